// Batched complex FFTs of 5-smooth length in shared memory (Stockham
// auto-sort, radix 2/3/4/5), used by the row and column passes of the
// k-space time stepping.  Twiddles come from a table exp(-2 pi i q / n),
// q < n, built in FP64 on the host and staged in shared memory.
#pragma once

#include <cuda_runtime.h>

namespace pat {

constexpr int kMaxStages = 12;

// Radix schedule of one FFT length: n = rad[0] * rad[1] * ... * rad[nrad-1].
struct FftDesc {
    int n;
    int nrad;
    int rad[kMaxStages];
    // per stage: ceil(2^32 / (n / rad)) and ceil(2^32 / Ns) (Ns: the sub-transforms already done), so that a division
    // of the stage's indices (below 2^20) is one multiplication
    unsigned inv_nb[kMaxStages];
    unsigned inv_ns[kMaxStages];
};

// Additions and real factors of complex values act on both parts alike: one packed instruction
// (fp32x2) each on the device, half the issue slots of two scalar ones at the same FP32 rate.
__host__ __device__ __forceinline__ float2 cadd(float2 a, float2 b) {
#ifdef __CUDA_ARCH__
    return __fadd2_rn(a, b);
#else
    return make_float2(a.x + b.x, a.y + b.y);
#endif
}
// a + s b
__host__ __device__ __forceinline__ float2 caxpy(float2 a, float s, float2 b) {
#ifdef __CUDA_ARCH__
    return __ffma2_rn(b, make_float2(s, s), a);
#else
    return make_float2(a.x + s * b.x, a.y + s * b.y);
#endif
}
__host__ __device__ __forceinline__ float2 csub(float2 a, float2 b) { return caxpy(a, -1.f, b); }
__host__ __device__ __forceinline__ float2 cscale(float2 a, float s) {
#ifdef __CUDA_ARCH__
    return __fmul2_rn(a, make_float2(s, s));
#else
    return make_float2(a.x * s, a.y * s);
#endif
}
// part by part
__host__ __device__ __forceinline__ float2 cprod(float2 a, float2 b) {
#ifdef __CUDA_ARCH__
    return __fmul2_rn(a, b);
#else
    return make_float2(a.x * b.x, a.y * b.y);
#endif
}
__host__ __device__ __forceinline__ float2 cmul(float2 a, float2 b) {
    return make_float2(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x);
}
// a * conj(b)
__host__ __device__ __forceinline__ float2 cmulc(float2 a, float2 b) {
    return make_float2(a.x * b.x + a.y * b.y, a.y * b.x - a.x * b.y);
}
// multiply by -i (forward) or +i (inverse)
template <bool INV, class C>
__host__ __device__ __forceinline__ C rot(C a) {
    return INV ? C{-a.y, a.x} : C{a.y, -a.x};
}
// the same in FP64, for the host's measurement of the transforms' gain
__host__ inline double2 cadd(double2 a, double2 b) { return {a.x + b.x, a.y + b.y}; }
__host__ inline double2 caxpy(double2 a, float s, double2 b) { return {a.x + double(s) * b.x, a.y + double(s) * b.y}; }
__host__ inline double2 csub(double2 a, double2 b) { return {a.x - b.x, a.y - b.y}; }
__host__ inline double2 cscale(double2 a, float s) { return {a.x * double(s), a.y * double(s)}; }
__host__ inline double2 cmul(double2 a, float2 b) { return {a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x}; }
__host__ inline double2 cmulc(double2 a, float2 b) { return {a.x * b.x + a.y * b.y, a.y * b.x - a.x * b.y}; }

// a + rot(b), a - rot(b): the parts change places, so these stay scalar
template <bool INV, class C>
__host__ __device__ __forceinline__ C crot_add(C a, C b) {
    return INV ? C{a.x - b.y, a.y + b.x} : C{a.x + b.y, a.y - b.x};
}
template <bool INV, class C>
__host__ __device__ __forceinline__ C crot_sub(C a, C b) {
    return crot_add<!INV>(a, b);
}

// In-register DFT of R points: v_q <- sum_m v_m exp(-+ 2 pi i m q / R).  C: float2, or double2 on the host (the
// same float constants in FP64 arithmetic).
template <int R, bool INV, class C>
__host__ __device__ __forceinline__ void dft_small(C (&v)[R]) {
    if constexpr (R == 2) {
        C a = v[0], b = v[1];
        v[0] = cadd(a, b);
        v[1] = csub(a, b);
    } else if constexpr (R == 3) {
        const float s3 = 0.86602540378443864676f;   // sin(2 pi / 3)
        const float sg = INV ? -s3 : s3;            // v1, v2 = m +- rot(s3 dif)
        C sum = cadd(v[1], v[2]);
        C dif = csub(v[1], v[2]);
        C m = caxpy(v[0], -0.5f, sum);
        v[0] = cadd(v[0], sum);
        v[1] = C{m.x + sg * dif.y, m.y - sg * dif.x};
        v[2] = C{m.x - sg * dif.y, m.y + sg * dif.x};
    } else if constexpr (R == 4) {
        C a = cadd(v[0], v[2]), b = csub(v[0], v[2]);
        C c = cadd(v[1], v[3]), d = csub(v[1], v[3]);
        v[0] = cadd(a, c);
        v[2] = csub(a, c);
        v[1] = crot_add<INV>(b, d);
        v[3] = crot_sub<INV>(b, d);
    } else if constexpr (R == 5) {
        const float c1 = 0.30901699437494742410f;    // cos(2 pi / 5)
        const float c2 = -0.80901699437494742410f;   // cos(4 pi / 5)
        const float s1 = 0.95105651629515357212f;    // sin(2 pi / 5)
        const float s2 = 0.58778525229247312917f;    // sin(4 pi / 5)
        C a1 = cadd(v[1], v[4]), b1 = csub(v[1], v[4]);
        C a2 = cadd(v[2], v[3]), b2 = csub(v[2], v[3]);
        C m1 = caxpy(caxpy(v[0], c1, a1), c2, a2);
        C m2 = caxpy(caxpy(v[0], c2, a1), c1, a2);
        C u1 = caxpy(cscale(b1, s1), s2, b2);
        C u2 = caxpy(cscale(b1, s2), -s1, b2);
        v[0] = cadd(cadd(v[0], a1), a2);
        v[1] = crot_add<INV>(m1, u1);
        v[4] = crot_sub<INV>(m1, u1);
        v[2] = crot_add<INV>(m2, u2);
        v[3] = crot_sub<INV>(m2, u2);
    }
}

// One Stockham stage of radix R over nseq sequences (stride ss) from src to dst.
// Ns is the length of the sub-transforms already done.
template <int R, bool INV>
__device__ __forceinline__ void stockham_stage(const float2* __restrict__ src, float2* __restrict__ dst,
                                               int n, int Ns, int nseq, int ss,
                                               const float2* __restrict__ tw, unsigned inv_nb, unsigned inv_ns) {
    const int nb = n / R;
    const int tstride = n / (Ns * R);
    const int total = nseq * nb;
    for (int t = threadIdx.x; t < total; t += blockDim.x) {
        const int s = nb > 1 ? int(__umulhi(unsigned(t), inv_nb)) : t;
        const int j = t - s * nb;
        const float2* in = src + s * ss;
        float2* out = dst + s * ss;
        const int k = Ns > 1 ? j - int(__umulhi(unsigned(j), inv_ns)) * Ns : 0;
        float2 v[R];
#pragma unroll
        for (int r = 0; r < R; ++r) v[r] = in[j + r * nb];
        if (Ns > 1) {
#pragma unroll
            for (int r = 1; r < R; ++r) {
                const float2 w = tw[r * k * tstride];
                v[r] = INV ? cmulc(v[r], w) : cmul(v[r], w);
            }
        }
        dft_small<R, INV>(v);
        const int base = (j - k) * R + k;
#pragma unroll
        for (int r = 0; r < R; ++r) out[base + r * Ns] = v[r];
    }
}

// FFT of nseq sequences of length fd.n held at a[s*ss + i]; b is scratch of
// the same shape.  Unnormalised; INV selects exp(+2 pi i ...).  All threads
// of the block must call it; it ends with __syncthreads().  Returns the
// buffer (a or b) that holds the result.
template <bool INV>
__device__ float2* fft_smem(float2* a, float2* b, int nseq, int ss, const FftDesc& fd,
                            const float2* __restrict__ tw) {
    int Ns = 1;
    for (int st = 0; st < fd.nrad; ++st) {
        const int R = fd.rad[st];
        switch (R) {
            case 2: stockham_stage<2, INV>(a, b, fd.n, Ns, nseq, ss, tw, fd.inv_nb[st], fd.inv_ns[st]); break;
            case 3: stockham_stage<3, INV>(a, b, fd.n, Ns, nseq, ss, tw, fd.inv_nb[st], fd.inv_ns[st]); break;
            case 4: stockham_stage<4, INV>(a, b, fd.n, Ns, nseq, ss, tw, fd.inv_nb[st], fd.inv_ns[st]); break;
            default: stockham_stage<5, INV>(a, b, fd.n, Ns, nseq, ss, tw, fd.inv_nb[st], fd.inv_ns[st]); break;
        }
        __syncthreads();
        float2* t = a;
        a = b;
        b = t;
        Ns *= R;
    }
    return a;
}

// One stage of stockham_stage for one sequence on the host, in FP64 arithmetic with the same float constants.
template <int R, bool INV>
inline void stockham_stage_host(const double2* src, double2* dst, int n, int Ns, const float2* tw) {
    const int nb = n / R, tstride = n / (Ns * R);
    for (int j = 0; j < nb; ++j) {
        const int k = j % Ns;
        double2 v[R];
        for (int r = 0; r < R; ++r) {
            v[r] = src[j + r * nb];
            if (r > 0 && Ns > 1) v[r] = INV ? cmulc(v[r], tw[r * k * tstride]) : cmul(v[r], tw[r * k * tstride]);
        }
        dft_small<R, INV>(v);
        for (int r = 0; r < R; ++r) dst[(j - k) * R + k + r * Ns] = v[r];
    }
}
template <bool INV>
inline double2* fft_host(double2* a, double2* b, const FftDesc& fd, const float2* tw) {
    int Ns = 1;
    for (int st = 0; st < fd.nrad; ++st) {
        switch (fd.rad[st]) {
            case 2: stockham_stage_host<2, INV>(a, b, fd.n, Ns, tw); break;
            case 3: stockham_stage_host<3, INV>(a, b, fd.n, Ns, tw); break;
            case 4: stockham_stage_host<4, INV>(a, b, fd.n, Ns, tw); break;
            default: stockham_stage_host<5, INV>(a, b, fd.n, Ns, tw); break;
        }
        double2* t = a;
        a = b;
        b = t;
        Ns *= fd.rad[st];
    }
    return a;
}

}  // namespace pat
