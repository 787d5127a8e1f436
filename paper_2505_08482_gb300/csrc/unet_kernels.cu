// Kernels of the learned warm start (a small U-Net on BF16 tensor cores):
// a BF16 GEMM with FP32 accumulation on the warp-level tensor-core
// instructions (mma.sync m16n8k16, operands staged with cp.async and read
// with ldmatrix), im2col for 3x3 convolutions in NHWC layout, transposes,
// pooling, upsampling, concatenation, bias/ReLU, the MSE loss and Adam.
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cstdint>

#include "kfixed.cuh"
#include "pat_internal.h"
#include "unet.h"

namespace pat {

// ---------------------------------------------------------------------------
// GEMM  C[M][N] = A[M][K] . B[N][K]^T  (both operands K-contiguous, K % 8 == 0)
// epilogue: (+ bias[n]) (ReLU) -> bf16 or fp32 store, or fp32 atomic add (split K)
namespace gemm {
constexpr int BM = 128, BN = 128, BK = 32, STAGES = 3, PITCH = BK + 8;   // bf16 elements per smem row
constexpr int THREADS = 256;

__device__ __forceinline__ uint32_t smem_u32(const void* p) {
    return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}
__device__ __forceinline__ void cp_async16(void* smem, const void* gmem, bool valid) {
    const int sz = valid ? 16 : 0;   // zero-fill outside the matrix
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;\n" ::"r"(smem_u32(smem)), "l"(gmem), "r"(sz));
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;\n" ::); }
template <int N>
__device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_group %0;\n" ::"n"(N)); }

__device__ __forceinline__ void ldmatrix_x4(uint32_t (&r)[4], const void* p) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];\n"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
                 : "r"(smem_u32(p)));
}
__device__ __forceinline__ void mma_bf16(float (&d)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
    asm volatile(
        "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, "
        "{%0,%1,%2,%3};\n"
        : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
        : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

struct Args {
    const __nv_bfloat16* A;
    const __nv_bfloat16* B;
    int M, N, K;
    int lda, ldb;          // row pitches (elements) of A and B
    const float* bias;     // [N] or null
    int relu;
    void* C;
    int ldc;
    int out_mode;          // 0 bf16 store, 1 fp32 store, 2 fp32 atomic add
    int ksplit;            // K range per blockIdx.z
};

__global__ void __launch_bounds__(THREADS) k_gemm(Args a) {
    extern __shared__ __align__(16) unsigned char smraw[];
    __nv_bfloat16* sA = reinterpret_cast<__nv_bfloat16*>(smraw);
    __nv_bfloat16* sB = sA + STAGES * BM * PITCH;
    const int tid = threadIdx.x, warp = tid / 32, lane = tid % 32;
    const int wm = warp / 4, wn = warp % 4;          // 2 x 4 warps, warp tile 64 x 32
    const int m0 = blockIdx.y * BM, n0 = blockIdx.x * BN;
    const int kb = blockIdx.z * a.ksplit;
    const int ke = min(a.K, kb + a.ksplit);
    const int nk = (ke - kb + BK - 1) / BK;
    float acc[4][4][4];
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j)
#pragma unroll
            for (int q = 0; q < 4; ++q) acc[i][j][q] = 0.f;

    auto load_stage = [&](int stage, int kt) {
        const int k0 = kb + kt * BK;
#pragma unroll
        for (int it = 0; it < 2; ++it) {
            const int c = tid + it * THREADS;       // 512 chunks of 8 bf16 per operand tile
            const int row = c / 4, kc = (c % 4) * 8;
            const int gk = k0 + kc;
            const bool kin = gk < ke;
            const int gm = m0 + row, gn = n0 + row;
            const bool va = kin && gm < a.M, vb = kin && gn < a.N;
            cp_async16(sA + (stage * BM + row) * PITCH + kc, a.A + (va ? size_t(gm) * a.lda + gk : 0), va);
            cp_async16(sB + (stage * BN + row) * PITCH + kc, a.B + (vb ? size_t(gn) * a.ldb + gk : 0), vb);
        }
    };
#pragma unroll
    for (int s = 0; s < STAGES - 1; ++s) {
        if (s < nk) load_stage(s, s);
        cp_async_commit();
    }
    for (int kt = 0; kt < nk; ++kt) {
        cp_async_wait<STAGES - 2>();
        __syncthreads();
        const int nxt = kt + STAGES - 1;
        if (nxt < nk) load_stage(nxt % STAGES, nxt);
        cp_async_commit();
        const __nv_bfloat16* tA = sA + (kt % STAGES) * BM * PITCH;
        const __nv_bfloat16* tB = sB + (kt % STAGES) * BN * PITCH;
#pragma unroll
        for (int kk = 0; kk < BK; kk += 16) {
            uint32_t af[4][4], bf[2][4];
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const int row = wm * 64 + i * 16 + (lane % 16);
                ldmatrix_x4(af[i], tA + row * PITCH + kk + (lane / 16) * 8);
            }
#pragma unroll
            for (int j = 0; j < 2; ++j) {
                const int row = wn * 32 + j * 16 + (lane % 8) + (lane / 16) * 8;
                ldmatrix_x4(bf[j], tB + row * PITCH + kk + ((lane / 8) % 2) * 8);
            }
#pragma unroll
            for (int i = 0; i < 4; ++i)
#pragma unroll
                for (int j = 0; j < 4; ++j) mma_bf16(acc[i][j], af[i], bf[j / 2][(j % 2) * 2], bf[j / 2][(j % 2) * 2 + 1]);
        }
    }
    cp_async_wait<0>();
    // epilogue
    const int g = lane / 4, t4 = lane % 4;
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j)
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const int m = m0 + wm * 64 + i * 16 + g + h * 8;
                const int n = n0 + wn * 32 + j * 8 + t4 * 2;
                if (m >= a.M) continue;
#pragma unroll
                for (int e = 0; e < 2; ++e) {
                    const int nn = n + e;
                    if (nn >= a.N) continue;
                    float v = acc[i][j][h * 2 + e];
                    if (a.bias) v += a.bias[nn];
                    if (a.relu) v = fmaxf(v, 0.f);
                    const size_t o = size_t(m) * a.ldc + nn;
                    if (a.out_mode == 0)
                        static_cast<__nv_bfloat16*>(a.C)[o] = __float2bfloat16(v);
                    else if (a.out_mode == 1)
                        static_cast<float*>(a.C)[o] = v;
                    else
                        atomicAdd(static_cast<float*>(a.C) + o, v);
                }
            }
}
}  // namespace gemm

int unet_gemm(cudaStream_t st, const __nv_bfloat16* A, int lda, const __nv_bfloat16* B, int ldb, int M, int N,
              int K, const float* bias, int relu, void* C, int ldc, int out_mode, int splitk) {
    if (K % 8 || lda % 8 || ldb % 8 || M <= 0 || N <= 0 || K <= 0) {
        set_error("unet_gemm: K and the operand pitches must be multiples of 8 (M=%d N=%d K=%d)", M, N, K);
        return PAT_EINVAL;
    }
    static bool configured = false;
    const size_t smem = size_t(gemm::STAGES) * (gemm::BM + gemm::BN) * gemm::PITCH * sizeof(__nv_bfloat16);
    if (!configured) {
        PAT_CUDA(cudaFuncSetAttribute(gemm::k_gemm, cudaFuncAttributeMaxDynamicSharedMemorySize, int(smem)));
        configured = true;
    }
    splitk = splitk < 1 ? 1 : splitk;
    int ks = (K + splitk - 1) / splitk;
    ks = (ks + gemm::BK - 1) / gemm::BK * gemm::BK;
    const int nz = (K + ks - 1) / ks;
    gemm::Args a{A, B, M, N, K, lda, ldb, bias, relu, C, ldc, out_mode, ks};
    dim3 grid((N + gemm::BN - 1) / gemm::BN, (M + gemm::BM - 1) / gemm::BM, nz);
    count_launch();
    gemm::k_gemm<<<grid, gemm::THREADS, smem, st>>>(a);
    cudaError_t e = cudaGetLastError();
    return e == cudaSuccess ? PAT_OK : cuda_fail(e, "k_gemm");
}

// ---------------------------------------------------------------------------
// elementwise / layout kernels (NHWC, channel counts padded to multiples of 8)
static unsigned nblk(size_t n) {
    size_t b = (n + 255) / 256;
    return unsigned(b > 65535 * 8 ? 65535 * 8 : (b < 1 ? 1 : b));
}
#define GRID_STRIDE(i, n) for (size_t i = size_t(blockIdx.x) * blockDim.x + threadIdx.x; i < (n); i += size_t(gridDim.x) * blockDim.x)

// Eight channels (16 bytes) per thread in the kernels below: NHWC with channel counts in multiples of 8.
union Bf8 {
    uint4 u;
    __nv_bfloat16 h[8];
};

// col[b][y][x][tap * C + c] = in[b][y+dy][x+dx][c] (zero outside), tap = (dy+1)*3 + (dx+1); flip: tap -> 8 - tap;
// rows of kp >= 9 C elements, the rest zero
__global__ void k_im2col(const __nv_bfloat16* __restrict__ in, __nv_bfloat16* __restrict__ col, int B, int H, int W,
                         int C, int ldc_in, int flip, int kp) {
    pdl_wait_then_release();
    const int C8 = C / 8, K8 = kp / 8;
    const size_t total = size_t(B) * H * W * K8;
    GRID_STRIDE(i, total) {
        const int k = int(i % K8);
        const size_t p = i / K8;
        const int tap = k / C8, c = k - tap * C8;
        const int x = int(p % W), y = int((p / W) % H);
        const int t = flip ? 8 - tap : tap;
        const int yy = y + t / 3 - 1, xx = x + t % 3 - 1;
        uint4 v = make_uint4(0, 0, 0, 0);
        if (tap < 9 && yy >= 0 && yy < H && xx >= 0 && xx < W)
            v = *reinterpret_cast<const uint4*>(in + (p + (yy - y) * (long long)W + (xx - x)) * ldc_in + c * 8);
        *reinterpret_cast<uint4*>(col + p * kp + size_t(k) * 8) = v;
    }
}

// out[c][r] = in[r][c] for an R x C bf16 matrix with row pitch ld
__global__ void k_transpose(const __nv_bfloat16* __restrict__ in, __nv_bfloat16* __restrict__ out, int R, int C,
                            int ld) {
    __shared__ __nv_bfloat16 t[32][33];
    for (int bx = blockIdx.x; bx < (C + 31) / 32; bx += gridDim.x)
        for (int by = blockIdx.y; by < (R + 31) / 32; by += gridDim.y) {
            const int c = bx * 32 + threadIdx.x;
            for (int j = threadIdx.y; j < 32; j += blockDim.y) {
                const int r = by * 32 + j;
                t[j][threadIdx.x] = (r < R && c < C) ? in[size_t(r) * ld + c] : __float2bfloat16(0.f);
            }
            __syncthreads();
            const int r2 = by * 32 + threadIdx.x;
            for (int j = threadIdx.y; j < 32; j += blockDim.y) {
                const int c2 = bx * 32 + j;
                if (c2 < C && r2 < R) out[size_t(c2) * R + r2] = t[threadIdx.x][j];
            }
            __syncthreads();
        }
}

// 2x2 max pooling (NHWC); idx records the argmax (0..3) for the backward
__global__ void k_maxpool(const __nv_bfloat16* __restrict__ in, __nv_bfloat16* __restrict__ out,
                          unsigned char* __restrict__ idx, int B, int H, int W, int C) {
    pdl_wait_then_release();
    const int Ho = H / 2, Wo = W / 2, C8 = C / 8;
    const size_t total = size_t(B) * Ho * Wo * C8;
    GRID_STRIDE(i, total) {
        const int c = int(i % C8) * 8;
        size_t r = i / C8;
        const int x = int(r % Wo);
        r /= Wo;
        const int y = int(r % Ho);
        const int b = int(r / Ho);
        Bf8 v[4], o;
        for (int q = 0; q < 4; ++q)
            v[q].u = *reinterpret_cast<const uint4*>(in + ((size_t(b) * H + 2 * y + q / 2) * W + 2 * x + q % 2) * C + c);
        unsigned char ix[8];
#pragma unroll
        for (int j = 0; j < 8; ++j) {
            float best = -3.0e38f;
            int bi = 0;
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const float f = __bfloat162float(v[q].h[j]);
                if (f > best) {
                    best = f;
                    bi = q;
                }
            }
            o.h[j] = __float2bfloat16(best);
            ix[j] = (unsigned char)bi;
        }
        *reinterpret_cast<uint4*>(out + i * 8) = o.u;
        *reinterpret_cast<uint2*>(idx + i * 8) = *reinterpret_cast<const uint2*>(ix);
    }
}

// gradient of an encoder output y (pooled and, from channel `off` of cat's gradient, skipped to the
// decoder): din = [y > 0] (unpool(dout) + cat[off ..]), rounded as the two steps one after the other
__global__ void k_enc_bwd(const __nv_bfloat16* __restrict__ dout, const unsigned char* __restrict__ idx,
                          const __nv_bfloat16* __restrict__ cat, int ldcat, int off, const __nv_bfloat16* __restrict__ yv,
                          __nv_bfloat16* __restrict__ din, int B, int H, int W, int C) {
    const int Ho = H / 2, Wo = W / 2, C8 = C / 8;
    const size_t total = size_t(B) * Ho * Wo * C8;
    GRID_STRIDE(i, total) {
        const int c = int(i % C8) * 8;
        size_t r = i / C8;
        const int x = int(r % Wo);
        r /= Wo;
        const int y = int(r % Ho);
        const int b = int(r / Ho);
        Bf8 d;
        d.u = *reinterpret_cast<const uint4*>(dout + i * 8);
        uint2 ixu = *reinterpret_cast<const uint2*>(idx + i * 8);
        const unsigned char* ix = reinterpret_cast<const unsigned char*>(&ixu);
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const size_t p = (size_t(b) * H + 2 * y + q / 2) * W + 2 * x + q % 2;
            Bf8 s, yy, o;
            s.u = *reinterpret_cast<const uint4*>(cat + p * ldcat + off + c);
            yy.u = *reinterpret_cast<const uint4*>(yv + p * C + c);
#pragma unroll
            for (int j = 0; j < 8; ++j) {
                const float v = (ix[j] == q ? __bfloat162float(d.h[j]) : 0.f) + __bfloat162float(s.h[j]);
                o.h[j] = __float2bfloat16(__bfloat162float(yy.h[j]) > 0.f ? v : 0.f);
            }
            *reinterpret_cast<uint4*>(din + p * C + c) = o.u;
        }
    }
}

// decoder input: cat = [nearest 2x upsampling of src (Cs channels) | skip (Ck channels)]
__global__ void k_concat(const __nv_bfloat16* __restrict__ src, const __nv_bfloat16* __restrict__ skip,
                         __nv_bfloat16* __restrict__ cat, int B, int Hs, int Ws, int Cs, int Ck) {
    pdl_wait_then_release();
    const int H = Hs * 2, W = Ws * 2, C8 = (Cs + Ck) / 8;
    const size_t total = size_t(B) * H * W * C8;
    GRID_STRIDE(i, total) {
        const int c = int(i % C8) * 8;
        const size_t p = i / C8;
        const int x = int(p % W), y = int((p / W) % H);
        const int b = int(p / (size_t(W) * H));
        const __nv_bfloat16* s = c < Cs ? src + ((size_t(b) * Hs + y / 2) * Ws + x / 2) * Cs + c : skip + p * Ck + (c - Cs);
        *reinterpret_cast<uint4*>(cat + i * 8) = *reinterpret_cast<const uint4*>(s);
    }
}

// backward of the nearest upsampling and of the ReLU below it: dsrc = [y > 0] sum of the 4 children of
// the first C channels of cat's gradient (fp32 sum)
__global__ void k_upsample_bwd(const __nv_bfloat16* __restrict__ cat, const __nv_bfloat16* __restrict__ yv,
                               __nv_bfloat16* __restrict__ dsrc, int B, int Hs, int Ws, int C, int ldo) {
    const int H = Hs * 2, W = Ws * 2, C8 = C / 8;
    const size_t total = size_t(B) * Hs * Ws * C8;
    GRID_STRIDE(i, total) {
        const int c = int(i % C8) * 8;
        size_t r = i / C8;
        const int x = int(r % Ws);
        r /= Ws;
        const int y = int(r % Hs);
        const int b = int(r / Hs);
        float s[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            Bf8 v;
            v.u = *reinterpret_cast<const uint4*>(cat + ((size_t(b) * H + 2 * y + q / 2) * W + 2 * x + q % 2) * ldo + c);
#pragma unroll
            for (int j = 0; j < 8; ++j) s[j] += __bfloat162float(v.h[j]);
        }
        Bf8 yy, o;
        yy.u = *reinterpret_cast<const uint4*>(yv + i * 8);
#pragma unroll
        for (int j = 0; j < 8; ++j) o.h[j] = __float2bfloat16(__bfloat162float(yy.h[j]) > 0.f ? s[j] : 0.f);
        *reinterpret_cast<uint4*>(dsrc + i * 8) = o.u;
    }
}

// ReLU backward in place: g *= (y > 0)
__global__ void k_relu_bwd(__nv_bfloat16* __restrict__ g, const __nv_bfloat16* __restrict__ y, size_t n8) {
    GRID_STRIDE(i, n8) {
        Bf8 a, b;
        a.u = reinterpret_cast<const uint4*>(g)[i];
        b.u = reinterpret_cast<const uint4*>(y)[i];
#pragma unroll
        for (int j = 0; j < 8; ++j)
            if (!(__bfloat162float(b.h[j]) > 0.f)) a.h[j] = __float2bfloat16(0.f);
        reinterpret_cast<uint4*>(g)[i] = a.u;
    }
}

// Bias gradient db[c] = sum_p g[p][c] in a fixed order: block (b, z) sums every gridDim.x-th group of 256 / G pixels
// for 8 G channels from 64 z on into part[b][C], four reads in flight per thread; the block that is done last
// sums the parts.
constexpr int kBiasBlocks = 296;
__global__ void __launch_bounds__(256) k_bias_grad(const __nv_bfloat16* __restrict__ g, float* __restrict__ part,
                                                   unsigned* __restrict__ done, float* __restrict__ db, size_t P, int C) {
    pdl_wait_then_release();
    __shared__ float red[256][9];
    __shared__ bool last;
    const int c0 = blockIdx.y * 64, G = min(8, (C - c0) / 8);
    const int R = 256 / G, cg = threadIdx.x % G, pr = threadIdx.x / G;
    float s[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
    if (pr < R) {
        const size_t step = size_t(gridDim.x) * R;
        const __nv_bfloat16* src = g + c0 + cg * 8;
        for (size_t p = size_t(blockIdx.x) * R + pr; p < P; p += 4 * step) {
            Bf8 v[4];
#pragma unroll
            for (int q = 0; q < 4; ++q)
                v[q].u = p + q * step < P ? *reinterpret_cast<const uint4*>(src + (p + q * step) * C) : make_uint4(0, 0, 0, 0);
#pragma unroll
            for (int q = 0; q < 4; ++q)
#pragma unroll
                for (int j = 0; j < 8; ++j) s[j] += __bfloat162float(v[q].h[j]);
        }
    }
#pragma unroll
    for (int j = 0; j < 8; ++j) red[threadIdx.x][j] = s[j];
    __syncthreads();
    if (threadIdx.x < 8 * G) {
        const int c = threadIdx.x / 8, j = threadIdx.x % 8;
        float t = 0.f;
        for (int r = 0; r < R; ++r) t += red[r * G + c][j];
        part[size_t(blockIdx.x) * C + c0 + c * 8 + j] = t;
    }
    __syncthreads();
    if (threadIdx.x == 0) {   // one fence for the block's parts, ordered by the barrier
        __threadfence();
        last = atomicAdd(done, 1u) == gridDim.x * gridDim.y - 1;
        if (last) *done = 0;
        __threadfence();
    }
    __syncthreads();
    if (!last) return;
    // 256 / C threads per channel (at least one), consecutive threads on consecutive channels
    float* sum = &red[0][0];
    const int per = max(1, 256 / C), nb = int(gridDim.x);
    for (int cb = 0; cb < C; cb += 256) {
        const int w = min(C - cb, 256), q = threadIdx.x / w, c = cb + threadIdx.x - q * w;
        float t = 0.f;
        if (q < per) {
#pragma unroll 8
            for (int b = q; b < nb; b += per) t += __ldcg(part + size_t(b) * C + c);
        }
        __syncthreads();
        sum[threadIdx.x] = t;
        __syncthreads();
        if (q == 0) {
            for (int i = 1; i < per; ++i) t += sum[i * w + threadIdx.x];
            db[c] = t;
        }
        __syncthreads();
    }
}

// Final 1x1 convolution to one channel: out[p] = sum_c y[p][c] w[c] + b.  A warp takes 16 pixels as the rows of
// m16n8k16 MMAs whose second operand has w in column 0 and zeros elsewhere: the same 16-channel sums, in the
// same order, as the GEMM above, for one read of y.
__global__ void __launch_bounds__(256) k_head(const __nv_bfloat16* __restrict__ y, const __nv_bfloat16* __restrict__ w,
                                              const float* __restrict__ bias, float* __restrict__ out, size_t P, int C) {
    const int lane = threadIdx.x & 31, g = lane >> 2, t2 = (lane & 3) * 2;
    const size_t warps = size_t(gridDim.x) * (blockDim.x >> 5);
    for (size_t p0 = (size_t(blockIdx.x) * (blockDim.x >> 5) + (threadIdx.x >> 5)) * 16; p0 < P; p0 += warps * 16) {
        float acc[4] = {0.f, 0.f, 0.f, 0.f};
        auto pair = [&](const __nv_bfloat16* row, bool ok, int c) {
            return ok && c < C ? *reinterpret_cast<const uint32_t*>(row + c) : 0u;
        };
        const bool ok0 = p0 + g < P, ok1 = p0 + g + 8 < P;
        const __nv_bfloat16* r0 = y + (p0 + g) * C;
        const __nv_bfloat16* r1 = r0 + size_t(8) * C;
        for (int c = 0; c < C; c += 16) {
            const uint32_t a[4] = {pair(r0, ok0, c + t2), pair(r1, ok1, c + t2), pair(r0, ok0, c + t2 + 8),
                                   pair(r1, ok1, c + t2 + 8)};
            gemm::mma_bf16(acc, a, pair(w, g == 0, c + t2), pair(w, g == 0, c + t2 + 8));
        }
        if (t2 == 0) {   // column 0 of rows g, g + 8
            if (ok0) out[p0 + g] = acc[0] + bias[0];
            if (ok1) out[p0 + g + 8] = acc[2] + bias[0];
        }
    }
}

// Loss L = mean (out - target)^2 and the backward of the final convolution in one pass over its input
// y: d = bf16(2 (out - target) / n) per pixel, dy = [y > 0] bf16(d w), and per block the partial sums of
// dW[c] = sum d y[c], db = sum d (part[b][C + 1]) and of the loss (lpart[b]).  Eight channels per thread, so that
// a block covers 2048 channels; blockIdx.y: the 2048 channels, of which the first also take db and the loss.
constexpr int kHeadBlocks = 296;
__global__ void __launch_bounds__(256) k_head_bwd(const float* __restrict__ out, const float* __restrict__ tgt,
                                                  const __nv_bfloat16* __restrict__ y,
                                                  const __nv_bfloat16* __restrict__ w, __nv_bfloat16* __restrict__ dy,
                                                  float* __restrict__ part, double* __restrict__ lpart, size_t P, int C) {
    __shared__ float red[256][9];
    __shared__ double lred[256];
    const int g0 = blockIdx.y * 256, G = min(256, C / 8 - g0), R = 256 / G;
    const int cg = g0 + threadIdx.x % G, pr = threadIdx.x / G;
    float wv[8], s[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f}, sb = 0.f;
    double ls = 0.0;
#pragma unroll
    for (int j = 0; j < 8; ++j) wv[j] = __bfloat162float(w[cg * 8 + j]);
    if (pr < R)
        for (size_t p = size_t(blockIdx.x) * R + pr; p < P; p += size_t(gridDim.x) * R) {
            const float e = out[p] - tgt[p];
            const float d = __bfloat162float(__float2bfloat16(2.f * e / float(P)));
            if (cg == 0) {
                ls += double(e) * e;
                sb += d;
            }
            Bf8 v, o;
            v.u = *reinterpret_cast<const uint4*>(y + p * C + cg * 8);
#pragma unroll
            for (int j = 0; j < 8; ++j) {
                const float f = __bfloat162float(v.h[j]);
                s[j] += d * f;
                o.h[j] = __float2bfloat16(f > 0.f ? d * wv[j] : 0.f);
            }
            *reinterpret_cast<uint4*>(dy + p * C + cg * 8) = o.u;
        }
#pragma unroll
    for (int j = 0; j < 8; ++j) red[threadIdx.x][j] = s[j];
    red[threadIdx.x][8] = sb;
    lred[threadIdx.x] = ls;
    __syncthreads();
    for (int t = threadIdx.x; t <= 8 * G; t += 256) {
        float v = 0.f;
        if (t < 8 * G)
            for (int r = 0; r < R; ++r) v += red[r * G + t / 8][t % 8];
        else
            for (int r = 0; r < R; ++r) v += red[r * G][8];
        if (t < 8 * G || g0 == 0) part[size_t(blockIdx.x) * (C + 1) + (t < 8 * G ? 8 * g0 + t : C)] = v;
    }
    for (int k = 128; k > 0; k >>= 1) {
        __syncthreads();
        if (threadIdx.x < k) lred[threadIdx.x] += lred[threadIdx.x + k];
    }
    if (threadIdx.x == 0 && g0 == 0) lpart[blockIdx.x] = lred[0];
}
__global__ void k_head_sum(const float* __restrict__ part, const double* __restrict__ lpart, int nblk,
                           float* __restrict__ dw, float* __restrict__ db, double* __restrict__ loss, double scale, int C) {
    const int lane = threadIdx.x, t = blockIdx.x;
    if (t <= C) {
        float s = 0.f;
        for (int b = lane; b < nblk; b += 32) s += part[size_t(b) * (C + 1) + t];
        for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
        if (lane == 0) *(t < C ? dw + t : db) = s;
    } else {
        double s = 0.0;
        for (int b = lane; b < nblk; b += 32) s += lpart[b];
        for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
        if (lane == 0) *loss = s * scale;
    }
}

// Adam on fp32 master weights
__global__ void k_adam(float* __restrict__ w, const float* __restrict__ g, float* __restrict__ m, float* __restrict__ v, size_t n, float lr, float b1, float b2, float eps,
                       float bc1, float bc2) {
    GRID_STRIDE(i, n) {
        const float gi = g[i];
        const float mi = b1 * m[i] + (1.f - b1) * gi;
        const float vi = b2 * v[i] + (1.f - b2) * gi * gi;
        m[i] = mi;
        v[i] = vi;
        const float wi = w[i] - lr * (mi / bc1) / (sqrtf(vi / bc2) + eps);
        w[i] = wi;
    }
}

// bf16 copies of every convolution's weights W[co][tap][ci] and, for the data gradient of the 3x3
// ones, Wt[ci][tap][co]; blockIdx.y: convolution
__global__ void k_weights(const float* __restrict__ param, __nv_bfloat16* __restrict__ wb, __nv_bfloat16* __restrict__ wt,
                          const ConvDesc* __restrict__ desc) {
    const ConvDesc d = desc[blockIdx.y];
    const int taps = d.k * d.k;
    const size_t n = size_t(d.cout) * taps * d.cin;
    GRID_STRIDE(i, n) {
        const __nv_bfloat16 v = __float2bfloat16(param[d.w_off + i]);
        wb[d.wb_off + i] = v;
        if (d.k == 3) {
            const int ci = int(i % d.cin);
            const size_t r = i / d.cin;
            const int tap = int(r % 9), co = int(r / 9);
            wt[d.wb_off + (size_t(ci) * 9 + tap) * d.cout + co] = v;
        }
    }
}

// input staging: fp32 [B][Cin][H][W] (NCHW, as the solver produces images) -> bf16 NHWC with C padded
__global__ void k_pack_input(const float* __restrict__ in, __nv_bfloat16* __restrict__ out, int B, int Cin, size_t HW,
                             int Cp) {
    const int C8 = Cp / 8;
    GRID_STRIDE(i, size_t(B) * HW * C8) {
        const size_t p = i % HW;   // pixels fastest: the reads of a channel plane are contiguous
        const int g = int((i / HW) % C8);
        const int b = int(i / (HW * C8));
        Bf8 v;
#pragma unroll
        for (int j = 0; j < 8; ++j) {
            const int c = g * 8 + j;
            v.h[j] = __float2bfloat16(c < Cin ? in[(size_t(b) * Cin + c) * HW + p] : 0.f);
        }
        *reinterpret_cast<uint4*>(out + (size_t(b) * HW + p) * Cp + g * 8) = v.u;
    }
}

// ---- launchers ----
#define LAUNCH_CHECK(name)                                                        \
    do {                                                                          \
        count_launch();                                                           \
        cudaError_t e_ = cudaGetLastError();                                      \
        if (e_ != cudaSuccess) return cuda_fail(e_, name);                        \
    } while (0)

int unet_im2col(cudaStream_t st, const __nv_bfloat16* in, __nv_bfloat16* col, int B, int H, int W, int C, int ldc_in,
                int flip, int kp) {
    k_im2col<<<nblk(size_t(B) * H * W * (kp / 8)), 256, 0, st>>>(in, col, B, H, W, C, ldc_in, flip, kp);
    LAUNCH_CHECK("k_im2col");
    return PAT_OK;
}
int unet_transpose(cudaStream_t st, const __nv_bfloat16* in, __nv_bfloat16* out, int R, int C, int ld) {
    dim3 grid(std::min((C + 31) / 32, 1024), std::min((R + 31) / 32, 1024));
    k_transpose<<<grid, dim3(32, 8), 0, st>>>(in, out, R, C, ld);
    LAUNCH_CHECK("k_transpose");
    return PAT_OK;
}
int unet_maxpool(cudaStream_t st, const __nv_bfloat16* in, __nv_bfloat16* out, unsigned char* idx, int B, int H, int W,
                 int C) {
    launch_pdl(k_maxpool, nblk(size_t(B) * H * W * C / 32), dim3(256), 0, st, true, in, out, idx, B, H, W, C);
    LAUNCH_CHECK("k_maxpool");
    return PAT_OK;
}
int unet_enc_bwd(cudaStream_t st, const __nv_bfloat16* dout, const unsigned char* idx, const __nv_bfloat16* cat, int ldcat,
                 int off, const __nv_bfloat16* y, __nv_bfloat16* din, int B, int H, int W, int C) {
    k_enc_bwd<<<nblk(size_t(B) * H * W * C / 32), 256, 0, st>>>(dout, idx, cat, ldcat, off, y, din, B, H, W, C);
    LAUNCH_CHECK("k_enc_bwd");
    return PAT_OK;
}
int unet_concat(cudaStream_t st, const __nv_bfloat16* src, const __nv_bfloat16* skip, __nv_bfloat16* cat, int B, int Hs,
                int Ws, int Cs, int Ck) {
    launch_pdl(k_concat, nblk(size_t(B) * Hs * Ws * 4 * (Cs + Ck) / 8), dim3(256), 0, st, true, src, skip, cat, B, Hs, Ws, Cs,
               Ck);
    LAUNCH_CHECK("k_concat");
    return PAT_OK;
}
int unet_upsample_bwd(cudaStream_t st, const __nv_bfloat16* cat, const __nv_bfloat16* y, __nv_bfloat16* dsrc, int B, int Hs,
                      int Ws, int C, int ldo) {
    k_upsample_bwd<<<nblk(size_t(B) * Hs * Ws * C / 8), 256, 0, st>>>(cat, y, dsrc, B, Hs, Ws, C, ldo);
    LAUNCH_CHECK("k_upsample_bwd");
    return PAT_OK;
}
int unet_relu_bwd(cudaStream_t st, __nv_bfloat16* g, const __nv_bfloat16* y, size_t n) {
    k_relu_bwd<<<nblk(n / 8), 256, 0, st>>>(g, y, n / 8);
    LAUNCH_CHECK("k_relu_bwd");
    return PAT_OK;
}
int unet_bias_grad(cudaStream_t st, const __nv_bfloat16* g, float* db, float* part, unsigned* done, size_t P, int C) {
    // at least 16 pixels per thread: the last block's sum grows with the blocks
    const size_t group = 256 / std::min(8, C / 8);
    const unsigned nb = unsigned(std::max<size_t>(1, std::min<size_t>(kBiasBlocks, P / (16 * group))));
    launch_pdl(k_bias_grad, dim3(nb, (C + 63) / 64), dim3(256), 0, st, true, g, part, done, db, P, C);
    LAUNCH_CHECK("k_bias_grad");
    return PAT_OK;
}
size_t unet_part_floats(int C) { return size_t(kBiasBlocks > kHeadBlocks ? kBiasBlocks : kHeadBlocks) * (C + 1); }
int unet_part_blocks() { return kHeadBlocks; }
int unet_head(cudaStream_t st, const __nv_bfloat16* y, const __nv_bfloat16* w, const float* bias, float* out, size_t P,
              int C) {
    k_head<<<unsigned(std::min<size_t>((P + 127) / 128, 65535)), 256, 0, st>>>(y, w, bias, out, P, C);
    LAUNCH_CHECK("k_head");
    return PAT_OK;
}
int unet_head_bwd(cudaStream_t st, const float* out, const float* tgt, const __nv_bfloat16* y, const __nv_bfloat16* w,
                  __nv_bfloat16* dy, float* part, double* lpart, float* dw, float* db, double* loss, size_t P, int C) {
    k_head_bwd<<<dim3(kHeadBlocks, (C / 8 + 255) / 256), 256, 0, st>>>(out, tgt, y, w, dy, part, lpart, P, C);
    LAUNCH_CHECK("k_head_bwd");
    k_head_sum<<<C + 2, 32, 0, st>>>(part, lpart, kHeadBlocks, dw, db, loss, 1.0 / double(P), C);
    LAUNCH_CHECK("k_head_sum");
    return PAT_OK;
}
int unet_adam(cudaStream_t st, float* w, const float* g, float* m, float* v, size_t n, float lr, float b1, float b2,
              float eps, float bc1, float bc2) {
    k_adam<<<nblk(n), 256, 0, st>>>(w, g, m, v, n, lr, b1, b2, eps, bc1, bc2);
    LAUNCH_CHECK("k_adam");
    return PAT_OK;
}
int unet_weights(cudaStream_t st, const float* param, __nv_bfloat16* wb, __nv_bfloat16* wt, const ConvDesc* desc, int n,
                 size_t most) {
    k_weights<<<dim3(std::min(nblk(most), 1024u), n), 256, 0, st>>>(param, wb, wt, desc);
    LAUNCH_CHECK("k_weights");
    return PAT_OK;
}
int unet_pack_input(cudaStream_t st, const float* in, __nv_bfloat16* out, int B, int Cin, int H, int W, int Cp) {
    k_pack_input<<<nblk(size_t(B) * H * W * Cp / 8), 256, 0, st>>>(in, out, B, Cin, size_t(H) * W, Cp);
    LAUNCH_CHECK("k_pack_input");
    return PAT_OK;
}

}  // namespace pat
