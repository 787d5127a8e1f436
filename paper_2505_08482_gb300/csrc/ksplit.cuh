// Split-axis passes of the k-space scheme: three launches per time step.
//
// The split-field scheme keeps u_x and rho_x apart from u_y and rho_y, and the PML factor of an
// x field depends on x alone.  Everything between the pressure and rho_x is therefore diagonal in
// ky: it can run on the lines (ky, x = 0..Ng-1) of the y half spectrum, and everything between the
// pressure and rho_y on the lines (kx, y = 0..Ng-1) of the x half spectrum.  A step is
//   to_lines : p = c^2 (rho_x + rho_y); R2C along y -> lines of axis 0, R2C along x -> axis 1
//   lines    : per line FFT, G, IFFT, velocity update, FFT, D, IFFT, density update
//   to_real  : C2R of the rho_x lines along y and of the rho_y lines along x
// and the discrete adjoint is the same three passes with their transposes.  kappa(kx, ky) is
// symmetric and both axes have the same spacing, so the two axes run the same code on the same
// tables.  Against the four-pass step (kfixed.cuh) this is 12 instead of 14 one-dimensional
// transforms of the half grid, 3 instead of 4 trips through L2 and three instead of seven
// half-spectrum packings; u and rho live as lines from step to step.
//
// Scaling (N = Ng, transforms unnormalised).  Pressure lines hold FFT(p), rho lines FFT(rho) / N (so
// that the inverse transform of to_real needs no factor) and u lines FFT(rho0 u) / sqrt(N); then G and
// D have the same multiplier, M = dt N^{-3/2} i k kappa exp(+-i k dx/2), without rho0, and so have the
// adjoint's G and D with rho lines FFT(rb), u lines FFT(ub / rho0) / sqrt(N) and q lines FFT(q) / N.
// The multiplier is one table, rounded once from FP64 (a factor rounded by itself would put the same
// relative error on every mode of every step, a wrong speed of sound) and divided by the gain of the float
// transform pairs that a mode meets (mode_gain, up to 7e-8 each): one along the line in each operator, one across the
// lines per step.
//
// What bounds the passes: with few data sets the latency of the three launches (L2 round trip and the
// chain of transforms, about ten warps per SM at 256^2, K = 8), with many the instruction issue of the
// transforms.  Measured on GB300, us per forward step, four-pass step -> this one: Ng 108, K = 1 11.5 ->
// 7.2; Ng 180, K = 4 14.3 -> 9.9; Ng 300, K = 8 23.3 -> 17.7; Ng 180, K = 64 64.6 -> 41.8; per gradient
// step (Ng 300, K = 8) 65.1 -> 50.0.  A pass takes its registers and shared memory sparingly: what it
// leaves free lets the CTAs of the next pass run their prologue (programmatic dependent launch).
#pragma once

#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstdint>
#include <type_traits>
#include <vector>

#include "dcheck.cuh"
#include "fft2l.cuh"
#include "geo.cuh"
#include "kfixed.cuh"

namespace pat {

// ---------------------------------------------------------------------------
// arguments (by value) of the three passes; lines are [axis][K][hc][N] float2, real fields [K][N][N]

enum { SP_COPY = 0, SP_PRESSURE = 1, SP_INIT = 2, SP_ADJOINT = 3 };

struct ToLinesArgs {
    int mode;
    const float* f0[2];   // field of axis 0 and 1: rho_x, rho_y (SP_PRESSURE), q_x, q_y (SP_ADJOINT), copied (SP_COPY)
    const float* f1[2];   // SP_COPY: a second field (gridDim.z = 2)
    float2* out0;
    float2* out1;
    float2 scale0, scale1;   // SP_COPY: factors of the lines (high and low part)
    const float* cg;      // c on the grid
    const float* p0;      // SP_INIT
    float* y;             // SP_PRESSURE, SP_INIT: traces, or null
    int tstep;
    float* hist;          // p^n written (SP_PRESSURE, SP_INIT; or null) or read (SP_ADJOINT)
    int slot;
    float* cbar;          // SP_ADJOINT
};

enum { SP_STEP = 0, SP_STEP_FIRST = 1, SP_STEP_ADJOINT = 2, SP_DIV = 3 };

struct LinesArgs {
    int mode;
    const float2* in;
    float2* u;
    float2* r;
    float2* out;   // SP_STEP_ADJOINT, SP_DIV
    float scale;   // SP_DIV: factor of out
};

struct ToRealArgs {
    const float2* in0;
    const float2* in1;   // gridDim.z = 2
    float* d0[2];
    float* d1[2];
    float2 scale0, scale1;   // factors (high and low part; {1, 0}: none)
    const float* resid;  // adjoint source added to axis 1 of field 0, or null
    int tstep;
    int zero;            // the lines are not read: the source alone (first adjoint step)
};

struct SplitOps {
    int ng, n1, n2;
    const double* (*mode_gain)();   // [ng] gain of a forward and inverse float transform per mode, minus 1
    int (*configure)();
    void (*to_lines)(const Geo&, cudaStream_t, const ToLinesArgs&, int fields, bool pdl);
    void (*lines)(const Geo&, cudaStream_t, const LinesArgs&);
    void (*to_real)(const Geo&, cudaStream_t, const ToRealArgs&, int fields);
};

const SplitOps* split_ops_for(int ng);   // nullptr: no split-axis passes for this grid side

// v (hi + lo): the factor to about twice FP32 precision, rounded once
__device__ __forceinline__ float2 scale2(float2 v, float2 s) { return caxpy(cscale(v, s.y), s.x, v); }

// ---------------------------------------------------------------------------
// real -> lines.  A CTA transforms PP pairs of neighbouring columns (axis 0) or rows (axis 1): a
// pair (a, b) is one complex transform of a + i b.  The pair index runs fastest over the threads,
// so that both the reads of axis 0 and the line writes (float4: both members of a pair) cover
// consecutive addresses of PP pairs.
//
// The real fields (to_lines) and the lines (to_real) of a tile come in through shared memory by
// asynchronous 16-byte copies, all in flight at once without registers: with register loads the
// compiler kept only a few in flight and the latency of the L2 round trips set the pass time.
// The transpose buffer takes the place of the staged tile once every thread has read it.
template <class F, int PP>
struct PairSmem {
    // stride of a staged row: members 2c, 2c+1 of the pairs of a warp on different banks, 16-byte rows
    static constexpr int S = F::N + ((4 - F::N % 8) + 8) % 8;
    static_assert(S >= F::N && S % 8 == 4, "row stride");
    static constexpr size_t z = size_t(F::ZS) * PP * sizeof(float2);
    static constexpr size_t tile = size_t(2) * 2 * PP * S * sizeof(float);            // two real fields
    static constexpr size_t ltile = size_t(F::N / 2 + 1) * PP * sizeof(float4);       // lines
    static constexpr size_t to_lines = F::N * sizeof(float2) + (z > tile ? z : tile);
    static constexpr size_t zl = ((z > ltile ? z : ltile) + 15) / 16 * 16;
    static constexpr int kMaxEnt = 32 * PP;                                           // staged source entries
    static constexpr size_t source = size_t(2 * PP * F::N + 3 * kMaxEnt) * sizeof(float);
    static constexpr size_t to_real = F::N * sizeof(float2) + zl;                     // + source with a source
};

// 16-byte copy global -> shared through L2 (the source may have been written by the preceding kernel)
__device__ __forceinline__ void cp16(void* dst, const void* src) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(s_addr(dst)), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_wait_all() { asm volatile("cp.async.wait_all;" ::: "memory"); }

// A tile of 2 PP columns (axis 0: [N][2 PP]) or rows (axis 1: [2 PP][S]) of a real field into shared
// memory, from column or row p0 on.  Rows of a multiple of 4 floats are copied by 16 bytes.  A thread's
// pieces lie at constant distances, so that a piece is one instruction.
template <int N, int PP, int S, int NT, int AX>
__device__ __forceinline__ void stage_tile(float* dst, const float* f, int p0) {
    constexpr int V = (N % 4 == 0 && (2 * PP) % 4 == 0) ? 4 : 2;
    auto piece = [](float* d, const float* src) {
        if constexpr (V == 4)
            cp16(d, src);
        else
            *reinterpret_cast<float2*>(d) = __ldcg(reinterpret_cast<const float2*>(src));
    };
    if constexpr (AX == 1) {
        const int rows = min(2 * PP, N - p0);
        for (int x = V * threadIdx.x; x < N; x += V * NT)
            static_for<0, 2 * PP>([&](auto R) {
                constexpr int r = decltype(R)::value;
                if (r < rows) piece(dst + r * S + x, f + size_t(p0) * N + x + size_t(r) * N);
            });
    } else {
        constexpr int per = 2 * PP / V, step = NT / per, steps = (N + step - 1) / step;
        static_assert(NT % per == 0, "whole rows per step");
        const int x = (threadIdx.x % per) * V, y0 = threadIdx.x / per;
        if (p0 + x < N)
            static_for<0, steps>([&](auto I) {
                constexpr int i = decltype(I)::value;
                if ((i + 1) * step <= N || y0 + i * step < N)
                    piece(dst + (y0 + i * step) * (2 * PP) + x, f + size_t(y0) * N + p0 + x + size_t(i) * step * N);
            });
    }
}

// the pair's members at a position: axis 0 two neighbours of a row, axis 1 two neighbours of a column
// (p at position 0); _l2: written by the preceding kernel
template <int AX, int N>
__device__ __forceinline__ float2 sp_load(const float* p, int pos) {
    return AX ? make_float2(p[pos], p[pos + N]) : *reinterpret_cast<const float2*>(p + size_t(pos) * N);
}
template <int AX, int N>
__device__ __forceinline__ float2 sp_load_l2(const float* p, int pos) {
    return AX ? make_float2(__ldcg(p + pos), __ldcg(p + pos + N))
              : __ldcg(reinterpret_cast<const float2*>(p + size_t(pos) * N));
}

template <int N1, int N2, int PP, bool ADJ>
__global__ void __launch_bounds__(PP * Fft2<N1, N2>::T) ks_to_lines(Geo g, ToLinesArgs a) {
    using F = Fft2<N1, N2>;
    constexpr int N = F::N, H = N / 2 + 1, NT = PP * F::T;
    extern __shared__ float2 sm[];
    float2* twA = sm;
    float2* Z = sm + N;
    constexpr int S = PairSmem<F, PP>::S;
    float* T0 = reinterpret_cast<float*>(Z);   // staged tiles of the two fields, before Z is written
    float* T1 = T0 + 2 * PP * S;
    constexpr int tiles = (N / 2 + PP - 1) / PP;
    const int axis = blockIdx.x >= tiles, tile = blockIdx.x - axis * tiles;
    const int k = blockIdx.y;
    const int c = threadIdx.x % PP, idx = threadIdx.x / PP;
    const int q0 = tile * PP;
    const bool ok = q0 + c < N / 2;
    const int q = ok ? q0 + c : N / 2 - 1;
    const bool aact = idx < N2, bact = idx < N1;
    const size_t kf = size_t(k) * N * N;
    const float* med = medium_of(g, a.cg, k);
    const int mode = ADJ ? int(SP_ADJOINT) : a.mode;
    // element (position, member) of the pair: axis 0 position y, members x = 2q, 2q+1; axis 1
    // position x, members y = 2q, 2q+1.  Each axis has its own copy of the loads (constant strides).
    auto for_axis = [&](auto f) {
        if (axis)
            f(std::integral_constant<int, 1>{});
        else
            f(std::integral_constant<int, 0>{});
    };
    const size_t o0 = axis ? size_t(2 * q) * N + idx : size_t(idx) * N + 2 * q;
    float2 cc[N1], hv[ADJ ? N1 : 1];
    const int hslot = a.hist ? in_range_or_zero(a.slot, g.s_eff, g.status) : 0;
    float* hb = a.hist ? a.hist + (size_t(k) * g.s_eff + hslot) * N * N : nullptr;
    const int yd = 2 * q - g.P;   // domain row of the pair's first member (axis 1)
    const bool in0 = yd >= 0 && yd < g.n, in1 = yd + 1 >= 0 && yd + 1 < g.n;
    float* cbr = ADJ ? a.cbar + (size_t(k) * g.n + (in0 || in1 ? yd : 0)) * g.n : nullptr;
    if (aact && (mode == SP_PRESSURE || mode == SP_ADJOINT))
        for_axis([&](auto A) {
            constexpr int AX = decltype(A)::value;
            static_for<0, N1>([&](auto I) {
                constexpr int n1 = decltype(I)::value;
                cc[n1] = sp_load<AX, N>(med + o0, N2 * n1);
                if constexpr (ADJ && AX == 1) {
                    const int xd = idx + N2 * n1 - g.P;
                    const bool xin = xd >= 0 && xd < g.n;
                    hv[n1] = make_float2(xin && in0 ? hb[o0 + N2 * n1] : 0.f, xin && in1 ? hb[o0 + N2 * n1 + N] : 0.f);
                }
            });
        });
    for (int i = threadIdx.x; i < N; i += NT) twA[i] = g.twA[i];
    // sensor entries of the tile's rows (axis 1)
    const int y0 = 2 * q0;
    const bool gather = !ADJ && axis == 1 && a.y != nullptr && (mode == SP_PRESSURE || mode == SP_INIT);
    int e0 = 0, e1 = 0;
    int2 se = make_int2(0, 0);     // the thread's first entry and its medium, fetched before the wait
    float4 sw = make_float4(0.f, 0.f, 0.f, 0.f);
    float c0 = 0.f, c1 = 0.f;
    auto entry = [&](int e) {
        se = g.sent[e];
        sw = g.sentw[e];
        const bool in = in_range(int(sw.w) - y0, 2 * PP, g.status) && in_range(se.y + 1, N, g.status) &&
                        in_range(se.x, g.m, g.status) && in_range(a.tstep, g.nt, g.status);
        if (!in) sw = make_float4(0.f, 0.f, 0.f, -1.f);
        if (in && mode == SP_PRESSURE) {
            const float* m = med + size_t(int(sw.w)) * N + se.y;
            c0 = m[0];
            c1 = m[1];
        }
    };
    if (gather) {
        e0 = g.srow[y0] + int(threadIdx.x);
        e1 = g.srow[min(y0 + 2 * PP, N)];
        if (e0 < e1) entry(e0);
    }
    pdl_wait_then_release();
    if (mode == SP_PRESSURE || mode == SP_ADJOINT) {
        for_axis([&](auto A) {
            constexpr int AX = decltype(A)::value;
            stage_tile<N, PP, S, NT, AX>(T0, a.f0[0] + kf, y0);
            stage_tile<N, PP, S, NT, AX>(T1, a.f0[1] + kf, y0);
        });
        cp_wait_all();
    }
    __syncthreads();   // twiddles, staged tiles
    float2 v[N1];
    if (aact) {
        if (mode == SP_PRESSURE || mode == SP_ADJOINT) {
            for_axis([&](auto A) {
                constexpr int AX = decltype(A)::value;
                static_for<0, N1>([&](auto I) {
                    constexpr int n1 = decltype(I)::value;
                    const int pos = idx + N2 * n1;
                    float2 t;
                    if constexpr (AX == 0) {
                        t = cadd(*reinterpret_cast<const float2*>(T0 + pos * (2 * PP) + 2 * c),
                                 *reinterpret_cast<const float2*>(T1 + pos * (2 * PP) + 2 * c));
                    } else {
                        t = make_float2(T0[2 * c * S + pos] + T1[2 * c * S + pos],
                                        T0[(2 * c + 1) * S + pos] + T1[(2 * c + 1) * S + pos]);
                    }
                    v[n1] = cprod(cprod(cc[n1], cc[n1]), t);
                    if constexpr (ADJ && AX == 1) {   // sum_n p^n pb (one addition per cell and step); 2 / c at the end
                        const int xd = pos - g.P;
                        if (ok && xd >= 0 && xd < g.n) {
                            if (in0) atomicAdd(cbr + xd, hv[n1].x * t.x);
                            if (in1) atomicAdd(cbr + g.n + xd, hv[n1].y * t.y);
                        }
                    }
                });
            });
        } else if (mode == SP_INIT) {
            static_for<0, N1>([&](auto I) {
                constexpr int n1 = decltype(I)::value;
                const int pos = idx + N2 * n1;
                const int xd = (axis ? pos : 2 * q) - g.P, yy = (axis ? 2 * q : pos) - g.P;
                const int dx = axis ? 0 : 1, dy = axis ? 1 : 0;
                auto at = [&](int yv, int xv) {
                    return (xv >= 0 && xv < g.n && yv >= 0 && yv < g.n) ? a.p0[(size_t(k) * g.n + yv) * g.n + xv] : 0.f;
                };
                v[n1] = make_float2(at(yy, xd), at(yy + dy, xd + dx));
            });
        } else {
            const float* f = (blockIdx.z ? a.f1[axis] : a.f0[axis]) + kf + o0;
            const float2 sc = blockIdx.z ? a.scale1 : a.scale0;
            for_axis([&](auto A) {
                constexpr int AX = decltype(A)::value;
                static_for<0, N1>([&](auto I) {
                    constexpr int n1 = decltype(I)::value;
                    v[n1] = scale2(sp_load_l2<AX, N>(f, N2 * n1), sc);
                });
            });
        }
        if (!ADJ && axis == 1 && hb && ok && mode != SP_COPY) {
            float* h = hb + o0;
            static_for<0, N1>([&](auto I) {
                constexpr int n1 = decltype(I)::value;
                h[N2 * n1] = v[n1].x;
                h[N2 * n1 + N] = v[n1].y;
            });
        }
    }
    if (gather) {
        for (int e = e0; e < e1; e += NT) {
            if (e != e0) entry(e);
            const int row = int(sw.w);
            if (row < 0) continue;
            float p0v, p1v;
            if (mode == SP_INIT) {
                const int xd = se.y - g.P, yy = row - g.P;
                auto at = [&](int xv) {
                    return (xv >= 0 && xv < g.n && yy >= 0 && yy < g.n) ? a.p0[(size_t(k) * g.n + yy) * g.n + xv] : 0.f;
                };
                p0v = at(xd);
                p1v = at(xd + 1);
            } else {
                const int o = (row - y0) * S + se.y;
                p0v = c0 * c0 * (T0[o] + T1[o]);
                p1v = c1 * c1 * (T0[o + 1] + T1[o + 1]);
            }
            // at most two adds (rows iy, iy+1) onto a zeroed sample: order-independent
            atomicAdd(&a.y[(size_t(k) * g.nt + a.tstep) * g.m + se.x], sw.z * (sw.x * p0v + sw.y * p1v));
        }
    }
    __syncthreads();   // the staged tiles are read: Z takes their place
    if (aact) F::template fwd_a_t<PP>(v, idx, Z + c, twA);
    __syncthreads();
    {
        float2 b[N2];
        if (bact) F::template fwd_b_load<PP>(b, idx, Z + c);
        __syncthreads();
        if (bact) {
            F::fwd_b(b);
            static_for<0, N2>([&](auto I) {
                Z[(idx + N1 * decltype(I)::value) * PP + c] = b[decltype(I)::value];
            });
        }
    }
    __syncthreads();
    float2* out = (blockIdx.z ? a.out1 : a.out0) + (size_t(axis) * g.K + k) * H * N;
    for (int i = threadIdx.x; i < H * PP; i += NT) {
        const int cq = i % PP, m = i / PP;
        if (q0 + cq >= N / 2) continue;
        const float2 zk = Z[m * PP + cq];
        const float2 zm = Z[(m == 0 ? 0 : N - m) * PP + cq];
        const float4 w = make_float4(0.5f * (zk.x + zm.x), 0.5f * (zk.y - zm.y), 0.5f * (zk.y + zm.y),
                                     -0.5f * (zk.x - zm.x));
        *reinterpret_cast<float4*>(out + size_t(m) * N + 2 * (q0 + cq)) = w;
    }
}

// ---------------------------------------------------------------------------
// lines -> real: the inverse of the above; the adjoint's source S^T r^n is added to axis 1
template <int N1, int N2, int PP>
__global__ void __launch_bounds__(PP * Fft2<N1, N2>::T) ks_to_real(Geo g, ToRealArgs a) {
    using F = Fft2<N1, N2>;
    constexpr int N = F::N, H = N / 2 + 1, NT = PP * F::T;
    constexpr int kMaxEnt = PairSmem<F, PP>::kMaxEnt;
    extern __shared__ float2 sm[];
    float2* twB = sm;
    float2* Z = sm + N;
    float4* W = reinterpret_cast<float4*>(Z);   // staged lines [H][PP], before Z is written
    float* S = reinterpret_cast<float*>(reinterpret_cast<char*>(Z) + PairSmem<F, PP>::zl);   // source rows [2 PP][N]
    int* s_col = reinterpret_cast<int*>(S + 2 * PP * N);
    float* s_wa = reinterpret_cast<float*>(s_col + kMaxEnt);
    float* s_wb = s_wa + kMaxEnt;
    constexpr int tiles = (N / 2 + PP - 1) / PP;
    const int axis = blockIdx.x >= tiles, tile = blockIdx.x - axis * tiles;
    const int k = blockIdx.y;
    const int c = threadIdx.x % PP, idx = threadIdx.x / PP;
    const int q0 = tile * PP;
    const bool ok = q0 + c < N / 2;
    const int q = ok ? q0 + c : N / 2 - 1;
    const bool bact = idx < N1, aact = idx < N2;
    for (int i = threadIdx.x; i < N; i += NT) twB[i] = g.twB[i];
    // The source of the tile's rows, accumulated before the wait (the residual is complete before
    // the reverse sweep starts): entries staged in parallel, then added in order, one thread per row.
    const int y0 = 2 * q0, y1 = min(y0 + 2 * PP, N);
    bool src = false;
    if (a.resid && axis == 1 && blockIdx.z == 0) {
        const int e0 = g.srow[y0], e1 = g.srow[y1];
        src = e1 > e0;
        if (src) {
            const float* rv = a.resid + (size_t(k) * g.nt + in_range_or_zero(a.tstep, g.nt, g.status)) * g.m;
            const bool staged = e1 - e0 <= kMaxEnt;
            for (int i = threadIdx.x; i < 2 * PP * N; i += NT) S[i] = 0.f;
            if (staged)
                for (int e = e0 + int(threadIdx.x); e < e1; e += NT) {
                    const int2 se = g.sent[e];
                    const float4 sw = g.sentw[e];
                    const bool in = in_range(se.x, g.m, g.status) && in_range(se.y + 1, N, g.status);
                    const float v = in ? rv[se.x] * sw.z : 0.f;
                    s_col[e - e0] = in ? se.y : 0;
                    s_wa[e - e0] = sw.x * v;
                    s_wb[e - e0] = sw.y * v;
                }
            __syncthreads();
            if (int(threadIdx.x) < y1 - y0) {
                float* Sr = S + threadIdx.x * N;
                const int ea = g.srow[y0 + threadIdx.x], eb = g.srow[y0 + threadIdx.x + 1];
                for (int e = ea; e < eb; ++e) {
                    if (staged) {
                        const int col = s_col[e - e0];
                        Sr[col] += s_wa[e - e0];
                        Sr[col + 1] += s_wb[e - e0];
                    } else {
                        const int2 se = g.sent[e];
                        const float4 sw = g.sentw[e];
                        if (!(in_range(se.x, g.m, g.status) && in_range(se.y + 1, N, g.status))) continue;
                        const float v = rv[se.x] * sw.z;
                        Sr[se.y] += sw.x * v;
                        Sr[se.y + 1] += sw.y * v;
                    }
                }
            }
        }
    }
    pdl_wait_then_release();
    if (!a.zero) {
        const float2* in = (blockIdx.z ? a.in1 : a.in0) + (size_t(axis) * g.K + k) * H * N + 2 * q0;
        constexpr int step = NT / PP, steps = (H + step - 1) / step;
        if (ok)
            static_for<0, steps>([&](auto I) {
                constexpr int i = decltype(I)::value;
                if ((i + 1) * step <= H || idx + i * step < H)
                    cp16(W + threadIdx.x + i * NT, in + size_t(idx) * N + 2 * c + size_t(i) * step * N);
            });
        cp_wait_all();
    }
    __syncthreads();   // twiddles, source rows, staged lines
    float2 b[N2];
    if (bact && !a.zero) {
        static_for<0, N2>([&](auto I) {
            constexpr int k2 = decltype(I)::value;
            const int kk = idx + N1 * k2;
            const bool low = 2 * kk <= N;
            float4 w = W[(low ? kk : N - kk) * PP + (ok ? c : 0)];
            if (kk == 0 || 2 * kk == N) {
                w.y = 0.f;
                w.w = 0.f;
            }
            b[k2] = low ? make_float2(w.x - w.w, w.y + w.z) : make_float2(w.x + w.w, w.z - w.y);
        });
    }
    __syncthreads();   // the staged lines are read: Z takes their place
    if (bact && !a.zero) F::template inv_b_t<PP>(b, idx, Z + c, twB);
    __syncthreads();
    if (!aact || !ok) return;
    float2 v[N1];
    if (!a.zero) {
        F::template inv_a_load<PP>(v, idx, Z + c);
        F::inv_a(v);
    } else {
        static_for<0, N1>([&](auto I) { v[decltype(I)::value] = make_float2(0.f, 0.f); });
    }
    const float2 scale = blockIdx.z ? a.scale1 : a.scale0;
    if (scale.x != 1.f)
        static_for<0, N1>([&](auto I) { v[decltype(I)::value] = scale2(v[decltype(I)::value], scale); });
    if (axis == 0) {
        float* d = (blockIdx.z ? a.d1[0] : a.d0[0]) + size_t(k) * N * N + 2 * q;
        static_for<0, N1>([&](auto I) {
            constexpr int n1 = decltype(I)::value;
            *reinterpret_cast<float2*>(d + size_t(idx + N2 * n1) * N) = v[n1];
        });
    } else {
        float* d = (blockIdx.z ? a.d1[1] : a.d0[1]) + size_t(k) * N * N + size_t(2 * q) * N;
        static_for<0, N1>([&](auto I) {
            constexpr int n1 = decltype(I)::value;
            const int x = idx + N2 * n1;
            float2 w = v[n1];
            if (src) {
                w.x += S[(2 * c) * N + x];
                w.y += S[(2 * c + 1) * N + x];
            }
            d[x] = w.x;
            d[N + x] = w.y;
        });
    }
}

// ---------------------------------------------------------------------------
// the lines pass: LL lines per CTA, T threads each.  The lines' state (into shared memory, by
// asynchronous copies), the multipliers (into the registers of the threads that use them, for both
// operators), the twiddles (likewise: one set for all four transforms, whose twiddles all sit on the
// A side) and the PML factors are fetched before the dependency wait.
template <class F, int LL>
struct LinesSmem {
    static constexpr int ZR = RowPad<F::N1, F::N2>::zs;
    static_assert(ZR >= F::ZS, "padded stride");
    static constexpr size_t bytes = size_t(2 * LL * F::N + 2 * LL * ZR) * sizeof(float2) + size_t(2) * F::N * sizeof(float);
};

template <int N1, int N2, int LL, bool ADJ>
__global__ void __launch_bounds__(LL * Fft2<N1, N2>::T) ks_lines(Geo g, LinesArgs a) {
    using F = Fft2<N1, N2>;
    constexpr int N = F::N, T = F::T, H = N / 2 + 1, NT = LL * T, ZR = LinesSmem<F, LL>::ZR;
    extern __shared__ float2 sm[];
    float2* SU = sm;                  // staged u and rho lines [LL][N]
    float2* SR = SU + LL * N;
    float2* Z0 = SR + LL * N;
    float2* Z1 = Z0 + LL * ZR;
    float* AC = reinterpret_cast<float*>(Z1 + LL * ZR);   // PML factors at cell centres and at +1/2 cell
    float* AS = AC + N;
    const int lines = 2 * g.K * H;
    const int r = threadIdx.x / T, idx = threadIdx.x - r * T;
    const int l = blockIdx.x * LL + r;
    const bool ok = l < lines;
    const bool aact = ok && idx < N2, bact = ok && idx < N1;
    const size_t base = size_t(l) * N + idx;
    float2 m[N2], w[N1];
    if (a.mode != SP_DIV) {   // the CTA's lines are contiguous
        const size_t o0 = size_t(blockIdx.x) * LL * N + 2 * threadIdx.x;
        const int pieces = min(LL, lines - int(blockIdx.x) * LL) * (N / 2);
        static_for<0, (LL * N / 2 + NT - 1) / NT>([&](auto I) {
            constexpr int i = decltype(I)::value * NT;
            if (int(threadIdx.x) + i < pieces) {
                cp16(SR + 2 * threadIdx.x + 2 * i, a.r + o0 + 2 * i);
                if (a.mode != SP_STEP_FIRST) cp16(SU + 2 * threadIdx.x + 2 * i, a.u + o0 + 2 * i);
            }
        });
    }
    if (bact) {   // M at the bins idx + N1 k2 of the line's row of the table
        const float2* md = g.md + size_t(l % H) * N + idx;
        static_for<0, N2>([&](auto I) { m[decltype(I)::value] = md[N1 * decltype(I)::value]; });
    }
    if (aact)
        static_for<1, N1>([&](auto I) { w[decltype(I)::value] = g.twA[decltype(I)::value * N2 + idx]; });
    for (int i = threadIdx.x; i < N; i += NT) {
        AC[i] = g.a_cell[i];
        AS[i] = g.a_stag[i];
    }
    pdl_wait_then_release();
    float2 v[N1];
    if (aact)
        static_for<0, N1>([&](auto I) { v[decltype(I)::value] = __ldcg(a.in + base + N2 * decltype(I)::value); });
    const float2* su = SU + r * N + idx;
    const float2* sr = SR + r * N + idx;
    cp_wait_all();
    __syncthreads();   // tables, staged state
    // IFFT(M FFT(v)); D: M -> -conj M
    auto apply = [&](auto div) {
        if (aact) F::fwd_a_w(v, idx, Z0 + r * ZR, w);
        __syncthreads();
        if (bact) {
            float2 b[N2];
            F::fwd_b_load(b, idx, Z0 + r * ZR);
            F::fwd_b(b);
            static_for<0, N2>([&](auto I) {
                constexpr int k2 = decltype(I)::value;
                const float2 mm = decltype(div)::value ? make_float2(-m[k2].x, m[k2].y) : m[k2];
                b[k2] = cmul(b[k2], mm);
            });
            F::inv_b_w(b, idx, Z1 + r * ZR);
        }
        __syncthreads();
        if (aact) {
            F::inv_a_load_w(v, idx, Z1 + r * ZR, w);
            F::inv_a(v);
        }
    };
    const std::false_type grad{};
    const std::true_type div{};
    if constexpr (!ADJ) {
        apply(grad);
        if (aact)
            static_for<0, N1>([&](auto I) {
                constexpr int n1 = decltype(I)::value;
                const float as = AS[idx + N2 * n1];
                const float2 uo = a.mode == SP_STEP_FIRST ? cscale(v[n1], 0.5f) : su[N2 * n1];
                v[n1] = cscale(csub(cscale(uo, as), v[n1]), as);
                a.u[base + N2 * n1] = v[n1];
            });
        apply(div);
        if (aact)
            static_for<0, N1>([&](auto I) {
                constexpr int n1 = decltype(I)::value;
                const float ac = AC[idx + N2 * n1];
                a.r[base + N2 * n1] = cscale(csub(cscale(sr[N2 * n1], ac), v[n1]), ac);
            });
    } else {
        if (a.mode == SP_STEP_ADJOINT) {
            if (aact)
                static_for<0, N1>([&](auto I) {
                    constexpr int n1 = decltype(I)::value;
                    const float ac = AC[idx + N2 * n1];
                    v[n1] = cscale(cadd(sr[N2 * n1], v[n1]), ac);
                    a.r[base + N2 * n1] = cscale(v[n1], ac);
                });
            apply(grad);
            if (aact)
                static_for<0, N1>([&](auto I) {
                    constexpr int n1 = decltype(I)::value;
                    const float as = AS[idx + N2 * n1];
                    v[n1] = cscale(cadd(su[N2 * n1], v[n1]), as);
                    a.u[base + N2 * n1] = cscale(v[n1], as);
                });
        }
        apply(div);
        if (aact)
            static_for<0, N1>([&](auto I) {
                constexpr int n1 = decltype(I)::value;
                a.out[base + N2 * n1] = a.mode == SP_DIV ? cscale(v[n1], a.scale) : v[n1];
            });
    }
}

// ---------------------------------------------------------------------------
// Shared memory a CTA asks for: at least a fixed slot of the SM while a launch has few CTAs per SM.
// The CTAs of a pass are placed while those of the pass before still run (programmatic dependent launch), wherever
// they fit; with small requests some SMs took several times their share and the pass ended with them.  With slots
// of one size for all three passes an SM holds at most `slots` CTAs of any mix, which is every SM's share.
// Ng 300, K = 8 (608 CTAs on 152 SMs): 17.7 us per forward step against 21.9 without slots, gradient step 50.0
// against 54.1; K = 4 12.7 against 17.4; Ng 180, K = 16 (five slots) 14.0 against 15.5.  Beyond five CTAs per SM a
// launch has waves enough to even out, and the slots would cost occupancy (Ng 180, K = 64: 41.8 free, 54.3 in four).
inline size_t slot_bytes(int ctas, int sms) {
    const int share = (ctas + sms - 1) / sms;
    if (share > 5) return 0;
    return share > 4 ? 38 * 1024 : 46 * 1024;   // five, four slots of an SM's 228 KB (1 KB per CTA reserved)
}

// PP pairs per CTA in the pair passes, LL lines per CTA in the lines pass
template <int N1, int N2, int PP, int LL>
struct SplitImpl {
    using F = Fft2<N1, N2>;
    static_assert(F::N % 2 == 0, "pairs of rows");
    static constexpr int N = F::N, H = N / 2 + 1;
    static constexpr size_t smem_tl = PairSmem<F, PP>::to_lines, smem_tr = PairSmem<F, PP>::to_real,
                            smem_src = PairSmem<F, PP>::source;
    static constexpr size_t smem_ln = LinesSmem<F, LL>::bytes;

    // request of a pass that needs `need` bytes: the slot, or a larger one where the lines need it
    static size_t request(const Geo& g, size_t need) {
        const int ctas = std::max(2 * ((N / 2 + PP - 1) / PP) * g.K, (2 * g.K * H + LL - 1) / LL);
        const size_t slot = slot_bytes(ctas, g.sms);
        return slot ? std::max({need, slot, smem_ln}) : need;
    }

    // A forward/inverse pair in float multiplies the mode exp(2 pi i k n / N) by 1 + gain[k], because the rounded
    // transform constants are not exactly unitary: measured with those constants in FP64 arithmetic, by the
    // same code on the host (once per process and side, a few ms).
    static std::vector<double> measure_gain() {
        std::vector<float2> tw(N), ta(N), tb(N);
        std::vector<double2> e(N), x(N), X(N), Z(F::ZS);
        for (int q = 0; q < N; ++q) {
            const double w = -2.0 * 3.14159265358979323846 * q / N;
            e[q] = double2{std::cos(w), -std::sin(w)};
            tw[q] = make_float2(float(std::cos(w)), float(std::sin(w)));
        }
        F::fill_tables(ta.data(), tb.data(), tw.data(), 0, 1);
        std::vector<double> gain(N);
        for (int k = 0; k < N; ++k) {
            for (int n2 = 0; n2 < N2; ++n2) {
                double2 a[N1];
                for (int n1 = 0; n1 < N1; ++n1) a[n1] = e[size_t(k) * (N2 * n1 + n2) % N];
                F::fwd_a_t(a, n2, Z.data(), ta.data());
            }
            for (int k1 = 0; k1 < N1; ++k1) {
                double2 b[N2];
                F::fwd_b_load(b, k1, Z.data());
                F::fwd_b(b);
                for (int k2 = 0; k2 < N2; ++k2) X[k1 + N1 * k2] = b[k2];
            }
            for (int k1 = 0; k1 < N1; ++k1) {
                double2 b[N2];
                for (int k2 = 0; k2 < N2; ++k2) b[k2] = X[k1 + N1 * k2];
                F::inv_b_t(b, k1, Z.data(), tb.data());
            }
            double s = 0.0;
            for (int n2 = 0; n2 < N2; ++n2) {
                double2 a[N1];
                F::inv_a_load(a, n2, Z.data());
                F::inv_a(a);
                for (int n1 = 0; n1 < N1; ++n1) {
                    const double2 o = e[size_t(k) * (N2 * n1 + n2) % N];
                    s += o.x * a[n1].x + o.y * a[n1].y;
                }
            }
            gain[k] = s / (double(N) * N) - 1.0;
        }
        return gain;
    }
    static const double* mode_gain() {
        static const std::vector<double> gain = measure_gain();
        return gain.data();
    }
    static int configure() {
        struct { const void* f; size_t b; } ks[] = {
            {(const void*)ks_to_lines<N1, N2, PP, false>, smem_tl}, {(const void*)ks_to_lines<N1, N2, PP, true>, smem_tl},
            {(const void*)ks_to_real<N1, N2, PP>, smem_tr + smem_src},
            {(const void*)ks_lines<N1, N2, LL, false>, smem_ln}, {(const void*)ks_lines<N1, N2, LL, true>, smem_ln}};
        for (const auto& k : ks) {
            const cudaError_t e = cudaFuncSetAttribute(k.f, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                                       int(std::max({k.b, size_t(46 * 1024), smem_ln})));
            if (e != cudaSuccess) return cuda_fail(e, "cudaFuncSetAttribute(split-axis passes)");
        }
        return PAT_OK;
    }
    static dim3 pair_grid(const Geo& g, int fields) { return dim3(2 * ((N / 2 + PP - 1) / PP), g.K, fields); }
    static void to_lines(const Geo& g, cudaStream_t st, const ToLinesArgs& a, int fields, bool pdl) {
        if (a.mode == SP_ADJOINT)
            launch_pdl(ks_to_lines<N1, N2, PP, true>, pair_grid(g, 1), dim3(PP * F::T), request(g, smem_tl), st, pdl, g, a);
        else
            launch_pdl(ks_to_lines<N1, N2, PP, false>, pair_grid(g, fields), dim3(PP * F::T), request(g, smem_tl), st, pdl, g, a);
    }
    static void lines(const Geo& g, cudaStream_t st, const LinesArgs& a) {
        const dim3 grid((2 * g.K * H + LL - 1) / LL);
        if (a.mode == SP_STEP_ADJOINT || a.mode == SP_DIV)
            launch_pdl(ks_lines<N1, N2, LL, true>, grid, dim3(LL * F::T), request(g, smem_ln), st, true, g, a);
        else
            launch_pdl(ks_lines<N1, N2, LL, false>, grid, dim3(LL * F::T), request(g, smem_ln), st, true, g, a);
    }
    static void to_real(const Geo& g, cudaStream_t st, const ToRealArgs& a, int fields) {
        launch_pdl(ks_to_real<N1, N2, PP>, pair_grid(g, fields), dim3(PP * F::T),
                   request(g, smem_tr + (a.resid ? smem_src : 0)), st, true, g, a);
    }
    static SplitOps ops() { return SplitOps{N, N1, N2, &mode_gain, &configure, &to_lines, &lines, &to_real}; }
};

}  // namespace pat
