// 3x3 convolutions of the warm-start network as implicit GEMMs on the fifth-generation tensor cores:
// no im2col buffer, no transposes.
//
// Forward and data gradient (k_conv): C[pixel][cout] = sum_{tap, c} in[pixel + off(tap)][c] W[cout][tap][c].
// A CTA computes an image tile of 16 x 8 pixels (the 128 rows of the MMA) by NT channels.  For every
// tap and block of KB channels, one TMA copy fetches the shifted 16 x 8 x KB box of the NHWC input
// (4-D tensor map; the zero fill outside the image is the convolution's padding) and one the weights'
// NT x KB tile.  The K index runs over (tap, channel) in 16-wide steps exactly as in the im2col
// GEMM, so the FP32 accumulation and every BF16 result are the same.  The epilogue adds the bias,
// applies the ReLU (or, in the data gradient, the ReLU mask of the layer below) and stores 16 bytes at a time.
//
// Weight gradient (k_wgrad): dW[cout][(tap, c)] = sum_pixel dz[pixel][cout] in[pixel + off(tap)][c], a
// contraction over the pixels, in which both operands are contiguous along the output dimensions
// ("MN-major"): the NHWC boxes are the MMA operands as they lie.  128 rows of (tap, c) by NT channels per CTA,
// 64 pixels (16 x 4) per stage, the pixels split over CTAs, FP32 atomics into dW.
//
// What bounds them: at 128 x 128 with 32 channels the L2 -> shared traffic of the nine shifted boxes;
// the im2col form wrote and read nine times the activations through HBM.  A small CTA (one tile,
// 20-100 KB of shared memory) leaves room for several per SM, which overlap one another's prologue,
// copies and epilogue.  Measured on GB300 (128 x 128, 4 levels, base 32, 32 images): all convolutions and their
// gradients 1.6 ms, against 20.5 ms of im2col, 3.5 of transposes and 4.5 of GEMMs; a 32 -> 32 convolution at full size
// 50 us (193 TFLOP/s), its weight gradient 28 us.
//
// The kernels of the convolutions, the bias sums, the pooling and the concatenation are launched with programmatic
// stream serialisation: a kernel's barriers and tensor memory are set up while the one before drains.  A CTA
// lets the next kernel start only once it has its tensor memory, so that a later kernel's allocation never keeps an
// earlier one waiting.  The weight gradient depends on nothing that the bias sum before it writes: it runs beside it
// and waits for it only before its own stores.  Forward of 8 images 0.341 -> 0.293 ms, gradients of 32 2.12 -> 1.91 ms.
//
// Every mbarrier wait is bounded as in unet_tc05.cu: a wait that gives up sets PAT_STATUS_TC05 and the CTA
// drains its copies, frees its tensor memory and returns without storing.
#include <algorithm>

#include "kfixed.cuh"
#include "pat_internal.h"
#include "tc05.cuh"
#include "unet.h"

namespace pat {
namespace tc05 {

constexpr int TX = 16, TY = 8;                    // pixel tile of k_conv
constexpr int WY = 4, WPIX = TX * WY;             // pixels of one k_wgrad stage: 16 x 4
constexpr int CONV_THREADS = 128;

struct ConvArgs {
    int H, W, tx, ty;        // image, tiles per row and column
    int cin, cout, nt;       // channels, N tile
    int stages, cols;        // ring depth, tensor-memory columns
    int taps;                // 9, or 1 (a 1x1 convolution)
    int flip;                // taps in reverse order (data gradient)
    const float* bias;       // [cout] or null
    int relu;
    const __nv_bfloat16* mask;   // zero where mask <= 0 (pitch cout), or null
    __nv_bfloat16* out;
    int ldo;
    int* status;
};

// Barriers and flags of a CTA behind its ring buffers.
struct Ring {
    uint64_t* full;
    uint64_t* empty;
    uint64_t* done;
    uint32_t* tslot;
    volatile int* abort_flag;
    int* issued;
    __device__ Ring(unsigned char* p, int stages) {
        full = reinterpret_cast<uint64_t*>(p);
        empty = full + stages;
        done = empty + stages;
        tslot = reinterpret_cast<uint32_t*>(done + 1);
        abort_flag = reinterpret_cast<volatile int*>(tslot + 1);
        issued = const_cast<int*>(abort_flag) + 1;
    }
    __device__ void init(int stages) {
        for (int s = 0; s < stages; ++s) {
            mbar_init(full + s, 1);
            mbar_init(empty + s, 1);
        }
        mbar_init(done, 1);
        *abort_flag = 0;
        *issued = 0;
    }
};

// set up barriers and tensor memory; returns the accumulator's address
__device__ __forceinline__ uint32_t begin(const Ring& r, int stages, uint32_t cols) {
    if (threadIdx.x == 0) const_cast<Ring&>(r).init(stages);
    if (threadIdx.x < 32) tmem_alloc(r.tslot, cols);
    fence_before();
    __syncthreads();
    fence_after();
    return *r.tslot;
}

// wait for the MMAs; true if every wait of the CTA succeeded (one decision for the whole CTA)
__device__ __forceinline__ bool finish(const Ring& r) {
    __syncwarp();
    const bool waited = mbar_wait_bounded(r.done, 0, kWaitNs);
    const bool ok = __syncthreads_and(waited && !*r.abort_flag) != 0;
    fence_after();
    return ok;
}

__device__ __forceinline__ void end(const Ring& r, bool ok, int stages, uint32_t tmem, uint32_t cols, int* status) {
    if (!ok && threadIdx.x == 0) {   // let the copies this CTA issued land before its shared memory goes
        const int n = *r.issued;
        for (int k = max(0, n - stages); k < n; ++k) mbar_wait_bounded(r.full + k % stages, (k / stages) & 1, kWaitNs);
        if (status) atomicOr(status, PAT_STATUS_TC05);
    }
    fence_before();
    __syncthreads();
    if (threadIdx.x < 32) {
        fence_after();
        tmem_free(tmem, cols);
    }
}

// HALO: the input comes in as three boxes of 16 x 10 pixels per channel block (one per horizontal shift), loaded once; a
// vertical shift is 16 rows of the box further on, a whole number of swizzle patterns.  Only the weights
// pass through the ring.  480 input pixels per tile instead of 1152.
constexpr int TH = TY + 2;
template <int KB, bool HALO>
__global__ void __launch_bounds__(CONV_THREADS) k_conv(const __grid_constant__ CUtensorMap ta,
                                                      const __grid_constant__ CUtensorMap tb, ConvArgs a) {
    constexpr uint32_t TILE_A = HALO ? 0 : TX * TY * KB * 2, BOX = TX * TH * KB * 2;
    extern __shared__ unsigned char smraw[];
    unsigned char* sm = reinterpret_cast<unsigned char*>((reinterpret_cast<uintptr_t>(smraw) + 1023) & ~uintptr_t(1023));
    const uint32_t tile_b = uint32_t(a.nt) * KB * 2;
    unsigned char* sA = sm;
    unsigned char* sB = sm + (HALO ? 3 * (a.cin / KB) * BOX : a.stages * TILE_A);
    unsigned char* sR = sB + ((a.stages * tile_b + 15u) & ~15u);
    uint64_t* input = reinterpret_cast<uint64_t*>(sR);   // HALO: the input boxes have landed
    const Ring ring(sR + 16, a.stages);
    const int t = blockIdx.x;
    const int b = t / (a.tx * a.ty), q = t - b * a.tx * a.ty;
    const int y0 = (q / a.tx) * TY, x0 = (q % a.tx) * TX, n0 = blockIdx.y * a.nt;
    const int per_tap = a.cin / KB, nk = a.taps * per_tap;
    if (HALO && threadIdx.x == 0) mbar_init(input, 1);
    const uint32_t tmem = begin(ring, a.stages, a.cols);
    pdl_wait_then_release();
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (warp == 0 && lane == 0) {   // producer
        if (HALO) {
            mbar_arrive_expect(input, 3 * per_tap * BOX);
            for (int j = 0; j < 3 * per_tap; ++j)
                tma_load_4d(sA + j * BOX, &ta, (j / 3) * KB, x0 + j % 3 - 1, y0 - 1, b, input);
        }
        for (int kt = 0; kt < nk; ++kt) {
            const int s = kt % a.stages;
            if (kt >= a.stages && !mbar_wait_bounded(ring.empty + s, ((kt / a.stages) - 1) & 1, kWaitNs)) {
                *ring.abort_flag = 1;
                break;
            }
            if (*ring.abort_flag) break;
            const int tap = kt / per_tap, c0 = (kt - tap * per_tap) * KB;
            mbar_arrive_expect(ring.full + s, TILE_A + tile_b);
            if (!HALO) {
                const int o = a.taps == 1 ? 4 : a.flip ? 8 - tap : tap;
                tma_load_4d(sA + s * TILE_A, &ta, c0, x0 + o % 3 - 1, y0 + o / 3 - 1, b, ring.full + s);
            }
            tma_load_2d(sB + s * tile_b, &tb, tap * a.cin + c0, n0, ring.full + s);
            *ring.issued = kt + 1;
        }
    } else if (warp == 1 && lane == 0) {   // MMA issuer
        const uint32_t id = (1u << 4) | (1u << 7) | (1u << 10) | (uint32_t(a.nt >> 3) << 17) | (uint32_t(128 >> 4) << 24);
        if (HALO && !mbar_wait_bounded(input, 0, kWaitNs)) *ring.abort_flag = 1;
        for (int kt = 0; kt < nk; ++kt) {
            const int s = kt % a.stages;
            if (*ring.abort_flag) break;
            if (!mbar_wait_bounded(ring.full + s, (kt / a.stages) & 1, kWaitNs)) {
                *ring.abort_flag = 1;
                break;
            }
            fence_after();
            uint32_t a0 = s_addr(sA + s * TILE_A);
            if (HALO) {
                const int tap = kt / per_tap, cb = kt - tap * per_tap, o = a.flip ? 8 - tap : tap;
                a0 = s_addr(sA + (3 * cb + o % 3) * BOX + (o / 3) * (TX * KB * 2));
            }
            const uint32_t b0 = s_addr(sB + s * tile_b);
#pragma unroll
            for (int kk = 0; kk < KB / 16; ++kk)
                mma_bf16(tmem, desc_sw<KB * 2>(a0 + 32 * kk, 16, 16 * KB), desc_sw<KB * 2>(b0 + 32 * kk, 16, 16 * KB), id,
                         (kt | kk) ? 1u : 0u);
            mma_commit(ring.empty + s);
        }
        mma_commit(ring.done);
    }
    const bool ok = finish(ring);
    const int m = warp * 32 + lane;
    const int y = y0 + m / TX, x = x0 + m % TX;
    if (ok) {
        const bool inside = y < a.H && x < a.W;
        const size_t p = (size_t(b) * a.H + y) * a.W + x;
        for (int c0 = 0; c0 < a.nt && n0 + c0 < a.cout; c0 += 16) {
            uint32_t v[16];
            __syncwarp();
            tmem_ld16(v, tmem + (uint32_t(warp * 32) << 16) + uint32_t(c0));
#pragma unroll
            for (int h = 0; h < 2; ++h) {   // channels come in multiples of 8
                const int n = n0 + c0 + 8 * h;
                if (!inside || n >= a.cout) continue;
                __nv_bfloat162 w[4];
                uint4 mk = make_uint4(0, 0, 0, 0);
                if (a.mask) mk = *reinterpret_cast<const uint4*>(a.mask + p * a.cout + n);
                const __nv_bfloat162* mv = reinterpret_cast<const __nv_bfloat162*>(&mk);
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    float f0 = __uint_as_float(v[8 * h + 2 * j]), f1 = __uint_as_float(v[8 * h + 2 * j + 1]);
                    if (a.bias) {
                        f0 += a.bias[n + 2 * j];
                        f1 += a.bias[n + 2 * j + 1];
                    }
                    if (a.relu) {
                        f0 = fmaxf(f0, 0.f);
                        f1 = fmaxf(f1, 0.f);
                    }
                    if (a.mask) {
                        const float2 g = __bfloat1622float2(mv[j]);
                        if (!(g.x > 0.f)) f0 = 0.f;
                        if (!(g.y > 0.f)) f1 = 0.f;
                    }
                    w[j] = __floats2bfloat162_rn(f0, f1);
                }
                *reinterpret_cast<uint4*>(a.out + p * a.ldo + n) = *reinterpret_cast<const uint4*>(w);
            }
        }
    }
    // (a given-up wait: the input boxes land before the shared memory goes, too)
    if (HALO && !ok && threadIdx.x == 0) mbar_wait_bounded(input, 0, kWaitNs);
    end(ring, ok, a.stages, tmem, a.cols, a.status);
}

struct WgradArgs {
    int tx, ty, tiles;       // 16 x 4 pixel tiles per row, column, in all
    int cin, rows;           // channels per tap, rows of the product: taps * cin
    int taps;                // 9, or 1 (the input is used unshifted)
    int cout, nt, stages, cols;
    int per;                 // pixel tiles per CTA (blockIdx.y)
    float* dW;               // [cout][kw]
    int kw;                  // row length of dW (rows >= kw are not stored)
    int* status;
};

// CA, CB: channels per box of the input and of dz (one swizzle row each)
template <int CA, int CB>
__global__ void __launch_bounds__(CONV_THREADS) k_wgrad(const __grid_constant__ CUtensorMap ta,
                                                       const __grid_constant__ CUtensorMap tb, WgradArgs a) {
    constexpr uint32_t BOX_A = WPIX * CA * 2, BOX_B = WPIX * CB * 2;
    constexpr int NA = 128 / CA;               // input boxes of a stage
    constexpr uint32_t TILE_A = NA * BOX_A;
    extern __shared__ unsigned char smraw[];
    unsigned char* sm = reinterpret_cast<unsigned char*>((reinterpret_cast<uintptr_t>(smraw) + 1023) & ~uintptr_t(1023));
    const int nb = a.nt / CB;
    const uint32_t tile_b = nb * BOX_B;
    unsigned char* sA = sm;
    unsigned char* sB = sm + a.stages * TILE_A;
    const Ring ring(sB + a.stages * tile_b, a.stages);
    const int r0 = blockIdx.x * 128, n0 = blockIdx.z * a.nt;
    const int na = min(NA, (a.rows - r0 + CA - 1) / CA);
    const int t0 = blockIdx.y * a.per, t1 = min(t0 + a.per, a.tiles), nk = t1 - t0;
    const uint32_t tmem = begin(ring, a.stages, a.cols);
    pdl_release();
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (warp == 0 && lane == 0) {
        for (int kt = 0; kt < nk; ++kt) {
            const int s = kt % a.stages;
            if (kt >= a.stages && !mbar_wait_bounded(ring.empty + s, ((kt / a.stages) - 1) & 1, kWaitNs)) {
                *ring.abort_flag = 1;
                break;
            }
            if (*ring.abort_flag) break;
            const int t = t0 + kt, b = t / (a.tx * a.ty), q = t - b * a.tx * a.ty;
            const int y = (q / a.tx) * WY, x = (q % a.tx) * TX;
            mbar_arrive_expect(ring.full + s, na * BOX_A + tile_b);
            for (int j = 0; j < na; ++j) {
                const int row = r0 + j * CA, tap = row / a.cin, c0 = row - tap * a.cin;
                const int dx = a.taps == 9 ? tap % 3 - 1 : 0, dy = a.taps == 9 ? tap / 3 - 1 : 0;
                tma_load_4d(sA + s * TILE_A + j * BOX_A, &ta, c0, x + dx, y + dy, b, ring.full + s);
            }
            for (int j = 0; j < nb; ++j)
                tma_load_4d(sB + s * tile_b + j * BOX_B, &tb, n0 + j * CB, x, y, b, ring.full + s);
            *ring.issued = kt + 1;
        }
    } else if (warp == 1 && lane == 0) {
        // both operands MN-major (bits 15, 16)
        const uint32_t id = (1u << 4) | (1u << 7) | (1u << 10) | (1u << 15) | (1u << 16) | (uint32_t(a.nt >> 3) << 17) |
                            (uint32_t(128 >> 4) << 24);
        for (int kt = 0; kt < nk; ++kt) {
            const int s = kt % a.stages;
            if (!mbar_wait_bounded(ring.full + s, (kt / a.stages) & 1, kWaitNs)) {
                *ring.abort_flag = 1;
                break;
            }
            fence_after();
            const uint32_t a0 = s_addr(sA + s * TILE_A), b0 = s_addr(sB + s * tile_b);
#pragma unroll
            for (int kk = 0; kk < WPIX / 16; ++kk)   // 16 pixels: 16 rows of each box
                mma_bf16(tmem, desc_sw<CA * 2>(a0 + kk * 32 * CA, BOX_A, 16 * CA),
                         desc_sw<CB * 2>(b0 + kk * 32 * CB, BOX_B, 16 * CB), id, (kt | kk) ? 1u : 0u);
            mma_commit(ring.empty + s);
        }
        mma_commit(ring.done);
    }
    const bool ok = finish(ring);
    pdl_wait();
    const int row = r0 + warp * 32 + lane;
    if (ok && nk > 0)
        for (int c0 = 0; c0 < a.nt && n0 + c0 < a.cout; c0 += 16) {
            uint32_t v[16];
            __syncwarp();
            tmem_ld16(v, tmem + (uint32_t(warp * 32) << 16) + uint32_t(c0));
#pragma unroll
            for (int j = 0; j < 16; ++j)
                if (row < a.kw && n0 + c0 + j < a.cout) atomicAdd(a.dW + size_t(n0 + c0 + j) * a.kw + row, __uint_as_float(v[j]));
        }
    end(ring, ok, a.stages, tmem, a.cols, a.status);
}

// The weight gradient of 32 input channels for all nine taps in one CTA: three boxes of 16 x 6 pixels (one per
// horizontal shift) hold every shifted 16 x 4 tile, a vertical shift being 16 rows of the box further on (a whole
// number of swizzle patterns), and dz is read once.  22 KB per 64 pixels instead of 60 KB in three CTAs, which the
// L2 -> shared traffic bounds.  Accumulators: one of 96 rows (dx, c) by NT columns per vertical shift.
constexpr int HY = WY + 2;
template <int CB>
__global__ void __launch_bounds__(CONV_THREADS) k_wgrad_halo(const __grid_constant__ CUtensorMap ta,
                                                            const __grid_constant__ CUtensorMap tb, WgradArgs a) {
    constexpr uint32_t BOX_A = TX * HY * 64, BOX_B = WPIX * CB * 2, TILE_A = 3 * BOX_A;
    extern __shared__ unsigned char smraw[];
    unsigned char* sm = reinterpret_cast<unsigned char*>((reinterpret_cast<uintptr_t>(smraw) + 1023) & ~uintptr_t(1023));
    const int nb = a.nt / CB;
    const uint32_t tile_b = nb * BOX_B;
    unsigned char* sA = sm;
    unsigned char* sB = sm + a.stages * TILE_A;   // at least 6 KB: the unused rows 96..127 of the last tile end here
    const Ring ring(sB + a.stages * tile_b, a.stages);
    const int c0 = blockIdx.x * 32, n0 = blockIdx.z * a.nt;
    const int t0 = blockIdx.y * a.per, t1 = min(t0 + a.per, a.tiles), nk = t1 - t0;
    const uint32_t tmem = begin(ring, a.stages, a.cols);
    pdl_release();
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (warp == 0 && lane == 0) {
        for (int kt = 0; kt < nk; ++kt) {
            const int s = kt % a.stages;
            if (kt >= a.stages && !mbar_wait_bounded(ring.empty + s, ((kt / a.stages) - 1) & 1, kWaitNs)) {
                *ring.abort_flag = 1;
                break;
            }
            if (*ring.abort_flag) break;
            const int t = t0 + kt, b = t / (a.tx * a.ty), q = t - b * a.tx * a.ty;
            const int y = (q / a.tx) * WY, x = (q % a.tx) * TX;
            mbar_arrive_expect(ring.full + s, TILE_A + tile_b);
            for (int j = 0; j < 3; ++j)
                tma_load_4d(sA + s * TILE_A + j * BOX_A, &ta, c0, x + j - 1, y - 1, b, ring.full + s);
            for (int j = 0; j < nb; ++j)
                tma_load_4d(sB + s * tile_b + j * BOX_B, &tb, n0 + j * CB, x, y, b, ring.full + s);
            *ring.issued = kt + 1;
        }
    } else if (warp == 1 && lane == 0) {
        const uint32_t id = (1u << 4) | (1u << 7) | (1u << 10) | (1u << 15) | (1u << 16) | (uint32_t(a.nt >> 3) << 17) |
                            (uint32_t(128 >> 4) << 24);
        for (int kt = 0; kt < nk; ++kt) {
            const int s = kt % a.stages;
            if (!mbar_wait_bounded(ring.full + s, (kt / a.stages) & 1, kWaitNs)) {
                *ring.abort_flag = 1;
                break;
            }
            fence_after();
            const uint32_t a0 = s_addr(sA + s * TILE_A), b0 = s_addr(sB + s * tile_b);
            for (int dy = 0; dy < 3; ++dy)
#pragma unroll
                for (int kk = 0; kk < WPIX / 16; ++kk)
                    mma_bf16(tmem + dy * a.nt, desc_sw<64>(a0 + (dy + kk) * (TX * 64), BOX_A, 512),
                             desc_sw<CB * 2>(b0 + kk * 32 * CB, BOX_B, 16 * CB), id, (kt | kk) ? 1u : 0u);
            mma_commit(ring.empty + s);
        }
        mma_commit(ring.done);
    }
    const bool ok = finish(ring);
    pdl_wait();
    if (ok && nk > 0)
        for (int cc = 0; cc < 3 * a.nt; cc += 16) {
            const int dy = cc / a.nt, n = n0 + cc - dy * a.nt;
            const int row = (dy * 3 + warp) * a.cin + c0 + lane;   // warp: the horizontal shift
            uint32_t v[16];
            __syncwarp();
            tmem_ld16(v, tmem + (uint32_t(warp * 32) << 16) + uint32_t(cc));
#pragma unroll
            for (int j = 0; j < 16; ++j)
                if (warp < 3 && n + j < a.cout) atomicAdd(a.dW + size_t(n + j) * a.kw + row, __uint_as_float(v[j]));
        }
    end(ring, ok, a.stages, tmem, a.cols, a.status);
}

namespace {

CUtensorMapSwizzle swizzle_of(int ch) {
    return ch == 64 ? CU_TENSOR_MAP_SWIZZLE_128B : ch == 32 ? CU_TENSOR_MAP_SWIZZLE_64B : CU_TENSOR_MAP_SWIZZLE_32B;
}

// NHWC activations [B][H][W] of C channels with pixel pitch ld; boxes of ch channels x 16 x bh pixels
int map_nhwc(CUtensorMap* m, const __nv_bfloat16* base, int B, int H, int W, int C, int ld, int ch, int bh) {
    const cuuint64_t dims[4] = {cuuint64_t(C), cuuint64_t(W), cuuint64_t(H), cuuint64_t(B)};
    const cuuint64_t st[3] = {cuuint64_t(ld) * 2, cuuint64_t(W) * ld * 2, cuuint64_t(H) * W * ld * 2};
    const cuuint32_t box[4] = {cuuint32_t(ch), cuuint32_t(TX), cuuint32_t(bh), 1};
    const cuuint32_t es[4] = {1, 1, 1, 1};
    const CUresult r = encoder()(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4, const_cast<__nv_bfloat16*>(base), dims, st, box,
                                 es, CU_TENSOR_MAP_INTERLEAVE_NONE, swizzle_of(ch), CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
                                 CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    if (r == CUDA_SUCCESS) return PAT_OK;
    set_error("unet_conv: cuTensorMapEncodeTiled failed (%d) for %d x %d x %d x %d, pitch %d", int(r), B, H, W, C, ld);
    return PAT_ECUDA;
}

int map_weights(CUtensorMap* m, const __nv_bfloat16* base, int rows, int K, int kb, int box_rows) {
    const cuuint64_t dims[2] = {cuuint64_t(K), cuuint64_t(rows)};
    const cuuint64_t st[1] = {cuuint64_t(K) * 2};
    const cuuint32_t box[2] = {cuuint32_t(kb), cuuint32_t(box_rows)};
    const cuuint32_t es[2] = {1, 1};
    const CUresult r = encoder()(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<__nv_bfloat16*>(base), dims, st, box,
                                 es, CU_TENSOR_MAP_INTERLEAVE_NONE, swizzle_of(kb), CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                                 CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    if (r == CUDA_SUCCESS) return PAT_OK;
    set_error("unet_conv: cuTensorMapEncodeTiled failed (%d) for %d x %d weights", int(r), rows, K);
    return PAT_ECUDA;
}

int chunk_of(int c) { return c % 64 == 0 ? 64 : c % 32 == 0 ? 32 : c % 16 == 0 ? 16 : 0; }
int columns(int nt) {
    int c = 32;
    while (c < nt) c *= 2;
    return c;
}
bool aligned16(const void* p) { return (reinterpret_cast<uintptr_t>(p) & 15) == 0; }

// raise a kernel's shared-memory limit to the most any launch uses (the limit is per kernel and device)
template <class K>
int allow_smem(K k) {
    PAT_CUDA(cudaFuncSetAttribute((const void*)k, cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024));
    return PAT_OK;
}

constexpr size_t kRingBytes = 1024 + 32 + 256;   // alignment of the ring, barriers

// ring depth: up to four stages within half of an SM's shared memory, at least two
int stages_for(size_t stage, int most) {
    int s = most;
    while (s > 2 && kRingBytes + s * stage > 100 * 1024) --s;
    return s;
}

template <int KB, bool HALO>
int launch_conv(cudaStream_t st, const CUtensorMap& ta, const CUtensorMap& tb, dim3 grid, size_t smem,
                const ConvArgs& a) {
    const int rc = allow_smem(k_conv<KB, HALO>);
    if (rc != PAT_OK) return rc;
    count_launch();
    launch_pdl(k_conv<KB, HALO>, grid, dim3(CONV_THREADS), smem, st, true, ta, tb, a);
    const cudaError_t e = cudaGetLastError();
    return e == cudaSuccess ? PAT_OK : cuda_fail(e, "k_conv");
}

template <int CB>
int launch_wgrad_halo(cudaStream_t st, const CUtensorMap& ta, const CUtensorMap& tb, dim3 grid, size_t smem,
                      const WgradArgs& a) {
    const int rc = allow_smem(k_wgrad_halo<CB>);
    if (rc != PAT_OK) return rc;
    count_launch();
    launch_pdl(k_wgrad_halo<CB>, grid, dim3(CONV_THREADS), smem, st, true, ta, tb, a);
    const cudaError_t e = cudaGetLastError();
    return e == cudaSuccess ? PAT_OK : cuda_fail(e, "k_wgrad_halo");
}

template <int CA, int CB>
int launch_wgrad(cudaStream_t st, const CUtensorMap& ta, const CUtensorMap& tb, dim3 grid, size_t smem,
                 const WgradArgs& a) {
    const int rc = allow_smem(k_wgrad<CA, CB>);
    if (rc != PAT_OK) return rc;
    count_launch();
    launch_pdl(k_wgrad<CA, CB>, grid, dim3(CONV_THREADS), smem, st, true, ta, tb, a);
    const cudaError_t e = cudaGetLastError();
    return e == cudaSuccess ? PAT_OK : cuda_fail(e, "k_wgrad");
}

int sm_count() {
    int dev = 0, sms = 148;
    if (cudaGetDevice(&dev) == cudaSuccess) cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    return sms;
}

}  // namespace
}  // namespace tc05

using namespace tc05;

// channel counts in whole 16-wide MMA steps per tap, 16-byte aligned pixels
bool unet_conv_supported(const __nv_bfloat16* in, int ldin, int cin, int cout) {
    return chunk_of(cin) != 0 && cout % 8 == 0 && ldin % 8 == 0 && aligned16(in) && encoder() != nullptr;
}

int unet_conv(cudaStream_t st, const __nv_bfloat16* in, int ldin, const __nv_bfloat16* W, int B, int H, int Wd, int cin,
              int cout, int taps, int kw, int flip, const float* bias, int relu, const __nv_bfloat16* mask,
              __nv_bfloat16* out, int ldo, int* d_status) {
    const int kb = chunk_of(cin);
    ConvArgs a{};
    a.H = H;
    a.W = Wd;
    a.tx = (Wd + TX - 1) / TX;
    a.ty = (H + TY - 1) / TY;
    a.cin = cin;
    a.cout = cout;
    const long long tiles = (long long)B * a.tx * a.ty;
    // the widest N tile (fewest reads of the input) that still gives every SM a CTA
    a.nt = std::min(256, (cout + 15) / 16 * 16);
    const int sms = sm_count();
    while (a.nt % 32 == 0 && a.nt > 32 && tiles * ((cout + a.nt - 1) / a.nt) < sms) a.nt /= 2;
    a.cols = columns(a.nt);
    // The three input boxes of all channel blocks next to a ring of weight tiles, where four CTAs fit an SM: the input
    // is then waited for once, which other CTAs have to cover.  128 x 128 x 32 images: 32 -> 32 channels 61 -> 50 us,
    // 32 -> 96 95 -> 81; with two CTAs per SM it is slower than the ring (64 -> 64 at 64 x 64 36 -> 42, 96 -> 32 134 -> 224).
    const size_t boxes = size_t(3) * TX * TH * cin * 2, wtile = size_t(a.nt) * kb * 2;
    const bool halo = taps == 9 && kRingBytes + boxes + 4 * wtile <= 56 * 1024;
    const size_t stage = halo ? wtile : size_t(TX * TY) * kb * 2 + wtile;
    a.stages = halo ? 4 : std::min(stages_for(stage, 6), taps * cin / kb);
    a.taps = taps;
    a.flip = flip;
    a.bias = bias;
    a.relu = relu;
    a.mask = mask;
    a.out = out;
    a.ldo = ldo;
    a.status = d_status;
    CUtensorMap ta, tb;
    int rc = map_nhwc(&ta, in, B, H, Wd, cin, ldin, kb, halo ? TH : TY);
    if (rc == PAT_OK) rc = map_weights(&tb, W, cout, kw, kb, a.nt);
    if (rc != PAT_OK) return rc;
    const dim3 grid(static_cast<unsigned>(tiles), (cout + a.nt - 1) / a.nt);
    const size_t smem = kRingBytes + a.stages * stage + (halo ? boxes : 0);
    if (kb == 64) return launch_conv<64, false>(st, ta, tb, grid, smem, a);   // the boxes of 64 channels exceed the limit
    if (kb == 32)
        return halo ? launch_conv<32, true>(st, ta, tb, grid, smem, a) : launch_conv<32, false>(st, ta, tb, grid, smem, a);
    return halo ? launch_conv<16, true>(st, ta, tb, grid, smem, a) : launch_conv<16, false>(st, ta, tb, grid, smem, a);
}

bool unet_wgrad_supported(const __nv_bfloat16* in, int ldin, int cin, int cout) {
    return chunk_of(cin) != 0 && chunk_of(cout) != 0 && ldin % 8 == 0 && aligned16(in) && encoder() != nullptr;
}

int unet_wgrad(cudaStream_t st, const __nv_bfloat16* in, int ldin, const __nv_bfloat16* dz, int B, int H, int Wd, int cin,
               int taps, int cout, float* dW, int kw, int* d_status) {
    const int ca = chunk_of(cin), cb = chunk_of(cout);
    WgradArgs a{};
    a.tx = (Wd + TX - 1) / TX;
    a.ty = (H + WY - 1) / WY;
    a.tiles = B * a.tx * a.ty;
    a.cin = cin;
    a.taps = taps;
    a.rows = taps * cin;
    a.cout = cout;
    a.nt = std::min(256, cout);
    if (a.nt % cb != 0) a.nt = a.nt / cb * cb;
    // 32 input channels per box (cin 32, 96, ...; 64 would need 192 rows per shift) and few enough output channels for
    // three accumulators: all taps in one CTA.  128 x 128 x 32 images, 32 -> 32: 87 us in the other form.
    const bool halo = taps == 9 && ca == 32 && cout <= 128;
    a.cols = columns(a.nt);
    const size_t stage = size_t(128 + a.nt) * WPIX * 2;
    a.stages = stages_for(stage, 4);
    if (halo) {
        a.cols = columns(3 * a.nt);
        const size_t hstage = size_t(3 * TX * HY * 64) + size_t(a.nt) * WPIX * 2;
        a.stages = stages_for(hstage, 4);
        const int want = std::max(1, 2 * sm_count() / (cin / 32));
        a.per = std::max((a.tiles + want - 1) / want, std::min(8, a.tiles));
        a.dW = dW;
        a.kw = kw;
        a.status = d_status;
        CUtensorMap ta, tb;
        int rc = map_nhwc(&ta, in, B, H, Wd, cin, ldin, 32, HY);
        if (rc == PAT_OK) rc = map_nhwc(&tb, dz, B, H, Wd, cout, cout, cb, WY);
        if (rc != PAT_OK) return rc;
        const dim3 grid(cin / 32, (a.tiles + a.per - 1) / a.per, 1);
        const size_t smem = kRingBytes + a.stages * hstage;
        return cb == 64   ? launch_wgrad_halo<64>(st, ta, tb, grid, smem, a)
               : cb == 32 ? launch_wgrad_halo<32>(st, ta, tb, grid, smem, a)
                          : launch_wgrad_halo<16>(st, ta, tb, grid, smem, a);
    }
    const int mt = (a.rows + 127) / 128, nz = (cout + a.nt - 1) / a.nt;
    // about four CTAs per SM, at least eight stages each
    const int want = std::max(1, 4 * sm_count() / std::max(1, mt * nz));
    a.per = std::max((a.tiles + want - 1) / want, std::min(8, a.tiles));
    const int split = (a.tiles + a.per - 1) / a.per;
    a.dW = dW;
    a.kw = kw;
    a.status = d_status;
    CUtensorMap ta, tb;
    int rc = map_nhwc(&ta, in, B, H, Wd, cin, ldin, ca, WY);
    if (rc == PAT_OK) rc = map_nhwc(&tb, dz, B, H, Wd, cout, cout, cb, WY);
    if (rc != PAT_OK) return rc;
    const dim3 grid(mt, split, nz);
    const size_t smem = kRingBytes + a.stages * stage;
#define WG(A, B_) \
    if (ca == A && cb == B_) return launch_wgrad<A, B_>(st, ta, tb, grid, smem, a);
    WG(64, 64) WG(64, 32) WG(64, 16) WG(32, 64) WG(32, 32) WG(32, 16) WG(16, 64) WG(16, 32) WG(16, 16)
#undef WG
    return PAT_EINVAL;
}

}  // namespace pat
