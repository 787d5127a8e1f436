// Kernel launchers of the learned warm start (unet_kernels.cu).
#pragma once

#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <cstddef>

namespace pat {

// C[M][N] = A[M][K] . B[N][K]^T (+bias)(ReLU); out_mode 0 bf16, 1 fp32, 2 fp32 atomic add (split K)
int unet_gemm(cudaStream_t st, const __nv_bfloat16* A, int lda, const __nv_bfloat16* B, int ldb, int M, int N,
              int K, const float* bias, int relu, void* C, int ldc, int out_mode, int splitk);
// the same GEMM on tcgen05 / TMEM / TMA (unet_tc05.cu); supported: K >= 64, pitches multiples of 8,
// 16-byte aligned operands.  d_status (may be null) gets PAT_STATUS_TC05 if a bounded wait gave up.
bool unet_gemm_tc05_supported(const __nv_bfloat16* A, int lda, const __nv_bfloat16* B, int ldb, int M, int N, int K);
int unet_gemm_tc05(cudaStream_t st, const __nv_bfloat16* A, int lda, const __nv_bfloat16* B, int ldb, int M, int N,
                   int K, const float* bias, int relu, void* C, int ldc, int out_mode, int splitk, int* d_status);
// 3x3 (taps 9) or 1x1 (taps 1) convolution without im2col (unet_conv.cu), weight rows of kw >= taps * cin or zero-
// extended elements: out[p][cout] (pitch ldo, bf16) = conv(in, W[cout][kw]) (+ bias)
// (ReLU) (zero where mask <= 0, pitch cout); flip: taps reversed (data gradient)
bool unet_conv_supported(const __nv_bfloat16* in, int ldin, int cin, int cout);
int unet_conv(cudaStream_t st, const __nv_bfloat16* in, int ldin, const __nv_bfloat16* W, int B, int H, int Wd, int cin,
              int cout, int taps, int kw, int flip, const float* bias, int relu, const __nv_bfloat16* mask,
              __nv_bfloat16* out, int ldo, int* d_status);
// dW[cout][kw] += sum_p dz[p][cout] in[p + off(tap)][c] at tap * cin + c < kw (taps 9, or 1 unshifted); dW zeroed by the caller;
// reads in and dz without waiting for the kernel before it in the stream, which must be the bias sum of the same dz
bool unet_wgrad_supported(const __nv_bfloat16* in, int ldin, int cin, int cout);
int unet_wgrad(cudaStream_t st, const __nv_bfloat16* in, int ldin, const __nv_bfloat16* dz, int B, int H, int Wd, int cin,
               int taps, int cout, float* dW, int kw, int* d_status);

struct ConvDesc {   // one convolution's weights in the parameter and bf16 arrays
    int cin, cout, k;
    size_t w_off, wb_off;
};

int unet_im2col(cudaStream_t st, const __nv_bfloat16* in, __nv_bfloat16* col, int B, int H, int W, int C, int ldc_in,
                int flip, int kp);
int unet_transpose(cudaStream_t st, const __nv_bfloat16* in, __nv_bfloat16* out, int R, int C, int ld);
int unet_maxpool(cudaStream_t st, const __nv_bfloat16* in, __nv_bfloat16* out, unsigned char* idx, int B, int H, int W,
                 int C);
int unet_enc_bwd(cudaStream_t st, const __nv_bfloat16* dout, const unsigned char* idx, const __nv_bfloat16* cat, int ldcat,
                 int off, const __nv_bfloat16* y, __nv_bfloat16* din, int B, int H, int W, int C);
int unet_concat(cudaStream_t st, const __nv_bfloat16* src, const __nv_bfloat16* skip, __nv_bfloat16* cat, int B, int Hs,
                int Ws, int Cs, int Ck);
int unet_upsample_bwd(cudaStream_t st, const __nv_bfloat16* cat, const __nv_bfloat16* y, __nv_bfloat16* dsrc, int B, int Hs,
                      int Ws, int C, int ldo);
int unet_relu_bwd(cudaStream_t st, __nv_bfloat16* g, const __nv_bfloat16* y, size_t n);
size_t unet_part_floats(int C);   // scratch of the two-step sums below
int unet_part_blocks();
int unet_bias_grad(cudaStream_t st, const __nv_bfloat16* g, float* db, float* part, unsigned* done, size_t P, int C);
int unet_head(cudaStream_t st, const __nv_bfloat16* y, const __nv_bfloat16* w, const float* bias, float* out, size_t P,
              int C);
int unet_head_bwd(cudaStream_t st, const float* out, const float* tgt, const __nv_bfloat16* y, const __nv_bfloat16* w,
                  __nv_bfloat16* dy, float* part, double* lpart, float* dw, float* db, double* loss, size_t P, int C);
int unet_adam(cudaStream_t st, float* w, const float* g, float* m, float* v, size_t n, float lr, float b1, float b2,
              float eps, float bc1, float bc2);
int unet_weights(cudaStream_t st, const float* param, __nv_bfloat16* wb, __nv_bfloat16* wt, const ConvDesc* desc, int n,
                 size_t most);
int unet_pack_input(cudaStream_t st, const float* in, __nv_bfloat16* out, int B, int Cin, int H, int W, int Cp);

}  // namespace pat
