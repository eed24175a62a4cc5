// Declarations of the surrogate network's kernels (lbpf_nn.cu).
#pragma once

#include <cuda_bf16.h>
#include <cuda_runtime.h>

namespace lbpf_nn {

// y = act(conv3x3(x, w) + bias), periodic padding, on the tensor cores
// (tcgen05); cin a multiple of 16; cout in equal tiles of at most 256
// channels, each a multiple of 16.  w: BF16 [tap][cout][cin].
cudaError_t conv3x3_fwd(const float* x, const __nv_bfloat16* w, const float* bias, float* y, int N, int H, int W,
                        int cin, int cout, int relu, cudaStream_t s);
// The kernel conv3x3_fwd takes for these (valid) sizes: 0 the gather kernel, 1
// the halo kernel with resident weights, 2 with streamed weights.
int conv3x3_form(int H, int W, int cin, int cout);
// Error word of the convolution kernels, a bit mask of the waits that gave up
// (forward: 1, 2 gather kernel, 16 halo loaders, 32 epilogue, 64 MMA issue, 128
// weight stream; weight gradient: 4 loaders, 8 the sums, 256 MMA issue); 0 when
// every wait completed, -1 when it cannot be read.
int conv_error();
// wt[tap][ci][co] = w[8 - tap][co][ci]: weights of the data-gradient convolution.
cudaError_t flip_weights(const __nv_bfloat16* w, __nv_bfloat16* wt, int cin, int cout, cudaStream_t s);
// dw[tap][co][ci] += sum_p dy[p][co] x[p + tap][ci], BF16 operands on the tensor
// cores, FP32 accumulation; cin, cout multiples of 16 (cin > 256: of 32).
cudaError_t conv3x3_wgrad(const float* x, const float* dy, float* dw, int N, int H, int W, int cin, int cout,
                          cudaStream_t s);
// The same two with the input given in two parts: ca channels at half the
// resolution (upsampled 2x, nearest), then cb channels (b NULL: cb = 0, a at
// full resolution).  Two parts need H a multiple of 16 and W of 8.
cudaError_t conv3x3_fwd_src(const float* a, const float* b, int ca, int cb, const __nv_bfloat16* w, const float* bias,
                            float* y, int N, int H, int W, int cout, int relu, cudaStream_t s);
cudaError_t conv3x3_wgrad_src(const float* a, const float* b, int ca, int cb, const float* dy, float* dw, int N, int H,
                              int W, int cout, cudaStream_t s);
// Gradient through a layer's ReLU and its bias gradient (act_bwd_kernel): in
// place; from the 2 x 2 children in src (sc channels a pixel); from the pooled
// gradient src plus the skip gradient (sc channels a pixel, from so on; may be
// NULL).  c a power of two, 16 .. 256.  The bias gradient comes as act_blocks(P, c)
// rows of c partial sums in part.
int act_blocks(long long P, int c);
cudaError_t act_bwd(const float* y, float* dy, float* part, long long P, int c, cudaStream_t s);
cudaError_t act_bwd_up(const float* y, const float* src, float* dst, float* part, int N, int H, int W, int c, int sc,
                       cudaStream_t s);
cudaError_t act_bwd_pool(const float* y, const float* src, const float* skip, float* dst, float* part, int N, int H,
                         int W, int c, int sc, int so, cudaStream_t s);
// Sums of partials, s[k].out[j] += sum over rows r of s[k].part[r * pitch + j], in
// an order that depends on the sizes alone.
struct PartialSums {
    struct Sum {
        const float* part;
        float* out;
        int rows, pitch, width;
    };
    Sum s[20];  // a layer's each, and the head's
    int n;
};
cudaError_t sum_partials(const PartialSums& q, cudaStream_t s);
cudaError_t pool_fwd(const float* x, float* y, int N, int H, int W, int c, cudaStream_t s);
// 1x1 head with the interface gate, c <= 64 channels in, 2 out; y may be NULL.
cudaError_t head_fwd(const float* x, const float* w, const float* b, const float* xin, int cx, float* out, float* y,
                     long long P, int c, cudaStream_t s);
// part: act_blocks(P, c) rows of 3 c + 2 partial sums: dw, db, the last layer's db.
cudaError_t head_bwd(const float* x, const float* dy, const float* w, const float* xin, int cx, float* dx, float* part,
                     long long P, int c, cudaStream_t s);
cudaError_t mse(const float* p, const float* t, const float* x, int cin, int cout, float alpha, float* dp, double* loss,
                long long n, cudaStream_t s);
cudaError_t adam(float* w, const float* g, float* m, float* v, __nv_bfloat16* wb, long long n, float lr, float b1,
                 float b2, float eps, int t, cudaStream_t s);
cudaError_t to_bf16(const float* a, __nv_bfloat16* b, long long n, cudaStream_t s);
cudaError_t pad_channels(const float* x, float* y, long long P, int cin, int cout, cudaStream_t s);
cudaError_t assemble(const float* phi, const float* u, const int* index, const float* tab, int nc, float* x, long long P,
                     cudaStream_t s);
cudaError_t apply(const float* y, float* phi, float* u, long long P, cudaStream_t s);
cudaError_t delta(const float* phi0, const float* u0, const float* phi1, const float* u1, float* y, long long P,
                  cudaStream_t s);
cudaError_t range_count(const float* phi, long long P, float lo, float hi, unsigned int* count, cudaStream_t s);

}  // namespace lbpf_nn
