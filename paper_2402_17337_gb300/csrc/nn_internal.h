// Launchers of the U-Net kernels (k_nn.cu, k_conv_tc.cu).  Activations are BF16 NHWC; a
// view of an activation is (buffer, channels per pixel ld, first channel off).
#pragma once
#include <cuda_bf16.h>
#include <cuda_runtime.h>

namespace ibm {
namespace nn {

using bf16 = __nv_bfloat16;

// What a convolution writes besides its output: its 2x2 average (pool, ldp
// channels a pixel) and its nearest 2x upsampling (up, ldu channels a pixel).
// A data gradient (no bias, no ReLU of its own) may take the activation it is
// the gradient of (act, an output of a ReLU): it is zeroed where act is not
// positive, and its sum over the pixels is added to db.
struct ConvAlso {
  bf16* pool = nullptr;
  int ldp = 0;
  bf16* up = nullptr;
  int ldu = 0;
  const bf16* act = nullptr;
  int lda = 0, offa = 0;
  float* db = nullptr;
};
// Y = act(conv3x3(X, W) + bias), zero padding, on the tcgen05 tensor cores
// (k_conv_tc.cu); Cin, Cout % 16 == 0, ldx, offx, ldy, offy % 8 == 0; wpk:
// the weights packed by pack_conv_weights; Y may be null (only the other
// outputs are wanted); yf: optional FP32 copy of output channel 0, [H][W].
// *pooled: whether also.pool was written (conv3x3_pools; else the caller pools).  Returns 0, or -1 with ibm_last_error set.
int conv3x3(cudaStream_t s, int H, int W, int Cin, int Cout, const bf16* X, int ldx, int offx, const bf16* wpk,
            const float* bias, bf16* Y, int ldy, int offy, bool relu, float* yf, ConvAlso also = ConvAlso{},
            bool* pooled = nullptr);
// whether a convolution of an H x W image can write its 2x2 average: rows of a
// whole tile, more than 64 pixels, and even sizes
bool conv3x3_pools(int H, int W);
// elements of the packed weights of a convolution with Cin inputs and Cout
// outputs, and the packing of w[Cout][9][Cin] (flip: of the data-gradient
// operator of a layer with weights w[Cin][9][Cout], W'[co][tap][ci] =
// w[ci][8 - tap][co])
size_t packed_conv_weights(int Cin, int Cout);
struct PackJob {
  int cin, cout, flip;
  const bf16* w;
  bf16* wpk;
};
PackJob pack_job(int Cin, int Cout, const bf16* w, bf16* wpk, bool flip);
// every job of the device array jobs_dev in one launch; max_elems: the
// largest job's packed_conv_weights
void pack_conv_weights(cudaStream_t s, const PackJob* jobs_dev, int njobs, long max_elems);
// true once a convolution kernel has given up a bounded wait
bool conv_tc_failed();
// dW[co][tap][ci] += sum_p G[p][co] X[p + shift(tap)][ci] on the tcgen05 tensor
// cores (k_conv_tc.cu); Cout <= 128; returns 0, or -1 with ibm_last_error set
int conv3x3_wgrad(cudaStream_t s, int H, int W, int Cin, int Cout, const bf16* G, int ldg, int offg, const bf16* X,
                   int ldx, int offx, float* dW);
void avgpool(cudaStream_t s, int H, int W, int C, const bf16* X, int ldx, int offx, bf16* Y, int ldy, int offy);
// The gradient g of a ReLU output (act; ld and off of its view) from the next
// level's: zeroed where act is not positive, its sum over the pixels added to
// db.  avgpool_grad: g += dY / 4 over each 2x2 block (H, W: the size of g).
// upsample_grad: g = the sum of each 2x2 block of dY (H, W: the size of dY).
void avgpool_grad(cudaStream_t s, int H, int W, int C, const bf16* dY, int ldy, bf16* g, int ldg, int offg,
                  const bf16* act, int lda, int offa, float* db);
void upsample_grad(cudaStream_t s, int H, int W, int C, const bf16* dY, int ldy, bf16* g, int ldg, const bf16* act,
                   int lda, float* db);
// db: the sum of dout's channel 0 is added to it
void mse(cudaStream_t s, long npix, const float* out, int ldo, const float* target, const float* mask, float inv_count,
         bf16* dout, int ldd, double* loss, float* db);
void adam(cudaStream_t s, long n, float* w, const float* g, float* m, float* v, bf16* wb, float lr, float b1, float b2,
          float eps, float c1, float c2);
void to_bf16(cudaStream_t s, long n, const float* a, bf16* b);
void pack_input(cudaStream_t s, long npix, int cin, int cpad, const float* f, bf16* x);

}  // namespace nn
}  // namespace ibm
