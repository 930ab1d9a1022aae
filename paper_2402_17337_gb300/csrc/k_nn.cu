// Kernels of the learned warm start: a 4-level convolutional U-Net with BF16
// weights and activations and FP32 accumulation, trained on the GPU.
//
// Layout: activations NHWC (channels contiguous), BF16; a layer may read or
// write a channel slice of a wider buffer (ld = channels per pixel of the
// buffer, off = first channel), which is how the decoder's concatenations
// are formed without copies.  Weights of a 3x3 convolution are [Cout][9][Cin]
// (tap = 3*(dy+1) + (dx+1)), i.e. K-contiguous columns of the GEMM operand B.
//
// The convolutions (forward, data gradient, weight gradient) run on the
// tcgen05 tensor cores (k_conv_tc.cu); this file holds the element-wise
// kernels around them.
#include <cuda_bf16.h>
#include <stdint.h>

#include "ibm_internal.h"

namespace ibm {
namespace nn {

using bf16 = __nv_bfloat16;

namespace {

// Kernels of the forward pass are programmatic dependent launches: each
// waits for the previous kernel on the stream to complete (and its writes to
// be visible) before touching global memory, then lets the next one start.
__device__ __forceinline__ void pdl_enter() {
  asm volatile("griddepcontrol.wait;" ::: "memory");
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}

template <typename... KArgs, typename... Args>
void launch_pdl(void (*k)(KArgs...), int grid, int block, cudaStream_t s, Args... args) {
  cudaLaunchConfig_t lc{};
  lc.gridDim = dim3(grid);
  lc.blockDim = dim3(block);
  lc.stream = s;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  lc.attrs = at;
  lc.numAttrs = 1;
  cudaLaunchKernelEx(&lc, k, static_cast<KArgs>(args)...);
}

// 8 BF16 channels (16 bytes) to FP32
__device__ inline void bf16x8_to_float(const uint4& u, float (&f)[8]) {
  const __nv_bfloat162* h = reinterpret_cast<const __nv_bfloat162*>(&u);
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    float2 t = __bfloat1622float2(h[j]);
    f[2 * j] = t.x;
    f[2 * j + 1] = t.y;
  }
}

// FP32 to 8 BF16 channels (16 bytes), round to nearest
__device__ inline uint4 bf16x8_to(const float (&f)[8]) {
  uint4 o;
  __nv_bfloat162* h = reinterpret_cast<__nv_bfloat162*>(&o);
#pragma unroll
  for (int j = 0; j < 4; ++j) h[j] = __floats2bfloat162_rn(f[2 * j], f[2 * j + 1]);
  return o;
}

// ---------------------------------------------------------- elementwise

// 2x2 average pool (H, W even): out[y][x][c] = mean of the 2x2 block; one
// thread per output pixel and 8 channels (C, the slices' ld and off are
// multiples of 8: 16-byte loads and stores)
__global__ void k_avgpool(int H, int W, int C, const bf16* __restrict__ X, int ldx, int offx, bf16* __restrict__ Y,
                          int ldy, int offy) {
  pdl_enter();
  const int H2 = H / 2, W2 = W / 2, G = C / 8;
  const int n = H2 * W2 * G;
  for (int k = blockIdx.x * blockDim.x + threadIdx.x; k < n; k += gridDim.x * blockDim.x) {
    const int g = k % G, p = k / G, x = p % W2, y = p / W2;
    auto at = [&](int yy, int xx) {
      return *reinterpret_cast<const uint4*>(X + ((size_t)yy * W + xx) * ldx + offx + 8 * g);
    };
    float a[8], b[8], c[8], d[8];
    bf16x8_to_float(at(2 * y, 2 * x), a);
    bf16x8_to_float(at(2 * y, 2 * x + 1), b);
    bf16x8_to_float(at(2 * y + 1, 2 * x), c);
    bf16x8_to_float(at(2 * y + 1, 2 * x + 1), d);
    uint4 o;
    __nv_bfloat162* oh = reinterpret_cast<__nv_bfloat162*>(&o);
#pragma unroll
    for (int j = 0; j < 4; ++j)
      oh[j] = __floats2bfloat162_rn(0.25f * (a[2 * j] + b[2 * j] + c[2 * j] + d[2 * j]),
                                    0.25f * (a[2 * j + 1] + b[2 * j + 1] + c[2 * j + 1] + d[2 * j + 1]));
    *reinterpret_cast<uint4*>(Y + (size_t)p * ldy + offy + 8 * g) = o;
  }
}

// The gradient of a ReLU output Y from the next level's gradient dY, through
// the average pool (FROM_POOL: G[p] += dY[p / 2] / 4) or the upsampling
// (FROM_UP: G[p] = the sum of the 2x2 block of dY), zeroed where Y <= 0, and
// that layer's bias gradient db[c] += sum_p G[p][c], in one pass over G (as
// two passes the six such layers of 32/64/128/128 at 256x512 took 30 and 52 us
// of a training step).  A block of 256 threads takes 256 / (C / 8) pixels at
// a time, each thread 8 channels of one pixel (16 bytes), sums over its
// pixels, then the block sums its threads' partials per channel in shared
// memory and adds them to db.  H, W: the size of G.
enum GradFrom { FROM_POOL, FROM_UP };
template <GradFrom FROM>
__global__ void k_resize_relu_grad(int H, int W, int C, const bf16* __restrict__ dY, int ldy, bf16* __restrict__ G,
                                   int ldg, int offg, const bf16* __restrict__ Y, int lda, int offa,
                                   float* __restrict__ db) {
  __shared__ float part[256][9];  // [thread][8 channels], padded against bank conflicts
  pdl_enter();
  const int Gc = C / 8, rows = blockDim.x / Gc, npix = H * W;
  const int g = threadIdx.x % Gc, r = threadIdx.x / Gc;
  float acc[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
  if (r < rows) {
    for (int p = blockIdx.x * rows + r; p < npix; p += gridDim.x * rows) {
      const int x = p % W, y = p / W;
      auto at = [&](size_t q, float (&f)[8]) {
        bf16x8_to_float(*reinterpret_cast<const uint4*>(dY + q * ldy + 8 * g), f);
      };
      uint4* gp = reinterpret_cast<uint4*>(G + (size_t)p * ldg + offg + 8 * g);
      float v[8], act[8];
      bf16x8_to_float(*reinterpret_cast<const uint4*>(Y + (size_t)p * lda + offa + 8 * g), act);
      if (FROM == FROM_POOL) {
        float d[8];
        bf16x8_to_float(*gp, v);
        at((size_t)(y / 2) * (W / 2) + x / 2, d);
#pragma unroll
        for (int j = 0; j < 8; ++j) v[j] += 0.25f * d[j];
      } else {
        float a[8], b[8], c[8], d[8];
        const size_t q = (size_t)(2 * y) * (2 * W) + 2 * x;
        at(q, a);
        at(q + 1, b);
        at(q + 2 * W, c);
        at(q + 2 * W + 1, d);
#pragma unroll
        for (int j = 0; j < 8; ++j) v[j] = a[j] + b[j] + c[j] + d[j];
      }
#pragma unroll
      for (int j = 0; j < 8; ++j)
        if (!(act[j] > 0.f)) v[j] = 0.f;
      const uint4 o = bf16x8_to(v);
      *gp = o;
      bf16x8_to_float(o, v);
#pragma unroll
      for (int j = 0; j < 8; ++j) acc[j] += v[j];
    }
  }
#pragma unroll
  for (int j = 0; j < 8; ++j) part[threadIdx.x][j] = acc[j];
  __syncthreads();
  // the rows of a channel split over the block's threads
  const int per = blockDim.x / C > 0 ? blockDim.x / C : 1;
  for (int t = threadIdx.x; t < C * per; t += blockDim.x) {
    const int c = t % C, cg = c / 8, j = c % 8;
    float sum = 0.f;
    for (int rr = t / C; rr < rows; rr += per) sum += part[rr * Gc + cg][j];
    atomicAdd(&db[c], sum);
  }
}

// loss = mean over masked pixels of (out[p][0] - target[p])^2 ; dOut = 2 (out - target) / count ; db += sum dOut
__global__ void k_mse(long npix, const float* __restrict__ out, int ldo, const float* __restrict__ target,
                      const float* __restrict__ mask, float inv_count, bf16* __restrict__ dout, int ldd,
                      double* __restrict__ loss, float* __restrict__ db) {
  pdl_enter();
  double s = 0.0;
  float sb = 0.f;
  for (long p = blockIdx.x * (long)blockDim.x + threadIdx.x; p < npix; p += (long)gridDim.x * blockDim.x) {
    float m = mask ? mask[p] : 1.f;
    float d = (out[p * ldo] - target[p]) * m;
    s += (double)d * d;
    // channel 0 of the pixel's ldd (a multiple of 8) channels, the others zero: 16-byte stores
    __nv_bfloat162 h = __floats2bfloat162_rn(2.f * d * inv_count, 0.f);
    sb += __low2float(h);
    uint4* o = reinterpret_cast<uint4*>(dout + p * ldd);
    o[0] = make_uint4(*reinterpret_cast<unsigned*>(&h), 0u, 0u, 0u);
    for (int c = 1; c < ldd / 8; ++c) o[c] = make_uint4(0u, 0u, 0u, 0u);
  }
  for (int o = 16; o > 0; o >>= 1) {
    s += __shfl_xor_sync(0xffffffffu, s, o);
    sb += __shfl_xor_sync(0xffffffffu, sb, o);
  }
  if ((threadIdx.x & 31) == 0) {
    atomicAdd(loss, s * inv_count);
    atomicAdd(db, sb);
  }
}

// Adam on FP32 master weights, BF16 copy for the kernels
__global__ void k_adam(long n, float* __restrict__ w, const float* __restrict__ g, float* __restrict__ m,
                       float* __restrict__ v, bf16* __restrict__ wb, float lr, float b1, float b2, float eps,
                       float c1, float c2) {
  pdl_enter();
  for (long k = blockIdx.x * (long)blockDim.x + threadIdx.x; k < n; k += (long)gridDim.x * blockDim.x) {
    float gk = g[k];
    float mk = b1 * m[k] + (1.f - b1) * gk, vk = b2 * v[k] + (1.f - b2) * gk * gk;
    m[k] = mk;
    v[k] = vk;
    float wk = w[k] - lr * (mk * c1) / (sqrtf(vk * c2) + eps);
    w[k] = wk;
    if (wb) wb[k] = __float2bfloat16_rn(wk);
  }
}

__global__ void k_to_bf16(long n, const float* __restrict__ a, bf16* __restrict__ b) {
  for (long k = blockIdx.x * (long)blockDim.x + threadIdx.x; k < n; k += (long)gridDim.x * blockDim.x)
    b[k] = __float2bfloat16_rn(a[k]);
}

// FP32 [H][W][cin] features -> BF16 [H][W][cpad] (zero padded channels;
// cpad a multiple of 8); one thread per pixel and 8 channels
__global__ void k_pack_input(long npix, int cin, int cpad, const float* __restrict__ f, bf16* __restrict__ x) {
  pdl_enter();
  const int G = cpad / 8;
  const long n = npix * G;
  for (long k = blockIdx.x * (long)blockDim.x + threadIdx.x; k < n; k += (long)gridDim.x * blockDim.x) {
    const long p = k / G;
    const int c0 = (int)(k % G) * 8;
    uint4 o;
    __nv_bfloat162* oh = reinterpret_cast<__nv_bfloat162*>(&o);
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const int c = c0 + 2 * j;
      oh[j] = __floats2bfloat162_rn(c < cin ? f[p * cin + c] : 0.f, c + 1 < cin ? f[p * cin + c + 1] : 0.f);
    }
    *reinterpret_cast<uint4*>(x + p * cpad + c0) = o;
  }
}

inline int grid1(long n) {
  long b = (n + 255) / 256;
  return (int)(b > 4096 ? 4096 : (b < 1 ? 1 : b));
}

}  // namespace

void avgpool(cudaStream_t s, int H, int W, int C, const bf16* X, int ldx, int offx, bf16* Y, int ldy, int offy) {
  launch_pdl(k_avgpool, grid1((long)H * W * C / 32), 256, s, H, W, C, X, ldx, offx, Y, ldy, offy);
}
static int resize_grad_blocks(long npix, int C) {
  const long rows = 256 / (C / 8), blocks = (npix + rows * 4 - 1) / (rows * 4);  // at least 4 pixels per thread
  return (int)(blocks > 1216 ? 1216 : blocks);
}
void avgpool_grad(cudaStream_t s, int H, int W, int C, const bf16* dY, int ldy, bf16* g, int ldg, int offg,
                  const bf16* act, int lda, int offa, float* db) {
  launch_pdl(k_resize_relu_grad<FROM_POOL>, resize_grad_blocks((long)H * W, C), 256, s, H, W, C, dY, ldy, g, ldg, offg,
             act, lda, offa, db);
}
void upsample_grad(cudaStream_t s, int H, int W, int C, const bf16* dY, int ldy, bf16* g, int ldg, const bf16* act,
                   int lda, float* db) {
  launch_pdl(k_resize_relu_grad<FROM_UP>, resize_grad_blocks((long)H * W / 4, C), 256, s, H / 2, W / 2, C, dY, ldy, g,
             ldg, 0, act, lda, 0, db);
}
void mse(cudaStream_t s, long npix, const float* out, int ldo, const float* target, const float* mask, float inv_count,
         bf16* dout, int ldd, double* loss, float* db) {
  launch_pdl(k_mse, grid1(npix), 256, s, npix, out, ldo, target, mask, inv_count, dout, ldd, loss, db);
}
void adam(cudaStream_t s, long n, float* w, const float* g, float* m, float* v, bf16* wb, float lr, float b1, float b2,
          float eps, float c1, float c2) {
  launch_pdl(k_adam, grid1(n), 256, s, n, w, g, m, v, wb, lr, b1, b2, eps, c1, c2);
}
void to_bf16(cudaStream_t s, long n, const float* a, bf16* b) { k_to_bf16<<<grid1(n), 256, 0, s>>>(n, a, b); }
void pack_input(cudaStream_t s, long npix, int cin, int cpad, const float* f, bf16* x) {
  launch_pdl(k_pack_input, grid1(npix * cpad / 8), 256, s, npix, cin, cpad, f, x);
}

}  // namespace nn
}  // namespace ibm
