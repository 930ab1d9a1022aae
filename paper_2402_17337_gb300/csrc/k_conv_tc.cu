// 3x3 convolutions of the warm-start U-Net on the fifth-generation tensor
// cores: tcgen05.mma with the accumulator in tensor memory, operands staged
// in shared memory by the tensor memory accelerator.
//
// The convolution is an implicit GEMM.  One CTA computes a tile of M = 128
// output pixels (R image rows of TW pixels, R TW = 128) times NT output
// channels; K runs over the input channels in chunks of KC (64, 32 or 16) and
// over the 9 taps, one MMA per tap and 16 channels.
//
//   A (pixels x channels): the input halo tile is loaded by TMA from a 3-D
//     tensor map over the activation view (channels, x, y), one box of KC
//     channels, so shared memory holds [row][pixel][KC], 2 KC bytes a pixel
//     with the swizzle of that width (K-major).  A tap's operand is a window of
//     that tile: with one image row per tile (R = 1) the box spans TW + 2
//     pixels and a tap's shift (dy, dx) moves the descriptor's start by dy
//     rows and dx pixels (the swizzle acts on the address, so a window may
//     start at any pixel); with R > 1 rows a pixel shift would wrap between
//     rows, so three boxes are loaded, each already shifted by its dx, and a
//     tap moves the start by dy rows only.  Out-of-image pixels are
//     zero-filled by the TMA unit, which is the convolution's zero padding.
//   B (output channels x channels): weights pre-packed (k_pack_conv_weights)
//     as shared-memory images without swizzling (core matrices of 8 rows x 16
//     bytes), copied by bulk copies.
//
// Consecutive convolutions are programmatic dependent launches (the next
// kernel's set-up overlaps the previous one's tail).  The CTAs are
// persistent and loop over tiles.  One thread issues the TMA
// loads and another the MMAs (a pipeline of 2-3 stages on mbarriers: full =
// data landed, empty = the MMAs reading a stage are done, signalled by
// tcgen05.commit); four epilogue warps read the accumulator from tensor
// memory (warp w owns lanes 32 w .. 32 w + 31, i.e. pixels) and apply bias
// and ReLU, while the next tile accumulates into a second accumulator.
// Every wait is bounded: a wait that gives up sets a flag in mapped host
// memory and the CTA skips the rest of its work.
//
// The weight gradient (k_conv3x3_wgrad_tc, below) is a GEMM over pixels
// whose operands come MN-major from boxes of the same form.
#include <cuda.h>
#include <cudaTypedefs.h>
#include <cuda_bf16.h>
#include <stdint.h>

#include <mutex>

#include "ibm_internal.h"
#include "nn_internal.h"

namespace ibm {
namespace nn {

namespace {

constexpr int TC_M = 128;
constexpr int TC_THREADS = 192;  // warps 0-3: epilogue; warp 4: TMA loads; warp 5: MMAs
constexpr int TC_STAGES_MAX = 4;
constexpr int TC_SMEM_MAX = 200 * 1024;  // dynamic shared memory a launch may ask for
constexpr int SM_SMEM = 228 * 1024;      // shared memory of one SM
constexpr long long TC_WAIT_CYCLES = 4000000000ll;  // about 2 s at the SM clock

__device__ __forceinline__ uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_expect_tx(uint32_t bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint32_t bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ bool mbar_test(uint32_t bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}\n"
      : "=r"(ok)
      : "r"(bar), "r"(parity)
      : "memory");
  return ok != 0;
}
// waits for the phase with the given parity to complete; false if it has
// not completed within TC_WAIT_CYCLES
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity) {
  const long long t0 = clock64();
  while (!mbar_test(bar, parity))
    if (clock64() - t0 > TC_WAIT_CYCLES) return false;
  return true;
}
__device__ __forceinline__ void tma_load_3d(uint32_t dst, const CUtensorMap* map, int c0, int c1, int c2,
                                            uint32_t bar) {
  asm volatile(
      "cp.async.bulk.tensor.3d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4}], "
      "[%5];" ::"r"(dst),
      "l"(reinterpret_cast<uint64_t>(map)), "r"(c0), "r"(c1), "r"(c2), "r"(bar)
      : "memory");
}
// adds an FP32 box of shared memory to global memory
__device__ __forceinline__ void tma_add_3d(const CUtensorMap* map, uint32_t src, int c0, int c1, int c2) {
  asm volatile("cp.reduce.async.bulk.tensor.3d.global.shared::cta.add.tile.bulk_group [%0, {%2, %3, %4}], [%1];" ::"l"(
                   reinterpret_cast<uint64_t>(map)),
               "r"(src), "r"(c0), "r"(c1), "r"(c2)
               : "memory");
}
__device__ __forceinline__ void bulk_load(uint32_t dst, const void* src, uint32_t bytes, uint32_t bar) {
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(dst),
               "l"(src), "r"(bytes), "r"(bar)
               : "memory");
}
__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }

// Shared-memory matrix descriptors as two words (descriptor version 1).  Low
// word: start address / 16, leading byte offset (core matrices of a K = 16
// slice without swizzling; unused with it); high word: stride byte offset
// (between 8-row groups), version, swizzle.
__device__ __forceinline__ uint32_t desc_lo(uint32_t addr, uint32_t lbo) { return (addr >> 4) | (lbo >> 4) << 16; }
__device__ __forceinline__ uint32_t desc_hi(uint32_t sbo) { return (sbo >> 4) | 1u << 14; }
// A K-major operand whose rows are row_bytes = 32, 64 or 128 wide with the
// swizzle of that width, 8-row groups contiguous.  The swizzle acts on the
// address, so a window may start at any row of the pattern and a K = 16 slice
// 32 bytes further along the row.
__device__ __forceinline__ uint32_t desc_hi_swizzled(uint32_t row_bytes) {
  return desc_hi(8 * row_bytes) | (row_bytes == 128 ? 2u : (row_bytes == 64 ? 4u : 6u)) << 29;
}
// instruction descriptor of kind::f16: FP32 accumulator, BF16 A and B, both
// K-major, N = n, M = 128
__device__ __forceinline__ uint32_t instr_desc(int n) {
  return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(n >> 3) << 17) | ((uint32_t)(TC_M >> 4) << 24);
}
// One thread of the warp, chosen so that the compiler knows the branch holds
// one thread and keeps the operands of the instructions below in uniform
// registers.  A 128 x N x 16 MMA reads 4 KB + 32 N bytes of shared memory and
// takes that over 128 bytes/clock: 40 clocks at N = 16, 48 at 64, 65 at 128
// issued this way (58 and more from a thread picked by its lane number).
__device__ __forceinline__ bool elect_one() {
  uint32_t p;
  asm volatile("{\n .reg .pred p;\n elect.sync _|p, 0xffffffff;\n selp.u32 %0, 1, 0, p;\n}\n" : "=r"(p));
  return p != 0;
}
// Descriptors come as low and high words; the loops below add to the low one.
__device__ __forceinline__ void tc_mma(uint32_t d, uint32_t a_lo, uint32_t a_hi, uint32_t b_lo, uint32_t b_hi,
                                       uint32_t idesc, uint32_t acc) {
  asm volatile(
      "{\n .reg .pred p;\n .reg .b64 a, b;\n setp.ne.b32 p, %6, 0;\n"
      " mov.b64 a, {%1, %2};\n mov.b64 b, {%3, %4};\n"
      " tcgen05.mma.cta_group::1.kind::f16 [%0], a, b, %5, p;\n}\n" ::"r"(d),
      "r"(a_lo), "r"(a_hi), "r"(b_lo), "r"(b_hi), "r"(idesc), "r"(acc)
      : "memory");
}
__device__ __forceinline__ void tc_commit(uint32_t bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ void prefetch_map(const CUtensorMap* map) {
  asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(map)) : "memory");
}
// 16 consecutive FP32 columns of this warp's 32 lanes
__device__ __forceinline__ void tmem_ld16(uint32_t taddr, float (&v)[16]) {
  uint32_t r[16];
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];\n"
      "tcgen05.wait::ld.sync.aligned;\n"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
        "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
      : "r"(taddr)
      : "memory");
#pragma unroll
  for (int j = 0; j < 16; ++j) v[j] = __uint_as_float(r[j]);
}

// Geometry of one launch (host-computed).
struct TcGeom {
  int TW, R;           // pixels per tile row, rows per MMA (TW R = 128)
  int RB;              // MMA rows a tile stacks (R = 1 only): RB accumulators from one halo box
  int KC;              // input channels per chunk: 64, 32 or 16
  int copies, boxw;    // A boxes per chunk (1 or 3), pixels per box row
  int a_region;        // bytes of one A box in shared memory (padded to 1024)
  int a_bytes, a_tx, stage_bytes, stages;  // a_tx: bytes the A boxes of a chunk bring
  int NT, tmem_cols, nchunks;
  int tiles_x, tiles_z, ntiles;  // tiles: TW-pixel columns x R-row bands x NT-channel groups
};

// waits for the phase with the given parity of an mbarrier unless the CTA
// has given up; gives up (sets *abort) after TC_WAIT_CYCLES
__device__ __forceinline__ bool wait_or_abort(uint32_t bar, uint32_t parity, volatile int* abort) {
  const long long t0 = clock64();
  while (!mbar_test(bar, parity)) {
    if (*abort) return false;
    if (clock64() - t0 > TC_WAIT_CYCLES) {
      *abort = 1;
      return false;
    }
  }
  return true;
}

// Persistent: CTA b computes tiles b, b + gridDim.x, ...  Warps 0-3 drain
// the accumulators (TMEM lanes 0-127 = the tile's pixels) and write the
// outputs; lane 0 of warp 4 issues the loads (a ring of G.stages stages over
// the sequence of (tile, chunk) pairs), lane 0 of warp 5 the MMAs.  Two accumulators in
// tensor memory alternate between tiles, so the MMAs of a tile run while
// the previous tile's epilogue reads the other one.
// GRAD (a data gradient): the epilogue applies the ReLU mask of the layer that
// made this convolution's input and sums that layer's bias gradient, a pass
// over the gradient (139 of 1025 us of a training step at 256x512) less.
enum ConvOut { OUT_PLAIN, OUT_RELU, OUT_GRAD };
template <ConvOut OUT>
__global__ void __launch_bounds__(TC_THREADS, 1)
    k_conv3x3_tc(const __grid_constant__ CUtensorMap tmX, const bf16* __restrict__ wpk, const float* __restrict__ bias,
                 bf16* __restrict__ Y, int ldy, int offy, float* __restrict__ yf, ConvAlso also, int H, int W, int Cout,
                 TcGeom G, unsigned int* __restrict__ err) {
  extern __shared__ __align__(1024) unsigned char smem_raw[];
  __shared__ __align__(8) unsigned long long bar_full[TC_STAGES_MAX], bar_empty[TC_STAGES_MAX];
  __shared__ __align__(8) unsigned long long bar_tfull[2], bar_tempty[2];
  __shared__ uint32_t tmem_slot;
  __shared__ int abort_flag;
  volatile int* abort = &abort_flag;
  const uint32_t sbase = (smem_u32(smem_raw) + 1023u) & ~1023u;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int nmine = (int)blockIdx.x < G.ntiles ? (G.ntiles - 1 - (int)blockIdx.x) / (int)gridDim.x + 1 : 0;
  const uint32_t half_cols = (uint32_t)G.tmem_cols / 2;  // column of the second accumulator
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_slot)),
                 "r"(G.tmem_cols)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  if (threadIdx.x == 32) {
    for (int s = 0; s < G.stages; ++s) {
      mbar_init(smem_u32(&bar_full[s]), 1);
      mbar_init(smem_u32(&bar_empty[s]), 1);
    }
    for (int b = 0; b < 2; ++b) {
      mbar_init(smem_u32(&bar_tfull[b]), 1);
      mbar_init(smem_u32(&bar_tempty[b]), 4);  // one arrival per epilogue warp
    }
    abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (threadIdx.x == 128) prefetch_map(&tmX);
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = tmem_slot;
  // Launched as a programmatic dependent of the previous kernel on the
  // stream: the set-up above (tensor memory, barriers) overlaps that
  // kernel's tail, and no thread touches global memory before the previous
  // kernel has completed and its writes are visible (griddepcontrol.wait);
  // then the next launch may be scheduled.
  asm volatile("griddepcontrol.wait;" ::: "memory");
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  // the biases, once per CTA (OUT_GRAD: the CTA's sums of the bias gradient)
  float* sb = reinterpret_cast<float*>(smem_raw + (sbase - smem_u32(smem_raw)) + G.stages * G.stage_bytes);
  if (warp < 4) {
    for (int k = threadIdx.x; k < Cout; k += 128) sb[k] = bias ? bias[k] : 0.f;
    asm volatile("bar.sync 1, 128;" ::: "memory");
  }
  auto coords = [&](int li, int& x0, int& y0, int& z) {
    int t = (int)blockIdx.x + li * (int)gridDim.x;
    z = t % G.tiles_z;
    t /= G.tiles_z;
    x0 = (t % G.tiles_x) * G.TW;
    y0 = (t / G.tiles_x) * G.R * G.RB;
  };

  const int nc = G.nchunks, S = G.stages, nq = nmine * nc;
  if (warp == 4) {
    // TMA producer: the ring of stages over the sequence of (tile, chunk)
    // pairs q = li nc + ch; a stage is reloaded once the MMAs that read it
    // have completed (empty barrier, committed by the MMA thread)
    if (lane == 0) {
      int issued = 0;
      for (int q = 0; q < nq; ++q) {
        const int li = q / nc, ch = q % nc, s = q % S;
        if (q >= S && !wait_or_abort(smem_u32(&bar_empty[s]), (uint32_t)(q / S - 1) & 1u, abort)) break;
        int x0, y0, z;
        coords(li, x0, y0, z);
        const uint32_t st = sbase + s * G.stage_bytes, bar = smem_u32(&bar_full[s]);
        // this tile's output channels of the packed weights: NT of them, fewer in the last tile
        const int n0 = z * G.NT, nt = Cout - n0 < G.NT ? Cout - n0 : G.NT, k16 = G.KC / 16;
        mbar_expect_tx(bar, G.a_tx + k16 * 9 * nt * 32);
        for (int cp = 0; cp < G.copies; ++cp)
          tma_load_3d(st + cp * G.a_region, &tmX, ch * G.KC, x0 + cp - 1, y0 - 1, bar);
        const bf16* w = wpk + (size_t)ch * k16 * 9 * Cout * 16 + (size_t)n0 * 16;
        if (nt == Cout)
          bulk_load(st + G.a_bytes, w, k16 * 9 * nt * 32, bar);
        else
          for (int t = 0; t < 9 * k16; ++t)
            bulk_load(st + G.a_bytes + t * G.NT * 32, w + (size_t)t * Cout * 16, nt * 32, bar);
        issued = q + 1;
      }
      if (*abort && issued > 0)  // the last load issued has landed (bounded) before the CTA may exit
        mbar_wait(smem_u32(&bar_full[(issued - 1) % S]), (uint32_t)((issued - 1) / S) & 1u);
    }
    __syncwarp();
  } else if (warp == 5) {
    // MMA issuer: never waits for its own MMAs, only for data (full) and for
    // the epilogue to have drained an accumulator (tempty).  An MMA costs this
    // thread two additions: building each descriptor took 105 clocks an MMA,
    // more than twice what the tensor cores need.
    if (elect_one()) {
      const uint32_t idesc = instr_desc(G.NT), row = (uint32_t)G.KC * 2;  // row: bytes of a pixel
      const uint32_t a_hi = desc_hi_swizzled(row), b_hi = desc_hi(256), b_step = (uint32_t)G.NT * 2;
      uint32_t a_tap[9];
#pragma unroll
      for (int tap = 0; tap < 9; ++tap)
        a_tap[tap] = (G.copies == 1 ? (uint32_t)((tap / 3) * G.boxw + tap % 3) * row
                                    : (uint32_t)(tap % 3 * G.a_region) + (uint32_t)(tap / 3 * G.TW) * row) >> 4;
      int s = 0, last = -1;
      uint32_t phase = 0;
      bool ok = true;
      for (int li = 0; li < nmine && ok; ++li) {
        const int buf = li & 1;
        const uint32_t d = tmem + (uint32_t)buf * half_cols;
        if (li >= 2) ok = wait_or_abort(smem_u32(&bar_tempty[buf]), (uint32_t)((li >> 1) - 1) & 1u, abort);
        for (int ch = 0; ch < nc; ++ch) {
          ok = ok && wait_or_abort(smem_u32(&bar_full[s]), phase, abort);
          if (!ok) break;
          tc_fence_after();
          const uint32_t st = sbase + s * G.stage_bytes;
          uint32_t ar = desc_lo(st, 0);
          // B: [K = 16 slice][tap][8-row group of output channels][channel group][8 rows][16 bytes]
          const uint32_t b0 = desc_lo(st + G.a_bytes, 128);
          for (int rb = 0; rb < G.RB; ++rb) {
            uint32_t b = b0, ak = ar;
            for (int k = 0; k < G.KC / 16; ++k) {
#pragma unroll
              for (int tap = 0; tap < 9; ++tap) {
                tc_mma(d + (uint32_t)(rb * G.NT), ak + a_tap[tap], a_hi, b, b_hi, idesc, (uint32_t)(ch | k | tap));
                b += b_step;
              }
              ak += 2;
            }
            ar += (uint32_t)G.boxw * row >> 4;
          }
          tc_commit(smem_u32(&bar_empty[s]));
          if (ch == nc - 1) tc_commit(smem_u32(&bar_tfull[buf]));
          last = s;
          if (++s == S) {
            s = 0;
            phase ^= 1u;
          }
        }
      }
      if (*abort) {
        // the MMAs issued have completed (bounded) before the accumulators are freed
        if (last >= 0) mbar_wait(smem_u32(&bar_empty[last]), last < s ? phase : phase ^ 1u);
        atomicOr_system(err, 1u);
      }
    }
    __syncwarp();
  } else {
    const int m = warp * 32 + lane;
    for (int li = 0; li < nmine; ++li) {
      const int buf = li & 1;
      if (!wait_or_abort(smem_u32(&bar_tfull[buf]), (uint32_t)(li >> 1) & 1u, abort)) {
        if (lane == 0) atomicOr_system(err, 1u);
        break;
      }
      tc_fence_after();
      int x0, y0, z;
      coords(li, x0, y0, z);
      const int x = x0 + m % G.TW, n0 = z * G.NT;
      for (int c0 = 0; c0 < G.NT && n0 + c0 < Cout; c0 += 16) {
        const int co = n0 + c0;
        float bv[16];  // OUT_GRAD: the pixel's sums over rb
#pragma unroll
        for (int j = 0; j < 16; ++j) bv[j] = OUT == OUT_GRAD ? 0.f : sb[co + j];
        uint32_t below[8];  // the tile row before, for the pooling
        for (int rb = 0; rb < G.RB; ++rb) {
          const int y = y0 + m / G.TW + rb;
          const bool valid = x < W && y < H;
          const size_t p = (size_t)y * W + x;
          uint4 mk[2] = {};
          if (OUT == OUT_GRAD && valid) {
            const uint4* src = reinterpret_cast<const uint4*>(also.act + p * also.lda + also.offa + co);
            mk[0] = src[0];
            mk[1] = src[1];
          }
          float v[16];
          tmem_ld16(tmem + ((uint32_t)(warp * 32) << 16) + (uint32_t)buf * half_cols + (uint32_t)(rb * G.NT + c0), v);
#pragma unroll
          for (int j = 0; j < 16; ++j) {
            if (OUT != OUT_GRAD) v[j] += bv[j];
            if (OUT == OUT_RELU) v[j] = fmaxf(v[j], 0.f);
          }
          if (yf && valid && co == 0) yf[p] = v[0];
          uint4 o[2];
          uint32_t* ow = reinterpret_cast<uint32_t*>(o);
#pragma unroll
          for (int j = 0; j < 8; ++j) {
            __nv_bfloat162 h = __floats2bfloat162_rn(v[2 * j], v[2 * j + 1]);
            ow[j] = *reinterpret_cast<uint32_t*>(&h);
          }
          if (OUT == OUT_GRAD) {
            // zero where the activation is not positive (mk is zero outside the image), then add to the sums
            const uint32_t* mw = reinterpret_cast<const uint32_t*>(mk);
#pragma unroll
            for (int j = 0; j < 8; ++j) {
              const float2 a = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&mw[j]));
              if (!(a.x > 0.f)) ow[j] &= 0xFFFF0000u;
              if (!(a.y > 0.f)) ow[j] &= 0x0000FFFFu;
              const float2 g = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&ow[j]));
              bv[2 * j] += g.x;
              bv[2 * j + 1] += g.y;
            }
          }
          if (Y && valid) {
            uint4* dst = reinterpret_cast<uint4*>(Y + p * ldy + offy + co);
            dst[0] = o[0];
            dst[1] = o[1];
          }
          if (also.up && valid) {
            // nearest 2x upsampling: the pixel's four copies
            uint4* d0 = reinterpret_cast<uint4*>(also.up + ((size_t)(2 * y) * (2 * W) + 2 * x) * also.ldu + co);
            uint4* d1 = reinterpret_cast<uint4*>(also.up + ((size_t)(2 * y) * (2 * W) + 2 * x + 1) * also.ldu + co);
            const size_t row = (size_t)(2 * W) * also.ldu / 8;  // uint4 per image row
            d0[0] = d1[0] = d0[row] = d1[row] = o[0];
            d0[1] = d1[1] = d0[row + 1] = d1[row + 1] = o[1];
          }
          if (also.pool) {
            if (rb & 1) {
              // 2x2 average of the stored (BF16) values: lane pairs hold x and x + 1; the even lane takes
              // channels 0-7, the odd lane 8-15 (W and H are even, so a pair is inside or outside as a whole)
              const bool odd = lane & 1;
              uint32_t lo[4], hi[4], oth_lo[4], oth_hi[4];
#pragma unroll
              for (int j = 0; j < 4; ++j) {
                lo[j] = odd ? below[j + 4] : below[j];
                hi[j] = odd ? ow[j + 4] : ow[j];
                oth_lo[j] = __shfl_xor_sync(0xffffffffu, odd ? below[j] : below[j + 4], 1);
                oth_hi[j] = __shfl_xor_sync(0xffffffffu, odd ? ow[j] : ow[j + 4], 1);
              }
              uint4 r;
              uint32_t* rw = reinterpret_cast<uint32_t*>(&r);
#pragma unroll
              for (int j = 0; j < 4; ++j) {
                auto f2 = [](uint32_t w) { return __bfloat1622float2(*reinterpret_cast<__nv_bfloat162*>(&w)); };
                const float2 a = f2(odd ? oth_lo[j] : lo[j]), b = f2(odd ? lo[j] : oth_lo[j]);
                const float2 c = f2(odd ? oth_hi[j] : hi[j]), d = f2(odd ? hi[j] : oth_hi[j]);
                __nv_bfloat162 h = __floats2bfloat162_rn(0.25f * (a.x + b.x + c.x + d.x), 0.25f * (a.y + b.y + c.y + d.y));
                rw[j] = *reinterpret_cast<uint32_t*>(&h);
              }
              if (valid)
                *reinterpret_cast<uint4*>(also.pool + ((size_t)(y / 2) * (W / 2) + x / 2) * also.ldp + co + (odd ? 8 : 0)) = r;
            } else {
#pragma unroll
              for (int j = 0; j < 8; ++j) below[j] = ow[j];
            }
          }
        }
        if (OUT == OUT_GRAD) {
          // sum over the warp's pixels: at each step a lane passes on half of its channels and adds the other
          // lane's share of the half it keeps; lanes 2c and 2c + 1 end with channel c
#pragma unroll
          for (int w = 8; w >= 1; w /= 2) {
            const bool up = lane & (2 * w);
#pragma unroll
            for (int j = 0; j < w; ++j) {
              const float got = __shfl_xor_sync(0xffffffffu, up ? bv[j] : bv[j + w], 2 * w);
              bv[j] = (up ? bv[j + w] : bv[j]) + got;
            }
          }
          bv[0] += __shfl_xor_sync(0xffffffffu, bv[0], 1);
          if (!(lane & 1)) atomicAdd(&sb[co + lane / 2], bv[0]);
        }
      }
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(smem_u32(&bar_tempty[buf]));
    }
    if (OUT == OUT_GRAD) {
      asm volatile("bar.sync 1, 128;" ::: "memory");
      for (int k = threadIdx.x; k < Cout; k += 128)
        if (sb[k] != 0.f) atomicAdd(also.db + k, sb[k]);
    }
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 0) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(G.tmem_cols) : "memory");
  }
}

// ------------------------------------------------------- weight gradient
//
// dW[co][tap][ci] += sum over pixels p of G[p][co] X[p + shift(tap)][ci], a
// GEMM with K = pixels, M = 128 output channels (a tile of them), and N = 3 CB:
// CB input channels (32 or 16) of the three image rows that the tap rows dy
// read.  One MMA per tap column dx and 16 pixels covers three taps, and a CTA
// all nine (three accumulators of 3 CB columns), so G and X are loaded once for
// them.  Both operands come as TMA boxes of [row][pixel][channels], i.e.
// MN-major with the swizzle of a pixel's width: 8-pixel groups (K) are
// contiguous; the leading byte offset takes A to its next channel block and B
// to the next image row.  X boxes start one row and one pixel before the
// chunk's (P pixels of RB rows) and dx moves the start by a pixel.  Rows of A
// beyond Cout read whatever lies there: they only reach accumulator lanes that
// nothing reads.  After its chunks the CTA adds its accumulators to dW with
// TMA reductions.
//
// The MMAs bound the large layers (each reads 4 KB of G and 96 CB bytes of X
// from shared memory at 128 bytes/clock), its fixed latency the small ones.  A
// training step of 32/64/128/128 at 256x512: 839 us with a CTA per tap row,
// N = 32 to 128 for each tap, boxes of 8 channels and vector atomics; 808 us
// with this tile and vector atomics; 763 us as it is.
struct WgGeom {
  int P, RB, XW;            // pixels (a multiple of 16, <= 128) and rows of a chunk; pixels of an X box row
  int CA, CB;               // channels of a block of G and of the tile of X
  int g_block, x_row;       // bytes of a G box and of a row of the X box
  int a_bytes, stage_bytes, stages;
  int nci, co_tiles;        // tiles of input and of output channels
  int tmem_cols, chunks_x, nchunks, ksplit;
};

__global__ void __launch_bounds__(TC_THREADS, 1)
    k_conv3x3_wgrad_tc(const __grid_constant__ CUtensorMap tmG, const __grid_constant__ CUtensorMap tmX,
                       const __grid_constant__ CUtensorMap tmW, int Cout, WgGeom G, unsigned int* __restrict__ err) {
  extern __shared__ __align__(1024) unsigned char smem_raw[];
  __shared__ __align__(8) unsigned long long bar_full[TC_STAGES_MAX], bar_empty[TC_STAGES_MAX], bar_acc;
  __shared__ uint32_t tmem_slot;
  __shared__ int abort_flag;
  volatile int* abort = &abort_flag;
  const uint32_t sbase = (smem_u32(smem_raw) + 1023u) & ~1023u;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  // work unit: blockIdx.x = (ksplit part, input-channel tile, output-channel tile)
  const int part = blockIdx.x % G.ksplit, unit = blockIdx.x / G.ksplit;
  const int ci0 = unit % G.nci * G.CB, co0 = unit / G.nci * 128;
  const int nb = (Cout - co0 < 128 ? Cout - co0 : 128) / G.CA;  // blocks of G in this tile
  const int c_begin = (int)((long)G.nchunks * part / G.ksplit), c_end = (int)((long)G.nchunks * (part + 1) / G.ksplit);
  const int nq = c_end - c_begin, S = G.stages;
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_slot)),
                 "r"(G.tmem_cols)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  if (threadIdx.x == 32) {
    for (int s = 0; s < S; ++s) {
      mbar_init(smem_u32(&bar_full[s]), 1);
      mbar_init(smem_u32(&bar_empty[s]), 1);
    }
    mbar_init(smem_u32(&bar_acc), 1);
    abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (threadIdx.x == 128) {
    prefetch_map(&tmG);
    prefetch_map(&tmX);
    prefetch_map(&tmW);
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = tmem_slot;
  asm volatile("griddepcontrol.wait;" ::: "memory");
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");

  if (warp == 4) {
    if (lane == 0) {
      const int tx_bytes = nb * G.g_block + (G.RB + 2) * G.x_row;
      int issued = 0;
      for (int q = 0; q < nq; ++q) {
        const int s = q % S, c = c_begin + q;
        if (q >= S && !wait_or_abort(smem_u32(&bar_empty[s]), (uint32_t)(q / S - 1) & 1u, abort)) break;
        const int x0 = (c % G.chunks_x) * G.P, y0 = c / G.chunks_x * G.RB;
        const uint32_t st = sbase + s * G.stage_bytes, bar = smem_u32(&bar_full[s]);
        mbar_expect_tx(bar, tx_bytes);
        for (int g = 0; g < nb; ++g) tma_load_3d(st + g * G.g_block, &tmG, co0 + g * G.CA, x0, y0, bar);
        tma_load_3d(st + G.a_bytes, &tmX, ci0, x0 - 1, y0 - 1, bar);
        issued = q + 1;
      }
      if (*abort && issued > 0) mbar_wait(smem_u32(&bar_full[(issued - 1) % S]), (uint32_t)((issued - 1) / S) & 1u);
    }
    __syncwarp();
  } else if (warp == 5) {
    if (elect_one()) {
      // both operands MN-major (transpose bits)
      const uint32_t idesc = instr_desc(3 * G.CB) | (1u << 15) | (1u << 16);
      const uint32_t a_hi = desc_hi_swizzled(2 * G.CA), b_hi = desc_hi_swizzled(2 * G.CB);
      const uint32_t a_step = 2 * G.CA, b_step = 2 * G.CB, dx_step = G.CB / 8, cols = 3 * G.CB;  // / 16 bytes; columns
      int done = 0;
      for (int q = 0; q < nq; ++q) {
        const int s = q % S;
        if (!wait_or_abort(smem_u32(&bar_full[s]), (uint32_t)(q / S) & 1u, abort)) break;
        tc_fence_after();
        const uint32_t st = sbase + s * G.stage_bytes;
        for (int r = 0; r < G.RB; ++r) {
          uint32_t a = desc_lo(st + r * G.P * G.CA * 2, G.g_block);
          uint32_t b = desc_lo(st + G.a_bytes + r * G.x_row, G.x_row);
          for (int ks = 0; ks < G.P / 16; ++ks) {
#pragma unroll
            for (int dx = 0; dx < 3; ++dx)
              tc_mma(tmem + dx * cols, a, a_hi, b + dx * dx_step, b_hi, idesc, (uint32_t)(q | r | ks));
            a += a_step;
            b += b_step;
          }
        }
        tc_commit(smem_u32(&bar_empty[s]));
        done = q + 1;
      }
      tc_commit(smem_u32(&bar_acc));
      if (*abort) {
        if (done > 0) mbar_wait(smem_u32(&bar_empty[(done - 1) % S]), (uint32_t)((done - 1) / S) & 1u);
        atomicOr_system(err, 1u);
      }
    }
    __syncwarp();
  } else if (nq > 0) {
    // epilogue: lane = output channel, 16 input channels of a tap per load; the accumulators go to shared memory
    // (free now) as one [co][CB] box per tap, swizzled against bank conflicts, and one TMA reduction per tap adds
    // it to dW
    const bool ok = wait_or_abort(smem_u32(&bar_acc), 0u, abort);
    if (!ok && lane == 0) atomicOr_system(err, 1u);
    const int row = threadIdx.x, rows = Cout < 128 ? Cout : 128;
    if (ok && warp * 32 < rows) {
      tc_fence_after();
      unsigned char* base = smem_raw + (sbase - smem_u32(smem_raw)) + row * G.CB * 4;
      const int swz = G.CB == 32 ? row & 7 : (row >> 1) & 3;
      for (int t = 0; t < 9; ++t)
        for (int c0 = 0; c0 < G.CB; c0 += 16) {
          float v[16];
          tmem_ld16(tmem + ((uint32_t)(warp * 32) << 16) + (uint32_t)(t * G.CB + c0), v);
          if (row >= rows) continue;
#pragma unroll
          for (int j = 0; j < 4; ++j)
            *reinterpret_cast<float4*>(base + t * rows * G.CB * 4 + (((c0 / 4 + j) ^ swz) * 16)) =
                make_float4(v[4 * j], v[4 * j + 1], v[4 * j + 2], v[4 * j + 3]);
        }
    }
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    asm volatile("bar.sync 1, 128;" ::: "memory");
    if (threadIdx.x == 0 && !*abort) {
      // accumulator columns are [dx][dy][CB]: tap 3 dy + dx
      for (int t = 0; t < 9; ++t) tma_add_3d(&tmW, sbase + t * rows * G.CB * 4, ci0, t % 3 * 3 + t / 3, co0);
      asm volatile("cp.async.bulk.commit_group;" ::: "memory");
      asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory");  // shared memory has been read
    }
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 0) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(G.tmem_cols) : "memory");
  }
}

// Packed weights of a convolution with Cin input and Cout output channels:
// for each 16 input channels the shared-memory image
//   [tap 9][8-row group Cout/8][channel group 2][row 8][8 channels]
// of W'[co][tap][ci]; a tile of output channels is a contiguous piece of each
// tap.  W' is the layer's weights
// w[Cout][9][Cin]; with flip it is the data-gradient operator of a layer
// whose weights are w[Cin][9][Cout]: W'[co][tap][ci] = w[ci][8 - tap][co].
// One launch packs every job (blockIdx.y = job).
__global__ void k_pack_conv_weights(const PackJob* __restrict__ jobs) {
  // a thread packs the 8 channels (16 bytes) of one output channel and tap: a
  // 16-byte load and store, and 32-bit index arithmetic (one element a thread
  // with 64-bit divisions took 28.8 us for the 32/64/128/128 network)
  asm volatile("griddepcontrol.wait;" ::: "memory");
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  const PackJob J = jobs[blockIdx.y];
  const int Cin = J.cin, Cout = J.cout, n = Cin / 16 * 9 * Cout * 2;
  for (int k = blockIdx.x * blockDim.x + threadIdx.x; k < n; k += gridDim.x * blockDim.x) {
    const int row = k & 7, g = (k >> 3) & 1;
    int r = k >> 4;
    const int ngrp = r % (Cout / 8);
    r /= Cout / 8;
    const int tap = r % 9, ch = r / 9;
    const int co = ngrp * 8 + row, ci = ch * 16 + g * 8;
    uint4 v;
    if (!J.flip) {
      v = *reinterpret_cast<const uint4*>(J.w + ((size_t)co * 9 + tap) * Cin + ci);
    } else {
      unsigned short h[8];
      const unsigned short* w = reinterpret_cast<const unsigned short*>(J.w);
#pragma unroll
      for (int e = 0; e < 8; ++e) h[e] = w[((size_t)(ci + e) * 9 + (8 - tap)) * Cout + co];
      v = make_uint4(h[0] | (unsigned)h[1] << 16, h[2] | (unsigned)h[3] << 16, h[4] | (unsigned)h[5] << 16,
                     h[6] | (unsigned)h[7] << 16);
    }
    reinterpret_cast<uint4*>(J.wpk)[k] = v;
  }
}

PFN_cuTensorMapEncodeTiled_v12000 encode_fn() {
  static PFN_cuTensorMapEncodeTiled_v12000 fn = nullptr;
  static std::once_flag once;
  std::call_once(once, [] {
    void* p = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) == cudaSuccess &&
        q == cudaDriverEntryPointSuccess)
      fn = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(p);
  });
  return fn;
}

// a flag the kernels set (system-scope atomic) when a wait gives up; mapped
// host memory, so the host reads it without a device synchronisation
unsigned int* error_flag(unsigned int** dev) {
  static unsigned int* host = nullptr;
  static unsigned int* devp = nullptr;
  static std::once_flag once;
  std::call_once(once, [] {
    void* h = nullptr;
    if (cudaHostAlloc(&h, sizeof(unsigned int), cudaHostAllocMapped | cudaHostAllocPortable) == cudaSuccess) {
      host = static_cast<unsigned int*>(h);
      *host = 0u;
      void* d = nullptr;
      if (cudaHostGetDevicePointer(&d, h, 0) == cudaSuccess) devp = static_cast<unsigned int*>(d);
    }
  });
  *dev = devp;
  return host;
}

// Least dynamic shared memory per CTA such that the CTAs that fit on one SM
// by shared memory (1 KB static and 1 KB reserved each) hold no more than the
// SM's 512 tensor-memory columns: then an allocation never waits for
// another CTA's.
int tmem_min_smem(int cols) {
  const int k = 512 / cols;  // CTAs whose columns fit
  return SM_SMEM / (k + 1) - 2048 + 1;
}

// kernel attributes (shared memory size and carveout) are set once per device
bool first_use_on_device(int which) {
  static std::mutex mu;
  static unsigned long long done[2] = {0ull, 0ull};
  int dev = 0;
  cudaGetDevice(&dev);
  if (dev < 0 || dev >= 64) return true;
  std::lock_guard<std::mutex> lock(mu);
  const unsigned long long bit = 1ull << dev;
  if (done[which] & bit) return false;
  done[which] |= bit;
  return true;
}

int pow2_at_least(int v) {
  int p = 1;
  while (p < v) p <<= 1;
  return p;
}

}  // namespace

// pixels of a tile row: those of a narrow image, else the tile's
static int conv_tile_width(int W) { return W >= TC_M ? TC_M : (pow2_at_least(W) < 8 ? 8 : pow2_at_least(W)); }

bool conv3x3_pools(int H, int W) { return conv_tile_width(W) == TC_M && H % 2 == 0 && W % 2 == 0; }

size_t packed_conv_weights(int Cin, int Cout) { return (size_t)Cout * 9 * Cin; }

PackJob pack_job(int Cin, int Cout, const bf16* w, bf16* wpk, bool flip) {
  return PackJob{Cin, Cout, flip ? 1 : 0, w, wpk};
}

void pack_conv_weights(cudaStream_t s, const PackJob* jobs_dev, int njobs, long max_elems) {
  const long b = (max_elems / 8 + 255) / 256;
  cudaLaunchConfig_t lc{};
  lc.gridDim = dim3((unsigned)(b > 256 ? 256 : (b < 1 ? 1 : b)), (unsigned)njobs);
  lc.blockDim = dim3(256);
  lc.stream = s;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  lc.attrs = at;
  lc.numAttrs = 1;
  cudaLaunchKernelEx(&lc, k_pack_conv_weights, jobs_dev);
}

int conv3x3_wgrad(cudaStream_t s, int H, int W, int Cin, int Cout, const bf16* Gd, int ldg, int offg, const bf16* X,
                   int ldx, int offx, float* dW) {
  // channel counts and slices were checked by the forward convolutions of the same layer
  PFN_cuTensorMapEncodeTiled_v12000 enc = encode_fn();
  unsigned int* err_dev = nullptr;
  error_flag(&err_dev);
  if (!enc || !err_dev || Cin % 16 || Cout % 16) {
    set_last_error("weight gradient: unsupported channel counts or no tensor-map encoder");
    return -1;
  }
  WgGeom G{};
  auto block = [](int C) { return C % 64 == 0 ? 64 : (C % 32 == 0 ? 32 : 16); };
  G.P = W >= 128 ? 128 : (pow2_at_least(W) < 16 ? 16 : pow2_at_least(W));
  G.RB = 256 / G.P;  // 256 pixels a chunk: 763 us a training step of 32/64/128/128 at 256x512, 765 with 128
  G.XW = G.P + 8;
  G.CA = block(Cout);
  G.CB = Cin % 32 == 0 ? 32 : 16;  // 9 CB accumulator columns
  G.nci = Cin / G.CB;
  G.co_tiles = (Cout + 127) / 128;
  G.g_block = G.RB * G.P * G.CA * 2;
  G.x_row = G.XW * G.CB * 2;
  G.a_bytes = ((Cout < 128 ? Cout : 128) / G.CA * G.g_block + 1023) / 1024 * 1024;
  G.stage_bytes = (G.a_bytes + (G.RB + 2) * G.x_row + 1023) / 1024 * 1024;
  // the last stage's A reads 128 / CA blocks, also where fewer are loaded
  const int over = 128 / G.CA * G.g_block - G.stage_bytes, extra = 1024 + (over > 0 ? over : 0);
  G.stages = 4;
  while (G.stages > 2 && G.stages * G.stage_bytes + extra > TC_SMEM_MAX) --G.stages;
  G.tmem_cols = pow2_at_least(9 * G.CB);
  G.chunks_x = (W + G.P - 1) / G.P;
  G.nchunks = (H + G.RB - 1) / G.RB * G.chunks_x;
  int smem = G.stages * G.stage_bytes + extra;
  const int smem_tmem = tmem_min_smem(G.tmem_cols);
  if (smem < smem_tmem) smem = smem_tmem;
  if (smem > TC_SMEM_MAX) {
    set_last_error("weight-gradient tile does not fit in shared memory");
    return -1;
  }
  auto swizzle = [](int C) {
    return C == 64 ? CU_TENSOR_MAP_SWIZZLE_128B : (C == 32 ? CU_TENSOR_MAP_SWIZZLE_64B : CU_TENSOR_MAP_SWIZZLE_32B);
  };
  CUtensorMap mg, mx, mw;
  cuuint32_t estr[3] = {1, 1, 1};
  {
    cuuint64_t dims[3] = {(cuuint64_t)Cout, (cuuint64_t)W, (cuuint64_t)H};
    cuuint64_t strides[2] = {(cuuint64_t)ldg * 2, (cuuint64_t)W * ldg * 2};
    cuuint32_t box[3] = {(cuuint32_t)G.CA, (cuuint32_t)G.P, (cuuint32_t)G.RB};
    if (enc(&mg, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, const_cast<bf16*>(Gd + offg), dims, strides, box, estr,
            CU_TENSOR_MAP_INTERLEAVE_NONE, swizzle(G.CA), CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
            CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS) {
      set_last_error("cuTensorMapEncodeTiled rejected a gradient view");
      return -1;
    }
  }
  {
    cuuint64_t dims[3] = {(cuuint64_t)Cin, (cuuint64_t)W, (cuuint64_t)H};
    cuuint64_t strides[2] = {(cuuint64_t)ldx * 2, (cuuint64_t)W * ldx * 2};
    cuuint32_t box[3] = {(cuuint32_t)G.CB, (cuuint32_t)G.XW, (cuuint32_t)(G.RB + 2)};
    if (enc(&mx, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, const_cast<bf16*>(X + offx), dims, strides, box, estr,
            CU_TENSOR_MAP_INTERLEAVE_NONE, swizzle(G.CB), CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
            CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS) {
      set_last_error("cuTensorMapEncodeTiled rejected an activation view");
      return -1;
    }
  }
  {
    cuuint64_t dims[3] = {(cuuint64_t)Cin, 9, (cuuint64_t)Cout};
    cuuint64_t strides[2] = {(cuuint64_t)Cin * 4, (cuuint64_t)Cin * 36};
    cuuint32_t box[3] = {(cuuint32_t)G.CB, 1, (cuuint32_t)(Cout < 128 ? Cout : 128)};
    if (enc(&mw, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 3, dW, dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
            G.CB == 32 ? CU_TENSOR_MAP_SWIZZLE_128B : CU_TENSOR_MAP_SWIZZLE_64B, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
            CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS) {
      set_last_error("cuTensorMapEncodeTiled rejected a weight gradient");
      return -1;
    }
  }
  if (first_use_on_device(1)) {
    cudaFuncSetAttribute(k_conv3x3_wgrad_tc, cudaFuncAttributeMaxDynamicSharedMemorySize, TC_SMEM_MAX);
    cudaFuncSetAttribute(k_conv3x3_wgrad_tc, cudaFuncAttributePreferredSharedMemoryCarveout,
                         (int)cudaSharedmemCarveoutMaxShared);
  }
  int dev = 0, nsm = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
  int per_sm = SM_SMEM / (smem + 2048);
  if (per_sm > 2048 / TC_THREADS) per_sm = 2048 / TC_THREADS;
  if (per_sm > 512 / G.tmem_cols) per_sm = 512 / G.tmem_cols;
  if (per_sm < 1) per_sm = 1;
  // split the pixel chunks so that the CTAs fill the device once
  const int units = G.nci * G.co_tiles;
  G.ksplit = (int)((long)nsm * per_sm / units);
  if (G.ksplit < 1) G.ksplit = 1;
  if (G.ksplit > G.nchunks) G.ksplit = G.nchunks;
  cudaLaunchConfig_t lc{};
  lc.gridDim = dim3(units * G.ksplit);
  lc.blockDim = dim3(TC_THREADS);
  lc.dynamicSmemBytes = smem;
  lc.stream = s;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  lc.attrs = at;
  lc.numAttrs = 1;
  if (cudaLaunchKernelEx(&lc, k_conv3x3_wgrad_tc, mg, mx, mw, Cout, G, err_dev) != cudaSuccess) {
    set_last_error("weight-gradient launch failed");
    return -1;
  }
  return 0;
}

bool conv_tc_failed() {
  unsigned int* dev = nullptr;
  unsigned int* host = error_flag(&dev);
  return host && *reinterpret_cast<volatile unsigned int*>(host) != 0u;
}

int conv3x3(cudaStream_t s, int H, int W, int Cin, int Cout, const bf16* X, int ldx, int offx, const bf16* wpk,
            const float* bias, bf16* Y, int ldy, int offy, bool relu, float* yf, ConvAlso also, bool* pooled) {
  if (Cin % 16 || Cout % 16 || ldx % 8 || offx % 8 || ldy % 8 || offy % 8) {
    set_last_error("convolution channel counts and slices must be multiples of 16 and 8");
    return -1;
  }
  PFN_cuTensorMapEncodeTiled_v12000 enc = encode_fn();
  unsigned int* err_dev = nullptr;
  error_flag(&err_dev);
  if (!enc || !err_dev) {
    set_last_error("cuTensorMapEncodeTiled or the mapped error flag is unavailable");
    return -1;
  }
  TcGeom G{};
  G.TW = conv_tile_width(W);
  G.R = TC_M / G.TW;
  G.copies = G.R == 1 ? 1 : 3;
  G.boxw = G.R == 1 ? G.TW + 2 : G.TW;
  G.tiles_x = (W + G.TW - 1) / G.TW;
  // Output channels per tile: all of them up to 128, halved (not below 32)
  // while the tiles are fewer than half the SMs.  A halving doubles the CTAs
  // and the loads of A: the forward pass of the 32/64/128/128 network on
  // 256x512 takes 170 us with a quarter of the SMs as the line, 163 with half,
  // 168 with all.
  G.NT = Cout <= 128 ? Cout : 128;
  while (G.NT >= 64 && G.NT % 32 == 0 && (long)G.tiles_x * ((H + G.R - 1) / G.R) * ((Cout + G.NT - 1) / G.NT) < 76)
    G.NT /= 2;
  G.tiles_z = (Cout + G.NT - 1) / G.NT;
  // With one image row per MMA a tile stacks RB rows: one halo box of RB + 2
  // rows serves RB accumulators, where RB tiles would load 3 RB rows, and the
  // weights of a chunk are loaded once.  RB NT <= 64: the forward pass of
  // 16/32/32/48 on 512x1024 takes 196 us with 32, 172 with 64, 176 with 128.
  // A layer keeps a tile for every SM.
  G.RB = 1;
  if (G.R == 1)
    for (int rb = 4; rb > 1 && G.RB == 1; rb /= 2)
      if (rb * G.NT <= 64 && (long)G.tiles_x * G.tiles_z * ((H + rb - 1) / rb) >= 152) G.RB = rb;
  // the pooling in the epilogue takes two rows of a tile
  if (also.pool && G.R == 1 && G.RB == 1 && 2 * G.NT <= 256) G.RB = 2;
  const bool pool = also.pool && conv3x3_pools(H, W);
  if (!pool) also.pool = nullptr;
  if (pooled) *pooled = pool;
  // Channels per chunk: the most of which two stages fit.  A TMA box moves
  // one contiguous run per pixel, so a chunk of 64 channels takes an eighth of
  // the runs that 8-channel boxes take: 163 us for 32/64/128/128 on 256x512,
  // against 180 with chunks of 16.
  const int rows = G.R * G.RB + 2, smem_extra = 1024 + Cout * 4;  // alignment slack, biases
  for (G.KC = 64;; G.KC /= 2) {
    G.a_region = (rows * G.boxw * G.KC * 2 + 1023) / 1024 * 1024;
    G.a_bytes = G.copies * G.a_region;
    G.a_tx = G.copies * rows * G.boxw * G.KC * 2;
    G.stage_bytes = (G.a_bytes + 9 * G.NT * G.KC * 2 + 1023) / 1024 * 1024;
    if (G.KC == 16 || (Cin % G.KC == 0 && 2 * G.stage_bytes + smem_extra <= TC_SMEM_MAX)) break;
  }
  // two sets of RB accumulators, each set at least 32 columns
  G.tmem_cols = pow2_at_least(2 * G.RB * G.NT < 64 ? 64 : 2 * G.RB * G.NT);
  G.nchunks = Cin / G.KC;
  G.stages = 3 * G.stage_bytes + smem_extra <= TC_SMEM_MAX ? 3 : 2;
  G.ntiles = G.tiles_x * ((H + G.R * G.RB - 1) / (G.R * G.RB)) * G.tiles_z;
  // dynamic shared memory: the stages, alignment slack and biases, at least
  // tmem_min_smem
  int smem = G.stages * G.stage_bytes + smem_extra;
  const int smem_tmem = tmem_min_smem(G.tmem_cols);
  if (smem < smem_tmem) smem = smem_tmem;
  if (smem > TC_SMEM_MAX) {
    set_last_error("convolution tile does not fit in shared memory");
    return -1;
  }
  CUtensorMap map;
  cuuint64_t dims[3] = {(cuuint64_t)Cin, (cuuint64_t)W, (cuuint64_t)H};
  cuuint64_t strides[2] = {(cuuint64_t)ldx * 2, (cuuint64_t)W * ldx * 2};
  cuuint32_t box[3] = {(cuuint32_t)G.KC, (cuuint32_t)G.boxw, (cuuint32_t)rows};
  const CUtensorMapSwizzle swz = G.KC == 64   ? CU_TENSOR_MAP_SWIZZLE_128B
                                 : G.KC == 32 ? CU_TENSOR_MAP_SWIZZLE_64B
                                              : CU_TENSOR_MAP_SWIZZLE_32B;
  cuuint32_t estr[3] = {1, 1, 1};
  CUresult cr = enc(&map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, const_cast<bf16*>(X + offx), dims, strides, box, estr,
                    CU_TENSOR_MAP_INTERLEAVE_NONE, swz, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
                    CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  if (cr != CUDA_SUCCESS) {
    set_last_error("cuTensorMapEncodeTiled rejected an activation view");
    return -1;
  }
  if (first_use_on_device(0)) {
    // the largest shared-memory carveout, so that several CTAs fit on an SM
    for (auto k : {k_conv3x3_tc<OUT_PLAIN>, k_conv3x3_tc<OUT_RELU>, k_conv3x3_tc<OUT_GRAD>}) {
      cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, TC_SMEM_MAX);
      cudaFuncSetAttribute(k, cudaFuncAttributePreferredSharedMemoryCarveout, (int)cudaSharedmemCarveoutMaxShared);
    }
  }
  // persistent CTAs: as many as fit on the device at once (shared memory,
  // with 1 KB static and 1 KB reserved per CTA; threads; tensor-memory
  // columns), at most one per tile
  int dev = 0, nsm = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
  auto kern = also.act ? k_conv3x3_tc<OUT_GRAD> : (relu ? k_conv3x3_tc<OUT_RELU> : k_conv3x3_tc<OUT_PLAIN>);
  int per_sm = SM_SMEM / (smem + 2048);
  if (per_sm > 2048 / TC_THREADS) per_sm = 2048 / TC_THREADS;
  if (per_sm > 512 / G.tmem_cols) per_sm = 512 / G.tmem_cols;
  if (per_sm < 1) per_sm = 1;
  const long slots = (long)nsm * per_sm;
  const int grid = (int)(G.ntiles < slots ? G.ntiles : slots);
  cudaLaunchConfig_t lc{};
  lc.gridDim = dim3(grid);
  lc.blockDim = dim3(TC_THREADS);
  lc.dynamicSmemBytes = smem;
  lc.stream = s;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  lc.attrs = at;
  lc.numAttrs = 1;
  if (cudaLaunchKernelEx(&lc, kern, map, wpk, bias, Y, ldy, offy, yf, also, H, W, Cout, G, err_dev) != cudaSuccess) {
    set_last_error("convolution launch failed");
    return -1;
  }
  return 0;
}

}  // namespace nn
}  // namespace ibm
