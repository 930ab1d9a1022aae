// Geometric multigrid for the pressure correction equation L_p e = r
// (FP32, inside the FP64 defect correction).
//
// The paper solves the pressure equation by red-black SOR (Sec. 2.2); this
// is a variant that reaches the same FP64 residual tolerance in fewer
// sweeps.  The hierarchy coarsens the stretched grid (Sec. 2.3) by merging
// pairs of cells (level l+1 has the faces x_f[0], x_f[2], ... of level l),
// and every level carries the same five-point operator per unit volume,
// rediscretised from its own faces:
//   (L e)_ij = pE_i (e_E - e) + pW_i (e_W - e) + pN_j (e_N - e) + pS_j (e_S - e).
// Transfers:
//   restriction  r_c(I,J) = sum over children of (dx_i / dX_I)(dy_j / dY_J) res_f(i,j)
//                (the volume-weighted average of the fine residual);
//   prolongation e_f(i,j) += bilinear interpolation of e_c between the
//                centre of the parent cell and the centres of the neighbours
//                on the fine cell's side, in the stretched coordinates (zero
//                slope at the domain boundary).
// Interpolation of order 2 and restriction of order 1 add up to more than
// the order of the operator, as cell-centred multigrid needs for V-cycles
// whose convergence does not degrade with the number of levels; piecewise
// constant interpolation (1 + 1) lost convergence on deep hierarchies.
// Smoothing is red-black Gauss-Seidel by the FP32 tile kernel of k_mixed.cu;
// the coarsest level (a few dozen cells) is solved by red-black SOR inside
// one CTA.  All arrays use the colour-split layout rb_at of the FP32 sweeps.
#include <algorithm>
#include <cstdint>

#include "ibm_internal.h"

namespace ibm {

namespace {

// Every kernel of a cycle is a programmatic dependent launch: it waits for the
// one before it and then lets the next one be scheduled (direct launches; with
// the small levels and the merged FCG passes below they take a cycle on
// 2048x1024 from 184.5 us of device time, as a graph per iteration of the
// kernels before, to 141.3).
__device__ __forceinline__ void pdl_enter() {
  asm volatile("griddepcontrol.wait;" ::: "memory");
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}
template <typename... KArgs, typename... Args>
void launch_pdl(void (*k)(KArgs...), dim3 grid, dim3 block, cudaStream_t s, Args... args) {
  cudaLaunchConfig_t lc{};
  lc.gridDim = grid;
  lc.blockDim = block;
  lc.stream = s;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  lc.attrs = at;
  lc.numAttrs = 1;
  cudaLaunchKernelEx(&lc, k, static_cast<KArgs>(args)...);
}

// One thread per coarse cell: residual of its (up to four) children,
// restricted.  Packed column I of the fine level holds the children's columns
// 2I and 2I + 1, one of each colour in each row, so the cells and their W and
// E neighbours are entries I - 1, I and I + 1 of the two colour rows: of the
// fine correction a warp reads whole lines (per-cell index arithmetic and its
// loads took 14.0 us for 2048x1024).
__global__ void k_mg_restrict(const MgLevel F, const float* __restrict__ ef, MgLevel C) {
  pdl_enter();
  const int I = blockIdx.x * blockDim.x + threadIdx.x, J = blockIdx.y * blockDim.y + threadIdx.y;
  if (I >= C.g.nx || J >= C.g.ny) return;
  const int nx = F.g.nx, ny = F.g.ny, pk = F.g.pk, i0 = 2 * I;
  const bool two = i0 + 1 < nx;
  // row j: cells 2I (colour j & 1) and 2I + 1 (the other colour)
  auto at2 = [&](const float* p, int j) {
    const size_t a = ((size_t)(j & 1) * ny + j) * pk + I, b = ((size_t)((j & 1) ^ 1) * ny + j) * pk + I;
    return make_float2(p[a], two ? p[b] : 0.f);
  };
  float acc = 0.f;
  const float2 zero = make_float2(0.f, 0.f);
  const int j0 = 2 * J;
  float2 s = j0 > 0 ? at2(ef, j0 - 1) : zero, x = at2(ef, j0), n;
#pragma unroll
  for (int b = 0; b < 2; ++b) {
    const int j = j0 + b;
    if (j >= ny) break;
    n = j + 1 < ny ? at2(ef, j + 1) : zero;
    // W of 2I: cell 2I - 1, the other colour at packed column I - 1; E of 2I + 1: cell 2I + 2, at I + 1
    const float w = I > 0 ? ef[((size_t)((j & 1) ^ 1) * ny + j) * pk + I - 1] : 0.f;
    const float e = i0 + 2 < nx ? ef[((size_t)(j & 1) * ny + j) * pk + I + 1] : 0.f;
    const float2 r = at2(F.r, j);
    const float cN = F.g.pN[j], cS = F.g.pS[j];
    // a neighbour outside the grid has coefficient zero
    float L0 = F.pE[i0] * (x.y - x.x);
    L0 = fmaf(F.pW[i0], w - x.x, L0);
    L0 = fmaf(cN, n.x - x.x, L0);
    L0 = fmaf(cS, s.x - x.x, L0);
    float row = F.wx[i0] * (r.x - L0);
    if (two) {
      float L1 = F.pE[i0 + 1] * (e - x.y);
      L1 = fmaf(F.pW[i0 + 1], x.x - x.y, L1);
      L1 = fmaf(cN, n.y - x.y, L1);
      L1 = fmaf(cS, s.y - x.y, L1);
      row = fmaf(F.wx[i0 + 1], r.y - L1, row);
    }
    acc = fmaf(F.wy[j], row, acc);
    s = x;
    x = n;
  }
  C.r[rb_at(I, J, C.g.ny, C.g.pk)] = acc;
}

// One thread per coarse column I and fine row j: the fine cells 2I and 2I + 1.
// Fine cell i takes parent i / 2 and its neighbour i / 2 + ox_i (ox_i in
// {-1, 0, +1}, 0 at the boundary) with weight ax_i on the neighbour, the same
// in y.
__global__ void k_mg_prolong(const MgLevel C, const float* __restrict__ ec, MgLevel F, float* __restrict__ ef) {
  pdl_enter();
  const int I = blockIdx.x * blockDim.x + threadIdx.x, j = blockIdx.y * blockDim.y + threadIdx.y;
  if (I >= C.g.nx || j >= F.g.ny) return;
  const int J = j >> 1, J2 = J + F.oy[j], ny = C.g.ny, pk = C.g.pk;
  const float ay = F.ay[j];
  const float e00 = ec[rb_at(I, J, ny, pk)], e01 = ec[rb_at(I, J2, ny, pk)];
#pragma unroll
  for (int a = 0; a < 2; ++a) {
    const int i = 2 * I + a;
    if (i >= F.g.nx) break;
    const int I2 = I + F.ox[i];
    const float ax = F.ax[i];
    const float e10 = ec[rb_at(I2, J, ny, pk)], e11 = ec[rb_at(I2, J2, ny, pk)];
    const float lo = fmaf(ax, e10 - e00, e00), hi = fmaf(ax, e11 - e01, e01);
    ef[((size_t)((i + j) & 1) * F.g.ny + j) * F.g.pk + I] += fmaf(ay, hi - lo, lo);
  }
}

inline dim3 grid_for(int nx, int ny) { return dim3((nx + 31) / 32, (ny + 7) / 8); }

// ---- the small levels of the hierarchy in one launch of one CTA
//
// Below some 9000 cells a level's four launches (smoothing twice,
// restriction, prolongation) are latency; from there down the whole V-cycle
// runs in one CTA.  Same operations as the per-level kernels: two red-black
// Gauss-Seidel sweeps before and after, residual and restriction, bilinear
// prolongation, SOR on the coarsest level; corrections from zero.  What binds
// is the chain of half-sweeps (about 100 of them, each a barrier and a few
// shared-memory loads), so a thread keeps the coefficients, right-hand sides
// and reciprocal diagonals of its cells in registers over a level's
// half-sweeps, corrections lie in shared memory inside a border of zeros (no
// tests at the boundary), and the coarsest level, at most 64 cells, runs in
// one warp.  Everything that does not change between cycles (coefficients,
// transfer weights, reciprocal diagonals of all levels) comes in one copy at
// the start.  (Reading it from global memory on every use, the levels below
// 128x64 alone took 49.8 us; a cluster of 16 CTAs with strips of rows and a
// cluster barrier per half-sweep took 68 us from 256x128 down.)
constexpr int kLowThreads = 1024;
constexpr int kLowRows = 4;  // cells of one colour a thread owns at most

struct LowCells {  // a thread's cells of one level: column pair k, rows g, g + G, ...
  int k, g, G;
  float cE[2], cW[2];                                     // per colour: the cell's column is fixed, G being even
  float cN[kLowRows], cS[kLowRows];
  float r[2][kLowRows], d[2][kLowRows];
};

// e[j + 1][i + 1] of a level, rows nx + 2 apart
__device__ __forceinline__ float* low_e(const MgLow& T, float* sm, int l) { return sm + T.lv[l].off; }
__device__ __forceinline__ float* low_r(const MgLow& T, float* sm, int l) {
  return sm + T.lv[l].off + (T.lv[l].ny + 2) * (T.lv[l].nx + 2);
}

// the constants of a level in shared memory, in the order mg_low_consts packs them
struct LowConst {
  const float *pE, *pW, *wx, *ax, *ox, *pN, *pS, *wy, *ay, *oy, *invd;
  __device__ __forceinline__ LowConst(const MgLowLevel& A, const float* base) {
    const float* p = base + A.coff;
    pE = p;
    pW = p + A.nx;
    wx = p + 2 * A.nx;
    ax = p + 3 * A.nx;
    ox = p + 4 * A.nx;
    p += 5 * A.nx;
    pN = p;
    pS = p + A.ny;
    wy = p + 2 * A.ny;
    ay = p + 3 * A.ny;
    oy = p + 4 * A.ny;
    invd = p + 5 * A.ny;
  }
};

__device__ __forceinline__ void low_load(const MgLowLevel& A, const LowConst& K, const float* r, LowCells& c) {
  const int nx = A.nx, ny = A.ny, w2 = (nx + 1) / 2;
  c.g = threadIdx.x / w2;
  c.k = threadIdx.x - c.g * w2;
  c.G = (kLowThreads / w2) & ~1;
  if (c.g >= c.G) c.g = ny;  // no cells
#pragma unroll
  for (int m = 0; m < kLowRows; ++m) {
    const int j = c.g + c.G * m;
    const bool in = j < ny;
    c.cN[m] = in ? K.pN[j] : 0.f;
    c.cS[m] = in ? K.pS[j] : 0.f;
#pragma unroll
    for (int col = 0; col < 2; ++col) {
      const int i = 2 * c.k + ((col + c.g) & 1);
      const bool cell = in && i < nx;
      if (m == 0) {
        c.cE[col] = cell ? K.pE[i] : 0.f;
        c.cW[col] = cell ? K.pW[i] : 0.f;
      }
      c.r[col][m] = cell ? r[j * nx + i] : 0.f;
      c.d[col][m] = cell ? K.invd[j * nx + i] : 0.f;
    }
  }
}

// two red-black Gauss-Seidel sweeps
__device__ __forceinline__ void low_relax(const MgLowLevel& A, float* e, const LowCells& c) {
  const int nx = A.nx, P = nx + 2;
#pragma unroll
  for (int h = 0; h < 4; ++h) {
    const int col = h & 1, i = 2 * c.k + ((col + c.g) & 1);
#pragma unroll
    for (int m = 0; m < kLowRows; ++m) {
      const int j = c.g + c.G * m;
      if (j < A.ny && i < nx) {
        float* p = e + (j + 1) * P + i + 1;
        float sum = c.cE[col] * p[1];
        sum = fmaf(c.cW[col], p[-1], sum);
        sum = fmaf(c.cN[m], p[P], sum);
        sum = fmaf(c.cS[m], p[-P], sum);
        const float gs = (sum - c.r[col][m]) * c.d[col][m];
        p[0] = fmaf(1.0f, gs - p[0], p[0]);
      }
    }
    __syncthreads();
  }
}

__global__ void __launch_bounds__(kLowThreads, 1) k_mg_low(const __grid_constant__ MgLow T, float* __restrict__ e_top) {
  extern __shared__ float low_smem[];
  const int tid = threadIdx.x;
  // the constants, before the wait (nothing writes them after set-up), and zero corrections
  float* konst = low_smem + T.nzero;
  for (int t = tid; t < T.nconst / 4; t += kLowThreads)
    reinterpret_cast<float4*>(konst)[t] = reinterpret_cast<const float4*>(T.consts)[t];
  for (int t = tid; t < T.nzero / 4; t += kLowThreads)
    reinterpret_cast<float4*>(low_smem)[t] = make_float4(0.f, 0.f, 0.f, 0.f);
  asm volatile("griddepcontrol.wait;" ::: "memory");
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  __syncthreads();
  const MgLowLevel& top = T.lv[0];
  {
    float* r = low_r(T, low_smem, 0);
    for (int t = tid; t < top.nx * top.ny; t += kLowThreads) {
      const int j = t / top.nx, i = t - j * top.nx;
      r[t] = top.r[rb_at(i, j, top.ny, top.pk)];
    }
  }
  __syncthreads();
  const int last = T.n - 1;
  LowCells c;
  for (int l = 0; l < last; ++l) {
    const MgLowLevel &A = T.lv[l], &C = T.lv[l + 1];
    float *e = low_e(T, low_smem, l), *r = low_r(T, low_smem, l), *rc = low_r(T, low_smem, l + 1);
    const LowConst K(A, konst);
    low_load(A, K, r, c);
    low_relax(A, e, c);
    const int P = A.nx + 2;
    for (int t = tid; t < C.nx * C.ny; t += kLowThreads) {
      const int J = t / C.nx, I = t - J * C.nx;
      float acc = 0.f;
#pragma unroll
      for (int b = 0; b < 2; ++b) {
        const int j = 2 * J + b;
        if (j >= A.ny) break;
        float row = 0.f;
#pragma unroll
        for (int a = 0; a < 2; ++a) {
          const int i = 2 * I + a;
          if (i >= A.nx) break;
          const float* p = e + (j + 1) * P + i + 1;
          const float x = p[0];
          float Le = K.pE[i] * (p[1] - x);
          Le = fmaf(K.pW[i], p[-1] - x, Le);
          Le = fmaf(K.pN[j], p[P] - x, Le);
          Le = fmaf(K.pS[j], p[-P] - x, Le);
          row = fmaf(K.wx[i], r[j * A.nx + i] - Le, row);
        }
        acc = fmaf(K.wy[j], row, acc);
      }
      rc[t] = acc;
    }
    __syncthreads();
  }
  {
    // coarsest level: red-black SOR; a lane owns up to two cells of each colour (more than 64 cells: the whole CTA)
    const MgLowLevel& Z = T.lv[last];
    const LowConst K(Z, konst);
    float *e = low_e(T, low_smem, last), *r = low_r(T, low_smem, last);
    const int nx = Z.nx, ny = Z.ny, P = nx + 2, w2 = (nx + 1) / 2;
    if (nx * ny <= 64) {
      if (tid < 32) {
        float aE[2][2], aW[2][2], aN[2][2], aS[2][2], rr[2][2], dd[2][2];
        float* p[2][2];
#pragma unroll
        for (int col = 0; col < 2; ++col)
#pragma unroll
          for (int q = 0; q < 2; ++q) {
            const int t = tid + 32 * q, j = t / w2, i = 2 * (t - j * w2) + ((col + j) & 1);
            const bool in = j < ny && i < nx;
            p[col][q] = in ? e + (j + 1) * P + i + 1 : nullptr;
            aE[col][q] = in ? K.pE[i] : 0.f;
            aW[col][q] = in ? K.pW[i] : 0.f;
            aN[col][q] = in ? K.pN[j] : 0.f;
            aS[col][q] = in ? K.pS[j] : 0.f;
            rr[col][q] = in ? r[j * nx + i] : 0.f;
            dd[col][q] = in ? K.invd[j * nx + i] : 0.f;
          }
        for (int s = 0; s < T.sweeps_c; ++s)
#pragma unroll
          for (int col = 0; col < 2; ++col) {
#pragma unroll
            for (int q = 0; q < 2; ++q)
              if (float* x = p[col][q]) {
                float sum = aE[col][q] * x[1];
                sum = fmaf(aW[col][q], x[-1], sum);
                sum = fmaf(aN[col][q], x[P], sum);
                sum = fmaf(aS[col][q], x[-P], sum);
                const float gs = (sum - rr[col][q]) * dd[col][q];
                x[0] = fmaf(T.omega_c, gs - x[0], x[0]);
              }
            __syncwarp();
          }
      }
    } else {
      for (int h = 0; h < 2 * T.sweeps_c; ++h) {
        for (int t = tid; t < ny * w2; t += kLowThreads) {
          const int j = t / w2, i = 2 * (t - j * w2) + ((h + j) & 1);
          if (i >= nx) continue;
          float* x = e + (j + 1) * P + i + 1;
          float sum = K.pE[i] * x[1];
          sum = fmaf(K.pW[i], x[-1], sum);
          sum = fmaf(K.pN[j], x[P], sum);
          sum = fmaf(K.pS[j], x[-P], sum);
          const float gs = (sum - r[j * nx + i]) * K.invd[j * nx + i];
          x[0] = fmaf(T.omega_c, gs - x[0], x[0]);
        }
        __syncthreads();
      }
    }
    __syncthreads();
  }
  for (int l = last - 1; l >= 0; --l) {
    const MgLowLevel &A = T.lv[l], &C = T.lv[l + 1];
    float *e = low_e(T, low_smem, l), *ec = low_e(T, low_smem, l + 1);
    const LowConst K(A, konst);
    low_load(A, K, low_r(T, low_smem, l), c);
    const int P = A.nx + 2, PC = C.nx + 2;
    for (int t = tid; t < A.nx * A.ny; t += kLowThreads) {
      const int j = t / A.nx, i = t - j * A.nx;
      const int I = (i >> 1) + 1, J = (j >> 1) + 1, I2 = I + __float_as_int(K.ox[i]), J2 = J + __float_as_int(K.oy[j]);
      const float ax = K.ax[i], ay = K.ay[j];
      const float e00 = ec[J * PC + I], e10 = ec[J * PC + I2];
      const float e01 = ec[J2 * PC + I], e11 = ec[J2 * PC + I2];
      const float lo = fmaf(ax, e10 - e00, e00), hi = fmaf(ax, e11 - e01, e01);
      e[(j + 1) * P + i + 1] += fmaf(ay, hi - lo, lo);
    }
    __syncthreads();
    low_relax(A, e, c);
  }
  const float* e = low_e(T, low_smem, 0);
  for (int t = tid; t < top.nx * top.ny; t += kLowThreads) {
    const int j = t / top.nx, i = t - j * top.nx;
    e_top[rb_at(i, j, top.ny, top.pk)] = e[(j + 1) * (top.nx + 2) + i + 1];
  }
}

constexpr int kFcgSlots = 128;

// ---- flexible conjugate gradients, FCG(1), preconditioned by the V-cycle,
// on level 0 in the volume-weighted inner product <a, b> = sum V_ij a_ij b_ij
// (L is self-adjoint in it).  Scalars stay on the device in FcgScalars:
// each inner product is accumulated in kFcgSlots FP64 slots (block b adds
// into slot b mod kFcgSlots, so the atomics do not pile onto one address);
// the last block of a reduction kernel (found by a counter after a memory
// fence) sums the slots, derives alpha or beta, and clears the slots and
// the counter for the next use.  Products and warp sums are FP32, block and
// slot sums FP64.
struct FcgScalars {
  double slot[3][kFcgSlots];  // <p, Lp>, <p, r>, <z, q>
  double pq;                  // <p, Lp> of the current direction
  float alpha, beta;
  unsigned int count;
};

// adds the block's sum of v into slots; returns true in the block that
// finished last (all other blocks' additions are then visible)
__device__ inline bool block_sum_add(float v, double* slots, unsigned int* count, bool last_check) {
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  __shared__ double ws[32];
  __shared__ bool last;
  const int t = threadIdx.x + threadIdx.y * blockDim.x, lane = t & 31, warp = t >> 5;
  const int nw = (blockDim.x * blockDim.y + 31) >> 5;
  __syncthreads();  // ws may still be read by a previous call
  if (lane == 0) ws[warp] = (double)v;
  __syncthreads();
  if (t == 0) {
    double a = 0.0;
    for (int w = 0; w < nw; ++w) a += ws[w];
    atomicAdd(&slots[(blockIdx.x + gridDim.x * blockIdx.y) % kFcgSlots], a);
    if (last_check) {
      __threadfence();
      last = atomicAdd(count, 1u) == gridDim.x * gridDim.y - 1;
    }
  }
  __syncthreads();
  return last_check && last;
}

// sum of one scalar's slots (warp 0 of the calling block), slots cleared
__device__ inline double take_slots(double* slots) {
  __shared__ double out;
  const int t = threadIdx.x + threadIdx.y * blockDim.x;
  if (t < 32) {
    double a = 0.0;
    for (int k = t; k < kFcgSlots; k += 32) {
      a += *(volatile double*)&slots[k];
      slots[k] = 0.0;
    }
    for (int o = 16; o > 0; o >>= 1) a += __shfl_xor_sync(0xffffffffu, a, o);
    if (t == 0) out = a;
  }
  __syncthreads();
  return out;
}

// The two reduction kernels run a grid-stride loop over 32 x 8 tiles with at
// most kReduceBlocks blocks, so the slot and counter atomics stay few.
constexpr int kReduceBlocks = 1216;  // 8 CTAs of 8 warps per SM: full occupancy to hide load latency

// <z, q>; the last block sets beta = -<z, q> / <p, Lp> of the previous direction
__global__ void k_fcg_dot(const MgLevel L, const float* __restrict__ dxv, const float* __restrict__ dyv,
                          const float* __restrict__ z, const float* __restrict__ q, FcgScalars* __restrict__ sc) {
  pdl_enter();
  const int tx = (L.g.nx + 31) / 32, nt = tx * ((L.g.ny + 7) / 8);
  float v = 0.f;
  for (int t = blockIdx.x; t < nt; t += gridDim.x) {
    const int i = (t % tx) * 32 + threadIdx.x, j = (t / tx) * 8 + threadIdx.y;
    if (i < L.g.nx && j < L.g.ny) {
      const size_t o = rb_at(i, j, L.g.ny, L.g.pk);
      v = fmaf(dxv[i] * dyv[j] * z[o], q[o], v);
    }
  }
  if (block_sum_add(v, sc->slot[2], &sc->count, true)) {
    const double zq = take_slots(sc->slot[2]);
    if (threadIdx.x == 0 && threadIdx.y == 0) {
      sc->beta = sc->pq != 0.0 ? (float)(-zq / sc->pq) : 0.f;
      sc->count = 0u;
    }
  }
}

// p = z (first) or z + beta p_old, formed on the fly at the cell and its
// neighbours (one pass instead of two), q = L p, <p, q>, <p, r>; the last block
// sets alpha = <p, r> / <p, q>
template <bool FIRST>
__global__ void k_fcg_apply(const MgLevel L, const float* __restrict__ dxv, const float* __restrict__ dyv,
                            const float* __restrict__ z, const float* __restrict__ p_old, float* __restrict__ p,
                            const float* __restrict__ r, float* __restrict__ q, FcgScalars* __restrict__ sc) {
  pdl_enter();
  const float beta = FIRST ? 0.f : sc->beta;
  auto dir = [&](size_t o) { return FIRST ? z[o] : fmaf(beta, p_old[o], z[o]); };
  float vpq = 0.f, vpr = 0.f;
  const int nx = L.g.nx, ny = L.g.ny, pk = L.g.pk;
  const int tx = (nx + 31) / 32, nt = tx * ((ny + 7) / 8);
  for (int t = blockIdx.x; t < nt; t += gridDim.x) {
    const int i = (t % tx) * 32 + threadIdx.x, j = (t / tx) * 8 + threadIdx.y;
    if (i >= nx || j >= ny) continue;
    const size_t o = rb_at(i, j, ny, pk);
    const float x = dir(o);
    const float xE = i < nx - 1 ? dir(rb_at(i + 1, j, ny, pk)) : x;
    const float xW = i > 0 ? dir(rb_at(i - 1, j, ny, pk)) : x;
    const float xN = j < ny - 1 ? dir(rb_at(i, j + 1, ny, pk)) : x;
    const float xS = j > 0 ? dir(rb_at(i, j - 1, ny, pk)) : x;
    float Lp = L.pE[i] * (xE - x);
    Lp = fmaf(L.pW[i], xW - x, Lp);
    Lp = fmaf(L.g.pN[j], xN - x, Lp);
    Lp = fmaf(L.g.pS[j], xS - x, Lp);
    p[o] = x;
    q[o] = Lp;
    const float Vx = dxv[i] * dyv[j] * x;
    vpq = fmaf(Vx, Lp, vpq);
    vpr = fmaf(Vx, r[o], vpr);
  }
  block_sum_add(vpq, sc->slot[0], &sc->count, false);
  if (block_sum_add(vpr, sc->slot[1], &sc->count, true)) {
    const double pq = take_slots(sc->slot[0]);
    const double pr = take_slots(sc->slot[1]);
    if (threadIdx.x == 0 && threadIdx.y == 0) {
      sc->pq = pq;
      sc->alpha = pq != 0.0 ? (float)(pr / pq) : 0.f;
      sc->count = 0u;
    }
  }
}

// x += alpha p; r -= alpha q, over the arrays as they lie (4 entries a thread;
// the padding of p and q is zero, so that of x and r stays zero while alpha is
// finite, and nothing reads it)
__global__ void k_fcg_update(int n4, const float4* __restrict__ p, const float4* __restrict__ q,
                             float4* __restrict__ x, float4* __restrict__ r, const FcgScalars* __restrict__ sc) {
  pdl_enter();
  const float alpha = sc->alpha;
  for (int o = blockIdx.x * blockDim.x + threadIdx.x; o < n4; o += gridDim.x * blockDim.x) {
    const float4 pp = p[o], qq = q[o];
    float4 xx = x[o], rr = r[o];
    xx.x = fmaf(alpha, pp.x, xx.x);
    xx.y = fmaf(alpha, pp.y, xx.y);
    xx.z = fmaf(alpha, pp.z, xx.z);
    xx.w = fmaf(alpha, pp.w, xx.w);
    rr.x = fmaf(-alpha, qq.x, rr.x);
    rr.y = fmaf(-alpha, qq.y, rr.y);
    rr.z = fmaf(-alpha, qq.z, rr.z);
    rr.w = fmaf(-alpha, qq.w, rr.w);
    x[o] = xx;
    r[o] = rr;
  }
}

}  // namespace

size_t fcg_scalars_bytes() { return sizeof(FcgScalars); }

inline int reduce_blocks(const MgLevel& L) {
  const int nt = ((L.g.nx + 31) / 32) * ((L.g.ny + 7) / 8);
  return nt < kReduceBlocks ? nt : kReduceBlocks;
}

void launch_fcg_dot(cudaStream_t s, const MgLevel& L, const float* dxv, const float* dyv, const float* z,
                    const float* q, void* sc) {
  launch_pdl(k_fcg_dot, dim3(reduce_blocks(L)), dim3(32, 8), s, L, dxv, dyv, z, q, (FcgScalars*)sc);
}
void launch_fcg_apply(cudaStream_t s, const MgLevel& L, const float* dxv, const float* dyv, const float* z,
                      const float* p_old, float* p, const float* r, float* q, void* sc, int first) {
  launch_pdl(first ? k_fcg_apply<true> : k_fcg_apply<false>, dim3(reduce_blocks(L)), dim3(32, 8), s, L, dxv, dyv, z,
             p_old, p, r, q, (FcgScalars*)sc);
}
void launch_fcg_update(cudaStream_t s, const MgLevel& L, const float* p, const float* q, float* x, float* r,
                       const void* sc) {
  const int n4 = 2 * L.g.ny * (L.g.pk / 4), blocks = (n4 + 255) / 256;
  launch_pdl(k_fcg_update, dim3(blocks < 2432 ? blocks : 2432), dim3(256), s, n4, (const float4*)p, (const float4*)q,
             (float4*)x, (float4*)r, (const FcgScalars*)sc);
}

// Fills T's shared-memory offsets for its n levels (nx, ny of lv set, finest
// first); false if the levels do not fit the CTA (threads or shared memory).
bool mg_low_layout(MgLow& T) {
  static PerDevice<bool> limit_set;
  const bool ok = limit_set.get(current_device(), [] {
    return cudaFuncSetAttribute(k_mg_low, cudaFuncAttributeMaxDynamicSharedMemorySize, kLowSmem) == cudaSuccess;
  });
  long off = 0, coff = 0;
  for (int l = 0; l < T.n; ++l) {
    MgLowLevel& A = T.lv[l];
    const int w2 = (A.nx + 1) / 2, G = (kLowThreads / w2) & ~1;
    if (l < T.n - 1 && (G < 2 || A.ny > G * kLowRows)) return false;
    A.off = (int)off;
    off += (long)(A.ny + 2) * (A.nx + 2) + (long)A.ny * A.nx;
    A.coff = (int)coff;
    coff += 5l * (A.nx + A.ny) + (long)A.nx * A.ny;
  }
  T.nzero = (int)((off + 3) / 4 * 4);
  T.nconst = (int)((coff + 3) / 4 * 4);
  T.smem = (T.nzero + T.nconst) * (int)sizeof(float);
  return ok && ((off + coff) * (long)sizeof(float) + 64) <= kLowSmem;
}

void launch_mg_low(cudaStream_t s, const MgLow& T, float* e_top) {
  cudaLaunchConfig_t lc{};
  cudaLaunchAttribute at[1];
  lc.gridDim = dim3(1);
  lc.blockDim = dim3(kLowThreads);
  lc.dynamicSmemBytes = T.smem;
  lc.stream = s;
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  lc.attrs = at;
  lc.numAttrs = 1;
  cudaLaunchKernelEx(&lc, k_mg_low, T, e_top);
}

void launch_mg_restrict(cudaStream_t s, const MgLevel& F, const float* ef, const MgLevel& C) {
  launch_pdl(k_mg_restrict, grid_for(C.g.nx, C.g.ny), dim3(32, 8), s, F, ef, C);
}

void launch_mg_prolong(cudaStream_t s, const MgLevel& C, const float* ec, const MgLevel& F, float* ef) {
  launch_pdl(k_mg_prolong, grid_for(C.g.nx, F.g.ny), dim3(32, 8), s, C, ec, F, ef);
}

}  // namespace ibm
