// FP64 red-black SOR of the pressure equation with the grid kept on chip for
// many sweeps (arXiv 2402.17337 Sec. 2.2, Sec. 3.1), including the residual
// checks: one launch runs up to a few thousand sweeps and leaves when the
// tolerance is met, so the host is asked once per launch, not once per check.
//
// The iterates are those of k_poisson_half / k_poisson_res (k_sor.cu): the
// same fma chains in the same order, the same reciprocal diagonal, the norm
// on the IEEE bit pattern; sweep counts and results are the same bit for bit.
//
// Two kernels, by size (rule in sor64_plan):
//   k_sor64_cluster  one thread-block cluster; each CTA owns a strip of rows.
//                    A half-sweep pushes its edge rows into the neighbours'
//                    shared memory and ends with a cluster barrier.
//   k_sor64_tiles    a cooperative launch of one CTA per SM; each CTA owns a
//                    rectangle with a halo of K cells that is recomputed for
//                    K half-sweeps between two exchanges through L2.
// FP64 issues one warp instruction per 16 clocks and SM here (2 lanes a
// clock), so an update (8 FP64 instructions) costs 128 clocks per 32 cells
// and SM; what the launch-per-half-sweep form spent on top of that was the
// launch (about 2.3 us) and, every check, a host wait (about 15 us).
#include <cstdint>
#include <mutex>

#include "ibm_internal.h"

namespace ibm {

namespace {

__device__ __forceinline__ unsigned long long abs_bits(double r) {
  return (unsigned long long)__double_as_longlong(fabs(r));
}

__device__ __forceinline__ unsigned long long warp_max(unsigned long long v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const unsigned long long w = __shfl_xor_sync(0xffffffffu, v, o);
    v = w > v ? w : v;
  }
  return v;
}

// the update and the residual of k_sor.cu
__device__ __forceinline__ double sor64(double aE, double aW, double aN, double aS, double xE, double xW, double xN,
                                        double xS, double b, double invd, double omega, double x) {
  double s = aE * xE;
  s = fma(aW, xW, s);
  s = fma(aN, xN, s);
  s = fma(aS, xS, s);
  const double gs = (s - b) * invd;
  return fma(omega, gs - x, x);
}
__device__ __forceinline__ double res64(double aE, double aW, double aN, double aS, double xE, double xW, double xN,
                                        double xS, double b, double x) {
  double L = aE * (xE - x);
  L = fma(aW, xW - x, L);
  L = fma(aN, xN - x, L);
  L = fma(aS, xS - x, L);
  return b - L;
}

// State of the sweep loop; every thread of the launch holds the same one, so
// all leave together.  Follows the host loop of solve_poisson: a check before
// the first sweep and every m sweeps, at most maxs sweeps.
struct Loop {
  int s, next;     // sweeps done, sweep count of the next check
  int last, status;
  unsigned long long bits;
};

// after a check with norm `bits`: true if the solve ends
__device__ __forceinline__ bool check_done(Loop& L, unsigned long long bits, double thr, int m, int maxs) {
  const double r = __longlong_as_double((long long)bits);
  L.last = L.s;
  L.bits = bits;
  L.next = L.s + m;
  if (!isfinite(r))
    L.status = SOR64_DIVERGED;
  else if (r <= thr)
    L.status = SOR64_OK;
  else if (L.s >= maxs)
    L.status = SOR64_NOCONV;
  return L.status != SOR64_MORE;
}

// ------------------------------------------------------------ one cluster

constexpr int CL_THREADS = 512;  // 16 warps: four per scheduler hide the FP64 latency
constexpr int CL_CPT = 2;        // cells of one colour a thread owns at most
constexpr size_t CL_SMEM = 100 * 1024;
// Which kernel a grid takes (us per sweep, checks every 8 sweeps included;
// the launch-per-half-sweep kernels of k_sor.cu in brackets):
//   70x45    cluster 1.8 [10.4], tiles 2.7
//   133x67   cluster 2.6 [10.7], tiles 3.1
//   192x128  cluster 4.8, tiles 3.7 [10]
//   512x256  tiles 6.5 [10.1]
//   1024x512 tiles 14.0 [10.3]
// so one cluster up to kClusterCells, tiles up to kTilesCells, and above
// that the kernels of k_sor.cu, whose launches are then long enough.
constexpr long kClusterCells = 12000, kTilesCells = 250000;
// Model of the tiles' time that picks their shape, in clocks, fitted to those
// measurements: one exchange, one half-sweep's barrier and latency, and 32
// updates (128 of FP64 issue, the rest index arithmetic and shared memory).
constexpr double kExchange = 7000.0, kHalf = 1300.0, kWarpUpdate = 200.0;

__device__ __forceinline__ uint32_t smem_addr(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }
__device__ __forceinline__ uint32_t map_rank(uint32_t addr, int rank) {
  uint32_t r;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(addr), "r"(rank));
  return r;
}
__device__ __forceinline__ void st_cluster(uint32_t addr, unsigned long long v) {
  asm volatile("st.shared::cluster.u64 [%0], %1;" ::"r"(addr), "l"(v) : "memory");
}
// every write above (shared memory of any CTA of the cluster) is seen by every read below
__device__ __forceinline__ void cluster_sync() {
  asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
  asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}

// CTA `rank` of `nrank` owns rows [ny rank / nrank, ny (rank+1) / nrank).  Its
// shared memory holds those rows of phi with one halo row above and below and
// a zero column on each side; a thread keeps the coefficients, b and the
// reciprocal diagonal of its cells in registers for the whole launch.  Every
// row of a strip is whole, so a half-sweep exchanges two rows and needs no
// redundant updates; with at most 16 SMs at work this pays while the grid is
// small enough for the barrier (about 0.2 us) not to be dwarfed by the
// updates.
__global__ void __launch_bounds__(CL_THREADS, 1) k_sor64_cluster(Sor64Args A, Sor64Result* __restrict__ out) {
  extern __shared__ __align__(16) double ph[];  // [(rows + 2)][nx + 2]
  __shared__ unsigned long long wmax[CL_THREADS / 32];
  __shared__ unsigned long long norms[16];
  int rank, nrank;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(rank));
  asm volatile("mov.u32 %0, %%cluster_nctarank;" : "=r"(nrank));
  const int nx = A.nx, ny = A.ny, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int j0 = (int)((long)ny * rank / nrank), j1 = (int)((long)ny * (rank + 1) / nrank), rows = j1 - j0;
  const int P = nx + 2;
  for (int t = tid; t < (rows + 2) * P; t += CL_THREADS) {
    const int r = t / P, i = t - r * P - 1, j = j0 + r - 1;
    ph[t] = (i >= 0 && i < nx && j >= 0 && j < ny) ? A.phi[A.off + (size_t)j * A.pitch + i] : 0.0;
  }
  // cells: entry k of colour c is the (tid + k threads)-th of the strip's cells of that colour
  const int w2 = (nx + 1) / 2;
  double aE[2][CL_CPT], aW[2][CL_CPT], aN[2][CL_CPT], aS[2][CL_CPT], bb[2][CL_CPT], dd[2][CL_CPT];
  int pos[2][CL_CPT];             // index into ph, 0: no cell
  uint32_t push[2][CL_CPT][2];    // copies in the neighbours' halo rows (shared::cluster), 0: none
#pragma unroll
  for (int c = 0; c < 2; ++c)
#pragma unroll
    for (int k = 0; k < CL_CPT; ++k) {
      const int t = tid + k * CL_THREADS, r = t / w2, j = j0 + r, i = 2 * (t - r * w2) + ((c + j) & 1);
      const bool in = r < rows && i < nx;
      aE[c][k] = in ? A.pE[i] : 0.0;
      aW[c][k] = in ? A.pW[i] : 0.0;
      aN[c][k] = in ? A.pN[j] : 0.0;
      aS[c][k] = in ? A.pS[j] : 0.0;
      const size_t o = A.off + (size_t)j * A.pitch + i;
      bb[c][k] = in ? A.b[o] : 0.0;
      dd[c][k] = !in ? 0.0 : A.invd ? A.invd[o] : 1.0 / (aE[c][k] + aW[c][k] + aN[c][k] + aS[c][k]);
      pos[c][k] = in ? (r + 1) * P + i + 1 : 0;
      push[c][k][0] = push[c][k][1] = 0u;
      if (in && r == 0 && rank > 0) {  // the last halo row of the strip below
        const int below = j0 - (int)((long)ny * (rank - 1) / nrank);
        push[c][k][0] = map_rank(smem_addr(ph + (below + 1) * P + i + 1), rank - 1);
      }
      if (in && r == rows - 1 && rank < nrank - 1) push[c][k][1] = map_rank(smem_addr(ph + i + 1), rank + 1);
    }
  cluster_sync();
  Loop L{0, 0, 0, SOR64_MORE, 0ull};
  for (;;) {
    if (L.s == L.next) {
      unsigned long long v = 0ull;
#pragma unroll
      for (int c = 0; c < 2; ++c)
#pragma unroll
        for (int k = 0; k < CL_CPT; ++k) {
          const int p = pos[c][k];
          if (!p) continue;
          const unsigned long long b = abs_bits(res64(aE[c][k], aW[c][k], aN[c][k], aS[c][k], ph[p + 1], ph[p - 1],
                                                      ph[p + P], ph[p - P], bb[c][k], ph[p]));
          v = b > v ? b : v;
        }
      v = warp_max(v);
      if (lane == 0) wmax[warp] = v;
      __syncthreads();
      if (warp == 0) {
        v = warp_max(lane < CL_THREADS / 32 ? wmax[lane] : 0ull);
        if (lane < nrank) st_cluster(map_rank(smem_addr(&norms[rank]), lane), v);
      }
      cluster_sync();
      v = warp_max(lane < nrank ? norms[lane] : 0ull);
      if (check_done(L, v, A.thr, A.m, A.maxs)) break;
      // the next write to norms comes after another cluster barrier (the next half-sweep's)
    }
    if (L.s >= A.maxs) {
      L.status = SOR64_NOCONV;
      break;
    }
    if (L.s >= A.chunk && L.s == L.last) break;  // hand back to the host, at a check
#pragma unroll
    for (int c = 0; c < 2; ++c) {
#pragma unroll
      for (int k = 0; k < CL_CPT; ++k) {
        const int p = pos[c][k];
        if (!p) continue;
        const double x = sor64(aE[c][k], aW[c][k], aN[c][k], aS[c][k], ph[p + 1], ph[p - 1], ph[p + P], ph[p - P],
                               bb[c][k], dd[c][k], A.omega, ph[p]);
        ph[p] = x;
        const unsigned long long xb = (unsigned long long)__double_as_longlong(x);
        if (push[c][k][0]) st_cluster(push[c][k][0], xb);
        if (push[c][k][1]) st_cluster(push[c][k][1], xb);
      }
      cluster_sync();
    }
    ++L.s;
  }
  for (int t = tid; t < rows * nx; t += CL_THREADS) {
    const int r = t / nx, i = t - r * nx;
    A.phi[A.off + (size_t)(j0 + r) * A.pitch + i] = ph[(r + 1) * P + i + 1];
  }
  if (rank == 0 && tid == 0) *out = Sor64Result{L.bits, L.last, L.s, L.status, 0};
}

// ------------------------------------------------- tiles over all SMs

constexpr int TL_THREADS = 512;

__device__ __forceinline__ unsigned ld_acquire(const unsigned* p) {
  unsigned v;
  asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ void st_release(unsigned* p, unsigned v) {
  asm volatile("st.release.gpu.global.u32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}
constexpr long long kWaitCycles = 2000000000ll;  // about 1 s at the SM clock
// waits until *p has reached v; false after kWaitCycles
__device__ __forceinline__ bool wait_flag(const unsigned* p, unsigned v) {
  if ((int)(ld_acquire(p) - v) >= 0) return true;
  const long long t0 = clock64();
  while ((int)(ld_acquire(p) - v) < 0)
    if (clock64() - t0 > kWaitCycles) return false;
  return true;
}

// CTA b owns tile (b % nbx, b / nbx) of the grid.  Shared memory holds phi, b
// and the reciprocal diagonal of the tile and a halo of K cells, and the 1-D
// coefficients.  Half-sweep h = 1 .. K after an exchange updates the tile and
// K - h cells round it (the halo shrinks by one cell each time), so the tile
// is exact after K half-sweeps; then each CTA publishes the K cells along its
// edges in one of two buffers (phi2 and phi in turn), raises its flag, waits
// for its neighbours' flags and refreshes its halo.  A buffer is written
// again two exchanges later, after the neighbours' flags of the exchange in
// between, which they raise after having read it.  All CTAs are resident at
// once (cooperative launch); a wait that lasts about a second gives up and
// the launch reports it.
__global__ void __launch_bounds__(TL_THREADS, 1) k_sor64_tiles(Sor64Args A, Sor64Tiles T, Sor64Result* __restrict__ out) {
  extern __shared__ __align__(16) double sm64[];
  __shared__ unsigned long long wmax[TL_THREADS / 32];
  const int nx = A.nx, ny = A.ny, K = T.K, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int bx = blockIdx.x % T.nbx, by = blockIdx.x / T.nbx, nb = T.nbx * T.nby;
  const int x0 = (int)((long)nx * bx / T.nbx), x1 = (int)((long)nx * (bx + 1) / T.nbx);
  const int y0 = (int)((long)ny * by / T.nby), y1 = (int)((long)ny * (by + 1) / T.nby);
  const int X0 = x0 - K, Y0 = y0 - K, RW = x1 - x0 + 2 * K, RH = y1 - y0 + 2 * K;  // region with its halo
  const int P = RW + 2;                                                         // one spare column on each side
  double* ph = sm64;                  // [RH + 2][P]
  double* sb = ph + (RH + 2) * P;     // [RH][RW]
  double* sd = sb + RH * RW;          // [RH][RW]
  double* cE = sd + RH * RW;          // [RW]
  double* cW = cE + RW;
  double* cN = cW + RW;               // [RH]
  double* cS = cN + RH;
  for (int t = tid; t < (RH + 2) * P; t += TL_THREADS) {
    const int r = t / P, i = X0 + (t - r * P) - 1, j = Y0 + r - 1;
    const bool in = i >= 0 && i < nx && j >= 0 && j < ny && i >= X0 && i < X0 + RW && j >= Y0 && j < Y0 + RH;
    ph[t] = in ? __ldcg(A.phi + A.off + (size_t)j * A.pitch + i) : 0.0;
  }
  for (int t = tid; t < RH * RW; t += TL_THREADS) {
    const int r = t / RW, i = X0 + (t - r * RW), j = Y0 + r;
    const bool in = i >= 0 && i < nx && j >= 0 && j < ny;
    const size_t o = A.off + (size_t)j * A.pitch + i;
    sb[t] = in ? A.b[o] : 0.0;
    sd[t] = in ? A.invd[o] : 0.0;
  }
  for (int t = tid; t < RW; t += TL_THREADS) {
    const int i = X0 + t;
    const bool in = i >= 0 && i < nx;
    cE[t] = in ? A.pE[i] : 0.0;
    cW[t] = in ? A.pW[i] : 0.0;
  }
  for (int t = tid; t < RH; t += TL_THREADS) {
    const int j = Y0 + t;
    const bool in = j >= 0 && j < ny;
    cN[t] = in ? A.pN[j] : 0.0;
    cS[t] = in ? A.pS[j] : 0.0;
  }
  // the neighbour this thread waits for in an exchange (the first 8 threads), -1: none
  int nbr = -1;
  if (tid < 8) {
    const int q = tid < 4 ? tid : tid + 1;  // 3 x 3 neighbourhood without its centre
    const int ax = bx + q % 3 - 1, ay = by + q / 3 - 1;
    if (ax >= 0 && ax < T.nbx && ay >= 0 && ay < T.nby) nbr = ay * T.nbx + ax;
  }
  __syncthreads();
  unsigned epoch = 0, checks = 0;
  bool dead = false;
  // refreshes the halo; false if a neighbour did not come
  auto exchange = [&]() {
    double* buf = (epoch & 1) ? A.phi : T.phi2;
    ++epoch;
    const int w = x1 - x0, h = y1 - y0;
    // the K cells along each edge of the tile (all of it if the tile is narrower than 2 K)
    for (int t = tid; t < w * h; t += TL_THREADS) {
      const int r = t / w, q = t - r * w;
      if (r < K || r >= h - K || q < K || q >= w - K)
        __stcg(buf + A.off + (size_t)(y0 + r) * A.pitch + x0 + q, ph[(r + K + 1) * P + q + K + 1]);
    }
    __syncthreads();
    if (tid == 0) {
      __threadfence();
      st_release(T.flags + blockIdx.x, epoch);
    }
    bool late = false;
    if (nbr >= 0) late = !wait_flag(T.flags + nbr, epoch);
    if (__syncthreads_or(late)) return false;
    const int top = K * RW, mid = h * 2 * K;  // halo cells: K rows below, K rows above, K columns on both sides
    for (int t = tid; t < 2 * top + mid; t += TL_THREADS) {
      int r, q;
      if (t < 2 * top) {
        r = t / RW;
        q = t - r * RW;
        if (r >= K) r += h;
      } else {
        const int u = t - 2 * top;
        r = u / (2 * K);
        q = u - r * 2 * K;
        r += K;
        if (q >= K) q += w;
      }
      const int i = X0 + q, j = Y0 + r;
      if (i >= 0 && i < nx && j >= 0 && j < ny)
        ph[(r + 1) * P + q + 1] = __ldcg(buf + A.off + (size_t)j * A.pitch + i);
    }
    __syncthreads();
    return true;
  };
  // half-sweep of colour c over the region without its outer h cells
  auto half = [&](int c, int h) {
    const int w = RW - 2 * h, hh = RH - 2 * h, w2 = (w + 1) / 2, n = hh * w2;
    const int dr = TL_THREADS / w2, dk = TL_THREADS - dr * w2;
    int r = tid / w2, k = tid - r * w2;
    for (int t = tid; t < n; t += TL_THREADS) {
      const int rr = h + r, q = h + 2 * k + ((c + Y0 + rr + X0 + h) & 1);
      if (q < RW - h) {
        const int p = (rr + 1) * P + q + 1, o = rr * RW + q;
        ph[p] = sor64(cE[q], cW[q], cN[rr], cS[rr], ph[p + 1], ph[p - 1], ph[p + P], ph[p - P], sb[o], sd[o], A.omega,
                      ph[p]);
      }
      r += dr;
      k += dk;
      if (k >= w2) {
        k -= w2;
        ++r;
      }
    }
    __syncthreads();
  };
  Loop L{0, 0, 0, SOR64_MORE, 0ull};
  int fresh = K;  // half-sweeps the halo is still good for (just loaded: all K)
  for (;;) {
    if (L.s == L.next) {
      if (fresh < 1) {
        if (!exchange()) { dead = true; break; }
        fresh = K;
      }
      unsigned long long v = 0ull;
      const int w = x1 - x0, n = w * (y1 - y0);
      for (int t = tid; t < n; t += TL_THREADS) {
        const int r = t / w, q = t - r * w + K, rr = r + K, p = (rr + 1) * P + q + 1;
        const unsigned long long b = abs_bits(res64(cE[q], cW[q], cN[rr], cS[rr], ph[p + 1], ph[p - 1], ph[p + P],
                                                    ph[p - P], sb[rr * RW + q], ph[p]));
        v = b > v ? b : v;
      }
      v = warp_max(v);
      if (lane == 0) wmax[warp] = v;
      __syncthreads();
      // the CTA's norm to its slot of this check's bank, then every CTA reads every slot
      unsigned long long* slots = T.norms + (checks & 1) * nb;
      ++checks;
      if (warp == 0) {
        v = warp_max(lane < TL_THREADS / 32 ? wmax[lane] : 0ull);
        if (lane == 0) {
          __stcg(slots + blockIdx.x, v);
          __threadfence();
          st_release(T.flags + nb + blockIdx.x, checks);
        }
      }
      v = 0ull;
      bool late = false;
      for (int t = tid; t < nb; t += TL_THREADS) {
        if (!wait_flag(T.flags + nb + t, checks)) { late = true; break; }
        const unsigned long long b = __ldcg(slots + t);
        v = b > v ? b : v;
      }
      v = warp_max(v);
      __syncthreads();  // warp 0 has read wmax
      if (lane == 0) wmax[warp] = v;
      if (__syncthreads_or(late)) { dead = true; break; }
      v = warp_max(lane < TL_THREADS / 32 ? wmax[lane] : 0ull);
      __syncthreads();  // wmax is written again by the next check
      if (check_done(L, v, A.thr, A.m, A.maxs)) break;
    }
    if (L.s >= A.maxs) {
      L.status = SOR64_NOCONV;
      break;
    }
    if (L.s >= A.chunk && L.s == L.last) break;
    if (fresh < 2) {
      if (!exchange()) { dead = true; break; }
      fresh = K;
    }
    half(0, K - fresh + 1);
    half(1, K - fresh + 2);
    fresh -= 2;
    ++L.s;
  }
  const int w = x1 - x0, n = w * (y1 - y0);
  if (!dead && L.s != L.last) {
    // an exchange may have followed the last check: every CTA has read its
    // halo from phi before any of them writes its whole tile there
    ++checks;
    if (tid == 0) {
      __threadfence();
      st_release(T.flags + nb + blockIdx.x, checks);
    }
    for (int t = tid; t < nb; t += TL_THREADS)
      if (!wait_flag(T.flags + nb + t, checks)) dead = true;
    dead = __syncthreads_or(dead);
  }
  if (!dead)
    for (int t = tid; t < n; t += TL_THREADS) {
      const int r = t / w, q = t - r * w;
      A.phi[A.off + (size_t)(y0 + r) * A.pitch + x0 + q] = ph[(r + K + 1) * P + q + K + 1];
    }
  if (dead && tid == 0) atomicOr(&out->late, 1);
  if (blockIdx.x == 0 && tid == 0) {
    out->bits = L.bits;
    out->checked = L.last;
    out->sweeps = L.s;
    out->status = L.status;
  }
}

}  // namespace

namespace {

// Device limits the plan depends on, asked once per device.
struct Sor64Dev {
  int sms = 0, coop = 0, smem = 0, cluster = 0;
};

const Sor64Dev& sor64_device() {
  static Sor64Dev dev[64];
  static std::once_flag once[64];
  static const Sor64Dev none;
  int d = 0;
  if (cudaGetDevice(&d) != cudaSuccess || d < 0 || d >= 64) return none;
  std::call_once(once[d], [d] {
    Sor64Dev v;
    cudaDeviceGetAttribute(&v.sms, cudaDevAttrMultiProcessorCount, d);
    cudaDeviceGetAttribute(&v.coop, cudaDevAttrCooperativeLaunch, d);
    cudaDeviceGetAttribute(&v.smem, cudaDevAttrMaxSharedMemoryPerBlockOptin, d);
    v.smem -= 1024;  // static shared memory of the kernels
    bool ok = cudaFuncSetAttribute(k_sor64_tiles, cudaFuncAttributeMaxDynamicSharedMemorySize, v.smem) == cudaSuccess;
    if (!ok) v.coop = 0;
    ok = cudaFuncSetAttribute(k_sor64_cluster, cudaFuncAttributeMaxDynamicSharedMemorySize, CL_SMEM) == cudaSuccess &&
         cudaFuncSetAttribute(k_sor64_cluster, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) == cudaSuccess;
    for (int c = 16; ok && c >= 8 && !v.cluster; c /= 2) {  // 16 where the device takes it, else the portable 8
      cudaLaunchConfig_t lc{};
      cudaLaunchAttribute at[1];
      lc.gridDim = dim3(c);
      lc.blockDim = dim3(CL_THREADS);
      lc.dynamicSmemBytes = CL_SMEM;
      at[0].id = cudaLaunchAttributeClusterDimension;
      at[0].val.clusterDim = {(unsigned)c, 1, 1};
      lc.attrs = at;
      lc.numAttrs = 1;
      int n = 0;
      if (cudaOccupancyMaxActiveClusters(&n, k_sor64_cluster, &lc) == cudaSuccess && n > 0) v.cluster = c;
    }
    cudaGetLastError();
    dev[d] = v;
  });
  return dev[d];
}

size_t tiles_smem(int w, int h, int K) {
  const size_t RW = w + 2 * K, RH = h + 2 * K;
  return sizeof(double) * ((RH + 2) * (RW + 2) + 2 * RH * RW + 2 * RW + 2 * RH);
}

}  // namespace

// Which kernel a grid takes, from its size alone.
Sor64Plan sor64_plan(int nx, int ny, bool tiles) {
  Sor64Plan p;
  const Sor64Dev& d = sor64_device();
  if (d.cluster && ny >= d.cluster) {
    const int rows = (ny + d.cluster - 1) / d.cluster, w2 = (nx + 1) / 2;
    if (rows * w2 <= CL_THREADS * CL_CPT && sizeof(double) * (rows + 2) * (nx + 2) <= CL_SMEM &&
        (!tiles || (long)nx * ny <= kClusterCells)) {
      p.kind = Sor64Plan::CLUSTER;
      p.nbx = d.cluster;
      return p;
    }
  }
  if (!tiles || !d.coop || d.sms < 1 || (long)nx * ny > kTilesCells) return p;
  // Tiles: the split and halo depth with the smallest modelled time per
  // half-sweep: the updates of the shrinking region, and an exchange every K
  // half-sweeps.
  double best = 0.0;
  for (int K = 2; K <= 8; K += 2)
    for (int nbx = 1; nbx <= d.sms && nbx * K <= nx; ++nbx) {
      int nby = d.sms / nbx;
      if (nby > ny / K) nby = ny / K;
      if (nby < 1) continue;
      const int w = (nx + nbx - 1) / nbx, h = (ny + nby - 1) / nby;
      const size_t smem = tiles_smem(w, h, K);
      if (smem > (size_t)d.smem) continue;
      double t = kExchange;
      for (int q = 1; q <= K; ++q) {
        const double n = (double)((w + 2 * (K - q) + 1) / 2) * (h + 2 * (K - q));
        const double warps = n / 32;
        t += kWarpUpdate * warps + kHalf;
      }
      t /= K;
      if (p.kind == Sor64Plan::NONE || t < best) {
        best = t;
        p.kind = Sor64Plan::TILES;
        p.nbx = nbx;
        p.nby = nby;
        p.K = K;
        p.smem = smem;
      }
    }
  return p;
}

int sor64_max_tiles() { return sor64_device().sms; }

cudaError_t launch_sor64(cudaStream_t s, const Sor64Plan& p, const Sor64Args& a, const Sor64Tiles& t, Sor64Result* out) {
  cudaError_t e = cudaMemsetAsync(out, 0, sizeof(Sor64Result), s);
  if (e != cudaSuccess) return e;
  if (p.kind == Sor64Plan::CLUSTER) {
    const int rows = (a.ny + p.nbx - 1) / p.nbx;
    cudaLaunchConfig_t lc{};
    cudaLaunchAttribute at[1];
    lc.gridDim = dim3(p.nbx);
    lc.blockDim = dim3(CL_THREADS);
    lc.dynamicSmemBytes = sizeof(double) * (rows + 2) * (a.nx + 2);
    lc.stream = s;
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim = {(unsigned)p.nbx, 1, 1};
    lc.attrs = at;
    lc.numAttrs = 1;
    return cudaLaunchKernelEx(&lc, k_sor64_cluster, a, out);
  }
  Sor64Tiles tt = t;
  tt.nbx = p.nbx;
  tt.nby = p.nby;
  tt.K = p.K;
  e = cudaMemsetAsync(tt.flags, 0, 2 * sizeof(unsigned) * p.nbx * p.nby, s);
  if (e != cudaSuccess) return e;
  Sor64Args aa = a;
  void* args[] = {&aa, &tt, &out};
  return cudaLaunchCooperativeKernel((const void*)k_sor64_tiles, dim3(p.nbx * p.nby), dim3(TL_THREADS), args, p.smem, s);
}

}  // namespace ibm
