// FP64 red-black SOR of the pressure equation with the grid kept on chip for
// many sweeps (arXiv 2402.17337 Sec. 2.2, Sec. 3.1), including the residual
// checks: one launch runs hundreds (tiles) or thousands (cluster) of sweeps and
// leaves when the tolerance is met, so the host is asked once per launch, not
// once per check (sor64_loop.h: when a launch checks and when it ends).
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
#include <type_traits>

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

// after a check with norm `bits`: true if the solve ends
__device__ __forceinline__ bool check_done(Sor64Loop& L, unsigned long long bits, const Sor64Args& A) {
  const double r = __longlong_as_double((long long)bits);
  return L.checked(A.span, bits, isfinite(r), r <= A.thr);
}

// ------------------------------------------------------------ one cluster

constexpr int CL_THREADS = 512;  // 16 warps: four per scheduler hide the FP64 latency
constexpr int CL_CPT = 2;        // cells of one colour a thread owns at most
constexpr size_t CL_SMEM = 100 * 1024;
// Which kernel a grid takes (us per sweep, checks every 8 sweeps included;
// the launch-per-half-sweep kernels of k_sor.cu in brackets):
//   70x45    cluster 1.8 [10.4], tiles 2.1
//   110x56   cluster 2.1 [10.5]
//   133x67   cluster 2.6 [10.7], tiles 2.9
//   160x80   cluster 3.0 [11.0], tiles 2.9
//   192x96   tiles 2.8 [11.0]
//   192x128  cluster 4.8, tiles 2.7 [10]
//   384x192  tiles 3.8 [11.0]
//   512x256  tiles 5.1 [10.1]
//   700x350  tiles 7.3 [10.2]
//   1024x512 tiles 12 [10.3]
// so one cluster up to kClusterCells, tiles up to kSor64TilesCells, and above
// that the kernels of k_sor.cu, whose launches are then long enough.  A
// half-sweep's floor is its chain of eight dependent FP64 instructions, about
// 160 clocks each, and a barrier: 0.9 us.
constexpr long kClusterCells = 10500;
// Model of the tiles' time that picks their shape, in clocks, fitted to those
// measurements: one exchange, one half-sweep's barrier and latency, and 32
// updates (128 of FP64 issue, the rest shared memory).
constexpr double kExchange = 1500.0, kHalf = 1500.0, kWarpUpdate = 190.0;

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
  Sor64Loop L(A.span);
  for (;;) {
    if (L.check_due()) {
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
      if (check_done(L, v, A)) break;
      // the next write to norms comes after another cluster barrier (the next half-sweep's)
    }
    if (L.stop(A.span)) break;
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

constexpr int TL_THREADS = 640;
constexpr int TL_CPT = 2;  // cells of one colour a thread owns at most

// A double with its exchange number: two 8-byte words {half, number}, each
// written and read whole, so a reader that sees the number in both has the
// value and needs no flag or fence (a fence here waits for every store of the
// SM: with data, fence and flag 512x256 took 6.4 us a sweep, with this 5.1).
__device__ __forceinline__ void post(unsigned long long* p, unsigned long long v, unsigned no) {
  const unsigned long long lo = (v & 0xffffffffull) | ((unsigned long long)no << 32);
  const unsigned long long hi = (v >> 32) | ((unsigned long long)no << 32);
  asm volatile("st.relaxed.gpu.global.v2.b64 [%0], {%1, %2};" ::"l"(p), "l"(lo), "l"(hi) : "memory");
}
__device__ __forceinline__ bool peek(const unsigned long long* p, unsigned no, unsigned long long& v) {
  unsigned long long lo, hi;
  asm volatile("ld.relaxed.gpu.global.v2.b64 {%0, %1}, [%2];" : "=l"(lo), "=l"(hi) : "l"(p) : "memory");
  v = (lo & 0xffffffffull) | (hi << 32);
  return (unsigned)(lo >> 32) == no && (unsigned)(hi >> 32) == no;
}
// waits for exchange number no at p; false after limit clocks (0: unless it is there already)
__device__ __forceinline__ bool fetch(const unsigned long long* p, unsigned no, unsigned long long& v, long long limit) {
  if (peek(p, no, v)) return true;
  const long long t0 = clock64();
  while (!peek(p, no, v))
    if (clock64() - t0 >= limit) return false;
  return true;
}

// Cell u of the perimeter of the w x h rectangle at (x, y), walked from its
// corner (x, y) along the bottom row, the right column, the top row and the
// left column; consecutive cells alternate in colour.
__device__ __forceinline__ void perimeter(int x, int y, int w, int h, int u, int& i, int& j) {
  if (u < w) {
    i = x + u;
    j = y;
  } else if ((u -= w) < h - 1) {
    i = x + w - 1;
    j = y + 1 + u;
  } else if ((u -= h - 1) < w - 1) {
    i = x + w - 2 - u;
    j = y + h - 1;
  } else {
    u -= w - 1;
    i = x;
    j = y + h - 2 - u;
  }
}

// CTA b owns tile (b % nbx, b / nbx) of the grid.  Shared memory holds phi of
// the tile and a halo of K cells.  Half-sweep h = 1 .. K after an exchange
// updates the tile and K - h cells round it, so the tile is exact after K
// half-sweeps; then each CTA posts the K cells along its edges and picks up
// its halo from its neighbours' posts (two buffers in turn: a buffer is
// written again two exchanges later, after the neighbours' posts of the
// exchange in between, which they make after having read it).  The cells of a
// colour are listed tile first, then ring by ring outwards, so those of
// half-sweep h are the first of the list; a thread keeps the coefficients, b
// and the reciprocal diagonal of its TL_CPT entries in registers.  All CTAs
// are resident at once (cooperative launch); a wait that lasts A.wait clocks
// gives up and the launch reports it.
__global__ void __launch_bounds__(TL_THREADS, 1) k_sor64_tiles(Sor64Args A, Sor64Tiles T, Sor64Result* __restrict__ out) {
  extern __shared__ __align__(16) double sm64[];
  __shared__ unsigned long long wmax[TL_THREADS / 32];
  const int nx = A.nx, ny = A.ny, K = T.K, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int bx = blockIdx.x % T.nbx, by = blockIdx.x / T.nbx, nb = T.nbx * T.nby;
  const int x0 = (int)((long)nx * bx / T.nbx), x1 = (int)((long)nx * (bx + 1) / T.nbx), w = x1 - x0;
  const int y0 = (int)((long)ny * by / T.nby), y1 = (int)((long)ny * (by + 1) / T.nby), h = y1 - y0;
  const int X0 = x0 - K, Y0 = y0 - K, P = w + 2 * K, RH = h + 2 * K;  // region with its halo
  double* ph = sm64;  // [RH][P]
  for (int t = tid; t < RH * P; t += TL_THREADS) {
    const int r = t / P, i = X0 + (t - r * P), j = Y0 + r;
    const bool in = i >= 0 && i < nx && j >= 0 && j < ny;
    ph[t] = in ? __ldcg(A.phi + A.off + (size_t)j * A.pitch + i) : 0.0;
  }
  const int w2 = (w + 1) / 2, n_own = h * w2;
  double aE[2][TL_CPT], aW[2][TL_CPT], aN[2][TL_CPT], aS[2][TL_CPT], bb[2][TL_CPT], dd[2][TL_CPT];
  int pos[2][TL_CPT];  // index into ph, 0: no cell
#pragma unroll
  for (int c = 0; c < 2; ++c)
#pragma unroll
    for (int k = 0; k < TL_CPT; ++k) {
      int t = tid + k * TL_THREADS, i, j;
      bool in = true;
      if (t < n_own) {
        const int r = t / w2;
        j = y0 + r;
        i = x0 + 2 * (t - r * w2) + ((c + x0 + j) & 1);
        in = i < x1;
      } else {
        t -= n_own;
        int q = 1;
        while (q < K && t >= w + h + 4 * q - 2) t -= w + h + 4 * q++ - 2;
        in = q < K;
        perimeter(x0 - q, y0 - q, w + 2 * q, h + 2 * q, 2 * t + ((c + x0 + y0) & 1), i, j);
      }
      in = in && i >= 0 && i < nx && j >= 0 && j < ny;
      aE[c][k] = in ? A.pE[i] : 0.0;
      aW[c][k] = in ? A.pW[i] : 0.0;
      aN[c][k] = in ? A.pN[j] : 0.0;
      aS[c][k] = in ? A.pS[j] : 0.0;
      const size_t o = A.off + (size_t)j * A.pitch + i;
      bb[c][k] = in ? A.b[o] : 0.0;
      dd[c][k] = !in ? 0.0 : A.invd ? A.invd[o] : 1.0 / (aE[c][k] + aW[c][k] + aN[c][k] + aS[c][k]);
      pos[c][k] = in ? (j - Y0) * P + i - X0 : 0;
    }
  __syncthreads();
  unsigned no = T.first;  // number of the last exchange or check
  unsigned exchanges = 0, checks = 0;  // each alternates between its two buffers
  bool dead = false;
  // refreshes the halo; false if a neighbour did not come
  auto exchange = [&]() {
    ++no;
    unsigned long long* buf = T.words + ((exchanges++ & 1) ? T.stride : 0);
    // the K outermost rings of the tile (all of it if it is narrower), then the K rings round it
    const int rings = min(K, (min(w, h) + 1) / 2);
    int total = 0;
    for (int q = 0; q < rings; ++q) {
      const int ww = w - 2 * q, hh = h - 2 * q, n = ww > 1 && hh > 1 ? 2 * (ww + hh) - 4 : ww * hh;
      for (int u = tid - total % TL_THREADS < 0 ? tid - total % TL_THREADS + TL_THREADS : tid - total % TL_THREADS; u < n;
           u += TL_THREADS) {
        int i, j;
        if (ww > 1 && hh > 1) {
          perimeter(x0 + q, y0 + q, ww, hh, u, i, j);
        } else {
          i = x0 + q + (ww > 1 ? u : 0);
          j = y0 + q + (ww > 1 ? 0 : u);
        }
        post(buf + 2 * ((size_t)j * nx + i), (unsigned long long)__double_as_longlong(ph[(j - Y0) * P + i - X0]), no);
      }
      total += n;
    }
    bool late = false;
    total = 0;
    for (int q = 1; q <= K; ++q) {
      const int n = 2 * (w + h) + 8 * q - 4;
      for (int u = tid - total % TL_THREADS < 0 ? tid - total % TL_THREADS + TL_THREADS : tid - total % TL_THREADS;
           u < n && !late; u += TL_THREADS) {
        int i, j;
        perimeter(x0 - q, y0 - q, w + 2 * q, h + 2 * q, u, i, j);
        if (i < 0 || i >= nx || j < 0 || j >= ny) continue;
        unsigned long long v;
        late = !fetch(buf + 2 * ((size_t)j * nx + i), no, v, A.wait);
        ph[(j - Y0) * P + i - X0] = __longlong_as_double((long long)v);
      }
      total += n;
    }
    return !__syncthreads_or(late);
  };
  // half-sweep hs of colour C after an exchange: the first n cells of the list
  auto half = [&](auto colour, int n) {
    constexpr int c = decltype(colour)::value;
#pragma unroll
    for (int k = 0; k < TL_CPT; ++k) {
      const int p = pos[c][k];
      if (p && tid + k * TL_THREADS < n)
        ph[p] = sor64(aE[c][k], aW[c][k], aN[c][k], aS[c][k], ph[p + 1], ph[p - 1], ph[p + P], ph[p - P], bb[c][k],
                      dd[c][k], A.omega, ph[p]);
    }
    __syncthreads();
  };
  Sor64Loop L(A.span);
  int fresh = K;  // half-sweeps the halo is still good for (just loaded: all K)
  for (;;) {
    if (L.check_due()) {
      if (fresh < 1) {
        if (!exchange()) { dead = true; break; }
        fresh = K;
      }
      unsigned long long v = 0ull;
#pragma unroll
      for (int c = 0; c < 2; ++c)
#pragma unroll
        for (int k = 0; k < TL_CPT; ++k) {
          const int p = pos[c][k];
          if (!p || tid + k * TL_THREADS >= n_own) continue;
          const unsigned long long b = abs_bits(res64(aE[c][k], aW[c][k], aN[c][k], aS[c][k], ph[p + 1], ph[p - 1],
                                                      ph[p + P], ph[p - P], bb[c][k], ph[p]));
          v = b > v ? b : v;
        }
      v = warp_max(v);
      if (lane == 0) wmax[warp] = v;
      __syncthreads();
      // the CTA's norm to its slot, then every CTA reads every slot
      ++no;
      // (a slot is written again two checks later: every CTA has read it before it posts to the check in between)
      unsigned long long* slots = T.norms + ((checks++ & 1) ? 2 * nb : 0);
      if (warp == 0) {
        v = warp_max(lane < TL_THREADS / 32 ? wmax[lane] : 0ull);
        if (lane == 0) post(slots + 2 * blockIdx.x, v, no);
      }
      v = 0ull;
      bool late = false;
      for (int t = tid; t < nb && !late; t += TL_THREADS) {
        unsigned long long b;
        late = !fetch(slots + 2 * t, no, b, A.wait);
        v = b > v ? b : v;
      }
      v = warp_max(v);
      __syncthreads();  // warp 0 has read wmax
      if (lane == 0) wmax[warp] = v;
      if (__syncthreads_or(late)) { dead = true; break; }
      v = warp_max(lane < TL_THREADS / 32 ? wmax[lane] : 0ull);
      __syncthreads();  // wmax is written again by the next check
      if (check_done(L, v, A)) break;
    }
    if (L.stop(A.span)) break;
    if (fresh < 2) {
      if (!exchange()) { dead = true; break; }
      fresh = K;
    }
    // rings 1 .. fresh - 1, then fresh - 2: (w + h + 4 q - 2) cells of a colour in ring q
    auto cells = [&](int q) { return n_own + q * (w + h - 2) + 2 * q * (q + 1); };
    half(std::integral_constant<int, 0>{}, cells(fresh - 1));
    half(std::integral_constant<int, 1>{}, cells(fresh - 2));
    fresh -= 2;
    ++L.s;
  }
  if (!dead)
    for (int t = tid; t < w * h; t += TL_THREADS) {
      const int r = t / w, q = t - r * w;
      A.phi[A.off + (size_t)(y0 + r) * A.pitch + x0 + q] = ph[(r + K) * P + q + K];
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

Sor64Dev sor64_device() {
  static PerDevice<Sor64Dev> dev;
  const int d = current_device();
  if (d < 0) return Sor64Dev{};
  return dev.get(d, [d] {
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
    return v;
  });
}

size_t tiles_smem(int w, int h, int K) { return sizeof(double) * (size_t)(w + 2 * K) * (h + 2 * K); }

// entries of a colour's list: the tile and K - 1 rings
long tiles_list(int w, int h, int K) {
  const int q = K - 1;
  return (long)h * ((w + 1) / 2) + (long)q * (w + h - 2) + 2l * q * (q + 1);
}

}  // namespace

// Which kernel a grid takes, from its size alone.
Sor64Plan sor64_plan(int nx, int ny) {
  Sor64Plan p;
  const Sor64Dev d = sor64_device();
  if (d.cluster && ny >= d.cluster) {
    const int rows = (ny + d.cluster - 1) / d.cluster, w2 = (nx + 1) / 2;
    if (rows * w2 <= CL_THREADS * CL_CPT && sizeof(double) * (rows + 2) * (nx + 2) <= CL_SMEM &&
        (!d.coop || (long)nx * ny <= kClusterCells)) {
      p.kind = Sor64Plan::CLUSTER;
      p.nbx = d.cluster;
      return p;
    }
  }
  if (!d.coop || d.sms < 1 || d.sms > kSor64MaxTiles || (long)nx * ny > kSor64TilesCells) return p;
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
      if (smem > (size_t)d.smem || tiles_list(w, h, K) > TL_THREADS * TL_CPT) continue;
      double t = kExchange;
      for (int q = 1; q <= K; ++q) t += kWarpUpdate * (tiles_list(w, h, q) / 32.0) + kHalf;
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
  Sor64Args aa = a;
  void* args[] = {&aa, &tt, &out};
  return cudaLaunchCooperativeKernel((const void*)k_sor64_tiles, dim3(p.nbx * p.nby), dim3(TL_THREADS), args, p.smem, s);
}

}  // namespace ibm
