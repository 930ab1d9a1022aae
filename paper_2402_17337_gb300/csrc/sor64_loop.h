// Control of the FP64 solve kept on chip (k_sor64.cu): when a launch checks
// the residual, when it ends, and which exchange numbers it may use.  Plain
// integer code, the same on the host and in the kernels.
#pragma once
#include <climits>

#ifdef __CUDACC__
#define SOR64_HD __host__ __device__ __forceinline__
#else
#define SOR64_HD inline
#endif

namespace ibm {

enum { SOR64_MORE = 0, SOR64_OK, SOR64_NOCONV, SOR64_DIVERGED };

// The most sweeps of one launch, whatever the interval between checks.  Tiles
// hold most of every SM's registers while they run, so a kernel of another
// stream that does not fit beside them waits for the end of their launch.  For
// 8000 sweeps of 384x192 / 512x256 / 700x350, a 2048x2048 matrix product beside
// them waits 28 / 43 / 64 ms with 8192 sweeps a launch, 3.3 / 5.2 / 7.8 ms with
// 1024 and 1.5 / 2.4 / 3.8 ms with 512; the solves take 28.7 / 43.3 / 64.1 ms,
// 28.8 / 43.4 / 64.2 and 29.0 / 43.6 / 64.4 (with 256: 2 % more).  A cluster
// leaves 136 of 152 SMs free.
constexpr int kSor64Chunk = 8192, kSor64TilesChunk = 512;
// Exchange numbers a launch reserves: it sees the sweep counts 0 .. chunk, and
// at each of them makes at most one exchange and one check.
constexpr unsigned kSor64Numbers = 2u * (kSor64Chunk + 1);

// What one launch is given, in sweeps counted from its own start.
struct Sor64Span {
  int next;   // first check (0: before the first sweep)
  int m;      // checks every m sweeps after that
  int maxs;   // sweeps left of the solve
  int chunk;  // the launch ends after so many
};

// State of a launch; every thread holds the same one, so all leave together.
struct Sor64Loop {
  int s = 0;      // sweeps done
  int next;       // sweep count of the next check
  int last = -1;  // sweep count of the last check, -1: none
  int status = SOR64_MORE;
  unsigned long long bits = 0ull;  // norm of the last check
  SOR64_HD explicit Sor64Loop(const Sor64Span& p) : next(p.next) {}
  SOR64_HD bool check_due() const { return s == next; }
  // after a check of the norm `bits_` (finite: not NaN or Inf; met: within the tolerance); true if the solve ends
  SOR64_HD bool checked(const Sor64Span& p, unsigned long long bits_, bool finite, bool met) {
    last = s;
    bits = bits_;
    next = s + p.m;
    if (!finite)
      status = SOR64_DIVERGED;
    else if (met)
      status = SOR64_OK;
    else if (s >= p.maxs)
      status = SOR64_NOCONV;
    return status != SOR64_MORE;
  }
  // after the check of this sweep count, if one was due: true if the launch ends
  SOR64_HD bool stop(const Sor64Span& p) {
    if (s >= p.maxs) status = SOR64_NOCONV;
    return status != SOR64_MORE || s >= p.chunk;
  }
};

// The launches of one solve: a check before the first sweep and every m
// sweeps, at most maxs sweeps, no launch longer than chunk sweeps.  A launch
// may lie between two checks as a whole.
struct Sor64Progress {
  int m, maxs, chunk;
  long long done = 0, due = 0;  // sweeps done; sweep count of the next check
  Sor64Span span() const {
    // a check beyond the launch needs no exact place (and the sums below stay within an int)
    const int far = chunk + 1, d = (int)(due - done < far ? due - done : far);
    const long long left = (long long)maxs - done;
    return Sor64Span{d, m < far ? m : far, (int)left, chunk};
  }
  // after a launch of that many sweeps whose last check was at `checked` (-1: none)
  void advance(int sweeps, int checked) {
    if (checked >= 0) due = done + checked + m;
    done += sweeps;
  }
};

// Reserves the exchange numbers first + 1 .. first + kSor64Numbers; *used: the
// last number reserved before on the same buffers (0: none).  True if the
// numbers have run out and start again: the buffers have to be cleared first.
inline bool sor64_reserve(unsigned* used, unsigned* first) {
  const bool wrap = *used > UINT_MAX - kSor64Numbers;
  if (wrap) *used = 0;
  *first = *used;
  *used += kSor64Numbers;
  return wrap;
}

}  // namespace ibm
