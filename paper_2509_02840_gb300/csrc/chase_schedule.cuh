// The chases of one rank-1 column (k_chase.cu's schedule): the op kinds, what
// each rotates, which op follows, the phases and each chase's first op.  Plain
// C++, without device code, so that the schedule can also be walked on the
// host.
#pragma once

#ifdef __CUDACC__
#define BDU_HD __host__ __device__
#else
#define BDU_HD
#endif

namespace bdu {
namespace chase {

constexpr int kLanes = 4;                    // lanes of a chase
constexpr int kSlots = 32 / kLanes;          // chases of a warp
constexpr int kRotWarps = 4;                 // warps that rotate (one per SM sub-partition)
constexpr int kGroup = kRotWarps * kSlots;   // chases of a group

enum : int { S_L0 = 0, S_R1 = 1, S_L1 = 2, S_A = 3, S_B = 4, S_C = 5, S_CL = 6, S_CR = 7, S_P2 = 8 };
constexpr int kStates = 9;

// Geometry of each op kind.  An op at position a rotates rows (a, a+1) over
// columns a-dl .. a-dl+w-1, or columns (a, a+1) over as many rows.  src 0: the
// entry eliminated is the first pair's second, 1: u(a+1) against u(a), 2: row
// 1's (1, a+1) against (1, a); S_R1 also rotates v(a), v(a+1).  next, dpos:
// the op that follows while the bulge exists, and its distance; it exists
// while a + loff <= N (limN) or <= n.
struct Geo {
  bool rows;
  int dl, w, src;
  bool withv;
  int next, dpos;
  bool limN;
  int loff;
};
BDU_HD constexpr Geo geo_of(int st) {
  return st == S_L0 ? Geo{true, 0, 3, 1, false, S_R1, 1, false, 2}
       : st == S_R1 ? Geo{false, 1, 4, 0, true, S_L1, 1, true, 2}
       : st == S_L1 ? Geo{true, 1, 4, 0, false, S_R1, 1, false, 2}
       : st == S_A  ? Geo{true, 0, 4, 0, false, S_B, 2, false, 3}
       : st == S_B  ? Geo{false, 2, 5, 0, false, S_CL, 1, true, 2}
       : st == S_C  ? Geo{false, 1, 4, 0, false, S_CL, 1, true, 2}
       : st == S_CL ? Geo{true, 1, 5, 0, false, S_CR, 2, false, 3}
       : st == S_CR ? Geo{false, 2, 5, 0, false, S_CL, 1, true, 2}
       :              Geo{false, 1, 4, 2, false, S_CL, 1, true, 2};  // S_P2
}
// Number of pairs rotated besides the source pair, and which of them holds the
// bulge (its first cell is the entry the chase looks at next).
BDU_HD constexpr int geo_pairs(int st) {
  return geo_of(st).w - (geo_of(st).src == 0 ? 1 : 0) + (geo_of(st).withv ? 1 : 0);
}
BDU_HD constexpr int geo_bulge(int st) { return geo_pairs(st) - 1 - (geo_of(st).withv ? 1 : 0); }

// The problem as a sequence of groups: phases 1, 2 and 3 in groups of kGroup
// chases (no group crosses a phase; phase 1 has one even without chases, since
// its last group does the fold).
BDU_HD inline int ceil_div(int a, int b) { return (a + b - 1) / b; }
struct Phases {
  int N, p1, p2, p3, g1, g2, g3;
};
BDU_HD inline Phases phases_of(int m, int n) {
  Phases f;
  f.N = m > n ? n + 1 : n;
  f.p1 = f.N - 1;
  f.p2 = n > 2 ? n - 2 : 0;
  f.p3 = 2 * (f.N == n + 1 ? n : n - 1);
  f.g1 = f.p1 > 0 ? ceil_div(f.p1, kGroup) : 1;
  f.g2 = ceil_div(f.p2, kGroup);
  f.g3 = ceil_div(f.p3, kGroup);
  return f;
}
// First op (state, position) of chase q (0-based) of a phase.  False when it
// does not exist, and the chase with it: the right rotation of P3c(i) for
// i + 2 > n, at the end of the band.  Nothing may decide that from the values
// there: the columns beyond n hold zeros only as long as every entry is
// finite (0 times a NaN or an infinity is NaN).
BDU_HD inline bool first_op(const Phases &F, int n, int phase, int q, int &st, int &pos) {
  if (phase == 1) { st = S_L0; pos = F.N - q - 1; }
  else if (phase == 2) { st = S_P2; pos = n - q - 1; }
  else { st = (q & 1) ? S_C : S_A; pos = q / 2 + 1 + (q & 1); }
  return st != S_C || pos + 1 <= n;
}

// Watchdog: steps a warp may take for a group where the caller names none.  A
// group needs up to about 1.3 n + 100.
BDU_HD inline long long default_steps(int n) { return 64LL * (n + 16) + 4096; }
// Polls of a wait before the kernel gives up.  A poll reads shared memory and
// takes 60 cycles at least (one of the storing warp, which reads global memory,
// 500: it has an eighth of them).  What it may have to wait for is the column:
// about 11 n steps of 3300 cycles, behind a spike of m - n rotations of 2500;
// and of a rank-r update every step also rotates rx later columns of U or V,
// four at a time, every spike rotation 32 at a time, about 1500 cycles each.
BDU_HD inline long long poll_limit(int m, int n, int rx) {
  return default_steps(n) * (256 + 16LL * ceil_div(rx, kLanes)) + 128LL * (m - n) * (1 + ceil_div(rx, 32));
}

}  // namespace chase
}  // namespace bdu
