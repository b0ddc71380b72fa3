// K2: rotation generation and bulge chasing for one rank-1 column
// (Sec. 3.4, Algorithm 2), in FP64.
//
// The reduction of the core M = Bd + u v^T is a sequence of "chases": each
// starts with one rotation and pushes the bulge it creates down the band.
// Chases are generated in a fixed order (the schedule below) and every chase
// moves monotonically down the band, so chase t may run concurrently with
// chase t-1 as long as it stays a few positions behind it: 3 between
// neighbouring phase-1 chases, 4 otherwise.  This keeps every band cell's
// read/write order that of the sequential algorithm, so the result equals a
// one-rotation-at-a-time execution.
//
// Schedule (1-based; N = n+1 if m > n else n):
//   spike:    j = m..n+2: left (j-1, j) zeroing u(j)              [one warp]
//   phase 1:  chase P1(j), j = N..2: left (j-1, j) zeroing u(j); then for
//             i = j-1, j+1, ...: right (i+1, i+2) zeroing M(i, i+2), left
//             (i+2, i+3) zeroing M(i+3, i+1), while the bulge exists
//   fold:     row 1 += u(1) v^T                                   [one warp]
//   phase 2:  chase P2(j), j = n..3: right (j-1, j) zeroing M(1, j), then
//             chase_lower(j-1)
//   phase 3:  chases P3b(i), P3c(i), i = 1..n-1 (and n when N = n+1):
//             P3b: left (i, i+1) zeroing M(i+1, i); right (i+2, i+3)
//                  zeroing M(i, i+3); chase_lower(i+2)
//             P3c: right (i+1, i+2) zeroing M(i, i+2); chase_lower(i+1)
//   chase_lower(k): left (k+1, k+2) zeroing M(k+2, k); right (k+3, k+4)
//             zeroing M(k+1, k+4); k += 3, while the bulge exists.
//
// The engine is a pipeline of groups of kGroup consecutive chases, one thread
// block a group.  A chase depends on earlier chases only, and only through
// rows that they have passed, so everything flows one way: a block loads the
// rows of the band behind the previous group's last chase into a circular
// window in its shared memory, its chases run there, and the rows behind its
// own last chase go back to global memory for the next group.  One word per
// group says up to which row all groups so far are done (release / acquire);
// its latency is paid once per kGroup chases, not on every step, and no block
// waits for a slower one behind it.  (Before, all chases of a column advanced
// together, one rotation per cluster barrier: 3.0 us a step at n = 4096, of
// which the FP64 sequence was a third.)
//
// Inside a block, four warps run the rotations, one per SM sub-partition: on
// GB300 a warp's FP64 instruction holds its sub-partition's FP64 unit for 64
// cycles whatever the number of active lanes, so what a step costs is the
// number of FP64 instructions in one warp's chain.  Each chase therefore has
// kLanes = 4 lanes: the rotation is computed by all four at once (c, s and r,
// products or quotients with one factor in common, in one instruction), and
// each lane rotates one of the up to four pairs: 12 FP64 instructions a step in
// the fast form (16 + 10 with a lane per chase), 22 in the exact one.  A fifth warp loads rows, a sixth stores
// them and publishes the group's word.  Groups are taken from a ticket
// counter in order, so a block that waits for the group before it waits for
// one that is already running: any number of resident blocks makes progress.
//
// Arithmetic.  Exact (FP64 form): every multiply, add, divide and square root
// is a separately rounded IEEE operation (__dmul_rn, __dadd_rn, __ddiv_rn,
// __dsqrt_rn), never a fused multiply-add, so each value is fully determined
// by its inputs.  Fast (mixed form, where Q and P are FP32 anyway): fused
// multiply-adds, and 1/sqrt(f^2 + g^2) from an FP32 seed refined by one
// third-order Newton step in FP64 (error well below an FP64 ulp), which
// avoids the long-latency FP64 division and square-root sequences.
#include <algorithm>

#include "bdu_internal.cuh"
#include "chase_schedule.cuh"

namespace bdu {
namespace {

using namespace chase;

// ----------------------------------------------------------------------------
// rotation arithmetic
// ----------------------------------------------------------------------------
__device__ __forceinline__ double mul(double a, double b) { return __dmul_rn(a, b); }
// x != 0 and |x| compared through the bit pattern, on the integer pipes
__device__ __forceinline__ bool nz(double x) { return (__double_as_longlong(x) << 1) != 0; }
__device__ __forceinline__ unsigned long long absbits(double x) {
  return (unsigned long long)__double_as_longlong(x) & 0x7fffffffffffffffULL;
}
__device__ __forceinline__ double add(double a, double b) { return __dadd_rn(a, b); }

// Rotation generator (Eqs. giv, giv1, zero handling of Sec. 3.4):
// [c s; -s c][f; g] = [r; 0], c >= 0, r = sign(f) hypot(f, g).  Returns false
// when g == 0 (no rotation); f == 0 gives c = 0, s = 1, r = g.  hypot uses
// power-of-two safe scaling.  Written without branches on the common path so
// that the lanes of a warp share its (long-latency) FP64 instructions.
__device__ __forceinline__ bool rotg_exact(double f, double g, double &c, double &s, double &r) {
  const unsigned long long bf = absbits(f), bg = absbits(g);
  const unsigned long long bm = bf > bg ? bf : bg;  // |x| order = bit-pattern order
  const double sigma = bm > 0x5F30000000000000ULL ? 0x1p-600 : (bm < 0x20B0000000000000ULL ? 0x1p600 : 1.0);
  const double fs = mul(f, sigma), gs = mul(g, sigma);
  const double h = __dsqrt_rn(add(mul(fs, fs), mul(gs, gs)));
  const double rs = copysign(h, f);
  const bool fz = bf == 0;
  const double den = fz ? 1.0 : rs;
  c = fz ? 0.0 : __ddiv_rn(fs, den);
  s = fz ? 1.0 : __ddiv_rn(gs, den);
  r = fz ? g : __ddiv_rn(rs, sigma);
  return bg != 0;
}

// FP32 value of x (|x| <= 2, or NaN), rounded to nearest even, formed from
// the bit pattern on the integer pipes: on GB300 an FP64 <-> FP32 conversion
// instruction holds the SM sub-partition's FP64 unit for about 90 cycles.
// Magnitudes below 2^-126 (under FP32's normal range) become signed zero.
__device__ __forceinline__ float f32_of(double x) {
  const unsigned long long b = (unsigned long long)__double_as_longlong(x);
  const unsigned long long mag = b & 0x7fffffffffffffffULL;
  const unsigned sign = (unsigned)(b >> 32) & 0x80000000u;
  unsigned long long t = mag >> 29;  // exponent and the top 23 mantissa bits
  const unsigned rem = (unsigned)(mag & 0x1fffffffULL);
  t += (rem > 0x10000000u || (rem == 0x10000000u && (t & 1))) ? 1 : 0;
  unsigned r = (unsigned)(t - (896ULL << 23));  // exponent bias 1023 -> 127
  r = mag < (897ULL << 52) ? 0u : r;
  r = mag >= 0x7ff0000000000000ULL ? 0x7fc00000u : r;
  return __uint_as_float(r | sign);
}

// A pair (x, y) after the rotation.
template <bool FAST> struct Arith;
template <> struct Arith<false> {
  static __device__ __forceinline__ double px(double c, double s, double x, double y) { return add(mul(c, x), mul(s, y)); }
  static __device__ __forceinline__ double py(double c, double s, double x, double y) { return add(mul(-s, x), mul(c, y)); }
};
template <> struct Arith<true> {
  static __device__ __forceinline__ double px(double c, double s, double x, double y) { return fma(c, x, s * y); }
  static __device__ __forceinline__ double py(double c, double s, double x, double y) { return fma(c, y, -(s * x)); }
};

// ----------------------------------------------------------------------------
// chases, groups, the window
// ----------------------------------------------------------------------------
constexpr int kThreads = 32 * (kRotWarps + 2);
// Rows of the window.  A group's chases are at most 6 positions apart while
// none of them has to wait for rows (lag 4, and a position advances by up to
// 3 at a time), and an op at position p touches rows p-2..p+4.
constexpr int kWin = 256;
static_assert(kWin >= 6 * kGroup + 16, "a group's chases must fit the window");
constexpr int kCells = 9;                    // per row: six diagonals, row 1, v, u
constexpr int kRowBytes = kCells * 8;        // (an odd number of doubles: no bank conflicts down a column)
constexpr int kWinBytes = kWin * kRowBytes;
constexpr int kR1 = 6, kV = 7, kU = 8;       // the last three cells of a row
constexpr int kPad = 8;                      // rows of zeros below the band
constexpr int kFar = 1 << 29;                // a position or row beyond every other
constexpr int kAborted = -1;                 // progress word of a group that gave up

// info word of a state: bit 0 rows, 1-2 bulge pair, 3-6 next, 7-8 dpos,
// 9 limN, 10-12 loff, 13 the chase ends when this op finds nothing to rotate
__host__ __device__ constexpr int geo_info(int st) {
  return (geo_of(st).rows ? 1 : 0) | geo_bulge(st) << 1 | geo_of(st).next << 3 | geo_of(st).dpos << 7 |
         (geo_of(st).limN ? 1 : 0) << 9 | geo_of(st).loff << 10 | (st == S_A ? 0 : 1) << 13;
}
// Byte offset of cell `cell` of the row `drow` away from the position, from
// the row two above it (the topmost an op touches).
__device__ __forceinline__ int rel(int drow, int cell) { return (drow + 2) * kRowBytes + cell * 8; }

// Progress words in shared memory (one CTA) and in global memory (the groups).
// What the word's writer stored before it is seen by the lane that read the
// word at once, and by the others after the warp's next __syncwarp() (a shuffle
// orders no memory).  In the loading and storing warps lane 0's reading counts,
// among the rotating ones that of a chase's first lane.
__device__ __forceinline__ int ld_cta(const int *p) {
  int v;
  asm volatile("ld.acquire.cta.shared.s32 %0, [%1];\n" : "=r"(v) : "r"((uint32_t)__cvta_generic_to_shared(p)) : "memory");
  return v;
}
__device__ __forceinline__ void st_cta(int *p, int v) {
  asm volatile("st.release.cta.shared.s32 [%0], %1;\n" ::"r"((uint32_t)__cvta_generic_to_shared(p)), "r"(v) : "memory");
}
__device__ __forceinline__ int ld_gpu(const int *p) {
  int v;
  asm volatile("ld.acquire.gpu.global.s32 %0, [%1];\n" : "=r"(v) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ void st_gpu(int *p, int v) {
  asm volatile("st.release.gpu.global.s32 [%0], %1;\n" ::"l"(p), "r"(v) : "memory");
}

__device__ __forceinline__ int of_lane0(int v) { return __shfl_sync(0xffffffffu, v, 0); }

struct Shared {
  double win[kWin * kCells];     // cell c of row r at (r mod kWin) * kCells + c
  int4 tab[kStates * kLanes];    // byte offsets of a lane's cells: source pair, rotated pair (x < 0: none)
  int info[kStates];
  int front[kRotWarps];          // position the next warp's first chase stays behind
  int least[kRotWarps];          // least position of the warp's unfinished chases
  int loaded;                    // rows up to this one are in the window (kAborted: give up)
  int flushed;                   // rows up to this one are back in global memory
  int before;                    // the previous group's word as last read
  int far;                       // kFar (what the first warp stays behind)
  int done;                      // rotating warps that have finished the group
  int loader_done;
  int ticket;
};

__device__ __forceinline__ double &cell_at(Shared &S, int off) {
  return *reinterpret_cast<double *>(reinterpret_cast<char *>(S.win) + off);
}
// byte offset of M(i, j) (row 1 dense)
__device__ __forceinline__ int cell_off(int i, int j) {
  return i == 1 ? (j & (kWin - 1)) * kRowBytes + kR1 * 8 : (i & (kWin - 1)) * kRowBytes + (j - i + 2) * 8;
}

__device__ __forceinline__ double make_f64(int hi, unsigned lo) { return __hiloint2double(hi, (int)lo); }

// y ~ 1/sqrt(q), q in [0.25, 2): an FP32 seed (q truncated to FP32 and the
// seed widened through the bit patterns, about 22 correct bits) refined by
// y0 (1 + e/2 + 3e^2/8), e = 1 - q y0^2 (third-order Newton step).
__device__ __forceinline__ double rsqrt_f64(double q) {
  const unsigned qf = __funnelshift_l((unsigned)__double2loint(q), (unsigned)__double2hiint(q), 3) - (896u << 23);
  const unsigned u = __float_as_uint(rsqrtf(__uint_as_float(qf)));
  const double y = make_f64((int)((u >> 3) + (896u << 20)), u << 29);
  const double e = fma(-(q * y), y, 1.0);
  return fma(y * e, fma(0.375, e, 0.5), y);
}

// The rotation of one chase by its four lanes (f, g the same in all of them;
// every lane of the warp calls it).  c and s end up in every lane, r in lanes
// 2 and 3.
//
// Fast: from y ~ 1/sqrt(f^2 + g^2) of the inputs scaled by the power of two
// that brings the larger into [0.5, 1) (exact, on the exponent fields; f^2 +
// g^2 then lies in [0.25, 2)).  Inputs whose scaling would leave the normal
// range -- the larger exponent outside [2, 2044], the smaller input subnormal
// or more than 2^1021 below the larger -- take the plain form.
//
// Exact: the square root and the two quotients are formed from y ~
// 1/sqrt(f^2 + g^2) by Newton corrections with exact remainders (Markstein,
// "IA-64 and Elementary Functions", ch. 8-9), and each is then compared with
// the rounding interval around it through its exact remainder: h is the
// rounded root of q iff q - h^2 lies in (-h ulp, h ulp], a quotient the
// rounded one iff its remainder is below half an ulp of it times h (a tie
// cannot occur).  16 FP64 instructions: the rotation took 4.4k cycles at n =
// 1024 with the library's square root and division and takes 1.8k.  The scaling by
// the larger exponent is exact and does not change any rounding while both
// inputs lie within 2^-500..2^500 and within 2^900 of each other; for others
// plain is set, and the caller takes the plain form (rot_plain: rotg_exact).
template <bool FAST>
__device__ __forceinline__ void rot_lanes(double f, double g, int lane, double &c, double &s, double &r, bool &plain) {
  const int role = lane & 3;
  const int fh = __double2hiint(f), gh = __double2hiint(g);
  const unsigned fl = (unsigned)__double2loint(f), gl = (unsigned)__double2loint(g);
  const bool fz = ((unsigned)(fh << 1) | fl) == 0, gz = ((unsigned)(gh << 1) | gl) == 0;
  const int ef = (fh >> 20) & 0x7ff, eg = (gh >> 20) & 0x7ff;
  const int ex = max(ef, eg), en = min(ef, eg);
  const int dk = (1022 - ex) << 20;
  const int sf = fh & (int)0x80000000;
  if (FAST) {
    plain = !gz && (ex < 2 || ex > 2044 || (!fz && (en == 0 || en + 1021 < ex)));
    const double fs = fz ? 0.0 : make_f64(fh + dk, fl), gs = gz ? 0.0 : make_f64(gh + dk, gl);
    const double q = fma(fs, fs, gs * gs);
    const double y = rsqrt_f64(q);
    // c = |fs| y, s = sign(f) gs y and the scaled |r| = q y in one instruction
    const double a = role == 0 ? fabs(fs) : role == 1 ? make_f64(__double2hiint(gs) ^ sf, (unsigned)__double2loint(gs)) : q;
    const double pr = a * y;
    c = __shfl_sync(0xffffffffu, pr, lane & ~3);
    s = __shfl_sync(0xffffffffu, pr, (lane & ~3) | 1);
    r = make_f64((__double2hiint(pr) - dk) ^ sf, (unsigned)__double2loint(pr));
  } else {
    plain = !gz && !fz && (en < 523 || ex > 1523 || ex - en > 900);
    const double fs = make_f64((fh & 0x7fffffff) + dk, fl), gs = make_f64((gh & 0x7fffffff) + dk, gl);  // magnitudes
    const double q = add(mul(fs, fs), mul(gs, gs));
    const double y = rsqrt_f64(q);
    const double num = (role & 1) ? gs : fs;
    const double s0 = q * y, c0 = num * y;
    const double h1 = fma(fma(-s0, s0, q), make_f64(__double2hiint(y) - (1 << 20), (unsigned)__double2loint(y)), s0);
    const long long hb = __double_as_longlong(h1);
    const long long rem = __double_as_longlong(fma(-h1, h1, q));
    const long long hu = hb + ((long long)((int)(hb >> 52) - (1023 + 52)) << 52);  // h1 times its ulp
    const long long rmag = rem & 0x7fffffffffffffffLL;
    int fix = rem >= 0 ? (rmag > hu ? 1 : 0) : (rmag >= hu || hb == 0x3FF0000000000000LL ? -1 : 0);
    const double h = __longlong_as_double(hb + fix);
    const double q1 = fma(fma(-c0, h, num), y, c0);
    const long long qb = __double_as_longlong(q1);
    const long long qrem = __double_as_longlong(fma(-q1, h, num));
    long long half = __double_as_longlong(h) + ((long long)((int)(qb >> 52) - (1023 + 53)) << 52);  // h times q1's half ulp
    if (qrem < 0 && (qb & 0xfffffffffffffLL) == 0) half -= 1LL << 52;  // (below a power of two ulps are half as wide)
    fix = (qrem & 0x7fffffffffffffffLL) > half ? (qrem < 0 ? -1 : 1) : 0;
    const double quo = __longlong_as_double(qb + fix);
    const double oth = __shfl_xor_sync(0xffffffffu, quo, 1);
    c = (role & 1) ? oth : quo;
    s = (role & 1) ? quo : oth;
    s = make_f64(__double2hiint(s) | ((fh ^ gh) & (int)0x80000000), (unsigned)__double2loint(s));
    r = make_f64((__double2hiint(h) - dk) | sf, (unsigned)__double2loint(h));
  }
  c = fz ? 0.0 : c;
  s = fz ? 1.0 : s;
  r = fz ? g : r;
}

__device__ __noinline__ void rot_plain(double f, double g, double &c, double &s, double &r) {
  rotg_exact(f, g, c, s, r);
}

// One op of a chase, as a lane sees it: byte offsets in the window of the
// source pair (f, g), which becomes (r, 0), and of the lane's own pair; info
// word of the state, negative when the lane has no pair.
struct Op {
  int f, g, x, y, info;
};
// (away from row 1)
__device__ __forceinline__ Op plan_op(Shared &S, int st, int pos, int q) {
  Op o;
  const int4 tb = S.tab[st * kLanes + q];
  o.info = S.info[st] | (tb.w & (int)0x80000000);
  const int base = ((pos - 2) & (kWin - 1)) * kRowBytes;
  // offsets past the window's end wrap (as unsigned, the smaller is in range)
  auto wrap = [](int off) { return (int)min((unsigned)off, (unsigned)(off - kWinBytes)); };
  o.f = wrap(base + tb.x);
  o.g = wrap(base + tb.y);
  o.x = wrap(base + tb.z);
  o.y = wrap(base + (tb.w & 0xffff));
  return o;
}
// The last position an op touches row 1 from; row 1 is kept apart.
constexpr int kNearTop = 3;
__device__ __forceinline__ Op plan_any(Shared &S, int st, int pos, int q) {
  Op o = plan_op(S, st, pos, q);
  if (pos <= kNearTop) {
    if (o.info & 1) {
      if (pos == 1) {  // S_L0 or S_A: rows 1 and 2, columns from 1 (2) on
        const int j = pos + q + (st == S_L0 ? 0 : 1);
        o.x = cell_off(1, j);
        o.y = cell_off(2, j);
        if (st == S_A) { o.f = cell_off(1, 1); o.g = cell_off(2, 1); }
      }
    } else if (pos - (st == S_B || st == S_CR ? 2 : 1) == 1) {  // columns whose first row is row 1
      o.f = cell_off(1, pos);
      o.g = cell_off(1, pos + 1);
      if (st == S_P2 && q == 0) o.info |= (int)0x80000000;  // (its first band pair is the source pair)
    }
  }
  return o;
}

// A group's chases, slots kSlots w .. kSlots w + kSlots - 1: warp w.
//
// A step's critical path is its FP64 chain; everything else that can be known
// before the chain ends is computed beside it, for the case that every bulge
// goes on: the next op and its addresses, whether it may run, what the warp
// publishes.  When some chase of the warp ends (or skips a step), that is
// thrown away and recomputed.  (One after the other, at n = 1024: 2.9k cycles
// a step in the mixed form, of which 1.35k the chain.)
template <bool FAST, bool EXTRA>
__device__ __forceinline__ void rotate_chases(const ChaseArgs &Ar, Shared &S, const Phases &F, int phase, int q0, int cnt,
                                              int w, int max_steps, int &steps, long long max_polls) {
  using A = Arith<FAST>;
  const int lane = threadIdx.x & 31, q = lane & 3, slot = w * kSlots + (lane >> 2);
  const int n = Ar.n, N = F.N;
  int st = S_A, pos = kFar;
  const bool mine = slot < cnt;
  bool done = !mine || !first_op(F, n, phase, q0 + slot, st, pos);
  if (done) pos = kFar;
  int eff = done ? 0 : pos;  // what the next chase stays behind
  // a finished chase passes on what it had to stay behind itself
  auto relay = [](int ahead) { return ahead >= kFar ? kFar : ahead - 1; };
  const int lag = phase == 1 ? 3 : 4;
  const int t = (phase == 1 ? 0 : phase == 2 ? F.p1 : F.p1 + F.p2) + q0 + slot;  // chase number
  const int cap = Ar.st.cap;
  // where the lane writes its part of a record: the pair (lane 0), c (1), s (3)
  char *recL = nullptr, *recR = nullptr;
  const int stride = q == 0 ? 4 : 8;
  if (mine && done && q == 0) Ar.st.Ln[t] = Ar.st.Rn[t] = 0;
  if (!done) {
    const size_t rec = (size_t)t * cap;
    if (q == 0) {
      recL = reinterpret_cast<char *>(Ar.st.La + rec); recR = reinterpret_cast<char *>(Ar.st.Ra + rec);
    } else if (FAST) {
      recL = reinterpret_cast<char *>(Ar.st.Lf + rec) + (q >> 1) * 4;
      recR = reinterpret_cast<char *>(Ar.st.Rf + rec) + (q >> 1) * 4;
    } else {
      recL = reinterpret_cast<char *>((q == 1 ? Ar.st.Lc : Ar.st.Ls) + rec);
      recR = reinterpret_cast<char *>((q == 1 ? Ar.st.Rc : Ar.st.Rs) + rec);
    }
  }
  const int *const before = w > 0 ? &S.front[w - 1] : &S.far;
  int nl = 0, nr = 0, tried = 0;
  bool full = false;  // a record did not fit
  long long polls = 0;
  int told = -1;  // last published front
  Op op = plan_any(S, st, done ? 4 : pos, q);
  bool may = false, any = false;  // may this chase's (some chase's) next op run?
  for (;;) {
    __syncwarp();
    if (!any) {
      const int pw = ld_cta(before);
      const int have = ld_cta(&S.loaded);
      int ahead = __shfl_up_sync(0xffffffffu, eff, kLanes);
      if (lane < kLanes) ahead = pw;
      if (done) eff = relay(ahead);
      may = !done && pos + lag <= ahead && pos + 4 <= have;
      any = __any_sync(0xffffffffu, may);
      __syncwarp();
      if (!any) {
        if (__any_sync(0xffffffffu, have == kAborted)) break;
        const int last = __shfl_sync(0xffffffffu, eff, 31);
        if (last != told) {
          told = last;
          if (lane == 31) st_cta(&S.front[w], last);
        }
        if (last >= kFar && __all_sync(0xffffffffu, done)) break;
        if (++polls > max_polls) {
          if (lane == 0) {
            atomicOr(Ar.status, ERR_STEPS);
            st_cta(&S.loaded, kAborted);
          }
          break;
        }
        continue;
      }
    }
    const int info = op.info;
    const bool rows = info & 1, has = info >= 0;
    const double f = cell_at(S, op.f), g = cell_at(S, op.g);
    const double x = cell_at(S, op.x), y = cell_at(S, op.y);
    // A chase runs when its first lane says so, by the progress words as that
    // lane has read them (the others follow behind the __syncwarp() above).
    // Asked for here, beside the loads: a column of 2048, exact, 35.6 ms, of
    // 4096, fast, 55.2 (as soon as the next step is planned: 37.1, 54.9; a
    // vote of the four lanes there: 37.5, 55.6).
    const bool run = __shfl_sync(0xffffffffu, (int)may, lane & ~3);
    // later columns of U (V), lane q those of number q, q + kLanes, ...: the
    // first one's entries are loaded before the rotation
    double *ex = nullptr;
    double eu = 0.0, ev = 0.0;
    if (EXTRA) {
      const int ldx = rows ? Ar.m : n;
      if (q < Ar.rx && run && pos < ldx) {
        ex = (rows ? Ar.Ux : Ar.Vx) + (size_t)q * ldx - 1 + pos;
        eu = __ldcg(ex);
        ev = __ldcg(ex + 1);
      }
    }
    // (relied on from the next step on, behind the __syncwarp() it starts with)
    const int pw = ld_cta(before);
    const int have = ld_cta(&S.loaded);
    // the rotation, and beside it the step after this one for the case that
    // every bulge goes on (in one basic block, for the compiler to interleave)
    double c, s, r;
    bool plain;
    rot_lanes<FAST>(f, g, lane, c, s, r, plain);
    const bool exists = pos + ((info >> 10) & 7) <= ((info >> 9) & 1 ? N : n);
    const int npos = run ? pos + ((info >> 7) & 3) : pos, nst = run ? (info >> 3) & 15 : st;
    Op nop = plan_op(S, nst, npos, q);
    int neff = done ? eff : npos;
    int ahead = __shfl_up_sync(0xffffffffu, neff, kLanes);
    ahead = lane < kLanes ? pw : ahead;
    neff = done ? relay(ahead) : neff;
    const bool nmay = !done && npos + lag <= ahead && npos + 4 <= have;
    const bool nany = __any_sync(0xffffffffu, nmay);
    int front = __shfl_sync(0xffffffffu, neff, 31);
    int least = __reduce_min_sync(0xffffffffu, npos);
    const bool ok = run && nz(g);
    const int k = rows ? nl : nr;
    char *const rp = (rows ? recL : recR) + (size_t)(unsigned)(k * stride);
    const bool put = ok && k < cap;
    full = full || (ok && k >= cap);
    nl += ok && rows ? 1 : 0;
    nr += ok && !rows ? 1 : 0;
    tried += run ? 1 : 0;
    // (scaling extremes; near row 1 the plan above does not hold)
    const bool top = __any_sync(0xffffffffu, least <= kNearTop);
    if (__any_sync(0xffffffffu, plain)) {
      if (plain) rot_plain(f, g, c, s, r);
    }
    const double nx = A::px(c, s, x, y), ny = A::py(c, s, x, y);
    if (FAST) {
      const int v = q == 0 ? pos : __float_as_int(f32_of(q == 1 ? c : s));
      if (put && q != 2) *reinterpret_cast<int *>(rp) = v;
    } else {
      if (put && q == 0) *reinterpret_cast<int *>(rp) = pos;
      if (put && (q & 1)) *reinterpret_cast<double *>(rp) = q == 1 ? c : s;
    }
    if (ok && has) { cell_at(S, op.x) = nx; cell_at(S, op.y) = ny; }
    if (ok && q == 2) { cell_at(S, op.f) = r; cell_at(S, op.g) = 0.0; }
    if (EXTRA) {
      if (ok && ex) {
        __stcg(ex, A::px(c, s, eu, ev));
        __stcg(ex + 1, A::py(c, s, eu, ev));
        for (int kx = q + kLanes; kx < Ar.rx; kx += kLanes) {
          const int ldx = rows ? Ar.m : n;
          double *X = (rows ? Ar.Ux : Ar.Vx) + (size_t)kx * ldx - 1 + pos;
          const double a0 = __ldcg(X), a1 = __ldcg(X + 1);
          __stcg(X, A::px(c, s, a0, a1));
          __stcg(X + 1, A::py(c, s, a0, a1));
        }
      }
    }
    const unsigned bulges = __ballot_sync(0xffffffffu, ok && has && nz(nx));
    const bool bulge = (bulges >> ((lane & ~3) + ((info >> 1) & 3))) & 1;
    const bool on = exists && (bulge || !((info >> 13) & 1));
    if (__all_sync(0xffffffffu, on || !run) && !top) {
      pos = npos;
      st = nst;
      op = nop;
      eff = neff;
      may = nmay;
      any = nany;
    } else {
      __syncwarp();
      if (run) {
        if (on) {
          pos = npos;
          st = nst;
        } else if (ok && st == S_R1 && pos + 3 <= n && nz(cell_at(S, cell_off(pos + 1, pos + 3)))) {
          pos += 2;
        } else if (ok && st == S_CL && pos + 4 <= N && nz(cell_at(S, cell_off(pos + 4, pos + 2)))) {
          pos += 3;
        } else {
          if (!ok && (st == S_R1 || st == S_L1 || st == S_CL || st == S_CR)) atomicOr(Ar.status, ERR_SCHEDULE);
          done = true;
          pos = kFar;
          if (q == 0) { Ar.st.Ln[t] = nl; Ar.st.Rn[t] = nr; }
        }
      }
      __syncwarp();
      eff = done ? eff : pos;
      ahead = __shfl_up_sync(0xffffffffu, eff, kLanes);
      ahead = lane < kLanes ? pw : ahead;
      if (done) eff = relay(ahead);  // (at once, or the chase behind it would lose steps)
      op = plan_any(S, st, done ? 4 : pos, q);
      any = false;
      front = __shfl_sync(0xffffffffu, eff, 31);
      least = __reduce_min_sync(0xffffffffu, pos);
    }
    told = front;
    __syncwarp();
    if (lane == 31) {
      st_cta(&S.front[w], front);
      st_cta(&S.least[w], least);
    }
    if (++steps > max_steps) {
      if (lane == 0) {
        atomicOr(Ar.status, ERR_STEPS);
        st_cta(&S.loaded, kAborted);
      }
      break;
    }
  }
  if (full) atomicOr(Ar.status, ERR_CAP);
  // rotation counts
  const int sl = __reduce_add_sync(0xffffffffu, q == 0 ? nl : 0);
  const int sr = __reduce_add_sync(0xffffffffu, q == 0 ? nr : 0);
  const int sa = __reduce_add_sync(0xffffffffu, q == 0 ? tried : 0);
  if (lane == 0) {
    if (sl) atomicAdd(&Ar.counters[phase], (unsigned long long)sl);
    if (sr) atomicAdd(&Ar.counters[4 + phase], (unsigned long long)sr);
    if (sa) atomicAdd(&Ar.counters[8], (unsigned long long)sa);
    __threadfence_block();
    atomicAdd(&S.done, 1);
  }
}

// Rows into the window, as far as the previous group has finished them and the
// window has room.
__device__ __forceinline__ void load_rows(const ChaseArgs &Ar, Shared &S, const Phases &F, int base, const int *prev,
                                          bool wait_all) {
  const int lane = threadIdx.x & 31, n = Ar.n, N = F.N, end = N + kPad;
  int have = base - 1, before = prev ? 0 : kFar;
  for (;;) {
    __syncwarp();
    if (of_lane0(ld_cta(&S.done)) == kRotWarps) break;
    if (before < kFar) {
      before = of_lane0(ld_gpu(prev));
      if (before == kAborted) {
        if (lane == 0) st_cta(&S.loaded, kAborted);
        break;
      }
      // phase 2 starts from row 1 as the fold leaves it: nothing is passed on before
      if (wait_all && before < kFar) continue;
      if (lane == 0) st_cta(&S.before, before);
    }
    int lim = before >= N ? end : before;
    lim = min(lim, of_lane0(ld_cta(&S.flushed)) + kWin);
    if (lim <= have) continue;
    __syncwarp();
    for (int r0 = have + 1; r0 <= lim; r0 += 32) {
      const int r = r0 + lane;
      if (r <= lim) {
        double v[kCells];
        const bool row = r <= N;
#pragma unroll
        for (int o = 0; o < 6; o++) {
          const int j = r + o - 2;
          v[o] = row && j >= 1 && j <= n ? __ldcg(Ar.band.dg[o] + r) : 0.0;
        }
        v[kR1] = r <= n ? __ldcg(Ar.band.r1 + r) : 0.0;
        v[kV] = r <= n ? __ldcg(Ar.band.v + r) : 0.0;
        v[kU] = row ? __ldcg(Ar.band.u + r) : 0.0;
        double *d = S.win + (r & (kWin - 1)) * kCells;
#pragma unroll
        for (int o = 0; o < kCells; o++) d[o] = v[o];
      }
    }
    have = lim;
    __syncwarp();
    if (lane == 0) {
      const int old = ld_cta(&S.loaded);  // (an abort mark set by another warp stays)
      __threadfence_block();
      if (old != kAborted) atomicCAS(&S.loaded, old, have);
    }
    __syncwarp();
  }
  if (lane == 0) st_cta(&S.loader_done, 1);
}

// Rows r0..r1 back to global memory.  Returns whether one of this lane's rows
// holds a nonzero (or a NaN) outside the matrix, which no rotation leaves there
// while every entry is finite.
__device__ __forceinline__ bool store_rows(const ChaseArgs &Ar, Shared &S, const Phases &F, int r0, int r1) {
  const int lane = threadIdx.x & 31, n = Ar.n, N = F.N;
  bool outside = false;
  for (int r = r0 + lane; r <= r1; r += 32) {
    const double *d = S.win + (r & (kWin - 1)) * kCells;
#pragma unroll
    for (int o = 0; o < 6; o++) {
      const int j = r + o - 2;
      outside |= nz(d[o]) && (r > N || j < 1 || j > n);
    }
    outside |= (r > n && (nz(d[kR1]) || nz(d[kV]))) || (r > N && nz(d[kU]));
    if (r <= N) {
#pragma unroll
      for (int o = 0; o < 6; o++) __stcg(Ar.band.dg[o] + r, d[o]);
      __stcg(Ar.band.u + r, d[kU]);
    }
    if (r <= n) {
      __stcg(Ar.band.r1 + r, d[kR1]);
      __stcg(Ar.band.v + r, d[kV]);
    }
  }
  return outside;
}

// Rows the group's last chase has left, back to global memory; then the
// group's word.  fold: the last group of phase 1.  stall (failure injection):
// 1: the word is never written, 2: it never says that the group is done.
template <bool FAST>
__device__ __forceinline__ void publish_rows(const ChaseArgs &Ar, Shared &S, const Phases &F, int base, const int *prev,
                                             int *word, bool fold, long long max_polls, int stall) {
  const int lane = threadIdx.x & 31, n = Ar.n;
  int flushed = base - 1, told = 0;
  bool outside = false;
  for (;;) {
    __syncwarp();
    // (the order of these loads: what is stored below was final before them)
    const bool all = of_lane0(ld_cta(&S.done) == kRotWarps && ld_cta(&S.loader_done));
    int least = kFar;
#pragma unroll
    for (int w = 0; w < kRotWarps; w++) least = min(least, ld_cta(&S.least[w]));
    least = of_lane0(least);
    const int have = of_lane0(ld_cta(&S.loaded));
    const int bf = of_lane0(ld_cta(&S.before));
    __syncwarp();
    if (have == kAborted) {
      if (lane == 0) st_gpu(word, kAborted);
      return;
    }
    if (!all) {
      const int lim = min(min(least - 3, have), flushed + kWin);
      if (lim > flushed) {
        outside |= store_rows(Ar, S, F, flushed + 1, lim);
        flushed = lim;
        __syncwarp();
        if (lane == 0) st_cta(&S.flushed, flushed);
      }
      const int f = min(flushed, bf);
      if (f > told) {
        told = f;
        __syncwarp();
        if (lane == 0 && stall != 1) st_gpu(word, f);
      }
      continue;
    }
    break;
  }
  // the group's chases are finished: the rest of its rows, then everything
  // below is as the groups before leave it
  const int loaded = of_lane0(ld_cta(&S.loaded));
  __syncwarp();
  outside |= store_rows(Ar, S, F, flushed + 1, loaded);
  if (outside) atomicOr(Ar.status, ERR_BAND);
  __syncwarp();
  int before = prev ? 0 : kFar;
  for (long long polls = 0; before < kFar; polls++) {
    before = of_lane0(ld_gpu(prev));
    if (before == kAborted || polls > max_polls) {
      if (lane == 0) {
        if (before != kAborted) atomicOr(Ar.status, ERR_STEPS);
        st_cta(&S.loaded, kAborted);
        st_gpu(word, kAborted);
      }
      return;
    }
    if (before < kFar && before > told) {
      told = before;
      if (lane == 0) st_gpu(word, before);
    }
  }
  if (fold) {  // row 1 += u(1) v^T
    __threadfence();
    __syncwarp();
    const double u1 = __ldcg(Ar.band.u + 1);
    for (int j = 1 + lane; j <= n; j += 32)
      __stcg(Ar.band.r1 + j, Arith<FAST>::px(1.0, u1, __ldcg(Ar.band.r1 + j), __ldcg(Ar.band.v + j)));
  }
  __syncwarp();
  if (lane == 0 && stall != 1) st_gpu(word, stall ? F.N : kFar);
}

// The spike (m > n): one sequential chain on u in global memory, by one warp:
// 32 entries of u are loaded together, the running entry stays in a register;
// lane k holds u (and, of a rank-r update, the later columns k, k + 32, ... of
// U go through global memory).
template <bool FAST>
__device__ __forceinline__ void run_spike(const ChaseArgs &Ar) {
  using A = Arith<FAST>;
  const int m = Ar.m, n = Ar.n, lane = threadIdx.x & 31;
  int ns = 0;
  double *u = Ar.band.u;
  if (m < n + 2) {
    if (lane == 0) Ar.st.Sn[0] = 0;
    return;
  }
  double run = __ldcg(u + m);  // u(j), as the rotations so far have left it
  for (int j0 = m; j0 >= n + 2; j0 -= 32) {
    const int cnt = min(32, j0 - (n + 1));  // rotations (j-1, j), j = j0 .. j0-cnt+1
    const double mine = lane < cnt ? __ldcg(u + j0 - 1 - lane) : 0.0;  // u(j0 - 1 - lane)
    double left = 0.0, kc = 0.0, ks = 0.0;  // u(j0 - lane) afterwards; the rotation of j = j0 - lane
    bool got = false;
    for (int k = 0; k < cnt; k++) {
      const int j = j0 - k;
      const double f = __shfl_sync(0xffffffffu, mine, k);
      double c = 1.0, s = 0.0, r = 0.0;
      bool plain;
      rot_lanes<FAST>(f, run, lane, c, s, r, plain);
      if (plain) rot_plain(f, run, c, s, r);
      const bool ok = nz(run);
      r = __shfl_sync(0xffffffffu, r, 2);
      if (lane == k) {
        left = ok ? 0.0 : run;
        kc = c; ks = s; got = ok;
      }
      if (ok) {
        for (int x = lane; x < Ar.rx; x += 32) {
          double *U = Ar.Ux + (size_t)x * m - 1;
          const double a = U[j - 1], b = U[j];
          U[j - 1] = A::px(c, s, a, b);
          U[j] = A::py(c, s, a, b);
        }
      }
      run = ok ? r : f;
    }
    if (lane < cnt) __stcg(u + j0 - lane, left);
    const unsigned have = __ballot_sync(0xffffffffu, got);
    if (got) {
      const int o = ns + __popc(have & ((1u << lane) - 1));
      Ar.st.Sc[o] = kc; Ar.st.Ss[o] = ks; Ar.st.Sa[o] = j0 - lane - 1;
      if (Ar.st.Sf) Ar.st.Sf[o] = make_float2(f32_of(kc), f32_of(ks));
    }
    ns += __popc(have);
  }
  if (lane == 0) {
    __stcg(u + n + 1, run);
    Ar.st.Sn[0] = ns;
    atomicAdd(&Ar.counters[0], (unsigned long long)ns);
  }
  __threadfence();
}

template <bool FAST, bool EXTRA>
__device__ __forceinline__ void engine(const ChaseArgs &Ar) {
  __shared__ Shared S;
  const int me = threadIdx.x, wid = me >> 5;
  const int m = Ar.m, n = Ar.n;
  const Phases F = phases_of(m, n);
  const int groups = F.g1 + F.g2 + F.g3;
  int *const ticket = Ar.sync, *const words = Ar.sync + 2;
  for (int e = me; e < kStates * kLanes; e += kThreads) {
    const int st = e / kLanes, q = e % kLanes;
    const Geo G = geo_of(st);
    const int qq = q + (G.src == 0 ? 1 : 0);
    int4 t;
    if (G.src == 1) { t.x = rel(0, kU); t.y = rel(1, kU); }
    else if (G.src == 2) { t.x = rel(0, kR1); t.y = rel(1, kR1); }
    else if (G.rows) { t.x = rel(0, 2 - G.dl); t.y = rel(1, 1 - G.dl); }
    else { t.x = rel(-G.dl, G.dl + 2); t.y = rel(-G.dl, G.dl + 3); }
    if (G.withv && q == geo_pairs(st) - 1) { t.z = rel(0, kV); t.w = rel(1, kV); }
    else if (G.rows) { t.z = rel(0, qq - G.dl + 2); t.w = rel(1, qq - G.dl + 1); }
    else { t.z = rel(qq - G.dl, G.dl - qq + 2); t.w = rel(qq - G.dl, G.dl - qq + 3); }
    if (q >= geo_pairs(st)) { t.z = t.x; t.w = t.y | (int)0x80000000; }
    S.tab[e] = t;
  }
  if (me < kStates) S.info[me] = geo_info(me);
  const int max_steps = (int)min(Ar.step_budget > 0 ? Ar.step_budget : default_steps(n), 0x7ffffffeLL);
  const long long polls = poll_limit(m, n, Ar.rx);
  const long long rot_polls = Ar.stall == 1 ? Ar.stall_polls : polls;
  const long long word_polls = Ar.stall == 2 ? Ar.stall_polls : polls / 8;
  int steps = 0;  // of this warp, on the group at hand
  if (me == 0) S.far = kFar;
  for (;;) {
    __syncthreads();
    if (me == 0) {
      S.ticket = atomicAdd(ticket, 1);
      S.before = S.done = S.loader_done = 0;
    }
    __syncthreads();
    const int s = S.ticket;
    if (s >= groups) return;
    steps = 0;
    const int phase = s < F.g1 ? 1 : s < F.g1 + F.g2 ? 2 : 3;
    const int q0 = (s - (phase == 1 ? 0 : phase == 2 ? F.g1 : F.g1 + F.g2)) * kGroup;
    const int cnt = min(kGroup, (phase == 1 ? F.p1 : phase == 2 ? F.p2 : F.p3) - q0);
    // the first row of the window: two above the topmost first position
    int st0, p0 = 1;
    if (cnt > 0) first_op(F, n, phase, phase == 3 ? q0 : q0 + cnt - 1, st0, p0);
    const int base = max(1, p0 - 2);
    int *const word = words + s;
    const int *const prev = s > 0 ? word - 1 : nullptr;
    if (me < kRotWarps) {
      S.front[me] = 0;
      int least = kFar;
      for (int k = me * kSlots; k < min(cnt, (me + 1) * kSlots); k++) {
        int a, p;
        if (first_op(F, n, phase, q0 + k, a, p)) least = min(least, p);
      }
      S.least[me] = least;
    }
    if (me == 0) {
      S.loaded = S.flushed = base - 1;
      if (s == 0) S.before = kFar;
    }
    if (s == 0 && wid == 0) run_spike<FAST>(Ar);
    __syncthreads();
    if (wid < kRotWarps) rotate_chases<FAST, EXTRA>(Ar, S, F, phase, q0, max(cnt, 0), wid, max_steps, steps, rot_polls);
    else if (wid == kRotWarps) load_rows(Ar, S, F, base, prev, s == F.g1);
    else publish_rows<FAST>(Ar, S, F, base, prev, word, s == F.g1 - 1, word_polls, s == 0 ? Ar.stall : 0);
    __syncthreads();
    if (S.loaded == kAborted) return;
  }
}

template <bool FAST, bool EXTRA>
__global__ void __launch_bounds__(kThreads) k_chase(ChaseArgs Ar) {
  engine<FAST, EXTRA>(Ar);
}

}  // namespace

int chase_sync_ints(int m, int n) {
  const Phases F = phases_of(m, n);
  return 2 + F.g1 + F.g2 + F.g3;
}

// Blocks for a column.  About n / (3 kGroup) groups are in flight in phases 2
// and 3, up to n / (2 kGroup) at the end of phase 1; three more cover the
// hand-over between groups.  A block that holds the ticket of a later group
// keeps its SM from the application that runs beside the chase: at 4096, 67
// blocks 83.9 ms an overlapped update, 35 blocks 75.5, 24 blocks 76.3 (the
// chase alone 54.2, 54.3, 56).  (Measured at 4096 in the fast form only.)
int chase_blocks(int m, int n) {
  const Phases F = phases_of(m, n);
  return std::min(F.g1 + F.g2 + F.g3, n / (4 * kGroup) + 3);
}

namespace {

// Many independent factorizations: blocks (i, .) run items[i] (so that every
// item has a block in the first wave).
template <bool FAST, bool EXTRA>
__global__ void __launch_bounds__(kThreads) k_chase_batch(const ChaseArgs *__restrict__ items) {
  __shared__ ChaseArgs Ar;  // (in shared memory: a copy in registers halves the blocks an SM holds)
  if (threadIdx.x == 0) Ar = items[blockIdx.x];
  __syncthreads();
  if ((int)blockIdx.y >= Ar.blocks) return;
  engine<FAST, EXTRA>(Ar);
}

}  // namespace

cudaError_t launch_chase_batch(const ChaseArgs *d_items, int count, int max_blocks, int fast, bool extra,
                               cudaStream_t s) {
  if (count <= 0) return cudaSuccess;
  const dim3 grid(count, max_blocks);
  auto *const k = fast ? (extra ? k_chase_batch<true, true> : k_chase_batch<true, false>)
                       : (extra ? k_chase_batch<false, true> : k_chase_batch<false, false>);
  k<<<grid, kThreads, 0, s>>>(d_items);
  return cudaGetLastError();
}

// Failure injection: BDU_INJECT_STEP_BUDGET sets the step budget of a column
// whose caller set none, BDU_INJECT_CHASE_STALL and BDU_INJECT_CHASE_UNDONE
// withhold the first group's progress word (altogether; that it is done) and
// set the polls after which the waits for it give up.
cudaError_t launch_chase(const ChaseArgs &a0, cudaStream_t s) {
  ChaseArgs a = a0;
  const Injection inj = injection();
  if (a.step_budget == 0 && inj.site == BDU_INJECT_STEP_BUDGET) a.step_budget = inj.value;
  a.stall = inj.site == BDU_INJECT_CHASE_STALL ? 1 : inj.site == BDU_INJECT_CHASE_UNDONE ? 2 : 0;
  a.stall_polls = inj.value;
  a.blocks = a.engine == 1 ? 1 : chase_blocks(a.m, a.n);
  const cudaError_t e = cudaMemsetAsync(a.sync, 0, sizeof(int) * chase_sync_ints(a.m, a.n), s);
  if (e != cudaSuccess) return e;
  auto *const k = a.fast ? (a.rx > 0 ? k_chase<true, true> : k_chase<true, false>)
                         : (a.rx > 0 ? k_chase<false, true> : k_chase<false, false>);
  k<<<a.blocks, kThreads, 0, s>>>(a);
  return cudaGetLastError();
}

}  // namespace bdu
