// K3: application of the rotation stream to the columns of Q (left
// rotations, Q+ = Q * prod G^T) or P (right rotations, P+ = P * prod H)
// (Sec. 3.2, Eq. bidiagplus).
//
// Rows of Q and P are independent under column rotations, so each CTA owns a
// slab of R rows, keeps it in shared memory for the whole rank-1 column and
// writes it back once: every element is read and written once per column.
// The slab is stored column by column, so that an FP32 rotation reaches 4 rows
// of both of its columns with each 16-byte shared access.
// The rotations of one chase act on disjoint column pairs, so a chase is
// applied by all threads at once -- FP32: one rotation per thread, looping over
// the slab's rows; FP64: see apply_slab64 -- and consecutive chases are
// separated by a barrier; the next rotations are prefetched into registers
// while the current ones are applied.  The spike chain (m > n) is sequential and runs first, one thread
// per row.  R is chosen so that the grid fills whole waves of SMs.
//
// FP64: each pair update is c*x + s*y with separately rounded operations, the
// same operations a one-rotation-at-a-time evaluation performs.  FP32 (the
// mixed form): the generator's FP32 copies of (c, s) are applied with fused
// multiply-adds.
//
// The slab is indexed with the columns that the records name, so a record whose
// pair lies outside the matrix is skipped and reported (ERR_RANGE).
#include <algorithm>

#include "bdu_internal.cuh"

namespace bdu {
namespace {

constexpr int kThreads = 512;
constexpr int kPer = 5;  // rotations per thread per chase held in registers

// One FP64 rotation of a pair.
__device__ __forceinline__ void rot64(double c, double s, double &x, double &y) {
  const double xo = x, yo = y;
  x = __dadd_rn(__dmul_rn(c, xo), __dmul_rn(s, yo));
  y = __dadd_rn(__dmul_rn(-s, xo), __dmul_rn(c, yo));
}
// One FP32 rotation, as recorded.
struct Coef {
  float c, s;
  static __device__ __forceinline__ Coef load(const RotStream &st, int side, size_t i) {
    const float2 v = side == 0 ? st.Lf[i] : st.Rf[i];
    Coef k; k.c = v.x; k.s = v.y; return k;
  }
  static __device__ __forceinline__ Coef load_spike(const RotStream &st, int i) {
    const float2 v = st.Sf[i];
    Coef k; k.c = v.x; k.s = v.y; return k;
  }
  __device__ __forceinline__ void rot(float &x, float &y) const {
    const float xo = x, yo = y;
    x = fmaf(c, xo, s * yo);
    y = fmaf(c, yo, -s * xo);
  }
};

constexpr int kVec = 4;  // floats of a 16-byte vector of the tile
__device__ __forceinline__ void rot_vec(const Coef &k, float4 &x, float4 &y) {
  k.rot(x.x, y.x); k.rot(x.y, y.y); k.rot(x.z, y.z); k.rot(x.w, y.w);
}

// Shared-memory tile: column-major, column c's R rows at tile[c*csw ...],
// csw = kVec * (odd count of 16-byte vectors) >= R, so that the columns touched
// by a stride-3 chase fall in distinct 16-byte bank groups.
__device__ __forceinline__ void apply_slab32(float *__restrict__ X, int64_t ld, int nrow, int ncol, int R, int csw,
                                             const RotStream &st, int side, int with_spike, int slab, int *status) {
  extern __shared__ __align__(16) unsigned char raw[];
  float *tile = reinterpret_cast<float *>(raw);
  const int r0 = slab * R;
  const int rows = min(R, nrow - r0);
  if (rows <= 0) return;
  const int tid = threadIdx.x;
  const int32_t *Ca = side == 0 ? st.La : st.Ra;
  const int32_t *Cn = side == 0 ? st.Ln : st.Rn;
  const int cap = st.cap, ntask = st.T;
  const int nv = R / kVec;  // vectors per column

  for (int64_t q = tid; q < (int64_t)R * ncol; q += kThreads) {
    const int col = (int)(q / R), rr = (int)(q % R);
    tile[(size_t)col * csw + rr] = (rr < rows) ? X[(size_t)col * ld + r0 + rr] : 0.f;
  }
  __syncthreads();

  if (with_spike) {
    const int ns = st.Sn[0];
    if (tid < rows) {
      float *row = tile + tid;
      for (int e = 0; e < ns; e++) {
        const int a = st.Sa[e] - 1;  // 0-based first column of the pair
        Coef::load_spike(st, e).rot(row[(size_t)a * csw], row[(size_t)(a + 1) * csw]);
      }
    }
    __syncthreads();
  }

  // A record outside the factor is dropped before its chase's turn, beside the
  // barrier, and reported at the end: order 257 0.73 to 0.75 ms a side, 0.84
  // with a test and a report a rotation (0.72 unchecked).
  bool outside = false;
  auto drop = [&](int (&a)[kPer]) {
    int most = a[0];
#pragma unroll
    for (int k = 1; k < kPer; k++) most = max(most, a[k]);
    if (most < ncol - 1) return;
    outside = true;
#pragma unroll
    for (int k = 0; k < kPer; k++) a[k] = a[k] < ncol - 1 ? a[k] : -1;
  };
  // the rotations of the current chase owned by this thread, in registers
  Coef cf[kPer];
  int ca[kPer];
  int cnt = ntask > 0 ? Cn[0] : 0;
#pragma unroll
  for (int k = 0; k < kPer; k++) {
    const int e = tid + k * kThreads;
    ca[k] = -1;
    if (e < cnt) {
      cf[k] = Coef::load(st, side, (size_t)e);
      ca[k] = Ca[e] - 1;
    }
  }
  drop(ca);
  for (int t = 0; t < ntask; t++) {
    // prefetch chase t+1
    Coef nf[kPer];
    int na[kPer];
    const int ncnt = (t + 1 < ntask) ? Cn[t + 1] : 0;
    const size_t nbase = (size_t)(t + 1) * cap;
#pragma unroll
    for (int k = 0; k < kPer; k++) {
      const int e = tid + k * kThreads;
      na[k] = -1;
      if (e < ncnt) {
        nf[k] = Coef::load(st, side, nbase + e);
        na[k] = Ca[nbase + e] - 1;
      }
    }
    // apply chase t: each owned rotation to all rows of the slab, V rows per access
#pragma unroll
    for (int k = 0; k < kPer; k++) {
      if (ca[k] >= 0) {
        float4 *pa = reinterpret_cast<float4 *>(tile + (size_t)ca[k] * csw);
        float4 *pb = reinterpret_cast<float4 *>(tile + (size_t)(ca[k] + 1) * csw);
        for (int q = 0; q < nv; q++) {
          float4 x = pa[q], y = pb[q];
          rot_vec(cf[k], x, y);
          pa[q] = x;
          pb[q] = y;
        }
      }
    }
    // chases longer than the register-held part
    const int ccnt = Cn[t];
    for (int e = tid + kPer * kThreads; e < ccnt; e += kThreads) {
      const size_t i = (size_t)t * cap + e;
      const Coef k = Coef::load(st, side, i);
      const int a = Ca[i] - 1;
      if ((unsigned)a >= (unsigned)(ncol - 1)) {
        outside = true;
        continue;
      }
      float4 *pa = reinterpret_cast<float4 *>(tile + (size_t)a * csw);
      float4 *pb = reinterpret_cast<float4 *>(tile + (size_t)(a + 1) * csw);
      for (int q = 0; q < nv; q++) {
        float4 x = pa[q], y = pb[q];
        rot_vec(k, x, y);
        pa[q] = x;
        pb[q] = y;
      }
    }
    drop(na);
    __syncthreads();
#pragma unroll
    for (int k = 0; k < kPer; k++) {
      cf[k] = nf[k];
      ca[k] = na[k];
    }
  }

  if (outside && status) atomicOr(status, ERR_RANGE);
  for (int64_t q = tid; q < (int64_t)rows * ncol; q += kThreads) {
    const int col = (int)(q / rows), rr = (int)(q % rows);
    X[(size_t)col * ld + r0 + rr] = tile[(size_t)col * csw + rr];
  }
}

// FP64 body.  A slab of R rows in shared memory (column stride csw, odd), all
// chases applied one after another, a barrier between two.  Six FP64
// operations a rotation and row at two FP64 results a clock and SM bound it at
// large n, the chase's chain of latencies at small n:
//   * a work item is 16 rotations x some of the slab's rows, two lanes a
//     rotation (one forms x', the other y': three FP64 instructions, and half
//     the latency of six); items are dealt so that every SM sub-partition
//     gets the same number of rotations and rows (parts of the rows to
//     warps 4 apart), since on GB300 a warp's FP64 instruction holds its
//     sub-partition's FP64 unit for 64 cycles whatever the active lanes;
//     A warp without an item in a chase issues none of them.
//   * each warp runs through its items of all chases as one stream and loads
//     the coefficients kAhead items ahead of their use, the counts of 32
//     chases at a time.
// Per side and column, before (a rotation of both rows and columns a thread,
// coefficients one chase ahead) and now: order 64 0.61 -> 0.21 ms, 256 1.27 ->
// 0.54, 512 5.6 -> 4.0, 1024 15.7 -> 12.3, 4096 750 -> 670 (the FP64 units'
// floor at 4096 is 490 ms).  Any number of rows a slab may have (4096 columns:
// 7, in 4 waves of blocks, where pairs of rows allowed 6 in 5).
constexpr int kGroupRot = 16;  // rotations of an item
constexpr int kAhead = 3;

struct Item64 {
  double c, s;  // as the lane uses them: own column times c, the other times s
  int a;        // 1-based first column of the lane's pair, 0: none (as loaded: arithmetic here would wait for the load)
  bool last;    // the warp's last item of its chase
};
// A warp's stream of items: chase t, group g; counts of chases t0 .. t0 + 31
// in the lanes.
struct Stream64 {
  int t, g, t0, cnt, mine;
};

__device__ __forceinline__ void apply_slab64(double *__restrict__ X, int64_t ld, int nrow, int ncol, int R, int csw,
                                             const RotStream &st, int side, int with_spike, int slab, int *status) {
  extern __shared__ __align__(16) unsigned char raw[];
  double *tile = reinterpret_cast<double *>(raw);
  const int r0 = slab * R;
  const int rows = min(R, nrow - r0);
  if (rows <= 0) return;
  const int tid = threadIdx.x, nth = blockDim.x, lane = tid & 31, w = tid >> 5, nw = nth >> 5;
  const int32_t *__restrict__ Ca = side == 0 ? st.La : st.Ra;
  const int32_t *__restrict__ Cn = side == 0 ? st.Ln : st.Rn;
  const double *__restrict__ Cc = side == 0 ? st.Lc : st.Rc;
  const double *__restrict__ Cs = side == 0 ? st.Ls : st.Rs;
  const int ntask = st.T, cap = st.cap;

  for (int64_t q = tid; q < (int64_t)R * ncol; q += nth) {
    const int col = (int)(q / R), rr = (int)(q % R);
    tile[(size_t)col * csw + rr] = (rr < rows) ? X[(size_t)col * ld + r0 + rr] : 0.0;
  }
  __syncthreads();

  if (with_spike) {
    const int ns = st.Sn[0];
    if (tid < rows && ns > 0) {
      double *row = tile + tid;
      double c = st.Sc[0], s = st.Ss[0];
      int a = st.Sa[0] - 1;
      for (int e = 0; e < ns; e++) {
        const int en = min(e + 1, ns - 1);  // the next rotation, while this one is applied
        const double nc = st.Sc[en], nsn = st.Ss[en];
        const int na = st.Sa[en] - 1;
        rot64(c, s, row[(size_t)a * csw], row[(size_t)(a + 1) * csw]);
        c = nc; s = nsn; a = na;
      }
    }
    __syncthreads();
  }

  // This warp's share of a chase's groups: parts of the slab's rows go to
  // warps 4 apart (the same sub-partition), the groups to the rest.
  const int q4 = nw >= 4 ? 4 : 1;              // nw: 1, or a multiple of 4
  const int upper = nw / q4;                   // warps of a sub-partition
  int parts = 1;
  while (parts * 2 <= upper && parts * 2 <= rows && ncol / (2 * kGroupRot) * parts < 2 * nw) parts *= 2;
  const int part = (w / q4) % parts;
  const int ra = rows * part / parts, rb = rows * (part + 1) / parts;
  const int g0 = w % q4 + q4 * (w / (q4 * parts)), gstep = nw / parts;
  const int h = lane & 1;  // 0: x', 1: y'

  Stream64 S{-1, 0, -32, 0, 0};
  // counts one batch ahead
  auto counts = [&](int t0) { return t0 + lane < ntask ? Cn[t0 + lane] : 0; };
  S.mine = 0;
  int next_mine = counts(0);
  auto next_item = [&]() {
    Item64 it;
    it.a = 0;
    it.last = true;
    it.c = it.s = 0.0;
    if (S.t >= ntask) return it;
    const bool more = S.t >= 0 && (S.g + gstep) * kGroupRot < S.cnt;
    if (more) {
      S.g += gstep;
    } else {
      S.t++;
      if (S.t >= ntask) return it;
      if (S.t - S.t0 >= 32) {
        S.t0 += 32;
        S.mine = next_mine;
        next_mine = counts(S.t0 + 32);
      }
      S.cnt = __shfl_sync(0xffffffffu, S.mine, S.t - S.t0);
      S.g = g0;
    }
    const int e = S.g * kGroupRot + (lane >> 1);
    if (e < S.cnt) {
      const size_t i = (size_t)S.t * cap + e;
      it.a = __ldg(Ca + i);
      it.c = __ldg(Cc + i);
      it.s = __ldg(Cs + i);
    }
    it.last = (S.g + gstep) * kGroupRot >= S.cnt;
    return it;
  };
  Item64 ring[kAhead];
#pragma unroll
  for (int k = 0; k < kAhead; k++) ring[k] = next_item();
  // (reported once, at the end: a branch an item costs 4 % of a batch of 16
  // FP64 sessions of 64..1024, 170 against 163 ms)
  int most = 0;  // greatest column named
  for (int t = 0; t < ntask;) {
#pragma unroll
    for (int k = 0; k < kAhead; k++) {  // (unrolled: the ring stays in registers)
      if (t >= ntask) break;
      const Item64 it = ring[k];
      ring[k] = next_item();
      // two rows at a time; both lanes of a pair have read before either writes
      const bool in = it.a > 0 && it.a < ncol;
      most = max(most, it.a);
      const int a = in ? it.a - 1 : 0;
      const double s = h ? -it.s : it.s;
      double *const own = tile + (size_t)(a + h) * csw, *const oth = tile + (size_t)(a + 1 - h) * csw;
      // (an item past the chase's last rotation costs no FP64 instruction)
      for (int r = __any_sync(0xffffffffu, in) ? ra : rb; r < rb; r += 2) {
        const bool two = r + 1 < rb;
        const double p0 = own[r], o0 = oth[r];
        const double p1 = two ? own[r + 1] : 0.0, o1 = two ? oth[r + 1] : 0.0;
        __syncwarp();
        const double v0 = __dadd_rn(__dmul_rn(it.c, p0), __dmul_rn(s, o0));
        if (in) own[r] = v0;
        if (two) {
          const double v1 = __dadd_rn(__dmul_rn(it.c, p1), __dmul_rn(s, o1));
          if (in) own[r + 1] = v1;
        }
      }
      if (it.last) {
        __syncthreads();
        t++;
      }
    }
  }

  if (most >= ncol && status) atomicOr(status, ERR_RANGE);
  for (int64_t q = tid; q < (int64_t)rows * ncol; q += nth) {
    const int col = (int)(q / rows), rr = (int)(q % rows);
    X[(size_t)col * ld + r0 + rr] = tile[(size_t)col * csw + rr];
  }
}

// gate (may be null): a device error word written by an earlier kernel on
// the stream; when it is nonzero the kernel leaves X untouched.
template <typename T>
__global__ void __launch_bounds__(kThreads) k_apply_slab(T *__restrict__ X, int64_t ld, int nrow,
                                                         int ncol, int R, int csw, RotStream st,
                                                         int side, int with_spike, int *status, const int *gate) {
  if (gate && *(volatile const int *)gate) return;
  if constexpr (sizeof(T) == 8) apply_slab64(X, ld, nrow, ncol, R, csw, st, side, with_spike, blockIdx.x, status);
  else apply_slab32(X, ld, nrow, ncol, R, csw, st, side, with_spike, blockIdx.x, status);
}

// Many matrices of uneven sizes in one launch: block b works on the slab
// b - first[i] of item i, where first[] is the prefix sum of the items' slab
// counts (found by binary search).
template <typename T>
__global__ void __launch_bounds__(kThreads) k_apply_batch(const ApplyItem *__restrict__ items,
                                                          const int *__restrict__ first, int count) {
  const int b = blockIdx.x;
  int lo = 0, hi = count - 1;
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (first[mid] <= b) lo = mid;
    else hi = mid - 1;
  }
  const ApplyItem it = items[lo];
  if constexpr (sizeof(T) == 8)
    apply_slab64((T *)it.X, it.ld, it.nrow, it.ncol, it.R, it.csw, it.st, it.side, it.with_spike, b - first[lo],
                 it.status);
  else
    apply_slab32((T *)it.X, it.ld, it.nrow, it.ncol, it.R, it.csw, it.st, it.side, it.with_spike, b - first[lo],
                 it.status);
}

}  // namespace

// Column stride of an FP64 slab of R rows: odd (consecutive columns in distinct
// banks) where that fits in smem_cap bytes, 0 when the slab does not fit.
static int stride64(int R, int ncol, size_t smem_cap) {
  if (sizeof(double) * (size_t)(R | 1) * ncol <= smem_cap) return R | 1;
  return sizeof(double) * (size_t)R * ncol <= smem_cap ? R : 0;
}
// Threads of an FP64 slab's block: as many warps as the longest chases (a
// rotation every second column) have items for, 4 to 16.
static int threads64(int ncol, int R) {
  const int items = (ncol / 2 + kGroupRot - 1) / kGroupRot * R;
  return items <= 4 ? 128 : items <= 12 ? 256 : 512;
}

// Rows per slab and column stride for an ncol-wide matrix within smem_cap
// bytes of shared memory: as many rows as fit, at most `most` (and the least
// there can be if that is fewer).
void apply_geometry(int precision, int ncol, size_t smem_cap, int most, int *R, int *csw) {
  const int esz = (precision == BDU_FP64) ? 8 : 4;
  const int V = 16 / esz;
  if (precision == BDU_FP64) {
    *R = *csw = 0;
    for (int r = 2; r <= std::max(most, 2); r++) {
      const int c = stride64(r, ncol, smem_cap);
      if (c == 0) break;
      *R = r; *csw = c;
    }
    return;
  }
  int bestR = 0, bestc = 0;
  for (int r = V; r <= std::max(most, V); r += V) {
    int w = r / V;
    if ((w & 1) == 0) w++;
    const int c = w * V;
    if ((size_t)esz * c * ncol > smem_cap) break;
    bestR = r; bestc = c;
  }
  *R = bestR; *csw = bestc;
}

cudaError_t launch_apply_batch(int precision, const ApplyItem *d_items, const int *d_first, int count,
                               int total_slabs, size_t smem, cudaStream_t s) {
  if (count <= 0 || total_slabs <= 0) return cudaSuccess;
  cudaError_t e;
  if (precision == BDU_FP64) {
    e = cudaFuncSetAttribute(k_apply_batch<double>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    k_apply_batch<double><<<total_slabs, kThreads, smem, s>>>(d_items, d_first, count);
  } else {
    e = cudaFuncSetAttribute(k_apply_batch<float>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    k_apply_batch<float><<<total_slabs, kThreads, smem, s>>>(d_items, d_first, count);
  }
  return cudaGetLastError();
}

cudaError_t launch_apply(int precision, void *X, int64_t ld, int nrow, int ncol,
                         const RotStream &st, int side, bool with_spike, cudaStream_t s, int *status,
                         int sm_reserve, bool desc_ready, int variant, const int *gate) {
  if (precision == BDU_MIXED && (st.Lf == nullptr || st.Rf == nullptr)) return cudaErrorInvalidValue;
  if (precision == BDU_MIXED && variant == 0 && ncol >= kBlockedFrom && st.tc_ws) variant = 128;
  if (precision == BDU_MIXED && is_tc_variant(variant))
    return launch_apply_tc((float *)X, ld, nrow, ncol, st, side, with_spike, status, desc_ready, variant, st.tc_ws,
                           st.tc_ws_bytes, s);
  if (precision == BDU_MIXED && variant != kSlabVariant) {
    cudaError_t e = launch_apply_reg((float *)X, ld, nrow, ncol, st, side, with_spike, status, sm_reserve,
                                     desc_ready, variant, s);
    if (e != cudaErrorNotSupported || variant != 0) return e;
    // no register layout covers the shape: the blocked tensor-core apply
    e = launch_apply_tc((float *)X, ld, nrow, ncol, st, side, with_spike, status, desc_ready, 128, st.tc_ws,
                        st.tc_ws_bytes, s);
    if (e != cudaErrorNotSupported) return e;
    cudaGetLastError();
  }
  int dev = 0, optin = 0, sms = 1;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  const int esz = (precision == BDU_FP64) ? 8 : 4;
  const int V = 16 / esz;
  // Rows per block.  FP32: a multiple of V, the column stride an odd number of
  // 16-byte vectors; FP64: 2 to 64.  Pick the R that minimizes waves x (R +
  // overhead).  (FP64 form: a positive variant fixes R instead)
  int best_R = 0, best_csw = 0;
  double best_cost = 1e300;
  const bool fixed = precision == BDU_FP64 && variant > 0;
  if (fixed && (variant < 2 || variant > 64)) return cudaErrorNotSupported;
  for (int R = 2; R <= 64; R++) {
    int csw = 0;
    if (precision == BDU_FP64) {
      csw = stride64(R, ncol, (size_t)optin);
      if (csw == 0) break;
    } else {
      if (R % V) continue;
      const int w = (R / V) | 1;
      csw = w * V;
      if ((size_t)esz * csw * ncol > (size_t)optin) break;
    }
    const int ctas = (nrow + R - 1) / R;
    const int waves = (ctas + sms - 1) / sms;
    const double cost = fixed ? (R == variant ? 0.0 : 1e299) : (double)waves * (R + 4);
    if (cost <= best_cost) { best_cost = cost; best_R = R; best_csw = csw; }
  }
  if (fixed && best_R != variant) return cudaErrorNotSupported;
  if (best_R == 0) return cudaErrorNotSupported;  // a single vector column does not fit
  const size_t smem = (size_t)esz * best_csw * ncol;
  const int blocks = (nrow + best_R - 1) / best_R;
  cudaError_t e;
  if (precision == BDU_FP64) {
    e = cudaFuncSetAttribute(k_apply_slab<double>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    k_apply_slab<double><<<blocks, threads64(ncol, best_R), smem, s>>>((double *)X, ld, nrow, ncol, best_R, best_csw, st,
                                                        side, with_spike ? 1 : 0, status, gate);
  } else {
    e = cudaFuncSetAttribute(k_apply_slab<float>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    k_apply_slab<float><<<blocks, kThreads, smem, s>>>((float *)X, ld, nrow, ncol, best_R, best_csw, st,
                                                       side, with_spike ? 1 : 0, status, gate);
  }
  return cudaGetLastError();
}

}  // namespace bdu
