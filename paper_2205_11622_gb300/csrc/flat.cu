// Row sums over windows of consecutive nonzeros, for the expressions whose
// output row is a weighted sum of gathered rows:
//
//   kSum       out(r,:) = sum_p vals[p] X(crd[p],:)
//   kSampled   out(r,:) = sum_p vals[p] <C(r,:), D(crd[p],:)> X(crd[p],:)
//              (fused <SDDMM,SpMM>, Fig. 2d: the scalar of each stored (i,j)
//              is formed and used at once)
//
// The nonzeros, not the rows, are split: lane group g of a warp (GS lanes, one
// gathered row at a time) owns a window of `win` consecutive nonzeros,
// whatever rows they belong to, so that every group has about the same work
// on any distribution of row lengths, in a single queue that needs no counter.
// k_flat_rows first notes the row of each window's first nonzero and zeroes
// the rows without nonzeros.  A row whose nonzeros lie in one window is
// written once.  One that spans windows leaves a tail piece in the window
// where it starts and a head piece in each later one; k_flat_combine adds
// tail and heads in window order.  Windows depend on sizes only, so results
// are the same on every run.
//
// What bounds it: waiting for the gathered rows, which come out of L2 (a group
// reads one or two whole rows per nonzero).  With every warp's loads in flight
// all the time this GPU gathers 21 TB/s; sums of 16M and 20M rows of 128 and 64
// reach 14, <SDDMM,SpMM> of 2M nonzeros at 64/64 9.5, sums of 2.4M rows of 32
// and <SDDMM,SpMM> of 0.6M at 100/48 4 to 6 (windows of few nonzeros, whose
// starts and ends are a larger part).  An ncu capture of the 64/64 call: 13
// warps on an SM, 6 of them waiting for loads for each that issues, issue slots
// 32 % used, L1 57 %, L2 40 %; of the sums of rows of 32: 28 warps, 53 %, 62 %, 21 %.
#include "flat.cuh"
#include "launch.h"

namespace slnr {
namespace {

using flat::Row;
using flat::u64;

enum FlatMode { kSum = 0, kSampled = 1 };

constexpr int kFlatThreads = 128;
constexpr int kFlatSms = 152;  // the window sizes are for this many SMs (sizes only: no device is asked)
constexpr int kStage = 64;  // nonzeros of a warp staged in shared memory at a time (two per lane)

// Rows in flight per lane group, and resident CTAs per SM (registers) the
// kernels are compiled for.  Measured: sum of 20M rows of 64 with 2 rows and 9
// CTAs 385 us, 4 and 8 435; <SDDMM,SpMM> (two gathered rows per nonzero), 100k
// rows at 64/64 and 3k rows, with 4 and 4 120 and 25.6 us, 2 and 6 124 and 27.
constexpr int kFlatU = 2, kFlatCtas = 9;
constexpr int kFlatU2 = 4, kFlatCtas2 = 4;
template <int NCH, int MODE>
constexpr int flat_u() {
  return (MODE == kSum ? kFlatU : kFlatU2) / NCH > 0 ? (MODE == kSum ? kFlatU : kFlatU2) / NCH : 1;
}
template <int NCH, int MODE>
constexpr int flat_ctas() {
  return NCH == 1 ? (MODE == kSum ? kFlatCtas : kFlatCtas2) : NCH == 2 ? 4 : 2;
}

// Rows of pos that a lane holds: a group looks at 8 rows a step (4 where it is
// one lane), or windows of short rows wait for pos again and again
// (<SDDMM,SpMM> 16/16 on R-MAT graphs of 30k rows, degrees 8 and 32: one row a
// lane 43 and 50 us, four 37 and 44; row kernel 31 and 41).
template <int GS>
constexpr int flat_look() {
  return GS >= 8 ? 1 : GS == 4 ? 2 : 4;
}

// Largest r in [lo, n) with pos[r] <= p, given lo < n and pos[lo] <= p; one
// thread.  The row is near lo as a rule: kProbe loads in flight first double
// the distance until a row lies past p, then cut the rows that are left by
// kProbe + 1.  Ends, with lo <= r < n, whatever pos holds.  A binary search of
// all rows left took 23 dependent loads per nonzero where an R-MAT graph is
// sparse: sums of 1.6M rows of 16, 400k rows 138 us, now 73; of 4M rows of 128,
// 1M rows 320 | 270.  Out of line, as its registers otherwise cost every window
// (uniform, 6.4M rows of 128: 403 us inline, 382).
constexpr int kProbe = 4;
__device__ __noinline__ int row_of(const int32_t* __restrict__ pos, int lo, int n, int p) {
  int hi = n - 1;
  for (int64_t d = 1; lo < hi; d <<= kProbe) {
    int k = 0;
    bool le[kProbe];
#pragma unroll
    for (int j = 0; j < kProbe; ++j) le[j] = lo + (d << j) < n && __ldg(pos + lo + (d << j)) <= p;
#pragma unroll
    for (int j = 0; j < kProbe; ++j) k += k == j && le[j];
    if (k < kProbe && lo + (d << k) <= hi) hi = (int)(lo + (d << k)) - 1;
    if (k > 0) lo += (int)(d << (k - 1));
    if (k < kProbe) break;
  }
  while (lo < hi) {
    const int step = (hi - lo + kProbe) / (kProbe + 1);
    int k = 0;
    bool le[kProbe];
#pragma unroll
    for (int j = 0; j < kProbe; ++j)
      le[j] = lo + (int64_t)(j + 1) * step <= hi && __ldg(pos + lo + (j + 1) * step) <= p;
#pragma unroll
    for (int j = 0; j < kProbe; ++j) k += k == j && le[j];
    lo += k * step;
    if (k < kProbe && (int64_t)lo + step <= hi) hi = lo + step - 1;
  }
  return lo;
}

struct FlatArgs {
  WsHeader* hdr;
  int nrows;
  int nnz;
  int win;     // nonzeros per window: a multiple of the group's share of a stage
  int nw;      // windows
  const int32_t* pos;
  const int32_t* crd;
  const float* vals;
  const float* X;
  const float* D;   // kSampled
  const float* C;   // kSampled
  int W;            // width of X and out
  int L;            // kSampled: width of C and D
  float* out;
  int* first;       // [nw] row of window w's first nonzero
  int* tail_row;    // [nw] row whose first piece ends window w and goes on, or -1
  float* head;      // [nw x W]
  float* tail;      // [nw x W]
};

// Before the windows: row r, lane r % 32 of its warp.  Row r holds the first
// nonzero of the windows w with pos[r] <= w win < pos[r+1]; rows without
// nonzeros are zero in out.
constexpr int kRowsThreads = 256;

__global__ void __launch_bounds__(kRowsThreads) k_flat_rows(const FlatArgs a) {
  constexpr unsigned FULL = 0xffffffffu;
  const int lane = threadIdx.x & 31;
  const int64_t r0 = ((int64_t)blockIdx.x * kRowsThreads + threadIdx.x) - lane, r = r0 + lane;
  flat::grid_launch();
  if (blockIdx.x == 0 && threadIdx.x == 0 && a.hdr != nullptr) a.hdr->error = 0;
  const bool in = r < a.nrows;
  const int p0 = in ? __ldg(a.pos + r) : 0, p1 = in ? __ldg(a.pos + r + 1) : 0;
  int w0 = 0, w1 = 0;
  if (p0 < p1) {
    w0 = (int)(((unsigned)p0 + (unsigned)a.win - 1u) / (unsigned)a.win);
    w1 = (int)(((unsigned)p1 + (unsigned)a.win - 1u) / (unsigned)a.win);
  }
  const bool many = w1 - w0 > 4;
  if (!many)
    for (int w = w0; w < w1; ++w) a.first[w] = (int)r;
  for (unsigned m = __ballot_sync(FULL, many); m != 0; m &= m - 1) {  // a long row: the whole warp
    const int b = __ffs(m) - 1, lo = __shfl_sync(FULL, w0, b), hi = __shfl_sync(FULL, w1, b);
    for (int w = lo + lane; w < hi; w += 32) a.first[w] = (int)r0 + b;
  }
  flat::zero_rows(a.out + r0 * a.W, a.W, __ballot_sync(FULL, in && p0 == p1), lane);
}

// One warp's staged nonzeros: entry i belongs to window i / NS of the warp.
struct FlatStage {
  int2 cv[kStage];  // coordinate, value
  int row[kStage];  // the row that starts at the entry, or -1
};

// This lane's places in the call's matrices.
template <int GS, int NCH, int MODE, int KIND>
struct FlatPtrs {
  using Ptr = flat::RowPtr<GS, NCH, KIND>;
  Ptr x, d, c, out;
  __device__ __forceinline__ FlatPtrs(const FlatArgs& a, int gl)
      : x(a.X, a.W, gl), d(a.D, a.L, gl), c(a.C, a.L, gl), out(a.out, a.W, gl) {}
};

// U nonzeros of each window of the warp, entries e0 .. e0 + U - 1 of this
// lane's group: the U gathered rows are in flight together, then summed in
// order.  any: some window of the warp has a row starting among them (bits
// 0 .. U - 1 of `starts` are this window's), or fewer than U nonzeros left
// (`live`); then the row so far is written where the next one begins.
template <int GS, int NCH, int MODE, int KIND, int U>
__device__ __forceinline__ void flat_batch(const FlatPtrs<GS, NCH, MODE, KIND>& m, const FlatStage& st, int e0,
                                           bool any, unsigned starts, int live, uint64_t pol, Row<GS, NCH, KIND>& acc,
                                           Row<GS, NCH, KIND>& c, const char*& dst, int& cur) {
  using R = Row<GS, NCH, KIND>;
  uint32_t crd[U];
  float val[U];
  if constexpr (U % 2 == 0) {
#pragma unroll
    for (int u = 0; u < U; u += 2) {
      const int4 q = *reinterpret_cast<const int4*>(st.cv + e0 + u);
      crd[u] = (uint32_t)q.x;
      val[u] = __int_as_float(q.y);
      crd[u + 1] = (uint32_t)q.z;
      val[u + 1] = __int_as_float(q.w);
    }
  } else {
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int2 q = st.cv[e0 + u];
      crd[u] = (uint32_t)q.x;
      val[u] = __int_as_float(q.y);
    }
  }
  R x[U], d[MODE == kSum ? 1 : U];
#pragma unroll
  for (int u = 0; u < U; ++u) {
    if constexpr (MODE != kSum) d[u].load(m.d, crd[u]);
    x[u].load(m.x, crd[u]);
  }
  if (!any) {  // warp-uniform
    if constexpr (MODE == kSampled) {  // the dot products of the batch side by side
      float y[U];
#pragma unroll
      for (int u = 0; u < U; ++u) y[u] = R::dot_part(m.d, c, d[u]);
#pragma unroll
      for (int o = GS / 2; o > 0; o >>= 1)
#pragma unroll
        for (int u = 0; u < U; ++u) y[u] += __shfl_xor_sync(0xffffffffu, y[u], o);
#pragma unroll
      for (int u = 0; u < U; ++u) val[u] *= y[u];
    }
#pragma unroll
    for (int u = 0; u < U; ++u) {
      acc.fma(flat::pack2(val[u]), x[u]);
    }
    return;
  }
  starts &= (1u << U) - 1u;
  R cn;  // kSampled: C's row of the first row that starts here, in flight with the others
  if constexpr (MODE == kSampled) {
    if (starts != 0) cn.load(m.c, (uint32_t)st.row[e0 + __ffs(starts) - 1]);
    if (!__any_sync(0xffffffffu, (starts & (starts - 1)) != 0 || live < U)) {
      // at most one row starts in each window: its nonzeros before and after
      // that are added apart, with one write between, and the dot products
      // stay side by side
      const int f = starts != 0 ? __ffs(starts) - 1 : U;
      float y[U];
#pragma unroll
      for (int u = 0; u < U; ++u) y[u] = u < f ? R::dot_part(m.d, c, d[u]) : R::dot_part(m.d, cn, d[u]);
#pragma unroll
      for (int o = GS / 2; o > 0; o >>= 1)
#pragma unroll
        for (int u = 0; u < U; ++u) y[u] += __shfl_xor_sync(0xffffffffu, y[u], o);
#pragma unroll
      for (int u = 0; u < U; ++u) {
        val[u] *= y[u];
        if (u < f) acc.fma(flat::pack2(val[u]), x[u]);
      }
      if (f < U) {
        if (dst != nullptr) acc.store_once(m.out, dst, pol);
        cur = st.row[e0 + f];
        dst = m.out.row((uint32_t)cur);
        acc.zero();
        c = cn;
#pragma unroll
        for (int u = 0; u < U; ++u)
          if (u >= f) acc.fma(flat::pack2(val[u]), x[u]);
      }
      return;
    }
  }
  const unsigned first = starts & (0u - starts);
#pragma unroll
  for (int u = 0; u < U; ++u) {
    if (starts >> u & 1) {
      if (dst != nullptr) acc.store_once(m.out, dst, pol);
      cur = st.row[e0 + u];
      dst = m.out.row((uint32_t)cur);
      acc.zero();
      if constexpr (MODE == kSampled) {
        if (first == 1u << u) c = cn; else c.load(m.c, (uint32_t)cur);
      }
    }
    float v = val[u];
    if constexpr (MODE == kSampled) v *= group_sum<GS>(R::dot_part(m.d, c, d[u]));
    if (u < live) acc.fma(flat::pack2(v), x[u]);
  }
}

template <int GS, int NCH, int MODE, int KIND>
__global__ void __launch_bounds__(kFlatThreads, flat_ctas<NCH, MODE>()) k_flat(const FlatArgs a) {
  using R = Row<GS, NCH, KIND>;
  constexpr int GPW = 32 / GS;      // groups (windows) per warp
  constexpr int NS = kStage / GPW;  // nonzeros of a window per stage
  constexpr int U0 = flat_u<NCH, MODE>();
  constexpr int U = NS < U0 ? NS : U0;
  constexpr int NB = flat_look<GS>();
  constexpr unsigned FULL = 0xffffffffu;
  static_assert(NS % U == 0 && NS == 2 * GS, "batches tile a stage");
  __shared__ __align__(16) FlatStage stage[kFlatThreads / 32];
  const int lane = threadIdx.x & 31, g = lane / GS, gl = lane % GS;
  const unsigned gmask = GS == 32 ? FULL : ((1u << (GS & 31)) - 1u) << (g * GS);
  const int64_t warp = ((int64_t)blockIdx.x * kFlatThreads + threadIdx.x) >> 5;
  const int64_t span = (int64_t)GPW * a.win, s0 = warp * span;
  FlatStage& st = stage[threadIdx.x >> 5];
  const uint64_t pol = flat::first_out();
  const FlatPtrs<GS, NCH, MODE, KIND> m(a, gl);
  // this lane's two entries of a stage: window i / NS, nonzero i % NS; loaded one stage ahead
  int ncrd[2];
  float nval[2];
  auto fetch = [&](int s) {
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const int i = lane + 32 * h;
      const int64_t q = s0 + (i / NS * a.win + i % NS + s);
      const bool ok = s < a.win && q < a.nnz;
      ncrd[h] = ok ? flat::ld_once(a.crd + q, pol) : 0;
      nval[h] = ok ? flat::ld_once(a.vals + q, pol) : 0.f;
    }
  };
  fetch(0);
  flat::grid_wait();  // k_flat_rows has written `first`
  flat::grid_launch();
  if (s0 >= a.nnz) return;  // warp-uniform
  const int64_t w = warp * GPW + g;
  int p = (int)(w * a.win < a.nnz ? w * a.win : a.nnz);  // first nonzero of the window's stage
  const int p1 = (int)((int64_t)p + a.win < a.nnz ? p + a.win : a.nnz);
  int rnext = p < p1 ? a.first[w] : a.nrows;  // rows before it start before nonzero p
  // pos of rows rnext + NB gl, ..., loaded ahead: NB rows a lane and the one after
  int b[NB + 1];
  auto peek = [&]() {
#pragma unroll
    for (int j = 0; j <= NB; ++j) {
      const unsigned r = item(rnext, NB * gl + j);
      b[j] = r < (unsigned)a.nrows ? __ldg(a.pos + r) : INT_MAX;
    }
  };
  peek();
  int cur = -1;               // the row being summed
  const char* dst = nullptr;  // where its piece goes
  R acc, c;                   // c: C's row of `cur` (kSampled)
  acc.zero();
  if constexpr (MODE == kSampled) c.load(m.c, (uint32_t)(rnext < a.nrows ? rnext : 0));
  if (__shfl_sync(FULL, b[0], g * GS) < p) {  // the window starts inside row rnext
    cur = rnext;
    dst = typename R::Ptr(a.head, a.W, gl).row((uint32_t)w);
  }
#pragma unroll 1
  for (int s = 0; s < a.win; s += NS) {
    if (s0 + s >= a.nnz) break;  // warp-uniform: the first group has the earliest window
    __syncwarp();
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      st.cv[lane + 32 * h] = make_int2(ncrd[h], __float_as_int(nval[h]));
      st.row[lane + 32 * h] = -1;
    }
    __syncwarp();
    fetch(s + NS);
    // mark the rows that start in [p, pe): NB GS rows of pos per group and step
    const int pe = step_end(p, NS, p1);
    bool more = p < pe;
    do {
      int rows = 0;  // of this lane that start before pe
      bool mark = false;
#pragma unroll
      for (int j = 0; j < NB; ++j) {
        const bool in = more && b[j] < pe, full = in && b[j + 1] > b[j] && b[j] >= p;
        if (full) st.row[g * NS + b[j] - p] = rnext + NB * gl + j;
        rows += in;
        mark |= full;
      }
      const unsigned marked = __ballot_sync(FULL, mark) & gmask;
      if constexpr (NB == 1) {
        rows = __popc(__ballot_sync(FULL, rows != 0) & gmask);
      } else {
#pragma unroll
        for (int o = GS / 2; o > 0; o >>= 1) rows += __shfl_xor_sync(FULL, rows, o);
      }
      rnext += rows;
      more = more && rows == NB * GS;
      if (more && marked == 0 && rnext < a.nrows) {  // empty rows: on to the row with the next nonzero
        rnext = row_of(a.pos, rnext, a.nrows, __ldg(a.pos + rnext));  // never back: every step passes a row
      }
      if (rows != 0) peek();
    } while (__any_sync(FULL, more));
    __syncwarp();
    const unsigned long long marks = (unsigned long long)__ballot_sync(FULL, st.row[lane] >= 0) |
                                     (unsigned long long)__ballot_sync(FULL, st.row[lane + 32] >= 0) << 32;
    // rows that start in this window, and in any window of the warp, by nonzero of the stage
    const unsigned long long mine = marks >> (g * NS);
    unsigned long long any = marks;
#pragma unroll
    for (int k = kStage / 2; k >= NS; k >>= 1) any |= any >> k;
    if (s0 + span > a.nnz) any = ~0ull;  // a window of the warp may end early
    const int live = pe - p;
#pragma unroll 1
    for (int u0 = 0; u0 < NS; u0 += U) {
      flat_batch<GS, NCH, MODE, KIND, U>(m, st, g * NS + u0, (any >> u0 & ((1u << U) - 1u)) != 0,
                                         (unsigned)(mine >> u0), live - u0, pol, acc, c, dst, cur);
    }
    p = pe;
  }
  if (p1 <= w * a.win) return;  // a window past the end
  const bool more = __ldg(a.pos + cur + 1) > p1;
  const bool head = dst == typename R::Ptr(a.head, a.W, gl).row((uint32_t)w);
  acc.store_once(m.out, more && !head ? typename R::Ptr(a.tail, a.W, gl).row((uint32_t)w) : dst, pol);
  if (gl == 0) a.tail_row[w] = more && !head ? cur : -1;
}

// Rows that span windows: out(r,:) = tail of the window where r starts + the
// heads of the windows after it up to r's last nonzero, in that order.  A CTA
// looks at four windows a lane group (at most one a thread), so that wide rows
// are not one group's chain (<SDDMM,SpMM> 30k rows 100/48: 78 us with 256
// windows, 72 with 64; 3k 64/64 24.3 | 22.6); rows of more than kLongRow heads
// are summed by the whole CTA (lane groups take heads g, g + G, ... in order,
// then a fixed pairwise tree), the others by a lane group each.
constexpr int kCombineThreads = 256;
template <int GS>
constexpr int combine_windows() {
  return 4 * (kCombineThreads / GS) < kCombineThreads ? 4 * (kCombineThreads / GS) : kCombineThreads;
}
constexpr int kLongRow = 32;

template <int GS, int NCH, int KIND>
__global__ void __launch_bounds__(kCombineThreads) k_flat_combine(FlatArgs a) {
  using R = Row<GS, NCH, KIND>;
  constexpr int G = kCombineThreads / GS;  // lane groups of the CTA
  constexpr int N = combine_windows<GS>();
  __shared__ int2 item[N];  // {window, heads}: short rows from the front, long ones from the back
  __shared__ int nshort, nlong;
  __shared__ u64 red[kCombineThreads * R::P];
  const int tid = threadIdx.x, g = tid / GS, gl = tid % GS;
  const typename R::Ptr out(a.out, a.W, gl), heads(a.head, a.W, gl), tails(a.tail, a.W, gl);
  if (tid == 0) nshort = nlong = 0;
  flat::grid_wait();  // k_flat's pieces
  __syncthreads();
  {
    const int64_t w = (int64_t)blockIdx.x * N + tid;
    const int r = tid < N && w < a.nw ? a.tail_row[w] : -1;
    if (r >= 0) {
      const int n = (int)((__ldg(a.pos + r + 1) - 1) / a.win - w);
      const int at = n > kLongRow ? N - 1 - atomicAdd(&nlong, 1) : atomicAdd(&nshort, 1);
      item[at] = make_int2((int)w, n);
    }
  }
  __syncthreads();
  const int ns = nshort, nl = nlong;
  for (int i = 0; i < nl; ++i) {
    const int2 it = item[N - 1 - i];
    const uint32_t h = (uint32_t)it.x + 1;  // the first head
    R acc;
    acc.zero();
    if (g == 0) acc.load_written(tails, (uint32_t)it.x);
    int k = g;
    for (; k + 3 * G < it.y; k += 4 * G) {
      R x[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) x[u].load_written(heads, h + k + u * G);
#pragma unroll
      for (int u = 0; u < 4; ++u) acc.add(x[u]);
    }
    for (; k < it.y; k += G) {
      R x;
      x.load_written(heads, h + k);
      acc.add(x);
    }
#pragma unroll
    for (int q = 0; q < R::P; ++q) red[q * kCombineThreads + tid] = acc.v[q];
    __syncthreads();
    for (int half = G / 2; half > 0; half >>= 1) {
      if (g < half)
#pragma unroll
        for (int q = 0; q < R::P; ++q)
          red[q * kCombineThreads + tid] =
              flat::add2(red[q * kCombineThreads + tid], red[q * kCombineThreads + tid + half * GS]);
      __syncthreads();
    }
    if (g == 0) {
#pragma unroll
      for (int q = 0; q < R::P; ++q) acc.v[q] = red[q * kCombineThreads + tid];
      acc.store(out, out.row((uint32_t)a.tail_row[it.x]));
    }
    __syncthreads();
  }
  for (int i = g; i < ns; i += G) {
    const int2 it = item[i];
    const uint32_t h = (uint32_t)it.x + 1;  // the first head
    R acc;
    acc.load_written(tails, (uint32_t)it.x);
    int k = 0;
    for (; k + 4 <= it.y; k += 4) {
      R x[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) x[u].load_written(heads, h + k + u);
#pragma unroll
      for (int u = 0; u < 4; ++u) acc.add(x[u]);
    }
    for (; k < it.y; ++k) {
      R x;
      x.load_written(heads, h + k);
      acc.add(x);
    }
    acc.store(out, out.row((uint32_t)a.tail_row[it.x]));
  }
}

bool aligned32(const void* p) { return (reinterpret_cast<uintptr_t>(p) & 31u) == 0; }

template <int GS, int NCH, int MODE, int KIND>
cudaError_t flat_launch(const FlatArgs& a, cudaStream_t s) {
  if (a.nw < 1) return cudaSuccess;
  cudaError_t e =
      flat::launch_early(k_flat<GS, NCH, MODE, KIND>,
                         SLNR_COUNTED(ceil_div(ceil_div(a.nw, 32 / GS), kFlatThreads / 32)), kFlatThreads, 0, s, a);
  if (e != cudaSuccess || a.nw < 2) return e;
  return flat::launch_early(k_flat_combine<GS, NCH, KIND>, SLNR_COUNTED(ceil_div(a.nw, combine_windows<GS>())),
                            kCombineThreads, 0, s, a);
}

template <int MODE, int KIND>
cudaError_t flat_width(int wm, const FlatArgs& a, cudaStream_t s) {
  if (wm <= 8) return flat_launch<1, 1, MODE, KIND>(a, s);
  if (wm <= 16) return flat_launch<2, 1, MODE, KIND>(a, s);
  if (wm <= 32) return flat_launch<4, 1, MODE, KIND>(a, s);
  if (wm <= 64) return flat_launch<8, 1, MODE, KIND>(a, s);
  if (wm <= 128) return flat_launch<16, 1, MODE, KIND>(a, s);
  if (wm <= 256) return flat_launch<32, 1, MODE, KIND>(a, s);
  if (wm <= 512) return flat_launch<32, 2, MODE, KIND>(a, s);
  return flat_launch<32, 4, MODE, KIND>(a, s);
}

FlatArgs flat_args(const CsrView& B, int W, float* out, const FlatPlan& plan) {
  FlatArgs a = {};
  a.hdr = plan.hdr;
  a.nrows = B.nrows;
  a.nnz = (int)B.nnz;
  a.win = plan.win;
  a.nw = plan.nw;
  a.pos = B.pos;
  a.crd = B.crd;
  a.vals = B.vals;
  a.W = W;
  a.out = out;
  a.first = plan.first;
  a.tail_row = plan.tail_row;
  a.head = plan.pieces;
  a.tail = plan.pieces + (size_t)plan.nw * W;
  return a;
}

template <int MODE>
cudaError_t flat_run(const FlatArgs& a, cudaStream_t s) {
  if (a.nrows <= 0) return cudaSuccess;
  const int wm = MODE == kSampled && a.L > a.W ? a.L : a.W;
  // 32-byte accesses where every row of every operand allows them
  const bool v8 = a.W % 8 == 0 && aligned32(a.X) && aligned32(a.out) && aligned32(a.D) && aligned32(a.C) &&
                  (MODE != kSampled || a.L % 8 == 0);
  if (!v8) return flat_width<MODE, flat::kV4>(wm, a, s);
  const bool whole = wm >= 8 && (wm & (wm - 1)) == 0 && (MODE != kSampled || a.L == a.W);
  return whole ? flat_width<MODE, flat::kWhole>(wm, a, s) : flat_width<MODE, flat::kV8>(wm, a, s);
}

}  // namespace

// The window: a multiple of the group's share of a stage (2 GS nonzeros) that
// leaves each resident group about six windows, so that costly windows (many
// short rows) even out.  Sums of rows: at most 9 stages, 3 for groups of half
// a warp or more, and odd multiples: windows a power of two apart ran up to
// 8 % slower (16.8M rows of 128: 96 nonzeros 661 us, 128 695, 256 708 or
// more).  Sampled sums pay for every row that starts in a window with a
// gather of C, so theirs are shorter where four or more windows share a warp
// (2M nonzeros at 64/64: 32 nonzeros 119 us, 48 125, 144 163; 3.1M at 128/32,
// two windows a warp: 96 222 us, 224 217).
int flat_window(int64_t nnz, int wm, bool sampled) {
  const int gs = wm <= 8 ? 1 : wm <= 16 ? 2 : wm <= 32 ? 4 : wm <= 64 ? 8 : wm <= 128 ? 16 : 32;
  const int64_t groups = (int64_t)kFlatSms * (sampled ? 16 : 24) * (32 / gs);
  int64_t k = nnz / (groups * 6 * 2 * gs);
  const int64_t most = gs >= 16 ? (sampled ? 7 : 3) : sampled ? 2 : 9;
  if (k > most) k = most;
  // at least 16 nonzeros, but for calls too small to fill the GPU with them
  const int64_t least = nnz < (int64_t(1) << 17) || gs >= 8 ? 1 : 16 / (2 * gs);
  if (k < least) k = least;
  if (most > 2 && k > 1) k += (k + 1) % 2;
  return (int)k * 2 * gs;
}

cudaError_t launch_flat_rows(const CsrView& B, int W, float* out, const FlatPlan& plan, cudaStream_t s) {
  if (B.nrows <= 0) return cudaSuccess;
  k_flat_rows<<<SLNR_COUNTED((unsigned)ceil_div(B.nrows, kRowsThreads)), kRowsThreads, 0, s>>>(
      flat_args(B, W, out, plan));
  return cudaGetLastError();
}

cudaError_t launch_flat_sum(const CsrView& B, const float* X, int W, float* out, const FlatPlan& plan, cudaStream_t s) {
  FlatArgs a = flat_args(B, W, out, plan);
  a.X = X;
  return flat_run<kSum>(a, s);
}

cudaError_t launch_flat_sampled(const CsrView& B, const float* C, const float* D, int L, const float* E, int K,
                                float* out, const FlatPlan& plan, cudaStream_t s) {
  FlatArgs a = flat_args(B, K, out, plan);
  a.X = E;
  a.D = D;
  a.C = C;
  a.L = L;
  return flat_run<kSampled>(a, s);
}

}  // namespace slnr
