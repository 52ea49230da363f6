// Fused MTTKRP and <MTTKRP,GEMM> over windows of consecutive nonzeros.
//
//   A(i,:) = sum_{j,k} B(i,j,k) C(j,:) .* D(k,:)
//
// Fused schedule (Sec. 4.2, Algorithm 1 removing C): the shared loops are the
// slice i and the fiber j; T(l) = sum_k B(i,j,k) D(k,l) of a fiber is formed in
// registers and T .* C(j,:) added to the slice's row at once.
//
// A warp owns a window of `win` consecutive nonzeros, whatever fibers and
// slices they belong to (Zipf slices hold from a few to millions of them).
// k_mt_first notes the slice and the fiber of each window's first nonzero and
// zeroes the rows of A that no nonzero reaches.  The warp walks its window 32
// nonzeros at a time: each lane loads one and finds its fiber among the next 32
// fiber starts (a binary search by shuffles), lane group g (GS lanes, 8 columns
// a lane: half the instructions per nonzero of 4) then gathers the D rows of
// the next GS nonzeros with 256-bit loads, sums each fiber's run in nonzero
// order and adds the run times C(j,:) where it ends.  Where a slice ends, the
// groups' rows are added and the row is written; a slice that spans
// windows leaves a tail piece where it starts and head pieces after that, which
// k_mt_combine adds in window order.  Windows depend on sizes only, so results
// are the same on every run.  <MTTKRP,GEMM> takes the slices' rows (nslices x L,
// in the workspace) times E in one product after that (premul.cu): multiplied
// inside the window's warp, tensors of many small slices took up to 1.5 times
// as long as with the separate launch (37k nonzeros in 6800 slices 89 us).
//
// What bounds it: L1 (72 % busy in an ncu capture of 10M nonzeros at L = 32, its
// data pipe 67 %; a C-row load of the few groups whose fiber ends costs as much
// as one of all eight) and the gathers' latency (7.7 warps waiting for loads for
// each that issues); 8.6 warp instructions per nonzero (19 with 4 columns a lane
// and a shuffle per value).
#include "flat.cuh"
#include "launch.h"

namespace slnr {
namespace {

using flat::Row;
using flat::u64;

constexpr int kMtThreads = 128;
constexpr int kMtWarps = kMtThreads / 32;
constexpr unsigned kFull = 0xffffffffu;

// Nonzeros of a group in flight, and resident CTAs per SM (registers).
// Measured, 10M nonzeros and 2M at rank 32 (us a call): 1 and 8 151 and 58, 1
// and 7 155 and 59, 1 and 9 (spills) 161 and 62, 2 and 6 165 and 61.
constexpr int kMtU = 1, kMtCtas = 8;

struct MtArgs {
  WsHeader* hdr;
  int d0, nslices, nfibers, nnz;
  int win, shift, nw;  // nonzeros per window (a power of two, 1 << shift), windows
  const int32_t *crd1, *pos2, *crd2, *pos3, *crd3;
  const float* vals;
  const float* C;
  const float* D;
  int L;
  float* U;          // NULL, or nslices x L: the slices' rows go here instead of A
  int M;             // width of A
  float* A;
  int* first_slice;  // [nw]
  int* first_fiber;  // [nw]
  int* tail_slice;   // [nw] slice whose first piece ends window w and goes on, or -1
  float* head;       // [nw x L]
  float* tail;       // [nw x L]
};

// First nonzero of slice s (s <= nslices).
__device__ __forceinline__ int slice_start(const MtArgs& a, int s) { return __ldg(a.pos3 + __ldg(a.pos2 + s)); }

constexpr int kFirstThreads = 256;
constexpr int kFibersPerThread = 4;

// The first `row_ctas` CTAs: a thread per row of A; the others a thread per fiber.
__global__ void __launch_bounds__(kFirstThreads) k_mt_first(const MtArgs a, int row_ctas) {
  flat::grid_launch();
  if (blockIdx.x == 0 && threadIdx.x == 0) a.hdr->error = 0;
  if ((int)blockIdx.x >= row_ctas) {
    const int64_t f0 = (int64_t)(blockIdx.x - row_ctas) * (kFirstThreads * kFibersPerThread) + threadIdx.x;
    int p[kFibersPerThread], e[kFibersPerThread];
#pragma unroll
    for (int k = 0; k < kFibersPerThread; ++k) {
      const int64_t f = f0 + k * kFirstThreads;
      p[k] = f < a.nfibers ? __ldg(a.pos3 + f) : 0;
      e[k] = f < a.nfibers ? __ldg(a.pos3 + f + 1) : 0;
    }
#pragma unroll
    for (int k = 0; k < kFibersPerThread; ++k)
      for (int w = (int)(((unsigned)p[k] + (unsigned)a.win - 1u) >> a.shift); w < a.nw && (unsigned)w << a.shift < (unsigned)e[k]; ++w)
        a.first_fiber[w] = (int)(f0 + k * kFirstThreads);
    return;
  }
  const int lane = threadIdx.x & 31;
  const int64_t i0 = (int64_t)blockIdx.x * kFirstThreads + threadIdx.x - lane, i = i0 + lane;
  const bool in = i < a.d0;
  int q = 0, p0 = 0, p1 = 0;
  if (in && a.nslices > 0) {
    int lo = 0, hi = a.nslices;  // first slice with crd1 >= i
    while (lo < hi) {
      const int mid = lo + ((hi - lo) >> 1);
      if (__ldg(a.crd1 + mid) < i) lo = mid + 1; else hi = mid;
    }
    q = lo;
    if (q < a.nslices && __ldg(a.crd1 + q) == i) {
      p0 = slice_start(a, q);
      p1 = slice_start(a, q + 1);
    }
  }
  int w0 = 0, w1 = 0;
  if (p0 < p1) {
    w0 = (int)(((unsigned)p0 + (unsigned)a.win - 1u) >> a.shift);
    w1 = (int)(((unsigned)p1 + (unsigned)a.win - 1u) >> a.shift);
  }
  for (unsigned m = __ballot_sync(kFull, w0 < w1); m != 0; m &= m - 1) {  // the warp writes each slice's windows
    const int b = __ffs(m) - 1, lo = __shfl_sync(kFull, w0, b), hi = __shfl_sync(kFull, w1, b),
              s = __shfl_sync(kFull, q, b);
    for (int w = lo + lane; w < hi; w += 32) a.first_slice[w] = s;
  }
  flat::zero_rows(a.A + i0 * a.M, a.M, __ballot_sync(kFull, in && p0 == p1), lane);
}

// Slice s's row is finished (every group of the warp holds it): row crd1[s] of
// A, or row s of U.
template <int GS, int NCH, int KIND>
__device__ __forceinline__ void finish_row(const MtArgs& a, const Row<GS, NCH, KIND>& u, int s, int lane) {
  if (lane >= GS) return;
  const typename Row<GS, NCH, KIND>::Ptr out(a.U != nullptr ? a.U : a.A, a.L, lane);
  u.store(out, out.row((uint32_t)(a.U != nullptr ? s : __ldg(a.crd1 + s))));
}

// Sum over the groups of the warp, in every group.
template <int GS, int NCH, int KIND>
__device__ __forceinline__ void group_total(Row<GS, NCH, KIND>& r) {
#pragma unroll
  for (int o = GS; o < 32; o <<= 1)
#pragma unroll
    for (int k = 0; k < Row<GS, NCH, KIND>::P; ++k) r.v[k] = flat::add2(r.v[k], __shfl_xor_sync(kFull, r.v[k], o));
}

template <int GS, int NCH, int KIND>
__global__ void __launch_bounds__(kMtThreads, NCH == 1 ? kMtCtas : 2) k_mt(const MtArgs a) {
  using R = Row<GS, NCH, KIND>;
  constexpr int B = GS;  // nonzeros of a group per step of 32
  constexpr int U0 = kMtU / NCH > 0 ? kMtU / NCH : 1, U = B < U0 ? B : U0;
  static_assert(B % U == 0, "batches tile a step");
  constexpr unsigned kBlocks = B == 1 ? ~0u : B == 2 ? 0x55555555u : B == 4 ? 0x11111111u : B == 8 ? 0x01010101u
                               : B == 16 ? 0x00010001u : 1u;  // the groups' first nonzeros
  __shared__ __align__(16) int2 kv[kMtWarps][32];  // k, value
  __shared__ int js[kMtWarps][32];
  const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5, g = lane / GS, gl = lane % GS;
  const int64_t w = (int64_t)blockIdx.x * kMtWarps + wib;
  const typename R::Ptr dp(a.D, a.L, gl), cp(a.C, a.L, gl);
  const uint64_t pol = flat::first_out();
  flat::grid_wait();  // k_mt_first
  flat::grid_launch();
  if (w >= a.nw) return;  // warp-uniform
  int q = (int)(w * a.win);
  const int pend = (w + 1) * a.win < a.nnz ? q + a.win : a.nnz;
  int sl = a.first_slice[w], f = a.first_fiber[w];
  bool head = slice_start(a, sl) < q;
  int send = slice_start(a, sl + 1), tail = -1;
  // a step's nonzero of this lane, and the starts and j of fibers f + 1 .. f + 32 (past the last: never)
  unsigned s;
  int jn, j0, kk;
  float vv;
  auto fetch = [&](int p0) {
    const unsigned fm = item(f, 1 + lane), p = item(p0, lane);
    s = fm <= (unsigned)a.nfibers ? (unsigned)__ldg(a.pos3 + fm) : ~0u;
    jn = fm < (unsigned)a.nfibers ? __ldg(a.crd2 + fm) : 0;
    j0 = f < a.nfibers ? __ldg(a.crd2 + f) : 0;
    kk = p < (unsigned)pend ? flat::ld_once(a.crd3 + p, pol) : 0;
    vv = p < (unsigned)pend ? flat::ld_once(a.vals + p, pol) : 0.f;
  };
  fetch(q);
  R acc;
  acc.zero();
  while (q < pend) {
    const int hi = send < pend ? send : pend;
    while (q < hi) {  // warp-uniform
      const unsigned s31 = __shfl_sync(kFull, s, 31);
      int qe = step_end(q, 32, hi);
      qe = s31 < (unsigned)qe ? (int)s31 : qe;  // labels stay inside the 32 starts
      const int n = qe - q;
      // the nonzeros where fibers start, and each lane's count of starts at or before its own
      const bool near = s - (unsigned)q < 32u;
      unsigned at = __reduce_or_sync(kFull, near ? 1u << (s - (unsigned)q) : 0u);
      int cnt = __popc(at & (2u << lane) - 1u);
      if (__popc(__ballot_sync(kFull, near)) != __popc(at)) {  // empty fibers share a start: count them all
        cnt = 0;
#pragma unroll
        for (int step = 16; step > 0; step >>= 1)
          if (__shfl_sync(kFull, s, cnt + step - 1) <= item(q, lane)) cnt += step;
      }
      const int jx = __shfl_sync(kFull, jn, cnt > 0 ? cnt - 1 : 0);
      __syncwarp();
      kv[wib][lane] = make_int2(kk, __float_as_int(vv));
      js[wib][lane] = cnt > 0 ? jx : j0;
      f += __popc(__ballot_sync(kFull, s <= (unsigned)qe));  // the fiber holding qe
      __syncwarp();
      fetch(qe);  // the next step's, in flight with this one's rows
      at |= kBlocks;  // every group begins a run at its first nonzero ...
      const unsigned starts = at >> (g * B);
      // ... and ends one at its last, before a start, and at the step's end
      const unsigned ends = n <= 0 ? 0u : ((at >> 1 | 1u << (n - 1)) & (~0u >> (32 - n))) >> (g * B);
      R t;
      t.zero();
#pragma unroll
      for (int u0 = 0; u0 < B; u0 += U) {
        R x[U], c[U];
        float v[U];
        if constexpr (U == 2) {
          const int4 e = *reinterpret_cast<const int4*>(&kv[wib][g * B + u0]);
          v[0] = __int_as_float(e.y);
          v[1] = __int_as_float(e.w);
          x[0].load(dp, (uint32_t)e.x);
          x[1].load(dp, (uint32_t)e.z);
        } else {
#pragma unroll
          for (int u = 0; u < U; ++u) {
            const int2 e = kv[wib][g * B + u0 + u];
            v[u] = __int_as_float(e.y);
            x[u].load(dp, (uint32_t)e.x);
          }
        }
#pragma unroll
        for (int u = 0; u < U; ++u) {
          if (ends >> (u0 + u) & 1) c[u].load(cp, (uint32_t)js[wib][g * B + u0 + u]);
        }
#pragma unroll
        for (int u = 0; u < U; ++u) {
          const u64 vp = flat::pack2(v[u]);
          if (starts >> (u0 + u) & 1) {
#pragma unroll
            for (int k = 0; k < R::P; ++k) t.v[k] = flat::mul2(vp, x[u].v[k]);
          } else {
            t.fma(vp, x[u]);
          }
          if (ends >> (u0 + u) & 1)
#pragma unroll
            for (int k = 0; k < R::P; ++k) acc.v[k] = flat::fma2(t.v[k], c[u].v[k], acc.v[k]);
        }
      }
      q = qe;
    }
    // the slice ends, or the window does
    group_total<GS, NCH, KIND>(acc);
    const bool whole = q == send && !head;
    if (whole) {
      finish_row<GS, NCH, KIND>(a, acc, sl, lane);
    } else if (lane < GS) {  // a piece: the head, or the tail (the slice goes on)
      const typename R::Ptr row(head ? a.head : a.tail, a.L, gl);
      acc.store(row, row.row((uint32_t)w));
    }
    if (q != send) {
      tail = head ? -1 : sl;
      break;
    }
    head = false;
    acc.zero();
    if (q < pend) {  // the next slice with nonzeros
      int k = 0;
      do {
        send = slice_start(a, ++sl + 1);
      } while (send <= q && ++k < 8);
      if (send <= q) {  // a long run of empty slices
        int lo = sl, hi2 = a.nslices - 1;
        while (lo < hi2) {
          const int mid = lo + ((hi2 - lo + 1) >> 1);
          if (slice_start(a, mid) <= q) lo = mid; else hi2 = mid - 1;
        }
        sl = lo;
        send = slice_start(a, sl + 1);
      }
    }
  }
  if (lane == 0) a.tail_slice[w] = tail;
}

// Slices that span windows: tail + heads in window order.  A CTA looks at four
// windows a warp; slices of more than kMtLong heads are summed by the whole CTA
// (lane groups take heads g, g + G, ... in order, then their sums are added in
// order), the others by a warp each (its groups the same way).  CTAs are large,
// so that the hub slice (3900 heads of 10M nonzeros) is a few rounds of loads
// long, and look at few windows, so that short slices are not one warp's chain
// (20k slices of 200 nonzeros, rank 16: 100 us with a window a thread, 72 with
// four a warp; 10k slices of 1000, rank 32: 157 | 151).
template <int NCH>
constexpr int mt_combine_threads() {
  return NCH == 1 ? 1024 : 256;  // 32 KB of shared memory
}
template <int NCH>
constexpr int mt_combine_windows() {
  return mt_combine_threads<NCH>() / 8;
}
constexpr int kMtLong = 64;

template <int GS, int NCH, int KIND>
__global__ void __launch_bounds__(mt_combine_threads<NCH>()) k_mt_combine(const MtArgs a) {
  using R = Row<GS, NCH, KIND>;
  constexpr int kMtCombineThreads = mt_combine_threads<NCH>();
  constexpr int W = kMtCombineThreads / 32, GW = 32 / GS, N = mt_combine_windows<NCH>();
  __shared__ int2 item[N];
  __shared__ int nshort, nlong;
  __shared__ u64 red[W][32 * R::P];
  const int tid = threadIdx.x, wib = tid >> 5, lane = tid & 31, g = lane / GS, gl = lane % GS;
  const typename R::Ptr heads(a.head, a.L, gl), tails(a.tail, a.L, gl);
  if (tid == 0) nshort = nlong = 0;
  flat::grid_wait();  // k_mt's pieces
  __syncthreads();
  {
    const int64_t w = (int64_t)blockIdx.x * N + tid;
    const int s = tid < N && w < a.nw ? a.tail_slice[w] : -1;
    if (s >= 0) {
      const int n = ((slice_start(a, s + 1) - 1) >> a.shift) - (int)w;
      const int at = n > kMtLong ? N - 1 - atomicAdd(&nlong, 1) : atomicAdd(&nshort, 1);
      item[at] = make_int2((int)w, n);
    }
  }
  __syncthreads();
  const int ns = nshort, nl = nlong;
  // heads k0, k0 + step, ... < n of the slice whose tail is in window w, 4 in flight
  auto add_heads = [&](R& acc, int w, int n, int k, int step) {
    const uint32_t h = (uint32_t)w + 1;
    for (; k + 3 * step < n; k += 4 * step) {
      R x[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) x[u].load_written(heads, h + (uint32_t)(k + u * step));
#pragma unroll
      for (int u = 0; u < 4; ++u) acc.add(x[u]);
    }
    for (; k < n; k += step) {
      R x;
      x.load_written(heads, h + (uint32_t)k);
      acc.add(x);
    }
  };
  for (int i = 0; i < nl; ++i) {
    const int2 it = item[N - 1 - i];
    R acc;
    acc.zero();
    if (wib == 0 && g == 0) acc.load_written(tails, (uint32_t)it.x);
    add_heads(acc, it.x, it.y, wib * GW + g, W * GW);
    group_total<GS, NCH, KIND>(acc);
#pragma unroll
    for (int k = 0; k < R::P; ++k) red[wib][k * 32 + lane] = acc.v[k];
    __syncthreads();
    if (wib == 0) {
#pragma unroll
      for (int k = 0; k < R::P; ++k) {
        u64 s = red[0][k * 32 + lane];
#pragma unroll
        for (int x = 1; x < W; ++x) s = flat::add2(s, red[x][k * 32 + lane]);
        acc.v[k] = s;
      }
      finish_row<GS, NCH, KIND>(a, acc, a.tail_slice[it.x], lane);
    }
    __syncthreads();
  }
  for (int i = wib; i < ns; i += W) {
    const int2 it = item[i];
    R acc;
    acc.zero();
    if (g == 0) acc.load_written(tails, (uint32_t)it.x);
    add_heads(acc, it.x, it.y, g, GW);
    group_total<GS, NCH, KIND>(acc);
    finish_row<GS, NCH, KIND>(a, acc, a.tail_slice[it.x], lane);
  }
}

bool aligned32(const void* p) { return (reinterpret_cast<uintptr_t>(p) & 31u) == 0; }

template <int GS, int NCH, int KIND>
cudaError_t mt_launch(const MtArgs& a, cudaStream_t s) {
  cudaError_t e =
      flat::launch_early(k_mt<GS, NCH, KIND>, SLNR_COUNTED(ceil_div(a.nw, kMtWarps)), kMtThreads, 0, s, a);
  if (e != cudaSuccess || a.nw < 2) return e;
  return flat::launch_early(k_mt_combine<GS, NCH, KIND>, SLNR_COUNTED(ceil_div(a.nw, mt_combine_windows<NCH>())),
                            mt_combine_threads<NCH>(), 0, s, a);
}

template <int KIND>
cudaError_t mt_width(const MtArgs& a, cudaStream_t s) {
  if (a.L <= 8) return mt_launch<1, 1, KIND>(a, s);
  if (a.L <= 16) return mt_launch<2, 1, KIND>(a, s);
  if (a.L <= 32) return mt_launch<4, 1, KIND>(a, s);
  if (a.L <= 64) return mt_launch<8, 1, KIND>(a, s);
  if (a.L <= 128) return mt_launch<16, 1, KIND>(a, s);
  if (a.L <= 256) return mt_launch<32, 1, KIND>(a, s);
  if (a.L <= 512) return mt_launch<32, 2, KIND>(a, s);
  return mt_launch<32, 4, KIND>(a, s);
}

MtArgs mt_args(const slnr_csf3& B, const float* C, const float* D, int L, float* U, int M, float* A,
               const MtPlan& plan) {
  MtArgs a = {};
  a.hdr = plan.hdr;
  a.d0 = B.dim[0];
  a.nslices = B.nslices;
  a.nfibers = B.nfibers;
  a.nnz = (int)B.nnz;
  a.win = plan.win;
  while ((1 << a.shift) < a.win) ++a.shift;
  a.nw = plan.nw;
  a.crd1 = B.crd1;
  a.pos2 = B.pos2;
  a.crd2 = B.crd2;
  a.pos3 = B.pos3;
  a.crd3 = B.crd3;
  a.vals = B.vals;
  a.C = C;
  a.D = D;
  a.L = L;
  a.U = U;
  a.M = M;
  a.A = A;
  a.first_slice = plan.first_slice;
  a.first_fiber = plan.first_fiber;
  a.tail_slice = plan.tail_slice;
  a.head = plan.pieces;
  a.tail = plan.pieces + (size_t)plan.nw * L;
  return a;
}

}  // namespace

// A power of two (k_mt_first divides by it for every fiber) that leaves each
// resident warp about three windows, so that costly ones even out, from 128
// to 256 nonzeros (10M: 128 163 us, 256 151, 512 157; 58k: 64 28 us, 128 23,
// 512 27), or 32 where the slices are short: each ends a step.
int mt_window(int64_t nnz, int64_t nslices) {
  if (nnz < 32 * nslices) return 32;
  return nnz / ((int64_t)152 * 32 * 3) < 192 ? 128 : 256;
}

cudaError_t launch_mt_first(const slnr_csf3& B, int L, int M, float* A, const MtPlan& plan, cudaStream_t s) {
  if (B.dim[0] <= 0) return cudaSuccess;
  const int64_t rows = ceil_div(B.dim[0], kFirstThreads), fibers = plan.nw > 0 ? ceil_div(B.nfibers, kFirstThreads * kFibersPerThread) : 0;
  k_mt_first<<<SLNR_COUNTED((unsigned)(rows + fibers)), kFirstThreads, 0, s>>>(
      mt_args(B, nullptr, nullptr, L, nullptr, M, A, plan), (int)rows);
  return cudaGetLastError();
}

cudaError_t launch_mt(const slnr_csf3& B, const float* C, const float* D, int L, float* U, float* A,
                      const MtPlan& plan, cudaStream_t s) {
  if (B.dim[0] <= 0 || plan.nw < 1) return cudaSuccess;
  const MtArgs a = mt_args(B, C, D, L, U, L, A, plan);
  const bool v8 = L % 8 == 0 && aligned32(C) && aligned32(D) && (U != nullptr || aligned32(A));
  if (!v8) return mt_width<flat::kV4>(a, s);
  return L >= 8 && (L & (L - 1)) == 0 ? mt_width<flat::kWhole>(a, s) : mt_width<flat::kV8>(a, s);
}

}  // namespace slnr
