// G = X . D (or (X .* X2) . D) on tcgen05 TF32 tensor cores: the dense first
// step of A = B . (X . D), X M x K, D K x L, both row-major fp32.
//
// X enters as the sum of two tf32 values per fp32 value (hi = x rounded, lo =
// x - hi rounded), so that only D's rounding is left in the product.  A D with
// infinities or NaN takes the hi parts alone: 0 times infinity in a lo product
// would turn an infinite result into NaN.
//
// What bounds it: the M (K + L) floats that X and G move through memory (both
// X and X2 with the Hadamard product); the MMAs of a 128 x 128 x 128 tile take
// a third of the time its rows need to arrive.  So a persistent CTA per SM
// keeps loads in flight across tiles:
//   16 producer warps: warp w loads rows 8w .. 8w + 7 of each chunk (128 rows x
//                32 columns of X) into registers, two or four chunks ahead (64
//                KB per SM in flight), splits them and stores hi and lo, 128B
//                swizzled and K-major, into a ring of four 32 KB stages;
//   MMA warp:    issues the 8 MMAs of a chunk, gives the stage back, and after
//                a tile's last chunk hands over one of two accumulators;
//   4 epilogue warps: tensor memory -> shared memory -> whole row pieces of G.
// A tile held whole (128 x 128 hi and lo is 128 KB beside D^T's 64 KB) had a
// single buffer, so loads, MMAs and stores of one tile followed one another.
// Whole calls with the product first, whole tiles | chunks: 1M rows 128/128 with
// the Hadamard product and 16M nonzeros 1068 | 980 us, without it 957 | 856;
// 128/32 664 | 549 (calls of that size now go row first); 100k rows 64/64 99 |
// 91; 4k rows 16/16 36 | 31.  A step of the ring holds 32
// columns because D^T (64 KB) and the epilogue's pieces (18 KB) leave 128 KB.
// Every wait is bounded; a wait that gives up sets kErrTimeout, and MMAs in
// flight are drained before the tensor memory is freed.
#include "launch.h"
#include "tcgen05.cuh"

namespace slnr {

namespace {

constexpr int kPtProducers = 16;
constexpr int kPtMmaWarp = kPtProducers;                // then the four epilogue warps
constexpr int kPtThreads = 32 * (kPtProducers + 1 + 4);
constexpr int kPtRows = 128;                            // MMA M
constexpr int kPtStages = 4;
constexpr int kPtBlock = kPtRows * 128;                 // 128 rows x 32 tf32 values
constexpr int kPtStage = 2 * kPtBlock;                  // hi, lo
static_assert(kPtRows == 8 * kPtProducers, "each producer warp owns eight rows of a chunk");

__host__ __device__ constexpr int pt_kt(int K) { return K < 32 ? 32 : K; }
__host__ __device__ constexpr int pt_chunk(int L) { return L < 32 ? L : 32; }  // columns the epilogue stages at a time
__host__ __device__ constexpr int pt_pitch(int L) { return pt_chunk(L) * 4 + 16; }
__host__ __device__ constexpr uint32_t pt_tmem_cols(int L) { return 2 * L < 32 ? 32u : (uint32_t)(2 * L); }
__host__ __device__ constexpr size_t pt_smem_bytes(int K, int L) {
  return (size_t)kPtStages * kPtStage + (size_t)L * pt_kt(K) * 4 + (size_t)4 * 32 * pt_pitch(L) + 1024;
}
static_assert(pt_smem_bytes(128, 128) <= (size_t)227 * 1024, "shared memory of a CTA");

// Waits for the phase with the given parity to complete; false after `limit` cycles.
__device__ __forceinline__ bool pt_wait(uint64_t* bar, uint32_t parity, long long limit) {
  const long long t0 = clock64();
  while (!tc::mbar_try_wait(bar, parity))
    if (clock64() - t0 > limit) return false;
  return true;
}

// v as the sum of two tf32 values each.  Infinities and NaN have no second
// part; the largest finite values, which would round to infinity, are cut off.
__device__ __forceinline__ void pt_split(const float4& v, uint4& hi, uint4& lo) {
  const float x[4] = {v.x, v.y, v.z, v.w};
  uint32_t h[4], l[4], most = 0;
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    h[i] = tc::to_tf32(x[i]);
    l[i] = tc::to_tf32(x[i] - __uint_as_float(h[i]));
    most = max(most, h[i] & 0x7FFFFFFFu);
  }
  if (most >= 0x7F800000u) {
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      if ((h[i] & 0x7F800000u) != 0x7F800000u) continue;
      const uint32_t bits = __float_as_uint(x[i]);
      const bool finite = (bits & 0x7F800000u) != 0x7F800000u;
      if (finite) h[i] = bits & 0xFFFFE000u;
      l[i] = finite ? tc::to_tf32(x[i] - __uint_as_float(h[i])) : 0u;
    }
  }
  hi = make_uint4(h[0], h[1], h[2], h[3]);
  lo = make_uint4(l[0], l[1], l[2], l[3]);
}

template <int K, int L, bool H>
__global__ void __launch_bounds__(kPtThreads, 1)
    k_tc_premul(WsHeader* hdr, int64_t M, const float* __restrict__ X, const float* __restrict__ X2,
                const float* __restrict__ D, float* __restrict__ G, long long wait_cycles) {
  constexpr int KT = pt_kt(K), KB = KT / 32;  // chunks per tile
  constexpr int PD = H ? 2 : 4;               // chunks a producer warp has in flight
  constexpr uint32_t IDESC = tc::idesc_tf32(kPtRows, L), NCOLS = pt_tmem_cols(L);
  static_assert((NCOLS & (NCOLS - 1)) == 0 && NCOLS >= 32 && NCOLS <= 512, "tensor memory allocation");
  __shared__ uint64_t full[kPtStages], empty[kPtStages], done[2], drained[2], last;
  __shared__ uint32_t tmem_base;
  __shared__ int failed;
  extern __shared__ uint8_t smem_raw[];
  uint8_t* sX = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  uint8_t* sD = sX + kPtStages * kPtStage;
  uint8_t* sE = sD + L * KT * 4;

  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  if (warp == kPtMmaWarp) {
    tc::tmem_alloc(&tmem_base, NCOLS);
    tc::tmem_relinquish();
  }
  if (tid == 0) {
    for (int i = 0; i < kPtStages; ++i) {
      tc::mbar_init(&full[i], kPtProducers);
      tc::mbar_init(&empty[i], 1);
    }
    for (int b = 0; b < 2; ++b) {
      tc::mbar_init(&done[b], 1);
      tc::mbar_init(&drained[b], 4);
    }
    tc::mbar_init(&last, 1);
    tc::fence_mbar_init();
    failed = 0;
  }
  // D^T as the B operand, tf32; the rows k >= K of a padded tile are zero
  int odd = 0;  // D holds an infinity or NaN
  for (int i = tid; i < KT * (L / 4); i += kPtThreads) {
    const int k = i / (L / 4), n4 = i % (L / 4);
    const float4 d = k < K ? __ldg(reinterpret_cast<const float4*>(D + (int64_t)k * L) + n4)
                           : make_float4(0.f, 0.f, 0.f, 0.f);
    const float dv[4] = {d.x, d.y, d.z, d.w};
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      const uint32_t t = tc::to_tf32(dv[e]);
      odd |= (t & 0x7F800000u) == 0x7F800000u;
      *reinterpret_cast<uint32_t*>(sD + tc::sw128_offset(4 * n4 + e, k, L)) = t;
    }
  }
  tc::fence_proxy_async_smem();
  tc::tc_fence_before_sync();
  const bool hi_only = __syncthreads_or(odd) != 0;
  tc::tc_fence_after_sync();
  const uint32_t tmem = tmem_base;

  const int ntiles = (int)((M + kPtRows - 1) / kPtRows);  // this CTA's: blockIdx.x, + gridDim.x, ...
  const int mine = (int)blockIdx.x < ntiles ? (ntiles - 1 - (int)blockIdx.x) / (int)gridDim.x + 1 : 0;

  if (warp < kPtProducers) {
    const int nchunks = mine * KB, lr = lane >> 3, lc = lane & 7;
    float4 x[PD][2], y[PD][2];
    auto load = [&](int c, float4 (&xv)[2], float4 (&yv)[2]) {
      const int64_t r0 = ((int64_t)blockIdx.x + (int64_t)(c / KB) * gridDim.x) * kPtRows + 8 * warp + lr;
      const int col = (c % KB) * 32 + 4 * lc;
#pragma unroll
      for (int i = 0; i < 2; ++i) {
        const int64_t r = r0 + 4 * i;
        const bool in = r < M && (K >= 32 || col < K);
        xv[i] = in ? __ldcs(reinterpret_cast<const float4*>(X + r * K + col)) : make_float4(0.f, 0.f, 0.f, 0.f);
        if constexpr (H)
          yv[i] = in ? __ldcs(reinterpret_cast<const float4*>(X2 + r * K + col)) : make_float4(0.f, 0.f, 0.f, 0.f);
      }
    };
#pragma unroll
    for (int u = 0; u < PD; ++u)
      if (u < nchunks) load(u, x[u], y[u]);
    bool ok = true;
    for (int c0 = 0; c0 < nchunks && ok; c0 += PD) {
#pragma unroll
      for (int u = 0; u < PD; ++u) {
        const int c = c0 + u, st = c % kPtStages;
        if (c >= nchunks || !ok) break;
        if (c >= kPtStages)
          ok = __all_sync(0xffffffffu, pt_wait(&empty[st], (c / kPtStages - 1) & 1, wait_cycles));
        if (!ok) {
          if (lane == 0) atomicOr(&failed, 1);
          break;
        }
        uint8_t* s = sX + st * kPtStage;
#pragma unroll
        for (int i = 0; i < 2; ++i) {
          float4 v = x[u][i];
          if constexpr (H) v = make_float4(v.x * y[u][i].x, v.y * y[u][i].y, v.z * y[u][i].z, v.w * y[u][i].w);
          uint4 hi, lo;
          pt_split(v, hi, lo);
          const int r = 8 * warp + 4 * i + lr, off = r * 128 + ((lc ^ (r & 7)) << 4);
          *reinterpret_cast<uint4*>(s + off) = hi;
          *reinterpret_cast<uint4*>(s + kPtBlock + off) = lo;
        }
        tc::fence_proxy_async_smem();
        __syncwarp();
        if (lane == 0) tc::mbar_arrive(&full[st]);
        if (c + PD < nchunks) load(c + PD, x[u], y[u]);
      }
    }
  } else if (warp == kPtMmaWarp) {
    if (lane == 0) {
      const uint32_t x_addr = tc::smem_u32(sX), d_addr = tc::smem_u32(sD);
      bool ok = true;
      for (int j = 0; j < mine && ok; ++j) {
        const int b = j & 1;
        if (j >= 2) ok = pt_wait(&drained[b], (j / 2 - 1) & 1, wait_cycles);
        for (int kb = 0; kb < KB && ok; ++kb) {
          const int c = j * KB + kb, st = c % kPtStages;
          ok = pt_wait(&full[st], (c / kPtStages) & 1, wait_cycles);
          if (!ok) break;
          tc::tc_fence_after_sync();
          for (int p = 0; p < (hi_only ? 1 : 2); ++p)
#pragma unroll
            for (int ks = 0; ks < 4; ++ks)
              tc::mma_tf32(tmem + (uint32_t)(b * L),
                           tc::desc_k_sw128(x_addr + st * kPtStage + p * kPtBlock + ks * 32),
                           tc::desc_k_sw128(d_addr + kb * L * 128 + ks * 32), IDESC, (kb | p | ks) != 0);
          tc::mma_commit(&empty[st]);
          if (kb == KB - 1) tc::mma_commit(&done[b]);
        }
      }
      if (!ok) atomicOr(&failed, 1);
    }
    __syncwarp();
  } else {
    const int q = warp & 3;  // tensor memory lanes 32 q .. 32 q + 31
    constexpr int CW = pt_chunk(L), PITCH = pt_pitch(L), LPR = CW / 4, RPI = 32 / LPR;
    uint8_t* stage = sE + (size_t)q * 32 * PITCH;
    for (int j = 0; j < mine; ++j) {
      const int b = j & 1;
      if (!__all_sync(0xffffffffu, pt_wait(&done[b], (j / 2) & 1, wait_cycles))) {
        if (lane == 0) atomicOr(&failed, 1);
        break;
      }
      tc::tc_fence_after_sync();
      const int64_t r0 = ((int64_t)blockIdx.x + (int64_t)j * gridDim.x) * kPtRows + 32 * q;
#pragma unroll 1
      for (int c = 0; c < L; c += CW) {
        float v[CW];
        if constexpr (CW == 32)
          tc::tmem_ld32(tmem + ((uint32_t)(32 * q) << 16) + (uint32_t)(b * L + c), v);
        else
          tc::tmem_ld16(tmem + ((uint32_t)(32 * q) << 16) + (uint32_t)(b * L + c), v);
        __syncwarp();  // the previous piece has been read
#pragma unroll
        for (int i = 0; i < CW / 4; ++i)
          *reinterpret_cast<float4*>(stage + (size_t)lane * PITCH + 16 * i) =
              make_float4(v[4 * i], v[4 * i + 1], v[4 * i + 2], v[4 * i + 3]);
        __syncwarp();
#pragma unroll
        for (int i = 0; i < 32 / RPI; ++i) {
          const int r = RPI * i + lane / LPR, part = lane % LPR;
          if (r0 + r < M)
            *reinterpret_cast<float4*>(G + (r0 + r) * L + c + 4 * part) =
                *reinterpret_cast<const float4*>(stage + (size_t)r * PITCH + 16 * part);
        }
      }
      tc::tc_fence_before_sync();
      __syncwarp();
      if (lane == 0) tc::mbar_arrive(&drained[b]);
    }
  }

  tc::tc_fence_before_sync();
  __syncthreads();
  if (failed) {
    if (warp == kPtMmaWarp && lane == 0) {  // the MMAs that were issued end before the tensor memory is freed
      tc::mma_commit(&last);
      pt_wait(&last, 0, kWaitCycles);
    }
    if (tid == 0) atomicOr(&hdr->error, kErrTimeout);
  }
  __syncthreads();
  tc::tc_fence_after_sync();
  if (warp == kPtMmaWarp) tc::tmem_dealloc(tmem, NCOLS);
}

template <int K, int L, bool H>
cudaError_t pt_launch(int64_t M, const float* X, const float* X2, const float* D, float* G, WsHeader* hdr,
                      cudaStream_t s) {
  constexpr size_t smem = pt_smem_bytes(K, L);
  const cudaError_t e =
      cudaFuncSetAttribute(k_tc_premul<K, L, H>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  int64_t grid = (M + kPtRows - 1) / kPtRows;
  if (grid > device_sm_count()) grid = device_sm_count();
  k_tc_premul<K, L, H><<<SLNR_COUNTED((unsigned)grid), kPtThreads, smem, s>>>(hdr, M, X, X2, D, G, wait_limit_cycles());
  return cudaGetLastError();
}

template <int K, int L>
cudaError_t pt_kind(int64_t M, const float* X, const float* X2, const float* D, float* G, WsHeader* hdr,
                    cudaStream_t s) {
  return X2 != nullptr ? pt_launch<K, L, true>(M, X, X2, D, G, hdr, s)
                       : pt_launch<K, L, false>(M, X, X2, D, G, hdr, s);
}

template <int K>
cudaError_t pt_width(int L, int64_t M, const float* X, const float* X2, const float* D, float* G, WsHeader* hdr,
                     cudaStream_t s) {
  switch (L) {
    case 16: return pt_kind<K, 16>(M, X, X2, D, G, hdr, s);
    case 32: return pt_kind<K, 32>(M, X, X2, D, G, hdr, s);
    case 64: return pt_kind<K, 64>(M, X, X2, D, G, hdr, s);
    case 128: return pt_kind<K, 128>(M, X, X2, D, G, hdr, s);
  }
  return cudaErrorInvalidValue;
}

}  // namespace

bool tc_split_supported(int K, int L) {
  return (K == 16 || K == 32 || K == 64 || K == 128) && (L == 16 || L == 32 || L == 64 || L == 128);
}

cudaError_t launch_tc_premul(int64_t M, int K, int L, const float* X, const float* X2, const float* D, float* G,
                             WsHeader* hdr, cudaStream_t s) {
  if (M <= 0) return cudaSuccess;
  switch (K) {
    case 16: return pt_width<16>(L, M, X, X2, D, G, hdr, s);
    case 32: return pt_width<32>(L, M, X, X2, D, G, hdr, s);
    case 64: return pt_width<64>(L, M, X, X2, D, G, hdr, s);
    case 128: return pt_width<128>(L, M, X, X2, D, G, hdr, s);
  }
  return cudaErrorInvalidValue;
}

}  // namespace slnr
