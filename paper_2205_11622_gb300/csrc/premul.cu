// G = X . D, or G = (X .* X2) . D, in fp32 on the CUDA cores: the dense
// contraction of A = B.X.D done once per row of X instead of once per row of
// B (api.cu chooses).  X, X2: M x K, D: K x L, all row-major; any K and L that
// are multiples of 4.
//
// A CTA computes kPmRows x BN values, kPmK columns of X and rows of D staged
// in shared memory at a time (X transposed, so that a thread's rows are
// consecutive); a thread holds RPT rows x 4 columns as pairs of rows, two
// products per instruction.  Every value is a k-ordered fp32 chain.  Bound by
// the FMA rate for wide D, by HBM below (100k x 64 x 64: 0.8 GFLOP, 51 MB).
#include "flat.cuh"
#include "launch.h"

namespace slnr {
namespace {

using flat::u64;

constexpr int kPmThreads = 256;
constexpr int kPmRows = 128;
constexpr int kPmK = 32;
constexpr int kPmPitch = kPmRows + 4;  // keeps 16-byte alignment and spreads the transposed stores

// kSlices: row r of X belongs to slice r of a CSF tensor and goes to row crd1[r]
// of G, unless the slice has no nonzeros.
enum PremulRows { kPlain = 0, kHadamard = 1, kSlices = 2 };

template <int BN, int ROWS>
__global__ void __launch_bounds__(kPmThreads) k_premul(int64_t M, int K, int L, const float* __restrict__ X,
                                                       const float* __restrict__ X2, const float* __restrict__ D,
                                                       float* __restrict__ G, const int32_t* __restrict__ crd1,
                                                       const int32_t* __restrict__ pos2,
                                                       const int32_t* __restrict__ pos3) {
  constexpr bool H = ROWS == kHadamard;
  constexpr int CG = BN / 4;                  // threads along the columns
  constexpr int RG = kPmThreads / CG;         // threads along the rows
  constexpr int RPT = kPmRows / RG;           // rows per thread
  static_assert(RPT >= 2 && RPT % 2 == 0, "pairs of rows");
  __shared__ __align__(16) float xs[kPmK][kPmPitch];
  __shared__ __align__(16) float ds[kPmK][BN];
  const int tid = threadIdx.x, cg = tid % CG, rg = tid / CG;
  const int64_t r0 = (int64_t)blockIdx.x * kPmRows;
  const int c0 = blockIdx.y * BN;
  u64 acc[RPT / 2][4];
#pragma unroll
  for (int i = 0; i < RPT / 2; ++i)
#pragma unroll
    for (int c = 0; c < 4; ++c) acc[i][c] = 0;
  for (int k0 = 0; k0 < K; k0 += kPmK) {
    const int kn = K - k0 < kPmK ? K - k0 : kPmK;  // a multiple of 4
#pragma unroll
    for (int i = 0; i < kPmRows * kPmK / 4 / kPmThreads; ++i) {
      const int e = tid + i * kPmThreads, k4 = e % (kPmK / 4), r = e / (kPmK / 4);
      float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
      if (r0 + r < M && 4 * k4 < kn) {
        v = __ldg(reinterpret_cast<const float4*>(X + (r0 + r) * K + k0) + k4);
        if constexpr (H) {
          const float4 y = __ldg(reinterpret_cast<const float4*>(X2 + (r0 + r) * K + k0) + k4);
          v.x *= y.x; v.y *= y.y; v.z *= y.z; v.w *= y.w;
        }
      }
      xs[4 * k4 + 0][r] = v.x;
      xs[4 * k4 + 1][r] = v.y;
      xs[4 * k4 + 2][r] = v.z;
      xs[4 * k4 + 3][r] = v.w;
    }
    for (int e = tid; e < kPmK * CG; e += kPmThreads) {
      const int k = e / CG, c = e % CG;
      *reinterpret_cast<float4*>(&ds[k][4 * c]) =
          k < kn && c0 + 4 * c < L ? __ldg(reinterpret_cast<const float4*>(D + (int64_t)(k0 + k) * L + c0) + c)
                                   : make_float4(0.f, 0.f, 0.f, 0.f);
    }
    __syncthreads();
#pragma unroll 4
    for (int k = 0; k < kn; ++k) {
      const float4 d = *reinterpret_cast<const float4*>(&ds[k][4 * cg]);
      const u64 dp[4] = {flat::pack2(d.x), flat::pack2(d.y), flat::pack2(d.z), flat::pack2(d.w)};
#pragma unroll
      for (int i = 0; i < RPT / 2; ++i) {
        const u64 x = *reinterpret_cast<const u64*>(&xs[k][rg * RPT + 2 * i]);
#pragma unroll
        for (int c = 0; c < 4; ++c) acc[i][c] = flat::fma2(x, dp[c], acc[i][c]);
      }
    }
    __syncthreads();
  }
  if (c0 + 4 * cg >= L) return;
#pragma unroll
  for (int i = 0; i < RPT / 2; ++i) {
    const float2 a = flat::unpack2(acc[i][0]), b = flat::unpack2(acc[i][1]), c = flat::unpack2(acc[i][2]),
                 d = flat::unpack2(acc[i][3]);
    const int64_t r = r0 + rg * RPT + 2 * i;
    auto put = [&](int64_t row, float4 v) {
      if (row >= M) return;
      if constexpr (ROWS == kSlices) {
        if (__ldg(pos3 + __ldg(pos2 + row)) == __ldg(pos3 + __ldg(pos2 + row + 1))) return;
        row = __ldg(crd1 + row);
      }
      reinterpret_cast<float4*>(G + row * L + c0)[cg] = v;
    };
    put(r, make_float4(a.x, b.x, c.x, d.x));
    put(r + 1, make_float4(a.y, b.y, c.y, d.y));
  }
}

template <int BN>
cudaError_t premul_launch(int64_t M, int K, int L, const float* X, const float* X2, const float* D, float* G,
                          const slnr_csf3* B, cudaStream_t s) {
  const dim3 grid((unsigned)SLNR_COUNTED(ceil_div(M, kPmRows)), (unsigned)ceil_div(L, BN));
  if (B != nullptr)
    k_premul<BN, kSlices><<<grid, kPmThreads, 0, s>>>(M, K, L, X, nullptr, D, G, B->crd1, B->pos2, B->pos3);
  else if (X2 != nullptr)
    k_premul<BN, kHadamard><<<grid, kPmThreads, 0, s>>>(M, K, L, X, X2, D, G, nullptr, nullptr, nullptr);
  else
    k_premul<BN, kPlain><<<grid, kPmThreads, 0, s>>>(M, K, L, X, nullptr, D, G, nullptr, nullptr, nullptr);
  return cudaGetLastError();
}

cudaError_t premul_width(int64_t M, int K, int L, const float* X, const float* X2, const float* D, float* G,
                         const slnr_csf3* B, cudaStream_t s) {
  if (M <= 0) return cudaSuccess;
  if (L <= 16) return premul_launch<16>(M, K, L, X, X2, D, G, B, s);
  if (L <= 32) return premul_launch<32>(M, K, L, X, X2, D, G, B, s);
  return premul_launch<64>(M, K, L, X, X2, D, G, B, s);
}

constexpr int kHadThreads = 256;
constexpr int kHadPer = 4;  // float4s a thread has in flight of each matrix

// P = X .* X2, n4 float4s: what the row kernel's Hadamard gathers would form
// for every nonzero.  Bound by HBM: 12 bytes per value.
__global__ void __launch_bounds__(kHadThreads) k_hadamard(int64_t n4, const float4* __restrict__ X,
                                                          const float4* __restrict__ X2, float4* __restrict__ P) {
  const int64_t i0 = (int64_t)blockIdx.x * (kHadThreads * kHadPer) + threadIdx.x;
  float4 x[kHadPer], y[kHadPer];
#pragma unroll
  for (int k = 0; k < kHadPer; ++k) {
    const int64_t i = i0 + k * kHadThreads;
    x[k] = i < n4 ? __ldcs(X + i) : make_float4(0.f, 0.f, 0.f, 0.f);
    y[k] = i < n4 ? __ldcs(X2 + i) : make_float4(0.f, 0.f, 0.f, 0.f);
  }
#pragma unroll
  for (int k = 0; k < kHadPer; ++k) {
    const int64_t i = i0 + k * kHadThreads;
    if (i < n4) P[i] = make_float4(x[k].x * y[k].x, x[k].y * y[k].y, x[k].z * y[k].z, x[k].w * y[k].w);
  }
}

}  // namespace

cudaError_t launch_hadamard(int64_t M, int K, const float* X, const float* X2, float* P, cudaStream_t s) {
  if (M <= 0) return cudaSuccess;
  const int64_t n4 = M * (K / 4);
  k_hadamard<<<SLNR_COUNTED((unsigned)ceil_div(n4, kHadThreads * kHadPer)), kHadThreads, 0, s>>>(
      n4, reinterpret_cast<const float4*>(X), reinterpret_cast<const float4*>(X2), reinterpret_cast<float4*>(P));
  return cudaGetLastError();
}

cudaError_t launch_premul(int64_t M, int K, int L, const float* X, const float* X2, const float* D, float* G,
                          cudaStream_t s) {
  return premul_width(M, K, L, X, X2, D, G, nullptr, s);
}

cudaError_t launch_slices_times(const slnr_csf3& B, int L, int M, const float* U, const float* E, float* A,
                                cudaStream_t s) {
  return premul_width(B.nslices, L, M, U, nullptr, E, A, &B, s);
}

}  // namespace slnr
