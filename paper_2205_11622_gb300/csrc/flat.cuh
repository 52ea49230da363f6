// Lane layout and 256-bit row accesses of the nonzero-window kernels (flat.cu).
//
// A dense row of W fp32 values (W a multiple of 4) is held by a group of GS
// lanes, each lane 8 NCH of its columns as 4 NCH packed pairs: lane gl the
// 8-column blocks gl + GS i, one 32-byte access each, or, where W or the
// addresses don't allow that, the float4 columns gl + GS i.  Lanes past W
// read column 0 (always in bounds) and are left out of dot products and
// stores.
#pragma once

#include <type_traits>

#include "common.cuh"

namespace slnr {
namespace flat {

typedef unsigned long long u64;  // two packed fp32 values

__device__ __forceinline__ u64 pack2(float v) {
  u64 y;
  asm("mov.b64 %0, {%1, %1};" : "=l"(y) : "f"(v));
  return y;
}
__device__ __forceinline__ float2 unpack2(u64 y) {
  float2 v;
  asm("mov.b64 {%0, %1}, %2;" : "=f"(v.x), "=f"(v.y) : "l"(y));
  return v;
}
// Two fp32 operations in one instruction, each rounded as the scalar one.
__device__ __forceinline__ u64 fma2(u64 a, u64 b, u64 c) {
  u64 d;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
  return d;
}
__device__ __forceinline__ u64 mul2(u64 a, u64 b) {
  u64 d;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
  return d;
}
__device__ __forceinline__ u64 add2(u64 a, u64 b) {
  u64 d;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
  return d;
}

// Programmatic dependent launch: lets the next kernel of the stream start, and
// waits for the results of the one before (kernels launched without it: none to wait for).
__device__ __forceinline__ void grid_launch() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void grid_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

// Data a call streams through once: first to leave L2.
__device__ __forceinline__ uint64_t first_out() {
  uint64_t pol;
  asm("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(pol));
  return pol;
}
__device__ __forceinline__ int ld_once(const int32_t* p, uint64_t pol) {
  int v;
  asm("ld.global.nc.L2::cache_hint.b32 %0, [%1], %2;" : "=r"(v) : "l"(p), "l"(pol));
  return v;
}
__device__ __forceinline__ float ld_once(const float* p, uint64_t pol) {
  float v;
  asm("ld.global.nc.L2::cache_hint.f32 %0, [%1], %2;" : "=f"(v) : "l"(p), "l"(pol));
  return v;
}

// Zeroes the rows of `rows` (of 32, W values each, from base on) whose bit of m
// is set; by a whole warp.
__device__ __forceinline__ void zero_rows(float* rows, int W, unsigned m, int lane) {
  const int w4 = W >> 2;
  float4* base = reinterpret_cast<float4*>(rows);
  const float4 z = make_float4(0.f, 0.f, 0.f, 0.f);
  if (m == 0xffffffffu) {
    for (int i = lane; i < 32 * w4; i += 32) base[i] = z;
    return;
  }
  if (__popc(m) * ceil_div(w4, 32) > w4) {  // narrow rows: 32 / w4 of them a step
    for (int i = lane; i < 32 * w4; i += 32)
      if (m >> (i / w4) & 1u) base[i] = z;
    return;
  }
  for (; m != 0; m &= m - 1) {
    const int b = __ffs(m) - 1;
    for (int i = lane; i < w4; i += 32) base[b * w4 + i] = z;
  }
}

// How the columns of a row are spread over its lane group.
enum RowKind {
  kWhole = 0,  // W = 8 GS NCH: every lane holds columns; 32-byte accesses
  kV8 = 1,     // W a multiple of 8, lanes past W idle; 32-byte accesses
  kV4 = 2,     // any W, rows on 16-byte boundaries; 16-byte accesses
};

// This lane's place in the rows of a row-major matrix of width W: one access
// is the matrix's base plus the row's byte offset plus a lane offset.
template <int GS, int NCH, int KIND>
struct RowPtr {
  static constexpr int NP = KIND == kV4 ? 2 * NCH : NCH;  // accesses per row
  static constexpr int STEP = KIND == kV4 ? 16 : 32;      // bytes per access
  const char* base;   // column of access 0
  uint32_t pitch;     // bytes per row
  uint32_t off[KIND == kWhole ? 1 : NP];  // the other accesses, from access 0
  bool on[KIND == kWhole ? 1 : NP];

  __device__ __forceinline__ RowPtr(const float* m, int W, int gl) {
    pitch = 4u * (uint32_t)W;
    const bool on0 = KIND == kWhole || STEP * gl < (int)pitch;
    base = reinterpret_cast<const char*>(m) + (on0 ? STEP * gl : 0);
    if constexpr (KIND != kWhole) {
#pragma unroll
      for (int i = 0; i < NP; ++i) {
        on[i] = STEP * (gl + GS * i) < (int)pitch;
        off[i] = on[i] ? (uint32_t)(STEP * GS * i) : 0u;  // a lane past W reads its access 0 again
      }
    }
  }
  __device__ __forceinline__ const char* row(uint32_t r) const { return base + (uint64_t)r * pitch; }
  __device__ __forceinline__ uint32_t at(int i) const { return KIND == kWhole ? (uint32_t)(STEP * GS * i) : off[i]; }
  __device__ __forceinline__ bool holds(int i) const { return KIND == kWhole || on[i]; }
};

// One row's columns of this lane.
template <int GS, int NCH, int KIND>
struct Row {
  using Ptr = RowPtr<GS, NCH, KIND>;
  static constexpr int P = 4 * NCH;   // pairs per lane
  static constexpr int NP = Ptr::NP;  // accesses per row
  static constexpr int PP = P / NP;   // pairs per access
  u64 v[P];

  __device__ __forceinline__ void zero() {
#pragma unroll
    for (int i = 0; i < P; ++i) v[i] = 0;
  }
  __device__ __forceinline__ void load(const Ptr& m, uint32_t r) {
    const char* p = m.row(r);
#pragma unroll
    for (int i = 0; i < NP; ++i) {
      const char* q = p + m.at(i);
      if constexpr (KIND == kV4)
        asm("ld.global.nc.v2.b64 {%0, %1}, [%2];" : "=l"(v[2 * i]), "=l"(v[2 * i + 1]) : "l"(q));
      else
        asm("ld.global.nc.v4.b64 {%0, %1, %2, %3}, [%4];"
            : "=l"(v[4 * i]), "=l"(v[4 * i + 1]), "=l"(v[4 * i + 2]), "=l"(v[4 * i + 3])
            : "l"(q));
    }
  }
  // the same from memory that a kernel before this one wrote
  __device__ __forceinline__ void load_written(const Ptr& m, uint32_t r) {
    const char* p = m.row(r);
#pragma unroll
    for (int i = 0; i < NP; ++i) {
      const char* q = p + m.at(i);
      if constexpr (KIND == kV4)
        asm volatile("ld.global.v2.b64 {%0, %1}, [%2];" : "=l"(v[2 * i]), "=l"(v[2 * i + 1]) : "l"(q) : "memory");
      else
        asm volatile("ld.global.v4.b64 {%0, %1, %2, %3}, [%4];"
                     : "=l"(v[4 * i]), "=l"(v[4 * i + 1]), "=l"(v[4 * i + 2]), "=l"(v[4 * i + 3])
                     : "l"(q)
                     : "memory");
    }
  }
  // to the row whose access 0 of this lane is at p (a Ptr's row()); m: its matrix
  __device__ __forceinline__ void store(const Ptr& m, const char* p) const {
#pragma unroll
    for (int i = 0; i < NP; ++i) {
      const char* q = p + m.at(i);
      if (m.holds(i)) {
        if constexpr (KIND == kV4)
          asm volatile("st.global.v2.b64 [%0], {%1, %2};" ::"l"(q), "l"(v[2 * i]), "l"(v[2 * i + 1]) : "memory");
        else
          asm volatile("st.global.v4.b64 [%0], {%1, %2, %3, %4};" ::"l"(q), "l"(v[4 * i]), "l"(v[4 * i + 1]),
                       "l"(v[4 * i + 2]), "l"(v[4 * i + 3])
                       : "memory");
      }
    }
  }
  // the same, marked first to leave L2
  __device__ __forceinline__ void store_once(const Ptr& m, const char* p, uint64_t pol) const {
#pragma unroll
    for (int i = 0; i < NP; ++i) {
      const char* q = p + m.at(i);
      if (m.holds(i)) {
        if constexpr (KIND == kV4)
          asm volatile("st.global.L2::cache_hint.v2.b64 [%0], {%1, %2}, %3;" ::"l"(q), "l"(v[2 * i]),
                       "l"(v[2 * i + 1]), "l"(pol)
                       : "memory");
        else
          asm volatile("st.global.L2::cache_hint.v4.b64 [%0], {%1, %2, %3, %4}, %5;" ::"l"(q), "l"(v[4 * i]),
                       "l"(v[4 * i + 1]), "l"(v[4 * i + 2]), "l"(v[4 * i + 3]), "l"(pol)
                       : "memory");
      }
    }
  }
  __device__ __forceinline__ void fma(u64 s, const Row& x) {
#pragma unroll
    for (int i = 0; i < P; ++i) v[i] = fma2(s, x.v[i], v[i]);
  }
  __device__ __forceinline__ void add(const Row& x) {
#pragma unroll
    for (int i = 0; i < P; ++i) v[i] = add2(v[i], x.v[i]);
  }
  // this lane's share of <a, b> over the columns of matrix m
  static __device__ __forceinline__ float dot_part(const Ptr& m, const Row& a, const Row& b) {
    u64 s = 0;
#pragma unroll
    for (int i = 0; i < NP; ++i) {
      u64 t = i == 0 ? mul2(a.v[0], b.v[0]) : fma2(a.v[PP * i], b.v[PP * i], s);
#pragma unroll
      for (int k = 1; k < PP; ++k) t = fma2(a.v[PP * i + k], b.v[PP * i + k], t);
      s = m.holds(i) ? t : s;
    }
    const float2 f = unpack2(s);
    return f.x + f.y;
  }
};

// A launch that may start while the kernel before it on the stream drains
// (its grid_wait() waits for that kernel's results).
template <typename Args>
cudaError_t launch_early(void (*kernel)(Args), int64_t grid, int threads, size_t smem, cudaStream_t s,
                         const typename std::remove_cv<Args>::type& a) {
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)grid);
  cfg.blockDim = dim3((unsigned)threads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kernel, a);
}

}  // namespace flat
}  // namespace slnr
