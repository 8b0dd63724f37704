// mttkrp_common.cuh - helpers shared by the fused spMTTKRP + remap kernels:
// lane layout of a rank-R row over a group of lanes, bulk-async copy and
// mbarrier PTX wrappers with bounded waits, and 16-byte factor-row loads.
#pragma once

#include <cuda_bf16.h>
#include <stdint.h>

#include <algorithm>

#include "engine.h"

namespace spm {


struct LaneCfg {
  int L;    // lanes per nonzero (power of two <= 32)
  int VW;   // elements per lane per load (4 fp32 / 8 bf16 for 16-byte loads, else 1)
  int RC;   // rank chunks per lane for the scalar path
  bool vec;
};

__host__ __device__ inline int pow2ceil(int x) {
  int p = 1;
  while (p < x) p <<= 1;
  return p;
}

// narrow_bf16: BF16 rows of R <= 32 values use 8-byte lane slices (4 values), so
// that a rank-32 row takes 8 lanes, as an FP32 one does (the warp-block form).
inline LaneCfg lane_config(int R, int dtype, bool aligned16, bool narrow_bf16 = false) {
  LaneCfg c;
  int vw = dtype == SPM_DTYPE_BF16 ? ((narrow_bf16 && R <= 32) ? 4 : 8) : 4;
  if (aligned16 && R % vw == 0 && R / vw <= 32) {
    c.vec = true;
    c.VW = vw;
    c.L = pow2ceil(R / vw);
    c.RC = 1;
  } else {
    c.vec = false;
    c.VW = 1;
    if (R <= 32) {
      c.L = pow2ceil(R);
      c.RC = 1;
    } else {
      c.L = 32;
      c.RC = pow2ceil((R + 31) / 32);
    }
  }
  return c;
}

// Lanes of the warp-block form: the widest piece (values per lane and load) that
// divides the rank, fits 32 lanes and suits the alignment of the factors and the
// output, so that a rank that is no multiple of four still loads 8 bytes a lane (or 4,
// or 2) with as many nonzeros per warp as its lanes allow.
inline LaneCfg warp_lane_config(int R, int dtype, size_t factor_align, size_t out_align) {
  const size_t es = dtype == SPM_DTYPE_BF16 ? 2 : 4;
  for (int vw : {8, 4, 2}) {
    if (vw == 8 && (dtype != SPM_DTYPE_BF16 || R <= 32)) continue;  // narrow BF16: FP32's lanes
    if (R % vw || R / vw > 32 || factor_align % (vw * es) || out_align % (vw >= 4 ? 16 : 4 * vw))
      continue;
    LaneCfg c;
    c.vec = true;
    c.VW = vw;
    c.L = pow2ceil(R / vw);
    c.RC = 1;
    return c;
  }
  return lane_config(R, dtype, false);
}

// Lanes of one or two values (ranks that are no multiple of four, or factors aligned
// to less than 16 bytes): built for 3 to 6 modes and up to 64 columns; other shapes run
// the runtime-modes kernel.
inline bool narrow_built(int nmodes, bool packed, const LaneCfg& c) {
  return nmodes >= 3 && nmodes <= 6 && !packed && c.VW * c.RC <= 2;
}

// Steps in flight (U) of the warp-block kernel for a shape: the dispatchers launch this many
// and the plan sizes its tiles by it.  A tile holds at least one chunk of U G nonzeros, so
// with one-lane groups (ranks 1, 2 and 4: G = 32) eight steps would stage 256 nonzeros: one
// CTA per SM, and no room for a ring of 3 or 4 stages.  They take four (3M nonzeros, 3 modes,
// rank 1, FP32: a sweep 0.235 ms, with eight 0.286), and two where a nonzero is wider than
// 32 bytes (1.5M, 10 modes, rank 4: 0.90 ms, with four 1.07).
inline int warp_steps(int nmodes, int es, int dtype, bool packed, const LaneCfg& c, int unroll) {
  if (c.L == 1 && es > 32) return 2;
  if (narrow_built(nmodes, packed, c)) {
    if (c.L == 1) return 4;
    return nmodes <= 4 || c.VW * c.RC == 1 ? 8 : 4;
  }
  if (c.VW == 8) return nmodes == 6 ? 2 : 4;
  if (c.VW == 4) {
    if (nmodes == 3)
      return c.L == 1 || (unroll == 4 && dtype == SPM_DTYPE_F32) ? 4 : 8;
    return nmodes == 6 && dtype == SPM_DTYPE_F32 ? 2 : 4;
  }
  return c.RC == 8 ? 2 : 4;
}

// ------------------------------------------------------------ stored nonzeros

// Index k of a stored nonzeros (plain: word k; packed: its bit field).
// A field of at most 31 bits lies in two neighbouring words: one funnel shift.
__device__ __forceinline__ uint32_t pk_field(const uint32_t* w, int off, int b) {
  const uint32_t lo = off < 32 ? w[0] : (off < 64 ? w[1] : w[2]);
  const uint32_t hi = off < 32 ? w[1] : (off < 64 ? w[2] : 0u);
  return __funnelshift_r(lo, hi, off & 31) & ((1u << b) - 1u);
}
__device__ __forceinline__ int elem_index(const uint8_t* ep, int k, const PackInfo& pk) {
  const uint32_t* w = reinterpret_cast<const uint32_t*>(ep);
  return pk.packed ? (int)pk_field(w, pk.off[k], pk.bits[k]) : (int)w[k];
}
__device__ __forceinline__ float elem_value(const uint8_t* ep, int N, const PackInfo& pk) {
  return reinterpret_cast<const float*>(ep)[pk.packed ? 3 : N];
}

// ------------------------------------------------------------ PTX helpers

__device__ __forceinline__ uint32_t smem_u32(const void* p) {
  return (uint32_t)__cvta_generic_to_shared(p);
}

__device__ __forceinline__ void mbar_init(uint64_t* bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count)
               : "memory");
}

__device__ __forceinline__ void fence_mbar_init() {
  asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}

__device__ __forceinline__ void fence_proxy_async_smem() {
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
}

__device__ __forceinline__ void mbar_expect_tx(uint64_t* bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)),
               "r"(bytes)
               : "memory");
}

// 1D bulk async copy global -> shared, completes `bytes` on the mbarrier.
// Both addresses 16-byte aligned, bytes a multiple of 16.
__device__ __forceinline__ void bulk_g2s(void* dst, const void* src, uint32_t bytes,
                                         uint64_t* bar) {
  asm volatile(
      "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
          smem_u32(dst)),
      "l"(src), "r"(bytes), "r"(smem_u32(bar))
      : "memory");
}

// 1D bulk async copy with an L2 cache policy (e.g. evict_first for streams).
__device__ __forceinline__ void bulk_g2s_hint(void* dst, const void* src, uint32_t bytes,
                                              uint64_t* bar, uint64_t policy) {
  asm volatile(
      "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes.L2::cache_hint "
      "[%0], [%1], %2, [%3], %4;" ::"r"(smem_u32(dst)),
      "l"(src), "r"(bytes), "r"(smem_u32(bar)), "l"(policy)
      : "memory");
}

// L2 cache policies: 0 = evict_normal, 1 = evict_first, 2 = evict_last.
__device__ __forceinline__ uint64_t make_policy(int kind) {
  uint64_t p;
  if (kind == 1)
    asm volatile("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(p));
  else if (kind == 2)
    asm volatile("createpolicy.fractional.L2::evict_last.b64 %0, 1.0;" : "=l"(p));
  else
    asm volatile("createpolicy.fractional.L2::evict_normal.b64 %0, 1.0;" : "=l"(p));
  return p;
}

// 16-byte global store with an L2 cache policy, not allocated in L1.
__device__ __forceinline__ void st_hint_v4(void* ptr, uint4 v, uint64_t policy) {
  asm volatile("st.global.L1::no_allocate.L2::cache_hint.v4.b32 [%0], {%1, %2, %3, %4}, %5;" ::"l"(
                   ptr),
               "r"(v.x), "r"(v.y), "r"(v.z), "r"(v.w), "l"(policy)
               : "memory");
}

// 32-byte global store (a whole DRAM sector) with an L2 cache policy; the
// address must be 32-byte aligned.  A full-sector write needs no read of the
// sector's old contents, unlike a 16-byte write into it.
__device__ __forceinline__ void st_hint_v8(void* ptr, uint4 lo, uint4 hi, uint64_t policy) {
  asm volatile(
      "st.global.L1::no_allocate.L2::cache_hint.v8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8}, "
      "%9;" ::"l"(ptr),
      "r"(lo.x), "r"(lo.y), "r"(lo.z), "r"(lo.w), "r"(hi.x), "r"(hi.y), "r"(hi.z), "r"(hi.w),
      "l"(policy)
      : "memory");
}

// 16-byte read-only global load with an L2 cache policy.
__device__ __forceinline__ uint4 ld_nc_hint_v4(const void* ptr, uint64_t policy) {
  uint4 v;
  asm volatile("ld.global.nc.L2::cache_hint.v4.u32 {%0, %1, %2, %3}, [%4], %5;"
               : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w)
               : "l"(ptr), "l"(policy));
  return v;
}

// 8-byte read-only global load with an L2 cache policy.
__device__ __forceinline__ uint2 ld_nc_hint_v2(const void* ptr, uint64_t policy) {
  uint2 v;
  asm volatile("ld.global.nc.L2::cache_hint.v2.u32 {%0, %1}, [%2], %3;"
               : "=r"(v.x), "=r"(v.y)
               : "l"(ptr), "l"(policy));
  return v;
}
// 4-byte read-only global load with an L2 cache policy.
__device__ __forceinline__ uint32_t ld_nc_hint_v1(const void* ptr, uint64_t policy) {
  uint32_t v;
  asm volatile("ld.global.nc.L2::cache_hint.u32 %0, [%1], %2;" : "=r"(v) : "l"(ptr), "l"(policy));
  return v;
}

// 16-byte read-only global load with an L1 choice and an L2 cache policy: rows
// marked hot are kept in L1 longest (evict_last), the others leave it first
// (evict_first), so that L1 favours the most frequently gathered factor rows.
__device__ __forceinline__ uint4 ld_nc_l1_v4(const void* ptr, uint64_t policy, bool keep) {
  uint4 v;
  if (keep)
    asm volatile("ld.global.nc.L1::evict_last.L2::cache_hint.v4.u32 {%0, %1, %2, %3}, [%4], %5;"
                 : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w)
                 : "l"(ptr), "l"(policy));
  else
    asm volatile("ld.global.nc.L1::evict_first.L2::cache_hint.v4.u32 {%0, %1, %2, %3}, [%4], %5;"
                 : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w)
                 : "l"(ptr), "l"(policy));
  return v;
}

// Paired FP32 arithmetic (two lanes of IEEE round-to-nearest per instruction;
// the same result as two scalar operations).
__device__ __forceinline__ float2 mul2(float2 a, float2 b) {
  unsigned long long r;
  asm("mul.rn.f32x2 %0, %1, %2;"
      : "=l"(r)
      : "l"(*reinterpret_cast<unsigned long long*>(&a)),
        "l"(*reinterpret_cast<unsigned long long*>(&b)));
  return *reinterpret_cast<float2*>(&r);
}
__device__ __forceinline__ float2 fma2(float2 a, float2 b, float2 c) {
  unsigned long long r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;"
      : "=l"(r)
      : "l"(*reinterpret_cast<unsigned long long*>(&a)),
        "l"(*reinterpret_cast<unsigned long long*>(&b)),
        "l"(*reinterpret_cast<unsigned long long*>(&c)));
  return *reinterpret_cast<float2*>(&r);
}

__device__ __forceinline__ uint64_t global_ns() {
  uint64_t t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}

constexpr unsigned long long kWaitLimitNs = 2000000000ull;  // default bounded-wait limit

// Bounded wait on an mbarrier phase: gives up after limit_ns and returns false.
__device__ __forceinline__ bool mbar_wait_bounded(uint64_t* bar, uint32_t parity,
                                                  unsigned long long limit_ns = kWaitLimitNs) {
  const uint32_t a = smem_u32(bar);
  const uint64_t t0 = global_ns();
  while (true) {
    uint32_t done;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(done)
        : "r"(a), "r"(parity)
        : "memory");
    if (done) return true;
    if (global_ns() - t0 > limit_ns) return false;
  }
}

// ------------------------------------------------------------ factor slices

template <typename T, int VW>
struct Slice;

template <>
struct Slice<float, 4> {
  __device__ __forceinline__ static void load(const void* base, int64_t row, int R, int sub,
                                              float* x) {
    const float4 v =
        __ldg(reinterpret_cast<const float4*>(static_cast<const float*>(base) + row * R) + sub);
    x[0] = v.x;
    x[1] = v.y;
    x[2] = v.z;
    x[3] = v.w;
  }
};

template <>
struct Slice<__nv_bfloat16, 8> {
  __device__ __forceinline__ static void unpack(uint4 v, float* x) {
    const uint32_t w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      x[2 * j] = __uint_as_float(w[j] << 16);
      x[2 * j + 1] = __uint_as_float(w[j] & 0xffff0000u);
    }
  }
  __device__ __forceinline__ static void load(const void* base, int64_t row, int R, int sub,
                                              float* x) {
    unpack(__ldg(reinterpret_cast<const uint4*>(static_cast<const __nv_bfloat16*>(base) + row * R) +
                 sub),
           x);
  }
};

template <typename T>
__device__ __forceinline__ float load_scalar(const void* base, int64_t idx);
template <>
__device__ __forceinline__ float load_scalar<float>(const void* base, int64_t idx) {
  return __ldg(static_cast<const float*>(base) + idx);
}
template <>
__device__ __forceinline__ float load_scalar<__nv_bfloat16>(const void* base, int64_t idx) {
  const unsigned short u = __ldg(reinterpret_cast<const unsigned short*>(base) + idx);
  return __uint_as_float((uint32_t)u << 16);
}

}  // namespace spm
