// mttkrp_kernel.cuh - the fused mode-n spMTTKRP + dynamic remap kernel, a persistent
// grid of warps taking small blocks of the split.
//
// A block [lo, hi) of the mode-n ordered working copy (the paper's thread block over a
// tensor partition, Algorithm 4, shrunk so far that no CTA-wide synchronisation is
// needed) is one warp's work.  The resident warps take the blocks in order: two each to
// begin with, then whatever a counter hands out, claimed a block ahead.  Lane 0 streams
// the warp's blocks tile by tile through a shared-memory ring by 1D bulk-async copies
// (cp.async.bulk) of the nonzeros and of their remap ids, completion is counted on
// per-warp mbarriers, and every wait is bounded.
//   * Remap (Algorithm 3): when a tile has landed, the warp's lanes copy its nonzeros
//     to their places in the next mode's order, T_out[next_pos[p]] = x_p.  Because the
//     blocks are small and taken in order, the warps store near each other's places in
//     the next order at nearly the same time, and L2 gathers sectors into whole lines
//     before it writes them (a lone 32-byte sector costs DRAM as much as its line).
//   * Elementwise computation (Algorithm 2): the warp is cut into G groups of L lanes,
//     each lane owning a slice of a rank-R row.  Nonzero u G + g of a chunk of U G
//     consecutive ones is step u of group g.  The ring holds the gathered slices
//     A_k[i_k, slice] (k != n) of one chunk: as each step is consumed, its place takes
//     the gathers of the same step of the next chunk, across tile and block ends, so
//     the warp always has close to U G nonzeros' rows in flight and never drains.
//     Neighbouring nonzeros of one row often share a fiber index, and the groups then
//     gather the same line in one request.
//   * Rows: while the output row does not change, the groups add to G partial rows in
//     registers, which are added when the row ends.  Chunks in which it changes put
//     their weighted products in a shared-memory scratch, and a short loop adds them
//     row by row.  The block's first and last row, where they continue outside the
//     block, are left as partials in `part`, summed by the fix-up kernel in block order.
// No atomics on data (the counter only hands out blocks, and a block's result does not
// depend on who takes it): results are bit-identical from run to run and every output
// row is written exactly once (the empty ones from a list that all warps share).
//
// What bounds it, measured on a GB300 (3 modes 120000 x 90000 x 2000000, 100M nonzeros,
// Zipf 1.1, rank 32 FP32): a sweep takes 7.70 ms against 8.79 of one 1.7K-nonzero block
// per warp with its groups on four separate runs; passes of modes 0 and 1 without the
// remap 1.43 ms against 1.91 and 1.95.  Three things set the shape:
//   * Shared memory is taken from L1, and the gathers in flight (up to 128 KB per SM)
//     need L1 lines to land in: a 128-nonzero tile and a 4 KB scratch per warp left
//     modes 0 and 1 at 2.1-2.2 ms without the remap, 64 and 2 KB take 1.4.
//   * Blocks of about 512 nonzeros: larger ones spread the remap stores over more of
//     the next order than L2 holds, smaller ones pay more for their ends.
//   * Code size: with the row ends' code unrolled into every step the kernel was 50-66
//     KB, and mode 2 (50 nonzeros per row) waited on instruction fetch at 2.9 ms without
//     the remap; as a loop over the scratch it takes 1.8.
// The remainder is gather latency and the DRAM cost of the scattered sectors.
#pragma once

#include "mttkrp_common.cuh"
#include "mttkrp_tile.cuh"  // the write-order tiles (kTileNnz, kTileWordW)

namespace spm {

constexpr int kWarps = kThreads / 32;

// Per-warp shared-memory layout (bytes, in order): the staged tiles, their remap
// ids, the row scratch, one descriptor per stage, and the mbarriers.
struct WarpLayout {
  size_t ebuf, npbuf, scratch, rows, desc, mbar, total;
};

// Row scratch of a warp: the weighted products of HS steps' nonzeros (floats; 2 KB, see
// above), and the places in them where rows begin.
constexpr int kScratch = 512;
__host__ __device__ constexpr int scratch_steps(int NV, int U) {
  return kScratch / (32 * NV) < U ? kScratch / (32 * NV) : U;
}

// Remap ids staged per tile of k nonzeros: k + 3 ids at most (the copy starts at
// the 16-byte boundary at or below the tile) rounded up to a multiple of 4 ints, so
// that every bulk-copy destination stays 16-byte aligned.
__host__ __device__ inline int np_stage_ints(int tw) { return (tw + 8 + 3) & ~3; }

__host__ __device__ inline WarpLayout warp_layout(int es, int tw, int stages, bool ids) {
  WarpLayout l;
  size_t o = 0;
  l.ebuf = o;
  o += (size_t)stages * tw * es;
  l.npbuf = o;
  if (ids) o += (size_t)stages * np_stage_ints(tw) * 4;
  l.scratch = o;
  o += (size_t)kScratch * 4;
  l.rows = o;
  o += (size_t)36 * 4;
  l.desc = o;
  o += (size_t)stages * 16;
  l.mbar = o;
  o += (size_t)(stages + 1) * 8;  // the ring, plus one barrier only the stall test waits on
  l.total = (o + 127) & ~(size_t)127;
  return l;
}

// NT: modes at compile time (0 = runtime); T: factor type; VW, RC: values per piece and
// pieces of a row per lane (Piece); U: steps in flight; MODE: output mode at compile
// time (3 modes only; -1 = runtime); ESB: element bytes when fixed (0: 32, or 16 for
// packed nonzeros (PK), with 4 to 6 modes at compile time; else the plan's).
// LOSS (3 modes, 16- or 32-byte nonzeros): the fused first pass of the CP loss.  Each
// nonzero's own factor row A_n[i_n] is gathered as well; the model value
// m_e = sum_r prod_k A_k[i_k, r] and the residual e = m_e - x_e replace the
// value in the pass (so `out` receives the mode-n gradient of L = 1/2 sum e^2),
// the remapped copy written is the residual copy (the value word holds e), and
// every block leaves its FP64 partial of sum e^2 in loss_part.
// Sums four per-lane partials m[0..3] over the L >= 4 lanes of a lane group
// (lane `sub` of the group; gmask: the group's lanes) and leaves the four totals
// in every lane.  A butterfly per value takes 4 log2(L) shuffles; here the lanes
// first split the values over the two highest lane bits (each keeps the half the
// partner passes), add over the remaining bits, and gather the totals back:
// log2(L) + 4 shuffles.  Every total adds the same pairs in the same order as
// the butterfly (xor L/2 first, then L/4, ...), so the results are bit-identical.
__device__ __forceinline__ void group_sum4(float (&m)[4], int sub, int L, unsigned gmask) {
  const int h = L >> 1, q = L >> 2;
  const bool bh = (sub & h) != 0, bq = (sub & q) != 0;
  // bit h: lanes with it clear keep values 0 and 1, the others 2 and 3
  const float k0 = (bh ? m[2] : m[0]) + __shfl_xor_sync(gmask, bh ? m[0] : m[2], h);
  const float k1 = (bh ? m[3] : m[1]) + __shfl_xor_sync(gmask, bh ? m[1] : m[3], h);
  // bit q: keep one of the two (value 2 bh + bq)
  float t = (bq ? k1 : k0) + __shfl_xor_sync(gmask, bq ? k0 : k1, q);
  for (int off = q >> 1; off > 0; off >>= 1) t += __shfl_xor_sync(gmask, t, off);
  // gather: the partner across bit q holds value 2 bh + !bq, across bit h 2 !bh + ..
  const float t2 = __shfl_xor_sync(gmask, t, q);
  const float lo = bq ? t2 : t, hi = bq ? t : t2;
  const float lo2 = __shfl_xor_sync(gmask, lo, h), hi2 = __shfl_xor_sync(gmask, hi, h);
  m[0] = bh ? lo2 : lo;
  m[1] = bh ? hi2 : hi;
  m[2] = bh ? lo : lo2;
  m[3] = bh ? hi : hi2;
}

// RWARP (3 modes, 32-byte nonzeros carrying remap ids and write orders; form 3):
// the CTA's last warp does the remap of the CTA's blocks, the other warps only
// compute.  The remap warp takes the 960-nonzero write-order tiles that start in
// the CTA's range of the mode order; it stages each with one bulk copy into its
// shared-memory region (`region`: an mbarrier, then the tile at +128) and stores
// the tile's nonzeros in the order of their destinations, so stores that land
// side by side leave together.  The two roles share nothing but the input.
constexpr int kRemapRegion = 128 + kTileNnz * 32;  // bytes of the remap warp's region
__device__ __forceinline__ void remap_warp_tiles(const MttkrpArgs& a, int mode, int cw,
                                                 uint8_t* region, unsigned long long wait_ns) {
  const int lane = threadIdx.x & 31;
  const int b0 = blockIdx.x * cw, b1 = min(b0 + cw, a.nblk) - 1;
  if (b0 > b1) return;
  // a tile belongs to the block holding its first nonzero; the tiles are taken
  // in the compute warps' wavefront order: the k-th tile of each block in turn
  int64_t ft[kWarps], et[kWarps];
  int64_t kmax = 0;
#pragma unroll
  for (int w = 0; w < kWarps; ++w) {
    ft[w] = et[w] = 0;
    if (w < cw && b0 + w <= b1) {
      const int4 bw = a.blkinfo[b0 + w];
      ft[w] = ((int64_t)bw.x + kTileNnz - 1) / kTileNnz;
      et[w] = ((int64_t)bw.y + kTileNnz - 1) / kTileNnz;
      kmax = max(kmax, et[w] - ft[w]);
    }
  }
  int64_t kk = 0;
  int ww = -1;
  auto next_tile = [&]() -> int64_t {  // advances (kk, ww); -1 when done
    for (;;) {
      if (++ww == cw) {
        ww = 0;
        ++kk;
      }
      if (kk >= kmax) return -1;
      int64_t t = -1;
#pragma unroll
      for (int w = 0; w < kWarps; ++w)
        if (w == ww && ft[w] + kk < et[w]) t = ft[w] + kk;
      if (t >= 0) return t;
    }
  };
  int64_t t = next_tile();
  if (t < 0) return;
  uint64_t* bar = reinterpret_cast<uint64_t*>(region);
  uint8_t* buf = region + 128;
  const int nx = (mode + 1) % 3;
  const uint64_t pol = make_policy(1);
  if (lane == 0) {
    mbar_init(bar, 1);
    fence_mbar_init();
  }
  __syncwarp();
  auto issue = [&](int64_t t) {  // lane 0: stage tile t
    const int64_t base = t * kTileNnz;
    const uint32_t bytes = (uint32_t)min((int64_t)kTileNnz, a.nnz - base) * 32u;
    fence_proxy_async_smem();
    mbar_expect_tx(bar, bytes);
    bulk_g2s_hint(buf, a.elems_in + base * 32, bytes, bar, make_policy(0));
  };
  if (lane == 0) issue(t);
  for (uint32_t it = 0; t >= 0; ++it) {
    const uint32_t parity = it & 1u;
    const bool ok = mbar_wait_bounded(bar, parity, wait_ns);
    if (!__all_sync(0xffffffffu, ok)) {
      // the copy did not complete in time: record it, wait (bounded) for it, leave
      if (lane == 0) {
        if (a.err) atomicOr(a.err, 1);
        (void)mbar_wait_bounded(bar, parity);
      }
      return;
    }
    const int len = (int)min((int64_t)kTileNnz, a.nnz - t * kTileNnz);
    for (int j = lane; j < len; j += 32) {
      const uint32_t wo = reinterpret_cast<const uint32_t*>(buf + (size_t)j * 32)[kTileWordW];
      const int k = (int)((wo >> (10 * mode)) & 1023u);
      if (k >= len) {  // damaged write order: skip and report
        if (a.err) atomicOr(a.err, 2);
        continue;
      }
      const uint4* sp = reinterpret_cast<const uint4*>(buf + (size_t)k * 32);
      const uint4 lo4 = sp[0], hi4 = sp[1];
      const uint32_t dst = (nx == 0 ? hi4.x : (nx == 1 ? hi4.y : hi4.z)) & kAlphaMask;
      if ((int64_t)dst >= a.nnz) {
        if (a.err) atomicOr(a.err, 2);
        continue;
      }
      st_hint_v8(a.elems_out + (int64_t)dst * 32, lo4, hi4, pol);
    }
    __syncwarp();  // every lane has read the tile before the next copy lands on it
    t = next_tile();
    if (lane == 0 && t >= 0) issue(t);
  }
}

// A lane's share of a factor row: RC pieces of VW consecutive values, piece j
// starting at value (sub + L j) VW.  One load per piece: 16 bytes (4 FP32 or 8
// BF16), 8 bytes (2 or 4) or a 4- or 2-byte load where the rank or the factors'
// alignment allows no more.  BF16 stays packed until use.
template <typename T, int VW>
struct Piece;
template <>
struct Piece<float, 4> {
  using type = uint4;
  __device__ __forceinline__ static type load(const uint8_t* p, uint64_t pol) {
    return ld_nc_hint_v4(p, pol);
  }
  __device__ __forceinline__ static void unpack(const type& v, float* x) {
    x[0] = __uint_as_float(v.x);
    x[1] = __uint_as_float(v.y);
    x[2] = __uint_as_float(v.z);
    x[3] = __uint_as_float(v.w);
  }
};
template <>
struct Piece<float, 2> {
  using type = uint2;
  __device__ __forceinline__ static type load(const uint8_t* p, uint64_t pol) {
    return ld_nc_hint_v2(p, pol);
  }
  __device__ __forceinline__ static void unpack(const type& v, float* x) {
    x[0] = __uint_as_float(v.x);
    x[1] = __uint_as_float(v.y);
  }
};
template <>
struct Piece<float, 1> {
  using type = uint32_t;
  __device__ __forceinline__ static type load(const uint8_t* p, uint64_t pol) {
    return ld_nc_hint_v1(p, pol);
  }
  __device__ __forceinline__ static void unpack(const type& v, float* x) {
    x[0] = __uint_as_float(v);
  }
};
template <>
struct Piece<__nv_bfloat16, 2> {
  using type = uint32_t;
  __device__ __forceinline__ static type load(const uint8_t* p, uint64_t pol) {
    return ld_nc_hint_v1(p, pol);
  }
  __device__ __forceinline__ static void unpack(const type& v, float* x) {
    x[0] = __uint_as_float(v << 16);
    x[1] = __uint_as_float(v & 0xffff0000u);
  }
};
template <>
struct Piece<__nv_bfloat16, 4> {
  using type = uint2;
  __device__ __forceinline__ static type load(const uint8_t* p, uint64_t pol) {
    return ld_nc_hint_v2(p, pol);
  }
  __device__ __forceinline__ static void unpack(const type& v, float* x) {
    Piece<__nv_bfloat16, 2>::unpack(v.x, x);
    Piece<__nv_bfloat16, 2>::unpack(v.y, x + 2);
  }
};
template <>
struct Piece<__nv_bfloat16, 8> {
  using type = uint4;
  __device__ __forceinline__ static type load(const uint8_t* p, uint64_t pol) {
    return ld_nc_hint_v4(p, pol);
  }
  __device__ __forceinline__ static void unpack(const type& v, float* x) {
    Piece<__nv_bfloat16, 2>::unpack(v.x, x);
    Piece<__nv_bfloat16, 2>::unpack(v.y, x + 2);
    Piece<__nv_bfloat16, 2>::unpack(v.z, x + 4);
    Piece<__nv_bfloat16, 2>::unpack(v.w, x + 6);
  }
};
template <>
struct Piece<__nv_bfloat16, 1> {
  using type = uint32_t;
  __device__ __forceinline__ static type load(const uint8_t* p, uint64_t) {
    return (uint32_t)__ldg(reinterpret_cast<const unsigned short*>(p));
  }
  __device__ __forceinline__ static void unpack(const type& v, float* x) {
    x[0] = __uint_as_float(v << 16);
  }
};

// Stores the VW consecutive values of one piece, times sc.
template <int VW>
__device__ __forceinline__ void store_piece(float* __restrict__ d, const float* v, float sc) {
  if constexpr (VW % 4 == 0) {
#pragma unroll
    for (int q = 0; q < VW / 4; ++q)
      reinterpret_cast<float4*>(d)[q] = make_float4(v[4 * q] * sc, v[4 * q + 1] * sc,
                                                    v[4 * q + 2] * sc, v[4 * q + 3] * sc);
  } else if constexpr (VW == 2) {
    *reinterpret_cast<float2*>(d) = make_float2(v[0] * sc, v[1] * sc);
  } else {
    d[0] = v[0] * sc;
  }
}

// CTAs per SM the register budget is cut for.  Wide lanes (16 bytes of every
// gathered row in flight) take 128 registers and two CTAs; lanes that hold at most 24
// registers in flight take three.
template <int NT, int VW, int RC, int U>
constexpr int warp_min_ctas() {
  return NT > 0 && VW * RC <= 2 && U * (NT - 1) * VW * RC <= 24 ? 3 : 2;
}

template <int NT, typename T, int VW, int RC, int U, int MODE, int ESB = 0, bool LOSS = false,
          bool RWARP = false, bool PK = false>
__global__ void __launch_bounds__(kThreads, (warp_min_ctas<NT, VW, RC, U>()))
    mttkrp_warp_kernel(const MttkrpArgs a, const int L) {
  static_assert(!LOSS || (NT == 3 && MODE >= 0 && VW > 1 && U == 4 && (ESB == 32 || ESB == 16)),
                "the fused CP-loss pass is built for 3 modes and 16- or 32-byte nonzeros");
  static_assert(!RWARP || (NT == 3 && MODE >= 0 && VW > 1 && ESB == 32 && !LOSS),
                "the remap warp is built for 3 modes and 32-byte nonzeros");
  static_assert(!PK || NT >= 4, "packed nonzeros have 4 or more modes");
  constexpr int CW = RWARP ? kWarps - 1 : kWarps;  // warps that compute
  constexpr int NV = VW * RC;
  const int N = NT > 0 ? NT : a.nmodes;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int G = 32 / L, sub = lane % L, gw = lane / L;
  // element stride: a compile-time constant when the layout is
  constexpr int ES_C = ESB > 0 ? ESB : (NT >= 4 ? (PK ? 16 : 32) : 0);
  const int es = ES_C > 0 ? ES_C : a.es;
  const int R = a.R, mode = MODE >= 0 ? MODE : a.mode;
  const int TW = a.tile, NPK = np_stage_ints(TW);
  const bool remap = a.elems_out != nullptr && !RWARP;  // RWARP: the remap warp's work
  const bool ids = remap && !a.alpha_word;              // remap ids from the next_pos array
  const int S = a.stages;
  const WarpLayout lay = warp_layout(es, TW, S, a.alpha_word == 0);
  if constexpr (RWARP) {
    if (warp == kWarps - 1) {
      extern __shared__ __align__(128) uint8_t smem_r[];
      if (a.elems_out)
        remap_warp_tiles(a, MODE, CW, smem_r + (size_t)CW * lay.total,
                         a.wait_ns ? a.wait_ns : kWaitLimitNs);
      return;
    }
  }
  const int nwarps = gridDim.x * CW;  // blocks w and w + nwarps are warp w's, then claimed ones

  extern __shared__ __align__(128) uint8_t smem[];
  uint8_t* wbase = smem + (size_t)warp * lay.total;
  uint8_t* ebuf = wbase + lay.ebuf;
  int32_t* npbuf = reinterpret_cast<int32_t*>(wbase + lay.npbuf);
  float* scratch = reinterpret_cast<float*>(wbase + lay.scratch);
  int* srows = reinterpret_cast<int*>(wbase + lay.rows);
  int4* desc = reinterpret_cast<int4*>(wbase + lay.desc);
  uint64_t* mbar = reinterpret_cast<uint64_t*>(wbase + lay.mbar);

  const float sc = a.scale ? __ldg(a.scale) : 1.0f;
  float* __restrict__ out = a.out;
  // L2 policies: the element stream, remap ids and remapped copy are touched
  // once per mode (evict first); factor rows are reused (evict last)
  const uint64_t pol_stream = make_policy((a.hints & 1) ? 1 : 0);
  const uint64_t pol_factor = make_policy((a.hints & 2) ? 2 : 0);
  const uint32_t rowb = (uint32_t)R * (uint32_t)sizeof(T);
  const unsigned long long wait_ns = a.wait_ns ? a.wait_ns : kWaitLimitNs;

  // ---- staging.  Lane 0 walks the warp's blocks tile by tile, one stage each: a
  // descriptor {first position, nonzeros | flags << 16, block, row before the block}, then one
  // mbarrier arrival with the tile's byte count.  A tile of no nonzeros ends the sequence.
  // (The first-tile flag and the row before are not read; built without them the 3-mode
  // kernel comes out 1 % slower, 7.83 ms for 7.76 on 100M nonzeros, at the same registers.)
  constexpr int kFirst = 4, kLast = 8;  // tile flags beside BLK_HEAD_SPLIT, BLK_TAIL_SPLIT
  int in_flight = 0;                    // tiles issued and not yet waited for
  // lane 0: block and position, the next block and its descriptor, the one after
  int ib = 0, ipos = 0, ihi = 0, ib1 = blockIdx.x * CW + warp, ib2 = ib1 + nwarps;
  int4 ibi = make_int4(0, 0, 0, 0), inext = make_int4(0, 0, 0, 0);
  if (lane == 0) {
    for (int q = 0; q <= S; ++q) mbar_init(&mbar[q], 1);  // mbar[S]: never completed
    fence_mbar_init();
    if (ib1 < a.nblk) inext = a.blkinfo[ib1];
  }
  __syncwarp();
  auto issue = [&](int st) {  // into stage st
    if (lane == 0) {
      while (ipos >= ihi && ib1 < a.nblk) {  // the next block that holds nonzeros
        ib = ib1;
        ibi = inext;
        ipos = ibi.x;
        ihi = ibi.y;
        ib1 = ib2;  // both are used one block later
        if (ib1 < a.nblk) inext = a.blkinfo[ib1];
        if (ib1 < a.nblk && a.nblk > 2 * nwarps) ib2 = 2 * nwarps + atomicAdd(a.sched, 1);
        else ib2 = a.nblk;
        if (LOSS && ipos >= ihi) a.loss_part[ib] = 0.0;
      }
      const int n = ipos < ihi ? min(TW, ihi - ipos) : 0;
      const int fl = ibi.w | (ipos == ibi.x ? kFirst : 0) | (ipos + n == ihi ? kLast : 0);
      desc[st] = make_int4(ipos, n | (fl << 16), ib, ibi.z);
      const uint32_t ebytes = (uint32_t)n * es;
      uint32_t npbytes = 0;
      const int np0 = ipos & ~3;
      if (ids && n > 0) npbytes = ((uint32_t)(ipos + n - np0) * 4u + 15u) & ~15u;
      fence_proxy_async_smem();
      mbar_expect_tx(&mbar[st], ebytes + npbytes);
      if (n > 0) {
        bulk_g2s_hint(ebuf + (size_t)st * TW * es, a.elems_in + (size_t)ipos * es, ebytes,
                      &mbar[st], pol_stream);
        if (npbytes)
          bulk_g2s_hint(npbuf + st * NPK, a.next_pos + np0, npbytes, &mbar[st], pol_stream);
      }
      ipos += n;
    }
    ++in_flight;
  };
  for (int st = 0; st < S; ++st) issue(st);

  // Waits for the oldest tile not yet waited for, in stage st with mbarrier phase
  // `phase`; false (after recording the error and awaiting, bounded, the
  // copies still in flight) when its copy did not complete in time.
  bool stall = a.stall_test;  // waits first on mbar[S], which no copy and no thread completes
  auto wait_tile = [&](int st, uint32_t phase) -> bool {
    const bool ok = mbar_wait_bounded(&mbar[stall ? S : st], stall ? 0u : phase, wait_ns);
    stall = false;
    if (__all_sync(0xffffffffu, ok)) {
      --in_flight;
      return true;
    }
    if (lane == 0) {
      atomicOr(a.err, 1);
      for (; in_flight > 0; --in_flight) {
        (void)mbar_wait_bounded(&mbar[st], phase);
        if (++st == S) {
          st = 0;
          phase ^= 1u;
        }
      }
    }
    return false;
  };

  auto do_remap = [&](int st) {  // Algorithm 3: a tile's nonzeros to their places in the next order
    const int4 d = desc[st];
    const int n = d.y & 0xffff;
    const uint8_t* eb = ebuf + (size_t)st * TW * es;
    const int32_t* np = npbuf + st * NPK + (d.x & 3);
    if (es % 32 == 0) {  // whole 32-byte sectors per store (no read of the old sector)
      const int nv = es >= 32 ? es / 32 : 1;
      const int aw = a.alpha_word;  // remap id carried in the staged nonzero (Section 3.5)
      for (int i = lane; i < n * nv; i += 32) {
        const int e = (nv == 1) ? i : i / nv, c = (nv == 1) ? 0 : i - e * nv;
        const uint4* src = reinterpret_cast<const uint4*>(eb + (size_t)e * es) + 2 * c;
        const uint4 lo4 = src[0], hi4 = src[1];
        // with the ids in the nonzero (32-byte stride, one sector: c == 0) the id is
        // word aw of the sector, i.e. component aw - 4 of its upper half
        // (bit 31 of the id words is a hot-row flag, not part of the id)
        const int dst = aw ? (int)((aw == 4 ? hi4.x : (aw == 5 ? hi4.y : hi4.z)) & 0x7fffffffu)
                           : np[e];
        st_hint_v8(a.elems_out + (size_t)dst * es + 32 * c, lo4, hi4, pol_stream);
      }
    } else {
      const int nv = es / 16;  // 16-byte vectors per element
      for (int i = lane; i < n * nv; i += 32) {
        const int e = (nv == 1) ? i : i / nv, c = (nv == 1) ? 0 : i - e * nv;
        const uint4 v = reinterpret_cast<const uint4*>(eb + (size_t)e * es)[c];
        st_hint_v4(reinterpret_cast<uint4*>(a.elems_out + (size_t)np[e] * es) + c, v, pol_stream);
      }
    }
  };

  // fields of the staged nonzero at ep
  uint32_t foff[NT > 0 ? NT : 1];  // plain nonzeros: byte offsets of the fields (output row first)
#pragma unroll
  for (int j = 0; j < (NT > 0 ? NT : 1); ++j) {
    int k = mode + j;
    if (k >= N) k -= N;
    foff[j] = 4u * (uint32_t)k;
  }
  auto row_of = [&](const uint8_t* ep) -> int {
    if constexpr (PK || NT == 0) {
      return elem_index(ep, mode, a.pk);
    } else if constexpr (MODE >= 0) {
      return reinterpret_cast<const int*>(ep)[MODE];
    } else {
      return *reinterpret_cast<const int*>(ep + foff[0]);
    }
  };
  // ---- output rows.  The warp's current row `cur` is summed in G parts (acc of each
  // lane group), which are added when the row ends.  Steps in which rows change put
  // their weighted products into the scratch; every HS steps these are added to their
  // rows in a loop (unrolled with the steps, the row ends' code outgrew the instruction
  // cache).
  constexpr int HS = scratch_steps(NV, U);
  static_assert(HS >= 1 && U % HS == 0, "the scratch holds whole steps");
  float acc[NV];
#pragma unroll
  for (int j = 0; j < NV; ++j) acc[j] = 0.f;
  int cur = -1;             // current row
  bool first = true;        // cur is the block's first row
  auto piece_rank = [&](int j) -> int { return (sub + L * j) * VW; };  // first value of piece j
  auto store_row = [&](float* d, const float (&v)[NV], float s) {
#pragma unroll
    for (int j = 0; j < RC; ++j)
      if (piece_rank(j) < R) store_piece<VW>(d + piece_rank(j), v + j * VW, s);
  };
  auto add_slot = [&](int k, float (&v)[NV]) {  // v += this lane's pieces of scratch row k
#pragma unroll
    for (int j = 0; j < RC; ++j) {
      const int c = piece_rank(j) < R ? piece_rank(j) : 0;
      const float* x = scratch + k * R + c;
      if constexpr (VW % 4 == 0) {
#pragma unroll
        for (int q = 0; q < VW / 4; ++q) {
          const float4 t = reinterpret_cast<const float4*>(x)[q];
          v[j * VW + 4 * q] += t.x;
          v[j * VW + 4 * q + 1] += t.y;
          v[j * VW + 4 * q + 2] += t.z;
          v[j * VW + 4 * q + 3] += t.w;
        }
      } else {
#pragma unroll
        for (int q = 0; q < VW; ++q) v[j * VW + q] += x[q];
      }
    }
  };
  // All lanes: the row `cur` ends: to the block's partials where it is split, else to M_n.
  auto close_row = [&](int stage, bool last) {
    const int4 d = desc[stage];
    const bool split = (first && ((d.y >> 16) & BLK_HEAD_SPLIT)) ||
                       (last && ((d.y >> 16) & BLK_TAIL_SPLIT));
    float* const to = (split ? a.part : out) + (size_t)(split ? 2 * d.z + (first ? 0 : 1) : cur) * R;
    const float s = split ? 1.f : sc;
    first = false;
#pragma unroll 1
    for (int o = L; o < 32; o <<= 1)
#pragma unroll
      for (int j = 0; j < NV; ++j) acc[j] += __shfl_xor_sync(0xffffffffu, acc[j], o);
    if (gw == 0) store_row(to, acc, s);
  };
  // Adds the n nonzeros whose weighted products lie in the scratch (staged from p0 on)
  // to their rows.
  auto add_rows = [&](int n, const uint8_t* p0, int stage) {
    __syncwarp();
#pragma unroll 1
    for (int b = 0; b < n; b += 32) {
      const int m = min(32, n - b);
      const int row = lane < m ? row_of(p0 + (b + lane) * es) : -1;
      int before = __shfl_up_sync(0xffffffffu, row, 1);
      if (lane == 0) before = cur;
      const unsigned starts = __ballot_sync(0xffffffffu, lane < m && row != before);
      const int nst = __popc(starts);
      // slot i of the list: where the batch's i-th new row begins; then its end
      if ((starts >> lane) & 1u) srows[__popc(starts & ((1u << lane) - 1u))] = lane;
      if (lane == 0) srows[nst] = m;
      __syncwarp();
      int j = 0, e = srows[0];
#pragma unroll 1
      while (true) {  // first the row `cur` up to its end, then the batch's last row
#pragma unroll 1
        for (int k = j + gw; k < e; k += G) add_slot(b + k, acc);
        if (nst == 0 || e == m) break;
        close_row(stage, false);
        // the rows between, a group each
        if (nst > 1) {
#pragma unroll 1
          for (int i = gw; i < nst - 1; i += G) {
            const int k0 = srows[i], k1 = srows[i + 1];
            const uint8_t* p = p0 + (b + k0) * es;
            const int r = row_of(p);
            float v[NV];
#pragma unroll
            for (int q = 0; q < NV; ++q) v[q] = 0.f;
#pragma unroll 1
            for (int k = k0; k < k1; ++k) add_slot(b + k, v);
            store_row(out + (int64_t)r * R, v, sc);
          }
        }
        j = srows[nst - 1];
        e = m;
        cur = row_of(p0 + (b + j) * es);
#pragma unroll
        for (int q = 0; q < NV; ++q) acc[q] = 0.f;
      }
      __syncwarp();
    }
  };
  double lsum = 0.0;  // LOSS: sum of squared residuals (FP32 per chunk, FP64 across)
  auto end_block = [&](int stage) {
    close_row(stage, true);
    if constexpr (LOSS) {  // fixed-order warp sum of the lanes' partials
      for (int off = 16; off > 0; off >>= 1) lsum += __shfl_down_sync(0xffffffffu, lsum, off);
      if (lane == 0) a.loss_part[desc[stage].z] = lsum;
      lsum = 0.0;
    }
  };

  // ---- the walk: chunks of U steps of G nonzeros (nonzero u G + g of the chunk is
  // step u of group g), a rolling ring of one chunk per warp.  While a chunk is
  // consumed, step after step, each step's place in the ring is filled at once with
  // the gathers of the same step of the next chunk, across tile and block ends, so the
  // warp always has close to U G nonzeros' rows in flight and never drains.
  const int CH = U * G;
  constexpr int NI = (NT > 0 ? NT : 2) - 1;
  using P = Piece<T, VW>;
  typename P::type raw[U][NI][RC];
  typename P::type rown[LOSS ? U : 1][RC];  // A_n[i_n] (fused loss)
  // this lane's pieces of the factor rows (pieces past R read piece 0 of the row;
  // their values are never stored)
  const uint8_t* base[NI];
  const uint8_t* own = nullptr;
  uint32_t poff[RC];
#pragma unroll
  for (int j = 0; j < RC; ++j)
    poff[j] = (piece_rank(j) < R ? (uint32_t)piece_rank(j) : 0u) * (uint32_t)sizeof(T);
#pragma unroll
  for (int j = 0; j < NI; ++j) {
    int k = mode + 1 + j;
    if (k >= N) k -= N;
    base[j] = static_cast<const uint8_t*>(a.factors[k]) + (RC == 1 ? poff[0] : 0u);
  }
  if constexpr (LOSS) own = static_cast<const uint8_t*>(a.factors[mode]) + poff[0];
  const bool lane_live = sub * VW < R;

  auto val_of = [&](const uint8_t* ep) -> float {
    if constexpr (NT == 0) return elem_value(ep, N, a.pk);
    else return reinterpret_cast<const float*>(ep)[PK ? 3 : NT];
  };
  // the rows to gather of the staged nonzero at ep (LOSS: its own row too)
  auto fetch = [&](const uint8_t* ep, int& row, int (&ix)[NI]) {
    if constexpr (NT == 3 && MODE >= 0) {
      const int4 v = *reinterpret_cast<const int4*>(ep);
      const int f[3] = {v.x, v.y, v.z};
      row = f[MODE];
      ix[0] = f[(MODE + 1) % 3];
      ix[1] = f[(MODE + 2) % 3];
    } else if constexpr (PK) {  // 4-6 modes in 16 bytes (bit fields)
      const uint4 w4 = *reinterpret_cast<const uint4*>(ep);
      const uint32_t w[3] = {w4.x, w4.y, w4.z};
#pragma unroll
      for (int j = 0; j < NI; ++j) {
        int k = mode + 1 + j;
        if (k >= N) k -= N;
        ix[j] = (int)pk_field(w, a.pk.off[k], a.pk.bits[k]);
      }
    } else if constexpr (NT > 0) {
#pragma unroll
      for (int j = 0; j < NI; ++j) ix[j] = *reinterpret_cast<const int*>(ep + foff[1 + j]);
    }
  };
  auto gather = [&](int u, int row, const int (&ix)[NI]) {
    if constexpr (LOSS) {
      const uint8_t* r = own + (uint64_t)(uint32_t)row * rowb;
#pragma unroll
      for (int q = 0; q < RC; ++q) rown[u][q] = P::load(r, pol_factor);
    }
#pragma unroll
    for (int j = 0; j < NI; ++j) {  // one 32 x 32 -> 64-bit multiply-add per row address
      const uint8_t* r = base[j] + (uint64_t)(uint32_t)ix[j] * rowb;
#pragma unroll
      for (int q = 0; q < RC; ++q) raw[u][j][q] = P::load(RC == 1 ? r : r + poff[q], pol_factor);
    }
  };
  auto product = [&](int u, float (&prod)[NV]) {  // of the gathered pieces, in mode order
#pragma unroll
    for (int q = 0; q < RC; ++q) P::unpack(raw[u][0][q], prod + q * VW);
#pragma unroll
    for (int j = 1; j < NI; ++j) {
      float x[NV];
#pragma unroll
      for (int q = 0; q < RC; ++q) P::unpack(raw[u][j][q], x + q * VW);
      if constexpr (NV % 2 == 0) {  // paired FP32: half the instructions
        float2* p2 = reinterpret_cast<float2*>(prod);
        const float2* x2 = reinterpret_cast<const float2*>(x);
#pragma unroll
        for (int q = 0; q < NV / 2; ++q) p2[q] = mul2(p2[q], x2[q]);
      } else {
#pragma unroll
        for (int q = 0; q < NV; ++q) prod[q] *= x[q];
      }
    }
  };
  // A chunk consumed (nc nonzeros, staged from pc on) while the next one (nn, staged
  // from pn on) is gathered into its places of the ring.  The fast body takes a whole
  // chunk inside one output row, or inside a row and the one numbered next (so that none
  // lies between; each is added in its own registers), the slow one any chunk through the
  // scratch: at 53 nonzeros per row (17M, BF16, rank 32, no remap) the two-row body took
  // a pass from 0.42 to 0.30 ms.  Which of them runs depends on the
  // block alone, never on what the warp takes next, so results do not depend on the
  // claims.  Each step reads the fields of the next one ahead of its own arithmetic;
  // the empty asm keeps the compiler from reading all steps' fields at once (the ring
  // holds most of the registers).
  const int gs = G * es;  // bytes from a group's nonzero to its next
  // (the two-row body below adds each group's nonzeros of the second row apart)
  auto add_to = [&](float (&to)[NV], const float (&prod)[NV], float v) {
    if constexpr (NV % 2 == 0) {
      float2* a2 = reinterpret_cast<float2*>(to);
      const float2* p2 = reinterpret_cast<const float2*>(prod);
      const float2 vv = make_float2(v, v);
#pragma unroll
      for (int q = 0; q < NV / 2; ++q) a2[q] = fma2(p2[q], vv, a2[q]);
    } else {
#pragma unroll
      for (int q = 0; q < NV; ++q) to[q] = fmaf(prod[q], v, to[q]);
    }
  };
  auto next_row = [&](const float (&acc2)[NV], int stage) {  // `cur` ends, row cur + 1 begins
    close_row(stage, false);
    ++cur;
#pragma unroll
    for (int q = 0; q < NV; ++q) acc[q] = acc2[q];
  };
  auto body_fast = [&](auto two, auto full, int nn, const uint8_t* pc, const uint8_t* pn,
                       int stage) {
    constexpr bool TWO = decltype(two)::value;    // rows cur and cur + 1
    constexpr bool FULL = decltype(full)::value;  // the next chunk is whole too
    float acc2[NV];
#pragma unroll
    for (int q = 0; q < NV; ++q) acc2[q] = 0.f;
    int row1 = 0;
    const uint8_t* ec = pc + gw * es;  // this group's nonzero of the step
    const uint8_t* en = pn + gw * es;  // and of the next chunk's step
    int nrow = 0, nix[NI];
#pragma unroll
    for (int j = 0; j < NI; ++j) nix[j] = 0;
    if (FULL || gw < nn) fetch(en, nrow, nix);
    float nval = val_of(ec);
    if (TWO) row1 = row_of(ec);
#pragma unroll
    for (int u = 0; u < U; ++u) {
      int ix_g[NI];
#pragma unroll
      for (int j = 0; j < NI; ++j) ix_g[j] = nix[j];
      const float v = nval;
      const int row = row1;
      if (u + 1 < U) {
        en += gs;
        ec += gs;
        if (FULL || (u + 1) * G + gw < nn) fetch(en, nrow, nix);
        nval = val_of(ec);
        if (TWO) row1 = row_of(ec);
        asm volatile("" ::: "memory");  // read here, a step before they are used
      }
      float prod[NV];
      product(u, prod);
      if (!TWO || row == cur) add_to(acc, prod, v);
      else add_to(acc2, prod, v);
      if (FULL || u * G + gw < nn) gather(u, 0, ix_g);
      asm volatile("" ::: "memory");
    }
    if (TWO) next_row(acc2, stage);
  };
  auto body_slow = [&](int nc, int nn, const uint8_t* pc, const uint8_t* pn, int stage) {
    int i = gw;
#pragma unroll
    for (int u = 0; u < U; ++u, i += G) {
      int nrow = 0, nix[NI];
#pragma unroll
      for (int j = 0; j < NI; ++j) nix[j] = 0;
      if (i < nn) fetch(pn + i * es, nrow, nix);
      const float v = i < nc ? val_of(pc + i * es) : 0.f;
      float prod[NV];
      product(u, prod);
      if (i < nc) store_row(scratch + ((u % HS) * G + gw) * R, prod, v);
      if (i < nn) gather(u, nrow, nix);
      if (u % HS == HS - 1) {
        const int u0 = (u - HS + 1) * G;
        if (u0 < nc) add_rows(min(nc - u0, HS * G), pc + u0 * es, stage);
      }
      asm volatile("" ::: "memory");
    }
  };
  // The fused CP-loss pass: the chunk's model values first (their products kept for the
  // gradient), the next chunk's gathers behind them, then the residuals and the rows.
  auto body_loss = [&](bool same, bool two, int nc, int nn, uint8_t* pc, const uint8_t* pn, int stage) {
    float m[U], hh[U][NV];
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int i = u * G + gw;
      int nrow = 0, nix[NI];
#pragma unroll
      for (int j = 0; j < NI; ++j) nix[j] = 0;
      if (i < nn) fetch(pn + i * es, nrow, nix);
      // the model value: m_e = sum over the lanes of the group of sum_q A_k1 A_k2 A_n
      float y[NV];
      product(u, hh[u]);
      P::unpack(rown[u][0], y);
      m[u] = 0.f;
#pragma unroll
      for (int q = 0; q < NV; ++q) m[u] = fmaf(hh[u][q], y[q], m[u]);
      if (!lane_live || i >= nc) m[u] = 0.f;
      if (i < nn) gather(u, nrow, nix);
      asm volatile("" ::: "memory");
    }
    if constexpr (U == 4) {  // (always, where this pass is built)
      // shuffles within the group's lanes
      if (L >= 4) {
        group_sum4(m, sub, L, 0xffffffffu);
      } else {
#pragma unroll
        for (int u = 0; u < U; ++u)
          for (int o = L / 2; o > 0; o >>= 1) m[u] += __shfl_xor_sync(0xffffffffu, m[u], o);
      }
    }
    float sq = 0.f;
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int i = u * G + gw;
      if (i < nc) {  // the residual e = m_e - x_e replaces the value
        m[u] -= val_of(pc + i * es);
        sq = fmaf(m[u], m[u], sq);
      }
    }
    if (sub == 0) lsum += (double)sq;
    __syncwarp();  // every lane has read the chunk's values
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int i = u * G + gw;
      if (sub == 0 && i < nc)  // the residual copy: the staged value becomes e
        reinterpret_cast<float*>(pc + i * es)[3] = m[u];
      if (same) add_to(acc, hh[u], m[u]);
    }
    if (same) return;
    if (two) {
      float acc2[NV];
#pragma unroll
      for (int q = 0; q < NV; ++q) acc2[q] = 0.f;
#pragma unroll
      for (int u = 0; u < U; ++u) {
        if (row_of(pc + (u * G + gw) * es) == cur) add_to(acc, hh[u], m[u]);
        else add_to(acc2, hh[u], m[u]);
      }
      next_row(acc2, stage);
      return;
    }
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int i = u * G + gw;
      if (i < nc) store_row(scratch + ((u % HS) * G + gw) * R, hh[u], m[u]);
      if (u % HS == HS - 1) {
        const int u0 = (u - HS + 1) * G;
        if (u0 < nc) add_rows(min(nc - u0, HS * G), pc + u0 * es, stage);
      }
    }
  };
  // Runtime number of modes: a chunk's nonzeros are gathered mode by mode when it is
  // consumed, all steps' pieces of a mode in flight at once.  Steps past a short chunk's end
  // gather its last nonzero again and are not used: with a test around each step's loads
  // they went out one after the other (1.5M nonzeros, FP32, a sweep: 16 modes at rank 25
  // 26.4 ms, now 14.1; 10 modes at rank 64 6.05 and 3.45; 2 modes at rank 32 0.335 and 0.255).
  auto body_generic = [&](bool same, int nc, const uint8_t* pc, int stage) {
    float pr[U][NV];
    int eo[U];  // byte offsets of this group's nonzeros
#pragma unroll
    for (int u = 0; u < U; ++u) {
      eo[u] = min(u * G + gw, nc - 1) * es;
#pragma unroll
      for (int j = 0; j < NV; ++j) pr[u][j] = 1.f;
    }
    for (int k = 0; k < N; ++k) {
      if (k == mode) continue;
      const uint8_t* Ak = static_cast<const uint8_t*>(a.factors[k]);
      typename P::type x[U][RC];
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const uint8_t* r = Ak + (uint64_t)(uint32_t)elem_index(pc + eo[u], k, a.pk) * rowb;
#pragma unroll
        for (int j = 0; j < RC; ++j) x[u][j] = P::load(r + poff[j], pol_factor);
      }
#pragma unroll
      for (int u = 0; u < U; ++u)
#pragma unroll
        for (int j = 0; j < RC; ++j) {
          float y[VW];
          P::unpack(x[u][j], y);
#pragma unroll
          for (int c = 0; c < VW; ++c) pr[u][j * VW + c] *= y[c];
        }
    }
    if (same) {
#pragma unroll
      for (int u = 0; u < U; ++u) add_to(acc, pr[u], val_of(pc + (u * G + gw) * es));
      return;
    }
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int i = u * G + gw;
      if (i < nc) store_row(scratch + ((u % HS) * G + gw) * R, pr[u], val_of(pc + i * es));
      if (u % HS == HS - 1) {
        const int u0 = (u - HS + 1) * G;
        if (u0 < nc) add_rows(min(nc - u0, HS * G), pc + u0 * es, stage);
      }
    }
  };

  if (!wait_tile(0, 0)) return;
  int stage = 0;        // the gathering side's tile: its stage, the phase of its barrier,
  uint32_t phase = 0;   // its flags, and its nonzeros not yet gathered
  int dy = desc[0].y, left = dy & 0xffff;
  if (remap && !LOSS) do_remap(0);
  uint8_t* pn = ebuf;
  int nn = min(CH, left);
  if constexpr (NT > 0) {
#pragma unroll
    for (int u = 0; u < U; ++u) {
      if (u * G + gw < nn) {
        int row = 0, nix[NI];
        fetch(pn + (u * G + gw) * es, row, nix);
        gather(u, row, nix);
      }
    }
  }
  bool block_start = true;
  const int last_off = (CH - 1) * es;
#pragma unroll 1
  while (nn > 0) {
    uint8_t* pc = pn;  // the chunk to consume
    const int nc = nn, cstage = stage;
    left -= nn;
    const bool tile_end = left == 0;
    bool block_end = false;
    if (tile_end) {
      block_end = ((dy >> 16) & kLast) != 0;
      if (++stage == S) {
        stage = 0;
        phase ^= 1u;
      }
      if (!wait_tile(stage, phase)) return;
      dy = desc[stage].y;
      left = dy & 0xffff;
      if (remap && !LOSS && left > 0) do_remap(stage);
      pn = ebuf + (size_t)stage * TW * es;
    } else {
      pn += CH * es;
    }
    nn = min(CH, left);
    if (block_start) {
      cur = row_of(pc);
      first = true;
#pragma unroll
      for (int j = 0; j < NV; ++j) acc[j] = 0.f;
      block_start = false;
    }
    if constexpr (NT == 0) {
      body_generic(nc == CH && row_of(pc + last_off) == cur, nc, pc, cstage);
    } else {
      const int over = nc == CH ? row_of(pc + last_off) - cur : -1;  // rows begun in the chunk
      const bool same = over == 0, two = over == 1;
      if constexpr (LOSS)
        body_loss(same, two, nc, nn, pc, pn, cstage);
      else if (same && nn == CH)
        body_fast(std::false_type{}, std::true_type{}, nn, pc, pn, cstage);
      else if (same)
        body_fast(std::false_type{}, std::false_type{}, nn, pc, pn, cstage);
      else if (two)
        body_fast(std::true_type{}, std::false_type{}, nn, pc, pn, cstage);
      else
        body_slow(nc, nn, pc, pn, cstage);
    }
    if (tile_end) {  // the consumed chunk was its tile's last: the tile's stage is free
      __syncwarp();
      if (LOSS && remap) {  // the residual nonzeros, now in shared memory, to the next order
        do_remap(cstage);
        __syncwarp();
      }
      if (block_end) {
        end_block(cstage);
        block_start = true;
        __syncwarp();
      }
      issue(cstage);
    }
  }
  // the empty rows, shared by all lane groups (each reads its next piece ahead)
  const int groups = nwarps * G;
  int g = (blockIdx.x * CW + warp) * G + gw;
  int2 z = g < a.ngap ? a.gaps[g] : make_int2(0, 0);
#pragma unroll
  for (int j = 0; j < NV; ++j) acc[j] = 0.f;
  for (; g < a.ngap; g += groups) {
    const int2 next = a.ngap - g > groups ? a.gaps[g + groups] : make_int2(0, 0);
    for (int r = z.x; r < z.y; ++r) store_row(out + (int64_t)r * R, acc, 1.f);
    z = next;
  }
}

// Nonzeros per warp tile for a requested size: a whole number of chunks (U steps
// of G nonzeros).
__host__ __device__ inline int warp_tile_for(int tile, int G, int U) {
  const int c = G * U;
  return c * (tile / c > 1 ? tile / c : 1);
}

// CTAs of the fused kernel that are resident at once on the current device with
// `smem` bytes of dynamic shared memory each (asked once per kernel, size and device).
int resident_ctas(const void* kernel, size_t smem, int* ctas);

template <int NT, typename T, int VW, int RC, int U, int MODE = -1, int ESB = 0, bool LOSS = false,
          bool RWARP = false, bool PK = false>
int launch_warp_kernel(const MttkrpArgs& a0, int L, cudaStream_t s) {
  const int G = 32 / L;
  MttkrpArgs a = a0;
  // (form 3's remap warp leaves its CTA less room)
  a.tile = warp_tile_for(RWARP ? std::min(a0.tile, 64) : a0.tile, G, U);
  constexpr int CW = RWARP ? kWarps - 1 : kWarps;  // warps that compute
  // form 3: seven compute warps' slots, then the remap warp's region
  const size_t smem = CW * warp_layout(a.es, a.tile, a.stages, a.alpha_word == 0).total +
                      (RWARP ? kRemapRegion : 0);
  auto kfn = mttkrp_warp_kernel<NT, T, VW, RC, U, MODE, ESB, LOSS, RWARP, PK>;
  int st = ensure_dyn_smem((const void*)kfn, smem, "cudaFuncSetAttribute(mttkrp_warp)");
  if (st) return st;
  int grid = (a.nblk + CW - 1) / CW;
  if (!RWARP) {  // (form 3's remap warps cover their CTA's own blocks)
    int ctas = 0;
    st = resident_ctas((const void*)kfn, smem, &ctas);
    if (st) return st;
    grid = std::min(std::max(grid, (a.ngap + CW * G - 1) / (CW * G)), ctas);
    // blocks past the warps' first two are claimed from a counter
    if (a.nblk > 2 * grid * CW) SPM_CUDA(cudaMemsetAsync(a.sched, 0, sizeof(int), s));
  }
  kfn<<<grid, kThreads, smem, s>>>(a, L);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return cuda_fail(e, "mttkrp_warp_kernel launch");
  return SPM_OK;
}

// 4 to 6 modes: nonzeros in 32-byte sectors, or packed in 16 bytes.
template <int NT, typename T, int VW, int U>
int launch_modes(const MttkrpArgs& a, int L, cudaStream_t s) {
  if (a.pk.packed) return launch_warp_kernel<NT, T, VW, 1, U, -1, 0, false, false, true>(a, L, s);
  return launch_warp_kernel<NT, T, VW, 1, U>(a, L, s);
}

inline bool narrow_built(const MttkrpArgs& a, const LaneCfg& c) {
  return narrow_built(a.nmodes, a.pk.packed, c);
}
inline int warp_steps(const MttkrpArgs& a, const LaneCfg& c) {
  return warp_steps(a.nmodes, a.es, a.dtype, a.pk.packed, c, a.unroll);
}
// The runtime-modes kernel with one- to four-value pieces (4 steps, or 2: warp_steps).
template <typename T, int VW>
int launch_any_modes(const MttkrpArgs& a, const LaneCfg& c, cudaStream_t s) {
  if (warp_steps(a, c) == 2) return launch_warp_kernel<0, T, VW, 1, 2>(a, c.L, s);
  return launch_warp_kernel<0, T, VW, 1, 4>(a, c.L, s);
}
int launch_narrow_f32(const MttkrpArgs& a, const LaneCfg& c, cudaStream_t s);
int launch_narrow_bf16(const MttkrpArgs& a, const LaneCfg& c, cudaStream_t s);

}  // namespace spm
