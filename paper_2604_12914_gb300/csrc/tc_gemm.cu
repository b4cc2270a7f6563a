// tcgen05 GEMM (kind::tf32 on TF32 operands, kind::f16 on BF16 operands) for sm_103a,
// persistent and warp-specialised: one CTA per SM walks a
// static list of (tile, K split) work units.  Warp 0 streams A/B K blocks with TMA (128-byte
// swizzle) into a 4-stage shared-memory ring, warp 1 issues tcgen05.mma into one of two TMEM
// accumulators, and warps 2-9 drain the other accumulator (tcgen05.ld -> registers ->
// shared-memory staging -> coalesced global stores), so the epilogue of one tile overlaps
// the main loop of the next.  Large products run as pairs of CTAs on 256-row tiles
// (tc_pair_kernel), the split modes as tc_split_kernel.  Every mbarrier wait is bounded (globaltimer); on timeout the
// kernel raises a device flag, stops every role, drains its own copies and MMAs with bounded
// waits, frees its TMEM and returns.
#include <cstdio>
#include <cstdlib>
#include <cuda.h>
#include <cudaTypedefs.h>

#include <map>
#include <mutex>
#include <tuple>
#include <type_traits>
#include <vector>

#include "engine.cuh"
#include "tc_gemm.cuh"
#include "tc_ptx.cuh"

namespace cclr {
namespace {

constexpr int BM = 128;      // UMMA M
constexpr int BKB = 128;     // bytes per K block = one 128-byte swizzle row (32 TF32 or 64 BF16)
constexpr int STAGES = 4;

struct TcParams {
  int M, N, K, BN;
  int nMt, nNt, band;   // tile counts; M tiles per raster band (N varies fastest inside a band)
  int kb_per_split;     // K blocks per split (splits of K are atomically summed)
  int splits;           // work units = tiles x splits, walked with stride gridDim.x
  const uint32_t *list; // the tiles to compute, (m << 16) | n, ntiles of them (nullptr: all, in raster order)
  int ntiles;
  int store;            // epilogue: a StoreMode
  float *C;
  View2 rv, cv;         // C rows and complex columns
  float ar, ai;
  int accumulate;       // add to C (always true when split)
  int atomic;           // split-K: combine partial tiles with atomicAdd
  int *err;
  float tau;            // the kernels that compare their sums instead of storing them (tc_magnitude_sums)
  uint32_t *words;
};

// work unit -> (m tile, n tile, split); banded rasterisation: consecutive units share one B
// tile column across a band of M tiles, so the band's A tiles and the current B tiles stay in L2
__device__ __forceinline__ void unit_coords(const TcParams &p, int u, int &m_tile, int &n_tile, int &split) {
  split = u / p.ntiles;
  const int id = u - split * p.ntiles;
  if (p.list) {
    const uint32_t mn = __ldg(p.list + id);
    m_tile = (int)(mn >> 16);
    n_tile = (int)(mn & 0xffff);
    return;
  }
  const int per_band = p.band * p.nNt;
  const int b = id / per_band;
  const int local = id - b * per_band;
  const int mb = min(p.band, p.nMt - b * p.band);
  m_tile = b * p.band + local % mb;
  n_tile = local / mb;
}

constexpr int EPI_PITCH = 18;  // floats per staged row (16 + 2): conflict-free float2 traffic

// How a warp writes its part of C: a lane per row; lanes along contiguous columns; the same two complex columns at a time
// (C 16-byte aligned, everything that its views add up to even)
enum StoreMode { STORE_ROWS = 0, STORE_COLS = 1, STORE_PAIRS = 2 };

// The rows of C (nullptr: beyond M) that a lane writes in every chunk of a unit, rows row0 + .. of the warp's 32
struct RowPtrs {
  float *p[8];
  __device__ __forceinline__ RowPtrs(const TcParams &q, int row0, int lane) {
    const int step = q.store == STORE_PAIRS ? 8 : 4;
    const int first = row0 + (q.store == STORE_PAIRS ? lane >> 2 : q.store == STORE_COLS ? lane >> 3 : lane);
#pragma unroll
    for (int k = 0; k < 8; ++k) {
      const int row = first + k * step;
      p[k] = row < q.M && k < (q.store == STORE_PAIRS ? 4 : q.store == STORE_COLS ? 8 : 1) ? q.C + 2 * v2off(q.rv, row) : nullptr;
    }
  }
};

// One 16-column chunk of a tile (columns n1 .., 32 rows) times alpha into C: sixteen values per lane, all loads before
// the stores (independent accesses in flight instead of one read-modify-write at a time).  The epilogue's two warps per
// scheduler are bound by their instructions: with the rows' addresses formed once per unit and 16 bytes per access a
// chunk takes a fraction of the 416 that it took (245760 x 240 x 240 complex 277 us before, 180 now; 92160 x 160 x 160
// 74 and 55).
__device__ __forceinline__ void store16(const TcParams &p, const uint32_t (&r)[16], float *stg, const RowPtrs &rows, int lane,
                                        int n1) {
  if (p.store == STORE_PAIRS) {
    // rows of 16 floats, their 16-byte units permuted so that neither side conflicts; 8 rows x 64 bytes per instruction
    float4 *st4 = reinterpret_cast<float4 *>(stg);
    const int u = lane & 3, rs = lane >> 2, n = n1 + 4 * u;
#pragma unroll
    for (int j = 0; j < 4; ++j)
      st4[4 * lane + (j ^ ((lane >> 1) & 3))] = make_float4(__uint_as_float(r[4 * j]), __uint_as_float(r[4 * j + 1]),
                                                            __uint_as_float(r[4 * j + 2]), __uint_as_float(r[4 * j + 3]));
    __syncwarp();
    const int64_t co = 2 * v2off(p.cv, n >> 1);
    float4 v[4];
    float *dst[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const int rl = 8 * k + rs;
      v[k] = st4[4 * rl + (u ^ ((rl >> 1) & 3))];
      dst[k] = rows.p[k] && n < p.N ? rows.p[k] + co : nullptr;
    }
    __syncwarp();
#pragma unroll
    for (int k = 0; k < 4; ++k)
      v[k] = make_float4(p.ar * v[k].x - p.ai * v[k].y, p.ar * v[k].y + p.ai * v[k].x, p.ar * v[k].z - p.ai * v[k].w,
                         p.ar * v[k].w + p.ai * v[k].z);
    if (p.atomic) {
#pragma unroll
      for (int k = 0; k < 4; ++k)
        if (dst[k]) atomicAdd(reinterpret_cast<float4 *>(dst[k]), v[k]);
      return;
    }
    if (p.accumulate) {
      float4 old[4];
#pragma unroll
      for (int k = 0; k < 4; ++k) old[k] = dst[k] ? *reinterpret_cast<const float4 *>(dst[k]) : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        v[k].x += old[k].x;
        v[k].y += old[k].y;
        v[k].z += old[k].z;
        v[k].w += old[k].w;
      }
    }
#pragma unroll
    for (int k = 0; k < 4; ++k)
      if (dst[k]) *reinterpret_cast<float4 *>(dst[k]) = v[k];
    return;
  }
  float *dst[8];
  float2 val[8];
  if (p.store == STORE_COLS) {
    // stage rows, then 4 rows x 8 complex per instruction (64 contiguous bytes per row)
    float2 *srow = reinterpret_cast<float2 *>(stg + lane * EPI_PITCH);
#pragma unroll
    for (int j = 0; j < 8; ++j) srow[j] = make_float2(__uint_as_float(r[2 * j]), __uint_as_float(r[2 * j + 1]));
    __syncwarp();
    const int jj = lane & 7, rs = lane >> 3, n = n1 + 2 * jj;
    const int64_t co = 2 * v2off(p.cv, n >> 1);
#pragma unroll
    for (int k = 0; k < 8; ++k) {
      val[k] = reinterpret_cast<const float2 *>(stg + (4 * k + rs) * EPI_PITCH)[jj];
      dst[k] = rows.p[k] && n < p.N ? rows.p[k] + co : nullptr;
    }
    __syncwarp();
  } else {
#pragma unroll
    for (int k = 0; k < 8; ++k) {
      const int n = n1 + 2 * k;
      val[k] = make_float2(__uint_as_float(r[2 * k]), __uint_as_float(r[2 * k + 1]));
      dst[k] = rows.p[0] && n < p.N ? rows.p[0] + 2 * v2off(p.cv, n >> 1) : nullptr;
    }
  }
#pragma unroll
  for (int k = 0; k < 8; ++k)
    val[k] = make_float2(p.ar * val[k].x - p.ai * val[k].y, p.ar * val[k].y + p.ai * val[k].x);
  if (p.atomic) {
#pragma unroll
    for (int k = 0; k < 8; ++k)
      if (dst[k]) {
        atomicAdd(dst[k], val[k].x);
        atomicAdd(dst[k] + 1, val[k].y);
      }
    return;
  }
  if (p.accumulate) {
    float2 old[8];
#pragma unroll
    for (int k = 0; k < 8; ++k) old[k] = dst[k] ? *reinterpret_cast<const float2 *>(dst[k]) : make_float2(0.f, 0.f);
#pragma unroll
    for (int k = 0; k < 8; ++k) val[k] = make_float2(val[k].x + old[k].x, val[k].y + old[k].y);
  }
#pragma unroll
  for (int k = 0; k < 8; ++k)
    if (dst[k]) *reinterpret_cast<float2 *>(dst[k]) = val[k];
}

// The same chunk compared with p.tau instead (tc_magnitude_sums): a column of 32 sums makes one word per ballot, and lane
// 4 c + k stores word k of complex column c.
__device__ __forceinline__ void check16(const TcParams &p, const uint32_t (&r)[16], int row0, int lane, int n1) {
  uint32_t w = 0;
#pragma unroll
  for (int k = 0; k < 16; ++k) {
    const float s = __uint_as_float(r[k]);
    const uint32_t reach = __ballot_sync(0xffffffffu, s >= p.tau), some = __ballot_sync(0xffffffffu, s != 0.f);
    if (lane == 4 * (k >> 1) + (k & 1)) w = reach;
    if (lane == 4 * (k >> 1) + 2 + (k & 1)) w = some;
  }
  const int col = (n1 >> 1) + (lane >> 2);
  if (row0 >= p.M || 2 * col >= p.N) return;
  p.words[4 * ((int64_t)(row0 >> 5) * (p.N >> 1) + col) + (lane & 3)] = w;
}
struct NoRows {
  __device__ __forceinline__ NoRows(const TcParams &, int, int) {}
};
template <bool CHECK> using Rows = std::conditional_t<CHECK, NoRows, RowPtrs>;

// CHECK: the sums are compared (check16), not stored
template <int KIND, bool CHECK>
__global__ void __launch_bounds__(320, 1)
    tc_gemm_kernel(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmB,
                   TcParams p) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t *smem = (uint8_t *)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
  constexpr int BK = BKB / (KIND == TC_BF16 ? 2 : 4);  // operand elements per K block
  const int BN = p.BN;
  uint8_t *sA = smem;
  uint8_t *sB = smem + STAGES * BM * BKB;
  float *stage = (float *)(smem + STAGES * (BM + BN) * BKB);  // 8 warps x 32 rows x EPI_PITCH
  // barriers: full[S], empty[S], tfull[2], tempty[2], drain
  uint64_t *bars = (uint64_t *)(stage + 8 * 32 * EPI_PITCH);
  uint64_t *full = bars, *empty = bars + STAGES, *tfull = bars + 2 * STAGES, *tempty = tfull + 2,
           *drain = tempty + 2;
  uint32_t *tslot = (uint32_t *)(drain + 1);
  int *issued = (int *)(tslot + 1);  // K blocks loaded (producer)
  int *consumed = issued + 1;        // K blocks whose full barrier the MMA warp passed
  volatile int *abort_flag = issued + 2;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int units = p.ntiles * p.splits;
  const int nk_all = (p.K + BK - 1) / BK;
  // accumulator columns: one buffer per power of two >= BN, two buffers
  const uint32_t half = BN <= 32 ? 32u : BN <= 64 ? 64u : BN <= 128 ? 128u : 256u;
  const uint32_t tcols = 2 * half;

  if (threadIdx.x == 0) {
    for (int s = 0; s < STAGES; ++s) {
      asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(su32(full + s)) : "memory");
      asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(su32(empty + s)) : "memory");
    }
    for (int b = 0; b < 2; ++b) {
      asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(su32(tfull + b)) : "memory");
      asm volatile("mbarrier.init.shared::cta.b64 [%0], 8;" ::"r"(su32(tempty + b)) : "memory");
    }
    asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(su32(drain)) : "memory");
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(&tmA)) : "memory");
    asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(&tmB)) : "memory");
    issued[0] = 0;
    consumed[0] = 0;
    *abort_flag = 0;
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(su32(tslot)),
                 "r"(tcols)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tmem = *tslot;

  if (warp == 0) {
    if (lane == 0) {
      // TMA producer: K blocks of every unit of this CTA, through the ring
      const uint32_t bytes = (uint32_t)(BM + BN) * BKB;
      int g = 0;
      bool ok = true;
      for (int u = blockIdx.x; u < units && ok; u += gridDim.x) {
        int mt, nt, sp;
        unit_coords(p, u, mt, nt, sp);
        const int kb0 = sp * p.kb_per_split;
        const int nk = max(0, min(nk_all - kb0, p.kb_per_split));
        for (int kb = 0; kb < nk; ++kb, ++g) {
          const int s = g % STAGES;
          const uint32_t ph = (uint32_t)(g / STAGES) & 1u;
          if (!mbar_wait_ab(su32(empty + s), ph ^ 1u, p.err, abort_flag)) { ok = false; break; }
          asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(su32(full + s)), "r"(bytes)
                       : "memory");
          tma_load_2d(sA + s * BM * BKB, &tmA, (kb0 + kb) * BK, mt * BM, su32(full + s));
          tma_load_2d(sB + s * BN * BKB, &tmB, (kb0 + kb) * BK, nt * BN, su32(full + s));
          issued[0] = g + 1;
        }
      }
    }
    __syncwarp();
  } else if (warp == 1) {
    if (lane == 0) {
      // MMA issuer: accumulator buffer it & 1 for the it-th unit of this CTA
      const uint32_t idesc = idesc_mma(KIND, BM, BN);
      int g = 0, it = 0;
      bool ok = true;
      for (int u = blockIdx.x; u < units && ok; u += gridDim.x, ++it) {
        int mt, nt, sp;
        unit_coords(p, u, mt, nt, sp);
        const int kb0 = sp * p.kb_per_split;
        const int nk = max(0, min(nk_all - kb0, p.kb_per_split));
        const int buf = it & 1;
        if (!mbar_wait_ab(su32(tempty + buf), ((uint32_t)(it >> 1) & 1u) ^ 1u, p.err, abort_flag)) break;
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        const uint32_t dacc = tmem + (uint32_t)buf * half;
        for (int kb = 0; kb < nk; ++kb, ++g) {
          const int s = g % STAGES;
          const uint32_t ph = (uint32_t)(g / STAGES) & 1u;
          if (!mbar_wait_ab(su32(full + s), ph, p.err, abort_flag)) { ok = false; break; }
          consumed[0] = g + 1;
          asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
          const uint64_t da = sw128_desc(su32(sA + s * BM * BKB));
          const uint64_t db = sw128_desc(su32(sB + s * BN * BKB));
#pragma unroll
          for (int kk = 0; kk < BKB / 32; ++kk)  // 32 bytes of K per instruction (+2 in 16-byte units)
            mma_issue<KIND>(dacc, da + 2 * kk, db + 2 * kk, idesc, (kb | kk) != 0 ? 1u : 0u);
          mma_commit(su32(empty + s));
        }
        if (ok) mma_commit(su32(tfull + buf));  // arrives once this unit's MMAs have completed
      }
      // every MMA issued above has completed once this arrives
      mma_commit(su32(drain));
      mbar_wait(su32(drain), 0, p.err);
    }
    __syncwarp();
  } else {
    // epilogue warps 2..9: warps w and w + 4 share TMEM lane quarter w % 4 (rows 32 (w % 4)
    // .. + 31 of the tile) and take alternate 16-column chunks
    const int q = warp & 3, h = (warp - 2) >> 2;
    float *stg = stage + (warp - 2) * 32 * EPI_PITCH;
    int it = 0;
    for (int u = blockIdx.x; u < units; u += gridDim.x, ++it) {
      int mt, nt, sp;
      unit_coords(p, u, mt, nt, sp);
      const int buf = it & 1;
      const Rows<CHECK> rows(p, mt * BM + q * 32, lane);
      bool ok = mbar_wait_ab(su32(tfull + buf), (uint32_t)(it >> 1) & 1u, p.err, abort_flag);
      ok = __shfl_sync(0xffffffffu, ok ? 1 : 0, 0) != 0;
      if (!ok) break;
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
      const int n0 = nt * BN;
      const uint32_t tbase = tmem + ((uint32_t)(q * 32) << 16) + (uint32_t)buf * half;
      if (16 * h >= BN) {  // no chunk for this warp: release the buffer at once
        asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
        __syncwarp();
        if (lane == 0) mbar_arrive(su32(tempty + buf));
        continue;
      }
      for (int c0 = 16 * h; c0 < BN; c0 += 32) {
        uint32_t r[16];
        tmem_ld16(tbase + (uint32_t)c0, r);
        if (c0 + 32 >= BN) {
          // the accumulator buffer is free for the next unit once every warp has read its part
          asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
          __syncwarp();
          if (lane == 0) mbar_arrive(su32(tempty + buf));
        }
        if constexpr (CHECK) check16(p, r, mt * BM + q * 32, lane, n0 + c0);
        else store16(p, r, stg, rows, lane, n0 + c0);
      }
    }
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  if (threadIdx.x == 0 && consumed[0] < issued[0]) {
    // error path: drain TMA copies issued but never consumed (bounded)
    for (int g = consumed[0]; g < issued[0]; ++g)
      mbar_wait(su32(full + g % STAGES), (uint32_t)(g / STAGES) & 1u, p.err);
  }
  __syncthreads();
  if (warp == 1)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(tcols) : "memory");
}

// The same GEMM by pairs of CTAs: a pair computes 256 x BN tiles (BN a multiple of 32), each CTA loading its 128 rows
// of A and half the rows of B, and the first CTA issuing the MMAs for both.  A 128-row CTA of its own loads 94 bytes
// per clock and SM at BN = 256, which L2 does not keep up with; here it is 62, and the ring holds six blocks instead
// of four.  TFLOP/s before and now: 28800 x 7680 x 1200 complex 924 and 1144, 3840^3 860 and 1131, 7680^3 894 and 1187,
// 25600 x 2560 x 800 849 and 1063.
constexpr int PAIR_STAGES = 6;

template <int KIND, bool CHECK>
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(320, 1)
    tc_pair_kernel(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmB, TcParams p) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t *smem = (uint8_t *)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
  constexpr int BK = BKB / (KIND == TC_BF16 ? 2 : 4);  // operand elements per K block
  const int BN = p.BN, HN = BN / 2;
  uint8_t *sA = smem;
  uint8_t *sB = smem + PAIR_STAGES * BM * BKB;
  float *stage = (float *)(smem + PAIR_STAGES * (BM + HN) * BKB);  // 8 warps x 32 rows x EPI_PITCH
  // full and tempty are waited for in CTA 0 only; empty and tfull arrive in both
  uint64_t *bars = (uint64_t *)(stage + 8 * 32 * EPI_PITCH);
  uint64_t *full = bars, *empty = bars + PAIR_STAGES, *tfull = empty + PAIR_STAGES, *tempty = tfull + 2, *drain = tempty + 2;
  uint32_t *tslot = (uint32_t *)(drain + 1);
  int *issued = (int *)(tslot + 1), *consumed = issued + 1;
  volatile int *abort_flag = issued + 2;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const uint32_t rank = cta_rank();
  const int pair = blockIdx.x >> 1, npairs = gridDim.x >> 1;
  const int units = p.ntiles * p.splits, nk_all = (p.K + BK - 1) / BK;
  const uint32_t half = BN <= 32 ? 32u : BN <= 64 ? 64u : BN <= 128 ? 128u : 256u;
  const uint32_t tcols = 2 * half;

  if (threadIdx.x == 0) {
    for (int s = 0; s < PAIR_STAGES; ++s) {
      asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(su32(full + s)) : "memory");
      asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(su32(empty + s)) : "memory");
    }
    for (int b = 0; b < 2; ++b) {
      asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(su32(tfull + b)) : "memory");
      asm volatile("mbarrier.init.shared::cta.b64 [%0], 16;" ::"r"(su32(tempty + b)) : "memory");  // 8 warps of both CTAs
    }
    asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(su32(drain)) : "memory");
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(&tmA)) : "memory");
    asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(&tmB)) : "memory");
    issued[0] = 0;
    consumed[0] = 0;
    *abort_flag = 0;
  }
  __syncthreads();
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(su32(tslot)), "r"(tcols)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  pair_sync();  // both CTAs' barriers are initialised
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tmem = *tslot;

  if (warp == 0) {
    if (lane == 0) {
      // TMA producer of this CTA's half of the operands; both halves count on CTA 0's full barrier
      const uint32_t bytes = (uint32_t)(2 * BM + BN) * BKB;
      int g = 0, s = 0;
      uint32_t ph = 0;
      bool ok = true;
      for (int u = pair; u < units && ok; u += npairs) {
        int mt, nt, sp;
        unit_coords(p, u, mt, nt, sp);
        const int kb0 = sp * p.kb_per_split;
        const int nk = max(0, min(nk_all - kb0, p.kb_per_split));
        const int y_a = (2 * mt + (int)rank) * BM, y_b = nt * BN + (int)rank * HN;
        for (int kb = 0; kb < nk; ++kb, ++g) {
          if (!mbar_wait_ab(su32(empty + s), ph ^ 1u, p.err, abort_flag)) { ok = false; break; }
          const uint32_t fb = pair_addr(su32(full + s), 0);
          if (rank == 0)
            asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(su32(full + s)), "r"(bytes)
                         : "memory");
          tma_load_2d_pair(sA + s * BM * BKB, &tmA, (kb0 + kb) * BK, y_a, fb);
          tma_load_2d_pair(sB + s * HN * BKB, &tmB, (kb0 + kb) * BK, y_b, fb);
          issued[0] = g + 1;
          if (++s == PAIR_STAGES) { s = 0; ph ^= 1u; }
        }
      }
    }
    __syncwarp();
  } else if (warp == 1) {
    if (rank == 0 && elect_one()) {
      // MMA issuer of the pair: accumulator buffer it & 1 for the it-th unit
      const uint32_t idesc = idesc_mma(KIND, 2 * BM, BN);
      int g = 0, it = 0, s = 0;
      uint32_t ph = 0;
      bool ok = true;
      for (int u = pair; u < units && ok; u += npairs, ++it) {
        int mt, nt, sp;
        unit_coords(p, u, mt, nt, sp);
        const int kb0 = sp * p.kb_per_split;
        const int nk = max(0, min(nk_all - kb0, p.kb_per_split));
        const int buf = it & 1;
        if (!mbar_wait_ab(su32(tempty + buf), ((uint32_t)(it >> 1) & 1u) ^ 1u, p.err, abort_flag)) break;
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        const uint32_t dacc = tmem + (uint32_t)buf * half;
        for (int kb = 0; kb < nk; ++kb, ++g) {
          if (!mbar_wait_ab(su32(full + s), ph, p.err, abort_flag)) { ok = false; break; }
          consumed[0] = g + 1;
          asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
          const uint64_t da = sw128_desc(su32(sA + s * BM * BKB));
          const uint64_t db = sw128_desc(su32(sB + s * HN * BKB));
#pragma unroll
          for (int kk = 0; kk < BKB / 32; ++kk)  // 32 bytes of K per instruction (+2 in 16-byte units)
            mma_issue_pair<KIND>(dacc, da + 2 * kk, db + 2 * kk, idesc, (kb | kk) != 0 ? 1u : 0u);
          mma_commit_pair(su32(empty + s));
          if (++s == PAIR_STAGES) { s = 0; ph ^= 1u; }
        }
        if (ok) mma_commit_pair(su32(tfull + buf));  // arrives once this unit's MMAs have completed
      }
      // every MMA issued above has completed once this arrives
      mma_commit_pair(su32(drain));
      mbar_wait(su32(drain), 0, p.err);
    }
    __syncwarp();
  } else {
    // epilogue warps 2..9, as above, for this CTA's 128 rows
    const int q = warp & 3, h = (warp - 2) >> 2;
    float *stg = stage + (warp - 2) * 32 * EPI_PITCH;
    int it = 0;
    for (int u = pair; u < units; u += npairs, ++it) {
      int mt, nt, sp;
      unit_coords(p, u, mt, nt, sp);
      const int buf = it & 1;
      const Rows<CHECK> rows(p, (2 * mt + (int)rank) * BM + q * 32, lane);
      bool ok = mbar_wait_ab(su32(tfull + buf), (uint32_t)(it >> 1) & 1u, p.err, abort_flag);
      ok = __shfl_sync(0xffffffffu, ok ? 1 : 0, 0) != 0;
      if (!ok) break;
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
      const int n0 = nt * BN;
      const uint32_t tbase = tmem + ((uint32_t)(q * 32) << 16) + (uint32_t)buf * half;
      for (int c0 = 16 * h; c0 < BN; c0 += 32) {
        uint32_t r[16];
        tmem_ld16(tbase + (uint32_t)c0, r);
        if (c0 + 32 >= BN) {
          // the accumulator buffer is free for the next unit once every warp of both CTAs has read its part
          asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
          __syncwarp();
          if (lane == 0) mbar_arrive_cluster(pair_addr(su32(tempty + buf), 0));
        }
        if constexpr (CHECK) check16(p, r, (2 * mt + (int)rank) * BM + q * 32, lane, n0 + c0);
        else store16(p, r, stg, rows, lane, n0 + c0);
      }
    }
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  if (threadIdx.x == 0 && *abort_flag) {
    // error path: drain the copies of both CTAs that CTA 0 expected but never consumed (bounded); copies of CTA 1 that
    // CTA 0 never expected have no barrier to wait for, so both CTAs stay for 10 ms, which no copy takes
    if (rank == 0)
      for (int g = consumed[0]; g < issued[0]; ++g)
        mbar_wait(su32(full + g % PAIR_STAGES), (uint32_t)(g / PAIR_STAGES) & 1u, p.err);
    const unsigned long long t0 = gtime();
    while (gtime() - t0 < 10000000ull) {}
  }
  __syncthreads();
  pair_sync();  // neither CTA leaves (or frees its TMEM) while the other's MMAs, copies or arrivals may touch it
  if (warp == 1)
    asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(tcols) : "memory");
}

// The split modes in one pass: each 64-byte K block of A_hi, A_lo, B_hi, B_lo is loaded once and gives three products,
// hi.hi into the main accumulator, hi.lo + lo.hi into the correction accumulator (both 256 columns: one set of
// accumulators for tiles wider than 128 columns, two otherwise).  After CHAIN blocks the epilogue warps add both to
// FP32 registers and give the accumulators back; the unit's sums are written once.  Against one pass per term over
// rows of [hi | hi | lo], with every 64 blocks of a pass added to C by atomics, it loads a third less of A and B and
// touches C once.  TFLOP/s of MMAs before and now: 3840^3 complex 3xTF32 784 and 1049, bf16x3 1507 and 2029;
// 25600 x 2560 x 800 757 and 945, 1338 and 1712 (bound by the tensor cores).
constexpr int SPLIT_STAGES = 4;
constexpr int CHAIN = 128;  // 64-byte K blocks per accumulation chain

template <int KIND>
__global__ void __launch_bounds__(320, 1)
    tc_split_kernel(const __grid_constant__ CUtensorMap tmAh, const __grid_constant__ CUtensorMap tmAl,
                    const __grid_constant__ CUtensorMap tmBh, const __grid_constant__ CUtensorMap tmBl, TcParams p) {
  constexpr int KB = 64 / (KIND == TC_BF16 ? 2 : 4);  // operand elements per K block
  extern __shared__ uint8_t smem_raw[];
  uint8_t *smem = (uint8_t *)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
  const int BN = p.BN, a_bytes = BM * 64, b_bytes = BN * 64, slot = 2 * (a_bytes + b_bytes);
  float *stage = (float *)(smem + SPLIT_STAGES * slot);
  uint64_t *bars = (uint64_t *)(stage + 8 * 32 * EPI_PITCH);
  uint64_t *full = bars, *empty = bars + SPLIT_STAGES, *tfull = empty + SPLIT_STAGES, *tempty = tfull + 2, *drain = tempty + 2;
  uint32_t *tslot = (uint32_t *)(drain + 1);
  int *issued = (int *)(tslot + 1), *consumed = issued + 1;
  volatile int *abort_flag = issued + 2;
  const int warp = __shfl_sync(0xffffffffu, threadIdx.x >> 5, 0), lane = threadIdx.x & 31;
  const int units = p.ntiles * p.splits, nk_all = (p.K + KB - 1) / KB;
  const uint32_t half = BN <= 32 ? 32u : BN <= 64 ? 64u : BN <= 128 ? 128u : 256u;
  const int nbuf = half == 256u ? 1 : 2;
  const uint32_t tcols = 2 * half * (uint32_t)nbuf;

  if (threadIdx.x == 0) {
    for (int s = 0; s < SPLIT_STAGES; ++s) {
      asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(su32(full + s)) : "memory");
      asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(su32(empty + s)) : "memory");
    }
    for (int b = 0; b < 2; ++b) {
      asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(su32(tfull + b)) : "memory");
      asm volatile("mbarrier.init.shared::cta.b64 [%0], 8;" ::"r"(su32(tempty + b)) : "memory");
    }
    asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(su32(drain)) : "memory");
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    issued[0] = 0;
    consumed[0] = 0;
    *abort_flag = 0;
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(su32(tslot)), "r"(tcols)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tmem = *tslot;

  if (warp == 0) {
    if (lane == 0) {
      int g = 0;
      bool ok = true;
      for (int u = blockIdx.x; u < units && ok; u += gridDim.x) {
        int mt, nt, sp;
        unit_coords(p, u, mt, nt, sp);
        const int kb0 = sp * p.kb_per_split, kb1 = min(nk_all, kb0 + p.kb_per_split);
        for (int kb = kb0; kb < kb1; ++kb, ++g) {
          const int s = g % SPLIT_STAGES;
          if (!mbar_wait_ab(su32(empty + s), ((uint32_t)(g / SPLIT_STAGES) & 1u) ^ 1u, p.err, abort_flag)) { ok = false; break; }
          asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(su32(full + s)), "r"((uint32_t)slot)
                       : "memory");
          uint8_t *d = smem + s * slot;
          tma_load_2d(d, &tmAh, kb * KB, mt * BM, su32(full + s));
          tma_load_2d(d + 2 * a_bytes, &tmBh, kb * KB, nt * BN, su32(full + s));
          tma_load_2d(d + 2 * a_bytes + b_bytes, &tmBl, kb * KB, nt * BN, su32(full + s));
          tma_load_2d(d + a_bytes, &tmAl, kb * KB, mt * BM, su32(full + s));
          issued[0] = g + 1;
        }
      }
    }
    __syncwarp();
  } else if (warp == 1) {
    if (lane == 0) {
      const uint32_t idesc = idesc_mma(KIND, BM, BN), base = sw64_lo(su32(smem));
      const uint32_t al = (uint32_t)a_bytes >> 4, bh = 2 * al, bl = bh + ((uint32_t)b_bytes >> 4);
      int g = 0, it = 0;  // K blocks, accumulation chains
      bool ok = true;
      for (int u = blockIdx.x; u < units && ok; u += gridDim.x) {
        int mt, nt, sp;
        unit_coords(p, u, mt, nt, sp);
        const int kb0 = sp * p.kb_per_split, kb1 = min(nk_all, kb0 + p.kb_per_split);
        for (int c0 = kb0; c0 < kb1 && ok; c0 += CHAIN, ++it) {
          const int buf = nbuf == 1 ? 0 : it & 1, use = nbuf == 1 ? it : it >> 1;
          if (!mbar_wait_ab(su32(tempty + buf), ((uint32_t)use & 1u) ^ 1u, p.err, abort_flag)) { ok = false; break; }
          asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
          const uint32_t dm = tmem + (uint32_t)buf * 2 * half, dc = dm + half;
          const int c1 = min(kb1, c0 + CHAIN);
          for (int kb = c0; kb < c1; ++kb, ++g) {
            const int s = g % SPLIT_STAGES;
            if (!mbar_wait_ab(su32(full + s), (uint32_t)(g / SPLIT_STAGES) & 1u, p.err, abort_flag)) { ok = false; break; }
            consumed[0] = g + 1;
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            const uint32_t sb = base + ((uint32_t)(s * slot) >> 4);
            const bool acc = kb > c0;
            mma_sw64<KIND>(dm, sb, sb + bh, idesc, acc);
            mma_sw64<KIND>(dm, sb + 2, sb + bh + 2, idesc, true);
            mma_sw64<KIND>(dc, sb, sb + bl, idesc, acc);
            mma_sw64<KIND>(dc, sb + 2, sb + bl + 2, idesc, true);
            mma_sw64<KIND>(dc, sb + al, sb + bh, idesc, true);
            mma_sw64<KIND>(dc, sb + al + 2, sb + bh + 2, idesc, true);
            mma_commit(su32(empty + s));
          }
          if (ok) mma_commit(su32(tfull + buf));
        }
      }
      mma_commit(su32(drain));
      mbar_wait(su32(drain), 0, p.err);
    }
    __syncwarp();
  } else {
    const int q = warp & 3, h = (warp - 2) >> 2;
    float *stg = stage + (warp - 2) * 32 * EPI_PITCH;
    int it = 0;
    bool ok = true;
    for (int u = blockIdx.x; u < units && ok; u += gridDim.x) {
      int mt, nt, sp;
      unit_coords(p, u, mt, nt, sp);
      const int kb0 = sp * p.kb_per_split, kb1 = min(nk_all, kb0 + p.kb_per_split);
      float sum[8][16];  // columns 16 h + 32 j + c of the warp's rows
      for (int c0 = kb0; c0 < kb1; c0 += CHAIN, ++it) {
        const int buf = nbuf == 1 ? 0 : it & 1, use = nbuf == 1 ? it : it >> 1;
        ok = __all_sync(0xffffffffu, mbar_wait_ab(su32(tfull + buf), (uint32_t)use & 1u, p.err, abort_flag));
        if (!ok) break;
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        const uint32_t tb = tmem + ((uint32_t)(q * 32) << 16) + (uint32_t)buf * 2 * half;
#pragma unroll
        for (int j = 0; j < 8; ++j) {
          const int c = 16 * h + 32 * j;
          if (c < BN) {
            uint32_t x[16];
            tmem_ld16(tb + half + (uint32_t)c, x);
#pragma unroll
            for (int k = 0; k < 16; ++k) sum[j][k] = __uint_as_float(x[k]) + (c0 == kb0 ? 0.f : sum[j][k]);
            tmem_ld16(tb + (uint32_t)c, x);
#pragma unroll
            for (int k = 0; k < 16; ++k) sum[j][k] += __uint_as_float(x[k]);
          }
        }
        asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
        __syncwarp();
        if (lane == 0) mbar_arrive(su32(tempty + buf));
      }
      if (!ok) break;
      // a rolled loop over the chunks, the front one of the registers each time
#pragma unroll 1
      for (int c = 16 * h; c < BN; c += 32) {
        uint32_t r[16];
#pragma unroll
        for (int k = 0; k < 16; ++k) r[k] = __float_as_uint(sum[0][k]);
        const RowPtrs rows(p, mt * BM + q * 32, lane);  // (kept over the loop they would spill)
        store16(p, r, stg, rows, lane, nt * BN + c);
#pragma unroll
        for (int j = 0; j < 7; ++j)
#pragma unroll
          for (int k = 0; k < 16; ++k) sum[j][k] = sum[j + 1][k];
      }
    }
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  if (threadIdx.x == 0 && consumed[0] < issued[0])  // error path: drain copies issued but never consumed (bounded)
    for (int g = consumed[0]; g < issued[0]; ++g)
      mbar_wait(su32(full + g % SPLIT_STAGES), (uint32_t)(g / SPLIT_STAGES) & 1u, p.err);
  __syncthreads();
  if (warp == 1)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(tcols) : "memory");
}

// A wait that nothing completes, bounded by timeout_ns (self-test of the give-up path).
__global__ void wait_never_kernel(unsigned long long timeout_ns, int *err) {
  __shared__ __align__(8) uint64_t bar;
  if (threadIdx.x == 0) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(su32(&bar)) : "memory");
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    const unsigned long long t0 = gtime();
    while (!mbar_try(su32(&bar), 0)) {
      if (gtime() - t0 > timeout_ns) {
        atomicExch(err, 1);
        break;
      }
    }
  }
  __syncthreads();
}

// ---------------- operand preparation ----------------
// Source contiguous along k (or along neither): a thread takes two neighbouring k of one row, TX threads along k and
// 256 / TX rows per block, so that rows are written in 16-byte pieces and an entry costs no division by the row
// length (92160 x 160 complex, TF32 columns: 60 us; one entry per thread in flat order took 80).
template <int KIND, bool ISB>
__global__ void __launch_bounds__(256) prep_rows_kernel(const float2 *__restrict__ src, View2 rv, View2 kv, int64_t R, int64_t K,
                                                        int64_t Kp, int tx, int seg, typename TcElem<KIND>::T *__restrict__ dst,
                                                        int64_t ldd) {
  const int x = threadIdx.x % tx, y = threadIdx.x / tx, ty = 256 / tx;
  for (int64_t r = (int64_t)blockIdx.x * ty + y; r < R; r += (int64_t)gridDim.x * ty) {
    const float2 *row = src + v2off(rv, r);
    for (int64_t k = 2 * (int64_t)(blockIdx.y * tx + x); k < Kp; k += 2 * (int64_t)tx * gridDim.y) {
      float2 v[2];
#pragma unroll
      for (int c = 0; c < 2; ++c) v[c] = k + c < K ? row[v2off(kv, k + c)] : make_float2(0.f, 0.f);
      if (ISB) tc_put_b_pair<KIND>(dst + (2 * r) * ldd, dst + (2 * r + 1) * ldd, k, Kp, seg, v[0], v[1]);
      else tc_put_a_pair<KIND>(dst + r * ldd, k, Kp, seg, v[0], v[1]);
    }
  }
}

// Transposing preparation: the source is contiguous along m (A) or n (B) and strided along
// k; 32 x 32 tiles through shared memory so that reads and writes are both coalesced.
template <int KIND>
__global__ void prep_tiled_kernel(const float2 *src, View2 mnv, View2 kv, int64_t MN, int64_t K, int64_t Kp, int seg,
                                  int isB, typename TcElem<KIND>::T *dst, int64_t ldd) {
  __shared__ float2 tile[32][33];
  const int64_t tmn = (MN + 31) / 32, tk = (Kp + 31) / 32;
  for (int64_t t = blockIdx.x; t < tmn * tk; t += gridDim.x) {
    const int64_t mn0 = (t % tmn) * 32, k0 = (t / tmn) * 32;
    for (int r = threadIdx.y; r < 32; r += blockDim.y) {
      const int64_t mn = mn0 + threadIdx.x, k = k0 + r;
      float2 v = make_float2(0.f, 0.f);
      if (mn < MN && k < K) v = src[v2off(mnv, mn) + v2off(kv, k)];
      tile[r][threadIdx.x] = v;
    }
    __syncthreads();
    for (int r = threadIdx.y; r < 32; r += blockDim.y) {
      const int64_t mn = mn0 + r, k = k0 + threadIdx.x;
      if (mn < MN && k < Kp) {
        const float2 v = tile[threadIdx.x][r];
        if (!isB) tc_put_a<KIND>(dst + mn * ldd, k, Kp, seg, v);
        else tc_put_b<KIND>(dst + (2 * mn) * ldd, dst + (2 * mn + 1) * ldd, k, Kp, seg, v);
      }
    }
    __syncthreads();
  }
}

PFN_cuTensorMapEncodeTiled_v12000 g_encode = nullptr;
constexpr int kMaxDevs = 64;
int *g_err_dev[kMaxDevs] = {};  // bounded-wait flag, one per device
std::mutex g_dev_mu;

std::once_flag g_enc_once;

void fetch_encoder() {
  // the driver entry point is fetched through the runtime, so the library does not link
  // against libcuda itself (it still loads on machines without a driver)
  cudaDriverEntryPointQueryResult q;
  void *fn = nullptr;
  CCLR_CUDA(cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &fn, 12000, cudaEnableDefault, &q));
  if (q != cudaDriverEntryPointSuccess || !fn) throw Error(4, "cuTensorMapEncodeTiled not available");
  g_encode = (PFN_cuTensorMapEncodeTiled_v12000)fn;
}

int current_device() {
  int dev = 0;
  CCLR_CUDA(cudaGetDevice(&dev));
  CCLR_REQUIRE(dev >= 0 && dev < kMaxDevs, "device ordinal beyond 63");
  return dev;
}

// raises the dynamic shared-memory limit of every kernel instantiation on the current device
void set_smem_limits() {
  CCLR_CUDA(cudaFuncSetAttribute(tc_gemm_kernel<TC_TF32, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024));
  CCLR_CUDA(cudaFuncSetAttribute(tc_gemm_kernel<TC_BF16, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024));
  CCLR_CUDA(cudaFuncSetAttribute(tc_pair_kernel<TC_TF32, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024));
  CCLR_CUDA(cudaFuncSetAttribute(tc_pair_kernel<TC_BF16, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024));
  CCLR_CUDA(cudaFuncSetAttribute(tc_gemm_kernel<TC_BF16, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024));
  CCLR_CUDA(cudaFuncSetAttribute(tc_pair_kernel<TC_BF16, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024));
  CCLR_CUDA(cudaFuncSetAttribute(tc_split_kernel<TC_TF32>, cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024));
  CCLR_CUDA(cudaFuncSetAttribute(tc_split_kernel<TC_BF16>, cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024));
}

// The current device's wait flag; the first use on a device allocates and clears it and raises
// the kernel's shared-memory limit there.
int *device_err() {
  const int dev = current_device();
  std::lock_guard<std::mutex> lock(g_dev_mu);
  if (!g_err_dev[dev]) {
    std::call_once(g_enc_once, fetch_encoder);
    int *p = nullptr;
    CCLR_CUDA(cudaMalloc(&p, sizeof(int)));
    CCLR_CUDA(cudaMemset(p, 0, sizeof(int)));
    set_smem_limits();
    g_err_dev[dev] = p;
  }
  return g_err_dev[dev];
}

// 2-D tensor map over a row-major operand (rows x cols elements, ld elements apart), boxes of
// box_bytes of K (one 128- or 64-byte swizzle row) by box_rows rows
CUtensorMap make_map(const void *base, int64_t rows, int64_t cols, int64_t ld, int box_rows, int box_bytes, int kind) {
  CUtensorMap m;
  const int64_t es = tc_esize(kind);
  cuuint64_t gdim[2] = {(cuuint64_t)cols, (cuuint64_t)rows};
  cuuint64_t gstride[1] = {(cuuint64_t)(ld * es)};
  cuuint32_t box[2] = {(cuuint32_t)(box_bytes / es), (cuuint32_t)box_rows};
  cuuint32_t estr[2] = {1, 1};
  CUresult r = g_encode(&m, kind == TC_BF16 ? CU_TENSOR_MAP_DATA_TYPE_BFLOAT16 : CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 2,
                        (void *)base, gdim, gstride, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
                        box_bytes == 64 ? CU_TENSOR_MAP_SWIZZLE_64B : CU_TENSOR_MAP_SWIZZLE_128B,
                        CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  if (r != CUDA_SUCCESS) throw Error(4, "cuTensorMapEncodeTiled failed: " + std::to_string((int)r));
  return m;
}

int num_sms() {
  int dev = 0, n = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess ||
      n <= 0) {
    (void)cudaGetLastError();
    return 152;
  }
  return n;
}

unsigned grid1d(int64_t n) {
  return (unsigned)std::max<int64_t>(1, std::min<int64_t>((n + 255) / 256, 152 * 32));
}

template <int KIND>
void prep_launch(const void *src, View2 mv, View2 kv, int64_t MN, int64_t K, int seg, int isB, void *dst, int64_t ldd,
                 cudaStream_t st) {
  using T = typename TcElem<KIND>::T;
  const int64_t Kp = ldd / (2 * seg);
  const bool tiled = kv.sin != 1 && mv.sin == 1;
  if (tiled) {
    const int64_t nt = ((MN + 31) / 32) * ((Kp + 31) / 32);
    prep_tiled_kernel<KIND><<<(unsigned)std::min<int64_t>(nt, 152 * 64), dim3(32, 8), 0, st>>>(
        (const float2 *)src, mv, kv, MN, K, Kp, seg, isB, (T *)dst, ldd);
  } else {
    int tx = 2;
    while (tx < 256 && 2 * tx < Kp) tx *= 2;
    // (k pairs beyond one pass of tx over blockIdx.y; rows over blockIdx.x; about 32 blocks per SM)
    const int64_t gy = std::min<int64_t>((Kp + 2 * tx - 1) / (2 * tx), 152 * 32);
    const int64_t gx = std::max<int64_t>(1, std::min<int64_t>((MN * tx + 255) / 256, (152 * 32 + gy - 1) / gy));
    const dim3 g((unsigned)gx, (unsigned)gy);
    if (isB) prep_rows_kernel<KIND, true><<<g, 256, 0, st>>>((const float2 *)src, mv, kv, MN, K, Kp, tx, seg, (T *)dst, ldd);
    else prep_rows_kernel<KIND, false><<<g, 256, 0, st>>>((const float2 *)src, mv, kv, MN, K, Kp, tx, seg, (T *)dst, ldd);
  }
}

}  // namespace

void tc_prep_a2(const void *A, View2 mv, View2 kv, int64_t M, int64_t K, int seg, int kind, void *dst, int64_t ldd,
                cudaStream_t st) {
  CCLR_REQUIRE(ldd >= 2 * K * seg && ldd % (2 * seg) == 0, "tc_prep_a: row too short");
  if (kind == TC_BF16) prep_launch<TC_BF16>(A, mv, kv, M, K, seg, 0, dst, ldd, st);
  else prep_launch<TC_TF32>(A, mv, kv, M, K, seg, 0, dst, ldd, st);
  count_launch();
  CCLR_CUDA(cudaGetLastError());
}

void tc_prep_b2(const void *B, View2 kv, View2 nv, int64_t K, int64_t N, int seg, int kind, void *dst, int64_t ldd,
                cudaStream_t st) {
  CCLR_REQUIRE(ldd >= 2 * K * seg && ldd % (2 * seg) == 0, "tc_prep_b: row too short");
  if (kind == TC_BF16) prep_launch<TC_BF16>(B, nv, kv, N, K, seg, 1, dst, ldd, st);
  else prep_launch<TC_TF32>(B, nv, kv, N, K, seg, 1, dst, ldd, st);
  count_launch();
  CCLR_CUDA(cudaGetLastError());
}

void tc_prep_a(const void *A, int64_t sam, int64_t sak, int64_t M, int64_t K, int seg, int kind, void *dst,
               int64_t ldd, cudaStream_t st) {
  tc_prep_a2(A, view1(sam), view1(sak), M, K, seg, kind, dst, ldd, st);
}

void tc_prep_b(const void *B, int64_t sbk, int64_t sbn, int64_t K, int64_t N, int seg, int kind, void *dst,
               int64_t ldd, cudaStream_t st) {
  tc_prep_b2(B, view1(sbk), view1(sbn), K, N, seg, kind, dst, ldd, st);
}

// Launch configuration: tile width BN, K splits and raster band (0 = the rule's choice), and whether pairs of CTAs take
// 256-row tiles (read with BN > 0 only).
struct TcCfg {
  int BN = 0, splits = 0, band = 0;
  bool pair = false;
};

// Clocks of a 128-byte K block of a BN-wide tile: four MMAs of BN / 2, but an MMA never takes less than 93, which
// makes narrow tiles dear (M = N = K = 5056 complex 497 TFLOP/s in 128-wide tiles, 800 in 256-wide ones), and in the
// one-pass kernels not less than L2 takes to feed an SM, about 84 bytes per clock.
constexpr int64_t block_clocks(int BN, bool pair, bool split) {
  const int64_t mma = 4 * std::max(BN / 2, 93), feed = (BM + (pair ? BN / 2 : BN)) * BKB / 84;
  return split ? 3 * mma : std::max(mma, feed);
}
constexpr int64_t epilogue_clocks(int BN) { return 32 * BN; }

// Time in clocks of M x N tiles of width BN with K in `splits`, each SM (or pair of SMs) taking every num_sms-th (or
// num_sms / 2-th) unit: whole waves of the longer of main loop and epilogue, and the last epilogue.
static int64_t cfg_clocks(int64_t M, int64_t Nreal, int nk, int BN, bool pair, int splits, int nsm, bool split) {
  const int64_t rows = pair ? 2 * BM : BM, slots = pair ? std::max(nsm / 2, 1) : nsm;
  const int64_t units = ((M + rows - 1) / rows) * ((Nreal + BN - 1) / BN) * splits, waves = (units + slots - 1) / slots;
  const int64_t main = (nk + splits - 1) / splits * block_clocks(BN, pair, split), epi = epilogue_clocks(BN) * (splits > 1 ? 2 : 1);
  return waves * std::max(main, epi) + epi;
}

// the cheapest number of K splits of at least eight blocks (1 unless it gains a twentieth)
static int best_splits(int64_t M, int64_t Nreal, int nk, int BN, bool pair, bool allow, int nsm, bool split) {
  int best = 1;
  if (!allow) return best;
  int64_t t = cfg_clocks(M, Nreal, nk, BN, pair, best, nsm, split);
  const int64_t rows = pair ? 2 * BM : BM, tiles = ((M + rows - 1) / rows) * ((Nreal + BN - 1) / BN);
  const int most = (int)std::min<int64_t>(nk / 8, std::max<int64_t>(32, (pair ? nsm : 2 * nsm) / std::max<int64_t>(tiles, 1)));
  for (int s = 2; s <= most; ++s) {
    const int64_t c = cfg_clocks(M, Nreal, nk, BN, pair, s, nsm, split);
    if (c * 20 < t * 19) { t = c; best = s; }
  }
  return best;
}

// the rule's tile width and splits: the cheapest by cfg_clocks, a narrower tile where it gains a tenth (per column it
// loads more of A: 25600 x 2560 x 800 complex 838 TFLOP/s at 256, 732 at 208, which would save half a wave); then
// pairs of CTAs for one pass if their best tile gains a twentieth (92160 x 160 x 160, bound by its output: 76 us by
// single CTAs, 80 by pairs)
static TcCfg rule_cfg(int64_t M, int64_t Nreal, int nk, bool allow, int nsm, bool split) {
  TcCfg r, q;
  int64_t t = -1, tq = -1;
  if (Nreal <= 256) {
    r.BN = (int)((Nreal + 15) / 16 * 16);
    r.splits = best_splits(M, Nreal, nk, r.BN, false, allow, nsm, split);
    t = cfg_clocks(M, Nreal, nk, r.BN, false, r.splits, nsm, split);
  } else {
    for (int bn = 256; bn >= 128; bn -= 16) {
      const int s = best_splits(M, Nreal, nk, bn, false, allow, nsm, split);
      const int64_t c = cfg_clocks(M, Nreal, nk, bn, false, s, nsm, split);
      if (t < 0 || c * 10 < t * 9) { t = c; r.BN = bn; r.splits = s; }
    }
  }
  if (split || Nreal < 128 || M <= BM) return r;
  q.pair = true;
  for (int bn = 256; bn >= 128; bn -= 32) {
    if (bn > 128 && bn - 32 >= Nreal) continue;
    const int s = best_splits(M, Nreal, nk, bn, true, allow, nsm, split);
    const int64_t c = cfg_clocks(M, Nreal, nk, bn, true, s, nsm, split);
    if (tq < 0 || c * 10 < tq * 9) { tq = c; q.BN = bn; q.splits = s; }
  }
  return tq * 20 < t * 19 ? q : r;
}

struct TuneKey {
  int dev, kind, transposed;
  int64_t M, N, K;
  bool operator<(const TuneKey &o) const {
    return std::tie(dev, kind, transposed, M, N, K) < std::tie(o.dev, o.kind, o.transposed, o.M, o.N, o.K);
  }
};
struct TuneRec {
  TcCfg cfg, rule;
  float ms_best = 0.f, ms_rule = 0.f;
  int tried = 0;
};
std::mutex g_tune_mu;
std::map<TuneKey, TuneRec> g_tune;
thread_local bool g_tune_on = false;

// a_cols: operand elements A actually holds per row (<= Kreal; the rest reads as zero).
// lda, ldb, Kreal in elements of the operand type; split: rows of two segments (hi, lo) of Kreal elements.  cfg
// overrides the rules; *used receives the configuration launched.  prepare: makes the list of tiles of that configuration if
// there is none yet, and launches nothing (the list is allocated and copied, which a timed launch should not contain).
static void tc_launch(const void *A, int64_t lda, const void *B, int64_t ldb, int64_t M, int64_t Nreal, int64_t Kreal,
                      int kind, bool split, float *C, View2 rv, View2 cv, zc alpha, bool accumulate, int *err,
                      cudaStream_t st, int64_t a_cols, TcCfg cfg, TcCfg *used, UpperTiles *upper, bool prepare = false) {
  const int64_t es = tc_esize(kind), BK = BKB / es;
  const int nk = (int)((Kreal + BK - 1) / BK), nsm = num_sms();
  // K splits need an accumulating or plain output (split partial tiles are added atomically)
  const bool plain = rv.din == TC_ONE_LEVEL && cv.din == TC_ONE_LEVEL && cv.sin == 1;
  if (cfg.BN <= 0) {
    const int band = cfg.band;
    cfg = rule_cfg(M, Nreal, nk, accumulate || plain, nsm, split);
    cfg.band = band;
  } else if (cfg.splits <= 0) {
    cfg.splits = best_splits(M, Nreal, nk, cfg.BN, cfg.pair, accumulate || plain, nsm, split);
  }
  const int BN = cfg.BN, rows = cfg.pair ? 2 * BM : BM;
  int splits = std::min({cfg.splits, nk, 65535});
  TcParams p;
  p.M = (int)M;
  p.N = (int)Nreal;
  p.K = (int)Kreal;
  p.BN = BN;
  p.nMt = (int)((M + rows - 1) / rows);
  p.nNt = (int)((Nreal + BN - 1) / BN);
  // band of M tiles swept by N: as many A rows as take 32 MB (they stay in L2), and at least 20 tiles, which makes
  // the running tiles' block of C about square (M = N = K = 7680 complex: 4 tiles 839 TFLOP/s, 20 tiles 894)
  p.band = cfg.band > 0 ? std::min(cfg.band, p.nMt)
                        : (int)std::min<int64_t>(p.nMt, std::max<int64_t>(20 * BM / rows, (32ll << 20) / (rows * Kreal * es + 1)));
  const int64_t tiles = (int64_t)p.nMt * p.nNt;
  p.kb_per_split = (nk + splits - 1) / splits;
  splits = (nk + p.kb_per_split - 1) / p.kb_per_split;  // every split has at least one K block
  if (split) p.kb_per_split *= 2;                       // (64-byte blocks there)
  p.splits = splits;
  p.C = C;
  p.rv = rv;
  p.cv = cv;
  // lanes along columns when C's columns run contiguously (two at a time where they make whole 16-byte units), one lane
  // per row otherwise
  const bool two_r = rv.din != TC_ONE_LEVEL, two_c = cv.din != TC_ONE_LEVEL;
  const bool even = Nreal % 4 == 0 && (uintptr_t)C % 16 == 0 && rv.sin % 2 == 0 && (!two_r || rv.sout % 2 == 0) &&
                    (!two_c || (cv.din % 2 == 0 && cv.sout % 2 == 0));
  p.store = cv.sin != 1 || (two_c && cv.din < 8) ? STORE_ROWS : even ? STORE_PAIRS : STORE_COLS;
  p.ar = (float)alpha.re;
  p.ai = (float)alpha.im;
  p.atomic = splits > 1 ? 1 : 0;
  p.accumulate = (accumulate || splits > 1) ? 1 : 0;
  p.err = err;
  p.ntiles = (int)tiles;
  p.list = upper ? upper->get(p.nMt, p.nNt, p.band, rows, BN / 2, 0, 0, M, st, &p.ntiles) : nullptr;
  if (prepare) return;
  if (splits > 1 && !accumulate) {
    CCLR_REQUIRE(rv.din == TC_ONE_LEVEL && cv.din == TC_ONE_LEVEL && cv.sin == 1,
                 "tc_gemm: split K without accumulation needs a plain C layout");
    CCLR_CUDA(cudaMemset2DAsync(C, (size_t)rv.sin * 8, 0, (size_t)Nreal * 4, (size_t)M, st));
  }
  const int64_t units = (int64_t)p.ntiles * splits;
  CCLR_REQUIRE(units < (1ll << 31), "tc_gemm: too many work units");
  static const bool trace = std::getenv("CCLR_TRACE") && std::getenv("CCLR_TRACE")[0] == '1';
  if (trace)
    std::fprintf(stderr, "cclr tc_gemm kind=%d M=%lld N=%lld K=%lld BN=%d pair=%d tiles=%lld splits=%d band=%d atomic=%d store=%d\n",
                 kind, (long long)M, (long long)Nreal, (long long)Kreal, BN, (int)cfg.pair, (long long)tiles, splits, p.band, p.atomic,
                 p.store);
  const unsigned grid = (unsigned)std::min<int64_t>(units, nsm);
  const size_t epi = (size_t)8 * 32 * EPI_PITCH * 4 + (2 * PAIR_STAGES + 5) * 8 + 16;
  if (split) {
    const char *Al = (const char *)A + Kreal * es, *Bl = (const char *)B + Kreal * es;
    const CUtensorMap ah = make_map(A, M, Kreal, lda, BM, 64, kind), al = make_map(Al, M, Kreal, lda, BM, 64, kind);
    const CUtensorMap bh = make_map(B, Nreal, Kreal, ldb, BN, 64, kind), bl = make_map(Bl, Nreal, Kreal, ldb, BN, 64, kind);
    const size_t smem = 1024 + (size_t)SPLIT_STAGES * 2 * (BM + BN) * 64 + epi;
    if (kind == TC_BF16) tc_split_kernel<TC_BF16><<<grid, 320, smem, st>>>(ah, al, bh, bl, p);
    else tc_split_kernel<TC_TF32><<<grid, 320, smem, st>>>(ah, al, bh, bl, p);
  } else {
    const CUtensorMap ma = make_map(A, M, a_cols < 0 ? Kreal : a_cols, lda, BM, BKB, kind);
    const CUtensorMap mb = make_map(B, Nreal, Kreal, ldb, cfg.pair ? BN / 2 : BN, BKB, kind);
    const size_t smem = 1024 + (cfg.pair ? (size_t)PAIR_STAGES * (BM + BN / 2) : (size_t)STAGES * (BM + BN)) * BKB + epi;
    if (cfg.pair) {
      const unsigned pairs = (unsigned)std::min<int64_t>(units, std::max(nsm / 2, 1));
      if (kind == TC_BF16) tc_pair_kernel<TC_BF16, false><<<2 * pairs, 320, smem, st>>>(ma, mb, p);
      else tc_pair_kernel<TC_TF32, false><<<2 * pairs, 320, smem, st>>>(ma, mb, p);
    } else if (kind == TC_BF16) tc_gemm_kernel<TC_BF16, false><<<grid, 320, smem, st>>>(ma, mb, p);
    else tc_gemm_kernel<TC_TF32, false><<<grid, 320, smem, st>>>(ma, mb, p);
  }
  count_launch();
  CCLR_CUDA(cudaGetLastError());
  if (used) {
    used->BN = BN;
    used->splits = splits;
    used->band = p.band;
    used->pair = cfg.pair;
  }
}

// Tiles as wide as 256 columns, by pairs of CTAs from 129 rows and 128 columns on; K in parts of at least four blocks where
// the tiles leave half the SMs idle.
bool tc_magnitude_sums(const void *A, int64_t lda, const void *B, int64_t ldb, int64_t M, int64_t Nreal, int64_t Kreal, float tau,
                       void *out, cudaStream_t st) {
  CCLR_REQUIRE(Nreal % 2 == 0 && lda % 8 == 0 && ldb % 8 == 0 && (uintptr_t)A % 16 == 0 && (uintptr_t)B % 16 == 0,
               "tc_magnitude_sums: operands must be whole 16-byte units");
  const int nsm = num_sms(), nk = (int)((Kreal + BKB / 2 - 1) / (BKB / 2));
  TcCfg cfg;
  cfg.pair = M > BM && Nreal >= 128;
  const int step = cfg.pair ? 32 : 16, rows = cfg.pair ? 2 * BM : BM, slots = cfg.pair ? std::max(nsm / 2, 1) : nsm;
  cfg.BN = (int)std::min<int64_t>(256, (Nreal + step - 1) / step * step);
  const int64_t tiles = ((M + rows - 1) / rows) * ((Nreal + cfg.BN - 1) / cfg.BN);
  cfg.splits = 2 * tiles <= slots ? std::max(1, std::min((int)(slots / tiles), nk / 4)) : 1;
  if (cfg.splits > 1) {
    tc_launch(A, lda, B, ldb, M, Nreal, Kreal, TC_BF16, false, (float *)out, view1(Nreal / 2), view1(1), zc(1.0), false,
              device_err(), st, -1, cfg, nullptr, nullptr);
    return false;
  }
  TcParams p = {};
  p.M = (int)M;
  p.N = (int)Nreal;
  p.K = (int)Kreal;
  p.BN = cfg.BN;
  p.nMt = (int)((M + rows - 1) / rows);
  p.nNt = (int)((Nreal + cfg.BN - 1) / cfg.BN);
  p.band = std::min(p.nMt, 20 * BM / rows);
  p.ntiles = (int)tiles;
  p.splits = 1;
  p.kb_per_split = nk;
  p.err = device_err();
  p.tau = tau;
  p.words = (uint32_t *)out;
  const CUtensorMap ma = make_map(A, M, Kreal, lda, BM, BKB, TC_BF16);
  const CUtensorMap mb = make_map(B, Nreal, Kreal, ldb, cfg.pair ? cfg.BN / 2 : cfg.BN, BKB, TC_BF16);
  const size_t smem = 1024 + (cfg.pair ? (size_t)PAIR_STAGES * (BM + cfg.BN / 2) : (size_t)STAGES * (BM + cfg.BN)) * BKB +
                      (size_t)8 * 32 * EPI_PITCH * 4 + (2 * PAIR_STAGES + 5) * 8 + 16;
  const unsigned grid = (unsigned)std::min<int64_t>(tiles, slots);
  if (cfg.pair) tc_pair_kernel<TC_BF16, true><<<2 * grid, 320, smem, st>>>(ma, mb, p);
  else tc_gemm_kernel<TC_BF16, true><<<grid, 320, smem, st>>>(ma, mb, p);
  count_launch();
  CCLR_CUDA(cudaGetLastError());
  return true;
}
// (2 tiles <= slots, tiles of 128 x 256 floats per SM)
int64_t tc_magnitude_sums_cap() { return (int64_t)num_sms() / 2 * BM * 256 * 4; }

// Candidate configurations around the rule's choice: other tile widths for wide outputs (each with its own best
// number of splits), more or fewer K splits, and the two extreme raster bands.
static std::vector<TcCfg> candidates(const TcCfg &rule, int64_t M, int64_t Nreal, int64_t Kreal, int kind, bool allow_split,
                                     bool split) {
  std::vector<TcCfg> c{rule};
  auto add = [&](TcCfg x) {
    for (const auto &y : c)
      if (y.BN == x.BN && y.splits == x.splits && y.band == x.band && y.pair == x.pair) return;
    c.push_back(x);
  };
  const int nk = (int)((Kreal + BKB / tc_esize(kind) - 1) / (BKB / tc_esize(kind)));
  if (Nreal > 256)
    for (int bn : {192, 256}) {
      TcCfg x = rule;
      x.BN = bn;
      x.splits = best_splits(M, Nreal, nk, bn, x.pair, allow_split, num_sms(), split);
      add(x);
    }
  if (rule.pair) {  // the same width by single CTAs
    TcCfg x = rule;
    x.pair = false;
    x.splits = best_splits(M, Nreal, nk, x.BN, false, allow_split, num_sms(), split);
    x.band = 0;
    add(x);
  }
  if (allow_split) {
    TcCfg x = rule;
    x.splits = std::max(1, rule.splits / 2); add(x);
    if (nk >= 16) { x.splits = std::min(nk / 4, 2 * rule.splits); add(x); }
  }
  const int rows = rule.pair ? 2 * BM : BM, nMt = (int)((M + rows - 1) / rows);
  if (nMt > 1) {
    TcCfg x = rule; x.band = 1; add(x);
    x.band = nMt; add(x);
  }
  return c;
}

static void tc_gemm_core(const void *A, int64_t lda, const void *B, int64_t ldb, int64_t M, int64_t Nreal,
                         int64_t Kreal, int kind, bool split, float *C, View2 rv, View2 cv, zc alpha, bool accumulate,
                         int *err, cudaStream_t st, int64_t a_cols = -1, UpperTiles *upper = nullptr) {
  if (M <= 0 || Nreal <= 0) return;
  const int64_t es = tc_esize(kind);
  CCLR_REQUIRE(Nreal % 2 == 0, "tc_gemm: real N must be even (complex pairs)");
  CCLR_REQUIRE((lda * es) % 16 == 0 && (ldb * es) % 16 == 0, "tc_gemm: row pitches must be multiples of 16 bytes");
  CCLR_REQUIRE(((uintptr_t)A % 16) == 0 && ((uintptr_t)B % 16) == 0, "tc_gemm: operands must be 16-byte aligned");
  CCLR_REQUIRE(M < (1ll << 31) && Nreal < (1ll << 31) && Kreal < (1ll << 31), "tc_gemm: dimension too large");
  const int transposed = (cv.sin == 1 && (cv.din == TC_ONE_LEVEL || cv.din >= 8)) ? 1 : 0;
  const TuneKey key{current_device(), kind, transposed + (upper ? 2 : 0) + (split ? 4 : 0), M, Nreal, Kreal};
  TcCfg cfg;
  bool have = false;
  {
    std::lock_guard<std::mutex> lock(g_tune_mu);
    auto it = g_tune.find(key);
    if (it != g_tune.end()) {
      cfg = it->second.cfg;
      have = true;
    }
  }
  cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
  CCLR_CUDA(cudaStreamIsCapturing(st, &cap));
  // Autotuning (first use of a shape while tuning is on, never inside a capture): every candidate
  // is timed with CUDA events on the real operands.  Outputs that are overwritten are tuned in
  // place (the launch below rewrites them); accumulated ones into a scratch block of the same
  // shape when it fits in 512 MB, else the rule stands.
  if (!have && g_tune_on && cap == cudaStreamCaptureStatusNone) {
    const size_t cbytes = (size_t)M * Nreal * 4;
    DevBuf scratch;
    float *Ct = C;
    View2 trv = rv, tcv = cv;
    bool ok = true;
    if (accumulate) {
      if (cbytes <= (512ull << 20)) {
        scratch.alloc(cbytes);
        Ct = scratch.as<float>();
        trv = view1(Nreal / 2);
        tcv = view1(1);
      } else {
        ok = false;
      }
    }
    TuneRec rec;
    if (ok) {
      TcCfg rule;
      tc_launch(A, lda, B, ldb, M, Nreal, Kreal, kind, split, Ct, trv, tcv, alpha, false, err, st, a_cols,
                TcCfg(), &rule, upper);
      rec.rule = rule;
      cudaEvent_t e0, e1;
      CCLR_CUDA(cudaEventCreate(&e0));
      CCLR_CUDA(cudaEventCreate(&e1));
      float best = 1e30f;
      // K splits need an accumulating or plain output (split partial tiles are added atomically)
      const bool plain = trv.din == TC_ONE_LEVEL && tcv.din == TC_ONE_LEVEL && tcv.sin == 1;
      for (const TcCfg &cand : candidates(rule, M, Nreal, Kreal, kind, accumulate || plain, split)) {
        TcCfg used;
        tc_launch(A, lda, B, ldb, M, Nreal, Kreal, kind, split, Ct, trv, tcv, alpha, false, err, st, a_cols, cand, nullptr,
                  upper, true);
        CCLR_CUDA(cudaEventRecord(e0, st));
        tc_launch(A, lda, B, ldb, M, Nreal, Kreal, kind, split, Ct, trv, tcv, alpha, false, err, st, a_cols,
                  cand, &used, upper);
        CCLR_CUDA(cudaEventRecord(e1, st));
        CCLR_CUDA(cudaEventSynchronize(e1));
        float ms = 0.f;
        CCLR_CUDA(cudaEventElapsedTime(&ms, e0, e1));
        if (rec.tried == 0) rec.ms_rule = ms;  // the first candidate is the rule's configuration
        ++rec.tried;
        if (ms < best) {
          best = ms;
          rec.cfg = used;
        }
      }
      rec.ms_best = best;
      CCLR_CUDA(cudaEventDestroy(e0));
      CCLR_CUDA(cudaEventDestroy(e1));
    } else {
      rec.cfg = TcCfg();
    }
    std::lock_guard<std::mutex> lock(g_tune_mu);
    g_tune[key] = rec;
    cfg = rec.cfg;
  }
  tc_launch(A, lda, B, ldb, M, Nreal, Kreal, kind, split, C, rv, cv, alpha, accumulate, err, st, a_cols, cfg,
            nullptr, upper);
}

void tc_gemm(const float *A, int64_t lda, const float *B, int64_t ldb, int64_t M, int64_t Nreal,
             int64_t Kreal, float *C, int64_t ldc_floats, zc alpha, bool accumulate, cudaStream_t st) {
  tc_gemm_core(A, lda, B, ldb, M, Nreal, Kreal, TC_TF32, false, C, view1(ldc_floats / 2), view1(1), alpha, accumulate,
               device_err(), st);
}

void tc_gemm_seg_v(const void *A, int64_t lda, const void *B, int64_t ldb, int64_t M, int64_t Nreal, int64_t Kseg,
                   int seg, int kind, float *C, View2 rv, View2 cv, zc alpha, bool accumulate, cudaStream_t st,
                   UpperTiles *upper) {
  tc_gemm_core(A, lda, B, ldb, M, Nreal, Kseg, kind, seg == 2, C, rv, cv, alpha, accumulate, device_err(), st, -1, upper);
}

void tc_gemm_a_inplace(const void *A, int64_t lda_cpx, int64_t K, const float *B, int64_t ldb, int64_t M,
                       int64_t Nreal, float *C, View2 rv, View2 cv, zc alpha, bool accumulate, cudaStream_t st) {
  tc_gemm_core(A, 2 * lda_cpx, B, ldb, M, Nreal, ldb, TC_TF32, false, C, rv, cv, alpha, accumulate, device_err(),
               st, 2 * K);
}

bool tc_a_inplace_ok(const void *A, int64_t lda_cpx, int64_t K) {
  return ((uintptr_t)A % 16) == 0 && lda_cpx % 2 == 0 && lda_cpx >= K && 8 * lda_cpx < (1ll << 40);
}

void tc_gemm_seg(const void *A, int64_t lda, const void *B, int64_t ldb, int64_t M, int64_t Nreal, int64_t Kseg,
                 int seg, int kind, float *C, int64_t ldc_floats, zc alpha, bool accumulate, cudaStream_t st,
                 UpperTiles *upper) {
  tc_gemm_seg_v(A, lda, B, ldb, M, Nreal, Kseg, seg, kind, C, view1(ldc_floats / 2), view1(1), alpha, accumulate, st, upper);
}

const uint32_t *UpperTiles::get(int nMt, int nNt, int band, int rows, int cols, int64_t m0, int64_t n0, int64_t M,
                                cudaStream_t st, int *n) {
  if (nMt > 0xffff || nNt > 0xffff) return nullptr;
  for (const auto &e : lists_)
    if (e->nMt == nMt && e->nNt == nNt && e->band == band && e->rows == rows && e->cols == cols && e->m0 == m0 &&
        e->n0 == n0 && e->M == M) {
      *n = e->n;
      return (const uint32_t *)e->buf.p;
    }
  cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
  CCLR_CUDA(cudaStreamIsCapturing(st, &cap));
  if (cap != cudaStreamCaptureStatusNone) return nullptr;
  std::vector<uint32_t> t;
  for (int b0 = 0; b0 < nMt; b0 += band)
    for (int nt = 0; nt < nNt; ++nt)
      for (int mt = b0; mt < std::min(nMt, b0 + band); ++mt) {
        const int64_t last_b = (std::min<int64_t>(M, m0 + (int64_t)(mt + 1) * rows) - 1) / v_;
        const int64_t first_a = (n0 + (int64_t)nt * cols) / v_;
        if (last_b > first_a) t.push_back((uint32_t)mt << 16 | (uint32_t)nt);
      }
  if (t.empty()) return nullptr;
  auto e = std::make_unique<List>();
  e->nMt = nMt; e->nNt = nNt; e->band = band; e->rows = rows; e->cols = cols;
  e->m0 = m0; e->n0 = n0; e->M = M;
  e->n = (int)t.size();
  try {
    e->buf.alloc(t.size() * sizeof(uint32_t));
  } catch (const Error &x) {
    if (x.status != 2) throw;
    return nullptr;  // no room: every tile is computed
  }
  CCLR_CUDA(cudaMemcpyAsync(e->buf.p, t.data(), e->buf.bytes, cudaMemcpyHostToDevice, st));
  CCLR_CUDA(cudaStreamSynchronize(st));  // t is pageable and goes out of scope
  lists_.push_back(std::move(e));
  *n = lists_.back()->n;
  return (const uint32_t *)lists_.back()->buf.p;
}

void tc_setup_device_flagged() {
  std::call_once(g_enc_once, fetch_encoder);
  set_smem_limits();
}

void tc_gemm_seg_flagged(const float *A, int64_t lda, const float *B, int64_t ldb, int64_t M, int64_t Nreal,
                         int64_t Kseg, int seg, float *C, int64_t ldc_floats, zc alpha, bool accumulate,
                         int *err, cudaStream_t st) {
  CCLR_REQUIRE(g_encode != nullptr, "tc_gemm_seg_flagged: tc_setup_device_flagged was not called");
  tc_gemm_core(A, lda, B, ldb, M, Nreal, Kseg, TC_TF32, seg == 2, C, view1(ldc_floats / 2), view1(1), alpha, accumulate,
               err, st);
}

int tc_selftest_timeout(int timeout_us, cudaStream_t st) {
  wait_never_kernel<<<1, 32, 0, st>>>((unsigned long long)timeout_us * 1000ull, device_err());
  count_launch();
  CCLR_CUDA(cudaGetLastError());
  return tc_error(st);
}

int *tc_device_err() { return device_err(); }
int tc_num_sms() { return num_sms(); }
CUtensorMap tc_make_map(const void *base, int64_t rows, int64_t cols, int64_t ld, int box_rows, int box_bytes, int kind) {
  return make_map(base, rows, cols, ld, box_rows, box_bytes, kind);
}

void tc_set_autotune(bool on) { g_tune_on = on; }

int tc_tuning_table(int cap, double *rec, int *pair) {
  const int dev = current_device();
  std::lock_guard<std::mutex> lock(g_tune_mu);
  int n = 0;
  for (const auto &kv : g_tune) {
    if (kv.first.dev != dev) continue;
    if (n < cap && pair) pair[n] = kv.second.cfg.pair ? 1 : 0;
    if (n < cap && rec) {
      double *r = rec + 10 * n;
      const TuneKey &k = kv.first;
      const TuneRec &t = kv.second;
      r[0] = k.kind; r[1] = (double)k.M; r[2] = (double)k.N; r[3] = (double)k.K;
      r[4] = t.cfg.BN; r[5] = t.cfg.splits; r[6] = t.cfg.band;
      r[7] = t.ms_best; r[8] = t.ms_rule; r[9] = t.tried;
    }
    ++n;
  }
  return n;
}

int tc_error(cudaStream_t st) {
  int *g_err = nullptr;
  {
    const int dev = current_device();
    std::lock_guard<std::mutex> lock(g_dev_mu);
    g_err = g_err_dev[dev];
  }
  if (!g_err) return 0;
  int h = 0;
  CCLR_CUDA(cudaMemcpyAsync(&h, g_err, sizeof(int), cudaMemcpyDeviceToHost, st));
  CCLR_CUDA(cudaStreamSynchronize(st));
  if (h) CCLR_CUDA(cudaMemsetAsync(g_err, 0, sizeof(int), st));
  return h;
}

}  // namespace cclr
