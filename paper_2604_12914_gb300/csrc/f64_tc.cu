// FP64-accurate complex GEMM on tcgen05 from exact 8-bit slices; see f64_tc.cuh.
//
// This GPU's FP64 pipe does two FMAs per clock and SM, so a complex GEMM on it stops near 1 TFLOP/s.  The
// 36 BF16 slice products (orders q <= 7) cost 36 times a BF16 GEMM and still leave some 25 times more.
// Measured (GEMM and output kernel, operands sliced): M = N = K = 1760 complex 1.24 ms (35 TFLOP/s, 1270 TFLOP/s of
// BF16 MMAs) against 42 ms on the FP64 pipe; 12100 x 1760 x 500 2.67 ms against 90; 400^3 49 us against 617 (44 without the
// comparison of the magnitudes, which runs beside the slice products).
// What bounds it: MMAs alone (never waiting for the epilogue) 0.89 ms at 1760^3; handing each sum to the epilogue and
// its accumulator back, 0.99 ms; with the epilogue's integer work, 1.24 ms.  With chunks of 32 real K (eight sums per
// chunk, each of its own order) and 128-row tiles by single CTAs it was 1.09, 1.5 and 1.81 ms: twice as many sums to
// hand over per MMA, and MMAs of 93 clocks instead of 64.
#include <atomic>
#include <cmath>
#include <type_traits>

#include "engine.cuh"
#include "f64_tc.cuh"
#include "tc_ptx.cuh"

namespace cclr {
namespace {

constexpr int S = F64_SLICES;
constexpr int BM = 128;
constexpr int KC = 64;                  // real K per chunk: 128-byte slice rows, and |S_q| <= 6 2^14 64 < 2^24 exact (q <= 5)
constexpr int A_SLOT = BM * KC * 2;     // bytes of one slice block of A
constexpr int NSLOT = S + 1;            // slots of (A_s, B_s): one chunk, and slice 0 of the next
__host__ __device__ constexpr int b_slot(int BN, bool pair) { return (pair ? BN / 2 : BN) * KC * 2; }
// slot of slice s in a chunk of parity par
__host__ __device__ constexpr int slot_of(int s, int par) { return s == 0 && par ? S : s; }
constexpr int NBUF = 4;                 // accumulators in TMEM, taken in turn
constexpr int MAX_CHUNKS = 1024;        // per launch, 65536 real K: |S_0| 2^32 stays below 2^62
constexpr int SPLIT_TILES = 76;         // K is split when at most this many tiles (half the SMs) exist

struct F64Params {
  int sA, sB, rA, rB;   // slice rows per slice of A and B, first slice row
  int nMt, nNt, splits, chunks_per_split;
  int uMt, band;        // work units: rows of tiles (of two tiles for pairs of CTAs), and those per raster band
  const uint32_t *list; // the units to compute, (m << 16) | n, ntiles of them (nullptr: all, in raster order)
  int ntiles;
  int chunk0, chunk1;   // chunks of KC of this K segment
  int K;                // real K
  long long *hi;        // integer sums, [split][tile][column][row]: hi + lo 2^-8, in units of 2^(ea + eb - 46)
  float *lo;
  int *err;
};

// C += or = alpha times the sums, through C's views
struct F64Out {
  int m0, n0, M, N;     // first row and complex column of the tiles; C's extents
  int nMt, nNt, splits, cols_fast, accumulate;
  const uint32_t *list; // as the GEMM's (K is not split then)
  int ntiles;
  const long long *hi;
  const float *lo;
  const uint32_t *ea, *eb;  // rows' and columns' maxima (scale_of gives the exponents)
  double *C;
  View2 rv, cv;
  double ar, ai;        // alpha (used unless pow2)
  int pow2, neg, sh;    // alpha = (-1)^neg 2^sh
  // entries that are summed directly: the words of tc_magnitude_sums, or its sums (then words is nullptr), for the rows from
  // m0 on and the ldw columns from n0 on; the operands, and the complex k of this launch
  const uint4 *words;
  const float2 *sums;
  int64_t ldw;
  float tau;
  const double2 *A, *B;
  int64_t ra, rb;  // their first row and column
  View2 arv, akv, brv, bkv;
  int64_t k0, k1;
};

__device__ __forceinline__ void unit_coords(const F64Params &p, int u, int &mt, int &nt, int &sp) {
  sp = u / p.ntiles;
  const int id = u - sp * p.ntiles;
  if (p.list) {
    const uint32_t mn = __ldg(p.list + id);
    mt = (int)(mn >> 16);
    nt = (int)(mn & 0xffff);
    return;
  }
  const int per_band = p.band * p.nNt, b = id / per_band, local = id - b * per_band;
  const int mb = min(p.band, p.uMt - b * p.band);
  mt = b * p.band + local % mb;
  nt = local / mb;
}

// W accumulator columns of the warp's 32 rows into registers (no wait), W = 8, 16 or 32
template <int W> __device__ __forceinline__ void tmem_ld(uint32_t a, uint32_t (&r)[W]);
template <> __device__ __forceinline__ void tmem_ld<8>(uint32_t a, uint32_t (&r)[8]) {
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
               : "r"(a));
}
template <> __device__ __forceinline__ void tmem_ld<16>(uint32_t a, uint32_t (&r)[16]) {
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
               : "r"(a));
}
template <> __device__ __forceinline__ void tmem_ld<32>(uint32_t a, uint32_t (&r)[32]) {
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, %16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]), "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]), "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
               : "r"(a));
}
// completes every load issued before it; hold() passes registers through so that no use of them moves above
__device__ __forceinline__ void tmem_wait() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }
template <int W> __device__ __forceinline__ void hold(uint32_t (&r)[W]) {
#pragma unroll
  for (int k = 0; k < W; ++k) asm volatile("" : "+r"(r[k])::"memory");
}

// scale e of a row from the largest high word of its entries' magnitudes: every |x| < 2^e
__device__ __forceinline__ int scale_of(uint32_t m) {
  const int ex = (int)(m >> 20);
  return ex == 0x7ff ? F64_NONFINITE : max(ex, 1) - 1022;
}

// H 2^8 + L for integers H = h wh and L = l wl (floats; |H| <= 3 2^20, |L| <= 2^22), from the bits of 2^23 + 0x34C000 + H
// and -(2^23 + 2^22 + L): H and L are their low bits, and the constants cancel modulo 2^32.
__device__ __forceinline__ int two_orders(uint32_t h, uint32_t l, float wh, float wl) {
  const uint32_t x = __float_as_uint(fmaf(__uint_as_float(h), wh, 11845632.f));
  const uint32_t y = __float_as_uint(fmaf(__uint_as_float(l), -wl, -12582912.f));
  return (int)((x << 8) + y);
}
constexpr uint32_t MAGIC = 0x4B400000u;  // 2^23 + 2^22: an integer of up to 22 bits is its low bits when added to it

// lo 2^s rounded to an integer (|result| < 2^62), from the bits of lo
__device__ __forceinline__ long long scaled_int(float lo, int s) {
  const uint32_t b = __float_as_uint(lo), ex = (b >> 23) & 0xff;
  const unsigned long long m = ex ? (b & 0x7fffffu) | 0x800000u : 0u;
  const int sh = (int)ex - 150 + s;
  const unsigned long long r = sh >= 0 ? m << sh : sh < -25 ? 0ull : ((m >> (-sh - 1)) + 1) >> 1;
  return (int)b < 0 ? -(long long)r : (long long)r;
}

// 2^e (hi 2^-46 + lo 2^-54), negated if neg: hi is shifted up as far as it goes (24 bits at most), lo rounded into
// the bits below it, and the sum rounded once to FP64 (ties to even), in integer arithmetic: the FP64 pipe would
// take longer for its conversions and scalings than the MMAs of a short K.
__device__ __forceinline__ double combine(long long hi, float lo, int e, int neg) {
  const int s = max(0, min(24, __clzll(hi < 0 ? -hi : hi) - 2));
  const long long tot = (hi << s) + scaled_int(lo, s - 8);
  if (tot == 0) return 0.0;
  unsigned long long m = (unsigned long long)(tot < 0 ? -tot : tot);
  const unsigned long long sign = ((tot < 0) != (neg != 0)) ? 1ull << 63 : 0ull;
  const int lz = __clzll(m), ex = 1023 + 63 - lz + e - 46 - s;  // biased exponent of the leading bit
  m <<= lz;
  m = (m + 0x3ffull + ((m >> 11) & 1)) < m ? 1ull << 53 : (m + 0x3ffull + ((m >> 11) & 1)) >> 11;
  if (ex > 0 && ex < 0x7fe) return __longlong_as_double((long long)(sign | (((unsigned long long)(ex - 1) << 52) + m)));
  // towards the ends of the range: [1, 2] scaled in steps that stay representable
  const double r = __longlong_as_double((long long)(sign | ((1022ull << 52) + m)));
  const int d = max(-2200, min(2200, ex - 1023)), d1 = d / 3, d2 = (d - d1) / 2;
  auto two = [](int k) { return __hiloint2double((1023 + k) << 20, 0); };
  return r * two(d1) * two(d2) * two(d - d1 - d2);
}

// product of slices i of A and j of B of a chunk of parity par, MMAs of 16 real K each (two if half, else four), into
// the accumulator at d (added to it if acc)
template <int BN, bool PAIR>
__device__ __forceinline__ void issue_product(uint32_t base, int par, bool half, int i, int j, uint32_t d, uint32_t idesc,
                                              bool acc) {
  constexpr uint32_t SLOT = (A_SLOT + b_slot(BN, PAIR)) >> 4;
  const uint32_t da = base + slot_of(i, par) * SLOT, db = base + slot_of(j, par) * SLOT + (A_SLOT >> 4);
  mma_sw128<PAIR>(d, da, db, idesc, acc);
  mma_sw128<PAIR>(d, da + 2, db + 2, idesc, true);
  if (half) return;
  mma_sw128<PAIR>(d, da + 4, db + 4, idesc, true);
  mma_sw128<PAIR>(d, da + 6, db + 6, idesc, true);
}
// `count` products of order q, slices of A from the digits of `list`, lowest first (a loop: unrolled, its addresses
// spill from the forty registers)
template <int BN, bool PAIR>
__device__ __forceinline__ void issue_list(uint32_t base, int par, bool half, int q, uint32_t list, int count, uint32_t d,
                                           uint32_t idesc, bool acc) {
#pragma unroll 1
  for (int k = 0; k < count; ++k, list >>= 4)
    issue_product<BN, PAIR>(base, par, half, (int)(list & 7), q - (int)(list & 7), d, idesc, acc || k > 0);
}
template <bool PAIR> __device__ __forceinline__ void commit(uint32_t bar) {
  if constexpr (PAIR) mma_commit_pair(bar);
  else mma_commit(bar);
}

// The accumulators are taken in turn: the next one and the parity of its use.
struct Turn {
  int buf = 0;
  uint32_t parity = 0;
  __device__ __forceinline__ Turn next() const {
    Turn t;
    t.buf = (buf + 1) % NBUF;
    t.parity = t.buf == 0 ? parity ^ 1u : parity;
    return t;
  }
};

struct Bars {
  uint32_t base;  // of the barriers: full, empty, tfull, tempty
  int *err;
  volatile int *abort_flag;
  __device__ __forceinline__ uint32_t at(int i) const {
    uint32_t a = base;
    asm volatile("" : "+r"(a));  // formed here, not kept in a register of its own
    return a + 8 * (uint32_t)i;
  }
};

// full barriers: slice 0 of even and odd chunks, slice 1, slices 6 and 7, 2 and 5, 3 and 4; empty barriers: slices 7,
// 6, 1, (3 and 5), 2, 4 (and 0, which is free when the next chunk's 4 is)
enum { F_0 = 0, F_1 = 2, F_67, F_25, F_34, NFULL };
enum { E_7 = 0, E_6, E_1, E_35, E_2, E_4, NEMPTY };
enum { B_EMPTY = NFULL, B_TFULL = B_EMPTY + NEMPTY, B_TEMPTY = B_TFULL + NBUF };
constexpr int GROUPS = 5;  // full barriers per chunk, in the order they are expected: 0, 67, 1, 25, 34

// All MMAs of the n-th chunk: order 0, order 1, orders 7 and 6 (one sum), then 2, 3, 5 and 4.  The sum of an order is
// handed over, and its accumulator handed back, about a microsecond after its MMAs have run; in this sequence each finds
// its accumulator, that of the fourth sum before it, free.  A slice block arrives as long after its slot was freed: the
// last orders read first what the next chunk begins with (slice 0 has two slots, slice 1 is read by their first four
// products, and order 7 begins with the slices that come first).
template <int BN, bool PAIR>
__device__ __forceinline__ bool issue_chunk(uint32_t base, uint32_t tmem, uint32_t idesc, const Bars &b, Turn &t, uint32_t n,
                                            bool half, int *consumed) {
  const int par = (int)(n & 1u);
  auto wait = [&](int bar, uint32_t parity) {
    const bool ok = mbar_wait_ab(b.at(bar), parity, b.err, b.abort_flag);
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    return ok;
  };
  auto list = [&](int q, uint32_t l, int count, int buf, bool acc) {
    issue_list<BN, PAIR>(base, par, half, q, l, count, tmem + (uint32_t)(buf * BN), idesc, acc);
  };
#pragma unroll 1
  for (int q = 0; q < 4; ++q) {
    if (q == 0 && !wait(F_0 + par, (n >> 1) & 1u)) return false;
    if (q == 1 && !wait(F_1, n & 1u)) return false;
    if (!wait(B_TEMPTY + t.buf, t.parity ^ 1u)) return false;
    list(q, 0x3210u, q + 1, t.buf, false);
    commit<PAIR>(b.at(B_TFULL + t.buf));
    t = t.next();
    if (q == 1) {
      if (!wait(F_67, n & 1u)) return false;
      consumed[0] = GROUPS * (int)n + 3;
      if (!wait(B_TEMPTY + t.buf, t.parity ^ 1u)) return false;
      list(7, 0x6170u, 4, t.buf, false);
      if (!wait(F_25, n & 1u)) return false;
      list(7, 0x52u, 2, t.buf, true);
      if (!wait(F_34, n & 1u)) return false;
      consumed[0] = GROUPS * (int)n + GROUPS;
      list(7, 0x43u, 2, t.buf, true);
      commit<PAIR>(b.at(B_EMPTY + E_7));
      list(6, 0x6543210u, 7, t.buf, true);
      commit<PAIR>(b.at(B_EMPTY + E_6));
      commit<PAIR>(b.at(B_TFULL + t.buf));
      t = t.next();
    }
  }
  const Turn t4 = t.next();
  if (!wait(B_TEMPTY + t.buf, t.parity ^ 1u)) return false;
  list(5, 0x41u, 2, t.buf, false);
  if (!wait(B_TEMPTY + t4.buf, t4.parity ^ 1u)) return false;
  list(4, 0x31u, 2, t4.buf, false);
  commit<PAIR>(b.at(B_EMPTY + E_1));
  list(5, 0x3250u, 4, t.buf, true);
  commit<PAIR>(b.at(B_TFULL + t.buf));
  commit<PAIR>(b.at(B_EMPTY + E_35));
  list(4, 0x2u, 1, t4.buf, true);
  commit<PAIR>(b.at(B_EMPTY + E_2));
  list(4, 0x40u, 2, t4.buf, true);
  commit<PAIR>(b.at(B_TFULL + t4.buf));
  commit<PAIR>(b.at(B_EMPTY + E_4));
  t = t4.next();
  return true;
}

// Warp 0 streams slice blocks with TMA, each as its slot is freed.  Warp 1 issues the MMAs.  Warps 4-11 add the sums of
// the orders 0 .. 4 to a 64-bit integer (two orders at a time as one 32-bit integer) and those of 5 and of 6 and 7 to a
// float per output, and store both once per unit.  The orders 6 and 7 share an accumulator: slice s is stored times
// 2^(-8 s), so they add up with their weights, and below 2^-48 of the total its 24 bits are plenty.  192 accumulator
// registers per thread: setmaxnreg gives the two epilogue warpgroups 232 and the first one 40 (of 168 at launch).
// PAIR: two CTAs share a unit of 256 rows; each loads its rows of A and half the rows of B, the first one issues the
// MMAs of both.  An MMA of 128 x 128 reads 8 KB of shared memory and takes 93 clocks instead of 64 for that; as half
// of a pair's it reads 6.
template <int BN, bool PAIR>
__global__ void __launch_bounds__(384, 1)
    f64_gemm_kernel(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmB, F64Params p) {
  constexpr int SLOT = A_SLOT + b_slot(BN, PAIR), NC = BN / 2;
  constexpr uint32_t TCOLS = NBUF * BN;
  extern __shared__ uint8_t smem_raw[];
  uint8_t *smem = (uint8_t *)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
  // (pairs: full and tempty are waited for in CTA 0 only; empty and tfull arrive in both)
  uint64_t *bars = (uint64_t *)(smem + NSLOT * SLOT);
  uint64_t *full = bars, *empty = full + NFULL, *tfull = empty + NEMPTY, *tempty = tfull + NBUF, *drain = tempty + NBUF;
  uint32_t *tslot = (uint32_t *)(drain + 1);
  int *issued = (int *)(tslot + 1), *consumed = issued + 1;
  volatile int *abort_flag = issued + 2;
  const int warp = __shfl_sync(0xffffffffu, threadIdx.x >> 5, 0), lane = threadIdx.x & 31;
  const int units = p.ntiles * p.splits;
  const int rank = PAIR ? (int)cta_rank() : 0, first = PAIR ? blockIdx.x >> 1 : blockIdx.x,
            step = PAIR ? gridDim.x >> 1 : gridDim.x;

  if (threadIdx.x == 0) {
    for (int s = 0; s < NFULL; ++s) asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(su32(full + s)) : "memory");
    for (int s = 0; s < NEMPTY; ++s) asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(su32(empty + s)) : "memory");
    for (int b = 0; b < NBUF; ++b) {
      asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(su32(tfull + b)) : "memory");
      asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(su32(tempty + b)), "r"(PAIR ? 16 : 8) : "memory");
    }
    asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(su32(drain)) : "memory");
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    issued[0] = 0;
    consumed[0] = 0;
    *abort_flag = 0;
  }
  __syncthreads();
  if (warp == 1) {
    if constexpr (PAIR) {
      asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(su32(tslot)), "r"(TCOLS)
                   : "memory");
      asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
    } else {
      asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(su32(tslot)), "r"(TCOLS)
                   : "memory");
      asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  if constexpr (PAIR) pair_sync();  // both CTAs' barriers are initialised
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tmem = __shfl_sync(0xffffffffu, *tslot, 0);

  if (warp < 4) {
    asm volatile("setmaxnreg.dec.sync.aligned.u32 40;");
    if (warp == 0 && lane == 0) {
      uint32_t n = 0;  // chunks so far
      bool ok = true;
      for (int u = first; u < units && ok; u += step) {
        int mt, nt, sp;
        unit_coords(p, u, mt, nt, sp);
        if (PAIR) mt = 2 * mt + rank;
        const int c0 = p.chunk0 + sp * p.chunks_per_split, c1 = min(p.chunk1, c0 + p.chunks_per_split);
        const int yA = p.rA + mt * BM, yB = p.rB + nt * BN + (PAIR ? rank * (BN / 2) : 0);
        for (int c = c0; c < c1 && ok; ++c, ++n) {
          const int par = (int)(n & 1u);
          // slices 0, 7, 6, 1, 5, 3, 2, 4, as they are freed (slice 0's slot was last read two chunks ago, before
          // slice 4 of the last one could be loaded); a loop, as forty registers do not hold eight slices' addresses
#pragma unroll 1
          for (int j = 0; j < S; ++j) {
            const int s = (0x42351670u >> (4 * j)) & 7, f = s == 0 ? F_0 + par : (0x33455420u >> (4 * s)) & 7;
            if (j > 0 && !(ok = mbar_wait_ab(su32(empty + (j <= 4 ? j - 1 : j - 2)), (n & 1u) ^ 1u, p.err, abort_flag))) break;
            if (j < 6 && j != 2) {  // the first slice of its group: one slice (0 and 1) or two
              if (!PAIR || rank == 0)
                asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(su32(full + f)),
                             "r"((uint32_t)(SLOT * (PAIR ? 2 : 1) * (s < 2 ? 1 : 2)))
                             : "memory");
              issued[0] = issued[0] + 1;
            }
            uint8_t *dst = smem + slot_of(s, par) * SLOT;
            if constexpr (PAIR) {
              const uint32_t fb = pair_addr(su32(full + f), 0);
              tma_load_2d_pair(dst, &tmA, c * KC, s * p.sA + yA, fb);
              tma_load_2d_pair(dst + A_SLOT, &tmB, c * KC, s * p.sB + yB, fb);
            } else {
              tma_load_2d(dst, &tmA, c * KC, s * p.sA + yA, su32(full + f));
              tma_load_2d(dst + A_SLOT, &tmB, c * KC, s * p.sB + yB, su32(full + f));
            }
          }
        }
      }
    } else if (warp == 1 && rank == 0 && elect_one()) {
      const uint32_t idesc = idesc_mma(TC_BF16, PAIR ? 2 * BM : BM, BN), base = sw64_lo(su32(smem));
      const Bars b{su32(bars), p.err, abort_flag};
      Turn t;
      uint32_t n = 0;  // chunks so far
      bool ok = true;
      for (int u = first; u < units && ok; u += step) {
        int mt, nt, sp;
        unit_coords(p, u, mt, nt, sp);
        const int c0 = p.chunk0 + sp * p.chunks_per_split, c1 = min(p.chunk1, c0 + p.chunks_per_split);
        for (int c = c0; c < c1 && ok; ++c, ++n) {
          // half: the rest of the chunk is zeros
          ok = issue_chunk<BN, PAIR>(base, tmem, idesc, b, t, n, p.K - c * KC <= KC / 2, consumed);
        }
      }
      commit<PAIR>(su32(drain));
      mbar_wait(su32(drain), 0, p.err);
    }
    __syncwarp();
  } else {
    asm volatile("setmaxnreg.inc.sync.aligned.u32 232;");
    const int quarter = warp & 3, h = (warp - 4) >> 2;
    const uint32_t tb = tmem + ((uint32_t)(quarter * 32) << 16) + (uint32_t)(h * NC);
    bool ok = true;
    uint32_t n = 0;  // chunks so far
    Turn t;
    for (int u = first; u < units && ok; u += step) {
      int mt, nt, sp;
      unit_coords(p, u, mt, nt, sp);
      if (PAIR) mt = 2 * mt + rank;
      const int c0 = p.chunk0 + sp * p.chunks_per_split, c1 = min(p.chunk1, c0 + p.chunks_per_split);
      long long hi[NC];
      float lo[NC];
#pragma unroll
      for (int c = 0; c < NC; ++c) { hi[c] = 0; lo[c] = 0.f; }
      auto wait = [&](int buf, uint32_t parity) {
        const bool w = mbar_wait_ab(su32(tfull + buf), parity, p.err, abort_flag);
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        return __all_sync(0xffffffffu, w) != 0;
      };
      auto release = [&](int buf) {
        asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
        __syncwarp();
        if (lane == 0) {
          if constexpr (PAIR) mbar_arrive_cluster(pair_addr(su32(tempty + buf), 0));
          else mbar_arrive(su32(tempty + buf));
        }
      };
      for (int ch = c0; ch < c1; ++ch, ++n) {
        constexpr int W1 = NC < 32 ? NC : 32, W2 = 8;  // columns per TMEM load (16 in pairs of accumulators spill)
        // two orders as one 32-bit integer, S_q 2^8 + S_(q+1), from the next two accumulators
        auto pair = [&](float wh, float wl, int shift) {
          const Turn x = t, y = t.next();
          t = y.next();
          if (!wait(x.buf, x.parity) || !wait(y.buf, y.parity)) return false;
#pragma unroll
          for (int c = 0; c < NC; c += W2) {
            uint32_t a[W2], b[W2];
            tmem_ld<W2>(tb + x.buf * BN + c, a);
            tmem_ld<W2>(tb + y.buf * BN + c, b);
            tmem_wait();
            hold(a);
            hold(b);
#pragma unroll
            for (int k = 0; k < W2; ++k) hi[c + k] += (long long)two_orders(a[k], b[k], wh, wl) * (1ll << shift);
          }
          release(x.buf);
          release(y.buf);
          return true;
        };
        auto low = [&]() {
          const Turn z = t;
          t = t.next();
          if (!wait(z.buf, z.parity)) return false;
#pragma unroll
          for (int c = 0; c < NC; c += W1) {
            uint32_t x[W1];
            tmem_ld<W1>(tb + z.buf * BN + c, x);
            tmem_wait();
            hold(x);
#pragma unroll
            for (int k = 0; k < W1; ++k) lo[c + k] = fmaf(__uint_as_float(x[k]), 0x1p40f, lo[c + k]);
          }
          release(z.buf);
          return true;
        };
        if (!(ok = pair(1.f, 0x1p8f, 24))) break;      // q = 0, 1
        if (!(ok = low())) break;                      // q = 7, 6
        if (!(ok = pair(0x1p16f, 0x1p24f, 8))) break;  // q = 2, 3
        if (!(ok = low())) break;                      // q = 5
        const Turn z = t;  // q = 4 (too large for the bits of a float near 2^23)
        t = t.next();
        if (!(ok = wait(z.buf, z.parity))) break;
#pragma unroll
        for (int c = 0; c < NC; c += W2) {
          uint32_t x[W2];
          tmem_ld<W2>(tb + z.buf * BN + c, x);
          tmem_wait();
          hold(x);
#pragma unroll
          for (int k = 0; k < W2; ++k) hi[c + k] += (long long)__float2int_rn(__uint_as_float(x[k]) * 0x1p32f);
        }
        release(z.buf);
      }
      if (!ok) break;
      if (PAIR && mt >= p.nMt) continue;
      const int64_t at = (((int64_t)sp * p.nMt * p.nNt + (int64_t)nt * p.nMt + mt) * BN + h * NC) * BM + quarter * 32 + lane;
#pragma unroll
      for (int c = 0; c < NC; ++c) {
        p.hi[at + c * BM] = hi[c];
        p.lo[at + c * BM] = lo[c];
      }
    }
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  // error path: drain copies issued but never consumed (bounded)
  if (threadIdx.x == 0 && (PAIR ? *abort_flag != 0 : consumed[0] < issued[0])) {
    if (rank == 0)
      for (int g = consumed[0]; g < issued[0]; ++g) {
        const int n = g / GROUPS, k = g % GROUPS, f = k == 0 ? F_0 + (n & 1) : k == 1 ? F_67 : k == 2 ? F_1 : k == 3 ? F_25 : F_34;
        mbar_wait(su32(full + f), (uint32_t)(k == 0 ? n >> 1 : n) & 1u, p.err);
      }
    if (PAIR) {  // copies of CTA 1 that CTA 0 never expected have no barrier to wait for: 10 ms, which no copy takes
      const unsigned long long t0 = gtime();
      while (gtime() - t0 < 10000000ull) {}
    }
  }
  __syncthreads();
  if constexpr (PAIR) pair_sync();  // neither CTA leaves while the other's MMAs, copies or arrivals may touch it
  if (warp == 1) {
    if constexpr (PAIR)
      asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(TCOLS) : "memory");
    else
      asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(TCOLS) : "memory");
  }
}

// Whether a part lies too far below the product of its row's and column's maxima for the slices: bit l of the word for row
// 32 g + l, or the sums of one entry.
__device__ __forceinline__ uint32_t small_bits(uint4 w) { return (w.z & ~w.x) | (w.w & ~w.y); }
__device__ __forceinline__ bool small_sum(float2 s, float tau) { return (s.x < tau && s.x != 0.f) || (s.y < tau && s.y != 0.f); }
// The FP64 sums alpha sum_k A(row, k) B(k, n) of the entries in 32 rows from r0 on and the columns c0 + lane whose words
// (lane by lane, the same in every warp) are not zero, which nobody else has written, by the block's 256 threads.  Many
// entries (64 of short sums, 256 of any): a thread per entry, in the order of k.  Else up to K = 1024 a warp per entry, and
// beyond it the block for up to four rows of a column, each thread every 32nd or 256th k and the threads' sums added up
// pairwise: few entries are bound by latency, many by the FP64 pipe, which the pairwise sums take too (all entries,
// 1760^3: 57 ms by four rows, 37 by threads; 12100 x 1760 x 500: 96 by warps, 72; the CUDA-core kernel 42 and 90).  In the long sums
// 32 terms that are all zero are passed over: the usual ones are those of a row or column that the difference of two equal
// products has left, a few roundings among zeros, and the FP64 pipe bounds the loop.  (256 x 256 entries of K = 12100 with
// 14 such rows: 0.73 ms without, 0.19 with.)  A call: inlined, it costs the conversion its registers.
__device__ __noinline__ void write_small(const F64Out &p, uint32_t word, int r0, int c0) {
  __shared__ double part[8][8];
  const int lane = threadIdx.x, y = threadIdx.y, thread = 32 * y + lane;
  auto write = [&](int row, int n, double re, double im) {
    double2 *dst = (double2 *)p.C + v2off(p.rv, row) + v2off(p.cv, n);
    double2 v = make_double2(p.ar * re - p.ai * im, p.ar * im + p.ai * re);
    if (p.accumulate) { const double2 o = *dst; v.x += o.x; v.y += o.y; }
    *dst = v;
  };
  auto nonzero = [](double2 z) {  // (in integers: comparisons are the FP64 pipe's too)
    return ((__double_as_longlong(z.x) | __double_as_longlong(z.y)) << 1) != 0;
  };
  const int total = __reduce_add_sync(0xffffffffu, __popc(word));
  if (total >= (p.k1 - p.k0 <= 256 ? 64 : 256)) {
    for (int t0 = 0; t0 < total; t0 += 256) {
      int left = t0 + thread, l = -1, n = 0;
#pragma unroll 1
      for (int j = 0; j < 16; ++j) {
        const uint32_t w = __shfl_sync(0xffffffffu, word, j);
        const int c = __popc(w);
        if (left >= 0 && left < c) {
          l = (int)__fns(w, 0, left + 1);
          n = c0 + j;
        }
        left -= c;
      }
      if (l < 0) continue;
      const double2 *a = p.A + v2off(p.arv, p.ra + r0 + l), *b = p.B + v2off(p.brv, p.rb + n);
      double re = 0.0, im = 0.0;
#pragma unroll 2
      for (int64_t k = p.k0; k < p.k1; ++k) {
        const double2 x = a[v2off(p.akv, k)], z = b[v2off(p.bkv, k)];
        re = fma(x.x, z.x, re);
        re = fma(-x.y, z.y, re);
        im = fma(x.x, z.y, im);
        im = fma(x.y, z.x, im);
      }
      write(r0 + l, n, re, im);
    }
    return;
  }
  auto add_lanes = [](double &x) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
  };
  if (p.k1 - p.k0 <= 1024) {
    int turn = 0;
    for (uint32_t c = __ballot_sync(0xffffffffu, word != 0); c; c &= c - 1) {
      const int j = __ffs(c) - 1, n = c0 + j;
      for (uint32_t w = __shfl_sync(0xffffffffu, word, j); w; w &= w - 1, ++turn) {
        if ((turn & 7) != y) continue;
        const int row = r0 + __ffs(w) - 1;
        const double2 *a = p.A + v2off(p.arv, p.ra + row), *b = p.B + v2off(p.brv, p.rb + n);
        double re = 0.0, im = 0.0;
        for (int64_t k = p.k0 + lane; k < p.k1; k += 128) {
          double2 x[4], z[4];
#pragma unroll
          for (int q = 0; q < 4; ++q) {
            const bool in = k + 32 * q < p.k1;
            x[q] = in ? a[v2off(p.akv, k + 32 * q)] : make_double2(0.0, 0.0);
            z[q] = in ? b[v2off(p.bkv, k + 32 * q)] : make_double2(0.0, 0.0);
          }
#pragma unroll
          for (int q = 0; q < 4; ++q) {
            re = fma(x[q].x, z[q].x, re);
            re = fma(-x[q].y, z[q].y, re);
            im = fma(x[q].x, z[q].y, im);
            im = fma(x[q].y, z[q].x, im);
          }
        }
        add_lanes(re);
        add_lanes(im);
        if (lane == 0) write(row, n, re, im);
      }
    }
    return;
  }
  for (uint32_t c = __ballot_sync(0xffffffffu, word != 0); c; c &= c - 1) {
    const int j = __ffs(c) - 1, n = c0 + j;
    const double2 *b = p.B + v2off(p.brv, p.rb + n);
    uint32_t w = __shfl_sync(0xffffffffu, word, j);
    while (w) {
      const int rows = min(4, __popc(w));
      int row[4];
      const double2 *a[4];
      double re[4] = {0.0, 0.0, 0.0, 0.0}, im[4] = {0.0, 0.0, 0.0, 0.0};
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        row[q] = w ? r0 + __ffs(w) - 1 : r0;
        a[q] = p.A + v2off(p.arv, p.ra + row[q]);
        w &= w - 1;
      }
      // (a block of the column is loaded under the sums of the one before, and one of zeros needs none of the rows)
      double2 zn = p.k0 + thread < p.k1 ? b[v2off(p.bkv, p.k0 + thread)] : make_double2(0.0, 0.0);
#pragma unroll 1
      for (int64_t k0 = p.k0; k0 < p.k1; k0 += 256) {
        const int64_t k = k0 + thread;
        const double2 z = zn;
        zn = k + 256 < p.k1 ? b[v2off(p.bkv, k + 256)] : make_double2(0.0, 0.0);
        if (!__any_sync(0xffffffffu, nonzero(z))) continue;
        const bool in = k < p.k1;
        const int64_t ko = in ? v2off(p.akv, k) : 0;
        double2 x[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) x[q] = in && q < rows ? a[q][ko] : make_double2(0.0, 0.0);
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          int some = __any_sync(0xffffffffu, nonzero(x[q]) && nonzero(z));
          asm volatile("" : "+r"(some));
#pragma unroll 1
          for (; some > 0; --some) {  // (a loop of at most one pass: as a condition it predicates the FMAs, which take the pipe)
            re[q] = fma(x[q].x, z.x, re[q]);
            re[q] = fma(-x[q].y, z.y, re[q]);
            im[q] = fma(x[q].x, z.y, im[q]);
            im[q] = fma(x[q].y, z.x, im[q]);
          }
        }
      }
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        if (q >= rows) break;
        add_lanes(re[q]);
        add_lanes(im[q]);
        if (lane == 0) {
          part[y][2 * q] = re[q];
          part[y][2 * q + 1] = im[q];
        }
      }
      __syncthreads();
#pragma unroll
      for (int q = 0; q < 4; ++q)
        if (thread == q && q < rows) {
          auto sum = [&](int i) {
            return ((part[0][i] + part[1][i]) + (part[2][i] + part[3][i])) + ((part[4][i] + part[5][i]) + (part[6][i] + part[7][i]));
          };
          write(row[q], n, sum(2 * q), sum(2 * q + 1));
        }
      __syncthreads();
    }
  }
}

// The integer sums to FP64: a block takes 32 rows by 16 complex columns of a tile, reads the sums of every K
// split along the rows (as the GEMM wrote them), adds them exactly, and writes C along its contiguous direction
// (through shared memory when that is the columns).  This is a kernel of its own because the conversion is some
// hundred dependent integer instructions per value: at the GEMM's eight warps per SM, with the accumulators
// holding all registers, it took 50 us per tile, as long as the MMAs of K = 250.
template <int BN>
__global__ void __launch_bounds__(256, 4) f64_out_kernel(const __grid_constant__ F64Out p) {
  __shared__ double2 T[32][17];
  const int lane = threadIdx.x, y = threadIdx.y;
  int b = blockIdx.x;
  const int cg = b % (BN / 32);
  b /= BN / 32;
  const int rg = b % 4;
  int tile = b / 4, mt = tile % p.nMt, nt = tile / p.nMt;
  if (p.list) {
    const uint32_t mn = __ldg(p.list + tile);
    mt = (int)(mn >> 16);
    nt = (int)(mn & 0xffff);
    tile = nt * p.nMt + mt;
  }
  const int r0 = p.m0 + mt * BM + rg * 32, c0 = p.n0 + nt * (BN / 2) + cg * 16;
  if (r0 >= p.M || c0 >= p.N) return;
  const int row = r0 + lane;
  const int er = row < p.M ? scale_of(p.ea[row]) : 0;
  const uint32_t finite = __ballot_sync(0xffffffffu, er < F64_NONFINITE / 2);
  const int64_t plane = (int64_t)p.nMt * p.nNt * BN * BM;
  double2 v[2];
#pragma unroll
  for (int q = 0; q < 2; ++q) {
    const int j = y + 8 * q, n = c0 + j;
    if (n < p.N) {
      const int64_t at = ((int64_t)tile * BN + cg * 32 + 2 * j) * BM + rg * 32 + lane;
      long long hr = 0, hm = 0;
      if (p.splits == 1) {
        hr = p.hi[at];
        hm = p.hi[at + BM];
      }
      float lr = p.lo[at], lm = p.lo[at + BM];
      if (p.splits > 1) {  // the low parts as integers of 2^-16
        long long ir = 0, im = 0;
#pragma unroll 4
        for (int s = 0; s < p.splits; ++s) {
          hr += p.hi[at + s * plane];
          hm += p.hi[at + s * plane + BM];
          ir += scaled_int(p.lo[at + s * plane], 16);
          im += scaled_int(p.lo[at + s * plane + BM], 16);
        }
        lr = (float)ir * 0x1p-16f;
        lm = (float)im * 0x1p-16f;
      }
      const int e = er + scale_of(p.eb[n]);
      v[q].x = combine(hr, lr, e + p.sh, p.neg);
      v[q].y = combine(hm, lm, e + p.sh, p.neg);
      if (!p.pow2) v[q] = make_double2(p.ar * v[q].x - p.ai * v[q].y, p.ar * v[q].y + p.ai * v[q].x);
      if (e >= F64_NONFINITE / 2) v[q].x = v[q].y = __longlong_as_double(0x7ff8000000000000ll);
      if (p.cols_fast) T[lane][j] = v[q];
    }
  }
  // the entries to be summed directly, written at the end (the words, of column c0 + lane, are used no earlier: the sums'
  // loads should not wait for theirs)
  uint32_t word = 0;
  if (p.words) {
    if (lane < 16 && c0 + lane < p.N) word = small_bits(__ldg(p.words + (int64_t)(mt * 4 + rg) * p.ldw + c0 + lane - p.n0));
  } else {
    const float2 *mine = p.sums + (int64_t)(row - p.m0) * p.ldw + c0 - p.n0;
#pragma unroll 8
    for (int j = 0; j < 16; ++j) {
      const float2 s = c0 + j < p.N && row < p.M ? __ldg(mine + j) : make_float2(0.f, 0.f);
      const uint32_t w = __ballot_sync(0xffffffffu, small_sum(s, p.tau));
      if (lane == j) word = w;
    }
  }
  if (word) word = scale_of(p.eb[c0 + lane]) < F64_NONFINITE / 2 ? word & finite : 0u;
  if (!p.cols_fast) {
#pragma unroll
    for (int q = 0; q < 2; ++q) {
      const int n = c0 + y + 8 * q;
      const uint32_t small = __shfl_sync(0xffffffffu, word, y + 8 * q);
      if (n >= p.N || row >= p.M || (small >> lane & 1)) continue;
      double2 *dst = (double2 *)p.C + v2off(p.rv, row) + v2off(p.cv, n);
      if (p.accumulate) { const double2 o = *dst; v[q].x += o.x; v[q].y += o.y; }
      *dst = v[q];
    }
  } else {
    __syncthreads();
    const int t = y * 32 + lane, j = t & 15, n = c0 + j;
    const uint32_t small = __shfl_sync(0xffffffffu, word, j);
    const int64_t co = n < p.N ? v2off(p.cv, n) : 0;
#pragma unroll
    for (int q = 0; q < 2; ++q) {
      const int rl = (t >> 4) + 16 * q;
      if (n >= p.N || r0 + rl >= p.M || (small >> rl & 1)) continue;
      double2 *dst = (double2 *)p.C + v2off(p.rv, r0 + rl) + co, z = T[rl][j];
      if (p.accumulate) { const double2 o = *dst; z.x += o.x; z.y += o.y; }
      *dst = z;
    }
  }
  if (__any_sync(0xffffffffu, word != 0)) write_small(p, word, r0, c0);
}

// The same for many K splits of a small C: a block takes 32 rows of one complex column, its eight warps share the
// splits.
template <int BN>
__global__ void __launch_bounds__(256, 4) f64_out_split_kernel(const __grid_constant__ F64Out p) {
  __shared__ long long T[4][8][33];
  const int lane = threadIdx.x, y = threadIdx.y;
  int b = blockIdx.x;
  const int j = b % (BN / 2);
  b /= BN / 2;
  const int rg = b % 4, tile = b / 4, mt = tile % p.nMt, nt = tile / p.nMt;
  const int row = p.m0 + mt * BM + rg * 32 + lane, n = p.n0 + nt * (BN / 2) + j;
  if (n >= p.N || p.m0 + mt * BM + rg * 32 >= p.M) return;
  const int er = row < p.M ? scale_of(p.ea[row]) : 0;
  const int64_t plane = (int64_t)p.nMt * p.nNt * BN * BM, at = ((int64_t)tile * BN + 2 * j) * BM + rg * 32 + lane;
  long long t[4] = {0, 0, 0, 0};  // hi and lo 2^16, real and imaginary
#pragma unroll 4
  for (int s = y; s < p.splits; s += 8) {
    t[0] += p.hi[at + s * plane];
    t[1] += p.hi[at + s * plane + BM];
    t[2] += scaled_int(p.lo[at + s * plane], 16);
    t[3] += scaled_int(p.lo[at + s * plane + BM], 16);
  }
#pragma unroll
  for (int k = 0; k < 4; ++k) T[k][y][lane] = t[k];
  __syncthreads();
  uint32_t small;
  if (p.words) {
    small = small_bits(__ldg(p.words + (int64_t)(mt * 4 + rg) * p.ldw + n - p.n0));
  } else {
    const float2 s = row < p.M ? __ldg(p.sums + (int64_t)(row - p.m0) * p.ldw + n - p.n0) : make_float2(0.f, 0.f);
    small = __ballot_sync(0xffffffffu, small_sum(s, p.tau));
  }
  small &= __ballot_sync(0xffffffffu, er + scale_of(p.eb[n]) < F64_NONFINITE / 2);
  if (y == 0 && row < p.M && !(small >> lane & 1)) {
#pragma unroll
    for (int k = 0; k < 4; ++k)
      for (int q = 1; q < 8; ++q) t[k] += T[k][q][lane];
    const int e = er + scale_of(p.eb[n]);
    double2 v;
    v.x = combine(t[0], (float)t[2] * 0x1p-16f, e + p.sh, p.neg);
    v.y = combine(t[1], (float)t[3] * 0x1p-16f, e + p.sh, p.neg);
    if (!p.pow2) v = make_double2(p.ar * v.x - p.ai * v.y, p.ar * v.y + p.ai * v.x);
    if (e >= F64_NONFINITE / 2) v.x = v.y = __longlong_as_double(0x7ff8000000000000ll);
    double2 *dst = (double2 *)p.C + v2off(p.rv, row) + v2off(p.cv, n);
    if (p.accumulate) { const double2 o = *dst; v.x += o.x; v.y += o.y; }
    *dst = v;
  }
  __syncwarp();
  if (small) write_small(p, lane == 0 ? small : 0u, row - lane, n);
}

// ---------------- slices ----------------
__device__ __forceinline__ uint32_t mag(double x) { return (uint32_t)__double2hiint(x) & 0x7fffffffu; }
__device__ __forceinline__ uint32_t mag2(double2 z) { return max(mag(z.x), mag(z.y)); }

// x 2^(63 - e) rounded to an integer (63 bits and sign), from the bits of x: no FP64 arithmetic
__device__ __forceinline__ long long fixed63(double x, int e) {
  const uint32_t h = (uint32_t)__double2hiint(x);
  const int ex = (int)((h >> 20) & 0x7ff);
  unsigned long long f = ((unsigned long long)((h & 0xfffffu) | (ex ? 0x100000u : 0u)) << 32) | (uint32_t)__double2loint(x);
  const int sh = max(ex, 1) - 1012 - e;  // at most 10
  if (sh >= 0) f <<= sh;
  else f = sh < -54 ? 0ull : ((f >> (-sh - 1)) + 1) >> 1;
  return (int)h < 0 ? -(long long)f : (long long)f;
}

// digit d (-128 .. 128) times 2^(-8 s) as BF16 bits
__device__ __forceinline__ uint32_t digit_bits(int d, int s) {
  return __float_as_uint((__uint_as_float(MAGIC + (uint32_t)d) - 12582912.f) * __uint_as_float((uint32_t)(127 - 8 * s) << 23)) >> 16;
}
// slice s > 0 from below: the next balanced digit (-128 .. 127)
__device__ __forceinline__ uint32_t digit(long long &X, int s) {
  const int d = (int)(signed char)(X & 0xff);
  X = (X - d) >> 8;
  return digit_bits(d, s);
}

// |x| 2^-e cut off to BF16 (bits); what is not zero counts as 2^-60 at least, so that its products stay above zero
__device__ __forceinline__ uint32_t magnitude_bits(double x, int e) {
  const uint32_t h = mag(x);
  const int ex = (int)(h >> 20), b = ex - 1023 - e + 127;
  return ex > 0 && b > 67 ? (uint32_t)b << 7 | ((h >> 13) & 0x7fu) : (h | (uint32_t)__double2loint(x)) ? 67u << 7 : 0u;
}

// eight slices and the magnitudes of one complex entry at real columns 2k, 2k+1 of slice row r (R rows per slice)
template <bool EMBED>
__device__ __forceinline__ void put_slices(uint32_t *dst, int64_t R, int64_t ld2, int64_t r, int64_t k, double2 z, int e) {
  const uint32_t ax = magnitude_bits(z.x, e), ay = magnitude_bits(z.y, e);
  if (EMBED) {
    uint32_t *row = dst + ((int64_t)S * 2 * R + 2 * r) * ld2 + k;
    row[0] = ax | (ay << 16);
    row[ld2] = ay | (ax << 16);
  } else {
    dst[((int64_t)S * R + r) * ld2 + k] = ax | (ay << 16);
  }
  long long X = fixed63(z.x, e), Y = fixed63(z.y, e);
  if (e == F64_NONFINITE) X = Y = 0;
#pragma unroll
  for (int s = S - 1; s >= 0; --s) {
    uint32_t a, b;
    if (s > 0) {
      a = digit(X, s);
      b = digit(Y, s);
    } else {  // the top digit, up to +-128
      a = digit_bits((int)X, 0);
      b = digit_bits((int)Y, 0);
    }
    if (EMBED) {
      uint32_t *row = dst + ((int64_t)s * 2 * R + 2 * r) * ld2 + k;
      row[0] = a | ((b ^ 0x8000u) << 16);
      row[ld2] = b | (a << 16);
    } else {
      dst[((int64_t)s * R + r) * ld2 + k] = a | (b << 16);
    }
  }
}

// Rows contiguous along k: T threads per row find the row's largest magnitude, then read it again (from
// L1/L2) and write its slices, coalesced along k.
template <int T, bool EMBED>
__global__ void __launch_bounds__(256) f64_slice_rows(const double2 *__restrict__ src, View2 rv, View2 kv, int64_t R, int64_t K,
                                                      uint32_t *__restrict__ dst, int64_t ld2, uint32_t *__restrict__ tops) {
  __shared__ uint32_t red[8];
  const int t = threadIdx.x % T;
  const int64_t r = (int64_t)blockIdx.x * (256 / T) + threadIdx.x / T;
  const double2 *row = src + (r < R ? v2off(rv, r) : 0);
  uint32_t m = 0;
  if (r < R)
    for (int64_t k = t; k < K; k += T) m = max(m, mag2(row[v2off(kv, k)]));
  m = __reduce_max_sync(0xffffffffu, m);
  if (T > 32) {
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = m;
    __syncthreads();
    for (int w = 0; w < T / 32; ++w) m = max(m, red[w]);
  }
  if (r >= R) return;
  if (t == 0) tops[r] = m;
  const int e = scale_of(m);
  for (int64_t k = t; k < K; k += T) put_slices<EMBED>(dst, R, ld2, r, k, row[v2off(kv, k)], e);
}

// The same for a few long rows: blocks over ranges of k, maxima first.
__global__ void __launch_bounds__(256) f64_rowmax(const double2 *__restrict__ src, View2 rv, View2 kv, int64_t K, int64_t kstep,
                                                  uint32_t *__restrict__ tops) {
  const double2 *row = src + v2off(rv, blockIdx.x);
  const int64_t k1 = min(K, (int64_t)(blockIdx.y + 1) * kstep);
  uint32_t m = 0;
  for (int64_t k = (int64_t)blockIdx.y * kstep + threadIdx.x; k < k1; k += 256) m = max(m, mag2(row[v2off(kv, k)]));
  m = __reduce_max_sync(0xffffffffu, m);
  if ((threadIdx.x & 31) == 0) atomicMax(tops + blockIdx.x, m);
}
template <bool EMBED>
__global__ void __launch_bounds__(256) f64_slice_range(const double2 *__restrict__ src, View2 rv, View2 kv, int64_t R, int64_t K,
                                                       int64_t kstep, uint32_t *__restrict__ dst, int64_t ld2,
                                                       const uint32_t *__restrict__ tops) {
  const int64_t r = blockIdx.x, k1 = min(K, (int64_t)(blockIdx.y + 1) * kstep);
  const double2 *row = src + v2off(rv, r);
  const int e = scale_of(tops[r]);
  for (int64_t k = (int64_t)blockIdx.y * kstep + threadIdx.x; k < k1; k += 256)
    put_slices<EMBED>(dst, R, ld2, r, k, row[v2off(kv, k)], e);
}

// Rows contiguous along r (k strided): maxima by threads along r over a range of k, then 32 x 32 transposing
// tiles.
__global__ void __launch_bounds__(256) f64_colmax(const double2 *__restrict__ src, View2 rv, View2 kv, int64_t R, int64_t K,
                                                  int64_t kstep, uint32_t *__restrict__ tops) {
  const int64_t r = (int64_t)blockIdx.x * 256 + threadIdx.x;
  if (r >= R) return;
  const double2 *row = src + v2off(rv, r);
  const int64_t k1 = min(K, (int64_t)(blockIdx.y + 1) * kstep);
  uint32_t m = 0;
#pragma unroll 4
  for (int64_t k = (int64_t)blockIdx.y * kstep; k < k1; ++k) m = max(m, mag2(row[v2off(kv, k)]));
  atomicMax(tops + r, m);
}
template <bool EMBED>
__global__ void __launch_bounds__(256) f64_slice_tiled(const double2 *__restrict__ src, View2 rv, View2 kv, int64_t R, int64_t K,
                                                       uint32_t *__restrict__ dst, int64_t ld2,
                                                       const uint32_t *__restrict__ tops) {
  __shared__ double2 tile[32][33];
  const int64_t tr = (R + 31) / 32, tk = (K + 31) / 32;
  for (int64_t t = blockIdx.x; t < tr * tk; t += gridDim.x) {
    const int64_t r0 = (t % tr) * 32, k0 = (t / tr) * 32;
    for (int q = threadIdx.y; q < 32; q += 8) {
      const int64_t r = r0 + threadIdx.x, k = k0 + q;
      tile[q][threadIdx.x] = (r < R && k < K) ? src[v2off(rv, r) + v2off(kv, k)] : make_double2(0.0, 0.0);
    }
    __syncthreads();
    for (int q = threadIdx.y; q < 32; q += 8) {
      const int64_t r = r0 + q, k = k0 + threadIdx.x;
      if (r < R && k < K) put_slices<EMBED>(dst, R, ld2, r, k, tile[threadIdx.x][q], scale_of(tops[r]));
    }
    __syncthreads();
  }
}

template <bool EMBED>
void prep_launch(const double2 *src, View2 rv, View2 kv, int64_t R, int64_t K, uint32_t *dst, uint32_t *tops, cudaStream_t st) {
  const int64_t ld2 = f64tc_ld(K) / 2;
  const bool kfast = kv.sin == 1 || rv.sin != 1;
  if (kfast && !(R < 2 * 152 && K >= 2048)) {
    if (K >= 512) f64_slice_rows<256, EMBED><<<(unsigned)R, 256, 0, st>>>(src, rv, kv, R, K, dst, ld2, tops);
    else f64_slice_rows<32, EMBED><<<(unsigned)((R + 7) / 8), 256, 0, st>>>(src, rv, kv, R, K, dst, ld2, tops);
    count_launch();
    return;
  }
  CCLR_CUDA(cudaMemsetAsync(tops, 0, (size_t)R * sizeof(uint32_t), st));
  if (kfast) {  // about four blocks per SM over ranges of at least 1024
    const int64_t ky = std::max<int64_t>(1, std::min<int64_t>({(4 * 152 + R - 1) / R, K / 1024, (int64_t)65535}));
    const int64_t kstep = (K + ky - 1) / ky;
    const dim3 g((unsigned)R, (unsigned)((K + kstep - 1) / kstep));
    f64_rowmax<<<g, 256, 0, st>>>(src, rv, kv, K, kstep, tops);
    f64_slice_range<EMBED><<<g, 256, 0, st>>>(src, rv, kv, R, K, kstep, dst, ld2, tops);
  } else {
    const int64_t bx = (R + 255) / 256;
    const int64_t ky = std::max<int64_t>(1, std::min<int64_t>({(4 * 152 + bx - 1) / bx, (K + 15) / 16, (int64_t)65535}));
    const int64_t kstep = (K + ky - 1) / ky;
    f64_colmax<<<dim3((unsigned)bx, (unsigned)((K + kstep - 1) / kstep)), 256, 0, st>>>(src, rv, kv, R, K, kstep, tops);
    const int64_t nt = ((R + 31) / 32) * ((K + 31) / 32);
    f64_slice_tiled<EMBED><<<(unsigned)std::min<int64_t>(nt, 152 * 64), dim3(32, 8), 0, st>>>(src, rv, kv, R, K, dst, ld2, tops);
  }
  count_launch(2);
}

template <int BN, bool PAIR> constexpr size_t smem_bytes() {
  return 1024 + (size_t)NSLOT * (A_SLOT + b_slot(BN, PAIR)) + (NFULL + NEMPTY + 2 * NBUF + 1) * 8 + 16;
}

// one launch of the GEMM over the units of p (rows of A from p.rA, columns of B from p.rB), and its output
template <int BN, bool PAIR>
void launch(const F64Op &A, const F64Op &B, const F64Params &p, F64Out &o, int64_t K, F64Side &side, cudaStream_t st) {
  static std::atomic<unsigned long long> attr_set{0};  // one bit per device
  constexpr int smem = (int)smem_bytes<BN, PAIR>();
  int dev = 0;
  CCLR_CUDA(cudaGetDevice(&dev));
  if (dev >= 64 || !(attr_set.load() & (1ull << dev))) {
    CCLR_CUDA(cudaFuncSetAttribute(f64_gemm_kernel<BN, PAIR>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem));
    if (dev < 64) attr_set |= 1ull << dev;
  }
  const int64_t ld = f64tc_ld(K);
  const CUtensorMap ma = tc_make_map(A.p, (int64_t)S * p.sA, 2 * K, ld, BM, 128, TC_BF16);
  const CUtensorMap mb = tc_make_map(B.p, (int64_t)S * p.sB, 2 * K, ld, PAIR ? BN / 2 : BN, 128, TC_BF16);
  const int64_t units = (int64_t)p.ntiles * p.splits;
  if constexpr (PAIR) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(2 * (unsigned)std::min<int64_t>(units, std::max(tc_num_sms() / 2, 1)));
    cfg.blockDim = dim3(384);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute at;
    at.id = cudaLaunchAttributeClusterDimension;
    at.val.clusterDim.x = 2;
    at.val.clusterDim.y = at.val.clusterDim.z = 1;
    cfg.attrs = &at;
    cfg.numAttrs = 1;
    CCLR_CUDA(cudaLaunchKernelEx(&cfg, f64_gemm_kernel<BN, PAIR>, ma, mb, p));
  } else {
    f64_gemm_kernel<BN, PAIR><<<(unsigned)std::min<int64_t>(units, tc_num_sms()), 384, smem, st>>>(ma, mb, p);
  }
  CCLR_CUDA(cudaGetLastError());
  o.hi = p.hi;
  o.lo = p.lo;
  o.nMt = p.nMt;
  o.nNt = p.nNt;
  o.splits = p.splits;
  side.join(st);
  if (p.splits > 8) f64_out_split_kernel<BN><<<(unsigned)(o.ntiles * 4 * (BN / 2)), dim3(32, 8), 0, st>>>(o);
  else f64_out_kernel<BN><<<(unsigned)(o.ntiles * 4 * (BN / 32)), dim3(32, 8), 0, st>>>(o);
  CCLR_CUDA(cudaGetLastError());
  count_launch(2);
}

// columns of tiles and rows of tiles of one launch, the K splits and the bytes of their sums
struct F64Plan {
  int BN, nMt, nNt, rows, cols;  // tiles in all; tile rows and tile columns per launch
  int64_t unit;                  // bytes of one tile's sums
};
// tiles whose sums take cap bytes: as many columns of accumulators at every width
int64_t tiles_that_fit(int BN, size_t cap) { return (int64_t)cap / (BM * 128 * 12) * (128 / BN); }
F64Plan plan_of(int64_t M, int64_t N, size_t cap) {
  F64Plan q;
  q.BN = 2 * N <= 32 ? 32 : 2 * N <= 64 ? 64 : 128;
  q.nMt = (int)((M + BM - 1) / BM);
  q.nNt = (int)((2 * N + q.BN - 1) / q.BN);
  q.unit = (int64_t)BM * q.BN * 12;
  const int64_t fit = tiles_that_fit(q.BN, cap);
  q.rows = (int)std::min<int64_t>(q.nMt, fit);
  q.cols = (int)std::max<int64_t>(1, std::min<int64_t>(q.nNt, fit / q.rows));
  return q;
}
// K splits of one launch: only when the tiles of the whole product leave half the SMs idle, two chunks at least each
int64_t splits_of(int64_t all_tiles, int64_t units, int slots, int n) {
  return all_tiles > SPLIT_TILES ? 1 : std::max<int64_t>(1, std::min<int64_t>(slots / units, n / 2));
}
constexpr size_t SUMS_CAP = 250u << 20;  // the most that the integer sums of one launch take

}  // namespace

F64Side::~F64Side() {
  if (s_) cudaStreamDestroy(s_);
  if (fork_) cudaEventDestroy(fork_);
  if (join_) cudaEventDestroy(join_);
}
cudaStream_t F64Side::fork(cudaStream_t st) {
  if (!s_) CCLR_CUDA(cudaStreamCreateWithFlags(&s_, cudaStreamNonBlocking));
  if (!fork_) CCLR_CUDA(cudaEventCreateWithFlags(&fork_, cudaEventDisableTiming));
  if (!join_) CCLR_CUDA(cudaEventCreateWithFlags(&join_, cudaEventDisableTiming));
  CCLR_CUDA(cudaEventRecord(fork_, st));
  CCLR_CUDA(cudaStreamWaitEvent(s_, fork_, 0));
  return s_;
}
void F64Side::join(cudaStream_t st) {
  CCLR_CUDA(cudaEventRecord(join_, s_));
  CCLR_CUDA(cudaStreamWaitEvent(st, join_, 0));
}

F64Op f64tc_prep(const void *src, View2 rv, View2 kv, int64_t R, int64_t K, bool embed, void *dst, uint32_t *tops,
                 cudaStream_t st) {
  CCLR_REQUIRE(R > 0 && K > 0 && (int64_t)F64_PLANES * 2 * R < (1ll << 31) && 2 * K < (1ll << 31), "f64tc_prep: bad dimensions");
  if (embed) prep_launch<true>((const double2 *)src, rv, kv, R, K, (uint32_t *)dst, tops, st);
  else prep_launch<false>((const double2 *)src, rv, kv, R, K, (uint32_t *)dst, tops, st);
  CCLR_CUDA(cudaGetLastError());
  F64Op op;
  op.p = dst;
  op.tops = tops;
  op.stride = R;
  op.src = src;
  op.rv = rv;
  op.kv = kv;
  return op;
}

// The largest need of any product of at most M rows and N columns, so that what a caller claims for its first (largest)
// block or chunk serves the others: a launch takes no more tiles than there are and than SUMS_CAP holds, K splits
// no more than one unit per SM, and the width of the tiles only grows with N.  (The need of the product itself
// is not monotone: fewer rows of tiles leave room for more columns of them.)
// Behind the integer sums lie the words of the launch's tiles, or the magnitudes' sums that they stand for: those are there
// only where the tiles leave half the SMs idle, and then the integer sums take one unit per SM at most.
size_t f64tc_scratch_bytes(int64_t M, int64_t N) {
  const F64Plan q = plan_of(M, N, SUMS_CAP);
  const int64_t tiles = std::min<int64_t>(tiles_that_fit(q.BN, SUMS_CAP), (int64_t)q.nMt * q.nNt);
  const int64_t small = std::min<int64_t>(std::max<int64_t>(M, 2) * 2 * N * 4, tc_magnitude_sums_cap());
  return (size_t)std::max<int64_t>(tiles * (q.unit + (BM / 32) * (q.BN / 2) * 16), tc_num_sms() * q.unit + small);
}

void f64tc_gemm(const F64Op &A, int64_t M, const F64Op &B, int64_t N, int64_t K, void *C, View2 rv, View2 cv, zc alpha,
                bool accumulate, void *scratch, F64Side &side, cudaStream_t st, UpperTiles *upper,
                int64_t upper_row, int64_t upper_col) {
  if (M <= 0 || N <= 0 || K <= 0) return;
  CCLR_REQUIRE(A.r0 + M <= A.stride && B.r0 + N <= B.stride, "f64tc_gemm: rows outside the prepared operand");
  CCLR_REQUIRE((uintptr_t)A.p % 16 == 0 && (uintptr_t)B.p % 16 == 0, "f64tc_gemm: operands must be 16-byte aligned");
  const F64Plan pl = plan_of(M, N, SUMS_CAP);
  F64Params p;
  p.sA = (int)A.stride;
  p.sB = (int)(2 * B.stride);
  p.err = tc_device_err();
  F64Out o;
  o.M = (int)M;
  o.N = (int)N;
  o.C = (double *)C;
  o.rv = rv;
  o.cv = cv;
  o.cols_fast = cv.sin == 1 && (cv.din == TC_ONE_LEVEL || cv.din >= 4) ? 1 : 0;
  o.ea = A.tops + A.r0;
  o.eb = B.tops + B.r0;
  o.ar = alpha.re;
  o.ai = alpha.im;
  int ex = 0;
  o.pow2 = alpha.im == 0.0 && std::abs(std::frexp(alpha.re, &ex)) == 0.5;
  o.sh = o.pow2 ? ex - 1 : 0;
  o.neg = o.pow2 && alpha.re < 0.0;
  o.A = (const double2 *)A.src;
  o.B = (const double2 *)B.src;
  o.ra = A.r0;
  o.rb = B.r0;
  o.arv = A.rv;
  o.akv = A.kv;
  o.brv = B.rv;
  o.bkv = B.kv;
  o.tau = (float)std::sqrt(2.0 * (double)K) * 0x1p-8f;
  const int64_t ld = f64tc_ld(K);
  const int nk = (int)((2 * K + KC - 1) / KC);
  p.K = (int)(2 * K);
  for (int t0 = 0; t0 < pl.nNt; t0 += pl.cols)
    for (int r0 = 0; r0 < pl.nMt; r0 += pl.rows) {
      p.nMt = std::min(pl.rows, pl.nMt - r0);
      p.nNt = std::min(pl.cols, pl.nNt - t0);
      o.m0 = r0 * BM;
      o.n0 = t0 * (pl.BN / 2);
      p.rA = (int)A.r0 + r0 * BM;
      p.rB = (int)(2 * B.r0) + t0 * pl.BN;
      const int64_t tiles = (int64_t)p.nMt * p.nNt, all = (int64_t)pl.nMt * pl.nNt;
      // tiles of 128 columns by pairs of CTAs, also where the second one has no rows (M <= 128): a single CTA's MMAs
      // take 93 clocks for 64 columns
      const bool pair = pl.BN == 128;
      const int slots = pair ? std::max(tc_num_sms() / 2, 1) : tc_num_sms();
      p.uMt = pair ? (p.nMt + 1) / 2 : p.nMt;
      p.band = std::min(p.uMt, pair ? 6 : 12);
      p.ntiles = p.uMt * p.nNt;
      o.ntiles = (int)tiles;
      p.list = o.list = nullptr;
      if (upper && all > SPLIT_TILES) {  // (a product with few tiles splits K instead)
        const int64_t um = upper_row + o.m0, un = upper_col + o.n0;
        o.list = upper->get(p.nMt, p.nNt, 12, BM, pl.BN / 2, um, un, upper_row + M, st, &o.ntiles);
        p.list = pair ? upper->get(p.uMt, p.nNt, p.band, 2 * BM, pl.BN / 2, um, un, upper_row + M, st, &p.ntiles) : o.list;
        if (!pair && o.list) p.ntiles = o.ntiles;
        if (!p.list || !o.list) {
          p.list = o.list = nullptr;
          p.ntiles = p.uMt * p.nNt;
          o.ntiles = (int)tiles;
        }
      }
      {
        // behind the integer sums of as many K splits as any segment of K below takes
        void *small = (char *)scratch + tiles * splits_of(all, (int64_t)p.uMt * p.nNt, slots, std::min(nk, MAX_CHUNKS)) * pl.unit;
        const int64_t mm = std::min<int64_t>(M - o.m0, (int64_t)p.nMt * BM);
        o.ldw = std::min<int64_t>(N - o.n0, (int64_t)p.nNt * (pl.BN / 2));
        const bool words = tc_magnitude_sums((const char *)A.p + ((int64_t)S * p.sA + p.rA) * ld * 2, ld,
                                             (const char *)B.p + ((int64_t)S * p.sB + p.rB) * ld * 2, ld, mm, 2 * o.ldw, 2 * K, o.tau,
                                             small, side.fork(st));
        o.words = words ? (const uint4 *)small : nullptr;
        o.sums = (const float2 *)small;
      }
      // segments of K that the integer sums can hold, one launch each
      for (p.chunk0 = 0; p.chunk0 < nk; p.chunk0 += MAX_CHUNKS) {
        p.chunk1 = std::min(nk, p.chunk0 + MAX_CHUNKS);
        const int n = p.chunk1 - p.chunk0;
        const int64_t splits = splits_of(all, (int64_t)p.uMt * p.nNt, slots, n);
        p.chunks_per_split = (int)((n + splits - 1) / splits);
        p.splits = (n + p.chunks_per_split - 1) / p.chunks_per_split;
        p.hi = (long long *)scratch;
        p.lo = (float *)(p.hi + tiles * p.splits * BM * pl.BN);
        o.accumulate = accumulate || p.chunk0 > 0;
        o.k0 = (int64_t)p.chunk0 * (KC / 2);
        o.k1 = std::min<int64_t>(K, (int64_t)p.chunk1 * (KC / 2));
        if (pl.BN == 32) launch<32, false>(A, B, p, o, K, side, st);
        else if (pl.BN == 64) launch<64, false>(A, B, p, o, K, side, st);
        else launch<128, true>(A, B, p, o, K, side, st);
      }
    }
}

}  // namespace cclr
