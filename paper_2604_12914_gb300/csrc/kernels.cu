// Generic device kernels of libcclr: strided complex GEMM on CUDA cores (FP64 DFMA and
// FP32 FFMA), arbitrary-stride permute/accumulate, and the HBM-bound vector kernels of the
// solver (axpy, bilinear and Hermitian dot products with FP64 accumulation, diagonal
// preconditioner, precision conversion).
#include "kernels.cuh"

#include <atomic>
#include <type_traits>

namespace cclr {

static std::atomic<unsigned long long> g_launches{0};
unsigned long long launch_count() { return g_launches.load(); }
void count_launch(unsigned long long n) { g_launches += n; }

// --------------------------------------------------------------------------------------
// Complex GEMM, C[b](m,n) (+)= alpha * sum_k A[b](m,k) B[b](k,n); arbitrary strides.
// Tile BM x BN x BK, each thread TM x TN outputs (interleaved rows/cols to spread banks).
// Bound by the loads from shared memory beside the FMAs (55 of 80 TFLOP/s).  4489 x 1139 x 270 in FP32: 236 us with
// loads and sums in turn in blocks of 16, 202 with each block's loads under the sums of the block before it in blocks
// of 8 (88 registers; blocks of 16 take 121).  8 x 4 outputs per thread: 245; packed FP32 pairs with the
// shared entries doubled to feed them: 272.
// --------------------------------------------------------------------------------------
template <typename T, int BM, int BN, int BK, int TM, int TN>
__global__ void __launch_bounds__((BM / TM) * (BN / TN))
    zgemm_simt(GemmArgs g, int64_t b0) {
  using C = typename cpx<T>::t;
  constexpr int NT = (BM / TM) * (BN / TN);
  constexpr int RX = BN / TN;  // threads along n
  constexpr int RY = BM / TM;  // threads along m
  __shared__ C As[BK][BM + 1];
  __shared__ C Bs[BK][BN + 1];

  const int64_t nMt = (g.M + BM - 1) / BM;
  const int64_t tile = blockIdx.x;
  const int64_t m0 = (tile % nMt) * BM;
  const int64_t n0 = (tile / nMt) * BN;
  const int64_t b = b0 + blockIdx.z;
  const C *A = (const C *)g.A + b * g.sAb;
  const C *B = (const C *)g.B + b * g.sBb;
  C *Cp = (C *)g.C + b * g.sCb;

  const int tid = threadIdx.x;
  const int tx = tid % RX, ty = tid / RX;
  C acc[TM][TN];
#pragma unroll
  for (int i = 0; i < TM; ++i)
#pragma unroll
    for (int j = 0; j < TN; ++j) acc[i][j] = C{T(0), T(0)};

  const bool a_kfast = (g.sAk == 1);
  const bool b_nfast = (g.sBn == 1);
  const int64_t kbeg = g.kchunk > 0 ? (int64_t)blockIdx.y * g.kchunk : 0;
  const int64_t kend = g.kchunk > 0 ? min(g.K, kbeg + g.kchunk) : g.K;
  // a block's loads are issued before the sums of the block before it, and each thread's entries of A and B are a
  // fixed step apart from block to block
  constexpr int NA = (BM * BK + NT - 1) / NT, NB = (BN * BK + NT - 1) / NT;
  C ra[NA], rb[NB];
  const C *pa[NA], *pb[NB];
  int ka[NA], kb[NB];
#pragma unroll
  for (int q = 0; q < NA; ++q) {
    const int e = tid + q * NT, mm = a_kfast ? e / BK : e % BM;
    ka[q] = e < BM * BK && m0 + mm < g.M ? (a_kfast ? e % BK : e / BM) : 1 << 30;
    pa[q] = ka[q] < BK ? A + (m0 + mm) * g.sAm + (kbeg + ka[q]) * g.sAk : A;
  }
#pragma unroll
  for (int q = 0; q < NB; ++q) {
    const int e = tid + q * NT, nn = b_nfast ? e % BN : e / BK;
    kb[q] = e < BN * BK && n0 + nn < g.N ? (b_nfast ? e / BN : e % BK) : 1 << 30;
    pb[q] = kb[q] < BK ? B + (n0 + nn) * g.sBn + (kbeg + kb[q]) * g.sBk : B;
  }
  auto fetch = [&](int64_t k0) {
    const int left = (int)min((int64_t)BK, kend - k0);
#pragma unroll
    for (int q = 0; q < NA; ++q) {
      ra[q] = ka[q] < left ? *pa[q] : C{T(0), T(0)};
      pa[q] += BK * g.sAk;
    }
#pragma unroll
    for (int q = 0; q < NB; ++q) {
      rb[q] = kb[q] < left ? *pb[q] : C{T(0), T(0)};
      pb[q] += BK * g.sBk;
    }
  };
  fetch(kbeg);
  for (int64_t k0 = kbeg; k0 < kend; k0 += BK) {
#pragma unroll
    for (int q = 0; q < NA; ++q) {
      const int e = tid + q * NT;
      if (e < BM * BK) As[a_kfast ? e % BK : e / BM][a_kfast ? e / BK : e % BM] = ra[q];
    }
#pragma unroll
    for (int q = 0; q < NB; ++q) {
      const int e = tid + q * NT;
      if (e < BN * BK) Bs[b_nfast ? e / BN : e % BK][b_nfast ? e % BN : e / BK] = rb[q];
    }
    __syncthreads();
    if (k0 + BK < kend) fetch(k0 + BK);
#pragma unroll
    for (int kk = 0; kk < BK; ++kk) {
      C a[TM], bb[TN];
#pragma unroll
      for (int i = 0; i < TM; ++i) a[i] = As[kk][ty + i * RY];
#pragma unroll
      for (int j = 0; j < TN; ++j) bb[j] = Bs[kk][tx + j * RX];
#pragma unroll
      for (int i = 0; i < TM; ++i)
#pragma unroll
        for (int j = 0; j < TN; ++j) {
          acc[i][j].x = fma(a[i].x, bb[j].x, acc[i][j].x);
          acc[i][j].x = fma(-a[i].y, bb[j].y, acc[i][j].x);
          acc[i][j].y = fma(a[i].x, bb[j].y, acc[i][j].y);
          acc[i][j].y = fma(a[i].y, bb[j].x, acc[i][j].y);
        }
    }
    __syncthreads();
  }
  const T ar = (T)g.alr, ai = (T)g.ali;
#pragma unroll
  for (int i = 0; i < TM; ++i) {
    int64_t m = m0 + ty + i * RY;
    if (m >= g.M) continue;
#pragma unroll
    for (int j = 0; j < TN; ++j) {
      int64_t n = n0 + tx + j * RX;
      if (n >= g.N) continue;
      C *dst = Cp + m * g.sCm + n * g.sCn;
      C v = acc[i][j];
      C r;
      r.x = ar * v.x - ai * v.y;
      r.y = ar * v.y + ai * v.x;
      if (g.kchunk > 0) {  // partial sum over this block's K range
        atomicAdd(&dst->x, r.x);
        atomicAdd(&dst->y, r.y);
        continue;
      }
      if (!g.overwrite) {
        C o = *dst;
        r.x += o.x;
        r.y += o.y;
      }
      *dst = r;
    }
  }
}

// The same with one output per thread in a TM x TN tile (TM TN = 256): little padding and many blocks.  In FP64,
// whose pipe does two FMAs per clock and SM, this is the kernel for every size: the pipe is busy 512 clocks per k
// of a 16 x 16 tile, far longer than its loads take, and what counts is that no padded entry is computed and that
// every SM has a block (o=10 v=40: M=40 N=10 K=40 98 us as one 128 x 16 tile, 28 so; M=N=10 K=16000 520 us as
// 64 x 64 tiles, 34 so).  In FP32 it serves the products whose 64 x 64 tiles would leave most SMs idle.
template <typename T, int TM, int TN>
__global__ void __launch_bounds__(256) zgemm_small(GemmArgs g, int64_t b0) {
  using C = typename cpx<T>::t;
  constexpr int BK = TM > 64 || TN > 64 ? 8 : 16, NA = (TM * BK + 255) / 256, NB = (TN * BK + 255) / 256;
  __shared__ C As[BK][TM + 1], Bs[BK][TN + 1];
  const int64_t nMt = (g.M + TM - 1) / TM;
  const int64_t m0 = ((int64_t)blockIdx.x % nMt) * TM, n0 = ((int64_t)blockIdx.x / nMt) * TN, b = b0 + blockIdx.z;
  const C *A = (const C *)g.A + b * g.sAb, *B = (const C *)g.B + b * g.sBb;
  const int tid = threadIdx.x, tn = tid % TN, tm = tid / TN;
  const bool a_kfast = g.sAk == 1, b_nfast = g.sBn == 1;
  const int64_t kbeg = g.kchunk > 0 ? (int64_t)blockIdx.y * g.kchunk : 0;
  const int64_t kend = g.kchunk > 0 ? min(g.K, kbeg + g.kchunk) : g.K;
  C ra[NA], rb[NB];
  auto fetch = [&](int64_t k0) {
#pragma unroll
    for (int q = 0; q < NA; ++q) {
      const int e = tid + q * 256, kk = a_kfast ? e % BK : e / TM, mm = a_kfast ? e / BK : e % TM;
      const int64_t m = m0 + mm, k = k0 + kk;
      ra[q] = (e < TM * BK && m < g.M && k < kend) ? A[m * g.sAm + k * g.sAk] : C{T(0), T(0)};
    }
#pragma unroll
    for (int q = 0; q < NB; ++q) {
      const int e = tid + q * 256, kk = b_nfast ? e / TN : e % BK, nn = b_nfast ? e % TN : e / BK;
      const int64_t n = n0 + nn, k = k0 + kk;
      rb[q] = (e < TN * BK && n < g.N && k < kend) ? B[k * g.sBk + n * g.sBn] : C{T(0), T(0)};
    }
  };
  C acc{T(0), T(0)};
  fetch(kbeg);
  for (int64_t k0 = kbeg; k0 < kend; k0 += BK) {
#pragma unroll
    for (int q = 0; q < NA; ++q) {
      const int e = tid + q * 256;
      if (e < TM * BK) As[a_kfast ? e % BK : e / TM][a_kfast ? e / BK : e % TM] = ra[q];
    }
#pragma unroll
    for (int q = 0; q < NB; ++q) {
      const int e = tid + q * 256;
      if (e < TN * BK) Bs[b_nfast ? e / TN : e % BK][b_nfast ? e % TN : e / BK] = rb[q];
    }
    __syncthreads();
    if (k0 + BK < kend) fetch(k0 + BK);  // the next block's loads overlap this block's sums
    if (m0 + tm < g.M && n0 + tn < g.N) {
      const int nk = (int)min((int64_t)BK, kend - k0);
#pragma unroll 4
      for (int kk = 0; kk < nk; ++kk) {
        const C x = As[kk][tm], y = Bs[kk][tn];
        acc.x = fma(x.x, y.x, acc.x);
        acc.x = fma(-x.y, y.y, acc.x);
        acc.y = fma(x.x, y.y, acc.y);
        acc.y = fma(x.y, y.x, acc.y);
      }
    }
    __syncthreads();
  }
  const int64_t m = m0 + tm, n = n0 + tn;
  if (m >= g.M || n >= g.N) return;
  C *dst = (C *)g.C + b * g.sCb + m * g.sCm + n * g.sCn;
  const T ar = (T)g.alr, ai = (T)g.ali;
  C r;
  r.x = ar * acc.x - ai * acc.y;
  r.y = ar * acc.y + ai * acc.x;
  if (g.kchunk > 0) {
    atomicAdd(&dst->x, r.x);
    atomicAdd(&dst->y, r.y);
    return;
  }
  if (!g.overwrite) {
    const C o = *dst;
    r.x += o.x;
    r.y += o.y;
  }
  *dst = r;
}

void launch_gemm(const GemmArgs &g, int dt, cudaStream_t st) {
  if (g.M <= 0 || g.N <= 0) return;
  if (g.K <= 0) {
    CCLR_REQUIRE(!g.overwrite, "gemm with K=0 and overwrite is not supported");
    return;
  }
  auto tiles_of = [&](int64_t tm, int64_t tn) { return ((g.M + tm - 1) / tm) * ((g.N + tn - 1) / tn); };
  // complex64: 64 x 64 tiles (flat ones for skinny outputs) when they fill two thirds of the SMs
  const int shape = (g.N <= 16 && g.M > 16) ? 1 : (g.M <= 16 && g.N > 16) ? 2 : 0;
  const int64_t big = shape == 1 ? tiles_of(128, 16) : shape == 2 ? tiles_of(16, 128) : tiles_of(64, 64);
  const bool small = dt == C128 || big * g.batch < 100;
  // one output per thread: the tile shape with the least padding (complex64, which its loads bound, keeps the square
  // one down to four columns: 64 x 4 tiles read A three times for N = 11, 37 us against 21)
  int tm = 16, tn = 16;
  if (small && (dt == C128 || std::min(g.M, g.N) <= 4))
    for (int t : {64, 256})
      for (int side = 0; side < 2; ++side) {
        const int m = side == 0 ? t : 256 / t, n = 256 / m;
        if (tiles_of(m, n) < tiles_of(tm, tn)) { tm = m; tn = n; }
      }
  const int64_t tiles = small ? tiles_of(tm, tn) : big;
  // split K over blocks (partial sums added atomically) when the tile grid cannot fill the GPU: at least 32 of K
  // per split in complex128; in complex64 as many splits as the large tiles would take, of at least 64 (twice as
  // many atomic FP32 additions made the error of an o=11 v=67 sigma half as large again)
  int64_t splits = 1;
  const int64_t bk = dt == C128 ? 8 : 16, fill = dt == C128 ? 4 * 152 : 2 * 152, least = dt == C128 ? 32 : 64;
  const int64_t units = (dt == C128 ? tiles : big) * g.batch;
  const bool plain_c = g.sCn == 1 && g.sCm == g.N && (g.batch == 1 || g.sCb == g.M * g.N);
  if (units < fill && g.K >= 2 * least && (!g.overwrite || plain_c) && g.batch <= 65535)
    splits = std::min<int64_t>((fill + units - 1) / units, g.K / least);
  GemmArgs ga = g;
  if (splits > 1) {
    ga.kchunk = ((g.K + splits - 1) / splits + bk - 1) / bk * bk;
    splits = (g.K + ga.kchunk - 1) / ga.kchunk;
    if (g.overwrite) {
      CCLR_CUDA(cudaMemsetAsync(g.C, 0, (size_t)g.batch * g.M * g.N * (dt == C128 ? 16 : 8), st));
      ga.overwrite = 0;
    }
  }
  for (int64_t b0 = 0; b0 < g.batch; b0 += 65535) {
    int64_t nb = std::min<int64_t>(65535, g.batch - b0);
    dim3 grid((unsigned)tiles, (unsigned)splits, (unsigned)nb);
    auto run_small = [&](auto zero) {
      using T = decltype(zero);
      if (tm == 16) zgemm_small<T, 16, 16><<<grid, 256, 0, st>>>(ga, b0);
      else if (tm == 64) zgemm_small<T, 64, 4><<<grid, 256, 0, st>>>(ga, b0);
      else if (tm == 4) zgemm_small<T, 4, 64><<<grid, 256, 0, st>>>(ga, b0);
      else if (tm == 256) zgemm_small<T, 256, 1><<<grid, 256, 0, st>>>(ga, b0);
      else zgemm_small<T, 1, 256><<<grid, 256, 0, st>>>(ga, b0);
    };
    if (dt == C128) run_small(0.0);
    else if (small) run_small(0.0f);
    else if (shape == 1) zgemm_simt<float, 128, 16, 16, 8, 1><<<grid, 256, 0, st>>>(ga, b0);
    else if (shape == 2) zgemm_simt<float, 16, 128, 16, 1, 8><<<grid, 256, 0, st>>>(ga, b0);
    else zgemm_simt<float, 64, 64, 8, 4, 4><<<grid, 256, 0, st>>>(ga, b0);
    count_launch();
    CCLR_CUDA(cudaGetLastError());
  }
}

// out = alpha * v (+ out): arithmetic in double only when either side is complex128 (the
// FP64 pipe of this GPU is far slower than its memory, even for a streaming copy).
template <typename TI, typename TO>
__device__ __forceinline__ typename cpx<TO>::t scale_acc(typename cpx<TI>::t v, double ar, double ai,
                                                         int acc, const typename cpx<TO>::t *dst) {
  using CT = typename std::conditional<sizeof(TI) == 8 || sizeof(TO) == 8, double, float>::type;
  const CT vr = (CT)v.x, vi = (CT)v.y;
  CT wr, wi;
  if (ar == 1.0 && ai == 0.0) { wr = vr; wi = vi; }
  else if (ai == 0.0) { wr = (CT)ar * vr; wi = (CT)ar * vi; }
  else { wr = (CT)ar * vr - (CT)ai * vi; wi = (CT)ar * vi + (CT)ai * vr; }
  typename cpx<TO>::t res;
  if (acc) {
    const typename cpx<TO>::t o = *dst;
    res.x = (TO)(wr + (CT)o.x);
    res.y = (TO)(wi + (CT)o.y);
  } else {
    res.x = (TO)wr;
    res.y = (TO)wi;
  }
  return res;
}

// --------------------------------------------------------------------------------------
// Permute / accumulate: out[idx] = alpha * in[perm idx] (+ out[idx]).  Iterates in the
// order of the output's own mode list (rank <= 8); strides in elements.
// --------------------------------------------------------------------------------------
template <typename TI, typename TO>
__global__ void permute_kernel(PermArgs a) {
  using CI = typename cpx<TI>::t;
  using CO = typename cpx<TO>::t;
  const CI *in = (const CI *)a.in;
  CO *out = (CO *)a.out;
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < a.total;
       e += (int64_t)gridDim.x * blockDim.x) {
    int64_t r = e, oi = 0, oo = 0;
#pragma unroll
    for (int d = 7; d >= 0; --d) {
      if (d >= a.rank) continue;
      int64_t c = r % a.dim[d];
      r /= a.dim[d];
      oi += c * a.sin[d];
      oo += c * a.sout[d];
    }
    out[oo] = scale_acc<TI, TO>(in[oi], a.alr, a.ali, a.acc, out + oo);
  }
}

// Contiguous-enough case: 32-bit index math over at most 4 merged modes.
template <typename TI, typename TO>
__global__ void permute_kernel32(PermArgs a) {
  using CI = typename cpx<TI>::t;
  using CO = typename cpx<TO>::t;
  const CI *in = (const CI *)a.in;
  CO *out = (CO *)a.out;
  const int rank = a.rank;
  const int d0 = (int)a.dim[0], d1 = (int)a.dim[1], d2 = (int)a.dim[2], d3 = (int)a.dim[3];
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < a.total;
       e += (int64_t)gridDim.x * blockDim.x) {
    unsigned r = (unsigned)e;
    int64_t oi = 0, oo = 0;
    if (rank > 3) { unsigned c = r % d3; r /= d3; oi += c * a.sin[3]; oo += c * a.sout[3]; }
    if (rank > 2) { unsigned c = r % d2; r /= d2; oi += c * a.sin[2]; oo += c * a.sout[2]; }
    if (rank > 1) { unsigned c = r % d1; r /= d1; oi += c * a.sin[1]; oo += c * a.sout[1]; }
    oi += (int64_t)r * a.sin[0];
    oo += (int64_t)r * a.sout[0];
    (void)d0;
    out[oo] = scale_acc<TI, TO>(in[oi], a.alr, a.ali, a.acc, out + oo);
  }
}

// Transpose-like case: the input's unit-stride mode (din) is not the output's innermost
// mode (dout).  32 x 32 tiles through shared memory, remaining modes as a batch.
struct TileArgs {
  int64_t Din, Dout;        // extents of the two tiled modes
  int64_t sin_din, sin_dout, sout_din, sout_dout;
  int nb_rank;
  int64_t bdim[6], bsin[6], bsout[6];
  int64_t nbatch;
};

template <typename TI, typename TO>
__global__ void permute_tiled(PermArgs a, TileArgs t) {
  using CI = typename cpx<TI>::t;
  using CO = typename cpx<TO>::t;
  __shared__ CI tile[32][33];
  const CI *in = (const CI *)a.in;
  CO *out = (CO *)a.out;
  const unsigned tin = (unsigned)((t.Din + 31) / 32), tout = (unsigned)((t.Dout + 31) / 32);
  const unsigned per = tin * tout;
  for (unsigned bt = blockIdx.x; bt < (unsigned)t.nbatch * per; bt += gridDim.x) {
    unsigned b = bt / per;
    const unsigned tt = bt - b * per;
    const int64_t i0 = (int64_t)(tt % tin) * 32, o0 = (int64_t)(tt / tin) * 32;
    int64_t bi = 0, bo = 0;
    for (int d = t.nb_rank - 1; d >= 0; --d) {
      const unsigned bd = (unsigned)t.bdim[d];
      const unsigned c = b % bd;
      b /= bd;
      bi += (int64_t)c * t.bsin[d];
      bo += (int64_t)c * t.bsout[d];
    }
    // load: threadIdx.x along din (unit stride in the input)
    for (int r = threadIdx.y; r < 32; r += blockDim.y) {
      const int64_t iin = i0 + threadIdx.x, iout = o0 + r;
      if (iin < t.Din && iout < t.Dout) tile[r][threadIdx.x] = in[bi + iin * t.sin_din + iout * t.sin_dout];
    }
    __syncthreads();
    // store: threadIdx.x along dout (unit stride in the output)
    for (int r = threadIdx.y; r < 32; r += blockDim.y) {
      const int64_t iout = o0 + threadIdx.x, iin = i0 + r;
      if (iin < t.Din && iout < t.Dout) {
        CO *dst = out + bo + iin * t.sout_din + iout * t.sout_dout;
        *dst = scale_acc<TI, TO>(tile[threadIdx.x][r], a.alr, a.ali, a.acc, dst);
      }
    }
    __syncthreads();
  }
}

template <typename TI, typename TO>
static void permute_dispatch(PermArgs a, cudaStream_t st) {
  // merge output-adjacent modes that are also adjacent (same order) in the input
  PermArgs m = a;
  int r = 0;
  for (int d = 0; d < a.rank; ++d) {
    if (r > 0 && m.sout[r - 1] == a.sout[d] * a.dim[d] && m.sin[r - 1] == a.sin[d] * a.dim[d]) {
      m.dim[r - 1] *= a.dim[d];
      m.sout[r - 1] = a.sout[d];
      m.sin[r - 1] = a.sin[d];
    } else {
      m.dim[r] = a.dim[d];
      m.sout[r] = a.sout[d];
      m.sin[r] = a.sin[d];
      ++r;
    }
  }
  m.rank = r;
  const int threads = 256;
  const int64_t blocks = std::min<int64_t>((m.total + threads - 1) / threads, 152 * 32);
  // unit-stride input mode that is not the output's innermost one -> tiled transpose
  int din = -1;
  for (int d = 0; d < m.rank; ++d)
    if (m.sin[d] == 1 && m.dim[d] > 1) din = d;
  const int dout = m.rank - 1;
  if (din >= 0 && din != dout && m.sout[dout] == 1 && m.dim[dout] >= 8 && m.dim[din] >= 8 && m.rank <= 8 &&
      m.total < (1ll << 40)) {
    TileArgs t;
    t.Din = m.dim[din]; t.Dout = m.dim[dout];
    t.sin_din = m.sin[din]; t.sin_dout = m.sin[dout];
    t.sout_din = m.sout[din]; t.sout_dout = m.sout[dout];
    t.nb_rank = 0;
    t.nbatch = 1;
    for (int d = 0; d < m.rank; ++d) {
      if (d == din || d == dout) continue;
      t.bdim[t.nb_rank] = m.dim[d];
      t.bsin[t.nb_rank] = m.sin[d];
      t.bsout[t.nb_rank] = m.sout[d];
      t.nbatch *= m.dim[d];
      ++t.nb_rank;
    }
    const int64_t ntile = t.nbatch * ((t.Din + 31) / 32) * ((t.Dout + 31) / 32);
    CCLR_REQUIRE(ntile < (1ll << 32), "permute: too many tiles");
    permute_tiled<TI, TO><<<(unsigned)std::min<int64_t>(ntile, 152 * 64), dim3(32, 8), 0, st>>>(m, t);
  } else if (m.rank <= 4 && m.total < (1ll << 31)) {
    permute_kernel32<TI, TO><<<(unsigned)blocks, threads, 0, st>>>(m);
  } else {
    permute_kernel<TI, TO><<<(unsigned)blocks, threads, 0, st>>>(m);
  }
}

void launch_permute(const PermArgs &a, int dt_in, int dt_out, cudaStream_t st) {
  if (a.total <= 0) return;
  if (dt_in == C128 && dt_out == C128) permute_dispatch<double, double>(a, st);
  else if (dt_in == C64 && dt_out == C64) permute_dispatch<float, float>(a, st);
  else if (dt_in == C128 && dt_out == C64) permute_dispatch<double, float>(a, st);
  else permute_dispatch<float, double>(a, st);
  count_launch();
  CCLR_CUDA(cudaGetLastError());
}

// --------------------------------------------------------------------------------------
// Antisymmetriser, one pass (o, o, v, v tensors):
//   S[ijab] += Rab[ijab] - Rab[ijba] + Rij[ijab] - Rij[jiab]
//            + R4[ijab] - R4[jiab] - R4[ijba] + R4[jiba]
// and its transpose (dir -1):  Rab += S - S(ab), Rij += S - S(ij), R4 += (1-P(ij))(1-P(ab)) S.
// --------------------------------------------------------------------------------------
template <typename T>
__global__ void antisym_kernel(int o, int v, int dir, const typename cpx<T>::t *Rab_c,
                               const typename cpx<T>::t *Rij_c, const typename cpx<T>::t *R4_c,
                               typename cpx<T>::t *S, typename cpx<T>::t *Rab, typename cpx<T>::t *Rij,
                               typename cpx<T>::t *R4) {
  using C = typename cpx<T>::t;
  const int64_t vv = (int64_t)v * v, n = (int64_t)o * o * vv;
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < n;
       e += (int64_t)gridDim.x * blockDim.x) {
    const int64_t ab = e % vv, ij = e / vv;
    const int a = (int)(ab / v), b = (int)(ab % v), i = (int)(ij / o), j = (int)(ij % o);
    const int64_t e_ba = ij * vv + (int64_t)b * v + a;
    const int64_t e_ji = ((int64_t)j * o + i) * vv + ab;
    const int64_t e_jiba = ((int64_t)j * o + i) * vv + (int64_t)b * v + a;
    if (dir > 0) {
      C r1 = Rab_c[e], r2 = Rab_c[e_ba], r3 = Rij_c[e], r4 = Rij_c[e_ji];
      C q1 = R4_c[e], q2 = R4_c[e_ji], q3 = R4_c[e_ba], q4 = R4_c[e_jiba];
      C s = S[e];
      s.x += r1.x - r2.x + r3.x - r4.x + q1.x - q2.x - q3.x + q4.x;
      s.y += r1.y - r2.y + r3.y - r4.y + q1.y - q2.y - q3.y + q4.y;
      S[e] = s;
    } else {
      const C s1 = S[e], s2 = S[e_ba], s3 = S[e_ji], s4 = S[e_jiba];
      C t;
      t = Rab[e]; t.x += s1.x - s2.x; t.y += s1.y - s2.y; Rab[e] = t;
      t = Rij[e]; t.x += s1.x - s3.x; t.y += s1.y - s3.y; Rij[e] = t;
      t = R4[e]; t.x += s1.x - s3.x - s2.x + s4.x; t.y += s1.y - s3.y - s2.y + s4.y; R4[e] = t;
    }
  }
}

// In-place projection onto tensors antisymmetric in (i,j) and in (a,b):
//   S <- 1/4 (S - S(ij) - S(ab) + S(ij)(ab)); entries with i = j or a = b become zero.
// Each orbit {ijab, jiab, ijba, jiba} is written by the thread of its i<j, a<b member.
template <typename T>
__global__ void antisym_project_kernel(int o, int v, typename cpx<T>::t *S) {
  using C = typename cpx<T>::t;
  const int64_t vv = (int64_t)v * v, n = (int64_t)o * o * vv;
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < n;
       e += (int64_t)gridDim.x * blockDim.x) {
    const int64_t ab = e % vv, ij = e / vv;
    const int a = (int)(ab / v), b = (int)(ab % v), i = (int)(ij / o), j = (int)(ij % o);
    if (i == j || a == b) {
      C z;
      z.x = 0;
      z.y = 0;
      S[e] = z;
    } else if (i < j && a < b) {
      const int64_t e_ba = ij * vv + (int64_t)b * v + a;
      const int64_t e_ji = ((int64_t)j * o + i) * vv + ab;
      const int64_t e_jiba = ((int64_t)j * o + i) * vv + (int64_t)b * v + a;
      const C s1 = S[e], s2 = S[e_ji], s3 = S[e_ba], s4 = S[e_jiba];
      C q;
      q.x = (T)0.25 * (s1.x - s2.x - s3.x + s4.x);
      q.y = (T)0.25 * (s1.y - s2.y - s3.y + s4.y);
      C mq;
      mq.x = -q.x;
      mq.y = -q.y;
      S[e] = q;
      S[e_ji] = mq;
      S[e_ba] = mq;
      S[e_jiba] = q;
    }
  }
}

// ---- tiled forms: one block per orbit {(i,j), (j,i)} x {(A,B), (B,A)} of 32 x 32 (a,b) tiles,
// i <= j and A <= B, so that every element is read and written once and the transposed images
// go through shared memory (coalesced in both orientations).

// the k-th pair (p <= q) of n values, row by row
__device__ __forceinline__ void tri_pair(int64_t k, int n, int &p, int &q) {
  int r = 0;
  while (k >= n - r) {
    k -= n - r;
    ++r;
  }
  p = r;
  q = r + (int)k;
}

template <typename T> __device__ __forceinline__ typename cpx<T>::t cz() {
  typename cpx<T>::t z;
  z.x = 0;
  z.y = 0;
  return z;
}
template <typename C> __device__ __forceinline__ C csub(C a, C b) { a.x -= b.x; a.y -= b.y; return a; }
template <typename C> __device__ __forceinline__ C cadd(C a, C b) { a.x += b.x; a.y += b.y; return a; }
template <typename C, typename T> __device__ __forceinline__ C cscale(C a, T s) { a.x *= s; a.y *= s; return a; }

// S <- 1/4 (S - S(ij) - S(ab) + S(ij)(ab)) in place (zero where i = j or a = b)
template <typename T>
__global__ void __launch_bounds__(256) antisym_project_tiled(int o, int v, typename cpx<T>::t *S) {
  using C = typename cpx<T>::t;
  __shared__ C P[32][33], Q[32][33];
  const int nt = (v + 31) / 32;
  const int64_t ntp = (int64_t)nt * (nt + 1) / 2;
  int i, j, tA, tB;
  tri_pair(blockIdx.x / ntp, o, i, j);
  tri_pair(blockIdx.x % ntp, nt, tA, tB);
  const int a0 = tA * 32, b0 = tB * 32, tx = threadIdx.x;
  const int64_t vv = (int64_t)v * v;
  C *Sij = S + ((int64_t)i * o + j) * vv, *Sji = S + ((int64_t)j * o + i) * vv;
  if (i == j) {
    for (int r = threadIdx.y; r < 32; r += 8) {
      if (a0 + r < v && b0 + tx < v) Sij[(int64_t)(a0 + r) * v + b0 + tx] = cz<T>();
      if (b0 + r < v && a0 + tx < v) Sij[(int64_t)(b0 + r) * v + a0 + tx] = cz<T>();
    }
    return;
  }
  for (int r = threadIdx.y; r < 32; r += 8) {
    int a = a0 + r, b = b0 + tx;
    P[r][tx] = (a < v && b < v) ? csub(Sij[(int64_t)a * v + b], Sji[(int64_t)a * v + b]) : cz<T>();
    b = b0 + r;
    a = a0 + tx;
    Q[r][tx] = (a < v && b < v) ? csub(Sij[(int64_t)b * v + a], Sji[(int64_t)b * v + a]) : cz<T>();
  }
  __syncthreads();
  for (int r = threadIdx.y; r < 32; r += 8) {
    const int a = a0 + r, b = b0 + tx;
    if (a < v && b < v) {
      C q = a == b ? cz<T>() : cscale(csub(P[r][tx], Q[tx][r]), (T)0.25);
      Sij[(int64_t)a * v + b] = q;
      Sji[(int64_t)a * v + b] = cscale(q, (T)-1);
    }
  }
  if (tA != tB)
    for (int r = threadIdx.y; r < 32; r += 8) {
      const int b = b0 + r, a = a0 + tx;
      if (a < v && b < v) {
        C q = cscale(csub(Q[r][tx], P[tx][r]), (T)0.25);
        Sij[(int64_t)b * v + a] = q;
        Sji[(int64_t)b * v + a] = cscale(q, (T)-1);
      }
    }
}

// S += P(ab) Rab + P(ij) Rij + P(ij)P(ab) R4 over one orbit.  With, at (a,b),
//   al_ij = Rab_ij - Rab_ij^T, al_ji likewise, be = Rij_ij - Rij_ji, ga = R4_ij - R4_ji - (R4_ij - R4_ji)^T
// and beT = (Rij_ij - Rij_ji) at (b,a):
//   S_ij(a,b) += al_ij + be + ga,  S_ji(a,b) += al_ji - be - ga,
//   S_ij(b,a) += -al_ij - ga + beT, S_ji(b,a) += -al_ji + ga - beT.
template <typename T>
__global__ void __launch_bounds__(256) antisym_apply_tiled(int o, int v, typename cpx<T>::t *S,
                                                           const typename cpx<T>::t *Rab,
                                                           const typename cpx<T>::t *Rij,
                                                           const typename cpx<T>::t *R4) {
  using C = typename cpx<T>::t;
  extern __shared__ __align__(16) unsigned char smem_as[];
  C(*T1)[33] = reinterpret_cast<C(*)[33]>(smem_as);   // Rab_ij at (b,a), later U1
  C(*T2)[33] = T1 + 32;                               // Rab_ji at (b,a), later U2
  C(*T3)[33] = T1 + 64;                               // (R4_ij - R4_ji) at (b,a)
  C(*T4)[33] = T1 + 96;                               // (Rij_ij - Rij_ji) at (b,a)
  const int nt = (v + 31) / 32;
  const int64_t ntp = (int64_t)nt * (nt + 1) / 2;
  int i, j, tA, tB;
  tri_pair(blockIdx.x / ntp, o, i, j);
  tri_pair(blockIdx.x % ntp, nt, tA, tB);
  const int a0 = tA * 32, b0 = tB * 32, tx = threadIdx.x;
  const int64_t vv = (int64_t)v * v, oij = ((int64_t)i * o + j) * vv, oji = ((int64_t)j * o + i) * vv;
  const bool same = i == j;
  for (int r = threadIdx.y; r < 32; r += 8) {
    const int b = b0 + r, a = a0 + tx;
    const bool in = a < v && b < v;
    const int64_t e = (int64_t)b * v + a;
    T1[r][tx] = in ? Rab[oij + e] : cz<T>();
    T2[r][tx] = in ? Rab[oji + e] : cz<T>();
    T3[r][tx] = in ? csub(R4[oij + e], R4[oji + e]) : cz<T>();
    T4[r][tx] = in ? csub(Rij[oij + e], Rij[oji + e]) : cz<T>();
  }
  __syncthreads();
  C u1[4], u2[4];
  for (int k = 0, r = threadIdx.y; r < 32; r += 8, ++k) {
    const int a = a0 + r, b = b0 + tx;
    u1[k] = cz<T>();
    u2[k] = cz<T>();
    if (!(a < v && b < v)) continue;
    const int64_t e = (int64_t)a * v + b;
    const C al_ij = csub(Rab[oij + e], T1[tx][r]);
    const C al_ji = csub(Rab[oji + e], T2[tx][r]);
    const C be = csub(Rij[oij + e], Rij[oji + e]);
    const C ga = csub(csub(R4[oij + e], R4[oji + e]), T3[tx][r]);
    if (same) {
      S[oij + e] = cadd(S[oij + e], al_ij);
    } else {
      S[oij + e] = cadd(S[oij + e], cadd(al_ij, cadd(be, ga)));
      S[oji + e] = cadd(S[oji + e], csub(al_ji, cadd(be, ga)));
    }
    u1[k] = cscale(cadd(al_ij, ga), (T)-1);
    u2[k] = csub(ga, al_ji);
  }
  if (tA == tB) return;  // the tile holds both (a,b) and (b,a): done
  __syncthreads();
  for (int k = 0, r = threadIdx.y; r < 32; r += 8, ++k) {
    T1[r][tx] = u1[k];
    T2[r][tx] = u2[k];
  }
  __syncthreads();
  for (int r = threadIdx.y; r < 32; r += 8) {
    const int b = b0 + r, a = a0 + tx;
    if (!(a < v && b < v)) continue;
    const int64_t e = (int64_t)b * v + a;
    if (same) {
      S[oij + e] = cadd(S[oij + e], T1[tx][r]);  // -al_ij at (a,b) (ga = 0 when i = j)
    } else {
      S[oij + e] = cadd(S[oij + e], cadd(T1[tx][r], T4[r][tx]));
      S[oji + e] = cadd(S[oji + e], csub(T2[tx][r], T4[r][tx]));
    }
  }
}

static int64_t orbit_blocks(int o, int v) {
  const int64_t nt = (v + 31) / 32;
  return (int64_t)o * (o + 1) / 2 * (nt * (nt + 1) / 2);
}

void antisym_project(int dt, int o, int v, void *S, cudaStream_t st) {
  const int64_t nb = orbit_blocks(o, v);
  CCLR_REQUIRE(nb < (1ll << 31), "antisym_project: too many tiles");
  if (dt == C128) antisym_project_tiled<double><<<(unsigned)nb, dim3(32, 8), 0, st>>>(o, v, (double2 *)S);
  else antisym_project_tiled<float><<<(unsigned)nb, dim3(32, 8), 0, st>>>(o, v, (float2 *)S);
  count_launch();
  CCLR_CUDA(cudaGetLastError());
}

void antisym_apply(int dt, int o, int v, int dir, void *S, void *Rab, void *Rij, void *R4, cudaStream_t st) {
  if (dir > 0) {
    const int64_t nb = orbit_blocks(o, v);
    CCLR_REQUIRE(nb < (1ll << 31), "antisym_apply: too many tiles");
    const size_t smem = (size_t)4 * 32 * 33 * (dt == C128 ? 16 : 8);
    static std::atomic<unsigned long long> attr_set{0};  // one bit per device
    int dev = 0;
    CCLR_CUDA(cudaGetDevice(&dev));
    if (dev < 64 && !(attr_set.load() & (1ull << dev))) {  // the complex128 tiles take 67 KB of shared memory
      CCLR_CUDA(cudaFuncSetAttribute(antisym_apply_tiled<double>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                     (int)((size_t)4 * 32 * 33 * 16)));
      attr_set |= 1ull << dev;
    }
    if (dt == C128)
      antisym_apply_tiled<double><<<(unsigned)nb, dim3(32, 8), smem, st>>>(o, v, (double2 *)S, (const double2 *)Rab,
                                                                          (const double2 *)Rij, (const double2 *)R4);
    else
      antisym_apply_tiled<float><<<(unsigned)nb, dim3(32, 8), smem, st>>>(o, v, (float2 *)S, (const float2 *)Rab,
                                                                         (const float2 *)Rij, (const float2 *)R4);
    count_launch();
    CCLR_CUDA(cudaGetLastError());
    return;
  }
  const int64_t n = (int64_t)o * o * v * v;
  const unsigned g = (unsigned)std::max<int64_t>(1, std::min<int64_t>((n + 255) / 256, 152 * 32));
  if (dt == C128)
    antisym_kernel<double><<<g, 256, 0, st>>>(o, v, dir, (const double2 *)Rab, (const double2 *)Rij,
                                              (const double2 *)R4, (double2 *)S, (double2 *)Rab,
                                              (double2 *)Rij, (double2 *)R4);
  else
    antisym_kernel<float><<<g, 256, 0, st>>>(o, v, dir, (const float2 *)Rab, (const float2 *)Rij,
                                             (const float2 *)R4, (float2 *)S, (float2 *)Rab, (float2 *)Rij,
                                             (float2 *)R4);
  count_launch();
  CCLR_CUDA(cudaGetLastError());
}

// --------------------------------------------------------------------------------------
// Vector kernels (contiguous complex arrays).
// --------------------------------------------------------------------------------------
template <typename T>
__global__ void axpy_kernel(int64_t n, double ar, double ai, const typename cpx<T>::t *x,
                            typename cpx<T>::t *y) {
  // a real scale takes half the FP64 operations (this GPU's FP64 rate, not HBM, bounds the
  // complex128 vector kernels)
  if (ai == 0.0) {
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n;
         i += (int64_t)gridDim.x * blockDim.x) {
      auto xv = x[i];
      auto yv = y[i];
      yv.x += (T)(ar * xv.x);
      yv.y += (T)(ar * xv.y);
      y[i] = yv;
    }
    return;
  }
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n;
       i += (int64_t)gridDim.x * blockDim.x) {
    auto xv = x[i];
    auto yv = y[i];
    yv.x += (T)(ar * xv.x - ai * xv.y);
    yv.y += (T)(ar * xv.y + ai * xv.x);
    y[i] = yv;
  }
}

template <typename T>
__global__ void scal_kernel(int64_t n, double ar, double ai, typename cpx<T>::t *y) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n;
       i += (int64_t)gridDim.x * blockDim.x) {
    auto v = y[i];
    typename cpx<T>::t r;
    r.x = (T)(ar * v.x - ai * v.y);
    r.y = (T)(ar * v.y + ai * v.x);
    y[i] = r;
  }
}

static unsigned grid_for(int64_t n) {
  int64_t b = (n + 255) / 256;
  return (unsigned)std::max<int64_t>(1, std::min<int64_t>(b, 152 * 16));
}

void vec_axpy(int dt, int64_t n, zc a, const void *x, void *y, cudaStream_t st) {
  if (n <= 0) return;
  if (dt == C128) axpy_kernel<double><<<grid_for(n), 256, 0, st>>>(n, a.re, a.im, (const double2 *)x, (double2 *)y);
  else axpy_kernel<float><<<grid_for(n), 256, 0, st>>>(n, a.re, a.im, (const float2 *)x, (float2 *)y);
  count_launch();
    CCLR_CUDA(cudaGetLastError());
}

void vec_scal(int dt, int64_t n, zc a, void *y, cudaStream_t st) {
  if (n <= 0) return;
  if (dt == C128) scal_kernel<double><<<grid_for(n), 256, 0, st>>>(n, a.re, a.im, (double2 *)y);
  else scal_kernel<float><<<grid_for(n), 256, 0, st>>>(n, a.re, a.im, (float2 *)y);
  count_launch();
    CCLR_CUDA(cudaGetLastError());
}

// Dot products with FP64 accumulation: mode 0 bilinear sum x*y, mode 1 Hermitian
// sum conj(x)*y.  Two passes (block partials, then one block) for a deterministic result.
template <typename T>
__global__ void dot_partial(int64_t n, const typename cpx<T>::t *x, const typename cpx<T>::t *y,
                            int herm, double2 *part) {
  double sr = 0.0, si = 0.0;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n;
       i += (int64_t)gridDim.x * blockDim.x) {
    double xr = x[i].x, xi = herm ? -(double)x[i].y : (double)x[i].y;
    double yr = y[i].x, yi = y[i].y;
    sr += xr * yr - xi * yi;
    si += xr * yi + xi * yr;
  }
  for (int o = 16; o > 0; o >>= 1) {
    sr += __shfl_down_sync(0xffffffffu, sr, o);
    si += __shfl_down_sync(0xffffffffu, si, o);
  }
  __shared__ double rs[32], is[32];
  int w = threadIdx.x / 32, l = threadIdx.x % 32;
  if (l == 0) { rs[w] = sr; is[w] = si; }
  __syncthreads();
  if (w == 0) {
    int nw = blockDim.x / 32;
    sr = l < nw ? rs[l] : 0.0;
    si = l < nw ? is[l] : 0.0;
    for (int o = 16; o > 0; o >>= 1) {
      sr += __shfl_down_sync(0xffffffffu, sr, o);
      si += __shfl_down_sync(0xffffffffu, si, o);
    }
    if (l == 0) part[blockIdx.x] = make_double2(sr, si);
  }
}

__global__ void dot_final(int nb, const double2 *part, double2 *out, int slot) {
  double sr = 0.0, si = 0.0;
  for (int i = threadIdx.x; i < nb; i += blockDim.x) {
    sr += part[i].x;
    si += part[i].y;
  }
  for (int o = 16; o > 0; o >>= 1) {
    sr += __shfl_down_sync(0xffffffffu, sr, o);
    si += __shfl_down_sync(0xffffffffu, si, o);
  }
  __shared__ double rs[32], is[32];
  int w = threadIdx.x / 32, l = threadIdx.x % 32;
  if (l == 0) { rs[w] = sr; is[w] = si; }
  __syncthreads();
  if (w == 0) {
    int nw = blockDim.x / 32;
    sr = l < nw ? rs[l] : 0.0;
    si = l < nw ? is[l] : 0.0;
    for (int o = 16; o > 0; o >>= 1) {
      sr += __shfl_down_sync(0xffffffffu, sr, o);
      si += __shfl_down_sync(0xffffffffu, si, o);
    }
    if (l == 0) out[slot] = make_double2(sr, si);
  }
}

void vec_dot(int dt, int64_t n, const void *x, const void *y, int herm, double2 *part,
             double2 *out, int slot, cudaStream_t st) {
  const int nb = 304;
  if (n <= 0) {
    CCLR_CUDA(cudaMemsetAsync(out + slot, 0, sizeof(double2), st));
    return;
  }
  if (dt == C128) dot_partial<double><<<nb, 256, 0, st>>>(n, (const double2 *)x, (const double2 *)y, herm, part);
  else dot_partial<float><<<nb, 256, 0, st>>>(n, (const float2 *)x, (const float2 *)y, herm, part);
  dot_final<<<1, 256, 0, st>>>(nb, part, out, slot);
  count_launch(2);
    CCLR_CUDA(cudaGetLastError());
}

// 1/x in FP64 by Newton-Raphson iteration for the reciprocal, y <- y (2 - x y), from the FP32
// reciprocal: each step squares the relative error (2^-24 -> 2^-48 -> below FP64 rounding), so two
// steps give the FP64 reciprocal to about an ulp with four FP64 FMAs instead of an FP64 division
// (this GPU's FP64 rate bounds the preconditioner). For normal x within FP32 range.
__device__ __forceinline__ double recip_newton(double x) {
  double y = (double)__frcp_rn((float)x);
  y = fma(y, fma(-x, y, 1.0), y);
  y = fma(y, fma(-x, y, 1.0), y);
  return y;
}

// Delta = r / (D - omega), D real; in place allowed.
template <typename T>
__global__ void precond_kernel(int64_t n, const double *D, double omega, double omega_im,
                               const typename cpx<T>::t *r, typename cpx<T>::t *out) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n;
       i += (int64_t)gridDim.x * blockDim.x) {
    auto v = r[i];
    typename cpx<T>::t o;
    if (omega_im == 0.0) {
      double d = D[i] - omega;
      if (fabs(d) < 1e-8) d = d < 0 ? -1e-8 : 1e-8;
      const double q = recip_newton(d);
      o.x = (T)(v.x * q);
      o.y = (T)(v.y * q);
    } else {  // v / (d - i w_im) = v (d + i w_im) / (d^2 + w_im^2)
      const double d = D[i] - omega, q = recip_newton(d * d + omega_im * omega_im);
      o.x = (T)((v.x * d - v.y * omega_im) * q);
      o.y = (T)((v.y * d + v.x * omega_im) * q);
    }
    out[i] = o;
  }
}

void vec_precond(int dt, int64_t n, const double *D, double omega, double omega_im, const void *r, void *out,
                 cudaStream_t st) {
  if (n <= 0) return;
  if (dt == C128)
    precond_kernel<double><<<grid_for(n), 256, 0, st>>>(n, D, omega, omega_im, (const double2 *)r, (double2 *)out);
  else
    precond_kernel<float><<<grid_for(n), 256, 0, st>>>(n, D, omega, omega_im, (const float2 *)r, (float2 *)out);
  count_launch();
    CCLR_CUDA(cudaGetLastError());
}

// pair (p < q) of n indices -> its row-major position among all pairs, and back
__host__ __device__ __forceinline__ int64_t pair_id(int64_t p, int64_t q, int64_t n) {
  return p * n - p * (p + 1) / 2 + (q - p - 1);
}
__device__ __forceinline__ void pair_of(int64_t k, int n, int &p, int &q) {
  // p = largest row with start(p) = p n - p (p + 1) / 2 <= k: the root of the quadratic in
  // single precision (this GPU's FP64 rate is low), then corrected by whole steps
  const float nn = 2.0f * (float)n - 1.0f;
  int r = (int)((nn - sqrtf(fmaxf(0.0f, nn * nn - 8.0f * (float)k))) * 0.5f);
  r = max(0, min(r, n - 2));
  while (r > 0 && pair_id(r, r + 1, n) > k) --r;
  while (r < n - 2 && pair_id(r + 1, r + 2, n) <= k) ++r;
  p = r;
  q = (int)(k - pair_id(r, r + 1, n)) + r + 1;
}

// D1[i,a] = Fvv_aa - Foo_ii ; D2p[(i<j),(a<b)] = Fvv_aa + Fvv_bb - Foo_ii - Foo_jj (real parts).
__global__ void diag_kernel(int o, int v, const double2 *Foo, const double2 *Fvv, double *D1, double *D2p) {
  const int64_t n1 = (int64_t)o * v;
  const int64_t Pv = (int64_t)v * (v - 1) / 2, n2 = (int64_t)o * (o - 1) / 2 * Pv;
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < n1 + n2;
       e += (int64_t)gridDim.x * blockDim.x) {
    if (e < n1) {
      int i = (int)(e / v), a = (int)(e % v);
      D1[e] = Fvv[(int64_t)a * v + a].x - Foo[(int64_t)i * o + i].x;
    } else {
      const int64_t r = e - n1;
      int i, j, a, b;
      pair_of(r / Pv, o, i, j);
      pair_of(r % Pv, v, a, b);
      D2p[r] = Fvv[(int64_t)a * v + a].x + Fvv[(int64_t)b * v + b].x - Foo[(int64_t)i * o + i].x -
               Foo[(int64_t)j * o + j].x;
    }
  }
}

// Y[p][j][q] += alpha * sum_k S(k, j) X[p][k][q] for short k and j (at most 64 each): the
// o x o matrices acting on one occupied index of an o^2 v^2 tensor.  One block of 128 threads takes
// 128 consecutive q of one p: S is staged in shared memory (broadcast reads), each thread copies its
// own column X[p][.][q] into shared memory once and forms eight j at a time from it, so X is read
// once and Y read and written once, all coalesced along q.
template <typename T>
__global__ void __launch_bounds__(128) smallk_kernel(int64_t P, int K, int J, int64_t Q,
                                                     const typename cpx<T>::t *__restrict__ S, int64_t sSk,
                                                     int64_t sSj, const typename cpx<T>::t *__restrict__ X,
                                                     int64_t sXp, int64_t sXk, typename cpx<T>::t *__restrict__ Y,
                                                     int64_t sYp, int64_t sYj, T ar, T ai) {
  using C2 = typename cpx<T>::t;
  extern __shared__ __align__(16) unsigned char smk_raw[];
  C2 *Ss = (C2 *)smk_raw;     // [K][J]
  C2 *Xs = Ss + K * J;         // [K][128], column threadIdx.x private to its thread
  for (int e = threadIdx.x; e < K * J; e += blockDim.x) {
    const int k = e / J, j = e % J;
    Ss[e] = S[(int64_t)k * sSk + (int64_t)j * sSj];
  }
  __syncthreads();
  const int64_t nqt = (Q + 127) / 128;
  for (int64_t t = blockIdx.x; t < P * nqt; t += gridDim.x) {
    const int64_t p = t / nqt, q = (t % nqt) * 128 + threadIdx.x;
    if (q >= Q) continue;
    const C2 *xp = X + p * sXp + q;
    // the column in batches of eight independent loads (latency overlapped), then to shared memory
    for (int k0 = 0; k0 < K; k0 += 8) {
      C2 xv[8];
#pragma unroll
      for (int u = 0; u < 8; ++u)
        if (k0 + u < K) xv[u] = xp[(int64_t)(k0 + u) * sXk];
#pragma unroll
      for (int u = 0; u < 8; ++u)
        if (k0 + u < K) Xs[(k0 + u) * 128 + threadIdx.x] = xv[u];
    }
    C2 *yp = Y + p * sYp + q;
    for (int j0 = 0; j0 < J; j0 += 8) {
      // the eight outputs' old values are loaded first, so their latency overlaps the sums
      C2 yv[8];
#pragma unroll
      for (int u = 0; u < 8; ++u)
        if (j0 + u < J) yv[u] = yp[(int64_t)(j0 + u) * sYj];
      T re[8], im[8];
#pragma unroll
      for (int u = 0; u < 8; ++u) { re[u] = 0; im[u] = 0; }
      for (int k = 0; k < K; ++k) {
        const C2 x = Xs[k * 128 + threadIdx.x];
        const C2 *sr = Ss + k * J + j0;
#pragma unroll
        for (int u = 0; u < 8; ++u) {
          if (j0 + u < J) {
            const C2 sv = sr[u];
            re[u] += sv.x * x.x - sv.y * x.y;
            im[u] += sv.x * x.y + sv.y * x.x;
          }
        }
      }
#pragma unroll
      for (int u = 0; u < 8; ++u) {
        if (j0 + u < J) {
          C2 y = yv[u];
          y.x += ar * re[u] - ai * im[u];
          y.y += ar * im[u] + ai * re[u];
          yp[(int64_t)(j0 + u) * sYj] = y;
        }
      }
    }
  }
}

// The complex64 case with k <= 32: each thread keeps two columns X[p][.][q], X[p][.][q + 128] in registers (all loads
// issued at once; KT is k rounded up to 8, S zero beyond), prefetches four outputs of each, and reads S two entries per
// load from shared memory, eight loads' issue time for 32 FMAs' (with one column and one entry per load the loads
// took as long as the FMAs: 32 x 32 on 32 x 32 x 240 x 240, 0.80 ms; the FMAs alone are 0.20, the memory 0.21).
template <int KT>
__global__ void __launch_bounds__(128) smallk_reg_kernel(int64_t P, int K, int J, int64_t Q,
                                                         const float2 *__restrict__ S, int64_t sSk, int64_t sSj,
                                                         const float2 *__restrict__ X, int64_t sXp, int64_t sXk,
                                                         float2 *__restrict__ Y, int64_t sYp, int64_t sYj, float ar,
                                                         float ai) {
  extern __shared__ __align__(16) unsigned char smr_raw[];
  float2 *Ss = (float2 *)smr_raw;  // [KT][JP], JP = J rounded up to 4
  const int JP = (J + 3) & ~3;
  for (int e = threadIdx.x; e < KT * JP; e += blockDim.x) {
    const int k = e / JP, j = e % JP;
    Ss[e] = k < K && j < J ? S[(int64_t)k * sSk + (int64_t)j * sSj] : make_float2(0.f, 0.f);
  }
  __syncthreads();
  const int64_t nqt = (Q + 255) / 256;
  for (int64_t t = blockIdx.x; t < P * nqt; t += gridDim.x) {
    const int64_t p = t / nqt, q = (t % nqt) * 256 + threadIdx.x;
    const bool in[2] = {q < Q, q + 128 < Q};
    if (!in[0]) continue;
    const float2 *xp = X + p * sXp + q;
    float2 x[2][KT];
#pragma unroll
    for (int k = 0; k < KT; ++k)
#pragma unroll
      for (int c = 0; c < 2; ++c)
        x[c][k] = k < K && in[c] ? xp[(int64_t)k * sXk + c * 128] : make_float2(0.f, 0.f);
    float2 *yp = Y + p * sYp + q;
    for (int j0 = 0; j0 < J; j0 += 4) {
      float2 yv[2][4], acc[2][4];
#pragma unroll
      for (int c = 0; c < 2; ++c)
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          yv[c][u] = j0 + u < J && in[c] ? yp[(int64_t)(j0 + u) * sYj + c * 128] : make_float2(0.f, 0.f);
          acc[c][u] = make_float2(0.f, 0.f);
        }
#pragma unroll
      for (int k = 0; k < KT; ++k) {
        const float4 s01 = *reinterpret_cast<const float4 *>(Ss + k * JP + j0);
        const float4 s23 = *reinterpret_cast<const float4 *>(Ss + k * JP + j0 + 2);
        const float2 sv[4] = {make_float2(s01.x, s01.y), make_float2(s01.z, s01.w), make_float2(s23.x, s23.y),
                              make_float2(s23.z, s23.w)};
#pragma unroll
        for (int c = 0; c < 2; ++c)
#pragma unroll
          for (int u = 0; u < 4; ++u) {
            acc[c][u].x += sv[u].x * x[c][k].x - sv[u].y * x[c][k].y;
            acc[c][u].y += sv[u].x * x[c][k].y + sv[u].y * x[c][k].x;
          }
      }
#pragma unroll
      for (int c = 0; c < 2; ++c)
#pragma unroll
        for (int u = 0; u < 4; ++u)
          if (j0 + u < J && in[c]) {
            float2 y = yv[c][u];
            y.x += ar * acc[c][u].x - ai * acc[c][u].y;
            y.y += ar * acc[c][u].y + ai * acc[c][u].x;
            yp[(int64_t)(j0 + u) * sYj + c * 128] = y;
          }
    }
  }
}

void contract_smallk(int dt, int64_t P, int K, int J, int64_t Q, const void *S, int64_t sSk, int64_t sSj,
                     const void *X, int64_t sXp, int64_t sXk, void *Y, int64_t sYp, int64_t sYj, zc alpha,
                     cudaStream_t st) {
  CCLR_REQUIRE(K >= 1 && K <= 64 && J >= 1 && J <= 64, "contract_smallk: k and j extents must be 1..64");
  if (P == 0 || Q == 0) return;
  const size_t es = dt == C128 ? 16 : 8;
  const size_t smem = (size_t)K * J * es + (size_t)K * 128 * es;  // at most 192 KB (complex128)
  static std::atomic<unsigned long long> attr_set{0};               // one bit per device
  int dev = 0;
  CCLR_CUDA(cudaGetDevice(&dev));
  if (dev < 64 && !(attr_set.load() & (1ull << dev))) {
    CCLR_CUDA(cudaFuncSetAttribute(smallk_kernel<double>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                   (int)((size_t)64 * 64 * 16 + (size_t)64 * 128 * 16)));
    CCLR_CUDA(cudaFuncSetAttribute(smallk_kernel<float>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                   (int)((size_t)64 * 64 * 8 + (size_t)64 * 128 * 8)));
    attr_set |= 1ull << dev;
  }
  const int64_t tiles = P * ((Q + 127) / 128);
  const unsigned grid = (unsigned)std::min<int64_t>(tiles, (int64_t)152 * 16);
  if (dt == C64 && K <= 32) {
    const int64_t t2 = P * ((Q + 255) / 256);
    const unsigned g2 = (unsigned)std::min<int64_t>(t2, (int64_t)152 * 16);
    auto go = [&](auto kt) {
      constexpr int KT = decltype(kt)::value;
      smallk_reg_kernel<KT><<<g2, 128, (size_t)KT * ((J + 3) & ~3) * 8, st>>>(
          P, K, J, Q, (const float2 *)S, sSk, sSj, (const float2 *)X, sXp, sXk, (float2 *)Y, sYp, sYj, (float)alpha.re,
          (float)alpha.im);
    };
    if (K <= 8) go(std::integral_constant<int, 8>());
    else if (K <= 16) go(std::integral_constant<int, 16>());
    else if (K <= 24) go(std::integral_constant<int, 24>());
    else go(std::integral_constant<int, 32>());
    count_launch();
    CCLR_CUDA(cudaGetLastError());
    return;
  }
  if (dt == C128)
    smallk_kernel<double><<<grid, 128, smem, st>>>(P, K, J, Q, (const double2 *)S, sSk, sSj, (const double2 *)X, sXp,
                                                   sXk, (double2 *)Y, sYp, sYj, alpha.re, alpha.im);
  else
    smallk_kernel<float><<<grid, 128, smem, st>>>(P, K, J, Q, (const float2 *)S, sSk, sSj, (const float2 *)X, sXp,
                                                  sXk, (float2 *)Y, sYp, sYj, (float)alpha.re, (float)alpha.im);
  count_launch();
  CCLR_CUDA(cudaGetLastError());
}

// y[r] += alpha * sum_c B[x] s[c] for a rank-4 tensor B whose modes are each either an output mode
// (r) or a contracted mode (c), s holding only contracted modes: the matrix-vector products of an
// o^2 v^2 tensor with an o x v vector.  One block per (x0, x1) reads the contiguous slab
// B[x0][x1][.][.] once, sums into shared-memory partials over the slab's output index (at most one
// of the two slab modes is an output mode), and adds them to y with atomics.
template <typename T>
__device__ __forceinline__ T warp_sum(T x) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
  return x;
}

template <typename T>
__global__ void __launch_bounds__(256) slab_gemv_kernel(int64_t d0, int64_t d1, int64_t d2, int64_t d3,
                                                        int rmask, const typename cpx<T>::t *B,
                                                        const typename cpx<T>::t *S, int64_t s0, int64_t s1,
                                                        int64_t s2, int64_t s3, typename cpx<T>::t *Y,
                                                        int64_t y0, int64_t y1, int64_t y2, int64_t y3, T ar,
                                                        T ai) {
  using C2 = typename cpx<T>::t;
  extern __shared__ __align__(16) unsigned char sg_raw[];
  T *part = (T *)sg_raw;  // [np][2]
  const bool r2 = rmask & 4, r3 = rmask & 8;
  const int64_t np = r2 ? d2 : (r3 ? d3 : 1);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nwarps = blockDim.x >> 5;
  for (int64_t t = blockIdx.x; t < d0 * d1; t += gridDim.x) {
    const int64_t x0 = t / d1, x1 = t % d1;
    for (int64_t e = threadIdx.x; e < 2 * np; e += blockDim.x) part[e] = 0;
    __syncthreads();
    const C2 *slab = B + t * d2 * d3;
    const C2 *sb = S + ((rmask & 1) ? 0 : x0 * s0) + ((rmask & 2) ? 0 : x1 * s1);
    if (r2) {  // one warp per row x2, lanes along the contiguous contracted x3
      for (int64_t x2 = warp; x2 < d2; x2 += nwarps) {
        T re = 0, im = 0;
#pragma unroll 4
        for (int64_t x3 = lane; x3 < d3; x3 += 32) {
          const C2 b = slab[x2 * d3 + x3], sv = sb[x3 * s3];
          re += b.x * sv.x - b.y * sv.y;
          im += b.x * sv.y + b.y * sv.x;
        }
        re = warp_sum(re);
        im = warp_sum(im);
        if (lane == 0) { part[2 * x2] = re; part[2 * x2 + 1] = im; }
      }
    } else {  // thread groups over rows x2, threads along x3 (the output index, or contracted too)
      const int64_t w3 = d3 < (int64_t)blockDim.x ? d3 : (int64_t)blockDim.x;
      const int64_t G = blockDim.x / w3, g = threadIdx.x / w3, c = threadIdx.x % w3;
      if (g < G) {
        for (int64_t x3 = c; x3 < d3; x3 += w3) {
          T re = 0, im = 0;
#pragma unroll 8
          for (int64_t x2 = g; x2 < d2; x2 += G) {
            const C2 b = slab[x2 * d3 + x3], sv = sb[(r3 ? 0 : x3 * s3) + x2 * s2];
            re += b.x * sv.x - b.y * sv.y;
            im += b.x * sv.y + b.y * sv.x;
          }
          const int64_t pi = r3 ? x3 : 0;
          atomicAdd(&part[2 * pi], re);
          atomicAdd(&part[2 * pi + 1], im);
        }
      }
    }
    __syncthreads();
    const int64_t yb = ((rmask & 1) ? x0 * y0 : 0) + ((rmask & 2) ? x1 * y1 : 0);
    for (int64_t pi = threadIdx.x; pi < np; pi += blockDim.x) {
      const T re = part[2 * pi], im = part[2 * pi + 1];
      T *yp = (T *)(Y + yb + (r2 ? pi * y2 : 0) + (r3 ? pi * y3 : 0));
      atomicAdd(yp, ar * re - ai * im);
      atomicAdd(yp + 1, ar * im + ai * re);
    }
    __syncthreads();
  }
}

void contract_slab_gemv(int dt, const int64_t *d, int rmask, const void *B, const void *S, const int64_t *ss,
                        void *Y, const int64_t *ys, zc alpha, cudaStream_t st) {
  CCLR_REQUIRE(!((rmask & 4) && (rmask & 8)), "contract_slab_gemv: at most one slab mode may be an output mode");
  if (d[0] * d[1] * d[2] * d[3] == 0) return;
  const int64_t np = (rmask & 4) ? d[2] : ((rmask & 8) ? d[3] : 1);
  const size_t smem = (size_t)np * 2 * (dt == C128 ? 8 : 4);
  CCLR_REQUIRE(smem <= 48 * 1024, "contract_slab_gemv: slab output index too long");
  const unsigned grid = (unsigned)std::min<int64_t>(d[0] * d[1], (int64_t)152 * 8);
  if (dt == C128)
    slab_gemv_kernel<double><<<grid, 256, smem, st>>>(d[0], d[1], d[2], d[3], rmask, (const double2 *)B,
                                                      (const double2 *)S, ss[0], ss[1], ss[2], ss[3], (double2 *)Y,
                                                      ys[0], ys[1], ys[2], ys[3], alpha.re, alpha.im);
  else
    slab_gemv_kernel<float><<<grid, 256, smem, st>>>(d[0], d[1], d[2], d[3], rmask, (const float2 *)B,
                                                     (const float2 *)S, ss[0], ss[1], ss[2], ss[3], (float2 *)Y, ys[0],
                                                     ys[1], ys[2], ys[3], (float)alpha.re, (float)alpha.im);
  count_launch();
  CCLR_CUDA(cudaGetLastError());
}

// y[r] += alpha sum_p B[p][r] w[p] for a contiguous [P][R] array: threads along r, blocks over ranges of p whose
// partial sums are added with atomics; one coalesced pass over B (memory-bound: 800 x 25600 complex64 113 us as a
// GEMM with one column).
template <typename T>
__global__ void __launch_bounds__(256) colsum_gemv_kernel(int64_t P, int64_t R, int64_t step, const typename cpx<T>::t *__restrict__ B,
                                                          const typename cpx<T>::t *__restrict__ w, int64_t sw,
                                                          typename cpx<T>::t *__restrict__ y, T ar, T ai) {
  const int64_t r = (int64_t)blockIdx.x * 256 + threadIdx.x;
  if (r >= R) return;
  const int64_t p1 = min(P, (int64_t)(blockIdx.y + 1) * step);
  T re = 0, im = 0;
#pragma unroll 8
  for (int64_t p = (int64_t)blockIdx.y * step; p < p1; ++p) {
    const auto b = B[p * R + r], s = w[p * sw];
    re += b.x * s.x - b.y * s.y;
    im += b.x * s.y + b.y * s.x;
  }
  atomicAdd(&y[r].x, ar * re - ai * im);
  atomicAdd(&y[r].y, ar * im + ai * re);
}

void contract_colsum_gemv(int dt, int64_t P, int64_t R, const void *B, const void *w, int64_t sw, void *y, zc alpha,
                          cudaStream_t st) {
  const int64_t bx = (R + 255) / 256;
  // about eight blocks per SM, of at least 32 rows
  const int64_t ny = std::max<int64_t>(1, std::min<int64_t>({(8 * 152 + bx - 1) / bx, P / 32, (int64_t)65535}));
  const int64_t step = (P + ny - 1) / ny;
  const dim3 g((unsigned)bx, (unsigned)((P + step - 1) / step));
  if (dt == C128)
    colsum_gemv_kernel<double><<<g, 256, 0, st>>>(P, R, step, (const double2 *)B, (const double2 *)w, sw, (double2 *)y,
                                                  alpha.re, alpha.im);
  else
    colsum_gemv_kernel<float><<<g, 256, 0, st>>>(P, R, step, (const float2 *)B, (const float2 *)w, sw, (float2 *)y,
                                                 (float)alpha.re, (float)alpha.im);
  count_launch();
  CCLR_CUDA(cudaGetLastError());
}

// tau of the CCSD energy over the packed doubles (complex128):
// tau[(i<j),(a<b)] = t2[(i<j),(a<b)] + t1[i,a] t1[j,b] - t1[i,b] t1[j,a].
__global__ void tau_packed_kernel(int o, int v, const double2 *t1, const double2 *t2p, double2 *tau) {
  const int64_t Pv = (int64_t)v * (v - 1) / 2, n = (int64_t)o * (o - 1) / 2 * Pv;
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < n; e += (int64_t)gridDim.x * blockDim.x) {
    int i, j, a, b;
    pair_of(e / Pv, o, i, j);
    pair_of(e % Pv, v, a, b);
    const double2 ia = t1[(int64_t)i * v + a], jb = t1[(int64_t)j * v + b];
    const double2 ib = t1[(int64_t)i * v + b], ja = t1[(int64_t)j * v + a];
    double2 z = t2p[e];
    z.x += (ia.x * jb.x - ia.y * jb.y) - (ib.x * ja.x - ib.y * ja.y);
    z.y += (ia.x * jb.y + ia.y * jb.x) - (ib.x * ja.y + ib.y * ja.x);
    tau[e] = z;
  }
}

void tau_packed(int o, int v, const void *t1, const void *t2p, void *tau, cudaStream_t st) {
  const int64_t n = (int64_t)o * (o - 1) / 2 * ((int64_t)v * (v - 1) / 2);
  if (n == 0) return;
  tau_packed_kernel<<<grid_for(n), 256, 0, st>>>(o, v, (const double2 *)t1, (const double2 *)t2p, (double2 *)tau);
  count_launch();
  CCLR_CUDA(cudaGetLastError());
}

__global__ void conj_kernel(int64_t n, const double2 *x, double2 *y) {
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < n; e += (int64_t)gridDim.x * blockDim.x) {
    const double2 z = x[e];
    y[e] = make_double2(z.x, -z.y);
  }
}

void vec_conj(int64_t n, const void *x, void *y, cudaStream_t st) {
  if (n == 0) return;
  conj_kernel<<<grid_for(n), 256, 0, st>>>(n, (const double2 *)x, (double2 *)y);
  count_launch();
  CCLR_CUDA(cudaGetLastError());
}

void build_diag(int o, int v, const void *Foo, const void *Fvv, double *D1, double *D2p,
                cudaStream_t st) {
  const int64_t n = (int64_t)o * v + (int64_t)o * (o - 1) / 2 * ((int64_t)v * (v - 1) / 2);
  diag_kernel<<<grid_for(n), 256, 0, st>>>(o, v, (const double2 *)Foo, (const double2 *)Fvv, D1, D2p);
  count_launch();
  CCLR_CUDA(cudaGetLastError());
}

// F (+)= alpha * unpack(P), one thread per full entry (writes coalesced; the packed row of one
// (i,j) pair is read with a stride that depends on the (a,b) order, from L2).
template <typename TP, typename TF>
__global__ void __launch_bounds__(256) unpack_doubles_kernel(int o, int v, const typename cpx<TP>::t *__restrict__ P,
                                                             typename cpx<TF>::t *__restrict__ F, double ar, double ai,
                                                             int acc, int unit) {
  // block (32, 8): b = blockIdx.x * 32 + x, a = blockIdx.y * 8 + y, (i, j) = blockIdx.z: no division
  const int b = blockIdx.x * 32 + threadIdx.x, a = blockIdx.y * 8 + threadIdx.y;
  if (a >= v || b >= v) return;
  const int i = blockIdx.z / o, j = blockIdx.z % o;
  const int64_t Pv = (int64_t)v * (v - 1) / 2;
  const int64_t e = ((int64_t)blockIdx.z * v + a) * v + b;
  TF zr = 0, zi = 0;
  if (i != j && a != b) {
    const int p = min(i, j), q = max(i, j), r = min(a, b), s2 = max(a, b);
    const typename cpx<TP>::t z = P[pair_id(p, q, o) * Pv + pair_id(r, s2, v)];
    const bool pos = (i < j) == (a < b);
    zr = pos ? (TF)z.x : -(TF)z.x;
    zi = pos ? (TF)z.y : -(TF)z.y;
  }
  // alpha = 1 (unit) takes no multiply: this GPU's FP64 rate would bound the complex128 case
  TF wr = zr, wi = zi;
  if (!unit) {
    wr = (TF)(ar * (double)zr - ai * (double)zi);
    wi = (TF)(ar * (double)zi + ai * (double)zr);
  }
  if (acc) {
    wr += F[e].x;
    wi += F[e].y;
  }
  typename cpx<TF>::t w;
  w.x = wr;
  w.y = wi;
  F[e] = w;
}

// P = F[i<j, a<b], one thread per packed entry (writes coalesced, reads along b).
template <typename TF, typename TP>
__global__ void pack_doubles_kernel(int o, int v, const typename cpx<TF>::t *F, typename cpx<TP>::t *P) {
  const int64_t Pv = (int64_t)v * (v - 1) / 2, n = (int64_t)o * (o - 1) / 2 * Pv;
  for (int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; k < n; k += (int64_t)gridDim.x * blockDim.x) {
    int i, j, a, b;
    pair_of(k / Pv, o, i, j);
    pair_of(k % Pv, v, a, b);
    const typename cpx<TF>::t f = F[(((int64_t)i * o + j) * v + a) * v + b];
    typename cpx<TP>::t w;
    w.x = (TP)f.x;
    w.y = (TP)f.y;
    P[k] = w;
  }
}

void unpack_doubles(int dt_p, int dt_f, int o, int v, const void *P, void *F, zc alpha, bool acc, cudaStream_t st) {
  if ((int64_t)o * o * v * v == 0) return;
  CCLR_REQUIRE((int64_t)o * o < 65536, "unpack_doubles: too many occupied pairs for the grid");
  const dim3 g((unsigned)((v + 31) / 32), (unsigned)((v + 7) / 8), (unsigned)(o * o)), b(32, 8);
  const int a = acc ? 1 : 0, u = (alpha.re == 1.0 && alpha.im == 0.0) ? 1 : 0;
  if (dt_p == C128 && dt_f == C128)
    unpack_doubles_kernel<double, double><<<g, b, 0, st>>>(o, v, (const double2 *)P, (double2 *)F, alpha.re, alpha.im, a, u);
  else if (dt_p == C128 && dt_f == C64)
    unpack_doubles_kernel<double, float><<<g, b, 0, st>>>(o, v, (const double2 *)P, (float2 *)F, alpha.re, alpha.im, a, u);
  else if (dt_p == C64 && dt_f == C128)
    unpack_doubles_kernel<float, double><<<g, b, 0, st>>>(o, v, (const float2 *)P, (double2 *)F, alpha.re, alpha.im, a, u);
  else
    unpack_doubles_kernel<float, float><<<g, b, 0, st>>>(o, v, (const float2 *)P, (float2 *)F, alpha.re, alpha.im, a, u);
  count_launch();
  CCLR_CUDA(cudaGetLastError());
}

// one block per i, threads over a; each thread sums over (j, b) with the packed entry's sign
__global__ void packed_dot_singles_kernel(int o, int v, const double2 *W, const double2 *x1, double2 *out1,
                                          double ar, double ai) {
  const int i = blockIdx.x;
  const int64_t Pv = (int64_t)v * (v - 1) / 2;
  for (int a = threadIdx.x; a < v; a += blockDim.x) {
    double sr = 0.0, si = 0.0;
    for (int j = 0; j < o; ++j) {
      if (j == i) continue;
      const int64_t row = pair_id(min(i, j), max(i, j), o) * Pv;
      const double sij = i < j ? 1.0 : -1.0;
      for (int b = 0; b < v; ++b) {
        if (b == a) continue;
        const double sg = (a < b) ? sij : -sij;
        const double2 w = W[row + pair_id(min(a, b), max(a, b), v)];
        const double2 x = x1[(int64_t)j * v + b];
        sr += sg * (w.x * x.x - w.y * x.y);
        si += sg * (w.x * x.y + w.y * x.x);
      }
    }
    double2 *p = out1 + (int64_t)i * v + a;
    p->x += ar * sr - ai * si;
    p->y += ar * si + ai * sr;
  }
}

void packed_doubles_dot_singles(int o, int v, const void *Wp, const void *x1, void *out1, zc alpha, cudaStream_t st) {
  if (o < 2 || v < 2) return;
  packed_dot_singles_kernel<<<o, 128, 0, st>>>(o, v, (const double2 *)Wp, (const double2 *)x1, (double2 *)out1,
                                               alpha.re, alpha.im);
  count_launch();
  CCLR_CUDA(cudaGetLastError());
}

void pack_doubles(int dt_f, int dt_p, int o, int v, const void *F, void *P, cudaStream_t st) {
  const int64_t n = (int64_t)o * (o - 1) / 2 * ((int64_t)v * (v - 1) / 2);
  if (n == 0) return;
  const unsigned g = grid_for(n);
  if (dt_f == C128 && dt_p == C128)
    pack_doubles_kernel<double, double><<<g, 256, 0, st>>>(o, v, (const double2 *)F, (double2 *)P);
  else if (dt_f == C64 && dt_p == C128)
    pack_doubles_kernel<float, double><<<g, 256, 0, st>>>(o, v, (const float2 *)F, (double2 *)P);
  else if (dt_f == C128 && dt_p == C64)
    pack_doubles_kernel<double, float><<<g, 256, 0, st>>>(o, v, (const double2 *)F, (float2 *)P);
  else
    pack_doubles_kernel<float, float><<<g, 256, 0, st>>>(o, v, (const float2 *)F, (float2 *)P);
  count_launch();
  CCLR_CUDA(cudaGetLastError());
}

// t2[i,j,a,b] = w[i,j,a,b] / (e_i + e_j - e_a - e_b)
__global__ void denom_kernel(int o, int v, const double *eps, double2 *t2) {
  int64_t n = (int64_t)o * o * v * v;
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < n;
       e += (int64_t)gridDim.x * blockDim.x) {
    int64_t r = e;
    int b = (int)(r % v); r /= v;
    int a = (int)(r % v); r /= v;
    int j = (int)(r % o); r /= o;
    int i = (int)r;
    double d = eps[i] + eps[j] - eps[o + a] - eps[o + b];
    double2 x = t2[e];
    t2[e] = make_double2(x.x / d, x.y / d);
  }
}

void apply_denominator(int o, int v, const double *eps, void *t2, cudaStream_t st) {
  int64_t n = (int64_t)o * o * v * v;
  denom_kernel<<<grid_for(n), 256, 0, st>>>(o, v, eps, (double2 *)t2);
  count_launch();
    CCLR_CUDA(cudaGetLastError());
}

// out[p,q] = value on the diagonal (complex128 square matrix), used for diag(eps).
__global__ void set_diag_kernel(int n, const double *d, double2 *out) {
  int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) out[(int64_t)i * n + i] = make_double2(d[i], 0.0);
}

void set_diag(int n, const double *d, void *out, cudaStream_t st) {
  set_diag_kernel<<<(n + 255) / 256, 256, 0, st>>>(n, d, (double2 *)out);
  count_launch();
    CCLR_CUDA(cudaGetLastError());
}

}  // namespace cclr
