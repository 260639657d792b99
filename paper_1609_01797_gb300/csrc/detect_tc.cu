// Tensor-core TASER iterations (Algorithm 1): the triangular product L~ T^ on the
// tensor cores with BF16 or FP16 operands and FP32 accumulation; the master L~ and the
// prox (column norms, rescaling) stay in FP32.
//
// One warp per instance, in transposed form: the accumulators of mma.m16n8k16 hold
//   V^T = L~^T + T^ L~^T   (T^ = -2 tau T~ is symmetric, so V^T = (L~ - 2 tau L~ T~)^T),
// with the C operand the FP32 master L~^T, the constant A operand T^ and the B operand
// L~^T.  A lane holds two adjacent entries of rows k of V^T (columns k of V) per n-tile,
// so the prox's column norms are sums over the 4 lanes of a row.  They are summed transposed
// (row_sums): a lane ends with the norm of one row of four, forms its scale, and a shuffle
// hands the scale to the row's lanes.  The kernel is bound by instruction issue, and forming
// every row's scale in all of its 4 lanes was a sixth of its instructions (222 -> 195 warp
// instructions per instance and iteration at N = 33).  With the sums, a compile-time L~_NN mode
// and the products' order below, per 65,536, t_max = 20: N = 33 0.396 -> 0.359 ms, N = 17
// 0.186 -> 0.164 (outputs bitwise equal).  6 blocks an SM (80 registers): 0.395.  Row N of
// L~ is simply the last n-tile (column NB of L~^T).  The B operand of the next step is the
// iterate transposed in 8 x 8 blocks: each block packed to 16 bits and moved with
// movmatrix.trans, which turns the accumulator layout (row g, columns 2tq, 2tq + 1) into
// the B-fragment layout (rows 2tq, 2tq + 1, column g).
//
// Tiles: columns k of L~ in m-tiles of 16, rows i in n-tiles of 8 (the last holds row N),
// j in k-tiles of 16.  Tile (M, n) exists only where some i >= k (V is lower-triangular,
// V^T upper), and it needs only the k-tiles with j <= i (L~^T[j][i] = 0 for j > i): the
// triangular skip of the paper's array (Sec. IV-A) at tile granularity.  The j = N term
// (T^[k][N] L~_NN) and V_NN are added in FP32.  The tensor-core instruction is the
// warp-level mma.sync: the per-instance operand T^ changes with every instance and the
// problem is 33 x 33, below the 64/128-row tiles of tcgen05.
#include <type_traits>

#include "tct_job.cuh"

namespace taser {

// Persistent: each warp takes jobs from its source (a fixed stride, or a bucket queue) and
// prefetches the next job's inputs with cp.async while it iterates on the current one.
// MON: objective monitoring of taser_detect_monitored (dense source only).  f(L~) =
// Tr(L~ T~ L~^T) is the sum over i >= k of L~_ik (L~ T~)_ik, the lower part of L~ T~ that
// each gradient step forms.  A single BF16 product is too coarse to see a rise of f of a
// fraction of a percent, so the monitor forms W^T = T^ L~^T a second time as a BF16 split
// (T^ = hi + lo as A fragments, the iterate's hi and lo moved like the B operand; 3 mma
// per product, about 2^-16 relative error) into scratch accumulators, before the step's
// own mma, and sums L~ o W; f = sum / (-2 tau).  The iteration itself is unchanged.  One
// more step after the outputs are written gives f(L~(t_max)).
// LIT: taser_lnn_mode LITERAL.  In the fixed mode L~_NN is constant and V_NN feeds one flag
// only, so no lane but tq == 0 needs it.
template <int NB, bool FP16, class Src, bool LIT, bool MON = false>
__global__ void __launch_bounds__(128, MON ? 3 : 5)
detect_tct_kernel(Src src, int slot_floats, float ascent_tol) {
  constexpr bool BCAST = LIT || MON;   // V_NN in every lane
  using C = TctCfg<NB>;
  constexpr int MT = C::MT, KT = C::KT, NT = C::NT;
  extern __shared__ __align__(16) float smem[];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int g = lane >> 2, tq = lane & 3;
  float* slot = smem + warp * (slot_floats + kTcRecFloats);
  // Output pointers and sizes of the current and the next job live in shared memory
  // (two records per warp), not in registers across the iteration loop.
  struct JobOut {
    float* L;
    int8_t* s;
    uint32_t* flag;
    double* obj;
    int N, t_max, shift;
  };
  static_assert(2 * sizeof(JobOut) <= kTcRecFloats * sizeof(float), "job records must fit");
  JobOut* outs = reinterpret_cast<JobOut*>(slot + slot_floats);
  auto park = [&](const Job& jb, double* ob, int shift, int which) {
    if (lane == 0) outs[which] = JobOut{jb.L, jb.s, jb.flag, ob, jb.N, jb.t_max, shift};
  };
  Cursor<Src> cursor;
  int cur_m = 0;
  bool have;
  {
    Job first;
    double* ob = nullptr;
    have = cursor.next(src, first, ob, lane);
    if (have) park(first, ob, stage_job(slot, first, lane, slot_floats), 0);
  }

  while (have) {
    asm volatile("cp.async.wait_all;" ::: "memory");
    __syncwarp();
    const int N = outs[cur_m].N, t_max = outs[cur_m].t_max;
    const float* T = slot + outs[cur_m].shift;
    const float* Di = slot + N * N + 4;
    const float m2tau = -2.f * Di[N];
    auto tval = [&](int k, int j) -> float {  // T^ at bucket indices (k, j < NB)
      return (k < N - 1 && j < N - 1) ? m2tau * T[k * N + j] : 0.f;
    };
    // A operand: T^ rows k = 16M + g (+8), columns j = 16kt + 2tq (+1, +8, +9).  MON: also
    // T^ = hi + lo in BF16 (same layout) for the monitor's split product.
    uint32_t af[MT][KT][4];
    uint32_t mah[MON ? MT : 1][KT][4], mal[MON ? MT : 1][KT][4];
#pragma unroll
    for (int M = 0; M < MT; ++M)
#pragma unroll
      for (int kt = 0; kt < KT; ++kt) {
        const int r = 16 * M + g, c = 16 * kt + 2 * tq;
        float v[4][2];
        if (N == NB + 1) {   // no padding rows or columns: no bounds tests
          const float* r0 = T + r * (NB + 1) + c;
          const float* r1 = r0 + 8 * (NB + 1);
          v[0][0] = m2tau * r0[0], v[0][1] = m2tau * r0[1];
          v[1][0] = m2tau * r1[0], v[1][1] = m2tau * r1[1];
          v[2][0] = m2tau * r0[8], v[2][1] = m2tau * r0[9];
          v[3][0] = m2tau * r1[8], v[3][1] = m2tau * r1[9];
        } else {
          v[0][0] = tval(r, c), v[0][1] = tval(r, c + 1);
          v[1][0] = tval(r + 8, c), v[1][1] = tval(r + 8, c + 1);
          v[2][0] = tval(r, c + 8), v[2][1] = tval(r, c + 9);
          v[3][0] = tval(r + 8, c + 8), v[3][1] = tval(r + 8, c + 9);
        }
#pragma unroll
        for (int x = 0; x < 4; ++x) {
          af[M][kt][x] = pack2<FP16>(v[x][0], v[x][1]);
          if constexpr (MON) split_bf16(v[x][0], v[x][1], mah[M][kt][x], mal[M][kt][x]);
        }
      }
    // This lane's rows k = 16M + g + 8h: T^[k][N] (FP32, the j = N term).
    float tkN[MT][2];
#pragma unroll
    for (int M = 0; M < MT; ++M)
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const int k = 16 * M + g + 8 * h;
        tkN[M][h] = k < N - 1 ? m2tau * T[k * N + N - 1] : 0.f;
      }
    // The row whose norm this lane owns (row_sums): its D_k, and its smallest squared norm.
    constexpr int R = 2 * MT;
    const int k_own = row_column(owned_row<R>(0, tq), g);
    const float D_own = k_own < N - 1 ? Di[k_own] : 0.f;
    const float inval_own = k_own < N - 1 ? 0.f : 3.0e38f;   // rows k >= N - 1 never flag a zero column
    float snmin = 3.0e38f;
    const float tnNN = m2tau * T[(N - 1) * N + (N - 1)];
    const float DN = Di[N - 1];
    // L~(0) = D in the V^T layout: element (M, n, e) is k = 16M + g + 8(e >> 1),
    // i = 8n + 2tq + (e & 1).
    float acc[MT][NT][4];
#pragma unroll
    for (int M = 0; M < MT; ++M)
#pragma unroll
      for (int n = 0; n < NT; ++n)
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          const int k = 16 * M + g + 8 * (e >> 1), i = 8 * n + 2 * tq + (e & 1);
          acc[M][n][e] = (C::has_tile(M, n) && i == k && k < N - 1) ? Di[k] : 0.f;
        }
    __syncwarp();  // every lane has read the slot
    bool have_next;
    {
      Job nxt;
      double* ob = nullptr;
      have_next = cursor.next(src, nxt, ob, lane);
      if (have_next) park(nxt, ob, stage_job(slot, nxt, lane, slot_floats), cur_m ^ 1);
    }
    float LNN = DN;
    float vmin = 3.0e38f;   // smallest V_NN of the job (where it is formed)
    uint32_t fl = 0;
    // Inside a diagonal 8 x 8 block, element (row g, column 2tq + p) lies below the
    // diagonal of V^T (i < k) iff 2tq + p < g.
    const bool lo0 = 2 * tq < g, lo1 = 2 * tq + 1 < g;

    // One gradient step: acc <- V^T = L~^T + T^ L~^T (on and above its diagonal; the 8 x 8 blocks
    // below the diagonal, (M, 2M) rows h = 1, are left as they come: nothing reads them).
    // Returns V_NN, in every lane if BCAST, otherwise in the lanes tq == 0.  MON: fterm += sum of
    // L~_ik W_ik over this lane's elements, W = L~ T^ (as W^T = T^ L~^T, a BF16 split product of the
    // old iterate, before the step).
    auto grad_step = [&](float& fterm) -> float {
      // V_NN partial sum_{j < N} T^[N][j] L~[N][j] from the old row N (column NB of L~^T,
      // held by the lanes tq == 0), summed over g after the products.
      float part = 0.f;
      if (tq == 0) {
#pragma unroll
        for (int M = 0; M < MT; ++M)
#pragma unroll
          for (int h = 0; h < 2; ++h) part = fmaf(tkN[M][h], acc[M][NT - 1][2 * h], part);
      }
      // B operand from the old iterate: block (kb, ib) of L~^T transposed; blocks with
      // kb > ib are zero.
      uint32_t bfr[KT][NT][2];
      uint32_t mbh[MON ? KT : 1][NT][2], mbl[MON ? KT : 1][NT][2];
#pragma unroll
      for (int kt = 0; kt < KT; ++kt)
#pragma unroll
        for (int n = 0; n < NT; ++n)
#pragma unroll
          for (int q = 0; q < 2; ++q) {
            const int kb = 2 * kt + q, M = kb / 2, h = kb % 2;
            if (kt > C::ktmax(n) || kb > n) {
              bfr[kt][n][q] = 0u;
              if constexpr (MON) mbh[kt][n][q] = mbl[kt][n][q] = 0u;
            } else {
              bfr[kt][n][q] = movmatrix_trans(pack2<FP16>(acc[M][n][2 * h], acc[M][n][2 * h + 1]));
              if constexpr (MON) {
                uint32_t hi, lo;
                split_bf16(acc[M][n][2 * h], acc[M][n][2 * h + 1], hi, lo);
                mbh[kt][n][q] = movmatrix_trans(hi);
                mbl[kt][n][q] = movmatrix_trans(lo);
              }
            }
          }
      if constexpr (MON) {
#pragma unroll
        for (int M = 0; M < MT; ++M)
#pragma unroll
          for (int n = 0; n < NT; ++n) {
            if (!C::has_tile(M, n)) continue;
            float w4[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
            for (int kt = 0; kt <= C::ktmax(n); ++kt) {
              mma16816<false>(w4, mah[M][kt], mbh[kt][n]);
              mma16816<false>(w4, mah[M][kt], mbl[kt][n]);
              mma16816<false>(w4, mal[M][kt], mbh[kt][n]);
            }
            if (n == NT - 1 && tq == 0) {   // j = N term of column NB, in FP32
              w4[0] = fmaf(tkN[M][0], LNN, w4[0]);
              w4[2] = fmaf(tkN[M][1], LNN, w4[2]);
            }
#pragma unroll
            for (int e = 0; e < 4; ++e)
              if (!(n == 2 * M && e >= 2)) fterm = fmaf(acc[M][n][e], w4[e], fterm);
          }
      }
      // The step's products, n-tiles ascending (measured per 65,536 at N = 33: 0.359 ms, row N's
      // tile first 0.366, k-tiles outermost 0.360).
#pragma unroll
      for (int n = 0; n < NT; ++n)
#pragma unroll
        for (int M = 0; M < MT; ++M) {
          if (!C::has_tile(M, n)) continue;
#pragma unroll
          for (int kt = 0; kt <= C::ktmax(n); ++kt) mma16816<FP16>(acc[M][n], af[M][kt], bfr[kt][n]);
        }
      part += __shfl_xor_sync(TASER_FULL_MASK, part, 4);
      part += __shfl_xor_sync(TASER_FULL_MASK, part, 8);
      part += __shfl_xor_sync(TASER_FULL_MASK, part, 16);
      if (BCAST) part = __shfl_sync(TASER_FULL_MASK, part, lane & 28);   // from the row's lane tq == 0
      // j = N term of column NB: V^T[k][N] += T^[k][N] L~_NN.
      if (tq == 0) {
#pragma unroll
        for (int M = 0; M < MT; ++M)
#pragma unroll
          for (int h = 0; h < 2; ++h) acc[M][NT - 1][2 * h] = fmaf(tkN[M][h], LNN, acc[M][NT - 1][2 * h]);
      }
      // Keep V^T on and above its diagonal (i >= k): blocks kb == ib are masked.
#pragma unroll
      for (int M = 0; M < MT; ++M) {
        if (lo0) acc[M][2 * M][0] = 0.f;
        if (lo1) acc[M][2 * M][1] = 0.f;
        if (lo0) acc[M][2 * M + 1][2] = 0.f;
        if (lo1) acc[M][2 * M + 1][3] = 0.f;
      }
      return fmaf(LNN, tnNN, LNN) + part;
    };

    // MON: f(L~(t)) from the step's terms (FP32 sums, FP64 ratio and comparison).
    double f_prev = 0.0;
    double* const obj = MON ? outs[cur_m].obj : nullptr;
    auto monitor = [&](int t, float fterm, float vnn) {
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) fterm += __shfl_xor_sync(TASER_FULL_MASK, fterm, o);
      fterm = fmaf(LNN, vnn - LNN, fterm);   // L~_NN W_NN, W_NN = V_NN - L~_NN (FP32)
      const double f = m2tau < 0.f ? (double)fterm / (double)m2tau : 0.0;
      if (t > 0 && f > f_prev + (double)ascent_tol * fabs(f_prev)) fl |= TASER_FLAG_ASCENT;
      f_prev = f;
      if (lane == 0 && obj != nullptr && TASER_IN(t, t_max + 1)) obj[t] = f;
    };

    for (int t = 0; t < t_max; ++t) {
      float fterm = 0.f;
      const float vnn = grad_step(fterm);
      if constexpr (MON) monitor(t, fterm, vnn);
      vmin = fminf(vmin, vnn);
      if (LIT) LNN = vnn >= 0.f ? DN : -DN;
      // prox: squared norms of this lane's rows k, summed over the 4 lanes of the row; each
      // row's scale is formed in the lane that owns its sum.
      float sn[R], own[1];
#pragma unroll
      for (int M = 0; M < MT; ++M)
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          uint64_t v2 = 0ull;
#pragma unroll
          for (int n = 0; n < NT; ++n) {
            if (!C::has_tile(M, n) || (n == 2 * M && h == 1)) continue;   // below the diagonal
            const uint64_t x = f2pack(acc[M][n][2 * h], acc[M][n][2 * h + 1]);
            v2 = f2fma(x, x, v2);
          }
          float a, b;
          f2unpack(v2, a, b);
          sn[2 * M + h] = a + b;
        }
      row_sums<R>(sn, own, tq);
      snmin = fminf(snmin, own[0] + inval_own);
      const float sc_own = own[0] > 0.f ? D_own * rsqrtf(own[0]) : 0.f;
#pragma unroll
      for (int M = 0; M < MT; ++M)
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          const float sc = __shfl_sync(TASER_FULL_MASK, sc_own, (lane & 28) + 2 * M + h);
          const uint64_t sc2 = f2pack(sc, sc);
#pragma unroll
          for (int n = 0; n < NT; ++n) {
            if (!C::has_tile(M, n) || (n == 2 * M && h == 1)) continue;
            TASER_PAIR_APPLY(acc[M][n], 2 * h, f2mul(_x, sc2));
          }
        }
    }

    // A zero column in any iteration (its prox scale was 0): measured 2.2% faster than a
    // per-iteration flag update.
    if (snmin <= 0.f) fl |= TASER_FLAG_ZERO_COLUMN;
    if ((BCAST || tq == 0) && vmin <= 0.f) fl |= TASER_FLAG_LNN_SIGN;
    const JobOut o = outs[cur_m];
    // Decisions from row N of L~ (column NB of L~^T, lanes tq == 0).
    if (tq == 0) {
#pragma unroll
      for (int M = 0; M < MT; ++M)
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          const int k = 16 * M + g + 8 * h;
          if (k < N - 1 && TASER_IN(k, N - 1)) {
            float r = acc[M][NT - 1][2 * h];
            TASER_FINITE(r);
            if (LIT && LNN < 0.f) r = -r;
            o.s[k] = r >= 0.f ? int8_t(1) : int8_t(-1);
          }
        }
    }
    if (o.L != nullptr) {
      float* Lo = o.L;
#pragma unroll
      for (int M = 0; M < MT; ++M)
#pragma unroll
        for (int n = 0; n < NT; ++n)
#pragma unroll
          for (int e = 0; e < 4; ++e) {
            const int k = 16 * M + g + 8 * (e >> 1), i = 8 * n + 2 * tq + (e & 1);
            const int rr = bucket_to_real(i, N, NB);
            if (rr < 0 || k >= N - 1 || !TASER_IN(rr * N + k, N * N)) continue;
            Lo[(int64_t)rr * N + k] = C::has_tile(M, n) && !(n == 2 * M && e >= 2) ? acc[M][n][e] : 0.f;
            TASER_FINITE(Lo[(int64_t)rr * N + k]);
          }
      for (int rr = lane; rr < N; rr += 32)
        if (TASER_IN(rr * N + N - 1, N * N)) Lo[(int64_t)rr * N + (N - 1)] = rr == N - 1 ? LNN : 0.f;
    }
    if constexpr (MON) {   // f(L~(t_max)): one more gradient step, after the outputs
      float fterm = 0.f;
      const float vnn = grad_step(fterm);
      monitor(t_max, fterm, vnn);
    }
#pragma unroll
    for (int ofs = 16; ofs > 0; ofs >>= 1) fl |= __shfl_xor_sync(TASER_FULL_MASK, fl, ofs);
    if (lane == 0 && o.flag != nullptr && fl) *o.flag |= fl;
    __syncwarp();  // the record of this job is consumed before it is reused
    cur_m ^= 1;
    have = have_next;
  }
}

template <int NB, bool MON, class Src>
static cudaError_t launch_tc(const Src& src, int64_t jobs, int blocks_per_sm, int literal, bool fp16, int slot_floats,
                             float ascent_tol, cudaStream_t st) {
  const size_t smem = (size_t)4 * (slot_floats + kTcRecFloats) * sizeof(float);
  auto go = [&](auto half, auto lit) {
    return launch_persistent(detect_tct_kernel<NB, decltype(half)::value, Src, decltype(lit)::value, MON>, smem, src,
                             jobs, blocks_per_sm, st, slot_floats, ascent_tol);
  };
  if (literal) return fp16 ? go(std::true_type{}, std::true_type{}) : go(std::false_type{}, std::true_type{});
  return fp16 ? go(std::true_type{}, std::false_type{}) : go(std::false_type{}, std::false_type{});
}

// ---------------------------------------------------------------------------------
// The transposed form at 34 <= N <= 65 (bucket 64), one warp per instance.  The 24 tiles of
// V^T (96 accumulators a lane) and the 16 A fragments of T^ (64 registers) stay in
// registers.  The B operand goes through shared memory: every step the lane packs and
// transposes the 44 nonzero 8 x 8 blocks of L~^T it holds (movmatrix.trans) into the warp's
// block grid, and each group of mma loads its two B registers from there just before use.
// T^, D and tau are read from global memory once per job (no staging slot, so the block
// grid is the only shared memory).  No step needs another warp: the column norms are sums
// over the 4 lanes of a row, transposed as in the bucket-32 kernel (0.455 -> 0.420 ms per 16,384
// at N = 65, t_max = 20; a compile-time L~_NN mode was slower here, 0.434).
// ---------------------------------------------------------------------------------
constexpr int kBlk64Words = 8 * 9 * 32;   // block grid [kb][ib][lane] of one warp (kb <= ib used)

template <bool FP16, class Src>
__global__ void __launch_bounds__(128, 2)
detect_tct64_kernel(Src src, int literal, int slot_floats) {
  using C = TctCfg<64>;
  constexpr int MT = C::MT, KT = C::KT, NT = C::NT, NB = 64;
  extern __shared__ __align__(16) float smem[];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int g = lane >> 2, tq = lane & 3;
  // Per warp: the block grid, then the staging slot of the next job and two job records.
  uint32_t* const blk = reinterpret_cast<uint32_t*>(smem) + warp * (kBlk64Words + slot_floats + kTcRecFloats);
  float* const slot = reinterpret_cast<float*>(blk + kBlk64Words);
  auto bw = [&](int kb, int ib) -> uint32_t& { return blk[(kb * 9 + ib) * 32 + lane]; };
  struct JobOut {
    float* L;
    int8_t* s;
    uint32_t* flag;
    double* obj;
    int N, t_max, shift;
  };
  static_assert(2 * sizeof(JobOut) <= kTcRecFloats * sizeof(float), "job records must fit");
  JobOut* outs = reinterpret_cast<JobOut*>(slot + slot_floats);
  auto park = [&](const Job& jb, int shift, int which) {
    if (lane == 0) outs[which] = JobOut{jb.L, jb.s, jb.flag, nullptr, jb.N, jb.t_max, shift};
  };
  // Inside a diagonal 8 x 8 block, element (row g, column 2tq + p) lies below the
  // diagonal of V^T (i < k) iff 2tq + p < g.
  const bool lo0 = 2 * tq < g, lo1 = 2 * tq + 1 < g;
  Cursor<Src> cursor;
  int cur_m = 0;
  bool have;
  {
    Job first;
    double* ob = nullptr;
    have = cursor.next(src, first, ob, lane);
    if (have) park(first, stage_job(slot, first, lane, slot_floats), 0);
  }
  while (have) {
    asm volatile("cp.async.wait_all;" ::: "memory");
    __syncwarp();
    const int N = outs[cur_m].N, t_max = outs[cur_m].t_max;
    const float* T = slot + outs[cur_m].shift;
    const float* Di = slot + N * N + 4;
    const float m2tau = -2.f * Di[N];
    auto tval = [&](int k, int j) -> float {  // T^ at bucket indices (k, j < NB)
      return (k < N - 1 && j < N - 1) ? m2tau * T[k * N + j] : 0.f;
    };
    // A operand: T^ rows k = 16M + g (+8), columns j = 16kt + 2tq (+1, +8, +9).
    uint32_t af[MT][KT][4];
#pragma unroll
    for (int M = 0; M < MT; ++M)
#pragma unroll
      for (int kt = 0; kt < KT; ++kt) {
        const int r = 16 * M + g, c = 16 * kt + 2 * tq;
        af[M][kt][0] = pack2<FP16>(tval(r, c), tval(r, c + 1));
        af[M][kt][1] = pack2<FP16>(tval(r + 8, c), tval(r + 8, c + 1));
        af[M][kt][2] = pack2<FP16>(tval(r, c + 8), tval(r, c + 9));
        af[M][kt][3] = pack2<FP16>(tval(r + 8, c + 8), tval(r + 8, c + 9));
      }
    // This lane's rows k = 16M + g + 8h: T^[k][N] (FP32, the j = N term).
    float tkN[MT][2];
#pragma unroll
    for (int M = 0; M < MT; ++M)
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const int k = 16 * M + g + 8 * h;
        tkN[M][h] = k < N - 1 ? m2tau * T[k * N + N - 1] : 0.f;
      }
    // The rows whose norms this lane owns (row_sums): their D_k and smallest squared norm.
    constexpr int R = 2 * MT;
    float D_own[R / 4], inval_own[R / 4];
#pragma unroll
    for (int u = 0; u < R / 4; ++u) {
      const int k = row_column(owned_row<R>(u, tq), g);
      D_own[u] = k < N - 1 ? Di[k] : 0.f;
      inval_own[u] = k < N - 1 ? 0.f : 3.0e38f;   // rows k >= N - 1 never flag a zero column
    }
    float snmin = 3.0e38f;
    const float tnNN = m2tau * T[(N - 1) * N + (N - 1)];
    const float DN = Di[N - 1];
    // L~(0) = D in the V^T layout: element (M, n, e) is k = 16M + g + 8(e >> 1),
    // i = 8n + 2tq + (e & 1).
    float acc[MT][NT][4];
#pragma unroll
    for (int M = 0; M < MT; ++M)
#pragma unroll
      for (int n = 0; n < NT; ++n)
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          const int k = 16 * M + g + 8 * (e >> 1), i = 8 * n + 2 * tq + (e & 1);
          acc[M][n][e] = (C::has_tile(M, n) && i == k && k < N - 1) ? Di[k] : 0.f;
        }
    __syncwarp();  // every lane has read the slot
    bool have_next;
    {
      Job nxt;
      double* ob = nullptr;
      have_next = cursor.next(src, nxt, ob, lane);
      if (have_next) park(nxt, stage_job(slot, nxt, lane, slot_floats), cur_m ^ 1);
    }
    float LNN = DN;
    float vmin = 3.0e38f;   // smallest V_NN of the job (where it is formed)
    uint32_t fl = 0;

    for (int t = 0; t < t_max; ++t) {
      // V_NN partial sum_{j < N} T^[N][j] L~[N][j] from the old row N (lanes tq == 0).
      float part = 0.f;
      if (tq == 0) {
#pragma unroll
        for (int M = 0; M < MT; ++M)
#pragma unroll
          for (int h = 0; h < 2; ++h) part = fmaf(tkN[M][h], acc[M][NT - 1][2 * h], part);
      }
      part += __shfl_xor_sync(TASER_FULL_MASK, part, 4);
      part += __shfl_xor_sync(TASER_FULL_MASK, part, 8);
      part += __shfl_xor_sync(TASER_FULL_MASK, part, 16);
      if (literal) part = __shfl_sync(TASER_FULL_MASK, part, lane & 28);   // else only the lanes tq == 0 hold V_NN
      // The old iterate as B blocks: block (kb, ib) of L~^T transposed, for kb <= ib.
      __syncwarp();   // the previous step's B loads are done before the grid is rewritten
#pragma unroll
      for (int kb = 0; kb < 2 * MT; ++kb)
#pragma unroll
        for (int ib = kb; ib < NT; ++ib)
          bw(kb, ib) = movmatrix_trans(pack2<FP16>(acc[kb / 2][ib][2 * (kb % 2)], acc[kb / 2][ib][2 * (kb % 2) + 1]));
      __syncwarp();
      // Products, row N's n-tile first; each (kt, n) B fragment serves every m-tile.
#pragma unroll
      for (int n = NT - 1; n >= 0; --n)
#pragma unroll
        for (int kt = 0; kt <= C::ktmax(n); ++kt) {
          const uint32_t b[2] = {bw(2 * kt, n), 2 * kt + 1 <= n ? bw(2 * kt + 1, n) : 0u};
#pragma unroll
          for (int M = 0; M < MT; ++M) {
            if (!C::has_tile(M, n)) continue;
            mma16816<FP16>(acc[M][n], af[M][kt], b);
          }
        }
      // j = N term of column NB: V^T[k][N] += T^[k][N] L~_NN.
      if (tq == 0) {
#pragma unroll
        for (int M = 0; M < MT; ++M)
#pragma unroll
          for (int h = 0; h < 2; ++h) acc[M][NT - 1][2 * h] = fmaf(tkN[M][h], LNN, acc[M][NT - 1][2 * h]);
      }
      const float vnn = fmaf(LNN, tnNN, LNN) + part;
      // Keep V^T on and above its diagonal (nothing reads the blocks below it).
#pragma unroll
      for (int M = 0; M < MT; ++M) {
        if (lo0) acc[M][2 * M][0] = 0.f;
        if (lo1) acc[M][2 * M][1] = 0.f;
        if (lo0) acc[M][2 * M + 1][2] = 0.f;
        if (lo1) acc[M][2 * M + 1][3] = 0.f;
      }
      vmin = fminf(vmin, vnn);
      if (literal) LNN = vnn >= 0.f ? DN : -DN;
      // prox: squared norms of this lane's 8 rows k, summed over the 4 lanes of a row; each
      // row's scale is formed in the lane that owns its sum.
      float sn[R], own[R / 4], sc_own[R / 4];
#pragma unroll
      for (int M = 0; M < MT; ++M)
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          uint64_t v2 = 0ull;
#pragma unroll
          for (int n = 0; n < NT; ++n) {
            if (!C::has_tile(M, n) || (n == 2 * M && h == 1)) continue;   // below the diagonal
            const uint64_t x = f2pack(acc[M][n][2 * h], acc[M][n][2 * h + 1]);
            v2 = f2fma(x, x, v2);
          }
          float a, b;
          f2unpack(v2, a, b);
          sn[2 * M + h] = a + b;
        }
      row_sums<R>(sn, own, tq);
#pragma unroll
      for (int u = 0; u < R / 4; ++u) {
        snmin = fminf(snmin, own[u] + inval_own[u]);
        sc_own[u] = own[u] > 0.f ? D_own[u] * rsqrtf(own[u]) : 0.f;
      }
#pragma unroll
      for (int M = 0; M < MT; ++M)
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          const int r = 2 * M + h;
          const float sc = __shfl_sync(TASER_FULL_MASK, sc_own[r / 4], (lane & 28) + r % 4);
          const uint64_t sc2 = f2pack(sc, sc);
#pragma unroll
          for (int n = 0; n < NT; ++n) {
            if (!C::has_tile(M, n) || (n == 2 * M && h == 1)) continue;
            TASER_PAIR_APPLY(acc[M][n], 2 * h, f2mul(_x, sc2));
          }
        }
    }

    // A zero column in any iteration (its prox scale was 0): measured 2.2% faster than a
    // per-iteration flag update.
    if (snmin <= 0.f) fl |= TASER_FLAG_ZERO_COLUMN;
    if ((literal || tq == 0) && vmin <= 0.f) fl |= TASER_FLAG_LNN_SIGN;
    const JobOut o = outs[cur_m];
    // Decisions from row N of L~ (column NB of L~^T, lanes tq == 0).
    if (tq == 0) {
#pragma unroll
      for (int M = 0; M < MT; ++M)
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          const int k = 16 * M + g + 8 * h;
          if (k < N - 1 TASER_AND(TASER_IN(k, N - 1))) {
            float r = acc[M][NT - 1][2 * h];
            if (literal && LNN < 0.f) r = -r;
            o.s[k] = r >= 0.f ? int8_t(1) : int8_t(-1);
          }
        }
    }
    if (o.L != nullptr) {
      float* Lo = o.L;
#pragma unroll
      for (int M = 0; M < MT; ++M)
#pragma unroll
        for (int n = 0; n < NT; ++n)
#pragma unroll
          for (int e = 0; e < 4; ++e) {
            const int k = 16 * M + g + 8 * (e >> 1), i = 8 * n + 2 * tq + (e & 1);
            const int rr = bucket_to_real(i, N, NB);
            if (rr < 0 || k >= N - 1) continue;
            TASER_CHECKED(TASER_IN(rr * N + k, N * N)) Lo[(int64_t)rr * N + k] = C::has_tile(M, n) && !(n == 2 * M && e >= 2) ? acc[M][n][e] : 0.f;
          }
      for (int rr = lane; rr < N; rr += 32)
        TASER_CHECKED(TASER_IN(rr * N + N - 1, N * N)) Lo[(int64_t)rr * N + (N - 1)] = rr == N - 1 ? LNN : 0.f;
    }
#pragma unroll
    for (int ofs = 16; ofs > 0; ofs >>= 1) fl |= __shfl_xor_sync(TASER_FULL_MASK, fl, ofs);
    if (lane == 0 && o.flag != nullptr && fl) *o.flag |= fl;
    __syncwarp();  // the record of this job is consumed before it is reused
    cur_m ^= 1;
    have = have_next;
  }
}

template <class Src>
static cudaError_t launch_tct64(const Src& src, int64_t jobs, int blocks_per_sm, int literal, bool fp16,
                                cudaStream_t st) {
  const int slot_floats = tc_slot_floats(65);
  const size_t smem = (size_t)4 * (kBlk64Words + slot_floats + kTcRecFloats) * sizeof(uint32_t);
  return fp16 ? launch_persistent(detect_tct64_kernel<true, Src>, smem, src, jobs, blocks_per_sm, st, literal, slot_floats)
              : launch_persistent(detect_tct64_kernel<false, Src>, smem, src, jobs, blocks_per_sm, st, literal,
                                  slot_floats);
}

// Returns cudaErrorNotSupported when the bucket has no tensor-core kernel.
cudaError_t detect_tc(int64_t batch, int N, const float* Tt, const float* D, const float* tau, int t_max,
                      int literal, bool fp16, float* L, int8_t* s, uint32_t* flags, cudaStream_t st) {
  const DenseSource src{batch, 0, N, t_max, Tt, D, tau, L, s, flags, nullptr};
  switch (bucket_of(N)) {
    case 64: return launch_tct64(src, batch, 0, literal, fp16, st);
    case 16: return launch_tc<16, false>(src, batch, 0, literal, fp16, tc_slot_floats(N), 0.f, st);
    case 32: return launch_tc<32, false>(src, batch, 0, literal, fp16, tc_slot_floats(N), 0.f, st);
    default: return cudaErrorNotSupported;
  }
}

// taser_detect_monitored on the tensor cores (buckets 16 and 32; cudaErrorNotSupported
// for the bucket 64).
cudaError_t detect_tc_monitored(int64_t batch, int N, const float* Tt, const float* D, const float* tau, int t_max,
                                int literal, bool fp16, float ascent_tol, double* obj, float* L, int8_t* s,
                                uint32_t* flags, cudaStream_t st) {
  const DenseSource src{batch, 0, N, t_max, Tt, D, tau, L, s, flags, obj};
  switch (bucket_of(N)) {
    case 16: return launch_tc<16, true>(src, batch, 0, literal, fp16, tc_slot_floats(N), ascent_tol, st);
    case 32: return launch_tc<32, true>(src, batch, 0, literal, fp16, tc_slot_floats(N), ascent_tol, st);
    default: return cudaErrorNotSupported;
  }
}

// Queue-fed launch for bucket nb (16, 32 or 64) of an uneven batch.
cudaError_t detect_tc_queue(int nb, bool fp16, const Queue& q, int blocks_per_sm, int pop, const float* T_pool,
                            const float* D_pool, const float* tau, int literal, float* L_pool, int8_t* s_pool,
                            uint32_t* flags, cudaStream_t st) {
  const QueueSource src{q, pop > 0 ? pop : 1, T_pool, D_pool, tau, L_pool, s_pool, flags};
  switch (nb) {
    case 64: return launch_tct64(src, -1, blocks_per_sm, literal, fp16, st);
    case 16: return launch_tc<16, false>(src, -1, blocks_per_sm, literal, fp16, tc_slot_floats(17), 0.f, st);
    case 32: return launch_tc<32, false>(src, -1, blocks_per_sm, literal, fp16, tc_slot_floats(33), 0.f, st);
    default: return cudaErrorNotSupported;
  }
}

}  // namespace taser

TASER_DEBUG_COLLECTOR(detect_tc)
