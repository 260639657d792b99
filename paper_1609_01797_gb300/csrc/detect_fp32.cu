// FP32 TASER iterations (Algorithm 1) on the CUDA cores.
//
// Mapping: NB / 2 lanes per instance (NB >= N - 1 columns: 8, 12, .., 32, 64), lane gl
// owning the columns ca = gl and cb = NB / 2 + gl of L~ and V (small batches: NB lanes, one column
// each).  Its columns of T^ = -2 tau T~ (negated so every product is one FMA) live in registers
// for all t_max iterations, as packed pairs (T^_kj, T^_k+1,j); the rows of L~(t-1) are broadcast
// from shared memory, and one LDS.128 feeds two packed f32x2 FMAs per column, which keep the
// even- and odd-k partial sums of the row.  The stored L~ is zero above the diagonal and in the row padding, so the last
// float4 of a row needs no masking.  Column norms of the prox (Sec. III-C) are then lane-local
// sums.  L~ never leaves the SM between iterations.
//
// Why two columns a lane: with one, the broadcasts (two cycles of register write-back each)
// kept the L1 data pipe 93% busy at N = 33.  Here one broadcast serves both columns and
// 32 / G instances, and rows < NB / 2 skip every cb at compile time; each column's sums keep
// their order.  What bounds it now is the register file: a packed FMA with three different
// 64-bit operands takes 3 cycles of operand reads, 2.3 to 2.6 with reuse, not the 2 of the
// FMA pipe (measured in a loop of them).  Per 65,536 problems, t_max = 20: N = 33 1.49 ->
// 1.09 ms, N = 17 0.292 -> 0.202 ms, N = 9 0.079 -> 0.056 ms.  Measured and not kept at
// N = 33: 168 registers (12 warps an SM) with and without the rows split over two warps, 1.22
// and 1.16 ms; four columns a lane with split rows 1.13 ms.
#include <type_traits>

#include "common.cuh"

namespace taser {

// NB <= 32: L~ and V columns in registers too, all loops unrolled.  COLS columns a lane: 2, or 1
// for batches that leave the GPU's schedulers without a second warp (one_column_max below).
template <int NB, int COLS>
struct FoldCfg {
  static constexpr int HALF = NB / COLS;             // columns ca of the lanes
  static constexpr int FB = COLS == 2 ? HALF : NB + 1;   // first row that a column cb reaches
  static constexpr int G = group_lanes(HALF);        // lanes of one instance, HALF of them at work
  static constexpr int IPW = 32 / G;                 // instances of a warp
  static constexpr int S = NB + 4;                   // smem row stride (floats), 16B rows
  static constexpr int ROWS = (NB + 1) * S;
  // Instances sit G banks apart (mod 32), so the column stores of a warp hit 32 banks.
  static constexpr int INST_FLOATS = ROWS + ((G - ROWS % 32) % 32 + 32) % 32;
  static constexpr int NP = NB / 2 + 1;              // pairs (k, k + 1) of a column of T^
  static constexpr int WARPS = 4;
  static constexpr int IPC = WARPS * IPW;            // instances per block
  static constexpr int SMEM_BYTES = IPC * INST_FLOATS * 4;
  // NB = 32 holds 118 floats of T^ and L~ a lane, NB = 24 90; the loads in flight need the rest.
  static constexpr int MIN_BLOCKS = COLS == 2 ? (NB >= 28 ? 2 : (NB >= 20 ? 3 : 4)) : (NB >= 20 ? 3 : 1);
};

// NB = 64: two warps per instance, lane j of the pair owning column j (the second warp skips
// rows < 32, all above its columns).  Two columns a lane do not pay here: their 130 registers
// of T^ leave no room for the columns of L~, and with those kept in shared memory one warp per
// instance took 1.25 ms per 8,192 at N = 65, t_max = 20 (from 1.41) but 0.136 ms (from 0.085)
// for 101 problems; two warps sharing the rows took 1.64 ms, four 1.84 ms (their four unrolled
// bodies miss the instruction cache).
struct PairCfg {
  static constexpr int WPI = 2;                      // warps per instance
  static constexpr int S = 64 + 4;                   // smem row stride (floats), 16B rows
  static constexpr int INST_FLOATS = 65 * S + 4;     // the iterate, then 4 words of exchange
  static constexpr int WARPS = 4;                    // warps per block
  static constexpr int IPC = WARPS / WPI;            // instances per block
  static constexpr int SMEM_BYTES = IPC * INST_FLOATS * 4;
  static constexpr int MIN_BLOCKS = 1;
};

template <int NB, int COLS = 2>
using Fp32Cfg = std::conditional_t<NB <= 32, FoldCfg<NB <= 32 ? NB : 32, COLS>, PairCfg>;

// Starts a row's two partial sums with the pair k = 0, 1: (l + q_0 t_0, q_1 t_1).
__device__ __forceinline__ uint64_t f2start(uint64_t q, uint64_t t, float l) {
  float q0, q1, t0, t1;
  f2unpack(q, q0, q1);
  f2unpack(t, t0, t1);
  return f2pack(fmaf(q0, t0, l), __fmul_rn(q1, t1));
}

// Scale of a column of squared norm n2 to norm D; a real column (r >= 0) of norm zero is flagged.
__device__ __forceinline__ float prox_scale(float n2, float D, int r, uint32_t& fl) {
  if (n2 > 0.f) return D * rsqrtf(n2);
  if (r >= 0) fl |= TASER_FLAG_ZERO_COLUMN;
  return 0.f;
}

// Runs Algorithm 1 for `jb` (inactive lanes compute on zeros and write nothing).
// t_loop: iterations the warp executes (the largest t_max among its instances).  MIXED:
// instances sharing the warp may have different t_max, so outputs are emitted inside the
// loop at each instance's own last iteration; otherwise once after the loop.
// MON: objective monitoring (taser_detect_monitored).  f(L~) = Tr(L~ T~ L~^T) equals
// sum_{i >= k} L~_ik (L~ T~)_ik, and the gradient step computes exactly that lower part:
// V = L~ - 2 tau tril(L~ T~), so f(L~(t)) = sum L~(t)_ik (L~(t)_ik - V(t+1)_ik) / (2 tau),
// accumulated from the iteration's own FP32 values (no extra product).  One more product
// after the last iteration gives f(L~(t_max)); its V is discarded.
template <int NB, int COLS, bool MIXED, bool MON>
__device__ __forceinline__ void fold_run(const Job& jb, bool active, int t_loop, float* Ls, int gl, int lane,
                                         int literal, double* obj, float ascent_tol) {
  using C = FoldCfg<NB, COLS>;
  constexpr int HALF = C::HALF, FB = C::FB, S = C::S, NP = C::NP;
  const unsigned gmask = (TASER_FULL_MASK >> (32 - C::G)) << (lane & ~(C::G - 1));
  const int N = active ? jb.N : NB + 1;
  const bool at_work = C::G == HALF || gl < HALF;   // the other lanes carry zeros
  const int ca = gl, cb = COLS == 2 ? (NB == 12 ? NB - 1 - gl : HALF + gl) : gl;
  const int ra = at_work && ca < N - 1 ? ca : -1;   // real columns (-1: padding)
  const int rb = COLS == 2 && at_work && cb < N - 1 ? cb : -1;
  const float tau = active ? *jb.tau : 0.f;
  const float m2tau = -2.f * tau;

  // The columns of T^ = -2 tau T~ (T~ symmetric: T~[k][j] read row by row).
  uint64_t ta[NP], tb[COLS == 2 ? NP : 1];
  auto load = [&](int k, int r) -> float {
    const int kr = k <= NB ? bucket_to_real(k, N, NB) : -1;
    return m2tau * (active && kr >= 0 && r >= 0 && TASER_IN(kr * N + r, N * N) ? jb.T[(int64_t)kr * N + r] : 0.f);
  };
#pragma unroll
  for (int p = 0; p < NP; ++p) {
    ta[p] = f2pack(load(2 * p, ra), load(2 * p + 1, ra));
    if constexpr (COLS == 2) tb[p] = f2pack(load(2 * p, rb), load(2 * p + 1, rb));
  }
  const float Da = (active && ra >= 0 && TASER_IN(ra, N)) ? jb.D[ra] : 0.f;
  const float Db = (active && rb >= 0 && TASER_IN(rb, N)) ? jb.D[rb] : 0.f;
  const float DN = active ? jb.D[N - 1] : 0.f;
  const float tnNN = m2tau * (active ? jb.T[(int64_t)(N - 1) * N + (N - 1)] : 0.f);

  // L~(0) = D (Algorithm 1 initialisation).
  for (int idx = gl; idx < C::ROWS; idx += C::G) Ls[idx] = 0.f;
  __syncwarp();
  if (at_work && TASER_IN(ca * S + ca, C::ROWS)) Ls[ca * S + ca] = Da;
  if (COLS == 2 && at_work && TASER_IN(cb * S + cb, C::ROWS)) Ls[cb * S + cb] = Db;
  if (gl == 0) Ls[NB * S + NB] = DN;
  float la[NB + 1], lb[COLS == 2 ? NB + 1 - FB : 1];   // columns ca (all rows) and cb (rows FB..NB)
#pragma unroll
  for (int i = 0; i <= NB; ++i) la[i] = (i == ca) ? Da : 0.f;
#pragma unroll
  for (int i = FB; i <= NB; ++i) lb[i - FB] = (i == cb) ? Db : 0.f;
  float LNN = DN;
  uint32_t fl = 0;
  __syncwarp();

  // Outputs of this instance (its lanes call this together).
  auto emit = [&]() {
    uint32_t f = fl;
#pragma unroll
    for (int o = C::G / 2; o > 0; o >>= 1) f |= __shfl_xor_sync(gmask, f, o);
    if (gl == 0 && jb.flag != nullptr && f) *jb.flag |= f;
    // Decisions s_k = sign(L~_{N,k}) (sign(0) = +1), times sign(L~_NN) in literal mode.
    const bool flip = literal && LNN < 0.f;
    auto decide = [&](int r, float v) {
      if (r < 0 || !TASER_IN(r, N - 1)) return;
      TASER_FINITE(v);
      jb.s[r] = ((flip ? -v : v) >= 0.f) ? int8_t(1) : int8_t(-1);
    };
    decide(ra, la[NB]);
    if constexpr (COLS == 2) decide(rb, lb[NB - FB]);
    if (jb.L != nullptr) {
#pragma unroll
      for (int i = 0; i <= NB; ++i) {
        const int ir = bucket_to_real(i, N, NB);
        if (ir < 0) continue;
        auto put = [&](int r, float v) {
          if (r < 0 || !TASER_IN(ir * N + r, N * N)) return;
          jb.L[(int64_t)ir * N + r] = v;
          TASER_FINITE(v);
        };
        put(ra, la[i]);
        if constexpr (COLS == 2) put(rb, i < FB ? 0.f : lb[i < FB ? 0 : i - FB]);
        if (gl == 0 && TASER_IN(ir * N + N - 1, N * N)) jb.L[(int64_t)ir * N + (N - 1)] = (ir == N - 1) ? LNN : 0.f;
      }
    }
  };

  double f_prev = 0.0;
  for (int t = 0; t < t_loop + (MON ? 1 : 0); ++t) {
    const bool last_pass = MON && t == t_loop;   // only f(L~(t_max)); L~ stays as it is
    // Partial of V_NN = L~_NN (1 - 2 tau T~_NN) - 2 tau sum_k L~_Nk T~_kN from L~(t-1).
    float tNa, tNb = 0.f, lNb = 0.f, unused;
    f2unpack(ta[NP - 1], tNa, unused);
    if constexpr (COLS == 2) {
      f2unpack(tb[NP - 1], tNb, unused);
      lNb = lb[NB - FB];
    }
    float part = column_halves<NB, COLS>(__fmul_rn(la[NB], tNa), __fmul_rn(lNb, tNb), gl, lane);
    float fa = 0.f, fb = 0.f;   // MON: sums of L~_ij (L~_ij - V_ij) over the lane's columns

    // V = L~ - tril(2 tau L~ T~): row i needs L~_ik, k <= i only (triangular skip).  The pair
    // k = 0, 1 starts a row's two partial sums (L~_ij joins the even one) without the moves
    // that a packed {L~_ij, 0} would need.
#pragma unroll
    for (int i = 0; i <= NB; ++i) {
      const float* row = Ls + i * S;
      uint64_t acca = 0ull, accb = 0ull;
#pragma unroll
      for (int k4 = 0; k4 <= i; k4 += 4) {
        const float4 q = *reinterpret_cast<const float4*>(row + k4);
        const uint64_t q0 = f2pack(q.x, q.y), q1 = f2pack(q.z, q.w);
        acca = k4 == 0 ? f2start(q0, ta[0], la[i]) : f2fma(q0, ta[k4 / 2], acca);
        if (i >= FB) accb = k4 == 0 ? f2start(q0, tb[0], lb[i < FB ? 0 : i - FB]) : f2fma(q0, tb[k4 / 2], accb);
        if (k4 + 2 <= i) {
          acca = f2fma(q1, ta[k4 / 2 + 1], acca);
          if (i >= FB) accb = f2fma(q1, tb[k4 / 2 + 1], accb);
        }
      }
      float a0, a1;
      f2unpack(acca, a0, a1);
      const float va = (i >= HALF || i >= ca) ? a0 + a1 : 0.f;   // ca < HALF
      if constexpr (MON) fa = fmaf(la[i], la[i] - va, fa);
      if (!last_pass) la[i] = va;   // la now holds column ca of V
      if (i >= FB) {
        f2unpack(accb, a0, a1);
        const float vb = (i >= cb) ? a0 + a1 : 0.f;
        if constexpr (MON) fb = fmaf(lb[i - FB], lb[i - FB] - vb, fb);
        if (!last_pass) lb[i - FB] = vb;
      }
    }
    float fterm = 0.f;
    if constexpr (MON) fterm = column_total<NB, COLS>(column_halves<NB, COLS>(fa, fb, gl, lane));
    part = column_total<NB, COLS>(part);   // its shuffles under the products: N = 25 1 to 2% faster than before them
    __syncwarp();  // every lane has finished reading L~(t-1)
    const float vnn = fmaf(LNN, tnNN, LNN) + part;
    if constexpr (MON) {
      fterm = fmaf(LNN, LNN - vnn, fterm);
      // f in FP64 from the FP32 sum; ascent when f(L~(t)) > f(L~(t-1)) + tol |f(L~(t-1))|.
      const double f = tau > 0.f ? (double)fterm / (2.0 * (double)tau) : 0.0;
      if (t > 0 && f > f_prev + (double)ascent_tol * fabs(f_prev)) fl |= TASER_FLAG_ASCENT;
      f_prev = f;
      if (active && obj != nullptr && gl == 0 && TASER_IN(t, t_loop + 1)) obj[t] = f;
      if (last_pass) break;
    }
    if (vnn <= 0.f) fl |= TASER_FLAG_LNN_SIGN;
    if (literal) LNN = vnn >= 0.f ? DN : -DN;

    // prox: each column rescaled to norm D_jj.
    float na = 0.f, nb = 0.f;
#pragma unroll
    for (int i = 0; i <= NB; ++i) {
      na = fmaf(la[i], la[i], na);
      if (i >= FB) nb = fmaf(lb[i - FB], lb[i - FB], nb);
    }
    const float sa = prox_scale(na, Da, ra, fl), sb = prox_scale(nb, Db, rb, fl);
#pragma unroll
    for (int i = 0; i <= NB; ++i) {
      la[i] *= sa;
      if (at_work && TASER_IN(i * S + ca, C::ROWS)) Ls[i * S + ca] = la[i];
      if (i >= FB) {
        lb[i - FB] *= sb;
        if (at_work && TASER_IN(i * S + cb, C::ROWS)) Ls[i * S + cb] = lb[i - FB];
      }
    }
    if (literal && gl == 0) Ls[NB * S + NB] = LNN;
    __syncwarp();

    if constexpr (MIXED) {
      if (t + 1 == (active ? jb.t_max : -1)) emit();
    }
  }
  if constexpr (!MIXED) {
    if (active) emit();
  }
}

// Barrier of the two warps of an instance (NB = 64).
__device__ __forceinline__ void sync_pair(int bar_id) {
  asm volatile("bar.sync %0, %1;" ::"r"(bar_id), "r"(64) : "memory");
}

// The same for NB = 64 (34 <= N <= 65), lane j of the warp pair owning column j; MON as in
// fold_run.
template <bool MON>
__device__ __forceinline__ void pair_run(const Job& jb, bool active, int t_loop, float* Ls, int lane, int warp,
                                         int bar_id, int literal, double* obj, float ascent_tol) {
  using C = PairCfg;
  constexpr int NB = 64;
  const int j = (warp % C::WPI) * 32 + lane;
  const int colbase = (warp % C::WPI) * 32;  // warp-uniform
  float* const xs = Ls + 65 * C::S;
  const int N = active ? jb.N : NB + 1;
  const int jr = j < N - 1 ? j : -1;                         // real column (variable)
  const float tau = active ? *jb.tau : 0.f;
  const float m2tau = -2.f * tau;

  // Column j of T^ = -2 tau T~ (T~ symmetric: T~[k][j] read row by row, coalesced), as
  // pairs (k, k + 1); pairs past k = NB are zero.
  constexpr int NP2 = NB / 2 + 2;
  uint64_t tn2[NP2];
  float tNB = 0.f;
#pragma unroll
  for (int p = 0; p < NP2; ++p) {
    float v2[2];
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const int k = 2 * p + h;
      float v = 0.f;
      if (k <= NB) {
        const int kr = bucket_to_real(k, N, NB);
        if (active && jr >= 0 && kr >= 0 && TASER_IN(kr * N + jr, N * N)) v = jb.T[(int64_t)kr * N + jr];
      }
      v2[h] = m2tau * v;
      if (k == NB) tNB = v2[h];
    }
    tn2[p] = f2pack(v2[0], v2[1]);
  }
  const float Dj = (active && jr >= 0 && TASER_IN(jr, N)) ? jb.D[jr] : 0.f;
  const float DN = active ? jb.D[N - 1] : 0.f;
  const float tnNN = m2tau * (active ? jb.T[(int64_t)(N - 1) * N + (N - 1)] : 0.f);

  // L~(0) = D (Algorithm 1 initialisation).
  for (int idx = j; idx < C::INST_FLOATS; idx += 64) Ls[idx] = 0.f;
  sync_pair(bar_id);
  if (TASER_IN(j * C::S + j, C::INST_FLOATS)) Ls[j * C::S + j] = Dj;
  if (j == 0) Ls[NB * C::S + NB] = DN;
  float l[NB + 1];
#pragma unroll
  for (int i = 0; i <= NB; ++i) l[i] = (i == j) ? Dj : 0.f;
  float LNN = DN;
  uint32_t fl = 0;
  sync_pair(bar_id);

  // Outputs of this instance (its lanes call this together).
  auto emit = [&]() {
    uint32_t f = fl;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) f |= __shfl_xor_sync(TASER_FULL_MASK, f, o);
    if (lane == 0 && jb.flag != nullptr && f) atomicOr(jb.flag, f);
    // Decisions s_k = sign(L~_{N,k}) (sign(0) = +1), times sign(L~_NN) in literal mode.
    if (jr >= 0 && TASER_IN(jr, N - 1)) {
      float r = l[NB];
      TASER_FINITE(r);
      if (literal && LNN < 0.f) r = -r;
      jb.s[jr] = (r >= 0.f) ? int8_t(1) : int8_t(-1);
    }
    if (jb.L != nullptr) {
#pragma unroll
      for (int i = 0; i <= NB; ++i) {
        const int ir = bucket_to_real(i, N, NB);
        if (ir < 0) continue;
        if (jr >= 0 && TASER_IN(ir * N + jr, N * N)) {
          jb.L[(int64_t)ir * N + jr] = l[i];
          TASER_FINITE(l[i]);
        }
        if (j == 0 && TASER_IN(ir * N + N - 1, N * N)) jb.L[(int64_t)ir * N + (N - 1)] = (ir == N - 1) ? LNN : 0.f;
      }
    }
  };

  double f_prev = 0.0;
  for (int t = 0; t < t_loop + (MON ? 1 : 0); ++t) {
    const bool last_pass = MON && t == t_loop;   // only f(L~(t_max)); L~ stays as it is
    // Partial of V_NN = L~_NN (1 - 2 tau T~_NN) - 2 tau sum_k L~_Nk T~_kN from L~(t-1).
    float part = l[NB] * tNB;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) part += __shfl_xor_sync(TASER_FULL_MASK, part, o);
    float fterm = 0.f;   // MON: this lane's sum of L~_ij (L~_ij - V_ij)

    // V = L~ - tril(2 tau L~ T~): row i needs L~_ik, k <= i only (triangular skip).
#pragma unroll
    for (int i = 0; i <= NB; ++i) {
      if (i < 32 && colbase != 0) {
        l[i] = 0.f;  // rows above every column of this warp
        continue;
      }
      uint64_t acc2 = f2pack(l[i], 0.f);
      const float* row = Ls + i * C::S;
#pragma unroll
      for (int k4 = 0; k4 <= i; k4 += 4) {
        const float4 q = *reinterpret_cast<const float4*>(row + k4);
        acc2 = f2fma(f2pack(q.x, q.y), tn2[k4 / 2], acc2);
        if (k4 + 2 <= i) acc2 = f2fma(f2pack(q.z, q.w), tn2[k4 / 2 + 1], acc2);
      }
      float a0, a1;
      f2unpack(acc2, a0, a1);
      const float v = (i >= j) ? a0 + a1 : 0.f;
      if constexpr (MON) {
        fterm = fmaf(l[i], l[i] - v, fterm);
        if (!last_pass) l[i] = v;
      } else {
        l[i] = v;  // l now holds column j of V
      }
    }
    if constexpr (MON) {
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) fterm += __shfl_xor_sync(TASER_FULL_MASK, fterm, o);
      if (lane == 0) xs[2 + warp % C::WPI] = fterm;
    }
    if (lane == 0) xs[warp % C::WPI] = part;
    sync_pair(bar_id);  // every lane has finished reading L~(t-1)
    part = xs[0] + xs[1];
    const float vnn = fmaf(LNN, tnNN, LNN) + part;
    if constexpr (MON) {
      fterm = xs[2] + xs[3];
      fterm = fmaf(LNN, LNN - vnn, fterm);
      // f in FP64 from the FP32 sum; ascent when f(L~(t)) > f(L~(t-1)) + tol |f(L~(t-1))|.
      const double f = tau > 0.f ? (double)fterm / (2.0 * (double)tau) : 0.0;
      if (t > 0 && f > f_prev + (double)ascent_tol * fabs(f_prev)) fl |= TASER_FLAG_ASCENT;
      f_prev = f;
      if (active && obj != nullptr && j == 0 && colbase == 0 && TASER_IN(t, t_loop + 1)) obj[t] = f;
      if (last_pass) {
        sync_pair(bar_id);   // xs is read before it is reused
        break;
      }
    }
    if (vnn <= 0.f) fl |= TASER_FLAG_LNN_SIGN;
    if (literal) LNN = vnn >= 0.f ? DN : -DN;

    // prox: column j rescaled to norm D_jj.
    float n2 = 0.f;
#pragma unroll
    for (int i = 0; i <= NB; ++i) {
      if (i < 32 && colbase != 0) continue;
      n2 = fmaf(l[i], l[i], n2);
    }
    float sc = 0.f;
    if (n2 > 0.f) {
      sc = Dj * rsqrtf(n2);
    } else if (jr >= 0) {
      fl |= TASER_FLAG_ZERO_COLUMN;
    }
#pragma unroll
    for (int i = 0; i <= NB; ++i) {
      if (i < 32 && colbase != 0) continue;
      l[i] *= sc;
      if (TASER_IN(i * C::S + j, C::INST_FLOATS)) Ls[i * C::S + j] = l[i];
    }
    if (literal && j == 0) Ls[NB * C::S + NB] = LNN;
    sync_pair(bar_id);
  }
  if (active) emit();
}

// (The monitor's FP64 division and its sums spill in 128 registers at NB = 16.)
template <int NB, int COLS, bool MON>
__global__ void __launch_bounds__(128, MON && NB == 16 && COLS == 2 ? 3 : Fp32Cfg<NB, COLS>::MIN_BLOCKS)
detect_fp32_kernel(int64_t batch, int N, const float* __restrict__ Tt, const float* __restrict__ Dg,
                   const float* __restrict__ tau_g, int t_max, int literal, float* __restrict__ Lout,
                   int8_t* __restrict__ s_hat, uint32_t* __restrict__ flags, double* __restrict__ obj,
                   float ascent_tol) {
  using C = Fp32Cfg<NB, COLS>;
  extern __shared__ __align__(16) float smem[];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int local = threadIdx.x / (128 / C::IPC);   // instance of the block
  const int64_t inst = (int64_t)blockIdx.x * C::IPC + local;
  const bool active = inst < batch;
  const Job jb = dense_job(active ? inst : 0, N, t_max, Tt, Dg, tau_g, Lout, s_hat, flags);
  double* ob = (MON && obj != nullptr) ? obj + (active ? inst : 0) * (int64_t)(t_max + 1) : nullptr;
  float* Ls = smem + local * C::INST_FLOATS;
  if constexpr (NB <= 32) {
    fold_run<NB, COLS, false, MON>(jb, active, t_max, Ls, lane % C::G, lane, literal, ob, ascent_tol);
  } else {
    pair_run<MON>(jb, active, t_max, Ls, lane, warp, 1 + local, literal, ob, ascent_tol);
  }
}

// Persistent, queue-fed: each warp (each warp pair for NB = 64) pops the next items of its
// bucket until the queue is empty, `rounds` warp-loads per pop (one atomic per rounds x IPW
// items: short jobs would otherwise queue on the counter).
template <int NB, int COLS>
__global__ void __launch_bounds__(128, Fp32Cfg<NB, COLS>::MIN_BLOCKS)
detect_fp32_queue_kernel(Queue q, int rounds, const float* __restrict__ T_pool, const float* __restrict__ D_pool,
                         const float* __restrict__ tau, int literal, float* __restrict__ L_pool,
                         int8_t* __restrict__ s_pool, uint32_t* __restrict__ flags) {
  using C = Fp32Cfg<NB, COLS>;
  extern __shared__ __align__(16) float smem[];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int local = threadIdx.x / (128 / C::IPC);   // instance of the block
  float* Ls = smem + local * C::INST_FLOATS;
  const int count = q.count();
  auto job = [&](int pos) {
    const int idx = pos < count ? q.item_at(pos) : 0;
    return item_job(q.items[idx], idx, T_pool, D_pool, tau, L_pool, s_pool, flags);
  };
  if constexpr (NB <= 32) {
    // Warps beyond the queue's pops leave the counter alone: 2,432 of them queued on it before the
    // few that had work, also in the buckets without items (500 items of N = 9 in two columns a lane
    // 37.5 -> 26.8 us, 8,000 of N = 17 64.3 -> 60.5; a kernel without items 4 to 5 -> 3 us).
    if ((int64_t)(blockIdx.x * C::WARPS + warp) * (C::IPW * rounds) >= count) return;
  }
  for (;;) {
    int base = 0;
    if constexpr (NB <= 32) {
      if (lane == 0) base = q.pop(C::IPW * rounds);
      base = __shfl_sync(TASER_FULL_MASK, base, 0);
      if (base >= count) break;                                   // uniform per warp
      for (int r = 0; r < rounds && base + r * C::IPW < count; ++r) {
        const int pos = base + r * C::IPW + lane / C::G;
        const Job jb = job(pos);
        const int t_loop = __reduce_max_sync(TASER_FULL_MASK, pos < count ? jb.t_max : 0);
        fold_run<NB, COLS, (C::IPW > 1), false>(jb, pos < count, t_loop, Ls, lane % C::G, lane, literal, nullptr, 0.f);
        __syncwarp();
      }
    } else {
      int* const slot = reinterpret_cast<int*>(Ls + 65 * C::S + 2);   // a word that only the monitor uses
      if (warp % C::WPI == 0 && lane == 0) *slot = q.pop(rounds);
      sync_pair(1 + local);
      base = *slot;
      sync_pair(1 + local);
      if (base >= count) break;                                   // uniform per warp pair
      for (int pos = base; pos < base + rounds && pos < count; ++pos) {
        const Job jb = job(pos);
        pair_run<false>(jb, true, jb.t_max, Ls, lane, warp, 1 + local, literal, nullptr, 0.f);
        sync_pair(1 + local);   // the iterate is read before the next job overwrites it
      }
    }
  }
}

// Largest batch that runs with one column a lane.  With two, a warp's chain of an iteration is 1.75
// times as long (506 against 289 packed FMAs at NB = 32), which nothing hides while every scheduler
// (4 an SM) holds at most one warp of the one-column layout.  One column against two, t_max = 20:
// N = 33 512 problems 19.5 / 25.6 us, 1,024 32.2 / 25.9; N = 25 13.4 / 17.0 and 21.3 / 17.6; N = 17
// 1,024 problems 8.6 / 11.1, 2,048 12.5 / 11.3; N = 9 2,048 5.8 / 6.4, 4,096 7.0 / 6.5; monitored,
// N = 17 512 problems 19.7 / 29.1.
template <int NB>
static cudaError_t one_column_max(int64_t& most, int& sms) {
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  most = (int64_t)sms * 4 * FoldCfg<NB, 1>::IPW;
  return e;
}

template <int NB, int COLS, bool MON>
static cudaError_t launch_dense(int64_t batch, int N, const float* Tt, const float* D, const float* tau,
                                int t_max, int literal, float* L, int8_t* s, uint32_t* flags, double* obj,
                                float ascent_tol, cudaStream_t st) {
  using C = Fp32Cfg<NB, COLS>;
  const int64_t blocks = (batch + C::IPC - 1) / C::IPC;
  if (C::SMEM_BYTES > 48 * 1024) {
    cudaError_t e = cudaFuncSetAttribute(detect_fp32_kernel<NB, COLS, MON>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         C::SMEM_BYTES);
    if (e != cudaSuccess) return e;
  }
  detect_fp32_kernel<NB, COLS, MON><<<(unsigned)blocks, 128, C::SMEM_BYTES, st>>>(batch, N, Tt, D, tau, t_max, literal,
                                                                                 L, s, flags, obj, ascent_tol);
  return cudaGetLastError();
}

template <int NB, bool MON>
static cudaError_t launch_fp32(int64_t batch, int N, const float* Tt, const float* D, const float* tau,
                               int t_max, int literal, float* L, int8_t* s, uint32_t* flags, double* obj,
                               float ascent_tol, cudaStream_t st) {
  if constexpr (NB <= 32) {
    int64_t most = 0;
    int sms = 0;
    const cudaError_t e = one_column_max<NB>(most, sms);
    if (e != cudaSuccess) return e;
    if (batch <= most)
      return launch_dense<NB, 1, MON>(batch, N, Tt, D, tau, t_max, literal, L, s, flags, obj, ascent_tol, st);
  }
  return launch_dense<NB, 2, MON>(batch, N, Tt, D, tau, t_max, literal, L, s, flags, obj, ascent_tol, st);
}

cudaError_t detect_fp32(int64_t batch, int N, const float* Tt, const float* D, const float* tau, int t_max,
                        int literal, float* L, int8_t* s, uint32_t* flags, cudaStream_t st) {
  // Column counts in steps of 4 up to 32: a problem pays for its own rows and columns, not for a
  // bucket twice its size (packed FMAs per warp and iteration: 506 at 32 columns, 394 / 296 / 212
  // at 28 / 24 / 20, 142 at 16, 86 at 12).  Per 10,007 problems, t_max = 20: N = 25 197 -> 131 us
  // against the 32-column layout.  The sums keep their order (V_NN: column_halves), so the results are
  // bitwise those of the queue-fed and the monitored kernels, which keep the buckets 8, 16, 32 and 64.
  auto go = [&](auto nb) {
    return launch_fp32<decltype(nb)::value, false>(batch, N, Tt, D, tau, t_max, literal, L, s, flags, nullptr, 0.f, st);
  };
  const int nv = N - 1;
  if (nv <= 8) return go(std::integral_constant<int, 8>{});
  if (nv <= 12) return go(std::integral_constant<int, 12>{});
  if (nv <= 16) return go(std::integral_constant<int, 16>{});
  if (nv <= 20) return go(std::integral_constant<int, 20>{});
  if (nv <= 24) return go(std::integral_constant<int, 24>{});
  if (nv <= 28) return go(std::integral_constant<int, 28>{});
  if (nv <= 32) return go(std::integral_constant<int, 32>{});
  return go(std::integral_constant<int, 64>{});
}

// taser_detect_monitored on the FP32 kernel: f(L~(t)) per iteration and the ascent flag.
cudaError_t detect_fp32_monitored(int64_t batch, int N, const float* Tt, const float* D, const float* tau,
                                  int t_max, int literal, float ascent_tol, double* obj, float* L, int8_t* s,
                                  uint32_t* flags, cudaStream_t st) {
  switch (bucket_of(N)) {
    case 8: return launch_fp32<8, true>(batch, N, Tt, D, tau, t_max, literal, L, s, flags, obj, ascent_tol, st);
    case 16: return launch_fp32<16, true>(batch, N, Tt, D, tau, t_max, literal, L, s, flags, obj, ascent_tol, st);
    case 32: return launch_fp32<32, true>(batch, N, Tt, D, tau, t_max, literal, L, s, flags, obj, ascent_tol, st);
    default: return launch_fp32<64, true>(batch, N, Tt, D, tau, t_max, literal, L, s, flags, obj, ascent_tol, st);
  }
}

// Queue-fed launch for bucket NB; pop items per queue pop (0: one warp-load), rounded up to whole
// warp-loads.
template <int NB, int COLS>
static cudaError_t launch_queue(const Queue& q, int sms, int blocks_per_sm, int pop, const float* T_pool,
                                const float* D_pool, const float* tau, int literal, float* L_pool, int8_t* s_pool,
                                uint32_t* flags, cudaStream_t st) {
  using C = Fp32Cfg<NB, COLS>;
  const auto kern = detect_fp32_queue_kernel<NB, COLS>;
  cudaError_t e = cudaSuccess;
  if (C::SMEM_BYTES > 48 * 1024)
    e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, C::SMEM_BYTES);
  int fit = 0;
  if (e == cudaSuccess) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&fit, kern, 128, C::SMEM_BYTES);
  if (e != cudaSuccess) return e;
  const int per_sm = blocks_per_sm > 0 && blocks_per_sm < fit ? blocks_per_sm : (fit > 0 ? fit : 1);
  int per_load = 1;   // items of a warp (pair)'s load
  if constexpr (NB <= 32) per_load = C::IPW;
  const int rounds = pop > per_load ? (pop + per_load - 1) / per_load : 1;
  kern<<<sms * per_sm, 128, C::SMEM_BYTES, st>>>(q, rounds, T_pool, D_pool, tau, literal, L_pool,
                                                 s_pool, flags);
  return cudaGetLastError();
}

template <int NB>
static cudaError_t launch_fp32_queue(const Queue& q, int blocks_per_sm, int pop, const float* T_pool,
                                     const float* D_pool, const float* tau, int literal, float* L_pool,
                                     int8_t* s_pool, uint32_t* flags, cudaStream_t st) {
  int64_t most = 0;
  int sms = 0;
  const cudaError_t e = one_column_max<NB <= 32 ? NB : 32>(most, sms);
  if (e != cudaSuccess) return e;
  // A queue's warp also waits for the counter, its items and their T~, so the one-column layout
  // leads for longer: per call of n items of one size, t_max 10 and 20 (one column / two): N = 9
  // n = 8,000 33.3 / 35.1 us, 12,000 38.8 / 36.1; N = 17 4,000 49.0 / 58.7, 6,000 60.3 / 59.7;
  // N = 33 2,000 65.8 / 71.8, 4,000 114.9 / 101.0.  Only the call's length is known here and the
  // bucket's may be shorter, so N = 17 keeps one column a little longer (3,000 of N = 9 and 3,000 of
  // N = 17 in one batch 55 / 66 us).
  if constexpr (NB <= 32) {
    if (q.n <= (NB == 16 ? 6 : 4) * most)
      return launch_queue<NB, 1>(q, sms, blocks_per_sm, pop, T_pool, D_pool, tau, literal, L_pool, s_pool, flags, st);
  }
  return launch_queue<NB, 2>(q, sms, blocks_per_sm, pop, T_pool, D_pool, tau, literal, L_pool, s_pool, flags, st);
}

cudaError_t detect_fp32_queue(int nb, const Queue& q, int blocks_per_sm, int pop, const float* T_pool,
                              const float* D_pool, const float* tau, int literal, float* L_pool, int8_t* s_pool,
                              uint32_t* flags, cudaStream_t st) {
  switch (nb) {
    case 8:
      return launch_fp32_queue<8>(q, blocks_per_sm, pop, T_pool, D_pool, tau, literal, L_pool, s_pool, flags, st);
    case 16:
      return launch_fp32_queue<16>(q, blocks_per_sm, pop, T_pool, D_pool, tau, literal, L_pool, s_pool, flags, st);
    case 32:
      return launch_fp32_queue<32>(q, blocks_per_sm, pop, T_pool, D_pool, tau, literal, L_pool, s_pool, flags, st);
    default:
      return launch_fp32_queue<64>(q, blocks_per_sm, pop, T_pool, D_pool, tau, literal, L_pool, s_pool, flags, st);
  }
}

}  // namespace taser

TASER_DEBUG_COLLECTOR(detect_fp32)
