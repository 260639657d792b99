// Unfolded TASER: Algorithm 1 with a learnable step per iteration, tau_t = alpha_t /
// ||T~||_2, its FP32 forward with checkpoints, and the hand-written adjoint.
//
// Forward (mode "fixed", L~_NN = D_NN):  V_t = L~(t-1) - tau_t tril(2 L~(t-1) T~),
// L~(t) = prox(V_t); soft output x_k = L~(t_max)_{N,k} / D_k (the last row of the
// unit-column factor L = L~ D^-1).  L~(kc) is saved every c iterations.
//
// Adjoint of one step, given Lbar = dloss/dL~(t):
//   G = tril(2 L~(t-1) T~),  u_k = V_{.k} / ||V_{.k}||,
//   Vbar_{.k} = (D_k / ||V_{.k}||) (Lbar_{.k} - u_k (u_k . Lbar_{.k}))  for k < N-1, Vbar_{.N} = 0,
//   taubar_t = - sum_{i >= j} Vbar_ij G_ij,
//   dloss/dL~(t-1) = tril(Vbar - tau_t Vbar (2 T~)).
// Neither G nor V is needed in reverse: with T~ symmetric,
//   <Vbar, G> = sum_{i >= k} L~(t-1)_ik P_ik,  P = Vbar (2 T~),
// reads the product that dloss/dL~(t-1) forms anyway (P_NN = sum_j Vbar_Nj 2 T~_jN for the
// constant L~_NN), u_k = L~(t)_{.k} / D_k, and D_k / ||V_{.k}|| is the scale of the forward
// prox.  So a segment costs its c forward steps (recomputed from the checkpoint, iterates and
// scales kept in shared memory) and one product per reverse step, 2 products per iteration
// against 2.75 at c = 4 when V was formed again; Vbar(t) overwrites L~(t).
//
// Mapping as in the FP32 detector: NB / 2 lanes per instance, lane gl owning columns ca = gl
// and cb = NB / 2 + gl of L~, V, Vbar and Lbar (or NB lanes, one column each: UfPlan); its columns
// of T~ stay in registers; rows of L~ and Vbar are broadcast from shared memory (one LDS.128 serves
// both columns of all the warp's instances), and both products keep the triangular skip.  Shared
// memory holds only the lower triangle: row i takes i + 1 floats rounded up to a multiple of 4
// (16-byte rows for the float4 broadcasts), 612 floats at bucket 32 instead of 33 x 36.
// Measured per 8,192, t_max = 10, c = 4 (GPU time), against one column a lane and V formed again in
// reverse: N = 33 forward 143 -> 101 us, adjoint 344 -> 224; N = 17 51 -> 23 and 137 -> 49; N = 9
// 25.8 -> 7.8 and 60 -> 17.6.  At N = 33 both hold 8 warps an SM (255 registers); 10 and 12 warps with
// fewer registers were 3 and 9% slower (forward).  Writing the checkpoints entry by entry from shared memory
// took a sixth of the forward's instructions.
#include <algorithm>
#include <cmath>

#include "common.cuh"

namespace taser {

// Offset (floats) of row i of a packed lower-triangular matrix whose row r holds
// (r + 1) rounded up to 4 floats: with i = 4q + m, 16 q (q + 1) / 2 + 4 m (q + 1).
__host__ __device__ constexpr int tri_off(int i) { return 4 * ((i >> 2) + 1) * (2 * (i >> 2) + (i & 3)); }
// Where the scale of column j is kept inside a packed iterate: floats 2 and 3 of the last quad of
// rows 4q and 4q + 1 (q = j / 4) are padding that no product uses (tri_rows skips that pair).
__device__ __forceinline__ int scale_off(int j) {
  return tri_off(4 * (j >> 2) + ((j >> 1) & 1)) + 4 * (j >> 2) + 2 + (j & 1);
}

// COLS columns a lane: 2, or 1 where too few warps would share an SM (UfPlan).
template <int NB, int COLS>
struct UfCfg {
  static constexpr int HALF = NB / COLS;            // columns ca of the lanes
  static constexpr int FB = COLS == 2 ? HALF : NB + 1;   // first row that a column cb reaches
  static constexpr int G = HALF;                    // lanes of one instance
  static constexpr int IPW = 32 / G;                // instances of a warp
  static constexpr int MAT = tri_off(NB + 1);       // one packed iterate (rows 0..NB)
  static constexpr int NP = NB / 2 + 1;             // pairs (k, k + 1) of a column of T~
  static constexpr int NBV = COLS == 2 ? NB + 1 - FB : 1;   // entries of a column cb
  // Floats between the instances of a warp holding `mats` iterates each: G banks apart.
  __host__ __device__ static constexpr int inst_floats(int mats) {
    return mats * MAT + ((G - mats * MAT % 32) % 32 + 32) % 32;
  }
  // Blocks (warps) per SM that the registers allow.
  static constexpr int FWD_MIN_BLOCKS = COLS == 2 ? (NB == 32 ? 8 : 16) : (NB == 8 ? 16 : 12);
  static constexpr int BWD_MIN_BLOCKS = NB == 32 ? 8 : (NB == 16 && COLS == 1 ? 12 : 16);   // adjoint: one warp per block
};

// What a lane keeps of its instance: columns ca < HALF <= cb and their T~ (COLS = 1: ca only).
template <int NB, int COLS>
struct UfLane {
  using C = UfCfg<NB, COLS>;
  int gl, ca, cb, ra, rb, N;        // ra, rb: real columns (-1: padding)
  uint64_t ta[C::NP], tb[COLS == 2 ? C::NP : 1];   // pairs (T~_kj, T~_k+1,j), k <= NB
  float Da, Db, DN;

  __device__ __forceinline__ UfLane(const float* T, const float* D, bool active, int n, int lane) {
    gl = lane % C::G;
    ca = gl;
    cb = COLS == 2 ? C::HALF + gl : gl;
    N = active ? n : NB + 1;
    ra = ca < N - 1 ? ca : -1;
    rb = COLS == 2 && cb < N - 1 ? cb : -1;
    auto load = [&](int k, int r) -> float {
      const int kr = k <= NB ? bucket_to_real(k, N, NB) : -1;
      return active && kr >= 0 && r >= 0 && TASER_IN(kr * N + r, N * N) ? T[(int64_t)kr * N + r] : 0.f;
    };
#pragma unroll
    for (int p = 0; p < C::NP; ++p) {
      ta[p] = f2pack(load(2 * p, ra), load(2 * p + 1, ra));
      if constexpr (COLS == 2) tb[p] = f2pack(load(2 * p, rb), load(2 * p + 1, rb));
    }
    Da = active && ra >= 0 && TASER_IN(ra, N) ? D[ra] : 0.f;
    Db = active && rb >= 0 && TASER_IN(rb, N) ? D[rb] : 0.f;
    DN = active ? D[N - 1] : 0.f;
  }
};

// f(i, a, b) for the rows i = 0..NB, a = 2 sum_{k <= i} R[i][k] T~_k,ca and (rows >= HALF) b the
// same for cb, R a packed lower-triangular matrix whose row padding within a used pair is zero.
template <int NB, int COLS, class F>
__device__ __forceinline__ void tri_rows(const float* R, const UfLane<NB, COLS>& L, F&& f) {
  constexpr int FB = UfCfg<NB, COLS>::FB;
#pragma unroll
  for (int i = 0; i <= NB; ++i) {
    const float* row = R + tri_off(i);
    uint64_t acca = 0ull, accb = 0ull;
#pragma unroll
    for (int k4 = 0; k4 <= i; k4 += 4) {
      const float4 q = *reinterpret_cast<const float4*>(row + k4);
      const uint64_t q0 = f2pack(q.x, q.y), q1 = f2pack(q.z, q.w);
      acca = k4 == 0 ? f2mul(q0, L.ta[0]) : f2fma(q0, L.ta[k4 / 2], acca);
      if (i >= FB) accb = k4 == 0 ? f2mul(q0, L.tb[0]) : f2fma(q0, L.tb[k4 / 2], accb);
      if (k4 + 2 <= i) {
        acca = f2fma(q1, L.ta[k4 / 2 + 1], acca);
        if (i >= FB) accb = f2fma(q1, L.tb[k4 / 2 + 1], accb);
      }
    }
    float a0, a1, b0, b1;
    f2unpack(acca, a0, a1);
    f2unpack(accb, b0, b1);
    f(i, 2.f * (a0 + a1), 2.f * (b0 + b1));
  }
}

// One forward step on the packed iterate Lin: va (rows 0..NB) and vb (rows HALF..NB) hold its
// columns ca and cb and become those of the next iterate, sa and sb their scales D_k / ||V_{.k}||.
// At bucket 32 the columns are read from Lin again, which frees their registers during the
// products (adjoint 0.256 against 0.283 ms per 8,192).
template <int NB, int COLS>
__device__ __forceinline__ void forward_step(const float* Lin, const UfLane<NB, COLS>& L, float tau, float (&va)[NB + 1],
                                             float (&vb)[UfCfg<NB, COLS>::NBV], float& sa, float& sb) {
  constexpr int HALF = UfCfg<NB, COLS>::HALF, FB = UfCfg<NB, COLS>::FB;
  float na = 0.f, nb = 0.f;
  tri_rows<NB, COLS>(Lin, L, [&](int i, float a, float b) {
    const float la = NB < 32 ? va[i] : Lin[tri_off(i) + (i >= HALF || i >= L.ca ? L.ca : 0)];
    va[i] = (i >= HALF || i >= L.ca) ? fmaf(-tau, a, la) : 0.f;
    if (i >= FB) {
      const float lb = NB < 32 ? vb[i < FB ? 0 : i - FB] : Lin[tri_off(i) + (i >= L.cb ? L.cb : 0)];
      vb[i - FB] = i >= L.cb ? fmaf(-tau, b, lb) : 0.f;
    }
  });
#pragma unroll
  for (int i = 0; i <= NB; ++i) {
    na = fmaf(va[i], va[i], na);
    if (i >= FB) nb = fmaf(vb[i - FB], vb[i - FB], nb);
  }
  sa = na > 0.f ? L.Da * rsqrtf(na) : 0.f;
  sb = nb > 0.f ? L.Db * rsqrtf(nb) : 0.f;
#pragma unroll
  for (int i = 0; i <= NB; ++i) {
    va[i] *= sa;
    if (i >= FB) vb[i - FB] *= sb;
  }
}

// Columns ca and cb into a packed matrix (on and below the diagonal).
template <int NB, int COLS>
__device__ __forceinline__ void put_columns(float* M, const UfLane<NB, COLS>& L, const float (&va)[NB + 1],
                                            const float (&vb)[UfCfg<NB, COLS>::NBV], bool own) {
  constexpr int HALF = UfCfg<NB, COLS>::HALF, FB = UfCfg<NB, COLS>::FB;
#pragma unroll
  for (int i = 0; i <= NB; ++i) {
    if (own && (i >= HALF || i >= L.ca)) M[tri_off(i) + L.ca] = va[i];
    if (i >= FB && own && i >= L.cb) M[tri_off(i) + L.cb] = vb[i - FB];
  }
}

// A checkpoint (full N x N in real indices, zeros above the diagonal) from and to the lanes'
// columns: a row of an instance is 2 runs of NB / 2 floats and column N.
template <int NB, int COLS>
__device__ __forceinline__ void store_ckpt(float* out, const UfLane<NB, COLS>& L, const float (&va)[NB + 1],
                                           const float (&vb)[UfCfg<NB, COLS>::NBV]) {
  constexpr int FB = UfCfg<NB, COLS>::FB;
  const int N = L.N;
#pragma unroll
  for (int i = 0; i <= NB; ++i) {
    const int ir = bucket_to_real(i, N, NB);
    if (ir < 0) continue;
    float* row = out + ir * N;
    if (L.ra >= 0 && TASER_IN(ir * N + L.ra, N * N)) row[L.ra] = va[i];
    if (L.rb >= 0 && TASER_IN(ir * N + L.rb, N * N)) row[L.rb] = i < FB ? 0.f : vb[i < FB ? 0 : i - FB];
    if (L.gl == 0 && TASER_IN(ir * N + N - 1, N * N)) row[N - 1] = i == NB ? L.DN : 0.f;
  }
}
template <int NB, int COLS>
__device__ __forceinline__ void load_ckpt(const float* in, const UfLane<NB, COLS>& L, float (&va)[NB + 1],
                                          float (&vb)[UfCfg<NB, COLS>::NBV]) {
  constexpr int HALF = UfCfg<NB, COLS>::HALF, FB = UfCfg<NB, COLS>::FB;
  const int N = L.N;
#pragma unroll
  for (int i = 0; i <= NB; ++i) {
    const int ir = bucket_to_real(i, N, NB);
    const float* row = in + ir * N;
    va[i] = ir >= 0 && L.ra >= 0 && (i >= HALF || i >= L.ca) && TASER_IN(ir * N + L.ra, N * N) ? row[L.ra] : 0.f;
    if (i >= FB)
      vb[i - FB] = ir >= 0 && L.rb >= 0 && i >= L.cb && TASER_IN(ir * N + L.rb, N * N) ? row[L.rb] : 0.f;
  }
}

// Power of two 2^e by which the adjoint multiplies the incoming gradient, and divides its result
// again (the adjoint is linear, so both are exact).  u (u . Lbar) is formed as L~ (L~ . Lbar) / D^2
// with Lbar of the order g / D, which leaves FP32's range although the result does not: e is the
// exponent of the smallest D below 2^-40, or of the largest above 2^40, and 0 in between.
template <int G>
__device__ __forceinline__ int grad_exponent(float Da, float Db) {
  float lo = fminf(Da > 0.f ? Da : 1.f, Db > 0.f ? Db : 1.f), hi = fmaxf(Da, Db);
#pragma unroll
  for (int o = G / 2; o > 0; o >>= 1) {
    lo = fminf(lo, __shfl_xor_sync(TASER_FULL_MASK, lo, o));
    hi = fmaxf(hi, __shfl_xor_sync(TASER_FULL_MASK, hi, o));
  }
  const float D = lo < 0x1p-40f ? lo : (hi > 0x1p40f ? hi : 1.f);
  return min(max((int)(__float_as_uint(D) >> 23) - 127, -126), 126);
}
__device__ __forceinline__ float pow2f(int e) { return __uint_as_float((uint32_t)(e + 127) << 23); }

template <int NB, int COLS>
__global__ void __launch_bounds__(32, UfCfg<NB, COLS>::FWD_MIN_BLOCKS)
unfolded_forward_kernel(int64_t batch, int N, const float* __restrict__ Tt, const float* __restrict__ Dg,
                        const float* __restrict__ inv_norm, const float* __restrict__ alpha_t, int t_max, int c,
                        float* __restrict__ ckpt, float* __restrict__ soft, int8_t* __restrict__ s_hat) {
  using C = UfCfg<NB, COLS>;
  constexpr int FB = C::FB, STRIDE = C::inst_floats(1);
  extern __shared__ __align__(16) float smem[];
  const int lane = threadIdx.x;
  const int64_t inst = (int64_t)blockIdx.x * C::IPW + lane / C::G;
  const bool active = inst < batch;
  float* const cur = smem + (lane / C::G) * STRIDE;
  const int64_t at = active ? inst : 0;
  const UfLane<NB, COLS> L(Tt + at * N * N, Dg + at * N, active, N, lane);
  const float inv = active ? inv_norm[inst] : 0.f;
  const int n_ckpt = (t_max + c - 1) / c;
  float va[NB + 1], vb[C::NBV];                // columns of the iterate
#pragma unroll
  for (int i = 0; i <= NB; ++i) {
    va[i] = i == L.ca ? L.Da : 0.f;
    if (i >= FB) vb[i - FB] = i == L.cb ? L.Db : 0.f;
  }
  for (int idx = lane; idx < C::IPW * STRIDE; idx += 32) smem[idx] = 0.f;
  __syncwarp();
  put_columns<NB, COLS>(cur, L, va, vb, true);
  if (L.gl == 0) cur[tri_off(NB) + NB] = L.DN;
  __syncwarp();
  for (int t = 0; t < t_max; ++t) {
    if (t % c == 0 && ckpt != nullptr && active && TASER_IN(inst * n_ckpt + t / c, batch * n_ckpt))
      store_ckpt<NB, COLS>(ckpt + (inst * n_ckpt + t / c) * (int64_t)N * N, L, va, vb);
    const float tau = TASER_IN(t, t_max) ? alpha_t[t] * inv : 0.f;
    float sa, sb;
    forward_step<NB, COLS>(cur, L, tau, va, vb, sa, sb);
    __syncwarp();   // every lane has read L~(t)
    put_columns<NB, COLS>(cur, L, va, vb, true);
    __syncwarp();
  }
  auto emit = [&](int r, float D, float x) {
    if (!active || r < 0 || !TASER_IN(inst * (N - 1) + r, batch * (N - 1))) return;
    const float y = D > 0.f ? x / D : 0.f;
    soft[inst * (N - 1) + r] = y;
    TASER_FINITE(y);
    if (s_hat != nullptr) s_hat[inst * (N - 1) + r] = x >= 0.f ? int8_t(1) : int8_t(-1);
  };
  emit(L.ra, L.Da, va[NB]);
  if constexpr (COLS == 2) emit(L.rb, L.Db, vb[NB - FB]);
}

// One warp per block, `ipw` instances on it: C::IPW, or fewer (a power of two) where the c + 1
// iterates of each fill the shared memory (UfPlan); the lanes of the other groups then follow
// the first one's data and store nothing.
template <int NB, int COLS>
__global__ void __launch_bounds__(32, UfCfg<NB, COLS>::BWD_MIN_BLOCKS)
unfolded_backward_kernel(int64_t batch, int N, const float* __restrict__ Tt, const float* __restrict__ Dg,
                         const float* __restrict__ inv_norm, const float* __restrict__ alpha_t, int t_max, int c,
                         int ipw, const float* __restrict__ ckpt, const float* __restrict__ grad_soft,
                         float* __restrict__ grad_tau) {
  using C = UfCfg<NB, COLS>;
  constexpr int HALF = C::HALF, FB = C::FB;
  extern __shared__ __align__(16) float smem[];
  const int lane = threadIdx.x;
  const int stride = C::inst_floats(c + 1);
  const int64_t first = (int64_t)blockIdx.x * ipw;
  const int grp = lane / C::G;
  const bool own = grp < ipw;                         // this group has shared memory
  const int64_t inst = first + grp;
  const bool active = own && inst < batch;
  float* const seg = smem + (own ? grp : 0) * stride;   // iterates L~(t0) .. L~(t1); Vbar replaces them
  const int64_t at = active ? inst : 0;
  const UfLane<NB, COLS> L(Tt + at * N * N, Dg + at * N, active, N, lane);
  const float inv = active ? inv_norm[inst] : 0.f;
  const float rDa = L.Da > 0.f ? 1.f / L.Da : 0.f, rDb = L.Db > 0.f ? 1.f / L.Db : 0.f;
  float tNa, tNb, unused;                             // T~_N,ca and T~_N,cb
  f2unpack(L.ta[C::NP - 1], tNa, unused);
  f2unpack(L.tb[COLS == 2 ? C::NP - 1 : 0], tNb, unused);
  for (int idx = lane; idx < ipw * stride; idx += 32) smem[idx] = 0.f;
  const int n_ckpt = (t_max + c - 1) / c;
  // Lbar(t_max): only the last row, dloss/dL~_{N,k} = dloss/dx_k / D_k (times 2^e)
  const int e = grad_exponent<C::G>(L.Da, L.Db);
  float la[NB + 1], lb[C::NBV];
#pragma unroll
  for (int i = 0; i <= NB; ++i) {
    la[i] = 0.f;
    if (i >= FB) lb[i - FB] = 0.f;
  }
  if (L.ra >= 0 && L.Da > 0.f && TASER_IN(inst * (N - 1) + L.ra, batch * (N - 1)))
    la[NB] = grad_soft[inst * (N - 1) + L.ra] * pow2f(e) / L.Da;
  if (COLS == 2 && L.rb >= 0 && L.Db > 0.f && TASER_IN(inst * (N - 1) + L.rb, batch * (N - 1)))
    lb[C::NBV - 1] = grad_soft[inst * (N - 1) + L.rb] * pow2f(e) / L.Db;
  __syncwarp();

  for (int kc = n_ckpt - 1; kc >= 0; --kc) {
    const int t0 = kc * c, t1 = min(t0 + c, t_max);
    // L~(t0) from the checkpoint into seg[0] (all loads in flight together), then L~(t0+1) ..
    // L~(t1) and their scales.
    float va[NB + 1], vb[C::NBV], sa, sb;
    if (active && TASER_IN(inst * n_ckpt + kc, batch * n_ckpt)) {
      load_ckpt<NB, COLS>(ckpt + (inst * n_ckpt + kc) * (int64_t)N * N, L, va, vb);
    } else {
#pragma unroll
      for (int i = 0; i <= NB; ++i) {
        va[i] = 0.f;
        if (i >= FB) vb[i - FB] = 0.f;
      }
    }
    put_columns<NB, COLS>(seg, L, va, vb, own);
    if (own && L.gl == 0) seg[tri_off(NB) + NB] = L.DN;
    __syncwarp();
#pragma unroll 1
    for (int s = t0 + 1; s <= t1; ++s) {
      const float* Lin = seg + (s - 1 - t0) * C::MAT;
      float* Lout = seg + (TASER_IN(s - t0, c + 1) ? s - t0 : 0) * C::MAT;
      forward_step<NB, COLS>(Lin, L, alpha_t[s - 1] * inv, va, vb, sa, sb);
      put_columns<NB, COLS>(Lout, L, va, vb, own);
      if (own) {
        Lout[scale_off(L.ca)] = sa;
        if (COLS == 2) Lout[scale_off(L.cb)] = sb;
        if (L.gl == 0) Lout[tri_off(NB) + NB] = L.DN;
      }
      __syncwarp();
    }
    // reverse through steps t1 .. t0+1 (step s maps L~(s-1) -> L~(s), uses tau_s)
#pragma unroll 1
    for (int s = t1; s > t0; --s) {
      const float* Lin = seg + (s - 1 - t0) * C::MAT;
      float* Ls = seg + (s - t0) * C::MAT;
      const float tau = alpha_t[s - 1] * inv;
      // Vbar = f (Lbar - u (u . Lbar)), u = L~(s) / D, f the prox scale; it overwrites Lbar and,
      // in shared memory, L~(s).
      float pa = 0.f, pb = 0.f;
#pragma unroll
      for (int i = 0; i <= NB; ++i) {
        pa = fmaf((i >= HALF || i >= L.ca) ? Ls[tri_off(i) + (i >= HALF || i >= L.ca ? L.ca : 0)] : 0.f, la[i], pa);
        if (i >= FB) pb = fmaf(i >= L.cb ? Ls[tri_off(i) + (i >= L.cb ? L.cb : 0)] : 0.f, lb[i - FB], pb);
      }
      pa = pa * rDa * rDa;   // in this order: 1 / D^2 by itself overflows below D = 2^-64
      pb = pb * rDb * rDb;
      const float fa = Ls[scale_off(L.ca)], fb = Ls[scale_off(L.cb)];
#pragma unroll
      for (int i = 0; i <= NB; ++i) {
        if (i >= HALF || i >= L.ca) la[i] = fa * fmaf(-Ls[tri_off(i) + L.ca], pa, la[i]);
        if (i >= FB && i >= L.cb) lb[i - FB] = fb * fmaf(-Ls[tri_off(i) + L.cb], pb, lb[i - FB]);
      }
      put_columns<NB, COLS>(Ls, L, la, lb, own);
      if (own && L.gl == 0) Ls[tri_off(NB) + NB] = 0.f;   // column N of Vbar is zero
      __syncwarp();
      // P = Vbar (2 T~);  <Vbar, G> = <L~(s-1), P>;  Lbar(s-1) = tril(Vbar - tau P)
      float ga = L.DN * 2.f * __fmul_rn(la[NB], tNa), gb = 0.f;   // by column
      if constexpr (COLS == 2) gb = L.DN * 2.f * __fmul_rn(lb[NB - FB], tNb);
      tri_rows<NB, COLS>(Ls, L, [&](int i, float a, float b) {
        if (i >= HALF || i >= L.ca) {
          ga = fmaf(Lin[tri_off(i) + L.ca], a, ga);
          la[i] = fmaf(-tau, a, la[i]);
        }
        if (i >= FB && i >= L.cb) {
          gb = fmaf(Lin[tri_off(i) + L.cb], b, gb);
          lb[i - FB] = fmaf(-tau, b, lb[i - FB]);
        }
      });
      const float tb = column_total<NB, COLS>(column_halves<NB, COLS>(ga, gb, L.gl, lane));
      if (active && L.gl == 0 && TASER_IN(inst * t_max + (s - 1), batch * t_max)) {
        grad_tau[inst * t_max + (s - 1)] = -tb * pow2f(-e);
        TASER_FINITE(tb);
      }
      __syncwarp();
    }
  }
}

// grad_alpha[t] = sum_n grad_tau[n][t] * inv_norm[n], one block per t, fixed-order tree.
__global__ void reduce_alpha_kernel(int64_t batch, int t_max, const float* __restrict__ grad_tau,
                                     const float* __restrict__ inv_norm, float* __restrict__ grad_alpha) {
  __shared__ float part[256];
  const int t = blockIdx.x;
  float acc = 0.f;
  for (int64_t n = threadIdx.x; n < batch; n += blockDim.x) acc = fmaf(grad_tau[n * t_max + t], inv_norm[n], acc);
  part[threadIdx.x] = acc;
  __syncthreads();
  for (int s = blockDim.x / 2; s > 0; s >>= 1) {
    if (threadIdx.x < s) part[threadIdx.x] += part[threadIdx.x + s];
    __syncthreads();
  }
  if (threadIdx.x == 0) grad_alpha[t] = part[0];
}

// Layout of a launch: columns a lane and, for the adjoint, instances a warp.  Two columns a lane do
// more per instruction, but a warp's chain of an iteration is longer, which nothing hides where few
// warps share an SM: in small batches, and in the adjoint where the iterates of a wide spacing fill
// the shared memory.  The layout with the smallest estimate is taken, in units of a one-column
// warp's chain, p instances an SM on W warps of n each:
//   chain x max(1, 0.12 ceil(p / n))                    while they fit at once (p <= W n),
//   chain x (max(1, 0.12 W) p / (W n) + 0.4)            in turns, the last one half empty,
// the chain of two columns 1.45 / 1.6 / 1.3 at NB = 8 / 16 / 32.  The constants are a fit to 591 pairs
// of times (N = 9 to 33, 64 to 20,000 instances, c = 1 to 200): the layout taken is on average 0.2%
// slower than the better one, at most 15%.
// Adjoint, one column / two: 512 instances of N = 33, c = 4, t_max = 10 35.9 / 45.5 us, 1,024 44.5 /
// 45.3, 2,048 86.7 / 65.0; of N = 17 1,024 17.2 / 24.3, 4,096 38.9 / 31.0; 4,096 of N = 33 with t_max =
// c = 5 87 / 67, 6 99 / 94, 8 125 / 130, 16 299 / 515, 24 600 / 762; of N = 17 with 8 32 / 25, 12 45 / 50,
// 48 289 / 415.  Forward: 512 of N = 17 7.7 / 10.9, 2,048 9.6 / 11.3, 4,096 15.4 / 14.1.
struct UfPlan {
  double cost = 1e300;
  bool two = false;
  int ipw = 0;
  size_t smem = 0;

  template <int NB, int COLS>
  void consider(bool backward, double per_sm, int c) {
    using C = UfCfg<NB, COLS>;
    constexpr double chain = COLS == 1 ? 1.0 : (NB == 32 ? 1.3 : (NB == 16 ? 1.6 : 1.45));
    for (int n = C::IPW; n >= 1; n /= 2) {
      const size_t bytes = (size_t)n * C::inst_floats(backward ? c + 1 : 1) * sizeof(float);
      if (bytes <= kMaxSmem) {
        const int fit = (int)((size_t)228 * 1024 / (bytes + 1024));   // an SM's memory; 1 KB a block is reserved
        const int warps = std::min(fit, backward ? C::BWD_MIN_BLOCKS : C::FWD_MIN_BLOCKS);
        const double turns = per_sm / (warps * n);
        const double t = chain * (turns <= 1.0 ? std::max(1.0, 0.12 * std::ceil(per_sm / n))
                                               : std::max(1.0, 0.12 * warps) * turns + 0.4);
        if (t < cost) {
          cost = t;
          two = COLS == 2;
          ipw = n;
          smem = bytes;
        }
      }
      if (!backward) break;   // the forward holds one iterate an instance: whole warps always fit
    }
  }
};

template <int NB, int COLS>
static cudaError_t launch_cols(const UfPlan& plan, bool backward, int64_t batch, int N, const float* Tt, const float* D,
                               const float* inv_norm, const float* alpha_t, int t_max, int c, float* ckpt,
                               float* soft, int8_t* s_hat, const float* grad_soft, float* grad_tau,
                               cudaStream_t st) {
  const int64_t blocks = (batch + plan.ipw - 1) / plan.ipw;   // one warp each
  if (!backward) {
    static_assert(UfCfg<NB, COLS>::IPW * UfCfg<NB, COLS>::inst_floats(1) * 4 <= 48 * 1024,
                  "above 48 KB a kernel must opt in");
    unfolded_forward_kernel<NB, COLS><<<(unsigned)blocks, 32, plan.smem, st>>>(batch, N, Tt, D, inv_norm, alpha_t,
                                                                              t_max, c, ckpt, soft, s_hat);
  } else {
    const cudaError_t e = allow_smem(unfolded_backward_kernel<NB, COLS>);
    if (e != cudaSuccess) return e;
    unfolded_backward_kernel<NB, COLS><<<(unsigned)blocks, 32, plan.smem, st>>>(
        batch, N, Tt, D, inv_norm, alpha_t, t_max, c, plan.ipw, ckpt, grad_soft, grad_tau);
  }
  return cudaGetLastError();
}

template <int NB>
static cudaError_t launch_unfolded(bool backward, int64_t batch, int N, const float* Tt, const float* D,
                                   const float* inv_norm, const float* alpha_t, int t_max, int c, float* ckpt,
                                   float* soft, int8_t* s_hat, const float* grad_soft, float* grad_tau,
                                   cudaStream_t st) {
  int dev = 0, sms = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  if (e != cudaSuccess) return e;
  UfPlan plan;
  plan.consider<NB, 2>(backward, (double)batch / sms, c);
  plan.consider<NB, 1>(backward, (double)batch / sms, c);
  if (plan.ipw == 0) return cudaErrorInvalidValue;
  if (plan.two)
    return launch_cols<NB, 2>(plan, backward, batch, N, Tt, D, inv_norm, alpha_t, t_max, c, ckpt, soft, s_hat,
                              grad_soft, grad_tau, st);
  return launch_cols<NB, 1>(plan, backward, batch, N, Tt, D, inv_norm, alpha_t, t_max, c, ckpt, soft, s_hat, grad_soft,
                            grad_tau, st);
}

// Bound on checkpoint spacing c at size N: the shared memory (bytes) of c + 2 iterates of one
// instance (the kernel holds c + 1 of them, aligned).
size_t unfolded_backward_smem(int N, int c) {
  const int NB = bucket_of(N);
  return (size_t)(c + 2) * tri_off(NB + 1) * sizeof(float);
}

cudaError_t unfolded_tc(bool backward, bool fp16, int64_t batch, int N, const float* Tt, const float* D,
                        const float* inv_norm, const float* alpha_t, int t_max, int c, float* ckpt, float* soft,
                        int8_t* s_hat, const float* grad_soft, float* grad_tau, cudaStream_t st);

// precision: TASER_FP32, or TASER_BF16_TC / TASER_FP16_TC (tensor-core kernels for bucket 32;
// smaller N runs the FP32 kernels).
cudaError_t unfolded(bool backward, int precision, int64_t batch, int N, const float* Tt, const float* D,
                     const float* inv_norm, const float* alpha_t, int t_max, int c, float* ckpt, float* soft,
                     int8_t* s_hat, const float* grad_soft, float* grad_tau, float* grad_alpha, cudaStream_t st) {
  cudaError_t e;
  const bool tc = precision != TASER_FP32 && bucket_of(N) == 32;
  switch (tc ? -1 : bucket_of(N)) {
    case -1:
      e = unfolded_tc(backward, precision == TASER_FP16_TC, batch, N, Tt, D, inv_norm, alpha_t, t_max, c, ckpt, soft,
                      s_hat, grad_soft, grad_tau, st);
      break;
    case 8:
      e = launch_unfolded<8>(backward, batch, N, Tt, D, inv_norm, alpha_t, t_max, c, ckpt, soft, s_hat, grad_soft,
                             grad_tau, st);
      break;
    case 16:
      e = launch_unfolded<16>(backward, batch, N, Tt, D, inv_norm, alpha_t, t_max, c, ckpt, soft, s_hat, grad_soft,
                              grad_tau, st);
      break;
    case 32:
      e = launch_unfolded<32>(backward, batch, N, Tt, D, inv_norm, alpha_t, t_max, c, ckpt, soft, s_hat, grad_soft,
                              grad_tau, st);
      break;
    default:
      return cudaErrorNotSupported;
  }
  if (e != cudaSuccess || !backward || grad_alpha == nullptr) return e;
  reduce_alpha_kernel<<<t_max, 256, 0, st>>>(batch, t_max, grad_tau, inv_norm, grad_alpha);
  return cudaGetLastError();
}

}  // namespace taser

TASER_DEBUG_COLLECTOR(unfolded)
