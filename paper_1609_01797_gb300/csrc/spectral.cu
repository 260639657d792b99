// ||T~||_2 and the step size tau = alpha / ||T~||_2 (Sec. III-B; inputs of Algorithm 1).
//
// ||T~||_2 of a symmetric matrix is its largest |eigenvalue|.  A power iteration is not
// used: on MU-MIMO matrices the two largest eigenvalues are often close and hundreds of
// steps still leave errors of 1e-3.  Instead each T~ is reduced to tridiagonal form with
// Householder reflections (FP32, backward stable), and the extreme eigenvalues of the
// tridiagonal matrix are found by Sturm-count multisection.  When T~ is known to be
// semidefinite (MU-MIMO: T = A^T A; JED: T = -A^T A) only that end is searched; otherwise
// lambda_max(T~) and lambda_max(-T~) are bracketed side by side.
//
// Layout: T~ is embedded in an (NV+1) x (NV+1) matrix with zero padding (zero rows and
// columns add zero eigenvalues, which do not change ||T~||_2 since ||T~||_2 >= 0).  The
// first reflection eliminates column 0, leaving an NV x NV trailing matrix whose columns
// 1..NV live in lane registers:
//  - spectral_fold_kernel (real): NV / 2 lanes per instance, two columns a lane (c and
//    NV + 1 - c), as packed pairs of rows (A[2p][c], A[2p+1][c]): one 16-byte read of a published
//    vector feeds four rows of both columns;
//  - spectral_herm_kernel (QPSK complex form): two columns a lane for NV <= 16, one at 24 and 32, as
//    {re, im} pairs (row pairs need 12 instead of 8 registers of duplicated factors a column and
//    were slower: 0.165 against 0.139 ms per 65,536 QPSK 128x16).
//
// A Householder step is a chain: norm of the column (shuffles), reflector scalars, publish v,
// p = beta A v, v^H p (shuffles), rank-2 update.  p is published before v^H p is known: with
// kk = beta v^H p (real), A - v w^H - w v^H = A - v (p - kk v)^H - p v^H, whose own-column
// factor alone needs kk, so its shuffles overlap the reads.  (Updating the next step's column
// by itself before the rest, so that its norm overlaps the update too, cost more instructions
// than it hid: 1.7% slower at N = 32, 0.7% for QPSK 128x16.)
#include <type_traits>

#include "common.cuh"

namespace taser {

// Householder steps per compiled block (a fully unrolled body misses the instruction cache; the
// longer a block, the more finished rows its steps carry along).  Measured: real NV = 64 4 beats 2
// by 6%, NV <= 32 2 beats 4 by 1 to 3%; complex UV <= 16 2 beats 4 by 2%.
template <int NV>
__host__ __device__ constexpr int real_block() { return NV == 64 ? 4 : 2; }
template <int UV>
__host__ __device__ constexpr int herm_block() { return UV >= 24 ? 4 : 2; }

// Calls f(std::integral_constant<int, KB>) for KB = 0, BLK, 2 BLK, ... < NV - 1.
template <int NV, int BLK, int KB = 0, typename F>
__device__ __forceinline__ void static_for_blocks(F&& f) {
  if constexpr (KB < NV - 1) {
    f(std::integral_constant<int, KB>{});
    static_for_blocks<NV, BLK, KB + BLK>(f);
  }
}

// Exponent e with 2^e <= m < 2^(e+1), clamped to [-126, 126] (0 for zero or non-finite m):
// the matrix is scaled by 2^-e (exact, both factors normal floats) so its largest entry
// lies in [1, 4) and tiny reflector norms are judged against that scale; ||T~|| is scaled
// back by 2^e.
__device__ __forceinline__ int scale_exponent(float m) {
  if (!(m > 0.f) || !(m <= 3.0e38f)) return 0;
  const int e = (int)((__float_as_uint(m) >> 23) & 0xffu) - 127;
  return e < -126 ? -126 : (e > 126 ? 126 : e);
}
__device__ __forceinline__ float pow2f(int e) { return __uint_as_float((uint32_t)(e + 127) << 23); }

// An int known at compile time, usable where a runtime int is expected.
template <int V>
struct SpecInt {
  __host__ __device__ constexpr operator int() const { return V; }
};

// Below this squared norm (relative to the scaled matrix, largest entry about 1) the
// column is already eliminated: the rest is rounding residue far under FP32's resolution.
constexpr float kTinyNorm2 = 0x1p-100f;

// Hardware reciprocal and reciprocal square root without the range handling of __fdividef and
// rsqrtf: every argument here is normal (at least kTinyNorm2 in the reflectors) or may count as
// zero (a pivot).  With the fused subtraction of the Sturm recurrence a step
// of it is about 5 instructions instead of 10: JED BPSK K = 32 780 -> 655 us per 131,072, QPSK
// 128x16 149 -> 132 us per 65,536, N = 65 (either sign) 340 -> 285 us per 8,192.
__device__ __forceinline__ float rcp_fast(float x) {
  float r;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
  return r;
}
__device__ __forceinline__ float rsqrt_fast(float x) {
  float r;
  asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
  return r;
}

// Sturm count: number of eigenvalues of the tridiagonal (sg*d, e) below sigma, as the
// number of negative pivots q_j of the LDL^T factorisation of (sg*T - sigma I).  No pivot
// guard sits in the recurrence: IEEE infinities carry a zero pivot through (Demmel, Dhillon
// and Ren, 1995).  A pivot +0 yields -inf next (counted), -0 yields +inf, and the pivot
// after an infinite one is finite again.  (rcp_fast flushes a denormal pivot to a zero of its sign,
// which is such a pivot.)  This needs e2 > 0 throughout (0 * inf would be a
// NaN), so callers floor the squared off-diagonals at kTinyNorm2.  The count reads the sign
// bit, so -0 counts as negative and +0 does not, matching the infinities they produce.
template <int NP>
__device__ __forceinline__ int sturm_count(const float (&d)[NP], const float (&e2)[NP], float sg, float sigma) {
  float q = sg * d[0] - sigma;
  int cnt = (int)(__float_as_uint(q) >> 31);
#pragma unroll
  for (int j = 1; j < NP; ++j) {
    q = fmaf(-e2[j - 1], rcp_fast(q), sg * d[j] - sigma);
    cnt += (int)(__float_as_uint(q) >> 31);
  }
  return cnt;
}

// sign_hint: +1 -> T~ is positive semidefinite (||T~|| = lambda_max), -1 -> negative
// semidefinite (||T~|| = lambda_max(-T~)), 0 -> unknown (both ends are searched).
//
// Lane gl < NV / 2 of an instance's G (the next power of two) holds columns ca = gl + 1 (1..NV/2)
// and cb = NV - gl.  From step NV / 2 on every ca column is finished, and those blocks drop it at
// compile time.
// Multisection: one-sided, each lane evaluates two of 2 G points (2 G + 1 parts); two-sided, one
// point on each side (G + 1 parts a side).  The parts stand beside ROUNDS1 and ROUNDS2; FP32's own
// spacing limits the result from about 2^24 = 1.7e7 on (300 tridiagonal matrices of order 65 on the
// CPU: mean error 4.6e-8 and largest 9.5e-8 with 1.8e7 parts and with 4.1e8).
// Measured per 131,072 JED BPSK matrices (B = 16), against pairs of columns {A[j][ca], A[j][cb]}
// (a 16-byte read for two rows, finished columns updated with zeros): K = 32 940 -> 780 us,
// K = 16 184 -> 171; per 20,000 BPSK matrices of N = 33 with the build 255 -> 226 us.  At NV = 32
// the 128-register bound spills a little; 168 registers and 3 blocks per SM were not faster.
template <int NV>
struct SpecFoldCfg {
  static constexpr int HALF = NV / 2;
  static constexpr int G = HALF <= 4 ? 4 : (HALF <= 8 ? 8 : (HALF <= 16 ? 16 : 32));   // lanes, HALF at work
  static constexpr int IPW = 32 / G;              // instances per warp
  static constexpr int NP = NV + 1;               // padded order
  static constexpr int P = NV / 2 + 1;            // row pairs
  static constexpr int VB = (2 * P + 3) & ~3;     // vector length, whole 16-byte quads
  static constexpr int WARPS = 4;
  static constexpr int IPC = WARPS * IPW;
  // v, p, d, e; the odd quad keeps the instances of a warp in different banks.
  static constexpr int INST_FLOATS = 4 * VB + 4;
  // Resolution (parts^rounds) of the one-sided search: 65^4 = 1.8e7, 33^5 = 3.9e7, 17^6 = 2.4e7,
  // 9^8 = 4.3e7; of the two-sided one: 33^5 = 3.9e7, 17^7 = 4.1e8, 9^9 = 3.9e8, 5^12 = 2.4e8.
  static constexpr int ROUNDS1 = G == 32 ? 4 : (G == 16 ? 5 : (G == 8 ? 6 : 8));
  static constexpr int ROUNDS2 = G == 32 ? 5 : (G == 16 ? 7 : (G == 8 ? 9 : 12));
};

// The row r (of rows FROM..TO, known at run time) of a column held as row pairs.
template <int FROM, int TO, int P>
__device__ __forceinline__ float pick_row(const uint64_t (&a)[P], int r) {
  float v = 0.f;
#pragma unroll
  for (int i = FROM; i <= TO; ++i) {
    float lo, hi;
    f2unpack(a[i / 2], lo, hi);
    v = r == i ? (i & 1 ? hi : lo) : v;
  }
  return v;
}

// MINB blocks per SM: 4 at NV = 32, 5 at 24, 6 below (131,072 JED bursts of K = 16, with the build,
// 302 -> 290 us).  At NV = 64 the lane's two columns are 132 registers: 3 blocks of 168 registers
// serve large batches (1.27 -> 1.16 ms per 30,000 at N = 65), 2 blocks without spills the batches that
// fit the GPU at once (49 against 56 us for 100 matrices).
template <int NV, int MINB>
__global__ void __launch_bounds__(128, MINB)
spectral_fold_kernel(int64_t batch, int N, const float* __restrict__ Tt, float alpha, int sign_hint,
                     float* __restrict__ tau, float* __restrict__ nrm_out) {
  using C = SpecFoldCfg<NV>;
  constexpr int NP = C::NP, VB = C::VB, G = C::G, HALF = C::HALF, P = C::P;
  constexpr int KBLK = real_block<NV>();
  static_assert(HALF % KBLK == 0, "a Householder block must not straddle step NV / 2");
  __shared__ __align__(16) float sm[C::IPC * C::INST_FLOATS];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int grp = lane / G, gl = lane % G;
  const int local = warp * C::IPW + grp;
  const int64_t inst = (int64_t)blockIdx.x * C::IPC + local;
  const bool active = inst < batch;
  float* vs = sm + local * C::INST_FLOATS;
  float* ps = vs + VB;
  float* db = ps + VB;
  float* eb = db + VB;
  // A lane not at work takes "column 0", which no step k >= 0 has live: its v and p are zero.
  const bool at_work = G == HALF || gl < HALF;
  const int ca = at_work ? gl + 1 : 0, cb = at_work ? NV - gl : 0;
  const float* T = Tt + (active ? inst : 0) * (int64_t)N * N;
  auto a_rc = [&](int r, int c) -> float {
    return active && r < N && c < N && TASER_IN(inst * N * N + r * N + c, batch * N * N) ? T[(int64_t)r * N + c] : 0.f;
  };
  uint64_t A[P], B[P];   // columns ca and cb
  float d0 = a_rc(0, 0), amax = fabsf(d0);
#pragma unroll
  for (int p = 0; p < P; ++p) {
    const float a0 = a_rc(2 * p, ca), a1 = a_rc(2 * p + 1, ca), b0 = a_rc(2 * p, cb), b1 = a_rc(2 * p + 1, cb);
    amax = fmaxf(fmaxf(amax, fmaxf(fabsf(a0), fabsf(a1))), fmaxf(fabsf(b0), fabsf(b1)));
    A[p] = f2pack(a0, a1);
    B[p] = f2pack(b0, b1);
  }
#pragma unroll
  for (int o = G / 2; o > 0; o >>= 1) amax = fmaxf(amax, __shfl_xor_sync(TASER_FULL_MASK, amax, o));
  const int ex = scale_exponent(amax);
  {
    const float sc = pow2f(-ex);
    const uint64_t sc2 = f2pack(sc, sc);
    d0 *= sc;
#pragma unroll
    for (int p = 0; p < P; ++p) {
      A[p] = f2mul(A[p], sc2);
      B[p] = f2mul(B[p], sc2);
    }
  }
  for (int i = gl; i < 2 * VB; i += G) vs[i] = 0.f;
  if (gl == 0) db[0] = d0;
  // x = row k of the lane's columns (A symmetric: the entries x_c of column k), k = 0.
  float xA = pick_row<0, 0>(A, 0), xB = pick_row<0, 0>(B, 0);
  __syncwarp();

  static_for_blocks<NV, KBLK>([&](auto kb) {
    constexpr int KB = decltype(kb)::value;
    constexpr int KE = (KB + KBLK < NV - 1) ? KB + KBLK : NV - 1;   // k in [KB, KE)
    constexpr bool LIVE_A = KB < HALF;   // k < NV / 2 throughout the block: some ca > k
    constexpr int P0 = (KB + 1) / 2;     // first row pair that v reaches
    if constexpr (KB == HALF) {          // the ca columns are finished
      if (TASER_IN(ca, VB)) vs[ca] = ps[ca] = 0.f;
      __syncwarp();
    }
#pragma unroll 1
    for (int k = KB; k < KE; ++k) {
      const bool liveA = LIVE_A && ca > k, liveB = cb > k;
      float sig2 = (liveA ? xA * xA : 0.f) + (liveB ? xB * xB : 0.f);
#pragma unroll
      for (int o = G / 2; o > 0; o >>= 1) sig2 += __shfl_xor_sync(TASER_FULL_MASK, sig2, o);
      // x_{k+1}: column k + 1 is ca of lane k (k < NV / 2) or cb of lane NV - 1 - k.
      const float x1 = __shfl_sync(TASER_FULL_MASK, LIVE_A ? xA : xB, grp * G + (LIVE_A ? k : NV - 1 - k));
      // Reflector H = I - beta v v^T, v = x - ah e_{k+1}, ah = -sign(x_{k+1}) ||x||, from a
      // reciprocal square root (a few ulp; the reflection stays orthogonal to that order).  A
      // column with ||x||^2 under kTinyNorm2 is left as it is (beta = 0).
      const bool refl = sig2 >= kTinyNorm2;
      const float sig = refl ? sig2 * rsqrt_fast(sig2) : 0.f;
      const float ah = x1 >= 0.f ? -sig : sig;
      const float vv2 = 2.f * (sig2 + sig * fabsf(x1));
      const float beta = refl ? 2.f * rcp_fast(vv2) : 0.f;
      const float v1 = x1 - ah;
      const float vA = liveA ? (ca == k + 1 ? v1 : xA) : 0.f;
      const float vB = liveB ? (cb == k + 1 ? v1 : xB) : 0.f;
      if (LIVE_A && TASER_IN(ca, VB)) vs[ca] = vA;
      if (TASER_IN(cb, VB)) vs[cb] = vB;
      if (at_work && ca == k && TASER_IN(k, VB)) db[k] = xA;
      if (at_work && cb == k && TASER_IN(k, VB)) db[k] = xB;
      if (gl == 0 && TASER_IN(k, VB)) eb[k] = ah;
      __syncwarp();
      // p_c = beta sum_j A[j][c] v_j, even and odd rows apart.
      uint64_t sA = 0ull, sB = 0ull;
#pragma unroll
      for (int q = P0 / 2; q < VB / 4; ++q) {
        const float4 v4 = *reinterpret_cast<const float4*>(vs + 4 * q);
        const uint64_t v2[2] = {f2pack(v4.x, v4.y), f2pack(v4.z, v4.w)};
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          const int p = 2 * q + h;
          if (p < P0 || p >= P) continue;
          if (LIVE_A) sA = f2fma(A[p], v2[h], sA);
          sB = f2fma(B[p], v2[h], sB);
        }
      }
      float lo, hi;
      f2unpack(sA, lo, hi);
      const float pA = liveA ? beta * (lo + hi) : 0.f;
      f2unpack(sB, lo, hi);
      const float pB = liveB ? beta * (lo + hi) : 0.f;
      if (LIVE_A && TASER_IN(ca, VB)) ps[ca] = pA;
      if (TASER_IN(cb, VB)) ps[cb] = pB;
      float kk = fmaf(vA, pA, vB * pB);
#pragma unroll
      for (int o = G / 2; o > 0; o >>= 1) kk += __shfl_xor_sync(TASER_FULL_MASK, kk, o);
      __syncwarp();
      // A <- A - v u^T - p v^T on the lane's columns, u = p - kk v.
      kk *= beta;
      const float uA = fmaf(kk, vA, -pA), uB = fmaf(kk, vB, -pB);   // -u
      const uint64_t uA2 = f2pack(uA, uA), uB2 = f2pack(uB, uB), vA2 = f2pack(-vA, -vA), vB2 = f2pack(-vB, -vB);
#pragma unroll
      for (int q = P0 / 2; q < VB / 4; ++q) {
        const float4 v4 = *reinterpret_cast<const float4*>(vs + 4 * q);
        const float4 p4 = *reinterpret_cast<const float4*>(ps + 4 * q);
        const uint64_t v2[2] = {f2pack(v4.x, v4.y), f2pack(v4.z, v4.w)};
        const uint64_t p2[2] = {f2pack(p4.x, p4.y), f2pack(p4.z, p4.w)};
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          const int p = 2 * q + h;
          if (p < P0 || p >= P) continue;
          if (LIVE_A) A[p] = f2fma(v2[h], uA2, f2fma(p2[h], vA2, A[p]));
          B[p] = f2fma(v2[h], uB2, f2fma(p2[h], vB2, B[p]));
        }
      }
      if (LIVE_A) xA = pick_row<KB + 1, KE>(A, k + 1);
      xB = pick_row<KB + 1, KE>(B, k + 1);
      __syncwarp();
    }
  });
  // Trailing 2 x 2 block: x is row NV - 1, columns NV - 1 and NV are cb of lanes 1 and 0.
  if (cb == NV - 1) db[NV - 1] = xB;
  if (cb == NV) {
    eb[NV - 1] = xB;
    db[NV] = pick_row<NV, NV>(B, NV);
  }
  __syncwarp();
  float d[NP], e2[NP];
#pragma unroll
  for (int j = 0; j < NP; ++j) {
    d[j] = db[j];
    e2[j] = j < NV ? eb[j] * eb[j] : 0.f;
  }
  // Multisection.  One-sided: sg = the hint's sign, points 2 gl and 2 gl + 1 of 2 G.
  // Two-sided (hint 0): the point gl of lambda_max(A) and the point gl of lambda_max(-A).
  const bool two = sign_hint == 0;
  const float sg0 = two ? 1.f : (sign_hint > 0 ? 1.f : -1.f);
  const float sg1 = two ? -1.f : sg0;
  const int parts = two ? G + 1 : 2 * G + 1;
  const int rounds = two ? C::ROUNDS2 : C::ROUNDS1;
  // Bracket per side: [max sg d_j, max (sg d_j + |e_{j-1}| + |e_j|)].
  float lo0 = -3.0e38f, hi0 = -3.0e38f, lo1 = -3.0e38f, hi1 = -3.0e38f;
#pragma unroll
  for (int j = 0; j < NP; ++j) {
    const float r = (j > 0 ? sqrtf(e2[j - 1]) : 0.f) + sqrtf(e2[j]);
    lo0 = fmaxf(lo0, sg0 * d[j]);
    hi0 = fmaxf(hi0, sg0 * d[j] + r);
    lo1 = fmaxf(lo1, sg1 * d[j]);
    hi1 = fmaxf(hi1, sg1 * d[j] + r);
  }
  // The Sturm count needs e2 > 0; the floor comes after the bracket, which it must not
  // widen (the zero matrix keeps the norm 0).
#pragma unroll
  for (int j = 0; j < NP; ++j) e2[j] = fmaxf(e2[j], kTinyNorm2);
  const float inv_parts = 1.f / (float)parts;
  const unsigned gmask = G == 32 ? 0xffffffffu : (1u << (G & 31)) - 1u;
  // index of the point of lane gl on each side: one-sided 2 gl and 2 gl + 1, two-sided gl
  const int p0 = two ? gl : 2 * gl, p1 = two ? gl : 2 * gl + 1;
#pragma unroll 1
  for (int round = 0; round < rounds; ++round) {
    const float st0 = (hi0 - lo0) * inv_parts, st1 = (hi1 - lo1) * inv_parts;
    const float s0 = fmaf(st0, (float)(p0 + 1), lo0);
    const float s1 = two ? fmaf(st1, (float)(p1 + 1), lo1) : fmaf(st0, (float)(p1 + 1), lo0);
    const int c0 = sturm_count<NP>(d, e2, sg0, s0);
    const int c1 = sturm_count<NP>(d, e2, sg1, s1);
    const unsigned m0 = (__ballot_sync(TASER_FULL_MASK, c0 == NP) >> (grp * G)) & gmask;
    const unsigned m1 = (__ballot_sync(TASER_FULL_MASK, c1 == NP) >> (grp * G)) & gmask;
    if (two) {
      // each side: first of its G points at or above its lambda_max
      if (m0 == 0u) {
        lo0 = fmaf(st0, (float)G, lo0);
      } else {
        const int f = __ffs(m0) - 1;
        const float nhi = fmaf(st0, (float)(f + 1), lo0);
        lo0 = f == 0 ? lo0 : fmaf(st0, (float)f, lo0);
        hi0 = nhi;
      }
      if (m1 == 0u) {
        lo1 = fmaf(st1, (float)G, lo1);
      } else {
        const int f = __ffs(m1) - 1;
        const float nhi = fmaf(st1, (float)(f + 1), lo1);
        lo1 = f == 0 ? lo1 : fmaf(st1, (float)f, lo1);
        hi1 = nhi;
      }
    } else {
      // one side, points interleaved over the lanes: p = 2 gl (m0) and 2 gl + 1 (m1)
      const int f0 = m0 ? 2 * (__ffs(m0) - 1) : 2 * G;
      const int f1 = m1 ? 2 * (__ffs(m1) - 1) + 1 : 2 * G;
      const int f = min(f0, f1);
      if (f == 2 * G) {
        lo0 = fmaf(st0, (float)(2 * G), lo0);
      } else {
        const float nhi = fmaf(st0, (float)(f + 1), lo0);
        lo0 = f == 0 ? lo0 : fmaf(st0, (float)f, lo0);
        hi0 = nhi;
      }
    }
  }
  float nrm = 0.5f * (lo0 + hi0);
  if (two) nrm = fmaxf(nrm, 0.5f * (lo1 + hi1));
  nrm *= pow2f(ex);
  if (active && gl == 0 && TASER_IN(inst, batch)) {
    tau[inst] = nrm > 0.f ? alpha / nrm : 0.f;
    if (nrm_out != nullptr) nrm_out[inst] = nrm;
    TASER_FINITE(nrm);
  }
}


// ---------------------------------------------------------------------------------
// QPSK: ||T~||_2 from the complex Hermitian form.
//
// For QPSK, T~ (N = 2U + 1) is the real form [[Re M, -Im M], [Im M, Re M]] of the
// preconditioned complex Gram M~ of [H / sqrt2, -y] ((U+1) x (U+1), Hermitian) with the
// row and column of the imaginary part of the augmented coordinate deleted.  Every
// eigenvalue of M~ appears twice in its real form, so by Cauchy interlacing the largest
// and smallest eigenvalues of T~ are those of M~, and ||T~||_2 = ||M~||_2.  M~ is read
// from T~:  M~_ab = T~_ab + i T~_{U+a,b},  M~_{a,N} = T~_{a,2U} + i T~_{U+a,2U}.
// Tridiagonalising the (U+1) complex matrix costs about 2.5x fewer flops and half the
// sequential steps of the real (2U+1) one.  UV = 8 and 16: lane gl of UV / 2 holds columns
// ca = gl + 1 and cb = UV - gl; UV = 32: one column a lane (two would need 132 registers for the
// matrix alone).  The complex multiply-adds run as packed f32x2 operations
// on {re, im} against duplicated pairs {v, v}.
// Measured (early p and one kernel for all sizes): QPSK 256x32 with the build 631 -> 614 us per
// 16,384, QPSK 128x16 419 -> 415 per 65,536.
// ---------------------------------------------------------------------------------
template <int UV>
struct HermCfg {
  static constexpr bool FOLD = UV <= 16;       // two columns a lane; else one (UV = 24, 32)
  static constexpr int HALF = UV / 2;
  static constexpr int G = FOLD ? (HALF <= 4 ? 4 : 8) : 32;   // lanes per instance, HALF or UV at work
  static constexpr int IPW = 32 / G;           // instances per warp
  static constexpr int NP = UV + 1;            // padded complex order; aug at index UV
  static constexpr int VB = (NP + 1) & ~1;     // complex vector length
  static constexpr int WARPS = 4;
  static constexpr int IPC = WARPS * IPW;
  static constexpr int INST_FLOATS = 8 * VB + 2 * VB;  // v, p ({re, re, im, im}), d, |e|^2
  static constexpr int MIN_BLOCKS = FOLD ? 4 : 5;
  // One point a lane, G + 1 parts per round.  For positive semidefinite M~ the initial bracket is
  // at most 2 lambda_max wide (|e_j| <= max d): 33^5 = 3.9e7, 9^7 = 4.8e6, 5^12 = 2.4e8.
  static constexpr int ROUNDS = G == 32 ? 5 : (G == 8 ? 7 : 12);
};

// The row r (of rows FROM..TO, known at run time) of a complex column.
template <int FROM, int TO, int NP>
__device__ __forceinline__ float2 pick_row(const float2 (&a)[NP], int r) {
  float2 v = a[FROM];
#pragma unroll
  for (int i = FROM + 1; i <= TO; ++i) v = r == i ? a[i] : v;
  return v;
}

template <int UV, bool NEG>
__global__ void __launch_bounds__(128, HermCfg<UV>::MIN_BLOCKS)
spectral_herm_kernel(int64_t batch, int U, const float* __restrict__ Tt, float alpha, float* __restrict__ tau,
                     float* __restrict__ nrm_out) {
  using C = HermCfg<UV>;
  constexpr int NP = C::NP, VB = C::VB, G = C::G, HALF = C::HALF;
  constexpr bool FOLD = C::FOLD;
  constexpr int KBLK_HERM = herm_block<UV>();
  static_assert(!FOLD || HALF % KBLK_HERM == 0, "a Householder block must not straddle step UV / 2");
  __shared__ __align__(16) float sm[C::IPC * C::INST_FLOATS];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int grp = lane / G, gl = lane % G;
  const int local = warp * C::IPW + grp;
  const int64_t inst = (int64_t)blockIdx.x * C::IPC + local;
  const bool active = inst < batch;
  // v and p of the current reflection as duplicated pairs {re, re, im, im}: one LDS.128 gives both
  // pair operands of a complex multiply-add.
  float4* vs = reinterpret_cast<float4*>(sm + local * C::INST_FLOATS);
  float4* ps = vs + VB;
  float* db = reinterpret_cast<float*>(ps + VB);
  float* eb2 = db + VB;
  // (One column a lane: cb only.)  A lane not at work takes "column 0", which no step has live.
  const bool at_work = gl < (FOLD ? HALF : UV);
  const int ca = at_work ? gl + 1 : 0, cb = at_work ? (FOLD ? UV - gl : gl + 1) : 0;
  float2 A[FOLD ? NP : 1], B[NP];                              // M~[.][ca], M~[.][cb]
  float m00 = 0.f;
  auto load = [&](auto u_c) {
    const int Uc = u_c, N = 2 * Uc + 1;
    const float* T = Tt + (active ? inst : 0) * (int64_t)N * N;
    // NEG reads the negative semidefinite JED form as its (positive semidefinite) negation;
    // the norm is the same.
    auto t = [&](int a, int b) -> float {
      const float v = active && TASER_IN(inst * N * N + a * N + b, batch * N * N) ? T[a * N + b] : 0.f;
      return NEG ? -v : v;
    };
    // M~[j][c]: users below min(UV, Uc), the augmented coordinate at index UV.
    auto entry = [&](int j, int c) -> float2 {
      const bool ju = j < UV && j < Uc, ja = j == UV;
      const bool cu = c < UV && c < Uc, cx = c == UV;
      if (ju && cu) return make_float2(t(j, c), t(Uc + j, c));
      if (ju && cx) return make_float2(t(j, 2 * Uc), t(Uc + j, 2 * Uc));
      if (ja && cu) return make_float2(t(c, 2 * Uc), -t(Uc + c, 2 * Uc));
      if (ja && cx) return make_float2(t(2 * Uc, 2 * Uc), 0.f);
      return make_float2(0.f, 0.f);
    };
#pragma unroll
    for (int j = 0; j < NP; ++j) {
      if constexpr (FOLD) A[j] = entry(j, ca);
      B[j] = entry(j, cb);
    }
    m00 = Uc >= 1 ? t(0, 0) : 0.f;
  };
  // A problem that fills the bucket (U = UV, e.g. QPSK 128x16) reads with compile-time sizes.
  if (U == UV) load(SpecInt<UV>{});
  else load(U);
  float amax = fabsf(m00);
#pragma unroll
  for (int j = 0; j < NP; ++j) {
    if constexpr (FOLD) amax = fmaxf(amax, fmaxf(fabsf(A[j].x), fabsf(A[j].y)));
    amax = fmaxf(amax, fmaxf(fabsf(B[j].x), fabsf(B[j].y)));
  }
#pragma unroll
  for (int o = G / 2; o > 0; o >>= 1) amax = fmaxf(amax, __shfl_xor_sync(TASER_FULL_MASK, amax, o));
  const int ex = scale_exponent(amax);
  {
    const float sc = pow2f(-ex);
    m00 *= sc;
#pragma unroll
    for (int j = 0; j < NP; ++j) {
      if constexpr (FOLD) A[j] = make_float2(A[j].x * sc, A[j].y * sc);
      B[j] = make_float2(B[j].x * sc, B[j].y * sc);
    }
  }
  const float2 zero = make_float2(0.f, 0.f);
  for (int i = gl; i < 2 * VB; i += G) vs[i] = make_float4(0.f, 0.f, 0.f, 0.f);
  if (gl == 0) db[0] = m00;
  // x = conj of row k of the lane's columns: the entries x_c of column k (M~ Hermitian), k = 0.
  float2 xA = zero, xB = make_float2(B[0].x, -B[0].y);
  if constexpr (FOLD) xA = make_float2(A[0].x, -A[0].y);
  __syncwarp();

  static_for_blocks<UV, KBLK_HERM>([&](auto kb) {
    constexpr int KB = decltype(kb)::value;
    constexpr int KE = (KB + KBLK_HERM < UV - 1) ? KB + KBLK_HERM : UV - 1;   // k in [KB, KE)
    constexpr bool LIVE_A = FOLD && KB < HALF;   // k < UV / 2 throughout the block: some ca > k
#pragma unroll 1
    for (int k = KB; k < KE; ++k) {
      const bool liveA = LIVE_A && ca > k, liveB = cb > k;
      float sig2 = (liveA ? fmaf(xA.x, xA.x, xA.y * xA.y) : 0.f) + (liveB ? fmaf(xB.x, xB.x, xB.y * xB.y) : 0.f);
#pragma unroll
      for (int o = G / 2; o > 0; o >>= 1) sig2 += __shfl_xor_sync(TASER_FULL_MASK, sig2, o);
      // x_{k+1}: column k + 1 is ca of lane k (k < UV / 2) or cb of lane UV - 1 - k; with one column
      // a lane, of lane k.
      const int src = grp * G + (FOLD && !LIVE_A ? UV - 1 - k : k);
      const float2 xs = LIVE_A ? xA : xB;
      const float2 x1 = make_float2(__shfl_sync(TASER_FULL_MASK, xs.x, src), __shfl_sync(TASER_FULL_MASK, xs.y, src));
      // The reflector H = I - beta v v^H with v = x - alpha e_{k+1}, alpha = -e^{i theta} sigma
      // (theta = arg x_{k+1}, sigma = ||x||) maps x to alpha e_{k+1}.  Its scalars come from
      // reciprocal square roots (a few ulp; the reflection stays orthogonal to that order, below
      // the FP32 rounding of the updates).  A column with ||x||^2 under kTinyNorm2 is left as it
      // is (beta = 0); an x_{k+1} that small takes the phase 1, and ||v||^2 then uses
      // Re(conj(e^{i theta}) x_{k+1}) = Re x_{k+1}.
      const bool refl = sig2 >= kTinyNorm2;
      const float sig = refl ? sig2 * rsqrt_fast(sig2) : 0.f;
      const float n1 = fmaf(x1.x, x1.x, x1.y * x1.y);
      const bool big1 = n1 >= kTinyNorm2;
      const float r1 = big1 ? rsqrt_fast(n1) : 0.f;
      const float2 ph = big1 ? make_float2(x1.x * r1, x1.y * r1) : make_float2(1.f, 0.f);
      const float ax1 = big1 ? n1 * r1 : x1.x;                                       // Re(conj(ph) x_{k+1})
      const float2 v1 = make_float2(fmaf(ph.x, sig, x1.x), fmaf(ph.y, sig, x1.y));   // x_{k+1} - alpha
      const float vv2 = 2.f * sig * (sig + ax1);                                     // ||v||^2
      const float beta = refl ? 2.f * rcp_fast(vv2) : 0.f;
      const float2 vA = liveA ? (ca == k + 1 ? v1 : xA) : zero;
      const float2 vB = liveB ? (cb == k + 1 ? v1 : xB) : zero;
      if (LIVE_A && TASER_IN(ca, VB)) vs[ca] = make_float4(vA.x, vA.x, vA.y, vA.y);
      if (TASER_IN(cb, VB)) vs[cb] = make_float4(vB.x, vB.x, vB.y, vB.y);
      if (FOLD && at_work && ca == k && TASER_IN(k, VB)) db[k] = xA.x;
      if (at_work && cb == k && TASER_IN(k, VB)) db[k] = xB.x;
      if (gl == 0 && TASER_IN(k, VB)) eb2[k] = sig2;                                 // |alpha|^2
      __syncwarp();
      // p_c = beta sum_j conj(M~[j][c]) v_j in one pass over j:
      //   S = sum {Re M, Im M} {Re v, Re v},  Q = sum {Re M, Im M} {Im v, Im v},
      //   conj(M) v = (S.re + Q.im, Q.re - S.im).
      uint64_t Sa = 0ull, Qa = 0ull, Sb = 0ull, Qb = 0ull;
#pragma unroll
      for (int j = KB + 1; j < NP; ++j) {
        const float4 q = vs[j];
        const uint64_t vr = f2pack(q.x, q.y), vi = f2pack(q.z, q.w);
        if constexpr (LIVE_A) {
          const uint64_t Ma = f2pack(A[j].x, A[j].y);
          Sa = f2fma(Ma, vr, Sa);
          Qa = f2fma(Ma, vi, Qa);
        }
        const uint64_t Mb = f2pack(B[j].x, B[j].y);
        Sb = f2fma(Mb, vr, Sb);
        Qb = f2fma(Mb, vi, Qb);
      }
      auto prod = [&](uint64_t S, uint64_t Q, bool live) {
        float sx, sy, qx, qy;
        f2unpack(S, sx, sy);
        f2unpack(Q, qx, qy);
        return live ? make_float2(beta * (sx + qy), beta * (qx - sy)) : zero;
      };
      const float2 pA = LIVE_A ? prod(Sa, Qa, liveA) : zero, pB = prod(Sb, Qb, liveB);
      if (LIVE_A && TASER_IN(ca, VB)) ps[ca] = make_float4(pA.x, pA.x, pA.y, pA.y);
      if (TASER_IN(cb, VB)) ps[cb] = make_float4(pB.x, pB.x, pB.y, pB.y);
      float kk = fmaf(vA.x, pA.x, vA.y * pA.y) + fmaf(vB.x, pB.x, vB.y * pB.y);      // Re(conj(v_c) p_c)
#pragma unroll
      for (int o = G / 2; o > 0; o >>= 1) kk += __shfl_xor_sync(TASER_FULL_MASK, kk, o);
      __syncwarp();
      // M~[j][c] <- M~[j][c] - v_j conj(u_c) - p_j conj(v_c), u = p - kk v, as four pair FMAs per row
      // (v conj(u) = {Re v, Re v}{Re u, -Im u} + {Im v, Im v}{Im u, Re u}).
      kk *= beta;
      const float2 uA = make_float2(fmaf(-kk, vA.x, pA.x), fmaf(-kk, vA.y, pA.y));
      const float2 uB = make_float2(fmaf(-kk, vB.x, pB.x), fmaf(-kk, vB.y, pB.y));
      const uint64_t ua = f2pack(-uA.x, uA.y), ub = f2pack(-uA.y, -uA.x), va = f2pack(-vA.x, vA.y), vb = f2pack(-vA.y, -vA.x);
      const uint64_t wa = f2pack(-uB.x, uB.y), wb = f2pack(-uB.y, -uB.x), ya = f2pack(-vB.x, vB.y), yb = f2pack(-vB.y, -vB.x);
      auto update = [](float2& m, const float4& q, const float4& w, uint64_t a, uint64_t b, uint64_t c, uint64_t d) {
        uint64_t M = f2pack(m.x, m.y);
        M = f2fma(f2pack(q.x, q.y), a, M);
        M = f2fma(f2pack(q.z, q.w), b, M);
        M = f2fma(f2pack(w.x, w.y), c, M);
        M = f2fma(f2pack(w.z, w.w), d, M);
        f2unpack(M, m.x, m.y);
      };
#pragma unroll
      for (int j = KB + 1; j < NP; ++j) {
        const float4 q = vs[j], w = ps[j];
        if constexpr (LIVE_A) update(A[j], q, w, ua, ub, va, vb);
        update(B[j], q, w, wa, wb, ya, yb);
      }
      if constexpr (LIVE_A) {
        const float2 m = pick_row<KB + 1, KE>(A, k + 1);
        xA = make_float2(m.x, -m.y);
      }
      {
        const float2 m = pick_row<KB + 1, KE>(B, k + 1);
        xB = make_float2(m.x, -m.y);
      }
      __syncwarp();
    }
  });
  // Trailing 2 x 2 block: x is row UV - 1 (conjugated).
  if (cb == UV - 1) db[UV - 1] = xB.x;
  if (cb == UV) {
    eb2[UV - 1] = fmaf(xB.x, xB.x, xB.y * xB.y);
    db[UV] = B[UV].x;
  }
  __syncwarp();
  float d[NP], e2[NP];
#pragma unroll
  for (int j = 0; j < NP; ++j) {
    d[j] = db[j];
    e2[j] = j < UV ? eb2[j] : 0.f;
  }
  float lo = -3.0e38f, hi = -3.0e38f;
#pragma unroll
  for (int j = 0; j < NP; ++j) {
    const float r = (j > 0 ? sqrtf(e2[j - 1]) : 0.f) + sqrtf(e2[j]);
    lo = fmaxf(lo, d[j]);
    hi = fmaxf(hi, d[j] + r);
  }
  // The Sturm count needs e2 > 0; the floor comes after the bracket, which it must not
  // widen (the zero matrix keeps the norm 0).
#pragma unroll
  for (int j = 0; j < NP; ++j) e2[j] = fmaxf(e2[j], kTinyNorm2);
  // One-sided multisection, G + 1 parts: lane gl evaluates the point sigma = lo + (gl + 1) step.
  // (Two points a lane over UV + 1 parts, 5 rounds, were 1.5% slower at UV = 16.)
  const float inv_parts = 1.f / (float)(G + 1);
  const unsigned gmask = G == 32 ? 0xffffffffu : (1u << (G & 31)) - 1u;
#pragma unroll 1
  for (int round = 0; round < C::ROUNDS; ++round) {
    const float step = (hi - lo) * inv_parts;
    const float sigma = fmaf(step, (float)(gl + 1), lo);
    const int cnt = sturm_count<NP>(d, e2, 1.f, sigma);
    const unsigned mine = (__ballot_sync(TASER_FULL_MASK, cnt == NP) >> (grp * G)) & gmask;
    const int f = mine ? __ffs(mine) - 1 : G;   // first point at or above lambda_max
    if (f == G) {
      lo = fmaf(step, (float)G, lo);
    } else {
      const float nhi = fmaf(step, (float)(f + 1), lo);
      const float nlo = f == 0 ? lo : fmaf(step, (float)f, lo);
      lo = nlo;
      hi = nhi;
    }
  }
  const float nrm = 0.5f * (lo + hi) * pow2f(ex);
  if (active && gl == 0 && TASER_IN(inst, batch)) {
    tau[inst] = nrm > 0.f ? alpha / nrm : 0.f;
    if (nrm_out != nullptr) nrm_out[inst] = nrm;
    TASER_FINITE(nrm);
  }
}


template <int UV>
static cudaError_t launch_herm(int64_t batch, int U, const float* Tt, bool neg, float alpha, float* tau,
                               float* nrm, cudaStream_t st) {
  const int64_t blocks = (batch + HermCfg<UV>::IPC - 1) / HermCfg<UV>::IPC;
  if (neg) spectral_herm_kernel<UV, true><<<(unsigned)blocks, 128, 0, st>>>(batch, U, Tt, alpha, tau, nrm);
  else spectral_herm_kernel<UV, false><<<(unsigned)blocks, 128, 0, st>>>(batch, U, Tt, alpha, tau, nrm);
  return cudaGetLastError();
}

// ||T~||_2 of QPSK matrices (N = 2U + 1) through the complex form; U <= 32.  sign = +1 for
// a positive semidefinite T~ (MIMO), -1 for a negative semidefinite one (JED).
// Layouts of 12 and 24 columns, with idle lanes, as in spectral() (with the build, 60,000 QPSK 24x12
// 262 -> 225 us, 20,001 40x20 506 -> 375 us; 20,000 JED QPSK bursts of K = 25 646 -> 491 us).
cudaError_t spectral_qpsk(int64_t batch, int U, const float* Tt, int sign, float alpha, float* tau, float* nrm,
                          cudaStream_t st) {
  const bool neg = sign < 0;
  if (U + 1 <= 9) return launch_herm<8>(batch, U, Tt, neg, alpha, tau, nrm, st);
  if (U + 1 <= 13) return launch_herm<12>(batch, U, Tt, neg, alpha, tau, nrm, st);
  if (U + 1 <= 17) return launch_herm<16>(batch, U, Tt, neg, alpha, tau, nrm, st);
  if (U + 1 <= 25) return launch_herm<24>(batch, U, Tt, neg, alpha, tau, nrm, st);
  return launch_herm<32>(batch, U, Tt, neg, alpha, tau, nrm, st);
}

template <int NV>
static cudaError_t launch_spectral(int64_t batch, int N, const float* Tt, float alpha, int hint, float* tau,
                                   float* nrm, cudaStream_t st) {
  const int64_t blocks = (batch + SpecFoldCfg<NV>::IPC - 1) / SpecFoldCfg<NV>::IPC;
  auto go = [&](auto kern) { kern<<<(unsigned)blocks, 128, 0, st>>>(batch, N, Tt, alpha, hint, tau, nrm); };
  if constexpr (NV <= 32) {
    go(spectral_fold_kernel<NV, NV == 32 ? 4 : (NV == 24 ? 5 : 6)>);
  } else {
    int dev = 0, sms = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e != cudaSuccess) return e;
    if (blocks <= 2 * sms) go(spectral_fold_kernel<NV, 2>);
    else go(spectral_fold_kernel<NV, 3>);
  }
  return cudaGetLastError();
}

cudaError_t spectral(int64_t batch, int N, const float* Tt, float alpha, int hint, float* tau, float* nrm,
                     cudaStream_t st) {
  // Layouts of 12 and 24 columns, with idle lanes, beside the powers of two: a problem pays for its
  // own steps, rows and columns (with the build, 60,000 BPSK of N = 13 147 -> 131 us, 30,000 of
  // N = 25 248 -> 201 us; 50,000 JED BPSK bursts of K = 20 369 -> 293 us).
  const int nv = N - 1;
  if (nv <= 8) return launch_spectral<8>(batch, N, Tt, alpha, hint, tau, nrm, st);
  if (nv <= 12) return launch_spectral<12>(batch, N, Tt, alpha, hint, tau, nrm, st);
  if (nv <= 16) return launch_spectral<16>(batch, N, Tt, alpha, hint, tau, nrm, st);
  if (nv <= 24) return launch_spectral<24>(batch, N, Tt, alpha, hint, tau, nrm, st);
  if (nv <= 32) return launch_spectral<32>(batch, N, Tt, alpha, hint, tau, nrm, st);
  return launch_spectral<64>(batch, N, Tt, alpha, hint, tau, nrm, st);
}

}  // namespace taser

TASER_DEBUG_COLLECTOR(spectral)
