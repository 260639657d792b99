// Fixed-point TASER: the 14-bit datapath of the paper's VLSI designs (Sec. IV-B operation
// modes, Sec. IV-D fixed-point parameters and inverse square-root LUT), computed exactly
// in integer arithmetic.
//
// Formats (two's complement, saturating to [-2^13, 2^13 - 1]):
//   L~, V rows < N: 8 fraction bits;  row N: 7;  L~_NN (constant register): 5;
//   T^ = 2 tau T~: 12 fraction bits (|T^_ij| <= 2 alpha < 2);  D_j: 8, D_N: 5.
// Rounding to a narrower format is round-half-up: (a + 2^(k-1)) >> k, arithmetic shift.
// The MAC accumulates exactly (row i < N at 20 fraction bits, row N at 19); the squared
// column norm is exact (16 fraction bits); its inverse square root comes from a LUT of
// 2^11 entries (13 fraction bits) indexed by the top 11 bits of the norm after an even
// normalisation x = m 4^e, m in [1, 4); the scale D_j * LUT keeps its power-of-two part
// as a shift and each PE rounds V_ij * scale once.  Only the constant-L~_NN mode exists.
//
// N <= 33: the products run on the tensor cores, exactly (detect_fxt_kernel below).
// 34 <= N <= 65: one warp per instance, lane j owns columns j and j + 32.  Its column of
// T^ lives in registers; L~ lives in shared memory, one int per entry, and its rows are
// broadcast to the lanes (one LDS.128 feeds four IMADs).  Products are below 2^26, so
// 16 of them (four partial sums of four) are summed in int32 before each 64-bit
// accumulate: exact for every input.
#include <type_traits>

#include "tct_job.cuh"

namespace taser {

template <int NB>
struct FxCfg {
  static_assert(NB == 64, "smaller buckets run on the tensor cores");
  static constexpr int CPL = 2;                    // columns per lane
  static constexpr int KC = 16;                    // products summed in int32 per chunk
  static constexpr int NCH = NB / KC;
  static constexpr int SLOT = (NB + 1) * NB;       // ints per warp: NB rows + row N
  static constexpr int WARPS = 4;
};

constexpr int kFxLutEntries = 2048;
constexpr int kFxLutInts = kFxLutEntries / 2;      // uint16 entries

// floor(x * scale + 1/2) as a 14-bit code (scale a power of two, so x * scale is exact and
// the + 1/2 is exact below 2^23; larger magnitudes saturate either way).  NaN -> 0.
__device__ __forceinline__ int fx_quant(float x, float scale, bool& sat) {
  const float v = floorf(__fadd_rn(__fmul_rn(x, scale), 0.5f));
  if (isnan(v)) {
    sat = true;
    return 0;
  }
  if (v < -8192.f) {
    sat = true;
    return -8192;
  }
  if (v > 8191.f) {
    sat = true;
    return 8191;
  }
  return (int)v;
}

__device__ __forceinline__ int fx_sat(long long a, bool& sat) {
  if (a < -8192) {
    sat = true;
    return -8192;
  }
  if (a > 8191) {
    sat = true;
    return 8191;
  }
  return (int)a;
}

// LUT[i] = round(2^13 / sqrt((i + 1/2) / 512)) = round(2^18 / sqrt(m)), m = 2i + 1, for i in
// [512, 2048): the r with (2r - 1)^2 m <= 2^38 < (2r + 1)^2 m, from an FP32 estimate corrected
// in integers.  Entries below 512 are unused (0).  (FP64 divisions and square roots here cost
// every block about 30 us: 2,048 entries on an FP64 pipe of a few lanes.)
__device__ __forceinline__ void fx_fill_lut(unsigned short* lut) {
  for (int i = threadIdx.x; i < kFxLutEntries; i += blockDim.x) {
    long long r = 0;
    if (i >= 512) {
      const long long m = 2 * i + 1;
      r = (long long)(262144.f * rsqrtf((float)m) + 0.5f);
      if ((2 * r - 1) * (2 * r - 1) * m > (1ll << 38)) --r;
      if ((2 * r + 1) * (2 * r + 1) * m <= (1ll << 38)) ++r;
    }
    lut[i] = (unsigned short)r;
  }
}

__device__ __forceinline__ long long fx_round_shift(long long a, int k) { return (a + (1ll << (k - 1))) >> k; }

// Algorithm 1 on one instance.  Lq: this warp's (NB + 1) x NB ints; lut: 2048 uint16.
template <int NB>
__device__ __forceinline__ void fx_run(const Job& jb, int* Lq, const unsigned short* lut, int lane) {
  using C = FxCfg<NB>;
  constexpr int CPL = C::CPL, KC = C::KC, NCH = C::NCH;
  const int N = jb.N, nv = N - 1;
  const float* T = jb.T;
  const float tau2 = __fadd_rn(*jb.tau, *jb.tau);
  bool sat = false;
  uint32_t fl = 0;

  // Quantised inputs: this lane's columns of T^ (bucket rows), T^_{N,j}, T^_{j,N} and D_j.
  int tc[CPL][NB], tNj[CPL], tjN[CPL], dq[CPL];
#pragma unroll
  for (int c = 0; c < CPL; ++c) {
    const int j = lane + 32 * c;
    const bool real = j < nv;
#pragma unroll
    for (int k = 0; k < NB; ++k)
      tc[c][k] = (real && k < nv && TASER_IN(k * N + j, N * N))
                     ? fx_quant(__fmul_rn(tau2, T[(int64_t)k * N + j]), 4096.f, sat)
                     : 0;
    const bool ok = real && TASER_IN(nv * N + j, N * N) && TASER_IN(j * N + nv, N * N) && TASER_IN(j, N);
    tNj[c] = ok ? fx_quant(__fmul_rn(tau2, T[(int64_t)nv * N + j]), 4096.f, sat) : 0;
    tjN[c] = ok ? fx_quant(__fmul_rn(tau2, T[(int64_t)j * N + nv]), 4096.f, sat) : 0;
    dq[c] = ok ? fx_quant(jb.D[j], 256.f, sat) : 0;
  }
  const int tNN = fx_quant(__fmul_rn(tau2, T[(int64_t)nv * N + nv]), 4096.f, sat);
  const int lnn = fx_quant(jb.D[nv], 32.f, sat);

  // L~(0) = D: diagonal codes, zero elsewhere (row N starts at zero).
  int* rowN = Lq + NB * NB;
  for (int i = lane; i < C::SLOT; i += 32) Lq[i] = 0;
  __syncwarp();
#pragma unroll
  for (int c = 0; c < CPL; ++c) {
    const int j = lane + 32 * c;
    if (j < nv && TASER_IN(j * NB + j, NB * NB)) Lq[j * NB + j] = dq[c];
  }
  __syncwarp();

  // acc[c] += sum over the KC columns k of chunk ch of L~_ik T^_kj, with four independent
  // int32 partial sums (each at most 4 products below 2^26: exact) for instruction-level
  // parallelism, then one 64-bit accumulate.
  auto chunk_mac = [&](const int* lrow, int ch, long long (&acc)[CPL]) {
    int p0[CPL], p1[CPL], p2[CPL], p3[CPL];
#pragma unroll
    for (int c = 0; c < CPL; ++c) p0[c] = p1[c] = p2[c] = p3[c] = 0;
#pragma unroll
    for (int kk = 0; kk < KC; kk += 4) {
      const int4 l4 = *reinterpret_cast<const int4*>(lrow + kk);
      const int k0 = ch * KC + kk;
#pragma unroll
      for (int c = 0; c < CPL; ++c) {
        p0[c] += l4.x * tc[c][k0];
        p1[c] += l4.y * tc[c][k0 + 1];
        p2[c] += l4.z * tc[c][k0 + 2];
        p3[c] += l4.w * tc[c][k0 + 3];
      }
    }
#pragma unroll
    for (int c = 0; c < CPL; ++c) acc[c] += (long long)((p0[c] + p1[c]) + (p2[c] + p3[c]));
  };

  for (int t = 0; t < jb.t_max; ++t) {
    long long x[CPL];
#pragma unroll
    for (int c = 0; c < CPL; ++c) x[c] = 0;

    // Gradient step, rows i < N: V_ij = round((L~_ij 2^12 - sum_k<=i L~_ik T^_kj) / 2^12).
    for (int i = 0; i < nv; ++i) {
      int* row = Lq + i * NB;
      long long acc[CPL];
#pragma unroll
      for (int c = 0; c < CPL; ++c) acc[c] = 0;
#pragma unroll
      for (int ch = 0; ch < NCH; ++ch) {
        if (ch * KC > i) break;                    // L~_ik = 0 for k > i
        chunk_mac(row + ch * KC, ch, acc);
      }
      int v[CPL];
#pragma unroll
      for (int c = 0; c < CPL; ++c) {
        const int j = lane + 32 * c;             // j <= i < nv <= NB: inside the row
        v[c] = j <= i ? fx_sat(fx_round_shift(((long long)row[j] << 12) - acc[c], 12), sat) : 0;
      }
      __syncwarp();                                // every lane has read row i
#pragma unroll
      for (int c = 0; c < CPL; ++c) {
        const int j = lane + 32 * c;
        if (j <= i && TASER_IN(i * NB + j, NB * NB)) {
          row[j] = v[c];
          x[c] += (long long)(v[c] * v[c]);
        }
      }
    }

    // Row N: 19 fraction bits; the L~_NN (5-bit) product is aligned by 2 bits.
    {
      long long acc[CPL];
#pragma unroll
      for (int c = 0; c < CPL; ++c) acc[c] = 0;
#pragma unroll
      for (int ch = 0; ch < NCH; ++ch) chunk_mac(rowN + ch * KC, ch, acc);
      // V_NN (for the flag only): L~_NN 2^14 - sum_k L~_Nk T^_kN - (L~_NN T^_NN) 2^2.
      long long part = 0;
#pragma unroll
      for (int c = 0; c < CPL; ++c) {
        const int j = lane + 32 * c;
        if (j < nv) part += (long long)(rowN[j] * tjN[c]);
      }
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) part += __shfl_xor_sync(TASER_FULL_MASK, part, o);
      const long long vnn = ((long long)lnn << 14) - part - ((long long)(lnn * tNN) << 2);
      if (vnn <= 0) fl |= TASER_FLAG_LNN_SIGN;
      int v[CPL];
#pragma unroll
      for (int c = 0; c < CPL; ++c) {
        const int j = lane + 32 * c;
        v[c] = 0;
        if (j < nv) {
          const long long a = ((long long)rowN[j] << 12) - acc[c] - ((long long)(lnn * tNj[c]) << 2);
          v[c] = fx_sat(fx_round_shift(a, 12), sat);
        }
      }
      __syncwarp();
#pragma unroll
      for (int c = 0; c < CPL; ++c) {
        const int j = lane + 32 * c;
        if (j < nv) {
          rowN[j] = v[c];
          x[c] += 4ll * (long long)(v[c] * v[c]);   // 7 -> 8 fraction bits before squaring
        }
      }
    }

    // Prox: scale unit (LUT inverse square root times D_j), then each PE rescales.
#pragma unroll
    for (int c = 0; c < CPL; ++c) {
      const int j = lane + 32 * c;
      if (j >= nv) continue;
      int cs = 0, sh = 13;
      if (x[c] > 0) {
        const unsigned long long ux = (unsigned long long)x[c];
        const int e = (63 - __clzll(x[c])) & ~1;
        const unsigned long long idx = e >= 9 ? (ux >> (e - 9)) : (ux << (9 - e));
        cs = TASER_IN(idx, 2048) ? dq[c] * (int)lut[idx] : 0;
        sh = 13 + (e >> 1);
      } else {
        fl |= TASER_FLAG_ZERO_COLUMN;
      }
      for (int i = j; i < nv; ++i) {
        if (!TASER_IN(i * NB + j, NB * NB)) continue;
        int* p = Lq + i * NB + j;
        *p = fx_sat(fx_round_shift((long long)(*p) * cs, sh), sat);
      }
      rowN[j] = fx_sat(fx_round_shift((long long)rowN[j] * cs, sh), sat);
    }
    __syncwarp();
  }

  // Outputs: flags, decisions sign(L~_N,j) (sign(0) = +1), L~ as reals.
  if (sat) fl |= TASER_FLAG_SATURATED;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) fl |= __shfl_xor_sync(TASER_FULL_MASK, fl, o);
  if (lane == 0 && jb.flag != nullptr && fl) atomicOr(jb.flag, fl);
#pragma unroll
  for (int c = 0; c < CPL; ++c) {
    const int j = lane + 32 * c;
    if (j < nv && TASER_IN(j, N - 1)) jb.s[j] = rowN[j] >= 0 ? int8_t(1) : int8_t(-1);
  }
  if (jb.L != nullptr) {
    for (int e = lane; e < N * N; e += 32) {
      const int r = e / N, cc = e - r * N;
      float val = 0.f;
      if (cc <= r) {
        if (r == nv) val = cc == nv ? (float)lnn * (1.f / 32.f) : (float)rowN[cc] * (1.f / 128.f);
        else val = TASER_IN(r * NB + cc, NB * NB) ? (float)Lq[r * NB + cc] * (1.f / 256.f) : 0.f;
      }
      jb.L[e] = val;
    }
  }
  __syncwarp();
}

// Persistent kernel: dense instances at a fixed stride, or items popped from a bucket queue.
template <int NB, bool QUEUE>
__global__ void __launch_bounds__(128, 1)
detect_fx14_kernel(int64_t batch, int N, int t_max, const float* __restrict__ Tt, const float* __restrict__ Dg,
                   const float* __restrict__ tau, float* __restrict__ L, int8_t* __restrict__ s,
                   uint32_t* __restrict__ flags, Queue q, const float* __restrict__ T_pool,
                   const float* __restrict__ D_pool, float* __restrict__ L_pool, int8_t* __restrict__ s_pool) {
  using C = FxCfg<NB>;
  extern __shared__ __align__(16) int fsm[];
  unsigned short* lut = reinterpret_cast<unsigned short*>(fsm);
  fx_fill_lut(lut);
  __syncthreads();
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  int* Lq = fsm + kFxLutInts + warp * C::SLOT;
  const int64_t stride = (int64_t)gridDim.x * C::WARPS;
  for (int64_t k = 0;; ++k) {
    Job jb;
    if constexpr (QUEUE) {
      int pos = 0;
      if (lane == 0) pos = q.pop(1);
      pos = __shfl_sync(TASER_FULL_MASK, pos, 0);
      if (pos >= q.count()) break;
      const int idx = q.item_at(pos);
      jb = item_job(q.items[idx], idx, T_pool, D_pool, tau, L_pool, s_pool, flags);
    } else {
      const int64_t inst = (int64_t)blockIdx.x * C::WARPS + warp + k * stride;
      if (inst >= batch) break;
      jb = dense_job(inst, N, t_max, Tt, Dg, tau, L, s, flags);
    }
    fx_run<NB>(jb, Lq, lut, lane);
  }
}

template <int NB, bool QUEUE>
static cudaError_t launch_fx14(int64_t batch, int N, int t_max, const float* Tt, const float* D, const float* tau,
                               float* L, int8_t* s, uint32_t* flags, const Queue& q, int blocks_per_sm,
                               const float* T_pool, const float* D_pool, float* L_pool, int8_t* s_pool,
                               cudaStream_t st) {
  using C = FxCfg<NB>;
  const size_t smem = (size_t)(kFxLutInts + C::WARPS * C::SLOT) * sizeof(int);
  auto kern = detect_fx14_kernel<NB, QUEUE>;
  int dev = 0, sms = 0, fit = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  if (e == cudaSuccess) e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e == cudaSuccess) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&fit, kern, 32 * C::WARPS, smem);
  if (e != cudaSuccess) return e;
  const int per_sm = blocks_per_sm > 0 && blocks_per_sm < fit ? blocks_per_sm : (fit > 0 ? fit : 1);
  int64_t blocks = (int64_t)sms * per_sm;
  if (!QUEUE) {
    const int64_t need = (batch + C::WARPS - 1) / C::WARPS;
    if (need < blocks) blocks = need;
  }
  kern<<<(unsigned)blocks, 32 * C::WARPS, smem, st>>>(batch, N, t_max, Tt, D, tau, L, s, flags, q, T_pool, D_pool,
                                                    L_pool, s_pool);
  return cudaGetLastError();
}

// ---------------------------------------------------------------------------------
// N <= 33: the transposed tensor-core form of detect_tc.cu (bucket 16 also for N <= 9, faster
// than the integer kernel there too), one warp per instance, on integer codes.  A 14-bit code
// splits as x = 128 h + l with h in [-64, 63] and l in [0, 127], both exact in FP16, so a product
// sum P = sum_k L_ik T_kj is
//   P = 2^14 sum h h' + 2^7 sum (h l' + l h') + sum l l',
// three mma chains (four mma per tile and k-tile) in FP32 accumulators.  The A operands are -4 h
// and -4 l of T^; the accumulators start at kMagic = 1.5 2^23, and while a chain's sum stays within
// +-2^22 they are integers in [2^23, 2^24), exact in any order, whose low mantissa bits are the sum
// itself, so no conversion is needed.  The largest sum, 4 NB (64 127 + 127 64), is 2.08e6 at NB = 32
// (the kernel asserts the bounds of all three chains and of the integer sums):
//   hh = L - 4 sum h h',  x = -4 sum (h l' + l h'),  ll = -4 sum l l',
//   V = (L 2^12 - P + 2^11) >> 12 = hh + ((2^13 + 2^7 x + ll) >> 14)       (exact in int32).
// L~ stays in registers as the bits of kMagic + code (the C operand of the hh chain, and its
// low half word is the code).  The squared norm is below 2^32 (32 x 2^26 + 4 x 2^26): uint32.
// What bounds it: issue (57%) and the ALU pipe (55%), 766 warp instructions per instance and
// iteration at N = 33 against 3,500 of the integer kernel (a 64-bit accumulate and rounding
// per entry, IMAD chains).  Per 8,192 problems, t_max = 20: N = 33 0.775 -> 0.204 ms, N = 17
// 0.367 -> 0.083, N = 9 0.229 -> 0.080; per 65,536 at N = 33 6.07 -> 1.51 ms.  5 blocks an SM
// (96 registers) 0.222 ms, 3 blocks 0.205 ms.
// ---------------------------------------------------------------------------------
constexpr uint32_t kMagic = 0x4b400000u;   // 1.5 * 2^23 as a float; its low 16 bits are zero

__device__ __forceinline__ void mma16816_c(float (&d)[4], const uint32_t (&a)[4], const uint32_t (&b)[2],
                                           float c0, float c1, float c2, float c3) {
  asm("mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, "
      "{%10,%11,%12,%13};"
      : "=f"(d[0]), "=f"(d[1]), "=f"(d[2]), "=f"(d[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b[0]), "r"(b[1]), "f"(c0), "f"(c1), "f"(c2), "f"(c3));
}

__device__ __forceinline__ uint32_t hadd2_bits(uint32_t a, uint32_t b) {
  const __half2 r = __hadd2(*reinterpret_cast<const __half2*>(&a), *reinterpret_cast<const __half2*>(&b));
  return *reinterpret_cast<const uint32_t*>(&r);
}

// max(-8192, min(8191, v)); any change leaves bits in `sat`.
__device__ __forceinline__ int fx_clamp(int v, int& sat) {
  const int c = max(-8192, min(8191, v));
  sat |= v ^ c;
  return c;
}

template <int NB, class Src>
__global__ void __launch_bounds__(128, 4)
detect_fxt_kernel(Src src, int slot_floats) {
  using C = TctCfg<NB>;
  constexpr int MT = C::MT, KT = C::KT, NT = C::NT;
  constexpr int64_t HH = 4 * NB * 64 * 64 + 8192, HL = 4 * NB * 2 * 64 * 127, LL = 4 * NB * 127 * 127;
  static_assert(HH <= 1 << 22 && HL <= 1 << 22 && LL <= 1 << 22, "the chains' sums must stay within 2^22 of kMagic");
  static_assert(128 * HL + LL + 8192 + (16ll << 26) < 1ll << 31, "the rounding sum (with row N's L~_NN term) is int32");
  static_assert((NB + 4ll) << 26 < 1ll << 32, "the squared column norm is uint32");
  extern __shared__ __align__(16) float smem[];
  unsigned short* lut = reinterpret_cast<unsigned short*>(smem);
  fx_fill_lut(lut);
  __syncthreads();
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int g = lane >> 2, tq = lane & 3;
  float* slot = smem + kFxLutInts + warp * (slot_floats + kTcRecFloats);
  struct JobOut {
    float* L;
    int8_t* s;
    uint32_t* flag;
    int N, t_max, shift;
  };
  static_assert(2 * sizeof(JobOut) <= kTcRecFloats * sizeof(float), "job records must fit");
  JobOut* outs = reinterpret_cast<JobOut*>(slot + slot_floats);
  auto park = [&](const Job& jb, int shift, int which) {
    if (lane == 0) outs[which] = JobOut{jb.L, jb.s, jb.flag, jb.N, jb.t_max, shift};
  };
  Cursor<Src> cursor;
  int cur = 0;
  bool have;
  {
    Job first;
    double* ob = nullptr;
    have = cursor.next(src, first, ob, lane);
    if (have) park(first, stage_job(slot, first, lane, slot_floats), 0);
  }
  // Element (M, n, e) of V^T is k = 16M + g + 8(e >> 1), i = 8n + 2tq + (e & 1).  `live`: it can
  // be nonzero (blocks above the diagonal of V are not, and of row N's tile only i = NB is).
  constexpr auto live = [](int M, int n, int e) {
    return C::has_tile(M, n) && !(n == 2 * M && e >= 2) && !(n == NT - 1 && (e & 1));
  };

  while (have) {
    asm volatile("cp.async.wait_all;" ::: "memory");
    __syncwarp();
    const int N = outs[cur].N, t_max = outs[cur].t_max;
    const float* T = slot + outs[cur].shift;
    const float* Di = slot + N * N + 4;
    const float tau2 = __fadd_rn(Di[N], Di[N]);
    bool qsat = false;
    auto tq14 = [&](int r, int c) -> int {   // T^ code at real indices
      return fx_quant(__fmul_rn(tau2, T[r * N + c]), 4096.f, qsat);
    };
    // A operands: rows are the columns j of V, columns the k of the contraction.
    uint32_t ah[MT][KT][4], al[MT][KT][4];
#pragma unroll
    for (int M = 0; M < MT; ++M)
#pragma unroll
      for (int kt = 0; kt < KT; ++kt)
#pragma unroll
        for (int x = 0; x < 4; ++x) {
          float h2[2], l2[2];
#pragma unroll
          for (int p = 0; p < 2; ++p) {
            const int j = 16 * M + g + 8 * (x & 1), k = 16 * kt + 2 * tq + 8 * (x >> 1) + p;
            const int t = (j < N - 1 && k < N - 1) ? tq14(k, j) : 0;
            h2[p] = (float)(-4 * (t >> 7));
            l2[p] = (float)(-4 * (t & 127));
          }
          ah[M][kt][x] = pack2<true>(h2[0], h2[1]);
          al[M][kt][x] = pack2<true>(l2[0], l2[1]);
        }
    const int lnn = fx_quant(Di[N - 1], 32.f, qsat);
    const int tNN = tq14(N - 1, N - 1);
    // V_NN <= 0  <=>  vnn0 <= sum_k L_Nk T^_kN.
    const int vnn0 = lnn * 16384 - 4 * (lnn * tNN);
    // This lane's rows k of V^T: T^_kN, D_k and the constant of the rounding sum (with row N's
    // L~_NN term, held by the lanes tq == 0).
    int tjN[MT][2], dq[MT][2];
    uint32_t kN[MT][2];
    constexpr uint32_t kRound = 8192u - 129u * kMagic;
#pragma unroll
    for (int M = 0; M < MT; ++M)
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const int k = 16 * M + g + 8 * h;
        const bool real = k < N - 1;
        tjN[M][h] = real ? tq14(k, N - 1) : 0;
        dq[M][h] = real ? fx_quant(Di[k], 256.f, qsat) : 0;
        const int tNj = real ? tq14(N - 1, k) : 0;
        kN[M][h] = kRound - (tq == 0 ? 16u * (uint32_t)(lnn * tNj) : 0u);
      }
    uint32_t m[MT][NT][4];   // kMagic + code
#pragma unroll
    for (int M = 0; M < MT; ++M)
#pragma unroll
      for (int n = 0; n < NT; ++n)
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          const int k = 16 * M + g + 8 * (e >> 1), i = 8 * n + 2 * tq + (e & 1);
          m[M][n][e] = kMagic + (live(M, n, e) && i == k ? (uint32_t)dq[M][e >> 1] : 0u);
        }
    // After row_sums a lane owns the sum of one row k: its D code.
    const int k_own = row_column(owned_row<2 * MT>(0, tq), g);
    const bool real_own = k_own < N - 1;
    int dq_own = 0;
#pragma unroll
    for (int r = 0; r < 2 * MT; ++r) dq_own = owned_row<2 * MT>(0, tq) == r ? dq[r / 2][r % 2] : dq_own;
    __syncwarp();  // every lane has read the slot
    bool have_next;
    {
      Job nxt;
      double* ob = nullptr;
      have_next = cursor.next(src, nxt, ob, lane);
      if (have_next) park(nxt, stage_job(slot, nxt, lane, slot_floats), cur ^ 1);
    }
    uint32_t fl = 0;
    int sat = qsat ? 1 : 0;
    const bool lo0 = 2 * tq < g, lo1 = 2 * tq + 1 < g;   // below V^T's diagonal inside its blocks
    const float fm = __uint_as_float(kMagic);

    for (int t = 0; t < t_max; ++t) {
      // V_NN (for the flag only), from the old row N.
      {
        int part = 0;
#pragma unroll
        for (int M = 0; M < MT; ++M)
#pragma unroll
          for (int h = 0; h < 2; ++h) part += (int)(m[M][NT - 1][2 * h] - kMagic) * tjN[M][h];
        part += __shfl_xor_sync(TASER_FULL_MASK, part, 4);
        part += __shfl_xor_sync(TASER_FULL_MASK, part, 8);   // at most 2^30 in magnitude
        const int other = __shfl_xor_sync(TASER_FULL_MASK, part, 16);
        if (tq == 0 && vnn0 - part <= other) fl |= TASER_FLAG_LNN_SIGN;
      }
      // The old iterate as B blocks: 8 x 8 blocks of codes, transposed.
      uint32_t pk[KT][NT][2];
#pragma unroll
      for (int kt = 0; kt < KT; ++kt)
#pragma unroll
        for (int n = 0; n < NT; ++n)
#pragma unroll
          for (int q = 0; q < 2; ++q) {
            const int kb = 2 * kt + q;
            if (kt <= C::ktmax(n) && kb <= n)
              pk[kt][n][q] = movmatrix_trans(
                  __byte_perm(m[kb / 2][n][2 * (kb % 2)], m[kb / 2][n][2 * (kb % 2) + 1], 0x5410));
          }
      int v[MT][NT][4];
#pragma unroll
      for (int n = NT - 1; n >= 0; --n) {
        // Codes to FP16: 0x6400 | x is 1024 + x for x < 1024; the high part's sign bit is
        // flipped to an offset of 64.
        uint32_t bh[KT][2], bl[KT][2];
#pragma unroll
        for (int kt = 0; kt <= C::ktmax(n); ++kt)
#pragma unroll
          for (int q = 0; q < 2; ++q) {
            bh[kt][q] = bl[kt][q] = 0u;
            if (2 * kt + q <= n) {
              const uint32_t p = pk[kt][n][q];
              bh[kt][q] = hadd2_bits(((p >> 7) & 0x007f007fu) ^ 0x64406440u, 0xe440e440u);   // - 1088
              bl[kt][q] = hadd2_bits((p & 0x007f007fu) ^ 0x64006400u, 0xe400e400u);          // - 1024
            }
          }
#pragma unroll
        for (int M = 0; M < MT; ++M) {
          if (!C::has_tile(M, n)) continue;
          float hh[4], xx[4], ll[4];
#pragma unroll
          for (int kt = 0; kt <= C::ktmax(n); ++kt) {
            if (kt == 0) {
              mma16816_c(hh, ah[M][0], bh[0], __uint_as_float(m[M][n][0]), __uint_as_float(m[M][n][1]),
                         __uint_as_float(m[M][n][2]), __uint_as_float(m[M][n][3]));
              mma16816_c(xx, ah[M][0], bl[0], fm, fm, fm, fm);
              mma16816_c(ll, al[M][0], bl[0], fm, fm, fm, fm);
            } else {
              mma16816<true>(hh, ah[M][kt], bh[kt]);
              mma16816<true>(xx, ah[M][kt], bl[kt]);
              mma16816<true>(ll, al[M][kt], bl[kt]);
            }
            mma16816<true>(xx, al[M][kt], bh[kt]);
          }
#pragma unroll
          for (int e = 0; e < 4; ++e) {
            v[M][n][e] = 0;
            if (!live(M, n, e)) continue;
            const uint32_t k0 = n == NT - 1 ? kN[M][e >> 1] : kRound;
            const int sh = (int)(__float_as_uint(xx[e]) * 128u + k0 + __float_as_uint(ll[e])) >> 14;
            int w = (int)(__float_as_uint(hh[e]) - kMagic) + sh;
            if ((n == 2 * M && e < 2) || (n == 2 * M + 1 && e >= 2)) w = (e & 1 ? lo1 : lo0) ? 0 : w;
            v[M][n][e] = fx_clamp(w, sat);
          }
        }
      }
      // Squared column norms (16 fraction bits; row N's codes have one bit less).
      uint32_t sn[2 * MT], own[1];
#pragma unroll
      for (int M = 0; M < MT; ++M)
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          uint32_t a = 0;
#pragma unroll
          for (int n = 0; n < NT; ++n)
#pragma unroll
            for (int p = 0; p < 2; ++p) {
              const int e = 2 * h + p;
              if (!live(M, n, e)) continue;
              const uint32_t sq = (uint32_t)(v[M][n][e] * v[M][n][e]);
              a += n == NT - 1 ? 4u * sq : sq;
            }
          sn[2 * M + h] = a;
        }
      row_sums<2 * MT>(sn, own, tq);   // each row's sum ends in one lane
      const uint32_t x = own[0];
      // Scale D_k LUT[.] 2^-sh of the owned row, sh - 13 in the low 4 bits.
      int cs = 0;
      if (x != 0u) {
        const int e = (31 - __clz(x)) & ~1;
        const uint32_t idx = e >= 9 ? x >> (e - 9) : x << (9 - e);
        cs = ((TASER_IN(idx, 2048) ? dq_own * (int)lut[idx] : 0) << 4) | (e >> 1);
      } else if (real_own) {
        fl |= TASER_FLAG_ZERO_COLUMN;
      }
#pragma unroll
      for (int M = 0; M < MT; ++M)
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          const int c4 = __shfl_sync(TASER_FULL_MASK, cs, (lane & 28) + 2 * M + h);
          const int sc = c4 >> 4, sh = 13 + (c4 & 15);
          const long long half = 1ll << (sh - 1);
#pragma unroll
          for (int n = 0; n < NT; ++n)
#pragma unroll
            for (int p = 0; p < 2; ++p) {
              const int e = 2 * h + p;
              if (!live(M, n, e)) continue;
              const long long prod = (long long)v[M][n][e] * sc + half;
              const int l = (int)__funnelshift_r((uint32_t)prod, (uint32_t)(prod >> 32), sh);
              m[M][n][e] = kMagic + (uint32_t)fx_clamp(l, sat);
            }
        }
    }

    // Outputs: decisions sign(L~_N,k) (sign(0) = +1), L~ as reals, flags.
    if (sat != 0) fl |= TASER_FLAG_SATURATED;
    const JobOut o = outs[cur];
    if (tq == 0) {
#pragma unroll
      for (int M = 0; M < MT; ++M)
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          const int k = 16 * M + g + 8 * h;
          if (k < N - 1 && TASER_IN(k, N - 1))
            o.s[k] = (int)(m[M][NT - 1][2 * h] - kMagic) >= 0 ? int8_t(1) : int8_t(-1);
        }
    }
    if (o.L != nullptr) {
#pragma unroll
      for (int M = 0; M < MT; ++M)
#pragma unroll
        for (int n = 0; n < NT; ++n)
#pragma unroll
          for (int e = 0; e < 4; ++e) {
            const int k = 16 * M + g + 8 * (e >> 1), i = 8 * n + 2 * tq + (e & 1);
            const int rr = bucket_to_real(i, N, NB);
            if (rr < 0 || k >= N - 1 || !TASER_IN(rr * N + k, N * N)) continue;
            const float unit = i == NB ? 1.f / 128.f : 1.f / 256.f;
            o.L[rr * N + k] = live(M, n, e) ? (float)(int)(m[M][n][e] - kMagic) * unit : 0.f;
          }
      for (int rr = lane; rr < N; rr += 32)
        if (TASER_IN(rr * N + N - 1, N * N)) o.L[rr * N + N - 1] = rr == N - 1 ? (float)lnn * (1.f / 32.f) : 0.f;
    }
#pragma unroll
    for (int ofs = 16; ofs > 0; ofs >>= 1) fl |= __shfl_xor_sync(TASER_FULL_MASK, fl, ofs);
    if (lane == 0 && o.flag != nullptr && fl) *o.flag |= fl;
    __syncwarp();  // the record of this job is consumed before it is reused
    cur ^= 1;
    have = have_next;
  }
}

template <int NB, class Src>
static cudaError_t launch_fxt(const Src& src, int64_t jobs, int blocks_per_sm, int slot_floats, cudaStream_t st) {
  const size_t smem = (kFxLutInts + (size_t)TctCfg<NB>::WARPS * (slot_floats + kTcRecFloats)) * sizeof(float);
  return launch_persistent(detect_fxt_kernel<NB, Src>, smem, src, jobs, blocks_per_sm, st, slot_floats);
}

cudaError_t detect_fx14(int64_t batch, int N, const float* Tt, const float* D, const float* tau, int t_max, float* L,
                        int8_t* s, uint32_t* flags, cudaStream_t st) {
  const Queue q{};
  const DenseSource src{batch, 0, N, t_max, Tt, D, tau, L, s, flags, nullptr};
  switch (bucket_of(N)) {
    case 8:
    case 16:
      return launch_fxt<16>(src, batch, 0, tc_slot_floats(N), st);
    case 32:
      return launch_fxt<32>(src, batch, 0, tc_slot_floats(N), st);
    default:
      return launch_fx14<64, false>(batch, N, t_max, Tt, D, tau, L, s, flags, q, 0, nullptr, nullptr, nullptr,
                                    nullptr, st);
  }
}

cudaError_t detect_fx14_queue(int nb, const Queue& q, int blocks_per_sm, const float* T_pool, const float* D_pool,
                              const float* tau, float* L_pool, int8_t* s_pool, uint32_t* flags, cudaStream_t st) {
  const QueueSource src{q, 1, T_pool, D_pool, tau, L_pool, s_pool, flags};
  switch (nb) {
    case 8:
    case 16:
      return launch_fxt<16>(src, -1, blocks_per_sm, tc_slot_floats(nb + 1), st);
    case 32:
      return launch_fxt<32>(src, -1, blocks_per_sm, tc_slot_floats(33), st);
    default:
      return launch_fx14<64, true>(0, 0, 0, nullptr, nullptr, tau, nullptr, nullptr, flags, q, blocks_per_sm, T_pool,
                                   D_pool, L_pool, s_pool, st);
  }
}

}  // namespace taser

TASER_DEBUG_COLLECTOR(detect_fx14)
