// Job plumbing of the persistent one-warp-per-instance tensor-core kernels (detect_tc.cu,
// detect_fx14.cu): where a warp's next job comes from, its asynchronous staging into shared
// memory, and the tiles of the transposed triangular product V^T = L~^T + T^ L~^T.
#pragma once

#include <type_traits>

#include "mma_tc.cuh"

namespace taser {

__device__ __forceinline__ void cp_async4(void* smem_dst, const void* gsrc) {
  const unsigned d = (unsigned)__cvta_generic_to_shared(smem_dst);
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(d), "l"(gsrc) : "memory");
}

__device__ __forceinline__ void cp_async16(void* smem_dst, const void* gsrc) {
  const unsigned d = (unsigned)__cvta_generic_to_shared(smem_dst);
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(d), "l"(gsrc) : "memory");
}

// Slot layout of a staged job: T~ at slot + shift (shift = 0..3, see stage_job), D at
// slot + N^2 + 4, tau after D.  Returns the floats a slot needs for size N.
__host__ __device__ constexpr int tc_slot_floats(int N) { return ((N * N + 4 + N + 1) + 3) & ~3; }

// Stage T~ (N x N), D (N) and tau of one job into the warp's shared slot.  An instance's T~
// starts at any 4-byte boundary (N^2 floats per instance), so it is placed `shift` floats
// into the slot, shift = (address / 4) mod 4: then its 16-byte groups in global and shared
// memory coincide, and all but at most 3 + 3 of the N^2 floats move as 16-byte copies
// (9 instead of 35 copies per lane at N = 33).  Returns shift.  (Staging only the lower
// triangle was measured: the DRAM bytes stayed at 4,490 per instance, because rows of
// N = 33 floats are not aligned to the 128-byte lines, so nearly every line still holds a
// part of the triangle; the triangle walk only added instructions.)
// A debug build checks every copy against the instance's N^2 floats and the slot's
// slot_floats.
__device__ __forceinline__ int stage_job(float* slot, const Job& jb, int lane, int slot_floats) {
  const int N = jb.N, nn = N * N;
  const int shift = (int)((reinterpret_cast<uintptr_t>(jb.T) >> 2) & 3u);
  float* dst = slot + shift;
  const int head = (4 - shift) & 3;
  const int nvec = nn > head ? (nn - head) >> 2 : 0;
  const int tail0 = head + 4 * nvec;
  if (lane < head && lane < nn && TASER_IN(shift + lane, slot_floats)) cp_async4(dst + lane, jb.T + lane);
  for (int v = lane; v < nvec; v += 32)
    if (TASER_IN(head + 4 * v + 3, nn) && TASER_IN(shift + head + 4 * v + 3, slot_floats))
      cp_async16(dst + head + 4 * v, jb.T + head + 4 * v);
  for (int i = tail0 + lane; i < nn; i += 32)
    if (TASER_IN(shift + i, slot_floats)) cp_async4(dst + i, jb.T + i);
  float* dd = slot + nn + 4;
  for (int i = lane; i < N; i += 32)
    if (TASER_IN(nn + 4 + i, slot_floats)) cp_async4(dd + i, jb.D + i);
  if (lane == 0 && TASER_IN(nn + 4 + N, slot_floats)) cp_async4(dd + N, jb.tau);
  asm volatile("cp.async.commit_group;" ::: "memory");
  return shift;
}

// Instances at a fixed stride (the dense batch of taser_detect).
struct DenseSource {
  int64_t batch, stride;
  int N, t_max;
  const float *Tt, *Dg, *tau;
  float* L;
  int8_t* s;
  uint32_t* flags;
  double* obj;   // objective trace [batch][t_max + 1] (monitored launches), or nullptr
  __device__ __forceinline__ bool get(int64_t k, Job& jb, double*& ob) const {  // k-th instance of this warp
    const int64_t inst = (int64_t)blockIdx.x * 4 + (threadIdx.x >> 5) + k * stride;
    if (inst >= batch) return false;
    jb = dense_job(inst, N, t_max, Tt, Dg, tau, L, s, flags);
    ob = obj != nullptr ? obj + inst * (int64_t)(t_max + 1) : nullptr;
    return true;
  }
};

// Items of one bucket's queue, popped `pop` at a time per warp.
struct QueueSource {
  Queue q;
  int pop;
  const float *T_pool, *D_pool, *tau;
  float* L_pool;
  int8_t* s_pool;
  uint32_t* flags;
};

template <class Src>
struct Cursor;

template <>
struct Cursor<DenseSource> {
  int64_t k = 0;
  __device__ __forceinline__ bool next(const DenseSource& src, Job& jb, double*& ob, int) {
    return src.get(k++, jb, ob);
  }
};

template <>
struct Cursor<QueueSource> {
  int base = 0, left = 0;
  __device__ __forceinline__ bool next(const QueueSource& src, Job& jb, double*& ob, int lane) {
    ob = nullptr;
    if (left == 0) {
      int b = 0;
      if (lane == 0) b = src.q.pop(src.pop);
      base = __shfl_sync(TASER_FULL_MASK, b, 0);
      left = src.pop;
    }
    const int pos = base++;
    --left;
    if (pos >= src.q.count()) {
      left = 0;
      base = 1 << 30;
      return false;
    }
    const int idx = src.q.item_at(pos);
    const taser_item it = src.q.items[idx];
    jb = item_job(it, idx, src.T_pool, src.D_pool, src.tau, src.L_pool, src.s_pool, src.flags);
    return true;
  }
};

// Shared-memory floats per warp after its staging slot: two job records (JobOut below).
constexpr int kTcRecFloats = 24;

template <int NB>
struct TctCfg {
  static constexpr int MT = NB / 16;      // m-tiles over the columns k of L~
  static constexpr int KT = NB / 16;      // k-tiles over j
  static constexpr int NT = NB / 8 + 1;   // n-tiles over the rows i of L~; the last holds row N (i = NB)
  static constexpr int WARPS = 4;
  // Tile (M, n) holds V^T[k][i] for k in 16M..16M+15, i in 8n..8n+7; rows i < k are zero.
  __host__ __device__ static constexpr bool has_tile(int M, int n) { return n >= 2 * M; }
  // k-tiles of j that reach n-tile n (L~^T[j][i] = 0 for j > i).
  __host__ __device__ static constexpr int ktmax(int n) { return n / 2 < KT - 1 ? n / 2 : KT - 1; }
};

__device__ __forceinline__ uint32_t movmatrix_trans(uint32_t x) {
  uint32_t y;
  asm volatile("movmatrix.sync.aligned.m8n8.trans.b16 %0, %1;" : "=r"(y) : "r"(x));
  return y;
}

// Sums of R = 2 MT per-row partials over the 4 lanes of a row group (tq = lane & 3), transposed:
// lane tq ends with the totals of rows r = 4u + tq (R = 2: row tq & 1, in two lanes), so the
// scalar work of a row (its norm, scale, flag) is done once instead of in 4 lanes, and the sums
// take R - 1 shuffles instead of 2 R.  Each total is (p0 + p1) + (p2 + p3), whichever the lane.
template <int R, typename V>
__device__ __forceinline__ void row_sums(const V (&p)[R], V (&own)[R < 4 ? 1 : R / 4], int tq) {
  V a[R / 2];
#pragma unroll
  for (int u = 0; u < R / 2; ++u) {
    const V keep = tq & 1 ? p[2 * u + 1] : p[2 * u], send = tq & 1 ? p[2 * u] : p[2 * u + 1];
    a[u] = keep + __shfl_xor_sync(TASER_FULL_MASK, send, 1);
  }
  if constexpr (R == 2) {
    own[0] = a[0] + __shfl_xor_sync(TASER_FULL_MASK, a[0], 2);
  } else {
#pragma unroll
    for (int u = 0; u < R / 4; ++u) {
      const V keep = tq & 2 ? a[2 * u + 1] : a[2 * u], send = tq & 2 ? a[2 * u] : a[2 * u + 1];
      own[u] = keep + __shfl_xor_sync(TASER_FULL_MASK, send, 2);
    }
  }
}

// The row index (M, h) -> r = 2M + h that row_sums leaves in this lane, u-th of it.
template <int R>
__device__ __forceinline__ int owned_row(int u, int tq) { return R == 2 ? tq & 1 : 4 * u + tq; }
// Column k of L~ that row r of lane group g is: 16M + g + 8h.
__device__ __forceinline__ int row_column(int r, int g) { return 8 * r + g; }

// Persistent launch of `kern` for a job source: `blocks_per_sm` blocks of 4 warps per SM (as many
// as fit if <= 0), fewer if the jobs are fewer (jobs < 0: unknown, a queue).
template <class Kern, class Src, class... Args>
static cudaError_t launch_persistent(Kern kern, size_t smem, Src src, int64_t jobs, int blocks_per_sm,
                                     cudaStream_t st, Args... args) {
  int dev = 0, sms = 0, fit = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  if (e == cudaSuccess && smem > 48 * 1024)
    e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e == cudaSuccess) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&fit, kern, 128, smem);
  if (e != cudaSuccess) return e;
  const int per_sm = blocks_per_sm > 0 && blocks_per_sm < fit ? blocks_per_sm : (fit > 0 ? fit : 1);
  const int64_t need = (jobs + 3) / 4;
  const int64_t resident = (int64_t)sms * per_sm;
  const int64_t blocks = jobs >= 0 && need < resident ? need : resident;
  if constexpr (std::is_same_v<Src, DenseSource>) src.stride = blocks * 4;
  kern<<<(unsigned)blocks, 128, smem, st>>>(src, args...);
  return cudaGetLastError();
}

}  // namespace taser
