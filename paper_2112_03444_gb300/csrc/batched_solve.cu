// Standalone batched dense complex solve A x = b: the fused linear solver of
// paper Sec. 6 (LU with partial pivoting on the augmented matrix [A b] and
// the triangular solve in one kernel, data kept in registers), measured on
// its own in the paper's Fig. 3 (1000 matrices of 4x4 to 20x20 against
// cuBLAS and MAGMA).  It is the same register-resident elimination the
// tracker runs per path (gj_solve in hc_device.cuh): one lane group per
// system, row i of [A | b] in lane i, Gauss-Jordan with partial pivoting, so
// the back substitution is folded into the elimination.
//
// The groups of a warp run the elimination in step (make_group): with group masks
// each ran it on its own (batch 100,000, FP32, together with the staging below:
// n = 4 12.6 -> 8.5 us, n = 8 31 -> 28, n = 20 327 -> 281; batch 1000, n = 8, device time
// of captured calls 4.1 -> 3.1; a call by itself takes 8 to 10 us either way, the host's).
//
// Data path: a block's systems are contiguous in A (row-major, system after
// system), so the block stages them through shared memory with consecutive
// threads reading consecutive complex numbers (coalesced), then each lane
// takes its row from shared memory; solutions go out the same way.
#include <atomic>
#include <cstdint>

#include <cuda_runtime.h>

#include "hc.h"
#include "hc_device.cuh"
#include "kernels.cuh"

namespace {

using hc::cx;

constexpr int kThreads = 128;

// Lanes per system with one row per lane; D divides them (rows per lane: D, or
// fewer where N leaves the last ones empty).
//
// FP64 is bound by its pipe (91 % busy at n = 13, batch 40,000, one row per lane),
// and 38 % of its instructions are the reciprocals of the pivots, which cost a
// warp the same whether its lanes belong to two systems or to eight.  With several
// rows per lane a warp's reciprocals serve D times the systems: batch 100,000, us,
// one row -> D rows: n = 5 289 -> 141, n = 8 494 -> 361, n = 12 1763 -> 977 (D = 4),
// n = 13 1981 -> 1594, n = 20 7550 -> 6475 (D = 2; four rows of 13 or more entries
// leave the registers).  Where they pay is decided by several_rows.  FP32 is bound
// by issue slots and its row updates: one row per lane (n = 20, batch 100,000: 281
// against 343 with two rows and two-wide updates).
template <int N, class R>
constexpr int wide_rows() {
  return sizeof(R) == 4 || N > 24 ? 1 : N > 12 || N <= 2 ? 2 : 4;
}
template <int N, int D>
constexpr int solve_lanes() {
  return (N <= 4 ? 4 : N <= 8 ? 8 : N <= 16 ? 16 : 32) / D;
}

// A block of D rows per lane holds D times the systems and takes longer, so what
// counts is how many rounds (blocks on the busiest SM) either form needs: 6 rounds of
// one-row blocks at n = 20 take 265 us, the 3 rounds of two-row blocks that hold the
// same systems 316 (the hardware gives some SM a fourth).  round_cost: a round of
// D-row blocks in percent of a round of one-row blocks, fitted to 60 batches of 1 to
// 34 rounds at every n; the sizes that fill their lanes (4, 8, 16) and n = 7 have the
// cheaper one-row rounds.  A third of a round is the wide form's longer latency.
constexpr int round_cost(int n) {
  return n <= 2                     ? 130
         : n == 4 || n == 7 || n == 8 ? 265
         : n <= 12                    ? 200
         : n <= 15                    ? 150
         : n <= 16                    ? 160
         : n <= 20                    ? 165
                                      : 175;
}
// Against one row per lane everywhere (us, one row / rule): n = 8, batch 9,728 48 / 39,
// n = 10, 3,648 49 / 41, n = 20, 2,432 178 / 161; where the other form is taken: n = 20,
// 3,648 265 (D rows 316), n = 24, 3,648 354 (D rows 435).
template <int N, class R>
bool several_rows(int64_t batch, int sms) {
  constexpr int D = wide_rows<N, R>();
  if constexpr (D == 1) return false;
  const int64_t one = kThreads / solve_lanes<N, 1>(), wide = kThreads / solve_lanes<N, D>();
  // (a last one-row block that is half empty costs half a round)
  const int64_t r1 = (batch - one / 2 + one * sms - 1) / (one * sms);
  const int64_t blocks = (batch + wide - 1) / wide;
  int64_t r = (blocks + sms - 1) / sms;
  // an odd round that is nearly full: the blocks beyond an even number per SM are not
  // spread evenly, and some SM gets two of them
  if (r > 2 && r % 2 == 1 && 10 * (r * sms - blocks) < 3 * sms) ++r;
  return 100 * r1 > round_cost(N) * r + 35;
}

// Shared memory of one block: the staged augmented matrices [G][N][N + 1],
// then per group the two pivot-row buffers and the solution scatter buffer.
template <int N, class R, int D>
constexpr size_t solve_smem_bytes() {
  constexpr int L = solve_lanes<N, D>(), G = kThreads / L;
  constexpr int S = (N + 2) & ~1;  // entries per pivot buffer (gj_solve, NR = 1)
  return sizeof(cx<R>) * ((((size_t)G * N * (N + 1) + 1) & ~(size_t)1) + (size_t)G * 2 * S +
                          (size_t)G * N);
}

// Blocks per SM to compile for (0: as the registers fall).  n = 8 in FP64 by six
// registers misses the fifth block, which a batch of five blocks per SM needs.
template <int N, class R, int D>
constexpr int min_blocks() {
  return sizeof(R) == 8 && D == 1 && N == 8 ? 5 : 0;
}

// MEET: the groups of a warp in step; otherwise each group runs by itself and those
// past the batch not at all (a few FP32 systems, see solve_dispatch).
template <int N, class R, int D, bool MEET>
__global__ void __launch_bounds__(kThreads, min_blocks<N, R, D>())
    batched_solve_kernel(int64_t batch, const cx<R>* __restrict__ A, const cx<R>* __restrict__ b,
                         cx<R>* __restrict__ x, int32_t* __restrict__ info) {
  constexpr int L = solve_lanes<N, D>(), G = kThreads / L, W = N + 1;
  constexpr int ROWS = (N + L - 1) / L;
  constexpr int S = (N + 2) & ~1;
  static_assert(MEET || ROWS == 1, "groups apart: one row per lane");
  extern __shared__ __align__(16) unsigned char smem[];
  cx<R>* stage = reinterpret_cast<cx<R>*>(smem);
  cx<R>* pvbuf = stage + (((size_t)G * N * W + 1) & ~(size_t)1);
  cx<R>* sbuf = pvbuf + (size_t)G * 2 * S;
  const hc::Group g = hc::make_group<L, MEET>();
  const int grp = threadIdx.x / L;
  cx<R>* pv = pvbuf + grp * 2 * S;
  cx<R>* sb = sbuf + grp * N;
  for (int64_t base = (int64_t)blockIdx.x * G; base < batch; base += (int64_t)gridDim.x * G) {
    const int cnt = (int)((batch - base) < G ? (batch - base) : G);
    // Coalesced staging of the block's matrices and right-hand sides: row r of the
    // block (N entries) lands at r W, so entry idx at idx + idx / N.
    const cx<R>* Ab = A + base * N * N;
#pragma unroll 4
    for (int idx = threadIdx.x; idx < cnt * N * N; idx += kThreads)
      stage[idx + (unsigned)idx / N] = Ab[idx];
    const cx<R>* bb = b + base * N;
    for (int idx = threadIdx.x; idx < cnt * N; idx += kThreads) stage[idx * W + N] = bb[idx];
    __syncthreads();
    // FP64: a warp without a system solves nothing.  In one with some, the groups
    // past the count take its last system again and the lanes past the last row ones:
    // their results go nowhere, but a reciprocal of zero takes the division's slow
    // path for the whole warp.  (us, with all groups of a block on zero rows -> now,
    // n = 9: batch 1000 19.6 -> 17.7, one system more than a block per SM 30.5 -> 20.0.
    // FP32 is bound by issue slots and pays more for the branch than for the rows.)
    constexpr bool FILL = sizeof(R) == 8;
    const bool live = grp < cnt;
    const bool work = MEET ? !FILL || (threadIdx.x & ~31) / L < cnt : live;
    const int sys = FILL && !live ? cnt - 1 : grp;
    cx<R> a[ROWS][W];
#pragma unroll
    for (int q = 0; q < ROWS; ++q)
#pragma unroll
      for (int j = 0; j < W; ++j)
        a[q][j] = (FILL || live) && g.gl + q * L < N ? stage[(sys * N + g.gl + q * L) * W + j]
                                                     : hc::mk<R>(R(FILL ? 1 : 0), R(0));
    __syncthreads();  // the stage is free for the next round once every row is in registers
    if (work) {
      cx<R> sol[ROWS];
      int col[ROWS];
      bool ok;
      if constexpr (ROWS == 1)
        ok = hc::gj_solve<N, 1, R, L, MEET>(g, a[0], sol, col[0], pv);
      else
        ok = hc::gj_solve_rows<N, L, ROWS, R>(g, a, sol, col, pv);
#pragma unroll
      for (int q = 0; q < ROWS; ++q)
        if (col[q] >= 0) sb[col[q]] = sol[q];
      __syncwarp(g.meet);
      if (live) {
#pragma unroll
        for (int q = 0; q < ROWS; ++q)
          if (g.gl + q * L < N) x[(base + grp) * N + g.gl + q * L] = sb[g.gl + q * L];
        if (g.gl == 0 && info) info[base + grp] = ok ? 0 : 1;
      }
      __syncwarp(g.meet);
    }
  }
}

constexpr int kMaxDevices = 64;

struct SolveRef {
  const void* fn;
  size_t smem;
  int per_block, per_sm;  // systems per block, resident blocks per SM (0: refused)
};

// The occupancy query costs as much as the launch of a small batch: once per
// kernel and device.
template <int N, class R, int D, bool MEET = true>
SolveRef solve_ref(int dev) {
  static std::atomic<int> known[kMaxDevices];
  SolveRef k{reinterpret_cast<const void*>(&batched_solve_kernel<N, R, D, MEET>),
             solve_smem_bytes<N, R, D>(), kThreads / solve_lanes<N, D>(),
             dev < kMaxDevices ? known[dev].load(std::memory_order_acquire) : 0};
  // (the attribute belongs to the context, which a program may have replaced)
  if (k.smem > 48 * 1024 &&
      cudaFuncSetAttribute(k.fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)k.smem) !=
          cudaSuccess) {
    k.per_sm = 0;
    return k;
  }
  if (k.per_sm > 0) return k;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&k.per_sm, k.fn, kThreads, k.smem) !=
      cudaSuccess)
    k.per_sm = 0;
  else if (k.per_sm < 1)
    k.per_sm = 1;
  if (dev < kMaxDevices) known[dev].store(k.per_sm, std::memory_order_release);
  return k;
}

template <class R, int N = 1>
SolveRef solve_dispatch(int n, int64_t batch, int sms, int dev) {
  if constexpr (N > 32) {
    return SolveRef{nullptr, 0, 0, 0};
  } else {
    if (n == N) {
      if (several_rows<N, R>(batch, sms)) return solve_ref<N, R, wide_rows<N, R>()>(dev);
      // A few FP32 systems: the group-wide maximum of one group is faster than the
      // butterfly that several share, and the other warps stay out of the way (one
      // system, device us, in step / apart: n = 8 2.8 / 2.6, n = 16 4.2 / 3.7, n = 32
      // 7.9 / 7.4; two systems: n = 8 2.8 / 3.2, n = 16 4.1 / 4.8, n = 32 8.2 / 7.9).
      if constexpr (sizeof(R) == 4)
        if (batch < (solve_lanes<N, 1>() == 32 ? 4 : 2)) return solve_ref<N, R, 1, false>(dev);
      return solve_ref<N, R, 1>(dev);
    }
    return solve_dispatch<R, N + 1>(n, batch, sms, dev);
  }
}

}  // namespace

extern "C" hc_status hc_batched_solve(int32_t n, int64_t batch, int32_t fp32, const void* A,
                                      const void* b, void* x, int32_t* info, void* stream) {
  if (n < 1 || n > 32 || batch < 0 || (batch > 0 && (!A || !b || !x)) || (fp32 != 0 && fp32 != 1)) {
    hc::set_last_error("hc_batched_solve: n must be 1..32, batch >= 0, A, b, x non-null");
    return HC_ERR_INVALID;
  }
  if (batch == 0) return HC_OK;
  cudaGetLastError();
  int dev = 0, sms = 0;
  if (cudaGetDevice(&dev) != cudaSuccess ||
      cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) {
    hc::set_last_error("hc_batched_solve: device query failed");
    return HC_ERR_CUDA;
  }
  const SolveRef k =
      fp32 ? solve_dispatch<float>(n, batch, sms, dev) : solve_dispatch<double>(n, batch, sms, dev);
  if (!k.fn) {
    hc::set_last_error("hc_batched_solve: no kernel for this size");
    return HC_ERR_UNSUPPORTED;
  }
  if (k.per_sm < 1) {
    hc::set_last_error("hc_batched_solve: shared-memory attribute or occupancy query refused");
    return HC_ERR_CUDA;
  }
  // one wave of resident blocks at most; each block strides over the batch
  const int64_t want = (batch + k.per_block - 1) / k.per_block;
  const int64_t cap = (int64_t)k.per_sm * sms;
  const unsigned grid = (unsigned)(want < cap ? want : cap);
  void* args[] = {&batch, &A, &b, &x, &info};
  if (cudaLaunchKernel(k.fn, dim3(grid), dim3(kThreads), args, k.smem,
                       static_cast<cudaStream_t>(stream)) != cudaSuccess) {
    hc::set_last_error("hc_batched_solve: launch failed");
    return HC_ERR_CUDA;
  }
  return HC_OK;
}
