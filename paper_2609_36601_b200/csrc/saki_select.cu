// Placement controls (Appendix "placement_control"): per trajectory, choose m = number of corrected
// valid positions, valid positions for the teacher-mode loss: uniformly (Random-TM) or without
// replacement with the positions' TV as weights (TV-Weighted-TM: the m smallest exponential-race keys
// -log U / TV, uniform fill if fewer than m positions have positive TV).
//
// One block per trajectory.  A position's key is a 64-bit integer that orders like
// (tier, float64 key value): bit 63 is the tier (0: weighted key, or any key in Random mode; 1: the
// uniform of a zero-TV position, used by the fill), the rest are the bits of the non-negative double.
// The m-th smallest key is found by a radix select, a byte per pass; equal keys go to the lower index by an
// ordered count.  The call touches N scalars, so what counts is the chain of steps in a block: the keys (a
// Philox call and a logarithm each) are formed once and kept in shared memory (a trajectory of more than KEEP
// positions recomputes them in every pass), the bin that holds the m-th key is found by a warp's scan of the
// histogram, and the passes stop as soon as a bin is chosen as a whole (after three of the eight as a rule).
// 16 trajectories of 512: 40 -> 10 us.
#include "saki_common.cuh"
#include <math_constants.h>

namespace saki {

constexpr int ST = 256;                              // threads per block
constexpr unsigned long long KEY_INVALID = ~0ull;    // not a valid position: never chosen (m <= number of valid positions)

__device__ __forceinline__ bool sel_valid(const SelectParams& P, int64_t i) {
  if (P.mask && P.mask[i] == 0) return false;
  const uint32_t unusable = SAKI_ROW_NONFINITE | SAKI_ROW_BAD_ID | SAKI_ROW_TIMEOUT | SAKI_ROW_NOT_COMPUTED;
  return !(P.rollout_status && (P.rollout_status[i] & unusable));
}
__device__ __forceinline__ unsigned long long sel_key(const SelectParams& P, int64_t i) {
  if (!sel_valid(P, i)) return KEY_INVALID;
  const double u = scalar_uniform(P.seed, P.row_offset + (uint64_t)i, STAGE_SELECT);
  if (P.mode == SAKI_SELECT_TV_WEIGHTED) {
    const double d = (double)P.tv[i];
    if (d > 0.0 && d < CUDART_INF) return (unsigned long long)__double_as_longlong(-log(u) / d);
    return (1ull << 63) | (unsigned long long)__double_as_longlong(u);
  }
  return (unsigned long long)__double_as_longlong(u);
}

// sum over the block, returned to every thread; `sh` holds ST/32 + 1 ints
__device__ __forceinline__ int block_sum_i(int v, int* sh) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  __syncthreads();
  if (lane == 0) sh[warp] = v;
  __syncthreads();
  int a = 0;
  for (int w = 0; w < ST / 32; ++w) a += sh[w];
  return a;
}

constexpr int KEEP = 4096;     // keys in shared memory (32 KB)

__global__ void __launch_bounds__(ST) select_kernel(const SelectParams P) {
  __shared__ unsigned long long keys[KEEP];
  __shared__ int hist[256];      // ST == 256 bins
  __shared__ int sh[ST / 32 + 1];
  __shared__ int pick[3];        // the chosen bin of a pass, the count below it, the count in it
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  launch_dependents();
  wait_for_predecessor();
  for (int64_t b = blockIdx.x; b < P.B; b += gridDim.x) {
    const int64_t lo = P.seq_start[b], hi = P.seq_start[b + 1];
    const bool keep = hi - lo <= KEEP;
    // the keys, and m = corrected valid positions of the trajectory
    int cnt = 0;
    for (int64_t i = lo + tid; i < hi; i += ST) {
      if (keep) {
        const unsigned long long k = sel_key(P, i);
        keys[i - lo] = k;
        cnt += (k != KEY_INVALID && P.corrected[i] != 0) ? 1 : 0;
      } else cnt += (sel_valid(P, i) && P.corrected[i] != 0) ? 1 : 0;
    }
    auto key = [&](int64_t i) { return keep ? keys[i - lo] : sel_key(P, i); };
    const int m = block_sum_i(cnt, sh);
    if (tid == 0 && P.m) P.m[b] = m;
    if (m == 0) {
      for (int64_t i = lo + tid; i < hi; i += ST) P.selected[i] = 0;
      continue;
    }
    // radix select of the m-th smallest key: after the passes, the keys below `prefix` (`below` of them) are chosen, and
    // of those that agree with it on `high_mask` the first m - below
    unsigned long long prefix = 0ull, high_mask = 0ull;
    int below = 0;
    for (int shift = 56; shift >= 0; shift -= 8) {
      hist[tid] = 0;
      __syncthreads();
      for (int64_t i = lo + tid; i < hi; i += ST) {
        const unsigned long long k = key(i);
        if ((k & high_mask) == prefix) atomicAdd(&hist[(int)((k >> shift) & 0xffull)], 1);
      }
      __syncthreads();
      if (warp == 0) {           // eight bins per lane
        int h[8], sum = 0;
#pragma unroll
        for (int q = 0; q < 8; ++q) { h[q] = hist[lane * 8 + q]; sum += h[q]; }
        int acc = sum;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
          const int up = __shfl_up_sync(0xffffffffu, acc, o);
          if (lane >= o) acc += up;
        }
        const unsigned reach = __ballot_sync(0xffffffffu, below + acc >= m);      // (the last lane's does)
        if (lane == __ffs(reach) - 1) {
          int a = below + acc - sum, q = 0;
#pragma unroll
          for (int z = 0; z < 7; ++z) if (q == z && a + h[z] < m) { a += h[z]; ++q; }
          int in_bin = 0;
#pragma unroll
          for (int z = 0; z < 8; ++z) if (q == z) in_bin = h[z];
          pick[0] = lane * 8 + q; pick[1] = a; pick[2] = in_bin;
        }
      }
      __syncthreads();
      prefix |= (unsigned long long)pick[0] << shift;
      high_mask |= 0xffull << shift;
      below = pick[1];
      if (below + pick[2] == m) break;       // the whole bin is chosen
    }
    int need = m - below;
    for (int64_t base = lo; base < hi; base += ST) {
      const int64_t i = base + tid;
      const unsigned long long k = i < hi ? key(i) : KEY_INVALID;
      const bool eq = (k & high_mask) == prefix && k != KEY_INVALID;
      // ordered rank of this thread among the chunk's keys of the bin
      const unsigned bal = __ballot_sync(0xffffffffu, eq);
      __syncthreads();
      if (lane == 0) sh[warp] = __popc(bal);
      __syncthreads();
      int before = 0, total = 0;
      for (int w = 0; w < ST / 32; ++w) { if (w < warp) before += sh[w]; total += sh[w]; }
      const int rank = before + __popc(bal & ((1u << lane) - 1u));
      if (i < hi) P.selected[i] = ((k & high_mask) < prefix || (eq && rank < need)) ? 1 : 0;
      need = max(0, need - total);
    }
    __syncthreads();
  }
}

cudaError_t launch_select(const SelectParams& p, cudaStream_t st, int* n_launches) {
  if (p.B <= 0) return cudaSuccess;
  const int grid = (int)std::min<int64_t>(p.B, 1 << 16);
  ++*n_launches;
  return launch_pdl(select_kernel, dim3((unsigned)grid), ST, 0, st, true, p);
}

}  // namespace saki
