// Proposal utility: x ~ softmax(s / tau) by Gumbel-max, key_v = s_v / tau - log(-log u_v) in float64, u_v from word v % 4
// of Philox block v / 4.
//
// A float64 key costs two logarithms, and all but a few keys are hopeless: every element gets a float32 UPPER BOUND of
// its key, and only those whose bound reaches the best exact key are evaluated in float64, so the result is the argmax of
// the float64 keys.  The bound: with v = 1 - u, -log u >= v + v^2/2, so the Gumbel term is at most -log(v + v^2/2), nearly
// exact where it is large (v small); v is taken from the upper 23 bits of the word, rounded down.  Per element that
// leaves a quarter of a Philox block (ten rounds of two wide multiplications and two xors: the integer pipe is the
// bound), one lg2 and a few float operations; the row is read once.
#include "saki_device.cuh"
#include <cooperative_groups.h>

namespace cg = cooperative_groups;

namespace saki {

namespace {

constexpr int PT = 256, PWARPS = PT / 32, PROPOSE_CS = 8;

struct ProposeShared {
  float ub[PWARPS];
  int blk[PWARPS];
  double key[PWARPS];
  int idx[PWARPS];
  double block_key;      // read by the other blocks of the cluster
  int block_idx;
  float block_ub;
  int block_blk;
};

template <typename T> struct Quad { float x[4]; };

// the four logits of Philox block blk (past the row's end: -inf)
template <typename T> __device__ __forceinline__ Quad<T> load_quad(const T* s, int blk, int V, bool vec) {
  Quad<T> q;
  if (vec && blk * 4 + 4 <= V) {
    if constexpr (sizeof(T) == 2) {
      const uint2 r = __ldg((const uint2*)(s + blk * 4));
      const float2 a = unpack_bf16x2(r.x), b = unpack_bf16x2(r.y);
      q.x[0] = a.x; q.x[1] = a.y; q.x[2] = b.x; q.x[3] = b.y;
    } else {
      const float4 r = __ldg((const float4*)(s + blk * 4));
      q.x[0] = r.x; q.x[1] = r.y; q.x[2] = r.z; q.x[3] = r.w;
    }
  } else {
#pragma unroll
    for (int k = 0; k < 4; ++k) q.x[k] = blk * 4 + k < V ? ld_as_float(s, blk * 4 + k) : -CUDART_INF_F;
  }
  return q;
}

__device__ __forceinline__ float lg2f(float x) {
  float y;
  asm("lg2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
// upper bound of the largest of a block's four keys, in units of log 2
template <typename T> __device__ __forceinline__ float bound(const Quad<T>& q, const uint32_t* w, float c) {
  float m = -CUDART_INF_F;
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    const float v = 1.99999988079071f - __uint_as_float(0x3f800000u | (w[k] >> 9));    // 1 - u, rounded down; may be 0
    m = fmaxf(m, fmaf(q.x[k], c, -lg2f(fmaf(v, 0.5f * v, v))));
  }
  return m;
}
__device__ __forceinline__ void better(double& key, int& idx, double k, int i) {
  if (k > key || (k == key && i < idx)) { key = k; idx = i; }
}
// the exact keys of a block's elements
template <typename T>
__device__ __noinline__ void exact_keys(const T* s, int blk, int V, double tau, uint64_t rid, uint64_t seed, double& key, int& idx) {
  uint32_t w[4];
  philox4x32_10((uint32_t)rid, (uint32_t)(rid >> 32), STAGE_PROPOSE, (uint32_t)blk, (uint32_t)seed, (uint32_t)(seed >> 32), w);
#pragma unroll 1
  for (int k = 0; k < 4; ++k) {
    const int v = blk * 4 + k;
    if (v >= V) break;
    const double u = ((double)(k == 0 ? w[0] : k == 1 ? w[1] : k == 2 ? w[2] : w[3]) + 0.5) * (1.0 / 4294967296.0);
    const double e = (double)ld_as_float(s, v) / tau - log(-log(u));
    if (e > -CUDART_INF) better(key, idx, e, v);
  }
}

// CS: blocks per row (1, or a cluster that shares the row)
template <typename T, int CS>
__global__ void __launch_bounds__(PT, 4) propose_kernel(const T* logits, int64_t ld, int64_t N, int V, double tau, float c,
                                                        uint64_t seed, uint64_t row_offset, int32_t* out) {
  __shared__ ProposeShared sh;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  int crank = 0;
  if constexpr (CS > 1) crank = (int)cg::this_cluster().block_rank();
  const int first = crank * PT + tid, step = PT * CS, nblk = (V + 3) / 4;
  for (int64_t row = blockIdx.x / CS; row < N; row += gridDim.x / CS) {
    const T* const s = logits + row * ld;
    const bool vec = ((uintptr_t)s & (4 * sizeof(T) - 1)) == 0;
    const uint64_t rid = row_offset + (uint64_t)row;
    // the two best blocks of this thread by their bounds, and the third best bound
    float b1 = -CUDART_INF_F, b2 = b1, b3 = b1;
    int i1 = 0, i2 = 0;
    Quad<T> next = load_quad(s, min(first, nblk - 1), V, vec);
#pragma unroll 1
    for (int blk = first; blk < nblk; blk += step) {
      const Quad<T> q = next;
      next = load_quad(s, min(blk + step, nblk - 1), V, vec);
      uint32_t w[4];
      philox4x32_10((uint32_t)rid, (uint32_t)(rid >> 32), STAGE_PROPOSE, (uint32_t)blk, (uint32_t)seed, (uint32_t)(seed >> 32), w);
      const float m = bound(q, w, c);
      b3 = fmaxf(b3, fminf(b2, m));
      const bool g1 = m > b1, g2 = m > b2;
      i2 = g1 ? i1 : (g2 ? blk : i2); b2 = g1 ? b1 : (g2 ? m : b2);
      i1 = g1 ? blk : i1; b1 = g1 ? m : b1;
    }
    // the block with the largest bound: its exact keys set the bar
    float mb = b1;
    int mi = i1;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      const float ob = __shfl_xor_sync(0xffffffffu, mb, o);
      const int oi = __shfl_xor_sync(0xffffffffu, mi, o);
      if (ob > mb) { mb = ob; mi = oi; }
    }
    if (lane == 0) { sh.ub[warp] = mb; sh.blk[warp] = mi; }
    __syncthreads();
#pragma unroll
    for (int w = 0; w < PWARPS; ++w) if (sh.ub[w] > mb) { mb = sh.ub[w]; mi = sh.blk[w]; }
    if constexpr (CS > 1) {
      if (tid == 0) { sh.block_ub = mb; sh.block_blk = mi; }
      cg::cluster_group cl = cg::this_cluster();
      cl.sync();
      for (int r = 0; r < CS; ++r) {
        const ProposeShared* const rs = cl.map_shared_rank(&sh, r);
        if (rs->block_ub > mb) { mb = rs->block_ub; mi = rs->block_blk; }
      }
    }
    double key = -CUDART_INF;
    int idx = 0x7fffffff;
    if (mb > -CUDART_INF_F) {
      double bar = -CUDART_INF;
      int bi = 0x7fffffff;
      exact_keys(s, mi, V, tau, rid, seed, bar, bi);                    // (every thread alike)
      // rounding of a bound: ~1e-7 of the scaled logit (the Gumbel term is within 33 of zero), and of lg2
      const float fb = (float)(bar * INV_LN2), thr = fb - (1e-4f + 1e-6f * (fminf(fabsf(fb), 1e30f) + 64.f));
      if (!(b1 < thr)) exact_keys(s, i1, V, tau, rid, seed, key, idx);
      if (!(b2 < thr) && b2 > -CUDART_INF_F) exact_keys(s, i2, V, tau, rid, seed, key, idx);
      if (!(b3 < thr) && b3 > -CUDART_INF_F) {                          // a third: every block of this thread that reaches the bar
#pragma unroll 1
        for (int blk = first; blk < nblk; blk += step) {
          uint32_t w[4];
          philox4x32_10((uint32_t)rid, (uint32_t)(rid >> 32), STAGE_PROPOSE, (uint32_t)blk, (uint32_t)seed, (uint32_t)(seed >> 32), w);
          if (!(bound(load_quad(s, blk, V, vec), w, c) < thr)) exact_keys(s, blk, V, tau, rid, seed, key, idx);
        }
      }
    } else {          // no finite bound (NaN or -inf logits only, or logits beyond float32's range once scaled)
#pragma unroll 1
      for (int blk = first; blk < nblk; blk += step) exact_keys(s, blk, V, tau, rid, seed, key, idx);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      const double ok = __shfl_xor_sync(0xffffffffu, key, o);
      const int oi = __shfl_xor_sync(0xffffffffu, idx, o);
      better(key, idx, ok, oi);
    }
    if (lane == 0) { sh.key[warp] = key; sh.idx[warp] = idx; }
    __syncthreads();
    if (tid == 0) {
      for (int w = 1; w < PWARPS; ++w) better(key, idx, sh.key[w], sh.idx[w]);
      if constexpr (CS == 1) out[row] = idx;
      else { sh.block_key = key; sh.block_idx = idx; }
    }
    if constexpr (CS > 1) {
      cg::cluster_group cl = cg::this_cluster();
      cl.sync();
      if (tid == 0 && crank == 0) {
        for (int r = 1; r < CS; ++r) {
          const ProposeShared* const rs = cl.map_shared_rank(&sh, r);
          better(key, idx, rs->block_key, rs->block_idx);
        }
        out[row] = idx;
      }
    }
  }
  if constexpr (CS > 1) cg::this_cluster().sync();   // no block leaves while a peer may still read its shared memory
}

template <typename T>
cudaError_t launch(const void* logits, int64_t ld, int64_t N, int V, float tau, uint64_t seed, uint64_t row_offset, int32_t* out,
                   int sms, cudaStream_t st) {
  const float c = (float)(INV_LN2 / (double)tau);
  // A row per cluster of 8 while that does not ask for more blocks than fit, and a block keeps a few hundred elements.
  const bool split = N * PROPOSE_CS <= 4 * (int64_t)sms && V >= 8192;
  cudaLaunchConfig_t cfg = {};
  cfg.blockDim = dim3(PT, 1, 1);
  cfg.stream = st;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = PROPOSE_CS; at[0].val.clusterDim.y = 1; at[0].val.clusterDim.z = 1;
  cfg.attrs = at; cfg.numAttrs = split ? 1 : 0;
  cfg.gridDim = dim3((unsigned)(split ? N * PROPOSE_CS : (N < (1 << 30) ? N : (1 << 30))), 1, 1);
  if (split) return cudaLaunchKernelEx(&cfg, propose_kernel<T, PROPOSE_CS>, (const T*)logits, ld, N, V, (double)tau, c, seed, row_offset, out);
  return cudaLaunchKernelEx(&cfg, propose_kernel<T, 1>, (const T*)logits, ld, N, V, (double)tau, c, seed, row_offset, out);
}

}  // namespace

cudaError_t launch_propose(const void* logits, int64_t ld, int64_t N, int V, int dtype, float tau, uint64_t seed,
                           uint64_t row_offset, int32_t* out, cudaStream_t st) {
  int dev = 0, sms = 148;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  return dtype == SAKI_BF16 ? launch<__nv_bfloat16>(logits, ld, N, V, tau, seed, row_offset, out, sms, st)
                            : launch<float>(logits, ld, N, V, tau, seed, row_offset, out, sms, st);
}

}  // namespace saki
