// Proposal utility: x ~ softmax(s / tau) by Gumbel-max, key_v = s_v / tau - log(-log u_v) in float64, u_v from word v % 4
// of Philox block v / 4.
//
// A float64 key costs two logarithms, and all but a few keys are hopeless: every element gets a float32 UPPER BOUND of
// its key, and only those whose bound reaches the best exact key are evaluated in float64, so the result is the argmax of
// the float64 keys.  The bound: with v = 1 - u, -log u >= v + v^2/2, so the Gumbel term is at most -log(v + v^2/2), nearly
// exact where it is large (v small); v is taken from the upper 23 bits of the word, rounded down.  Per element that
// leaves a quarter of a Philox block (ten rounds of two wide multiplications and two xors) and about eight more
// instructions, half of them shared by the elements of a packed pair or of a group of eight: the integer pipes are the
// bound (512 rows of 151936: 68 us; the Philox blocks alone take 40, at 74 cycles per warp and scheduler, a wide multiply
// occupying its pipe for four).  Two independent groups at a time, and one bar per row from the exact keys of each warp's
// best group (one float64 evaluation on the chain of a block instead of two): 83.5 -> 68.5 us.  The row is read once.
// (The kernel works with minus the bound, in units of log 2: the smallest counts.)
#include "saki_device.cuh"
#include <cooperative_groups.h>

namespace cg = cooperative_groups;

namespace saki {

namespace {

constexpr int PT = 256, PWARPS = PT / 32, PROPOSE_CS = 8;
constexpr int G = 8;       // elements of a group: two Philox blocks, the unit that is bounded and remembered

// The Philox key of every round: row-invariant, and an operand from the constant bank instead of two additions a round.
struct Keys { uint32_t k0[10], k1[10]; };

struct ProposeShared {
  double key[PWARPS];
  int idx[PWARPS];
  double block_key, last_key;      // read by the other blocks of the cluster: before and after the groups that reach the bar
  int block_idx, last_idx;
};

// The eight logits of a group, as stored (past the row's end: -inf).
template <typename T> struct Raw;
template <> struct Raw<__nv_bfloat16> {
  uint32_t r[4];
  __device__ __forceinline__ float2 pair(int i) const { return unpack_bf16x2(r[i]); }
  __device__ __forceinline__ void set(const float* x) {
#pragma unroll
    for (int i = 0; i < 4; ++i) r[i] = pack_bf16x2(x[2 * i], x[2 * i + 1]);
  }
};
template <> struct Raw<float> {
  float r[8];
  __device__ __forceinline__ float2 pair(int i) const { return make_float2(r[2 * i], r[2 * i + 1]); }
  __device__ __forceinline__ void set(const float* x) {
#pragma unroll
    for (int i = 0; i < 8; ++i) r[i] = x[i];
  }
};
template <typename T> __device__ __forceinline__ Raw<T> load_full(const T* at) {
  Raw<T> q;
  const uint4 a = __ldg((const uint4*)at);
  if constexpr (sizeof(T) == 2) { q.r[0] = a.x; q.r[1] = a.y; q.r[2] = a.z; q.r[3] = a.w; }
  else {
    const uint4 b = __ldg((const uint4*)at + 1);
    q.r[0] = __uint_as_float(a.x); q.r[1] = __uint_as_float(a.y); q.r[2] = __uint_as_float(a.z); q.r[3] = __uint_as_float(a.w);
    q.r[4] = __uint_as_float(b.x); q.r[5] = __uint_as_float(b.y); q.r[6] = __uint_as_float(b.z); q.r[7] = __uint_as_float(b.w);
  }
  return q;
}
template <typename T> __device__ __forceinline__ Raw<T> load_raw(const T* s, int grp, int V, bool vec) {
  if (vec && grp * G + G <= V) return load_full(s + grp * G);
  float x[G];
#pragma unroll
  for (int k = 0; k < G; ++k) x[k] = grp * G + k < V ? ld_as_float(s, grp * G + k) : -CUDART_INF_F;
  Raw<T> q;
  q.set(x);
  return q;
}

__device__ __forceinline__ float lg2f(float x) {
  float y;
  asm("lg2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
__device__ __forceinline__ void philox_keys(uint64_t rid, uint32_t blk, const Keys& K, uint32_t (&w)[4]) {
  uint32_t c0 = (uint32_t)rid, c1 = (uint32_t)(rid >> 32), c2 = STAGE_PROPOSE, c3 = blk;
#pragma unroll
  for (int r = 0; r < 10; ++r) {
    const uint64_t p0 = (uint64_t)0xD2511F53u * c0, p1 = (uint64_t)0xCD9E8D57u * c2;
    c0 = (uint32_t)(p1 >> 32) ^ c1 ^ K.k0[r]; c1 = (uint32_t)p1;
    c2 = (uint32_t)(p0 >> 32) ^ c3 ^ K.k1[r]; c3 = (uint32_t)p0;
  }
  w[0] = c0; w[1] = c1; w[2] = c2; w[3] = c3;
}
// lower bound of minus a group's largest key, in units of log 2 and one too large (nc = -log2(e) / tau)
template <typename T> __device__ __forceinline__ float lower(const Raw<T>& q, int grp, uint64_t rid, const Keys& K, float nc) {
  float m = CUDART_INF_F;
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    uint32_t w[4];
    philox_keys(rid, (uint32_t)(2 * grp + h), K, w);
#pragma unroll
    for (int k = 0; k < 2; ++k) {
      // (0x7f : ~w) >> 9 is the float 1 + v, v = 1 - u rounded down to 23 bits (may be 0): 2 (v + v^2/2) = (1 + v)^2 - 1
      // by one multiply-add, rounded once
      const float gx = __uint_as_float(__funnelshift_r(~w[2 * k], 0x7fu, 9)), gy = __uint_as_float(__funnelshift_r(~w[2 * k + 1], 0x7fu, 9));
      const float2 g = make_float2(gx, gy), l = ffma2(g, g, splat(-1.f)), d = ffma2(q.pair(2 * h + k), splat(nc), make_float2(lg2f(l.x), lg2f(l.y)));
      m = fminf(fminf(m, d.x), d.y);
    }
  }
  return m;
}
__device__ __forceinline__ void better(double& key, int& idx, double k, int i) {
  if (k > key || (k == key && i < idx)) { key = k; idx = i; }
}
// a group's exact keys, one per lane (lanes 0 to 7 of the warp): each lane keeps its best
template <typename T>
__device__ __noinline__ void exact_keys(const T* s, int grp, int V, double tau, uint64_t rid, uint64_t seed, double& key, int& idx) {
  const int lane = threadIdx.x & 31, v = grp * G + lane;
  if (lane < G && v < V) {
    uint32_t w[4];
    philox4x32_10((uint32_t)rid, (uint32_t)(rid >> 32), STAGE_PROPOSE, (uint32_t)(v >> 2), (uint32_t)seed, (uint32_t)(seed >> 32), w);
    const int k = v & 3;
    const double u = ((double)(k == 0 ? w[0] : k == 1 ? w[1] : k == 2 ? w[2] : w[3]) + 0.5) * (1.0 / 4294967296.0);
    const double e = (double)ld_as_float(s, v) / tau - log(-log(u));
    if (e > -CUDART_INF) better(key, idx, e, v);
  }
}
__device__ __forceinline__ void warp_better(double& key, int& idx) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const double ok = __shfl_xor_sync(0xffffffffu, key, o);
    const int oi = __shfl_xor_sync(0xffffffffu, idx, o);
    better(key, idx, ok, oi);
  }
}

// CS: blocks per row (1, or a cluster that shares the row)
template <typename T, int CS>
__global__ void __launch_bounds__(PT, 3) propose_kernel(const T* logits, int64_t ld, int64_t N, int V, double tau, float nc,
                                                        const Keys K, uint64_t seed, uint64_t row_offset, int32_t* out) {
  __shared__ ProposeShared sh;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  wait_for_predecessor();
  int crank = 0;
  if constexpr (CS > 1) crank = (int)cg::this_cluster().block_rank();
  const int first = crank * PT + tid, step = PT * CS, ngrp = (V + G - 1) / G;
  for (int64_t row = blockIdx.x / CS; row < N; row += gridDim.x / CS) {
    const T* const s = logits + row * ld;
    const bool vec = ((uintptr_t)s & 15) == 0;
    const uint64_t rid = row_offset + (uint64_t)row;
    // the best group of this thread by its bound, and the second best bound
    float b1 = CUDART_INF_F, b2 = b1;
    int i1 = 0;
    auto note = [&](float m, int grp) {
      b2 = fminf(b2, fmaxf(b1, m));
      i1 = m < b1 ? grp : i1;
      b1 = fminf(b1, m);
    };
    // two groups at a time (independent chains), the logits of the next on their way
    int grp = first;
    if (vec) {
      const int nfull = V / G;
      const T* at = s + (int64_t)grp * G;
      Raw<T> next = {};
      if (grp < nfull) next = load_full(at);
#pragma unroll 1
      for (; grp + step < nfull; grp += 2 * step) {
        const Raw<T> raw0 = next, raw1 = load_full(at + step * G);
        at += 2 * step * G;
        if (grp + 2 * step < nfull) next = load_full(at);
        const float m0 = lower(raw0, grp, rid, K, nc), m1 = lower(raw1, grp + step, rid, K, nc);
        note(m0, grp);
        note(m1, grp + step);
      }
    }
#pragma unroll 1
    for (; grp < ngrp; grp += step) note(lower(load_raw(s, grp, V, vec), grp, rid, K, nc), grp);
    // (not earlier: blocks of the next launch would take up what this one leaves of each SM, unevenly)
    launch_dependents();
    // each warp's best group by its bound: the largest of their exact keys sets the bar
    float mb = b1;
    int mi = i1;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      const float ob = __shfl_xor_sync(0xffffffffu, mb, o);
      const int oi = __shfl_xor_sync(0xffffffffu, mi, o);
      if (ob < mb || (ob == mb && oi < mi)) { mb = ob; mi = oi; }
    }
    double key = -CUDART_INF;
    int idx = 0x7fffffff;
    if (mb < CUDART_INF_F) {
      exact_keys(s, mi, V, tau, rid, seed, key, idx);
      warp_better(key, idx);
    } else {
      mi = -1;
    }
    if (lane == 0) { sh.key[warp] = key; sh.idx[warp] = idx; }
    __syncthreads();
    key = sh.key[0]; idx = sh.idx[0];
#pragma unroll
    for (int w = 1; w < PWARPS; ++w) better(key, idx, sh.key[w], sh.idx[w]);
    if constexpr (CS > 1) {
      if (tid == 0) { sh.block_key = key; sh.block_idx = idx; }
      cg::cluster_group cl = cg::this_cluster();
      cl.sync();
      for (int r = 0; r < CS; ++r) {
        const ProposeShared* const rs = cl.map_shared_rank(&sh, r);
        better(key, idx, rs->block_key, rs->block_idx);
      }
    }
    // the groups whose bound reaches the bar as well (few rows have one).  Rounding of a bound: ~1e-7 of the scaled logit
    // (the Gumbel term is within 33 of zero), and of lg2.  No bar (NaN or -inf logits only, or logits beyond float32's
    // range once scaled): every group
    const bool bounded = key > -CUDART_INF;
    const float fb = 1.f - (float)(key * INV_LN2);
    const float thr = fb + (1e-4f + 1e-6f * (fminf(fabsf(fb), 1e30f) + 64.f));
    auto reaches = [&](float b) { return !(b > thr) && b < CUDART_INF_F; };
    const bool wanted = reaches(b1) && i1 != mi, all = !bounded || reaches(b2);
    const bool more = __syncthreads_or(wanted || all);
    if (more) {
      // the warp evaluates the groups its lanes ask for, one after the other
      auto evaluate = [&](bool which, int grp) {
        for (unsigned m = __ballot_sync(0xffffffffu, which); m; m &= m - 1)
          exact_keys(s, __shfl_sync(0xffffffffu, grp, __ffs(m) - 1), V, tau, rid, seed, key, idx);
      };
      if (!__any_sync(0xffffffffu, all)) {
        evaluate(wanted, i1);
      } else {      // a second group of a thread reaches the bar: the warp bounds its groups again
#pragma unroll 1
        for (int g0 = first - lane; g0 < ngrp; g0 += step) {
          const int grp = min(g0 + lane, ngrp - 1);
          evaluate(!bounded || !(lower(load_raw(s, grp, V, vec), grp, rid, K, nc) > thr), grp);
        }
      }
      warp_better(key, idx);
      if (lane == 0) { sh.key[warp] = key; sh.idx[warp] = idx; }
      __syncthreads();
      if (tid == 0)
        for (int w = 0; w < PWARPS; ++w) better(key, idx, sh.key[w], sh.idx[w]);
    }
    if constexpr (CS == 1) {
      if (tid == 0) out[row] = idx;
      if (more) __syncthreads();       // the next row writes where thread 0 reads
    } else {
      if (tid == 0) { sh.last_key = key; sh.last_idx = idx; }
      cg::cluster_group cl = cg::this_cluster();
      cl.sync();
      if (tid == 0 && crank == 0) {
        for (int r = 1; r < CS; ++r) {
          const ProposeShared* const rs = cl.map_shared_rank(&sh, r);
          better(key, idx, rs->last_key, rs->last_idx);
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
  const float nc = -(float)(INV_LN2 / (double)tau);
  Keys K;
  for (int r = 0; r < 10; ++r) {
    K.k0[r] = (uint32_t)seed + (uint32_t)r * 0x9E3779B9u;
    K.k1[r] = (uint32_t)(seed >> 32) + (uint32_t)r * 0xBB67AE85u;
  }
  // Blocks per row: the number that takes the least time, a block on every SM taking a + 0.112 V / 1000 / blocks
  // microseconds (fitted to V = 2048 to 151936 and 8 to 888 rows; a grows with the exchange between the blocks).  Rows of
  // 151936: 8 rows 20.9 / 13.9 / 9.7 / 8.3 us with 1 / 2 / 4 / 8 blocks, 148 rows 21 / 22 / 32 / 39, 200 rows 37 / 31 / 37 /
  // 50, 512 rows 74 / 69 / 85 / 126.
  static const double a[4] = {0.4, 1.35, 1.9, 2.05};
  int cs = 1;
  double best = 1e300;
  for (int i = 0; (1 << i) <= PROPOSE_CS; ++i) {
    const double c = (double)((((int64_t)N << i) + sms - 1) / sms) * (a[i] + 0.112e-3 * V / (1 << i));
    if (c < best) { best = c; cs = 1 << i; }
  }
  cudaLaunchConfig_t cfg = {};
  cfg.blockDim = dim3(PT, 1, 1);
  cfg.stream = st;
  cudaLaunchAttribute at[2];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  at[1].id = cudaLaunchAttributeClusterDimension;
  at[1].val.clusterDim.x = (unsigned)cs; at[1].val.clusterDim.y = 1; at[1].val.clusterDim.z = 1;
  cfg.attrs = at; cfg.numAttrs = cs > 1 ? 2 : 1;
  cfg.gridDim = dim3((unsigned)((N < (1 << 27) ? N : (1 << 27)) * cs), 1, 1);
  auto go = [&](auto kernel) { return cudaLaunchKernelEx(&cfg, kernel, (const T*)logits, ld, N, V, (double)tau, nc, K, seed, row_offset, out); };
  switch (cs) {
    case 1: return go(propose_kernel<T, 1>);
    case 2: return go(propose_kernel<T, 2>);
    case 4: return go(propose_kernel<T, 4>);
    default: return go(propose_kernel<T, 8>);
  }
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
