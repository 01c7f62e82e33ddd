// Cluster kernel for bf16 rows: the latency path (calls of a few long rows).
//
// One vocabulary row per thread-block cluster of CS CTAs x 256 threads.  Each CTA owns a contiguous slice of the row in
// shared memory, fetched by one 1-D bulk async copy per array (cp.async.bulk + mbarrier), so the row pair is read from HBM
// exactly once; each thread owns an odd number of contiguous chunks of 8 elements
// (up to 11: 88 elements; 40 at V = 151936 with 16 CTAs).  What bounds a call here is the chain of steps of a
// single row, and much of that was instruction fetch: with the row in registers every pass was 40 unrolled pairs of code
// that ran once.  The passes are loops over shared memory now, and the registers that frees let the scalar steps be
// inlined.  With what that made possible (warp 0 gathers all sums and goes on to the scalars, up to 16 CTAs per row, sums
// taken chunk by chunk) 8 rows of 151936 went from 23.6 to 18.7 us, 1 row from 22.9 to 15.7, 32 rows from 32.1 to 24.5.
// Passes:
//   lse      2 exponentials/element: both log-sum-exps (computed under the
//            CTA's own maxima rounded up to whole powers of two, then moved
//            exactly onto the row's maxima, which the CTAs exchange while the
//            pass runs), moments of the teacher-student logit difference under
//            p (initial guess of lambda), KL(T||p) (saturation test), teacher
//            argmax index
//   solve    1 exponential/element per evaluation of KL(q_beta||p) and the first
//            four cumulants of the logit difference under q_beta; lambda = root of
//            the fourth-order Taylor model inside a bisection bracket, one
//            evaluation for most rows (Eqs. "bridge", "trust_region")
//   final    2 exponentials/element: TV = sum [q-p]_+ with per-thread ordered
//            partial sums for the inverse-CDF residual draw (Eqs. "accept",
//            "residual"), and the gradient row (Eq. "general_objective")
// Per-element work is float32 (packed f32x2 FMAs, ex2.approx); every
// cross-thread combination and every per-row scalar is float64.  Per-warp
// partial sums travel to all CTAs of the cluster as asynchronous
// distributed-shared-memory stores that complete on the receiver's mbarrier
// (no cluster barrier, no fence on the row loop); each CTA then forms the
// same scalars redundantly from the same numbers in the same order, so
// control flow is uniform across the cluster.
#define SAKI_SCALARS_INLINE 1
#include "saki_device.cuh"
#include <cooperative_groups.h>
#include <math_constants.h>
#include <mutex>

namespace cg = cooperative_groups;

namespace saki {

constexpr int CT = 256;                 // threads per CTA
constexpr int CW = CT / 32;             // warps per CTA
constexpr int MAX_CHUNKS = 11;          // 16-byte chunks (8 bf16) per thread and row, at most; always an odd number: a thread's
                                        // chunks are contiguous, and an odd stride keeps 128-bit shared loads free of conflicts
constexpr int SLICE_CAP = CT * MAX_CHUNKS * 8;      // elements of one row a CTA can hold
constexpr int MAX_V = 163840;
constexpr int MAX_CS = 16;
constexpr int NSLOT = MAX_CS * CW;      // per-warp partial slots of a cluster
constexpr int NV = 8;                   // doubles per partial vector
constexpr uint32_t SENTINEL = 0xFF7FFF7Fu;   // two bf16 "most negative finite": exp -> 0, difference 0

constexpr int OFF_RED = 0;                                      // [2][NV][NSLOT] doubles: per-warp partials
constexpr int OFF_MX = OFF_RED + 2 * NV * NSLOT * 8;            // [2][MAX_CS][2] doubles: per-CTA maxima
constexpr int OFF_GAT = OFF_MX + 2 * MAX_CS * 2 * 8;            // [NV] doubles: cluster totals
constexpr int OFF_BC = OFF_GAT + NV * 8;                        // [2][BC_DOUBLES] broadcast scalars
constexpr int OFF_WMAX = OFF_BC + 2 * BC_DOUBLES * 8;           // [2][2][CW] floats: per-warp maxima
constexpr int OFF_MBAR = OFF_WMAX + 2 * 2 * CW * 4;             // copy barrier, 2 exchange barriers, 2 maxima barriers
constexpr int OFF_S = (OFF_MBAR + 5 * 8 + 127) / 128 * 128;     // the slice of the student's row, then the teacher's
static int slice_of(int V, int cs) { return ((V + cs - 1) / cs + 7) & ~7; }
static int smem_bytes(int slice_len) { return OFF_S + 2 * ((slice_len * 2 + 127) / 128 * 128); }
static_assert(OFF_MBAR % 8 == 0, "alignment");

template <int CS>
__global__ void __launch_bounds__(CT, CS > 8 ? 1 : 2) cluster_kernel(const RowParams P, const int n_clusters) {
  extern __shared__ __align__(128) unsigned char smem[];
  launch_dependents();
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const unsigned rank = cg::this_cluster().block_rank();
  const int cluster_id = blockIdx.x / CS;

  const __nv_bfloat16* slot_s = (const __nv_bfloat16*)(smem + OFF_S);
  double* red = (double*)(smem + OFF_RED);
  double* mx = (double*)(smem + OFF_MX);
  double* gat = (double*)(smem + OFF_GAT);
  float* wmax = (float*)(smem + OFF_WMAX);
  uint64_t* mbar = (uint64_t*)(smem + OFF_MBAR);   // [0] row copy, [1..2] partial exchange, [3..4] maxima exchange
  const uint32_t red_s = smem_addr(red), mx_s = smem_addr(mx), bar_s = smem_addr(mbar);

  const int V = P.V;
  const int slice_len = ((V + CS - 1) / CS + 7) & ~7;
  const int off_t = OFF_S + (slice_len * 2 + 127) / 128 * 128;
  const __nv_bfloat16* slot_t = (const __nv_bfloat16*)(smem + off_t);
  const int slice_start = (int)rank * slice_len;
  const int my_len = max(0, min(slice_len, V - slice_start));
  const uint32_t slice_bytes = (uint32_t)my_len * 2u;
  const int chunks = ((slice_len + 8 * CT - 1) / (8 * CT)) | 1;     // per thread
  const int ept = chunks * 8, thr_first = tid * ept;                // elements of a thread, its first within the slice

  const float c32 = (float)(1.4426950408889634 / (double)P.temperature);     // log2(e)/temperature
  Consts K;
  K.tau = (double)P.temperature; K.rtau = 1.0 / K.tau; K.eps = (double)P.eps; K.c64 = (double)c32;
  K.rc64 = 1.0 / K.c64; K.grad_scale = (double)P.grad_scale; K.sqrt_eps = sqrtf(P.eps); K.V = V;

  bool dead = false;   // a wait timed out: this CTA stops fetching and the cluster flags its rows
  auto row_ptrs = [&](int64_t row, const __nv_bfloat16*& s, const __nv_bfloat16*& t) {
    const int64_t b = row / P.K1;
    const int j = (int)(row - b * P.K1);
    s = (const __nv_bfloat16*)P.s + b * P.s_seq + (int64_t)j * P.s_pos;
    t = (const __nv_bfloat16*)P.t + b * P.t_seq + (int64_t)j * P.t_pos;
  };
  auto issue = [&](int64_t row) {   // one thread: fetch this CTA's slice of both rows
    const __nv_bfloat16 *s, *t;
    row_ptrs(row, s, t);
    mbar_expect_tx(&mbar[0], 2u * slice_bytes);
    if (slice_bytes) {
      bulk_load(smem + OFF_S, s + slice_start, slice_bytes, &mbar[0]);
      bulk_load(smem + off_t, t + slice_start, slice_bytes, &mbar[0]);
    }
  };
  // one exchange: every warp's totals, value lane / 4 in each lane (n of them), to slot rank*CW+warp of red[p] in every CTA
  auto push = [&](double v, int n, int p) {
    const int k = lane >> 2;
    if (k < n) {
      const uint32_t dst = red_s + (uint32_t)(((p * NV + k) * NSLOT + rank * CW + warp) * 8), bar = bar_s + (uint32_t)((1 + p) * 8);
#pragma unroll
      for (int r = lane & 3; r < CS; r += 4) st_async_f64(map_to_rank(dst, r), v, map_to_rank(bar, r));
    }
  };
  // warp 0: cluster total of value lane / 4 (fixed order, the same in every CTA)
  auto gather = [&](int p) {
    const double* base = red + (size_t)(p * NV + (lane >> 2)) * NSLOT;
    double a = 0.0;
#pragma unroll
    for (int slot = lane & 3; slot < CS * CW; slot += 4) a += base[slot];
    a += __shfl_xor_sync(0xffffffffu, a, 2);
    a += __shfl_xor_sync(0xffffffffu, a, 1);
    return a;
  };
  // warp 0, for a draw: the warp of the cluster that owns the inverse-CDF target (ordered scan of the warps' weights)
  auto find_owner = [&](double* bc, const double* weight) {
    constexpr int NW = CS * CW, PER = NW > 32 ? NW / 32 : 1;
    double w[PER], mine = 0.0;
#pragma unroll
    for (int q = 0; q < PER; ++q) {
      w[q] = lane * PER + q < NW ? weight[lane * PER + q] : 0.0;
      mine += w[q];
    }
    double inc = mine;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const double up = __shfl_up_sync(0xffffffffu, inc, o);
      if (lane >= o) inc += up;
    }
    const double target = bc[BC_UDRAW] * __shfl_sync(0xffffffffu, inc, 31);
    const unsigned hit = __ballot_sync(0xffffffffu, inc > target), pos = __ballot_sync(0xffffffffu, mine > 0.0);
    // rounding left no crossing: the last position with positive weight
    if (lane == (hit ? __ffs(hit) - 1 : pos ? 31 - __clz(pos) : 0)) {
      double before = inc - mine;
      int owner = 0;
#pragma unroll
      for (int q = 0; q < PER - 1; ++q)
        if (owner == q && (hit ? !(before + w[q] > target) : true)) { before += w[q]; ++owner; }
      if (!hit) {
#pragma unroll
        for (int q = 0; q < PER; ++q) if (w[q] > 0.0) owner = q;
        before = 0.0;
      }
      bc[BC_OWNER_WARP] = (double)(lane * PER + owner); bc[BC_BEFORE] = before; bc[BC_TARGET] = target; bc[BC_TAKE_LAST] = hit ? 0.0 : 1.0;
    }
  };
  // this thread's chunks of the slice: body(first element within the slice, student, teacher); beyond the slice's end the
  // elements are "most negative finite"
  auto for_chunks = [&](auto&& body) {
#pragma unroll 2
    for (int j = 0; j < chunks; ++j) {
      const int e0 = thr_first + j * 8;
      uint4 a = make_uint4(SENTINEL, SENTINEL, SENTINEL, SENTINEL), b = a;
      if (e0 < my_len && !dead) {
        a = *reinterpret_cast<const uint4*>(slot_s + e0);
        b = *reinterpret_cast<const uint4*>(slot_t + e0);
      }
      const uint32_t sw[4] = {a.x, a.y, a.z, a.w}, tw[4] = {b.x, b.y, b.z, b.w};
      body(e0, sw, tw);
    }
  };

  if (tid == 0) {
#pragma unroll
    for (int i = 0; i < 5; ++i) mbar_init(&mbar[i], 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  cg::this_cluster().sync();   // every CTA's barriers exist before any peer signals them
  wait_for_predecessor();
  if (tid == 0 && cluster_id < P.n_rows) issue(cluster_id);
  uint32_t phase = 0, xph0 = 0, xph1 = 0, mph0 = 0, mph1 = 0;
  int parity = 0, rb = 0;

  for (int64_t row = cluster_id; row < P.n_rows; row += n_clusters, rb ^= 1) {
    double* bc = (double*)(smem + OFF_BC) + rb * BC_DOUBLES;
    const uint64_t rid = P.row_offset + (uint64_t)row;
    const int64_t seq = row / P.K1;
    const int pos = (int)(row - seq * P.K1);
    const bool bonus = P.spec && (pos == P.K1 - 1);
    const int x = bonus ? 0 : (P.spec ? P.proposal[seq * P.prop_ld + pos] : P.proposal[row]);
    const bool masked = (P.mask != nullptr) && (P.mask[row] == 0);
    const __nv_bfloat16 *g_s, *g_t;
    row_ptrs(row, g_s, g_t);
    __nv_bfloat16* g_out = P.dlogits ? (__nv_bfloat16*)P.dlogits + row * P.ld_g : nullptr;

    if (row != cluster_id) {                 // the slot is free once every thread is done with the last row
      __syncthreads();
      if (tid == 0 && !dead) {
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        issue(row);
      }
    }
    // row scalars that do not depend on the passes, while the copy is on its way
    if (tid == 32) bc[BC_UACC] = scalar_uniform(P.seed, rid, STAGE_ACCEPT);
    if (tid == 64) bc[BC_UDRAW] = scalar_uniform(P.seed, rid, bonus ? STAGE_BONUS : STAGE_RESIDUAL);
    if (tid == 96) {
      const bool ok = (x >= 0 && x < V);
      bc[BC_SX] = ok ? (double)__bfloat162float(g_s[x]) : 0.0;
      bc[BC_TX] = ok ? (double)__bfloat162float(g_t[x]) : 0.0;
    }

    // ------------------------------------------------ the slice has arrived; its maxima
    if (!dead) {
      if (!mbar_wait_bounded(&mbar[0], phase)) dead = true;
      else phase ^= 1u;
    }
    // maxima of this CTA's slice (packed bf16), via shuffles and one CTA barrier
    float my_mt;
    {
      uint32_t a = SENTINEL, b = SENTINEL;
      for_chunks([&](int, const uint32_t* sw, const uint32_t* tw) {
        a = max_bf16x2(a, max_bf16x2(max_bf16x2(sw[0], sw[1]), max_bf16x2(sw[2], sw[3])));
        b = max_bf16x2(b, max_bf16x2(max_bf16x2(tw[0], tw[1]), max_bf16x2(tw[2], tw[3])));
      });
      const float2 fb0 = unpack_bf16x2(b);
      my_mt = fmaxf(fb0.x, fb0.y);
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) {
        a = max_bf16x2(a, __shfl_xor_sync(0xffffffffu, a, o));
        b = max_bf16x2(b, __shfl_xor_sync(0xffffffffu, b, o));
      }
      if (lane == 0) {
        const float2 fa = unpack_bf16x2(a), fb = unpack_bf16x2(b);
        wmax[(rb * 2 + 0) * CW + warp] = fmaxf(fa.x, fa.y);
        wmax[(rb * 2 + 1) * CW + warp] = fmaxf(fb.x, fb.y);
      }
    }
    if (__syncthreads_or(dead ? 1 : 0)) dead = true;
    if (tid == 0) {
      mbar_expect_tx(&mbar[3 + rb], (uint32_t)(CS * 16));          // maxima of all CTAs
      mbar_expect_tx(&mbar[1 + parity], (uint32_t)(CS * CW * 8 * 8));   // partials of pass "lse"
    }
    float ms_r = wmax[(rb * 2 + 0) * CW], mt_r = wmax[(rb * 2 + 1) * CW];
#pragma unroll
    for (int w = 1; w < CW; ++w) {
      ms_r = fmaxf(ms_r, wmax[(rb * 2 + 0) * CW + w]);
      mt_r = fmaxf(mt_r, wmax[(rb * 2 + 1) * CW + w]);
    }
    if (tid < CS) {   // this CTA's maxima to every CTA (a CTA that timed out sends NaN: the row is flagged)
      const uint32_t dst = map_to_rank(mx_s + (uint32_t)(((rb * MAX_CS) + rank) * 16), tid);
      const uint32_t bar = map_to_rank(bar_s + (uint32_t)((3 + rb) * 8), tid);
      st_async_f64(dst, dead ? CUDART_NAN : (double)ms_r, bar);
      st_async_f64(dst + 8, (double)mt_r, bar);
    }
    // whole-number shifts: every exponent argument is <= 0, and sums taken under different
    // shifts differ by exact powers of two
    const float k0r = -ceilf(c32 * fmaxf(ms_r, -1e30f)), k1r = -ceilf(c32 * fmaxf(mt_r, -1e30f));

    // teacher argmax candidate of this thread (exact compare on stored values, lowest index)
    uint32_t cand = 0xffffffffu;
    if (my_mt == mt_r) {
      for_chunks([&](int e0, const uint32_t*, const uint32_t* tw) {
#pragma unroll
        for (int k = 3; k >= 0; --k) {
          const float2 f = unpack_bf16x2(tw[k]);
          if (f.y == mt_r) cand = min(cand, (uint32_t)(slice_start + e0 + 2 * k + 1));
          if (f.x == mt_r) cand = min(cand, (uint32_t)(slice_start + e0 + 2 * k));
        }
      });
    }

    // ------------------------------------------------ pass "lse"
    float k0, k1;        // the row's shifts
    bool row_timeout;
    {
      float2 Ss = splat(0.f), St = splat(0.f), M1 = splat(0.f), M2 = splat(0.f), M3 = splat(0.f), M4 = splat(0.f),
             N1 = splat(0.f);
      const float2 cc = splat(c32), kk0 = splat(k0r), kk1 = splat(k1r), neg1 = splat(-1.f);
      for_chunks([&](int, const uint32_t* sw, const uint32_t* tw) {
        float2 cs = splat(0.f), ct = splat(0.f);   // per chunk first: a dominant element swamps fewer small ones
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          const float2 sf = unpack_bf16x2(sw[i]), tf = unpack_bf16x2(tw[i]);
          const float2 d = ffma2(sf, neg1, tf);
          const float2 es = ex2f2(ffma2(sf, cc, kk0));
          const float2 et = ex2f2(ffma2(tf, cc, kk1));
          cs = i == 0 ? es : fadd2(cs, es);
          ct = i == 0 ? et : fadd2(ct, et);
          const float2 d2 = fmul2(d, d);
          M1 = ffma2(es, d, M1);
          const float2 u = fmul2(es, d2);
          M2 = fadd2(M2, u);
          M3 = ffma2(u, d, M3);
          M4 = ffma2(u, d2, M4);
          N1 = ffma2(et, d, N1);
        }
        Ss = fadd2(Ss, cs);
        St = fadd2(St, ct);
      });
      // the row's maxima have arrived meanwhile: move the partial sums onto the row's shifts
      bool mx_timeout = false;
      if (!mbar_wait_bounded(&mbar[3 + rb], rb ? mph1 : mph0)) mx_timeout = true;
      if (rb) mph1 ^= 1u; else mph0 ^= 1u;
      float gms = -CUDART_INF_F, gmt = -CUDART_INF_F;
      bool poisoned = mx_timeout;
#pragma unroll
      for (int r = 0; r < CS; ++r) {
        const double a = mx[(rb * MAX_CS + r) * 2 + 0], b = mx[(rb * MAX_CS + r) * 2 + 1];
        if (a != a) poisoned = true;
        gms = fmaxf(gms, (float)a); gmt = fmaxf(gmt, (float)b);
      }
      row_timeout = poisoned;
      if (mx_timeout) dead = true;
      k0 = -ceilf(c32 * fmaxf(gms, -1e30f)); k1 = -ceilf(c32 * fmaxf(gmt, -1e30f));
      const double fs = pow2_exact((int)(k0 - k0r)), ft = pow2_exact((int)(k1 - k1r));
      auto tot = [](const float2 a) { return (double)a.x + (double)a.y; };
      // (the place of the argmax in the vector: its index, and the largest index where this CTA does not hold the maximum)
      const double v[8] = {fs * tot(Ss), ft * tot(St), fs * tot(M1), fs * tot(M2), fs * tot(M3), ft * tot(N1), 0.0, fs * tot(M4)};
      const uint32_t wc = __reduce_min_sync(0xffffffffu, mt_r == gmt ? cand : 0xffffffffu);
      const double total = warp_sum8(v, lane);
      push((lane >> 2) == 6 ? (double)wc : total, 8, parity);
      if (warp == 0) {
        if (!mbar_wait_bounded(&mbar[1 + parity], parity ? xph1 : xph0)) dead = true;
        const double g = gather(parity);
        const double* const ci = red + (size_t)(parity * NV + 6) * NSLOT;
        double am = 4294967295.0;
        for (int slot = lane; slot < CS * CW; slot += 32) am = fmin(am, ci[slot]);
        const uint32_t best = __reduce_min_sync(0xffffffffu, (uint32_t)am);
        if ((lane & 3) == 0) gat[lane >> 2] = (lane >> 2) == 6 ? (double)best : g;
        __syncwarp();
      }
      if (parity) xph1 ^= 1u; else xph0 ^= 1u;
      parity ^= 1;
      if (tid < 2) {   // lane 0: the student's sum, lane 1: the teacher's; then lane 0 alone
        double rS, G;
        lse_of_sum(gat[lane], lane ? (double)k1 : (double)k0, rS, G);
        const double rSt = __shfl_sync(0x3u, rS, 1), G1 = __shfl_sync(0x3u, G, 1);
        // (sums that are not finite: a logit is not, or the difference of two logits, one of them masked with the type's lowest
        // value say, has no square in float32; the float64 kernel tells the two apart and routes the second)
        if (tid == 0) scalar_after_lse_tail(bc, gat, K, k0, k1, x, bonus, masked, row_timeout, 1.f, true, rS, rSt, G, G1, gat + 7);
      }
      if (tid == 0) {
        if ((int)bc[BC_MODE] == MODE_SOLVE) mbar_expect_tx(&mbar[1 + parity], (uint32_t)(CS * CW * 5 * 8));
        else if ((int)bc[BC_MODE] == MODE_FINAL) mbar_expect_tx(&mbar[1 + parity], (uint32_t)(CS * CW * 3 * 8));
      }
      __syncthreads();
    }

    // ------------------------------------------------ pass "solve" (repeated)
    while ((int)bc[BC_MODE] == MODE_SOLVE) {
      const float cb = (float)bc[BC_CB], kb = (float)bc[BC_KB];
      float2 S0 = splat(0.f), S1 = splat(0.f), S2 = splat(0.f), S3 = splat(0.f), S4 = splat(0.f);
      const float2 cc = splat(c32), cbb = splat(cb), kbb = splat(kb), neg1 = splat(-1.f);
      for_chunks([&](int, const uint32_t* sw, const uint32_t* tw) {
        float2 c0 = splat(0.f), c1 = splat(0.f);
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          const float2 sf = unpack_bf16x2(sw[i]), tf = unpack_bf16x2(tw[i]);
          const float2 d = ffma2(sf, neg1, tf);
          const float2 e = ex2f2(ffma2(d, cbb, ffma2(sf, cc, kbb)));
          const float2 d2 = fmul2(d, d);
          c0 = i == 0 ? e : fadd2(c0, e);
          c1 = i == 0 ? fmul2(e, d) : ffma2(e, d, c1);
          const float2 u = fmul2(e, d2);
          S2 = fadd2(S2, u);
          S3 = ffma2(u, d, S3);
          S4 = ffma2(u, d2, S4);
        }
        S0 = fadd2(S0, c0);
        S1 = fadd2(S1, c1);
      });
      auto tot = [](const float2 a) { return (double)a.x + (double)a.y; };
      const double v[8] = {tot(S0), tot(S1), tot(S2), tot(S3), tot(S4), 0.0, 0.0, 0.0};
      push(warp_sum8(v, lane), 5, parity);
      if (warp == 0) {
        if (!mbar_wait_bounded(&mbar[1 + parity], parity ? xph1 : xph0)) dead = true;
        const double g = gather(parity);
        if ((lane & 3) == 0 && lane < 20) gat[lane >> 2] = g;
        __syncwarp();
      }
      if (parity) xph1 ^= 1u; else xph0 ^= 1u;
      parity ^= 1;
      if (tid == 0) {
        scalar_after_solve4(bc, gat, K, k0, k1, x, bonus, masked);
        if ((int)bc[BC_MODE] == MODE_SOLVE) mbar_expect_tx(&mbar[1 + parity], (uint32_t)(CS * CW * 5 * 8));   // next evaluation
        else if ((int)bc[BC_MODE] == MODE_FINAL) mbar_expect_tx(&mbar[1 + parity], (uint32_t)(CS * CW * 3 * 8));   // pass "final"
      }
      __syncthreads();
    }

    // ------------------------------------------------ flagged row: zero outputs, zero gradient
    if ((int)bc[BC_MODE] == MODE_FLAGGED || (int)bc[BC_MODE] == MODE_REDO) {
      const bool redo = (int)bc[BC_MODE] == MODE_REDO;   // ill-conditioned for float32: the float64 kernel routes it
      if (rank == 0 && tid == 0) {
        if (redo) {
          const unsigned int slot = atomicAdd(P.redo_count, 1u);
          P.redo_list[slot] = (int32_t)row;
          if (P.redo_guess) P.redo_guess[slot] = (float)bc[BC_BETA];     // where the float64 kernel starts its iteration
        }
        else {
          write_row(P.out, row, zero_row((uint32_t)bc[BC_STATUS]), !P.spec);
          atomicAdd(P.flagged, 1ull);
        }
      }
      if (g_out && !redo) {
#pragma unroll 1
        for (int e0 = thr_first; e0 < min(thr_first + ept, my_len); e0 += 8)
          *reinterpret_cast<uint4*>(g_out + slice_start + e0) = make_uint4(0, 0, 0, 0);
      }
      continue;
    }

    // ------------------------------------------------ pass "final"
    const bool need_draw = bonus || bc[BC_CORR] != 0.0;
    float my_part;       // this thread's ordered weight for the inverse-CDF draw
    const float cl = (float)bc[BC_CL], kq = (float)bc[BC_KQ];
    const float iq = (float)bc[BC_IQ], ip = (float)bc[BC_IP];
    {
      const float KGf = (float)bc[BC_KG];
      const float kg = (float)(bc[BC_KG] * (double)ip);     // gradient entry = e_p * kg
      const bool want_g = (g_out != nullptr);
      float2 Sq[2] = {splat(0.f), splat(0.f)}, R[2] = {splat(0.f), splat(0.f)};
      const float2 cc = splat(c32), cll = splat(cl), kqq = splat(kq), kk0 = splat(k0), neg1 = splat(-1.f);
      const float2 iqq = splat(iq), nip = splat(-ip), kgg = splat(kg);
      for_chunks([&](int e0, const uint32_t* sw, const uint32_t* tw) {
        uint32_t gp[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) {
          const int h = k & 1;
          const float2 sf = unpack_bf16x2(sw[k]), tf = unpack_bf16x2(tw[k]);
          const float2 d = ffma2(sf, neg1, tf);
          const float2 ep = ex2f2(ffma2(sf, cc, kk0));
          const float2 eq = ex2f2(ffma2(d, cll, ffma2(sf, cc, kqq)));
          Sq[h] = fadd2(Sq[h], eq);
          float2 r = ffma2(eq, iqq, fmul2(ep, nip));     // q_i - p_i
          r.x = fmaxf(r.x, 0.f); r.y = fmaxf(r.y, 0.f);
          R[h] = fadd2(R[h], r);
          const float2 gv = fmul2(ep, kgg);
          gp[k] = pack_bf16x2(gv.x, gv.y);
        }
        if (want_g && e0 < my_len) *reinterpret_cast<uint4*>(g_out + slice_start + e0) = make_uint4(gp[0], gp[1], gp[2], gp[3]);
      });
      const float sq_f = (Sq[0].x + Sq[0].y) + (Sq[1].x + Sq[1].y);
      const float r_f = (R[0].x + R[0].y) + (R[1].x + R[1].y);
      my_part = bonus ? sq_f * iq : r_f;
      // the thread that owns the supervised token subtracts the one-hot part of the gradient
      if (want_g) {
        const int tok = (int)bc[BC_TOK];
        const int loc = tok - slice_start - thr_first;
        if (tok >= 0 && loc >= 0 && loc < ept && tok - slice_start < my_len) {
          const float ep = ex2f(fmaf(__bfloat162float(g_s[tok]), c32, k0));
          g_out[tok] = __float2bfloat16_rn(fmaf(ep, kg, -KGf));
        }
      }
      const double v[8] = {(double)sq_f, (double)r_f, (double)my_part, 0.0, 0.0, 0.0, 0.0, 0.0};
      push(warp_sum8(v, lane), 3, parity);
      if (warp == 0) {
        if (!mbar_wait_bounded(&mbar[1 + parity], parity ? xph1 : xph0)) dead = true;
        const double tv = __shfl_sync(0xffffffffu, gather(parity), 4);
        if (lane == 0) bc[BC_TV] = (bc[BC_LAMBDA] > 0.0) ? tv : 0.0;
        if (need_draw) find_owner(bc, red + (size_t)(parity * NV + 2) * NSLOT);
        if (lane == 0) {
          if (!need_draw && rank == 0) write_result(bc, P.out, !P.spec, row, 0, x, false, K.c64, g_s, g_t);
        }
      }
      if (parity) xph1 ^= 1u; else xph0 ^= 1u;
      parity ^= 1;
    }

    // ------------------------------------------------ the draw (corrected and bonus rows only)
    if (need_draw) {
      __syncthreads();
      if ((int)rank * CW + warp == (int)bc[BC_OWNER_WARP]) {
        // inverse CDF inside the owning warp: lanes are in index order
        const double target = bc[BC_TARGET], before = bc[BC_BEFORE];
        const bool take_last = bc[BC_TAKE_LAST] != 0.0;
        double inc = (double)my_part;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
          const double up = __shfl_up_sync(0xffffffffu, inc, o);
          if (lane >= o) inc += up;
        }
        const unsigned posm = __ballot_sync(0xffffffffu, my_part > 0.f);
        const unsigned hit = take_last ? 0u : __ballot_sync(0xffffffffu, before + inc > target);
        int owner_lane;
        bool last_mode = take_last;
        if (hit) owner_lane = __ffs(hit) - 1;
        else { owner_lane = posm ? 31 - __clz(posm) : 0; last_mode = true; }
        double running = __shfl_sync(0xffffffffu, before + inc - (double)my_part, owner_lane);
        const int first = slice_start + (warp * 32 + owner_lane) * ept;
        const int n_el = max(0, min(ept, slice_start + my_len - first));
        int y = -1, last_pos = -1;
        const __nv_bfloat16 *es = slot_s + (first - slice_start), *et = slot_t + (first - slice_start);   // the warp walks the owner's elements together
        for (int base = 0; base < n_el && y < 0; base += 32) {
          const int e = base + lane;
          float w = 0.f;
          if (e < n_el) {
            const float sf = __bfloat162float(es[e]), tf = __bfloat162float(et[e]);
            const float d = tf - sf;
            const float ep = ex2f(fmaf(sf, c32, k0));
            const float eq = ex2f(fmaf(d, cl, fmaf(sf, c32, kq)));
            w = bonus ? eq * iq : fmaxf(fmaf(eq, iq, -(ep * ip)), 0.f);
          }
          double wi = (double)w;
#pragma unroll
          for (int o = 1; o < 32; o <<= 1) {
            const double up = __shfl_up_sync(0xffffffffu, wi, o);
            if (lane >= o) wi += up;
          }
          const unsigned pm = __ballot_sync(0xffffffffu, w > 0.f);
          const unsigned hm = last_mode ? 0u : __ballot_sync(0xffffffffu, running + wi > target);
          if (pm) last_pos = first + base + 31 - __clz(pm);
          if (hm) y = first + base + __ffs(hm) - 1;
          running += __shfl_sync(0xffffffffu, wi, 31);
        }
        if (y < 0) y = (last_pos >= 0) ? last_pos : min(V - 1, first + max(n_el - 1, 0));
        if (lane == 0) write_result(bc, P.out, !P.spec, row, bonus ? 0 : 1, y, bonus, K.c64, g_s, g_t);
      }
    }
  }

  // a CTA that gave up on a copy still waits (bounded) for what it has in flight before leaving
  if (dead && tid == 0) (void)mbar_wait_bounded(&mbar[0], phase);
  cg::this_cluster().sync();   // no CTA leaves while a peer may still write its shared memory
}

// ---------------------------------------------------------------- host side
// CTAs per row: as many as a row needs (a slice fits a CTA's shared memory), and more while no more than two share an SM
// and each keeps 2048 elements (forward and gradient: 32 rows of 65536 with 2 or 4 CTAs each 20.1 / 18.2 us, 8 rows of
// 32000 with 2 or 4 13.9 / 13.3 us).  By V alone, up to 8, where the kernel is pinned (rows = 0).
static int pick_cs(int V, int64_t rows, int sms) {
  const int most = rows > 0 ? MAX_CS : 8;
  int cs = 1;
  while (cs < most && (cs * SLICE_CAP < V || (V >= 4096 * cs && rows * cs <= sms))) cs *= 2;
  return cs;
}

bool cluster_can_serve(const RowParams& p, int dtype) {
  if (dtype != SAKI_BF16) return false;
  if (p.V < 2048 || p.V % 8 != 0 || p.V > MAX_V) return false;
  if (p.n_rows > 0x7fffffffLL) return false;     // the redo list keeps row numbers in 32 bits
  auto al16 = [](const void* q) { return ((uintptr_t)q & 15) == 0; };
  if (!al16(p.s) || !al16(p.t)) return false;
  if (p.s_seq % 8 || p.s_pos % 8 || p.t_seq % 8 || p.t_pos % 8) return false;
  if (p.dlogits && (!al16(p.dlogits) || p.ld_g % 8)) return false;
  return true;
}

template <int CS>
static cudaError_t launch_cs(const RowParams& p, cudaStream_t st) {
  static_assert(CS <= MAX_CS, "partial slots");
  static std::mutex mu;
  static int cached_dev = -1, cached_clusters = 0;
  auto kern = cluster_kernel<CS>;
  int dev = 0;
  cudaGetDevice(&dev);
  cudaLaunchConfig_t cfg = {};
  cudaLaunchAttribute at[2];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = CS; at[0].val.clusterDim.y = 1; at[0].val.clusterDim.z = 1;
  at[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[1].val.programmaticStreamSerializationAllowed = 1;
  cfg.blockDim = dim3(CT); cfg.dynamicSmemBytes = smem_bytes(SLICE_CAP); cfg.stream = st;
  cfg.attrs = at; cfg.numAttrs = 1;
  int n_clusters;
  {
    std::lock_guard<std::mutex> lock(mu);
    if (cached_dev != dev) {
      cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, smem_bytes(SLICE_CAP));
      if (e == cudaSuccess && CS > 8) e = cudaFuncSetAttribute(kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
      if (e != cudaSuccess) return e;
      cfg.gridDim = dim3(CS * 64);
      int n = 0;
      e = cudaOccupancyMaxActiveClusters(&n, kern, &cfg);
      if (e != cudaSuccess) return e;
      if (n < 1 && CS <= 8) return cudaErrorLaunchOutOfResources;
      cached_clusters = n; cached_dev = dev;
    }
    n_clusters = cached_clusters;
  }
  if (CS > 8 && n_clusters < p.n_rows) return launch_cs<8>(p, st);       // (clusters of 16 need that many SMs in one part of the chip)
  if ((int64_t)n_clusters > p.n_rows) n_clusters = (int)p.n_rows;
  cfg.gridDim = dim3(CS * n_clusters);
  cfg.dynamicSmemBytes = smem_bytes(slice_of(p.V, CS));
  cfg.numAttrs = 2;
  return cudaLaunchKernelEx(&cfg, kern, p, n_clusters);
}

cudaError_t launch_cluster(const RowParams& p, cudaStream_t st, int* n_launches, bool* served) {
  *served = false;
  if (p.n_rows <= 0) { *served = true; return cudaSuccess; }
  int dev = 0, sms = 148;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  cudaError_t e;
  switch (pick_cs(p.V, p.call_rows, sms)) {
    case 1: e = launch_cs<1>(p, st); break;
    case 2: e = launch_cs<2>(p, st); break;
    case 4: e = launch_cs<4>(p, st); break;
    case 8: e = launch_cs<8>(p, st); break;
    default: e = launch_cs<16>(p, st); break;
  }
  if (e == cudaSuccess) { *served = true; if (n_launches) *n_launches += 1; }
  return e;
}

}  // namespace saki
