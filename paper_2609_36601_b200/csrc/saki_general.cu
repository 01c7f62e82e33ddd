// General row kernel: any V, dtype and strides, float64 arithmetic throughout.  It serves the layouts the bf16
// kernels do not (fp32 logits, odd strides, ragged V), and it is their second tier (rows they hand over through
// the row list).  Steps follow the method's definition:
//   log-softmax x2 -> lambda (Eqs. "bridge", "trust_region") -> TV and the
//   maximal coupling (Eqs. "accept", "residual") -> routed loss (Eqs.
//   "k1_loss_token", "teacher_mode_loss") -> gradient (Eq. "general_objective").
//
// What bounds it: the float64 pipe (64 lanes per clock and SM; a warp instruction occupies its scheduler's half of
// it for two clocks).  Hence:
//   - 2^y costs eight float64 operations (saki_exp2.cuh);
//   - three passes over the row: "sums" (two exponentials), one or two evaluations of KL with its first four
//     derivatives (one exponential each: the root of the fourth-order model, as in the bf16 kernels, here accepted
//     when the dropped terms move lambda by less than about 1e-11), "final" (two exponentials; total variation, draw
//     weights and the gradient in one pass).  The row's maxima come out of pass "sums" itself: every warp runs
//     under shifts fixed from its first elements (whole powers of two, so warps combine exactly) and repeats its
//     part with the true maxima if they turn out so much larger that its sums could have overflowed;
//   - the moments of the logit difference that only feed the first guess of lambda are float32.
// A warp owns a contiguous segment of the row in every pass (the residual draw is in index order), a row is owned by
// one block or by a cluster of blocks that add up their warps' partial sums through distributed shared memory.
#include "saki_exp2.cuh"
#include <cooperative_groups.h>
#include <algorithm>
#include <atomic>
#include <cmath>
#include <type_traits>

namespace cg = cooperative_groups;

namespace saki {

namespace {

constexpr int GT = 256;        // threads per block
constexpr int GW = GT / 32;    // warps per block
constexpr int MAX_CS = 8;      // blocks per row, at most
constexpr int NPART = 12;      // doubles a warp leaves per phase

struct Shared {
  double tab[EXP2_TAB * EXP2_COPIES];
  double part[2][GW][NPART];   // alternates from phase to phase: one barrier per phase is enough
  double bc[32];               // scalars broadcast to the block
  double sub[GW];
  alignas(16) unsigned char answer[16];
  uint64_t bar;
  int next[2];
};
enum { G_STATUS = 0, G_MODE, G_BETA, G_KP, G_CC, G_LSE_T, G_LAM, G_LOGZ, G_KL, G_LO, G_HI, G_ITER, G_AM, G_OWNER, G_BEFORE,
       G_TARGET, G_LAST, G_TV, G_TOK, G_SC, G_CORR, G_ACC, G_LPX, G_LTX, G_LOSS, G_ZERO, G_UACC, G_UDRAW, G_COUNT };
static_assert(G_COUNT <= 32, "broadcast area too small");
enum { PA_KS = 0, PA_KT, PA_SS, PA_ST, PA_N1, PA_M1, PA_M2, PA_M3, PA_M4, PA_MS, PA_MT, PA_AM };   // pass "sums" (AM: -1 - index if a logit is not finite)
enum { G_SOLVE = 0, G_FINAL = 1, G_FLAG = 2 };
constexpr int LOST = -2;

__device__ __forceinline__ double pow2_down(double n) {      // 2^n for whole n <= 0; 0 below -1000
  return n < -1000.0 ? 0.0 : __longlong_as_double((long long)(1023 + (int)n) << 52);
}

// Sixteen bytes of a row: eight bf16 or four fp32 elements.
template <typename T> struct Chunk;
template <> struct Chunk<__nv_bfloat16> {
  static constexpr int W = 8;
  uint32_t r[4];
  __device__ __forceinline__ float get(int i) const { return __uint_as_float((i & 1) ? r[i >> 1] & 0xffff0000u : r[i >> 1] << 16); }
  __device__ __forceinline__ void set2(int i, double a, double b) { r[i >> 1] = pack_bf16x2(to_odd(a), to_odd(b)); }
  static __device__ __forceinline__ void put(__nv_bfloat16* g, double v) { *g = __float2bfloat16_rn(to_odd(v)); }
};
template <> struct Chunk<float> {
  static constexpr int W = 4;
  uint32_t r[4];
  __device__ __forceinline__ float get(int i) const { return __uint_as_float(r[i]); }
  __device__ __forceinline__ void set2(int i, double a, double b) { r[i] = __float_as_uint((float)a); r[i + 1] = __float_as_uint((float)b); }
  static __device__ __forceinline__ void put(float* g, double v) { *g = (float)v; }
};
template <typename T> __device__ __forceinline__ Chunk<T> load_chunk(const T* p, bool vec) {
  Chunk<T> c;
  if (vec) {
    const uint4 q = __ldg((const uint4*)p);
    c.r[0] = q.x; c.r[1] = q.y; c.r[2] = q.z; c.r[3] = q.w;
  } else {   // a row whose 16-byte boundaries are not the student row's
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      if constexpr (sizeof(T) == 4) c.r[i] = __float_as_uint(p[i]);
      else c.r[i] = (uint32_t)__bfloat16_as_ushort(p[2 * i]) | ((uint32_t)__bfloat16_as_ushort(p[2 * i + 1]) << 16);
    }
  }
  return c;
}

// A warp's part of the row: the chunks [c0, c1) of the 16-byte chunks that start `head` elements into the row (the
// student row's first 16-byte boundary); the first warp also takes the elements before them, the last one those after.
struct Part { int c0, c1, head, x0, x1; };     // x0, x1: the extra elements (x0 == x1: none)

// The chunks and extra elements of a warp's part: chunk(first element, s, t) and element(v, s, t).  The next chunk is on
// its way while one is worked on (eight elements take a warp longer than a trip to memory).
template <typename T, typename FC, typename FE>
__device__ __forceinline__ void for_elements(const T* __restrict__ s, const T* __restrict__ t, bool tvec, const Part& pt, int lane,
                                             FC&& chunk, FE&& element) {
  constexpr int W = Chunk<T>::W;
  int k = pt.c0 + lane;
  if (k < pt.c1) {
    Chunk<T> a = load_chunk(s + pt.head + k * W, true), b = load_chunk(t + pt.head + k * W, tvec);
#pragma unroll 1
    for (; k < pt.c1; k += 32) {
      const int n = min(k + 32, pt.c1 - 1);
      const Chunk<T> na = load_chunk(s + pt.head + n * W, true), nb = load_chunk(t + pt.head + n * W, tvec);
      chunk(pt.head + k * W, a, b);
      a = na; b = nb;
    }
  }
#pragma unroll 1
  for (int v = pt.x0 + lane; v < pt.x1; v += 32) element(v, ld_as_float(s, v), ld_as_float(t, v));
}
template <typename T, typename FE>
__device__ __forceinline__ void for_elements(const T* __restrict__ s, const T* __restrict__ t, bool tvec, const Part& pt, int lane,
                                             FE&& element) {
  for_elements(s, t, tvec, pt, lane,
    [&](int v, const Chunk<T>& a, const Chunk<T>& b) {
#pragma unroll
      for (int i = 0; i < Chunk<T>::W; ++i) element(v + i, a.get(i), b.get(i));
    }, element);
}

// 1 / x of a sum of exponentials: short while x is in float32's range
__device__ __forceinline__ double rcp_sum(double x) { return x > 1e-30 && x < 1e30 ? rcp_fast(x) : 1.0 / x; }

// The scalars between the passes, on one warp per block (all lanes alike): first_guess, solve_step.
__device__ __noinline__ double first_guess(double m1, double m2, double m3, double m4, double rtau, double kl1, double eps) {
  const double var = m2 - m1 * m1, m1s = m1 * m1;
  const double c3 = m3 - 3.0 * m1 * m2 + 2.0 * m1 * m1s;
  const double c4 = m4 - 4.0 * m3 * m1 - 3.0 * m2 * m2 + 12.0 * m2 * m1s - 6.0 * m1s * m1s;
  const float rt = (float)rtau, vd = fmaxf((float)var * rt * rt, 1e-30f), k3 = (float)c3 * rt * rt * rt, k4 = (float)c4 * (rt * rt) * (rt * rt);
  const float e2 = 2.f * (float)eps;
  float b = sqrtf(__fdividef(e2, vd));
#pragma unroll 1
  for (int it = 0; it < 3; ++it) {
    const float bb = fminf(b, 1.f);
    const float den = vd + (2.f / 3.f) * bb * k3 + 0.25f * bb * bb * k4;
    if (den > 0.25f * vd) b = sqrtf(__fdividef(e2, den));
  }
  if (b > 0.45f) b = anchored_guess(b, vd, k3, k4, (float)kl1, (float)eps);
  if (!(b > 1e-7f)) b = 1e-7f;
  if (!(b < 0.98f)) b = 0.98f;
  return (double)b;
}

// One evaluation at beta: v[k] = sum p exp(beta d) d^k.  Returns true when lambda is settled (bc[G_LAM], bc[G_LOGZ], bc[G_KL]).
__device__ __noinline__ bool solve_step(double* bc, const double* v, double eps) {
  const double beta = bc[G_BETA], r0 = rcp_sum(v[0]), L = log(v[0]);
  const double m1 = v[1] * r0, m2 = v[2] * r0, m3 = v[3] * r0, m4 = v[4] * r0, m1s = m1 * m1;
  if (beta == 0.0) {                                         // the moments under p, for a guess on their scale (below)
    const double b = sqrt(2.0 * eps / (m2 - m1s)), top = 0.5 * bc[G_HI];
    __syncwarp();
    bc[G_BETA] = b > 0.0 && b < top ? b : top; bc[G_ZERO] = 1.0;
    __syncwarp();
    return false;
  }
  const double var = fmax(m2 - m1s, 0.0), k3 = m3 - 3.0 * m2 * m1 + 2.0 * m1s * m1;
  const double k4 = m4 - 4.0 * m3 * m1 - 3.0 * m2 * m2 + 12.0 * m2 * m1s - 6.0 * m1s * m1s;
  const double kl = beta * m1 - L, slope = beta * var;
  const double c2 = 0.5 * (beta * k3 + var), c3 = beta * k4 * (1.0 / 6.0) + k3 * (1.0 / 3.0), c4 = 0.125 * k4;
  double lo = bc[G_LO], hi = bc[G_HI];
  if (kl <= eps) lo = fmax(lo, beta); else hi = fmin(hi, beta);
  const int iter = (int)bc[G_ITER] + 1;
  // Lambda may lie on the scale of 1 / d of logits that the teacher masks (down to 1e-39 for float32's lowest value): there
  // steps and bracket are judged relative to beta.
  const double unit = beta < 1e-7 ? beta : 1.0;           // (below every first guess)
  // root of the fourth-order model of KL(beta + h) - eps
  const double f0 = eps - kl;
  double h = f0 / slope;
  bool ok = slope > 0.0;
#pragma unroll 1
  for (int it = 0; it < 20 && ok; ++it) {
    const double pv = h * (slope + h * (c2 + h * (c3 + h * c4))) - f0;
    const double dv = slope + h * (2.0 * c2 + h * (3.0 * c3 + h * (4.0 * c4)));
    if (!(dv > 0.25 * slope)) { ok = false; break; }
    const double dh = pv * rcp_sum(dv);
    h -= dh;
    if (fabs(dh) <= 1e-9 * fabs(h)) break;                   // (the next step would be the square of this one)
  }
  if (!ok) h = f0 / slope;                                   // the model bends over: Newton's step
  double nb = beta + h;
  bool bisected = false;
  if (!(nb > lo && nb < hi)) {
    // a step that is nothing but rounding may end on the wrong side of the bracket; a real one is halved (or, far apart on
    // the scale of masked logits, the bracket's exponent is).  With nothing known yet of the side of 0, the moments at 0 tell
    // the scale: the first guess had them in float32, where those of masked logits overflow.
    if (fabs(h) < 1e-13 * unit) nb = fmin(fmax(nb, lo), hi);
    else { nb = unit < 1.0 && lo > 0.0 && hi > 16.0 * lo ? sqrt(lo) * sqrt(hi) : 0.5 * (lo + hi); bisected = true; }
    if (bisected && lo == 0.0 && bc[G_ZERO] == 0.0) nb = 0.0;
  }
  h = nb - beta;
  // the first dropped term moves lambda by (k5 / k2) h^4 / 24; with D a scale of d under q, that is D^3 h^4 / 24
  const double rv = 1.0 / var, D2 = fmax(var, fmax(k3 * rv * k3 * rv, fabs(k4) * rv)), h2 = h * h;
  const bool done = (ok && !bisected && D2 * sqrt(D2) * h2 * h2 <= 2e-10 * unit) || fabs(h) < 1e-13 * unit || hi - lo < 1e-15 * unit || iter >= 100;
  __syncwarp();                                              // every lane has read the state
  if (done) {
    bc[G_LAM] = nb;
    bc[G_LOGZ] = L + h * (m1 + h * (0.5 * var + h * ((1.0 / 6.0) * k3 + h * (1.0 / 24.0) * k4)));
    bc[G_KL] = kl + h * (slope + h * (c2 + h * (c3 + h * c4)));
  } else {
    bc[G_BETA] = nb; bc[G_LO] = lo; bc[G_HI] = hi; bc[G_ITER] = (double)iter;
  }
  __syncwarp();
  return done;
}

}  // namespace

// CS: blocks per row (1, or a cluster of CS blocks); KS: blocks per SM.
template <typename T, int CS, int KS>
__global__ void __launch_bounds__(GT, KS) general_kernel(const RowParams P, const int steal, const double rtau, const double c) {
  __shared__ Shared sh;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int V = P.V;
  int crank = 0;
  if constexpr (CS > 1) crank = (int)cg::this_cluster().block_rank();
  constexpr int NWC = GW * CS;                               // warps of the row, in index order of their segments
  const int gw = crank * GW + warp;

  if (P.from_list) {
    wait_for_predecessor();
    launch_dependents();
  }
  if (P.from_list && *(volatile unsigned int*)P.redo_count == 0u) {      // an empty row list, as a rule
    if (blockIdx.x == 0) move_counters(P.redo_count);
    return;
  }
  const int64_t n_work = P.from_list ? (int64_t)*(volatile unsigned int*)P.redo_count : P.n_rows;
  if ((int64_t)(blockIdx.x / CS) >= n_work) {                // the whole cluster: nothing to do
    if (P.from_list) close_counters(P.redo_count);
    return;
  }
  exp2_table(sh.tab, tid, GT);
  if (tid == 0) {
    mbar_init(&sh.bar, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  __syncthreads();
  const Exp2 ex2(sh.tab, lane);
  if (!P.from_list) {
    if (steal) launch_dependents();
    wait_for_predecessor();
  }

  const double eps = (double)P.eps;     // (rtau = 1 / tau, c = log2(e) / tau)
  int ph = 0;
  double* const bc = sh.bc;

  // all warps' partial sums of a phase are in place
  auto phase_barrier = [&]() {
    if constexpr (CS == 1) __syncthreads(); else cg::this_cluster().sync();
  };
  // the record of warp w of the row (its segment order)
  auto part_of = [&](int w) -> const double* {
    if constexpr (CS == 1) return sh.part[ph][w];
    else return cg::this_cluster().map_shared_rank(&sh.part[ph][w % GW][0], w / GW);
  };

  const int64_t stride = gridDim.x / CS;
  int turn = 0, nxt = -1;
  for (int64_t item = blockIdx.x / CS; item >= 0 && item < n_work; item = steal ? (int64_t)nxt : item + stride) {
    const int64_t row = P.from_list ? (int64_t)P.redo_list[item] : item;   // list mode: rows handed over by the float32 kernels
    const int64_t b = P.K1 == 1 ? row : row / P.K1;
    const int j = (int)(row - b * P.K1);
    const T* const s = (const T*)P.s + b * P.s_seq + (int64_t)j * P.s_pos;
    const T* const t = (const T*)P.t + b * P.t_seq + (int64_t)j * P.t_pos;
    const bool bonus = P.spec && (j == P.K1 - 1);
    int x = 0;
    if (!bonus) x = P.spec ? P.proposal[b * P.prop_ld + j] : P.proposal[row];
    // the proposal's logits, for the scalar phase
    const int xc = min(max(x, 0), V - 1);
    const float sx = ld_as_float(s, xc), tx = ld_as_float(t, xc);
    const uint64_t rid = P.row_offset + (uint64_t)row;
    const bool masked = (P.mask != nullptr) && (P.mask[row] == 0);
    T* const g = P.dlogits ? (T*)P.dlogits + row * P.ld_g : nullptr;
    // this warp's part of the row
    constexpr int CW = Chunk<T>::W;
    const int head = min(V, (int)(((16u - (uint32_t)((uintptr_t)s & 15u)) & 15u) / sizeof(T)));
    const int nck = (V - head) / CW, cseg = (nck + NWC - 1) / NWC;
    Part pt;
    pt.head = head; pt.c0 = min(nck, gw * cseg); pt.c1 = min(nck, pt.c0 + cseg);
    pt.x0 = gw == 0 ? 0 : V; pt.x1 = gw == 0 ? head : V;
    if (gw == NWC - 1) pt.x0 = head + nck * CW;
    const bool tvec = ((uintptr_t)(t + head) & 15u) == 0, gvec = ((uintptr_t)(g + head) & 15u) == 0;
    auto part_begin = [&](int w) { return w == 0 ? 0 : head + min(nck, w * cseg) * CW; };
    auto part_end = [&](int w) { return w == NWC - 1 ? V : head + min(nck, (w + 1) * cseg) * CW; };
    if (steal && tid == 0 && crank == 0) steal_request(sh.answer, &sh.bar);
    // the row's uniforms, on a warp that does no scalars (the last row's are read before a barrier that this warp has passed)
    if (tid == 32) bc[G_UACC] = scalar_uniform(P.seed, rid, STAGE_ACCEPT);
    if (tid == 64) bc[G_UDRAW] = scalar_uniform(P.seed, rid, bonus ? STAGE_BONUS : STAGE_RESIDUAL);
    const float d0 = ld_as_float(t, 0) - ld_as_float(s, 0);  // the logit difference is taken about this one: no offset of hundreds in its moments

    // ---- pass "sums"
    {
      float ms = -CUDART_INF_F, mt = -CUDART_INF_F;
      const int seg0 = part_begin(gw), seg1 = part_end(gw);
      for (int v = seg0 + lane, u = 0; v < seg1 && u < 4; v += 32, ++u) { ms = fmaxf(ms, ld_as_float(s, v)); mt = fmaxf(mt, ld_as_float(t, v)); }
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) { ms = fmaxf(ms, __shfl_xor_sync(0xffffffffu, ms, o)); mt = fmaxf(mt, __shfl_xor_sync(0xffffffffu, mt, o)); }
      double ks = 0.0, kt = 0.0, ss, st, n1;
      float m1, m2, m3, m4;
      int am;
      bool again = false;
#pragma unroll 1
      for (int pass = 0; pass < 2; ++pass) {
        if (seg0 < seg1) { ks = -ceil(c * (double)ms); kt = -ceil(c * (double)mt); }
        ss = st = n1 = 0.0; m1 = m2 = m3 = m4 = 0.f;
        am = 0x7fffffff;
        float xs = -CUDART_INF_F, xt = -CUDART_INF_F;
        float2 f1 = {0.f, 0.f}, f2 = f1, f3 = f1, f4 = f1;
        const float2 nd0 = make_float2(-d0, -d0);
        auto pair = [&](float a0, float b0, float a1, float b1) {
          const double s0 = (double)a0, s1 = (double)a1, t0 = (double)b0, t1 = (double)b1;
          const double es0 = ex2(fma(c, s0, ks)), es1 = ex2(fma(c, s1, ks)), et0 = ex2(fma(c, t0, kt)), et1 = ex2(fma(c, t1, kt));
          ss += es0; ss += es1; st += et0; st += et1;
          n1 = fma(et0, t0 - s0, n1); n1 = fma(et1, t1 - s1, n1);
          const float2 d = fadd2(fadd2(make_float2(b0, b1), make_float2(-a0, -a1)), nd0), e = make_float2((float)es0, (float)es1);
          const float2 w1 = fmul2(e, d), q = fmul2(d, d);
          f1 = fadd2(f1, w1); f2 = ffma2(e, q, f2); f3 = ffma2(w1, q, f3); f4 = ffma2(fmul2(e, q), q, f4);
        };
        for_elements(s, t, tvec, pt, lane,
          [&](int v, const Chunk<T>& a, const Chunk<T>& bt) {
            float cx = bt.get(0);
#pragma unroll
            for (int i = 0; i < CW; i += 2) {
              pair(a.get(i), bt.get(i), a.get(i + 1), bt.get(i + 1));
              xs = fmaxf(fmaxf(xs, a.get(i)), a.get(i + 1)); cx = fmaxf(fmaxf(cx, bt.get(i)), bt.get(i + 1));
            }
            if (cx > xt) { xt = cx; am = v; }                // (the chunk; its element is found at the end)
          },
          [&](int v, float a, float bt) {
            const double s0 = (double)a, t0 = (double)bt, es = ex2(fma(c, s0, ks)), et = ex2(fma(c, t0, kt));
            ss += es; st += et; n1 = fma(et, t0 - s0, n1);
            const float d = (bt - a) - d0, e = (float)es, q = d * d;
            f1.x += e * d; f2.x += e * q; f3.x += e * d * q; f4.x += e * q * q;
            xs = fmaxf(xs, a);
            if (bt > xt || (bt == xt && v < am)) { xt = bt; am = v; }     // (the elements before the first chunk come after it here)
          });
        m1 = f1.x + f1.y; m2 = f2.x + f2.y; m3 = f3.x + f3.y; m4 = f4.x + f4.y;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
          xs = fmaxf(xs, __shfl_xor_sync(0xffffffffu, xs, o));
          const float oxt = __shfl_xor_sync(0xffffffffu, xt, o);
          const int oam = __shfl_xor_sync(0xffffffffu, am, o);
          if (oxt > xt || (oxt == xt && oam < am)) { xt = oxt; am = oam; }
        }
        {                                                    // the first element of that value in its chunk
          const int v = am + lane;
          const unsigned same = __ballot_sync(0xffffffffu, am < V && lane < CW && v < V && ld_as_float(t, min(v, V - 1)) == xt);
          if (same) am += __ffs(same) - 1;
        }
        again = fma(c, (double)xs, ks) > 300.0 || fma(c, (double)xt, kt) > 300.0;   // 2^y left its range: once more under the true maxima
        ms = xs; mt = xt;
        if (!again) break;
      }
      const double v8[8] = {ss, st, n1, (double)m1, (double)m2, (double)m3, (double)m4, 0.0};
      const double a = warp_sum8(v8, lane);
      // a logit that is not finite leaves n1 so (an exponential is never 0 and the difference is then infinite or NaN)
      const bool inf = __any_sync(0xffffffffu, lane < 12 && !(fabs(a) < CUDART_INF));
      double* const p = sh.part[ph][warp];
      static_assert(PA_ST == PA_SS + 1 && PA_N1 == PA_SS + 2 && PA_M4 == PA_SS + 6, "seven sums side by side");
      if ((lane & 3) == 0 && lane < 28) p[PA_SS + (lane >> 2)] = a;
      if (lane == 0) {
        p[PA_KS] = ks; p[PA_KT] = kt;
        p[PA_MS] = (double)ms; p[PA_MT] = (double)mt; p[PA_AM] = inf ? -1.0 : (double)am;
      }
    }
    if (steal && tid == 0 && crank == 0) {     // the next row, decided while pass "sums" ran: its number, -1 for none, or LOST - number
      int next = -1;
      if (mbar_wait_bounded(&sh.bar, (uint32_t)(turn & 1), P.wait_limit > 0 ? P.wait_limit : WAIT_LIMIT_CYCLES)) {
        const int first = steal_answer(sh.answer);
        next = first < 0 ? -1 : first / CS;
      } else if (mbar_wait_bounded(&sh.bar, (uint32_t)(turn & 1))) {     // late: the row it took over, if any, is flagged and no other is asked for
        const int first = steal_answer(sh.answer);
        next = first < 0 ? -1 : LOST - first / CS;
      } else {
        atomicAdd(P.flagged, 1ull);            // no answer at all: saki_check reports that a row may have been lost
      }
      sh.next[turn & 1] = next;
    }
    phase_barrier();
    if (steal) {
      if constexpr (CS == 1) nxt = sh.next[turn & 1];
      else nxt = *cg::this_cluster().map_shared_rank(&sh.next[turn & 1], 0);
      ++turn;
    }
    // the coupling decision and the constants of pass "final" (warp 0, once lambda is known)
    auto decide_row = [&](uint32_t status) {
      const double lam = bc[G_LAM], lse_s = -LN2 * bc[G_KP], lse_t = bc[G_LSE_T];
      double lp_x = 0.0, lT_x = 0.0, acc = 1.0;
      int corrected = 0, tok = -1;
      if (!bonus) {
        lp_x = (double)sx * rtau - lse_s;
        lT_x = (double)tx * rtau - lse_t;
        if (lam > 0.0) {
          acc = exp2_fast(fmin(0.0, lam * (lT_x - lp_x) - bc[G_LOGZ]) * INV_LN2);
          corrected = (bc[G_UACC] < acc) ? 0 : 1;
        }
      }
      double loss = 0.0, coef = 0.0;                         // gradient = coef (p - onehot(tok)) / tau
      if (masked) status |= SAKI_ROW_MASKED;
      else if (!bonus) {
        if (!corrected) { loss = (lp_x - lT_x) * lp_x; coef = -(lp_x - lT_x); tok = x; }
        else { coef = 1.0; tok = (int)bc[G_AM]; }            // (the loss, -log p(v*), is filled in when the row is written)
      }
      __syncwarp();
      bc[G_STATUS] = (double)status; bc[G_CORR] = (double)corrected; bc[G_TOK] = (double)tok;
      bc[G_SC] = (double)P.grad_scale * coef * rtau;
      bc[G_ACC] = acc; bc[G_LPX] = lp_x; bc[G_LTX] = lT_x; bc[G_LOSS] = loss; bc[G_MODE] = (double)G_FINAL;
    };
    if (warp == 0) {
      double S = 0.0, St = 0.0, N1 = 0.0, M1 = 0.0, M2 = 0.0, M3 = 0.0, M4 = 0.0, ms = -CUDART_INF, mt = -CUDART_INF, am = 2147483647.0;
      bool finite = true;
      for (int w = lane; w < NWC; w += 32) {
        const double* const p = part_of(w);
        if (p[PA_AM] < 0.0) finite = false;
        ms = fmax(ms, p[PA_MS]);
        if (p[PA_MT] > mt || (p[PA_MT] == mt && p[PA_AM] < am)) { mt = p[PA_MT]; am = p[PA_AM]; }
      }
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) {
        ms = fmax(ms, __shfl_xor_sync(0xffffffffu, ms, o));
        const double omt = __shfl_xor_sync(0xffffffffu, mt, o), oam = __shfl_xor_sync(0xffffffffu, am, o);
        if (omt > mt || (omt == mt && oam < am)) { mt = omt; am = oam; }
      }
      finite = __all_sync(0xffffffffu, finite);
      const double ks = -ceil(c * ms), kt = -ceil(c * mt);
      for (int w = lane; w < NWC; w += 32) {
        const double* const p = part_of(w);
        if (!(p[PA_MS] > -CUDART_INF)) continue;             // an empty segment
        const double fs = pow2_down(ks - p[PA_KS]), ft = pow2_down(kt - p[PA_KT]);
        S += fs * p[PA_SS]; St += ft * p[PA_ST]; N1 += ft * p[PA_N1];
        M1 += fs * p[PA_M1]; M2 += fs * p[PA_M2]; M3 += fs * p[PA_M3]; M4 += fs * p[PA_M4];
      }
      const double v8[8] = {S, St, N1, M1, M2, M3, M4, 0.0};
      const double a = warp_sum8(v8, lane);
      auto total = [&](int k) { return __shfl_sync(0xffffffffu, a, 4 * k); };
      S = total(0); St = total(1); N1 = total(2); M1 = total(3); M2 = total(4); M3 = total(5); M4 = total(6);
      uint32_t status = 0;
      if (!finite) status = SAKI_ROW_NONFINITE;
      else if (!bonus && (x < 0 || x >= V)) status = SAKI_ROW_BAD_ID;
      bc[G_AM] = am;
      if (status) { bc[G_STATUS] = (double)status; bc[G_MODE] = (double)G_FLAG; }
      else {
        // (as few roundings as there are: KL takes those of lse_s one to one, those of the short logarithm too)
        const double lse_s = fma(-LN2, ks, log(S)), lse_t = fma(-LN2, kt, log(St)), cc = lse_t - lse_s;
        bc[G_KP] = -INV_LN2 * lse_s; bc[G_CC] = cc; bc[G_LSE_T] = lse_t;
        const double kl1 = N1 * rcp_sum(St) * rtau - cc;      // KL(T || p)
        const bool endpoint = !(eps > 0.0) || kl1 <= eps;
        bc[G_LOGZ] = 0.0; bc[G_STATUS] = 0.0;
        bc[G_LAM] = !(eps > 0.0) ? 0.0 : 1.0; bc[G_KL] = !(eps > 0.0) ? 0.0 : kl1;
        __syncwarp();
        if (endpoint) decide_row(!(eps > 0.0) ? SAKI_ROW_EPS_ZERO : SAKI_ROW_SATURATED);
        else {
          const double rS = rcp_sum(S);
          double beta = first_guess(M1 * rS, M2 * rS, M3 * rS, M4 * rS, rtau, kl1, eps);
          if (P.from_list && P.redo_guess) {     // the float32 kernel's value of lambda, good to ~1e-5: one evaluation from here
            const double g0 = (double)P.redo_guess[item];
            if (g0 > 0.0 && g0 < 1.0) beta = g0;
          }
          bc[G_BETA] = beta; bc[G_LO] = 0.0; bc[G_HI] = 1.0; bc[G_ITER] = 0.0; bc[G_ZERO] = 0.0; bc[G_MODE] = (double)G_SOLVE;
        }
      }
    }
    __syncthreads();
    ph ^= 1;

    if ((int)bc[G_MODE] == G_FLAG) {   // flagged row: zero outputs, zero gradient row
      if (tid == 0 && crank == 0) {
        write_row(P.out, row, zero_row((uint32_t)bc[G_STATUS]), !P.spec);
        atomicAdd(P.flagged, 1ull);
      }
      if (g) for (int v = part_begin(gw) + lane; v < part_end(gw); v += 32) st_from_float(g, v, 0.f);
      continue;
    }

    // ---- pass "solve": one evaluation of KL(q_beta || p) and its derivatives
    const double kp = bc[G_KP], cc = bc[G_CC];
    while ((int)bc[G_MODE] == G_SOLVE) {
      const double bi = bc[G_BETA] * INV_LN2;
      double a0 = 0.0, a1 = 0.0, a2 = 0.0, a3 = 0.0, a4 = 0.0;
      for_elements(s, t, tvec, pt, lane, [&](int, float a, float bt) {
        const double sd = (double)a, d = fma((double)bt - sd, rtau, -cc);
        const double e = ex2(fma(bi, d, fma(c, sd, kp)));
        const double w1 = e * d, q = d * d, w2 = e * q;
        a0 += e; a1 += w1; a2 += w2; a3 = fma(w1, q, a3); a4 = fma(w2, q, a4);
      });
      const double v8[8] = {a0, a1, a2, a3, a4, 0.0, 0.0, 0.0};
      const double a = warp_sum8(v8, lane);
      if ((lane & 3) == 0 && lane < 20) sh.part[ph][warp][lane >> 2] = a;
      phase_barrier();
      if (warp == 0) {
        double v[5] = {0.0, 0.0, 0.0, 0.0, 0.0};
        for (int w = lane; w < NWC; w += 32) {
          const double* const p = part_of(w);
#pragma unroll
          for (int k = 0; k < 5; ++k) v[k] += p[k];
        }
        const double v8[8] = {v[0], v[1], v[2], v[3], v[4], 0.0, 0.0, 0.0};
        const double a = warp_sum8(v8, lane);
#pragma unroll
        for (int k = 0; k < 5; ++k) v[k] = __shfl_sync(0xffffffffu, a, 4 * k);
        if (solve_step(bc, v, eps)) decide_row(0u);
      }
      __syncthreads();
      ph ^= 1;
    }

    // (not earlier where the call leaves room: blocks of the next launch would take up what it leaves of each SM, unevenly;
    // 128 fp32 rows of 1024: 18.9 -> 14.9 us)
    if (!P.from_list && !steal) launch_dependents();
    // ---- pass "final": total variation, draw weights (of a bonus row: q itself) and the gradient
    // log2 q = cq s + cl t + kq: two operations instead of the four that the logit difference d takes
    const double lam = bc[G_LAM], cl = lam * c, cq = c - cl, kq = kp - INV_LN2 * (lam * cc + bc[G_LOGZ]);
    const bool corrected = bc[G_CORR] != 0.0, draw = corrected || bonus;
    // p = p_v, q = q_v; returns q - p
    auto diff = [&](float a, float bt, double& p, double& q) {
      const double sd = (double)a;
      p = ex2(fma(c, sd, kp));
      q = ex2(fma(cl, (double)bt, fma(cq, sd, kq)));
      return q - p;
    };
    double tv = 0.0, wq = 0.0;
    if (g) {
      const double sc = bc[G_SC];
      const int tok = (int)bc[G_TOK];
      auto grad = [&](float a, float bt) {
        double p, q;
        const double r = diff(a, bt, p, q);
        if (__double2hiint(r) >= 0) tv += r;                 // (the sign, without the float64 pipe)
        return sc * p;
      };
      auto at_token = [&]() { return sc * (ex2(fma(c, (double)ld_as_float(s, tok), kp)) - 1.0); };
      for_elements(s, t, tvec, pt, lane,
        [&](int v, const Chunk<T>& a, const Chunk<T>& bt) {
          Chunk<T> o;
#pragma unroll
          for (int i = 0; i < CW; i += 2) {
            const double g0 = grad(a.get(i), bt.get(i)), g1 = grad(a.get(i + 1), bt.get(i + 1));
            o.set2(i, g0, g1);
          }
          if (gvec) *(uint4*)(g + v) = make_uint4(o.r[0], o.r[1], o.r[2], o.r[3]);
          else {
#pragma unroll
            for (int i = 0; i < CW; ++i) st_from_float(g, v + i, o.get(i));
          }
          if ((unsigned)(tok - v) < (unsigned)CW) Chunk<T>::put(g + tok, at_token());
        },
        [&](int v, float a, float bt) { const double gv = grad(a, bt); Chunk<T>::put(g + v, v == tok ? at_token() : gv); });
    } else if (bonus) {
      for_elements(s, t, tvec, pt, lane, [&](int, float a, float bt) { double p, q; const double r = diff(a, bt, p, q); if (__double2hiint(r) >= 0) tv += r; wq += q; });
    } else if (lam > 0.0) {
      for_elements(s, t, tvec, pt, lane, [&](int, float a, float bt) { double p, q; const double r = diff(a, bt, p, q); if (__double2hiint(r) >= 0) tv += r; });
    }
    tv = warp_sum(tv);
    if (bonus) wq = warp_sum(wq);
    if (lane == 0) { sh.part[ph][warp][0] = tv; sh.part[ph][warp][1] = bonus ? wq : tv; }
    phase_barrier();
    if (warp == 0) {   // the total, and for a draw the warp that owns the inverse-CDF target
      double tvs = 0.0, wa[2] = {0.0, 0.0};
      constexpr int PER = NWC > 32 ? 2 : 1;                  // consecutive warps per lane: index order
#pragma unroll
      for (int q = 0; q < PER; ++q) {
        const int w = lane * PER + q;
        if (w < NWC) { const double* const p = part_of(w); tvs += p[0]; wa[q] = p[1]; }
      }
      tvs = warp_sum(tvs);
      int owner = 0;
      if (draw) {
        double inc = wa[0] + wa[1];
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
          const double up = __shfl_up_sync(0xffffffffu, inc, o);
          if (lane >= o) inc += up;
        }
        const double target = bc[G_UDRAW] * __shfl_sync(0xffffffffu, inc, 31);
        const unsigned hit = __ballot_sync(0xffffffffu, inc > target), pos = __ballot_sync(0xffffffffu, wa[0] + wa[1] > 0.0);
        // rounding left no crossing: the last index with positive weight
        const int ol = hit ? __ffs(hit) - 1 : (pos ? 31 - __clz(pos) : 0);
        double before = inc - (wa[0] + wa[1]);
        int q = 0;
        if (PER == 2 && (hit ? !(before + wa[0] > target) : wa[1] > 0.0)) { q = 1; before += wa[0]; }
        before = __shfl_sync(0xffffffffu, before, ol);
        owner = ol * PER + __shfl_sync(0xffffffffu, q, ol);
        bc[G_OWNER] = (double)owner; bc[G_BEFORE] = before; bc[G_TARGET] = target; bc[G_LAST] = hit ? 0.0 : 1.0;
      }
      bc[G_TV] = tvs;
    }
    int y = x;
    bool writer = tid == 0 && crank == 0;
    if (draw) {        // (all threads of the block agree)
      __syncthreads();
      const int owner = (int)bc[G_OWNER];
      writer = false;
      if (owner / GW == crank) {
        // the owner's segment once more, an eighth per warp; the warp whose part holds the target walks it
        const double target = bc[G_TARGET];
        bool last = bc[G_LAST] != 0.0;
        const int o0 = part_begin(owner), o1 = part_end(owner), sl = (((o1 - o0 + GW - 1) / GW) + 31) & ~31;
        auto weight = [&](int v) {
          double p, q;
          const double r = diff(ld_as_float(s, v), ld_as_float(t, v), p, q);
          return bonus ? q : fmax(r, 0.0);
        };
        double w = 0.0;
#pragma unroll 4
        for (int v = o0 + warp * sl + lane; v < min(o1, o0 + (warp + 1) * sl); v += 32) w += weight(v);
        w = warp_sum(w);
        if (lane == 0) sh.sub[warp] = w;
        __syncthreads();
        double running = bc[G_BEFORE], at = running;
        int mine = -1, lastpos = 0;
        double lastat = running;
        for (int k = 0; k < GW; ++k) {
          const double wk = sh.sub[k];
          if (wk > 0.0) { lastpos = k; lastat = running; }
          if (mine < 0 && !last && running + wk > target) { mine = k; at = running; }
          running += wk;
        }
        if (mine < 0) { mine = lastpos; at = lastat; last = true; }
        if (warp == mine) {
          int last_pos = -1, found = -1;
          const int e1 = min(o1, o0 + (mine + 1) * sl);
          const int b1 = o0 + mine * sl;
          double next = b1 + lane < e1 ? weight(b1 + lane) : 0.0;
          for (int v0 = b1; v0 < e1 && found < 0; v0 += 32) {
            const int v = v0 + lane;
            const double r = next;
            next = v + 32 < e1 ? weight(v + 32) : 0.0;       // (on its way while these are looked through)
            double inc = r;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
              const double up = __shfl_up_sync(0xffffffffu, inc, o);
              if (lane >= o) inc += up;
            }
            const unsigned pos = __ballot_sync(0xffffffffu, r > 0.0);
            const unsigned hit = last ? 0u : __ballot_sync(0xffffffffu, at + inc > target && v < e1);
            if (pos) last_pos = v0 + 31 - __clz(pos);
            if (hit) found = v0 + __ffs(hit) - 1;
            at += __shfl_sync(0xffffffffu, inc, 31);
          }
          if (found < 0) found = last_pos >= 0 ? last_pos : V - 1;
          y = found;
          writer = lane == 0;
        }
      }
    }
    if (writer) {
      const double lse_s = -LN2 * kp, lse_t = bc[G_LSE_T], Lam = bc[G_LOGZ];
      const double lp_x = bc[G_LPX], lT_x = bc[G_LTX];
      RowResult r;
      r.status = (uint32_t)bc[G_STATUS];
      r.corrected = corrected ? 1 : 0; r.token = y; r.vstar = (int)bc[G_AM];
      r.lambda = (float)lam; r.kl = (float)bc[G_KL];
      r.tv = lam > 0.0 ? (float)bc[G_TV] : 0.f;
      r.accept = bonus ? 0.f : (float)bc[G_ACC];
      r.logp_x = (float)lp_x; r.logT_x = (float)lT_x;
      r.logq_x = bonus ? 0.f : (float)(lp_x + lam * (lT_x - lp_x) - Lam);
      const double lp_y = (double)(y == x ? sx : ld_as_float(s, y)) * rtau - lse_s, lT_y = (double)(y == x ? tx : ld_as_float(t, y)) * rtau - lse_t;
      r.logp_y = (float)lp_y; r.logT_y = (float)lT_y;
      r.logq_y = (float)(lp_y + lam * (lT_y - lp_y) - Lam);
      r.loss = (float)bc[G_LOSS];
      if (corrected && !masked) r.loss = (float)-((double)ld_as_float(s, r.vstar) * rtau - lse_s);
      write_row(P.out, row, r, !P.spec);
    }
    ph ^= 1;
  }
  if (steal && nxt <= LOST) {                          // a row whose launch was cancelled by a request that was answered too late
    const int64_t row = (int64_t)LOST - nxt;
    if (tid == 0 && crank == 0) {
      write_row(P.out, row, zero_row(SAKI_ROW_TIMEOUT), !P.spec);
      atomicAdd(P.flagged, 1ull);
    }
    if (P.dlogits) for (int v = crank * GT + tid; v < V; v += CS * GT) st_from_float((T*)P.dlogits + row * P.ld_g, v, 0.f);
  }
  if constexpr (CS > 1) cg::this_cluster().sync();   // no block leaves while a peer may still read its shared memory
  if (P.from_list) close_counters(P.redo_count);
}

// blocks (clusters) that are resident at once: the grid, so that none starts after the others have finished
template <typename T, int CS, int KS>
static cudaError_t resident_rows(int dev, int sms, int* rows) {
  static std::atomic<int> fit_of[64];
  int fit = dev < 64 ? fit_of[dev].load(std::memory_order_relaxed) : 0;
  if (fit <= 0) {
    int n = 0;
    cudaError_t e;
    if (CS > 1) {
      cudaLaunchConfig_t cfg = {};
      cudaLaunchAttribute at[1];
      at[0].id = cudaLaunchAttributeClusterDimension;
      at[0].val.clusterDim.x = CS; at[0].val.clusterDim.y = 1; at[0].val.clusterDim.z = 1;
      cfg.blockDim = dim3(GT, 1, 1); cfg.gridDim = dim3(CS, 1, 1);
      cfg.attrs = at; cfg.numAttrs = 1;
      e = cudaOccupancyMaxActiveClusters(&n, general_kernel<T, CS, KS>, &cfg);
    } else {
      e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, general_kernel<T, CS, KS>, GT, 0);
      n *= sms;
    }
    if (e != cudaSuccess) return e;
    fit = n > 0 ? n : 1;
    if (dev < 64) fit_of[dev].store(fit, std::memory_order_relaxed);
  }
  *rows = fit;
  return cudaSuccess;
}

template <typename T, int CS, int KS>
static cudaError_t launch_cs(const RowParams& p, int dev, int sms, cudaStream_t st) {
  int fit = 1;
  const cudaError_t e = resident_rows<T, CS, KS>(dev, sms, &fit);
  if (e != cudaSuccess) return e;
  cudaLaunchConfig_t cfg = {};
  cfg.blockDim = dim3(GT, 1, 1);
  cfg.stream = st;
  cudaLaunchAttribute at[2];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[1].id = cudaLaunchAttributeClusterDimension;
  at[1].val.clusterDim.x = CS; at[1].val.clusterDim.y = 1; at[1].val.clusterDim.z = 1;
  cfg.attrs = at; cfg.numAttrs = CS > 1 ? 2 : 1;
  // One cluster per row where the hardware can be asked for the next one (a row's solve takes one evaluation or two,
  // and the rows do not divide evenly); in list mode, and for more rows than a grid may have blocks, a fixed stride.
  const bool steal = !p.from_list && p.n_rows > fit && p.n_rows <= (1 << 27);
  const double rtau = 1.0 / (double)p.temperature;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  if (p.from_list) fit = std::min(fit, std::max(1, sms / CS));     // as a rule they only find the list empty
  cfg.gridDim = dim3((unsigned)(CS * (p.n_rows < fit || steal ? p.n_rows : fit)), 1, 1);
  return cudaLaunchKernelEx(&cfg, general_kernel<T, CS, KS>, p, (int)steal, rtau, INV_LN2 * rtau);
}

// How a call is laid out: blocks per row (cs) and blocks per SM (k, by the registers a thread is given: 128, 80 or 64).  Two
// blocks per SM run a row soonest, more of them hide one another's serial steps and share an SM's slots out more finely.
//   - A call whose blocks are all resident two to an SM, and whose rows stay in L2 between the passes (200 MB: a pass behind
//     another finds most of 126 MB of L2 all the same), takes two, and as many blocks per row as fit and keep 4000 elements or more
//     (us, against as many blocks per row as are resident at four to an SM: fp32 64 rows of 1024 12.1 / 10.9, 64 of 16000 30.4 / 21.4,
//     148 of 50000 114 / 77; at three, bf16 148 rows of 16001 40.9 / 31.5, 64 of 100001 91 / 68).
//     Clusters of four and eight do not fill every SM (71 and 33 of them are resident, not 74 and 37): what does not fit takes half
//     the blocks per row (us, with the one or two rows of a second turn and now: fp32 34 rows of 32000 38 / 30, 72 of 64000 86 / 68, bf16 37 of 33001 46 / 33).
//     Where that leaves SMs out, or some SMs would have two blocks and others one, twice the blocks at three to an SM, if they are all
//     resident and keep 5000 elements or more (8000 in clusters of eight): fp32
//     190 rows of 50000 135 -> 113, 89 of 120000 183 -> 138, bf16 42 rows of 123205 79 -> 67.
//   - Of the others the one that takes the least by a cost model: turns, times what a turn takes of a row's serial steps, its
//     elements and the rows in flight beyond L2.  Fitted to the times of 605 calls of 200 to 4000 rows of 1024 to 151937, every layout
//     of the list: the choice is 0.9 % (fp32) and 0.6 % (bf16) above the best of them on average, 5 and 4 % or more for one call in
//     twenty, 9 and 24 % at worst (350 fp32 rows of 32000, 350 bf16 rows of 80001).
// The kernel pinned (call_rows = 0), the rows do not count, so that pieces of a batch agree with the whole to the bit: blocks per row
// by V alone, so many that the rows in flight stay in L2.  In list mode (a handful of rows as a rule; the host does not know
// their number) as many blocks per row as a row has 2048 elements for.
struct Layout { int cs, k; };
// fits(l): all rows of the call are resident at once in layout l
template <typename F>
static Layout pick_layout(int V, int64_t rows, bool from_list, bool f32, int sms, F&& fits) {
  const int64_t row_bytes = 2 * (int64_t)V * (f32 ? 4 : 2);
  int cs = 1;
  if (from_list || rows <= 0) {
    const int k = from_list ? 2 : f32 ? 4 : 3;
    while (cs < MAX_CS && V >= (from_list ? 2048 : 4096) * cs && (from_list || (int64_t)k * sms / cs * row_bytes > (150 << 20))) cs *= 2;
    return {cs, cs == 8 ? 2 : k};
  }
  if (rows <= 2 * sms && rows * row_bytes <= 200000000) {
    while (cs < MAX_CS && rows * 2 * cs <= 2 * sms && V >= 8000 * cs) cs *= 2;
    bool parted = false;
    while (cs > 1 && !fits(Layout{cs, 2})) { cs /= 2; parted = true; }
    const int wide = 2 * cs;
    if (wide <= MAX_CS && (parted || rows * cs > sms) && V >= (wide == 8 ? 64000 : 10000 * cs) && fits(Layout{wide, 3})) return {wide, 3};
    return {cs, 2};
  }
  static const Layout all[] = {{1, 2}, {1, 3}, {2, 2}, {4, 2}, {8, 2}, {1, 4}, {2, 4}, {4, 4}};     // (the last three: fp32)
  // bf16, fp32, in microseconds: a row's serial steps, 1000 elements of a block (by blocks per SM, two to four), a doubling of the
  // blocks; the part of a turn that is waited for to its end (blocks take over rows that have not started); 126 MB in flight beyond L2
  static const double serial[2][3] = {{15.2, 20.3}, {8.65, 10.5, 14.4}}, element[2][3] = {{2.42, 3.56}, {2.06, 3.35, 3.81}};
  static const double join[2] = {0.67, 0.45}, whole[2] = {0.014, 0.155}, beyond[2] = {0.49, 0.002};
  Layout best = all[0];
  double least = 1e300;
  for (int i = 0; i < (f32 ? 8 : 5); ++i) {
    const Layout l = all[i];
    if (l.cs > 1 && V < 4000 * l.cs) continue;
    const double slots = (double)(l.k * sms / l.cs), turns = (double)rows / slots, in_flight = std::min((double)rows, slots) * (double)row_bytes;
    if (l.cs == 1 && l.k > 2 && in_flight > 126e6) continue;         // (1024 fp32 rows of 32000: 336 us with four to an SM, 293 with two)
    double t = serial[f32][l.k - 2] + element[f32][l.k - 2] * 1e-3 * V / l.cs + join[f32] * std::log2((double)l.cs);
    t *= 1.0 + beyond[f32] * std::max(0.0, in_flight / 126e6 - 1.0);
    if (turns > 1.0) t *= whole[f32] * std::ceil(turns) + (1.0 - whole[f32]) * (turns + 0.5);
    if (t < least) { least = t; best = l; }
  }
  return best;
}

// f(blocks per row, blocks per SM) as constants, of the layouts that pick_layout gives for T
template <typename T, typename F>
static cudaError_t with_layout(Layout l, F&& f) {
  using std::integral_constant;
  if constexpr (sizeof(T) == 4) {
    switch (l.cs * 16 + l.k) {
      case 16 + 4: return f(integral_constant<int, 1>{}, integral_constant<int, 4>{});
      case 32 + 4: return f(integral_constant<int, 2>{}, integral_constant<int, 4>{});
      case 64 + 4: return f(integral_constant<int, 4>{}, integral_constant<int, 4>{});
    }
  }
  switch (l.cs * 16 + l.k) {
    case 16 + 3: return f(integral_constant<int, 1>{}, integral_constant<int, 3>{});
    case 32 + 2: return f(integral_constant<int, 2>{}, integral_constant<int, 2>{});
    case 32 + 3: return f(integral_constant<int, 2>{}, integral_constant<int, 3>{});
    case 64 + 2: return f(integral_constant<int, 4>{}, integral_constant<int, 2>{});
    case 64 + 3: return f(integral_constant<int, 4>{}, integral_constant<int, 3>{});
    case 128 + 2: return f(integral_constant<int, 8>{}, integral_constant<int, 2>{});
    case 128 + 3: return f(integral_constant<int, 8>{}, integral_constant<int, 3>{});
    default: return f(integral_constant<int, 1>{}, integral_constant<int, 2>{});
  }
}

static thread_local int g_layout[3];     // of the thread's last call: blocks per row, blocks per SM, rows resident at once
void general_layout(int* out) { std::copy(g_layout, g_layout + 3, out); }

template <typename T>
static cudaError_t launch_t(const RowParams& p, int dev, int sms, cudaStream_t st) {
  auto resident = [&](Layout l, int* rows) {
    return with_layout<T>(l, [&](auto cs, auto k) { return resident_rows<T, cs, k>(dev, sms, rows); });
  };
  auto fits = [&](Layout l) {              // (an error comes again, and is returned, where the layout is launched)
    int n = 0;
    return resident(l, &n) != cudaSuccess || p.call_rows <= n;
  };
  const Layout l = pick_layout(p.V, p.call_rows, p.from_list != 0, sizeof(T) == 4, sms, fits);
  if (!p.from_list) {
    g_layout[0] = l.cs; g_layout[1] = l.k;
    const cudaError_t e = resident(l, &g_layout[2]);
    if (e != cudaSuccess) return e;
  }
  return with_layout<T>(l, [&](auto cs, auto k) { return launch_cs<T, cs, k>(p, dev, sms, st); });
}

cudaError_t launch_general(const RowParams& p, int dtype, cudaStream_t st, int* n_launches) {
  if (p.n_rows <= 0) return cudaSuccess;
  int dev = 0, sms = 148;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  if (n_launches) *n_launches += 1;
  return dtype == SAKI_BF16 ? launch_t<__nv_bfloat16>(p, dev, sms, st) : launch_t<float>(p, dev, sms, st);
}

}  // namespace saki
