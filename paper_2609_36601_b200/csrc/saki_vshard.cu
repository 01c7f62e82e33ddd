// Vocabulary-sharded routing: every rank holds a contiguous slice [v0, v0 + V_local) of each logit row
// (as a tensor-parallel lm-head produces them) and the row is routed without ever gathering it.  The work
// is cut into stages; in each stage a rank reduces its slice to a few numbers per row (a "partial", a
// kernel here), the ranks exchange the partials (the caller's all-gather: ~100 bytes per row and stage),
// and every rank combines them, in rank order, into the same per-row state (a kernel here, and the same
// function compiled for the host).  What is computed is the definition (Eqs. "bridge", "trust_region",
// "accept", "residual", "k1_loss_token", "teacher_mode_loss", "general_objective"); sums, scalars and every
// combine in float64.  An evaluation
// of q_beta costs every rank a pass over its slice and the ranks an exchange, so the solver makes each one
// count: it carries the first four cumulants of the logit difference, the first guess is the root of the
// fourth-order series of KL(q_beta||p) at beta = 0, and each wave moves to the root of the fourth-order model
// at its beta (inside a bisection bracket); a step shorter than VS_SETTLE_STEP is taken without another look.
//   stage A  maxima, teacher argmax, the two sums of exponentials and the moments of the logit
//            difference under p (four) and T (one), each under the slice's own shift; the combine rescales
//   stage B  one evaluation of q_beta per wave: sum e delta^k, k = 0..4; repeated until every
//            row's lambda has settled (two waves as a rule)
//   stage C  the slice's share of TV = sum [q - p]_+ and of KL(q||p), the student's logit at the teacher's
//            argmax, and the gradient slice (acceptance is decided when lambda settles); the combine finds the rank
//            that owns the inverse-CDF target
//   stage D  on the owning rank the residual draw; the last combine writes the outputs (a caller that gives the
//            gradient's buffer here instead gets it from a pass of its own)
// Two families of slice kernels: float64 throughout (one block of 16 warps per row; any dtype, any alignment),
// and, further down, float32 per element for aligned bf16 slices.
#include "saki_exp2.cuh"
#include <math_constants.h>
#include <cmath>

namespace saki {

// per-row state, in doubles (the same on every rank after each combine)
enum { VS_MODE = 0,      // 0 solving, 1 settled, 2 flagged
       VS_STATUS, VS_MS, VS_MT, VS_VSTAR, VS_LSE_S, VS_LSE_T, VS_SX, VS_TX, VS_SV,
       VS_BETA, VS_LO, VS_HI, VS_ITER, VS_LAM, VS_LOGZ, VS_KL, VS_TV, VS_ACC, VS_CORR,
       VS_OWNER, VS_BEFORE, VS_TARGET, VS_TAKE_LAST, VS_TOK, VS_COEF, VS_LOSS, VS_Y, VS_SY, VS_TY,
       VS_F64,        // 1: the row is ill-conditioned for the float32 slice kernels, the float64 ones take it
       VS_COUNT };
static_assert(VS_COUNT <= SAKI_VSHARD_STATE, "state record too small");
enum { VS_SOLVING = 0, VS_SETTLED = 1, VS_FLAGGED = 2 };

struct VsConsts {
  int64_t N;
  int32_t V, world;
  double eps, tau;
  uint64_t seed, row_offset;
  const int32_t* proposal;
  const uint8_t* mask;
  int fast;          // the float32 slice kernels may be at work (a property of the call, the same on every rank)
};

// the second to fourth cumulants of delta from the sums  a_k = sum w delta^k, k = 0..4
__host__ __device__ inline void vs_cumulants(double a0, double a1, double a2, double a3, double a4, double& k2, double& k3,
                                             double& k4) {
  const double m1 = a1 / a0, r2 = a2 / a0, r3 = a3 / a0, r4 = a4 / a0;
  const double mu2 = r2 - m1 * m1;
  const double mu3 = r3 - 3.0 * m1 * r2 + 2.0 * m1 * m1 * m1;
  const double mu4 = r4 - 4.0 * m1 * r3 + 6.0 * m1 * m1 * r2 - 3.0 * m1 * m1 * m1 * m1;
  k2 = mu2; k3 = mu3; k4 = mu4 - 3.0 * mu2 * mu2;
}
// a wave's step shorter than this is taken without another evaluation: the model's error in lambda is of
// the order of (k5 / k2) step^4 / 24
constexpr double VS_SETTLE_STEP = 3e-3;

// The coupling decision and the gradient's coefficient of a row whose lambda is settled: they need no further sums, so
// the gradient can be written by the pass that takes the shares of TV.
__host__ __device__ inline void vs_decide(const VsConsts& c, int64_t i, double* st) {
  const double lam = st[VS_LAM];
  const double lp_x = st[VS_SX] / c.tau - st[VS_LSE_S], lT_x = st[VS_TX] / c.tau - st[VS_LSE_T];
  double acc = 1.0;
  int corrected = 0;
  if (lam > 0.0) {
    acc = exp(fmin(0.0, lam * (lT_x - lp_x) - st[VS_LOGZ]));
    corrected = (scalar_uniform(c.seed, c.row_offset + (uint64_t)i, STAGE_ACCEPT) < acc) ? 0 : 1;
  }
  const bool masked = c.mask != nullptr && c.mask[i] == 0;
  double loss = 0.0, coef = 0.0;
  int tok = -1;
  if (!masked) {
    if (!corrected) { loss = (lp_x - lT_x) * lp_x; coef = -(lp_x - lT_x); tok = c.proposal[i]; }
    else { coef = 1.0; tok = (int)st[VS_VSTAR]; }         // (the loss, -log p(v*), when the slices have sent s[v*])
  }
  st[VS_ACC] = acc; st[VS_CORR] = (double)corrected; st[VS_COEF] = coef; st[VS_TOK] = (double)tok; st[VS_LOSS] = loss;
}

// ---------------------------------------------------------------- the combine steps (host and device)
// `part`: row i's partial of rank 0, of SAKI_VSHARD_PARTIALS numbers; that of rank r stands r * rs further on.
struct VsMaxima { double ms, mt, am; bool finite; };
__host__ __device__ inline VsMaxima vs_maxima(const VsConsts& c, const double* part, int64_t rs) {
  VsMaxima m = {-INFINITY, -INFINITY, 2147483647.0, true};
  for (int r = 0; r < c.world; ++r) {
    const double* p = part + r * rs;
    if (p[3] == 0.0) m.finite = false;
    if (p[0] > m.ms) m.ms = p[0];
    if (p[1] > m.mt || (p[1] == m.mt && p[2] < m.am)) { m.mt = p[1]; m.am = p[2]; }   // lowest index among ties
  }
  return m;
}
// a rank's sums of stage A, from its own shifts onto the row's
enum { VA_SS = 0, VA_ST, VA_TD, VA_SD, VA_SD2, VA_SD3, VA_SD4, VA_COUNT };
__host__ __device__ inline void vs_rescale(const VsConsts& c, const double* p, const VsMaxima& m, double* v) {
  const double fs = p[4] > 0.0 ? exp((p[0] - m.ms) / c.tau) : 0.0, ft = p[5] > 0.0 ? exp((p[1] - m.mt) / c.tau) : 0.0;
  v[VA_SS] = v[VA_SD] = v[VA_SD2] = v[VA_SD3] = v[VA_SD4] = v[VA_ST] = v[VA_TD] = 0.0;
  if (p[4] > 0.0) { v[VA_SS] = fs * p[4]; v[VA_SD] = fs * p[7]; v[VA_SD2] = fs * p[8]; v[VA_SD3] = fs * p[12]; v[VA_SD4] = fs * p[13]; }
  if (p[5] > 0.0) { v[VA_ST] = ft * p[5]; v[VA_TD] = ft * p[6]; }
}
// `scaled`: the ranks' records of vs_rescale, `vs` apart; null: formed here
__host__ __device__ inline void vs_combine_a(const VsConsts& c, int64_t i, const double* part, int64_t rs, double* st,
                                             const VsMaxima& m, const double* scaled, int64_t vs) {
  for (int k = 0; k < SAKI_VSHARD_STATE; ++k) st[k] = 0.0;
  const double ms = m.ms, mt = m.mt, am = m.am;
  const bool finite = m.finite;
  const int x = c.proposal[i];
  uint32_t status = 0;
  if (!finite || !(ms > -INFINITY) || !(mt > -INFINITY)) status = SAKI_ROW_NONFINITE;
  else if (x < 0 || x >= c.V) status = SAKI_ROW_BAD_ID;
  st[VS_MS] = ms; st[VS_MT] = mt; st[VS_VSTAR] = am < 2147483647.0 ? am : 0.0;
  if (status) { st[VS_STATUS] = (double)status; st[VS_MODE] = VS_FLAGGED; return; }
  double Ss = 0.0, St = 0.0, Td = 0.0, Sd = 0.0, Sd2 = 0.0, Sd3 = 0.0, Sd4 = 0.0, sx = 0.0, tx = 0.0;
  for (int r = 0; r < c.world; ++r) {      // rank order: the summation order is part of the protocol
    const double* p = part + r * rs;
    double own[VA_COUNT];
    if (!scaled) vs_rescale(c, p, m, own);
    const double* const v = scaled ? scaled + r * vs : own;
    Ss += v[VA_SS]; St += v[VA_ST]; Td += v[VA_TD]; Sd += v[VA_SD]; Sd2 += v[VA_SD2]; Sd3 += v[VA_SD3]; Sd4 += v[VA_SD4];
    sx += p[9]; tx += p[10];
  }
  const double lse_s = ms / c.tau + log(Ss), lse_t = mt / c.tau + log(St);
  st[VS_LSE_S] = lse_s; st[VS_LSE_T] = lse_t; st[VS_SX] = sx; st[VS_TX] = tx;
  if (!(c.eps > 0.0)) {                                  // lambda = 0, log Z = 0
    st[VS_STATUS] = (double)SAKI_ROW_EPS_ZERO; st[VS_MODE] = VS_SETTLED;
    vs_decide(c, i, st);
    return;
  }
  const double cc = lse_t - lse_s;                       // d = delta - cc with delta = (t - s) / tau
  const double kl1 = Td / St - cc;                       // KL(T || p)
  if (kl1 <= c.eps) {                                    // teacher endpoint: q = T, log Z(1) = 0
    st[VS_LAM] = 1.0; st[VS_STATUS] = (double)SAKI_ROW_SATURATED; st[VS_MODE] = VS_SETTLED;
    vs_decide(c, i, st);
    return;
  }
  // First guess: d KL(q_beta||p) / d beta = beta Var_{q_beta}(d) and the variance under q_beta is
  // k2 + k3 beta + k4 beta^2 / 2 + ... in the cumulants of d under p (those of delta: d differs by a constant),
  // so KL = k2 beta^2 / 2 + k3 beta^3 / 3 + k4 beta^4 / 8 + ...; the root of that polynomial at eps, by Newton
  // from the root of its first term.
  double k2, k3, k4;
  vs_cumulants(Ss, Sd, Sd2, Sd3, Sd4, k2, k3, k4);
  double beta = sqrt(2.0 * c.eps / fmax(k2, 1e-300));
  if (!(beta > 0.0 && beta < 1.0)) beta = 0.5;
  {
    double b = beta;
    bool ok = true;
    for (int it = 0; it < 12 && ok; ++it) {
      const double f = b * b * (0.5 * k2 + b * (k3 / 3.0 + b * 0.125 * k4)) - c.eps;
      const double fp = b * (k2 + b * (k3 + b * 0.5 * k4));
      if (!(fp > 0.0)) { ok = false; break; }
      const double nb = b - f / fp;
      if (!(nb > 0.0 && nb < 1.0)) { ok = false; break; }
      const bool done = fabs(nb - b) < 1e-9;
      b = nb;
      if (done) break;
    }
    if (ok) beta = b;
  }
  st[VS_BETA] = beta; st[VS_LO] = 0.0; st[VS_HI] = 1.0; st[VS_MODE] = VS_SOLVING;
}

// One wave of the solver: from the sums at beta, KL(q_beta||p), the cumulants of d under q_beta and with them
// the model  KL(beta + h) = KL(beta) + int_0^h (beta + u) (k2 + k3 u + k4 u^2 / 2) du;  h = its root at eps (Newton
// from the first-order step), kept inside the bisection bracket.  Returns 1 if the row needs another wave.
__host__ __device__ inline int vs_combine_b(const VsConsts& c, int64_t i, const double* part, int64_t rs, double* st) {
  if ((int)st[VS_MODE] != VS_SOLVING) return 0;
  double a0 = 0.0, a1 = 0.0, a2 = 0.0, a3 = 0.0, a4 = 0.0;
  for (int r = 0; r < c.world; ++r) {
    const double* p = part + r * rs;
    a0 += p[0]; a1 += p[1]; a2 += p[2]; a3 += p[3]; a4 += p[4];
  }
  const double beta = st[VS_BETA], cc = st[VS_LSE_T] - st[VS_LSE_S];
  const double kb = ((1.0 - beta) * st[VS_MS] + beta * st[VS_MT]) / c.tau;    // the shift the partials were taken under
  double k2, k3, k4;
  vs_cumulants(a0, a1, a2, a3, a4, k2, k3, k4);
  const double E = a1 / a0 - cc;
  const double logZ = log(a0) + kb - (1.0 - beta) * st[VS_LSE_S] - beta * st[VS_LSE_T];
  const double kl = beta * E - logZ;
  double lo = st[VS_LO], hi = st[VS_HI];
  if (kl <= c.eps) lo = beta; else hi = beta;
  const int it = (int)st[VS_ITER] + 1;
  double h = (c.eps - kl) / (beta * k2);
  {
    double u = h;
    bool ok = isfinite(u);
    for (int n = 0; n < 12 && ok; ++n) {
      const double g = kl - c.eps + beta * u * (k2 + u * (0.5 * k3 + u * k4 / 6.0)) + u * u * (0.5 * k2 + u * (k3 / 3.0 + u * 0.125 * k4));
      const double gp = (beta + u) * (k2 + u * (k3 + u * 0.5 * k4));
      if (!(gp > 0.0)) { ok = false; break; }
      const double nu = u - g / gp;
      if (!isfinite(nu)) { ok = false; break; }
      const bool done = fabs(nu - u) < 1e-15;
      u = nu;
      if (done) break;
    }
    if (ok && fabs(u) <= 2.0 * fabs(h) + 1e-300) h = u;     // the model's root, unless it ran away from the first-order step
  }
  const bool inside = isfinite(h) && beta + h > lo && beta + h < hi;
  if (hi - lo < 1e-13 || it >= 100) h = 0.0;
  else if (!(inside && fabs(h) < VS_SETTLE_STEP)) {
    st[VS_BETA] = inside ? beta + h : 0.5 * (lo + hi);
    st[VS_LO] = lo; st[VS_HI] = hi; st[VS_ITER] = (double)it;
    return 1;
  }
  if (c.fast && st[VS_F64] == 0.0) {
    // The float32 slice kernels resolve KL to a few 1e-7 x (largest probability of either row).  Where that
    // would move lambda by more than a tenth of its tolerance (a very flat KL: nearly one-hot rows, whose TV
    // and acceptance probability move many times faster than lambda) the row goes on in float64.
    const double pmax = fmin(1.0, exp(fmax(st[VS_MS] / c.tau - st[VS_LSE_S], st[VS_MT] / c.tau - st[VS_LSE_T])));
    if (3e-7 * pmax > 1e-6 * beta * k2) {
      st[VS_F64] = 1.0;
      st[VS_BETA] = inside ? beta + h : beta;
      st[VS_LO] = 0.0; st[VS_HI] = 1.0; st[VS_ITER] = (double)it;     // the bracket came from float32 sums: start it over
      return 1;
    }
  }
  st[VS_LAM] = beta + h;
  st[VS_LOGZ] = logZ + h * (E + h * (0.5 * k2 + h * (k3 / 6.0 + h * k4 / 24.0)));   // log Z along beta: the cumulant series of d under q_beta
  st[VS_MODE] = VS_SETTLED;
  vs_decide(c, i, st);
  return 0;
}

// TV, KL, the coupling decision, the routed loss and the owner of the residual draw
__host__ __device__ inline void vs_combine_c(const VsConsts& c, int64_t i, const double* part, int64_t rs, double* st) {
  if ((int)st[VS_MODE] == VS_FLAGGED) return;
  double tv = 0.0, kl = 0.0, sv = 0.0;
  for (int r = 0; r < c.world; ++r) {
    const double* p = part + r * rs;
    tv += p[0]; kl += p[1]; sv += p[2];
  }
  const int x = c.proposal[i];
  const uint64_t rid = c.row_offset + (uint64_t)i;
  const bool corrected = st[VS_CORR] != 0.0;
  if (!(st[VS_LAM] > 0.0)) { tv = 0.0; kl = 0.0; }
  st[VS_SV] = sv; st[VS_TV] = tv; st[VS_KL] = kl;
  st[VS_OWNER] = -1.0; st[VS_Y] = (double)x; st[VS_SY] = st[VS_SX]; st[VS_TY] = st[VS_TX];
  if (corrected) {        // inverse CDF in index order: slices are contiguous, so rank order is index order
    const double target = scalar_uniform(c.seed, rid, STAGE_RESIDUAL) * tv;
    int owner = -1;
    double before = 0.0;
    for (int r = 0; r < c.world; ++r) {
      const double w = part[r * rs];
      if (before + w > target) { owner = r; break; }
      before += w;
    }
    double take_last = 0.0;
    if (owner < 0) {      // rounding left no crossing: the last index with positive weight
      take_last = 1.0; before = 0.0;
      for (int r = c.world - 1; r >= 0; --r) if (part[r * rs] > 0.0) { owner = r; break; }
      if (owner < 0) owner = c.world - 1;
    }
    st[VS_OWNER] = (double)owner; st[VS_BEFORE] = before; st[VS_TARGET] = target; st[VS_TAKE_LAST] = take_last;
  }
  if (c.mask != nullptr && c.mask[i] == 0) st[VS_STATUS] = (double)((uint32_t)st[VS_STATUS] | SAKI_ROW_MASKED);
  else if (corrected) st[VS_LOSS] = -(sv / c.tau - st[VS_LSE_S]);
}

// the drawn token and the per-position outputs
__host__ __device__ inline void vs_combine_d(const VsConsts& c, int64_t i, const double* part, int64_t rs, double* st, const saki_out& o) {
  if ((int)st[VS_MODE] == VS_FLAGGED) { write_row(o, i, zero_row((uint32_t)st[VS_STATUS]), true); return; }
  if (st[VS_CORR] != 0.0) {
    double y = -1.0, sy = 0.0, ty = 0.0;
    for (int r = 0; r < c.world; ++r) {
      const double* p = part + r * rs;
      if (p[0] >= 0.0) { y = p[0]; sy = p[1]; ty = p[2]; }
    }
    st[VS_Y] = y; st[VS_SY] = sy; st[VS_TY] = ty;
  }
  const double lam = st[VS_LAM], logZ = st[VS_LOGZ];
  RowResult r;
  r.corrected = (int)st[VS_CORR]; r.token = (int)st[VS_Y]; r.vstar = (int)st[VS_VSTAR];
  r.lambda = (float)lam; r.kl = (float)st[VS_KL]; r.tv = (float)st[VS_TV]; r.accept = (float)st[VS_ACC];
  const double lp_x = st[VS_SX] / c.tau - st[VS_LSE_S], lT_x = st[VS_TX] / c.tau - st[VS_LSE_T];
  const double lp_y = st[VS_SY] / c.tau - st[VS_LSE_S], lT_y = st[VS_TY] / c.tau - st[VS_LSE_T];
  r.logp_x = (float)lp_x; r.logT_x = (float)lT_x; r.logq_x = (float)(lp_x + lam * (lT_x - lp_x) - logZ);
  r.logp_y = (float)lp_y; r.logT_y = (float)lT_y; r.logq_y = (float)(lp_y + lam * (lT_y - lp_y) - logZ);
  r.loss = (float)st[VS_LOSS]; r.status = (uint32_t)st[VS_STATUS];
  write_row(o, i, r, true);
}

// ---------------------------------------------------------------- partial kernels: one block per row
constexpr int VT = 512, VW = VT / 32;

template <int NV>
__device__ __forceinline__ void vs_block_sum(double (&v)[NV], double* sh) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
  for (int k = 0; k < NV; ++k) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v[k] += __shfl_xor_sync(0xffffffffu, v[k], o);
  }
  if (lane == 0) {
#pragma unroll
    for (int k = 0; k < NV; ++k) sh[k * VW + warp] = v[k];
  }
  __syncthreads();
#pragma unroll
  for (int k = 0; k < NV; ++k) {
    double a = 0.0;
#pragma unroll
    for (int w = 0; w < VW; ++w) a += sh[k * VW + w];
    v[k] = a;
  }
  __syncthreads();
}

struct VsSlice {
  const void *s, *t;
  int64_t ld_s, ld_t, N;
  int32_t V_local, v0, rank;
  double tau;
  const int32_t* proposal;
  double* partial;
  void* dlogits;         // stages C and D; NULL: not wanted
  int64_t ld_g;
  int32_t fast;          // the float32 kernels can read this slice
};
// The slices of one launch (blockIdx.y): one for a rank of a distributed call, all of them where a process holds several
// ranks' slices (one launch per stage instead of one per rank: a slice of a thousand rows keeps the chip busy for 20 us).
constexpr int VS_GROUP = 16;
struct VsGroup { VsSlice s[VS_GROUP]; };

// The residual draw on the rank that owns the inverse-CDF target (all threads of the block call; NW warps).
// Every warp adds up the residual weights of its contiguous segment; the warp whose segment holds the target
// (segments in index order) walks it 32 elements at a time.  float64, whichever kernel family calls.
template <typename T, int NW>
__device__ __forceinline__ void vs_draw(const T* s, const T* t, int Vl, double rtau, const double* st, double* red, int* stoken, const Exp2& ex2) {
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const double lam = st[VS_LAM], lse_s = st[VS_LSE_S], lse_t = st[VS_LSE_T], logZ = st[VS_LOGZ];
  const double target = st[VS_TARGET];
  const bool take_last = st[VS_TAKE_LAST] != 0.0;
  const int seg = (Vl + NW - 1) / NW, v_lo = min(Vl, warp * seg), v_hi = min(Vl, v_lo + seg);
  auto weight = [&](int v) {
    const double lp = (double)ld_as_float(s, v) * rtau - lse_s, lT = (double)ld_as_float(t, v) * rtau - lse_t;
    return fmax(ex2((lp + lam * (lT - lp) - logZ) * INV_LN2) - ex2(lp * INV_LN2), 0.0);
  };
  double wsum = 0.0;
#pragma unroll 4
  for (int v = v_lo + lane; v < v_hi; v += 32) wsum += weight(v);
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) wsum += __shfl_xor_sync(0xffffffffu, wsum, o);
  if (lane == 0) red[warp] = wsum;
  __syncthreads();
  // the first warp whose running total passes the target; none (rounding, or the rule "last positive
  // element"): the last warp with weight
  double before = st[VS_BEFORE];
  int own_w = -1, last_w = -1;
  for (int w = 0; w < NW; ++w) {
    if (red[w] > 0.0) last_w = w;
    if (own_w < 0 && !take_last && before + red[w] > target) own_w = w;
    if (own_w < 0) before += red[w];
  }
  const bool walk_last = own_w < 0;
  if (walk_last) own_w = last_w;
  if (warp == own_w) {
    double running = before;
    int last_pos = -1, found = -1;
    for (int v0 = v_lo; v0 < v_hi && found < 0; v0 += 32) {
      const int v = v0 + lane;
      const double r = v < v_hi ? weight(v) : 0.0;
      double inc = r;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const double up = __shfl_up_sync(0xffffffffu, inc, o);
        if (lane >= o) inc += up;
      }
      const unsigned pos = __ballot_sync(0xffffffffu, r > 0.0);
      const unsigned hit = walk_last ? 0u : __ballot_sync(0xffffffffu, (running + inc > target) && v < v_hi);
      if (pos) last_pos = v0 + 31 - __clz(pos);
      if (hit) found = v0 + __ffs(hit) - 1;
      running += __shfl_sync(0xffffffffu, inc, 31);
    }
    if (found < 0) found = last_pos >= 0 ? last_pos : max(v_hi - 1, 0);   // rounding: the last element with weight in the segment
    if (lane == 0) *stoken = found;
  }
  if (own_w < 0 && tid == 0) *stoken = max(Vl - 1, 0);   // no weight anywhere in the slice
}

template <typename T>
__global__ void __launch_bounds__(VT) vs_partial_kernel(const __grid_constant__ VsGroup Gr, const int stage, const double* state,
                                                        const double grad_scale) {
  const VsSlice& S = Gr.s[blockIdx.y];
  double* const partial = S.partial;
  void* const dlogits = S.dlogits;
  const int64_t ld_g = S.ld_g;
  const bool only_flagged = S.fast != 0;     // the float32 kernel has the other rows
  __shared__ double red[7 * VW];
  __shared__ float smax[2][VW];
  __shared__ int sarg[VW];
  __shared__ int stoken;
  __shared__ unsigned char marks[VT];
  __shared__ double row_state[SAKI_VSHARD_STATE];
  __shared__ double tab[EXP2_TAB * EXP2_COPIES];
  bool table = false;
  const Exp2 ex2(tab, threadIdx.x & 31);
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int Vl = S.V_local;
  const double rtau = 1.0 / S.tau;
  // (in this order: the float32 kernel of the same stage, launched right behind, starts without a wait of its own from stage B on)
  wait_for_predecessor();
  launch_dependents();
  // rows in groups of VT, dealt out to the blocks; where only marked rows count, a thread looks at one row's mark (as a
  // rule none is marked, and a block is done after one load; before the first combine none can be)
  const int64_t n_rows = only_flagged && stage == 0 ? 0 : S.N;
  for (int64_t base = blockIdx.x; base < n_rows; base += (int64_t)gridDim.x * VT) {
    const int64_t mine_row = base + (int64_t)tid * gridDim.x;
    if (only_flagged) {
      const bool marked = mine_row < S.N && __ldcg(state + mine_row * SAKI_VSHARD_STATE + VS_F64) != 0.0;
      marks[tid] = marked ? 1 : 0;
      if (!__syncthreads_or(marked)) continue;
    }
    if (!table) {
      exp2_table(tab, tid, VT);
      __syncthreads();
      table = true;
    }
    for (int64_t row = base; row < S.N && row < base + (int64_t)gridDim.x * VT; row += gridDim.x) {
      const T* s = (const T*)S.s + row * S.ld_s;
      const T* t = (const T*)S.t + row * S.ld_t;
      double* out = partial + row * SAKI_VSHARD_PARTIALS;
      if (only_flagged && !marks[(row - base) / gridDim.x]) continue;   // the float32 kernel has this row
      const double* const st = row_state;
      if (state) {
        __syncthreads();                       // the last row is done with row_state
        if (tid < SAKI_VSHARD_STATE) row_state[tid] = __ldcg(state + row * SAKI_VSHARD_STATE + tid);
        __syncthreads();
      }
      if (stage == 0) {
        // ---- stage A: maxima and argmax, then the sums under this slice's own shifts
        float ms = -CUDART_INF_F, mt = -CUDART_INF_F;
        int am = 0x7fffffff, finite = 1;
#pragma unroll 4
        for (int v = tid; v < Vl; v += VT) {
          const float a = ld_as_float(s, v), c = ld_as_float(t, v);
          finite &= (isfinite(a) && isfinite(c)) ? 1 : 0;
          ms = fmaxf(ms, a);
          if (c > mt) { mt = c; am = v; }
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
          ms = fmaxf(ms, __shfl_xor_sync(0xffffffffu, ms, o));
          const float omt = __shfl_xor_sync(0xffffffffu, mt, o);
          const int oam = __shfl_xor_sync(0xffffffffu, am, o);
          if (omt > mt || (omt == mt && oam < am)) { mt = omt; am = oam; }
        }
        if (lane == 0) { smax[0][warp] = ms; smax[1][warp] = mt; sarg[warp] = am; }
        finite = __syncthreads_and(finite);
        ms = smax[0][0]; mt = smax[1][0]; am = sarg[0];
        for (int w = 1; w < VW; ++w) {
          ms = fmaxf(ms, smax[0][w]);
          if (smax[1][w] > mt || (smax[1][w] == mt && sarg[w] < am)) { mt = smax[1][w]; am = sarg[w]; }
        }
        __syncthreads();
        double a[7] = {0.0, 0.0, 0.0, 0.0, 0.0, 0.0, 0.0};
        if (finite && Vl > 0) {
          const double zms = (double)ms * rtau, zmt = (double)mt * rtau;
#pragma unroll 4
          for (int v = tid; v < Vl; v += VT) {
            const double zs = (double)ld_as_float(s, v) * rtau, zt = (double)ld_as_float(t, v) * rtau;
            const double es = ex2((zs - zms) * INV_LN2), et = ex2((zt - zmt) * INV_LN2), dl = zt - zs, ed = es * dl, ed2 = ed * dl;
            a[0] += es; a[1] += et; a[2] += et * dl; a[3] += ed; a[4] += ed2; a[5] += ed2 * dl; a[6] += ed2 * dl * dl;
          }
        }
        vs_block_sum<7>(a, red);
        if (tid == 0) {
          const int x = S.proposal[row] - S.v0;
          const bool own = x >= 0 && x < Vl;
          out[0] = (double)ms; out[1] = (double)mt; out[2] = am == 0x7fffffff ? 2147483647.0 : (double)(S.v0 + am);
          out[3] = finite ? 1.0 : 0.0;
          out[4] = a[0]; out[5] = a[1]; out[6] = a[2]; out[7] = a[3]; out[8] = a[4];
          out[9] = own ? (double)ld_as_float(s, x) : 0.0; out[10] = own ? (double)ld_as_float(t, x) : 0.0;
          out[11] = own ? 1.0 : 0.0;
          out[12] = a[5]; out[13] = a[6]; out[14] = 0.0; out[15] = 0.0;
        }
      } else if (stage == 1) {
        // ---- stage B: one evaluation at the row's current beta, under the row's global shift
        double a[5] = {0.0, 0.0, 0.0, 0.0, 0.0};
        if ((int)st[VS_MODE] == VS_SOLVING) {
          const double beta = st[VS_BETA];
          const double kb = ((1.0 - beta) * st[VS_MS] + beta * st[VS_MT]) * rtau;
#pragma unroll 4
          for (int v = tid; v < Vl; v += VT) {
            const double zs = (double)ld_as_float(s, v) * rtau, zt = (double)ld_as_float(t, v) * rtau;
            const double dl = zt - zs, e = ex2((zs + beta * dl - kb) * INV_LN2), ed = e * dl, ed2 = ed * dl;
            a[0] += e; a[1] += ed; a[2] += ed2; a[3] += ed2 * dl; a[4] += ed2 * dl * dl;
          }
        }
        vs_block_sum<5>(a, red);
        if (tid == 0) {
          for (int k = 0; k < SAKI_VSHARD_PARTIALS; ++k) out[k] = 0.0;
          out[0] = a[0]; out[1] = a[1]; out[2] = a[2]; out[3] = a[3]; out[4] = a[4];
        }
      } else if (stage == 2) {
        // ---- stage C: the slice's share of TV and KL(q||p); the student's logit at the teacher's argmax
        double a[2] = {0.0, 0.0};
        const bool live = (int)st[VS_MODE] == VS_SETTLED;
        const double lam = st[VS_LAM];
        if (live && lam > 0.0) {
          const double lse_s = st[VS_LSE_S], lse_t = st[VS_LSE_T], logZ = st[VS_LOGZ];
          // per-warp segments in index order, summed in warp order: close to the index-order sum of the definition
          const int seg = (Vl + VW - 1) / VW, v_lo = warp * seg, v_hi = min(Vl, v_lo + seg);
#pragma unroll 4
          for (int v = v_lo + lane; v < v_hi; v += 32) {
            const double lp = (double)ld_as_float(s, v) * rtau - lse_s, lT = (double)ld_as_float(t, v) * rtau - lse_t;
            const double lq = lp + lam * (lT - lp) - logZ, q = ex2(lq * INV_LN2);
            a[0] += fmax(q - ex2(lp * INV_LN2), 0.0);
            a[1] += q * (lq - lp);
          }
        }
        vs_block_sum<2>(a, red);
        if (tid == 0) {
          for (int k = 0; k < SAKI_VSHARD_PARTIALS; ++k) out[k] = 0.0;
          const int vs = (int)st[VS_VSTAR] - S.v0;
          out[0] = a[0]; out[1] = a[1];
          out[2] = (live && vs >= 0 && vs < Vl) ? (double)ld_as_float(s, vs) : 0.0;
        }
      } else {
        // ---- stage D: on the owning rank the residual draw
        const int mode = (int)st[VS_MODE];
        if (tid == 0) stoken = -1;
        __syncthreads();
        const bool mine = mode == VS_SETTLED && st[VS_CORR] != 0.0 && (int)st[VS_OWNER] == S.rank;
        if (mine) vs_draw<T, VW>(s, t, Vl, rtau, st, red, &stoken, ex2);
        __syncthreads();
        if (tid == 0) {
          for (int k = 0; k < SAKI_VSHARD_PARTIALS; ++k) out[k] = 0.0;
          out[0] = -1.0;
          if (mine && stoken >= 0 && stoken < Vl) {
            out[0] = (double)(S.v0 + stoken);
            out[1] = (double)ld_as_float(s, stoken); out[2] = (double)ld_as_float(t, stoken);
          }
        }
        __syncthreads();
      }
      if (stage >= 2 && dlogits) {
        // ---- the gradient slice (with stage C, or with stage D)
        const int mode = (int)st[VS_MODE];
        T* g = (T*)dlogits + row * ld_g;
        const double sc = mode == VS_FLAGGED ? 0.0 : grad_scale * st[VS_COEF] * rtau;
        const double lse_s = st[VS_LSE_S];
        const int tok = mode == VS_FLAGGED ? -1 : (int)st[VS_TOK] - S.v0;
#pragma unroll 4
        for (int v = tid; v < Vl; v += VT) {
          double gv = 0.0;
          if (sc != 0.0) gv = sc * (ex2(((double)ld_as_float(s, v) * rtau - lse_s) * INV_LN2) - (v == tok ? 1.0 : 0.0));
          if constexpr (sizeof(T) == 2) g[v] = __float2bfloat16_rn(to_odd(gv));
          else g[v] = (float)gv;
        }
      }
    }
    if (only_flagged) __syncthreads();       // a warp that is through with the group overwrites its marks with the next group's
  }
}

// ---------------------------------------------------------------- the float32 slice kernels
// The same partials for bf16 slices that start on a 16-byte boundary, with the per-element arithmetic of the
// row-per-SM kernel: packed f32x2 FMAs, ex2.approx under whole-number exponent shifts (the factor between such
// a shift and the one the partial is defined under is applied once per row, in float64), float32 sums per thread,
// float64 across threads.  One block of four warps per row slice, several blocks per SM.  A row whose state says
// VS_F64 is left to the float64 kernel, which is launched for those rows only and runs beside this one.
constexpr int FT = 128, FW = FT / 32;
constexpr uint32_t VF_FILLER = 0xFF7FFF7Fu;       // two bf16 of the most negative finite value
constexpr double VF_LOG2E = 1.4426950408889634;

template <int NV>
__device__ __forceinline__ void vf_block_sum(double (&v)[NV], double* sh) {   // the totals are valid in thread 0
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
  for (int k = 0; k < NV; ++k) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v[k] += __shfl_xor_sync(0xffffffffu, v[k], o);
  }
  if (lane == 0) {
#pragma unroll
    for (int k = 0; k < NV; ++k) sh[k * FW + warp] = v[k];
  }
  __syncthreads();
  if (threadIdx.x == 0) {
#pragma unroll
    for (int k = 0; k < NV; ++k) {
      double a = 0.0;
#pragma unroll
      for (int w = 0; w < FW; ++w) a += sh[k * FW + w];
      v[k] = a;
    }
  }
  __syncthreads();
}
__device__ __forceinline__ uint4 vf_ld(const __nv_bfloat16* p) {
  uint4 v;
  asm volatile("ld.global.nc.L1::no_allocate.v4.u32 {%0, %1, %2, %3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "l"(p));
  return v;
}
__device__ __forceinline__ double vf_tot(const float2 a) { return (double)a.x + (double)a.y; }
// sums of e (d - D)^k, k = 0..4, to sums of e d^k (in place): the kernels take the moments about a constant near the
// mean of the logit difference, where float32 products keep their digits; the partials are defined about zero
__device__ __forceinline__ void vf_uncentre(double D, double a0, double& a1, double& a2, double& a3, double& a4) {
  const double D2 = D * D, D3 = D2 * D, D4 = D2 * D2;
  a4 = a4 + 4.0 * D * a3 + 6.0 * D2 * a2 + 4.0 * D3 * a1 + D4 * a0;
  a3 = a3 + 3.0 * D * a2 + 3.0 * D2 * a1 + D3 * a0;
  a2 = a2 + 2.0 * D * a1 + D2 * a0;
  a1 = a1 + D * a0;
}

// The residual draw of the float32 kernels on the owning rank (all threads of the block call): weights
// [q - p]_+ per element in float32 (in units of fq, like stage C), sums in float64.  Every warp adds up its
// contiguous range of chunks; the warp that holds the target walks its range 32 chunks at a time, the lane whose
// chunk holds it walks the chunk's 8 elements.
__device__ __forceinline__ void vf_draw(const __nv_bfloat16* s, const __nv_bfloat16* t, int n_chunks, float c32, double c64,
                                        double tau, const double* st, double* red, int* stoken) {
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const double lam = st[VS_LAM], target = st[VS_TARGET];
  const bool take_last = st[VS_TAKE_LAST] != 0.0;
  float cl = (float)(c64 * lam);
  const float ccl = c32 - cl;
  cl = c32 - ccl;
  const float msf = (float)st[VS_MS], mtf = (float)st[VS_MT];
  // (the log-sum-exps relative to the maxima: what the sums of 2^(c s'), 2^(c t') came to)
  const double ls = st[VS_LSE_S] - st[VS_MS] / tau, lt = st[VS_LSE_T] - st[VS_MT] / tau;
  const double kp2 = ls * VF_LOG2E, kq2 = ((1.0 - lam) * ls + lam * lt + st[VS_LOGZ]) * VF_LOG2E;
  const float kpi = floorf((float)kp2 - 1e-3f), kqi = floorf((float)kq2 - 1e-3f);
  const double fp = exp2((double)kpi - kp2), fq = exp2((double)kqi - kq2);
  const float2 cc = splat(c32), cll = splat(cl), ccll = splat(ccl), kpp = splat(-kpi), kqq = splat(-kqi);
  const float2 nms = splat(-msf), nmt = splat(-mtf);
  const float2 nrho = splat(-(float)(fp / fq));
  auto weights_of = [&](const uint4 s4, const uint4 t4, float (&w)[8]) {
    const uint32_t sw[4] = {s4.x, s4.y, s4.z, s4.w}, tw[4] = {t4.x, t4.y, t4.z, t4.w};
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const float2 sf = fadd2(unpack_bf16x2(sw[i]), nms), tf = fadd2(unpack_bf16x2(tw[i]), nmt);
      const float2 ep = ex2f2(ffma2(sf, cc, kpp));
      const float2 eq = ex2f2(ffma2(tf, cll, ffma2(sf, ccll, kqq)));
      const float2 r = ffma2(ep, nrho, eq);
      w[2 * i] = fmaxf(r.x, 0.f); w[2 * i + 1] = fmaxf(r.y, 0.f);
    }
  };
  auto total = [&](const float (&w)[8]) { return fq * (double)(((w[0] + w[1]) + (w[2] + w[3])) + ((w[4] + w[5]) + (w[6] + w[7]))); };
  auto weights = [&](int c, float (&w)[8]) { weights_of(vf_ld(s + (size_t)c * 8), vf_ld(t + (size_t)c * 8), w); };
  const int seg = (n_chunks + FW - 1) / FW, c_lo = min(n_chunks, warp * seg), c_hi = min(n_chunks, c_lo + seg);
  double wsum = 0.0;
#pragma unroll 1
  for (int b = c_lo + lane; b < c_hi; b += 4 * 32) {       // (four chunks on their way at a time)
    uint4 sv[4], tv[4];
#pragma unroll
    for (int u = 0; u < 4; ++u)
      if (b + u * 32 < c_hi) { sv[u] = vf_ld(s + (size_t)(b + u * 32) * 8); tv[u] = vf_ld(t + (size_t)(b + u * 32) * 8); }
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      if (b + u * 32 >= c_hi) break;
      float w[8];
      weights_of(sv[u], tv[u], w);
      wsum += total(w);
    }
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) wsum += __shfl_xor_sync(0xffffffffu, wsum, o);
  if (lane == 0) red[warp] = wsum;
  __syncthreads();
  double before = st[VS_BEFORE];
  int own_w = -1, last_w = -1;
  for (int w = 0; w < FW; ++w) {
    if (red[w] > 0.0) last_w = w;
    if (own_w < 0 && !take_last && before + red[w] > target) own_w = w;
    if (own_w < 0) before += red[w];
  }
  const bool walk_last = own_w < 0;
  if (walk_last) own_w = last_w;
  if (warp == own_w) {
    double running = before;
    int found = -1, last_c = -1;
    float next[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
    if (c_lo + lane < c_hi) weights(c_lo + lane, next);
    for (int c0 = c_lo; c0 < c_hi && found < 0; c0 += 32) {
      const int c = c0 + lane;
      float w[8];
#pragma unroll
      for (int i = 0; i < 8; ++i) { w[i] = next[i]; next[i] = 0.f; }
      if (c + 32 < c_hi) weights(c + 32, next);       // (on its way while this step is looked through)
      const double mine = total(w);
      double inc = mine;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const double up = __shfl_up_sync(0xffffffffu, inc, o);
        if (lane >= o) inc += up;
      }
      const unsigned pos = __ballot_sync(0xffffffffu, mine > 0.0);
      const unsigned hit = walk_last ? 0u : __ballot_sync(0xffffffffu, running + inc > target);
      if (pos) last_c = c0 + 31 - __clz(pos);
      if (hit) {
        const int src = __ffs(hit) - 1;
        int f = -1;
        if (lane == src) {
          double run = running + inc - mine;
#pragma unroll
          for (int i = 0; i < 8; ++i) {
            run += fq * (double)w[i];
            if (f < 0 && run > target) f = c * 8 + i;
          }
          if (f < 0) {                                // rounding inside the chunk: its last element with weight
#pragma unroll
            for (int i = 0; i < 8; ++i) if (w[i] > 0.f) f = c * 8 + i;
          }
        }
        found = __shfl_sync(0xffffffffu, f, src);
      }
      running += __shfl_sync(0xffffffffu, inc, 31);
    }
    if (found < 0 && last_c >= 0) {                   // no crossing: the last element with weight in the range
      float w[8];
      weights(last_c, w);
#pragma unroll
      for (int i = 0; i < 8; ++i) if (w[i] > 0.f) found = last_c * 8 + i;
    }
    if (found < 0) found = max(c_hi * 8 - 1, 0);
    if (lane == 0) *stoken = found;
  }
  if (own_w < 0 && tid == 0) *stoken = max(n_chunks * 8 - 1, 0);   // no weight anywhere in the slice
}

template <int STAGE>
__global__ void __launch_bounds__(FT) vs_fast_kernel(const __grid_constant__ VsGroup Gr, const double* state, const double grad_scale,
                                                     const bool beside) {
  const VsSlice& S = Gr.s[blockIdx.y];
  // beside: the float64 kernel of the same stage was launched right before and lets this one start once all of its blocks
  // have seen the combine before it complete.  The two touch different rows, so the marked rows are routed while this
  // kernel runs, and the wait stands at the end: the next combine starts when both are done.  (With the float64 kernel
  // behind this one it could only start with the last of these blocks, and 28 of the 31 us that it takes in stage C
  // for 1024 rows of 151936 in eight slices came on top.)
  // Not in stage A (rows of slices of either kind): it reads the caller's logits and proposals, which the kernel in front of the
  // call may just have written, past no wait of its own.  From stage B on those are old, and what the combine wrote is read with
  // __ldcg.
  if (!beside) wait_for_predecessor();
  launch_dependents();
  if (!S.fast) {
    if (beside) wait_for_predecessor();
    return;
  }
  double* const partial = S.partial;
  void* const dlogits = S.dlogits;
  const int64_t ld_g = S.ld_g;
  __shared__ double red[7 * FW];
  __shared__ float smax[2][FW];
  __shared__ int sarg[FW];
  __shared__ int stoken;
  __shared__ double row_state[SAKI_VSHARD_STATE];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int Vl = S.V_local, n_chunks = Vl >> 3;
  const double rtau = 1.0 / S.tau;
  const float c32 = (float)(VF_LOG2E / S.tau);
  const double c64 = (double)c32;                  // the multiplier the elements really see
  const float2 cc = splat(c32), neg1 = splat(-1.f);
  // Every element enters as its distance below the row's maxima, s' = s - max s and t' = t - max t (exact in
  // float32 for bf16 logits): exponents are then sums of small terms, and the logit difference d' = t' - s'
  // is taken about the difference of the maxima, so float32 products keep their digits whatever offsets the two
  // models' logits carry.  Partials that are defined about zero are converted in float64, once per row.
  for (int64_t turn = blockIdx.x; turn < S.N; turn += gridDim.x) {
    // stage B from the last row to the first: it begins with what stage A, and stage C with what stage B, has left in L2
    const int64_t row = STAGE == 1 ? S.N - 1 - turn : turn;
    const __nv_bfloat16* s = (const __nv_bfloat16*)S.s + row * S.ld_s;
    const __nv_bfloat16* t = (const __nv_bfloat16*)S.t + row * S.ld_t;
    double* out = partial + row * SAKI_VSHARD_PARTIALS;
    // (one load by one warp: in the later waves and stage D a block has little more to do than this look at its row.  Past
    // L1: a launch that does not wait at its start has no claim on what another wrote)
    const double* const st = row_state;
    if (STAGE > 0) {
      __syncthreads();                         // the last row is done with row_state
      if (tid < SAKI_VSHARD_STATE) row_state[tid] = __ldcg(state + row * SAKI_VSHARD_STATE + tid);
      __syncthreads();
      if (st[VS_F64] != 0.0) continue;
    }
    const int mode = STAGE > 0 ? (int)st[VS_MODE] : 0;
    __nv_bfloat16* const g = STAGE >= 2 && dlogits ? (__nv_bfloat16*)dlogits + row * ld_g : nullptr;
    // the gradient slice on its own (a row without a TV pass, or a caller that asks for it at stage D)
    auto gradient_only = [&]() {
        const double sc = mode == VS_FLAGGED ? 0.0 : grad_scale * st[VS_COEF] * rtau;
        if (sc == 0.0) {
          for (int c = tid; c < n_chunks; c += FT) *reinterpret_cast<uint4*>(g + (size_t)c * 8) = make_uint4(0, 0, 0, 0);
        } else {
          const float msf = (float)st[VS_MS];
          const double kp2 = (st[VS_LSE_S] - st[VS_MS] * rtau) * VF_LOG2E;
          const float kpi = floorf((float)kp2 - 1e-3f);
          const float kgf = (float)(sc * exp2((double)kpi - kp2)), scf = (float)sc;     // gradient entry = e_p * kgf (- sc at the token)
          const float2 kpp = splat(-kpi), kgg = splat(kgf), nms = splat(-msf);
          const int tok = (int)st[VS_TOK] - S.v0;
          const int tok_c = (tok >= 0 && tok < Vl) ? (tok >> 3) : -1;
          for (int c = tid; c < n_chunks; c += FT) {
            const uint4 s4 = vf_ld(s + (size_t)c * 8);
            const uint32_t sw[4] = {s4.x, s4.y, s4.z, s4.w};
            float gv[8];
#pragma unroll
            for (int i = 0; i < 4; ++i) {
              const float2 ep = ex2f2(ffma2(fadd2(unpack_bf16x2(sw[i]), nms), cc, kpp));
              const float2 v = fmul2(ep, kgg);
              gv[2 * i] = v.x; gv[2 * i + 1] = v.y;
            }
            if (c == tok_c) {
#pragma unroll
              for (int i = 0; i < 8; ++i) if (i == (tok & 7)) gv[i] -= scf;
            }
            *reinterpret_cast<uint4*>(g + (size_t)c * 8) =
                make_uint4(pack_bf16x2(gv[0], gv[1]), pack_bf16x2(gv[2], gv[3]), pack_bf16x2(gv[4], gv[5]), pack_bf16x2(gv[6], gv[7]));
          }
        }
    };
    if (STAGE == 0) {
      // ---- stage A, first sweep: the slice's maxima, and the first chunk that holds the teacher's
      uint32_t run_s = VF_FILLER;
      float mt_run = -CUDART_INF_F;
      int arg_c = 0x7fffffff;
      for (int c = tid; c < n_chunks; c += FT) {
        const uint4 s4 = vf_ld(s + (size_t)c * 8), t4 = vf_ld(t + (size_t)c * 8);
        run_s = max_bf16x2(run_s, max_bf16x2(max_bf16x2(s4.x, s4.y), max_bf16x2(s4.z, s4.w)));
        const float2 cmt = unpack_bf16x2(max_bf16x2(max_bf16x2(t4.x, t4.y), max_bf16x2(t4.z, t4.w)));
        const float cm = fmaxf(cmt.x, cmt.y);
        if (cm > mt_run) { mt_run = cm; arg_c = c; }
      }
      const float2 rs2 = unpack_bf16x2(run_s);
      float ms = fmaxf(rs2.x, rs2.y), mt = mt_run;
      int ac = arg_c;
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) {
        ms = fmaxf(ms, __shfl_xor_sync(0xffffffffu, ms, o));
        const float omt = __shfl_xor_sync(0xffffffffu, mt, o);
        const int oac = __shfl_xor_sync(0xffffffffu, ac, o);
        if (omt > mt || (omt == mt && oac < ac)) { mt = omt; ac = oac; }
      }
      if (lane == 0) { smax[0][warp] = ms; smax[1][warp] = mt; sarg[warp] = ac; }
      __syncthreads();
      ms = smax[0][0]; mt = smax[1][0]; ac = sarg[0];
#pragma unroll
      for (int w = 1; w < FW; ++w) {
        ms = fmaxf(ms, smax[0][w]);
        if (smax[1][w] > mt || (smax[1][w] == mt && sarg[w] < ac)) { mt = smax[1][w]; ac = sarg[w]; }
      }
      __syncthreads();
      if (n_chunks == 0) { ms = -CUDART_INF_F; mt = -CUDART_INF_F; }
      // ---- second sweep: the sums under the slice's own maxima.  That is the partial's definition (no factor to apply), and
      // the float32 products need it: the exponent argument of the largest terms is then 0 or near it, exact, where one of
      // size a carries an error of a 2^-24.  (One sweep under the maxima of the slice's first 1024 logits takes 593 us instead
      // of 654 for 1024 rows of 151936 in eight slices, and moves log-sum-exps by 1e-7 and with them draws.)
      float2 Ss = splat(0.f), St = splat(0.f), Td = splat(0.f), M1 = splat(0.f), M2 = splat(0.f), M3 = splat(0.f), M4 = splat(0.f);
      const float msc = fminf(fmaxf(ms, -1e30f), 1e30f), mtc = fminf(fmaxf(mt, -1e30f), 1e30f);
      const float2 nms = splat(-msc), nmt = splat(-mtc);
#pragma unroll 2
      for (int c = tid; c < n_chunks; c += FT) {
        const uint4 s4 = vf_ld(s + (size_t)c * 8), t4 = vf_ld(t + (size_t)c * 8);
        const uint32_t sw[4] = {s4.x, s4.y, s4.z, s4.w}, tw[4] = {t4.x, t4.y, t4.z, t4.w};
        float2 cs = splat(0.f), ct = splat(0.f);     // per chunk first: a running sum takes one addition per chunk
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          const float2 sf = fadd2(unpack_bf16x2(sw[i]), nms), tf = fadd2(unpack_bf16x2(tw[i]), nmt);
          const float2 d = ffma2(sf, neg1, tf);
          const float2 es = ex2f2(fmul2(sf, cc));
          const float2 et = ex2f2(fmul2(tf, cc));
          cs = i == 0 ? es : fadd2(cs, es);
          ct = i == 0 ? et : fadd2(ct, et);
          Td = ffma2(et, d, Td);
          const float2 d2 = fmul2(d, d);
          M1 = ffma2(es, d, M1);
          const float2 u = fmul2(es, d2);
          M2 = fadd2(M2, u);
          M3 = ffma2(u, d, M3);
          M4 = ffma2(u, d2, M4);
        }
        Ss = fadd2(Ss, cs);
        St = fadd2(St, ct);
      }
      double a[7] = {vf_tot(Ss), vf_tot(St), vf_tot(Td), vf_tot(M1), vf_tot(M2), vf_tot(M3), vf_tot(M4)};
      vf_block_sum<7>(a, red);
      if (tid == 0) {
        int am = 0x7fffffff;                       // lowest index of the teacher's maximum inside its first chunk
        if (n_chunks > 0 && ac != 0x7fffffff) {
          for (int i = 7; i >= 0; --i) if (__bfloat162float(t[(size_t)ac * 8 + i]) == mt) am = ac * 8 + i;
        }
        bool finite = true;
#pragma unroll
        for (int k = 0; k < 7; ++k) finite = finite && isfinite(a[k]);
        finite = finite && (n_chunks == 0 || (ms > -1e30f && mt > -1e30f && ms < 1e30f && mt < 1e30f));
        const int x = S.proposal[row] - S.v0;
        const bool own = x >= 0 && x < Vl;
        for (int k = 0; k < SAKI_VSHARD_PARTIALS; ++k) out[k] = 0.0;
        out[0] = (double)ms; out[1] = (double)mt; out[2] = am == 0x7fffffff ? 2147483647.0 : (double)(S.v0 + am);
        out[3] = finite ? 1.0 : 0.0;
        if (finite && n_chunks > 0) {
          const double r2 = rtau * rtau, D = (double)mtc - (double)msc;
          a[2] += D * a[1];
          vf_uncentre(D, a[0], a[3], a[4], a[5], a[6]);
          out[4] = a[0]; out[5] = a[1]; out[6] = a[2] * rtau;
          out[7] = a[3] * rtau; out[8] = a[4] * r2; out[12] = a[5] * r2 * rtau; out[13] = a[6] * r2 * r2;
        }
        out[9] = own ? (double)__bfloat162float(s[x]) : 0.0; out[10] = own ? (double)__bfloat162float(t[x]) : 0.0;
        out[11] = own ? 1.0 : 0.0;
      }
    } else if (STAGE == 1) {
      // ---- stage B: one evaluation at the row's current beta, under the row's shift (its maxima: no factor)
      if (mode != VS_SOLVING) continue;            // (block-uniform; its partial is not read)
      const double beta = st[VS_BETA];
      float cb = (float)(c64 * beta);
      const float ccb = c32 - cb;                  // the exponent is formed as (c - cb) s' + cb t'
      cb = c32 - ccb;                              // (so that the pair adds up to c exactly)
      const float msf = (float)st[VS_MS], mtf = (float)st[VS_MT];
      const float2 cbb = splat(cb), ccbb = splat(ccb), nms = splat(-msf), nmt = splat(-mtf);
      float2 S0 = splat(0.f), S1 = splat(0.f), S2 = splat(0.f), S3 = splat(0.f), S4 = splat(0.f);
      // (the loads of three chunks per thread before the first is worked on, here, and of two in stage C: the waves that
      // find few rows unsettled are the latency of one slice; 1024 rows of 151936 in eight slices 655 -> 630 us when stage A was one sweep)
#pragma unroll 1
      for (int b = tid; b < n_chunks; b += 3 * FT) {
        uint4 sv[3], tv[3];
#pragma unroll
        for (int u = 0; u < 3; ++u)
          if (b + u * FT < n_chunks) { sv[u] = vf_ld(s + (size_t)(b + u * FT) * 8); tv[u] = vf_ld(t + (size_t)(b + u * FT) * 8); }
#pragma unroll
        for (int u = 0; u < 3; ++u) {
          const int c = b + u * FT;
          if (c >= n_chunks) break;
          const uint4 s4 = sv[u], t4 = tv[u];
          const uint32_t sw[4] = {s4.x, s4.y, s4.z, s4.w}, tw[4] = {t4.x, t4.y, t4.z, t4.w};
          float2 c0 = splat(0.f), c1 = splat(0.f);      // the chunk's share of S0 and S1
#pragma unroll
          for (int i = 0; i < 4; ++i) {
            const float2 sf = fadd2(unpack_bf16x2(sw[i]), nms), tf = fadd2(unpack_bf16x2(tw[i]), nmt);
            const float2 d = ffma2(sf, neg1, tf);
            const float2 e = ex2f2(ffma2(tf, cbb, fmul2(sf, ccbb)));
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
        }
      }
      double a[5] = {vf_tot(S0), vf_tot(S1), vf_tot(S2), vf_tot(S3), vf_tot(S4)};
      vf_block_sum<5>(a, red);
      if (tid == 0) {
        const double r2 = rtau * rtau;
        vf_uncentre((double)mtf - (double)msf, a[0], a[1], a[2], a[3], a[4]);
        for (int k = 0; k < SAKI_VSHARD_PARTIALS; ++k) out[k] = 0.0;
        out[0] = a[0]; out[1] = a[1] * rtau; out[2] = a[2] * r2; out[3] = a[3] * r2 * rtau; out[4] = a[4] * r2 * r2;
      }
    } else if (STAGE == 2) {
      // ---- stage C: the slice's share of TV and KL(q||p); the student's logit at the teacher's argmax; the gradient
      // slice (the row's coefficient has been known since its lambda settled)
      const bool live = mode == VS_SETTLED;
      const double lam = st[VS_LAM];
      double a[3] = {0.0, 0.0, 0.0};
      double fq = 0.0, D = 0.0;
      if (live && lam > 0.0) {
        const double lse_s = st[VS_LSE_S], lse_t = st[VS_LSE_T], logZ = st[VS_LOGZ];
        float cl = (float)(c64 * lam);
        const float ccl = c32 - cl;
        cl = c32 - ccl;
        const float msf = (float)st[VS_MS], mtf = (float)st[VS_MT];
        D = (double)mtf - (double)msf;
        // p = 2^(c s' - kp2), q = 2^((c - cl) s' + cl t' - kq2); whole-number shifts kpi <= kp2, kqi <= kq2 (both
        // arguments stay below 1), the factors between them applied in float64
        // (with the log-sum-exps relative to the maxima: what the sums of 2^(c s'), 2^(c t') came to)
        const double ls = lse_s - st[VS_MS] * rtau, lt = lse_t - st[VS_MT] * rtau;
        const double kp2 = ls * VF_LOG2E, kq2 = ((1.0 - lam) * ls + lam * lt + logZ) * VF_LOG2E;
        const float kpi = floorf((float)kp2 - 1e-3f), kqi = floorf((float)kq2 - 1e-3f);
        const double fp = exp2((double)kpi - kp2);
        fq = exp2((double)kqi - kq2);
        const float2 cll = splat(cl), ccll = splat(ccl), kpp = splat(-kpi), kqq = splat(-kqi), nrho = splat(-(float)(fp / fq));
        const float2 nms = splat(-msf), nmt = splat(-mtf);
        // the gradient entry is e_p * kgf (- sc at the token)
        const double sc = grad_scale * st[VS_COEF] * rtau;
        const float kgf = (float)(sc * fp), scf = (float)sc;
        const float2 kgg = splat(kgf);
        const int tok = (int)st[VS_TOK] - S.v0, tok_c = (tok >= 0 && tok < Vl) ? (tok >> 3) : -1;
        float2 R = splat(0.f), Sq = splat(0.f), Sqd = splat(0.f);
#pragma unroll 1
        for (int b = tid; b < n_chunks; b += 2 * FT) {
          uint4 sv[2], tv[2];
#pragma unroll
          for (int u = 0; u < 2; ++u)
            if (b + u * FT < n_chunks) { sv[u] = vf_ld(s + (size_t)(b + u * FT) * 8); tv[u] = vf_ld(t + (size_t)(b + u * FT) * 8); }
#pragma unroll
          for (int u = 0; u < 2; ++u) {
            const int c = b + u * FT;
            if (c >= n_chunks) break;
            const uint4 s4 = sv[u], t4 = tv[u];
            const uint32_t sw[4] = {s4.x, s4.y, s4.z, s4.w}, tw[4] = {t4.x, t4.y, t4.z, t4.w};
            float2 gv[4];
#pragma unroll
            for (int i = 0; i < 4; ++i) {
              const float2 sf = fadd2(unpack_bf16x2(sw[i]), nms), tf = fadd2(unpack_bf16x2(tw[i]), nmt);
              const float2 d = ffma2(sf, neg1, tf);
              const float2 ep = ex2f2(ffma2(sf, cc, kpp));
              gv[i] = fmul2(ep, kgg);
              const float2 eq = ex2f2(ffma2(tf, cll, ffma2(sf, ccll, kqq)));
              float2 r = ffma2(ep, nrho, eq);          // (q_i - p_i) / fq
              r.x = fmaxf(r.x, 0.f); r.y = fmaxf(r.y, 0.f);
              R = fadd2(R, r);
              Sq = fadd2(Sq, eq);
              Sqd = ffma2(eq, d, Sqd);
            }
            if (g) {
              if (c == tok_c) {
#pragma unroll
                for (int i = 0; i < 8; ++i) if (i == (tok & 7)) { if (i & 1) gv[i >> 1].y -= scf; else gv[i >> 1].x -= scf; }
              }
              __stcs(reinterpret_cast<uint4*>(g + (size_t)c * 8), make_uint4(pack_bf16x2(gv[0].x, gv[0].y), pack_bf16x2(gv[1].x, gv[1].y),
                                                                             pack_bf16x2(gv[2].x, gv[2].y), pack_bf16x2(gv[3].x, gv[3].y)));
            }
          }
        }
        a[0] = vf_tot(R); a[1] = vf_tot(Sq); a[2] = vf_tot(Sqd);
      } else if (g) gradient_only();
      vf_block_sum<3>(a, red);
      if (tid == 0) {
        for (int k = 0; k < SAKI_VSHARD_PARTIALS; ++k) out[k] = 0.0;
        if (live && lam > 0.0) {
          const double cc0 = st[VS_LSE_T] - st[VS_LSE_S];      // log q - log p = lam ((t - s)/tau - cc0) - log Z
          out[0] = fq * a[0];
          out[1] = fq * (lam * rtau * (a[2] + D * a[1]) - (lam * cc0 + st[VS_LOGZ]) * a[1]);
        }
        const int vs = (int)st[VS_VSTAR] - S.v0;
        out[2] = (live && vs >= 0 && vs < Vl) ? (double)__bfloat162float(s[vs]) : 0.0;
      }
    } else {
      // ---- stage D: on the owning rank the residual draw; the gradient slice, if stage C has not written it
      if (g) gradient_only();
      const bool mine = mode == VS_SETTLED && st[VS_CORR] != 0.0 && (int)st[VS_OWNER] == S.rank;      // (block-uniform)
      int y = -1;
      if (mine) {
        if (tid == 0) stoken = -1;
        __syncthreads();
        vf_draw(s, t, n_chunks, c32, c64, S.tau, st, red, &stoken);
        __syncthreads();
        y = stoken;
        __syncthreads();
        if (y >= Vl) y = -1;
      }
      if (tid < SAKI_VSHARD_PARTIALS)
        out[tid] = tid == 0 ? (y >= 0 ? (double)(S.v0 + y) : -1.0) : tid == 1 && y >= 0 ? (double)__bfloat162float(s[y])
                 : tid == 2 && y >= 0 ? (double)__bfloat162float(t[y]) : 0.0;
    }
  }
  if (beside) wait_for_predecessor();
}

// Stage D of a group of slices, a block per row: the draw on the slice that owns the target, if any, and the records of
// all of them (a block per row and slice is 8192 blocks for 1024 rows in eight slices, most of which only write a record).
__global__ void __launch_bounds__(FT, 6) vs_draw_kernel(const __grid_constant__ VsGroup Gr, const double* state, const int members, const bool beside) {
  if (!beside) wait_for_predecessor();         // (as in vs_fast_kernel)
  launch_dependents();
  __shared__ double red[FW], row_state[SAKI_VSHARD_STATE];
  __shared__ int stoken;
  const int tid = threadIdx.x;
  const float c32 = (float)(VF_LOG2E / Gr.s[0].tau);
  const double c64 = (double)c32;
  for (int64_t row = blockIdx.x; row < Gr.s[0].N; row += gridDim.x) {
    const double* const st = row_state;
    __syncthreads();
    if (tid < SAKI_VSHARD_STATE) row_state[tid] = __ldcg(state + row * SAKI_VSHARD_STATE + tid);
    __syncthreads();
    if (st[VS_F64] != 0.0) continue;
    int own = -1, y = -1;
    if ((int)st[VS_MODE] == VS_SETTLED && st[VS_CORR] != 0.0)
      for (int k = 0; k < members; ++k) if (Gr.s[k].rank == (int)st[VS_OWNER]) own = k;
    float sy = 0.f, ty = 0.f;
    if (own >= 0) {
      const VsSlice& O = Gr.s[own];
      const __nv_bfloat16* const s = (const __nv_bfloat16*)O.s + row * O.ld_s;
      const __nv_bfloat16* const t = (const __nv_bfloat16*)O.t + row * O.ld_t;
      if (tid == 0) stoken = -1;
      __syncthreads();
      vf_draw(s, t, O.V_local >> 3, c32, c64, O.tau, st, red, &stoken);
      __syncthreads();
      y = stoken;
      if (y >= O.V_local) y = -1;
      if (y >= 0) { sy = __bfloat162float(s[y]); ty = __bfloat162float(t[y]); }
    }
    for (int k = tid; k < members * SAKI_VSHARD_PARTIALS; k += FT) {
      const int r = k / SAKI_VSHARD_PARTIALS, f = k % SAKI_VSHARD_PARTIALS;
      const bool mine = r == own && y >= 0;
      Gr.s[r].partial[row * SAKI_VSHARD_PARTIALS + f] = f == 0 ? (mine ? (double)(Gr.s[r].v0 + y) : -1.0) : f == 1 && mine ? (double)sy : f == 2 && mine ? (double)ty : 0.0;
    }
  }
  if (beside) wait_for_predecessor();
}

// A row's combine is a chain of float64 scalars on one thread.  What surrounds the chain is spread over the row's VC_LANES
// threads: partials and state come into shared memory side by side (a thread that fetched them one after the other, rank
// by rank, waited for memory at each), the exponentials of stage A are formed one rank per thread, the state leaves as a
// block.  The sums themselves stay in rank order.
constexpr int VC_ROWS = 8, VC_LANES = 8, VC_THREADS = VC_ROWS * VC_LANES, VC_WORLD = 16;
__global__ void __launch_bounds__(VC_THREADS) vs_combine_kernel(const VsConsts C, const int stage, const double* part, double* state,
                                  const saki_out o, unsigned int* n_solving, unsigned int* n_marked) {
  constexpr int P = SAKI_VSHARD_PARTIALS, S = SAKI_VSHARD_STATE;
  __shared__ double sp[VC_ROWS][VC_WORLD][P + 1], sst[VC_ROWS][S + 1], scaled[VC_ROWS][VC_WORLD][VA_COUNT];
  launch_dependents();
  wait_for_predecessor();
  const int tid = threadIdx.x, lr = tid / VC_LANES, lane = tid % VC_LANES;
  const int64_t row0 = (int64_t)blockIdx.x * VC_ROWS, i = row0 + lr;
  const int rows = (int)min((int64_t)VC_ROWS, C.N - row0);
  const bool held = C.world <= VC_WORLD;                     // (more ranks: read where they are)
  if (held) {
#pragma unroll 8
    for (int k = tid; k < C.world * rows * P; k += VC_THREADS) {
      const int r = k / (rows * P), q = k - r * rows * P;
      sp[q / P][r][q % P] = part[((int64_t)r * C.N + row0) * P + q];
    }
  }
  if (stage > 0)
    for (int k = tid; k < rows * S; k += VC_THREADS) sst[k / S][k % S] = state[row0 * S + k];
  __syncthreads();
  const double* const mine = held ? &sp[lr][0][0] : part + i * P;
  const int64_t rs = held ? P + 1 : C.N * P;
  VsMaxima m = {};
  if (stage == 0) {
    if (lr < rows) {
      m = vs_maxima(C, mine, rs);
      if (held) for (int r = lane; r < C.world; r += VC_LANES) vs_rescale(C, mine + r * rs, m, scaled[lr][r]);
    }
    __syncthreads();
  }
  if (lr < rows && lane == 0) {
    double* const st = sst[lr];
    if (stage == 0) {
      vs_combine_a(C, i, mine, rs, st, m, held ? &scaled[lr][0][0] : nullptr, VA_COUNT);
      if ((int)st[VS_MODE] == VS_SOLVING && n_solving) atomicAdd(n_solving, 1u);
    } else if (stage == 1) {
      const double was = st[VS_F64];
      if (vs_combine_b(C, i, mine, rs, st) && n_solving) atomicAdd(n_solving, 1u);
      if (n_marked && st[VS_F64] != was) atomicAdd(n_marked, 1u);
    }
    else if (stage == 2) vs_combine_c(C, i, mine, rs, st);
    else vs_combine_d(C, i, mine, rs, st, o);
  }
  __syncthreads();
  for (int k = tid; k < rows * S; k += VC_THREADS) state[row0 * S + k] = sst[k / S][k % S];
}

// the call may use the float32 slice kernels: a property of the call's arguments alone, so that every rank's
// combine takes the same decisions (a rank whose own slice is not aligned for them simply computes in float64)
static bool vshard_fast_call(const saki_vshard_in& in, bool allow_fast) {
  return allow_fast && in.dtype == SAKI_BF16 && in.eps >= 0.02f;   // below, KL needs the float64 sums (or a quadrature)
}

cudaError_t launch_vshard_partial(const saki_vshard_in* in, int n, int stage, const double* state, double* const* partial,
                                  void* const* dlogits, const int64_t* ld_g, float grad_scale, bool allow_fast, int flags,
                                  int* n_launches, cudaStream_t st) {
  int dev = 0, sms = 148;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  auto al16 = [](const void* q) { return ((uintptr_t)q & 15) == 0; };
  for (int i0 = 0; i0 < n; i0 += VS_GROUP) {
    const int m = n - i0 < VS_GROUP ? n - i0 : VS_GROUP;
    VsGroup Gr;
    int n_fast = 0;
    for (int k = 0; k < m; ++k) {
      const saki_vshard_in& a = in[i0 + k];
      VsSlice& S = Gr.s[k];
      S.s = a.student_logits; S.t = a.teacher_logits; S.ld_s = a.ld_s; S.ld_t = a.ld_t; S.N = a.N;
      S.V_local = a.V_local; S.v0 = a.v0; S.rank = a.rank; S.tau = (double)a.temperature; S.proposal = a.proposal;
      S.partial = partial[i0 + k];
      S.dlogits = stage >= 2 && dlogits ? dlogits[i0 + k] : nullptr;
      S.ld_g = S.dlogits ? ld_g[i0 + k] : 0;
      S.fast = vshard_fast_call(a, allow_fast) && a.V_local % 8 == 0 && a.ld_s % 8 == 0 && a.ld_t % 8 == 0 && al16(S.s) &&
               al16(S.t) && (!S.dlogits || (al16(S.dlogits) && S.ld_g % 8 == 0));
      n_fast += S.fast;
    }
    const int64_t N = in[i0].N;
    const double gs = (double)grad_scale;
    const bool marks = n_fast < m || !(stage == 0 || (flags & SAKI_VSHARD_NONE_MARKED));    // (no row is marked before the first combine)
    if (marks) {
      const int64_t blocks = (3LL * sms + m - 1) / m;
      const dim3 grid((unsigned)(N < blocks ? N : blocks), (unsigned)m, 1);
      auto go = [&](auto kernel) { return launch_pdl(kernel, grid, VT, 0, st, true, Gr, stage, state, gs); };
      cudaError_t e = in[i0].dtype == SAKI_BF16 ? go(vs_partial_kernel<__nv_bfloat16>) : go(vs_partial_kernel<float>);
      *n_launches += 1;
      if (e != cudaSuccess) return e;
    }
    if (n_fast > 0) {
      // (A block per row and slice, in the later waves and stage 3 too, where most rows have nothing left to do: with one
      // per two or four rows those that have wait for one another, 715 -> 738, 753 us for 1024 rows in eight slices.)
      const bool draw = stage == 3 && n_fast == m && !dlogits;
      const dim3 grid((unsigned)(N < 8LL * sms ? N : 8LL * sms), draw ? 1u : (unsigned)m, 1);
      const bool beside = marks && stage > 0;
      auto go = [&](auto kernel) { return launch_pdl(kernel, grid, FT, 0, st, true, Gr, state, gs, beside); };
      cudaError_t e = draw ? launch_pdl(vs_draw_kernel, grid, FT, 0, st, true, Gr, state, m, beside)
                    : stage == 0 ? go(vs_fast_kernel<0>) : stage == 1 ? go(vs_fast_kernel<1>) : stage == 2 ? go(vs_fast_kernel<2>) : go(vs_fast_kernel<3>);
      *n_launches += 1;
      if (e != cudaSuccess) return e;
    }
  }
  return cudaSuccess;
}

static VsConsts consts_of(const saki_vshard_in& in, bool allow_fast) {
  VsConsts c;
  c.N = in.N; c.V = in.V; c.world = in.world; c.eps = (double)in.eps; c.tau = (double)in.temperature;
  c.seed = in.seed; c.row_offset = in.row_offset; c.proposal = in.proposal; c.mask = in.mask;
  c.fast = vshard_fast_call(in, allow_fast) ? 1 : 0;
  return c;
}

cudaError_t launch_vshard_combine(const saki_vshard_in& in, int stage, const double* gathered, double* state, const saki_out& out,
                                  unsigned int* n_solving, unsigned int* n_marked, bool allow_fast, cudaStream_t st) {
  const VsConsts c = consts_of(in, allow_fast);
  return launch_pdl(vs_combine_kernel, dim3((unsigned)((in.N + VC_ROWS - 1) / VC_ROWS)), VC_THREADS, 0, st, true, c, stage, gathered,
                    state, out, n_solving, n_marked);
}

// the same combine on HOST buffers (a caller without a GPU at hand, and the multi-process tests of the exchange)
int vshard_combine_host(const saki_vshard_in& in, int stage, const double* gathered, double* state, const saki_out& out,
                        bool allow_fast) {
  const VsConsts c = consts_of(in, allow_fast);
  int solving = 0;
  for (int64_t i = 0; i < in.N; ++i) {
    double* st = state + i * SAKI_VSHARD_STATE;
    const double* const mine = gathered + i * SAKI_VSHARD_PARTIALS;
    const int64_t rs = c.N * SAKI_VSHARD_PARTIALS;
    if (stage == 0) {
      vs_combine_a(c, i, mine, rs, st, vs_maxima(c, mine, rs), nullptr, 0);
      solving += (int)st[VS_MODE] == VS_SOLVING;
    }
    else if (stage == 1) solving += vs_combine_b(c, i, mine, rs, st);
    else if (stage == 2) vs_combine_c(c, i, mine, rs, st);
    else vs_combine_d(c, i, mine, rs, st, out);
  }
  return solving;
}

}  // namespace saki
