// Row-per-SM kernel, the variant with one CTA of 512 threads per SM, and the choice between the five
// variants (the implementation is saki_rowsm_impl.cuh).
#include "saki_rowsm_impl.cuh"
#include <cmath>

namespace saki {

// Where the kernel is pinned, rows up to this length go to the variant with two CTAs of 256 threads per SM: their passes are short
// against the serial phases between them (block reductions, float64 scalars), and a second CTA on the
// SM runs its passes meanwhile.  Longer rows stay with one CTA per SM: with two rows in flight per SM
// the streamed parts of all rows no longer stay in L2 between the passes.  Measured (fwd+bwd, M rows/s,
// one / two CTAs per SM): V = 8192 15.9 / 25.3, 32000 9.9 / 12.7, 65536 6.5 / 7.5, 81920 5.6 / 6.3,
// 100000 4.85 / 5.06, 131072 3.95 / 3.76.
constexpr int HALF_MAX_V = 98304;
// Shorter rows still go to the variant with four CTAs of 128 threads per SM: more of the SM's rows are in a
// pass at any time.  Measured (M rows/s, two / four CTAs per SM): V = 4096 29.7 / 44.4, 8192 26.0 / 35.0,
// 16384 19.6 / 21.7, 32000 13.1 / 14.3, 49152 9.8 / 10.0, 65536 7.8 / 7.5.
constexpr int QUARTER_MAX_V = 49152;
// Rows of more than this many elements do not go to two SMs in blocks of 512 threads (why: see the choice below).
constexpr int WIDE_MAX_V = 98304;

bool rowsm_can_serve(const RowParams& p, int dtype) {
  if (dtype != SAKI_BF16) return false;
  if (p.V < 2048 || p.V % 8 != 0 || p.V > full_sm::max_v()) return false;
  if (p.n_rows > 0x7fffffffLL) return false;     // row numbers are kept in 32 bits (redo list, divisions)
  auto al16 = [](const void* q) { return ((uintptr_t)q & 15) == 0; };
  if (!al16(p.s) || !al16(p.t)) return false;
  if (p.s_seq % 8 || p.s_pos % 8 || p.t_seq % 8 || p.t_pos % 8) return false;
  if (p.dlogits && (!al16(p.dlogits) || p.ld_g % 8)) return false;
  return true;
}

struct Variant {
  cudaError_t (*launch)(const RowParams&, cudaStream_t, int*, bool*);
  int blocks_per_row, blocks_per_sm;
};
static const Variant FULL = {full_sm::launch, 1, 1}, HALF = {half_sm::launch, 1, 2}, QUARTER = {quarter_sm::launch, 1, 4},
                     PAIR = {pair_sm::launch, 2, 2}, WIDE = {wide_sm::launch, 2, 1};

// The variant that routes this number of rows soonest.  All figures: forward + gradient, rows from memory, us, calls one after the
// other in a graph.
//   - A row or less for two SMs: two CTAs of 512 threads on two SMs to a row (one SM per row / two: 74 rows of 98304 42.3 / 31.4,
//     of 65536 34.2 / 25.8, of 32000 23.7 / 20.1); a row or less per SM: the pair of CTAs of 256 threads (148 rows of 151936
//     68.6 / 59.8, of 65536 38.2 / 35.4, of 24000 22.6 / 20.8).  Below V = 20000 the exchange costs about what it saves: two CTAs
//     per SM (148 rows of 16384 19.6, the pair 19.0; 37 rows 15.6, 15.7; 148 rows of 12288 18.2, 18.5).  49 shapes of up to 148 rows: 0.3 %
//     above the best variant on average, 5 % at worst, beside what follows.
//   - Beyond V = 98304 the pair takes those few rows too, which costs a quarter to a third (74 rows of 151936 52.3, 40.1 with 512
//     threads; 37 rows 49.4, 36.4; one SM per row 56.9 and 52.8): its sixteen warps add up a row's sums in the order of the pinned
//     variant, and a test compares 40 such rows with it to the bit.
//   - Rows beyond V = 131072, more than 40 per SM: one CTA per SM.  The pair's lead, the last turn, is gone there, and each row waits for
//     the slower of its SMs (loops of half a second over three batches, one SM / pair: 16384 rows of 151936 4489 / 4541, 8192 2290 /
//     2297, 8192 of 163840 2463 / 2471, 16384 of 139264 4128 / 4145).  Up to V = 131072 (16384 rows of 131072 3919 / 3925, of 118784 3614 /
//     3592, of 98312 3239 / 3161) and for fewer rows (4096 of 151936 1182 / 1178, 2000 597 / 584) it is even or the other way round.
//   - More rows than SMs otherwise: the variant that takes the least by a cost model, start + (serial + element V / 1000) turns, where a
//     turn is waited for to its end only in part (CTAs take over rows that have not started) and costs more where the rows in
//     flight are more than L2 holds.  Fitted to 754 shapes (V = 2048 to 163840, 149 to 16384 rows), each with rows from memory, with
//     rows in L2, and forward alone: 0.2, 0.2 and 0.4 % above the best variant on average, 3 % or more for 15, 18 and 40 of the
//     shapes, 7, 9 and 11 % at worst.  (Where two fit, e.g. 16384 rows of 118784, the gradient's stores decide: pair / two per SM
//     3600 / 3693, forward alone 3500 / 3204.  The choice does not look at that, so that both calls give the same bits.)
//     The pair takes 149 to some 175 rows of 49152 and to some 235 of 98304, from V = 65536 on a second turn that has just begun, and from
//     V = 115000 on all calls (320 rows of 151936 149 on one SM each, 121 on the pair; 1200 390 / 365); two and four CTAs per SM the others
//     (2000 rows of 65536 259, the pair 304; of 16384 86 with four, 97 with two).
// Not where saki_set_kernel pins the kernel: then the variant goes by V alone, and pieces of a batch agree with the whole to the bit.
static const Variant& pick_variant(const RowParams& p) {
  const int64_t n = p.call_rows;
  if (n <= 0) return p.V <= QUARTER_MAX_V ? QUARTER : p.V <= HALF_MAX_V ? HALF : FULL;
  int dev = 0, sms = 148;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  if (n <= sms) {
    if (p.V < 20000) return HALF;
    return 2 * n <= sms && p.V <= WIDE_MAX_V ? WIDE : PAIR;
  }
  if (p.V > 131072 && n > 40 * (int64_t)sms) return FULL;
  // max_v: the longest row; per_sm: rows in flight per SM; whole: the part of a turn that is waited for to its end; late: how far
  // into its turn an average CTA is when no row is left; beyond: for each 126 MB in flight beyond L2
  struct Model { const Variant* v; int max_v; double per_sm, start, serial, element, whole, late, beyond; };
  const Model models[] = {{&HALF, half_sm::max_v(), 2, 7.30, 4.71, 0.4938, 0.214, 0.308, 1.812},
                          {&QUARTER, QUARTER_MAX_V, 4, 7.52, 2.83, 1.0473, 0.153, 0.249, 0.317},
                          {&PAIR, pair_sm::max_v(), 1, 8.72, 11.92, 0.1921, 0.0, 0.109, 0.125}};
  const Variant* best = &PAIR;
  double least = 1e300;
  for (const Model& m : models) {
    if (p.V > m.max_v) continue;
    const double slots = m.per_sm * sms, turns = (double)n / slots, in_flight = std::min((double)n, slots) * 4.0 * p.V;
    const double t = turns > 1.0 ? m.whole * std::ceil(turns) + (1.0 - m.whole) * (turns + m.late) : 1.0;
    const double c = m.start + (m.serial + m.element * 1e-3 * p.V) * t * (1.0 + m.beyond * std::max(0.0, in_flight / 126e6 - 1.0));
    if (c < least) { least = c; best = m.v; }
  }
  return *best;
}

static thread_local int g_layout[2];      // of the thread's last routing call: blocks per row, blocks per SM
void rowsm_layout(int* out) { std::copy(g_layout, g_layout + 2, out); }
void rowsm_layout_none() { g_layout[0] = g_layout[1] = 0; }

cudaError_t launch_rowsm(const RowParams& p, cudaStream_t st, int* n_launches, bool* served) {
  const Variant& v = pick_variant(p);
  const cudaError_t e = v.launch(p, st, n_launches, served);
  if (e == cudaSuccess && *served) { g_layout[0] = v.blocks_per_row; g_layout[1] = v.blocks_per_sm; }
  return e;
}

}  // namespace saki
