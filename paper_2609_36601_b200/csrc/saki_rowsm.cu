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

// The variant that routes this number of rows soonest, by 231 shapes (V = 8192 to 151936, 20 to 5000 rows, every variant timed): the
// choice is 0.6 % above the best of them on average, 3 % or more for one shape in fifteen, 13 % at worst.
//   - A row or less for two SMs: two CTAs of 512 threads on two SMs to a row (us, one SM per row / two: 74 rows of 98304 37.9 /
//     26.1, of 65536 32.4 / 23.7, of 32768 22.5 / 19.0); a row or less per SM: the pair of CTAs of 256 threads (148 rows of
//     151936 60.8 / 58.3, of 65536 33.8 / 30.1, of 24000 20.9 / 19.1).  Rows of V > 98304 take the pair there too (37 rows of 151936
//     50.2 / 36.6, 32.8 with 512 threads; 74 rows 50.7 / 49.3, 33.8): its sixteen warps give the bits of the pinned variant, which
//     callers and tests of such pieces compare with.  Below V = 20000 the exchange costs what it saves: two
//     CTAs per SM (148 rows of 16384 17.9, the pair 17.5; 20 rows 15.3, 15.4).
//   - More: the variant that takes the least by a cost model, start + (serial + element V / 1000) turns, where a turn is waited
//     for to its end only in part (CTAs take over rows that have not started) and costs more where the rows in flight are more than
//     L2 holds.  The pair is what 149 to some 1000 long rows take (us, one CTA per SM / pair: 300 rows of 151936 147 / 116, 1200 395 / 372), two
//     and four CTAs per SM shorter ones (2000 rows of 65536 314 / 267 with two; of 16384 157 / 88 with four).
//   - Rows beyond V = 131072 by the thousands: one CTA per SM (16384 rows of 151936 4517, the pair 4550; 4096 rows 1167, 1162).
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
  // max_v: the longest row; per_sm: rows in flight per SM; whole: the part of a turn that is waited for to its end; late: how far into its turn an
  // average CTA is when no row is left; beyond: for each 126 MB in flight beyond L2
  struct Model { const Variant* v; int max_v; double per_sm, start, serial, element, whole, late, beyond; };
  const Model models[] = {{&FULL, full_sm::max_v(), 1, 4.64, 6.52, 0.2485, 0.548, 1.0, 0.05}, {&HALF, half_sm::max_v(), 2, 7.40, 3.64, 0.5366, 0.156, 0.253, 0.221},
                          {&QUARTER, QUARTER_MAX_V, 4, 5.68, 4.31, 1.0593, 0.091, 0.246, 0.131}, {&PAIR, pair_sm::max_v(), 1, 4.70, 6.03, 0.2368, 0.121, 0.535, 0.05}};
  if (p.V > 131072 && n > 40 * (int64_t)sms) return FULL;
  const Variant* best = &FULL;
  double least = 1e300;
  for (const Model& m : models) {
    if (p.V > m.max_v) continue;
    const double slots = m.per_sm * sms, turns = (double)n / slots, in_flight = std::min((double)n, slots) * 4.0 * p.V;
    const double t = turns > 1.0 ? m.whole * std::ceil(turns) + (1.0 - m.whole) * (turns + m.late) : 1.0;
    const double c = m.start + (m.serial + m.element * 1e-3 * p.V) * std::max(1.0, t) * (1.0 + m.beyond * std::max(0.0, in_flight / 126e6 - 1.0));
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
