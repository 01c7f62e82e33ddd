// Row-per-SM kernel, the variant with one CTA of 512 threads per SM, and the choice between the three
// variants (the implementation is saki_rowsm_impl.cuh).
#include "saki_rowsm_impl.cuh"

namespace saki {

// Rows up to this length go to the variant with two CTAs of 256 threads per SM: their passes are short
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

// The variant that routes this number of rows soonest.  A variant with k CTAs per SM takes ceil(rows / (k SMs))
// turns of a + b V / 1000 microseconds each (fitted to V = 2048 to 98304 and 8 to 1776 rows, within 10 %):
//   k = 1: 6.2, 0.302     k = 2: 5.0, 0.535     k = 4: 6.0, 1.06
// so that, e.g., 888 rows of 32000 take three turns of k = 2 (73 us) and not two of k = 4 (83 us), 296 rows of 49152 one
// turn of k = 2 (38 us against 48 with k = 1 and 51 with k = 4); a call with a row or less per SM takes k = 1, or k = 2
// where its inlined scalar steps outweigh the longer passes (below V = 16384: 14.1 against 16.2 us at 8192).  The limits on V above
// hold here too, except that rows in flight that fit in L2 anyway (two per SM) may be longer.  Not where saki_set_kernel
// pins the kernel: then the variant goes by V alone, and pieces of a batch agree with the whole to the bit.
cudaError_t launch_rowsm(const RowParams& p, cudaStream_t st, int* n_launches, bool* served) {
  if (p.call_rows > 0) {
    int dev = 0, sms = 148;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    const int64_t n = p.call_rows;
    const double kv = p.V * 1e-3;
    auto cost = [&](int k, double a, double b) { return (double)((n + (int64_t)k * sms - 1) / ((int64_t)k * sms)) * (a + b * kv); };
    const double c1 = cost(1, 6.2, 0.302);
    const double c2 = p.V <= HALF_MAX_V || (n <= 2 * sms && p.V <= half_sm::max_v()) ? cost(2, 5.0, 0.535) : 1e30;
    const double c4 = p.V <= QUARTER_MAX_V ? cost(4, 6.0, 1.06) : 1e30;
    if (n <= sms ? p.V >= 16384 : (c1 < c2 && c1 < c4)) return full_sm::launch(p, st, n_launches, served);
    if (n <= sms || c2 < c4) return half_sm::launch(p, st, n_launches, served);
    return quarter_sm::launch(p, st, n_launches, served);
  }
  if (p.V <= QUARTER_MAX_V && p.V <= quarter_sm::max_v()) return quarter_sm::launch(p, st, n_launches, served);
  if (p.V <= HALF_MAX_V && p.V <= half_sm::max_v()) return half_sm::launch(p, st, n_launches, served);
  return full_sm::launch(p, st, n_launches, served);
}

}  // namespace saki
