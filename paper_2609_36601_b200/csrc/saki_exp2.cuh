// 2^y in float64 at eight operations of the float64 pipe, for the kernels that work in float64 throughout.
// y is split by a magic-number addition into n + i/256 + r; 2^(i/256) comes from a table in shared memory and 2^r from its
// Taylor polynomial (|r| <= 1/512: the first dropped term is 4e-17).  A degree less would be seen: KL is a difference of sums of
// these of the size of 1, an error e of theirs moves lambda by e / (2 eps) of itself.  The table is stored 16 times over, one copy per
// 64-bit bank, so the lookups of a half-warp never conflict (32 KB).
#pragma once
#include "saki_device.cuh"

namespace saki {

constexpr int EXP2_TAB = 256, EXP2_COPIES = 16;

// fills the table (all threads of the block; a barrier is the caller's)
__device__ __forceinline__ void exp2_table(double* tab, int tid, int n_threads) {
  for (int i = tid; i < EXP2_TAB; i += n_threads) {
    double e = exp2((double)i * (1.0 / EXP2_TAB));
    e = __hiloint2double(__double2hiint(e) - (i << 12), __double2loint(e));
#pragma unroll 1
    for (int c = 0; c < EXP2_COPIES; ++c) tab[i * EXP2_COPIES + ((c + tid) & (EXP2_COPIES - 1))] = e;
  }
}

// The entry of 2^(i/256) has i << 12 taken off its high word: adding the low word of y + M, shifted by 12, then puts
// the exponent in and the index back in one addition.
// The coefficients are read from the constant bank (as operands: three 64-bit immediates cost two moves each per
// exponential once registers are short, and a float64 operation on three register operands runs at two thirds of the rate).
static __constant__ double EXP2_COEF[4] = {9.618129107628477e-03, 5.550410866482158e-02, 2.402265069591007e-01, 6.931471805599453e-01};   // ln2^i / i!, i = 4..1
struct Exp2 {
  uint32_t lane8;   // this lane's copy of the table: byte offset among the 16 copies of an entry
  const double* tab;
  __device__ __forceinline__ Exp2(const double* table, int lane) : lane8((uint32_t)(lane & (EXP2_COPIES - 1)) * 8u), tab(table) {}
  // 2^y for y <= ~1000; y below -1000 counts as -1000 (clamped through the high word: an unsigned minimum)
  __device__ __forceinline__ double operator()(double y) const {
    const uint32_t hi = min((uint32_t)__double2hiint(y), 0xC08F4000u);
    y = __hiloint2double((int)hi, __double2loint(y));
    const double M = 26388279066624.0;                       // 1.5 * 2^44: the low word of y + M is round(256 y)
    const double t = y + M;
    const double r = y - (t - M);
    const int k = __double2loint(t);
    double T = *(const double*)((const char*)tab + ((((uint32_t)k << 7) & 0x7f80u) | lane8));
    double q = fma(r, EXP2_COEF[0], EXP2_COEF[1]);
    q = fma(r, q, EXP2_COEF[2]);
    q = fma(r, q, EXP2_COEF[3]);
    T = __hiloint2double(__double2hiint(T) + (k << 12), __double2loint(T));
    return fma(T * r, q, T);
  }
};

// float64 to float, ready to be rounded to bf16: truncated, with the last bit set if anything was dropped (rounded to
// odd), so that the second rounding is the only one.  (The low 29 bits of a float64 do not fit a normal float.)
__device__ __forceinline__ float to_odd(double v) {
  return __uint_as_float(__float_as_uint(__double2float_rz(v)) | (uint32_t)((__double2loint(v) << 3) != 0));
}

}  // namespace saki
