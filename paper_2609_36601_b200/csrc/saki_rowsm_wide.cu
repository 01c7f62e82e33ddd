// Row-per-SM kernel, the variant with one CTA of 512 threads per SM and two CTAs per row (the implementation is
// saki_rowsm_impl.cuh).
#define SAKI_ROWSM_WIDE 1
#include "saki_rowsm_impl.cuh"
