// The streaming gradient kernel's fp32 variants (grad_rows.cuh).
#include "grad_rows.cuh"

namespace pgc {

GradRowsKernel grad_rows_kernel_f32(int g, int lpr, int nch, int r, bool full) { return pick_rows_kernel<float>(g, lpr, nch, r, full); }

}  // namespace pgc
