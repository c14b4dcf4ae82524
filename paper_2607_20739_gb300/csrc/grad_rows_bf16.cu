// The streaming gradient kernel's bf16 variants (grad_rows.cuh).
#include "grad_rows.cuh"

namespace pgc {

GradRowsKernel grad_rows_kernel_bf16(int g, int lpr, int nch, int r, bool full) { return pick_rows_kernel<uint16_t>(g, lpr, nch, r, full); }

}  // namespace pgc
