// Host side of the streaming gradient kernel (grad_rows.cuh): the variant a row
// length takes, its stages, the launch.
#include "grad_rows.cuh"

namespace pgc {

namespace {

// id = bf16 << 30 | G << 24 | R << 20 | LPR << 8 | NCH
struct RowsVariant {
  int g, r, lpr, nch, bf16;
};
RowsVariant unpack(int id) {
  return {(id >> 24) & 31, (id >> 20) & 15, (id >> 8) & 63, id & 31, (id >> 30) & 1};
}

int64_t max_features(int dtype) { return dtype == PGC_BF16 ? 32768 : 16384; }

StageCfg stage_cfg(int variant, int64_t ld, int tail) {
  const RowsVariant v = unpack(variant);
  const int64_t rb = ld * (v.bf16 ? 2 : 4);
  const int unit = v.r * (32 / v.lpr);   // rows of one batch
  StageCfg c;
  // stages of 48 KB (a stage's fixed cost is a few hundred cycles: 32 KB took up
  // to 1.2x as long, d = 128 and 1152), 64 KB where the teams' batches then split it
  // evenly
  const int kb = v.bf16 && v.nch >= 3 && v.nch <= 5 && (v.g == 4 || (v.g == 2 && v.nch == 5)) ? 64 : 48;
  int sr = (int)(kb * 1024 / rb) / unit * unit;
  sr = sr < unit ? unit : (sr > 512 ? 512 : sr);
  c.SR = sr;
  c.stage_bytes = (uint32_t)((c.SR * rb + 127) / 128 * 128);
  c.LS = ((c.SR + 3 + 3) / 4) * 4;   // labels of SR rows read from a 4-row-aligned start
  c.red_bytes = v.g == kNW ? 0 : (size_t)(kNW / v.g) * ld * sizeof(float);
  c.plan_bytes = tail == 2 ? sizeof(DecodePlan) : 0;
  const size_t budget = 220 * 1024;
  int S = 10;
  while (S > 2 && fixed_bytes(S, c.LS, c.red_bytes, c.plan_bytes) + (size_t)S * c.stage_bytes > budget) --S;
  c.S = S;
  c.smem = fixed_bytes(S, c.LS, c.red_bytes, c.plan_bytes) + (size_t)S * c.stage_bytes;
  return c;
}

}  // namespace

// nc = 512-byte warp-wide chunks per row.  G and R were chosen by timing the
// neighbours on 400 MB of features (us per step; chosen / other):
//   nc = 1    R = 8 / R = 4                 fp32 62.7 / 65.7   bf16 67.7 / 80.9
//   nc = 8    G = 2, R = 4 / R = 2          fp32 62.5 / 63.5   bf16 70.8 / 80.8
//   nc = 9    fp32 G = 2, R = 2 / G = 4, R = 4   67.3 / 71.1
//             bf16 G = 2, R = 4 / G = 4, R = 4   80.2 / 89.0
//   nc = 16   fp32 G = 2, R = 2 / G = 4, R = 4   63.8 / 68.5
//             bf16 G = 4, R = 4 / G = 2, R = 4   77.8 / 114.8
//   nc = 20   G = 4, R = 4 / G = 8, R = 4   fp32 71.4 / 72.2   bf16 90.1 / 102.1
//   nc = 32   G = 8, R = 4 / R = 2          fp32 75.8 / 82.4   bf16 72.6 / 97.1
//   nc = 64   G = 8, R = 2 / R = 1          fp32 66.9 / 74.3   bf16 98.0 / 124.4
// Short rows take R = 4 where R = 8 would leave SMs without a batch for every
// warp (4 partitions of 256 x 64).
int grad_rows_variant(int dtype, int64_t d, int64_t rows_per_sm, int64_t* ld_out) {
  if (d > max_features(dtype)) return -1;
  const bool bf16 = dtype == PGC_BF16;
  const int vec = bf16 ? 8 : 4;
  const int64_t nv = (d + vec - 1) / vec;               // 16-byte chunks per row
  *ld_out = nv * vec;
  const int nc = (int)((nv + 31) / 32);
  int g, r, lpr = 32, nch;
  if (nc <= 4) {
    g = 1;
    lpr = nv <= 8 ? 8 : nv <= 16 ? 16 : 32;
    r = nc <= 2 && rows_per_sm >= kNW * 8 * (32 / lpr) ? 8 : 4;
  } else if (nc <= 8 || (bf16 && nc <= 10)) {
    g = 2;
    r = 4;
  } else if (nc <= 16) {
    g = bf16 ? 4 : 2;
    r = bf16 ? 4 : 2;
  } else if (nc <= 24) {
    g = r = 4;
  } else {
    g = 8;
    r = nc <= 32 ? 4 : nc <= 64 ? 2 : 1;
  }
  nch = (nc + g - 1) / g;
  if (nch > 8) nch = (nch + 1) / 2 * 2;
  return (bf16 ? 1 << 30 : 0) | g << 24 | r << 20 | lpr << 8 | nch;
}

int grad_rows_min_item(int variant) {
  const RowsVariant v = unpack(variant);
  return kNW / v.g * v.r * (32 / v.lpr);
}

bool grad_rows_unpadded(int dtype, int64_t d) {
  const int64_t least = dtype == PGC_BF16 ? 64 : 32;
  return d >= least && d <= max_features(dtype) && (d & (d - 1)) == 0;
}

int grad_rows_stage_rows(int variant, int64_t ld, int dtype) {
  (void)dtype;
  return stage_cfg(variant, ld, 0).SR;
}

cudaError_t launch_grad_rows(const GradRowsArgs& a, int variant, cudaStream_t st) {
  if (a.nitems <= 0) return cudaSuccess;
  const RowsVariant v = unpack(variant);
  const bool full = a.ld == (int64_t)v.nch * v.g * v.lpr * (v.bf16 ? 8 : 4);
  const GradRowsKernel kern =
      v.bf16 ? grad_rows_kernel_bf16(v.g, v.lpr, v.nch, v.r, full) : grad_rows_kernel_f32(v.g, v.lpr, v.nch, v.r, full);
  const StageCfg c = stage_cfg(variant, a.ld, a.tail);
  if (!kern || c.smem > 227 * 1024) return cudaErrorInvalidValue;
  // the ranges' CTAs, a persistent grid when items are taken dynamically, else one CTA per item
  const int grid = a.cta_item0 ? a.grid : a.work_ctr ? (a.grid < a.nitems ? a.grid : a.nitems) : a.nitems;
  if (grid < 1) return cudaErrorInvalidValue;
  cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)c.smem);
  if (e != cudaSuccess) return e;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)grid);
  cfg.blockDim = dim3(kThreads);
  cfg.dynamicSmemBytes = c.smem;
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = a.pdl ? 1 : 0;
  return cudaLaunchKernelEx(&cfg, kern, a, c);
}

}  // namespace pgc
