// Standalone tail kernels of a step (used when the gradient kernel does not
// fuse them; see tail.cuh for the arithmetic):
//   K4 commit_kernel  one CTA column-slice per evaluated partition: the new
//                     gradient g_e = (1/m_e) * ordered sum of its partials,
//                     written into every store that keeps the copy (§VI-A).
//                     Below 2^20 parameters the decode kernel does it first.
//   K6 decode_kernel  decode coefficients derived on the device from the
//                     straggler mask (§IV-A, §V-B), decode, SGD (§III).
// Both may be launched as programmatic dependents of the previous kernel:
// they wait for it (griddepcontrol.wait) before reading its results, and the
// decode derives its coefficients (which need only the mask) before waiting.
#include "tail.cuh"

namespace pgc {

// One CTA per (column slice, evaluated partition); a thread sums one float4
// column over the partition's items (in item order), eight loads in flight.
__global__ void commit_slice_kernel(CommitArgs a, int64_t slice4) {
  grid_dep_launch();
  grid_dep_wait();
  const int e = blockIdx.y;
  const int i0 = a.e_item0[e], i1 = a.e_item0[e + 1];
  const int64_t P4 = a.P / 4;
  const int64_t c0 = (int64_t)blockIdx.x * slice4;
  if (c0 >= P4) return;
  const int64_t w4 = c0 + slice4 <= P4 ? slice4 : P4 - c0;
  const float4* src = reinterpret_cast<const float4*>(a.partials);
  const float sc = a.e_scale[e];
  const int32_t* dest = a.e_dest + (int64_t)e * a.ndest;
  for (int64_t j = threadIdx.x; j < w4; j += blockDim.x) {
    const int64_t p = c0 + j;
    float4 acc = f4zero();
    for (int it = i0; it < i1; it += 8) {
      float4 v[8];
#pragma unroll
      for (int u = 0; u < 8; ++u) v[u] = it + u < i1 ? __ldcg(src + (int64_t)(it + u) * P4 + p) : f4zero();
#pragma unroll
      for (int u = 0; u < 8; ++u) acc = f4add(acc, v[u]);
    }
    acc = make_float4(acc.x * sc, acc.y * sc, acc.z * sc, acc.w * sc);
    for (int k = 0; k < a.ndest; ++k) {
      const int dst = dest[k];
      if (dst >= 0) reinterpret_cast<float4*>(a.store)[(int64_t)dst * P4 + p] = acc;
    }
  }
}

template <typename K, typename... Args>
static cudaError_t launch_maybe_pdl(bool pdl, K kern, dim3 grid, dim3 block, cudaStream_t st, Args... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = 0;
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = pdl ? 1 : 0;
  return cudaLaunchKernelEx(&cfg, kern, args...);
}

cudaError_t launch_commit(const CommitArgs& a, cudaStream_t st, bool pdl) {
  if (a.nE <= 0) return cudaSuccess;
  const int64_t P4 = a.P / 4;
  const int threads = 128;
  // one float4 column per thread: slices of 128 columns per CTA, one grid row
  // per partition (the sums are short and latency-bound: many CTAs)
  const int64_t slice4 = threads;
  const int64_t bx = (P4 + slice4 - 1) / slice4;
  return launch_maybe_pdl(pdl, commit_slice_kernel, dim3((unsigned)bx, (unsigned)a.nE), dim3(threads), st, a, slice4);
}

// kCommit: the step's commit first, for the same columns (a column's decode
// reads only that column of the stores, so a CTA barrier is enough): thread
// row y sums the items of partitions y, y + kY, ..., in item order.  One
// launch instead of two.
template <bool kCommit, int kY, bool kAll>
__global__ void __launch_bounds__(256) decode_kernel(DecodeArgs a, CommitArgs cm) {
  constexpr int kX = 256 / kY;
  __shared__ DecodePlan pl;
  __shared__ float4 red[2 * kY][kX];
  grid_dep_launch();
  if (threadIdx.x < 32) derive_plan_warp(a, pl, threadIdx.x);   // needs only the mask
  __syncthreads();
  grid_dep_wait();
  if (blockIdx.x == 0 && threadIdx.x < 32) write_coeffs_warp(a, threadIdx.x);
  const int64_t P4 = a.P / 4, nq = (P4 + kX - 1) / kX;
  auto bar = [] { __syncthreads(); };
  for (int64_t q = blockIdx.x; q < nq; q += gridDim.x) {
    if constexpr (kCommit) {
      const int64_t p = q * kX + threadIdx.x % kX;
      if (p < P4) {
        const float4* src = reinterpret_cast<const float4*>(cm.partials) + p;
        for (int e = threadIdx.x / kX; e < cm.nE; e += kY) {
          const int i0 = cm.e_item0[e], i1 = cm.e_item0[e + 1];
          float4 acc = f4zero();
          for (int it = i0; it < i1; it += 8) {
            float4 v[8];
#pragma unroll
            for (int u = 0; u < 8; ++u) v[u] = it + u < i1 ? __ldcg(src + (int64_t)(it + u) * P4) : f4zero();
#pragma unroll
            for (int u = 0; u < 8; ++u) acc = f4add(acc, v[u]);
          }
          const float sc = cm.e_scale[e];
          acc = make_float4(acc.x * sc, acc.y * sc, acc.z * sc, acc.w * sc);
          for (int k = 0; k < cm.ndest; ++k) {
            const int dst = cm.e_dest[(int64_t)e * cm.ndest + k];
            if (dst >= 0) reinterpret_cast<float4*>(cm.store)[(int64_t)dst * P4 + p] = acc;
          }
        }
      }
      __syncthreads();
    }
    decode_chunk<kY, kAll>(a, pl, red, (int)threadIdx.x, q, bar);
  }
}

// Sum of cnt float4 loads base[off(j)], j = 0..cnt-1, issued eight at a time
// so that each thread keeps eight independent loads in flight.
template <class Off>
__device__ __forceinline__ float4 sum_loads8(const float4* base, int cnt, Off off) {
  float4 acc = f4zero();
  for (int j0 = 0; j0 < cnt; j0 += 8) {
    float4 v[8];
#pragma unroll
    for (int j = 0; j < 8; ++j) v[j] = j0 + j < cnt ? __ldcg(base + off(j0 + j)) : f4zero();
#pragma unroll
    for (int j = 0; j < 8; ++j) acc = f4add(acc, v[j]);
  }
  return acc;
}

// Decode + SGD for large P: one thread per float4 column, grid-stride, no
// barriers after the plan.  Same arithmetic as decode_chunk.
__global__ void __launch_bounds__(256) decode_wide_kernel(DecodeArgs a) {
  __shared__ DecodePlan pl;
  grid_dep_launch();
  if (threadIdx.x < 32) derive_plan_warp(a, pl, threadIdx.x);   // needs only the mask
  __syncthreads();
  grid_dep_wait();
  if (blockIdx.x == 0 && threadIdx.x < 32) write_coeffs_warp(a, threadIdx.x);
  const int64_t P4 = a.P / 4;
  const int c = a.c;
  const float4* store = reinterpret_cast<const float4*>(a.store);
  float4* U = reinterpret_cast<float4*>(a.U);
  const int64_t slotP = (int64_t)c * P4;           // float4s per store
  if (a.pre && a.u_ready && a.slot >= 0) {
    // the slots other than o_t were summed early: add U[o_t] and the
    // deviating stores' slot o_t
    const float4* pre = reinterpret_cast<const float4*>(a.pre);
    for (int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; p < P4; p += (int64_t)gridDim.x * blockDim.x) {
      float4 w = __ldcg(reinterpret_cast<const float4*>(a.w) + p);
      float4 g = f4fma(pl.B, __ldcg(U + (int64_t)a.slot * P4 + p), __ldcg(pre + p));
      const float4* cur = store + (int64_t)a.slot * P4 + p;
      for (int q0 = 0; q0 < pl.ndev; q0 += 8) {
        float4 v[8];
#pragma unroll
        for (int j = 0; j < 8; ++j) v[j] = q0 + j < pl.ndev ? __ldcg(cur + (int64_t)pl.dev[q0 + j] * slotP) : f4zero();
#pragma unroll
        for (int j = 0; j < 8; ++j)
          if (q0 + j < pl.ndev) g = f4fma(pl.devc[q0 + j], v[j], g);
      }
      w = f4fma(-a.lr, g, w);
      store_outputs_any(a, p, g, w);
    }
    return;
  }
  for (int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; p < P4; p += (int64_t)gridDim.x * blockDim.x) {
    float4 V = f4zero(), w = __ldcg(reinterpret_cast<const float4*>(a.w) + p);
    if (a.slot < 0) {
      for (int o = 0; o < c; ++o) {
        const float4 u = sum_loads8(store + (int64_t)o * P4 + p, a.owners, [&](int r) { return (int64_t)r * slotP; });
        U[(int64_t)o * P4 + p] = u;
        V = f4add(V, u);
      }
    } else {
      const int skip = a.u_ready ? -1 : a.slot;      // the slot re-summed below
      const int nu = a.u_ready ? c : c - 1;
      V = sum_loads8(U + p, nu, [&](int j) { return (int64_t)(skip >= 0 && j >= skip ? j + 1 : j) * P4; });
      if (!a.u_ready) {
        const float4 u =
            sum_loads8(store + (int64_t)a.slot * P4 + p, a.owners, [&](int r) { return (int64_t)r * slotP; });
        U[(int64_t)a.slot * P4 + p] = u;
        V = f4add(V, u);
      }
    }
    float4 D = f4zero();
    for (int q = 0; q < pl.ndev; ++q) {
      const float4 Cr = sum_loads8(store + (int64_t)pl.dev[q] * slotP + p, c, [&](int o) { return (int64_t)o * P4; });
      D = f4fma(pl.devc[q], Cr, D);
    }
    const float4 g = f4fma(pl.B, V, D);
    w = f4fma(-a.lr, g, w);
    store_outputs_any(a, p, g, w);
  }
}

// Columns from which the one-thread-per-column decode is used (8 x 700 x 4096,
// K = 300: 86 us per step, the kernel above 90; 16 x 1000 x 4096, K = 1000: 426, 443).
constexpr int64_t kWideDecodeMinP4 = 1 << 18;

bool decode_commits(int64_t P) { return P / 4 < kWideDecodeMinP4; }

template <bool kCommit, bool kAll>
static auto decode_instance(int y) {
  return y == 8 ? decode_kernel<kCommit, 8, kAll> : y == 4 ? decode_kernel<kCommit, 4, kAll> : decode_kernel<kCommit, 2, kAll>;
}

cudaError_t launch_decode(const DecodeArgs& a, const CommitArgs* cm, cudaStream_t st, bool pdl, int sm_count) {
  if (a.n > kMaxWorkers || a.owners > kMaxWorkers) return cudaErrorInvalidValue;
  if (a.P / 4 >= kWideDecodeMinP4) {
    if (cm) return cudaErrorInvalidValue;
    int64_t blocks = (a.P / 4 + 255) / 256;
    if (blocks > (int64_t)sm_count * 8) blocks = (int64_t)sm_count * 8;
    return launch_maybe_pdl(pdl, decode_wide_kernel, dim3((unsigned)blocks), dim3(256), st, a);
  }
  // Thread rows per column: each column's loads are one latency, so first a grid that
  // is resident at once (8 CTAs per SM), then as many rows as that leaves.  us per
  // step with 8 / 4 / 2 / 1 rows (terms of a column in brackets):
  //   n = 12, K = 33,  d = 3072 [27]   154 / 158 / 160 / 165    one wave with 8 rows
  //   n = 12, K = 100, d = 3072 [27]   228 / 224 / 233 / 237    with 4
  //   n = 8,  K = 128, d = 4096 [12]    71 /  66 /  64 /  65    with 2
  //   n = 16, K = 250, d = 2048 [41]    73 /  70 /  69 /  74    with 2
  //   n = 8,  K = 200, d = 4096 [12]    83 /   - /  73 /  72    with 1
  //   n = 32, K = 240, d = 4096 [95]   171 /   - / 164 / 170    with 1: two rows at least
  const int64_t P4 = a.P / 4, wave = (int64_t)sm_count * 8;
  int y = 8;
  while (y > 2 && (P4 + 256 / y - 1) / (256 / y) > wave) y /= 2;
  int64_t blocks = (P4 + 256 / y - 1) / (256 / y);
  blocks = blocks > wave ? wave : blocks < 1 ? 1 : blocks;
  // the refresh of every slot has instances of its own: its registers are not the steady step's
  const bool all = a.slot < 0;
  auto kern = cm ? (all ? decode_instance<true, true>(y) : decode_instance<true, false>(y))
                 : (all ? decode_instance<false, true>(y) : decode_instance<false, false>(y));
  return launch_maybe_pdl(pdl, kern, dim3((unsigned)blocks), dim3(256), st, a, cm ? *cm : CommitArgs{});
}

// ---------------------------------------------------------------------------
// fp32 -> bf16 (round to nearest even)
// ---------------------------------------------------------------------------
__global__ void f32_to_bf16_kernel(const float* __restrict__ src, uint16_t* __restrict__ dst, int64_t count) {
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < count; i += (int64_t)gridDim.x * blockDim.x) {
    __nv_bfloat16 b = __float2bfloat16_rn(src[i]);
    dst[i] = *reinterpret_cast<uint16_t*>(&b);
  }
}

cudaError_t launch_f32_to_bf16(const float* src, uint16_t* dst, int64_t count, cudaStream_t st) {
  if (count <= 0) return cudaSuccess;
  int64_t blocks = (count + 255) / 256;
  if (blocks > 4096) blocks = 4096;
  f32_to_bf16_kernel<<<(unsigned)blocks, 256, 0, st>>>(src, dst, count);
  return cudaGetLastError();
}

}  // namespace pgc
