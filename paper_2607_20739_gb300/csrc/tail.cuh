// Block-level pieces of a step's tail, shared by the standalone commit /
// decode kernels and by the gradient kernel's fused tail:
//
//   commit_block      g_e = scale * (ordered sum of partition e's partial
//                     sums), written to each store that keeps this copy
//                     (§VI-A: every worker keeps its latest gradients).
//   derive_plan_warp  the decode coefficients from the straggler mask, by one
//                     warp (§IV-A FR: one coded gradient per group, times
//                     1/n; §V-B CR: every received coded gradient, times
//                     1/(n mu) = 1/((n-s)c)).
//   decode_columns /  ghat = B * sum_o U[o] + sum_{stores r with b_r != B}
//   decode_chunk      (b_r - B) * sum_o store[r][o], fused with the SGD update
//                     beta <- beta - eta * ghat (§III); U[o_t] is refreshed.
//
// Decode arithmetic.  Coded gradient of store r: C_r = sum_o store[r][o]
// (every coefficient 1, §IV-A / §V-B).  Slot totals U[o] = sum_r store[r][o].
// With b_r the summed coefficient of the workers sharing store r and a
// baseline B,  ghat = sum_r b_r C_r = B sum_o U[o] + sum_{b_r != B} (b_r - B) C_r.
// FR: every group's coefficient is 1/n = B, so ghat = (1/n) sum_o U[o].
// CR: B = 1/((n-s)c) and only the s stragglers deviate (b_r = 0).  This reads
// (owners + c + s c) gradients instead of the (n - s) c of the literal sum.
//
// Data written by other CTAs of the same grid is read with ld.global.cg (L2)
// after a release (writer fence + atomic) / acquire (reader atomic + fence)
// handshake.
#pragma once

#include "dev_common.cuh"
#include "pgc_internal.h"
#include "pgc.h"

namespace pgc {

__device__ __forceinline__ float4 f4add(float4 a, float4 b) {
  return make_float4(a.x + b.x, a.y + b.y, a.z + b.z, a.w + b.w);
}
__device__ __forceinline__ float4 f4fma(float s, float4 a, float4 b) {
  return make_float4(fmaf(s, a.x, b.x), fmaf(s, a.y, b.y), fmaf(s, a.z, b.z), fmaf(s, a.w, b.w));
}
__device__ __forceinline__ float4 f4zero() { return make_float4(0.f, 0.f, 0.f, 0.f); }

__device__ __forceinline__ void grid_dep_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void grid_dep_launch() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

// ---------------------------------------------------------------------------
// commit
// ---------------------------------------------------------------------------
__device__ __forceinline__ void commit_block(const float* partials, int64_t P, int i0, int i1, float scale,
                                             const int32_t* dest, int ndest, float* store, int tid, int nthr) {
  constexpr int kB = 20;          // partials loaded per batch (one item per SM: 152 / 8 = 19 at n = 8)
  const int64_t P4 = P / 4;
  const float4* src = reinterpret_cast<const float4*>(partials);
  for (int64_t p = tid; p < P4; p += nthr) {
    float4 acc = f4zero();
    for (int it = i0; it < i1; it += kB) {
      float4 v[kB];
#pragma unroll
      for (int j = 0; j < kB; ++j) v[j] = it + j < i1 ? __ldcg(src + (int64_t)(it + j) * P4 + p) : f4zero();
#pragma unroll
      for (int j = 0; j < kB; ++j) acc = f4add(acc, v[j]);
    }
    acc = make_float4(acc.x * scale, acc.y * scale, acc.z * scale, acc.w * scale);
    for (int j = 0; j < ndest; ++j) {
      const int dst = dest[j];
      if (dst >= 0) reinterpret_cast<float4*>(store)[(int64_t)dst * P4 + p] = acc;
    }
  }
}

// ---------------------------------------------------------------------------
// decode plan
// ---------------------------------------------------------------------------
struct DecodePlan {
  float B;                     // baseline coefficient
  int ndev;                    // stores whose summed coefficient differs from B
  int dev[kMaxWorkers];        // ascending
  float devc[kMaxWorkers];     // b_r - B
};

__device__ __forceinline__ bool straggles(const MaskBits& m, int i) { return (m.w[i >> 5] >> (i & 31)) & 1u; }

// FR: representative of group g = lowest-index non-straggler, or -1.
__device__ __forceinline__ int fr_rep(const DecodeArgs& a, int g) {
  for (int l = 0; l < a.c; ++l)
    if (!straggles(a.mask, g * a.c + l)) return g * a.c + l;
  return -1;
}

// One warp derives the plan; invalid masks set kErrBadMask.  It depends only
// on the mask, so it can run before the step's gradients exist.  Plan: a
// DecodePlan, or a struct of the same members with shorter dev / devc arrays
// (more deviating stores than they hold also set kErrBadMask).
template <class Plan>
__device__ __forceinline__ void derive_plan_warp(const DecodeArgs& a, Plan& pl, int lane) {
  constexpr int kCap = (int)(sizeof(pl.dev) / sizeof(pl.dev[0]));
  const bool cr = a.scheme == PGC_CR;
  const float A = cr ? 1.0f / (float)((a.n - a.s) * a.c) : 1.0f / (float)a.n;
  int cnt = 0;
  for (int i = lane; i < a.n; i += 32) cnt += straggles(a.mask, i) ? 1 : 0;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) cnt += __shfl_xor_sync(0xffffffffu, cnt, o);
  int nd = 0;
  for (int base = 0; base < a.owners; base += 32) {
    const int r = base + lane;
    float br = A;
    if (r < a.owners) {
      if (cr) {
        br = straggles(a.mask, r) ? 0.f : A;         // one store per worker
      } else {
        const bool alive = fr_rep(a, r) >= 0;        // 1/n from the group's representative
        br = alive ? A : 0.f;
        if (!alive) atomicOr(a.status, kErrBadMask);
      }
    }
    const bool devr = r < a.owners && br != A;
    const unsigned bal = __ballot_sync(0xffffffffu, devr);
    if (devr) {
      const int pos = nd + __popc(bal & ((1u << lane) - 1u));
      if (pos < kCap) {
        pl.dev[pos] = r;
        pl.devc[pos] = br - A;
      }
    }
    nd += __popc(bal);
  }
  if (lane == 0) {
    pl.ndev = nd < kCap ? nd : kCap;
    pl.B = A;
    if (cnt != a.s || nd > kCap) atomicOr(a.status, kErrBadMask);
  }
  __syncwarp();
}

// The per-worker coefficients a_i, written by one warp of the decoding CTA.
__device__ __forceinline__ void write_coeffs_warp(const DecodeArgs& a, int lane) {
  if (!a.coeff_out) return;
  const bool cr = a.scheme == PGC_CR;
  const float A = cr ? 1.0f / (float)((a.n - a.s) * a.c) : 1.0f / (float)a.n;
  for (int i = lane; i < a.n; i += 32)
    a.coeff_out[i] = cr ? (straggles(a.mask, i) ? 0.f : A) : (fr_rep(a, i / a.c) == i ? A : 0.f);
}

// Four parameters (float4 column i) as three bf16 parts each, w = w1 + w2 + w3
// up to 2^-27 |w| (round to nearest); part j of the array starts at j * stride.
// Beyond bf16's largest value (3.39e38; a class masked by fp32's lowest value or by
// -infinity) a part is that value, not the infinity it would round to, whose
// remainder has the other sign or is NaN; an infinity becomes three of them.
constexpr float kBf16Max = 3.3895313892515355e38f;           // (2 - 2^-7) 2^127
__device__ __forceinline__ float bf16_range(float v) {
  return fabsf(v) > kBf16Max ? copysignf(kBf16Max, v) : v;   // NaN stays
}
__device__ __forceinline__ void store_split4(uint16_t* dst, int64_t stride, int64_t i, float4 v) {
  const bool beyond = fmaxf(fmaxf(fabsf(v.x), fabsf(v.y)), fmaxf(fabsf(v.z), fabsf(v.w))) > kBf16Max;
#pragma unroll
  for (int j = 0; j < 3; ++j) {
    float4 r = v;
    if (beyond) r = make_float4(bf16_range(v.x), bf16_range(v.y), bf16_range(v.z), bf16_range(v.w));
    const __nv_bfloat162 lo = __floats2bfloat162_rn(r.x, r.y), hi = __floats2bfloat162_rn(r.z, r.w);
    uint2 pk;
    pk.x = *reinterpret_cast<const uint32_t*>(&lo);
    pk.y = *reinterpret_cast<const uint32_t*>(&hi);
    reinterpret_cast<uint2*>(dst + j * stride)[i] = pk;
    v = make_float4(v.x - __low2float(lo), v.y - __high2float(lo), v.z - __low2float(hi), v.w - __high2float(hi));
  }
}

// The caller's copies of ghat and beta, written without the padding of the
// parameter rows.  kUserSame: rows of ld = d floats, 16-byte aligned.
// kUserPrefix: one class, the caller's array ends after user_n floats.
// kUserRows: [K][user_d] behind rows of 4 row4 floats, any 4-byte alignment.
enum { kUserSame = 0, kUserPrefix = 1, kUserRows = 2 };
__device__ __forceinline__ void put4(float* dst, int n, float4 v) {
  if (n >= 4 && (reinterpret_cast<uintptr_t>(dst) & 15) == 0) {
    *reinterpret_cast<float4*>(dst) = v;
    return;
  }
  if (n > 0) dst[0] = v.x;
  if (n > 1) dst[1] = v.y;
  if (n > 2) dst[2] = v.z;
  if (n > 3) dst[3] = v.w;
}
template <int kUser>
__device__ __forceinline__ void store_user(const DecodeArgs& a, int64_t p, float4 g, float4 w) {
  if constexpr (kUser == kUserSame) {
    if (a.w_user) reinterpret_cast<float4*>(a.w_user)[p] = w;
    if (a.g_user) reinterpret_cast<float4*>(a.g_user)[p] = g;
  } else {
    int64_t off = 4 * p, n = a.user_n - off;
    if constexpr (kUser == kUserRows) {
      const uint32_t k = (uint32_t)p / a.row4;                // P / 4 < 2^32: 4096 classes of 2^20 features
      const int64_t j = 4 * (int64_t)((uint32_t)p - k * a.row4);
      off = (int64_t)k * a.user_d + j;
      n = a.user_d - j;
    }
    const int m = n < 4 ? (int)n : 4;
    if (a.w_user) put4(a.w_user + off, m, w);
    if (a.g_user) put4(a.g_user + off, m, g);
  }
}

template <int kUser>
__device__ __forceinline__ void store_outputs(const DecodeArgs& a, int64_t p, float4 g, float4 w) {
  reinterpret_cast<float4*>(a.w)[p] = w;
  reinterpret_cast<float4*>(a.gout)[p] = g;
  store_user<kUser>(a, p, g, w);
  if (a.wb) {
    __nv_bfloat162 lo = __floats2bfloat162_rn(w.x, w.y);
    __nv_bfloat162 hi = __floats2bfloat162_rn(w.z, w.w);
    uint2 pk;
    pk.x = *reinterpret_cast<uint32_t*>(&lo);
    pk.y = *reinterpret_cast<uint32_t*>(&hi);
    reinterpret_cast<uint2*>(a.wb)[p] = pk;
  }
}

// store_outputs for the standalone decode kernels, which serve every path:
// beta as three bf16 parts, and the caller's arrays in any layout (the fused
// tails are compiled for theirs: one more branch cost the few-class kernel 2 us
// of its 57).
__device__ __forceinline__ void store_outputs_any(const DecodeArgs& a, int64_t p, float4 g, float4 w) {
  reinterpret_cast<float4*>(a.w)[p] = w;
  reinterpret_cast<float4*>(a.gout)[p] = g;
  if (a.g_user || a.w_user) {
    if (a.user_d) store_user<kUserRows>(a, p, g, w);
    else store_user<kUserPrefix>(a, p, g, w);
  }
  if (a.wb_stride) {
    store_split4(a.wb, a.wb_stride, p, w);
  } else if (a.wb) {
    __nv_bfloat162 lo = __floats2bfloat162_rn(w.x, w.y);
    __nv_bfloat162 hi = __floats2bfloat162_rn(w.z, w.w);
    uint2 pk;
    pk.x = *reinterpret_cast<uint32_t*>(&lo);
    pk.y = *reinterpret_cast<uint32_t*>(&hi);
    reinterpret_cast<uint2*>(a.wb)[p] = pk;
  }
}

// Decode + SGD of the float4 columns [q0, q1), every column handled by one
// thread (tid of nthr) and no barriers.  When the counts fit the unrolled
// bounds all loads of a column are issued back to back; otherwise plain loops.
template <int kUser>
__device__ __forceinline__ void decode_columns(const DecodeArgs& a, const DecodePlan& pl, int64_t q0, int64_t q1,
                                               int tid, int nthr) {
  constexpr int kMaxO = 8, kMaxC = 4, kMaxD = 4;
  const int64_t P4 = a.P / 4;
  const int c = a.c;
  const float B = pl.B;
  const int ndev = pl.ndev;
  const float4* store = reinterpret_cast<const float4*>(a.store);
  float4* U = reinterpret_cast<float4*>(a.U);
  const bool small = a.owners <= kMaxO && c <= kMaxC && ndev <= kMaxD && a.slot >= 0 && !a.u_ready;
  for (int64_t p = q0 + tid; p < q1; p += nthr) {
    float4 V = f4zero(), D = f4zero();
    // in the streaming kernel's tail beta is read with the terms (4 x 256 x 64: 9.8
    // us per step after them, 9.5 with them); the few-class kernel has no registers
    // for it (32 x 4096 x 3072: 56.8 after, 58.2 with)
    constexpr bool kEarly = kUser == kUserPrefix;
    float4 w = kEarly ? __ldcg(reinterpret_cast<const float4*>(a.w) + p) : f4zero();
    if (small) {
      float4 u[kMaxO], o4[kMaxC], dv[kMaxD][kMaxC];
#pragma unroll
      for (int r = 0; r < kMaxO; ++r)
        u[r] = r < a.owners ? __ldcg(store + ((int64_t)r * c + a.slot) * P4 + p) : f4zero();
#pragma unroll
      for (int o = 0; o < kMaxC; ++o)
        o4[o] = (o < c && o != a.slot) ? __ldcg(U + (int64_t)o * P4 + p) : f4zero();
#pragma unroll
      for (int q = 0; q < kMaxD; ++q)
#pragma unroll
        for (int o = 0; o < kMaxC; ++o)
          dv[q][o] = (q < ndev && o < c) ? __ldcg(store + ((int64_t)pl.dev[q] * c + o) * P4 + p) : f4zero();
      float4 un = f4zero();
#pragma unroll
      for (int r = 0; r < kMaxO; ++r) un = f4add(un, u[r]);
      U[(int64_t)a.slot * P4 + p] = un;
#pragma unroll
      for (int o = 0; o < kMaxC; ++o) V = f4add(V, o < c && o == a.slot ? un : o4[o]);
#pragma unroll
      for (int q = 0; q < kMaxD; ++q) {
        float4 Cr = f4zero();
#pragma unroll
        for (int o = 0; o < kMaxC; ++o) Cr = f4add(Cr, dv[q][o]);
        if (q < ndev) D = f4fma(pl.devc[q], Cr, D);
      }
    } else {
      for (int o = 0; o < c; ++o) {
        if (a.slot < 0 || (o == a.slot && !a.u_ready)) {
          float4 u = f4zero();
          for (int r = 0; r < a.owners; ++r) u = f4add(u, __ldcg(store + ((int64_t)r * c + o) * P4 + p));
          U[(int64_t)o * P4 + p] = u;
          V = f4add(V, u);
        } else {
          V = f4add(V, __ldcg(U + (int64_t)o * P4 + p));
        }
      }
      for (int q = 0; q < ndev; ++q) {
        float4 Cr = f4zero();
        for (int o = 0; o < c; ++o) Cr = f4add(Cr, __ldcg(store + ((int64_t)pl.dev[q] * c + o) * P4 + p));
        D = f4fma(pl.devc[q], Cr, D);
      }
    }
    const float4 g = f4fma(B, V, D);
    if (!kEarly) w = __ldcg(reinterpret_cast<const float4*>(a.w) + p);
    w = f4fma(-a.lr, g, w);
    store_outputs<kUser>(a, p, g, w);
  }
}

// Decode + SGD of 256 / kY float4 columns (chunk q), their terms split over kY
// thread rows (for large P, many CTAs).  Must be called by exactly 256 threads,
// all of which pass every bar().  red: [2 kY][256 / kY].  kAll: every slot is
// refreshed (a.slot < 0), else the one slot.
// Steady steps: each thread row sums its share of the refreshed slot's stores
// (the new U[o_t]) and, with their coefficients, of the other slot totals and
// the deviating stores' slots, all loads of a column in flight over the rows;
// one exchange.  (One slot after the other, with two barriers each, a step of
// 12 x 4096 x 3072, K = 100 spent 21 us here, 16 with one exchange.)  beta is read
// with the terms, not after them: 1 to 2 us of a step.
template <int kY, bool kAll, class Bar>
__device__ void decode_chunk(const DecodeArgs& a, const DecodePlan& pl, float4 (*red)[256 / kY], int tid, int64_t q,
                             Bar bar) {
  constexpr int kX = 256 / kY;
  const int x = tid % kX, y = tid / kX;
  const int64_t P4 = a.P / 4;
  const int c = a.c;
  const float B = pl.B;
  const int ndev = pl.ndev;
  const float4* store = reinterpret_cast<const float4*>(a.store);
  float4* U = reinterpret_cast<float4*>(a.U);
  const int64_t p = q * kX + x;
  const bool inb = p < P4;
  if constexpr (!kAll) {
    float4 un = f4zero(), rest = f4zero(), w = f4zero();
    if (inb) {
      if (y == 0) w = __ldcg(reinterpret_cast<const float4*>(a.w) + p);
      if (!a.u_ready) {
        const float4* s0 = store + (int64_t)a.slot * P4 + p;
        for (int r0 = y; r0 < a.owners; r0 += 4 * kY) {
          float4 v[4];
#pragma unroll
          for (int j = 0; j < 4; ++j)
            v[j] = r0 + j * kY < a.owners ? __ldcg(s0 + (int64_t)(r0 + j * kY) * c * P4) : f4zero();
#pragma unroll
          for (int j = 0; j < 4; ++j) un = f4add(un, v[j]);
        }
      } else if (y == 0) {
        un = __ldcg(U + (int64_t)a.slot * P4 + p);
      }
      // term t: slot total t (t < c, t != o_t), then slot o of deviating store d
      const int nt = c + ndev * c;
      for (int t0 = y; t0 < nt; t0 += 4 * kY) {
        float4 v[4];
        float f[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          const int t = t0 + j * kY;
          v[j] = f4zero();
          f[j] = B;
          if (t < c) {
            if (t != a.slot) v[j] = __ldcg(U + (int64_t)t * P4 + p);
          } else if (t < nt) {
            const int d = (t - c) / c, o = (t - c) - d * c;
            f[j] = pl.devc[d];
            v[j] = __ldcg(store + ((int64_t)pl.dev[d] * c + o) * P4 + p);
          }
        }
#pragma unroll
        for (int j = 0; j < 4; ++j) rest = f4fma(f[j], v[j], rest);
      }
    }
    red[y][x] = un;
    red[kY + y][x] = rest;
    bar();
    if (y == 0 && inb) {
#pragma unroll
      for (int j = 1; j < kY; ++j) {
        un = f4add(un, red[j][x]);
        rest = f4add(rest, red[kY + j][x]);
      }
      if (!a.u_ready) U[(int64_t)a.slot * P4 + p] = un;
      const float4 g = f4fma(B, un, rest);
      w = f4fma(-a.lr, g, w);
      store_outputs_any(a, p, g, w);
    }
    bar();
    return;
  }
  // warm-up, gradient coding: two slots per exchange (one: 26.1 us per step at
  // 16 x 1000 x 1000, K = 10; two: 24.8; four: 24.7, but their shared memory kept CTAs from
  // starting beside the kernel before)
  float4 V = f4zero(), w = f4zero();
  if (inb && y == 0) w = __ldcg(reinterpret_cast<const float4*>(a.w) + p);
  for (int o0 = 0; o0 < c; o0 += 2) {
    float4 part[2];
#pragma unroll
    for (int j = 0; j < 2; ++j) part[j] = f4zero();
    if (inb)
      for (int r = y; r < a.owners; r += kY)
#pragma unroll
        for (int j = 0; j < 2; ++j)
          if (o0 + j < c) part[j] = f4add(part[j], __ldcg(store + ((int64_t)r * c + o0 + j) * P4 + p));
#pragma unroll
    for (int j = 0; j < 2; ++j) red[j * kY + y][x] = part[j];
    bar();
    if (y == 0) {
#pragma unroll
      for (int j = 0; j < 2; ++j) {
        if (o0 + j >= c) break;
        float4 u = red[j * kY][x];
#pragma unroll
        for (int i = 1; i < kY; ++i) u = f4add(u, red[j * kY + i][x]);
        if (inb) U[(int64_t)(o0 + j) * P4 + p] = u;
        V = f4add(V, u);
      }
    }
    bar();
  }
  float4 dv = f4zero();
  if (inb)
    for (int qq = y; qq < ndev; qq += kY) {
      const int r = pl.dev[qq];
      float4 Cr = f4zero();
      for (int o = 0; o < c; ++o) Cr = f4add(Cr, __ldcg(store + ((int64_t)r * c + o) * P4 + p));
      dv = f4fma(pl.devc[qq], Cr, dv);
    }
  red[y][x] = dv;
  bar();
  if (y == 0 && inb) {
    float4 D = red[0][x];
#pragma unroll
    for (int j = 1; j < kY; ++j) D = f4add(D, red[j][x]);
    const float4 g = f4fma(B, V, D);
    w = f4fma(-a.lr, g, w);
    store_outputs_any(a, p, g, w);
  }
  bar();
}

}  // namespace pgc
