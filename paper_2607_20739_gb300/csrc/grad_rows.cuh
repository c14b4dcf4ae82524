// K1 — per-partition gradient of logistic and least-squares losses, one pass
// over the features (§III: g_k = (1/m_k) sum_{x in D_k} grad f; the 1/m_k is
// applied when the partition is committed).
//
// Work: the evaluated partitions' rows are cut into work items (contiguous
// row ranges of one partition) and every CTA, one per SM, takes a run of
// consecutive items of about equal cost (or, on request, CTAs take items
// dynamically).  Each item's sum over its rows of r(x) * x goes to its own
// partial slot, so the result does not depend on which CTA took which item.
//
// Per CTA: one producer thread streams each item's rows from HBM into a ring
// of S shared-memory stages with 1-D bulk async copies (rows and their labels,
// completion counted on the stage's mbarrier); 8 consumer warps dot each row
// with w, form the residual r = sigmoid(x.w) - y (logistic) or x.w - y (least
// squares) and accumulate r * x while the row sits in shared memory, so every
// feature byte is read from HBM once.
//
// Rows are stored with no more padding than the 16-byte alignment of the bulk
// copies asks for, and a row is read in 16-byte chunks: chunk (j G + g) LPR + l
// by lane l (of LPR lanes) of warp g (of the G warps that share a row), for
// j < NCH.  Chunks past the row are skipped, so what follows the row in shared
// memory never enters its sums.  Each lane keeps its
// columns of w and of its accumulator in registers (at most 64 fp32 or 128 bf16
// columns), so G grows with the row length; rows of less than 32 chunks share
// a warp (LPR = 8, 16).  A team of G warps takes R rows at a time: R independent
// dot products per lane (packed FMAs), one butterfly that reduces all R
// together (6 shuffles for R = 4 instead of 20), one exchange of partial dots
// between the team's warps (G > 1), one residual per lane group, then R updates.
// What bounds a team is the latency of that chain, over a thousand cycles
// whatever R; what bounds the kernel is HBM, as long as about 48 KB of rows are
// in some team's hands: 8 / G teams times R rows (grad_rows.cu has the choice).
// us per step, 400 MB of features (59 at the measured copy rate; 16 workers,
// least squares), with one row at a time in rows padded to powers of two, and
// now:
//   d        64  100  128  256  300  512 1024 1100 1500 2048 2500 3001 4096 5000 6000 8192 10000 12000 16384
//   fp32    192  166  125   86  114   66   62  214  163  119  162  140  105  140  122   88   121   106    79
//   now      63   62   62   62   62   61   62   67   67   63   71   72   76   86   86   67    72    73    76
//   bf16    376  278  213  138  168   98   86  275  209  154  226  195  145  186  160  118   185   162   122
//   now      64   77   64   66   80   62   61   86   75   68   84   81   75   90   84   71    95    90    98
// Beyond 16384 bf16 features a lane's 160 to 256 columns of w and sums no longer fit
// its registers (412 to 1296 bytes of spills per thread); still faster than before:
//   d     16392 18000 20000 22528 24576 28000 32768
//   bf16    442   414   378   344   320   289   252
//   now     168   213   196   237   215   228   243
// Item ends: consumers hand their accumulators to a tail warp (through a
// shared buffer and two mbarriers) and keep streaming.  The tail warp sums the
// teams' accumulators in a fixed order into the item's partial slot and,
// with tail >= 1, counts the item for its partition.  When that count
// completes a partition, the consumers commit it at their next item end (or
// after their last item): ordered sum of the partition's partials, scaled by
// 1/m, into its destination stores.  With tail == 2 the CTA that commits the
// last partition also derives the decode coefficients from the mask, decodes
// and applies the SGD update.
//
// Programmatic dependent launch: the producer streams its first item before
// waiting for the previous step's kernel; consumers wait before reading w.
//
// Every wait is bounded (mbarrier try_wait with an iteration and time limit).
// Consumer warps synchronise through mbarriers, never named barriers, so a
// wait that gives up cannot leave another warp blocked: the CTA then skips
// its remaining work, flags the status word and exits.
#pragma once

#include "pgc.h"
#include "tail.cuh"

namespace pgc {

constexpr int kNW = 8;                 // consumer warps per CTA
constexpr int kNT = kNW * 32;          // consumer threads
constexpr int kThreads = kNT + 64;     // + a producer warp + a tail warp
constexpr int kProducer = kNT;        // producer thread
constexpr int kTailWarp = kNW + 1;     // warp index of the tail warp
constexpr int64_t kPrefetchChunkRows = 16;

constexpr int kMaxTeams = 4;           // teams that exchange (G > 1)

struct StageHdr {
  int item;      // work item, or -1: no more work
  int e;         // evaluated-partition position of the item
  int rows;      // rows in this stage
  int lab_off;   // index of the stage's first label in its label slot
  int last;      // last stage of the item
  int pad[3];
};

struct StageCfg {
  int SR;              // rows per stage
  int S;               // stages
  uint32_t stage_bytes;
  int LS;              // floats per label slot
  size_t red_bytes;    // item-end reduction buffer
  size_t plan_bytes;   // decode plan (fused decode only)
  size_t smem;         // dynamic shared memory
};

__device__ __forceinline__ float residual(int loss, float z, float y) {
  return loss == PGC_LOGISTIC ? 1.0f / (1.0f + expf(-z)) - y : z - y;
}

// Item handoff between the consumers and the tail warp.
struct Handoff {
  int item;            // item whose accumulators are in red, or -1: no more items
  int e;
  int commit;          // set by the tail warp: partition to commit, or -1
  int decode;          // set by the consumers: this CTA decodes
  unsigned sync_count; // arrivals at the consumer barrier (ConsumerSync)
};

// Shared memory: [full S | empty S | sync, red_full, red_free, tail_done]
//                [handoff] [S headers] [S label slots] [red / decode scratch]
//                [dot exchange] [S stages]
struct Smem {
  uint64_t* full;
  uint64_t* empty;
  uint64_t* sync;       // consumer barrier (count kNW)
  uint64_t* red_full;   // consumers -> tail warp (count kNW)
  uint64_t* red_free;   // tail warp -> consumers (count 1)
  uint64_t* team_sync;  // [kMaxTeams] dot exchange of the warps that share rows (count G)
  Handoff* ho;
  DecodePlan* plan;     // decode coefficients (tail == 2), derived at kernel start
  StageHdr* hdr;
  float* lab;
  uint8_t* red;
  float* xdot;
  uint8_t* stages;
};

__host__ __device__ inline size_t a128(size_t v) { return (v + 127) & ~size_t(127); }

constexpr size_t kXdotBytes = 2 * 4 * kNW * sizeof(float);   // two buffers of R <= 4 rows per team of G warps

__host__ __device__ inline size_t fixed_bytes(int S, int LS, size_t red, size_t plan) {
  return a128(sizeof(uint64_t) * (2 * S + 3 + kMaxTeams)) + a128(sizeof(Handoff)) + a128(plan) +
         a128(sizeof(StageHdr) * S) + a128(sizeof(float) * LS * S) + a128(red) + a128(kXdotBytes);
}

__device__ __forceinline__ Smem carve(uint8_t* base, const StageCfg& c) {
  Smem m;
  size_t off = 0;
  m.full = reinterpret_cast<uint64_t*>(base);
  m.empty = m.full + c.S;
  m.sync = m.empty + c.S;
  m.red_full = m.sync + 1;
  m.red_free = m.sync + 2;
  m.team_sync = m.sync + 3;
  off = a128(sizeof(uint64_t) * (2 * c.S + 3 + kMaxTeams));
  m.ho = reinterpret_cast<Handoff*>(base + off);
  off = a128(off + sizeof(Handoff));
  m.plan = reinterpret_cast<DecodePlan*>(base + off);
  off = a128(off + c.plan_bytes);
  m.hdr = reinterpret_cast<StageHdr*>(base + off);
  off = a128(off + sizeof(StageHdr) * c.S);
  m.lab = reinterpret_cast<float*>(base + off);
  off = a128(off + sizeof(float) * c.LS * c.S);
  m.red = base + off;
  off = a128(off + c.red_bytes);
  m.xdot = reinterpret_cast<float*>(base + off);
  off = a128(off + kXdotBytes);
  m.stages = base + off;
  return m;
}

// A barrier of the 8 consumer warps on an mbarrier (count kNW), bounded.
// Each warp also counts its arrival on a shared counter; the warp whose
// arrival is the kNW-th knows every other warp is already through its
// pre-barrier work and does not wait (waiting on a phase it completed itself
// was measured to cost microseconds).
struct ConsumerSync {
  uint64_t* bar;
  unsigned* count;
  uint32_t phase;
  int* status;
  __device__ __forceinline__ bool operator()() {
    __syncwarp();
    int last = 0;
    if ((threadIdx.x & 31) == 0) {
      last = (atomic_add_cta_acq_rel(count, 1u) + 1u) % (unsigned)kNW == 0u;
      mbar_arrive(bar);
    }
    last = __shfl_sync(0xffffffffu, last, 0);
    __syncwarp();                        // lane 0's acquire covers the whole warp
    bool ok = true;
    if (!last) ok = mbar_wait(bar, phase, status);
    phase ^= 1u;
    return __all_sync(0xffffffffu, ok);
  }
};

// A plain barrier of the G warps of a team on its own mbarrier, bounded: used
// once per batch, where the warps arrive at about the same time.
struct TeamSync {
  uint64_t* bar;
  uint32_t phase;
  int* status;
  __device__ __forceinline__ bool operator()() {
    __syncwarp();
    if ((threadIdx.x & 31) == 0) mbar_arrive(bar);
    const bool ok = mbar_wait(bar, phase, status);
    phase ^= 1u;
    return __all_sync(0xffffffffu, ok);
  }
};

// ---------------------------------------------------------------------------
// producer
// ---------------------------------------------------------------------------
__device__ inline void produce(const GradRowsArgs& a, const Smem& sm, const StageCfg& c, int64_t rb) {
  const uint64_t pol = policy_evict_first();
  const uint8_t* X = static_cast<const uint8_t*>(a.X);
  const uint8_t* Y = reinterpret_cast<const uint8_t*>(a.y);
  int i = 0;                     // stages issued
  bool ok = true, waited = false;
  int item = blockIdx.x, end = a.nitems;
  if (a.cta_item0) {
    item = a.cta_item0[blockIdx.x];
    end = a.cta_item0[blockIdx.x + 1];
  }
  if (item < end) {
    // Beyond the S stages it can hold, optionally warm L2 with the next rows
    // of the first item while the previous step finishes (a.prefetch_bytes;
    // on the streaming workloads this traffic slowed the previous step's
    // serial tail more than it saved, so the library passes 0).
    const WorkItem it = a.items[item];
    const int64_t r0 = it.row0 + (int64_t)c.S * c.SR;
    int64_t rows = it.rows - (int64_t)c.S * c.SR;
    const int64_t cap = a.prefetch_bytes / rb;
    rows = rows < cap ? rows : cap;
    for (int64_t r = 0; r < rows; r += kPrefetchChunkRows) {
      const int64_t n = rows - r < kPrefetchChunkRows ? rows - r : kPrefetchChunkRows;
      prefetch_l2(X + (r0 + r) * rb, (uint32_t)(n * rb));
    }
  }
  while (ok && item < end) {
    const WorkItem it = a.items[item];
    const int nst = (int)((it.rows + c.SR - 1) / c.SR);
    for (int j = 0; j < nst; ++j) {
      const int s = i % c.S;
      if (i >= c.S && !mbar_wait(&sm.empty[s], ((i / c.S) - 1) & 1, a.status)) { ok = false; break; }
      const int64_t r0 = it.row0 + (int64_t)j * c.SR;
      const int rows = (int)(it.rows - (int64_t)j * c.SR < c.SR ? it.rows - (int64_t)j * c.SR : c.SR);
      const int64_t la = r0 & ~int64_t(3);                      // 16-byte aligned label start
      const uint32_t lbytes = (uint32_t)(((r0 + rows - la) * 4 + 15) & ~int64_t(15));
      StageHdr h;
      h.item = item; h.e = it.e; h.rows = rows; h.lab_off = (int)(r0 - la); h.last = j == nst - 1;
      sm.hdr[s] = h;
      const uint32_t xbytes = (uint32_t)(rows * rb);
      mbar_arrive_expect_tx(&sm.full[s], xbytes + lbytes);
      bulk_g2s_stream(sm.stages + (size_t)s * c.stage_bytes, X + r0 * rb, xbytes, &sm.full[s], pol);
      bulk_g2s(sm.lab + (size_t)s * c.LS, Y + la * 4, lbytes, &sm.full[s]);
      ++i;
    }
    if (!ok) break;
    if (a.cta_item0) { ++item; continue; }
    if (!a.work_ctr) break;
    if (a.pdl && !waited) { grid_dep_wait(); waited = true; }   // counters belong to the previous step until now
    item = (int)gridDim.x + atomicAdd(a.work_ctr, 1);
  }
  if (ok) {   // end marker: a stage without data
    const int s = i % c.S;
    if (i < c.S || mbar_wait(&sm.empty[s], ((i / c.S) - 1) & 1, a.status)) {
      sm.hdr[s].item = -1;
      mbar_arrive(&sm.full[s]);
      ++i;
    }
  }
  if (a.work_ctr) {
    if (a.pdl && !waited) grid_dep_wait();
    // the last producer to finish resets the item counter for the next step
    if (atomicAdd(a.prod_done, 1) == (int)gridDim.x - 1) {
      *a.work_ctr = 0;
      *a.prod_done = 0;
    }
  }
  // no copy may outlive the CTA: wait for the last use of every stage
  for (int s = 0; s < c.S && s < i; ++s) {
    const int last = ((i - 1 - s) / c.S) * c.S + s;
    mbar_wait(&sm.full[s], (last / c.S) & 1, a.status);
  }
}

// ---------------------------------------------------------------------------
// tail warp: per-item reduction and partition counting
// ---------------------------------------------------------------------------
__device__ inline void tail_warp(const GradRowsArgs& a, const Smem& sm, int teams) {
  const int lane = threadIdx.x & 31;
  if (a.tail == 2) derive_plan_warp(a.dec, *sm.plan, lane);   // depends only on the mask
  if (a.pdl) grid_dep_wait();          // partials and counters belong to the previous step until now
  const float* red = reinterpret_cast<const float*>(sm.red);
  for (uint32_t j = 0;; ++j) {
    if (!__all_sync(0xffffffffu, mbar_wait(sm.red_full, j & 1u, a.status))) break;
    const int item = sm.ho->item, e = sm.ho->e;
    if (item < 0) break;
    if (teams > 1) {
      // fixed-order sum of the teams' accumulators into the item's partial
      float4* out = reinterpret_cast<float4*>(a.partials + (size_t)item * a.ld);
      const float4* r4 = reinterpret_cast<const float4*>(red);
      const int64_t L4 = a.ld / 4;
      for (int64_t q = lane; q < L4; q += 32) {
        float4 acc = r4[q];
#pragma unroll
        for (int t = 1; t < kNW; ++t)
          if (t < teams) acc = f4add(acc, r4[(size_t)t * L4 + q]);
        out[q] = acc;
      }
    }
    int commit = -1;
    if (a.tail) {
      __syncwarp();
      if (lane == 0) {
        // release this item's partial (written by this warp, or by the
        // consumers before red_full) and acquire the other items' partials
        const int prev = atomic_add_acq_rel(&a.cnt_e[e], 1);
        if (prev == a.e_item0[e + 1] - a.e_item0[e] - 1) {
          a.cnt_e[e] = 0;              // every item of e has arrived: reset for the next step
          commit = e;
        }
      }
      commit = __shfl_sync(0xffffffffu, commit, 0);
    }
    if (lane == 0) {
      sm.ho->commit = commit;
      mbar_arrive(sm.red_free);
    }
    __syncwarp();
  }
}

// Consumers: commit partition e (all 256 consumer threads), then count it;
// the CTA completing the last partition decodes when tail == 2.
__device__ inline void consumer_commit(const GradRowsArgs& a, const Smem& sm, int e, int tid, ConsumerSync& bar, bool& ok) {
  // the tail warp acquired the other CTAs' partials (atomic + fence) before
  // handing e over through red_free
  commit_block(a.partials, a.ld, a.e_item0[e], a.e_item0[e + 1], a.e_scale[e], a.e_dest + (int64_t)e * a.ndest,
               a.ndest, a.store, tid, kNT);
  if (!bar()) { ok = false; return; }
  if (tid == 0) {
    // release the stores written by the whole CTA (ordered before this by the
    // barrier) and acquire the other committers' stores
    const bool all = atomic_add_acq_rel(a.cnt_all, 1) == a.nE - 1;
    if (all) *a.cnt_all = 0;
    if (all && a.tail == 2) sm.ho->decode = 1;
  }
}

__device__ inline void consumer_decode(const GradRowsArgs& a, const Smem& sm, int tid) {
  if (tid < 32) write_coeffs_warp(a.dec, tid);
  decode_columns<kUserPrefix>(a.dec, *sm.plan, 0, a.dec.P / 4, tid, kNT);
}

// Item end, consumer side, called by all 8 warps at the same stage.
// handover_begin: wait until the tail warp has taken the previous item (so
// red and the handoff slot are free) and run the commit it asked for.
__device__ __forceinline__ bool handover_begin(const GradRowsArgs& a, const Smem& sm, uint32_t ends, ConsumerSync& bar,
                                               bool& ok) {
  if (ends == 0) return true;
  if (!__all_sync(0xffffffffu, mbar_wait(sm.red_free, (ends - 1) & 1u, a.status))) { ok = false; return false; }
  const int ce = sm.ho->commit;          // written by the tail warp before red_free: same for every warp
  if (ce >= 0) {
    consumer_commit(a, sm, ce, (int)threadIdx.x, bar, ok);
    if (!ok) return false;
  }
  return true;
}

// handover_end: publish the item (or -1: no more) to the tail warp.
__device__ __forceinline__ void handover_end(const Smem& sm, int item, int e, uint32_t& ends) {
  if (threadIdx.x == 0) { sm.ho->item = item; sm.ho->e = e; }
  __syncwarp();
  if ((threadIdx.x & 31) == 0) mbar_arrive(sm.red_full);
  ++ends;
}

// After the last item: final handoff, pending commit, decode if this CTA
// committed the last partition.
__device__ __forceinline__ void consumers_finish(const GradRowsArgs& a, const Smem& sm, uint32_t& ends,
                                                 ConsumerSync& bar, bool& ok) {
  if (ok && handover_begin(a, sm, ends, bar, ok)) {
    handover_end(sm, -1, -1, ends);
    if (!bar()) ok = false;              // the decode flag is written before this barrier
    if (ok && sm.ho->decode) consumer_decode(a, sm, (int)threadIdx.x);
  } else if (threadIdx.x < kNT) {
    // release the tail warp even on failure: it stops at item -1 or at its own bound
    handover_end(sm, -1, -1, ends);
  }
}

// ---------------------------------------------------------------------------
// consumers
// ---------------------------------------------------------------------------
// Pairs of fp32 values for the packed FMA (one instruction for two products).
using f32x2 = unsigned long long;
__device__ __forceinline__ f32x2 pack2(float a, float b) {
  f32x2 r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
  return r;
}
__device__ __forceinline__ void unpack2(f32x2 v, float& a, float& b) {
  asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(v));
}
__device__ __forceinline__ f32x2 fma2(f32x2 a, f32x2 b, f32x2 c) {
  f32x2 r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
  return r;
}
__device__ __forceinline__ f32x2 mul2(f32x2 a, f32x2 b) {
  f32x2 r;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ f32x2 add2(f32x2 a, f32x2 b) {
  f32x2 r;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
// a 16-byte chunk of a row as pairs
template <typename T> struct Chunk;
template <> struct Chunk<float> {
  static constexpr int kPairs = 2;
  __device__ __forceinline__ static void widen(const uint4& r, f32x2* x) {
    x[0] = pack2(__uint_as_float(r.x), __uint_as_float(r.y));
    x[1] = pack2(__uint_as_float(r.z), __uint_as_float(r.w));
  }
};
template <> struct Chunk<uint16_t> {
  static constexpr int kPairs = 4;
  __device__ __forceinline__ static void widen(const uint4& r, f32x2* x) {
    const uint32_t w[4] = {r.x, r.y, r.z, r.w};
#pragma unroll
    for (int i = 0; i < 4; ++i) x[i] = pack2(__uint_as_float(w[i] << 16), __uint_as_float(w[i] & 0xffff0000u));
  }
};

// Sums v[0..N) over the LPR lanes that share a row, all together: each step
// halves the values a lane holds while two are left, then the lanes.  Returns
// the total number row_of_lane<N, LPR>(l).
template <int N, int LPR>
__device__ __forceinline__ float reduce_rows(float (&v)[N], int l) {
  int w = LPR / 2;
#pragma unroll
  for (int n = N; n > 1; n /= 2, w /= 2) {
    const bool up = (l & w) != 0;
#pragma unroll
    for (int k = 0; k < N / 2; ++k) {
      if (k < n / 2) {
        const float send = up ? v[k] : v[k + n / 2], keep = up ? v[k + n / 2] : v[k];
        v[k] = keep + __shfl_xor_sync(0xffffffffu, send, w);
      }
    }
  }
#pragma unroll
  for (; w > 0; w /= 2) v[0] += __shfl_xor_sync(0xffffffffu, v[0], w);
  return v[0];
}
template <int N, int LPR>
__device__ __forceinline__ int row_of_lane(int l) { return l / (LPR / N); }

// Whether chunk j of a lane lies inside the row.  Only the last j can lie past it
// (the last two where NCH is rounded up to an even count, beyond 8), and none
// if FULL: the longest rows' own variants, where the check on two chunks cost
// 64 x 2048 x 16384 2.5 % (1256 us per step against 1225).
template <int G, int LPR, int NCH, bool FULL>
__device__ __forceinline__ bool chunk_in(int j, int g, int l, int nv) {
  return FULL || j < NCH - (NCH > 8 ? 2 : 1) || (j * G + g) * LPR + l < nv;
}

// One team's batch of RR x SUB rows from row r0 of the stage (rows: its row count).
template <typename T, int G, int LPR, int NCH, int RR, bool FULL, class Sync>
__device__ __forceinline__ bool consume_batch(const GradRowsArgs& a, const uint8_t* st, const float* lab, float* xd,
                                              int r0, int rows, int rb, int nv, int g, int lane, const f32x2* wr,
                                              f32x2* acc, Sync& sync) {
  constexpr int H = Chunk<T>::kPairs, SUB = 32 / LPR;
  constexpr int C = RR >= 4 ? 1 : RR == 2 ? 2 : H;   // chains of pair sums per row
  const int sub = lane / LPR, l = lane % LPR;
  // rows of this lane: r0 + i SUB + sub; only a single-row batch may run past the stage
  const bool live = RR > 1 || SUB == 1 || r0 + sub < rows;
  const uint8_t* p0 = st + (r0 + sub) * rb + (g * LPR + l) * 16;
  auto load = [&](int i, int j) -> uint4 {
    if (chunk_in<G, LPR, NCH, FULL>(j, g, l, nv) && live)
      return *reinterpret_cast<const uint4*>(p0 + i * SUB * rb + j * (G * LPR * 16));
    return make_uint4(0u, 0u, 0u, 0u);
  };
  // the batch stays in registers, as stored, for the update below where w, the
  // accumulator and the batch fit about 128 of them; else it is read again
  // (holding only part of it cost more in spills than it saved in reads)
  constexpr int HN = 4 * RR * NCH + 4 * H * NCH <= 128 ? NCH : 0;
  uint4 raw[RR][HN > 0 ? HN : 1];
  const int own = row_of_lane<RR, LPR>(l);
  const float y = live ? lab[r0 + own * SUB + sub] : 0.f;
  f32x2 part[RR][C];
#pragma unroll
  for (int i = 0; i < RR; ++i)
#pragma unroll
    for (int q = 0; q < C; ++q) part[i][q] = 0;
#pragma unroll
  for (int j = 0; j < NCH; ++j)
#pragma unroll
    for (int i = 0; i < RR; ++i) {
      const uint4 v4 = load(i, j);
      if (j < HN) raw[i][j < HN ? j : 0] = v4;
      f32x2 x[H];
      Chunk<T>::widen(v4, x);
#pragma unroll
      for (int v = 0; v < H; ++v) part[i][v % C] = fma2(x[v], wr[j * H + v], part[i][v % C]);
    }
  float dot[RR];
#pragma unroll
  for (int i = 0; i < RR; ++i) {
    dot[i] = 0.f;
#pragma unroll
    for (int q = 0; q < C; ++q) {
      float lo, hi;
      unpack2(part[i][q], lo, hi);
      dot[i] += lo + hi;
    }
  }
  // held chunks are widened again below, not held wide; the others read again
#pragma unroll
  for (int i = 0; i < RR; ++i)
#pragma unroll
    for (int j = 0; j < HN; ++j)
      asm volatile("" : "+r"(raw[i][j].x), "+r"(raw[i][j].y), "+r"(raw[i][j].z), "+r"(raw[i][j].w));
  if (HN < NCH) asm volatile("" ::: "memory");
  float z = reduce_rows<RR, LPR>(dot, l);
  if constexpr (G > 1) {
    if (l % (LPR / RR) == 0) xd[own * G + g] = z;
    if (!sync()) return false;
    float q[G];
#pragma unroll
    for (int k = 0; k < G; k += G < 4 ? G : 4) {
      if constexpr (G == 2) {
        const float2 v = *reinterpret_cast<const float2*>(xd + own * G);
        q[0] = v.x; q[1] = v.y;
      } else {
        const float4 v = *reinterpret_cast<const float4*>(xd + own * G + k);
        q[k] = v.x; q[k + 1] = v.y; q[k + 2] = v.z; q[k + 3] = v.w;
      }
    }
#pragma unroll
    for (int n = G / 2; n > 0; n /= 2)
#pragma unroll
      for (int k = 0; k < n; ++k) q[k] += q[k + n];
    z = q[0];
  }
  const float res = live ? residual(a.loss, z, y) : 0.f;
  f32x2 r[RR];
#pragma unroll
  for (int i = 0; i < RR; ++i) {
    const float ri = RR > 1 ? __shfl_sync(0xffffffffu, res, sub * LPR + i * (LPR / RR)) : res;
    r[i] = pack2(ri, ri);
  }
  // the batch's rows are summed first, then added: a chain of rows / RR additions
  // (8 x 8192 x 1024: error against fp64 1.1e-7 -> 0.99e-7, 1.0e-7 with one row at a time)
#pragma unroll
  for (int j = 0; j < NCH; ++j) {
    f32x2 t[H];
#pragma unroll
    for (int i = 0; i < RR; ++i) {
      f32x2 x[H];
      if (j < HN) Chunk<T>::widen(raw[i][j < HN ? j : 0], x);
      else Chunk<T>::widen(load(i, j), x);
#pragma unroll
      for (int v = 0; v < H; ++v) {
        if (RR == 1) acc[j * H + v] = fma2(r[i], x[v], acc[j * H + v]);
        else t[v] = i == 0 ? mul2(r[i], x[v]) : fma2(r[i], x[v], t[v]);
      }
    }
    if (RR > 1) {
#pragma unroll
      for (int v = 0; v < H; ++v) acc[j * H + v] = add2(acc[j * H + v], t[v]);
    }
  }
  return true;
}

template <typename T, int G, int LPR, int NCH, int R, bool FULL>
__device__ void consume_rows(const GradRowsArgs& a, const Smem& sm, const StageCfg& c, int rb) {
  constexpr int VEC = 16 / (int)sizeof(T), H = VEC / 2, SUB = 32 / LPR, TEAMS = kNW / G, U = R * SUB, E2 = NCH * H;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int team = warp / G, g = warp % G, sub = lane / LPR, l = lane % LPR;
  const int nv = (int)(a.ld / VEC);
  ConsumerSync bar{sm.sync, &sm.ho->sync_count, 0u, a.status};
  TeamSync sync{sm.team_sync + team, 0u, a.status};
  if (a.pdl) grid_dep_wait();                       // w is the previous step's output
  f32x2 wr[E2], acc[E2];
#pragma unroll
  for (int j = 0; j < NCH; ++j) {
    const bool in = chunk_in<G, LPR, NCH, FULL>(j, g, l, nv);
    const float4* w4 = reinterpret_cast<const float4*>(a.w) + ((j * G + g) * LPR + l) * (VEC / 4);
#pragma unroll
    for (int q = 0; q < VEC / 4; ++q) {
      const float4 v = in ? w4[q] : make_float4(0.f, 0.f, 0.f, 0.f);
      wr[j * H + 2 * q] = pack2(v.x, v.y);
      wr[j * H + 2 * q + 1] = pack2(v.z, v.w);
      acc[j * H + 2 * q] = acc[j * H + 2 * q + 1] = 0;
    }
  }
  float* red = reinterpret_cast<float*>(sm.red);
  float* xd = sm.xdot + team * (2 * R * G);         // two buffers: a batch's reads and the next one's writes
  uint32_t ends = 0;
  int turn = 0, xbuf = 0;                           // team that takes the stage's first batch
  int s = 0;
  uint32_t phase = 0;
  bool ok = true;
  while (ok) {
    if (!__all_sync(0xffffffffu, mbar_wait(&sm.full[s], phase, a.status))) { ok = false; break; }
    const StageHdr h = sm.hdr[s];
    if (h.item < 0) break;
    const uint8_t* st = sm.stages + (size_t)s * c.stage_bytes;
    const float* lab = sm.lab + (size_t)s * c.LS + h.lab_off;
    const int nb = (h.rows + U - 1) / U;
    int b = team - turn;
    if (b < 0) b += TEAMS;
    for (; b < nb && ok; b += TEAMS) {
      const int r0 = b * U;
      if (r0 + U <= h.rows) {
        ok = consume_batch<T, G, LPR, NCH, R, FULL>(a, st, lab, xd + xbuf * (R * G), r0, h.rows, rb, nv, g, lane, wr, acc, sync);
        xbuf ^= 1;
      } else {
        for (int r = r0; r < h.rows && ok; r += SUB) {
          ok = consume_batch<T, G, LPR, NCH, 1, FULL>(a, st, lab, xd + xbuf * (R * G), r, h.rows, rb, nv, g, lane, wr, acc, sync);
          xbuf ^= 1;
        }
      }
    }
    if (!ok) break;
    __syncwarp();
    if (lane == 0) mbar_arrive(&sm.empty[s]);
    turn = (turn + nb) % TEAMS;
    if (++s == c.S) { s = 0; phase ^= 1u; }
    if (h.last) {
      if (!handover_begin(a, sm, ends, bar, ok)) break;
      // one team: straight to the item's partial; more: the tail warp adds the teams' sums
      float4* out = reinterpret_cast<float4*>(TEAMS == 1 ? a.partials + (size_t)h.item * a.ld : red + (size_t)team * a.ld);
#pragma unroll
      for (int j = 0; j < NCH; ++j) {
#pragma unroll
        for (int q = 0; q < VEC / 4; ++q) {
          float4 v;
          unpack2(acc[j * H + 2 * q], v.x, v.y);
          unpack2(acc[j * H + 2 * q + 1], v.z, v.w);
          if constexpr (SUB > 1) {
            // the warp's row groups hold sums of the same columns
#pragma unroll
            for (int w = LPR; w < 32; w *= 2)
              v = f4add(v, make_float4(__shfl_xor_sync(0xffffffffu, v.x, w), __shfl_xor_sync(0xffffffffu, v.y, w),
                                       __shfl_xor_sync(0xffffffffu, v.z, w), __shfl_xor_sync(0xffffffffu, v.w, w)));
          }
          if (sub == 0 && chunk_in<G, LPR, NCH, FULL>(j, g, l, nv)) out[((j * G + g) * LPR + l) * (VEC / 4) + q] = v;
          acc[j * H + 2 * q] = acc[j * H + 2 * q + 1] = 0;
        }
      }
      handover_end(sm, h.item, h.e, ends);
    }
  }
  consumers_finish(a, sm, ends, bar, ok);
  if (!ok) atomicOr(a.status, kErrWaitTimeout);
}

template <typename T, int G, int LPR, int NCH, int R, bool FULL>
__global__ void __launch_bounds__(kThreads, 1) grad_rows_kernel(GradRowsArgs a, StageCfg c) {
  extern __shared__ __align__(128) uint8_t smem[];
  const Smem sm = carve(smem, c);
  const int64_t rb = a.ld * (int64_t)sizeof(T);
  if (threadIdx.x == 0) {
    for (int s = 0; s < c.S; ++s) {
      mbar_init(&sm.full[s], 1);
      mbar_init(&sm.empty[s], kNW);
    }
    mbar_init(sm.sync, kNW);
    mbar_init(sm.red_full, kNW);
    mbar_init(sm.red_free, 1);
    for (int t = 0; t < kMaxTeams; ++t) mbar_init(sm.team_sync + t, G);
    sm.ho->item = -1;
    sm.ho->e = -1;
    sm.ho->commit = -1;
    sm.ho->decode = 0;
    sm.ho->sync_count = 0;
    fence_mbar_init();
    grid_dep_launch();
  }
  __syncthreads();
  const int warp = threadIdx.x >> 5;
  if (warp == kTailWarp) {
    tail_warp(a, sm, kNW / G);
  } else if (threadIdx.x >= kNT) {
    if (threadIdx.x == kProducer) produce(a, sm, c, rb);
  } else {
    consume_rows<T, G, LPR, NCH, R, FULL>(a, sm, c, (int)rb);
  }
  __syncthreads();
}

// Kernel of one variant (grad_rows_f32.cu, grad_rows_bf16.cu), nullptr if unknown.
using GradRowsKernel = void (*)(GradRowsArgs, StageCfg);
GradRowsKernel grad_rows_kernel_f32(int g, int lpr, int nch, int r, bool full);
GradRowsKernel grad_rows_kernel_bf16(int g, int lpr, int nch, int r, bool full);

template <typename T>
GradRowsKernel pick_rows_kernel(int g, int lpr, int nch, int r, bool full) {
#define PGC_ROWS(G, L, N, R) \
  if (g == G && lpr == L && nch == N && r == R) return grad_rows_kernel<T, G, L, N, R, false>;
  if (full && g == 8 && nch > 8) {
    switch (nch) {
      case 10: return grad_rows_kernel<T, 8, 32, 10, 1, true>;
      case 12: return grad_rows_kernel<T, 8, 32, 12, 1, true>;
      case 14: return grad_rows_kernel<T, 8, 32, 14, 1, true>;
      case 16: return grad_rows_kernel<T, 8, 32, 16, 1, true>;
      default: return nullptr;
    }
  }
  PGC_ROWS(1, 8, 1, 4) PGC_ROWS(1, 16, 1, 4) PGC_ROWS(1, 32, 1, 4) PGC_ROWS(1, 32, 2, 4)
  PGC_ROWS(1, 8, 1, 8) PGC_ROWS(1, 16, 1, 8) PGC_ROWS(1, 32, 1, 8) PGC_ROWS(1, 32, 2, 8)
  PGC_ROWS(1, 32, 3, 4) PGC_ROWS(1, 32, 4, 4) PGC_ROWS(2, 32, 3, 4) PGC_ROWS(2, 32, 4, 4)
  if constexpr (sizeof(T) == 4) {
    PGC_ROWS(2, 32, 5, 2) PGC_ROWS(2, 32, 6, 2) PGC_ROWS(2, 32, 7, 2) PGC_ROWS(2, 32, 8, 2)
  } else {
    PGC_ROWS(2, 32, 5, 4) PGC_ROWS(4, 32, 3, 4) PGC_ROWS(4, 32, 4, 4)
  }
  PGC_ROWS(4, 32, 5, 4) PGC_ROWS(4, 32, 6, 4) PGC_ROWS(8, 32, 4, 4)
  PGC_ROWS(8, 32, 5, 2) PGC_ROWS(8, 32, 6, 2) PGC_ROWS(8, 32, 7, 2) PGC_ROWS(8, 32, 8, 2)
  PGC_ROWS(8, 32, 10, 1) PGC_ROWS(8, 32, 12, 1) PGC_ROWS(8, 32, 14, 1) PGC_ROWS(8, 32, 16, 1)
#undef PGC_ROWS
  return nullptr;
}

}  // namespace pgc
