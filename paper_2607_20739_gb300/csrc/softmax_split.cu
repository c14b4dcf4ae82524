// Softmax gradient in single precision on the tensor cores, up to 128 classes
// (§III with f = log sum_k exp(w_k.x) - w_y.x): fp32 features, and bf16
// features outside the few-class and many-class kernels.  Two kernels:
//
//   logits    Z = X W^T, R = softmax(Z) - onehot(y)
//   gradient  G_e = R_e^T X_e for every evaluated partition e
//
// The CUDA-core kernels that did this ran at 11-17 TFLOP/s; the tensor cores
// take bf16.  So operands are cut into bf16 parts and multiplied by tcgen05.mma
// (kind::f16, fp32 accumulators).  W and R, rounded to nearest, are three parts
// each, w = w1 + w2 + w3 up to 2^-27 |w|; an fp32 x is cut into three 8-bit
// pieces, x = x1 + x2 + x3 exactly; a bf16 x is x1.  The products kept are
// x1 (w1 w2 w3), x2 (w1 w2), x3 w1: what is left out is below 2^-24 |x w| and of
// either sign.  The parts of W (R) stand side by side along the MMA's N axis,
// 3 Kp columns (Kp = K rounded up to 16).  x1 w1 has an accumulator of its own;
// the corrections have two, x1 w2 + x2 w1 (about 2^-8 of it) and
// x1 w3 + x2 w2 + x3 w1 (2^-16), added in fp32 at the end, smallest first.
//
// The tensor core cuts a sum off (it does not round it) at every K step, so a
// long sum drifts: one leading accumulator over all 4096 rows (3072 features)
// left the gradient 4.7e-6 off, 9.2e-7 with the CUDA-core sums.  So the
// leading accumulator is emptied into fp32 registers every two stages (128
// products; 2.0e-7), from 33 classes on every four (3.2e-7; 6.0e-7 with eight),
// alternating with a second one where tensor memory has room.
//
// Measured, us per step, before (three CUDA-core kernels) and with this file:
// 12 partitions of 4096 x 3072 bf16, 100 classes: 3561 -> 222; 8 of 4096 x 784
// fp32, 10 classes: 915 -> 60.  fp32 with 97 to 128 classes spills registers in the
// epilogue's sums (logits 456 bytes per thread, gradient 324) and gains less: 12 of 4096 x 3072
// 3540 -> 438 (97 classes) to 454 (128), 390 with 96; 4 of 300 x 700 131 -> 47 to 54.
// X is read once per kernel (twice per step).  The
// instructions of the single-thread roles bound an earlier form (282 and 102,
// with ring positions divided out and descriptors rebuilt for every MMA).
//
// Both kernels are one GEMM skeleton (kMode selects): a cluster of one or two
// CTAs takes units of h rows of X per CTA (logits; h <= 128, the MMA's M, chosen so
// that every SM streams about the same rows) or of 128 features per CTA
// (gradient) and streams its A tiles, 64 columns (rows) a stage, through a ring of
// TMA stages, with the B tile (W: 3 Kp x 64, K-major; R: 64 rows x 3 Kp,
// MN-major).  From 33 classes on, where B outweighs A, two CTAs share it: each
// loads half and multicasts it.  X is read through one tensor map per
// partition, so that rows past the partition read as zero and never as the next
// partition's.
//   bf16 X: the MMA reads A from the stage (K-major; gradient: MN-major).
//   fp32 X: eight (four) warps cut a stage's A tile into parts and put them into
//           tensor memory (one lane per row, or per feature), 32 K elements
//           (48 columns) at a time, in a ring of up to four buffers.
// Four epilogue warps add the accumulators and form R (one row per
// thread) as its three parts, or write the gradient's columns (one feature per
// thread) into the partition's partial or, if one unit holds the whole
// partition, times 1/m_e straight into the stores.
//
// The same logits with a third epilogue give the loss F (any K): a unit is a
// row tile and a block of up to 128 classes (X comes from L2 for all but one of a
// tile's blocks); every row's max and sum of exp per block go to memory and a
// small kernel combines them.  Before, the tiled CUDA-core logits
// went through memory, and one more kernel reduced them: a step with its loss on
// 8 partitions of about 600 x 1500 bf16, 300 classes, took 473 us; now 140
// (184 against 144 with the class blocks of a tile one after the other in one
// cluster: 20 of 76 clusters busy).
//
// Every wait is bounded; on a failure the kernel flags the status word, all
// roles wind down, and TMEM is released after the MMAs issued so far.
#include <cuda.h>
#include <cudaTypedefs.h>

#include <cstring>

#include "pgc.h"
#include "tc_common.cuh"

namespace pgc {

namespace {

constexpr int kSM = 128;                       // rows (features) per CTA
constexpr int kSK = 64;                        // K elements per stage
constexpr uint32_t kSTmem = 512;
constexpr uint32_t kSBufCols = 48;             // A buffer: 32 K elements x 3 parts, two per column
constexpr int kSMaxBuf = 4;
constexpr int kSMaxStages = 8;
constexpr size_t kSSmemBudget = 200 * 1024;

// Warps: producer, MMA, four epilogue warps; fp32 features: four warps per half
// of a stage that cut it into parts, or four in all where the epilogue's sums
// need the registers.
template <typename T, int NCH> constexpr int split_conv() { return sizeof(T) == 2 ? 0 : NCH <= 2 ? 8 : 4; }
template <typename T, int NCH> constexpr int split_threads() { return 192 + 32 * split_conv<T, NCH>(); }
template <typename T> constexpr uint32_t split_a_bytes() { return kSM * kSK * sizeof(T); }

// Tensor memory, A buffers from the top.  Up to 32 classes (stack): two
// accumulators of 3 Kp columns, leading products and corrections side by side, so
// one MMA multiplies x1 with all parts; more: nmain accumulators of the leading
// products (Kp columns), ncorr of the corrections (2 Kp).
struct SplitGeom {
  int stages, nmain, ncorr, nbuf;
  bool stack;
  uint32_t b_bytes;                            // B tile, a multiple of 1 KB
};
// nb: 3 Kp (logits: rows of W) or 3 Kp rounded up to 64 (gradient: columns of R)
__host__ __device__ inline SplitGeom split_geom(int esize, int Kp, int nb) {
  SplitGeom g;
  g.b_bytes = (uint32_t)nb * 128;
  const uint32_t stage = (uint32_t)(kSM * kSK) * (uint32_t)esize + g.b_bytes;
  g.stages = (int)(kSSmemBudget / stage);
  if (g.stages > kSMaxStages) g.stages = kSMaxStages;
  const int room = (int)kSTmem - (esize == 4 ? 2 * (int)kSBufCols : 0);
  g.stack = Kp <= 32;
  g.nmain = 4 * Kp <= room ? 2 : 1;
  g.ncorr = 6 * Kp <= room ? 2 : 1;
  g.nbuf = esize == 4 ? ((int)kSTmem - (g.nmain + 2 * g.ncorr) * Kp) / (int)kSBufCols : 0;
  if (g.nbuf > kSMaxBuf) g.nbuf = kSMaxBuf;
  return g;
}

// 16 columns of this thread's TMEM lane added to v
__device__ __forceinline__ void tmem_add16(uint32_t taddr, float* v) {
  uint32_t r[16];
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
        "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
      : "r"(taddr));
  tmem_ld_wait();
#pragma unroll
  for (int c = 0; c < 16; ++c) v[c] += __uint_as_float(r[c]);
}
__device__ __forceinline__ void tmem_st16(uint32_t taddr, const uint32_t (&r)[16]) {
  asm volatile(
      "tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16};" ::"r"(
          taddr),
      "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]), "r"(r[8]), "r"(r[9]),
      "r"(r[10]), "r"(r[11]), "r"(r[12]), "r"(r[13]), "r"(r[14]), "r"(r[15])
      : "memory");
}
__device__ __forceinline__ void tmem_st_wait() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }

// A from tensor memory (K-major), B from shared memory
__device__ __forceinline__ void umma_bf16_ta(uint32_t tmem_d, uint32_t tmem_a, uint64_t db, uint32_t idesc,
                                             uint32_t acc) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n\t}" ::"r"(tmem_d),
      "r"(tmem_a), "l"(db), "r"(idesc), "r"(acc)
      : "memory");
}

// two fp32 values -> their high halves packed (truncation), the remainders left in a, b
__device__ __forceinline__ uint32_t cut_pair(float& a, float& b) {
  const uint32_t ua = __float_as_uint(a), ub = __float_as_uint(b);
  const uint32_t pk = __byte_perm(ua, ub, 0x7632);
  a -= __uint_as_float(ua & 0xffff0000u);
  b -= __uint_as_float(ub & 0xffff0000u);
  return pk;
}

// eight fp32 values -> their three bf16 parts (round to nearest)
__device__ __forceinline__ void split8(const float* v, uint4& p1, uint4& p2, uint4& p3) {
  uint32_t a[4], b[4], c[4];
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    float x = v[2 * j], y = v[2 * j + 1];
    __nv_bfloat162 h = __floats2bfloat162_rn(x, y);
    a[j] = *reinterpret_cast<uint32_t*>(&h);
    x -= __low2float(h); y -= __high2float(h);
    h = __floats2bfloat162_rn(x, y);
    b[j] = *reinterpret_cast<uint32_t*>(&h);
    x -= __low2float(h); y -= __high2float(h);
    h = __floats2bfloat162_rn(x, y);
    c[j] = *reinterpret_cast<uint32_t*>(&h);
  }
  p1 = make_uint4(a[0], a[1], a[2], a[3]);
  p2 = make_uint4(b[0], b[1], b[2], b[3]);
  p3 = make_uint4(c[0], c[1], c[2], c[3]);
}

}  // namespace

template <int kMode, typename T, int NCH>
__global__ void __launch_bounds__(split_threads<T, NCH>(), 1)
split_gemm_kernel(const __grid_constant__ CUtensorMap tmB, SplitArgs p) {
  extern __shared__ __align__(1024) uint8_t smem_raw[];
  __shared__ uint64_t full[kSMaxStages], empty[kSMaxStages];
  __shared__ uint64_t acc_full[2], acc_empty[2], corr_empty[2], a_full[kSMaxBuf], a_empty[kSMaxBuf], drained;
  __shared__ uint32_t tmem_slot;
  constexpr bool kF32 = sizeof(T) == 4, kGrad = kMode == kSplitGrad;
  constexpr uint32_t kABytes = split_a_bytes<T>();
  uint8_t* sm = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  const int Kp = p.Kp;
  const int nb = kGrad ? p.C3 : 3 * Kp;
  const SplitGeom G = split_geom((int)sizeof(T), Kp, nb);
  const int S = G.stages;
  const uint32_t stage_bytes = kABytes + G.b_bytes;

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int rank = (int)cluster_rank();
  constexpr bool kStack = NCH == 1;        // split_geom's stack
  constexpr int CL = kStack ? 1 : 2;       // CTAs of the cluster (split_cluster)
  constexpr uint16_t kBoth = 0x3;
  if (threadIdx.x == 0) {
    for (int s = 0; s < S; ++s) {
      mbar_init(&full[s], 1);
      mbar_init(&empty[s], CL);          // every CTA's MMAs have read the stage
    }
    for (int a = 0; a < 2; ++a) {
      mbar_init(&acc_full[a], 1);
      mbar_init(&acc_empty[a], 4);
      mbar_init(&corr_empty[a], 4);
    }
    for (int a = 0; a < kSMaxBuf; ++a) {
      mbar_init(&a_full[a], 4);
      mbar_init(&a_empty[a], 1);
    }
    mbar_init(&drained, 1);
    fence_mbar_init();
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_slot)),
                 "r"(kSTmem)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  __syncthreads();
  tc_fence_before();
  cluster_sync_all();                    // the peer's barriers exist before any multicast
  tc_fence_after();
  const uint32_t tmem = tmem_slot;
  if (threadIdx.x == 0) grid_dep_launch();
  grid_dep_wait();                       // W (R) is the previous kernel's output

  const int ncl = (int)gridDim.x / CL, cid = (int)blockIdx.x / CL;
  // loss: unit = class block e of a row tile, the blocks of a tile side by side
  const int my_units = p.nunits > cid ? (p.nunits - cid + ncl - 1) / ncl : 0;
  auto unit = [&](int i) {
    const int n = cid + i * ncl;
    if constexpr (kMode == kSplitLoss) return SplitUnit{n % p.ncb, 0, 0, n / p.ncb * CL * p.h, (int)p.rows, 0, 0, 0};
    else return p.units[n];
  };
  // The producer and the MMA issuer run as whole, converged warps (elect_one): 8 to
  // 11 % of a step with fp32 features (8 x 4096 x 784, K = 10: 67.2 us against 61.8;
  // 8 x 2000 x 2000, K = 20: 126 against 112), 2 to 3 % in bf16 up to 64 classes.
  // Not so for more classes in bf16, where one thread each is faster (12 x 4096
  // x 3072, K = 100: 226 against 233).
  constexpr bool kWhole = kF32 || NCH <= 2;
  auto one = [] { return kWhole ? elect_one() : true; };
  auto wait = [&](uint64_t* bar, uint32_t parity) {
    return kWhole ? mbar_wait_warp(bar, parity, p.status) : mbar_wait(bar, parity, p.status);
  };
  auto join = [] { if (kWhole) __syncwarp(); };
  auto uniform = [](const SplitUnit& u) {    // known to be warp-uniform to the compiler
    if (!kWhole) return u;
    auto sh = [](int v) { return __shfl_sync(0xffffffffu, v, 0); };
    return SplitUnit{sh(u.e), sh(u.map), sh(u.x), sh(u.r0), sh(u.rows), sh(u.z0), sh(u.item), 0};
  };
  auto blocks_of = [&](const SplitUnit& u) { return kGrad ? (u.rows + kSK - 1) / kSK : p.nkb; };

  if (warp == 0 && (kWhole || lane == 0)) {
    // ---- producer ----------------------------------------------------------
    // (ring positions and phases are counted, not divided out: the single-thread
    // roles' instructions are on every stage's critical path)
    const uint32_t a_bytes = kGrad ? kABytes : (uint32_t)p.h * kSK * (uint32_t)sizeof(T);
    const int part = 3 * Kp / CL;
    int it = 0, s = 0;
    uint32_t ph = 1;                                         // phase of the empty barrier: passes at once in the first round
    bool ok = true;
    for (int i = 0; i < my_units && ok; ++i) {
      const SplitUnit u = uniform(unit(i));
      const CUtensorMap* tmA = reinterpret_cast<const CUtensorMap*>(p.tmX) + u.map;
      const int nkb = blocks_of(u);
      const int r0 = u.r0 + (kGrad ? 0 : rank * p.h), f0 = (CL * u.x + rank) * kSM;
      const int wrow = (kMode == kSplitLoss ? u.e * 3 * Kp : 0) + rank * part;
      for (int kb = 0; kb < nkb; ++kb, ++it) {
        if (it >= S && !wait(&empty[s], ph)) { ok = false; break; }
        uint8_t* a_dst = sm + (size_t)s * stage_bytes;
        uint8_t* b_dst = a_dst + kABytes;
        if (one()) {
          mbar_arrive_expect_tx(&full[s], a_bytes + G.b_bytes);
          if constexpr (!kGrad) {
            tma_load_2d(a_dst, tmA, kb * kSK, r0, &full[s]);
            if (kF32) tma_load_2d(a_dst + kABytes / 2, tmA, kb * kSK + 32, r0, &full[s]);
            if (CL == 1) tma_load_2d(b_dst, &tmB, kb * kSK, wrow, &full[s]);
            else tma_load_2d_mc(b_dst + (size_t)rank * part * 128, &tmB, kb * kSK, wrow, &full[s], kBoth);
          } else {
            const int r = r0 + kb * kSK;
            tma_load_2d(a_dst, tmA, f0, r, &full[s]);
            if (!kF32) tma_load_2d(a_dst + kABytes / 2, tmA, f0 + 64, r, &full[s]);
            for (int q = 0; q < nb / 64; ++q) {
              if (CL == 1) tma_load_2d(b_dst + q * 8192, &tmB, q * 64, u.z0 + r, &full[s]);
              else tma_load_2d_mc(b_dst + q * 8192 + rank * 4096, &tmB, q * 64, u.z0 + r + rank * 32, &full[s], kBoth);
            }
          }
        }
        join();
        if (++s == S) { s = 0; ph ^= 1u; }
      }
    }
    // no copy may outlive the CTA
    for (int q = 0; q < S && q < it; ++q) {
      const int last = ((it - 1 - q) / S) * S + q;
      wait(&full[q], (last / S) & 1);
    }
  } else if (warp == 1 && (kWhole || lane == 0)) {
    // ---- MMA issuer --------------------------------------------------------
    constexpr uint32_t idesc0 = idesc_bf16_f32(kSM, 0, kGrad && !kF32, kGrad);
    auto idesc = [&](int N) { return idesc0 | ((uint32_t)(N >> 3) << 17); };
    const uint32_t id1 = idesc(Kp), id2 = idesc(2 * Kp), id3 = idesc(kStack ? 3 * Kp : Kp);
    // x1 times parts 2 and 3: columns Kp .. 3 Kp of B.  MN-major, an operand that
    // starts inside a 64-column block must end there: two MMAs if it does not.
    const int na = kGrad && Kp % 64 != 0 && 2 * Kp > 64 - Kp % 64 ? 64 - Kp % 64 : 2 * Kp, nrest = 2 * Kp - na;
    const uint32_t ida = idesc(na), idr = idesc(nrest);
    // descriptors of stage 0; a stage further is stage_bytes / 16, a K step (16)
    // 32 bytes along the swizzled row (K-major) or two 8-row groups (MN-major)
    auto boff = [&](int n) {                                 // column n of B, in 16-byte units
      return kGrad ? (uint32_t)(n / 64) * 512u + (uint32_t)(n % 64) / 8u : (uint32_t)n * 8u;
    };
    constexpr uint32_t kStepA = kGrad ? 128 : 2, kStepB = kGrad ? 128 : 2;
    const uint32_t base = smem_u32(sm);
    const uint64_t da0 = smem_desc_sw128(base, kGrad ? 8192 : 16, 1024);
    const uint64_t db0 = smem_desc_sw128(base + kABytes, kGrad ? 8192 : 16, 1024);
    const uint32_t bK = boff(Kp), bR = boff(Kp + na), stage16 = stage_bytes / 16;
    int s = 0, ab = 0, acc = 0, cor = 0, left = 0;           // left: K blocks until the leading accumulator is handed over
    uint32_t ph = 0, ph_a = 0, ph_acc = 1, ph_cor = 1;       // phases; those of freed accumulators pass at once in the first round
    int used = 0;                                            // accumulators taken so far (up to 2)
    auto hand_over = [&](int stage, int a, bool done) {      // the stage is read, the accumulator complete
      if (CL == 1) umma_commit(&empty[stage]);
      else umma_commit_mc(&empty[stage], kBoth);
      if (done) umma_commit(&acc_full[a]);
    };
    bool ok = true;
    for (int i = 0; i < my_units && ok; ++i) {
      const SplitUnit u = uniform(unit(i));
      const int nkb = blocks_of(u);
      left = 0;
      uint32_t d = 0;
      const uint32_t dc = tmem + (uint32_t)((G.nmain + 2 * cor) * Kp);
      if (!kStack) {
        if (i >= G.ncorr && !wait(&corr_empty[cor], ph_cor)) { ok = false; break; }
        if (++cor == G.ncorr) { cor = 0; ph_cor ^= 1u; }
      }
      for (int kb = 0; kb < nkb && ok; ++kb) {
        bool fresh = false;
        if (left == 0) {                                     // the next leading accumulator, drained
          if (used >= G.nmain && !wait(&acc_empty[acc], ph_acc)) { ok = false; break; }
          if (used < G.nmain) ++used;
          left = p.chunk;
          fresh = true;
          d = tmem + (uint32_t)(acc * (kStack ? 3 * Kp : Kp));
          tc_fence_after();
        }
        if (!wait(&full[s], ph)) { ok = false; break; }
        const uint64_t da = da0 + (uint32_t)s * stage16, db = db0 + (uint32_t)s * stage16;
        const bool done = left == 1 || kb == nkb - 1;        // the accumulator is handed over after this block
        if constexpr (!kF32) {
          tc_fence_after();
          if (one()) {
#pragma unroll
            for (int kk = 0; kk < kSK / 16; ++kk) {
              const uint64_t dak = da + kk * kStepA, dbk = db + kk * kStepB;
              const uint32_t in1 = fresh && kk == 0 ? 0u : 1u;
              if constexpr (kStack) {
                umma_bf16(d, dak, dbk, id3, in1);
              } else {
                const uint32_t in2 = kb == 0 && kk == 0 ? 0u : 1u;
                umma_bf16(d, dak, dbk, id1, in1);
                umma_bf16(dc, dak, dbk + bK, ida, in2);
                if (nrest) umma_bf16(dc + (uint32_t)na, dak, dbk + bR, idr, in2);
              }
            }
            hand_over(s, acc, done);
          }
        } else {
#pragma unroll
          for (int h = 0; h < 2; ++h) {
            if (!ok) break;
            if (!wait(&a_full[ab], ph_a)) { ok = false; break; }
            tc_fence_after();
            const uint32_t ta = tmem + kSTmem - (uint32_t)(ab + 1) * kSBufCols;
            if (one()) {
#pragma unroll
              for (int k2 = 0; k2 < 2; ++k2) {
                const int kk = h * 2 + k2;
                const uint32_t ak = ta + (uint32_t)(k2 * 8);
                const uint64_t dbk = db + kk * kStepB;
                const uint32_t in1 = fresh && kk == 0 ? 0u : 1u;
                if constexpr (kStack) {
                  umma_bf16_ta(d, ak, dbk, id3, in1);
                  umma_bf16_ta(d + (uint32_t)Kp, ak + 16u, dbk, id2, 1u);
                  umma_bf16_ta(d + (uint32_t)(2 * Kp), ak + 32u, dbk, id1, 1u);
                } else {
                  const uint32_t in2 = kb == 0 && kk == 0 ? 0u : 1u;
                  umma_bf16_ta(d, ak, dbk, id1, in1);
                  umma_bf16_ta(dc, ak, dbk + bK, ida, in2);
                  if (nrest) umma_bf16_ta(dc + (uint32_t)na, ak, dbk + bR, idr, in2);
                  umma_bf16_ta(dc, ak + 16u, dbk, id2, 1u);
                  umma_bf16_ta(dc + (uint32_t)Kp, ak + 32u, dbk, id1, 1u);
                }
              }
              umma_commit(&a_empty[ab]);
            }
            join();
            if (++ab == G.nbuf) { ab = 0; ph_a ^= 1u; }
          }
          if (!ok) break;
          if (one()) hand_over(s, acc, done);
        }
        join();
        if (++s == S) { s = 0; ph ^= 1u; }
        --left;
        if (done) {
          left = 0;
          if (++acc == G.nmain) { acc = 0; ph_acc ^= 1u; }
        }
      }
    }
    // every MMA has completed before TMEM is released (and, on a failure,
    // before the CTA's shared memory goes away)
    if (one()) umma_commit(&drained);
    join();
    wait(&drained, 0);
  } else if (kF32 && warp >= 6) {
    // ---- fp32 features: cut a stage's A tile into parts in tensor memory -----
    // Eight warps: each half of a stage (32 K elements, one A buffer) has its
    // own four; four warps: they take the halves in turn.
    constexpr int kConv = split_conv<T, NCH>();
    const int q = warp & 3, t = q * 32 + lane;               // row (logits) or feature (gradient)
    const int h0 = kConv == 8 ? (warp - 6) >> 2 : 0;
    int it = 0, s = 0;
    uint32_t ph = 0;
    bool ok = true;
    for (int i = 0; i < my_units && ok; ++i) {
      const SplitUnit u = unit(i);
      const int nkb = blocks_of(u);
      for (int kb = 0; kb < nkb && ok; ++kb, ++it) {
        if (!__all_sync(0xffffffffu, mbar_wait(&full[s], ph, p.status))) { ok = false; break; }
        const uint8_t* a = sm + (size_t)s * stage_bytes;
        if (++s == S) { s = 0; ph ^= 1u; }
        for (int h = h0; h < (kConv == 8 ? h0 + 1 : 2); ++h) {
          const uint32_t ah = 2 * (uint32_t)it + (uint32_t)h, use = ah / (uint32_t)G.nbuf, ab = ah - use * (uint32_t)G.nbuf;
          float x[32];
          if constexpr (!kGrad) {
            const uint8_t* row = a + h * (kABytes / 2) + t * 128;
#pragma unroll
            for (int c = 0; c < 8; ++c) {
              const float4 v = *reinterpret_cast<const float4*>(row + ((c ^ (t & 7)) << 4));
              x[4 * c] = v.x; x[4 * c + 1] = v.y; x[4 * c + 2] = v.z; x[4 * c + 3] = v.w;
            }
          } else {
            const float* col = reinterpret_cast<const float*>(a) + (size_t)h * 32 * kSM + t;
#pragma unroll
            for (int r = 0; r < 32; ++r) x[r] = col[r * kSM];
          }
          if (use > 0 && !__all_sync(0xffffffffu, mbar_wait(&a_empty[ab], (use - 1) & 1u, p.status))) {
            ok = false;
            break;
          }
          tc_fence_after();
          const uint32_t ta = tmem + ((uint32_t)(q * 32) << 16) + kSTmem - (ab + 1) * kSBufCols;
#pragma unroll
          for (int part = 0; part < 3; ++part) {
            uint32_t w[16];
#pragma unroll
            for (int j = 0; j < 16; ++j) w[j] = cut_pair(x[2 * j], x[2 * j + 1]);
            tmem_st16(ta + (uint32_t)(part * 16), w);
          }
          tmem_st_wait();
          tc_fence_before();
          __syncwarp();
          if (lane == 0) mbar_arrive(&a_full[ab]);
        }
      }
    }
  } else if (warp >= 2 && warp < 6) {
    // ---- epilogue ----------------------------------------------------------
    const int q = warp & 3, t = q * 32 + lane;               // row (logits) or feature (gradient) of the CTA's 128
    int tt = 0;
    bool ok = true;
    for (int i = 0; i < my_units && ok; ++i) {
      const SplitUnit u = unit(i);
      const int nkb = blocks_of(u), nchunk = (nkb + p.chunk - 1) / p.chunk;
      float z[NCH * 32];
#pragma unroll
      for (int c = 0; c < NCH * 32; ++c) z[c] = 0.f;
      const uint32_t lane_base = tmem + ((uint32_t)(q * 32) << 16);
      for (int ck = 0; ck < nchunk; ++ck, ++tt) {
        const int acc = G.nmain == 2 ? tt & 1 : 0;
        if (!__all_sync(0xffffffffu, mbar_wait(&acc_full[acc], (G.nmain == 2 ? tt / 2 : tt) & 1, p.status))) {
          ok = false;
          break;
        }
        tc_fence_after();
        if (kStack) {
          if constexpr (NCH == 1) {
            float v[32];
#pragma unroll
            for (int c = 0; c < 32; ++c) v[c] = 0.f;
#pragma unroll
            for (int j = 2; j >= 0; --j)                     // smallest first
#pragma unroll
              for (int c = 0; c < 32; c += 16)
                if (c < Kp) tmem_add16(lane_base + (uint32_t)((acc * 3 + j) * Kp + c), v + c);
#pragma unroll
            for (int c = 0; c < 32; ++c) z[c] += v[c];
          }
        } else {
#pragma unroll
          for (int c = 0; c < NCH * 32; c += 16)
            if (c < Kp) tmem_add16(lane_base + (uint32_t)(acc * Kp + c), z + c);
        }
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(&acc_empty[acc]);
      }
      if (!ok) break;
      if (!kStack) {
        // the corrections, 2^-16 and 2^-8 times smaller than the leading sum
        const int cor = G.ncorr == 2 ? i & 1 : 0;
        const uint32_t cb = lane_base + (uint32_t)((G.nmain + 2 * cor) * Kp);
#pragma unroll
        for (int c = 0; c < NCH * 32; c += 16) {
          if (c < Kp) {
            float v[16];
#pragma unroll
            for (int j = 0; j < 16; ++j) v[j] = 0.f;
            tmem_add16(cb + (uint32_t)(Kp + c), v);
            tmem_add16(cb + (uint32_t)c, v);
#pragma unroll
            for (int j = 0; j < 16; ++j) z[c + j] += v[j];
          }
        }
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(&corr_empty[cor]);
      }
      if constexpr (kMode == kSplitLoss) {
        // this thread's row: max and sum of exp over the class block, the label's
        // logit if it is one of them
        const int row = u.r0 + rank * p.h + t;
        if (t < p.h && row < u.rows) {
          const int c0 = u.e * Kp, nc = p.K - c0 < Kp ? p.K - c0 : Kp;
          const int lab = p.y[row] - c0;
          float m = -INFINITY, sum = 0.f;
#pragma unroll
          for (int c = 0; c < NCH * 32; ++c) {
            if (c < nc) m = fmaxf(m, z[c]);
            if (c < nc && c == lab) p.row_lab[row] = z[c];
          }
          const float base = m == -INFINITY ? 0.f : m;       // every class of the block masked: sum 0 (NaN logits still count)
#pragma unroll
          for (int c = 0; c < NCH * 32; ++c)
            if (c < nc) sum += expf(z[c] - base);
          p.row_stats[(int64_t)u.e * p.rows + row] = make_float2(m, sum);
        }
      } else if constexpr (!kGrad) {
        // R = softmax(Z) - onehot(y) of this thread's row (rows of R past the
        // partition, which the gradient's last K block reads, stay zero)
        const int row = u.r0 + rank * p.h + t;
        if (t < p.h && row < u.rows) {
          const int lab = p.y[(int64_t)u.x + row];
          float m = -INFINITY;
#pragma unroll
          for (int c = 0; c < NCH * 32; ++c)
            if (c < p.K) m = fmaxf(m, z[c]);
          // rest: the sum over the classes other than the label.  The label's
          // residual is -rest / (rest + e_label): p - 1 would lose the digits
          // of a row that the model already gets right.
          float rest = 0.f, own = 0.f;
#pragma unroll
          for (int c = 0; c < NCH * 32; ++c) {
            z[c] = c < p.K ? expf(z[c] - m) : 0.f;
            if (c == lab) own = z[c]; else rest += z[c];
          }
          const float inv = 1.0f / (rest + own);
          uint16_t* out = p.R3 + (int64_t)(u.z0 + row) * p.C3;
#pragma unroll
          for (int c = 0; c < NCH * 32; c += 8) {
            if (c < Kp) {
              float v[8];
#pragma unroll
              for (int j = 0; j < 8; ++j)
                v[j] = c + j < p.K ? (c + j == lab ? -rest : z[c + j]) * inv : 0.f;
              uint4 p1, p2, p3;
              split8(v, p1, p2, p3);
              *reinterpret_cast<uint4*>(out + c) = p1;
              *reinterpret_cast<uint4*>(out + Kp + c) = p2;
              *reinterpret_cast<uint4*>(out + 2 * Kp + c) = p3;
            }
          }
        }
      } else {
        const int f = (CL * u.x + rank) * kSM + t;
        if (f < p.ld) {
          if (u.item >= 0) {
            float* out = p.partials + (int64_t)u.item * p.P + f;
#pragma unroll
            for (int c = 0; c < NCH * 32; ++c)
              if (c < p.K) out[(int64_t)c * p.ld] = z[c];
          } else {
            // the unit holds the whole partition: its gradient, into every store that keeps it
            const float sc = p.e_scale[u.e];
            for (int k = 0; k < p.ndest; ++k) {
              const int dst = p.e_dest[u.e * p.ndest + k];
              if (dst < 0) continue;
              float* out = p.store + (int64_t)dst * p.P + f;
#pragma unroll
              for (int c = 0; c < NCH * 32; ++c)
                if (c < p.K) out[(int64_t)c * p.ld] = z[c] * sc;
            }
          }
        }
      }
    }
  }
  __syncthreads();
  tc_fence_before();
  cluster_sync_all();                    // no multicast or remote arrive is still aimed at this CTA
  tc_fence_after();
  if (warp == 1)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(kSTmem) : "memory");
}

// ---------------------------------------------------------------------------
// host side
// ---------------------------------------------------------------------------
namespace {

using SplitKernel = void (*)(const CUtensorMap, SplitArgs);

template <int kMode, typename T>
SplitKernel pick(int Kp) {
  switch ((Kp + 31) / 32) {
    case 1: return split_gemm_kernel<kMode, T, 1>;
    case 2: return split_gemm_kernel<kMode, T, 2>;
    case 3: return split_gemm_kernel<kMode, T, 3>;
    case 4: return split_gemm_kernel<kMode, T, 4>;
    default: return nullptr;
  }
}
template <typename T>
SplitKernel pick_mode(int mode, int Kp) {
  return mode == kSplitLogits ? pick<kSplitLogits, T>(Kp) : mode == kSplitGrad ? pick<kSplitGrad, T>(Kp)
                                                                              : pick<kSplitLoss, T>(Kp);
}
SplitKernel split_kernel(int mode, int dtype, int Kp) {
  return dtype == PGC_BF16 ? pick_mode<uint16_t>(mode, Kp) : pick_mode<float>(mode, Kp);
}

size_t split_smem(int mode, int dtype, int Kp) {
  const int es = dtype == PGC_BF16 ? 2 : 4;
  const SplitGeom g = split_geom(es, Kp, mode == kSplitGrad ? split_cols(Kp) : 3 * Kp);
  return 1024 + (size_t)g.stages * ((size_t)kSM * kSK * es + g.b_bytes);
}

void split_config(cudaLaunchConfig_t& cfg, cudaLaunchAttribute* attr, int mode, int dtype, int Kp, int cl, int clusters) {
  cfg = {};
  cfg.gridDim = dim3((unsigned)(cl * clusters));
  cfg.blockDim = dim3((unsigned)(dtype == PGC_BF16 ? split_threads<uint16_t, 1>()
                                                   : Kp <= 64 ? split_threads<float, 2>() : split_threads<float, 4>()));
  cfg.dynamicSmemBytes = split_smem(mode, dtype, Kp);
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = (unsigned)cl;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[1].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
}

}  // namespace

int split_max_clusters(int mode, int dtype, int64_t K) {
  const int Kp = split_kp(K);
  const SplitKernel k = split_kernel(mode, dtype, Kp);
  if (!k || cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)split_smem(mode, dtype, Kp)) !=
                cudaSuccess)
    return 0;
  cudaLaunchConfig_t cfg;
  cudaLaunchAttribute attr[2];
  split_config(cfg, attr, mode, dtype, Kp, split_cluster(Kp), 1);
  int nc = 0;
  return cudaOccupancyMaxActiveClusters(&nc, k, &cfg) == cudaSuccess ? nc : 0;
}

cudaError_t launch_split(int mode, int dtype, const void* tmB, const SplitArgs& a, int nclusters, bool pdl,
                         cudaStream_t st) {
  if (a.nunits <= 0) return cudaSuccess;
  const SplitKernel k = split_kernel(mode, dtype, a.Kp);
  if (!k || nclusters < 1) return cudaErrorInvalidValue;
  cudaError_t e =
      cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)split_smem(mode, dtype, a.Kp));
  if (e != cudaSuccess) return e;
  cudaLaunchConfig_t cfg;
  cudaLaunchAttribute attr[2];
  split_config(cfg, attr, mode, dtype, a.Kp, a.cl, nclusters < a.nunits ? nclusters : a.nunits);
  cfg.stream = st;
  cfg.numAttrs = pdl ? 2 : 1;
  CUtensorMap b;
  std::memcpy(&b, tmB, sizeof(CUtensorMap));
  return cudaLaunchKernelEx(&cfg, k, b, a);
}

// Sum over the rows of log sum_k exp(z_k) - z_y from the class blocks' (max, sum
// of exp) and the label's logit; the last block to finish adds the blocks'
// sums in order and divides by the rows (ticket returns to 0).
__global__ void __launch_bounds__(256) loss_combine_kernel(const float2* __restrict__ stats, const float* __restrict__ lab,
                                                           int64_t rows, int ncb, double* blocksum, int* ticket,
                                                           double* out) {
  __shared__ double red[8];
  __shared__ int last;
  grid_dep_wait();
  double acc = 0.0;
  for (int64_t r = (int64_t)blockIdx.x * 256 + threadIdx.x; r < rows; r += (int64_t)gridDim.x * 256) {
    float M = -INFINITY;
    for (int b = 0; b < ncb; ++b) M = fmaxf(M, stats[b * rows + r].x);
    float s = 0.f;
    for (int b = 0; b < ncb; ++b) {
      const float2 v = stats[b * rows + r];
      s += v.y * expf(v.x - M);
    }
    acc += (double)M + log((double)s) - (double)lab[r];
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = acc;
  __syncthreads();
  if (threadIdx.x == 0) {
    double t = 0.0;
    for (int i = 0; i < 8; ++i) t += red[i];
    blocksum[blockIdx.x] = t;
    last = atomic_add_acq_rel(ticket, 1) == (int)gridDim.x - 1;
  }
  __syncthreads();
  if (last && threadIdx.x < 32) {
    __threadfence();
    double t = 0.0;
    for (int i = threadIdx.x; i < (int)gridDim.x; i += 32) t += __ldcg(blocksum + i);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
    if (threadIdx.x == 0) {
      *out = t / (double)rows;
      *ticket = 0;
    }
  }
}

cudaError_t launch_loss_combine(const float2* stats, const float* lab, int64_t rows, int ncb, double* blocksum,
                                int max_blocks, int* ticket, double* out, bool pdl, cudaStream_t st) {
  int64_t blocks = (rows + 255) / 256;
  if (blocks > max_blocks) blocks = max_blocks;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)blocks);
  cfg.blockDim = dim3(256);
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = pdl ? 1 : 0;
  return cudaLaunchKernelEx(&cfg, loss_combine_kernel, stats, lab, rows, ncb, blocksum, ticket, out);
}

// fp32 [K][ld] -> bf16 parts [K / Kp blocks][3][Kp][ld] (Kp classes per block)
__global__ void split_weights_kernel(const float* __restrict__ src, uint16_t* __restrict__ dst, int64_t K, int64_t ld,
                                     int Kp) {
  const int64_t row4 = ld / 4, stride = (int64_t)Kp * ld;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < K * row4; i += (int64_t)gridDim.x * blockDim.x)
    store_split4(dst + i / row4 / Kp * 2 * stride, stride, i, reinterpret_cast<const float4*>(src)[i]);
}

cudaError_t launch_split_weights(const float* src, uint16_t* dst, int64_t K, int64_t ld, int Kp, cudaStream_t st) {
  int64_t blocks = (K * (ld / 4) + 255) / 256;
  if (blocks > 4096) blocks = 4096;
  if (blocks > 0) split_weights_kernel<<<(unsigned)blocks, 256, 0, st>>>(src, dst, K, ld, Kp);
  return cudaGetLastError();
}

}  // namespace pgc
