// Warp-specialized tcgen05 GEMM fed by TMA, for complex operands prepared as
// four K-major 16-bit planes {re_hi, re_lo, im_hi, im_lo} (see k_split.cu).
//
// Paper: Sec. "Tensor Contraction Using Fused Permutation and Multiplication"
// (dense case: high compute density contraction at near-peak rate) and Sec.
// "A Mixed-Precision Computation Method via Adaptive Precision Scaling"
// (half-precision products, single-precision accumulation).
//
// Complex product on real tensor cores, planar form:
//   Dr = Ar Br - Ai Bi,  Di = Ar Bi + Ai Br,
// FP32 accumulation in TMEM (Dr and Di take TN columns each), the minus sign
// through the MMA's negate-A bit.  Split precision (four planes re_hi, re_lo,
// im_hi, im_lo) expands each real product X Y as Xhi Yhi + Xhi Ylo + Xlo Yhi
// and bounds the tensor core's truncating accumulation to short chunks of K;
// single precision (two planes re, im) keeps one 16-bit product and
// accumulates all of K in one chunk.  Both run in gemm_tma_chunked, one
// persistent CTA per SM with double-buffered accumulators.
//
// Adaptive scaling (Sec. "A Mixed-Precision Computation Method via Adaptive
// Precision Scaling"): a plane tensor stores x 2^-e with a per-unit integer
// exponent e and records the largest stored component.  The GEMM predicts a
// bound 2 K maxA maxB on its stored output, picks r so that the bound stays
// below 2^15 (inside fp16 range), writes C 2^-(eA+eB+r) and records
// eC = eA + eB + r and the actual maximum.  A unit whose values turn
// non-finite, or whose operand maximum fell below 2^-10 (most of the 16-bit
// range lost to underflow), is flagged for the executor's filter.
//
// Roles: warp 0 lane 0 issues TMA loads of one K stage (a 128-row A tile and a
// TN-row B tile, all planes; a row holds up to 32 complex K values in split
// precision, 64 in single, see row_bytes) into a ring of stages guarded by
// full/empty mbarriers; warp 1 lane 0 issues the tcgen05.mma instructions and
// commits each stage back to its empty barrier; warp 2 owns the TMEM
// allocation; warps 4.. read the accumulators (tcgen05.ld) and write complex64
// C, or C's 16-bit planes, through per-row and per-column offsets (the output
// permutation).  Every wait is bounded: on expiry the CTA records an error code
// and stops issuing work; before it leaves, the producer waits (bounded) for
// every TMA load it issued and the MMA warp for every MMA it issued, so no
// asynchronous copy or MMA still targets the CTA's shared memory or TMEM when
// it releases them.  Each CTA loads its own operand tiles from this GPU's
// memory (no clusters).
#include <cuda.h>
#include <cudaTypedefs.h>
#include <cuda_bf16.h>
#include <cuda_fp16.h>

#include <algorithm>
#include <atomic>
#include <cstdlib>
#include <mutex>
#include <type_traits>

#include "device_common.h"
#include "kernels.h"
#include "per_device.h"

namespace tn {

namespace {

constexpr int TM = 128;
constexpr int SMEM_BUDGET = 196 * 1024;
constexpr long long kWaitLimit = 1ll << 24;  // default polls of a pipeline wait
constexpr long long kDrainLimit = 1ll << 24;  // polls of a wait for this CTA's own copies / MMAs on the way out
constexpr int GROUP_M_DEFAULT = 16;

// Bytes of one operand row in a K stage: the largest of 32, 64 and (two planes)
// 128 that K fills, each with the TMA / MMA swizzle of that width, so a short K
// copies and multiplies no zeros; 16 stands for K = 8 by bulk copies (below).
// The four-plane kernel stops at 64-byte rows: its 128-byte stages would be
// 128 KB, one per SM.
constexpr int K8_ROWB = 16;
int row_bytes(int64_t kp, int np) { return np == 2 && kp >= 64 ? 128 : kp >= 32 ? 64 : 32; }

// Stage geometry: a K stage holds A's NP planes of TM rows, then B's of TN rows.
template <int TN, int NP, int ROWB>
struct Cfg2 {
  static constexpr int TKC = ROWB == K8_ROWB ? 8 : ROWB / 2;  // complex K per stage
  static constexpr int KSTEPS = (TKC + 15) / 16;              // 16-K MMA steps
  static constexpr int ROW = ROWB == K8_ROWB ? 32 : ROWB;     // shared memory per row
  static constexpr int A_PLANE = TM * ROW, B_PLANE = TN * ROW;
  static constexpr int A_STAGE = NP * A_PLANE;
  static constexpr int STAGE = A_STAGE + NP * B_PLANE;
};

__device__ __forceinline__ uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ void mbar_init(uint64_t* bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count));
}

// Polls of every pipeline wait of the kernels below on this device (set by
// set_tc_wait_limit; 0 makes every pipeline wait give up at once).
__device__ long long g_wait_limit = kWaitLimit;

__device__ __forceinline__ bool mbar_wait(uint64_t* bar, uint32_t parity, long long limit) {
  const uint32_t a = smem_u32(bar);
  for (long long it = 0; it < limit; ++it) {
    uint32_t ok;
    asm volatile(
        "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}\n"
        : "=r"(ok)
        : "r"(a), "r"(parity)
        : "memory");
    if (ok) return true;
  }
  return false;
}

__device__ __forceinline__ void mbar_expect_tx(uint64_t* bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes) : "memory");
}

__device__ __forceinline__ void tma_load_5d(void* dst, const CUtensorMap* map, uint64_t* bar, int c0, int c1, int c2,
                                            int c3, int c4) {
  asm volatile(
      "cp.async.bulk.tensor.5d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4, %5, %6}], "
      "[%7];" ::"r"(smem_u32(dst)),
      "l"(reinterpret_cast<uint64_t>(map)), "r"(c0), "r"(c1), "r"(c2), "r"(c3), "r"(c4), "r"(smem_u32(bar))
      : "memory");
}

// One contiguous run of global memory into shared memory (16-byte aligned
// addresses, a multiple of 16 bytes), completing on the stage's barrier.
__device__ __forceinline__ void bulk_load(void* dst, const void* src, uint32_t bytes, uint64_t* bar) {
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
                   smem_u32(dst)),
               "l"(src), "r"(bytes), "r"(smem_u32(bar))
               : "memory");
}

// Shared-memory operand descriptors, K-major, version 1 (bits 46-47), as low
// word (start address >> 4, leading byte offset >> 4 at bit 16) and high word
// (stride byte offset >> 4, version at bit 14, swizzle mode at bit 29).
// Swizzled rows of ROWB bytes: 8-row groups 8 ROWB bytes apart, swizzle mode 6
// (32 bytes), 4 (64) or 2 (128).  K8_ROWB: no swizzle, core matrices of 8 rows x
// 16 bytes, each 128 contiguous bytes; 16 ROWS bytes between the two core
// matrices of a 16-K step, 128 between 8-row groups.
template <int ROWB, int ROWS>
struct OperandDesc {
  static constexpr uint32_t LO = ROWB == K8_ROWB ? (uint32_t)((ROWS * 16) >> 4) << 16 : 1u << 16;
  static constexpr uint32_t HI = (uint32_t)((ROWB == K8_ROWB ? 128 : 8 * ROWB) >> 4) | (1u << 14) |
                                 (uint32_t)(ROWB == 128  ? 2
                                            : ROWB == 64 ? 4
                                            : ROWB == 32 ? 6
                                                         : 0)
                                     << 29;
};

// kind::f16 instruction descriptor: FP32 accumulate, A/B 16-bit format
// (0 fp16, 1 bf16), optional negate-A (bit 13), K-major A and B, N >> 3 at
// bit 17, M >> 4 at bit 24.
__host__ __device__ constexpr uint32_t idesc2(bool bf16, int M, int N, bool neg_a) {
  return (1u << 4) | ((bf16 ? 1u : 0u) << 7) | ((bf16 ? 1u : 0u) << 10) | ((neg_a ? 1u : 0u) << 13) |
         ((uint32_t)(N >> 3) << 17) | ((uint32_t)(M >> 4) << 24);
}

template <int ROWB, int TN>
__device__ __forceinline__ void mma(uint32_t d, uint32_t a_lo, uint32_t b_lo, uint32_t idesc, uint32_t acc) {
  asm volatile(
      "{\n .reg .pred p;\n .reg .b64 da, db;\n setp.ne.b32 p, %6, 0;\n mov.b64 da, {%1, %2};\n mov.b64 db, {%3, "
      "%4};\n"
      " tcgen05.mma.cta_group::1.kind::f16 [%0], da, db, %5, p;\n}\n" ::"r"(d),
      "r"(a_lo), "n"(OperandDesc<ROWB, TM>::HI), "r"(b_lo), "n"(OperandDesc<ROWB, TN>::HI), "r"(idesc), "r"(acc));
}

// The MMAs of one 16-K step: Dr (at dr) and Di (at di) += A B from the stage's
// planes, a and b0 their descriptors' low words; `acc` 0 starts the sums.
template <int NP, int TN, int ROWB>
__device__ __forceinline__ void mma_step(uint32_t dr, uint32_t di, uint32_t a, uint32_t b0, int kk, uint32_t I,
                                         uint32_t IN, uint32_t acc) {
  using CF = Cfg2<TN, NP, ROWB>;
  uint32_t A_[NP], B_[NP];
#pragma unroll
  for (int p = 0; p < NP; ++p) {
    A_[p] = a + ((p * CF::A_PLANE + kk * 32) >> 4);
    B_[p] = b0 + ((p * CF::B_PLANE + kk * 32) >> 4);
  }
  auto mm = [&](uint32_t dst, int pa, int pb, uint32_t id, uint32_t ac) { mma<ROWB, TN>(dst, A_[pa], B_[pb], id, ac); };
  if constexpr (NP == 4) {
    // planes: 0 re_hi, 1 re_lo, 2 im_hi, 3 im_lo; the chunk is short, so the
    // hi*lo + lo*hi terms share the hi*hi accumulator
    mm(dr, 0, 0, I, acc);
    mm(dr, 0, 1, I, 1u);
    mm(dr, 1, 0, I, 1u);
    mm(dr, 2, 2, IN, 1u);
    mm(dr, 2, 3, IN, 1u);
    mm(dr, 3, 2, IN, 1u);
    mm(di, 0, 2, I, acc);
    mm(di, 0, 3, I, 1u);
    mm(di, 1, 2, I, 1u);
    mm(di, 2, 0, I, 1u);
    mm(di, 2, 1, I, 1u);
    mm(di, 3, 0, I, 1u);
  } else {
    // planes: 0 re, 1 im
    mm(dr, 0, 0, I, acc);
    mm(dr, 1, 1, IN, 1u);
    mm(di, 0, 1, I, acc);
    mm(di, 1, 0, I, 1u);
  }
}

// One lane of the (converged) warp.  The compiler knows that a single thread
// runs what this guards and keeps the operands of TMA and MMA instructions in
// uniform registers; under `lane == 0` it cannot, and issuing an MMA took about
// as long as running it.  Measured (log2 M, N, K), with the K stages' row widths
// below: two planes, (11, 11, 10) x 1024 units 1238 -> 1636 TFLOP/s; four planes,
// (13, 11, 9) x 128 units 478 -> 581 counted (1743 issued), (11, 11, 12) 524 ->
// 570.
__device__ __forceinline__ bool elect_one() {
  uint32_t p;
  asm volatile("{\n .reg .pred p;\n elect.sync _|p, 0xffffffff;\n selp.u32 %0, 1, 0, p;\n}\n" : "=r"(p));
  return p != 0;
}

// A pipeline wait by a whole warp; false for every lane if any lane gave up.
__device__ __forceinline__ bool mbar_wait_warp(uint64_t* bar, uint32_t parity, long long limit) {
  return __all_sync(0xffffffffu, mbar_wait(bar, parity, limit));
}

__device__ __forceinline__ void commit(uint64_t* bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(smem_u32(bar))
               : "memory");
}

__device__ __forceinline__ int32_t bit_offset(int64_t x, int nb, const int32_t* st) {
  int32_t o = 0;
  for (int i = 0; i < nb; ++i)
    if ((x >> i) & 1) o += st[i];
  return o;
}

// One element as packed 16-bit planes, re in the low halves' plane order:
// four planes (x = hi + lo, hi = rn16(x), lo = rn16(x - hi)): e[0] = re_hi |
// re_lo << 16, e[1] = im_hi | im_lo << 16; two planes: e[0] = re | im << 16.
// Plane p sits in half p & 1 of e[p >> 1].
template <int NP>
__device__ __forceinline__ void pack_planes(bool bf16, float re, float im, uint32_t* e) {
  uint32_t hu, lu = 0;
  if (bf16) {
    const __nv_bfloat162 h = __floats2bfloat162_rn(re, im);
    hu = *reinterpret_cast<const uint32_t*>(&h);
    if (NP == 4) {
      const float2 hf = __bfloat1622float2(h);
      const __nv_bfloat162 l = __floats2bfloat162_rn(re - hf.x, im - hf.y);
      lu = *reinterpret_cast<const uint32_t*>(&l);
    }
  } else {
    const __half2 h = __floats2half2_rn(re, im);
    hu = *reinterpret_cast<const uint32_t*>(&h);
    if (NP == 4) {
      const float2 hf = __half22float2(h);
      const __half2 l = __floats2half2_rn(re - hf.x, im - hf.y);
      lu = *reinterpret_cast<const uint32_t*>(&l);
    }
  }
  if (NP == 4) {
    e[0] = __byte_perm(hu, lu, 0x5410);
    e[NP / 2 - 1] = __byte_perm(hu, lu, 0x7632);
  } else {
    e[0] = hu;
  }
}

// Number of leading tile column bits that are C's fastest indices in order
// (strides 1, 2, 4, ..): runs of 2^vb tile columns are contiguous in C.
__device__ __forceinline__ int vec_bits(const GemmDesc& d) {
  int v = 0;
  while (v < 4 && v < d.nn && d.cn[v] == (1 << v)) ++v;
  return v;
}

// C offset of tile column j of 16 from the strides of its four bits.
__device__ __forceinline__ int32_t col_offset(const int32_t (&cs)[4], int j) {
  return ((j & 1) ? cs[0] : 0) + ((j & 2) ? cs[1] : 0) + ((j & 4) ? cs[2] : 0) + ((j & 8) ? cs[3] : 0);
}

// One thread's 16 consecutive tile columns of one row (packed elements, see
// pack_planes) as NP 16-bit planes, P at the row and first column: each
// contiguous run of 2^vb columns goes out as one store per plane (the run
// starts at a multiple of 2^vb elements: every other index of C has a larger
// stride).
template <int NP>
__device__ __forceinline__ uint32_t plane_pair(const uint32_t (&e)[NP / 2][16], int p, int j) {
  return __byte_perm(e[p >> 1][j], e[p >> 1][j + 1], (p & 1) ? 0x7632 : 0x5410);
}
template <int NP>
__device__ __forceinline__ void store_planes(uint16_t* P, int64_t plane, const int32_t (&cs)[4], int vb,
                                             const uint32_t (&e)[NP / 2][16]) {
  auto pk = [&](int p, int j) { return plane_pair<NP>(e, p, j); };
  if (vb >= 3) {
#pragma unroll
    for (int r = 0; r < 2; ++r)
#pragma unroll
      for (int p = 0; p < NP; ++p)
        *reinterpret_cast<uint4*>(P + p * plane + col_offset(cs, 8 * r)) =
            make_uint4(pk(p, 8 * r), pk(p, 8 * r + 2), pk(p, 8 * r + 4), pk(p, 8 * r + 6));
  } else if (vb == 2) {
#pragma unroll
    for (int r = 0; r < 4; ++r)
#pragma unroll
      for (int p = 0; p < NP; ++p)
        *reinterpret_cast<uint2*>(P + p * plane + col_offset(cs, 4 * r)) = make_uint2(pk(p, 4 * r), pk(p, 4 * r + 2));
  } else if (vb == 1) {
#pragma unroll
    for (int r = 0; r < 8; ++r)
#pragma unroll
      for (int p = 0; p < NP; ++p) *reinterpret_cast<uint32_t*>(P + p * plane + col_offset(cs, 2 * r)) = pk(p, 2 * r);
  } else {
#pragma unroll
    for (int j = 0; j < 16; ++j)
#pragma unroll
      for (int p = 0; p < NP; ++p)
        P[p * plane + col_offset(cs, j)] = (uint16_t)((p & 1) ? e[p >> 1][j] >> 16 : e[p >> 1][j] & 0xffffu);
  }
}

// x0 f and x1 f in one instruction (x as register bits).
__device__ __forceinline__ void mul_pair(uint32_t x0, uint32_t x1, float f, float& y0, float& y1) {
  asm("{\n .reg .b64 a, b;\n mov.b64 a, {%2, %3};\n mov.b64 b, {%4, %4};\n mul.rn.f32x2 a, a, b;\n mov.b64 {%0, %1}, a;\n}\n"
      : "=f"(y0), "=f"(y1)
      : "r"(x0), "r"(x1), "f"(f));
}
__device__ __forceinline__ float max_nan(float a, float b) {
  float r;
  asm("max.NaN.f32 %0, %1, %2;" : "=f"(r) : "f"(a), "f"(b));
  return r;
}
__device__ __forceinline__ void sts64(uint32_t a, uint32_t x, uint32_t y) {
  asm volatile("st.shared.v2.b32 [%0], {%1, %2};" ::"r"(a), "r"(x), "r"(y) : "memory");
}
__device__ __forceinline__ void sts32(uint32_t a, uint32_t x) {
  asm volatile("st.shared.b32 [%0], %1;" ::"r"(a), "r"(x) : "memory");
}
__device__ __forceinline__ uint4 lds128(uint32_t a) {
  uint4 v;
  asm volatile("ld.shared.v4.b32 {%0, %1, %2, %3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "r"(a) : "memory");
  return v;
}

template <int NREG>
__device__ __forceinline__ void tmem_ld(uint32_t taddr, uint32_t* v);
template <>
__device__ __forceinline__ void tmem_ld<16>(uint32_t taddr, uint32_t* v) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
      : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]),
        "=r"(v[8]), "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]), "=r"(v[14]), "=r"(v[15])
      : "r"(taddr));
}

// Producer's way out: wait (bounded) until the TMA loads of the last
// min(issued, ns) stages it filled have landed.  Earlier stages were waited
// for by the MMA warp before their slots were refilled; on the normal path
// these phases have completed already and every wait returns at once.
__device__ __forceinline__ void drain_loads(uint64_t* full, int ns, int64_t issued, int* err) {
  for (int64_t q = issued > ns ? issued - ns : 0; q < issued; ++q)
    if (!mbar_wait(&full[q % ns], (uint32_t)((q / ns) & 1), kDrainLimit)) {
      atomicExch(err, 9);
      return;
    }
}

// Staged output.  A warp's 32 x 16 sub-tile (lanes = tile row bits 0..4,
// columns = tile column bits 0..3) covers 512 elements of C; sorted by their C
// stride these 9 bits give each element a C-order index.  The warp writes its
// values to shared memory at their C-order index and reads them back in C
// order, consecutive lanes taking consecutive 16-byte pieces (2 complex64
// values, or 8 values of one 16-bit plane): the first `run` sorted strides are
// 1, 2, 4, .., so each store instruction writes runs of 2^run values.  Only a
// complex64 output whose lanes already cover consecutive elements, or one whose
// fastest indices lie outside the sub-tile, goes out directly.
constexpr int STAGE_SLOTS = 512 + 64;  // 8-byte slots per warp: 512 elements, 2 padding slots after every 16

struct StageMap {
  bool on;
  int lane_idx;        // this lane's bits of its elements' C-order index
  int rank_c[4];       // C-order rank of column bits 0..3
  int32_t off_c64;     // C offset of this lane's pair (C-order index 2 lane) in read-back step 0
  int32_t step_c64[3]; // C offset added by bits 0..2 of the complex64 read-back step
  int32_t off_pl;      // C offset of this lane's 8 values (C-order index 8 lane) in read-back step 0
  int32_t step_pl;     // C offset added by the second plane read-back step
};

__device__ __forceinline__ StageMap stage_map(const GemmDesc& d, int lane, bool planes, bool wide) {
  StageMap m;
  int32_t st[9], sst[9];
  int rnk[9];
  for (int b = 0; b < 5; ++b) st[b] = d.cm[b];
  for (int b = 0; b < 4; ++b) st[5 + b] = d.cn[b];
  for (int b = 0; b < 9; ++b) {  // the strides of C's indices are distinct powers of two
    int r = 0;
    for (int o = 0; o < 9; ++o) r += st[o] < st[b];
    rnk[b] = r;
    sst[r] = st[b];
  }
  int run = 0;
  while (run < 9 && sst[run] == (1 << run)) ++run;
  int lane_run = 0;
  while (lane_run < 5 && d.cm[lane_run] == (1 << lane_run)) ++lane_run;
  m.on = planes ? run >= 3 : run >= 1 && lane_run < 5 && wide;
  m.lane_idx = 0;
  for (int b = 0; b < 5; ++b) m.lane_idx |= ((lane >> b) & 1) << rnk[b];
  for (int b = 0; b < 4; ++b) m.rank_c[b] = rnk[5 + b];
  // read-back step t, lane l: complex64 pair l + 32 t (C-order index bits
  // 1..5 from the lane, 6..8 from t); plane group of 8 values l + 32 t (bits
  // 3..7 from the lane, bit 8 from t)
  m.off_c64 = 0;
  m.off_pl = 0;
  for (int b = 0; b < 5; ++b) {
    m.off_c64 += ((lane >> b) & 1) * sst[1 + b];
    m.off_pl += ((lane >> b) & 1) * sst[3 + b];
  }
  for (int b = 0; b < 3; ++b) m.step_c64[b] = sst[6 + b];
  m.step_pl = sst[8];
  return m;
}

// 8-byte slot of a C-order index (complex64, or four packed planes), and 4-byte
// slot (two packed planes); both pad 16 bytes after every 128.
__device__ __forceinline__ int stage_slot(int idx) { return idx + ((idx >> 4) << 1); }
__device__ __forceinline__ int stage_slot4(int idx) { return idx + ((idx >> 5) << 2); }
static_assert(511 + (511 >> 4) * 2 < STAGE_SLOTS, "the last element's slot lies inside the warp's slots");
static_assert(511 + (511 >> 5) * 4 < 2 * STAGE_SLOTS, "the last element's slot lies inside the warp's slots");

__device__ __forceinline__ void tmem_st16(uint32_t taddr, const uint32_t* v) {
  asm volatile(
      "tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16};" ::"r"(
          taddr),
      "r"(v[0]), "r"(v[1]), "r"(v[2]), "r"(v[3]), "r"(v[4]), "r"(v[5]), "r"(v[6]), "r"(v[7]), "r"(v[8]), "r"(v[9]),
      "r"(v[10]), "r"(v[11]), "r"(v[12]), "r"(v[13]), "r"(v[14]), "r"(v[15])
      : "memory");
}

// The GEMM: one persistent CTA per SM walks the (unit, tile) work items; the
// K-stage ring runs on across items, and two TMEM accumulator buffers let the
// epilogue warps drain one item while the MMA warp accumulates the next.
//
// Chunked accumulation (split precision).  The tensor core adds into its FP32
// accumulator with truncation, so over a long K the error grows linearly and is
// biased toward zero.  Here every chunk of `chunk` K stages starts a fresh
// accumulator, and the epilogue warps add the chunks with round-to-nearest
// FP32 adds, so the bias scales with the chunk length, not with K.  (Single
// precision, whose 16-bit products dominate the error, runs as one chunk.)
//
// TMEM holds two buffers of 2 TN columns (Dr, Di).  The CTA's t-th tile keeps
// its running sum R in buffer t & 1: its first chunk accumulates there
// directly; every later chunk accumulates in the other buffer P, which the
// epilogue folds into R (R += P, read P, read R, add, write R) and releases.
// After the last chunk the epilogue scales and stores R while the MMA warp
// already runs the next tile's first chunk in the other buffer (the next
// tile's R), so the MMA warp waits only for the folds, never for a store.
// K stages per chunk (32 complex K each): 16 unless TN_SPLIT_CHUNK says
// otherwise; the bias grows with the chunk length, so longer chunks trade
// accuracy for fewer folds.
int split_chunk() {
  static const int c = [] {
    const char* e = getenv("TN_SPLIT_CHUNK");
    const int v = e ? atoi(e) : 16;
    return v >= 1 && v <= 4096 ? v : 16;
  }();
  return c;
}

// Chunked kernel with EW epilogue warps (4 or 8): 128 + 32 EW threads.  Eight
// epilogue warps (two per TMEM lane quarter, taking alternate 16-column
// chunks) double the epilogue's latency hiding for output-bound steps; their
// staging buffers leave room for fewer operand stages.
template <int TN, int NP, int ROWB, int EW>
struct ChunkCfg {
  static constexpr int THREADS = 128 + 32 * EW;
  static constexpr int STAGE_BYTES = EW * STAGE_SLOTS * 8;
  static constexpr int BUDGET = EW == 4 ? SMEM_BUDGET : 227 * 1024 - STAGE_BYTES - 1024 - 4096;
  static constexpr int STAGE = Cfg2<TN, NP, ROWB>::STAGE;
  static constexpr int NS = (BUDGET / STAGE) < 8 ? (BUDGET / STAGE) : 8;
  static constexpr int SMEM = NS * STAGE + 1024 + STAGE_BYTES;
  static_assert(NS >= 2, "at least two operand stages");
};

// Planes of one operand for K = 8 (16-byte rows): byte address of plane p,
// row r of the unit (zlo, zhi) = base + zlo st_lo + zhi st_hi + p plane + 16 r.
// A null base selects the tensor-map loads.
struct BulkPlanes {
  const uint8_t* base;
  int64_t st_lo, st_hi, plane;
};

template <int TN, int NP, int ROWB, int EW, bool PARTS>
__global__ void __launch_bounds__(ChunkCfg<TN, NP, ROWB, EW>::THREADS, 1)
    gemm_tma_chunked(const __grid_constant__ CUtensorMap mapA, const __grid_constant__ CUtensorMap mapB,
                     float2* __restrict__ C0, const GemmDesc d, int kp, int a_zlo, int a_zhi, int b_zlo, int b_zhi,
                     int out_flags, const ScaleIO sio, int chunk, int fold, bool bf16, int* __restrict__ err,
                     const BulkPlanes ba, const BulkPlanes bb, int parts_arg, float2* __restrict__ part) {
  using CC = ChunkCfg<TN, NP, ROWB, EW>;
  using CF = Cfg2<TN, NP, ROWB>;
  constexpr bool K8 = ROWB == K8_ROWB;  // K = 8 by bulk copies (ba, bb)
  constexpr int NS = CC::NS;
  constexpr int NT = CC::THREADS;
  constexpr int ET = 32 * EW;  // epilogue threads
  constexpr uint32_t BUF = 2 * TN;  // columns of one buffer
  constexpr uint32_t COLS = 2 * BUF < 32 ? 32 : 2 * BUF;
  static_assert(2 * BUF <= 512, "two accumulator buffers must fit in TMEM");
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = (uint8_t*)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
  __shared__ uint64_t full[NS], empty[NS], acc_full[2], acc_empty[2], mma_done;
  __shared__ uint32_t tmem_slot;
  __shared__ volatile int abort_flag;

  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const long long wl = g_wait_limit;
  const int64_t first = blockIdx.x, stride = gridDim.x;
  // fold > 1: `fold` consecutive hi units share A, and their N = 2^nn columns
  // side by side form the TN columns of one tile (so TN = fold * 2^nn)
  const int nsub = 1 << d.nn;
  const int ntm = (int)((int64_t(1) << d.nm) / TM), ntn = fold > 1 ? 1 : (int)((int64_t(1) << d.nn) / TN);
  const int tiles = ntm * ntn;
  // PARTS: each accumulation chunk of a tile is an item of its own, whose sum
  // goes to `part` ([chunk][unit][C's elements]) unscaled; combine_kernel adds
  // them in chunk order, as the folds below do
  const int parts = PARTS ? parts_arg : 1;
  const int64_t items = (int64_t)tiles * (d.units / fold) * parts;
  const int nkt = (kp + CF::TKC - 1) / CF::TKC;
  const int nch = PARTS ? 1 : (nkt + chunk - 1) / chunk;
  const int GM = d.group_m > 0 ? d.group_m : GROUP_M_DEFAULT;
  const bool items32 = items < (int64_t(1) << 31);
  auto decode = [&](int64_t item, int& unit, int& m0, int& n0, int& cp) {
    int t;
    cp = 0;
    if (PARTS) {
      cp = (int)(item % parts);
      item /= parts;
    }
    if (items32) {  // 32-bit division: a 64-bit one is a long dependent sequence
      unit = (int)((uint32_t)item / (uint32_t)tiles);
      t = (int)((uint32_t)item - (uint32_t)unit * (uint32_t)tiles);
    } else {
      unit = (int)(item / tiles);
      t = (int)(item % tiles);
    }
    const int per_group = GM * ntn;
    const int g = t / per_group, r = t % per_group;
    const int gm = min(GM, ntm - g * GM);
    m0 = (g * GM + r % gm) * TM;
    n0 = (r / gm) * TN;
  };

  if (tid == 0) {
    for (int s = 0; s < NS; ++s) { mbar_init(&full[s], 1); mbar_init(&empty[s], 1); }
    for (int b = 0; b < 2; ++b) { mbar_init(&acc_full[b], 1); mbar_init(&acc_empty[b], ET); }
    mbar_init(&mma_done, 1);
    abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(&mapA)) : "memory");
    asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(&mapB)) : "memory");
  }
  // K = 8: each operand plane sits in a stage as its 16-byte rows (one bulk
  // copy) followed by as many zero bytes, the second core matrix of every
  // 16-K MMA step; the zeros are written once here
  if constexpr (K8) {
    for (int s = 0; s < NS; ++s) {
      uint8_t* st = smem + s * CF::STAGE;
      for (int i = tid; i < NP * TM; i += NT) {
        const int p = i / TM, o = i % TM;
        reinterpret_cast<uint4*>(st + p * CF::A_PLANE + TM * 16)[o] = make_uint4(0u, 0u, 0u, 0u);
      }
      for (int i = tid; i < NP * TN; i += NT) {
        const int p = i / TN, o = i % TN;
        reinterpret_cast<uint4*>(st + CF::A_STAGE + p * CF::B_PLANE + TN * 16)[o] = make_uint4(0u, 0u, 0u, 0u);
      }
    }
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");  // visible to the tensor core's reads
  }
  if (warp == 2) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_slot)),
                 "r"(COLS));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tmem = tmem_slot;
  let_next_start();
  after_previous();

  if (warp == 0) {
    // ---- TMA producer (the whole warp waits, one lane issues): the stage ring
    // runs on across items
    const bool leader = elect_one();
    int64_t g = 0;
    int s = 0;
    uint32_t lap = 0;  // times round the ring
    bool ok = true;
    for (int64_t it = first; ok && it < items; it += stride) {
      int unit, m0, n0, cp;
      decode(it, unit, m0, n0, cp);
      const int ulo = unit % d.units_lo, uhi = (unit / d.units_lo) * fold;
      const int za_lo = a_zlo ? ulo : 0, za_hi = a_zhi ? uhi : 0;
      const int zb_lo = b_zlo ? ulo : 0, zb_hi = b_zhi ? uhi : 0;
      if (__any_sync(0xffffffffu, abort_flag)) break;
      const int kt1 = PARTS ? min(nkt, (cp + 1) * chunk) : nkt;
      for (int kt = cp * chunk; kt < kt1; ++kt, ++g) {
        if (lap > 0 && !mbar_wait_warp(&empty[s], (lap - 1) & 1, wl)) {
          if (leader) {
            atomicExch(err, 31);
            abort_flag = 1;
          }
          ok = false;
          break;
        }
        uint8_t* st = smem + s * CF::STAGE;
        uint64_t* fb = &full[s];
        if (leader) {
          if constexpr (K8) {
            // a 2 KB run of each of A's planes and a run of each of B's (per folded unit)
            mbar_expect_tx(fb, NP * TM * 16 + NP * TN * 16);
            const uint8_t* ga = ba.base + za_lo * ba.st_lo + za_hi * ba.st_hi + (int64_t)m0 * 16;
#pragma unroll
            for (int p = 0; p < NP; ++p) bulk_load(st + p * CF::A_PLANE, ga + p * ba.plane, TM * 16, fb);
            for (int f = 0; f < fold; ++f) {
              const uint8_t* gb = bb.base + zb_lo * bb.st_lo + (fold > 1 ? uhi + f : zb_hi) * bb.st_hi +
                                  (int64_t)(fold > 1 ? 0 : n0) * 16;
              const int rows = fold > 1 ? nsub : TN;
#pragma unroll
              for (int p = 0; p < NP; ++p)
                bulk_load(st + CF::A_STAGE + p * CF::B_PLANE + f * rows * 16, gb + p * bb.plane, rows * 16, fb);
            }
          } else {
            mbar_expect_tx(fb, CF::STAGE);
            tma_load_5d(st, &mapA, fb, kt * CF::TKC, m0, 0, za_lo, za_hi);
            if (fold == 1) {
              tma_load_5d(st + CF::A_STAGE, &mapB, fb, kt * CF::TKC, n0, 0, zb_lo, zb_hi);
            } else {
              // the B map's box is one plane of 2^nn rows: plane p of hi unit
              // uhi + f goes to rows f * 2^nn.. of plane p in the stage
              for (int f = 0; f < fold; ++f)
#pragma unroll
                for (int p = 0; p < NP; ++p)
                  tma_load_5d(st + CF::A_STAGE + p * CF::B_PLANE + f * nsub * ROWB, &mapB, fb, kt * CF::TKC, 0, p,
                              zb_lo, uhi + f);
            }
          }
        }
        if (++s == NS) {
          s = 0;
          ++lap;
        }
      }
    }
    if (leader) drain_loads(full, NS, g, err);  // g = stages issued
    __syncwarp();
  } else if (warp == 1) {
    // ---- MMA issuer (the whole warp waits, one lane issues).  Chunk 0 of the
    // t-th tile goes to buffer t & 1, later chunks to the other one; the n-th
    // use of a buffer (n >= 1) waits for the epilogue's (n-1)-th release of it.
    const bool leader = elect_one();
    const uint32_t I = idesc2(bf16, TM, TN, false), IN = idesc2(bf16, TM, TN, true);
    const uint32_t smem0 = smem_u32(smem) >> 4;
    int64_t g = 0, t = 0;
    int s = 0;
    uint32_t ph = 0;
    uint32_t used[2] = {0u, 0u};
    bool ok = true;
    for (int64_t it = first; ok && it < items; it += stride, ++t) {
      if (__any_sync(0xffffffffu, abort_flag)) break;
      const int rb = (int)(t & 1);
      for (int c = 0; c < nch && ok; ++c) {
        const int b = c == 0 ? rb : 1 - rb;
        if (used[b] >= 1 && !mbar_wait_warp(&acc_empty[b], (used[b] - 1) & 1, wl)) {
          if (leader) {
            atomicExch(err, 32);
            abort_flag = 1;
          }
          ok = false;
          break;
        }
        ++used[b];
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        const uint32_t dr = tmem + (uint32_t)b * BUF, di = dr + TN;
        const int k0 = (PARTS ? (int)(it % parts) : c) * chunk, k1 = min(nkt, k0 + chunk);
        for (int kt = k0; kt < k1; ++kt, ++g) {
          if (!mbar_wait_warp(&full[s], ph, wl)) {
            if (leader) {
              atomicExch(err, 33);
              abort_flag = 1;
            }
            ok = false;
            break;
          }
          asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
          if (leader) {
            const uint32_t a = smem0 + (uint32_t)s * (CF::STAGE >> 4) + OperandDesc<ROWB, TM>::LO;
            const uint32_t b0 = smem0 + (uint32_t)s * (CF::STAGE >> 4) + (CF::A_STAGE >> 4) + OperandDesc<ROWB, TN>::LO;
#pragma unroll
            for (int kk = 0; kk < CF::KSTEPS; ++kk) {
              mma_step<NP, TN, ROWB>(dr, di, a, b0, kk, I, IN, (kt > k0 || kk) ? 1u : 0u);
            }
            commit(&empty[s]);
          }
          __syncwarp();
          if (++s == NS) {
            s = 0;
            ph ^= 1;
          }
        }
        if (leader) commit(&acc_full[b]);  // also after an abort, so the epilogue's wait ends
        __syncwarp();
      }
    }
    // every MMA issued has finished reading shared memory and writing TMEM
    // before this warp reaches the final barrier
    if (leader && g > 0) {
      commit(&mma_done);
      if (!mbar_wait(&mma_done, 0, kDrainLimit)) atomicExch(err, 36);
    }
    __syncwarp();
  } else if (warp >= 4) {
    // ---- epilogue: fold chunks 1.. into R; after the last one, store R.
    // Warp 4 + e reads TMEM lane quarter q = warp % 4 (the hardware's rule)
    // and, with eight epilogue warps, every other 16-column chunk (h).  The
    // warps share nothing but the accumulator barriers.  What bounds an
    // output-bound step here is the warps' instruction latency, so every
    // address is a sum of few terms set up once: shared-memory slots per
    // column, C offsets per read-back step, and per tile the offsets of its
    // upper row and column bits, each one warp sum over the bits' strides.
    // Measured against column offsets in a shared table behind barriers and
    // per-element scaling branches: 16-bit planes, (11, 10, 5) x 4096 units 20.1
    // -> 12.4 ms; four planes, (15, 9, 7) x 128 units 7.2 -> 5.3 ms; complex64,
    // (14, 14, 5) 832 -> 518 us.
    const int e = warp - 4, q = warp & 3, h = e >> 2;
    constexpr int CS = 16 * (EW / 4);  // column stride between a warp's chunks
    const uint32_t lane_off = (uint32_t)(q * 32) << 16;
    const bool planes = (out_flags & 1) != 0, wide = (out_flags & 2) != 0;
    const StageMap sm = stage_map(d, lane, planes, wide);
    const int vb = wide || planes ? vec_bits(d) : 0;
    // this lane's slots: the C-order index of (lane, jj) is lane_idx | (jj's
    // bits at their ranks); the two parts have disjoint bits, so their slots add
    const bool slot4 = NP == 2 && planes;  // 4-byte slots
    const uint32_t slots = smem_u32(smem + NS * CF::STAGE) + e * STAGE_SLOTS * 8;
    auto slot_of = [&](int idx) { return (uint32_t)(slot4 ? stage_slot4(idx) * 4 : stage_slot(idx) * 8); };
    uint32_t slot[16];
    {
      uint32_t cs[4];
      for (int b = 0; b < 4; ++b) cs[b] = slot_of(1 << sm.rank_c[b]);
#pragma unroll
      for (int jj = 0; jj < 16; ++jj)
        slot[jj] = slots + slot_of(sm.lane_idx) + ((jj & 1) ? cs[0] : 0) + ((jj & 2) ? cs[1] : 0) +
                   ((jj & 4) ? cs[2] : 0) + ((jj & 8) ? cs[3] : 0);
    }
    const uint32_t rd = slots + slot_of(planes ? 8 * lane : 2 * lane);
    int32_t back[8];  // C offset of this lane's piece in read-back step t
#pragma unroll
    for (int t = 0; t < 8; ++t)
      back[t] = planes ? sm.off_pl + ((t & 1) ? sm.step_pl : 0)
                       : sm.off_c64 + ((t & 1) ? sm.step_c64[0] : 0) + ((t & 2) ? sm.step_c64[1] : 0) +
                             ((t & 4) ? sm.step_c64[2] : 0);
    const int32_t lane_row = bit_offset(lane, 5, d.cm);  // direct stores: this lane's row
    const int32_t cn_lo[4] = {d.cn[0], d.cn[1], d.cn[2], d.cn[3]};
    // strides of the tile's row bits 5.. and column bits 7.. (lane b: bit b), and of column bits 4..6
    const int32_t my_cm = lane >= 5 && lane < d.nm ? d.cm[lane] : 0;
    const int32_t my_cn = lane >= 4 && lane < d.nn ? d.cn[lane] : 0;
    const int32_t cn_mid[3] = {d.nn > 4 ? d.cn[4] : 0, d.nn > 5 ? d.cn[5] : 0, d.nn > 6 ? d.cn[6] : 0};
    auto bit_sum = [&](int x, int32_t st) {
      return (int32_t)__reduce_add_sync(0xffffffffu, (uint32_t)(((x >> lane) & 1) ? st : 0));
    };
    const int64_t plane = int64_t(1) << (d.nm + d.nn);
    const int gw = fold > 1 ? nsub : TN;  // tile columns of one unit
    // maximum / filter tracking only where the formats need it
    const bool track = sio.mc != nullptr || sio.flag != nullptr;
    // Scaled formats: exponents of the operands of the tile's f-th unit (a
    // folded tile holds `fold` hi units side by side, f = column / 2^nn, with A
    // shared and B, C of their own) and the output shift r that keeps the
    // predicted bound 2 K maxA maxB below 2^15.
    float vmax[2] = {0.f, 0.f};
    bool weak = false;
    int ea = 0, eb = 0, r = 0, scaled_unit = -1;
    Pow2 sc(0);
    auto unit_scale = [&](int ulo, int uhi, int f) {
      const int un = ulo + (uhi + f) * d.units_lo;
      if (!sio.ea || un == scaled_unit) return;
      scaled_unit = un;
      const int za = (a_zlo ? ulo : 0) + (a_zhi ? uhi : 0) * (a_zlo ? d.units_lo : 1);
      const int zb = (b_zlo ? ulo : 0) + (b_zhi ? uhi + f : 0) * (b_zlo ? d.units_lo : 1);
      ea = sio.ea[za];
      eb = sio.eb[zb];
      const float ma = sio.ma[za], mb = sio.mb[zb];
      weak = !(ma >= 0x1p-10f) || !(mb >= 0x1p-10f);
      const float bound = 2.f * ldexpf(ma * mb, d.nk);
      r = 0;
      if (bound > 0.f && isfinite(bound)) {
        int x;
        frexpf(bound, &x);
        r = x - 15;
      }
      if (!PARTS) sc = Pow2(planes ? -r : ea + eb);
    };
    int64_t t = 0;
    uint32_t seen[2] = {0u, 0u};
    bool ok = true;
    for (int64_t it = first; ok && it < items; it += stride, ++t) {
      int unit, m0, n0, cp;
      decode(it, unit, m0, n0, cp);
      const int ulo = unit % d.units_lo, uhi = (unit / d.units_lo) * fold;
      unit_scale(ulo, uhi, 0);  // (loads in flight while the accumulator fills)
      float2* const Cu = PARTS ? part + (((int64_t)cp * d.units + unit) << (d.nm + d.nn))
                                   : C0 + ((int64_t)ulo * d.c_lo + (int64_t)uhi * d.c_hi);
      const int32_t tile_off = bit_sum(m0 + q * 32, my_cm) + (fold > 1 ? 0 : bit_sum(n0, my_cn));
      const int rb = (int)(t & 1);
      const uint32_t R = tmem + lane_off + (uint32_t)rb * BUF, P = tmem + lane_off + (uint32_t)(1 - rb) * BUF;
      for (int c = 0; c < nch; ++c) {
        const int b = c == 0 ? rb : 1 - rb;
        ok = mbar_wait_warp(&acc_full[b], seen[b] & 1, wl);
        ++seen[b];
        if (!ok) {
          if (lane == 0) {
            atomicExch(err, 34);
            abort_flag = 1;
          }
          break;
        }
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        if (c == 0) continue;  // the first chunk accumulated in R itself
#pragma unroll 1
        for (int c0 = 16 * h; c0 < TN; c0 += CS) {
          uint32_t pr[16], pi[16], rr[16], ri[16];
          tmem_ld<16>(P + (uint32_t)c0, pr);
          tmem_ld<16>(P + (uint32_t)(TN + c0), pi);
          tmem_ld<16>(R + (uint32_t)c0, rr);
          tmem_ld<16>(R + (uint32_t)(TN + c0), ri);
          asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
          for (int jj = 0; jj < 16; ++jj) {
            rr[jj] = __float_as_uint(__uint_as_float(rr[jj]) + __uint_as_float(pr[jj]));
            ri[jj] = __float_as_uint(__uint_as_float(ri[jj]) + __uint_as_float(pi[jj]));
          }
          tmem_st16(R + (uint32_t)c0, rr);
          tmem_st16(R + (uint32_t)(TN + c0), ri);
        }
        // R complete before it is read again; P free for the next chunk
        asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
        asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
        asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(&acc_empty[1 - rb])) : "memory");
      }
      if (!ok) break;
#pragma unroll 1
      for (int c0 = 16 * h; c0 < TN; c0 += CS) {
        // columns of a folded tile belong to hi unit uhi + c0 / 2^nn (N >= 16:
        // a 16-column chunk never straddles two units); the warp's first and
        // last chunks among a unit's gw columns open and close its records
        const int f = fold > 1 ? (c0 >> d.nn) : 0;
        if (c0 % gw < CS) {
          if (f > 0) unit_scale(ulo, uhi, f);
          vmax[0] = vmax[1] = 0.f;
        }
        uint32_t ur[16], ui[16];
        tmem_ld<16>(R + (uint32_t)c0, ur);
        tmem_ld<16>(R + (uint32_t)(TN + c0), ui);
        const int cc = fold > 1 ? (c0 & (nsub - 1)) : c0;
        float2* const C = Cu + (int64_t)f * d.c_hi;
        const int32_t off = tile_off + ((cc & 16) ? cn_mid[0] : 0) + ((cc & 32) ? cn_mid[1] : 0) +
                            ((cc & 64) ? cn_mid[2] : 0);
        asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
        if (c0 + CS >= TN) {
          // R read out: the MMA warp may start a later tile's chunks in it
          asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
          asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(&acc_empty[rb])) : "memory");
        }
        float vr[16], vi[16];
        if (sc.direct) {
#pragma unroll
          for (int jj = 0; jj < 16; jj += 2) {
            mul_pair(ur[jj], ur[jj + 1], sc.f, vr[jj], vr[jj + 1]);
            mul_pair(ui[jj], ui[jj + 1], sc.f, vi[jj], vi[jj + 1]);
          }
        } else {
#pragma unroll
          for (int jj = 0; jj < 16; ++jj) {
            vr[jj] = ldexpf(__uint_as_float(ur[jj]), sc.e);
            vi[jj] = ldexpf(__uint_as_float(ui[jj]), sc.e);
          }
        }
        if (planes) {
          uint16_t* const Pl = reinterpret_cast<uint16_t*>(C) + off;
          if (track) {
            // (two chains; a NaN passes through to the maximum, so a unit whose
            // values turned non-finite ends with an infinity or a NaN)
#pragma unroll
            for (int jj = 0; jj < 16; ++jj) vmax[jj & 1] = max_nan(vmax[jj & 1], max_nan(fabsf(vr[jj]), fabsf(vi[jj])));
          }
          uint32_t x[NP / 2][16];
          auto pack = [&](bool fmt) {
#pragma unroll
            for (int jj = 0; jj < 16; ++jj) {
              uint32_t y[NP / 2];
              pack_planes<NP>(fmt, vr[jj], vi[jj], y);
#pragma unroll
              for (int u = 0; u < NP / 2; ++u) x[u][jj] = y[u];
            }
          };
          if (bf16) pack(true);
          else pack(false);
          if (sm.on) {
            // planes of one element packed in one slot (4 NP / 2 bytes), in C order
#pragma unroll
            for (int jj = 0; jj < 16; ++jj) {
              if constexpr (NP == 4) sts64(slot[jj], x[0][jj], x[1][jj]);
              else sts32(slot[jj], x[0][jj]);
            }
            __syncwarp();
            uint4 y2[2][NP];  // C-order values 8 (lane + 32 t2) .. + 7, one slot each
#pragma unroll
            for (int t2 = 0; t2 < 2; ++t2)
#pragma unroll
              for (int u = 0; u < NP; ++u)
                y2[t2][u] = lds128(rd + 16 * u + t2 * (NP == 4 ? (256 + 32) * 8 : (256 + 32) * 4));
#pragma unroll
            for (int t2 = 0; t2 < 2; ++t2) {
              uint32_t v[NP / 2][8];
#pragma unroll
              for (int u = 0; u < NP; ++u) {
                const uint4 y = y2[t2][u];
                if constexpr (NP == 4) {
                  v[0][2 * u] = y.x;
                  v[NP / 2 - 1][2 * u] = y.y;
                  v[0][2 * u + 1] = y.z;
                  v[NP / 2 - 1][2 * u + 1] = y.w;
                } else {
                  v[0][4 * u] = y.x;
                  v[0][4 * u + 1] = y.y;
                  v[0][4 * u + 2] = y.z;
                  v[0][4 * u + 3] = y.w;
                }
              }
#pragma unroll
              for (int pl = 0; pl < NP; ++pl) {
                auto pp = [&](int e0) {
                  return __byte_perm(v[pl >> 1][e0], v[pl >> 1][e0 + 1], (pl & 1) ? 0x7632 : 0x5410);
                };
                *reinterpret_cast<uint4*>(Pl + pl * plane + back[t2]) = make_uint4(pp(0), pp(2), pp(4), pp(6));
              }
            }
            __syncwarp();
          } else {
            store_planes<NP>(Pl + lane_row, plane, cn_lo, vb, x);
          }
        } else if (sm.on) {
#pragma unroll
          for (int jj = 0; jj < 16; ++jj) sts64(slot[jj], __float_as_uint(vr[jj]), __float_as_uint(vi[jj]));
          __syncwarp();
          float2* const Co = C + off;
          uint4 y[8];  // C-order values 2 (lane + 32 t2) and the next one: two adjacent slots
#pragma unroll
          for (int t2 = 0; t2 < 8; ++t2) y[t2] = lds128(rd + t2 * (64 + 8) * 8);
#pragma unroll
          for (int t2 = 0; t2 < 8; ++t2) *reinterpret_cast<uint4*>(Co + back[t2]) = y[t2];
          __syncwarp();
        } else {
          float2* const Co = C + off + lane_row;
#pragma unroll
          for (int jj = 0; jj < 16; ++jj) Co[col_offset(cn_lo, jj)] = make_float2(vr[jj], vi[jj]);
        }
        if (c0 % gw + CS >= gw && track) {
          // the unit's columns are done: its largest stored component,
          // exponent and filter flag (launch unit ulo + (uhi + f) units_lo)
          const int un = fold > 1 ? ulo + (uhi + f) * d.units_lo : unit;
          // (as unsigned bits NaN > infinity > any finite value)
          const float wmax = __uint_as_float(
              __reduce_max_sync(0xffffffffu, max(__float_as_uint(vmax[0]), __float_as_uint(vmax[1]))));
          const bool bad = planes && !(wmax < __int_as_float(0x7f800000));
          if (lane == 0) {
            if (sio.mc && planes) atomicMax(sio.mc + un, __float_as_uint(wmax));
            if (sio.ec && planes && q == 0 && m0 == 0 && n0 == 0) sio.ec[un] = ea + eb + r;
            if (sio.flag && (bad || weak)) sio.flag[sio.flag_by_lo ? ulo : un] = 1;
          }
        }
      }
    }
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  if (warp == 2) {
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(COLS));
  }
}

// The same GEMM with A read as complex64 (one unit, N <= 64: one column tile,
// so A is needed once).  Writing A's planes first and reading them back would
// move three times its bytes, and here A is nearly all the bytes.  So the eight
// epilogue warps also prepare A's stages: they load the 128 x 32 tile front to
// back in A's own order (the tile holds A's fastest indices, order_for_direct),
// turn it in shared memory, convert it as the split pass does and write the
// swizzled plane rows, with two stages' loads in flight in registers.  Warp 0
// copies B's planes by TMA, warp 1 issues the MMAs.
//
// TMEM holds the running sum R (buffer 0) and two partial buffers, so the chunk
// of K that the workers are converting never waits for the previous chunk's
// fold, which they do after it.  The workers decide together, at each stage's
// barrier, whether one of them gave up a wait.
constexpr int DTK = 32;                         // complex K per stage
constexpr int RAW_BYTES = TM * DTK * 8;         // a stage's tile as complex64
template <int TN, int NP>
struct DirectCfg {
  using CF = Cfg2<TN, NP, 64>;
  static constexpr int THREADS = 128 + 256;
  static constexpr int BUDGET = 227 * 1024 - 2 * RAW_BYTES - 1024 - 2048;
  static constexpr int NS = (BUDGET / CF::STAGE) < 4 ? (BUDGET / CF::STAGE) : 4;
  static constexpr int SMEM = NS * CF::STAGE + 2 * RAW_BYTES + 1024;
  static constexpr uint32_t BUF = 2 * TN;       // TMEM columns of one buffer
  static constexpr uint32_t COLS = TN == 64 ? 512 : TN == 32 ? 256 : 128;
  static_assert(NS >= 2 && 3 * BUF <= COLS, "two stages, three accumulator buffers");
  static_assert(8 * STAGE_SLOTS * 8 <= 2 * RAW_BYTES, "the output staging reuses the raw tiles");
};

// The tile's index bits (K bits 0..4, then row bits 0..6 of the descriptor) in
// A's order: stride and shared slot; and the slots in tile order.
// in_off, in_put: the sums over A's order bits 9..11.
struct DirectMap {
  int32_t in_src[12], in_slot[12], out_slot[12];
  int32_t in_off[8], in_put[8];
};

__device__ __forceinline__ bool workers_any(bool failed) {  // barrier of the 256 workers
  uint32_t r;
  asm volatile(
      "{\n .reg .pred p, q;\n setp.ne.u32 p, %1, 0;\n barrier.cta.red.or.pred q, 1, 256, p;\n selp.u32 %0, 1, 0, q;\n}\n"
      : "=r"(r)
      : "r"((uint32_t)failed)
      : "memory");
  return r != 0;
}

template <int TN, int NP, bool BF16>
__global__ void __launch_bounds__(DirectCfg<TN, NP>::THREADS, 1)
    gemm_direct(const __grid_constant__ CUtensorMap mapB, const float2* A, float2* __restrict__ C,
                const GemmDesc d, const __grid_constant__ DirectMap dm, const unsigned* maxA,
                const int* exp_b, int a_vec, int out_wide, int chunk, int* __restrict__ err) {
  using DC = DirectCfg<TN, NP>;
  using CF = typename DC::CF;
  constexpr int NS = DC::NS;
  constexpr uint32_t BUF = DC::BUF;
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = (uint8_t*)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
  float2* const raw = reinterpret_cast<float2*>(smem + NS * CF::STAGE);  // [2][4096]
  __shared__ uint64_t full_a[NS], full_b[NS], empty[NS], acc_full[3], acc_empty[3], mma_done;
  __shared__ uint32_t tmem_slot;
  __shared__ volatile int abort_flag;

  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const long long wl = g_wait_limit;
  const int items = 1 << (d.nm - 7), first = blockIdx.x, stride = gridDim.x;
  const int nkt = 1 << (d.nk - 5);
  const int nch = (nkt + chunk - 1) / chunk;

  if (tid == 0) {
    for (int s = 0; s < NS; ++s) {
      mbar_init(&full_a[s], 8);
      mbar_init(&full_b[s], 1);
      mbar_init(&empty[s], 1);
    }
    for (int b = 0; b < 3; ++b) {
      mbar_init(&acc_full[b], 1);
      mbar_init(&acc_empty[b], 8);
    }
    mbar_init(&mma_done, 1);
    abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(&mapB)) : "memory");
  }
  if (warp == 2) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_slot)),
                 "r"(DC::COLS));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tmem = tmem_slot;
  let_next_start();
  after_previous();

  if (warp == 0) {
    // ---- B's stages
    const bool leader = elect_one();
    int64_t g = 0;
    int s = 0;
    uint32_t lap = 0;
    bool ok = true;
    for (int it = first; ok && it < items; it += stride) {
      if (__any_sync(0xffffffffu, abort_flag)) break;
      for (int kt = 0; kt < nkt; ++kt, ++g) {
        if (lap > 0 && !mbar_wait_warp(&empty[s], (lap - 1) & 1, wl)) {
          if (leader) {
            atomicExch(err, 41);
            abort_flag = 1;
          }
          ok = false;
          break;
        }
        if (leader) {
          mbar_expect_tx(&full_b[s], NP * CF::B_PLANE);
          tma_load_5d(smem + s * CF::STAGE + CF::A_STAGE, &mapB, &full_b[s], kt * DTK, 0, 0, 0, 0);
        }
        if (++s == NS) {
          s = 0;
          ++lap;
        }
      }
    }
    if (leader) drain_loads(full_b, NS, g, err);
    __syncwarp();
  } else if (warp == 1) {
    // ---- MMA issuer: chunk 0 of a tile into buffer 0, later ones into 1 and 2 in turn
    const bool leader = elect_one();
    constexpr uint32_t I = idesc2(BF16, TM, TN, false), IN = idesc2(BF16, TM, TN, true);
    const uint32_t smem0 = smem_u32(smem) >> 4;
    int64_t g = 0;
    int s = 0;
    uint32_t ph = 0;
    uint32_t used[3] = {0u, 0u, 0u};
    bool ok = true;
    for (int it = first; ok && it < items; it += stride) {
      if (__any_sync(0xffffffffu, abort_flag)) break;
      for (int c = 0; c < nch && ok; ++c) {
        const int b = c == 0 ? 0 : 1 + ((c - 1) & 1);
        if (used[b] >= 1 && !mbar_wait_warp(&acc_empty[b], (used[b] - 1) & 1, wl)) {
          if (leader) {
            atomicExch(err, 42);
            abort_flag = 1;
          }
          ok = false;
          break;
        }
        ++used[b];
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        const uint32_t dr = tmem + (uint32_t)b * BUF, di = dr + TN;
        const int k0 = c * chunk, k1 = min(nkt, k0 + chunk);
        for (int kt = k0; kt < k1; ++kt, ++g) {
          if (!mbar_wait_warp(&full_b[s], ph, wl) || !mbar_wait_warp(&full_a[s], ph, wl)) {
            if (leader) {
              atomicExch(err, 43);
              abort_flag = 1;
            }
            ok = false;
            break;
          }
          asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
          if (leader) {
            const uint32_t a = smem0 + (uint32_t)s * (CF::STAGE >> 4) + OperandDesc<64, TM>::LO;
            const uint32_t b0 = smem0 + (uint32_t)s * (CF::STAGE >> 4) + (CF::A_STAGE >> 4) + OperandDesc<64, TN>::LO;
#pragma unroll
            for (int kk = 0; kk < CF::KSTEPS; ++kk)
              mma_step<NP, TN, 64>(dr, di, a, b0, kk, I, IN, (kt > k0 || kk) ? 1u : 0u);
            commit(&empty[s]);
          }
          __syncwarp();
          if (++s == NS) {
            s = 0;
            ph ^= 1;
          }
        }
        if (leader) commit(&acc_full[b]);
        __syncwarp();
      }
    }
    if (leader && g > 0) {
      commit(&mma_done);
      if (!mbar_wait(&mma_done, 0, kDrainLimit)) atomicExch(err, 46);
    }
    __syncwarp();
  } else if (warp >= 4) {
    // ---- workers
    const int t = tid - 128, w = warp - 4, q = warp & 3, h = w >> 2;
    int ea = 0;
    if (maxA) ea = scale_exponent(__uint_as_float(*maxA));
    const Pow2 sa(-ea), sc(ea + (exp_b ? *exp_b : 0));
    // loads: pairs t + 256 j of A-adjacent elements; A's order bits 1..8 from t, 9..11 from j
    int32_t so = 0, slot = 0;
#pragma unroll
    for (int b = 0; b < 8; ++b)
      if ((t >> b) & 1) {
        so += dm.in_src[1 + b];
        slot ^= dm.in_slot[1 + b];
      }
    const int32_t my_am = lane >= 7 && lane < d.nm ? d.am[lane] : 0;
    const int32_t my_ak = lane >= 5 && lane < d.nk ? d.ak[lane] : 0;
    auto bit_sum = [&](int x, int32_t st) {
      return (int32_t)__reduce_add_sync(0xffffffffu, (uint32_t)(((x >> lane) & 1) ? st : 0));
    };
    // two stages' loads in flight: one stage ahead left an SM waiting for their
    // latency, 2 us per 32 KB stage
    float4 pf0[8], pf1[8];
    auto load = [&](float4(&pf)[8], int it, int kt) {
      const float2* src = A + so + bit_sum(it << 7, my_am) + bit_sum(kt << 5, my_ak);
#pragma unroll
      for (int j = 0; j < 8; ++j) {
        const float2* p = src + dm.in_off[j];
        if (a_vec) {
          pf[j] = *reinterpret_cast<const float4*>(p);
        } else {
          const float2 x = p[0], y = p[1];
          pf[j] = make_float4(x.x, x.y, y.x, y.y);
        }
      }
    };
    // conversions: K octets t and t + 256 of the tile: octet o = row o / 4, K chunk
    // o % 4, i.e. rows t / 4 and t / 4 + 64, whose swizzles agree
    const int oplace = (t >> 2) * 64 + (((t & 3) ^ ((t >> 3) & 3)) << 4);
    int32_t oslot[2];
#pragma unroll
    for (int u = 0; u < 2; ++u) {
      oslot[u] = 0;
#pragma unroll
      for (int b = 0; b < 9; ++b)
        if (((t + 256 * u) >> b) & 1) oslot[u] ^= dm.out_slot[3 + b];
    }
    const uint32_t tq = tmem + ((uint32_t)(q * 32) << 16);
    uint32_t seen[3] = {0u, 0u, 0u};
    bool failed = false, stop = false;
    auto wait_acc = [&](int b) {
      if (!mbar_wait_warp(&acc_full[b], seen[b] & 1, wl)) {
        failed = true;
        if (lane == 0) {
          atomicExch(err, 44);
          abort_flag = 1;
        }
      }
      ++seen[b];
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    };
    auto release = [&](int b) {
      asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
      __syncwarp();
      if (lane == 0) asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(&acc_empty[b])) : "memory");
    };
    auto fold = [&](int c) {
      const int b = 1 + ((c - 1) & 1);
      if (c == 1) wait_acc(0);
      wait_acc(b);
      if (failed) return;
      const uint32_t R = tq, P = tq + (uint32_t)b * BUF;
#pragma unroll 1
      for (int c0 = 16 * h; c0 < TN; c0 += 32) {
        uint32_t pr[16], pi[16], rr[16], ri[16];
        tmem_ld<16>(P + (uint32_t)c0, pr);
        tmem_ld<16>(P + (uint32_t)(TN + c0), pi);
        tmem_ld<16>(R + (uint32_t)c0, rr);
        tmem_ld<16>(R + (uint32_t)(TN + c0), ri);
        asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
        for (int jj = 0; jj < 16; ++jj) {
          rr[jj] = __float_as_uint(__uint_as_float(rr[jj]) + __uint_as_float(pr[jj]));
          ri[jj] = __float_as_uint(__uint_as_float(ri[jj]) + __uint_as_float(pi[jj]));
        }
        tmem_st16(R + (uint32_t)c0, rr);
        tmem_st16(R + (uint32_t)(TN + c0), ri);
      }
      asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
      release(b);
    };
    int s = 0;
    uint32_t lap = 0;
    int64_t g = 0;
    // the load position: two stages past the one being converted
    int lit = first, lkt = 0;
    auto load_next = [&](float4(&pf)[8]) {
      if (lit >= items) return;
      load(pf, lit, lkt);
      if (++lkt == nkt) {
        lkt = 0;
        lit += stride;
      }
    };
    load_next(pf0);
    load_next(pf1);
    for (int it = first; !stop && it < items; it += stride) {
      for (int c = 0; c < nch && !stop; ++c) {
        const int k1 = min(nkt, (c + 1) * chunk);
        for (int kt = c * chunk; kt < k1; ++kt, ++g) {
          float2* const tile = raw + (g & 1) * (TM * DTK);
          auto land = [&](float4(&pf)[8]) {
#pragma unroll
            for (int j = 0; j < 8; ++j) {
              const int32_t p = slot ^ dm.in_put[j];
              tile[p] = make_float2(pf[j].x, pf[j].y);
              tile[p ^ dm.in_slot[0]] = make_float2(pf[j].z, pf[j].w);
            }
            load_next(pf);
          };
          if (g & 1) land(pf1);
          else land(pf0);
          if (lap > 0 && !failed && !mbar_wait_warp(&empty[s], (lap - 1) & 1, wl)) {
            failed = true;
            if (lane == 0) {
              atomicExch(err, 45);
              abort_flag = 1;
            }
          }
          // the tile is complete and its stage free; or everyone stops
          if (workers_any(failed)) {
            stop = true;
            break;
          }
          uint8_t* const st = smem + s * CF::STAGE;
          // (the shift is a single multiply but for exponents out of range)
          auto convert = [&](auto scale) {
#pragma unroll
            for (int u = 0; u < 2; ++u) {
              f32x2 x[8];
#pragma unroll
              for (int v = 0; v < 4; ++v) {
                const ulonglong2 y = *reinterpret_cast<const ulonglong2*>(&tile[oslot[u] ^ (2 * v)]);
                x[2 * v] = scale(y.x);
                x[2 * v + 1] = scale(y.y);
              }
              uint4 p[NP];
              planes8<NP, BF16>(x, p);
              // 64-byte rows, 16-byte chunks swizzled by row bits 1, 2
#pragma unroll
              for (int i = 0; i < NP; ++i) *reinterpret_cast<uint4*>(st + oplace + u * 64 * 64 + i * CF::A_PLANE) = p[i];
            }
          };
          if (sa.direct && sa.f == 1.f) {
            convert([](f32x2 y) { return y; });
          } else if (sa.direct) {
            const f32x2 f = pack2(sa.f, sa.f);
            convert([&](f32x2 y) { return mul2(y, f); });
          } else {
            convert([&](f32x2 y) {
              const float2 v = unpack2(y);
              return pack2(sa(v.x), sa(v.y));
            });
          }
          asm volatile("fence.proxy.async.shared::cta;" ::: "memory");  // visible to the tensor core's reads
          __syncwarp();
          if (lane == 0) asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(&full_a[s])) : "memory");
          if (++s == NS) {
            s = 0;
            ++lap;
          }
        }
        if (!stop && c >= 2) fold(c - 1);
      }
      if (stop) break;
      if (nch >= 2) fold(nch - 1);
      else wait_acc(0);
      // every worker is done with the raw tiles, whose memory now stages the output
      if (workers_any(failed)) break;
      // output addressing, as in gemm_tma_chunked (set up per tile: it would hold
      // registers that the loads need)
      const StageMap sm = stage_map(d, lane, false, out_wide != 0);
      const uint32_t slots = smem_u32(raw) + w * STAGE_SLOTS * 8;
      uint32_t cslot[4];
      for (int b = 0; b < 4; ++b) cslot[b] = (uint32_t)stage_slot(1 << sm.rank_c[b]) * 8;
      const uint32_t lslot = slots + (uint32_t)stage_slot(sm.lane_idx) * 8;
      const uint32_t rd = slots + (uint32_t)stage_slot(2 * lane) * 8;
      const int32_t lane_row = bit_offset(lane, 5, d.cm);
      const int32_t cn_lo[4] = {d.cn[0], d.cn[1], d.cn[2], d.cn[3]};
      const int32_t cn_mid[2] = {d.nn > 4 ? d.cn[4] : 0, d.nn > 5 ? d.cn[5] : 0};
      const int32_t my_cm = lane >= 5 && lane < d.nm ? d.cm[lane] : 0;
      const int32_t tile_off = bit_sum((it << 7) + q * 32, my_cm);
#pragma unroll 1
      for (int c0 = 16 * h; c0 < TN; c0 += 32) {
        uint32_t ur[16], ui[16];
        tmem_ld<16>(tq + (uint32_t)c0, ur);
        tmem_ld<16>(tq + (uint32_t)(TN + c0), ui);
        float2* const Co = C + (tile_off + ((c0 & 16) ? cn_mid[0] : 0) + ((c0 & 32) ? cn_mid[1] : 0));
        asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
        float vr[16], vi[16];
        if (sc.direct) {
#pragma unroll
          for (int jj = 0; jj < 16; jj += 2) {
            mul_pair(ur[jj], ur[jj + 1], sc.f, vr[jj], vr[jj + 1]);
            mul_pair(ui[jj], ui[jj + 1], sc.f, vi[jj], vi[jj + 1]);
          }
        } else {
#pragma unroll
          for (int jj = 0; jj < 16; ++jj) {
            vr[jj] = sc(__uint_as_float(ur[jj]));
            vi[jj] = sc(__uint_as_float(ui[jj]));
          }
        }
        if (sm.on) {
#pragma unroll
          for (int jj = 0; jj < 16; ++jj)
            sts64(lslot + ((jj & 1) ? cslot[0] : 0) + ((jj & 2) ? cslot[1] : 0) + ((jj & 4) ? cslot[2] : 0) +
                      ((jj & 8) ? cslot[3] : 0),
                  __float_as_uint(vr[jj]), __float_as_uint(vi[jj]));
          __syncwarp();
          uint4 y[8];
#pragma unroll
          for (int t2 = 0; t2 < 8; ++t2) y[t2] = lds128(rd + t2 * (64 + 8) * 8);
#pragma unroll
          for (int t2 = 0; t2 < 8; ++t2)
            *reinterpret_cast<uint4*>(Co + sm.off_c64 + ((t2 & 1) ? sm.step_c64[0] : 0) +
                                      ((t2 & 2) ? sm.step_c64[1] : 0) + ((t2 & 4) ? sm.step_c64[2] : 0)) = y[t2];
          __syncwarp();
        } else {
#pragma unroll
          for (int jj = 0; jj < 16; ++jj) Co[lane_row + col_offset(cn_lo, jj)] = make_float2(vr[jj], vi[jj]);
        }
      }
      release(0);
      if (workers_any(failed)) break;  // the raw tiles' memory is free again
    }
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  if (warp == 2) {
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(DC::COLS));
  }
}

// C = the chunks' sums added in order, times 2^(eA + eB): the folds and the
// scaling of gemm_tma_chunked for items that were one chunk each, with the same
// additions in the same order.  Bound by the sums' trip through L2 (they were
// written microseconds before; at most 256 MB).
__global__ void __launch_bounds__(256) combine_kernel(const float2* part, int parts, float2* __restrict__ C,
                                                      const GemmDesc d, const ScaleIO sio, int a_zlo, int a_zhi,
                                                      int b_zlo, int b_zhi) {
  let_next_start();
  after_previous();
  const int unit = blockIdx.y, ulo = unit % d.units_lo, uhi = unit / d.units_lo;
  int e = 0;
  if (sio.ea)
    e = sio.ea[(a_zlo ? ulo : 0) + (a_zhi ? uhi : 0) * (a_zlo ? d.units_lo : 1)] +
        sio.eb[(b_zlo ? ulo : 0) + (b_zhi ? uhi : 0) * (b_zlo ? d.units_lo : 1)];
  const Pow2 sc(e);
  const int64_t n = int64_t(1) << (d.nm + d.nn);
  const int64_t i = (int64_t)blockIdx.x * 256 + threadIdx.x;  // n is a multiple of 256
  const float2* p = part + unit * n + i;
  float2 s = p[0];
#pragma unroll 4
  for (int c = 1; c < parts; ++c) {
    const float2 x = p[(int64_t)c * d.units * n];
    s.x += x.x;
    s.y += x.y;
  }
  C[(int64_t)ulo * d.c_lo + (int64_t)uhi * d.c_hi + i] = make_float2(sc(s.x), sc(s.y));
}

PFN_cuTensorMapEncodeTiled_v12000 encode_fn() {
  static PFN_cuTensorMapEncodeTiled_v12000 fn = nullptr;
  static std::once_flag once;
  std::call_once(once, [] {
    void* p = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) ==
            cudaSuccess &&
        q == cudaDriverEntryPointSuccess)
      fn = (PFN_cuTensorMapEncodeTiled_v12000)p;
  });
  return fn;
}

// 5-D map over one operand's planes: [hi unit][lo unit][plane][row][k] of
// 16-bit values; box = row_bytes / 2 k x box_rows x box_planes x 1 x 1
// (box_planes 0: all np planes; row > 0: rows of that many bytes).  A plane row holds K >= 8 values (16 bytes or
// more); when K = 8 the box reaches past it and the copy fills those K positions with
// zeros (the other operand's are zero as well, so the products vanish), and
// the stage still receives the box's full byte count.
bool encode_planes(CUtensorMap* map, const PlaneOperand& o, int box_rows, int box_planes = 0, int row = 0) {
  auto fn = encode_fn();
  if (!fn) return false;
  const int64_t set = (int64_t)o.np * o.rows * o.kp * 2;  // bytes of one plane set
  cuuint64_t dims[5] = {(cuuint64_t)o.kp, (cuuint64_t)o.rows, (cuuint64_t)o.np, (cuuint64_t)o.nlo, (cuuint64_t)o.nhi};
  cuuint64_t strides[4] = {(cuuint64_t)(o.kp * 2), (cuuint64_t)(o.rows * o.kp * 2),
                           (cuuint64_t)(o.nlo > 1 ? o.st_lo : set), (cuuint64_t)(o.nhi > 1 ? o.st_hi : set)};
  const int rowb = row > 0 ? row : row_bytes(o.kp, o.np);
  cuuint32_t box[5] = {(cuuint32_t)(rowb / 2), (cuuint32_t)box_rows, (cuuint32_t)(box_planes > 0 ? box_planes : o.np), 1, 1};
  cuuint32_t estr[5] = {1, 1, 1, 1, 1};
  CUresult r = fn(map, CU_TENSOR_MAP_DATA_TYPE_UINT16, 5, const_cast<uint16_t*>(o.base), dims, strides, box, estr,
                  CU_TENSOR_MAP_INTERLEAVE_NONE,
                  rowb == 128  ? CU_TENSOR_MAP_SWIZZLE_128B
                  : rowb == 64 ? CU_TENSOR_MAP_SWIZZLE_64B
                               : CU_TENSOR_MAP_SWIZZLE_32B,
                  CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                  CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  return r == CUDA_SUCCESS;
}

// SM count of the current device (one CTA per SM for the persistent kernels).
int sm_count() {
  static std::atomic<int> known[64] = {};
  int dev = 0, sms = 0;
  cudaGetDevice(&dev);
  const bool keep = dev >= 0 && dev < 64;
  if (keep) sms = known[dev].load(std::memory_order_relaxed);
  if (sms > 0) return sms;
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  if (keep && sms > 0) known[dev].store(sms, std::memory_order_relaxed);
  return sms > 0 ? sms : 148;
}

template <int TN, int NP, int ROWB, int EW, bool PARTS>
cudaError_t launch_chunked_ew(const CUtensorMap& ma, const CUtensorMap& mb, float2* C, const GemmDesc& d, int kp,
                              const int z[4], int out_flags, const ScaleIO& sio, int fold, bool bf16, int* err,
                              cudaStream_t s, const BulkPlanes& ba, const BulkPlanes& bb, int parts, float2* part) {
  using CC = ChunkCfg<TN, NP, ROWB, EW>;
  static PerDevice once;
  const cudaError_t e = allow_smem(once, gemm_tma_chunked<TN, NP, ROWB, EW, PARTS>, CC::SMEM);
  if (e != cudaSuccess) return e;
  const int64_t M = int64_t(1) << d.nm, N = int64_t(1) << d.nn;
  const int64_t items = (M / TM) * (fold > 1 ? 1 : N / TN) * (d.units / fold) * parts;
  const int chunk = NP == 4 ? split_chunk() : 1 << 30;
  const unsigned grid = (unsigned)std::min<int64_t>(items, sm_count());
  return launch_overlapped(gemm_tma_chunked<TN, NP, ROWB, EW, PARTS>, dim3(grid), dim3(CC::THREADS), CC::SMEM, s, ma,
                           mb, C, d, kp, z[0], z[1], z[2], z[3], out_flags, sio, chunk, fold, bf16, err, ba, bb, parts, part);
}

// Eight epilogue warps where the epilogue dominates a tile (a short K, at
// most four operand stages, and tiles of 64 or 128 columns: each warp then
// still has two or more column chunks per tile), four where the main loop
// does and the extra operand stage matters.
template <int TN, int NP>
cudaError_t launch_chunked(const CUtensorMap& ma, const CUtensorMap& mb, float2* C, const GemmDesc& d, int kp,
                           const int z[4], int out_flags, const ScaleIO& sio, int fold, bool bf16, int* err,
                           cudaStream_t s, const BulkPlanes& ba, const BulkPlanes& bb, int parts, float2* part) {
  constexpr int EWS = TN >= 64 ? 8 : 4;  // a single K stage or a few
  using std::integral_constant;
  auto run = [&](auto rowb, auto ew, auto p) {
    return launch_chunked_ew<TN, NP, decltype(rowb)::value, decltype(ew)::value, decltype(p)::value>(
        ma, mb, C, d, kp, z, out_flags, sio, fold, bf16, err, s, ba, bb, parts, part);
  };
  auto go = [&](auto rowb, auto ew) { return run(rowb, ew, integral_constant<bool, false>{}); };
  if (ba.base) return go(integral_constant<int, K8_ROWB>{}, integral_constant<int, EWS>{});
  const int rowb = row_bytes(kp, NP);
  if (rowb == 32) return go(integral_constant<int, 32>{}, integral_constant<int, EWS>{});
  constexpr int WIDE = NP == 4 ? 64 : 128;
  if constexpr (WIDE == 128)
    if (rowb == 64) return go(integral_constant<int, 64>{}, integral_constant<int, EWS>{});
  // (chunks as items, two or more: a K of several stages, at any chunk length)
  if constexpr (NP == 4)
    if (parts > 1) return run(integral_constant<int, WIDE>{}, integral_constant<int, 4>{}, integral_constant<bool, true>{});
  if (EWS == 8 && kp <= 4 * (WIDE / 2)) return go(integral_constant<int, WIDE>{}, integral_constant<int, EWS>{});
  return go(integral_constant<int, WIDE>{}, integral_constant<int, 4>{});
}

template <int NP>
cudaError_t launch_tn(int TNv, const CUtensorMap& ma, const CUtensorMap& mb, float2* C, const GemmDesc& d, int kp,
                      const int z[4], int cp, const ScaleIO& sio, int fold, bool bf16, int* err, cudaStream_t s,
                      const BulkPlanes& ba, const BulkPlanes& bb, int parts, float2* part) {
  switch (TNv) {
    case 128: return launch_chunked<128, NP>(ma, mb, C, d, kp, z, cp, sio, fold, bf16, err, s, ba, bb, parts, part);
    case 64: return launch_chunked<64, NP>(ma, mb, C, d, kp, z, cp, sio, fold, bf16, err, s, ba, bb, parts, part);
    case 32: return launch_chunked<32, NP>(ma, mb, C, d, kp, z, cp, sio, fold, bf16, err, s, ba, bb, parts, part);
    case 16: return launch_chunked<16, NP>(ma, mb, C, d, kp, z, cp, sio, fold, bf16, err, s, ba, bb, parts, part);
    default: return cudaErrorInvalidValue;
  }
}

DirectMap direct_map(const GemmDesc& d) {
  DirectMap m{};
  int32_t st[12];
  for (int b = 0; b < 12; ++b) st[b] = b < 5 ? d.ak[b] : d.am[b - 5];
  int order[12];  // tile bits by A stride
  for (int i = 0; i < 12; ++i) {
    int j = i;
    for (; j > 0 && st[order[j - 1]] > st[i]; --j) order[j] = order[j - 1];
    order[j] = i;
  }
  turn_slots<12>(order, m.out_slot);
  for (int l = 0; l < 12; ++l) {
    m.in_src[l] = st[order[l]];
    m.in_slot[l] = m.out_slot[order[l]];
  }
  for (int j = 0; j < 8; ++j)
    for (int b = 0; b < 3; ++b)
      if ((j >> b) & 1) {
        m.in_off[j] += m.in_src[9 + b];
        m.in_put[j] ^= m.in_slot[9 + b];
      }
  return m;
}

template <int TN, int NP, bool BF16>
cudaError_t launch_direct_as(const CUtensorMap& mb, const float2* A, float2* C, const GemmDesc& d, const unsigned* maxA,
                             const int* exp_b, int* err, cudaStream_t s) {
  using DC = DirectCfg<TN, NP>;
  static PerDevice once;
  const cudaError_t e = allow_smem(once, gemm_direct<TN, NP, BF16>, DC::SMEM);
  if (e != cudaSuccess) return e;
  const unsigned grid = (unsigned)std::min<int64_t>(int64_t(1) << (d.nm - 7), sm_count());
  const int chunk = NP == 4 ? split_chunk() : 1 << 30;
  const int av = (reinterpret_cast<uintptr_t>(A) & 15) == 0, cv = (reinterpret_cast<uintptr_t>(C) & 15) == 0;
  return launch_overlapped(gemm_direct<TN, NP, BF16>, dim3(grid), dim3(DC::THREADS), DC::SMEM, s, mb, A, C, d,
                           direct_map(d), maxA, exp_b, av, cv, chunk, err);
}

}  // namespace

cudaError_t set_tc_wait_limit(long long polls) {
  const long long v = polls < 0 ? kWaitLimit : polls;
  return cudaMemcpyToSymbol(g_wait_limit, &v, sizeof v);
}

// Tile width: 128 columns where the tiles fill the chip; narrower ones where
// that spreads the work over more SMs, by waves over 152 SMs times the time of
// a tile relative to 128 columns (a narrow MMA is less efficient, and a tile's
// A copy does not shrink).  Every width gives the same bits.
int tma_tile_widths(const GemmDesc& d, int (&widths)[3]) {
  int n = 0;
  const int def = d.nn >= 7 ? 128 : (1 << d.nn);
  for (int tn = def; tn >= (def < 32 ? def : 32); tn /= 2) widths[n++] = tn;
  return n;
}

int tma_tile_n(const GemmDesc& d) {
  int widths[3];
  const int n = tma_tile_widths(d, widths), def = widths[0];
  if (d.tile_n >= 16 && d.tile_n <= def) return d.tile_n;
  int best = def;
  double best_cost = 1e300;
  for (int i = 0; i < n; ++i) {
    const int tn = widths[i];
    const int64_t items = ((int64_t(1) << d.nm) / TM) * ((int64_t(1) << d.nn) / tn) * d.units;
    const double rel = tn == 128 ? 1.0 : tn == 64 ? 0.55 : tn == 32 ? 0.35 : 0.3;
    const double cost = (double)((items + 151) / 152) * rel;
    if (cost < best_cost) {
      best = tn;
      best_cost = cost;
    }
  }
  return best;
}

int64_t split_plane_elems(int nrow_bits, int nk_bits, int np) {
  const int64_t kp = int64_t(1) << nk_bits;  // K >= 8 (tensor-core shapes): rows of >= 16 bytes
  return np * (int64_t(1) << nrow_bits) * kp;
}

// Accumulation chunks that launch_gemm_tma makes items of their own (1: none).
// With at most half as many tiles as SMs, a long K leaves the chip to a few
// serial chains of chunks of about 5 us each; one more launch and the sums' bytes
// cost less than one chunk.  Per tn_contract_pair call, split bf16, random
// orders, chunks in a chain -> spread, log2 M, N, K (tiles x chunks): (7, 7, 13)
// 4 x 16 209 -> 55 us, (8, 5, 11) 2 x 4 83 -> 49, (9, 6, 10) 8 x 2 61 -> 47,
// (9, 8, 12) 32 x 8 129 -> 67, (9, 9, 10) 64 x 2 60 -> 51, (9, 9, 14) 64 x 32
// 408 -> 246, (13, 5, 11) 64 x 4 121 -> 112.  From 128 tiles on, 152 SMs have at
// most one chunk in six to gain, and the sums are as many bytes as the planes.
static int chunk_parts(const GemmDesc& d, int np, bool c_planes) {
  if (np != 4 || c_planes) return 1;
  const int64_t K = int64_t(1) << d.nk;
  const int64_t nkt = (K + 31) / 32, nch = (nkt + split_chunk() - 1) / split_chunk();
  const int64_t tiles = ((int64_t(1) << d.nm) / TM) * ((int64_t(1) << d.nn) / tma_tile_n(d)) * d.units;
  const bool fits = (nch * d.units) << (d.nm + d.nn) <= int64_t(1) << 25;  // 256 MB of sums
  return nch > 1 && tiles <= 76 && fits ? (int)nch : 1;
}

int64_t tc_part_elems(const GemmDesc& d, int np, bool c_planes) {
  const int parts = chunk_parts(d, np, c_planes);
  return parts > 1 ? 4 * parts * (int64_t)d.units << (d.nm + d.nn) : 0;
}

cudaError_t launch_gemm_tma(const PlaneOperand& a, const PlaneOperand& b, float2* C, bool c_planes, const GemmDesc& d,
                            bool bf16, const ScaleIO& sio, int* err, cudaStream_t s, float2* part) {
  if (!tc_shape_ok(d) || d.units > 65535 || a.kp != b.kp || a.kp % 8 || a.np != b.np ||
      (a.np != 2 && a.np != 4))
    return cudaErrorInvalidValue;
  int TNv = tma_tile_n(d);
  const int parts = part ? chunk_parts(d, a.np, c_planes) : 1;
  // Narrow N with A shared by the hi units (e.g. one slice-only tensor against
  // the bitstrings of a group): fold consecutive hi units into the columns of
  // one tile, so that the MMAs run 128 columns wide and A is read once for
  // all of them (with scaling, the epilogue takes each unit's exponents for
  // its own columns).
  int fold = 1;
  if (parts == 1 && d.nn < 7 && a.nhi == 1 && b.nhi > 1 && d.units_lo > 0) {
    const int uh = d.units / d.units_lo;
    while (fold * 2 <= (128 >> d.nn) && uh % (fold * 2) == 0) fold *= 2;
    if (fold > 1) TNv = (1 << d.nn) * fold;
  }

  const int b_rows = fold > 1 ? (1 << d.nn) : TNv;
  CUtensorMap ma, mb;
  if (!encode_planes(&ma, a, TM) || !encode_planes(&mb, b, b_rows, fold > 1 ? 1 : 0)) return cudaErrorInvalidValue;
  const int kpi = (int)a.kp;
  const int z[4] = {a.nlo > 1, a.nhi > 1, b.nlo > 1, b.nhi > 1};
  // bit 0: plane output; bit 1: every even element of C on a 16-byte boundary
  const int cp = (c_planes ? 1 : 0) |
                 (parts > 1 || ((reinterpret_cast<uintptr_t>(C) & 15) == 0 && (d.c_lo & 1) == 0 && (d.c_hi & 1) == 0)
                      ? 2
                      : 0);
  // K = 8: the operands' 16-byte rows go by contiguous bulk copies (one per
  // plane) instead of tensor-map boxes of 16-byte rows; every address and
  // size must be a multiple of 16 bytes, else the tensor maps serve
  auto bulk = [](const PlaneOperand& o) {
    BulkPlanes q;
    q.base = reinterpret_cast<const uint8_t*>(o.base);
    q.st_lo = o.nlo > 1 ? o.st_lo : 0;
    q.st_hi = o.nhi > 1 ? o.st_hi : 0;
    q.plane = o.rows * o.kp * 2;
    return q;
  };
  BulkPlanes qa = bulk(a), qb = bulk(b);
  auto aligned = [](const BulkPlanes& q) {
    return (reinterpret_cast<uintptr_t>(q.base) % 16) == 0 && q.st_lo % 16 == 0 && q.st_hi % 16 == 0 &&
           q.plane % 16 == 0;
  };
  if (kpi != 8 || !aligned(qa) || !aligned(qb)) qa = qb = BulkPlanes{};
  const cudaError_t e =
      a.np == 4 ? launch_tn<4>(TNv, ma, mb, C, d, kpi, z, cp, sio, fold, bf16, err, s, qa, qb, parts, part)
                : launch_tn<2>(TNv, ma, mb, C, d, kpi, z, cp, sio, fold, bf16, err, s, qa, qb, 1, nullptr);
  if (e != cudaSuccess || parts == 1) return e;
  return launch_overlapped(combine_kernel, dim3((1u << (d.nm + d.nn)) / 256, (unsigned)d.units), dim3(256), 0, s, part,
                           parts, C, d, sio, z[0], z[1], z[2], z[3]);
}

// Where converting A in the GEMM beats a split pass: enough row tiles to fill
// the chip most of the time, and a K long enough that a tile's output, which
// the same warps store, is a small part of it.  Measured per call with random
// orders, split pass -> here: (16, 6, 13) split fp16 2675 -> 2064 us, (17, 6, 9)
// split bf16 307 -> 223, (14, 6, 12) split fp16 391 -> 303, (17, 6, 7) 152 -> 128;
// but (17, 6, 5) 84 -> 87, (13, 6, 14) split bf16 694 -> 882.
bool direct_ok(const GemmDesc& d) {
  return d.units == 1 && tc_shape_ok(d) && d.nn <= 6 && d.nk >= 7 && d.nm >= 14;
}

void order_for_direct(GemmDesc& d) {
  bool in[kMaxBits] = {};
  int count = 0;
  auto take = [&](int i) {
    if (!in[i] && count < 7) {
      in[i] = true;
      ++count;
    }
  };
  // A's fastest indices that are rows, then C's fastest rows
  for (int i = 0; i < d.nm; ++i)
    if (d.am[i] < 32) take(i);
  order_by_output(d, in);
  count = 0;
  for (int i = 0; i < d.nm; ++i) count += in[i];
  for (int i = 0; i < d.nm; ++i) take(i);
  // the tile's rows first, each part in C's order
  int32_t am[kMaxBits], cm[kMaxBits];
  int n = 0;
  for (int part = 1; part >= 0; --part)
    for (int i = 0; i < d.nm; ++i)
      if (in[i] == (part != 0)) {
        am[n] = d.am[i];
        cm[n++] = d.cm[i];
      }
  for (int i = 0; i < d.nm; ++i) {
    d.am[i] = am[i];
    d.cm[i] = cm[i];
  }
}

cudaError_t launch_gemm_direct(const float2* A, const PlaneOperand& b, float2* C, const GemmDesc& d, bool bf16,
                               const unsigned* maxA, const int* exp_b, int* err, cudaStream_t s) {
  if (!direct_ok(d)) return cudaErrorInvalidValue;
  const int tn = 1 << d.nn;
  CUtensorMap mb;
  if (!encode_planes(&mb, b, tn, 0, 64)) return cudaErrorInvalidValue;
  auto go = [&](auto n, auto np, auto fmt) {
    return launch_direct_as<decltype(n)::value, decltype(np)::value, decltype(fmt)::value>(mb, A, C, d, maxA, exp_b, err,
                                                                                           s);
  };
  auto go_n = [&](auto n) {
    using std::integral_constant;
    if (b.np == 4)
      return bf16 ? go(n, integral_constant<int, 4>{}, std::true_type{}) : go(n, integral_constant<int, 4>{}, std::false_type{});
    return bf16 ? go(n, integral_constant<int, 2>{}, std::true_type{}) : go(n, integral_constant<int, 2>{}, std::false_type{});
  };
  if (tn == 64) return go_n(std::integral_constant<int, 64>{});
  if (tn == 32) return go_n(std::integral_constant<int, 32>{});
  return go_n(std::integral_constant<int, 16>{});
}

}  // namespace tn
