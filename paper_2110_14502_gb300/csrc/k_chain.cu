// Runs of consecutive small steps in one launch.
//
// A slice's contraction starts with many tiny steps (a few leaves at a time),
// and a small circuit has nothing else.  Launched one by one, each costs a
// launch and the latency of one dependent pass through memory for a
// microsecond's work or less.  The units of a launch do not depend on one
// another, so one CTA per unit walks the whole run: a barrier between steps
// takes the place of a launch, the tensors stay in cache, and nothing waits for
// the other units.
//
// What bounds it: latency (a descriptor, the operands' trip from L2, K dependent
// multiply-adds per output) and shared-memory reads.  So the next step's
// descriptor is fetched while the current one runs; both operands are copied
// front to back into shared memory, because reads through the index strides
// would touch a cache line per lane; and a thread item is a 2 x 2 block of
// outputs, four reads for four complex multiply-adds.  An element sits at its
// index with bits 4..7 and 8..11 folded onto bits 0..3, which spreads the lanes'
// power-of-two strides over the banks.  Items follow C's memory order, so the
// stores need no permutation.  Each output adds its products with k ascending
// in the order of the kernel that would run the step alone, so results do not
// depend on which steps share a launch.
//
// Measured on the sixteen steps of a 4 x 4 circuit, one unit: sixteen launches
// 115 us of kernel time, this kernel 26; the whole call 160 -> 102 us (150 with
// the operands read through their strides instead of from shared memory).
#include <algorithm>

#include "device_common.h"
#include "kernels.h"
#include "per_device.h"

namespace tn {

namespace {

__host__ __device__ __forceinline__ int chain_slot(int i) { return i ^ ((i >> 4) & 15) ^ ((i >> 8) & 15); }

__device__ __forceinline__ float2* chain_ptr(const ChainBase& b, int space, int64_t off, int64_t lo, int64_t hi) {
  switch (space) {
    case 0: return b.store + off;
    case 1: return b.inv + off;
    case 2: return b.sarena + off + lo * b.slice_elems;
    default: return b.parena + off + (lo + hi * b.gs) * b.unit_elems;
  }
}

template <bool IM_FIRST>
__device__ __forceinline__ void chain_mac(float2& c, float2 a, float2 b) {
  if (IM_FIRST) {
    c.x = fmaf(a.x, b.x, fmaf(-a.y, b.y, c.x));
    c.y = fmaf(a.x, b.y, fmaf(a.y, b.x, c.y));
  } else {
    c.x = fmaf(a.x, b.x, c.x);
    c.x = fmaf(-a.y, b.y, c.x);
    c.y = fmaf(a.x, b.y, c.y);
    c.y = fmaf(a.y, b.x, c.y);
  }
}

template <bool TILE, bool IM_FIRST>
__device__ __forceinline__ void chain_items(const ChainStep& S, const float2* sA, const float2* sB, float2* C,
                                            const int2* kt) {
  const int n = 1 << S.items, K = 1 << S.nk;
  for (int i = threadIdx.x; i < n; i += blockDim.x) {
    int o = 0, a0 = 0, b0 = 0;
    for (int b = 0; b < S.items; ++b)
      if ((i >> b) & 1) {
        o += S.oc[b];
        a0 ^= S.ha[b];
        b0 ^= S.hb[b];
      }
    if (TILE) {
      const int b1 = b0 ^ S.hb[S.items], a1 = a0 ^ S.ha[S.items + 1];
      float2 c00 = make_float2(0.f, 0.f), c01 = c00, c10 = c00, c11 = c00;  // [M bit][N bit]
#pragma unroll 4
      for (int k = 0; k < K; ++k) {
        const int2 t = kt[k];
        const float2 x0 = sA[a0 ^ t.x], x1 = sA[a1 ^ t.x], y0 = sB[b0 ^ t.y], y1 = sB[b1 ^ t.y];
        chain_mac<IM_FIRST>(c00, x0, y0);
        chain_mac<IM_FIRST>(c01, x0, y1);
        chain_mac<IM_FIRST>(c10, x1, y0);
        chain_mac<IM_FIRST>(c11, x1, y1);
      }
      const int on = S.oc[S.items], om = S.oc[S.items + 1];
      C[o] = c00;
      C[o + on] = c01;
      C[o + om] = c10;
      C[o + on + om] = c11;
    } else {
      float2 c = make_float2(0.f, 0.f);
#pragma unroll 4
      for (int k = 0; k < K; ++k) {
        const int2 t = kt[k];
        chain_mac<IM_FIRST>(c, sA[a0 ^ t.x], sB[b0 ^ t.y]);
      }
      C[o] = c;
    }
  }
}

__global__ void __launch_bounds__(512) chain_kernel(const ChainStep* __restrict__ steps, int count, uint64_t forms,
                                                    const ChainBase base, const float2* __restrict__ leaf_store,
                                                    const LeafGather* __restrict__ leaves, int nleaves,
                                                    float2* gather_arena, int64_t gather_stride,
                                                    const GroupArg group) {
  extern __shared__ float2 operands[];
  __shared__ ChainStep S[2];
  __shared__ int2 kt[1 << kChainMaxK];
  const int nt = blockDim.x, tid = threadIdx.x;
  const int u = blockIdx.x;
  const int64_t lo = u % base.gs, hi = u / base.gs;
  constexpr int WORDS = sizeof(ChainStep) / 4;
  static_assert(sizeof(ChainStep) % 4 == 0, "descriptors are copied by words");
  auto fetch = [&](int i) {
    const uint32_t* p = reinterpret_cast<const uint32_t*>(steps + i);
    uint32_t* q = reinterpret_cast<uint32_t*>(&S[i & 1]);
    for (int w = tid; w < WORDS; w += nt) q[w] = p[w];
  };
  fetch(0);  // (the descriptors never change)
  let_next_start();
  after_previous();
  // the unit's leaves first, when this run opens its phase: one warp per leaf
  const GroupInfo grp = nleaves > 0 && group.slot ? *group.slot : group.now;
  for (int l = tid >> 5; l < nleaves; l += nt >> 5) {
    const LeafGather& L = leaves[l];
    const int64_t from = leaf_fixed_offset(L, grp, u);
    float2* dst = gather_arena + (int64_t)u * gather_stride + L.dst_off;
    for (int e = tid & 31; e < (1 << L.nkept); e += 32) dst[e] = leaf_store[leaf_kept_offset(L, from, e)];
  }
  __syncthreads();
  for (int i = 0; i < count; ++i) {
    const ChainStep& s = S[i & 1];
    const int na = 1 << s.abits, nb = 1 << s.bbits;
    float2 *sA = operands, *sB = operands + na;
    const float2* A = chain_ptr(base, s.space[0], s.off[0], lo, hi);
    const float2* B = chain_ptr(base, s.space[1], s.off[1], lo, hi);
    float2* C = chain_ptr(base, s.space[2], s.off[2], lo, hi);
#pragma unroll 4
    for (int e = tid; e < na; e += nt) sA[chain_slot(e)] = A[e];
#pragma unroll 4
    for (int e = tid; e < nb; e += nt) sB[chain_slot(e)] = B[e];
    for (int k = tid; k < (1 << s.nk); k += nt) {
      int a = 0, b = 0;
      for (int l = 0; l < s.nk; ++l)
        if ((k >> l) & 1) {
          a ^= s.ka[l];
          b ^= s.kb[l];
        }
      kt[k] = make_int2(a, b);
    }
    __syncthreads();  // operands and kt ready; S[(i + 1) & 1] no longer read
    if (i + 1 < count) fetch(i + 1);
    if ((forms >> i) & 1) {
      if (s.tile) chain_items<true, true>(s, sA, sB, C, kt);
      else chain_items<false, true>(s, sA, sB, C, kt);
    } else {
      if (s.tile) chain_items<true, false>(s, sA, sB, C, kt);
      else chain_items<false, false>(s, sA, sB, C, kt);
    }
    __syncthreads();  // C written before the next step reads it
  }
}

constexpr int CHAIN_SMEM = 2 * (1 << kChainMaxOperand) * (int)sizeof(float2);

}  // namespace

bool chain_shape_ok(const GemmDesc& d, int64_t units) {
  // One CTA runs a step alone: with few units that beats a launch (2-3 us, and
  // 12 us for a 2^5 x 2^4 x 2^7 step in the FP32 GEMM) up to 2^16 multiply-adds;
  // with enough units to fill the chip the step's own kernel, which tiles and
  // streams, wins earlier.
  const int limit = units <= 4 ? 16 : units < 152 ? 15 : 12;
  return d.nm + d.nn <= kChainMaxC && d.nk <= kChainMaxK && d.nm + d.nk <= kChainMaxOperand &&
         d.nn + d.nk <= kChainMaxOperand && d.nm + d.nn + d.nk <= limit && !reduce_shape_ok(d);
}

void make_chain_step(const GemmDesc& d, const int space[3], const int64_t off[3], ChainStep& s) {
  s = ChainStep{};
  s.nk = d.nk;
  s.abits = d.nm + d.nk;
  s.bbits = d.nn + d.nk;
  for (int i = 0; i < 3; ++i) {
    s.space[i] = space[i];
    s.off[i] = off[i];
  }
  // C's index bit b is the M or N bit with output stride 2^b
  const int nc = d.nm + d.nn;
  int32_t sa[kChainMaxC] = {}, sb[kChainMaxC] = {};
  for (int i = 0; i < d.nm; ++i) sa[__builtin_ctz((unsigned)d.cm[i])] = d.am[i];
  for (int j = 0; j < d.nn; ++j) sb[__builtin_ctz((unsigned)d.cn[j])] = d.bn[j];
  // the 2 x 2 block takes C's slowest N bit and slowest M bit, the items the rest in order
  s.tile = d.nm > 0 && d.nn > 0;
  int top[2] = {-1, -1};  // N, M
  if (s.tile)
    for (int b = 0; b < nc; ++b) top[sa[b] != 0] = b;
  int n = 0;
  auto put = [&](int b) {
    s.oc[n] = 1 << b;
    s.ha[n] = chain_slot(sa[b]);
    s.hb[n] = chain_slot(sb[b]);
    ++n;
  };
  for (int b = 0; b < nc; ++b)
    if (b != top[0] && b != top[1]) put(b);
  s.items = n;
  if (s.tile) {
    put(top[0]);
    put(top[1]);
  }
  for (int l = 0; l < d.nk; ++l) {
    s.ka[l] = chain_slot(d.ak[l]);
    s.kb[l] = chain_slot(d.bk[l]);
  }
}

void chain_add(ChainRun& run, const GemmDesc& d, bool im_first) {
  if (im_first) run.forms |= uint64_t(1) << run.count;
  ++run.count;
  run.items = std::max(run.items, d.nm + d.nn - (d.nm > 0 && d.nn > 0 ? 2 : 0));
  run.elems = std::max(run.elems, (1 << (d.nm + d.nk)) + (1 << (d.nn + d.nk)));
}

cudaError_t launch_chain(const ChainStep* steps, const ChainRun& run, const ChainBase& base, int units,
                         const float2* leaf_store, const LeafGather* leaves, int nleaves, float2* gather_arena,
                         int64_t gather_stride, const GroupArg& group, cudaStream_t s) {
  if (run.count < 1 || run.count > 64 || units < 1) return cudaErrorInvalidValue;
  static PerDevice once;
  const cudaError_t e = allow_smem(once, chain_kernel, CHAIN_SMEM);
  if (e != cudaSuccess) return e;
  // threads for the widest step's items, and enough to copy the operands in
  // about eight loads each; fewer once the units fill the SMs by themselves
  const int cap = units >= 304 ? 128 : 512;
  int nt = 64;
  while (nt < cap && (nt < (1 << run.items) || nt * 8 < run.elems)) nt *= 2;
  return launch_overlapped(chain_kernel, dim3((unsigned)units), dim3(nt), run.elems * sizeof(float2), s, steps, run.count,
                           run.forms, base, leaf_store, leaves, nleaves, gather_arena, gather_stride, group);
}

}  // namespace tn
