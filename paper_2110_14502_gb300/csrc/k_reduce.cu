// Bandwidth-bound contraction for steps with few outputs and a long
// contracted index: M N <= 64 outputs, K >= 256 (for example the last steps
// of a slice, which contract two wide tensors into the open-qubit batch).
//
// Paper: Sec. "Tensor Contraction Using Fused Permutation and
// Multiplication", imbalanced case: a memory-bound contraction whose operands
// are each streamed once.  Here one CTA takes one unit; thread t takes the
// contracted values k = t, t + 256, ..; it keeps partial sums of all M N
// outputs in registers, and the CTA combines them with warp shuffles and one
// pass through shared memory.  Consecutive threads read consecutive k, so the
// reads coalesce when the contracted indices are the operands' fastest ones
// (the planner's layout puts them there).
#include "kernels.h"
#include "per_device.h"

namespace tn {

namespace {

constexpr int NT = 256;
constexpr int LOW = 8;  // bits of k taken by the thread index

__device__ __forceinline__ int32_t bit_offset(int64_t x, int lo, int hi, const int32_t* st) {
  int32_t o = 0;
  for (int i = lo; i < hi; ++i)
    if ((x >> (i - lo)) & 1) o += st[i];
  return o;
}

template <int NM, int NN>
__global__ void __launch_bounds__(NT) reduce_kernel(const float2* __restrict__ A, const float2* __restrict__ B,
                                                    float2* __restrict__ C, const GemmDesc d) {
  constexpr int M = 1 << NM, N = 1 << NN;
  const int64_t ulo = blockIdx.x % d.units_lo, uhi = blockIdx.x / d.units_lo;
  A += ulo * d.a_lo + uhi * d.a_hi;
  B += ulo * d.b_lo + uhi * d.b_hi;
  C += ulo * d.c_lo + uhi * d.c_hi;
  __shared__ int32_t offA[M], offB[N];
  __shared__ float2 part[NT / 32][M * N];
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  if (tid < M) offA[tid] = bit_offset(tid, 0, NM, d.am);
  if (tid >= 64 && tid < 64 + N) offB[tid - 64] = bit_offset(tid - 64, 0, NN, d.bn);
  __syncthreads();
  float2 acc[M * N];
#pragma unroll
  for (int i = 0; i < M * N; ++i) acc[i] = make_float2(0.f, 0.f);
  const int32_t ka = bit_offset(tid, 0, LOW, d.ak), kb = bit_offset(tid, 0, LOW, d.bk);
  const int64_t nhigh = int64_t(1) << (d.nk - LOW);
  for (int64_t kh = 0; kh < nhigh; ++kh) {
    const int32_t oa = ka + bit_offset(kh, LOW, d.nk, d.ak), ob = kb + bit_offset(kh, LOW, d.nk, d.bk);
    float2 a[M], b[N];
#pragma unroll
    for (int m = 0; m < M; ++m) a[m] = __ldg(A + offA[m] + oa);
#pragma unroll
    for (int n = 0; n < N; ++n) b[n] = __ldg(B + offB[n] + ob);
#pragma unroll
    for (int m = 0; m < M; ++m)
#pragma unroll
      for (int n = 0; n < N; ++n) {
        float2& c = acc[m * N + n];
        c.x = fmaf(a[m].x, b[n].x, fmaf(-a[m].y, b[n].y, c.x));
        c.y = fmaf(a[m].x, b[n].y, fmaf(a[m].y, b[n].x, c.y));
      }
  }
#pragma unroll
  for (int i = 0; i < M * N; ++i) {
    float x = acc[i].x, y = acc[i].y;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      x += __shfl_xor_sync(0xffffffffu, x, o);
      y += __shfl_xor_sync(0xffffffffu, y, o);
    }
    if (lane == 0) part[warp][i] = make_float2(x, y);
  }
  __syncthreads();
  if (tid < M * N) {
    float2 s = part[0][tid];
#pragma unroll
    for (int w = 1; w < NT / 32; ++w) {
      s.x += part[w][tid].x;
      s.y += part[w][tid].y;
    }
    const int m = tid / N, n = tid % N;
    C[bit_offset(m, 0, NM, d.cm) + bit_offset(n, 0, NN, d.cn)] = s;
  }
}

// The same sums with one unit spread over the chip, for launches with fewer
// units than SMs (one CTA per unit leaves the rest idle and walks K alone: a
// 2^3 x 2^3 x 2^18 step took 4.15 ms that way, 8 GB/s).
//
// What bounds it: every output is a sum in a fixed order -- per thread t of 256
// over k = t, t + 256, .., then a shuffle tree over each warp's lanes, then the
// eight warps in order -- and that order is kept, so the results are those of
// reduce_kernel bit for bit and do not depend on the number of units.  The
// K / 256 dependent multiply-adds per thread are the serial chain; the bytes
// are an L2 -> SM stream.  So the eight warps' shares of k go to the eight CTAs
// of a cluster, and the outputs in 2 x 2 blocks to clusters: 128 SMs for
// 64 outputs, each reading 4 operand rows (2 of A, 2 of B) of its k share once
// for 4 outputs, one warp per output.  Four more warps only copy: the rows
// arrive by cp.async through a ring of 16-value groups, 7 of 8 in flight, and
// one barrier per group paces both, so an addition chain (16 values of two
// dependent FMAs) runs while the copies of a later group are issued.  The copies
// move 8 bytes per lane in any index order, or 16 past L1 when the five lowest
// contracted indices are both operands' fastest.  The CTAs' partial sums meet in
// the first one's shared memory.  Measured per
// tn_contract_pair call, 2^3 x 2^3 x 2^18 with contiguous K: one CTA 3260 us,
// copies and sums by the same warps 45 us, now 33 us; 1 x 1 x 2^19 102 -> 26 us.
constexpr int SP_G = 16;                   // values of k per thread and group (bits LOW .. LOW + 3)
constexpr int SP_RING = 8;
constexpr int SP_ROWS = 4;                 // at most 2 rows of A and 2 of B per CTA
constexpr int SP_SMEM = SP_RING * SP_G * SP_ROWS * 32 * (int)sizeof(float2);

__device__ __forceinline__ void cp_async8(uint32_t dst, const void* src) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 8;\n" ::"r"(dst), "l"(src) : "memory");
}

__device__ __forceinline__ void cp_async16(uint32_t dst, const void* src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(dst), "l"(src) : "memory");
}

// WIDE: lane bits 0..4 of k have strides 1, 2, 4, 8, 16 in A and B, every
// 32-value run starts on a 16-byte boundary, and a group has 16 values of k.
template <bool WIDE>
__global__ void __cluster_dims__(8, 1, 1) __launch_bounds__(256)
    reduce_spread_kernel(const float2* __restrict__ A, const float2* __restrict__ B, float2* __restrict__ C,
                         const GemmDesc d) {
  constexpr int RING = SP_RING;
  extern __shared__ __align__(16) float2 ring[];  // [RING][SP_G][row][32]
  __shared__ float2 part[8][4];                   // first CTA of the cluster: [original warp][output]
  const int64_t ulo = blockIdx.y % d.units_lo, uhi = blockIdx.y / d.units_lo;
  A += ulo * d.a_lo + uhi * d.a_hi;
  B += ulo * d.b_lo + uhi * d.b_hi;
  C += ulo * d.c_lo + uhi * d.c_hi;
  // the cluster's CTAs have all started once this barrier's phase completes
  // (awaited before the first store to another CTA's shared memory)
  asm volatile("barrier.cluster.arrive.relaxed.aligned;" ::: "memory");
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int share = blockIdx.x & 7, blk = blockIdx.x >> 3;  // cluster rank, output block
  const int wm = d.nm > 0 ? 1 : 0, wn = d.nn > 0 ? 1 : 0;   // the block's rows and columns (log2)
  const int nblk_n = 1 << (d.nn - wn);
  const int m0 = (blk / nblk_n) << wm, n0 = (blk % nblk_n) << wn;
  const int ra = 1 << wm, rows = ra + (1 << wn);
  const int m_l = warp >> wn, n_l = warp & ((1 << wn) - 1);  // this warp's output in the block
  const int gbits = d.nk - LOW < 4 ? d.nk - LOW : 4;
  const int glen = 1 << gbits;
  const int64_t ngroups = int64_t(1) << (d.nk - LOW - gbits);
  const int t = share * 32 + lane;  // the thread of the 256 whose values this lane sums
  const int sums = 1 << (wm + wn);  // warps 0 .. sums - 1 add, warp sums + r copies row r
  float2 c = make_float2(0.f, 0.f);
  if (warp >= sums) {
    // everything an issue needs is in registers: the offsets of a group's 16
    // values, and one stride of the group index per lane, summed over the warp
    const int r = warp - sums;
    const bool isa = r < ra;
    const int32_t* ks = isa ? d.ak : d.bk;
    const float2* src = isa ? A + bit_offset(m0 + r, 0, d.nm, d.am) : B + bit_offset(n0 + r - ra, 0, d.nn, d.bn);
    // WIDE: a lane copies values 2 (lane % 16), + 1 of the share's run, for the
    // group's even (lanes 0..15) or odd (16..31) values of k
    src += WIDE ? bit_offset(share * 32, 0, LOW, ks) + 2 * (lane & 15) + (lane >> 4) * ks[LOW]
                : bit_offset(t, 0, LOW, ks);
    const int32_t gst = LOW + gbits + lane < d.nk ? ks[LOW + gbits + lane] : 0;
    int32_t tab[SP_G];
#pragma unroll
    for (int i = 0; i < SP_G; ++i) {
      tab[i] = 0;
#pragma unroll
      for (int b = 0; b < 4; ++b)
        if (((i >> b) & 1) && b < gbits) tab[i] += ks[LOW + b];
    }
    const uint32_t base = (uint32_t)__cvta_generic_to_shared(ring) + (uint32_t)r * 256u +
                          (WIDE ? (uint32_t)((lane >> 4) * SP_ROWS) * 256u + (uint32_t)(lane & 15) * 16u
                                : (uint32_t)lane * 8u);
    auto issue = [&](int g) {
      const float2* p = src + (int32_t)__reduce_add_sync(0xffffffffu, (uint32_t)(((g >> lane) & 1) ? gst : 0));
      const uint32_t slot = base + (uint32_t)((g % RING) * SP_G * SP_ROWS) * 256u;
      if constexpr (WIDE) {
#pragma unroll
        for (int i = 0; i < SP_G; i += 2) cp_async16(slot + (uint32_t)(i * SP_ROWS) * 256u, p + tab[i]);
      } else {
#pragma unroll
        for (int i = 0; i < SP_G; ++i)
          if (i < glen) cp_async8(slot + (uint32_t)(i * SP_ROWS) * 256u, p + tab[i]);
      }
    };
    for (int g = 0; g < RING - 1; ++g) {
      if (g < ngroups) issue(g);
      asm volatile("cp.async.commit_group;\n" ::: "memory");
    }
    for (int g = 0; g < (int)ngroups; ++g) {
      asm volatile("cp.async.wait_group %0;\n" ::"n"(RING - 2) : "memory");
      __syncthreads();  // group g landed for every warp; group g - 1's slot is free
      if (g + RING - 1 < ngroups) issue(g + RING - 1);
      asm volatile("cp.async.commit_group;\n" ::: "memory");
    }
  } else {
    for (int g = 0; g < (int)ngroups; ++g) {
      __syncthreads();
      const float2* pa = ring + ((g % RING) * SP_G * SP_ROWS + m_l) * 32 + lane;
      const float2* pb = ring + ((g % RING) * SP_G * SP_ROWS + ra + n_l) * 32 + lane;
      auto mac = [&](float2 a, float2 b) {
        c.x = fmaf(a.x, b.x, fmaf(-a.y, b.y, c.x));
        c.y = fmaf(a.x, b.y, fmaf(a.y, b.x, c.y));
      };
      if (glen == SP_G) {
        float2 a[SP_G], b[SP_G];
#pragma unroll
        for (int i = 0; i < SP_G; ++i) {
          a[i] = pa[i * SP_ROWS * 32];
          b[i] = pb[i * SP_ROWS * 32];
        }
#pragma unroll
        for (int i = 0; i < SP_G; ++i) mac(a[i], b[i]);
      } else {
        for (int i = 0; i < glen; ++i) mac(pa[i * SP_ROWS * 32], pb[i * SP_ROWS * 32]);
      }
    }
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    c.x += __shfl_xor_sync(0xffffffffu, c.x, o);
    c.y += __shfl_xor_sync(0xffffffffu, c.y, o);
  }
  asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
  if (warp < sums && lane == 0) {
    uint32_t dst;
    asm volatile("mapa.shared::cluster.u32 %0, %1, 0;" : "=r"(dst)
                 : "r"((uint32_t)__cvta_generic_to_shared(&part[share][warp])));
    asm volatile("st.shared::cluster.v2.f32 [%0], {%1, %2};" ::"r"(dst), "f"(c.x), "f"(c.y) : "memory");
  }
  asm volatile("barrier.cluster.arrive.release.aligned;\n barrier.cluster.wait.acquire.aligned;" ::: "memory");
  if (share == 0 && warp < sums && lane == 0) {
    float2 s = part[0][warp];
#pragma unroll
    for (int w = 1; w < 8; ++w) {
      s.x += part[w][warp].x;
      s.y += part[w][warp].y;
    }
    C[bit_offset(m0 + m_l, 0, d.nm, d.cm) + bit_offset(n0 + n_l, 0, d.nn, d.cn)] = s;
  }
}

// One unit per CTA fills the chip from one unit per SM on; below that the
// spread kernel is used whatever K is (both at 2^3 x 2^3 x 2^8, one unit: one
// group of loads each).
constexpr int SPREAD_UNITS = 152;

template <bool WIDE>
cudaError_t launch_spread_as(const float2* A, const float2* B, float2* C, const GemmDesc& d, cudaStream_t s) {
  static PerDevice once;
  const cudaError_t e = allow_smem(once, reduce_spread_kernel<WIDE>, SP_SMEM);
  if (e != cudaSuccess) return e;
  const int wm = d.nm > 0 ? 1 : 0, wn = d.nn > 0 ? 1 : 0;
  const dim3 grid(8u << (d.nm - wm + d.nn - wn), (unsigned)d.units);
  const unsigned warps = (1u << (wm + wn)) + (1u << wm) + (1u << wn);  // adding, copying
  reduce_spread_kernel<WIDE><<<grid, 32u * warps, SP_SMEM, s>>>(A, B, C, d);
  return cudaGetLastError();
}

cudaError_t launch_spread(const float2* A, const float2* B, float2* C, const GemmDesc& d, cudaStream_t s) {
  // 16-byte copies: runs of 32 values in both operands (every other stride is
  // then a multiple of 32), aligned bases, even unit strides, whole groups
  auto runs = [&](const float2* p, const int32_t* ks, int64_t lo, int64_t hi) {
    bool ok = (reinterpret_cast<uintptr_t>(p) & 15) == 0 && (lo & 1) == 0 && (hi & 1) == 0;
    for (int i = 0; i < 5; ++i) ok &= ks[i] == (int32_t(1) << i);
    return ok;
  };
  if (d.nk - LOW >= 4 && runs(A, d.ak, d.a_lo, d.a_hi) && runs(B, d.bk, d.b_lo, d.b_hi))
    return launch_spread_as<true>(A, B, C, d, s);
  return launch_spread_as<false>(A, B, C, d, s);
}

template <int NM, int NN>
cudaError_t launch(const float2* A, const float2* B, float2* C, const GemmDesc& d, cudaStream_t s) {
  reduce_kernel<NM, NN><<<(unsigned)d.units, NT, 0, s>>>(A, B, C, d);
  return cudaGetLastError();
}

template <int NM>
cudaError_t launch_nn(const float2* A, const float2* B, float2* C, const GemmDesc& d, cudaStream_t s) {
  switch (d.nn) {
    case 0: return launch<NM, 0>(A, B, C, d, s);
    case 1: if constexpr (NM + 1 <= 6) return launch<NM, 1>(A, B, C, d, s); break;
    case 2: if constexpr (NM + 2 <= 6) return launch<NM, 2>(A, B, C, d, s); break;
    case 3: if constexpr (NM + 3 <= 6) return launch<NM, 3>(A, B, C, d, s); break;
    case 4: if constexpr (NM + 4 <= 6) return launch<NM, 4>(A, B, C, d, s); break;
    case 5: if constexpr (NM + 5 <= 6) return launch<NM, 5>(A, B, C, d, s); break;
    case 6: if constexpr (NM + 6 <= 6) return launch<NM, 6>(A, B, C, d, s); break;
    default: break;
  }
  return cudaErrorInvalidValue;
}

}  // namespace

bool reduce_shape_ok(const GemmDesc& d) { return d.nm + d.nn <= 6 && d.nk >= LOW && d.nk <= 30; }

cudaError_t launch_reduce(const float2* A, const float2* B, float2* C, const GemmDesc& d, cudaStream_t s) {
  if (!reduce_shape_ok(d) || d.units < 1 || d.units > (int64_t(1) << 31) - 1) return cudaErrorInvalidValue;
  if (d.units < SPREAD_UNITS) return launch_spread(A, B, C, d, s);
  switch (d.nm) {
    case 0: return launch_nn<0>(A, B, C, d, s);
    case 1: return launch_nn<1>(A, B, C, d, s);
    case 2: return launch_nn<2>(A, B, C, d, s);
    case 3: return launch_nn<3>(A, B, C, d, s);
    case 4: return launch_nn<4>(A, B, C, d, s);
    case 5: return launch_nn<5>(A, B, C, d, s);
    case 6: return launch_nn<6>(A, B, C, d, s);
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace tn
