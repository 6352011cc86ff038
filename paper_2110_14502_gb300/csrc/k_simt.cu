// Fused permute-GEMM on FP32 CUDA cores (complex64 in, complex64 out): the
// plain complex64 path, FP32 products and sums, no tensor cores.
//
// Paper: Sec. "Tensor Contraction Using Fused Permutation and Multiplication",
// dense case: the permutation of each operand is folded into the fetch of its
// tile rather than run as a separate pass.  Every element offset comes from
// the operand's per-bit strides (the analogue of the paper's pre-computed
// position array): a row's offset is computed once per CTA, and a K offset
// splits into the chunk's high bits (once per chunk) plus a per-thread
// constant for the low bits.
//
// Tiling: 256 threads compute a BM x BN tile of C over K chunks of BK, each
// thread an RM-row x RN-column complex micro-tile.  The tiles are staged in
// shared memory k-major ([k][row], rows contiguous) with two buffers: the
// global loads of chunk c+1 are in flight in registers while chunk c is
// computed, then stored to the other buffer; one barrier per chunk.  They are
// issued before the barrier, which holds ordinary loads back: log2 M, N, K =
// (7, 9, 12) 317 us, after it 333; (12, 12, 9) 1399 and 1450, (13, 13, 5) 635 and
// 694, (6, 4, 12) 182 and 196; with 128 x 64 tiles (16, 6, 11) 1747 and 1755, (14, 6,
// 12) in planner order 910 and 914 but in random orders 1007 and 993.
//
// Arithmetic: packed FP32 (fma.rn.f32x2), one instruction for two of a complex
// multiply-add's four FMAs: (re, im) += (ar, ar) (br, bi), then += (-ai, ai)
// (bi, br).  The same four roundings in the same order as scalar FMAs, k
// ascending, so every tile shape gives the same bits.  A sits in shared memory
// already as (ar, ar, -ai, ai), so its operands are one 16-byte load; B's
// swapped pair costs a register move, which issues beside the packed FMAs.  The
// 128 x 64 tile (8 x 4 outputs per thread) keeps scalar FMAs: per multiply-add it
// reads twice the shared memory of the 128 x 128 tile, and the doubled A costs
// more than packing saves (log2 M, N, K, scalar and packed: (16, 6, 11) 1781 and
// 2014 us, (14, 6, 12) 1037 and 1125, (17, 6, 8) 466 and 507; packed with two
// CTAs per SM and spills 1872, 1381, 469).
//
// What bounds the 128 x 128 tile: two warps per scheduler (246 registers, one CTA
// per SM) do not cover the packed FMAs' latency.  Counters at (13, 13, 9), 5.6 ms:
// FMA pipe busy 63% of the cycles, an instruction issued in 41%; per issue a warp
// waits 1.3 cycles on a fixed latency, 1.0 on the FMA pipe and 0.3 each on
// instruction fetch and shared memory; shared memory 10% and DRAM 2% busy.
//
// Global loads: when the operand's two fastest indices are its first two K
// bits (the planner's layouts put contracted indices innermost), a thread
// reads 4 consecutive K values of one row as two 16-byte loads and the lanes
// of a warp read consecutive rows at the same K quad (one 32-byte sector per
// row); otherwise each lane reads one element, lanes on consecutive rows.
#include <algorithm>
#include <cmath>
#include <type_traits>

#include "device_common.h"
#include "kernels.h"
#include "per_device.h"

namespace tn {

namespace {

constexpr int NT = 256;

__device__ __forceinline__ int32_t bit_offset(int64_t x, int nb, const int32_t* st) {
  int32_t o = 0;
  for (int i = 0; i < nb; ++i)
    if ((x >> i) & 1) o += st[i];
  return o;
}

__host__ __device__ constexpr int ilog2(int x) { return x <= 1 ? 0 : 1 + ilog2(x / 2); }

// Offset of the K bits at and above bit LOW of k0 (a multiple of 2^LOW).
template <int LOW>
__device__ __forceinline__ int32_t k_high_offset(int64_t k0, int nk, const int32_t* st) {
  int32_t o = 0;
  for (int i = LOW; i < nk; ++i)
    if ((k0 >> i) & 1) o += st[i];
  return o;
}

__device__ __forceinline__ f32x2 swap2(f32x2 v) {
  const float2 r = unpack2(v);
  return pack2(r.y, r.x);
}
__device__ __forceinline__ void acc2(f32x2& c, f32x2 a, f32x2 b) { c = fma2(a, b, c); }

// One operand tile of R rows x BK K values: what this thread loads, where from
// and where it goes in shared memory.  Thread t takes row t % R at K positions
// (t / R) + (256 / R) j -- single values, or quads of 4 (vec).
template <int R, int BK>
struct TileLoader {
  static constexpr int NE = R * BK / NT;   // elements per thread
  static constexpr int NQ = NE / 4;        // quads per thread (vector path)
  static constexpr int STEP = NT / R;
  static_assert(NE >= 4, "tile too small");
  bool vec;
  int64_t K;
  int row, kk0;
  int32_t row_off;
  int32_t low[NE];        // offsets of this thread's K positions within a chunk (vector path: of its quads)
  float2 v[NE];           // staged values (vector path: quad q's 4 values at 4 q ..)

  __device__ void init(const GemmDesc& d, int nrow_bits, const int32_t* rst, const int32_t* kst, int64_t r0,
                       bool vector_ok) {
    const int t = threadIdx.x;
    constexpr int LOW = ilog2(BK);
    K = int64_t(1) << d.nk;
    vec = vector_ok;
    row = t % R;
    kk0 = t / R;
    row_off = r0 + row < (int64_t(1) << nrow_bits) ? bit_offset(r0 + row, nrow_bits, rst) : -1;
    const int lb = d.nk < LOW ? d.nk : LOW;
    if (vec) {
#pragma unroll
      for (int j = 0; j < NQ; ++j) low[j] = bit_offset(4 * (kk0 + STEP * j), lb, kst);
    } else {
#pragma unroll
      for (int j = 0; j < NE; ++j) low[j] = bit_offset(kk0 + STEP * j, lb, kst);
    }
  }

  __device__ __forceinline__ void load(const float2* src, int64_t k0, int32_t khi) {
    if (vec) {
#pragma unroll
      for (int q = 0; q < NQ; ++q) {
        float4 x = make_float4(0.f, 0.f, 0.f, 0.f), y = x;
        if (row_off >= 0 && k0 + 4 * (kk0 + STEP * q) < K) {
          const float4* p = reinterpret_cast<const float4*>(src + row_off + khi + low[q]);
          x = p[0];
          y = p[1];
        }
        v[4 * q + 0] = make_float2(x.x, x.y);
        v[4 * q + 1] = make_float2(x.z, x.w);
        v[4 * q + 2] = make_float2(y.x, y.y);
        v[4 * q + 3] = make_float2(y.z, y.w);
      }
    } else {
#pragma unroll
      for (int j = 0; j < NE; ++j) {
        float2 x = make_float2(0.f, 0.f);
        if (row_off >= 0 && k0 + kk0 + STEP * j < K) x = src[row_off + khi + low[j]];
        v[j] = x;
      }
    }
  }

  // every staged value with its tile position [BK][R]
  template <class F>
  __device__ __forceinline__ void store(F&& put) const {
    if (vec) {
#pragma unroll
      for (int q = 0; q < NQ; ++q)
#pragma unroll
        for (int j = 0; j < 4; ++j) put((4 * (kk0 + STEP * q) + j) * R + row, v[4 * q + j]);
    } else {
#pragma unroll
      for (int j = 0; j < NE; ++j) put((kk0 + STEP * j) * R + row, v[j]);
    }
  }
};

template <int BM, int BN, int BK, int RM, int RN, bool PACKED>
struct SimtCfg {
  static_assert(BM / RM * (BN / RN) == NT, "256 threads");
  static constexpr int A_BUF = BK * BM * (PACKED ? 16 : 8), B_BUF = BK * BN * 8;
  static constexpr int SMEM = 2 * (A_BUF + B_BUF);
};

// flags: bit 0 A vector loads, bit 1 B vector loads, bit 2 C pair stores
template <int BM, int BN, int BK, int RM, int RN, bool PACKED>
__global__ void __launch_bounds__(NT, BM * BN >= 128 * 64 ? 1 : 2) gemm_simt_kernel(const float2* A,
                                                           const float2* B,
                                                           float2* __restrict__ C, const GemmDesc d, int flags) {
  using CF = SimtCfg<BM, BN, BK, RM, RN, PACKED>;
  constexpr int CG = BN / RN;        // column groups
  constexpr int BAND = 2 * CG;       // columns 2 tn, 2 tn + 1 of each band of BAND columns (RN = 1: column tn)
  extern __shared__ __align__(16) uint8_t smem[];
  using AT = std::conditional_t<PACKED, float4, float2>;           // (ar, ar, -ai, ai), or (ar, ai)
  AT* As = reinterpret_cast<AT*>(smem);                            // [2][BK][BM]
  float2* Bs = reinterpret_cast<float2*>(smem + 2 * CF::A_BUF);    // [2][BK][BN]
  const int64_t K = int64_t(1) << d.nk;
  const int64_t m0 = (int64_t)blockIdx.x * BM, n0 = (int64_t)blockIdx.y * BN;
  let_next_start();
  after_previous();
  const int64_t ulo = blockIdx.z % d.units_lo, uhi = blockIdx.z / d.units_lo;
  A += ulo * d.a_lo + uhi * d.a_hi;
  B += ulo * d.b_lo + uhi * d.b_hi;
  C += ulo * d.c_lo + uhi * d.c_hi;
  const int tid = threadIdx.x;
  const int tn = tid % CG, tm = tid / CG;

  TileLoader<BM, BK> la;
  TileLoader<BN, BK> lb;
  la.init(d, d.nm, d.am, d.ak, m0, (flags & 1) != 0);
  lb.init(d, d.nn, d.bn, d.bk, n0, (flags & 2) != 0);

  f32x2 acc[RM][RN];   // PACKED
  float accr[RM][RN], acci[RM][RN];
#pragma unroll
  for (int i = 0; i < RM; ++i)
#pragma unroll
    for (int j = 0; j < RN; ++j) {
      acc[i][j] = 0ull;
      accr[i][j] = acci[i][j] = 0.f;
    }
  auto result = [&](int i, int j) {
    if constexpr (PACKED) return unpack2(acc[i][j]);
    else return make_float2(accr[i][j], acci[i][j]);
  };

  auto store_tiles = [&](int buf) {
    AT* at = As + buf * BK * BM;
    float2* bt = Bs + buf * BK * BN;
    la.store([&](int p, float2 x) {
      if constexpr (PACKED) at[p] = make_float4(x.x, x.x, -x.y, x.y);
      else at[p] = x;
    });
    lb.store([&](int p, float2 x) { bt[p] = x; });
  };
  const int64_t nch = (K + BK - 1) / BK;
  const int kn = K < BK ? (int)K : BK;  // K values of a chunk
  auto load_chunk = [&](int64_t c) {
    const int64_t k = c * BK;
    la.load(A, k, k_high_offset<ilog2(BK)>(k, d.nk, d.ak));
    lb.load(B, k, k_high_offset<ilog2(BK)>(k, d.nk, d.bk));
  };
  load_chunk(0);
  store_tiles(0);
  if (nch > 1) load_chunk(1);
  __syncthreads();
  for (int64_t c = 0; c < nch; ++c) {
    const int buf = (int)(c & 1);
    const AT* const a0 = As + buf * BK * BM + RM * tm;
    const ulonglong2* at = reinterpret_cast<const ulonglong2*>(a0);
    const float2* bt = Bs + buf * BK * BN;
    auto scalar_step = [&](int kk) {
      float ar[RM], ai[RM], br[RN], bi[RN];
#pragma unroll
      for (int i = 0; i < RM; i += 2) {
        const float4 x = *reinterpret_cast<const float4*>(a0 + kk * BM + i);
        ar[i] = x.x;
        ai[i] = x.y;
        ar[i + 1] = x.z;
        ai[i + 1] = x.w;
      }
#pragma unroll
      for (int j = 0; j < RN; j += 2) {
        const float4 x = *reinterpret_cast<const float4*>(bt + kk * BN + BAND / 2 * j + 2 * tn);
        br[j] = x.x;
        bi[j] = x.y;
        br[j + 1] = x.z;
        bi[j + 1] = x.w;
      }
#pragma unroll
      for (int i = 0; i < RM; ++i)
#pragma unroll
        for (int j = 0; j < RN; ++j) {
          accr[i][j] = fmaf(ar[i], br[j], accr[i][j]);
          accr[i][j] = fmaf(-ai[i], bi[j], accr[i][j]);
          acci[i][j] = fmaf(ar[i], bi[j], acci[i][j]);
          acci[i][j] = fmaf(ai[i], br[j], acci[i][j]);
        }
    };
    auto packed_step = [&](int kk) {
      f32x2 b[RN], bs[RN];
      if constexpr (RN == 1) {
        b[0] = *reinterpret_cast<const f32x2*>(bt + kk * BN + tn);
      } else {
#pragma unroll
        for (int j = 0; j < RN / 2; ++j) {
          const ulonglong2 x = *reinterpret_cast<const ulonglong2*>(bt + kk * BN + BAND * j + 2 * tn);
          b[2 * j] = x.x;
          b[2 * j + 1] = x.y;
        }
      }
#pragma unroll
      for (int j = 0; j < RN; ++j) bs[j] = swap2(b[j]);
#pragma unroll
      for (int i = 0; i < RM; ++i) {
        const ulonglong2 a = at[kk * BM + i];
#pragma unroll
        for (int j = 0; j < RN; ++j) acc2(acc[i][j], a.x, b[j]);
#pragma unroll
        for (int j = 0; j < RN; ++j) acc2(acc[i][j], a.y, bs[j]);
      }
    };
    auto step = [&](int kk) {
      if constexpr (PACKED) packed_step(kk);
      else scalar_step(kk);
    };
    if (kn == BK) {
#pragma unroll 16
      for (int kk = 0; kk < BK; ++kk) step(kk);
    } else {
      for (int kk = 0; kk < kn; ++kk) step(kk);
    }
    if (c + 1 < nch) store_tiles(buf ^ 1);
    if (c + 2 < nch) load_chunk(c + 2);
    __syncthreads();
  }

  // epilogue: C offsets of this thread's rows and columns
  const int64_t M = int64_t(1) << d.nm, N = int64_t(1) << d.nn;
  int32_t cc[RN];
#pragma unroll
  for (int j = 0; j < RN; ++j) {
    const int64_t n = n0 + (RN == 1 ? tn : BAND * (j >> 1) + 2 * tn + (j & 1));
    cc[j] = n < N ? bit_offset(n, d.nn, d.cn) : -1;
  }
  const bool pairs = RN > 1 && (flags & 4) != 0;  // columns 2 tn, 2 tn + 1 adjacent in C (16-byte store)
#pragma unroll
  for (int i = 0; i < RM; ++i) {
    const int64_t m = m0 + RM * tm + i;
    if (m >= M) continue;
    const int32_t rc = bit_offset(m, d.nm, d.cm);
    if (pairs) {
#pragma unroll
      for (int j = 0; j < RN; j += 2)
        if (cc[j] >= 0) {
          const float2 x = result(i, j), y = result(i, RN > 1 ? j + 1 : j);
          *reinterpret_cast<float4*>(C + rc + cc[j]) = make_float4(x.x, x.y, y.x, y.y);
        }
    } else {
#pragma unroll
      for (int j = 0; j < RN; ++j)
        if (cc[j] >= 0) C[rc + cc[j]] = result(i, j);
    }
  }
}

template <int BM, int BN, int BK, int RM, int RN, bool PACKED = true>
cudaError_t launch_tile(const float2* A, const float2* B, float2* C, const GemmDesc& d, int flags, cudaStream_t s) {
  constexpr int SMEM = SimtCfg<BM, BN, BK, RM, RN, PACKED>::SMEM;
  static PerDevice once;
  const cudaError_t e = allow_smem(once, gemm_simt_kernel<BM, BN, BK, RM, RN, PACKED>, SMEM);
  if (e != cudaSuccess) return e;
  const int64_t M = int64_t(1) << d.nm, N = int64_t(1) << d.nn;
  dim3 grid((unsigned)((M + BM - 1) / BM), (unsigned)((N + BN - 1) / BN), (unsigned)d.units);
  return launch_overlapped(gemm_simt_kernel<BM, BN, BK, RM, RN, PACKED>, grid, dim3(NT), SMEM, s, A, B,
                           C, d, flags);
}

// Vector loads of 4 consecutive K values need the operand's two fastest
// indices to be its K bits 0 and 1 and every such quad to start on a 16-byte
// boundary: the base and the unit strides even (in complex elements), and the
// other strides even, which holds once bits 0 and 1 take strides 1 and 2.
bool quad_ok(const float2* base, int nk, const int32_t* kst, int64_t lo, int64_t hi) {
  return nk >= 2 && kst[0] == 1 && kst[1] == 2 && (reinterpret_cast<uintptr_t>(base) & 15) == 0 && (lo & 1) == 0 &&
         (hi & 1) == 0;
}

}  // namespace

// Tile choice: the estimated time of each tile shape, waves over 152 SMs times
// the tile's multiply-adds (padding included) over the shape's rate relative to
// the largest (46 TFLOP/s on (12, 12, 9); scalar FMAs reached 44).  The small
// shapes matter where the large one would leave SMs idle or compute padding:
// (5, 4, 7) 41 -> 12 us, (5, 3, 8) x 2 units 82 -> 18 us, (6, 4, 12) x 128 units
// 1.08 -> 0.57 ms, (16, 5, 10) 901 -> 558 us.  Every shape gives the same bits, so this is speed alone.
// Column tiles are counted by grid.y, which ends at 65535: a shape with more of
// them (16 columns from N = 2^20 on, 32 from 2^21, 64 from 2^22) is no choice.
SimtTile simt_tile(const GemmDesc& d) {
  const int64_t M = int64_t(1) << d.nm, N = int64_t(1) << d.nn;
  auto cost = [&](int bm, int bn, double rate) {
    const int64_t rows = (M + bm - 1) / bm, cols = (N + bn - 1) / bn;
    if (cols > 65535) return HUGE_VAL;
    const double tiles = (double)rows * (double)cols * d.units;
    return (double)((int64_t)((tiles + 151) / 152)) * bm * bn / rate;
  };
  const double c128 = cost(128, 128, 1.0), c64 = cost(128, 64, 0.85), cm = cost(64, 32, 0.55), cs = cost(32, 16, 0.25);
  const double best = std::min(std::min(c128, c64), std::min(cm, cs));
  if (best == c128) return {128, 128};
  if (best == c64) return {128, 64};
  if (best == cm) return {64, 32};
  return {32, 16};
}

cudaError_t launch_gemm_simt(const float2* A, const float2* B, float2* C, const GemmDesc& d, cudaStream_t s) {
  int flags = 0;
  if (quad_ok(A, d.nk, d.ak, d.a_lo, d.a_hi)) flags |= 1;
  if (quad_ok(B, d.nk, d.bk, d.b_lo, d.b_hi)) flags |= 2;
  // column bit 0 with C stride 1: columns 2j, 2j + 1 are adjacent and the
  // pair starts on an even element (every other stride of C is even)
  if (d.nn >= 1 && d.cn[0] == 1 && (reinterpret_cast<uintptr_t>(C) & 15) == 0 && (d.c_lo & 1) == 0 &&
      (d.c_hi & 1) == 0)
    flags |= 4;
  const SimtTile t = simt_tile(d);
  if (t.rows == 128 && t.cols == 128) return launch_tile<128, 128, 16, 8, 8>(A, B, C, d, flags, s);
  if (t.rows == 128) return launch_tile<128, 64, 16, 8, 4, false>(A, B, C, d, flags, s);
  if (t.rows == 64) return launch_tile<64, 32, 32, 4, 2>(A, B, C, d, flags, s);
  return launch_tile<32, 16, 64, 2, 1>(A, B, C, d, flags, s);
}

}  // namespace tn
