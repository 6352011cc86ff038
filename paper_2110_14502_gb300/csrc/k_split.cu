// Operand preparation for the TMA-fed tensor-core GEMM: gather a complex64
// operand through its per-bit strides (the index permutation) and write it
// once as four K-major 16-bit planes {re_hi, re_lo, im_hi, im_lo} of K (>= 8)
// values per row; the GEMM's TMA box reads past a short K as zeros.
//
// Paper: Sec. "Tensor Contraction Using Fused Permutation and Multiplication",
// imbalanced case (TTGT: one permuted copy of each operand feeds the GEMM; the
// position of every element comes from a pre-computed offset) and Sec. "A
// Mixed-Precision Computation Method via Adaptive Precision Scaling" (half
// precision operands: here each value is split as x = hi + lo,
// hi = rn16(x), lo = rn16(x - hi)).
#include <algorithm>
#include <type_traits>

#include "device_common.h"
#include "kernels.h"

namespace tn {

namespace {

constexpr int NT = 256;

// Largest |component| of each distinct tensor z (float bits, atomicMax).  The
// operand is a dense block of 2^bits elements whatever its index order, so the
// pass reads it front to back, 16 bytes per load.
__global__ void __launch_bounds__(NT) max_kernel(const float2* __restrict__ src, int bits, int nlo, int64_t lo,
                                                 int64_t hi, int vec, unsigned* __restrict__ maxbits) {
  const int64_t z = blockIdx.y;
  src += (z % nlo) * lo + (z / nlo) * hi;
  float m = 0.f;
  const int64_t step = (int64_t)gridDim.x * NT;
  const int64_t at = (int64_t)blockIdx.x * NT + threadIdx.x;
  if (vec) {
    const float4* p = reinterpret_cast<const float4*>(src);
    const int64_t n = int64_t(1) << (bits - 1);
    int64_t e = at;
    for (; e + 7 * step < n; e += 8 * step) {
      float4 v[8];
#pragma unroll
      for (int j = 0; j < 8; ++j) v[j] = __ldg(p + e + j * step);
#pragma unroll
      for (int j = 0; j < 8; ++j)
        m = fmaxf(m, fmaxf(fmaxf(fabsf(v[j].x), fabsf(v[j].y)), fmaxf(fabsf(v[j].z), fabsf(v[j].w))));
    }
    for (; e < n; e += step) {
      const float4 v = __ldg(p + e);
      m = fmaxf(m, fmaxf(fmaxf(fabsf(v.x), fabsf(v.y)), fmaxf(fabsf(v.z), fabsf(v.w))));
    }
  } else {
    const int64_t n = int64_t(1) << bits;
    for (int64_t e = at; e < n; e += step) {
      const float2 v = __ldg(src + e);
      m = fmaxf(m, fmaxf(fabsf(v.x), fabsf(v.y)));
    }
  }
  for (int o = 16; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
  __shared__ float wm[NT / 32];
  if ((threadIdx.x & 31) == 0) wm[threadIdx.x >> 5] = m;
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int w = 1; w < NT / 32; ++w) m = fmaxf(m, wm[w]);
    atomicMax(maxbits + z, __float_as_uint(m));
  }
}

// The split pass as a tiled transpose.  An operand is a dense block of 2^R
// elements and so is each plane; they differ in the order of their R index
// bits.  A tile is the 2^T elements spanned by T of those bits, chosen to hold
// both the output's fastest bits and the input's fastest ones, so whatever the
// order, a CTA reads runs of 2^(T/2) input elements and writes runs of
// 2^(T/2) values per plane, and turns the tile in shared memory.  (Reading 8
// values per thread through the index strides touched a 32-byte sector per
// 8-byte element on random orders: a 2^29-element operand took 2.8 ms for its
// maximum and 3.4 ms for its split, whose bytes move in 0.64 and 1.3 ms; the
// (16, 6, 13) contraction it belongs to went from 7.3 to 3.4 ms with this.)  The
// loads go past L1, where a line would stay for nothing: log2 M, N, K = (13, 6, 13)
// in scaled fp16 302 us per call, through L1 about 20 us more.
struct TileMap {
  int nout;                 // index bits outside the tile
  int32_t out_src[kMaxBits];   // their strides in the input ..
  int8_t out_dst[kMaxBits];    // .. and their bit positions in a plane
  // the tile's bits in input order (fastest first): input stride, and what the
  // bit flips in the element's shared-memory slot
  int32_t in_src[12], in_slot[12];
  // .. and in output order: what the bit flips in the slot, bit position in a plane
  int32_t out_slot[12];
  int8_t dst[12];
};

// One operand of a launch: its tensors (z: number nlo per lo stride, then hi),
// where their planes go, and the scaled formats' maxima and exponents.
struct SplitJob {
  const float2* src;
  uint16_t* dst;
  int bits, nlo, vec;
  int64_t lo, hi;
  const unsigned* maxbits;
  int* e_out;
  float* m_out;
};

template <int NP, int T, bool BF16>
__device__ __forceinline__ void split_tile(const SplitJob& job, const TileMap& tm, unsigned blk, int64_t z) {
  let_next_start();
  after_previous();
  constexpr int E = 1 << T;
  __shared__ __align__(16) float2 tile[E];
  const float2* src = job.src + (z % job.nlo) * job.lo + (z / job.nlo) * job.hi;
  const bool vec = job.vec != 0;
  int e = 0;
  if (job.maxbits) {
    const float mx = __uint_as_float(job.maxbits[z]);
    e = scale_exponent(mx);
    if (blk == 0 && threadIdx.x == 0) {
      job.e_out[z] = e;
      job.m_out[z] = ldexpf(mx, -e);
    }
  }
  const Pow2 sc(-e);
  const int64_t plane = int64_t(1) << job.bits;
  uint16_t* out = job.dst + z * NP * plane;
  {
    int32_t so = 0;
    int64_t dofs = 0;
    for (int b = 0; b < tm.nout; ++b)
      if ((blk >> b) & 1) {
        so += tm.out_src[b];
        dofs += int64_t(1) << tm.out_dst[b];
      }
    src += so;
    out += dofs;
  }
  const int t = threadIdx.x;
  // load: pairs of input-adjacent elements, pair q = t + NT j (bits 1.. of the input order)
  constexpr int PAIRS = E / 2, PL = PAIRS < NT ? PAIRS : NT, NJ = PAIRS / PL;
  constexpr int TB = PL == 256 ? 8 : PL == 128 ? 7 : 6;  // bits of t in a pair index
  static_assert(PL == (1 << TB), "tile size");
  if (t < PL) {
    int32_t so = 0, slot = 0;
#pragma unroll
    for (int b = 0; b < TB; ++b)
      if ((t >> b) & 1) {
        so += tm.in_src[1 + b];
        slot ^= tm.in_slot[1 + b];
      }
    float2 v[NJ][2];
#pragma unroll
    for (int j = 0; j < NJ; ++j) {
      int32_t o = so;
#pragma unroll
      for (int b = 0; b < T - 1 - TB; ++b)
        if ((j >> b) & 1) o += tm.in_src[1 + TB + b];
      if (vec) {
        const float4 x = __ldcg(reinterpret_cast<const float4*>(src + o));
        v[j][0] = make_float2(x.x, x.y);
        v[j][1] = make_float2(x.z, x.w);
      } else {
        v[j][0] = __ldcg(src + o);
        v[j][1] = __ldcg(src + o + 1);
      }
    }
#pragma unroll
    for (int j = 0; j < NJ; ++j) {
      int32_t p = slot;
#pragma unroll
      for (int b = 0; b < T - 1 - TB; ++b)
        if ((j >> b) & 1) p ^= tm.in_slot[1 + TB + b];
      tile[p] = v[j][0];
      tile[p ^ tm.in_slot[0]] = v[j][1];
    }
  }
  __syncthreads();
  // store: eight consecutive output elements per thread
  constexpr int GROUPS = E / 8, GL = GROUPS < NT ? GROUPS : NT;
  if (t < GL) {
#pragma unroll
    for (int g0 = 0; g0 < GROUPS; g0 += GL) {
      const int g = g0 + t;
      int32_t slot = 0;
      int64_t o = 0;
#pragma unroll
      for (int b = 3; b < T; ++b)
        if ((g >> (b - 3)) & 1) {
          slot ^= tm.out_slot[b];
          o += int64_t(1) << tm.dst[b];
        }
      f32x2 v[8];
#pragma unroll
      for (int c = 0; c < 4; ++c) {
        const ulonglong2 y = *reinterpret_cast<const ulonglong2*>(&tile[slot ^ (2 * c)]);
        v[2 * c] = y.x;
        v[2 * c + 1] = y.y;
      }
      // (one multiply but for exponents out of a float's range)
      if (sc.direct) {
#pragma unroll
        for (int j = 0; j < 8; ++j) v[j] = mul2(v[j], pack2(sc.f, sc.f));
      } else {
#pragma unroll
        for (int j = 0; j < 8; ++j) {
          const float2 x = unpack2(v[j]);
          v[j] = pack2(sc(x.x), sc(x.y));
        }
      }
      uint4 p[NP];
      planes8<NP, BF16>(v, p);
#pragma unroll
      for (int i = 0; i < NP; ++i) *reinterpret_cast<uint4*>(out + o + i * plane) = p[i];
    }
  }
}

template <int NP, int T, bool BF16>
__global__ void __launch_bounds__(NT) split_kernel(const SplitJob job, const __grid_constant__ TileMap tm) {
  split_tile<NP, T, BF16>(job, tm, blockIdx.x, blockIdx.y);
}

// Both operands of one contraction in one launch: the first blocks take A's
// tiles, the others B's.
template <int NP, int T, bool BF16>
__global__ void __launch_bounds__(NT) split_pair_kernel(const SplitJob a, const __grid_constant__ TileMap ta,
                                                        const SplitJob b, const __grid_constant__ TileMap tb) {
  const unsigned na = 1u << (a.bits - T);
  if (blockIdx.x < na) split_tile<NP, T, BF16>(a, ta, blockIdx.x, 0);
  else split_tile<NP, T, BF16>(b, tb, blockIdx.x - na, 0);
}

// The tile of T bits for an operand whose output bit i (K bits, then row bits)
// has input stride st[i], R bits in all.
template <int T>
TileMap split_tile_map(const SplitDesc& d) {
  TileMap m{};
  const int R = d.nk + d.nrow;
  int32_t st[kMaxBits];
  for (int i = 0; i < R; ++i) st[i] = i < d.nk ? d.k_st[i] : d.row_st[i - d.nk];
  bool in[kMaxBits] = {};
  int count = 0;
  auto take = [&](int i) {
    if (!in[i] && count < T) {
      in[i] = true;
      ++count;
    }
  };
  for (int i = 0; i < T / 2; ++i) take(i);
  for (int i = 0; i < R; ++i)
    if (st[i] < (int32_t(1) << ((T + 1) / 2))) take(i);
  for (int i = 0; i < R; ++i) take(i);
  int pos[kMaxBits];  // output-order position in the tile
  int nd = 0;
  for (int i = 0; i < R; ++i) {
    if (in[i]) {
      pos[i] = nd;
      m.dst[nd++] = (int8_t)i;
    } else {
      m.out_src[m.nout] = st[i];
      m.out_dst[m.nout++] = (int8_t)i;
    }
  }
  int order[12], n = 0;  // the tile's output bits by input stride
  for (int i = 0; i < R; ++i)
    if (in[i]) {
      int j = n++;
      for (; j > 0 && st[order[j - 1]] > st[i]; --j) order[j] = order[j - 1];
      order[j] = i;
    }
  int tile_order[12];
  for (int l = 0; l < T; ++l) tile_order[l] = pos[order[l]];
  turn_slots<T>(tile_order, m.out_slot);
  for (int l = 0; l < T; ++l) {
    m.in_src[l] = st[order[l]];
    m.in_slot[l] = m.out_slot[pos[order[l]]];
  }
  return m;
}

// Tile size for an operand of 2^R elements, nz of them: 2^12 once there are four
// such tiles per SM (six CTAs fit one); smaller tiles spread a small operand over
// more SMs.
int tile_bits(int R, int nz) {
  return R >= 12 && (int64_t(1) << (R - 12)) * nz >= 152 * 4 ? 12 : R >= 10 ? 10 : 7;
}

template <class F>
cudaError_t for_format(int np, bool bf16, int T, F&& f) {
  using std::integral_constant;
  auto t = [&](auto n, auto fmt) {
    return T == 12   ? f(n, integral_constant<int, 12>{}, fmt)
           : T == 10 ? f(n, integral_constant<int, 10>{}, fmt)
                     : f(n, integral_constant<int, 7>{}, fmt);
  };
  auto n = [&](auto fmt) { return np == 4 ? t(integral_constant<int, 4>{}, fmt) : t(integral_constant<int, 2>{}, fmt); };
  return bf16 ? n(std::true_type{}) : n(std::false_type{});
}

bool vec_ok(const float2* src, const SplitDesc& d) {
  return (reinterpret_cast<uintptr_t>(src) & 15) == 0 && (d.lo & 1) == 0 && (d.hi & 1) == 0;
}

SplitJob split_job(const float2* src, uint16_t* dst, const SplitDesc& d, const unsigned* maxbits, int* e_out,
                   float* m_out) {
  return {src, dst, d.nk + d.nrow, d.nlo, vec_ok(src, d), d.lo, d.hi, maxbits, e_out, m_out};
}

// Both maxima of a contraction's operands by one CTA each, stored (no clearing,
// no atomics): for operands that one CTA reads in a microsecond or two.
constexpr int MAX_SMALL_BITS = 15;
__global__ void __launch_bounds__(1024) max_small_kernel(const float2* a, int abits, const float2* b, int bbits,
                                                         unsigned* __restrict__ maxbits) {
  let_next_start();
  after_previous();
  const float2* p = blockIdx.x ? b : a;
  const int n = 1 << (blockIdx.x ? bbits : abits);
  float m = 0.f;
#pragma unroll 8
  for (int e = threadIdx.x; e < n; e += 1024) {
    const float2 v = p[e];
    m = fmaxf(m, fmaxf(fabsf(v.x), fabsf(v.y)));
  }
  __shared__ unsigned wm[32];
  const unsigned w = __reduce_max_sync(0xffffffffu, __float_as_uint(m));
  if ((threadIdx.x & 31) == 0) wm[threadIdx.x >> 5] = w;
  __syncthreads();
  if (threadIdx.x < 32) {
    const unsigned x = __reduce_max_sync(0xffffffffu, wm[threadIdx.x]);
    if (threadIdx.x == 0) maxbits[blockIdx.x] = x;
  }
}

}  // namespace

cudaError_t launch_max(const float2* src, int bits, int nz, int nlo, int64_t lo, int64_t hi, bool vec, unsigned* maxbits,
                       cudaStream_t s) {
  // 8 loads of 16 bytes per thread where there is enough to fill the chip
  const int64_t n = int64_t(1) << (bits - 1);
  const int64_t blocks = std::max<int64_t>(1, std::min<int64_t>(n / (NT * 8), 152 * 8));
  max_kernel<<<dim3((unsigned)blocks, (unsigned)nz), NT, 0, s>>>(src, bits, nlo, lo, hi, vec, maxbits);
  return cudaGetLastError();
}

cudaError_t launch_split(const float2* src, uint16_t* dst, const SplitDesc& d, int nz, bool bf16, int np,
                         unsigned* maxbits, int* e_out, float* m_out, cudaStream_t s, bool max_ready) {
  const int R = d.nk + d.nrow;
  if (nz < 1 || nz > 65535 || R < 7 || R > 30 || (np != 2 && np != 4)) return cudaErrorInvalidValue;
  if (maxbits && !max_ready) {
    const cudaError_t e = launch_max(src, R, nz, d.nlo, d.lo, d.hi, vec_ok(src, d), maxbits, s);
    if (e != cudaSuccess) return e;
  }
  const SplitJob job = split_job(src, dst, d, maxbits, e_out, m_out);
  return for_format(np, bf16, tile_bits(R, nz), [&](auto n, auto t, auto fmt) {
    constexpr int T = decltype(t)::value;
    return launch_overlapped(split_kernel<decltype(n)::value, T, decltype(fmt)::value>,
                             dim3(1u << (R - T), (unsigned)nz), dim3(NT), 0, s, job, split_tile_map<T>(d));
  });
}

namespace {
void split_desc(int nrow, const int32_t* row_st, int nk, const int32_t* k_st, int nlo, int64_t lo, int64_t hi,
                SplitDesc& sd) {
  sd.nrow = nrow;
  sd.nk = nk;
  sd.nlo = nlo;
  sd.lo = lo;
  sd.hi = hi;
  for (int i = 0; i < nrow; ++i) sd.row_st[i] = row_st[i];
  for (int i = 0; i < nk; ++i) sd.k_st[i] = k_st[i];
}
int distinct(const GemmDesc& d, int64_t lo, int64_t hi) {
  return (lo ? d.units_lo : 1) * (hi ? d.units / d.units_lo : 1);
}
}  // namespace

int64_t split_scratch_elems(const GemmDesc& d, bool which_b, int np) {
  return which_b ? split_plane_elems(d.nn, d.nk, np) * distinct(d, d.b_lo, d.b_hi)
                 : split_plane_elems(d.nm, d.nk, np) * distinct(d, d.a_lo, d.a_hi);
}

int64_t tc2_scratch_elems(const GemmDesc& d) { return split_scratch_elems(d, false, 4) + split_scratch_elems(d, true, 4); }

namespace {
// An operand's split view, number of distinct tensors, and its planes at `scratch`.
SplitDesc operand_view(const GemmDesc& d, bool which_b, int np, const uint16_t* scratch, int& nz, PlaneOperand& out) {
  const int64_t lo = which_b ? d.b_lo : d.a_lo, hi = which_b ? d.b_hi : d.a_hi;
  const int nrow = which_b ? d.nn : d.nm;
  SplitDesc sd;
  split_desc(nrow, which_b ? d.bn : d.am, d.nk, which_b ? d.bk : d.ak, lo ? d.units_lo : 1, lo, hi, sd);
  nz = distinct(d, lo, hi);
  const int64_t K = int64_t(1) << d.nk;  // tensor-core shapes have K >= 8: whole 16-byte chunks, no padding
  const int64_t set = (int64_t)np * (int64_t(1) << nrow) * K * 2;
  out.base = scratch;
  out.np = np;
  out.kp = K;
  out.rows = int64_t(1) << nrow;
  out.nlo = lo ? d.units_lo : 1;
  out.nhi = hi ? d.units / d.units_lo : 1;
  out.st_lo = set;
  out.st_hi = set * out.nlo;
  return sd;
}
}  // namespace

cudaError_t split_operand(const float2* src, const GemmDesc& d, bool which_b, bool bf16, int np, bool scaled,
                          unsigned* maxbits, int* e_out, float* m_out, uint16_t* scratch, PlaneOperand& out,
                          cudaStream_t s, bool max_ready) {
  int nz;
  const SplitDesc sd = operand_view(d, which_b, np, scratch, nz, out);
  return launch_split(src, scratch, sd, nz, bf16, np, scaled ? maxbits : nullptr, e_out, m_out, s, max_ready);
}

// The maxima of a one-unit contraction's operands, mx[0] of A and mx[1] of B.
static cudaError_t pair_maxima(const float2* A, const float2* B, const GemmDesc& d, unsigned* mx, cudaStream_t s) {
  const int ra = d.nm + d.nk, rb = d.nn + d.nk;
  if (ra <= MAX_SMALL_BITS && rb <= MAX_SMALL_BITS) {
    return launch_overlapped(max_small_kernel, dim3(2), dim3(1024), 0, s, A, ra, B, rb, mx);
  }
  cudaError_t e = cudaMemsetAsync(mx, 0, 2 * sizeof(unsigned), s);
  const auto vec = [](const float2* p) { return (reinterpret_cast<uintptr_t>(p) & 15) == 0; };
  if (e == cudaSuccess) e = launch_max(A, ra, 1, 1, 0, 0, vec(A), mx, s);
  if (e == cudaSuccess) e = launch_max(B, rb, 1, 1, 0, 0, vec(B), mx + 1, s);
  return e;
}

// Both operands of a one-unit contraction: one launch where one tile size suits
// both (a launch saved is 3 us of a call that small), else one each.  mx (may be
// null): their maxima, with ex, ms receiving the exponents and stored maxima.
static cudaError_t split_pair(const float2* A, const float2* B, const GemmDesc& d, bool bf16, int np, unsigned* mx,
                              int* ex, float* ms, uint16_t* scratch, PlaneOperand& pa, PlaneOperand& pb,
                              cudaStream_t s) {
  int nz;
  uint16_t* const sb = scratch + split_scratch_elems(d, false, np);
  const SplitDesc da = operand_view(d, false, np, scratch, nz, pa), db = operand_view(d, true, np, sb, nz, pb);
  const int ra = d.nm + d.nk, rb = d.nn + d.nk;
  const int ta = tile_bits(ra, 1), tb = tile_bits(rb, 1);
  const SplitJob ja = split_job(A, scratch, da, mx, ex, ms);
  const SplitJob jb = split_job(B, sb, db, mx ? mx + 1 : nullptr, ex ? ex + 1 : nullptr, ms ? ms + 1 : nullptr);
  const int T = ta < tb ? ta : tb, large = ra > rb ? ra : rb;
  if (ta == tb || (T == 10 && large <= 20) || (T == 7 && large <= 14))
    return for_format(np, bf16, T, [&](auto n, auto t, auto fmt) {
      constexpr int TT = decltype(t)::value;
      return launch_overlapped(split_pair_kernel<decltype(n)::value, TT, decltype(fmt)::value>,
                               dim3((1u << (ra - TT)) + (1u << (rb - TT))), dim3(NT), 0, s, ja, split_tile_map<TT>(da),
                               jb, split_tile_map<TT>(db));
    });
  const cudaError_t e = launch_split(A, scratch, da, 1, bf16, np, mx, ex, ms, s, true);
  return e != cudaSuccess ? e
                          : launch_split(B, sb, db, 1, bf16, np, mx ? mx + 1 : nullptr, ex ? ex + 1 : nullptr,
                                         ms ? ms + 1 : nullptr, s, true);
}

bool planes_in_place(const float2* base, const GemmDesc& d, bool which_b, int np, PlaneOperand& out) {
  const int nrow = which_b ? d.nn : d.nm;
  const int32_t* rs = which_b ? d.bn : d.am;
  const int32_t* ks = which_b ? d.bk : d.ak;
  const int64_t K = int64_t(1) << d.nk;
  if (K < 8) return false;
  for (int l = 0; l < d.nk; ++l)
    if (ks[l] != (int32_t(1) << l)) return false;
  for (int i = 0; i < nrow; ++i)
    if ((int64_t)rs[i] != (K << i)) return false;
  const int64_t lo = which_b ? d.b_lo : d.a_lo, hi = which_b ? d.b_hi : d.a_hi;
  out.base = reinterpret_cast<const uint16_t*>(base);
  out.np = np;
  out.kp = K;
  out.rows = int64_t(1) << nrow;
  out.nlo = lo ? d.units_lo : 1;
  out.nhi = hi ? d.units / d.units_lo : 1;
  out.st_lo = lo * 8;
  out.st_hi = hi * 8;
  return true;
}

int64_t tc2_pair_scratch_elems(const GemmDesc& d, bool sums) {
  return direct_ok(d) ? split_scratch_elems(d, true, 4) : tc2_scratch_elems(d) + (sums ? tc_part_elems(d, 4, false) : 0);
}

static float2* part_space(const GemmDesc& d, int np, uint16_t* scratch, bool sums) {
  return sums && tc_part_elems(d, np, false) > 0 ? reinterpret_cast<float2*>(scratch + tc2_scratch_elems(d)) : nullptr;
}

cudaError_t run_gemm_tc2(const float2* A, const float2* B, float2* C, const GemmDesc& d0, bool bf16, bool sums,
                         uint16_t* scratch, int* err, cudaStream_t s) {
  PlaneOperand pa, pb;
  GemmDesc d = d0;
  if (direct_ok(d)) {
    order_for_direct(d);
    const cudaError_t e = split_operand(B, d, true, bf16, 4, false, nullptr, nullptr, nullptr, scratch, pb, s);
    return e != cudaSuccess ? e : launch_gemm_direct(A, pb, C, d, bf16, nullptr, nullptr, err, s);
  }
  // the split pass reads any order of rows at the same speed, so they follow C
  // (random orders, scaled bf16 (14, 14, 5): 2040 -> 832 us per call)
  order_by_output(d);
  const cudaError_t e = split_pair(A, B, d, bf16, 4, nullptr, nullptr, nullptr, scratch, pa, pb, s);
  if (e != cudaSuccess) return e;
  const ScaleIO none{};
  return launch_gemm_tma(pa, pb, C, false, d, bf16, none, err, s, part_space(d, 4, scratch, sums));
}

cudaError_t run_gemm_tc2_scaled(const float2* A, const float2* B, float2* C, const GemmDesc& d0, bool bf16, int np,
                                bool sums, uint16_t* scratch, void* aux, int* err, cudaStream_t s) {
  unsigned* mx = reinterpret_cast<unsigned*>(aux);
  int* ex = reinterpret_cast<int*>(mx + 2);
  float* ms = reinterpret_cast<float*>(ex + 2);
  GemmDesc d = d0;
  cudaError_t e = pair_maxima(A, B, d, mx, s);
  if (e != cudaSuccess) return e;
  PlaneOperand pa, pb;
  if (direct_ok(d)) {
    order_for_direct(d);
    e = split_operand(B, d, true, bf16, np, true, mx + 1, ex + 1, ms + 1, scratch, pb, s, true);
    return e != cudaSuccess ? e : launch_gemm_direct(A, pb, C, d, bf16, mx, ex + 1, err, s);
  }
  order_by_output(d);
  e = split_pair(A, B, d, bf16, np, mx, ex, ms, scratch, pa, pb, s);
  if (e != cudaSuccess) return e;
  ScaleIO sio{};
  sio.ea = ex;
  sio.ma = ms;
  sio.eb = ex + 1;
  sio.mb = ms + 1;
  return launch_gemm_tma(pa, pb, C, false, d, bf16, sio, err, s, part_space(d, np, scratch, sums));
}

}  // namespace tn
