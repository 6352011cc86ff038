// Device helpers shared by the kernels.
#pragma once

#include <cuda_bf16.h>
#include <cuda_fp16.h>
#include <cuda_runtime.h>

#include <utility>

#include "kernels.h"

namespace tn {

// Slice selection: offset in the leaf store of unit u's sub-tensor of a leaf
// (its fixed indices set to the unit's slice id and bitstring bits), and of the
// sub-tensor's element e.
__device__ __forceinline__ int64_t leaf_fixed_offset(const LeafGather& L, const GroupInfo& g, int u) {
  const int64_t s = g.slice0 + u % g.nslice;
  const int64_t b = g.b0 + u / g.nslice;
  int64_t o = L.store_off;
  for (int f = 0; f < L.nfixed; ++f) {
    const int src = L.fixed_src[f];
    int v;
    if (src >= 0) v = (int)((s >> src) & 1);
    else {
      const int q = -src - 2;
      v = (int)((g.bits[b * g.words + (q >> 6)] >> (q & 63)) & 1);
    }
    if (v) o += L.fixed_stride[f];
  }
  return o;
}
__device__ __forceinline__ int64_t leaf_kept_offset(const LeafGather& L, int64_t fixed_off, int e) {
  int64_t o = fixed_off;
  for (int p = 0; p < L.nkept; ++p)
    if ((e >> (L.nkept - 1 - p)) & 1) o += L.kept_stride[p];
  return o;
}

// Multiplication by 2^e for the exponent shifts of the scaled formats.  A
// power of two in the normal range multiplies exactly, so one multiply gives
// the correctly rounded x 2^e (the value ldexpf returns); shifts outside
// [-126, 127] go through ldexpf.
struct Pow2 {
  int e;
  float f;
  bool direct;
  __device__ explicit Pow2(int e_) {
    e = e_;
    direct = e_ >= -126 && e_ <= 127;
    f = __int_as_float((min(max(e_, -126), 127) + 127) << 23);
  }
  __device__ float operator()(float x) const { return direct ? x * f : ldexpf(x, e); }
};

// Packed FP32: two values per instruction.
using f32x2 = unsigned long long;
__device__ __forceinline__ f32x2 pack2(float x, float y) {
  f32x2 r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(x), "f"(y));
  return r;
}
__device__ __forceinline__ float2 unpack2(f32x2 v) {
  float2 r;
  asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(v));
  return r;
}
__device__ __forceinline__ f32x2 mul2(f32x2 a, f32x2 b) {
  f32x2 r;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ f32x2 fma2(f32x2 a, f32x2 b, f32x2 c) {
  f32x2 r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
  return r;
}

// Eight complex values (consecutive in K order) as NP 16-bit planes of 16 bytes:
// four planes, x = hi + lo with hi = rn16(x) and lo = rn16(x - hi), in the order
// re_hi, re_lo, im_hi, im_lo; or two, x rounded once, re, im.
template <int NP, bool BF16>
__device__ __forceinline__ void planes8(const f32x2 (&v)[8], uint4 (&out)[NP]) {
  uint32_t hi[8], lo[8];  // re | im << 16
  const f32x2 minus = pack2(-1.f, -1.f);
#pragma unroll
  for (int j = 0; j < 8; ++j) {
    const float2 x = unpack2(v[j]);
    float2 f;
    if (BF16) {
      const __nv_bfloat162 h = __floats2bfloat162_rn(x.x, x.y);
      hi[j] = *reinterpret_cast<const uint32_t*>(&h);
      f = __bfloat1622float2(h);
    } else {
      const __half2 h = __floats2half2_rn(x.x, x.y);
      hi[j] = *reinterpret_cast<const uint32_t*>(&h);
      f = __half22float2(h);
    }
    if (NP == 4) {
      const float2 d = unpack2(fma2(pack2(f.x, f.y), minus, v[j]));  // x - hi, rounded once
      if (BF16) {
        const __nv_bfloat162 l = __floats2bfloat162_rn(d.x, d.y);
        lo[j] = *reinterpret_cast<const uint32_t*>(&l);
      } else {
        const __half2 l = __floats2half2_rn(d.x, d.y);
        lo[j] = *reinterpret_cast<const uint32_t*>(&l);
      }
    }
  }
  auto row = [](const uint32_t* x, unsigned half) {
    return make_uint4(__byte_perm(x[0], x[1], half), __byte_perm(x[2], x[3], half), __byte_perm(x[4], x[5], half),
                      __byte_perm(x[6], x[7], half));
  };
  constexpr unsigned RE = 0x5410, IM = 0x7632;
  out[0] = row(hi, RE);
  out[NP / 2] = row(hi, IM);
  if (NP == 4) {
    out[1] = row(lo, RE);
    out[NP - 1] = row(lo, IM);
  }
}

// Exponent putting a maximum into [2^13, 2^14) (0 for none or a non-finite one).
__device__ __forceinline__ int scale_exponent(float mx) {
  if (!(mx > 0.f) || !isfinite(mx)) return 0;
  int x;
  frexpf(mx, &x);  // mx in [2^(x-1), 2^x)
  return x - 14;
}

// Shared-memory slots of a 2^T-element tile that is written in one index order
// and read in another.  order[l]: the read-order bit that is the l-th of the
// write order.  The element with read-order index x sits at x with bits 4 and 5
// folded onto bits 1 and 2 -- a thread reads 8 elements as four 16-byte loads,
// lanes 64 bytes apart, and the fold spreads every quarter-warp over all banks
// -- and with bits 6.. folded onto bits 1..3 where that makes the slots of a
// half-warp's stores (write-order bits 1..4 vary) independent in the 16 banks.
// slot[b]: what read-order bit b flips.
template <int T>
inline void turn_slots(const int* order, int32_t* slot) {
  for (int b = 0; b < T; ++b) slot[b] = (1 << b) ^ (b == 4 ? 2 : b == 5 ? 4 : 0);
  // span of the chosen lane bits' low four slot bits (bitmap of the 16 vectors)
  unsigned span = 1;
  auto add = [&](int v) {
    unsigned s = span;
    for (int x = 0; x < 16; ++x)
      if ((span >> x) & 1) s |= 1u << (x ^ v);
    span = s;
  };
  for (int l = 1; l <= 4; ++l)
    if (order[l] < 6) add(slot[order[l]] & 15);
  for (int l = 1; l <= 4; ++l) {
    const int p = order[l];
    if (p < 6) continue;
    for (int v = 2; v < 16; v += 2)
      if (!((span >> v) & 1)) {
        slot[p] ^= v;
        add(v);
        break;
      }
  }
}

// Launches that overlap the end of the kernel before them in the stream: the
// next grid's blocks may start once every block of this one has called
// let_next_start (or ended), and hold at after_previous until the whole previous
// grid has finished and its writes are visible.  A kernel launched this way
// calls after_previous before it touches memory that others write or read, and
// reads what earlier kernels wrote by ordinary loads or __ldcg: no __ldg, and no
// `const T* __restrict__` parameter, from which the compiler makes the same
// read-only loads.  Those take the memory as constant for the life of the grid,
// which it is not when the grid starts before its producer has ended, and nothing
// keeps them below the wait.  (What no kernel writes, descriptors and leaves, may be
// read that way.)  A step of a small circuit is a few microseconds, of which a plain
// launch is one or two.
__device__ __forceinline__ void let_next_start() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void after_previous() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

template <class... P, class... A>
inline cudaError_t launch_overlapped(void (*kernel)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t s,
                                     A&&... args) {
  cudaLaunchConfig_t c{};
  c.gridDim = grid;
  c.blockDim = block;
  c.dynamicSmemBytes = smem;
  c.stream = s;
  cudaLaunchAttribute a{};
  a.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  a.val.programmaticStreamSerializationAllowed = 1;
  c.attrs = &a;
  // in a captured sequence, whose replay has no launch cost to hide, plainly
  // (5x5 circuit, 24 kernels: 289 us replayed, 294 with overlapping edges)
  cudaStreamCaptureStatus capture = cudaStreamCaptureStatusNone;
  if (cudaStreamIsCapturing(s, &capture) != cudaSuccess) {
    cudaGetLastError();
    capture = cudaStreamCaptureStatusActive;
  }
  c.numAttrs = capture == cudaStreamCaptureStatusNone ? 1 : 0;
  return cudaLaunchKernelEx(&c, kernel, std::forward<A>(args)...);
}

}  // namespace tn
