// Arithmetic shared by the stencil kernels (aew_stencil.cu streams planes from HBM,
// aew_brick.cuh keeps a small grid on chip): the face updates, the source and the packing
// helpers.  Both families call the same expressions, so their results are bitwise equal.
#pragma once

#include <cuda_bf16.h>

#include "aew_gemm.cuh"
#include "aew_internal.cuh"

namespace aew {

__device__ __forceinline__ void st4(float* p, size_t i, float4 v) {
  *reinterpret_cast<float4*>(p + i) = v;
}
__device__ __forceinline__ float& comp(float4& v, int c) {
  return c == 0 ? v.x : (c == 1 ? v.y : (c == 2 ? v.z : v.w));
}
__device__ __forceinline__ float4 z4() { return make_float4(0.f, 0.f, 0.f, 0.f); }
// the source's force on the z-faces of the 4 nodes (k, y, i0 .. i0 + 3): dts times the
// spread weight of each face inside the source box (a point source: the one face, 1)
template <class Step>
__device__ __forceinline__ void add_source(float4& v, int k, int y, int i0, const Step& a,
                                           float dts) {
  if (a.sk < 0) return;
  const int W = 2 * a.sr + 1;
  const int dk = k - a.sk + a.sr, dy = y - a.sj + a.sr;
  if ((unsigned)dk >= (unsigned)W || (unsigned)dy >= (unsigned)W) return;
  const float* w = a.src_w + ((size_t)dk * W + dy) * W;
#pragma unroll
  for (int d = 0; d < 4; ++d) {
    const int dx = i0 + d - a.si + a.sr;
    if ((unsigned)dx < (unsigned)W) comp(v, d) = fmaf(dts, __ldg(w + dx), comp(v, d));
  }
}
// The m e products are plain multiplies; the face updates below subtract them with
// __fsub_rn, which the compiler never merges with a multiply, so every face is
// fma(dth, round(m_hi e_hi) - round(m_lo e_lo), v) wherever it is computed: by its
// owner, or recomputed at a chunk's first plane or by the neighbouring lane.  (Left to
// the compiler, a subtraction could absorb one product into an FMA at one site and not
// at another, and the results then depended in the last bit on the z-chunk depth.)
__device__ __forceinline__ float4 mul4(float4 a, float4 b) {
  return make_float4(a.x * b.x, a.y * b.y, a.z * b.z, a.w * b.w);
}
__device__ __forceinline__ float4 fma4(float4 a, float4 b, float4 c) {
  return make_float4(fmaf(a.x, b.x, c.x), fmaf(a.y, b.y, c.y), fmaf(a.z, b.z, c.z),
                     fmaf(a.w, b.w, c.w));
}
// 1 / s for a block maximum m >= 0 given as float bits, equal to
// gemm::block_inv_scale(m) (s = 2^max(e, -100), m = f 2^e with f in [0.5, 1); 0 for
// m = 0) but from the exponent field: e = biased - 126 for normal m, and subnormal m
// falls under the clamp.  Maxima of 2^126 and above take the library path.
__device__ __forceinline__ float inv_scale_bits(uint32_t mb) {
  const int eb = (int)(mb >> 23);
  if (mb == 0u) return 0.f;
  if (eb >= 253) return gemm::block_inv_scale(__uint_as_float(mb));
  const int e = max(eb - 126, gemm::kExpMin);
  return __uint_as_float((uint32_t)(127 - e) << 23);
}
__device__ __forceinline__ float hmax4(float4 a) {
  return fmaxf(fmaxf(fabsf(a.x), fabsf(a.y)), fmaxf(fabsf(a.z), fabsf(a.w)));
}
__device__ __forceinline__ uint32_t pack2bf(float a, float b) {
  __nv_bfloat162 t = __floats2bfloat162_rn(a, b);
  return *reinterpret_cast<uint32_t*>(&t);
}
// face update v' = v + dth (hi - lo), the difference rounded on its own (see above)
__device__ __forceinline__ float fupd(float dth, float hi, float lo, float v) {
  return fmaf(dth, __fsub_rn(hi, lo), v);
}
__device__ __forceinline__ float4 fupd4(float dth, float4 hi, float4 lo, float4 v) {
  return make_float4(fupd(dth, hi.x, lo.x, v.x), fupd(dth, hi.y, lo.y, v.y),
                     fupd(dth, hi.z, lo.z, v.z), fupd(dth, hi.w, lo.w, v.w));
}
// lam' = (lam + inj) + dth (mu - mu_hi)
__device__ __forceinline__ float lupd(float dth, float mu_hi, float mu, float l) {
  return fmaf(dth, mu - mu_hi, l);
}
__device__ __forceinline__ float4 lupd4(float dth, float4 hi, float4 lo, float4 l) {
  return make_float4(lupd(dth, hi.x, lo.x, l.x), lupd(dth, hi.y, lo.y, l.y),
                     lupd(dth, hi.z, lo.z, l.z), lupd(dth, hi.w, lo.w, l.w));
}

__device__ __forceinline__ bool sticky_error(const int* err) {
  return err && *reinterpret_cast<const volatile int*>(err) != 0;
}

// The same value in FP64, by integer instructions: GB300 converts at its FP64 rate, which made
// the conversions half of a window's flush into the FP64 sum (a 256^3 two-step adjoint pass
// that ends a window: 249 -> 216 us; the on-chip loops, short of registers, gain nothing by it
// and convert by instruction).
__device__ __forceinline__ double widen(float v) {
  uint32_t u = __float_as_uint(v);
  int bias = 1023 - 127;
  if ((u & 0x7f800000u) == 0) {   // subnormal or zero: exact as 2^64 v
    u = __float_as_uint(v * 18446744073709551616.f);
    bias -= 64;
  }
  const int e = (int)(u >> 23 & 0xffu);
  const uint32_t ed = e == 255 ? 2047u : e == 0 ? 0u : (uint32_t)(e + bias);
  return __hiloint2double((int)((u & 0x80000000u) | ed << 20 | (u & 0x7fffffu) >> 3), (int)(u << 29));
}
// acc[0 .. 3] += v
__device__ __forceinline__ void add_wide(double* acc, float4 v) {
  double2* p = reinterpret_cast<double2*>(acc);
  double2 lo = p[0], hi = p[1];
  lo.x += widen(v.x);
  lo.y += widen(v.y);
  hi.x += widen(v.z);
  hi.y += widen(v.w);
  p[0] = lo;
  p[1] = hi;
}

// ---- four nodes as two pairs ---------------------------------------------------------
namespace quad {
// The paired FP32 instructions round each lane as the scalar ones do.
struct F4 {
  uint64_t a, b;
};
__device__ __forceinline__ F4 f4(float4 v) {
  return F4{gemm::f2::make(v.x, v.y), gemm::f2::make(v.z, v.w)};
}
__device__ __forceinline__ float4 v4(F4 f) {
  float4 v;
  gemm::f2::split(f.a, v.x, v.y);
  gemm::f2::split(f.b, v.z, v.w);
  return v;
}
__device__ __forceinline__ F4 add(F4 x, F4 y) { return F4{gemm::f2::add(x.a, y.a), gemm::f2::add(x.b, y.b)}; }
__device__ __forceinline__ F4 sub(F4 x, F4 y) { return F4{gemm::f2::sub(x.a, y.a), gemm::f2::sub(x.b, y.b)}; }
__device__ __forceinline__ F4 mul(F4 x, F4 y) { return F4{gemm::f2::mul(x.a, y.a), gemm::f2::mul(x.b, y.b)}; }
__device__ __forceinline__ F4 fma(F4 x, F4 y, F4 z) {
  return F4{gemm::f2::fma(x.a, y.a, z.a), gemm::f2::fma(x.b, y.b, z.b)};
}
__device__ __forceinline__ F4 lds(const float4* p) { return f4(*p); }
__device__ __forceinline__ void sts(float4* p, F4 v) { *p = v4(v); }
// l plus the residual row's component (r points at it) at the receivers of four nodes
__device__ __forceinline__ F4 injected(F4 f, const int* rec_map, const float* r) {
  const int4 m = __ldg(reinterpret_cast<const int4*>(rec_map));
  float4 l = v4(f);
  if (m.x >= 0) l.x += __ldg(r + 3 * m.x);
  if (m.y >= 0) l.y += __ldg(r + 3 * m.y);
  if (m.z >= 0) l.z += __ldg(r + 3 * m.z);
  if (m.w >= 0) l.w += __ldg(r + 3 * m.w);
  return f4(l);
}
}  // namespace quad

__device__ __forceinline__ float4 ldg4(const float* p) {
  return __ldg(reinterpret_cast<const float4*>(p));
}
__device__ __forceinline__ float4 bf4(uint2 b) {
  return make_float4(__uint_as_float(b.x << 16), __uint_as_float(b.x & 0xffff0000u),
                     __uint_as_float(b.y << 16), __uint_as_float(b.y & 0xffff0000u));
}
// some of four nodes carry a receiver (rec_map points at theirs)
__device__ __forceinline__ bool has_rec(const int* rec_map) {
  const int4 m = __ldg(reinterpret_cast<const int4*>(rec_map));
  return m.x >= 0 || m.y >= 0 || m.z >= 0 || m.w >= 0;
}
// the face values of four nodes to the receiver row d
__device__ __forceinline__ void record(const int* rec_map, float* d, float4 x, float4 y, float4 z) {
  const int4 r = __ldg(reinterpret_cast<const int4*>(rec_map));
  const int rr[4] = {r.x, r.y, r.z, r.w};
#pragma unroll
  for (int c = 0; c < 4; ++c)
    if (rr[c] >= 0) {
      d[3 * rr[c] + 0] = comp(x, c);
      d[3 * rr[c] + 1] = comp(y, c);
      d[3 * rr[c] + 2] = comp(z, c);
    }
}

}  // namespace aew
