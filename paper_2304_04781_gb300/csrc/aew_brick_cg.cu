// The prior solve of grids that fit the SMs: all of its CG iterations in one launch.
//
// A launch per pass took 15 us and more however small the grid.  Here x, r and A p stay in
// registers and p in shared memory, with its halos exchanged as in the time loops
// (aew_brick.cuh), and both inner products of an iteration are all-reduced through one
// tagged word pair per CTA: three L2 round trips per iteration bound it, with the reductions'
// dependent adds.  us per iteration, before -> now: 32^3 21 -> 8, 64^3 37 -> 12, 128^3
// 45 -> 17.
//
// The sums are pairs of floats (value and accumulated rounding error, Knuth's two-sum), as
// exact as FP64 here and without FP64 instructions, whose rate on this GPU would make the
// reductions the longest part.  Every CTA adds the same pairs in the same order, so all take
// the same steps and stop together.
#include "aew_brick.cuh"

namespace aew {
namespace brick {

struct Pair {
  float s, c;
  __device__ __forceinline__ void add(float x, float e = 0.f) {
    const float t = __fadd_rn(s, x), z = __fsub_rn(t, s);
    c = __fadd_rn(__fadd_rn(c, e), __fadd_rn(__fsub_rn(s, __fsub_rn(t, z)), __fsub_rn(x, z)));
    s = t;
  }
};
__device__ __forceinline__ Pair warp_sum(Pair p) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const float s = __shfl_xor_sync(0xffffffffu, p.s, o), c = __shfl_xor_sync(0xffffffffu, p.c, o);
    // both lanes add the lower lane's value first: the same result in both
    const bool up = threadIdx.x & o;
    Pair q{up ? s : p.s, up ? c : p.c};
    q.add(up ? p.s : s, up ? p.c : c);
    p = q;
  }
  return p;
}
// the sum over all CTAs of the threads' pairs (slot: the words of this reduction)
// (*stop: a wait gave up, the same for all threads)
__device__ __forceinline__ Pair all_sum(Pair p, ulonglong2* words, int ctas, uint32_t tag, Pair* scr,
                                        volatile int* dead, int* err, int* stop) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
  p = warp_sum(p);
  if (lane == 0) scr[warp] = p;
  __syncthreads();
  if (warp == 0) {
    Pair q = lane < nw ? scr[lane] : Pair{0.f, 0.f};
    q = warp_sum(q);
    if (lane == 0) {
      const unsigned long long t = (unsigned long long)tag << 32;
      asm volatile("st.relaxed.gpu.global.v2.b64 [%0], {%1, %2};" ::"l"(words + blockIdx.x),
                   "l"(t | __float_as_uint(q.s)), "l"(t | __float_as_uint(q.c))
                   : "memory");
    }
  }
  Pair q{0.f, 0.f};
  for (int i = threadIdx.x; i < ctas; i += blockDim.x) {
    uint32_t t0 = 0;
    for (uint32_t it = 1; !*dead; ++it) {
      const ulonglong2 v = ld_words(words + i);
      if ((uint32_t)(v.x >> 32) == tag && (uint32_t)(v.y >> 32) == tag) {
        q.add(__uint_as_float((uint32_t)v.x), __uint_as_float((uint32_t)v.y));
        break;
      }
      if ((it & 63u) == 0 && !keep_waiting(t0, dead, err)) break;
    }
  }
  q = warp_sum(q);
  Pair* const scr2 = scr + 32;
  if (lane == 0) scr2[warp] = q;
  *stop = __syncthreads_or(*dead);
  Pair r = scr2[0];
  const int n = min(nw, (ctas + 31) / 32);
  for (int w = 1; w < n; ++w) r.add(scr2[w].s, scr2[w].c);
  return r;
}
// a / b in one rounding or so
__device__ __forceinline__ float ratio(Pair a, Pair b) {
  const float q = __fdiv_rn(a.s, b.s);
  return q + __fdiv_rn(fmaf(-q, b.s, a.s) + fmaf(-q, b.c, a.c), b.s);
}

template <int BZ>
__global__ void __launch_bounds__(tmax(BZ), 1) cg_kernel(const __grid_constant__ BrickCg a) {
  using X = Ctx<BZ>;
  constexpr int PE = X::PE;
  extern __shared__ __align__(16) unsigned char smem[];
  __shared__ int dead_s;
  __shared__ Pair scr[64];
  if (sticky_error(a.err)) return;
  float4* const f = reinterpret_cast<float4*>(smem);
  volatile int* dead = &dead_s;
  const Geo g(a);
  const X c(g, a.halo, a.by, a.py, a.pz, a.ny, a.nz);
  const int tid = g.tid, nq = g.nq, ctas = a.py * a.pz;
  if (tid == 0) dead_s = 0;
  if (tid < 64) scr[tid] = Pair{0.f, 0.f};
  c.clear(f);
  ulonglong2* const red = c.wd.base + (2 * (size_t)ctas * (4 * X::TP) + 2 * (size_t)ctas * 4 * BZ * nq);
  const bool y0 = g.y > 0, y1 = g.y + 1 < a.ny, x0 = g.q > 0, x1 = g.q < nq - 1;
  float4* const E = f + X::oE + tid;

  float4 x[BZ], r[BZ], v[BZ];
#pragma unroll
  for (int k = 0; k < BZ; ++k) {
    x[k] = r[k] = z4();
    if (c.bits >> k & 1u) {
      const float4 w = ldg4(a.w + (g.row + k * g.P));
      r[k] = make_float4(a.sc * w.x, a.sc * w.y, a.sc * w.z, a.sc * w.w);
      E[k * PE] = r[k];   // p = r
      if (c.fl & (kLow | kHi)) c.publish_y(g, r[k], a.by, 0, a.tag, k);
    }
  }
  c.publish_z(g, f, 0, a.tag);
  Pair rr{a.rr_hi, a.rr_lo};
  int it = 0, ok = 0, stop = 0;
#pragma unroll 1
  while (it < a.max_iter) {
    const int par = it & 1;
    const uint32_t tag = a.tag + it;
    const float4 below = v4(c.template receive_halos<true>(g, f, a.by, a.py, par, tag, dead, a.err));
    // ---- v = A p and p.v
    Pair acc{0.f, 0.f};
    float4 zm = below;
#pragma unroll
    for (int k = 0; k < BZ; ++k) {
      if (k >= g.ka) continue;
      const float4 p = E[k * PE], zp = E[(k + 1) * PE], ym = E[k * PE - nq], yp = E[k * PE + nq];
      float xl = __shfl_up_sync(0xffffffffu, p.w, 1), xr = __shfl_down_sync(0xffffffffu, p.x, 1);
      if (c.fl & kP0) xl = E[k * PE - 1].w;
      if (c.fl & kP31) xr = E[k * PE + 1].x;
      const bool z0 = g.k0 + k > 0, z1 = g.k0 + k + 1 < a.nz;
      const float pc[4] = {p.x, p.y, p.z, p.w}, am[4] = {ym.x, ym.y, ym.z, ym.w}, ap[4] = {yp.x, yp.y, yp.z, yp.w},
                  bm[4] = {zm.x, zm.y, zm.z, zm.w}, bp[4] = {zp.x, zp.y, zp.z, zp.w};
      float o[4];
#pragma unroll
      for (int q = 0; q < 4; ++q) {   // the order of the streaming operator
        float lap = 0.f;
        if (q > 0 || x0) lap += (q == 0 ? xl : pc[q > 0 ? q - 1 : 0]) - pc[q];
        if (q < 3 || x1) lap += (q == 3 ? xr : pc[q < 3 ? q + 1 : 3]) - pc[q];
        if (y0) lap += am[q] - pc[q];
        if (y1) lap += ap[q] - pc[q];
        if (z0) lap += bm[q] - pc[q];
        if (z1) lap += bp[q] - pc[q];
        o[q] = a.alpha * pc[q] - a.at * lap;
      }
      v[k] = make_float4(o[0], o[1], o[2], o[3]);
      if (c.bits >> k & 1u)
        acc.add(fmaf(p.x, o[0], fmaf(p.y, o[1], fmaf(p.z, o[2], p.w * o[3]))));
      zm = p;
    }
    const Pair pap = all_sum(acc, red + (size_t)par * ctas, ctas, tag, scr, dead, a.err, &stop);
    const float al = pap.s > 0.f ? ratio(rr, pap) : 0.f;
    // ---- x += a p, r -= a A p and r.r
    acc = Pair{0.f, 0.f};
#pragma unroll
    for (int k = 0; k < BZ; ++k) {
      if (!(c.bits >> k & 1u)) continue;
      const float4 p = E[k * PE];
      x[k].x += al * p.x; x[k].y += al * p.y; x[k].z += al * p.z; x[k].w += al * p.w;
      r[k].x -= al * v[k].x; r[k].y -= al * v[k].y; r[k].z -= al * v[k].z; r[k].w -= al * v[k].w;
      acc.add(fmaf(r[k].x, r[k].x, fmaf(r[k].y, r[k].y, fmaf(r[k].z, r[k].z, r[k].w * r[k].w))));
    }
    const Pair rn = all_sum(acc, red + (size_t)(2 + par) * ctas, ctas, tag, scr, dead, a.err, &stop);
    const bool last = it + 1 == a.max_iter;
    if (((it & 7) == 7 || last) && (rn.s - a.tol_hi) + (rn.c - a.tol_lo) <= 0.f) ok = 1;
    const float be = rr.s > 0.f ? ratio(rn, rr) : 0.f;
    rr = rn;
    ++it;
    if (ok || last || stop) break;   // stop: the values are void, and the error flag is set
    // ---- p = r + b p
#pragma unroll
    for (int k = 0; k < BZ; ++k) {
      if (!(c.bits >> k & 1u)) continue;
      const float4 p = E[k * PE];
      const float4 q = make_float4(fmaf(be, p.x, r[k].x), fmaf(be, p.y, r[k].y), fmaf(be, p.z, r[k].z),
                                   fmaf(be, p.w, r[k].w));
      E[k * PE] = q;
      if (c.fl & (kLow | kHi)) c.publish_y(g, q, a.by, par ^ 1, tag + 1, k);
    }
    c.publish_z(g, f, par ^ 1, tag + 1);
  }
#pragma unroll
  for (int k = 0; k < BZ; ++k)
    if (c.bits >> k & 1u)
      st4(a.x, g.row + k * g.P, make_float4(a.inv_sc * x[k].x, a.inv_sc * x[k].y, a.inv_sc * x[k].z, a.inv_sc * x[k].w));
  if (blockIdx.x == 0 && tid == 0) {
    a.result[0] = it;
    a.result[1] = ok;
  }
}

}  // namespace brick

cudaError_t launch_brick_cg(BrickCg a, const BrickPlan& p, unsigned char* halo, uint32_t* tag, int* err,
                            cudaStream_t s) {
  if (!halo || !err || a.max_iter < 1) return cudaErrorInvalidValue;
  const cudaError_t e = brick_tags(tag, (uint32_t)a.max_iter, a.nx, p, halo, s);
  if (e != cudaSuccess) return e;
  a.by = p.by;
  a.bz = p.bz;
  a.py = p.py;
  a.pz = p.pz;
  a.halo = halo;
  a.tag = *tag + 1;   // the caller moves the tag on by the iterations taken
  a.err = err;
  switch (p.bz) {
    case 1: return brick::launch_coop<brick::cg_kernel<1>>(a, p, s);
    case 2: return brick::launch_coop<brick::cg_kernel<2>>(a, p, s);
    case 3: return brick::launch_coop<brick::cg_kernel<3>>(a, p, s);
    case 4: return brick::launch_coop<brick::cg_kernel<4>>(a, p, s);
    case 5: return brick::launch_coop<brick::cg_kernel<5>>(a, p, s);
    case 6: return brick::launch_coop<brick::cg_kernel<6>>(a, p, s);
    case 7: return brick::launch_coop<brick::cg_kernel<7>>(a, p, s);
    case 8: return brick::launch_coop<brick::cg_kernel<8>>(a, p, s);
  }
  return cudaErrorInvalidValue;
}

}  // namespace aew
