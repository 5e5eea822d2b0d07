// The prior solve of grids that fit the SMs: up to 1024 CG iterations per launch.
//
// A launch per pass took 15 us and more however small the grid.  Here x, r and A p stay in
// registers and p in shared memory, with its halos exchanged as in the time loops
// (aew_brick.cuh), and both inner products of an iteration are all-reduced through one
// tagged word pair per CTA: three L2 round trips per iteration bound it, with the reductions'
// dependent adds.  us per iteration, launch per pass -> now: 32^3 21 -> 7, 64^3 37 -> 9, 128^3
// 45 -> 16.
//
// The inner products: four products are summed by FP32 FMAs, as in the streaming passes; from
// there a thread's and a warp's sums keep their rounding errors in two more floats (72 bits
// against FP64's 53, and FP64 instructions in every warp would be the longest part of an
// iteration), and one warp per CTA adds the warps' and the CTAs' parts in as many bits or in FP64.
// Every CTA adds the same parts in the same order, so all take the same steps and stop together.
#include "aew_brick.cuh"

namespace aew {
namespace brick {

// a sum in three floats: value, accumulated rounding errors, and theirs
struct Sum3 {
  float s, c, d;
  __device__ __forceinline__ void add(float x) {
    float e, f;
    s = two_sum(s, x, e);
    c = two_sum(c, e, f);
    d = __fadd_rn(d, f);
  }
  __device__ __forceinline__ void add(float x, float y, float z) {   // the same in either order
    float e, f, g;
    s = two_sum(s, x, e);
    c = two_sum(c, y, f);
    c = two_sum(c, e, g);
    d = __fadd_rn(__fadd_rn(d, z), __fadd_rn(f, g));
  }
  __device__ __forceinline__ double value() const { return (double)s + ((double)c + (double)d); }
};
__device__ __forceinline__ Sum3 warp_sum(Sum3 p) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1)
    p.add(__shfl_xor_sync(0xffffffffu, p.s, o), __shfl_xor_sync(0xffffffffu, p.c, o),
          __shfl_xor_sync(0xffffffffu, p.d, o));
  return p;
}
__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}
constexpr int kParts = 5;   // CTAs per lane and round: one round on 152 SMs
struct Shared {
  Sum3 warp[32], total;
  int pass, dead;
};
// The sum over all CTAs of the threads' sums (words: two per CTA of this reduction); one warp per CTA
// fetches the CTAs' sums, all missing ones in flight at once.  They travel and are added as FP64
// numbers, or on one-plane bricks (THREE) as the three floats, which saves the small grids the FP64
// adds' latency and costs the large ones a second word per CTA.  us per iteration with every thread
// polling a word of FP32 pairs / so: 16^3 7.8 / 8.0, 32^3 8.0 / 7.3, 64^3 12.3 / 8.6, 96^3 13.5 / 10.3,
// 128^3 17.1 / 15.6; the other way round 32^3 9.3, 64^3 10.7, 128^3 18.6.
// test: sh.pass tells whether the total is at most tol2 (in FP64).
// (*stop: a wait gave up, the same for all threads)
template <bool THREE>
__device__ __forceinline__ Sum3 all_sum(Sum3 p, ulonglong2* words, int ctas, uint32_t tag, bool test, double tol2,
                                        Shared& sh, int* err, int* stop) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
  volatile int* const dead = &sh.dead;
  p = warp_sum(p);
  if (lane == 0) sh.warp[warp] = p;
  __syncthreads();
  if (warp == 0) {
    const Sum3 q = warp_sum(lane < nw ? sh.warp[lane] : Sum3{0.f, 0.f, 0.f});
    if (lane == 0) {
      const unsigned long long t = (unsigned long long)tag << 32, b = __double_as_longlong(q.value());
      const unsigned long long x = THREE ? __float_as_uint(q.s) : b >> 32,
                               y = THREE ? __float_as_uint(q.c) : b & 0xffffffffull;
      asm volatile("st.relaxed.gpu.global.v2.b64 [%0], {%1, %2};" ::"l"(words + blockIdx.x), "l"(t | x), "l"(t | y)
                   : "memory");
      if (THREE)
        asm volatile("st.relaxed.gpu.global.v2.b64 [%0], {%1, %2};" ::"l"(words + ctas + blockIdx.x),
                     "l"(t | __float_as_uint(q.d)), "l"(t)
                     : "memory");
    }
    double v = 0.0;
    Sum3 v3{0.f, 0.f, 0.f};
    for (int i0 = lane; i0 < ctas; i0 += 32 * kParts) {
      ulonglong2 w[kParts], u[THREE ? kParts : 1];
      uint32_t need = 0, t0 = 0;
#pragma unroll
      for (int k = 0; k < kParts; ++k) {
        w[k] = make_ulonglong2(0, 0);
        if (THREE) u[THREE ? k : 0] = w[k];
        if (i0 + 32 * k < ctas) need |= 1u << k;
      }
      for (uint32_t it = 1; need && !*dead; ++it) {
#pragma unroll
        for (int k = 0; k < kParts; ++k)
          if (need >> k & 1u) {
            w[k] = ld_words(words + i0 + 32 * k);
            if (THREE) u[THREE ? k : 0] = ld_words(words + ctas + i0 + 32 * k);
          }
#pragma unroll
        for (int k = 0; k < kParts; ++k)
          if (fresh(w[k], THREE ? u[THREE ? k : 0] : w[k], tag)) need &= ~(1u << k);
        if (need && (it & 63u) == 0 && !keep_waiting(t0, dead, err)) break;
      }
#pragma unroll
      for (int k = 0; k < kParts; ++k) {
        if (THREE)
          v3.add(__uint_as_float((uint32_t)w[k].x), __uint_as_float((uint32_t)w[k].y),
                 __uint_as_float((uint32_t)u[THREE ? k : 0].x));
        else
          v += __longlong_as_double((long long)(w[k].x << 32 | (w[k].y & 0xffffffffull)));
      }
    }
    if (THREE) v3 = warp_sum(v3);
    else v = warp_sum(v);
    if (lane == 0) {
      if (!THREE) {
        v3.s = (float)v;
        v3.c = (float)(v - (double)v3.s);
      }
      sh.total = v3;
      if (test) sh.pass = (THREE ? v3.value() : v) <= tol2;
    }
  }
  *stop = __syncthreads_or(*dead);
  return sh.total;
}
// a / b in one rounding or so
__device__ __forceinline__ float ratio(const Sum3& a, const Sum3& b) {
  const float q = __fdiv_rn(a.s, b.s);
  return q + __fdiv_rn(fmaf(-q, b.s, a.s) + fmaf(-q, b.c, a.c), b.s);
}

template <int BZ>
__global__ void __launch_bounds__(tmax(BZ), 1) cg_kernel(const __grid_constant__ BrickCg a) {
  using X = Ctx<BZ>;
  constexpr int PE = X::PE;
  extern __shared__ __align__(16) unsigned char smem[];
  __shared__ Shared sh;
  if (sticky_error(a.err)) return;
  float4* const f = reinterpret_cast<float4*>(smem);
  volatile int* dead = &sh.dead;
  const Geo g(a);
  const X c(g, a.halo, a.by, a.py, a.pz, a.ny, a.nz);
  const int tid = g.tid, nq = g.nq, ctas = a.py * a.pz;
  if (tid == 0) sh.dead = 0;
  c.clear(f);
  ulonglong2* const red = c.wd.base + (2 * (size_t)ctas * (4 * X::TP) + 2 * (size_t)ctas * 4 * BZ * nq);
  const bool y0 = g.y > 0, y1 = g.y + 1 < a.ny, x0 = g.q > 0, x1 = g.q < nq - 1;
  float4* const E = f + X::oE + tid;

  float4 x[BZ], r[BZ], v[BZ];
#pragma unroll
  for (int k = 0; k < BZ; ++k) {
    x[k] = r[k] = z4();
    if (c.bits >> k & 1u) {
      const uint32_t i = g.row + k * g.P;
      float4 p;
      if (a.resume) {
        x[k] = *reinterpret_cast<const float4*>(a.x + i);
        r[k] = *reinterpret_cast<const float4*>(a.r + i);
        p = *reinterpret_cast<const float4*>(a.p + i);
      } else {
        const float4 w = ldg4(a.w + i);
        p = r[k] = make_float4(a.sc * w.x, a.sc * w.y, a.sc * w.z, a.sc * w.w);
      }
      E[k * PE] = p;
      if (c.fl & (kLow | kHi)) c.publish_y(g, p, a.by, 0, a.tag, k);
    }
  }
  c.publish_z(g, f, 0, a.tag);
  Sum3 rr{a.rr_hi, a.rr_lo, 0.f};
  if (a.resume) {
    rr.s = __ldg(a.rr_in);
    rr.c = __ldg(a.rr_in + 1);
  }
  int it = 0, ok = 0, stop = 0;
#pragma unroll 1
  while (it < a.max_iter) {
    const int par = it & 1;
    const uint32_t tag = a.tag + it;
    const float4 below = v4(c.template receive_halos<true>(g, f, a.by, a.py, par, tag, dead, a.err));
    // ---- v = A p and p.v
    Sum3 acc{0.f, 0.f, 0.f};
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
    const Sum3 pap = all_sum<BZ == 1>(acc, red + (size_t)par * 2 * ctas, ctas, tag, false, a.tol2, sh, a.err, &stop);
    const float al = pap.s > 0.f ? ratio(rr, pap) : 0.f;
    // ---- x += a p, r -= a A p and r.r
    acc = Sum3{0.f, 0.f, 0.f};
#pragma unroll
    for (int k = 0; k < BZ; ++k) {
      if (!(c.bits >> k & 1u)) continue;
      const float4 p = E[k * PE];
      x[k].x += al * p.x; x[k].y += al * p.y; x[k].z += al * p.z; x[k].w += al * p.w;
      r[k].x -= al * v[k].x; r[k].y -= al * v[k].y; r[k].z -= al * v[k].z; r[k].w -= al * v[k].w;
      acc.add(fmaf(r[k].x, r[k].x, fmaf(r[k].y, r[k].y, fmaf(r[k].z, r[k].z, r[k].w * r[k].w))));
    }
    const bool last = it + 1 == a.max_iter, test = (it & 7) == 7 || last;
    const Sum3 rn = all_sum<BZ == 1>(acc, red + (size_t)(2 + par) * 2 * ctas, ctas, tag, test, a.tol2, sh, a.err, &stop);
    if (test && sh.pass) ok = 1;
    const float be = rr.s > 0.f ? ratio(rn, rr) : 0.f;
    rr = rn;
    ++it;
    if (ok || (last && !a.more) || stop) break;   // stop: the values are void, and the error flag is set
    // ---- p = r + b p
#pragma unroll
    for (int k = 0; k < BZ; ++k) {
      if (!(c.bits >> k & 1u)) continue;
      const float4 p = E[k * PE];
      const float4 q = make_float4(fmaf(be, p.x, r[k].x), fmaf(be, p.y, r[k].y), fmaf(be, p.z, r[k].z),
                                   fmaf(be, p.w, r[k].w));
      E[k * PE] = q;
      if (!last && (c.fl & (kLow | kHi))) c.publish_y(g, q, a.by, par ^ 1, tag + 1, k);
    }
    if (!last) c.publish_z(g, f, par ^ 1, tag + 1);
  }
  if (a.more && !ok) {   // to go on with
#pragma unroll
    for (int k = 0; k < BZ; ++k)
      if (c.bits >> k & 1u) {
        const uint32_t i = g.row + k * g.P;
        st4(a.x, i, x[k]);
        st4(a.r, i, r[k]);
        st4(a.p, i, E[k * PE]);
      }
    if (blockIdx.x == 0 && tid == 0) {
      a.result[0] = it;
      a.result[1] = 0;
      a.rr_out[0] = rr.s;
      a.rr_out[1] = rr.c;
    }
    return;
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
  if (!halo || !err || a.max_iter < 1 || (a.more && a.max_iter % 8) || ((a.more || a.resume) && (!a.r || !a.p || !a.rr_in || !a.rr_out || a.rr_in == a.rr_out)))
    return cudaErrorInvalidValue;
  const cudaError_t e = brick_tags(tag, (uint32_t)a.max_iter, a.nx, p, halo, s);
  if (e != cudaSuccess) return e;
  a.by = p.by;
  a.bz = p.bz;
  a.py = p.py;
  a.pz = p.pz;
  a.halo = halo;
  a.tag = *tag + 1;
  *tag += (uint32_t)a.max_iter + 1;
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
