// Two time steps in one pass over HBM (temporal blocking).
//
// What bounds it.  A single step reads and writes the whole state: 36 B per node forward, 48
// B adjoint, at 90-96% of the measured copy bandwidth.  Taking two steps while a plane is on
// chip halves that.  A CTA marches through z with a column of whole thread rows: at plane k
// it runs the first step, and behind it at plane k - 1 the second one.  The column's first
// and last thread rows (and, where the grid is wider than 64 float4, a column of float4 on
// each side of the x tile) take part in the first step only; they are recomputed by the
// neighbouring CTA, by the identical expressions, so results are bitwise those of two
// single steps.  z chunks overlap by two planes the same way.
//   256^3, us per step: forward 95 -> 57 (44 for its bytes at the copy rate), forward and
//   adjoint with the whole history 225 -> 144, with the time codec 274 -> 202; 160^3 34 -> 18
//   forward; 512 x 512 x 256 350 -> 276.
//
// Layout.  Thread (j, q) owns four nodes of row j.  The state of the two planes in flight is
// in its registers (the next plane's loads too); y neighbours go through four plane buffers
// in shared memory, x neighbours by shuffle, z neighbours are the thread's own.  Per plane:
//   A  faces of plane k (step 1) and x-, y-faces of plane k - 1 (step 2)
//   B  nodes of plane k (step 1), z-faces and nodes of plane k - 1 (step 2), stores
// with a barrier after each (forward_kernel, forward_pack_kernel and adjoint_kernel: one per
// plane).  The rows beyond the column (one m e row, and one y-face row below) come by cp.async
// into a small ring, so that they cost no registers.
#pragma once

#include "aew_stencil.cuh"
#include "aew_twostep.h"

namespace aew {
namespace two {

using namespace quad;

constexpr int kThreads = 512;
constexpr int kMaxTileQ = 64;   // float4 per x tile
constexpr int kRing = 4;        // extra rows: planes in the cp.async ring
// Planes of the threads' own nodes in the rings of forward_kernel and adjoint_kernel: fields that
// are used in two iterations (m, mu) and the others; two iterations of loads are in flight.
constexpr int kEarly = 4, kLate = 3;
constexpr int kOwnRing = 2 * kEarly + 3 * kLate;   // forward_kernel: m and e, and the faces
constexpr int kPackRing = kEarly + 4 * kLate;      // forward_pack_kernel: m, and e and the faces
constexpr int kExtra = 3;                          // planes of the extra rows there
constexpr int kAdjRing = kEarly + 2 * kLate;   // mu, and lx and ly

using Cut = TwoCut;

__device__ __forceinline__ void cp16(float4* dst, const float* src, bool ok) {
  const uint32_t d = tc::smem_u32(dst);
  const int n = ok ? 16 : 0;   // 0: the 16 bytes are zero-filled and src is not read
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(d), "l"(src), "r"(n) : "memory");
}
__device__ __forceinline__ void cp_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_wait() {
  asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}

// the thread's place
struct Place {
  int j, q, gq, y, i0, kb, ke;
  bool valid, inner, first_x, last_x, p31, p0, edge_y, last_y, top, bot;
  __device__ __forceinline__ Place(const Cut& c, int ny, int nz) {
    const int tid = threadIdx.x, lane = tid & 31;
    j = tid / c.W;
    q = tid - j * c.W;
    const int bx = blockIdx.x % c.ntx, by = blockIdx.x / c.ntx % c.nty, bz = blockIdx.x / c.ntx / c.nty;
    const int hl = bx > 0 ? 1 : 0, cnt = min(c.nqt, c.nq - bx * c.nqt);
    gq = bx * c.nqt + q - hl;
    y = by * (c.rows - 2) + j - 1;
    i0 = 4 * gq;
    kb = bz * c.kc;
    ke = min(kb + c.kc, nz);
    const bool live = j < c.rows && gq >= 0 && gq < c.nq && q <= hl + cnt;
    valid = live && y >= 0 && y < ny;
    inner = valid && j >= 1 && j <= c.rows - 2 && q >= hl && q < hl + cnt;
    first_x = gq <= 0;
    last_x = gq >= c.nq - 1;
    p31 = lane == 31 && q < c.W - 1;
    p0 = lane == 0 && q > 0;
    edge_y = y <= 0 || y >= ny - 1;
    last_y = y >= ny - 1;
    bot = j == 0;                // the row below comes from outside the column
    top = j == c.rows - 1;       // the row above does
  }
};

// four nodes' values with the grid's boundary nodes 0
__device__ __forceinline__ F4 bounded(F4 f, const Place& p, bool zedge) {
  float4 v = v4(f);
  if (p.edge_y || zedge) v = z4();
  if (p.first_x) v.x = 0.f;
  if (p.last_x) v.w = 0.f;
  return f4(v);
}
// a product whose only use is a difference: the paired multiply and subtract can be merged
// into one rounding by the assembler, these scalar ones are not
__device__ __forceinline__ F4 mul_rn(float4 a, float4 b) {
  return f4(make_float4(__fmul_rn(a.x, b.x), __fmul_rn(a.y, b.y), __fmul_rn(a.z, b.z), __fmul_rn(a.w, b.w)));
}
__device__ __forceinline__ float4 ldz(const float* p, bool ok) {
  return ok ? __ldg(reinterpret_cast<const float4*>(p)) : z4();
}
__device__ __forceinline__ float4 ldz16(const uint16_t* p, bool ok) {
  return ok ? bf4(__ldg(reinterpret_cast<const uint2*>(p))) : z4();
}

// Packed strain (time codec): the thread's 8 bytes of its vector's row, and the vectors'
// maxima, collected per pair of planes in a shared table (a column holds parts of a few
// rows of vectors) and folded into the window's with one atomic per vector and pair.
constexpr int kTable = 128;
struct Pack {
  float m;         // max |e| of the thread's nodes in the current pair of planes
  __device__ __forceinline__ void plane(F4 f, unsigned* cell, uint2* at, int k) {
    const float4 v = v4(f);
    *at = make_uint2(pack2bf(v.x, v.y), pack2bf(v.z, v.w));
    m = fmaxf(k & 1 ? m : 0.f, hmax4(v));
    if ((k & 1) && m > 0.f) atomicMax(cell, __float_as_uint(m));
  }
};
// the place of four nodes of plane 0 in the packed window (slot 0); planes 2 apart are
// nx * ny / 64 vectors apart
__device__ __forceinline__ size_t pack_place(int nx, const Place& p) {
  return ((size_t)(p.y >> 3) * (nx >> 3) + (p.i0 >> 3)) * 2048 + (p.y & 7) * 8 + (p.i0 & 7);
}
// after the barrier that ends a pair's last plane: the table of planes k - 1, k into vmax
__device__ __forceinline__ void fold_table(unsigned* table, unsigned* vmax, const Cut& c, int nx, int ny, int k) {
  const int t = threadIdx.x;
  if (t >= kTable) return;
  const unsigned m = table[t];
  if (!m) return;
  table[t] = 0;
  const int vx = c.nqt >> 1, bx = blockIdx.x % c.ntx, by = blockIdx.x / c.ntx % c.nty;
  const size_t yb = (by * (c.rows - 2) >> 3) + t / vx, xb = (size_t)bx * vx + t % vx;
  atomicMax(vmax + ((size_t)(k >> 1) * (ny >> 3) + yb) * (nx >> 3) + xb, m);
}

// Forward steps.  One barrier per plane: a thread computes the faces below and left of its nodes
// itself, from the neighbours' old faces in their ring slots (step 1) or their faces after step 1
// (step 2), by the expressions of the thread that owns them.
//   me: m e of the plane, rows -1 .. R; me1, vy1: after step 1, rows 0 .. R - 1; all in two
//   buffers by the plane's parity.
__global__ void __launch_bounds__(kThreads, 1) forward_kernel(const __grid_constant__ TwoFwd a,
                                                              const __grid_constant__ Cut cut) {
  extern __shared__ __align__(16) unsigned char smem[];
  if (sticky_error(a.err)) return;
  const Place p(cut, a.ny, a.nz);
  const int W = cut.W, R = cut.rows, tid = threadIdx.x, warp = tid >> 5, N = kThreads + 2 * W;
  float4* const ring = reinterpret_cast<float4*>(smem) + tid;   // [kOwnRing][kThreads]
  float4* const me_s = reinterpret_cast<float4*>(smem) + kOwnRing * kThreads + tid;   // [2][N]: row j - 1
  float4* const me1_s = me_s + 2 * N;
  float4* const vy1_s = me1_s + 2 * N;
  float4* const ex = vy1_s - tid + 2 * N;      // [kRing][3][W] e, m, vy of the row below ..
  float4* const eh = ex + kRing * 3 * W;       // [kRing][2][W] e, m of the row above
  float* const sx = reinterpret_cast<float*>(eh + kRing * 2 * W);   // [2][warps]: lane 31's last x-face
  const F4 dth = f4(make_float4(a.dth, a.dth, a.dth, a.dth));
  const size_t P = (size_t)a.nx * a.ny;
  const size_t i0 = p.valid ? (size_t)p.y * a.nx + p.i0 : 0;
  const int nz = a.nz;
  const bool live_q = p.gq >= 0 && p.gq < cut.nq;
  // rare work: the columns meet the source box; the quad has receivers
  const bool src = a.sk >= 0 && p.valid && abs(p.y - a.sj) <= a.sr && p.i0 + 3 >= a.si - a.sr &&
                   p.i0 <= a.si + a.sr;
  const int krec = p.inner && a.krec >= p.kb && a.krec < p.ke && (a.d[0] || a.d[1]) &&
                           has_rec(a.rec_map + i0)
                       ? a.krec
                       : -1;

  auto ok = [&](int k) { return p.valid && k >= 0 && k < nz; };
  auto em_at = [&](int k) { return ring + (size_t)((k & (kEarly - 1)) * 2) * kThreads; };
  auto v_at = [&](int k) { return ring + (size_t)(2 * kEarly + k % kLate * 3) * kThreads; };
  auto issue_em = [&](int k) {
    const bool v = ok(k) && k <= p.ke + 1;
    const size_t i = v ? i0 + (size_t)k * P : 0;
    cp16(em_at(k), a.e + i, v);
    cp16(em_at(k) + kThreads, a.m + i, v);
  };
  auto issue_v = [&](int k) {
    const bool v = ok(k) && k <= p.ke;
    const size_t i = v ? i0 + (size_t)k * P : 0;
    cp16(v_at(k), a.vx + i, v);
    cp16(v_at(k) + kThreads, a.vy + i, v);
    cp16(v_at(k) + 2 * kThreads, a.vz + i, v);
  };
  // the extra rows of plane k into slot k % kRing, and the end of the plane's group
  auto ex_at = [&](int k) { return (p.bot ? ex + k % kRing * 3 * W : eh + k % kRing * 2 * W) + p.q; };
  auto issue_extra = [&](int k) {
    if (p.bot || p.top) {
      const int ye = p.bot ? p.y - 1 : p.y + 1;
      const bool v = k <= p.ke + 1 && live_q && ye >= 0 && ye < a.ny && k < nz;
      const size_t i = v ? (size_t)ye * a.nx + p.i0 + (size_t)k * P : 0;
      cp16(ex_at(k), a.e + i, v);
      cp16(ex_at(k) + W, a.m + i, v);
      if (p.bot) cp16(ex_at(k) + 2 * W, a.vy + i, v);
    }
    cp_commit();
  };
  // m e of the own row and the extra ones into plane k's buffer
  auto put_me = [&](int k, F4 me) {
    float4* const d = me_s + (k & 1) * N;
    if (p.j < R) d[W] = v4(me);
    if (p.bot) d[0] = v4(mul_rn(ex_at(k)[W], ex_at(k)[0]));
    if (p.top) d[2 * W] = v4(mul_rn(ex_at(k)[W], ex_at(k)[0]));
  };

  const int k0 = max(p.kb - 1, 0);
  issue_em(k0);
  issue_em(k0 + 1);
  issue_v(k0);
  issue_extra(k0);
  issue_em(k0 + 2);
  issue_v(k0 + 1);
  issue_extra(k0 + 1);
  F4 vzl1 = f4(z4());   // z-face below plane k0 after step 1
  float4 eb = z4(), mb = z4(), vb = z4();
  if (k0 >= 1) {
    const size_t i = i0 + (size_t)(k0 - 1) * P;
    eb = ldz(a.e + i, p.valid);
    mb = ldz(a.m + i, p.valid);
    vb = ldz(a.vz + i, p.valid);
  }
  cp_wait<1>();
  F4 e_c = lds(em_at(k0)), me_c = mul(lds(em_at(k0) + kThreads), e_c);
  if (k0 >= 1) {
    vzl1 = fma(dth, sub(me_c, mul_rn(mb, eb)), f4(vb));
    if (src && abs(k0 - 1 - a.sk) <= a.sr) {
      float4 v = v4(vzl1);
      add_source(v, k0 - 1, p.y, p.i0, a, a.dts[0]);
      vzl1 = f4(v);
    }
  }
  put_me(k0, me_c);
  __syncthreads();

  F4 vx1p = f4(z4()), vy1p = vx1p, vz1p = vzl1, e1p = vx1p, me1p = vx1p, vz2p = vx1p;
  for (int k = k0; k <= p.ke; ++k) {
    const int cur = (k & 1) * N, old = N - cur;
    // ---- loads of the planes ahead, into the slots of plane k - 1
    issue_em(k + 3);
    issue_v(k + 2);
    issue_extra(k + 2);
    const F4 e_n = lds(em_at(k + 1)), me_n = mul(lds(em_at(k + 1) + kThreads), e_n);
    // ---- step 1 of plane k
    F4 vx1, vy1, vz1, e1, me1;
    {
      const float4* const me = me_s + cur;
      const float4* const v = v_at(k);
      const float4 m = v4(me_c);
      float mx1 = __shfl_down_sync(0xffffffffu, m.x, 1);
      if (p.p31) mx1 = me[W + 1].x;
      float4 x = v4(fma(dth, f4(make_float4(__fsub_rn(m.y, m.x), __fsub_rn(m.z, m.y), __fsub_rn(m.w, m.z),
                                            __fsub_rn(mx1, m.w))),
                        lds(v)));
      if (p.last_x) x.w = 0.f;
      vx1 = f4(x);
      float vxl = __shfl_up_sync(0xffffffffu, x.w, 1);
      if (p.p0) vxl = __fmaf_rn(a.dth, __fsub_rn(m.x, me[W - 1].w), v[-1].w);
      if (p.first_x) vxl = 0.f;
      vy1 = fma(dth, sub(lds(me + 2 * W), me_c), lds(v + kThreads));
      if (p.last_y) vy1 = f4(z4());
      const F4 vyl = fma(dth, sub(me_c, lds(me)), lds(p.bot ? ex_at(k) + 2 * W : v + kThreads - W));
      vz1 = fma(dth, sub(me_n, me_c), lds(v + 2 * kThreads));
      if (k >= nz - 1) vz1 = f4(z4());
      if (src && abs(k - a.sk) <= a.sr) {
        float4 z = v4(vz1);
        add_source(z, k, p.y, p.i0, a, a.dts[0]);
        vz1 = f4(z);
      }
      const F4 dx = f4(make_float4(x.x - vxl, x.y - x.x, x.z - x.y, x.w - x.z));
      const F4 s = add(add(dx, sub(vy1, vyl)), sub(vz1, vz1p));
      e1 = bounded(fma(dth, s, e_c), p, k == 0 || k >= nz - 1);
      me1 = mul(lds(em_at(k) + kThreads), e1);
      if ((tid & 31) == 31) sx[(k & 1) * (kThreads / 32) + warp] = x.w;
    }
    if (p.inner && k >= p.kb && k < p.ke) {
      if (a.e1) st4(a.e1, i0 + (size_t)k * P, v4(e1));
      if (k == krec && a.d[0]) record(a.rec_map + i0, a.d[0], v4(vx1), v4(vy1), v4(vz1));
    }
    // ---- step 2 of plane k - 1
    F4 vz2 = fma(dth, sub(me1, me1p), vz1p);
    if (k - 1 >= nz - 1) vz2 = f4(z4());
    if (src && abs(k - 1 - a.sk) <= a.sr && k > k0) {
      float4 z = v4(vz2);
      add_source(z, k - 1, p.y, p.i0, a, a.dts[1]);
      vz2 = f4(z);
    }
    if (k - 1 >= p.kb && k > k0) {
      const float4* const me = me1_s + old;
      const float4 m = v4(me1p);
      float mx1 = __shfl_down_sync(0xffffffffu, m.x, 1);
      if (p.p31) mx1 = me[W + 1].x;
      float4 x = v4(fma(dth, f4(make_float4(__fsub_rn(m.y, m.x), __fsub_rn(m.z, m.y), __fsub_rn(m.w, m.z),
                                            __fsub_rn(mx1, m.w))),
                        vx1p));
      if (p.last_x) x.w = 0.f;
      float vxl = __shfl_up_sync(0xffffffffu, x.w, 1);
      if (p.p0)
        vxl = __fmaf_rn(a.dth, __fsub_rn(m.x, me[W - 1].w), sx[((k - 1) & 1) * (kThreads / 32) + warp - 1]);
      if (p.first_x) vxl = 0.f;
      F4 vy2 = fma(dth, sub(lds(me + 2 * W), me1p), vy1p);
      if (p.last_y) vy2 = f4(z4());
      const F4 vyl = fma(dth, sub(me1p, lds(me)), lds(vy1_s + old));
      const F4 dx = f4(make_float4(x.x - vxl, x.y - x.x, x.z - x.y, x.w - x.z));
      const F4 s = add(add(dx, sub(vy2, vyl)), sub(vz2, vz2p));
      const F4 e2 = bounded(fma(dth, s, e1p), p, k - 1 == 0 || k - 1 >= nz - 1);
      const size_t i = i0 + (size_t)(k - 1) * P;
      if (p.inner) {
        st4(a.e2, i, v4(e2));
        st4(a.vx2, i, x);
        st4(a.vy2, i, v4(vy2));
        st4(a.vz2, i, v4(vz2));
        if (k - 1 == krec && a.d[1]) record(a.rec_map + i0, a.d[1], x, v4(vy2), v4(vz2));
      }
    }
    // ---- the next plane
    me1_s[cur + W] = v4(me1);
    vy1_s[cur + W] = v4(vy1);
    cp_wait<1>();   // what the last iteration asked for
    put_me(k + 1, me_n);
    vz2p = vz2;
    vx1p = vx1;
    vy1p = vy1;
    vz1p = vz1;
    e1p = e1;
    me1p = me1;
    me_c = me_n;
    e_c = e_n;
    __syncthreads();
  }
}

// The same with window packing (time codec), a kernel of its own: e^{n+1} and e^{n+2} as BF16 go
// through a stage in shared memory, so that the 16-byte rows of a vector leave together (a thread's
// own 8 bytes would touch 16 lines per warp), and their maxima through the tables above.  256^3:
// 147 us a pass with the stores of each thread, 137 now (111 without packing).  Room for the
// stage: e and the extra rows in three planes; with that layout the kernel above is 5% slower.
__global__ void __launch_bounds__(kThreads, 1) forward_pack_kernel(const __grid_constant__ TwoFwd a,
                                                                   const __grid_constant__ Cut cut) {
  extern __shared__ __align__(16) unsigned char smem[];
  if (sticky_error(a.err)) return;
  const Place p(cut, a.ny, a.nz);
  const int W = cut.W, R = cut.rows, tid = threadIdx.x, warp = tid >> 5, N = kThreads + 2 * W;
  float4* const ring = reinterpret_cast<float4*>(smem) + tid;   // [kPackRing][kThreads]
  float4* const me_s = reinterpret_cast<float4*>(smem) + kPackRing * kThreads + tid;   // [2][N]: row j - 1
  float4* const me1_s = me_s + 2 * N;
  float4* const vy1_s = me1_s + 2 * N;
  float4* const ex = vy1_s - tid + 2 * N;      // [kExtra][3][W] e, m, vy of the row below ..
  float4* const eh = ex + kExtra * 3 * W;      // [kExtra][2][W] e, m of the row above
  float* const sx = reinterpret_cast<float*>(eh + kExtra * 2 * W);   // [2][warps]: lane 31's last x-face
  unsigned* const table = reinterpret_cast<unsigned*>(sx + 2 * (kThreads / 32));   // [2][kTable]
  // packed strain on its way out: [2][step][R][pitch] quads of the tile's own columns
  const int pitch = cut.nqt + 2, SB = R * pitch;   // + 16 bytes per row: conflict-free columns
  uint2* const stage = reinterpret_cast<uint2*>(table + 2 * kTable);
  if (tid < 2 * kTable) table[tid] = 0;
  const F4 dth = f4(make_float4(a.dth, a.dth, a.dth, a.dth));
  const size_t P = (size_t)a.nx * a.ny;
  const size_t i0 = p.valid ? (size_t)p.y * a.nx + p.i0 : 0;
  const int nz = a.nz;
  const bool live_q = p.gq >= 0 && p.gq < cut.nq;
  // rare work: the columns meet the source box; the quad has receivers
  const bool src = a.sk >= 0 && p.valid && abs(p.y - a.sj) <= a.sr && p.i0 + 3 >= a.si - a.sr &&
                   p.i0 <= a.si + a.sr;
  const int krec = p.inner && a.krec >= p.kb && a.krec < p.ke && (a.d[0] || a.d[1]) &&
                           has_rec(a.rec_map + i0)
                       ? a.krec
                       : -1;

  auto ok = [&](int k) { return p.valid && k >= 0 && k < nz; };
  // the thread's slots: m; by c, the plane's number modulo 3 counted from k0, e and vx, vy, vz
  auto m_at = [&](int k) { return ring + (k & (kEarly - 1)) * kThreads; };
  auto e_at = [&](int c) { return ring + (kEarly + c) * kThreads; };
  auto v_at = [&](int c) { return ring + (kEarly + (c + 1) * kLate) * kThreads; };
  auto issue_em = [&](int k, int c) {
    const bool v = ok(k) && k <= p.ke + 1;
    const size_t i = v ? i0 + (size_t)k * P : 0;
    cp16(e_at(c), a.e + i, v);
    cp16(m_at(k), a.m + i, v);
  };
  auto issue_v = [&](int k, int c) {
    const bool v = ok(k) && k <= p.ke;
    const size_t i = v ? i0 + (size_t)k * P : 0;
    cp16(v_at(c), a.vx + i, v);
    cp16(v_at(c) + kThreads, a.vy + i, v);
    cp16(v_at(c) + 2 * kThreads, a.vz + i, v);
  };
  // the extra rows of plane k into their slot, and the end of the plane's group
  auto ex_at = [&](int c) { return (p.bot ? ex + c * 3 * W : eh + c * 2 * W) + p.q; };
  auto issue_extra = [&](int k, int c) {
    if (p.bot || p.top) {
      const int ye = p.bot ? p.y - 1 : p.y + 1;
      const bool v = k <= p.ke + 1 && live_q && ye >= 0 && ye < a.ny && k < nz;
      const size_t i = v ? (size_t)ye * a.nx + p.i0 + (size_t)k * P : 0;
      cp16(ex_at(c), a.e + i, v);
      cp16(ex_at(c) + W, a.m + i, v);
      if (p.bot) cp16(ex_at(c) + 2 * W, a.vy + i, v);
    }
    cp_commit();
  };
  // m e of the own row and the extra ones into plane k's buffer
  auto put_me = [&](int k, int c, F4 me) {
    float4* const d = me_s + (k & 1) * N;
    if (p.j < R) d[W] = v4(me);
    if (p.bot) d[0] = v4(mul_rn(ex_at(c)[W], ex_at(c)[0]));
    if (p.top) d[2 * W] = v4(mul_rn(ex_at(c)[W], ex_at(c)[0]));
  };

  const int k0 = max(p.kb - 1, 0);
  int c0 = 0, c1 = 1, c2 = 2;   // slots of planes k, k + 1, k + 2
  issue_em(k0, c0);
  issue_em(k0 + 1, c1);
  issue_v(k0, c0);
  issue_extra(k0, c0);
  issue_em(k0 + 2, c2);
  issue_v(k0 + 1, c1);
  issue_extra(k0 + 1, c1);
  F4 vzl1 = f4(z4());   // z-face below plane k0 after step 1
  float4 eb = z4(), mb = z4(), vb = z4();
  if (k0 >= 1) {
    const size_t i = i0 + (size_t)(k0 - 1) * P;
    eb = ldz(a.e + i, p.valid);
    mb = ldz(a.m + i, p.valid);
    vb = ldz(a.vz + i, p.valid);
  }
  cp_wait<1>();
  F4 e_c = lds(e_at(c0)), me_c = mul(lds(m_at(k0)), e_c);
  if (k0 >= 1) {
    vzl1 = fma(dth, sub(me_c, mul_rn(mb, eb)), f4(vb));
    if (src && abs(k0 - 1 - a.sk) <= a.sr) {
      float4 v = v4(vzl1);
      add_source(v, k0 - 1, p.y, p.i0, a, a.dts[0]);
      vzl1 = f4(v);
    }
  }
  put_me(k0, c0, me_c);
  __syncthreads();

  F4 vx1p = f4(z4()), vy1p = vx1p, vz1p = vzl1, e1p = vx1p, me1p = vx1p, vz2p = vx1p;
  Pack pk1{0.f}, pk2{0.f};
  unsigned* cell = table;
  uint2* put = stage;   // the thread's quad in the stage
  // Write-out: half of the threads take a row of 8 nodes of one vector each for step 1, half for
  // step 2; consecutive lanes take the rows of a vector, whose 16-byte rows are contiguous.
  const int which = tid >> 8;
  const size_t pair = P / 64 * 2048;   // a pair of planes further in the window
  uint16_t* to = nullptr;
  const uint2* from = stage;
  const int bx = blockIdx.x % cut.ntx, by = blockIdx.x / cut.ntx % cut.nty, vx = cut.nqt >> 1;
  const int item = tid & 255, v = item / (R - 2), r = item - v * (R - 2), y = by * (R - 2) + r;
  uint16_t* const window = which ? a.tpack[1] : a.tpack[0];
  if (window && 2 * v < min(cut.nqt, cut.nq - bx * cut.nqt) && y < a.ny)
    to = window + (which ? a.tslot[1] : a.tslot[0]) * 128 +
         ((size_t)(y >> 3) * (a.nx >> 3) + bx * vx + v) * 2048 + (y & 7) * 8;
  from += which * SB + (r + 1) * pitch + 2 * v;
  if (p.inner) {
    cell += ((p.y >> 3) - (by * (R - 2) >> 3)) * vx + (p.gq >> 1) - bx * vx;
    put += p.j * pitch + p.gq - bx * cut.nqt;
  }
  // what iteration k - 1 staged: plane k - 1 after step 1, plane k - 2 after step 2
  auto write_out = [&](int k) {
    const int w = k - 1 - which;
    if (to && w >= p.kb && w < p.ke)
      *reinterpret_cast<uint4*>(to + (w >> 1) * pair + (w & 1) * 64) =
          *reinterpret_cast<const uint4*>(from + (k - 1 & 1) * 2 * SB);
  };

  for (int k = k0; k <= p.ke; ++k) {
    const int cur = (k & 1) * N, old = N - cur;
    // ---- loads of the planes ahead, into the slots of plane k - 1
    issue_em(k + 3, c0);
    issue_v(k + 2, c2);
    issue_extra(k + 2, c2);
    const F4 e_n = lds(e_at(c1)), me_n = mul(lds(m_at(k + 1)), e_n);
    if (k > k0) {   // the pairs of planes that the last iteration ended
      write_out(k);
      if (a.tpack[0] && !(k & 1) && k - 1 >= p.kb) fold_table(table, a.vmax[0], cut, a.nx, a.ny, k - 1);
      if (a.tpack[1] && (k & 1) && k - 2 >= p.kb) fold_table(table + kTable, a.vmax[1], cut, a.nx, a.ny, k - 2);
    }
    // ---- step 1 of plane k
    F4 vx1, vy1, vz1, e1, me1;
    {
      const float4* const me = me_s + cur;
      const float4* const v = v_at(c0);
      const float4 m = v4(me_c);
      float mx1 = __shfl_down_sync(0xffffffffu, m.x, 1);
      if (p.p31) mx1 = me[W + 1].x;
      float4 x = v4(fma(dth, f4(make_float4(__fsub_rn(m.y, m.x), __fsub_rn(m.z, m.y), __fsub_rn(m.w, m.z),
                                            __fsub_rn(mx1, m.w))),
                        lds(v)));
      if (p.last_x) x.w = 0.f;
      vx1 = f4(x);
      float vxl = __shfl_up_sync(0xffffffffu, x.w, 1);
      if (p.p0) vxl = __fmaf_rn(a.dth, __fsub_rn(m.x, me[W - 1].w), v[-1].w);
      if (p.first_x) vxl = 0.f;
      vy1 = fma(dth, sub(lds(me + 2 * W), me_c), lds(v + kThreads));
      if (p.last_y) vy1 = f4(z4());
      const F4 vyl = fma(dth, sub(me_c, lds(me)), lds(p.bot ? ex_at(c0) + 2 * W : v + kThreads - W));
      vz1 = fma(dth, sub(me_n, me_c), lds(v + 2 * kThreads));
      if (k >= nz - 1) vz1 = f4(z4());
      if (src && abs(k - a.sk) <= a.sr) {
        float4 z = v4(vz1);
        add_source(z, k, p.y, p.i0, a, a.dts[0]);
        vz1 = f4(z);
      }
      const F4 dx = f4(make_float4(x.x - vxl, x.y - x.x, x.z - x.y, x.w - x.z));
      const F4 s = add(add(dx, sub(vy1, vyl)), sub(vz1, vz1p));
      e1 = bounded(fma(dth, s, e_c), p, k == 0 || k >= nz - 1);
      me1 = mul(lds(m_at(k)), e1);
      if ((tid & 31) == 31) sx[(k & 1) * (kThreads / 32) + warp] = x.w;
    }
    if (p.inner && k >= p.kb && k < p.ke) {
      if (a.e1) st4(a.e1, i0 + (size_t)k * P, v4(e1));
      if (k == krec && a.d[0]) record(a.rec_map + i0, a.d[0], v4(vx1), v4(vy1), v4(vz1));
    }
    if (a.tpack[0] && p.inner && k >= p.kb && k < p.ke)
      pk1.plane(e1, cell, put + (k & 1) * 2 * SB, k);
    // ---- step 2 of plane k - 1
    F4 vz2 = fma(dth, sub(me1, me1p), vz1p);
    if (k - 1 >= nz - 1) vz2 = f4(z4());
    if (src && abs(k - 1 - a.sk) <= a.sr && k > k0) {
      float4 z = v4(vz2);
      add_source(z, k - 1, p.y, p.i0, a, a.dts[1]);
      vz2 = f4(z);
    }
    if (k - 1 >= p.kb && k > k0) {
      const float4* const me = me1_s + old;
      const float4 m = v4(me1p);
      float mx1 = __shfl_down_sync(0xffffffffu, m.x, 1);
      if (p.p31) mx1 = me[W + 1].x;
      float4 x = v4(fma(dth, f4(make_float4(__fsub_rn(m.y, m.x), __fsub_rn(m.z, m.y), __fsub_rn(m.w, m.z),
                                            __fsub_rn(mx1, m.w))),
                        vx1p));
      if (p.last_x) x.w = 0.f;
      float vxl = __shfl_up_sync(0xffffffffu, x.w, 1);
      if (p.p0)
        vxl = __fmaf_rn(a.dth, __fsub_rn(m.x, me[W - 1].w), sx[((k - 1) & 1) * (kThreads / 32) + warp - 1]);
      if (p.first_x) vxl = 0.f;
      F4 vy2 = fma(dth, sub(lds(me + 2 * W), me1p), vy1p);
      if (p.last_y) vy2 = f4(z4());
      const F4 vyl = fma(dth, sub(me1p, lds(me)), lds(vy1_s + old));
      const F4 dx = f4(make_float4(x.x - vxl, x.y - x.x, x.z - x.y, x.w - x.z));
      const F4 s = add(add(dx, sub(vy2, vyl)), sub(vz2, vz2p));
      const F4 e2 = bounded(fma(dth, s, e1p), p, k - 1 == 0 || k - 1 >= nz - 1);
      const size_t i = i0 + (size_t)(k - 1) * P;
      if (p.inner) {
        st4(a.e2, i, v4(e2));
        st4(a.vx2, i, x);
        st4(a.vy2, i, v4(vy2));
        st4(a.vz2, i, v4(vz2));
        if (k - 1 == krec && a.d[1]) record(a.rec_map + i0, a.d[1], x, v4(vy2), v4(vz2));
      }
      if (a.tpack[1] && p.inner)
        pk2.plane(e2, cell + kTable, put + ((k & 1) * 2 + 1) * SB, k - 1);
    }
    // ---- the next plane
    me1_s[cur + W] = v4(me1);
    vy1_s[cur + W] = v4(vy1);
    cp_wait<1>();   // what the last iteration asked for
    put_me(k + 1, c1, me_n);
    const int c = c0;
    c0 = c1;
    c1 = c2;
    c2 = c;
    vz2p = vz2;
    vx1p = vx1;
    vy1p = vy1;
    vz1p = vz1;
    e1p = e1;
    me1p = me1;
    me_c = me_n;
    e_c = e_n;
    __syncthreads();
  }
  write_out(p.ke + 1);
  // the last pairs: planes ke - 1 of step 1 (ended one iteration ago) and of step 2
  if (a.tpack[0] && p.ke - 1 >= k0 && (p.ke & 1)) fold_table(table, a.vmax[0], cut, a.nx, a.ny, p.ke - 1);
  if (a.tpack[1]) fold_table(table + kTable, a.vmax[1], cut, a.nx, a.ny, p.ke - 1);
}

// Incremental steps: + G(dm e) with FP32 (INCR 1) or BF16 e (2).  TP: window packing.
template <int INCR, bool TP>
__global__ void __launch_bounds__(kThreads, 1) fwd_kernel(const __grid_constant__ TwoFwd a,
                                                          const __grid_constant__ Cut cut) {
  extern __shared__ __align__(16) unsigned char smem[];
  if (sticky_error(a.err)) return;
  const Place p(cut, a.ny, a.nz);
  const int W = cut.W, R = cut.rows, tid = threadIdx.x, warp = tid >> 5;
  static_assert(INCR == 1 || INCR == 2, "");
  constexpr int NE = 4;   // extra fields of the m e row: e, m, dm, e of the step
  // plane buffers, rows W apart: me0 [R + 1], vy1 [1 + R], me1 [R], vy2 [1 + R]; every index is
  // rounded up to whole threads
  float4* const sa = reinterpret_cast<float4*>(smem);
  float4* const sb = sa + kThreads + 2 * W;
  float4* const sc = sb + kThreads + 2 * W;
  float4* const sd = sc + kThreads + 2 * W;
  float4* const ex = sd + kThreads + 2 * W;                      // [kRing][NE + 1][W] rows below ..
  float4* const eh = ex + kRing * (NE + 1) * W;                  // [kRing][NE][W] .. and above
  float* const sx1 = reinterpret_cast<float*>(eh + kRing * NE * W);
  float* const sx2 = sx1 + kThreads / 32;
  unsigned* const table = reinterpret_cast<unsigned*>(sx2 + kThreads / 32);   // [2][kTable]
  if (TP && tid < 2 * kTable) table[tid] = 0;
  const F4 dth = f4(make_float4(a.dth, a.dth, a.dth, a.dth));
  const size_t P = (size_t)a.nx * a.ny;
  const size_t i0 = p.valid ? (size_t)p.y * a.nx + p.i0 : 0;
  const int nz = a.nz;
  const bool live_q = p.gq >= 0 && p.gq < cut.nq;
  const bool has_ef0 = a.ef[0] || a.ef16[0], has_ef1 = a.ef[1] || a.ef16[1];
  // rare work: the columns meet the source box; the quad has receivers
  const bool src = a.sk >= 0 && p.valid && abs(p.y - a.sj) <= a.sr && p.i0 + 3 >= a.si - a.sr &&
                   p.i0 <= a.si + a.sr;
  const int krec = p.inner && a.krec >= p.kb && a.krec < p.ke && (a.d[0] || a.d[1]) &&
                           has_rec(a.rec_map + i0)
                       ? a.krec
                       : -1;

  auto ok = [&](int k) { return p.valid && k >= 0 && k < nz; };
  // m e (+ dm e^n) of the own nodes in plane k
  struct Raw {
    float4 e, m, dm, f32;
    uint2 f16;
  };
  // m, dm and the strain of step s (plane k; m and dm come from L1 the second time)
  auto load_coef = [&](Raw& r, int k, int s) {
    const bool v = ok(k);
    const size_t i = i0 + (size_t)k * P;
    r.m = ldz(a.m + i, v);
    r.dm = ldz(a.dm + i, v);
    if (INCR == 1) r.f32 = ldz(a.ef[s] + i, v && a.ef[s]);
    else r.f16 = v && a.ef16[s] ? __ldg(reinterpret_cast<const uint2*>(a.ef16[s] + i)) : make_uint2(0u, 0u);
  };
  auto load_em = [&](int k) {
    Raw r;
    r.e = ldz(a.e + (i0 + (size_t)k * P), ok(k));
    load_coef(r, k, 0);
    return r;
  };
  auto with_dm = [&](const Raw& r, F4 v, bool has) {
    if (has) v = fma(f4(r.dm), f4(INCR == 2 ? bf4(r.f16) : r.f32), v);
    return v;
  };
  auto me_of = [&](const Raw& r) { return with_dm(r, mul(f4(r.m), f4(r.e)), has_ef0); };
  // the extra rows of plane k into ring slot k % kRing: below row 0 (e, m, .., vy), above the last
  auto issue_extra = [&](int k, bool want) {
    if (p.bot || p.top) {
      const int ye = p.bot ? p.y - 1 : p.y + 1;
      const bool v = want && live_q && p.j < R && ye >= 0 && ye < a.ny && k >= 0 && k < nz;
      const size_t i = v ? (size_t)ye * a.nx + p.i0 + (size_t)k * P : 0;
      const int s = (k + kRing) % kRing;
      float4* d = (p.bot ? ex + s * (NE + 1) * W : eh + s * NE * W) + p.q;
      cp16(d, a.e + i, v);
      cp16(d + W, a.m + i, v);
      cp16(d + 2 * W, a.dm + i, v);
      if (has_ef0 && INCR == 1) cp16(d + 3 * W, a.ef[0] + i, v);
      if (has_ef0 && INCR == 2) {   // BF16: 8 bytes
        const uint32_t dd = tc::smem_u32(d + 3 * W);
        asm volatile("cp.async.ca.shared.global [%0], [%1], 8, %2;" ::"r"(dd), "l"(a.ef16[0] + i),
                     "r"(v ? 8 : 0)
                     : "memory");
      }
      if (p.bot) cp16(d + NE * W, a.vy + i, v);
    }
    cp_commit();
  };
  auto extra_me = [&](int k) {   // m e of the extra row in plane k
    const int s = (k + kRing) % kRing;
    const float4* d = (p.bot ? ex + s * (NE + 1) * W : eh + s * NE * W) + p.q;
    F4 v = mul_rn(d[W], d[0]);
    if (has_ef0)
      v = fma(lds(d + 2 * W), INCR == 2 ? f4(bf4(*reinterpret_cast<const uint2*>(d + 3 * W))) : lds(d + 3 * W), v);
    return v;
  };

  const int k0 = max(p.kb - 1, 0);
  Raw raw = load_em(k0);   // plane k + 1 as it arrives
  F4 me_c = me_of(raw), e_c = f4(raw.e);
  F4 vzl1 = f4(z4());   // z-face below plane k0 after step 1
  if (k0 >= 1) {
    const Raw b = load_em(k0 - 1);
    vzl1 = fma(dth, sub(me_c, with_dm(b, mul_rn(b.m, b.e), has_ef0)),
               f4(ldz(a.vz + i0 + (size_t)(k0 - 1) * P, ok(k0 - 1))));
    if (src && abs(k0 - 1 - a.sk) <= a.sr) {
      float4 v = v4(vzl1);
      add_source(v, k0 - 1, p.y, p.i0, a, a.dts[0]);
      vzl1 = f4(v);
    }
  }
  raw = load_em(k0 + 1);
  float4 vxr = ldz(a.vx + i0 + (size_t)k0 * P, ok(k0)), vyr = ldz(a.vy + i0 + (size_t)k0 * P, ok(k0)),
         vzr = ldz(a.vz + i0 + (size_t)k0 * P, ok(k0));
  issue_extra(k0, true);
  issue_extra(k0 + 1, true);
  cp_wait<1>();   // plane k0's extra rows
  // rows of sa: own at j, the row above the column at R; sb, sd: own at j + 1
  const int at = tid;
  if (p.j < R) sa[at] = v4(me_c);
  if (p.top && p.j < R) sa[R * W + p.q] = v4(extra_me(k0));
  __syncthreads();

  F4 vx1p = f4(z4()), vy1p = vx1p, vz1p = vzl1, e1p = vx1p, me1p = vx1p, vz2p = vx1p;
  Pack pk1{0.f}, pk2{0.f};
  unsigned* cell = table;
  const size_t pk0 = TP && p.inner ? pack_place(a.nx, p) : 0, pair = P / 64 * 2048;
  if (TP && p.inner) {
    const int by = blockIdx.x / cut.ntx % cut.nty, bx = blockIdx.x % cut.ntx, vx = cut.nqt >> 1;
    cell += ((p.y >> 3) - (by * (R - 2) >> 3)) * vx + (p.gq >> 1) - bx * vx;
  }

  for (int k = k0; k <= p.ke; ++k) {
    // ---- loads of the planes ahead
    const F4 me_n = me_of(raw), e_n = f4(raw.e);
    raw = load_em(k + 2 <= p.ke + 1 ? k + 2 : nz);
    Raw coef;
    load_coef(coef, k, 1);
    const bool vv = ok(k + 1) && k + 1 <= p.ke;
    const size_t in = i0 + (size_t)(k + 1) * P;
    const float4 vxn = ldz(a.vx + in, vv), vyn = ldz(a.vy + in, vv), vzn = ldz(a.vz + in, vv);
    issue_extra(k + 2, k + 2 <= p.ke + 1);
    if (TP && k > k0) {   // the pairs of planes that the last iteration ended
      if (a.tpack[0] && !(k & 1) && k - 1 >= p.kb) fold_table(table, a.vmax[0], cut, a.nx, a.ny, k - 1);
      if (a.tpack[1] && (k & 1) && k - 2 >= p.kb) fold_table(table + kTable, a.vmax[1], cut, a.nx, a.ny, k - 2);
    }
    // ---- A: faces of plane k after step 1
    F4 vx1, vy1, vz1;
    {
      const F4 me_yp = lds(sa + at + W);
      const float4 m = v4(me_c);
      float mx1 = __shfl_down_sync(0xffffffffu, m.x, 1);
      if (p.p31) mx1 = sa[at + 1].x;
      float4 x = v4(fma(dth, f4(make_float4(__fsub_rn(m.y, m.x), __fsub_rn(m.z, m.y), __fsub_rn(m.w, m.z),
                                            __fsub_rn(mx1, m.w))),
                        f4(vxr)));
      if (p.last_x) x.w = 0.f;
      vx1 = f4(x);
      if ((tid & 31) == 31) sx1[warp] = x.w;
      vy1 = fma(dth, sub(me_yp, me_c), f4(vyr));
      if (p.last_y) vy1 = f4(z4());
      vz1 = fma(dth, sub(me_n, me_c), f4(vzr));
      if (k >= nz - 1) vz1 = f4(z4());
      if (src && abs(k - a.sk) <= a.sr) {
        float4 v = v4(vz1);
        add_source(v, k, p.y, p.i0, a, a.dts[0]);
        vz1 = f4(v);
      }
      sts(sb + at + W, vy1);
      if (p.bot) {   // the y-face below the column, as its owner computes it
        const float4* d = ex + ((k + kRing) % kRing) * (NE + 1) * W + p.q;
        sts(sb + p.q, fma(dth, sub(me_c, extra_me(k)), lds(d + NE * W)));
      }
    }
    // ---- A: x- and y-faces of plane k - 1 after step 2
    F4 vx2, vy2;
    {
      const F4 me_yp = lds(sc + at + W);
      const float4 m = v4(me1p);
      float mx1 = __shfl_down_sync(0xffffffffu, m.x, 1);
      if (p.p31) mx1 = sc[at + 1].x;
      float4 x = v4(fma(dth, f4(make_float4(__fsub_rn(m.y, m.x), __fsub_rn(m.z, m.y), __fsub_rn(m.w, m.z),
                                            __fsub_rn(mx1, m.w))),
                        vx1p));
      if (p.last_x) x.w = 0.f;
      vx2 = f4(x);
      if ((tid & 31) == 31) sx2[warp] = x.w;
      vy2 = fma(dth, sub(me_yp, me1p), vy1p);
      if (p.last_y) vy2 = f4(z4());
      sts(sd + at + W, vy2);
    }
    cp_wait<1>();   // the extra rows of plane k + 1
    __syncthreads();
    // ---- B: nodes of plane k after step 1
    F4 e1, me1;
    {
      const float4 x = v4(vx1);
      float vxl = __shfl_up_sync(0xffffffffu, x.w, 1);
      if (p.p0) vxl = sx1[warp - 1];
      if (p.first_x) vxl = 0.f;
      const F4 dx = f4(make_float4(x.x - vxl, x.y - x.x, x.z - x.y, x.w - x.z));
      const F4 s = add(add(dx, sub(vy1, lds(sb + at))), sub(vz1, vz1p));
      e1 = bounded(fma(dth, s, e_c), p, k == 0 || k >= nz - 1);
      me1 = with_dm(coef, mul(f4(coef.m), e1), has_ef1);
    }
    sts(sc + at, me1);
    const bool mine = p.inner && k >= p.kb && k < p.ke;
    if (mine) {
      if (a.e1) st4(a.e1, i0 + (size_t)k * P, v4(e1));
      if (k == krec && a.d[0]) record(a.rec_map + i0, a.d[0], v4(vx1), v4(vy1), v4(vz1));
    }
    if (TP && a.tpack[0] && p.inner && k >= p.kb && k < p.ke)
      pk1.plane(e1, cell,
                reinterpret_cast<uint2*>(a.tpack[0] + (k >> 1) * pair + a.tslot[0] * 128 + (k & 1) * 64 + pk0), k);
    // ---- B: z-faces and nodes of plane k - 1 after step 2
    F4 vz2 = fma(dth, sub(me1, me1p), vz1p);
    if (k - 1 >= nz - 1) vz2 = f4(z4());
    if (src && abs(k - 1 - a.sk) <= a.sr && k > k0) {
      float4 v = v4(vz2);
      add_source(v, k - 1, p.y, p.i0, a, a.dts[1]);
      vz2 = f4(v);
    }
    {
      const float4 x = v4(vx2);
      float vxl = __shfl_up_sync(0xffffffffu, x.w, 1);
      if (p.p0) vxl = sx2[warp - 1];
      if (p.first_x) vxl = 0.f;
      const F4 dx = f4(make_float4(x.x - vxl, x.y - x.x, x.z - x.y, x.w - x.z));
      const F4 s = add(add(dx, sub(vy2, lds(sd + at))), sub(vz2, vz2p));
      const F4 e2 = bounded(fma(dth, s, e1p), p, k - 1 == 0 || k - 1 >= nz - 1);
      if (k - 1 >= p.kb && k > k0) {
        const size_t i = i0 + (size_t)(k - 1) * P;
        if (p.inner) {
          st4(a.e2, i, v4(e2));
          st4(a.vx2, i, v4(vx2));
          st4(a.vy2, i, v4(vy2));
          st4(a.vz2, i, v4(vz2));
          if (k - 1 == krec && a.d[1]) record(a.rec_map + i0, a.d[1], v4(vx2), v4(vy2), v4(vz2));
        }
        if (TP && a.tpack[1] && p.inner)
          pk2.plane(e2, cell + kTable,
                    reinterpret_cast<uint2*>(a.tpack[1] + (k - 1 >> 1) * pair + a.tslot[1] * 128 +
                                             (k - 1 & 1) * 64 + pk0),
                    k - 1);
      }
    }
    // ---- the next plane
    if (p.j < R) sa[at] = v4(me_n);
    if (p.top && p.j < R) sa[R * W + p.q] = v4(extra_me(k + 1));
    vz2p = vz2;
    vx1p = vx1;
    vy1p = vy1;
    vz1p = vz1;
    e1p = e1;
    me1p = me1;
    me_c = me_n;
    e_c = e_n;
    vxr = vxn;
    vyr = vyn;
    vzr = vzn;
    __syncthreads();
  }
  if (TP) {   // the last pairs: planes ke - 1 of step 1 (ended one iteration ago) and of step 2
    if (a.tpack[0] && p.ke - 1 >= k0 && (p.ke & 1)) fold_table(table, a.vmax[0], cut, a.nx, a.ny, p.ke - 1);
    if (a.tpack[1]) fold_table(table + kTable, a.vmax[1], cut, a.nx, a.ny, p.ke - 1);
  }
}

// Two adjoint steps with gradient accumulation, one barrier per plane as in forward_kernel.
// B16: the strain is BF16.  CLOSE: a window ends with one of the steps (FP64 instructions slow
// the loop even where they are skipped: 238 us instead of 140 at 256^3, so the other launches
// are built without them).  mu, lx and ly, which neighbours read, come through the ring; the
// fields that only their own thread uses stay in registers, one plane ahead (through the ring
// too the pass was 15% slower).  Full gradient at 256^3: 153 us per step with two barriers, 148
// with one; 52 B per node and pass bound it from 128 us a pass, issue slots at about 175.
template <bool B16, bool CLOSE>
__global__ void __launch_bounds__(kThreads, 1) adjoint_kernel(const __grid_constant__ TwoAdj a,
                                                              const __grid_constant__ Cut cut) {
  extern __shared__ __align__(16) unsigned char smem[];
  if (sticky_error(a.err)) return;
  const Place p(cut, a.ny, a.nz);
  const int W = cut.W, R = cut.rows, tid = threadIdx.x, warp = tid >> 5, N = kThreads + 2 * W;
  float4* const ring = reinterpret_cast<float4*>(smem) + tid;   // [kAdjRing][kThreads]
  float4* const mu_s = reinterpret_cast<float4*>(smem) + kAdjRing * kThreads + tid;   // [2][N]: row j - 1
  float4* const mu1_s = mu_s + 2 * N;
  float4* const ly1_s = mu1_s + 2 * N;
  float4* const ex = ly1_s - tid + 2 * N;      // [kRing][2][W] mu, ly of the row below ..
  float4* const eh = ex + kRing * 2 * W;       // [kRing][W] mu of the row above
  float* const sx = reinterpret_cast<float*>(eh + kRing * W);   // [2][warps]: lane 31's last x-face
  const F4 dth = f4(make_float4(a.dth, a.dth, a.dth, a.dth));
  const F4 ndth = f4(make_float4(-a.dth, -a.dth, -a.dth, -a.dth));
  const size_t P = (size_t)a.nx * a.ny;
  const size_t i0 = p.valid ? (size_t)p.y * a.nx + p.i0 : 0;
  const int nz = a.nz;
  const bool live_q = p.gq >= 0 && p.gq < cut.nq;
  // receivers on the own nodes, on those of the row below, on the node left of them
  const int* const map = a.rec_map + i0;
  const bool rz = p.valid && a.krec >= 0 && (a.resid[0] || a.resid[1]) && a.krec >= p.kb - 2 && a.krec <= p.ke;
  const bool rec = rz && has_rec(map), rec_y = rz && p.y > 0 && has_rec(map - a.nx);
  const int rec_x = rz && p.p0 && p.gq > 0 ? __ldg(map - 1) : -1;
  const bool open = a.open, close1 = CLOSE && a.close[0], close2 = CLOSE && a.close[1];

  auto ok = [&](int k) { return p.valid && k >= 0 && k < nz; };
  auto mu_at = [&](int k) { return ring + (size_t)(k & (kEarly - 1)) * kThreads; };
  auto l_at = [&](int c) { return ring + (kEarly + c * 2) * kThreads; };   // by slot
  auto issue_mu = [&](int k) {
    const bool v = ok(k) && k <= p.ke + 1;
    cp16(mu_at(k), a.mu + (v ? i0 + (size_t)k * P : 0), v);
  };
  auto issue_l = [&](int k, int c) {
    const bool v = ok(k) && k <= p.ke;
    const size_t i = v ? i0 + (size_t)k * P : 0;
    cp16(l_at(c), a.lx + i, v);
    cp16(l_at(c) + kThreads, a.ly + i, v);
  };
  // the extra rows of plane k into slot k % kRing, and the end of the plane's group
  auto ex_at = [&](int k) { return (p.bot ? ex + k % kRing * 2 * W : eh + k % kRing * W) + p.q; };
  auto issue_extra = [&](int k) {
    if (p.bot || p.top) {
      const int ye = p.bot ? p.y - 1 : p.y + 1;
      const bool v = k <= p.ke + 1 && live_q && ye >= 0 && ye < a.ny && k < nz;
      const size_t i = v ? (size_t)ye * a.nx + p.i0 + (size_t)k * P : 0;
      cp16(ex_at(k), a.mu + i, v);
      if (p.bot) cp16(ex_at(k) + W, a.ly + i, v);
    }
    cp_commit();
  };
  auto put_mu = [&](int k, F4 mu) {
    float4* const d = mu_s + (k & 1) * N;
    if (p.j < R) d[W] = v4(mu);
    if (p.bot) d[0] = ex_at(k)[0];
    if (p.top) d[2 * W] = ex_at(k)[0];
  };
  // strain of step s in plane k (own nodes)
  struct Strain {
    float4 f32;
    uint2 f16;
  };
  auto load_en = [&](int s, int k) {
    Strain e{z4(), make_uint2(0u, 0u)};
    if (p.inner && k >= p.kb && k < p.ke) {
      const size_t i = i0 + (size_t)k * P;
      if (B16) {
        if (a.en16[s]) e.f16 = __ldg(reinterpret_cast<const uint2*>(a.en16[s] + i));
      } else if (a.en[s]) {
        e.f32 = ldg4(a.en[s] + i);
      }
    }
    return e;
  };
  auto load_w = [&](int k) {
    return !open && p.inner && k >= p.kb && k < p.ke
               ? *reinterpret_cast<const float4*>(a.acc32 + (i0 + (size_t)k * P))
               : z4();
  };
  auto flush = [&](size_t i, F4 f) { add_wide(a.acc64 + i, v4(f)); };
  auto val = [&](const Strain& e) { return f4(B16 ? bf4(e.f16) : e.f32); };

  const int k0 = max(p.kb - 1, 0);
  issue_mu(k0);
  issue_mu(k0 + 1);
  int c0 = 0, c1 = 1, c2 = 2;   // slots of planes k, k + 1, k + 2 (modulo 3)
  issue_l(k0, c0);
  issue_extra(k0);
  issue_mu(k0 + 2);
  issue_l(k0 + 1, c1);
  issue_extra(k0 + 1);
  float4 mub = z4(), lzb = z4();
  if (k0 >= 1) {
    const size_t i = i0 + (size_t)(k0 - 1) * P;
    mub = ldz(a.mu + i, p.valid);
    lzb = ldz(a.lz + i, p.valid);
  }
  const size_t ik = i0 + (size_t)k0 * P;
  float4 lzr = ldz(a.lz + ik, ok(k0)), mr = ldz(a.m + ik, ok(k0));
  Strain e1r = load_en(0, k0), e2r = load_en(1, k0);
  float4 wr = load_w(k0);
  cp_wait<1>();
  F4 mu_c = lds(mu_at(k0));
  F4 lzl1 = f4(z4());   // z-face below plane k0 after the first step
  if (k0 >= 1) {
    F4 l = f4(lzb);
    if (rec && a.krec == k0 - 1 && a.resid[0]) l = injected(l, map, a.resid[0] + 2);
    lzl1 = fma(dth, sub(f4(mub), mu_c), l);
  }
  put_mu(k0, mu_c);
  __syncthreads();

  F4 lx1p = f4(z4()), ly1p = lx1p, lz1p = lzl1, mu1p = lx1p, lz2p = lx1p, mp = lx1p, gp = lx1p;
  Strain e2p{z4(), make_uint2(0u, 0u)};

  for (int k = k0; k <= p.ke; ++k) {
    const int cur = (k & 1) * N, old = N - cur;
    // ---- loads of the planes ahead, into the slots of plane k - 1
    issue_mu(k + 3);
    issue_l(k + 2, c2);
    issue_extra(k + 2);
    const F4 mu_n = lds(mu_at(k + 1));
    const F4 m_c = f4(mr), w_c = f4(wr);
    const Strain e1c = e1r, e2c = e2r;
    F4 lz1 = f4(lzr);
    {
      const bool vv = ok(k + 1) && k + 1 <= p.ke;
      const size_t in = i0 + (size_t)(k + 1) * P;
      lzr = ldz(a.lz + in, vv);
      mr = ldz(a.m + in, vv);
      e1r = load_en(0, k + 1);
      e2r = load_en(1, k + 1);
      wr = load_w(k + 1);
    }
    // ---- the first step of plane k
    F4 lx1, ly1, mu1, g;
    {
      const float4* const me = mu_s + cur;
      const float4* const l = l_at(c0);
      lx1 = lds(l);
      ly1 = lds(l + kThreads);
      F4 lyl = lds(p.bot ? ex_at(k) + W : l + kThreads - W);
      float lxl_old = p.p0 ? l[-1].w : 0.f;
      if (k == a.krec && a.resid[0]) {
        if (rec) {
          lx1 = injected(lx1, map, a.resid[0]);
          ly1 = injected(ly1, map, a.resid[0] + 1);
          lz1 = injected(lz1, map, a.resid[0] + 2);
        }
        if (rec_y) lyl = injected(lyl, map - a.nx, a.resid[0] + 1);
        if (rec_x >= 0) lxl_old += __ldg(a.resid[0] + 3 * rec_x);
      }
      const float4 m = v4(mu_c);
      float mx1 = __shfl_down_sync(0xffffffffu, m.x, 1);
      if (p.p31) mx1 = me[W + 1].x;
      float4 x = v4(fma(dth, f4(make_float4(m.x - m.y, m.y - m.z, m.z - m.w, m.w - mx1)), lx1));
      if (p.last_x) x.w = 0.f;
      lx1 = f4(x);
      float lxl = __shfl_up_sync(0xffffffffu, x.w, 1);
      if (p.p0) lxl = __fmaf_rn(a.dth, __fsub_rn(me[W - 1].w, m.x), lxl_old);
      if (p.first_x) lxl = 0.f;
      ly1 = fma(dth, sub(mu_c, lds(me + 2 * W)), ly1);
      if (p.last_y) ly1 = f4(z4());
      lyl = fma(dth, sub(lds(me), mu_c), lyl);
      lz1 = fma(dth, sub(mu_c, mu_n), lz1);
      if (k >= nz - 1) lz1 = f4(z4());
      const F4 dx = f4(make_float4(x.x - lxl, x.y - x.x, x.z - x.y, x.w - x.z));
      const F4 s = add(add(dx, sub(ly1, lyl)), sub(lz1, lz1p));
      const F4 dq = bounded(mul(ndth, s), p, k == 0 || k >= nz - 1);
      mu1 = fma(m_c, dq, mu_c);
      g = fma(val(e1c), dq, w_c);
      if ((tid & 31) == 31) sx[(k & 1) * (kThreads / 32) + warp] = x.w;
    }
    // ---- the second step of plane k - 1
    F4 lz2 = lz1p;
    const bool rec2 = k - 1 == a.krec && k > k0 && a.resid[1];
    if (rec2 && rec) lz2 = injected(lz2, map, a.resid[1] + 2);
    lz2 = fma(dth, sub(mu1p, mu1), lz2);
    if (k - 1 >= nz - 1) lz2 = f4(z4());
    if (k - 1 >= p.kb && k > k0) {
      const float4* const me = mu1_s + old;
      F4 lx2 = lx1p, ly2 = ly1p, lyl = lds(ly1_s + old);
      float lxl_old = p.p0 ? sx[((k - 1) & 1) * (kThreads / 32) + warp - 1] : 0.f;
      if (rec2) {
        if (rec) {
          lx2 = injected(lx2, map, a.resid[1]);
          ly2 = injected(ly2, map, a.resid[1] + 1);
        }
        if (rec_y) lyl = injected(lyl, map - a.nx, a.resid[1] + 1);
        if (rec_x >= 0) lxl_old += __ldg(a.resid[1] + 3 * rec_x);
      }
      const float4 m = v4(mu1p);
      float mx1 = __shfl_down_sync(0xffffffffu, m.x, 1);
      if (p.p31) mx1 = me[W + 1].x;
      float4 x = v4(fma(dth, f4(make_float4(m.x - m.y, m.y - m.z, m.z - m.w, m.w - mx1)), lx2));
      if (p.last_x) x.w = 0.f;
      float lxl = __shfl_up_sync(0xffffffffu, x.w, 1);
      if (p.p0) lxl = __fmaf_rn(a.dth, __fsub_rn(me[W - 1].w, m.x), lxl_old);
      if (p.first_x) lxl = 0.f;
      ly2 = fma(dth, sub(mu1p, lds(me + 2 * W)), ly2);
      if (p.last_y) ly2 = f4(z4());
      lyl = fma(dth, sub(lds(me), mu1p), lyl);
      const F4 dx = f4(make_float4(x.x - lxl, x.y - x.x, x.z - x.y, x.w - x.z));
      const F4 s = add(add(dx, sub(ly2, lyl)), sub(lz2, lz2p));
      const F4 dq = bounded(mul(ndth, s), p, k - 1 == 0 || k - 1 >= nz - 1);
      if (p.inner) {
        const size_t i = i0 + (size_t)(k - 1) * P;
        st4(a.mu2, i, v4(fma(mp, dq, mu1p)));
        st4(a.lx2, i, x);
        st4(a.ly2, i, v4(ly2));
        st4(a.lz2, i, v4(lz2));
        // dJ/dm += dt e q of both steps; a window that ends is flushed
        if (close1) flush(i, gp);
        const F4 sum = fma(val(e2p), dq, close1 ? f4(z4()) : gp);
        if (close2) flush(i, sum);
        else st4(a.acc32, i, v4(sum));
      }
    }
    // ---- the next plane
    mu1_s[cur + W] = v4(mu1);
    ly1_s[cur + W] = v4(ly1);
    cp_wait<1>();   // what the last iteration asked for
    put_mu(k + 1, mu_n);
    const int c = c0;
    c0 = c1;
    c1 = c2;
    c2 = c;
    lz2p = lz2;
    lx1p = lx1;
    ly1p = ly1;
    lz1p = lz1;
    mu1p = mu1;
    mp = m_c;
    gp = g;
    e2p = e2c;
    mu_c = mu_n;
    __syncthreads();
  }
}

}  // namespace two
}  // namespace aew
