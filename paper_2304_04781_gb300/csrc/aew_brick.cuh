// On-chip time loops.  A grid of up to about 14,300 nodes per SM (128^3) keeps its state in
// registers and shared memory for many steps: one cooperative launch, one CTA (brick) per
// SM, and per step only the bricks' face values go through L2.
//
// What bounds it.  A step launched by itself takes 8 us on a 32^3 grid and 14 us (36 B per
// node through L2) at 128^3 whatever the arithmetic costs.  Here a step is bounded by
// the shared-memory traffic of the y-neighbour exchange (7 accesses of 16 B per four
// nodes) on large bricks and by one L2 store-to-load round trip on small ones.
//
// Layout.  A brick is `by` rows (y) x up to BZ planes (z) of whole x rows.  Thread
// (j, q) owns the four nodes 4q .. 4q + 3 of row j in every plane: x neighbours come by
// shuffle, z neighbours are the thread's own, y neighbours go through shared memory.
//   forward   vx, vz, e in registers; vy, m and m e (+ dm e^n) in shared memory
//   adjoint   lam_x, lam_z and the window accumulator in registers; lam_y, m and mu in
//             shared memory
// (some planes of e / the accumulator in shared memory too where registers run short).
// The exchanged fields carry the halo rows and planes in place, so that every thread reads
// its neighbours at one fixed distance whoever owns them.  The z planes are taken ZC at a
// time: the faces of a chunk, a barrier, its nodes.  (Updating the faces of plane i and the
// nodes of plane i - 1 between the same two barriers costs registers that the deep bricks
// do not have: 14.7 against 13.3 us per gradient step at 128^3.)
//
// Exchange.  Every brick publishes the values its neighbours' faces need (m e, or mu) of
// its first and last rows and planes, and its neighbours recompute the faces they share
// by the owner's expression, so one exchange per step is enough and results are bitwise
// those of the streaming kernels.  Each FP32 value travels in one 64-bit word beside the
// tag of its step, so its arrival is its own signal: no fence and no flag, half the
// latency of a flag that follows the data.  Words are double-buffered by step parity; a
// brick overwrites a word only after it has received the neighbour's next values, which
// the neighbour computed from it.  Tags never repeat within a handle.
//
// Every wait is bounded (2 s, or the error flag of another CTA); a wait that gives up
// sets the sticky error flag and the kernel runs to its end without waiting again.
#pragma once

#include "aew_brick.h"
#include "aew_stencil.cuh"

namespace aew {
namespace brick {

using namespace quad;

constexpr uint64_t kWaitNs = 2000000000ull;
constexpr int kSmemMax = 232448;   // 227 KB
constexpr int kMaxBz = 8;

// Limits and layout by depth.  Each depth is compiled for itself, so the tables trade registers
// (65,536 per SM), shared memory (smem_bytes below) and barriers; bytes spilled per thread are
// -Xptxas -v's for the FP32 adjoint, the tightest kernel of each depth.
// Threads: a kernel needs about 45 working registers and 8 to 12 per plane, so two planes fit
// 65,536 / 640 = 102 registers, up to seven 128, eight 168.
__host__ __device__ constexpr int tmax(int bz) {
  return bz <= 2 ? 640 : bz <= 7 ? 512 : 384;
}
// Longest x row, in float4: the exchanged field holds two rows beyond the brick and the y faces one
// in every plane.  128 (512 nodes) where that is a small part; 64 from five planes on; at seven only
// 32 fits beside four shared planes of the third field (225,216 of 231,424 B; 64 would take 236,992).
__host__ __device__ constexpr int nqmax(int bz) { return bz <= 4 ? 128 : bz == 7 ? 32 : 64; }
// Planes per chunk of the forward and the adjoint kernels: a chunk is a barrier, so two where the
// registers of a second plane's faces are there.  In the adjoint they are up to four planes (from
// five on two would spill 64 B for 8, 204 for 72, 340 for 184, 48 for 0), in the forward kernel up to
// five (six would spill 44 B for 20, seven 88 for 56), with dm e^n in flight up to four.
__host__ __device__ constexpr int zc(int bz, bool incr) { return bz <= 2 ? bz : bz <= (incr ? 4 : 5) ? 2 : 1; }
__host__ __device__ constexpr int zca(int bz) { return bz <= 1 ? bz : bz <= 4 ? 2 : 1; }
// Planes whose third register field (e, or the accumulator) lives in shared memory instead, each for
// 16 B per thread and access: two at five planes (8 B spilled; 44 with none), three at six (72; 212
// with none, 24 with a fourth, which was not timed), four at seven, as many as fit (184; 372 with
// none), two at eight (0; 44 with none).
__host__ __device__ constexpr int ks(int bz) { return bz == 5 || bz == 8 ? 2 : bz == 6 ? 3 : bz == 7 ? 4 : 0; }
// row pitches (float4) of the exchanged field (a halo row on both sides), of the y faces (one
// below) and of the private fields: constants, so that plane offsets are immediates
__host__ __device__ constexpr int pe(int bz) { return tmax(bz) + 2 * nqmax(bz); }
__host__ __device__ constexpr int pv(int bz) { return tmax(bz) + nqmax(bz); }

__host__ __device__ constexpr int smem_bytes(int bz) {
  // exchanged field and the plane above it; y faces; m; third field; last x-faces of warps
  return ((bz + 1) * pe(bz) + bz * pv(bz) + (bz + ks(bz)) * tmax(bz)) * 16 + bz * (tmax(bz) / 32) * 4;
}
static_assert(smem_bytes(7) <= kSmemMax - 1024 && smem_bytes(6) <= kSmemMax - 1024 &&
              smem_bytes(4) <= kSmemMax - 1024 && smem_bytes(8) <= kSmemMax - 1024 &&
              smem_bytes(5) <= kSmemMax - 1024 && smem_bytes(3) <= kSmemMax - 1024 &&
              smem_bytes(2) <= kSmemMax - 1024 && smem_bytes(1) <= kSmemMax - 1024, "");

// v, but unknown to the optimiser: what is computed from it inside a step is computed there
// instead of being held in registers across the time loop
__device__ __forceinline__ uint32_t fresh_copy(uint32_t v) {
  asm volatile("" : "+r"(v));
  return v;
}

// ---- the exchange buffer ---------------------------------------------------------------
// z faces: [parity][cta][face][half][tmax] of 16 B, face 0 the first plane, 1 the last;
// y faces: [parity][cta][face][plane][half][nq] behind them
template <int BZ>
struct Words {
  static constexpr int TP = tmax(BZ);
  ulonglong2* base;
  uint32_t nq, ctas, cta;
  __device__ __forceinline__ Words(unsigned char* b, int nq_, int ctas_)
      : base(reinterpret_cast<ulonglong2*>(b)), nq(nq_), ctas(ctas_), cta(blockIdx.x) {}
  // z face 0 / 1 of the brick `step` CTAs on, at parity par, thread tid
  __device__ __forceinline__ ulonglong2* z(int par, int step, int face, uint32_t tid) const {
    return base + ((par * ctas + cta + step) * (4 * TP) + face * (2 * TP) + tid);
  }
  // y face 0 / 1: plane k, quad q
  __device__ __forceinline__ ulonglong2* y(int par, int step, int face, uint32_t k, uint32_t q) const {
    return base + (2 * ctas * (4 * TP) + (((par * ctas + cta + step) * 4 + face * 2) * BZ + 2 * k) * nq + q);
  }
  __device__ __forceinline__ uint32_t ypar() const { return ctas * 4 * BZ * nq; }   // parity distance
};

__device__ __forceinline__ void publish(ulonglong2* p, int stride, float4 v, uint32_t tag) {
  const unsigned long long t = (unsigned long long)tag << 32;
  asm volatile("st.relaxed.gpu.global.v2.b64 [%0], {%1, %2};" ::"l"(p), "l"(t | __float_as_uint(v.x)),
               "l"(t | __float_as_uint(v.y))
               : "memory");
  asm volatile("st.relaxed.gpu.global.v2.b64 [%0], {%1, %2};" ::"l"(p + stride),
               "l"(t | __float_as_uint(v.z)), "l"(t | __float_as_uint(v.w))
               : "memory");
}
__device__ __forceinline__ ulonglong2 ld_words(const ulonglong2* p) {
  ulonglong2 r;
  asm volatile("ld.relaxed.gpu.global.v2.b64 {%0, %1}, [%2];" : "=l"(r.x), "=l"(r.y) : "l"(p) : "memory");
  return r;
}
__device__ __forceinline__ bool fresh(const ulonglong2& a, const ulonglong2& b, uint32_t tag) {
  return (((uint32_t)(a.x >> 32) ^ tag) | ((uint32_t)(a.y >> 32) ^ tag) |
          ((uint32_t)(b.x >> 32) ^ tag) | ((uint32_t)(b.y >> 32) ^ tag)) == 0;
}
__device__ __forceinline__ float4 value(const ulonglong2& a, const ulonglong2& b) {
  return make_float4(__uint_as_float((uint32_t)a.x), __uint_as_float((uint32_t)a.y),
                     __uint_as_float((uint32_t)b.x), __uint_as_float((uint32_t)b.y));
}
// A wait that has not ended after a while: false once it is to be given up.  `dead`
// (shared): a wait of this CTA gave up before.
__device__ __forceinline__ bool keep_waiting(uint32_t& t0, volatile int* dead, int* err) {
  const uint32_t t = (uint32_t)(tc::globaltimer() >> 10) | 1u;   // about microseconds
  if (t0 == 0) t0 = t;
  if (t - t0 <= (uint32_t)(kWaitNs >> 10) && !*dead && *reinterpret_cast<volatile int*>(err) == 0) return true;
  *dead = 1;
  atomicExch(err, 1);
  return false;
}
// the value of one words group into *dst (shared)
__device__ __forceinline__ void receive(const ulonglong2* p, int stride, float4* dst, uint32_t tag,
                                        volatile int* dead, int* err) {
  uint32_t t0 = 0;
  for (uint32_t it = 1;; ++it) {
    const ulonglong2 a = ld_words(p), b = ld_words(p + stride);
    if (fresh(a, b, tag)) {
      *dst = value(a, b);
      return;
    }
    if ((it & 63u) == 0 && !keep_waiting(t0, dead, err)) return;
  }
}

// ---- geometry of one CTA and one thread ------------------------------------------------
struct Geo {
  int nq, tid, j, q, i0, y, k0, ka, cta;
  bool act, ylo, yhi, zlo, zhi;   // the thread has nodes; the brick has neighbours
  bool jlo, jhi;                  // the thread's row is the brick's first / last
  uint32_t P, C, row;             // plane and grid sizes (< 2^22 nodes); the thread's nodes in plane k0
  template <class A>
  __device__ __forceinline__ explicit Geo(const A& a) {
    nq = a.nx >> 2;
    tid = threadIdx.x;
    j = tid / nq;
    q = tid - j * nq;
    cta = blockIdx.x;
    const int cy = cta % a.py, cz = cta / a.py;
    const int y0 = cy * a.by;
    k0 = cz * a.bz;
    const int rows = min(a.by, a.ny - y0);
    ka = min(a.bz, a.nz - k0);
    act = j < rows;
    y = y0 + j;
    i0 = 4 * q;
    ylo = cy > 0;
    yhi = cy + 1 < a.py;
    zlo = cz > 0;
    zhi = cz + 1 < a.pz;
    jlo = act && j == 0;
    jhi = act && j == rows - 1;
    P = (uint32_t)a.nx * a.ny;
    C = P * a.nz;
    row = k0 * P + (uint32_t)y * a.nx + i0;
  }
};

// A field of BZ planes of which the first KS live in shared memory
template <int BZ, int KS>
struct Split {
  F4 r[BZ - KS];
  __device__ __forceinline__ F4 get(const float4* s, int k) const {
    return k < KS ? lds(s + k * tmax(BZ)) : r[k < KS ? 0 : k - KS];
  }
  __device__ __forceinline__ void set(float4* s, int k, F4 v) {
    if (k < KS) sts(s + k * tmax(BZ), v);
    else r[k < KS ? 0 : k - KS] = v;
  }
};

// What the forward and adjoint kernels share: where the thread's values are, its place in
// the grid and the exchange of the field E (m e, or mu).  The place is kept in a few packed
// words, unpacked anew in every step: the state leaves no registers for more.
enum : uint32_t {
  kAct = 1u, kZlo = 2u, kZhi = 4u, kLow = 8u, kHi = 16u, kP31 = 32u, kP0 = 64u, kFirstX = 128u,
  kLastX = 256u, kEdgeY = 512u, kLastY = 1024u, kBelow = 2048u, kYin = 4096u
};
template <int BZ>
struct Ctx {
  static constexpr int TP = tmax(BZ), PE = pe(BZ), PV = pv(BZ), NW = TP / 32, NQ = nqmax(BZ);
  // shared memory, in float4 from its start: E rows from NQ (row -1 before them), V rows from
  // NQ (the face below before them), M, the third field's shared planes, the last x-faces
  static constexpr int oE = NQ, oV = (BZ + 1) * PE + NQ, oM = (BZ + 1) * PE + BZ * PV, oS = oM + BZ * TP,
                       oX = oS + ks(BZ) * TP;
  Words<BZ> wd;
  uint32_t fl;     // flags above
  uint32_t bits;   // bits 0-7 planes in which the thread has nodes, 8-15 planes on the boundary,
                   // 16-31 planes with rare work
  uint32_t row;    // the thread's nodes in plane k0
  uint32_t yin;    // the thread's halo row item at parity 0
  uint32_t ydst;   // .. and its place (float4)

  __device__ __forceinline__ Ctx(const Geo& g, unsigned char* halo, int by, int py, int pz, int ny, int nz)
      : wd(halo, g.nq, py * pz) {
    const int lane = g.tid & 31;
    const bool edge_y = g.y == 0 || g.y >= ny - 1;
    fl = (g.act ? kAct : 0) | (g.act && g.zlo ? kZlo : 0) | (g.act && g.zhi ? kZhi : 0) |
         (g.jlo && g.ylo ? kLow : 0) | (g.jhi && g.yhi ? kHi : 0) |
         (lane == 31 && g.q < g.nq - 1 ? kP31 : 0) | (lane == 0 && g.q > 0 ? kP0 : 0) |
         (g.q == 0 ? kFirstX : 0) | (g.q == g.nq - 1 ? kLastX : 0) | (edge_y ? kEdgeY : 0) |
         (g.y >= ny - 1 ? kLastY : 0);
    bits = (g.act ? (1u << g.ka) - 1 : 0) | (g.k0 == 0 ? 256u : 0u) |
           (g.k0 + g.ka == nz ? 256u << (g.ka - 1) : 0u);
    row = g.row;
    yin = ydst = 0;
    if (g.tid < 2 * g.ka * g.nq && yitem(g, by, g.tid, yin, ydst)) fl |= kYin;
  }
  // halo row item w: plane and quad of the row below (w < ka nq) or above the brick
  __device__ __forceinline__ bool yitem(const Geo& g, int by, int w, uint32_t& src, uint32_t& dst) const {
    const int n = g.ka * g.nq;
    const bool up = w >= n;
    if (!(up ? g.yhi : g.ylo)) return false;
    if (up) w -= n;
    const int k = w / g.nq, q = w - k * g.nq;
    src = (uint32_t)(wd.y(0, up ? 1 : -1, up ? 0 : 1, k, q) - wd.base);
    // the row below is at - nq of row 0; the one above follows the brick's rows
    dst = oE + k * PE + (up ? by * g.nq : -g.nq) + q;
    return true;
  }
  // start of a step: the halo rows into E (spread over the threads), the plane below
  // returned, and with ABOVE the plane above into its place; then the barrier that also ends
  // the step before.  Without ABOVE the kernel fetches the plane above while it works on the
  // planes before it (fetch_above, take_above): three fetches at once cost it spills.
  template <bool ABOVE>
  __device__ __forceinline__ F4 receive_halos(const Geo& g, float4* f, int by, int py, int par, uint32_t tag,
                                              volatile int* dead, int* err) const {
    const uint32_t tid = fresh_copy(threadIdx.x);
    uint32_t want = fresh_copy(fl) & (kZlo | (ABOVE ? kZhi : 0u) | kYin);
    float4 below = z4();
    if (*dead) want = 0;
    uint32_t t0 = 0;
    const ulonglong2* lo = wd.z(par, -py, 1, tid);
    const ulonglong2* hi = wd.z(par, py, 0, tid);
    const ulonglong2* yw = wd.base + (yin + (par ? wd.ypar() : 0u));
    for (uint32_t it = 1; want; ++it) {
      ulonglong2 a0, a1, b0, b1, c0, c1;
      if (want & kZlo) {
        a0 = ld_words(lo);
        a1 = ld_words(lo + TP);
      }
      if (ABOVE && (want & kZhi)) {
        b0 = ld_words(hi);
        b1 = ld_words(hi + TP);
      }
      if (want & kYin) {
        c0 = ld_words(yw);
        c1 = ld_words(yw + wd.nq);
      }
      if ((want & kZlo) && fresh(a0, a1, tag)) {
        below = value(a0, a1);
        want &= ~kZlo;
      }
      if (ABOVE && (want & kZhi) && fresh(b0, b1, tag)) {
        f[oE + g.ka * PE + tid] = value(b0, b1);
        want &= ~kZhi;
      }
      if ((want & kYin) && fresh(c0, c1, tag)) {
        f[ydst] = value(c0, c1);
        want &= ~kYin;
      }
      if ((it & 63u) == 0 && !keep_waiting(t0, dead, err)) break;
    }
    for (int w = tid + blockDim.x; w < 2 * g.ka * g.nq; w += blockDim.x) {   // short bricks only
      uint32_t src, dst;
      if (yitem(g, by, w, src, dst) && !*dead)
        receive(wd.base + (src + (par ? wd.ypar() : 0u)), wd.nq, f + dst, tag, dead, err);
    }
    __syncthreads();
    return f4(below);
  }
  struct Above {
    ulonglong2 a, b;
  };
  __device__ __forceinline__ Above fetch_above(int py, int par) const {
    Above v{make_ulonglong2(0, 0), make_ulonglong2(0, 0)};
    if (fl & kZhi) {
      const ulonglong2* p = wd.z(par, py, 0, fresh_copy(threadIdx.x));
      v.a = ld_words(p);
      v.b = ld_words(p + TP);
    }
    return v;
  }
  __device__ __forceinline__ void take_above(const Above& v, const Geo& g, float4* f, int py, int par, uint32_t tag,
                                             volatile int* dead, int* err) const {
    if (!(fl & kZhi)) return;
    const uint32_t tid = fresh_copy(threadIdx.x);
    float4* dst = f + oE + g.ka * PE + tid;
    if (fresh(v.a, v.b, tag)) *dst = value(v.a, v.b);
    else if (!*dead) receive(wd.z(par, py, 0, tid), TP, dst, tag, dead, err);
  }
  // plane k of E, v, for the y neighbours (threads of the first and last rows)
  __device__ __forceinline__ void publish_y(const Geo& g, float4 v, int by, int par, uint32_t tag, int k) const {
    const uint32_t tid = fresh_copy(threadIdx.x);
    if (fl & kLow) publish(wd.y(par, 0, 0, k, tid), wd.nq, v, tag);
    if (fl & kHi) publish(wd.y(par, 0, 1, k, tid - (by - 1) * wd.nq), wd.nq, v, tag);
  }
  __device__ __forceinline__ void publish_z(const Geo& g, const float4* f, int par, uint32_t tag) const {
    const uint32_t tid = fresh_copy(threadIdx.x);
    if (fl & kZlo) publish(wd.z(par, 0, 0, tid), TP, f[oE + tid], tag);
    if (fl & kZhi) publish(wd.z(par, 0, 1, tid), TP, f[oE + (g.ka - 1) * PE + tid], tag);
  }
  // zero E and V: halo planes and rows that no neighbour fills stay 0
  __device__ __forceinline__ void clear(float4* f) const {
    for (int i = threadIdx.x; i < oM; i += blockDim.x) f[i] = z4();
    __syncthreads();
  }
};
// the node values of plane k, 0 on the grid's boundary
__device__ __forceinline__ F4 masked(F4 f, uint32_t fl, bool zplane) {
  float4 v = v4(f);
  if ((fl & kEdgeY) || zplane) v = z4();
  if (fl & kFirstX) v.x = 0.f;
  if (fl & kLastX) v.w = 0.f;
  return f4(v);
}

// ---------------------------------------------------------------------------------
// forward-type steps
// ---------------------------------------------------------------------------------
// INCR 0: forward; 1: + G(dm e^n) with FP32 e^n; 2: with BF16 e^n.  TPACK: window packing.
template <int BZ, int INCR, bool TPACK>
__global__ void __launch_bounds__(tmax(BZ), 1) fwd_kernel(const __grid_constant__ BrickFwd a) {
  constexpr int ZC = zc(BZ, INCR != 0), NC = (BZ + ZC - 1) / ZC, KS = ks(BZ);
  using X = Ctx<BZ>;
  constexpr int PE = X::PE, PV = X::PV, TP = X::TP, NW = X::NW;
  extern __shared__ __align__(16) unsigned char smem[];
  __shared__ int dead_s;
  if (sticky_error(a.err)) return;
  float4* const f = reinterpret_cast<float4*>(smem);
  volatile int* dead = &dead_s;
  const Geo g(a);
  X c(g, a.halo, a.by, a.py, a.pz, a.ny, a.nz);
  if (g.tid == 0) dead_s = 0;
  c.clear(f);
  const F4 dth = f4(make_float4(a.dth, a.dth, a.dth, a.dth));
  const int nq = a.nx >> 2;
  // planes with rare work: bit 16 + k the source, 24 + k receivers
  if (g.act) {
    if (a.sk >= 0 && abs(g.y - a.sj) <= a.sr && g.i0 + 3 >= a.si - a.sr && g.i0 <= a.si + a.sr) {
      for (int k = 0; k < g.ka; ++k)
        if (abs(g.k0 + k - a.sk) <= a.sr) c.bits |= 0x10000u << k;
      if (g.zlo && abs(g.k0 - 1 - a.sk) <= a.sr) c.fl |= kBelow;
    }
    if (a.d_out && a.krec >= g.k0 && a.krec < g.k0 + g.ka &&
        has_rec(a.rec_map + (size_t)g.y * a.nx + g.i0))
      c.bits |= 0x1000000u << (a.krec - g.k0);
  }

  F4 vx[BZ], vz[BZ], vzl = f4(z4());
  Split<BZ, KS> e;
  float tm[TPACK ? BZ : 1];
  {
    const int tid = g.tid;
#pragma unroll
    for (int k = 0; k < BZ; ++k) {
      if (TPACK) tm[k] = 0.f;
      float4 m4 = z4(), me = z4(), vy4 = z4(), e4 = z4(), vx4 = z4(), vz4 = z4();
      if (c.bits >> k & 1u) {
        const uint32_t i = g.row + k * g.P;
        m4 = ldg4(a.m + i);
        if (a.e) {
          e4 = ldg4(a.e + i);
          vx4 = ldg4(a.vx + i);
          vy4 = ldg4(a.vy + i);
          vz4 = ldg4(a.vz + i);
          me = mul4(m4, e4);
          if (c.fl & kLow) f[X::oV + k * PV + tid - nq] = ldg4(a.vy + (i - a.nx));
        }
        if (INCR && a.ef_first == 0)
          me = fma4(ldg4(a.dm + i),
                    INCR == 2 ? bf4(__ldg(reinterpret_cast<const uint2*>(a.ef16 + i))) : ldg4(a.ef + i), me);
        f[X::oE + k * PE + tid] = me;
        f[X::oV + k * PV + tid] = vy4;
        if (c.fl & (kLow | kHi)) c.publish_y(g, me, a.by, 0, a.tag, k);
      }
      f[X::oM + k * TP + tid] = m4;
      vx[k] = f4(vx4);
      vz[k] = f4(vz4);
      e.set(f + X::oS + tid, k, f4(e4));
    }
    if ((c.fl & kZlo) && a.e) vzl = f4(ldg4(a.vz + (g.row - g.P)));
    c.publish_z(g, f, 0, a.tag);
  }

  int next_store = 0;
#pragma unroll 1
  for (int n = 0; n < a.nsteps; ++n) {
    const int par = n & 1;
    const uint32_t tag = a.tag + n;
    const bool more = n + 1 < a.nsteps;
    const bool inc = INCR && more && n + 1 >= a.ef_first;   // next step's dm e^n
    const F4 below = c.template receive_halos<NC == 1>(g, f, a.by, a.py, par, tag, dead, a.err);
    const uint32_t tid = fresh_copy(threadIdx.x), fl = fresh_copy(c.fl), bits = fresh_copy(c.bits);
    float4* const E = f + X::oE + tid;
    float4* const V = f + X::oV + tid;
    float* const sx = reinterpret_cast<float*>(f + X::oX) + (tid >> 5);
    F4 me_c = lds(E);
    // the face below the brick, as the brick below computes it
    vzl = fma(dth, sub(me_c, below), vzl);
    if (fl & kBelow) {
      float4 v = v4(vzl);
      add_source(v, g.k0 - 1, g.y, g.i0, a, __ldg(a.dts + n));
      vzl = f4(v);
    }
    typename X::Above above;
#pragma unroll
    for (int ch = 0; ch < NC; ++ch) {
      if (NC > 1 && ch == NC - 2) above = c.fetch_above(a.py, par);
      if (NC > 1 && ch == NC - 1) c.take_above(above, g, f, a.py, par, tag, dead, a.err);
      F4 vyc[ZC];
      float4 dme[INCR ? ZC : 1], efe[INCR == 1 ? ZC : 1];
      uint2 efb[INCR == 2 ? ZC : 1];
      // ---- faces
#pragma unroll
      for (int z = 0; z < ZC; ++z) {
        const int k = ch * ZC + z;
        if (k >= BZ) continue;
        if (INCR && inc && (bits >> k & 1u)) {   // in flight
          const uint32_t i = c.row + k * g.P;
          dme[z] = ldg4(a.dm + i);
          if (INCR == 2) efb[z] = __ldg(reinterpret_cast<const uint2*>(a.ef16 + (size_t)(n + 1) * g.C + i));
          else efe[z] = ldg4(a.ef + (size_t)(n + 1) * g.C + i);
        }
        const F4 me_n = lds(E + (k + 1) * PE);
        const F4 me_yp = lds(E + k * PE + nq);
        const float4 m = v4(me_c);
        float mx1 = __shfl_down_sync(0xffffffffu, m.x, 1);
        if (fl & kP31) mx1 = E[k * PE + 1].x;
        const float4 d = make_float4(__fsub_rn(m.y, m.x), __fsub_rn(m.z, m.y), __fsub_rn(m.w, m.z),
                                     __fsub_rn(mx1, m.w));
        float4 x = v4(fma(dth, f4(d), vx[k]));
        if (fl & kLastX) x.w = 0.f;   // unused last face
        vx[k] = f4(x);
        if ((tid & 31) == 31) sx[k * NW] = x.w;
        const F4 vy = fma(dth, sub(me_yp, me_c), lds(V + k * PV));
        sts(V + k * PV, vy);
        vyc[z] = vy;
        vz[k] = fma(dth, sub(me_n, me_c), vz[k]);
        if (bits >> k & 0x10000u) {
          float4 v = v4(vz[k]);
          add_source(v, g.k0 + k, g.y, g.i0, a, __ldg(a.dts + n));
          vz[k] = f4(v);
        }
        me_c = me_n;
      }
      if (fl & kLow) {   // the y-faces below the brick, as the brick below computes them
#pragma unroll
        for (int z = 0; z < ZC; ++z) {
          const int k = ch * ZC + z;
          if (k < BZ)
            sts(V + k * PV - nq, fma(dth, sub(lds(E + k * PE), lds(E + k * PE - nq)), lds(V + k * PV - nq)));
        }
      }
      __syncthreads();
      // ---- nodes
#pragma unroll
      for (int z = 0; z < ZC; ++z) {
        const int k = ch * ZC + z;
        if (k >= BZ) continue;
        const float4 x = v4(vx[k]);
        float vxl = __shfl_up_sync(0xffffffffu, x.w, 1);
        if (fl & kP0) vxl = sx[k * NW - 1];
        if (fl & kFirstX) vxl = 0.f;
        const F4 dx = f4(make_float4(x.x - vxl, x.y - x.x, x.z - x.y, x.w - x.z));
        const F4 dy = sub(vyc[z], lds(V + k * PV - nq));
        const F4 dz = sub(vz[k], k ? vz[k ? k - 1 : 0] : vzl);
        const F4 e1 = masked(fma(dth, add(add(dx, dy), dz), e.get(f + X::oS + tid, k)), fl, bits >> k & 0x100u);
        e.set(f + X::oS + tid, k, e1);
        F4 me = mul(lds(f + X::oM + k * TP + tid), e1);
        if (INCR && inc && (bits >> k & 1u)) me = fma(f4(dme[z]), f4(INCR == 2 ? bf4(efb[z]) : efe[z]), me);
        if (bits >> k & 1u) {
          sts(E + k * PE, me);
          if (n < a.nhist) __stcs(reinterpret_cast<float4*>(a.hist + (size_t)n * g.C + (c.row + k * g.P)), v4(e1));
          if (TPACK && n < a.npack) {
            const float4 ev = v4(e1);
            const int kk = g.k0 + k, NBx = a.nx >> 3, NBy = a.ny >> 3;
            const uint32_t v = ((uint32_t)(kk >> 1) * NBy + (g.y >> 3)) * NBx + (g.i0 >> 3);
            *reinterpret_cast<uint2*>(a.tpack + (size_t)v * 2048 + (a.tslot + n) * 128 + (kk & 1) * 64 +
                                      (g.y & 7) * 8 + (g.i0 & 7)) =
                make_uint2(pack2bf(ev.x, ev.y), pack2bf(ev.z, ev.w));
            tm[k] = fmaxf(tm[k], hmax4(ev));
          }
        }
      }
      if (more && (fl & (kLow | kHi))) {
#pragma unroll
        for (int z = 0; z < ZC; ++z)
          if (ch * ZC + z < BZ && (bits >> (ch * ZC + z) & 1u))
            c.publish_y(g, E[(ch * ZC + z) * PE], a.by, par ^ 1, tag + 1, ch * ZC + z);
      }
    }
    if (more) c.publish_z(g, f, par ^ 1, tag + 1);
    if (INCR == 0 && !TPACK && next_store < a.nstore && a.store_at[next_store] == n) {   // a checkpoint
      float* const o = a.store[next_store++];
#pragma unroll
      for (int k = 0; k < BZ; ++k)
        if (bits >> k & 1u) {
          const uint32_t i = c.row + k * g.P;
          st4(o, i, v4(e.get(f + X::oS + tid, k)));
          st4(o, i + g.C, v4(vx[k]));
          st4(o, i + 2 * g.C, fl & kLastY ? z4() : V[k * PV]);
          st4(o, i + 3 * g.C, g.k0 + k == a.nz - 1 ? z4() : v4(vz[k]));
        }
    }
    if (bits & 0xff000000u) {   // receivers
#pragma unroll
      for (int k = 0; k < BZ; ++k)
        if (bits >> k & 0x1000000u)   // the last y- and z-faces of the grid are unused: 0
          record(a.rec_map + (size_t)g.y * a.nx + g.i0, a.d_out + (size_t)n * a.nrow, v4(vx[k]),
                 fl & kLastY ? z4() : V[k * PV], g.k0 + k == a.nz - 1 ? z4() : v4(vz[k]));
    }
  }

  // ---- state out
  const int tid = g.tid;
#pragma unroll
  for (int k = 0; k < BZ; ++k) {
    if (!(c.bits >> k & 1u)) continue;
    const uint32_t i = g.row + k * g.P;
    if (a.e1) {
      st4(a.e1, i, v4(e.get(f + X::oS + tid, k)));
      st4(a.vx1, i, v4(vx[k]));
      st4(a.vy1, i, c.fl & kLastY ? z4() : f[X::oV + k * PV + tid]);
      st4(a.vz1, i, g.k0 + k == a.nz - 1 ? z4() : v4(vz[k]));
    }
    if (TPACK && tm[k] > 0.f) {
      const uint32_t v = ((uint32_t)((g.k0 + k) >> 1) * (a.ny >> 3) + (g.y >> 3)) * (a.nx >> 3) + (g.i0 >> 3);
      atomicMax(a.vmax + v, __float_as_uint(tm[k]));
    }
  }
}

// ---------------------------------------------------------------------------------
// adjoint steps
// ---------------------------------------------------------------------------------
// B16: the strain is BF16
template <int BZ, bool B16>
__global__ void __launch_bounds__(tmax(BZ), 1) adj_kernel(const __grid_constant__ BrickAdj a) {
  constexpr int ZC = zca(BZ), NC = (BZ + ZC - 1) / ZC, KS = ks(BZ);
  using X = Ctx<BZ>;
  constexpr int PE = X::PE, PV = X::PV, TP = X::TP, NW = X::NW;
  extern __shared__ __align__(16) unsigned char smem[];
  __shared__ int dead_s;
  if (sticky_error(a.err)) return;
  float4* const f = reinterpret_cast<float4*>(smem);
  volatile int* dead = &dead_s;
  const Geo g(a);
  X c(g, a.halo, a.by, a.py, a.pz, a.ny, a.nz);
  if (g.tid == 0) dead_s = 0;
  c.clear(f);
  const F4 dth = f4(make_float4(a.dth, a.dth, a.dth, a.dth));
  const int nq = a.nx >> 2;
  // planes with receivers: bit 16 + k on the thread's own nodes, 24 + k on the row below
  if (g.act && a.resid) {
    const int kr = a.krec - g.k0;
    const int* map = a.rec_map + (size_t)g.y * a.nx + g.i0;
    if (kr >= 0 && kr < g.ka) {
      if (has_rec(map)) c.bits |= 0x10000u << kr;
      if ((c.fl & kLow) && has_rec(map - a.nx)) c.bits |= 0x1000000u << kr;
    }
    if (kr == -1 && g.zlo && has_rec(map)) c.fl |= kBelow;
  }

  F4 lx[BZ], lz[BZ], lzl = f4(z4());
  Split<BZ, KS> acc;
  {
    const int tid = g.tid;
#pragma unroll
    for (int k = 0; k < BZ; ++k) {
      float4 m4 = z4(), mu = z4(), ly4 = z4(), ac = z4(), lx4 = z4(), lz4 = z4();
      if (c.bits >> k & 1u) {
        const uint32_t i = g.row + k * g.P;
        m4 = ldg4(a.m + i);
        if (a.mu) {
          mu = ldg4(a.mu + i);
          lx4 = ldg4(a.lx + i);
          ly4 = ldg4(a.ly + i);
          lz4 = ldg4(a.lz + i);
          if (c.fl & kLow) f[X::oV + k * PV + tid - nq] = ldg4(a.ly + (i - a.nx));
        }
        if (a.w0 > 0) ac = *reinterpret_cast<const float4*>(a.acc32 + i);
        f[X::oE + k * PE + tid] = mu;
        f[X::oV + k * PV + tid] = ly4;
        if (c.fl & (kLow | kHi)) c.publish_y(g, mu, a.by, 0, a.tag, k);
      }
      f[X::oM + k * TP + tid] = m4;
      lx[k] = f4(lx4);
      lz[k] = f4(lz4);
      acc.set(f + X::oS + tid, k, f4(ac));
    }
    if ((c.fl & kZlo) && a.mu) lzl = f4(ldg4(a.lz + (g.row - g.P)));
    c.publish_z(g, f, 0, a.tag);
  }
  int w = a.w0;   // place in the accumulation window

#pragma unroll 1
  for (int n = 0; n < a.nsteps; ++n) {
    const int par = n & 1;
    const uint32_t tag = a.tag + n;
    const bool more = n + 1 < a.nsteps;
    const float* const en_n = B16 ? nullptr : a.nlist ? a.en_list[n] : a.en - (size_t)n * g.C;
    const bool has_e = a.nlist ? en_n != nullptr : n < a.en_steps;
    const F4 below = c.template receive_halos<NC == 1>(g, f, a.by, a.py, par, tag, dead, a.err);
    const uint32_t tid = fresh_copy(threadIdx.x), fl = fresh_copy(c.fl), bits = fresh_copy(c.bits);
    float4* const E = f + X::oE + tid;
    float4* const V = f + X::oV + tid;
    float* const sx = reinterpret_cast<float*>(f + X::oX) + (tid >> 5);
    F4 mu_c = lds(E);
    if (bits & 0xffff0000u) {   // receivers: the residual comes first
      const int* map = a.rec_map + (size_t)g.y * a.nx + g.i0;
      const float* r = a.resid - (size_t)n * a.nrow;
#pragma unroll
      for (int k = 0; k < BZ; ++k) {
        if (bits >> k & 0x10000u) {
          lx[k] = injected(lx[k], map, r);
          sts(V + k * PV, injected(lds(V + k * PV), map, r + 1));
          lz[k] = injected(lz[k], map, r + 2);
        }
        if (bits >> k & 0x1000000u)
          sts(V + k * PV - nq, injected(lds(V + k * PV - nq), map - a.nx, r + 1));
      }
    }
    if (fl & kBelow)
      lzl = injected(lzl, a.rec_map + (size_t)g.y * a.nx + g.i0, a.resid - (size_t)n * a.nrow + 2);
    if (fl & kZlo) lzl = fma(dth, sub(below, mu_c), lzl);
    typename X::Above above;
#pragma unroll
    for (int ch = 0; ch < NC; ++ch) {
      if (NC > 1 && ch == NC - 2) above = c.fetch_above(a.py, par);
      if (NC > 1 && ch == NC - 1) c.take_above(above, g, f, a.py, par, tag, dead, a.err);
      F4 lyc[ZC], muc[ZC];
      float4 en[B16 ? 1 : ZC];
      uint2 enb[B16 ? ZC : 1];
      // ---- faces
#pragma unroll
      for (int z = 0; z < ZC; ++z) {
        const int k = ch * ZC + z;
        if (k >= BZ) continue;
        if (has_e && (bits >> k & 1u)) {   // in flight
          const uint32_t i = c.row + k * g.P;
          if (B16) {
            enb[z] = __ldg(reinterpret_cast<const uint2*>(a.en16 - (size_t)n * g.C + i));
          } else {
            en[z] = ldg4(en_n + i);
            // the next step's strain comes from HBM: into L2 now
            if (n + 1 < a.en_steps) asm volatile("prefetch.global.L2 [%0];" ::"l"(en_n + i - g.C));
          }
        }
        const F4 mu_n = lds(E + (k + 1) * PE);
        const F4 mu_yp = lds(E + k * PE + nq);
        const float4 m = v4(mu_c);
        float mx1 = __shfl_down_sync(0xffffffffu, m.x, 1);
        if (fl & kP31) mx1 = E[k * PE + 1].x;
        float4 x = v4(fma(dth, f4(make_float4(m.x - m.y, m.y - m.z, m.z - m.w, m.w - mx1)), lx[k]));
        if (fl & kLastX) x.w = 0.f;
        lx[k] = f4(x);
        if ((tid & 31) == 31) sx[k * NW] = x.w;
        const F4 ly = fma(dth, sub(mu_c, mu_yp), lds(V + k * PV));
        sts(V + k * PV, ly);
        lyc[z] = ly;
        lz[k] = fma(dth, sub(mu_c, mu_n), lz[k]);
        muc[z] = mu_c;
        mu_c = mu_n;
      }
      if (fl & kLow) {
#pragma unroll
        for (int z = 0; z < ZC; ++z) {
          const int k = ch * ZC + z;
          if (k < BZ)
            sts(V + k * PV - nq, fma(dth, sub(lds(E + k * PE - nq), lds(E + k * PE)), lds(V + k * PV - nq)));
        }
      }
      __syncthreads();
      // ---- nodes
#pragma unroll
      for (int z = 0; z < ZC; ++z) {
        const int k = ch * ZC + z;
        if (k >= BZ) continue;
        const float4 x = v4(lx[k]);
        float lxl = __shfl_up_sync(0xffffffffu, x.w, 1);
        if (fl & kP0) lxl = sx[k * NW - 1];
        if (fl & kFirstX) lxl = 0.f;
        const F4 dx = f4(make_float4(x.x - lxl, x.y - x.x, x.z - x.y, x.w - x.z));
        const F4 dy = sub(lyc[z], lds(V + k * PV - nq));
        const F4 dz = sub(lz[k], k ? lz[k ? k - 1 : 0] : lzl);
        const F4 ndth = f4(make_float4(-a.dth, -a.dth, -a.dth, -a.dth));
        const F4 dq = masked(mul(ndth, add(add(dx, dy), dz)), fl, bits >> k & 0x100u);
        if (bits >> k & 1u) {
          sts(E + k * PE, fma(lds(f + X::oM + k * TP + tid), dq, muc[z]));
          // dJ/dm += dt e^n q
          if (has_e)
            acc.set(f + X::oS + tid, k, fma(f4(B16 ? bf4(enb[z]) : en[z]), dq, acc.get(f + X::oS + tid, k)));
        }
      }
      if (more && (fl & (kLow | kHi))) {
#pragma unroll
        for (int z = 0; z < ZC; ++z)
          if (ch * ZC + z < BZ && (bits >> (ch * ZC + z) & 1u))
            c.publish_y(g, E[(ch * ZC + z) * PE], a.by, par ^ 1, tag + 1, ch * ZC + z);
      }
    }
    if (more) c.publish_z(g, f, par ^ 1, tag + 1);
    if (w == a.W - 1 || (a.last && !more)) {   // the window ends: flush it
#pragma unroll
      for (int k = 0; k < BZ; ++k) {
        if (!(bits >> k & 1u)) continue;
        const float4 s = v4(acc.get(f + X::oS + tid, k));
        double2* p64 = reinterpret_cast<double2*>(a.acc64 + (c.row + k * g.P));
        double2 lo = p64[0], hi = p64[1];
        lo.x += (double)s.x;
        lo.y += (double)s.y;
        hi.x += (double)s.z;
        hi.y += (double)s.w;
        p64[0] = lo;
        p64[1] = hi;
        acc.set(f + X::oS + tid, k, f4(z4()));
        if (k % 3 == 2) asm volatile("" ::: "memory");   // three planes in flight
      }
      w = 0;
    } else {
      ++w;
    }
  }

  const int tid = g.tid;
#pragma unroll
  for (int k = 0; k < BZ; ++k) {
    if (!(c.bits >> k & 1u)) continue;
    const uint32_t i = g.row + k * g.P;
    if (a.mu1) {
      st4(a.mu1, i, f[X::oE + k * PE + tid]);
      st4(a.lx1, i, v4(lx[k]));
      st4(a.ly1, i, c.fl & kLastY ? z4() : f[X::oV + k * PV + tid]);
      st4(a.lz1, i, g.k0 + k == a.nz - 1 ? z4() : v4(lz[k]));
    }
    if (w > 0) st4(a.acc32, i, v4(acc.get(f + X::oS + tid, k)));
  }
}

// ---------------------------------------------------------------------------------
template <auto kernel, class A>
cudaError_t launch_coop(const A& a, const BrickPlan& p, cudaStream_t s) {
  // once per instantiation (thread-safe static initialisation)
  static const cudaError_t attr = cudaFuncSetAttribute(
      kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemMax - 1024);
  if (attr != cudaSuccess) return attr;
  void* args[] = {const_cast<A*>(&a)};
  return cudaLaunchCooperativeKernel(reinterpret_cast<const void*>(kernel), dim3(p.py * p.pz),
                                     dim3(p.threads), args, smem_bytes(p.bz), s);
}

}  // namespace brick
}  // namespace aew
