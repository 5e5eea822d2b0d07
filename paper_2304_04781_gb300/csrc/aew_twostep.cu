// Two time steps per pass: how a grid is cut, and the launches.
#include "aew_twostep.cuh"

#include <algorithm>

namespace aew {

// Equal x tiles of 16 to 64 float4, as many thread rows as 512 threads hold, and z chunks,
// chosen together: a CTA takes about the same time for each plane it walks, and a chunk costs
// about six more than it owns (three or four walked, and the start), so the best cut has the
// least planes times whole waves of one CTA per SM.  Tiles narrower than the grid have halo
// columns and unaligned rows: a plane takes 1.2 times as long (256^3 forward 57 us per step in
// one tile, 73 in two; 512 x 512 x 256 301, 283, 276 and 292 in two to five).
//
// Against single steps.  A pass takes about 1.5 us per plane of that cost in one wave, 1.15 in
// more (a second wave's start hides).  Where rows are whole 128-node tiles of the single-step
// kernels and the state (36 B per node) stays in L2, a single step takes 7.45 us per million
// nodes and no less than 11.4, and passes of several x tiles lose.  us per forward step (nz x ny
// x nx), single / two: 8 x 512 x 512 15.6 / 17.6, 8 x 256 x 1024 15.6 / 18.7, 16 x 256 x 512 15.6
// / 16.7, 4 x 64 x 4096 11.4 / 12.4; but 64 x 64 x 512 15.6 / 14.6, 16 x 512 x 512 30.3 / 28.3,
// and rows that fill no tile 40 x 200 x 320 20.8 / 17.2, one x tile 160^3 36 / 18.6.  Adjoint steps
// divide alike; incremental ones gain on all but the first two (18.2 / 19.1, 18.4 / 19.6), and the
// time codec's solves gain on 32 x 128 x 512, where forward steps lose (15.6 / 16.6; gradient step
// 48.5 / 46.0).
TwoCut two_cut(int nx, int ny, int nz, int sms) {
  TwoCut best{};
  double least = 0.0;
  const int nq = nx / 4;
  for (int ntx = (nq + two::kMaxTileQ - 1) / two::kMaxTileQ; ntx == 1 || nq / ntx >= 16; ++ntx) {
    TwoCut c{};
    c.nq = nq;
    c.nqt = (nq + ntx - 1) / ntx;
    if (nq % 2 == 0) c.nqt += c.nqt & 1;   // whole 8-node vectors per tile
    c.ntx = (nq + c.nqt - 1) / c.nqt;
    c.W = c.nqt + std::min(c.ntx - 1, 2);
    const int by = std::min(two::kThreads / c.W - 2, ny);
    c.nty = (ny + by - 1) / by;
    c.rows = (ny + c.nty - 1) / c.nty + 2;
    c.nty = (ny + c.rows - 3) / (c.rows - 2);
    const long long cols = (long long)c.ntx * c.nty;
    for (c.kc = 4; c.kc <= std::max(nz, 4); c.kc += 2) {
      c.ntz = (nz + c.kc - 1) / c.kc;
      const double cost = (double)((cols * c.ntz + sms - 1) / sms) * (std::min(c.kc, nz) + 6) *
                          (c.ntx > 1 ? 1.2 : 1.0);
      if (best.ntx == 0 || cost < least) {
        least = cost;
        best = c;
      }
    }
  }
  const double m = (double)nx * ny * nz / 1e6;
  const double pass = ((long long)best.ntx * best.nty * best.ntz <= sms ? 1.5 : 1.15) * least;
  const bool close = best.ntx > 1 && nx % 128 == 0 && 36.0 * m <= 96.0;
  best.vs_single = close ? pass / (2.0 * std::max(11.4, 7.45 * m)) : 0.0;
  return best;
}

namespace {

// shared memory: own ring, plane buffers, `planes` planes of `extra_rows` rows beyond the
// column, edge words and maxima tables, the packed strain's stage
template <auto kernel, class A>
cudaError_t go(const A& a, const TwoCut& c, int ring, int buffers, int planes, int extra_rows, bool stage,
               cudaStream_t s) {
  const size_t smem = ((size_t)ring * two::kThreads + buffers * (size_t)(two::kThreads + 2 * c.W) +
                       (size_t)planes * extra_rows * c.W) * 16 +
                      2 * two::kThreads / 32 * 4 + 2 * two::kTable * 4 +
                      (stage ? 4 * (size_t)c.rows * (c.nqt + 2) * 8 : 0);
  // once per instantiation (thread-safe static initialisation)
  static const cudaError_t attr =
      cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024);
  if (attr != cudaSuccess) return attr;
  kernel<<<(unsigned)((long long)c.ntx * c.nty * c.ntz), two::kThreads, smem, s>>>(a, c);
  return cudaGetLastError();
}

}  // namespace

cudaError_t launch_two_fwd(const TwoFwd& a, const TwoCut& cut, cudaStream_t s) {
  const bool tp = a.tpack[0] || a.tpack[1];
  if (tp && (a.nx % 8 || a.ny % 8 || a.nz % 2)) return cudaErrorInvalidValue;
  if (!a.err || (a.ef[0] && a.ef16[0]) || (a.ef[1] && a.ef16[1])) return cudaErrorInvalidValue;
  if (a.dm) {
    const bool b16 = a.ef16[0] || a.ef16[1];
    if (tp) return b16 ? go<two::fwd_kernel<2, true>>(a, cut, 0, 4, two::kRing, 9, false, s) : cudaErrorInvalidValue;
    return b16 ? go<two::fwd_kernel<2, false>>(a, cut, 0, 4, two::kRing, 9, false, s) : go<two::fwd_kernel<1, false>>(a, cut, 0, 4, two::kRing, 9, false, s);
  }
  return tp ? go<two::forward_pack_kernel>(a, cut, two::kPackRing, 6, two::kExtra, 5, true, s)
            : go<two::forward_kernel>(a, cut, two::kOwnRing, 6, two::kRing, 5, false, s);
}

cudaError_t launch_two_adj(const TwoAdj& a, const TwoCut& cut, cudaStream_t s) {
  if (!a.err || (a.en[0] && a.en16[0]) || (a.en[1] && a.en16[1])) return cudaErrorInvalidValue;
  const bool close = a.close[0] || a.close[1];
  if (a.en16[0] || a.en16[1])
    return close ? go<two::adjoint_kernel<true, true>>(a, cut, two::kAdjRing, 6, two::kRing, 3, false, s)
                 : go<two::adjoint_kernel<true, false>>(a, cut, two::kAdjRing, 6, two::kRing, 3, false, s);
  return close ? go<two::adjoint_kernel<false, true>>(a, cut, two::kAdjRing, 6, two::kRing, 3, false, s)
               : go<two::adjoint_kernel<false, false>>(a, cut, two::kAdjRing, 6, two::kRing, 3, false, s);
}

}  // namespace aew
