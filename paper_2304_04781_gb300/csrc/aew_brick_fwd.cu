// On-chip time loops: how a grid is cut into bricks, and the forward kernels' launches.
#include "aew_brick.cuh"

#include <algorithm>

namespace aew {

// One brick per SM at most.  Among the depths that fit, the one with the least work in its
// largest brick (warps x planes, counting a plane's fixed cost as one warp); a grid whose
// bricks need more threads or shared memory than a CTA has is left to the streaming kernels.
bool brick_plan(int nx, int ny, int nz, int sms, BrickPlan* p) {
  const int nq = nx / 4;
  double best = 0.0;
  bool found = false;
  for (int bz = 1; bz <= brick::kMaxBz; ++bz) {
    const int pz = (nz + bz - 1) / bz;
    if (pz > sms) continue;
    int py = std::min(ny, sms / pz);
    const int by = (ny + py - 1) / py;
    py = (ny + by - 1) / by;
    const int threads = (by * nq + 31) / 32 * 32;
    if (threads > brick::tmax(bz)) continue;
    if (nq > brick::nqmax(bz)) continue;
    const double cost = (double)(threads / 32 + 1) * bz;
    if (!found || cost < best) {
      found = true;
      best = cost;
      *p = BrickPlan{by, bz, py, pz, threads};
    }
  }
  return found;
}

size_t brick_halo_bytes(int nx, const BrickPlan& p) {
  const size_t ctas = (size_t)p.py * p.pz;
  return 2 * ctas * 2 * 2 * ((size_t)brick::tmax(p.bz) + (size_t)p.bz * (nx / 4)) * 16 +
         8 * ctas * 16;   // two sums of two parities, two words each, per CTA
}

cudaError_t brick_tags(uint32_t* tag, uint32_t steps, int nx, const BrickPlan& p, unsigned char* halo,
                       cudaStream_t s) {
  if ((uint64_t)*tag + steps + 4 <= 0xffffffffull) return cudaSuccess;
  *tag = 0;
  return cudaMemsetAsync(halo, 0, brick_halo_bytes(nx, p), s);
}

namespace {
template <int BZ>
cudaError_t go(const BrickFwd& a, const BrickPlan& p, cudaStream_t s) {
  if (a.tpack) return brick::launch_coop<brick::fwd_kernel<BZ, 0, true>>(a, p, s);
  return brick::launch_coop<brick::fwd_kernel<BZ, 0, false>>(a, p, s);
}
}  // namespace

cudaError_t launch_brick_fwd(BrickFwd a, const BrickPlan& p, unsigned char* halo, uint32_t* tag,
                             int* err, cudaStream_t s) {
  if (!halo || !err || a.nsteps < 1 || a.nstore > kBrickList || (a.nstore && (a.dm || a.tpack)))
    return cudaErrorInvalidValue;
  const cudaError_t e = brick_tags(tag, (uint32_t)a.nsteps, a.nx, p, halo, s);
  if (e != cudaSuccess) return e;
  a.by = p.by;
  a.bz = p.bz;
  a.py = p.py;
  a.pz = p.pz;
  a.halo = halo;
  a.tag = *tag + 1;
  a.err = err;
  *tag += (uint32_t)a.nsteps + 1;
  if (a.dm) return a.tpack ? cudaErrorInvalidValue : launch_brick_incr(a, p, s);
  switch (p.bz) {
    case 1: return go<1>(a, p, s);
    case 2: return go<2>(a, p, s);
    case 3: return go<3>(a, p, s);
    case 4: return go<4>(a, p, s);
    case 5: return go<5>(a, p, s);
    case 6: return go<6>(a, p, s);
    case 7: return go<7>(a, p, s);
    case 8: return go<8>(a, p, s);
  }
  return cudaErrorInvalidValue;
}

}  // namespace aew
