// On-chip time loops: launches of the adjoint kernels.
#include "aew_brick.cuh"

namespace aew {
namespace {
template <int BZ>
cudaError_t go(const BrickAdj& a, const BrickPlan& p, cudaStream_t s) {
  if (a.en16) return brick::launch_coop<brick::adj_kernel<BZ, true>>(a, p, s);
  return brick::launch_coop<brick::adj_kernel<BZ, false>>(a, p, s);
}
}  // namespace

cudaError_t launch_brick_adj(BrickAdj a, const BrickPlan& p, unsigned char* halo, uint32_t* tag,
                             int* err, cudaStream_t s) {
  if (!halo || !err || a.nsteps < 1 || (a.nlist && a.nlist != a.nsteps) || a.nlist > kBrickList)
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
