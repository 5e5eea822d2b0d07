// On-chip time loops: launches of the incremental forward kernels.
#include "aew_brick.cuh"

namespace aew {
namespace {
template <int BZ>
cudaError_t go(const BrickFwd& a, const BrickPlan& p, cudaStream_t s) {
  if (a.ef16) return brick::launch_coop<brick::fwd_kernel<BZ, 2, false>>(a, p, s);
  return brick::launch_coop<brick::fwd_kernel<BZ, 1, false>>(a, p, s);
}
}  // namespace

cudaError_t launch_brick_incr(const BrickFwd& a, const BrickPlan& p, cudaStream_t s) {
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
