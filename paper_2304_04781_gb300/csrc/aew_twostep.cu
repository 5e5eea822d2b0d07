// Two time steps per pass: how a grid is cut, and the launches.
#include "aew_twostep.cuh"

#include <algorithm>

namespace aew {
namespace {

// Whole x rows up to 64 float4, else the fewest equal tiles; as many thread rows as 512
// threads hold; and the z chunk whose CTAs fill whole waves of one CTA per SM with the least
// planes walked (a chunk walks about three more than it owns).
two::Cut make_cut(int nx, int ny, int nz, int sms) {
  two::Cut c{};
  c.nq = nx / 4;
  c.ntx = (c.nq + two::kMaxTileQ - 1) / two::kMaxTileQ;
  c.nqt = (c.nq + c.ntx - 1) / c.ntx;
  if (c.nq % 2 == 0) c.nqt += c.nqt & 1;   // whole 8-node vectors per tile
  c.ntx = (c.nq + c.nqt - 1) / c.nqt;
  c.W = c.nqt + std::min(c.ntx - 1, 2);
  const int by = std::min(two::kThreads / c.W - 2, ny);
  c.nty = (ny + by - 1) / by;
  c.rows = (ny + c.nty - 1) / c.nty + 2;
  c.nty = (ny + c.rows - 3) / (c.rows - 2);
  const long long cols = (long long)c.ntx * c.nty;
  double best = 0.0;
  for (int kc = 4; kc <= std::max(nz, 4); kc += 2) {
    const long long n = cols * ((nz + kc - 1) / kc);
    const double cost = (double)((n + sms - 1) / sms) * (std::min(kc, nz) + 3.5);
    if (best == 0.0 || cost < best) {
      best = cost;
      c.kc = kc;
    }
  }
  c.ntz = (nz + c.kc - 1) / c.kc;
  return c;
}

template <auto kernel, class A>
cudaError_t go(const A& a, int sms, int extra_rows, cudaStream_t s) {
  const two::Cut c = make_cut(a.nx, a.ny, a.nz, sms > 0 ? sms : 1);
  const size_t smem = (4 * (size_t)(two::kThreads + 2 * c.W) + (size_t)two::kRing * extra_rows * c.W) * 16 +
                      2 * two::kThreads / 32 * 4 + 2 * two::kTable * 4;
  // once per instantiation (thread-safe static initialisation)
  static const cudaError_t attr =
      cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, 160 * 1024);
  if (attr != cudaSuccess) return attr;
  kernel<<<(unsigned)((long long)c.ntx * c.nty * c.ntz), two::kThreads, smem, s>>>(a, c);
  return cudaGetLastError();
}

}  // namespace

cudaError_t launch_two_fwd(const TwoFwd& a, int sms, cudaStream_t s) {
  const bool tp = a.tpack[0] || a.tpack[1];
  if (tp && (a.nx % 8 || a.ny % 8 || a.nz % 2)) return cudaErrorInvalidValue;
  if (!a.err || (a.ef[0] && a.ef16[0]) || (a.ef[1] && a.ef16[1])) return cudaErrorInvalidValue;
  if (a.dm) {
    const bool b16 = a.ef16[0] || a.ef16[1];
    if (tp) return b16 ? go<two::fwd_kernel<2, true>>(a, sms, 9, s) : cudaErrorInvalidValue;
    return b16 ? go<two::fwd_kernel<2, false>>(a, sms, 9, s) : go<two::fwd_kernel<1, false>>(a, sms, 9, s);
  }
  return tp ? go<two::fwd_kernel<0, true>>(a, sms, 5, s) : go<two::fwd_kernel<0, false>>(a, sms, 5, s);
}

cudaError_t launch_two_adj(const TwoAdj& a, int sms, cudaStream_t s) {
  if (!a.err || (a.en[0] && a.en16[0]) || (a.en[1] && a.en16[1])) return cudaErrorInvalidValue;
  const bool close = a.close[0] || a.close[1];
  if (a.en16[0] || a.en16[1])
    return close ? go<two::adj_kernel<true, true>>(a, sms, 3, s) : go<two::adj_kernel<true, false>>(a, sms, 3, s);
  return close ? go<two::adj_kernel<false, true>>(a, sms, 3, s) : go<two::adj_kernel<false, false>>(a, sms, 3, s);
}

}  // namespace aew
