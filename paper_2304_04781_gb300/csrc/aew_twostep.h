// Two leapfrog (or adjoint) steps in one pass over HBM, for grids too large for the on-chip
// loops (aew_twostep.cu).
#pragma once

#include <cuda_runtime.h>
#include <cstddef>
#include <cstdint>

#include "aew_internal.cuh"

namespace aew {

// how a grid is cut: x tiles of nqt float4 (W with the halo columns), columns of `rows` thread
// rows (rows - 2 of their own), z chunks of kc planes
struct TwoCut {
  int nq, nqt, ntx, W, rows, nty, kc, ntz;
  // estimated time of a forward or adjoint pass by that of two single steps, where these may be
  // the faster ones (otherwise 0)
  double vs_single;
};
TwoCut two_cut(int nx, int ny, int nz, int sms);

// steps n and n + 1 of a forward-type solve: state n -> state n + 2
struct TwoFwd {
  const float* m;
  const float* e;      // state n
  const float* vx;
  const float* vy;
  const float* vz;
  float* e1;           // optional: e^{n+1} (FP32)
  float* e2;           // state n + 2 (no field of state n)
  float* vx2;
  float* vy2;
  float* vz2;
  int nx, ny, nz;
  float dth;
  float dts[2];        // dt s^n, dt s^{n+1} (sk >= 0)
  int si, sj, sk, sr;
  const float* src_w;
  int krec;
  const int* rec_map;
  float* d[2];         // receiver rows of d^{n+1}, d^{n+2} (null: none)
  // incremental solve: + G(dm e), e of steps n and n + 1 as FP32 or BF16 (a null one: none)
  const float* dm;
  const float* ef[2];
  const uint16_t* ef16[2];
  // window packing (time codec): e^{n+1} and e^{n+2} into slots of their windows (null: none)
  uint16_t* tpack[2];
  unsigned* vmax[2];
  int tslot[2];
  int* err;
};

// reverse steps n and n - 1
struct TwoAdj {
  const float* m;
  const float* mu;
  const float* lx;
  const float* ly;
  const float* lz;
  float* mu2;
  float* lx2;
  float* ly2;
  float* lz2;
  int nx, ny, nz;
  float dth;
  // strain of the two steps, FP32 or BF16 (a null one: zero)
  const float* en[2];
  const uint16_t* en16[2];
  float* acc32;
  double* acc64;
  bool open;           // the first step opens an accumulation window
  bool close[2];       // the first / second step ends one
  int krec;
  const int* rec_map;
  const float* resid[2];   // residual rows r^{n+1}, r^n (null: none)
  int* err;
};

cudaError_t launch_two_fwd(const TwoFwd& a, const TwoCut& cut, cudaStream_t s);
cudaError_t launch_two_adj(const TwoAdj& a, const TwoCut& cut, cudaStream_t s);

}  // namespace aew
