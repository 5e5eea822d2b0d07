// Interface of the on-chip stencil kernels (aew_brick.cuh): time loops of grids whose
// state fits the SMs' registers and shared memory, many steps per launch.
#pragma once

#include <cuda_runtime.h>
#include <cstddef>
#include <cstdint>

namespace aew {

// How a grid is cut: py x pz bricks of by rows and bz planes (whole x rows), one CTA each;
// the last brick of either axis may be smaller.
struct BrickPlan {
  int by = 0, bz = 0, py = 0, pz = 0;
  int threads = 0;   // by * nx / 4 rounded up to whole warps
};

// entries of the per-step lists below
constexpr int kBrickList = 32;

// One launch: `nsteps` forward-type steps n = 0 .. nsteps - 1 (indices inside the launch).
struct BrickFwd {
  const float* m;
  const float* e;      // state in (null: the zero state; then vx, vy, vz are not read)
  const float* vx;
  const float* vy;
  const float* vz;
  float* e1;           // state out (null: not kept); not the state in
  float* vx1;
  float* vy1;
  float* vz1;
  int nx, ny, nz;
  float dth;
  int nsteps;
  const float* dts;    // device [nsteps]: dt s^n (read where sk >= 0)
  int si, sj, sk, sr;  // source, as in FwdStep
  const float* src_w;
  int krec;            // receiver plane (-1: none)
  const int* rec_map;
  float* d_out;        // row of step 0's output, rows nrow floats apart (null: none)
  size_t nrow;
  float* hist;         // e^{n+1} of step n to hist + n C for n < nhist (null: none)
  int nhist;
  // checkpoints: the state after step store_at[i] (increasing) also to store[i] (e, vx, vy, vz
  // one after the other)
  int nstore;
  int store_at[kBrickList];
  float* store[kBrickList];
  // incremental solve: step n adds G(dm e^n), e^n = ef + n C (FP32) or ef16 + n C (BF16);
  // ef_first: the first step that has it (the initial strain is 0)
  const float* dm;
  const float* ef;
  const uint16_t* ef16;
  int ef_first;
  // window packing (time codec), as in FwdStep: the output of step n < npack goes to slot
  // tslot + n
  int npack;
  uint16_t* tpack;
  unsigned* vmax;
  int tslot;
  // filled in by the launcher
  int by, bz, py, pz;
  unsigned char* halo;
  uint32_t tag;
  int* err;
};

// One launch: `nsteps` adjoint steps, in the order they run.
struct BrickAdj {
  const float* m;
  const float* mu;     // state in (null: the zero state)
  const float* lx;
  const float* ly;
  const float* lz;
  float* mu1;          // state out (null: not kept); not the state in
  float* lx1;
  float* ly1;
  float* lz1;
  int nx, ny, nz;
  float dth;
  int nsteps;
  // strain of step n: en - n C (FP32) or en16 - n C (BF16); steps n >= en_steps have none
  const float* en;
  const uint16_t* en16;
  int en_steps;
  // .. or, with nlist = nsteps, en_list[n] (null: none)
  int nlist;
  const float* en_list[kBrickList];
  const float* resid;  // residual row of step 0; step n reads resid - n nrow (null: none)
  size_t nrow;
  int krec;
  const int* rec_map;
  float* acc32;        // window accumulator: read if w0 > 0, written if the launch ends inside
  double* acc64;
  int w0, W;           // step 0's place in its window of W steps
  bool last;           // the launch's last step also ends its window
  int by, bz, py, pz;
  unsigned char* halo;
  uint32_t tag;
  int* err;
};

// CG for A x = w of the prior's operator (aew_newton.cu), up to max_iter iterations in one launch:
// r = sc w at the start, x scaled by 1 / sc at the end; the residual test every 8 iterations
// (and after the last): r.r <= tol2.  Where more iterations may follow (more; max_iter is then a
// multiple of 8) a launch that did not pass leaves x unscaled, r, p and r.r for the next one (resume).
struct BrickCg {
  const float* w;
  float* x;
  float* r;                // between launches
  float* p;
  bool resume, more;
  int nx, ny, nz;
  float alpha, at, sc, inv_sc;
  float rr_hi, rr_lo;      // r.r at the start, as a pair of floats
  double tol2;
  int max_iter;
  int* result;             // device [2]: iterations, 1 if the test passed
  const float* rr_in;      // device [2] each: r.r as a pair of floats, from the launch before and
  float* rr_out;           // for the next one (two places: all CTAs read the one, CTA 0 writes the other)
  int by, bz, py, pz;
  unsigned char* halo;
  uint32_t tag;
  int* err;
};

// false where the grid does not fit (or sms is not known)
bool brick_plan(int nx, int ny, int nz, int sms, BrickPlan* p);
// bytes of the halo exchange buffer (zeroed once by its owner)
size_t brick_halo_bytes(int nx, const BrickPlan& p);
// halo / tag: the handle's exchange buffer and its running tag, advanced by the launch
cudaError_t launch_brick_fwd(BrickFwd a, const BrickPlan& p, unsigned char* halo, uint32_t* tag,
                             int* err, cudaStream_t s);
cudaError_t launch_brick_adj(BrickAdj a, const BrickPlan& p, unsigned char* halo, uint32_t* tag,
                             int* err, cudaStream_t s);
cudaError_t launch_brick_cg(BrickCg a, const BrickPlan& p, unsigned char* halo, uint32_t* tag,
                            int* err, cudaStream_t s);
// before a launch that uses up to `steps` tags: where they would wrap, the buffer is cleared and
// they start over
cudaError_t brick_tags(uint32_t* tag, uint32_t steps, int nx, const BrickPlan& p, unsigned char* halo,
                       cudaStream_t s);
// per kernel family (internal to the launchers)
cudaError_t launch_brick_incr(const BrickFwd& a, const BrickPlan& p, cudaStream_t s);

}  // namespace aew
