// Several 2D leapfrog steps per launch (step2d_tile.cu): the split of the
// domain into regions and the launch arguments.
#pragma once

#include "wave_internal.cuh"

namespace wave {

// Regions of 128 x rh cells, outx x outy of them owned inside the domain;
// consecutive regions overlap by 2 h with h = r * steps.  rb: rows per warp.
struct Tile2DPlan {
  int rb, rh, steps, h;
  int outx, outy;
  int nkx, nky;
};

// First cell of region k along an axis of n cells cut into nk regions of w
// cells: every `out` cells, the last one ends at n.
__host__ __device__ __forceinline__ int tile_start(int k, int nk, int out, int n, int w) {
  return k < nk - 1 ? k * out : n - w;
}
// Owned cells [lo, hi): from where the previous region's stop to h before the
// region's own end; the first from 0, the last to n.
__host__ __device__ __forceinline__ int tile_own_lo(int k, int out, int w, int h) {
  return k == 0 ? 0 : (k - 1) * out + w - h;
}
__host__ __device__ __forceinline__ int tile_own_hi(int k, int nk, int out, int n, int w, int h) {
  return k == nk - 1 ? n : k * out + w - h;
}

struct Tile2DArgs {
  Geom g;
  Tile2DPlan plan;
  int nfields;            // 1, or 2 that advance together
  int mix;                // two fields u, lambda: acc -= (lambda - lambda_new)(u - u_new)
  const float* prev[2];   // level n-1 of each field
  const float* cur[2];    // level n
  float* oprev[2];        // level n+nsteps-1 (other buffers than prev, cur)
  float* ocur[2];         // level n+nsteps
  const float* coef;
  const float* bmat;      // density form: b = 1/rho
  float da, dbs;          // density form: as StepArgs
  float* acc;             // sensitivity accumulator (nullable), updated in place
  float* comp;            // Kahan compensation (nullable)
  float acc_scale;        // +1 or -1 (one field; two have -1 and +1)
  int nsteps;             // <= plan.steps
  int overlap;            // the launch before in the stream is a step of the same pass: start while it ends
  int mass_lo, mass_hi;   // steps of the launch that accumulate the (mass) term
  int stiff_lo, stiff_hi; // density form: steps that accumulate the stiffness term
  int level0, dlevel;     // recorded / injected level of the first step, and its change per step
  // receivers (lists per region: entries ptr[t] .. ptr[t+1])
  int nrec;
  const int* tptr;
  const int2* tent;       // {row * 128 + column in the region | owned << 31, receiver}
  float* resid;           // record u - d, time-major (nullable)
  const float* observed;
  int64_t obs_ld;
  float* traces;          // record u, receiver-major (nullable)
  int64_t tr_ld;
  const float* resid_in;  // inject -k w e, time-major residuals (nullable)
  const double* k_dev;
  float weight[2];        // w of each field
  int rec_fields, src_fields;   // two fields: bit f set if field f takes the receivers' / the source's force
  // source
  int sx, sy;
  const float* wavelet;   // nullable
  float h2;
};

cudaError_t launch_tile2d(const Tile2DArgs& a, int physics, int order, cudaStream_t s);
cudaError_t launch_tile2d_o2(const Tile2DArgs& a, cudaStream_t s);   // one translation unit each
cudaError_t launch_tile2d_o4(const Tile2DArgs& a, cudaStream_t s);
cudaError_t launch_tile2d_o6(const Tile2DArgs& a, cudaStream_t s);
cudaError_t launch_tile2d_o8(const Tile2DArgs& a, cudaStream_t s);
cudaError_t launch_tile2d_density(const Tile2DArgs& a, cudaStream_t s);
cudaError_t launch_tile2d_lists(const Tile2DPlan& p, const Geom& g, const int64_t* rec_p, int nrec, int* count,
                                int* ptr, int* cursor, void* ent, cudaStream_t s);
cudaError_t launch_tile2d_skipped(const int64_t* rec_p, int nrec, int lo, int hi, float* resid, float* traces,
                                  int64_t tr_ld, cudaStream_t s);

}  // namespace wave
