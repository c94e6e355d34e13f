// Several 2D steps per launch: per-region lists of receivers, and the dispatch.
#include "step2d_tile.cuh"

namespace wave {
namespace {

// ---- per-region lists of receivers -------------------------------------------
// A receiver belongs to every region that holds its cell; the region that owns
// the cell has the sign bit set.  count = nullptr in the filling pass.
//
// Neighbouring receivers mostly fall into the same region, so a warp's lanes
// with the same region share one atomic: the regions are few, and an atomic per
// receiver queues up on their counters (a forward of 20 steps of 2048^2, order 2,
// with 1e6 receivers in a block: 1.98 ms that way, 0.48 this way).  All lanes
// therefore walk the same number of candidate regions: those of the evenly
// placed ones that can hold a cell, then the last.
__global__ void tile2d_list_kernel(Tile2DPlan P, Geom g, const int64_t* __restrict__ rec_p, int nrec,
                                   int* __restrict__ count, int* __restrict__ cursor, int2* __restrict__ ent) {
  const int r = blockIdx.x * blockDim.x + threadIdx.x, lane = threadIdx.x & 31;
  const int64_t p = r < nrec ? rec_p[r] : -1;
  const bool in = p >= 0;
  const int y = in ? (int)(p / g.px) : 0, x = in ? (int)(p - (int64_t)y * g.px) : 0;
  const int nx = (int)g.nx, ny = (int)g.ny;
  const int ky0 = y < P.rh ? 0 : (y - P.rh) / P.outy + 1, kx0 = x < kStrip ? 0 : (x - kStrip) / P.outx + 1;
  const int by = min((P.rh - 1) / P.outy + 1, P.nky - 1), bx = min((kStrip - 1) / P.outx + 1, P.nkx - 1);
  for (int iy = 0; iy <= by; ++iy) {
    const int ky = iy < by ? ky0 + iy : P.nky - 1;
    const int ys = tile_start(ky, P.nky, P.outy, ny, P.rh);
    const bool yin = in && (iy == by || ky < P.nky - 1) && y >= ys && y < ys + P.rh;
    if (!__any_sync(0xffffffffu, yin)) continue;
    for (int ix = 0; ix <= bx; ++ix) {
      const int kx = ix < bx ? kx0 + ix : P.nkx - 1;
      const int xs = tile_start(kx, P.nkx, P.outx, nx, kStrip);
      const bool here = yin && (ix == bx || kx < P.nkx - 1) && x >= xs && x < xs + kStrip;
      if (!__any_sync(0xffffffffu, here)) continue;
      const int t = here ? ky * P.nkx + kx : -1;
      const unsigned same = __match_any_sync(0xffffffffu, t);
      const int leader = __ffs(same) - 1;
      if (count) {   // nothing waits for these
        if (here && lane == leader) atomicAdd(count + t, __popc(same));
        continue;
      }
      int first = 0;
      if (here && lane == leader) first = atomicAdd(cursor + t, __popc(same));
      first = __shfl_sync(0xffffffffu, first, leader) + __popc(same & ((1u << lane) - 1u));
      if (here) {
        const bool own = y >= tile_own_lo(ky, P.outy, P.rh, P.h) && y < tile_own_hi(ky, P.nky, P.outy, ny, P.rh, P.h) &&
                         x >= tile_own_lo(kx, P.outx, kStrip, P.h) && x < tile_own_hi(kx, P.nkx, P.outx, nx, kStrip, P.h);
        const int pos = (y - ys) * kStrip + (x - xs);
        ent[first] = make_int2(pos | (own ? (int)0x80000000 : 0), r);
      }
    }
  }
}

// ptr[0..n] = exclusive prefix sums of count[0..n-1]; cursor = ptr (one block)
__global__ void tile2d_scan_kernel(const int* __restrict__ count, int n, int* __restrict__ ptr, int* __restrict__ cursor) {
  __shared__ int wsum[32];
  __shared__ int carry;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  if (threadIdx.x == 0) carry = 0;
  __syncthreads();
  for (int base = 0; base < n; base += blockDim.x) {
    const int i = base + threadIdx.x;
    const int v = i < n ? count[i] : 0;
    int s = v;
    for (int o = 1; o < 32; o <<= 1) {
      const int t = __shfl_up_sync(0xffffffffu, s, o);
      if (lane >= o) s += t;
    }
    if (lane == 31) wsum[warp] = s;
    __syncthreads();
    if (warp == 0) {
      int w = wsum[lane];
      for (int o = 1; o < 32; o <<= 1) {
        const int t = __shfl_up_sync(0xffffffffu, w, o);
        if (lane >= o) w += t;
      }
      wsum[lane] = w;
    }
    __syncthreads();
    const int excl = carry + (warp ? wsum[warp - 1] : 0) + s - v;
    if (i < n) {
      ptr[i] = excl;
      cursor[i] = excl;
    }
    __syncthreads();
    if (threadIdx.x == 0) carry += wsum[31];
    __syncthreads();
  }
  if (threadIdx.x == 0) ptr[n] = carry;
}

// receivers outside the grid: zero trace, zero residual at levels lo..hi
__global__ void tile2d_skipped_kernel(const int64_t* __restrict__ rec_p, int nrec, int lo, int hi, float* resid,
                                      float* traces, int64_t tr_ld) {
  const int r = blockIdx.x * blockDim.x + threadIdx.x;
  if (r >= nrec || rec_p[r] >= 0) return;
  for (int n = lo; n <= hi; ++n) {
    if (traces) traces[r * tr_ld + n] = 0.f;
    if (resid) resid[(int64_t)n * nrec + r] = 0.f;
  }
}

}  // namespace

cudaError_t launch_tile2d(const Tile2DArgs& a, int physics, int order, cudaStream_t s) {
  if (physics == WAVE_DENSITY) return launch_tile2d_density(a, s);
  switch (order) {
    case 2: return launch_tile2d_o2(a, s);
    case 4: return launch_tile2d_o4(a, s);
    case 6: return launch_tile2d_o6(a, s);
    case 8: return launch_tile2d_o8(a, s);
  }
  return cudaErrorInvalidValue;
}

cudaError_t launch_tile2d_lists(const Tile2DPlan& p, const Geom& g, const int64_t* rec_p, int nrec, int* count,
                                int* ptr, int* cursor, void* ent, cudaStream_t s) {
  if (nrec <= 0) return cudaSuccess;
  const int n = p.nkx * p.nky, blocks = (nrec + 255) / 256;
  cudaError_t e = cudaMemsetAsync(count, 0, n * sizeof(int), s);
  if (e != cudaSuccess) return e;
  tile2d_list_kernel<<<blocks, 256, 0, s>>>(p, g, rec_p, nrec, count, nullptr, nullptr);
  tile2d_scan_kernel<<<1, 1024, 0, s>>>(count, n, ptr, cursor);
  tile2d_list_kernel<<<blocks, 256, 0, s>>>(p, g, rec_p, nrec, nullptr, cursor, static_cast<int2*>(ent));
  count_launch(3);
  return cudaGetLastError();
}

cudaError_t launch_tile2d_skipped(const int64_t* rec_p, int nrec, int lo, int hi, float* resid, float* traces,
                                  int64_t tr_ld, cudaStream_t s) {
  if (nrec <= 0 || lo > hi) return cudaSuccess;
  tile2d_skipped_kernel<<<(nrec + 255) / 256, 256, 0, s>>>(rec_p, nrec, lo, hi, resid, traces, tr_ld);
  count_launch();
  return cudaGetLastError();
}

}  // namespace wave
