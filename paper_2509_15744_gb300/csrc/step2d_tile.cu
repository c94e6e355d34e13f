// 2D velocity form, FP32 storage: several leapfrog steps per launch.
//
// Same arithmetic per cell and step, operation by operation, as
// step2d_velocity_kernel followed by the source / receiver kernel (Eq.
// FDstencil1 in squared-slowness form, the increment and the sources of
// Algorithm 1), so traces, residuals, levels and sensitivities are
// bit-identical.
//
// What bounds a 2D time loop is not the memory: a 2048^2 problem lives in the
// L2, and a 251^2 one is 15 warps' worth of work per step, so a launch per
// step and one per source injection leaves the chip waiting for launches and
// for dependent loads.  Here a CTA takes a region of 128 x RH cells through S
// steps:
//
// * warp w owns RB rows of the region, a lane 4 cells of each row: both time
//   levels, coef and the accumulator stay in registers for all S steps;
// * per step a warp hands its edge rows to its neighbours through shared
//   memory (double buffered, one barrier per step); x neighbours come by
//   shuffle (orders 2 and 4) or from the shared rows (orders 6 and 8);
// * the outer h = r S cells of the region (not at domain edges) lose validity
//   by r cells a step; the CTA writes back only the cells that stay valid, so
//   neighbouring regions overlap by 2 h and no CTA waits on another;
// * regions never leave the domain: the first starts at 0 and the last ends
//   at n, so boundary ghosts are formed from cells at fixed places (the own
//   quad in x, the first / last rows in y);
// * levels go from one pair of buffers to another, since a neighbour still
//   reads the old ones; acc (each cell owned by one CTA) is updated in place.
//
// Sources and receivers inside a region are listed per region once per call
// (count, scan, fill); each step the CTA records its own receivers from the
// shared rows and adds the forces to u^{n-1} in every region that holds the
// cell.
#include "stencil_common.cuh"
#include "step2d_tile.cuh"

namespace wave {
namespace {

constexpr int kSW = kStrip + 8;   // shared row: 4 spare cells each side

__device__ __forceinline__ float4 shfl_up4(const float4& v, int n) {
  float4 r = make_float4(0.f, 0.f, 0.f, 0.f);
  r.w = __shfl_up_sync(0xffffffffu, v.w, 1);
  if (n > 1) r.z = __shfl_up_sync(0xffffffffu, v.z, 1);
  return r;
}
__device__ __forceinline__ float4 shfl_down4(const float4& v, int n) {
  float4 r = make_float4(0.f, 0.f, 0.f, 0.f);
  r.x = __shfl_down_sync(0xffffffffu, v.x, 1);
  if (n > 1) r.y = __shfl_down_sync(0xffffffffu, v.y, 1);
  return r;
}

// Adds a force to a shared cell (cells may repeat) with the rounding of the
// global atomics of the one-step path: the product rounded first, subnormals
// flushed.
__device__ __forceinline__ void add_force(float* p, float v) {
  int* const q = reinterpret_cast<int*>(p);
  int old = *reinterpret_cast<volatile int*>(q), seen;
  do {
    seen = old;
    float sum;
    asm("add.ftz.f32 %0, %1, %2;" : "=f"(sum) : "f"(__int_as_float(seen)), "f"(v));
    old = atomicCAS(q, seen, __float_as_int(sum));
  } while (old != seen);
}

// ACC: 0 none, 1 acc, 2 with compensation; the increment's sign is SGN.
template <int R, int RB, int NW, int ACC, int SGN>
__global__ void __launch_bounds__(NW * 32, 1) tile2d_velocity_kernel(Tile2DArgs a) {
  extern __shared__ __align__(16) float smem[];
  __shared__ uint32_t s_flag[2][4];   // rows of the region with a force / with a receiver to record
  const Tile2DPlan& P = a.plan;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int rh = P.rh, nthreads = blockDim.x;
  float* const share = smem;                       // [2][rh][kSW]: rows of u^n
  float* const force = smem + 2 * rh * kSW;        // [rh][kStrip]: rows of u^{n-1} that take a force
  const int kx = blockIdx.x, ky = blockIdx.y;
  const int nx = (int)a.g.nx, ny = (int)a.g.ny;
  const int xs = tile_start(kx, P.nkx, P.outx, nx, kStrip), ys = tile_start(ky, P.nky, P.outy, ny, rh);
  const int ox0 = tile_own_lo(kx, P.outx, kStrip, P.h), ox1 = tile_own_hi(kx, P.nkx, P.outx, nx, kStrip, P.h);
  const int oy0 = tile_own_lo(ky, P.outy, rh, P.h), oy1 = tile_own_hi(ky, P.nky, P.outy, ny, rh, P.h);
  const int r0 = warp * RB;                        // first region row of the warp
  const int xl = xs + 4 * lane;
  const bool aligned = (xs & 3) == 0;
  const bool left = lane == 0 && xs == 0, right = lane == 31 && xs + kStrip == nx;

  auto ld = [&](const float* p, int64_t off) -> float4 {
    if (aligned) return __ldg(reinterpret_cast<const float4*>(p + off));
    return make_float4(__ldg(p + off), __ldg(p + off + 1), __ldg(p + off + 2), __ldg(p + off + 3));
  };
  const int64_t off0 = (int64_t)(ys + r0) * a.g.px + xl;
  float4 u0[RB], u1[RB], cf[RB], ac[RB], cp[ACC == 2 ? RB : 1];
  const float4 zero4 = make_float4(0.f, 0.f, 0.f, 0.f);
  const bool xown = xl + 4 > ox0 && xl < ox1;      // some cell of the lane's quads is owned
  const bool whole = aligned && xl >= ox0 && xl + 4 <= ox1;
  auto ldown = [&](const float* p, int64_t off) -> float4 {   // owned cells only: a neighbour updates the others
    if (whole) return *reinterpret_cast<const float4*>(p + off);
    return make_float4(xl >= ox0 && xl < ox1 ? p[off] : 0.f, xl + 1 >= ox0 && xl + 1 < ox1 ? p[off + 1] : 0.f,
                       xl + 2 >= ox0 && xl + 2 < ox1 ? p[off + 2] : 0.f, xl + 3 >= ox0 && xl + 3 < ox1 ? p[off + 3] : 0.f);
  };
#pragma unroll
  for (int i = 0; i < RB; ++i) {
    const int64_t off = off0 + i * a.g.px;
    u0[i] = ld(a.prev, off);
    u1[i] = ld(a.cur, off);
    cf[i] = ld(a.coef, off);
    ac[i] = zero4;
    if (ACC == 2) cp[i] = zero4;
    const int y = ys + r0 + i;
    if (ACC && xown && y >= oy0 && y < oy1) {
      ac[i] = ldown(a.acc, off);
      if (ACC == 2) cp[i] = ldown(a.comp, off);
    }
  }

  // ---- the region's sources and receivers ------------------------------------
  const int tile = ky * P.nkx + kx;
  int e0 = 0, ne = 0;
  if (a.nrec > 0 && (a.resid || a.traces || a.resid_in)) {
    e0 = a.tptr[tile];
    ne = a.tptr[tile + 1] - e0;
  }
  const bool src_here = a.wavelet && a.sx >= xs && a.sx < xs + kStrip && a.sy >= ys && a.sy < ys + rh;
  const int src_p = (a.sy - ys) * kStrip + (a.sx - xs);
  if (tid < 8) s_flag[tid >> 2][tid & 3] = 0u;
  for (int i = tid; i < 2 * rh * 8; i += nthreads)   // the spare cells of the shared rows are read, never used: finite
    share[(i >> 3) * kSW + ((i & 7) < 4 ? (i & 7) : kStrip + (i & 7))] = 0.f;
  __syncthreads();
  // A thread keeps its first list entry, its force scale and the next step's
  // residual or datum in registers (most regions hold fewer entries than
  // threads), so no step waits for them; further entries are read each step.
  int2 my = make_int2(0, 0);
  float my_inj = 0.f, my_next = 0.f;
  auto entry_value = [&](const int2& en, int level) -> float {   // residual to inject, or datum to subtract
    if (a.resid_in) return a.resid_in[(int64_t)level * a.nrec + en.y];
    return a.observed && en.x < 0 ? a.observed[en.y * a.obs_ld + level] : 0.f;
  };
  auto entry_inj = [&](const int2& en) -> float {
    const int pos = en.x & 0x3fffffff, row = pos / kStrip, col = pos - row * kStrip;
    return a.coef[(int64_t)(ys + row) * a.g.px + xs + col] * a.h2;
  };
  for (int e = tid; e < ne; e += nthreads) {
    const int2 en = a.tent[e0 + e];
    const int row = (en.x & 0x3fffffff) / kStrip;
    if (e == tid) {
      my = en;
      my_next = entry_value(en, a.level0);
      if (a.resid_in) my_inj = entry_inj(en);
    }
    if (a.resid_in) atomicOr(&s_flag[0][row >> 5], 1u << (row & 31));
    if ((a.resid || a.traces) && en.x < 0) atomicOr(&s_flag[1][row >> 5], 1u << (row & 31));
  }
  const bool src_mine = src_here && tid == nthreads - 1;
  float src_inj = 0.f, src_next = 0.f;
  if (src_mine) {
    src_inj = a.coef[(int64_t)a.sy * a.g.px + a.sx] * a.h2;
    src_next = a.wavelet[a.level0];
  }
  if (src_here && tid == 0) atomicOr(&s_flag[0][(a.sy - ys) >> 5], 1u << ((a.sy - ys) & 31));
  __syncthreads();
  const bool forced = (s_flag[0][0] | s_flag[0][1] | s_flag[0][2] | s_flag[0][3]) != 0u;   // uniform over the CTA
  const uint32_t fmask = (s_flag[0][r0 >> 5] >> (r0 & 31)) & ((1u << RB) - 1u);   // RB divides 32
  const uint32_t gmask = (s_flag[1][r0 >> 5] >> (r0 & 31)) & ((1u << RB) - 1u);
  const float kw = a.resid_in ? (float)(*a.k_dev) * a.weight : 0.f;

  // rows above / below the warp's block: the neighbour's rows, or the mirror
  // rows at a domain edge (Dirichlet: row -1 zero, row -1-j = -row j-1;
  // Neumann: row -1-j = row j); a region edge inside the domain: row 0 / rh-1
  int ru[R], rd[R];
  float su[R], sd[R];
  const bool edge = r0 < R || r0 + RB + R > rh;
#pragma unroll
  for (int j = 1; j <= R; ++j) {
    ru[j - 1] = r0 - j;
    rd[j - 1] = r0 + RB - 1 + j;
    su[j - 1] = sd[j - 1] = 1.f;
    if (ru[j - 1] < 0) {
      const int o = -1 - ru[j - 1];                 // 0-based distance behind the edge
      if (ys != 0) ru[j - 1] = 0;
      else if (a.g.bc == WAVE_NEUMANN) ru[j - 1] = o;
      else { su[j - 1] = o == 0 ? 0.f : -1.f; ru[j - 1] = o == 0 ? 0 : o - 1; }
    }
    if (rd[j - 1] >= rh) {
      const int o = rd[j - 1] - rh;
      if (ys + rh != ny) rd[j - 1] = rh - 1;
      else if (a.g.bc == WAVE_NEUMANN) rd[j - 1] = rh - 1 - o;
      else { sd[j - 1] = o == 0 ? 0.f : -1.f; rd[j - 1] = o == 0 ? rh - 1 : rh - o; }
    }
  }

  auto step = [&](float4 (&c)[RB], float4 (&p)[RB], int s) {   // c = u^n, p: u^{n-1} -> u^{n+1}
    float* const sh = share + (s & 1) * rh * kSW;
#pragma unroll
    for (int i = 0; i < RB; ++i)
      if (R > 2 || i < R || i >= RB - R || ((gmask >> i) & 1u))
        *reinterpret_cast<float4*>(sh + (r0 + i) * kSW + 4 + 4 * lane) = c[i];
    if (fmask) {
#pragma unroll
      for (int i = 0; i < RB; ++i)
        if ((fmask >> i) & 1u) *reinterpret_cast<float4*>(force + (r0 + i) * kStrip + 4 * lane) = p[i];
    }
    __syncthreads();
    const int level = a.level0 + s * a.dlevel;
    auto visit = [&](const int2& en, float v, float inj) {
      const int pos = en.x & 0x3fffffff;
      if (en.x < 0) {   // the region that owns the cell records it
        const int row = pos / kStrip;
        const float u = sh[row * (kSW - kStrip) + 4 + pos];
        if (a.traces) a.traces[en.y * a.tr_ld + level] = u;
        if (a.resid) a.resid[(int64_t)level * a.nrec + en.y] = u - v;
      }
            if (a.resid_in) add_force(force + pos, __fmul_rn(inj, __fmul_rn(kw, v)));
    };
    if (tid < ne) {
      visit(my, my_next, my_inj);
      if (s + 1 < a.nsteps) my_next = entry_value(my, level + a.dlevel);
      for (int e = tid + nthreads; e < ne; e += nthreads) {
        const int2 en = a.tent[e0 + e];
        visit(en, entry_value(en, level), a.resid_in ? entry_inj(en) : 0.f);
      }
    }
    if (src_mine) {
      add_force(force + src_p, __fmul_rn(-src_inj, src_next));
      if (s + 1 < a.nsteps) src_next = a.wavelet[level + a.dlevel];
    }
    if (forced) {
      __syncthreads();
      if (fmask) {
#pragma unroll
        for (int i = 0; i < RB; ++i)
          if ((fmask >> i) & 1u) p[i] = *reinterpret_cast<const float4*>(force + (r0 + i) * kStrip + 4 * lane);
      }
    }
    float4 hu[R], hd[R];
#pragma unroll
    for (int j = 0; j < R; ++j) {
      hu[j] = *reinterpret_cast<const float4*>(sh + ru[j] * kSW + 4 + 4 * lane);
      hd[j] = *reinterpret_cast<const float4*>(sh + rd[j] * kSW + 4 + 4 * lane);
      if (edge) {
        hu[j] = f4_scale(hu[j], su[j]);
        hd[j] = f4_scale(hd[j], sd[j]);
      }
    }
    const bool mass = ACC != 0 && s >= a.mass_lo && s < a.mass_hi;
#pragma unroll
    for (int i = 0; i < RB; ++i) {
      float4 A, C;
      const float4 u = c[i];
      if constexpr (R <= 2) {
        A = shfl_up4(u, R);
        C = shfl_down4(u, R);
      } else {
        A = *reinterpret_cast<const float4*>(sh + (r0 + i) * kSW + 4 * lane);
        C = *reinterpret_cast<const float4*>(sh + (r0 + i) * kSW + 8 + 4 * lane);
      }
      if (left) A = left_ghosts(u, a.g.bc);
      if (right) C = right_ghosts(u, a.g.bc);
      float lap[4];
      x_terms_abc<R>(A, u, C, lap, 2.f * cw<R>(0));
#pragma unroll
      for (int j = 1; j <= R; ++j) {
        const float4& up = i - j >= 0 ? c[i - j >= 0 ? i - j : 0] : hu[i - j < 0 ? j - i - 1 : 0];
        const float4& dn = i + j < RB ? c[i + j < RB ? i + j : 0] : hd[i + j >= RB ? i + j - RB : 0];
        lap[0] = fmaf(cw<R>(j), up.x + dn.x, lap[0]);
        lap[1] = fmaf(cw<R>(j), up.y + dn.y, lap[1]);
        lap[2] = fmaf(cw<R>(j), up.z + dn.z, lap[2]);
        lap[3] = fmaf(cw<R>(j), up.w + dn.w, lap[3]);
      }
      float4 un;
      un.x = fmaf(cf[i].x, lap[0], 2.f * u.x - p[i].x);
      un.y = fmaf(cf[i].y, lap[1], 2.f * u.y - p[i].y);
      un.z = fmaf(cf[i].z, lap[2], 2.f * u.z - p[i].z);
      un.w = fmaf(cf[i].w, lap[3], 2.f * u.w - p[i].w);
      if (mass) {
        const float d0 = un.x - u.x, d1 = un.y - u.y, d2 = un.z - u.z, d3 = un.w - u.w;
        constexpr float sg = (float)SGN;
        if constexpr (ACC == 2) {
          kahan_add(ac[i].x, cp[i].x, sg * d0 * d0);
          kahan_add(ac[i].y, cp[i].y, sg * d1 * d1);
          kahan_add(ac[i].z, cp[i].z, sg * d2 * d2);
          kahan_add(ac[i].w, cp[i].w, sg * d3 * d3);
        } else {
          ac[i].x = fmaf(sg * d0, d0, ac[i].x);
          ac[i].y = fmaf(sg * d1, d1, ac[i].y);
          ac[i].z = fmaf(sg * d2, d2, ac[i].z);
          ac[i].w = fmaf(sg * d3, d3, ac[i].w);
        }
      }
      p[i] = un;
    }
  };

  for (int s = 0; s + 1 < a.nsteps; s += 2) {
    step(u1, u0, s);
    step(u0, u1, s + 1);
  }
  if (a.nsteps & 1) {
    step(u1, u0, a.nsteps - 1);
#pragma unroll
    for (int i = 0; i < RB; ++i) {
      const float4 t = u0[i];
      u0[i] = u1[i];
      u1[i] = t;
    }
  }

  if (!xown) return;
  auto st = [&](float* q, int64_t off, const float4& v) {
    if (whole) {
      *reinterpret_cast<float4*>(q + off) = v;
    } else {
      if (xl >= ox0 && xl < ox1) q[off] = v.x;
      if (xl + 1 >= ox0 && xl + 1 < ox1) q[off + 1] = v.y;
      if (xl + 2 >= ox0 && xl + 2 < ox1) q[off + 2] = v.z;
      if (xl + 3 >= ox0 && xl + 3 < ox1) q[off + 3] = v.w;
    }
  };
#pragma unroll
  for (int i = 0; i < RB; ++i) {
    const int y = ys + r0 + i;
    if (y < oy0 || y >= oy1) continue;
    const int64_t off = off0 + i * a.g.px;
    st(a.oprev, off, u0[i]);
    st(a.ocur, off, u1[i]);
    if (ACC) st(a.acc, off, ac[i]);
    if (ACC == 2) st(a.comp, off, cp[i]);
  }
}

// ---- per-region lists of receivers -------------------------------------------
// A receiver belongs to every region that holds its cell; the region that owns
// the cell has the sign bit set.  count = nullptr in the filling pass.
__global__ void tile2d_list_kernel(Tile2DPlan P, Geom g, const int64_t* __restrict__ rec_p, int nrec,
                                   int* __restrict__ count, int* __restrict__ cursor, int2* __restrict__ ent) {
  const int r = blockIdx.x * blockDim.x + threadIdx.x;
  if (r >= nrec) return;
  const int64_t p = rec_p[r];
  if (p < 0) return;
  const int x = (int)(p % g.px), y = (int)(p / g.px);
  const int nx = (int)g.nx, ny = (int)g.ny;
  for (int ky = max(0, (y - P.rh) / P.outy - 1); ky < P.nky; ++ky) {
    if (ky < P.nky - 1 && ky * P.outy > y) {   // starts below the cell: only the last region may still hold it
      ky = P.nky - 1;
    }
    const int ys = tile_start(ky, P.nky, P.outy, ny, P.rh);
    if (y < ys || y >= ys + P.rh) continue;
    const bool yo = y >= tile_own_lo(ky, P.outy, P.rh, P.h) && y < tile_own_hi(ky, P.nky, P.outy, ny, P.rh, P.h);
    for (int kx = max(0, (x - kStrip) / P.outx - 1); kx < P.nkx; ++kx) {
      if (kx < P.nkx - 1 && kx * P.outx > x) kx = P.nkx - 1;
      const int xs = tile_start(kx, P.nkx, P.outx, nx, kStrip);
      if (x < xs || x >= xs + kStrip) continue;
      const bool xo = x >= tile_own_lo(kx, P.outx, kStrip, P.h) && x < tile_own_hi(kx, P.nkx, P.outx, nx, kStrip, P.h);
      const int t = ky * P.nkx + kx;
      if (count) {
        atomicAdd(count + t, 1);
      } else {
        const int pos = (y - ys) * kStrip + (x - xs);
        ent[atomicAdd(cursor + t, 1)] = make_int2(pos | (yo && xo ? (int)0x80000000 : 0), r);
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

template <int R, int RB, int NW, int ACC, int SGN>
cudaError_t launch_vel(const Tile2DArgs& a, cudaStream_t s) {
  const int bytes = tile2d_smem(a.plan);
  const auto kernel = tile2d_velocity_kernel<R, RB, NW, ACC, SGN>;
  cudaError_t e = set_smem_limit_once(reinterpret_cast<const void*>(kernel), (2 * kSW + kStrip) * 4 * RB * NW);
  if (e != cudaSuccess) return e;
  kernel<<<dim3(a.plan.nkx, a.plan.nky), a.plan.rh / RB * 32, bytes, s>>>(a);
  count_launch();
  e = cudaGetLastError();
  if (e != cudaSuccess) note_error("step kernel launch", e);
  return e;
}

template <int R, int RB, int NW>
cudaError_t launch_vel_acc(const Tile2DArgs& a, cudaStream_t s) {
  if (!a.acc) return launch_vel<R, RB, NW, 0, 1>(a, s);
  if (a.acc_scale > 0.f) return a.comp ? launch_vel<R, RB, NW, 2, 1>(a, s) : launch_vel<R, RB, NW, 1, 1>(a, s);
  return a.comp ? launch_vel<R, RB, NW, 2, -1>(a, s) : launch_vel<R, RB, NW, 1, -1>(a, s);
}

template <int R>
cudaError_t launch_vel_r(const Tile2DArgs& a, cudaStream_t s) {
  switch (a.plan.rb) {
    case 2: return launch_vel_acc<R, 2, 16>(a, s);
    case 4: return launch_vel_acc<R, 4, 16>(a, s);
  }
  return cudaErrorInvalidValue;
}

}  // namespace

int tile2d_smem(const Tile2DPlan& p) { return (2 * kSW + kStrip) * 4 * p.rh; }

cudaError_t launch_tile2d_velocity(const Tile2DArgs& a, int order, cudaStream_t s) {
  switch (order) {
    case 2: return launch_vel_r<1>(a, s);
    case 4: return launch_vel_r<2>(a, s);
    case 6: return launch_vel_r<3>(a, s);
    case 8: return launch_vel_r<4>(a, s);
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
