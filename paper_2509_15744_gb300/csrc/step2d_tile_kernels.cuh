// 2D, FP32 storage: several leapfrog steps per launch (kernels; one
// translation unit per order instantiates them).
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
#pragma once

#include <type_traits>

#include "stencil_common.cuh"
#include "step2d_tile.cuh"

namespace wave {
namespace {

constexpr int kTileWarps = 16;   // of a region, at most
constexpr int kSW = kStrip + 8;   // shared row: 4 spare cells each side
constexpr int kNoForce = 0x7fa5a5a5;   // bits of a force-plane cell without a force (a NaN no force has)

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

// Programmatic dependent launch: the next launch may start where SMs are free,
// and reads what this one wrote only behind its own wait.
__device__ __forceinline__ void let_next_start() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void wait_for_previous() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

// Place of the CTA's region and of the thread's cells in it.
struct Region {
  int xs, ys, ox0, ox1, oy0, oy1;   // first cell; owned cells [ox0, ox1) x [oy0, oy1)
  int xl;                           // first of the lane's 4 cells
  int tile;
  bool aligned, whole, xown;        // 16-byte loads possible; the whole quad / some cell of it is owned
  bool left, right;                 // the quad ends at the domain's edge
  __device__ __forceinline__ Region(const Tile2DArgs& a, int lane) {
    const Tile2DPlan& P = a.plan;
    const int kx = blockIdx.x, ky = blockIdx.y, nx = (int)a.g.nx, ny = (int)a.g.ny;
    xs = tile_start(kx, P.nkx, P.outx, nx, kStrip);
    ys = tile_start(ky, P.nky, P.outy, ny, P.rh);
    ox0 = tile_own_lo(kx, P.outx, kStrip, P.h);
    ox1 = tile_own_hi(kx, P.nkx, P.outx, nx, kStrip, P.h);
    oy0 = tile_own_lo(ky, P.outy, P.rh, P.h);
    oy1 = tile_own_hi(ky, P.nky, P.outy, ny, P.rh, P.h);
    xl = xs + 4 * lane;
    tile = ky * P.nkx + kx;
    aligned = (xs & 3) == 0;
    whole = aligned && xl >= ox0 && xl + 4 <= ox1;
    xown = xl + 4 > ox0 && xl < ox1;
    left = lane == 0 && xs == 0;
    right = lane == 31 && xs + kStrip == nx;
  }
  __device__ __forceinline__ bool own_row(int y) const { return xown && y >= oy0 && y < oy1; }
  // NC: not written by a launch that may still be running
  template <bool NC>
  __device__ __forceinline__ float4 load(const float* p, int64_t off) const {
    if constexpr (NC) {
      if (aligned) return __ldg(reinterpret_cast<const float4*>(p + off));
      return make_float4(__ldg(p + off), __ldg(p + off + 1), __ldg(p + off + 2), __ldg(p + off + 3));
    } else {
      if (aligned) return *reinterpret_cast<const float4*>(p + off);
      return make_float4(p[off], p[off + 1], p[off + 2], p[off + 3]);
    }
  }
  // owned cells only: a neighbour updates the others
  __device__ __forceinline__ float4 load_own(const float* p, int64_t off) const {
    if (whole) return *reinterpret_cast<const float4*>(p + off);
    return make_float4(xl >= ox0 && xl < ox1 ? p[off] : 0.f, xl + 1 >= ox0 && xl + 1 < ox1 ? p[off + 1] : 0.f,
                       xl + 2 >= ox0 && xl + 2 < ox1 ? p[off + 2] : 0.f, xl + 3 >= ox0 && xl + 3 < ox1 ? p[off + 3] : 0.f);
  }
  __device__ __forceinline__ void store_own(float* q, int64_t off, const float4& v) const {
    if (whole) {
      *reinterpret_cast<float4*>(q + off) = v;
    } else {
      if (xl >= ox0 && xl < ox1) q[off] = v.x;
      if (xl + 1 >= ox0 && xl + 1 < ox1) q[off + 1] = v.y;
      if (xl + 2 >= ox0 && xl + 2 < ox1) q[off + 2] = v.z;
      if (xl + 3 >= ox0 && xl + 3 < ox1) q[off + 3] = v.w;
    }
  }
};

// The region's sources and receivers: the list entries, then the source, one
// per thread (most regions hold fewer than threads; the rest are looped over).
//
// Forces of one field whose cells are all different go through two shared
// planes, written a step ahead: a step's force is there when its barrier has
// passed, and the owner adds it to u^{n-1} in registers.  The per-step work of
// a thread is then one multiply-and-store or one record, with the coming value
// loaded a step ahead; what a region with a source costs more per step is 0.1
// us (0.3 with the branches of the general form in every warp).  Cells that
// take more than one force (a receiver twice, or on the source), and two
// fields (whose rows leave no room for the planes), hand the rows of u^{n-1} to
// a shared plane, add there and take them back, behind a second barrier.
template <int RB, int NF>
struct Points {
  int e0, ne;
  int2 my;                 // this thread's entry
  float val;               // its coming value: residual, wavelet sample or datum
  const float* from;       // where `val` came from, and the step to the next
  int stride;
  float m1, m2;            // force = m1 (m2 val)
  int pos;                 // its place in the force plane / the shared rows
  float* out;              // record: where to, and the step to the next
  int ostride;
  int kind;                // 0 none, 1 inject through the planes, 2 record
  float src_inj;
  int src_p;
  bool src_here, src_mine;
  bool forced;             // a force somewhere in the region (uniform over the CTA)
  bool ahead;              // it goes through the planes written a step ahead (uniform)
  uint32_t fmask, gmask;   // rows of the warp that take a force / hold a receiver to record
  float kw[NF];

  __device__ __forceinline__ float value(const Tile2DArgs& a, const int2& en, int level) const {
    if (a.resid_in) return a.resid_in[(int64_t)level * a.nrec + en.y];   // residual to inject
    return a.observed && en.x < 0 ? a.observed[en.y * a.obs_ld + level] : 0.f;   // datum to subtract
  }
  __device__ __forceinline__ float scale(const Tile2DArgs& a, const Region& rg, const int2& en) const {
    const int p = en.x & 0x3fffffff, row = p / kStrip, c = p - row * kStrip;
    return a.coef[(int64_t)(rg.ys + row) * a.g.px + rg.xs + c] * a.h2;
  }
  __device__ __forceinline__ void record(const Tile2DArgs& a, const int2& en, int level, const float* sh) const {
    if (en.x >= 0) return;   // the region that owns the cell records it
    const int p = en.x & 0x3fffffff;
    const float u = sh[p / kStrip * (kSW - kStrip) + 4 + p];
    if (a.traces) a.traces[en.y * a.tr_ld + level] = u;
    if (a.resid) a.resid[(int64_t)level * a.nrec + en.y] = u - value(a, en, level);
  }

  // Contains CTA barriers; s_flag: shared scratch; force: [2][rh][kStrip].
  __device__ __forceinline__ void init(const Tile2DArgs& a, const Region& rg, uint32_t (&s_flag)[3][4], int r0, float* force) {
    const int tid = threadIdx.x, nthreads = blockDim.x;
    e0 = ne = 0;
    if (a.nrec > 0 && (a.resid || a.traces || a.resid_in)) {
      e0 = a.tptr[rg.tile];
      ne = a.tptr[rg.tile + 1] - e0;
    }
    src_here = a.wavelet && a.sx >= rg.xs && a.sx < rg.xs + kStrip && a.sy >= rg.ys && a.sy < rg.ys + a.plan.rh;
    src_p = (a.sy - rg.ys) * kStrip + (a.sx - rg.xs);
    if (tid < 12) s_flag[tid >> 2][tid & 3] = 0u;
    const bool planes = NF == 1 && (src_here || (a.resid_in && ne > 0));
    if (planes) {
      const float none = __int_as_float(kNoForce);
      for (int i = tid; i < 2 * a.plan.rh * (kStrip / 4); i += nthreads)
        *reinterpret_cast<float4*>(force + 4 * i) = make_float4(none, none, none, none);
    }
    __syncthreads();
    auto claim = [&](int p) {   // a cell taken twice: not through the planes
      if (planes && atomicExch(reinterpret_cast<int*>(force) + p, 0) != kNoForce) s_flag[2][0] = 1u;
    };
    my = make_int2(0, 0);
    for (int e = tid; e < ne; e += nthreads) {
      const int2 en = a.tent[e0 + e];
      const int p = en.x & 0x3fffffff, row = p / kStrip;
      if (e == tid) my = en;
      if (a.resid_in) {
        atomicOr(&s_flag[0][row >> 5], 1u << (row & 31));
        claim(p);
      }
      if ((a.resid || a.traces) && en.x < 0) atomicOr(&s_flag[1][row >> 5], 1u << (row & 31));
    }
    src_mine = src_here && tid == min(ne, nthreads - 1);
    src_inj = 0.f;
    if (src_mine) {
      src_inj = a.coef[(int64_t)a.sy * a.g.px + a.sx] * a.h2;
      atomicOr(&s_flag[0][(a.sy - rg.ys) >> 5], 1u << ((a.sy - rg.ys) & 31));
      claim(src_p);
    }
    __syncthreads();
    forced = (s_flag[0][0] | s_flag[0][1] | s_flag[0][2] | s_flag[0][3]) != 0u;
    ahead = planes && s_flag[2][0] == 0u;
    fmask = (s_flag[0][r0 >> 5] >> (r0 & 31)) & ((1u << RB) - 1u);   // RB divides 32
    gmask = (s_flag[1][r0 >> 5] >> (r0 & 31)) & ((1u << RB) - 1u);
#pragma unroll
    for (int f = 0; f < NF; ++f) kw[f] = a.resid_in ? (float)(*a.k_dev) * a.weight[f] : 0.f;

    kind = 0;
    from = nullptr;
    out = nullptr;
    val = m1 = m2 = 0.f;
    stride = ostride = pos = 0;
    if (tid < ne) {
      pos = my.x & 0x3fffffff;
      if (a.resid_in) {
        kind = ahead ? 1 : 0;
        from = a.resid_in + (int64_t)a.level0 * a.nrec + my.y;
        stride = a.dlevel * a.nrec;
        m1 = scale(a, rg, my);
        m2 = kw[0];
        val = *from;
      } else if (my.x < 0 && !(a.traces && a.resid)) {
        kind = 2;
        pos = pos / kStrip * (kSW - kStrip) + 4 + pos;
        out = a.traces ? a.traces + my.y * a.tr_ld + a.level0 : a.resid + (int64_t)a.level0 * a.nrec + my.y;
        ostride = a.traces ? a.dlevel : a.dlevel * a.nrec;
        if (a.resid && a.observed) {
          from = a.observed + my.y * a.obs_ld + a.level0;
          stride = a.dlevel;
          val = *from;
        }
      }
    } else if (src_mine) {
      kind = ahead ? 1 : 0;
      pos = src_p;
      from = a.wavelet + a.level0;
      stride = a.dlevel;
      m1 = -src_inj;
      m2 = 1.f;
      val = *from;
    }
    if (ahead) write_ahead(a, rg, force, 0);   // visible after the first step's barrier
  }
  // Forces of step s into its plane.
  __device__ __forceinline__ void write_ahead(const Tile2DArgs& a, const Region& rg, float* force, int s) {
    float* const pl = force + (s & 1) * a.plan.rh * kStrip;
    if (kind == 1) {
      pl[pos] = __fmul_rn(m1, __fmul_rn(m2, val));
      if (s + 1 < a.nsteps) {
        from += stride;
        val = *from;
      }
    }
    if (ne >= (int)blockDim.x) {   // uniform
      const int level = a.level0 + s * a.dlevel;
      if (a.resid_in) {
        for (int e = threadIdx.x + blockDim.x; e < ne; e += blockDim.x) {
          const int2 en = a.tent[e0 + e];
          pl[en.x & 0x3fffffff] = __fmul_rn(scale(a, rg, en), __fmul_rn(kw[0], value(a, en, level)));
        }
      }
      if (src_mine) pl[src_p] = __fmul_rn(-src_inj, a.wavelet[level]);
    }
  }
  // u^{n-1} of a row that takes a force, in registers.
  __device__ __forceinline__ static void add_ahead(float4& p, const float* row) {
    const float4 v = *reinterpret_cast<const float4*>(row);
    auto add = [](float& q, float w) {
      float sum;   // rounding of the global atomics of the one-step path: subnormals flushed
      asm("add.ftz.f32 %0, %1, %2;" : "=f"(sum) : "f"(q), "f"(w));
      if (__float_as_int(w) != kNoForce) q = sum;
    };
    add(p.x, v.x);
    add(p.y, v.y);
    add(p.z, v.z);
    add(p.w, v.w);
  }
  // Record / inject of step s, behind its barrier: sh = rows of u^n (field 0).
  __device__ __forceinline__ void visit(const Tile2DArgs& a, const Region& rg, const float* sh, float* force, int s) {
    if (kind == 2) {
      *out = sh[pos] - val;
      out += ostride;
      if (from && s + 1 < a.nsteps) {
        from += stride;
        val = *from;
      }
    }
    if (ahead && s + 1 < a.nsteps) write_ahead(a, rg, force, s + 1);
    const bool all = !ahead && forced;   // uniform: the general form of the forces
    if (!all && ne <= (int)blockDim.x && !(a.traces && a.resid)) return;
    const int level = a.level0 + s * a.dlevel, plane = a.plan.rh * kStrip;
    for (int e = threadIdx.x; e < ne; e += blockDim.x) {
      const int2 en = a.tent[e0 + e];
      if (!a.resid_in) {
        if (e >= (int)blockDim.x || kind != 2) record(a, en, level, sh);
      } else if (all) {
        const float er = value(a, en, level), inj = scale(a, rg, en);
#pragma unroll
        for (int f = 0; f < NF; ++f)
          if (NF == 1 || ((a.rec_fields >> f) & 1))
            add_force(force + f * plane + (en.x & 0x3fffffff), __fmul_rn(inj, __fmul_rn(kw[f], er)));
      }
    }
    if (all && src_mine) {
#pragma unroll
      for (int f = 0; f < NF; ++f)
        if (NF == 1 || ((a.src_fields >> f) & 1)) add_force(force + f * plane + src_p, __fmul_rn(-src_inj, a.wavelet[level]));
    }
  }
};

// Rows above / below a warp's block of RB rows: the neighbour's rows, or the
// mirror rows at a domain edge (Dirichlet: row -1 zero, row -1-j = -row j-1;
// Neumann: row -1-j = row j); at a region edge inside the domain row 0 / rh-1
// (those cells are not valid any more).
template <int R>
struct EdgeRows {
  int up[R], dn[R];
  float su[R], sd[R];
  bool edge;
  __device__ __forceinline__ EdgeRows(const Tile2DArgs& a, const Region& rg, int r0, int RB) {
    const int rh = a.plan.rh;
    edge = r0 < R || r0 + RB + R > rh;
#pragma unroll
    for (int j = 1; j <= R; ++j) {
      up[j - 1] = r0 - j;
      dn[j - 1] = r0 + RB - 1 + j;
      su[j - 1] = sd[j - 1] = 1.f;
      if (up[j - 1] < 0) {
        const int o = -1 - up[j - 1];                 // 0-based distance behind the edge
        if (rg.ys != 0) up[j - 1] = 0;
        else if (a.g.bc == WAVE_NEUMANN) up[j - 1] = o;
        else { su[j - 1] = o == 0 ? 0.f : -1.f; up[j - 1] = o == 0 ? 0 : o - 1; }
      }
      if (dn[j - 1] >= rh) {
        const int o = dn[j - 1] - rh;
        if (rg.ys + rh != (int)a.g.ny) dn[j - 1] = rh - 1;
        else if (a.g.bc == WAVE_NEUMANN) dn[j - 1] = rh - 1 - o;
        else { sd[j - 1] = o == 0 ? 0.f : -1.f; dn[j - 1] = o == 0 ? rh - 1 : rh - o; }
      }
    }
  }
  __device__ __forceinline__ void load(const float* sh, int lane, float4 (&hu)[R], float4 (&hd)[R]) const {
#pragma unroll
    for (int j = 0; j < R; ++j) {
      hu[j] = *reinterpret_cast<const float4*>(sh + up[j] * kSW + 4 + 4 * lane);
      hd[j] = *reinterpret_cast<const float4*>(sh + dn[j] * kSW + 4 + 4 * lane);
      if (edge) {
        hu[j] = f4_scale(hu[j], su[j]);
        hd[j] = f4_scale(hd[j], sd[j]);
      }
    }
  }
};

// The spare cells of the shared rows are read, never used: finite.
__device__ __forceinline__ void clear_spare(float* share, int rows) {
  for (int i = threadIdx.x; i < rows * 8; i += blockDim.x)
    share[(i >> 3) * kSW + ((i & 7) < 4 ? (i & 7) : kStrip + (i & 7))] = 0.f;
}

// New level of 4 cells of row i: c = u^n, p = u^{n-1}, hu / hd the rows beyond the block.
template <int R, int RB>
__device__ __forceinline__ float4 velocity_row(int i, const float4 (&c)[RB], const float4& p, const float4& cf,
                                               const float4 (&hu)[R], const float4 (&hd)[R], const float* srow,
                                               int lane, const Region& rg, int bc) {
  float4 A, C;
  const float4 u = c[i];
  if constexpr (R <= 2) {
    A = shfl_up4(u, R);
    C = shfl_down4(u, R);
  } else {
    A = *reinterpret_cast<const float4*>(srow + 4 * lane);
    C = *reinterpret_cast<const float4*>(srow + 8 + 4 * lane);
  }
  if (rg.left) A = left_ghosts(u, bc);
  if (rg.right) C = right_ghosts(u, bc);
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
  return make_float4(fmaf(cf.x, lap[0], 2.f * u.x - p.x), fmaf(cf.y, lap[1], 2.f * u.y - p.y),
                     fmaf(cf.z, lap[2], 2.f * u.z - p.z), fmaf(cf.w, lap[3], 2.f * u.w - p.w));
}

// acc += sg (un - u)^2
__device__ __forceinline__ void add_square(float sg, const float4& un, const float4& u, float4& ac) {
  const float d0 = un.x - u.x, d1 = un.y - u.y, d2 = un.z - u.z, d3 = un.w - u.w;
  ac.x = fmaf(sg * d0, d0, ac.x);
  ac.y = fmaf(sg * d1, d1, ac.y);
  ac.z = fmaf(sg * d2, d2, ac.z);
  ac.w = fmaf(sg * d3, d3, ac.w);
}
__device__ __forceinline__ void add_square_kahan(float sg, const float4& un, const float4& u, float4& ac, float4& cp) {
  const float d0 = un.x - u.x, d1 = un.y - u.y, d2 = un.z - u.z, d3 = un.w - u.w;
  kahan_add(ac.x, cp.x, sg * d0 * d0);
  kahan_add(ac.y, cp.y, sg * d1 * d1);
  kahan_add(ac.z, cp.z, sg * d2 * d2);
  kahan_add(ac.w, cp.w, sg * d3 * d3);
}

// One field.  ACC: 0 none, 1 acc, 2 with compensation; the increment's sign is SGN.
template <int R, int RB, int ACC, int SGN>
__global__ void __launch_bounds__(kTileWarps * 32, 1) tile2d_velocity_kernel(Tile2DArgs a) {
  extern __shared__ __align__(16) float smem[];
  __shared__ uint32_t s_flag[3][4];   // rows of the region with a force, with a receiver to record; [2][0]: cells taken twice
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int rh = a.plan.rh;
  float* const share = smem;                       // [2][rh][kSW]: rows of u^n
  float* const force = smem + 2 * rh * kSW;        // [2][rh][kStrip]: forces, or rows of u^{n-1} that take them
  const Region rg(a, lane);
  const int r0 = warp * RB;                        // first region row of the warp
  const int64_t off0 = (int64_t)(rg.ys + r0) * a.g.px + rg.xl;
  float4 u0[RB], u1[RB], cf[RB], ac[RB], cp[ACC == 2 ? RB : 1];
  auto load_levels = [&](auto nc) {
#pragma unroll
    for (int i = 0; i < RB; ++i) {
      const int64_t off = off0 + i * a.g.px;
      u0[i] = rg.load<nc>(a.prev[0], off);
      u1[i] = rg.load<nc>(a.cur[0], off);
      ac[i] = make_float4(0.f, 0.f, 0.f, 0.f);
      if (ACC == 2) cp[i] = ac[i];
      if (ACC && rg.own_row(rg.ys + r0 + i)) {
        ac[i] = rg.load_own(a.acc, off);
        if (ACC == 2) cp[i] = rg.load_own(a.comp, off);
      }
    }
  };
  let_next_start();
  if (!a.overlap) load_levels(std::true_type());
#pragma unroll
  for (int i = 0; i < RB; ++i) cf[i] = rg.load<true>(a.coef, off0 + i * a.g.px);
  if (R > 2) clear_spare(share, 2 * rh);
  Points<RB, 1> pts;
  pts.init(a, rg, s_flag, r0, force);
  if (a.overlap) {   // the coefficients and lists do not depend on the launch before, the levels do
    wait_for_previous();
    load_levels(std::false_type());
  }
  const EdgeRows<R> er(a, rg, r0, RB);

  // c = u^n, p: u^{n-1} -> u^{n+1}; lists: the region holds a source or receiver
  auto step = [&](float4 (&c)[RB], float4 (&p)[RB], int s, auto lists) {
    float* const sh = share + (s & 1) * rh * kSW;
#pragma unroll
    for (int i = 0; i < RB; ++i) {
      if (R > 2 || i < R || i >= RB - R || (lists && ((pts.gmask >> i) & 1u)))
        *reinterpret_cast<float4*>(sh + (r0 + i) * kSW + 4 + 4 * lane) = c[i];
      if (lists && !pts.ahead && ((pts.fmask >> i) & 1u))
        *reinterpret_cast<float4*>(force + (r0 + i) * kStrip + 4 * lane) = p[i];
    }
    __syncthreads();
    if (lists) pts.visit(a, rg, sh, force, s);
    if (lists && pts.forced) {
      if (!pts.ahead) __syncthreads();
      const float* const fr = force + (pts.ahead ? (s & 1) * rh * kStrip : 0) + r0 * kStrip + 4 * lane;
#pragma unroll
      for (int i = 0; i < RB; ++i)
        if ((pts.fmask >> i) & 1u) {
          if (pts.ahead) pts.add_ahead(p[i], fr + i * kStrip);
          else p[i] = *reinterpret_cast<const float4*>(fr + i * kStrip);
        }
    }
    float4 hu[R], hd[R];
    er.load(sh, lane, hu, hd);
    const bool mass = ACC != 0 && s >= a.mass_lo && s < a.mass_hi;
#pragma unroll
    for (int i = 0; i < RB; ++i) {
      const float4 un = velocity_row<R, RB>(i, c, p[i], cf[i], hu, hd, sh + (r0 + i) * kSW, lane, rg, a.g.bc);
      if (mass) {
        if constexpr (ACC == 2) add_square_kahan((float)SGN, un, c[i], ac[i], cp[i]);
        else add_square((float)SGN, un, c[i], ac[i]);
      }
      p[i] = un;
    }
  };
  const bool odd = a.nsteps & 1;
  auto steps = [&](auto lists) {
    for (int s = 0; s + 1 < a.nsteps; s += 2) {
      step(u1, u0, s, lists);
      step(u0, u1, s + 1, lists);
    }
    if (odd) step(u1, u0, a.nsteps - 1, lists);
  };
  // most regions of a large grid hold neither: a loop without that code
  if (pts.ne > 0 || pts.src_here) steps(std::true_type());
  else steps(std::false_type());

#pragma unroll
  for (int i = 0; i < RB; ++i) {
    if (!rg.own_row(rg.ys + r0 + i)) continue;
    const int64_t off = off0 + i * a.g.px;
    rg.store_own(odd ? a.ocur[0] : a.oprev[0], off, u0[i]);
    rg.store_own(odd ? a.oprev[0] : a.ocur[0], off, u1[i]);
    if (ACC) rg.store_own(a.acc, off, ac[i]);
    if (ACC == 2) rg.store_own(a.comp, off, cp[i]);
  }
}

// ---- coefficients and accumulator in tensor memory ------------------------------
// Two fields (the +-k pair, or u and lambda of the reverse-time mode), or the
// density form with its six face weights per cell, hold more than registers
// take.  The tensor memory of the SM (128 lanes x 512 columns of 32 bits, used
// by no tile of this kernel otherwise) keeps, per thread, 4 columns per row
// and quantity: what a row needs is read when the row is computed, the
// accumulator written back.  16 warps share 4 lane quarters, so a warp has 128
// columns: RB = 4 rows of 32.
__device__ __forceinline__ void tm_ld4(uint32_t ta, float4& v) {
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0, %1, %2, %3}, [%4];"
               : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "r"(ta) : "memory");
}
__device__ __forceinline__ void tm_st4(uint32_t ta, const float4& v) {
  asm volatile("tcgen05.st.sync.aligned.32x32b.x4.b32 [%0], {%1, %2, %3, %4};"
               :: "r"(ta), "f"(v.x), "f"(v.y), "f"(v.z), "f"(v.w) : "memory");
}
__device__ __forceinline__ void tm_wait_st() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }
// wait for the loads; the registers pass through so that no use moves above it
__device__ __forceinline__ void tm_use(float4& v) {
  asm volatile("" : "+f"(v.x), "+f"(v.y), "+f"(v.z), "+f"(v.w) :: "memory");
}
__device__ __forceinline__ void tm_wait_ld() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }

// Flux and squared-difference weights of a face seen from cell i (harmonic
// mean of b, and its derivative with respect to b_i), as face() of the
// one-step density kernel.
__device__ __forceinline__ float face_flux(float bi, float bj) { return 2.f * bi * bj / (bi + bj); }
__device__ __forceinline__ float face_grad(float bi, float bj) {
  const float sum = bi + bj;
  return 2.f * bj * bj / (sum * sum);
}

// ACC: 0 none, 1 acc, 2 with compensation, 3 the mixed term of the exact
// reverse-time mode (fields u, lambda).  With two fields of modes 1 and 2 the
// increments have the signs -1 (field 0) and +1 (field 1); with one it is a.acc_scale.
template <int R, bool DEN, int NF, int ACC>
__global__ void __launch_bounds__(512, 1) tile2d_tmem_kernel(Tile2DArgs a) {
  constexpr int RB = 4;
  constexpr int kCols = DEN ? 128 : (ACC == 2 ? 48 : 32);   // columns of a warp
  constexpr uint32_t kAlloc = DEN ? 512u : (ACC == 2 ? 256u : 128u);
  // column of a quantity within a row's group: quantities q of row i at (q RB + i) 4
  enum { kCoef = 0, kAcc = 1, kComp = 2, kFx = 2, kFy = 3, kGxm = 4, kGxp = 5, kGym = 6, kGyp = 7 };
  extern __shared__ __align__(16) float smem[];
  __shared__ uint32_t s_flag[3][4];
  __shared__ uint32_t s_tm;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int rh = a.plan.rh;
  float* const share = smem;                             // [NF][2][rh][kSW]: rows of u^n
  float* const force = smem + NF * 2 * rh * kSW;         // [2][rh][kStrip]: forces, or rows of u^{n-1} per field
  if (warp == 0) {
    const uint32_t sa = (uint32_t)__cvta_generic_to_shared(&s_tm);
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(sa), "r"(kAlloc) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  const Region rg(a, lane);
  const int r0 = warp * RB;
  const int64_t off0 = (int64_t)(rg.ys + r0) * a.g.px + rg.xl;
  float4 u0[NF][RB], u1[NF][RB], cp[DEN && ACC == 2 ? RB : 1];
  auto load_levels = [&](auto nc) {
#pragma unroll
    for (int f = 0; f < NF; ++f)
#pragma unroll
      for (int i = 0; i < RB; ++i) {
        u0[f][i] = rg.load<nc>(a.prev[f], off0 + i * a.g.px);
        u1[f][i] = rg.load<nc>(a.cur[f], off0 + i * a.g.px);
      }
  };
  if (!a.overlap) load_levels(std::true_type());
  if (R > 2) clear_spare(share, NF * 2 * rh);
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  Points<RB, NF> pts;
  pts.init(a, rg, s_flag, r0, force);   // CTA barriers: the allocation is visible after them
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  // Only now, when every CTA of this launch holds its tensor memory, may the
  // next launch start.  Its CTAs allocate before they wait for this launch: on
  // an SM that CTAs of several launches share (regions of few rows), one that
  // came before a CTA of this launch had its columns could take them and wait
  // for the CTA that then never gets any.  This way what a CTA waits for,
  // columns or a launch, is always held or run by CTAs that have their columns.
  let_next_start();
  const uint32_t tm_base = s_tm;
  const uint32_t tm = tm_base + ((uint32_t)(32 * (warp & 3)) << 16) + (uint32_t)((warp >> 2) * kCols);
  auto col = [&](int q, int i) -> uint32_t { return tm + (uint32_t)((q * RB + i) * 4); };
  // density: flux weights of the faces above the block, and of the face left
  // of the quad in each of the 4 rows (per thread, in shared memory)
  float4* const bedge = reinterpret_cast<float4*>(smem + (2 * NF * kSW + 2 * kStrip) * rh) + 2 * threadIdx.x;
  {
    auto brow = [&](int y) -> float4 {   // ghost material = boundary material
      y = min(max(y, 0), (int)a.g.ny - 1);
      return rg.load<true>(a.bmat, (int64_t)y * a.g.px + rg.xl);
    };
    float4 bm, bc, bp;
    if constexpr (DEN) {
      bm = brow(rg.ys + r0 - 1);
      bc = brow(rg.ys + r0);
      bedge[0] = make_float4(face_flux(bc.x, bm.x), face_flux(bc.y, bm.y), face_flux(bc.z, bm.z), face_flux(bc.w, bm.w));
    }
#pragma unroll
    for (int i = 0; i < RB; ++i) {
      const int64_t off = off0 + i * a.g.px;
      const int y = rg.ys + r0 + i;
      tm_st4(col(kCoef, i), rg.load<true>(a.coef, off));
      if constexpr (DEN) {
        bp = brow(y + 1);
        float bl = __shfl_up_sync(0xffffffffu, bc.w, 1), br = __shfl_down_sync(0xffffffffu, bc.x, 1);
        if (lane == 0) bl = bc.x;
        if (lane == 31) br = bc.w;
        (&bedge[1].x)[i] = face_flux(bc.x, bl);
        tm_st4(col(kFx, i), make_float4(face_flux(bc.x, bc.y), face_flux(bc.y, bc.z), face_flux(bc.z, bc.w), face_flux(bc.w, br)));
        tm_st4(col(kFy, i), make_float4(face_flux(bc.x, bp.x), face_flux(bc.y, bp.y), face_flux(bc.z, bp.z), face_flux(bc.w, bp.w)));
        if constexpr (ACC != 0) {
          const bool dir = a.g.bc == WAVE_DIRICHLET;   // a Dirichlet ghost's material follows its cell
          float4 gxm = make_float4(face_grad(bc.x, bl), face_grad(bc.y, bc.x), face_grad(bc.z, bc.y), face_grad(bc.w, bc.z));
          float4 gxp = make_float4(face_grad(bc.x, bc.y), face_grad(bc.y, bc.z), face_grad(bc.z, bc.w), face_grad(bc.w, br));
          float4 gym = make_float4(face_grad(bc.x, bm.x), face_grad(bc.y, bm.y), face_grad(bc.z, bm.z), face_grad(bc.w, bm.w));
          float4 gyp = make_float4(face_grad(bc.x, bp.x), face_grad(bc.y, bp.y), face_grad(bc.z, bp.z), face_grad(bc.w, bp.w));
          if (dir && rg.left) gxm.x = 1.f;
          if (dir && rg.right) gxp.w = 1.f;
          if (dir && y == 0) gym = make_float4(1.f, 1.f, 1.f, 1.f);
          if (dir && y == (int)a.g.ny - 1) gyp = make_float4(1.f, 1.f, 1.f, 1.f);
          tm_st4(col(kGxm, i), gxm);
          tm_st4(col(kGxp, i), gxp);
          tm_st4(col(kGym, i), gym);
          tm_st4(col(kGyp, i), gyp);
        }
        bm = bc;
        bc = bp;
      }
    }
  }
  if (a.overlap) {   // the weights and lists do not depend on the launch before, the levels and acc do
    wait_for_previous();
    load_levels(std::false_type());
  }
  if constexpr (ACC != 0) {
#pragma unroll
    for (int i = 0; i < RB; ++i) {
      const int64_t off = off0 + i * a.g.px;
      const bool own = rg.own_row(rg.ys + r0 + i);
      const float4 zero4 = make_float4(0.f, 0.f, 0.f, 0.f);
      tm_st4(col(kAcc, i), own ? rg.load_own(a.acc, off) : zero4);
      if (ACC == 2) {
        const float4 v = own ? rg.load_own(a.comp, off) : zero4;
        if constexpr (DEN) cp[i] = v;
        else tm_st4(col(kComp, i), v);
      }
    }
  }
  tm_wait_st();
  const EdgeRows<R> er(a, rg, r0, RB);

  // plain_q: the quad's element whose x pair the one-step kernel adds unfused (x mod 4 = 3)
  auto step = [&](float4 (&c)[NF][RB], float4 (&p)[NF][RB], int s, auto plain_q, auto lists) {
#pragma unroll
    for (int f = 0; f < NF; ++f) {
      float* const sh = share + (2 * f + (s & 1)) * rh * kSW;
#pragma unroll
      for (int i = 0; i < RB; ++i) {
        if (R > 2 || i < R || i >= RB - R || (lists && f == 0 && ((pts.gmask >> i) & 1u)))
          *reinterpret_cast<float4*>(sh + (r0 + i) * kSW + 4 + 4 * lane) = c[f][i];
        if (lists && !pts.ahead && ((pts.fmask >> i) & 1u))
          *reinterpret_cast<float4*>(force + (f * rh + r0 + i) * kStrip + 4 * lane) = p[f][i];
      }
    }
    __syncthreads();
    if (lists) pts.visit(a, rg, share + (s & 1) * rh * kSW, force, s);
    if (lists && pts.forced) {
      if (!pts.ahead) __syncthreads();
#pragma unroll
      for (int f = 0; f < NF; ++f)
#pragma unroll
        for (int i = 0; i < RB; ++i)
          if ((pts.fmask >> i) & 1u) {
            if (NF == 1 && pts.ahead) pts.add_ahead(p[f][i], force + ((s & 1) * rh + r0 + i) * kStrip + 4 * lane);
            else p[f][i] = *reinterpret_cast<const float4*>(force + (f * rh + r0 + i) * kStrip + 4 * lane);
          }
    }
    const bool mass = ACC != 0 && s >= a.mass_lo && s < a.mass_hi;
    const bool stiff = DEN && ACC != 0 && s >= a.stiff_lo && s < a.stiff_hi;
#pragma unroll
    for (int f = 0; f < NF; ++f) {
      const float sg = NF == 2 ? (f == 0 ? -1.f : 1.f) : a.acc_scale;
      const float* const sh = share + (2 * f + (s & 1)) * rh * kSW;
      if constexpr (!DEN) {
        float4 hu[R], hd[R];
        er.load(sh, lane, hu, hd);
#pragma unroll
        for (int i = 0; i < RB; ++i) {
          float4 cf, ac, cpv;
          const bool inc = mass && (ACC != 3 || f == 1);
          tm_ld4(col(kCoef, i), cf);
          if (inc) tm_ld4(col(kAcc, i), ac);
          if (ACC == 2 && inc) tm_ld4(col(kComp, i), cpv);
          tm_wait_ld();
          tm_use(cf);
          if (inc) tm_use(ac);
          if (ACC == 2 && inc) tm_use(cpv);
          const float4 un = velocity_row<R, RB>(i, c[f], p[f][i], cf, hu, hd, sh + (r0 + i) * kSW, lane, rg, a.g.bc);
          if (inc) {
            if constexpr (ACC == 3) {   // acc -= (lambda - lambda_new)(u - u_new)
              const float4 u = c[0][i], v = p[0][i], l = c[NF - 1][i];
              ac.x = fmaf(-(l.x - un.x), u.x - v.x, ac.x);
              ac.y = fmaf(-(l.y - un.y), u.y - v.y, ac.y);
              ac.z = fmaf(-(l.z - un.z), u.z - v.z, ac.z);
              ac.w = fmaf(-(l.w - un.w), u.w - v.w, ac.w);
            } else if constexpr (ACC == 2) {
              add_square_kahan(sg, un, c[f][i], ac, cpv);
              tm_st4(col(kComp, i), cpv);
            } else {
              add_square(sg, un, c[f][i], ac);
            }
            tm_st4(col(kAcc, i), ac);
          }
          p[f][i] = un;
        }
        if (mass) tm_wait_st();
      } else {
        // in two parts per row, the update first, to hold few weights at a time
        float4 by = bedge[0];                                // flux weights and differences of the faces above
        float4 hrow = *reinterpret_cast<const float4*>(sh + er.up[0] * kSW + 4 + 4 * lane);
        if (er.edge) hrow = f4_scale(hrow, er.su[0]);
        float4 dy = make_float4(c[f][0].x - hrow.x, c[f][0].y - hrow.y, c[f][0].z - hrow.z, c[f][0].w - hrow.w);
#pragma unroll
        for (int i = 0; i < RB; ++i) {
          float4 cf, fx, fy;
          tm_ld4(col(kCoef, i), cf);
          tm_ld4(col(kFx, i), fx);
          tm_ld4(col(kFy, i), fy);
          const float4 u = c[f][i];
          float ul = __shfl_up_sync(0xffffffffu, u.w, 1), ur = __shfl_down_sync(0xffffffffu, u.x, 1);
          if (rg.left) ul = a.g.bc == WAVE_NEUMANN ? u.x : 0.f;
          if (rg.right) ur = a.g.bc == WAVE_NEUMANN ? u.w : 0.f;
          float4 below;
          if (i + 1 < RB) {
            below = c[f][i + 1 < RB ? i + 1 : 0];
          } else {
            below = *reinterpret_cast<const float4*>(sh + er.dn[0] * kSW + 4 + 4 * lane);
            if (er.edge) below = f4_scale(below, er.sd[0]);
          }
          const float dx[5] = {u.x - ul, u.y - u.x, u.z - u.y, u.w - u.z, ur - u.w};   // u_{x} - u_{x-1}
          const float dm[4] = {dy.x, dy.y, dy.z, dy.w};                                  // u_y - u_{y-1}
          const float dp[4] = {below.x - u.x, below.y - u.y, below.z - u.z, below.w - u.w};
          const float bxl = (&bedge[1].x)[i];
          tm_wait_ld();
          tm_use(cf);
          tm_use(fx);
          tm_use(fy);
          const float bx[5] = {bxl, fx.x, fx.y, fx.z, fx.w};
          const float bym[4] = {by.x, by.y, by.z, by.w}, byp[4] = {fy.x, fy.y, fy.z, fy.w};
          float flux[4];
#pragma unroll
          for (int q = 0; q < 4; ++q) {
            // rounding of the one-step kernel, as compiled: the lower face's
            // product rounded, the upper one fused onto it (not in the x pair
            // of cells with x mod 4 = 3)
            const float mx = __fmul_rn(bx[q], dx[q]), my = __fmul_rn(bym[q], dm[q]);
            const float fxs = q != plain_q ? fmaf(bx[q + 1], dx[q + 1], -mx) : __fsub_rn(__fmul_rn(bx[q + 1], dx[q + 1]), mx);
            const float fys = fmaf(byp[q], dp[q], -my);
            flux[q] = __fadd_rn(fxs, fys);
          }
          float4 un;
          un.x = fmaf(cf.x, flux[0], 2.f * u.x - p[f][i].x);
          un.y = fmaf(cf.y, flux[1], 2.f * u.y - p[f][i].y);
          un.z = fmaf(cf.z, flux[2], 2.f * u.z - p[f][i].z);
          un.w = fmaf(cf.w, flux[3], 2.f * u.w - p[f][i].w);
          p[f][i] = un;
          if (mass) {
            float4 ac;
            float g[4] = {0.f, 0.f, 0.f, 0.f};
            tm_ld4(col(kAcc, i), ac);
            if (stiff) {
              float4 wm, wp;
              tm_ld4(col(kGxm, i), wm);
              tm_ld4(col(kGxp, i), wp);
              tm_wait_ld();
              tm_use(wm);
              tm_use(wp);
              const float gm[4] = {wm.x, wm.y, wm.z, wm.w}, gp[4] = {wp.x, wp.y, wp.z, wp.w};
#pragma unroll
              for (int q = 0; q < 4; ++q) {
                const float lo = __fmul_rn(__fmul_rn(gm[q], dx[q]), dx[q]), hi = __fmul_rn(gp[q], dx[q + 1]);
                g[q] = q != plain_q ? fmaf(hi, dx[q + 1], lo) : __fadd_rn(__fmul_rn(hi, dx[q + 1]), lo);
              }
              tm_ld4(col(kGym, i), wm);
              tm_ld4(col(kGyp, i), wp);
              tm_wait_ld();
              tm_use(wm);
              tm_use(wp);
              const float hm[4] = {wm.x, wm.y, wm.z, wm.w}, hp[4] = {wp.x, wp.y, wp.z, wp.w};
#pragma unroll
              for (int q = 0; q < 4; ++q)
                g[q] = __fadd_rn(g[q], fmaf(__fmul_rn(hp[q], dp[q]), dp[q], __fmul_rn(__fmul_rn(hm[q], dm[q]), dm[q])));
            } else {
              tm_wait_ld();
            }
            tm_use(ac);
            const float d[4] = {un.x - u.x, un.y - u.y, un.z - u.z, un.w - u.w};
            float v[4];
#pragma unroll
            for (int q = 0; q < 4; ++q) {
              v[q] = __fmul_rn(__fmul_rn(a.da, d[q]), d[q]);
              if (stiff) v[q] = fmaf(-a.dbs, g[q], v[q]);
            }
            if constexpr (ACC == 2) {
              kahan_add(ac.x, cp[i].x, sg * v[0]);
              kahan_add(ac.y, cp[i].y, sg * v[1]);
              kahan_add(ac.z, cp[i].z, sg * v[2]);
              kahan_add(ac.w, cp[i].w, sg * v[3]);
            } else {
              ac.x = fmaf(sg, v[0], ac.x);
              ac.y = fmaf(sg, v[1], ac.y);
              ac.z = fmaf(sg, v[2], ac.z);
              ac.w = fmaf(sg, v[3], ac.w);
            }
            tm_st4(col(kAcc, i), ac);
          }
          by = fy;
          dy = make_float4(dp[0], dp[1], dp[2], dp[3]);
        }
        if (mass) tm_wait_st();
      }
    }
  };
  const bool odd = a.nsteps & 1;
  auto steps = [&](auto plain_q, auto lists) {
    for (int s = 0; s + 1 < a.nsteps; s += 2) {
      step(u1, u0, s, plain_q, lists);
      step(u0, u1, s + 1, plain_q, lists);
    }
    if (odd) step(u1, u0, a.nsteps - 1, plain_q, lists);
  };
  if (DEN && !rg.aligned) steps(3 - (rg.xs & 3), std::true_type());
  else if (pts.ne > 0 || pts.src_here) steps(std::integral_constant<int, 3>(), std::true_type());
  else steps(std::integral_constant<int, 3>(), std::false_type());

#pragma unroll
  for (int i = 0; i < RB; ++i) {
    float4 ac, cpv;
    if constexpr (ACC != 0) {   // warp-wide loads, whatever the lanes own
      tm_ld4(col(kAcc, i), ac);
      if (ACC == 2 && !DEN) tm_ld4(col(kComp, i), cpv);
      tm_wait_ld();
      tm_use(ac);
      if (ACC == 2 && !DEN) tm_use(cpv);
      if (ACC == 2 && DEN) cpv = cp[i];
    }
    if (!rg.own_row(rg.ys + r0 + i)) continue;
    const int64_t off = off0 + i * a.g.px;
#pragma unroll
    for (int f = 0; f < NF; ++f) {
      rg.store_own(odd ? a.ocur[f] : a.oprev[f], off, u0[f][i]);
      rg.store_own(odd ? a.oprev[f] : a.ocur[f], off, u1[f][i]);
    }
    if (ACC) rg.store_own(a.acc, off, ac);
    if (ACC == 2) rg.store_own(a.comp, off, cpv);
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  if (warp == 0) {
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tm_base), "r"(kAlloc) : "memory");
  }
}

template <typename K>
cudaError_t launch_tile(K kernel, int rb, const Tile2DArgs& a, cudaStream_t s, int per_thread = 0) {
  // shared bytes per region row: rows of both levels, force rows, per-thread data
  const int row = (2 * a.nfields * kSW + 2 * kStrip) * 4 + per_thread * 32 / rb;
  cudaError_t e = set_smem_limit_once(reinterpret_cast<const void*>(kernel), row * rb * kTileWarps);
  if (e != cudaSuccess) return e;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(a.plan.nkx, a.plan.nky);
  cfg.blockDim = dim3(a.plan.rh / rb * 32);
  cfg.dynamicSmemBytes = row * a.plan.rh;
  cfg.stream = s;
  cudaLaunchAttribute attr = {};
  attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr.val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = &attr;
  cfg.numAttrs = a.overlap ? 1 : 0;
  e = cudaLaunchKernelEx(&cfg, kernel, a);
  count_launch();
  if (e == cudaSuccess) e = cudaGetLastError();
  if (e != cudaSuccess) note_error("step kernel launch", e);
  return e;
}

template <int R, int RB>
cudaError_t launch_vel(const Tile2DArgs& a, cudaStream_t s) {
  if (!a.acc) return launch_tile(tile2d_velocity_kernel<R, RB, 0, 1>, RB, a, s);
  if (a.acc_scale > 0.f)
    return a.comp ? launch_tile(tile2d_velocity_kernel<R, RB, 2, 1>, RB, a, s)
                  : launch_tile(tile2d_velocity_kernel<R, RB, 1, 1>, RB, a, s);
  return a.comp ? launch_tile(tile2d_velocity_kernel<R, RB, 2, -1>, RB, a, s)
                : launch_tile(tile2d_velocity_kernel<R, RB, 1, -1>, RB, a, s);
}

template <int R>
cudaError_t launch_vel_r(const Tile2DArgs& a, cudaStream_t s) {
  if (a.nfields == 1) return a.plan.rb == 2 ? launch_vel<R, 2>(a, s) : launch_vel<R, 4>(a, s);
  if (a.mix) return launch_tile(tile2d_tmem_kernel<R, false, 2, 3>, 4, a, s);
  return a.comp ? launch_tile(tile2d_tmem_kernel<R, false, 2, 2>, 4, a, s)
                : launch_tile(tile2d_tmem_kernel<R, false, 2, 1>, 4, a, s);
}

}  // namespace
}  // namespace wave
