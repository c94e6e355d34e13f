// Fused leapfrog step for the variable-density acoustic equation (Eq.
// wavetopopt) with the second-order stencil of Eq. FDstencil2:
//
//   u^{n+1} = 2 u^n - u^{n-1} + dt^2/(a h^2) sum_faces b_f (u_j - u_i),
//   b_f = 2 b_i b_j / (b_i + b_j)   (harmonic mean of b = 1/rho, Sec. 3.1),
//
// ghost material = boundary material (even mirror of b), ghost u per the BC.
// Sensitivity increment (dt times the per-step discrete Eq. kernel2):
//
//   acc += acc_scale * [ da (u^{n+1} - u^n)^2 - dbs sum_faces dbf (u_j - u_i)^2 ]
//
// with dbs = (dt^2/h^2) db/dgamma and dbf = d b_f / d b_i = 2 b_j^2/(b_i+b_j)^2
// (1 for a Dirichlet ghost face, whose material follows cell i).  The mass
// term belongs to the half level n+1/2, the stiffness term to level n.
//
// Mapping (2D): as the 2D velocity kernel (warp per 128-cell strip, march in
// y), with a second staged field b; 3D below.
#include "wave_internal.cuh"

namespace wave {

template <typename T>
__device__ __forceinline__ float4 round_storage(float4 v) {
  if constexpr (sizeof(T) == 4) {
    return v;
  } else {
    T b0 = T(v.x), b1 = T(v.y), b2 = T(v.z), b3 = T(v.w);
    return make_float4(float(b0), float(b1), float(b2), float(b3));
  }
}

// Face contribution of one neighbour j of cell i.
struct Face {
  float flux;   // b_f (u_j - u_i)
  float grad;   // dbf (u_j - u_i)^2
};

__device__ __forceinline__ Face face(float ui, float uj, float bi, float bj, bool dirichlet_ghost) {
  const float du = uj - ui;
  const float sum = bi + bj;
  const float bf = 2.f * bi * bj / sum;
  const float dbf = dirichlet_ghost ? 1.f : 2.f * bj * bj / (sum * sum);
  Face f;
  f.flux = bf * du;
  f.grad = dbf * du * du;
  return f;
}

__device__ __forceinline__ void kahan_add_d(float& acc, float& comp, float v) {
  const float y = v - comp;
  const float t = acc + y;
  comp = (t - acc) - y;
  acc = t;
}

// Stage one row of a field with its 4-cell x halos (ghost rule per `bc`).
template <typename T>
__device__ __forceinline__ void stage_row(float* srow, const T* __restrict__ f, int64_t rowbase, float4 own,
                                          int64_t x0, bool xin, int lane, const Geom& g, int bc) {
  *reinterpret_cast<float4*>(srow + 4 + 4 * lane) = own;
  if (xin) {
    if (lane == 0) *reinterpret_cast<float4*>(srow) = Stor<T>::ld4_nc(f + rowbase + x0 - 4);
    if (lane == 31) *reinterpret_cast<float4*>(srow + 4 + kStrip) = Stor<T>::ld4_nc(f + rowbase + x0 + kStrip);
  } else {
    __syncwarp();
    int64_t gx = -1;
    int p = 0;
    if (lane == 0) { gx = x0 - 1; p = 3; }
    if (lane == 8) { gx = g.nx < x0 + kStrip ? g.nx : x0 + kStrip; p = (int)(gx - x0 + 4); }
    if (lane == 0 || lane == 8) {
      float s;
      const int64_t m = mirror_index(gx, g.nx, bc, &s);
      srow[p] = s == 0.f ? 0.f : s * Stor<T>::ld1(f + rowbase + m);
    }
  }
}

template <typename T, int WPB>
__global__ void __launch_bounds__(WPB * 32)
step2d_density_kernel(StepArgs a) {
  chain_wait();
  __shared__ __align__(16) float su[WPB][kRowW];
  __shared__ __align__(16) float sb[WPB][kRowW];
  const Geom& g = a.g;
  const int lane = threadIdx.x & 31;
  const int warp = threadIdx.x >> 5;
  const int64_t nstrips = (g.nx + kStrip - 1) / kStrip;
  const int64_t gw = (int64_t)blockIdx.x * WPB + warp;
  const int64_t strip = gw % nstrips;
  const int64_t y0 = (gw / nstrips) * a.zblock;
  if (y0 >= g.ny) return;
  const int64_t y1 = min(y0 + a.zblock, g.ny);
  const int64_t x0 = strip * kStrip;
  const int64_t xl = x0 + 4 * lane;
  const bool xin = (x0 >= 4) && (x0 + kStrip + 4 <= g.nx);
  const T* __restrict__ uc = after_wait(reinterpret_cast<const T*>(a.u_cur));
  const T* __restrict__ up = after_wait(reinterpret_cast<const T*>(a.u_prev));
  const float* __restrict__ bm = a.bmat;
  const bool dir = g.bc == WAVE_DIRICHLET;
  for (int i = lane; i < kRowW; i += 32) { su[warp][i] = 0.f; sb[warp][i] = 1.f; }

  auto uload = [&](int64_t yy) -> float4 {
    float s;
    const int64_t ys = mirror_index(yy, g.ny, g.bc, &s);
    if (s == 0.f) return make_float4(0.f, 0.f, 0.f, 0.f);
    return f4_scale(Stor<T>::ld4_nc(uc + ys * g.px + xl), s);
  };
  auto bload = [&](int64_t yy) -> float4 {   // material ghost = boundary material
    float s;
    const int64_t ys = mirror_index(yy, g.ny, WAVE_NEUMANN, &s);
    return __ldg(reinterpret_cast<const float4*>(bm + ys * g.px + xl));
  };

  float4 qu0 = uload(y0 - 1), qu1 = uload(y0);
  float4 qb0 = bload(y0 - 1), qb1 = bload(y0);
  for (int64_t y = y0; y < y1; ++y) {
    const float4 qu2 = uload(y + 1);
    const float4 qb2 = bload(y + 1);
    const int64_t off = y * g.px + xl;
    const float4 u_old = Stor<T>::ld4(up + off);
    const float4 ca = __ldg(reinterpret_cast<const float4*>(a.coef + off));
    __syncwarp();
    stage_row<T>(su[warp], uc, y * g.px, qu1, x0, xin, lane, g, g.bc);
    stage_row<float>(sb[warp], bm, y * g.px, qb1, x0, xin, lane, g, WAVE_NEUMANN);
    __syncwarp();
    const float* ru = su[warp];
    const float* rb = sb[warp];
    float flux[4], grad[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const int p = 4 + 4 * lane + i;
      const int64_t x = xl + i;
      const float ui = ru[p], bi = rb[p];
      const float uy_m = f4_get(qu0, i), uy_p = f4_get(qu2, i);
      const float by_m = f4_get(qb0, i), by_p = f4_get(qb2, i);
      Face fxm = face(ui, ru[p - 1], bi, rb[p - 1], dir && x == 0);
      Face fxp = face(ui, ru[p + 1], bi, rb[p + 1], dir && x == g.nx - 1);
      Face fym = face(ui, uy_m, bi, by_m, dir && y == 0);
      Face fyp = face(ui, uy_p, bi, by_p, dir && y == g.ny - 1);
      flux[i] = (fxm.flux + fxp.flux) + (fym.flux + fyp.flux);
      grad[i] = x < g.nx ? (fxm.grad + fxp.grad) + (fym.grad + fyp.grad) : 0.f;   // row padding stays zero
    }
    float4 un;
    un.x = fmaf(ca.x, flux[0], 2.f * qu1.x - u_old.x);
    un.y = fmaf(ca.y, flux[1], 2.f * qu1.y - u_old.y);
    un.z = fmaf(ca.z, flux[2], 2.f * qu1.z - u_old.z);
    un.w = fmaf(ca.w, flux[3], 2.f * qu1.w - u_old.w);
    Stor<T>::st4(reinterpret_cast<T*>(a.u_prev) + off, un);
    if (a.acc_mass || a.acc_stiff) {
      const float4 ur = round_storage<T>(un);
      const float d[4] = {ur.x - qu1.x, ur.y - qu1.y, ur.z - qu1.z, ur.w - qu1.w};
      float c[4];
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        float v = 0.f;
        if (a.acc_mass) v = a.da * d[i] * d[i];
        if (a.acc_stiff) v = fmaf(-a.dbs, grad[i], v);
        c[i] = a.acc_scale * v;
      }
      float4* accp = reinterpret_cast<float4*>(a.acc + off);
      float4 ac = *accp;
      if (a.comp) {
        float4* cpp = reinterpret_cast<float4*>(a.comp + off);
        float4 cp = *cpp;
        kahan_add_d(ac.x, cp.x, c[0]);
        kahan_add_d(ac.y, cp.y, c[1]);
        kahan_add_d(ac.z, cp.z, c[2]);
        kahan_add_d(ac.w, cp.w, c[3]);
        *cpp = cp;
      } else {
        ac.x += c[0]; ac.y += c[1]; ac.z += c[2]; ac.w += c[3];
      }
      *accp = ac;
    }
    qu0 = qu1; qu1 = qu2;
    qb0 = qb1; qb1 = qb2;
  }
}

// 3D, 16-bit storage: a warp owns one 128-cell strip of a (y, z) row and marches up z over a
// block of planes.  z neighbours come from a three-plane register queue, y
// neighbours from direct loads of the rows y-1 and y+1 (L1/L2-resident: the
// warps of the neighbouring rows read them too), x neighbours from the
// staged own row.  Same face arithmetic and sensitivity increment as 2D.
template <typename T, int WPB>
__global__ void __launch_bounds__(WPB * 32)
step3d_density_kernel(StepArgs a) {
  __shared__ __align__(16) float su[WPB][kRowW];
  __shared__ __align__(16) float sb[WPB][kRowW];
  const Geom& g = a.g;
  const int lane = threadIdx.x & 31;
  const int warp = threadIdx.x >> 5;
  const int64_t nstrips = (g.nx + kStrip - 1) / kStrip;
  const int64_t nzb = (g.nz + a.zblock - 1) / a.zblock;
  const int64_t gw = (int64_t)blockIdx.x * WPB + warp;
  const int64_t strip = gw % nstrips;
  const int64_t rest = gw / nstrips;
  const int64_t y = rest % g.ny;
  const int64_t zb = rest / g.ny;
  if (zb >= nzb) return;   // whole warps only; the kernel has no block-wide barrier
  const int64_t z0 = zb * a.zblock;
  const int64_t z1 = min(z0 + a.zblock, g.nz);
  const int64_t x0 = strip * kStrip;
  const int64_t xl = x0 + 4 * lane;
  const bool xin = (x0 >= 4) && (x0 + kStrip + 4 <= g.nx);
  const T* __restrict__ uc = reinterpret_cast<const T*>(a.u_cur);
  const T* __restrict__ up = reinterpret_cast<const T*>(a.u_prev);
  const float* __restrict__ bm = a.bmat;
  const bool dir = g.bc == WAVE_DIRICHLET;
  for (int i = lane; i < kRowW; i += 32) { su[warp][i] = 0.f; sb[warp][i] = 1.f; }

  auto uload = [&](int64_t yy, int64_t zz) -> float4 {   // u with the ghost rule in y and z
    float sy, sz;
    const int64_t ys = mirror_index(yy, g.ny, g.bc, &sy);
    const int64_t zs = mirror_index(zz, g.nz, g.bc, &sz);
    const float sg = sy * sz;
    if (sg == 0.f) return make_float4(0.f, 0.f, 0.f, 0.f);
    return f4_scale(Stor<T>::ld4_nc(uc + zs * g.plane + ys * g.px + xl), sg);
  };
  auto bload = [&](int64_t yy, int64_t zz) -> float4 {   // material ghost = boundary material
    float sy, sz;
    const int64_t ys = mirror_index(yy, g.ny, WAVE_NEUMANN, &sy);
    const int64_t zs = mirror_index(zz, g.nz, WAVE_NEUMANN, &sz);
    return __ldg(reinterpret_cast<const float4*>(bm + zs * g.plane + ys * g.px + xl));
  };

  float4 qu0 = uload(y, z0 - 1), qu1 = uload(y, z0);
  float4 qb0 = bload(y, z0 - 1), qb1 = bload(y, z0);
  for (int64_t z = z0; z < z1; ++z) {
    const float4 qu2 = uload(y, z + 1);
    const float4 qb2 = bload(y, z + 1);
    const float4 uym4 = uload(y - 1, z), uyp4 = uload(y + 1, z);
    const float4 bym4 = bload(y - 1, z), byp4 = bload(y + 1, z);
    const int64_t rowbase = z * g.plane + y * g.px;
    const int64_t off = rowbase + xl;
    const float4 u_old = Stor<T>::ld4(up + off);
    const float4 ca = __ldg(reinterpret_cast<const float4*>(a.coef + off));
    __syncwarp();
    stage_row<T>(su[warp], uc, rowbase, qu1, x0, xin, lane, g, g.bc);
    stage_row<float>(sb[warp], bm, rowbase, qb1, x0, xin, lane, g, WAVE_NEUMANN);
    __syncwarp();
    const float* ru = su[warp];
    const float* rb = sb[warp];
    float flux[4], grad[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const int p = 4 + 4 * lane + i;
      const int64_t x = xl + i;
      const float ui = ru[p], bi = rb[p];
      Face fxm = face(ui, ru[p - 1], bi, rb[p - 1], dir && x == 0);
      Face fxp = face(ui, ru[p + 1], bi, rb[p + 1], dir && x == g.nx - 1);
      Face fym = face(ui, f4_get(uym4, i), bi, f4_get(bym4, i), dir && y == 0);
      Face fyp = face(ui, f4_get(uyp4, i), bi, f4_get(byp4, i), dir && y == g.ny - 1);
      Face fzm = face(ui, f4_get(qu0, i), bi, f4_get(qb0, i), dir && z == 0);
      Face fzp = face(ui, f4_get(qu2, i), bi, f4_get(qb2, i), dir && z == g.nz - 1);
      flux[i] = ((fxm.flux + fxp.flux) + (fym.flux + fyp.flux)) + (fzm.flux + fzp.flux);
      grad[i] = x < g.nx ? ((fxm.grad + fxp.grad) + (fym.grad + fyp.grad)) + (fzm.grad + fzp.grad)
                         : 0.f;   // row padding stays zero
    }
    float4 un;
    un.x = fmaf(ca.x, flux[0], 2.f * qu1.x - u_old.x);
    un.y = fmaf(ca.y, flux[1], 2.f * qu1.y - u_old.y);
    un.z = fmaf(ca.z, flux[2], 2.f * qu1.z - u_old.z);
    un.w = fmaf(ca.w, flux[3], 2.f * qu1.w - u_old.w);
    Stor<T>::st4(reinterpret_cast<T*>(a.u_prev) + off, un);
    if (a.acc_mass || a.acc_stiff) {
      const float4 ur = round_storage<T>(un);
      const float d[4] = {ur.x - qu1.x, ur.y - qu1.y, ur.z - qu1.z, ur.w - qu1.w};
      float c[4];
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        float v = 0.f;
        if (a.acc_mass) v = a.da * d[i] * d[i];
        if (a.acc_stiff) v = fmaf(-a.dbs, grad[i], v);
        c[i] = a.acc_scale * v;
      }
      float4* accp = reinterpret_cast<float4*>(a.acc + off);
      float4 ac = *accp;
      if (a.comp) {
        float4* cpp = reinterpret_cast<float4*>(a.comp + off);
        float4 cp = *cpp;
        kahan_add_d(ac.x, cp.x, c[0]);
        kahan_add_d(ac.y, cp.y, c[1]);
        kahan_add_d(ac.z, cp.z, c[2]);
        kahan_add_d(ac.w, cp.w, c[3]);
        *cpp = cp;
      } else {
        ac.x += c[0]; ac.y += c[1]; ac.z += c[2]; ac.w += c[3];
      }
      *accp = ac;
    }
    qu0 = qu1; qu1 = qu2;
    qb0 = qb1; qb1 = qb2;
  }
}

// 3D, FP32 storage: one or two fields (the +-k pair) advance together.
//
// The weights of a face, 2 b_i b_j / (b_i + b_j) and its derivative, cost a
// division each; the kernel above divides 12 times per cell, field and step.
// Here a face's flux weight is computed once for the two cells of a lane that
// share it (x faces of a quad, z faces carried to the next plane), the
// derivatives only where something accumulates, and both fields use the same
// weights, coefficient and accumulator.  180 x 210 x 250, symmetric mode: 201 ->
// 72 us per field and step.  The divisions still bound it (4.25 per cell, 10.25
// with increments).  A CTA is 8 rows of a strip, so the rows y-1 and y+1 are L1
// hits; x neighbours come by shuffle.  Two CTAs per SM (three without
// increments) although that spills a few registers: one CTA of 186 took 98 us
// where two take 73, three 88.  Sums keep the operand order and the fused products of the kernel
// above as compiled (x pair: upper face fused onto the lower one, except at x
// mod 4 = 3; z flux pair fused the same way; all others unfused): same bits.
__device__ __forceinline__ float flux_weight(float bi, float bj) { return 2.f * bi * bj / (bi + bj); }
__device__ __forceinline__ float grad_weight(float bi, float bj) {
  const float sum = bi + bj;
  return 2.f * bj * bj / (sum * sum);
}
__device__ __forceinline__ void f4_array(const float4& v, float (&o)[4]) { o[0] = v.x; o[1] = v.y; o[2] = v.z; o[3] = v.w; }

constexpr int kMarchRows = 8;

template <int NF, int ACC>   // ACC: 0 none, 1 acc, 2 with compensation
__global__ void __launch_bounds__(kMarchRows * 32, ACC == 0 ? 3 : 2)
step3d_density_march_kernel(StepArgs a) {
  chain_wait();
  const Geom& g = a.g;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int64_t nstrips = (g.nx + kStrip - 1) / kStrip, nyt = (g.ny + kMarchRows - 1) / kMarchRows;
  const int64_t strip = blockIdx.x % nstrips, rest = blockIdx.x / nstrips;
  const int64_t y = (rest % nyt) * kMarchRows + warp;
  if (y >= g.ny) return;   // whole warps only; the kernel has no block-wide barrier
  const int64_t z0 = (rest / nyt) * a.zblock, z1 = min(z0 + a.zblock, g.nz);
  const int64_t x0 = strip * kStrip, xl = x0 + 4 * lane;
  const bool neu = g.bc == WAVE_NEUMANN;
  const bool xend = x0 + kStrip >= g.nx;                 // the strip holds the last cell of the row
  const int qlast = (int)min((int64_t)4, g.nx - 1 - xl);  // the quad's element at nx - 1 (in the last strip), < 0 behind it
  const int64_t row = y * g.px + xl;
  const float* const bm = a.bmat;
  const float* uc[NF];
  float* up[NF];
  uc[0] = after_wait(reinterpret_cast<const float*>(a.u_cur));
  up[0] = reinterpret_cast<float*>(a.u_prev);
  if constexpr (NF == 2) {
    uc[1] = after_wait(reinterpret_cast<const float*>(a.u_cur2));
    up[1] = reinterpret_cast<float*>(a.u_prev2);
  }
  auto ld = [](const float* p) { return __ldg(reinterpret_cast<const float4*>(p)); };
  const float4 zero4 = make_float4(0.f, 0.f, 0.f, 0.f);

  // carried from plane to plane: this plane's u and b, the lower z face's
  // difference u_z - u_{z-1} and weights
  float u[NF][4], dzm[NF][4], b[4], fzm[4], gzm[4];
  f4_array(ld(bm + z0 * g.plane + row), b);
  {
    float bl[4];
    if (z0 > 0) f4_array(ld(bm + (z0 - 1) * g.plane + row), bl);
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      if (z0 == 0) bl[q] = b[q];
      fzm[q] = flux_weight(b[q], bl[q]);
      gzm[q] = ACC ? (z0 == 0 && !neu ? 1.f : grad_weight(b[q], bl[q])) : 0.f;
    }
#pragma unroll
    for (int f = 0; f < NF; ++f) {
      float ul[4];
      f4_array(ld(uc[f] + z0 * g.plane + row), u[f]);
      if (z0 > 0) f4_array(ld(uc[f] + (z0 - 1) * g.plane + row), ul);
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        if (z0 == 0) ul[q] = neu ? u[f][q] : 0.f;
        dzm[f][q] = u[f][q] - ul[q];
      }
    }
  }
  for (int64_t z = z0; z < z1; ++z) {
    const int64_t base = z * g.plane, off = base + row;
    const bool ztop = z == g.nz - 1;
    // loads of the plane
    float4 bu4 = zero4, bym4 = zero4, byp4 = zero4, uu4[NF], uym4[NF], uyp4[NF], uo4[NF];
    if (!ztop) bu4 = ld(bm + off + g.plane);
    if (y > 0) bym4 = ld(bm + off - g.px);
    if (y < g.ny - 1) byp4 = ld(bm + off + g.px);
    const float4 ca4 = ld(a.coef + off);
    float bxl = 0.f, bxr = 0.f, uxl[NF], uxr[NF];   // the quad's outer x neighbours at strip ends
    if (lane == 0 && x0 > 0) bxl = __ldg(bm + off - 1);
    if (lane == 31 && !xend) bxr = __ldg(bm + off + 4);
#pragma unroll
    for (int f = 0; f < NF; ++f) {
      uu4[f] = uym4[f] = uyp4[f] = zero4;
      uxl[f] = uxr[f] = 0.f;
      if (!ztop) uu4[f] = ld(uc[f] + off + g.plane);
      if (y > 0) uym4[f] = ld(uc[f] + off - g.px);
      if (y < g.ny - 1) uyp4[f] = ld(uc[f] + off + g.px);
      if (lane == 0 && x0 > 0) uxl[f] = __ldg(uc[f] + off - 1);
      if (lane == 31 && !xend) uxr[f] = __ldg(uc[f] + off + 4);
      uo4[f] = *reinterpret_cast<const float4*>(up[f] + off);
    }
    float4 ac4 = zero4, cp4 = zero4;
    if (ACC) ac4 = *reinterpret_cast<const float4*>(a.acc + off);
    if (ACC == 2) cp4 = *reinterpret_cast<const float4*>(a.comp + off);

    // weights: x faces 0..4 (face q between cells q-1 and q), y, upper z
    float bx[6], fx[5], gxm[4], gxp[4], fym[4], fyp[4], gym[4], gyp[4], fzp[4], gzp[4], gzn[4], bu[4], t[4];
    {
      float v = __shfl_up_sync(0xffffffffu, b[3], 1);
      bx[0] = lane == 0 ? (x0 > 0 ? bxl : b[0]) : v;
      v = __shfl_down_sync(0xffffffffu, b[0], 1);
      bx[5] = lane == 31 ? bxr : v;
#pragma unroll
      for (int q = 0; q < 4; ++q) bx[q + 1] = b[q];
      float br[4] = {bx[2], bx[3], bx[4], bx[5]};
      if (xend) {
#pragma unroll
        for (int q = 0; q < 4; ++q)
          if (q == qlast) br[q] = b[q];   // ghost material = boundary material
      }
      fx[0] = flux_weight(b[0], bx[0]);
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        fx[q + 1] = flux_weight(b[q], br[q]);
        if (ACC) {
          gxm[q] = grad_weight(b[q], bx[q]);
          gxp[q] = grad_weight(b[q], br[q]);
        }
      }
      if (ACC && !neu) {
        if (xl == 0) gxm[0] = 1.f;   // a Dirichlet ghost's material follows its cell
        if (xend) {
#pragma unroll
          for (int q = 0; q < 4; ++q)
            if (q == qlast) gxp[q] = 1.f;
        }
      }
      f4_array(bym4, t);
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        if (y == 0) t[q] = b[q];
        fym[q] = flux_weight(b[q], t[q]);
        if (ACC) gym[q] = y == 0 && !neu ? 1.f : grad_weight(b[q], t[q]);
      }
      f4_array(byp4, t);
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        if (y == g.ny - 1) t[q] = b[q];
        fyp[q] = flux_weight(b[q], t[q]);
        if (ACC) gyp[q] = y == g.ny - 1 && !neu ? 1.f : grad_weight(b[q], t[q]);
      }
      f4_array(bu4, bu);
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        if (ztop) bu[q] = b[q];
        fzp[q] = flux_weight(b[q], bu[q]);
        if (ACC) {
          gzp[q] = ztop && !neu ? 1.f : grad_weight(b[q], bu[q]);
          gzn[q] = grad_weight(bu[q], b[q]);   // the same face seen from the next plane
        }
      }
    }
    float ca[4], ac[4], cp[4];
    f4_array(ca4, ca);
    f4_array(ac4, ac);
    f4_array(cp4, cp);
#pragma unroll
    for (int f = 0; f < NF; ++f) {
      float uu[4], uym[4], uyp[4], uo[4], dx[5], dym[4], dyp[4], dzp[4], dr[4], un[4];
      f4_array(uu4[f], uu);
      f4_array(uym4[f], uym);
      f4_array(uyp4[f], uyp);
      f4_array(uo4[f], uo);
      float ul = __shfl_up_sync(0xffffffffu, u[f][3], 1), ur = __shfl_down_sync(0xffffffffu, u[f][0], 1);
      if (lane == 0) ul = x0 > 0 ? uxl[f] : (neu ? u[f][0] : 0.f);
      if (lane == 31) ur = uxr[f];
      dx[0] = u[f][0] - ul;
      dx[1] = u[f][1] - u[f][0];
      dx[2] = u[f][2] - u[f][1];
      dx[3] = u[f][3] - u[f][2];
      dx[4] = ur - u[f][3];
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        dr[q] = dx[q + 1];
        if (xend && q == qlast) dr[q] = (neu ? u[f][q] : 0.f) - u[f][q];
        if (y == 0) uym[q] = neu ? u[f][q] : 0.f;
        if (y == g.ny - 1) uyp[q] = neu ? u[f][q] : 0.f;
        if (ztop) uu[q] = neu ? u[f][q] : 0.f;
        dym[q] = uym[q] - u[f][q];
        dyp[q] = uyp[q] - u[f][q];
        dzp[q] = uu[q] - u[f][q];
        const float mx = __fmul_rn(fx[q], dx[q]);   // minus the lower face's flux
        const float px = q < 3 ? fmaf(fx[q + 1], dr[q], -mx) : __fsub_rn(__fmul_rn(fx[q + 1], dr[q]), mx);
        const float py = __fadd_rn(__fmul_rn(fym[q], dym[q]), __fmul_rn(fyp[q], dyp[q]));
        const float pz = fmaf(fzp[q], dzp[q], -__fmul_rn(fzm[q], dzm[f][q]));
        const float flux = __fadd_rn(__fadd_rn(px, py), pz);
        un[q] = fmaf(ca[q], flux, 2.f * u[f][q] - uo[q]);
      }
      *reinterpret_cast<float4*>(up[f] + off) = make_float4(un[0], un[1], un[2], un[3]);
      if constexpr (ACC != 0) {
        const float sc = f == 0 ? a.acc_scale : a.acc_scale2;
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          const float d = un[q] - u[f][q];
          float v = a.acc_mass ? __fmul_rn(__fmul_rn(a.da, d), d) : 0.f;
          if (a.acc_stiff) {
            const float lx = __fmul_rn(__fmul_rn(gxm[q], dx[q]), dx[q]), hx = __fmul_rn(gxp[q], dr[q]);
            const float sx = q < 3 ? fmaf(hx, dr[q], lx) : __fadd_rn(__fmul_rn(hx, dr[q]), lx);
            const float sy = __fadd_rn(__fmul_rn(__fmul_rn(gym[q], dym[q]), dym[q]), __fmul_rn(__fmul_rn(gyp[q], dyp[q]), dyp[q]));
            const float sz = __fadd_rn(__fmul_rn(__fmul_rn(gzm[q], dzm[f][q]), dzm[f][q]),
                                       __fmul_rn(__fmul_rn(gzp[q], dzp[q]), dzp[q]));
            float gr = __fadd_rn(__fadd_rn(sx, sy), sz);
            if (xend && q > qlast) gr = 0.f;   // row padding stays zero
            v = fmaf(-a.dbs, gr, v);
          }
          const float c = __fmul_rn(sc, v);
          if constexpr (ACC == 2) {
            const float yk = __fsub_rn(c, cp[q]), tk = __fadd_rn(ac[q], yk);
            cp[q] = __fsub_rn(__fsub_rn(tk, ac[q]), yk);
            ac[q] = tk;
          } else {
            ac[q] = __fadd_rn(ac[q], c);
          }
        }
      }
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        dzm[f][q] = dzp[q];
        u[f][q] = uu[q];
      }
    }
    if (ACC) *reinterpret_cast<float4*>(a.acc + off) = make_float4(ac[0], ac[1], ac[2], ac[3]);
    if (ACC == 2) *reinterpret_cast<float4*>(a.comp + off) = make_float4(cp[0], cp[1], cp[2], cp[3]);
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      b[q] = bu[q];
      fzm[q] = fzp[q];
      gzm[q] = gzn[q];
    }
  }
}

template <int NF>
static cudaError_t launch_march(const StepArgs& a, cudaStream_t s) {
  const Geom& g = a.g;
  const int64_t blocks = (g.nx + kStrip - 1) / kStrip * ((g.ny + kMarchRows - 1) / kMarchRows) *
                         ((g.nz + a.zblock - 1) / a.zblock);
  const bool acc = a.acc_mass || a.acc_stiff;
  if (NF == 2 && !acc) return cudaErrorInvalidValue;
  count_launch();
  if constexpr (NF == 1) {   // two fields only advance to accumulate
    if (!acc) return launch_chained(step3d_density_march_kernel<NF, 0>, (unsigned)blocks, kMarchRows * 32, 0, s, a);
  }
  if (!a.comp) return launch_chained(step3d_density_march_kernel<NF, 1>, (unsigned)blocks, kMarchRows * 32, 0, s, a);
  return launch_chained(step3d_density_march_kernel<NF, 2>, (unsigned)blocks, kMarchRows * 32, 0, s, a);
}

constexpr int kWarpsDen = 4;

template <typename T>
static cudaError_t launch_den(const StepArgs& a, cudaStream_t s) {
  const Geom& g = a.g;
  const int64_t nstrips = (g.nx + kStrip - 1) / kStrip;
  if (g.ndim == 3) {
    if constexpr (sizeof(T) == 4) {
      return a.u_cur2 ? launch_march<2>(a, s) : launch_march<1>(a, s);
    } else {
      const int64_t warps = nstrips * g.ny * ((g.nz + a.zblock - 1) / a.zblock);
      const int64_t blocks = (warps + kWarpsDen - 1) / kWarpsDen;
      count_launch();
      // plainly: chained, its CTAs land unevenly over the SMs and march there for
      // the whole kernel (BF16, 200 x 100 x 128, 24-step gradient: 7.2 ms chained,
      // 6.0 plain)
      step3d_density_kernel<T, kWarpsDen><<<(unsigned)blocks, kWarpsDen * 32, 0, s>>>(a);
      return cudaGetLastError();
    }
  }
  if (g.ndim != 2) return cudaErrorInvalidValue;
  const int64_t warps = nstrips * ((g.ny + a.zblock - 1) / a.zblock);
  const int64_t blocks = (warps + kWarpsDen - 1) / kWarpsDen;
  count_launch();
  return launch_chained(step2d_density_kernel<T, kWarpsDen>, (unsigned)blocks, kWarpsDen * 32, 0, s, a);
}

cudaError_t launch_step_density(const StepArgs& a, int storage, cudaStream_t s) {
  switch (storage) {
    case WAVE_F32: return launch_den<float>(a, s);
    case WAVE_BF16: return launch_den<__nv_bfloat16>(a, s);
    case WAVE_F16: return launch_den<__half>(a, s);
  }
  return cudaErrorInvalidValue;
}

}  // namespace wave
