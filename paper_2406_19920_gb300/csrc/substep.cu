// substep.cu -- one RK stage of Eq. 2a-2h (ibm_substep).
//
// Order of work (the paper's flowchart for one stage, Sec. 2.3):
//   E1  explicit terms: du = u^e - u^{n-1}
//         = dt [(a+b) nu L u - (a+b) G p - gamma N(u) - zeta N^{n-2}]   (Eq. 2a)
//       and N(u) stored for the next stage's zeta term;
//   L2  marker positions / surface velocity at the stage start time;
//   L1  U^e = interp(u^{n-1} + du) (Eq. 2b), F = (U^d - U^e)/dt (Eq. 2c),
//       du += dt spread(F) (Eq. 2d);
//   S1  three Helmholtz solves.  Eq. 2e, (I - c L) u* = u^e - c L u^{n-1} +
//       dt f with c = beta dt nu, is solved in increment form
//       (I - c L) delta = du, u* = u^{n-1} + delta (same system: subtract
//       (I - c L) u^{n-1} from both sides); u* overwrites u;
//   E2  b = D u* / ((a+b) dt)                                          (Eq. 2f)
//   S2  Poisson solve L phi = b (refined on the FP32 path)
//   E3  u^n = u* - (a+b) dt G phi, p^n = p + phi - c L phi             (Eq. 2g, 2h)
// RK coefficients: Rai & Moin's low-storage scheme, which the paper cites
// without printing.  Advection is the conservative MAC form div(u u) with
// two-point averages (the paper names second-order central differences).
#include <cmath>
#include <mutex>

#include "plan.h"
#include "tma.cuh"

namespace ibm {

template <typename T>
cudaError_t launch_interp(const ibm_plan_s *p, int n, const T *X, const T *u, const T *v, const T *w,
                          const T *du, const T *dv, const T *dw, T *U, const T *Ud, double inv_dt, T *F,
                          const T *X0, T *Xout, T *Udout, int kind, const double *params, double t,
                          cudaStream_t st);
template <typename T>
cudaError_t launch_spread(const ibm_plan_s *p, int n, const T *X, const T *F, const T *dV, T *fu, T *fv, T *fw,
                          double scale, cudaStream_t st);

static const double kAlpha[3] = {4.0 / 15.0, 1.0 / 15.0, 1.0 / 6.0};
static const double kBeta[3] = {4.0 / 15.0, 1.0 / 15.0, 1.0 / 6.0};
static const double kGamma[3] = {8.0 / 15.0, 5.0 / 12.0, 3.0 / 4.0};
static const double kZeta[3] = {0.0, -17.0 / 60.0, -5.0 / 12.0};

struct Geo {
  int nx, ny, nz;
  double ihx, ihy, ihz;  // 1/h
};

// field accessor with periodic x, z
template <typename T> struct F3 {
  const T *f;
  int nx, nz;
  __device__ __forceinline__ T at(int j, int k, int i) const {
    i = i < 0 ? i + nx : (i >= nx ? i - nx : i);
    k = k < 0 ? k + nz : (k >= nz ? k - nz : k);
    return f[((size_t)j * nz + k) * nx + i];
  }
};

// E1, all three components.  A CTA owns a TX x TZ column tile (a thread two
// columns, neighbours in z) and marches up a range of y planes; the planes j
// and j + 1 of u, v, w and j of p sit in shared memory with a one-cell periodic
// halo in x and z, copied there asynchronously two planes ahead (16 bytes a
// copy, the halo columns one by one), and N^{n-2} is loaded a plane ahead, so
// every field is read from HBM about once.  What a thread needs of plane j - 1 it still holds
// in registers, and so it does the advective fluxes it formed there: with
//   XY(i, j) = (u_{j-1} + u_j)(v_{i-1} + v_i),  XZ(i, k) = (u_{k-1} + u_k)(w_{i-1} + w_i),
//   YZ(j, k) = (v_{k-1} + v_k)(w_{j-1} + w_j)
// (times 4, on the cell edges) one flux serves the two components it
// transports, and the y and z neighbours' fluxes are the thread's own but at
// the ends.  That leaves some 80 operations a point (111 with every flux formed
// where it is used) and 16 shared-memory loads (40).  Every difference of two
// fluxes is one FMA on the second one's factors, with the first one's rounded
// product, and the y term, the largest between walls, is the last one added,
// unrounded: with two rounded products and the sum in another order N_v loses 4 % of
// its accuracy in FP32.
// Wall rules in y: u, w cell-centred with the no-slip ghost (-value) in the
// Laplacian and zero wall flux in the advective y-flux; v on faces, zero at
// the walls (j = 0 stored as the wall, j = ny not stored).
//
// IO: the inflow-outflow walls of Sec. 3 instead.  The y = 0 face carries
// v = v_lo with u = w = 0 there (the ghost -value and the zero y-flux of
// u, w are unchanged; v's lower neighbour at j = 1 is v_lo); the y = Ly
// wall carries the outlet planes uo, wo (u, w at the wall: ghost 2 g - u in
// the Laplacian, flux v_face * g) and vo (v on the outlet face), [nz][nx].
// Measured (one column a thread, planes j - 1 .. j + 1 in shared memory, 256
// threads, 16 planes a CTA, against now): FP32 128^3 35.7 -> 23.4 us, 384 x 256
// x 256 369 -> 240 us (1.31 GB: 5.4 TB/s; bound by instruction issue before, by
// HBM and the latency of its loads now), FP64 96 x 65 x 64 145 -> 81 us (bound
// by FP64 operations, 53 us at the pipe's rate, in 24 tiles on 152 SMs).  CTAs of
// 256 threads: 247 us at 384 x 256 x 256, one plane ahead 277 us.
constexpr int kExTX = 32, kExTY = 4, kExTZ = 2 * kExTY, kExThreads = kExTX * kExTY;

template <typename T> struct ExTile {
  static constexpr int VEC = 16 / (int)sizeof(T);     // elements of a 16-byte copy
  static constexpr int PITCH = kExTX + 2 * VEC;       // a row: VEC (the last is the left halo), TX, VEC
  static constexpr int ROWS = kExTZ + 2;
  static constexpr int PL = ROWS * PITCH;
  static constexpr int CPR = kExTX / VEC;             // 16-byte copies a row
  static constexpr int OPS = ROWS * (CPR + 2);        // copies a plane (and field)
  static constexpr int NQ = (OPS + kExThreads - 1) / kExThreads;
  static constexpr size_t bytes = sizeof(T) * (size_t)PL * 15;  // 4 planes of u, v, w, 3 of p
};

// Coefficients with the constant factors folded in: dt (a + b) nu / h^2 (vx,
// vy, vz), dt (a + b) / h (px, py, pz), 1 / (4 h) (qx, qy, qz), dt gamma, dt zeta.
template <typename T> struct ExCoef {
  T vx, vy, vz, px, py, pz, qx, qy, qz, gam, zet;
};

template <typename T, bool IO>
__global__ void __launch_bounds__(kExThreads, sizeof(T) == 4 ? 4 : 2)
k_explicit(int nx, int ny, int nz, int jc, const T *__restrict__ u_, const T *__restrict__ v_,
           const T *__restrict__ w_, const T *__restrict__ p_, T *Nu, T *Nv, T *Nw, T *__restrict__ du,
           T *__restrict__ dv, T *__restrict__ dw, ExCoef<T> cf, T v_lo, const T *__restrict__ uo,
           const T *__restrict__ vo, const T *__restrict__ wo) {
  using Cfg = ExTile<T>;
  constexpr int VEC = Cfg::VEC, PI = Cfg::PITCH, PL = Cfg::PL, CPR = Cfg::CPR, NQ = Cfg::NQ;
  extern __shared__ __align__(128) unsigned char smem_raw[];
  T *su = reinterpret_cast<T *>(smem_raw), *sv = su + 4 * PL, *sw = sv + 4 * PL, *sp = sw + 4 * PL;
  const int tx = threadIdx.x % kExTX, ty = threadIdx.x / kExTX;
  const int i0 = blockIdx.x * kExTX, k0 = blockIdx.y * kExTZ;
  const int jb = blockIdx.z * jc, je = min(ny, jb + jc);
  const size_t plane = (size_t)nz * nx;
  // this thread's copies of a plane: source offset, destination, 16 bytes or one element
  int src[NQ], dst[NQ];
  bool wide[NQ];
#pragma unroll
  for (int q = 0; q < NQ; ++q) {
    const int op = threadIdx.x + q * kExThreads;
    const int r = op < Cfg::OPS ? op / (CPR + 2) : 0, e = op - r * (CPR + 2);
    const int kk = (k0 - 1 + r + nz) % nz;
    const int last = min(kExTX, nx - i0);  // the right halo follows the last column of the tile
    wide[q] = e < CPR;
    const int x = e < CPR ? i0 + e * VEC : e == CPR ? i0 - 1 + (i0 == 0 ? nx : 0) : (i0 + last == nx ? 0 : i0 + last);
    src[q] = (op < Cfg::OPS && (e >= CPR || x < nx)) ? kk * nx + x : -1;
    dst[q] = r * PI + (e < CPR ? VEC + e * VEC : e == CPR ? VEC - 1 : VEC + last);
  }
  auto copy = [&](const T *F, int jj, T *buf) {
    const T *f = F + (size_t)jj * plane;
#pragma unroll
    for (int q = 0; q < NQ; ++q) {
      if (src[q] < 0) continue;
      if (wide[q]) cp_async16(buf + dst[q], f + src[q]);
      else if constexpr (sizeof(T) == 8) cp_async8(buf + dst[q], f + src[q]);
      else cp_async4(buf + dst[q], f + src[q]);
    }
  };
  // slots of planes j, j + 1 and of the two planes in flight (rotated each plane)
  int s0 = 0, s1 = PL, s2 = 2 * PL, s3 = 3 * PL;
  pdl_wait();
  copy(u_, jb, su + s0); copy(v_, jb, sv + s0); copy(w_, jb, sw + s0); copy(p_, jb, sp);
  if (jb + 1 < ny) { copy(u_, jb + 1, su + s1); copy(v_, jb + 1, sv + s1); copy(w_, jb + 1, sw + s1); }
  const int i = i0 + tx, k = k0 + 2 * ty;
  const bool inside = i < nx && k < nz;  // nz is even: both columns or none
  const int c = (2 * ty + 1) * PI + VEC + tx;  // column 0 in a tile plane; column 1 is c + PI
  const size_t col = inside ? (size_t)k * nx + i : 0;
  const T v_wall = IO ? v_lo : (T)0;
  // of plane j - 1: u (and at i + 1), v, w (and at k + 2), p
  T ud[2] = {}, uEd[2] = {}, vd[2] = {}, wd[3] = {}, pd[2] = {};
  if (inside && jb > 0) {
    const size_t below = (size_t)(jb - 1) * plane;
    const T *pu = u_ + below, *pv = v_ + below, *pw = w_ + below, *pp = p_ + below;
    const size_t ce = i + 1 < nx ? col + 1 : col + 1 - nx;
    const size_t cn = k + 2 < nz ? col + 2 * (size_t)nx : (size_t)i;
#pragma unroll
    for (int z = 0; z < 2; ++z) {
      ud[z] = pu[col + (size_t)z * nx];
      uEd[z] = pu[ce + (size_t)z * nx];
      vd[z] = jb == 1 ? v_wall : pv[col + (size_t)z * nx];
      wd[z] = pw[col + (size_t)z * nx];
      pd[z] = pp[col + (size_t)z * nx];
    }
    wd[2] = pw[cn];
  }
  cp_async_commit();
  if (jb + 2 < ny && jb + 1 < je) { copy(u_, jb + 2, su + s2); copy(v_, jb + 2, sv + s2); copy(w_, jb + 2, sw + s2); }
  if (jb + 1 < je) copy(p_, jb + 1, sp + PL);
  cp_async_commit();
  cp_async_wait_group<1>();
  __syncthreads();
  // of plane j, from the step before: u, u at i + 1, v at k - 1 .. k + 2, v at i -+ 1, w at k .. k + 2
  T u0[2], uE[2], vc[4], vW[2], vE[2], w0[3];
  const T *U = su + s0 + c, *V = sv + s0 + c, *W = sw + s0 + c;
#pragma unroll
  for (int z = 0; z < 2; ++z) {
    u0[z] = U[z * PI];
    uE[z] = U[z * PI + 1];
    vW[z] = V[z * PI - 1];
    vE[z] = V[z * PI + 1];
  }
#pragma unroll
  for (int z = 0; z < 4; ++z) vc[z] = V[(z - 1) * PI];
#pragma unroll
  for (int z = 0; z < 3; ++z) w0[z] = W[z * PI];
  // fluxes XY, YZ on the lower edges of plane j (zero at the wall j = 0), their differences to the next edge along x
  // and z, and twice the average of v under the plane
  T xy[2] = {}, dxy[2] = {}, yz[2] = {}, dyz[2] = {}, va[2] = {};
  if (jb > 0) {
    T A[3], B[3];
#pragma unroll
    for (int z = 0; z < 3; ++z) { A[z] = vc[z] + vc[z + 1]; B[z] = wd[z] + w0[z]; }
#pragma unroll
    for (int z = 0; z < 2; ++z) {
      xy[z] = (vW[z] + vc[z + 1]) * (ud[z] + u0[z]);
      dxy[z] = fma(vc[z + 1] + vE[z], uEd[z] + uE[z], -xy[z]);
      yz[z] = A[z] * B[z];
      dyz[z] = fma(A[z + 1], B[z + 1], -yz[z]);
      va[z] = vd[z] + vc[z + 1];
    }
  }
  const bool n_prev = cf.zet != (T)0;  // N^{n-2} unused (and maybe unset) at stage 1
  int ps = 0;                          // p slot of plane j
  size_t at = (size_t)jb * plane + col;
  T nuN[2] = {}, nvN[2] = {}, nwN[2] = {};
  auto fetch_n = [&](size_t o) {
    if (n_prev && inside) {
#pragma unroll
      for (int z = 0; z < 2; ++z) {
        nuN[z] = Nu[o + (size_t)z * nx];
        nvN[z] = Nv[o + (size_t)z * nx];
        nwN[z] = Nw[o + (size_t)z * nx];
      }
    }
  };
  fetch_n(at);
  for (int j = jb; j < je; ++j, at += plane) {
    if (j > jb) {
      cp_async_wait_group<1>();
      __syncthreads();  // planes j + 1 of u, v, w and j of p have landed; plane j - 1's slots are free
    }
    const bool lo = j == 0, hi = j + 1 >= ny;
    if (j + 2 < je) {
      copy(p_, j + 2, sp + (ps == 0 ? 2 * PL : ps - PL));
      if (j + 3 < ny) { copy(u_, j + 3, su + s3); copy(v_, j + 3, sv + s3); copy(w_, j + 3, sw + s3); }
    }
    cp_async_commit();
    // N^{n-2} of this plane arrived during the last one
    T nu[2], nv[2], nw[2];
#pragma unroll
    for (int z = 0; z < 2; ++z) { nu[z] = nuN[z]; nv[z] = nvN[z]; nw[z] = nwN[z]; }
    if (j + 1 < je) fetch_n(at + plane);
    // plane j + 1 and the fluxes on the upper edges
    T u1[2], uE1[2], vc1[4], vW1[2], vE1[2], w1[3], xy1[2], dxy1[2], yz1[2], dyz1[2], uu[2], wu[2], vu[2];
    T xyj[2], yzj[2];  // differences of XY, YZ along y
    if (!hi) {
      const T *U1 = su + s1 + c, *V1 = sv + s1 + c, *W1 = sw + s1 + c;
#pragma unroll
      for (int z = 0; z < 2; ++z) {
        u1[z] = U1[z * PI];
        uE1[z] = U1[z * PI + 1];
        vW1[z] = V1[z * PI - 1];
        vE1[z] = V1[z * PI + 1];
      }
#pragma unroll
      for (int z = 0; z < 4; ++z) vc1[z] = V1[(z - 1) * PI];
#pragma unroll
      for (int z = 0; z < 3; ++z) w1[z] = W1[z * PI];
      T A[3], B[3];
#pragma unroll
      for (int z = 0; z < 3; ++z) { A[z] = vc1[z] + vc1[z + 1]; B[z] = w0[z] + w1[z]; }
#pragma unroll
      for (int z = 0; z < 2; ++z) {
        const T a = vW1[z] + vc1[z + 1], b = u0[z] + u1[z];
        xy1[z] = a * b;
        xyj[z] = fma(a, b, -xy[z]);
        dxy1[z] = fma(vc1[z + 1] + vE1[z], uE[z] + uE1[z], -xy1[z]);
        yz1[z] = A[z] * B[z];
        yzj[z] = fma(A[z], B[z], -yz[z]);
        dyz1[z] = fma(A[z + 1], B[z + 1], -yz1[z]);
        uu[z] = u1[z];
        wu[z] = w1[z];
        vu[z] = vc1[z + 1];
      }
    } else {
      // the wall above: no plane, no flux; IO: the outlet's values
#pragma unroll
      for (int z = 0; z < 2; ++z) {
        u1[z] = uE1[z] = vW1[z] = vE1[z] = xy1[z] = dxy1[z] = yz1[z] = dyz1[z] = (T)0;
        xyj[z] = -xy[z];
        yzj[z] = -yz[z];
        uu[z] = -u0[z];
        wu[z] = -w0[z];
        vu[z] = (T)0;
      }
#pragma unroll
      for (int z = 0; z < 4; ++z) vc1[z] = (T)0;
#pragma unroll
      for (int z = 0; z < 3; ++z) w1[z] = (T)0;
      if (IO && inside) {
#pragma unroll
        for (int z = 0; z < 2; ++z) {
          const int kz = k + z, iw = i == 0 ? nx - 1 : i - 1, ks = kz == 0 ? nz - 1 : kz - 1;
          const T ug = uo[kz * nx + i], wg = wo[kz * nx + i], vg = vo[kz * nx + i];
          uu[z] = 2 * ug - u0[z];
          wu[z] = 2 * wg - w0[z];
          vu[z] = vg;
          xyj[z] = fma(vo[kz * nx + iw] + vg, ug + ug, -xy[z]);
          yzj[z] = fma(vo[ks * nx + i] + vg, wg + wg, -yz[z]);
        }
      }
    }
    const T vb[2] = {lo ? v_wall : vc[1], lo ? v_wall : vc[2]};
    // the rest of plane j
    U = su + s0 + c; V = sv + s0 + c; W = sw + s0 + c;
    const T *Pp = sp + ps + c;
    const T uS = U[-PI], uN = U[2 * PI], uES = U[1 - PI], wS = W[-PI];
    const T uk[4] = {uS, u0[0], u0[1], uN};     // u at k - 1 .. k + 2
    const T wk[4] = {wS, w0[0], w0[1], w0[2]};  // w at k - 1 .. k + 2
    const T uEk[3] = {uES, uE[0], uE[1]};       // u at i + 1, k - 1 .. k + 1
    const T pS = Pp[-PI];
    T wW[3], xzA[3], xzB[3], wa[3], p0[2];
#pragma unroll
    for (int z = 0; z < 3; ++z) {
      wW[z] = W[z * PI - 1];
      xzA[z] = wW[z] + w0[z];
      xzB[z] = uk[z] + uk[z + 1];
      wa[z] = wk[z] + wk[z + 1];
    }
#pragma unroll
    for (int z = 0; z < 2; ++z) p0[z] = Pp[z * PI];
#pragma unroll
    for (int z = 0; z < 2; ++z) {
      const size_t o = at + (size_t)z * nx;
      const T uw = U[z * PI - 1], wE = W[z * PI + 1];
      const T xz = xzA[z] * xzB[z], va1 = vb[z] + vu[z];
      // u (x-faces)
      {
        const T a = u0[z] + uE[z], b = uw + u0[z];  // twice the averages
        const T N = fma(xyj[z], cf.qy, fma(fma(a, a, -(b * b)), cf.qx, fma(xzA[z + 1], xzB[z + 1], -xz) * cf.qz));
        const T lx = uE[z] - 2 * u0[z] + uw, lz = uk[z + 2] - 2 * u0[z] + uk[z];
        const T ly = uu[z] - 2 * u0[z] + (lo ? -u0[z] : ud[z]);
        if (inside) {
          du[o] = lx * cf.vx + lz * cf.vz + ly * cf.vy - (p0[z] - Pp[z * PI - 1]) * cf.px - cf.gam * N - cf.zet * nu[z];
          Nu[o] = N;
        }
      }
      // w (z-faces)
      {
        const T N = fma(yzj[z], cf.qy, fma(fma(wa[z + 1], wa[z + 1], -(wa[z] * wa[z])), cf.qz,
                                           fma(w0[z] + wE, uEk[z] + uEk[z + 1], -xz) * cf.qx));
        const T lx = wE - 2 * w0[z] + wW[z], lz = wk[z + 2] - 2 * w0[z] + wk[z];
        const T ly = wu[z] - 2 * w0[z] + (lo ? -w0[z] : wd[z]);
        if (inside) {
          dw[o] = lx * cf.vx + lz * cf.vz + ly * cf.vy - (p0[z] - (z == 0 ? pS : p0[0])) * cf.pz - cf.gam * N -
                  cf.zet * nw[z];
          Nw[o] = N;
        }
      }
      // v (y-faces, interior j = 1 .. ny - 1)
      {
        const T v0 = vc[z + 1];
        const T N = fma(fma(va1, va1, -(va[z] * va[z])), cf.qy, fma(dxy[z], cf.qx, dyz[z] * cf.qz));
        const T lx = vE[z] - 2 * v0 + vW[z], lz = vc[z + 2] - 2 * v0 + vc[z];
        const T ly = vu[z] - 2 * v0 + vd[z];
        if (inside) {
          dv[o] = lo ? (T)0
                     : lx * cf.vx + lz * cf.vz + ly * cf.vy - (p0[z] - pd[z]) * cf.py - cf.gam * N - cf.zet * nv[z];
          Nv[o] = lo ? (T)0 : N;
        }
      }
      va[z] = va1;
    }
    // plane j becomes plane j - 1
#pragma unroll
    for (int z = 0; z < 2; ++z) {
      ud[z] = u0[z]; u0[z] = u1[z]; uE[z] = uE1[z];
      vd[z] = vb[z]; vW[z] = vW1[z]; vE[z] = vE1[z];
      xy[z] = xy1[z]; dxy[z] = dxy1[z]; yz[z] = yz1[z]; dyz[z] = dyz1[z];
      pd[z] = p0[z];
    }
#pragma unroll
    for (int z = 0; z < 4; ++z) vc[z] = vc1[z];
#pragma unroll
    for (int z = 0; z < 3; ++z) { wd[z] = w0[z]; w0[z] = w1[z]; }
    const int t = s0;
    s0 = s1; s1 = s2; s2 = s3; s3 = t;
    ps = ps == 2 * PL ? 0 : ps + PL;
  }
}

// Planes a CTA marches: the split of ny whose CTAs take the fewest rounds of
// plane steps, a CTA's start counted as two (its first planes are read with
// nothing to compute).  per_sm: resident CTAs that add to each other's speed
// (FP32, waiting on memory: all 4; FP64, bound by the SM's FP64 pipe: 1; at
// 128^3 FP32 a split for 1 takes 33 us and for 4 23 us).
static int explicit_planes(int nx, int ny, int nz, int per_sm) {
  static std::once_flag once;
  static int sms = 0;
  std::call_once(once, [] {
    int dev = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  });
  const long tiles = (long)ceil_div(nx, kExTX) * ceil_div(nz, kExTZ);
  long best = 0;
  int jc = ny;
  for (int n = 1; n <= ny; ++n) {  // n chunks
    const int c = ceil_div(ny, n);
    if (c < 4 && n > 1) break;
    const long slots = (long)sms * per_sm;
    const long cost = ((tiles * ceil_div(ny, c) + slots - 1) / slots) * (c + 2);
    if (n == 1 || cost < best) { best = cost; jc = c; }
  }
  return jc;
}

template <typename T, bool IO>
static cudaError_t launch_explicit(const Geo &g, const T *u, const T *v, const T *w, const T *p, T *Nu, T *Nv, T *Nw,
                                   T *du, T *dv, T *dw, double visc, double pres, double gam, double zet, double dt,
                                   T v_lo, const T *uo, const T *vo, const T *wo, cudaStream_t st) {
  ExCoef<T> cf;
  cf.vx = (T)(dt * visc * g.ihx * g.ihx); cf.vy = (T)(dt * visc * g.ihy * g.ihy); cf.vz = (T)(dt * visc * g.ihz * g.ihz);
  cf.px = (T)(dt * pres * g.ihx); cf.py = (T)(dt * pres * g.ihy); cf.pz = (T)(dt * pres * g.ihz);
  cf.qx = (T)(0.25 * g.ihx); cf.qy = (T)(0.25 * g.ihy); cf.qz = (T)(0.25 * g.ihz);
  cf.gam = (T)(dt * gam); cf.zet = (T)(dt * zet);
  IBM_KTRY((ensure_max_smem<k_explicit<T, IO>>()));
  const int jc = explicit_planes(g.nx, g.ny, g.nz, sizeof(T) == 4 ? 4 : 1);
  const dim3 grid(ceil_div(g.nx, kExTX), ceil_div(g.nz, kExTZ), ceil_div(g.ny, jc));
  return launch_pdl(k_explicit<T, IO>, grid, dim3(kExThreads), ExTile<T>::bytes, st, g.nx, g.ny, g.nz, jc, u, v, w, p,
                    Nu, Nv, Nw, du, dv, dw, cf, v_lo, uo, vo, wo);
}

__device__ __forceinline__ void atomic_max_nonneg(double *addr, double v) {
  atomicMax(reinterpret_cast<unsigned long long *>(addr), (unsigned long long)__double_as_longlong(v));
}

// E2: b = D u * inv_scale in plain working precision (the right-hand side of
// Eq. 2f); with dmax, additionally max |D u| evaluated exactly: float-float
// differences for FP32 fields, FP64 for FP64 fields (the projection check).
// The wall faces carry v_lo (y = 0) and v_hi ([nz][nx] at y = Ly, NULL for
// 0).
template <typename T> struct DivExact;
template <> struct DivExact<float> {
  static __device__ __forceinline__ float eval(float ue, float uw, float vn, float vs, float wt, float wb,
                                               const ff &ihx, const ff &ihy, const ff &ihz) {
    ff d = ff_mul(two_sum(ue, -uw), ihx);
    d = ff_add(d, ff_mul(two_sum(vn, -vs), ihy));
    d = ff_add(d, ff_mul(two_sum(wt, -wb), ihz));
    return fabsf(__fadd_rn(d.hi, d.lo));
  }
};
template <> struct DivExact<double> {
  static __device__ __forceinline__ double eval(double ue, double uw, double vn, double vs, double wt, double wb,
                                                const ff &ihx, const ff &ihy, const ff &ihz) {
    return fabs((ue - uw) * (double)ihx.hi + (vn - vs) * (double)ihy.hi + (wt - wb) * (double)ihz.hi +
                ((ue - uw) * (double)ihx.lo + (vn - vs) * (double)ihy.lo + (wt - wb) * (double)ihz.lo));
  }
};

template <typename T>
__global__ void __launch_bounds__(128)
k_divergence(Geo g, const T *__restrict__ u_, const T *__restrict__ v_, const T *__restrict__ w_, T *b,
             T inv_scale, T ihx_t, T ihy_t, T ihz_t, ff ihx, ff ihy, ff ihz, double *dmax, T v_lo,
             const T *__restrict__ v_hi) {
  pdl_wait();
  int i, k, j;
  const bool inside = stencil_index(g.nx, g.nz, i, k, j);
  const size_t idx = ((size_t)j * g.nz + k) * g.nx + i;
  T mx = 0;
  if (inside) {
    const F3<T> U{u_, g.nx, g.nz}, V{v_, g.nx, g.nz}, W{w_, g.nx, g.nz};
    const T vs = j == 0 ? v_lo : V.at(j, k, i);
    const T vn = j + 1 >= g.ny ? (v_hi ? v_hi[k * g.nx + i] : (T)0) : V.at(j + 1, k, i);
    const T ue = U.at(j, k, i + 1), uw = U.at(j, k, i), wt = W.at(j, k + 1, i), wb = W.at(j, k, i);
    if (b) b[idx] = ((ue - uw) * ihx_t + (vn - vs) * ihy_t + (wt - wb) * ihz_t) * inv_scale;
    if (dmax) mx = DivExact<T>::eval(ue, uw, vn, vs, wt, wb, ihx, ihy, ihz);
  }
  if (dmax) {
    const unsigned full = 0xffffffffu;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) mx = fmax(mx, __shfl_xor_sync(full, mx, o));
    if (((threadIdx.y * blockDim.x + threadIdx.x) & 31) == 0) atomic_max_nonneg(dmax, (double)mx);
  }
}

// E3: u -= k G phi (in place), p += phi - c L phi (Neumann ghosts); the
// y = 0 face of v is set to v_lo.  kx .. = k / h, lx .. = c / h^2: with the
// factors folded on the host 16 operations a point instead of 28 (FP64 is bound
// by them: 96 x 65 x 64 21.7 -> 16.5 us).
template <typename T>
__global__ void __launch_bounds__(128)
k_project(int nx, int ny, int nz, T *__restrict__ u, T *__restrict__ v, T *__restrict__ w, T *__restrict__ p,
          const T *__restrict__ phi_, T kx, T ky, T kz, T lx, T ly, T lz, T v_lo) {
  pdl_wait();
  int i, k, j;
  if (!stencil_index(nx, nz, i, k, j)) return;
  const size_t idx = ((size_t)j * nz + k) * nx + i;
  const F3<T> Ph{phi_, nx, nz};
  const T f0 = Ph.at(j, k, i);
  const T dw = f0 - Ph.at(j, k, i - 1), ds = f0 - Ph.at(j, k - 1, i);
  const T dd = j > 0 ? f0 - Ph.at(j - 1, k, i) : (T)0;
  const T de = Ph.at(j, k, i + 1) - f0, dn = Ph.at(j, k + 1, i) - f0;
  const T du = j + 1 < ny ? Ph.at(j + 1, k, i) - f0 : (T)0;
  u[idx] -= kx * dw;
  w[idx] -= kz * ds;
  if (j > 0) v[idx] -= ky * dd;
  else v[idx] = v_lo;
  p[idx] += f0 - ((de - dw) * lx + (dn - ds) * lz + (du - dd) * ly);
}

// FP32 versions of E2 and E3 with four consecutive x points per thread:
// float4 rows, the x neighbours from the same float4 plus one or two
// scalars, shared index arithmetic (the one-point kernels are load-latency
// bound).  Each point's arithmetic is the one-point kernel's, in the same
// order.  Grid (ceil(nz nx / 4 / 128), ny), 128 threads; nx % 4 == 0 and
// 16-byte aligned fields.
__device__ __forceinline__ float4 ld4(const float *p) { return *reinterpret_cast<const float4 *>(p); }
__device__ __forceinline__ float comp4(const float4 &a, int q) { return q == 0 ? a.x : q == 1 ? a.y : q == 2 ? a.z : a.w; }
__device__ __forceinline__ void set4(float4 &a, int q, float v) {
  if (q == 0) a.x = v; else if (q == 1) a.y = v; else if (q == 2) a.z = v; else a.w = v;
}

__global__ void __launch_bounds__(128)
k_divergence_f32v(Geo g, const float *__restrict__ u_, const float *__restrict__ v_, const float *__restrict__ w_,
                  float *b, float inv_scale, float ihx_t, float ihy_t, float ihz_t, ff ihx, ff ihy, ff ihz,
                  double *dmax, float v_lo, const float *__restrict__ v_hi) {
  pdl_wait();
  const int q4 = g.nx >> 2;
  const int t = blockIdx.x * blockDim.x + threadIdx.x;
  const int j = blockIdx.y;
  float mx = 0.f;
  if (t < q4 * g.nz) {
    const int k = t / q4, i0 = 4 * (t - k * q4);
    const size_t pl = (size_t)g.nx * g.nz;
    const size_t at = (size_t)j * pl + (size_t)k * g.nx + i0;
    const float4 uc = ld4(u_ + at);
    const float uE = u_[at - i0 + (i0 + 4 == g.nx ? 0 : i0 + 4)];
    const float4 vs = j == 0 ? make_float4(v_lo, v_lo, v_lo, v_lo) : ld4(v_ + at);
    const float4 vn = j + 1 >= g.ny ? (v_hi ? ld4(v_hi + (size_t)k * g.nx + i0) : make_float4(0.f, 0.f, 0.f, 0.f))
                                    : ld4(v_ + at + pl);
    const float4 wb = ld4(w_ + at);
    const float4 wt = ld4(w_ + at + (k + 1 == g.nz ? -(long)(g.nz - 1) * g.nx : (long)g.nx));
    float4 out;
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const float ue = q < 3 ? comp4(uc, q + 1) : uE, uw = comp4(uc, q);
      const float vnq = comp4(vn, q), vsq = comp4(vs, q), wtq = comp4(wt, q), wbq = comp4(wb, q);
      set4(out, q, ((ue - uw) * ihx_t + (vnq - vsq) * ihy_t + (wtq - wbq) * ihz_t) * inv_scale);
      if (dmax) mx = fmaxf(mx, DivExact<float>::eval(ue, uw, vnq, vsq, wtq, wbq, ihx, ihy, ihz));
    }
    if (b) *reinterpret_cast<float4 *>(b + at) = out;
  }
  if (dmax) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
    if ((threadIdx.x & 31) == 0) atomic_max_nonneg(dmax, (double)mx);
  }
}

__global__ void __launch_bounds__(128)
k_project_f32v(Geo g, float *__restrict__ u, float *__restrict__ v, float *__restrict__ w, float *__restrict__ p,
               const float *__restrict__ phi, float kproj, float cvisc, float v_lo) {
  pdl_wait();
  const int q4 = g.nx >> 2;
  const int t = blockIdx.x * blockDim.x + threadIdx.x;
  const int j = blockIdx.y;
  if (t >= q4 * g.nz) return;
  const int k = t / q4, i0 = 4 * (t - k * q4);
  const size_t pl = (size_t)g.nx * g.nz;
  const size_t at = (size_t)j * pl + (size_t)k * g.nx + i0;
  const float ihx = (float)g.ihx, ihy = (float)g.ihy, ihz = (float)g.ihz;
  const float4 f0 = ld4(phi + at);
  const float fW = phi[at - i0 + (i0 == 0 ? g.nx - 1 : i0 - 1)];
  const float fE = phi[at - i0 + (i0 + 4 == g.nx ? 0 : i0 + 4)];
  const float4 fs = ld4(phi + at + (k == 0 ? (long)(g.nz - 1) * g.nx : -(long)g.nx));
  const float4 fn = ld4(phi + at + (k + 1 == g.nz ? -(long)(g.nz - 1) * g.nx : (long)g.nx));
  const float4 fd = j > 0 ? ld4(phi + at - pl) : f0;
  const float4 fu = j + 1 < g.ny ? ld4(phi + at + pl) : f0;
  float4 uu = ld4(u + at), vv = ld4(v + at), ww = ld4(w + at), pp = ld4(p + at);
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    const float c0 = comp4(f0, q);
    const float fw = q == 0 ? fW : comp4(f0, q - 1), fe = q < 3 ? comp4(f0, q + 1) : fE;
    const float fsq = comp4(fs, q), fnq = comp4(fn, q), fdq = comp4(fd, q), fuq = comp4(fu, q);
    set4(uu, q, comp4(uu, q) - kproj * (c0 - fw) * ihx);
    set4(ww, q, comp4(ww, q) - kproj * (c0 - fsq) * ihz);
    set4(vv, q, j > 0 ? comp4(vv, q) - kproj * (c0 - fdq) * ihy : v_lo);
    const float lap = (fe - 2 * c0 + fw) * ihx * ihx + (fnq - 2 * c0 + fsq) * ihz * ihz + (fuq - 2 * c0 + fdq) * ihy * ihy;
    set4(pp, q, comp4(pp, q) + (c0 - cvisc * lap));
  }
  *reinterpret_cast<float4 *>(u + at) = uu;
  *reinterpret_cast<float4 *>(v + at) = vv;
  *reinterpret_cast<float4 *>(w + at) = ww;
  *reinterpret_cast<float4 *>(p + at) = pp;
}

// E2 / E3 launches: the four-point FP32 kernels, the one-point kernels for FP64.
template <typename T>
static cudaError_t launch_divergence(const Geo &g, const Launch3 &L3, const T *u, const T *v, const T *w, T *b,
                                     double inv_scale, const ff &fx, const ff &fy, const ff &fz, double *dmax, T v_lo,
                                     const T *v_hi, cudaStream_t st) {
  if constexpr (sizeof(T) == 4) {
    const dim3 grid((unsigned)ceil_div(g.nz * (g.nx / 4), 128), (unsigned)g.ny);
    return launch_pdl(k_divergence_f32v, grid, dim3(128), 0, st, g, u, v, w, b, (float)inv_scale, (float)g.ihx,
                      (float)g.ihy, (float)g.ihz, fx, fy, fz, dmax, v_lo, v_hi);
  } else {
    return launch_pdl(k_divergence<T>, L3.grid, L3.block, 0, st, g, u, v, w, b, (T)inv_scale, (T)g.ihx, (T)g.ihy,
                      (T)g.ihz, fx, fy, fz, dmax, v_lo, v_hi);
  }
}
template <typename T>
static cudaError_t launch_project(const Geo &g, const Launch3 &L3, T *u, T *v, T *w, T *p, const T *phi, double kproj,
                                  double cvisc, T v_lo, cudaStream_t st) {
  if constexpr (sizeof(T) == 4) {
    const dim3 grid((unsigned)ceil_div(g.nz * (g.nx / 4), 128), (unsigned)g.ny);
    return launch_pdl(k_project_f32v, grid, dim3(128), 0, st, g, u, v, w, p, phi, (float)kproj, (float)cvisc, v_lo);
  } else {
    return launch_pdl(k_project<T>, L3.grid, L3.block, 0, st, g.nx, g.ny, g.nz, u, v, w, p, phi, (T)(kproj * g.ihx),
                      (T)(kproj * g.ihy), (T)(kproj * g.ihz), (T)(cvisc * g.ihx * g.ihx), (T)(cvisc * g.ihy * g.ihy),
                      (T)(cvisc * g.ihz * g.ihz), v_lo);
  }
}

// Outlet condition of the inflow-outflow configuration (Sec. 3):
// d phi/dt + C d phi/dy = 0 at y = Ly, advanced over the stage step
// (alpha + beta) dt by first-order upwinding from the last interior value
// (cu = step C / (hy/2) for u, w at the wall, cv = step C / hy for v's outlet
// face).  Also stores v = v_in on the inflow face (plane 0 of v) and writes
// each CTA's FP64 sum of the new outlet v to part[blockIdx.x] (fixed-order
// tree, so the total is reproducible).
constexpr int kOutT = 256;
template <typename T>
__global__ void __launch_bounds__(kOutT)
k_outflow_update(int ncol, const T *__restrict__ ul, const T *__restrict__ vl, const T *__restrict__ wl, T *uo,
                 T *vo, T *wo, T *v0, T cu, T cv, T v_in, double *part) {
  pdl_wait();
  __shared__ double ws[kOutT / 32];
  const int col = blockIdx.x * kOutT + threadIdx.x;
  double s = 0.0;
  if (col < ncol) {
    uo[col] -= cu * (uo[col] - ul[col]);
    wo[col] -= cu * (wo[col] - wl[col]);
    const T vn = vo[col] - cv * (vo[col] - vl[col]);
    vo[col] = vn;
    v0[col] = v_in;
    s = (double)vn;
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  if ((threadIdx.x & 31) == 0) ws[threadIdx.x >> 5] = s;
  __syncthreads();
  if (threadIdx.x == 0) {
    double t = 0.0;
#pragma unroll
    for (int q = 0; q < kOutT / 32; ++q) t += ws[q];
    part[blockIdx.x] = t;
  }
}

// Global mass balance: the outlet v is shifted by a constant so that its
// mean equals v_in (outflow = inflow; the Poisson right-hand side then has
// zero mean).  Every CTA sums the nparts partial sums in the same order.
template <typename T>
__global__ void __launch_bounds__(kOutT)
k_outflow_shift(int ncol, T *vo, double v_in, const double *__restrict__ part, int nparts, double inv_ncol) {
  pdl_wait();
  __shared__ double ws[kOutT / 32];
  __shared__ double shift;
  double s = 0.0;
  for (int q = threadIdx.x; q < nparts; q += kOutT) s += part[q];
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  if ((threadIdx.x & 31) == 0) ws[threadIdx.x >> 5] = s;
  __syncthreads();
  if (threadIdx.x == 0) {
    double t = 0.0;
#pragma unroll
    for (int q = 0; q < kOutT / 32; ++q) t += ws[q];
    shift = v_in - t * inv_ncol;
  }
  __syncthreads();
  const int col = blockIdx.x * kOutT + threadIdx.x;
  if (col < ncol) vo[col] = (T)((double)vo[col] + shift);
}

static ff ff_host(double v) {
  ff r;
  r.hi = (float)v;
  r.lo = (float)(v - (double)r.hi);
  return r;
}

static int ensure_substep_buffers(ibm_plan_s *p, int nmk) {
  for (int q = 0; q < 4; ++q) {
    if (!p->sub[q]) {
      cudaError_t e = cudaMalloc(&p->sub[q], p->npts * p->esz);
      if (e != cudaSuccess) { p->sub[q] = nullptr; return cuda_error(e, "substep workspace"); }
      p->bytes += p->npts * p->esz;
    }
  }
  const size_t need = (size_t)nmk * 3 * p->esz;
  if (need > p->mkcap) {
    if (p->mkbuf) { cudaFree(p->mkbuf); p->bytes -= p->mkcap; p->mkbuf = nullptr; p->mkcap = 0; }
    cudaError_t e = cudaMalloc(&p->mkbuf, need);
    if (e != cudaSuccess) { p->mkbuf = nullptr; return cuda_error(e, "marker workspace"); }
    p->mkcap = need;
    p->bytes += need;
  }
  return IBM_OK;
}

template <typename T>
static int substep_t(ibm_plan_s *p, ibm_state *s, const ibm_inout *io, int stage, double dt, double nu,
                     ibm_markers *mk, cudaStream_t st, ibm_info *info) {
  const int n = stage - 1;
  const double a = kAlpha[n], b = kBeta[n], gm = kGamma[n], zt = kZeta[n];
  const double ab = a + b;
  const double cH = b * dt * nu;  // Helmholtz coefficient of Eq. 2e
  const int nmk = mk ? mk->n : 0;
  int rc = ensure_substep_buffers(p, nmk);
  if (rc) return rc;
  Geo g{p->nx, p->ny, p->nz, 1.0 / p->h[0], 1.0 / p->h[1], 1.0 / p->h[2]};
  T *u = (T *)s->u, *v = (T *)s->v, *w = (T *)s->w, *pr = (T *)s->p;
  T *du = (T *)p->sub[0], *dv = (T *)p->sub[1], *dw = (T *)p->sub[2], *phi = (T *)p->sub[3];
  T *rhs = (T *)p->bsave;
  const Launch3 L3 = stencil_launch(p->nx, p->ny, p->nz);
  InfoTrace trace(p, info != nullptr);
  if (info) {
    IBM_CUDA_TRY(cudaMemsetAsync(p->dsc + 8, 0, 2 * sizeof(double), st));
    IBM_CUDA_TRY(cudaEventRecord(p->ev0, st));
  }
  // inflow-outflow walls: outlet values advanced to the end of the stage
  // and made mass-conserving; they are the wall data of the whole stage
  const T v_lo = io ? (T)io->v_in : (T)0;
  T *uo = io ? (T *)io->u_out : nullptr, *vo = io ? (T *)io->v_out : nullptr, *wo = io ? (T *)io->w_out : nullptr;
  if (io) {
    ProfScope ps(p, IBM_K_OUTFLOW, st, 2);
    const int ncol = p->nx * p->nz, nparts = ceil_div(ncol, kOutT);
    const size_t last = (size_t)(p->ny - 1) * ncol;
    const double step = ab * dt;
    double *part = (double *)p->work;
    IBM_CUDA_TRY(launch_pdl(k_outflow_update<T>, dim3(nparts), dim3(kOutT), 0, st, ncol, (const T *)(u + last),
                            (const T *)(v + last), (const T *)(w + last), uo, vo, wo, v,
                            (T)(step * io->c_out * 2.0 * g.ihy), (T)(step * io->c_out * g.ihy), v_lo, part));
    IBM_CUDA_TRY(launch_pdl(k_outflow_shift<T>, dim3(nparts), dim3(kOutT), 0, st, ncol, vo, io->v_in,
                            (const double *)part, nparts, 1.0 / ncol));
  }
  // E1
  {
    ProfScope ps(p, IBM_K_EXPLICIT, st);
    if (io)
      IBM_CUDA_TRY((launch_explicit<T, true>(g, u, v, w, pr, (T *)s->Nu, (T *)s->Nv, (T *)s->Nw, du, dv, dw, ab * nu,
                                             ab, gm, zt, dt, v_lo, uo, vo, wo, st)));
    else
      IBM_CUDA_TRY((launch_explicit<T, false>(g, u, v, w, pr, (T *)s->Nu, (T *)s->Nv, (T *)s->Nw, du, dv, dw, ab * nu,
                                              ab, gm, zt, dt, (T)0, nullptr, nullptr, nullptr, st)));
  }
  // L2 + L1
  if (nmk > 0) {
    T *F = mk->F ? (T *)mk->F : (T *)p->mkbuf;
    {
      // L2 (rigid marker motion at the stage start time) fused with L1's
      // interpolation and force
      ProfScope ps(p, IBM_K_INTERP, st);
      IBM_CUDA_TRY(launch_interp<T>(p, nmk, (const T *)mk->X, u, v, w, du, dv, dw, nullptr, (const T *)mk->Ud,
                                    1.0 / dt, F, (const T *)mk->X0, (T *)mk->X, (T *)mk->Ud, mk->motion, mk->params,
                                    s->t, st));
    }
    {
      ProfScope ps(p, IBM_K_SPREAD, st);
      IBM_CUDA_TRY(launch_spread<T>(p, nmk, (const T *)mk->X, F, (const T *)mk->dV, du, dv, dw, dt, st));
    }
  }
  // S1: Helmholtz, increment form, u* written over u; the three components
  // go through the same launches
  {
    const int bcs[3] = {IBM_FIELD_CELL_DIRICHLET, IBM_FIELD_FACE_DIRICHLET, IBM_FIELD_CELL_DIRICHLET};
    const void *in3[3] = {du, dv, dw};
    void *out3[3] = {u, v, w};
    const void *add3[3] = {u, v, w};
    if ((rc = plan_solve_fields(p, cH, 3, bcs, in3, out3, add3, st))) return rc;
  }
  // E2
  const ff fx = ff_host(g.ihx), fy = ff_host(g.ihy), fz = ff_host(g.ihz);
  {
    ProfScope ps(p, IBM_K_DIVERGENCE, st);
    IBM_CUDA_TRY(launch_divergence<T>(g, L3, u, v, w, rhs, 1.0 / (ab * dt), fx, fy, fz, info ? p->dsc + 9 : nullptr,
                                      v_lo, (const T *)vo, st));
  }
  // S2
  if ((rc = plan_solve(p, 0, 0.0, 0, rhs, phi, nullptr, st, nullptr))) return rc;
  // E3
  {
    ProfScope ps(p, IBM_K_PROJECT, st);
    IBM_CUDA_TRY(launch_project<T>(g, L3, u, v, w, pr, phi, ab * dt, cH, v_lo, st));
  }
  if (info) {
    IBM_CUDA_TRY(cudaEventRecord(p->ev1, st));
    IBM_CUDA_TRY(launch_divergence<T>(g, L3, u, v, w, (T *)nullptr, 1.0, fx, fy, fz, p->dsc + 8, v_lo,
                                      (const T *)vo, st));
    IBM_CUDA_TRY(cudaMemcpyAsync(p->hsc, p->dsc, 16 * sizeof(double), cudaMemcpyDeviceToHost, st));
    IBM_CUDA_TRY(cudaStreamSynchronize(st));
    float ms = 0.f;
    IBM_CUDA_TRY(cudaEventElapsedTime(&ms, p->ev0, p->ev1));
    trace.read(info->phase_ms);
    if ((rc = plan_status(p, st))) return rc;
    info->rel_residual = -1.0;
    info->removed_mean = p->hsc[0];
    info->div_max = p->hsc[8];
    info->div_before = p->hsc[9];
    info->t_ms = ms;
    info->refine_iters = p->precision == IBM_FP32_REFINED ? p->refine : 0;
  }
  s->t += ab * dt;
  return IBM_OK;
}

}  // namespace ibm

using namespace ibm;

static int substep_entry(ibm_plan plan, ibm_state *st, const ibm_inout *io, int rk_stage, double dt, double nu,
                         ibm_markers *mk, void *stream, ibm_info *info) {
  if (!plan || !st) return set_error(IBM_ERR_ARG, "ibm_substep: NULL plan or state");
  if (plan->bc != IBM_BC_PXZ_WALL_Y)
    return set_error(IBM_ERR_UNSUPPORTED, "ibm_substep: the RK stage is built for the wall-bounded branch only");
  if (rk_stage < 1 || rk_stage > 3) return set_error(IBM_ERR_ARG, "ibm_substep: rk_stage %d", rk_stage);
  if (!(dt > 0) || !std::isfinite(dt) || !(nu > 0) || !std::isfinite(nu))
    return set_error(IBM_ERR_ARG, "ibm_substep: dt and nu must be finite and > 0");
  void *fields[] = {st->u, st->v, st->w, st->p, st->Nu, st->Nv, st->Nw};
  for (void *f : fields)
    if (!f || !aligned_to(f, 16)) return set_error(IBM_ERR_ARG, "ibm_substep: NULL or non-16-byte-aligned field");
  if (mk && mk->n > 0) {
    if (!mk->X0 || !mk->dV || !mk->X || !mk->Ud)
      return set_error(IBM_ERR_ARG, "ibm_substep: markers need X0, dV, X and Ud");
    if (mk->motion < IBM_MOTION_STATIC || mk->motion > IBM_MOTION_HEAVE)
      return set_error(IBM_ERR_ARG, "ibm_substep: motion %d", mk->motion);
    if (mk->motion == IBM_MOTION_HEAVE && !(mk->params[1] > 0))
      return set_error(IBM_ERR_ARG, "ibm_substep: heave period must be > 0");
    if (mk->n > (1 << 26)) return set_error(IBM_ERR_ARG, "ibm_substep: too many markers");
  } else if (mk && mk->n < 0) {
    return set_error(IBM_ERR_ARG, "ibm_substep: negative marker count");
  }
  if (io) {
    if (!std::isfinite(io->v_in) || !std::isfinite(io->c_out) || io->c_out < 0)
      return set_error(IBM_ERR_ARG, "ibm_substep_inout: v_in must be finite and c_out finite and >= 0");
    const void *planes[] = {io->u_out, io->v_out, io->w_out};
    for (const void *f : planes)
      if (!f || !aligned_to(f, 16))
        return set_error(IBM_ERR_ARG, "ibm_substep_inout: NULL or non-16-byte-aligned outlet plane");
  }
  if (plan->precision == IBM_FP64)
    return substep_t<double>(plan, st, io, rk_stage, dt, nu, mk, (cudaStream_t)stream, info);
  return substep_t<float>(plan, st, io, rk_stage, dt, nu, mk, (cudaStream_t)stream, info);
}

namespace ibm {
double stage_time_advance(int rk_stage, double dt) { return (kAlpha[rk_stage - 1] + kBeta[rk_stage - 1]) * dt; }

int substep_checked(ibm_plan_s *p, ibm_state *st, int rk_stage, double dt, double nu, ibm_markers *mk,
                    cudaStream_t stream) {
  return substep_entry(p, st, nullptr, rk_stage, dt, nu, mk, stream, nullptr);
}

int prepare_substep(ibm_plan_s *p, int nmk) {
  int rc = ensure_substep_buffers(p, nmk);
  if (rc) return rc;
  for (int b = 0; b < 2; ++b) {  // the spectra of the stage's three-field Helmholtz launches
    if (!p->Sx[b] && !p->use_slab_fields) {
      cudaError_t e = cudaMalloc(&p->Sx[b], p->nspec * 2 * p->esz);
      if (e != cudaSuccess) { p->Sx[b] = nullptr; return cuda_error(e, "field spectrum"); }
      p->bytes += p->nspec * 2 * p->esz;
    }
  }
  return IBM_OK;
}
}  // namespace ibm

extern "C" int ibm_substep(ibm_plan plan, ibm_state *st, int rk_stage, double dt, double nu, ibm_markers *mk,
                           void *stream, ibm_info *info) {
  return substep_entry(plan, st, nullptr, rk_stage, dt, nu, mk, stream, info);
}

extern "C" int ibm_substep_inout(ibm_plan plan, ibm_state *st, const ibm_inout *io, int rk_stage, double dt,
                                 double nu, ibm_markers *mk, void *stream, ibm_info *info) {
  if (!io) return set_error(IBM_ERR_ARG, "ibm_substep_inout: NULL inflow-outflow data");
  return substep_entry(plan, st, io, rk_stage, dt, nu, mk, stream, info);
}
