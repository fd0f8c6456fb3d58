// stencil.cu -- 7-point residual of the Poisson / Helmholtz operators.
//
// r = b - (sigma x + tau L_h x), L_h the second-order central Laplacian of
// Sec. 2.1 with periodic x, z and the ghost rule of the field's wall kind
// along y (Appendix B; periodic for the triply periodic branch).  Poisson:
// sigma = 0, tau = 1; Helmholtz (I - c L):
// sigma = 1, tau = -c.  In FP32 the second differences of the stored values
// are taken exactly (hi + lo) and the other terms, all O(|b|), are summed in
// FP32 (residual_point below): a plain FP32 stencil would lose the residual
// in the cancelling second differences.  Optionally the
// FP64 sums of r^2, b^2, r and b are accumulated for the relative residual.
// An optional device scalar is subtracted from b first (the Poisson
// right-hand side's removed mean), so the residual is that of the compatible
// system.
#include <algorithm>
#include <mutex>

#include "stencil.cuh"

namespace ibm {

// Four consecutive x points per thread, marching up jc planes of y: the planes
// below and above a point are registers that move down, so x is read from
// beyond L1 about once (three times with a thread a plane), and the next plane
// of x and b is on its way while a plane is computed.  Grid (ceil(nz nx / 4 /
// 128), ceil(ny / jc)), 128 threads.  Bound by HBM: 512 x 256 x 256 75 -> 67.5 us
// (6.0 TB/s), 384 x 200 x 192 36 -> 31.6 us.
template <int BC, bool SIGMA>
__global__ void __launch_bounds__(128)
k_residual_f32v(ResidualArgs A, const float *__restrict__ b, const float *__restrict__ x, float *__restrict__ r,
                double *norms, int jc) {
  pdl_wait();
  const int q = A.nx >> 2;
  const int t = blockIdx.x * blockDim.x + threadIdx.x;
  const int ja = blockIdx.y * jc, je = min(A.ny, ja + jc);
  double r2 = 0.0, b2 = 0.0, r1 = 0.0, b1 = 0.0;
  if (t < q * A.nz) {
    const int k = t / q, i0 = 4 * (t - k * q);
    const size_t pl = (size_t)A.nx * A.nz;
    const int off = k * A.nx + i0;
    const int oW = i0 == 0 ? A.nx - 1 : -1, oE = i0 + 4 == A.nx ? 4 - A.nx : 4;
    const int dn = k + 1 == A.nz ? -(A.nz - 1) * A.nx : A.nx, ds = k == 0 ? (A.nz - 1) * A.nx : -A.nx;
    const float4 zero = make_float4(0.f, 0.f, 0.f, 0.f);
    float2 m = make_float2(0.f, 0.f);
    if (A.boff) m = *reinterpret_cast<const float2 *>(A.boff + 1);
    // plane jj of x at the four points (walls: 0 for the faces; the ghost kinds take theirs from x0 below)
    auto plane_of = [&](int jj) {
      if (BC == BC_PERIODIC) jj = jj < 0 ? jj + A.ny : jj >= A.ny ? jj - A.ny : jj;
      const bool in = jj >= (BC == BC_FACE_DIRICHLET ? 1 : 0) && jj < A.ny;
      return in ? *reinterpret_cast<const float4 *>(x + jj * pl + off) : zero;
    };
    constexpr float gs = BC == BC_NEUMANN ? 1.0f : -1.0f;
    constexpr bool ghost = BC == BC_NEUMANN || BC == BC_CELL_DIRICHLET;
    float4 xd = plane_of(ja - 1), x0 = plane_of(ja), xu = plane_of(ja + 1);
    float4 bv = *reinterpret_cast<const float4 *>(b + ja * pl + off);
    for (int j = ja; j < je; ++j) {
      const float *xc = x + j * pl + off;
      const float xW = xc[oW], xE = xc[oE];
      const float4 xn = *reinterpret_cast<const float4 *>(xc + dn);
      const float4 xs = *reinterpret_cast<const float4 *>(xc + ds);
      float4 xnext = zero, bnext = zero;
      if (j + 1 < je) {
        xnext = plane_of(j + 2);
        bnext = *reinterpret_cast<const float4 *>(b + (j + 1) * pl + off);
      }
      float4 lo = xd, hi = xu, res = zero, bt = zero;
      if (ghost && j == 0) lo = make_float4(gs * x0.x, gs * x0.y, gs * x0.z, gs * x0.w);
      if (ghost && j + 1 == A.ny) hi = make_float4(gs * x0.x, gs * x0.y, gs * x0.z, gs * x0.w);
      if (BC != BC_FACE_DIRICHLET || j > 0) {
        res.x = residual_point<SIGMA>(A, bv.x, m, x0.x, x0.y, xW, xn.x, xs.x, hi.x, lo.x, bt.x);
        res.y = residual_point<SIGMA>(A, bv.y, m, x0.y, x0.z, x0.x, xn.y, xs.y, hi.y, lo.y, bt.y);
        res.z = residual_point<SIGMA>(A, bv.z, m, x0.z, x0.w, x0.y, xn.z, xs.z, hi.z, lo.z, bt.z);
        res.w = residual_point<SIGMA>(A, bv.w, m, x0.w, xE, x0.z, xn.w, xs.w, hi.w, lo.w, bt.w);
      }
      if (norms) residual4_norms(res, bt, r2, b2, r1, b1);
      *reinterpret_cast<float4 *>(r + j * pl + off) = res;
      xd = x0; x0 = xu; xu = xnext; bv = bnext;
    }
  }
  if (norms) block_accumulate(r2, b2, r1, b1, norms);
}

__global__ void __launch_bounds__(128)
k_residual_f64(ResidualArgs A, const double *__restrict__ b, const double *__restrict__ x,
               double *__restrict__ r, double *norms) {
  pdl_wait();
  int i, k, j;
  const bool inside = stencil_index(A.nx, A.nz, i, k, j);
  const size_t idx = ((size_t)j * A.nz + k) * A.nx + i;
  double rr = 0.0, bb = 0.0;
  if (inside) {
    const size_t row = (size_t)A.nx;
    const size_t pl = (size_t)A.nx * A.nz;
    const double bv = A.boff ? b[idx] - *A.boff : b[idx];
    double res;
    if (A.bc == BC_FACE_DIRICHLET && j == 0) {
      res = 0.0;
    } else {
      const double x0 = x[idx];
      const double xe = x[idx - i + (i + 1 == A.nx ? 0 : i + 1)];
      const double xw = x[idx - i + (i == 0 ? A.nx - 1 : i - 1)];
      const size_t rowbase = idx - (size_t)k * row;
      const double xn = x[rowbase + (size_t)(k + 1 == A.nz ? 0 : k + 1) * row];
      const double xs = x[rowbase + (size_t)(k == 0 ? A.nz - 1 : k - 1) * row];
      double xu, xd;
      if (A.bc == BC_FACE_DIRICHLET) {
        xd = (j - 1 >= 1) ? x[idx - pl] : 0.0;
        xu = (j + 1 <= A.ny - 1) ? x[idx + pl] : 0.0;
      } else if (A.bc == BC_PERIODIC) {
        xd = j > 0 ? x[idx - pl] : x[idx + (size_t)(A.ny - 1) * pl];
        xu = j + 1 < A.ny ? x[idx + pl] : x[idx - (size_t)(A.ny - 1) * pl];
      } else {
        const double gsign = (A.bc == BC_NEUMANN) ? 1.0 : -1.0;
        xd = (j > 0) ? x[idx - pl] : gsign * x0;
        xu = (j + 1 < A.ny) ? x[idx + pl] : gsign * x0;
      }
      const double L = (xe + xw - 2.0 * x0) * A.cxd + (xn + xs - 2.0 * x0) * A.czd + (xu + xd - 2.0 * x0) * A.cyd;
      res = bv - A.sigmad * x0 - A.taud * L;
    }
    r[idx] = res;
    rr = res;
    bb = (A.bc == BC_FACE_DIRICHLET && j == 0) ? 0.0 : bv;
  }
  if (norms) block_accumulate(rr * rr, bb * bb, rr, bb, norms);
}


template <int BC, bool SIGMA>
static cudaError_t launch_residual_f32(const ResidualArgs &A, const float *b, const float *x, float *r, double *norms,
                                       cudaStream_t st) {
  // Planes a CTA marches: the fewest that let every CTA be resident at once,
  // if that is at most 32, else 8 (384 x 200 x 192: 24 planes, one wave, 31.6 us,
  // 16 planes, 1.6 waves, 34.1; 512 x 256 x 256: 8 planes 67.5 us, 16 70.9, 32 69.9).
  static std::once_flag once;
  static int slots = 0;
  std::call_once(once, [] {
    int dev = 0, sms = 0, per_sm = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_residual_f32v<BC, SIGMA>, 128, 0);
    slots = sms * std::max(per_sm, 1);
  });
  const int cols = ceil_div(A.nz * (A.nx / 4), 128);
  const int one = ceil_div(A.ny, std::max(1, slots / cols));
  const int jc = one <= 32 ? one : 8;
  IBM_KTRY(launch_pdl(k_residual_f32v<BC, SIGMA>, dim3((unsigned)cols, (unsigned)ceil_div(A.ny, jc)), 128, 0, st, A, b,
                      x, r, norms, jc));
  return cudaGetLastError();
}

template <>
cudaError_t launch_residual<float>(int nx, int ny, int nz, const StencilCoef &c, const float *b, const float *x,
                                   float *r, const double *boff, double *norms, cudaStream_t st) {
  if (nx % 4 != 0 || ((uintptr_t)b | (uintptr_t)x | (uintptr_t)r) & 15u) return cudaErrorInvalidValue;
  const ResidualArgs A = make_args(nx, ny, nz, c, boff);
  const bool sg = c.sigma != 0.0;
#define IBM_RES_BC(B)                                                                             \
  case B:                                                                                         \
    return sg ? launch_residual_f32<B, true>(A, b, x, r, norms, st) : launch_residual_f32<B, false>(A, b, x, r, norms, st);
  switch (c.bc) {
    IBM_RES_BC(BC_NEUMANN)
    IBM_RES_BC(BC_CELL_DIRICHLET)
    IBM_RES_BC(BC_FACE_DIRICHLET)
    IBM_RES_BC(BC_PERIODIC)
    default: return cudaErrorInvalidValue;
  }
#undef IBM_RES_BC
}

// Wall data's share of the 7-point operator, moved to the right-hand side
// (Appendix B: the first and last rows of each pencil carry the boundary
// values; BC2.2 forms the same terms from the FFT of the ghost planes): dst =
// src, with clo g_lo added to plane jlo and chi g_hi to plane jhi (either g may
// be NULL).  16 bytes per thread; nx % 4 == 0, so no thread straddles planes.
// (A copy and a launch over the two planes took 7 us at 192 x 129 x 96: solve 56.5 -> 52.2 us.)
template <typename T>
__global__ void __launch_bounds__(256)
k_wall_rhs(size_t nvec, const T *__restrict__ src, T *__restrict__ dst, int vplane, int jlo, int jhi,
           const T *__restrict__ glo, const T *__restrict__ ghi, T clo, T chi) {
  constexpr int V = 16 / sizeof(T);
  struct alignas(16) Vec { T v[V]; };
  pdl_wait();
  const size_t e = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= nvec) return;
  Vec x = reinterpret_cast<const Vec *>(src)[e];
  auto add = [&](const T *g, int j, T c) {
    const size_t e0 = (size_t)j * vplane;
    if (g && e >= e0 && e < e0 + vplane) {
      const Vec w = reinterpret_cast<const Vec *>(g)[e - e0];
#pragma unroll
      for (int q = 0; q < V; ++q) x.v[q] += c * w.v[q];
    }
  };
  add(glo, jlo, clo);
  add(ghi, jhi, chi);
  reinterpret_cast<Vec *>(dst)[e] = x;
}

template <typename T>
cudaError_t launch_wall_rhs(int nx, int ny, int nz, const T *src, T *dst, int jlo, int jhi, const T *glo, const T *ghi,
                            double clo, double chi, cudaStream_t st) {
  constexpr int V = 16 / sizeof(T);
  const int vplane = nx * nz / V;
  const size_t nvec = (size_t)vplane * ny;
  IBM_KTRY(launch_pdl(k_wall_rhs<T>, (unsigned)((nvec + 255) / 256), 256, 0, st, nvec, src, dst, vplane, jlo, jhi, glo,
                      ghi, (T)clo, (T)chi));
  return cudaGetLastError();
}
template cudaError_t launch_wall_rhs<float>(int, int, int, const float *, float *, int, int, const float *,
                                            const float *, double, double, cudaStream_t);
template cudaError_t launch_wall_rhs<double>(int, int, int, const double *, double *, int, int, const double *,
                                             const double *, double, double, cudaStream_t);

template <>
cudaError_t launch_residual<double>(int nx, int ny, int nz, const StencilCoef &c, const double *b, const double *x,
                                    double *r, const double *boff, double *norms, cudaStream_t st) {
  const Launch3 L = stencil_launch(nx, ny, nz);
  IBM_KTRY(launch_pdl(k_residual_f64, L.grid, L.block, 0, st, make_args(nx, ny, nz, c, boff), b, x, r, norms));
  return cudaGetLastError();
}

}  // namespace ibm
