// transforms.cu -- Fourier transforms along the two periodic axes (x, z).
//
// The paper's doubly periodic branch (Sec. 2.3.3, S1.1/S2.1) feeds the
// pencil solver with the 2-D real FFT of the right-hand side over the
// periodic planes and inverts it afterwards (S1.2/S2.2).  Here each y-plane
// [nz][nx] (real) maps to a spectrum plane [nz][nx/2+1] (complex, kx
// fastest), unnormalised forward and scaled by 1/(nx nz) on the way back.
//
// Real rows are transformed in pairs: rows a and b form z = a + i b, one
// complex FFT of length nx gives Z, and A_k = (Z_k + conj Z_{N-k})/2,
// B_k = -i (Z_k - conj Z_{N-k})/2 for k = 0..nx/2.  The inverse rebuilds
// Z_k = A_k + i B_k from the two Hermitian half spectra.
//
// Three kernel families, chosen per plan by its plane mode:
//   plane kernels   (mode 1, plane.cuh) one CTA per y-plane: the x transform
//                   of every row pair lands in a shared-memory plane, the z
//                   transform of every column leaves it; one HBM read and
//                   one write per direction;
//   axis kernels    (mode 0, axis.cu) x-rows and z-columns in two passes;
//   cluster kernels (modes 2, 4, 8, cplane.cu) C CTAs per plane.
// Plane and axis kernels run the two-step register transform of fft2.cuh.  This
// file holds the choice between them.
#include <algorithm>
#include <mutex>

#include "plane.cuh"

namespace ibm {

// --------------------------------------------------------------------------
// dispatch
// --------------------------------------------------------------------------
#define IBM_FOR_EACH_N(X) X(8) X(12) X(16) X(24) X(32) X(48) X(64) X(96) X(128) X(192) X(256) X(384) X(512)

// FP64 plane kernels (the tuner's; FP32: plane.cuh)
#define IBM_PLANE_SHAPES(X)                                                    \
  X(8, 8) X(12, 12) X(16, 16) X(24, 24) X(32, 32) X(48, 48) X(64, 64) X(96, 96) \
  X(128, 128) X(192, 192) X(256, 128) X(128, 256) X(64, 128) X(128, 64)

template <typename T> static bool plane_supported(int nx, int nz) {
  if constexpr (sizeof(T) == 4) {
#define X(N) if (nx == N) return plane_dispatch<N>(nz, [](auto) {}, PlaneLengths{});
    IBM_FOR_EACH_N(X)
#undef X
  } else {
#define X(a, b) if (nx == a && nz == b) return PlaneCfg<T, a, b>::ok;
    IBM_PLANE_SHAPES(X)
#undef X
  }
  return false;
}

static cudaError_t plane_forward(const TransformGeom &g, Ptr3<const float *> in, Ptr3<float2 *> S, const float2 *twx,
                                 const float2 *twz, const PlaneResidual &res, cudaStream_t st) {
#define X(N) if (g.nx == N) return plane_forward_f32<N>(g, in, S, twx, twz, res, st);
  IBM_FOR_EACH_N(X)
#undef X
  return cudaErrorNotSupported;
}

template <typename T>
cudaError_t launch_forward(const TransformGeom &g, Ptr3<const T *> in, Ptr3<cplx<T> *> S, const cplx<T> *twx,
                           const cplx<T> *twz, cudaStream_t st) {
  const int nx = g.nx, ny = g.ny, nz = g.nz;
  if constexpr (sizeof(T) == 4) {
    if (g.use_plane == kPlaneDft && g.dft_fwd) return launch_dft_forward(g, in, S, st);
  }
  if (g.use_plane >= 2 && cplane_supported<T>(nx, nz, g.use_plane))
    return launch_cplane_forward<T>(g, g.use_plane, in, S, twx, twz, st);
  if (g.use_plane == 1 && plane_supported<T>(nx, nz)) {
    if constexpr (sizeof(T) == 4) {
      return plane_forward(g, in, S, twx, twz, PlaneResidual{}, st);
    } else {
#define X(a, b)                                                                                  \
  if (nx == a && nz == b) {                                                                      \
    if constexpr (PlaneCfg<T, a, b>::ok) {                                                       \
      { cudaError_t e = ensure_max_smem<k_plane_fwd<T, a, b>>(); if (e) return e; }              \
      IBM_KTRY(launch_pdl(k_plane_fwd<T, a, b>, dim3(ny, g.nb), PlaneCfg<T, a, b>::THREADS, PlaneCfg<T, a, b>::bytes, st, in, S, twx, twz, g.zrhs, PlaneResidual{})); \
      return cudaGetLastError();                                                                 \
    }                                                                                            \
  }
      IBM_PLANE_SHAPES(X)
#undef X
    }
  }
  // axis path: x rows then z columns
  return launch_axis_forward<T>(g, in, S, twx, twz, st);
}

bool plane_residual_fused(const TransformGeom &g) { return g.use_plane == 1 && plane_supported<float>(g.nx, g.nz); }

cudaError_t launch_plane_residual_forward(const TransformGeom &g, const StencilCoef &c, const float *b, const float *x,
                                          float2 *S, const float2 *twx, const float2 *twz, const double *boff,
                                          cudaStream_t st) {
  const PlaneResidual res{x, make_args(g.nx, g.ny, g.nz, c, boff)};
  return plane_forward(g, ptr3(b), ptr3(S), twx, twz, res, st);
}

template <typename T>
cudaError_t launch_inverse(const TransformGeom &g, Ptr3<cplx<T> *> S, Ptr3<T *> out, Ptr3<const T *> addend,
                           const cplx<T> *twx, const cplx<T> *twz, T scale, cudaStream_t st) {
  const int nx = g.nx, ny = g.ny, nz = g.nz;
  if constexpr (sizeof(T) == 4) {
    if (g.use_plane == kPlaneDft && g.dft_inv) return launch_dft_inverse(g, S, out, addend, scale, st);
  }
  if (g.use_plane >= 2 && cplane_supported<T>(nx, nz, g.use_plane))
    return launch_cplane_inverse<T>(g, g.use_plane, S, out, addend, twx, twz, scale, st);
  if (g.use_plane == 1 && plane_supported<T>(nx, nz)) {
    if constexpr (sizeof(T) == 4) {
#define X(N) if (nx == N) return plane_inverse_f32<N>(g, S, out, addend, twx, twz, scale, st);
      IBM_FOR_EACH_N(X)
#undef X
    } else {
#define X(a, b)                                                                                  \
  if (nx == a && nz == b) {                                                                      \
    if constexpr (PlaneCfg<T, a, b>::ok) {                                                       \
      { cudaError_t e = ensure_max_smem<k_plane_inv<T, a, b>>(); if (e) return e; }              \
      IBM_KTRY(launch_pdl(k_plane_inv<T, a, b>, dim3(ny, g.nb), PlaneCfg<T, a, b>::THREADS, PlaneCfg<T, a, b>::bytes, st, S, out, addend, twx, twz, (T)0.5 * scale, g.zsol)); \
      return cudaGetLastError();                                                                 \
    }                                                                                            \
  }
      IBM_PLANE_SHAPES(X)
#undef X
    }
  }
  return launch_axis_inverse<T>(g, S, out, addend, twx, twz, scale, st);
}

template cudaError_t launch_forward<float>(const TransformGeom &, Ptr3<const float *>, Ptr3<float2 *>, const float2 *,
                                           const float2 *, cudaStream_t);
template cudaError_t launch_forward<double>(const TransformGeom &, Ptr3<const double *>, Ptr3<double2 *>,
                                            const double2 *, const double2 *, cudaStream_t);
template cudaError_t launch_inverse<float>(const TransformGeom &, Ptr3<float2 *>, Ptr3<float *>, Ptr3<const float *>,
                                           const float2 *, const float2 *, float, cudaStream_t);
template cudaError_t launch_inverse<double>(const TransformGeom &, Ptr3<double2 *>, Ptr3<double *>,
                                            Ptr3<const double *>, const double2 *, const double2 *, double,
                                            cudaStream_t);

template <typename T> int transform_launches(const TransformGeom &g) {
  if (g.use_plane == kPlaneDft) return (sizeof(T) == 4 && g.dft_fwd) ? 1 : 2;
  if (g.use_plane >= 2) return cplane_supported<T>(g.nx, g.nz, g.use_plane) ? 1 : 2;
  return (g.use_plane == 1 && plane_supported<T>(g.nx, g.nz)) ? 1 : 2;
}
template int transform_launches<float>(const TransformGeom &);
template int transform_launches<double>(const TransformGeom &);

template <typename T> int plane_modes(int nx, int nz, int *modes) {
  int n = 0;
  if (sizeof(T) == 4 && dft_tc_supported(nx, nz)) modes[n++] = kPlaneDft;
  modes[n++] = 0;
  if (plane_supported<T>(nx, nz)) modes[n++] = 1;
  for (int c = 2; c <= 8; c *= 2)
    if (cplane_supported<T>(nx, nz, c)) modes[n++] = c;
  return n;
}
template int plane_modes<float>(int, int, int *);
template int plane_modes<double>(int, int, int *);

static int sm_count() {
  static std::once_flag once;
  static int sms = 0;
  std::call_once(once, [] {
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
      sms = 0;
  });
  return std::max(sms, 1);  // (without a device the plan is refused later)
}

// The last wave of n CTAs, one an SM, fills more than a third of the SMs.
static bool last_wave_filled(int n, int sms) {
  const int last = n % sms;
  return last == 0 || 20 * last >= 7 * sms;
}

template <typename T> int default_plane_mode(int nx, int ny, int nz) {
  // FP64 (arithmetic-bound) takes the split passes at every size, and so does
  // FP32 beyond the planes below.  The lines follow refined FP32 Poisson and
  // Helmholtz solves timed on GB300 (152 SMs) for every plane shape at 28 ny from 8
  // to 512, split passes against plane kernels with the residual in the forward
  // transform (us, Poisson):
  //   planes up to 128 x 128 (in place, two CTAs an SM or more) win by their
  //   launches (6 against 11) and, once they fill the SMs, by bytes: 48x33x24
  //   30.3 / 21.1, 96x16x96 30.5 / 29.9, 96x512x96 96.2 / 86.3, 128x80x128
  //   44.9 / 39.7, 128x512x128 153.5 / 133.0; not the few large planes that
  //   leave SMs idle: 128x33x128 34.0 / 38.6, 128x64x128 37.5 / 38.7,
  //   96x33x128 33.1 / 35.5;
  //   other small planes at any ny where the rows are short, with long rows up
  //   to one CTA an SM: 192x512x32 74.6 / 68.0, 256x128x32 38.0 / 31.0,
  //   256x512x32 77.4 / 91.6;
  //   other middle planes from about a third of the SMs on, and beyond one
  //   wave where the last one is not nearly empty: 48x56x192 39.5 / 33.9,
  //   64x153x192 57.0 / 63.8, 64x228x192 69.2 / 70.8, 64x256x192 71.4 / 69.2,
  //   64x305x192 90.1 / 96.9; 192x153x48 49.5 / 47.1 (short columns) and its
  //   like at every ny;
  //   other large planes (one CTA an SM) where their CTAs fill most of one
  //   wave, or of two with short rows: 192x80x96 46.0 / 43.5, 96x80x256 55.9 /
  //   59.6, 96x100x256 64.9 / 62.4, 256x100x96 55.0 / 59.2, 256x128x96 62.5 /
  //   59.7, 192x256x128 126.8 / 115.6, 192x512x128 241.4 / 266.6.
  if (sizeof(T) == 4 && plane_supported<T>(nx, nz)) {
    const int area = nx * nz, sms = sm_count();
    const bool one = ny <= sms;                                             // one wave
    const bool two = nx <= 192 && 19 * ny >= 30 * sms && ny <= 2 * sms;     // most of two
    if (nx <= 128 && nz <= 128) return area <= 9216 || (area <= 12288 ? 5 : 4) * ny >= 2 * sms;
    if (area <= 8192) return one || (nx <= 192 && nz <= 256);
    if (area <= 12288 && nx <= 192 && nz <= 192)
      return 11 * ny >= 4 * sms && (one || nz <= 48 || last_wave_filled(ny, sms));
    if (area <= kPlaneArea) {
      const bool most = area <= 18432 ? 19 * ny >= 10 * sms : nx <= 192 ? 9 * ny >= 5 * sms : 11 * ny >= 8 * sms;
      return (one && most) || two;
    }
  }
  return 0;
}
template int default_plane_mode<float>(int, int, int);
template int default_plane_mode<double>(int, int, int);

template <typename T> int default_plane_mode_fields(int nx, int ny, int nz) {
  // Three fields a launch.  Measured on GB300 for every plane shape up to 24,576
  // points at 19 ny from 8 to 512 (one FP32 stage, plane kernels over split
  // passes): planes up to 96 x 96 and 192 x 48 0.8 to 0.99 at any ny; 128 x 128
  // 1.05, 1.02, 1.01 at ny = 8, 16, 24, 0.90 to 1.0 from 33 on; 192 x 96, one CTA an
  // SM, by the last wave of its 3 ny CTAs: 0.92 at ny = 50 (150 CTAs), 1.06 at 56,
  // 1.00 at 80, 0.95 at 100, 1.03 at 256 (768 CTAs), 0.99 at 304; other small planes
  // up to one wave: 256 x 32 0.92 at 50, 1.03 at 56; not 96 x 192 (1.03 at 128), 192 x
  // 128 (1.04), 256 x 64 (1.06).
  if (sizeof(T) == 4 && plane_supported<T>(nx, nz)) {
    const int area = nx * nz, sms = sm_count(), ctas = 3 * ny;
    if (nx <= 128 && nz <= 128) return area <= 9216 || 20 * ctas >= 9 * sms;
    if (nx <= 192 && nz <= 96) return area <= 9216 || last_wave_filled(ctas, sms);
    if (area <= 8192) return ctas <= sms;
  }
  return 0;
}
template int default_plane_mode_fields<float>(int, int, int);
template int default_plane_mode_fields<double>(int, int, int);

bool transform_size_supported(int n) {
#define X(N) if (n == N) return true;
  IBM_FOR_EACH_N(X)
#undef X
  return false;
}

}  // namespace ibm
