// periodic.cu -- the pencil step of the triply periodic branch.
//
// With y periodic as well (Sec. 2.3.3, S2), every (kx, kz) pencil of the
// x/z spectrum is diagonalised by a Fourier transform along y too: the
// solve is a forward y-transform, a divide by the eigenvalue of each
// (kx, ky, kz) mode, and an inverse y-transform (scaled by 1/ny), all in
// place on the spectrum.  Eigenvalues (Appendix A): lambda = lambda_x(kx) +
// lambda_y(ky) + lambda_z(kz), lambda_d = (2/h_d^2)(1 - cos theta_d);
//   Poisson    x = -f / lambda, the (0,0,0) mode set to 0 (mean(phi) = 0);
//   Helmholtz  x =  f / (1 + c lambda).
// A CTA takes W consecutive pencils (every access a run of W complex
// values).  With N = N1 N2 the forward transform's step 3 leaves the modes
// ky = k2 + N2 k1, k1 < N1, in the registers of the thread of k2, and those
// are one step-1 group of the inverse transform split the other way round
// (N2 lanes, length-N1 DFTs): the thread divides them by their eigenvalues
// and runs on into the inverse, whose exchange goes back to the very entries
// of shared memory the thread read.  Two exchanges and three barriers per
// pencil in one buffer; bound by the global accesses (512 x 256 x 256 FP32:
// 104 us a launch with the divide a pass of its own and a second buffer, 61 us
// now, 4.4 TB/s).  For the Poisson solve an extra CTA sums the FP64 plane sums
// of b (from the forward x/z transform) into the removed mean.
#include "fft2.cuh"
#include "internal.h"

namespace ibm {

template <typename T, int N> struct YCfg {
  static constexpr int N1 = TwoStep<N>::N1, N2 = TwoStep<N>::N2;
  static constexpr int WMIN = sizeof(T) == 4 ? 16 : 8, WMAX = 64;
  static constexpr int WT0 = (sizeof(T) == 4 ? 256 : 64) / N1;
  static constexpr int W = WT0 < WMIN ? WMIN : (WT0 > WMAX ? WMAX : WT0);
  static constexpr int THREADS = W * N1;
  static constexpr size_t smem = sizeof(cplx<T>) * ((size_t)N + (size_t)N * W) + sizeof(T) * N;
};

template <typename T, int N>
__global__ void __launch_bounds__(YCfg<T, N>::THREADS)
k_ypencil(cplx<T> *__restrict__ S, const cplx<T> *__restrict__ tw, const T *__restrict__ lamx,
          const T *__restrict__ lamz, const T *__restrict__ lamy, PencilParams pp, double *mean_out) {
  using Cfg = YCfg<T, N>;
  constexpr int N1 = Cfg::N1, N2 = Cfg::N2, W = Cfg::W;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  cplx<T> *tw2 = reinterpret_cast<cplx<T> *>(smem_raw);
  cplx<T> *X = tw2 + N;  // [N1][N2][W] exchange of both transforms
  T *ly = reinterpret_cast<T *>(X + N * W);  // lambda_y
  load_step_twiddles<T, N>(tw2, tw);
  for (int i = threadIdx.x; i < N; i += blockDim.x) ly[i] = lamy[i];
  pdl_wait();
  if (pp.zero_mode && blockIdx.x == gridDim.x - 1) {
    // removed mean of b: the FP64 sum of the plane sums (zrhs) / (nx ny nz)
    if (threadIdx.x < 32) {
      double s = 0.0;
      for (int j = threadIdx.x; j < N; j += 32) s += pp.zrhs[j];
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
      if (threadIdx.x == 0 && mean_out) {
        const double m = s * pp.inv_nxnz * pp.inv_ny;
        mean_out[0] = m;
        float2 f;
        f.x = (float)m;
        f.y = (float)(m - (double)f.x);
        *reinterpret_cast<float2 *>(mean_out + 1) = f;
      }
    }
    return;
  }
  __syncthreads();
  const size_t plane = (size_t)pp.nz * pp.P;
  const int npen = pp.nz * pp.P;
  const int tid = threadIdx.x;
  const int c = tid % W;
  const int p = blockIdx.x * W + c;
  const bool live = p < npen;
  const int kz = live ? p / pp.P : 0, kx = live ? p - kz * pp.P : 0;
  cplx<T> *base = S + (live ? p : 0);
  const T lxz = lamx[kx] + lamz[kz];
  const T g_add = (T)pp.g_add, g_mul = (T)pp.g_mul;
  const T sgn = pp.neg_rhs ? (T)-1 : (T)1;
  const T inv_n = (T)1 / (T)N;
  // forward y-transform, step 1
  if (live) col_step1<T, N, false, W>(base, plane, tid / W, tw2, X + (tid / W) * N2 * W + c, false, mk<T>(0, 0));
  __syncthreads();
  // forward step 3, the divide and the inverse's step 1, in the registers of the thread of k2
  if (live) {
    for (int k2 = tid / W; k2 < N2; k2 += N1) {
      cplx<T> *x = X + k2 * W + c;  // entries N2 W apart
      cplx<T> u[N1];
#pragma unroll
      for (int n1 = 0; n1 < N1; ++n1) u[n1] = x[n1 * N2 * W];
      reg_dft<false, N1>(u);
#pragma unroll
      for (int k1 = 0; k1 < N1; ++k1) {
        const T eig = g_add + g_mul * (lxz + ly[k2 + N2 * k1]);
        const T s = eig != (T)0 ? sgn * inv_n / eig : (T)0;  // the (0,0,0) Poisson mode -> 0
        u[k1] = cscale(u[k1], s);
      }
      reg_dft<true, N1>(u);
      x[0] = u[0];
#pragma unroll
      for (int m = 1; m < N1; ++m) x[m * N2 * W] = cmulc(u[m], tw2[k2 * N1 + m]);
    }
  }
  __syncthreads();
  // inverse step 3: rows m + N1 j
  if (live) {
    const int m = tid / W;
    cplx<T> u[N2];
#pragma unroll
    for (int k2 = 0; k2 < N2; ++k2) u[k2] = X[(m * N2 + k2) * W + c];
    reg_dft<true, N2>(u);
#pragma unroll
    for (int j = 0; j < N2; ++j) base[(size_t)(m + N1 * j) * plane] = u[j];
  }
}

#define IBM_Y_N(X) X(8) X(12) X(16) X(24) X(32) X(48) X(64) X(96) X(128) X(192) X(256) X(384) X(512)

template <typename T>
cudaError_t launch_ypencil(const PencilParams &pp, Ptr3<cplx<T> *> S3, const cplx<T> *twy, const T *lamx,
                           const T *lamz, const T *lamy, double *mean_out, cudaStream_t st) {
  const int npen = pp.nz * pp.P;
  for (int b = 0; b < pp.nb; ++b) {
    bool done = false;
#define X(N)                                                                                      \
    if (pp.ny == N) {                                                                             \
      using Cfg = YCfg<T, N>;                                                                     \
      { cudaError_t e = ensure_max_smem<k_ypencil<T, N>>(); if (e) return e; }                   \
      const int grid = ceil_div(npen, Cfg::W) + (pp.zero_mode ? 1 : 0);                           \
      IBM_KTRY(launch_pdl(k_ypencil<T, N>, grid, Cfg::THREADS, Cfg::smem, st, S3[b], twy, lamx, lamz, lamy, pp, \
                          mean_out));                                                             \
      done = true;                                                                                \
    }
    IBM_Y_N(X)
#undef X
    if (!done) return cudaErrorInvalidValue;
  }
  return cudaSuccess;
}

template cudaError_t launch_ypencil<float>(const PencilParams &, Ptr3<float2 *>, const float2 *, const float *,
                                           const float *, const float *, double *, cudaStream_t);
template cudaError_t launch_ypencil<double>(const PencilParams &, Ptr3<double2 *>, const double2 *, const double *,
                                            const double *, const double *, double *, cudaStream_t);

}  // namespace ibm
