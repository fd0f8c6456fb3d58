// plane.cuh -- the plane transform kernels: one CTA per y-plane (plane mode 1).
//
// Instantiated per plane shape, FP32 in plane_*.cu (one file per range of x
// lengths, so that they compile in parallel), FP64 in transforms.cu.
#pragma once

#include "fft2.cuh"
#include "internal.h"
#include "stencil.cuh"

namespace ibm {

// The refinement residual formed inside the forward transform: x NULL for
// none, else the input is b and the kernel transforms r = b - A x (FP32).
struct PlaneResidual {
  const float *x;
  ResidualArgs A;
};

// r of plane j (b: its first value) into shared memory, row k at r + k pitch.
// The wall kind is a run-time value here: the planes below and above, and the
// ghost's sign, are the same for the whole plane.  (sigma = 0 goes through the
// sigma form: -0 x + b = b.)
template <int NX, int NZ>
__device__ __forceinline__ void plane_residual(const PlaneResidual &res, const float *b, int j, float *r, int pitch,
                                               int tid, int nthr) {
  const ResidualArgs &A = res.A;
  constexpr int Q = NX / 4;
  const float *xc = res.x + (size_t)j * NX * NZ;
  const float *xlo = j > 0 ? xc - NX * NZ : nullptr, *xhi = j + 1 < A.ny ? xc + NX * NZ : nullptr;
  float gs = 1.f;
  if (A.bc == BC_CELL_DIRICHLET) gs = -1.f;
  if (A.bc == BC_FACE_DIRICHLET) {  // faces 0 and ny are walls (0)
    gs = 0.f;
    if (j == 1) xlo = nullptr;
  }
  if (A.bc == BC_PERIODIC) {
    if (!xlo) xlo = res.x + (size_t)(A.ny - 1) * NX * NZ;
    if (!xhi) xhi = res.x;
  }
  float2 m = make_float2(0.f, 0.f);
  if (A.boff) m = *reinterpret_cast<const float2 *>(A.boff + 1);
  for (int t = tid; t < Q * NZ; t += nthr) {
    const int k = t / Q, i0 = 4 * (t - k * Q);
    float4 bt, v = make_float4(0.f, 0.f, 0.f, 0.f);
    if (A.bc != BC_FACE_DIRICHLET || j > 0) v = residual4_ghost<true>(A, gs, b, xc, xlo, xhi, k * NX + i0, i0, k, m, bt);
    float2 *d = reinterpret_cast<float2 *>(r + k * pitch + i0);
    d[0] = make_float2(v.x, v.y);
    d[1] = make_float2(v.z, v.w);
  }
}

// Shared memory (complex entries): tw2x [NX], tw2z [NZ], the spectrum plane
// [NZ][P], and one exchange buffer reused by the x chunks (CP row pairs,
// [CP][N1x][N2x+1]) and the z chunks (CW columns, [N1z][N2z][CW]); chunk
// sizes fill what the plane leaves of the 227 KB.
template <typename T, int NX, int NZ> struct PlaneCfg {
  using C = cplx<T>;
  static constexpr int P = NX / 2 + 1;
  static constexpr int N1X = TwoStep<NX>::N1, N2X = TwoStep<NX>::N2, XPITCH = N2X + 1;
  static constexpr size_t fixed = sizeof(C) * ((size_t)NX + NZ + (size_t)NZ * P);
  static constexpr size_t room = fixed < kPlaneSmemLimit ? kPlaneSmemLimit - fixed : 0;
  static constexpr size_t pair_bytes = sizeof(C) * N1X * XPITCH;
  static constexpr size_t col_bytes = sizeof(C) * NZ;
  static constexpr int CP0 = (int)(room / pair_bytes), CW0 = (int)(room / col_bytes);
  static constexpr int CP = CP0 < NZ / 2 ? CP0 : NZ / 2;
  static constexpr int CW = CW0 < P ? CW0 : P;
  static constexpr bool ok = CP >= (NZ / 2 < 8 ? NZ / 2 : 8) && CW >= (P < 8 ? P : 8);
  static constexpr size_t xbytes = (size_t)CP * pair_bytes > (size_t)CW * col_bytes ? (size_t)CP * pair_bytes
                                                                                    : (size_t)CW * col_bytes;
  static constexpr size_t bytes = fixed + xbytes;
  // threads: enough for the largest of the x step-1, x step-3 and z step-1
  // job counts in one round (z step 3 takes N2z / N1z rounds), <= 1024
  static constexpr int N1Z = TwoStep<NZ>::N1;
  static constexpr int J3 = N2X / 2;
  static constexpr int JMAX0 = CP * N1X > CP * J3 ? CP * N1X : CP * J3;
  static constexpr int JMAX = JMAX0 > CW * N1Z ? JMAX0 : CW * N1Z;
  static constexpr int THREADS = JMAX >= 1024 ? 1024 : (JMAX + 31) / 32 * 32;
};

template <typename T, int NX, int NZ>
__global__ void __launch_bounds__(PlaneCfg<T, NX, NZ>::THREADS)
k_plane_fwd(Ptr3<const T *> in_, Ptr3<cplx<T> *> S_, const cplx<T> *__restrict__ twx,
            const cplx<T> *__restrict__ twz, double *zrhs, PlaneResidual res) {
  const T *__restrict__ in = in_[blockIdx.y];
  cplx<T> *__restrict__ S = S_[blockIdx.y];
  using Cfg = PlaneCfg<T, NX, NZ>;
  constexpr int P = Cfg::P, N1X = Cfg::N1X, XPITCH = Cfg::XPITCH, CP = Cfg::CP, CW = Cfg::CW;
  constexpr int kPlaneThreads_ = Cfg::THREADS;
  constexpr int N1Z = TwoStep<NZ>::N1, N2Z = TwoStep<NZ>::N2, J3 = Cfg::N2X / 2;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  cplx<T> *tw2x = reinterpret_cast<cplx<T> *>(smem_raw);
  cplx<T> *tw2z = tw2x + NX;
  cplx<T> *plane = tw2z + NZ;  // [NZ][P]
  cplx<T> *X = plane + NZ * P;
  const int j = blockIdx.x;
  const int tid = threadIdx.x;
  load_step_twiddles<T, NX>(tw2x, twx);
  load_step_twiddles<T, NZ>(tw2z, twz);
  pdl_wait();  // the fields below are the predecessor's output
  __syncthreads();
  const T *src = in + (size_t)j * NZ * NX;
  int pitch = NX;
  if constexpr (sizeof(T) == 4) {
    if (res.x) {
      // refinement: the rows of r = b - A x instead, each where its spectrum row will go (2 P values)
      float *r = reinterpret_cast<float *>(plane);
      plane_residual<NX, NZ>(res, src, j, r, 2 * P, tid, kPlaneThreads_);
      __syncthreads();
      src = r;
      pitch = 2 * P;
    }
  }
  for (int p0 = 0; p0 < NZ / 2; p0 += CP) {
    const int np = min(CP, NZ / 2 - p0);
    for (int job = tid; job < np * N1X; job += kPlaneThreads_) {
      const int p = job / N1X, n1 = job - p * N1X;
      rfwd_step1<T, NX>(src + (size_t)(p0 + p) * 2 * pitch, pitch, n1, tw2x, X + (p * N1X + n1) * XPITCH);
    }
    __syncthreads();
    for (int job = tid; job < np * J3; job += kPlaneThreads_) {
      const int p = job / J3, q = job - p * J3;
      cplx<T> *dA = plane + (p0 + p) * 2 * P;
      rfwd_step3<T, NX, XPITCH>(X + p * N1X * XPITCH, q, dA, dA + P);
    }
    __syncthreads();
  }
  cplx<T> *dst = S + (size_t)j * NZ * P;
  for (int c0 = 0; c0 < P; c0 += CW) {
    const int nc = min(CW, P - c0);
    for (int job = tid; job < CW * N1Z; job += kPlaneThreads_) {
      const int n1 = job / CW, c = job - n1 * CW;
      if (c < nc)
        col_step1<T, NZ, false, CW>(plane + c0 + c, P, n1, tw2z, X + n1 * N2Z * CW + c, false, mk<T>((T)0, (T)0));
    }
    __syncthreads();
    for (int job = tid; job < CW * N2Z; job += kPlaneThreads_) {
      const int k2 = job / CW, c = job - k2 * CW;
      if (c < nc) {
        const cplx<T> u0 = col_step3<T, NZ, false, CW>(X, c, k2, dst + c0 + c, P);
        if (zrhs && c0 + c == 0 && k2 == 0) zrhs[j] = 0.5 * (double)u0.x;
      }
    }
    __syncthreads();
  }
}

// Inverse: spectrum plane -> out = addend + scale * result.
template <typename T, int NX, int NZ>
__global__ void __launch_bounds__(PlaneCfg<T, NX, NZ>::THREADS)
k_plane_inv(Ptr3<cplx<T> *> S_, Ptr3<T *> out_, Ptr3<const T *> add_, const cplx<T> *__restrict__ twx,
            const cplx<T> *__restrict__ twz, T scale, const double *zsol) {
  const cplx<T> *__restrict__ S = S_[blockIdx.y];
  T *out = out_[blockIdx.y];
  const T *addend = add_[blockIdx.y];
  using Cfg = PlaneCfg<T, NX, NZ>;
  constexpr int P = Cfg::P, N1X = Cfg::N1X, N2X = Cfg::N2X, XPITCH = Cfg::XPITCH, CP = Cfg::CP, CW = Cfg::CW;
  constexpr int kPlaneThreads_ = Cfg::THREADS;
  constexpr int N1Z = TwoStep<NZ>::N1, N2Z = TwoStep<NZ>::N2;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  cplx<T> *tw2x = reinterpret_cast<cplx<T> *>(smem_raw);
  cplx<T> *tw2z = tw2x + NX;
  cplx<T> *plane = tw2z + NZ;
  cplx<T> *X = plane + NZ * P;
  const int j = blockIdx.x;
  const int tid = threadIdx.x;
  load_step_twiddles<T, NX>(tw2x, twx);
  load_step_twiddles<T, NZ>(tw2z, twz);
  pdl_wait();  // the fields below are the predecessor's output
  __syncthreads();
  const cplx<T> *src = S + (size_t)j * NZ * P;
  const cplx<T> z0 = zsol ? mk<T>((T)(2.0 * zsol[j]), (T)0) : mk<T>((T)0, (T)0);
  for (int c0 = 0; c0 < P; c0 += CW) {
    const int nc = min(CW, P - c0);
    for (int job = tid; job < CW * N1Z; job += kPlaneThreads_) {
      const int n1 = job / CW, c = job - n1 * CW;
      if (c < nc)
        col_step1<T, NZ, true, CW>(src + c0 + c, P, n1, tw2z, X + n1 * N2Z * CW + c, zsol && c0 + c == 0, z0);
    }
    __syncthreads();
    for (int job = tid; job < CW * N2Z; job += kPlaneThreads_) {
      const int k2 = job / CW, c = job - k2 * CW;
      if (c < nc) col_step3<T, NZ, true, CW>(X, c, k2, plane + c0 + c, P);
    }
    __syncthreads();
  }
  T *dst = out + (size_t)j * NZ * NX;
  const T *add = addend ? addend + (size_t)j * NZ * NX : nullptr;
  for (int p0 = 0; p0 < NZ / 2; p0 += CP) {
    const int np = min(CP, NZ / 2 - p0);
    for (int job = tid; job < np * N1X; job += kPlaneThreads_) {
      const int p = job / N1X, n1 = job - p * N1X;
      const cplx<T> *sA = plane + (p0 + p) * 2 * P;
      rinv_step1<T, NX>(sA, sA + P, n1, tw2x, X + (p * N1X + n1) * XPITCH);
    }
    __syncthreads();
    for (int job = tid; job < np * N2X; job += kPlaneThreads_) {
      const int p = job / N2X, k2 = job - p * N2X;
      const size_t r = (size_t)(p0 + p) * 2 * NX;
      rinv_step3<T, NX, XPITCH>(X + p * N1X * XPITCH, k2, dst + r, dst + r + NX, add ? add + r : nullptr,
                                add ? add + r + NX : nullptr, scale);
    }
    __syncthreads();
  }
}

// --------------------------------------------------------------------------
// The same transforms in place (FP32): one buffer holds the plane and every
// exchange.  Each thread keeps its job's values in registers over the barrier
// between a step's reads and its writes, so the CTA needs about the plane's
// bytes (128 x 128: 72 KB instead of 139) and two CTAs share an SM, each with
// barriers of its own to wait at.  For lengths up to 128, where what a thread
// holds over a barrier is at most 16 complex values: one job's of x step 1 (N2X),
// x step 3 (2 N1X) and z step 1 (N2Z), or its RZ3 jobs' of z step 3 (N1Z each; up
// to three jobs, at z lengths 12 and 48).  Measured against
// the separate buffers: 128 x 512 x 128 refined solve 163 -> 133 us, 128 x 256 x
// 128 78 -> 66, 128^3 44.1 -> 43.3, 96^3 32.5 -> 31.5, 48 x 33 x 24 21.8 -> 20.0.
// --------------------------------------------------------------------------
template <int NX, int NZ> struct PlaneInPlace {
  static constexpr int P = NX / 2 + 1;
  static constexpr int N1X = TwoStep<NX>::N1, N2X = TwoStep<NX>::N2, XPITCH = N2X + 1;
  static constexpr int N1Z = TwoStep<NZ>::N1, N2Z = TwoStep<NZ>::N2;
  static constexpr int X1 = NZ / 2 * N1X, X3 = NZ / 2 * (N2X / 2), Z1 = P * N1Z, Z3 = P * N2Z;  // jobs of each step
  static constexpr int mx(int a, int b) { return a > b ? a : b; }
  static constexpr int THREADS = (mx(mx(X1, X3), Z1) + 31) / 32 * 32;
  static constexpr int RZ3 = (Z3 + THREADS - 1) / THREADS;  // rounds of z step 3
  // CTAs an SM the registers are sized for (at least 56 a thread)
  static constexpr int CTAS = 1152 / THREADS < 2 ? 2 : 1152 / THREADS > 8 ? 8 : 1152 / THREADS;
  static constexpr int BUF = mx(NZ * P, NZ / 2 * N1X * XPITCH);
  static constexpr size_t bytes = sizeof(float2) * ((size_t)NX + NZ + BUF);
  static constexpr bool ok = NX <= 128 && NZ <= 128 && THREADS <= 576 && RZ3 * N1Z <= 16;
};

template <int NX, int NZ>
__global__ void __launch_bounds__(PlaneInPlace<NX, NZ>::THREADS, PlaneInPlace<NX, NZ>::CTAS)
k_plane_fwd_ip(Ptr3<const float *> in_, Ptr3<float2 *> S_, const float2 *__restrict__ twx,
               const float2 *__restrict__ twz, double *zrhs, PlaneResidual res) {
  using Cfg = PlaneInPlace<NX, NZ>;
  constexpr int P = Cfg::P, N1X = Cfg::N1X, N2X = Cfg::N2X, XPITCH = Cfg::XPITCH, N1Z = Cfg::N1Z, N2Z = Cfg::N2Z;
  const float *__restrict__ in = in_[blockIdx.y];
  float2 *__restrict__ S = S_[blockIdx.y];
  extern __shared__ __align__(16) unsigned char smem_raw[];
  float2 *tw2x = reinterpret_cast<float2 *>(smem_raw);
  float2 *tw2z = tw2x + NX;
  float2 *buf = tw2z + NZ;  // the plane [NZ][P], or an exchange
  const int j = blockIdx.x, tid = threadIdx.x;
  load_step_twiddles<float, NX>(tw2x, twx);
  load_step_twiddles<float, NZ>(tw2z, twz);
  pdl_wait();  // the fields below are the predecessor's output
  const float *src = in + (size_t)j * NZ * NX;
  int pitch = NX;
  if (res.x) {
    float *r = reinterpret_cast<float *>(buf);
    plane_residual<NX, NZ>(res, src, j, r, 2 * P, tid, Cfg::THREADS);
    src = r;
    pitch = 2 * P;
  }
  __syncthreads();
  {  // x step 1
    const int p = tid / N1X, n1 = tid - p * N1X;
    const bool job = tid < Cfg::X1;
    float2 v[N2X];
    if (job) {
      const float *a = src + (size_t)p * 2 * pitch + n1;
#pragma unroll
      for (int n2 = 0; n2 < N2X; ++n2) v[n2] = make_float2(a[N1X * n2], a[pitch + N1X * n2]);
      reg_dft<false, N2X>(v);
    }
    if (res.x) __syncthreads();  // the rows have been read
    if (job) {
      float2 *x = buf + tid * XPITCH;
      x[0] = v[0];
#pragma unroll
      for (int k2 = 1; k2 < N2X; ++k2) x[k2] = cmul(v[k2], tw2x[k2 * N1X + n1]);
    }
  }
  __syncthreads();
  {  // x step 3 (rfwd_step3 with the barrier between its reads and writes)
    constexpr int J3 = N2X / 2;
    const int p = tid / J3, q = tid - p * J3;
    const bool job = tid < Cfg::X3, own = q == 0;
    const int qb = own ? N2X / 2 : N2X - q;
    float2 u[N1X], w[N1X];
    if (job) {
      const float2 *xp = buf + p * N1X * XPITCH;
#pragma unroll
      for (int n1 = 0; n1 < N1X; ++n1) { u[n1] = xp[n1 * XPITCH + q]; w[n1] = xp[n1 * XPITCH + qb]; }
      reg_dft<false, N1X>(u);
      reg_dft<false, N1X>(w);
    }
    __syncthreads();
    if (job) {
      float2 *dA = buf + p * 2 * P, *dB = dA + P;
#pragma unroll
      for (int k1 = 0; k1 < N1X / 2; ++k1) {
        const float2 zu = own ? u[(N1X - k1) % N1X] : w[N1X - 1 - k1];
        const float2 zw = own ? w[N1X - 1 - k1] : u[N1X - 1 - k1];
        split_put(u[k1], zu, dA + q + N2X * k1, dB + q + N2X * k1);
        split_put(w[k1], zw, dA + qb + N2X * k1, dB + qb + N2X * k1);
      }
      if (own) split_put(u[N1X / 2], u[N1X / 2], dA + NX / 2, dB + NX / 2);
    }
  }
  __syncthreads();
  {  // z step 1
    const int n1 = tid / P, c = tid - n1 * P;
    const bool job = tid < Cfg::Z1;
    float2 v[N2Z];
    if (job) {
#pragma unroll
      for (int n2 = 0; n2 < N2Z; ++n2) v[n2] = buf[(n1 + N1Z * n2) * P + c];
      reg_dft<false, N2Z>(v);
    }
    __syncthreads();
    if (job) {
      float2 *x = buf + n1 * N2Z * P + c;
      x[0] = v[0];
#pragma unroll
      for (int k2 = 1; k2 < N2Z; ++k2) x[k2 * P] = cmul(v[k2], tw2z[k2 * N1Z + n1]);
    }
  }
  __syncthreads();
  float2 *dst = S + (size_t)j * NZ * P;
  for (int job = tid; job < Cfg::Z3; job += Cfg::THREADS) {
    const int k2 = job / P, c = job - k2 * P;
    const float2 u0 = col_step3<float, NZ, false, P>(buf, c, k2, dst + c, P);
    if (zrhs && job == 0) zrhs[j] = 0.5 * (double)u0.x;
  }
}

template <int NX, int NZ>
__global__ void __launch_bounds__(PlaneInPlace<NX, NZ>::THREADS, PlaneInPlace<NX, NZ>::CTAS)
k_plane_inv_ip(Ptr3<float2 *> S_, Ptr3<float *> out_, Ptr3<const float *> add_, const float2 *__restrict__ twx,
               const float2 *__restrict__ twz, float scale, const double *zsol) {
  using Cfg = PlaneInPlace<NX, NZ>;
  constexpr int P = Cfg::P, N1X = Cfg::N1X, N2X = Cfg::N2X, XPITCH = Cfg::XPITCH, N1Z = Cfg::N1Z, N2Z = Cfg::N2Z;
  constexpr int RZ3 = Cfg::RZ3;
  const float2 *__restrict__ S = S_[blockIdx.y];
  float *out = out_[blockIdx.y];
  const float *addend = add_[blockIdx.y];
  extern __shared__ __align__(16) unsigned char smem_raw[];
  float2 *tw2x = reinterpret_cast<float2 *>(smem_raw);
  float2 *tw2z = tw2x + NX;
  float2 *buf = tw2z + NZ;
  const int j = blockIdx.x, tid = threadIdx.x;
  load_step_twiddles<float, NX>(tw2x, twx);
  load_step_twiddles<float, NZ>(tw2z, twz);
  pdl_wait();  // the fields below are the predecessor's output
  __syncthreads();
  if (tid < Cfg::Z1) {  // z step 1
    const int n1 = tid / P, c = tid - n1 * P;
    const float2 z0 = zsol ? make_float2((float)(2.0 * zsol[j]), 0.f) : make_float2(0.f, 0.f);
    col_step1<float, NZ, true, P>(S + (size_t)j * NZ * P + c, P, n1, tw2z, buf + n1 * N2Z * P + c, zsol && c == 0, z0);
  }
  __syncthreads();
  {  // z step 3
    float2 u[RZ3][N1Z];
#pragma unroll
    for (int r = 0; r < RZ3; ++r) {
      const int job = tid + r * Cfg::THREADS;
      if (job < Cfg::Z3) {
        const int k2 = job / P, c = job - k2 * P;
#pragma unroll
        for (int n1 = 0; n1 < N1Z; ++n1) u[r][n1] = buf[(n1 * N2Z + k2) * P + c];
        reg_dft<true, N1Z>(u[r]);
      }
    }
    __syncthreads();
#pragma unroll
    for (int r = 0; r < RZ3; ++r) {
      const int job = tid + r * Cfg::THREADS;
      if (job < Cfg::Z3) {
        const int k2 = job / P, c = job - k2 * P;
#pragma unroll
        for (int k1 = 0; k1 < N1Z; ++k1) buf[(k2 + N2Z * k1) * P + c] = u[r][k1];
      }
    }
  }
  __syncthreads();
  {  // x step 1 (rinv_step1 with the barrier between its reads and writes)
    const int p = tid / N1X, n1 = tid - p * N1X;
    const bool job = tid < Cfg::X1;
    float2 v[N2X];
    if (job) {
      rinv_load<float, NX>(buf + p * 2 * P, buf + p * 2 * P + P, n1, v);
      reg_dft<true, N2X>(v);
    }
    __syncthreads();
    if (job) {
      float2 *x = buf + tid * XPITCH;
      x[0] = v[0];
#pragma unroll
      for (int k2 = 1; k2 < N2X; ++k2) x[k2] = cmulc(v[k2], tw2x[k2 * N1X + n1]);
    }
  }
  __syncthreads();
  float *dst = out + (size_t)j * NZ * NX;
  const float *add = addend ? addend + (size_t)j * NZ * NX : nullptr;
  for (int job = tid; job < NZ / 2 * N2X; job += Cfg::THREADS) {
    const int p = job / N2X, k2 = job - p * N2X;
    const size_t r = (size_t)p * 2 * NX;
    rinv_step3<float, NX, XPITCH>(buf + p * N1X * XPITCH, k2, dst + r, dst + r + NX, add ? add + r : nullptr,
                                  add ? add + r + NX : nullptr, scale);
  }
}

// Plane shapes with FP32 kernels: every pair of supported lengths up to
// kPlaneArea values whose spectrum fits in shared memory, and three larger
// ones for the tuner.
constexpr int kPlaneArea = 24576;
template <int NX, int NZ> constexpr bool plane_shape_f32() {
  constexpr bool extra = (NX == 192 && NZ == 192) || (NX == 256 && NZ == 128) || (NX == 128 && NZ == 256);
  if constexpr (NX * NZ <= kPlaneArea || extra) return PlaneCfg<float, NX, NZ>::ok;
  else return false;
}

template <int... N> struct Lengths {};
using PlaneLengths = Lengths<8, 12, 16, 24, 32, 48, 64, 96, 128, 192, 256, 384, 512>;

// f(NZ) for the instantiated shape NX x nz; false if there is none.
template <int NX, typename F, int... NZ> inline bool plane_dispatch(int nz, F &&f, Lengths<NZ...>) {
  bool found = false;
  auto one = [&](auto c) {
    constexpr int Z = decltype(c)::value;
    if constexpr (plane_shape_f32<NX, Z>()) {
      if (nz == Z) {
        found = true;
        f(c);
      }
    }
  };
  (one(std::integral_constant<int, NZ>{}), ...);
  return found;
}

// One x length's FP32 launches (defined in plane_*.cu); cudaErrorNotSupported
// for a z length without an instantiation.
template <int NX>
cudaError_t plane_forward_f32(const TransformGeom &g, Ptr3<const float *> in, Ptr3<float2 *> S, const float2 *twx,
                              const float2 *twz, const PlaneResidual &res, cudaStream_t st);
template <int NX>
cudaError_t plane_inverse_f32(const TransformGeom &g, Ptr3<float2 *> S, Ptr3<float *> out, Ptr3<const float *> addend,
                              const float2 *twx, const float2 *twz, float scale, cudaStream_t st);

#ifdef IBM_PLANE_DEFINE
template <int NX>
cudaError_t plane_forward_f32(const TransformGeom &g, Ptr3<const float *> in, Ptr3<float2 *> S, const float2 *twx,
                              const float2 *twz, const PlaneResidual &res, cudaStream_t st) {
  cudaError_t err = cudaErrorNotSupported;
  plane_dispatch<NX>(g.nz, [&](auto c) {
    constexpr int NZ = decltype(c)::value;
    if constexpr (PlaneInPlace<NX, NZ>::ok) {
      using Cfg = PlaneInPlace<NX, NZ>;
      if ((err = ensure_max_smem<k_plane_fwd_ip<NX, NZ>>())) return;
      err = launch_pdl(k_plane_fwd_ip<NX, NZ>, dim3(g.ny, g.nb), Cfg::THREADS, Cfg::bytes, st, in, S, twx, twz, g.zrhs,
                       res);
    } else {
      using Cfg = PlaneCfg<float, NX, NZ>;
      if ((err = ensure_max_smem<k_plane_fwd<float, NX, NZ>>())) return;
      err = launch_pdl(k_plane_fwd<float, NX, NZ>, dim3(g.ny, g.nb), Cfg::THREADS, Cfg::bytes, st, in, S, twx, twz,
                       g.zrhs, res);
    }
  }, PlaneLengths{});
  return err;
}
template <int NX>
cudaError_t plane_inverse_f32(const TransformGeom &g, Ptr3<float2 *> S, Ptr3<float *> out, Ptr3<const float *> addend,
                              const float2 *twx, const float2 *twz, float scale, cudaStream_t st) {
  cudaError_t err = cudaErrorNotSupported;
  plane_dispatch<NX>(g.nz, [&](auto c) {
    constexpr int NZ = decltype(c)::value;
    if constexpr (PlaneInPlace<NX, NZ>::ok) {
      using Cfg = PlaneInPlace<NX, NZ>;
      if ((err = ensure_max_smem<k_plane_inv_ip<NX, NZ>>())) return;
      err = launch_pdl(k_plane_inv_ip<NX, NZ>, dim3(g.ny, g.nb), Cfg::THREADS, Cfg::bytes, st, S, out, addend, twx, twz,
                       0.5f * scale, g.zsol);
    } else {
      using Cfg = PlaneCfg<float, NX, NZ>;
      if ((err = ensure_max_smem<k_plane_inv<float, NX, NZ>>())) return;
      err = launch_pdl(k_plane_inv<float, NX, NZ>, dim3(g.ny, g.nb), Cfg::THREADS, Cfg::bytes, st, S, out, addend, twx,
                       twz, 0.5f * scale, g.zsol);
    }
  }, PlaneLengths{});
  return err;
}
#define IBM_PLANE_INSTANCE(NX)                                                                                    \
  template cudaError_t plane_forward_f32<NX>(const TransformGeom &, Ptr3<const float *>, Ptr3<float2 *>,          \
                                             const float2 *, const float2 *, const PlaneResidual &, cudaStream_t); \
  template cudaError_t plane_inverse_f32<NX>(const TransformGeom &, Ptr3<float2 *>, Ptr3<float *>,                \
                                             Ptr3<const float *>, const float2 *, const float2 *, float, cudaStream_t);
#endif

}  // namespace ibm
