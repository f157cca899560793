// dg_misc.cu -- layout conversion and diagnostics kernels.
#include <cuda_runtime.h>

#include "dg_internal.h"
#include "dg_physics.cuh"

namespace dgk {

// ---------------------------------------------------------------------------
// Layout conversion (one plane at a time, grid-stride, coalesced)
// ---------------------------------------------------------------------------
template <class TS>
__global__ void plane_in_kernel(const double* __restrict__ src, StateBuf<TS> dst, int kind, int idx,
                                long ncell) {
  for (long i = blockIdx.x * (long)blockDim.x + threadIdx.x; i < ncell;
       i += (long)gridDim.x * blockDim.x) {
    double v = src[i];
    if (kind == 0) dst.c0[(size_t)idx * ncell + i] = v;
    else dst.sl[(size_t)idx * ncell + i] = (TS)v;
  }
}

template <class TS>
__global__ void plane_out_kernel(StateBuf<TS> src, double* __restrict__ dst, int kind, int idx,
                                 long ncell) {
  for (long i = blockIdx.x * (long)blockDim.x + threadIdx.x; i < ncell;
       i += (long)gridDim.x * blockDim.x) {
    dst[i] = kind == 0 ? src.c0[(size_t)idx * ncell + i] : (double)src.sl[(size_t)idx * ncell + i];
  }
}

static inline unsigned grid_for(long n, int threads) {
  long b = (n + threads - 1) / threads;
  if (b > 152L * 16) b = 152L * 16;
  if (b < 1) b = 1;
  return (unsigned)b;
}

template <class TS>
cudaError_t launch_plane_in(const double* src, StateBuf<TS> dst, int kind, int idx, long ncell,
                            cudaStream_t st) {
  plane_in_kernel<TS><<<grid_for(ncell, 256), 256, 0, st>>>(src, dst, kind, idx, ncell);
  return cudaGetLastError();
}
template <class TS>
cudaError_t launch_plane_out(StateBuf<TS> src, double* dst, int kind, int idx, long ncell,
                             cudaStream_t st) {
  plane_out_kernel<TS><<<grid_for(ncell, 256), 256, 0, st>>>(src, dst, kind, idx, ncell);
  return cudaGetLastError();
}
// All planes of one problem in one launch (blockIdx.y = plane): the interchange planes
// at src into the state (the adjoint's checkpoints; dg_load.cu loads a context's state).
template <class TS>
__global__ void state_in_kernel(const double* __restrict__ src, StateBuf<TS> dst, PlaneMap map,
                                long ncell) {
  const int k = blockIdx.y, kind = map.kind[k];
  const size_t o = (size_t)map.idx[k] * ncell;
  const double* s = src + (size_t)k * ncell;
  for (long i = blockIdx.x * (long)blockDim.x + threadIdx.x; i < ncell;
       i += (long)gridDim.x * blockDim.x) {
    const double v = s[i];
    if (kind == 0) dst.c0[o + i] = v;
    else dst.sl[o + i] = (TS)v;
  }
}

static inline dim3 state_grid(long ncell, int nplanes) {
  long b = (ncell + 255) / 256, cap = 152L * 16 / (nplanes > 0 ? nplanes : 1);
  if (b > cap) b = cap;
  if (b < 1) b = 1;
  return dim3((unsigned)b, (unsigned)nplanes);
}

template <class TS>
cudaError_t launch_state_in(const double* src, StateBuf<TS> dst, const PlaneMap& map, long ncell,
                            cudaStream_t st) {
  state_in_kernel<TS><<<state_grid(ncell, map.nplanes), 256, 0, st>>>(src, dst, map, ncell);
  return cudaGetLastError();
}
template cudaError_t launch_state_in<double>(const double*, StateBuf<double>, const PlaneMap&,
                                             long, cudaStream_t);
template cudaError_t launch_state_in<float>(const double*, StateBuf<float>, const PlaneMap&, long,
                                            cudaStream_t);
template cudaError_t launch_plane_in<double>(const double*, StateBuf<double>, int, int, long,
                                             cudaStream_t);
template cudaError_t launch_plane_in<float>(const double*, StateBuf<float>, int, int, long,
                                            cudaStream_t);
template cudaError_t launch_plane_out<double>(StateBuf<double>, double*, int, int, long,
                                              cudaStream_t);
template cudaError_t launch_plane_out<float>(StateBuf<float>, double*, int, int, long,
                                             cudaStream_t);

// ---------------------------------------------------------------------------
// Neumaier-compensated totals: per block (sum, compensation) pairs, then one
// block combines the partials in a fixed order (deterministic).
// ---------------------------------------------------------------------------
__device__ __forceinline__ void neumaier_add(double& s, double& c, double x) {
  double t = s + x;
  if (fabs(s) >= fabs(x)) c += (s - t) + x;
  else c += (x - t) + s;
  s = t;
}

__global__ void totals_partial_kernel(const double* __restrict__ c0, long ncell,
                                      double* __restrict__ partial) {
  const int v = blockIdx.y;
  double s = 0.0, c = 0.0;
  for (long i = blockIdx.x * (long)blockDim.x + threadIdx.x; i < ncell;
       i += (long)gridDim.x * blockDim.x)
    neumaier_add(s, c, c0[(size_t)v * ncell + i]);
  __shared__ double ss[256], cc[256];
  ss[threadIdx.x] = s;
  cc[threadIdx.x] = c;
  __syncthreads();
  if (threadIdx.x == 0) {
    double S = 0.0, C = 0.0;
    for (int k = 0; k < (int)blockDim.x; ++k) {
      neumaier_add(S, C, ss[k]);
      C += cc[k];
    }
    partial[((size_t)v * gridDim.x + blockIdx.x) * 2] = S;
    partial[((size_t)v * gridDim.x + blockIdx.x) * 2 + 1] = C;
  }
}

__global__ void totals_final_kernel(const double* __restrict__ partial, int nblk, int nv,
                                    double* __restrict__ out) {
  int v = threadIdx.x;
  if (v >= nv) return;
  double S = 0.0, C = 0.0;
  for (int b = 0; b < nblk; ++b) {
    neumaier_add(S, C, partial[((size_t)v * nblk + b) * 2]);
    C += partial[((size_t)v * nblk + b) * 2 + 1];
  }
  out[v] = S + C;
}

cudaError_t launch_totals(const double* c0, int nv, long ncell, double* partial, double* out,
                          cudaStream_t st) {
  const int nblk = 256;
  totals_partial_kernel<<<dim3(nblk, nv), 256, 0, st>>>(c0, ncell, partial);
  totals_final_kernel<<<1, 32, 0, st>>>(partial, nblk, nv, out);
  return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// Sec. 2.6 Stokes div-B estimate per cell (2D MHD): the face-normal field at
// each face Gauss point is the average of both one-sided polynomial values.
// Internal indices: averages b1 = 4, b2 = 5; coefficients a1 = 8, a2 = 9, a3 = 10.
// ---------------------------------------------------------------------------
template <class TS>
__global__ void divb_kernel(StateBuf<TS> s, int nx, int ny, double dx, double dy,
                            double* __restrict__ out) {
  const long ncell = (long)nx * ny;
  const double o = 0.28867513459481288225;  // 1/(2 sqrt 3)
  for (long c = blockIdx.x * (long)blockDim.x + threadIdx.x; c < ncell;
       c += (long)gridDim.x * blockDim.x) {
    int i = (int)(c % nx), j = (int)(c / nx);
    auto BX = [&](long cell, double x, double y) {
      return s.c0[4 * ncell + cell] + (double)s.sl[10 * ncell + cell] * x +
             (double)s.sl[8 * ncell + cell] * y;
    };
    auto BY = [&](long cell, double x, double y) {
      return s.c0[5 * ncell + cell] + (double)s.sl[9 * ncell + cell] * x -
             (double)s.sl[10 * ncell + cell] * y;
    };
    long xp = (long)j * nx + (i + 1) % nx, xm = (long)j * nx + (i + nx - 1) % nx;
    long yp = (long)((j + 1) % ny) * nx + i, ym = (long)((j + ny - 1) % ny) * nx + i;
    double acc = 0.0;
    for (int g = 0; g < 2; ++g) {
      double ty = (g ? 1.0 : -1.0) * o * dy, tx = (g ? 1.0 : -1.0) * o * dx;
      acc += 0.5 * dy * 0.5 * (BX(c, 0.5 * dx, ty) + BX(xp, -0.5 * dx, ty));
      acc -= 0.5 * dy * 0.5 * (BX(c, -0.5 * dx, ty) + BX(xm, 0.5 * dx, ty));
      acc += 0.5 * dx * 0.5 * (BY(c, tx, 0.5 * dy) + BY(yp, tx, -0.5 * dy));
      acc -= 0.5 * dx * 0.5 * (BY(c, tx, -0.5 * dy) + BY(ym, tx, 0.5 * dy));
    }
    out[c] = acc / (dx * dy);
  }
}

template <class TS>
cudaError_t launch_divb(StateBuf<TS> s, int nx, int ny, double dx, double dy, double* out,
                        cudaStream_t st) {
  long n = (long)nx * ny;
  divb_kernel<TS><<<grid_for(n, 256), 256, 0, st>>>(s, nx, ny, dx, dy, out);
  return cudaGetLastError();
}
template cudaError_t launch_divb<double>(StateBuf<double>, int, int, double, double, double*,
                                         cudaStream_t);
template cudaError_t launch_divb<float>(StateBuf<float>, int, int, double, double, double*,
                                        cudaStream_t);

}  // namespace dgk
