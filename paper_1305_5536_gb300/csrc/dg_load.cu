// dg_load.cu -- a whole context's state in or out in one launch.
//
// In: every problem's interchange planes to the internal layout, the Courant signal
// speed of the averages on the way, and, by the last block of each problem, the reset
// and commit of its control block and the control block's copy in page-locked host
// memory.  One launch where separate layout (one per problem), reset, Courant (one per
// problem, reading the averages again), commit and read-back operations stood: at 2D
// MHD 512^2 a pass (set, four steps, get) went from 385 to 356 us, with 48 batched problems
// from 2.50 to 1.71 ms.
// Bound by the memory traffic of the planes for large states and by the launch for
// small ones: one thread per cell, all its planes in flight (coalesced: consecutive
// threads take consecutive cells of every plane).
// Out: the same mapping back.
#include <cuda_runtime.h>

#include "dg_internal.h"
#include "dg_stage2d.cuh"
#include "dg_stage3d.cuh"
#include "dg_stage3m.cuh"

namespace dgk {

namespace {

constexpr int kLoadThreads = 256;

template <int EQ, int DIM>
struct Planes {
  static constexpr int NT = DIM + 2;                     // Taylor variables
  static constexpr int NB = EQ == 1 ? DIM : 0;           // field averages
  static constexpr int NC = EQ == 1 ? (DIM == 2 ? 3 : 8) : 0;  // field coefficients
  static constexpr int NV = NT + NB, NS = NT * DIM + NC;
  static constexpr int NP = NV + NS;
  // interchange plane of average v and of derivative coefficient k
  __device__ __forceinline__ static constexpr int avg(int v) {
    return v < NT ? v * (DIM + 1) : NT * (DIM + 1) + (v - NT);
  }
  __device__ __forceinline__ static constexpr int slope(int k) {
    return k < NT * DIM ? (k / DIM) * (DIM + 1) + 1 + k % DIM : NT * (DIM + 1) + NB + (k - NT * DIM);
  }
};

__device__ __forceinline__ int problem_of_block(const LoadProb* tab, int nprob, int b) {
  int lo = 0, hi = nprob - 1;
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (tab[mid].blk0 <= b) lo = mid;
    else hi = mid - 1;
  }
  return lo;
}

// Courant signal speed of one cell's averages (as in the stage kernels' reduction);
// a non-physical or non-finite state sets err and counts as zero.
template <int EQ, int DIM, class TC>
__device__ __forceinline__ TC signal_speed(const Gas<TC>& G, const double* a, const double* ih,
                                           unsigned& err) {
  constexpr int NV = Planes<EQ, DIM>::NV;
  TC c[NV], W[NV], s[DIM];
#pragma unroll
  for (int v = 0; v < NV; ++v) c[v] = Cvt<TC>::to_tc(a[v]);
  if constexpr (DIM == 2) prims2d<EQ, TC>(G, c, W, err);
  else if constexpr (EQ == 0) prims3d<TC>(G, c, W, err);
  else prims3m<TC>(G, c, W, err);
  if constexpr (EQ == 0) {
    s[0] = sqrts(G.g * W[DIM + 1] * rcpv(W[0]));
#pragma unroll
    for (int d = 1; d < DIM; ++d) s[d] = s[0];
  } else {
    TC b2 = TC(0);
#pragma unroll
    for (int d = 0; d < DIM; ++d) b2 += W[DIM + 2 + d] * W[DIM + 2 + d];
#pragma unroll
    for (int d = 0; d < DIM; ++d) s[d] = fast_speed(G, W[0], W[DIM + 1], b2, W[DIM + 2 + d]);
  }
  TC sp = TC(0);
#pragma unroll
  for (int d = 0; d < DIM; ++d) sp += (fabs(W[1 + d]) + s[d]) * TC(ih[d]);
  if (!courant_ok(sp, W[0], W[DIM + 1])) {
    err |= ERR_NONPHYS;
    sp = TC(0);
  }
  return sp;
}

template <int EQ, int DIM, class TS>
__global__ void __launch_bounds__(kLoadThreads) state_load_kernel(const LoadArgs<TS> A) {
  using P = Planes<EQ, DIM>;
  const int ip = problem_of_block(A.tab, A.nprob, blockIdx.x);
  const LoadProb p = A.tab[ip];
  const Gas<TS> G = gas_of<TS>(A.gas);
  const size_t n = (size_t)p.ncell;
  double* c0 = A.c0 + p.c0_off;
  TS* sl = A.sl + p.sl_off;
  TS m = TS(0);
  unsigned err = 0;
  const long step = (long)p.nblk * kLoadThreads;
  for (long i = (long)(blockIdx.x - p.blk0) * kLoadThreads + threadIdx.x; i < p.ncell; i += step) {
    double a[P::NV];
    if (A.src) {
      const double* s = A.src + p.plane_off + i;
      double g[P::NS];
#pragma unroll
      for (int v = 0; v < P::NV; ++v) a[v] = s[P::avg(v) * n];
#pragma unroll
      for (int k = 0; k < P::NS; ++k) g[k] = s[P::slope(k) * n];
#pragma unroll
      for (int v = 0; v < P::NV; ++v) c0[v * n + i] = a[v];
#pragma unroll
      for (int k = 0; k < P::NS; ++k) sl[k * n + i] = (TS)g[k];
    } else {
#pragma unroll
      for (int v = 0; v < P::NV; ++v) a[v] = c0[v * n + i];
    }
    const TS sp = signal_speed<EQ, DIM, TS>(G, a, p.ih, err);
    m = sp > m ? sp : m;
  }
  // block and grid maximum; the problem's last block commits
  __shared__ TS red[kLoadThreads / 32];
  __shared__ unsigned s_err;
  if (threadIdx.x == 0) s_err = 0;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const TS t = __shfl_xor_sync(0xffffffffu, m, o);
    m = t > m ? t : m;
  }
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = m;
  __syncthreads();
  if (err) atomicOr(&s_err, err);
  __syncthreads();
  if (threadIdx.x != 0) return;
#pragma unroll
  for (int w = 1; w < kLoadThreads / 32; ++w) m = red[w] > m ? red[w] : m;
  LoadAcc* acc = A.acc + ip;
  atomicMax(&acc->vmax, (unsigned long long)__double_as_longlong(Cvt<TS>::to_f64(m)));
  if (s_err) atomicOr(&acc->err, s_err);
  __threadfence();
  if (atomicAdd(&acc->ticket, 1u) != (unsigned)p.nblk - 1) return;
  __threadfence();
  const double vm = __longlong_as_double((long long)atomicExch(&acc->vmax, 0ull));
  unsigned e = atomicExch(&acc->err, 0u);
  acc->ticket = 0u;
  if (!(vm > 0.0)) e |= ERR_NONPHYS;
  Ctl* ctl = A.ctl + ip;
  ctl->vmax_cur = vm;
  ctl->dt_cur = A.cfl / vm;
  ctl->vmax_next = 0ull;
  ctl->t = 0.0;
  ctl->dt_last = 0.0;
  ctl->step = 0;
  ctl->ticket = 0u;
  ctl->err = e;
  ctl->err_step = e ? 0 : -1;
  A.host[ip] = *ctl;
}

template <int EQ, int DIM, class TS>
__global__ void __launch_bounds__(kLoadThreads)
    state_save_kernel(const LoadProb* tab, int nprob, const double* c0a, const TS* sla, double* dst) {
  using P = Planes<EQ, DIM>;
  const LoadProb p = tab[problem_of_block(tab, nprob, blockIdx.x)];
  const size_t n = (size_t)p.ncell;
  const double* c0 = c0a + p.c0_off;
  const TS* sl = sla + p.sl_off;
  const long step = (long)p.nblk * kLoadThreads;
  for (long i = (long)(blockIdx.x - p.blk0) * kLoadThreads + threadIdx.x; i < p.ncell; i += step) {
    double* d = dst + p.plane_off + i;
    double a[P::NV];
    TS g[P::NS];
#pragma unroll
    for (int v = 0; v < P::NV; ++v) a[v] = c0[v * n + i];
#pragma unroll
    for (int k = 0; k < P::NS; ++k) g[k] = sl[k * n + i];
#pragma unroll
    for (int v = 0; v < P::NV; ++v) d[P::avg(v) * n] = a[v];
#pragma unroll
    for (int k = 0; k < P::NS; ++k) d[P::slope(k) * n] = (double)g[k];
  }
}

}  // namespace

int load_blocks(long ncell) {
  const long b = (ncell + kLoadThreads - 1) / kLoadThreads, cap = 152L * 8;
  return (int)(b < cap ? b : cap);
}

template <class TS>
cudaError_t launch_state_load(int eq, int dim, int blocks, const LoadArgs<TS>& A, cudaStream_t st) {
  if (dim == 2) {
    if (eq == 0) state_load_kernel<0, 2, TS><<<blocks, kLoadThreads, 0, st>>>(A);
    else state_load_kernel<1, 2, TS><<<blocks, kLoadThreads, 0, st>>>(A);
  } else {
    if (eq == 0) state_load_kernel<0, 3, TS><<<blocks, kLoadThreads, 0, st>>>(A);
    else state_load_kernel<1, 3, TS><<<blocks, kLoadThreads, 0, st>>>(A);
  }
  return cudaGetLastError();
}

template <class TS>
cudaError_t launch_state_save(int eq, int dim, int blocks, const LoadProb* tab, int nprob,
                              const double* c0, const TS* sl, double* dst, cudaStream_t st) {
  if (dim == 2) {
    if (eq == 0) state_save_kernel<0, 2, TS><<<blocks, kLoadThreads, 0, st>>>(tab, nprob, c0, sl, dst);
    else state_save_kernel<1, 2, TS><<<blocks, kLoadThreads, 0, st>>>(tab, nprob, c0, sl, dst);
  } else {
    if (eq == 0) state_save_kernel<0, 3, TS><<<blocks, kLoadThreads, 0, st>>>(tab, nprob, c0, sl, dst);
    else state_save_kernel<1, 3, TS><<<blocks, kLoadThreads, 0, st>>>(tab, nprob, c0, sl, dst);
  }
  return cudaGetLastError();
}

template cudaError_t launch_state_load<double>(int, int, int, const LoadArgs<double>&, cudaStream_t);
template cudaError_t launch_state_load<float>(int, int, int, const LoadArgs<float>&, cudaStream_t);
template cudaError_t launch_state_save<double>(int, int, int, const LoadProb*, int, const double*,
                                               const double*, double*, cudaStream_t);
template cudaError_t launch_state_save<float>(int, int, int, const LoadProb*, int, const double*,
                                              const float*, double*, cudaStream_t);

}  // namespace dgk
