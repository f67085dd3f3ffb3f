// Deterministic sums over a grid, finished on the device by its last block.
#pragma once

#include "spfd_internal.cuh"

namespace spfd {

// ------------------------------------------------------------ accumulators
// Per-thread running sum: FP64 for double kernels, compensated FP32 for float
// kernels (about FP64 accuracy over the few dozen terms a thread adds).
template <typename T> struct Acc;
template <> struct Acc<double> {
  double s = 0.0;
  __device__ __forceinline__ void add(double v) { s += v; }
  __device__ __forceinline__ double get() const { return s; }
};
template <> struct Acc<float> {
  float s = 0.f, c = 0.f;
  __device__ __forceinline__ void add(float v) {
    const float y = v - c;
    const float t = s + y;
    c = (t - s) - y;
    s = t;
  }
  __device__ __forceinline__ double get() const { return (double)s - (double)c; }
};

// ------------------------------------------------------------ reductions
// Block sums of the threads' NV FP64 values, left in warp 0 (every lane),
// for blocks of at most MT threads.  The values pass through shared memory
// and warp 0 adds them (lane l the values of threads l, l + 32, ..., then a
// butterfly): NV * (warps + 4) FP64 warp instructions per block, against
// 5 NV per warp plus 5 NV for a butterfly in every warp, on GB300's narrow
// FP64 pipe.  The NV chains of dependent additions run side by side and their
// loads ahead of them (MT bounds the loop): the tail of a reduction is their
// latency, once in each block and once more in the last one (32^3 sphere
// solve 1107 -> 1082 us, 16 mm step 2058 -> 2037; no change at 2 mm).
template <int NV, int MT = NT>
__device__ __forceinline__ void block_sum(double (&v)[NV]) {
  __shared__ double sm[NV][MT];
  const int t = threadIdx.x, lane = t & 31, w = t >> 5;
  const int nw = (blockDim.x + 31) >> 5;
#pragma unroll
  for (int k = 0; k < NV; ++k) sm[k][t] = v[k];
  __syncthreads();
  if (w == 0) {
#pragma unroll
    for (int k = 0; k < NV; ++k) v[k] = sm[k][lane];
#pragma unroll
    for (int i = 1; i < MT / 32; ++i)
      if (i < nw)
#pragma unroll
        for (int k = 0; k < NV; ++k) v[k] += sm[k][lane + 32 * i];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1)
#pragma unroll
      for (int k = 0; k < NV; ++k) v[k] += __shfl_xor_sync(0xffffffffu, v[k], o);
  }
  __syncthreads();
}

// The tail of the grid reductions, once thread 0 has written this block's NV
// partials: a ticket finds the last of the nblk blocks, which adds every
// block's partials in a fixed order.  Returns true in thread 0 of the last
// block, with tot[] = grid totals.
template <int NV, int MT = NT>
__device__ bool grid_finish(double *partials, unsigned *ticket, double (&tot)[NV],
                            unsigned nblk) {
  __shared__ bool last;
  if (threadIdx.x == 0) {
    __threadfence();
    unsigned prev = atomicAdd(ticket, 1u);
    last = prev == nblk - 1;
  }
  __syncthreads();
  if (!last) return false;
  __threadfence();
  double a[NV];
#pragma unroll
  for (int k = 0; k < NV; ++k) a[k] = 0.0;
  for (unsigned i = threadIdx.x; i < nblk; i += blockDim.x)
#pragma unroll
    for (int k = 0; k < NV; ++k) a[k] += __ldcg(&partials[(size_t)i * NV + k]);
  block_sum<NV, MT>(a);
  if (threadIdx.x != 0) return false;
#pragma unroll
  for (int k = 0; k < NV; ++k) tot[k] = a[k];
  *ticket = 0u;
  return true;
}

// Grid totals of the threads' values over nblk blocks, this one number blk.
template <int NV, int MT = NT>
__device__ bool grid_sum(double (&v)[NV], double *partials, unsigned *ticket,
                         double (&tot)[NV], unsigned blk, unsigned nblk) {
  block_sum<NV, MT>(v);
  if (threadIdx.x == 0)
#pragma unroll
    for (int k = 0; k < NV; ++k) partials[(size_t)blk * NV + k] = v[k];
  return grid_finish<NV, MT>(partials, ticket, tot, nblk);
}

// hi + lo += oh + ol with the rounding error of the high parts kept (TwoSum).
__device__ __forceinline__ void two_sum_add(float &hi, float &lo, float oh, float ol) {
  const float s = hi + oh, bb = s - hi;
  const float e = (hi - (s - bb)) + (oh - bb);
  hi = s;
  lo = lo + ol + e;
}

// A sum of three FP32 parts h + m + l, for adding many FP32 pairs without
// the FP64 pipe and with no larger error than FP64 additions: the rounding
// errors of the high parts go to the middle ones, and theirs to the low ones,
// whose own are below (c 2^-24)^3 of the sum of magnitudes after c additions
// in a row.
struct Sum3 {
  float h, m, l;
};
__host__ __device__ __forceinline__ float two_sum(float a, float b, float &err) {
  const float s = a + b, bb = s - a;
  err = (a - (s - bb)) + (b - bb);
  return s;
}
__host__ __device__ __forceinline__ void sum3_add(Sum3 &t, float h, float m, float l) {
  float e1, e2, e3;
  t.h = two_sum(t.h, h, e1);
  t.m = two_sum(t.m, m, e2);
  t.m = two_sum(t.m, e1, e3);
  t.l = (t.l + l) + (e2 + e3);
}
__host__ __device__ __forceinline__ double sum3_value(const Sum3 &t) {
  return (double)t.h + ((double)t.m + (double)t.l);
}
__device__ __forceinline__ void sum3_warp(Sum3 &t) {  // the warp's total in every lane
#pragma unroll
  for (int o = 16; o > 0; o >>= 1)
    sum3_add(t, __shfl_xor_sync(0xffffffffu, t.h, o), __shfl_xor_sync(0xffffffffu, t.m, o),
             __shfl_xor_sync(0xffffffffu, t.l, o));
}

// grid_sum for per-thread FP32 pairs (value hi + lo): the warps and the block
// add them as TwoSum pairs in FP32, and only the block's total is widened to
// FP64 (in thread 0).  An FP64 conversion or addition takes a 16-clock slot
// of GB300's narrow FP64 pipe for its warp whatever its lane mask, so
// widening in every thread put an FP64 tail of several microseconds at the
// end of the FP32 reduction kernels.
template <int NV, int MT = NT>
__device__ bool grid_sum_f32(float (&hi)[NV], float (&lo)[NV], double *partials,
                             unsigned *ticket, double (&tot)[NV], unsigned blk,
                             unsigned nblk) {
  __shared__ float sh[32][NV], sl[32][NV];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int nw = (blockDim.x + 31) >> 5;
#pragma unroll
  for (int k = 0; k < NV; ++k)
#pragma unroll
    for (int o = 16; o > 0; o >>= 1)
      two_sum_add(hi[k], lo[k], __shfl_xor_sync(0xffffffffu, hi[k], o),
                  __shfl_xor_sync(0xffffffffu, lo[k], o));
  if (lane == 0)
#pragma unroll
    for (int k = 0; k < NV; ++k) {
      sh[w][k] = hi[k];
      sl[w][k] = lo[k];
    }
  __syncthreads();
  if (w == 0) {
#pragma unroll
    for (int k = 0; k < NV; ++k) {
      float h = lane < nw ? sh[lane][k] : 0.f, l = lane < nw ? sl[lane][k] : 0.f;
#pragma unroll
      for (int o = 16; o > 0; o >>= 1)
        two_sum_add(h, l, __shfl_xor_sync(0xffffffffu, h, o), __shfl_xor_sync(0xffffffffu, l, o));
      if (lane == 0) partials[(size_t)blk * NV + k] = (double)h + (double)l;
    }
  }
  return grid_finish<NV, MT>(partials, ticket, tot, nblk);
}

// One warp's part of NV sums in FP32: the thread's N values of each and the
// warp's are added without rounding error (TwoSum), and lane 0 stores the
// pairs (hi, lo) at pairs[NV warp + k], for launch_finish_pairs.  (Finishing
// the sums in the same launch, with a fence and a ticket per warp, doubled
// the time of the FP32 CG operator, 48 -> 94 us on the 2 mm body.)
template <int NV, int N>
__device__ __forceinline__ void warp_pairs(const float (&v)[NV][N], int warp, double *pairs) {
#pragma unroll
  for (int k = 0; k < NV; ++k) {
    float hi = v[k][0], lo = 0.f;
#pragma unroll
    for (int i = 1; i < N; ++i) {
      const float sh = hi + v[k][i], bb = sh - hi;
      lo += (hi - (sh - bb)) + (v[k][i] - bb);
      hi = sh;
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1)
      two_sum_add(hi, lo, __shfl_xor_sync(0xffffffffu, hi, o),
                  __shfl_xor_sync(0xffffffffu, lo, o));
    if ((threadIdx.x & 31) == 0)
      reinterpret_cast<float2 *>(pairs)[(size_t)NV * warp + k] = make_float2(hi, lo);
  }
}

// grid_sum of per-thread accumulators: FP64 sums directly, compensated FP32
// sums (value s - c) as FP32 pairs.
template <typename T, int NV, int MT = NT>
__device__ bool grid_sum_acc(const Acc<T> (&a)[NV], double *partials, unsigned *ticket,
                             double (&tot)[NV], unsigned blk, unsigned nblk) {
  if constexpr (sizeof(T) == 8) {
    double v[NV];
#pragma unroll
    for (int k = 0; k < NV; ++k) v[k] = a[k].s;
    return grid_sum<NV, MT>(v, partials, ticket, tot, blk, nblk);
  } else {
    float h[NV], l[NV];
#pragma unroll
    for (int k = 0; k < NV; ++k) {
      h[k] = a[k].s;
      l[k] = -a[k].c;
    }
    return grid_sum_f32<NV, MT>(h, l, partials, ticket, tot, blk, nblk);
  }
}

// p.q into the Scalars, and the CG step alpha = rz / p.q.
__device__ __forceinline__ void set_pq(Scalars *sc, double pq) {
  sc->pq = pq;
  const double al = pq > 0.0 ? sc->rz / pq : 0.0;
  sc->alpha = al;
  sc->alpha_f = (float)al;
}

// r.z (tot[0]) and the sum of z over the unknowns (tot[1]) into the Scalars:
// beta = rz / rz_old (0 on the first iteration or after a restart) and the
// mean of z for its projection.
__device__ __forceinline__ void set_rz(Scalars *sc, const double (&tot)[2], int first) {
  const double old = sc->rz;
  sc->rz_old = old;
  sc->rz = tot[0];
  const double beta = (first || sc->restart || old == 0.0) ? 0.0 : tot[0] / old;
  sc->restart = 0;
  sc->beta = beta;
  sc->beta_f = (float)beta;
  sc->zsum = tot[1];
  sc->zmean = tot[1] * sc->inv_ndof;
  sc->zmean_f = (float)sc->zmean;
}

}  // namespace spfd
