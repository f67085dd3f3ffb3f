// V-cycle kernels of small levels: one block per quarter brick.
//
// A level of a few hundred bricks or less does not fill the GPU with one
// 512-thread block per brick, and what its sweeps cost is latency: the 27
// FP64 multiply-adds of 16 warps pass one after the other through one SM's
// FP64 pipe (16 clocks a warp instruction, 3.3 us a brick) while most SMs
// idle, after two dependent rounds of loads.  Here a brick is cut into four
// slabs of two z-layers, 128 nodes and one 128-thread block each, so a
// brick's multiply-adds take a quarter of that; and since the operator
// (coefficients, weights, activity bits, brick tables) is constant during a
// solve, it is read into registers before the kernel waits for its
// predecessor (pdl_early), so that after the wait one round of loads of the
// vector is left.  The order of every sum is that of the one-brick kernels
// (spfd_cycle.cu): results are the same bit for bit.
#include "spfd_internal.cuh"
#include "spfd_tile.cuh"

namespace spfd {

constexpr int SLAB = 128;               // nodes (and threads) per slab
constexpr int SLABS = BV / SLAB;        // slabs per brick

// This thread's slot of the slab: FP64 (compaction) the slab's n-th active
// slot for thread n, FP32 its own.  mine: the thread computes at ts; idle:
// its own slot q * SLAB + t is inactive and gets the zero-row result.
template <typename T>
__device__ __forceinline__ SlotMap slab_slot(const Grid &g, int bk, int q) {
  const int t = threadIdx.x;
  const uint4 a = __ldg(reinterpret_cast<const uint4 *>(g.act + (size_t)bk * 16) + q);
  const unsigned own = t < 32 ? a.x : t < 64 ? a.y : t < 96 ? a.z : a.w;
  SlotMap m;
  m.idle = !((own >> (t & 31)) & 1u);
  if constexpr (!compact27<T>()) {
    m.mine = !m.idle;
    m.ts = q * SLAB + t;
  } else {
    const int c0 = __popc(a.x), c1 = c0 + __popc(a.y), c2 = c1 + __popc(a.z),
              c3 = c2 + __popc(a.w);
    m.mine = t < c3;
    const int j = (t >= c0) + (t >= c1) + (t >= c2);
    unsigned w = j == 0 ? a.x : j == 1 ? a.y : j == 2 ? a.z : a.w;
    int k = t - (j == 0 ? 0 : j == 1 ? c0 : j == 2 ? c1 : c2);
    m.ts = m.mine ? q * SLAB + j * 32 + nth_bit(w, k) : q * SLAB;
  }
  return m;
}

// Residual r = b - A x (JAC = false) or weighted-Jacobi sweep
// out = x + wdinv (b - A x) (JAC = true) on slab blockIdx.x & 3 of brick
// blockIdx.x >> 2: the slab's 4 x 10 x 10 values of x (two layers and the
// halo) go to shared memory.
template <typename T, bool JAC>
__global__ void __launch_bounds__(SLAB)
k_slab27(Grid g, const T *__restrict__ st, const T *__restrict__ wdinv, const T *x,
         const T *b, T *out) {
  __shared__ T tl[4][10][10];
  pdl_trigger();
  const int bk = blockIdx.x / SLABS, q = blockIdx.x % SLABS, t = threadIdx.x;
  const size_t S = (size_t)g.nb * BV, base = (size_t)bk * BV;
  const SlotMap m = slab_slot<T>(g, bk, q);
  T cf[27];
  if (m.mine) load27(st, S, base + m.ts, cf);
  const size_t sa = base + m.ts, si = base + q * SLAB + t;
  T wa = T(0), wi = T(0);
  if (JAC) {
    if (m.mine) wa = wdinv[sa];
    if (m.idle) wi = wdinv[si];
  }
  // where this thread's tile values (400 over 128 threads) are read from
  constexpr int NV = (400 + SLAB - 1) / SLAB;
  int src[NV];
#pragma unroll
  for (int k = 0; k < NV; ++k) {
    const int u = t + k * SLAB;
    src[k] = -1;
    if (u < 400) {
      const int z = 2 * q - 1 + u / 100, y = (u / 10) % 10 - 1, xx = u % 10 - 1;
      const int e = sidx(xx >> 3, y >> 3, z >> 3);
      const int nb = e == 13 ? bk : __ldg(&g.nbr[(size_t)bk * 27 + e]);
      if (nb >= 0) src[k] = nb * BV + ((z & 7) * 8 + (y & 7)) * 8 + (xx & 7);
    }
  }
  const size_t off = (size_t)blockIdx.y * S;
  x += off; b += off; out += off;
  pdl_wait();
  T v[NV];
#pragma unroll
  for (int k = 0; k < NV; ++k) v[k] = src[k] >= 0 ? x[src[k]] : T(0);
  const T ba = m.mine ? b[sa] : T(0), bi = m.idle ? b[si] : T(0);
#pragma unroll
  for (int k = 0; k < NV; ++k)
    if (t + k * SLAB < 400) (&tl[0][0][0])[t + k * SLAB] = v[k];
  __syncthreads();
  auto at = [&](int ts, int dz, int dy, int dx) {
    return tl[((ts >> 6) & 1) + 1 + dz][((ts >> 3) & 7) + 1 + dy][(ts & 7) + 1 + dx];
  };
  if (m.idle) {  // zero row: r = b
    if (JAC) out[si] = at(t, 0, 0, 0) + wi * bi;
    else out[si] = bi;
  }
  if (m.mine) {
    T acc = 0;
#pragma unroll
    for (int e = 0; e < 27; ++e)
      acc += cf[e] * at(m.ts, e / 9 - 1, (e / 3) % 3 - 1, e % 3 - 1);
    const T r = ba - acc;
    if (JAC) out[sa] = at(m.ts, 0, 0, 0) + wa * r;
    else out[sa] = r;
  }
}

// Restriction onto slab blockIdx.x & 3 of coarse brick blockIdx.x >> 2 (its
// 5 x 17 x 17 fine values in shared memory); with xc, also the coarse level's
// first sweep from the zero guess, xc = wdinv b.
template <typename T>
__global__ void __launch_bounds__(SLAB)
k_slab_restrict(Grid gc, size_t Sf, const T *__restrict__ P, const T *__restrict__ wdinv,
                const T *rf, T *bc, T *xc) {
  __shared__ T fs[5][17][17];
  __shared__ int sk[27];
  pdl_trigger();
  const int bk = blockIdx.x / SLABS, q = blockIdx.x % SLABS, t = threadIdx.x;
  const size_t Sc = (size_t)gc.nb * BV, s = (size_t)bk * BV + q * SLAB + t;
  if (t < 27) sk[t] = gc.kid[(size_t)bk * 27 + t];
  const bool on = (__ldg(&gc.act[(size_t)bk * 16 + q * 4 + (t >> 5)]) >> (t & 31)) & 1u;
  T w[27];
  if (on) load27(P, Sc, s, w);
  const T wd = xc ? wdinv[s] : T(0);
  __syncthreads();
  constexpr int NF = 5 * 289, NV = (NF + SLAB - 1) / SLAB;
  int src[NV];
#pragma unroll
  for (int k = 0; k < NV; ++k) {
    const int u = t + k * SLAB;
    src[k] = -1;
    if (u < NF) {
      const int fz = 4 * q + u / 289, fy = (u / 17) % 17, fx = u % 17;
      const int nb = sk[((fz + 7) >> 3) * 9 + ((fy + 7) >> 3) * 3 + ((fx + 7) >> 3)];
      if (nb >= 0)
        src[k] = nb * BV + (((fz - 1) & 7) * 8 + ((fy - 1) & 7)) * 8 + ((fx - 1) & 7);
    }
  }
  rf += (size_t)blockIdx.y * Sf;
  bc += (size_t)blockIdx.y * Sc;
  if (xc) xc += (size_t)blockIdx.y * Sc;
  pdl_wait();
  T v[NV];
#pragma unroll
  for (int k = 0; k < NV; ++k) v[k] = src[k] >= 0 ? rf[src[k]] : T(0);
#pragma unroll
  for (int k = 0; k < NV; ++k)
    if (t + k * SLAB < NF) (&fs[0][0][0])[t + k * SLAB] = v[k];
  __syncthreads();
  T acc = 0;
  if (on) {
    const int cx = 2 * (t & 7) + 1, cy = 2 * ((t >> 3) & 7) + 1, cz = 2 * (t >> 6) + 1;
#pragma unroll
    for (int d = 0; d < 27; ++d)
      acc += w[d] * fs[cz + d / 9 - 1][cy + (d / 3) % 3 - 1][cx + d % 3 - 1];
  }
  bc[s] = acc;
  if (xc) xc[s] = wd * acc;
}

template <typename T>
void launch_slab27(const Grid &g, const T *st27, const T *wdinv, const T *x, const T *b, T *out,
                   cudaStream_t st, int nk) {
  const dim3 grid((unsigned)g.nb * SLABS, (unsigned)nk);
  if (wdinv) pdl_early(k_slab27<T, true>, grid, SLAB, st)(g, st27, wdinv, x, b, out);
  else pdl_early(k_slab27<T, false>, grid, SLAB, st)(g, st27, wdinv, x, b, out);
}
template <typename T>
void launch_slab_restrict(const Grid &gc, size_t Sf, const T *P, const T *wdinv, const T *rf,
                          T *bc, T *xc, cudaStream_t st, int nk) {
  pdl_early(k_slab_restrict<T>, dim3((unsigned)gc.nb * SLABS, (unsigned)nk), SLAB, st)(
      gc, Sf, P, wdinv, rf, bc, xc);
}
#define INST_SLAB(T)                                                                       \
  template void launch_slab27<T>(const Grid &, const T *, const T *, const T *, const T *, \
                                 T *, cudaStream_t, int);                                  \
  template void launch_slab_restrict<T>(const Grid &, size_t, const T *, const T *,        \
                                        const T *, T *, T *, cudaStream_t, int);
INST_SLAB(double)
INST_SLAB(float)

}  // namespace spfd
