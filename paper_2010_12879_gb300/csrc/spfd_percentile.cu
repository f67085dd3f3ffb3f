// Step 6 of the pipeline (Sec. II-A, step 6; Sec. III-E): the 99th
// percentile of the voxel-averaged |E|, per tissue and over the whole body.
//
// The p-quantile of n values is the nearest-rank value: the k-th smallest,
// k the least integer >= p * n in exact arithmetic (k >= 1).  It is taken
// over the conducting voxels of the context (sigma > 0) carrying each label
// 0..L-1 (groups 0..L-1) and over every conducting voxel (group L).
//
// Method: an exact most-significant-digit radix select on the bit patterns
// of |E|.  For non-negative doubles the IEEE-754 bit pattern, read as an
// unsigned 64-bit integer, orders like the value, so selecting the k-th
// smallest key selects the k-th smallest value and the answer is one of the
// inputs, bit for bit.
//   1. field digit: one pass over the mask, E and the labels counts the first
//      digit (16 bits after the sign for up to 62 labels, 32 buckets an
//      octave) of every conducting voxel in its group's row of a table in
//      L2; the body's row is the sum of the rows;
//   2. select: a block per group sums its row (the group's voxels), forms the
//      rank and finds the bucket that holds it;
//   3. while these buckets hold more than an eighth of the voxels (a narrow or
//      tied field, many groups), the next digit is counted over the field in
//      the same way, for the voxels in their group's bucket and for those in
//      the body's;
//   4. collect: another pass lists the keys in their group's bucket or in
//      the body's (their number is known from the buckets);
//   5. further digits over the list: histogram, then select.
// An ordinary field is read twice and nothing is moved: 0.81 -> 0.42 ms per
// call on the 2 mm body with 40 labels, against counting, scattering every
// key twice (18 M keys, its tissue's segment and the body's) and rereading
// the segments for two digits.
//
// What a pass costs beyond its reads is atomics on one address, about 4 ns
// each.  A warp adds equal counters together, and equal steps of its eight;
// a table with few rows is kept in several copies (PctTable), added up before
// the select; a warp takes its places in the list with one atomic for its
// eight steps; and a narrow field is not listed.  Us per call on the 2 mm
// body's grid, one table, two atomics a warp step and every key listed
// against this: log-normal field without labels 1798 -> 391, with 40 labels
// 529 -> 488, with 2048 1358 -> 965; values within 1e-3 of each other 2879 ->
// 532 (40 labels); one value 1958 -> 574; 32^3 voxels, 40 labels 168 -> 166.
#include <cstring>

#include "spfd_ctx.cuh"

namespace spfd {
namespace {

constexpr int PT = 256;              // threads per block
constexpr int PCT_UNROLL = 8;        // voxels per thread and step
constexpr int PCT_BINS = 1 << 13;    // bins of the later digits' histograms
constexpr int PCT_MAX_LABELS = 2048;
constexpr unsigned long long PCT_LIST_MIN = 65536;  // keys that are always listed
constexpr int PCT_BAD_E = 1;         // status bit: negative or non-finite |E|
constexpr int PCT_BAD_RANK = 2;      // status bit: a rank or list entry out of place

constexpr long long PCT_TABLE = 4LL << 20;  // counters of the field digits' table
// Copies of the rows (as many as the table holds) and of the body's row: one
// for every 2^18 voxels, at most so many.
constexpr int PCT_COPY_VOXELS = 18;
constexpr int PCT_COPIES = 32;
constexpr int PCT_BODY_COPIES = 16;

// Width of a field digit: 16 bits while the table of G + 1 rows stays
// within 16 MB, a bit less for every doubling beyond.
int field_width(int G) {
  int w = 16;
  while (w > 8 && ((long long)(G + 1) << w) > PCT_TABLE) --w;
  return w;
}

// Key of a conducting voxel's |E|: its bit pattern (+0 for -0), or flags it.
__device__ __forceinline__ unsigned long long e_key(double e, int *status) {
  const unsigned long long u = f64_bits(e);
  if ((u << 1) == 0ull) return 0ull;
  if (u >= 0x7ff0000000000000ull) {  // negative, infinite or NaN
    atomicOr(status, PCT_BAD_E);
    return 0ull;
  }
  return u;
}

// Least integer k >= p * n, at least 1 (0 when n = 0), p = m / 2^s (p in (0,
// 1] read as its binary fraction, m < 2^54).
__device__ unsigned long long rank_of(unsigned long long m, int s, unsigned long long n) {
  if (n == 0) return 0;
  if (s >= 127) return 1;
  const unsigned __int128 one = 1, x = (unsigned __int128)m * n;
  const unsigned long long k = (unsigned long long)((x + ((one << s) - 1)) >> s);
  return k < 1 ? 1 : k;
}

// Calls f(on, key, group) with PCT_UNROLL voxels a thread (on: the voxel
// conducts); a group is the label when it is one of 0..L-1, else L (the voxel
// counts for the body only).  Whole warps call f.
template <typename F>
__device__ __forceinline__ void each_voxels(const unsigned char *__restrict__ mask,
                                            const double *__restrict__ E,
                                            const int *__restrict__ labels, long long nv, int L,
                                            int *status, const F &f) {
  const long long step = (long long)gridDim.x * PT * PCT_UNROLL;
  for (long long base = (long long)blockIdx.x * PT * PCT_UNROLL; base < nv; base += step) {
    bool on[PCT_UNROLL], any = false;
    double e[PCT_UNROLL];
    int lab[PCT_UNROLL];
#pragma unroll
    for (int q = 0; q < PCT_UNROLL; ++q) {
      const long long v = base + q * PT + threadIdx.x;
      on[q] = v < nv && mask[v];
      any |= on[q];
    }
    if (!__any_sync(0xffffffffu, any)) continue;
#pragma unroll
    for (int q = 0; q < PCT_UNROLL; ++q) {
      const long long v = base + q * PT + threadIdx.x;
      e[q] = on[q] ? E[v] : 0.0;
      lab[q] = on[q] && labels ? labels[v] : -1;
    }
    unsigned long long key[PCT_UNROLL];
#pragma unroll
    for (int q = 0; q < PCT_UNROLL; ++q) {
      key[q] = on[q] ? e_key(e[q], status) : 0ull;
      if (lab[q] < 0 || lab[q] >= L) lab[q] = L;
    }
    f(on, key, lab);
  }
}

// cnt[i] += times for every lane with on, one atomic per distinct i.
__device__ __forceinline__ void warp_count(unsigned *cnt, unsigned i, bool on,
                                           unsigned times = 1) {
  const unsigned act = __ballot_sync(0xffffffffu, on);
  if (!on) return;
  const unsigned peers = __match_any_sync(act, i);
  if ((int)(threadIdx.x & 31) == __ffs(peers) - 1) atomicAdd(&cnt[i], times * __popc(peers));
}

// The same for PCT_UNROLL counters a lane (NO_COUNT: none); steps in which
// every lane repeats its counter of the step before are added together.
constexpr unsigned NO_COUNT = 0xffffffffu;
__device__ __forceinline__ void warp_counts(unsigned *cnt, const unsigned (&i)[PCT_UNROLL]) {
  unsigned times = 1;
#pragma unroll
  for (int q = 0; q < PCT_UNROLL; ++q) {
    if (q + 1 < PCT_UNROLL && __all_sync(0xffffffffu, i[q] == i[q + 1])) {
      ++times;
      continue;
    }
    warp_count(cnt, i[q], i[q] != NO_COUNT, times);
    times = 1;
  }
}

struct PctGroup {
  unsigned long long count;   // voxels of the group
  unsigned long long rank;    // 1-based rank inside the buckets chosen so far
  unsigned long long prefix;  // the digits chosen so far
  unsigned long long listed;  // keys in the buckets chosen over the field
};

// The table of a field digit: `copies` copies of rows 0..L (a block counts in
// copy blockIdx.x mod copies), then `bcopies` copies of the body's row.  The
// sums land in the first copies.
struct PctTable {
  unsigned *cnt;
  int L, width, copies, bcopies;
  __host__ __device__ size_t rows() const { return (size_t)(L + 1) << width; }
  __host__ __device__ size_t body() const { return copies * rows(); }
  __host__ __device__ size_t size() const { return body() + ((size_t)bcopies << width); }
};

// 1, 3. A digit of every conducting voxel: the first (FIRST), in the rows of
// the groups only, or one further down, of the voxels whose higher digits are
// their group's, and of those whose higher digits are the body's.
template <bool FIRST>
__global__ void __launch_bounds__(PT)
k_pct_field(const unsigned char *__restrict__ mask, const double *__restrict__ E,
            const int *__restrict__ labels, long long nv, PctTable tab, int shift,
            const PctGroup *__restrict__ grp, int *status) {
  extern __shared__ unsigned long long want[];  // higher digits, L + 1 (not FIRST)
  const int L = tab.L, hi = shift + tab.width;
  const unsigned dmask = (1u << tab.width) - 1u;
  unsigned *rows = tab.cnt + (blockIdx.x % tab.copies) * tab.rows();
  unsigned *body = tab.cnt + tab.body() + ((size_t)(blockIdx.x % tab.bcopies) << tab.width);
  if constexpr (!FIRST) {
    for (int g = threadIdx.x; g <= L; g += PT) want[g] = grp[g].prefix >> hi;
    __syncthreads();
  }
  each_voxels(mask, E, labels, nv, L, status,
              [&](const bool (&on)[PCT_UNROLL], const unsigned long long (&k)[PCT_UNROLL],
                  const int (&g)[PCT_UNROLL]) {
    unsigned i[PCT_UNROLL];
#pragma unroll
    for (int q = 0; q < PCT_UNROLL; ++q) {
      const bool in = on[q] && (FIRST || (g[q] < L && (k[q] >> hi) == want[g[q]]));
      i[q] = in ? ((unsigned)g[q] << tab.width) + ((unsigned)(k[q] >> shift) & dmask) : NO_COUNT;
    }
    warp_counts(rows, i);
    if constexpr (!FIRST) {
#pragma unroll
      for (int q = 0; q < PCT_UNROLL; ++q)
        i[q] = on[q] && (k[q] >> hi) == want[L] ? (unsigned)(k[q] >> shift) & dmask : NO_COUNT;
      warp_counts(body, i);
    }
  });
}

// Adds the copies up; after the first digit the body's row is the sum of the
// rows (zero before).  Block y takes rows y, y + gridDim.y, ...
template <bool FIRST>
__global__ void __launch_bounds__(PT) k_pct_rows(PctTable tab) {
  const int bin = blockIdx.x * PT + threadIdx.x;
  if (bin >> tab.width) return;
  unsigned sum = 0;
  for (int g = blockIdx.y; g <= tab.L; g += gridDim.y) {
    unsigned *row = tab.cnt + ((size_t)g << tab.width) + bin, s = 0;
    for (int c = 0; c < tab.copies; ++c) s += row[c * tab.rows()];
    if (tab.copies > 1) *row = s;
    sum += s;
  }
  unsigned *body = tab.cnt + tab.body() + bin;
  if constexpr (FIRST) {
    if (sum) atomicAdd(body, sum);
  } else if (blockIdx.y == 0) {
    unsigned s = 0;
    for (int c = 0; c < tab.bcopies; ++c) s += body[(size_t)c << tab.width];
    *body = s;
  }
}

// The bucket of row (nbin entries, per thread PER consecutive ones of the
// block's PT * PER) that holds the r-th count; *excl: counts before it.
// Every thread of the block calls it; returns -1 where no bucket holds it.
__device__ int pct_bucket(const unsigned *__restrict__ row, int nbin,
                          unsigned long long *total, const unsigned long long *rank_in,
                          unsigned long long m, int s, unsigned long long *excl_out) {
  __shared__ unsigned long long part[PT];
  __shared__ int bucket;
  __shared__ unsigned long long before;
  const int per = (nbin + PT - 1) / PT, b0 = threadIdx.x * per, b1 = min(b0 + per, nbin);
  unsigned long long own = 0;
  for (int b = b0; b < b1; ++b) own += row[b];
  part[threadIdx.x] = own;
  if (threadIdx.x == 0) bucket = -1;
  __syncthreads();
  for (int o = 1; o < PT; o <<= 1) {
    const unsigned long long add = threadIdx.x >= o ? part[threadIdx.x - o] : 0ull;
    __syncthreads();
    part[threadIdx.x] += add;
    __syncthreads();
  }
  const unsigned long long n = part[PT - 1];
  *total = n;
  const unsigned long long r = rank_in ? *rank_in : rank_of(m, s, n);
  unsigned long long cum = part[threadIdx.x] - own;
  if (cum < r && r <= cum + own)
    for (int b = b0; b < b1; ++b) {
      if (cum + row[b] >= r) {
        bucket = b;
        before = cum;
        break;
      }
      cum += row[b];
    }
  __syncthreads();
  *excl_out = before;
  return bucket;
}

// 2. Per group (block L: the body): the digit at `shift` of the group's
// answer, after the first one (FIRST) also the group's count and rank.
template <bool FIRST>
__global__ void __launch_bounds__(PT)
k_pct_select_field(PctTable tab, int shift, unsigned long long m, int s,
                   PctGroup *__restrict__ grp, int *status) {
  const int g = blockIdx.x;
  const unsigned *row = tab.cnt + (g < tab.L ? (size_t)g << tab.width : tab.body());
  PctGroup q{0, 0, 0, 0};
  if constexpr (!FIRST) {
    q = grp[g];
    if (q.count == 0) return;
  }
  unsigned long long n, excl;
  const unsigned long long rank = q.rank;
  const int b = pct_bucket(row, 1 << tab.width, &n, FIRST ? nullptr : &rank, m, s, &excl);
  if (threadIdx.x) return;
  if (FIRST) q.count = n;
  if (q.count) {
    if (b < 0) atomicOr(status, PCT_BAD_RANK);
    else {
      q.rank = (FIRST ? rank_of(m, s, n) : rank) - excl;
      q.prefix |= (unsigned long long)b << shift;
      q.listed = row[b];
    }
  }
  grp[g] = q;
}

// 4. The keys in their group's buckets and in the body's (chosen down to the
// digit at `shift`), with the group.
__global__ void __launch_bounds__(PT)
k_pct_collect(const unsigned char *__restrict__ mask, const double *__restrict__ E,
              const int *__restrict__ labels, long long nv, int L, int shift,
              const PctGroup *__restrict__ grp, unsigned long long *__restrict__ key,
              int *__restrict__ kgrp, unsigned long long cap,
              unsigned long long *__restrict__ cursor, int *status) {
  extern __shared__ unsigned long long want[];  // digits, L + 1
  for (int g = threadIdx.x; g <= L; g += PT) want[g] = grp[g].count ? grp[g].prefix >> shift : ~0ull;
  __syncthreads();
  const unsigned lane = threadIdx.x & 31, below = (1u << lane) - 1u;
  each_voxels(mask, E, labels, nv, L, status,
              [&](const bool (&on)[PCT_UNROLL], const unsigned long long (&k)[PCT_UNROLL],
                  const int (&g)[PCT_UNROLL]) {
    unsigned mt[PCT_UNROLL], mb[PCT_UNROLL], n = 0;
#pragma unroll
    for (int q = 0; q < PCT_UNROLL; ++q) {
      const unsigned long long d = k[q] >> shift;
      mt[q] = __ballot_sync(0xffffffffu, on[q] && g[q] < L && d == want[g[q]]);
      mb[q] = __ballot_sync(0xffffffffu, on[q] && d == want[L]);
      n += __popc(mt[q]) + __popc(mb[q]);
    }
    if (!n) return;
    unsigned long long pos = 0;
    if (lane == 0) pos = atomicAdd(cursor, (unsigned long long)n);
    pos = __shfl_sync(0xffffffffu, pos, 0);
    auto append = [&](unsigned m, unsigned long long kk, int gg) {
      if ((m >> lane) & 1u) {
        const unsigned long long at = pos + __popc(m & below);
        if (at < cap) {  // more than counted: the inputs changed during the call
          key[at] = kk;
          kgrp[at] = gg;
        } else {
          atomicOr(status, PCT_BAD_RANK);
        }
      }
      pos += __popc(m);
    };
#pragma unroll
    for (int q = 0; q < PCT_UNROLL; ++q) {
      append(mt[q], k[q], g[q]);
      append(mb[q], k[q], L);
    }
  });
}

// 5a. Digit histogram of the listed keys that match their group's prefix.
// *listed entries were written; want, as many as the buckets counted, when
// the inputs did not change during the call.  Fewer are flagged, and no entry
// past them is read: its group would be any number.
__global__ void __launch_bounds__(PT)
k_pct_hist(const unsigned long long *__restrict__ key, const int *__restrict__ kgrp,
           const unsigned long long *__restrict__ listed, unsigned long long want,
           const PctGroup *__restrict__ grp, int shift, int width,
           unsigned *__restrict__ hist, int *status) {
  const unsigned long long n = min(*listed, want);
  if (n != want && blockIdx.x == 0 && threadIdx.x == 0) atomicOr(status, PCT_BAD_RANK);
  const int hi = shift + width;
  const unsigned dmask = (1u << width) - 1u;
  const unsigned long long stride = (unsigned long long)gridDim.x * PT;
  for (unsigned long long i0 = (unsigned long long)blockIdx.x * PT; i0 < n; i0 += stride) {
    const unsigned long long i = i0 + threadIdx.x;
    const bool in = i < n;
    const unsigned long long k = in ? key[i] : 0ull;
    const int g = in ? kgrp[i] : 0;
    warp_count(hist, (unsigned)g * PCT_BINS + ((unsigned)(k >> shift) & dmask),
               in && (k >> hi) == (grp[g].prefix >> hi));
  }
}

// 5b. One block per group: the digit whose bucket holds the remaining rank;
// clears the group's row for the next digit.
__global__ void __launch_bounds__(PT)
k_pct_select(unsigned *__restrict__ hist, PctGroup *__restrict__ grp, int shift, int width,
             int *status) {
  const int g = blockIdx.x;
  if (grp[g].count == 0) return;
  unsigned *row = hist + (size_t)g * PCT_BINS;
  unsigned long long n, excl;
  const unsigned long long rank = grp[g].rank;
  const int b = pct_bucket(row, 1 << width, &n, &rank, 0, 0, &excl);
  if (threadIdx.x == 0) {
    if (b < 0) atomicOr(status, PCT_BAD_RANK);
    else {
      grp[g].prefix |= (unsigned long long)b << shift;
      grp[g].rank = rank - excl;
    }
  }
  for (int i = threadIdx.x; i < (1 << width); i += PT) row[i] = 0u;
}

}  // namespace
}  // namespace spfd

using namespace spfd;

extern "C" spfd_status spfd_percentile(spfd_ctx *ctx, const double *E_dev,
                                       const int32_t *labels_dev, int n_labels, double p,
                                       double *values_host, int64_t *counts_host) {
  if (!ctx) return fail(SPFD_EINVAL, "ctx is NULL");
  if (!E_dev || !values_host || (n_labels > 0 && !labels_dev))
    return fail(SPFD_EINVAL, "null argument");
  if (n_labels < 0 || n_labels > PCT_MAX_LABELS)
    return fail(SPFD_EINVAL, "n_labels must be in 0..%d (got %d)", PCT_MAX_LABELS, n_labels);
  if (!(p > 0.0 && p <= 1.0)) return fail(SPFD_EINVAL, "p must be in (0, 1]");
  spfd_ctx *c = ctx;
  cudaStream_t st = c->stream;
  const int L = n_labels, G = L + 1, width = field_width(G);
  const long long nv = (long long)c->nx * c->ny * c->nz;
  // without labels every conducting voxel counts for the body only
  const int *lab = L > 0 ? (const int *)labels_dev : nullptr;
  // p = m / 2^s
  int pe = 0;
  const double pf = std::frexp(p, &pe);
  const unsigned long long pm = (unsigned long long)std::ldexp(pf, 53);
  const int ps = 53 - pe;
  // scratch: the field digits' table, the later digits' (zero between calls),
  // the groups, list cursor and status, and their pinned mirror
  const int many = (int)std::min<long long>(std::max<long long>(nv >> PCT_COPY_VOXELS, 1), PCT_COPIES);
  PctTable tab{nullptr, L, width, 1, std::min(many, PCT_BODY_COPIES)};
  tab.copies = (int)std::max<long long>(std::min<long long>(many, PCT_TABLE / (long long)tab.rows()), 1);
  if (c->pct_tcap < tab.size()) {
    dfree(c, c->pct_first);
    c->pct_tcap = 0;
    TRY(dalloc(c, &c->pct_first, tab.size()));
    c->pct_tcap = tab.size();
  }
  tab.cnt = c->pct_first;
  if (c->pct_gcap < G) {
    dfree(c, c->pct_hist);
    dfree(c, c->pct_grp);
    c->pct_gcap = 0;
    TRY(dalloc(c, &c->pct_hist, (size_t)G * PCT_BINS));
    TRY(dalloc(c, &c->pct_grp, (size_t)4 * G + 2));
    TRY(halloc(c, &c->pct_hgrp, (size_t)4 * G + 2));
    CU(cudaMemsetAsync(c->pct_hist, 0, (size_t)G * PCT_BINS * sizeof(unsigned), st));
    c->pct_gcap = G;
  }
  static_assert(sizeof(PctGroup) == 32, "PctGroup layout");
  PctGroup *grp = (PctGroup *)c->pct_grp;
  unsigned long long *cursor = c->pct_grp + 4 * (size_t)G;
  int *status = (int *)(cursor + 1);
  const size_t small = ((size_t)4 * G + 2) * 8, want_smem = (size_t)G * sizeof(unsigned long long);
  const PctGroup *hg = (const PctGroup *)c->pct_hgrp;
  const int *hstatus = (const int *)(c->pct_hgrp + 4 * (size_t)G + 1);
  CU(cudaMemsetAsync(c->pct_grp, 0, small, st));
  const long long steps = (nv + PT * PCT_UNROLL - 1) / (PT * PCT_UNROLL);
  const int grid = (int)std::max(1LL, std::min(steps, (long long)c->nsm * 8));
  // algorithmic bytes: the mask of every voxel, E and the label of each
  // conducting one (counted from the previous call; all voxels on the first)
  const double ncv = c->pct_nc > 0 ? (double)c->pct_nc : (double)nv;
  // digits over the field, until the chosen buckets hold few enough keys to
  // list (or nothing is left to choose)
  unsigned long long listed = 0;
  int left = 63;
  do {
    const bool first = left == 63;
    tab.width = std::min(width, left);
    left -= tab.width;
    // after the first digit the body's row is a sum into its first copy
    const size_t used = first ? tab.body() + ((size_t)1 << tab.width) : tab.size();
    CU(cudaMemsetAsync(tab.cnt, 0, used * sizeof(unsigned), st));
    const dim3 rgrid(((1 << tab.width) + PT - 1) / PT, std::min(G, std::max(1, (256 * 1024) >> tab.width)));
    if (first) {
      SPFD_LAUNCH(c, "percentile_first", false, 1, nv + 12.0 * ncv, 0,
                  (k_pct_field<true><<<grid, PT, 0, st>>>(c->mask, E_dev, lab, nv, tab, left, grp,
                                                          status)));
      SPFD_LAUNCH(c, "percentile_select", false, 2, 8.0 * tab.rows(), 0,
                  (k_pct_rows<true><<<rgrid, PT, 0, st>>>(tab),
                   k_pct_select_field<true><<<G, PT, 0, st>>>(tab, left, pm, ps, grp, status)));
    } else {
      SPFD_LAUNCH(c, "percentile_field", false, 1, nv + 12.0 * ncv, 0,
                  (k_pct_field<false><<<grid, PT, want_smem, st>>>(c->mask, E_dev, lab, nv, tab,
                                                                   left, grp, status)));
      SPFD_LAUNCH(c, "percentile_select", false, 2, 8.0 * tab.rows(), 0,
                  (k_pct_rows<false><<<rgrid, PT, 0, st>>>(tab),
                   k_pct_select_field<false><<<G, PT, 0, st>>>(tab, left, pm, ps, grp, status)));
    }
    TRY(launch_check("percentile field digit"));
    CU(cudaMemcpyAsync(c->pct_hgrp, c->pct_grp, small, cudaMemcpyDeviceToHost, st));
    TRY(sync_check(c, "percentile field digit"));
    if (*hstatus & PCT_BAD_E)
      return fail(SPFD_EINVAL, "|E| holds a negative or non-finite value on a conducting voxel");
    listed = 0;
    for (int g = 0; g < G; ++g) listed += hg[g].listed;
  } while (left > 0 && !(*hstatus & PCT_BAD_RANK) &&
           listed > std::max<unsigned long long>(hg[L].count / 8, PCT_LIST_MIN));
  c->pct_nc = (long long)hg[L].count;
  if (listed > 0 && left > 0 && !(*hstatus & PCT_BAD_RANK)) {
    if (c->pct_keycap < (long long)listed) {
      dfree(c, c->pct_keys);
      dfree(c, c->pct_keyg);
      c->pct_keycap = 0;
      const size_t cap = (size_t)listed + (size_t)listed / 4;
      TRY(dalloc(c, &c->pct_keys, cap));
      TRY(dalloc(c, &c->pct_keyg, cap));
      c->pct_keycap = (long long)cap;
    }
    SPFD_LAUNCH(c, "percentile_collect", false, 1, nv + 12.0 * ncv + 12.0 * listed, 0,
                (k_pct_collect<<<grid, PT, want_smem, st>>>(c->mask, E_dev, lab, nv, L, left, grp,
                                                            c->pct_keys, c->pct_keyg, listed,
                                                            cursor, status)));
    const int hgrid =
        (int)std::min<unsigned long long>((listed + PT - 1) / PT, (unsigned long long)c->nsm * 8);
    while (left > 0) {
      const int w = std::min(left, 13), shift = left - w;
      SPFD_LAUNCH(c, "percentile_hist", false, 2, 12.0 * listed, 0,
                  (k_pct_hist<<<hgrid, PT, 0, st>>>(c->pct_keys, c->pct_keyg, cursor, listed,
                                                    grp, shift, w, c->pct_hist, status),
                   k_pct_select<<<G, PT, 0, st>>>(c->pct_hist, grp, shift, w, status)));
      left = shift;
    }
    TRY(launch_check("percentile digits"));
    CU(cudaMemcpyAsync(c->pct_hgrp, c->pct_grp, small, cudaMemcpyDeviceToHost, st));
    TRY(sync_check(c, "percentile"));
  }
  TRY(prof_flush(c));
  if (*hstatus & PCT_BAD_RANK) {
    // a row of the later digits may be left behind
    CU(cudaMemsetAsync(c->pct_hist, 0, (size_t)c->pct_gcap * PCT_BINS * sizeof(unsigned), st));
    return fail(SPFD_EINTERNAL, "percentile selection lost its rank (|E| or labels "
                                "changed during the call?)");
  }
  for (int g = 0; g < G; ++g) {
    double v = NAN;
    if (hg[g].count) memcpy(&v, &hg[g].prefix, 8);
    values_host[g] = v;
    if (counts_host) counts_host[g] = (int64_t)hg[g].count;
  }
  return SPFD_OK;
}
