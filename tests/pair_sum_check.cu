// Host check of Sum3 (the three-part FP32 sums of the mixed form's p.q and
// r.z): the finishing kernel's order of additions, on pairs like those the
// row kernels write, against a sum of about 106 bits, beside FP64 additions
// in the order of a grid of 152 blocks.  Prints "ok <cases> <rms error of
// Sum3> <of FP64>", both relative to the sum of magnitudes; exit status 1
// when a case passes its bound: 8 block totals rounded once each and 7 FP64
// additions of them, (8 + 7) 2^-53 of the sum of magnitudes, with one more
// 2^-53 for the low parts' own rounding ((57 2^-24)^3 at most).
#include <cmath>
#include <cstdio>
#include <random>
#include <vector>

#include "spfd_reduce.cuh"

struct Pair { float h, l; };

static double exact(const std::vector<Pair> &p, double &mag) {
  double hi = 0.0, lo = 0.0;
  mag = 0.0;
  auto add = [&](double v) {
    const double s = hi + v, bb = s - hi;
    lo += (hi - (s - bb)) + (v - bb);
    hi = s;
    mag += std::fabs(v);
  };
  for (const Pair &q : p) { add(q.h); add(q.l); }
  return hi + lo;
}

// Butterfly over 32 values, the same tree in every lane: lane 0's.
template <typename T, typename F>
static T warp(std::vector<T> v, const F &add) {
  for (int o = 16; o > 0; o >>= 1) {
    std::vector<T> u = v;
    for (int i = 0; i < 32; ++i) u[i] = add(v[i], v[i ^ o]);
    v = u;
  }
  return v[0];
}

static double by_sum3(const std::vector<Pair> &p) {
  using spfd::Sum3;
  auto add = [](Sum3 a, Sum3 b) { spfd::sum3_add(a, b.h, b.m, b.l); return a; };
  double tot = 0.0;
  for (int b = 0; b < 8; ++b) {
    std::vector<Sum3> warps(32);
    for (int w = 0; w < 32; ++w) {
      std::vector<Sum3> lanes(32, Sum3{0.f, 0.f, 0.f});
      for (int l = 0; l < 32; ++l)
        for (size_t i = b * 1024 + w * 32 + l; i < p.size(); i += 8192)
          spfd::sum3_add(lanes[l], p[i].h, p[i].l, 0.f);
      warps[w] = warp(lanes, add);
    }
    tot += spfd::sum3_value(warp(warps, add));
  }
  return tot;
}

static double by_f64(const std::vector<Pair> &p) {
  auto add = [](double a, double b) { return a + b; };
  const int blocks = (int)std::min<size_t>(152, (p.size() + 511) / 512);
  auto block = [&](const std::vector<double> &v) {  // lane l adds l, l + 32, ...
    std::vector<double> lanes(32, 0.0);
    for (size_t i = 0; i < v.size(); ++i) lanes[i % 32] += v[i];
    return warp(lanes, add);
  };
  std::vector<double> part;
  for (int b = 0; b < blocks; ++b) {
    std::vector<double> t(512, 0.0);
    for (int k = 0; k < 512; ++k)
      for (size_t i = (size_t)b * 512 + k; i < p.size(); i += (size_t)blocks * 512)
        t[k] += (double)p[i].h + (double)p[i].l;
    part.push_back(block(t));
  }
  return block(part);
}

int main() {
  std::mt19937_64 rng(2010);
  std::normal_distribution<double> nd;
  double s3 = 0.0, s64 = 0.0;
  int n = 0, bad = 0;
  for (int kind = 0; kind < 4; ++kind)
    for (int size : {4, 60, 824, 13648, 89120, 700000})
      for (int rep = 0; rep < (size > 100000 ? 2 : 6); ++rep, ++n) {
        std::vector<Pair> p(size);
        for (Pair &q : p) {
          double v = nd(rng);                          // signs cancel
          if (kind == 1) v = v * v;                    // r.z, p.q: positive
          if (kind == 2) v = std::exp(12.0 * v);       // many magnitudes
          if (kind == 3) v = v * 1e-3 + 1.0;           // nearly equal
          q.h = (float)v;
          q.l = (float)(v - (double)q.h);
        }
        double mag;
        const double want = exact(p, mag), e3 = std::fabs(by_sum3(p) - want) / mag,
                     e64 = std::fabs(by_f64(p) - want) / mag;
        if (!(e3 <= 16.0 * 0x1p-53)) {
          std::printf("kind %d size %d: error %g\n", kind, size, e3);
          ++bad;
        }
        s3 += e3 * e3;
        s64 += e64 * e64;
      }
  if (!bad) std::printf("ok %d %.3g %.3g\n", n, std::sqrt(s3 / n), std::sqrt(s64 / n));
  return bad ? 1 : 0;
}
