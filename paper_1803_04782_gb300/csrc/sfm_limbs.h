// sfm_limbs.h -- the fixed-point form of the product's tables (sfm_product.cu):
// T = L0 / s0 + L1 / (s0 s1), the limbs L0 and L1 integers that FP16 holds.  The
// cells' L1 is any integer up to 65504 and takes two tables, what FP16 holds of
// it and what that leaves.
// Plain functions, compiled for the device and for the host.
//
// The tensor cores add limbs in FP32, so a sum is exact, whatever the order, as
// long as every partial sum of either limb stays below 2^24.  limb_scales looks
// at the limbs themselves: a law that is nearly flat has large second limbs all
// over its window, which no bound by the law's largest entry shows.
#pragma once
#include <math.h>

#include <algorithm>
#include <vector>

#ifdef __CUDACC__
#define SFM_LIMB_HD __host__ __device__ __forceinline__
#else
#define SFM_LIMB_HD inline
#endif

namespace sfm {

// Fixed-point scales, powers of two.
struct ProductScales {
  double s0 = 0.0, s1 = 0.0;
};

// the nearest integer that FP16 holds (|v| < 65520): any up to 2048, every
// second one up to 4096, and so on
SFM_LIMB_HD double limb16(double v) {
  double step = 1.0;
  for (double top = 2048.0; fabs(v) > top; top *= 2.0) step *= 2.0;
  return rint(v / step) * step;
}

// Entry (dx, dy) of plane ch of a crowd (0 presence; the heading axes 1 E-W,
// 2 N-S, 3 NE-SW, 4 NW-SE), v = k d^a being that of plane 0.
SFM_LIMB_HD double crowd_entry(double v, double gamma, int dx, int dy, double d, int ch) {
  const double q = 0.70710678118654752440;  // 1 / sqrt(2)
  if (ch == 1) return v * (gamma * dx / d);
  if (ch == 2) return v * (gamma * dy / d);
  if (ch == 3) return v * (gamma * q * (dx + dy) / d);
  if (ch == 4) return v * (gamma * q * (dy - dx) / d);
  return v;
}

// An offset of the window that stands for `count` of them (by the window's
// symmetries, which map the heading axes onto one another), and its entries: a
// sum holds `first` or not, and at most one of `others`.
struct LimbOffset {
  double count, first;
  double others[4];
};

// The largest scales, s0 largest first, for which every partial sum over a full
// window is below 2^24 (planes are added one after the other, `first`'s before
// the others': a sum holds all of `first`'s or none, or some of them alone).
// `big` bounds the entries; `either`: the others come with both signs.  A limb on
// the edge between two integers may fall either way (the device's pow is not the
// host's): it counts with both signs too.
inline bool limb_scales(const std::vector<LimbOffset>& w, double big, bool either, double most0,
                        double most1, ProductScales* out) {
  if (!(big > 0.0) || !isfinite(big)) return false;
  const double top = 16777215.0, grow = 1.0 + ldexp(1.0, -9);  // FP16's rounding of large limbs
  double n = 0.0, mag = 0.0;
  for (const LimbOffset& o : w) {
    double m = 0.0;
    for (double v : o.others) m = std::max(m, fabs(v));
    n += o.count;
    mag += o.count * (fabs(o.first) + m);
  }
  double s0 = ldexp(1.0, (int)floor(log2(most0 / big)));
  while (mag * s0 * grow + 2.0 * n > top) s0 *= 0.5;
  // what the first limbs leave: largest sums up and down, with `first` and
  // without it, and largest single rest
  double sums[4] = {0.0, 0.0, 0.0, 0.0}, rest_max = 0.0;
  struct Rest {
    double up, down;
  };
  auto rest = [&](double v, bool both) {
    const double x = v * s0, hi = limb16(x), e = x - hi;
    both = both || limb16(hi + 1.000002 * e) != hi;  // half a step off, or as good as
    rest_max = std::max(rest_max, fabs(e));
    return both ? Rest{fabs(e), fabs(e)} : Rest{e, -e};
  };
  for (const LimbOffset& o : w) {
    Rest m{0.0, 0.0};
    for (double v : o.others) {
      const Rest e = rest(v, either);
      m.up = std::max(m.up, e.up);
      m.down = std::max(m.down, e.down);
    }
    const Rest e = rest(o.first, false);
    sums[0] += o.count * std::max(0.0, e.up + m.up);
    sums[1] += o.count * std::max(0.0, e.down + m.down);
    sums[2] += o.count * m.up;
    sums[3] += o.count * m.down;
  }
  const double sum = *std::max_element(sums, sums + 4);
  double s1 = most1;
  while (sum * s1 * grow + 2.0 * n > top || rest_max * s1 > 65504.0) s1 *= 0.5;
  if (!(s0 > 1e-30 && s0 * s1 < 1e30)) return false;  // the limbs' weights are FP32
  out->s0 = s0;
  out->s1 = s1;
  return true;
}

// what the limbs of v leave of it; whole: a second limb of two tables
inline double limb_error(double v, const ProductScales& s, bool whole) {
  const double x = v * s.s0, rest = (x - limb16(x)) * s.s1;
  return fabs((whole ? rint(rest) : limb16(rest)) - rest) / (s.s0 * s.s1);
}

// the window's offsets (x, y), 0 <= y <= x <= r, and how many each stands for
template <class F>
inline void for_octant(int r, F f) {
  for (int x = 1; x <= r; ++x)
    for (int y = 0; y <= x; ++y) f(x, y, y == 0 || y == x ? 4.0 : 8.0);
}

// A crowd's law k d^a (1 + gamma h . u).  false: its range over the window is
// too wide for the two limbs: what a pedestrian adds to a su would be off by
// more than 2^-21 of k d^a there.  The gathers' FP32 sums of a crowd are off by
// that and more (3e-7 to 9e-7), but a lone pedestrian's entry, which they hold
// to 2^-24, is not: the exact sums leave no room for a third limb in FP32.  The
// default law's entries are off by 2.1e-7 at most up to radius 40 (a
// pedestrian without heading 1.1e-7), by 4.2e-7 at 44.
inline bool crowd_limb_scales(int r, double k, double a, double gamma, ProductScales* out) {
  std::vector<LimbOffset> w;
  double big = 0.0;
  for_octant(r, [&](int x, int y, double count) {
    const double d = sqrt((double)(x * x + y * y)), v = k * pow(d, a);
    LimbOffset o{count, v, {}};
    for (int j = 0; j < 4; ++j) o.others[j] = crowd_entry(v, gamma, x, y, d, 1 + j);
    for (double e : {o.first, o.others[0], o.others[1], o.others[2], o.others[3]})
      big = isfinite(e) ? std::max(big, fabs(e)) : INFINITY;
    w.push_back(o);
  });
  if (!limb_scales(w, big, true, 16384.0, 8192.0, out)) return false;
  for (const LimbOffset& o : w) {
    double e = 0.0;
    for (double v : o.others) e = std::max(e, limb_error(v, *out, false));
    if (!(limb_error(o.first, *out, false) + e <= ldexp(fabs(o.first), -21))) return false;
  }
  return true;
}

// Walls (k0 d^a0) and exits (k1 d^a1): a su is one or the other, or neither.
// false: an entry would be further from its law than FP32's rounding puts it
// (2^-24 of itself), which a su that sees a single wall far away would show.
// Two FP16 limbs are 22 bits and up, so the second one has two tables: the
// defaults' entries at radius 40 are off by 5.6e-8 at most (2.1e-7 with one).
inline bool cell_limb_scales(int r, double k0, double a0, double k1, double a1, ProductScales* out) {
  std::vector<LimbOffset> w;
  double big = 0.0;
  for_octant(r, [&](int x, int y, double count) {
    const double d = sqrt((double)(x * x + y * y)), p = pow(d, a0);
    const double v0 = k0 * p, v1 = k1 * (a1 == a0 ? p : pow(d, a1));
    w.push_back(LimbOffset{count, 0.0, {v0, v1, 0.0, 0.0}});
    big = std::max(big, std::max(fabs(v0), fabs(v1)));
    if (!isfinite(v0) || !isfinite(v1)) big = INFINITY;
  });
  if (!limb_scales(w, big, false, 8192.0, 16384.0, out)) return false;
  for (const LimbOffset& o : w)
    for (double v : {o.others[0], o.others[1]})
      if (!(limb_error(v, *out, true) <= ldexp(fabs(v), -24))) return false;
  return true;
}

}  // namespace sfm
