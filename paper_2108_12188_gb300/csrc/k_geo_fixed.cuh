// Geometric factors in fixed point, rebuilt from an element's trilinear coefficients: the values
// k_fixed_factors stores (X = G_ab 2^(sg + c_a + c_b), signed 32-bit halves), for the on-the-fly variant of
// the slice operators.
//
// The rows c_0 = x_s x x_t, c_1 = x_t x x_r, c_2 = x_r x x_s of the cofactor matrix are bilinear in
// the two coordinates along their row's own plane, without the mixed term: with P, M, K the linear functions
//   row 0 (of r)  P = a2 + a4 r, M = a3 + a5 r, K = a6 + a7 r   c_0 = P x M + s P x K + t K x M
//   row 1 (of s)  P = a3 + a6 s, M = a1 + a4 s, K = a5 + a7 s   c_1 = P x M + t P x K + r K x M
//   row 2 (of t)  P = a1 + a5 t, M = a2 + a6 t, K = a4 + a7 t   c_2 = P x M + r P x K + s K x M
// so three crosses per row index of each direction replace those of every point. A point then takes four
// products per component of C, det J = x_t . c_2, F = w_i w_j w_k / det J and G_ab = (c_a . c_b) F, all as
// 64-bit fixed point on the integer and FMA pipes, where GB300 runs 64 or 128 a clock per SM against two FP64
// multiply-adds (k_ax: 45 FP64 instructions per point for the same). A quotient F on the FP64 pipe (a Newton step
// and a correction, 8 instructions) made the kernel slower, N = 9 2.01 -> 2.15 ms: its chain is longer than
// the integer one.
#pragma once

#include <cmath>
#include <cstdint>
#include <cstring>

namespace sem {

#ifdef __CUDA_ARCH__
#define SEM_HD __host__ __device__ __forceinline__
#else
#define SEM_HD __host__ __device__ inline
#endif

// A 64-bit value as signed halves, v = h 2^32 + l (the layout of the stored factors).
struct __align__(8) Fx {
  int l, h;
};
SEM_HD Fx fx_split(long long v) {
  return {static_cast<int>(static_cast<uint32_t>(v)),
          static_cast<int>(v >> 32) + static_cast<int>(static_cast<uint32_t>(v) >> 31)};
}
SEM_HD long long fx_shl(long long v, int s) { return static_cast<long long>(static_cast<unsigned long long>(v) << s); }
// Sum of products without the low by low terms, in units of 2^64 (h) and 2^32 (m).
struct FxSum {
  long long h = 0, m = 0;
  SEM_HD void add(const Fx& a, const Fx& b) {
    h += static_cast<long long>(a.h) * b.h;
    m += static_cast<long long>(a.h) * b.l;
    m += static_cast<long long>(a.l) * b.h;
  }
  SEM_HD void sub(const Fx& a, const Fx& b) {
    h -= static_cast<long long>(a.h) * b.h;
    m -= static_cast<long long>(a.h) * b.l;
    m -= static_cast<long long>(a.l) * b.h;
  }
  // sum / 2^64. one: 1, in a register the compiler does not see through: a sign extension and a 64-bit
  // addition as one wide multiply-add.
  SEM_HD long long get(int one) const { return h + static_cast<long long>(static_cast<int>(m >> 32)) * one; }
  SEM_HD long long get_shl(int s) const { return fx_shl(h, s) + (m >> (32 - s)); }  // sum / 2^(64 - s)
};
SEM_HD long long fx_fma(const Fx& a, const Fx& b, long long c, int one) {
  FxSum s;
  s.h = c;
  s.add(a, b);
  return s.get(one);
}

// One element: its coefficients a1..a7 and the scales of its factors.
struct __align__(16) GeoElement {
  long long a[7][3];  // in units of 2^-qa
  int sg;             // X = G_ab 2^(sg + c_a + c_b); kGeoNone: not in fixed point
  int s, s2;          // shifts of the rows 0, 1 and of row 2 from units of 2^(64 - 2 qa) to 2^-q and 2^-q2
  int down;           // q2 - q: c_d in units of 2^-q in the products c_a . c_b, c_2 in units of 2^-q2 for det J
  int lz;             // F in the units of a point whose det J has this many leading zeros: the most of the element
  int up;             // (c_a . c_b / 2^64) F / 2^(64 - up) uses 62 bits; 8 bits up: its right shift to X less the row scales
};
constexpr int kGeoNone = 1 << 20;
// Bits of det J an element has to have in fixed point, and the most that `up` and the rows' shifts may be; beyond, the factors
// would come out less exact than FP64 has them, and a mesh with such an element keeps k_ax. Relative rms error of the
// factors against 80 bits, here and in FP64, over 200 elements with vertices moved by 15%, N = 9: 3.9e-17 and 2.5e-16 (up 9),
// ten times as long along r, s or t 3.9e-17 or less and 2.5e-16, along t 30 times 7.5e-17 and 2.3e-16 (shift 14) and 100 times 1.4e-16 and
// 2.2e-16 (shift 15; 300 times, 17, 3.7e-16), sheared by 5 4.7e-17 and 2.9e-16; moved by 30% 1.6e-16 and 2.4e-16 (up 12), N = 11 2.2e-16
// and 2.4e-16 (up 12; with 14 3.2e-16).
constexpr int kGeoBits = 52, kGeoUp = 12, kGeoShift = 15;

// Node values: coordinates in units of 2^-62, weights times 2^c (c: fixed_row_scale) below 2^62.
template <int NP>
struct GeoNodes {
  Fx x[NP], w[NP];
};
// Units of 2^-(62 + geo_weight_scale) for the weights times 2^c.
inline int geo_weight_scale(const double* w, const int* c, int np) {
  double top = 0.0;
  for (int i = 0; i < np; ++i) top = std::fmax(top, std::ldexp(w[i], c[i]));
  return -std::ilogb(top) - 1;
}

// v 2^q truncated, |v 2^q| < 2^62.
SEM_HD long long geo_fixed(double v, int q) {
  uint64_t b;
  memcpy(&b, &v, 8);
  const int e = static_cast<int>((b >> 52) & 0x7ffu), s = 1075 - e - q;  // significand / 2^s
  if (e == 0) return 0;
  uint64_t f = (b & 0xfffffffffffffull) | 0x10000000000000ull;
  f = s >= 0 ? (s < 64 ? f >> s : 0) : f << (-s < 63 ? -s : 63);
  return (b >> 63) ? -static_cast<long long>(f) : static_cast<long long>(f);
}

// The scales from the exponents (frexp) of these numbers of an element: coef: for each component the sum of
// |a_1| .. |a_7|, the largest of the three; row: largest |c_d| and 4 times its slopes; det: smallest det J, less 2^-40 of it; top:
// largest G_ab 2^(c_a + c_b); all: largest G_ab 2^(c_0 + c_1 + c_2); sw: geo_weight_scale.
// |c| 2^q < 2^62 bounds the products: |c_a . c_b| / 2^64 < 2^60, and the mixed terms of a sum of three stay below
// 2^63. F < 2^62, and X <= 2^59.
SEM_HD int geo_scale(GeoElement& g, int coef, const int (&row)[3], int det, int top, int all, int sw) {
  int most = row[0] > row[1] ? row[0] : row[1];
  most = most > row[2] ? most : row[2];
  const int qa = 61 - coef, q = 62 - most, q2 = 62 - row[2];
  g.s = q - (2 * qa - 64);
  g.s2 = q2 - (2 * qa - 64);
  g.down = q2 - q;
  const int d = det - 1 + qa + q2 - 64;  // det J in fixed point is at least 2^d
  g.lz = 63 - d;
  const int unit = 2 * q + 3 * sw + 61 - qa - q2 - g.lz;  // c_a . c_b F / 2^128 = G 2^(c_0 + c_1 + c_2 + unit)
  const int up = 62 - (all + unit);
  g.sg = 59 - top < unit + up - 2 ? 59 - top : unit + up - 2;
  g.up = up | (unit + up - g.sg) << 8;
  bool ok = d >= kGeoBits && d <= 61 && g.s >= 0 && g.s <= kGeoShift && g.s2 <= kGeoShift && up >= 0 && up <= kGeoUp &&
            unit + up - g.sg <= 40;
  for (int v : {coef, row[0], row[1], row[2], det, top, all}) ok = ok && v > -200 && v < 200;
  if (!ok) g.sg = kGeoNone;
  return qa;
}

// Row tables, one entry per component: alpha + y beta + z gamma (y, z the coordinates of P x K and K x M above), the
// slopes times four (a coordinate is in units of 2^-62). Row 0 has x_t = a + s b too.
struct GeoEntry {
  long long a;
  Fx b, g;
};
struct GeoEntryT {
  long long a;
  Fx b;
};
// Component c of row d at node coordinate v.
SEM_HD GeoEntry geo_entry(const GeoElement& e, int d, int c, const Fx& v, int one, GeoEntryT* xt) {
  // rows of a (a1 is 0) of P, M, K: value and slope
  const int p0 = d == 0 ? 1 : d == 1 ? 2 : 0, p1 = d == 0 ? 3 : d == 1 ? 5 : 4;
  const int m0 = d == 0 ? 2 : d == 1 ? 0 : 1, m1 = d == 0 ? 4 : d == 1 ? 3 : 5;
  const int k0 = d == 0 ? 5 : d == 1 ? 4 : 3;
  const int y = c == 2 ? 0 : c + 1, z = c == 0 ? 2 : c - 1;
  auto at = [&](int r0, int r1, int q) { return fx_fma(fx_split(fx_shl(e.a[r1][q], 2)), v, e.a[r0][q], one); };
  const Fx py = fx_split(at(p0, p1, y)), pz = fx_split(at(p0, p1, z)), my = fx_split(at(m0, m1, y)),
           mz = fx_split(at(m0, m1, z)), ky = fx_split(at(k0, 6, y)), kz = fx_split(at(k0, 6, z));
  const int s = d == 2 ? e.s2 : e.s;
  auto cross = [&](const Fx& ay, const Fx& az, const Fx& by, const Fx& bz, int sh) {
    FxSum t;
    t.add(ay, bz);
    t.sub(az, by);
    // (of two short vectors the difference is small and sh large: the low by low products count)
    t.m += (static_cast<long long>(ay.l) * bz.l - static_cast<long long>(az.l) * by.l) >> 32;
    return t.get_shl(sh);
  };
  if (d == 0) *xt = {at(m0, m1, c), fx_split(fx_shl(at(k0, 6, c), 2))};
  return {cross(py, pz, my, mz, s), fx_split(cross(py, pz, ky, kz, s + 2)), fx_split(cross(ky, kz, my, mz, s + 2))};
}

// 2^124 / v for v in [2^62, 2^63): a 24-bit start, one step of third order. Error below 4 units.
SEM_HD long long geo_recip(unsigned long long v) {
  const uint32_t vh = static_cast<uint32_t>(v >> 32), vl = static_cast<uint32_t>(v);
#ifdef __CUDA_ARCH__
  const uint32_t s = __float2uint_rz(__fdividef(2305843009213693952.0f, __uint2float_rn(vh)));
#else
  const uint32_t s = static_cast<uint32_t>(2305843009213693952.0f / static_cast<float>(vh));
#endif
  const uint32_t y0 = s < 0x7fffffffu ? s : 0x7fffffffu;
  const unsigned long long p = static_cast<unsigned long long>(vh) * y0 +
                               ((static_cast<unsigned long long>(vl) * y0) >> 32);  // v y0 2^-32 ~ 2^61
  const long long r = static_cast<long long>(2305843009213693952ull - p);             // 1 - v y0 in units of 2^-61
  const int rs = static_cast<int>(r >> 8);
  const long long r2 = r + ((static_cast<long long>(rs) * rs) >> 45);
  const long long hi = static_cast<long long>(static_cast<int>(y0)) * static_cast<int>(r2 >> 8);
  const uint32_t lo = static_cast<uint32_t>((static_cast<uint64_t>(y0) * static_cast<uint32_t>(r2 & 255)) >> 30);
  return (static_cast<long long>(y0) << 31) + (hi >> 22) + lo;
}

// The rows of one k-column (i, j) of an element.
struct GeoColumn {
  long long a0[3], a1[3];
  Fx xt[3], r, s, w;
  int one;

  // e0: [3] of node i, e1: of node j; et: of node i
  SEM_HD void init(const GeoEntry* e0, const GeoEntry* e1, const GeoEntryT* et, const Fx& xi, const Fx& xj, const Fx& wi,
                   const Fx& wj, int one_) {
    r = xi;
    s = xj;
    one = one_;
    FxSum p;
    p.add(wi, wj);
    w = fx_split(p.get_shl(2));
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      a0[c] = fx_fma(e0[c].b, s, e0[c].a, one);
      a1[c] = fx_fma(e1[c].g, r, e1[c].a, one);
      xt[c] = fx_split(fx_fma(et[c].b, s, et[c].a, one));
    }
  }
  // The six factors at node k (e2 of it, coordinate t, weight wk): out(m, value) in the order 00, 01, 02, 11,
  // 12, 22, the value times 2^((up >> 8) + c_0 + c_1 + c_2 - c_a - c_b).
  template <typename F>
  SEM_HD void point(const GeoEntry* e0, const GeoEntry* e1, const GeoEntry* e2, const Fx& t, const Fx& wk, int down,
                    int lzmax, int up, F&& out) const {
    Fx c0[3], c1[3], c2[3];
    FxSum d;
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      FxSum q;
      q.h = e2[c].a;
      q.add(e2[c].b, r);
      q.add(e2[c].g, s);
      const long long v = q.get(one);
      d.add(xt[c], fx_split(v));
      c2[c] = fx_split(v >> down);
    }
    const long long det = d.get(one);
#ifdef __CUDA_ARCH__
    const int lz = __clzll(det);
#else
    const int lz = det > 0 ? __builtin_clzll(static_cast<unsigned long long>(det)) : det < 0 ? 0 : 64;
#endif
    FxSum fw;
    fw.add(fx_split(fx_fma(w, wk, 0, one)), fx_split(geo_recip(static_cast<unsigned long long>(det) << ((lz - 1) & 63))));
    const int fs = lzmax - lz;
    const Fx f = fx_split(fw.get_shl(4) >> (fs > 0 ? fs & 63 : 0));
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      c0[c] = fx_split(fx_fma(e0[c].g, t, a0[c], one));
      c1[c] = fx_split(fx_fma(e1[c].b, t, a1[c], one));
    }
    auto mixed = [&](int m, const Fx(&p)[3], const Fx(&q)[3]) {
      FxSum n;
#pragma unroll
      for (int c = 0; c < 3; ++c) n.add(p[c], q[c]);
      FxSum x;
      x.add(fx_split(n.get(one)), f);
      out(m, x.get_shl(up));
    };
    auto square = [&](int m, const Fx(&p)[3]) {
      FxSum n;
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        n.h += static_cast<long long>(p[c].h) * p[c].h;
        n.m += static_cast<long long>(p[c].h) * p[c].l;
      }
      FxSum x;
      x.add(fx_split(n.h + (n.m >> 31)), f);
      out(m, x.get_shl(up));
    };
    square(5, c2);
    mixed(2, c0, c2);
    mixed(4, c1, c2);
    square(0, c0);
    mixed(1, c0, c1);
    square(3, c1);
  }
};

}  // namespace sem
