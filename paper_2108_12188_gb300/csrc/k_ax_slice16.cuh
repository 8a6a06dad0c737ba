// The operator of k_ax_slice.cuh at 9 to 12 points per direction: the same digits, fixed point and
// error analysis on a box of 16 x 16 points per k-plane, one element per block and one k-plane per warp.
// A contraction over 16 points is one k-step of mma.sync per pair of digits, so a group C_g takes
// g + 1 of them; the groups from magic_groups on exceed the 2^22 that fit on top of kMagic and are split
// in FP32.
//
// 17.6, 16.2 and 16.0M points, FP64 (k_ax) against this kernel: N = 9 2.03 and 1.47 ms, N = 10 1.79 and 1.03, N = 11 2.06 and
// 0.81; 180 elements at N = 11 68 and 30 us. It is bound as k_ax_slice is, and works on 256 points of
// every plane where the element has (N + 1)^2 (N = 9 100), with 9 to 12 warps per SM.
#pragma once

#include "k_ax_slice.cuh"

namespace sem {
namespace {

template <int NP>
struct Slice16Shape {
  static constexpr int kThreads = 32 * NP;
  static constexpr int kRowBytes = 272;                           // 16 rows of 8 digits, 16 bytes of padding
  static constexpr int kHalf = 16 * kRowBytes;                    // i half b of a digit: 16 k-planes
  static constexpr int kDigit = 2 * kHalf;
  static constexpr int kPlaneX = 136;                             // exchange: [2][NP][136] 64-bit
  static constexpr unsigned kElemBytes = 48u * NP * NP * NP;
  static constexpr size_t kOffD = (kElemBytes + 127) / 128 * 128; // digits [kSlices][2][16][17][8] FP16
  static constexpr size_t kOffX = kOffD + kSlices * kDigit;
  static constexpr size_t kOffT = kOffX + 2 * NP * kPlaneX * 8;   // fragments [2][kSlices][32] 16 bytes
  static constexpr size_t kOffM = kOffT + 2 * kSlices * 32 * 16;  // maxima [2][NP]
  static constexpr size_t kOffBar = kOffM + (2 * NP * 4 + 7) / 8 * 8;
  static constexpr size_t kOffTab = (kOffBar + 8 + 15) / 16 * 16;  // on the fly: row tables
  static constexpr int kFew = kThreads / 4;  // every thread holds points, see kNear
  static_assert(kSlices * kDigit >= 24 * NP * NP * NP, "the digits' buffer holds the arrays of elements_fp64");
  using Geometry = OtfGeometry<NP, 1, kThreads>;
  static constexpr size_t bytes(bool otf) { return otf ? kOffTab + sizeof(typename Geometry::Tables) : kOffBar + 8; }
};

// As combine() with fewer groups on top of kMagic: C_4 = 1024 t + r with t joining C_3, and for three groups
// C_3 = 1024 t' + r' the same way, |r| and |r'| <= 512.
template <int GROUPS>
__device__ __forceinline__ long long combine16(float f0, float f1, float f2, float f3, float f4, float f5, float f6) {
  constexpr unsigned long long kBase =
      0ull - static_cast<unsigned long long>(kMagicBits) * (1ull + (1ull << 13) + (1ull << 23)) -
      static_cast<unsigned long long>(kMagicBits) * (GROUPS == 4 ? 1ull << 13 : 1ull << 23) -
      (static_cast<unsigned long long>(static_cast<uint32_t>((kMagicBits << 1) + (kMagicBits << 11))) << 32);
  const float t = fmaf(f4, 1.0f / 1024.0f, kMagic), tq = __fsub_rn(t, kMagic);
  const float low = fmaf(fmaf(tq, -1024.0f, f4), 8.0f, fmaf(fmaf(f6, 1.0f / 1024.0f, f5), 1.0f / 128.0f, kMagic));
  unsigned long long v = madw<1>(__float_as_uint(low), kBase);
  if constexpr (GROUPS == 4) {
    v = madw<8192>(__float_as_uint(f3) + __float_as_uint(t), v);
    v = madw<8388608>(__float_as_uint(f2), v);
  } else {
    const float t3 = fmaf(f3, 1.0f / 1024.0f, kMagic), r3 = fmaf(__fsub_rn(t3, kMagic), -1024.0f, f3);
    v = madw<8192>(__float_as_uint(__fadd_rn(__fadd_rn(r3, tq), kMagic)), v);
    v = madw<8388608>(__float_as_uint(f2) + __float_as_uint(t3), v);
  }
  const uint32_t hi = static_cast<uint32_t>(v >> 32) + (__float_as_uint(f1) << 1) + (__float_as_uint(f0) << 11);
  return static_cast<long long>((static_cast<unsigned long long>(hi) << 32) | static_cast<uint32_t>(v));
}

// Products of digits s and t (of the table), summed by group: c[g] over s + t = g. Lines: the table is the A operand (outputs in the rows), b[s] the lines' B fragment. Rows: a[s]
// holds rows of points and the table's half h is the B operand (outputs 8 h .. 8 h + 7 in the columns).
template <int GROUPS>
__device__ __forceinline__ void groups_lines(const float (&m)[4], const uint4* tab, const uint32_t (&b)[kSlices][2],
                                             float (&c)[7][4]) {
#pragma unroll
  for (int t = 0; t < kSlices; ++t) {
    const uint4 a = tab[32 * t];
#pragma unroll
    for (int s = 0; s < kSlices; ++s) {
      const int g = s + t;
      if (g > 6) continue;
      if (t == 0 || g == 6 && t == 1) {  // the group's first product
        if (g < GROUPS)
          mma_start(c[g], a, b[s][0], b[s][1], m);
        else
          mma_zero(c[g], a, b[s][0], b[s][1]);
      } else {
        mma_add(c[g], a, b[s][0], b[s][1]);
      }
    }
  }
}
template <int GROUPS>
__device__ __forceinline__ void groups_rows(const float (&m)[4], const uint4* tab, int h, const uint4 (&a)[kSlices],
                                            float (&c)[7][4]) {
#pragma unroll
  for (int t = 0; t < kSlices; ++t) {
    const uint4 d = tab[32 * t];
    const uint32_t b0 = h ? d.y : d.x, b1 = h ? d.w : d.z;
#pragma unroll
    for (int s = 0; s < kSlices; ++s) {
      const int g = s + t;
      if (g > 6) continue;
      if (t == 0 || g == 6 && t == 1) {
        if (g < GROUPS)
          mma_start(c[g], a[s], b0, b1, m);
        else
          mma_zero(c[g], a[s], b0, b1);
      } else {
        mma_add(c[g], a[s], b0, b1);
      }
    }
  }
}
// Value x of the lane's row (0: lane / 4, 1: lane / 4 + 8).
template <int GROUPS>
__device__ __forceinline__ long long value16(const float (&c)[7][4], int row, int x) {
  const int q = 2 * row + x;
  return combine16<GROUPS>(c[0][q], c[1][q], c[2][q], c[3][q], c[4][q], c[5][q], c[6][q]);
}

// Warp k holds plane k; the lane's points are j = lane / 4 + 8 a, i = 2 (lane % 4) + 8 b + x (a, b, x in
// {0, 1}), values [a][b][x]. Phases as in k_ax_slice; in the k contractions warp k takes the lines of plane
// j = k.
template <int NP, bool CG, bool OTF>
__global__ void __launch_bounds__(Slice16Shape<NP>::kThreads, 1)
    k_ax_slice16(const __grid_constant__ GllParam<NP, double> tab, const __grid_constant__ SliceTab<NP> sl,
                 const __grid_constant__ GeoNodes<NP> nodes, int64_t E, const double* __restrict__ u,
                 double* __restrict__ w, const int2* __restrict__ G, const int* __restrict__ gexp,
                 const GeoElement* __restrict__ geo, const double* __restrict__ r, const double* __restrict__ minv,
                 double* __restrict__ x, double* __restrict__ p, CgScalars* __restrict__ st,
                 double* __restrict__ partials, int* __restrict__ err) {
  using S = Slice16Shape<NP>;
  constexpr int NP2 = NP * NP, P = NP2 * NP, kMg = magic_groups(NP);
  extern __shared__ __align__(128) unsigned char smem[];
  int2* sG = reinterpret_cast<int2*>(smem);
  double* abc = reinterpret_cast<double*>(smem + S::kOffD);  // elements_fp64, in place of the digits
  long long* sX = reinterpret_cast<long long*>(smem + S::kOffX);
  uint4* sT = reinterpret_cast<uint4*>(smem + S::kOffT);
  unsigned* sMax = reinterpret_cast<unsigned*>(smem + S::kOffM);
  uint64_t* bar = reinterpret_cast<uint64_t*>(smem + S::kOffBar);
  __shared__ double sRed[32];
  __shared__ __align__(16) float sStart[4];

  double beta = 0.0, alpha = 0.0;
  if constexpr (CG) {
    if (st->done) return;  // uniform over the grid: set by an earlier launch
    beta = st->beta;
    alpha = st->alpha;
  }
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int g = lane >> 2, q2 = 2 * (lane & 3);
  auto load_factors = [&](int64_t e) {  // one thread
    fence_proxy_async();
    mbar_expect_tx(bar, S::kElemBytes);
    tma_load_1d(sG, G + e * 6 * P, S::kElemBytes, bar);
  };
  typename S::Geometry::Tables* tables = reinterpret_cast<typename S::Geometry::Tables*>(smem + S::kOffTab);
  if constexpr (OTF) {
    S::Geometry::nodes(tables, nodes);
  } else if (threadIdx.x == 0) {
    mbar_init(bar, 1);
    load_factors(blockIdx.x);
  }
  if (threadIdx.x < 4) sStart[threadIdx.x] = kMagic;
  for (unsigned q = threadIdx.x; q < kSlices * S::kDigit / 4; q += S::kThreads)
    reinterpret_cast<uint32_t*>(smem + S::kOffD)[q] = 0u;
  if (warp < 2)
#pragma unroll
    for (int t = 0; t < kSlices; ++t) {
      const auto& d = sl.d[warp][t];
      sT[(warp * kSlices + t) * 32 + lane] =
          make_uint4(d[g][lane & 3], d[g + 8][lane & 3], d[g][4 + (lane & 3)], d[g + 8][4 + (lane & 3)]);
    }
  const uint4* tF = sT + lane;
  const uint4* tT = sT + kSlices * 32 + lane;
  const uint32_t sD32 = smem_u32(smem + S::kOffD);
  const int mi = lane >> 3, row = lane & 7;
  // k-lines of plane j = warp and j-lines of plane k = warp: rows 0-7, 8-15 of digit s, then of digit s + 1
  const uint32_t ldK = sD32 + (mi >> 1) * S::kDigit + (row + 8 * (mi & 1)) * S::kRowBytes + warp * 16;
  const uint32_t ldJ = sD32 + (mi >> 1) * S::kDigit + warp * S::kRowBytes + (row + 8 * (mi & 1)) * 16;
  // i-rows: rows j 0-7, 8-15 of i half 0, then of half 1
  const uint32_t ldI = sD32 + (mi >> 1) * S::kHalf + warp * S::kRowBytes + (row + 8 * (mi & 1)) * 16;
  auto put_digits = [&](int a, int b, const uint32_t (&d)[kSlices]) {
#pragma unroll
    for (int s = 0; s < kSlices; ++s)
      *reinterpret_cast<uint32_t*>(smem + S::kOffD + s * S::kDigit + b * S::kHalf + warp * S::kRowBytes + (g + 8 * a) * 16 +
                                   (lane & 3) * 4) = d[s];
  };
  auto at_x = [&](int b, int k, int j) { return sX + (b * NP + k) * S::kPlaneX + j * 8 + q2; };
  double dot = 0.0;
  unsigned parity = 0;
  __syncthreads();
  float m4[4];
  lds_quad(m4, smem_u32(sStart));

  // k-lines of plane j = warp through table `tab16`, to the exchange buffer; the magnitudes' bits
  auto k_lines = [&](const uint4* tab16) {
    unsigned m = 0;
#pragma unroll
    for (int b = 0; b < 2; ++b) {
      uint32_t f[kSlices][2];
#pragma unroll
      for (int s = 0; s < kSlices; s += 2)
        ldsm4t(f[s][0], f[s][1], f[s + 1][0], f[s + 1][1], ldK + s * S::kDigit + b * S::kHalf);
      float c[7][4];
      groups_lines<kMg>(m4, tab16, f, c);
#pragma unroll
      for (int a = 0; a < 2; ++a) {
        const long long v0 = value16<kMg>(c, a, 0), v1 = value16<kMg>(c, a, 1);
        if (g + 8 * a < NP) *reinterpret_cast<longlong2*>(at_x(b, g + 8 * a, warp)) = make_longlong2(v0, v1);
        m |= magnitude(v0) | magnitude(v1);
      }
    }
    return m;
  };

  for (int64_t e = blockIdx.x; e < E; e += gridDim.x) {
    const int64_t base = e * P + warp * NP2;
    const bool more = e + gridDim.x < E;
    auto in = [&](int a, int b, int y) { return g + 8 * a < NP && q2 + 8 * b + y < NP; };
    auto off = [&](int a, int b) { return (g + 8 * a) * NP + q2 + 8 * b; };
    // the lane's pair (a, b); 16-byte aligned where NP is even
    auto load2 = [&](const double* __restrict__ src, int a, int b, double (&o)[2]) {
      const double* s = src + base + off(a, b);
      o[0] = o[1] = 0.0;
      if constexpr (NP % 2 == 0) {
        if (in(a, b, 0)) {
          const double2 v = *reinterpret_cast<const double2*>(s);
          o[0] = v.x;
          o[1] = v.y;
        }
      } else {
        if (in(a, b, 0)) o[0] = s[0];
        if (in(a, b, 1)) o[1] = s[1];
      }
    };
    auto store2 = [&](double* __restrict__ dst, int a, int b, const double (&o)[2]) {
      double* s = dst + base + off(a, b);
      if constexpr (NP % 2 == 0) {
        if (in(a, b, 0)) *reinterpret_cast<double2*>(s) = make_double2(o[0], o[1]);
      } else {
        if (in(a, b, 0)) s[0] = o[0];
        if (in(a, b, 1)) s[1] = o[1];
      }
    };
    // phase 0
    double v[2][2][2];
#pragma unroll
    for (int a = 0; a < 2; ++a)
#pragma unroll
      for (int b = 0; b < 2; ++b) {
        if constexpr (CG) {
          double rv[2], pv[2], xv[2], mv[2];
          load2(r, a, b, rv);
          load2(p, a, b, pv);
          load2(x, a, b, xv);
          if (minv) load2(minv, a, b, mv);
#pragma unroll
          for (int y = 0; y < 2; ++y) {
            v[a][b][y] = fma(beta, pv[y], minv ? mv[y] * rv[y] : rv[y]);
            xv[y] = fma(alpha, pv[y], xv[y]);
          }
          store2(p, a, b, v[a][b]);
          store2(x, a, b, xv);
        } else {
          load2(u, a, b, v[a][b]);
        }
      }
    if constexpr (OTF) S::Geometry::rows(tables, geo, e, 1);
    const int sg = __ldg(OTF ? &geo[e].sg : gexp + e);
    unsigned mh = 0;
    bool nonzero = false;
#pragma unroll
    for (int a = 0; a < 2; ++a)
#pragma unroll
      for (int b = 0; b < 2; ++b)
#pragma unroll
        for (int y = 0; y < 2; ++y) {
          mh = max(mh, static_cast<unsigned>(__double2hiint(v[a][b][y])) & 0x7fffffffu);
          nonzero |= v[a][b][y] != 0.0;
        }
    mh = near_word(mh, __reduce_max_sync(0xffffffffu, mh), 0xffffffffu);
    if (lane == 0) sMax[warp] = mh;
    __syncthreads();
    const unsigned all = lane < NP ? sMax[lane] : 0u;
    int emax = static_cast<int>(__reduce_max_sync(0xffffffffu, all) >> 20);
    const bool near = static_cast<int>(all >> 20) + kNearWarp >= emax;
    bool slow = emax == 2047 || abs(1080 - emax + sg) > 700 || __reduce_add_sync(0xffffffffu, near ? all & 63u : 0u) < S::kFew;
    if (emax < 64) {  // zero, or too small for fixed point
      slow = __syncthreads_or(nonzero || sg < kSgFinite);
      emax = 1080;
    }
    if (threadIdx.x == 0 && more) {  // the next element's vectors into L2
      if constexpr (OTF) l2_prefetch(geo + e + gridDim.x, sizeof(GeoElement));
      if constexpr (P % 2 == 0) {
        const int64_t at = (e + gridDim.x) * P;
        if constexpr (CG) {
          l2_prefetch(r + at, 8u * P);
          l2_prefetch(p + at, 8u * P);
          l2_prefetch(x + at, 8u * P);
          if (minv) l2_prefetch(minv + at, 8u * P);
        } else {
          l2_prefetch(u + at, 8u * P);
        }
      }
    }
#pragma unroll
    for (int a = 0; a < 2; ++a)
#pragma unroll
      for (int b = 0; b < 2; ++b) {
        uint32_t d[kSlices];
        digit_pairs(to_fixed(v[a][b][0], emax), to_fixed(v[a][b][1], emax), d);
        put_digits(a, b, d);
      }
    if constexpr (OTF) S::Geometry::columns(tables, geo, e, 1, sG);
    __syncthreads();

    // phase 1
    long long vr[2][2][2], vs[2][2][2];
    if (!slow) {
      unsigned m = k_lines(tF);
      {
        uint4 f[kSlices];
#pragma unroll
        for (int s = 0; s < kSlices; ++s) {
          uint32_t t[4];
          ldsm4(t, ldI + s * S::kDigit);
          f[s] = make_uint4(t[0], t[1], t[2], t[3]);
        }
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          float c[7][4];
          groups_rows<kMg>(m4, tF, h, f, c);
#pragma unroll
          for (int a = 0; a < 2; ++a)
#pragma unroll
            for (int y = 0; y < 2; ++y) vr[a][h][y] = value16<kMg>(c, a, y);
        }
      }
#pragma unroll
      for (int b = 0; b < 2; ++b) {
        uint32_t f[kSlices][2];
#pragma unroll
        for (int s = 0; s < kSlices; s += 2)
          ldsm4t(f[s][0], f[s][1], f[s + 1][0], f[s + 1][1], ldJ + s * S::kDigit + b * S::kHalf);
        float c[7][4];
        groups_lines<kMg>(m4, tF, f, c);
#pragma unroll
        for (int a = 0; a < 2; ++a)
#pragma unroll
          for (int y = 0; y < 2; ++y) vs[a][b][y] = value16<kMg>(c, a, y);
      }
#pragma unroll
      for (int a = 0; a < 2; ++a)
#pragma unroll
        for (int b = 0; b < 2; ++b)
#pragma unroll
          for (int y = 0; y < 2; ++y) m |= magnitude(vr[a][b][y]) | magnitude(vs[a][b][y]);
      m = __reduce_or_sync(0xffffffffu, m);
      if (lane == 0) sMax[NP + warp] = m;
    } else {  // u over the digits
#pragma unroll
      for (int a = 0; a < 2; ++a)
#pragma unroll
        for (int b = 0; b < 2; ++b)
#pragma unroll
          for (int y = 0; y < 2; ++y)
            if (in(a, b, y)) abc[warp * NP2 + off(a, b) + y] = v[a][b][y];
    }
    bool ok = true;
    if constexpr (!OTF) ok = mbar_wait_bounded(bar, parity);  // this element's factors
    parity ^= 1u;
    if (__syncthreads_or(!ok)) {  // the factor copy did not arrive: report and leave together
      if (threadIdx.x == 0) {
        mbar_wait_bounded(bar, parity ^ 1u);  // give the copy in flight one more bounded wait
        atomicExch(err, static_cast<int>(SEM_ERR_TIMEOUT));
        if constexpr (CG) {
          st->status = SEM_ERR_TIMEOUT;
          st->done = 1;
        }
      }
      return;
    }

    double wv[2][2][2];
    if (!slow) {
      // phase 2: geometry on V 2^lv, |V| 2^lv < 2^61
      unsigned m = 0;
#pragma unroll
      for (int q = 0; q < NP; ++q) m |= sMax[NP + q];
      const int lv = __clz(m) - 3;
#pragma unroll
      for (int a = 0; a < 2; ++a)
#pragma unroll
        for (int b = 0; b < 2; ++b) {
          // (the fixed-point factors beyond the element's points: none, their V is 0)
          const int j = g + 8 * a < NP ? g + 8 * a : 0;
          const longlong2 ut = *reinterpret_cast<const longlong2*>(at_x(b, warp, j));
          long long vt[2] = {ut.x, ut.y};
          int2 gm[6][2];
#pragma unroll
          for (int q = 0; q < 6; ++q) {
            const int2* src = sG + q * P + warp * NP2 + off(a, b);
            if constexpr (NP % 2 == 0) {
              const int4 t = in(a, b, 0) ? *reinterpret_cast<const int4*>(src) : make_int4(0, 0, 0, 0);
              gm[q][0] = make_int2(t.x, t.y);
              gm[q][1] = make_int2(t.z, t.w);
            } else {
#pragma unroll
              for (int y = 0; y < 2; ++y) gm[q][y] = in(a, b, y) ? src[y] : make_int2(0, 0);
            }
          }
#pragma unroll
          for (int y = 0; y < 2; ++y) {
            const long long ar = vr[a][b][y] << lv, as = vs[a][b][y] << lv, at = vt[y] << lv;
            const int rl = low_half(ar), rh = high_half(ar), jl = low_half(as), jh = high_half(as), tl = low_half(at),
                      th = high_half(at);
            auto row3 = [&](const int2& f0, const int2& f1, const int2& f2) {
              Acc2 s{0, 0};
              s.add(f0.x, f0.y, rl, rh);
              s.add(f1.x, f1.y, jl, jh);
              s.add(f2.x, f2.y, tl, th);
              return s.value();
            };
            vr[a][b][y] = row3(gm[0][y], gm[1][y], gm[2][y]);
            vs[a][b][y] = row3(gm[1][y], gm[3][y], gm[4][y]);
            vt[y] = row3(gm[2][y], gm[4][y], gm[5][y]);
          }
          uint32_t d[kSlices];
          digit_pairs(vt[0], vt[1], d);
          put_digits(a, b, d);
        }
      // phase 3
      long long sum[2][2][2];
      {
        uint4 f[kSlices];
        uint32_t d[2][2][kSlices];
#pragma unroll
        for (int a = 0; a < 2; ++a)
#pragma unroll
          for (int b = 0; b < 2; ++b) digit_pairs(vr[a][b][0], vr[a][b][1], d[a][b]);
#pragma unroll
        for (int s = 0; s < kSlices; ++s) f[s] = make_uint4(d[0][0][s], d[1][0][s], d[0][1][s], d[1][1][s]);
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          float c[7][4];
          groups_rows<kMg>(m4, tT, h, f, c);
#pragma unroll
          for (int a = 0; a < 2; ++a)
#pragma unroll
            for (int y = 0; y < 2; ++y) sum[a][h][y] = value16<kMg>(c, a, y);
        }
      }
#pragma unroll
      for (int b = 0; b < 2; ++b) {
        uint32_t f[kSlices][2], d[kSlices];
#pragma unroll
        for (int a = 0; a < 2; ++a) {
          digit_pairs(vs[a][b][0], vs[a][b][1], d);
#pragma unroll
          for (int s = 0; s < kSlices; ++s) f[s][a] = transpose8x8(d[s]);
        }
        float c[7][4];
        groups_lines<kMg>(m4, tT, f, c);
#pragma unroll
        for (int a = 0; a < 2; ++a)
#pragma unroll
          for (int y = 0; y < 2; ++y) sum[a][b][y] += value16<kMg>(c, a, y);
      }
      __syncthreads();  // the digits of vt; the factors are consumed
      if (!OTF && threadIdx.x == 0 && more) load_factors(e + gridDim.x);
      k_lines(tT);
      __syncthreads();
      // w = sum 2^-sc: u 2^(1080 - emax), D 2^e / 2^57 twice, V 2^lv, G 2^sg / 2^64
      const int scale = -(1080 - emax + lv + sg - 64 + 2 * (sl.e - 57));
#pragma unroll
      for (int a = 0; a < 2; ++a)
#pragma unroll
        for (int b = 0; b < 2; ++b) {
          const longlong2 t = *reinterpret_cast<const longlong2*>(at_x(b, warp, g + 8 * a < NP ? g + 8 * a : 0));
          wv[a][b][0] = to_double(sum[a][b][0] + t.x, scale);
          wv[a][b][1] = to_double(sum[a][b][1] + t.y, scale);
        }
    } else {
      elements_fp64<NP, 1>(tab, sG, OTF ? &geo[e].sg : gexp + e, 0, 1, abc);
#pragma unroll
      for (int a = 0; a < 2; ++a)
#pragma unroll
        for (int b = 0; b < 2; ++b)
#pragma unroll
          for (int y = 0; y < 2; ++y) {
            const double* s = abc + warp * NP2 + off(a, b) + y;
            wv[a][b][y] = in(a, b, y) ? s[0] + s[P] + s[2 * P] : 0.0;
          }
      __syncthreads();
      for (unsigned q = threadIdx.x; q < kSlices * S::kDigit / 4; q += S::kThreads)  // beyond the points, as at the start
        reinterpret_cast<uint32_t*>(smem + S::kOffD)[q] = 0u;
      if (!OTF && threadIdx.x == 0 && more) load_factors(e + gridDim.x);
    }
#pragma unroll
    for (int a = 0; a < 2; ++a)
#pragma unroll
      for (int b = 0; b < 2; ++b) {
        if constexpr (CG) {
#pragma unroll
          for (int y = 0; y < 2; ++y)
            if (in(a, b, y)) {
              w[e * P + cg_pos(NP, q2 + 8 * b + y, g + 8 * a, warp)] = wv[a][b][y];
              dot = fma(v[a][b][y], wv[a][b][y], dot);
            }
        } else {
          store2(w, a, b, wv[a][b]);
        }
      }
  }
  if constexpr (CG) {
    const double s = block_sum(dot, sRed);
    if (threadIdx.x == 0) partials[blockIdx.x] = s;
  }
}

template <int NP, bool CG, bool OTF>
sem_status launch_slice16_t(int N, const AxLaunch& a, cudaStream_t s) {
  using S = Slice16Shape<NP>;
  static const int max_blocks = [] {
    cudaFuncSetAttribute(k_ax_slice16<NP, CG, OTF>, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(S::bytes(OTF)));
    int dev = 0, sms = 0, per_sm = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_ax_slice16<NP, CG, OTF>, S::kThreads, S::bytes(OTF));
    return (per_sm > 0 ? per_sm : 1) * (sms > 0 ? sms : 1);
  }();
  static const SliceTab<NP> sl = make_slice_tab<NP>(N);
  static const GllParam<NP, double> tab = make_gll_param<NP, double>(N);
  static const GeoNodes<NP> nodes = make_geo_nodes<NP>(N);
  int grid = max_blocks < kRedMax ? max_blocks : kRedMax;
  if (a.E < grid) grid = static_cast<int>(a.E);
  if (a.grid_out) *a.grid_out = grid;
  k_ax_slice16<NP, CG, OTF><<<grid, S::kThreads, S::bytes(OTF), s>>>(
      tab, sl, nodes, a.E, static_cast<const double*>(a.u), static_cast<double*>(a.w), static_cast<const int2*>(a.G),
      a.gexp, a.geo, static_cast<const double*>(a.r), static_cast<const double*>(a.minv), static_cast<double*>(a.x),
      static_cast<double*>(a.p), a.st, a.partials, a.err);
  count_launch();
  SEM_CUDA_TRY(cudaGetLastError());
  return SEM_OK;
}

}  // namespace
}  // namespace sem
