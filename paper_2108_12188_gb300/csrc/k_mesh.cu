// Element geometry kernels: trilinear-map coefficients, geometric factors G and mass B
// (Eq. 4's G^e; Section 4.2's six factors per point), physical coordinates, the local
// diagonal of A_L (Jacobi), the right-hand side B f, and small vector utilities.
//
// A trilinear hexahedron with vertices X_v, v = a + 2b + 4c, is
//   x(xi, eta, gam) = sum_v X_v phi_a(xi) phi_b(eta) phi_c(gam),  phi_0 = (1-t)/2, phi_1 = (1+t)/2
//                   = a0 + a1 xi + a2 eta + a3 gam + a4 xi eta + a5 xi gam + a6 eta gam + a7 xi eta gam
// with a_m = (1/8) sum_v s_m(v) X_v and s_m the products of the corner signs (2a-1, 2b-1, 2c-1)
// selected by the monomial. a1..a7 are differences of vertices, so rounding them to FP32
// keeps their relative accuracy (absolute coordinates would lose bits to cancellation).
#include "k_common.cuh"

namespace sem {
namespace {

constexpr int kThreads = 256;

struct GllAll {  // xi and w of one order, FP64
  double xi[kMaxNp], w[kMaxNp];
};
GllAll gll_all(int N) {
  const GllTable& t = gll_table(N);
  GllAll g{};
  for (int a = 0; a <= N; ++a) {
    g.xi[a] = t.xi[a];
    g.w[a] = t.w[a];
  }
  return g;
}

__global__ void k_coefficients(int64_t E, const double* __restrict__ X, double* __restrict__ c64,
                               float* __restrict__ c32) {
  const int64_t e = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x;
  if (e >= E) return;
  const double* x = X + e * 24;
  for (int comp = 0; comp < 3; ++comp) {
    double a[8] = {0, 0, 0, 0, 0, 0, 0, 0};
    for (int v = 0; v < 8; ++v) {
      const double sa = (v & 1) ? 1.0 : -1.0, sb = (v & 2) ? 1.0 : -1.0, sc = (v & 4) ? 1.0 : -1.0;
      const double xv = x[v * 3 + comp];
      a[0] += xv;
      a[1] += sa * xv;
      a[2] += sb * xv;
      a[3] += sc * xv;
      a[4] += sa * sb * xv;
      a[5] += sa * sc * xv;
      a[6] += sb * sc * xv;
      a[7] += sa * sb * sc * xv;
    }
    for (int m = 0; m < 8; ++m) {
      const double am = 0.125 * a[m];
      c64[e * 24 + m * 3 + comp] = am;
      c32[e * 24 + m * 3 + comp] = static_cast<float>(am);
    }
  }
}

struct PointGeom {
  double g[3][3];  // g[b] = dx/dxi_b
};

__device__ __forceinline__ void jacobian_columns(const double* a, double xi, double eta, double gam, double g0[3],
                                                 double g1[3], double g2[3]) {
  for (int c = 0; c < 3; ++c) {
    const double a1 = a[3 + c], a2 = a[6 + c], a3 = a[9 + c], a4 = a[12 + c], a5 = a[15 + c], a6 = a[18 + c],
                 a7 = a[21 + c];
    g0[c] = a1 + a4 * eta + a5 * gam + a7 * eta * gam;
    g1[c] = a2 + a4 * xi + a6 * gam + a7 * xi * gam;
    g2[c] = a3 + a5 * xi + a6 * eta + a7 * xi * eta;
  }
}

__device__ __forceinline__ void cross3(const double a[3], const double b[3], double out[3]) {
  out[0] = a[1] * b[2] - a[2] * b[1];
  out[1] = a[2] * b[0] - a[0] * b[2];
  out[2] = a[0] * b[1] - a[1] * b[0];
}

// C C^T with the cofactor rows c_b = g_{b+1} x g_{b+2}, and det J.
__device__ void point_cofactors(const double* a, double xi, double eta, double gam, double cc[6], double* det_out) {
  double g0[3], g1[3], g2[3], c0[3], c1[3], c2[3];
  jacobian_columns(a, xi, eta, gam, g0, g1, g2);
  cross3(g1, g2, c0);
  cross3(g2, g0, c1);
  cross3(g0, g1, c2);
  *det_out = g0[0] * c0[0] + g0[1] * c0[1] + g0[2] * c0[2];
  auto d = [](const double* p, const double* q) { return p[0] * q[0] + p[1] * q[1] + p[2] * q[2]; };
  cc[0] = d(c0, c0);
  cc[1] = d(c0, c1);
  cc[2] = d(c0, c2);
  cc[3] = d(c1, c1);
  cc[4] = d(c1, c2);
  cc[5] = d(c2, c2);
}

// G = w |det J| J^-1 J^-T = (w / det) C C^T; B = w det.
__device__ void point_geometry(const double* a, double xi, double eta, double gam, double wq, double G[6],
                               double* B, double* det_out) {
  double det;
  point_cofactors(a, xi, eta, gam, G, &det);
  const double s = wq / det;
  for (int m = 0; m < 6; ++m) G[m] = s * G[m];
  *B = wq * det;
  *det_out = det;
}

// Arrays of a mesh's geometry, each may be null: G in FP64, FP32 and as float pairs (high, low), B, and the scale of the
// on-the-fly factors w / det J. gs64, gs32: words per element of G.
struct GeometryOut {
  double* G64;
  float* G32;
  double* B64;
  float* B32;
  int64_t gs64, gs32;
  double* S64;
  float* S32;
  float* GX;
  __device__ __forceinline__ void put(int64_t e, int P, int r, const double (&G)[6], double B, double sc) const {
    for (int m = 0; m < 6; ++m) {
      if (G64) G64[e * gs64 + m * P + r] = G[m];
      if (G32) G32[e * gs32 + m * P + r] = static_cast<float>(G[m]);
      if (GX) {  // high = G rounded to FP32, low = the rest rounded to FP32
        const float h = static_cast<float>(G[m]);
        GX[2 * (e * gs64 + m * P + r)] = h;
        GX[2 * (e * gs64 + m * P + r) + 1] = static_cast<float>(G[m] - static_cast<double>(h));
      }
    }
    const int64_t idx = e * P + r;
    if (B64) B64[idx] = B;
    if (B32) B32[idx] = static_cast<float>(B);
    if (S64) S64[idx] = sc;
    if (S32) S32[idx] = static_cast<float>(sc);
  }
};

__global__ void k_geometry(const __grid_constant__ GllAll tab, int Np, int64_t E, const double* __restrict__ coef,
                           const __grid_constant__ GeometryOut out, int* __restrict__ bad) {
  const int64_t P = static_cast<int64_t>(Np) * Np * Np;
  const int64_t idx = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x;
  if (idx >= E * P) return;
  const int64_t e = idx / P;
  const int r = static_cast<int>(idx - e * P);
  const int i = r % Np, j = (r / Np) % Np, k = r / (Np * Np);
  const double wq = tab.w[i] * tab.w[j] * tab.w[k];
  double G[6], B, det;
  point_geometry(coef + e * 24, tab.xi[i], tab.xi[j], tab.xi[k], wq, G, &B, &det);
  if (!(det > 0.0) || !isfinite(det)) atomicOr(bad, 1);
  out.put(e, static_cast<int>(P), r, G, B, wq / det);
}

// The same with one element per block at the orders of ax_slice_order, with G as their fixed point too: sg = 59 -
// (exponent of the element's largest entry, row scales included), and the element for factors rebuilt on the fly (sw:
// geo_weight_scale). X null: not G. sG: 6 P doubles of dynamic shared memory (if X). bad: bit 0 det J <= 0, bit 1
// an element that fixed point rebuilds with less than FP64's precision. Bound by the FP64 pipe, as k_geometry is; exponents
// are taken from the bits.
__global__ void k_fixed_factors(const __grid_constant__ GllAll tab, int Np, int sw, const double* __restrict__ coef,
                                const __grid_constant__ GeometryOut out, int2* __restrict__ X, int* __restrict__ gexp,
                                GeoElement* __restrict__ geo, int* __restrict__ bad) {
  extern __shared__ double sG[];
  // largest exponents (as frexp has them) of |c_0|, |c_1|, |c_2| and their slopes, of G 2^(c_a + c_b) and of
  // G 2^(c_0 + c_1 + c_2); the smallest of det J
  __shared__ int sMax[5], sMin;
  const int P = Np * Np * Np;
  const int64_t e = blockIdx.x;
  const double* a = coef + e * 24;
  if (threadIdx.x < 5) sMax[threadIdx.x] = -4000;
  if (threadIdx.x == 0) sMin = 4000;
  __syncthreads();
  int most[5] = {-4000, -4000, -4000, -4000, -4000}, least = 4000;
  auto exponent = [](double v) {  // (4000: no finite number, see kSgFinite)
    const int ex = (__double2hiint(v) >> 20) & 0x7ff;
    return ex == 0 ? -4000 : ex == 0x7ff ? 4000 : ex - 1022;
  };
  // of a bound that rounding may have put below a power of two it reaches: the high word one up
  auto exponent_up = [&](double v) { return exponent(__hiloint2double(__double2hiint(v) + 1, 0)); };
  for (int r = threadIdx.x; r < P; r += blockDim.x) {
    const int i = r % Np, j = (r / Np) % Np, k = r / (Np * Np);
    const double wq = tab.w[i] * tab.w[j] * tab.w[k];
    double G[6], det;
    point_cofactors(a, tab.xi[i], tab.xi[j], tab.xi[k], G, &det);
    if (!(det > 0.0) || !isfinite(det)) atomicOr(bad, 1);
    least = min(least, exponent(__hiloint2double(__double2hiint(det) - 1, 0)));
    for (int d = 0; d < 3; ++d) {
      const int ex = exponent_up(G[d == 0 ? 0 : d == 1 ? 3 : 5]);  // |c|^2 < 2^ex
      most[d] = max(most[d], ex <= -4000 ? ex : (ex + 1) >> 1);
    }
    const double sc = wq / det;
    const int c[3] = {fixed_row_scale(Np, i), fixed_row_scale(Np, j), fixed_row_scale(Np, k)};
    for (int m = 0; m < 6; ++m) {
      G[m] = sc * G[m];
      const int ca = c[m < 3 ? 0 : m < 5 ? 1 : 2] + c[m < 3 ? m : m < 5 ? m - 2 : 2];
      most[3] = max(most[3], exponent(G[m]) + ca);
      most[4] = max(most[4], exponent_up(G[m]) + c[0] + c[1] + c[2]);
      if (X) sG[m * P + r] = exponent(G[m]) > -4000 ? __hiloint2double(__double2hiint(G[m]) + (ca << 20), __double2loint(G[m])) : 0.0;
    }
    out.put(e, P, r, G, wq * det, sc);
  }
  for (int q = threadIdx.x; q < 3 * Np; q += blockDim.x) {  // 4 P x K and 4 K x M of row q % 3, node q / 3
    const int d = q % 3, p0 = d == 0 ? 2 : d == 1 ? 3 : 1, p1 = d == 0 ? 4 : d == 1 ? 6 : 5, m0 = d == 0 ? 3 : d == 1 ? 1 : 2,
              m1 = d == 0 ? 5 : d == 1 ? 4 : 6, k0 = d == 0 ? 6 : d == 1 ? 5 : 4;
    double p[3], m[3], k[3], v[3];
    for (int c = 0; c < 3; ++c) {
      const double xi = tab.xi[q / 3];
      p[c] = a[3 * p0 + c] + a[3 * p1 + c] * xi;
      m[c] = a[3 * m0 + c] + a[3 * m1 + c] * xi;
      k[c] = a[3 * k0 + c] + a[21 + c] * xi;
    }
    int ex = -4000;
    cross3(p, k, v);
    for (int c = 0; c < 3; ++c) ex = max(ex, exponent_up(v[c]) + 2);
    cross3(k, m, v);
    for (int c = 0; c < 3; ++c) ex = max(ex, exponent_up(v[c]) + 2);
    for (int r = 0; r < 3; ++r)
      if (r == d) most[r] = max(most[r], ex);
  }
  for (int m = 0; m < 5; ++m) atomicMax(&sMax[m], most[m]);
  atomicMin(&sMin, least);
  __syncthreads();
  const int sg = 59 - sMax[3];
  if (threadIdx.x == 0) {
    double size = 0.0;
    for (int c = 0; c < 3; ++c) {
      double t = 0.0;
      for (int m = 1; m < 8; ++m) t += fabs(a[3 * m + c]);
      size = fmax(size, t);
    }
    const int row[3] = {sMax[0], sMax[1], sMax[2]};
    GeoElement g;
    const int qa = geo_scale(g, exponent_up(size), row, sMin, sMax[3], sMax[4], sw);
    for (int m = 0; m < 7; ++m)
      for (int c = 0; c < 3; ++c) g.a[m][c] = geo_fixed(a[3 * m + 3 + c], qa);
    geo[e] = g;
    if (g.sg == kGeoNone) atomicOr(bad, 2);
    if (gexp) gexp[e] = sg;
  }
  if (!X) return;
  for (int q = threadIdx.x; q < 6 * P; q += blockDim.x) {
    const long long x = (geo_fixed(sG[q], sg + 1) + 1) >> 1;  // rounded
    const int lo = static_cast<int>(static_cast<uint32_t>(x));
    X[e * 6 * P + q] = make_int2(lo, static_cast<int>((x - lo) >> 32));
  }
}

__global__ void k_coords(const __grid_constant__ GllAll tab, int Np, int64_t E, const double* __restrict__ coef,
                         double* __restrict__ xyz, int64_t n) {
  const int64_t P = static_cast<int64_t>(Np) * Np * Np;
  const int64_t idx = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x;
  if (idx >= E * P) return;
  const int64_t e = idx / P;
  const int r = static_cast<int>(idx - e * P);
  const double xi = tab.xi[r % Np], eta = tab.xi[(r / Np) % Np], gam = tab.xi[r / (Np * Np)];
  const double* a = coef + e * 24;
  for (int c = 0; c < 3; ++c)
    xyz[c * n + idx] = a[c] + a[3 + c] * xi + a[6 + c] * eta + a[9 + c] * gam + a[12 + c] * xi * eta +
                       a[15 + c] * xi * gam + a[18 + c] * eta * gam + a[21 + c] * xi * eta * gam;
}

// Diagonal of D^T G D at (i, j, k):
//   sum_l D_li^2 G11(l,j,k) + sum_l D_lj^2 G22(i,l,k) + sum_l D_lk^2 G33(i,j,l)
//   + 2 D_ii D_jj G12 + 2 D_ii D_kk G13 + 2 D_jj D_kk G23.
// One block per element; G of the element is built in shared memory first.
__global__ void k_local_diag(const __grid_constant__ GllTable tab, int Np, int64_t E, const double* __restrict__ coef,
                             double* __restrict__ d) {
  extern __shared__ double sG[];  // [6][P]
  const int P = Np * Np * Np;
  const int64_t e = blockIdx.x;
  for (int r = threadIdx.x; r < P; r += blockDim.x) {
    const int i = r % Np, j = (r / Np) % Np, k = r / (Np * Np);
    double G[6], B, det;
    point_geometry(coef + e * 24, tab.xi[i], tab.xi[j], tab.xi[k], tab.w[i] * tab.w[j] * tab.w[k], G, &B, &det);
    for (int m = 0; m < 6; ++m) sG[m * P + r] = G[m];
  }
  __syncthreads();
  for (int r = threadIdx.x; r < P; r += blockDim.x) {
    const int i = r % Np, j = (r / Np) % Np, k = r / (Np * Np);
    double s = 0.0;
    for (int l = 0; l < Np; ++l) {
      const double dli = tab.D[l * Np + i], dlj = tab.D[l * Np + j], dlk = tab.D[l * Np + k];
      s += dli * dli * sG[0 * P + (k * Np + j) * Np + l];
      s += dlj * dlj * sG[3 * P + (k * Np + l) * Np + i];
      s += dlk * dlk * sG[5 * P + (l * Np + j) * Np + i];
    }
    const double dii = tab.D[i * Np + i], djj = tab.D[j * Np + j], dkk = tab.D[k * Np + k];
    s += 2.0 * dii * djj * sG[1 * P + r] + 2.0 * dii * dkk * sG[2 * P + r] + 2.0 * djj * dkk * sG[4 * P + r];
    d[e * P + r] = s;
  }
}

// (-1)^(n / 2) / n!, the coefficients of the sine's and cosine's Taylor sums.
struct TaylorTab {
  double v[18];
};
TaylorTab taylor_tab() {
  TaylorTab t{};
  double f = 1.0;
  for (int n = 0; n < 18; ++n) {
    if (n > 0) f /= n;
    t.v[n] = n / 2 % 2 ? -f : f;
  }
  return t;
}

// Terms of the sums that leave less than 2^-55 out for |t| <= pi slope; 0: too large for them.
__device__ __forceinline__ int taylor_terms(double slope) {
  const double a = fabs(slope);
  return a <= 1.0 / 32 ? 4 : a <= 1.0 / 16 ? 5 : a <= 1.0 / 8 ? 6 : a <= 1.0 / 4 ? 8 : 0;
}
// sin t and cos t up to t^(2 terms + 1) and t^(2 terms).
__device__ __forceinline__ void sincos_small(const TaylorTab& k, int terms, double t, double* s, double* c) {
  const double t2 = t * t;
  double p = k.v[2 * terms + 1], q = k.v[2 * terms];
#pragma unroll 1
  for (int n = terms - 1; n >= 1; --n) {
    p = fma(p, t2, k.v[2 * n + 1]);
    q = fma(q, t2, k.v[2 * n]);
  }
  *s = fma(t * t2, p, t);
  *c = fma(t2, q, 1.0);
}

// (B f)(x) with f = (a^2+b^2+c^2) pi^2 sin(a pi x) sin(b pi y) sin(c pi z), `split` threads per i-row of an
// element (each every split-th pair of points +-xi), epb elements per block or, for chunk < rows, `chunk`
// rows of one element. The kernel is bound by
// FP64 instructions (2 multiply-adds per clock per SM), and three sinpi and the Jacobian at every point
// are 190 of them. Along a row x is linear in xi, so sin(a pi x) is a rotation of the row's midpoint value
// by angles +-a pi B xi_i, whose sines and cosines are short sums and serve two points each (the GLL nodes
// are symmetric); the midpoints follow the same way from one value per k-plane. Along the row det J is a
// quadratic in xi, formed once. 55 of them per point at N = 9: with the gather-scatter 2.14 ->
// 0.83 ms at 8.0M points, the FP64 pipe 90% busy. Elements too large for the short sums (|a B| > 1/4) take sincospi and sinpi.
__global__ void k_rhs_local(const __grid_constant__ GllAll tab, const __grid_constant__ TaylorTab tay, int Np, int epb,
                            int split, int chunk, int64_t E, const double* __restrict__ coef, int fa, int fb, int fc,
                            double* __restrict__ out) {
  extern __shared__ double sh[];  // [epb][P] values, then [epb][Np][3] (sin, cos) of the planes' midpoints
  constexpr double kPi = 3.14159265358979323846;
  const int P = Np * Np * Np, rows = Np * Np;
  double2* plane = reinterpret_cast<double2*>(sh + static_cast<size_t>(epb) * P + (static_cast<size_t>(epb) * P) % 2);
  const int parts = (rows + chunk - 1) / chunk, row0 = blockIdx.x % parts * chunk;  // (parts > 1: epb = 1)
  const int64_t e0 = static_cast<int64_t>(blockIdx.x / parts) * epb;
  const int count = static_cast<int>(E - e0 < epb ? E - e0 : epb);
  const int my_rows = parts > 1 ? min(chunk, rows - row0) : count * rows;
  const double f[3] = {static_cast<double>(fa), static_cast<double>(fb), static_cast<double>(fc)};
  for (int q = threadIdx.x; q < count * Np * 3; q += blockDim.x) {
    const int c = q % 3, k = q / 3 % Np;
    const double* a = coef + (e0 + q / (3 * Np)) * 24;
    double s, co;
    sincospi(f[c] * fma(a[9 + c], tab.xi[k], a[c]), &s, &co);
    plane[q] = make_double2(s, co);
  }
  __syncthreads();
  for (int q = threadIdx.x; q < my_rows * split; q += blockDim.x) {
    const int part = q % split, row = row0 + q / split, el = row / rows, j = row % rows % Np, k = row % rows / Np;
    const double* a = coef + (e0 + el) * 24;
    const double eta = tab.xi[j], gam = tab.xi[k], eg = eta * gam;
    double g0[3], p[3], pq[3], r[3], rs[3], S[3], C[3], base[3], turn[3];
    int terms[3];
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      const double a1 = a[3 + c], a2 = a[6 + c], a3 = a[9 + c], a4 = a[12 + c], a5 = a[15 + c], a6 = a[18 + c],
                   a7 = a[21 + c];
      g0[c] = a1 + a4 * eta + a5 * gam + a7 * eg;  // dx/dxi, constant along the row
      p[c] = a2 + a6 * gam;                        // dx/deta = p + xi pq
      pq[c] = a4 + a7 * gam;
      r[c] = a3 + a6 * eta;                        // dx/dgam = r + xi rs
      rs[c] = a5 + a7 * eta;
      const double mid = fma(a3, gam, a[c]), up = f[c] * p[c];
      const double2 m = plane[(el * Np + k) * 3 + c];
      S[c] = m.x;
      C[c] = m.y;
      base[c] = f[c] * fma(p[c], eta, mid);
      if (const int n = taylor_terms(up)) {
        double ds, dc;
        sincos_small(tay, n, kPi * up * eta, &ds, &dc);
        S[c] = fma(m.x, dc, m.y * ds);
        C[c] = fma(m.y, dc, -m.x * ds);
      } else {
        sincospi(base[c], &S[c], &C[c]);
      }
      const double along = f[c] * g0[c];
      terms[c] = taylor_terms(along);
      turn[c] = terms[c] ? kPi * along : along;
    }
    double h1[3], h2[3];  // det J = (p + xi pq) . ((r + xi rs) cross g0)
    cross3(r, g0, h1);
    cross3(rs, g0, h2);
    auto dot = [](const double* x, const double* y) { return x[0] * y[0] + x[1] * y[1] + x[2] * y[2]; };
    const double pi2 = 9.869604401089358;  // pi^2
    const double w = tab.w[j] * tab.w[k] * ((fa * fa + fb * fb + fc * fc) * pi2);
    const double d0 = w * dot(p, h1), d1 = w * (dot(p, h2) + dot(pq, h1)), d2 = w * dot(pq, h2);
    double* o = sh + (row - row0) * Np;
#pragma unroll 1
    for (int i = part; 2 * i < Np; i += split) {
      const double xi = tab.xi[i];
      double lo = tab.w[i], hi = lo;  // the points xi and -xi
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        if (terms[c]) {
          double ds, dc;
          sincos_small(tay, terms[c], turn[c] * xi, &ds, &dc);
          const double sc = S[c] * dc;
          lo *= fma(C[c], ds, sc);
          hi *= fma(-C[c], ds, sc);
        } else {
          lo *= sinpi(fma(turn[c], xi, base[c]));
          hi *= sinpi(fma(turn[c], -xi, base[c]));
        }
      }
      o[i] = lo * fma(xi, fma(xi, d2, d1), d0);
      o[Np - 1 - i] = hi * fma(-xi, fma(-xi, d2, d1), d0);
    }
  }
  __syncthreads();
  for (int q = threadIdx.x; q < my_rows * Np; q += blockDim.x) out[e0 * P + row0 * Np + q] = sh[q];
}

template <typename T>
__global__ void k_scatter(int64_t n, const int32_t* __restrict__ glo, const T* __restrict__ ug, T* __restrict__ ul) {
  for (int64_t i = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x; i < n;
       i += static_cast<int64_t>(gridDim.x) * blockDim.x)
    ul[i] = ug[glo[i]];
}

__global__ void k_invert(int64_t n, const double* __restrict__ d, double* __restrict__ m64, float* __restrict__ m32) {
  for (int64_t i = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x; i < n;
       i += static_cast<int64_t>(gridDim.x) * blockDim.x) {
    const double v = 1.0 / d[i];
    if (m64) m64[i] = v;
    if (m32) m32[i] = static_cast<float>(v);
  }
}

__global__ void k_cast(int64_t n, const double* __restrict__ in, float* __restrict__ out) {
  for (int64_t i = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x; i < n;
       i += static_cast<int64_t>(gridDim.x) * blockDim.x)
    out[i] = static_cast<float>(in[i]);
}

int sm_count() {
  static const int n = [] {
    int dev = 0, sms = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    return sms > 0 ? sms : 1;
  }();
  return n;
}

// One thread per item, at most 32 blocks per SM (grid-stride beyond).
int grid_for(int64_t n) {
  const int cap = 32 * sm_count();
  const int64_t b = (n + kThreads - 1) / kThreads;
  return static_cast<int>(b < cap ? (b > 0 ? b : 1) : cap);
}

}  // namespace

sem_status launch_coefficients(int64_t E, const double* X, double* coef64, float* coef32, cudaStream_t s) {
  k_coefficients<<<ceil_div(E, 128), 128, 0, s>>>(E, X, coef64, coef32);
  count_launch();
  SEM_CUDA_TRY(cudaGetLastError());
  return SEM_OK;
}

sem_status launch_geometry(int N, int64_t E, const double* coef64, double* G64, float* G32, double* B64, float* B32,
                           int* bad, int64_t gs64, int64_t gs32, cudaStream_t s, double* S64, float* S32,
                           float* GX, int2* X, int* gexp, GeoElement* geo) {
  const int Np = N + 1, P = Np * Np * Np;
  const GeometryOut out{G64, G32, B64, B32, gs64, gs32, S64, S32, GX};
  if (geo) {
    int c[kMaxNp];
    for (int i = 0; i < Np; ++i) c[i] = fixed_row_scale(Np, i);
    static const cudaError_t attr = cudaFuncSetAttribute(k_fixed_factors, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                                         6 * kMaxNp * kMaxNp * kMaxNp * static_cast<int>(sizeof(double)));
    SEM_CUDA_TRY(attr);
    k_fixed_factors<<<static_cast<unsigned>(E), P < 128 ? 64 : P < 600 ? 128 : 256,
                      X ? 6 * static_cast<size_t>(P) * sizeof(double) : 0, s>>>(
        gll_all(N), Np, geo_weight_scale(gll_table(N).w, c, Np), coef64, out, X, gexp, geo, bad);
  } else {
    k_geometry<<<ceil_div(E * P, kThreads), kThreads, 0, s>>>(gll_all(N), Np, E, coef64, out, bad);
  }
  count_launch();
  SEM_CUDA_TRY(cudaGetLastError());
  return SEM_OK;
}

sem_status launch_coords(int N, int64_t E, const double* coef64, double* xyz, int64_t n, cudaStream_t s) {
  k_coords<<<ceil_div(n, kThreads), kThreads, 0, s>>>(gll_all(N), N + 1, E, coef64, xyz, n);
  count_launch();
  SEM_CUDA_TRY(cudaGetLastError());
  return SEM_OK;
}

sem_status launch_local_diag(int N, int64_t E, const double* coef64, double* d, cudaStream_t s) {
  const int Np = N + 1, P = Np * Np * Np;
  const size_t smem = 6 * static_cast<size_t>(P) * sizeof(double);
  static const cudaError_t attr = cudaFuncSetAttribute(k_local_diag, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                                       6 * kMaxNp * kMaxNp * kMaxNp * static_cast<int>(sizeof(double)));
  SEM_CUDA_TRY(attr);
  // E blocks: at most 2^31 / 8 elements (the local-size limit), within the grid x limit
  k_local_diag<<<static_cast<unsigned>(E), P < 512 ? P : 512, smem, s>>>(gll_table(N), Np, E, coef64, d);
  count_launch();
  SEM_CUDA_TRY(cudaGetLastError());
  return SEM_OK;
}

sem_status launch_rhs_local(int N, int64_t E, const double* coef64, int a, int b, int c, double* out, cudaStream_t s) {
  constexpr int kBlock = 128;
  const int Np = N + 1, P = Np * Np * Np, rows = Np * Np;
  // Meshes whose rows do not give every scheduler four warps: a thread per pair of points (the row's share
  // of the work repeated) and blocks of one pass over at most 128 of them, for a short chain on many
  // SMs (4^3 elements at N = 7, with the gather-scatter: 21 us; a thread per row 35 us).
  const int split = E * rows < static_cast<int64_t>(sm_count()) * 512 ? (Np + 1) / 2 : 1;
  const int chunk = split > 1 ? kBlock / split : rows;
  // elements per block: the fewest idle lanes in the block's last pass over its rows, 32 KB of values at most
  int epb = 1;
  auto waste = [&](int q) { return 1.0 - static_cast<double>(q) * rows / (ceil_div(static_cast<int64_t>(q) * rows, kBlock) * kBlock); };
  if (split == 1)
    for (int q = 2; q * P <= 4096; ++q)
      if (waste(q) < waste(epb) - 1e-9) epb = q;
  const size_t smem = (static_cast<size_t>(epb) * P + 1 + 6 * static_cast<size_t>(epb) * Np) * sizeof(double);
  static const TaylorTab tay = taylor_tab();
  const int64_t blocks = split > 1 ? E * ceil_div(rows, chunk) : ceil_div(E, epb);
  k_rhs_local<<<static_cast<unsigned>(blocks), kBlock, smem, s>>>(gll_all(N), tay, Np, epb, split,
                                                                  chunk < rows ? chunk : rows, E, coef64, a, b, c, out);
  count_launch();
  SEM_CUDA_TRY(cudaGetLastError());
  return SEM_OK;
}

sem_status launch_scatter(sem_prec prec, int64_t n, const int32_t* glo, const void* ug, void* ul, cudaStream_t s) {
  if (prec == SEM_F64)
    k_scatter<double><<<grid_for(n), kThreads, 0, s>>>(n, glo, static_cast<const double*>(ug), static_cast<double*>(ul));
  else
    k_scatter<float><<<grid_for(n), kThreads, 0, s>>>(n, glo, static_cast<const float*>(ug), static_cast<float*>(ul));
  count_launch();
  SEM_CUDA_TRY(cudaGetLastError());
  return SEM_OK;
}

sem_status launch_invert(int64_t n, const double* d, double* m64, float* m32, cudaStream_t s) {
  k_invert<<<grid_for(n), kThreads, 0, s>>>(n, d, m64, m32);
  count_launch();
  SEM_CUDA_TRY(cudaGetLastError());
  return SEM_OK;
}

sem_status launch_cast(int64_t n, const double* in, float* out, cudaStream_t s) {
  k_cast<<<grid_for(n), kThreads, 0, s>>>(n, in, out);
  count_launch();
  SEM_CUDA_TRY(cudaGetLastError());
  return SEM_OK;
}

}  // namespace sem
