// FP64 local operator w = A_L u = D^T G D u (Eq. 4, Section 3.1) with stored factors or with factors
// rebuilt on the fly (k_geo_fixed.cuh), its line contractions on the tensor cores with more than FP64 accuracy: the products run exactly, on
// integer digits (the error-free splitting of Ozaki, Ogita, Oishi and Rump, "Error-free
// transformations of matrix multiplication by using fast routines of matrix multiplication and
// its applications", Numerical Algorithms 59, 2012), and everything between the input and
// the output is 64-bit fixed point on the integer and FP32 pipes.
//
// Why: GB300 runs 2 FP64 multiply-adds per clock per SM. The FP64 operator (k_ax) issues 48 FP64
// instructions per point and is bound by that pipe at ten times its HBM time. Here no FP64
// instruction is left in the contractions and the geometry.
//
// Fixed point. The element's values are scaled by one power of two to |U| < 2^58 (from the
// largest exponent in the element) and cut into kSlices balanced digits of 10 bits,
// U = sum_s u_s 2^(50 - 10 s), |u_s| <= 512, |u_0| <= 256; D (and D^T) likewise, D 2^e =
// sum_t d_t 2^(50 - 10 t). The digits are exact FP16 integers, and
//   C_g = sum over s + t = g of sum_l d_t(i, l) u_s(l)
// is an integer below 2^24, so mma.sync with FP32 accumulators forms it exactly. The groups
// g = 0..6 are kept, V = sum_g C_g 2^(43 - 10 g) (weight 2^60 / 2^57 of the product), the rest is
// below 2^-7 units of V. Groups 0..4 accumulate on top of 1.5 2^23 (make_slice_tab checks that
// |C_g| < 2^22), so their bits are the integers and V takes five integer multiply-adds.
//
// Geometry. The mesh keeps G as 64-bit fixed point (k_fixed_factors), X = G_ab / (s_a s_b) 2^sg with
// |X| <= 2^59 and sg one number per element (fixed_row_scale has s). The derivatives are shifted up
// by the same count over the element, to |V| < 2^61; with 32-bit halves
//   R = sum_b X_ab V_b / 2^64 = sum xh vh + (sum xh vl + xl vh) / 2^32
// takes nine wide multiply-adds per row (the dropped xl vl is below one unit) and stays below
// 2^58, so its digits are cut without another scaling. The three transposed contractions are added
// as integers and rounded to FP64 once.
//
// What bounds it: dependent integer work. Of 371 instructions per point (429 in CG mode) 154 (168) run on the ALU, 134 (150) are
// integer and FP32 multiply-adds of the heavy FMA pipe, 25.5 mma.sync. A probe of either kind or both mixed ran 64 lanes a
// clock per SM; at that rate the two take 72% of the time (66%), with 38% and 45% of their pipes' cycles, and what is left is
// latency: four warps per scheduler (128 registers) that wait on the instruction before (1.8 of 7 stalled), on the pipes
// (1.1), on barriers and shared memory. 16.8M points, N = 7: 1.497 ms in FP64 (k_ax, 95% of the FP64 peak by Eq. 11 flops) ->
// 0.337 ms, 0.46 of the HBM bandwidth. In CG mode with the fused prologue 0.411 ms (0.62); the prologue takes 0.02 ms and saves
// 0.067 in the update kernel: one Jacobi-CG iteration 1.779 -> 0.554 ms.
//
// On the fly (Section 5.1's rematerialised factors) the same kernel fills its factor buffer from the element's
// coefficients, with about 700 instructions per point on the same pipes, still far below the 45 FP64 instructions
// of k_ax for it. A_L in ms, k_ax and this kernel, 16.0 to 17.6M points: N = 3 2.84 and 1.17, N = 5 3.31 and 1.74, N = 6 3.23 and
// 1.49, N = 7 2.89 and 0.99, N = 9 4.07 and 2.36, N = 10 3.13 and 1.76, N = 11 3.49 and 1.45 (of these the factors take
// 0.5 ms, the row tables 0.05 and at N = 3 0.2); with the per-point scale of SEM_AX_OTF_SCALE, which is not read
// here, k_ax takes 0.8 to 0.9 of that. Error against long double (jittered elements, random u, N = 9) as with k_ax or below:
// 1.9e-16 and 2.6e-16, stored 2.4e-16 and 2.6e-16.
//
// Error against 64 bits (relative 2-norm of w, N = 7, jittered elements, CPU model of both
// kernels against an 80-bit reference; k_ax in brackets): random u 8e-17 (1.8e-16), a sine over 8^3
// elements 4e-16 (1.4e-14), one plus 1e-8 of a sine 5e-9 (1.2e-6), aspect ratio 100 4e-12 (5e-11),
// exp(-3 (x + y + z)) over two elements 6e-16 (3.0e-15). Fixed point is relative to the element's
// largest value, and so is the error at every node, see kNear.
//
// Elements that fixed point does not take (an infinity or NaN, magnitudes within about 2^60 of the
// ends of the FP64 range, few values near the largest, see kNear) run the FP64 lines of k_ax, in elements_fp64.
#pragma once

#include <cuda_fp16.h>

#include <algorithm>
#include <cmath>

#include "k_ax.cuh"
#include "k_geo_fixed.cuh"
#include "k_tma.cuh"

namespace sem {
namespace {

constexpr int kSlices = 6;                 // digits of every operand
constexpr float kMagic = 12582912.0f;      // 1.5 2^23: adding it leaves an integer in the low bits
constexpr uint32_t kMagicBits = 0x4b400000u;

// Digits of D ([0]) and D^T ([1]) as FP16 pairs: d[m][t][row][q] holds columns 2q and 2q + 1 of
// digit t (top digit first); M = digits * 2^-e. The rows of D (and with them the columns of D^T)
// are scaled by 2^-fixed_row_scale. For NP <= 4 the matrix repeats along the diagonal, once per element
// of the block's row of elements; entries beyond NP points are zero.
template <int NP>
struct SliceTab {
  static constexpr int R = NP <= 8 ? 8 : 16;
  uint32_t d[2][kSlices][R][R / 2];
  int e;
};

// D is used as diag(s) D and G_ab as G_ab / (s_a s_b), s = 2^-fixed_row_scale (at the two ends, 1
// inside): the end rows of D are the largest and the quadrature weights there the smallest, so
// with both evened out the factors and derivatives of an element use their leading bits better.

// Points per direction an element takes of a block's 8: eight elements of 4 points share a block.
__host__ __device__ constexpr int slice_width(int NP) { return NP <= 4 ? 4 : 8; }

inline uint32_t half_bits(int v) {  // |v| <= 2048: exact
  const __half h = __float2half_rn(static_cast<float>(v));
  uint16_t b;
  static_assert(sizeof(h) == sizeof(b), "FP16 is two bytes");
  memcpy(&b, &h, 2);
  return b;
}

// Groups that accumulate on top of kMagic: as many as stay below 2^22 at the order without giving up more
// than one bit of D (five groups would cost N = 9 four bits of D, four N = 11 four).
__host__ __device__ constexpr int magic_groups(int NP) { return NP <= 8 ? 5 : NP <= 11 ? 4 : 3; }

// The largest e such that |D 2^e| <= 511 2^50, every |C_g| that accumulates on kMagic stays below 2^22
// for any digits |u_0| <= 256, |u_s| <= 512, and |V| = |U D 2^e| / 2^57 stays below 2^61.
template <int NP>
SliceTab<NP> make_slice_tab(int N) {
  constexpr int kGroups = magic_groups(NP), R = SliceTab<NP>::R;
  const GllTable& t = gll_table(N);
  SliceTab<NP> r{};
  for (int e = 60;; --e) {
    bool ok = true;
    int dig[2][kSlices][NP][NP];
    for (int m = 0; m < 2 && ok; ++m)
      for (int i = 0; i < NP && ok; ++i) {
        double sum = 0.0, cg[kGroups] = {};
        for (int l = 0; l < NP && ok; ++l) {
          const double v = std::ldexp(m == 0 ? t.D[i * NP + l] : t.D[l * NP + i], e - fixed_row_scale(NP, m == 0 ? i : l));
          ok = std::fabs(v) <= std::ldexp(511.0, 50);
          if (!ok) break;
          sum += std::fabs(v);
          int64_t x = std::llrint(v);
          for (int q = kSlices - 1; q > 0; --q) {
            const int64_t low = ((x + 512) & 1023) - 512;
            dig[m][q][i][l] = static_cast<int>(low);
            x = (x - low) >> 10;
          }
          dig[m][0][i][l] = static_cast<int>(x);
          for (int g = 0; g < kGroups; ++g)
            for (int s = 0; s <= g; ++s) cg[g] += (s == 0 ? 256.0 : 512.0) * std::abs(dig[m][g - s][i][l]);
        }
        for (double c : cg) ok = ok && c < 4194304.0;
        ok = ok && sum * 2.0 < std::ldexp(1.0, 61);
      }
    if (!ok) continue;
    r.e = e;
    for (int m = 0; m < 2; ++m)
      for (int q = 0; q < kSlices; ++q)
        for (int i = 0; i < NP; ++i)
          for (int l = 0; l < NP; ++l)
            for (int b = 0; b < (NP <= 8 ? 8 : 1); b += slice_width(NP))
              r.d[m][q][(b + i) % R][(b + l) / 2 % (R / 2)] |= half_bits(dig[m][q][i][l]) << (16 * (l % 2));
    return r;
  }
}

__device__ __forceinline__ void mma_f16(float (&d)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint32_t b0,
                                        uint32_t b1, float c0, float c1, float c2, float c3) {
  asm("mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%10,%11,%12,%13};"
      : "=f"(d[0]), "=f"(d[1]), "=f"(d[2]), "=f"(d[3])
      : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1), "f"(c0), "f"(c1), "f"(c2), "f"(c3));
}
// Accumulator start values kept in registers for the whole kernel: read back from shared memory,
// so that the compiler cannot rebuild them (four moves) before each of the mma they start.
struct Start {
  float m[4], h[4];  // (magic x 4), (magic, magic, 0, 0)
};
__device__ __forceinline__ void mma_start(float (&d)[4], const uint4& a, uint32_t b0, uint32_t b1, const float (&c)[4]) {
  mma_f16(d, a.x, a.y, a.z, a.w, b0, b1, c[0], c[1], c[2], c[3]);
}
__device__ __forceinline__ void mma_zero(float (&d)[4], const uint4& a, uint32_t b0, uint32_t b1) {
  mma_f16(d, a.x, a.y, a.z, a.w, b0, b1, 0.f, 0.f, 0.f, 0.f);
}
__device__ __forceinline__ void lds_quad(float (&q)[4], uint32_t addr) {
  asm volatile("ld.shared.v4.f32 {%0,%1,%2,%3}, [%4];" : "=f"(q[0]), "=f"(q[1]), "=f"(q[2]), "=f"(q[3]) : "r"(addr));
}
__device__ __forceinline__ void mma_add(float (&d)[4], const uint4& a, uint32_t b0, uint32_t b1) {
  mma_f16(d, a.x, a.y, a.z, a.w, b0, b1, d[0], d[1], d[2], d[3]);
}

__device__ __forceinline__ void ldsm4(uint32_t (&r)[4], uint32_t addr) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
               : "r"(addr)
               : "memory");
}
__device__ __forceinline__ void ldsm4t(uint32_t& r0, uint32_t& r1, uint32_t& r2, uint32_t& r3, uint32_t addr) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];"
               : "=r"(r0), "=r"(r1), "=r"(r2), "=r"(r3)
               : "r"(addr)
               : "memory");
}
__device__ __forceinline__ uint32_t transpose8x8(uint32_t v) {
  uint32_t r;
  asm volatile("movmatrix.sync.aligned.m8n8.trans.b16 %0, %1;" : "=r"(r) : "r"(v));
  return r;
}

// U of x: the signed significand scaled so that a value with biased exponent emax has its leading
// bit at 2^57, truncated.
__device__ __forceinline__ long long to_fixed(double x, int emax) {
  const uint32_t hi = static_cast<uint32_t>(__double2hiint(x)), lo = static_cast<uint32_t>(__double2loint(x));
  const int sh = min(63, 5 + emax - static_cast<int>((hi >> 20) & 0x7ffu));
  const uint32_t fh = (__funnelshift_l(lo, hi, 10) & 0x3fffffffu) | 0x40000000u;
  const unsigned long long f = ((static_cast<unsigned long long>(fh) << 32) | (lo << 10)) >> sh;
  const long long s = static_cast<int>(hi) >> 31;
  return (static_cast<long long>(f) ^ s) - s;
}

// Digits of U_a and U_b as FP16 pairs (a in the low half), top digit first. With 512 added at every
// digit position the digits are plain 10-bit fields; 0x6400 | field is 1024 + field in FP16.
__device__ __forceinline__ void digit_pairs(long long ua, long long ub, uint32_t (&d)[kSlices]) {
  constexpr unsigned long long kBias = 512ull * (1ull + (1ull << 10) + (1ull << 20) + (1ull << 30) + (1ull << 40) + (1ull << 50));
  const unsigned long long a = static_cast<unsigned long long>(ua) + kBias, b = static_cast<unsigned long long>(ub) + kBias;
  const uint32_t al = static_cast<uint32_t>(a), ah = static_cast<uint32_t>(a >> 32);
  const uint32_t bl = static_cast<uint32_t>(b), bh = static_cast<uint32_t>(b >> 32);
  auto field = [](uint32_t p) {
    const uint32_t f = (p & 0x03ff03ffu) | 0x64006400u;
    __half2 h;
    memcpy(&h, &f, 4);
    const uint32_t k = 0xe600e600u;  // -1536
    __half2 c;
    memcpy(&c, &k, 4);
    h = __hadd2(h, c);
    uint32_t r;
    memcpy(&r, &h, 4);
    return r;
  };
  d[5] = field(__byte_perm(al, bl, 0x5410));                                                   // bits 0..9
  d[4] = field(__byte_perm(al, bl, 0x6521) >> 2);                                              // 10..19
  d[3] = field(__byte_perm(al, bl, 0x7632) >> 4);                                              // 20..29
  d[2] = field(__byte_perm(__funnelshift_r(al, ah, 24), __funnelshift_r(bl, bh, 24), 0x5410) >> 6);  // 30..39
  d[1] = field(__byte_perm(ah, bh, 0x6521));                                                   // 40..49
  d[0] = field(__byte_perm(ah, bh, 0x7632) >> 2);                                              // 50..59
}

// a K + c as one wide integer multiply-add (the FMA pipes have room, the ALU does not).
template <unsigned K>
__device__ __forceinline__ unsigned long long madw(uint32_t a, unsigned long long c) {
  unsigned long long r;
  asm("mad.wide.u32 %0, %1, %2, %3;" : "=l"(r) : "r"(a), "n"(K), "l"(c));
  return r;
}

// V = sum_g C_g 2^(43 - 10 g) from the accumulators of the seven groups (0..4 on top of kMagic).
__device__ __forceinline__ long long combine(float f0, float f1, float f2, float f3, float f4, float f5, float f6) {
  constexpr unsigned long long kBase =
      0ull - static_cast<unsigned long long>(kMagicBits) * (1ull + (1ull << 3) + (1ull << 13) + (1ull << 23)) -
      (static_cast<unsigned long long>(static_cast<uint32_t>((kMagicBits << 1) + (kMagicBits << 11))) << 32);
  const float low = fmaf(fmaf(f6, 1.0f / 1024.0f, f5), 1.0f / 128.0f, kMagic);
  unsigned long long v = madw<1>(__float_as_uint(low), kBase);
  v = madw<8>(__float_as_uint(f4), v);
  v = madw<8192>(__float_as_uint(f3), v);
  v = madw<8388608>(__float_as_uint(f2), v);
  const uint32_t hi = static_cast<uint32_t>(v >> 32) + (__float_as_uint(f1) << 1) + (__float_as_uint(f0) << 11);
  return static_cast<long long>((static_cast<unsigned long long>(hi) << 32) | static_cast<uint32_t>(v));
}

// One tile of eight lines, outputs in the rows: acc rows 0..7 of acc[G] are group 2G, rows 8..15
// group 2G + 1; b[s] is the tile's digit s (k = contraction index, n = line), fa the lane's
// A fragments [d_o, d_(o+1); d_(o-1), d_o] for o = 0, 2, 4, 6. Value x (0, 1) of the lane: line
// 2 (lane % 4) + x, output lane / 4.
__device__ __forceinline__ void contract_lines(const Start& s0, const uint4* fa, const uint32_t (&b)[kSlices],
                                               long long (&v)[2]) {
  const uint4 a0 = fa[0], a2 = fa[32], a4 = fa[64], a6 = fa[96];
  float c0[4], c1[4], c2[4], c3[4];
  mma_start(c0, a0, b[0], b[1], s0.m);
  mma_start(c1, a2, b[0], b[1], s0.m);
  mma_start(c2, a4, b[0], b[1], s0.h);
  mma_zero(c3, a6, b[0], b[1]);
  mma_add(c1, a0, b[2], b[3]);
  mma_add(c2, a2, b[2], b[3]);
  mma_add(c3, a4, b[2], b[3]);
  mma_add(c2, a0, b[4], b[5]);
  mma_add(c3, a2, b[4], b[5]);
#pragma unroll
  for (int x = 0; x < 2; ++x) v[x] = combine(c0[x], c0[2 + x], c1[x], c1[2 + x], c2[x], c2[2 + x], c3[x]);
}

// Two tiles of eight lines in the rows (tile t: rows 8t..8t+7), outputs in the columns: a[S] holds
// the tiles' digits 2S and 2S + 1, fb the lane's B fragments [d_o; d_(o-1)] for o = 0..6. Value
// x of tile t: line lane / 4, output 2 (lane % 4) + x.
__device__ __forceinline__ void contract_rows(const Start& s0, const uint2* fb, const uint4 (&a)[3],
                                              long long (&v)[2][2]) {
  float c[7][4];
#pragma unroll
  for (int g = 0; g < 7; ++g) {
    const uint2 b = fb[32 * g];
    if (g < 5)
      mma_start(c[g], a[0], b.x, b.y, s0.m);
    else
      mma_zero(c[g], a[0], b.x, b.y);
  }
#pragma unroll
  for (int g = 2; g < 7; ++g) {
    const uint2 b = fb[32 * (g - 2)];
    mma_add(c[g], a[1], b.x, b.y);
  }
#pragma unroll
  for (int g = 4; g < 7; ++g) {
    const uint2 b = fb[32 * (g - 4)];
    mma_add(c[g], a[2], b.x, b.y);
  }
#pragma unroll
  for (int t = 0; t < 2; ++t)
#pragma unroll
    for (int x = 0; x < 2; ++x) {
      const int q = 2 * t + x;
      v[t][x] = combine(c[0][q], c[1][q], c[2][q], c[3][q], c[4][q], c[5][q], c[6][q]);
    }
}

// The high half of v for 32-bit signed halves: v = vh 2^32 + vl.
__device__ __forceinline__ int low_half(long long v) { return static_cast<int>(static_cast<uint32_t>(v)); }
__device__ __forceinline__ int high_half(long long v) {
  return static_cast<int>(v >> 32) + static_cast<int>(static_cast<uint32_t>(v) >> 31);
}

// The bits of the high word that v's magnitude uses.
__device__ __forceinline__ unsigned magnitude(long long v) {
  const int h = static_cast<int>(v >> 32);
  return static_cast<unsigned>(h ^ (h >> 31));
}

struct Acc2 {  // (sum xh vh, sum xh vl + xl vh)
  long long h, m;
  __device__ __forceinline__ void add(int xl, int xh, int vl, int vh) {
    h += static_cast<long long>(xh) * vh;
    m += static_cast<long long>(xh) * vl;
    m += static_cast<long long>(xl) * vh;
  }
  __device__ __forceinline__ long long value() const { return h + (m >> 32); }
};

// v 2^k rounded to nearest (|v| < 2^62, the result a normal number or zero), on the integer pipes: three
// FP64 instructions per point would keep the FP64 pipe busy for a quarter of the kernel's time.
__device__ __forceinline__ double to_double(long long v, int k) {
  const long long s = v >> 63;
  const unsigned long long a = static_cast<unsigned long long>((v ^ s) - s);
  const uint32_t hi = static_cast<uint32_t>(a >> 32);
  const int lz = hi ? __clz(static_cast<int>(hi)) : 32 + __clz(static_cast<int>(static_cast<uint32_t>(a)));
  const unsigned long long m = ((a << (lz - 1)) + 512ull) >> 10;  // significand in bits 52..0 (2^53 when rounded up)
  const uint32_t h = static_cast<uint32_t>(m >> 32) + (static_cast<uint32_t>(1023 + 62 - (lz - 1) + k - 1) << 20);
  const uint32_t sign = static_cast<uint32_t>(static_cast<unsigned long long>(v) >> 32) & 0x80000000u;
  return a ? __hiloint2double(static_cast<int>(h | sign), static_cast<int>(static_cast<uint32_t>(m))) : 0.0;
}

// Fixed point is relative to the element's largest |u|: where only a few of an element's values come near it, the
// others lose bits that FP64 keeps, so such an element takes FP64 lines. A thread's largest value counts if it is
// within 2^kNear of its warp's and that within 2^kNearWarp of the element's (by exponent); fewer than a quarter of the threads
// with points: FP64. Relative 2-norm error of w over an element, CPU model of both, 2000 fields with spikes, decays and ridges:
// without this rule up to 3.5e-15 at N = 3, 4.9e-14 at N = 7, 1.8e-13 at N = 11 (FP64 lines 2e-16), with it at most 1.5e-15,
// 2.5e-15 and 3.3e-15, on average as FP64. Random fields have 2e-16 either way; in CG with a smooth or a random right-hand
// side 37% of the threads or more count in every element and iteration, with a point source a quarter is missed in the first
// 12% of them. A_L in us at 4.1M points where every element takes FP64 lines, k_ax in brackets: N = 3 294 (282), N = 5 417 (344), N = 6
// 412 (371), N = 7 371 (378), N = 9 595 (530), N = 10 558 (422), N = 11 570 (500); on the fly 414 (695), 522 (750), 543 (774), 462
// (719), 770 (941), 703 (735), 707 (841). The rule itself, and u kept for such elements: N = 3 344 -> 354 us at 16.8M points, N = 7
// 345 -> 335 and in CG 547 -> 554 an iteration, the other orders within 2%.
constexpr int kNear = 4, kNearWarp = 3;

// A warp's word on its values (or those of an element in it): the largest exponent above the number of threads within 2^kNear.
__device__ __forceinline__ unsigned near_word(unsigned top, unsigned most, unsigned lanes) {
  return (most & 0x7ff00000u) | __popc(__ballot_sync(0xffffffffu, (top >> 20) + kNear >= (most >> 20)) & lanes);
}

// `count` elements in FP64, as k_ax computes them (lines through the even/odd split of D). abc: the arrays A, B, C
// of ELEMS NP^3 doubles each in shared memory; A holds u, and w = A + B + C on return. G: the elements' fixed-point factors in
// shared memory, sg[q sg_step] the exponent of element q. Called by all threads after a barrier, ends with one.
template <int NP, int ELEMS>
__device__ __noinline__ void elements_fp64(const GllParam<NP, double>& tab, const int2* G, const int* __restrict__ sg,
                                           int sg_step, int count, double* abc) {
  constexpr int NP2 = NP * NP, P = NP2 * NP;
  double *A = abc, *B = A + ELEMS * P, *C = B + ELEMS * P;
  const int t = threadIdx.x, nt = blockDim.x, lines = count * NP2;
  auto line = [&](const EoMat<NP, double>& M, const double* src, double* dst, int q, int dir) {
    const int r = q % NP2, a = r % NP, b = r / NP;
    const int base = q / NP2 * P + (dir == 0 ? (a + b * NP) * NP : dir == 1 ? a + b * NP2 : r);
    const int step = dir == 0 ? 1 : dir == 1 ? NP : NP2;
    double in[NP], o[NP];
#pragma unroll
    for (int l = 0; l < NP; ++l) in[l] = src[base + l * step];
    eo_apply<NP, double>(M, in, o);
#pragma unroll
    for (int l = 0; l < NP; ++l) dst[base + l * step] = o[l];
  };
#pragma unroll 1
  for (int q = t; q < 2 * lines; q += nt) {
    const bool rows = q < lines;
    line(tab.Df, A, rows ? B : C, rows ? q : q - lines, rows ? 0 : 2);
  }
  __syncthreads();
#pragma unroll 1
  for (int q = t; q < lines; q += nt) line(tab.Df, A, A, q, 1);
  __syncthreads();
#pragma unroll 1
  for (int q = t; q < count * P; q += nt) {
    const int el = q / P, r = q % P, e = __ldg(sg + el * sg_step);
    const int c[3] = {fixed_row_scale(NP, r % NP), fixed_row_scale(NP, r / NP % NP), fixed_row_scale(NP, r / NP2)};
    double g[6];
#pragma unroll
    for (int m = 0; m < 6; ++m) {
      const int2 x = G[(el * 6 + m) * P + r];
      const long long v = static_cast<long long>(x.y) * 4294967296ll + x.x;
      const int k = -(e + c[m < 3 ? 0 : m < 5 ? 1 : 2] + c[m < 3 ? m : m < 5 ? m - 2 : 2]);
      // (to_double wants a normal result)
      g[m] = abs(e) < 900    ? to_double(v, k)
             : e > kSgFinite ? scalbn(static_cast<double>(v), k)
                             : __hiloint2double(0x7ff80000, 0);
    }
    const double ur = B[q], us = A[q], ut = C[q];
    B[q] = g[0] * ur + g[1] * us + g[2] * ut;
    A[q] = g[1] * ur + g[3] * us + g[4] * ut;
    C[q] = g[2] * ur + g[4] * us + g[5] * ut;
  }
  __syncthreads();
#pragma unroll 1
  for (int q = t; q < 3 * lines; q += nt) {
    const int dir = q / lines;
    double* v = dir == 0 ? B : dir == 1 ? A : C;
    line(tab.Dt, v, v, q - dir * lines, dir);
  }
  __syncthreads();
}

// On the fly: the row tables of one group's elements in shared memory, and the group's factors from
// them (k_geo_fixed.cuh). THREADS threads take kParts parts of every k-column, or points.
template <int NP, int ELEMS, int THREADS>
struct OtfGeometry {
  static constexpr int NP2 = NP * NP, P = NP2 * NP;
  static constexpr int kParts = THREADS / (ELEMS * NP2) > 1 ? THREADS / (ELEMS * NP2) : 1;
  // Point by point (each sets its column up again) where that takes fewer rounds of the block and measures faster:
  // A_L at 16M points by columns and by points, N = 6 (four and three rounds) 1.45 and 1.37 ms, N = 11 (six and five)
  // 1.50 and 1.46; but N = 10 (six and four) 1.78 and 1.83, and at the other orders the rounds are the same.
  static constexpr bool kByPoint = NP != 11 && (ELEMS * P + THREADS - 1) / THREADS < (NP + kParts - 1) / kParts;
  struct Tables {
    GeoEntry e[ELEMS][3][NP][3];
    GeoEntryT t[ELEMS][NP][3];
    GeoNodes<NP> n;
    int one;
  };
  static __device__ __forceinline__ int one_of(const Tables* s) {
    int one;
    asm volatile("ld.shared.b32 %0, [%1];" : "=r"(one) : "r"(smem_u32(&s->one)));
    return one;
  }
  static __device__ __forceinline__ void nodes(Tables* s, const GeoNodes<NP>& n) {
    if (threadIdx.x < NP) {
      s->n.x[threadIdx.x] = n.x[threadIdx.x];
      s->n.w[threadIdx.x] = n.w[threadIdx.x];
    }
    if (threadIdx.x == 0) s->one = 1;
  }
  static __device__ __forceinline__ void rows(Tables* s, const GeoElement* __restrict__ geo, int64_t e0, int count) {
    const int one = one_of(s);
    for (int q = threadIdx.x; q < 9 * NP * count; q += THREADS) {
      const int el = q / (9 * NP), d = q / (3 * NP) % 3, i = q / 3 % NP, c = q % 3;
      s->e[el][d][i][c] = geo_entry(geo[e0 + el], d, c, s->n.x[i], one, &s->t[el][i][c]);
    }
  }
  static __device__ __forceinline__ void columns(const Tables* s, const GeoElement* __restrict__ geo, int64_t e0, int count,
                                                 int2* sG) {
    const int one = one_of(s);
    auto column = [&](int el, int i, int j, int k0, int k1) {
      const GeoEntry *e_i = s->e[el][0][i], *e_j = s->e[el][1][j];
      const int down = __ldg(&geo[e0 + el].down), lz = __ldg(&geo[e0 + el].lz);
      const int up = __ldg(&geo[e0 + el].up) & 255, b = __ldg(&geo[e0 + el].up) >> 8;
      GeoColumn c;
      c.init(e_i, e_j, s->t[el][i], s->n.x[i], s->n.x[j], s->n.w[i], s->n.w[j], one);
      const int ci = fixed_row_scale(NP, i), cj = fixed_row_scale(NP, j);
      int2* out = sG + el * 6 * P + j * NP + i;
#pragma unroll 1
      for (int k = k0; k < k1; ++k) {
        const int ck = fixed_row_scale(NP, k);
        const int sh[6] = {b + cj + ck - ci, b + ck, b + cj, b + ci + ck - cj, b + ci, b + ci + cj - ck};
        c.point(e_i, e_j, s->e[el][2][k], s->n.x[k], s->n.w[k], down, lz, up, [&](int m, long long v) {
          const Fx x = fx_split(v >> sh[m]);
          out[m * P + k * NP2] = make_int2(x.l, x.h);
        });
      }
    };
    if constexpr (kByPoint) {
      for (int q = threadIdx.x; q < P * count; q += THREADS) {
        const int el = q / P, k = q % P / NP2;
        column(el, q % NP, q % NP2 / NP, k, k + 1);
      }
    } else {
      for (int q = threadIdx.x; q < NP2 * kParts * count; q += THREADS) {
        const int el = q / (NP2 * kParts), part = q / NP2 % kParts;
        column(el, q % NP2 % NP, q % NP2 / NP, part * NP / kParts, (part + 1) * NP / kParts);
      }
    }
  }
};
template <int NP>
GeoNodes<NP> make_geo_nodes(int N) {
  const GllTable& t = gll_table(N);
  int c[NP];
  for (int i = 0; i < NP; ++i) c[i] = fixed_row_scale(NP, i);
  const int sw = geo_weight_scale(t.w, c, NP);
  GeoNodes<NP> n{};
  for (int i = 0; i < NP; ++i) {
    n.x[i] = fx_split(std::llrint(std::ldexp(t.xi[i], 62)));
    n.w[i] = fx_split(std::llrint(std::ldexp(t.w[i], 62 + sw + c[i])));
  }
  return n;
}

template <int NP>
struct SliceShape {
  static constexpr int kW = slice_width(NP);   // an element takes kW of the block's 8 points per direction,
  static constexpr int kSub = 8 / kW;          // so a block holds kSub^3 elements at a time
  static constexpr int kElems = kSub * kSub * kSub;
  static_assert(kElems == ax_slice_elements(NP - 1), "elements per block");
  static constexpr int kPlanes = kSub > 1 ? 8 : NP;      // k-planes of the block that hold points
  static constexpr int kWarps = (kPlanes + 1) / 2;       // a warp takes two (two j-planes in the k contractions)
  static constexpr int kThreads = 32 * kWarps;
  static constexpr int kSlots = kSub == 2 ? 2 : kWarps;  // warps that share an element
  static constexpr int kPlane = 72;            // values per plane of 8 x 8 in shared memory: 8 of padding
  static constexpr int kDigit = 8 * kPlane;
  static constexpr unsigned kElemBytes = 48u * NP * NP * NP;
  static constexpr size_t kBytesG = (kElems * static_cast<size_t>(kElemBytes) + 127) / 128 * 128;
  static constexpr size_t kOffD = kBytesG;                         // digits [kSlices][8][72] FP16
  static constexpr size_t kOffX = kOffD + kSlices * kDigit * 2;    // exchange [8][72] 64-bit
  // (the digits and the exchange together also hold the three arrays of elements_fp64)
  static constexpr size_t kBytesDX = kSlices * kDigit * 2 + 8 * kPlane * 8, kBytes64 = 24ull * kElems * NP * NP * NP;
  static constexpr size_t kOffA = kOffD + (kBytes64 > kBytesDX ? kBytes64 : kBytesDX);  // A fragments [2][4][32] 16 bytes
  static constexpr size_t kOffB = kOffA + 2 * 4 * 32 * 16;         // B fragments [2][7][32] 8 bytes
  static constexpr size_t kOffC = kOffB + 2 * 7 * 32 * 8;          // Start
  static constexpr size_t kOffM = kOffC + 32;                      // maxima [3][kElems][kSlots]
  static constexpr size_t kOffBar = kOffM + (3 * kElems * kSlots * 4 + 7) / 8 * 8;
  static constexpr size_t kOffTab = (kOffBar + 8 + 15) / 16 * 16;  // on the fly: row tables
  static constexpr int kHolders = NP * ((NP + 1) / 2) * ((NP + 1) / 2);  // threads with points of one element
  static constexpr int kFew = (kHolders + 3) / 4;  // see kNear
  using Geometry = OtfGeometry<NP, kElems, kThreads>;
  static constexpr size_t bytes(bool otf) { return otf ? kOffTab + sizeof(typename Geometry::Tables) : kOffBar + 8; }
};

// OR or maximum of v over the lanes of the warp that hold points of one of the eight elements of a
// block: lane bit 0 counts pairs of points along i, bits 2-3 points along j (or k).
template <typename F>
__device__ __forceinline__ unsigned over_element(unsigned v, F&& op) {
  v = op(v, __shfl_xor_sync(0xffffffffu, v, 1));
  v = op(v, __shfl_xor_sync(0xffffffffu, v, 4));
  return op(v, __shfl_xor_sync(0xffffffffu, v, 8));
}

// A block takes a group of kElems elements as one 8 x 8 x 8 box of points (one element for NP > 4).
// Warp q holds the points of planes k = 2q and 2q + 1, lane (j = lane / 4, i = 2 (lane % 4) + {0, 1}), both
// of one element; lanes and planes beyond an element's points hold zeros. Phases of a group:
//   0  u (CG, fused_cg: the previous iteration's x += alpha p, p = M^-1 r + beta p) to registers; largest
//      exponent and how many threads come near it (kNear); digits of U to shared memory
//   1  k-lines (a warp takes j = 2q, 2q + 1): ut, exchanged through shared memory; i-rows and j-lines
//      of the own planes: ur, us stay in the lane that owns the point; largest magnitude
//   2  geometry; digits of vt to shared memory
//   3  digits of vr and vs in registers (vs transposed), D^T on i-rows and j-lines, then (after a
//      barrier) on k-lines, exchanged back; w
// The factors of the next group arrive by one TMA bulk copy during phase 3 and the next phase 0.
// OTF: the factors are rebuilt (OtfGeometry: row tables in phase 0, the factors before phase 1) instead of
// copied; three blocks per SM there (168 registers; N = 7 1% slower with four, N = 3 100 and 96 us at 1.3M points), four at N = 5, whose blocks of 96 threads have the registers (CG 2.19 ms with three, 2.13 with four).
template <int NP, bool CG, bool OTF>
__global__ void __launch_bounds__(SliceShape<NP>::kThreads, OTF && NP != 6 ? 3 : 4)
    k_ax_slice(const __grid_constant__ GllParam<NP, double> tab, const __grid_constant__ SliceTab<NP> sl,
               const __grid_constant__ GeoNodes<NP> nodes, int64_t E, const double* __restrict__ u,
               double* __restrict__ w, const int2* __restrict__ G, const int* __restrict__ gexp,
               const GeoElement* __restrict__ geo, const double* __restrict__ r, const double* __restrict__ minv,
               double* __restrict__ x, double* __restrict__ p, CgScalars* __restrict__ st,
               double* __restrict__ partials, int* __restrict__ err) {
  using S = SliceShape<NP>;
  constexpr int NP2 = NP * NP, P = NP2 * NP, PL = S::kPlane;
  extern __shared__ __align__(128) unsigned char smem[];
  int2* sG = reinterpret_cast<int2*>(smem);
  uint32_t* sD = reinterpret_cast<uint32_t*>(smem + S::kOffD);  // FP16 pairs
  double* abc = reinterpret_cast<double*>(smem + S::kOffD);     // elements_fp64, in place of sD and sX
  long long* sX = reinterpret_cast<long long*>(smem + S::kOffX);
  uint4* sA = reinterpret_cast<uint4*>(smem + S::kOffA);
  uint2* sB = reinterpret_cast<uint2*>(smem + S::kOffB);
  unsigned* sMax = reinterpret_cast<unsigned*>(smem + S::kOffM);  // of |u| (near_word); of ur and us; of ut
  uint64_t* bar = reinterpret_cast<uint64_t*>(smem + S::kOffBar);
  __shared__ double sRed[32];

  double beta = 0.0, alpha = 0.0;
  if constexpr (CG) {
    if (st->done) return;  // uniform over the grid: set by an earlier launch
    beta = st->beta;
    alpha = st->alpha;
  }
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int j = lane >> 2, i0 = 2 * (lane & 3), k0 = 2 * warp;
  // the group's element that holds the lane's points, and the one of its k-line values (k = lane / 4,
  // j = k0 + {0, 1})
  const int si = i0 / S::kW, sj = j / S::kW, sk = k0 / S::kW;
  const int own = si + S::kSub * (sj + S::kSub * sk), own_k = si + S::kSub * (sk + S::kSub * sj);
  const int slot = S::kSub == 1 ? warp : (warp & 1);
  const int li = i0 % S::kW, lj = j % S::kW, lk = k0 % S::kW;
  const int off = lk * NP2 + lj * NP + li;
  const int64_t n_groups = (E + S::kElems - 1) / S::kElems;
  auto group_size = [&](int64_t grp) {
    const int64_t left = E - grp * S::kElems;
    return static_cast<unsigned>(left < S::kElems ? left : S::kElems);
  };
  auto load_factors = [&](int64_t grp) {  // one thread
    const unsigned bytes = S::kElemBytes * group_size(grp);
    fence_proxy_async();
    mbar_expect_tx(bar, bytes);
    tma_load_1d(sG, G + grp * S::kElems * 6 * P, bytes, bar);
  };
  typename S::Geometry::Tables* tables = reinterpret_cast<typename S::Geometry::Tables*>(smem + S::kOffTab);
  if constexpr (OTF) {
    S::Geometry::nodes(tables, nodes);
  } else if (threadIdx.x == 0) {
    mbar_init(bar, 1);
    load_factors(blockIdx.x);
  }
  for (int q = threadIdx.x; q < kSlices * S::kDigit / 2; q += S::kThreads) sD[q] = 0u;
  if (threadIdx.x < 8) reinterpret_cast<float*>(smem + S::kOffC)[threadIdx.x] = threadIdx.x < 6 ? kMagic : 0.f;
  if (warp < 2) {  // fragment tables of D (warp 0) and D^T (warp 1)
    uint32_t d[kSlices + 3];  // d[0] = 0, d[1 + t] = digit t, then zeros
    d[0] = d[kSlices + 1] = d[kSlices + 2] = 0u;
#pragma unroll
    for (int t = 0; t < kSlices; ++t) d[1 + t] = sl.d[warp][t][lane >> 2][lane & 3];
#pragma unroll
    for (int o = 0; o <= 6; ++o) {
      sB[(warp * 7 + o) * 32 + lane] = make_uint2(d[1 + o], d[o]);
      if (o % 2 == 0) sA[(warp * 4 + o / 2) * 32 + lane] = make_uint4(d[1 + o], d[2 + o], d[o], d[1 + o]);
    }
  }
  const uint32_t sD32 = smem_u32(sD);
  const int mi = lane >> 3, row = lane & 7;  // ldmatrix: matrix and row this lane addresses
  // k-lines of planes j = k0, k0 + 1: matrices (digit s, j0), (s + 1, j0), (s, j1), (s + 1, j1), rows k
  const uint32_t ldK = sD32 + 2u * ((mi & 1) * S::kDigit + row * PL + (k0 + (mi >> 1)) * 8);
  // i-rows: (s, k0), (s, k1), (s + 1, k0), (s + 1, k1), rows j
  const uint32_t ldI = sD32 + 2u * ((mi >> 1) * S::kDigit + (k0 + (mi & 1)) * PL + row * 8);
  // j-lines: (s, k0), (s + 1, k0), (s, k1), (s + 1, k1), rows j, transposed on load
  const uint32_t ldJ = sD32 + 2u * ((mi & 1) * S::kDigit + (k0 + (mi >> 1)) * PL + row * 8);
  const uint4* fAf = sA + lane;
  const uint4* fAt = sA + 4 * 32 + lane;
  const uint2* fBf = sB + lane;
  const uint2* fBt = sB + 7 * 32 + lane;
  auto by_max = [](unsigned a, unsigned b) { return a > b ? a : b; };
  auto by_or = [](unsigned a, unsigned b) { return a | b; };
  // one value per element and warp into row a of sMax, combined over the warps after a barrier
  auto put = [&](int a, int elem, unsigned m) { sMax[(a * S::kElems + elem) * S::kSlots + slot] = m; };
  auto get = [&](int a, int q) { return sMax[(a * S::kElems + own) * S::kSlots + q]; };
  double dot = 0.0;
  unsigned parity = 0;
  __syncthreads();
  Start s0;
  lds_quad(s0.m, smem_u32(smem + S::kOffC));
  lds_quad(s0.h, smem_u32(smem + S::kOffC) + 16);

  for (int64_t grp = blockIdx.x; grp < n_groups; grp += gridDim.x) {
    const int64_t e0 = grp * S::kElems, e = e0 + own, base = e * P + off;
    const bool more = grp + gridDim.x < n_groups;
    bool in[2][2];
#pragma unroll
    for (int t = 0; t < 2; ++t)
#pragma unroll
      for (int x = 0; x < 2; ++x)
        in[t][x] = (S::kElems == 1 || e < E) && (NP == S::kW || (lk + t < NP && lj < NP && li + x < NP));
    // the lane's pair of plane k0 + t (16-byte aligned where NP is even)
    auto load2 = [&](const double* __restrict__ src, int t, double (&o)[2]) {
      const double* s = src + base + t * NP2;
      o[0] = o[1] = 0.0;
      if constexpr (NP % 2 == 0) {
        if (in[t][0]) {
          const double2 a = *reinterpret_cast<const double2*>(s);
          o[0] = a.x;
          o[1] = a.y;
        }
      } else {
        if (in[t][0]) o[0] = s[0];
        if (in[t][1]) o[1] = s[1];
      }
    };
    auto store2 = [&](double* __restrict__ dst, int t, const double (&o)[2]) {
      double* s = dst + base + t * NP2;
      if constexpr (NP % 2 == 0) {
        if (in[t][0]) *reinterpret_cast<double2*>(s) = make_double2(o[0], o[1]);
      } else {
        if (in[t][0]) s[0] = o[0];
        if (in[t][1]) s[1] = o[1];
      }
    };
    // phase 0
    double v[2][2];
    if constexpr (CG) {
      double rv[2][2], pv[2][2], xv[2][2], mv[2][2];
#pragma unroll
      for (int t = 0; t < 2; ++t) {
        load2(r, t, rv[t]);
        load2(p, t, pv[t]);
        load2(x, t, xv[t]);
        if (minv) load2(minv, t, mv[t]);
      }
#pragma unroll
      for (int t = 0; t < 2; ++t) {
#pragma unroll
        for (int q = 0; q < 2; ++q) {
          v[t][q] = fma(beta, pv[t][q], minv ? mv[t][q] * rv[t][q] : rv[t][q]);
          xv[t][q] = fma(alpha, pv[t][q], xv[t][q]);
        }
        store2(p, t, v[t]);
        store2(x, t, xv[t]);
      }
    } else {
#pragma unroll
      for (int t = 0; t < 2; ++t) load2(u, t, v[t]);
    }
    if constexpr (OTF) S::Geometry::rows(tables, geo, e0, group_size(grp));
    const int sg = S::kElems == 1 || e < E ? __ldg(OTF ? &geo[e].sg : gexp + e) : 0;
    unsigned mh = 0;
#pragma unroll
    for (int t = 0; t < 2; ++t)
#pragma unroll
      for (int x = 0; x < 2; ++x) mh = max(mh, static_cast<unsigned>(__double2hiint(v[t][x])) & 0x7fffffffu);
    const unsigned top = mh;
    if constexpr (S::kSub == 1)
      mh = near_word(top, __reduce_max_sync(0xffffffffu, mh), 0xffffffffu);
    else
      mh = near_word(top, over_element(mh, by_max), 0x3333u << (lane & 18));
    put(0, own, mh);
    __syncthreads();
    int emax;
    unsigned n;  // threads that count
    if constexpr (S::kSub == 1) {
      const unsigned all = lane < S::kSlots ? sMax[lane] : 0u;
      emax = static_cast<int>(__reduce_max_sync(0xffffffffu, all) >> 20);
      n = __reduce_add_sync(0xffffffffu, static_cast<int>(all >> 20) + kNearWarp >= emax ? all & 63u : 0u);
    } else {
      const unsigned m0 = get(0, 0), m1 = get(0, 1);
      emax = static_cast<int>(by_max(m0, m1) >> 20);
      n = (static_cast<int>(m0 >> 20) + kNearWarp >= emax ? m0 & 63u : 0u) +
          (static_cast<int>(m1 >> 20) + kNearWarp >= emax ? m1 & 63u : 0u);
    }
    bool general = emax == 2047 || abs(1080 - emax + sg) > 700 || n < S::kFew;
    if (emax < 64) {  // zero, or too small for fixed point
      general = v[0][0] != 0.0 || v[0][1] != 0.0 || v[1][0] != 0.0 || v[1][1] != 0.0 || sg < kSgFinite;
      emax = 1080;
    }
    if (threadIdx.x == 0 && more) {  // the next group's vectors into L2
      if constexpr (OTF)
        l2_prefetch(geo + e0 + static_cast<int64_t>(gridDim.x) * S::kElems,
                    static_cast<unsigned>(sizeof(GeoElement)) * group_size(grp + gridDim.x));
      if constexpr (P % 2 == 0) {
        const int64_t at = (e0 + static_cast<int64_t>(gridDim.x) * S::kElems) * P;
        const unsigned bytes = 8u * P * group_size(grp + gridDim.x);
        if constexpr (CG) {
          l2_prefetch(r + at, bytes);
          l2_prefetch(p + at, bytes);
          l2_prefetch(x + at, bytes);
          if (minv) l2_prefetch(minv + at, bytes);
        } else {
          l2_prefetch(u + at, bytes);
        }
      }
    }
#pragma unroll
    for (int t = 0; t < 2; ++t) {
      uint32_t d[kSlices];
      digit_pairs(to_fixed(v[t][0], emax), to_fixed(v[t][1], emax), d);
      if (S::kPlanes % 2 == 0 || k0 + t < S::kPlanes) {
#pragma unroll
        for (int s = 0; s < kSlices; ++s) sD[(s * S::kDigit + (k0 + t) * PL) / 2 + lane] = d[s];
      }
    }
    if constexpr (OTF) S::Geometry::columns(tables, geo, e0, group_size(grp), sG);
    const bool slow = __syncthreads_or(general);  // for the whole group

    // phase 1
    long long vr[2][2], vs[2][2];
    if (!slow) {
      unsigned m = 0;
      {
        uint32_t b[2][kSlices];
#pragma unroll
        for (int s = 0; s < kSlices; s += 2) ldsm4t(b[0][s], b[0][s + 1], b[1][s], b[1][s + 1], ldK + 2u * s * S::kDigit);
#pragma unroll
        for (int t = 0; t < 2; ++t) {
          long long r[2];
          contract_lines(s0, fAf, b[t], r);
          *reinterpret_cast<longlong2*>(sX + j * PL + (k0 + t) * 8 + i0) = make_longlong2(r[0], r[1]);  // k = lane / 4
          m |= magnitude(r[0]) | magnitude(r[1]);
        }
      }
      if constexpr (S::kSub > 1) {
        put(2, own_k, over_element(m, by_or));
        m = 0;
      }
      {
        uint4 a[3];
#pragma unroll
        for (int s = 0; s < 3; ++s) {
          uint32_t r[4];
          ldsm4(r, ldI + 4u * s * S::kDigit);
          a[s] = make_uint4(r[0], r[1], r[2], r[3]);
        }
        contract_rows(s0, fBf, a, vr);
      }
      {
        uint32_t b[2][kSlices];
#pragma unroll
        for (int s = 0; s < kSlices; s += 2) ldsm4t(b[0][s], b[0][s + 1], b[1][s], b[1][s + 1], ldJ + 2u * s * S::kDigit);
#pragma unroll
        for (int t = 0; t < 2; ++t) contract_lines(s0, fAf, b[t], vs[t]);
      }
#pragma unroll
      for (int t = 0; t < 2; ++t)
#pragma unroll
        for (int x = 0; x < 2; ++x) m |= magnitude(vr[t][x]) | magnitude(vs[t][x]);
      if constexpr (S::kSub == 1)
        m = __reduce_or_sync(0xffffffffu, m);
      else
        m = over_element(m, by_or);
      put(1, own, m);
    } else {  // u over the digits and the exchange
#pragma unroll
      for (int t = 0; t < 2; ++t)
#pragma unroll
        for (int x = 0; x < 2; ++x)
          if (in[t][x]) abc[own * P + t * NP2 + off + x] = v[t][x];
    }
    bool ok = true;
    if constexpr (!OTF) ok = mbar_wait_bounded(bar, parity);  // this group's factors
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

    double wv[2][2];
    if (!slow) {
      // phase 2: geometry on V 2^lv, |V| 2^lv < 2^61
      unsigned m = 0;
#pragma unroll
      for (int q = 0; q < S::kSlots; ++q) m |= S::kSub > 1 ? get(1, q) | get(2, q) : get(1, q);
      const int lv = __clz(m) - 3;
      long long vt[2][2];
#pragma unroll
      for (int t = 0; t < 2; ++t) {
        const longlong2 ut = *reinterpret_cast<const longlong2*>(sX + (k0 + t) * PL + j * 8 + i0);
        vt[t][0] = ut.x;
        vt[t][1] = ut.y;
        int2 g[6][2];
#pragma unroll
        for (int q = 0; q < 6; ++q) {
          const int2* src = sG + (own * 6 + q) * P + t * NP2 + off;
          if constexpr (NP == S::kW) {  // beyond the mesh's last element: what was there, times V = 0
            const int4 a = *reinterpret_cast<const int4*>(src);
            g[q][0] = make_int2(a.x, a.y);
            g[q][1] = make_int2(a.z, a.w);
          } else {
#pragma unroll
            for (int x = 0; x < 2; ++x) g[q][x] = in[t][x] ? src[x] : make_int2(0, 0);
          }
        }
#pragma unroll
        for (int x = 0; x < 2; ++x) {
          const long long ar = vr[t][x] << lv, as = vs[t][x] << lv, at = vt[t][x] << lv;
          const int rl = low_half(ar), rh = high_half(ar), sl_ = low_half(as), sh = high_half(as), tl = low_half(at),
                    th = high_half(at);
          auto row3 = [&](const int2& a, const int2& b, const int2& c) {
            Acc2 s{0, 0};
            s.add(a.x, a.y, rl, rh);
            s.add(b.x, b.y, sl_, sh);
            s.add(c.x, c.y, tl, th);
            return s.value();
          };
          vr[t][x] = row3(g[0][x], g[1][x], g[2][x]);
          vs[t][x] = row3(g[1][x], g[3][x], g[4][x]);
          vt[t][x] = row3(g[2][x], g[4][x], g[5][x]);
        }
      }
#pragma unroll
      for (int t = 0; t < 2; ++t) {
        uint32_t d[kSlices];
        digit_pairs(vt[t][0], vt[t][1], d);
        if (S::kPlanes % 2 == 0 || k0 + t < S::kPlanes) {
#pragma unroll
          for (int s = 0; s < kSlices; ++s) sD[(s * S::kDigit + (k0 + t) * PL) / 2 + lane] = d[s];
        }
      }
      // phase 3
      long long sum[2][2];
      {
        uint32_t d[2][kSlices];
#pragma unroll
        for (int t = 0; t < 2; ++t) digit_pairs(vr[t][0], vr[t][1], d[t]);
        uint4 a[3];
#pragma unroll
        for (int s = 0; s < 3; ++s) a[s] = make_uint4(d[0][2 * s], d[1][2 * s], d[0][2 * s + 1], d[1][2 * s + 1]);
        contract_rows(s0, fBt, a, sum);
      }
#pragma unroll
      for (int t = 0; t < 2; ++t) {
        uint32_t d[kSlices];
        digit_pairs(vs[t][0], vs[t][1], d);
#pragma unroll
        for (int s = 0; s < kSlices; ++s) d[s] = transpose8x8(d[s]);
        long long r[2];
        contract_lines(s0, fAt, d, r);
        sum[t][0] += r[0];
        sum[t][1] += r[1];
      }
      __syncthreads();  // the digits of vt; the factors are consumed
      if (!OTF && threadIdx.x == 0 && more) load_factors(grp + gridDim.x);
      {
        uint32_t b[2][kSlices];
#pragma unroll
        for (int s = 0; s < kSlices; s += 2) ldsm4t(b[0][s], b[0][s + 1], b[1][s], b[1][s + 1], ldK + 2u * s * S::kDigit);
#pragma unroll
        for (int t = 0; t < 2; ++t) {
          long long r[2];
          contract_lines(s0, fAt, b[t], r);
          *reinterpret_cast<longlong2*>(sX + j * PL + (k0 + t) * 8 + i0) = make_longlong2(r[0], r[1]);
        }
      }
      __syncthreads();
      // w = sum 2^-sc: u 2^(1080 - emax), D 2^e / 2^57 twice, V 2^lv, G 2^sg / 2^64
      const int scale = -(1080 - emax + lv + sg - 64 + 2 * (sl.e - 57));
#pragma unroll
      for (int t = 0; t < 2; ++t) {
        const longlong2 r = *reinterpret_cast<const longlong2*>(sX + (k0 + t) * PL + j * 8 + i0);
        wv[t][0] = to_double(sum[t][0] + r.x, scale);
        wv[t][1] = to_double(sum[t][1] + r.y, scale);
      }
    } else {
      elements_fp64<NP, S::kElems>(tab, sG, OTF ? &geo[e0].sg : gexp + e0, OTF ? static_cast<int>(sizeof(GeoElement) / 4) : 1,
                                   static_cast<int>(group_size(grp)), abc);
#pragma unroll
      for (int t = 0; t < 2; ++t)
#pragma unroll
        for (int x = 0; x < 2; ++x) {
          const double* s = abc + own * P + t * NP2 + off + x;
          wv[t][x] = in[t][x] ? s[0] + s[S::kElems * P] + s[2 * S::kElems * P] : 0.0;
        }
      __syncthreads();
      for (int q = threadIdx.x; q < kSlices * S::kDigit / 2; q += S::kThreads) sD[q] = 0u;  // beyond the points, as at the start
      if (!OTF && threadIdx.x == 0 && more) load_factors(grp + gridDim.x);
    }
    if constexpr (CG) {
#pragma unroll
      for (int t = 0; t < 2; ++t)
#pragma unroll
        for (int x = 0; x < 2; ++x)
          if (in[t][x]) {
            w[e * P + cg_pos(NP, li + x, lj, lk + t)] = wv[t][x];
            dot = fma(v[t][x], wv[t][x], dot);
          }
    } else {
#pragma unroll
      for (int t = 0; t < 2; ++t) store2(w, t, wv[t]);
    }
  }
  if constexpr (CG) {
    const double s = block_sum(dot, sRed);
    if (threadIdx.x == 0) partials[blockIdx.x] = s;
  }
}

template <int NP, bool CG, bool OTF>
sem_status launch_slice_t(int N, const AxLaunch& a, cudaStream_t s) {
  using S = SliceShape<NP>;
  static const int max_blocks = [] {
    cudaFuncSetAttribute(k_ax_slice<NP, CG, OTF>, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(S::bytes(OTF)));
    int dev = 0, sms = 0, per_sm = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_ax_slice<NP, CG, OTF>, S::kThreads, S::bytes(OTF));
    return (per_sm > 0 ? per_sm : 1) * (sms > 0 ? sms : 1);
  }();
  static const SliceTab<NP> sl = make_slice_tab<NP>(N);
  static const GllParam<NP, double> tab = make_gll_param<NP, double>(N);
  static const GeoNodes<NP> nodes = make_geo_nodes<NP>(N);
  const int64_t groups = (a.E + S::kElems - 1) / S::kElems;
  int grid = max_blocks < kRedMax ? max_blocks : kRedMax;
  if (groups < grid) grid = static_cast<int>(groups);
  if (a.grid_out) *a.grid_out = grid;
  k_ax_slice<NP, CG, OTF><<<grid, S::kThreads, S::bytes(OTF), s>>>(
      tab, sl, nodes, a.E, static_cast<const double*>(a.u), static_cast<double*>(a.w), static_cast<const int2*>(a.G),
      a.gexp, a.geo, static_cast<const double*>(a.r), static_cast<const double*>(a.minv), static_cast<double*>(a.x),
      static_cast<double*>(a.p), a.st, a.partials, a.err);
  count_launch();
  SEM_CUDA_TRY(cudaGetLastError());
  return SEM_OK;
}

}  // namespace
}  // namespace sem
