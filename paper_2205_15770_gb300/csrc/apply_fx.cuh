// 3D cell kernel of Q2-Q1 in FP64 by 64-bit fixed-point arithmetic (launch shape 5 for double, k = 2):
// one thread per (cell, velocity component, z plane of the cell).  Same operator as the other cell
// kernels (paper Sec. 3.1: K x = sum_tau P_tau K_tau P_tau^T x by sum factorisation; Sec. 2 forms
// a(u,v) = mu grad u : grad v + gamma rho u.v and b(v,q) = -q div v).
//
// Why integers: this GPU issues 1.7 FP64 multiply-adds per SM and clock, but 50 of 32 x 32 + 64 bit
// integer ones and 60 of the other integer operations (a probe kernel of independent chains, 64
// warps per SM), and the floating-point cell kernel kept the FP64 pipe 85 % busy.  The product of
// two 62-bit numbers takes three integer multiply-adds and one addition (FxInt::mad).
//
// Why a plane per thread: the whole 27-node tensor in one thread is a straight line of 10,000
// instructions, which starved on instruction fetch (5.1 of 10 stall cycles an issue) at 255
// registers; a plane is 2,000 at about half the registers, and gives small levels three times the threads.
// A warp holds 10 cells of one component, lane = z * 10 + cell; the z contractions exchange planes by
// shuffles, x and y stay in registers.
//
// 1D tables of Q2 at the Gauss points 1/2 -+ r, 1/2 (r = sqrt(0.15)), node values a, b, c:
//   values      q0 = (0.3 + r) a + 0.4 b + (0.3 - r) c, q1 = b, q2 mirrored
//   derivatives 2r d/dx = (-3, 4, -1), (-1, 0, 1), (1, -4, 3) times (q0, q1, q2): whole numbers
//   pressure    q0, q2 = (p0 + p1) / 2 +- r (p0 - p1), q1 = (p0 + p1) / 2
// The factors 1 / (2r) are folded into the coefficients.  Along z a thread forms its own Gauss value
// and derivative from the three node planes; whole parts of the table are added, not multiplied, which
// keeps every table entry below 1/2.
//
// Ranges, for any input: a thread's velocity values are integers times a common power of two, the largest of
// the cell and component in [2^57, 2^58].  Gauss values are at most 2^59 (rows of S sum to 1.175 in absolute
// value), scaled derivatives 6.7 times the nodal values, 2^60.8; the x and y fluxes of A together
// 2^58.8 (rows of G, 2^62), each of B^T's 2^57 (pressure integers 2^59, columns of C 2^62); test sums of a plane 2^62.6, an eighth of them
// enters the transposed interpolation, whose sums stay below 2^62.5.  Sums of three products stay below 2^63 in
// both words.  Each rounding is to nearest at 2^-53 to 2^-58 of the stage's bound, where floating point rounds
// every operation, and the coefficients are formed from 106 bits: measured against extended precision on six meshes the
// operator's error is 0.10-0.37 of the FP64 column kernel's on random vectors, 0.15-0.62 on smooth ones and 0.19-0.49
// under large pressures (tests/test_gpu_fixed_point.py asserts that it is no larger).  One rounding to FP64 before the
// scatter.
//
// Measured (us, floating-point column kernel -> this kernel): 32^3 trilinear K 348 -> 97, A 264 -> 62, B^T 136 ->
// 36, B 146 -> 32; 32^3 Cartesian K 401 -> 80, A 327 -> 52; 16^3 trilinear K 61 -> 19; 8^3 K 23 -> 11.  Bound by
// the instruction chains of 12 resident warps per SM (168 registers): issue 38 % busy, most stalls fixed latencies.
//
// Warps with a value that is not finite, or whose largest is outside 2^-850 .. 2^850, take the same
// steps in floating point (FxDbl): infinities and NaN spread as they do there.
#pragma once
#include <algorithm>
#include <cmath>
#include <type_traits>

#include "common.cuh"
#include "host_tables.h"
#include "vec.cuh"

namespace smf {

typedef long long i64;

constexpr int kFxCells = 10;   // cells per warp
constexpr int kFxThreads = 96;  // a CTA is the three components of one group of 10 cells
// Stored coefficients of a level, int2 entries: [group of 10 cells] times a block of G 00 01 02 11 12 22 and W and a
// block of C (column c at 3 c), each [y, x point][field][lane], so that a launch copies what it needs of a group as one
// or two contiguous pieces; then two scales per cell.
constexpr int kFxG = 7, kFxC = 9;
__host__ __device__ inline long long fx_group_entries() { return 9ll * (kFxG + kFxC) * 32; }
__host__ __device__ inline long long fx_entries(long long cells) {
  return (cells + kFxCells - 1) / kFxCells * fx_group_entries() + cells;
}

struct Dig {  // h 2^32 + l, l signed
  int h, l;
};
__host__ __device__ __forceinline__ Dig fx_split(i64 v) {
  const int l = (int)v;
  return {(int)(v >> 32) + (int)((unsigned)l >> 31), l};
}
// a b + c in one instruction (written in C++ the compiler mixes the products with the splitting above:
// three times the instructions)
__device__ __forceinline__ i64 fx_wide(int a, int b, i64 c) {
  i64 r;
  asm("mad.wide.s32 %0, %1, %2, %3;" : "=l"(r) : "r"(a), "r"(b), "l"(c));
  return r;
}

template <int B>
__device__ __forceinline__ i64 fx_wide_imm(int a, i64 c) {
  i64 r;
  asm("mad.wide.s32 %0, %1, %2, %3;" : "=l"(r) : "r"(a), "n"(B), "l"(c));
  return r;
}
constexpr int kFxWUp = 3;    // W's digits stand for 2^-kFxWUp of its scale (FxInt::value_up)
constexpr int kFxTDown = 3;  // integers: places the test sums are shifted down before the transposed interpolation

template <int H, int L>
struct FxTab {};  // the constant (H 2^32 + L) / 2^64

struct FxInt {
  typedef i64 V;
  typedef Dig C;
  static constexpr bool SPLIT = true;  // whole parts of table entries are added apart (entries stay below 1/2)
  static __device__ __forceinline__ C tab(int h, int l) { return {h, l}; }
  static __device__ __forceinline__ V zero() { return 0; }
  // base + sum of c v / 2^64, rounded to nearest: rounding down would add up over the cells (the product of
  // the two low words, below one unit and of either sign, is left out)
  static constexpr i64 HALF = 1ll << 31;
  struct Sum {
    i64 hi, mid;
  };
  static __device__ __forceinline__ Sum start(V base, C c, V v) {
    const Dig d = fx_split(v);
    return {fx_wide(d.h, c.h, base), fx_wide(d.h, c.l, fx_wide(d.l, c.h, HALF))};
  }
  static __device__ __forceinline__ void add(Sum &s, C c, V v) {
    const Dig d = fx_split(v);
    s.hi = fx_wide(d.h, c.h, s.hi);
    s.mid = fx_wide(d.h, c.l, s.mid);
    s.mid = fx_wide(d.l, c.h, s.mid);
  }
  template <int H, int L>
  static __device__ __forceinline__ Sum start(V base, FxTab<H, L>, V v) {
    const Dig d = fx_split(v);
    return {fx_wide_imm<H>(d.h, base), fx_wide_imm<L>(d.h, fx_wide_imm<H>(d.l, HALF))};
  }
  template <int H, int L>
  static __device__ __forceinline__ void add(Sum &s, FxTab<H, L>, V v) {
    const Dig d = fx_split(v);
    s.hi = fx_wide_imm<H>(d.h, s.hi);
    s.mid = fx_wide_imm<L>(d.h, s.mid);
    s.mid = fx_wide_imm<H>(d.l, s.mid);
  }
  static __device__ __forceinline__ V value(const Sum &s) { return fx_wide_imm<1>((int)(s.mid >> 32), s.hi); }
  // 2^N times the sum, its last places from the fraction
  template <int N>
  static __device__ __forceinline__ V value_up(const Sum &s) {
    return (s.hi << N) + ((s.mid + ((1ll << (31 - N)) - HALF)) >> (32 - N));
  }
  template <int N>
  static __device__ __forceinline__ V down(V v) {  // v / 2^N, halves to even
    return (v + ((1 << (N - 1)) - 1) + ((v >> N) & 1)) >> N;
  }
  static __device__ __forceinline__ V half(V v) { return down<1>(v); }
  static __device__ __forceinline__ V tdown(V v) { return down<kFxTDown>(v); }
  static __device__ __forceinline__ V down_by(V v, int n) { return v >> n; }  // n large: the lost part is below the other term's rounding
};
template <typename T>
struct FxFloat {
  typedef T V;
  typedef T C;
  static constexpr bool SPLIT = false;
  static __device__ __forceinline__ C tab(int h, int l) { return (T)(h * 0x1p-32 + l * 0x1p-64); }
  static __device__ __forceinline__ V zero() { return T(0); }
  struct Sum {
    T s;
  };
  static __device__ __forceinline__ Sum start(V base, C c, V v) { return {base + c * v}; }
  static __device__ __forceinline__ void add(Sum &s, C c, V v) { s.s += c * v; }
  template <int H, int L>
  static __device__ __forceinline__ Sum start(V base, FxTab<H, L>, V v) {
    return {base + (T)(H * 0x1p-32 + L * 0x1p-64) * v};
  }
  template <int H, int L>
  static __device__ __forceinline__ void add(Sum &s, FxTab<H, L>, V v) {
    s.s += (T)(H * 0x1p-32 + L * 0x1p-64) * v;
  }
  static __device__ __forceinline__ V value(const Sum &s) { return s.s; }
  template <int N>
  static __device__ __forceinline__ V value_up(const Sum &s) {
    return s.s;
  }
  static __device__ __forceinline__ V half(V v) { return T(0.5) * v; }
  static __device__ __forceinline__ V tdown(V v) { return v; }
  static __device__ __forceinline__ V down_by(V v, int) { return v; }
};
typedef FxFloat<double> FxDbl;
typedef FxFloat<float> FxFlt;
// Table entries (times 2^64 as digits).
using FxTS00M = FxTab<-1343043426, -896144430>;     // 0.3 + r - 1 (the unit part is the base of the sum)
using FxTS01 = FxTab<1717986918, 1717986918>;    // 0.4
using FxTS02 = FxTab<-374943492, -821842488>;             // 0.3 - r
using FxTR = FxTab<1663433681, -37150971>;               // r

// node values -> Gauss values along one line in registers (the middle value is the middle node's)
template <typename P>
__device__ __forceinline__ void fx_interp(typename P::V &a, const typename P::V &b, typename P::V &c) {
  typename P::Sum q0 = P::start(a, FxTS00M{}, a), q2 = P::start(c, FxTS00M{}, c);
  P::add(q0, FxTS01{}, b);
  P::add(q2, FxTS01{}, b);
  P::add(q0, FxTS02{}, c);
  P::add(q2, FxTS02{}, a);
  a = P::value(q0);
  c = P::value(q2);
}
// its transpose
template <typename P>
__device__ __forceinline__ void fx_interp_t(typename P::V &a, typename P::V &b, typename P::V &c) {
  b = P::value(P::start(b, FxTS01{}, a + c));
  typename P::Sum y0 = P::start(a, FxTS00M{}, a), y2 = P::start(c, FxTS00M{}, c);
  P::add(y0, FxTS02{}, c);
  P::add(y2, FxTS02{}, a);
  a = P::value(y0);
  c = P::value(y2);
}
// pressure: two node values -> three Gauss values, and the transpose
template <typename P>
__device__ __forceinline__ void fx_pre(typename P::V p0, typename P::V p1, typename P::V (&q)[3]) {
  const typename P::V m = P::half(p0 + p1), d = P::value(P::start(P::zero(), FxTR{}, p0 - p1));
  q[0] = m + d;
  q[1] = m;
  q[2] = m - d;
}
template <typename P>
__device__ __forceinline__ void fx_pre_t(typename P::V q0, typename P::V q1, typename P::V q2, typename P::V &p0,
                                         typename P::V &p1) {
  const typename P::V e = P::half(q0 + q1 + q2), o = P::value(P::start(P::zero(), FxTR{}, q0 - q2));
  p0 = e + o;
  p1 = e - o;
}

// ---- doubles in and out: on the FP64 pipe, which the integer work leaves idle ----------------------------
__device__ __forceinline__ double fx_pow2(int e) { return __hiloint2double((1023 + e) << 20, 0); }  // |e| <= 1022
// digits of x 2^-e (|x| 2^-e <= 2^60; scale = 2^-e), and the value they stand for
__host__ __device__ inline Dig fx_coef(double x, double scale) { return fx_split((i64)rint(x * scale)); }
__device__ __forceinline__ double fx_coef_value(Dig d, int e) { return ldexp(d.h * 0x1p32 + d.l, e); }
// smallest e with x < 2^e (0 has a very small one)
__host__ __device__ inline int fx_exp(double x) { return x > 0.0 ? ilogb(x) + 1 : -4000; }
// Scales of a cell's coefficients: the x and y rows of G together, and its z row, sum to at most 2^62 in absolute
// value (only x and y fluxes add up in a plane's test sums), W (stored 2^-kFxWUp of
// its scale, FxInt::value_up) to 2^62; columns of C to 2^62.
__host__ __device__ inline int fx_scale_g(double xy, double z, double w) {
  const int a = fx_exp(xy > z ? xy : z) - 62, b = fx_exp(w) - 62 - kFxWUp;
  return a > b ? a : b;
}
__host__ __device__ inline int fx_scale_c(double cols) { return fx_exp(cols) - 62; }

constexpr double kFxAlpha = 1.2909944487358056;   // 1 / (2r)
constexpr double kFxAlpha2 = 1.6666666666666667;  // its square

// Cartesian levels: the coefficients of every weight class (number of middle points among x, y and z; the
// tensor Gauss weight is (5/18)^(3-m) (8/18)^m), formed on the host at the launch.  Cells with their own
// viscosity scale gd themselves.
__host__ __device__ constexpr double fx_weight(int m) {
  return m == 0 ? 125.0 / 5832.0 : (m == 1 ? 200.0 / 5832.0 : (m == 2 ? 320.0 / 5832.0 : 512.0 / 5832.0));
}
struct FxCart {
  int2 g[3][4], w[4], c[3][4];
  double gd[3], wd, cd[3];  // without weight; gd without the viscosity
  double xy, zz, wtop;      // row sums of gd and wd times the largest weight
  int eg, ec;
};
inline FxCart fx_cart(const LevelDesc<double> &L) {
  FxCart K{};
  const double *h = L.h;
  const double a2 = kFxAlpha2;
  K.gd[0] = a2 * h[1] * h[2] / h[0];
  K.gd[1] = a2 * h[0] * h[2] / h[1];
  K.gd[2] = a2 * h[0] * h[1] / h[2];
  K.wd = L.gamma_rho * h[0] * h[1] * h[2];
  K.cd[0] = kFxAlpha * h[1] * h[2];
  K.cd[1] = kFxAlpha * h[0] * h[2];
  K.cd[2] = kFxAlpha * h[0] * h[1];
  K.xy = (K.gd[0] + K.gd[1]) * fx_weight(3);
  K.zz = K.gd[2] * fx_weight(3);
  K.wtop = K.wd * fx_weight(3);
  K.eg = fx_scale_g(K.xy * L.mu, K.zz * L.mu, K.wtop);
  K.ec = fx_scale_c(std::max(K.cd[0], std::max(K.cd[1], K.cd[2])) * fx_weight(3));
  auto dig = [](double x, int e) {
    const Dig d = fx_coef(x, ldexp(1.0, -e));
    return make_int2(d.h, d.l);
  };
  for (int m = 0; m < 4; ++m) {
    for (int a = 0; a < 3; ++a) {
      K.g[a][m] = dig(K.gd[a] * L.mu * fx_weight(m), K.eg);
      K.c[a][m] = dig(K.cd[a] * fx_weight(m), K.ec);
    }
    K.w[m] = dig(K.wd * fx_weight(m), K.eg + kFxWUp);
  }
  return K;
}

// ---- coefficients at the points of a thread's plane ---------------------------------------------------
// Trilinear cells: stored digits.  Cartesian cells: G and C are diagonal, times the tensor Gauss weight,
// which in a plane takes three values (by the number of middle points among x and y).
template <typename P, bool CART>
struct FxGeo;
template <>
struct FxGeo<FxInt, false> {
  const int2 *g, *cc;  // shared memory: this lane's first entries of the staged blocks
  __device__ __forceinline__ Dig at(int pt, int f) const {
    const int2 v = g[(pt * kFxG + f) * 32];
    return {v.x, v.y};
  }
  __device__ __forceinline__ Dig col(int pt, int c, int a) const {
    const int2 v = cc[(pt * kFxC + 3 * c + a) * 32];
    return {v.x, v.y};
  }
  template <int MODE>
  __device__ __forceinline__ const FxGeo &point(int, int) const {
    return *this;
  }
};
template <>
struct FxGeo<FxDbl, false> {
  FxGeo<FxInt, false> d;
  int eg, ec;
  __device__ __forceinline__ double at(int pt, int f) const {
    return fx_coef_value(d.at(pt, f), f < 6 ? eg : eg + kFxWUp);
  }
  __device__ __forceinline__ double col(int pt, int c, int a) const { return fx_coef_value(d.col(pt, c, a), ec); }
  template <int MODE>
  __device__ __forceinline__ const FxGeo &point(int, int) const {
    return *this;
  }
};
// FP32: quads of (G00, G01, G02, G11), (G12, G22, W, -) and a column of C per component, one point in registers.
template <>
struct FxGeo<FxFlt, false> {
  const float4 *g, *cc;  // shared memory: this lane's first quads of the staged blocks
  struct Point {
    float4 a, b, d;
    __device__ __forceinline__ float at(int, int i) const {
      return i == 0 ? a.x : (i == 1 ? a.y : (i == 2 ? a.z : (i == 3 ? a.w : (i == 4 ? b.x : (i == 5 ? b.y : b.z)))));
    }
    __device__ __forceinline__ float col(int, int, int k) const { return k == 0 ? d.x : (k == 1 ? d.y : d.z); }
  };
  template <int MODE>
  __device__ __forceinline__ Point point(int pt, int c) const {
    Point q;
    if (MODE & kApplyA) {
      q.a = g[2 * pt * 32];
      q.b = g[(2 * pt + 1) * 32];
    }
    if (MODE & (kApplyB | kApplyBT)) q.d = cc[(3 * pt + c) * 32];
    return q;
  }
};
// What a launch stages: the G block with an A block, the C block with B or B^T.
template <int MODE>
struct FxStage {
  static constexpr int G = (MODE & kApplyA) ? 9 * kFxG * 32 * (int)sizeof(int2) : 0;
  static constexpr int C = (MODE & (kApplyB | kApplyBT)) ? 9 * kFxC * 32 * (int)sizeof(int2) : 0;
};
template <typename P>
struct FxGeo<P, true> {
  typename P::C g[3][3], w[3], cc[3];  // [direction][weight class]
};

template <int MODE, typename P>
__device__ __forceinline__ const FxGeo<P, true> &fx_point(const FxGeo<P, true> &g, int, int) {
  return g;
}
template <int MODE, typename P>
__device__ __forceinline__ decltype(auto) fx_point(const FxGeo<P, false> &g, int pt, int c) {
  return g.template point<MODE>(pt, c);
}

// The element action on a thread's plane.  v: in the 9 node values of plane z (scaled integers, or
// doubles), out the 9 test sums of that node plane times 2^-kFxTDown;
// pr: the cell's 8 pressure values; qn: out, the sums of the four pressure nodes at z = 0 (lanes of
// plane 0) or z = 1 (plane 2).  sa: right shift of the fluxes of A.
template <typename P, int MODE, bool CART>
__device__ __forceinline__ void fx_plane(typename P::V (&v)[3][3], const typename P::V (&pr)[2][2][2],
                                         typename P::V (&qn)[2][2], const FxGeo<P, CART> &geo, int c, int z, int lane,
                                         int sa) {
  typedef typename P::V V;
  typedef typename P::C Cf;
  constexpr bool DO_A = MODE & kApplyA, DO_BT = MODE & kApplyBT, DO_B = MODE & kApplyB;
  constexpr bool NEED_U = DO_A || DO_B;
  constexpr unsigned FULL = 0xffffffffu;
  const int l1 = lane < 20 ? lane + 10 : (lane < 30 ? lane - 20 : lane), l2 = lane < 10 ? lane + 20 : (lane < 30 ? lane - 10 : lane);
  // coefficients of planes z, z + 1, z + 2 (mod 3) in this plane's Gauss value (less the unit part of the
  // own plane) and scaled derivative (less the whole parts (-2, 2, 0), (0, 1, -1), (2, 0, -2))
  Cf s0, s1, s2, d0, d1, d2;
  {
    const Cf o = P::tab(0, 0), S00M = P::tab(-1343043426, -896144430), S01 = P::tab(1717986918, 1717986918),
             S02 = P::tab(-374943492, -821842488);
    const Cf e0 = P::tab(109106475, -784691517), ne0 = P::tab(-109106475, 784691517),    // 0.8 - 2r
             e2 = P::tab(-1827093393, -933295402), ne2 = P::tab(1827093393, 933295402),  // 2r - 1.2
             e3 = P::tab(-968099934, -74301943), ne3 = P::tab(968099934, 74301943),  // 2r - 1
             nS01 = P::tab(-1717986918, -1717986918);
    s0 = z == 1 ? o : S00M;
    s1 = z == 0 ? S01 : (z == 1 ? o : S02);
    s2 = z == 0 ? S02 : (z == 1 ? o : S01);
    d0 = z == 0 ? e0 : (z == 1 ? o : ne0);
    d1 = z == 0 ? S01 : (z == 1 ? e3 : ne2);
    d2 = z == 0 ? e2 : (z == 1 ? ne3 : nS01);
    if constexpr (!P::SPLIT) {  // the whole parts belong to the table
      s0 += P::zero() + 1;
      d0 += z == 0 ? -2 : (z == 1 ? 0 : 2);
      d1 += z == 0 ? 2 : (z == 1 ? 1 : 0);
      d2 += z == 0 ? 0 : (z == 1 ? -1 : -2);
    }
  }
  V pq[3][3];
  if (DO_BT) {
    const Cf rz = z == 0 ? P::tab(1663433681, -37150971) : (z == 1 ? P::tab(0, 0) : P::tab(-1663433681, 37150971));
    V t[2][3];
#pragma unroll
    for (int y = 0; y < 2; ++y) {
      V m[2];
#pragma unroll
      for (int x = 0; x < 2; ++x)
        m[x] = P::value(P::start(P::half(pr[0][y][x] + pr[1][y][x]), rz, pr[0][y][x] - pr[1][y][x]));
      fx_pre<P>(m[0], m[1], t[y]);
    }
#pragma unroll
    for (int x = 0; x < 3; ++x) {
      V q[3];
      fx_pre<P>(t[0][x], t[1][x], q);
#pragma unroll
      for (int y = 0; y < 3; ++y) pq[y][x] = q[y];
    }
  }
  V gz[3][3];
  if (NEED_U) {
#pragma unroll
    for (int y = 0; y < 3; ++y) fx_interp<P>(v[y][0], v[y][1], v[y][2]);
#pragma unroll
    for (int x = 0; x < 3; ++x) fx_interp<P>(v[0][x], v[1][x], v[2][x]);
#pragma unroll
    for (int y = 0; y < 3; ++y)
#pragma unroll
      for (int x = 0; x < 3; ++x) {
        const V a = v[y][x], b = __shfl_sync(FULL, a, l1), e = __shfl_sync(FULL, a, l2);
        V qb = P::zero(), gb = P::zero();
        if constexpr (P::SPLIT) {
          const V w = (z == 2 ? a : b) - (z == 0 ? a : e);
          qb = a;
          gb = z == 1 ? w : 2 * w;
        }
        typename P::Sum q = P::start(qb, s0, a), g = P::start(gb, d0, a);
        P::add(q, s1, b);
        P::add(g, d1, b);
        P::add(q, s2, e);
        P::add(g, d2, e);
        v[y][x] = P::value(q);
        gz[y][x] = P::value(g);
      }
  }
  // point operation, one row of points at a time; t: test sums of the plane, gz becomes the z flux
  V t[3][3], qa[3][3];
#pragma unroll
  for (int y = 0; y < 3; ++y)
#pragma unroll
    for (int x = 0; x < 3; ++x) t[y][x] = P::zero();
  V dy[3], ey[3];
  if (NEED_U) {
#pragma unroll
    for (int x = 0; x < 3; ++x) {
      dy[x] = v[2][x] - v[0][x];
      ey[x] = 2 * (v[0][x] + v[2][x] - 2 * v[1][x]);
    }
  }
#pragma unroll
  for (int y = 0; y < 3; ++y) {
    V f0[3];
    V dx = P::zero(), ex = P::zero();
    if (NEED_U) {
      dx = v[y][2] - v[y][0];
      ex = 2 * (v[y][0] + v[y][2] - 2 * v[y][1]);
    }
#pragma unroll
    for (int x = 0; x < 3; ++x) {
      const int pt = y * 3 + x, m = (x == 1) + (y == 1);
      V gx = P::zero(), gy = P::zero();
      if (NEED_U) {
        gx = x == 0 ? dx - ex : (x == 1 ? dx : dx + ex);
        gy = y == 0 ? dy[x] - ey[x] : (y == 1 ? dy[x] : dy[x] + ey[x]);
      }
      const V gzp = NEED_U ? gz[y][x] : P::zero();
      V a0 = P::zero(), a1 = P::zero(), a2 = P::zero();
      decltype(auto) pg = fx_point<MODE>(geo, pt, c);
      if constexpr (DO_A) {
        V w;
        if constexpr (CART) {
          a0 = P::value(P::start(P::zero(), geo.g[0][m], gx));
          a1 = P::value(P::start(P::zero(), geo.g[1][m], gy));
          a2 = P::value(P::start(P::zero(), geo.g[2][m], gzp));
          w = P::template value_up<kFxWUp>(P::start(P::zero(), geo.w[m], v[y][x]));
        } else {
          const Cf g1 = pg.at(pt, 1), g2 = pg.at(pt, 2), g4 = pg.at(pt, 4);
          typename P::Sum q0 = P::start(P::zero(), pg.at(pt, 0), gx), q1 = P::start(P::zero(), g1, gx),
                          q2 = P::start(P::zero(), g2, gx);
          P::add(q0, g1, gy);
          P::add(q1, pg.at(pt, 3), gy);
          P::add(q2, g4, gy);
          P::add(q0, g2, gzp);
          P::add(q1, g4, gzp);
          P::add(q2, pg.at(pt, 5), gzp);
          a0 = P::value(q0);
          a1 = P::value(q1);
          a2 = P::value(q2);
          w = P::template value_up<kFxWUp>(P::start(P::zero(), pg.at(pt, 6), v[y][x]));
        }
        if (DO_BT) {
          a0 = P::down_by(a0, sa);
          a1 = P::down_by(a1, sa);
          a2 = P::down_by(a2, sa);
          w = P::down_by(w, sa);
        }
        t[y][x] += w;
      }
      if constexpr (DO_BT || DO_B) {
        if constexpr (CART) {
          const Cf k = geo.cc[m];
          if (DO_BT) {
            const V d = P::value(P::start(P::zero(), k, pq[y][x]));
            a0 -= c == 0 ? d : P::zero();
            a1 -= c == 1 ? d : P::zero();
            a2 -= c == 2 ? d : P::zero();
          }
          if (DO_B) qa[y][x] = -P::value(P::start(P::zero(), k, c == 0 ? gx : (c == 1 ? gy : gzp)));
        } else {
          const Cf c0 = pg.col(pt, c, 0), c1 = pg.col(pt, c, 1), c2 = pg.col(pt, c, 2);
          if (DO_BT) {
            a0 -= P::value(P::start(P::zero(), c0, pq[y][x]));
            a1 -= P::value(P::start(P::zero(), c1, pq[y][x]));
            a2 -= P::value(P::start(P::zero(), c2, pq[y][x]));
          }
          if (DO_B) {
            typename P::Sum q = P::start(P::zero(), c0, gx);
            P::add(q, c1, gy);
            P::add(q, c2, gzp);
            qa[y][x] = -P::value(q);
          }
        }
      }
      if (DO_A || DO_BT) {
        f0[x] = a0;
        gz[y][x] = a2;
        if (y == 0) {
          t[0][x] -= 3 * a1;
          t[1][x] += 4 * a1;
          t[2][x] -= a1;
        } else if (y == 1) {
          t[0][x] -= a1;
          t[2][x] += a1;
        } else {
          t[0][x] += a1;
          t[1][x] -= 4 * a1;
          t[2][x] += 3 * a1;
        }
      }
    }
    if (DO_A || DO_BT) {
      const V a = f0[0] - f0[2];
      t[y][0] -= 2 * f0[0] + f0[1] + a;
      t[y][1] += 4 * a;
      t[y][2] += 2 * f0[2] + f0[1] - a;
    }
  }
  if (DO_A || DO_BT) {
    // this plane's contributions to node planes z, z + 1, z + 2 (the transposes of s and d by symmetry
    // of position: plane z's coefficient of plane m), summed over the three planes
#pragma unroll
    for (int y = 0; y < 3; ++y)
#pragma unroll
      for (int x = 0; x < 3; ++x) {
        const V a = P::tdown(t[y][x]), f = P::tdown(gz[y][x]);
        V b0 = P::zero(), b1 = P::zero(), b2 = P::zero();
        if constexpr (P::SPLIT) {
          const V w = z == 1 ? f : 2 * f;
          b0 = a + (z == 0 ? -w : (z == 1 ? P::zero() : w));
          b1 = z == 2 ? P::zero() : w;
          b2 = z == 0 ? P::zero() : -w;
        }
        typename P::Sum c0 = P::start(b0, s0, a), c1 = P::start(b1, s1, a), c2 = P::start(b2, s2, a);
        P::add(c0, d0, f);
        P::add(c1, d1, f);
        P::add(c2, d2, f);
        // c1 belongs to plane z + 1: it arrives there from l2 (the plane before); c2 from l1
        v[y][x] = P::value(c0) + __shfl_sync(FULL, P::value(c1), l2) + __shfl_sync(FULL, P::value(c2), l1);
      }
#pragma unroll
    for (int x = 0; x < 3; ++x) fx_interp_t<P>(v[0][x], v[1][x], v[2][x]);
#pragma unroll
    for (int y = 0; y < 3; ++y) fx_interp_t<P>(v[y][0], v[y][1], v[y][2]);
  }
  if (DO_B) {
    V r[3][2], w[2][2];
#pragma unroll
    for (int y = 0; y < 3; ++y) fx_pre_t<P>(qa[y][0], qa[y][1], qa[y][2], r[y][0], r[y][1]);
#pragma unroll
    for (int x = 0; x < 2; ++x) fx_pre_t<P>(r[0][x], r[1][x], r[2][x], w[0][x], w[1][x]);
#pragma unroll
    for (int y = 0; y < 2; ++y)
#pragma unroll
      for (int x = 0; x < 2; ++x) {
        const V a = w[y][x], b = __shfl_sync(FULL, a, l1), e = __shfl_sync(FULL, a, l2);
        // plane 0: own - plane 2 (l2); plane 2: own - plane 0 (l1); both sums add r times that
        qn[y][x] = P::value(P::start(P::half(a + b + e), FxTR{}, a - (z == 0 ? e : b)));
      }
  }
}

// ---- a warp's cells of one component: indices, gathers, scatter (any precision) ---------------------------
struct PlaneIdx {
  int lane, z, cx, cy, cz;
  bool fast;  // FP32: every node of the warp's cells is free, no per-node predicates (FP64's code is long enough)
  bool pad, valid, fx[3], fy[3];
  unsigned cell;
  long long N0, P0, P01, vbase, pbase;
};
template <typename T>
__device__ __forceinline__ PlaneIdx plane_index(const LevelDesc<T> &L, long long group, int c) {
  PlaneIdx I;
  I.lane = threadIdx.x & 31;
  I.pad = I.lane >= 30;
  I.z = I.pad ? 0 : I.lane / 10;
  const int s = I.pad ? 0 : I.lane - 10 * I.z;
  const long long cell_raw = group * kFxCells + s;
  I.valid = !I.pad && cell_raw < L.n_cells;
  I.cell = (unsigned)(I.valid ? cell_raw : 0);  // launches hold n_cells below 2^31
  I.cx = (int)(I.cell % (unsigned)L.n[0]);
  const unsigned rr = I.cell / (unsigned)L.n[0];
  I.cy = (int)(rr % (unsigned)L.n[1]);
  I.cz = (int)(rr / (unsigned)L.n[1]);
  const int gx0 = 2 * I.cx, gy0 = 2 * I.cy, gz0 = 2 * I.cz + I.z;
  const bool fz = I.valid && !((L.faces & 16u) && gz0 == 0) && !((L.faces & 32u) && gz0 == L.N[2] - 1);
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    I.fx[i] = fz && !((L.faces & 1u) && gx0 + i == 0) && !((L.faces & 2u) && gx0 + i == L.N[0] - 1);
    I.fy[i] = !((L.faces & 4u) && gy0 + i == 0) && !((L.faces & 8u) && gy0 + i == L.N[1] - 1);
  }
  I.fast = sizeof(T) == 4 && __all_sync(0xffffffffu, I.pad || (I.fx[0] && I.fx[1] && I.fx[2] && I.fy[0] && I.fy[1] && I.fy[2]));
  I.N0 = L.N[0];
  I.vbase = c * L.nv + ((long long)gz0 * L.N[1] + gy0) * I.N0 + gx0;
  I.P0 = L.Pn[0];
  I.P01 = (long long)L.Pn[0] * L.Pn[1];
  I.pbase = ((long long)I.cz * L.Pn[1] + I.cy) * I.P0 + I.cx;
  return I;
}
// The 9 node values of the thread's plane and the cell's 8 pressure values.  FUSED: the Fuse combinations, and
// the owner of each node performs their side effects (see Fuse and cc_group).
template <int MODE, bool FUSED, typename T>
__device__ __forceinline__ void plane_gather(const LevelDesc<T> &L, const PlaneIdx &I, int c, const T *__restrict__ u,
                                             const T *__restrict__ p, const Fuse<T> &F, T (&uv)[3][3], T (&pv)[2][2][2]) {
  constexpr bool NEED_U = MODE & (kApplyA | kApplyB), DO_BT = MODE & kApplyBT;
  if constexpr (FUSED) {
    const bool oz = I.valid && (I.z < 2 || I.cz == L.n[2] - 1);
    bool ox[3], oy[3];  // this cell owns the node (local index below the last, or last cell)
#pragma unroll
    for (int i = 0; i < 3; ++i) {
      ox[i] = oz && (i < 2 || I.cx == L.n[0] - 1);
      oy[i] = i < 2 || I.cy == L.n[1] - 1;
    }
    T raw[kFuseVel + 2][3][3];  // every load first
#pragma unroll
    for (int iy = 0; iy < 3; ++iy)
#pragma unroll
      for (int ix = 0; ix < 3; ++ix) {
        const long long gi = I.vbase + iy * I.N0 + ix;
        const bool need = (NEED_U && I.fx[ix] && I.fy[iy]) || (ox[ix] && oy[iy] && F.vstore);
        if (F.nv > 0) {
#pragma unroll
          for (int j = 0; j < kFuseVel; ++j) raw[j][iy][ix] = (need && j < F.nv) ? F.vv[j][gi] : T(0);
          raw[kFuseVel][iy][ix] = (need && F.vd) ? F.vd[gi] : T(1);
          raw[kFuseVel + 1][iy][ix] = (need && F.vb) ? F.vb[gi] : T(0);
        } else {
          raw[0][iy][ix] = need ? u[gi] : T(0);
        }
      }
#pragma unroll
    for (int iy = 0; iy < 3; ++iy)
#pragma unroll
      for (int ix = 0; ix < 3; ++ix) {
        const long long gi = I.vbase + iy * I.N0 + ix;
        T val = raw[0][iy][ix];
        if (F.nv > 0) {
          T sum = F.vc[0] * raw[0][iy][ix];
#pragma unroll
          for (int j = 1; j < kFuseVel; ++j)
            if (j < F.nv) sum += F.vc[j] * raw[j][iy][ix];
          val = raw[kFuseVel + 1][iy][ix] + raw[kFuseVel][iy][ix] * sum;
        }
        uv[iy][ix] = (I.fx[ix] && I.fy[iy]) ? val : T(0);
        if (ox[ix] && oy[iy]) {
          if (F.vstore) F.vstore[gi] = val;
          if (F.vzero[0]) F.vzero[0][gi] = T(0);
          if (F.vzero[1]) F.vzero[1][gi] = T(0);
        }
      }
  } else if (NEED_U) {
    const T *ub = u + I.vbase;
    if (I.fast) {
#pragma unroll
      for (int iy = 0; iy < 3; ++iy)
#pragma unroll
        for (int ix = 0; ix < 3; ++ix) uv[iy][ix] = ub[iy * I.N0 + ix];
    } else {
#pragma unroll
      for (int iy = 0; iy < 3; ++iy)
#pragma unroll
        for (int ix = 0; ix < 3; ++ix) uv[iy][ix] = (I.fx[ix] && I.fy[iy]) ? ub[iy * I.N0 + ix] : T(0);
    }
  }
  if (DO_BT) {
#pragma unroll
    for (int a3 = 0; a3 < 2; ++a3)
#pragma unroll
      for (int a2 = 0; a2 < 2; ++a2)
#pragma unroll
        for (int a1 = 0; a1 < 2; ++a1) {
          const long long gi = I.pbase + a3 * I.P01 + a2 * I.P0 + a1;
          T val = T(0);
          if (I.valid) {
            if (FUSED && F.np > 0) {
              T sum = T(0);
#pragma unroll
              for (int j = 0; j < kFusePre; ++j)
                if (j < F.np) sum += F.pc[j] * F.pv[j][gi];
              val = F.pd[gi] * sum;
            } else {
              val = p[gi];
            }
          }
          pv[a3][a2][a1] = val;
        }
    if constexpr (FUSED) {  // once per node: component 0, planes 0 and 2 for the two z nodes
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        const int a1 = i & 1, a2 = (i >> 1) & 1, a3 = i >> 2;
        if (I.valid && c == 0 && I.z == 2 * a3 && (a1 < 1 || I.cx == L.n[0] - 1) && (a2 < 1 || I.cy == L.n[1] - 1) &&
            (a3 < 1 || I.cz == L.n[2] - 1)) {
          const long long gi = I.pbase + a3 * I.P01 + a2 * I.P0 + a1;
          if (F.pacc) F.pacc[gi] += pv[a3][a2][a1];
#pragma unroll
          for (int j = 0; j < kFusePre; ++j)
            if (F.pzero[j]) F.pzero[j][gi] = T(0);
        }
      }
    }
  }
}
template <int MODE, typename T>
__device__ __forceinline__ void plane_scatter(const PlaneIdx &I, T *__restrict__ yu, T *__restrict__ yp, const T (&yv)[3][3],
                                              const T (&qv)[2][2]) {
  if (MODE & (kApplyA | kApplyBT)) {
    T *yb = yu + I.vbase;
    if (I.fast) {
      if (!I.pad) {
#pragma unroll
        for (int iy = 0; iy < 3; ++iy)
#pragma unroll
          for (int ix = 0; ix < 3; ++ix) atomicAdd(&yb[iy * I.N0 + ix], yv[iy][ix]);
      }
    } else {
#pragma unroll
      for (int iy = 0; iy < 3; ++iy)
#pragma unroll
        for (int ix = 0; ix < 3; ++ix)
          if (I.fx[ix] && I.fy[iy]) atomicAdd(&yb[iy * I.N0 + ix], yv[iy][ix]);
    }
  }
  if (MODE & kApplyB) {
    if (I.valid && I.z != 1) {
#pragma unroll
      for (int iy = 0; iy < 2; ++iy)
#pragma unroll
        for (int ix = 0; ix < 2; ++ix) atomicAdd(&yp[I.pbase + (I.z >> 1) * I.P01 + iy * I.P0 + ix], qv[iy][ix]);
    }
  }
}
// A contiguous block to shared memory in 16-byte pieces, without waiting.
template <int BYTES>
__device__ __forceinline__ void plane_stage(const void *src, void *dst) {
  const int4 *s = static_cast<const int4 *>(src) + threadIdx.x;
  const unsigned d = (unsigned)__cvta_generic_to_shared(static_cast<int4 *>(dst) + threadIdx.x);
  constexpr int N = BYTES / 16;
#pragma unroll
  for (int i = 0; i < (N + kFxThreads - 1) / kFxThreads; ++i)
    if ((i + 1) * kFxThreads <= N || (int)threadIdx.x < N - i * kFxThreads)
      asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(d + i * kFxThreads * 16), "l"(s + i * kFxThreads)
                   : "memory");
}

// One warp's cells of one component in FP64.
template <int MODE, bool CART, bool FUSED>
__device__ __forceinline__ void fx_group(const LevelDesc<double> &L, const double *__restrict__ u,
                                         const double *__restrict__ p, double *__restrict__ yu, double *__restrict__ yp,
                                         const int2 *__restrict__ geo, long long group, int c, const FxCart &K, const Fuse<double> &F) {
  constexpr bool DO_A = MODE & kApplyA, DO_BT = MODE & kApplyBT, DO_B = MODE & kApplyB;
  constexpr bool NEED_U = DO_A || DO_B;
  constexpr unsigned FULL = 0xffffffffu;
  // Trilinear cells: the group's coefficients go to shared memory while the values are gathered (without
  // it a warp waited for them at every point: 10.4 of 15 stall cycles an issue).
  extern __shared__ int4 fx_smem[];
  using ST = FxStage<MODE>;
  if constexpr (!CART) {
    const int2 *src = geo + group * fx_group_entries();
    plane_stage<ST::G>(src, fx_smem);
    plane_stage<ST::C>(src + 9 * kFxG * 32, fx_smem + ST::G / 16);
    asm volatile("cp.async.commit_group;" ::: "memory");
  }
  const PlaneIdx I = plane_index(L, group, c);
  const int lane = I.lane, z = I.z;
  const unsigned cell = I.cell;
  double uv[3][3], pv[2][2][2];
  plane_gather<MODE, FUSED>(L, I, c, u, p, F, uv, pv);

  // ---- coefficients and scales ---------------------------------------------------------------------
  int eg, ec;
  if constexpr (CART) {
    eg = K.eg;
    ec = K.ec;
    if (L.mu_cell && DO_A) eg = fx_scale_g(K.xy * L.mu_cell[cell], K.zz * L.mu_cell[cell], K.wtop);
  } else {
    const int2 e = __ldg(geo + (L.n_cells + kFxCells - 1) / kFxCells * fx_group_entries() + cell);
    eg = e.x;
    ec = e.y;
  }
  int tu = 0, tp = 0;
  if (NEED_U) {
#pragma unroll
    for (int i = 0; i < 9; ++i) tu = max(tu, __double2hiint(uv[i / 3][i % 3]) & 0x7fffffff);
    const int l1 = lane < 20 ? lane + 10 : (I.pad ? lane : lane - 20), l2 = lane < 10 ? lane + 20 : (I.pad ? lane : lane - 10);
    tu = max(tu, max(__shfl_sync(FULL, tu, l1), __shfl_sync(FULL, tu, l2)));
  }
  if (DO_BT) {
#pragma unroll
    for (int i = 0; i < 8; ++i) tp = max(tp, __double2hiint(pv[i >> 2][(i >> 1) & 1][i & 1]) & 0x7fffffff);
  }
  const int eu = tu >> 20, ep = tp >> 20;              // biased; 0: all zero (or below 2^-1042)
  const int su = eu - 1022 - 58, sp = ep - 1022 - 59;  // the integers are multiples of 2^su, 2^sp
  const int ea = su + eg + 64, eb = sp + ec + 64;      // scales of the fluxes
  int ev = DO_A ? ea : eb, sa = 0, more = 0;
  bool ok = true;
  if (NEED_U) ok = ok && (tu == 0 || (eu > 173 && eu < 1873));
  if (DO_BT) ok = ok && (tp == 0 || (ep > 173 && ep < 1873));
  if (DO_A && DO_BT) {
    if (tp != 0 && (tu == 0 || eb > ea)) {
      ev = eb;
      sa = tu == 0 ? 0 : min(eb - ea, 63);
    } else {
      more = tp == 0 ? 0 : min(ea - eb, 63);
    }
  }
  if (DO_A || DO_BT) ok = ok && ((tu == 0 && tp == 0) || (ev > -900 && ev < 850));
  if (DO_B) ok = ok && (tu == 0 || (su + ec + 64 > -900 && su + ec + 64 < 850));

  if constexpr (!CART) {  // the staged coefficients
    asm volatile("cp.async.wait_all;" ::: "memory");
    __syncthreads();
  }
  double yv[3][3], qv[2][2];
  if (__all_sync(FULL, ok)) {
    i64 v[3][3], pi[2][2][2], qn[2][2];
    const double ku = tu == 0 ? 0.0 : fx_pow2(-su), kp = tp == 0 ? 0.0 : fx_pow2(-sp - more);
    if (NEED_U) {
#pragma unroll
      for (int i = 0; i < 9; ++i) v[i / 3][i % 3] = __double2ll_rn(uv[i / 3][i % 3] * ku);
    }
    if (DO_BT) {
#pragma unroll
      for (int i = 0; i < 8; ++i)
        pi[i >> 2][(i >> 1) & 1][i & 1] = __double2ll_rn(pv[i >> 2][(i >> 1) & 1][i & 1] * kp);
    }
    FxGeo<FxInt, CART> g;
    if constexpr (CART) {
#pragma unroll
      for (int m = 0; m < 3; ++m) {
        auto pick = [&](const int2 &a, const int2 &b) { return z == 1 ? Dig{b.x, b.y} : Dig{a.x, a.y}; };
        if (DO_A) {
#pragma unroll
          for (int a = 0; a < 3; ++a) g.g[a][m] = pick(K.g[a][m], K.g[a][m + 1]);
          g.w[m] = pick(K.w[m], K.w[m + 1]);
        }
        if (DO_B || DO_BT) g.cc[m] = pick(K.c[c][m], K.c[c][m + 1]);
      }
      if (DO_A && L.mu_cell) {
        const double mu = L.mu_cell[cell], kg = ldexp(1.0, -eg);
#pragma unroll
        for (int m = 0; m < 3; ++m) {
          const double w = kg * fx_weight(m + (z == 1));
#pragma unroll
          for (int a = 0; a < 3; ++a) g.g[a][m] = fx_coef(K.gd[a] * mu, w);
          g.w[m] = fx_coef(K.wd, w * (1.0 / (1 << kFxWUp)));
        }
      }
    } else {
      g.g = reinterpret_cast<const int2 *>(fx_smem) + lane;
      g.cc = reinterpret_cast<const int2 *>(fx_smem + ST::G / 16) + lane;
    }
    fx_plane<FxInt, MODE, CART>(v, pi, qn, g, c, z, lane, sa);
    const double kv = tu == 0 && tp == 0 ? 0.0 : fx_pow2(ev + kFxTDown), kq = tu == 0 ? 0.0 : fx_pow2(su + ec + 64);
    if (DO_A || DO_BT) {
#pragma unroll
      for (int i = 0; i < 9; ++i) yv[i / 3][i % 3] = (double)v[i / 3][i % 3] * kv;
    }
    if (DO_B) {
#pragma unroll
      for (int i = 0; i < 4; ++i) qv[i >> 1][i & 1] = (double)qn[i >> 1][i & 1] * kq;
    }
  } else {
    FxGeo<FxDbl, CART> g;
    if constexpr (CART) {
      const double mu = L.mu_cell ? L.mu_cell[cell] : L.mu;
#pragma unroll
      for (int m = 0; m < 3; ++m) {
        const double w = fx_weight(m + (z == 1));
#pragma unroll
        for (int a = 0; a < 3; ++a) g.g[a][m] = K.gd[a] * mu * w;
        g.w[m] = K.wd * w;
        g.cc[m] = K.cd[c] * w;
      }
    } else {
      g.d.g = reinterpret_cast<const int2 *>(fx_smem) + lane;
      g.d.cc = reinterpret_cast<const int2 *>(fx_smem + ST::G / 16) + lane;
      g.eg = eg;
      g.ec = ec;
    }
    double qn[2][2];
    fx_plane<FxDbl, MODE, CART>(uv, pv, qn, g, c, z, lane, 0);
#pragma unroll
    for (int i = 0; i < 9; ++i) yv[i / 3][i % 3] = uv[i / 3][i % 3];
#pragma unroll
    for (int i = 0; i < 4; ++i) qv[i >> 1][i & 1] = qn[i >> 1][i & 1];
  }

  plane_scatter<MODE>(I, yu, yp, yv, qv);
}

template <int MODE, bool CART>
__global__ void __launch_bounds__(kFxThreads, 4)
    stokes_cell_apply_fx(const LevelDesc<double> L, const double *__restrict__ u, const double *__restrict__ p,
                         double *__restrict__ yu, double *__restrict__ yp, const int2 *__restrict__ geo, const __grid_constant__ FxCart K,
                         const long long ld) {
  pdl_enter();
  fx_group<MODE, CART, false>(L, column(u, ld), column(p, ld), column(yu, ld), column(yp, ld), geo, blockIdx.x, threadIdx.x >> 5, K, Fuse<double>{});
}
template <int MODE, bool CART>
__global__ void __launch_bounds__(kFxThreads, 4)
    stokes_cell_apply_fx_fused(const LevelDesc<double> L, const double *__restrict__ u, const double *__restrict__ p,
                               double *__restrict__ yu, double *__restrict__ yp, const int2 *__restrict__ geo,
                               const __grid_constant__ FxCart K, const Fuse<double> F) {
  pdl_enter();
  fx_group<MODE, CART, true>(L, u, p, yu, yp, geo, blockIdx.x, threadIdx.x >> 5, K, F);
}

// ---- the stored coefficients of trilinear cells ----------------------------------------------------------
// Formed at setup in pairs of doubles (about 106 bits): FP64 geometry would leave more error in the operator
// than the fixed-point arithmetic does.
struct Dd {
  double h, l;
};
__device__ __forceinline__ Dd dd_two(double a, double b) {  // exact sum, any order
  const double s = a + b, t = s - a;
  return {s, (a - (s - t)) + (b - t)};
}
__device__ __forceinline__ Dd operator+(Dd a, Dd b) {
  const Dd s = dd_two(a.h, b.h);
  const double l = s.l + (a.l + b.l), h = s.h + l;
  return {h, l - (h - s.h)};
}
__device__ __forceinline__ Dd operator-(Dd a) { return {-a.h, -a.l}; }
__device__ __forceinline__ Dd operator-(Dd a, Dd b) { return a + (-b); }
__device__ __forceinline__ Dd operator*(Dd a, Dd b) {
  const double p = a.h * b.h, l = fma(a.h, b.h, -p) + (a.h * b.l + a.l * b.h), h = p + l;
  return {h, l - (h - p)};
}
__device__ __forceinline__ Dd dd_div(Dd a, Dd b) {
  const double q = a.h / b.h;
  const Dd r = a - Dd{q, 0.0} * b;
  return dd_two(q, r.h / b.h);
}

// One warp per cell, a lane per Gauss point: T_tau's Jacobian J from the 8 vertices (Sec. 2), G = mu w adj(J)
// adj(J)^T / det J, W = gamma rho w det J, C = w adj(J), times 1 / (2r)^2, 1 and 1 / (2r).
template <int K>
__global__ void k_fx_geometry(const LevelDesc<double> L, int2 *__restrict__ out) {
  pdl_enter();
  constexpr Dd X[3] = {{0.11270166537925831, -2.5675694035077516e-19}, {0.5, 0.0}, {0.8872983346207417, -1.3621030867463682e-17}};
  constexpr Dd Wt[3] = {{0.2777777777777778, -1.2335811384723961e-17}, {0.4444444444444444, 2.4671622769447922e-17}, {0.2777777777777778, -1.2335811384723961e-17}};
  constexpr Dd A1{1.2909944487358056, 2.861143208346483e-17}, A2{1.6666666666666667, -7.401486830834377e-17};
  const int lane = threadIdx.x & 31, pt = lane < 27 ? lane : 0;
  const int ix = pt % 3, iy = (pt / 3) % 3, iz = pt / 9;
  const Dd xi = ix == 0 ? X[0] : (ix == 1 ? X[1] : X[2]), eta = iy == 0 ? X[0] : (iy == 1 ? X[1] : X[2]),
           zeta = iz == 0 ? X[0] : (iz == 1 ? X[1] : X[2]);
  const Dd w = (ix == 1 ? Wt[1] : Wt[0]) * (iy == 1 ? Wt[1] : Wt[0]) * (iz == 1 ? Wt[1] : Wt[0]);
  const long long warps = (long long)gridDim.x * (blockDim.x >> 5);
  int2 *scales = out + (L.n_cells + kFxCells - 1) / kFxCells * fx_group_entries();
  for (long long cell = (long long)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5); cell < L.n_cells; cell += warps) {
    const int cx = (int)(cell % L.n[0]);
    const long long rr = cell / L.n[0];
    const int cy = (int)(rr % L.n[1]), cz = (int)(rr / L.n[1]);
    Dd J[3][3];  // J[a][b] = d x_a / d xi_b
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      double v[8];
#pragma unroll
      for (int i = 0; i < 8; ++i)
        v[i] = L.vert[(((long long)(cz + (i >> 2)) * (L.n[1] + 1) + (cy + ((i >> 1) & 1))) * (L.n[0] + 1) + (cx + (i & 1))) * 3 + a];
      auto lerp = [](Dd p, Dd q, Dd t) { return p + t * (q - p); };
      auto dif = [&](int i, int j) { return dd_two(v[i], -v[j]); };
      J[a][0] = lerp(lerp(dif(1, 0), dif(3, 2), eta), lerp(dif(5, 4), dif(7, 6), eta), zeta);
      J[a][1] = lerp(lerp(dif(2, 0), dif(3, 1), xi), lerp(dif(6, 4), dif(7, 5), xi), zeta);
      J[a][2] = lerp(lerp(dif(4, 0), dif(5, 1), xi), lerp(dif(6, 2), dif(7, 3), xi), eta);
    }
    Dd adj[3][3];  // adj[b][a]: rows c1 x c2, c2 x c0, c0 x c1 of J's columns
#pragma unroll
    for (int b = 0; b < 3; ++b)
#pragma unroll
      for (int a = 0; a < 3; ++a) {
        const int b1 = (b + 1) % 3, b2 = (b + 2) % 3, a1 = (a + 1) % 3, a2 = (a + 2) % 3;
        adj[b][a] = J[a1][b1] * J[a2][b2] - J[a2][b1] * J[a1][b2];
      }
    const Dd det = J[0][0] * adj[0][0] + J[1][0] * adj[0][1] + J[2][0] * adj[0][2];
    const Dd mu = {L.mu_cell ? L.mu_cell[cell] : L.mu, 0.0};
    const Dd wd = dd_div(A2 * mu * w, det);
    Dd f[kFxG + kFxC];
    {
      auto dot = [&](int i, int j) { return wd * (adj[i][0] * adj[j][0] + adj[i][1] * adj[j][1] + adj[i][2] * adj[j][2]); };
      f[0] = dot(0, 0);
      f[1] = dot(0, 1);
      f[2] = dot(0, 2);
      f[3] = dot(1, 1);
      f[4] = dot(1, 2);
      f[5] = dot(2, 2);
      f[6] = Dd{L.gamma_rho, 0.0} * w * det;
      const Dd wa = A1 * w;
#pragma unroll
      for (int c = 0; c < 3; ++c)
#pragma unroll
        for (int a = 0; a < 3; ++a) f[7 + 3 * c + a] = wa * adj[a][c];
    }
    double xy = fabs(f[0].h) + 2.0 * fabs(f[1].h) + fabs(f[2].h) + fabs(f[3].h) + fabs(f[4].h);
    double zz = fabs(f[2].h) + fabs(f[4].h) + fabs(f[5].h);
    double cols = 0.0, wm = fabs(f[6].h);
#pragma unroll
    for (int c = 0; c < 3; ++c) cols = fmax(cols, fabs(f[7 + 3 * c].h) + fabs(f[8 + 3 * c].h) + fabs(f[9 + 3 * c].h));
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      xy = fmax(xy, __shfl_xor_sync(0xffffffffu, xy, o));
      zz = fmax(zz, __shfl_xor_sync(0xffffffffu, zz, o));
      cols = fmax(cols, __shfl_xor_sync(0xffffffffu, cols, o));
      wm = fmax(wm, __shfl_xor_sync(0xffffffffu, wm, o));
    }
    const int eg = fx_scale_g(xy, zz, wm), ec = fx_scale_c(cols);
    if (lane < 27) {
      int2 *q = out + (cell / kFxCells) * fx_group_entries() + iz * 10 + cell % kFxCells;
#pragma unroll
      for (int i = 0; i < kFxG + kFxC; ++i) {
        const double s = ldexp(1.0, -(i < 6 ? eg : (i == 6 ? eg + kFxWUp : ec)));
        const Dig d = fx_split(__double2ll_rn(f[i].h * s) + __double2ll_rn(f[i].l * s));
        q[(i < kFxG ? (lane % 9) * kFxG + i : 9 * kFxG + (lane % 9) * kFxC + (i - kFxG)) * 32] = make_int2(d.h, d.l);
      }
    }
    if (lane == 0) scales[cell] = make_int2(eg, ec);
  }
}

// Launches one mode (its own translation unit: these are long kernels).
template <int MODE>
int launch_fx_mode(const LevelDesc<double> &L, const double *u, const double *p, double *yu, double *yp, const void *geo,
                   const Fuse<double> *F, cudaStream_t s, int cols, long long ld) {
  const dim3 grid((unsigned)((L.n_cells + kFxCells - 1) / kFxCells), F ? 1u : (unsigned)cols), block(kFxThreads);
  const int2 *g = static_cast<const int2 *>(geo);
  const FxCart K = L.cartesian ? fx_cart(L) : FxCart{};
  if (F) {
    if (L.cartesian)
      launch_kernel(stokes_cell_apply_fx_fused<MODE, true>, grid, block, 0, s, L, u, p, yu, yp, g, K, *F);
    else
      launch_kernel(stokes_cell_apply_fx_fused<MODE, false>, grid, block, FxStage<MODE>::G + FxStage<MODE>::C, s, L, u, p, yu, yp, g, K, *F);
  } else {
    if (L.cartesian)
      launch_kernel(stokes_cell_apply_fx<MODE, true>, grid, block, 0, s, L, u, p, yu, yp, g, K, ld);
    else
      launch_kernel(stokes_cell_apply_fx<MODE, false>, grid, block, FxStage<MODE>::G + FxStage<MODE>::C, s, L, u, p, yu, yp, g, K, ld);
  }
  return 0;
}

}  // namespace smf
