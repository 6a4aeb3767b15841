// chanfs_fix.cuh -- the FP64 transforms in block fixed point.
//
// GB300 executes 2 FP64 instructions per SM per clock against 64 integer
// ones, and a Stockham FFT in FP64 needs 12 to 14 of them per real point: the
// FP64 pipe bounds it at a tenth of the memory bandwidth.  Here a line (or
// column) of doubles is turned into 64-bit integers under one common power of
// two, transformed with integer additions and 32 x 32 + 64 -> 64 bit
// multiply-adds, and turned back into doubles once, at the end.
//
// Range.  Let B be the largest sum of |re| + |im| over the inputs of one
// first-pass butterfly and S the sum over the line.  The twiddle products come
// out divided by D = 4 (a 62-bit value times a 62-bit twiddle, the high half), so
// every pass after the first grows its values by R / D at most, and none exceeds
// S / D.  The scale 2^s is the largest with 2^s C < 2^headroom, C = max(B, min(B G,
// S / D_2)), G = max(1, R_2/D_2, R_2 R_3/(D_2 D_3), ..): no overflow for any input.
// The pass by pass division keeps the bits below a long line's sums that a bound on
// the whole line at the start (N max|x|, or S) would give away.  Transforms with few
// passes leave S out (C = B G), which costs them at most two bits.
// Precision.  Values start with 61 bits less the growth G below B and lose what the
// passes divide by beyond what they gain; additions are exact, a product is rounded
// to the last place of 62, the result is rounded to a double once.  D = 4 suits
// radix 8 and 6 and costs a radix-3 pass up to two bits of its values: a few such
// passes fit the eight bits over a double's 53, more do not, so D = 2 in the
// radix-3 passes of long plans of them (fix_halves).  Relative L2 errors in
// units of 2^-53 of columns like 1/k^2, one dominant value, white noise and
// magnitudes over 12 decades, D = 4 against 2: 729 7.9 8.7 1.8 3.3 against 0.7 0.6
// 0.9 1.4; 2187 24 34 4.0 9.5 against 0.8 1.1 2.0 4.5; 972 along x, inverse, 3.1 3.2
// 1.3 2.7 against 1.0 1.0 1.3 2.8; FP64 passes 1.5 to 4.4.
#pragma once

#include <cuda_runtime.h>
#include <math.h>

#include <vector>

namespace chanfs {

// A complex value.  (Twiddles are int4 (re hi, re lo, im hi, im lo): hi 2^-30 +
// lo 2^-62, lo signed.)
struct __align__(16) Fix {
  long long x, y;
};

// Radix of pass p of length n = 2^a 3^b (0 past the last pass): the fewest passes
// of radix 8, 6, 4, 3 and at most one 2 (16 as 4 x 4), in that order, the 6s last but
// for 3s.  PAIR (the real transform along x): the last radix is at most 6, since
// its last pass holds two mirrored butterflies in registers; the inverse takes
// the passes in the opposite order.
template <bool PAIR> __host__ __device__ constexpr int fix_radix(int n, int p) {
  int a = 0, b = 0;
  for (int m = n; m % 2 == 0; m /= 2) ++a;
  for (int m = n; m % 3 == 0; m /= 3) ++b;
  const int tail = PAIR && b == 0 ? 2 : 0;  // a closing radix 4
  a -= tail;
  int sixes = 0, least = 99;
  for (int c = 0; c <= a && c <= b; ++c) {
    const int passes = c + (b - c) + (a - c) / 3 + ((a - c) % 3 ? 1 : 0);
    const int cost =  // two per pass, one more for a lone radix 2
        2 * passes + ((a - c) % 3 == 1 && a - c < 4 ? 1 : 0);
    if (cost < least) {
      least = cost;
      sixes = c;
    }
  }
  a -= sixes;
  b -= sixes;
  int r[16] = {}, c = 0;
  const bool fours = a % 3 == 1 && a >= 4;
  for (int i = 0; i < (fours ? a / 3 - 1 : a / 3); ++i) r[c++] = 8;
  if (fours) {
    r[c++] = 4;
    r[c++] = 4;
  } else if (a % 3) {
    r[c++] = a % 3 == 1 ? 2 : 4;
  }
  for (int i = 0; i < sixes; ++i) r[c++] = 6;
  for (int i = 0; i < b; ++i) r[c++] = 3;
  if (tail) r[c++] = 4;
  return p < c ? r[p] : 0;
}
template <bool PAIR> __host__ __device__ constexpr int fix_npass(int n) {
  int p = 0;
  while (fix_radix<PAIR>(n, p)) ++p;
  return p;
}
// Pass p in execution order, its span and its twiddles' offset: entry (r, k),
// 1 <= r < radix, k < span, at twoff + (r - 1) span + k.
template <bool PAIR, bool INV> __host__ __device__ constexpr int fix_rad(int n, int p) {
  return fix_radix<PAIR>(n, INV && PAIR ? fix_npass<PAIR>(n) - 1 - p : p);
}
template <bool PAIR, bool INV> __host__ __device__ constexpr int fix_span(int n, int p) {
  int L = 1;
  for (int i = 0; i < p; ++i) L *= fix_rad<PAIR, INV>(n, i);
  return L;
}
template <bool PAIR, bool INV> __host__ __device__ constexpr int fix_twoff(int n, int p) {
  int o = 0;
  for (int i = 0; i < p; ++i) o += fix_span<PAIR, INV>(n, i) * (fix_rad<PAIR, INV>(n, i) - 1);
  return o;
}

// Whether the radix-3 passes divide by 2: in plans of five and more passes of radix
// 6 and 3 with two and more of radix 3 (243, 486, 729, 972, 1458, 1944, 2187, 2916;
// none has a compiled kernel).  Shorter plans lose nothing by 4, and 3888, with one
// radix-3 pass, gains nothing by 2.
template <bool PAIR> __host__ __device__ constexpr bool fix_halves(int n) {
  int threes = 0;
  for (int p = 0; p < fix_npass<PAIR>(n); ++p) threes += fix_radix<PAIR>(n, p) == 3;
  const int first = fix_radix<PAIR>(n, 0);
  return fix_npass<PAIR>(n) >= 5 && threes >= 2 && (first == 6 || first == 3);
}
// Kernels of their own, radix 6 and 3 only (a test per pass in the general ones would
// cost the other lengths 2 %): y at 64 x 729 x 64 103.6 us against 96.5 dividing by 4,
// x at 1458 x 64 x 64 105 us forward and 82 inverse against 125 and 86.
constexpr int kHalved = -1;  // (as a length)
// The bits that a pass p after the first divides by, and those of all of them.
template <bool PAIR, bool INV> __host__ __device__ constexpr int fix_div(int n, int p) {
  return fix_halves<PAIR>(n) && fix_rad<PAIR, INV>(n, p) == 3 ? 1 : 2;
}
template <bool PAIR, bool INV> __host__ __device__ constexpr int fix_drop(int n) {
  int d = 0;
  for (int p = 1; p < fix_npass<PAIR>(n); ++p) d += fix_div<PAIR, INV>(n, p);
  return d;
}

// ceil(log2) of the largest growth max(1, R_2/D_2, R_2 R_3/(D_2 D_3), ..) after the
// first pass.
template <bool PAIR, bool INV> __host__ __device__ constexpr int fix_growth(int n) {
  int lg = 0;
  double g = 1.0;
  for (int p = 1; p < fix_npass<PAIR>(n); ++p) {
    g *= (double)fix_rad<PAIR, INV>(n, p) / (1 << fix_div<PAIR, INV>(n, p));
    while (g > (double)(1 << lg)) ++lg;
  }
  return lg;
}

// Whether the sum over the line is worth its reduction: where the growth and the
// divisions take 7 bits or more, a line with one dominant value would otherwise
// keep fewer than a double's bits.
template <bool PAIR, bool INV> __host__ __device__ constexpr bool fix_uses_sum(int n) {
  return fix_growth<PAIR, INV>(n) + fix_drop<PAIR, INV>(n) >= 7;
}

// The lengths with kernels of their own (every radix, span and offset a constant:
// about half the time of the general ones): 2^a 3^b, b <= 3, from 16 to 2048.
#define CHANFS_FIX_LENGTHS                                                                  \
  CHANFS_FIX_LEN(16) CHANFS_FIX_LEN(18) CHANFS_FIX_LEN(24) CHANFS_FIX_LEN(32)               \
  CHANFS_FIX_LEN(36) CHANFS_FIX_LEN(48) CHANFS_FIX_LEN(54) CHANFS_FIX_LEN(64)               \
  CHANFS_FIX_LEN(72) CHANFS_FIX_LEN(96) CHANFS_FIX_LEN(108) CHANFS_FIX_LEN(128)             \
  CHANFS_FIX_LEN(144) CHANFS_FIX_LEN(192) CHANFS_FIX_LEN(216) CHANFS_FIX_LEN(256)           \
  CHANFS_FIX_LEN(288) CHANFS_FIX_LEN(384) CHANFS_FIX_LEN(432) CHANFS_FIX_LEN(512)           \
  CHANFS_FIX_LEN(576) CHANFS_FIX_LEN(768) CHANFS_FIX_LEN(864) CHANFS_FIX_LEN(1024)          \
  CHANFS_FIX_LEN(1152) CHANFS_FIX_LEN(1536) CHANFS_FIX_LEN(1728) CHANFS_FIX_LEN(2048)

// Shared-memory place of element e: one 16-byte element of padding per 8, so
// that the 8 lanes of a 128-byte access phase fall on different banks also in
// the first pass's stride-R writes.
__host__ __device__ constexpr int fix_pad(int e) { return e + (e >> 3); }

// exp(-+2 pi i e / n) in units of 2^-62, the low words signed.  The values of
// an eighth of the circle are computed once, in long double; the others are
// their reflections.
class FixRoots {
 public:
  explicit FixRoots(int n) : n_(n) {
    const long double half_pi = 1.57079632679489661923132169163975144L;
    for (int r = 0; 2 * r <= n; r += 4) add(half_pi * (long double)r / (long double)n);
    if (n % 4) {  // the remainders of 4 e / n run over more than multiples of 4
      cs_.clear();
      for (int r = 0; 2 * r <= n; ++r) add(half_pi * (long double)r / (long double)n);
    }
  }
  int4 at(long long e, bool conj) const {
    e %= n_;
    const long long q = 4 * e / n_, rest = 4 * e - q * n_;  // quarter turns, rest / n of the next
    const bool swap = 2 * rest > n_;
    const long long i = swap ? n_ - rest : rest;
    const longlong2 cs = cs_[n_ % 4 ? i : i / 4];
    const long long u = swap ? cs.y : cs.x, v = swap ? cs.x : cs.y;
    const long long re = q == 0 ? u : q == 1 ? -v : q == 2 ? -u : v;
    const long long im = q == 0 ? v : q == 1 ? u : q == 2 ? -v : -u;  // e^{+i angle}
    int4 w;
    split(re, &w.x, &w.y);
    split(conj ? im : -im, &w.z, &w.w);
    return w;
  }

 private:
  void add(long double a) {
    cs_.push_back(make_longlong2(llroundl(cosl(a) * 4611686018427387904.0L),
                                 llroundl(sinl(a) * 4611686018427387904.0L)));
  }
  static void split(long long x, int* hi, int* lo) {
    long long l = (long long)(int)(x & 0xffffffffll);
    if (l == -2147483648ll) l = -2147483647ll;  // its negative is used too
    *hi = (int)((x - l) >> 32);
    *lo = (int)l;
  }
  long long n_;
  std::vector<longlong2> cs_;
};

// (CHANFS_FIX_ON_HOST: a host test compiles the arithmetic with its own
// definitions of the intrinsics.)
#if defined(__CUDACC__) || defined(CHANFS_FIX_ON_HOST)

__device__ __forceinline__ Fix fadd(Fix a, Fix b) { return {a.x + b.x, a.y + b.y}; }
__device__ __forceinline__ Fix fsub(Fix a, Fix b) { return {a.x - b.x, a.y - b.y}; }
template <bool INV> __device__ __forceinline__ Fix frot(Fix a) {  // times -i (forward) or +i
  return INV ? Fix{-a.y, a.x} : Fix{a.y, -a.x};
}

__device__ __forceinline__ long long mad_wide(int a, int b, long long c) {
#ifdef __CUDA_ARCH__
  long long d;
  asm("mad.wide.s32 %0, %1, %2, %3;" : "=l"(d) : "r"(a), "r"(b), "l"(c));
  return d;
#else
  return (long long)((unsigned long long)((long long)a * b) + (unsigned long long)c);
#endif
}

// v = h 2^32 + l with a signed low word.
__device__ __forceinline__ int fix_lo(long long v) { return (int)v; }
__device__ __forceinline__ int fix_hi(long long v) {
  return (int)(v >> 32) + (int)((unsigned)(int)v >> 31);
}

// (sum << 2) with the two bits below it taken from the cross products.
__device__ __forceinline__ long long fix_join(long long sum, long long cross) {
  const unsigned sl = (unsigned)sum, sh = (unsigned)((unsigned long long)sum >> 32);
  const unsigned lo = __funnelshift_l((unsigned)cross, sl, 2);
  const unsigned hi = __funnelshift_l(sl, sh, 2);
  return (long long)(((unsigned long long)hi << 32) | lo);
}

// The products of a w for |a| <= 2^62: cross products (low by high words) from
// `start` up, then the high products, in units of 2^32 / 4, on top of those
// sums' high words by `carry`; the products of the two low words, below the last
// place, are left out.
template <class Carry>
__device__ __forceinline__ void fmul_sums(Fix a, int4 w, long long start, Carry carry,
                                          long long& sr, long long& si, long long& cr,
                                          long long& ci) {
  const int xl = fix_lo(a.x), xh = fix_hi(a.x), yl = fix_lo(a.y), yh = fix_hi(a.y);
  const int nh = -w.z, nl = -w.w;
  cr = mad_wide(xl, w.x, start);
  ci = mad_wide(xl, w.z, start);
  cr = mad_wide(xh, w.y, cr);
  ci = mad_wide(xh, w.w, ci);
  cr = mad_wide(yl, nh, cr);
  ci = mad_wide(yl, w.x, ci);
  cr = mad_wide(yh, nl, cr);
  ci = mad_wide(yh, w.y, ci);
  sr = mad_wide(xh, w.x, carry(cr));
  si = mad_wide(xh, w.z, carry(ci));
  sr = mad_wide(yh, nh, sr);
  si = mad_wide(yh, w.x, si);
}

// A pass's twiddled points are a w / 4 + kFixBias (1 + i), rounded to nearest:
// the cross products start at 2^63 (they stay within 2^62.5 of it), so their high
// word is unsigned and carries over without a sign extension.  The untwiddled
// point gets the same bias, and the DFT gathers it in its output 0, R times,
// where it is taken off.
constexpr long long kFixBias = 1ll << 31;
__device__ __forceinline__ Fix fmul4(Fix a, int4 w) {
  Fix s;
  long long cr, ci;
  fmul_sums(a, w, (long long)((1ull << 63) + (1ull << 31)),
            [](long long c) { return (long long)((unsigned long long)c >> 32); }, s.x, s.y, cr,
            ci);
  return s;
}
// The untwiddled point of a pass, a / 4, rounded: rounding down would add the
// same fraction to every butterfly, and the passes that follow would gather it
// in a few outputs.
__device__ __forceinline__ Fix fquarter(Fix a) {
  return {(a.x + (4 * kFixBias + 2)) >> 2, (a.y + (4 * kFixBias + 2)) >> 2};
}

// a w, rounded to nearest: two more bits, from the cross products.
__device__ __forceinline__ Fix fmul(Fix a, int4 w) {
  long long sr, si, cr, ci;
  fmul_sums(a, w, 1ll << 29, [](long long c) { return c >> 32; }, sr, si, cr, ci);
  return {fix_join(sr, cr), fix_join(si, ci)};
}

// v (1 + f) for a constant f = fh 2^-32 + fl 2^-64, |f| < 1/2.
__device__ __forceinline__ long long fix_scale1(long long v, int fh, int fl) {
  const int l = fix_lo(v), h = fix_hi(v);
  long long c = mad_wide(l, fh, 1ll << 31);
  c = mad_wide(h, fl, c);
  return mad_wide(h, fh, v + (c >> 32));
}
// 1/sqrt(2) - 1 and sqrt(3)/2 - 1 in units of 2^-64
__device__ __forceinline__ long long mul_rsqrt2(long long v) {
  return fix_scale1(v, -1257966796, -102865788);
}
__device__ __forceinline__ long long mul_sqrt3_2(long long v) {
  return fix_scale1(v, -575416509, -1033546850);
}

// Small DFTs, kernel e^{-2 pi i / R} forward, conjugate inverse.
template <bool INV> __device__ __forceinline__ void fdft3(Fix& a, Fix& b, Fix& c) {
  const Fix s = fadd(b, c), d = fsub(b, c);
  const Fix t = {a.x - s.x / 2, a.y - s.y / 2};  // (towards zero: no common sign)
  a = fadd(a, s);
  const Fix u = frot<INV>(Fix{mul_sqrt3_2(d.x), mul_sqrt3_2(d.y)});
  b = fadd(t, u);
  c = fsub(t, u);
}
template <bool INV> __device__ __forceinline__ void fdft4(Fix& a, Fix& b, Fix& c, Fix& d) {
  const Fix t0 = fadd(a, c), t1 = fsub(a, c), t2 = fadd(b, d), t3 = frot<INV>(fsub(b, d));
  a = fadd(t0, t2);
  b = fadd(t1, t3);
  c = fsub(t0, t2);
  d = fsub(t1, t3);
}
template <int R, bool INV> __device__ __forceinline__ void fdft(Fix* v) {
  if constexpr (R == 2) {
    const Fix t = fsub(v[0], v[1]);
    v[0] = fadd(v[0], v[1]);
    v[1] = t;
  } else if constexpr (R == 3) {
    fdft3<INV>(v[0], v[1], v[2]);
  } else if constexpr (R == 4) {
    fdft4<INV>(v[0], v[1], v[2], v[3]);
  } else if constexpr (R == 6) {  // 3 x 2 without twiddles (index maps modulo 6)
    fdft3<INV>(v[0], v[2], v[4]);
    fdft3<INV>(v[3], v[5], v[1]);
    const Fix a0 = v[0], a1 = v[2], a2 = v[4], b0 = v[3], b1 = v[5], b2 = v[1];
    v[0] = fadd(a0, b0);
    v[3] = fsub(a0, b0);
    v[4] = fadd(a1, b1);
    v[1] = fsub(a1, b1);
    v[2] = fadd(a2, b2);
    v[5] = fsub(a2, b2);
  } else {
    fdft4<INV>(v[0], v[2], v[4], v[6]);
    fdft4<INV>(v[1], v[3], v[5], v[7]);
    // W8 v3 = r (x + y, y - x) forward, r (x - y, x + y) inverse; W8^3 = -+i W8
    const Fix o1 = v[3], o3 = v[7];
    const long long p1 = mul_rsqrt2(INV ? o1.x - o1.y : o1.x + o1.y);
    const long long q1 = mul_rsqrt2(INV ? o1.x + o1.y : o1.y - o1.x);
    const long long p3 = mul_rsqrt2(INV ? o3.x + o3.y : o3.x - o3.y);
    const long long q3 = mul_rsqrt2(INV ? o3.x - o3.y : o3.x + o3.y);
    const Fix w1 = {p1, q1}, w3 = {-p3, INV ? q3 : -q3};
    const Fix w0 = v[1], w2 = frot<INV>(v[5]), e0 = v[0], e1 = v[2], e2 = v[4], e3 = v[6];
    v[0] = fadd(e0, w0);
    v[4] = fsub(e0, w0);
    v[1] = fadd(e1, w1);
    v[5] = fsub(e1, w1);
    v[2] = fadd(e2, w2);
    v[6] = fsub(e2, w2);
    v[3] = fadd(e3, w3);
    v[7] = fsub(e3, w3);
  }
}

// --- the scale of a line ----------------------------------------------------

// Adds |v| to a butterfly's maximum (as the high word of a double) and to its sum
// (as a float from the double's leading bits; values outside the range of
// floats are below every bound that the sum is used for, or switch it off).
__device__ __forceinline__ void fix_gather(double v, unsigned& top, float& sum) {
  const unsigned u = (unsigned)__double2hiint(v) & 0x7fffffffu;
  top = max(top, u);
  sum += __uint_as_float((max(u, 0x38100000u) - 0x38000000u) << 3);
}
__device__ __forceinline__ void fix_gather(double2 v, unsigned& top, float& sum) {
  fix_gather(v.x, top, sum);
  fix_gather(v.y, top, sum);
}

// A line's scale, and how its results leave.  kind 0: by a shift of the exponent;
// kind 1: by the library's scalbn (a line that was moved first, see fix_move); kind
// 2: an infinity or NaN (every output of the line is then NaN).
struct FixScale {
  int s, kind;
};

// Whether a line whose largest value has this high word is scaled as it is: within
// 2^+-90, where its sums fit the floats.
__device__ __forceinline__ bool fix_near(unsigned top) { return (top >> 20) - 933u <= 180u; }

// A line farther from 1 is moved first: all its values times 2^k, which brings its
// largest near 1, exactly (what that takes below the subnormals is below 2^-1000 of
// the largest).  So a power of two in the data comes out as that power of two, to
// the last bit.  A line of subnormals moves to 1 .. 2^52.  (The kernels
// do this in a call of their own.  With the moves among the code that every line runs,
// the x and y stages took 330 / 341 and 438 / 441 us at 512 x 384 x 384, y at 64 x 729 x
// 64 103; with the call 327 / 322, 428 / 436 and 63; with neither 324 / 333, 432 / 439
// and 96, the conversions then testing every value for the far cases.)
__device__ __forceinline__ int fix_move(unsigned top) {
  const int e = (int)(top >> 20);
  return fix_near(top) || e == 0x7ff ? 0 : e ? 1023 - e : 1074;
}
__device__ __forceinline__ double fix_moved(double v, int k) {  // |k| <= 1074
  const int h = k / 2;
  return v * __hiloint2double((1023 + h) << 20, 0) * __hiloint2double((1023 + k - h) << 20, 0);
}
__device__ __forceinline__ double2 fix_moved(double2 v, int k) {
  return k ? make_double2(fix_moved(v.x, k), fix_moved(v.y, k)) : v;
}
// Whether a line must be moved, as far as one thread knows: from its largest value,
// or, where that is 0 or below 2^-1042, from the thread's own.
template <int N> __device__ __forceinline__ bool fix_far(unsigned top, const double2* v) {
  if (top) return fix_move(top) != 0;
  int low = 0;
#pragma unroll
  for (int r = 0; r < N; ++r) low |= __double2loint(v[r].x) | __double2loint(v[r].y);
  return low != 0;
}

// A butterfly's sum in units of 2^-19 of the power of two above the largest one
// (integers add up to the same in any order); 0 if the line does not use it.
__device__ __forceinline__ unsigned fix_quanta(float sum, unsigned top, unsigned most) {
  if (!fix_near(top)) return 0u;
  return __float2uint_ru(sum * __uint_as_float((272u - ((most + 256u) >> 23)) << 23));
}

// The scale of a (moved) line, from its largest value (high word), largest butterfly
// sum B (float bits) and, unless it is 0, the sum of the butterflies' quanta.  A
// line of zeros takes s = 0.
__device__ __forceinline__ FixScale fix_scale_of(unsigned top, unsigned most, unsigned quanta,
                                                 int growth, int headroom, int div) {
  if (!fix_near(top)) return {0, top >= 0x7ff00000u ? 2 : 0};
  const int eb = (int)((most + 256u) >> 23) - 126;  // B < 2^eb
  int ec = eb + growth;
  // S / D_2 < 2^(eb - 19 + bits(quanta) - div)
  if (quanta) ec = max(eb, min(ec, eb + 13 - div - __clz((int)quanta)));
  return {headroom - ec, 0};
}
// The scale of the line before it was moved by 2^k.
__device__ __forceinline__ FixScale fix_moved_back(FixScale f, int k) {
  return {f.s + k, k ? 1 : f.kind};
}

static __device__ __noinline__ double fix_to_far(long long v, int s, int kind) {
  return kind == 2 ? __longlong_as_double(0x7ff8000000000000ll) : scalbn((double)v, -s);
}

// trunc(v 2^s): the significand, its leading bit at 62, shifted down.  (In a line
// with an infinity or NaN the shift may be out of range: any value will do.)
__device__ __forceinline__ long long fix_from(double v, int s) {
  const int hi = __double2hiint(v);
  const unsigned lo = (unsigned)__double2loint(v);
  const int t = 1085 - s - (int)(((unsigned)hi & 0x7fffffffu) >> 20);
  const unsigned mh = ((unsigned)hi & 0xfffffu) | 0x100000u;
  const unsigned long long m =
      ((((unsigned long long)__funnelshift_l(lo, mh, 10)) << 32) | (lo << 10)) >>
      min((unsigned)t, 63u);
  const long long sg = hi >> 31;
  return ((long long)m ^ sg) - sg;
}
__device__ __forceinline__ Fix fix_from(double2 v, int s) {
  return {fix_from(v.x, s), fix_from(v.y, s)};
}

// v 2^-s, rounded to nearest (the exponent is adjusted on the encoding).
__device__ __forceinline__ double fix_to(long long v, int s, int kind) {
  if (kind) return fix_to_far(v, s, kind);
  const double d = __ll2double_rn(v);
  const int hi = __double2hiint(d);
  return __hiloint2double(hi ? hi - (s << 20) : 0, __double2loint(d));
}
__device__ __forceinline__ double2 fix_to(Fix v, int s, int kind) {
  return make_double2(fix_to(v.x, s, kind), fix_to(v.y, s, kind));
}

// The DFT of a pass after the first: v[r] w[r - 1] / D, transformed.  (HALF, for
// radix 3, D = 2: whole products and sums, which stay below 3 x 2^61, then the
// division, towards zero: no common sign.)
template <int R, bool INV, bool HALF>
__device__ __forceinline__ void fix_twiddle_dft(Fix* v, const int4* __restrict__ tw, int stride) {
  if constexpr (HALF) {
#pragma unroll
    for (int r = 1; r < R; ++r) v[r] = fmul(v[r], __ldg(tw + (r - 1) * stride));
    fdft<R, INV>(v);
#pragma unroll
    for (int r = 0; r < R; ++r) v[r] = {v[r].x / 2, v[r].y / 2};
  } else {
    v[0] = fquarter(v[0]);
#pragma unroll
    for (int r = 1; r < R; ++r) v[r] = fmul4(v[r], __ldg(tw + (r - 1) * stride));
    fdft<R, INV>(v);
    v[0].x -= R * kFixBias;
    v[0].y -= R * kFixBias;
  }
}

// One Stockham radix-R butterfly: item j of a batch whose element e lives at
// at(e): points j + r q of `in`, twiddles (over D), DFT, positions (j - k) R + k
// + r L of `out`, k = j mod L.
template <int R, bool INV, bool HALF, class At>
__device__ __forceinline__ void fix_butterfly(const Fix* in, Fix* out, int j, int q, int L,
                                              const int4* __restrict__ tw, At at) {
  Fix v[R];
#pragma unroll
  for (int r = 0; r < R; ++r) v[r] = in[at(j + r * q)];
  const int k = j % L;
  fix_twiddle_dft<R, INV, HALF>(v, tw + k, L);
  const int o = (j - k) * R + k;
#pragma unroll
  for (int r = 0; r < R; ++r) out[at(o + r * L)] = v[r];
}

#endif

}  // namespace chanfs
