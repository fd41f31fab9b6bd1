// 64-bit block fixed point: the line transforms of the FP64 path on the integer units (sm_103a).
//
// The chip issues two FP64 operations per SM and cycle and 64 to 128 integer ones, so a line FFT
// in FP64 spends 16 cycles of an SM per warp instruction whatever else the kernel does.  Here a
// line's values are 64-bit integers v with one exponent e per line, value = v 2^e: an addition is
// two integer instructions, a product with a twiddle three 32 x 32 -> 64 multiply-adds.
//
// Precision.  Every value keeps |v| <= 2^61; a transform over K inputs is entered at
// |v| < 2^61 / ((4/pi) K), so nothing overflows, and rounds to nearest at one unit: 2^-57 to 2^-55
// of the line's largest input, where FP64 rounds every operand at 2^-53 of itself.  After EVERY
// transform the line is shifted back up to 2^61 and its exponent adjusted (fx_top, fx_up): a
// transform's outputs lie up to six bits below the headroom it was given, and a following one that
// is entered at its own headroom would round them away.
//
// Inf and NaN: a line that holds one has exponent kFxBad and is NaN as a whole when it is
// converted back, as the transform of such a line is.  Results beyond the range of a double are
// Inf; subnormal inputs and results are kept.
#pragma once
#include "common.cuh"

namespace ll {

struct fx64 {
  long long v;
  __host__ __device__ __forceinline__ fx64() {}
  __host__ __device__ __forceinline__ explicit constexpr fx64(long long a) : v(a) {}
};
__host__ __device__ __forceinline__ fx64 add_rn(fx64 a, fx64 b) { return fx64(a.v + b.v); }
__host__ __device__ __forceinline__ fx64 operator-(fx64 a) { return fx64(-a.v); }
__host__ __device__ __forceinline__ fx64 operator+(fx64 a, fx64 b) { return fx64(a.v + b.v); }

constexpr int kFxBad = 1 << 20;       // exponent of a line with an Inf or a NaN (sums stay above kFxBad / 2)

// A factor w, |w| <= 1, as w = (h + l 2^-31) 2^-31 with |l| <= 2^30 (h = 2^31 - 1, l = 2^31 - 1 for
// w = 1).  A twiddle holds -y too: both occur in a complex product.
struct FxTw { int xh, xl, yh, yl, nh, nl; };
__host__ __device__ __forceinline__ FxTw conj_tw(FxTw w) { return FxTw{w.xh, w.xl, w.nh, w.nl, w.yh, w.yl}; }

// a * w for the split a = ah 2^31 + al: ah wh + (ah wl + al wh) 2^-31, the middle sum rounded (the
// product of the low parts is below half a unit).  |a| <= 2^61 and |w| <= 1 (a complex factor's
// modulus) keep the middle sum below 2^63.
__host__ __device__ __forceinline__ int fx_hi(fx64 a) { return (int)(a.v >> 31); }
__host__ __device__ __forceinline__ int fx_lo(fx64 a) { return (int)(a.v & 0x7fffffff); }
__host__ __device__ __forceinline__ fx64 fx_mul(fx64 a, int wh, int wl) {
  const int h = fx_hi(a), l = fx_lo(a);
  const long long t = (1LL << 30) + (long long)h * wl + (long long)l * wh;
  return fx64((t >> 31) + (long long)h * wh);
}
// the complex product with w = (xh, xl) + i (yh, yl), (nh, nl) = -y
__host__ __device__ __forceinline__ cplx<fx64> cmul_rn(cplx<fx64> a, FxTw w) {
  const int xh = fx_hi(a.x), xl = fx_lo(a.x), yh = fx_hi(a.y), yl = fx_lo(a.y);
  const long long tr = (1LL << 30) + (long long)xh * w.xl + (long long)yh * w.nl + (long long)xl * w.xh + (long long)yl * w.nh;
  const long long ti = (1LL << 30) + (long long)xh * w.yl + (long long)yh * w.xl + (long long)xl * w.yh + (long long)yl * w.xh;
  return mk(fx64((tr >> 31) + (long long)xh * w.xh + (long long)yh * w.nh),
            fx64((ti >> 31) + (long long)xh * w.yh + (long long)yh * w.xh));
}
// SIGN i w
template <int SIGN> __host__ __device__ __forceinline__ FxTw turn_tw(FxTw w) {
  return SIGN > 0 ? FxTw{w.nh, w.nl, w.xh, w.xl, -w.xh, -w.xl} : FxTw{w.yh, w.yl, -w.xh, -w.xl, w.xh, w.xl};
}
template <int SIGN> __host__ __device__ __forceinline__ void third(cplx<fx64> a, cplx<fx64> sum, cplx<fx64> dif, cplx<fx64>* v) {
  // sqrt(3)/2 in limbs
  constexpr int sh = 1859775393, sl = 815355111;
  const long long mx = a.x.v - ((sum.x.v + 1) >> 1), my = a.y.v - (sum.y.v >> 1);
  const long long dx = fx_mul(dif.x, sh, sl).v, dy = fx_mul(dif.y, sh, sl).v;
  v[1] = SIGN > 0 ? mk(fx64(mx - dy), fx64(my + dx)) : mk(fx64(mx + dy), fx64(my - dx));
  v[2] = SIGN > 0 ? mk(fx64(mx + dy), fx64(my - dx)) : mk(fx64(mx - dy), fx64(my + dx));
}
__device__ __forceinline__ cplx<fx64> shfl_pair(cplx<fx64> v, unsigned mask) {
  return mk(fx64(__shfl_xor_sync(mask, v.x.v, 1)), fx64(__shfl_xor_sync(mask, v.y.v, 1)));
}

// limbs of the signed 62-bit fraction w 2^-62
__host__ __device__ __forceinline__ void fx_limbs(long long w, int& h, int& l) {
  const long long t = (w + (1LL << 30)) >> 31;
  h = (int)t;
  l = (int)(w - (t << 31));
}

// The limbs of exp(-2 pi i e / n) (x, y, -y) in exact integer arithmetic: the angle reduced to an
// eighth of a turn, the Taylor series in 64-bit fractions.
static inline void fx_twiddle_limbs(int e, int n, int* out) {
  const int q = 4 * e / n, r = 4 * e - q * n;   // angle = (pi/2) (q + r/n)
  const bool swap = 2 * r > n;
  const unsigned __int128 half_pi = ((unsigned __int128)1 << 64) | 0x921FB54442D18469ull;   // pi/2 in 64-bit fractions
  const uint64_t x = (uint64_t)(half_pi * (unsigned)(swap ? n - r : r) / (unsigned)n);
  auto mul = [](uint64_t a, uint64_t b) { return (uint64_t)(((unsigned __int128)a * b) >> 64); };
  unsigned __int128 c = (unsigned __int128)1 << 64, s = x;
  uint64_t term = x;                             // x^k / k!
  for (int k = 2; k < 24 && term; ++k) {
    term = mul(term, x) / (unsigned)k;
    if (k % 4 == 2) c -= term;
    if (k % 4 == 3) s -= term;
    if (k % 4 == 0) c += term;
    if (k % 4 == 1) s += term;
  }
  long long cc = (long long)((c + 2) >> 2), ss = (long long)((s + 2) >> 2);   // 2^-62
  if (swap) { const long long t = cc; cc = ss; ss = t; }
  const long long co[4] = {cc, -ss, -cc, ss}, si[4] = {ss, cc, -ss, -cc};     // cos, sin of the angle
  const long long w[3] = {co[q & 3], -si[q & 3], si[q & 3]};
  for (int i = 0; i < 3; ++i) {
    const long long one = 1LL << 62;
    if (w[i] >= one) out[2 * i] = out[2 * i + 1] = 0x7fffffff;                // 1 - 2^-62
    else fx_limbs(w[i], out[2 * i], out[2 * i + 1]);
  }
}

// ---- doubles ------------------------------------------------------------------------------
// A transform over k inputs is entered at |v| < 2^(61 - growth).  An output's real part is a sum of
// k terms re cos - im sin: at most (4/pi) k times the largest input, the mean of |cos| + |sin| over
// equally spaced angles with 0 among them being at most 4/pi (a trapezoid rule on a concave
// function).  What lies between (a twiddled transform over a half or a third of the inputs, up to
// two of its terms) stays below sqrt(2) (2/3) k.  ceil(log2 (4/pi) k), with 4% to spare for the
// roundings at every side.
__host__ __device__ constexpr int fx_growth(int k) {
  int g = 1;
  while ((1L << g) * 10000 < 12733L * k) ++g;
  return g;
}
__host__ __device__ __forceinline__ int fx_hiword(long long bits) { return (int)(bits >> 32); }
// sign and fraction of the double `bits` as an integer below 2^(53 + s0), rounded to nearest, in a
// line whose largest biased exponent is E >= 1 (subnormals have exponent 1 and no leading bit);
// the line's exponent is fx_exp(E, s0)
__host__ __device__ __forceinline__ long long fx_from(long long bits, int E, int s0) {
  const int ex = (int)(bits >> 52) & 0x7ff;
  const long long m = ((bits & 0xfffffffffffffLL) | ((long long)(ex > 0) << 52)) << s0;
  const int sh = E - (ex > 1 ? ex : 1);
  const long long r = sh > 62 ? 0 : (m + ((1LL << sh) >> 1)) >> sh;
  return bits < 0 ? -r : r;
}
__host__ __device__ __forceinline__ int fx_exp(int E, int s0) { return E == 0x7ff ? kFxBad : E - 1075 - s0; }
// v 2^e as a double, rounded to nearest (a tie away from zero)
__host__ __device__ __forceinline__ long long fx_bits(long long v, int e) {
  if (e > kFxBad / 2) return 0x7ff8000000000000LL;
  const unsigned long long u = v < 0 ? 0ull - (unsigned long long)v : (unsigned long long)v;
#ifdef __CUDA_ARCH__
  const int lz = __clzll((long long)u);
#else
  const int lz = u ? __builtin_clzll(u) : 64;
#endif
  const int be = 63 + 1023 + e - lz;   // biased exponent of the leading bit
  const unsigned long long n = u << (lz & 63);
  const int sh = 11 + (be < 1 ? 1 - be : 0);   // a subnormal result keeps fewer bits
  const unsigned long long m = (sh < 64 ? n >> sh : 0) + (sh < 65 ? (n >> (sh - 1)) & 1 : 0);
  long long r = ((long long)(be < 1 ? 0 : be - 1) << 52) + (long long)m;
  if (be > 2046) r = 0x7ff0000000000000LL;
  if (u == 0) r = 0;
  return v < 0 ? (r | (long long)0x8000000000000000ull) : r;
}
// limbs of a factor: the double as a fraction below 1/2 of 2^e, e = fx_coef_exp(E) (E: the largest
// biased exponent among the factors)
__host__ __device__ __forceinline__ void fx_coef(long long bits, int E, int& h, int& l) { fx_limbs(fx_from(bits, E, 8), h, l); }
__host__ __device__ __forceinline__ int fx_coef_exp(int E) { return fx_exp(E, 8) + 62; }

// ---- a line in registers: H points of this lane, P lanes (mask: the pair) --------------------
// The largest biased exponent of a line that holds doubles' bits (at least 1).
template <int P, int H>
__device__ __forceinline__ int fx_line_exp(const cplx<fx64> (&l)[H], unsigned mask) {
  int m = 0;
#pragma unroll
  for (int i = 0; i < H; ++i) m = max(m, max(fx_hiword(l[i].x.v) & 0x7fffffff, fx_hiword(l[i].y.v) & 0x7fffffff));
  if (P == 2) m = max(m, __shfl_xor_sync(mask, m, 1));
  return max(m >> 20, 1);
}
// doubles' bits -> fixed point at 2^(53 + S0)
template <int S0, int H>
__device__ __forceinline__ void fx_line_from(cplx<fx64> (&l)[H], int E) {
#pragma unroll
  for (int i = 0; i < H; ++i) l[i] = mk(fx64(fx_from(l[i].x.v, E, S0)), fx64(fx_from(l[i].y.v, E, S0)));
}
// The left shift that brings a line's largest value to 2^60 .. 2^61.
template <int P, int H>
__device__ __forceinline__ int fx_top(const cplx<fx64> (&l)[H], unsigned mask) {
  int m = 0;
#pragma unroll
  for (int i = 0; i < H; ++i) {
    const int a = fx_hiword(l[i].x.v), b = fx_hiword(l[i].y.v);
    m |= (a ^ (a >> 31)) | (b ^ (b >> 31));
  }
  if (P == 2) m |= __shfl_xor_sync(mask, m, 1);
  return max(__clz(m) - 3, 0);
}
// shifted left by c, then right by G with rounding
template <int G, int H>
__device__ __forceinline__ void fx_up(cplx<fx64> (&l)[H], int c) {
#pragma unroll
  for (int i = 0; i < H; ++i) {
    l[i] = mk(fx64(l[i].x.v << c), fx64(l[i].y.v << c));
    if constexpr (G > 0) l[i] = mk(fx64((l[i].x.v + (1LL << (G - 1))) >> G), fx64((l[i].y.v + (1LL << (G - 1))) >> G));
  }
}
// right by s >= 1 with rounding (s > 62: 0)
__device__ __forceinline__ cplx<fx64> fx_down(cplx<fx64> a, int s) {
  const long long half = 1LL << (s - 1);
  return mk(fx64((a.x.v + half) >> s), fx64((a.y.v + half) >> s));
}

}  // namespace ll
