// FP64 numbers as seven balanced digits, for exact products on the FP16 tensor cores (the splitting of k_ozaki.cu, Ozaki,
// Ogita, Oishi and Rump, 2012, with balanced digits):
//   x = 2^(e - 57) F, F = round(x 2^(57 - e)) = sum_{i=1..7} d_i 256^(7 - i), |d_1| <= 512, -128 <= d_i <= 127
// where 2^e bounds |x|.  Products of digits i + j <= 9 are kept; the sums of equal i + j of up to TC_WIN 16 products are
// exact in FP32 (13 2^14 4 16 < 2^24) and move to 64-bit integers then.
#pragma once

namespace tlr {

constexpr int TC_P = 7;    // digits
constexpr int TC_WIN = 4;  // steps of 16 products of an exact window

// Exponent e with |x| < 2^e for the largest |x| whose high word is hw (1 for a zero column: any bound will do)
__device__ __forceinline__ int tc_exp(unsigned hw) { return hw == 0 ? 1 : (int)(hw >> 20) - 1022; }
// a column of tiny, huge or non-finite numbers
__device__ __forceinline__ bool tc_odd(int e) { return e < -900 || e > 900; }
// What tc_pairs takes of a column with |x| < 2^e (-900 <= e <= 900)
__device__ __forceinline__ int tc_shift(int e) { return (e + 1022) << 20; }
// |F| + 0x6600808080808080 as two words: the bytes are d_7 + 128, ..., d_2 + 128 and the FP16 number 1536 + d_1.
// Rounds to nearest; the sign of bad is set unless |x| < 2^e; zeros and denormals give 0.
__device__ __forceinline__ uint2 tc_digits(double x, int shift, int& bad) {
  const unsigned hi = (unsigned)__double2hiint(x), lo = (unsigned)__double2loint(x);
  // |x| 2^(58 - e) = (mantissa 2^5) >> (e + 1022 - exponent field)
  const int t = shift - (int)(hi & 0x7ff00000u);
  bad |= t;
  unsigned long long w = ((unsigned long long)((__funnelshift_l(lo, hi, 5) & 0x01ffffffu) | 0x02000000u) << 32) | (lo << 5);
  asm("shr.u64 %0, %0, %1;" : "+l"(w) : "r"((unsigned)t >> 20));  // 0 from 64 on
  w = (w + (2 * 0x6600808080808080ull + 1)) >> 1;
  return make_uint2((unsigned)w, (unsigned)(w >> 32));
}
__device__ __forceinline__ unsigned tc_fma2(unsigned a, unsigned b, unsigned c) {
  unsigned r;
  asm("fma.rn.f16x2 %0, %1, %2, %3;" : "=r"(r) : "r"(a), "r"(b), "r"(c));
  return r;
}
__device__ __forceinline__ unsigned tc_mul2(unsigned a, unsigned b) {
  unsigned r;
  asm("mul.rn.f16x2 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(b));
  return r;
}
__device__ __forceinline__ float tc_half(unsigned a, int high) {
  float r;
  asm("cvt.f32.f16 %0, %1;" : "=f"(r) : "h"((unsigned short)(high ? a >> 16 : a)));
  return r;
}
// the seven digit pairs of entries a, b with the signs of the high words sa, sb: FP16 (1024 + byte) s - (1024 + 128) s
__device__ __forceinline__ void tc_pairs(uint2 a, uint2 b, unsigned sa, unsigned sb, unsigned (&d)[TC_P]) {
  const unsigned p0 = __byte_perm(a.x, b.x, 0x5140u), p1 = __byte_perm(a.x, b.x, 0x7362u), p2 = __byte_perm(a.y, b.y, 0x5140u);
  const unsigned sg = __byte_perm(sa, sb, 0x7632u) & 0x80008000u;
  const unsigned one = 0x64646464u, s = sg ^ 0x3c003c00u, bias = sg ^ 0xe480e480u, bias1 = sg ^ 0xe600e600u;
  d[6] = tc_fma2(__byte_perm(p0, one, 0x4140u), s, bias);  // byte 0: the least significant digit
  d[5] = tc_fma2(__byte_perm(p0, one, 0x4342u), s, bias);
  d[4] = tc_fma2(__byte_perm(p1, one, 0x4140u), s, bias);
  d[3] = tc_fma2(__byte_perm(p1, one, 0x4342u), s, bias);
  d[2] = tc_fma2(__byte_perm(p2, one, 0x4140u), s, bias);
  d[1] = tc_fma2(__byte_perm(p2, one, 0x4342u), s, bias);
  d[0] = tc_fma2(__byte_perm(a.y, b.y, 0x7632u), s, bias1);
}
// Group sums of a window; the totals: hi of the groups 0-3, lo of 4-7 (weights 256^-g); est: estimates of the sums of
// |x y|, FP16 in the layout of the products, 2^11 for the product of the two bounds (infinite past 2^5 of them).  The
// estimate multiplies the leading digits: nothing of a number below 2^-10 of its bound, at most twice a larger one.
//
// What an estimate has to reach for a result to be as accurate as an FP64 sum: K terms x y in units of the two bounds are
// off by the roundings of x and y, 2^-58 / sqrt(3) in the mean square each, so the result by
// 2^-58.8 sqrt(sum x^2 + y^2), up to 2^-58.3 sqrt(K) and for entries spread over their range about 2^-60 sqrt(K); an FP64
// sum by 2^-53 / sqrt(3) of its size s from its last rounding and about as much again from the others.  Hence
// s >= sqrt(K) / 64 (tc_least; in the worst case, all roundings of one sign, K 2^-57 against FP64's K 2^-53 s).
struct TcAcc {
  float f[8][4];
  long long hi[4], lo[4];
  unsigned est[2];
  int win, bad;
};
__host__ __device__ __forceinline__ float tc_least(float K) { return 32.f * sqrtf(K); }  // in the estimates' units
// |leading digits|, of the second factor times 2^-7
__device__ __forceinline__ unsigned tc_abs2(unsigned d) { return d & 0x7fff7fffu; }
__device__ __forceinline__ unsigned tc_abs2s(unsigned d) { return tc_mul2(d & 0x7fff7fffu, 0x20002000u); }
__device__ __forceinline__ void tc_init(TcAcc& a) {
#pragma unroll
  for (int c = 0; c < 4; ++c) {
    a.hi[c] = a.lo[c] = 0;
#pragma unroll
    for (int g = 0; g < 8; ++g) a.f[g][c] = 0.f;
  }
  a.est[0] = a.est[1] = 0;
  a.win = a.bad = 0;
}
__device__ __forceinline__ void tc_drain(TcAcc& a) {
#pragma unroll
  for (int c = 0; c < 4; ++c) {
    long long h = 0, l = 0;
#pragma unroll
    for (int g = 0; g < 4; ++g) {
      h = h * 256 + __float2int_rn(a.f[g][c]);
      l = l * 256 + __float2int_rn(a.f[g + 4][c]);
      a.f[g][c] = a.f[g + 4][c] = 0.f;
    }
    a.hi[c] += h;
    a.lo[c] += l;
  }
  a.win = 0;
}
// value of a total: digits i, j carry 2^(-1 - 8 i) each (i, j from 1): group g = i + j - 2 carries 2^(-18 - 8 g)
__device__ __forceinline__ double tc_value(long long hi, long long lo, int e) {
  return ldexp(fma((double)hi, 4294967296.0, (double)lo), e - 74);
}

}  // namespace tlr
