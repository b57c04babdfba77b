// dig.cuh -- matrix products of FP64 accuracy on the tensor cores: fixed-point digits.
//
// The FP64 pipe of a GB300 does 0.53 T multiply-adds per second; its tensor cores do 300 T per
// second on FP16 operands through mma.sync (measured with register-resident operands).  A product
// of FP64 matrices is therefore formed from products of short integers, the method of Ozaki,
// Ogita, Oishi and Rump (Numer. Algorithms 59, 2012) in the tensor-core form of Mukunoki et al.
// (ISC 2020):
//   - the values of a row (or matrix) are scaled by a common power of two to integers X of 61 to
//     62 bits, exact for every value within 2^-8 of the largest one and within 2^-61 of the
//     largest one otherwise;
//   - X = sum_i d_i 256^i with eight balanced digits d_i in [-128, 127];
//   - a product of two digits fits 14 bits plus sign, and the products of one level i + j
//     accumulate exactly in an FP32 accumulator as long as their sum stays within 2^24: at most
//     eight pairs per level times DIG_FLUSH = 128 products along k;
//   - the levels are added in two 64-bit integers (every DIG_FLUSH products) and the result is
//     rounded once, to its own leading bits (a sum cut at a fixed 2^-52 of the product of the maxima
//     was further off than FP64 where the largest values do not meet).
// Operands are cut (toward zero) at their last bit, and eight levels (36 of the 64 digit products) leave out
// up to 2^-57 of the product of the two maxima per term, 2^-60 on average and of either sign; an FP64 sum of
// K products rounds K times at 2^-53 of its partial sums.  These errors are relative to the operands' largest
// elements: where all products of a sum are many octaves smaller, the kernels sum in FP64 (ph.cu PH_SPAN,
// iterate.cu PP_FAR).  Measured from MBPT2 amplitudes, largest error of an element's own sum of absolute
// products: ladder N = 66, n^2 <= 14, 2.8e-15 against 3.2e-15 in FP64; ph term 6.0e-16 against 1.1e-15.
// Seven levels (28 products) drop terms below 2^-54, which left the FP32-pair results, whose 48 bits
// would allow it, further from the exact ladder than FP32-pair arithmetic (1.8e-14 against 1.4e-14 of
// the norm: the interaction spans many orders of magnitude, its maximum is far above its mean).
// A digit word stores X + 0x8080808080808080: byte i is d_i + 128.  Matrices that are read once
// per product are kept as the words of two elements interleaved by digit (16 bytes, the most
// significant digits first), so that one byte permutation brings a digit of both elements into
// FP16 position: 0x6400 | b is 1024 + b, and subtracting 1152 leaves d.  Matrices read by many
// warps are kept as FP16 digits.
#pragma once
#include <cuda_fp16.h>

#include <type_traits>

#include "pnm_internal.cuh"

typedef unsigned long long dig_t;
constexpr dig_t DIG_BIAS = 0x8080808080808080ull;  // the word of zero
constexpr int DIG_LEVELS = 8;
constexpr int DIG_FLUSH = 128;                      // products along k between two integer drains
constexpr int DIG_NONFINITE = 0x7ff;                // exponent of a set with an infinity or a NaN

// Biased exponent of x, at least 1 (0x7ff for infinities and NaN); |x| < 2^(exponent - 1022).
__device__ __forceinline__ int dig_exp(double x) { return max((__double2hiint(x) >> 20) & 0x7ff, 1); }

// x 2^(61 - (e - 1022)) truncated to an integer, for dig_exp(x) <= e: |result| < 2^61.
__device__ __forceinline__ long long dig_fixed(double x, int e) {
  const int hi = __double2hiint(x), ex = (hi >> 20) & 0x7ff;
  const unsigned mh = (hi & 0xfffff) | (ex ? 0x100000 : 0);
  const long long m = (long long)(((dig_t)mh << 32) | (unsigned)__double2loint(x));
  const long long a = (m << 8) >> min(e - max(ex, 1), 63);
  return hi < 0 ? -a : a;
}

// The leading 16 bits of a magnitude among those an integer of its scale can have.
__device__ __forceinline__ unsigned dig_top(long long x) { return (unsigned)((x < 0 ? -x : x) >> 46); }

__device__ __forceinline__ dig_t dig_word(long long x) { return (dig_t)x + DIG_BIAS; }

// s 2^p rounded to FP64, without the FP64 pipe where the result is a normal number.
__device__ __forceinline__ double dig_to_double(long long s, int p) {
  if (s == 0) return 0.0;
  const dig_t a = s < 0 ? (dig_t)0 - (dig_t)s : (dig_t)s;
  const int z = __clzll((long long)a);
  const int e = p + 63 - z + 1023;
  if (e < 1 || e > 2045) return scalbn((double)s, p);
  // the leading bit adds one to the exponent field; rounding may carry into it
  const dig_t m = ((a << z) >> 11) + (((a << z) >> 10) & 1);
  return __longlong_as_double((long long)((((dig_t)(e - 1)) << 52) + m) | (s & (long long)0x8000000000000000ull));
}

// s 2^p as an FP32 pair: rounded to 24 bits, and the rest to 24 more.
__device__ __forceinline__ f2 dig_to_f2(long long s, int p) {
  if (s == 0) return f2{0.0f, 0.0f};
  const dig_t a = s < 0 ? (dig_t)0 - (dig_t)s : (dig_t)s;
  const int z = __clzll((long long)a);
  const dig_t m = a << z;
  auto scaled = [](float v, int e) {  // v 2^e
    return e < -126 ? 0.0f : v * __int_as_float((min(e, 127) + 127) << 23);
  };
  const unsigned top = (unsigned)(m >> 40) + (unsigned)((m >> 39) & 1);
  const long long rest = (long long)(m - ((dig_t)top << 40));  // within 2^39; top 2^24 wraps around
  const float h = scaled(__uint2float_rn(top), p - z + 40), l = scaled(__int2float_rn((int)(rest >> 8)), p - z + 8);
  return s < 0 ? f2{-h, -l} : f2{h, l};
}

template <typename Out>
__device__ __forceinline__ Out dig_out(long long s, int p) {
  if constexpr (std::is_same<Out, f2>::value) return dig_to_f2(s, p);
  else return dig_to_double(s, p);
}

// The words of two elements interleaved: 32-bit part r holds the digits 2r and 2r + 1 (from the
// most significant) of both.
__device__ __forceinline__ uint4 dig_interleave(dig_t w0, dig_t w1) {
  const uint32_t h0 = (uint32_t)(w0 >> 32), h1 = (uint32_t)(w1 >> 32), l0 = (uint32_t)w0, l1 = (uint32_t)w1;
  return make_uint4(__byte_perm(h0, h1, 0x6273), __byte_perm(h0, h1, 0x4051), __byte_perm(l0, l1, 0x6273),
                    __byte_perm(l0, l1, 0x4051));
}
// FP16 digits (two elements: low and high half) of an interleaved pair: out[j] is digit j from the
// most significant.
template <int COUNT>
__device__ __forceinline__ void dig_expand(uint4 v, uint32_t (&out)[COUNT]) {
  const uint32_t p[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
  for (int j = 0; j < COUNT; j++) {
    const uint32_t x = __byte_perm(p[j >> 1], 0x64646464u, (j & 1) ? 0x4342 : 0x4140);
    const __half2 h = __hsub2(*reinterpret_cast<const __half2*>(&x), __half2half2(__ushort_as_half(0x6480)));
    out[j] = *reinterpret_cast<const uint32_t*>(&h);
  }
}
// The same for element k of the pair v (low half) and of the pair w (high half).
__device__ __forceinline__ void dig_expand_across(uint4 v, uint4 w, int k, uint32_t (&out)[DIG_LEVELS]) {
  const uint32_t p[4] = {v.x, v.y, v.z, v.w}, q[4] = {w.x, w.y, w.z, w.w};
  const uint32_t even = 0x0400u + 0x0101u * k, odd = even + 0x0202u;
#pragma unroll
  for (int j = 0; j < DIG_LEVELS; j++) {
    const uint32_t x = (__byte_perm(p[j >> 1], q[j >> 1], (j & 1) ? odd : even) & 0x00ff00ffu) | 0x64006400u;
    const __half2 h = __hsub2(*reinterpret_cast<const __half2*>(&x), __half2half2(__ushort_as_half(0x6480)));
    out[j] = *reinterpret_cast<const uint32_t*>(&h);
  }
}

__device__ __forceinline__ void dig_mma16(float (&d)[4], const uint32_t a0, const uint32_t a1, const uint32_t a2,
                                          const uint32_t a3, const uint32_t b0, const uint32_t b1) {
  asm volatile(
      "mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3},{%4,%5,%6,%7},{%8,%9},{%0,%1,%2,%3};"
      : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
      : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}

__device__ __forceinline__ void dig_mma8(float (&d)[4], const uint32_t a0, const uint32_t a1, const uint32_t b0) {
  asm volatile("mma.sync.aligned.m16n8k8.row.col.f32.f16.f16.f32 {%0,%1,%2,%3},{%4,%5},{%6},{%0,%1,%2,%3};"
               : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
               : "r"(a0), "r"(a1), "r"(b0));
}
// The 36 digit products of a 16 x 8 x 16 block (half: of its first 8 columns along k).
__device__ __forceinline__ void dig_block(float (&acc)[DIG_LEVELS][4], const uint32_t (&a)[4][DIG_LEVELS],
                                          const uint32_t (&b)[2][DIG_LEVELS], bool half) {
  if (half) {
#pragma unroll
    for (int i = 0; i < DIG_LEVELS; i++)
#pragma unroll
      for (int j = 0; i + j < DIG_LEVELS; j++) dig_mma8(acc[i + j], a[0][i], a[1][i], b[0][j]);
  } else {
#pragma unroll
    for (int i = 0; i < DIG_LEVELS; i++)
#pragma unroll
      for (int j = 0; i + j < DIG_LEVELS; j++)
        dig_mma16(acc[i + j], a[0][i], a[1][i], a[2][i], a[3][i], b[0][j], b[1][j]);
  }
}

// An exact sum hi 2^32 + lo of digit products in units of 256^7 256^0 (the lowest level kept).
struct DigSum {
  long long hi, lo;
};

// sum_l acc_l 256^(7 - l) of accumulator element e: acc_l holds level l (the pairs of digits whose
// distances from the top add up to l).
__device__ __forceinline__ DigSum dig_drain(const float (&acc)[DIG_LEVELS][4], int e) {
  long long hi = 0, lo = 0;
#pragma unroll
  for (int l = 0; l < 4; l++) {
    hi = hi * 256 + (long long)__float2int_rn(acc[l][e]);
    lo = lo * 256 + (long long)__float2int_rn(acc[l + 4][e]);
  }
  return DigSum{hi, lo};
}

// The same for accumulators within 2^22, sums of at most DIG_SMALL_K products (level 7 has six
// pairs of full digits and two with a leading digit, of at most 65 and 92 in magnitude): adding
// 1.5 2^23 leaves the integer in the low bits of the float, an FMA-pipe addition instead of a
// conversion at an eighth of its rate, and two levels fit 32 bits.
constexpr int DIG_SMALL_K = 35;
__device__ __forceinline__ DigSum dig_drain_small(const float (&acc)[DIG_LEVELS][4], int e) {
  int p[4];
#pragma unroll
  for (int l = 0; l < 4; l++) {
    // both floats carry the bits 0x4b400000: 257 of them in the sum, modulo 2^32
    const unsigned a = __float_as_uint(acc[2 * l][e] + 12582912.0f), b = __float_as_uint(acc[2 * l + 1][e] + 12582912.0f);
    p[l] = (int)(a * 256u + b - 0x4b400000u * 257u);
  }
  return DigSum{(long long)p[0] * 65536 + p[1], (long long)p[2] * 65536 + p[3]};
}

// x + y in units of lo.
__device__ __forceinline__ DigSum dig_add_low(DigSum x, long long y) {
  return DigSum{x.hi + (y >> 32), x.lo + (y & 0xffffffffll)};
}

// The sum as m 2^shift with the 62 leading bits in m (shift 0: exact).
__device__ __forceinline__ long long dig_leading(DigSum x, int& shift) {
  x.hi += x.lo >> 32;
  x.lo &= 0xffffffffll;
  const long long a = x.hi < 0 ? -x.hi : x.hi;
  shift = max(0, 34 - __clzll(a));  // |hi| < 2^30 leaves room for all of lo
  return (x.hi << (32 - shift)) + (x.lo >> shift);
}

// The sum scaled by 2^p as a result.
template <typename Out>
__device__ __forceinline__ Out dig_result(DigSum x, int p) {
  int shift;
  const long long m = dig_leading(x, shift);
  return dig_out<Out>(m, p + shift);
}

// Power of two of the unit of a sum: the operands' integers carry 2^(61 - (e - 1022)) each, the
// levels are counted from 256^7 256^7 = 2^112 down to 2^56.
__device__ __forceinline__ int dig_power(int ea, int eb) { return 56 - 122 + (ea + eb - 2044); }

// The antisymmetrized Minnesota element of v_minnesota_as as an integer, from the table of the
// Gaussians as integers of one scale (interleaved R, T, S with protons, as the FP64 table): sums
// of table entries with small integer weights, exact.  The states conserve momentum.
__device__ __forceinline__ long long v_minnesota_fixed(char4 p, char4 q, char4 r, char4 s,
                                                       const long long* __restrict__ xlut) {
  const int d1 = dot3(p.x - r.x, p.y - r.y, p.z - r.z), d2 = dot3(p.x - s.x, p.y - s.y, p.z - s.z);
  if (p.w <= 1 && p.w >= -1) {
    const int sf = (p.w == r.w && q.w == s.w) - (p.w == s.w && q.w == r.w);
    const long long v = xlut[d1] + xlut[d2];
    return sf > 0 ? v : (sf < 0 ? -v : 0);
  }
  auto tz = [](int w) { return w > 0 ? 1 : -1; };
  const int tp = tz(p.w), tq = tz(q.w), tr = tz(r.w), ts = tz(s.w);
  const int sp = p.w - 4 * tp, sq = q.w - 4 * tq, sr = r.w - 4 * tr, ss = s.w - 4 * ts;
  const int one = (sp == sr && sq == ss && tp == tr && tq == ts), ps = (sp == ss && sq == sr && tp == tr && tq == ts);
  const int pt = (sp == sr && sq == ss && tp == ts && tq == tr), pst = (sp == ss && sq == sr && tp == ts && tq == tr);
  const int cR = 2 * (one - pst), cT = one + ps - pt - pst, cS = one - ps + pt - pst;
  const long long *x1 = xlut + 3 * d1, *x2 = xlut + 3 * d2;
  return (cR * (x1[0] + x2[0]) + cT * (x1[1] + x2[1]) + cS * (x1[2] + x2[2])) >> 1;
}

// Stage the interaction table of one system as integers (all threads of the CTA); returns the
// exponent of their scale, which bounds every element: two table entries for neutrons, with
// protons half the sum of six entries of weights up to two.  Leaves a barrier to the caller.
__device__ __forceinline__ int stage_fixed_lut(const double* __restrict__ lut, int elems, bool protons,
                                               long long* __restrict__ xlut, int* sh_max) {
  if (threadIdx.x == 0) *sh_max = 1;
  __syncthreads();
  int e = 1;
  for (int m = threadIdx.x; m < elems; m += blockDim.x) e = max(e, dig_exp(lut[m]));
  atomicMax(sh_max, e);
  __syncthreads();
  e = *sh_max;
  if (e >= DIG_NONFINITE) return DIG_NONFINITE;
  e += protons ? 3 : 1;
  for (int m = threadIdx.x; m < elems; m += blockDim.x) xlut[m] = dig_fixed(lut[m], e);
  return e;
}
