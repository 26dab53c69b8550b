// FP64 Legendre stages on the tensor cores, by digit slices.
//
// On this GPU the FP64 pipe runs at 1/64 of the FP32 rate, so a Legendre
// stage whose sums are FP64 fused multiply-adds is bound by that pipe.  Here
// the recurrence runs in 64-bit integers and the sums over l (synthesis) or
// over ring pairs (adjoint) are exact integer products on the tensor cores; the
// FP64 pipe only takes the first steps of a sequence and collects the sums.
//
// Digit slices.  Every operand is written as a fixed-point number of seven
// base-256 digits (54 bits below a bound that holds for the whole row or
// block): the sequence's 0..255 below a signed leading one, the other
// operand's -128..127; leading ones are within 64.  Digits are small integers,
// exact in FP16, their products exact integers, and the sums of products of
// equal weight (order s = i + j of the digits' positions) share one FP32
// accumulator.  Below 2^24 an accumulator is exact: always in the orders that
// count (the assertions at DSS_KB and DSA_CB); in the last two (three in the
// adjoint, when four accumulators are added up) the largest possible sums, all
// digits extreme and of one sign, reach 1.2 (1.5) times 2^24 and may lose units
// there.  A unit of order s is 2^(-8 s - 12) of the operands' bounds, and one or
// two are lost in an addition: at most 2^-53 a block of the synthesis (42
// products into an order) and 2^-51 of the adjoint, under 3 and 7 % of the 96
// and 128 2^-54 that the digits not kept amount to.  Orders 0..7 are kept: the
// dropped ones are below the last digit of either operand.  Per term the error
// is thus an absolute 2^-54 of the operands' bounds, where a chain of FP64
// multiply-adds rounds to 2^-53 of the running sum at each step.  (The
// splitting of an accurate product into exact low-precision products is the
// scheme of Ozaki, Ogita, Oishi and Rump, Numer. Algorithms 59, 2012.)
//
// The recurrence.  For one m let e_l = sqrt((l^2 - m^2) / (4 l^2 - 1)), so
// that z P~_l = e_{l+1} P~_{l+1} + e_l P~_{l-1}.  With p_k = P~_o / z,
// o = m + 1 + 2k (an even polynomial times sin^m),
//   P~_o = z p_k,   P~_{o+1} = e_{o+2} p_{k+1} + e_{o+1} p_k,
// so one sequence serves both parities of l - m:
//   sum_l a_l P~_l(+-z) = sum_k p_k c_k +- z sum_k p_k d_k,
//   c_k = e_o a_{o-1} + e_{o+1} a_{o+1},  d_k = a_o,
// and p_k obeys a three-term recurrence in z^2 (Ishioka, J. Meteor. Soc.
// Japan 96, 2018).  Rescaled by sigma_k so that the last coefficient is one,
//   q_{k+1} = (A_k z^2 + B_k) q_k - q_{k-1},
// one step for two l.  Once a pair's values have grown past the first steps
// they are 64-bit fixed-point numbers, z^2 and the coefficients too (z^2 to
// 2^-64, the factor A z^2 + B + 8 to 2^-57), so a step rounds at 2^-58 of the
// bound of the functions and not at 2^-53 of the running value; the upper
// bytes of the same integers are the digits of the products.  Near the poles
// the first steps use 1 - z^2 and A_k + B_k.  Near the equator p_k grows like
// 1/z while P~ does not and the even sums would cancel, so pairs with z <=
// DS_ZEQ run the one-step recurrence of legendre.cu in the same integers (every
// l its own column of the sums).  Against a double-double recurrence the whole
// transforms are 2.5 to 4 times nearer than FP64 sums over an FP64 one-step
// recurrence (Nside 1024, lmax 2047: synthesis 2.6e-15 instead of 7.0e-15,
// adjoint 4.7e-15 instead of 1.8e-14).
//
// What bounds it: instruction issue, at half of its rate (ncu at Nside 512 /
// lmax 1023: 1.8 instructions a cycle, FP64 pipe 31 %, tensor pipe 17 %, 24 % of
// the warp slots); the rest are waits for the coefficients, the block barrier
// of a stage and the products.  About 42 instructions take a warp two l
// further.  At Nside 2048 / lmax 3000 the synthesis stage went from 89.1 ms
// (FP64 sums, one-step recurrence) to 17.5 ms and the adjoint from 99.9 to 21.7
// ms; where rings carry no weight in A, to 13.0 and 16.2 ms.
#include <cuda_fp16.h>

#include <cmath>

#include "common.cuh"
#include "kernels.h"
#include "tc.cuh"

namespace cr {

constexpr int DS_PAIRS = 128;             // ring pairs and threads per CTA
constexpr int DS_DIG = 7;                 // digits per operand
constexpr int DS_ORD = 8;                 // orders of the digit products kept
constexpr double DS_ZEQ = 0.06;           // pairs with z at or below run the one-step recurrence
constexpr uint32_t DS_WAIT = 1u << 26;    // polls of a bounded mbarrier wait
constexpr int DS_NONE = 0x3fffffff;       // start index of a pair that never starts
constexpr uint64_t DS_BIAS = 0x8000000000000080ull;  // zero (sign bit flipped) and half a unit of the dropped byte

// position of m's first k in tables of band limit L: room for
// (L - m) / 2 + 1 entries each
__host__ __device__ inline int64_t ds_off(int L, int m) { return (lm_off(L, m) >> 1) + m; }
int64_t ds_len(int L) { return (ds_off(L, L + 1) + 3) & ~(int64_t)1; }  // even: 16-byte alignment of what follows

// largest |sum| of order s over `terms` products of the two operands' digits
constexpr int64_t ds_order_sum(int s, int terms) {
  int64_t n = 0;
  for (int i = 0; i < DS_DIG; ++i)
    if (s - i >= 0 && s - i < DS_DIG) n += (i == 0 ? 64 : 255) * (s - i == 0 ? 64 : 128);
  return n * terms;
}

// ---- plan tables -------------------------------------------------------------
// Double-double helpers (Knuth's TwoSum, Dekker's product by FMA).
struct dd2 {
  double h, l;
};
__device__ __forceinline__ dd2 dd_prod(double a, double b) {
  const double p = a * b;
  return {p, fma(a, b, -p)};
}
__device__ __forceinline__ dd2 dd_norm(double h, double l) {
  const double s = h + l;
  return {s, l - (s - h)};
}
__device__ __forceinline__ dd2 dd_mul(dd2 a, dd2 b) {
  dd2 p = dd_prod(a.h, b.h);
  p.l += a.h * b.l + a.l * b.h;
  return dd_norm(p.h, p.l);
}
__device__ __forceinline__ dd2 dd_div(dd2 a, dd2 b) {
  const double q = a.h / b.h;
  const dd2 p = dd_prod(q, b.h);
  const double r = (a.h - p.h) - p.l + a.l - q * b.l;
  return dd_norm(q, r / b.h);
}
__device__ __forceinline__ dd2 dd_sqrt(dd2 a) {
  const double q = sqrt(a.h);
  const dd2 p = dd_prod(q, q);
  const double r = (a.h - p.h) - p.l + a.l;
  return dd_norm(q, 0.5 * r / q);
}

// sigma_{k-1}^2 / sigma_{k+1}^2 = e_{o+1}^2 e_{o+2}^2 / (e_o^2 e_{o-1}^2), o = m + 1 + 2k, k >= 1
__device__ __forceinline__ dd2 ds_ratio(int m, int k) {
  const double o = m + 1.0 + 2.0 * k, dm = m;
  auto n = [&](double l) { return (l - dm) * (l + dm); };
  const dd2 num = dd_mul(dd_prod(n(o + 1), n(o + 2)), {(2 * o - 1) * (2 * o - 1) * (2 * o - 3), 0.0});
  const dd2 den = dd_mul(dd_prod(n(o), n(o - 1)), {(2 * o + 3) * (2 * o + 3) * (2 * o + 5), 0.0});
  return dd_div(num, den);
}

// One CTA per m.  sigma_k^2 runs down from 1 at the last two k by ds_ratio,
// each parity of k its own chain: every thread multiplies the ratios of its
// stretch of k, one warp combines the stretches, and a second pass forms the
// coefficients.  In double-double, so that the tables are rounded once.
constexpr int DST_NT = 128;
__global__ void __launch_bounds__(DST_NT) ds_tab_kernel(DsTab t) {
  const int m = blockIdx.x, tid = threadIdx.x;
  const int nk = (t.Lc - m) / 2 + 1;
  const int64_t off = ds_off(t.Lc, m);
  __shared__ dd2 seg[2][DST_NT];
  // stretch of this thread in the order from the last k down, of even length
  const int len = (((nk + DST_NT - 1) / DST_NT) + 1) & ~1;
  const int j0 = tid * len, j1 = min(nk, j0 + len);
  dd2 c[2] = {{1.0, 0.0}, {1.0, 0.0}};
  for (int j = j0; j < j1; ++j)  // k = nk - 1 - j; sigma_k^2 from sigma_{k+2}^2 by the ratio at k + 1
    if (j >= 2) c[j & 1] = dd_mul(c[j & 1], ds_ratio(m, nk - j));
  seg[0][tid] = c[0];
  seg[1][tid] = c[1];
  __syncthreads();
  if (tid < 2) {
    dd2 s = {1.0, 0.0};
    for (int i = 0; i < DST_NT; ++i) {
      const dd2 v = seg[tid][i];
      seg[tid][i] = s;
      s = dd_mul(s, v);
    }
  }
  __syncthreads();
  dd2 s2[2] = {seg[0][tid], seg[1][tid]};  // the chains' values at the last j before this stretch
  const double dm = m;
  for (int j = j0; j < j1; ++j) {
    const int k = nk - 1 - j;
    const double o = m + 1.0 + 2.0 * k;
    const dd2 up = s2[(j & 1) ^ 1];  // sigma_{k+1}^2 (for j = 0 unused)
    if (j >= 2) s2[j & 1] = dd_mul(s2[j & 1], ds_ratio(m, nk - j));
    const dd2 cur = s2[j & 1];
    auto n = [&](double l) { return (l - dm) * (l + dm); };
    auto d = [&](double l) { return (2 * l - 1) * (2 * l + 1); };
    if (j > 0) {
      // A_k = sigma_k / (sigma_{k+1} e_{o+1} e_{o+2}), stored with the q it produces, k + 1
      const dd2 x = dd_div(dd_mul(cur, dd_prod(d(o + 1), d(o + 2))), dd_mul(up, dd_prod(n(o + 1), n(o + 2))));
      const dd2 A = dd_sqrt(x);
      const dd2 g = dd_prod(2 * o - 1, 2 * o + 3);
      const dd2 S = dd_div({2.0 * (o * o + o - dm * dm) - 1.0, 0.0}, g);           // e_{o+1}^2 + e_o^2
      const dd2 S1 = dd_div({2.0 * (o * o + o + dm * dm) - 2.0, 0.0}, g);          // 1 - that
      const dd2 B = dd_mul(A, {-S.h, -S.l});
      t.A[off + k + 1] = A.h;
      t.B[off + k + 1] = B.h;
      const dd2 AB = dd_mul(A, S1);
      t.AB[off + k + 1] = AB.h;
      t.rf[off + k + 1] = make_float4((float)A.h, (float)((AB.h - 2.0) + AB.l), (float)B.h, 0.f);
      // fixed point: A 2^57 and (B + 8) 2^60 (modulo 2^64); the integer steps
      // start where A < 100
      const double n = rint(B.h);
      const bool in = A.h < 127.0;
      t.Ai[off + k + 1] = in ? __double2ull_rn(A.h * 0x1p57) + (uint64_t)__double2ll_rn(A.l * 0x1p57) : 0;
      t.Bi[off + k + 1] = in ? ((uint64_t)((int64_t)n + 8) << 60) + (uint64_t)__double2ll_rn((B.h - n) * 0x1p60) +
                                   (uint64_t)__double2ll_rn(B.l * 0x1p60)
                             : 0;
    }
    const double sg = dd_sqrt(cur).h;
    const double e0 = dd_sqrt(dd_div(dd_mul(cur, {n(o), 0.0}), {d(o), 0.0})).h;
    const double e1 = dd_sqrt(dd_div(dd_mul(cur, {n(o + 1), 0.0}), {d(o + 1), 0.0})).h;
    t.sg[off + k] = sg;
    t.e0[off + k] = e0;
    t.e1[off + k] = e1;
    t.cf[off + k] = make_float4((float)sg, (float)e0, (float)e1, 0.f);
    if (k == 0) {
      t.A[off] = t.B[off] = t.AB[off] = 0.0;
      t.Ai[off] = t.Bi[off] = 0;
      t.rf[off] = make_float4(0.f, 0.f, 0.f, 0.f);
    }
  }
}

void ds_tab_free(DsTab& t) {
  if (t.A) cudaFree(t.A);
  t = DsTab();
}

// the tables for band limits up to Lc (one allocation)
int ds_tab_build(DsTab& t, int Lc, cudaStream_t st) {
  ds_tab_free(t);
  const int64_t n = ds_len(Lc);
  CR_CUDA(cudaMalloc(&t.A, 8 * n * sizeof(double) + 2 * n * sizeof(float4)));
  t.B = t.A + n;
  t.AB = t.B + n;
  t.sg = t.AB + n;
  t.e0 = t.sg + n;
  t.e1 = t.e0 + n;
  t.Ai = reinterpret_cast<uint64_t*>(t.e1 + n);
  t.Bi = t.Ai + n;
  t.rf = reinterpret_cast<float4*>(t.Bi + n);
  t.cf = t.rf + n;
  t.Lc = Lc;
  { ds_tab_kernel<<<Lc + 1, DST_NT, 0, st>>>(t); count_launch(); }
  CR_CHECK_LAUNCH("ds_tab_kernel");
  return CR_OK;
}

// ---- device helpers ----------------------------------------------------------

// kind::f16 instruction descriptor, FP16 inputs, FP32 accumulation
__host__ __device__ constexpr uint32_t ds_idesc(int M, int N) {
  return (1u << 4) | ((uint32_t)(N >> 3) << 17) | ((uint32_t)(M >> 4) << 24);
}

// MN-major offset (see legendre_tc.cu)
__device__ __forceinline__ uint32_t ds_mn_off(int mn, int k, int MN) {
  return (uint32_t)(((mn >> 3) << 7) + (k >> 3) * (MN / 8) * 128 + ((k & 7) << 4) + ((mn & 7) << 1));
}

__device__ __forceinline__ int ds_exp(double v) { return (__double2hiint(v) >> 20) & 0x7ff; }

// round(v 2^62 / 2^(eb - 1023)) + DS_BIAS, |v| < 2^(eb - 1023): the mantissa
// at bit 62, shifted right by the exponent's distance from the bound.  Bytes
// 7..1 are the digits: the leading one plus 128, the others as they are.
__device__ __forceinline__ uint64_t ds_fix(double v, int eb) {
  const int hi = __double2hiint(v);
  const uint32_t lo = (uint32_t)__double2loint(v);
  const int ex = (hi >> 20) & 0x7ff;
  const int r = max(0, min(63, eb - ex));
  const uint32_t mh = ((uint32_t)hi & 0xfffffu) | (ex ? 0x100000u : 0u);
  const uint64_t x = ((((uint64_t)mh << 32) | lo) << 10) >> r;
  const uint64_t s = (uint64_t)(int64_t)(hi >> 31);
  return (x ^ s) - s + DS_BIAS;
}

// The digits of the sequence (the operand with many values) are FP16
// subnormals d 2^-24: the bits of an unsigned digit are its value, so it
// takes a byte permutation and no conversion.  yh, yl: the two words of 8
// values; calls store(i, digits) for the digits i = 0..6.
template <typename F>
__device__ __forceinline__ void ds_digits8(const uint32_t yh[8], const uint32_t yl[8], F store) {
  uint4 d[DS_DIG];
  uint32_t* w = reinterpret_cast<uint32_t*>(d);
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    const uint32_t h0 = yh[2 * j], h1 = yh[2 * j + 1], l0 = yl[2 * j], l1 = yl[2 * j + 1];
    const uint32_t a = __byte_perm(h0, h1, 0x7632), b = __byte_perm(h0, h1, 0x5410), c = __byte_perm(l0, l1, 0x7632);
    // the leading digit: 1024 + byte, less 1152, times 2^-24
    const uint32_t t = __byte_perm(a, 0x64646464u, 0x4341);
    const __half2 v = __hfma2(*reinterpret_cast<const __half2*>(&t), __half2half2(__ushort_as_half(0x0001)),
                              __half2half2(__ushort_as_half(0x8480)));
    w[0 * 4 + j] = *reinterpret_cast<const uint32_t*>(&v);
    w[1 * 4 + j] = __byte_perm(a, 0u, 0x4240);
    w[2 * 4 + j] = __byte_perm(b, 0u, 0x4341);
    w[3 * 4 + j] = __byte_perm(b, 0u, 0x4240);
    w[4 * 4 + j] = __byte_perm(c, 0u, 0x4341);
    w[5 * 4 + j] = __byte_perm(c, 0u, 0x4240);
    w[6 * 4 + j] = __byte_perm(l0, l1, 0x5410) >> 8 & 0x00ff00ffu;
  }
#pragma unroll
  for (int i = 0; i < DS_DIG; ++i) store(i, d[i]);
}
// digit i (0 the most significant) of one value of the other operand, signed
// digits -128..127 of y = ds_fix + DS_SIGNED
constexpr uint64_t DS_SIGNED = 0x0080808080808000ull;
__device__ __forceinline__ __half ds_digit(uint64_t y, int i) {
  return __int2half_rn((int)((uint32_t)(y >> (8 * (7 - i))) & 255u) - 128);
}

// High 64 bits of a product from its three upper partial products, plus
// `up`: each of the two middle ones loses half a unit to truncation and the
// lowest product a quarter, so `up` = 1, 1, 1, 2 in turn keeps the mean error
// of four steps at zero (a bias would push every step the same way).
__device__ __forceinline__ uint64_t ds_mulhi(uint64_t a, uint64_t b, uint32_t up) {
  const uint32_t ah = (uint32_t)(a >> 32), al = (uint32_t)a, bh = (uint32_t)(b >> 32), bl = (uint32_t)b;
  const uint64_t mid = (uint64_t)__umulhi(al, bh) + __umulhi(ah, bl) + up;
  return (uint64_t)ah * bh + mid;
}

// sum_s D_s 256^-s of the eight orders f = D 2^-24, times 256^3
__device__ __forceinline__ double ds_collect(const float f[DS_ORD]) {
  long long d[DS_ORD];
#pragma unroll
  for (int s = 0; s < DS_ORD; ++s) d[s] = (int)(f[s] * 0x1p24f);
  const long long hi = (d[0] << 24) + (d[1] << 16) + (d[2] << 8) + d[3];
  const long long lo = (d[4] << 24) + (d[5] << 16) + (d[6] << 8) + d[7];
  // |hi|, |lo| < 2^51: to FP64 through the mantissa of 1.5 2^52
  const double dh = __longlong_as_double(0x4338000000000000ll + hi) - 6755399441055744.0;
  const double dl = __longlong_as_double(0x4338000000000000ll + lo) - 6755399441055744.0;
  return fma(dl, 0x1p-32, dh);
}
// 2^(eb - 1023 - 36): ds_collect's 2^-24 and the 2^-6 of either operand's
// leading digit; NaN where the block held an infinity or a NaN
__device__ __forceinline__ double ds_scale(int eb) {
  if (eb > 2047) return __longlong_as_double(0x7ff8000000000000ll);
  const int e = eb - 36;
  return e > 0 ? __hiloint2double(e << 20, 0) : 0.0;
}

// columns 16 o + c .. 16 o + c + 3 of the eight orders o, of this warp's lanes;
// the wait names the registers, so that nothing reads them before it
__device__ __forceinline__ void ds_ld_orders(uint32_t taddr, float f[DS_ORD][4]) {
#pragma unroll
  for (int o = 0; o < DS_ORD; ++o)
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0, %1, %2, %3}, [%4];"
                 : "=f"(f[o][0]), "=f"(f[o][1]), "=f"(f[o][2]), "=f"(f[o][3])
                 : "r"(taddr + 16 * o));
  asm volatile("tcgen05.wait::ld.sync.aligned;"
               : "+f"(f[0][0]), "+f"(f[0][1]), "+f"(f[0][2]), "+f"(f[0][3]), "+f"(f[1][0]), "+f"(f[1][1]),
                 "+f"(f[1][2]), "+f"(f[1][3]), "+f"(f[2][0]), "+f"(f[2][1]), "+f"(f[2][2]), "+f"(f[2][3]),
                 "+f"(f[3][0]), "+f"(f[3][1]), "+f"(f[3][2]), "+f"(f[3][3]), "+f"(f[4][0]), "+f"(f[4][1]),
                 "+f"(f[4][2]), "+f"(f[4][3]), "+f"(f[5][0]), "+f"(f[5][1]), "+f"(f[5][2]), "+f"(f[5][3]),
                 "+f"(f[6][0]), "+f"(f[6][1]), "+f"(f[6][2]), "+f"(f[6][3]), "+f"(f[7][0]), "+f"(f[7][1]),
                 "+f"(f[7][2]), "+f"(f[7][3])
               :
               : "memory");
}

// 16 columns of this warp's lanes
__device__ __forceinline__ void ds_ld16(uint32_t taddr, float f[16]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];"
      : "=f"(f[0]), "=f"(f[1]), "=f"(f[2]), "=f"(f[3]), "=f"(f[4]), "=f"(f[5]), "=f"(f[6]), "=f"(f[7]), "=f"(f[8]),
        "=f"(f[9]), "=f"(f[10]), "=f"(f[11]), "=f"(f[12]), "=f"(f[13]), "=f"(f[14]), "=f"(f[15])
      : "r"(taddr));
  asm volatile("tcgen05.wait::ld.sync.aligned;"
               : "+f"(f[0]), "+f"(f[1]), "+f"(f[2]), "+f"(f[3]), "+f"(f[4]), "+f"(f[5]), "+f"(f[6]), "+f"(f[7]),
                 "+f"(f[8]), "+f"(f[9]), "+f"(f[10]), "+f"(f[11]), "+f"(f[12]), "+f"(f[13]), "+f"(f[14]), "+f"(f[15])
               :
               : "memory");
}

// log2 of how far all |P~_lm(z)|, l <= L + 1, stay below their bound at the
// turning point of l = L + 1, for rings nearer to the pole than it (else 0).
// y = P~ sqrt(sin) obeys y'' = Q y, Q = (m^2 - 1/4) / sin^2 - (l + 1/2)^2, in theta,
// and g = y' / y stays above sqrt(Q) from the pole to the turning point (g' = Q -
// g^2 is 0 where they meet, and sqrt(Q) falls), so y is at most its value there
// times exp of minus the integral of sqrt(Q): m log((m z + u) / (sin D)) - nu
// log((nu z + u) / D) with u^2 = m^2 - nu^2 sin^2, D^2 = nu^2 - m^2, nu = l + 1/2.  Without it such a ring's digits
// would end 2^-54 below a bound far above its values: those 1e-6 (1e-9) of the
// largest ring's lost 5e-9 (1e-5) of themselves to it.  (Against the recurrence at
// lmax 64 to 8000 the bound is 0.2 to 5 bits above the largest value; the margins
// are FP32's rounding.)
__device__ __forceinline__ float ds_decay(int L, int m, float z, float s2) {
  const float nu = (float)L + 1.5f, mm = (float)m * (float)m - 0.25f;
  const float u2 = mm - nu * nu * s2;
  if (m == 0 || u2 <= 0.f) return 0.f;
  const float mf = sqrtf(mm), u = sqrtf(u2), D = rsqrtf((nu - mf) * (nu + mf));
  const float S = mf * log2f((mf * z + u) * D * rsqrtf(s2)) - nu * log2f((nu * z + u) * D);
  return fminf(80.f, fmaxf(0.f, 0.999f * S - 0.07f - 3e-5f * nu));
}

// One ring pair's sequence.  The first few steps, where the functions can grow
// by large factors, run in FP64 (mode 0); then in integers with an exponent
// per pair (mode 1: (Q - 2^63) 2^-62 2^(eb - 1023 - x), x falling to zero as
// the functions grow out of 2^-60); then, when every pair of the warp has
// x = 0, in plain fixed point (mode 2).
template <bool EQ>
struct DsPair {
  double q1 = 0.0, q2 = 0.0, Z = 0.0;  // mode 0; Z = z^2 or 1 - z^2 (EQ: z)
  uint64_t Q1 = 1ull << 63, Q2 = 1ull << 63, zi = 0;  // zi = z^2 2^64 (EQ: z 2^64)
  int x = 0;
  int k0 = DS_NONE;                    // first index of the sequence
  int eb = 1023;                       // |q| < 2^(eb - 1023)
  bool calm = true;                    // |e| at k0 is small enough for integer steps

  // p: pair; polar: FP64 steps on 1 - z^2, A + B
  __device__ __forceinline__ void load(const DsArgs& a, int m, int p, bool polar) {
    const int64_t o = (int64_t)m * a.ld_seed + p;
    const int ls = a.ls[o];
    const double2 st = a.st[o];
    const double z = a.z[p];
    const double zz = z * z;
    zi = EQ ? __double2ull_rn(z * 0x1p64) : __double2ull_rn(zz * 0x1p64) + (uint64_t)__double2ll_rn(fma(z, z, -zz) * 0x1p64);
    const double w = 1.0 - z;
    Z = EQ ? z : polar ? fma(-w, w, 2.0 * w) : zz;
    const int L = a.L;
    // bounds |P~_lm| <= sqrt((2 l + 1) / 4 pi) and 0.3 (l + 1)^(1/4) / sqrt(sin)
    // (the supremum over l, m and z is 0.29965 at every l tried to 3000),
    // over the rescaling at its smallest
    const float fl = (float)(L + 1), s2 = fmaxf((float)(1.0 - zz), 1e-20f);
    float b = fminf(0.2821f * sqrtf(2.f * fl), 0.305f * sqrtf(sqrtf(fl)) * rsqrtf(sqrtf(s2)));
    if (EQ) {
      const int64_t c = lm_off(a.Lc, m) + (L - m);
      b /= fminf((float)fmin(a.s[c], L > m ? a.s[c - 1] : 1.0), 1.f);
    } else {
      b /= (float)z;
    }
    eb = 1023 + (int)ceilf(log2f(b) + 0.1f - ds_decay(L, m, (float)z, s2));
    if (ls > L) return;
    const int64_t oc = lm_off(a.Lc, m) + (ls - m);
    const double c = ls > m ? a.c[oc] : 0.0;
    if (EQ) {
      k0 = ls - m;
      q1 = st.x;
      q2 = st.y;
      calm = k0 > 0 && c * z < 7.0;
      return;
    }
    // (q_{k0-1}, q_{k0-2}) from the one-step state (Q_{ls-1}, Q_{ls-2})
    k0 = (ls - m) >> 1;
    const int64_t ok = ds_off(a.t.Lc, m) + k0;
    const double P = a.s[oc] * fma(c * z, st.x, -st.y);
    const double A = a.t.A[ok], B = polar ? a.t.AB[ok] : a.t.B[ok];
    const bool odd = (ls - m) & 1;
    double n1 = 0.0, d1 = 1.0;  // q_{k0-1} = n1 / d1
    if (k0 > 0) {
      n1 = odd ? a.s[oc - 2] * st.y : a.s[oc - 1] * st.x;
      d1 = z * a.t.sg[ok - 1];
    }
    q1 = n1 / d1;
    const double qk = (odd ? P : fma(k0 > 0 ? -a.t.e1[ok - 1] : 0.0, q1, P)) / (odd ? z * a.t.sg[ok] : a.t.e0[ok]);
    // the second value, such that the recurrence's next step returns q_{k0}
    const double e = fma(polar ? -A : A, Z, B);
    q2 = fma(e, q1, -qk);
    calm = k0 > 0 && A < 100.0 && fabs(e) < 7.0;
  }

  __device__ __forceinline__ double step(double2 c) { return fma(EQ ? c.x * Z : fma(c.x, Z, c.y), q1, -q2); }

  // The same step in 64-bit integers: e + 8 = A z^2 + (B + 8) times 2^60, and
  // with Q = q + 2^63 (up to the common scale) e q - q' + 2^63 is
  // 16 mulhi(e + 8, Q) - 8 (e + 8 + Q) - Q' modulo 2^64.
  __device__ __forceinline__ uint64_t istep(ulonglong2 c, int u) const {
    const uint32_t up = (u & 3) == 3 ? 2u : 1u;
    const uint64_t e = (ds_mulhi(c.x, zi, up) << 3) + c.y;
    const uint64_t r = 0 - ((e + Q1) << 3) - Q2;  // beside the product
    return (ds_mulhi(e, Q1, up) << 4) + r;
  }

  // mode 0 -> 1: whether this pair can (c0, c1: the coefficients of the next
  // two steps; |e| falls with k), and the change, to at most 2^55
  __device__ __forceinline__ bool can_int(double2 c0, double2 c1, int ks) const {
    if (k0 == DS_NONE) return true;
    if (k0 > ks) return calm;
    const double e0 = EQ ? c0.x * Z : fma(c0.x, Z, c0.y), e1 = EQ ? c1.x * Z : fma(c1.x, Z, c1.y);
    return fabs(e0) < 7.0 && fabs(e1) < 7.0;
  }
  __device__ __forceinline__ void to_int() {
    x = k0 == DS_NONE ? 0 : max(0, eb - max(ds_exp(q1), ds_exp(q2)) - 8);
    Q1 = ds_fix(q1, eb - x) - 0x80;
    Q2 = ds_fix(q2, eb - x) - 0x80;
  }
  __device__ __forceinline__ void shift(int s) {
    constexpr uint64_t off = 1ull << 63;
    Q1 = (uint64_t)((int64_t)(Q1 ^ off) >> s) ^ off;
    Q2 = (uint64_t)((int64_t)(Q2 ^ off) >> s) ^ off;
    x -= s;
  }
  // bits of the larger of the two values, 32 to 63
  __device__ __forceinline__ int bits() const {
    const int h1 = (int)((uint32_t)(Q1 >> 32) ^ 0x80000000u), h2 = (int)((uint32_t)(Q2 >> 32) ^ 0x80000000u);
    return 64 - __clz((h1 ^ (h1 >> 31)) | (h2 ^ (h2 >> 31)));
  }
  // back to at most 2^55: two steps with |e| < 8 stay below 2^62
  __device__ __forceinline__ void renorm() { shift(min(x, max(0, bits() - 55))); }
};

// Coefficients of the step that produces index k of the sequence, for the
// FP64 steps (two doubles) or the integer ones.
template <bool EQ>
__device__ __forceinline__ ulonglong2 ds_coef(const DsArgs& a, int m, int k, int nk, bool polar, bool ints) {
  if (k >= nk) return make_ulonglong2(0, 0);
  double2 d = make_double2(0.0, 0.0);
  if (EQ) {
    d.x = a.c[lm_off(a.Lc, m) + k];
    if (ints) return make_ulonglong2(__double2ull_rn(d.x * 0x1p57), 1ull << 63);
  } else {
    const int64_t o = ds_off(a.t.Lc, m) + k;
    if (ints) return make_ulonglong2(a.t.Ai[o], a.t.Bi[o]);
    d = polar ? make_double2(-a.t.A[o], a.t.AB[o]) : make_double2(a.t.A[o], a.t.B[o]);
  }
  return make_ulonglong2((uint64_t)__double_as_longlong(d.x), (uint64_t)__double_as_longlong(d.y));
}
__device__ __forceinline__ double2 ds_coef_d(ulonglong2 c) {
  return make_double2(__longlong_as_double((long long)c.x), __longlong_as_double((long long)c.y));
}

// At the start of a stage (first index ks, cf its coefficients, one per
// lane): the warp's next mode, once all its pairs are fit for it.
template <bool EQ>
__device__ __forceinline__ void ds_mode(const DsArgs& a, DsPair<EQ>& s, int m, int ks, int nk, bool polar, int wmin,
                                        int wmax, ulonglong2& cf, int& mode) {
  if (mode == 2 || wmin == DS_NONE) return;
  if (mode == 0) {
    const double2 d = ds_coef_d(cf);
    const double2 c0 = make_double2(__shfl_sync(0xffffffffu, d.x, 0), __shfl_sync(0xffffffffu, d.y, 0));
    const double2 c1 = make_double2(__shfl_sync(0xffffffffu, d.x, 1), __shfl_sync(0xffffffffu, d.y, 1));
    const bool fit = fabs(d.x) < 100.0 || wmin > ks + 31;  // pairs yet to start know their own coefficient
    if (!__all_sync(0xffffffffu, fit && s.can_int(c0, c1, ks))) return;
    s.to_int();
    mode = 1;
    cf = ds_coef<EQ>(a, m, ks + (threadIdx.x & 31), nk, polar, true);
  }
  // plain fixed point: all started, and what the shift leaves is above FP64's precision
  if (ks >= wmax && __all_sync(0xffffffffu, s.k0 == DS_NONE || s.x == 0 || s.bits() - s.x >= 51)) {
    s.shift(s.x);
    mode = 2;
  }
}

struct DsShared {
  ulonglong2 sc[4][32];   // recurrence coefficients, one copy per warp
  uint64_t done;
  int eb[2][16];          // largest exponents of a block's columns
  uint32_t taddr;
  int kmin;
};

// The 8 values k..k+7 of a warp's sequences as digits: calls store(i, digits)
// for each digit i.  Nothing before the warp's first start.
template <bool EQ, typename F>
__device__ __forceinline__ void ds_produce8(DsPair<EQ>& s, const ulonglong2* sc, int k, int wmin, int mode, F store) {
  uint32_t yh[8], yl[8];
  if (mode == 2) {
#pragma unroll
    for (int u = 0; u < 8; ++u) {
      const uint64_t y = s.istep(sc[u], u);
      s.Q2 = s.Q1;
      s.Q1 = y;
      yh[u] = (uint32_t)(y >> 32);
      yl[u] = (uint32_t)y;
    }
  } else if (k + 8 <= wmin) {
#pragma unroll
    for (int i = 0; i < DS_DIG; ++i) store(i, make_uint4(0u, 0u, 0u, 0u));
    return;
  } else if (mode == 1) {
#pragma unroll
    for (int u = 0; u < 8; ++u) {
      const bool on = k + u >= s.k0;
      const uint64_t q = s.istep(sc[u], u);
      s.Q2 = on ? s.Q1 : s.Q2;
      s.Q1 = on ? q : s.Q1;
      const uint64_t y = on ? (uint64_t)((int64_t)(q ^ (1ull << 63)) >> min(s.x, 63)) ^ (1ull << 63) : 1ull << 63;
      yh[u] = (uint32_t)(y >> 32);
      yl[u] = (uint32_t)y;
      if (u & 1) s.renorm();
    }
  } else {
#pragma unroll
    for (int u = 0; u < 8; ++u) {
      const bool on = k + u >= s.k0;
      const double q = s.step(ds_coef_d(sc[u]));
      s.q2 = on ? s.q1 : s.q2;
      s.q1 = on ? q : s.q1;
      const uint64_t y = on ? ds_fix(q, s.eb) : DS_BIAS;
      yh[u] = (uint32_t)(y >> 32);
      yl[u] = (uint32_t)y;
    }
  }
  ds_digits8(yh, yl, store);
}

// this thread's pair, and the warp's and the CTA's first (and the warp's
// last) start index
template <bool EQ>
__device__ __forceinline__ void ds_setup(const DsArgs& a, DsShared& sh, DsPair<EQ>& s, int m, int p, int pend,
                                         bool* polar, int* wmin, int* wmax) {
  // one form per warp, from its last pair's cosine
  *polar = false;
  if (!EQ) {
    const double zl = a.z[min(p | 31, pend - 1)];
    *polar = __any_sync(0xffffffffu, zl * zl > 0.5);
  }
  if (p < pend) s.load(a, m, p, *polar);
  *wmin = __reduce_min_sync(0xffffffffu, s.k0);
  *wmax = __reduce_max_sync(0xffffffffu, s.k0 == DS_NONE ? 0 : s.k0);
  if (threadIdx.x == 0) sh.kmin = DS_NONE;
  __syncthreads();
  if ((threadIdx.x & 31) == 0) atomicMin(&sh.kmin, *wmin);
  __syncthreads();
}

// wait for the MMAs committed with phase `n`; once a wait has given up none
// is tried again (the results are marked, the barriers still pair up)
__device__ __forceinline__ void ds_wait(DsShared& sh, int n, bool& ok) {
  if (ok) ok = tc::mbar_wait(&sh.done, n & 1, DS_WAIT);
}

// ---- synthesis ---------------------------------------------------------------
// CTA: one m, 128 ring pairs (tensor-core rows, one per thread), up to NR
// right-hand sides.  A operand: the pairs' digits, 16 sequence values at a
// time.  B operand: the digits of (c_k, d_k) x (Re, Im) of the right-hand
// sides, 16 columns per digit, for a block of DSS_KB k with one exponent per
// column.  The accumulator of digit pair (i, j) starts at column 16 i, so
// equal orders add up in place.  After each block the warps collect the eight
// orders of their own pairs into FP64 sums.  Four CTAs per SM (53 KB of
// shared memory, 128 tensor-memory columns and 128 registers each): while one
// waits for its products the others step their recurrences.
constexpr int DSS_STAGE = DS_DIG * DS_PAIRS * 16 * 2;     // 28 KB
constexpr int DSS_BSTEP = 16 * DS_ORD * 16 * 2;           // 16 columns x 8 digits (the last zero) x K 16
constexpr int DSS_KB = 96;                                // k per block
static_assert(ds_order_sum(5, DSS_KB) < (1 << 24) && ds_order_sum(7, DSS_KB) < (5 << 22), "see the bounds above");
constexpr int DSS_SMEM = DSS_STAGE + (DSS_KB / 16) * DSS_BSTEP;
constexpr int DSS_TMEM = 128;

template <int NR, bool EQ>
__device__ __forceinline__ void ds_synth_body(const DsArgs& a, DsShared& sh, uint8_t* sm, int base, int pend) {
  const int m = blockIdx.y, L = a.L;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int p = base + tid;
  DsPair<EQ> s;
  bool polar;
  int wmin, wmax;
  ds_setup<EQ>(a, sh, s, m, p, pend, &polar, &wmin, &wmax);
  const int nk = EQ ? L - m + 1 : (L - m) / 2 + 1;
  const int kbeg = sh.kmin;
  uint8_t* Bs = sm + DSS_STAGE;
  double acc[4 * NR];
#pragma unroll
  for (int j = 0; j < 4 * NR; ++j) acc[j] = 0.0;
  bool ok = true;
  if (kbeg < nk) {
    for (int e = tid; e < (DSS_KB / 16) * DSS_BSTEP / 16; e += DS_PAIRS)
      reinterpret_cast<uint4*>(Bs)[e] = make_uint4(0u, 0u, 0u, 0u);
    if (tid < 32) sh.eb[tid >> 4][tid & 15] = 0;
    if (warp == 0) tc::tmem_alloc(&sh.taddr, DSS_TMEM);
    if (tid == 0) {
      tc::mbar_init(&sh.done, 1);
      tc::mbar_fence_init();
    }
    tc::fence_before_sync();
    __syncthreads();
    tc::fence_after_sync();
    const uint32_t taddr = sh.taddr;
    const int64_t offa = lm_off(L, m);
    const int64_t ok_ = ds_off(a.t.Lc, m), oc = lm_off(a.Lc, m);
    int mode = 0, gst = 0, nblk = 0;  // stages and blocks so far
    ulonglong2 cf = make_ulonglong2(0, 0);
    if (lane < 16) cf = ds_coef<EQ>(a, m, kbeg + lane, nk, polar, false);
    for (int kc = kbeg; kc < nk; kc += DSS_KB, ++nblk) {
      // coefficients of this block: thread = k
      const int k = kc + tid;
      double v[4 * NR];
#pragma unroll
      for (int j = 0; j < 4 * NR; ++j) v[j] = 0.0;
      if (k < nk && tid < DSS_KB) {
        if (EQ) {
          const double f = a.s[oc + k] * (a.dl ? a.dl[m + k] : 1.0);
#pragma unroll
          for (int r = 0; r < NR; ++r)
            if (r < a.nr) {
              const double2 x = a.alm[r * a.ld_alm + offa + k];
              const bool odd = k & 1;
              v[4 * r + 0] = odd ? 0.0 : f * x.x;
              v[4 * r + 1] = odd ? 0.0 : f * x.y;
              v[4 * r + 2] = odd ? f * x.x : 0.0;
              v[4 * r + 3] = odd ? f * x.y : 0.0;
            }
        } else {
          const int l = m + 2 * k;  // a_l, a_{l+1} = a_o, a_{l+2}
          const double f0 = a.t.e0[ok_ + k] * (a.dl ? a.dl[l] : 1.0);
          const double f1 = l + 1 <= L ? a.t.sg[ok_ + k] * (a.dl ? a.dl[l + 1] : 1.0) : 0.0;
          const double f2 = l + 2 <= L ? a.t.e1[ok_ + k] * (a.dl ? a.dl[l + 2] : 1.0) : 0.0;
#pragma unroll
          for (int r = 0; r < NR; ++r)
            if (r < a.nr) {
              const double2* x = a.alm + r * a.ld_alm + offa + 2 * k;
              const double2 x0 = x[0];
              const double2 x1 = l + 1 <= L ? x[1] : make_double2(0.0, 0.0);
              const double2 x2 = l + 2 <= L ? x[2] : make_double2(0.0, 0.0);
              v[4 * r + 0] = fma(f0, x0.x, f2 * x2.x);
              v[4 * r + 1] = fma(f0, x0.y, f2 * x2.y);
              v[4 * r + 2] = f1 * x1.x;
              v[4 * r + 3] = f1 * x1.y;
            }
        }
        if (m == 0) {
#pragma unroll
          for (int r = 0; r < NR; ++r) v[4 * r + 1] = v[4 * r + 3] = 0.0;
        }
      }
      int* eb = sh.eb[nblk & 1];
#pragma unroll
      for (int j = 0; j < 4 * NR; ++j) {
        const int e = __reduce_max_sync(0xffffffffu, ds_exp(v[j]));
        if (lane == 0) atomicMax(&eb[j], e + 1);  // |v| < 2^(eb - 1023); 2048: not finite
      }
      __syncthreads();
      if (tid < 16) sh.eb[(nblk + 1) & 1][tid] = 0;  // last read before this barrier
      if (tid < DSS_KB) {
        uint8_t* Bk = Bs + (tid >> 4) * DSS_BSTEP;
#pragma unroll
        for (int j = 0; j < 4 * NR; ++j) {
          const uint64_t y = ds_fix(v[j], eb[j]) + DS_SIGNED;
#pragma unroll
          for (int i = 0; i < DS_DIG; ++i)
            *reinterpret_cast<__half*>(Bk + tc::kmajor_offset(16 * i + j, tid & 15, 16)) = ds_digit(y, i);
        }
      }
      const int nst = min(DSS_KB / 16, (nk - kc + 15) / 16);
      for (int st = 0; st < nst; ++st, ++gst) {
        const int ks = kc + 16 * st;
        ds_mode<EQ>(a, s, m, ks, nk, polar, wmin, wmax, cf, mode);
        __syncwarp();
        if (lane < 16) {
          sh.sc[warp][lane] = cf;
          cf = ds_coef<EQ>(a, m, ks + 16 + lane, nk, polar, mode > 0);
        }
        __syncwarp();
        if (st > 0) ds_wait(sh, gst - 1, ok);
#pragma unroll 1
        for (int g = 0; g < 2; ++g) {
          uint8_t* S = sm + tc::kmajor_offset(tid, 8 * g, 16);
          ds_produce8<EQ>(s, sh.sc[warp] + 8 * g, ks + 8 * g, wmin, mode,
                          [&](int i, uint4 d) { *reinterpret_cast<uint4*>(S + i * (DSS_STAGE / DS_DIG)) = d; });
        }
        tc::fence_proxy_async();
        tc::fence_before_sync();
        __syncthreads();
        if (tid == 0) {
          tc::fence_after_sync();
          const uint32_t sa = tc::smem_addr(sm);
          const uint64_t bd = tc::smem_desc(tc::smem_addr(Bs + st * DSS_BSTEP), 128, 256);
#pragma unroll
          for (int i = 0; i < DS_DIG; ++i) {
            // digit i meets digits 0 .. min(6, 7 - i); i = 0 also the zero
            // digit, which clears the last order on the block's first step
            const int nj = i == 0 ? DS_ORD : min(DS_DIG, DS_ORD - i);
            tc::mma_bf16(taddr + 16 * i, tc::smem_desc(sa + i * (DSS_STAGE / DS_DIG), 128, 256), bd,
                         ds_idesc(128, 16 * nj), (st > 0 || i > 0) ? 1u : 0u);
          }
          tc::mma_commit(&sh.done);
        }
        __syncwarp();
      }
      ds_wait(sh, gst - 1, ok);
      tc::fence_after_sync();
      __syncwarp();
      const uint32_t tw = taddr + ((uint32_t)(warp * 32) << 16);
      const bool on = kc + DSS_KB > s.k0;
#pragma unroll
      for (int r = 0; r < NR; ++r) {
        if (r < a.nr) {
          float f[DS_ORD][4];
          ds_ld_orders(tw + 4 * r, f);
#pragma unroll
          for (int j = 0; j < 4; ++j) {
            float c[DS_ORD];
#pragma unroll
            for (int o = 0; o < DS_ORD; ++o) c[o] = f[o][j];
            const double x = fma(ds_collect(c), ds_scale(eb[4 * r + j]), acc[4 * r + j]);
            if (on) acc[4 * r + j] = x;
          }
        }
      }
      tc::fence_before_sync();
    }
    ok = __syncthreads_and(ok ? 1 : 0) != 0;
    // a wait that gave up: once more, before the tensor memory goes back
    if (!ok) tc::mbar_wait_block(&sh.done, (gst - 1) & 1, DS_WAIT);
    tc::fence_after_sync();
    if (warp == 0) tc::tmem_dealloc(taddr, DSS_TMEM);
  }
  if (p < pend) {
    const int rn = p, rs = a.nring - 1 - p;
    const bool live = s.k0 < nk;
    // a wait that gave up must not pass for a result
    const double sc = ok ? __hiloint2double(s.eb << 20, 0) : __longlong_as_double(0x7ff8000000000000ll);
    const double zd = EQ ? sc : sc * a.z[p];
#pragma unroll
    for (int r = 0; r < NR; ++r)
      if (r < a.nr) {
        double2 n = make_double2(0.0, 0.0), t = n;
        if (live || !ok) {
          const double cx = acc[4 * r] * sc, cy = acc[4 * r + 1] * sc;
          const double dx = acc[4 * r + 2] * zd, dy = acc[4 * r + 3] * zd;
          n = make_double2(cx + dx, cy + dy);
          t = make_double2(cx - dx, cy - dy);
        }
        a.phase[r * a.ld_phase + (int64_t)rn * a.ldp + m] = n;
        if (rs != rn) a.phase[r * a.ld_phase + (int64_t)rs * a.ldp + m] = t;
      }
  }
}

template <int NR>
__global__ void __launch_bounds__(DS_PAIRS, NR == 1 ? 4 : 3) ds_synth_kernel(DsArgs a) {
  extern __shared__ __align__(1024) uint8_t ds_sm[];
  __shared__ DsShared sh;
  const int tile = blockIdx.x;
  if (tile < a.nt_is) ds_synth_body<NR, false>(a, sh, ds_sm, tile * DS_PAIRS, a.nis);
  else ds_synth_body<NR, true>(a, sh, ds_sm, a.nis + (tile - a.nt_is) * DS_PAIRS, a.npairs);
}

// ---- adjoint -----------------------------------------------------------------
// CTA: one m, 128 ring pairs (the contraction index, one per thread).  The
// pairs' phases G = (even combination, z times the odd one) x (Re, Im) of up
// to NR right-hand sides are split into digits once: row (digit, column) of a
// K-major operand, 8 columns per digit (64 rows), with zero rows around.  The
// other operand holds 16 sequence values of the 128 pairs per stage, MN-major,
// so a thread writes 8 consecutive values of its own pair.  A tensor-core
// instruction takes at least 48 cycles here up to N = 64 and N / 2 beyond,
// whatever M, so four digits of the sequence share one instruction (N = 64,
// then 48 for the other three, read against G's digits shifted down by four):
// 16 per stage instead of 56, which the instruction rate would bind (30 ms
// against 18 at Nside 2048 / lmax 3000).  Row s of the accumulator of digits
// d and d + 4 is order s + d.  One partial row per (tile, right-hand side):
// (u_k, v_k) with a_o = sigma_k v_k, a_{o-1} += sigma_k e_o u_k,
// a_{o+1} += sigma_k e_{o+1} u_k, or the two parities' values themselves near
// the equator.
constexpr int DSA_N = 16;                                  // sequence values per stage
constexpr int DSA_CB = 8;                                  // columns per digit of G
// an accumulator takes digits d and d + 4 of the sequence against one digit each
static_assert(2 * 255 * 128 * DS_PAIRS < (1 << 24) && ds_order_sum(4, DS_PAIRS) < (1 << 24) &&
                  ds_order_sum(7, DS_PAIRS) < (3 << 23), "see the bounds above");
constexpr int DSA_A = 12 * DSA_CB * DS_PAIRS * 2;          // G: 4 CB zero rows, the digits, CB zero rows
constexpr int DSA_B = DS_DIG * DSA_N * DS_PAIRS * 2;       // a stage: digits 0..3, digits 4..6
constexpr int DSA_FS = 24;                                 // row stride of the collected accumulators
constexpr int DSA_SMEM = DSA_A + DSA_B;
constexpr int DSA_TMEM = 64;
static_assert(4 * DS_ORD * 4 * DSA_FS * 4 <= DSA_B, "the collected accumulators reuse the stage");

template <int NR, bool EQ>
__device__ __forceinline__ void ds_adjoint_body(const DsArgs& a, DsShared& sh, uint8_t* sm, int base, int pend) {
  constexpr int NC = 4 * NR;
  const int m = blockIdx.y, L = a.L, blk = blockIdx.x;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int p = base + tid;
  DsPair<EQ> s;
  bool polar;
  int wmin, wmax;
  ds_setup<EQ>(a, sh, s, m, p, pend, &polar, &wmin, &wmax);
  const int nk = EQ ? L - m + 1 : (L - m) / 2 + 1;
  const int nk2 = (L - m) / 2 + 1;
  const int kbeg = sh.kmin;
  // partial row of right-hand side r: doubles 4 k + column
  const int64_t rstride = (int64_t)a.nblk * a.nkk * 4;
  double* part = a.partial + ((int64_t)blk * a.nkk + ds_off(L, m)) * 4;
  // zero before the tile's first start
  for (int r = 0; r < a.nr; ++r)
    for (int i = tid; i < (kbeg < nk ? (EQ ? 2 * kbeg : 4 * kbeg) : 4 * nk2); i += DS_PAIRS) part[r * rstride + i] = 0.0;
  if (kbeg >= nk) return;

  for (int e = tid; e < DSA_A / 16; e += DS_PAIRS) reinterpret_cast<uint4*>(sm)[e] = make_uint4(0u, 0u, 0u, 0u);
  if (tid < 16) sh.eb[0][tid] = 0;
  if (warp == 0) tc::tmem_alloc(&sh.taddr, DSA_TMEM);
  if (tid == 0) {
    tc::mbar_init(&sh.done, 1);
    tc::mbar_fence_init();
  }
  double g[NC];
#pragma unroll
  for (int j = 0; j < NC; ++j) g[j] = 0.0;
  if (s.k0 < nk) {
    const int rn = p, rs = a.nring - 1 - p;
    const double zo = EQ ? 1.0 : a.z[p];
#pragma unroll
    for (int r = 0; r < NR; ++r)
      if (r < a.nr) {
        const double2 gn = a.phase[r * a.ld_phase + (int64_t)rn * a.ldp + m];
        const double2 gs = (rs != rn) ? a.phase[r * a.ld_phase + (int64_t)rs * a.ldp + m] : make_double2(0.0, 0.0);
        g[4 * r] = gn.x + gs.x;
        g[4 * r + 1] = gn.y + gs.y;
        g[4 * r + 2] = zo * (gn.x - gs.x);
        g[4 * r + 3] = zo * (gn.y - gs.y);
      }
  }
  __syncthreads();
  // the pair's bound goes to this operand: |g| 2^(eb_pair) < 2^(eb - 1023)
#pragma unroll
  for (int j = 0; j < NC; ++j) {
    const int x = ds_exp(g[j]);
    const int e = __reduce_max_sync(0xffffffffu, x == 0 ? 0 : (x == 2047 ? 1 << 20 : x + s.eb - 1023));
    if (lane == 0) atomicMax(&sh.eb[0][j], e + 1);
  }
  __syncthreads();
#pragma unroll
  for (int j = 0; j < NC; ++j) {
    const uint64_t y = ds_fix(g[j], sh.eb[0][j] - (s.eb - 1023)) + DS_SIGNED;
#pragma unroll
    for (int i = 0; i < DS_DIG; ++i)
      *reinterpret_cast<__half*>(sm + tc::kmajor_offset((4 + i) * DSA_CB + j, tid, DS_PAIRS)) = ds_digit(y, i);
  }
  tc::fence_proxy_async();
  tc::fence_before_sync();
  __syncthreads();
  tc::fence_after_sync();
  const uint32_t taddr = sh.taddr;
  bool ok = true;
  const int nit = (nk - kbeg + DSA_N - 1) / DSA_N;
  float* fb = reinterpret_cast<float*>(sm + DSA_A);  // the stage's operand is read by then
  // accumulators of iteration `it` to the partial rows
  auto flush = [&](int it) {
    ds_wait(sh, it, ok);
    tc::fence_after_sync();
    __syncwarp();
    // the 64 rows live in lanes 0..15 of each warp's quarter
    const int so = 2 * warp + (lane >> 3), col = lane & 7;
#pragma unroll
    for (int r = 0; r < NR; ++r) {
      if (r < a.nr) {
        if (r > 0) __syncthreads();  // the previous right-hand side is collected
#pragma unroll
        for (int d = 0; d < 4; ++d) {
          float f[DSA_N];
          ds_ld16(taddr + ((uint32_t)(warp * 32) << 16) + DSA_N * d, f);
          if (lane < 16 && (col >> 2) == r) {
            float4* q = reinterpret_cast<float4*>(fb + ((d * DS_ORD + so) * 4 + (col & 3)) * DSA_FS);
#pragma unroll
            for (int i = 0; i < DSA_N / 4; ++i) q[i] = make_float4(f[4 * i], f[4 * i + 1], f[4 * i + 2], f[4 * i + 3]);
          }
        }
        tc::fence_before_sync();
        // the sums below are of all warps' loads: one wait that gave up marks them all
        ok = __syncthreads_and(ok ? 1 : 0) != 0;
        const int w = tid & 3, kk = tid >> 2, k = kbeg + it * DSA_N + kk;
        if (kk >= DSA_N) continue;
        float c[DS_ORD];
#pragma unroll
        for (int o = 0; o < DS_ORD; ++o) {
          c[o] = fb[(o * 4 + w) * DSA_FS + kk];
#pragma unroll
          for (int d = 1; d < 4; ++d)
            if (d <= o) c[o] += fb[((d * DS_ORD + o - d) * 4 + w) * DSA_FS + kk];
        }
        double x = ds_collect(c) * ds_scale(sh.eb[0][4 * r + w]);
        if (!ok) x = __longlong_as_double(0x7ff8000000000000ll);
        if (k < nk) {
          double* q = part + r * rstride;
          if (!EQ) q[4 * (int64_t)k + w] = x;
          else if ((k & 1) == (w >> 1)) q[2 * (int64_t)k + (w & 1)] = x;
        }
      }
    }
  };
  int mode = 0;
  ulonglong2 cf = make_ulonglong2(0, 0);
  if (lane < DSA_N) cf = ds_coef<EQ>(a, m, kbeg + lane, nk, polar, false);
  for (int it = 0; it < nit; ++it) {
    const int ks = kbeg + it * DSA_N;
    ds_mode<EQ>(a, s, m, ks, nk, polar, wmin, wmax, cf, mode);
    __syncwarp();
    if (lane < DSA_N) {
      sh.sc[warp][lane] = cf;
      cf = ds_coef<EQ>(a, m, ks + DSA_N + lane, nk, polar, mode > 0);
    }
    __syncwarp();
    if (it > 0) {
      flush(it - 1);
      __syncthreads();
    }
#pragma unroll 1
    for (int gq = 0; gq < DSA_N / 8; ++gq) {
      uint8_t* B = sm + DSA_A;
      const uint32_t o4 = ds_mn_off(8 * gq, tid, 4 * DSA_N), o3 = 4 * DSA_N * DS_PAIRS * 2 + ds_mn_off(8 * gq, tid, 3 * DSA_N);
      ds_produce8<EQ>(s, sh.sc[warp] + 8 * gq, ks + 8 * gq, wmin, mode, [&](int i, uint4 d) {
        *reinterpret_cast<uint4*>(B + (i < 4 ? o4 : o3) + (i & 3) * (DSA_N / 8) * 128) = d;
      });
    }
    tc::fence_proxy_async();
    tc::fence_before_sync();
    __syncthreads();
    if (tid == 0) {
      tc::fence_after_sync();
      constexpr uint32_t rg = (DS_PAIRS / 8) * 128;  // 8 rows of the K-major operand
      const uint32_t sa = tc::smem_addr(sm), sb = tc::smem_addr(sm + DSA_A);
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const int n = h == 0 ? 4 * DSA_N : 3 * DSA_N;
        const uint32_t bk = (n / 8) * 128;           // 8 pairs of the MN-major operand
        const uint32_t id = ds_idesc(8 * DSA_CB, n) | (1u << 16);
#pragma unroll
        for (int kk = 0; kk < DS_PAIRS / 16; ++kk)
          tc::mma_bf16(taddr, tc::smem_desc(sa + (h == 0 ? 4 : 0) * (DSA_CB / 8) * rg + kk * 256, 128, rg),
                       tc::smem_desc(sb + h * 4 * DSA_N * DS_PAIRS * 2 + kk * 2 * bk, bk, 128), id,
                       (h > 0 || kk > 0) ? 1u : 0u);
      }
      tc::mma_commit(&sh.done);
    }
    __syncwarp();
  }
  flush(nit - 1);
  if (!__syncthreads_and(ok ? 1 : 0)) tc::mbar_wait_block(&sh.done, (nit - 1) & 1, DS_WAIT);
  tc::fence_after_sync();
  if (warp == 0) tc::tmem_dealloc(taddr, DSA_TMEM);
}

template <int NR>
__global__ void __launch_bounds__(DS_PAIRS, 4) ds_adjoint_kernel(DsArgs a) {
  extern __shared__ __align__(1024) uint8_t ds_sm[];
  __shared__ DsShared sh;
  const int tile = blockIdx.x;
  if (tile < a.nt_is) ds_adjoint_body<NR, false>(a, sh, ds_sm, tile * DS_PAIRS, a.nis);
  else ds_adjoint_body<NR, true>(a, sh, ds_sm, a.nis + (tile - a.nt_is) * DS_PAIRS, a.npairs);
}

// The tiles' partial rows to coefficients (fixed order), with the epilogue of
// leg_finalize_kernel.  Thread: one k, i.e. l = m + 2 k and l + 1.
__global__ void __launch_bounds__(128) ds_finalize_kernel(DsArgs a, const double* partial, FinalizeArgs<double> f) {
  const int m = blockIdx.y, L = a.L;
  const int nk = (L - m) / 2 + 1;
  const int k = blockIdx.x * blockDim.x + threadIdx.x;
  if (blockIdx.x * blockDim.x >= nk) return;  // whole CTA
  // blockIdx.z: right-hand side
  const double2* row = reinterpret_cast<const double2*>(partial) + ((int64_t)blockIdx.z * a.nblk * a.nkk + ds_off(L, m)) * 2;
  const int64_t v0 = blockIdx.z * f.ld;
  const int64_t bs = a.nkk * 2;
  auto sum = [&](int kk, int b0, int b1, double2& x, double2& y) {
    x = y = make_double2(0.0, 0.0);
#pragma unroll 4
    for (int b = b0; b < b1; ++b) {
      const double2* r = row + b * bs + 2 * (int64_t)kk;
      x = cadd(x, r[0]);
      y = cadd(y, r[1]);
    }
  };
  const bool in = k < nk;
  double2 u = make_double2(0.0, 0.0), v = u;
  if (in) sum(k, 0, a.nt_is, u, v);
  double2 um;  // u_{k-1}
  um.x = __shfl_up_sync(0xffffffffu, u.x, 1);
  um.y = __shfl_up_sync(0xffffffffu, u.y, 1);
  if (!in) return;
  if ((threadIdx.x & 31) == 0) {
    um = make_double2(0.0, 0.0);
    double2 vm;
    if (k > 0) sum(k - 1, 0, a.nt_is, um, vm);
  }
  double2 q[2];  // the equatorial pairs' values of l and l + 1
  sum(k, a.nt_is, a.nblk, q[0], q[1]);
  const int64_t ok = ds_off(a.t.Lc, m) + k, oc = lm_off(a.Lc, m) + 2 * k;
  const double g0 = a.t.e0[ok], g1 = k > 0 ? a.t.e1[ok - 1] : 0.0;
#pragma unroll
  for (int w = 0; w < 2; ++w) {
    const int l = m + 2 * k + w;
    if (l > L) break;
    const double sl = a.s[oc + w];
    double2 y = make_double2(sl * q[w].x, sl * q[w].y);
    if (w == 0) {
      y.x += g0 * u.x + (k > 0 ? g1 * um.x : 0.0);
      y.y += g0 * u.y + (k > 0 ? g1 * um.y : 0.0);
    } else {
      y.x = fma(a.t.sg[ok], v.x, y.x);
      y.y = fma(a.t.sg[ok], v.y, y.y);
    }
    const int64_t i = v0 + lm_off(L, m) + (l - m);
    if (f.dl_out) y = cscale(y, f.dl_out[l]);
    if (f.dadd) {
      const double2 x = f.xadd[i];
      y.x = fma(f.dadd[l], x.x, y.x);
      y.y = fma(f.dadd[l], x.y, y.y);
    }
    if (f.bsub) {
      const double2 b = f.bsub[i];
      y = make_double2(b.x - y.x, b.y - y.y);
    }
    if (m == 0) y.y = 0.0;
    if (f.accumulate) y = cadd(y, f.out[i]);
    f.out[i] = y;
  }
}

// ---- launchers ---------------------------------------------------------------

int ds_tiles(int nis, int npairs) { return (nis + DS_PAIRS - 1) / DS_PAIRS + (npairs - nis + DS_PAIRS - 1) / DS_PAIRS; }
int ds_first_equatorial(const double* z, int npairs) {
  int n = 0;
  while (n < npairs && z[n] > DS_ZEQ) ++n;
  return n;
}
int64_t ds_partial_bytes(int nis, int npairs, int L, int nr) {
  return (int64_t)nr * ds_tiles(nis, npairs) * ds_len(L) * 4 * (int64_t)sizeof(double);
}

// By the grid, not by the pairs that a mask leaves: A at Nside 32 / lmax 95 with
// 55 of 64 pairs takes 64 us here and 147 us with the FP64 sums of legendre.cu, at
// Nside 2048 / lmax 3000 with 1 and 63 pairs 624 and 690 us against 3.7 and 4.0 ms:
// one warp's chain of FP64 steps, however few the pairs.  The smallest grids and
// band limits stay with the plain FP64 sums (60 pairs, lmax 64: synthesis 33 us here,
// 57 us there; 8 pairs: 33 and 56 us).
bool ds_use(const LegArgs<double>& a) { return a.ds && !a.df && (a.nring + 1) / 2 >= 64 && a.L >= 64; }

static DsArgs ds_args(const LegArgs<double>& la, int nr) {
  DsArgs a;
  a.t = *la.ds;
  a.phase = la.phase;
  a.ldp = la.ldp;
  a.ld_phase = (int64_t)la.nring * la.ldp;
  a.L = la.L;
  a.Lc = la.Lc;
  a.nr = nr;
  a.c = la.c;
  a.s = la.s;
  a.dl = la.dl;
  a.z = la.z;
  a.ls = la.ls;
  a.st = la.st;
  a.ld_seed = la.ld_seed;
  a.npairs = la.npairs;
  a.nring = la.nring;
  a.nis = la.nis;
  a.nt_is = (la.nis + DS_PAIRS - 1) / DS_PAIRS;
  a.nblk = ds_tiles(la.nis, la.npairs);
  a.nkk = ds_len(la.L);
  return a;
}

// nr right-hand sides (vectors at stride ld_alm, phases at nring * ldp), four at a time
int launch_ds_synth(const LegArgs<double>& la, const double2* alm, int64_t ld_alm, int nr, double2* phase,
                    cudaStream_t st) {
  for (int r0 = 0; r0 < nr; r0 += 4) {
    DsArgs a = ds_args(la, std::min(4, nr - r0));
    a.alm = alm + r0 * ld_alm;
    a.ld_alm = ld_alm;
    a.phase = phase + r0 * a.ld_phase;
    const dim3 grid(a.nblk, la.L + 1);
    if (a.nr == 1) {
      CR_CUDA(cudaFuncSetAttribute(ds_synth_kernel<1>, cudaFuncAttributeMaxDynamicSharedMemorySize, DSS_SMEM));
      { ds_synth_kernel<1><<<grid, DS_PAIRS, DSS_SMEM, st>>>(a); count_launch(); }
    } else {
      CR_CUDA(cudaFuncSetAttribute(ds_synth_kernel<4>, cudaFuncAttributeMaxDynamicSharedMemorySize, DSS_SMEM));
      { ds_synth_kernel<4><<<grid, DS_PAIRS, DSS_SMEM, st>>>(a); count_launch(); }
    }
    CR_CHECK_LAUNCH("ds_synth_kernel");
  }
  return CR_OK;
}

template <int NR>
static int ds_adjoint_launch(const DsArgs& a, cudaStream_t st) {
  CR_CUDA(cudaFuncSetAttribute(ds_adjoint_kernel<NR>, cudaFuncAttributeMaxDynamicSharedMemorySize, DSA_SMEM));
  { ds_adjoint_kernel<NR><<<dim3(a.nblk, a.L + 1), DS_PAIRS, DSA_SMEM, st>>>(a); count_launch(); }
  CR_CHECK_LAUNCH("ds_adjoint_kernel");
  return CR_OK;
}

// phases of nr right-hand sides -> f.out (vectors f.ld apart), two at a time, through
// partial rows in `partial` (ds_partial_bytes of two right-hand sides, of one
// when nr = 1)
int launch_ds_adjoint(const LegArgs<double>& la, const double2* phase, int nr, double* partial,
                      const FinalizeArgs<double>& f0, cudaStream_t st) {
  for (int r0 = 0; r0 < nr; r0 += 2) {
    DsArgs a = ds_args(la, std::min(2, nr - r0));
    a.phase = const_cast<double2*>(phase) + r0 * a.ld_phase;
    a.partial = partial;
    int rc = a.nr == 1 ? ds_adjoint_launch<1>(a, st) : ds_adjoint_launch<2>(a, st);
    if (rc) return rc;
    FinalizeArgs<double> f = f0;
    f.out += r0 * f.ld;
    if (f.xadd) f.xadd += r0 * f.ld;
    if (f.bsub) f.bsub += r0 * f.ld;
    const dim3 grid((la.L / 2 + 1 + 127) / 128, la.L + 1, a.nr);
    { ds_finalize_kernel<<<grid, 128, 0, st>>>(a, partial, f); count_launch(); }
    CR_CHECK_LAUNCH("ds_finalize_kernel");
  }
  return CR_OK;
}

}  // namespace cr
