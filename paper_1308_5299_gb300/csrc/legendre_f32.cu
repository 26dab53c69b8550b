// FP32 Legendre stages on the CUDA cores.
//
// The two-step sequence of legendre_ds.cu: with p_k = P~_o / z, o = m + 1 + 2k,
//   sum_l a_l P~_l(+-z) = sum_k p_k c_k +- z sum_k p_k d_k,
//   c_k = e_o a_{o-1} + e_{o+1} a_{o+1},  d_k = a_o,
// and q_k = p_k / sigma_k obeys q_{k+1} = e_k q_k - q_{k-1}, e_k = A_k z^2 + B_k.
// Per two l and ring pair that is 2 (or 3) operations of recurrence and 4 of
// sums, where the one-step recurrence takes 4 (or 6) and 4.  Three forms of the
// step keep FP32's rounding down, each on a range of pairs (a warp has one):
//  - polar, z > LF_ZPOLAR: the difference form on s = 1 - z^2,
//      d = ((A + B - 2) - A s) q + d, q = q + d
//    (q varies slowly in k there; e - 2 is carried at full relative precision);
//  - middle: q_{k+1} = (A z^2 + B) q_k - q_{k-1};
//  - equatorial, z < LF_ZEQ: the one-step recurrence, P~_l = s_l q_l, q_l = c_l z
//    q_{l-1} - q_{l-2}, with w = z q at odd l - m (q_l = c_l w_{l-1} - q_{l-2}, w_l =
//    c_l z^2 q_{l-1} - w_{l-2}: one product less; the odd sums are divided by z).
//    p_k grows like min(L, 1 / z) there while P~ does not, so
//    that the two-step form's even sums cancel by that factor (the ring on the
//    equator would be off by 5e-6, 1.4e-5, 4e-5 at lmax 384, 1023, 3000).
// The argument of each has four copies that differ in the last place and
// average to the exact value, used in turn: a single rounded one would act the
// same way at every step.  The lines lie where the forms on either side are
// about equally near or the cheaper one is.
// Ring by ring against FP64 (white spectrum, Nside 64 / lmax 384, 512 / 1023, 2048 /
// 3000): 3e-7, 5e-7, 8e-7 for z < 0.015, at most 5e-7, 1e-6, 2.5e-6 for z < LF_ZEQ,
// 2e-6, 4.7e-6, 1.3e-5 just below LF_ZPOLAR, 1.2e-6, 2.8e-6, 7e-6 above it; over the
// map 7.5e-7, 1.6e-6, 4.9e-6.  One-step kernels with rounded arguments throughout:
// 3e-7, 5e-7, 9e-7 for z < 0.015, 3.8e-6, 9e-6, 2.5e-5 at z = 0.7, 1.8e-6, 4.4e-6,
// 1.2e-5 over the map.  No ring is further off than theirs.
//
// One warp per block of 32 RP pairs of one m (RP per thread), without block
// barriers; m in blockIdx.y, so the longest warps start first.  Each warp
// stages the chunk's coefficients itself; a group of 8 k runs unchecked once
// all of the warp's pairs have started (start tables, |P~| >= 2^-60).  Bound by
// FP32 issue: 6.5 operations per pair and k beside two shared loads per k and
// warp (ncu at Nside 1024 / lmax 2047: synthesis 2.8, adjoint 2.65 instructions a
// cycle, the adjoint's transpose near the shared-memory rate as well).  At Nside
// 2048 / lmax 3000, in A, against the one-step kernels with two ring pairs packed
// into an instruction and a launch each for polar and other pairs: synthesis
// 2.4 -> 1.52 ms, adjoint 3.3 -> 2.06 ms; alone, with every ring, 1.92 and 2.58 ms.
#include <cmath>

#include "common.cuh"
#include "kernels.h"

namespace cr {

constexpr double LF_ZPOLAR = 0.8, LF_ZEQ = 0.15;
constexpr int LF_CH = 128;       // k per staged chunk
constexpr int LF_FUSED = 8;      // most warps of one m whose sums one CTA collects
constexpr int LF_FUSED_SMEM = 64 * 1024;  // and its shared memory: three CTAs per SM

void lf_zones(const double* z, int npairs, int* n1, int* n2) {
  int i = 0;
  while (i < npairs && z[i] > LF_ZPOLAR) ++i;
  *n1 = i;
  while (i < npairs && z[i] >= LF_ZEQ) ++i;
  *n2 = i;
}

// arguments of a pair's steps: four copies of 1 - z^2 (polar) or z^2
void lf_args(const double* z, int npairs, int n1, float4* out) {
  for (int p = 0; p < npairs; ++p) {
    // the exact value as x + xl
    double x, xl;
    if (p < n1) {
      const double w = 1.0 - z[p], u = 2.0 * w;  // exact
      x = std::fma(-w, w, u);
      xl = std::fma(-w, w, u - x);
    } else {
      x = z[p] * z[p];
      xl = std::fma(z[p], z[p], -x);
    }
    const float h = (float)x;
    float c[4] = {h, h, h, h};
    if (h > 0.f) {
      const float up = nextafterf(h, 2.f) - h;
      const int t = (int)lrint(4.0 * ((x - h) + xl) / up);
      for (int j = 0; j < 4; ++j) c[j] = h + (j < abs(t) ? (t > 0 ? up : -up) : 0.f);
    }
    out[p] = make_float4(c[0], c[1], c[2], c[3]);
  }
}

// One warp's pairs: arguments, states, start indices.  ZONE 0 polar, 1 middle,
// 2 equatorial (one-step: two l, of either parity of l - m, per k).
template <int ZONE, int RP>
struct LfPairs {
  float q1[RP], q2[RP], Z[RP][4];
  int k0[RP], p[RP];
  int kmin, kmax;  // first and last start of the warp's live pairs

  __device__ __forceinline__ void load(const LegArgs<float>& a, int m, int base, int pend) {
    const int lane = threadIdx.x & 31;
    const int none = 0x3fffffff;
    int lo = none, hi = 0;
#pragma unroll
    for (int j = 0; j < RP; ++j) {
      p[j] = base + 32 * j + lane;
      k0[j] = none;
      q1[j] = q2[j] = 0.f;
      float4 z = make_float4(0.f, 0.f, 0.f, 0.f);
      if (p[j] < pend) {
        z = a.zi[p[j]];
        const int64_t o = (int64_t)m * a.ld_seed + p[j];
        const int l = a.ls[o];
        if (l <= a.L) {
          const float2 st = a.sti[o];
          k0[j] = (l - m) >> 1;
          q1[j] = st.x;
          q2[j] = st.y;
          lo = min(lo, k0[j]);
          hi = max(hi, k0[j]);
        }
      }
      Z[j][0] = z.x;
      Z[j][1] = z.y;
      Z[j][2] = z.z;
      Z[j][3] = z.w;
    }
    kmin = __reduce_min_sync(0xffffffffu, lo);
    kmax = __reduce_max_sync(0xffffffffu, hi);
  }
  // the next value of pair j, for the even and the odd sums (ZONE 2: the next
  // q and w), and the state behind it if `on`; u: its k modulo 4
  __device__ __forceinline__ float2 next(float2 r, int j, int u, bool on) {
    const float z = Z[j][u & 3];
    float qe, qo, second;
    if (ZONE == 2) {
      qe = fmaf(r.x, q1[j], -q2[j]);
      qo = fmaf(r.y * z, qe, -q1[j]);
      second = qe;
    } else if (ZONE == 1) {
      qe = qo = fmaf(fmaf(r.x, z, r.y), q1[j], -q2[j]);
      second = q1[j];
    } else {
      second = fmaf(fmaf(r.x, z, r.y), q1[j], q2[j]);
      qe = qo = q1[j] + second;
    }
    if (on) {
      q2[j] = second;
      q1[j] = qo;
    }
    return make_float2(qe, qo);
  }
};

// coefficients of step k: (factor of the argument, constant) from (A, A + B - 2,
// B), or those of l = m + 2k and l + 1 (ZONE 2)
template <int ZONE>
__device__ __forceinline__ float2 lf_step(const LegArgs<float>& a, int m, int k) {
  if (ZONE == 2) {
    const float* c = a.c + lm_off(a.Lc, m) + 2 * k;
    return make_float2(c[0], m + 2 * k + 1 <= a.L ? c[1] : 0.f);
  }
  const float4 t = a.rf[(lm_off(a.Lc, m) >> 1) + m + k];
  return ZONE == 0 ? make_float2(-t.x, t.y) : make_float2(t.x, t.z);
}

// factor of the odd sums (on the equator they are zero)
template <int ZONE>
__device__ __forceinline__ float lf_odd(float z) { return ZONE < 2 ? z : z > 0.f ? 1.f / z : 0.f; }

struct LfStage {
  float2 r[LF_CH];
  float4 c[LF_CH];
};

// ---- synthesis ---------------------------------------------------------------

template <int ZONE, int RP>
__device__ __forceinline__ void lf_synth(const LegArgs<float>& a, LfStage& sh, int m, int base, int pend) {
  const int L = a.L, lane = threadIdx.x;
  const int nk = (L - m) / 2 + 1;
  LfPairs<ZONE, RP> s;
  s.load(a, m, base, pend);
  float cx[RP], cy[RP], dx[RP], dy[RP];
#pragma unroll
  for (int j = 0; j < RP; ++j) cx[j] = cy[j] = dx[j] = dy[j] = 0.f;
  const int64_t offa = lm_off(L, m), offk = (lm_off(a.Lc, m) >> 1) + m;
  // chunks start at a multiple of 8
  for (int kc = s.kmin & ~7; kc < nk; kc += LF_CH) {
    const int n = min(LF_CH, nk - kc);
    __syncwarp();
#pragma unroll
    for (int i = lane; i < LF_CH; i += 32) {
      const int k = kc + i;
      if (i < n) {
        const int l = m + 2 * k;
        const float2* x = a.alm + offa + 2 * k;
        const float2 x0 = x[0];
        const float2 x1 = l + 1 <= L ? x[1] : make_float2(0.f, 0.f);
        const float2 x2 = ZONE < 2 && l + 2 <= L ? x[2] : make_float2(0.f, 0.f);
        float f0, f1, f2 = 0.f;
        if (ZONE == 2) {
          const float* s1 = a.s + lm_off(a.Lc, m) + 2 * k;
          f0 = s1[0];
          f1 = l + 1 <= L ? s1[1] : 0.f;
        } else {
          const float4 g = a.cf[offk + k];
          f0 = g.y;
          f1 = g.x;
          f2 = g.z;
        }
        if (a.dl) {
          f0 *= a.dl[l];
          f1 *= l + 1 <= L ? a.dl[l + 1] : 0.f;
          f2 *= l + 2 <= L ? a.dl[l + 2] : 0.f;
        }
        float4 c = make_float4(fmaf(f0, x0.x, f2 * x2.x), fmaf(f0, x0.y, f2 * x2.y), f1 * x1.x, f1 * x1.y);
        if (m == 0) c.y = c.w = 0.f;
        sh.c[i] = c;
        sh.r[i] = lf_step<ZONE>(a, m, k);
      }
    }
    __syncwarp();
    for (int i8 = 0; i8 < n; i8 += 8) {
      const int k = kc + i8;
      if (s.kmin >= k + 8) continue;
      if (s.kmax <= k && i8 + 8 <= n) {
#pragma unroll
        for (int u = 0; u < 8; ++u) {
          const float2 r = sh.r[i8 + u];
          const float4 c = sh.c[i8 + u];
#pragma unroll
          for (int j = 0; j < RP; ++j) {
            const float2 q = s.next(r, j, u, true);
            cx[j] = fmaf(q.x, c.x, cx[j]);
            cy[j] = fmaf(q.x, c.y, cy[j]);
            dx[j] = fmaf(q.y, c.z, dx[j]);
            dy[j] = fmaf(q.y, c.w, dy[j]);
          }
        }
      } else {
#pragma unroll
        for (int u = 0; u < 8; ++u) {
          if (i8 + u >= n) break;
          const float2 r = sh.r[i8 + u];
          const float4 c = sh.c[i8 + u];
#pragma unroll
          for (int j = 0; j < RP; ++j) {
            const bool on = k + u >= s.k0[j];
            const float2 q = s.next(r, j, u, on);
            if (on) {
              cx[j] = fmaf(q.x, c.x, cx[j]);
              cy[j] = fmaf(q.x, c.y, cy[j]);
              dx[j] = fmaf(q.y, c.z, dx[j]);
              dy[j] = fmaf(q.y, c.w, dy[j]);
            }
          }
        }
      }
    }
  }
#pragma unroll
  for (int j = 0; j < RP; ++j)
    if (s.p[j] < pend) {
      const int rn = s.p[j], rs = a.nring - 1 - rn;
      const float z = lf_odd<ZONE>(a.z[rn]);
      a.phase[(int64_t)rn * a.ldp + m] = make_float2(fmaf(z, dx[j], cx[j]), fmaf(z, dy[j], cy[j]));
      if (rs != rn) a.phase[(int64_t)rs * a.ldp + m] = make_float2(fmaf(-z, dx[j], cx[j]), fmaf(-z, dy[j], cy[j]));
    }
}

// warp blocks of a zone of n pairs
template <int RP>
__host__ __device__ inline int lf_blocks(int n) { return (n + 32 * RP - 1) / (32 * RP); }

// The equatorial zone, whose steps are the longest and whose pairs often fill
// less than half of a warp's: half as many per thread then.
template <int RP>
__device__ __forceinline__ void lf_synth_eq(const LegArgs<float>& a, LfStage& sh, int m, int base) {
  if (a.npairs - base <= 16 * RP) lf_synth<2, RP / 2>(a, sh, m, base, a.npairs);
  else lf_synth<2, RP>(a, sh, m, base, a.npairs);
}

template <int RP, int MT>
__global__ void __launch_bounds__(32) lf_synth_kernel(LegArgs<float> a) {
  __shared__ LfStage sh;
  const int b0 = lf_blocks<RP>(a.n1), b1 = lf_blocks<RP>(a.n2 - a.n1);
  const int b = blockIdx.x;
#pragma unroll 1
  for (int mi = 0; mi < MT; ++mi) {
    const int m = mi == 0 ? (int)blockIdx.y : a.L - (int)blockIdx.y;
    if (mi > 0 && m <= (int)blockIdx.y) break;
    if (b < b0) lf_synth<0, RP>(a, sh, m, b * 32 * RP, a.n1);
    else if (b < b0 + b1) lf_synth<1, RP>(a, sh, m, a.n1 + (b - b0) * 32 * RP, a.n2);
    else lf_synth_eq<RP>(a, sh, m, a.n2 + (b - b0 - b1) * 32 * RP);
    __syncwarp();
  }
}

// ---- adjoint -----------------------------------------------------------------
// u_k = sum_pairs q_k (G_m(z) + G_m(-z)), v_k = sum_pairs q_k z (G_m(z) - G_m(-z));
// a_o = sigma_k v_k, a_{o-1} += sigma_k e_o u_k, a_{o+1} += sigma_k e_{o+1} u_k.
// ZONE 2: the sums of q_l (w_l / z) themselves, l = m + 2k and m + 2k + 1; a_l = s_l times it.
// The four real sums of a k over a thread's RP pairs go to a shared-memory
// row; per 8 k, lane (k, part) adds every fourth lane's entry and two exchange
// steps leave one of the four sums per lane, 128 contiguous bytes of the
// warp's row.  Rows are 36 entries apart: 16-byte reads of two rows fall on
// different banks.
constexpr int LF_RS = 36;
typedef unsigned long long lf_u64;
__device__ __forceinline__ lf_u64 lf_add2(lf_u64 a, lf_u64 b) {
  lf_u64 d;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
  return d;
}

struct LfAdjStage {
  float2 r[LF_CH];
  float4 b[8][LF_RS];
};

// row: this warp's sums, 4 floats per k
template <int ZONE, int RP>
__device__ __forceinline__ void lf_adjoint(const LegArgs<float>& a, LfAdjStage& sh, int m, int base, int pend,
                                           float* row) {
  const int L = a.L, lane = threadIdx.x & 31;
  const int nk = (L - m) / 2 + 1;
  LfPairs<ZONE, RP> s;
  s.load(a, m, base, pend);
  float2 ge[RP], go[RP];
#pragma unroll
  for (int j = 0; j < RP; ++j) {
    ge[j] = go[j] = make_float2(0.f, 0.f);
    if (s.k0[j] < nk) {
      const int rn = s.p[j], rs = a.nring - 1 - rn;
      const float z = lf_odd<ZONE>(a.z[rn]);
      const float2 gn = a.phase[(int64_t)rn * a.ldp + m];
      const float2 gs = rs != rn ? a.phase[(int64_t)rs * a.ldp + m] : make_float2(0.f, 0.f);
      ge[j] = cadd(gn, gs);
      go[j] = make_float2(z * (gn.x - gs.x), z * (gn.y - gs.y));
    }
  }
  const int kbeg = min(s.kmin, nk) & ~7;
  for (int i = lane; i < 4 * kbeg; i += 32) row[i] = 0.f;  // before the first start
  if (s.kmin >= nk) {
    for (int i = 4 * kbeg + lane; i < 4 * nk; i += 32) row[i] = 0.f;
    return;
  }
  for (int kc = kbeg; kc < nk; kc += LF_CH) {
    const int n = min(LF_CH, nk - kc);
    __syncwarp();
#pragma unroll
    for (int i = lane; i < LF_CH; i += 32)
      if (i < n) sh.r[i] = lf_step<ZONE>(a, m, kc + i);
    __syncwarp();
    for (int i8 = 0; i8 < n; i8 += 8) {
      const int k = kc + i8;
      const bool full = s.kmax <= k && i8 + 8 <= n;
      if (full) {
#pragma unroll
        for (int u = 0; u < 8; ++u) {
          const float2 r = sh.r[i8 + u];
          float4 t = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
          for (int j = 0; j < RP; ++j) {
            const float2 q = s.next(r, j, u, true);
            t.x = fmaf(q.x, ge[j].x, t.x);
            t.y = fmaf(q.x, ge[j].y, t.y);
            t.z = fmaf(q.y, go[j].x, t.z);
            t.w = fmaf(q.y, go[j].y, t.w);
          }
          sh.b[u][lane] = t;
        }
      } else {
#pragma unroll
        for (int u = 0; u < 8; ++u) {
          float4 t = make_float4(0.f, 0.f, 0.f, 0.f);
          if (i8 + u < n) {
            const float2 r = sh.r[i8 + u];
#pragma unroll
            for (int j = 0; j < RP; ++j) {
              const bool on = k + u >= s.k0[j];
              const float2 q = s.next(r, j, u, on);
              if (on) {
                t.x = fmaf(q.x, ge[j].x, t.x);
                t.y = fmaf(q.x, ge[j].y, t.y);
                t.z = fmaf(q.y, go[j].x, t.z);
                t.w = fmaf(q.y, go[j].y, t.w);
              }
            }
          }
          sh.b[u][lane] = t;
        }
      }
      __syncwarp();
      const int u = lane >> 2, part = lane & 3;
      const ulonglong2* e = reinterpret_cast<const ulonglong2*>(&sh.b[u][part]);
      ulonglong2 t = e[0];
#pragma unroll
      for (int i = 1; i < 8; ++i) {
        const ulonglong2 w = e[4 * i];
        t.x = lf_add2(t.x, w.x);
        t.y = lf_add2(t.y, w.y);
      }
      __syncwarp();  // the rows are rewritten by the next group
      const float2 tu = *reinterpret_cast<const float2*>(&t.x), tv = *reinterpret_cast<const float2*>(&t.y);
      // parts 0, 1 keep u and 2, 3 keep v; then even parts the real part
      const bool hi = part & 2, im = part & 1;
      const float s0 = __shfl_xor_sync(0xffffffffu, hi ? tu.x : tv.x, 2);
      const float s1 = __shfl_xor_sync(0xffffffffu, hi ? tu.y : tv.y, 2);
      const float w0 = (hi ? tv.x : tu.x) + s0, w1 = (hi ? tv.y : tu.y) + s1;
      float w = (im ? w1 : w0) + __shfl_xor_sync(0xffffffffu, im ? w0 : w1, 1);
      if (i8 + u < n) row[4 * (k + u) + part] = w;
    }
  }
}

template <int RP>
__device__ __forceinline__ void lf_adjoint_eq(const LegArgs<float>& a, LfAdjStage& sh, int m, int base, float* row) {
  if (a.npairs - base <= 16 * RP) lf_adjoint<2, RP / 2>(a, sh, m, base, a.npairs, row);
  else lf_adjoint<2, RP>(a, sh, m, base, a.npairs, row);
}

// Warps per SM that the registers leave room for.  32, all that an SM takes of
// CTAs this small, cost 8 registers at RP = 4 (72 without the bound): adjoint at
// Nside 2048 / lmax 3000 2610 -> 2577 us, 1024 / 2047 677 -> 661, 512 / 1023 134 -> 132
// (in A there, with a mask, 108 -> 111).
template <int RP, int MT>
__global__ void __launch_bounds__(32, RP <= 2 ? 32 : RP == 4 ? (MT == 1 ? 32 : 24) : RP == 8 ? 16 : 8) lf_adjoint_kernel(LegArgs<float> a, float* partial, int64_t nkk) {
  __shared__ LfAdjStage sh;
  const int b0 = lf_blocks<RP>(a.n1), b1 = lf_blocks<RP>(a.n2 - a.n1);
  const int b = blockIdx.x;
#pragma unroll 1
  for (int mi = 0; mi < MT; ++mi) {
    const int m = mi == 0 ? (int)blockIdx.y : a.L - (int)blockIdx.y;
    if (mi > 0 && m <= (int)blockIdx.y) break;
    float* row = partial + ((int64_t)b * nkk + ((lm_off(a.L, m) >> 1) + m)) * 4;
    if (b < b0) lf_adjoint<0, RP>(a, sh, m, b * 32 * RP, a.n1, row);
    else if (b < b0 + b1) lf_adjoint<1, RP>(a, sh, m, a.n1 + (b - b0) * 32 * RP, a.n2, row);
    else lf_adjoint_eq<RP>(a, sh, m, a.n2 + (b - b0 - b1) * 32 * RP, row);
    __syncwarp();
  }
}

// a_l (l = m + 2k + w) from the summed (u_k, v_k), u_{k-1} and the one-step
// zone's sums q, and the epilogue of leg_finalize_kernel
__device__ __forceinline__ void lf_emit(const LegArgs<float>& a, const FinalizeArgs<float>& f, int m, int k, float4 t,
                                        float2 um, float4 q) {
  const int L = a.L;
  const float* sl = a.s + lm_off(a.Lc, m) + 2 * k;
  const int64_t ok = (lm_off(a.Lc, m) >> 1) + m + k;
  const float4 g = a.cf[ok];
  const float g1 = k > 0 ? a.cf[ok - 1].z : 0.f;
#pragma unroll
  for (int w = 0; w < 2; ++w) {
    const int l = m + 2 * k + w;
    if (l > L) break;
    float2 y = w == 0 ? make_float2(fmaf(g.y, t.x, g1 * um.x), fmaf(g.y, t.y, g1 * um.y))
                      : make_float2(g.x * t.z, g.x * t.w);
    y.x = fmaf(sl[w], w == 0 ? q.x : q.z, y.x);
    y.y = fmaf(sl[w], w == 0 ? q.y : q.w, y.y);
    const int64_t i = lm_off(L, m) + (l - m);
    if (f.dl_out) y = cscale(y, f.dl_out[l]);
    if (f.dadd) {
      const float2 x = f.xadd[i];
      y.x = fmaf(f.dadd[l], x.x, y.x);
      y.y = fmaf(f.dadd[l], x.y, y.y);
    }
    if (f.bsub) {
      const float2 b = f.bsub[i];
      y = make_float2(b.x - y.x, b.y - y.y);
    }
    if (m == 0) y.y = 0.f;
    if (f.accumulate) y = cadd(y, f.out[i]);
    f.out[i] = y;
  }
}

// The warps' rows in a fixed order (n2s of the two-step zones, then the one-step
// zone's); thread = one k.
__global__ void __launch_bounds__(128) lf_finalize_kernel(LegArgs<float> a, FinalizeArgs<float> f, const float4* partial,
                                                          int64_t nkk, int n2s, int nblk) {
  const int m = blockIdx.y;
  const int nk = (a.L - m) / 2 + 1;
  const int k = blockIdx.x * blockDim.x + threadIdx.x;
  if ((int)(blockIdx.x * blockDim.x) >= nk) return;  // whole CTA
  const float4* row = partial + ((lm_off(a.L, m) >> 1) + m);
  // two-step rows to t, one-step rows to q, all loads in one loop
  auto sum = [&](int kk, float4& t, float4& q) {
    t = q = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll 4
    for (int b = 0; b < nblk; ++b) {
      const float4 w = row[b * nkk + kk];
      const bool two = b < n2s;
      t = make_float4(t.x + (two ? w.x : 0.f), t.y + (two ? w.y : 0.f), t.z + (two ? w.z : 0.f), t.w + (two ? w.w : 0.f));
      q = make_float4(q.x + (two ? 0.f : w.x), q.y + (two ? 0.f : w.y), q.z + (two ? 0.f : w.z), q.w + (two ? 0.f : w.w));
    }
  };
  float4 t = make_float4(0.f, 0.f, 0.f, 0.f), q = t;
  if (k < nk) sum(k, t, q);
  float2 um = make_float2(__shfl_up_sync(0xffffffffu, t.x, 1), __shfl_up_sync(0xffffffffu, t.y, 1));
  if (k >= nk) return;
  if ((threadIdx.x & 31) == 0) {
    um = make_float2(0.f, 0.f);
    if (k > 0) {
      float4 w, wq;
      sum(k - 1, w, wq);
      um = make_float2(w.x, w.y);
    }
  }
  lf_emit(a, f, m, k, t, um, q);
}

// All warps of one m in one CTA (grids of few pairs): the rows stay in shared
// memory and the same kernel finishes the coefficients -- one launch instead
// of two, no partial rows.
template <int RP>
__global__ void __launch_bounds__(32 * LF_FUSED) lf_adjoint_fused_kernel(LegArgs<float> a, FinalizeArgs<float> f) {
  extern __shared__ __align__(16) unsigned char lf_dyn[];
  const int b0 = lf_blocks<RP>(a.n1), b1 = lf_blocks<RP>(a.n2 - a.n1);
  const int b = threadIdx.x >> 5, nw = blockDim.x >> 5, m = blockIdx.x;
  const int nk = (a.L - m) / 2 + 1;
  LfAdjStage& sh = reinterpret_cast<LfAdjStage*>(lf_dyn)[b];
  float4* rows = reinterpret_cast<float4*>(lf_dyn + nw * sizeof(LfAdjStage));
  const int ld = a.L / 2 + 1;
  float* row = reinterpret_cast<float*>(rows + b * ld);
  if (b < b0) lf_adjoint<0, RP>(a, sh, m, b * 32 * RP, a.n1, row);
  else if (b < b0 + b1) lf_adjoint<1, RP>(a, sh, m, a.n1 + (b - b0) * 32 * RP, a.n2, row);
  else lf_adjoint_eq<RP>(a, sh, m, a.n2 + (b - b0 - b1) * 32 * RP, row);
  __syncthreads();
  for (int k = threadIdx.x; k < nk; k += blockDim.x) {
    float4 t = make_float4(0.f, 0.f, 0.f, 0.f), q = t;
    float2 um = make_float2(0.f, 0.f);
    const int n2s = b0 + b1;
    for (int w = 0; w < n2s; ++w) {
      const float4 x = rows[w * ld + k];
      t = make_float4(t.x + x.x, t.y + x.y, t.z + x.z, t.w + x.w);
      if (k > 0) {
        const float4 y = rows[w * ld + k - 1];
        um = make_float2(um.x + y.x, um.y + y.y);
      }
    }
    for (int w = n2s; w < nw; ++w) {
      const float4 x = rows[w * ld + k];
      q = make_float4(q.x + x.x, q.y + x.y, q.z + x.z, q.w + x.w);
    }
    lf_emit(a, f, m, k, t, um, q);
  }
}

// ---- launchers ---------------------------------------------------------------

// warps of one m: those of the two-step zones, and of all zones
static int lf_blocks2(const LegArgs<float>& a, int rp) {
  auto nb = [&](int n) { return (n + 32 * rp - 1) / (32 * rp); };
  return nb(a.n1) + nb(a.n2 - a.n1);
}
static int lf_nblocks(const LegArgs<float>& a, int rp) {
  return lf_blocks2(a, rp) + (a.npairs - a.n2 + 32 * rp - 1) / (32 * rp);
}
int64_t lf_partial_bytes(int npairs, int L) {
  return (int64_t)((npairs + 63) / 64 + 3) * ds_len(L) * (int64_t)sizeof(float4);
}

// ring pairs per thread where nothing was tuned: 4, or 2 where 4 would leave
// fewer than `least` warps per SM.  Measured (us, 2 against 4 pairs): synthesis
// Nside 512 / 1023 81 : 94, Nside 1024 / 2047 504 : 497; adjoint Nside 128 / 384
// 19 : 23, Nside 256 / 512 36 : 33.
static int lf_default_rp(const LegArgs<float>& a, int least) {
  return (int64_t)lf_nblocks(a, 4) * (a.L + 1) < 152 * (int64_t)least ? 2 : 4;
}

template <int RP>
static void lf_synth_launch(const LegArgs<float>& a, cudaStream_t st) {
  const int nb = lf_nblocks(a, RP);
  if (a.mt_synth == 2) lf_synth_kernel<RP, 2><<<dim3(nb, (a.L + 2) / 2), 32, 0, st>>>(a);
  else lf_synth_kernel<RP, 1><<<dim3(nb, a.L + 1), 32, 0, st>>>(a);
  count_launch();
}

int launch_lf_synth(const LegArgs<float>& a, cudaStream_t st) {
  const int rp = a.rp_synth ? a.rp_synth : lf_default_rp(a, 128);
  if (rp == 2) lf_synth_launch<2>(a, st);
  else if (rp == 8) lf_synth_launch<8>(a, st);
  else lf_synth_launch<4>(a, st);
  CR_CHECK_LAUNCH("lf_synth_kernel");
  return CR_OK;
}

template <int RP>
static int lf_adjoint_launch(const LegArgs<float>& a, const FinalizeArgs<float>& f, cudaStream_t st) {
  const int nb = lf_nblocks(a, RP);
  const size_t smem = nb * (sizeof(LfAdjStage) + (size_t)(a.L / 2 + 1) * sizeof(float4));
  if constexpr (RP <= 4) {
    // few pairs: one CTA per m.  The kernel's limit is the most it may take, not
    // this launch's size, which another thread's launch could exceed.
    if (a.mt_adj == 1 && nb <= LF_FUSED && smem <= LF_FUSED_SMEM) {
      CR_CUDA(cudaFuncSetAttribute(lf_adjoint_fused_kernel<RP>, cudaFuncAttributeMaxDynamicSharedMemorySize, LF_FUSED_SMEM));
      { lf_adjoint_fused_kernel<RP><<<a.L + 1, 32 * nb, smem, st>>>(a, f); count_launch(); }
      CR_CHECK_LAUNCH("lf_adjoint_fused_kernel");
      return CR_OK;
    }
  }
  float* part = reinterpret_cast<float*>(a.partial);
  const int64_t nkk = ds_len(a.L);
  if (a.mt_adj == 2) lf_adjoint_kernel<RP, 2><<<dim3(nb, (a.L + 2) / 2), 32, 0, st>>>(a, part, nkk);
  else lf_adjoint_kernel<RP, 1><<<dim3(nb, a.L + 1), 32, 0, st>>>(a, part, nkk);
  count_launch();
  CR_CHECK_LAUNCH("lf_adjoint_kernel");
  const dim3 grid((a.L / 2 + 1 + 127) / 128, a.L + 1);
  { lf_finalize_kernel<<<grid, 128, 0, st>>>(a, f, reinterpret_cast<const float4*>(part), nkk,
                                           lf_blocks2(a, RP), nb); count_launch(); }
  CR_CHECK_LAUNCH("lf_finalize_kernel");
  return CR_OK;
}

int launch_lf_adjoint(const LegArgs<float>& a, const FinalizeArgs<float>& f, cudaStream_t st) {
  const int rp = a.rp_adj ? a.rp_adj : lf_default_rp(a, 16);
  if (rp == 2) return lf_adjoint_launch<2>(a, f, st);
  if (rp == 8) return lf_adjoint_launch<8>(a, f, st);
  if (rp == 16) return lf_adjoint_launch<16>(a, f, st);
  return lf_adjoint_launch<4>(a, f, st);
}

}  // namespace cr
