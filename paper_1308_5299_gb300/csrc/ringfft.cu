// Per-ring azimuthal stages of synthesis Y and adjoint synthesis Y^T
// (Section 2.1; the per-ring DFTs of Section 3.3), without cuFFT.
//
// Ring r has n (even) pixels at phi_j = pi (2 j + s) / n, s in {0, 1} (HEALPix
// and Gauss-Legendre rings both have this form).
//
// Synthesis of a real field from F_m (m = 0..L):
//   map_j = Re sum_{m} w_m F_m e^{i m phi_j},  w_0 = 1, w_{m>0} = 2
//         = sum_{b<n} H'_b e^{2 pi i b j / n},
//   H_b  = sum_{m = b mod n} w_m F_m e^{i pi s m / n}  (band limits above n/2
//          fold onto the ring's n bins), H'_b = (H_b + conj H_{n-b}) / 2.
// H' is Hermitian, so the length-n real inverse DFT is done as one complex
// inverse DFT of length nh = n/2 on Z_k = (H'_k + conj H'_{nh-k})
// + i w^k (H'_k - conj H'_{nh-k}), w = e^{2 pi i / n}; z = IDFT(Z) gives
// map_{2t} = Re z_t, map_{2t+1} = Im z_t.
// Adjoint: Yhat_b = sum_j y_j e^{-2 pi i b j / n} from a length-nh forward
// DFT of z_t = y_{2t} + i y_{2t+1}; then G_m = e^{-i pi s m / n} Yhat_{m mod n}
// (conjugate-symmetric extension for m mod n > n/2): the exact transpose of
// the folding above.
//
// Length-nh DFTs: radix-2 in shared memory when nh is a power of two,
// otherwise Bluestein's chirp-z with a power-of-two convolution of size
// M >= 2 nh - 1 (forward FFT from natural to bit-reversed order, pointwise
// product with the precomputed kernel spectrum stored in bit-reversed order,
// inverse FFT back to natural order: no bit-reversal passes).  The chirp
// e^{i pi k^2 / nh} = e^{i pi (2 k^2 mod 2n) / n} comes from an exact integer
// reduction into the ring length's table of e^{i pi u / n}, u < 2n.
//
// One CTA per ring and right-hand side; mode 2 keeps the ring's map in shared
// memory between the synthesis and the adjoint (map * N^-1 never touches HBM).
#include <algorithm>
#include <cstdio>
#include <map>
#include <vector>

#include "common.cuh"
#include "kernels.h"

namespace cr {

constexpr int RF_NT = 256;
// The most shared memory of a CTA.  The kernels' limit is set to it whatever a
// launch takes: it is one per kernel and process, so a limit of a launch's own
// size could fall below that of another thread's launch.
constexpr int RF_SMEM = 227 * 1024;

// Shared-memory position of FFT buffer element i: bits 4..15 XOR-folded into
// bits 0..3 (a bijection on [0, 2^16)).  With 8-byte elements a bank pair
// holds positions equal mod 16; the fold spreads every access pattern of
// the kernels below -- consecutive, the radix-8 passes' strides 8^p, and the
// bit-reversed scatter and gather -- over all 16 bank pairs.
__device__ __forceinline__ int swz(int i) { return i ^ (((i >> 4) ^ (i >> 8) ^ (i >> 12)) & 15); }

__device__ __forceinline__ int bitrev(int k, int logM) {
  return logM ? (int)(__brev((unsigned)k) >> (32 - logM)) : 0;
}

// e^{-2 pi i v / 16}, v < 4, and the half steps of 32: the constant factors of
// the twiddles inside one pass (cos and sin of 2 pi v / 16)
__device__ constexpr double RC16[4] = {1.0, 0.923879532511286756128, 0.707106781186547524401, 0.382683432365089771728};
__device__ constexpr double RS16[4] = {0.0, 0.382683432365089771728, 0.707106781186547524401, 0.923879532511286756128};

// Radix-2 butterfly a' = a + w b, b' = a - w b in six fused operations: a' by
// two per component, b' = 2 a - a'.  (Both transforms below are arranged so
// that the twiddle multiplies an input; the form with the twiddle on the
// difference takes eight.)
template <typename C>
__device__ __forceinline__ void bf_fma(C& a, C& b, C w) {
  using T = decltype(C().x);
  const T x = fma(w.x, b.x, fma(-w.y, b.y, a.x));
  const T y = fma(w.x, b.y, fma(w.y, b.x, a.y));
  b = mk(fma((T)2, a.x, -x), fma((T)2, a.y, -y));
  a = mk(x, y);
}
// the same with w = 1, and with w = sign i
template <typename C>
__device__ __forceinline__ void bf_one(C& a, C& b) {
  const C t = b;
  b = csub(a, t);
  a = cadd(a, t);
}
template <typename C>
__device__ __forceinline__ void bf_rot(C& a, C& b, int sign) {
  const C t = sign > 0 ? mk(-b.y, b.x) : mk(b.y, -b.x);
  b = csub(a, t);
  a = cadd(a, t);
}

// One pass of NS consecutive radix-2 stages on groups of 2^NS elements
// j0 + i h (i < 2^NS) held in registers.
//  - FWD (natural input, bit-reversed output, e^{-}): a block of the pass is a
//    polynomial modulo x^len - c^2, split into x^(len/2) -+ c; at depth d
//    block B has c = e^{-2 pi i brv_d(B) / 2^(d+1)}, so a group has one c per
//    stage, c_s = e^{-2 pi i brv_t(B) / 2^(t+s+1)}, times e^{-2 pi i brv_s(j) /
//    2^(s+1)} for the j-th part of stage s.  post (may be null): the output is
//    multiplied by post at its positions (the pointwise product of a
//    convolution, fused into the last pass).
//  - inverse (bit-reversed input, natural output, e^{+}): stage s joins spans
//    2^s h with w = e^{2 pi i (k + u h) / (2^(s+1) h)} = c_s e^{2 pi i u / 2^(s+1)}.
// Either way a stage's upper half of constants is i (or -i) times the lower
// half, one table value per stage and group serves it, and the pass whose
// table values are all 1 (TRIV: the first of either transform) has constant
// twiddles only.
template <typename C, int NS, bool FWD, bool TRIV>
__device__ __forceinline__ void fft_pass(C* buf, int M, int lg, const C* __restrict__ tw, int Mmax,
                                         const C* __restrict__ post) {
  using T = decltype(C().x);
  constexpr int R = 1 << NS;
  constexpr int sign = FWD ? -1 : 1;
  // FWD: lg = depth t of the pass (2^t blocks), h = len / R; inverse: h = 2^lg
  const int lh = FWD ? (31 - __clz(M)) - lg - NS : lg;
  const int h = 1 << lh;
  const int ng = M >> NS;
  for (int g = threadIdx.x; g < ng; g += blockDim.x) {
    const int k = g & (h - 1), B = g >> lh;
    const int j0 = (B << (lh + NS)) + k;
    C c[NS];
    if (!TRIV) {
      const int idx = FWD ? (lg ? (int)(__brev((unsigned)B) >> (32 - lg)) : 0) : k;
#pragma unroll
      for (int s = 0; s < NS; ++s) {
        c[s] = tw[idx * (Mmax >> (FWD ? lg + s + 1 : lh + s + 1))];
        if (!FWD) c[s] = cconj(c[s]);
      }
    }
    C e[R];
#pragma unroll
    for (int t = 0; t < R; ++t) e[t] = buf[swz(j0 + t * h)];
#pragma unroll
    for (int s = 0; s < NS; ++s) {
      // span of the stage in i; q-th twiddle of the stage's 2^s
      const int S = FWD ? R >> (s + 1) : 1 << s;
#pragma unroll
      for (int q = 0; q < (1 << s); ++q) {
        // constant e^{sign 2 pi i v / 2^(s+1)}: v = q, or its bit reversal; 16ths
        int v = q;
        if (FWD) {
          v = 0;
#pragma unroll
          for (int z = 0; z < s; ++z) v |= ((q >> z) & 1) << (s - 1 - z);
        }
        const int v16 = v << (3 - s);
        const bool rot = v16 >= 4;  // an extra factor sign i
        const int vv = v16 & 3;
        C w = mk((T)RC16[vv], (T)(sign > 0 ? RS16[vv] : -RS16[vv]));
        if (!TRIV) w = vv ? cmul(c[s], w) : c[s];
        if (rot) w = sign > 0 ? mk(-w.y, w.x) : mk(w.y, -w.x);
#pragma unroll
        for (int r = 0; r < R / 2 / (1 << s); ++r) {
          const int i = FWD ? q * 2 * S + r : r * 2 * S + q;
          if (TRIV && vv == 0) {
            if (rot) bf_rot(e[i], e[i + S], sign);
            else bf_one(e[i], e[i + S]);
          } else {
            bf_fma(e[i], e[i + S], w);
          }
        }
      }
    }
    // the last pass: h = 1, and a thread's R consecutive values in 16-byte loads (A
    // in FP32, Nside 2048 / 1024 / 512: 857 / 247 / 78 -> 845 / 232 / 75 us; one
    // value a load touched every line R times)
    if (post) {
      if constexpr (sizeof(T) == 4) {
#pragma unroll
        for (int t = 0; t < R; t += 2) {
          const float4 v = *reinterpret_cast<const float4*>(post + j0 + t);
          e[t] = cmul(e[t], mk(v.x, v.y));
          e[t + 1] = cmul(e[t + 1], mk(v.z, v.w));
        }
      } else {
#pragma unroll
        for (int t = 0; t < R; ++t) e[t] = cmul(e[t], post[j0 + t]);
      }
    }
#pragma unroll
    for (int t = 0; t < R; ++t) buf[swz(j0 + t * h)] = e[t];
  }
}

// Stages per pass.  FP32: 4 in BIG (rings with M >= 4096: fewer barriers and
// shared-memory round trips), 3 otherwise (fewer registers, so more CTAs per
// SM), also where that leaves threads without a group: small rings wait for
// barriers and round trips, not for arithmetic (A at Nside 64, lmax 383: 21.9 us
// with one group per thread at least, 18.3 us so).  FP64 keeps a quarter of the
// threads busy, as an SM's FP64 units are spread over its four schedulers
// (Nside 32, lmax 95: 29.2 us with a group per thread, 27.4 us with a quarter,
// 34.7 us without a limit).
template <typename C, bool FWD, bool TRIV, bool BIG>
__device__ __forceinline__ void fft_pass_ns(int ns, C* buf, int M, int lg, const C* __restrict__ tw, int Mmax,
                                            const C* __restrict__ post) {
  if (BIG && ns == 4) fft_pass<C, 4, FWD, TRIV>(buf, M, lg, tw, Mmax, post);
  else if (ns >= 3) fft_pass<C, 3, FWD, TRIV>(buf, M, lg, tw, Mmax, post);
  else if (ns == 2) fft_pass<C, 2, FWD, TRIV>(buf, M, lg, tw, Mmax, post);
  else fft_pass<C, 1, FWD, TRIV>(buf, M, lg, tw, Mmax, post);
}

// In-place transforms, one barrier per pass: inverse (e^{+2 pi i jk/M},
// unnormalised) from bit-reversed to natural order, forward from natural to
// bit-reversed order.
template <bool FWD, bool BIG, typename C>
__device__ void fft_run(C* buf, int M, int logM, const C* __restrict__ tw, int Mmax,
                        const C* __restrict__ post = nullptr) {
  const int cap = BIG ? 4 : sizeof(C) == 8 ? 3 : max(1, min(3, logM - 29 + __clz((int)blockDim.x)));
  int lg = 0;
  while (lg < logM) {
    const int ns = min(cap, logM - lg);
    const C* pp = lg + ns == logM ? post : nullptr;
    if (lg == 0) fft_pass_ns<C, FWD, true, BIG>(ns, buf, M, lg, tw, Mmax, pp);
    else fft_pass_ns<C, FWD, false, BIG>(ns, buf, M, lg, tw, Mmax, pp);
    __syncthreads();
    lg += ns;
  }
  if (logM == 0 && post && threadIdx.x == 0) buf[swz(0)] = cmul(buf[swz(0)], post[0]);
  if (logM == 0 && post) __syncthreads();
}

// CTAs per SM that the register allocation leaves room for: FP32 rings are bound
// by the latency of their barriers and shared-memory round trips, so resident
// CTAs count.  A (FP32, L = 2 Nside - 1; us at Nside 2048 / 1024 / 512) with
// (BIG, other) CTAs unbounded: 1109 / 364 / 105; (3, -) 974 / 340 / 106;
// (4, -) 932 / 315 / 106; (4, 5) 919 / 274 / 83; (4, 6) 920 / 271 / 85; (4, 8)
// 934 / 282 / 97; three stages per pass in BIG instead of four: (4, -) 999.
// (With later changes to the folds and the loads these became 845 / 232 / 75.)
// FP64 rings are bound by the FP64 pipe; 2 CTAs hold them to 128 registers
// instead of 138 (A at Nside 1024, lmax 2047 2574 -> 2389 us, Nside 2048, lmax
// 3000 10.45 -> 10.07 ms, eight right-hand sides at Nside 512 4.46 -> 4.20 ms;
// Nside 128, lmax 383 57 -> 63 us; with 3 CTAs the same within 3 %).
template <typename T, int MODE, bool BIG>
__global__ void __launch_bounds__(RF_NT, sizeof(T) == 8 ? 2 : BIG ? 4 : 5) ring_fft_kernel(RingArgs<T> a) {
  using C = typename Tr<T>::C;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  C* buf = reinterpret_cast<C*>(smem_raw);
  const int r = a.rings[a.rbase + blockIdx.x];
  const RingFFT f = a.fft[r];
  const C* __restrict__ tab = a.tab + f.tab;
  const C* __restrict__ vh = a.vhat + f.vhat;
  const int n = f.n, nh = f.nh, M = f.M, lg = f.logM;
  const int twon = 2 * n;
  C* row = a.phase + blockIdx.y * a.ld_phase + (int64_t)r * a.ldp;  // blockIdx.y: right-hand side
  const int L = a.L;
  const int tid = threadIdx.x;
  const int NT = blockDim.x;
  // rings with fewer bins than rows may keep the row in shared memory behind the
  // FFT buffer
  const bool staged = a.stage && n <= L;
  C* srow = buf + a.stage;
  if (MODE == 2 && a.live && !a.live[r]) {
    if (min(r, a.nring - 1 - r) < a.np_live)
      for (int m = tid; m <= L; m += NT) row[m] = mk((T)0, (T)0);
    return;
  }
  // e^{i pi (2 k^2 mod 2n) / n}; 2 k^2 < 2^31 for k < 2^15
  auto chirp = [&](int k) -> C { return tab[(int)((2u * (unsigned)k * (unsigned)k) % (unsigned)twon)]; };

  if (MODE != 1) {
    // The folds of bins k and nh - k together: sums over m = b + q n, q = j mod g
    // (b = k, n - k, nh - k, nh + k), four loads in flight a step; with
    // e^{i pi s m / n} = e^{i pi s b / n} (-1)^{s q} the phase waits for the sum.
    // A = H'_k and B = conj H'_{nh-k} (twice the Hermitian halves).
    auto fold4 = [&](auto load, int k, int j, int g, C& A, C& B) {
      const int b1 = k == 0 ? 0 : n - k, b2 = nh - k, b3 = nh + k;
      C h0 = mk((T)0, (T)0), h1 = h0, h2 = h0, h3 = h0;
      T sg = f.shift && (j & 1) ? (T)-1 : (T)1;
      const T fl = f.shift && g == 1 ? (T)-1 : (T)1;
      for (int q = j * n; q + k <= L; q += g * n) {
        const C v0 = load(q + k);  // half of m = 0, which the two sums of bin 0 share
        const C v1 = q + b1 <= L ? load(q + b1) : mk((T)0, (T)0);
        const C v2 = q + b2 <= L ? load(q + b2) : mk((T)0, (T)0);
        const C v3 = q + b3 <= L ? load(q + b3) : mk((T)0, (T)0);
        const T s0 = q + k == 0 ? (T)0.5 * sg : sg;
        h0 = mk(fma(s0, v0.x, h0.x), fma(s0, v0.y, h0.y));
        const T s1 = q + b1 == 0 ? (T)0.5 * sg : sg;
        h1 = mk(fma(s1, v1.x, h1.x), fma(s1, v1.y, h1.y));
        h2 = mk(fma(sg, v2.x, h2.x), fma(sg, v2.y, h2.y));
        h3 = mk(fma(sg, v3.x, h3.x), fma(sg, v3.y, h3.y));
        sg *= fl;
      }
      if (f.shift) {
        h0 = cmul(h0, tab[k]);
        h1 = cmul(h1, tab[b1]);
        h2 = cmul(h2, tab[b2]);
        h3 = cmul(h3, tab[b3]);
      }
      A = cadd(h0, cconj(h1));
      B = cadd(cconj(h2), h3);
    };
    // with S = H'_k + conj H'_{nh-k} and T = i w^k (H'_k - conj H'_{nh-k}),
    // Z_k = S + T and Z_{nh-k} = conj(S - T)
    auto put = [&](int k, C Z) {
      if (!f.bluestein) buf[swz(bitrev(k, lg))] = Z;
      else buf[swz(k)] = cmul(Z, chirp(k));
    };
    auto put2 = [&](int k, C A, C B) {
      const C S = cadd(A, B), D = cmuli(cmul(tab[2 * k], csub(A, B)));
      put(k, cadd(S, D));
      if (k > 0 && 2 * k < nh) put(nh - k, cconj(csub(S, D)));
    };
    // rings with fewer bins than threads split each fold over g lanes (a power
    // of two <= 32) and sum the parts in a fixed shuffle order
    auto folds = [&](auto load) {
      const int nk = nh / 2 + 1;
      int g = 1;
      while (g < 32 && nk * g * 2 <= NT) g <<= 1;
      if (g == 1) {
        for (int k = tid; k < nk; k += NT) {
          C A, B;
          fold4(load, k, 0, 1, A, B);
          put2(k, A, B);
        }
        return;
      }
      const int k = tid / g, j = tid & (g - 1);
      C A = mk((T)0, (T)0), B = A;
      if (k < nk) fold4(load, k, j, g, A, B);
      for (int o = g >> 1; o > 0; o >>= 1) {
        A.x += __shfl_xor_sync(0xffffffffu, A.x, o);
        A.y += __shfl_xor_sync(0xffffffffu, A.y, o);
        B.x += __shfl_xor_sync(0xffffffffu, B.x, o);
        B.y += __shfl_xor_sync(0xffffffffu, B.y, o);
      }
      if (k < nk && j == 0) put2(k, A, B);
    };
    if (!staged) {
      folds([&](int m) -> C { return row[m]; });
    } else {
#pragma unroll 4
      for (int m = tid; m <= L; m += NT) srow[swz(m)] = row[m];
      __syncthreads();
      folds([&](int m) -> C { return srow[swz(m)]; });
    }
    if (f.bluestein)
      for (int k = nh + tid; k < M; k += NT) buf[swz(k)] = mk((T)0, (T)0);
    __syncthreads();
    if (!f.bluestein) {
      fft_run<false, BIG>(buf, M, lg, a.tw, a.Mmax);
    } else {
      fft_run<true, BIG>(buf, M, lg, a.tw, a.Mmax, vh);  // times the kernel spectrum
      fft_run<false, BIG>(buf, M, lg, a.tw, a.Mmax);
    }
    // z_t = (map_{2t}, map_{2t+1}) = buf[t] (times the chirp for Bluestein rings)
    auto z_of = [&](int t) -> C { return f.bluestein ? cmul(buf[swz(t)], chirp(t)) : buf[swz(t)]; };
    if (MODE == 0) {
      C* out = reinterpret_cast<C*>(a.map_out + blockIdx.y * a.ld_map + f.off);
      for (int t = tid; t < nh; t += NT) out[t] = z_of(t);
      return;
    }
    // MODE 2: multiply by the pixel diagonal and continue with the adjoint.
    const C* dg = reinterpret_cast<const C*>(a.pixdiag + f.off);
    C* mo = a.map_out ? reinterpret_cast<C*>(a.map_out + blockIdx.y * a.ld_map + f.off) : nullptr;
    for (int t = tid; t < nh; t += NT) {
      C z = z_of(t);
      if (mo) mo[t] = z;
      const C d = dg[t];
      z.x *= d.x;
      z.y *= d.y;
      buf[swz(t)] = f.bluestein ? cmul(cconj(z), chirp(t)) : z;
    }
    if (f.bluestein)
      for (int k = nh + tid; k < M; k += NT) buf[swz(k)] = mk((T)0, (T)0);
    __syncthreads();
  } else {
    const C* in = reinterpret_cast<const C*>(a.map_in + blockIdx.y * a.ld_map + f.off);
    for (int t = tid; t < nh; t += NT) {
      const C z = in[t];
      buf[swz(t)] = f.bluestein ? cmul(cconj(z), chirp(t)) : z;
    }
    if (f.bluestein)
      for (int k = nh + tid; k < M; k += NT) buf[swz(k)] = mk((T)0, (T)0);
    __syncthreads();
  }

  // forward length-nh DFT of z_t = y_{2t} + i y_{2t+1}
  if (!f.bluestein) {
    fft_run<true, BIG>(buf, M, lg, a.tw, a.Mmax);  // Z'_k at buf[bitrev(k)]
  } else {
    fft_run<true, BIG>(buf, M, lg, a.tw, a.Mmax, vh);  // times the kernel spectrum
    fft_run<false, BIG>(buf, M, lg, a.tw, a.Mmax);     // Z'_k = conj(buf[k] chirp(k))
  }
  auto getZ = [&](int k) -> C {
    return f.bluestein ? cconj(cmul(buf[swz(k)], chirp(k))) : buf[swz(bitrev(k, lg))];
  };
  // bins b and nh - b together: with E = (Z_b + conj Z_{nh-b}) / 2 and
  // T = i w^-b (Z_b - conj Z_{nh-b}) / 2, Yhat_b = E - T and Yhat_{nh-b} =
  // conj(E + T); row m is bin m mod n, or the conjugate of bin n - m mod n,
  // times e^{-i pi s m / n}
  auto bins = [&](auto out) {
    for (int b = tid; 2 * b <= nh; b += NT) {
      const C Zb = getZ(b);
      const C Zc = cconj(getZ(b == 0 ? 0 : nh - b));
      const C E = cscale(cadd(Zb, Zc), (T)0.5);
      const C D = cmuli(cmul(cconj(tab[2 * b]), cscale(csub(Zb, Zc), (T)0.5)));
      const C Y0 = csub(E, D), Y1 = cconj(cadd(E, D));
      out(b, Y0);
      if (b > 0) out(n - b, cconj(Y0));
      if (2 * b < nh) {
        out(nh - b, Y1);
        if (b > 0) out(nh + b, cconj(Y1));
      }
    }
  };
  auto turn = [&](int m, C Y) -> C { return f.shift ? cmul(Y, cconj(tab[m])) : Y; };
  if (!staged) {
    // every row of a bin from its thread: e^{-i pi s m / n} turns by (-1)^s a period
    bins([&](int b, C Y) {
      if (b > L) return;
      C v = turn(b, Y);
      for (int m = b; m <= L; m += n) {
        row[m] = v;
        if (f.shift) v = mk(-v.x, -v.y);
      }
    });
    return;
  }
  bins([&](int b, C Y) { srow[swz(b)] = turn(b, Y); });
  __syncthreads();
  int b = tid % n;
  bool odd = f.shift && ((tid / n) & 1);
  const int db = NT % n;
  const bool dodd = f.shift && ((NT / n) & 1);
  for (int m = tid; m <= L; m += NT) {
    const C v = srow[swz(b)];
    row[m] = odd ? mk(-v.x, -v.y) : v;
    b += db;
    odd ^= dodd;
    if (b >= n) {
      b -= n;
      odd ^= f.shift != 0;
    }
  }
}

template <typename T, bool BIG>
static int ring_fft_launch(const RingArgs<T>& b, int mode, int cnt, int nt, size_t smem, cudaStream_t st) {
  switch (mode) {
    case 0:
      CR_CUDA(cudaFuncSetAttribute(ring_fft_kernel<T, 0, BIG>, cudaFuncAttributeMaxDynamicSharedMemorySize, RF_SMEM));
      { ring_fft_kernel<T, 0, BIG><<<dim3(cnt, b.nrhs), nt, smem, st>>>(b); count_launch(); }
      break;
    case 1:
      CR_CUDA(cudaFuncSetAttribute(ring_fft_kernel<T, 1, BIG>, cudaFuncAttributeMaxDynamicSharedMemorySize, RF_SMEM));
      { ring_fft_kernel<T, 1, BIG><<<dim3(cnt, b.nrhs), nt, smem, st>>>(b); count_launch(); }
      break;
    default:
      CR_CUDA(cudaFuncSetAttribute(ring_fft_kernel<T, 2, BIG>, cudaFuncAttributeMaxDynamicSharedMemorySize, RF_SMEM));
      { ring_fft_kernel<T, 2, BIG><<<dim3(cnt, b.nrhs), nt, smem, st>>>(b); count_launch(); }
      break;
  }
  return CR_OK;
}

// One launch per FFT-size class (rings ordered by their FFT size M), each
// with the shared memory and block size its rings need.
template <typename T>
int launch_ring_fft(const RingArgs<T>& a, int mode, cudaStream_t st) {
  using C = typename Tr<T>::C;
  for (int c = 0; c < a.nclass; ++c) {
    const int M = a.cls_M[c];
    const int cnt = a.cls_start[c + 1] - a.cls_start[c];
    if (cnt <= 0) continue;
    size_t smem = (size_t)M * sizeof(C);
    if (smem > RF_SMEM || M > 65536) return fail(CR_EINVAL, "ring FFT buffer exceeds shared memory");
    // at least 128 threads: small rings split their folds over the idle lanes
    const int nt = std::max(128, std::min(RF_NT, M / 8));
    RingArgs<T> b = a;
    // The smallest rings fold each row many times over: the row is staged where
    // it is long.  A with | without staging: FP32 Nside 1024, lmax 2047 247 | 264
    // us, Nside 2048, lmax 3000 856 | 891; FP64 10.44 | 10.59 ms; but FP32 Nside
    // 512, lmax 1023 78.9 | 77.6 us, and staging the larger classes as well loses
    // what the first gains (Nside 2048: 922 us; fewer CTAs per SM).
    const size_t rows = ((size_t)a.L + 16) / 16 * 16 * sizeof(C);
    b.stage = c == 0 && 2 * a.L > 3 * M && smem + rows <= RF_SMEM ? M : 0;
    if (b.stage) smem += rows;
    b.rbase = a.cls_start[c];
    // FP32 rings with M >= 4096: the 4-stage passes with computed twiddles
    int rc;
    if constexpr (sizeof(T) == 4)
      rc = M >= 4096 ? ring_fft_launch<T, true>(b, mode, cnt, nt, smem, st)
                     : ring_fft_launch<T, false>(b, mode, cnt, nt, smem, st);
    else
      rc = ring_fft_launch<T, false>(b, mode, cnt, nt, smem, st);
    if (rc) return rc;
    CR_CHECK_LAUNCH("ring_fft_kernel");
  }
  return CR_OK;
}
template int launch_ring_fft<double>(const RingArgs<double>&, int, cudaStream_t);
template int launch_ring_fft<float>(const RingArgs<float>&, int, cudaStream_t);

// ---------------------------------------------------------------------------
// plan-time tables

struct LenDesc {
  int n, nh, M, logM, bluestein;
  int64_t tab, vhat;
};

__global__ void tab_kernel(const LenDesc* lens, double2* tab) {
  const LenDesc d = lens[blockIdx.x];
  for (int u = threadIdx.x; u < 2 * d.n; u += blockDim.x) {
    double s, c;
    sincospi((double)u / (double)d.n, &s, &c);
    tab[d.tab + u] = make_double2(c, s);
  }
}

__global__ void tw_kernel(double2* tw, int Mmax) {
  for (int j = blockIdx.x * blockDim.x + threadIdx.x; j < Mmax / 2; j += gridDim.x * blockDim.x) {
    double s, c;
    sincospi(-2.0 * (double)j / (double)Mmax, &s, &c);
    tw[j] = make_double2(c, s);
  }
}

// Bluestein kernel spectrum: v_d = e^{-i pi d^2 / nh}, |d| < nh, wrapped into
// length M, forward FFT, divided by M, kept in bit-reversed order.
__global__ void vhat_kernel(const LenDesc* lens, const double2* tab, const double2* tw, int Mmax, double2* vhat) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  double2* buf = reinterpret_cast<double2*>(smem_raw);
  const LenDesc d = lens[blockIdx.x];
  if (!d.bluestein) return;
  const int64_t twon = 2 * (int64_t)d.n;
  for (int k = threadIdx.x; k < d.M; k += blockDim.x) {
    int dd = -1;
    if (k < d.nh) dd = k;
    else if (k > d.M - d.nh) dd = d.M - k;
    buf[swz(k)] = (dd >= 0) ? cconj(tab[d.tab + (int)((2 * (int64_t)dd * dd) % twon)]) : make_double2(0.0, 0.0);
  }
  __syncthreads();
  fft_run<true, false>(buf, d.M, d.logM, tw, Mmax);
  for (int k = threadIdx.x; k < d.M; k += blockDim.x) vhat[d.vhat + k] = cscale(buf[swz(k)], 1.0 / d.M);
}

__global__ void to_f32_kernel(const double2* in, float2* out, int64_t n) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
    out[i] = make_float2((float)in[i].x, (float)in[i].y);
}
__global__ void to_f32r_kernel(const double* in, float* out, int64_t n) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
    out[i] = (float)in[i];
}

static int ilog2i(int M) {
  int l = 0;
  while ((1 << l) < M) ++l;
  return l;
}

int build_fft_tables(Grid& g, cudaStream_t st) {
  // distinct ring lengths
  std::map<int, int> idx;
  std::vector<LenDesc> lens;
  int64_t tab_len = 0, vhat_len = 0;
  int Mmax = 2;
  for (auto& f : g.fft) {
    if (idx.count(f.n)) continue;
    LenDesc d{};
    d.n = f.n;
    d.nh = f.n / 2;
    const bool p2 = (d.nh & (d.nh - 1)) == 0;
    d.bluestein = p2 ? 0 : 1;
    d.M = p2 ? d.nh : 1;
    if (!p2)
      while (d.M < 2 * d.nh - 1) d.M <<= 1;
    d.logM = ilog2i(d.M);
    d.tab = tab_len;
    tab_len += 2 * (int64_t)d.n;
    d.vhat = vhat_len;
    if (d.bluestein) vhat_len += d.M;
    Mmax = std::max(Mmax, d.M);
    idx[f.n] = (int)lens.size();
    lens.push_back(d);
  }
  for (auto& f : g.fft) {
    const LenDesc& d = lens[idx[f.n]];
    f.nh = d.nh;
    f.M = d.M;
    f.logM = d.logM;
    f.bluestein = d.bluestein;
    f.tab = d.tab;
    f.vhat = d.vhat;
  }
  if ((size_t)Mmax * sizeof(double2) > RF_SMEM) return fail(CR_EINVAL, "ring too long for the shared-memory FFT");
  g.Mmax = Mmax;
  g.tab_len = tab_len;
  g.vhat_len = vhat_len;
  LenDesc* d_lens = nullptr;
  CR_CUDA(cudaMalloc(&d_lens, lens.size() * sizeof(LenDesc)));
  CR_CUDA(cudaMemcpyAsync(d_lens, lens.data(), lens.size() * sizeof(LenDesc), cudaMemcpyHostToDevice, st));
  CR_CUDA(cudaMalloc(&g.d_tab, tab_len * sizeof(double2)));
  CR_CUDA(cudaMalloc(&g.d_tab32, tab_len * sizeof(float2)));
  CR_CUDA(cudaMalloc(&g.d_vhat, std::max<int64_t>(vhat_len, 1) * sizeof(double2)));
  CR_CUDA(cudaMalloc(&g.d_vhat32, std::max<int64_t>(vhat_len, 1) * sizeof(float2)));
  CR_CUDA(cudaMalloc(&g.d_tw, std::max(Mmax / 2, 1) * sizeof(double2)));
  CR_CUDA(cudaMalloc(&g.d_tw32, std::max(Mmax / 2, 1) * sizeof(float2)));
  tab_kernel<<<(int)lens.size(), 256, 0, st>>>(d_lens, g.d_tab);
  CR_CHECK_LAUNCH("tab_kernel");
  tw_kernel<<<std::max(1, std::min(1024, Mmax / 512)), 256, 0, st>>>(g.d_tw, Mmax);
  CR_CHECK_LAUNCH("tw_kernel");
  if (vhat_len > 0) {
    const size_t smem = (size_t)Mmax * sizeof(double2);
    CR_CUDA(cudaFuncSetAttribute(vhat_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, RF_SMEM));
    vhat_kernel<<<(int)lens.size(), 256, smem, st>>>(d_lens, g.d_tab, g.d_tw, Mmax, g.d_vhat);
    CR_CHECK_LAUNCH("vhat_kernel");
  }
  to_f32_kernel<<<256, 256, 0, st>>>(g.d_tab, g.d_tab32, tab_len);
  if (vhat_len > 0) to_f32_kernel<<<256, 256, 0, st>>>(g.d_vhat, g.d_vhat32, vhat_len);
  to_f32_kernel<<<64, 256, 0, st>>>(g.d_tw, g.d_tw32, Mmax / 2);
  CR_CHECK_LAUNCH("to_f32_kernel");
  // rings ordered by FFT size; one launch class per distinct size
  {
    std::vector<int> order(g.fft.size());
    for (size_t i = 0; i < order.size(); ++i) order[i] = (int)i;
    std::stable_sort(order.begin(), order.end(), [&](int x, int y) { return g.fft[x].M < g.fft[y].M; });
    g.cls_M.clear();
    g.cls_start.clear();
    // sizes up to 1024 share one class (their shared memory is small anyway)
    auto key = [&](int r) { return std::max(g.fft[r].M, std::min(1024, Mmax)); };
    for (size_t i = 0; i < order.size(); ++i) {
      if (g.cls_M.empty() || key(order[i]) != g.cls_M.back()) {
        g.cls_M.push_back(key(order[i]));
        g.cls_start.push_back((int)i);
      }
    }
    g.cls_start.push_back((int)order.size());
    CR_CUDA(cudaMalloc(&g.d_rings, order.size() * sizeof(int)));
    CR_CUDA(cudaMemcpyAsync(g.d_rings, order.data(), order.size() * sizeof(int), cudaMemcpyHostToDevice, st));
  }
  CR_CUDA(cudaMalloc(&g.d_fft, g.fft.size() * sizeof(RingFFT)));
  CR_CUDA(cudaMemcpyAsync(g.d_fft, g.fft.data(), g.fft.size() * sizeof(RingFFT), cudaMemcpyHostToDevice, st));
  CR_CUDA(cudaStreamSynchronize(st));
  CR_CUDA(cudaFree(d_lens));
  return CR_OK;
}

// Seeds P~_mm(z) = -sqrt((2m+1)/(2m)) sin(theta) P~_{m-1,m-1}, P~_00 = 1/sqrt(4 pi)
// (Section 3.3 normalisation, Condon-Shortley phase), iterated per ring pair
// in FP64 with level tracking, stored [m][pair] for FP64 and FP32.
__global__ void seed_kernel(const double* sth, const double* fac, int Lseed, int npairs, double* seed, int* lev,
                            float* seed32, int* lev32) {
  const int p = blockIdx.x * blockDim.x + threadIdx.x;
  if (p >= npairs) return;
  const double st = sth[p];
  const double lo = exp2((double)(Tr<double>::THR - Tr<double>::S));
  const double up = exp2((double)Tr<double>::S);
  double v = 0.28209479177387814347;  // 1/sqrt(4 pi)
  int e = 0;
  for (int m = 0; m <= Lseed; ++m) {
    if (m > 0) {
      v = -v * fac[m] * st;
      if (fabs(v) < lo && v != 0.0) {
        v *= up;
        e -= 1;
      }
    }
    const int64_t o = (int64_t)m * npairs + p;
    seed[o] = v;
    lev[o] = e;
    // FP32 representation: true = v 2^(600 e); want v32 in [2^(THR-S), 2^THR)
    float v32 = 0.f;
    int e32 = 0;
    if (v != 0.0) {
      const int E = ilogb(v) + Tr<double>::S * e;
      if (E >= Tr<float>::THR - Tr<float>::S) {
        v32 = (float)ldexp(v, Tr<double>::S * e);
        e32 = 0;
      } else {
        const int k = (Tr<float>::THR - Tr<float>::S - E + Tr<float>::S - 1) / Tr<float>::S;
        v32 = (float)ldexp(v, Tr<double>::S * e + Tr<float>::S * k);
        e32 = -k;
      }
    } else {
      e32 = -1;
    }
    seed32[o] = v32;
    lev32[o] = e32;
  }
}

int build_seeds(Grid& g, int Lseed, cudaStream_t st) {
  std::vector<double> fac(Lseed + 1, 0.0);
  for (int m = 1; m <= Lseed; ++m) fac[m] = std::sqrt((2.0 * m + 1.0) / (2.0 * m));
  double* d_fac = nullptr;
  CR_CUDA(cudaMalloc(&d_fac, (Lseed + 1) * sizeof(double)));
  CR_CUDA(cudaMemcpyAsync(d_fac, fac.data(), (Lseed + 1) * sizeof(double), cudaMemcpyHostToDevice, st));
  const int64_t n = (int64_t)(Lseed + 1) * g.npairs;
  CR_CUDA(cudaMalloc(&g.d_seed, n * sizeof(double)));
  CR_CUDA(cudaMalloc(&g.d_lev, n * sizeof(int)));
  CR_CUDA(cudaMalloc(&g.d_seed32, n * sizeof(float)));
  CR_CUDA(cudaMalloc(&g.d_lev32, n * sizeof(int)));
  seed_kernel<<<(g.npairs + 127) / 128, 128, 0, st>>>(g.d_sth, d_fac, Lseed, g.npairs, g.d_seed, g.d_lev, g.d_seed32,
                                                       g.d_lev32);
  CR_CHECK_LAUNCH("seed_kernel");
  CR_CUDA(cudaStreamSynchronize(st));
  CR_CUDA(cudaFree(d_fac));
  g.Lseed = Lseed;
  return CR_OK;
}

}  // namespace cr
