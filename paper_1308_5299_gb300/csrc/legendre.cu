// Legendre stages of spherical-harmonic synthesis Y and adjoint synthesis Y^T
// (Section 2.1, Eq. sh-synthesis; normalised P~_lm of Section 3.3): the plan's
// start tables, the dispatch, and the FP64 kernels of small grids and of the
// smoother's diagonal.  FP32 stages are those of legendre_f32.cu, FP64 stages of
// at least 64 ring pairs and lmax >= 64 those of legendre_ds.cu.
//
// For one m and one north/south ring pair (z, -z):
//   synthesis  F_m(+-z) = sum_{l=m..L} a_lm P~_lm(+-z),
//   adjoint    a_lm    += P~_lm(z) G_m(z) + P~_lm(-z) G_m(-z),
// with P~_lm(-z) = (-1)^(l+m) P~_lm(z), so one recurrence serves both rings
// through even/odd (l-m) accumulators.
//
// P~_lm is generated on the fly in registers by the three-term recurrence in
// the rescaled form Q_l = P~_lm / s_lm,
//   Q_l = c_lm z Q_{l-1} - Q_{l-2},
// where s_lm and c_lm are plan-time tables (s_mm = s_{m+1,m} = 1).  Starting
// from (Q_{m-1}, Q_{m-2}) = (0, -P~_mm) makes the first step return the seed,
// so the loop is uniform from l = m.  a_lm is multiplied by s_lm when staged
// (synthesis) and the adjoint result by s_lm when written.
//
// Each (m, ring pair) starts where |P~_lm| first reaches a threshold tau
// (2^-60 for the transforms of both precisions, with the FP64 state there
// for the FP64 kernels; 2^-100 for the squared sums of the smoother's
// diagonal): the plan-time start tables hold
// that l and the recurrence state there, computed once from the seed
// P~_mm in scaled FP64 (build_start_tables).  Terms with |P~_lm| < tau are
// dropped: below FP32 rounding by ten orders of magnitude and below FP64
// rounding by two, and decaying geometrically away from the start, so their
// sum stays under the rounding of either sum.  Before its start a pair neither steps nor
// accumulates; pairs that never reach tau within the band limit hold a zero
// state.  Each warp classifies every group of 8 l as idle (no pair started
// yet), full (every live pair started: the unchecked loop) or ramp (per-pair
// start test), so the region below the turning point where the functions are
// negligible costs nothing.
//
// Work decomposition: one CTA per (m, block of LEG_NT*RP ring pairs) with
// the ring-pair blocks of one m adjacent in launch order (blockIdx.x) and m
// in blockIdx.y, so the longest CTAs (small m) are dispatched first, the
// short ones (m near L) last, and the CTAs of one m share its coefficients
// in L2; RP
// (2, 4 or 8 pairs per thread: the ring-block size) chosen per grid, band
// limit and precision by the plan's autotuner (default 4);
// each warp owns 32*RP consecutive pairs (lane + 32 j), so its pairs'
// start points are close.  The a_lm of the CTA's m (synthesis) and the
// recurrence coefficients are staged through shared memory in chunks of
// LEG_CH l-values from the CTA's earliest start.  The adjoint reduces over
// ring pairs with a warp-shuffle transpose reduction over 8 consecutive l
// (each lane ends with one l) into per-warp rows of shared memory, one
// fixed-order cross-warp sum per chunk of LEG_CH l (a single barrier per
// chunk), and one partial row per ring block summed in a second,
// deterministic kernel.
#include "common.cuh"
#include "kernels.h"

namespace cr {

constexpr int LEG_NT = 128;
constexpr int LEG_RP = 4;      // default ring pairs per thread
constexpr int LEG_RP_MIN = 2;  // smallest choice of the autotuner
constexpr int LEG_CH = 256;
constexpr int LEG_NW = LEG_NT / 32;

// One recurrence step Q_l = c z Q_{l-1} - Q_{l-2}; returns Q_l and advances
// the state (s1, s2) = (Q_{l-1}, Q_{l-2}).
__device__ __forceinline__ double rstep(double c, double z, double& s1, double& s2) {
  const double q = fma(c * z, s1, -s2);
  s2 = s1;
  s1 = q;
  return q;
}

// Per-thread pair setup shared by both kernels: start point, state, and the
// warp's earliest / latest start over its live pairs (a pair is live when it
// starts at or below L).  Returns false when the warp has no live pair.
template <int RP>
__device__ __forceinline__ bool load_pairs(const LegArgs<double>& a, int m, int warp, int lane, int p[RP], int ls[RP],
                                           double P1[RP], double P2[RP], double zz[RP], int* wmin, int* wmax) {
  int lo = a.L + 1, hi = m;
#pragma unroll
  for (int j = 0; j < RP; ++j) {
    p[j] = (int)blockIdx.x * (LEG_NT * RP) + warp * (32 * RP) + j * 32 + lane;
    ls[j] = a.L + 1;
    P1[j] = 0;
    P2[j] = 0;
    zz[j] = 0;
    if (p[j] < a.npairs) {
      const int64_t o = (int64_t)m * a.ld_seed + p[j];
      const int l = a.ls[o];
      zz[j] = a.z[p[j]];
      if (l <= a.L) {
        const double2 st = a.st[o];
        ls[j] = l;
        P1[j] = st.x;
        P2[j] = st.y;
        lo = min(lo, l);
        hi = max(hi, l);
      }
    }
  }
  *wmin = __reduce_min_sync(0xffffffffu, lo);
  *wmax = __reduce_max_sync(0xffffffffu, hi);
  return *wmin <= a.L;
}

template <int RP, int MT = 1>
__global__ void __launch_bounds__(LEG_NT) leg_synth_kernel(LegArgs<double> a) {
  using T = double;
  using C = double2;
  // m tile: this CTA takes m = blockIdx.y and, with MT = 2, then
  // m = L - blockIdx.y, so that every CTA has about the same l range
#pragma unroll 1
  for (int mi = 0; mi < MT; ++mi) {
    const int m = mi == 0 ? (int)blockIdx.y : a.L - (int)blockIdx.y;
    if (mi > 0 && m <= (int)blockIdx.y) break;
    if (mi > 0) __syncthreads();  // the shared buffers of the previous m are free
    const int L = a.L;
    const int tid = threadIdx.x;
    const int warp = tid >> 5, lane = tid & 31;
    // each warp stages its own chunks (no block-wide barrier in the loop)
    __shared__ C sa_all[LEG_NW][LEG_CH];
    __shared__ T sc_all[LEG_NW][LEG_CH];
    C* sa = sa_all[warp];
    T* sc = sc_all[warp];

    T P1[RP], P2[RP], zz[RP];
    int ls[RP], p[RP];
    C accE[RP], accO[RP];
#pragma unroll
    for (int j = 0; j < RP; ++j) {
      accE[j] = mk((T)0, (T)0);
      accO[j] = mk((T)0, (T)0);
    }
    const int yb = (int)blockIdx.x;
    int wmin, wmax;
    const bool live = load_pairs<RP>(a, m, warp, lane, p, ls, P1, P2, zz, &wmin, &wmax);
    const int64_t offa = lm_off(L, m);
    const int64_t offc = lm_off(a.Lc, m);

    // chunks start at an offset from m that is a multiple of 8, so l - m and
    // the group index agree in parity; a warp starts at its earliest pair
    const int lbeg = live ? m + ((wmin - m) & ~7) : L + 1;
    for (int l0 = lbeg; l0 <= L; l0 += LEG_CH) {
      const int nl = min(LEG_CH, L - l0 + 1);
      __syncwarp();
      for (int i = lane; i < nl; i += 32) {
        const int l = l0 + i;
        C v = a.alm[offa + (l - m)];
        if (m == 0) v.y = 0;
        T f = a.s[offc + (l - m)];
        if (a.dl) f *= a.dl[l];
        sa[i] = cscale(v, f);
        sc[i] = a.c[offc + (l - m)];
      }
      __syncwarp();
      for (int i8 = 0; i8 < nl; i8 += 8) {
        const int lg = l0 + i8;
        const int ng = min(8, nl - i8);
        if (wmin >= lg + ng) continue;  // no pair of the warp has started
        if (wmax <= lg && ng == 8) {
#pragma unroll
          for (int u = 0; u < 8; u += 2) {
            const T c0 = sc[i8 + u], c1 = sc[i8 + u + 1];
            const C a0 = sa[i8 + u], a1 = sa[i8 + u + 1];
#pragma unroll
            for (int j = 0; j < RP; ++j) {
              const T q0 = rstep(c0, zz[j], P1[j], P2[j]);
              const T q1 = rstep(c1, zz[j], P1[j], P2[j]);
              accE[j].x = fma(q0, a0.x, accE[j].x);
              accE[j].y = fma(q0, a0.y, accE[j].y);
              accO[j].x = fma(q1, a1.x, accO[j].x);
              accO[j].y = fma(q1, a1.y, accO[j].y);
            }
          }
        } else {
          for (int u = 0; u < ng; ++u) {
            const int l = lg + u;
            const T c0 = sc[i8 + u];
            const C a0 = sa[i8 + u];
#pragma unroll
            for (int j = 0; j < RP; ++j) {
              if (l >= ls[j]) {
                const T q0 = rstep(c0, zz[j], P1[j], P2[j]);
                if (u & 1) {
                  accO[j].x = fma(q0, a0.x, accO[j].x);
                  accO[j].y = fma(q0, a0.y, accO[j].y);
                } else {
                  accE[j].x = fma(q0, a0.x, accE[j].x);
                  accE[j].y = fma(q0, a0.y, accE[j].y);
                }
              }
            }
          }
        }
      }
    }
    const int pend = a.npairs;
#pragma unroll
    for (int j = 0; j < RP; ++j) {
      if (p[j] < pend) {
        const int rn = p[j], rs = a.nring - 1 - p[j];
        a.phase[(int64_t)rn * a.ldp + m] = cadd(accE[j], accO[j]);
        if (rs != rn) a.phase[(int64_t)rs * a.ldp + m] = csub(accE[j], accO[j]);
      }
    }
  }
}

template <typename T>
__device__ __forceinline__ T shfl_x(T v, int mask) {
  return __shfl_xor_sync(0xffffffffu, v, mask);
}

// Transpose reduction of 8 complex values over the 32 lanes of a warp: on
// return lane l holds in v[0] the warp sum of the value with index l >> 2.
template <typename C>
__device__ __forceinline__ void warp_reduce8(C v[8]) {
  const int lane = threadIdx.x & 31;
  {
    const bool hi = lane & 16;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      C send = hi ? v[i] : v[i + 4];
      C keep = hi ? v[i + 4] : v[i];
      send.x = shfl_x(send.x, 16);
      send.y = shfl_x(send.y, 16);
      v[i] = cadd(keep, send);
    }
  }
  {
    const bool hi = lane & 8;
#pragma unroll
    for (int i = 0; i < 2; ++i) {
      C send = hi ? v[i] : v[i + 2];
      C keep = hi ? v[i + 2] : v[i];
      send.x = shfl_x(send.x, 8);
      send.y = shfl_x(send.y, 8);
      v[i] = cadd(keep, send);
    }
  }
  {
    const bool hi = lane & 4;
    C send = hi ? v[0] : v[1];
    C keep = hi ? v[1] : v[0];
    send.x = shfl_x(send.x, 4);
    send.y = shfl_x(send.y, 4);
    v[0] = cadd(keep, send);
  }
  v[0].x += shfl_x(v[0].x, 2);
  v[0].y += shfl_x(v[0].y, 2);
  v[0].x += shfl_x(v[0].x, 1);
  v[0].y += shfl_x(v[0].y, 1);
}

// SQ: accumulate P~^2 times a per-ring value (ringval) instead of P~ times
// the ring's phase G_m: sum_k P~_lm(z_k)^2 v_k, used for the diagonal of
// Y^T N^-1 Y (the Delta m = 0 term of the ring formula).
template <int RP, bool SQ = false, int MT = 1>
__global__ void __launch_bounds__(LEG_NT) leg_adjoint_kernel(LegArgs<double> a) {
  using T = double;
  using C = double2;
  // m tile: this CTA takes m = blockIdx.y and, with MT = 2, then
  // m = L - blockIdx.y, so that every CTA has about the same l range
#pragma unroll 1
  for (int mi = 0; mi < MT; ++mi) {
    const int m = mi == 0 ? (int)blockIdx.y : a.L - (int)blockIdx.y;
    if (mi > 0 && m <= (int)blockIdx.y) break;
    if (mi > 0) __syncthreads();  // the shared buffers of the previous m are free
    const int L = a.L;
    const int tid = threadIdx.x;
    const int warp = tid >> 5, lane = tid & 31;
    // per-warp copies of the recurrence coefficients (staged by each warp),
    // and per-warp sums of the chunk's l
    __shared__ T sc_all[LEG_NW][LEG_CH];
    __shared__ C red[LEG_NW][LEG_CH];
    __shared__ int s_min;
    T* sc = sc_all[warp];

    T P1[RP], P2[RP], zz[RP];
    int ls[RP], p[RP];
    C GE[RP], GO[RP];
    const int yb = (int)blockIdx.x;
    int wmin, wmax;
    const bool live = load_pairs<RP>(a, m, warp, lane, p, ls, P1, P2, zz, &wmin, &wmax);
    const int pend = a.npairs;
#pragma unroll
    for (int j = 0; j < RP; ++j) {
      GE[j] = mk((T)0, (T)0);
      GO[j] = mk((T)0, (T)0);
      if (p[j] < pend && ls[j] <= L) {
        const int rn = p[j], rs = a.nring - 1 - p[j];
        if (SQ) {
          const T v = a.ringval[rn] + ((rs != rn) ? a.ringval[rs] : (T)0);
          GE[j] = mk(v, (T)0);
          GO[j] = GE[j];
        } else {
          const C gn = a.phase[(int64_t)rn * a.ldp + m];
          const C gs = (rs != rn) ? a.phase[(int64_t)rs * a.ldp + m] : mk((T)0, (T)0);
          GE[j] = cadd(gn, gs);
          GO[j] = csub(gn, gs);
        }
      }
    }
    if (tid == 0) s_min = L + 1;
    __syncthreads();
    if (lane == 0 && live) atomicMin(&s_min, wmin);
    __syncthreads();
    const int cmin = s_min;
    const int64_t offa = lm_off(L, m);
    const int64_t offc = lm_off(a.Lc, m);
    C* part = a.partial + (int64_t)yb * n_lm(L);
    const int lbeg = (cmin <= L) ? m + ((cmin - m) & ~7) : L + 1;
    // rows before the block's earliest start are zero
    for (int l = m + tid; l < lbeg; l += LEG_NT) part[offa + (l - m)] = mk((T)0, (T)0);

    for (int l0 = lbeg; l0 <= L; l0 += LEG_CH) {
      const int nl = min(LEG_CH, L - l0 + 1);
      __syncthreads();  // the previous chunk's sums are read
      __syncwarp();
      for (int i = lane; i < nl; i += 32) {
        sc[i] = a.c[offc + (l0 - m) + i];
      }
      __syncwarp();
      for (int i8 = 0; i8 < nl; i8 += 8) {
        const int lg = l0 + i8;
        const int ng = min(8, nl - i8);
        if (!live || wmin >= lg + ng) {
          // no pair of this warp has started: its share of the sums is zero
          if (lane < 8) red[warp][i8 + lane] = mk((T)0, (T)0);
        } else {
          C acc[8];
#pragma unroll
          for (int u = 0; u < 8; ++u) acc[u] = mk((T)0, (T)0);
          if (wmax <= lg && ng == 8) {
#pragma unroll
            for (int u = 0; u < 8; u += 2) {
              const T c0 = sc[i8 + u], c1 = sc[i8 + u + 1];
#pragma unroll
              for (int j = 0; j < RP; ++j) {
                T q0 = rstep(c0, zz[j], P1[j], P2[j]);
                T q1 = rstep(c1, zz[j], P1[j], P2[j]);
                if (SQ) {
                  q0 *= q0;
                  q1 *= q1;
                }
                acc[u].x = fma(q0, GE[j].x, acc[u].x);
                acc[u].y = fma(q0, GE[j].y, acc[u].y);
                acc[u + 1].x = fma(q1, GO[j].x, acc[u + 1].x);
                acc[u + 1].y = fma(q1, GO[j].y, acc[u + 1].y);
              }
            }
          } else {
#pragma unroll
            for (int u = 0; u < 8; ++u) {
              if (u < ng) {
                const int l = lg + u;
                const T c0 = sc[i8 + u];
#pragma unroll
                for (int j = 0; j < RP; ++j) {
                  if (l >= ls[j]) {
                    T q0 = rstep(c0, zz[j], P1[j], P2[j]);
                    if (SQ) q0 *= q0;
                    const C g = (u & 1) ? GO[j] : GE[j];
                    acc[u].x = fma(q0, g.x, acc[u].x);
                    acc[u].y = fma(q0, g.y, acc[u].y);
                  }
                }
              }
            }
          }
          warp_reduce8(acc);
          if ((lane & 3) == 0) red[warp][i8 + (lane >> 2)] = acc[0];
        }
      }
      // one barrier per chunk: the warps' sums in a fixed order
      __syncthreads();
      for (int i = tid; i < nl; i += LEG_NT) {
        const int l = l0 + i;
        C sum = red[0][i];
#pragma unroll
        for (int w = 1; w < LEG_NW; ++w) sum = cadd(sum, red[w][i]);
        const T sc_ = a.s[offc + (l - m)];
        part[offa + (l - m)] = cscale(sum, SQ ? sc_ * sc_ : sc_);
      }
    }
  }
}

// y_lm = dl_out[l] * sum_blk partial[blk][lm] + dadd[l] * xadd_lm; zero at
// inactive l (dl_out = dadd = 0 there) and Im(a_l0) = 0.
template <typename T>
__global__ void __launch_bounds__(256) leg_finalize_kernel(FinalizeArgs<T> a) {
  using C = typename Tr<T>::C;
  const int64_t nlm = n_lm(a.L);
  const C* part = a.partial + (int64_t)blockIdx.y * a.nblk * nlm;  // blockIdx.y: right-hand side
  const int64_t v0 = blockIdx.y * a.ld;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < nlm; i += (int64_t)gridDim.x * blockDim.x) {
    C s = part[i];
#pragma unroll 4
    for (int b = 1; b < a.nblk; ++b) s = cadd(s, part[(int64_t)b * nlm + i]);
    // recover l, m from the flat index (m-major layout)
    int m = (int)((2.0 * (a.L + 1) + 1.0 - sqrt((2.0 * (a.L + 1) + 1.0) * (2.0 * (a.L + 1) + 1.0) - 8.0 * (double)i)) * 0.5);
    while (m > 0 && lm_off(a.L, m) > i) --m;
    while (m < a.L && lm_off(a.L, m + 1) <= i) ++m;
    const int l = m + (int)(i - lm_off(a.L, m));
    T f = a.dl_out ? a.dl_out[l] : (T)1;
    C y = cscale(s, f);
    if (a.dadd) {
      C x = a.xadd[v0 + i];
      y.x = fma(a.dadd[l], x.x, y.x);
      y.y = fma(a.dadd[l], x.y, y.y);
    }
    if (a.bsub) {
      const C bb = a.bsub[v0 + i];
      y = mk(bb.x - y.x, (m == 0) ? (T)0 : bb.y - y.y);
    }
    if (m == 0) y.y = 0;
    if (a.accumulate) y = cadd(y, a.out[v0 + i]);
    a.out[v0 + i] = y;
  }
}

static inline void pair_blocks(int npairs, int rp, int* nb) { *nb = (npairs + LEG_NT * rp - 1) / (LEG_NT * rp); }

// ring pairs per thread of a launch: 2, 4 or 8 (other values: the default)
static inline int legal_rp(int rp) { return (rp == 2 || rp == 4 || rp == 8) ? rp : LEG_RP; }

// rows of m of a launch: L + 1, or (L + 2) / 2 when each CTA pairs m with L - m
static inline int m_rows(int L, int mt) { return mt == 2 ? (L + 2) / 2 : L + 1; }

template <int RP>
static void synth_launch(const LegArgs<double>& a, int nb, cudaStream_t st) {
  const dim3 grid(nb, m_rows(a.L, a.mt_synth));
  if (a.mt_synth == 2) leg_synth_kernel<RP, 2><<<grid, LEG_NT, 0, st>>>(a);
  else leg_synth_kernel<RP, 1><<<grid, LEG_NT, 0, st>>>(a);
  count_launch();
}
template <int RP>
static void adjoint_launch(const LegArgs<double>& a, int nb, cudaStream_t st) {
  const dim3 grid(nb, m_rows(a.L, a.mt_adj));
  if (a.mt_adj == 2) leg_adjoint_kernel<RP, false, 2><<<grid, LEG_NT, 0, st>>>(a);
  else leg_adjoint_kernel<RP, false, 1><<<grid, LEG_NT, 0, st>>>(a);
  count_launch();
}

template <>
int launch_leg_synth<float>(const LegArgs<float>& a, cudaStream_t st) {
  return a.L < 0 ? CR_OK : launch_lf_synth(a, st);
}
template <>
int launch_leg_adjoint<float>(const LegArgs<float>& a, const FinalizeArgs<float>& f, cudaStream_t st) {
  return a.L < 0 ? CR_OK : launch_lf_adjoint(a, f, st);
}

template <>
int launch_leg_synth<double>(const LegArgs<double>& a, cudaStream_t st) {
  if (a.L < 0) return CR_OK;
  if (a.df) return launch_leg_synth_df(a, st);
  if (ds_use(a)) return launch_ds_synth(a, a.alm, n_lm(a.L), 1, a.phase, st);
  const int rp = legal_rp(a.rp_synth);
  int nb;
  pair_blocks(a.npairs, rp, &nb);
  if (rp == 2) synth_launch<2>(a, nb, st);
  else if (rp == 8) synth_launch<8>(a, nb, st);
  else synth_launch<4>(a, nb, st);
  CR_CHECK_LAUNCH("leg_synth_kernel");
  return CR_OK;
}

template <>
int launch_leg_adjoint<double>(const LegArgs<double>& a, const FinalizeArgs<double>& f, cudaStream_t st) {
  if (a.L < 0) return CR_OK;
  int nb = 0;
  if (a.df) {
    int rc = launch_leg_adjoint_df(a, &nb, st);
    if (rc) return rc;
  } else if (ds_use(a)) {
    return launch_ds_adjoint(a, a.phase, 1, reinterpret_cast<double*>(a.partial), f, st);
  } else {
    const int rp = legal_rp(a.rp_adj);
    pair_blocks(a.npairs, rp, &nb);
    if (rp == 2) adjoint_launch<2>(a, nb, st);
    else if (rp == 8) adjoint_launch<8>(a, nb, st);
    else adjoint_launch<4>(a, nb, st);
    CR_CHECK_LAUNCH("leg_adjoint_kernel");
  }
  FinalizeArgs<double> ff = f;
  ff.partial = a.partial;
  ff.nblk = nb;
  ff.L = a.L;
  return launch_leg_finalize<double>(ff, st);
}

template <typename T>
int launch_leg_finalize(const FinalizeArgs<T>& f, cudaStream_t st) {
  const int64_t nlm = n_lm(f.L);
  int blocks = (int)std::min<int64_t>((nlm + 255) / 256, 152 * 16);
  { leg_finalize_kernel<T><<<dim3(blocks, f.nrhs), 256, 0, st>>>(f); count_launch(); }
  CR_CHECK_LAUNCH("leg_finalize_kernel");
  return CR_OK;
}

// out_lm = sum_k P~_lm(z_k)^2 ringval_k on the observation grid (FP64)
int launch_leg_diag(cr_plan* P, const double* ringval, double2* out) {
  const Grid& g = P->obs;
  LegArgs<double> a;
  a.ldp = P->lmax + 1;
  a.L = P->lmax;
  a.Lc = P->Lcoef;
  a.c = P->d_c;
  a.s = P->d_s;
  a.z = g.d_z;
  a.ls = g.d_ls64;
  a.st = g.d_st64;
  a.ld_seed = g.npairs;
  a.npairs = g.npairs;
  a.nring = g.nring;
  a.ringval = ringval;
  a.partial = reinterpret_cast<double2*>(P->ws.partial);
  int nbe;
  pair_blocks(a.npairs, LEG_RP, &nbe);
  { leg_adjoint_kernel<LEG_RP, true><<<dim3(nbe, a.L + 1), LEG_NT, 0, P->stream>>>(a); count_launch(); }
  CR_CHECK_LAUNCH("leg_adjoint_kernel<SQ>");
  FinalizeArgs<double> ff;
  ff.partial = a.partial;
  ff.nblk = nbe;
  ff.L = a.L;
  ff.out = out;
  const int64_t nlm = n_lm(a.L);
  { leg_finalize_kernel<double><<<(int)std::min<int64_t>((nlm + 255) / 256, 152 * 16), 256, 0, P->stream>>>(ff); count_launch(); }
  CR_CHECK_LAUNCH("leg_finalize_kernel");
  return CR_OK;
}

// The start state (value before k0, second value) of one pair of the FP32
// sequences (legendre_f32.cu), from the FP64 state (Q_{l-1}, Q_{l-2}) and Q_l at
// its start l: such that the zone's step returns q_{k0}, k0 = (l - m) / 2 (the
// one-step zone: (z Q, Q) before Q_{m + 2 k0}, one step back where l is the second
// of its two).
__device__ float2 lf_start(const DsTab& t, const double* c, const double* s, int Lc, int m, int l, double z, int zone,
                           double Q, double Q1, double Q2) {
  const int k0 = (l - m) >> 1;
  const int64_t oc = lm_off(Lc, m) + (l - m), ok = ((lm_off(t.Lc, m) >> 1) + m) + k0;
  const bool odd = (l - m) & 1;
  if (zone == 2)
    return odd ? make_float2((float)(z * Q2), (float)(c[oc - 1] * z * Q2 - Q1)) : make_float2((float)(z * Q1), (float)Q2);
  const double P = s[oc] * Q;
  double q1 = 0.0;
  if (k0 > 0) q1 = (odd ? s[oc - 2] * Q2 : s[oc - 1] * Q1) / (z * t.sg[ok - 1]);
  const double qk = (odd ? P : P - (k0 > 0 ? t.e1[ok - 1] * q1 : 0.0)) / (odd ? z * t.sg[ok] : t.e0[ok]);
  if (zone == 0) {
    const double w = 1.0 - z;
    const double e = k0 > 0 ? (t.AB[ok] - 2.0) - t.A[ok] * (w * (2.0 - w)) : 0.0;
    return make_float2((float)q1, (float)(qk - q1 - e * q1));
  }
  const double e = k0 > 0 ? fma(t.A[ok], z * z, t.B[ok]) : 0.0;
  return make_float2((float)q1, (float)(e * q1 - qk));
}

// Start tables (see Grid): for each m <= Lseed and ring pair, the scaled FP64
// recurrence from the seed P~_mm up to the first l with |P~_lm| >= tau.
__global__ void start_kernel(const double* z, const double* seed, const int* lev, int ld, const double* c,
                             const double* s, int Lc, int Lseed, int npairs, int npolar32, int* ls64,
                             double2* st64, int* ls32, float2* st32, double2* st64b, DsTab t, int n1, int n2,
                             float2* sti) {
  const int m = blockIdx.y;
  const int p = blockIdx.x * blockDim.x + threadIdx.x;
  if (p >= npairs) return;
  const int64_t o = (int64_t)m * ld + p;
  const double zz = z[p];
  const int64_t offc = lm_off(Lc, m);
  const double thr = exp2((double)Tr<double>::THR);
  const double down = exp2(-(double)Tr<double>::S);
  const double tau64 = exp2(-100.0), tau32 = exp2(-60.0);
  double q1 = 0.0, q2 = -seed[o];
  int e = lev[o];
  int f64 = Lseed + 1, f32 = Lseed + 1;
  double2 s64 = make_double2(0.0, 0.0), s64b = make_double2(0.0, 0.0);
  float2 s32 = make_float2(0.f, 0.f), si = s32;
  for (int l = m; l <= Lseed; ++l) {
    const double q = c[offc + (l - m)] * zz * q1 - q2;
    if (e == 0) {
      const double pv = fabs(s[offc + (l - m)] * q);
      if (f64 > Lseed && pv >= tau64) {
        f64 = l;
        s64 = make_double2(q1, q2);
      }
      if (pv >= tau32) {  // tau32 > tau64: the FP32 start comes last
        f32 = l;
        s32 = (p < npolar32) ? make_float2((float)q1, (float)(q1 - q2)) : make_float2((float)q1, (float)q2);
        s64b = make_double2(q1, q2);
        si = lf_start(t, c, s, Lc, m, l, zz, p < n1 ? 0 : p < n2 ? 1 : 2, q, q1, q2);
        break;
      }
    }
    q2 = q1;
    q1 = q;
    if (e < 0 && fabs(q1) > thr) {
      q1 *= down;
      q2 *= down;
      ++e;
    }
  }
  ls64[o] = f64;
  st64[o] = s64;
  ls32[o] = f32;
  st32[o] = s32;
  st64b[o] = s64b;
  sti[o] = si;
}

int build_start_tables(cr_plan* P, Grid& g) {
  const int Ls = g.Lseed;
  if (Ls < 0) return CR_OK;
  if (Ls > P->Lcoef) return fail(CR_EINVAL, "start tables: grid band limit above the recurrence tables");
  void* ptrs[] = {g.d_ls64, g.d_st64, g.d_ls32, g.d_st32, g.d_st64b, g.d_sti};
  for (void* q : ptrs)
    if (q) cudaFree(q);
  const int64_t n = (int64_t)(Ls + 1) * g.npairs;
  CR_CUDA(cudaMalloc(&g.d_ls64, n * sizeof(int)));
  CR_CUDA(cudaMalloc(&g.d_st64, n * sizeof(double2)));
  CR_CUDA(cudaMalloc(&g.d_ls32, n * sizeof(int)));
  CR_CUDA(cudaMalloc(&g.d_st32, n * sizeof(float2)));
  CR_CUDA(cudaMalloc(&g.d_st64b, n * sizeof(double2)));
  CR_CUDA(cudaMalloc(&g.d_sti, n * sizeof(float2)));
  dim3 grid((g.npairs + 127) / 128, Ls + 1);
  { start_kernel<<<grid, 128, 0, P->stream>>>(g.d_z, g.d_seed, g.d_lev, g.npairs, P->d_c, P->d_s, P->Lcoef, Ls,
                                               g.npairs, g.npolar32, g.d_ls64, g.d_st64, g.d_ls32, g.d_st32,
                                               g.d_st64b, *P->ds, g.n1, g.n2, g.d_sti);
    count_launch(); }
  CR_CHECK_LAUNCH("start_kernel");
  CR_CUDA(cudaStreamSynchronize(P->stream));
  return CR_OK;
}

// upper bound on the partial rows of the FP64 CUDA-core and double-float adjoints
int leg_partial_blocks(int npairs) {
  return std::max((npairs + LEG_NT * LEG_RP_MIN - 1) / (LEG_NT * LEG_RP_MIN), df_pair_blocks(npairs));
}

template int launch_leg_finalize<double>(const FinalizeArgs<double>&, cudaStream_t);
template int launch_leg_finalize<float>(const FinalizeArgs<float>&, cudaStream_t);

}  // namespace cr
