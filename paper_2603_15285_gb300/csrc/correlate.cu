// Step a3: the per-degree contraction of Eq. (sigmalmm), with the radial
// quadrature in place of the ball-harmonic radial index:
//   c^l_{mn} = sum_s w_s f_lm(r_s) conj(h_ln(r_s)).
// Negative orders come from f_{l,-m} = (-1)^m conj(f_lm) (real volumes).
// Output layout: the grouped layout of the plan (pairs (m, n), m >= |n|, taken
// two at a time with equal m, components of the two partners interleaved);
// each (pair, l), l = m..L_J, holds (c^l_{mn}, c^l_{nm}).
#include <stdint.h>
#include <algorithm>
#include "internal.cuh"

namespace matcha {

template <typename T> struct Cplx2;
template <> struct Cplx2<float> { using type = float2; };
template <> struct Cplx2<double> { using type = double2; };

// One CTA per (particle, degree pair {l, L-l}): the coefficients of both
// degrees (all shells, orders 0..l) are staged in shared memory with the
// template side pre-multiplied by the radial weight, then one thread per
// 2 x 2 block of orders (a, b) of one degree produces their (c^l_mn, c^l_nm); the two
// degrees share one item loop, so pairing l with L - l balances the
// (l+1)^2 + (L-l+1)^2 items of a CTA.  The signs of the negative order -|n|
// are applied once after the shell sums.
//
// FP64 (bound by its pipe) and the FP32 plans that k_correlate_rec does not serve
// better (launch_correlate).
//
// With BALL (plans with the ball-harmonic radial basis) the staged rows are
// the projections on the retained radial functions instead of the shells:
// f_klm = sum_s W_lk(s) f_lm(r_s), W_lk(s) = w_s N_lk j_l(lambda_lk r_s / R),
// for k < |K_l| (both sides), and the products run over those |K_l| rows:
// c^l_mn = sum_{k in K_l} f_klm conj(h_kln), Eq. (sigmalmm) itself, i.e. A_l
// through its rank-|K_l| factors, so a degree costs |K_l| (2l+1)^2 products
// instead of S (2l+1)^2.
template <typename T, bool BALL>
__global__ void __launch_bounds__(256)
k_correlate_deg(const T *__restrict__ f, const T *__restrict__ h, int S, int L, long h_stride,
                const double *__restrict__ wrad, const int *__restrict__ pair_base, long nc,
                T *__restrict__ c, const T *__restrict__ ballW, const int *__restrict__ ballK,
                int Kmax) {
  using C2 = typename Cplx2<T>::type;
  const long b = blockIdx.y;
  const int nlm = (L + 1) * (L + 2) / 2;
  const T *fb = f + 2 * b * (long)S * nlm;
  const T *hb = h + 2 * (b * h_stride) * (long)S * nlm;
  T *cb = c + 4 * b * nc;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  C2 *sF = reinterpret_cast<C2 *>(smem_raw);
  const int l_lo = blockIdx.x, l_hi = L - blockIdx.x;
  const int npass = l_hi == l_lo ? 1 : 2;
  // stage: degree d's orders 0..l at [S][l+1] (F) and [S][l+1] (w H)
  const int no0 = l_lo + 1, no1 = l_hi + 1;
  const int R0 = BALL ? Kmax : S;  // rows reserved per degree
  C2 *F0 = sF, *H0 = sF + R0 * no0, *F1 = sF + 2 * R0 * no0, *H1 = F1 + R0 * no1;
  // rows summed per degree: the shells, or the retained radial functions
  const int S0 = BALL ? ballK[l_lo] : S, S1 = BALL ? ballK[l_hi] : S;
  for (int d = 0; d < npass; ++d) {
    const int l = d ? l_hi : l_lo, no = l + 1, base = l * (l + 1) / 2;
    C2 *Fd = d ? F1 : F0, *Hd = d ? H1 : H0;
    if (BALL) {
      const int Kl = d ? S1 : S0;
      const T *Wl = ballW + (long)l * Kmax * S;
      for (int t = threadIdx.x; t < Kl * no; t += blockDim.x) {
        const int k = t / no, m = t - k * no;
        C2 fv{T(0), T(0)}, hv{T(0), T(0)};
        for (int s = 0; s < S; ++s) {
          const T w = Wl[k * S + s];
          const long src = 2 * ((long)s * nlm + base + m);
          fv.x = fma(w, fb[src], fv.x); fv.y = fma(w, fb[src + 1], fv.y);
          hv.x = fma(w, hb[src], hv.x); hv.y = fma(w, hb[src + 1], hv.y);
        }
        Fd[t] = fv; Hd[t] = hv;
      }
    } else {
      for (int t = threadIdx.x; t < S * no; t += blockDim.x) {
        int s = t / no, m = t - s * no;
        long src = 2 * ((long)s * nlm + base + m);
        T w = (T)wrad[s];
        C2 fv, hv;
        fv.x = fb[src]; fv.y = fb[src + 1];
        hv.x = w * hb[src]; hv.y = w * hb[src + 1];
        Fd[t] = fv; Hd[t] = hv;
      }
    }
  }
  __syncthreads();
  // Products over the shells for every order pair (a, b), 0 <= a, b <= l:
  //   A = sum f_a.re h_b.re, B = sum f_a.im h_b.im, C = sum f_a.im h_b.re, D = sum f_a.re h_b.im,
  // so that P1 = sum f_a conj(h_b) = (A + B) + i (C - D) and P2 = sum f_a h_b =
  // (A - B) + i (C + D).  With f_{l,-k} = (-1)^k conj(f_{lk}) (real volumes):
  //   c_mn = P1[m][n] (n >= 0),  (-1)^|n| P2[m][|n|] (n < 0),
  //   c_nm = P1[n][m] (n >= 0),  (-1)^|n| conj(P2[|n|][m]) (n < 0).
  // One thread per 2 x 2 block of (a, b): two 128-bit loads per shell feed 16
  // multiply-adds.
  const int h0 = (l_lo + 2) / 2, h1 = (l_hi + 2) / 2;  // blocks per side
  const int t_lo = h0 * h0, t_tot = t_lo + (npass == 2 ? h1 * h1 : 0);
  for (int t = threadIdx.x; t < t_tot; t += blockDim.x) {
    const int d = t < t_lo ? 0 : 1, tt = d ? t - t_lo : t, hh = d ? h1 : h0;
    const int l = d ? l_hi : l_lo, no = l + 1;
    const int a0 = 2 * (tt / hh), b0 = 2 * (tt - (tt / hh) * hh);
    // rows past l read a zero-weighted copy of row l (loaded, never stored)
    const int a1 = a0 + 1 <= l ? a0 + 1 : a0, b1 = b0 + 1 <= l ? b0 + 1 : b0;
    T acc[2][2][4];
#pragma unroll
    for (int u = 0; u < 2; ++u)
#pragma unroll
      for (int v = 0; v < 2; ++v)
#pragma unroll
        for (int k = 0; k < 4; ++k) acc[u][v][k] = 0;
    const C2 *F = d ? F1 : F0, *H = d ? H1 : H0;
    const int Sd = d ? S1 : S0;
    for (int s = 0; s < Sd; ++s, F += no, H += no) {
      const C2 fa[2] = {F[a0], F[a1]}, hb[2] = {H[b0], H[b1]};
#pragma unroll
      for (int u = 0; u < 2; ++u)
#pragma unroll
        for (int v = 0; v < 2; ++v) {
          acc[u][v][0] = fma(fa[u].x, hb[v].x, acc[u][v][0]);
          acc[u][v][1] = fma(fa[u].y, hb[v].y, acc[u][v][1]);
          acc[u][v][2] = fma(fa[u].y, hb[v].x, acc[u][v][2]);
          acc[u][v][3] = fma(fa[u].x, hb[v].y, acc[u][v][3]);
        }
    }
#pragma unroll
    for (int u = 0; u < 2; ++u)
#pragma unroll
      for (int v = 0; v < 2; ++v) {
        const int ai = a0 + u, bi = b0 + v;
        if (ai > l || bi > l) continue;
        const T A = acc[u][v][0], B = acc[u][v][1], C = acc[u][v][2], D = acc[u][v][3];
        const T p1r = A + B, p1i = C - D, p2r = A - B, p2i = C + D;
        // P1[ai][bi]: c_mn of pair (ai, bi) when ai >= bi; c_nm of pair (bi, ai) when ai <= bi
        if (ai >= bi) {
          const int m = ai, n = bi, q = m * m + n + m;
          T *o = cb + pair_base[q] + 8L * (l - m);
          o[0] = p1r; o[2] = p1i;
          if (n == m) { o[4] = p1r; o[6] = p1i; o[1] = 0; o[3] = 0; o[5] = 0; o[7] = 0; }
        }
        if (ai < bi) {
          const int m = bi, n = ai, q = m * m + n + m;
          T *o = cb + pair_base[q] + 8L * (l - m);
          o[4] = p1r; o[6] = p1i;
        }
        // P2[ai][bi] with the smaller index k > 0 as |n|: pair (max, -min)
        const int mx = ai > bi ? ai : bi, k = ai > bi ? bi : ai;
        if (k > 0) {
          const T sg = (k & 1) ? T(-1) : T(1);
          const int q = mx * mx - k + mx;
          T *o = cb + pair_base[q] + 8L * (l - mx);
          if (ai >= bi) { o[0] = sg * p2r; o[2] = sg * p2i; }    // c_{m,-k} = (-1)^k P2[m][k]
          if (ai <= bi) { o[4] = sg * p2r; o[6] = -sg * p2i; }   // c_{-k,m} = (-1)^k conj(P2[k][m])
        }
      }
  }
}

// N complex values from a 16-byte aligned address
template <int N>
__device__ __forceinline__ void ld_orders(const float2 *p, float2 (&v)[N]) {
#pragma unroll
  for (int i = 0; i < N; i += 2) {
    const float4 q = *reinterpret_cast<const float4 *>(p + i);
    v[i] = make_float2(q.x, q.y);
    v[i + 1] = make_float2(q.z, q.w);
  }
}
// 2 x 4 blocks of orders of degree l
__host__ __device__ __forceinline__ int blocks_of(int l) { return ((l + 2) / 2) * ((l + 4) / 4); }
// row lengths of the staged orders 0..l of F and H, and of the products
__host__ __device__ __forceinline__ int f_row(int l) { return (l + 2) & ~1; }
__host__ __device__ __forceinline__ int h_row(int l) { return (l + 4) & ~3; }
__host__ __device__ __forceinline__ int p_row(int l) { return (l + 1) | 1; }

// The same in FP32 with whole output records.  A thread takes a block of 2 x 4 orders:
// per shell three 16-byte loads (a row of F is broadcast) and 16 packed multiply-adds.
// The block's products go through shared memory, so that the records of the output are
// written whole (neighbouring lanes write a record's halves) instead of as single reals.
// 256 particles, 32 shells, L_J = 32: 88 -> 71 us (15 to read and write the
// coefficients), bound by the latencies of its three phases.
template <bool BALL>
__global__ void __launch_bounds__(256)
k_correlate_rec(const float *__restrict__ f, const float *__restrict__ h, int S, int L, long h_stride,
                const double *__restrict__ wrad, long nc, float *__restrict__ c, const float *__restrict__ ballW,
                const int *__restrict__ ballK, int Kmax) {
  using T = float;
  using C2 = float2;
  const long b = blockIdx.y;
  const int nlm = (L + 1) * (L + 2) / 2;
  const T *fb = f + 2 * b * (long)S * nlm;
  const T *hb = h + 2 * (b * h_stride) * (long)S * nlm;
  T *cb = c + 4 * b * nc;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  C2 *sF = reinterpret_cast<C2 *>(smem_raw);
  const int l_lo = blockIdx.x, l_hi = L - blockIdx.x;
  const int npass = l_hi == l_lo ? 1 : 2;
  // stage: degree d's orders 0..l at [S][f_row] (F) and [S][h_row] (w H)
  const int R0 = BALL ? Kmax : S;  // rows reserved per degree
  C2 *F0 = sF, *H0 = F0 + R0 * f_row(l_lo), *F1 = H0 + R0 * h_row(l_lo), *H1 = F1 + R0 * f_row(l_hi);
  // rows summed per degree: the shells, or the retained radial functions
  const int S0 = BALL ? ballK[l_lo] : S, S1 = BALL ? ballK[l_hi] : S;
  __shared__ T wsh[256];  // the radial weights, converted once
  const bool wtab = !BALL && S <= 256;
  if (wtab)
    for (int s = threadIdx.x; s < S; s += blockDim.x) wsh[s] = (T)wrad[s];
  __syncthreads();
  for (int d = 0; d < npass; ++d) {
    const int l = d ? l_hi : l_lo, no = l + 1, base = l * (l + 1) / 2, fr = f_row(l), hr = h_row(l);
    C2 *Fd = d ? F1 : F0, *Hd = d ? H1 : H0;
    const FastDiv dno(no);
    if (BALL) {
      const int Kl = d ? S1 : S0;
      const T *Wl = ballW + (long)l * Kmax * S;
      for (int t = threadIdx.x; t < Kl * no; t += blockDim.x) {
        const int k = dno.div(t), m = t - k * no;
        C2 fv{T(0), T(0)}, hv{T(0), T(0)};
        for (int s = 0; s < S; ++s) {
          const T w = Wl[k * S + s];
          const long src = 2 * ((long)s * nlm + base + m);
          fv.x = fma(w, fb[src], fv.x); fv.y = fma(w, fb[src + 1], fv.y);
          hv.x = fma(w, hb[src], hv.x); hv.y = fma(w, hb[src + 1], hv.y);
        }
        Fd[k * fr + m] = fv; Hd[k * hr + m] = hv;
      }
    } else {
#pragma unroll 4
      for (int t = threadIdx.x; t < S * no; t += blockDim.x) {
        const int s = dno.div(t), m = t - s * no;
        const long src = 2 * ((long)s * nlm + base + m);
        const T w = wtab ? wsh[s] : (T)wrad[s];
        C2 fv, hv;
        fv.x = fb[src]; fv.y = fb[src + 1];
        hv.x = w * hb[src]; hv.y = w * hb[src + 1];
        Fd[s * fr + m] = fv; Hd[s * hr + m] = hv;
      }
    }
  }
  __syncthreads();
  // Products over the shells for every order pair (a, b), 0 <= a, b <= l:
  //   A = sum f_a.re h_b.re, B = sum f_a.im h_b.im, C = sum f_a.im h_b.re, D = sum f_a.re h_b.im,
  // so that P1 = sum f_a conj(h_b) = (A + B) + i (C - D) and P2 = sum f_a h_b =
  // (A - B) + i (C + D).  With f_{l,-k} = (-1)^k conj(f_{lk}) (real volumes):
  //   c_mn = P1[m][n] (n >= 0),  (-1)^|n| P2[m][|n|] (n < 0),
  //   c_nm = P1[n][m] (n >= 0),  (-1)^|n| conj(P2[|n|][m]) (n < 0).
  // (a, b) past l read whatever the rows' padding holds and are never stored.
  constexpr int V = 4;
  const int t_lo = blocks_of(l_lo), t_tot = t_lo + (npass == 2 ? blocks_of(l_hi) : 0);
  C2 ad[2][V], cbq[2][V];  // (A, D), (C, B)
  auto products = [&](int t) {
    const int d = t < t_lo ? 0 : 1, tt = d ? t - t_lo : t;
    const int l = d ? l_hi : l_lo, hh = (l + V) / V, fr = f_row(l), hr = h_row(l);
    const int aq = tt / hh, a0 = 2 * aq, b0 = V * (tt - aq * hh);
#pragma unroll
    for (int u = 0; u < 2; ++u)
#pragma unroll
      for (int v = 0; v < V; ++v) ad[u][v].x = ad[u][v].y = cbq[u][v].x = cbq[u][v].y = T(0);
    const C2 *F = (d ? F1 : F0) + a0, *H = (d ? H1 : H0) + b0;
    const int Sd = d ? S1 : S0;
    for (int s = 0; s < Sd; ++s, F += fr, H += hr) {
      C2 fa[2], hv[V];
      ld_orders(F, fa);
      ld_orders(H, hv);
#pragma unroll
      for (int u = 0; u < 2; ++u)
#pragma unroll
        for (int v = 0; v < V; ++v) {
          ad[u][v] = __ffma2_rn(make_float2(fa[u].x, fa[u].x), hv[v], ad[u][v]);
          cbq[u][v] = __ffma2_rn(make_float2(fa[u].y, fa[u].y), hv[v], cbq[u][v]);
        }
    }
  };
  // [l+1][p_row] of P1, then of P2, of both degrees; a thread has at most one block
  // per sweep, and the sweeps of a CTA write after all have read
  C2 *P0 = sF + R0 * (f_row(l_lo) + h_row(l_lo) + (npass == 2 ? f_row(l_hi) + h_row(l_hi) : 0));
  if (blockDim.x >= t_tot) P0 = sF;
  auto p_of = [&](int d) { return P0 + (d ? 2 * (l_lo + 1) * p_row(l_lo) : 0); };
  for (int t0 = 0; t0 < t_tot; t0 += blockDim.x) {
    const int t = t0 + threadIdx.x;
    if (t < t_tot) products(t);
    if (P0 == sF) __syncthreads();
    if (t >= t_tot) continue;
    const int d = t < t_lo ? 0 : 1, tt = d ? t - t_lo : t, l = d ? l_hi : l_lo, hh = (l + V) / V;
    const int aq = tt / hh, a0 = 2 * aq, b0 = V * (tt - aq * hh), pr = p_row(l);
    C2 *P1 = p_of(d), *P2 = P1 + (l + 1) * pr;
#pragma unroll
    for (int u = 0; u < 2; ++u)
#pragma unroll
      for (int v = 0; v < V; ++v) {
        const int ai = a0 + u, bi = b0 + v;
        if (ai > l || bi > l) continue;
        const T A = ad[u][v].x, D = ad[u][v].y, C = cbq[u][v].x, B = cbq[u][v].y;
        P1[ai * pr + bi] = C2{A + B, C - D};
        P2[ai * pr + bi] = C2{A - B, C + D};
      }
  }
  __syncthreads();
  // half records: (c_mn) for n = n0, n0 + 1, then (c_nm)
  for (int d = 0; d < npass; ++d) {
    const int l = d ? l_hi : l_lo, pr = p_row(l);
    const C2 *P1 = p_of(d), *P2 = P1 + (l + 1) * pr;
    for (int t = threadIdx.x; t < (l + 1) * (l + 2); t += blockDim.x) {
      const int g = t >> 1, m = tri_floor(g), j = g - m * (m + 1) / 2;
      const bool second = t & 1;
      T o[4];
#pragma unroll
      for (int hh = 0; hh < 2; ++hh) {
        const int n = 2 * j - m + hh, k = n < 0 ? -n : n;
        C2 v{T(0), T(0)};
        if (n <= m) {
          v = (n < 0 ? P2 : P1)[second ? k * pr + m : m * pr + k];
          if (n < 0) {
            const T sg = (k & 1) ? T(-1) : T(1);
            v.x = sg * v.x;
            v.y = second ? -sg * v.y : sg * v.y;
          }
        }
        o[hh] = v.x;
        o[2 + hh] = v.y;
      }
      const int tm = m * (m + 1);
      const int go = (L + 2) * (tm / 2) - tm * (2 * m + 1) / 6 + j * (L - m + 1);
      T *dst = cb + 8L * (go + l - m) + 4 * second;
      *reinterpret_cast<float4 *>(dst) = make_float4(o[0], o[1], o[2], o[3]);
    }
  }
}

template <typename T>
cudaError_t launch_correlate(const Plan &p, const T *f, const T *h, int B, int hstride, T *c,
                             cudaStream_t st) {
  if (B == 0) return cudaSuccess;
  if (sizeof(T) == 4 && p.tc)
    return launch_correlate_tc(p, (const float *)f, (const float *)h, B, hstride, (float *)c, st);
  const bool ball = p.ball_kmax > 0;
  const int rows = ball ? p.ball_kmax : p.S;
  const size_t direct = sizeof(T) * 4 * (size_t)rows * (p.LJ + 2);  // both degrees of a pair
  const dim3 grid(p.LJ / 2 + 1, B);
  cudaError_t e;
  if constexpr (sizeof(T) == 4) {
    // threads: the fewest sweeps of at most 256 over the blocks of the pair {0, L_J}, the
    // largest but for a few; staged rows and products of the pair that needs most
    int most = 0;
    size_t stage = 0, prod = 0;
    for (int q = 0; 2 * q <= p.LJ; ++q) {
      const int l0 = q, l1 = p.LJ - q, two = l0 != l1;
      most = std::max(most, blocks_of(l0) + two * blocks_of(l1));
      stage = std::max(stage, (size_t)(f_row(l0) + h_row(l0) + two * (f_row(l1) + h_row(l1))));
      prod = std::max(prod, 2 * (size_t)((l0 + 1) * p_row(l0) + two * (l1 + 1) * p_row(l1)));
    }
    const int sweeps = (most + 255) / 256;
    const long ctas = (long)B * (p.LJ / 2 + 1);
    // (all 256 for few CTAs, whose staging and stores they share)
    const int threads = ctas <= 2L * p.sms ? 256 : std::max(128, ((most + sweeps - 1) / sweeps + 31) / 32 * 32);
    stage *= 2 * sizeof(T) * rows;
    prod *= 2 * sizeof(T);
    // a single sweep's products take the place of the staged rows
    const size_t both = sweeps == 1 ? std::max(stage, prod) : stage + prod;
    // The records win while all CTAs run at once, while shared memory leaves as many on an
    // SM as without them (three at most count), or two where the stores weigh more than the products (300 particles: 24
    // shells, L_J = 64, 603 -> 523 us; 40 shells, L_J = 50, 430 -> 476; 100 shells, L_J =
    // 60, 1.55 -> 2.09 ms on one instead of two), and not in small plans while SMs are idle,
    // where their third phase is one more latency (36 particles, L_J = 14, 9.4 -> 10.9
    // us; 100: 13.0 -> 11.9).
    auto fit = [](size_t bytes) { return 228 * 1024 / (bytes + 2048); };
    const bool residency = ctas <= (long)(p.sms * fit(both)) || fit(both) >= std::min<size_t>(3, fit(direct)) || (fit(both) == 2 && 2 * prod >= 3 * stage);
    const bool small = p.LJ <= 24 && ctas <= 4L * p.sms;
    if (prod <= 72 * 1024 && both <= 200 * 1024 && residency && !small && (uintptr_t)c % 16 == 0) {
      auto kern = ball ? k_correlate_rec<true> : k_correlate_rec<false>;
      if ((e = allow_smem(kern, both, 1024)) != cudaSuccess) return e;
      kern<<<grid, threads, both, st>>>(f, h, p.S, p.LJ, hstride, p.wrad, p.nc, c,
                                        ball ? (const T *)p.ball_W : nullptr, ball ? p.ball_K : nullptr,
                                        ball ? p.ball_kmax : 0);
      return cudaGetLastError();
    }
  }
  auto kern = ball ? k_correlate_deg<T, true> : k_correlate_deg<T, false>;
  if ((e = allow_smem(kern, direct)) != cudaSuccess) return e;
  kern<<<grid, 256, direct, st>>>(f, h, p.S, p.LJ, hstride, p.wrad, p.pair_base, p.nc, c,
                                  ball ? (const T *)p.ball_W : nullptr, ball ? p.ball_K : nullptr,
                                  ball ? p.ball_kmax : 0);
  return cudaGetLastError();
}

template cudaError_t launch_correlate<float>(const Plan &, const float *, const float *, int, int,
                                             float *, cudaStream_t);
template cudaError_t launch_correlate<double>(const Plan &, const double *, const double *, int,
                                              int, double *, cudaStream_t);

}  // namespace matcha
