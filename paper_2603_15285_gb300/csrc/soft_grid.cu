// Steps a4+a5 through memory: C_{L0} on the SOFFT grid (Section 2.3) written
// to HBM, then its P strongest local maxima, for grids that no on-chip kernel
// of soft.cu holds (L0 = 30, K = 2: 124^3 points per particle) and wherever
// the caller passes a grid and only the slice-streaming kernel would fit.
//
//   k_soft_beta   S_mn(beta_k) = sum_l c^l_mn d^l_mn(beta_k), rows m >= 0, with
//                 the threads along k (the transposed d table is read in
//                 order, the c of a group is one broadcast);
//   k_soft_slab   per beta slice the two DFT stages as register-tiled products
//                 against shared operand tables, packed FP32x2 in 32 bits;
//   k_soft_peaks  a cluster of CTAs per particle: separable 3x3x3 maximum in
//                 registers, the exact (value, index) test for the points that
//                 equal it, per-warp best-P lists merged through distributed
//                 shared memory.
//
// GB300, 32 particles at 124 points per angle (FP32): beta 0.053, slab 0.47,
// peaks 0.13 ms (one kernel with untiled stages and one search CTA per particle:
// 2.09 + 2.26); 121 particles at 72 points: 0.013 + 0.125 + 0.153 ms (streamed on
// one CTA per particle: 2.37).
//
// Rounding: the sums take their terms in the order of k_soft_stream
// (soft.cu), as x + (a b - c d) with the difference fused once, so every grid
// value has the bits that kernel gives; the folded signs are exact.
#include <algorithm>
#include <cooperative_groups.h>
#include <float.h>
#include <limits.h>
#include "internal.cuh"

namespace matcha {
namespace {

namespace cg = cooperative_groups;

template <typename T> struct Pair;
template <> struct Pair<float> { typedef float2 type; };
template <> struct Pair<double> { typedef double2 type; };
template <typename T> struct alignas(4 * sizeof(T) > 16 ? 16 : 4 * sizeof(T)) Quad { T v[4]; };

__device__ __forceinline__ float2 pfma(float2 a, float2 b, float2 c) { return __ffma2_rn(a, b, c); }
__device__ __forceinline__ float2 pmul(float2 a, float2 b) { return __fmul2_rn(a, b); }
__device__ __forceinline__ float2 padd(float2 a, float2 b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ double2 pfma(double2 a, double2 b, double2 c) {
  return make_double2(__fma_rn(a.x, b.x, c.x), __fma_rn(a.y, b.y, c.y));
}
__device__ __forceinline__ double2 pmul(double2 a, double2 b) {
  return make_double2(__dmul_rn(a.x, b.x), __dmul_rn(a.y, b.y));
}
__device__ __forceinline__ double2 padd(double2 a, double2 b) {
  return make_double2(__dadd_rn(a.x, b.x), __dadd_rn(a.y, b.y));
}
__device__ __forceinline__ float2 pdup(float x) { return make_float2(x, x); }
__device__ __forceinline__ double2 pdup(double x) { return make_double2(x, x); }
__device__ __forceinline__ float2 pset(float x, float y) { return make_float2(x, y); }
__device__ __forceinline__ double2 pset(double x, double y) { return make_double2(x, y); }

// The beta slice k of a particle owns the grid rows (i, k, 0..ns-1) for every
// i; until k_soft_slab writes them they hold the sums of the slice's order
// pairs: real f of the flat [pair q = m^2 + n + m][Re, Im of (m, n), Re, Im of
// (n, m)] array sits at row i = f / ns, column f % ns.  4 (L0+1)^2 <= ns^2.
__device__ __forceinline__ long stash_at(int f, int ns, int k, const FastDiv &dns) {
  const int i = dns.div(f);
  return ((long)i * ns + k) * ns + (f - i * ns);
}

// One thread per beta slice; a block takes a few partner groups (m, n_a),
// (m, n_a + 1) one after the other for two particles, so each read of
// the transposed d table (in order along the slices) serves both; the c of a
// degree are broadcast loads.  VEC: c and the grid rows are 16-byte aligned.
constexpr int BETA_GROUPS = 2, BETA_NB = 2;

template <typename T, bool VEC>
__global__ void __launch_bounds__(128)
k_soft_beta(const T *__restrict__ c, long nc, int LJ, int L0, int ns, int B,
            const T *__restrict__ dT, T *__restrict__ grid) {
  const int b0 = blockIdx.y * BETA_NB, nb = min(BETA_NB, B - b0);
  const int ng = (L0 + 1) * (L0 + 2) / 2;
  const FastDiv dns(ns);
  const long cs = nb > 1 ? 4 * nc : 0;  // a missing second particle reads the first
  // groups gridDim.x apart: every block gets long and short ones
  for (int g = blockIdx.x; g < ng; g += gridDim.x) {
    const int m = tri_floor(g), j = g - m * (m + 1) / 2, na = 2 * j - m;
    const long t = (long)m * (m + 1) / 2, m3 = (long)m * (m + 1) * (2 * m + 1) / 6;
    // entries of group (m, j) in the L_J layout; of pair (m, n_a) in the SOFFT layout
    const T *cp = c + 4 * b0 * nc + 8 * ((long)(LJ + 2) * t - m3 + (long)j * (LJ - m + 1));
    const long d0 = (long)(L0 + 1) * m * m - (long)m * (m - 1) * (4 * m + 1) / 6 +
                    (long)(na + m) * (L0 - m + 1);
    const bool two = na < m;
    const int len = L0 - m + 1;
    for (int k = threadIdx.x; k < ns; k += blockDim.x) {
      const T *da = dT + d0 * ns + k, *db = two ? da + (long)len * ns : da;
      T s[BETA_NB][8];  // (Re, Im of c_mn, c_nm) x 2 slots
#pragma unroll
      for (int u = 0; u < BETA_NB; ++u)
#pragma unroll
        for (int q = 0; q < 8; ++q) s[u][q] = T(0);
#pragma unroll 2
      for (int l = 0; l < len; ++l) {
        T e[BETA_NB][8];
#pragma unroll
        for (int u = 0; u < BETA_NB; ++u) {
          const T *ce = cp + u * cs + 8 * l;
          if (VEC) {
            const Quad<T> x = *reinterpret_cast<const Quad<T> *>(ce);
            const Quad<T> y = *reinterpret_cast<const Quad<T> *>(ce + 4);
#pragma unroll
            for (int q = 0; q < 4; ++q) { e[u][q] = x.v[q]; e[u][4 + q] = y.v[q]; }
          } else {
#pragma unroll
            for (int q = 0; q < 8; ++q) e[u][q] = ce[q];
          }
        }
        const T va = __ldg(da + (long)l * ns), vb = __ldg(db + (long)l * ns);
#pragma unroll
        for (int u = 0; u < BETA_NB; ++u)
#pragma unroll
          for (int q = 0; q < 4; ++q) {
            s[u][2 * q] = fma(e[u][2 * q], va, s[u][2 * q]);
            s[u][2 * q + 1] = fma(e[u][2 * q + 1], vb, s[u][2 * q + 1]);
          }
      }
#pragma unroll
      for (int u = 0; u < BETA_NB; ++u) {
        if (u >= nb) continue;
        T *gb = grid + (b0 + u) * (long)ns * ns * ns;
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          const int n = na + h, f = 4 * (m * m + n + m);
          if (n > m) continue;
          const bool odd = (m - n) & 1;  // d^l_nm = (-1)^{m-n} d^l_mn
          const Quad<T> r{s[u][h], s[u][2 + h], odd ? -s[u][4 + h] : s[u][4 + h],
                          odd ? -s[u][6 + h] : s[u][6 + h]};
          if (VEC) {
            *reinterpret_cast<Quad<T> *>(gb + stash_at(f, ns, k, dns)) = r;
          } else {
#pragma unroll
            for (int q = 0; q < 4; ++q) gb[stash_at(f + q, ns, k, dns)] = r.v[q];
          }
        }
      }
    }
  }
}

// Geometry of k_soft_slab, shared by the launcher: KS beta slices per CTA, IC
// alpha rows per operand table.
template <typename T> struct Tile;
template <> struct Tile<float> { static constexpr int I = 8, J = 8; };
template <> struct Tile<double> { static constexpr int I = 4, J = 4; };
__host__ __device__ __forceinline__ int round_up(int x, int a) { return (x + a - 1) / a * a; }
__host__ __device__ __forceinline__ int slab_pairs(int L0) { return round_up(L0 + 1, 4) / 2; }
template <typename T>
__host__ __device__ __forceinline__ long slab_reals(int L0, int ns, int KS, int IC) {
  const int W = 2 * L0 + 1, NJ = round_up(ns, Tile<T>::J);
  return round_up(2 * ns, 4) + (long)KS * W * slab_pairs(L0) * 4 + (long)KS * 2 * (L0 + 1) * NJ +
         2L * (L0 + 1) * IC;
}

// Two DFT stages of KS beta slices of one particle:
//   G_m(j) = sum_n S_mn e^{i n g_j};  C(i, j) = Re G_0(j) + 2 sum_{m>=1} Re(G_m(j) e^{i m a_i}).
// Bound by the FP32 pipe (the difference of each complex product is rounded
// before it is added, so a packed product pair costs three operations, not two;
// 0.47 ms against 0.29 of pure packed arithmetic at 32 x 124^3 points).  Stage 2 items are 4
// rows m (two packed pairs, one 16-byte broadcast of S each) x 4 gammas a quarter
// of the padded range apart (neighbouring lanes then gather twiddles at index
// steps of n, which spread over the banks; four adjacent gammas would step by
// 4 n and meet in four bank groups); stage
// 3 items are 8 x 8 tiles (4 x 4 in FP64) whose alpha operands come as packed
// pairs and whose rows and columns are two quads half the padded range apart,
// so that the lanes of a 16-byte shared load read consecutive quads.  As many
// slices share a CTA as give its 256 threads one tile each.
// FP64 is bound by its pipe, an operation holding a quarter SM as long for one lane as
// for 32, so stage 2 items are one pair of rows x one gamma there, enough for all warps
// (four rows x four gammas at 52 points: 52 items on two of the four quarters), and two
// CTAs share an SM, one's arithmetic over the other's barriers.  140 particles at 52
// points: 5.35 ms -> 3.02 (4.46 streamed on one CTA per particle).
template <typename T>
__global__ void __launch_bounds__(256, 2)
k_soft_slab(int L0, int ns, int KS, int IC, const T *__restrict__ tw, T *__restrict__ grid, int vec) {
  typedef typename Pair<T>::type P2;
  constexpr int TI = Tile<T>::I, TJ = Tile<T>::J, QI = TI / 4, QJ = TJ / 4;
  constexpr int SV = sizeof(T) == 8 ? 1 : 2, SU = sizeof(T) == 8 ? 1 : 4;  // stage 2 item: row pairs, gammas
  const long b = blockIdx.y;
  const int k0 = blockIdx.x * KS, nk = min(KS, ns - k0);
  const int W = 2 * L0 + 1, M1 = L0 + 1, MP = slab_pairs(L0), NJ = round_up(ns, TJ);
  const int tid = threadIdx.x, NT = blockDim.x;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  T *tws = reinterpret_cast<T *>(smem_raw);          // [ns][2]
  T *Sp = tws + round_up(2 * ns, 4);                  // [KS][W][MP][4]: (re, re, im, im) of rows 2p, 2p+1
  T *G = Sp + (long)KS * W * MP * 4;                  // [KS][M1][re|im][NJ]
  T *At = G + (long)KS * 2 * M1 * NJ;                 // [M1][cos|-sin][IC]
  T *gb = grid + b * (long)ns * ns * ns;
  const FastDiv dns(ns);
  for (int t = tid; t < 2 * ns; t += NT) tws[t] = tw[t];
  __syncthreads();
  // alpha operands cos m a_i, -sin m a_i of rows ib .. ib + ni - 1
  auto alpha_table = [&](int ib, int ni) {
    const FastDiv dni(ni);
    for (int t = tid; t < M1 * ni; t += NT) {
      const int m = dni.div(t), i = t - m * ni;
      const int mi = m * (ib + i), r = mi - dns.div(mi) * ns;
      At[(2 * m) * IC + i] = tws[2 * r];
      At[(2 * m + 1) * IC + i] = -tws[2 * r + 1];
    }
  };
  // S rows m >= 0 from the stashed pairs and their images; the first loads are
  // in flight while the first operand table is made
  {
    constexpr int NL = 4;
    const int np0 = M1 * M1, tot = nk * np0;
    const FastDiv dnp(np0);
    T r[NL][4];
    auto load = [&](int t0) {
#pragma unroll
      for (int x = 0; x < NL; ++x) {
        const int t = t0 + x * NT;
        if (t >= tot) continue;
        const int kk = dnp.div(t), f = 4 * (t - kk * np0);
        if (vec) {
          const Quad<T> v = *reinterpret_cast<const Quad<T> *>(gb + stash_at(f, ns, k0 + kk, dns));
#pragma unroll
          for (int e = 0; e < 4; ++e) r[x][e] = v.v[e];
        } else {
#pragma unroll
          for (int e = 0; e < 4; ++e) r[x][e] = gb[stash_at(f + e, ns, k0 + kk, dns)];
        }
      }
    };
    load(tid);
    alpha_table(0, min(IC, round_up(ns, TI)));
    for (int t0 = tid; t0 < tot; t0 += NL * NT) {
      if (t0 != tid) load(t0);
#pragma unroll
      for (int x = 0; x < NL; ++x) {
        const int t = t0 + x * NT;
        if (t >= tot) continue;
        const int kk = dnp.div(t), q = t - kk * np0, m = isqrt_floor(q), n = q - m * m - m;
        T *S = Sp + (long)kk * W * MP * 4;
        auto put = [&](int u, int v, T re, T im) {
          T *o = S + ((v + L0) * MP + (u >> 1)) * 4 + (u & 1);
          o[0] = re;
          o[2] = im;
        };
        put(m, n, r[x][0], r[x][1]);
        if (n != m && n != -m) {  // (n, m), and (-n, -m) its conjugate
          if (n >= 0) put(n, m, r[x][2], r[x][3]);
          if (n <= 0) put(-n, -m, r[x][2], -r[x][3]);
        }
      }
    }
    const int pad = (2 * MP - M1) * W;  // rows past M1 are zero
    for (int t = tid; t < nk * pad; t += NT) {
      const int kk = t / pad, q = t - kk * pad, u = M1 + q / W;
      T *o = Sp + ((long)kk * W * MP + (q % W) * MP + (u >> 1)) * 4 + (u & 1);
      o[0] = o[2] = T(0);
    }
  }
  __syncthreads();
  {
    const int jt = NJ / SU, mt = ((M1 + 1) / 2 + SV - 1) / SV;
    const FastDiv djt(jt), dmt(mt);
    for (int t = tid; t < nk * mt * jt; t += NT) {
      const int km = djt.div(t), jq = t - km * jt, kk = dmt.div(km), mq = km - kk * mt;
      int tt[SU], js[SU];
#pragma unroll
      for (int u = 0; u < SU; ++u) {
        const int j = jq + u * jt;
        js[u] = j < ns ? j : 0;  // columns of the padding are computed as column 0, never stored
        const int lj = L0 * js[u], r = lj - dns.div(lj) * ns;
        tt[u] = r ? ns - r : 0;  // (-L0 j) mod ns
      }
      P2 re[SV][SU], im[SV][SU];
#pragma unroll
      for (int v = 0; v < SV; ++v)
#pragma unroll
        for (int u = 0; u < SU; ++u) re[v][u] = im[v][u] = pdup(T(0));
      const T *row = Sp + ((long)kk * W * MP + SV * mq) * 4;
      for (int n = 0; n < W; ++n, row += 4 * MP) {
        P2 sr[SV], si[SV];
#pragma unroll
        for (int v = 0; v < SV; ++v) {
          const Quad<T> s = *reinterpret_cast<const Quad<T> *>(row + 4 * v);
          sr[v] = pset(s.v[0], s.v[1]);
          si[v] = pset(s.v[2], s.v[3]);
        }
#pragma unroll
        for (int u = 0; u < SU; ++u) {
          const P2 e = *reinterpret_cast<const P2 *>(tws + 2 * tt[u]);
          const P2 cr = pdup(e.x), ci = pdup(e.y), ni = pdup(-e.y);
#pragma unroll
          for (int v = 0; v < SV; ++v) {
            re[v][u] = padd(re[v][u], pfma(sr[v], cr, pmul(si[v], ni)));
            im[v][u] = padd(im[v][u], pfma(sr[v], ci, pmul(si[v], cr)));
          }
          tt[u] += js[u];
          if (tt[u] >= ns) tt[u] -= ns;
        }
      }
#pragma unroll
      for (int v = 0; v < SV; ++v)
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          const int m = 2 * (SV * mq + v) + h;
          if (m >= M1) continue;
          T *o = G + ((long)kk * M1 + m) * 2 * NJ + jq;
#pragma unroll
          for (int u = 0; u < SU; ++u) {
            o[u * jt] = h ? re[v][u].y : re[v][u].x;
            o[NJ + u * jt] = h ? im[v][u].y : im[v][u].x;
          }
        }
    }
  }
  const int jt = NJ / TJ, jh = NJ / 4 / QJ;  // tiles, quads per half
  for (int ib = 0; ib < ns; ib += IC) {
    const int ni = min(IC, round_up(ns - ib, TI));
    if (ib) {
      __syncthreads();
      alpha_table(ib, ni);
    }
    __syncthreads();
    const int it = ni / TI, ih = ni / 4 / QI;
    const FastDiv djt(jt), dit(it);
    for (int t = tid; t < nk * it * jt; t += NT) {
      const int ki = djt.div(t), jq = t - ki * jt, kk = dit.div(ki), iq = ki - kk * it;
      const T *Gk = G + (long)kk * M1 * 2 * NJ + 4 * jq, *Ai = At + 4 * iq;
      P2 acc[TI / 2][TJ];
#pragma unroll
      for (int u = 0; u < TI / 2; ++u)
#pragma unroll
        for (int v = 0; v < TJ; ++v) acc[u][v] = pdup(T(0));
      for (int m = 1; m < M1; ++m) {
        P2 co[TI / 2], sn[TI / 2];
        const T *am = Ai + 2 * m * IC, *gm = Gk + (long)m * 2 * NJ;
#pragma unroll
        for (int q = 0; q < QI; ++q) {
          const Quad<T> x = *reinterpret_cast<const Quad<T> *>(am + 4 * q * ih);
          const Quad<T> y = *reinterpret_cast<const Quad<T> *>(am + IC + 4 * q * ih);
          co[2 * q] = pset(x.v[0], x.v[1]); co[2 * q + 1] = pset(x.v[2], x.v[3]);
          sn[2 * q] = pset(y.v[0], y.v[1]); sn[2 * q + 1] = pset(y.v[2], y.v[3]);
        }
#pragma unroll
        for (int q = 0; q < QJ; ++q) {
          const Quad<T> gr = *reinterpret_cast<const Quad<T> *>(gm + 4 * q * jh);
          const Quad<T> gi = *reinterpret_cast<const Quad<T> *>(gm + NJ + 4 * q * jh);
#pragma unroll
          for (int v = 0; v < 4; ++v) {
            const P2 a = pdup(gr.v[v]), bb = pdup(gi.v[v]);
#pragma unroll
            for (int u = 0; u < TI / 2; ++u)
              acc[u][4 * q + v] = padd(acc[u][4 * q + v], pfma(a, co[u], pmul(bb, sn[u])));
          }
        }
      }
      T g0[TJ];
#pragma unroll
      for (int q = 0; q < QJ; ++q) {
        const Quad<T> g = *reinterpret_cast<const Quad<T> *>(Gk + 4 * q * jh);
#pragma unroll
        for (int v = 0; v < 4; ++v) g0[4 * q + v] = g.v[v];
      }
#pragma unroll
      for (int u = 0; u < TI; ++u) {
        const int i = ib + 4 * (iq + (u >> 2) * ih) + (u & 3);
        if (i >= ns) continue;
        T *o = gb + ((long)i * ns + k0 + kk) * ns;
#pragma unroll
        for (int q = 0; q < QJ; ++q) {
          const int j = 4 * (jq + q * jh);
          Quad<T> r;
#pragma unroll
          for (int v = 0; v < 4; ++v)
            r.v[v] = g0[4 * q + v] +
                     2 * ((u & 1) ? acc[u >> 1][4 * q + v].y : acc[u >> 1][4 * q + v].x);
          if (vec) {
            if (j < ns) *reinterpret_cast<Quad<T> *>(o + j) = r;
          } else {
#pragma unroll
            for (int v = 0; v < 4; ++v)
              if (j + v < ns) o[j + v] = r.v[v];
          }
        }
      }
    }
  }
}

// ---- local maxima -----------------------------------------------------------

template <typename T>
__device__ __forceinline__ bool before(T va, int ia, T vb, int ib) {
  return va > vb || (va == vb && ia < ib);
}

// Order keys for the maximum filter: a NaN in the window must win (its
// neighbours are no maxima) and -0 equals +0.  FP32 uses max.NaN; FP64 takes
// the doubles' order as 64-bit integers, because FP64 comparisons run at the
// FP64 rate.
__device__ __forceinline__ float key_of(float v) { return v; }
__device__ __forceinline__ long long key_of(double v) {
  long long x = __double_as_longlong(v);
  if ((x & 0x7fffffffffffffffLL) > 0x7ff0000000000000LL) return LLONG_MAX;
  if (x == LLONG_MIN) x = 0;
  return x < 0 ? x ^ 0x7fffffffffffffffLL : x;
}
__device__ __forceinline__ long long key_max(long long a, long long b) { return a > b ? a : b; }
__device__ __forceinline__ float key_max3(float a, float b, float c) {  // one instruction on sm_100+
  float d;
  asm("max.NaN.f32 %0, %1, %2, %3;" : "=f"(d) : "f"(a), "f"(b), "f"(c));
  return d;
}
__device__ __forceinline__ long long key_max3(long long a, long long b, long long c) {
  return key_max(key_max(a, b), c);
}
__device__ __forceinline__ void key_low(float &k) { k = -INFINITY; }
__device__ __forceinline__ void key_low(long long &k) { k = LLONG_MIN; }
__device__ __forceinline__ bool key_is(float v, float m) { return v == m; }
__device__ __forceinline__ bool key_is(long long v, long long m) { return v == m && v != LLONG_MAX; }
template <typename T> struct Key;
template <> struct Key<float> { typedef float type; };
template <> struct Key<double> { typedef long long type; };

// A warp's sorted best-P list, rank r in lane r (index INT_MAX: empty).
template <typename T> struct Best {
  T v;
  int i;
  // inserts (cv, ci), the same in every lane; false when it does not enter
  __device__ __forceinline__ bool insert(T cv, int ci, int lane, int P) {
    const bool first = lane < P && i != INT_MAX && before(v, i, cv, ci);
    const int pos = __popc(__ballot_sync(0xffffffffu, first));
    const T uv = __shfl_up_sync(0xffffffffu, v, 1);
    const int ui = __shfl_up_sync(0xffffffffu, i, 1);
    if (pos >= P) return false;
    if (lane > pos && lane < P) { v = uv; i = ui; }
    if (lane == pos) { v = cv; i = ci; }
    return true;
  }
};

constexpr int PEAK_THREADS = 256;
template <typename T> struct PeakRows { static constexpr int N = sizeof(T) == 4 ? 2 : 1; };

// P strongest local maxima of a materialised grid, one cluster of CTAs per
// particle.  A lane holds a quad of gammas of TI alpha rows and walks in beta:
// each step loads TI + 2 rows (two steps ahead), takes the
// 3-gamma maxima (the neighbour quads' edges by shuffles), the 3-row maxima, and
// compares the previous slice with the maximum over three slices.  A warp takes
// as many row blocks as its lanes hold whole rows (31 quads at 124 points per
// angle), or runs of 30 quads with a halo lane on each side; the steps are dealt
// to the cluster's warps in equal contiguous shares.  A point equal to its 3x3x3
// maximum takes the exact test against its 26 neighbours: it must precede each
// in the order (value desc, index asc), alpha and gamma wrapping and beta
// neighbours outside the grid skipped; NaN is never a maximum.  VEC: rows are
// whole 16-byte aligned quads; else quads are loaded by element, wrapping past
// the row's end (ns is even).
template <typename T, bool VEC>
__global__ void __launch_bounds__(PEAK_THREADS)
k_soft_peaks(const T *__restrict__ grid, int ns, int P_max, const int *__restrict__ P_per,
             int *__restrict__ idx_out, double *__restrict__ euler_out,
             double *__restrict__ score_out, int *__restrict__ n_cand_out) {
  typedef typename Key<T>::type K;
  constexpr int NW = PEAK_THREADS / 32, TI = PeakRows<T>::N;
  cg::cluster_group cl = cg::this_cluster();
  const int ctas = (int)cl.num_blocks(), rank = (int)cl.block_rank();
  const long b = blockIdx.x / ctas;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int n2 = ns * ns;
  const T *g = grid + b * (long)n2 * ns;
  __shared__ int cnt;
  __shared__ T lv[NW * 32], mv[32];
  __shared__ int li[NW * 32], mi[32];
  if (threadIdx.x == 0) cnt = 0;
  __syncthreads();
  Best<T> best{T(0), INT_MAX};
  int found = 0;
  int thi = INT_MAX;  // last entry of a full list
  T thv = T(0);
  const int nq = (ns + 3) / 4;
  const bool whole = nq <= 32;  // a row fits the warp
  const int rpw = whole ? 32 / nq : 1, njc = whole ? 1 : (nq + 29) / 30;
  const int nib = (ns + TI - 1) / TI, ncol = (nib + rpw - 1) / rpw * njc;
  const int sub = whole ? min(lane / nq, rpw - 1) : 0;
  const int left = whole ? (lane - sub * nq == 0 ? sub * nq + nq - 1 : lane - 1) : max(lane - 1, 0);
  const int right = whole ? (lane - sub * nq == nq - 1 ? sub * nq : lane + 1) : min(lane + 1, 31);
  K low;
  key_low(low);
  const long steps = (long)ncol * ns;
  const int share = warp * ctas + rank;
  long at = steps * share / (NW * ctas);
  const long end = steps * (share + 1) / (NW * ctas);
  while (at < end) {
    const int col = (int)(at / ns), ic = col / njc, jc = col - ic * njc;
    const int ka = (int)(at - (long)col * ns), kb = (int)min((long)ns, ka + (end - at));
    at += kb - ka;
    const int i0 = (ic * rpw + sub) * TI;
    const int q0 = whole ? lane - sub * nq : jc * 30 - 1 + lane;
    const bool out = whole ? lane < rpw * nq : lane >= 1 && lane <= 30 && q0 < nq;
    const int j0 = 4 * (q0 < 0 ? q0 + (VEC ? nq : 0) : (VEC ? q0 % nq : q0));
    int jo[4];  // wrapped gamma of each component
#pragma unroll
    for (int e = 0; e < 4; ++e) jo[e] = VEC ? j0 + e : (j0 + e + ns) % ns;
    const T *row[TI + 2];
#pragma unroll
    for (int q = 0; q < TI + 2; ++q) row[q] = g + (long)((i0 - 1 + q + ns) % ns) * n2;
    auto load = [&](int k, T (&nx)[TI + 2][4]) {
#pragma unroll
      for (int q = 0; q < TI + 2; ++q) {
        const T *r = row[q] + (long)k * ns;
        if (VEC) {
          const Quad<T> x = *reinterpret_cast<const Quad<T> *>(r + jo[0]);
#pragma unroll
          for (int e = 0; e < 4; ++e) nx[q][e] = x.v[e];
        } else {
#pragma unroll
          for (int e = 0; e < 4; ++e) nx[q][e] = r[jo[e]];
        }
      }
    };
    unsigned mask = out ? 0xffu : 0u;  // the lane's points, bit 4 * row + component
#pragma unroll
    for (int q = 0; q < TI; ++q)
      if (i0 + q >= ns) mask &= ~(15u << (4 * q));
    if (!VEC)
#pragma unroll
      for (int e = 0; e < 4; ++e)
        if (4 * q0 + e >= ns) mask &= ~(0x11u << e);
    const int ks = max(ka - 1, 0), ke = min(kb, ns - 1);  // slices loaded
    // Slice k (in nx, reloaded with slice k + 2): its 3 x 3 maxima, then the test
    // of slice k - 1 (values vc, maxima mc; those of slice k - 2 in mp), whose
    // place in mp the new maxima take.
    K vc[TI][4];
    auto step = [&](int k, T (&nx)[TI + 2][4], K (&mp)[TI][4], K (&mc)[TI][4]) {
      K vn[TI][4], mn[TI][4];  // (none past the grid)
      if (k <= ke) {
        K rm[TI + 2][4];
#pragma unroll
        for (int q = 0; q < TI + 2; ++q) {
          K x[4];
#pragma unroll
          for (int e = 0; e < 4; ++e) x[e] = key_of(nx[q][e]);
          K xl = __shfl_sync(0xffffffffu, x[3], left);
          const K xr = __shfl_sync(0xffffffffu, x[0], right);
          if (!VEC) {  // the last quad ends in the middle: column ns - 1 is component 1
            const K xe = __shfl_sync(0xffffffffu, x[1], left);
            if (whole && ns % 4 && q0 == 0) xl = xe;
          }
          rm[q][0] = key_max3(xl, x[0], x[1]);
          rm[q][1] = key_max3(x[0], x[1], x[2]);
          rm[q][2] = key_max3(x[1], x[2], x[3]);
          rm[q][3] = key_max3(x[2], x[3], xr);
          if (q >= 1 && q <= TI)
#pragma unroll
            for (int e = 0; e < 4; ++e) vn[q - 1][e] = x[e];
        }
        if (k + 1 < ke) load(k + 2, nx);
#pragma unroll
        for (int q = 0; q < TI; ++q)
#pragma unroll
          for (int e = 0; e < 4; ++e) mn[q][e] = key_max3(rm[q][e], rm[q + 1][e], rm[q + 2][e]);
      } else {
#pragma unroll
        for (int q = 0; q < TI; ++q)
#pragma unroll
          for (int e = 0; e < 4; ++e) vn[q][e] = mn[q][e] = low;
      }
      const int kc = k - 1;  // the slice tested
      bool any = false;
#pragma unroll
      for (int q = 0; q < TI; ++q)
#pragma unroll
        for (int e = 0; e < 4; ++e)
          any = any || key_is(vc[q][e], key_max3(mp[q][e], mc[q][e], mn[q][e]));
      if (__any_sync(0xffffffffu, any && kc >= ka && mask)) {
        unsigned is = 0;
#pragma unroll
        for (int q = 0; q < TI; ++q)
#pragma unroll
          for (int e = 0; e < 4; ++e)
            if (key_is(vc[q][e], key_max3(mp[q][e], mc[q][e], mn[q][e]))) is |= 1u << (4 * q + e);
        is &= mask;
        while (__any_sync(0xffffffffu, is)) {  // one point of each lane at a time
          bool ok = is != 0;
          const int bit = ok ? __ffs(is) - 1 : 0;
          is &= is - 1;
          const int i = i0 + (bit >> 2), j = jo[0] + (bit & 3), p = (i * ns + kc) * ns + j;
          T v = T(0);
          if (ok) v = g[p];
          // with a full list the count no longer matters, and a point that
          // does not precede the list's last entry needs no test
          if (thi != INT_MAX) ok = ok && before(v, p, thv, thi);
          if (ok) {
            // all neighbours of a row triple are loaded before any is compared
            for (int di = -1; di <= 1 && ok; ++di) {
              int ii = i + di;
              ii = ii < 0 ? ii + ns : (ii >= ns ? ii - ns : ii);
              T w[3][3];
              int wq[3][3];
#pragma unroll
              for (int dk = 0; dk < 3; ++dk)
#pragma unroll
                for (int dj = 0; dj < 3; ++dj) {
                  const int kk = min(max(kc + dk - 1, 0), ns - 1);
                  int jj = j + dj - 1;
                  jj = jj < 0 ? jj + ns : (jj >= ns ? jj - ns : jj);
                  wq[dk][dj] = (ii * ns + kk) * ns + jj;
                  w[dk][dj] = g[wq[dk][dj]];
                }
#pragma unroll
              for (int dk = 0; dk < 3; ++dk)
#pragma unroll
                for (int dj = 0; dj < 3; ++dj) {
                  const bool skip = kc + dk - 1 < 0 || kc + dk - 1 >= ns || wq[dk][dj] == p;
                  ok = ok && (skip || before(v, p, w[dk][dj], wq[dk][dj]));
                }
            }
          }
          found += ok;
          unsigned hit = __ballot_sync(0xffffffffu, ok);
          while (hit) {
            const int src = __ffs(hit) - 1;
            hit &= hit - 1;
            best.insert(__shfl_sync(0xffffffffu, v, src), __shfl_sync(0xffffffffu, p, src), lane,
                        P_max);
            thv = __shfl_sync(0xffffffffu, best.v, P_max - 1);
            thi = __shfl_sync(0xffffffffu, best.i, P_max - 1);
          }
        }
      }
#pragma unroll
      for (int q = 0; q < TI; ++q)
#pragma unroll
        for (int e = 0; e < 4; ++e) { mp[q][e] = mn[q][e]; vc[q][e] = vn[q][e]; }
    };
    T xa[TI + 2][4], xb[TI + 2][4];
    K ma[TI][4], mb[TI][4];
#pragma unroll
    for (int q = 0; q < TI; ++q)
#pragma unroll
      for (int e = 0; e < 4; ++e) ma[q][e] = mb[q][e] = vc[q][e] = low;
    load(ks, xa);
    if (ks < ke) load(ks + 1, xb);
    for (int k = ks; k <= kb; k += 2) {
      step(k, xa, ma, mb);
      if (k < kb) step(k + 1, xb, mb, ma);
    }
  }
  for (int o = 16; o > 0; o >>= 1) found += __shfl_xor_sync(0xffffffffu, found, o);
  if (lane == 0) atomicAdd(&cnt, found);
  lv[warp * 32 + lane] = best.v;
  li[warp * 32 + lane] = lane < P_max ? best.i : INT_MAX;
  __syncthreads();
  if (warp == 0) {  // the CTA's list; an entry that does not enter ends its list
    for (int w = 1; w < NW; ++w)
      for (int e = 0; e < P_max; ++e) {
        const int i = li[w * 32 + e];
        if (i == INT_MAX || !best.insert(lv[w * 32 + e], i, lane, P_max)) break;
      }
    mv[lane] = best.v;
    mi[lane] = best.i;
  }
  cl.sync();
  if (rank == 0 && warp == 0) {
    int n_max = cnt;
    for (int c = 1; c < ctas; ++c) {
      n_max += *cl.map_shared_rank(&cnt, c);
      const T *rv = cl.map_shared_rank(mv, c);
      const int *ri = cl.map_shared_rank(mi, c);
      const T tv = rv[lane];
      const int ti = ri[lane];
      for (int e = 0; e < P_max; ++e) {
        const T v = __shfl_sync(0xffffffffu, tv, e);
        const int i = __shfl_sync(0xffffffffu, ti, e);
        if (i == INT_MAX || !best.insert(v, i, lane, P_max)) break;
      }
    }
    const int Pb = max(P_per ? min(P_per[b], P_max) : P_max, 0), kept = min(Pb, n_max);
    if (lane < P_max) {
      const long o = b * P_max + lane;
      const bool has = lane < kept;
      const int i = has ? best.i : 0;
      const int ia = i / n2, kq = (i / ns) % ns, jg = i % ns;
      idx_out[o] = has ? i : -1;
      score_out[o] = has ? (double)best.v : __longlong_as_double(0x7ff8000000000000LL);
      euler_out[3 * o] = has ? 2.0 * M_PI * ia / ns : 0.0;
      euler_out[3 * o + 1] = has ? M_PI * (2.0 * kq + 1.0) / (2.0 * ns) : 0.0;
      euler_out[3 * o + 2] = has ? 2.0 * M_PI * jg / ns : 0.0;
    }
    if (lane == 0) n_cand_out[b] = kept;
  }
  cl.sync();  // the lists stay readable until rank 0 has merged them
}

template <typename T>
long slab_rows(const Plan &p, int KS) {  // alpha rows whose operand table fits (0: none)
  const long room = (sizeof(T) == 4 ? 112 : 226) * 1024, most = 226 * 1024;
  const int TI = Tile<T>::I, all = round_up(p.ns, TI);
  if ((long)sizeof(T) * slab_reals<T>(p.L0, p.ns, KS, all) <= room) return all;
  int IC = all;
  while (IC > TI && (long)sizeof(T) * slab_reals<T>(p.L0, p.ns, KS, IC) > most) IC = round_up(IC / 2, TI);
  return (long)sizeof(T) * slab_reals<T>(p.L0, p.ns, KS, IC) <= most ? IC : 0;
}

}  // namespace

template <typename T>
cudaError_t launch_soft_grid(const Plan &p, const T *c, int B, const int *P_per, T *grid, int *idx,
                             double *euler, double *score, int *n_cand, cudaStream_t st) {
  const int ng = (p.L0 + 1) * (p.L0 + 2) / 2;
  const bool vec = p.ns % 4 == 0 && reinterpret_cast<uintptr_t>(grid) % 16 == 0;
  const bool cvec = vec && reinterpret_cast<uintptr_t>(c) % 16 == 0;
  // beta slices per CTA: as many as give its threads one tile each, while the
  // batch still fills two CTAs on every SM and two fit an SM
  const int tiles = (round_up(p.ns, Tile<T>::I) / Tile<T>::I) * (round_up(p.ns, Tile<T>::J) / Tile<T>::J);
  int KS = std::max(1, 256 / tiles);
  while (KS > 1 && ((long)B * p.ns < 2L * p.sms * KS || slab_rows<T>(p, KS) < round_up(p.ns, Tile<T>::I))) --KS;
  const int IC = (int)slab_rows<T>(p, KS);
  if (IC == 0) return cudaErrorInvalidConfiguration;
  const size_t smem = sizeof(T) * slab_reals<T>(p.L0, p.ns, KS, IC);
  cudaError_t e = allow_smem(k_soft_slab<T>, smem);
  if (e != cudaSuccess) return e;
  (cvec ? k_soft_beta<T, true> : k_soft_beta<T, false>)
      <<<dim3((ng + BETA_GROUPS - 1) / BETA_GROUPS, (B + BETA_NB - 1) / BETA_NB), 128, 0, st>>>(
          c, p.nc, p.LJ, p.L0, p.ns, B, (const T *)p.soft_dT, grid);
  if ((e = cudaGetLastError()) != cudaSuccess) return e;
  k_soft_slab<T><<<dim3((p.ns + KS - 1) / KS, B), 256, smem, st>>>(p.L0, p.ns, KS, IC,
                                                                   (const T *)p.soft_tw, grid, vec);
  e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  // CTAs per particle: as many as the SMs take at two each
  cudaLaunchConfig_t cfg = {};
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = 8;
  while (at[0].val.clusterDim.x > 1 && (long)B * at[0].val.clusterDim.x > 2L * p.sms) at[0].val.clusterDim.x /= 2;
  at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
  cfg.gridDim = dim3(at[0].val.clusterDim.x * B);
  cfg.blockDim = dim3(PEAK_THREADS);
  cfg.stream = st;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, vec ? k_soft_peaks<T, true> : k_soft_peaks<T, false>,
                            (const T *)grid, p.ns, p.P, P_per, idx, euler, score, n_cand);
}
template cudaError_t launch_soft_grid<float>(const Plan &, const float *, int, const int *, float *,
                                             int *, double *, double *, int *, cudaStream_t);
template cudaError_t launch_soft_grid<double>(const Plan &, const double *, int, const int *, double *,
                                              int *, double *, double *, int *, cudaStream_t);

}  // namespace matcha
