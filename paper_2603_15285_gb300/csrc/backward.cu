// Gradient of the refined alignment score with respect to the template.
//
// Loss Lambda = sum_b w_b C_{L_J}(theta*_b): the refined score of each
// particle (Algorithm 1), weighted by the caller's w_b (the upstream
// gradient).  The template enters through c^l_{mn} = sum_s w_s f_lm
// conj(h_ln) (Eq. sigmalmm); the refined rotation theta* moves with it so
// that grad C stays zero, and the implicit function theorem turns that into
// a shift of the evaluation point (Section 2.2 gives grad and Hessian):
//
//   dLambda_b/dh = d/dh Re sum c^l_{mn} E'^l_{mn},   v = H^{-1} grad C (held fixed),
//   E'^l_{mn} = exp(i(m a + n g)) [ d^l_{mn}(b) (1 - i(m v_a + n v_g)) - v_b d'^l_{mn}(b) ].
//
// Four kernels, Wigner d recomputed by the l-recurrence (nothing stored
// from the forward pass):
//   k_bwd_point  one CTA per particle: C, grad, Hessian at theta* from c, and
//                v = H^{-1} grad (FP64 solve);
//   k_bwd_coef   one CTA per particle and range of shells: per degree l, E'^l (rows m = -l..l,
//                columns n = 0..l) into shared memory, then
//                X_ln(s) = w_b w_s sum_m f_lm(r_s) E'^l_{mn}, doubled for
//                n > 0 (the stored h_ln also drives h_{l,-n} = (-1)^n
//                conj(h_ln), and that term equals X_ln);
//   k_bwd_reduce sums X over the particles that share one template;
//   k_bwd_synth  one CTA per (template, shell, range of rings): the transpose of the shell
//                analysis (Legendre sum, then the phi series at the
//                samples) and of the trilinear sampling (FP64 atomic adds
//                into the voxel gradient), on the forward pass's own
//                sample coordinates.
#include <math.h>
#include <string.h>
#include <type_traits>
#include "internal.cuh"

namespace matcha {
namespace {

constexpr int BWD_THREADS = 256;

// first (group, l) entry of group (m, j) in the grouped layout:
// sum_{m' < m} (m'+1)(L-m'+1) + j (L-m+1)
// (32-bit: the bandwidths whose state fits in shared memory are below 128)
__device__ __forceinline__ int goff_dev(int m, int j, int L) {
  const unsigned u = m, t = u * (u + 1);
  return (int)((L + 2) * (t / 2) - t * (2 * u + 1) / 6) + j * (L - m + 1);
}

// cos and sin of b and b / 2 for the block: one sincos for a warp (each costs dozens
// of FP64 instructions, and FP64 runs at 1/64 of the FP32 rate).
template <typename T>
__device__ __forceinline__ void beta_trig(double be, T (&t)[4]) {
  __shared__ T tr[4];
  if (threadIdx.x < 2) {
    double sd, cd;
    sincos(threadIdx.x ? 0.5 * be : be, &sd, &cd);
    tr[2 * threadIdx.x] = (T)cd;
    tr[2 * threadIdx.x + 1] = (T)sd;
  }
  __syncthreads();
#pragma unroll
  for (int i = 0; i < 4; ++i) t[i] = tr[i];
}

// Powers x^k, k = 0 .. n - 1, by repeated products, of x = ch (thread 0) and sh (a
// thread of another warp); a loop per seed serialised a whole warp, at each degree.
constexpr int pw_len(int L) { return 2 * L + 3; }
template <typename T>
__device__ __forceinline__ void power_tables(T *chp, T *shp, int n, T ch, T sh) {
  if (threadIdx.x != 0 && threadIdx.x != 32) return;
  T *o = threadIdx.x ? shp : chp;
  const T x = threadIdx.x ? sh : ch;
  T r = T(1);
  for (int i = 0; i < n; ++i) {
    o[i] = r;
    r *= x;
  }
}
// x^k from the table, and 0 for k < 0 (those terms carry a zero integer factor)
template <typename T> __device__ __forceinline__ T pw(const T *t, int k) { return k < 0 ? T(0) : t[k]; }

// d^m_{mn}(b) and its first two b-derivatives at the seed degree l = m:
// sigma K ch^a sh^c with a = m + n, c = m - n, sigma = (-1)^c, ch = cos(b/2),
// sh = sin(b/2); d/db (ch^a sh^c) = (c ch^{a+1} sh^{c-1} - a ch^{a-1} sh^{c+1}) / 2.
template <typename T>
__device__ __forceinline__ void seed3(int m, int n, T K, const T *ch, const T *sh, T &d, T &d1, T &d2) {
  const int a = m + n, c = m - n;
  const T g = (c & 1) ? -K : K;
  d = g * pw(ch, a) * pw(sh, c);
  d1 = g * T(0.5) * (T(c) * pw(ch, a + 1) * pw(sh, c - 1) - T(a) * pw(ch, a - 1) * pw(sh, c + 1));
  d2 = g * T(0.25) *
       (T(c * (c - 1)) * pw(ch, a + 2) * pw(sh, c - 2) -
        T(c * (a + 1) + a * (c + 1)) * pw(ch, a) * pw(sh, c) +
        T(a * (a - 1)) * pw(ch, a - 2) * pw(sh, c + 2));
}

// Adds one image (u, v) with weight W of the sums S0 = sum c d, S1 = sum c d',
// S2 = sum c d'' (complex) to (C, C_a, C_b, C_g, C_aa, C_ab, C_ag, C_bb, C_bg,
// C_gg): the phase exp(i(u a + v g)) brings i u under d/da and i v under d/dg.
__device__ __forceinline__ void add_img(double (&acc)[10], double W, double u, double v, double er,
                                        double ei, double s0r, double s0i, double s1r, double s1i,
                                        double s2r, double s2i) {
  const double zr0 = s0r * er - s0i * ei, zi0 = __fma_rn(s0i, er, __dmul_rn(s0r, ei));
  const double zr1 = s1r * er - s1i * ei, zi1 = __fma_rn(s1i, er, __dmul_rn(s1r, ei));
  const double zr2 = s2r * er - s2i * ei;
  acc[0] += W * zr0;
  acc[1] -= W * u * zi0;
  acc[2] += W * zr1;
  acc[3] -= W * v * zi0;
  acc[4] -= W * u * u * zr0;
  acc[5] -= W * u * zi1;
  acc[6] -= W * u * v * zr0;
  acc[7] += W * zr2;
  acc[8] -= W * v * zi1;
  acc[9] -= W * v * v * zr0;
}

// 3x3 solve H v = g by Gaussian elimination with partial pivoting; false
// (v = 0) when a pivot falls below 1e-14 ||H||_F.
__device__ bool solve3(const double *H, const double *g, double *v) {
  double A[3][4], nf = 0.0;
  for (int i = 0; i < 3; ++i) {
    for (int j = 0; j < 3; ++j) {
      A[i][j] = H[3 * i + j];
      nf += H[3 * i + j] * H[3 * i + j];
    }
    A[i][3] = g[i];
  }
  nf = sqrt(nf);
  for (int k = 0; k < 3; ++k) {
    int piv = k;
    for (int i = k + 1; i < 3; ++i)
      if (fabs(A[i][k]) > fabs(A[piv][k])) piv = i;
    if (!(fabs(A[piv][k]) > 1e-14 * nf)) {
      v[0] = v[1] = v[2] = 0.0;
      return false;
    }
    if (piv != k)
      for (int j = 0; j < 4; ++j) {
        const double t = A[k][j];
        A[k][j] = A[piv][j];
        A[piv][j] = t;
      }
    for (int i = k + 1; i < 3; ++i) {
      const double f = A[i][k] / A[k][k];
      for (int j = k; j < 4; ++j) A[i][j] -= f * A[k][j];
    }
  }
  for (int k = 2; k >= 0; --k) {
    double s = A[k][3];
    for (int j = k + 1; j < 3; ++j) s -= A[k][j] * v[j];
    v[k] = s / A[k][k];
  }
  return true;
}

// An 8-real record of the grouped layout; VEC: 16-byte loads (p 16-byte aligned).
template <bool VEC, typename T>
__device__ __forceinline__ void load8(const T *p, T (&v)[8]) {
  if constexpr (VEC) {
    constexpr int W = 16 / sizeof(T);
#pragma unroll
    for (int i = 0; i < 8; i += W) {
      const uint4 q = __ldg(reinterpret_cast<const uint4 *>(p + i));
      memcpy(v + i, &q, 16);
    }
  } else {
#pragma unroll
    for (int i = 0; i < 8; ++i) v[i] = __ldg(p + i);
  }
}

// C, grad, Hessian of C_{L} at theta*_b from the grouped coefficients, then
// shift[b] = (v, C) with v = H^{-1} grad; flags[b] bit 4 when H is singular.
//
// A thread takes the two pairs (m, n) of a group along their l-recurrence, a record
// of c and one of the coefficients per degree, the next ones in flight.  Bound by the
// FP64 pipe (64 cycles of a quarter SM per warp and operation): a sincos and about
// thirty operations per image.  At a refined rotation grad C is a cancelled sum whose
// last bits carry over into v, so the phases, the order of the sums and the tree of the
// reduction are part of the result; the tree is evaluated by all threads from shared
// memory, not as 50 shuffled additions in every warp.  512 particles, L_J = 32, FP32:
// 318 -> 198 us (the pipe alone: about 170).
template <typename T, bool VEC>
__global__ void __launch_bounds__(BWD_THREADS)
    k_bwd_point(const T *__restrict__ c, long cper, const T *__restrict__ rcoef,
                const T *__restrict__ seedK, int L, const double *__restrict__ euler,
                double *__restrict__ shift, int *__restrict__ flags) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  double *red = reinterpret_cast<double *>(smem_raw);  // [10][BWD_THREADS]
  T *chp = reinterpret_cast<T *>(red + 10 * BWD_THREADS), *shp = chp + pw_len(L);
  const long b = blockIdx.x;
  const T *cb = c + b * cper;
  const double al = euler[3 * b], be = euler[3 * b + 1], ga = euler[3 * b + 2];
  T trig[4];
  beta_trig(be, trig);
  const T x = trig[0], s = trig[1], ch = trig[2], sh = trig[3];
  power_tables(chp, shp, pw_len(L), ch, sh);
  __syncthreads();
  double acc[10];
#pragma unroll
  for (int i = 0; i < 10; ++i) acc[i] = 0.0;
  const int ng = (L + 1) * (L + 2) / 2;
  for (int g = threadIdx.x; g < ng; g += blockDim.x) {
    const int m = tri_floor(g), j = g - m * (m + 1) / 2;
    const int e0 = goff_dev(m, j, L);
    T d[2], d1[2], d2[2], p0[2] = {0, 0}, p1[2] = {0, 0}, p2[2] = {0, 0};
    T s0r[2] = {0, 0}, s0i[2] = {0, 0}, s1r[2] = {0, 0}, s1i[2] = {0, 0}, s2r[2] = {0, 0},
      s2i[2] = {0, 0};  // c_mn sums
    T t0r[2] = {0, 0}, t0i[2] = {0, 0}, t1r[2] = {0, 0}, t1i[2] = {0, 0}, t2r[2] = {0, 0},
      t2i[2] = {0, 0};  // c_nm sums
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      d[h] = d1[h] = d2[h] = T(0);
      if (h == 0 || j < m) seed3<T>(m, 2 * j - m + h, seedK[4L * g + h], chp, shp, d[h], d1[h], d2[h]);
    }
    const T *cp = cb + 8L * e0, *rp = rcoef + 8L * e0;
    T cn[8], rn[8];
    load8<VEC>(cp, cn);
    if (m < L) load8<VEC>(rp, rn);
    for (int l = m; l <= L; ++l) {
      T ce[8], re[8];
#pragma unroll
      for (int i = 0; i < 8; ++i) { ce[i] = cn[i]; re[i] = rn[i]; }
      if (l < L) load8<VEC>(cp + 8 * (l + 1 - m), cn);
      if (l + 1 < L) load8<VEC>(rp + 8 * (l + 1 - m), rn);
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const T cr = ce[h], ci = ce[2 + h], dr = ce[4 + h], di = ce[6 + h];
        s0r[h] += cr * d[h]; s0i[h] += ci * d[h]; s1r[h] += cr * d1[h];
        s1i[h] += ci * d1[h]; s2r[h] += cr * d2[h]; s2i[h] += ci * d2[h];
        t0r[h] += dr * d[h]; t0i[h] += di * d[h]; t1r[h] += dr * d1[h];
        t1i[h] += di * d1[h]; t2r[h] += dr * d2[h]; t2i[h] += di * d2[h];
        if (l < L) {  // d^{l+1} = (a x - b) d^l - e d^{l-1}, differentiated in b
          const T A = re[h], NB = re[2 + h], NE = re[4 + h];
          const T t = A * x + NB;
          const T n0 = t * d[h] + NE * p0[h];
          const T n1 = t * d1[h] - A * s * d[h] + NE * p1[h];
          const T n2 = t * d2[h] - T(2) * A * s * d1[h] - A * x * d[h] + NE * p2[h];
          p0[h] = d[h]; p1[h] = d1[h]; p2[h] = d2[h];
          d[h] = n0; d1[h] = n1; d2[h] = n2;
        }
      }
    }
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const int n = 2 * j - m + h;
      if (n > m) break;
      double sn, cn;
      // image (m, n), weight 1 for (0, 0) else 2 (with its conjugate (-m, -n))
      sincos(m * al + n * ga, &sn, &cn);
      add_img(acc, (m == 0 && n == 0) ? 1.0 : 2.0, m, n, cn, sn, s0r[h], s0i[h], s1r[h], s1i[h], s2r[h],
              s2i[h]);
      // image (n, m): d^l_nm = (-1)^{m-n} d^l_mn; absent for n = +-m
      if (n != m && n != -m) {
        sincos(n * al + m * ga, &sn, &cn);
        add_img(acc, ((m - n) & 1) ? -2.0 : 2.0, n, m, cn, sn, t0r[h], t0i[h], t1r[h], t1i[h], t2r[h],
                t2i[h]);
      }
    }
  }
  // a warp's 32 terms as the tree (i, i + 16), (i, i + 8), ..., then the warps in order
#pragma unroll
  for (int i = 0; i < 10; ++i) red[i * BWD_THREADS + threadIdx.x] = acc[i];
  for (int o = 16; o > 0; o >>= 1) {
    __syncthreads();
    for (int t = threadIdx.x; t < 10 * (BWD_THREADS / 32) * o; t += BWD_THREADS) {
      double *x = red + t / o * 32 + t % o;
      x[0] += x[o];
    }
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    double r[10];
    for (int i = 0; i < 10; ++i) {
      r[i] = 0.0;
      for (int w = 0; w < BWD_THREADS / 32; ++w) r[i] += red[i * BWD_THREADS + 32 * w];
    }
    const double grad[3] = {r[1], r[2], r[3]};
    const double H[9] = {r[4], r[5], r[6], r[5], r[7], r[8], r[6], r[8], r[9]};
    double v[3];
    const bool ok = solve3(H, grad, v);
    shift[4 * b] = v[0];
    shift[4 * b + 1] = v[1];
    shift[4 * b + 2] = v[2];
    shift[4 * b + 3] = r[0];
    if (flags) flags[b] = ok ? 0 : 16;
  }
}

// Shared memory of k_bwd_coef, in reals: recurrence state [4][(L+1)^2], E' rows
// [2L+1] of column pairs, phase tables [4][2L+1], powers, two scales per shell and two
// buffers of a degree's coefficients of the shells.
__host__ __device__ __forceinline__ int bwd_cols(int L) { return (L + 2) & ~1; }
__host__ __device__ __forceinline__ long bwd_coef_reals(int L, int shells) {
  return 4L * (L + 1) * (L + 1) + 2L * (2 * L + 1) * bwd_cols(L) + 4L * (2 * L + 1) + 2L * pw_len(L) +
         2L * shells + 2 + 4L * shells * (L + 1);
}

// products that the compiler may not fuse
__device__ __forceinline__ float mul_rn(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ double mul_rn(double a, double b) { return __dmul_rn(a, b); }

// pairs of columns: packed in FP32
__device__ __forceinline__ float2 p_mul(float a, float2 b) { return __fmul2_rn(make_float2(a, a), b); }
__device__ __forceinline__ float2 p_fma(float a, float2 b, float2 c) { return __ffma2_rn(make_float2(a, a), b, c); }
__device__ __forceinline__ float2 p_add(float2 a, float2 b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ double2 p_mul(double a, double2 b) { return make_double2(a * b.x, a * b.y); }
__device__ __forceinline__ double2 p_fma(double a, double2 b, double2 c) {
  return make_double2(fma(a, b.x, c.x), fma(a, b.y, c.y));
}
__device__ __forceinline__ double2 p_add(double2 a, double2 b) {
  return make_double2(__dadd_rn(a.x, b.x), __dadd_rn(a.y, b.y));
}
template <typename T> struct PairOf;
template <> struct PairOf<float> { typedef float2 type; };
template <> struct PairOf<double> { typedef double2 type; };

__device__ __forceinline__ void ld_pairs(const float *p, float2 &a, float2 &b) {
  const float4 q = *reinterpret_cast<const float4 *>(p);
  a = make_float2(q.x, q.y);
  b = make_float2(q.z, q.w);
}
__device__ __forceinline__ void ld_pairs(const double *p, double2 &a, double2 &b) {
  a = *reinterpret_cast<const double2 *>(p);
  b = *reinterpret_cast<const double2 *>(p + 2);
}

// A real into shared memory, asynchronously.
template <typename T>
__device__ __forceinline__ void stage_real(T *dst, const T *src) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], %2;" ::"r"((unsigned)__cvta_generic_to_shared(dst)),
               "l"(src), "n"(sizeof(T)) : "memory");
}

// A thread's tile of the product is TS shells x two columns n: per row m (and -m)
// one 16-byte load of E' and one of each shell's coefficient serve 4 TS packed
// multiply-adds, in the order of m.  The products of a term are fused once and rounded
// before they are added; which of the two is fused follows the sign of a row's term.
// Bound by issue (57% of the slots; two barriers per degree): 512 particles of 32
// shells, L_J = 32, FP32: 468 -> 252 us (4 shells per tile 262, 1 shell slower still).
// Before, an output's coefficients and E' were read once per product, and the seeds'
// power loops and a trigonometric function per thread held the block at every degree.
// FP64: one shell, since a tile of few lanes holds a quarter SM as long as a full warp
// (140 particles of 12 shells, L_J = 16: 54 tiles of two shells on two of the four
// quarters; with one 196 us, 253 as one output per thread).
template <typename T> constexpr int BWD_TS = sizeof(T) == 8 ? 1 : 2;
template <typename T>
__global__ void __launch_bounds__(BWD_THREADS, sizeof(T) == 4 ? 4 : 3)
    k_bwd_coef(const T *__restrict__ f, int S, int Sc, int L, const double *__restrict__ wrad,
               const T *__restrict__ rcoef, const T *__restrict__ seedK,
               const double *__restrict__ euler, const double *__restrict__ shift,
               const double *__restrict__ weight, T *__restrict__ X) {
  typedef typename PairOf<T>::type P2;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const long b = blockIdx.x;
  const int s0 = blockIdx.y * Sc, ns = min(Sc, S - s0);
  const int np = (L + 1) * (L + 1), nlm = (L + 1) * (L + 2) / 2, R2 = 2 * L + 1, LN = bwd_cols(L);
  // [m + L][n / 2]: re, re, im, im; rows m < 0 times (-1)^m
  T *Es = reinterpret_cast<T *>(smem_raw);
  T *dc = Es + 2L * R2 * LN;  // d^l
  T *dp = dc + np;            // d^{l-1}
  T *d1c = dp + np;           // d'^l
  T *d1p = d1c + np;          // d'^{l-1}
  T *pa = d1p + np;           // cos, sin (k a), k = -L..L
  T *pg = pa + 2 * R2;        // cos, sin (k g)
  T *sc = pg + 2 * R2;        // w_b w_s, 2 w_b w_s
  T *chp = sc + 2 * Sc;       // powers of cos(b/2), sin(b/2)
  T *shp = chp + pw_len(L);
  // an even number of reals before the coefficient pairs
  T *fs = Es + (2L * R2 * LN + 4L * np + 4L * R2 + 2L * Sc + 2L * pw_len(L) + 1) / 2 * 2;
  const double al = euler[3 * b], be = euler[3 * b + 1], ga = euler[3 * b + 2];
  const T va = (T)shift[4 * b], vb = (T)shift[4 * b + 1], vg = (T)shift[4 * b + 2];
  const double wb = weight ? weight[b] : 1.0;
  T trig[4];
  beta_trig(be, trig);
  const T x = trig[0], s = trig[1], ch = trig[2], sh = trig[3];
  for (int k = threadIdx.x; k < 2 * (L + 1); k += blockDim.x) {  // and of -k: the conjugates
    const int q = k <= L ? k : k - L - 1;
    T *o = (k <= L ? pa : pg) + 2 * L;
    double sd, cd;
    sincos(q * (k <= L ? al : ga), &sd, &cd);
    o[2 * q] = o[-2 * q] = (T)cd;
    o[2 * q + 1] = (T)sd;
    if (q) o[-2 * q + 1] = (T)-sd;
  }
  for (int k = threadIdx.x; k < ns; k += blockDim.x) {
    sc[2 * k] = (T)(wb * wrad[s0 + k] * 1.0);
    sc[2 * k + 1] = (T)(wb * wrad[s0 + k] * 2.0);
  }
  power_tables(chp, shp, pw_len(L), ch, sh);
  const T *fb = f + 2L * (b * S + s0) * nlm;
  T *Xb = X + 2L * (b * S + s0) * nlm;
  // degree l of every shell into buffer l & 1
  auto stage = [&](int l) {
    T *buf = fs + (l & 1) * 2 * Sc * (L + 1);
    const int run = 2 * (l + 1);
    const FastDiv dr(run);
    for (int t = threadIdx.x; t < ns * run; t += blockDim.x) {
      const int q = dr.div(t), i = t - q * run;
      stage_real(buf + q * 2 * (L + 1) + i, fb + 2L * ((long)q * nlm + l * (l + 1) / 2) + i);
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
  };
  stage(0);
  __syncthreads();
  for (int l = 0; l <= L; ++l) {
    // 1. d^l, d'^l of every pair (m, n), m = isqrt(q), n = q - m^2 - m, with
    //    m <= l; then E' of its images with a non-negative second index
    for (int q = threadIdx.x; q < (l + 1) * (l + 1); q += blockDim.x) {
      const int m = isqrt_floor(q), n = q - m * m - m;
      const int j = (n + m) >> 1, h = (n + m) & 1;
      T d, d1;
      if (m == l) {
        T d2;
        seed3<T>(m, n, seedK[4L * (m * (m + 1) / 2 + j) + h], chp, shp, d, d1, d2);
        dp[q] = T(0); d1p[q] = T(0);
      } else {  // step l-1 -> l with the coefficients of entry (group, l-1)
        const T *re = rcoef + 8L * (goff_dev(m, j, L) + (l - 1) - m) + h;
        const T A = re[0], NB = re[2], NE = re[4];
        const T t = A * x + NB, od = dc[q], od1 = d1c[q];
        d = t * od + NE * dp[q];
        d1 = t * od1 - A * s * od + NE * d1p[q];
        dp[q] = od; d1p[q] = od1;
      }
      dc[q] = d; d1c[q] = d1;
      // images (u, w) with w >= 0 and d^l_uw = sg d^l_mn: (n, m) sg (-1)^{m-n}; (m, n)
      // sg 1 for n >= 0; (-m, -n) sg (-1)^{m-n} for n <= 0
      const T sgm = ((m - n) & 1) ? T(-1) : T(1), tm = T(m), tn = T(n);
      auto image = [&](int u, int w, T tu, T tw, T sg0) {
        const T sg = u < 0 && (u & 1) ? -sg0 : sg0;
        const T dd = sg * d, dd1 = sg * d1;
        // exp(i(u a + w g)) [dd - vb dd1 - i (u va + w vg) dd]
        const T ar = pa[2 * (u + L)], ai = pa[2 * (u + L) + 1];
        const T gr = pg[2 * (w + L)], gi = pg[2 * (w + L) + 1];
        const T er = ar * gr - ai * gi, ei = ar * gi + ai * gr;
        const T br = dd - vb * dd1, bi = -fma(tw, vg, mul_rn(tu, va)) * dd;
        T *o = Es + 2 * ((u + L) * LN + (w & ~1)) + (w & 1);
        o[0] = er * br - ei * bi;
        o[2] = er * bi + ei * br;
      };
      image(n, m, tn, tm, sgm);
      if (n < 0) image(-m, -n, -tm, -tn, sgm);
      else image(m, n, tm, tn, T(1));
      if (n == 0 && m > 0) image(-m, 0, -tm, T(0), sgm);
    }
    asm volatile("cp.async.wait_all;" ::: "memory");
    __syncthreads();
    if (l < L) stage(l + 1);
    // 2. X_ln(s) = w_b w_s (2 if n > 0) sum_{m=-l..l} f_lm(r_s) E'_mn, with
    //    f_{l,-m} = (-1)^m conj(f_lm) (the sign is in the rows of E')
    const int lm0 = l * (l + 1) / 2, nn = (l + 2) / 2;
    const FastDiv dn(nn);
    for (int o = threadIdx.x; o < (ns + BWD_TS<T> - 1) / BWD_TS<T> * nn; o += blockDim.x) {
      const int st = dn.div(o), n = 2 * (o - st * nn);
      const T *fq[BWD_TS<T>];
#pragma unroll
      for (int u = 0; u < BWD_TS<T>; ++u) {
        const int sidx = min(BWD_TS<T> * st + u, ns - 1);
        fq[u] = fs + (l & 1) * 2 * Sc * (L + 1) + sidx * 2 * (L + 1);
      }
      const T *ep = Es + 2 * (L * LN + n);
      P2 xr[BWD_TS<T>], xi[BWD_TS<T>];
#pragma unroll
      for (int u = 0; u < BWD_TS<T>; ++u) xr[u].x = xr[u].y = xi[u].x = xi[u].y = T(0);
      auto rows = [&](int m, auto kind) {  // rows m and -m; kind 0: m = 0, else m's parity
        constexpr int KIND = decltype(kind)::value;
        P2 e0, e1, g0, g1, ne1, ng0;
        ld_pairs(ep + 2 * m * LN, e0, e1);
        ne1.x = -e1.x; ne1.y = -e1.y;
        if (KIND) {
          ld_pairs(ep - 2 * m * LN, g0, g1);
          ng0.x = -g0.x; ng0.y = -g0.y;
        }
#pragma unroll
        for (int u = 0; u < BWD_TS<T>; ++u) {
          const P2 v = *reinterpret_cast<const P2 *>(fq[u] + 2 * m);
          const T fr = v.x, fi = v.y;
          xr[u] = p_add(xr[u], p_fma(fr, e0, p_mul(fi, ne1)));
          xi[u] = p_add(xi[u], p_fma(fr, e1, p_mul(fi, e0)));
          if (KIND) {
            xr[u] = p_add(xr[u], p_fma(fr, g0, p_mul(fi, g1)));
            xi[u] = p_add(xi[u], KIND == 1 ? p_fma(fi, ng0, p_mul(fr, g1)) : p_fma(fr, g1, p_mul(fi, ng0)));
          }
        }
      };
      rows(0, std::integral_constant<int, 0>{});
      for (int m = 1; m <= l; m += 2) {
        rows(m, std::integral_constant<int, 1>{});
        if (m < l) rows(m + 1, std::integral_constant<int, 2>{});
      }
#pragma unroll
      for (int u = 0; u < BWD_TS<T>; ++u) {
        const int sidx = BWD_TS<T> * st + u;
        if (sidx >= ns) break;
        T *xo = Xb + 2L * ((long)sidx * nlm + lm0 + n);
        const T q0 = sc[2 * sidx + (n > 0)], q1 = sc[2 * sidx + 1];
        xo[0] = q0 * xr[u].x;
        xo[1] = q0 * xi[u].x;
        if (n + 1 <= l) {
          xo[2] = q1 * xr[u].y;
          xo[3] = q1 * xi[u].y;
        }
      }
    }
    __syncthreads();
  }
}

// G[s][lm] = sum_b X[b][s][lm] (FP64 sums, fixed order).  A CTA takes RED_X elements
// and RED_Y interleaved runs of b, RED_K particles at a time.  FP32: these are summed
// as an unevaluated sum of three FP32 values (Knuth's two-sum: v enters s, the exact
// rounding error of that enters e, and that one's enters r), which then enter the FP64
// sum.  Only the additions into r round: with M the sum of the block's magnitudes, e is
// below 15 2^-24 M and r below 120 2^-48 M, so less than 2^-61 M is lost, where FP64
// additions of the 16 lose up to 15 2^-53 M.  FP64 conversions and additions, which
// bound the plain loop, are three sixteenths.  512 x 35,904 values: 83 us as FP64
// additions, 24 here (reading them: 11).
constexpr int RED_X = 32, RED_Y = 8, RED_K = 16;
// s + v into s; returns its rounding error, exact
__device__ __forceinline__ float two_sum(float &s, float v) {
  const float t = __fadd_rn(s, v), z = __fadd_rn(t, -s);
  const float err = __fadd_rn(__fadd_rn(s, -__fadd_rn(t, -z)), __fadd_rn(v, -z));
  s = t;
  return err;
}
template <typename T>
__global__ void __launch_bounds__(RED_X *RED_Y)
    k_bwd_reduce(const T *__restrict__ X, int B, long per, T *__restrict__ G) {
  __shared__ double red[RED_Y][RED_X];
  const long i = (long)blockIdx.x * RED_X + threadIdx.x;
  double acc = 0.0;
  if (i < per)
    for (int b0 = RED_K * threadIdx.y; b0 < B; b0 += RED_K * RED_Y) {
      T v[RED_K];
#pragma unroll
      for (int k = 0; k < RED_K; ++k) v[k] = b0 + k < B ? X[(long)(b0 + k) * per + i] : T(0);
      if constexpr (sizeof(T) == 4) {
        float s = v[0], e = 0.f, r = 0.f;
#pragma unroll
        for (int k = 1; k < RED_K; ++k) r = __fadd_rn(r, two_sum(e, two_sum(s, v[k])));
        if (isfinite(s)) {
          acc += (double)s;
          acc += (double)e;
          acc += (double)r;
          continue;
        }
      }
#pragma unroll
      for (int k = 0; k < RED_K; ++k) acc += (double)v[k];
    }
  red[threadIdx.y][threadIdx.x] = acc;
  __syncthreads();
  if (threadIdx.y || i >= per) return;
#pragma unroll
  for (int k = 1; k < RED_Y; ++k) acc += red[k][threadIdx.x];
  G[i] = (T)acc;
}

// Transpose of the analysis of one shell s of template t: the sample
// gradient du(j, k) = Re sum_m A_m(j) exp(i m phi_k) with
// A_m(j) = sum_l ptab[j][lm] G_lm(r_s), ptab = w_j (2 pi / n_phi) Pbar_lm(x_j),
// then the transpose of the trilinear sampling at the forward pass's own
// coordinates (same clamping of the corner), by FP64 atomic adds.  A CTA takes JB
// rings of the shell: with one template, a CTA per shell left 120 SMs idle (32 shells
// of 33 rings: 52 -> 30 us, now latency of the ring sums and the atomics).
template <typename T>
__global__ void __launch_bounds__(BWD_THREADS)
    k_bwd_synth(const T *__restrict__ G, int S, int L, int N, int JB, const T *__restrict__ ptab,
                const T *__restrict__ phi_cs, const T *__restrict__ ring, double *__restrict__ vox) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int sidx = blockIdx.x;
  const long t = blockIdx.y;
  const int nt = L + 1, nph = 2 * L + 2, nlm = (L + 1) * (L + 2) / 2;
  const int jb = blockIdx.z * JB, nj = min(JB, nt - jb);
  T *A = reinterpret_cast<T *>(smem_raw);  // [JB][L+1][2]
  T *cs = A + 2 * JB * (L + 1);             // [nph][2]
  const T *Gs = G + 2L * (t * S + sidx) * nlm;
  for (int k = threadIdx.x; k < 2 * nph; k += blockDim.x) cs[k] = phi_cs[k];
  for (int it = threadIdx.x; it < nj * (L + 1); it += blockDim.x) {
    const int j = it / (L + 1), m = it - j * (L + 1);
    T ar = 0, ai = 0;
#pragma unroll 8
    for (int l = m; l <= L; ++l) {
      const int lm = l * (l + 1) / 2 + m;
      const T p = ptab[(long)(jb + j) * nlm + lm];
      ar += p * Gs[2 * lm];
      ai += p * Gs[2 * lm + 1];
    }
    A[2 * it] = ar;
    A[2 * it + 1] = ai;
  }
  __syncthreads();
  const T c0 = (T)(0.5 * N), hi = (T)(N - 1);
  const long NN = (long)N * N;
  double *vt = vox + t * NN * N;
  for (int it = threadIdx.x; it < nj * nph; it += blockDim.x) {
    const int j = it / nph, k = it - j * nph;
    T du = 0;
    int mk = 0;  // m k mod n_phi
    for (int m = 0; m <= L; ++m) {
      du += A[2 * (j * (L + 1) + m)] * cs[2 * mk] - A[2 * (j * (L + 1) + m) + 1] * cs[2 * mk + 1];
      mk += k;
      if (mk >= nph) mk -= nph;
    }
    const T rho = ring[2 * ((long)sidx * nt + jb + j)], pz = ring[2 * ((long)sidx * nt + jb + j) + 1];
    const T px = c0 + rho * cs[2 * k], py = c0 + rho * cs[2 * k + 1];
    const T fx = floor(px), fy = floor(py), fz = floor(pz);
    const bool inside = px >= T(0) && py >= T(0) && pz >= T(0) && px <= hi && py <= hi && pz <= hi;
    int i0, j0, k0;
    T tx, ty, tz;
    if (inside) {
      i0 = min((int)fx, N - 2); j0 = min((int)fy, N - 2); k0 = min((int)fz, N - 2);
      tx = px - (T)i0; ty = py - (T)j0; tz = pz - (T)k0;
    } else {
      i0 = (int)fx; j0 = (int)fy; k0 = (int)fz;
      tx = px - fx; ty = py - fy; tz = pz - fz;
    }
    for (int dz = 0; dz < 2; ++dz)
      for (int dy = 0; dy < 2; ++dy)
        for (int dx = 0; dx < 2; ++dx) {
          const int ii = i0 + dx, jj = j0 + dy, kk = k0 + dz;
          if (ii < 0 || jj < 0 || kk < 0 || ii >= N || jj >= N || kk >= N) continue;
          const T w = (dx ? tx : T(1) - tx) * (dy ? ty : T(1) - ty) * (dz ? tz : T(1) - tz);
          atomicAdd(vt + (long)kk * NN + (long)jj * N + ii, (double)w * (double)du);
        }
  }
}

}  // namespace

// one shell per CTA at least
size_t bwd_coef_smem(const Plan &p) { return (p.fp64 ? 8 : 4) * (size_t)bwd_coef_reals(p.LJ, 1); }
bool backward_fits(const Plan &p) { return bwd_coef_smem(p) <= 227 * 1024; }

template <typename T>
cudaError_t launch_template_grad(const Plan &p, const T *f, const T *c, int B, int tstride,
                                 const double *euler, const double *weight, T *X, T *coef_grad,
                                 double *vox_grad, double *shift, int *flags, cudaStream_t st) {
  if (B == 0) return cudaSuccess;
  const long per = 2L * p.S * p.nlm;
  const bool vec = (uintptr_t)c % 16 == 0;
  const size_t ps = sizeof(double) * 10 * BWD_THREADS + 2 * sizeof(T) * pw_len(p.LJ);
  auto point = vec ? k_bwd_point<T, true> : k_bwd_point<T, false>;
  // Shells per CTA: each CTA repeats the recurrence, so the shells are split, evenly,
  // only as far as all CTAs run at once: one on an SM in FP64, whose pipe it fills, two
  // in FP32 where they fit (twice the CTAs of the chip, whatever the type, cost FP64 130
  // particles of 24 shells, L_J = 40, 7.51 ms against 2.99 in one part, 76 particles 3.92
  // against 2.18 in two; FP32 130, L_J = 64, 1.93 against 0.90); more parts where the
  // coefficients do not fit.
  const size_t most = SMEM_MOST / sizeof(T) - 4;
  auto shells = [&](long parts) { return (int)(((p.S + parts - 1) / parts + BWD_TS<T> - 1) / BWD_TS<T> * BWD_TS<T>); };
  auto at_once = [&](long parts) {
    const size_t bytes = sizeof(T) * (size_t)bwd_coef_reals(p.LJ, shells(parts)) + 2048;
    return p.sms * (sizeof(T) == 4 && 2 * bytes <= 228 * 1024 ? 2L : 1L);
  };
  long parts = 1;
  while (parts * BWD_TS<T> < p.S && (size_t)bwd_coef_reals(p.LJ, shells(parts)) > most) ++parts;
  while (2 * parts * BWD_TS<T> <= p.S && 2 * parts * B <= at_once(2 * parts)) parts *= 2;
  int Sc = shells(parts);
  while (Sc > 1 && (size_t)bwd_coef_reals(p.LJ, Sc) > most) --Sc;
  const size_t smem = sizeof(T) * (size_t)bwd_coef_reals(p.LJ, Sc);
  cudaError_t e = allow_smem(k_bwd_coef<T>, smem, 4 * sizeof(T));
  if (e != cudaSuccess) return e;
  T *Xo = tstride ? coef_grad : X;
  point<<<B, BWD_THREADS, ps, st>>>(c, 4L * p.nc, (const T *)p.rcoef, (const T *)p.seedK, p.LJ, euler,
                                    shift, flags);
  if ((e = cudaGetLastError()) != cudaSuccess) return e;
  k_bwd_coef<T><<<dim3(B, (p.S + Sc - 1) / Sc), BWD_THREADS, smem, st>>>(
      f, p.S, Sc, p.LJ, p.wrad, (const T *)p.rcoef, (const T *)p.seedK, euler, shift, weight, Xo);
  if ((e = cudaGetLastError()) != cudaSuccess) return e;
  const int ntmpl = tstride ? B : 1;
  if (!tstride)
    k_bwd_reduce<T><<<(int)((per + RED_X - 1) / RED_X), dim3(RED_X, RED_Y), 0, st>>>(X, B, per, coef_grad);
  if ((e = cudaGetLastError()) != cudaSuccess) return e;
  if (vox_grad) {
    const long nv = (long)p.N * p.N * p.N * ntmpl;
    e = cudaMemsetAsync(vox_grad, 0, sizeof(double) * nv, st);
    if (e != cudaSuccess) return e;
    // rings per CTA: a shell's, or few enough that there are four CTAs per SM
    const int nt = p.LJ + 1, want = (int)(4L * p.sms / ((long)p.S * ntmpl) + 1);
    const int JB = (nt + want - 1) / want;
    const size_t ss = sizeof(T) * (2 * (size_t)JB * nt + 2 * (size_t)(2 * p.LJ + 2));
    if ((e = allow_smem(k_bwd_synth<T>, ss)) != cudaSuccess) return e;
    k_bwd_synth<T><<<dim3(p.S, ntmpl, (nt + JB - 1) / JB), BWD_THREADS, ss, st>>>(
        coef_grad, p.S, p.LJ, p.N, JB, (const T *)p.ptab, (const T *)p.phi_cs, (const T *)p.ring, vox_grad);
  }
  return cudaGetLastError();
}

template cudaError_t launch_template_grad<float>(const Plan &, const float *, const float *, int,
                                                 int, const double *, const double *, float *,
                                                 float *, double *, double *, int *, cudaStream_t);
template cudaError_t launch_template_grad<double>(const Plan &, const double *, const double *, int,
                                                  int, const double *, const double *, double *,
                                                  double *, double *, double *, int *, cudaStream_t);

}  // namespace matcha
