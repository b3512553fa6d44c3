// Pieces shared by the refinement kernels (newton.cu: a CTA per particle;
// newton_spread.cu: a cluster of CTAs per particle): paired arithmetic, shared
// loads, the rescaled seeds, one recurrence step, the Newton step rule.
#pragma once
#include <math.h>
#include "internal.cuh"

namespace matcha {
namespace {

enum { ST_RUN = 0, ST_TRIAL = 1, ST_STOP = 2, ST_DEAD = 3 };

template <typename T>
__device__ __forceinline__ T ipow_t(T x, int e) {
  T r = T(1);
  while (e) {
    if (e & 1) r *= x;
    x *= x;
    e >>= 1;
  }
  return r;
}

template <typename T> __device__ __forceinline__ T tcos(T x);
template <typename T> __device__ __forceinline__ T tsin(T x);
template <> __device__ __forceinline__ float tcos<float>(float x) { return cosf(x); }
template <> __device__ __forceinline__ float tsin<float>(float x) { return sinf(x); }
template <> __device__ __forceinline__ double tcos<double>(double x) { return cos(x); }
template <> __device__ __forceinline__ double tsin<double>(double x) { return sin(x); }

// Asynchronous global -> shared copies (no registers involved).
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;\n" ::); }
template <int N> __device__ __forceinline__ void cp_async_wait() {
  asm volatile("cp.async.wait_group %0;\n" ::"n"(N));
}

// Shared-memory addressing: the hot loops address shared memory through
// 32-bit shared-window addresses and ld.shared, so every load is a shared
// load with 32-bit address arithmetic.
__device__ __forceinline__ unsigned smem_u32(const void *p) {
  return (unsigned)__cvta_generic_to_shared(p);
}
__device__ __forceinline__ void lds1(unsigned a, float &x) {
  asm volatile("ld.shared.f32 %0, [%1];\n" : "=f"(x) : "r"(a));
}
__device__ __forceinline__ void lds1(unsigned a, double &x) {
  asm volatile("ld.shared.f64 %0, [%1];\n" : "=d"(x) : "r"(a));
}
__device__ __forceinline__ void lds2(unsigned a, float2 &v) {
  asm volatile("ld.shared.v2.f32 {%0, %1}, [%2];\n" : "=f"(v.x), "=f"(v.y) : "r"(a));
}
__device__ __forceinline__ void lds2(unsigned a, double2 &v) {
  asm volatile("ld.shared.v2.f64 {%0, %1}, [%2];\n" : "=d"(v.x), "=d"(v.y) : "r"(a));
}
// two pairs: 16 bytes in FP32 (one vector load), 32 bytes in FP64
__device__ __forceinline__ void lds4(unsigned a, float2 &lo, float2 &hi) {
  asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];\n"
               : "=f"(lo.x), "=f"(lo.y), "=f"(hi.x), "=f"(hi.y)
               : "r"(a));
}
__device__ __forceinline__ void lds4(unsigned a, double2 &lo, double2 &hi) {
  lds2(a, lo);
  lds2(a + 16, hi);
}

// Two-wide values: the two halves of a partner group (pairs (m, n) and
// (m, n+1)) advance together.  FP32 uses the packed FP32x2 instructions of the
// sm_100 family (one FFMA2 does both halves); FP64 issues two scalar FMAs.
template <typename T> struct Vec2;
template <> struct Vec2<float> { using type = float2; };
template <> struct Vec2<double> { using type = double2; };
template <typename T> using v2 = typename Vec2<T>::type;

__device__ __forceinline__ float2 vfma(float2 a, float2 b, float2 c) { return __ffma2_rn(a, b, c); }
__device__ __forceinline__ float2 vmul(float2 a, float2 b) { return __fmul2_rn(a, b); }
__device__ __forceinline__ float2 vadd(float2 a, float2 b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ double2 vfma(double2 a, double2 b, double2 c) {
  return make_double2(fma(a.x, b.x, c.x), fma(a.y, b.y, c.y));
}
__device__ __forceinline__ double2 vmul(double2 a, double2 b) {
  return make_double2(a.x * b.x, a.y * b.y);
}
__device__ __forceinline__ double2 vadd(double2 a, double2 b) {
  return make_double2(a.x + b.x, a.y + b.y);
}
template <typename T> __device__ __forceinline__ v2<T> vset(T x, T y);
template <> __device__ __forceinline__ float2 vset<float>(float x, float y) { return make_float2(x, y); }
template <> __device__ __forceinline__ double2 vset<double>(double x, double y) {
  return make_double2(x, y);
}
template <typename T> __device__ __forceinline__ v2<T> vld(unsigned a0, unsigned a1) {
  T x, y;
  lds1(a0, x);
  lds1(a1, y);
  return vset<T>(x, y);
}

// Per-candidate tables, candidate index fastest with an odd stride
// cand_stride(P) >= P, so the lanes of a sub-slot (one candidate each) read
// distinct banks.  Power table: two rows (cos(b/2)^k, sin(b/2)^k), each
// PW_PAD zeros followed by k = 0 .. 2 L_J + 3.  Phase table: four rows
// (cos k a, sin k a, cos k g, sin k g) for k = -L_J .. L_J + 1 (index k + L_J).
// Element (row r, position k, candidate p) is at (r * row_len + k) * stride + p.
constexpr int PW_PAD = 4;
__host__ __device__ __forceinline__ int pw_row(int LJ) { return PW_PAD + 2 * LJ + 4; }
__host__ __device__ __forceinline__ int ph_row(int LJ) { return 2 * LJ + 2; }
__host__ __device__ __forceinline__ int cand_stride(int P) { return P | 1; }

// 2^e as a float for -126 <= e <= 127, 0 below (values that small times a
// state below 2^32 are far under FP32 resolution of any sum they enter).
__device__ __forceinline__ float pow2f(int e) {
  return e < -126 ? 0.f : __int_as_float((min(e, 127) + 127) << 23);
}

// Extended-range power x^k = mant 2^expo (mant in [0.5, 1), or 0 for x = 0,
// k > 0) by binary powering with the exponent carried as an integer, so
// that powers far below the FP32 range keep their leading bits.
__device__ __forceinline__ void xpow(float x, int k, float &mant, int &expo) {
  int ex;
  float xm = frexpf(x, &ex);
  float rm = 1.f;
  int re = 0;
  while (k) {
    if (k & 1) {
      int t;
      rm = frexpf(rm * xm, &t);
      re += ex + t;
    }
    k >>= 1;
    if (k) {
      int t;
      xm = frexpf(xm * xm, &t);
      ex = 2 * ex + t;
    }
  }
  if (rm == 0.f) re = 0;
  int t;
  mant = frexpf(rm, &t);
  expo = re + t;
}

// Seeds of the rescaled recurrence (32-bit plans above L_J = 64).  The
// powers come as (mantissa, exponent) from the extended-range tables: pc,
// ps address ch^aa and sh^ba, pe is the byte offset of the exponent rows.
// The states D0, D1, D2 of half h are the true seeds divided by 2^E_h,
// E_h = the exponent of K ch^a sh^b, so the state of d starts near 1 however
// small the true seed is; D1 and D2 keep their ratio to D0.
template <bool FULL>
__device__ __forceinline__ void group_seed_rs(unsigned pc, unsigned ps, unsigned pe, unsigned z,
                                              v2<float> K, int aa, int ba, v2<float> &D0,
                                              v2<float> &D1, v2<float> &D2, int &E0, int &E1) {
  auto ldm = [&](unsigned a, float &m, int &e) {
    float ef;
    lds1(a, m);
    lds1(a + pe, ef);
    e = (int)ef;
  };
  float c0, c1, s0, sm1;
  int ec0, ec1, es0, esm1;
  ldm(pc, c0, ec0); ldm(pc + z, c1, ec1);
  ldm(ps, s0, es0); ldm(ps - z, sm1, esm1);
  int kex, key;
  const float kmx = frexpf(K.x, &kex), kmy = frexpf(K.y, &key);
  const int R0 = ec0 + es0, R1 = ec1 + esm1;  // reference exponents of ch^a sh^b
  E0 = kex + R0;
  E1 = key + R1;
  const float g0 = kmx, g1 = -kmy;            // sigma K of both halves, mantissas
  D0 = vset<float>(g0 * c0 * s0, g1 * c1 * sm1);
  if (FULL) {
    float c2, c3, cm1, cm2, s1, s2, sm2, sm3;
    int ec2, ec3, ecm1, ecm2, es1, es2, esm2, esm3;
    ldm(pc + 2 * z, c2, ec2); ldm(pc + 3 * z, c3, ec3);
    ldm(pc - z, cm1, ecm1); ldm(pc - 2 * z, cm2, ecm2);
    ldm(ps + z, s1, es1); ldm(ps + 2 * z, s2, es2);
    ldm(ps - 2 * z, sm2, esm2); ldm(ps - 3 * z, sm3, esm3);
    // ch^i sh^j relative to 2^R
    auto rel = [](float cm, int ce, float sm, int se, int R) { return cm * sm * pow2f(ce + se - R); };
    const float fa = (float)aa, fb = (float)ba;
    // half 0: a = aa, b = ba; half 1: a = aa + 1, b = ba - 1
    const float t1a = fb * rel(c1, ec1, sm1, esm1, R0), t2a = fa * rel(cm1, ecm1, s1, es1, R0);
    const float t1b = (fb - 1.f) * rel(c2, ec2, sm2, esm2, R1), t2b = (fa + 1.f) * rel(c0, ec0, s0, es0, R1);
    D1 = vset<float>(0.5f * g0 * (t1a - t2a), 0.5f * g1 * (t1b - t2b));
    const float A0 = fa, B0 = fb, A1 = fa + 1.f, B1 = fb - 1.f;
    const float u1a = B0 * (B0 - 1.f) * rel(c2, ec2, sm2, esm2, R0);
    const float u2a = (B0 * (A0 + 1.f) + A0 * (B0 + 1.f)) * rel(c0, ec0, s0, es0, R0);
    const float u3a = A0 * (A0 - 1.f) * rel(cm2, ecm2, s2, es2, R0);
    const float u1b = B1 * (B1 - 1.f) * rel(c3, ec3, sm3, esm3, R1);
    const float u2b = (B1 * (A1 + 1.f) + A1 * (B1 + 1.f)) * rel(c1, ec1, sm1, esm1, R1);
    const float u3b = A1 * (A1 - 1.f) * rel(cm1, ecm1, s1, es1, R1);
    D2 = vset<float>(0.25f * g0 * (u1a + u3a - u2a), 0.25f * g1 * (u1b + u3b - u2b));
  }
}

// One staged degree entry of a partner group: c of both halves, the
// recurrence coefficients (a, -b, -e) of the step to the next degree, and
// -l(l+1) of the entry's own degree l.
template <typename T> struct Coef {
  v2<T> CR, CI, DR, DI;
};
template <typename T> struct Rec {
  v2<T> A, NB, NE, NL;
};

// Z += c d (and c d', c d'' when FULL) for one entry; with ODE the third
// sums take -l(l+1) c d (passed as D2 = -l(l+1) d) instead of c d''.
template <typename T, bool FULL>
__device__ __forceinline__ void accumulate(const Coef<T> &e, const v2<T> &D0, const v2<T> &D1,
                                           const v2<T> &D2, v2<T> (&Z)[12]) {
  Z[0] = vfma(e.CR, D0, Z[0]); Z[1] = vfma(e.CI, D0, Z[1]);
  Z[2] = vfma(e.DR, D0, Z[2]); Z[3] = vfma(e.DI, D0, Z[3]);
  if (FULL) {
    Z[4] = vfma(e.CR, D1, Z[4]); Z[5] = vfma(e.CI, D1, Z[5]);
    Z[6] = vfma(e.DR, D1, Z[6]); Z[7] = vfma(e.DI, D1, Z[7]);
    Z[8] = vfma(e.CR, D2, Z[8]); Z[9] = vfma(e.CI, D2, Z[9]);
    Z[10] = vfma(e.DR, D2, Z[10]); Z[11] = vfma(e.DI, D2, Z[11]);
  }
}
// One recurrence step from (d^l, d^{l-1}) = (D, P); d^{l+1} overwrites P:
//   d^{l+1} = t d - e p,  t = a x - b,
//   d'^{l+1} = t d' - a s d - e p',  d''^{l+1} = t d'' - 2 a s d' - a x d - e p''.
template <typename T, bool FULL, bool ODE = false>
__device__ __forceinline__ void step_into(const Rec<T> &r, v2<T> X, v2<T> NS, v2<T> NX,
                                          const v2<T> &D0, const v2<T> &D1, const v2<T> &D2,
                                          v2<T> &P0, v2<T> &P1, v2<T> &P2) {
  const v2<T> t = vfma(r.A, X, r.NB);
  P0 = vfma(t, D0, vmul(r.NE, P0));
  if (FULL && ODE) {
    const v2<T> nAs = vmul(r.A, NS);
    P1 = vfma(t, D1, vfma(nAs, D0, vmul(r.NE, P1)));
  } else if (FULL) {
    const v2<T> nAs = vmul(r.A, NS);
    P1 = vfma(t, D1, vfma(nAs, D0, vmul(r.NE, P1)));
    const v2<T> nAx = vmul(r.A, NX);
    P2 = vfma(t, D2, vfma(vadd(nAs, nAs), D1, vfma(nAx, D0, vmul(r.NE, P2))));
  }
}

// x mod 2 pi in [0, 2 pi).  The refinement only meets |x| < 4 pi (a wrapped
// angle plus a clamped step, or plus pi after a reflection of beta), where a
// few compare-and-add steps give the same result as x - 2 pi floor(x / 2 pi)
// without a double-precision division; other inputs take that formula first.
__device__ __forceinline__ double mod2pi_d(double x) {
  const double t = 2.0 * M_PI;
  if (!(x < 4.0 * t && x >= -4.0 * t)) x -= t * floor(x / t);
  for (int k = 0; k < 4 && x >= t; ++k) x -= t;
  for (int k = 0; k < 4 && x < 0.0; ++k) x += t;
  return x;
}

__device__ __forceinline__ void wrap_d(double *v) {
  double a = v[0], b = v[1], g = v[2];
  if (b < 0) { b = -b; a += M_PI; g += M_PI; }
  else if (b > M_PI) { b = 2.0 * M_PI - b; a += M_PI; g += M_PI; }
  v[0] = mod2pi_d(a); v[1] = b; v[2] = mod2pi_d(g);
}

// Newton direction from grad g and Hessian H (row-major 3x3) in the solve
// precision S; returns flag bits.  A Cholesky pivot of -H counts as positive
// above piv_rel ||H||_F, set by the precision H was summed in (1e-12 for FP64
// sums, 1e-6 for FP32 sums: above the rounding level of H's entries).
template <typename S>
__device__ __forceinline__ int newton_dir(const S *g, const S *H, int L, S *d, double piv_rel,
                                          bool grad) {
  S hn = 0;
#pragma unroll
  for (int i = 0; i < 9; ++i) hn += H[i] * H[i];
  hn = sqrt(hn);
  const S tol = S(piv_rel) * hn;
  // Cholesky of A = -H
  S a00 = -H[0], a10 = -H[3], a20 = -H[6], a11 = -H[4], a21 = -H[7], a22 = -H[8];
  bool ok = !grad && a00 > tol;  // grad: the gradient method, never the Newton step
  S L00 = 0, L10 = 0, L20 = 0, L11 = 0, L21 = 0, L22 = 0;
  if (ok) {
    L00 = sqrt(a00); L10 = a10 / L00; L20 = a20 / L00;
    S p11 = a11 - L10 * L10;
    ok = p11 > tol;
    if (ok) {
      L11 = sqrt(p11); L21 = (a21 - L20 * L10) / L11;
      S p22 = a22 - L20 * L20 - L21 * L21;
      ok = p22 > tol;
      if (ok) L22 = sqrt(p22);
    }
  }
  int fl = 0;
  if (ok) {
    S y0 = g[0] / L00;
    S y1 = (g[1] - L10 * y0) / L11;
    S y2 = (g[2] - L20 * y0 - L21 * y1) / L22;
    S x2 = y2 / L22;
    S x1 = (y1 - L21 * x2) / L11;
    S x0 = (y0 - L10 * x1 - L20 * x2) / L00;
    d[0] = x0; d[1] = x1; d[2] = x2;
  } else {
    fl = grad ? 0 : 2;
#pragma unroll
    for (int i = 0; i < 3; ++i) d[i] = hn > 0 ? g[i] / hn : S(0);
  }
  S nrm = sqrt(d[0] * d[0] + d[1] * d[1] + d[2] * d[2]);
  S cap = S(M_PI / (2.0 * (L + 1.0)));
  if (nrm > cap) {
    S f = cap / nrm;
#pragma unroll
    for (int i = 0; i < 3; ++i) d[i] *= f;
  }
  return fl;
}

// sm: pointers to the CTA's per-candidate state (th, tr, del, Cc, res, state,
// tries, fl).  Candidate tid has C, grad, H of its current point in res: record C, stop on
// a non-finite value (flag bit 0), take the Newton direction (solved in
// precision S), stop the level when the increment is below step_tol, else
// prepare the first trial (angles in FP64).
template <typename S, typename State>
__device__ __forceinline__ void start_step(int tid, int L, double step_tol, bool grad, const State &sm,
                                           double piv_rel) {
  const double *r = sm.res + 10 * tid;
  const double C = r[0];
  const S g[3] = {S(r[1]), S(r[2]), S(r[3])};
  const S H[9] = {S(r[4]), S(r[5]), S(r[6]), S(r[5]), S(r[7]), S(r[8]), S(r[6]), S(r[8]), S(r[9])};
  bool fin = true;
#pragma unroll
  for (int i = 0; i < 10; ++i) fin = fin && isfinite(r[i]);
  sm.Cc[tid] = C;
  if (!fin) {
    sm.fl[tid] |= 1;
    sm.state[tid] = ST_DEAD;
    return;
  }
  S d[3];
  sm.fl[tid] |= newton_dir<S>(g, H, L, d, piv_rel, grad);
  if (sqrt(d[0] * d[0] + d[1] * d[1] + d[2] * d[2]) < S(step_tol)) {
    sm.state[tid] = ST_STOP;
    return;
  }
  double tr[3] = {sm.th[3 * tid] + (double)d[0], sm.th[3 * tid + 1] + (double)d[1],
                  sm.th[3 * tid + 2] + (double)d[2]};
  wrap_d(tr);
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    sm.del[3 * tid + i] = (double)d[i];
    sm.tr[3 * tid + i] = tr[i];
  }
  sm.tries[tid] = 0;
  sm.state[tid] = ST_TRIAL;
}

// Candidate tid has been evaluated at its point (start: a level's start point) or
// trial point: accepts or halves the step, and prepares the next trial.  last:
// the plan's final level, whose 3x3 solves run in FP64.
template <typename T, typename State>
__device__ __forceinline__ void after_evaluation(int tid, int L, bool start, bool last, int M,
                                                 double step_tol, double acc_tol, bool grad,
                                                 const State &sm, double piv_rel) {
  const double Ct = sm.res[10 * tid];
  if (start) {
    sm.steps[tid] = 0;
  } else if (Ct >= sm.Cc[tid] - acc_tol * fabs(sm.Cc[tid])) {
    for (int i = 0; i < 3; ++i) sm.th[3 * tid + i] = sm.tr[3 * tid + i];
    sm.Cc[tid] = Ct;
    if (sm.steps[tid] >= M - 1) {
      sm.state[tid] = ST_STOP;
      return;
    }
    ++sm.steps[tid];  // derivatives at the accepted point
  } else if (++sm.tries[tid] == 3) {
    sm.fl[tid] |= 4;
    sm.state[tid] = ST_STOP;  // a repeated step from the same point rejects again
    return;
  } else {
    double tr[3];
    for (int i = 0; i < 3; ++i) {
      sm.del[3 * tid + i] *= 0.5;
      tr[i] = sm.th[3 * tid + i] + sm.del[3 * tid + i];
    }
    wrap_d(tr);
    for (int i = 0; i < 3; ++i) sm.tr[3 * tid + i] = tr[i];
    return;
  }
  if (last) start_step<double>(tid, L, step_tol, grad, sm, piv_rel);
  else start_step<T>(tid, L, step_tol, grad, sm, piv_rel);
}

}  // namespace
}  // namespace matcha
