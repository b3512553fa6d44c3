// Step a6: frequency-marched Newton refinement (Sections 2.2-2.4, Algorithm 1)
// and step a7: the final argmax over candidates.
//
// C_L(a,b,g) = Re sum_{l<=L} sum_{m,n} c^l_{mn} e^{i(m a + n g)} d^l_{mn}(b),
// grad and Hessian in (a, b, g): d/da brings i m, d/dg brings i n, d/db acts
// on d^l (Appendix A.4).  Every evaluation runs the three-term l-recurrence
// of d and d' for each order pair (m, n) with m >= |n|; the second
// derivative comes from the differential equation of the Wigner functions,
//   d'' = -cot(b) d' + ((m^2 + n^2 - 2mn cos b) / sin^2 b - l(l+1)) d,
// applied to the sums over l (the plans with the rescaled 32-bit recurrence
// above L_J = 64 run a third recurrence for d'' instead).  It uses
//   d^l_{nm} = (-1)^{m-n} d^l_{mn}            (transposed image),
//   term(-m,-n) = conj(term(m,n))              (real volumes),
// so one recurrence serves the four orders (m,n), (n,m), (-m,-n), (-n,-m).
//
// Work layout (32-bit plans that fill the SMs, and the cost-sorted queue; others are
// spread further, newton_spread.cu): one CTA per particle holds all P candidates.  A warp is split
// into sub-slots of `cpw` lanes (cpw = P rounded up to a power of two); lane
// p of a sub-slot follows candidate p.  A sub-slot walks partner groups (the
// two order pairs (m, n), (m, n+1) of one m, stored interleaved), and each
// lane advances both pairs of a group with paired (FP32x2 / 2 x FP64)
// operations: c^l, the recurrence coefficients and the recurrence state are
// pairs over the two partners, so no packed operand is a broadcast pair.  The
// entries are staged in shared memory with cp.async, in batches of up to four
// consecutive groups of the sub-slot.  Per-lane partial sums are reduced in a fixed order (the two
// halves, shuffles across sub-slots, then warps in index order), all in the
// plan's working precision and converted to FP64 at the end, so results do
// not depend on scheduling.
//
// Step rule (the paper gives only the plain update theta - H^{-1} grad):
//   delta = -H^{-1} grad when -H is positive definite (Cholesky pivots
//   > 1e-12 ||H||_F for FP64 sums, > 1e-6 ||H||_F for FP32 sums), else
//   grad / ||H||_F (flag bit 1); ||delta|| clamped to pi / (2 (L+1)); the
//   level ends early when ||delta|| < step_tol (Section 2.4); trial
//   theta' = wrap(theta + delta) is accepted when
//   C(theta') >= C(theta) - acc_tol |C(theta)| (acc_tol above the rounding
//   level of the sums), else delta is halved (at most twice); three
//   rejected trials end the level for that candidate (flag bit 2), since a
//   repeated step from the same point would reject again.  Angles, the
//   acceptance test and the scores are FP64 in every plan; the 3x3 solve is
//   FP64 on the final level and in the plan's precision (FP32 for the 32-bit
//   plans) on the earlier levels.
#include <algorithm>
#include "newton_common.cuh"

namespace matcha {

constexpr int NEWTON_THREADS = 256;
constexpr int NEWTON_WARPS = NEWTON_THREADS / 32;

struct NewtonArgs {
  int LJ, nlev, M, P, cpw, nslots;
  int grad;  // 1: gradient steps grad / ||H||_F instead of Newton steps
  int Ls[MATCHA_MAX_LEVELS];
  double tol, acc_tol;
  long nc;
};

struct SmemLayout {
  double *th, *tr, *del, *Cc, *res;
  void *red;  // [warps][P][10] working precision
  int *state, *steps, *tries, *fl;
  void *ea, *pw, *stage;
};

__device__ __forceinline__ void cp_async16s(unsigned sa, const void *gmem) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 16;\n" ::"r"(sa), "l"(gmem));
}
struct Group {
  int m, na, off;  // order, first partner's n, offset in (group, l) entries
};
// The groups of a sub-slot come in increasing g: the order m and the offset
// of the first group of m advance with g instead of being solved for.
struct GroupWalk {
  int m = 0, tri = 0, base = 0;  // tri = m(m+1)/2, base = offset of group (m, 0)
  __device__ __forceinline__ Group at(int g, int LJ) {
    while (g >= tri + m + 1) {
      base += (m + 1) * (LJ - m + 1);
      tri += m + 1;
      ++m;
    }
    const int j = g - tri;
    return {m, 2 * j - m, base + j * (LJ - m + 1)};
  }
};

// Staging buffer of one sub-slot, per half (double buffering), in reals: a
// header (below), then per degree entry 16 reals: the 8 c reals of the group
// entry, then its 8 recurrence reals (a_a, a_b, -b_a, -b_b, -e_a, -e_b,
// -l(l+1), -l(l+1)); L_J + 1 entries.
// Batched staging: a half buffer takes a run of up to STAGE_BATCH consecutive
// groups of its sub-slot whose entries fit in L_J + 1 entries; its header
// holds 8 reals per group: (K_a, K_b, 0, 0) from the seed table, then (m,
// n_a, first entry) written by the sub-slot's first lane, then one pad.
constexpr int STAGE_BATCH = 4;
constexpr int STAGE_HDR = 8 * STAGE_BATCH;  // reals
__host__ __device__ __forceinline__ int stage_half(int LJ) { return STAGE_HDR + 16 * (LJ + 1); }

// Seeds at l = m of both halves: d = sigma K ch^a sh^b with a = m+n,
// b = m-n, sigma = (-1)^b; with FULL also d' and d'' (Appendix A.4 applied to
// the closed form: d/db (ch^a sh^b) = (b ch^{a+1} sh^{b-1} - a ch^{a-1} sh^{b+1})/2).
// The first half has a = aa, b = ba (both even, so sigma = +1); the second
// a = aa + 1, b = ba - 1 (sigma = -1).  pc, ps: shared addresses of ch^aa,
// sh^ba in the padded power tables; a term whose integer coefficient is zero
// may read a zero pad, so it adds exactly 0.  z: bytes between consecutive
// powers in the table.
template <typename T, bool FULL, bool ODE = false>
__device__ __forceinline__ void group_seed(unsigned pc, unsigned ps, unsigned z, v2<T> K, int aa,
                                           int ba, v2<T> &D0, v2<T> &D1, v2<T> &D2) {
  T c0, c1, s0, sm1;
  lds1(pc, c0); lds1(pc + z, c1);
  lds1(ps, s0); lds1(ps - z, sm1);
  const v2<T> mone = vset<T>(T(-1), T(-1));
  const v2<T> GK = vmul(K, vset<T>(T(1), T(-1)));
  const v2<T> pp0 = vmul(vset<T>(c0, c1), vset<T>(s0, sm1));  // ch^a sh^b
  D0 = vmul(GK, pp0);
  if (FULL) {
    T c2, c3, cm1, cm2, s1, s2, sm2, sm3;
    lds1(pc + 2 * z, c2); lds1(pc + 3 * z, c3); lds1(pc - z, cm1); lds1(pc - 2 * z, cm2);
    lds1(ps + z, s1); lds1(ps + 2 * z, s2); lds1(ps - 2 * z, sm2); lds1(ps - 3 * z, sm3);
    const T fa = T(aa), fb = T(ba);
    const v2<T> A = vset<T>(fa, fa + T(1)), B = vset<T>(fb, fb - T(1));
    const v2<T> one = vset<T>(T(1), T(1));
    const v2<T> t1 = vmul(B, vmul(vset<T>(c1, c2), vset<T>(sm1, sm2)));
    const v2<T> t2 = vmul(A, vmul(vset<T>(cm1, c0), vset<T>(s1, s0)));
    D1 = vmul(vmul(GK, vset<T>(T(0.5), T(0.5))), vfma(t2, mone, t1));
    if (ODE) return;  // d'' comes from the differential equation
    // b(b-1) ch^{a+2} sh^{b-2} - (b(a+1) + a(b+1)) ch^a sh^b + a(a-1) ch^{a-2} sh^{b+2}
    const v2<T> u1 = vmul(vmul(B, vadd(B, mone)), vmul(vset<T>(c2, c3), vset<T>(sm2, sm3)));
    const v2<T> u2 = vmul(vfma(B, vadd(A, one), vmul(A, vadd(B, one))), pp0);
    const v2<T> u3 = vmul(vmul(A, vadd(A, mone)), vmul(vset<T>(cm2, cm1), vset<T>(s2, s1)));
    D2 = vmul(vmul(GK, vset<T>(T(0.25), T(0.25))), vfma(u2, mone, vadd(u1, u3)));
  }
}

// Entries interleaved: 8 c reals, then 8 recurrence reals.
template <typename T> __device__ __forceinline__ void load_coef(unsigned a, Coef<T> &e) {
  lds4(a, e.CR, e.CI);
  lds4(a + 4 * sizeof(T), e.DR, e.DI);
}
template <typename T> __device__ __forceinline__ void load_rec(unsigned a, Rec<T> &r) {
  lds4(a + 8 * sizeof(T), r.A, r.NB);
  lds4(a + 12 * sizeof(T), r.NE, r.NL);
}
// Sums over l = m..m+last of one partner group for one candidate: Z[0..3] =
// sum d (Re c_mn, Im c_mn, Re c_nm, Im c_nm), then the same with d' (Z[4..7])
// and d'' (Z[8..11]) when FULL; each a pair over the two halves.  With ODE
// the second-derivative recurrence is not run: Z[8..11] gets -l(l+1) d in
// place of d'' (the caller completes it with the differential equation).
// a: shared address of the group's first staged entry (16 reals per entry).
// The loop takes two degrees per trip with the roles of (D, P) swapped in the
// second; c is loaded one degree ahead of its use, the step coefficients at
// the start of their degree.
template <typename T, bool FULL, bool ODE = false>
__device__ __forceinline__ void group_sum(unsigned a, int last, v2<T> X, v2<T> NS, v2<T> NX,
                                          v2<T> D0, v2<T> D1, v2<T> D2, v2<T> (&Z)[12]) {
  constexpr unsigned ES = 16 * sizeof(T);
  const v2<T> zero = vset<T>(T(0), T(0));
  v2<T> P0, P1 = zero, P2 = zero;
  auto acc = [&](const Coef<T> &e, const v2<T> &S0, const v2<T> &S1, const v2<T> &S2,
                 const v2<T> &NL) {
    if (ODE) accumulate<T, FULL>(e, S0, S1, vmul(NL, S0), Z);
    else accumulate<T, FULL>(e, S0, S1, S2, Z);
  };
  Coef<T> e0, e1;
  Rec<T> r;
  load_coef(a, e0);
  load_rec(a, r);
  // degree m: the sums start from its products (a product rounds as the
  // multiply-add onto zero does)
  {
    const v2<T> S2 = ODE ? vmul(r.NL, D0) : D2;
    Z[0] = vmul(e0.CR, D0); Z[1] = vmul(e0.CI, D0); Z[2] = vmul(e0.DR, D0); Z[3] = vmul(e0.DI, D0);
    if (FULL) {
      Z[4] = vmul(e0.CR, D1); Z[5] = vmul(e0.CI, D1); Z[6] = vmul(e0.DR, D1); Z[7] = vmul(e0.DI, D1);
      Z[8] = vmul(e0.CR, S2); Z[9] = vmul(e0.CI, S2); Z[10] = vmul(e0.DR, S2); Z[11] = vmul(e0.DI, S2);
    } else {
#pragma unroll
      for (int q = 4; q < 12; ++q) Z[q] = zero;
    }
  }
  if (last == 0) return;
  // the step from degree m, whose predecessor state is zero
  {
    const v2<T> t = vfma(r.A, X, r.NB);
    P0 = vmul(t, D0);
    if (FULL) {
      const v2<T> nAs = vmul(r.A, NS);
      P1 = vfma(t, D1, vmul(nAs, D0));
      if (!ODE) {
        const v2<T> nAx = vmul(r.A, NX);
        P2 = vfma(t, D2, vfma(vadd(nAs, nAs), D1, vmul(nAx, D0)));
      }
    }
  }
  a += ES;
  load_coef(a, e1);
  // two degrees per trip: degree i in (P0, P1, P2), degree i + 1 in (D0, D1, D2)
  int i = 1;
  for (; i + 2 <= last; i += 2, a += 2 * ES) {
    load_rec(a, r);
    load_coef(a + ES, e0);
    acc(e1, P0, P1, P2, r.NL);
    step_into<T, FULL, ODE>(r, X, NS, NX, P0, P1, P2, D0, D1, D2);
    load_rec(a + ES, r);
    load_coef(a + 2 * ES, e1);
    acc(e0, D0, D1, D2, r.NL);
    step_into<T, FULL, ODE>(r, X, NS, NX, D0, D1, D2, P0, P1, P2);
  }
  v2<T> nl = zero;
  if (i < last) {  // degrees i (with a step) and last = i + 1
    load_rec(a, r);
    load_coef(a + ES, e0);
    acc(e1, P0, P1, P2, r.NL);
    step_into<T, FULL, ODE>(r, X, NS, NX, P0, P1, P2, D0, D1, D2);
    if (ODE && FULL) lds2(a + ES + 14 * sizeof(T), nl);
    acc(e0, D0, D1, D2, nl);
  } else {         // degree last = i
    if (ODE && FULL) lds2(a + 14 * sizeof(T), nl);
    acc(e1, P0, P1, P2, nl);
  }
}

// group_sum for the rescaled states of group_seed_rs: the true d, d', d'' of
// half h are the states times 2^E_h.  Each accumulation multiplies the state
// by SC = 2^E (0 while the true values are below 2^-126); after each step a
// half whose state has grown past 2^32 while E_h < 0 is scaled down by 2^32
// (exactly) and E_h raised by 32, so the states neither overflow nor lose the
// digits of seeds far below the FP32 range (per-degree rescaling).
__device__ __forceinline__ void rescale_half(float &p0, float &p1, float &p2, float &d0, float &d1,
                                             float &d2, int &E, float &sc) {
  if (E < 0 && fabsf(p0) > 4294967296.f) {
    const float f = 2.3283064365386963e-10f;  // 2^-32
    p0 *= f; p1 *= f; p2 *= f; d0 *= f; d1 *= f; d2 *= f;
    E += 32;
    sc = pow2f(E);
  }
}

template <bool FULL>
__device__ __forceinline__ void group_sum_rs(unsigned a, int last, v2<float> X, v2<float> NS,
                                             v2<float> NX, v2<float> D0, v2<float> D1, v2<float> D2,
                                             int E0, int E1, v2<float> (&Z)[12]) {
  constexpr unsigned ES = 16 * sizeof(float);
  const v2<float> zero = vset<float>(0.f, 0.f);
  v2<float> P0 = zero, P1 = zero, P2 = zero;
#pragma unroll
  for (int q = 0; q < 12; ++q) Z[q] = zero;
  float scx = pow2f(E0), scy = pow2f(E1);
  Coef<float> e;
  Rec<float> r;
  auto acc = [&](const v2<float> &S0, const v2<float> &S1, const v2<float> &S2) {
    const v2<float> SC = vset<float>(scx, scy);
    accumulate<float, FULL>(e, vmul(S0, SC), vmul(S1, SC), vmul(S2, SC), Z);
  };
  for (int i = 0; i <= last; ++i, a += ES) {
    load_coef(a, e);
    if (i & 1) acc(P0, P1, P2);
    else acc(D0, D1, D2);
    if (i == last) break;
    load_rec(a, r);
    if (i & 1) {
      step_into<float, FULL>(r, X, NS, NX, P0, P1, P2, D0, D1, D2);
      rescale_half(D0.x, D1.x, D2.x, P0.x, P1.x, P2.x, E0, scx);
      rescale_half(D0.y, D1.y, D2.y, P0.y, P1.y, P2.y, E1, scy);
    } else {
      step_into<float, FULL>(r, X, NS, NX, D0, D1, D2, P0, P1, P2);
      rescale_half(P0.x, P1.x, P2.x, D0.x, D1.x, D2.x, E0, scx);
      rescale_half(P0.y, P1.y, P2.y, D0.y, D1.y, D2.y, E1, scy);
    }
  }
}

// Adds one image of both halves to the candidate's sums.  The image has phase
// E = e^{i(u a + v g)} and weight W; (zr0, zi0) = S0 E, (zr1, zi1) = S1 E,
// zr2 = Re S2 E for the d, d', d'' sums S0, S1, S2.  d/da brings i u and d/dg
// brings i v, so with AU = -W u, GV = -W v:
//   C += W zr0, C_a += AU zi0, C_b += W zr1, C_g += GV zi0,
//   C_aa += AU u zr0, C_ab += AU zi1, C_ag += AU v zr0, C_bb += W zr2,
//   C_bg += GV zi1, C_gg += GV v zr0.
template <typename T, bool FULL>
__device__ __forceinline__ void add_image(v2<T> (&acc)[10], v2<T> W, v2<T> U, v2<T> V,
                                          const v2<T> &ER, const v2<T> &EI, const v2<T> &NEI,
                                          const v2<T> &S0r, const v2<T> &S0i, const v2<T> &S1r,
                                          const v2<T> &S1i, const v2<T> &S2r, const v2<T> &S2i) {
  const v2<T> zr0 = vfma(S0r, ER, vmul(S0i, NEI));
  acc[0] = vfma(W, zr0, acc[0]);
  if (FULL) {
    const v2<T> mone = vset<T>(T(-1), T(-1));
    const v2<T> zi0 = vfma(S0r, EI, vmul(S0i, ER));
    const v2<T> zr1 = vfma(S1r, ER, vmul(S1i, NEI));
    const v2<T> zi1 = vfma(S1r, EI, vmul(S1i, ER));
    const v2<T> zr2 = vfma(S2r, ER, vmul(S2i, NEI));
    const v2<T> NW = vmul(W, mone);
    const v2<T> AU = vmul(NW, U), GV = vmul(NW, V);
    acc[1] = vfma(AU, zi0, acc[1]);
    acc[2] = vfma(W, zr1, acc[2]);
    acc[3] = vfma(GV, zi0, acc[3]);
    acc[4] = vfma(vmul(AU, U), zr0, acc[4]);
    acc[5] = vfma(AU, zi1, acc[5]);
    acc[6] = vfma(vmul(AU, V), zr0, acc[6]);
    acc[7] = vfma(W, zr2, acc[7]);
    acc[8] = vfma(GV, zi1, acc[8]);
    acc[9] = vfma(vmul(GV, V), zr0, acc[9]);
  }
}

// Phase pair E = (cos, sin) rows product: E = EA EG with EA = (ar + i ai),
// EG = (gr + i gi) pairs; returns Re, Im and -Im.
template <typename T>
__device__ __forceinline__ void phase(v2<T> Ar, v2<T> Ai, v2<T> Gr, v2<T> Gi, v2<T> &ER,
                                      v2<T> &EI, v2<T> &NEI) {
  const v2<T> mone = vset<T>(T(-1), T(-1));
  ER = vfma(Ar, Gr, vmul(vmul(Ai, mone), Gi));
  EI = vfma(Ar, Gi, vmul(Ai, Gr));
  NEI = vmul(EI, mone);
}

// Evaluates C (and grad, Hessian when FULL) at pts[p] for the candidates with
// need[p] != 0; results in res[p][0..9] (FP64).  Called by the whole CTA.
//
// Lane layout: a warp holds 32 / cpw sub-slots of cpw lanes; lane p of a
// sub-slot follows candidate p.  Sub-slot `slot` walks the partner groups of
// bandwidth L in its alternating order; the next batch of its groups is
// copied into the other half of the slot's buffer while the current batch is
// summed, and the lanes of a sub-slot read the same staged entries (one
// shared-memory broadcast per load).
template <typename T, bool FULL, bool RS>
__device__ __forceinline__ void evaluate(const NewtonArgs &A, int L, const T *__restrict__ cb,
                                         const T *__restrict__ rcoef, const T *__restrict__ seedK,
                                         const double *pts, const int *need, SmemLayout &sm) {
  constexpr unsigned z = sizeof(T);
  const int P = A.P, cpw = A.cpw, LJ = A.LJ;
  const int NPW = pw_row(LJ), RW = ph_row(LJ), PS = cand_stride(P);
  T *ph = (T *)sm.ea;    // [4][RW][PS]: cos k a, sin k a, cos k g, sin k g
  T *pw = (T *)sm.pw;    // [2][NPW][PS]: PW_PAD zeros, then ch^k (sh^k), k = 0..2LJ+3
  const int tid = threadIdx.x;
  // Each thread takes the cosines and sines it needs from the point itself
  // (no table and no barrier before the tables below).
  // powers k = 0..2L+3 of cos(beta/2) and sin(beta/2): runs of 8 consecutive
  // powers per item, the first by binary powering, the rest by one product each
  constexpr int RUN = 8;
  const int npk = 2 * L + 4, nrun = (npk + RUN - 1) / RUN;
  const FastDiv dw(nrun);
  for (int t = tid; t < 2 * P * nrun; t += blockDim.x) {
    int pr = dw.div(t), k0 = (t - pr * nrun) * RUN;
    int p = pr >> 1, which = pr & 1;
    if (!need[p]) continue;
    const T hb = (T)pts[3 * p + 1] * T(0.5);
    const T x = which ? tsin(hb) : tcos(hb);
    const int k1 = min(k0 + RUN, npk);
    if (RS) {  // mantissa rows, then exponent rows (2 NPW rows further on)
      for (int k = k0; k < k1; ++k) {
        float mt;
        int ex;
        xpow((float)x, k, mt, ex);
        pw[(which * NPW + PW_PAD + k) * PS + p] = (T)mt;
        pw[((2 + which) * NPW + PW_PAD + k) * PS + p] = (T)ex;
      }
    } else {
      T v = ipow_t(x, k0);
      T *o = pw + (which * NPW + PW_PAD + k0) * PS + p;
      o[0] = v;
      for (int k = k0 + 1; k < k1; ++k) {
        v *= x;
        o += PS;
        o[0] = v;
      }
    }
  }
  // phase rows cos, sin of k alpha and k gamma, k = -L..L+1: eight chains per
  // (candidate, angle), chain q holding k = q, q + 8, ... (start e^{i q x},
  // step e^{8 i x})
  for (int t = tid; t < 16 * P; t += blockDim.x) {
    const int pq = t >> 3, q = t & 7, p = pq >> 1, which = pq & 1;
    if (need[p]) {
      const T ang = (T)pts[3 * p + 2 * which];  // alpha or gamma
      const T c1 = tcos(ang), s1 = tsin(ang);
      T *cr_ = ph + ((2 * which) * RW + LJ) * PS + p, *ci_ = cr_ + RW * PS;
      // e^{2ix}, e^{4ix}, e^{8ix} and e^{iqx} by binary powering
      const T c2 = c1 * c1 - s1 * s1, s2 = T(2) * c1 * s1;
      const T c4 = c2 * c2 - s2 * s2, s4 = T(2) * c2 * s2;
      const T c8 = c4 * c4 - s4 * s4, s8 = T(2) * c4 * s4;
      T cr = 1, ci = 0;
      if (q & 1) { cr = c1; ci = s1; }
      if (q & 2) { const T nr = cr * c2 - ci * s2, ni = cr * s2 + ci * c2; cr = nr; ci = ni; }
      if (q & 4) { const T nr = cr * c4 - ci * s4, ni = cr * s4 + ci * c4; cr = nr; ci = ni; }
      for (int m = q; m <= L + 1; m += 8) {
        cr_[m * PS] = cr; ci_[m * PS] = ci;
        if (m > 0 && m <= L) { cr_[-m * PS] = cr; ci_[-m * PS] = -ci; }
        const T nr = cr * c8 - ci * s8, ni = cr * s8 + ci * c8;
        cr = nr; ci = ni;
      }
    }
  }
  __syncthreads();

  const int lane = tid & 31, warp = tid >> 5;
  const int spw = 32 / cpw;
  const int p = lane & (cpw - 1);
  const int sub = lane / cpw;
  const int slot = warp * spw + sub;
  const int nslots = A.nslots;  // sub-slots with a staging buffer (<= NEWTON_WARPS * spw)
  const unsigned submask = cpw == 32 ? 0xffffffffu : (((1u << cpw) - 1u) << (sub * cpw));
  const bool act = p < P && need[p];
  const int pc = p < P ? p : 0;
  const T bt = (T)pts[3 * pc + 1];
  const T xb = tcos(bt), sb = tsin(bt);
  const v2<T> X = vset<T>(xb, xb), NS = vset<T>(-sb, -sb), NX = vset<T>(-xb, -xb);
  // constants of the differential equation for d'' (the non-rescaled path):
  // 1/sin^2 b and -cot b with sin b floored away from zero, and the pole form
  // of the numerator of Q (sign of n in m -/+ n, and +4 sin^2(b/2) or -4 cos^2(b/2))
  v2<T> IS2, NCOT, QSG, QC4;
  {
    const T sfl = sizeof(T) == 8 ? T(1e-150) : T(1e-18);
    const T se = sb > sfl ? sb : sfl;
    const T is2 = T(1) / (se * se), ncot = -xb / se;
    const T chb = tcos(bt * T(0.5)), shb = tsin(bt * T(0.5));
    const bool north = xb >= T(0);
    const T sg = north ? T(-1) : T(1), c4 = north ? T(4) * shb * shb : T(-4) * chb * chb;
    IS2 = vset<T>(is2, is2); NCOT = vset<T>(ncot, ncot);
    QSG = vset<T>(sg, sg); QC4 = vset<T>(c4, c4);
  }
  // shared addresses of this candidate's tables (index 0 of each row)
  const unsigned zs = z * PS;  // bytes between consecutive positions of a row
  const unsigned pcu = smem_u32(pw + PW_PAD * PS + pc);
  const unsigned psu = pcu + zs * NPW;
  const unsigned eacu = smem_u32(ph + LJ * PS + pc);  // k = 0 of cos k a
  const unsigned easu = eacu + zs * RW, egcu = easu + zs * RW, egsu = egcu + zs * RW;
  v2<T> acc[10];
#pragma unroll
  for (int i = 0; i < 10; ++i) acc[i] = vset<T>(T(0), T(0));

  const int ng = (L + 1) * (L + 2) / 2;
  const unsigned HB = z * stage_half(LJ);  // bytes per half buffer
  const unsigned stg = smem_u32(sm.stage) + (unsigned)(slot < nslots ? slot : 0) * 2 * HB;
  // Copy duty of this lane: 16-byte chunk `part` of every entry e = e0,
  // e0 + estep, ...; parts below CPE/2 come from c, the rest from the
  // recurrence table.
  constexpr int CH = 16 / (int)sizeof(T), CPE = 16 / CH;  // reals per chunk, chunks per entry
  const int part = p % CPE, e0 = p / CPE, estep = cpw / CPE;
  const T *srcb = (part < CPE / 2 ? cb : rcoef) + CH * (part % (CPE / 2)) + 8 * e0;
  const unsigned dsto = z * (STAGE_HDR + 16 * e0 + CH * part);
  // Sub-slot `slot` takes group k * nslots + slot in even rounds k and
  // k * nslots + (nslots - 1 - slot) in odd ones: groups come in increasing g
  // (non-increasing length), so the alternating order balances the sub-slots
  // while keeping every sum's order fixed.
  auto group_at = [&](int k) {
    return k * nslots + ((k & 1) ? nslots - 1 - slot : slot);
  };
  if (slot < nslots && slot < ng) {
    GroupWalk walk;
    int k = 0;  // next group of this sub-slot's sequence
    // Copies the next batch of groups into half buffer hb; returns its size
    // (0 when the sub-slot has no group left).
    auto issue_batch = [&](unsigned hb) -> int {
      int cnt = 0, eoff = 0;
      while (cnt < STAGE_BATCH) {
        const int g = group_at(k);
        if (g >= ng) break;
        const Group G = walk.at(g, LJ);
        const int len = L - G.m + 1;
        if (cnt > 0 && eoff + len > LJ + 1) break;
        const T *src = srcb + 8L * G.off;
        unsigned dst = hb + dsto + 16 * z * eoff;
        for (int e = e0; e < len; e += estep, src += 8 * estep, dst += 16 * z * estep)
          cp_async16s(dst, src);
        const unsigned hd = hb + z * 8 * cnt;
        if (p < 4 / CH) cp_async16s(hd + 16 * p, seedK + 4L * g + CH * p);
        if (p == 0) {
          T *h = reinterpret_cast<T *>(__cvta_shared_to_generic(hd));
          h[4] = T(G.m); h[5] = T(G.na); h[6] = T(eoff);
        }
        eoff += len;
        ++cnt;
        ++k;
      }
      return cnt;
    };
    int cur = 0;
    int ncur = issue_batch(stg);
    cp_async_commit();
    while (ncur > 0) {
      const int nnext = issue_batch(stg + (cur ^ 1) * HB);
      cp_async_commit();
      cp_async_wait<1>();
      __syncwarp(submask);
      if (act) {
       for (int t = 0; t < ncur; ++t) {
        const unsigned buf = stg + cur * HB, hd = buf + z * 8 * t;
        T hm, hn, he;
        lds1(hd + 4 * z, hm); lds1(hd + 5 * z, hn); lds1(hd + 6 * z, he);
        const int m = (int)hm, na = (int)hn, eoff = (int)he, aa = m + na, ba = m - na;
        const unsigned ent = buf + z * (STAGE_HDR + 16 * eoff);
        v2<T> K, D0, D1, D2, Z[12];
        lds2(hd, K);
        D1 = D2 = vset<T>(T(0), T(0));
        if constexpr (RS) {
          int E0, E1;
          group_seed_rs<FULL>(pcu + zs * aa, psu + zs * ba, zs * 2 * NPW, zs, K, aa, ba, D0, D1,
                              D2, E0, E1);
          group_sum_rs<FULL>(ent, L - m, X, NS, NX, D0, D1, D2, E0, E1, Z);
        } else {
          group_seed<T, FULL, true>(pcu + zs * aa, psu + zs * ba, zs, K, aa, ba, D0, D1, D2);
          group_sum<T, FULL, true>(ent, L - m, X, NS, NX, D0, D1, D2, Z);
          if (FULL) {
            // d'' = -cot(b) d' + (Q - l(l+1)) d with Q = (m^2 + n^2 - 2mn cos b) / sin^2 b,
            // the numerator as (m - n)^2 + 4mn sin^2(b/2) (beta <= pi/2) or
            // (m + n)^2 - 4mn cos^2(b/2) (beta > pi/2), free of cancellation at the pole
            const v2<T> mm = vset<T>(T(m), T(m)), nh = vset<T>(T(na), T(na + 1));
            const v2<T> dd = vfma(nh, QSG, mm);
            const v2<T> Q = vmul(vfma(vmul(mm, nh), QC4, vmul(dd, dd)), IS2);
#pragma unroll
            for (int q = 0; q < 4; ++q) Z[8 + q] = vfma(NCOT, Z[4 + q], vfma(Q, Z[q], Z[8 + q]));
          }
        }
        const T fm = T(m), fa = T(na);
        const v2<T> MM = vset<T>(fm, fm), NN = vset<T>(fa, fa + T(1));
        // image (m, n): phase e^{i(m a + n g)}, weight 1 for (0, 0) else 2
        // (the image (-m, -n) is the conjugate); an empty half has weight 0
        {
          v2<T> ER, EI, NEI;
          T ar, ai;
          lds1(eacu + zs * m, ar);
          lds1(easu + zs * m, ai);
          phase<T>(vset<T>(ar, ar), vset<T>(ai, ai), vld<T>(egcu + zs * na, egcu + zs * (na + 1)),
                   vld<T>(egsu + zs * na, egsu + zs * (na + 1)), ER, EI, NEI);
          const v2<T> Wt = vset<T>(m == 0 ? T(1) : T(2), na < m ? T(2) : T(0));
          add_image<T, FULL>(acc, Wt, MM, NN, ER, EI, NEI, Z[0], Z[1], Z[4], Z[5], Z[8], Z[9]);
        }
        // image (n, m): c^l_nm d^l_nm e^{i(n a + m g)}, d^l_nm = (-1)^{m-n} d^l_mn
        // (m - n even in the first half, odd in the second); absent when n = +-m
        {
          v2<T> ER, EI, NEI;
          T gr, gi;
          lds1(egcu + zs * m, gr);
          lds1(egsu + zs * m, gi);
          phase<T>(vld<T>(eacu + zs * na, eacu + zs * (na + 1)),
                   vld<T>(easu + zs * na, easu + zs * (na + 1)), vset<T>(gr, gr), vset<T>(gi, gi),
                   ER, EI, NEI);
          const v2<T> Wt = vset<T>(na == m || na == -m ? T(0) : T(2), na + 1 < m ? T(-2) : T(0));
          add_image<T, FULL>(acc, Wt, NN, MM, ER, EI, NEI, Z[2], Z[3], Z[6], Z[7], Z[10], Z[11]);
        }
       }
      }
      __syncwarp(submask);
      cur ^= 1;
      ncur = nnext;
    }
    cp_async_wait<0>();
  }
  // both halves, then the sub-slots of the warp that follow the same candidate,
  // then (below) the warps in index order: all in the working precision
  const int nq = FULL ? 10 : 1;
  T r[10];
#pragma unroll
  for (int i = 0; i < 10; ++i) r[i] = acc[i].x + acc[i].y;
  for (int o = cpw; o < 32; o <<= 1)
#pragma unroll
    for (int i = 0; i < 10; ++i)
      if (i < nq) r[i] += __shfl_xor_sync(0xffffffffu, r[i], o);
  if (lane < cpw && p < P)
#pragma unroll
    for (int i = 0; i < 10; ++i)
      if (i < nq) ((T *)sm.red)[(warp * P + p) * 10 + i] = r[i];
  __syncthreads();
  for (int idx = tid; idx < P * nq; idx += blockDim.x) {
    int pp = idx / nq, i = idx - pp * nq;
    if (need[pp]) {
      T v = 0;
      for (int w = 0; w < NEWTON_WARPS; ++w) v += ((const T *)sm.red)[(w * P + pp) * 10 + i];
      sm.res[pp * 10 + i] = (double)v;
    }
  }
  __syncthreads();
}

// Carves the refinement kernels' shared memory (layout of newton_smem_bytes).
template <typename T, bool RS>
__device__ __forceinline__ int *carve_smem(unsigned char *smem_raw, int P, int LJ, SmemLayout &sm) {
  double *dp = reinterpret_cast<double *>(smem_raw);
  sm.th = dp; dp += 3 * P;
  sm.tr = dp; dp += 3 * P;
  sm.del = dp; dp += 3 * P;
  sm.Cc = dp; dp += P;
  sm.res = dp; dp += 10 * P;
  int *ip = reinterpret_cast<int *>(dp);
  sm.state = ip; ip += P;
  sm.steps = ip; ip += P;
  sm.tries = ip; ip += P;
  sm.fl = ip; ip += P;
  int *need = ip; ip += P;
  uintptr_t u = reinterpret_cast<uintptr_t>(ip);
  u = (u + 15) & ~uintptr_t(15);
  T *tp = reinterpret_cast<T *>(u);
  sm.red = tp; tp += 10 * P * NEWTON_WARPS;
  sm.ea = tp; tp += 4 * cand_stride(P) * ph_row(LJ);
  sm.pw = tp; tp += (RS ? 4 : 2) * cand_stride(P) * pw_row(LJ);
  tp = reinterpret_cast<T *>((reinterpret_cast<uintptr_t>(tp) + 31) & ~uintptr_t(31));
  sm.stage = tp;
  for (int t = threadIdx.x; t < (RS ? 4 : 2) * cand_stride(P) * pw_row(LJ); t += blockDim.x)
    ((T *)sm.pw)[t] = T(0);  // pads
  return need;
}

// C_L, its gradient and Hessian (Section 2.2) at Q given rotations per
// particle: the refinement kernel's evaluation, one CTA per particle.
// out[b][q][10] = (C, C_a, C_b, C_g, C_aa, C_ab, C_ag, C_bb, C_bg, C_gg).
template <typename T, bool RS>
__global__ void __launch_bounds__(NEWTON_THREADS, sizeof(T) == 8 ? 1 : 2)
k_objective(const T *__restrict__ c, const T *__restrict__ rcoef, const T *__restrict__ seedK,
            NewtonArgs A, int L, int Q, const double *__restrict__ pts, double *__restrict__ out) {
  const long b = blockIdx.x;
  const int tid = threadIdx.x;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  SmemLayout sm;
  int *need = carve_smem<T, RS>(smem_raw, A.P, A.LJ, sm);
  if (tid < A.P) {
    const bool on = tid < Q;
    for (int i = 0; i < 3; ++i) sm.th[3 * tid + i] = on ? pts[3 * (b * Q + tid) + i] : 0.0;
    need[tid] = on;
  }
  __syncthreads();
  evaluate<T, true, RS>(A, L, c + 4 * b * A.nc, rcoef, seedK, sm.th, need, sm);
  for (int t = tid; t < Q * 10; t += blockDim.x) out[10 * b * Q + t] = sm.res[t];
}

// The march of all candidates of particle b by the whole CTA.
template <typename T, bool RS>
__device__ __forceinline__ void newton_particle(const T *__restrict__ c, const T *__restrict__ rcoef,
                                                const T *__restrict__ seedK, const NewtonArgs &A,
                                                const int *__restrict__ n_cand,
                                                double *__restrict__ euler, double *__restrict__ score,
                                                int *__restrict__ cflags, long long *__restrict__ work,
                                                long b, unsigned char *smem_raw) {
  const int P = A.P, tid = threadIdx.x;
  SmemLayout sm;  // staging buffers: [slots][2][stage_half(L_J)]
  int *need = carve_smem<T, RS>(smem_raw, P, A.LJ, sm);
  const int nc_b = n_cand[b];
  if (tid < P) {
    double *e = euler + 3 * (b * P + tid);
    sm.th[3 * tid] = e[0]; sm.th[3 * tid + 1] = e[1]; sm.th[3 * tid + 2] = e[2];
    sm.state[tid] = tid < nc_b ? ST_RUN : ST_DEAD;
    sm.fl[tid] = 0;
    sm.Cc[tid] = __longlong_as_double(0x7ff8000000000000LL);
  }
  __syncthreads();
  const T *cb = c + 4 * b * A.nc;
  const double piv_rel = sizeof(T) == 8 ? 1e-12 : 1e-6;  // H summed in T
  long long work_full = 0, work_val = 0;  // counted by thread 0

  // A trial point that is accepted is where the next step needs C, grad and
  // H, so trials are evaluated with derivatives except on a level's last
  // step: per level one derivative evaluation at the start point, then one
  // evaluation per trial.  The points, the arithmetic at each point and the
  // decisions are those of "evaluate at theta, step, test the trial".
  for (int lev = 0; lev < A.nlev; ++lev) {
    const int L = A.Ls[lev];
    // recurrence steps of one evaluation: sum_{m<=L} (2m+1)(L-m+1)
    long long steps_L = 0;
    for (int mm = 0; mm <= L; ++mm) steps_L += (long long)(2 * mm + 1) * (L - mm + 1);
    int want = 0;
    if (tid < P) { need[tid] = sm.state[tid] != ST_DEAD; want = need[tid]; }
    if (!__syncthreads_or(want)) break;
    if (tid == 0)
      for (int q = 0; q < P; ++q) work_full += need[q] ? steps_L : 0;
    evaluate<T, true, RS>(A, L, cb, rcoef, seedK, sm.th, need, sm);
    // the 3x3 solves of the final level run in FP64 in every plan
    const bool last = lev == A.nlev - 1;
    auto step_from = [&]() {
      if (last) start_step<double>(tid, L, A.tol, A.grad != 0, sm, piv_rel);
      else start_step<T>(tid, L, A.tol, A.grad != 0, sm, piv_rel);
    };
    if (tid < P && need[tid]) {
      sm.steps[tid] = 0;
      step_from();
    }
    for (int round = 0; round < 3 * A.M; ++round) {
      int tw = 0, wf = 0;
      if (tid < P) {
        need[tid] = sm.state[tid] == ST_TRIAL;
        tw = need[tid];
        wf = tw && sm.steps[tid] < A.M - 1;
      }
      if (!__syncthreads_or(tw)) break;
      const bool full = __syncthreads_or(wf);
      if (tid == 0)
        for (int q = 0; q < P; ++q) (full ? work_full : work_val) += need[q] ? steps_L : 0;
      if (full) evaluate<T, true, RS>(A, L, cb, rcoef, seedK, sm.tr, need, sm);
      else evaluate<T, false, RS>(A, L, cb, rcoef, seedK, sm.tr, need, sm);
      if (tid < P && need[tid]) {
        double Ct = sm.res[10 * tid];
        if (Ct >= sm.Cc[tid] - A.acc_tol * fabs(sm.Cc[tid])) {
          for (int i = 0; i < 3; ++i) sm.th[3 * tid + i] = sm.tr[3 * tid + i];
          sm.Cc[tid] = Ct;
          if (sm.steps[tid] < A.M - 1) {
            ++sm.steps[tid];
            step_from();  // derivatives at the accepted point
          } else {
            sm.state[tid] = ST_STOP;
          }
        } else if (++sm.tries[tid] == 3) {
          sm.fl[tid] |= 4;
          sm.state[tid] = ST_STOP;  // a repeated step from the same point rejects again
        } else {
          double tr[3];
          for (int i = 0; i < 3; ++i) {
            sm.del[3 * tid + i] *= 0.5;
            tr[i] = sm.th[3 * tid + i] + sm.del[3 * tid + i];
          }
          wrap_d(tr);
          for (int i = 0; i < 3; ++i) sm.tr[3 * tid + i] = tr[i];
        }
      }
    }
    __syncthreads();
  }
  if (tid < P) {
    long o = b * P + tid;
    if (tid < nc_b) {
      euler[3 * o] = sm.th[3 * tid];
      euler[3 * o + 1] = sm.th[3 * tid + 1];
      euler[3 * o + 2] = sm.th[3 * tid + 2];
      score[o] = sm.Cc[tid];
    }
    cflags[o] = sm.fl[tid];
  }
  if (tid == 0 && work) {
    work[2 * b] = work_full;
    work[2 * b + 1] = work_val;
  }
}

// One CTA per particle, in index order.
template <typename T, bool RS>
__global__ void __launch_bounds__(NEWTON_THREADS, sizeof(T) == 8 ? 1 : 2)
k_newton(const T *__restrict__ c, const T *__restrict__ rcoef,
         const T *__restrict__ seedK, NewtonArgs A, const int *__restrict__ n_cand,
         double *__restrict__ euler, double *__restrict__ score, int *__restrict__ cflags,
         long long *__restrict__ work) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  newton_particle<T, RS>(c, rcoef, seedK, A, n_cand, euler, score, cflags, work, blockIdx.x,
                         smem_raw);
}

// Persistent CTAs (as many as fit on the GPU at once) pulling particles from a
// cost-sorted queue: order[] lists the particles by decreasing refinement cost
// (candidates to march), and a CTA takes the next entry with an atomic ticket,
// so the most expensive particles start first and the cheap ones fill the tail
// (longest processing time first).  Each particle's arithmetic is that of
// k_newton, so the results are bit-identical.
template <typename T, bool RS>
__global__ void __launch_bounds__(NEWTON_THREADS, sizeof(T) == 8 ? 1 : 2)
k_newton_queue(const T *__restrict__ c, const T *__restrict__ rcoef, const T *__restrict__ seedK,
               NewtonArgs A, const int *__restrict__ n_cand, double *__restrict__ euler,
               double *__restrict__ score, int *__restrict__ cflags, long long *__restrict__ work,
               const int *__restrict__ order, int B, int *__restrict__ ticket) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ int next;
  for (;;) {
    __syncthreads();
    if (threadIdx.x == 0) next = atomicAdd(ticket, 1);
    __syncthreads();
    const int q = next;
    if (q >= B) break;
    newton_particle<T, RS>(c, rcoef, seedK, A, n_cand, euler, score, cflags, work, order[q],
                           smem_raw);
  }
}

// order[] = the particles by decreasing candidate count (stable in the index),
// by a counting sort in one CTA; also resets the queue's ticket.
__global__ void k_cost_order(const int *__restrict__ n_cand, int B, int P, int *__restrict__ order,
                             int *__restrict__ ticket) {
  __shared__ int start[MATCHA_MAX_P + 2];
  const int tid = threadIdx.x;
  if (tid <= P + 1) start[tid] = 0;
  __syncthreads();
  for (int b = tid; b < B; b += blockDim.x) atomicAdd(&start[P - min(max(n_cand[b], 0), P) + 1], 1);
  __syncthreads();
  if (tid == 0) {
    for (int k = 1; k <= P + 1; ++k) start[k] += start[k - 1];
    *ticket = 0;
  }
  __syncthreads();
  // stable placement: each bin is filled in index order by one warp per bin
  const int warp = tid >> 5, lane = tid & 31, nw = blockDim.x >> 5;
  for (int k = warp; k <= P; k += nw) {
    int pos = start[k];
    for (int b0 = 0; b0 < B; b0 += 32) {
      const int b = b0 + lane;
      const bool in = b < B && P - min(max(n_cand[b], 0), P) == k;
      const unsigned m = __ballot_sync(0xffffffffu, in);
      if (in) order[pos + __popc(m & ((1u << lane) - 1u))] = b;
      pos += __popc(m);
    }
  }
}

// Lanes per warp sub-slot: one per candidate, at least 16.
static int newton_cpw(int P) { return P <= 16 ? 16 : 32; }

// Shared memory of k_newton with `slots` staging buffers.
// Above this bandwidth the 32-bit plans run the rescaled recurrence: seeds
// flushed below the FP32 range would otherwise grow into significant terms
// (at L_J = 100 a seed under 2^-126 reaches 2.6e-4).
constexpr int RESCALE_ABOVE_L = 64;
bool newton_rescaled(const Plan &p) { return !p.fp64 && p.LJ > RESCALE_ABOVE_L; }

static size_t newton_smem_bytes(const Plan &p, size_t tsize, int slots) {
  size_t P = p.P;
  const size_t pw_rows = newton_rescaled(p) ? 4 : 2;
  size_t bytes = sizeof(double) * (3 * P * 3 + P + 10 * P);
  bytes += sizeof(int) * 5 * P;
  bytes = (bytes + 15) / 16 * 16;
  const size_t PS = cand_stride(p.P);
  bytes += tsize * (10 * P * NEWTON_WARPS + 4 * PS * ph_row(p.LJ) + pw_rows * PS * pw_row(p.LJ)) + 32;
  bytes += tsize * (size_t)slots * 2 * stage_half(p.LJ);
  return bytes;
}

// Staging buffers that fit: one per sub-slot when possible, else fewer (the
// other sub-slots then idle); 0 when even one does not fit.
static int newton_slots(const Plan &p, size_t tsize) {
  const size_t limit = 227 * 1024;
  int slots = NEWTON_WARPS * (32 / newton_cpw(p.P));
  while (slots > 0 && newton_smem_bytes(p, tsize, slots) > limit) --slots;
  return slots;
}

int newton_slots(const Plan &p) { return newton_slots(p, p.fp64 ? 8 : 4); }
size_t newton_smem(const Plan &p) { return newton_smem_bytes(p, p.fp64 ? 8 : 4, newton_slots(p)); }
bool newton_fits(const Plan &p) { return newton_slots(p) > 0; }

template <typename T>
cudaError_t launch_newton(const Plan &p, const T *c, int B, const int *n_cand, double *euler,
                          double *score, int *cflags, long long *work, cudaStream_t st, int batch) {
  if (B == 0) return cudaSuccess;
  cudaError_t e;
  if (launch_newton_spread<T>(p, c, B, std::max(B, batch), n_cand, euler, score, cflags, work, st, &e)) return e;
  if constexpr (sizeof(T) == 8) {
    return cudaErrorInvalidConfiguration;  // FP64 plans have a spread shape each
  } else {
    NewtonArgs A;
    A.LJ = p.LJ; A.nlev = p.nlev; A.M = p.M; A.P = p.P;
    A.cpw = newton_cpw(p.P);
    A.nslots = newton_slots(p, sizeof(T));
    if (A.nslots == 0) return cudaErrorInvalidConfiguration;
    for (int i = 0; i < MATCHA_MAX_LEVELS; ++i) A.Ls[i] = i < p.nlev ? p.Ls[i] : 0;
    A.tol = p.step_tol;
    A.acc_tol = p.accept_tol;
    A.grad = p.refine;
    A.nc = p.nc;
    const size_t smem = newton_smem_bytes(p, sizeof(T), A.nslots);
    auto kern = newton_rescaled(p) ? k_newton<T, true> : k_newton<T, false>;
    if ((e = allow_smem(kern, smem)) != cudaSuccess) return e;
    kern<<<B, NEWTON_THREADS, smem, st>>>(c, (const T *)p.rcoef, (const T *)p.seedK, A, n_cand, euler, score,
                                          cflags, work);
    return cudaGetLastError();
  }
}

template <typename T>
cudaError_t launch_newton_queue(const Plan &p, const T *c, int B, const int *n_cand, double *euler,
                                double *score, int *cflags, long long *work, int *order,
                                int *ticket, cudaStream_t st) {
  if (B == 0) return cudaSuccess;
  NewtonArgs A;
  A.LJ = p.LJ; A.nlev = p.nlev; A.M = p.M; A.P = p.P;
  A.cpw = newton_cpw(p.P);
  A.nslots = newton_slots(p, sizeof(T));
  if (A.nslots == 0) return cudaErrorInvalidConfiguration;
  for (int i = 0; i < MATCHA_MAX_LEVELS; ++i) A.Ls[i] = i < p.nlev ? p.Ls[i] : 0;
  A.tol = p.step_tol; A.acc_tol = p.accept_tol; A.grad = p.refine; A.nc = p.nc;
  const size_t smem = newton_smem_bytes(p, sizeof(T), A.nslots);
  k_cost_order<<<1, 1024, 0, st>>>(n_cand, B, p.P, order, ticket);
  cudaError_t launched = cudaGetLastError();
  if (launched != cudaSuccess) return launched;
  int dev = 0, sms = 0, per_sm = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  auto go = [&](auto kern) {
    const cudaError_t e = allow_smem(kern, smem, 16);
    if (e != cudaSuccess) return e;
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, NEWTON_THREADS, smem);
    const int grid = std::max(1, std::min(B, std::max(per_sm, 1) * sms));
    kern<<<grid, NEWTON_THREADS, smem, st>>>(c, (const T *)p.rcoef, (const T *)p.seedK, A, n_cand,
                                             euler, score, cflags, work, order, B, ticket);
    return cudaGetLastError();
  };
  if constexpr (sizeof(T) == 4) {
    if (newton_rescaled(p)) return go(k_newton_queue<T, true>);
  }
  return go(k_newton_queue<T, false>);
}
template cudaError_t launch_newton_queue<float>(const Plan &, const float *, int, const int *,
                                                double *, double *, int *, long long *, int *,
                                                int *, cudaStream_t);
template cudaError_t launch_newton_queue<double>(const Plan &, const double *, int, const int *,
                                                 double *, double *, int *, long long *, int *,
                                                 int *, cudaStream_t);

template <typename T>
cudaError_t launch_objective(const Plan &p, const T *c, int B, int L, int Q, const double *pts,
                             double *out, cudaStream_t st) {
  if (B == 0 || Q == 0) return cudaSuccess;
  cudaError_t e;
  if (launch_objective_spread<T>(p, c, B, L, Q, pts, out, st, &e)) return e;
  if constexpr (sizeof(T) == 8) {
    return cudaErrorInvalidConfiguration;  // as launch_newton
  } else {
    NewtonArgs A;
    A.LJ = p.LJ; A.nlev = p.nlev; A.M = p.M; A.P = p.P;
    A.cpw = newton_cpw(p.P);
    A.nslots = newton_slots(p, sizeof(T));
    if (A.nslots == 0) return cudaErrorInvalidConfiguration;
    for (int i = 0; i < MATCHA_MAX_LEVELS; ++i) A.Ls[i] = i < p.nlev ? p.Ls[i] : 0;
    A.tol = p.step_tol; A.acc_tol = p.accept_tol; A.grad = p.refine; A.nc = p.nc;
    const size_t smem = newton_smem_bytes(p, sizeof(T), A.nslots);
    auto kern = newton_rescaled(p) ? k_objective<T, true> : k_objective<T, false>;
    if ((e = allow_smem(kern, smem)) != cudaSuccess) return e;
    kern<<<B, NEWTON_THREADS, smem, st>>>(c, (const T *)p.rcoef, (const T *)p.seedK, A, L, Q, pts, out);
    return cudaGetLastError();
  }
}
template cudaError_t launch_objective<float>(const Plan &, const float *, int, int, int,
                                             const double *, double *, cudaStream_t);
template cudaError_t launch_objective<double>(const Plan &, const double *, int, int, int,
                                              const double *, double *, cudaStream_t);

template cudaError_t launch_newton<float>(const Plan &, const float *, int, const int *, double *,
                                          double *, int *, long long *, cudaStream_t, int);
template cudaError_t launch_newton<double>(const Plan &, const double *, int, const int *, double *,
                                           double *, int *, long long *, cudaStream_t, int);

// Eight lanes per particle: the candidates' scores and flags are read together and
// three lanes take one angle's sincos each.  (A thread per particle: 10.5 us for one
// particle, a chain of loads and six FP64 trigonometric functions.)
__global__ void k_final_select(int B, int P, const int *P_per, const int *n_cand,
                               const double *ce, const double *cs, const int *cf, double *euler,
                               double *R, double *score, int *best_p, int *flags) {
  const int t = blockIdx.x * blockDim.x + threadIdx.x, lane = t & 7;
  const bool live = (t >> 3) < B;
  const int b = live ? t >> 3 : B - 1;
  const int nc = n_cand[b];
  const int Pb = P_per ? min(P_per[b], P) : P;
  int best = -1, fl = nc < Pb ? 8 : 0;
  double bs = -INFINITY;
  for (int q = lane; q < nc; q += 8) {
    const double s = cs[(long)b * P + q];
    fl |= cf[(long)b * P + q];
    if (s > bs) { bs = s; best = q; }
  }
  for (int o = 4; o > 0; o >>= 1) {  // the first of the largest
    const double os = __shfl_xor_sync(0xffffffffu, bs, o);
    const int ob = __shfl_xor_sync(0xffffffffu, best, o);
    fl |= __shfl_xor_sync(0xffffffffu, fl, o);
    if (ob >= 0 && (best < 0 || os > bs || (os == bs && ob < best))) { bs = os; best = ob; }
  }
  const double ang = best >= 0 && lane < 3 ? ce[3 * ((long)b * P + best) + lane] : 0.0;
  double sn, cn;
  sincos(ang, &sn, &cn);
  const double ca = __shfl_sync(0xffffffffu, cn, 0, 8), sa = __shfl_sync(0xffffffffu, sn, 0, 8);
  const double cb = __shfl_sync(0xffffffffu, cn, 1, 8), sb = __shfl_sync(0xffffffffu, sn, 1, 8);
  const double cg = __shfl_sync(0xffffffffu, cn, 2, 8), sg = __shfl_sync(0xffffffffu, sn, 2, 8);
  if (!live) return;
  if (lane < 3) euler[3 * b + lane] = ang;
  if (lane) return;
  // R = r_z(a) r_y(b) r_z(g)
  double *r = R + 9 * b;
  r[0] = ca * cb * cg - sa * sg; r[1] = -ca * cb * sg - sa * cg; r[2] = ca * sb;
  r[3] = sa * cb * cg + ca * sg; r[4] = -sa * cb * sg + ca * cg; r[5] = sa * sb;
  r[6] = -sb * cg;               r[7] = sb * sg;                 r[8] = cb;
  score[b] = best >= 0 ? bs : __longlong_as_double(0x7ff8000000000000LL);
  best_p[b] = best;
  flags[b] = fl;
}

cudaError_t launch_final_select(const Plan &p, int B, const int *P_per, const int *n_cand,
                                const double *cand_euler, const double *cand_score,
                                const int *cand_flags, double *euler, double *R, double *score,
                                int *best_p, int *flags, cudaStream_t st) {
  if (B == 0) return cudaSuccess;
  k_final_select<<<(B + 15) / 16, 128, 0, st>>>(B, p.P, P_per, n_cand, cand_euler, cand_score,
                                                  cand_flags, euler, R, score, best_p, flags);
  return cudaGetLastError();
}

}  // namespace matcha
