// Step a6 for batches that leave SMs idle with one CTA per particle (newton.cu):
// the same march, bit for bit, with each particle spread over more warps and,
// where that helps, over a cluster of CTAs.  newton.cu explains the objective,
// the recurrences and the step rule.
//
// newton.cu fixes the order of a particle's sums: up to 16 sub-slots (8 with more
// than 16 candidates), each adding its own sequence of partner groups, then pairs
// of sub-slots, then the pairs in order.  Here a warp holds as many sub-slots as
// P lanes each fit (a chain group), and W warps (workers) share a chain group:
// worker w computes rounds w, w + W, ... of its sub-slots' groups, i.e. everything
// up to the images' sums z of each group, and leaves them in shared memory; after
// each chunk of rounds the workers add the chunk's z to the chains' accumulators in
// round order, each worker some of the ten quantities.  The long recurrences of a chain so run on W warps at once while its sum
// keeps its order.  A particle's chain groups are dealt to the CTAs of a cluster;
// every CTA receives all chains' sums through distributed shared memory, takes
// the same step decisions, and the first one writes the results.
//
// What bounds it: latency of the recurrence steps at the few warps a small batch
// gives (per degree and pair of order pairs 20 packed operations in a dependent
// chain), then the tables each CTA makes per evaluation and the step rule.
//
// Staging: each warp copies its sub-slots' degree entries, recurrence
// coefficients and group descriptors with cp.async into a ring of its own, one
// piece (a group, or STAGE_ENTRIES degrees of a long one) per slot and one piece
// ahead, so the ring does not grow with L_J.  All sub-slots of a warp take as
// many degrees as the longest one's group has; entries past a group's end, and
// groups past the last, are zero-filled and add exactly nothing.
#include <algorithm>
#include <cooperative_groups.h>
#include "newton_common.cuh"

namespace matcha {
namespace {

constexpr int SPREAD_THREADS = 256;

struct SpreadArgs {
  int LJ, nlev, M, P, nslots;
  int spw, ngrp;  // sub-slots per chain group, chain groups per particle
  int cpc, W;     // chain groups per CTA, workers per chain group
  int ctas;       // CTAs per particle
  int chunk;      // rounds between two accumulations, a multiple of W
  int pairs;      // sub-slots are summed in pairs (P <= 16) before the fixed-order sum
  int grad;       // 1: gradient steps grad / ||H||_F instead of Newton steps
  int Ls[MATCHA_MAX_LEVELS];
  double tol, acc_tol;
  long nc;
  const int4 *sched;  // [nslots][nrounds]: newton_schedule
  int nrounds;
  int o_red, o_z, o_trig, o_ph, o_pw, o_stage;  // byte offsets in shared memory
};

// A CTA's shared memory: per candidate the current point, the trial point and
// step, C, the last evaluation's results, the step state; then (byte offsets made
// by the launcher) the partial sums, the tables and the staging rings.  Accessors
// rather than pointers, so that none is held in registers through an evaluation.
struct Smem {
  const SpreadArgs &A;
  unsigned char *base;
  __device__ __forceinline__ double *th() const { return reinterpret_cast<double *>(base); }
  __device__ __forceinline__ double *tr() const { return th() + 3 * A.P; }
  __device__ __forceinline__ double *del() const { return th() + 6 * A.P; }
  __device__ __forceinline__ double *Cc() const { return th() + 9 * A.P; }
  __device__ __forceinline__ double *res() const { return th() + 10 * A.P; }
  // recurrence steps counted by thread 0: with derivatives, values only
  __device__ __forceinline__ long long *work() const { return reinterpret_cast<long long *>(th() + 20 * A.P); }
  __device__ __forceinline__ int *state() const { return reinterpret_cast<int *>(th() + 20 * A.P + 2); }
  __device__ __forceinline__ int *steps() const { return state() + A.P; }
  __device__ __forceinline__ int *tries() const { return state() + 2 * A.P; }
  __device__ __forceinline__ int *fl() const { return state() + 3 * A.P; }
  __device__ __forceinline__ int *need() const { return state() + 4 * A.P; }
  __device__ __forceinline__ int *turn() const { return state() + 5 * A.P; }  // red buffer in use
  template <typename T> __device__ __forceinline__ T *red() const { return reinterpret_cast<T *>(base + A.o_red); }
  template <typename T> __device__ __forceinline__ T *z() const { return reinterpret_cast<T *>(base + A.o_z); }
  template <typename T> __device__ __forceinline__ T *trig() const { return reinterpret_cast<T *>(base + A.o_trig); }
  template <typename T> __device__ __forceinline__ T *ph() const { return reinterpret_cast<T *>(base + A.o_ph); }
  template <typename T> __device__ __forceinline__ T *pw() const { return reinterpret_cast<T *>(base + A.o_pw); }
};

// The pointers the step rule works on, made where it runs.
struct StepState {
  double *th, *tr, *del, *Cc, *res;
  int *state, *steps, *tries, *fl;
  __device__ __forceinline__ explicit StepState(const Smem &s)
      : th(s.th()), tr(s.tr()), del(s.del()), Cc(s.Cc()), res(s.res()), state(s.state()),
        steps(s.steps()), tries(s.tries()), fl(s.fl()) {}
};

// 16 bytes global -> shared; zeros when !live (nothing is read).
__device__ __forceinline__ void cp_async16(unsigned dst, const void *src, bool live) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 16, %2;\n" ::"r"(dst), "l"(src), "r"(live ? 16 : 0));
}
__device__ __forceinline__ int lds_int(unsigned a) {
  int v;
  asm volatile("ld.shared.b32 %0, [%1];\n" : "=r"(v) : "r"(a));
  return v;
}
__device__ __forceinline__ void sts2(unsigned a, float2 x) {
  asm volatile("st.shared.v2.f32 [%0], {%1, %2};\n" ::"r"(a), "f"(x.x), "f"(x.y) : "memory");
}
__device__ __forceinline__ void sts2(unsigned a, double2 x) {
  asm volatile("st.shared.v2.f64 [%0], {%1, %2};\n" ::"r"(a), "d"(x.x), "d"(x.y) : "memory");
}
__device__ __forceinline__ float smul(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ double smul(double a, double b) { return __dmul_rn(a, b); }
__device__ __forceinline__ float sfma(float a, float b, float c) { return __fmaf_rn(a, b, c); }
__device__ __forceinline__ double sfma(double a, double b, double c) { return __fma_rn(a, b, c); }
// a b - c d, rounded as group_seed of newton.cu rounds it: both products in FP32,
// the second alone in FP64 (the compiler fuses the first there)
__device__ __forceinline__ float sdiff(float a, float b, float c, float d) {
  return __fsub_rn(__fmul_rn(a, b), __fmul_rn(c, d));
}
__device__ __forceinline__ double sdiff(double a, double b, double c, double d) {
  return __fma_rn(a, b, -__dmul_rn(c, d));
}

// Ring slot of one sub-slot, in reals: the group's descriptor (layout:
// k_group_desc in plan_tables.cu), the round's schedule entry (16 bytes), then 8
// c reals per degree entry, then 8 recurrence reals per entry (a_a, a_b, -b_a,
// -b_b, -e_a, -e_b, -l(l+1), -l(l+1)).  STAGE_ENTRIES is even, so a group
// resumed in the next slot finds the two recurrence states in their usual roles.
constexpr int STAGE_SLOTS = 2, STAGE_ENTRIES = 24;
template <typename T> constexpr int STAGE_HEAD = GROUP_DESC + 16 / (int)sizeof(T);
template <typename T> constexpr int STAGE_SUB = STAGE_HEAD<T> + 16 * STAGE_ENTRIES;

// Trigonometric table (candidate fastest, stride cand_stride): cos, sin of b/2, a
// and g, cos b, sin b, 1 / sin^2 b and -cot b (sin b floored away from zero).
constexpr int TRIG = 10;
// Sums of a group that a worker leaves per (sub-slot, round), as pairs over the
// halves: zr0, zi0, zr1, zi1, zr2 of both images, candidate fastest, then the
// images' weights.
__host__ __device__ __forceinline__ int z_row(int P) { return 20 * P + 24; }

// Seeds at l = m of both halves: d = sigma K ch^a sh^b with a = m+n,
// b = m-n, sigma = (-1)^b; with FULL also d' (Appendix A.4 applied to the
// closed form: d/db (ch^a sh^b) = (b ch^{a+1} sh^{b-1} - a ch^{a-1} sh^{b+1})/2);
// d'' comes from the differential equation.  The first half has a = aa, b = ba
// (both even, so sigma = +1); the second a = aa + 1, b = ba - 1 (sigma = -1).
// pc, ps: shared addresses of ch^aa, sh^ba in the padded power tables; a term
// whose integer coefficient is zero may read a zero pad, so it adds exactly 0.
// z: bytes between consecutive powers in the table.  d: shared address of the
// descriptor, which holds sigma K, sigma K / 2 and the integers a, b as pairs.
// Scalar products: packing the table values into register pairs would cost a
// move each, and a packed product occupies the pipe as long as two scalar ones.
template <typename T, bool FULL>
__device__ __forceinline__ void group_seed(unsigned pc, unsigned ps, unsigned z, unsigned d,
                                           v2<T> &D0, v2<T> &D1) {
  T c0, c1, s0, sm1;
  lds1(pc, c0); lds1(pc + z, c1);
  lds1(ps, s0); lds1(ps - z, sm1);
  v2<T> GK, GH;
  lds4(d, GK, GH);
  D0.x = smul(GK.x, smul(c0, s0));
  D0.y = smul(GK.y, smul(c1, sm1));
  if (FULL) {
    T c2, cm1, s1, sm2;
    lds1(pc + 2 * z, c2); lds1(pc - z, cm1);
    lds1(ps + z, s1); lds1(ps - 2 * z, sm2);
    v2<T> A, B;
    lds4(d + 4 * sizeof(T), A, B);
    D1.x = smul(GH.x, sdiff(B.x, smul(c1, sm1), A.x, smul(cm1, s1)));
    D1.y = smul(GH.y, sdiff(B.y, smul(c2, sm2), A.y, smul(c0, s0)));
  }
}

template <typename T> __device__ __forceinline__ void load_coef(unsigned a, Coef<T> &e) {
  lds4(a, e.CR, e.CI);
  lds4(a + 4 * sizeof(T), e.DR, e.DI);
}
// the recurrence reals of the entry whose c is at a
template <typename T> __device__ __forceinline__ void load_rec(unsigned a, Rec<T> &r) {
  lds4(a + 8 * STAGE_ENTRIES * sizeof(T), r.A, r.NB);
  lds4(a + (8 * STAGE_ENTRIES + 4) * sizeof(T), r.NE, r.NL);
}
// n staged degrees of one partner group for one candidate, added to Z[0..3] =
// sum d (Re c_mn, Im c_mn, Re c_nm, Im c_nm), and with FULL the same with d'
// (Z[4..7]) and -l(l+1) d (Z[8..11], completed by the caller with the
// differential equation); each a pair over the two halves.  a: shared address
// of the piece's first c entry.  The state holds d^l in (D0, D1) and d^{l-1} in
// (P0, P1), zero before degree m; two degrees per trip with the roles swapped
// in the second.  A piece that ends its group (fin) takes no step past its last
// degree; any other has an even number of degrees.
template <typename T, bool FULL>
__device__ __forceinline__ void group_sum(unsigned a, int n, bool fin, v2<T> X, v2<T> NS, v2<T> &D0,
                                          v2<T> &D1, v2<T> &P0, v2<T> &P1, v2<T> (&Z)[12]) {
  constexpr unsigned ES = 8 * sizeof(T);
  const v2<T> none = vset<T>(T(0), T(0));
  v2<T> u = none;
  auto acc = [&](const Coef<T> &e, const v2<T> &S0, const v2<T> &S1, const v2<T> &NL) {
    accumulate<T, FULL>(e, S0, S1, FULL ? vmul(NL, S0) : S0, Z);
  };
  Coef<T> e0, e1;
  Rec<T> r;
  load_coef(a, e0);
  for (int t = (fin ? n - 1 : n) >> 1; t > 0; --t, a += 2 * ES) {
    load_rec(a, r);
    load_coef(a + ES, e1);
    acc(e0, D0, D1, r.NL);
    step_into<T, FULL, true>(r, X, NS, none, D0, D1, u, P0, P1, u);
    load_rec(a + ES, r);
    load_coef(a + 2 * ES, e0);
    acc(e1, P0, P1, r.NL);
    step_into<T, FULL, true>(r, X, NS, none, P0, P1, u, D0, D1, u);
  }
  if (!fin) return;
  v2<T> nl = none;
  if (!(n & 1)) {  // two degrees left
    load_rec(a, r);
    load_coef(a + ES, e1);
    acc(e0, D0, D1, r.NL);
    step_into<T, FULL, true>(r, X, NS, none, D0, D1, u, P0, P1, u);
    if (FULL) lds2(a + ES + (8 * STAGE_ENTRIES + 6) * sizeof(T), nl);
    acc(e1, P0, P1, nl);
  } else {
    if (FULL) lds2(a + (8 * STAGE_ENTRIES + 6) * sizeof(T), nl);
    acc(e0, D0, D1, nl);
  }
}

// group_sum for the rescaled states of group_seed_rs, with a recurrence for d''
// (D2, P2): the true d, d', d'' of half h are the states times 2^E_h.  Each
// accumulation multiplies the state by SC = 2^E (0 while the true values are
// below 2^-126); after each step a half whose state has grown past 2^32 while
// E_h < 0 is scaled down by 2^32 (exactly) and E_h raised by 32, so the states
// neither overflow nor lose the digits of seeds far below the FP32 range
// (per-degree rescaling).
struct Scaled {
  v2<float> D0, D1, D2, P0, P1, P2, SC;
  int E0, E1;
};
__device__ __forceinline__ void rescale_half(float &p0, float &p1, float &p2, float &d0, float &d1,
                                             float &d2, int &E, float &sc) {
  const float f = 2.3283064365386963e-10f;  // 2^-32
  p0 *= f; p1 *= f; p2 *= f; d0 *= f; d1 *= f; d2 *= f;
  E += 32;
  sc = pow2f(E);
}

template <bool FULL>
__device__ __forceinline__ void group_sum_rs(unsigned a, int n, bool fin, v2<float> X, v2<float> NS,
                                             v2<float> NX, Scaled &s, v2<float> (&Z)[12]) {
  constexpr unsigned ES = 8 * sizeof(float);
  constexpr float BIG = 4294967296.f;
  Coef<float> e;
  Rec<float> r;
  auto acc = [&](const v2<float> &S0, const v2<float> &S1, const v2<float> &S2) {
    accumulate<float, FULL>(e, vmul(S0, s.SC), FULL ? vmul(S1, s.SC) : S1, FULL ? vmul(S2, s.SC) : S2, Z);
  };
  // one step from (A) into (B)
  auto step = [&](v2<float> &A0, v2<float> &A1, v2<float> &A2, v2<float> &B0, v2<float> &B1, v2<float> &B2) {
    step_into<float, FULL>(r, X, NS, NX, A0, A1, A2, B0, B1, B2);
    if (fmaxf(fabsf(B0.x), fabsf(B0.y)) > BIG) {
      if (s.E0 < 0 && fabsf(B0.x) > BIG) rescale_half(B0.x, B1.x, B2.x, A0.x, A1.x, A2.x, s.E0, s.SC.x);
      if (s.E1 < 0 && fabsf(B0.y) > BIG) rescale_half(B0.y, B1.y, B2.y, A0.y, A1.y, A2.y, s.E1, s.SC.y);
    }
  };
  for (int t = (fin ? n - 1 : n) >> 1; t > 0; --t, a += 2 * ES) {
    load_coef(a, e);
    load_rec(a, r);
    acc(s.D0, s.D1, s.D2);
    step(s.D0, s.D1, s.D2, s.P0, s.P1, s.P2);
    load_coef(a + ES, e);
    load_rec(a + ES, r);
    acc(s.P0, s.P1, s.P2);
    step(s.P0, s.P1, s.P2, s.D0, s.D1, s.D2);
  }
  if (!fin) return;
  load_coef(a, e);
  acc(s.D0, s.D1, s.D2);
  if (n & 1) return;
  load_rec(a, r);
  step(s.D0, s.D1, s.D2, s.P0, s.P1, s.P2);
  load_coef(a + ES, e);
  acc(s.P0, s.P1, s.P2);
}

// The sums of one image of both halves for one candidate, written to o (rows of
// `row` bytes): the image has phase E = e^{i(u a + v g)}; zr0 + i zi0 = S0 E, zr1 + i
// zi1 = S1 E, zr2 = Re S2 E for the d, d', d'' sums S0, S1, S2 (zr0 only when !FULL).
template <typename T, bool FULL>
__device__ __forceinline__ void put_image(unsigned o, unsigned row, const v2<T> &ER, const v2<T> &EI,
                                          const v2<T> &S0r, const v2<T> &S0i, const v2<T> &S1r,
                                          const v2<T> &S1i, const v2<T> &S2r, const v2<T> &S2i) {
  const v2<T> NEI = vset<T>(-EI.x, -EI.y);
  sts2(o, vfma(S0r, ER, vmul(S0i, NEI)));
  if (FULL) {
    sts2(o + row, vfma(S0r, EI, vmul(S0i, ER)));
    sts2(o + 2 * row, vfma(S1r, ER, vmul(S1i, NEI)));
    sts2(o + 3 * row, vfma(S1r, EI, vmul(S1i, ER)));
    sts2(o + 4 * row, vfma(S2r, ER, vmul(S2i, NEI)));
  }
}

// Adds one image of both halves to the candidate's sums.  The image has phase
// E = e^{i(u a + v g)} and weight W; (zr0, zi0) = S0 E, (zr1, zi1) = S1 E,
// zr2 = Re S2 E for the d, d', d'' sums S0, S1, S2.  d/da brings i u and d/dg
// brings i v, so with AU = -W u, GV = -W v:
//   C += W zr0, C_a += AU zi0, C_b += W zr1, C_g += GV zi0,
//   C_aa += AU u zr0, C_ab += AU zi1, C_ag += AU v zr0, C_bb += W zr2,
//   C_bg += GV zi1, C_gg += GV v zr0.
// w: shared address of the weights (W, AU, GV, AU u, AU v, GV v as pairs, exact
// integers made once per plan).
template <typename T, bool FULL>
__device__ __forceinline__ void add_image(v2<T> (&acc)[10], unsigned w, const v2<T> &ER,
                                          const v2<T> &EI, const v2<T> &S0r, const v2<T> &S0i,
                                          const v2<T> &S1r, const v2<T> &S1i, const v2<T> &S2r,
                                          const v2<T> &S2i) {
  const v2<T> NEI = vset<T>(-EI.x, -EI.y);
  v2<T> W, AU;
  lds4(w, W, AU);
  const v2<T> zr0 = vfma(S0r, ER, vmul(S0i, NEI));
  acc[0] = vfma(W, zr0, acc[0]);
  if (FULL) {
    v2<T> GV, AUU, AUV, GVV;
    lds4(w + 4 * sizeof(T), GV, AUU);
    lds4(w + 8 * sizeof(T), AUV, GVV);
    const v2<T> zi0 = vfma(S0r, EI, vmul(S0i, ER));
    const v2<T> zr1 = vfma(S1r, ER, vmul(S1i, NEI));
    const v2<T> zi1 = vfma(S1r, EI, vmul(S1i, ER));
    const v2<T> zr2 = vfma(S2r, ER, vmul(S2i, NEI));
    acc[1] = vfma(AU, zi0, acc[1]);
    acc[2] = vfma(W, zr1, acc[2]);
    acc[3] = vfma(GV, zi0, acc[3]);
    acc[4] = vfma(AUU, zr0, acc[4]);
    acc[5] = vfma(AU, zi1, acc[5]);
    acc[6] = vfma(AUV, zr0, acc[6]);
    acc[7] = vfma(W, zr2, acc[7]);
    acc[8] = vfma(GV, zi1, acc[8]);
    acc[9] = vfma(GVV, zr0, acc[9]);
  }
}

// Phase of both halves: E_h = (ar_h + i ai_h)(gr_h + i gi_h), scalar (the
// factors come as single table values).
template <typename T>
__device__ __forceinline__ void phase(T ar0, T ai0, T ar1, T ai1, T gr0, T gi0, T gr1, T gi1,
                                      v2<T> &ER, v2<T> &EI) {
  ER.x = sfma(ar0, gr0, smul(-ai0, gi0));
  ER.y = sfma(ar1, gr1, smul(-ai1, gi1));
  EI.x = sfma(ar0, gi0, smul(ai0, gr0));
  EI.y = sfma(ar1, gi1, smul(ai1, gr1));
}

// All CTAs of the particle's cluster (or the one CTA).
__device__ __forceinline__ void particle_sync(const SpreadArgs &A) {
  if (A.ctas > 1) cooperative_groups::this_cluster().sync();
  else __syncthreads();
}

// Evaluates C (and grad, Hessian when FULL) at pts[p] for the candidates with
// need[p] != 0; results in res[p][0..9] (FP64) of every CTA of the particle.
// Called by all of them.
// SPLIT (32-bit plans): W workers per chain group and z in shared memory; else (FP64)
// one, which adds its groups' images to accumulators in registers.
template <typename T, bool FULL, bool RS, bool SPLIT>
__device__ __forceinline__ void evaluate(const SpreadArgs &A, int L, const T *__restrict__ cb,
                                         const T *__restrict__ rcoef, const T *__restrict__ gdesc,
                                         const double *pts, const Smem &sm) {
  constexpr unsigned z = sizeof(T);
  // copies: a field read through the reference again would be a load each time
  const int P = A.P, spw = A.spw, LJ = A.LJ, allrounds = A.nrounds, ctas = A.ctas;
  const int W = SPLIT ? A.W : 1, chunk = SPLIT ? A.chunk : 1 << 20;
  const int NPW = pw_row(LJ), RW = ph_row(LJ), PS = cand_stride(P);
  T *ph = sm.ph<T>();    // [4][RW][PS]: cos k a, sin k a, cos k g, sin k g
  T *pw = sm.pw<T>();    // [2][NPW][PS]: PW_PAD zeros, then ch^k (sh^k), k = 0..2LJ+3
  T *tg = sm.trig<T>();  // [TRIG][PS]
  const int *need = sm.need();
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int rank = ctas > 1 ? (int)cooperative_groups::this_cluster().block_rank() : 0;
  const int grp = warp / W, wk = warp - grp * W;  // chain group in the CTA, worker
  const int sub = min(lane / P, spw - 1);
  const int p = lane - sub * P;                   // candidate; lanes past the last sub-slot: p >= P
  const int slot0 = rank * A.cpc * spw;           // first sub-slot of the CTA
  const int slot = slot0 + grp * spw + sub;
  const int nslots = A.nslots;
  const unsigned stage = smem_u32(sm.base + A.o_stage) + z * STAGE_SUB<T> * (warp * STAGE_SLOTS * spw);
  const int pc = p < P ? p : 0;

  // ---- staging.  Sub-slot `slot` takes group k * nslots + slot in even rounds k
  // and k * nslots + (nslots - 1 - slot) in odd ones: groups come in increasing g
  // (non-increasing length), so the alternating order balances the sub-slots
  // while keeping every sum's order fixed; this warp stages and sums rounds wk,
  // wk + W, ...  The plan's schedule lists, per sub-slot, each round's (order m,
  // first entry, group, smallest order of the chain group's groups); a group of
  // order m has L - m + 1 degrees, none past L.
  constexpr int CH = 16 / (int)z;                  // reals per copy
  constexpr int CE = 8 / CH;                       // copies per entry and kind
  const int4 *sched = A.sched + (slot < nslots ? slot : nslots - 1) * allrounds;
  const bool idle = slot >= nslots;                // a sub-slot without groups
  const int ng = (L + 1) * (L + 2) / 2, nrounds = (ng + nslots - 1) / nslots;  // rounds at L
  const bool works = slot0 + grp * spw < nslots;   // the warp has a sub-slot
  auto slot_at = [&](int i) { return stage + z * STAGE_SUB<T> * (i * spw + sub); };
  int ki = wk, ei = 0;  // next piece to issue: its round and first degree entry
  int4 round = sched[min(ki, allrounds - 1)];
  // Issues the next piece into ring slot i.
  auto issue = [&](int i) {
    if (works && ki < nrounds) {
      const int longest = L + 1 - round.w - ei;  // degrees left of the longest group
      const bool exists = !idle && round.x <= L;
      const int have = exists ? CE * (L + 1 - round.x - ei) : 0;
      const int want = CE * min(longest, STAGE_ENTRIES);
      if (p < P) {
        unsigned dst = slot_at(i) + 16 * p;
        const T *ds = gdesc + GROUP_DESC * round.z + CH * p;
        for (int x = p; x <= GROUP_DESC / CH; x += P, dst += 16 * P, ds += CH * P) {
          if (x < GROUP_DESC / CH) cp_async16(dst, ds, exists);
          else cp_async16(dst, sched + ki, true);
        }
        dst = slot_at(i) + z * STAGE_HEAD<T> + 16 * p;
        const int o = 8 * (round.y + ei) + CH * p;
        const T *cs = cb + o, *rs = rcoef + o;
        for (int x = p; x < want; x += P, dst += 16 * P, cs += CH * P, rs += CH * P) {
          cp_async16(dst, cs, x < have);
          cp_async16(dst + z * 8 * STAGE_ENTRIES, rs, x < have);
        }
      }
      if (longest > STAGE_ENTRIES) {
        ei += STAGE_ENTRIES;
      } else if (longest > 0) {  // past the last group the schedule entry alone is copied
        ei = 0;
        ki += W;
        if (ki < nrounds) round = sched[ki];
      }
    }
    cp_async_commit();
  };
#pragma unroll
  for (int i = 0; i < STAGE_SLOTS - 1; ++i) issue(i);

  // ---- tables.  Trigonometric values of the needed candidates first: item
  // (candidate, b/2 | a | g | b).
  for (int t = tid; t < 4 * P; t += blockDim.x) {
    const int q = t >> 2, w = t & 3;
    if (!need[q]) continue;
    const T bt = (T)pts[3 * q + 1];
    const T x = w == 0 ? bt * T(0.5) : w == 3 ? bt : (T)pts[3 * q + 2 * (w - 1)];
    const T c = tcos(x), s = tsin(x);
    T *o = tg + 2 * w * PS + q;
    o[0] = c;
    o[PS] = s;
    if (w == 3) {
      const T sfl = sizeof(T) == 8 ? T(1e-150) : T(1e-18);
      const T se = s > sfl ? s : sfl;
      o[2 * PS] = T(1) / (se * se);
      o[3 * PS] = -c / se;
    }
  }
  __syncthreads();
  // powers k = 0..2L+3 of cos(beta/2) and sin(beta/2): runs of 8 consecutive
  // powers per item, the first by binary powering, the rest by one product each
  constexpr int RUN = 8;
  const int npk = 2 * L + 4, nrun = (npk + RUN - 1) / RUN;
  const FastDiv dw(nrun);
  for (int t = tid; t < 2 * P * nrun; t += blockDim.x) {
    int pr = dw.div(t), k0 = (t - pr * nrun) * RUN;
    int q = pr >> 1, which = pr & 1;
    if (!need[q]) continue;
    const T x = tg[which * PS + q];
    const int k1 = min(k0 + RUN, npk);
    if (RS) {  // mantissa rows, then exponent rows (2 NPW rows further on)
      for (int kk = k0; kk < k1; ++kk) {
        float mt;
        int ex;
        xpow((float)x, kk, mt, ex);
        pw[(which * NPW + PW_PAD + kk) * PS + q] = (T)mt;
        pw[((2 + which) * NPW + PW_PAD + kk) * PS + q] = (T)ex;
      }
    } else {
      T v = ipow_t(x, k0);
      T *o = pw + (which * NPW + PW_PAD + k0) * PS + q;
      o[0] = v;
      for (int kk = k0 + 1; kk < k1; ++kk) {
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
    const int pq = t >> 3, q = t & 7, cp = pq >> 1, which = pq & 1;
    if (need[cp]) {
      const T c1 = tg[(2 + 2 * which) * PS + cp], s1 = tg[(3 + 2 * which) * PS + cp];
      T *cr_ = ph + ((2 * which) * RW + LJ) * PS + cp, *ci_ = cr_ + RW * PS;
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

  const T xb = tg[6 * PS + pc], sb = tg[7 * PS + pc];
  const v2<T> X = vset<T>(xb, xb), NS = vset<T>(-sb, -sb), NX = vset<T>(-xb, -xb);
  // constants of the differential equation for d'' (the non-rescaled path):
  // 1/sin^2 b, -cot b, and the pole form of the numerator of Q
  // (+4 sin^2(b/2) or -4 cos^2(b/2))
  const bool north = xb >= T(0);
  const T is2 = tg[8 * PS + pc], ncot = tg[9 * PS + pc];
  T qc4;
  {
    const T chb = tg[pc], shb = tg[PS + pc];
    qc4 = north ? T(4) * shb * shb : T(-4) * chb * chb;
  }
  // shared addresses of this candidate's tables (index 0 of each row)
  const unsigned zs = z * PS;  // bytes between consecutive positions of a row
  const unsigned pcu = smem_u32(pw + PW_PAD * PS + pc);
  const unsigned psu = pcu + zs * NPW;
  const unsigned eacu = smem_u32(ph + LJ * PS + pc);  // k = 0 of cos k a
  const unsigned row = zs * RW;                        // cos k a -> sin k a -> cos k g -> sin k g
  // ---- accumulators of this lane's sub-slot and candidate: quantities wk, wk + W, ...
  const int nsub = A.cpc * spw, zrow = z_row(P), nq = FULL ? 10 : 1;
  T *zb = sm.z<T>();
  constexpr int NACC = SPLIT ? 5 : 10;
  v2<T> acc[NACC];
#pragma unroll
  for (int j = 0; j < NACC; ++j) acc[j] = vset<T>(T(0), T(0));
  // the sub-slot's rounds at L: the last one may have no group for it
  const int kl = nrounds - 1;
  const int mine = slot < nslots ? nrounds - (kl * nslots + ((kl & 1) ? nslots - 1 - slot : slot) >= ng ? 1 : 0) : 0;

  // a group's state, kept between its pieces
  v2<T> D0, D1, P0, P1, Z[12];
  Scaled S;
  int ring = 0;
  for (int k0 = 0, buf = 0; k0 < nrounds; k0 += chunk, buf ^= 1) {
    for (int k = k0 + wk; works && k < min(k0 + chunk, nrounds); k += W) {
      const unsigned zo = smem_u32(zb + ((buf * chunk + k - k0) * nsub + grp * spw + sub) * zrow + 2 * pc);
      for (int e = 0;; e += STAGE_ENTRIES) {
        issue(ring == 0 ? STAGE_SLOTS - 1 : ring - 1);  // the slot summed last
        cp_async_wait<STAGE_SLOTS - 1>();
        __syncwarp();
        const unsigned dsc = slot_at(ring), ent = dsc + z * STAGE_HEAD<T>;
        // the longest of the warp's groups sets the degrees of all (missing ones, or
        // an absent group, are zeros)
        const int left = L + 1 - lds_int(dsc + z * GROUP_DESC + 12) - e;
        if (left <= 0) break;  // no group in this round (the last one)
        const bool fin = left <= STAGE_ENTRIES;
        const int n = fin ? left : STAGE_ENTRIES;
        const int m = lds_int(dsc + z * 14), na = lds_int(dsc + z * 15);
        if (e == 0) {
          const v2<T> zero = vset<T>(T(0), T(0));
#pragma unroll
          for (int q = 0; q < 12; ++q) Z[q] = zero;
          const unsigned pa = pcu + zs * (m + na), pb = psu + zs * (m - na);
          if constexpr (RS) {
            v2<T> GK, GH;
            lds4(dsc, GK, GH);
            group_seed_rs<FULL>(pa, pb, zs * 2 * NPW, zs, vset<T>(GK.x, -GK.y), m + na, m - na, S.D0,
                                S.D1, S.D2, S.E0, S.E1);
            S.P0 = S.P1 = S.P2 = zero;
            S.SC = vset<T>(pow2f(S.E0), pow2f(S.E1));
          } else {
            group_seed<T, FULL>(pa, pb, zs, dsc, D0, D1);
            P0 = P1 = zero;
          }
        }
        if constexpr (RS) group_sum_rs<FULL>(ent, n, fin, X, NS, NX, S, Z);
        else group_sum<T, FULL>(ent, n, fin, X, NS, D0, D1, P0, P1, Z);
        if (fin) {
          if (!RS && FULL) {
            // d'' = -cot(b) d' + (Q - l(l+1)) d with Q = (m^2 + n^2 - 2mn cos b) / sin^2 b,
            // the numerator as (m - n)^2 + 4mn sin^2(b/2) (beta <= pi/2) or
            // (m + n)^2 - 4mn cos^2(b/2) (beta > pi/2), free of cancellation at the pole
            v2<T> mn, sqn, sqs, none;
            lds4(dsc + 8 * z, mn, sqn);
            lds4(dsc + 12 * z, sqs, none);
            const v2<T> sq = vset<T>(north ? sqn.x : sqs.x, north ? sqn.y : sqs.y);
            const v2<T> Q = vset<T>(smul(sfma(mn.x, qc4, sq.x), is2), smul(sfma(mn.y, qc4, sq.y), is2));
            const v2<T> NCOT = vset<T>(ncot, ncot);
#pragma unroll
            for (int q = 0; q < 4; ++q) Z[8 + q] = vfma(NCOT, Z[4 + q], vfma(Q, Z[q], Z[8 + q]));
          }
          const unsigned am = eacu + zs * m, an = eacu + zs * na;
          T amr, ami, gmr, gmi, ar0, ai0, ar1, ai1, gr0, gi0, gr1, gi1;
          lds1(am, amr); lds1(am + row, ami); lds1(am + 2 * row, gmr); lds1(am + 3 * row, gmi);
          lds1(an, ar0); lds1(an + row, ai0); lds1(an + 2 * row, gr0); lds1(an + 3 * row, gi0);
          lds1(an + zs, ar1); lds1(an + zs + row, ai1); lds1(an + zs + 2 * row, gr1);
          lds1(an + zs + 3 * row, gi1);
          v2<T> ER, EI;
          // image (m, n): phase e^{i(m a + n g)}, weight 1 for (0, 0) else 2
          // (the image (-m, -n) is the conjugate); an empty half has weight 0
          phase<T>(amr, ami, amr, ami, gr0, gi0, gr1, gi1, ER, EI);
          const unsigned zr = 2 * z * P;
          if constexpr (!SPLIT)
            add_image<T, FULL>(acc, dsc + 16 * z, ER, EI, Z[0], Z[1], Z[4], Z[5], Z[8], Z[9]);
          else if (p < P)
            put_image<T, FULL>(zo, zr, ER, EI, Z[0], Z[1], Z[4], Z[5], Z[8], Z[9]);
          // image (n, m): c^l_nm d^l_nm e^{i(n a + m g)}, d^l_nm = (-1)^{m-n} d^l_mn
          // (m - n even in the first half, odd in the second); absent when n = +-m
          phase<T>(ar0, ai0, ar1, ai1, gmr, gmi, gmr, gmi, ER, EI);
          if constexpr (!SPLIT) {
            add_image<T, FULL>(acc, dsc + 28 * z, ER, EI, Z[2], Z[3], Z[6], Z[7], Z[10], Z[11]);
          } else if (p < P) {
            put_image<T, FULL>(zo + 5 * zr, zr, ER, EI, Z[2], Z[3], Z[6], Z[7], Z[10], Z[11]);
            for (int x = p; x < 12; x += P) {
              v2<T> w;
              lds2(dsc + z * (16 + 2 * x), w);
              sts2(zo + 2 * z * (10 * P + x - p), w);
            }
          }
        }
        __syncwarp();
        ring = ring == STAGE_SLOTS - 1 ? 0 : ring + 1;
        if (fin) break;
      }
    }
    if constexpr (!SPLIT) break;
    __syncthreads();
    // the chunk's rounds in order, image (m, n) before (n, m); the other buffer takes
    // the next chunk meanwhile
    const unsigned zc = smem_u32(zb + (buf * chunk * nsub + grp * spw + sub) * zrow), zs1 = z * nsub * zrow;
    const int nk = min(chunk, mine - k0);
#pragma unroll
    for (int j = 0; j < 5; ++j) {
      const int i = wk + j * W;  // C, a, b, g, aa, ab, ag, bb, bg, gg
      if (i >= nq) break;
      const int wi = (int)((0x5204132010ull >> (4 * i)) & 15), zi = (int)((0x0340301210ull >> (4 * i)) & 15);
      unsigned zp = zc + 2 * z * (zi * P + pc), wp = zc + 2 * z * (10 * P + wi);
      for (int k = 0; k < nk; ++k, zp += zs1, wp += zs1) {
        v2<T> z1, z2, w1, w2;
        lds2(wp, w1);
        lds2(zp, z1);
        lds2(wp + 12 * z, w2);
        lds2(zp + 10 * z * P, z2);
        acc[j] = vfma(w1, z1, acc[j]);
        acc[j] = vfma(w2, z2, acc[j]);
      }
    }
  }
  cp_async_wait<0>();
  // both halves of each chain to every CTA of the particle (two buffers in turn,
  // since a CTA may still read the previous evaluation's), then the pairs of
  // sub-slots and the pairs in index order: all in the working precision
  T *red = sm.red<T>();
  if (ctas > 1) red += *sm.turn() * nslots * P * 10;
  if (p < P && slot < nslots)
#pragma unroll
    for (int j = 0; j < NACC; ++j) {
      const int i = wk + j * W;
      if (i >= nq) break;
      const T v = acc[j].x + acc[j].y;
      T *o = red + (slot * P + p) * 10 + i;
      for (int d = 0; d < ctas; ++d)
        *(ctas > 1 ? cooperative_groups::this_cluster().map_shared_rank(o, d) : o) = v;
    }
  particle_sync(A);
  if (tid == 0) *sm.turn() ^= 1;
  for (int idx = tid; idx < P * nq; idx += blockDim.x) {
    const int pp = idx / nq, i = idx - pp * nq;
    if (!need[pp]) continue;
    const T *x = red + pp * 10 + i;
    T v = 0;
    for (int s = 0; s < nslots; s += A.pairs ? 2 : 1) {
      T y = x[s * P * 10];
      if (A.pairs && s + 1 < nslots) y += x[(s + 1) * P * 10];
      v += y;
    }
    sm.res()[pp * 10 + i] = (double)v;
  }
  __syncthreads();
}

// Zeroes the power tables (their pads stay zero) and, in a cluster, waits until
// all CTAs of the particle have started (they write to each other's sums).
template <typename T, bool RS>
__device__ __forceinline__ void init_smem(const Smem &sm) {
  const SpreadArgs &A = sm.A;
  for (int t = threadIdx.x; t < (RS ? 4 : 2) * cand_stride(A.P) * pw_row(A.LJ); t += blockDim.x)
    sm.pw<T>()[t] = T(0);
  if (threadIdx.x == 0) *sm.turn() = 0;
  particle_sync(A);
}

// C_L, its gradient and Hessian at Q given rotations per particle (k_objective of
// newton.cu).
template <typename T, bool RS, bool SPLIT>
__global__ void __launch_bounds__(SPREAD_THREADS, sizeof(T) == 8 ? 1 : 2)
k_objective_spread(const T *__restrict__ c, const T *__restrict__ rcoef, const T *__restrict__ gdesc,
                   const __grid_constant__ SpreadArgs A, int L, int Q, const double *__restrict__ pts,
                   double *__restrict__ out) {
  const long b = blockIdx.x / A.ctas;
  const int tid = threadIdx.x;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const Smem sm{A, smem_raw};
  init_smem<T, RS>(sm);
  if (tid < A.P) {
    const bool on = tid < Q;
    for (int i = 0; i < 3; ++i) sm.th()[3 * tid + i] = on ? pts[3 * (b * Q + tid) + i] : 0.0;
    sm.need()[tid] = on;
  }
  __syncthreads();
  evaluate<T, true, RS, SPLIT>(A, L, c + 4 * b * A.nc, rcoef, gdesc, sm.th(), sm);
  if (blockIdx.x % A.ctas == 0)
    for (int t = tid; t < Q * 10; t += blockDim.x) out[10 * b * Q + t] = sm.res()[t];
}

// The march of all candidates of one particle (k_newton of newton.cu).
template <typename T, bool RS, bool SPLIT>
__global__ void __launch_bounds__(SPREAD_THREADS, sizeof(T) == 8 ? 1 : 2)
k_newton_spread(const T *__restrict__ c, const T *__restrict__ rcoef, const T *__restrict__ gdesc,
                const __grid_constant__ SpreadArgs A, const int *__restrict__ n_cand,
                double *__restrict__ euler, double *__restrict__ score, int *__restrict__ cflags,
                long long *__restrict__ work) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const Smem sm{A, smem_raw};
  init_smem<T, RS>(sm);
  const long b = blockIdx.x / A.ctas;
  const int P = A.P, tid = threadIdx.x;
  const int nc_b = n_cand[b];
  if (tid < P) {
    const double *e = euler + 3 * (b * P + tid);
    for (int i = 0; i < 3; ++i) sm.th()[3 * tid + i] = e[i];
    sm.state()[tid] = tid < nc_b ? ST_RUN : ST_DEAD;
    sm.fl()[tid] = 0;
    sm.Cc()[tid] = __longlong_as_double(0x7ff8000000000000LL);
  }
  if (tid == 0) sm.work()[0] = sm.work()[1] = 0;
  // the start points are read by every CTA before the first one may write results
  particle_sync(A);
  const T *cb = c + 4 * b * A.nc;
  const double piv_rel = sizeof(T) == 8 ? 1e-12 : 1e-6;  // H summed in T
  // Trials are evaluated with derivatives except on a level's last step (newton.cu);
  // round -1 of a level is the evaluation at its start point.
  bool alive = true;
  for (int lev = 0; lev < A.nlev && alive; ++lev) {
    const int L = A.Ls[lev];
    for (int round = -1; round < 3 * A.M; ++round) {
      const bool start = round < 0;
      int tw = 0, wf = 0;
      if (tid < P) {
        tw = start ? sm.state()[tid] != ST_DEAD : sm.state()[tid] == ST_TRIAL;
        wf = tw && (start || sm.steps()[tid] < A.M - 1);
        sm.need()[tid] = tw;
      }
      if (!__syncthreads_or(tw)) {
        alive = !start;
        break;
      }
      const bool full = __syncthreads_or(wf);
      if (tid == 0) {
        // recurrence steps of one evaluation: sum_{m<=L} (2m+1)(L-m+1)
        const long long steps_L = (long long)(L + 1) * (L + 2) * (2 * L + 3) / 6;
        for (int q = 0; q < P; ++q) sm.work()[full ? 0 : 1] += sm.need()[q] ? steps_L : 0;
      }
      const double *pts = start ? sm.th() : sm.tr();
      if (full) evaluate<T, true, RS, SPLIT>(A, L, cb, rcoef, gdesc, pts, sm);
      else evaluate<T, false, RS, SPLIT>(A, L, cb, rcoef, gdesc, pts, sm);
      if (tid < P && sm.need()[tid])
        after_evaluation<T>(tid, L, start, lev == A.nlev - 1, A.M, A.tol, A.acc_tol, A.grad != 0,
                            StepState(sm), piv_rel);
    }
    __syncthreads();
  }
  if (blockIdx.x % A.ctas) return;
  if (tid < P) {
    const long o = b * P + tid;
    if (tid < nc_b) {
      for (int i = 0; i < 3; ++i) euler[3 * o + i] = sm.th()[3 * tid + i];
      score[o] = sm.Cc()[tid];
    }
    cflags[o] = sm.fl()[tid];
  }
  if (tid == 0 && work) {
    work[2 * b] = sm.work()[0];
    work[2 * b + 1] = sm.work()[1];
  }
}

// Sub-slots of a chain group: as many as P lanes each fit in a warp.
int spread_spw(const Plan &p, int nslots) { return std::min(32 / p.P, nslots); }

// Lays out the shared memory of a CTA; returns its size.
size_t spread_smem(const Plan &p, size_t tsize, SpreadArgs &A) {
  const size_t P = p.P, PS = cand_stride(p.P), nsub = (size_t)A.cpc * A.spw;
  size_t o = (8 * (20 * P + 2) + 4 * (5 * P + 1) + 15) / 16 * 16;
  auto take = [&](size_t reals) {
    const size_t at = o;
    o = (o + tsize * reals + 15) / 16 * 16;
    return (int)at;
  };
  A.o_red = take((A.ctas > 1 ? 2 : 1) * 10 * P * A.nslots);
  A.o_z = take(A.W > 1 ? 2 * A.chunk * nsub * z_row(p.P) : 0);
  A.o_trig = take(TRIG * PS);
  A.o_ph = take(4 * PS * ph_row(p.LJ));
  A.o_pw = take((newton_rescaled(p) ? 4 : 2) * PS * pw_row(p.LJ));
  A.o_stage = take((size_t)A.cpc * A.W * STAGE_SLOTS * A.spw *
                   (tsize == 8 ? STAGE_SUB<double> : STAGE_SUB<float>));
  return o;
}

// The shape for B particles, or false where one CTA per particle is as fast.
//
// FP64: one worker per chain group, and a shape for every plan (one chain group per CTA
// fits wherever the plan's refinement does).  An SM's FP64 pipe is full from about four of
// these warps on (40 particles to L = 32: 8.1 ms at eight warps per SM, 4.5 at
// four, 4.4 at two), so a wave of resident CTAs costs max(4, its warps); one CTA
// per particle, 9.0 ms, is never faster.
//
// 32-bit plans: several workers per chain group, worth it only while SMs are
// idle.  In units of one CTA per particle alone on its SM, W workers take
// a + f (1 - a) / W, where a, the share of the tables and the step rule, falls
// with the entries per sub-slot (560 / (700 + entries)) and f is 1.3 with eight
// warps on an SM, 1.6 with sixteen (eight particles of 16 candidates: to L = 16 141 us,
// W = 4 119, W = 8 114; L = 32 242, 153, 138; L = 64 822, 332, 245; L = 100 8.73 ms,
// 2.50, 1.58).  One CTA per particle takes 1 per wave of one CTA per SM and 1.5
// with two (96 and 304 particles: 500, 760 us).
//
// A wave holds as many clusters as run at once (clusters_at_once), not its share of the
// SMs: 76 particles to L = 48 in clusters of four, two waves of SMs but three of
// clusters, took 653 us against 448 as single CTAs.
bool spread_shape(const Plan &p, size_t tsize, int B, SpreadArgs &out, size_t *smem) {
  SpreadArgs A = {};
  A.LJ = p.LJ; A.nlev = p.nlev; A.M = p.M; A.P = p.P;
  A.nslots = newton_slots(p);
  if (A.nslots == 0) return false;
  for (int i = 0; i < MATCHA_MAX_LEVELS; ++i) A.Ls[i] = i < p.nlev ? p.Ls[i] : 0;
  A.tol = p.step_tol; A.acc_tol = p.accept_tol; A.grad = p.refine; A.nc = p.nc;
  A.sched = p.sched;
  A.nrounds = p.nrounds;
  A.spw = spread_spw(p, A.nslots);
  A.ngrp = (A.nslots + A.spw - 1) / A.spw;
  A.pairs = p.P <= 16;
  const bool fp64 = tsize == 8;
  const long sm_bytes = 228 * 1024, most = 227 * 1024, reg_warps = fp64 ? 8 : 16, sms = p.sms;
  const double entries = (double)p.nc / 2 / A.nslots, a = 560 / (700 + entries);
  const long one = std::max(1L, std::min<long>(sm_bytes / (long)(newton_smem(p) + 1024), reg_warps / 8));
  double best = fp64 ? 1e30 : 0.95 * (B <= sms ? 1 : ((B + one * sms - 1) / (one * sms)) * (one > 1 ? 1.5 : 1));
  bool found = false;
  for (int W = fp64 ? 1 : 4; W <= (fp64 ? 1 : 8); W *= 2)
    for (int cpc = std::min(8 / W, A.ngrp); cpc >= 1; --cpc) {
      A.W = W;
      A.cpc = cpc;
      A.ctas = (A.ngrp + cpc - 1) / cpc;
      if ((A.ngrp + A.ctas - 1) / A.ctas != cpc) continue;  // fewer per CTA at the same count
      A.chunk = 8;
      size_t bytes = spread_smem(p, tsize, A);
      if (W == 4 && 2 * bytes > (size_t)sm_bytes - 2048) {
        A.chunk = 4;
        bytes = spread_smem(p, tsize, A);
      }
      if ((long)bytes > most) continue;
      const long resident = std::max(1L, std::min<long>(sm_bytes / (long)(bytes + 1024), reg_warps / (cpc * W)));
      const long n = (long)B * A.ctas, held = clusters_at_once(p, (int)resident, A.ctas), waves = (B + held - 1) / held;
      const long per_sm = std::min(resident, (n + sms - 1) / sms), warps = per_sm * cpc * W;
      const double t = fp64 ? waves * std::max(4.0, (double)per_sm * cpc)
                            : waves * (a + (1 - a) / W * (warps > 8 ? 1.6 : warps > 4 ? 1.3 : 1));
      if (t < best) {
        best = t;
        out = A;
        *smem = bytes;
        found = true;
      }
    }
  return found;
}

template <typename... Args>
cudaError_t launch_clusters(void (*kern)(Args...), int B, const SpreadArgs &A, size_t smem,
                            cudaStream_t st, Args... args) {
  const cudaError_t e = allow_smem(kern, smem);
  if (e != cudaSuccess) return e;
  cudaLaunchConfig_t cfg = {};
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = A.ctas;
  at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
  cfg.gridDim = dim3((unsigned)(B * A.ctas));
  cfg.blockDim = dim3(32 * A.cpc * A.W);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cfg.attrs = at;
  cfg.numAttrs = A.ctas > 1 ? 1 : 0;
  return cudaLaunchKernelEx(&cfg, kern, args...);
}

}  // namespace

// The sub-slots' rounds at the plan's L_J, [slot][round]: (order m of the
// sub-slot's group, L_J + 1 past the last group; its first (group, l) entry; its
// index; the smallest order of the groups of the sub-slots that share its warp).
int newton_schedule(const Plan &p, std::vector<int4> &out) {
  const int ns = newton_slots(p), spw = spread_spw(p, ns);
  const int rounds = (p.ngroups + ns - 1) / ns;
  out.assign((size_t)ns * rounds, int4{p.LJ + 1, 0, 0, p.LJ + 1});
  std::vector<int> order(p.ngroups), first(p.ngroups);
  for (int m = 0, g = 0, e = 0; m <= p.LJ; ++m)
    for (int j = 0; j <= m; ++j, ++g, e += p.LJ - m + 1) { order[g] = m; first[g] = e; }
  for (int s = 0; s < ns; ++s)
    for (int k = 0; k < rounds; ++k) {
      const int g = k * ns + ((k & 1) ? ns - 1 - s : s);
      if (g < p.ngroups) out[(size_t)s * rounds + k] = int4{order[g], first[g], g, order[g]};
    }
  for (int s = 0; s < ns; ++s)
    for (int k = 0; k < rounds; ++k) {
      int4 &a = out[(size_t)s * rounds + k];
      for (int t = s / spw * spw; t < std::min(ns, s / spw * spw + spw); ++t)
        a.w = std::min(a.w, out[(size_t)t * rounds + k].x);
    }
  return rounds;
}

// False when one CTA per particle is expected to be as fast (32-bit plans).
template <typename T>
bool launch_newton_spread(const Plan &p, const T *c, int B, int batch, const int *n_cand, double *euler,
                          double *score, int *cflags, long long *work, cudaStream_t st, cudaError_t *e) {
  SpreadArgs A;
  size_t smem;
  if (!spread_shape(p, sizeof(T), batch, A, &smem)) return false;
  auto kern = k_newton_spread<T, false, sizeof(T) == 4>;
  if constexpr (sizeof(T) == 4)
    if (newton_rescaled(p)) kern = k_newton_spread<T, true, true>;
  *e = launch_clusters(kern, B, A, smem, st, c, (const T *)p.rcoef, (const T *)p.gdesc, A, n_cand, euler,
                       score, cflags, work);
  return true;
}
template bool launch_newton_spread<float>(const Plan &, const float *, int, int, const int *, double *,
                                          double *, int *, long long *, cudaStream_t, cudaError_t *);
template bool launch_newton_spread<double>(const Plan &, const double *, int, int, const int *, double *,
                                           double *, int *, long long *, cudaStream_t, cudaError_t *);

template <typename T>
bool launch_objective_spread(const Plan &p, const T *c, int B, int L, int Q, const double *pts,
                             double *out, cudaStream_t st, cudaError_t *e) {
  SpreadArgs A;
  size_t smem;
  if (!spread_shape(p, sizeof(T), B, A, &smem)) return false;
  auto kern = k_objective_spread<T, false, sizeof(T) == 4>;
  if constexpr (sizeof(T) == 4)
    if (newton_rescaled(p)) kern = k_objective_spread<T, true, true>;
  *e = launch_clusters(kern, B, A, smem, st, c, (const T *)p.rcoef, (const T *)p.gdesc, A, L, Q, pts, out);
  return true;
}
template bool launch_objective_spread<float>(const Plan &, const float *, int, int, int, const double *,
                                             double *, cudaStream_t, cudaError_t *);
template bool launch_objective_spread<double>(const Plan &, const double *, int, int, int, const double *,
                                              double *, cudaStream_t, cudaError_t *);

}  // namespace matcha
