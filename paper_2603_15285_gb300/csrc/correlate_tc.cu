// Step a3 on the tensor cores (tcgen05, sm_103a): the per-degree contraction
//   c^l_{mn} = sum_s w_s f_lm(r_s) conj(h_ln(r_s))                 (Eq. sigmalmm)
// as one real matrix product per (particle, degree pair {l, L-l}):
//   D[r][j] = sum_k A[r][k] B[j][k],   k < 2S (zero-padded to a multiple of 16),
// A row of degree d, order m >= 0:  (Re f_dm(r_0..r_{S-1}), Im f_dm(r_0..r_{S-1})),
// B rows of degree d, n = -d..d:    (w Re h_dn, w Im h_dn)   -> column of Re c^d_{mn},
//                                   (-w Im h_dn, w Re h_dn)  -> column of Im c^d_{mn},
// negative orders from h_{d,-n} = (-1)^n conj(h_dn) (real volumes).  Both
// degrees of the pair share one M = 128 tile (rows 0..l, then l+1..L+1) and
// one N tile (4(L+1) columns padded to 16), so one chain of MMAs covers the
// pair; the cross blocks are computed and never read.  Operands are TF32
// (cvt.rna) or BF16 (round to nearest) in shared memory, canonical K-major
// layout without swizzle (8-row x 16-byte core matrices, K-adjacent core
// matrices 128 bytes apart); the accumulator is FP32 in tensor memory.
//
// Persistent CTAs (two per SM, each holding 256 tensor-memory columns for its
// lifetime) walk the items (particle, degree pair) with two operand buffers:
// the operands of the next item are staged (generic stores, proxy fence)
// while the MMAs of the current one run; one thread issues the MMAs and
// commits them to an mbarrier; all threads wait on it with an iteration
// limit (on expiry: error bit, the CTA stops); warps 0-3 copy their
// accumulator lanes into the buffer the finished MMAs read; the next item's
// MMAs are issued; and the epilogue writes the grouped layout (see
// internal.cuh) while they run: c^l_{mn} from row m, c^l_{nm} from row n or,
// for n < 0, from (-1)^{m+n} conj of row -n.  That kernel serves a template per
// particle (and the sizes whose tile, table and operands do not fit beside one
// another); one template for all particles takes k_correlate_tc_shared below.
#include <cuda_bf16.h>
#include <stdint.h>
#include "internal.cuh"

namespace matcha {
namespace {

constexpr int TC_THREADS = 256;  // warps 0-3 own the 128 accumulator lanes
constexpr int TC_M = 128;
constexpr long TC_WAIT_LIMIT = 1L << 24;  // mbarrier polls before giving up

__device__ __forceinline__ uint32_t su32(const void *p) {
  return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}

// Shared-memory matrix descriptor: start address, leading-dimension byte
// offset (between K-adjacent core matrices), stride-dimension byte offset
// (between M/N-adjacent core matrices), descriptor version 1, no swizzle.
__host__ __device__ __forceinline__ uint64_t smem_desc(uint32_t saddr, uint32_t lbo, uint32_t sbo) {
  uint64_t d = 0;
  d |= (uint64_t)((saddr >> 4) & 0x3FFFu);
  d |= (uint64_t)((lbo >> 4) & 0x3FFFu) << 16;
  d |= (uint64_t)((sbo >> 4) & 0x3FFFu) << 32;
  d |= (uint64_t)1 << 46;
  return d;
}

// Instruction descriptor: FP32 accumulator, A and B of format `fmt` (TF32 = 2
// under kind::tf32, BF16 = 1 under kind::f16), both K-major, N >> 3, M >> 4.
__host__ __device__ __forceinline__ uint32_t instr_desc(int fmt, int M, int N) {
  return (1u << 4) | ((uint32_t)fmt << 7) | ((uint32_t)fmt << 10) | ((uint32_t)(N >> 3) << 17) |
         ((uint32_t)(M >> 4) << 24);
}

template <int BF16> struct Op;
template <> struct Op<0> {  // TF32 in 32-bit containers
  static constexpr int bytes = 4;
  __device__ static void put(unsigned char *base, long off, float v) {
    uint32_t t;
    asm("cvt.rna.tf32.f32 %0, %1;" : "=r"(t) : "f"(v));
    *reinterpret_cast<uint32_t *>(base + off) = t;
  }
  __device__ static void mma(uint32_t tmem, uint64_t ad, uint64_t bd, uint32_t id, int acc) {
    asm volatile(
        "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::tf32 [%0], %1, %2, %3, p;\n\t}\n" ::"r"(tmem),
        "l"(ad), "l"(bd), "r"(id), "r"(acc));
  }
};
template <> struct Op<1> {  // BF16
  static constexpr int bytes = 2;
  __device__ static void put(unsigned char *base, long off, float v) {
    *reinterpret_cast<__nv_bfloat16 *>(base + off) = __float2bfloat16_rn(v);
  }
  __device__ static void mma(uint32_t tmem, uint64_t ad, uint64_t bd, uint32_t id, int acc) {
    asm volatile(
        "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}\n" ::"r"(tmem),
        "l"(ad), "l"(bd), "r"(id), "r"(acc));
  }
};

}  // namespace

// Tile geometry shared by the launcher and the kernel.  One operand buffer
// holds A's used row groups followed by B; the A descriptor spans 128 rows,
// which reach into B (rows past L+1 are never read back).  The accumulator
// tile copied out of tensor memory reuses the buffer whose MMAs are done.
struct TcGeom {
  int Kp, KC, SBO, RA, RAg, N, DS, ncols;
  long a_range, b_off, b_range, d_bytes, buf;
};
__host__ __device__ inline TcGeom tc_geom(int S, int L, int bytes) {
  TcGeom g;
  g.Kp = (2 * S + 15) / 16 * 16;
  g.KC = g.Kp * bytes / 16;    // 16-byte chunks along K
  g.SBO = g.KC * 128;          // bytes between 8-row groups
  g.RA = L + 2;                // A rows used: degree l (l+1 rows) then L-l (L-l+1 rows)
  g.RAg = (g.RA + 7) / 8;
  g.N = (4 * (L + 1) + 15) / 16 * 16;
  g.ncols = 32;
  while (g.ncols < g.N) g.ncols <<= 1;
  g.a_range = (long)(TC_M / 8) * g.SBO;  // what the A descriptor spans
  g.b_off = (long)g.RAg * g.SBO;
  g.b_range = (long)(g.N / 8) * g.SBO;
  g.DS = g.N + 1;  // odd row stride of the accumulator copy (no bank conflicts)
  g.d_bytes = 4L * g.RA * g.DS;
  long s = g.b_off + g.b_range;
  if (g.a_range > s) s = g.a_range;
  if (g.d_bytes > s) s = g.d_bytes;
  g.buf = (s + 1023) / 1024 * 1024;
  return g;
}
// Two operand buffers; at least 77 KB so that no more than two CTAs share an
// SM (each holds 256 of the SM's 512 tensor-memory columns for its lifetime).
__host__ __device__ inline long tc_smem(const TcGeom &g) {
  long s = 2 * g.buf;
  return s < 77 * 1024 ? 77 * 1024 : s;
}
bool correlate_tc_fits(int S, int L, int bytes) {
  TcGeom g = tc_geom(S, L, bytes);
  return g.N <= 256 && g.RA <= TC_M && g.ncols <= 256 && tc_smem(g) <= 200 * 1024;
}

namespace {

// Persistent CTAs, each over items (particle, degree pair) blockIdx.x,
// blockIdx.x + gridDim.x, ...; software pipeline per item i:
//   stage operands of i+1 (other buffer)   | MMAs of i run
//   wait for i, copy the accumulator to shared memory
//   issue the MMAs of i+1                   | epilogue of i (global stores)
template <int BF16>
__global__ void __launch_bounds__(TC_THREADS, 1)
    k_correlate_tc(const float *__restrict__ f, const float *__restrict__ h, int S, int L,
                   long h_stride, const double *__restrict__ wrad, long nc, float *__restrict__ c,
                   int B, int *__restrict__ err, long wait_limit) {
  using O = Op<BF16>;
  extern __shared__ __align__(1024) unsigned char smem_raw[];
  __shared__ __align__(8) uint64_t mbar;
  __shared__ uint32_t tmem_base;
  __shared__ float wsh[128];
  const TcGeom G = tc_geom(S, L, O::bytes);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int nlm = (L + 1) * (L + 2) / 2;
  const int npair = L / 2 + 1;
  const long nitems = (long)B * npair;
  const long first = blockIdx.x;
  const int nmine = first < nitems ? (int)((nitems - 1 - first) / gridDim.x + 1) : 0;
  constexpr int E = 16 / O::bytes;  // elements per 16-byte chunk
  auto off = [&](int r, int k) -> long {
    return (long)(r >> 3) * G.SBO + (long)(k / E) * 128 + (r & 7) * 16 + (k % E) * O::bytes;
  };
  auto bufp = [&](int i) { return smem_raw + (i & 1) * G.buf; };
  for (int s = tid; s < S; s += TC_THREADS) wsh[s] = (float)wrad[s];
  if (tid == 0) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(su32(&mbar)));
    asm volatile("fence.mbarrier_init.release.cluster;");
  }
  const int kpad = G.Kp - 2 * S;
  __syncthreads();

  // Operands of item `it` into buffer `u`.  The K padding of every row is
  // zeroed each time (the accumulator copy of an earlier item may have
  // overwritten it); rows and columns that are never read back (A rows past
  // L+1, B rows past 4(L+1), the second block of the single-degree item
  // l = L/2) may hold anything: they reach only unread accumulator entries.
  auto stage = [&](long it, int u) {
    const long b = it / npair;
    const int q = (int)(it - b * npair);
    const int d0 = q, d1 = L - q, nd = d0 == d1 ? 1 : 2;
    const float *fb = f + 2 * b * (long)S * nlm;
    const float *hb = h + 2 * (b * h_stride) * (long)S * nlm;
    unsigned char *As = bufp(u), *Bs = As + G.b_off;
    for (int t = tid; t < G.RA * kpad; t += TC_THREADS)
      O::put(As, off(t / kpad, 2 * S + t % kpad), 0.0f);
    for (int t = tid; t < G.N * kpad; t += TC_THREADS)
      O::put(Bs, off(t / kpad, 2 * S + t % kpad), 0.0f);
    int r0 = 0, cbase = 0;
    for (int dd = 0; dd < nd; ++dd) {
      const int d = dd ? d1 : d0;
      const int lm0 = d * (d + 1) / 2, no = d + 1, w2 = 2 * d + 1;
      // item (s, m): f_dm(r_s) -> A row m; h_dm(r_s) -> the B rows of n = m and
      // n = -m.  Items go in tiles of 8 orders x 4 shells, a warp per tile, so
      // a warp's stores fall in 32 distinct banks; all loads of a round are
      // issued before any store.
      const int mt = (no + 7) >> 3;
      const int na = mt * ((S + 3) >> 2) * 32;
      const FastDiv dv(mt);
      auto item = [&](int t, int &s, int &m) {
        const int T = t >> 5, ln = t & 31, ts = dv.div(T);
        m = ((T - ts * mt) << 3) + (ln & 7);
        s = (ts << 2) + (ln >> 3);
        return m < no && s < S;
      };
      for (int t0 = tid; t0 < na; t0 += 8 * TC_THREADS) {
        float2 fv[8], hv[8];
#pragma unroll
        for (int k = 0; k < 8; ++k) {
          const int t = t0 + k * TC_THREADS;
          int s, m;
          if (t < na && item(t, s, m)) {
            const long o = 2 * ((long)s * nlm + lm0 + m);
            fv[k] = __ldg(reinterpret_cast<const float2 *>(fb + o));
            hv[k] = __ldg(reinterpret_cast<const float2 *>(hb + o));
          }
        }
#pragma unroll
        for (int k = 0; k < 8; ++k) {
          const int t = t0 + k * TC_THREADS;
          int s, m;
          if (t < na && item(t, s, m)) {
            O::put(As, off(r0 + m, s), fv[k].x);
            O::put(As, off(r0 + m, S + s), fv[k].y);
            const float w = wsh[s], hr = w * hv[k].x, hi = w * hv[k].y;
            const int rp = cbase + d + m;  // n = m
            O::put(Bs, off(rp, s), hr);
            O::put(Bs, off(rp, S + s), hi);
            O::put(Bs, off(rp + w2, s), -hi);
            O::put(Bs, off(rp + w2, S + s), hr);
            if (m > 0) {  // n = -m: (-1)^m conj(h)
              const float sr = (m & 1) ? -hr : hr, si = (m & 1) ? hi : -hi;
              const int rn = cbase + d - m;
              O::put(Bs, off(rn, s), sr);
              O::put(Bs, off(rn, S + s), si);
              O::put(Bs, off(rn + w2, s), -si);
              O::put(Bs, off(rn + w2, S + s), sr);
            }
          }
        }
      }
      r0 = d0 + 1;
      cbase = 2 * (2 * d0 + 1);
    }
  };
  const uint32_t id = instr_desc(BF16 ? 1 : 2, TC_M, G.N);
  const int nk = G.Kp * O::bytes / 32;  // K per MMA: 8 TF32 or 16 BF16 = two 16-byte chunks
  auto issue = [&](int u) {             // one thread
    const uint32_t a0 = su32(bufp(u)), b0 = a0 + (uint32_t)G.b_off;
    for (int ks = 0; ks < nk; ++ks)
      O::mma(tmem_base, smem_desc(a0 + ks * 256, 128, G.SBO), smem_desc(b0 + ks * 256, 128, G.SBO),
             id, ks > 0);
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(
                     su32(&mbar))
                 : "memory");
  };

  // tensor-memory columns for the accumulator, held for the CTA's lifetime
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                     su32(&tmem_base)),
                 "r"(G.ncols));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
  }
  if (nmine > 0) stage(first, 0);
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tmem = tmem_base;
  if (tid == 0 && nmine > 0) issue(0);

  int ok = 1, fail_i = -1;
  for (int i = 0; i < nmine && ok; ++i) {
    const long it = first + (long)i * gridDim.x;
    if (i + 1 < nmine) stage(it + gridDim.x, (i + 1) & 1);
    uint32_t done = 0;
    for (long w = 0; w < wait_limit && !done; ++w)
      asm volatile(
          "{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
          "selp.u32 %0, 1, 0, p;\n\t}\n"
          : "=r"(done)
          : "r"(su32(&mbar)), "r"((uint32_t)(i & 1))
          : "memory");
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    float *Dt = reinterpret_cast<float *>(bufp(i));  // MMAs of item i are done with it
    if (__syncthreads_and(done) == 0) {
      ok = 0;
      fail_i = i;
      break;
    }
    if (32 * (warp & 3) < G.RA) {
      // warps w and w + 4 read lanes 32 (w % 4) .. + 31 (rows), alternate
      // 16-column chunks of them
      const int row = 32 * (warp & 3) + lane;
      const uint32_t ta = tmem + ((uint32_t)(32 * (warp & 3)) << 16);
      for (int cc = 16 * (warp >> 2); cc < G.N; cc += 32) {
        uint32_t v[16];
        asm volatile(
            "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];\n"
            : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]),
              "=r"(v[7]), "=r"(v[8]), "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]),
              "=r"(v[13]), "=r"(v[14]), "=r"(v[15])
            : "r"(ta + (uint32_t)cc));
        asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
        if (row < G.RA)
#pragma unroll
          for (int k = 0; k < 16; ++k) Dt[(long)row * G.DS + cc + k] = __uint_as_float(v[k]);
      }
    }
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    if (tid == 0 && i + 1 < nmine) issue((i + 1) & 1);
    // epilogue of item i: one thread per partner group (m, j) of each degree
    {
      const long b = it / npair;
      const int q = (int)(it - b * npair);
      const int d0 = q, d1 = L - q, nd = d0 == d1 ? 1 : 2;
      float *cb = c + 4 * b * nc;
      int r0 = 0, cbase = 0;
      for (int dd = 0; dd < nd; ++dd) {
        const int d = dd ? d1 : d0;
        const int cre = cbase, cim = cbase + 2 * d + 1;
        const float *Dr = Dt + (long)r0 * G.DS;
        const int ng = (d + 1) * (d + 2) / 2;
        for (int g = tid; g < ng; g += TC_THREADS) {
          const int m = tri_floor(g), j = g - m * (m + 1) / 2;
          float e[8];
#pragma unroll
          for (int hh = 0; hh < 2; ++hh) {
            const int n = 2 * j - m + hh;
            float a = 0, bq = 0, cr = 0, ci = 0;
            if (n <= m) {
              a = Dr[(long)m * G.DS + cre + n + d];
              bq = Dr[(long)m * G.DS + cim + n + d];
              if (n >= 0) {
                cr = Dr[(long)n * G.DS + cre + m + d];
                ci = Dr[(long)n * G.DS + cim + m + d];
              } else {  // c_{n m} = (-1)^{m+n} conj(c_{-n,-m})
                const float sg = ((m + n) & 1) ? -1.0f : 1.0f;
                cr = sg * Dr[(long)(-n) * G.DS + cre - m + d];
                ci = -sg * Dr[(long)(-n) * G.DS + cim - m + d];
              }
            }
            e[hh] = a; e[2 + hh] = bq; e[4 + hh] = cr; e[6 + hh] = ci;
          }
          // entry (group, d): goff(m, j) + d - m, 8 reals
          const long t = (long)m * (m + 1) / 2;
          const long go =
              (long)(L + 2) * t - (long)m * (m + 1) * (2 * m + 1) / 6 + (long)j * (L - m + 1);
          float4 *o = reinterpret_cast<float4 *>(cb + 8 * (go + d - m));
          o[0] = make_float4(e[0], e[1], e[2], e[3]);
          o[1] = make_float4(e[4], e[5], e[6], e[7]);
        }
        r0 = d0 + 1;
        cbase = 2 * (2 * d0 + 1);
      }
    }
    __syncthreads();  // the accumulator copy and the buffer are free for item i + 2
  }
  if (!ok) {
    if (tid == 0) atomicOr(err, 1);
    // the MMAs of item fail_i are still in flight: wait for them (bounded)
    // before the columns they write are freed
    uint32_t done = 0;
    for (long w = 0; w < TC_WAIT_LIMIT && !done; ++w)
      asm volatile(
          "{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
          "selp.u32 %0, 1, 0, p;\n\t}\n"
          : "=r"(done)
          : "r"(su32(&mbar)), "r"((uint32_t)(fail_i & 1))
          : "memory");
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  if (warp == 0)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(G.ncols));
}

}  // namespace

// One template for the whole batch.  A unit is (block of PB particles, degree pair):
// B is staged once for the block, and a pass multiplies the A rows of PM particles,
// stacked in the 128-row tile at multiples of 8 RAg, with it.  One CTA per SM of 16
// warps; A, the accumulator columns and their barriers are double-buffered, so the
// next pass's MMAs run during this one's epilogue, and its coefficients are loaded
// into registers before that.  The epilogue's addresses are the same for every pass
// of a unit and are tabulated once; neighbouring lanes write the halves of a record,
// so a store touches 16 lines, not 32 (431 -> 351 us).  768 particles, 32 shells, L_J =
// 48, TF32: 854 us with both operands staged for every particle (conversions and
// 4-byte stores; one CTA of 8 warps on an SM) -> 351; reading and writing the
// coefficients is 111 us.  Bound by the shared-memory accesses of the epilogue and the
// phases' barriers; 1,024 threads: 373.
struct TcShared {
  int PM;
  long a_buf, a_off, d_off, t_off, smem;
};
constexpr int TS_THREADS = 512;
__host__ __device__ inline TcShared tc_shared(const TcGeom &g, int L, int PM) {
  TcShared q;
  q.PM = PM;
  q.a_off = g.b_range;
  q.a_buf = (long)PM * g.RAg * g.SBO;
  q.d_off = q.a_off + 2 * q.a_buf;
  q.t_off = (q.d_off + 4L * PM * g.RA * g.DS + 15) / 16 * 16;
  // groups of a pair: (d+1)(d+2)/2 of both degrees, at most those of degrees 0 and L
  q.smem = q.t_off + 16L * ((L + 1) * (L + 2) / 2 + 1);
  const long span = q.a_off + q.a_buf + g.a_range;  // what the second buffer's descriptor spans
  if (q.smem < span) q.smem = span;
  if (q.smem < 115 * 1024) q.smem = 115 * 1024;  // one CTA per SM: each holds its 512 columns
  return q;
}
// Particles per tile: as many as fit its rows and shared memory, at most four; 0: none.
inline int tc_shared_stack(const TcGeom &g, int S, int L) {
  if (g.N > 256 || g.RA > TC_M || S > 128) return 0;
  for (int PM = 4; PM >= 1; PM /= 2)
    if (PM * 8 * g.RAg <= TC_M && tc_shared(g, L, PM).smem <= 220 * 1024) return PM;
  return 0;
}

namespace {

__device__ __forceinline__ uint32_t mbar_wait(uint64_t *bar, uint32_t parity, long limit) {
  uint32_t done = 0;
  for (long w = 0; w < limit && !done; ++w)
    asm volatile(
        "{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}\n"
        : "=r"(done)
        : "r"(su32(bar)), "r"(parity)
        : "memory");
  return done;
}

template <int BF16>
__global__ void __launch_bounds__(TS_THREADS, 1)
    k_correlate_tc_shared(const float *__restrict__ f, const float *__restrict__ h, int S, int L,
                          const double *__restrict__ wrad, long nc, float *__restrict__ c, int B,
                          int PB, int PM, int *__restrict__ err, long wait_limit) {
  using O = Op<BF16>;
  extern __shared__ __align__(1024) unsigned char smem_raw[];
  __shared__ __align__(8) uint64_t mbar[2];
  __shared__ uint32_t tmem_base;
  __shared__ float wsh[128];
  const TcGeom G = tc_geom(S, L, O::bytes);
  const TcShared Q = tc_shared(G, L, PM);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int nlm = (L + 1) * (L + 2) / 2, npair = L / 2 + 1;
  const int nunit = (B + PB - 1) / PB * npair;
  constexpr int E = 16 / O::bytes;  // elements per 16-byte chunk
  auto off = [&](int r, int k) -> int {
    return (r >> 3) * G.SBO + (k / E) * 128 + (r & 7) * 16 + (k % E) * O::bytes;
  };
  unsigned char *Bs = smem_raw;
  auto abuf = [&](int i) { return smem_raw + Q.a_off + (i & 1) * Q.a_buf; };
  float *Dt = reinterpret_cast<float *>(smem_raw + Q.d_off);
  uint4 *tab = reinterpret_cast<uint4 *>(smem_raw + Q.t_off);
  const uint2 *half = reinterpret_cast<const uint2 *>(tab);
  for (int s = tid; s < S; s += TS_THREADS) wsh[s] = (float)wrad[s];
  const int kpad = G.Kp - 2 * S;  // the K padding stays zero
  if (kpad > 0) {
    const int rows = 2 * PM * G.RAg * 8;
    for (int t = tid; t < rows * kpad; t += TS_THREADS)
      O::put(smem_raw + Q.a_off, off(t / kpad, 2 * S + t % kpad), 0.0f);
    for (int t = tid; t < G.N * kpad; t += TS_THREADS) O::put(Bs, off(t / kpad, 2 * S + t % kpad), 0.0f);
  }
  if (tid == 0) {
    for (int k = 0; k < 2; ++k)
      asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(su32(&mbar[k])));
    asm volatile("fence.mbarrier_init.release.cluster;");
  }
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                     su32(&tmem_base)),
                 "r"(2 * G.ncols));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tmem = tmem_base;
  const uint32_t id = instr_desc(BF16 ? 1 : 2, TC_M, G.N);
  const int nk = G.Kp * O::bytes / 32;  // K per MMA: 8 TF32 or 16 BF16 = two 16-byte chunks
  auto issue = [&](int n) {             // pass n of this CTA; one thread
    const uint32_t a0 = su32(abuf(n)), b0 = su32(Bs);
    for (int ks = 0; ks < nk; ++ks)
      O::mma(tmem + (uint32_t)((n & 1) * G.ncols), smem_desc(a0 + ks * 256, 128, G.SBO),
             smem_desc(b0 + ks * 256, 128, G.SBO), id, ks > 0);
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(
                     su32(&mbar[n & 1]))
                 : "memory");
  };
  // Items (s, m) go in tiles of 8 orders x 4 shells, a warp per tile, so a warp's
  // stores fall in 32 distinct banks.
  const int ts4 = (S + 3) >> 2;
  constexpr int BL = 2048 / TS_THREADS;
  constexpr int AHEAD = 4096 / TS_THREADS;  // items of a thread loaded ahead of their pass
  int ok = 1, n = 0;        // n: passes issued
  int last = -1;            // the last pass waited for
  for (int unit = blockIdx.x; unit < nunit && ok; unit += gridDim.x) {
    const int blk = unit / npair, q = unit - blk * npair;
    const int d0 = q, d1 = L - q, nd = d0 == d1 ? 1 : 2;
    const int b0 = blk * PB, nb = min(PB, B - b0), npass = (nb + PM - 1) / PM;
    const int mt0 = (d0 + 8) >> 3, mt1 = nd > 1 ? (d1 + 8) >> 3 : 0, mts = mt0 + mt1;
    const int tiles = mts * ts4;                   // per particle
    const FastDiv dtile(tiles), dmts(mts);
    const float *fu = f + 2 * (long)b0 * S * nlm;
    float *cu = c + 4 * (long)b0 * nc;
    // item t of a pass: particle of the pass, row, order, shell, and where its
    // coefficient is from the pass's first particle's
    auto item = [&](int t, int &pq, int &row, int &m, int &s, int &src) {
      const int T = t >> 5, ln = t & 31;
      pq = dtile.div(T);
      const int rest = T - pq * tiles, ts = dmts.div(rest), mt = rest - ts * mts;
      const bool second = mt >= mt0;
      const int d = second ? d1 : d0;
      m = ((second ? mt - mt0 : mt) << 3) + (ln & 7);
      s = (ts << 2) + (ln >> 3);
      row = pq * 8 * G.RAg + (second ? d0 + 1 : 0) + m;
      src = (pq * S + s) * nlm + d * (d + 1) / 2 + m;
      return m <= d && s < S;
    };
    const int nitem = PM * tiles * 32;
    // the thread's first items, the same in every pass: coefficient (particle of the
    // pass above bit 28; -1: none) and the two elements they go to
    int from[AHEAD], to[AHEAD];
#pragma unroll
    for (int k = 0; k < AHEAD; ++k) {
      const int t = tid + k * TS_THREADS;
      int pq, row, m, s, src;
      from[k] = -1;
      if (t < nitem && item(t, pq, row, m, s, src)) {
        from[k] = src | pq << 28;
        to[k] = off(row, s) / O::bytes | off(row, S + s) / O::bytes << 16;
      }
    }
    float2 pre[AHEAD];
    auto load = [&](int pass) {
      const float2 *fp = reinterpret_cast<const float2 *>(fu) + (long)pass * PM * S * nlm;
      const int np = min(PM, nb - pass * PM);
#pragma unroll
      for (int k = 0; k < AHEAD; ++k)
        if (from[k] >= 0 && from[k] >> 28 < np) pre[k] = __ldg(fp + (from[k] & 0xfffffff));
    };
    auto put = [&](int pass, unsigned char *As) {  // (rows of absent particles: any values)
#pragma unroll
      for (int k = 0; k < AHEAD; ++k)
        if (from[k] >= 0) {
          O::put(As, (to[k] & 0xffff) * O::bytes, pre[k].x);
          O::put(As, (int)((unsigned)to[k] >> 16) * O::bytes, pre[k].y);
        }
      for (int t = tid + AHEAD * TS_THREADS; t < nitem; t += TS_THREADS) {
        int pq, row, m, s, src;
        if (!item(t, pq, row, m, s, src) || pass * PM + pq >= nb) continue;
        const float2 v = __ldg(reinterpret_cast<const float2 *>(fu) + (long)pass * PM * S * nlm + src);
        O::put(As, off(row, s), v.x);
        O::put(As, off(row, S + s), v.y);
      }
    };
#pragma unroll
    for (int k = 0; k < AHEAD; ++k) pre[k] = make_float2(0.f, 0.f);
    load(0);
    // B: h_dm(r_s) -> the rows of n = m and n = -m (all earlier MMAs have been waited for)
    for (int t0 = tid; t0 < tiles * 32; t0 += BL * TS_THREADS) {
      float2 hv[BL];
      int pq, row, m, s, src;
#pragma unroll
      for (int k = 0; k < BL; ++k) {
        const int t = t0 + k * TS_THREADS;
        if (t < tiles * 32 && item(t, pq, row, m, s, src)) hv[k] = __ldg(reinterpret_cast<const float2 *>(h) + src);
      }
#pragma unroll
      for (int k = 0; k < BL; ++k) {
        const int t = t0 + k * TS_THREADS;
        if (t >= tiles * 32 || !item(t, pq, row, m, s, src)) continue;
        const bool second = row >= d0 + 1 && nd > 1;
        const int d = second ? d1 : d0, cbase = second ? 2 * (2 * d0 + 1) : 0, w2 = 2 * d + 1;
        const float w = wsh[s], hr = w * hv[k].x, hi = w * hv[k].y;
        const int rp = cbase + d + m;  // n = m
        O::put(Bs, off(rp, s), hr);
        O::put(Bs, off(rp, S + s), hi);
        O::put(Bs, off(rp + w2, s), -hi);
        O::put(Bs, off(rp + w2, S + s), hr);
        if (m > 0) {  // n = -m: (-1)^m conj(h)
          const float sr = (m & 1) ? -hr : hr, si = (m & 1) ? hi : -hi;
          const int rn = cbase + d - m;
          O::put(Bs, off(rn, s), sr);
          O::put(Bs, off(rn, S + s), si);
          O::put(Bs, off(rn + w2, s), -si);
          O::put(Bs, off(rn + w2, S + s), sr);
        }
      }
    }
    // the epilogue's table, per half record of a partner group (m, j) of each degree,
    // (c_mn) for n = n0, n0 + 1, then (c_nm): offsets of the two real parts in the
    // accumulator copy; output entry, offset to the imaginary parts, signs of the four
    // values, and whether there is no n0 + 1
    const int ng0 = (d0 + 1) * (d0 + 2) / 2, ng = ng0 + (nd > 1 ? (d1 + 1) * (d1 + 2) / 2 : 0);
    for (int t = tid; t < ng; t += TS_THREADS) {
      const bool second = t >= ng0;
      const int d = second ? d1 : d0, g = second ? t - ng0 : t;
      const int r0 = second ? d0 + 1 : 0, cre = second ? 2 * (2 * d0 + 1) : 0;
      const int m = tri_floor(g), j = g - m * (m + 1) / 2;
      unsigned po[2], sg = 0;
#pragma unroll
      for (int hh = 0; hh < 2; ++hh) {
        const int k = 2 * j - m + hh;  // n
        if (k >= 0) {
          po[hh] = (r0 + min(k, m)) * G.DS + cre + m + d;
        } else {  // c_{n m} = (-1)^{m+n} conj(c_{-n,-m})
          po[hh] = (r0 - k) * G.DS + cre - m + d;
          sg |= (((m + k) & 1) ? 1u : 4u) << hh;
        }
      }
      const int tm = m * (m + 1);
      const int go = (L + 2) * (tm / 2) - tm * (2 * m + 1) / 6 + j * (L - m + 1);
      const unsigned own = (r0 + m) * G.DS + cre + 2 * j - m + d;
      const unsigned at = (unsigned)(go + d - m) | (unsigned)(2 * d + 1) << 16 | (unsigned)(j == m) << 27;
      tab[t] = make_uint4(own | (own + (j < m)) << 16, at, po[0] | po[1] << 16, at | sg << 28);
    }
    put(0, abuf(n));
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    if (tid == 0) issue(n);
    if (npass > 1) load(1);
    for (int i = 0; i < npass; ++i, ++n) {
      if (i + 1 < npass) {
        put(i + 1, abuf(n + 1));
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
        __syncthreads();
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        if (tid == 0) issue(n + 1);
      } else {
        __syncthreads();  // the epilogue of the pass before is done with the copy
      }
      // (uniform over the warp, which reads tensor memory together)
      const int done = __all_sync(0xffffffffu, mbar_wait(&mbar[n & 1], (uint32_t)((n >> 1) & 1), wait_limit));
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
      const int quad = 32 * (warp & 3);
      if (done && quad < PM * 8 * G.RAg) {
        // the warps of a lane quadrant take its 16-column chunks in turn
        const int row = quad + lane, pq = row / (8 * G.RAg), r = row - pq * 8 * G.RAg;
        const uint32_t ta = tmem + ((uint32_t)quad << 16) + (uint32_t)((n & 1) * G.ncols);
        float *Dr = Dt + (pq * G.RA + r) * G.DS;
        for (int cc = 16 * (warp >> 2); cc < G.N; cc += TS_THREADS / 8) {
          uint32_t v[16];
          asm volatile(
              "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];\n"
              : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]),
                "=r"(v[7]), "=r"(v[8]), "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]),
                "=r"(v[13]), "=r"(v[14]), "=r"(v[15])
              : "r"(ta + (uint32_t)cc));
          asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
          if (pq < PM && r < G.RA)
#pragma unroll
            for (int k = 0; k < 16; ++k) Dr[cc + k] = __uint_as_float(v[k]);
        }
      }
      asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
      if (__syncthreads_and(done) == 0) {
        ok = 0;
        n += i + 1 < npass;  // the last pass in flight
        break;
      }
      last = n;
      if (i + 2 < npass) load(i + 2);
      for (int pq = 0; pq < PM && i * PM + pq < nb; ++pq) {
        const float *D = Dt + pq * G.RA * G.DS;
        float4 *o = reinterpret_cast<float4 *>(cu + 4 * (long)(i * PM + pq) * nc);
        for (int t = tid; t < 2 * ng; t += TS_THREADS) {
          const uint2 e = half[t];
          const float *pa = D + (e.x & 0xffff), *pb = D + (e.x >> 16);
          const int im = e.y >> 16 & 0x7ff;
          uint32_t v[4] = {__float_as_uint(pa[0]), __float_as_uint(pb[0]), __float_as_uint(pa[im]),
                           __float_as_uint(pb[im])};
          const bool none = e.y >> 27 & 1;
          float4 x;
          x.x = __uint_as_float(v[0] ^ (e.y >> 28 << 31));
          x.y = none ? 0.f : __uint_as_float(v[1] ^ (e.y >> 29 << 31));
          x.z = __uint_as_float(v[2] ^ (e.y >> 30 << 31));
          x.w = none ? 0.f : __uint_as_float(v[3] ^ (e.y >> 31 << 31));
          o[2 * (e.y & 0xffff) + (t & 1)] = x;
        }
      }
    }
    __syncthreads();  // the table, the copy and the operands are free for the next unit
  }
  if (!ok) {
    if (tid == 0) atomicOr(err, 1);
    // passes last + 1 .. n are in flight: wait for them (bounded) before their columns
    // are freed
    for (int k = last + 1; k <= n; ++k) mbar_wait(&mbar[k & 1], (uint32_t)((k >> 1) & 1), TC_WAIT_LIMIT);
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  if (warp == 0)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(2 * G.ncols));
}

}  // namespace

// Particles per block: their passes share one staging of B, worth about 2.5 particles,
// but the blocks have to fill the SMs (at most 16: those in flight then write about 64
// MB, so that the degrees of an output line meet in L2).  An item of k_correlate_tc, two
// on an SM, takes about as long as 4.2 particles of a pass.  768 particles, 32 shells,
// L_J = 48, TF32: 387 us with 8, 351 with 16; 17 and 64 particles, 24 shells, L_J = 33:
// 14 and 31 us with k_correlate_tc, 20 and 34 in blocks of two, 17 and 23 in blocks of
// four and eight.
// 0: k_correlate_tc.
int correlate_tc_block(const Plan &p, int B, int hstride) {
  const int nsm = p.sms;
  const int PM = hstride ? 0 : tc_shared_stack(tc_geom(p.S, p.LJ, p.tc == 2 ? 2 : 4), p.S, p.LJ);
  const int pairs = p.LJ / 2 + 1;
  const long items = (long)B * pairs;
  int PB = 0;
  double best = 1e30;
  for (int q = PM; q && q <= 16; q *= 2) {
    const long units = (long)((B + q - 1) / q) * pairs;
    const double t = (units + nsm - 1) / nsm * (2.5 + q);
    if (t < best) { best = t; PB = q; }
  }
  return items > 2L * nsm && best <= 4.2 * ((items + 2L * nsm - 1) / (2L * nsm)) ? PB : 0;
}

cudaError_t launch_correlate_tc(const Plan &p, const float *f, const float *h, int B, int hstride,
                                float *c, cudaStream_t st) {
  if (B == 0) return cudaSuccess;
  const int bf16 = p.tc == 2;
  const TcGeom g = tc_geom(p.S, p.LJ, bf16 ? 2 : 4);
  if (!correlate_tc_fits(p.S, p.LJ, bf16 ? 2 : 4) || p.S > 128) return cudaErrorInvalidConfiguration;
  const int nsm = p.sms, PB = correlate_tc_block(p, B, hstride);
  const long items = (long)B * (p.LJ / 2 + 1);
  if (PB) {
    const int PM = tc_shared_stack(g, p.S, p.LJ);
    const long units = (long)((B + PB - 1) / PB) * (p.LJ / 2 + 1);
    const int smem1 = (int)tc_shared(g, p.LJ, PM).smem;
    const long limit = p.wait_limit >= 0 ? p.wait_limit : TC_WAIT_LIMIT;
    auto kern = bf16 ? k_correlate_tc_shared<1> : k_correlate_tc_shared<0>;
    const cudaError_t e = allow_smem(kern, smem1, 1024);
    if (e != cudaSuccess) return e;
    kern<<<(int)(units < nsm ? units : nsm), TS_THREADS, smem1, st>>>(f, h, p.S, p.LJ, p.wrad, p.nc, c, B,
                                                                      PB, PM, p.dev_err, limit);
    return cudaGetLastError();
  }
  const long per_sm = p.tune_tc_ctas == 1 ? 1 : 2;
  const int grid = (int)(items < per_sm * nsm ? items : per_sm * nsm);
  const size_t smem = (size_t)tc_smem(g);
  const long wait_limit = p.wait_limit >= 0 ? p.wait_limit : TC_WAIT_LIMIT;
  const cudaError_t e = bf16 ? allow_smem(k_correlate_tc<1>, smem, 1024) : allow_smem(k_correlate_tc<0>, smem, 1024);
  if (e != cudaSuccess) return e;
  if (bf16) {
    k_correlate_tc<1><<<grid, TC_THREADS, smem, st>>>(f, h, p.S, p.LJ, hstride, p.wrad, p.nc, c, B,
                                                      p.dev_err, wait_limit);
  } else {
    k_correlate_tc<0><<<grid, TC_THREADS, smem, st>>>(f, h, p.S, p.LJ, hstride, p.wrad, p.nc, c, B,
                                                      p.dev_err, wait_limit);
  }
  return cudaGetLastError();
}

}  // namespace matcha
