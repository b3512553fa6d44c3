// Translation search of the 6-D pose (the appendix "Alternating search over
// rotations and translations"; three alternations in Section 5.2).
//
// For a fixed rotation g the objective <f, g o S_tau h> is the
// cross-correlation CC(t) = sum_x f(x) u(x - t) of the particle f and the
// rotated template u = g o h at t = g tau.  CC is the circular correlation a
// 3-D FFT computes:
//   1. Z = FFT3(f + i u): both real volumes in one complex transform
//      (mixed radix 4/2/3/5 Stockham passes along x, y and z, each line held
//      in shared memory, loads and stores coalesced along x);
//   2. X(k) = F(k) conj(U(k)) from Z(k) and Z(-k) (the two spectra of a
//      packed pair), in place, by the CTA that made both in its z transform;
//   3. CC(t) = N^-3 Re sum_k X(k) e^{2 pi i k.t/N} (k in [-N/2, N/2)^3, the
//      trigonometric interpolant of CC) only where it is needed, by three
//      separable partial inverse DFTs (z, then y, then x): first on the
//      integer window [-m, m]^3, then on a grid of 2 floor(0.75 U) + 1
//      points per axis at spacing 1/U around the integer peak (the upsampled
//      DFT of Guizar-Sicairos et al. that the paper cites for sub-voxel
//      accuracy);
//   4. the maximum of each grid (ties to the smaller [z][y][x] index, NaN
//      never wins) gives t, and tau = R^T t.
// A pose kernel makes the rotated template u(x) = h(R^T (x - c0) + c0) and
// the shifted template (S_tau h)(x) = h(x - tau) by trilinear interpolation.
#include <math.h>
#include <algorithm>
#include <type_traits>
#include "internal.cuh"

namespace matcha {

template <typename T> struct alignas(2 * sizeof(T)) C2 { T x, y; };

template <typename T>
__device__ __forceinline__ C2<T> cmul(C2<T> a, C2<T> b) {
  return C2<T>{a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x};
}
template <typename T> __device__ __forceinline__ C2<T> cadd(C2<T> a, C2<T> b) { return {a.x + b.x, a.y + b.y}; }
template <typename T> __device__ __forceinline__ C2<T> csub(C2<T> a, C2<T> b) { return {a.x - b.x, a.y - b.y}; }
// s * i * a
template <typename T> __device__ __forceinline__ C2<T> cmuli(C2<T> a, T s) { return {-s * a.y, s * a.x}; }
template <typename T> __device__ __forceinline__ C2<T> cscale(C2<T> a, T s) { return {s * a.x, s * a.y}; }

// Rounded multiply and add that the compiler may not contract into an FMA:
// the FP64 pose transform then rounds exactly as the oracle's plain C.
__device__ __forceinline__ double mul_rn(double a, double b) { return __dmul_rn(a, b); }
__device__ __forceinline__ double add_rn(double a, double b) { return __dadd_rn(a, b); }
__device__ __forceinline__ float mul_rn(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ float add_rn(float a, float b) { return __fadd_rn(a, b); }

// ---- volume pose ------------------------------------------------------------
// out_b(x) = vol_b(R_b^T (x - c0) + c0 - s_b), trilinear, zero outside, one
// thread per output voxel.  R (row-major [B][9]) and s ([B][3]) are nullable
// (identity, zero).  A thread takes STEPS voxels along z, which spreads the block's
// indices, the pose (its conversion from FP64 runs at that rate) and the rows' products
// over them.  All index arithmetic is 32-bit: corner indices are clamped next to the box
// (they are outside all the same), the weights keep the unclamped coordinates; one test
// replaces the eight guards where all corners are inside.
__device__ __forceinline__ int corner_index(float f, int N) {  // -2 .. N + 1 (a NaN gives -2)
  return (int)fmin(fmax(f, -2.f), (float)(N + 1));
}
__device__ __forceinline__ int corner_index(double f, int N) {  // the conversion saturates
  return min(max(__double2int_rz(f), -2), N + 1);
}
template <typename T>
__device__ __forceinline__ float pose_sample(const float *__restrict__ src, int N, int NN, T px, T py, T pz) {
  const T fx0 = floor(px), fy0 = floor(py), fz0 = floor(pz);
  const int i0 = corner_index(fx0, N), j0 = corner_index(fy0, N), k0 = corner_index(fz0, N);
  const T tx = add_rn(px, -fx0), ty = add_rn(py, -fy0), tz = add_rn(pz, -fz0);
  float val[8];
  const unsigned last = N - 1;
  if ((unsigned)i0 < last && (unsigned)j0 < last && (unsigned)k0 < last) {  // all corners inside
    const float *p0 = src + (k0 * N + j0) * N + i0, *p1 = p0 + N, *p2 = p0 + NN, *p3 = p1 + NN;
    val[0] = __ldg(p0); val[1] = __ldg(p0 + 1);
    val[2] = __ldg(p1); val[3] = __ldg(p1 + 1);
    val[4] = __ldg(p2); val[5] = __ldg(p2 + 1);
    val[6] = __ldg(p3); val[7] = __ldg(p3 + 1);
  } else {
#pragma unroll
    for (int c = 0; c < 8; ++c) {
      const int ii = i0 + (c & 1), jj = j0 + (c >> 1 & 1), kk = k0 + (c >> 2);
      val[c] = 0.f;
      if ((unsigned)ii < (unsigned)N && (unsigned)jj < (unsigned)N && (unsigned)kk < (unsigned)N)
        val[c] = __ldg(src + (kk * N + jj) * N + ii);
    }
  }
  const T ux = add_rn(T(1), -tx), uy = add_rn(T(1), -ty), uz = add_rn(T(1), -tz);
  T acc = 0;
#pragma unroll
  for (int c = 0; c < 8; ++c) {
    const T w = mul_rn(mul_rn(c & 1 ? tx : ux, c >> 1 & 1 ? ty : uy), c >> 2 ? tz : uz);
    acc = add_rn(acc, mul_rn(w, (T)val[c]));
  }
  return (float)acc;
}

// FP32: a CTA takes a brick of 16 x 4 x 4 STEPS voxels, whose rotated corners share
// cache lines in all directions (a run of 256 along x does not).  96 volumes of 64^3:
// rotated 652 -> 170 us, shifted 266 -> 111 (one voxel per thread 260 and 240; two 208
// and 140; four 185 and 122), of which the traffic is 30; then the issue of coordinates
// and weights.
constexpr int POSE_X = 16, POSE_Y = 4, POSE_Z = 4, POSE_THREADS = POSE_X * POSE_Y * POSE_Z;
template <int STEPS>
__global__ void __launch_bounds__(POSE_THREADS)
k_pose_volume(int N, int nbx, const float *__restrict__ vol, long vstride,
              const double *__restrict__ R, const double *__restrict__ sh, float *__restrict__ out) {
  const long b = blockIdx.z;
  const int by = blockIdx.x / nbx;
  const int i = (blockIdx.x - by * nbx) * POSE_X + threadIdx.x % POSE_X;
  const int j = by * POSE_Y + threadIdx.x / POSE_X % POSE_Y;
  const int kb = blockIdx.y * POSE_Z * STEPS + threadIdx.x / (POSE_X * POSE_Y);
  __shared__ float r[12];  // R, then s: converted once, conversions from FP64 run at its rate
  if (threadIdx.x < 9) r[threadIdx.x] = R ? (float)R[9 * b + threadIdx.x] : float(threadIdx.x % 4 == 0);
  else if (threadIdx.x < 12) r[threadIdx.x] = sh ? (float)sh[3 * b + threadIdx.x - 9] : 0.f;
  __syncthreads();
  if (i >= N || j >= N) return;
  const float *src = vol + b * vstride;
  float *dst = out + b * (long)N * N * N + j * N + i;
  const float s0 = r[9], s1 = r[10], s2 = r[11];
  const float c0 = 0.5f * (float)N;
  const float x = (float)i - c0, y = (float)j - c0;
  // column c of R dotted with (x, y, z), then + c0 - s, left to right
  const float xy0 = add_rn(mul_rn(r[0], x), mul_rn(r[3], y)), xy1 = add_rn(mul_rn(r[1], x), mul_rn(r[4], y)),
              xy2 = add_rn(mul_rn(r[2], x), mul_rn(r[5], y));
  const float r6 = r[6], r7 = r[7], r8 = r[8];
  const int NN = N * N;
#pragma unroll
  for (int q = 0; q < STEPS; ++q) {
    const int k = kb + q * POSE_Z;
    if (k >= N) break;
    const float z = (float)k - c0;
    const float px = add_rn(add_rn(add_rn(xy0, mul_rn(r6, z)), c0), -s0);
    const float py = add_rn(add_rn(add_rn(xy1, mul_rn(r7, z)), c0), -s1);
    const float pz = add_rn(add_rn(add_rn(xy2, mul_rn(r8, z)), c0), -s2);
    dst[k * NN] = pose_sample<float>(src, N, NN, px, py, pz);
  }
}

// FP64: bound by its pipe, where an operation takes as long for one lane as for 32, so a
// CTA takes 256 consecutive voxels of a plane, or of the volume where a thread takes
// one (bricks of 16 leave a quarter of the lanes idle at N = 24), and the clamps work on
// integers.  64 volumes of 64^3: 2.46 ms before, 2.13 here; of 24^3: 197 us in bricks, 133
// here.
template <int STEPS>
__global__ void __launch_bounds__(POSE_THREADS)
k_pose_volume64(int N, const float *__restrict__ vol, long vstride, const double *__restrict__ R,
                const double *__restrict__ sh, float *__restrict__ out) {
  const long b = blockIdx.z;
  const int v = blockIdx.x * POSE_THREADS + threadIdx.x, q = v / N, i = v - q * N;
  const int kb = STEPS == 1 ? q / N : blockIdx.y * STEPS, j = STEPS == 1 ? q - kb * N : q;
  if (j >= N || kb >= N) return;
  double r[9], s[3];
#pragma unroll
  for (int c = 0; c < 9; ++c) r[c] = R ? R[9 * b + c] : (c % 4 == 0 ? 1.0 : 0.0);
#pragma unroll
  for (int c = 0; c < 3; ++c) s[c] = sh ? sh[3 * b + c] : 0.0;
  const float *src = vol + b * vstride;
  float *dst = out + b * (long)N * N * N + j * N + i;
  const double c0 = 0.5 * (double)N, x = (double)i - c0, y = (double)j - c0;
  // column c of R dotted with (x, y, z), then + c0 - s, left to right
  const double xy0 = add_rn(mul_rn(r[0], x), mul_rn(r[3], y)), xy1 = add_rn(mul_rn(r[1], x), mul_rn(r[4], y)),
               xy2 = add_rn(mul_rn(r[2], x), mul_rn(r[5], y));
  const int NN = N * N;
#pragma unroll
  for (int u = 0; u < STEPS; ++u) {
    const int k = kb + u;
    if (k >= N) break;
    const double z = (double)k - c0;
    const double px = add_rn(add_rn(add_rn(xy0, mul_rn(r[6], z)), c0), -s[0]);
    const double py = add_rn(add_rn(add_rn(xy1, mul_rn(r[7], z)), c0), -s[1]);
    const double pz = add_rn(add_rn(add_rn(xy2, mul_rn(r[8], z)), c0), -s[2]);
    dst[k * NN] = pose_sample<double>(src, N, NN, px, py, pz);
  }
}

cudaError_t launch_pose_volumes(int N, const float *vol, int B, long vol_stride, const double *R,
                                const double *shift, bool fp64, int sms, float *out, cudaStream_t st) {
  if (B <= 0) return cudaSuccess;
  if (fp64) {
    // four voxels per thread where that leaves at most a thirtieth of the lanes idle and
    // makes six CTAs on each SM, whose work then ends evenly; else one
    const int planes = (N * N + POSE_THREADS - 1) / POSE_THREADS, quads = (N + 3) / 4;
    if (30L * N * N * N >= 29L * planes * POSE_THREADS * quads * 4 && (long)planes * quads * B >= 6L * sms)
      k_pose_volume64<4><<<dim3(planes, quads, B), POSE_THREADS, 0, st>>>(N, vol, vol_stride, R, shift, out);
    else
      k_pose_volume64<1><<<dim3((N * N * N + POSE_THREADS - 1) / POSE_THREADS, 1, B), POSE_THREADS, 0, st>>>(
          N, vol, vol_stride, R, shift, out);
    return cudaGetLastError();
  }
  const int nbx = (N + POSE_X - 1) / POSE_X, nby = (N + POSE_Y - 1) / POSE_Y;
  auto run = [&](auto steps) {
    constexpr int ST = decltype(steps)::value;
    const dim3 grid((unsigned)(nbx * nby), (unsigned)((N + POSE_Z * ST - 1) / (POSE_Z * ST)), B);
    k_pose_volume<ST><<<grid, POSE_THREADS, 0, st>>>(N, nbx, vol, vol_stride, R, shift, out);
  };
  // eight voxels per thread where that still makes four CTAs on each SM
  if ((long)nbx * nby * ((N + 31) / 32) * B >= 4L * sms) run(std::integral_constant<int, 8>{});
  else run(std::integral_constant<int, 2>{});
  return cudaGetLastError();
}

// ---- box FFT ------------------------------------------------------------------
struct FftDesc {
  int N, npass;
  int radix[16];
};

// v, rounded: what follows may not be contracted with the operations that made it.
__device__ __forceinline__ C2<float> rounded(C2<float> v) {
  asm("" : "+f"(v.x), "+f"(v.y));
  return v;
}
__device__ __forceinline__ C2<double> rounded(C2<double> v) {
  asm("" : "+d"(v.x), "+d"(v.y));
  return v;
}

// Size-R DFT in place, V_q = sum_r v_r e^{-2 pi i q r / R}.
template <int R, typename T>
__device__ __forceinline__ void dft(C2<T> *v) {
  if (R == 2) {
    C2<T> a = v[0], b = v[1];
    v[0] = cadd(a, b); v[1] = csub(a, b);
  } else if (R == 4) {
    C2<T> s02 = cadd(v[0], v[2]), d02 = csub(v[0], v[2]);
    C2<T> s13 = cadd(v[1], v[3]), d13 = cmuli(csub(v[1], v[3]), T(-1));
    v[0] = cadd(s02, s13); v[2] = csub(s02, s13);
    v[1] = cadd(d02, d13); v[3] = csub(d02, d13);
  } else if (R == 3) {
    const T h3 = T(0.86602540378443864676);  // sin(2 pi / 3)
    C2<T> t1 = cadd(v[1], v[2]), t2 = cmuli(csub(v[1], v[2]), -h3);
    C2<T> a = csub(v[0], cscale(t1, T(0.5)));
    v[0] = cadd(v[0], t1);
    v[1] = cadd(a, t2);
    v[2] = csub(a, t2);
  } else {
    const T c1 = T(0.30901699437494742410), c2 = T(-0.80901699437494742410);  // cos(2pi/5), cos(4pi/5)
    const T s1 = T(0.95105651629515357212), s2 = T(0.58778525229247312917);   // sin(2pi/5), sin(4pi/5)
    C2<T> t1 = cadd(v[1], v[4]), t2 = cadd(v[2], v[3]);
    C2<T> t3 = csub(v[1], v[4]), t4 = csub(v[2], v[3]);
    C2<T> a1 = cadd(v[0], cadd(cscale(t1, c1), cscale(t2, c2)));
    C2<T> a2 = cadd(v[0], cadd(cscale(t1, c2), cscale(t2, c1)));
    C2<T> b1 = rounded(cmuli(cadd(cscale(t3, s1), cscale(t4, s2)), T(-1)));
    C2<T> b2 = rounded(cmuli(csub(cscale(t3, s2), cscale(t4, s1)), T(-1)));
    v[0] = cadd(v[0], cadd(t1, t2));
    v[1] = cadd(a1, b1); v[4] = csub(a1, b1);
    v[2] = cadd(a2, b2); v[3] = csub(a2, b2);
  }
}

// v w rounded as written, whatever follows (left to the compiler the outer
// operation could join the transform's additions, which would change last bits).
__device__ __forceinline__ C2<float> twiddle(C2<float> v, C2<float> w) {
  return {__fmaf_rn(v.x, w.x, -__fmul_rn(v.y, w.y)), __fmaf_rn(v.x, w.y, __fmul_rn(v.y, w.x))};
}
__device__ __forceinline__ C2<double> twiddle(C2<double> v, C2<double> w) {
  return {__fma_rn(v.x, w.x, -__dmul_rn(v.y, w.y)), __fma_rn(v.x, w.y, __dmul_rn(v.y, w.x))};
}

// One Stockham autosort pass of radix R over NB lines of length N: butterfly j of
// a line reads elements j + r N/R, applies the twiddles e^{-2 pi i k r / (Ns R)} (k =
// j mod Ns, Ns = product of earlier radices) and writes elements (j / Ns) Ns R + k +
// r Ns.  ld(line, e) and st(line, e, v): the elements.  Neighbouring threads take
// neighbouring lines, and a thread stays on its line where the lines divide the
// block.  tw: the twiddles in shared memory.
template <typename F>
__device__ __forceinline__ void fft_tasks(int n, int NB, F &&task) {
  if (blockDim.x % NB == 0) {
    const int j0 = threadIdx.x / NB, line = threadIdx.x - j0 * NB;
    for (int j = j0; j < n; j += blockDim.x / NB) task(line, j);
    return;
  }
  const FastDiv dl(NB);
  for (int t = threadIdx.x; t < NB * n; t += blockDim.x) {
    const int j = dl.div(t);
    task(t - j * NB, j);
  }
}
template <int R, typename T, typename Ld, typename St>
__device__ __forceinline__ void fft_pass(Ld ld, St st, int N, int NB, int Ns, const C2<T> *tw) {
  const FastDiv dn(Ns);
  if constexpr (R != 16) {
    const int NR = N / R, span = N / (Ns * R);
    fft_tasks(NR, NB, [&](int line, int j) {
      const int jn = dn.div(j), k = j - jn * Ns;
      C2<T> v[R];
#pragma unroll
      for (int r = 0; r < R; ++r) v[r] = ld(line, j + r * NR);
      if (Ns > 1)
#pragma unroll
        for (int r = 1; r < R; ++r) v[r] = twiddle(v[r], tw[k * r * span]);
      dft<R>(v);
#pragma unroll
      for (int r = 0; r < R; ++r) st(line, jn * Ns * R + k + r * Ns, v[r]);
    });
  } else {
    // two radix-4 passes in one, the 16 values between them in registers: the first
    // one's butterflies j + q N/16 write what the second one's, k + r Ns, read
    const int M = N / 16, s1 = N / (Ns * 4), s2 = N / (Ns * 16);
    fft_tasks(M, NB, [&](int line, int j) {
      const int jn = dn.div(j), k = j - jn * Ns;
      C2<T> v[4][4];  // [q][r]
#pragma unroll
      for (int r = 0; r < 4; ++r)
#pragma unroll
        for (int q = 0; q < 4; ++q) v[q][r] = ld(line, j + (4 * r + q) * M);
      if (Ns > 1)
#pragma unroll
        for (int r = 1; r < 4; ++r) {
          const C2<T> w = tw[k * r * s1];
#pragma unroll
          for (int q = 0; q < 4; ++q) v[q][r] = twiddle(v[q][r], w);
        }
#pragma unroll
      for (int q = 0; q < 4; ++q) dft<4>(v[q]);
#pragma unroll
      for (int r = 0; r < 4; ++r) {
        C2<T> u[4] = {v[0][r], v[1][r], v[2][r], v[3][r]};
#pragma unroll
        for (int q = 1; q < 4; ++q) u[q] = twiddle(u[q], tw[(k + r * Ns) * q * s2]);
        dft<4>(u);
#pragma unroll
        for (int q = 0; q < 4; ++q) st(line, jn * Ns * 16 + k + (r + 4 * q) * Ns, u[q]);
      }
    });
  }
}

// All passes of NB lines in the buffers src and dst (shared memory; element e of
// line l at l * ls + e * es, ls odd or es a row of lines, so that no banks collide).
// The first pass reads src, or gld(line, e) if one is given; the last leaves the
// result in src, or hands it to gst(line, e, v) and needs no more of the block.
struct InSmem {};
template <typename T, typename Gld = InSmem, typename Gst = InSmem>
__device__ __forceinline__ void fft_lines(C2<T> *&src, C2<T> *&dst, const FftDesc &fd, int ls, int es,
                                          int NB, const C2<T> *tw, Gld gld = {}, Gst gst = {}) {
  const int N = fd.N;
  int Ns = 1;
  for (int q = 0; q < fd.npass; ++q) {
    int R = fd.radix[q];
    const bool head = q == 0;
    if (R == 4 && q + 1 < fd.npass && fd.radix[q + 1] == 4 && (sizeof(T) == 4 || NB * (N / 16) >= 32)) {
      R = 16;
      ++q;
    }
    const bool tail = q + 1 >= fd.npass;
    auto sld = [=](int l, int e) { return src[l * ls + e * es]; };
    auto sst = [=](int l, int e, C2<T> v) { dst[l * ls + e * es] = v; };
    auto pass = [&](auto ld, auto st) {
      if (R == 16) fft_pass<16>(ld, st, N, NB, Ns, tw);
      else if (R == 4) fft_pass<4>(ld, st, N, NB, Ns, tw);
      else if (R == 2) fft_pass<2>(ld, st, N, NB, Ns, tw);
      else if (R == 3) fft_pass<3>(ld, st, N, NB, Ns, tw);
      else fft_pass<5>(ld, st, N, NB, Ns, tw);
    };
    constexpr bool GL = !std::is_same<Gld, InSmem>::value, GS = !std::is_same<Gst, InSmem>::value;
    static_assert(!(GL && GS), "one of the two");
    if constexpr (GL) {
      if (head) pass(gld, sst);
      else pass(sld, sst);
    } else if constexpr (GS) {
      if (tail) {
        pass(sld, gst);
        return;
      }
      pass(sld, sst);
    } else {
      pass(sld, sst);
    }
    __syncthreads();
    C2<T> *tmp = src; src = dst; dst = tmp;
    Ns *= R;
  }
}

// Forward x and y transforms of one z plane of the packed pair fre + i fim: the
// plane stays in shared memory between them, so the volume crosses HBM once.  A
// thread has 16 voxels of each volume in flight (loads of a loop that did not batch
// them left the warps waiting: 208 us), and the last y pass stores to memory.  96
// pairs of 64^3 in FP32: two passes of k_fft_axis 532 us, this 141, of which the
// traffic is 60; then the issue of the butterflies (72% busy).
template <typename T>
__global__ void __launch_bounds__(256)
k_fft_plane(C2<T> *__restrict__ data, const float *__restrict__ fre, const float *__restrict__ fim,
            const __grid_constant__ FftDesc fd, const C2<T> *__restrict__ twg) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int N = fd.N, LS = N | 1, N2 = N * N;
  C2<T> *src = reinterpret_cast<C2<T> *>(smem_raw), *dst = src + N * LS, *tw = dst + N * LS;
  const long o = blockIdx.y * (long)N2 * N + blockIdx.x * (long)N2;
  const FastDiv dN(N);
  constexpr int U = 16;  // voxels of a thread in flight
  for (int t0 = threadIdx.x; t0 < N2; t0 += U * blockDim.x) {
    float re[U], im[U];
#pragma unroll
    for (int q = 0; q < U; ++q) {
      const int t = t0 + q * blockDim.x;
      re[q] = t < N2 ? __ldg(fre + o + t) : 0.f;
      im[q] = t < N2 ? __ldg(fim + o + t) : 0.f;
    }
#pragma unroll
    for (int q = 0; q < U; ++q) {
      const int t = t0 + q * blockDim.x;
      if (t < N2) src[t + dN.div(t) * (LS - N)] = C2<T>{(T)re[q], (T)im[q]};
    }
  }
  for (int t = threadIdx.x; t < N; t += blockDim.x) tw[t] = twg[t];
  __syncthreads();
  fft_lines(src, dst, fd, LS, 1, N, tw);
  C2<T> *out = data + o;
  fft_lines(src, dst, fd, 1, LS, N, tw, InSmem{}, [=](int l, int e, C2<T> v) { out[e * N + l] = v; });
}

// Length-N transforms of NB lines of each volume along `axis` (0 x, 1 y), in
// place, for planes that do not fit in shared memory.  Axis 0: NB consecutive
// rows of the packed pair fre + i fim of float volumes; axis 1: NB consecutive x
// columns of one z plane, so every global access runs along x.
template <typename T>
__global__ void __launch_bounds__(256)
k_fft_axis(C2<T> *__restrict__ data, const float *__restrict__ fre, const float *__restrict__ fim,
           int axis, const __grid_constant__ FftDesc fd, const C2<T> *__restrict__ twg, int NB) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int N = fd.N, LS = N | 1;
  C2<T> *src = reinterpret_cast<C2<T> *>(smem_raw), *dst = src + NB * LS, *tw = dst + NB * LS;
  for (int t = threadIdx.x; t < N; t += blockDim.x) tw[t] = twg[t];
  const long b = blockIdx.y;
  const long N2 = (long)N * N, N3 = N2 * N;
  C2<T> *vol = data + b * N3;
  const int tid = threadIdx.x, NT = blockDim.x;
  const long g = blockIdx.x;
  long row0 = 0, ob = 0;
  int x0 = 0;
  if (axis == 0) {
    row0 = g * NB;
  } else {
    const int ntile = (N + NB - 1) / NB;
    const long outer = g / ntile;
    x0 = (int)(g - outer * ntile) * NB;
    ob = outer * N2;
  }
  const FastDiv dN(axis == 0 ? N : NB);
  auto at = [&](int idx, int &line, int &e, long &off) {
    const int q = dN.div(idx), w = idx - q * dN.d;
    line = axis == 0 ? q : w;
    e = axis == 0 ? w : q;
    off = axis == 0 ? (row0 + line) * N + e : ob + (long)e * N + x0 + line;
    return axis == 0 ? row0 + line < N2 : x0 + line < N;
  };
  for (int idx = tid; idx < NB * N; idx += NT) {
    int line, e;
    long off;
    C2<T> v{T(0), T(0)};
    if (at(idx, line, e, off))
      v = axis == 0 ? C2<T>{(T)__ldg(fre + b * N3 + off), (T)__ldg(fim + b * N3 + off)} : vol[off];
    src[line * LS + e] = v;
  }
  __syncthreads();
  fft_lines(src, dst, fd, LS, 1, NB, tw);
  for (int idx = tid; idx < NB * N; idx += NT) {
    int line, e;
    long off;
    if (at(idx, line, e, off)) vol[off] = src[line * LS + e];
  }
}

// The z transform and, still in shared memory, the cross spectrum: X(k) = F(k)
// conj(U(k)) from the packed spectrum Z = FFT(f + i u): F = (Z(k) + conj Z(-k)) / 2,
// U = (Z(k) - conj Z(-k)) / (2i), so X(k) = (i/4) (Z(k) + conj Z(-k)) (conj Z(k) -
// Z(-k)) and X(-k) = conj X(k) (CC is real).  A CTA takes NB columns kx of plane ky
// and the columns -kx of plane -ky (the columns 0 .. N/2 where ky = -ky), so that
// both members of every conjugate pair are at hand; the member with the smaller
// linear index plays k.  96 volumes of 64^3 in FP32: 383 us as a transform and a
// pass of its own, 112 here (traffic 60; 65% of the issue slots): the first pass reads
// memory directly, with no staging copy and barrier before it.
template <typename T>
__global__ void __launch_bounds__(128)
k_fft_cross(C2<T> *__restrict__ Z, const __grid_constant__ FftDesc fd, const C2<T> *__restrict__ twg,
            int NB) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int N = fd.N, N2 = N * N, L2 = 2 * NB, tid = threadIdx.x;
  C2<T> *src = reinterpret_cast<C2<T> *>(smem_raw), *dst = src + N * L2, *tw = dst + N * L2;
  C2<T> *zb = Z + blockIdx.y * (long)N2 * N;
  // planes 0 and (N even) N/2 are their own partners and come first
  const int nself = N % 2 ? 1 : 2, tself = (N / 2 + NB) / NB, tfull = (N + NB - 1) / NB;
  int ky, x0, nx;
  if ((int)blockIdx.x < nself * tself) {
    const int q = blockIdx.x / tself;
    ky = q ? N / 2 : 0;
    x0 = (blockIdx.x - q * tself) * NB;
    nx = N / 2 + 1;
  } else {
    const int g = blockIdx.x - nself * tself, q = g / tfull;
    ky = q + 1;
    x0 = (g - q * tfull) * NB;
    nx = N;
  }
  const int my = ky ? N - ky : 0;
  for (int t = tid; t < N; t += blockDim.x) tw[t] = twg[t];
  // this thread's line w (2 NB divides the block): column x0 + w of plane ky (w <
  // NB), or the mirror of column x0 + w - NB in plane -ky
  const int z0 = tid / L2, w = tid - z0 * L2, dz = blockDim.x / L2, x = x0 + (w < NB ? w : w - NB);
  const int mx = x ? N - x : 0;
  const bool live = x < nx;
  C2<T> *col = zb + (w < NB ? ky * N + x : my * N + mx);
  __syncthreads();
  // the first pass reads the thread's line w from memory
  fft_lines(src, dst, fd, 1, L2, L2, tw,
            [=](int, int kz) { return live ? col[kz * N2] : C2<T>{T(0), T(0)}; });
  const bool own = ky == my && x == mx;  // the column is its own partner
  if (live) {
    // the pairs (kz of the column, -kz of its partner) are shared between the
    // threads of the two lines: first halves of kz here, second halves there
    for (int q = w < NB ? z0 : z0 + dz; q < N; q += 2 * dz) {
      const int kz = q, mz = kz ? N - kz : 0, wa = w < NB ? w : w - NB;
      if (own && mz < kz) continue;
      C2<T> *pa = src + kz * L2 + wa, *pc = src + mz * L2 + (own ? wa : NB + wa);
      // the smaller linear index first
      const bool first = kz != mz ? kz < mz : ky != my ? ky < my : x <= mx;
      if (!first) { C2<T> *tmp = pa; pa = pc; pc = tmp; }
      const C2<T> A = *pa, C = *pc;
      const C2<T> s{A.x + C.x, A.y - C.y};    // Z(k) + conj Z(-k)
      const C2<T> d{A.x - C.x, -A.y - C.y};   // conj Z(k) - Z(-k)
      const C2<T> p = cmul(s, d);
      const C2<T> X{-T(0.25) * p.y, T(0.25) * p.x};
      *pa = X;
      if (pa != pc) *pc = C2<T>{X.x, -X.y};
    }
  }
  __syncthreads();
  if (live && !(own && w >= NB))  // its own partner: stored once
#pragma unroll 8
    for (int kz = z0; kz < N; kz += dz) col[kz * N2] = src[kz * L2 + w];
}

// Grid point j of axis a of particle b: t = org[b][a] + (j + j0) / den (org
// nullable), rounded as the oracle rounds it.
__device__ __forceinline__ double grid_t(const double *org, long b, int a, int j, int j0, int den) {
  return (org ? org[3 * b + a] : 0.0) + (double)(j + j0) / (double)den;
}

// E[b][a][k][j] = e^{2 pi i kk t / N} at the grid points t, kk = k or k - N
// (the symmetric frequency range); a = 0, 1, 2 for the x, y, z components.  One
// run of CTAs per (b, a); the points' FP64 divisions are made once per CTA.
template <typename T>
__global__ void __launch_bounds__(256)
k_idft_factors(C2<T> *__restrict__ E, int N, int nt, const double *__restrict__ org, int j0, int den) {
  __shared__ double ts[256];
  const int run = (N * nt + blockDim.x - 1) / blockDim.x;  // CTAs per (b, a)
  const int ba = blockIdx.x / run, b = ba / 3, a = ba - 3 * b;
  const bool pow2 = (N & (N - 1)) == 0;
  const double inv = 1.0 / N;
  for (int j = threadIdx.x; j < nt; j += blockDim.x) ts[j] = grid_t(org, b, a, j, j0, den);
  __syncthreads();
  const FastDiv dt(nt);
  const int q = (blockIdx.x - ba * run) * blockDim.x + threadIdx.x;
  if (q >= N * nt) return;
  const int k = dt.div(q), kk = k < (N + 1) / 2 ? k : k - N;
  const double u = 2.0 * kk * ts[q - k * nt];
  const double x = pow2 ? u * inv : u / N;  // the same bits: 1/N is exact
  T s, c;
  if (sizeof(T) == 8) {
    double sd, cd;
    sincospi(x, &sd, &cd);
    s = (T)sd; c = (T)cd;
  } else {
    float sf, cf;
    sincospif((float)x, &sf, &cf);
    s = (T)sf; c = (T)cf;
  }
  E[(long)ba * N * nt + q] = C2<T>{c, s};
}

// v e added to a, each part's two products fused once and rounded before they are
// added: a.x + (v.x e.x - v.y e.y), a.y + (v.y e.x + v.x e.y), the first product of
// each exact in the fused sum; q holds (e.x, e.x, -e.y, e.y).
__device__ __forceinline__ float2 cmac(float2 a, float2 v, const float4 &q) {
  const float2 m = __fmul2_rn(make_float2(v.y, v.x), make_float2(q.z, q.w));
  return __fadd2_rn(a, __ffma2_rn(v, make_float2(q.x, q.y), m));
}
struct alignas(16) Double4 { double x, y, z, w; };
__device__ __forceinline__ double2 cmac(double2 a, double2 v, const Double4 &q) {
  return make_double2(__dadd_rn(a.x, __fma_rn(v.x, q.x, __dmul_rn(v.y, q.z))),
                      __dadd_rn(a.y, __fma_rn(v.y, q.y, __dmul_rn(v.x, q.w))));
}
template <typename T> struct CPair;
template <> struct CPair<float> { typedef float2 type; typedef float4 quad; };
template <> struct CPair<double> { typedef double2 type; typedef Double4 quad; };

// out[b][a][j][c] = sum_k in[b][a][k][c] E[b][axis][k][j]: the partial inverse
// DFT along a middle (y) or outer (z) axis.  A thread takes CB columns c, JB grid
// points j at a time in registers against the factors in shared memory (one 16-byte
// broadcast per CB products of three packed operations); four rows k of its columns
// are in flight while the four before are multiplied.  PACK: one of the A C columns (a,
// c), and SP CTAs share a tile of them, each with every SP-th group of JB points (else
// the rows a are CTAs' and SP is 1).  es: elements between the particles' factors (0:
// shared).
//
// FP32, many volumes: 96 volumes of 64^3, 11 and 29 grid points: the z stage 139 and 171 us
// -> 76 and 97 (one column per thread 97 and 117; two without the loads ahead 128 and
// 143), then bound by its FMAs (floor 33) and, past 16 points, by reading the volume
// again.  One volume, 41 points: 41 and 40 us in the z and y stages on 16 and 41 CTAs;
// with one column and four points per CTA 14 and 12.
// FP64: bound by its pipe, where an operation takes as long for one lane as for 32 and
// a padded point as long as a real one, so no point is padded and the columns of all a
// are packed into warps; one column, four points and a CTA per group of points spread the
// work evenly.  64 volumes of 64^3, 41 points: 7.5 and 4.8 ms (eight padded points, two
// columns in the z stage: 9.0 and 5.8); one volume: 165 and 112 us (1,304 and 633).
template <typename T, int JB, int CB, bool PACK>
__global__ void __launch_bounds__(128)
k_idft_mid(const C2<T> *__restrict__ in, C2<T> *__restrict__ out, const C2<T> *__restrict__ E,
           int N, int nt, int A, int C, int axis, long es, int SP) {
  typedef typename CPair<T>::type P2;
  typedef typename CPair<T>::quad Q;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  Q *Es = reinterpret_cast<Q *>(smem_raw);  // [N][JB]
  const long b = blockIdx.z;
  static_assert(!PACK || CB == 1, "packed columns are single");
  const int tid = threadIdx.x, tile = PACK ? blockIdx.x / SP : blockIdx.x;
  const int c0 = tile * blockDim.x * CB + tid;
  const bool idle = c0 >= (PACK ? A * C : C);
  const int a = PACK ? min(c0, A * C - 1) / C : blockIdx.y;
  const int c = PACK ? min(c0, A * C - 1) - a * C : blockIdx.x * blockDim.x * CB + threadIdx.x;
  const P2 *src = reinterpret_cast<const P2 *>(in) + (b * A + a) * (long)N * C + c;
  const C2<T> *eb = E + b * es + (long)axis * N * nt;
  P2 *dst = reinterpret_cast<P2 *>(out) + (b * A + a) * (long)nt * C + c;
  int off[CB];  // a column past the end reads the thread's first
#pragma unroll
  for (int u = 0; u < CB; ++u) off[u] = !PACK && c + u * (int)blockDim.x < C ? u * blockDim.x : 0;
  for (int j0 = PACK ? (blockIdx.x - tile * SP) * JB : 0; j0 < nt; j0 += PACK ? SP * JB : JB) {
    __syncthreads();
    for (int t = tid; t < N * JB; t += blockDim.x) {
      const int k = t / JB, j = j0 + t % JB;
      const C2<T> e = j < nt ? eb[k * nt + j] : C2<T>{T(0), T(0)};
      Es[t] = Q{e.x, e.x, -e.y, e.y};
    }
    __syncthreads();
    if (idle) continue;
    P2 acc[CB][JB];
#pragma unroll
    for (int u = 0; u < CB; ++u)
#pragma unroll
      for (int j = 0; j < JB; ++j) acc[u][j].x = acc[u][j].y = T(0);
    constexpr int U = 4;
    P2 nx[U][CB];
    auto load = [&](int k0) {
#pragma unroll
      for (int q = 0; q < U; ++q)
#pragma unroll
        for (int u = 0; u < CB; ++u)
          if (k0 + q < N) nx[q][u] = src[(long)(k0 + q) * C + off[u]];
    };
    load(0);
    for (int k0 = 0; k0 < N; k0 += U) {
      P2 v[U][CB];
#pragma unroll
      for (int q = 0; q < U; ++q)
#pragma unroll
        for (int u = 0; u < CB; ++u) v[q][u] = nx[q][u];
      load(k0 + U);
#pragma unroll
      for (int q = 0; q < U; ++q) {
        if (k0 + q >= N) break;
#pragma unroll
        for (int j = 0; j < JB; ++j) {
          if (sizeof(T) == 8 && j0 + j >= nt) break;
          const Q e = Es[(k0 + q) * JB + j];
#pragma unroll
          for (int u = 0; u < CB; ++u) acc[u][j] = cmac(acc[u][j], v[q][u], e);
        }
      }
    }
#pragma unroll
    for (int u = 0; u < CB; ++u)
      if (u == 0 || off[u])
#pragma unroll
        for (int j = 0; j < JB; ++j)
          if (j0 + j < nt) dst[(long)(j0 + j) * C + off[u]] = acc[u][j];
  }
}

// CC[b][r][j] = scale Re sum_k Y[b][r][k] E[b][0][k][j]: the x stage, rows r =
// (tz, ty).  One CTA per (tile of ROWS rows, b).
template <typename T>
__global__ void __launch_bounds__(256)
k_idft_x(const C2<T> *__restrict__ Y, T *__restrict__ CC, const C2<T> *__restrict__ E, int N,
         int nt, int rows, T scale, long es) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  constexpr int ROWS = 8;
  C2<T> *ys = reinterpret_cast<C2<T> *>(smem_raw);  // [ROWS][N]
  C2<T> *Es = ys + ROWS * N;                         // [N][nt]
  const long b = blockIdx.y;
  const int r0 = blockIdx.x * ROWS;
  const int tid = threadIdx.x, NT = blockDim.x;
  const C2<T> *yb = Y + b * (long)rows * N;
  for (int idx = tid; idx < ROWS * N; idx += NT) {
    const int r = idx / N;
    ys[idx] = r0 + r < rows ? yb[(long)r0 * N + idx] : C2<T>{T(0), T(0)};
  }
  const C2<T> *eb = E + b * es;
  for (int idx = tid; idx < N * nt; idx += NT) Es[idx] = eb[idx];
  __syncthreads();
  for (int o = tid; o < ROWS * nt; o += NT) {
    const int r = o / nt, j = o - r * nt;
    if (r0 + r >= rows) continue;
    T re = 0;
    for (int k = 0; k < N; ++k) {
      const C2<T> v = ys[r * N + k], e = Es[k * nt + j];
      re += v.x * e.x - v.y * e.y;
    }
    CC[b * (long)rows * nt + (long)(r0 + r) * nt + j] = scale * re;
  }
}

// Maximum of each particle's nt^3 grid (value desc, index asc; NaN never
// wins): its grid point t, the value, flag bit 5 when an integer peak lies on
// the window's edge |t_a| = edge, and tau = R^T t.
template <typename T>
__global__ void __launch_bounds__(256)
k_cc_argmax(const T *__restrict__ CC, int nt, const double *__restrict__ org, int j0, int den,
            int edge, int flag_mode, const double *__restrict__ R, double *__restrict__ t_out,
            double *__restrict__ tau_out, double *__restrict__ cc_out, int *__restrict__ flags) {
  __shared__ T sv[256];
  __shared__ int si[256];
  const long b = blockIdx.x;
  const int n3 = nt * nt * nt, tid = threadIdx.x;
  const T *cb = CC + b * (long)n3;
  T bv = T(0);
  int bi = -1;
  for (int q = tid; q < n3; q += blockDim.x) {
    const T v = cb[q];
    if (v == v && (bi < 0 || v > bv)) { bv = v; bi = q; }  // q ascends: ties keep the first
  }
  sv[tid] = bv; si[tid] = bi;
  __syncthreads();
  for (int s = blockDim.x / 2; s > 0; s >>= 1) {
    if (tid < s) {
      const T ov = sv[tid + s];
      const int oi = si[tid + s];
      if (oi >= 0 && (si[tid] < 0 || ov > sv[tid] || (ov == sv[tid] && oi < si[tid]))) {
        sv[tid] = ov; si[tid] = oi;
      }
    }
    __syncthreads();
  }
  if (tid == 0) {
    const int q = si[0];
    double t[3];
    double v;
    if (q < 0) {
      t[0] = t[1] = t[2] = 0.0;
      v = __longlong_as_double(0x7ff8000000000000LL);
    } else {
      const int jx = q % nt, jy = (q / nt) % nt, jz = q / (nt * nt);
      const int jj[3] = {jx, jy, jz};
      for (int a = 0; a < 3; ++a) t[a] = grid_t(org, b, a, jj[a], j0, den);
      v = (double)sv[0];
    }
    for (int a = 0; a < 3; ++a) t_out[3 * b + a] = t[a];
    if (cc_out) cc_out[b] = v;
    int fl = 0;
    if (edge > 0)
      for (int a = 0; a < 3; ++a)
        if (fabs(t[a]) == (double)edge) fl = 32;
    if (q < 0) fl |= 1;
    if (flag_mode == 1) flags[b] = fl;
    else if (flag_mode == 2) flags[b] |= fl;
    if (tau_out) {
      const double *r = R + 9 * b;
      for (int a = 0; a < 3; ++a) tau_out[3 * b + a] = r[a] * t[0] + r[3 + a] * t[1] + r[6 + a] * t[2];
    }
  }
}

static int fine_points(int upsample) { return 2 * (int)floor(0.75 * upsample) + 1; }

size_t shift_ws_bytes(const Plan &p, int B, int max_shift, int upsample, char *base, ShiftWs *w) {
  const size_t cs = p.fp64 ? 16 : 8, rs = p.fp64 ? 8 : 4;
  const long N = p.N, N2 = N * N, N3 = N2 * N;
  const int nw = 2 * max_shift + 1, nf = fine_points(upsample);
  const long nt = nw > nf ? nw : nf;
  size_t off = 0;
  auto take = [&](size_t bytes) {
    char *r = base ? base + off : nullptr;
    off = align_up(off + bytes);
    return r;
  };
  ShiftWs tmp;
  ShiftWs *o = w ? w : &tmp;
  o->Z = take(cs * (size_t)B * N3);
  o->Y1 = take(cs * (size_t)B * nt * N2);
  o->Y2 = take(cs * (size_t)B * nt * nt * N);
  o->E = take(cs * (size_t)B * 3 * N * nt);
  o->CC = take(rs * (size_t)B * nt * nt * nt);
  o->t0 = reinterpret_cast<double *>(take(sizeof(double) * 3 * (size_t)B));
  return off;
}

// the three partial inverse-DFT stages and the maximum, on one grid
template <typename T>
static cudaError_t idft_grid(const Plan &p, int B, int nt, const double *org, int j0, int den,
                             int edge, int flag_mode, const double *R, const ShiftWs &w,
                             double *t_out, double *tau_out, double *cc_out, int *flags,
                             cudaStream_t st) {
  const int N = p.N;
  const long N2 = (long)N * N;
  // the integer window has the same factors for every particle
  const int nb = org ? B : 1;
  const long es = org ? 3L * N * nt : 0;
  k_idft_factors<T><<<3 * nb * ((N * nt + 255) / 256), 256, 0, st>>>((C2<T> *)w.E, N, nt, org, j0, den);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  // z stage: X[b][kz][ky kx] -> Y1[b][tz][ky kx], then y stage: Y1[b][tz][ky][kx]
  // -> Y2[b][tz][ty][kx].  FP32: the grid points per pass over a column are the fewest
  // passes of at most 16, rounded up to 4, with two columns per thread in the z stage,
  // which has N^2 of them per volume (rows of the y stage are short, one column keeps
  // their CTAs many: 11 points 23 against 33 us); where that makes fewer CTAs than SMs,
  // and in FP64, one column and four points per CTA.
  const size_t cs = sizeof(C2<T>);
  const int passes = (nt + 15) / 16, wide = ((nt + passes - 1) / passes + 3) / 4 * 4;
  const int narrow = (nt + 3) / 4, ty = N <= 64 ? 64 : 128;
  const bool fewz = sizeof(T) == 8 || (N2 + 255) / 256 * B < p.sms;
  const bool fewy = sizeof(T) == 8 || (long)((N + ty - 1) / ty) * nt * B < p.sms;
  auto pick = [&](auto cb, bool few) {
    constexpr int CB = decltype(cb)::value;
    if constexpr (sizeof(T) == 4) {
      if (!few)
        return wide == 4 ? k_idft_mid<T, 4, CB, false> : wide == 8 ? k_idft_mid<T, 8, CB, false>
             : wide == 12 ? k_idft_mid<T, 12, CB, false> : k_idft_mid<T, 16, CB, false>;
    }
    return k_idft_mid<T, 4, 1, true>;
  };
  auto midz = pick(std::integral_constant<int, 2>{}, fewz), midy = pick(std::integral_constant<int, 1>{}, fewy);
  const size_t smz = 2 * cs * (size_t)N * (fewz ? 4 : wide), smy = 2 * cs * (size_t)N * (fewy ? 4 : wide);
  // x stage: Y2[b][tz ty][kx] -> CC[b][tz ty][tx]
  const int rows = nt * nt;
  const size_t smx = cs * (8 * (size_t)N + (size_t)N * nt);
  if ((e = allow_smem(midz, smz)) != cudaSuccess || (e = allow_smem(midy, smy)) != cudaSuccess ||
      (e = allow_smem(k_idft_x<T>, smx)) != cudaSuccess)
    return e;
  // FP64: CTAs of two warps, which end more evenly (64 volumes of 24^3, 11 points, z
  // stage: 139 us with four, 120 with two)
  const int thp = sizeof(T) == 8 ? 64 : 128;
  auto packed = [&](long cols) { return dim3((unsigned)((cols + thp - 1) / thp * narrow), 1, B); };
  midz<<<fewz ? packed(N2) : dim3((unsigned)((N2 + 255) / 256), 1, B), fewz ? thp : 128, smz, st>>>(
      (const C2<T> *)w.Z, (C2<T> *)w.Y1, (const C2<T> *)w.E, N, nt, 1, (int)N2, 2, es, narrow);
  if ((e = cudaGetLastError()) != cudaSuccess) return e;
  midy<<<fewy ? packed((long)nt * N) : dim3((N + ty - 1) / ty, nt, B), fewy ? thp : ty, smy, st>>>(
      (const C2<T> *)w.Y1, (C2<T> *)w.Y2, (const C2<T> *)w.E, N, nt, nt, N, 1, es, narrow);
  if ((e = cudaGetLastError()) != cudaSuccess) return e;
  k_idft_x<T><<<dim3((rows + 7) / 8, B), 256, smx, st>>>(
      (const C2<T> *)w.Y2, (T *)w.CC, (const C2<T> *)w.E, N, nt, rows, T(1.0 / ((double)N2 * N)), es);
  if ((e = cudaGetLastError()) != cudaSuccess) return e;
  k_cc_argmax<T><<<B, 256, 0, st>>>((const T *)w.CC, nt, org, j0, den, edge, flag_mode, R, t_out,
                                    tau_out, cc_out, flags);
  return cudaGetLastError();
}

template <typename T>
cudaError_t launch_shift_search(const Plan &p, const float *f, const float *u, int B,
                                int max_shift, int upsample, const double *R, const ShiftWs &w,
                                double *t, double *tau, double *cc, int *flags, cudaStream_t st) {
  if (B <= 0) return cudaSuccess;
  const int N = p.N;
  const long N2 = (long)N * N;
  FftDesc fd;
  fd.N = N;
  fd.npass = p.fft_npass;
  for (int q = 0; q < 16; ++q) fd.radix[q] = p.fft_radix[q];
  const size_t cs = sizeof(C2<T>);
  C2<T> *Z = (C2<T> *)w.Z;
  const C2<T> *tw = (const C2<T> *)p.fft_tw;
  // planes of which two buffers fit an SM (N <= 112 in FP32, 79 in FP64) are transformed
  // whole; larger ones a direction at a time
  cudaError_t e;
  const size_t plane = cs * (2 * (size_t)N * (N | 1) + N);
  if (plane <= 200 * 1024) {
    if ((e = allow_smem(k_fft_plane<T>, plane)) != cudaSuccess) return e;
    // FP64: a thread per radix-4 butterfly at most (64 planes x 16 of 16^2: idle warps'
    // registers kept other planes off the SM, 49 us with 256 threads, 24 with 64)
    const int threads = sizeof(T) == 8 ? std::min(256, std::max(64, (N * N / 4 + 31) / 32 * 32)) : 256;
    k_fft_plane<T><<<dim3(N, B), threads, plane, st>>>(Z, f, u, fd, tw);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
  } else {
    // rows, then columns (at least 16, so their rows stay coalesced), about 4096
    // elements per CTA; fewer where they and the twiddles exceed shared memory (FP64
    // from N = 450 on: eight columns, 128 bytes of a row)
    auto lines = [&](int nb) { return cs * (2 * (size_t)nb * (N | 1) + N); };
    const int NB0 = 4096 / N > 0 ? 4096 / N : 1;
    int NB = 4096 / N > 16 ? 4096 / N : 16;
    while (lines(NB) > SMEM_MOST) NB /= 2;
    const size_t sm0 = lines(NB0), sm1 = lines(NB);
    if ((e = allow_smem(k_fft_axis<T>, sm0 > sm1 ? sm0 : sm1)) != cudaSuccess) return e;
    k_fft_axis<T><<<dim3((unsigned)((N2 + NB0 - 1) / NB0), B), 256, sm0, st>>>(Z, f, u, 0, fd, tw, NB0);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    k_fft_axis<T><<<dim3((unsigned)(N * ((N + NB - 1) / NB)), B), 256, sm1, st>>>(Z, nullptr, nullptr, 1,
                                                                               fd, tw, NB);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
  }
  // columns of the z transform per CTA: 128-byte rows while four buffers of them
  // leave two CTAs on an SM
  int NBz = 128 / (int)cs;
  while (NBz > 1 && cs * (4 * (size_t)NBz + 1) * N > 112 * 1024) NBz /= 2;
  const size_t smz = cs * (4 * (size_t)NBz + 1) * N;
  if ((e = allow_smem(k_fft_cross<T>, smz)) != cudaSuccess) return e;
  const int nself = N % 2 ? 1 : 2, npair = (N - nself) / 2;
  const unsigned zt = nself * ((N / 2 + NBz) / NBz) + npair * ((N + NBz - 1) / NBz);
  k_fft_cross<T><<<dim3(zt, B), 128, smz, st>>>(Z, fd, tw, NBz);
  if ((e = cudaGetLastError()) != cudaSuccess) return e;
  // integer window [-m, m]^3
  const int nw = 2 * max_shift + 1;
  e = idft_grid<T>(p, B, nw, nullptr, -max_shift, 1, max_shift, 1, nullptr, w, w.t0,
                   nullptr, nullptr, flags, st);
  if (e != cudaSuccess) return e;
  // fine grid around the integer peak
  const int h = (int)floor(0.75 * upsample), nf = 2 * h + 1;
  return idft_grid<T>(p, B, nf, w.t0, -h, upsample, 0, 0, R, w, t, tau,
                      cc, flags, st);
}

template cudaError_t launch_shift_search<float>(const Plan &, const float *, const float *, int,
                                                int, int, const double *, const ShiftWs &,
                                                double *, double *, double *, int *, cudaStream_t);
template cudaError_t launch_shift_search<double>(const Plan &, const float *, const float *, int,
                                                 int, int, const double *, const ShiftWs &,
                                                 double *, double *, double *, int *, cudaStream_t);

}  // namespace matcha
