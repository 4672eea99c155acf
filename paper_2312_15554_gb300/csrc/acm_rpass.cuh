// acm_rpass.cuh -- strided passes: complex FFTs along y or z held in registers.
//
// A line (one kx column of one y or z pencil) of N = E x TL points belongs to TL
// threads of E values each; thread t holds x[t + TL m], m = 0..E-1. The transform
// is a Stockham FFT of radices E, E, ..., N / E^k: the first stage reads exactly
// those positions and the last stage leaves X[t + TL m] in the same thread, so a
// pass loads rows t + TL m straight from global memory, crosses shared memory
// once per further stage (once up to N = E^2, twice at N = 512) and stores the
// same rows; an operator between a forward and an inverse transform finds its
// wavevectors where the inverse wants them.
//
// A tile is W consecutive kx columns of one pencil (W x 8 bytes of a row per
// access in FP32); thread (col, t) = (tid % W, tid / W % TL). When n2/2 and the
// number of pencils are multiples of W, the lone Nyquist column kx = n2/2 of W
// consecutive pencils forms one more tile (lane column `col` takes pencil
// W g + col), so no tile carries idle columns; the tiles of a problem are
// numbered regular ones first (pencil-major), then the Nyquist tiles, and a z
// pass writes one partial-sum record per tile.
//
// A thread holds one component only. The plain y passes give every component a
// block of its own; the passes that combine components (the z operators of
// Eq. 13 and Eq. 20, the y passes of the solute iteration) run one group of
// W x TL threads per component and meet in shared memory. With 16 complex values
// a thread instead of two components' 32 the FP32 kernels fit 64 to 80 registers,
// so 24 to 32 warps stay on an SM and their 16 loads each cover the memory
// latency without software pipelining.
//
// Bank conflicts: position n of a column sits at n + n / E and the columns lie
// an odd multiple of (wavefront slots / W) apart, so that the W columns and the
// consecutive t of one wavefront fall on distinct banks in every stage.
#pragma once
#include "acm_fft.cuh"
#include "acm_types.h"

namespace acm {

// OP_FWD_SOL (y forward of the solute iteration): lines (tau_0, tau_1, s') in,
//   (tau_0, s' + i d1 tau_1) out.
// OP_STOKES (z): Eq. 13 per wavevector with the q^ update of Eq. 9 and the
//   Parseval partials of the divergence residuals.
// OP_SOLUTE (z): (tau_0, s'') in, F^ = s'' + i d0 tau_0, Eq. 20 with the Parseval
//   partials of Eq. 19, (i d0 chi^, chi^) out, chi^ as component SOL_B.
// OP_INV_SOL (y inverse): (a, b) in (b is component SOL_B), lines (a, i d1 b, i d2 b)
//   inverse-transformed out.
enum { OP_FWD = 0, OP_INV = 1, OP_INV_SCALE = 2, OP_STOKES = 3, OP_SOLUTE = 4, OP_DERIV = 5, OP_FWD_SOL = 6,
       OP_INV_SOL = 7 };

// the spectral component (of four per solute problem) that carries chi^ from the z
// pass to the y inverse pass, apart from the latter's outputs
constexpr int SOL_B = 3;

template <typename T>
struct PassArgs {
  cx<T>* spec;
  long long probStride, compStride, rowStride, outerStride;
  // plain passes: where the lines come from and go to (spec and its strides unless
  // the caller's own array takes the place of one of them)
  const cx<T>* src;
  cx<T>* dst;
  long long srcRow, srcOuter, dstRow, dstOuter;
  int Pu;           // used kx columns
  Sym<T> sym;
  const cx<T>* twg; // W_TW_MAX^k
  // operator state
  cx<T>* st0;       // Stokes: q^ ; solute: chi^
  cx<T>* st1;       // Stokes: div^ of the previous iteration
  StokesDev* sprm;
  SoluteDev* cprm;
  double* part;     // per-tile partial sums (stride 4 doubles)
  double invV;
  int nkx;          // n2 / 2 (Nyquist column index)
  int dm;           // OP_DERIV: axis of the derivative
  int nouter;       // pencils along the other strided axis
};

// values per thread: 16 in FP32; short FP64 lines take smaller shares, for more warps
// on the two-lane FP64 pipes (a 32^3 z Stokes pass, 68 tiles of three warps at eight
// values and 136 of half the columns at four: 22 us a launch and 17)
template <typename T>
__host__ __device__ constexpr int lp_ept(int N) {
  if (sizeof(T) == 4) return ept(N);
  return N >= 512 ? 8 : (N >= 128 ? 16 : (N >= 64 ? 8 : (N >= 8 ? 4 : N)));
}

template <typename T, int N, int W>
struct LCfg {
  static constexpr int E = lp_ept<T>(N);
  static constexpr int TL = N / E;   // threads per line
  static constexpr int NT = W * TL;  // threads per component group
  static constexpr int WS = wave_slots<T>();
  // column stride of an exchange buffer
  static constexpr int stride() {
    const int q = W >= WS ? 1 : WS / W;
    int s = N + N / E;
    while (s % q != 0 || (s / q) % 2 == 0) ++s;
    return s;
  }
  static constexpr int BS = stride();
  __device__ static __forceinline__ int at(int n) { return n + n / E; }
};

// The passes that combine components, and their thread groups.
__host__ __device__ constexpr int lp_groups(int op) {
  return op == OP_STOKES ? 3 : (op == OP_SOLUTE || op == OP_FWD_SOL ? 2 : 1);
}

template <typename T, int N, int OP, int W>
__host__ __device__ constexpr int lp_smem() {
  return lp_groups(OP) * W * LCfg<T, N, W>::BS * (int)sizeof(cx<T>);
}

// Blocks per SM the launch bound asks for. FP32: 768 threads an SM, 80 registers a
// thread (64 at 1024 threads in the solute z and y passes, which fit them: z 19 us
// instead of 23 at 128^3); FP64: 512 threads, 128 registers. At most 16 blocks are
// asked for, which leaves one-warp blocks 128 registers, and whole ones: FP64 z Stokes
// in blocks of 192 or 384 threads may take 168, and at N = 512, 768 threads, 80. The
// FP32 z operators spill 4 to 12 bytes at 80 registers, the FP64 Stokes ones 32 in
// blocks of 96 threads at N = 128 and 24 (40 in the plane pass) at 512.
template <typename T, int N, int OP, int W>
__host__ __device__ constexpr int lp_minblocks() {
  const int threads = lp_groups(OP) * LCfg<T, N, W>::NT;
  const int want = sizeof(T) == 8 ? 512 : (OP == OP_SOLUTE || OP == OP_FWD_SOL || OP == OP_INV_SOL ? 1024 : 768);
  const int b = want / threads;
  return b < 1 ? 1 : (b > 16 ? 16 : b);
}

// The live tiles of one problem: nreg = gxr pencils x column blocks, then (when
// the Nyquist column is packed) nouter / W Nyquist tiles.
struct RTiles {
  int gxr;     // regular column blocks per pencil
  int nouter;  // pencils
  int nyq;     // 1: the Nyquist column is packed into tiles of its own
  int nlive;   // tiles per problem
};

__host__ __device__ inline RTiles rr_tiles(int Pu, int nouter, int W) {
  RTiles r;
  r.nouter = nouter;
  r.nyq = ((Pu - 1) % W == 0 && nouter % W == 0) ? 1 : 0;
  r.gxr = r.nyq ? (Pu - 1) / W : (Pu + W - 1) / W;
  r.nlive = r.gxr * nouter + (r.nyq ? nouter / W : 0);
  return r;
}

// pencil and kx column of lane column `col` in tile r of a problem
__device__ __forceinline__ void rr_tile_lane(const RTiles& tl, int r, int W, int col, int Pu, int* outer, int* kx) {
  const int nreg = tl.gxr * tl.nouter;
  if (r < nreg) {
    *outer = r / tl.gxr;
    *kx = (r % tl.gxr) * W + col;
  } else {
    *outer = (r - nreg) * W + col;
    *kx = Pu - 1;
  }
}

// W_N^{e}, or its conjugate for the inverse transform (0 <= e < N). The threads of
// a warp share at most 32 / W values of t, so a read of the table is a broadcast.
template <typename T, int N, int SIGN>
__device__ __forceinline__ cx<T> lp_tw(const cx<T>* __restrict__ twg, int e) {
  cx<T> w = twg[e * (TW_MAX / N)];
  if constexpr (SIGN > 0) w.y = -w.y;
  return w;
}

// Stages after the first, from span Ns on (see the head of the file). b: the
// column's exchange buffer, holding the outputs of the previous stage.
template <typename T, int N, int W, int Ns, int SIGN, int F>
__device__ __forceinline__ void lp_stage(cx<T> (&v)[LCfg<T, N, W>::E], cx<T>* b, const cx<T>* __restrict__ twg, int t) {
  using C = LCfg<T, N, W>;
  constexpr int E = C::E, TL = C::TL, R = N / Ns >= E ? E : N / Ns, NB = E / R;
  cx<T> u[E];
#pragma unroll
  for (int i = 0; i < NB; ++i) {
    const int j = t + TL * i, jm = j & (Ns - 1);
#pragma unroll
    for (int r = 0; r < R; ++r) u[i * R + r] = b[C::at(j + r * (N / R))];
#pragma unroll
    for (int r = 1; r < R; ++r) u[i * R + r] = cmul_fma<F>(u[i * R + r], lp_tw<T, N, SIGN>(twg, jm * r * (N / (Ns * R))));
    dft<R, SIGN>(&u[i * R]);
  }
  if constexpr (Ns * R == N) {
#pragma unroll
    for (int i = 0; i < NB; ++i)
#pragma unroll
      for (int r = 0; r < R; ++r) v[i + NB * r] = u[i * R + r];
  } else {
    __syncthreads();  // every thread has read its inputs
#pragma unroll
    for (int i = 0; i < NB; ++i) {
      const int j = t + TL * i, jm = j & (Ns - 1);
#pragma unroll
      for (int r = 0; r < R; ++r) b[C::at((j - jm) * R + jm + r * Ns)] = u[i * R + r];
    }
    __syncthreads();
    lp_stage<T, N, W, Ns * R, SIGN, F>(v, b, twg, t);
  }
}

// Transform of one line: v[m] = x[t + TL m] in, X[t + TL m] out. b must be free on
// entry and may still be read by other threads of the line on return.
template <typename T, int N, int W, int SIGN, int F = (SIGN < 0 ? 0 : 1)>
__device__ __forceinline__ void lp_fft(cx<T> (&v)[LCfg<T, N, W>::E], cx<T>* b, const cx<T>* __restrict__ twg, int t) {
  using C = LCfg<T, N, W>;
  constexpr int E = C::E;
  dft<E, SIGN>(v);
  if constexpr (N > E) {
#pragma unroll
    for (int r = 0; r < E; ++r) b[C::at(t * E + r)] = v[r];
    __syncthreads();
    lp_stage<T, N, W, E, SIGN, F>(v, b, twg, t);
  }
}

// DFT of radix R of x[k] d[k], the first butterflies x_k d_k +- x_l d_l (l = k +
// R/2) as one multiply-add on the rounded product x_l d_l
template <int R>
__device__ __forceinline__ void dft_scaled(cx<float>* x, const float* d) {
  cx<float> s[R / 2], q[R / 2];
#pragma unroll
  for (int k = 0; k < R / 2; ++k) {
    const cx<float> a = x[k];
    const float px = __fmul_rn(x[k + R / 2].x, d[k + R / 2]), py = __fmul_rn(x[k + R / 2].y, d[k + R / 2]);
    s[k] = mk<float>(__fmaf_rn(a.x, d[k], px), __fmaf_rn(a.y, d[k], py));
    q[k] = mk<float>(__fmaf_rn(a.x, d[k], -px), __fmaf_rn(a.y, d[k], -py));
  }
  dft_tail<R, +1>(s, q, x);
}

// Inverse transform in the other order of the two stages (radix TL, then 16): the
// same result up to rounding; d (SCALED) multiplies the inputs. The row-segment
// widths (SEG, tile choices -16 and -8 in FP32) have always used it at N = 64 and
// 128, and keep it, like their contraction, so that tuned results stay as they were.
template <typename T, int N, int W, bool SCALED>
__device__ __forceinline__ void lp_ifft_dit(cx<T> (&v)[LCfg<T, N, W>::E], const T* d, cx<T>* b,
                                            const cx<T>* __restrict__ twg, int s) {
  using C = LCfg<T, N, W>;
  constexpr int E = C::E, TL = C::TL, NB = E / TL;
#pragma unroll
  for (int i = 0; i < NB; ++i) {
    const int k1 = s + TL * i;
    cx<T> u[TL];
    T du[TL];
#pragma unroll
    for (int k2 = 0; k2 < TL; ++k2) {
      u[k2] = v[i + NB * k2];
      if constexpr (SCALED) du[k2] = d[i + NB * k2];
    }
    if constexpr (SCALED) dft_scaled<TL>(u, du);
    else dft<TL, +1>(u);
#pragma unroll
    for (int tt = 1; tt < TL; ++tt) u[tt] = cmul_fma<1>(u[tt], lp_tw<T, N, +1>(twg, tt * k1));
#pragma unroll
    for (int tt = 0; tt < TL; ++tt) b[C::at(tt * E + k1)] = u[tt];
  }
  __syncthreads();
#pragma unroll
  for (int k1 = 0; k1 < E; ++k1) v[k1] = b[C::at(s * E + k1)];
  dft<E, +1>(v);
}

template <typename T, int N>
__host__ __device__ constexpr bool lp_has_dit() { return sizeof(T) == 4 && (N == 64 || N == 128); }

template <typename T, int N, int W, bool SEG>
__device__ __forceinline__ void lp_inverse(cx<T> (&v)[LCfg<T, N, W>::E], cx<T>* b, const cx<T>* __restrict__ twg,
                                           int t) {
  if constexpr (SEG && lp_has_dit<T, N>()) lp_ifft_dit<T, N, W, false>(v, nullptr, b, twg, t);
  else lp_fft<T, N, W, +1>(v, b, twg, t);
}

// the inverse of x[m] d[m] in the SEG rounding (N <= 256: one exchange)
template <int N, int W>
__device__ __forceinline__ void lp_inverse_scaled(cx<float> (&v)[LCfg<float, N, W>::E], const float* d, cx<float>* b,
                                                  const cx<float>* __restrict__ twg, int t) {
  if constexpr (lp_has_dit<float, N>()) {
    lp_ifft_dit<float, N, W, true>(v, d, b, twg, t);
  } else {
    using C = LCfg<float, N, W>;
    dft_scaled<C::E>(v, d);
#pragma unroll
    for (int r = 0; r < C::E; ++r) b[C::at(t * C::E + r)] = v[r];
    __syncthreads();
    lp_stage<float, N, W, C::E, +1, 1>(v, b, twg, t);
  }
}

template <typename T, int E>
__device__ __forceinline__ void lp_load(cx<T> (&v)[E], const cx<T>* __restrict__ src, long long step, bool ok) {
#pragma unroll
  for (int m = 0; m < E; ++m) v[m] = ok ? src[m * step] : mk<T>(0, 0);
}

template <typename T, int E>
__device__ __forceinline__ void lp_store(const cx<T> (&v)[E], cx<T>* __restrict__ dst, long long step, bool ok) {
  if (!ok) return;
#pragma unroll
  for (int m = 0; m < E; ++m) dst[m * step] = v[m];
}

// Plain passes (OP_FWD, OP_INV, OP_INV_SCALE, and OP_DERIV: forward, times
// i d / V, inverse): block (tile, component, problem).
template <typename T, int N, int OP, int W, bool SEG>
__global__ void __launch_bounds__(LCfg<T, N, W>::NT, (lp_minblocks<T, N, OP, W>())) k_lpass(PassArgs<T> a) {
  using C = LCfg<T, N, W>;
  constexpr int E = C::E, TL = C::TL;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int p = blockIdx.z;
  if ((a.sprm && a.sprm[p].done) || (a.cprm && a.cprm[p].done)) return;
  const int col = threadIdx.x % W, t = threadIdx.x / W;
  cx<T>* b = reinterpret_cast<cx<T>*>(smem_raw) + col * C::BS;
  const RTiles tl = rr_tiles(a.Pu, a.nouter, W);
  int outer, kx;
  rr_tile_lane(tl, blockIdx.x, W, col, a.Pu, &outer, &kx);
  const bool ok = kx < a.Pu;
  const long long field = p * a.probStride + blockIdx.y * a.compStride + kx;
  cx<T> v[E];
  lp_load(v, a.src + field + outer * a.srcOuter + t * a.srcRow, TL * a.srcRow, ok);
  if constexpr (OP == OP_FWD) {
    lp_fft<T, N, W, -1, SEG ? 1 : 0>(v, b, a.twg, t);
  } else {
    if constexpr (OP == OP_INV_SCALE) {
      const T s = (T)a.invV;
#pragma unroll
      for (int m = 0; m < E; ++m) v[m] = mk<T>(mul_rn(v[m].x, s), mul_rn(v[m].y, s));
    }
    if constexpr (OP == OP_DERIV) {
      lp_fft<T, N, W, -1, SEG ? 1 : 0>(v, b, a.twg, t);
      __syncthreads();  // the buffer is free for the inverse
      const T invV = (T)a.invV;
#pragma unroll
      for (int m = 0; m < E; ++m) {
        const T d = !ok ? (T)0 : (a.dm == 0 ? a.sym.d0[t + TL * m] : (a.dm == 1 ? a.sym.d1[outer] : a.sym.d2[kx]));
        const cx<T> x = mul_i(v[m]);
        v[m] = mk<T>(mul_rn(x.x, d * invV), mul_rn(x.y, d * invV));
      }
    }
    lp_inverse<T, N, W, SEG>(v, b, a.twg, t);
  }
  lp_store(v, a.dst + field + outer * a.dstOuter + t * a.dstRow, TL * a.dstRow, ok);
}

// The y forward pass of the solute iteration, two groups of threads a block. Of
// three blocks two take tau_1 and s' of one tile each, one per group, and one takes
// two tiles of tau_0, which stands alone. (All three lines in one block held tau_0 at
// the others' barriers: 237 us a launch at 256^3 and three problems, now 215.)
// Blocks (job, problem).
template <typename T, int N, int OP, int W, bool SEG>
__global__ void __launch_bounds__(2 * LCfg<T, N, W>::NT, (lp_minblocks<T, N, OP, W>())) k_lpass_fsol(PassArgs<T> a) {
  using C = LCfg<T, N, W>;
  constexpr int E = C::E, TL = C::TL, NT = C::NT;
  static_assert(OP == OP_FWD_SOL, "y forward pass of the solute iteration");
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int p = blockIdx.y;
  if (a.cprm && a.cprm[p].done) return;
  const int grp = threadIdx.x / NT, lid = threadIdx.x % NT, col = lid % W, t = lid / W;
  cx<T>* bufs = reinterpret_cast<cx<T>*>(smem_raw);
  cx<T>* b = bufs + (grp * W + col) * C::BS;
  const RTiles tl = rr_tiles(a.Pu, a.nouter, W);
  const int m3 = blockIdx.x % 3;
  const bool pair = m3 < 2;
  const int tile = 2 * ((int)blockIdx.x / 3) + (pair ? m3 : grp);
  int outer, kx;
  rr_tile_lane(tl, tile, W, col, a.Pu, &outer, &kx);
  const bool ok = kx < a.Pu && tile < tl.nlive;
  cx<T>* base = a.spec + p * a.probStride + (long long)outer * a.outerStride + kx + t * a.rowStride;
  const long long step = TL * a.rowStride;
  cx<T> v[E];
  lp_load(v, base + (pair ? 1 + grp : 0) * a.compStride, step, ok);
  lp_fft<T, N, W, -1, SEG ? 1 : 0>(v, b, a.twg, t);
  if (pair) {
    __syncthreads();  // all reads of the exchange buffers are done
    // tau_1^ to the group that holds s'^, through slots private to (lid, m)
    cx<T>* slot = bufs + lid;
    if (grp == 0) {
#pragma unroll
      for (int m = 0; m < E; ++m) slot[m * NT] = v[m];
    }
    __syncthreads();
    if (grp == 0) return;
#pragma unroll
    for (int m = 0; m < E; ++m) v[m] = v[m] + cscale(mul_i(slot[m * NT]), a.sym.d1[t + TL * m]);
  }
  lp_store(v, base + (pair ? 1 : 0) * a.compStride, step, ok);
}

// The y inverse pass of the solute iteration: a (component 0) and b (component 3,
// SOL_B) in, the inverse transforms of a, i d1 b and i d2 b out as components 0, 1 and
// 2. b lies apart from the outputs, so each line is a block of its own with no
// barrier between lines, and the two blocks that read b run side by side (the second
// read hits L2). Blocks (3 tile + line, problem). At 256^3 and three problems, us a
// launch: three lines in one thread's turn 220, two groups sharing b 229 to 243, b
// parked in shared memory 282; this 205.
template <typename T, int N, int OP, int W, bool SEG>
__global__ void __launch_bounds__(LCfg<T, N, W>::NT, (lp_minblocks<T, N, OP, W>())) k_lpass_isol(PassArgs<T> a) {
  using C = LCfg<T, N, W>;
  constexpr int E = C::E, TL = C::TL;
  static_assert(OP == OP_INV_SOL, "y inverse pass of the solute iteration");
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int p = blockIdx.y;
  if (a.cprm && a.cprm[p].done) return;
  const int col = threadIdx.x % W, t = threadIdx.x / W;
  cx<T>* b = reinterpret_cast<cx<T>*>(smem_raw) + col * C::BS;
  const RTiles tl = rr_tiles(a.Pu, a.nouter, W);
  const int line = blockIdx.x % 3;
  int outer, kx;
  rr_tile_lane(tl, blockIdx.x / 3, W, col, a.Pu, &outer, &kx);
  const bool ok = kx < a.Pu;
  cx<T>* base = a.spec + p * a.probStride + (long long)outer * a.outerStride + kx + t * a.rowStride;
  const long long step = TL * a.rowStride;
  cx<T> v[E];
  lp_load(v, base + (line == 0 ? 0 : SOL_B) * a.compStride, step, ok);
  if (line == 1) {
    // i d1(ky) b before the inverse transform along axis 1
    T d[E];
#pragma unroll
    for (int m = 0; m < E; ++m) {
      v[m] = mul_i(v[m]);
      d[m] = a.sym.d1[t + TL * m];
    }
    if constexpr (SEG && sizeof(T) == 4) {
      lp_inverse_scaled<N, W>(v, d, b, a.twg, t);
    } else {
#pragma unroll
      for (int m = 0; m < E; ++m) v[m] = mk<T>(mul_rn(v[m].x, d[m]), mul_rn(v[m].y, d[m]));
      lp_inverse<T, N, W, SEG>(v, b, a.twg, t);
    }
  } else {
    lp_inverse<T, N, W, SEG>(v, b, a.twg, t);
    if (line == 2) {
      // i d2(kx), a factor per column, after the (linear) transform
      const T d2 = ok ? a.sym.d2[kx] : (T)0;
#pragma unroll
      for (int m = 0; m < E; ++m) v[m] = cscale(mul_i(v[m]), d2);
    }
  }
  lp_store(v, base + line * a.compStride, step, ok);
}

// The z passes with the Green operators: one group of threads per component. The
// transformed components meet in slots of the exchange buffers (component c of
// element e of thread lid at bufs[c][e NT + lid]), where the groups share the
// elements out (e = grp, grp + NC, ...); the operator state of a thread's share is
// read once its own component has left the registers (with the inputs it would
// live through the forward transform: spills, 577 us a launch against 544 at
// 256^3 and three problems). Issue slots bound these passes (40% busy, DRAM at
// half its rate): two transforms and the operator are about 1750 instructions a
// thread. Against one thread per line holding two components at a time (166
// registers, 12 warps an SM) z Stokes takes 544 us for 606, z solute 327 for 338
// in the block-wide tile it used; 512^3 lines, block-wide before, 5.56 ms for 6.56.
//
// PLANE: lines along axis 1 of a cell of one plane (n0 = 1, kz = 0). Axis 0 has no
// transform there, so this is the whole of y forward, Green step and y inverse: three
// launches of 5 to 6 us at 128 x 128 become one. Blocks (tile, problem).
template <typename T, int N, int OP, int W, bool SEG, bool PLANE>
__global__ void __launch_bounds__(lp_groups(OP) * LCfg<T, N, W>::NT, (lp_minblocks<T, N, OP, W>()))
    k_lpass_z(PassArgs<T> a) {
  using C = LCfg<T, N, W>;
  constexpr int E = C::E, TL = C::TL, NT = C::NT, NC = lp_groups(OP), K = (E + NC - 1) / NC;
  constexpr int CB = W * C::BS;
  static_assert(CB >= E * NT, "a component's slots fit its exchange buffer");
  extern __shared__ __align__(16) unsigned char smem_raw[];
  cx<T>* bufs = reinterpret_cast<cx<T>*>(smem_raw);
  __shared__ T red[4 * 32];
  __shared__ T opar[5];
  const int p = blockIdx.y;
  if ((a.sprm && a.sprm[p].done) || (a.cprm && a.cprm[p].done)) return;
  const int grp = threadIdx.x / NT, lid = threadIdx.x % NT, col = lid % W, t = lid / W;
  const RTiles tl = rr_tiles(a.Pu, a.nouter, W);
  int outer, kx;
  rr_tile_lane(tl, blockIdx.x, W, col, a.Pu, &outer, &kx);
  const bool ok = kx < a.Pu;
  const long long off = (long long)outer * a.outerStride + kx + t * a.rowStride;
  const long long step = TL * a.rowStride;
  cx<T>* base = a.spec + p * a.probStride + grp * a.compStride + off;
  cx<T>* st0 = a.st0 + (long long)p * a.compStride + off;
  cx<T>* st1 = OP == OP_STOKES ? a.st1 + (long long)p * a.compStride + off : nullptr;
  cx<T> v[E], sa[K], sb[K];
  lp_load(v, base, step, ok);
  if (threadIdx.x == 0) {
    // the operator's parameters, converted once per block
    if constexpr (OP == OP_STOKES) {
      opar[0] = (T)a.sprm[p].nu;
      opar[1] = (T)a.sprm[p].psi[1];
      opar[2] = (T)a.sprm[p].psi[2];
    } else {
      opar[0] = (T)a.cprm[p].A0;
      for (int k = 0; k < 3; ++k) opar[1 + k] = (T)a.cprm[p].B0[k];
    }
    opar[4] = (T)a.invV;
  }
  lp_fft<T, N, W, -1, SEG ? 1 : 0>(v, bufs + grp * CB + col * C::BS, a.twg, t);
  __syncthreads();
  cx<T>* slot = bufs + lid;
#pragma unroll
  for (int e = 0; e < E; ++e) slot[grp * CB + e * NT] = v[e];
#pragma unroll
  for (int k = 0; k < K; ++k) {
    const int e = grp + NC * k;
    const bool in = ok && e < E;
    sa[k] = in ? st0[e * step] : mk<T>(0, 0);
    if constexpr (OP == OP_STOKES) sb[k] = in ? st1[e * step] : mk<T>(0, 0);
  }
  __syncthreads();
  const T invV = opar[4];
  const T d2 = ok ? a.sym.d2[kx] : (T)0, l2 = ok ? a.sym.l2[kx] : (T)0;
  const T wgt = (kx == 0 || kx == a.nkx) ? (T)1 : (T)2;
  // symbols of the other strided axis (read once: the stores below may alias them)
  const T db = PLANE ? a.sym.d0[0] : a.sym.d1[outer], lb = PLANE ? a.sym.l0[0] : a.sym.l1[outer];
  const T lb2 = lb + l2, db2 = sum2<false>(db, db, d2, d2);
  T acc[3] = {(T)0, (T)0, (T)0};
#pragma unroll
  for (int k = 0; k < K; ++k) {
    const int e = grp + NC * k;
    if (e >= E) break;
    const int row = t + TL * e, kz = PLANE ? 0 : row, ky = PLANE ? row : outer;
    // the symbols of the line's axis, per element, beside the block's own
    const T dline = PLANE ? a.sym.d1[row] : a.sym.d0[row], lr = PLANE ? a.sym.l1[row] : a.sym.l0[row];
    const T d0 = PLANE ? db : dline, l0 = PLANE ? lb : lr, d1 = PLANE ? dline : db, l1 = PLANE ? lr : lb;
    const T l12 = PLANE ? l1 + l2 : lb2, d12 = PLANE ? sum2<false>(d1, d1, d2, d2) : db2;
    const T L = l0 + l12, dd = d0 * d0 + d12;
    const bool k0 = (kz == 0 && ky == 0 && kx == 0);
    cx<T>* s0 = slot + e * NT;
    cx<T>* s1 = s0 + CB;
    if constexpr (OP == OP_STOKES) {
      const T nu = opar[0], beta = opar[1], b = opar[2];
      cx<T>* s2 = s1 + CB;
      const cx<T> qh = sa[k];
      // r = w^ - i d q^ (+ g V at k = 0)
      const cx<T> iq = mul_i(qh);
      cx<T> r0 = *s0 - cscale(iq, d0), r1 = *s1 - cscale(iq, d1), r2 = *s2 - cscale(iq, d2);
      if (k0) {
        const StokesDev& P = a.sprm[p];
        const T Vt = (T)(1.0 / a.invV);
        r0.x += (T)P.g[0] * Vt;
        r1.x += (T)P.g[1] * Vt;
        r2.x += (T)P.g[2] * Vt;
      }
      // Eq. 13: (nu L + b) u^ + beta d (d.u^) = r, solved as
      //   d.u^ = d.r / (c + beta |d|^2),  u^ = (r - beta d (d.u^)) / c,  c = nu L + b
      const T c0 = nu * L + b;
      const T ic0 = (T)1 / c0;
      const cx<T> dr = mk<T>(fma_rn(r2.x, d2, sum2<true>(r0.x, d0, r1.x, d1)),
                             fma_rn(r2.y, d2, sum2<false>(r0.y, d0, r1.y, d1)));
      const cx<T> du = cscale(dr, (T)1 / fma_rn(beta, dd, c0));
      const cx<T> f = cscale(du, beta);
      const cx<T> u0 = cscale(r0 - cscale(f, d0), ic0);
      const cx<T> u1 = cscale(r1 - cscale(f, d1), ic0);
      const cx<T> u2 = cscale(r2 - cscale(f, d2), ic0);
      // div u^ = i d.u^ (taken from the solve, free of the cancellation of
      // summing d_c u^_c when beta is large); Eq. 9: q^ <- q^ - beta div u^
      const cx<T> dv = mul_i(du);
      const cx<T> qn = mk<T>(qh.x - mul_rn(dv.x, beta), qh.y - mul_rn(dv.y, beta));
      if (ok) {
        st0[e * step] = qn;
        st1[e * step] = dv;
        const cx<T> ddv = dv - sb[k];
        acc[0] += wgt * cabs2(dv);
        acc[1] += wgt * cabs2(ddv);
        acc[2] += wgt * cabs2(qn);
      }
      if (k0) {
        a.sprm[p].mean_u[0] = (double)u0.x * a.invV;
        a.sprm[p].mean_u[1] = (double)u1.x * a.invV;
        a.sprm[p].mean_u[2] = (double)u2.x * a.invV;
      }
      *s0 = cscale(u0, invV);
      *s1 = cscale(u1, invV);
      *s2 = cscale(u2, invV);
    } else {
      // F^ = s^ + i d.tau^ (Eq. 18 in Fourier space): the axis-2 and axis-1
      // terms were added in the x and y passes, component 1 holds s''
      const T A0 = opar[0];
      const cx<T> F = mk<T>(fma_rn(-s0->y, d0, s1->x), fma_rn(s0->x, d0, s1->y));
      // Eq. 20: chi^ = F^ / (i B0.d + A0 L), chi^(0) = 0
      const T dre = mul_rn(A0, L), dim = sum2<false>(opar[1], d0, opar[2], d1) + mul_rn(opar[3], d2);
      cx<T> chi = mk<T>(0, 0);
      if (!k0 && ok) {
        const T den = (T)1 / sum2<true>(dre, dre, dim, dim);
        chi = mk<T>(sum2<true>(F.x, dre, F.y, dim) * den, sum2<false>(F.y, dre, -F.x, dim) * den);
      }
      if (ok) {
        const cx<T> dch = chi - sa[k];
        st0[e * step] = chi;
        acc[0] += wgt * cabs2(dch);
        acc[1] += wgt * dd * cabs2(dch);
      }
      // i d0 chi^ and chi^, normalised for the inverse transform (the axis-1 and
      // axis-2 derivatives are taken in the later passes)
      const cx<T> cs = cscale(chi, invV);
      *s0 = cscale(mul_i(cs), d0);
      *s1 = cs;
    }
  }
  block_sum_store<3>(acc, red, a.part + ((long long)p * tl.nlive + blockIdx.x) * 4);
  __syncthreads();
#pragma unroll
  for (int e = 0; e < E; ++e) v[e] = slot[grp * CB + e * NT];
  __syncthreads();  // every thread holds its slots before the buffers carry the inverse
  lp_inverse<T, N, W, SEG>(v, bufs + grp * CB + col * C::BS, a.twg, t);
  if (OP == OP_SOLUTE && grp == 1) base += (SOL_B - 1) * a.compStride;
  lp_store(v, base, step, ok);
}

}  // namespace acm
