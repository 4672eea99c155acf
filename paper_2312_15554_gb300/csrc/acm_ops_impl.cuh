// acm_ops_impl.cuh -- definitions of the launch wrappers; included once per
// precision (acm_f32.cu, acm_f64.cu) followed by an explicit instantiation.
#pragma once
#include <cstdlib>

#include "acm_kernels.cuh"
#include "acm_ops.h"

namespace acm {

// The default tile width (kx columns) a strided pass reports (see tx_ok; it runs the
// width that lp_width takes from the grid): about 256 threads over its components, at
// least 2 columns, at most 64 KB of shared memory.
constexpr int pick_tx(int csize, int N, int NC) {
  int tl = N / ept(N);
  int tx = 16;
  while (tx > 2 && (NC * tx * tl > 256 || NC * tx * line_stride(N, tl, tx, 128 / csize) * csize > 64 * 1024)) tx /= 2;
  return tx;
}

template <typename K>
static cudaError_t set_smem(K* k, int bytes) {
  return bytes > 48 * 1024 ? cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes)
                           : cudaSuccess;
}

// the strided passes also take lines of one point (axis 0 of a single plane):
// the transform is the identity and the pass applies its operator
#define ACM_DISPATCH_NS(n, FN, ...)             \
  switch (n) {                                  \
    case 1: return FN<T, 1>(__VA_ARGS__);       \
    case 8: return FN<T, 8>(__VA_ARGS__);       \
    case 16: return FN<T, 16>(__VA_ARGS__);     \
    case 32: return FN<T, 32>(__VA_ARGS__);     \
    case 64: return FN<T, 64>(__VA_ARGS__);     \
    case 128: return FN<T, 128>(__VA_ARGS__);   \
    case 256: return FN<T, 256>(__VA_ARGS__);   \
    case 512: return FN<T, 512>(__VA_ARGS__);   \
    default: return cudaErrorInvalidValue;      \
  }

#define ACM_DISPATCH_N(n, FN, ...)     \
  switch (n) {                         \
    case 8: return FN<T, 8>(__VA_ARGS__);     \
    case 16: return FN<T, 16>(__VA_ARGS__);   \
    case 32: return FN<T, 32>(__VA_ARGS__);   \
    case 64: return FN<T, 64>(__VA_ARGS__);   \
    case 128: return FN<T, 128>(__VA_ARGS__); \
    case 256: return FN<T, 256>(__VA_ARGS__); \
    case 512: return FN<T, 512>(__VA_ARGS__); \
    default: return cudaErrorInvalidValue;    \
  }

#define ACM_DISPATCH_NI(n, FN)   \
  switch (n) {                   \
    case 8: return FN<T, 8>();     \
    case 16: return FN<T, 16>();   \
    case 32: return FN<T, 32>();   \
    case 64: return FN<T, 64>();   \
    case 128: return FN<T, 128>(); \
    case 256: return FN<T, 256>(); \
    case 512: return FN<T, 512>(); \
    default: return 1;             \
  }

template <typename T, int N2>
static cudaError_t l_x_local(const Geo& g, int nprob, void* spec, void* u, void* lam, const uint8_t* H,
                             const uint32_t* Hb, StokesDev* prm, double* part, const void* tw, cudaStream_t s) {
  constexpr int smem = xs_smem_bytes<T, N2, 2, 0>();
  static const cudaError_t attr = set_smem(k_x_stokes_local<T, N2>, smem);
  if (attr != cudaSuccess) return attr;
  const XGrid x = xs_grid(g.n0 * g.n1 / XL<T, N2>::LPW);
  k_x_stokes_local<T, N2><<<dim3(x.blocks, nprob, x.csplit), x.warps * 32, xs_smem_bytes<T, N2, 2, 0>(x.warps), s>>>(
      (cx<T>*)spec, (T*)u, (T*)lam, H, Hb, prm, part, g, (const cx<T>*)tw, x.gpw);
  return cudaGetLastError();
}

template <typename T, int N2>
static cudaError_t l_x_rhs(const Geo& g, int nprob, void* spec, const void* u, const void* lam, const uint8_t* H,
                           const uint32_t* Hb, const StokesDev* prm, const void* tw, cudaStream_t s) {
  constexpr int smem = xs_smem_bytes<T, N2, 1, 0>();
  static const cudaError_t attr = set_smem(k_x_stokes_rhs<T, N2>, smem);
  if (attr != cudaSuccess) return attr;
  const XGrid x = xs_grid(g.n0 * g.n1 / XL<T, N2>::LPW);
  k_x_stokes_rhs<T, N2><<<dim3(x.blocks, nprob, x.csplit), x.warps * 32, xs_smem_bytes<T, N2, 1, 0>(x.warps), s>>>(
      (cx<T>*)spec, (const T*)u, (const T*)lam, H, Hb, prm, g, (const cx<T>*)tw, x.gpw);
  return cudaGetLastError();
}

template <typename T, int N2>
static cudaError_t l_x_solute(const Geo& g, int nprob, void* spec, const void* u, const uint8_t* H,
                              const uint32_t* Hb, const SoluteDev* prm, const void* tw, const T* d2, bool central,
                              cudaStream_t s) {
  constexpr int smem = xs_smem_bytes<T, N2, 2, 2 * XL<T, N2>::E>();
  static const cudaError_t attr0 = set_smem(k_x_solute<T, N2, false>, smem);
  static const cudaError_t attr1 = set_smem(k_x_solute<T, N2, true>, smem);
  if (attr0 != cudaSuccess) return attr0;
  if (attr1 != cudaSuccess) return attr1;
  // On grids large enough for gpw > 1, problems that share the velocity and the
  // indicator loop inside the kernel (up to XS_PCACHE per block), with fewer line
  // groups per warp so that the grid keeps its size. On smaller ones the velocity
  // stays in L2 and each problem gets blocks of its own.
  XGrid x = xs_grid(g.n0 * g.n1 / XL<T, N2>::LPW);
  int pshare = 1;
  if (g.us == 0 && g.hs == 0 && x.gpw > 1) {
    pshare = nprob < XS_PCACHE ? nprob : XS_PCACHE;
    x.gpw = XS_GPW / pshare > 1 ? XS_GPW / pshare : 1;
    x.blocks = (g.n0 * g.n1 / XL<T, N2>::LPW + x.warps * x.gpw - 1) / (x.warps * x.gpw);
  }
  const dim3 grid(x.blocks, (nprob + pshare - 1) / pshare);
  auto* k = central ? k_x_solute<T, N2, true> : k_x_solute<T, N2, false>;
  k<<<grid, x.warps * 32, xs_smem_bytes<T, N2, 2, 2 * XL<T, N2>::E>(x.warps), s>>>(
      (cx<T>*)spec, (const T*)u, H, Hb, prm, g, (const cx<T>*)tw, d2, nprob, x.gpw, pshare);
  return cudaGetLastError();
}

template <typename T, int N2, int NC>
static cudaError_t l_x_r2c_nc(const Geo& g, int nprob, void* spec, long long sps, const void* in, long long ips,
                              const void* tw, cudaStream_t s) {
  constexpr int smem = x_smem_bytes<T, N2, NC>();
  static const cudaError_t attr = set_smem(k_x_r2c<T, N2, NC>, smem);
  if (attr != cudaSuccess) return attr;
  dim3 grid((g.n0 * g.n1 + XCfg<T, N2>::LPB - 1) / XCfg<T, N2>::LPB, nprob);
  k_x_r2c<T, N2, NC><<<grid, NC * 64, smem, s>>>((cx<T>*)spec, (const T*)in, g, ips, sps, (const cx<T>*)tw);
  return cudaGetLastError();
}
template <typename T, int N2>
static cudaError_t l_x_r2c(const Geo& g, int nprob, int nc, void* spec, long long sps, const void* in,
                           long long ips, const void* tw, cudaStream_t s) {
  if (nc == 1) return l_x_r2c_nc<T, N2, 1>(g, nprob, spec, sps, in, ips, tw, s);
  if (nc == 3) return l_x_r2c_nc<T, N2, 3>(g, nprob, spec, sps, in, ips, tw, s);
  return cudaErrorInvalidValue;
}

template <typename T, int N2>
static cudaError_t l_x_r2c_lr(const Geo& g, void* spec, const void* in, const void* tw, cudaStream_t s) {
  constexpr int smem = xr_smem_bytes<T, N2>();
  static const cudaError_t attr = set_smem(k_x_r2c_lr<T, N2>, smem);
  if (attr != cudaSuccess) return attr;
  const XGrid x = xs_grid(g.n0 * g.n1 / XL<T, N2>::LPW);
  k_x_r2c_lr<T, N2><<<x.blocks, x.warps * 32, xr_smem_bytes<T, N2>(x.warps), s>>>((cx<T>*)spec, (const T*)in, g,
                                                                                  (const cx<T>*)tw, x.gpw);
  return cudaGetLastError();
}

template <typename T, int N2, int NC>
static cudaError_t l_x_c2r_nc(const Geo& g, int nprob, const void* spec, long long sps, void* out, long long ops,
                              const void* tw, cudaStream_t s) {
  constexpr int smem = x_smem_bytes<T, N2, NC>();
  static const cudaError_t attr = set_smem(k_x_c2r<T, N2, NC>, smem);
  if (attr != cudaSuccess) return attr;
  dim3 grid((g.n0 * g.n1 + XCfg<T, N2>::LPB - 1) / XCfg<T, N2>::LPB, nprob);
  k_x_c2r<T, N2, NC><<<grid, NC * 64, smem, s>>>((const cx<T>*)spec, (T*)out, g, ops, sps, (const cx<T>*)tw);
  return cudaGetLastError();
}
// The line-resident kernel stores voxel pairs as vectors: it runs when `out`
// is aligned to a pair (the strides are even); otherwise the block-phase
// kernel with element stores does.
template <typename T, int N2>
static cudaError_t l_x_c2r(const Geo& g, int nprob, int nc, const void* spec, long long sps, void* out,
                           long long ops, const void* tw, cudaStream_t s) {
  if ((uintptr_t)out % (2 * sizeof(T)) == 0 && ops % 2 == 0 && g.V % 2 == 0) {
    constexpr int smem = xs_smem_bytes<T, N2, 1, 0>();
    static const cudaError_t attr = set_smem(k_x_c2r_lr<T, N2>, smem);
    if (attr != cudaSuccess) return attr;
    const XGrid x = xs_grid(g.n0 * g.n1 / XL<T, N2>::LPW);
    k_x_c2r_lr<T, N2><<<dim3(x.blocks, nprob * nc), x.warps * 32, xs_smem_bytes<T, N2, 1, 0>(x.warps), s>>>(
        (const cx<T>*)spec, (T*)out, g, nc, ops, sps, (const cx<T>*)tw, x.gpw);
    return cudaGetLastError();
  }
  if (nc == 1) return l_x_c2r_nc<T, N2, 1>(g, nprob, spec, sps, out, ops, tw, s);
  if (nc == 3) return l_x_c2r_nc<T, N2, 3>(g, nprob, spec, sps, out, ops, tw, s);
  return cudaErrorInvalidValue;
}

// Tile choices of a pass (Geo::txs): 0 lets the pass pick its width from the
// grid; the solver passes at N >= 64 also take -1, 1, 2 (half, double, four
// times the default width reported) and, at N = 64, 128 and 256, 3 and 4 (a full and
// a half 128-byte row segment, reported as -W). FP32 lines of 128 and 256 points also
// take 5, a quarter segment: what a pass of a small grid picks by itself, so the tuner
// has to be able to pick it too (z Stokes, us a launch at half and quarter segments:
// 22.4 and 17.0 at 256 x 32 x 64, 15.3 and 13.5 at 128 x 64 x 32; y at 16 x 256 x 64
// 10.3 and 8.4).
template <int N, int OP, int NC>
constexpr bool tunable() {
  return N >= 64 && ((OP == OP_FWD && NC == 3) || (OP == OP_INV && NC == 3) || OP == OP_STOKES || OP == OP_SOLUTE ||
                     OP == OP_FWD_SOL || OP == OP_INV_SOL);
}

// Which positive widths are offered: a list that callers may have saved, so it stays
// what it was when a tile of TX columns was one block of at most 1536 line threads and
// 200 KB of shared memory. A pass runs the nearest width it is compiled for
// (lp_width), so several of them can name one kernel.
template <typename T, int N, int OP, int NC, int TX>
constexpr bool tx_ok() {
  return TX >= 2 && TX <= 32 && NC * TX * (N / ept(N)) <= 1536 &&
         (NC * TX * line_stride(N, N / ept(N), TX, wave_slots<T>()) + tw_total(N)) * (int)sizeof(cx<T>) <= 200 * 1024;
}

template <typename T, int N, int OP, int NC>
constexpr bool rr_ok() {
  return (N == 64 || N == 128 || N == 256) && tunable<N, OP, NC>();
}

// columns of one 128-byte row segment (16 in FP32, 8 in FP64)
template <typename T>
constexpr int rr_wdef() { return 128 / (int)sizeof(cx<T>); }

// whether lines of N are compiled for a quarter of that
template <typename T, int N>
constexpr bool rr_quarter() { return sizeof(T) == 4 && (N == 128 || N == 256); }

// the width (T, N, OP, NC) reports under the choice `shift`
template <typename T, int N, int OP, int NC>
constexpr int resolved_tx(int shift) {
  constexpr int TX0 = pick_tx((int)sizeof(cx<T>), N, NC);
  if constexpr (rr_ok<T, N, OP, NC>()) {
    if (shift == 3) return -rr_wdef<T>();
    if (shift == 4) return -rr_wdef<T>() / 2;
    if (shift == 5 && rr_quarter<T, N>()) return -rr_wdef<T>() / 4;
  }
  if (tunable<N, OP, NC>()) {
    if (shift < 0 && tx_ok<T, N, OP, NC, TX0 / 2>()) return TX0 / 2;
    if (shift == 1 && tx_ok<T, N, OP, NC, TX0 * 2>()) return TX0 * 2;
    if (shift == 2 && tx_ok<T, N, OP, NC, TX0 * 4>()) return TX0 * 4;
  }
  return TX0;
}

// Compiled widths of (T, N): powers of two from max(4, the width that fills a
// warp) to a full 128-byte row segment (half of one at N = 512, where three
// groups of wider tiles pass 1024 threads), or the one that fills a warp alone.
template <typename T, int N>
constexpr int lp_wmin() {
  constexpr int TL = N / lp_ept<T>(N);
  return TL >= 8 ? 4 : 32 / TL;
}
static_assert(lp_wmin<float, 128>() == rr_wdef<float>() / 4 && lp_wmin<float, 256>() == rr_wdef<float>() / 4);
template <typename T, int N>
constexpr int lp_wmax() {
  constexpr int m = N == 512 ? rr_wdef<T>() / 2 : rr_wdef<T>();
  return m < lp_wmin<T, N>() ? lp_wmin<T, N>() : m;
}

// The width a pass runs with. Asked for one, the nearest compiled. Left to
// itself, the widest that gives a problem two tiles per SM (152), at most half
// a row segment in the z operators (their three groups of a full segment fill an
// SM's thread budget with one block), so that small grids spread over the SMs and
// large ones read long segments. Depends on the grid alone: a problem's partial
// sums do not depend on how many share its launch.
template <typename T, int N>
static int lp_width(const Geo& g, int axis, int op, int reported) {
  constexpr int lo = lp_wmin<T, N>(), hi = lp_wmax<T, N>();
  const int sh = g.txs[sizeof(T) == 8][axis][op];
  int w = hi;
  if (sh == 0) {
    if ((op == OP_STOKES || op == OP_SOLUTE) && w > lo && w > rr_wdef<T>() / 2) w /= 2;
    const int nouter = axis == 1 ? g.n0 : g.n1;
    while (w > lo && rr_tiles(g.Pu, nouter, w).nlive < 304) w /= 2;
    return w;
  }
  const int want = reported < 0 ? -reported : reported;
  while (w > lo && w > want) w /= 2;
  return w;
}

template <typename T>
static PassArgs<T> pass_args(const Geo& g, int axis, void* spec, long long probStride, const Sym<T>& sym,
                             const void* tw, void* st0, void* st1, StokesDev* sprm, SoluteDev* cprm, double* part,
                             int dm) {
  PassArgs<T> a;
  a.spec = (cx<T>*)spec;
  a.probStride = probStride;
  a.compStride = g.S;
  if (axis == 1) {
    a.rowStride = g.P;
    a.outerStride = (long long)g.n1 * g.P;
  } else {
    a.rowStride = (long long)g.n1 * g.P;
    a.outerStride = g.P;
  }
  a.Pu = g.Pu;
  a.sym = sym;
  a.twg = (const cx<T>*)tw;
  a.st0 = (cx<T>*)st0;
  a.st1 = (cx<T>*)st1;
  a.sprm = sprm;
  a.cprm = cprm;
  a.part = part;
  a.invV = 1.0 / (double)g.V;
  a.nkx = g.n2 / 2;
  a.dm = dm;
  a.nouter = axis == 1 ? g.n0 : g.n1;
  a.src = a.dst = a.spec;
  a.srcRow = a.dstRow = a.rowStride;
  a.srcOuter = a.dstOuter = a.outerStride;
  return a;
}

template <typename T, int N, int OP, int W, bool SEG, bool PLANE = false>
static cudaError_t l_pass_w(const PassArgs<T>& a, int nc, int nprob, cudaStream_t s) {
  using C = LCfg<T, N, W>;
  constexpr int smem = lp_smem<T, N, OP, W>(), threads = lp_groups(OP) * C::NT;
  constexpr auto k = [] {
    if constexpr (OP == OP_STOKES || OP == OP_SOLUTE) return k_lpass_z<T, N, OP, W, SEG, PLANE>;
    else if constexpr (OP == OP_FWD_SOL) return k_lpass_fsol<T, N, OP, W, SEG>;
    else if constexpr (OP == OP_INV_SOL) return k_lpass_isol<T, N, OP, W, SEG>;
    else return k_lpass<T, N, OP, W, SEG>;
  }();
  static const cudaError_t attr = set_smem(k, smem);
  if (attr != cudaSuccess) return attr;
  const int nlive = rr_tiles(a.Pu, a.nouter, W).nlive;
  const dim3 grid = OP == OP_FWD_SOL     ? dim3((nlive + 1) / 2 * 3, nprob)
                    : OP == OP_INV_SOL   ? dim3(3 * nlive, nprob)
                    : lp_groups(OP) == 1 ? dim3(nlive, nc, nprob)
                                         : dim3(nlive, nprob);
  k<<<grid, threads, smem, s>>>(a);
  return cudaGetLastError();
}

template <typename T, int N, int OP, int W, bool SEG>
static cudaError_t l_pass_pick(int w, const PassArgs<T>& a, int nc, int nprob, cudaStream_t s) {
  if constexpr (W > lp_wmin<T, N>())
    if (w < W) return l_pass_pick<T, N, OP, W / 2, SEG>(w, a, nc, nprob, s);
  return l_pass_w<T, N, OP, W, SEG>(a, nc, nprob, s);
}

// Plane cells: y forward, Eq. 13 and y inverse in one pass along axis 1. A plane has
// at most 65 tiles of the narrowest width, so that is the one compiled. The rounding
// follows the y passes' choices, which have to be of one kind (see plane_pass).
template <typename T, int N>
static cudaError_t l_plane(const PassArgs<T>& a, bool seg, int nprob, cudaStream_t s) {
  if constexpr (N >= 8) {
    constexpr int W = lp_wmin<T, N>();
    if constexpr (sizeof(T) == 4 && (N == 64 || N == 128 || N == 256))
      if (seg) return l_pass_w<T, N, OP_STOKES, W, true, true>(a, 3, nprob, s);
    return l_pass_w<T, N, OP_STOKES, W, false, true>(a, 3, nprob, s);
  }
  return cudaErrorInvalidValue;
}
template <typename T, int N>
static cudaError_t l_fft_z(const PassArgs<T>& a, const Geo& g, bool inverse, cudaStream_t s) {
  const int w = lp_width<T, N>(g, 0, OP_FWD, 0);
  return inverse ? l_pass_pick<T, N, OP_INV_SCALE, lp_wmax<T, N>(), false>(w, a, 1, 1, s)
                 : l_pass_pick<T, N, OP_FWD, lp_wmax<T, N>(), false>(w, a, 1, 1, s);
}
template <typename T, int N>
static int l_wmin() { return lp_wmin<T, N>(); }

template <typename T, int N, int OP, int NC>
static cudaError_t l_pass_k(const Geo& g, int axis, int nprob, void* spec, long long probStride, const Sym<T>& sym,
                            const void* tw, void* st0, void* st1, StokesDev* sprm, SoluteDev* cprm, double* part,
                            cudaStream_t s, int dm) {
  const PassArgs<T> a = pass_args<T>(g, axis, spec, probStride, sym, tw, st0, st1, sprm, cprm, part, dm);
  const int sh = g.txs[sizeof(T) == 8][axis][OP];
  const int w = lp_width<T, N>(g, axis, OP, resolved_tx<T, N, OP, NC>(sh));
  // the tuned row-segment widths keep their own rounding (lp_ifft_dit, cmul_fma)
  if constexpr (rr_ok<T, N, OP, NC>() && sizeof(T) == 4)
    if (sh >= 3) return l_pass_pick<T, N, OP, lp_wmax<T, N>(), true>(w, a, NC, nprob, s);
  return l_pass_pick<T, N, OP, lp_wmax<T, N>(), false>(w, a, NC, nprob, s);
}

template <typename T, int N>
static int l_pass_tx(int op, int nc, int shift) {
#define ACM_TX(OPV, NCV) \
  if (op == OPV && nc == NCV) return resolved_tx<T, N, OPV, NCV>(shift);
  ACM_TX(OP_FWD, 1)
  ACM_TX(OP_FWD, 3)
  ACM_TX(OP_INV, 1)
  ACM_TX(OP_INV, 3)
  ACM_TX(OP_INV_SCALE, 1)
  ACM_TX(OP_STOKES, 3)
  ACM_TX(OP_SOLUTE, 2)
  ACM_TX(OP_FWD_SOL, 3)
  ACM_TX(OP_INV_SOL, 3)
  ACM_TX(OP_DERIV, 1)
#undef ACM_TX
  return 0;
}

// the width a pass runs with under g's choice
template <typename T, int N>
static int l_pass_w(const Geo& g, int axis, int op, int nc) {
  return lp_width<T, N>(g, axis, op, l_pass_tx<T, N>(op, nc, g.txs[sizeof(T) == 8][axis][op]));
}

template <typename T, int N>
static cudaError_t l_pass(const Geo& g, int axis, int op, int nc, int nprob, void* spec, long long ps,
                          const Sym<T>& sym, const void* tw, void* st0, void* st1, StokesDev* sprm, SoluteDev* cprm,
                          double* part, cudaStream_t s, int dm) {
#define ACM_PASS(OPV, NCV)                                                                                    \
  if (op == OPV && nc == NCV)                                                                                 \
    return l_pass_k<T, N, OPV, NCV>(g, axis, nprob, spec, ps, sym, tw, st0, st1, sprm, cprm, part, s, dm);
  ACM_PASS(OP_FWD, 1)
  ACM_PASS(OP_FWD, 3)
  ACM_PASS(OP_INV, 1)
  ACM_PASS(OP_INV, 3)
  ACM_PASS(OP_INV_SCALE, 1)
  ACM_PASS(OP_STOKES, 3)
  ACM_PASS(OP_SOLUTE, 2)
  ACM_PASS(OP_FWD_SOL, 3)
  ACM_PASS(OP_INV_SOL, 3)
  ACM_PASS(OP_DERIV, 1)
#undef ACM_PASS
  return cudaErrorInvalidValue;
}

template <typename T>
int Ops<T>::x_blocks(const Geo& g) {
  const int M = g.n2 / 2;
  const int TL = M / xl_ept<T>(M);
  const XGrid x = xs_grid(g.n0 * g.n1 / (32 / TL));
  return x.blocks * x.csplit;
}

template <typename T>
int Ops<T>::pass_tx(const Geo& g, int axis, int op, int nc) {
  const int n = axis == 1 ? g.n1 : g.n0;
  const int sh = g.txs[sizeof(T) == 8][axis][op];
  switch (n) {
    case 1: return l_pass_tx<T, 1>(op, nc, sh);
    case 8: return l_pass_tx<T, 8>(op, nc, sh);
    case 16: return l_pass_tx<T, 16>(op, nc, sh);
    case 32: return l_pass_tx<T, 32>(op, nc, sh);
    case 64: return l_pass_tx<T, 64>(op, nc, sh);
    case 128: return l_pass_tx<T, 128>(op, nc, sh);
    case 256: return l_pass_tx<T, 256>(op, nc, sh);
    case 512: return l_pass_tx<T, 512>(op, nc, sh);
    default: return 0;
  }
}

template <typename T>
bool Ops<T>::tx_variant(int n, int op, int nc, int shift) {
  Geo g;
  g.n0 = g.n1 = n;
  const int t0 = pass_tx(g, 0, op, nc);
  g.txs[sizeof(T) == 8][0][op] = (signed char)shift;
  const int t1 = pass_tx(g, 0, op, nc);
  if (shift >= 3) return t1 < 0;
  return shift == 0 || (t1 != t0 && t1 > 0);
}

template <typename T>
int Ops<T>::pass_columns(const Geo& g, int axis, int op, int nc) {
  switch (axis == 1 ? g.n1 : g.n0) {
    case 1: return l_pass_w<T, 1>(g, axis, op, nc);
    case 8: return l_pass_w<T, 8>(g, axis, op, nc);
    case 16: return l_pass_w<T, 16>(g, axis, op, nc);
    case 32: return l_pass_w<T, 32>(g, axis, op, nc);
    case 64: return l_pass_w<T, 64>(g, axis, op, nc);
    case 128: return l_pass_w<T, 128>(g, axis, op, nc);
    case 256: return l_pass_w<T, 256>(g, axis, op, nc);
    case 512: return l_pass_w<T, 512>(g, axis, op, nc);
    default: return 1;
  }
}

template <typename T>
int Ops<T>::z_blocks(const Geo& g, int op) {
  if (op == P_STOKES && plane_pass(g) >= 0) {
    auto wmin = [&]() -> int { ACM_DISPATCH_NI(g.n1, l_wmin) };
    return rr_tiles(g.Pu, 1, wmin()).nlive;
  }
  return rr_tiles(g.Pu, g.n1, pass_columns(g, 0, op, op == P_SOLUTE ? 2 : 3)).nlive;
}

template <typename T>
cudaError_t Ops<T>::x_stokes_local(const Geo& g, int nprob, void* spec, void* u, void* lam, const uint8_t* H,
                                   const uint32_t* Hb, StokesDev* prm, double* part, const void* tw, cudaStream_t s) {
  ACM_DISPATCH_N(g.n2, l_x_local, g, nprob, spec, u, lam, H, Hb, prm, part, tw, s)
}

template <typename T>
cudaError_t Ops<T>::x_stokes_rhs(const Geo& g, int nprob, void* spec, const void* u, const void* lam,
                                 const uint8_t* H, const uint32_t* Hb, const StokesDev* prm, const void* tw,
                                 cudaStream_t s) {
  ACM_DISPATCH_N(g.n2, l_x_rhs, g, nprob, spec, u, lam, H, Hb, prm, tw, s)
}

template <typename T>
cudaError_t Ops<T>::x_solute(const Geo& g, int nprob, void* spec, const void* u, const uint8_t* H,
                             const uint32_t* Hb, const SoluteDev* prm, const void* tw, const Sym<T>& sym,
                             bool central, cudaStream_t s) {
  ACM_DISPATCH_N(g.n2, l_x_solute, g, nprob, spec, u, H, Hb, prm, tw, sym.d2, central, s)
}

template <typename T>
cudaError_t Ops<T>::x_r2c(const Geo& g, int nprob, int nc, void* spec, long long sps, const void* in, long long ips,
                          const void* tw, cudaStream_t s) {
  ACM_DISPATCH_N(g.n2, l_x_r2c, g, nprob, nc, spec, sps, in, ips, tw, s)
}

template <typename T>
cudaError_t Ops<T>::x_r2c_lr(const Geo& g, void* spec, const void* in, const void* tw, cudaStream_t s) {
  ACM_DISPATCH_N(g.n2, l_x_r2c_lr, g, spec, in, tw, s)
}

template <typename T>
cudaError_t Ops<T>::x_c2r(const Geo& g, int nprob, int nc, const void* spec, long long sps, void* out,
                          long long ops, const void* tw, cudaStream_t s) {
  ACM_DISPATCH_N(g.n2, l_x_c2r, g, nprob, nc, spec, sps, out, ops, tw, s)
}

template <typename T>
cudaError_t Ops<T>::pass(const Geo& g, int axis, int op, int nc, int nprob, void* spec, long long ps,
                         const Sym<T>& sym, const void* tw, void* st0, void* st1, StokesDev* sprm, SoluteDev* cprm,
                         double* part, cudaStream_t s, int dm) {
  const int n = axis == 1 ? g.n1 : g.n0;
  if ((op == P_STOKES || op == P_SOLUTE || op == P_DERIV) && axis != 0) return cudaErrorInvalidValue;
  if ((op == P_FWD_SOL || op == P_INV_SOL) && axis != 1) return cudaErrorInvalidValue;
  ACM_DISPATCH_NS(n, l_pass, g, axis, op, nc, nprob, spec, ps, sym, tw, st0, st1, sprm, cprm, part, s, dm)
}

// codes of the y passes a plane pass stands for: both left to the grid or tuned to
// row segments (-1: mixed, the three passes run in turn)
template <typename T>
int Ops<T>::plane_pass(const Geo& g) {
  if (g.n0 != 1) return -1;
  const auto& t = g.txs[sizeof(T) == 8];
  const bool f = t[1][P_FWD] >= 3, i = t[1][P_INV] >= 3;
  return f != i ? -1 : f;
}

template <typename T>
cudaError_t Ops<T>::plane_stokes(const Geo& g, int nprob, void* spec, long long ps, const Sym<T>& sym, const void* tw,
                                 void* st0, void* st1, StokesDev* sprm, double* part, cudaStream_t s) {
  const int seg = plane_pass(g);
  if (seg < 0) return cudaErrorInvalidValue;
  const PassArgs<T> a = pass_args<T>(g, 1, spec, ps, sym, tw, st0, st1, sprm, nullptr, part, 0);
  ACM_DISPATCH_N(g.n1, l_plane, a, seg == 1, nprob, s)
}

template <typename T>
cudaError_t Ops<T>::fft_z(const Geo& g, bool inverse, const void* src, long long srcPitch, void* dst,
                          long long dstPitch, const void* tw, cudaStream_t s) {
  PassArgs<T> a = pass_args<T>(g, 0, dst, g.S, Sym<T>{}, tw, nullptr, nullptr, nullptr, nullptr, nullptr, 0);
  a.src = (const cx<T>*)src;
  a.dst = (cx<T>*)dst;
  a.srcRow = g.n1 * srcPitch;
  a.srcOuter = srcPitch;
  a.dstRow = g.n1 * dstPitch;
  a.dstOuter = dstPitch;
  ACM_DISPATCH_NS(g.n0, l_fft_z, a, g, inverse, s)
}

template <typename T>
cudaError_t Ops<T>::pore_products(const Geo& g, const void* f, const uint8_t* H, double* part, int nblk,
                                  cudaStream_t s) {
  k_pore_products<T><<<nblk, 256, 0, s>>>((const T*)f, H, g.V, part);
  return cudaGetLastError();
}

template <typename T>
cudaError_t Ops<T>::field_sums(const Geo& g, int nprob, const void* u, const uint8_t* H, double* part, int nblk,
                               cudaStream_t s) {
  dim3 grid(nblk, nprob);
  k_field_sums<T><<<grid, 256, 0, s>>>((const T*)u, H, g.V, g.us, g.hs, part);
  return cudaGetLastError();
}

template <typename T>
cudaError_t Ops<T>::diffusivity(const Geo& g, int nprob, const void* chi, const void* grad, const void* u,
                                const uint8_t* H, const SoluteDev* prm, double* part, int nblk, cudaStream_t s) {
  dim3 grid(nblk, nprob);
  k_diffusivity<T><<<grid, 256, 0, s>>>((const T*)chi, (const T*)grad, (const T*)u, H, g.V, g.us, g.hs, prm, part);
  return cudaGetLastError();
}

template <typename T>
cudaError_t Ops<T>::mask_solid(const Geo& g, const void* in, void* out, const uint8_t* H, cudaStream_t s) {
  k_mask_solid<T><<<608, 256, 0, s>>>((const T*)in, (T*)out, H, g.V);
  return cudaGetLastError();
}

template <typename T>
cudaError_t Ops<T>::div_spec(const Geo& g, const void* uh, void* dv, const Sym<T>& sym, cudaStream_t s) {
  k_div_spec<T><<<608, 256, 0, s>>>((const cx<T>*)uh, (cx<T>*)dv, g, sym);
  return cudaGetLastError();
}

template <typename T>
cudaError_t Ops<T>::q_from_a(const Geo& g, const void* ah, void* q, const Sym<T>& sym, cudaStream_t s) {
  k_q_from_a<T><<<608, 256, 0, s>>>((const cx<T>*)ah, (cx<T>*)q, g, sym);
  return cudaGetLastError();
}

}  // namespace acm
