// acm_fno.cu -- the learned warm start: a 3D Fourier neural operator with
// hand-written forward and backward kernels (BF16 weights and stored
// activations, FP32 arithmetic and accumulation) and an AdamW step.
//
// Model (width W, `modes` per axis, L layers) on a grid (n0, n1, n2):
//   features a = (H, x0, x1, x2) with x_c = (i_c + 1/2)/n_c
//   lift     v0 = P a + p
//   layer l  v_{l+1} = gelu(z_l),  z_l = G(R_l F(v_l)) + M_l v_l + m_l
//            F: forward DFT on the kept modes; G(Y) = (1/V) sum_k w_k Re[Y(k) e^{2 pi i k.x/n}]
//            (w_k = 1 on the k2 = 0 plane, 2 elsewhere); R_l(k): W x W complex per kept mode
//   project  out = Q v_L + q   (u and lambda, 6 channels)
// Kept modes: k2 in [0, modes), k1 and k0 in [0, modes) U [n - modes, n).
// Loss: (1/(B V)) sum [ |out_u - t_u|^2 + H |out_lambda - t_lambda|^2 ].
//
// F and G are pruned to the kept modes. With C = batch x W fields the spectra pass
// through three compact buffers:
//   A [C][n0][n1][modes]            after the transform along axis 2,
//   B [C][n0][2 modes][modes]       after the one along axis 1 (kept k1 rows),
//   X [C][2 modes][2 modes][modes]  after the one along axis 0: the kept modes;
// G goes the same way back. Each transform is the one-dimensional transform of the
// solver passes (same stages, same rounding); rows and columns that the truncation
// drops or that are zero are not moved. The last step back, along axis 2, also
// applies the pointwise layer, so the W x W contraction and the activation read
// the spectral term from shared memory.
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstring>
#include <type_traits>
#include <vector>

#include "acm.h"
#include "acm_kernels.cuh"
#include "acm_ops.h"

using namespace acm;

namespace {

constexpr int NRB = 512;  // most blocks (partials) of the loss and weight-gradient reductions

struct FnoDims {
  int n0, n1, n2, W, md, L;
  long long V;
  int M;  // kept modes
};

__device__ __forceinline__ float bf(const __nv_bfloat16 x) { return __bfloat162float(x); }

__device__ __forceinline__ float gelu_f(float z) { return 0.5f * z * (1.0f + erff(z * 0.70710678118654752f)); }

__device__ __forceinline__ float gelu_grad_f(float z) {
  return 0.5f * (1.0f + erff(z * 0.70710678118654752f)) + z * 0.3989422804014327f * expf(-0.5f * z * z);
}

// two FP32 multiply-adds in one issue slot (each rounded as fmaf); pairs travel as
// float2 in one 64-bit register
__device__ __forceinline__ float2 fma2(float2 a, float2 b, float2 c) {
  unsigned long long d;
  asm("fma.rn.f32x2 %0, %1, %2, %3;"
      : "=l"(d)
      : "l"(*reinterpret_cast<unsigned long long*>(&a)), "l"(*reinterpret_cast<unsigned long long*>(&b)),
        "l"(*reinterpret_cast<unsigned long long*>(&c)));
  return *reinterpret_cast<float2*>(&d);
}

// ---------------------------------------------------------------------------
// lift: v0[b][c][x] = sum_a P[c][a] a_a(x) + p[c]
// ---------------------------------------------------------------------------
template <int W>
__global__ void __launch_bounds__(256) k_lift(const uint8_t* __restrict__ H, const __nv_bfloat16* __restrict__ P,
                                             const __nv_bfloat16* __restrict__ pb, __nv_bfloat16* __restrict__ v0,
                                             FnoDims d, int B) {
  __shared__ float sP[W * 4], sp[W];
  for (int i = threadIdx.x; i < W * 4; i += blockDim.x) sP[i] = bf(P[i]);
  for (int i = threadIdx.x; i < W; i += blockDim.x) sp[i] = bf(pb[i]);
  __syncthreads();
  const long long total = (long long)B * d.V;
  for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < total; t += (long long)gridDim.x * blockDim.x) {
    const long long b = t / d.V, x = t - b * d.V;
    const int i2 = (int)(x % d.n2), i1 = (int)((x / d.n2) % d.n1), i0 = (int)(x / ((long long)d.n2 * d.n1));
    const float a[4] = {(float)H[t], (i0 + 0.5f) / d.n0, (i1 + 0.5f) / d.n1, (i2 + 0.5f) / d.n2};
    __nv_bfloat16* o = v0 + b * W * d.V + x;
#pragma unroll 4
    for (int c = 0; c < W; ++c)
      o[c * d.V] = __float2bfloat16(sp[c] + sP[c * 4] * a[0] + sP[c * 4 + 1] * a[1] + sP[c * 4 + 2] * a[2] +
                                    sP[c * 4 + 3] * a[3]);
  }
}

// ---------------------------------------------------------------------------
// pruned transforms
// ---------------------------------------------------------------------------
// F along axis 2: real lines (BF16 activations or FP32) to the kept columns of A.
// Bound by its reads: 67 MB of BF16 or 134 MB of FP32 at 64^3 with 128 fields.
template <int N2, typename In>
__global__ void __launch_bounds__(64) k_fno_x_fwd(const In* __restrict__ in, cx<float>* __restrict__ A, int md,
                                                 const cx<float>* __restrict__ twg) {
  using C = XCfg<float, N2>;
  constexpr int M = C::M, VEC = 16 / (int)sizeof(In);  // values per 16-byte load
  extern __shared__ __align__(16) unsigned char smem_raw[];
  cx<float>* sm = reinterpret_cast<cx<float>*>(smem_raw);
  cx<float>* tw = sm + C::LPB * C::LS;
  load_tw_x<float, N2>(tw, twg);
  const long long line0 = (long long)blockIdx.x * C::LPB;
  for (int idx = threadIdx.x; idx < C::LPB * N2 / VEC; idx += 64) {
    const int l = idx / (N2 / VEC), n = (idx % (N2 / VEC)) * VEC;
    const uint4 q = *reinterpret_cast<const uint4*>(in + (line0 + l) * N2 + n);
    cx<float>* s = sm + l * C::LS;
    if constexpr (sizeof(In) == 2) {
      const unsigned w[4] = {q.x, q.y, q.z, q.w};
#pragma unroll
      for (int k = 0; k < 4; ++k)
        s[pad(n / 2 + k)] = mk<float>(__uint_as_float(w[k] << 16), __uint_as_float(w[k] & 0xffff0000u));
    } else {
      s[pad(n / 2)] = mk<float>(__uint_as_float(q.x), __uint_as_float(q.y));
      s[pad(n / 2 + 1)] = mk<float>(__uint_as_float(q.z), __uint_as_float(q.w));
    }
  }
  __syncthreads();
  x_fft<float, N2, 1, -1>(sm, tw);
  __syncthreads();
  const cx<float>* post = tw + tw_total(M);
  cx<float>* dst = A + line0 * md;
  for (int idx = threadIdx.x; idx < C::LPB * md; idx += 64) {
    const int l = idx / md, k = idx - l * md;
    const cx<float>* s = sm + l * C::LS;
    const cx<float> Zk = s[pad(k)];
    if (k == 0) {
      dst[idx] = mk<float>(Zk.x + Zk.y, 0.f);
    } else {
      const cx<float> Zm = s[pad(M - k)];
      const cx<float> ak = cscale(Zk + cconj(Zm), 0.5f), bk = cscale(Zk - cconj(Zm), 0.5f);
      dst[idx] = ak - mul_i(cmul_fma<0>(post[k], bk));
    }
  }
}

// A strided line set of the pruned transforms: column q of a field lies at
// (q / cw) zs + q % cw, its row r at r rs further; fields fs apart.
struct LineSet {
  long long fs, zs, rs;
};

// F (SIGN < 0) or G (SIGN > 0) along axis 1 or 0 on W columns a block: forward
// reads N rows and stores the 2 md kept ones, inverse reads the kept ones (the
// others are zero) and stores N. Values of column kx = q % md are multiplied by s0
// (kx = 0) or s1. Blocks (column tile, field).
template <int N, int W, int SIGN>
__global__ void __launch_bounds__(LCfg<float, N, W>::NT) k_fno_line(const cx<float>* __restrict__ in,
                                                                   cx<float>* __restrict__ out, LineSet li, LineSet lo,
                                                                   int ncol, int cw, int md, float s0, float s1,
                                                                   const cx<float>* __restrict__ twg) {
  using C = LCfg<float, N, W>;
  constexpr int E = C::E, TL = C::TL;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int col = threadIdx.x % W, t = threadIdx.x / W;
  cx<float>* b = reinterpret_cast<cx<float>*>(smem_raw) + col * C::BS;
  const int q = blockIdx.x * W + col;
  const bool ok = q < ncol;
  const int qz = q / cw, qx = q - qz * cw;
  const float s = q % md == 0 ? s0 : s1;
  const cx<float>* ip = in + blockIdx.y * li.fs + qz * li.zs + qx;
  cx<float>* op = out + blockIdx.y * lo.fs + qz * lo.zs + qx;
  // kept row of grid row r, or -1
  auto kept = [&](int r) { return r < md ? r : (r >= N - md ? r - (N - 2 * md) : -1); };
  cx<float> v[E];
#pragma unroll
  for (int m = 0; m < E; ++m) {
    const int r = t + TL * m, j = SIGN < 0 ? r : kept(r);
    v[m] = ok && j >= 0 ? ip[j * li.rs] : mk<float>(0.f, 0.f);
    if (SIGN > 0) v[m] = mk<float>(mul_rn(v[m].x, s), mul_rn(v[m].y, s));
  }
  lp_fft<float, N, W, SIGN>(v, b, twg, t);
#pragma unroll
  for (int m = 0; m < E; ++m) {
    const int r = t + TL * m, j = SIGN < 0 ? kept(r) : r;
    if (ok && j >= 0) op[j * lo.rs] = SIGN < 0 ? cscale(v[m], s) : v[m];
  }
}

// G along axis 2 from the columns of A, with the pointwise layer on the way out.
//   forward   z = G + M v + m (BF16), v' = gelu(z) (BF16), v the layer's input;
//   backward  dv = G + M^T dz (FP32), v the FP32 dz.
// Real-part semantics on the k2 = 0 column: its imaginary part is dropped. A
// block takes R rows of all W channels: the lanes of a line transform it in
// registers (acm_xline.cuh) and leave its voxel pairs in its line buffer, then each
// thread forms the W outputs of one voxel pair, the W inputs in registers and the
// matrix read as broadcasts of four entries. Bound by issue: 64 multiply-adds, 8
// broadcasts and two erf per pair and channel (132 us a layer at 64^3, W = 32, batch 4,
// for 333 us of separate inverse transform, column clean-up and pointwise kernels).
// Packed multiply-adds on a doubled matrix (161 us) and four voxels a thread in
// blocks of half the size (232 us) lost: both leave too few loads in flight.
constexpr int FX_NT = 128;
template <int N2>
__host__ __device__ constexpr int fx_rows() { return FX_NT / (N2 / 2) < 1 ? 1 : FX_NT / (N2 / 2); }
template <int N2, int W>
__host__ __device__ constexpr int fx_smem() {
  return ((XL<float, N2>::TW + 1) / 2 * 2 + fx_rows<N2>() * W * XL<float, N2>::template lb<1>()) * (int)sizeof(cx<float>) +
         (W * W + W) * (int)sizeof(float);
}

template <int N2, int W, bool FWD>
__global__ void __launch_bounds__(FX_NT) k_fno_x_inv(const cx<float>* __restrict__ A, const void* __restrict__ vin,
                                                    const __nv_bfloat16* __restrict__ Mw,
                                                    const __nv_bfloat16* __restrict__ mb, void* __restrict__ out,
                                                    __nv_bfloat16* __restrict__ vout, int md, long long rows,
                                                    const cx<float>* __restrict__ twg) {
  using L = XL<float, N2>;
  constexpr int M = L::M, E = L::E, TL = L::TL, R = fx_rows<N2>(), LB = L::template lb<1>();
  constexpr int TWS = (L::TW + 1) / 2 * 2;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  cx<float>* tw = reinterpret_cast<cx<float>*>(smem_raw);
  float* sM = reinterpret_cast<float*>(tw + TWS);
  float* sm = sM + W * W;
  cx<float>* lines = reinterpret_cast<cx<float>*>(sm + W);
  const long long row0 = (long long)blockIdx.x * R, V = rows * N2;
  const long long f0 = (long long)blockIdx.y * W;  // first field of the sample
  xl_load_tw<float, N2, TW_MAX>(tw, twg);
  for (int i = threadIdx.x; i < W * W; i += FX_NT) {
    const int r = i / W, c = i - r * W;
    sM[FWD ? i : c * W + r] = bf(Mw[i]);
  }
  if (FWD)
    for (int i = threadIdx.x; i < W; i += FX_NT) sm[i] = bf(mb[i]);
  for (int idx = threadIdx.x; idx < R * W * (M + 1); idx += FX_NT) {
    const int l = idx / (M + 1), k = idx - l * (M + 1), r = l / W, ch = l - r * W;
    cx<float> x = mk<float>(0.f, 0.f);
    if (k < md) x = A[((f0 + ch) * rows + row0 + r) * md + k];
    if (k == 0) x.y = 0.f;
    lines[l * LB + pad(k)] = x;
  }
  __syncthreads();
  for (int task = threadIdx.x; task < R * W * TL; task += FX_NT) {  // whole warps: R W TL is a multiple of 32
    const int l = task / TL, t = task % TL;
    cx<float>* sl = lines + l * LB;
    cx<float> y[E];
    xl_inverse<float, N2>(sl, tw, t, xl_mask(), y);
#pragma unroll
    for (int m = 0; m < E; ++m) sl[t + TL * m] = y[m];
  }
  __syncthreads();
  for (int pi = threadIdx.x; pi < R * M; pi += FX_NT) {
    const int r = pi / M, k = pi - r * M;
    const long long x = (row0 + r) * N2 + 2 * k;
    const cx<float>* yl = lines + r * W * LB + k;
    float2 vv[W];
#pragma unroll
    for (int j = 0; j < W; ++j) {
      if constexpr (FWD) {
        const unsigned q = *reinterpret_cast<const unsigned*>((const __nv_bfloat16*)vin + (f0 + j) * V + x);
        vv[j] = make_float2(__uint_as_float(q << 16), __uint_as_float(q & 0xffff0000u));
      } else {
        vv[j] = *reinterpret_cast<const float2*>((const float*)vin + (f0 + j) * V + x);
      }
    }
#pragma unroll 2
    for (int i = 0; i < W; ++i) {
      const cx<float> y = yl[i * LB];
      float2 acc = FWD ? make_float2(y.x + sm[i], y.y + sm[i]) : make_float2(0.f, 0.f);
#pragma unroll
      for (int j = 0; j < W; j += 4) {
        const float4 m4 = *reinterpret_cast<const float4*>(&sM[i * W + j]);
        const float mm[4] = {m4.x, m4.y, m4.z, m4.w};
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          acc.x += mm[e] * vv[j + e].x;
          acc.y += mm[e] * vv[j + e].y;
        }
      }
      const long long o = (f0 + i) * V + x;
      if constexpr (FWD) {
        __nv_bfloat162 z2, g2;
        z2.x = __float2bfloat16(acc.x);
        z2.y = __float2bfloat16(acc.y);
        g2.x = __float2bfloat16(gelu_f(acc.x));
        g2.y = __float2bfloat16(gelu_f(acc.y));
        *reinterpret_cast<__nv_bfloat162*>((__nv_bfloat16*)out + o) = z2;
        *reinterpret_cast<__nv_bfloat162*>(vout + o) = g2;
      } else {
        *reinterpret_cast<float2*>((float*)out + o) = make_float2(acc.x + y.x, acc.y + y.y);
      }
    }
  }
}

// ---------------------------------------------------------------------------
// per-mode channel mix, MPB consecutive modes a block so that the [field][mode]
// spectra move in whole sectors
// ---------------------------------------------------------------------------
constexpr int MIX_NT = 256;

// Eight lanes hold eight modes of one field, four fields a warp: rows of a matrix
// lie W + 1 words apart and matrices 4 words (mod 32), spectra of a mode an odd
// number of elements, so the lanes fall on distinct banks (with equal strides mod 32
// the forward mix took 82 us at 6912 modes, W = 32, batch 4).
template <int W>
__host__ __device__ constexpr int mix_rs() {  // words per matrix
  int q = W * (W + 1);
  while (q % 32 != 4) ++q;
  return q;
}
__host__ __device__ constexpr int mix_fs(int F) { return F + 1 - F % 2; }  // elements per mode of a spectrum

template <int W>
__device__ __forceinline__ void mix_load_r(const __nv_bfloat16* __restrict__ R, unsigned* sR, int m0, int nm) {
  const unsigned* src = reinterpret_cast<const unsigned*>(R) + (long long)m0 * W * W;
  for (int e = threadIdx.x; e < nm * W * W; e += MIX_NT)
    sR[e / (W * W) * mix_rs<W>() + e / W % W * (W + 1) + e % W] = src[e];
}
__device__ __forceinline__ cx<float> mix_r(unsigned q) {
  return mk<float>(__uint_as_float(q << 16), __uint_as_float(q & 0xffff0000u));
}

// Y[b][i] = sum_j R[i][j] X[b][j]
template <int W>
__global__ void __launch_bounds__(MIX_NT) k_mix_fwd(const cx<float>* __restrict__ X, const __nv_bfloat16* __restrict__ R,
                                                   cx<float>* __restrict__ Y, int M, int B, int mpb) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int m0 = blockIdx.x * mpb, nm = min(mpb, M - m0), F = B * W, FS = mix_fs(F);
  cx<float>* sX = reinterpret_cast<cx<float>*>(smem_raw);        // [mpb][FS]
  unsigned* sR = reinterpret_cast<unsigned*>(sX + mpb * FS);  // [mpb][mix_rs]
  mix_load_r<W>(R, sR, m0, nm);
  for (int e = threadIdx.x; e < F * mpb; e += MIX_NT) {
    const int f = e / mpb, m = e - f * mpb;
    if (m < nm) sX[m * FS + f] = X[(long long)f * M + m0 + m];
  }
  __syncthreads();
  // one (field, mode) an output, modes fastest for the stores
  for (int e = threadIdx.x; e < F * mpb; e += MIX_NT) {
    const int m = e % mpb, f = e / mpb, b = f / W, i = f - b * W;
    if (m >= nm) continue;
    const unsigned* r = sR + m * mix_rs<W>() + i * (W + 1);
    const cx<float>* x = sX + m * FS + b * W;
    cx<float> acc = mk<float>(0.f, 0.f);
#pragma unroll 8
    for (int j = 0; j < W; ++j) acc = acc + cmul_fma<1>(mix_r(r[j]), x[j]);
    Y[(long long)f * M + m0 + m] = acc;
  }
}

// gR[i][j] = sum_b gY[b][i] conj(X[b][j]);  gX[b][j] = sum_i conj(R[i][j]) gY[b][i]
template <int W>
__global__ void __launch_bounds__(MIX_NT) k_mix_bwd(const cx<float>* __restrict__ X, const cx<float>* __restrict__ gY,
                                                   const __nv_bfloat16* __restrict__ R, float* __restrict__ gR,
                                                   cx<float>* __restrict__ gX, int M, int B, int mpb) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int m0 = blockIdx.x * mpb, nm = min(mpb, M - m0), F = B * W, FS = mix_fs(F);
  cx<float>* sX = reinterpret_cast<cx<float>*>(smem_raw);
  cx<float>* sG = sX + mpb * FS;
  unsigned* sR = reinterpret_cast<unsigned*>(sG + mpb * FS);
  mix_load_r<W>(R, sR, m0, nm);
  for (int e = threadIdx.x; e < F * mpb; e += MIX_NT) {
    const int f = e / mpb, m = e - f * mpb;
    if (m < nm) {
      sX[m * FS + f] = X[(long long)f * M + m0 + m];
      sG[m * FS + f] = gY[(long long)f * M + m0 + m];
    }
  }
  __syncthreads();
  float2* gRm = reinterpret_cast<float2*>(gR) + (long long)m0 * W * W;
  for (int e = threadIdx.x; e < nm * W * W; e += MIX_NT) {
    const int m = e / (W * W), i = e / W % W, j = e % W;
    cx<float> acc = mk<float>(0.f, 0.f);
    for (int b = 0; b < B; ++b) acc = acc + cmul(sG[m * FS + b * W + i], cconj(sX[m * FS + b * W + j]));
    gRm[e] = make_float2(acc.x, acc.y);
  }
  for (int e = threadIdx.x; e < F * mpb; e += MIX_NT) {
    const int m = e % mpb, f = e / mpb, b = f / W, j = f - b * W;
    if (m >= nm) continue;
    cx<float> acc = mk<float>(0.f, 0.f);
#pragma unroll 8
    for (int i = 0; i < W; ++i) acc = acc + cmul(cconj(mix_r(sR[m * mix_rs<W>() + i * (W + 1) + j])), sG[m * FS + b * W + i]);
    gX[(long long)f * M + m0 + m] = acc;
  }
}

// projection, loss and its gradient: out = Q v + q; d = (out - t) * mask;
// dout = 2 d / (B V); partial sums of d^2 per block
template <int W>
__global__ void __launch_bounds__(256) k_project(const __nv_bfloat16* __restrict__ v, const __nv_bfloat16* __restrict__ Q,
                                                const __nv_bfloat16* __restrict__ q, const float* __restrict__ target,
                                                const uint8_t* __restrict__ H, float* __restrict__ out,
                                                float* __restrict__ dout, double* __restrict__ lpart, FnoDims d, int B) {
  __shared__ float sQ[6 * W], sq[6];
  __shared__ double red[32];
  for (int i = threadIdx.x; i < 6 * W; i += blockDim.x) sQ[i] = bf(Q[i]);
  for (int i = threadIdx.x; i < 6; i += blockDim.x) sq[i] = bf(q[i]);
  __syncthreads();
  const long long total = (long long)B * d.V;
  const float sc = 2.0f / (float)total;
  float acc = 0.f;
  for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < total; t += (long long)gridDim.x * blockDim.x) {
    const long long b = t / d.V, x = t - b * d.V;
    float r6[6];
#pragma unroll
    for (int o = 0; o < 6; ++o) r6[o] = sq[o];
#pragma unroll 4
    for (int j = 0; j < W; ++j) {
      const float vj = bf(v[b * W * d.V + j * d.V + x]);
#pragma unroll
      for (int o = 0; o < 6; ++o) r6[o] += sQ[o * W + j] * vj;
    }
    const bool solid = H[t] != 0;
#pragma unroll
    for (int o = 0; o < 6; ++o) {
      const float r = r6[o];
      const long long oi = (b * 6 + o) * d.V + x;
      if (out) out[oi] = r;
      if (target) {
        const float dd = (o < 3 || solid) ? r - target[oi] : 0.f;
        acc += dd * dd;
        dout[oi] = sc * dd;
      }
    }
  }
  if (!target) return;
  double a = acc;
  for (int o = 16; o > 0; o >>= 1) a += __shfl_xor_sync(0xffffffffu, a, o);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = a;
  __syncthreads();
  if (threadIdx.x == 0) {
    double s = 0;
    for (int w = 0; w < (int)(blockDim.x >> 5); ++w) s += red[w];
    lpart[blockIdx.x] = s;
  }
}

// dv = Q^T dout
template <int W>
__global__ void __launch_bounds__(256) k_project_bwd(const float* __restrict__ dout, const __nv_bfloat16* __restrict__ Q,
                                                    float* __restrict__ dv, FnoDims d, int B) {
  __shared__ float sQ[6 * W];
  for (int i = threadIdx.x; i < 6 * W; i += blockDim.x) sQ[i] = bf(Q[i]);
  __syncthreads();
  const long long total = (long long)B * d.V;
  for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < total; t += (long long)gridDim.x * blockDim.x) {
    const long long b = t / d.V, x = t - b * d.V;
    float g[6];
#pragma unroll
    for (int o = 0; o < 6; ++o) g[o] = dout[(b * 6 + o) * d.V + x];
#pragma unroll 4
    for (int j = 0; j < W; ++j) {
      float acc = 0.f;
#pragma unroll
      for (int o = 0; o < 6; ++o) acc += sQ[o * W + j] * g[o];
      dv[b * W * d.V + j * d.V + x] = acc;
    }
  }
}

// Weight gradients G[i][j] = sum_x A_i(x) B_j(x) and g[i] = sum_x A_i(x) over all
// voxels of the batch, as block partials [blocks][AD * BD + AD].
// A: FP32 [b][AD][V]; with ACT it is dv, and A = dv gelu'(z) is formed here and stored
// in dz. B: BF16 [b][BD][V], or the features (H, x0, x1, x2) when LIFT.
//
// A thread loads one voxel's A and B rows into shared memory; a warp then goes
// through its own 32 voxels with one column of the wider operand per lane and the
// narrower one as broadcasts of four, all sums in registers. Sums of 32 voxels are
// added to the running sums, so a partial is never a chain longer than 32 + its
// tiles. Bound by issue (W = 32: 16 packed multiply-adds to 9 shared loads a voxel); the
// former kernel, two scalar shared loads to a multiply-add, took 1246 us a layer at
// 64^3, W = 32, batch 4 (and 121 for the activation), this one about 205.
template <int D>
__host__ __device__ constexpr int wg_stride() {  // floats per row: whole float4s, an odd number of them
  int q = (D + 3) / 4;
  return 4 * (q % 2 ? q : q + 1);
}
template <int AD, int BD>
__host__ __device__ constexpr int wg_smem() {
  const int rows = 256 * (wg_stride<AD>() + wg_stride<BD>()) * 4, sums = 8 * (AD * BD + AD) * 4;
  return rows > sums ? rows : sums;
}

template <int AD, int BD, bool LIFT, bool ACT>
__global__ void __launch_bounds__(256, 2) k_wgrad(const float* __restrict__ A, const __nv_bfloat16* __restrict__ Bv,
                                              const uint8_t* __restrict__ H, const __nv_bfloat16* __restrict__ z,
                                              float* __restrict__ dz, float* __restrict__ part, FnoDims d, int B) {
  constexpr int NE = AD * BD + AD;
  constexpr int SA = wg_stride<AD>(), SB = wg_stride<BD>();
  constexpr bool WIDEB = !LIFT;                   // the operand spread over the lanes: B, or A of the lift
  constexpr int WD = WIDEB ? BD : AD, ND = WIDEB ? AD : BD;
  static_assert(WD <= 32 && 32 % WD == 0, "one lane per wide column");
  constexpr int VS = 32 / WD;                     // voxels a warp takes at once
  constexpr int NP = (ND + 1) / 2;                // narrow columns in pairs (ND is even)
  extern __shared__ __align__(16) float wsm[];
  float* ra = wsm + threadIdx.x * SA;
  float* rb = wsm + 256 * SA + threadIdx.x * SB;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, w = lane % WD, vs = lane / WD;
  const float* wa = wsm + warp * 32 * SA;
  const float* wb = wsm + 256 * SA + warp * 32 * SB;
  constexpr int NBI = (AD + WD - 1) / WD;         // bias sums of A_w, A_{w + WD}, ...
  float acc[ND], ab[NBI];
#pragma unroll
  for (int n = 0; n < NBI; ++n) ab[n] = 0.f;
#pragma unroll
  for (int n = 0; n < ND; ++n) acc[n] = 0.f;
  const long long total = (long long)B * d.V;
  const long long tiles = (total + 255) / 256, per = (tiles + gridDim.x - 1) / gridDim.x;
  const long long lo = blockIdx.x * per, hi = min(tiles, lo + per);
  for (long long tile = lo; tile < hi; ++tile) {
    const long long t = tile * 256 + threadIdx.x;
    const bool in = t < total;
    const long long b = in ? t / d.V : 0, x = in ? t - b * d.V : 0;
    constexpr int CH = AD < 8 ? 4 : 8;  // rows whose loads are in flight together
#pragma unroll
    for (int c0 = 0; c0 < AD; c0 += CH) {
      float q[CH], zz[CH];
#pragma unroll
      for (int e = 0; e < CH; ++e) {
        const bool use = in && c0 + e < AD;
        const long long o = (b * AD + c0 + e) * d.V + x;
        q[e] = use ? A[o] : 0.f;
        if constexpr (ACT) zz[e] = use ? bf(z[o]) : 0.f;
      }
#pragma unroll
      for (int e = 0; e < CH; ++e) {
        if constexpr (ACT) {
          q[e] *= gelu_grad_f(zz[e]);
          if (in) dz[(b * AD + c0 + e) * d.V + x] = q[e];
        }
      }
#pragma unroll
      for (int e = 0; e < CH; e += 4)
        *reinterpret_cast<float4*>(ra + c0 + e) = make_float4(q[e], q[e + 1], q[e + 2], q[e + 3]);
    }
    if constexpr (LIFT) {
      const int i2 = (int)(x % d.n2), i1 = (int)((x / d.n2) % d.n1), i0 = (int)(x / ((long long)d.n2 * d.n1));
      *reinterpret_cast<float4*>(rb) = in ? make_float4((float)H[t], (i0 + 0.5f) / d.n0, (i1 + 0.5f) / d.n1,
                                                        (i2 + 0.5f) / d.n2)
                                          : make_float4(0.f, 0.f, 0.f, 0.f);
    } else {
#pragma unroll
      for (int c0 = 0; c0 < BD; c0 += BD < 16 ? 4 : 16) {
        constexpr int CB = BD < 16 ? 4 : 16;
        float q[CB];
#pragma unroll
        for (int e = 0; e < CB; ++e) q[e] = in ? bf(Bv[(b * BD + c0 + e) * d.V + x]) : 0.f;
#pragma unroll
        for (int e = 0; e < CB; e += 4)
          *reinterpret_cast<float4*>(rb + c0 + e) = make_float4(q[e], q[e + 1], q[e + 2], q[e + 3]);
      }
    }
    __syncwarp();
    float sb[NBI];
#pragma unroll
    for (int n = 0; n < NBI; ++n) sb[n] = 0.f;
    // 16 narrow columns at a time: fewer tile sums live beside the running sums
    constexpr int HP = NP < 8 ? NP : 8;
    static_assert(NP % HP == 0, "whole parts");
#pragma unroll
    for (int h = 0; h < NP; h += HP) {
      float2 s[HP];
#pragma unroll
      for (int n = 0; n < HP; ++n) s[n] = make_float2(0.f, 0.f);
#pragma unroll 4
      for (int v = vs; v < 32; v += VS) {
        const float wide = WIDEB ? wb[v * SB + w] : wa[v * SA + w];
        const float* nar = (WIDEB ? wa + v * SA : wb + v * SB) + 2 * h;
        const float2 w2 = make_float2(wide, wide);
#pragma unroll
        for (int n = 0; n < HP; n += 2) {
          const float4 q = *reinterpret_cast<const float4*>(nar + 2 * n);
          s[n] = fma2(make_float2(q.x, q.y), w2, s[n]);
          if (n + 1 < HP) s[n + 1] = fma2(make_float2(q.z, q.w), w2, s[n + 1]);
        }
        if (h == 0) {
#pragma unroll
          for (int n = 0; n < NBI; ++n) sb[n] += WIDEB ? (w + WD * n < AD ? wa[v * SA + w + WD * n] : 0.f) : wide;
        }
      }
#pragma unroll
      for (int n = 0; n < 2 * HP; ++n) acc[2 * h + n] += n & 1 ? s[n / 2].y : s[n / 2].x;
    }
#pragma unroll
    for (int n = 0; n < NBI; ++n) ab[n] += sb[n];
    __syncwarp();
  }
  // lanes that share a column, then the warps of the block
#pragma unroll
  for (int o = WD; o < 32; o <<= 1) {
#pragma unroll
    for (int n = 0; n < ND; ++n) acc[n] += __shfl_xor_sync(0xffffffffu, acc[n], o);
#pragma unroll
    for (int n = 0; n < NBI; ++n) ab[n] += __shfl_xor_sync(0xffffffffu, ab[n], o);
  }
  __syncthreads();
  float* my = wsm + warp * NE;
  if (vs == 0) {
#pragma unroll
    for (int n = 0; n < ND; ++n) my[WIDEB ? n * BD + w : w * BD + n] = acc[n];
#pragma unroll
    for (int n = 0; n < NBI; ++n)
      if (w + WD * n < AD) my[AD * BD + w + WD * n] = ab[n];
  }
  __syncthreads();
  for (int e = threadIdx.x; e < NE; e += 256) {
    float sum = 0.f;
#pragma unroll
    for (int k = 0; k < 8; ++k) sum += wsm[k * NE + e];
    part[(long long)blockIdx.x * NE + e] = sum;
  }
}

// sum the nrec partials in FP64, a warp per element: out_w[e] for e < AD*BD, out_b[e]
// for the biases (one thread per element walked the 512 records in 77 us)
__global__ void __launch_bounds__(256) k_reduce_parts(const float* __restrict__ part, int nrec, int ne, int nab,
                                                     float* __restrict__ out_w, float* __restrict__ out_b) {
  const int e = blockIdx.x * 8 + (threadIdx.x >> 5), lane = threadIdx.x & 31;
  if (e >= ne) return;
  double s = 0;
  for (int r = lane; r < nrec; r += 32) s += part[(long long)r * ne + e];
  s = warp_sum(s);
  if (lane != 0) return;
  if (e < nab) out_w[e] = (float)s;
  else out_b[e - nab] = (float)s;
}

__global__ void k_adamw(float* __restrict__ th, __nv_bfloat16* __restrict__ tb, const float* __restrict__ g,
                        float* __restrict__ m1, float* __restrict__ m2, long long n, float lr, float b1, float b2,
                        float eps, float wd, float c1, float c2) {
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
    const float gi = g[i];
    const float a = b1 * m1[i] + (1.f - b1) * gi;
    const float v = b2 * m2[i] + (1.f - b2) * gi * gi;
    m1[i] = a;
    m2[i] = v;
    const float t = th[i] - lr * ((a / c1) / (sqrtf(v / c2) + eps) + wd * th[i]);
    th[i] = t;
    tb[i] = __float2bfloat16(t);
  }
}

__global__ void k_f32_to_bf16(const float* __restrict__ in, __nv_bfloat16* __restrict__ out, long long n) {
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x)
    out[i] = __float2bfloat16(in[i]);
}

}  // namespace

// ---------------------------------------------------------------------------
// host side
// ---------------------------------------------------------------------------
struct acm_fno {
  FnoDims d;
  Geo g;
  int Bmax;
  cudaStream_t st;
  long long np;
  // parameter offsets (elements) in the flat vector
  long long oP, op, oQ, oq;
  std::vector<long long> oR, oM, om;
  float* theta = nullptr;          // FP32 master
  __nv_bfloat16* tb = nullptr;     // BF16 copy used by the kernels
  float* grad = nullptr;
  float* m1 = nullptr;
  float* m2 = nullptr;
  long long step = 0;
  // activations
  __nv_bfloat16* v = nullptr;      // [L+1][Bmax][W][V]
  __nv_bfloat16* z = nullptr;      // [L][Bmax][W][V]
  cx<float>* X = nullptr;          // [L][Bmax][W][M]
  cx<float>* Y = nullptr;          // [Bmax][W][M]
  cx<float>* gX = nullptr;         // [Bmax][W][M]
  float* r0 = nullptr;             // [Bmax][W][V] FP32 scratch
  float* r1 = nullptr;             // [Bmax][W][V] FP32 scratch
  float* dout = nullptr;           // [Bmax][6][V]
  float* tgt = nullptr;            // [Bmax][6][V] staging of host targets
  uint8_t* Hs = nullptr;           // [Bmax][V] staging of indicators
  uint8_t* Hp = nullptr;           // [Bmax][V] axis-swapped indicators (warm start, allocated on first use)
  cx<float>* spec = nullptr;       // compact spectra A, then B (see the head of the file)
  float* part = nullptr;           // [NRB][W*W + W]
  double* lpart = nullptr;         // [NRB]
  void* tw = nullptr;              // FP32 twiddles
};

namespace {

#define FK(x)                              \
  do {                                     \
    if ((x) != cudaSuccess) {              \
      cudaGetLastError();                  \
      return ACM_ERR_CUDA;                 \
    }                                      \
  } while (0)

#define CKF(x)                   \
  do {                           \
    acm_status s_ = (x);         \
    if (s_ != ACM_OK) return s_; \
  } while (0)

int blocks_for(long long n) { return (int)std::min<long long>(4 * 152, (n + 255) / 256); }

// columns a block of the pruned strided transforms takes
template <int N>
constexpr int fno_w() {
  constexpr int TL = N / ept(N);
  return N == 512 ? 8 : (TL >= 2 ? 16 : 32);
}

template <int N, int SIGN>
acm_status fno_line_n(acm_fno* f, const cx<float>* in, cx<float>* out, LineSet li, LineSet lo, int ncol, int cw, int C,
                      float s0, float s1) {
  constexpr int W = fno_w<N>();
  using L = LCfg<float, N, W>;
  constexpr int smem = W * L::BS * (int)sizeof(cx<float>);
  static_assert(smem <= 48 * 1024, "static limit");
  k_fno_line<N, W, SIGN><<<dim3((ncol + W - 1) / W, C), L::NT, smem, f->st>>>(in, out, li, lo, ncol, cw, f->d.md, s0, s1,
                                                                              (const cx<float>*)f->tw);
  FK(cudaGetLastError());
  return ACM_OK;
}

template <int SIGN>
acm_status fno_line(acm_fno* f, int n, const cx<float>* in, cx<float>* out, LineSet li, LineSet lo, int ncol, int cw,
                    int C, float s0, float s1) {
  switch (n) {
    case 8: return fno_line_n<8, SIGN>(f, in, out, li, lo, ncol, cw, C, s0, s1);
    case 16: return fno_line_n<16, SIGN>(f, in, out, li, lo, ncol, cw, C, s0, s1);
    case 32: return fno_line_n<32, SIGN>(f, in, out, li, lo, ncol, cw, C, s0, s1);
    case 64: return fno_line_n<64, SIGN>(f, in, out, li, lo, ncol, cw, C, s0, s1);
    case 128: return fno_line_n<128, SIGN>(f, in, out, li, lo, ncol, cw, C, s0, s1);
    case 256: return fno_line_n<256, SIGN>(f, in, out, li, lo, ncol, cw, C, s0, s1);
    case 512: return fno_line_n<512, SIGN>(f, in, out, li, lo, ncol, cw, C, s0, s1);
    default: return ACM_ERR_UNSUPPORTED_SIZE;
  }
}

// the line sets of the three compact spectra (columns (i0, k2) along axis 1, (k1, k2) along axis 0)
cx<float>* buf_b(acm_fno* f) {  // B lies behind A
  const FnoDims& d = f->d;
  return f->spec + (long long)f->Bmax * d.W * d.n0 * d.n1 * d.md;
}

template <int N2, typename In>
acm_status fno_x_fwd_n(acm_fno* f, const In* in, int C) {
  constexpr int smem = x_smem_bytes<float, N2, 1>();
  static const cudaError_t attr =
      smem > 48 * 1024 ? cudaFuncSetAttribute(k_fno_x_fwd<N2, In>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem)
                       : cudaSuccess;
  FK(attr);
  const long long lines = (long long)C * f->d.n0 * f->d.n1;
  k_fno_x_fwd<N2, In><<<(unsigned)(lines / XCfg<float, N2>::LPB), 64, smem, f->st>>>(in, f->spec, f->d.md,
                                                                                     (const cx<float>*)f->tw);
  FK(cudaGetLastError());
  return ACM_OK;
}

// F: C real fields -> their kept modes X, times s0 (k2 = 0) or s1
template <typename In>
acm_status fno_fwd_dft(acm_fno* f, const In* in, cx<float>* X, int C, float s0, float s1) {
  const FnoDims& d = f->d;
  switch (d.n2) {
    case 8: CKF((fno_x_fwd_n<8, In>(f, in, C))); break;
    case 16: CKF((fno_x_fwd_n<16, In>(f, in, C))); break;
    case 32: CKF((fno_x_fwd_n<32, In>(f, in, C))); break;
    case 64: CKF((fno_x_fwd_n<64, In>(f, in, C))); break;
    case 128: CKF((fno_x_fwd_n<128, In>(f, in, C))); break;
    case 256: CKF((fno_x_fwd_n<256, In>(f, in, C))); break;
    case 512: CKF((fno_x_fwd_n<512, In>(f, in, C))); break;
    default: return ACM_ERR_UNSUPPORTED_SIZE;
  }
  const long long q = 2LL * d.md * d.md;
  const LineSet ya = {(long long)d.n0 * d.n1 * d.md, (long long)d.n1 * d.md, d.md}, yb = {d.n0 * q, q, d.md};
  CKF(fno_line<-1>(f, d.n1, f->spec, buf_b(f), ya, yb, d.n0 * d.md, d.md, C, 1.f, 1.f));
  const LineSet zb = {d.n0 * q, 0, q}, zx = {d.M, 0, q};
  return fno_line<-1>(f, d.n0, buf_b(f), X, zb, zx, (int)q, (int)q, C, s0, s1);
}

// G along axes 0 and 1: kept modes Y times s0 (k2 = 0) or s1 -> A
acm_status fno_inv_dft(acm_fno* f, const cx<float>* Y, int C, float s0, float s1) {
  const FnoDims& d = f->d;
  const long long q = 2LL * d.md * d.md;
  const LineSet zb = {d.n0 * q, 0, q}, zx = {d.M, 0, q};
  CKF(fno_line<+1>(f, d.n0, Y, buf_b(f), zx, zb, (int)q, (int)q, C, s0, s1));
  const LineSet ya = {(long long)d.n0 * d.n1 * d.md, (long long)d.n1 * d.md, d.md}, yb = {d.n0 * q, q, d.md};
  return fno_line<+1>(f, d.n1, buf_b(f), f->spec, yb, ya, d.n0 * d.md, d.md, C, 1.f, 1.f);
}

template <int N2, int W, bool FWD>
acm_status fno_x_inv_n(acm_fno* f, int B, const void* vin, const __nv_bfloat16* Mw, const __nv_bfloat16* mb, void* out,
                       __nv_bfloat16* vout) {
  constexpr int smem = fx_smem<N2, W>();
  static_assert(smem <= 227 * 1024, "shared memory of a block");
  static const cudaError_t attr =
      smem > 48 * 1024
          ? cudaFuncSetAttribute(k_fno_x_inv<N2, W, FWD>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem)
          : cudaSuccess;
  FK(attr);
  const long long rows = (long long)f->d.n0 * f->d.n1;
  k_fno_x_inv<N2, W, FWD><<<dim3((unsigned)(rows / fx_rows<N2>()), B), FX_NT, smem, f->st>>>(
      f->spec, vin, Mw, mb, out, vout, f->d.md, rows, (const cx<float>*)f->tw);
  FK(cudaGetLastError());
  return ACM_OK;
}

template <int W, bool FWD>
acm_status fno_x_inv(acm_fno* f, int B, const void* vin, const __nv_bfloat16* Mw, const __nv_bfloat16* mb, void* out,
                     __nv_bfloat16* vout) {
  switch (f->d.n2) {
    case 8: return fno_x_inv_n<8, W, FWD>(f, B, vin, Mw, mb, out, vout);
    case 16: return fno_x_inv_n<16, W, FWD>(f, B, vin, Mw, mb, out, vout);
    case 32: return fno_x_inv_n<32, W, FWD>(f, B, vin, Mw, mb, out, vout);
    case 64: return fno_x_inv_n<64, W, FWD>(f, B, vin, Mw, mb, out, vout);
    case 128: return fno_x_inv_n<128, W, FWD>(f, B, vin, Mw, mb, out, vout);
    case 256: return fno_x_inv_n<256, W, FWD>(f, B, vin, Mw, mb, out, vout);
    case 512: return fno_x_inv_n<512, W, FWD>(f, B, vin, Mw, mb, out, vout);
    default: return ACM_ERR_UNSUPPORTED_SIZE;
  }
}

// modes per block of the mix (a power of two up to 8): spectra and matrices within 96 KB
template <int W>
int mix_mpb(int B, int spectra, int* smem) {
  int m = 8;
  auto bytes = [&](int k) { return k * (spectra * mix_fs(B * W) * (int)sizeof(cx<float>) + mix_rs<W>() * (int)sizeof(unsigned)); };
  while (m > 1 && bytes(m) > 96 * 1024) m /= 2;
  *smem = bytes(m);
  return m;
}

template <int W>
acm_status mix_fwd(acm_fno* f, int B, const cx<float>* X, const __nv_bfloat16* R, cx<float>* Y) {
  static const cudaError_t attr =
      cudaFuncSetAttribute(k_mix_fwd<W>, cudaFuncAttributeMaxDynamicSharedMemorySize, 96 * 1024);
  FK(attr);
  int smem;
  const int mpb = mix_mpb<W>(B, 1, &smem);
  k_mix_fwd<W><<<(f->d.M + mpb - 1) / mpb, MIX_NT, smem, f->st>>>(X, R, Y, f->d.M, B, mpb);
  FK(cudaGetLastError());
  return ACM_OK;
}

template <int W>
acm_status mix_bwd(acm_fno* f, int B, const cx<float>* X, const cx<float>* gY, const __nv_bfloat16* R, float* gR,
                   cx<float>* gX) {
  static const cudaError_t attr =
      cudaFuncSetAttribute(k_mix_bwd<W>, cudaFuncAttributeMaxDynamicSharedMemorySize, 96 * 1024);
  FK(attr);
  int smem;
  const int mpb = mix_mpb<W>(B, 2, &smem);
  k_mix_bwd<W><<<(f->d.M + mpb - 1) / mpb, MIX_NT, smem, f->st>>>(X, gY, R, gR, gX, f->d.M, B, mpb);
  FK(cudaGetLastError());
  return ACM_OK;
}

template <int W>
acm_status fno_forward_impl(acm_fno* f, int B, const uint8_t* Hd, const float* target, float* out, double* loss) {
  const FnoDims& d = f->d;
  const long long BV = (long long)B * d.V;
  const long long act = (long long)f->Bmax * W * d.V;
  const int C = B * W;
  const float invV = (float)(1.0 / (double)d.V);
  k_lift<W><<<blocks_for(BV), 256, 0, f->st>>>(Hd, f->tb + f->oP, f->tb + f->op, f->v, d, B);
  FK(cudaGetLastError());
  for (int l = 0; l < d.L; ++l) {
    __nv_bfloat16* vl = f->v + l * act;
    cx<float>* Xl = f->X + (long long)l * f->Bmax * W * d.M;
    CKF(fno_fwd_dft(f, vl, Xl, C, 1.f, 1.f));
    CKF(mix_fwd<W>(f, B, Xl, f->tb + f->oR[l], f->Y));
    CKF(fno_inv_dft(f, f->Y, C, invV, invV));
    CKF((fno_x_inv<W, true>(f, B, vl, f->tb + f->oM[l], f->tb + f->om[l], f->z + l * act, f->v + (l + 1) * act)));
  }
  k_project<W><<<NRB, 256, 0, f->st>>>(f->v + d.L * act, f->tb + f->oQ, f->tb + f->oq, target, Hd, out, f->dout,
                                       f->lpart, d, B);
  FK(cudaGetLastError());
  if (loss) {
    std::vector<double> lp(NRB);
    FK(cudaMemcpyAsync(lp.data(), f->lpart, NRB * sizeof(double), cudaMemcpyDeviceToHost, f->st));
    FK(cudaStreamSynchronize(f->st));
    double s = 0;
    for (double x : lp) s += x;
    *loss = s / (double)BV;
  }
  return ACM_OK;
}

template <int AD, int BD, bool LIFT, bool ACT>
acm_status wgrad(acm_fno* f, int B, const float* A, const __nv_bfloat16* Bv, const uint8_t* H, const __nv_bfloat16* z,
                 float* dz, float* gw, float* gb) {
  constexpr int smem = wg_smem<AD, BD>();
  static const cudaError_t attr =
      cudaFuncSetAttribute(k_wgrad<AD, BD, LIFT, ACT>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
  FK(attr);
  // one wave: as many blocks as the SMs hold (two of the W = 32 kernel, by registers; held
  // to three it spills: 300 us a layer for 205)
  constexpr int per_sm = AD * BD >= 1024 ? 2 : 3;
  constexpr int blocks = std::min(NRB, 152 * per_sm);
  k_wgrad<AD, BD, LIFT, ACT><<<blocks, 256, smem, f->st>>>(A, Bv, H, z, dz, f->part, f->d, B);
  FK(cudaGetLastError());
  const int ne = AD * BD + AD;
  k_reduce_parts<<<(ne + 7) / 8, 256, 0, f->st>>>(f->part, blocks, ne, AD * BD, gw, gb);
  FK(cudaGetLastError());
  return ACM_OK;
}

template <int W>
acm_status fno_backward_impl(acm_fno* f, int B, const uint8_t* Hd) {
  const FnoDims& d = f->d;
  const long long BV = (long long)B * d.V;
  const long long act = (long long)f->Bmax * W * d.V;
  const int C = B * W;
  const float invV = 1.0f / (float)d.V;
  // projection
  CKF((wgrad<6, W, false, false>(f, B, f->dout, f->v + d.L * act, nullptr, nullptr, nullptr, f->grad + f->oQ,
                                 f->grad + f->oq)));
  k_project_bwd<W><<<blocks_for(BV), 256, 0, f->st>>>(f->dout, f->tb + f->oQ, f->r0, d, B);  // r0 = dv
  FK(cudaGetLastError());
  for (int l = d.L - 1; l >= 0; --l) {
    __nv_bfloat16* vl = f->v + l * act;
    cx<float>* Xl = f->X + (long long)l * f->Bmax * W * d.M;
    // r1 = dz, with its weight gradients
    CKF((wgrad<W, W, false, true>(f, B, f->r0, vl, nullptr, f->z + l * act, f->r1, f->grad + f->oM[l],
                                  f->grad + f->om[l])));
    // gY = (w_k / V) F(dz) on the kept modes
    CKF(fno_fwd_dft(f, f->r1, f->Y, C, invV, 2.f * invV));
    CKF(mix_bwd<W>(f, B, Xl, f->Y, f->tb + f->oR[l], f->grad + f->oR[l], f->gX));
    // dv = sum_k Re[gX e^{i k.x}] (the unnormalised inverse of gX / w_k) + M^T dz
    CKF(fno_inv_dft(f, f->gX, C, 1.f, 0.5f));
    CKF((fno_x_inv<W, false>(f, B, f->r1, f->tb + f->oM[l], nullptr, f->r0, nullptr)));
  }
  CKF((wgrad<W, 4, true, false>(f, B, f->r0, nullptr, Hd, nullptr, nullptr, f->grad + f->oP, f->grad + f->op)));
  return ACM_OK;
}

// Linear index of the voxel whose axes 0 and j (1 or 2) are swapped, on an
// n x n x n grid. The swap is its own inverse.
__device__ __forceinline__ long long swap_axes(long long i, int n, int j) {
  const int c = (int)(i % n), b = (int)((i / n) % n), a = (int)(i / ((long long)n * n));
  return j == 1 ? ((long long)b * n + a) * n + c : ((long long)c * n + b) * n + a;
}

__global__ void k_swap_h(const uint8_t* __restrict__ H, uint8_t* __restrict__ Hp, int n, int j, long long V,
                         long long total) {
  for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < total; t += (long long)gridDim.x * blockDim.x) {
    const long long b = t / V, i = t - b * V;
    Hp[t] = H[b * V + swap_axes(i, n, j)];
  }
}

// Predictions out' [B][6][V] for the load e_0 on the swapped cell become the
// warm start of load e_j on the cell: u_c(x) = u'_{s(c)}(s x) with s the swap
// of 0 and j (the identity for j = 0); the multiplier transforms alike.
// Outputs [B][3 loads][3][V]; this writes the slot of load j.
__global__ void k_unswap_out(const float* __restrict__ o, float* __restrict__ u, float* __restrict__ lam, int n, int j,
                             long long V, long long total) {
  for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < total; t += (long long)gridDim.x * blockDim.x) {
    const long long b = t / V, i = t - b * V;
    const long long si = j == 0 ? i : swap_axes(i, n, j);
    const float* ob = o + b * 6 * V;
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      const int sc = c == j ? 0 : (c == 0 ? j : c);
      const long long dst = ((b * 3 + j) * 3 + c) * V + i;
      u[dst] = ob[sc * V + si];
      lam[dst] = ob[(3 + sc) * V + si];
    }
  }
}

}  // namespace


namespace {

bool fno_on_device(const void* p) {
  cudaPointerAttributes a;
  if (cudaPointerGetAttributes(&a, p) != cudaSuccess) {
    cudaGetLastError();
    return false;
  }
  return a.type == cudaMemoryTypeDevice || a.type == cudaMemoryTypeManaged;
}

template <typename F>
acm_status dispatch_w(int W, F&& fn) {
  switch (W) {
    case 4: return fn(std::integral_constant<int, 4>());
    case 8: return fn(std::integral_constant<int, 8>());
    case 16: return fn(std::integral_constant<int, 16>());
    case 32: return fn(std::integral_constant<int, 32>());
    default: return ACM_ERR_ARG;
  }
}

void fno_free(acm_fno* f) {
  void* ps[] = {f->theta, f->tb, f->grad, f->m1, f->m2, f->v, f->z, f->X, f->Y, f->gX, f->r0, f->r1,
                f->dout, f->tgt, f->Hs, f->Hp, f->spec, f->part, f->lpart, f->tw};
  for (void* p : ps)
    if (p) cudaFree(p);
  cudaGetLastError();
}

}  // namespace

extern "C" {

acm_status acm_fno_create(acm_fno** out, int n0, int n1, int n2, int width, int modes, int layers, int max_batch,
                          void* stream) {
  if (!out) return ACM_ERR_ARG;
  *out = nullptr;
  auto p2 = [](int n) { return n >= 8 && n <= 512 && (n & (n - 1)) == 0; };
  if (!p2(n0) || !p2(n1) || !p2(n2)) return ACM_ERR_UNSUPPORTED_SIZE;
  if (!(width == 4 || width == 8 || width == 16 || width == 32) || modes < 1 || 2 * modes > n0 || 2 * modes > n1 ||
      modes > n2 / 2 || layers < 1 || layers > 16 || max_batch < 1 || max_batch > 64)
    return ACM_ERR_ARG;
  acm_fno* f = new (std::nothrow) acm_fno();
  if (!f) return ACM_ERR_NOMEM;
  FnoDims& d = f->d;
  d.n0 = n0;
  d.n1 = n1;
  d.n2 = n2;
  d.W = width;
  d.md = modes;
  d.L = layers;
  d.V = (long long)n0 * n1 * n2;
  d.M = 4 * modes * modes * modes;
  Geo& g = f->g;
  g.n0 = n0;
  g.n1 = n1;
  g.n2 = n2;
  g.Pu = n2 / 2 + 1;
  g.P = n2 / 2 + 4;
  g.V = d.V;
  g.S = (long long)n0 * n1 * g.P;
  g.hs = 0;
  g.us = 0;
  g.lph = 1;
  f->Bmax = max_batch;
  f->st = (cudaStream_t)stream;
  long long o = 0;
  f->oP = o;
  o += 4LL * width;
  f->op = o;
  o += width;
  for (int l = 0; l < layers; ++l) {
    f->oR.push_back(o);
    o += 2LL * d.M * width * width;
    f->oM.push_back(o);
    o += (long long)width * width;
    f->om.push_back(o);
    o += width;
  }
  f->oQ = o;
  o += 6LL * width;
  f->oq = o;
  o += 6;
  f->np = o;
  const long long act = (long long)max_batch * width * d.V;
  const long long ne = std::max((long long)width * width + width, 6LL * width + 6);
  const long long spec_elems = (long long)max_batch * width * n0 * modes * (n1 + 2LL * modes);
  bool ok = cudaMalloc(&f->theta, f->np * 4) == cudaSuccess && cudaMalloc(&f->tb, f->np * 2) == cudaSuccess &&
            cudaMalloc(&f->grad, f->np * 4) == cudaSuccess && cudaMalloc(&f->m1, f->np * 4) == cudaSuccess &&
            cudaMalloc(&f->m2, f->np * 4) == cudaSuccess &&
            cudaMalloc(&f->v, (layers + 1) * act * 2) == cudaSuccess &&
            cudaMalloc(&f->z, layers * act * 2) == cudaSuccess &&
            cudaMalloc(&f->X, (long long)layers * max_batch * width * d.M * sizeof(cx<float>)) == cudaSuccess &&
            cudaMalloc(&f->Y, (long long)max_batch * width * d.M * sizeof(cx<float>)) == cudaSuccess &&
            cudaMalloc(&f->gX, (long long)max_batch * width * d.M * sizeof(cx<float>)) == cudaSuccess &&
            cudaMalloc(&f->r0, act * 4) == cudaSuccess && cudaMalloc(&f->r1, act * 4) == cudaSuccess &&
            cudaMalloc(&f->dout, (long long)max_batch * 6 * d.V * 4) == cudaSuccess &&
            cudaMalloc(&f->tgt, (long long)max_batch * 6 * d.V * 4) == cudaSuccess &&
            cudaMalloc(&f->Hs, (long long)max_batch * d.V) == cudaSuccess &&
            cudaMalloc(&f->spec, spec_elems * sizeof(cx<float>)) == cudaSuccess &&
            cudaMalloc(&f->part, NRB * ne * 4) == cudaSuccess &&
            cudaMalloc(&f->lpart, NRB * sizeof(double)) == cudaSuccess &&
            cudaMalloc(&f->tw, 2 * TW_MAX * sizeof(float)) == cudaSuccess;
  if (!ok) {
    cudaGetLastError();
    fno_free(f);
    delete f;
    return ACM_ERR_NOMEM;
  }
  std::vector<float> tw(2 * TW_MAX);
  const double PI = 3.14159265358979323846;
  for (int k = 0; k < TW_MAX; ++k) {
    tw[2 * k] = (float)std::cos(2.0 * PI * k / TW_MAX);
    tw[2 * k + 1] = (float)(-std::sin(2.0 * PI * k / TW_MAX));
  }
  if (cudaMemcpy(f->tw, tw.data(), tw.size() * 4, cudaMemcpyHostToDevice) != cudaSuccess ||
      cudaMemset(f->theta, 0, f->np * 4) != cudaSuccess || cudaMemset(f->tb, 0, f->np * 2) != cudaSuccess ||
      cudaMemset(f->m1, 0, f->np * 4) != cudaSuccess || cudaMemset(f->m2, 0, f->np * 4) != cudaSuccess ||
      cudaMemset(f->grad, 0, f->np * 4) != cudaSuccess) {
    cudaGetLastError();
    fno_free(f);
    delete f;
    return ACM_ERR_CUDA;
  }
  *out = f;
  return ACM_OK;
}

acm_status acm_fno_destroy(acm_fno* f) {
  if (!f) return ACM_ERR_ARG;
  if (f->st) cudaStreamSynchronize(f->st);
  else cudaDeviceSynchronize();
  fno_free(f);
  delete f;
  return ACM_OK;
}

acm_status acm_fno_num_params(acm_fno* f, long long* n) {
  if (!f || !n) return ACM_ERR_ARG;
  *n = f->np;
  return ACM_OK;
}

acm_status acm_fno_set_params(acm_fno* f, const float* theta) {
  if (!f || !theta) return ACM_ERR_ARG;
  FK(cudaMemcpyAsync(f->theta, theta, f->np * 4, cudaMemcpyDefault, f->st));
  k_f32_to_bf16<<<blocks_for(f->np), 256, 0, f->st>>>(f->theta, f->tb, f->np);
  FK(cudaGetLastError());
  FK(cudaMemsetAsync(f->m1, 0, f->np * 4, f->st));
  FK(cudaMemsetAsync(f->m2, 0, f->np * 4, f->st));
  f->step = 0;
  FK(cudaStreamSynchronize(f->st));
  return ACM_OK;
}

acm_status acm_fno_get_params(acm_fno* f, float* theta) {
  if (!f || !theta) return ACM_ERR_ARG;
  FK(cudaMemcpyAsync(theta, f->theta, f->np * 4, cudaMemcpyDefault, f->st));
  FK(cudaStreamSynchronize(f->st));
  return ACM_OK;
}

static acm_status stage_inputs(acm_fno* f, int B, const uint8_t* H, const uint8_t** Hd) {
  if (fno_on_device(H)) {
    *Hd = H;
  } else {
    FK(cudaMemcpyAsync(f->Hs, H, (size_t)B * f->d.V, cudaMemcpyHostToDevice, f->st));
    *Hd = f->Hs;
  }
  return ACM_OK;
}

acm_status acm_fno_forward(acm_fno* f, int batch, const uint8_t* H, float* out) {
  if (!f || !H || batch < 1 || batch > f->Bmax) return ACM_ERR_ARG;
  const uint8_t* Hd = nullptr;
  CKF(stage_inputs(f, batch, H, &Hd));
  float* o = out && fno_on_device(out) ? out : f->dout;
  CKF(dispatch_w(f->d.W, [&](auto w) { return fno_forward_impl<decltype(w)::value>(f, batch, Hd, nullptr, o, nullptr); }));
  if (out && o != out) FK(cudaMemcpyAsync(out, o, (size_t)batch * 6 * f->d.V * 4, cudaMemcpyDeviceToHost, f->st));
  FK(cudaStreamSynchronize(f->st));
  return ACM_OK;
}

acm_status acm_fno_warm_start(acm_fno* f, int batch, const uint8_t* H, float* init_u, float* init_lambda) {
  if (!f || !H || !init_u || !init_lambda || batch < 1 || batch > f->Bmax) return ACM_ERR_ARG;
  const Geo& g = f->g;
  if (g.n0 != g.n1 || g.n0 != g.n2) return ACM_ERR_UNSUPPORTED_SIZE;
  if (!fno_on_device(init_u) || !fno_on_device(init_lambda)) return ACM_ERR_ARG;
  const uint8_t* Hd = nullptr;
  CKF(stage_inputs(f, batch, H, &Hd));
  if (!f->Hp) FK(cudaMalloc(&f->Hp, (size_t)f->Bmax * f->d.V));
  const long long total = (long long)batch * f->d.V;
  for (int j = 0; j < 3; ++j) {
    const uint8_t* Hj = Hd;
    if (j > 0) {
      k_swap_h<<<blocks_for(total), 256, 0, f->st>>>(Hd, f->Hp, g.n0, j, f->d.V, total);
      FK(cudaGetLastError());
      Hj = f->Hp;
    }
    CKF(dispatch_w(f->d.W, [&](auto w) {
      return fno_forward_impl<decltype(w)::value>(f, batch, Hj, nullptr, f->dout, nullptr);
    }));
    k_unswap_out<<<blocks_for(total), 256, 0, f->st>>>(f->dout, init_u, init_lambda, g.n0, j, f->d.V, total);
    FK(cudaGetLastError());
  }
  FK(cudaStreamSynchronize(f->st));
  return ACM_OK;
}

acm_status acm_fno_backward(acm_fno* f, int batch, const uint8_t* H, const float* target, double* loss, float* grad) {
  if (!f || !H || !target || batch < 1 || batch > f->Bmax) return ACM_ERR_ARG;
  const uint8_t* Hd = nullptr;
  CKF(stage_inputs(f, batch, H, &Hd));
  const float* t = target;
  if (!fno_on_device(target)) {
    FK(cudaMemcpyAsync(f->tgt, target, (size_t)batch * 6 * f->d.V * 4, cudaMemcpyHostToDevice, f->st));
    t = f->tgt;
  }
  double L = 0;
  CKF(dispatch_w(f->d.W, [&](auto w) {
    acm_status s = fno_forward_impl<decltype(w)::value>(f, batch, Hd, t, nullptr, &L);
    if (s != ACM_OK) return s;
    return fno_backward_impl<decltype(w)::value>(f, batch, Hd);
  }));
  if (loss) *loss = L;
  if (grad) FK(cudaMemcpyAsync(grad, f->grad, f->np * 4, cudaMemcpyDefault, f->st));
  FK(cudaStreamSynchronize(f->st));
  return ACM_OK;
}

acm_status acm_fno_adamw(acm_fno* f, double lr, double beta1, double beta2, double eps, double weight_decay) {
  if (!f || !(lr > 0) || !(beta1 >= 0 && beta1 < 1) || !(beta2 >= 0 && beta2 < 1) || !(eps > 0) ||
      !(weight_decay >= 0))
    return ACM_ERR_ARG;
  f->step += 1;
  const float c1 = (float)(1.0 - std::pow(beta1, (double)f->step));
  const float c2 = (float)(1.0 - std::pow(beta2, (double)f->step));
  k_adamw<<<blocks_for(f->np), 256, 0, f->st>>>(f->theta, f->tb, f->grad, f->m1, f->m2, f->np, (float)lr,
                                                  (float)beta1, (float)beta2, (float)eps, (float)weight_decay, c1, c2);
  FK(cudaGetLastError());
  return ACM_OK;
}

}  // extern "C"
