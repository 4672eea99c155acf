// acm_misc.cu -- precision-independent kernels: FP64 finalize steps of both
// iterations, precision conversion and the solid-voxel count.
#include "acm_fft.cuh"
#include "acm_kernels.cuh"
#include "acm_ops.h"

namespace acm {
// ---------------------------------------------------------------------------
// finalize kernels: deterministic FP64 sums of the partials, Eq. 10-12, Eq. 22
// ---------------------------------------------------------------------------
// One finalize block per problem. FP64 runs on two lanes an SM, so the block sums
// eight values at once by halving: a warp's lanes exchange half of their values at
// each of the first three steps (4 + 2 + 1 + 1 + 1 additions a lane, against 40
// for eight butterflies), and the residuals, tolerances and penalties are formed
// by one lane each. A problem's whole step took 18 us a launch as eight butterflies
// and one thread's chain of square roots, divisions and loads of its control block.
constexpr int FIN_VALS = 8;
constexpr int FIN_MAXW = 32;

// Sums v[0..7] over the block; lane k (mod 8) of warp 0 returns the total of value
// k. scratch: FIN_VALS * FIN_MAXW doubles. Deterministic for a fixed block size.
__device__ __forceinline__ double block_sum8(double (&v)[FIN_VALS], double* scratch) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
  // after the step over bit `o` a lane holds the values whose index has the lane's
  // bit there: value index k = lane & 7
#pragma unroll
  for (int o = 4, n = 4; o >= 1; o >>= 1, n >>= 1) {
#pragma unroll
    for (int i = 0; i < n; ++i) {
      const bool up = lane & o;
      const double keep = up ? v[i + n] : v[i], give = up ? v[i] : v[i + n];
      v[i] = keep + __shfl_xor_sync(0xffffffffu, give, o);
    }
  }
  double a = v[0];
  a += __shfl_xor_sync(0xffffffffu, a, 8);
  a += __shfl_xor_sync(0xffffffffu, a, 16);
  if (lane < FIN_VALS) scratch[warp * FIN_VALS + lane] = a;
  __syncthreads();
  double r = 0.0;
  if (warp == 0) {
    for (int w = lane >> 3; w < nw; w += 4) r += scratch[w * FIN_VALS + (lane & 7)];
    r += __shfl_xor_sync(0xffffffffu, r, 8);
    r += __shfl_xor_sync(0xffffffffu, r, 16);
  }
  return r;
}

// adds the records part[i][0..NV) (stride doubles apart, pairs 16-byte aligned) of
// the thread's share to v[0..NV)
template <int NV>
__device__ __forceinline__ void add_partials(const double* __restrict__ part, int nblk, int stride, double* v) {
#pragma unroll 4
  for (int i = threadIdx.x; i < nblk; i += blockDim.x) {
    const double2* q = reinterpret_cast<const double2*>(part + (long long)i * stride);
#pragma unroll
    for (int k = 0; k < NV; k += 2) {
      const double2 x = q[k / 2];
      v[k] += x.x;
      if (k + 1 < NV) v[k + 1] += x.y;
    }
  }
}

// Stagnation test of an FP32 phase (off when win = 0): the distance to the
// tolerance m = max_k r[k] / t[k] must fall below STALL_DROP times its best
// value within `win` iterations, else the phase has reached its rounding floor.
__device__ __forceinline__ bool stalled(int win, int& n, double& best, double m) {
  if (win <= 0) return false;
  if (m < STALL_DROP * best) {
    best = m;
    n = 0;
    return false;
  }
  return ++n >= win;
}

__device__ __forceinline__ double shfl(double x, int src) { return __shfl_sync(0xffffffffu, x, src); }

__global__ void __launch_bounds__(1024) k_stokes_finalize(StokesDev* __restrict__ prm, const double* __restrict__ part_x,
                                                         int nbx, const double* __restrict__ part_z, int nbz,
                                                         double V, double* __restrict__ hist, int hist_cap) {
  __shared__ double red[FIN_VALS * FIN_MAXW];
  const int p = blockIdx.x;
  StokesDev* P = prm + p;
  if (P->done) return;
  const int lane = threadIdx.x;
  const bool first = threadIdx.x < 32;
  // warp 0 reads the control block while the partial sums travel: lane k holds
  // entry k of the vectors
  const int k3 = lane < 3 ? lane : 0;
  double psi = 0, phi = 0, tau = 0, psi_min = 0, mean = 0, e = 0, b_next = 0;
  int adaptive = 0, max_iter = 0, iter = 0, iter_base = 0, stall_win = 0;
  if (first) {
    psi = P->psi[k3];
    phi = P->phi[k3];
    tau = P->tau[k3];
    psi_min = P->psi_min[k3];
    mean = P->mean_u[k3];
    e = P->eps;
    b_next = P->b_next;
    adaptive = P->adaptive;
    max_iter = P->max_iter;
    iter = P->iter;
    iter_base = P->iter_base;
    stall_win = P->stall_win;
  }
  // values 0..4: the x pass (||Hu~||^2, ||H(u~ - u~_old)||^2, ||u - u~||^2,
  // ||u - u_old||^2, ||lambda||^2), 5..7: the z pass (V times ||div u||^2,
  // ||div (u - u_old)||^2, ||q||^2)
  double v[FIN_VALS] = {0, 0, 0, 0, 0, 0, 0, 0};
  add_partials<5>(part_x + (long long)p * nbx * 8, nbx, 8, v);
  add_partials<3>(part_z + (long long)p * nbz * 4, nbz, 4, v + 5);
  const double total = block_sum8(v, red);
  if (!first) return;
  // lane k: the norm of value k (all 32 lanes compute, eight distinct values)
  const double nrm = sqrt((lane & 7) >= 5 ? total / V : total);
  const double n0 = shfl(nrm, 0), n1 = shfl(nrm, 1), n2 = shfl(nrm, 2), n3 = shfl(nrm, 3), nl = shfl(nrm, 4);
  const double z0 = shfl(nrm, 5), z1 = shfl(nrm, 6), nq = shfl(nrm, 7);
  const double alpha = shfl(psi, 0), beta = shfl(psi, 1), b = shfl(psi, 2);
  // lane k < 6: residual k (Eq. 10) and its tolerance (Eq. 11-12); a = H lambda
  const double r = lane == 0 ? n0 : lane == 1 ? alpha * n1 : lane == 2 ? z0 : lane == 3 ? beta * z1
                   : lane == 4 ? n2 : b * n3;
  const bool pair2 = (lane >> 1) == 1;
  const double s = sqrt(pair2 ? V : 3.0 * V) * e, nm = pair2 ? nq : nl;
  const double t = s + e * ((lane & 1) ? nm : fmax(r, nm));
  const unsigned six = 0x3fu;
  const bool conv = (__ballot_sync(0xffffffffu, r <= t) & six) == six;
  const bool finite = (__ballot_sync(0xffffffffu, isfinite(r)) & six) == six;
  const int it = iter + 1;
  if (lane < 6) {
    P->res[lane] = r;
    P->tol[lane] = t;
  }
  if (hist && it + iter_base <= hist_cap) {
    double* h = hist + ((long long)p * hist_cap + (it + iter_base - 1)) * STOKES_HIST;
    if (lane < 6) {
      h[lane] = r;
      h[6 + lane] = t;
    }
    if (lane < 3) {
      h[12 + lane] = psi;
      h[15 + lane] = mean;
    }
    if (lane < 2) h[18 + lane] = 0.0;
  }
  const double rp = shfl(r, 2 * k3), rd = shfl(r, 2 * k3 + 1);
  if (lane < 3) {
    P->psi_last[lane] = psi;
    P->psi_prev[lane] = psi;
    double next = psi, guess = psi;  // guess: the change of this iteration once more
    if (adaptive) {  // Eq. 22: pair k drives (alpha, beta, b)[k]
      if (rp > tau * rd) {
        next = phi * psi;
        guess = phi * next;
      } else if (rd > tau * rp) {
        next = fmax(psi / phi, psi_min);
        guess = fmax(next / phi, psi_min);
      }
      P->psi[lane] = next;
    }
    if (lane == 2) {
      P->rhs_ok = next == b_next;
      P->b_next = guess;
    }
  }
  double m = 0.0;
  if (stall_win > 0) {
    const double q = lane < 6 ? (t > 0.0 ? r / t : r) : 0.0;
    for (int i = 0; i < 6; ++i) m = fmax(m, shfl(q, i));
  }
  if (lane != 0) return;
  P->iter = it;
  if (!finite) {
    P->done = 1;
    P->status = ST_NONFINITE;
  } else if (conv) {
    P->done = 1;
    P->converged = 1;
    P->status = ST_OK;
  } else if (stalled(stall_win, P->stall_n, P->stall_best, m)) {
    P->done = 1;
    P->status = ST_STALLED;
  } else if (it >= max_iter) {
    P->done = 1;
    P->status = ST_MAXITER;
  }
}

__global__ void __launch_bounds__(1024) k_solute_finalize(SoluteDev* __restrict__ prm, const double* __restrict__ part_z,
                                                         int nbz, double V, double* __restrict__ hist, int hist_cap) {
  __shared__ double red[FIN_VALS * FIN_MAXW];
  const int p = blockIdx.x;
  SoluteDev* P = prm + p;
  if (P->done) return;
  const int lane = threadIdx.x;
  const bool first = threadIdx.x < 32;
  double eps = 0, rmin = 0;
  int max_iter = 0, iter = 0, iter_base = 0, stall_win = 0;
  if (first) {
    eps = P->eps;
    rmin = P->rmin;
    max_iter = P->max_iter;
    iter = P->iter;
    iter_base = P->iter_base;
    stall_win = P->stall_win;
  }
  double v[FIN_VALS] = {0, 0, 0, 0, 0, 0, 0, 0};
  add_partials<2>(part_z + (long long)p * nbz * 4, nbz, 4, v);
  const double total = block_sum8(v, red);
  if (!first) return;
  // lane 0: r1 and its tolerance, lane 1: r2 (Eq. 19)
  const double r = sqrt(total / V), t = sqrt((lane & 1) ? 3.0 * V : V) * eps;
  const int it = iter + 1;
  if (lane < 2) {
    P->res[lane] = r;
    P->tol[lane] = t;
    if (hist && it + iter_base <= hist_cap) {
      double* h = hist + ((long long)p * hist_cap + (it + iter_base - 1)) * SOLUTE_HIST;
      h[lane] = r;
      h[2 + lane] = t;
    }
  }
  const bool finite = (__ballot_sync(0xffffffffu, isfinite(r)) & 3u) == 3u;
  const bool conv = (__ballot_sync(0xffffffffu, r <= t) & 3u) == 3u;
  const double q = stall_win > 0 ? (t > 0.0 ? r / t : r) : 0.0, q1 = shfl(q, 1);
  if (lane != 0) return;
  P->iter = it;
  const double rn = r / (1.0 + t);
  if (!finite) {
    P->done = 1;
    P->status = ST_NONFINITE;
    return;
  }
  if (conv) {
    P->done = 1;
    P->converged = 1;
    P->status = ST_OK;
    return;
  }
  if (it > 20 && rn > 1e3 * rmin) {
    P->done = 1;
    P->status = ST_DIVERGED;
    return;
  }
  if (rn < rmin) P->rmin = rn;
  if (stalled(stall_win, P->stall_n, P->stall_best, fmax(fmax(0.0, q), q1))) {
    P->done = 1;
    P->status = ST_STALLED;
    return;
  }
  if (it >= max_iter) {
    P->done = 1;
    P->status = ST_MAXITER;
  }
}

// solid-pore faces of the periodic voxel grid: each voxel counts the faces it
// shares with its +1 neighbours along the three axes where H changes (a grid of
// one plane has no face along axis 0)
__global__ void k_count_faces(const uint8_t* __restrict__ H, int n0, int n1, int n2, unsigned long long* out) {
  const long long V = (long long)n0 * n1 * n2;
  unsigned long long c = 0;
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < V; i += (long long)gridDim.x * blockDim.x) {
    const int i2 = (int)(i % n2);
    const long long r = i / n2;
    const int i1 = (int)(r % n1), i0 = (int)(r / n1);
    const uint8_t h = H[i] != 0;
    const long long a0 = ((long long)((i0 + 1) % n0) * n1 + i1) * n2 + i2;
    const long long a1 = ((long long)i0 * n1 + (i1 + 1) % n1) * n2 + i2;
    const long long a2 = ((long long)i0 * n1 + i1) * n2 + (i2 + 1) % n2;
    c += (unsigned long long)(h != (H[a0] != 0)) + (h != (H[a1] != 0)) + (h != (H[a2] != 0));
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) c += __shfl_xor_sync(0xffffffffu, c, o);
  if ((threadIdx.x & 31) == 0 && c) atomicAdd(out, c);
}

__global__ void k_count_solid(const uint8_t* __restrict__ H, long long V, unsigned long long* out) {
  unsigned long long c = 0;
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < V; i += (long long)gridDim.x * blockDim.x)
    c += H[i] ? 1ull : 0ull;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) c += __shfl_xor_sync(0xffffffffu, c, o);
  if ((threadIdx.x & 31) == 0 && c) atomicAdd(out, c);
}

__global__ void __launch_bounds__(256) k_loop_control(LoopCtl c) {
  __shared__ int any;
  if (threadIdx.x == 0) any = 0;
  __syncthreads();
  int mine = 0;
  for (int gi = 0; gi < c.ngroups; ++gi)
    for (int i = threadIdx.x; i < c.n[gi]; i += blockDim.x)
      mine |= (*reinterpret_cast<const int*>(c.base[gi] + (size_t)i * c.stride[gi] + c.done_off) == 0);
  if (mine) any = 1;
  __syncthreads();
  if (threadIdx.x == 0) {
    const unsigned int it = *c.counter + c.step;
    *c.counter = it;
    cudaGraphSetConditional(c.handle, (any && it < c.cap) ? 1u : 0u);
  }
}

cudaError_t loop_control(const LoopCtl& c, cudaStream_t s) {
  k_loop_control<<<1, 256, 0, s>>>(c);
  return cudaGetLastError();
}

// a thread of the finalize block takes about four records, in blocks of 128 to 1024
static int fin_threads(int records) {
  int t = 128;
  while (t < 1024 && records > 4 * t) t *= 2;
  return t;
}

cudaError_t stokes_finalize(int nprob, StokesDev* prm, const double* part_x, int nbx, const double* part_z,
                            int nbz, double V, double* hist, int hist_cap, cudaStream_t s) {
  k_stokes_finalize<<<nprob, fin_threads(nbx > nbz ? nbx : nbz), 0, s>>>(prm, part_x, nbx, part_z, nbz, V, hist, hist_cap);
  return cudaGetLastError();
}

cudaError_t solute_finalize(int nprob, SoluteDev* prm, const double* part_z, int nbz, double V, double* hist,
                            int hist_cap, cudaStream_t s) {
  k_solute_finalize<<<nprob, fin_threads(nbz), 0, s>>>(prm, part_z, nbz, V, hist, hist_cap);
  return cudaGetLastError();
}

// one bit per voxel of H: word w holds voxels 32 w .. 32 w + 31 (n a multiple of
// 32, so every warp of the grid-stride loop sees 32 valid voxels)
__global__ void k_hbits(const uint8_t* __restrict__ H, uint32_t* __restrict__ Hb, long long n) {
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
    const unsigned b = __ballot_sync(0xffffffffu, H[i] != 0);
    if ((threadIdx.x & 31) == 0) Hb[i >> 5] = b;
  }
}

cudaError_t pack_hbits(const uint8_t* H, uint32_t* Hb, long long n, cudaStream_t s) {
  if (n % 32 != 0) return cudaErrorInvalidValue;
  k_hbits<<<608, 256, 0, s>>>(H, Hb, n);
  return cudaGetLastError();
}

cudaError_t count_solid(const uint8_t* H, long long V, unsigned long long* out, cudaStream_t s) {
  cudaError_t e = cudaMemsetAsync(out, 0, sizeof(unsigned long long), s);
  if (e != cudaSuccess) return e;
  k_count_solid<<<304, 256, 0, s>>>(H, V, out);
  return cudaGetLastError();
}

cudaError_t count_faces_add(const uint8_t* H, int n0, int n1, int n2, unsigned long long* out, cudaStream_t s) {
  k_count_faces<<<304, 256, 0, s>>>(H, n0, n1, n2, out);
  return cudaGetLastError();
}

cudaError_t count_solid_add(const uint8_t* H, long long V, unsigned long long* out, cudaStream_t s) {
  k_count_solid<<<304, 256, 0, s>>>(H, V, out);
  return cudaGetLastError();
}

cudaError_t convert_f2d(const float* in, double* out, long long n, cudaStream_t s) {
  k_convert<float, double><<<608, 256, 0, s>>>(in, out, n);
  return cudaGetLastError();
}

cudaError_t convert_d2f(const double* in, float* out, long long n, cudaStream_t s) {
  k_convert<double, float><<<608, 256, 0, s>>>(in, out, n);
  return cudaGetLastError();
}

}  // namespace acm
