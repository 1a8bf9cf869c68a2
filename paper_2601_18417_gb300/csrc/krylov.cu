// krylov.cu -- vector kernels of the flexible GMRES outer solver and the
// compact-stencil approximate-Jacobian preconditioner (arXiv 2601.18417,
// Sec. 4.1).
//
// Reductions are deterministic: each block writes a partial sum, and the
// last block to finish (an atomic ticket, no waiting) adds the partials in
// block order and publishes the result to device memory, where the next
// kernel on the stream reads it.  No host round trip is needed inside Jv or
// inside the preconditioner.
#include <stdlib.h>

#include "hofv_internal.cuh"
#include "reduce.cuh"

namespace hofv {

constexpr int kRedThreads = 256;

// Sums of NV values a thread over the block, value k in lane 0 of warp k: the
// warps' lanes first, one warp a value, so that FP64 additions, which hold
// the pipe for 16 cycles a warp, are 13 a value and not 40.
template <int NV>
__device__ __forceinline__ double block_sums(const double (&v)[NV], double* sh) {
  constexpr int NW = kRedThreads / 32;
  static_assert(NV <= NW, "a warp a value");
#pragma unroll
  for (int k = 0; k < NV; ++k) sh[k * kRedThreads + threadIdx.x] = v[k];
  __syncthreads();
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  double t = 0.0;
  if (wid < NV) {
    double q[NW];
#pragma unroll
    for (int i = 0; i < NW; ++i) q[i] = sh[wid * kRedThreads + i * 32 + lane];
#pragma unroll
    for (int h = NW / 2; h > 0; h /= 2)  // pairwise: the additions' latency counts
#pragma unroll
      for (int i = 0; i < h; ++i) q[i] += q[i + h];
    t = q[0];
    for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
  }
  return t;
}

// True in all threads of the last of n blocks to come here; the writers of what
// that block reads have each put a fence behind their writes.
__device__ __forceinline__ bool last_to_come(unsigned int* count, unsigned int n) {
  __shared__ bool last;
  __syncthreads();
  if (threadIdx.x == 0) {
    last = atomicAdd(count, 1u) == n - 1;
    __threadfence();
  }
  __syncthreads();
  return last;
}

// out[k0 + k] = x_k . y for NV vectors x_k = X + (k0 + k) * ldx
template <int NV>
__device__ __forceinline__ void mdot(const double* __restrict__ X, int64_t ldx, const double* __restrict__ y,
                                     int64_t n, int k0, double* red, unsigned int* count, double* out, int mode,
                                     double* sh) {
  double s[NV];
#pragma unroll
  for (int k = 0; k < NV; ++k) s[k] = 0.0;
  const double* __restrict__ x = X + k0 * ldx;
#pragma unroll 4
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n;
       i += (int64_t)gridDim.x * blockDim.x) {
    const double yi = y[i];
#pragma unroll
    for (int k = 0; k < NV; ++k) s[k] = fma(x[k * ldx + i], yi, s[k]);
  }
  const double t = block_sums<NV>(s, sh);
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  if (wid < NV && lane == 0) {
    __stcg(red + (k0 + wid) * gridDim.x + blockIdx.x, t);
    __threadfence();
  }
  if (last_to_come(count + blockIdx.y, gridDim.x)) {
    if (wid < NV) {  // a warp a vector, in block order
      const double* r = red + (k0 + wid) * gridDim.x;
      double a = 0.0;
#pragma unroll 8
      for (unsigned int b = lane; b < gridDim.x; b += 32) a += __ldcg(r + b);
      for (int o = 16; o > 0; o >>= 1) a += __shfl_xor_sync(0xffffffffu, a, o);
      if (lane == 0) out[k0 + wid] = mode == 1 ? sqrt(a) : a;
    }
    if (threadIdx.x == 0) count[blockIdx.y] = 0;
  }
}

// kMdot vectors a block.  The pass is bound by the FP64 pipe (22 us for 16
// vectors of 64^3 x 3); one vector a block with a shuffle tree in each warp
// took 35 us (27 on 512^2 x 2, pipe 15), this 31 (23): y is read a quarter as often
// and the reductions are a tenth of the FP64 instructions.
constexpr int kMdot = 4;
__global__ void __launch_bounds__(kRedThreads)
    k_mdot(const double* __restrict__ X, int64_t ldx, const double* __restrict__ y, int nvec, int64_t n,
           double* red, unsigned int* count, double* out, int mode) {
  __shared__ double sh[kMdot * kRedThreads];
  const int k0 = blockIdx.y * kMdot;
  switch (min(nvec - k0, kMdot)) {
    case 1: return mdot<1>(X, ldx, y, n, k0, red, count, out, mode, sh);
    case 2: return mdot<2>(X, ldx, y, n, k0, red, count, out, mode, sh);
    case 3: return mdot<3>(X, ldx, y, n, k0, red, count, out, mode, sh);
    default: return mdot<kMdot>(X, ldx, y, n, k0, red, count, out, mode, sh);
  }
}

void launch_dots(const double* X, int64_t ldx, const double* y, int nvec, int64_t n, double* red,
                 unsigned int* count, double* out, int blocks, cudaStream_t st, int mode) {
  // few blocks per vector: every block ends in FP64 warp reductions
  blocks = (int)std::min<int64_t>(std::max(blocks / 4, 1), (n + kRedThreads - 1) / kRedThreads);
  dim3 grid((unsigned)blocks, (unsigned)((nvec + kMdot - 1) / kMdot));
  k_mdot<<<grid, kRedThreads, 0, st>>>(X, ldx, y, nvec, n, red, count, out, mode);
}

void launch_norm2(const double* x, int64_t n, double* red, unsigned int* count, double* out,
                  int blocks, cudaStream_t st) {
  launch_dots(x, 0, x, 1, n, red, count, out, blocks, st, 1);
}

// sc[1] = ||v||, sc[0] = ||u|| (slice 1, where the launch has it), then
// sc[2] = eps = sqrt(2^-52) (1 + ||u||) / ||v|| (1 if v = 0) and sc[3] = 1 / eps,
// which the assembly would divide out in every thread.  One launch for
// what took three, each mostly latency: a product on 13^3 hexes 92 -> 84 us.
// A step's rounding passes through eps to the whole difference quotient, so the
// sums are in the order of separate norms, block_sum's.
__global__ void k_jv_norms(const double* __restrict__ v, const double* __restrict__ u, int64_t n, double* red,
                           unsigned int* count, unsigned int* slices, double* sc) {
  __shared__ double sh[32];
  const int k = blockIdx.y;
  const double* x = k == 0 ? v : u;
  double s = 0.0;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n;
       i += (int64_t)gridDim.x * blockDim.x)
    s = fma(x[i], x[i], s);
  const double bs = block_sum(s, sh);
  if (threadIdx.x == 0) {
    __stcg(red + k * gridDim.x + blockIdx.x, bs);
    __threadfence();
  }
  if (last_to_come(count + k, gridDim.x)) {
    const double t = warp0_sum(red + k * gridDim.x, gridDim.x);
    if (threadIdx.x == 0) {
      __stcg(sc + 1 - k, sqrt(t));
      count[k] = 0;
      __threadfence();
      if (atomicAdd(slices, 1u) == gridDim.y - 1) {  // both norms are there
        __threadfence();
        const double vn = __ldcg(sc + 1);
        const double eps = vn > 0.0 ? 1.4901161193847656e-08 * (1.0 + __ldcg(sc)) / vn : 1.0;
        sc[2] = eps;
        sc[3] = 1.0 / eps;
        *slices = 0;
      }
    }
  }
}
void launch_jv_norms(const double* v, const double* u, int64_t n, double* red, unsigned int* count, double* sc,
                     int blocks, cudaStream_t st) {
  blocks = (int)std::min<int64_t>(std::max(blocks / 4, 1), (n + kRedThreads - 1) / kRedThreads);
  k_jv_norms<<<dim3((unsigned)blocks, u ? 2 : 1), kRedThreads, 0, st>>>(v, u, n, red, count, count + 255, sc);
}

// y = x + sign * alpha[0] * v   (alpha read on the device)
__global__ void k_axpy_dev(double* __restrict__ y, const double* __restrict__ x,
                           const double* __restrict__ v, const double* alpha, double sign,
                           int64_t n) {
  const double a = sign * alpha[0];
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n;
       i += (int64_t)gridDim.x * blockDim.x)
    y[i] = fma(a, v[i], x[i]);
}
void launch_waxpy_dev(double* y, const double* x, const double* v, const double* alpha,
                      double sign, int64_t n, cudaStream_t st) {
  k_axpy_dev<<<(unsigned)std::min<int64_t>((n + 255) / 256, 4096), 256, 0, st>>>(y, x, v, alpha,
                                                                              sign, n);
}

// y = x * s[0] (invert: x / s[0])
__global__ void k_scale_copy(double* __restrict__ y, const double* __restrict__ x,
                             const double* s, int invert, int64_t n) {
  __shared__ double f;  // one quotient a block, on the FP64 pipe for 16 cycles an instruction
  if (threadIdx.x == 0) f = invert ? 1.0 / s[0] : s[0];
  __syncthreads();
#pragma unroll 4
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n;
       i += (int64_t)gridDim.x * blockDim.x)
    y[i] = x[i] * f;
}
void launch_scale_copy(double* y, const double* x, const double* s, int invert, int64_t n, int blocks,
                       cudaStream_t st) {
  // four blocks an SM at most: 512^2 x 2 7.9 -> 3.6 us with the quotient once a block
  k_scale_copy<<<(unsigned)std::min<int64_t>((n + 255) / 256, blocks), 256, 0, st>>>(y, x, s, invert, n);
}

// w -= sum_k coef[k] V_k  (coef on the device)
__global__ void k_multi_axpy(double* __restrict__ w, const double* __restrict__ V,
                             const double* __restrict__ coef, int k, int64_t n, int64_t ld) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n;
       i += (int64_t)gridDim.x * blockDim.x) {
    double s = w[i];
    for (int j = 0; j < k; ++j) s = fma(-coef[j], V[j * ld + i], s);
    w[i] = s;
  }
}
void launch_multi_axpy(double* w, const double* V, const double* coef, int k, int64_t n,
                       int64_t ld, cudaStream_t st) {
  k_multi_axpy<<<(unsigned)std::min<int64_t>((n + 255) / 256, 8192), 256, 0, st>>>(w, V, coef, k,
                                                                                 n, ld);
}

// x += sum_k y[k] Z_k  (y on the device)
__global__ void k_combine(double* __restrict__ x, const double* __restrict__ Z,
                          const double* __restrict__ y, int k, int64_t n, int64_t ld) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n;
       i += (int64_t)gridDim.x * blockDim.x) {
    double s = x[i];
    for (int j = 0; j < k; ++j) s = fma(y[j], Z[j * ld + i], s);
    x[i] = s;
  }
}
void launch_combine(double* x, const double* Z, const double* y, int k, int64_t n, int64_t ld,
                    cudaStream_t st) {
  k_combine<<<(unsigned)std::min<int64_t>((n + 255) / 256, 8192), 256, 0, st>>>(x, Z, y, k, n, ld);
}

// y = a x + b y
__global__ void k_axpby(double* __restrict__ y, double a, const double* __restrict__ x, double b,
                        int64_t n) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n;
       i += (int64_t)gridDim.x * blockDim.x)
    y[i] = fma(a, x[i], b * y[i]);
}
void launch_axpby(double* y, double a, const double* x, double b, int64_t n, cudaStream_t st) {
  k_axpby<<<(unsigned)std::min<int64_t>((n + 255) / 256, 4096), 256, 0, st>>>(y, a, x, b, n);
}

// ---------------------------------------------------------------------
// approximate Jacobian A = Kbar * A1 (Sec. 4.1), A1 negative definite with
// Kbar = 1.  z = A^{-1} v solves B z = -v / Kbar with B = -A1 (SPD), by a
// fixed number of Jacobi-preconditioned conjugate-gradient iterations on
// all `dim` right-hand sides at once, in the single-reduction form of
// Chronopoulos & Gear (J. Comput. Appl. Math. 25, 1989): per iteration one
// product w = B u (u = D^{-1} r) and the two inner products (r,u), (w,u),
// with s = B p carried by recurrence.  One kernel per iteration: the vector
// updates of iteration i-1 are recomputed on the fly for the neighbours
// that the product of iteration i reads (r, w and s are double-buffered),
// so no grid-wide synchronisation is needed.  T = float or double.
// Scalars (double): sc[0..d) gamma_prev, sc[d..2d) alpha, sc[2d..3d) beta.
// ---------------------------------------------------------------------
template <typename T, int DIM>
__device__ __forceinline__ void cg_finalize(const double* red, unsigned int nb, double* sh,
                                            double* sc, bool first) {
  for (int j = 0; j < DIM; ++j) {
    const double gamma = warp0_sum<T>(red + (2 * j) * nb, nb);
    const double delta = warp0_sum<T>(red + (2 * j + 1) * nb, nb);
    if (threadIdx.x == 0) {
      double alpha, beta;
      if (first) {
        beta = 0.0;
        alpha = delta != 0.0 ? gamma / delta : 0.0;
      } else {
        const double gp = sc[j], ap = sc[DIM + j];
        beta = gp != 0.0 ? gamma / gp : 0.0;
        const double den = ap != 0.0 ? delta - beta * gamma / ap : 0.0;
        alpha = den != 0.0 ? gamma / den : 0.0;
      }
      sc[j] = gamma;
      sc[DIM + j] = alpha;
      sc[2 * DIM + j] = beta;
    }
  }
}

// r0 = b = -v/Kbar, w0 = B D^{-1} r0; x = p = 0, s_{-1} = 0; alpha0 = gamma0/delta0
template <typename T, int DIM, int NLF>
__global__ void k_cg_init(int64_t nc, const double* __restrict__ v, double inv_kbar,
                          const T* __restrict__ diag, const T* __restrict__ invd,
                          const int32_t* __restrict__ col,
                          const T* __restrict__ off, T* __restrict__ r0, T* __restrict__ w0,
                          T* __restrict__ sm1, T* __restrict__ x, T* __restrict__ p, double* red,
                          unsigned int* count, double* sc) {
  __shared__ double sh[32];
  T pg[DIM], pd[DIM];  // per-thread partials in the vector precision
#pragma unroll
  for (int j = 0; j < DIM; ++j) pg[j] = pd[j] = (T)0;
  for (int64_t c = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; c < nc;
       c += (int64_t)gridDim.x * blockDim.x) {
    const T D = -diag[c], iD = invd[c];
    T u[DIM], w[DIM];
#pragma unroll
    for (int j = 0; j < DIM; ++j) {
      const T b = (T)(-v[j * nc + c] * inv_kbar);
      r0[j * nc + c] = b;
      u[j] = b * iD;
      w[j] = D * u[j];
      x[j * nc + c] = (T)0;
      p[j * nc + c] = (T)0;
      sm1[j * nc + c] = (T)0;
      pg[j] += b * u[j];
    }
#pragma unroll
    for (int lf = 0; lf < NLF; ++lf) {
      const int32_t nb = col[c * NLF + lf];
      if (nb < 0) continue;
      const T o = off[c * NLF + lf] * invd[nb];
#pragma unroll
      for (int j = 0; j < DIM; ++j) w[j] -= o * (T)(-v[j * nc + nb] * inv_kbar);
    }
#pragma unroll
    for (int j = 0; j < DIM; ++j) {
      w0[j * nc + c] = w[j];
      pd[j] += w[j] * u[j];
    }
  }
#pragma unroll
  for (int j = 0; j < DIM; ++j) {
    const double a = block_sum_t(pg[j], sh);
    const double b = block_sum_t(pd[j], sh);
    if (threadIdx.x == 0) {
      red[(2 * j) * gridDim.x + blockIdx.x] = a;
      red[(2 * j + 1) * gridDim.x + blockIdx.x] = b;
    }
  }
  if (last_block(count, gridDim.x)) {
    __threadfence();
    cg_finalize<T, DIM>(red, gridDim.x, sh, sc, true);
    if (threadIdx.x == 0) count[0] = 0;
  }
}

// iteration i: from r_{i-1}, w_{i-1}, s_{i-2} and alpha_{i-1}, beta_{i-1}:
//   s_{i-1} = w_{i-1} + beta s_{i-2};  r_i = r_{i-1} - alpha s_{i-1}
//   p_{i-1} = u_{i-1} + beta p_{i-2};  x += alpha p_{i-1}
//   w_i = B u_i, u_i = D^{-1} r_i;  partial (r_i, u_i), (w_i, u_i)
template <typename T, int DIM, int NLF>
__global__ void k_cg_iter(int64_t nc, const T* __restrict__ diag, const T* __restrict__ invd,
                          const int32_t* __restrict__ col,
                          const T* __restrict__ off, const T* __restrict__ r_old,
                          const T* __restrict__ w_old, const T* __restrict__ s_oldold,
                          T* __restrict__ r_new, T* __restrict__ w_new, T* __restrict__ s_new,
                          T* __restrict__ x, T* __restrict__ p, double* red, unsigned int* count,
                          double* sc) {
  __shared__ double sh[32];
  T alpha[DIM], beta[DIM];
  T pg[DIM], pd[DIM];  // per-thread partials in the vector precision
#pragma unroll
  for (int j = 0; j < DIM; ++j) {
    alpha[j] = (T)sc[DIM + j];
    beta[j] = (T)sc[2 * DIM + j];
    pg[j] = pd[j] = 0.0;
  }
  for (int64_t c = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; c < nc;
       c += (int64_t)gridDim.x * blockDim.x) {
    const T D = -diag[c], iD = invd[c];
    T un[DIM], w[DIM];
#pragma unroll
    for (int j = 0; j < DIM; ++j) {
      const int64_t i = j * nc + c;
      const T ro = r_old[i];
      const T s1 = w_old[i] + beta[j] * s_oldold[i];
      const T rn = ro - alpha[j] * s1;
      const T pp = ro * iD + beta[j] * p[i];
      p[i] = pp;
      x[i] += alpha[j] * pp;
      s_new[i] = s1;
      r_new[i] = rn;
      un[j] = rn * iD;
      w[j] = D * un[j];
      pg[j] += rn * un[j];
    }
#pragma unroll
    for (int lf = 0; lf < NLF; ++lf) {
      const int32_t nb = col[c * NLF + lf];
      if (nb < 0) continue;
      const T o = off[c * NLF + lf] * invd[nb];
#pragma unroll
      for (int j = 0; j < DIM; ++j) {
        const int64_t i = j * nc + nb;
        const T rn = r_old[i] - alpha[j] * (w_old[i] + beta[j] * s_oldold[i]);
        w[j] -= o * rn;
      }
    }
#pragma unroll
    for (int j = 0; j < DIM; ++j) {
      w_new[j * nc + c] = w[j];
      pd[j] += w[j] * un[j];
    }
  }
#pragma unroll
  for (int j = 0; j < DIM; ++j) {
    const double a = block_sum_t(pg[j], sh);
    const double b = block_sum_t(pd[j], sh);
    if (threadIdx.x == 0) {
      red[(2 * j) * gridDim.x + blockIdx.x] = a;
      red[(2 * j + 1) * gridDim.x + blockIdx.x] = b;
    }
  }
  if (last_block(count, gridDim.x)) {
    __threadfence();
    cg_finalize<T, DIM>(red, gridDim.x, sh, sc, false);
    if (threadIdx.x == 0) count[0] = 0;
  }
}

// z = x + alpha (u + beta p), u = D^{-1} r (the last step's update), in FP64
template <typename T, int DIM>
__global__ void k_cg_finish(int64_t nc, const T* __restrict__ invd, const T* __restrict__ r,
                            const T* __restrict__ x, const T* __restrict__ p,
                            const double* __restrict__ sc, double* __restrict__ z) {
  const int64_t c = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (c >= nc) return;
  const T iD = invd[c];
#pragma unroll
  for (int j = 0; j < DIM; ++j) {
    const int64_t i = j * nc + c;
    const T alpha = (T)sc[DIM + j], beta = (T)sc[2 * DIM + j];
    z[i] = (double)(x[i] + alpha * (r[i] * iD + beta * p[i]));
  }
}

// ---------------------------------------------------------------------
// The same iteration in one persistent cooperative launch: the blocks are
// co-resident (cudaLaunchCooperativeKernel) and meet at one grid barrier
// per iteration, after which every block forms the scalars from the
// per-block partial sums in the same fixed order.  The barrier's spin is
// bounded: on time-out the kernel sets an error flag and returns, and the
// host reports the error at its next synchronisation.
//
// An iteration touches a few hundred bytes a cell, all of it in L2 (or
// registers), so its time is latency: the barrier, the reductions and the
// gathers, 16 us an iteration on 32^2 quads and 24 us on 45^3 hexes when each
// of these was a chain.  Hence:
//  * One block of 1024 cells each, no more blocks than the cells need: 32^2
//    quads run in one block and meet at its own barrier.
//  * The 2 DIM inner products go together: interleaved shuffles, then one
//    warp each for the sum over the warps and for the sum over the blocks.
//  * Blocks wait on the arrivals themselves, without a sleep.
//  * A cell's r, w and s are one vector load each for its neighbours; with a
//    cell a thread (RES: at most 1024 cells a block and SM) its own values,
//    its row of the matrix and x, p stay in registers.
//  * In RES a neighbour of the same block is read as its new r from shared
//    memory, after one more block barrier; only the others' r, w and s go
//    through L2, and only cells that another block reads are stored there
//    (45^3 hexes, 30 iterations: 293 -> 272 us).
//  * In FP32 alpha needs no quotient of the previous alpha: beta gamma /
//    alpha_prev = beta^2 (delta - ...)_prev, gamma / beta = gamma_prev; the
//    scalars are doubles, so the roundings are far below the vectors'.  FP64
//    keeps the quotients: 1 / gamma overflows where gamma is a subnormal number.
// The sums keep their order (a warp's cells by shuffles in T, warps of 1024
// cells in double, blocks in T), whatever the number of blocks.
// ---------------------------------------------------------------------
constexpr unsigned int kBarrierSpinLimit = 1u << 22;  // polls of an L2 word, ~0.3 us each: ~1 s

struct GridBarrier {
  unsigned int* count;  // arrivals since the launch began
  unsigned int* done;   // blocks that finished (the last one clears both)
  int* err;
};

// Whether an earlier launch's wait ran out and the host has not cleared the
// flag yet: its counters are then not those of a new launch.  Thread 0 reads
// it when the kernel begins and hands it to the barriers.
__device__ __forceinline__ bool barrier_failed(const GridBarrier& gb) {
  return threadIdx.x == 0 && *(volatile int*)gb.err != 0;
}

// Arrive, and wait until `target` arrivals have been counted since the
// launch began.  Returns false (the same for the whole block) when the wait
// ran out, another block's did, or an earlier launch's had (failed).
__device__ __forceinline__ bool grid_barrier(const GridBarrier& gb, unsigned int target, bool failed,
                                             unsigned int spin_limit = kBarrierSpinLimit) {
  __shared__ int s_ok;
  __syncthreads();
  if (threadIdx.x == 0) {
    int ok = !failed;
    if (ok) {
      __threadfence();
      atomicAdd(gb.count, 1u);
      unsigned int spins = 0, now;
      for (;;) {
        asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(now) : "l"(gb.count) : "memory");
        if (now >= target) break;
        if (++spins > spin_limit || ((spins & 1023u) == 0 && *(volatile int*)gb.err)) {
          ok = 0;
          break;
        }
      }
    }
    if (!ok) atomicExch(gb.err, 1);
    __threadfence();
    s_ok = ok;
  }
  __syncthreads();
  return s_ok != 0;
}

// end of a launch whose blocks met at grid_barrier: the last block to get
// here clears the counters for the next one
__device__ __forceinline__ void grid_barrier_leave(const GridBarrier& gb) {
  if (threadIdx.x == 0) {
    __threadfence();
    if (atomicAdd(gb.done, 1u) == gridDim.x - 1) {
      atomicExch(gb.count, 0u);
      atomicExch(gb.done, 0u);
    }
  }
}

// a product rounded by itself: where a sum of two products could be fused
// either way, the order of rounding is written out
__device__ __forceinline__ float mul_rn(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ double mul_rn(double a, double b) { return __dmul_rn(a, b); }

// a cell's DIM values as one (DIM = 2, or float) or two vector accesses, past
// L1: other SMs write them between barriers
template <typename T, int DIM>
struct CellVec {
  static constexpr int N = DIM == 2 ? 2 : 4;  // elements a cell
  static __device__ __forceinline__ void ld(const T* a, int64_t c, T (&v)[DIM]) {
    if constexpr (sizeof(T) == 4 && DIM == 2) {
      const float2 x = __ldcg(reinterpret_cast<const float2*>(a) + c);
      v[0] = x.x, v[1] = x.y;
    } else if constexpr (sizeof(T) == 4) {
      const float4 x = __ldcg(reinterpret_cast<const float4*>(a) + c);
      v[0] = x.x, v[1] = x.y, v[2] = x.z;
    } else {
      const double2 x = __ldcg(reinterpret_cast<const double2*>(a + c * N));
      v[0] = x.x, v[1] = x.y;
      if constexpr (DIM == 3) v[2] = __ldcg(a + c * N + 2);
    }
  }
  static __device__ __forceinline__ void st(T* a, int64_t c, const T (&v)[DIM]) {
    if constexpr (sizeof(T) == 4 && DIM == 2) {
      __stcg(reinterpret_cast<float2*>(a) + c, make_float2(v[0], v[1]));
    } else if constexpr (sizeof(T) == 4) {
      __stcg(reinterpret_cast<float4*>(a) + c, make_float4(v[0], v[1], v[2], 0.f));
    } else {
      __stcg(reinterpret_cast<double2*>(a + c * N), make_double2(v[0], v[1]));
      if constexpr (DIM == 3) __stcg(a + c * N + 2, v[2]);
    }
  }
};

constexpr int kPersistThreads = 1024;
constexpr int kPersistWarps = kPersistThreads / 32;

// rwork: r, w, s of even and odd iterations, CellVec::N * nc elements each;
// xwork: x and p, DIM * nc each (not RES)
template <typename T, int DIM, int NLF, bool RES>
__global__ void __launch_bounds__(kPersistThreads)
    k_cg_persist(int64_t nc, int iters, const double* __restrict__ v, double inv_kbar,
                 const T* __restrict__ diag, const T* __restrict__ invd,
                 const int32_t* __restrict__ col, const T* __restrict__ off, T* rwork, T* xwork,
                 double* part, GridBarrier gb, double* __restrict__ zout) {
  using CV = CellVec<T, DIM>;
  constexpr int NS = 2 * DIM;              // inner products: gamma_j, delta_j interleaved
  __shared__ double sh[NS][kPersistWarps];
  __shared__ double s_sum[NS];
  __shared__ T s_ab[2 * DIM];              // alpha, beta in the vector precision
  const unsigned int nb = gridDim.x;
  const bool failed = nb > 1 && barrier_failed(gb);
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const int64_t nv = CV::N * nc;
  T* r[2] = {rwork, rwork + nv};
  T* w[2] = {rwork + 2 * nv, rwork + 3 * nv};
  T* s[2] = {rwork + 4 * nv, rwork + 5 * nv};
  T* xa = xwork;
  T* pa = xwork + (RES ? 0 : DIM * nc);
  const int64_t c0 = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  const int64_t cstep = (int64_t)gridDim.x * blockDim.x;
  T pg[DIM], pd[DIM];  // per-thread partials in the vector precision
  // threads j < DIM: 1 / gamma, gamma, denominator and alpha of the last iteration
  double inv_gp = 0.0, gamma_p = 0.0, den_p = 0.0, alpha_p = 0.0;
  // the thread's cell (RES): its row of the matrix and its vectors; a
  // neighbour of the same block is an index into rs, another's is global
  constexpr bool ROW = RES && NLF <= 6;    // the row fits in registers
  __shared__ T rs[RES ? DIM * kPersistThreads : 1];  // the block's new r
  T rD = 0, riD = 0, ro_r[DIM], wo_r[DIM], so_r[DIM], xr[DIM], pr[DIM], row_o[ROW ? NLF : 1];
  int32_t row_c[ROW ? NLF : 1];
  const int32_t cb = (int32_t)(blockIdx.x * (int64_t)blockDim.x);  // the block's first cell (RES)
  bool seen = !RES;                        // another block reads this cell
  // ---- iteration 0: r0 = b, w0 = B D^-1 r0, x = p = 0, s_{-1} = 0
#pragma unroll
  for (int j = 0; j < DIM; ++j) {
    pg[j] = pd[j] = (T)0;
    ro_r[j] = wo_r[j] = so_r[j] = xr[j] = pr[j] = (T)0;
  }
  for (int64_t c = c0; c < nc; c += cstep) {
    const T D = -diag[c], iD = invd[c];
    T u[DIM], ww[DIM], bb[DIM];
#pragma unroll
    for (int j = 0; j < DIM; ++j) {
      const T b = (T)(-v[j * nc + c] * inv_kbar);
      bb[j] = b;
      u[j] = mul_rn(b, iD);
      ww[j] = mul_rn(D, u[j]);
      pg[j] = fma(b, u[j], pg[j]);
    }
#pragma unroll
    for (int lf = 0; lf < NLF; ++lf) {
      const int32_t n2 = col[c * NLF + lf];
      if (ROW) row_c[lf] = n2;
      if (n2 < 0) continue;
      const T o = mul_rn(off[c * NLF + lf], invd[n2]);
      if (ROW) row_o[lf] = o;
      if (RES) seen |= (uint32_t)(n2 - cb) >= (uint32_t)kPersistThreads;
#pragma unroll
      for (int j = 0; j < DIM; ++j) ww[j] = fma(-o, (T)(-v[j * nc + n2] * inv_kbar), ww[j]);
    }
    if (seen) {
      const T zero[DIM] = {};
      CV::st(r[0], c, bb);
      CV::st(w[0], c, ww);
      CV::st(s[1], c, zero);
    }
#pragma unroll
    for (int j = 0; j < DIM; ++j) {
      pd[j] = fma(ww[j], u[j], pd[j]);
      if (RES) {
        ro_r[j] = bb[j];
        wo_r[j] = ww[j];
      } else {
        xa[j * nc + c] = (T)0;
        pa[j * nc + c] = (T)0;
      }
    }
    if (RES) rD = D, riD = iD;
  }
  for (int it = 0; it < iters; ++it) {
    // the block's sums: a warp's cells by shuffles in T, its warps in double
    T q[NS];
#pragma unroll
    for (int j = 0; j < DIM; ++j) q[2 * j] = pg[j], q[2 * j + 1] = pd[j];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1)
#pragma unroll
      for (int k = 0; k < NS; ++k) q[k] += __shfl_xor_sync(0xffffffffu, q[k], o);
    if (lane == 0) {
#pragma unroll
      for (int k = 0; k < NS; ++k) sh[k][wid] = (double)q[k];
    }
    __syncthreads();
    double* pp = part + (int64_t)(it & 1) * NS * nb;  // [2j (+1)][block], by parity
    if (wid < NS) {
      double t = sh[wid][lane];
      for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
      if (lane == 0) {
        if (nb == 1) s_sum[wid] = (double)(T)t;
        else __stcg(pp + wid * nb + blockIdx.x, t);
      }
    }
    if (nb == 1) {
      __syncthreads();
    } else {
      if (!grid_barrier(gb, (unsigned int)(it + 1) * nb, failed)) return;
      if (wid < NS) {  // every block forms the same sums in the same order
        T t = (T)0;
#pragma unroll 5
        for (unsigned int b = lane; b < nb; b += 32) t += (T)__ldcg(pp + wid * nb + b);
        for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
        if (lane == 0) s_sum[wid] = (double)t;
      }
      __syncthreads();
    }
    if (threadIdx.x < DIM) {
      const int j = threadIdx.x;
      const double gamma = s_sum[2 * j], delta = s_sum[2 * j + 1];
      double beta, den;
      if constexpr (sizeof(T) == 8) {  // the quotients themselves
        beta = gamma_p != 0.0 ? gamma / gamma_p : 0.0;  // 0 in the first iteration
        den = it == 0 ? delta : alpha_p != 0.0 ? delta - beta * gamma / alpha_p : 0.0;
        gamma_p = gamma;
      } else {
        beta = gamma * inv_gp;
        den = it == 0 ? delta : alpha_p != 0.0 ? fma(-(beta * beta), den_p, delta) : 0.0;
        den_p = den;
      }
      const double alpha = den != 0.0 ? gamma / den : 0.0;
      alpha_p = alpha;
      s_ab[j] = (T)alpha;
      s_ab[DIM + j] = (T)beta;
    }
    __syncthreads();
    // the next beta's divisor, while the other warps go on
    if (sizeof(T) == 4 && threadIdx.x < DIM) {
      const double gamma = s_sum[2 * threadIdx.x];
      inv_gp = gamma != 0.0 ? 1.0 / gamma : 0.0;
    }
    T alpha[DIM], beta[DIM];
#pragma unroll
    for (int j = 0; j < DIM; ++j) {
      alpha[j] = s_ab[j];
      beta[j] = s_ab[DIM + j];
    }
    const int i = it + 1;  // the iteration this pass computes
    const T* ro_ = r[(i - 1) & 1];
    const T* wo_ = w[(i - 1) & 1];
    const T* so_ = s[i & 1];
    if (i == iters) {
      // last step: z = x + alpha (u + beta p), u = D^-1 r
      for (int64_t c = c0; c < nc; c += cstep) {
        const T iD = RES ? riD : invd[c];
        T ro[DIM];
        if (RES) {
#pragma unroll
          for (int j = 0; j < DIM; ++j) ro[j] = ro_r[j];
        } else {
          CV::ld(ro_, c, ro);
        }
#pragma unroll
        for (int j = 0; j < DIM; ++j) {
          const T x = RES ? xr[j] : xa[j * nc + c], p = RES ? pr[j] : pa[j * nc + c];
          zout[j * nc + c] = (double)fma(alpha[j], fma(ro[j], iD, mul_rn(beta[j], p)), x);
        }
      }
      if (nb > 1) grid_barrier_leave(gb);
      return;
    }
    T* rn_ = r[i & 1];
    T* wn_ = w[i & 1];
    T* sn_ = s[(i - 1) & 1];
#pragma unroll
    for (int j = 0; j < DIM; ++j) pg[j] = pd[j] = (T)0;
    if constexpr (RES) {
      T ww[DIM], un[DIM];
      if (c0 < nc) {
        T rn[DIM], s1[DIM];
#pragma unroll
        for (int j = 0; j < DIM; ++j) {
          s1[j] = fma(beta[j], so_r[j], wo_r[j]);
          rn[j] = fma(-alpha[j], s1[j], ro_r[j]);
          pr[j] = fma(ro_r[j], riD, mul_rn(beta[j], pr[j]));
          xr[j] = fma(alpha[j], pr[j], xr[j]);
          un[j] = mul_rn(rn[j], riD);
          ww[j] = mul_rn(rD, un[j]);
          pg[j] = fma(rn[j], un[j], pg[j]);
          rs[j * kPersistThreads + threadIdx.x] = rn[j];
          ro_r[j] = rn[j];
          so_r[j] = s1[j];
        }
        if (seen) {
          CV::st(sn_, c0, s1);
          CV::st(rn_, c0, rn);
        }
      }
      __syncthreads();
      if (c0 < nc) {
#pragma unroll
        for (int lf = 0; lf < NLF; ++lf) {
          const int32_t n2 = ROW ? row_c[ROW ? lf : 0] : col[c0 * NLF + lf];
          if (n2 < 0) continue;
          const T o = ROW ? row_o[ROW ? lf : 0] : mul_rn(off[c0 * NLF + lf], invd[n2]);
          T rb[DIM];
          const uint32_t k = (uint32_t)(n2 - cb);
          if (k < (uint32_t)kPersistThreads) {
#pragma unroll
            for (int j = 0; j < DIM; ++j) rb[j] = rs[j * kPersistThreads + k];
          } else {
            T wb[DIM], sb[DIM];
            CV::ld(ro_, n2, rb);
            CV::ld(wo_, n2, wb);
            CV::ld(so_, n2, sb);
#pragma unroll
            for (int j = 0; j < DIM; ++j) rb[j] = fma(-alpha[j], fma(beta[j], sb[j], wb[j]), rb[j]);
          }
#pragma unroll
          for (int j = 0; j < DIM; ++j) ww[j] = fma(-o, rb[j], ww[j]);
        }
        if (seen) CV::st(wn_, c0, ww);
#pragma unroll
        for (int j = 0; j < DIM; ++j) {
          pd[j] = fma(ww[j], un[j], pd[j]);
          wo_r[j] = ww[j];
        }
      }
    } else {
      for (int64_t c = c0; c < nc; c += cstep) {
        const T D = -diag[c], iD = invd[c];
        T ro[DIM], wo[DIM], so[DIM], rn[DIM], s1[DIM], un[DIM], ww[DIM];
        CV::ld(ro_, c, ro);
        CV::ld(wo_, c, wo);
        CV::ld(so_, c, so);
#pragma unroll
        for (int j = 0; j < DIM; ++j) {
          s1[j] = fma(beta[j], so[j], wo[j]);
          rn[j] = fma(-alpha[j], s1[j], ro[j]);
          const T pv = fma(ro[j], iD, mul_rn(beta[j], pa[j * nc + c]));
          pa[j * nc + c] = pv;
          xa[j * nc + c] = fma(alpha[j], pv, xa[j * nc + c]);
          un[j] = mul_rn(rn[j], iD);
          ww[j] = mul_rn(D, un[j]);
          pg[j] = fma(rn[j], un[j], pg[j]);
        }
        CV::st(sn_, c, s1);
        CV::st(rn_, c, rn);
#pragma unroll
        for (int lf = 0; lf < NLF; ++lf) {
          const int32_t n2 = col[c * NLF + lf];
          if (n2 < 0) continue;
          const T o = mul_rn(off[c * NLF + lf], invd[n2]);
          T rb[DIM], wb[DIM], sb[DIM];
          CV::ld(ro_, n2, rb);
          CV::ld(wo_, n2, wb);
          CV::ld(so_, n2, sb);
#pragma unroll
          for (int j = 0; j < DIM; ++j)
            ww[j] = fma(-o, fma(-alpha[j], fma(beta[j], sb[j], wb[j]), rb[j]), ww[j]);
        }
        CV::st(wn_, c, ww);
#pragma unroll
        for (int j = 0; j < DIM; ++j) pd[j] = fma(ww[j], un[j], pd[j]);
      }
    }
  }
}

template <typename T, int DIM, int NLF, bool RES>
static bool cg_persist_launch(hofv_ctx* c, const T* diag, const T* invd, const T* off, T* work,
                              int iters, const double* v, double* zout) {
  static int mb = -1;  // co-resident blocks of this instantiation, found once
  if (mb < 0) {
    int per_sm = 0, dev = 0, nsm = 0, coop = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, dev);
    cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
    if (!coop ||
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_cg_persist<T, DIM, NLF, RES>,
                                                      kPersistThreads, 0) != cudaSuccess)
      per_sm = 0;
    int blocks = std::min(per_sm, 1) * nsm;
    const char* env = getenv("HOFV_CG_PERSISTENT");
    if (env && env[0] == '0') blocks = 0;
    mb = blocks;
  }
  if (mb <= 0 || !c->d_bar) return false;
  int64_t nc = c->nc;
  const int64_t need = (nc + kPersistThreads - 1) / kPersistThreads;
  if (RES && need > mb) return false;
  const unsigned int nb = (unsigned int)std::min<int64_t>(need, mb);
  int iters_ = std::max(iters, 1);
  double inv_kbar = 1.0 / c->mat.kbar;
  T* rwork = work;
  T* xwork = work + 6 * CellVec<T, DIM>::N * nc;
  double* part = c->d_red;
  GridBarrier gb{c->d_bar, c->d_bar + 1, reinterpret_cast<int*>(c->d_bar + 2)};
  void* args[] = {&nc, &iters_, (void*)&v, &inv_kbar, (void*)&diag, (void*)&invd,
                  (void*)&c->d_aj_col, (void*)&off, &rwork, &xwork, &part, &gb, &zout};
  const cudaError_t e = cudaLaunchCooperativeKernel((const void*)k_cg_persist<T, DIM, NLF, RES>,
                                                    dim3(nb), dim3(kPersistThreads), args, 0,
                                                    c->stream);
  if (e != cudaSuccess) {
    cudaGetLastError();
    return false;
  }
  return true;
}

template <typename T, int DIM, int NLF>
static bool cg_persist_run(hofv_ctx* c, const T* diag, const T* invd, const T* off, T* work,
                           int iters, const double* v, double* zout) {
  // a cell a thread where one block an SM has threads for all cells (doubles
  // do not fit the 64 registers of 1024 threads)
  if constexpr (sizeof(T) == 4) {
    if (c->nc <= (int64_t)kPersistThreads * c->sm_count &&
        cg_persist_launch<T, DIM, NLF, true>(c, diag, invd, off, work, iters, v, zout))
      return true;
  }
  return cg_persist_launch<T, DIM, NLF, false>(c, diag, invd, off, work, iters, v, zout);
}

template <typename T, int DIM, int NLF>
static void cg_run(hofv_ctx* c, const T* diag, const T* invd, const T* off, T* work, int iters,
                   const double* v, double* zout) {
  const int64_t nc = c->nc, n = DIM * nc;
  T* x = work;
  T* p = work + n;
  T* r[2] = {work + 2 * n, work + 3 * n};
  T* w[2] = {work + 4 * n, work + 5 * n};
  T* s[2] = {work + 6 * n, work + 7 * n};
  const int blocks = c->red_blocks;
  double* red = c->d_red;
  unsigned int* cnt = c->d_count;
  double* sc = c->d_scal + 32;  // slots 32..40
  cudaStream_t st = c->stream;
  if (iters < 1) iters = 1;
  k_cg_init<T, DIM, NLF><<<blocks, kRedThreads, 0, st>>>(nc, v, 1.0 / c->mat.kbar, diag, invd, c->d_aj_col,
                                                   off, r[0], w[0], s[1], x, p, red, cnt, sc);
  for (int i = 1; i < iters; ++i)
    k_cg_iter<T, DIM, NLF><<<blocks, kRedThreads, 0, st>>>(nc, diag, invd, c->d_aj_col, off, r[(i - 1) & 1],
                                                     w[(i - 1) & 1], s[i & 1], r[i & 1], w[i & 1],
                                                     s[(i - 1) & 1], x, p, red, cnt, sc);
  k_cg_finish<T, DIM><<<(unsigned)((nc + 255) / 256), 256, 0, st>>>(nc, invd, r[(iters - 1) & 1], x,
                                                                     p, sc, zout);
}

// Two co-resident blocks at a barrier.  With extra = 1 it expects one more
// arrival than exists: the wait must run out and latch the error flag.
__global__ void k_barrier_probe(GridBarrier gb, unsigned int extra, unsigned int spin_limit, unsigned int* passed) {
  const bool failed = barrier_failed(gb);
  // the count stays: the host clears it
  if (grid_barrier(gb, gridDim.x + extra, failed, spin_limit) && threadIdx.x == 0) atomicExch(passed, 1u);
}

// A wait that runs out, and behind it, before the host looks, a launch whose
// arrivals are already counted: neither may pass.
int barrier_selftest(hofv_ctx* c, int* timed_out) {
  *timed_out = 0;
  if (!c->d_bar) return fail(c, HOFV_ESTATE, "hofv_build_stencils must come first");
  GridBarrier gb{c->d_bar, c->d_bar + 1, reinterpret_cast<int*>(c->d_bar + 2)};
  unsigned int limit = 1u << 14, extra;
  unsigned int* passed = c->d_bar + 3;
  void* args[] = {&gb, &extra, &limit, &passed};
  for (unsigned int e : {1u, 0u}) {
    extra = e;
    HOFV_CUDA(c, cudaLaunchCooperativeKernel((const void*)k_barrier_probe, dim3(2), dim3(32), args, 0,
                                             c->stream));
  }
  HOFV_CUDA(c, cudaStreamSynchronize(c->stream));
  int flags[2] = {0, 0};  // the error flag, and `passed`
  HOFV_CUDA(c, cudaMemcpy(flags, c->d_bar + 2, sizeof(flags), cudaMemcpyDeviceToHost));
  *timed_out = flags[0] != 0 && flags[1] == 0;
  HOFV_CUDA(c, cudaMemset(c->d_bar, 0, 4 * sizeof(unsigned int)));
  return 0;
}

// the persistent cooperative solve when it fits on the device, else one
// launch per iteration; NLF = faces per cell (4 / 6 for quads / hexes,
// 3 / 4 for triangles / tetrahedra, 8 slots for polygons, 16 for polyhedra)
template <typename T, int DIM, int NLF>
static void aj_run(hofv_ctx* c, const T* diag, const T* invd, const T* off, T* work, int iters,
                   const double* v, double* z) {
  if (!cg_persist_run<T, DIM, NLF>(c, diag, invd, off, work, iters, v, z))
    cg_run<T, DIM, NLF>(c, diag, invd, off, work, iters, v, z);
}

template <typename T>
static void aj_dispatch(hofv_ctx* c, const T* diag, const T* invd, const T* off, T* work, int iters,
                        const double* v, double* z) {
  const bool simplex = c->nlf == c->dim + 1;
  if (c->dim == 2) {
    if (simplex) aj_run<T, 2, 3>(c, diag, invd, off, work, iters, v, z);
    else if (c->poly) aj_run<T, 2, kPolyMaxSides>(c, diag, invd, off, work, iters, v, z);
    else aj_run<T, 2, 4>(c, diag, invd, off, work, iters, v, z);
  } else {
    if (simplex) aj_run<T, 3, 4>(c, diag, invd, off, work, iters, v, z);
    else if (c->polyh) aj_run<T, 3, kPolyhedronMaxFaces>(c, diag, invd, off, work, iters, v, z);
    else aj_run<T, 3, 6>(c, diag, invd, off, work, iters, v, z);
  }
}

int aj_precondition(hofv_ctx* c, int kind, int iters, const double* v, double* z) {
  if (c->nlf != 2 * c->dim && c->nlf != c->dim + 1 && !(c->poly && c->nlf == kPolyMaxSides) &&
      !(c->polyh && c->nlf == kPolyhedronMaxFaces))
    return fail(c, HOFV_ENOTSUP, "cell shape without an approximate-Jacobian kernel");
  if (kind == HOFV_PC_AJ64)
    aj_dispatch<double>(c, c->d_aj_diag, c->d_aj_invd, c->d_aj_off, c->d_cg64, iters, v, z);
  else
    aj_dispatch<float>(c, c->d_aj_diag32, c->d_aj_invd32, c->d_aj_off32, c->d_cg32, iters, v, z);
  HOFV_CUDA(c, cudaGetLastError());
  return 0;
}

}  // namespace hofv
