// residual.cu -- the matrix-free residual R(u) of the high-order
// cell-centred finite-volume scheme (arXiv 2601.18417):
//
//   k_ustar : cell-ordered; extrapolated face values of the alpha
//             stabilisation, u*_{f,P} = u_P + sum_N e_N u_N (eq. alphaJump,
//             App. B, with the Taylor terms folded into e at set-up)
//   k_flux  : face-ordered, 32 faces per tile; (1) displacement gradient at
//             every Gauss point, grad u = sum_N c_N (x) u_N (+ ghost node,
//             eq. faceQuadGrad), (2) the law (App. A) and traction T a_q,
//             (3) Gauss quadrature over the face plus the stabilisation
//             traction alpha Kbar / |d.n| (u*_N - u*_P) Gamma (eq. alpha)
//   k_cell  : cell-ordered, fixed face order (no atomics):
//             R_P = sum_f +-flux_f + source_P (eq. divStressDiscret +
//             eq. bodyTerm); optional epilogue (R - R0) / eps for Jv.
//   k_tflux : the linear law in contracted form, flux_f = sum_N T_N u_N
//             (replaces k_flux when enabled)
//   k_extend, k_sym_other : symmetry faces (reflected ghost values, mirrored
//             stabilisation value), only when the mesh has symmetry faces
//   k_cell_avg : inertia term of the BDF2 dynamics, only when enabled
//
// Operands and results are FP64; the contractions over the stencils are formed
// in fixed point where that is as exact as FP64 FMAs, whose rate does not bound
// it, by those FMAs elsewhere or, on request, in double-float arithmetic.  A tile's (face, row) pairs are laid
// out so that consecutive threads own consecutive coefficient rows.
#include <algorithm>
#include <type_traits>

#include "fixed_point.cuh"
#include "hofv_internal.cuh"

namespace hofv {

// ---------------------------------------------------------------------
// Fixed-point contraction of FP64 coefficients with FP64 values (the
// arithmetic of HOFV_PREC_FP64; fixed_point.cuh).
//
// GB300 issues 2 FP64 FMAs a clock and SM, a fraction of what one coefficient
// a product needs at HBM speed, but many times that of 32 x 32 -> 64 bit
// integer multiply-adds.  So a sum sum_N c_N u_N is formed exactly but for
// the representation of its operands: the coefficients of a row as integers
// of 59 bits in units of 2^-59 of a power of two 2^e, the values of a stencil
// as integers of 55 bits in units of 2^-55 of their largest binade, both rounded
// and each as two limbs; the products of the high limbs and of the high with
// the low ones are summed without rounding in 64 bits, and the sum is rounded
// once.  Left out are the products of the low limbs (zero on average, the value's
// low limb being signed).  2^e is above each coefficient, and sum |c_N| <= 15 2^e;
// with that, |U1| <= 2^27, |U0| <= 2^27, |C0| <= 2^28 and kMaxS = 128 slots both sums
// stay below 2^63.
//
// The error of that scales with the largest coefficient times the largest value,
// the error of FMAs with the partial sums.  Where the products are all small
// against those maxima (one value among zeros, a far cell's large value, a
// field falling by ten a cell) FMAs are the more accurate, and they are taken
// then: a row's sum is left in fixed point only if some of its products, the nearest
// cells' among them, add up to 2^-4 (2-D) or 2^-5 (3-D) of 2^e times the values'
// binade (fx_sure, fx_row).
// Errors of this rule and of FMAs alone over sum |c_N u_N|, rms over the gradient
// rows of jittered p = 3 hexes (quads), and the rows left in fixed point:
//   smooth field         1.7e-17 and 1.5e-16 (1.3e-17 and 5.6e-17)   all
//   random values        1.8e-17 and 1.3e-16 (3.4e-17 and 1.1e-16)   all (99 %)
//   zero across the face 2.0e-17 and 1.6e-16 (3.2e-17 and 1.2e-16)   all (98.9 %)
//   falling by e a cell  4.2e-17 and 9.2e-17 (4.1e-17 and 6.1e-17)   99.9 % (85 %)
//   falling by 10 a cell 9.2e-17 and 1.0e-16 (5.7e-17 and 6.5e-17)   28 % (8 %)
//   one value            4.6e-17 and 4.6e-17 (4.7e-17 and 4.7e-17)   6 % (9 %)
//
// What bounds it: integer issue.  A coefficient takes about 17 instructions to
// split and, for three components, nine multiply-adds at 32 a clock and SM (209
// of the 494 us on 32^3 hexes; the bytes take 257).  Measured on smooth fields,
// FP64 FMAs alone -> this (without the check and the way to FMAs), us: k_flux 32^3
// hexes p = 3 neo-Hookean 1427 -> 494 (475), 12^3 45 (41), 20^3 151 (132: one row's
// FMAs), 40^3 p = 2 1077 -> 385 (355), 2 255^2 triangles 110 -> 81 (76), 20-layer
// prisms 1104 -> 426 (390), 6 17^3 tetrahedra 272 -> 132 (119); k_ustar 32^3 hexes
// 107 -> 73 (65), 40^3 148 -> 106 (97), 512^2 quads 83 -> 68 (65).  A state that takes
// nearly all rows to FMAs (values spread over 2^40): k_flux 1326, 937, 134, 982, 298
// (32^3, 40^3, triangles, prisms, tetrahedra), k_ustar 122, 178, 103.  Strides known to
// the compiler and a loop without range checks gave 666 -> 497 of the first when
// nothing was checked.  Not kept: every 5th slot by FP64 FMAs beside the others (515
// for 467), two of five (682); the FMAs behind a barrier (516 for 499) or inlined (504);
// a lone row's FMAs with a lane a slot, or its operands loaded ahead (no gain); the
// second look out of line (a state spread over 2^40: 2053 for 1326); the limbs cut from
// one 64-bit integer (684).
//
// Rows and stencils whose largest binade lies outside [kFxMin, kFxMax] (tiny,
// huge, infinite or NaN values) are summed by FP64 FMAs too.
// ---------------------------------------------------------------------
// the exponent that scales each coefficient row of [tile][S][cs]
__global__ void k_row_exponents(const double* __restrict__ a, int S, int cs, int64_t n,
                                uint16_t* __restrict__ out) {
  const int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;  // (tile, row)
  if (e >= n) return;
  const double* __restrict__ p = a + e / cs * S * cs + e % cs;
  int mx = 0;
  bool zero = true;
  double sum = 0.0;
  for (int k = 0; k < S; ++k) {
    const double v = p[(int64_t)k * cs];
    zero &= v == 0.0;
    mx = max(mx, (__double2hiint(v) >> 20) & 0x7ff);
    sum += fabs(v);
  }
  out[e] = fx_row_exponent(mx, zero, sum);
}

void launch_row_exponents(const double* a, int S, int cs, int64_t tiles, uint16_t* out, cudaStream_t st) {
  const int64_t n = tiles * cs;
  if (n > 0) k_row_exponents<<<(unsigned)((n + 255) / 256), 256, 0, st>>>(a, S, cs, n, out);
}

// The values at the stencils of `items` consecutive faces or cells (item0 the
// first) as limbs in shared memory, ua[n * STRIDE + k] components 0 and 1 and
// ub component 2 of slot n of item k, and each item's exponents in ex (0 where
// the item is to be summed by FMAs).  Called by the whole block.
template <int DIM, int THREADS, int STRIDE>
__device__ __forceinline__ void fx_gather(const int32_t* __restrict__ sten, const double* __restrict__ w,
                                          int64_t ws, int S, int64_t item0, int items, int4* ua, int2* ub,
                                          int* ex) {
  constexpr int U = 4, stride = STRIDE, step = THREADS / STRIDE;
  const int k = threadIdx.x % stride, s0 = threadIdx.x / stride;
  const bool on = k < items && s0 < step;
  const int64_t g = item0 + k;
  const int32_t* __restrict__ st = sten + g / kTile * (int64_t)S * kTile + g % kTile;
  for (int i = threadIdx.x; i < stride * DIM; i += THREADS) ex[i] = 0;
  __syncthreads();
  if (on) {
    int mx[DIM];
#pragma unroll
    for (int j = 0; j < DIM; ++j) mx[j] = 0;
    for (int n0 = s0; n0 < S; n0 += U * step) {
      int32_t id[U];  // the cells first: one wait for their list, one for their values
#pragma unroll
      for (int d = 0; d < U; ++d) id[d] = n0 + d * step < S ? __ldg(st + (n0 + d * step) * kTile) : 0;
      double v[U][DIM];
#pragma unroll
      for (int d = 0; d < U; ++d)
#pragma unroll
        for (int j = 0; j < DIM; ++j) v[d][j] = __ldg(w + j * ws + id[d]);
#pragma unroll
      for (int d = 0; d < U; ++d) {
        const int n = n0 + d * step;
        if (n >= S) break;
        int h[DIM], l[DIM];
#pragma unroll
        for (int j = 0; j < DIM; ++j) {
          h[j] = __double2hiint(v[d][j]);
          l[j] = __double2loint(v[d][j]);
          mx[j] = max(mx[j], (h[j] & 0x7fffffff) | (l[j] != 0));
        }
        ua[n * stride + k] = make_int4(h[0], l[0], h[1], l[1]);
        if constexpr (DIM == 3) ub[n * stride + k] = make_int2(h[2], l[2]);
      }
    }
#pragma unroll
    for (int j = 0; j < DIM; ++j) atomicMax(ex + k * DIM + j, mx[j]);
  }
  __syncthreads();
  int E[DIM];
  bool fx = true;
  if (on) {
#pragma unroll
    for (int j = 0; j < DIM; ++j) {
      const int key = ex[k * DIM + j];
      E[j] = key >> 20;
      fx &= key == 0 || (E[j] >= kFxMin && E[j] <= kFxMax);
      if (key == 0) E[j] = kFxZero;
    }
  }
  __syncthreads();
  if (on) {
    if (s0 == 0) {
#pragma unroll
      for (int j = 0; j < DIM; ++j) ex[k * DIM + j] = fx ? E[j] : 0;
    }
    if (fx)
      for (int n = s0; n < S; n += step) {  // a thread converts what it stored
        const int4 a = ua[n * stride + k];
        const FxLimbs x = fx_value(a.x, a.y, E[0]), y = fx_value(a.z, a.w, E[1]);
        ua[n * stride + k] = make_int4(x.hi, x.lo, y.hi, y.lo);
        if constexpr (DIM == 3) {
          const int2 b = ub[n * stride + k];
          const FxLimbs z = fx_value(b.x, b.y, E[2]);
          ub[n * stride + k] = make_int2(z.hi, z.lo);
        }
      }
  }
  __syncthreads();
}

// Streams the S coefficients of the row co (CS between slots) as limbs to
// mac(limbs, n0, d), slot n0 + d, or, with CHECK, to mac.check(limbs, n); E is the
// row's exponent.  K slots are requested ahead in registers (begin, before the
// values are ready); K slots from n0 (round), all from n0 on (rest).
template <int K, int CS>
struct FxRow {
  double c[K];
  __device__ __forceinline__ void begin(const double* __restrict__ co, int S) {
#pragma unroll
    for (int d = 0; d < K; ++d) c[d] = d < S ? __ldg(co + d * CS) : 0.0;
  }
  template <bool CHECK, typename F>
  static __device__ __forceinline__ void put(FxLimbs q, int n0, int d, F& mac) {
    if constexpr (CHECK) mac.check(q, n0 + d);
    else mac(q, n0, d);
  }
  template <typename F>
  __device__ __forceinline__ void round(const double* __restrict__ co, int n0, int S, int E, F& mac) {
#pragma unroll
    for (int d = 0; d < K; ++d) {
      const FxLimbs q = fx_coef(c[d], E);
      if (n0 + K + d < S) c[d] = __ldg(co + (n0 + K + d) * CS);
      if (n0 + d < S) mac.check(q, n0 + d);
    }
  }
  template <bool CHECK, typename F>
  __device__ __forceinline__ void rest(const double* __restrict__ co, int n0, int S, int E, F& mac) {
    co += (n0 + K) * CS;
    for (; n0 + 2 * K <= S; n0 += K) {  // every request in range
#pragma unroll
      for (int d = 0; d < K; ++d) {
        const FxLimbs q = fx_coef(c[d], E);
        c[d] = __ldg(co + d * CS);
        put<CHECK>(q, n0, d, mac);
      }
      co += K * CS;
    }
#pragma unroll
    for (int d = 0; d < K; ++d) {
      const FxLimbs q = fx_coef(c[d], E);
      if (n0 + K + d < S) c[d] = __ldg(co + d * CS);
      if (n0 + d < S) put<CHECK>(q, n0, d, mac);
    }
#pragma unroll
    for (int d = 0; d < K; ++d)
      if (n0 + K + d < S) put<CHECK>(fx_coef(c[d], E), n0, K + d, mac);
  }
};

// mac of all components of an item, its limbs ua, ub STRIDE apart a slot
template <int DIM, int STRIDE>
struct FxAll {
  const int4* ua;
  const int2* ub;
  FxSum s[DIM];
  uint32_t size[DIM];
  __device__ __forceinline__ void operator()(FxLimbs q, int n0, int d) {
    const int4 a = ua[n0 * STRIDE + d * STRIDE];
    s[0].mac(q, a.x, a.y);
    s[1].mac(q, a.z, a.w);
    if constexpr (DIM == 3) {
      const int2 b = ub[n0 * STRIDE + d * STRIDE];
      s[2].mac(q, b.x, b.y);
    }
  }
  __device__ __forceinline__ void check(FxLimbs q, int n) {
    (*this)(q, n, 0);
    const int4 a = ua[n * STRIDE];
    size[0] += fx_size(q, a.x);
    size[1] += fx_size(q, a.z);
    if constexpr (DIM == 3) size[2] += fx_size(q, ub[n * STRIDE].x);
  }
  // the sums are exact enough, or all coefficients (exponent E) or values
  // (exponents ex) are zero; least: the size that is enough
  __device__ __forceinline__ bool sure(int E, const int* ex, uint32_t least = fx_sure(DIM)) const {
    bool r = true;
#pragma unroll
    for (int j = 0; j < DIM; ++j) r &= size[j] >= least || ex[j] == kFxZero;
    return r || E == kFxZero;
  }
  // sure from here on: a size stays below 15 2^26 by the scale of the row
  __device__ __forceinline__ void pass() {
#pragma unroll
    for (int j = 0; j < DIM; ++j) size[j] += 1u << 30;
  }
};

// All slots of a row whose exponents are in range (fx); true if the sum stands.
// Ten slots are checked, the nearest cells.  In 3-D a row that does not pass by them,
// but comes within a factor 4 (noise: 1e-5 to 1e-3 of the rows of smooth fields),
// is judged by all its slots, with 5/4 as the bar, since what is left out weighs
// more where the far cells' values decide; its warp then checks them all.  A lone
// row's FMAs would hold its block up by 20 us (a chain of 85 slots, 2400 cycles for
// four).  The rule looks at a row's own values only, so that a face's flux depends
// on its stencil alone to the last bit.  Called by whole warps in 3-D.
template <int K, int CS, int DIM, int STRIDE>
__device__ __forceinline__ bool fx_row(FxRow<K, CS>& r, const double* __restrict__ co, int S, int E, const int* ex,
                                       bool fx, FxAll<DIM, STRIDE>& a) {
  bool ok = false, near = false;
  if (fx) {
    r.round(co, 0, S, E, a);
    r.round(co, K, S, E, a);
    ok = a.sure(E, ex);
    near = DIM == 3 && a.sure(E, ex, fx_sure(DIM) / 4);
  }
  if (DIM == 3 && __any_sync(0xffffffffu, near && !ok)) {
    if (near) {
      if (ok) a.pass();
      r.template rest<true>(co, 2 * K, S, E, a);
      ok = a.sure(E, ex, fx_sure(DIM) / 4 * 5);
    }
  } else if (ok) {
    r.template rest<false>(co, 2 * K, S, E, a);
  }
  return ok;
}

// the same sum by FP64 FMAs, SL slots CS apart, U slots' requests at a time
template <int DIM>
struct PlainSum {
  double v[DIM];
};
template <int DIM, int CS>
__device__ __noinline__ PlainSum<DIM> plain_row(const double* __restrict__ co, int SL,
                                                const int32_t* __restrict__ st,
                                                const double* __restrict__ w, int64_t ws) {
  constexpr int U = DIM == 2 ? 5 : 4;
  PlainSum<DIM> s;
#pragma unroll
  for (int j = 0; j < DIM; ++j) s.v[j] = 0.0;
  int n = 0;
  for (; n + U <= SL; n += U) {
    int32_t id[U];
    double c[U], u[U][DIM];
#pragma unroll
    for (int d = 0; d < U; ++d) id[d] = __ldg(st + (n + d) * kTile);
#pragma unroll
    for (int d = 0; d < U; ++d) {
      c[d] = __ldg(co + (int64_t)(n + d) * CS);
#pragma unroll
      for (int j = 0; j < DIM; ++j) u[d][j] = __ldg(w + j * ws + id[d]);
    }
#pragma unroll
    for (int d = 0; d < U; ++d)
#pragma unroll
      for (int j = 0; j < DIM; ++j) s.v[j] = fma(c[d], u[d][j], s.v[j]);
  }
  for (; n < SL; ++n) {
    const int32_t id = __ldg(st + n * kTile);
    const double c = __ldg(co + (int64_t)n * CS);
#pragma unroll
    for (int j = 0; j < DIM; ++j) s.v[j] = fma(c, __ldg(w + j * ws + id), s.v[j]);
  }
  return s;
}

// shared memory of the limbs of a number of items
template <int DIM>
static size_t fx_smem_bytes(int S, int items) {
  return (size_t)S * items * DIM * sizeof(int2);
}

// ---------------------------------------------------------------------
// stabilisation extrapolation: W threads per (cell, local face), each with a
// part of the stencil (their integer sums add up exactly)
// ---------------------------------------------------------------------
// NLF = faces per cell: 4 / 6 for quads / hexes, 3 / 4 for triangles / tetrahedra
template <int DIM, int NLF>
struct UstarShape {
  // the limbs of a 3-D stencil fill shared memory before its rows fill the
  // SM with threads: fewer cells a block, more threads a row
  static constexpr int CPB = DIM == 2 ? 32 : 16;
  static constexpr int ROWS = CPB * NLF;
  // four threads a row: 32^3 hexes 73 -> 59 us; two on 512^2 quads 57 -> 71 (both
  // before the sums were checked, 73 and 68 now); 6 17^3 tetrahedra 64 -> 44
  static constexpr int W = NLF >= 8 || DIM == 2 ? 1 : 4;
  static constexpr int THREADS = ROWS * W;
  static constexpr int BLOCKS = 1152 / THREADS;
  // the parts' sums: FxTotal's h and l, or a double in h's place
  static size_t smem(int S) {
    return fx_smem_bytes<DIM>(S, CPB) + (sizeof(int64_t) + sizeof(uint32_t)) * (W - 1) * ROWS * DIM;
  }
};

template <int DIM, int NLF>
__global__ void __launch_bounds__(UstarShape<DIM, NLF>::THREADS, UstarShape<DIM, NLF>::BLOCKS)
    k_ustar(DevMesh m, const double* __restrict__ w, double* __restrict__ ustar) {
  using SH = UstarShape<DIM, NLF>;
  constexpr int CPB = SH::CPB, ROWS = SH::ROWS, W = SH::W, CS = kTile * NLF;
  extern __shared__ __align__(16) double sm[];
  __shared__ int ex[CPB * DIM];
  __shared__ uint32_t size[W > 1 ? W * DIM * ROWS : 1];  // the parts' FxAll::size
  const int S = m.S;
  int4* ua = reinterpret_cast<int4*>(sm);                                        // [S][CPB]
  int2* ub = reinterpret_cast<int2*>(ua + S * CPB);                              // [S][CPB]
  int64_t* part = reinterpret_cast<int64_t*>(ub + (DIM == 3 ? S * CPB : 0));     // [W-1][DIM][ROWS]
  uint32_t* part_l = reinterpret_cast<uint32_t*>(part + (W - 1) * ROWS * DIM);   // the same
  const int64_t cell0 = (int64_t)blockIdx.x * CPB;
  const int it = threadIdx.x % ROWS, p = threadIdx.x / ROWS;
  const int ci = it / NLF, lf = it % NLF;
  const int64_t cell = cell0 + ci, tile = cell0 / kTile;
  const bool on = cell < m.nc;
  const int row = (int)(cell % kTile) * NLF + lf;
  const int n0 = p * S / W, len = (p + 1) * S / W - n0;  // this thread's slots
  const double* __restrict__ co = m.cex + tile * (int64_t)S * CS + row + (int64_t)n0 * CS;
  FxRow<5, CS> r;
  r.begin(co, on ? len : 0);
  const int E = on ? m.cexp[tile * CS + row] : kFxPlain;
  const int64_t ws = m.wst;  // stride of the state read
  fx_gather<DIM, SH::THREADS, CPB>(m.cst, w, ws, S, cell0, (int)min((int64_t)CPB, m.nc - cell0), ua, ub, ex);
  bool fx = E != kFxPlain && ex[ci * DIM] != 0;
  FxTotal t[DIM];
  FxAll<DIM, CPB> a{ua + n0 * CPB + ci, ub + n0 * CPB + ci, {}, {}};
  if (W == 1) {
    if (DIM == 3 || fx) fx = fx_row(r, co, len, E, ex + ci * DIM, fx, a);
  } else if (fx) {  // ten slots of the first part are checked, five of each other
    r.round(co, 0, len, E, a);
    if (p == 0) r.round(co, 5, len, E, a);
    r.template rest<false>(co, p == 0 ? 10 : 5, len, E, a);
#pragma unroll
    for (int j = 0; j < DIM; ++j) size[(p * DIM + j) * ROWS + it] = a.size[j];
  }
#pragma unroll
  for (int j = 0; j < DIM; ++j) {
    t[j] = a.s[j].total();
    if (W > 1 && p > 0) {
      part[((p - 1) * DIM + j) * ROWS + it] = t[j].h;
      part_l[((p - 1) * DIM + j) * ROWS + it] = t[j].l;
    }
  }
  bool again = W == 1 && !fx;  // some row of the block is to be summed by FMAs
  if (W > 1) {
    __syncthreads();
    if (fx) {
#pragma unroll
      for (int j = 0; j < DIM; ++j)
#pragma unroll
        for (int k = 0; k < W; ++k)
          if (k != p) a.size[j] += size[(k * DIM + j) * ROWS + it];
      fx = a.sure(E, ex + ci * DIM);
    }
    again = __syncthreads_or(on && !fx);
  }
  PlainSum<DIM> acc;
  if (again) {
    if (on && !fx)
      acc = plain_row<DIM, CS>(co, len, m.cst + tile * (int64_t)S * kTile + n0 * kTile + cell % kTile, w, ws);
    if (W > 1) {
      if (on && !fx && p > 0) {
#pragma unroll
        for (int j = 0; j < DIM; ++j)
          part[((p - 1) * DIM + j) * ROWS + it] = __double_as_longlong(acc.v[j]);
      }
      __syncthreads();
    }
  }
  if (!on || p > 0) return;
#pragma unroll
  for (int j = 0; j < DIM; ++j) {
    if (fx) {
#pragma unroll
      for (int k = 0; k < W - 1; ++k) {
        t[j].h += part[(k * DIM + j) * ROWS + it];
        t[j].l += part_l[(k * DIM + j) * ROWS + it];
      }
      acc.v[j] = fx_scale(t[j], E, ex[ci * DIM + j]);
    } else {
#pragma unroll
      for (int k = 0; k < W - 1; ++k) acc.v[j] += __longlong_as_double(part[(k * DIM + j) * ROWS + it]);
    }
    ustar[(cell * NLF + lf) * DIM + j] = w[j * ws + cell] + acc.v[j];
  }
}

// ---------------------------------------------------------------------
// inertia: cell average of the cell fit over the cell's Gauss points,
// ubar_P = u_P + sum_N cmass_N u_N (eq. inertiaTerm with the Taylor
// extrapolation of eq. alphaJump; u_P alone for one point per cell), and,
// scaled, the u-dependent part -rho Omega_P c2 ubar_P of the BDF2 term
// ---------------------------------------------------------------------
template <int DIM, bool SCALE>
__global__ void k_cell_avg(DevMesh m, const double* __restrict__ w, int64_t ws,
                           double* __restrict__ out) {
  const int64_t c = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (c >= m.nc) return;
  const int64_t nc = m.nc;
  double acc[DIM];
#pragma unroll
  for (int j = 0; j < DIM; ++j) acc[j] = w[j * ws + c];
  if (m.cmass) {
    const int64_t tile = c / kTile, ci = c % kTile;
    const int32_t* __restrict__ st = m.cst + tile * m.S * kTile + ci;
    const double* __restrict__ e = m.cmass + tile * m.S * kTile + ci;
    for (int n = 0; n < m.S; ++n) {
      const int32_t id = __ldg(st + n * kTile);
      const double en = __ldg(e + n * kTile);
#pragma unroll
      for (int j = 0; j < DIM; ++j) acc[j] = fma(en, __ldg(w + j * ws + id), acc[j]);
    }
  }
  const double sc = SCALE ? m.mscale[c] : 1.0;
#pragma unroll
  for (int j = 0; j < DIM; ++j) out[j * nc + c] = SCALE ? sc * acc[j] : acc[j];
}

void launch_cell_average(const DevMesh& m, const double* u, double* ubar, cudaStream_t st) {
  const unsigned g = (unsigned)((m.nc + 127) / 128);
  if (m.dim == 2)
    k_cell_avg<2, false><<<g, 128, 0, st>>>(m, u, m.nc, ubar);
  else
    k_cell_avg<3, false><<<g, 128, 0, st>>>(m, u, m.nc, ubar);
}

__global__ void k_combine4(int64_t n, double a, const double* __restrict__ x, double b,
                           const double* __restrict__ y, double g, const double* __restrict__ z,
                           double e, const double* __restrict__ w, double* __restrict__ out) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n;
       i += (int64_t)gridDim.x * blockDim.x) {
    double s = 0.0;
    if (x) s += a * x[i];
    if (y) s += b * y[i];
    if (z) s += g * z[i];
    if (w) s += e * w[i];
    out[i] = s;
  }
}

void launch_combine4(int64_t n, double a, const double* x, double b, const double* y, double g,
                     const double* z, double e, const double* w, double* out, cudaStream_t st) {
  k_combine4<<<(unsigned)std::min<int64_t>((n + 255) / 256, 4096), 256, 0, st>>>(n, a, x, b, y, g,
                                                                                 z, e, w, out);
}

__global__ void k_scale_rows(int dim, int64_t nc, const double* __restrict__ s, double* out) {
  const int64_t c = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (c >= nc) return;
  for (int j = 0; j < dim; ++j) out[j * nc + c] *= s[c];
}

void launch_scale_rows(int dim, int64_t nc, const double* s, double* out, cudaStream_t st) {
  k_scale_rows<<<(unsigned)((nc + 255) / 256), 256, 0, st>>>(dim, nc, s, out);
}

// ---------------------------------------------------------------------
// laws: traction t = T a from G[i][j] = du_j/dx_i
// ---------------------------------------------------------------------
template <int DIM, int LAW>
__device__ __forceinline__ void traction(const double (&G)[3][3], const double* a, const Material& mt,
                                         double* t) {
  if (LAW == HOFV_LAW_LINEAR) {
    // sigma = mu (G + G^T) + lambda tr(G) I, eq. (linearElastic)
    double tr = 0.0;
#pragma unroll
    for (int i = 0; i < DIM; ++i) tr += G[i][i];
#pragma unroll
    for (int i = 0; i < DIM; ++i) {
      double s = mt.lam * tr * a[i];
#pragma unroll
      for (int j = 0; j < DIM; ++j) s = fma(mt.mu * (G[i][j] + G[j][i]), a[j], s);
      t[i] = s;
    }
  } else {
    // neo-Hookean, eq. (neoHook), first Piola-Kirchhoff P = J sigma F^{-T}
    // (eq. nanson).  With B = F F^T, w = cof(F) a and r = J^{-1/3}:
    //   J sigma = mu J^{-2/3} (B - tr(B)/3 I) + kappa/2 (J^2 - 1) I,
    //   t = P a = J sigma w / J = alpha B w + beta w,
    //   alpha = mu r^5,  beta = kappa/2 (J^2 - 1) r^3 - alpha tr(B) / 3,
    // and since F^T cof(F) = J I, B w = F (F^T w) = J F a.
    double F[3][3];
#pragma unroll
    for (int i = 0; i < 3; ++i)
#pragma unroll
      for (int j = 0; j < 3; ++j) F[i][j] = (i == j ? 1.0 : 0.0) + G[j][i];
    double C[3][3];  // cofactor matrix
    C[0][0] = F[1][1] * F[2][2] - F[1][2] * F[2][1];
    C[0][1] = F[1][2] * F[2][0] - F[1][0] * F[2][2];
    C[0][2] = F[1][0] * F[2][1] - F[1][1] * F[2][0];
    C[1][0] = F[0][2] * F[2][1] - F[0][1] * F[2][2];
    C[1][1] = F[0][0] * F[2][2] - F[0][2] * F[2][0];
    C[1][2] = F[0][1] * F[2][0] - F[0][0] * F[2][1];
    C[2][0] = F[0][1] * F[1][2] - F[0][2] * F[1][1];
    C[2][1] = F[0][2] * F[1][0] - F[0][0] * F[1][2];
    C[2][2] = F[0][0] * F[1][1] - F[0][1] * F[1][0];
    const double J = F[0][0] * C[0][0] + F[0][1] * C[0][1] + F[0][2] * C[0][2];
    // J^{-1/3}; not defined for J <= 0 (an inverted element): NaN, so the
    // caller's finiteness checks reject the state
    const double r = inv_cbrt(J);
    const double r3 = r * r * r;
    const double alpha = mt.mu * (r * r) * r3;
    double trB = 0.0;  // tr(F F^T): the squares of F's entries
#pragma unroll
    for (int i = 0; i < 3; ++i)
#pragma unroll
      for (int j = 0; j < 3; ++j) trB = fma(F[i][j], F[i][j], trB);
    const double beta = 0.5 * mt.kappa * fma(J, J, -1.0) * r3 - alpha * trB * (1.0 / 3.0);
    const double aJ = alpha * J;
#pragma unroll
    for (int i = 0; i < DIM; ++i) {
      double wi = 0.0, fa = 0.0;
#pragma unroll
      for (int l = 0; l < DIM; ++l) {
        wi = fma(C[i][l], a[l], wi);
        fa = fma(F[i][l], a[l], fa);
      }
      t[i] = fma(aJ, fa, beta * wi);
    }
  }
}

// ---------------------------------------------------------------------
// face fluxes: FPB consecutive faces a block (a block may span two tiles),
// one thread a (face, row) for the gradients, a (face, point) for the law and
// a (face, component) for the quadrature
// ---------------------------------------------------------------------
// Blocks of 192 threads at most: 467 us against 478 with 384 (32^3 hexes p = 3),
// 353 against 372 (40^3 p = 2), as more blocks mix their phases; 1152 threads an
// SM: 478 against 537 with 768 (all before the sums were checked).
template <int DIM, int Q>
struct FluxShape {
  static constexpr int R = Q * DIM;  // rows a face, at most 96 (8 fan slots of 2 x 2 points)
  static constexpr int kMaxT = 192;
  static constexpr int FPB = kMaxT / R < kTile ? kMaxT / R : kTile;
  static constexpr int THREADS = (FPB * R + 31) / 32 * 32;
  static constexpr int BLOCKS = 1152 / THREADS < 32 ? 1152 / THREADS : 32;
  // Three rows a face do not pay for the split of its values: one point a face in 3-D
  // is summed by FMAs alone (32^3 hexes p = 1: 119 us in fixed point, 95 so; 6 10^3
  // tetrahedra 34, 20)
  static constexpr bool FX = DIM == 2 || Q > 1;
  static size_t smem(int S) { return (FX ? fx_smem_bytes<DIM>(S, FPB) : 0) + sizeof(double) * FPB * (R * DIM + R); }
};

template <int DIM, int LAW, int Q>
__global__ void __launch_bounds__(FluxShape<DIM, Q>::THREADS, FluxShape<DIM, Q>::BLOCKS)
    k_flux(DevMesh m, Material mt, const double* __restrict__ w, const double* __restrict__ ustar,
           const double* __restrict__ ubq, const double* __restrict__ ubf, double* __restrict__ flux) {
  using SH = FluxShape<DIM, Q>;
  constexpr int R = SH::R, FPB = SH::FPB;
  extern __shared__ __align__(16) double sm[];
  __shared__ int ex[FPB * DIM];
  const int S = m.S;
  int4* ua = reinterpret_cast<int4*>(sm);                                // [S][FPB] components 0, 1
  int2* ub = reinterpret_cast<int2*>(ua + S * FPB);                      // [S][FPB] component 2
  double* Gs = SH::FX ? reinterpret_cast<double*>(ub + (DIM == 3 ? S * FPB : 0)) : sm;  // [FPB][R][DIM]
  double* Ts = Gs + FPB * R * DIM;                                       // [FPB][Q][DIM]
  const int64_t f0 = (int64_t)blockIdx.x * FPB;
  const int nf = (int)min((int64_t)FPB, m.nfid - f0);
  const int it = threadIdx.x;
  const int64_t nc = m.wst;  // stride of the state read
  // (1) gradient rows: thread (fi, r) accumulates sum_N c_{r,N} u_N
  {
    const int fi = it / R, r = it % R;
    const int64_t f = f0 + fi, tile = f / kTile;
    const int row = (int)(f % kTile) * R + r;
    // rows of points without area (polyhedral fan slots past a face's last
    // corner) are neither read nor formed
    const bool live = fi < nf && (m.fql == nullptr || r < __ldg(m.fql + f) * DIM);
    const double* __restrict__ co = m.fco + tile * (int64_t)S * kTile * R + row;
    FxRow<5, kTile * R> rw;
    int E = kFxPlain;
    if constexpr (SH::FX) {
      rw.begin(co, live ? S : 0);
      if (live) E = m.fexp[tile * kTile * R + row];
      fx_gather<DIM, SH::THREADS, FPB>(m.fst, w, nc, S, f0, nf, ua, ub, ex);
    }
    double acc[DIM];
#pragma unroll
    for (int j = 0; j < DIM; ++j) acc[j] = 0.0;
    if (DIM == 3 || live) {
      bool fx = false;
      if constexpr (SH::FX) {
        FxAll<DIM, FPB> a{ua + fi, ub + fi, {}, {}};
        fx = fx_row(rw, co, S, E, ex + fi * DIM, live && E != kFxPlain && ex[fi * DIM] != 0, a);
        if (fx) {
#pragma unroll
          for (int j = 0; j < DIM; ++j) acc[j] = fx_scale(a.s[j].total(), E, ex[fi * DIM + j]);
        }
      }
      if (live && !fx) {
        const PlainSum<DIM> s =
            plain_row<DIM, kTile * R>(co, S, m.fst + tile * (int64_t)S * kTile + f % kTile, w, nc);
#pragma unroll
        for (int j = 0; j < DIM; ++j) acc[j] = s.v[j];
      }
    }
    if (live) {
      if (f >= m.nfi && f < m.nfi + m.nfd) {  // ghost node of a displacement face
        const int64_t fd = f - m.nfi;
        const double cg = m.gco[fd * R + r];
        const int q = r / DIM;
#pragma unroll
        for (int j = 0; j < DIM; ++j) acc[j] = fma(cg, ubq[(fd * Q + q) * DIM + j], acc[j]);
      }
    }
    if (fi < nf) {
#pragma unroll
      for (int j = 0; j < DIM; ++j) Gs[(fi * R + r) * DIM + j] = acc[j];
    }
  }
  __syncthreads();
  // (2) law and traction at each Gauss point
  if (it < nf * Q) {
    const int fi = it / Q, q = it % Q;
    const int64_t f = f0 + fi;
    double t[DIM];
    double G[3][3] = {{0, 0, 0}, {0, 0, 0}, {0, 0, 0}};
#pragma unroll
    for (int i = 0; i < DIM; ++i)
#pragma unroll
      for (int j = 0; j < DIM; ++j) G[i][j] = Gs[(fi * R + q * DIM + i) * DIM + j];
    double a[3];
#pragma unroll
    for (int k = 0; k < DIM; ++k) a[k] = m.aq[(f * Q + q) * 3 + k];
    traction<DIM, LAW>(G, a, mt, t);
#pragma unroll
    for (int i = 0; i < DIM; ++i) Ts[(fi * Q + q) * DIM + i] = t[i];
  }
  __syncthreads();
  // (3) quadrature over the face + alpha stabilisation
  if (it < nf * DIM) {
    const int fi = it / DIM, i = it % DIM;
    const int64_t f = f0 + fi;
    double s = 0.0;
    for (int q = 0; q < Q; ++q) s += Ts[(fi * Q + q) * DIM + i];
    const int32_t sp = m.fstar[2 * f], sn = m.fstar[2 * f + 1];
    const double other = sn >= 0 ? ustar[(int64_t)sn * DIM + i] : ubf[(f - m.nfi) * DIM + i];
    const double coef = mt.alpha * mt.kbar * m.fstab[f];
    flux[f * DIM + i] = fma(coef, other - ustar[(int64_t)sp * DIM + i], s);
  }
}

// ---------------------------------------------------------------------
// cell assembly; out = R, or (R - R0) * inv_eps when R0 != nullptr
// ---------------------------------------------------------------------
template <int DIM, int NLF>
__global__ void k_cell(DevMesh m, const double* __restrict__ flux, const double* __restrict__ src,
                       const double* __restrict__ R0, const double* __restrict__ d_eps,
                       double* __restrict__ out) {
  const int64_t c = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (c >= m.nc) return;
  double r[DIM];
#pragma unroll
  for (int j = 0; j < DIM; ++j) r[j] = src ? src[j * m.nc + c] : 0.0;
#pragma unroll
  for (int lf = 0; lf < NLF; ++lf) {
    const int32_t code = m.cface[c * NLF + lf];
    if (code == 0) continue;
    const int64_t f = (code > 0 ? code : -code) - 1;
#pragma unroll
    for (int j = 0; j < DIM; ++j) {
      const double v = flux[f * DIM + j];
      r[j] = code > 0 ? r[j] + v : r[j] - v;
    }
  }
  if (m.mscale) {
#pragma unroll
    for (int j = 0; j < DIM; ++j) r[j] += m.inert[j * m.nc + c];
  }
  if (R0) {
    const double ie = d_eps[1];
#pragma unroll
    for (int j = 0; j < DIM; ++j) out[j * m.nc + c] = (r[j] - R0[j * m.nc + c]) * ie;
  } else {
#pragma unroll
    for (int j = 0; j < DIM; ++j) out[j * m.nc + c] = r[j];
  }
}

template <int DIM>
__global__ void __launch_bounds__(32 * DIM)
    k_tflux(DevMesh m, const double* __restrict__ tco, double alpha_kbar,
            const double* __restrict__ w, const double* __restrict__ ustar,
            const double* __restrict__ ubf, double* __restrict__ flux);

// ---------------------------------------------------------------------
// symmetry faces (Sec. 3.5.3): the state extended by the ghosts' reflected
// values R u_src = u - 2 n (n . u), and, after the stabilisation
// extrapolation, the mirror R u*_P of each symmetry face's own value as the
// value beyond the face (its jump then penalises the normal component only)
// ---------------------------------------------------------------------
template <int DIM>
__global__ void k_extend(DevMesh m, const double* __restrict__ w, double* __restrict__ wext) {
  const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  const int64_t nc = m.nc, ws = m.wst;
  if (i < nc) {
#pragma unroll
    for (int j = 0; j < DIM; ++j) wext[j * ws + i] = w[j * nc + i];
  } else if (i < ws) {
    const int64_t g = i - nc;
    const int32_t src = m.gsrc[g];
    const double* n = m.nrm + 3 * (int64_t)m.gface[g];
    double u[DIM], un = 0.0;
#pragma unroll
    for (int j = 0; j < DIM; ++j) {
      u[j] = w[j * nc + src];
      un += n[j] * u[j];
    }
#pragma unroll
    for (int j = 0; j < DIM; ++j) wext[j * ws + i] = u[j] - 2.0 * un * n[j];
  }
}

template <int DIM>
__global__ void k_sym_other(DevMesh m, const double* __restrict__ ustar) {
  const int64_t b = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (b >= m.nfy) return;
  const int64_t f = m.nfi + m.nfd + b;
  const double* us = ustar + (int64_t)m.fstar[2 * f] * DIM;
  const double* n = m.nrm + 3 * f;
  double un = 0.0;
#pragma unroll
  for (int j = 0; j < DIM; ++j) un += n[j] * us[j];
#pragma unroll
  for (int j = 0; j < DIM; ++j) m.ubfw[(f - m.nfi) * DIM + j] = us[j] - 2.0 * un * n[j];
}

// faces per cell as a compile-time constant: d + 1 (triangles /
// tetrahedra), 2 d (quads / hexes), kPolyMaxSides slots (2-D polygons),
// kPolyhedronMaxFaces slots (3-D polyhedra)
template <int DIM, typename F>
static void by_faces_per_cell(const DevMesh& m, F&& launch) {
  if (m.nlf == DIM + 1)
    launch(std::integral_constant<int, DIM + 1>{});
  else if (m.nlf == 2 * DIM)
    launch(std::integral_constant<int, 2 * DIM>{});
  else if constexpr (DIM == 2)
    launch(std::integral_constant<int, kPolyMaxSides>{});
  else
    launch(std::integral_constant<int, kPolyhedronMaxFaces>{});
}

// Gauss points per face as a compile-time constant: q^(d-1) for q = 1..4 in
// 2-D, 1..3 in 3-D; on polyhedra 4 or 8 fan slots of q^2 points for q = 1, 2
template <int DIM, typename F>
static void by_points(const DevMesh& m, F&& launch) {
  if constexpr (DIM == 2) {
    switch (m.Q) {
      case 1: return launch(std::integral_constant<int, 1>{});
      case 2: return launch(std::integral_constant<int, 2>{});
      case 3: return launch(std::integral_constant<int, 3>{});
      default: return launch(std::integral_constant<int, 4>{});
    }
  } else {
    switch (m.Q) {
      case 1: return launch(std::integral_constant<int, 1>{});
      case 4: return launch(std::integral_constant<int, 4>{});
      case 8: return launch(std::integral_constant<int, 8>{});
      case 16: return launch(std::integral_constant<int, 16>{});
      case 32: return launch(std::integral_constant<int, 32>{});
      default: return launch(std::integral_constant<int, 9>{});
    }
  }
}

template <int DIM, int LAW>
static void residual_impl(const DevMesh& m, const Material& mat, const double* w,
                          const double* d_eps, const double* R0, double* out, double* ustar,
                          double* flux, const double* ubq, const double* ubf, const double* src,
                          cudaStream_t st, cudaEvent_t* ev) {
  if (ev) cudaEventRecord(ev[0], st);
  if (m.ng > 0) {
    k_extend<DIM><<<(unsigned)((m.wst + 255) / 256), 256, 0, st>>>(m, w, m.wext);
    w = m.wext;
  }
  by_faces_per_cell<DIM>(m, [&](auto nlf) {
    constexpr int NLF = decltype(nlf)::value;
    using SH = UstarShape<DIM, NLF>;
    k_ustar<DIM, NLF><<<(unsigned)((m.nc + SH::CPB - 1) / SH::CPB), SH::THREADS, SH::smem(m.S), st>>>(m, w, ustar);
  });
  if (m.nfy > 0) k_sym_other<DIM><<<(unsigned)((m.nfy + 127) / 128), 128, 0, st>>>(m, ustar);
  if (ev) cudaEventRecord(ev[1], st);
  if (m.nftile > 0) {
    if (LAW == HOFV_LAW_LINEAR && m.tco) {
      k_tflux<DIM><<<(unsigned)m.nftile, 32 * DIM, 0, st>>>(m, m.tco, mat.alpha * mat.kbar, w,
                                                            ustar, ubf, flux);
    } else {
      by_points<DIM>(m, [&](auto q) {
        constexpr int Q = decltype(q)::value;
        using SH = FluxShape<DIM, Q>;
        k_flux<DIM, LAW, Q><<<(unsigned)((m.nfid + SH::FPB - 1) / SH::FPB), SH::THREADS, SH::smem(m.S), st>>>(
            m, mat, w, ustar, ubq, ubf, flux);
      });
    }
  }
  if (ev) cudaEventRecord(ev[2], st);
  if (m.mscale)
    k_cell_avg<DIM, true><<<(unsigned)((m.nc + 127) / 128), 128, 0, st>>>(m, w, m.wst, m.inert);
  const unsigned cgrid = (unsigned)((m.nc + 255) / 256);
  by_faces_per_cell<DIM>(m, [&](auto nlf) {
    constexpr int NLF = decltype(nlf)::value;
    k_cell<DIM, NLF><<<cgrid, 256, 0, st>>>(m, flux, src, R0, d_eps, out);
  });
  if (ev) cudaEventRecord(ev[3], st);
}

void launch_residual_df(const DevMesh& m, const Material& mat, const double* w,
                        const double* d_eps, const double* R0, double* out, double* ustar,
                        double* flux, const double* ubq, const double* ubf, const double* src,
                        cudaStream_t st, cudaEvent_t* ev);

void launch_residual(const DevMesh& m, const Material& mat, const double* w, const double* /*v*/,
                     const double* d_eps, const double* R0, double* out, double* ustar,
                     double* flux, const double* ubq, const double* ubf, const double* src,
                     cudaStream_t st, cudaEvent_t* ev) {
  if (m.prec == HOFV_PREC_DF64) {
    launch_residual_df(m, mat, w, d_eps, R0, out, ustar, flux, ubq, ubf, src, st, ev);
    return;
  }
  if (m.dim == 2) {
    if (mat.law == HOFV_LAW_LINEAR)
      residual_impl<2, 0>(m, mat, w, d_eps, R0, out, ustar, flux, ubq, ubf, src, st, ev);
    else
      residual_impl<2, 1>(m, mat, w, d_eps, R0, out, ustar, flux, ubq, ubf, src, st, ev);
  } else {
    if (mat.law == HOFV_LAW_LINEAR)
      residual_impl<3, 0>(m, mat, w, d_eps, R0, out, ustar, flux, ubq, ubf, src, st, ev);
    else
      residual_impl<3, 1>(m, mat, w, d_eps, R0, out, ustar, flux, ubq, ubf, src, st, ev);
  }
}

// ---------------------------------------------------------------------
// constant source per cell: integrated body force + traction-face fluxes
// sum_q |a_q| T_{b,q} (eq. divStressDiscret, traction term)
// ---------------------------------------------------------------------
__global__ void k_source(int dim, int nlf, int Q, int64_t nc, int64_t nfi, int64_t nfd,
                         const int64_t* __restrict__ cf, const int32_t* __restrict__ ftag,
                         const double* __restrict__ aq, const double* __restrict__ tbq,
                         const double* __restrict__ body, const double* __restrict__ gflux,
                         double* __restrict__ src) {
  const int64_t c = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (c >= nc) return;
  for (int j = 0; j < dim; ++j) {
    double s = body ? body[j * nc + c] : 0.0;
    if (gflux)
      for (int lf = 0; lf < nlf; ++lf) {
        const int64_t f = cf[c * nlf + lf];  // -1: polygon slot without a face
        if (f >= 0 && ftag[f] == 0) s += gflux[(f - nfi) * dim + j];
      }
    if (tbq) {
      for (int lf = 0; lf < nlf; ++lf) {
        const int64_t f = cf[c * nlf + lf];
        if (f < 0 || ftag[f] != 1) continue;
        const int64_t b = f - nfi - nfd;
        for (int q = 0; q < Q; ++q) {
          const double* a = aq + (f * Q + q) * 3;
          const double mag = sqrt(a[0] * a[0] + a[1] * a[1] + a[2] * a[2]);
          s += mag * tbq[(b * Q + q) * dim + j];
        }
      }
    }
    src[j * nc + c] = s;
  }
}

void launch_source(const hofv_ctx* c, cudaStream_t st) {
  k_source<<<(unsigned)((c->nc + 127) / 128), 128, 0, st>>>(
      c->dim, c->nlf, c->Q, c->nc, c->nfi, c->nfd + c->nfy, c->d_cf, c->d_ftag, c->d_aq,
      c->nft > 0 ? c->d_tbq : nullptr, c->d_body,
      (c->contract && c->tco_valid && c->mat.law == HOFV_LAW_LINEAR && c->nfd > 0) ? c->d_gflux
                                                                                  : nullptr,
      c->d_src);
}

}  // namespace hofv

namespace hofv {
// per-cell sum of |flux_f| over the cell's internal and displacement faces
// (the force scale F_s = max over cells), from the last residual's fluxes
template <int DIM, int NLF>
__global__ void k_flux_scale(DevMesh m, const double* __restrict__ flux, double* __restrict__ out) {
  const int64_t c = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (c >= m.nc) return;
  double s = 0.0;
#pragma unroll
  for (int lf = 0; lf < NLF; ++lf) {
    const int32_t code = m.cface[c * NLF + lf];
    if (code == 0) continue;
    const int64_t f = (code > 0 ? code : -code) - 1;
    double q = 0.0;
#pragma unroll
    for (int j = 0; j < DIM; ++j) q += flux[f * DIM + j] * flux[f * DIM + j];
    s += sqrt(q);
  }
  out[c] = s;
}

void launch_flux_scale(const DevMesh& m, const double* flux, double* out, cudaStream_t st) {
  const unsigned grid = (unsigned)((m.nc + 255) / 256);
  if (m.dim == 2 && m.nlf == 3)
    k_flux_scale<2, 3><<<grid, 256, 0, st>>>(m, flux, out);
  else if (m.dim == 2 && m.nlf == kPolyMaxSides)
    k_flux_scale<2, kPolyMaxSides><<<grid, 256, 0, st>>>(m, flux, out);
  else if (m.dim == 2)
    k_flux_scale<2, 4><<<grid, 256, 0, st>>>(m, flux, out);
  else if (m.nlf == 4)
    k_flux_scale<3, 4><<<grid, 256, 0, st>>>(m, flux, out);
  else if (m.nlf == kPolyhedronMaxFaces)
    k_flux_scale<3, kPolyhedronMaxFaces><<<grid, 256, 0, st>>>(m, flux, out);
  else
    k_flux_scale<3, 6><<<grid, 256, 0, st>>>(m, flux, out);
}
}  // namespace hofv

// ---------------------------------------------------------------------
// Linear elasticity with the law and the face quadrature folded into the
// coefficients (an exact re-association of eq. divStressDiscret for Hooke's
// law): with sigma = mu (G + G^T) + lambda tr(G) I and G = sum_N c_N (x) u_N,
//   flux_i = sum_N sum_k T_N[i][k] u_N[k],
//   T_N[i][k] = sum_q mu c_qN,i a_q,k + mu (c_qN . a_q) delta_ik + lambda a_q,i c_qN,k.
// One d x d matrix per face and stencil cell replaces Q d coefficients and
// the per-point law: d^2 FMAs per cell instead of Q d^2.  The ghost node of
// a displacement face only multiplies prescribed data, so its part is a
// constant folded into the cell source.
// ---------------------------------------------------------------------
namespace hofv {

__device__ __forceinline__ float2 ld_pair(const float2* __restrict__ pl, int i, int rows, int np);

// tco[tile][N][fi][i][k] from fco[tile][N][fi][q*d + i] and aq
template <int DIM>
__global__ void k_build_tco(DevMesh m, double mu, double lam, double* __restrict__ tco) {
  const int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;  // (tile, N, fi)
  const int64_t total = m.nftile * m.S * kTile;
  if (e >= total) return;
  const int fi = (int)(e % kTile);
  const int64_t tile = e / ((int64_t)m.S * kTile);
  const int64_t f = tile * kTile + fi;
  double T[DIM][DIM];
#pragma unroll
  for (int i = 0; i < DIM; ++i)
#pragma unroll
    for (int k = 0; k < DIM; ++k) T[i][k] = 0.0;
  if (f < m.nfid) {
    const double* co = m.fco + e * m.R;
    const int np = kTile * m.Q;  // points of the tile: planes of the pairs' layout
    const float2* pairs = reinterpret_cast<const float2*>(m.fco) + (e - fi) * m.R + fi * m.Q;  // tile, slot
    for (int q = 0; q < m.Q; ++q) {
      double c[DIM], a[DIM], ca = 0.0;
#pragma unroll
      for (int i = 0; i < DIM; ++i) {
        if (m.prec == HOFV_PREC_DF64) {  // stored as a double-float pair
          const float2 p = ld_pair(pairs + q, i, DIM, np);
          c[i] = (double)p.x + (double)p.y;
        } else {
          c[i] = co[q * DIM + i];
        }
        a[i] = m.aq[(f * m.Q + q) * 3 + i];
        ca += c[i] * a[i];
      }
#pragma unroll
      for (int i = 0; i < DIM; ++i)
#pragma unroll
        for (int k = 0; k < DIM; ++k)
          T[i][k] += mu * c[i] * a[k] + lam * a[i] * c[k] + (i == k ? mu * ca : 0.0);
    }
  }
#pragma unroll
  for (int i = 0; i < DIM; ++i)
#pragma unroll
    for (int k = 0; k < DIM; ++k) tco[(e * DIM + i) * DIM + k] = T[i][k];
}

// ghost-node flux of each displacement face: sum_q Tg_q u_bq (constant data)
template <int DIM>
__global__ void k_ghost_flux(DevMesh m, double mu, double lam, const double* __restrict__ ubq,
                             double* __restrict__ gflux) {
  const int64_t fd = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (fd >= m.nfd) return;
  const int64_t f = m.nfi + fd;
  double out[DIM];
#pragma unroll
  for (int i = 0; i < DIM; ++i) out[i] = 0.0;
  for (int q = 0; q < m.Q; ++q) {
    double c[DIM], a[DIM], u[DIM], ca = 0.0, cu = 0.0, au = 0.0;
#pragma unroll
    for (int i = 0; i < DIM; ++i) {
      c[i] = m.gco[fd * m.R + q * DIM + i];
      a[i] = m.aq[(f * m.Q + q) * 3 + i];
      u[i] = ubq[(fd * m.Q + q) * DIM + i];
      ca += c[i] * a[i];
      cu += c[i] * u[i];
      au += a[i] * u[i];
    }
#pragma unroll
    for (int i = 0; i < DIM; ++i) out[i] += mu * c[i] * au + mu * ca * u[i] + lam * a[i] * cu;
  }
#pragma unroll
  for (int i = 0; i < DIM; ++i) gflux[fd * DIM + i] = out[i];
}

// face fluxes from the contracted matrices: thread (face, row i), 32 faces
// per block; every FP64 instruction runs with full warps (32 d threads)
template <int DIM>
__global__ void __launch_bounds__(32 * DIM)
    k_tflux(DevMesh m, const double* __restrict__ tco, double alpha_kbar,
            const double* __restrict__ w, const double* __restrict__ ustar,
            const double* __restrict__ ubf, double* __restrict__ flux) {
  const int64_t tile = blockIdx.x;
  const int it = threadIdx.x;  // fi * DIM + i
  const int fi = it / DIM, i = it % DIM;
  const int64_t f = tile * kTile + fi;
  const int S = m.S;
  const int64_t nc = m.wst;  // stride of the state read
  const int32_t* __restrict__ st = m.fst + tile * S * kTile + fi;
  const double* __restrict__ tc = tco + tile * (int64_t)S * kTile * DIM * DIM + it * DIM;
  double acc = 0.0;
#pragma unroll 4
  for (int n = 0; n < S; ++n) {
    const int32_t id = __ldg(st + n * kTile);
    const double* t = tc + (int64_t)n * kTile * DIM * DIM;
#pragma unroll
    for (int k = 0; k < DIM; ++k) acc = fma(__ldg(t + k), __ldg(w + k * nc + id), acc);
  }
  if (f < m.nfid) {
    const int32_t sp = m.fstar[2 * f], sn = m.fstar[2 * f + 1];
    const double other = sn >= 0 ? ustar[(int64_t)sn * DIM + i] : ubf[(f - m.nfi) * DIM + i];
    flux[f * DIM + i] = fma(alpha_kbar * m.fstab[f], other - ustar[(int64_t)sp * DIM + i], acc);
  }
}

void launch_build_tco(const DevMesh& m, double mu, double lam, double* tco, cudaStream_t st) {
  const int64_t total = m.nftile * m.S * kTile;
  if (total == 0) return;
  if (m.dim == 2)
    k_build_tco<2><<<(unsigned)((total + 127) / 128), 128, 0, st>>>(m, mu, lam, tco);
  else
    k_build_tco<3><<<(unsigned)((total + 127) / 128), 128, 0, st>>>(m, mu, lam, tco);
}

void launch_ghost_flux(const DevMesh& m, double mu, double lam, const double* ubq, double* gflux,
                       cudaStream_t st) {
  if (m.nfd == 0) return;
  if (m.dim == 2)
    k_ghost_flux<2><<<(unsigned)((m.nfd + 127) / 128), 128, 0, st>>>(m, mu, lam, ubq, gflux);
  else
    k_ghost_flux<3><<<(unsigned)((m.nfd + 127) / 128), 128, 0, st>>>(m, mu, lam, ubq, gflux);
}

void launch_tflux(const DevMesh& m, const double* tco, double alpha_kbar, const double* w,
                  const double* ustar, const double* ubf, double* flux, cudaStream_t st) {
  if (m.nftile == 0) return;
  if (m.dim == 2)
    k_tflux<2><<<(unsigned)m.nftile, 32 * 2, 0, st>>>(m, tco, alpha_kbar, w, ustar, ubf, flux);
  else
    k_tflux<3><<<(unsigned)m.nftile, 32 * 3, 0, st>>>(m, tco, alpha_kbar, w, ustar, ubf, flux);
}

}  // namespace hofv


// =====================================================================
// Gradient contraction in double-float arithmetic (HOFV_PREC_DF64).
//
// GB300 issues FP64 at 2 FMAs per clock per SM and FP32 at 128, while the
// per-point face kernel does d FP64 FMAs per 8-byte coefficient: it is bound
// by the FP64 pipe at 20-35 % of HBM.  Here every coefficient is stored as a
// pair of floats (hi, lo) in the same 8 bytes and the state is split the
// same way once per call; each product c u is formed as hi*hi exactly
// (TwoProduct by FMA, Dekker 1971) plus the cross terms, and accumulated by
// TwoSum with a compensation float (Dot2, Ogita, Rump & Oishi 2005): twelve
// FP32 operations per product, two products an instruction where they pair.
// The sum is converted to FP64 for the law, the quadrature, the stabilisation
// jump and the assembly, which stay FP64.
//
// Jv must not difference two residuals contracted separately: each carries
// an independent rounding of 2^-48 relative, which the division by eps
// (~1e-8) would amplify.  For the linear law the residual is affine and the
// difference quotient is evaluated exactly as the homogeneous residual of v
// (no boundary data or sources).  For the neo-Hookean law the kernels
// contract v alone and difference the tractions of grad u + eps grad v and
// grad u in FP64, with grad u and its tractions taken from a cache filled
// once per linearisation point, so the rounding of grad u cancels exactly.
// =====================================================================
namespace hofv {

// modes of the double-float face kernel
constexpr int kDfResidual = 0;  // flux of u (split a, extrapolated values ua)
constexpr int kDfHomog = 1;     // linear law: flux of v without ghost data or prescribed values
constexpr int kDfFill = 2;      // neo-Hookean: gradient rows and tractions of u into the cache
constexpr int kDfJv = 3;        // neo-Hookean: flux(u + eps v) - flux(u) from the cache

__device__ __forceinline__ void ff_mac(float ch, float cl, float uh, float ul, float& s, float& e) {
  const float p = __fmul_rn(ch, uh);
  float r = __fmaf_rn(ch, uh, -p);  // exact rounding error of ch * uh
  r = __fmaf_rn(ch, ul, r);
  r = __fmaf_rn(cl, uh, r);
  const float t = __fadd_rn(s, p);
  const float z = __fsub_rn(t, s);
  const float q = __fadd_rn(__fsub_rn(s, __fsub_rn(t, z)), __fsub_rn(p, z));  // TwoSum error
  s = t;
  e = __fadd_rn(e, __fadd_rn(q, r));
}

__device__ __forceinline__ double ff_value(float s, float e) { return (double)s + (double)e; }

// two floats in a 64-bit register: Blackwell's packed FP32 instructions do
// both halves in one issue slot (the contractions are short of issue slots,
// not of FP32 lanes)
typedef unsigned long long f32x2;
__device__ __forceinline__ f32x2 pack2(float a, float b) {
  f32x2 r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
  return r;
}
__device__ __forceinline__ float2 unpack2(f32x2 v) {
  float2 r;
  asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(v));
  return r;
}
__device__ __forceinline__ f32x2 mul2(f32x2 a, f32x2 b) {
  f32x2 r;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ f32x2 add2(f32x2 a, f32x2 b) {
  f32x2 r;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ f32x2 sub2(f32x2 a, f32x2 b) {
  f32x2 r;
  asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ f32x2 fma2(f32x2 a, f32x2 b, f32x2 c) {
  f32x2 r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
  return r;
}

// ff_mac on both halves, bit for bit (the product is formed negated, which
// changes no rounding); nch = -ch
__device__ __forceinline__ void ff_mac2(f32x2 ch, f32x2 nch, f32x2 cl, f32x2 uh, f32x2 ul, f32x2& s,
                                        f32x2& e) {
  const f32x2 np = mul2(nch, uh);
  f32x2 r = fma2(ch, uh, np);
  r = fma2(ch, ul, r);
  r = fma2(cl, uh, r);
  const f32x2 t = sub2(s, np);
  const f32x2 z = sub2(t, s);
  const f32x2 q = sub2(sub2(s, sub2(t, z)), add2(np, z));
  s = t;
  e = add2(e, add2(q, r));
}
__device__ __forceinline__ f32x2 neg2(f32x2 a) { return a ^ 0x8000000080000000ull; }

// Coefficient pairs of a point's rows are stored two rows together, ready
// for ff_mac2: plane 2k holds (hi, hi) and plane 2k + 1 (lo, lo) of rows 2k
// and 2k + 1; an odd last row keeps its plane (hi, lo).  This reads row i of
// a point whose planes lie np apart.
__device__ __forceinline__ float2 ld_pair(const float2* __restrict__ pl, int i, int rows, int np) {
  if ((rows & 1) && i == rows - 1) return pl[(int64_t)i * np];
  const float2 h = pl[(int64_t)(i & ~1) * np], l = pl[(int64_t)(i | 1) * np];
  return (i & 1) ? make_float2(h.y, l.y) : make_float2(h.x, l.x);
}

__device__ __forceinline__ void split_value(double a, float& h, float& l) {
  h = __double2float_rn(a);
  l = __double2float_rn(a - (double)h);  // a - h is exact in FP64
}

// a double as hi + mid + lo, three floats, exactly (24 + 24 bits, then the
// at most 5 remaining significant bits)
__device__ __forceinline__ float4 split3(double a) {
  const float h = __double2float_rn(a);
  const double r = a - (double)h;  // exact
  const float m = __double2float_rn(r);
  return make_float4(h, m, __double2float_rn(r - (double)m), 0.f);
}

// n cells of a state read with stride ws -> three-float splits
template <int DIM>
__global__ void k_split(int64_t n, int64_t ws, const double* __restrict__ u, float4* __restrict__ su) {
  const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (i >= n) return;
#pragma unroll
  for (int j = 0; j < DIM; ++j) su[i * DIM + j] = split3(u[j * ws + i]);
}

__device__ __forceinline__ void two_sum(float a, float b, float& s, float& e) {
  s = __fadd_rn(a, b);
  const float z = __fsub_rn(s, a);
  e = __fadd_rn(__fsub_rn(a, __fsub_rn(s, z)), __fsub_rn(b, z));
}

// x - r from their three-float splits as a double-float pair: the high and
// middle differences exactly (TwoSum), the low parts' difference rounded
// once (2^-72 of the values), renormalised
__device__ __forceinline__ float2 diff3(const float4 x, const float4 r) {
  float s1, e1, s2, e2, h, e3;
  two_sum(x.x, -r.x, s1, e1);
  two_sum(x.y, -r.y, s2, e2);
  two_sum(s1, s2, h, e3);
  const float l = __fadd_rn(e3, __fadd_rn(e1, __fadd_rn(e2, __fsub_rn(x.z, r.z))));
  const float dh = __fadd_rn(h, l);
  return make_float2(dh, __fsub_rn(l, __fsub_rn(dh, h)));
}

// Coefficient arrays in place between doubles and double-float pairs.  An
// array is a list of chunks (one tile and stencil slot each) of np points
// (face Gauss points, or cells) with `rows` coefficients a point: doubles as
// [np][rows], pairs as planes [rows][np] (ld_pair), so that a thread that
// takes a point reads its rows coalesced with its neighbours'.  One block a
// chunk.
__global__ void __launch_bounds__(256) k_coef_format(double* __restrict__ a, int np, int rows, int to_df) {
  extern __shared__ double2 chunk_raw[];
  double* chunk = reinterpret_cast<double*>(chunk_raw);
  const int n = np * rows;
  double* g = a + (int64_t)blockIdx.x * n;
  for (int k = threadIdx.x; k < n; k += blockDim.x) chunk[k] = g[k];
  __syncthreads();
  for (int k = threadIdx.x; k < n; k += blockDim.x) {
    if (to_df) {  // k = plane * np + point
      const int pl = k / np;
      const double* c = chunk + (k % np) * rows;
      float2 v;
      if ((rows & 1) && pl == rows - 1) {
        split_value(c[pl], v.x, v.y);
      } else {
        float h0, l0, h1, l1;
        split_value(c[pl & ~1], h0, l0);
        split_value(c[pl | 1], h1, l1);
        v = (pl & 1) ? make_float2(l0, l1) : make_float2(h0, h1);
      }
      reinterpret_cast<float2*>(g)[k] = v;
    } else {  // k = point * rows + i
      const float2 p = ld_pair(reinterpret_cast<const float2*>(chunk) + k / rows, k % rows, rows, np);
      g[k] = ff_value(p.x, p.y);
    }
  }
}

// fcsum[tile][i][point] = sum_n of the stored pairs of row i of the point
__global__ void k_row_sums(DevMesh m, double* __restrict__ fcsum) {
  const int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;  // (tile, row, point)
  const int np = kTile * m.Q, cs = kTile * m.R;
  if (e >= m.nftile * cs) return;
  const int64_t tile = e / cs;
  const int i = (int)(e % cs) / np, p = (int)(e % cs) % np;
  const float2* co = reinterpret_cast<const float2*>(m.fco) + tile * (int64_t)m.S * cs + p;
  double sum = 0.0;
  for (int n = 0; n < m.S; ++n) {
    const float2 c = ld_pair(co + (int64_t)n * cs, i, m.dim, np);
    sum += ff_value(c.x, c.y);
  }
  fcsum[e] = sum;
}

void launch_row_sums(const DevMesh& m, double* fcsum, cudaStream_t st) {
  const int64_t n = m.nftile * kTile * m.R;
  if (n > 0) k_row_sums<<<(unsigned)((n + 255) / 256), 256, 0, st>>>(m, fcsum);
}

void launch_coef_format(double* a, int64_t chunks, int np, int rows, int to_df, cudaStream_t st) {
  if (chunks <= 0) return;
  k_coef_format<<<(unsigned)chunks, 256, sizeof(double) * np * rows, st>>>(a, np, rows, to_df);
}

// Stabilisation extrapolation of the state w (split sw):
//   out[(cell * NLF + lf) * DIM + j] = w_P + sum_N e_N w_N.
// A block takes a tile of 32 cells, lane = cell.  A warp takes RPG of the
// cells' rows and every W-th stencil slot: each gathered value serves RPG
// rows, and the slots of a cell are spread over W warps, so that a mesh of a
// few tiles still keeps its loads in flight.  The warps' partial sums meet in
// shared memory as float pairs and are added in a fixed order.  Rows without
// a flux (polygon and polyhedron slots past a cell's last face, traction
// faces) are never read back and, where slots may be empty, load nothing.
// A warp's slots past the last take its cell, with zero coefficients: a cell of
// the stencil, so that a value that is not finite reaches no other cell by them.
// Measured (us, one thread a (cell, face) -> this): 13^3 hexes p = 3 60 -> 25
// (four warps a tile hide each other's latency), 48^3 hexes p = 3 187 -> 137
// (0.55 of HBM: the gathers and the packed products), p = 2 148 -> 111, 512^2
// quads p = 3 76 -> 66, 24-layer prisms 58 -> 48, 6 17^3 tetrahedra 54 -> 31.
template <int NLF>
struct UsShape {
  static constexpr int RPG = NLF >= 8 ? 4 : NLF;   // rows a warp takes
  static constexpr int NG = NLF / RPG;             // row groups
  static constexpr bool SPARSE = NLF >= 8;         // cells with empty face slots
  // few: no tile for each SM (13^3 hexes 15.9 -> 10.5 us with eight)
  static constexpr int split(int S, bool few) { return NLF == 16 ? 2 : S <= 32 ? 2 : few && NLF < 8 ? 8 : 4; }
  static constexpr int THREADS = 256;              // at most
};

template <int DIM, int NLF>
__global__ void __launch_bounds__(UsShape<NLF>::THREADS, 512 / UsShape<NLF>::THREADS)
    k_ustar_df(DevMesh m, const float4* __restrict__ sw, const double* __restrict__ w,
               double* __restrict__ out) {
  using SH = UsShape<NLF>;
  constexpr int RPG = SH::RPG, NP = RPG / 2, NV = NLF * DIM, U = 4;
  constexpr bool ODD = RPG & 1;
  extern __shared__ float2 part[];     // [W][NV][33]
  const int S = m.S;
  const int64_t tile = blockIdx.x;
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const int W = (blockDim.x >> 5) / SH::NG, g = wid / W, k = wid % W;
  const int64_t cell = tile * kTile + lane;
  const int32_t* __restrict__ st = m.cst + tile * (int64_t)S * kTile + lane;
  const float2* __restrict__ ex =
      reinterpret_cast<const float2*>(m.cex) + tile * (int64_t)S * kTile * NLF + g * RPG * kTile + lane;
  unsigned live = ~0u;                 // bit r: rows 2r, 2r + 1 are needed
  if (SH::SPARSE) {
    live = 0;
    if (cell < m.nc)
#pragma unroll
      for (int r = 0; r < RPG; ++r)
        if (__ldg(m.cface + cell * NLF + g * RPG + r) != 0) live |= 1u << (r / 2);
  }
  f32x2 s[NP][DIM], e[NP][DIM];
  float so[DIM], eo[DIM];              // an odd last row
#pragma unroll
  for (int j = 0; j < DIM; ++j) {
    so[j] = eo[j] = 0.f;
#pragma unroll
    for (int r = 0; r < NP; ++r) s[r][j] = e[r][j] = 0;
  }
  int32_t id[U];
#pragma unroll
  for (int d = 0; d < U; ++d) id[d] = __ldg(st + min(k + d * W, S - 1) * kTile);
  for (int n0 = k; n0 < S; n0 += U * W) {
    float2 c[U][RPG], u[U][DIM];
#pragma unroll
    for (int d = 0; d < U; ++d) {
      const int n = n0 + d * W;
#pragma unroll
      for (int r = 0; r < RPG; ++r)
        c[d][r] = n < S && (live >> (r / 2) & 1) ? __ldg(ex + ((int64_t)n * NLF + r) * kTile)
                                                 : make_float2(0.f, 0.f);
#pragma unroll
      for (int j = 0; j < DIM; ++j)
        u[d][j] = __ldg(reinterpret_cast<const float2*>(sw + (int64_t)id[d] * DIM + j));
    }
#pragma unroll
    for (int d = 0; d < U; ++d) id[d] = __ldg(st + min(n0 + (U + d) * W, S - 1) * kTile);
#pragma unroll
    for (int d = 0; d < U; ++d) {
#pragma unroll
      for (int j = 0; j < DIM; ++j) {
        const f32x2 uh = pack2(u[d][j].x, u[d][j].x), ul = pack2(u[d][j].y, u[d][j].y);
#pragma unroll
        for (int r = 0; r < NP; ++r) {
          const f32x2 ch = pack2(c[d][2 * r].x, c[d][2 * r].y);
          ff_mac2(ch, neg2(ch), pack2(c[d][2 * r + 1].x, c[d][2 * r + 1].y), uh, ul, s[r][j], e[r][j]);
        }
        if (ODD) ff_mac(c[d][RPG - 1].x, c[d][RPG - 1].y, u[d][j].x, u[d][j].y, so[j], eo[j]);
      }
    }
  }
  {
    float2* p = part + ((int64_t)k * NV + g * RPG * DIM) * 33 + lane;
#pragma unroll
    for (int j = 0; j < DIM; ++j) {
#pragma unroll
      for (int r = 0; r < NP; ++r) {
        const float2 a = unpack2(s[r][j]), b = unpack2(e[r][j]);
        p[(2 * r * DIM + j) * 33] = make_float2(a.x, b.x);
        p[((2 * r + 1) * DIM + j) * 33] = make_float2(a.y, b.y);
      }
      if (ODD) p[((RPG - 1) * DIM + j) * 33] = make_float2(so[j], eo[j]);
    }
  }
  __syncthreads();
  for (int t = threadIdx.x; t < kTile * NV; t += blockDim.x) {
    const int ci = t / NV, v = t % NV;
    const int64_t c = tile * kTile + ci;
    if (c >= m.nc) break;
    float2 a = part[v * 33 + ci];
    for (int q = 1; q < W; ++q) {
      const float2 b = part[(q * NV + v) * 33 + ci];
      float h, l;
      two_sum(a.x, b.x, h, l);
      a = make_float2(h, __fadd_rn(l, __fadd_rn(a.y, b.y)));
    }
    out[c * NV + v] = w[(v % DIM) * m.wst + c] + ff_value(a.x, a.y);
  }
}

// component i of the mirror (I - 2 n n) x of the extrapolated value x of a
// symmetry face (the value beyond the face, as k_sym_other)
template <int DIM>
__device__ __forceinline__ double mirror_i(const double* x, const double* n, int i) {
  double un = 0.0;
#pragma unroll
  for (int j = 0; j < DIM; ++j) un += n[j] * x[j];
  return x[i] - 2.0 * un * n[i];
}

// Face fluxes, double-float gradient rows.  One thread takes one Gauss point
// of one face: its DIM coefficient rows (DIM x DIM products a stencil cell),
// then the law at that point in registers; the tractions meet in shared
// memory only for the sum over the face.  QD points a face, FPB consecutive
// faces a block (a group may span two tiles); sw is the three-float split of the state contracted (u, or v in the Jv modes), wd
// the same state in FP64 and ws its extrapolated values.
//
// Each gradient is contracted against the differences to a reference cell,
// the face's nearest stencil cell N0:
//   sum_N c_N w_N = sum_N c_N (w_N - w_N0) + w_N0 sum_N c_N,
// an exact identity; the differences are small where the field is smooth,
// so the rounding of the products and sums of the contraction scales with
// them and not with |w| (on fine meshes |w| exceeds h |grad w| by orders of
// magnitude), and the last term is one FP64 product with the FP64 row sum
// of the stored coefficients.  The stored pairs differ from the FP64
// coefficients by up to 2^-48 of each; through the row sum that difference
// still meets w_N0 itself (the sum of the pairs, not of the originals).
// The block first forms its faces' differences (exact differences of the
// splits) in shared memory, slots 1 .. S-1; the reference's own difference
// is zero and its coefficient enters only through the row sum.  Each thread
// then streams its DIM rows through a ring of RING slots in registers: the
// coefficients of slot n + RING are requested when slot n is consumed.  The
// pairs are stored by plane (k_coef_format), so every request of a warp is
// 256 contiguous bytes.
// Points without area (polyhedral fan slots past a face's last corner) load
// nothing.
//
// PACK: polyhedral faces of 8 fan slots (QD = 32).  A group is a run of
// consecutive faces of one tile whose points with area fill the block's
// kPackPoints threads (at most kPackMaxFaces faces; the host builds the runs,
// DevMesh::pgrp); thread it takes the group's it-th point with area.
// What bounds it and what was measured (GB300, 2070 MHz; us of the kernel in
// a Jacobian-vector product: one thread a coefficient row before -> this):
// 48^3 hexes p = 3 neo-Hookean 1554 -> 1132, 48^3 hexes p = 2 807 -> 502,
// 512^2 quads p = 3 linear 197 -> 129, 24-layer prisms 524 -> 344, 6 17^3
// tetrahedra 158 -> 104; 32^3 hexes face by face (16 points a face) 670 -> 453,
// neo-Hookean 846 -> 502, with one point a fan slot (4) 178 -> 121, 24-layer
// prisms with one (8) 207 -> 129, 200^2 polygons (2) 57 -> 35.  The coefficient
// stream is 85 % of measured HBM at p = 3; the rest is the FP64 law (without it:
// 1009 of 1266 us at that stage) and, at p = 2, the gather of the differences (442
// of 582 us without).  A plane of a prism's triangle is 96 bytes, which DRAM
// reads as 128: 11 % more bytes than needed on prisms (4 % with a face's rows together).
//  * A thread a point instead of a row: a difference read from shared memory
//    serves DIM rows, the gradient never leaves registers, and no barrier
//    stands between contraction and law, so one warp's FP64 law runs beside
//    other warps' contraction.
//  * Small groups (14 faces of 9 points fill 126 of 128 threads; 16 faces of
//    4): the phases of more blocks mix.  32 faces a block, two an SM: 1657 us;
//    16 faces (144 of 160 threads): 1423; 14: 1383.
//  * AHEAD: the pairs of slot n + RING + AHEAD are prefetched into L2, so the
//    ring only has to cover an L2 hit, and five blocks an SM fit in registers:
//    1383 -> 1270 us (4 to 16 slots ahead alike; 2-D 4, of its 19 slots).
//  * Packed FP32 instructions (ff_mac2): 1266 -> 1155 us at p = 3, 582 -> 500
//    at p = 2, 147 -> 129 on the quads.
//  * A ring of 4 (3 in 2-D, whose twelve blocks an SM need 56 registers);
//    ten stencil cells' ids of a thread loaded before their values: 3 %.
// Not kept: the pair widened to double by integer operations (1 % slower),
// the operands of the law prefetched at the start (no gain).
template <int DIM, int QD, bool PACK>
struct DfShape {
  static constexpr int FPB = PACK       ? kPackMaxFaces
                             : DIM == 2 ? 32
                             : QD == 1  ? 32
                             : QD == 9  ? 14
                             : QD == 16 ? 8
                                        : 16;  // faces per group
  static constexpr int THREADS = PACK ? kPackPoints : (FPB * QD + 31) / 32 * 32;
  static constexpr int RING = DIM == 2 ? 3 : 4;    // slots requested ahead in registers
  static constexpr int AHEAD = DIM == 2 ? 4 : 8;   // ... and beyond them into L2
  static constexpr int IDS = DIM == 2 ? 7 : 10;    // stencil ids of a thread loaded together
  static constexpr int BLOCKS = (DIM == 2 ? 1152 : PACK || QD == 9 ? 640 : 512) / THREADS;
  static constexpr int MIN_BLOCKS = BLOCKS < 32 ? BLOCKS : 32;  // an SM holds 32 at most
};

// dynamic shared memory: the differences (DIM pairs a slot and face), the
// tractions of the block's points
template <int DIM, int QD, bool PACK>
static size_t df_smem_bytes(int S) {
  using SH = DfShape<DIM, QD, PACK>;
  return (size_t)(S - 1) * SH::FPB * DIM * 8 + sizeof(double) * SH::THREADS * DIM;
}

__device__ __forceinline__ void prefetch_l2(const void* p) {
  asm volatile("prefetch.global.L2 [%0];" ::"l"(p));
}

template <int DIM, int LAW, int MODE, int QD, bool PACK>
__global__ void __launch_bounds__(DfShape<DIM, QD, PACK>::THREADS, DfShape<DIM, QD, PACK>::MIN_BLOCKS)
    k_flux_df(DevMesh m, Material mt, const float4* __restrict__ sw, const double* __restrict__ wd,
              const double* __restrict__ ws, const double* __restrict__ ubq,
              const double* __restrict__ ubf, const double* __restrict__ d_eps,
              double* __restrict__ flux) {
  using SH = DfShape<DIM, QD, PACK>;
  constexpr int FPB = SH::FPB, T = SH::THREADS, Q = QD, K = SH::RING;
  constexpr int NP = kTile * Q;        // points of a tile: plane stride of the coefficients
  constexpr int CS = NP * DIM;         // coefficient stride between stencil slots
  extern __shared__ __align__(16) double sm[];
  const int S = m.S;
  float4* ua = reinterpret_cast<float4*>(sm);                            // [S-1][FPB] components 0, 1
  float2* ub = reinterpret_cast<float2*>(ua + (size_t)(S - 1) * FPB);    // [S-1][FPB] component 2
  double* Ts = reinterpret_cast<double*>(ub + (DIM == 3 ? (size_t)(S - 1) * FPB : 0));  // [T][DIM]
  __shared__ int rowp[PACK ? FPB + 1 : 1];  // points with area before each face of the group
  const int it = threadIdx.x;
  int64_t f0;
  int nf;                              // faces of the group
  int fi = it / Q, q = it % Q;         // this thread's face in the group and its point
  bool live;
  if (PACK) {
    f0 = m.pgrp[2 * (int64_t)blockIdx.x];
    nf = m.pgrp[2 * (int64_t)blockIdx.x + 1];
    if (it == 0) {
      int acc = 0;
      rowp[0] = 0;
      for (int k = 0; k < FPB; ++k) rowp[k + 1] = acc += k < nf ? m.fql[f0 + k] : 0;
    }
    __syncthreads();
    fi = 0;
    while (fi + 1 < nf && rowp[fi + 1] <= it) ++fi;
    live = it < rowp[nf];
    q = live ? it - rowp[fi] : 0;
  } else {
    f0 = (int64_t)blockIdx.x * FPB;
    nf = (int)(m.nfid - f0 < FPB ? m.nfid - f0 : FPB);
    live = fi < nf && (m.fql == nullptr || q < __ldg(m.fql + f0 + fi));
    if (fi >= nf) fi = 0;
  }
  const int64_t f = f0 + fi;
  const int64_t tile = f / kTile;
  const int pt = (int)(f % kTile) * Q + q;  // point within the tile
  const float2* __restrict__ co =
      reinterpret_cast<const float2*>(m.fco) + tile * (int64_t)S * CS + CS + pt;  // slot 1
  const int SL = live ? S - 1 : 0;     // stencil slots this thread contracts: 1 .. S-1
  float2 cq[K][DIM];
#pragma unroll
  for (int d = 0; d < K; ++d)
#pragma unroll
    for (int i = 0; i < DIM; ++i)
      cq[d][i] = d < SL ? __ldg(co + d * CS + i * NP) : make_float2(0.f, 0.f);
  constexpr int PD = SH::AHEAD;
#pragma unroll
  for (int d = K; d < K + PD; ++d)
#pragma unroll
    for (int i = 0; i < DIM; ++i)
      if (d < SL) prefetch_l2(co + d * CS + i * NP);
  // the group's differences; a thread keeps one face, STEP slots at a time
  {
    constexpr int STEP = T / FPB, IDB = SH::IDS;
    const int fj = it % FPB;
    if (fj < nf && it < STEP * FPB) {
      const int64_t fg = f0 + fj;
      const int32_t* __restrict__ st = m.fst + fg / kTile * (int64_t)S * kTile + fg % kTile;
      float4 r[DIM];
      const int32_t id0 = __ldg(st);
#pragma unroll
      for (int j = 0; j < DIM; ++j) r[j] = __ldg(sw + (int64_t)id0 * DIM + j);
      for (int n0 = 1 + it / FPB; n0 < S; n0 += IDB * STEP) {
        int32_t id[IDB];  // the cells first: one wait for their list, one for their values
#pragma unroll
        for (int k = 0; k < IDB; ++k) id[k] = n0 + k * STEP < S ? __ldg(st + (n0 + k * STEP) * kTile) : 0;
#pragma unroll
        for (int k = 0; k < IDB; ++k) {
          const int n = n0 + k * STEP;
          if (n >= S) break;
          float4 x[DIM];
#pragma unroll
          for (int j = 0; j < DIM; ++j) x[j] = __ldg(sw + (int64_t)id[k] * DIM + j);
          const float2 a = diff3(x[0], r[0]), b = diff3(x[1], r[1]);
          ua[(n - 1) * FPB + fj] = make_float4(a.x, b.x, a.y, b.y);
          if constexpr (DIM == 3) ub[(n - 1) * FPB + fj] = diff3(x[2], r[2]);
        }
      }
    }
  }
  __syncthreads();
  // gradient rows: sum_N c_{i,N} (w_N - w_N0), rows 0 and 1 together for each
  // component; in 3-D row 2 takes components 0 and 1 together, then 2 alone
  f32x2 s01[DIM], e01[DIM], s2 = 0, e2 = 0;
  float s22 = 0.f, e22 = 0.f;
#pragma unroll
  for (int j = 0; j < DIM; ++j) s01[j] = e01[j] = 0;
  auto mac_slot = [&](int n, const float2 (&c)[DIM]) {
    const float4 a = ua[n * FPB + fi];  // (hi, hi, lo, lo) of components 0, 1
    const f32x2 ch = pack2(c[0].x, c[0].y), cl = pack2(c[1].x, c[1].y), nch = neg2(ch);
    ff_mac2(ch, nch, cl, pack2(a.x, a.x), pack2(a.z, a.z), s01[0], e01[0]);
    ff_mac2(ch, nch, cl, pack2(a.y, a.y), pack2(a.w, a.w), s01[1], e01[1]);
    if constexpr (DIM == 3) {
      const float2 b = ub[n * FPB + fi];
      ff_mac2(ch, nch, cl, pack2(b.x, b.x), pack2(b.y, b.y), s01[2], e01[2]);
      const f32x2 c2 = pack2(c[2].x, c[2].x);
      ff_mac2(c2, neg2(c2), pack2(c[2].y, c[2].y), pack2(a.x, a.y), pack2(a.z, a.w), s2, e2);
      ff_mac(c[2].x, c[2].y, b.x, b.y, s22, e22);
    }
  };
  int n0 = 0;
  // steady part: every request in range
  for (; n0 + 2 * K <= SL; n0 += K) {
    const float2* cn = co + (int64_t)(n0 + K) * CS;
#pragma unroll
    for (int d = 0; d < K; ++d) {
      float2 c[DIM];
#pragma unroll
      for (int i = 0; i < DIM; ++i) {
        c[i] = cq[d][i];
        cq[d][i] = __ldg(cn + d * CS + i * NP);
      }
      const float2* pf = co + (int64_t)min(n0 + d + K + PD, SL - 1) * CS;
#pragma unroll
      for (int i = 0; i < DIM; ++i) prefetch_l2(pf + i * NP);
      mac_slot(n0 + d, c);
    }
  }
  // the operands of what follows are requested while the last slots run
  const int64_t tp = tile * NP;        // first point of the tile in the per-point arrays
  double cs[DIM], w0[DIM], a[3];
#pragma unroll
  for (int i = 0; i < DIM; ++i) cs[i] = w0[i] = a[i] = 0.0;
  if (live) {
    const int32_t id0 = __ldg(m.fst + tile * (int64_t)S * kTile + f % kTile);
#pragma unroll
    for (int i = 0; i < DIM; ++i) {
      cs[i] = __ldg(m.fcsum + tp * DIM + i * NP + pt);
      a[i] = __ldg(m.aq + (f * Q + q) * 3 + i);
      w0[i] = __ldg(wd + i * m.wst + id0);
    }
  }
  // the last K .. 2 K - 1 slots (fewer if S <= K)
#pragma unroll
  for (int d = 0; d < K; ++d) {
    const int n = n0 + d;
    if (n < SL) {
      float2 c[DIM];
#pragma unroll
      for (int i = 0; i < DIM; ++i) {
        c[i] = cq[d][i];
        if (n + K < SL) cq[d][i] = __ldg(co + (int64_t)(n + K) * CS + i * NP);
      }
      mac_slot(n, c);
    }
  }
  double gu[DIM][DIM], tu[DIM];        // the linearisation (Jv)
  if (MODE == kDfJv && live) {
#pragma unroll
    for (int i = 0; i < DIM; ++i) {
      tu[i] = m.tcache[tp * DIM + i * NP + pt];
#pragma unroll
      for (int j = 0; j < DIM; ++j) gu[i][j] = m.gcache[(tp * DIM + i * NP) * DIM + j * NP + pt];
    }
  }
#pragma unroll
  for (int d = 0; d < K; ++d)
    if (n0 + K + d < SL) mac_slot(n0 + K + d, cq[d]);
  float s[DIM][DIM], e[DIM][DIM];
#pragma unroll
  for (int j = 0; j < DIM; ++j) {
    const float2 a = unpack2(s01[j]), b = unpack2(e01[j]);
    s[0][j] = a.x, s[1][j] = a.y, e[0][j] = b.x, e[1][j] = b.y;
  }
  if constexpr (DIM == 3) {
    const float2 a = unpack2(s2), b = unpack2(e2);
    s[2][0] = a.x, s[2][1] = a.y, s[2][2] = s22;
    e[2][0] = b.x, e[2][1] = b.y, e[2][2] = e22;
  }
  double t[DIM];
#pragma unroll
  for (int i = 0; i < DIM; ++i) t[i] = 0.0;
  if (live) {
    const double eps = MODE == kDfJv ? __ldg(d_eps) : 0.0;
    double G[3][3] = {{0, 0, 0}, {0, 0, 0}, {0, 0, 0}};
#pragma unroll
    for (int i = 0; i < DIM; ++i)  // + w_N0 sum_N c_N, in FP64
#pragma unroll
      for (int j = 0; j < DIM; ++j) G[i][j] = fma(cs[i], w0[j], ff_value(s[i][j], e[i][j]));
    if (MODE == kDfResidual || MODE == kDfFill) {
      if (f >= m.nfi && f < m.nfi + m.nfd) {  // ghost node of a displacement face (prescribed data)
        const int64_t fd = f - m.nfi;
#pragma unroll
        for (int i = 0; i < DIM; ++i) {
          const double cg = m.gco[(fd * Q + q) * DIM + i];
#pragma unroll
          for (int j = 0; j < DIM; ++j) G[i][j] = fma(cg, ubq[(fd * Q + q) * DIM + j], G[i][j]);
        }
      }
    }
#pragma unroll
    for (int i = 0; i < DIM; ++i)
#pragma unroll
      for (int j = 0; j < DIM; ++j) {
        if (MODE == kDfFill) m.gcache[(tp * DIM + i * NP) * DIM + j * NP + pt] = G[i][j];
        if (MODE == kDfJv) G[i][j] = fma(eps, G[i][j], gu[i][j]);  // grad (u + eps v)
      }
    traction<DIM, LAW>(G, a, mt, t);
#pragma unroll
    for (int i = 0; i < DIM; ++i) {
      if (MODE == kDfFill) m.tcache[tp * DIM + i * NP + pt] = t[i];
      if (MODE == kDfJv) t[i] -= tu[i];
    }
  }
  if constexpr (MODE != kDfFill) {
#pragma unroll
    for (int i = 0; i < DIM; ++i) Ts[it * DIM + i] = t[i];
    // quadrature over the face + alpha stabilisation, a thread a component of
    // a face (SUMS of them where a face has fewer points than components);
    // what does not depend on the tractions is loaded before they are ready
    constexpr int SUMS = (FPB * DIM + T - 1) / T;
    double up[SUMS], other[SUMS], coef[SUMS];
#pragma unroll
    for (int k = 0; k < SUMS; ++k) {
      const int fs = (it + k * T) / DIM, i = (it + k * T) % DIM;
      const int64_t ff = f0 + fs;
      up[k] = other[k] = coef[k] = 0.0;
      if (fs < nf) {
        const int32_t sp = m.fstar[2 * ff], sn = m.fstar[2 * ff + 1];
        const bool sym = sn < 0 && ff >= m.nfi + m.nfd;
        up[k] = ws[(int64_t)sp * DIM + i];
        // beyond a displacement face: the prescribed value (the homogeneous and
        // Jv modes differentiate it away)
        other[k] = sn >= 0 ? ws[(int64_t)sn * DIM + i]
                   : sym   ? mirror_i<DIM>(ws + (int64_t)sp * DIM, m.nrm + 3 * ff, i)
                   : MODE == kDfResidual ? ubf[(ff - m.nfi) * DIM + i]
                                         : 0.0;
        // the stabilisation is linear: its difference at u + eps v and u is
        // eps times its value at v
        coef[k] = mt.alpha * mt.kbar * m.fstab[ff] * (MODE == kDfJv ? __ldg(d_eps) : 1.0);
      }
    }
    __syncthreads();
#pragma unroll
    for (int k = 0; k < SUMS; ++k) {
      const int fs = (it + k * T) / DIM, i = (it + k * T) % DIM;
      const int64_t ff = f0 + fs;
      if (fs < nf) {
        const int p0 = PACK ? rowp[fs] : fs * Q, p1 = PACK ? rowp[fs + 1] : p0 + Q;
        double acc = 0.0;
        for (int p = p0; p < p1; ++p) acc += Ts[p * DIM + i];
        flux[ff * DIM + i] = fma(coef[k], other[k] - up[k], acc);
      }
    }
  }
}

// contracted linear form, homogeneous part at v: sum_N T_N v_N plus the
// stabilisation of v with zero prescribed values (symmetry faces mirror)
template <int DIM>
__global__ void __launch_bounds__(32 * DIM)
    k_tflux_hom(DevMesh m, const double* __restrict__ tco, double alpha_kbar,
                const double* __restrict__ v, const double* __restrict__ vstar,
                double* __restrict__ flux) {
  const int64_t tile = blockIdx.x;
  const int it = threadIdx.x;  // fi * DIM + i
  const int fi = it / DIM, i = it % DIM;
  const int64_t f = tile * kTile + fi;
  const int S = m.S;
  const int64_t ws = m.wst;
  const int32_t* __restrict__ st = m.fst + tile * S * kTile + fi;
  const double* __restrict__ tc = tco + tile * (int64_t)S * kTile * DIM * DIM + it * DIM;
  double acc = 0.0;
#pragma unroll 4
  for (int n = 0; n < S; ++n) {
    const int32_t id = __ldg(st + n * kTile);
    const double* t = tc + (int64_t)n * kTile * DIM * DIM;
#pragma unroll
    for (int k = 0; k < DIM; ++k) acc = fma(__ldg(t + k), __ldg(v + k * ws + id), acc);
  }
  if (f < m.nfid) {
    const int32_t sp = m.fstar[2 * f], sn = m.fstar[2 * f + 1];
    const bool sym = sn < 0 && f >= m.nfi + m.nfd;
    const double up = vstar[(int64_t)sp * DIM + i];
    const double other = sn >= 0 ? vstar[(int64_t)sn * DIM + i]
                         : sym   ? mirror_i<DIM>(vstar + (int64_t)sp * DIM, m.nrm + 3 * f, i)
                                 : 0.0;
    flux[f * DIM + i] = fma(alpha_kbar * m.fstab[f], other - up, acc);
  }
}

// Jv assembly from face-flux differences: out = sum_f +-dflux_f / eps, plus
// the inertia term of v (linear, so its difference quotient is exact)
template <int DIM, int NLF>
__global__ void k_cell_diff(DevMesh m, const double* __restrict__ flux,
                            const double* __restrict__ d_eps, double* __restrict__ out) {
  const int64_t c = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (c >= m.nc) return;
  double r[DIM];
#pragma unroll
  for (int j = 0; j < DIM; ++j) r[j] = 0.0;
#pragma unroll
  for (int lf = 0; lf < NLF; ++lf) {
    const int32_t code = m.cface[c * NLF + lf];
    if (code == 0) continue;
    const int64_t f = (code > 0 ? code : -code) - 1;
#pragma unroll
    for (int j = 0; j < DIM; ++j) {
      const double v = flux[f * DIM + j];
      r[j] = code > 0 ? r[j] + v : r[j] - v;
    }
  }
  const double ie = d_eps[1];
#pragma unroll
  for (int j = 0; j < DIM; ++j)
    out[j * m.nc + c] = m.mscale ? fma(r[j], ie, m.inert[j * m.nc + c]) : r[j] * ie;
}

template <int DIM>
static void launch_ustar_df(const DevMesh& m, const float4* sw, const double* w, double* out,
                            cudaStream_t st) {
  by_faces_per_cell<DIM>(m, [&](auto nlf) {
    constexpr int NLF = decltype(nlf)::value;
    using SH = UsShape<NLF>;
    const int W = SH::split(m.S, m.nctile <= m.sms);
    k_ustar_df<DIM, NLF><<<(unsigned)m.nctile, 32 * SH::NG * W, sizeof(float2) * W * NLF * DIM * 33, st>>>(
        m, sw, w, out);
  });
}

template <int DIM, int LAW, int MODE, int QD, bool PACK = false>
static void launch_flux_df_q(const DevMesh& m, const Material& mat, const float4* sw,
                             const double* wd, const double* ws, const double* ubq,
                             const double* ubf, const double* d_eps, double* flux,
                             cudaStream_t st) {
  using SH = DfShape<DIM, QD, PACK>;
  const int64_t groups = PACK ? m.npg : (m.nfid + SH::FPB - 1) / SH::FPB;
  if (groups == 0) return;
  k_flux_df<DIM, LAW, MODE, QD, PACK><<<(unsigned)groups, SH::THREADS, df_smem_bytes<DIM, QD, PACK>(m.S), st>>>(
      m, mat, sw, wd, ws, ubq, ubf, d_eps, flux);
}

// 8 fan slots of 4 points always run with their packed groups
template <int DIM, int LAW, int MODE>
static void launch_flux_df(const DevMesh& m, const Material& mat, const float4* sw,
                           const double* wd, const double* ws, const double* ubq,
                           const double* ubf, const double* d_eps, double* flux, cudaStream_t st) {
  by_points<DIM>(m, [&](auto q) {
    constexpr int Q = decltype(q)::value;
    launch_flux_df_q<DIM, LAW, MODE, Q, Q == 32>(m, mat, sw, wd, ws, ubq, ubf, d_eps, flux, st);
  });
}

// the state (extended by the mirror nodes when the mesh has symmetry faces)
// split into double-float pairs; returns the FP64 state the kernels read
template <int DIM>
static const double* split_state(const DevMesh& m, const double* u, double* ext, float4* su,
                                 cudaStream_t st) {
  const unsigned g = (unsigned)((m.wst + 255) / 256);
  if (m.ng > 0) {
    k_extend<DIM><<<g, 256, 0, st>>>(m, u, ext);
    u = ext;
  }
  k_split<DIM><<<g, 256, 0, st>>>(m.wst, m.wst, u, su);
  return u;
}

template <int DIM, int LAW>
static void residual_impl_df(const DevMesh& m, const Material& mat, const double* w,
                             const double* d_eps, const double* R0, double* out, double* ustar,
                             double* flux, const double* ubq, const double* ubf, const double* src,
                             cudaStream_t st, cudaEvent_t* ev) {
  if (ev) cudaEventRecord(ev[0], st);
  w = split_state<DIM>(m, w, m.wext, m.su, st);
  launch_ustar_df<DIM>(m, m.su, w, ustar, st);
  if (ev) cudaEventRecord(ev[1], st);
  if (m.nftile > 0) {
    if (LAW == HOFV_LAW_LINEAR && m.tco) {
      if (m.nfy > 0) k_sym_other<DIM><<<(unsigned)((m.nfy + 127) / 128), 128, 0, st>>>(m, ustar);
      k_tflux<DIM><<<(unsigned)m.nftile, 32 * DIM, 0, st>>>(m, m.tco, mat.alpha * mat.kbar, w,
                                                            ustar, ubf, flux);
    } else {
      launch_flux_df<DIM, LAW, kDfResidual>(m, mat, m.su, w, ustar, ubq, ubf, nullptr, flux, st);
    }
  }
  if (ev) cudaEventRecord(ev[2], st);
  if (m.mscale)
    k_cell_avg<DIM, true><<<(unsigned)((m.nc + 127) / 128), 128, 0, st>>>(m, w, m.wst, m.inert);
  const unsigned cgrid = (unsigned)((m.nc + 255) / 256);
  by_faces_per_cell<DIM>(m, [&](auto nlf) {
    constexpr int NLF = decltype(nlf)::value;
    k_cell<DIM, NLF><<<cgrid, 256, 0, st>>>(m, flux, src, R0, d_eps, out);
  });
  if (ev) cudaEventRecord(ev[3], st);
}

template <int DIM, int LAW>
static void jv_impl_df(const DevMesh& m, const Material& mat, const double* v,
                       const double* d_eps, double* out, double* flux, cudaStream_t st,
                       cudaEvent_t* ev) {
  if (ev) cudaEventRecord(ev[0], st);
  v = split_state<DIM>(m, v, m.vext, m.sv, st);
  launch_ustar_df<DIM>(m, m.sv, v, m.ustar_v, st);
  if (ev) cudaEventRecord(ev[1], st);
  if (m.nftile > 0) {
    if (LAW == HOFV_LAW_LINEAR && m.tco)
      k_tflux_hom<DIM><<<(unsigned)m.nftile, 32 * DIM, 0, st>>>(m, m.tco, mat.alpha * mat.kbar, v,
                                                                m.ustar_v, flux);
    else if (LAW == HOFV_LAW_LINEAR)
      launch_flux_df<DIM, LAW, kDfHomog>(m, mat, m.sv, v, m.ustar_v, nullptr, nullptr, nullptr,
                                         flux, st);
    else
      launch_flux_df<DIM, LAW, kDfJv>(m, mat, m.sv, v, m.ustar_v, nullptr, nullptr, d_eps, flux,
                                      st);
  }
  if (ev) cudaEventRecord(ev[2], st);
  if (m.mscale)
    k_cell_avg<DIM, true><<<(unsigned)((m.nc + 127) / 128), 128, 0, st>>>(m, v, m.wst, m.inert);
  const unsigned cgrid = (unsigned)((m.nc + 255) / 256);
  by_faces_per_cell<DIM>(m, [&](auto nlf) {
    constexpr int NLF = decltype(nlf)::value;
    if (LAW == HOFV_LAW_LINEAR)  // the homogeneous residual: J v itself
      k_cell<DIM, NLF><<<cgrid, 256, 0, st>>>(m, flux, nullptr, nullptr, nullptr, out);
    else
      k_cell_diff<DIM, NLF><<<cgrid, 256, 0, st>>>(m, flux, d_eps, out);
  });
  if (ev) cudaEventRecord(ev[3], st);
}

void launch_residual_df(const DevMesh& m, const Material& mat, const double* w,
                        const double* d_eps, const double* R0, double* out, double* ustar,
                        double* flux, const double* ubq, const double* ubf, const double* src,
                        cudaStream_t st, cudaEvent_t* ev) {
  if (m.dim == 2) {
    if (mat.law == HOFV_LAW_LINEAR)
      residual_impl_df<2, 0>(m, mat, w, d_eps, R0, out, ustar, flux, ubq, ubf, src, st, ev);
    else
      residual_impl_df<2, 1>(m, mat, w, d_eps, R0, out, ustar, flux, ubq, ubf, src, st, ev);
  } else {
    if (mat.law == HOFV_LAW_LINEAR)
      residual_impl_df<3, 0>(m, mat, w, d_eps, R0, out, ustar, flux, ubq, ubf, src, st, ev);
    else
      residual_impl_df<3, 1>(m, mat, w, d_eps, R0, out, ustar, flux, ubq, ubf, src, st, ev);
  }
}

void launch_jv_df(const DevMesh& m, const Material& mat, const double* v, const double* d_eps,
                  double* out, double* flux, cudaStream_t st, cudaEvent_t* ev) {
  if (m.dim == 2) {
    if (mat.law == HOFV_LAW_LINEAR)
      jv_impl_df<2, 0>(m, mat, v, d_eps, out, flux, st, ev);
    else
      jv_impl_df<2, 1>(m, mat, v, d_eps, out, flux, st, ev);
  } else {
    if (mat.law == HOFV_LAW_LINEAR)
      jv_impl_df<3, 0>(m, mat, v, d_eps, out, flux, st, ev);
    else
      jv_impl_df<3, 1>(m, mat, v, d_eps, out, flux, st, ev);
  }
}

// the face kernels' differences and limbs exceed the default 48 KB of dynamic
// shared memory for large stencils: raise the limit of every instantiation to what
// kMaxS stencil cells need.  The limit belongs to the device, so each set-up
// raises it on its own (0.04 ms; never during stream capture)
template <int DIM, int LAW, int MODE, int QD, bool PACK>
static void raise_smem(cudaError_t& e) {
  const cudaError_t r =
      cudaFuncSetAttribute((const void*)k_flux_df<DIM, LAW, MODE, QD, PACK>,
                           cudaFuncAttributeMaxDynamicSharedMemorySize,
                           (int)df_smem_bytes<DIM, QD, PACK>(kMaxS));
  if (r != cudaSuccess) e = r;
}
template <int DIM, int QD, bool PACK = false>
static void raise_smem_all(cudaError_t& e) {
  raise_smem<DIM, 0, kDfResidual, QD, PACK>(e);
  raise_smem<DIM, 1, kDfResidual, QD, PACK>(e);
  raise_smem<DIM, 0, kDfHomog, QD, PACK>(e);
  raise_smem<DIM, 1, kDfFill, QD, PACK>(e);
  raise_smem<DIM, 1, kDfJv, QD, PACK>(e);
}
template <typename K>
static void raise_smem_fx(cudaError_t& e, K* kernel, size_t bytes) {
  const cudaError_t r =
      cudaFuncSetAttribute((const void*)kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
  if (r != cudaSuccess) e = r;
}
template <int DIM, int NLF>
static void raise_smem_ustar(cudaError_t& e) {
  raise_smem_fx(e, k_ustar<DIM, NLF>, UstarShape<DIM, NLF>::smem(kMaxS));
}
template <int DIM, int Q>
static void raise_smem_flux(cudaError_t& e) {
  raise_smem_fx(e, k_flux<DIM, HOFV_LAW_LINEAR, Q>, FluxShape<DIM, Q>::smem(kMaxS));
  raise_smem_fx(e, k_flux<DIM, HOFV_LAW_NEOHOOKEAN, Q>, FluxShape<DIM, Q>::smem(kMaxS));
}
int setup_face_kernels() {
  cudaError_t e = cudaSuccess;
  raise_smem_ustar<2, 3>(e);
  raise_smem_ustar<2, 4>(e);
  raise_smem_ustar<2, kPolyMaxSides>(e);
  raise_smem_ustar<3, 4>(e);
  raise_smem_ustar<3, 6>(e);
  raise_smem_ustar<3, kPolyhedronMaxFaces>(e);
  raise_smem_flux<2, 1>(e);
  raise_smem_flux<2, 2>(e);
  raise_smem_flux<2, 3>(e);
  raise_smem_flux<2, 4>(e);
  raise_smem_flux<3, 1>(e);
  raise_smem_flux<3, 4>(e);
  raise_smem_flux<3, 9>(e);
  raise_smem_flux<3, 8>(e);
  raise_smem_flux<3, 16>(e);
  raise_smem_flux<3, 32>(e);
  raise_smem_all<2, 1>(e);
  raise_smem_all<2, 2>(e);
  raise_smem_all<2, 3>(e);
  raise_smem_all<2, 4>(e);
  raise_smem_all<3, 1>(e);
  raise_smem_all<3, 4>(e);
  raise_smem_all<3, 9>(e);
  raise_smem_all<3, 8>(e);
  raise_smem_all<3, 16>(e);
  raise_smem_all<3, 32, true>(e);
  return e == cudaSuccess ? 0 : (int)e;
}

void launch_jv_cache_fill(const DevMesh& m, const Material& mat, const double* u,
                          const double* ubq, cudaStream_t st) {
  if (m.nftile == 0) return;
  if (m.dim == 2) {
    const double* w = split_state<2>(m, u, m.wext, m.su, st);
    launch_flux_df<2, 1, kDfFill>(m, mat, m.su, w, nullptr, ubq, nullptr, nullptr, nullptr, st);
  } else {
    const double* w = split_state<3>(m, u, m.wext, m.su, st);
    launch_flux_df<3, 1, kDfFill>(m, mat, m.su, w, nullptr, ubq, nullptr, nullptr, nullptr, st);
  }
}

}  // namespace hofv
