// Levels held by one CTA in 2 x 2 blocks of fine points: block (bi, bj) holds
//   A = (2bi+1, 2bj+1), B = (2bi+2, 2bj+1), C = (2bi+1, 2bj+2), D = (2bi+2, 2bj+2),
// one point of each Gauss-Seidel colour in the sweep's order, and coincides
// with the coarse cell (bi+1, bj+1) of the interpolation (A its centre, C its
// x-edge point, B its y-edge point, D its coarse point).  One thread owns a
// block for the whole of a sweep sequence: its coefficients stay in registers,
// and the four colours live in four planes of shared memory of (blocks + 2)
// entries per side, so that a colour phase reads its neighbours from planes
// that no thread is writing, without bank conflicts, and stores one value.
// Every row sum takes the operands and the order of row_residual.
#pragma once

#include "cycle_device.cuh"

namespace bmg {
namespace dev {

template <typename T>
struct BlockCoef {
  T aw, as, asw, anw, ad;   // the couplings W, S, SW, NW and 1/a_O of A, B, C, D
  T bw, bs, bsw, bnw, bd;
  T cw, cs, csw, cnw, cd;
  T dw, ds, dsw, dnw, dd;
  T be, de;                 // E couplings of B and D (W of the blocks to the right)
  T cn, dn;                 // N couplings of C and D (S of the blocks above)
  T bne, cne, dne;          // NE couplings of B, C, D
  T ase, bse, dse;          // SE couplings of A, B, D
};

// get(plane, i, j): plane 1 .. 5 = W, S, SW, NW, D at fine point (i, j).  vb,
// vd ... say which of the block's points are interior; the couplings of the
// others are not read.
template <typename T, typename G>
__device__ __forceinline__ void block_coef(BlockCoef<T>& k, int i, int j, bool va, bool vb, bool vc, bool vd, G&& get) {
  k = BlockCoef<T>{};
  if (va) {
    k.aw = get(1, i, j), k.as = get(2, i, j), k.asw = get(3, i, j), k.anw = get(4, i, j), k.ad = get(5, i, j);
    k.ase = get(4, i + 1, j - 1);
    // couplings of B, C and D that are A's to the east, north and north-east
    k.bw = get(1, i + 1, j), k.cs = get(2, i, j + 1), k.dsw = get(3, i + 1, j + 1);
  }
  if (vb) {
    k.bs = get(2, i + 1, j), k.bsw = get(3, i + 1, j), k.bd = get(5, i + 1, j);
    k.be = get(1, i + 2, j), k.bne = get(3, i + 2, j + 1), k.bse = get(4, i + 2, j - 1);
    k.ds = get(2, i + 1, j + 1);
  }
  if (va) k.bnw = get(4, i + 1, j);   // B's NW coupling, C's SE coupling
  if (vc) {
    k.cw = get(1, i, j + 1), k.csw = get(3, i, j + 1), k.cnw = get(4, i, j + 1), k.cd = get(5, i, j + 1);
    k.cn = get(2, i, j + 2), k.cne = get(3, i + 1, j + 2);
    k.dw = get(1, i + 1, j + 1);
  }
  if (vd) {
    k.dnw = get(4, i + 1, j + 1), k.dd = get(5, i + 1, j + 1);
    k.de = get(1, i + 2, j + 1), k.dn = get(2, i + 1, j + 2);
    k.dne = get(3, i + 2, j + 2), k.dse = get(4, i + 2, j);
  }
}

// The four colour planes of a level and this thread's entry in them.
template <typename T>
struct BlockPlanes {
  T *a, *b, *c, *d;   // at the thread's own entry
  int p;              // plane pitch (blocks + 2)
};

template <typename T>
__device__ __forceinline__ BlockPlanes<T> block_planes(T* base, int pitch, int rows, int bi, int bj) {
  const int e = (bj + 1) * pitch + bi + 1, ps = pitch * rows;
  return {base + e, base + ps + e, base + 2 * ps + e, base + 3 * ps + e, pitch};
}

template <typename T>
struct BlockX {
  T a, b, c, d;
};

// s minus the couplings of A (B, C, D) to its neighbours, in the canonical order.
template <bool NINE, bool FU, typename T>
__device__ __forceinline__ T block_sum_a(T s, const BlockCoef<T>& k, const BlockX<T>& x, const BlockPlanes<T>& q) {
  s = msub<FU>(s, k.aw, q.b[-1]);
  s = msub<FU>(s, k.bw, x.b);
  s = msub<FU>(s, k.as, q.c[-q.p]);
  s = msub<FU>(s, k.cs, x.c);
  if (NINE) {
    s = msub<FU>(s, k.asw, q.d[-q.p - 1]);
    s = msub<FU>(s, k.dsw, x.d);
    s = msub<FU>(s, k.anw, q.d[-1]);
    s = msub<FU>(s, k.ase, q.d[-q.p]);
  }
  return s;
}
template <bool NINE, bool FU, typename T>
__device__ __forceinline__ T block_sum_b(T s, const BlockCoef<T>& k, const BlockX<T>& x, const BlockPlanes<T>& q) {
  s = msub<FU>(s, k.bw, x.a);
  s = msub<FU>(s, k.be, q.a[1]);
  s = msub<FU>(s, k.bs, q.d[-q.p]);
  s = msub<FU>(s, k.ds, x.d);
  if (NINE) {
    s = msub<FU>(s, k.bsw, q.c[-q.p]);
    s = msub<FU>(s, k.bne, q.c[1]);
    s = msub<FU>(s, k.bnw, x.c);
    s = msub<FU>(s, k.bse, q.c[1 - q.p]);
  }
  return s;
}
template <bool NINE, bool FU, typename T>
__device__ __forceinline__ T block_sum_c(T s, const BlockCoef<T>& k, const BlockX<T>& x, const BlockPlanes<T>& q) {
  s = msub<FU>(s, k.cw, q.d[-1]);
  s = msub<FU>(s, k.dw, x.d);
  s = msub<FU>(s, k.cs, x.a);
  s = msub<FU>(s, k.cn, q.a[q.p]);
  if (NINE) {
    s = msub<FU>(s, k.csw, q.b[-1]);
    s = msub<FU>(s, k.cne, q.b[q.p]);
    s = msub<FU>(s, k.cnw, q.b[q.p - 1]);
    s = msub<FU>(s, k.bnw, x.b);
  }
  return s;
}
template <bool NINE, bool FU, typename T>
__device__ __forceinline__ T block_sum_d(T s, const BlockCoef<T>& k, const BlockX<T>& x, const BlockPlanes<T>& q) {
  s = msub<FU>(s, k.dw, x.c);
  s = msub<FU>(s, k.de, q.c[1]);
  s = msub<FU>(s, k.ds, x.b);
  s = msub<FU>(s, k.dn, q.b[q.p]);
  if (NINE) {
    s = msub<FU>(s, k.dsw, x.a);
    s = msub<FU>(s, k.dne, q.a[q.p + 1]);
    s = msub<FU>(s, k.dnw, q.a[q.p]);
    s = msub<FU>(s, k.dse, q.a[1]);
  }
  return s;
}

// One Gauss-Seidel sweep of the block's points (four colours, or red = A, D
// then black = B, C for 5-point levels).  ZERO: the iterate is zero on entry,
// so the terms of points not yet updated are left out (a term a * 0 changes no
// sum but the sign of a zero one); a dependent FP64 operation costs 63 cycles
// and the first sweep of a coarse level then needs 16 of its 32 terms.  sync()
// orders a phase's stores before the next phase's loads.
template <bool NINE, bool FU, bool ZERO, typename T, typename F>
__device__ __forceinline__ void block_sweep(const BlockCoef<T>& k, const BlockX<T>& f, BlockX<T>& x,
                                            const BlockPlanes<T>& q, bool va, bool vb, bool vc, bool vd, F&& sync) {
  if constexpr (NINE) {
    if (va) {
      x.a = rmul(ZERO ? f.a : block_sum_a<true, FU>(f.a, k, x, q), k.ad);
      *q.a = x.a;
    }
    sync();
    if (vb) {
      T s = f.b;
      if constexpr (ZERO) {
        s = msub<FU>(s, k.bw, x.a);
        s = msub<FU>(s, k.be, q.a[1]);
      } else {
        s = block_sum_b<true, FU>(s, k, x, q);
      }
      x.b = rmul(s, k.bd);
      *q.b = x.b;
    }
    sync();
    if (vc) {
      T s = f.c;
      if constexpr (ZERO) {
        s = msub<FU>(s, k.cs, x.a);
        s = msub<FU>(s, k.cn, q.a[q.p]);
        s = msub<FU>(s, k.csw, q.b[-1]);
        s = msub<FU>(s, k.cne, q.b[q.p]);
        s = msub<FU>(s, k.cnw, q.b[q.p - 1]);
        s = msub<FU>(s, k.bnw, x.b);
      } else {
        s = block_sum_c<true, FU>(s, k, x, q);
      }
      x.c = rmul(s, k.cd);
      *q.c = x.c;
    }
    sync();
    if (vd) {
      x.d = rmul(block_sum_d<true, FU>(f.d, k, x, q), k.dd);
      *q.d = x.d;
    }
    sync();
  } else {
    if (va) {
      x.a = rmul(ZERO ? f.a : block_sum_a<false, FU>(f.a, k, x, q), k.ad);
      *q.a = x.a;
    }
    if (vd) {
      x.d = rmul(ZERO ? f.d : block_sum_d<false, FU>(f.d, k, x, q), k.dd);
      *q.d = x.d;
    }
    sync();
    if (vb) {
      x.b = rmul(block_sum_b<false, FU>(f.b, k, x, q), k.bd);
      *q.b = x.b;
    }
    if (vc) {
      x.c = rmul(block_sum_c<false, FU>(f.c, k, x, q), k.cd);
      *q.c = x.c;
    }
    sync();
  }
}

// Residuals of the block's points (zero at points that are not interior).
template <bool NINE, bool FU, typename T>
__device__ __forceinline__ BlockX<T> block_resid(const BlockCoef<T>& k, const BlockX<T>& o, const BlockX<T>& f,
                                                 const BlockX<T>& x, const BlockPlanes<T>& q, bool va, bool vb,
                                                 bool vc, bool vd) {
  BlockX<T> r{};
  if (va) r.a = block_sum_a<NINE, FU>(msub<FU>(f.a, o.a, x.a), k, x, q);
  if (vb) r.b = block_sum_b<NINE, FU>(msub<FU>(f.b, o.b, x.b), k, x, q);
  if (vc) r.c = block_sum_c<NINE, FU>(msub<FU>(f.c, o.c, x.c), k, x, q);
  if (vd) r.d = block_sum_d<NINE, FU>(msub<FU>(f.d, o.d, x.d), k, x, q);
  return r;
}

// The Fig. 2 restriction at the block's coarse point (its D): planes a, b, c
// hold the residuals.  w(plane, dic, djc): weight at coarse cell (ic + dic, jc + djc).
template <bool FU, typename T, typename W>
__device__ __forceinline__ T block_restrict(const BlockX<T>& r, const BlockPlanes<T>& q, W&& w) {
  T t = rmul(w(CI_LNE, 0, 0), r.a);
  t = madd<FU>(t, w(CI_LA, 0, 0), r.b);
  t = madd<FU>(t, w(CI_LNW, 1, 0), q.a[1]);
  t = madd<FU>(t, w(CI_LR, 0, 0), r.c);
  t = radd(t, r.d);
  t = madd<FU>(t, w(CI_LL, 1, 0), q.c[1]);
  t = madd<FU>(t, w(CI_LSE, 0, 1), q.a[q.p]);
  t = madd<FU>(t, w(CI_LB, 0, 1), q.b[q.p]);
  t = madd<FU>(t, w(CI_LSW, 1, 1), q.a[q.p + 1]);
  return t;
}

// x += P e on the block's points, the interpolated value formed first; e_sw,
// e_se, e_nw, e_ne: the coarse cell's corner values, w(plane): its weights.
template <bool FU, typename T, typename W>
__device__ __forceinline__ void block_interp(BlockX<T>& x, T e_sw, T e_se, T e_nw, T e_ne, bool va, bool vb, bool vc,
                                             bool vd, W&& w) {
  if (vd) x.d = radd(x.d, e_ne);
  if (vc) {
    T t = rmul(w(CI_LL), e_nw);
    t = madd<FU>(t, w(CI_LR), e_ne);
    x.c = radd(x.c, t);
  }
  if (vb) {
    T t = rmul(w(CI_LB), e_se);
    t = madd<FU>(t, w(CI_LA), e_ne);
    x.b = radd(x.b, t);
  }
  if (va) {
    T t = rmul(w(CI_LSW), e_sw);
    t = madd<FU>(t, w(CI_LSE), e_se);
    t = madd<FU>(t, w(CI_LNW), e_nw);
    t = madd<FU>(t, w(CI_LNE), e_ne);
    x.a = radd(x.a, t);
  }
}

// ---- coarsest solve by one warp ---------------------------------------------------------
// L L^T x = f.  m = 9 unknowns (the default coarsest level; 12 or 16 with
// periodic sides): lane i holds
// unknown i's partial sum, a step's quotient goes to the others by shuffle.
// Forward, right-looking: row i subtracts L_ik y_k as soon as y_k is known, the
// increasing-k order of the row-by-row loop.  Backward: row i's terms are
// subtracted in increasing k > i, so its chain starts when x_{i+1} is known; the
// products L_ki x_k of all rows are formed as soon as x_k is.  What is left is a
// chain of 45 differences, 18 products and 18 quotients (quot, four operations
// each), about 63 cycles an operation.
constexpr int COARSE_LANES = 9;
template <int M>
struct CoarseFactor {       // lane i: L(i, k), L(k, i), L(i, i) and its reciprocal
  double row[M], col[M], dg, y, yl;
};
template <int M>
__device__ __forceinline__ void coarse_load(CoarseFactor<M>& c, const double* L) {
  const int lane = threadIdx.x & 31, i = lane < M ? lane : 0;
#pragma unroll
  for (int k = 0; k < M; ++k) {
    c.row[k] = L[i * M + k];
    c.col[k] = L[k * M + i];
  }
  c.dg = L[i * M + i];
}
// lane i < M: f_i in, x_i out (other lanes compute along and are ignored)
template <int M>
__device__ __forceinline__ double coarse_substitute(const CoarseFactor<M>& c, double f) {
  const int lane = threadIdx.x & 31;
  double s = f;
#pragma unroll
  for (int k = 0; k < M; ++k) {
    const double q = quot(s, c.dg, c.y, c.yl);
    const double yk = __shfl_sync(0xffffffffu, q, k);
    s = lane == k ? yk : (lane > k ? rsub(s, rmul(c.row[k], yk)) : s);
  }
  double pr[M], x = s;      // s = y_i
#pragma unroll
  for (int k = M - 1; k >= 0; --k) {
    double t = s;           // lane k: every x_j, j > k, is known
#pragma unroll
    for (int j = 1; j < M; ++j)
      if (j > k) t = rsub(t, pr[j]);
    const double q = quot(t, c.dg, c.y, c.yl);
    if (lane == k) x = q;
    const double xk = __shfl_sync(0xffffffffu, q, k);
    pr[k] = rmul(c.col[k], xk);
  }
  return x;
}

// Any m, one warp, y in memory that the warp can see (m doubles): the same
// order of every row's terms; the backward products of a row in parallel.
template <typename T>
__device__ __forceinline__ void warp_coarse(int n, const double* __restrict__ L, const T* f, T* x, double* y) {
  const int lane = threadIdx.x & 31, m = n * n, ld = n + 2;
  for (int k = lane; k < m; k += 32) y[k] = (double)f[(size_t)(k / n + 1) * ld + (k % n + 1)];
  __syncwarp();
  for (int k = 0; k < m; ++k) {
    const double yk = rdiv(y[k], L[(size_t)k * m + k]);
    for (int i = k + 1 + lane; i < m; i += 32) y[i] = rsub(y[i], rmul(L[(size_t)i * m + k], yk));
    __syncwarp();
    if (lane == 0) y[k] = yk;
  }
  __syncwarp();
  for (int i = m - 1; i >= 0; --i) {
    double s = y[i];
    for (int k0 = i + 1; k0 < m; k0 += 32) {
      const int k = k0 + lane;
      const double p = k < m ? rmul(L[(size_t)k * m + i], y[k]) : 0.0;
      const int cnt = m - k0 < 32 ? m - k0 : 32;
      for (int q = 0; q < cnt; ++q) s = rsub(s, __shfl_sync(0xffffffffu, p, q));
    }
    const double xi = rdiv(s, L[(size_t)i * m + i]);
    __syncwarp();
    if (lane == 0) y[i] = xi;
    __syncwarp();
  }
  for (int k = lane; k < m; k += 32) x[(size_t)(k / n + 1) * ld + (k % n + 1)] = (T)y[k];
  __syncwarp();
}

// The coarsest solve as a launch of its own (one warp).
template <typename T>
__device__ __forceinline__ void coarse_body(int n, const double* __restrict__ L, const T* f, T* x) {
  __shared__ double y[COARSE_M_MAX];
  const int lane = threadIdx.x & 31;
  if (n * n == COARSE_LANES) {
    CoarseFactor<COARSE_LANES> c;
    coarse_load(c, L);
    c.y = quot_recip(c.dg, &c.yl);
    const int p = lane < COARSE_LANES ? (lane / 3 + 1) * 5 + lane % 3 + 1 : 6;
    const T v = (T)coarse_substitute(c, (double)f[p]);
    if (lane < COARSE_LANES) x[p] = v;
  } else {
    warp_coarse<T>(n, L, f, x, y);
  }
}

}  // namespace dev
}  // namespace bmg
