// Setup kernels of the BoxMG hierarchy (FP64): input preparation, Dendy
// operator-dependent interpolation, the Galerkin coarse operator
// A_c = P^T A P, reciprocal diagonals, the coarsest Cholesky factor and the
// FP32 / BF16 copies used by the mixed-precision cycle.
//
// Every formula keeps the operation order stated in the interface header so
// that results are reproducible bit for bit (no fused multiply-add).
#include "common.cuh"
#include "kernels.h"
#include "rap_device.cuh"

namespace bmg {

namespace {

constexpr int BX = 32, BY = 8;

// Copy a caller stencil (kind 5: O, W, S; kind 9: O, W, S, SW, NW) on an
// nx x ny grid ((ny+2) x (nx+2) planes) into the six-plane layout of the
// n x n level 0, dropping the ghost ring and ghost couplings.  With nx, ny < n
// the caller's points keep their (i, j) and every other interior point gets
// the identity row O = 1 (general sizes: the embedding reading).
__global__ void k_prepare(int n, int nx, int ny, int kind, const double* __restrict__ in, double* __restrict__ st) {
  int i = blockIdx.x * blockDim.x + threadIdx.x;
  int j = blockIdx.y * blockDim.y + threadIdx.y;
  int ld = n + 2;
  if (i > n + 1 || j > n + 1) return;
  size_t ps = plane_size(n), p = (size_t)j * ld + i;
  const size_t psi = (size_t)(nx + 2) * (ny + 2), q = (size_t)j * (nx + 2) + i;
  const bool caller = i >= 1 && i <= nx && j >= 1 && j <= ny;
  const bool extra = !caller && i >= 1 && i <= n && j >= 1 && j <= n;
  double o = extra ? 1.0 : 0.0, w = 0, s = 0, sw = 0, nw = 0;
  if (caller) {
    o = in[q];
    if (i > 1) w = in[psi + q];
    if (j > 1) s = in[2 * psi + q];
    if (kind == 9) {
      if (i > 1 && j > 1) sw = in[3 * psi + q];
      if (i > 1 && j < ny) nw = in[4 * psi + q];
    }
  }
  if (!BMG_IN(DBG_SETUP_STORE, p, ps)) return;
  st[p] = o;
  st[ps + p] = w;
  st[2 * ps + p] = s;
  st[3 * ps + p] = sw;
  st[4 * ps + p] = nw;
  st[5 * ps + p] = 0.0;
}

__global__ void k_dinv(int n, double* __restrict__ st, int* err) {
  int i = blockIdx.x * blockDim.x + threadIdx.x + 1;
  int j = blockIdx.y * blockDim.y + threadIdx.y + 1;
  if (i > n || j > n) return;
  size_t ps = plane_size(n), p = (size_t)j * (n + 2) + i;
  double o = st[p];
  if (!(o > 0.0)) atomicExch(err, 1);
  if (BMG_IN(DBG_SETUP_STORE, p, ps)) st[5 * ps + p] = rdiv(1.0, o);
}

// ---- Dendy interpolation -------------------------------------------------
// x-edge fine point (2ic-1, 2jc), 1 <= ic <= nc+1, 1 <= jc <= nc:
//   D = (a_S + a_O) + a_N, LL = -((a_SW + a_W) + a_NW) / D, LR = -((a_SE + a_E) + a_NE) / D.
// y-edge fine point (2ic, 2jc-1), 1 <= ic <= nc, 1 <= jc <= nc+1:
//   D = (a_W + a_O) + a_E, LB = -((a_SW + a_S) + a_SE) / D, LA = -((a_NW + a_N) + a_NE) / D.
// Outside those ranges the weights are 0 (the point is a ghost point).
// Galerkin operators of coarse levels are not M-matrices in general, so D may
// be negative (the weights then stay a partition of unity); only D = 0 or a
// non-finite D is an error.
struct EdgeW {
  double lo, hi;
};

__device__ __forceinline__ EdgeW xedge(const Planes<double>& A, int ld, int nc, int ic, int jc, int* err) {
  if (ic < 1 || ic > nc + 1 || jc < 1 || jc > nc) return EdgeW{0.0, 0.0};
  size_t p = (size_t)(2 * jc) * ld + (2 * ic - 1);
  double D = radd(radd(A.a<3>(p, ld), A.a<0>(p, ld)), A.a<4>(p, ld));
  if (!(fabs(D) > 0.0) || isinf(D)) atomicExch(err, 2);   // zero or non-finite: no weight exists
  double ll = -rdiv(radd(radd(A.a<5>(p, ld), A.a<1>(p, ld)), A.a<7>(p, ld)), D);
  double lr = -rdiv(radd(radd(A.a<8>(p, ld), A.a<2>(p, ld)), A.a<6>(p, ld)), D);
  return EdgeW{ll, lr};
}

__device__ __forceinline__ EdgeW yedge(const Planes<double>& A, int ld, int nc, int ic, int jc, int* err) {
  if (ic < 1 || ic > nc || jc < 1 || jc > nc + 1) return EdgeW{0.0, 0.0};
  size_t p = (size_t)(2 * jc - 1) * ld + 2 * ic;
  double D = radd(radd(A.a<1>(p, ld), A.a<0>(p, ld)), A.a<2>(p, ld));
  if (!(fabs(D) > 0.0) || isinf(D)) atomicExch(err, 2);   // zero or non-finite: no weight exists
  double lb = -rdiv(radd(radd(A.a<5>(p, ld), A.a<3>(p, ld)), A.a<8>(p, ld)), D);
  double la = -rdiv(radd(radd(A.a<7>(p, ld), A.a<4>(p, ld)), A.a<6>(p, ld)), D);
  return EdgeW{lb, la};
}

// One thread per coarse cell (ic, jc), 1..nc+1 each: its x-edge and y-edge
// points and the centre point (2ic-1, 2jc-1), whose row of A is solved with
// the four edge neighbours already interpolated:
//   LSW = -((a_SW + a_W LB_w) + a_S LL_s) / a_O, LSE = -((a_SE + a_E LB_e) + a_S LR_s) / a_O,
//   LNW = -((a_NW + a_W LA_w) + a_N LL_n) / a_O, LNE = -((a_NE + a_E LA_e) + a_N LR_n) / a_O.
// A CTA's edge points (and the row below, the column to the left) are formed
// once each, into shared memory: FP64 divisions bound this kernel, and a thread
// forming its neighbours' edges again needs twelve of them, now eight.
__global__ void __launch_bounds__(BX* BY) k_dendy(int n, const double* __restrict__ st, double* __restrict__ ci,
                                                  int* err) {
  __shared__ EdgeW sx[BY + 1][BX], sy[BY][BX + 1];   // x-edges of rows jc0 - 1 .., y-edges of columns ic0 - 1 ..
  const int tx = threadIdx.x, ty = threadIdx.y, tid = ty * BX + tx;
  const int ic0 = blockIdx.x * BX, jc0 = blockIdx.y * BY, ic = ic0 + tx, jc = jc0 + ty;
  const int nc = (n - 1) / 2, ldc = nc + 2, ld = n + 2;
  Planes<double> A = planes_at(st, plane_size(n));
  const EdgeW xe = xedge(A, ld, nc, ic, jc, err), ye = yedge(A, ld, nc, ic, jc, err);
  sx[ty + 1][tx] = xe;
  sy[ty][tx + 1] = ye;
  if (tid < BX) sx[0][tid] = xedge(A, ld, nc, ic0 + tid, jc0 - 1, err);
  else if (tid < BX + BY) sy[tid - BX][0] = yedge(A, ld, nc, ic0 - 1, jc0 + tid - BX, err);
  __syncthreads();
  if (ic > nc + 1 || jc > nc + 1) return;
  size_t pc = (size_t)jc * ldc + ic, psc = plane_size(nc);
  if (!BMG_IN(DBG_SETUP_STORE, pc, psc)) return;
  if (ic == 0 || jc == 0) {
#pragma unroll
    for (int k = 0; k < 8; ++k) ci[k * psc + pc] = 0.0;
    return;
  }
  const EdgeW yw = sy[ty][tx];   // west neighbour of the centre
  const EdgeW xs = sx[ty][tx];   // south neighbour of the centre
  size_t p = (size_t)(2 * jc - 1) * ld + (2 * ic - 1);
  double aO = A.a<0>(p, ld), aW = A.a<1>(p, ld), aE = A.a<2>(p, ld), aS = A.a<3>(p, ld), aN = A.a<4>(p, ld);
  double aSW = A.a<5>(p, ld), aNE = A.a<6>(p, ld), aNW = A.a<7>(p, ld), aSE = A.a<8>(p, ld);
  if (!(aO > 0.0)) atomicExch(err, 2);
  double yl;
  const double y = quot_recip(aO, &yl);   // four quotients by one divisor
  double sw = -quot(radd(radd(aSW, rmul(aW, yw.lo)), rmul(aS, xs.lo)), aO, y, yl);
  double se = -quot(radd(radd(aSE, rmul(aE, ye.lo)), rmul(aS, xs.hi)), aO, y, yl);
  double nw = -quot(radd(radd(aNW, rmul(aW, yw.hi)), rmul(aN, xe.lo)), aO, y, yl);
  double ne = -quot(radd(radd(aNE, rmul(aE, ye.hi)), rmul(aN, xe.hi)), aO, y, yl);
  ci[CI_LSW * psc + pc] = sw;
  ci[CI_LSE * psc + pc] = se;
  ci[CI_LNW * psc + pc] = nw;
  ci[CI_LNE * psc + pc] = ne;
  ci[CI_LL * psc + pc] = xe.lo;
  ci[CI_LR * psc + pc] = xe.hi;
  ci[CI_LB * psc + pc] = ye.lo;
  ci[CI_LA * psc + pc] = ye.hi;
}

// One coarse entry per thread: blockIdx.z picks O, W, S, SW or NW (the five
// entries one after the other kept a small level's few threads busy for 21 us).
__global__ void k_rap(int n, const double* __restrict__ st, const double* __restrict__ ci,
                      double* __restrict__ stc) {
  int ic = blockIdx.x * blockDim.x + threadIdx.x;
  int jc = blockIdx.y * blockDim.y + threadIdx.y;
  int nc = (n - 1) / 2, ldc = nc + 2, ld = n + 2;
  if (ic > nc + 1 || jc > nc + 1) return;
  size_t psc = plane_size(nc), pc = (size_t)jc * ldc + ic;
  if (!BMG_IN(DBG_SETUP_STORE, pc, psc)) return;
  if (ic == 0 || jc == 0 || ic == nc + 1 || jc == nc + 1) {
    stc[blockIdx.z * psc + pc] = 0.0;
    if (blockIdx.z == 0) stc[5 * psc + pc] = 0.0;
    return;
  }
  Planes<double> A = planes_at(st, plane_size(n));
  const int k = blockIdx.z;
  double v;
  bool in = true;
  switch (k) {
    case 0: v = rapdev::rap_entry<0, 0>(A, ld, ci, psc, ldc, nc, ic, jc); break;
    case 1: v = rapdev::rap_entry<-1, 0>(A, ld, ci, psc, ldc, nc, ic, jc), in = ic > 1; break;
    case 2: v = rapdev::rap_entry<0, -1>(A, ld, ci, psc, ldc, nc, ic, jc), in = jc > 1; break;
    case 3: v = rapdev::rap_entry<-1, -1>(A, ld, ci, psc, ldc, nc, ic, jc), in = ic > 1 && jc > 1; break;
    default: v = rapdev::rap_entry<-1, 1>(A, ld, ci, psc, ldc, nc, ic, jc), in = ic > 1 && jc < nc; break;
  }
  stc[k * psc + pc] = in ? v : 0.0;
  if (k == 0) stc[5 * psc + pc] = 0.0;
}

// ---- coarsest Cholesky (one CTA; m = n^2 <= 225) --------------------------
// Dense A over lexicographic unknowns, then right-looking Cholesky: for each
// pivot k, L_kk = sqrt(a_kk), L_ik = a_ik / L_kk, then a_ij -= L_ik L_jk for
// j = k+1.., i = j.. (lower triangle), the entries of a step in parallel (one
// thread took 40 us for m = 9).  `a` in shared memory when it fits.
constexpr int FACTOR_SMEM_M = 64;
__global__ void __launch_bounds__(256) k_factor(int n, const double* __restrict__ st, double* __restrict__ L,
                                                double* __restrict__ work, int* err) {
  __shared__ double sa[FACTOR_SMEM_M * FACTOR_SMEM_M];
  const int m = n * n, ld = n + 2;
  double* a = m <= FACTOR_SMEM_M ? sa : work;
  Planes<double> A = planes_at(st, plane_size(n));
  for (int k = threadIdx.x; k < m * m; k += blockDim.x) {
    a[k] = 0.0;
    L[k] = 0.0;
  }
  __syncthreads();
  for (int r = threadIdx.x; r < m; r += blockDim.x) {
    const int i = r % n + 1, j = r / n + 1;
    size_t p = (size_t)j * ld + i;
    double v[9] = {A.a<0>(p, ld), A.a<1>(p, ld), A.a<2>(p, ld), A.a<3>(p, ld), A.a<4>(p, ld),
                   A.a<5>(p, ld), A.a<6>(p, ld), A.a<7>(p, ld), A.a<8>(p, ld)};
    for (int k = 0; k < 9; ++k) {
      int ii = i + nbr_dx(k), jj = j + nbr_dy(k);
      if (ii >= 1 && ii <= n && jj >= 1 && jj <= n) a[(size_t)r * m + (jj - 1) * n + (ii - 1)] = v[k];
    }
  }
  __syncthreads();
  for (int k = 0; k < m; ++k) {
    const double akk = a[(size_t)k * m + k];
    if (!(akk > 0.0)) {
      if (threadIdx.x == 0) atomicExch(err, 3);
      return;
    }
    const double lkk = __dsqrt_rn(akk);
    if (threadIdx.x == 0) L[(size_t)k * m + k] = lkk;
    for (int i = k + 1 + threadIdx.x; i < m; i += blockDim.x)
      L[(size_t)i * m + k] = rdiv(a[(size_t)i * m + k], lkk);
    __syncthreads();
    const int w = m - k - 1;
    for (int e = threadIdx.x; e < w * w; e += blockDim.x) {
      const int i = k + 1 + e / w, j = k + 1 + e % w;
      if (j <= i)
        a[(size_t)i * m + j] = rsub(a[(size_t)i * m + j], rmul(L[(size_t)i * m + k], L[(size_t)j * m + k]));
    }
    __syncthreads();
  }
}

// ---- FP32 / BF16 copies -----------------------------------------------------
__global__ void k_round32(size_t count, const double* __restrict__ in, float* __restrict__ out) {
  for (size_t k = blockIdx.x * (size_t)blockDim.x + threadIdx.x; k < count; k += (size_t)gridDim.x * blockDim.x)
    out[k] = __double2float_rn(in[k]);
}

__device__ __forceinline__ float bf16_of(double v) { return __bfloat162float(__float2bfloat16_rn(__double2float_rn(v))); }

// The FP32 planes O, W, S, SW, NW, D of a level, and (pk) their packed copy
// d, w, s, sw, nw per point, in one pass (seven launches a level before).
__global__ void k_lower32(int n, const double* __restrict__ st, float* __restrict__ st32, float* __restrict__ pk,
                          size_t pst) {
  const size_t ps = plane_size(n);
  for (size_t p = blockIdx.x * (size_t)blockDim.x + threadIdx.x; p < ps; p += (size_t)gridDim.x * blockDim.x) {
    float v[6];
#pragma unroll
    for (int k = 0; k < 6; ++k) {
      v[k] = __double2float_rn(st[k * ps + p]);
      st32[k * pst + p] = v[k];
    }
    if (pk) {
      float* o = pk + PK_WORDS_F32 * p;
      o[0] = v[5];
#pragma unroll
      for (int k = 1; k < 5; ++k) o[k] = v[k];
    }
  }
}

// off16: W, S, SW, NW as bf16(fl32(a)); od32: O32, D32 with
// O32 = fl32(sum_NBR a) - W_b - E_b - S_b - N_b - SW_b - NE_b - NW_b - SE_b, D32 = 1 / O32.
__global__ void k_lower_bf16(int n, const double* __restrict__ st, __nv_bfloat16* __restrict__ off16,
                             float* __restrict__ od32, float* __restrict__ pk, size_t pst) {
  int i = blockIdx.x * blockDim.x + threadIdx.x;
  int j = blockIdx.y * blockDim.y + threadIdx.y;
  int ld = n + 2;
  if (i > n + 1 || j > n + 1) return;
  size_t ps = plane_size(n), p = (size_t)j * ld + i;
  unsigned half[4];
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    const __nv_bfloat16 b = __float2bfloat16_rn(__double2float_rn(st[(k + 1) * ps + p]));
    off16[k * pst + p] = b;
    half[k] = (unsigned)__bfloat16_as_ushort(b);
  }
  unsigned* w = reinterpret_cast<unsigned*>(pk + PK_WORDS_BF16 * p);   // d, w | s << 16, sw | nw << 16
  w[1] = half[0] | (half[1] << 16);
  w[2] = half[2] | (half[3] << 16);
  if (i < 1 || i > n || j < 1 || j > n) {
    od32[p] = 0.0f;
    od32[pst + p] = 0.0f;
    w[0] = 0u;
    return;
  }
  Planes<double> A = planes_at(st, ps);
  double rs = A.a<0>(p, ld);
  rs = radd(rs, A.a<1>(p, ld));
  rs = radd(rs, A.a<2>(p, ld));
  rs = radd(rs, A.a<3>(p, ld));
  rs = radd(rs, A.a<4>(p, ld));
  rs = radd(rs, A.a<5>(p, ld));
  rs = radd(rs, A.a<6>(p, ld));
  rs = radd(rs, A.a<7>(p, ld));
  rs = radd(rs, A.a<8>(p, ld));
  float o = __double2float_rn(rs);
  o = rsub(o, bf16_of(A.a<1>(p, ld)));
  o = rsub(o, bf16_of(A.a<2>(p, ld)));
  o = rsub(o, bf16_of(A.a<3>(p, ld)));
  o = rsub(o, bf16_of(A.a<4>(p, ld)));
  o = rsub(o, bf16_of(A.a<5>(p, ld)));
  o = rsub(o, bf16_of(A.a<6>(p, ld)));
  o = rsub(o, bf16_of(A.a<7>(p, ld)));
  o = rsub(o, bf16_of(A.a<8>(p, ld)));
  const float d = rdiv(1.0f, o);
  od32[p] = o;
  od32[pst + p] = d;
  w[0] = __float_as_uint(d);
}

dim3 grid2(int nx, int ny) { return dim3((nx + BX - 1) / BX, (ny + BY - 1) / BY); }

}  // namespace

// Interior of an nx x ny grid array into / out of the n x n layout (the other
// points of the destination are left as they are).
__global__ void k_embed_vec(int nx, int ny, int n, const double* __restrict__ in, double* __restrict__ out, int back) {
  int i = blockIdx.x * blockDim.x + threadIdx.x + 1;
  int j = blockIdx.y * blockDim.y + threadIdx.y + 1;
  if (i > nx || j > ny) return;
  const size_t pc = (size_t)j * (nx + 2) + i, pn = (size_t)j * (n + 2) + i;
  if (back)
    out[pc] = in[pn];
  else
    out[pn] = in[pc];
}

void launch_embed_vec(int nx, int ny, int n, const double* in, double* out, bool back, cudaStream_t s) {
  k_embed_vec<<<grid2(nx, ny), dim3(BX, BY), 0, s>>>(nx, ny, n, in, out, back ? 1 : 0);
  count_launch();
}

void launch_prepare(int n, int nx, int ny, int kind, const double* coef_in, double* st, int* err, cudaStream_t s) {
  k_prepare<<<grid2(n + 2, n + 2), dim3(BX, BY), 0, s>>>(n, nx, ny, kind, coef_in, st);
  count_launch();
  k_dinv<<<grid2(n, n), dim3(BX, BY), 0, s>>>(n, st, err);
  count_launch();
}

void launch_dendy(int n, const double* st, double* ci, int* err, cudaStream_t s) {
  int nc = (n - 1) / 2;
  k_dendy<<<grid2(nc + 2, nc + 2), dim3(BX, BY), 0, s>>>(n, st, ci, err);
  count_launch();
}

void launch_rap(int n, const double* st, const double* ci, double* stc, cudaStream_t s) {
  int nc = (n - 1) / 2;
  dim3 g = grid2(nc + 2, nc + 2);
  g.z = 5;
  k_rap<<<g, dim3(BX, BY), 0, s>>>(n, st, ci, stc);
  count_launch();
}

void launch_dinv(int n, double* st, int* err, cudaStream_t s) {
  k_dinv<<<grid2(n, n), dim3(BX, BY), 0, s>>>(n, st, err);
  count_launch();
}

void launch_factor(int n, const double* st, double* L, double* work, int* err, cudaStream_t s) {
  k_factor<<<1, 256, 0, s>>>(n, st, L, work, err);
  count_launch();
}

static unsigned blocks_for(size_t count) { return (unsigned)((count + 255) / 256 < 4096 ? (count + 255) / 256 : 4096); }

void launch_round32(size_t count, const double* in, float* out, cudaStream_t s) {
  k_round32<<<blocks_for(count), 256, 0, s>>>(count, in, out);
  count_launch();
}

void launch_lower32(int n, const double* st, float* st32, float* pk, cudaStream_t s) {
  k_lower32<<<blocks_for(plane_size(n)), 256, 0, s>>>(n, st, st32, pk, plane_stride32(n));
  count_launch();
}

void launch_lower_bf16(int n, const double* st, __nv_bfloat16* off16, float* od32, float* pk, cudaStream_t s) {
  k_lower_bf16<<<grid2(n + 2, n + 2), dim3(BX, BY), 0, s>>>(n, st, off16, od32, pk, plane_stride32(n));
  count_launch();
}

}  // namespace bmg
