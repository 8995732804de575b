// One level's half of the cycle in one launch: the pre-smoothing sweeps, the
// residual and its restriction (k_level_down), and the interpolation, the
// correction and the post-smoothing sweeps (k_level_up), for the small and
// middle levels, where a launch per colour pair, residual or interpolation
// costs more than its arithmetic (a dependent launch takes about 3 us in the
// cycle's graph, eight of them per level).
//
// Every CTA takes a tile of 32 x rows blocks of 2 x 2 points (block_device.cuh)
// with a halo and computes the halo's points itself: a sweep's value at a block
// depends on old values up to two blocks away along x and one along y (the
// colours c1, c2 of a row, then c3, c4), the residual and restriction on one
// block more, so after nu1 sweeps a tile owns its blocks from 2 nu1 + 1 columns
// and nu1 + 1 rows inside.  Rows of blocks that no owned value depends on any
// more are skipped; a warp is a row.  Values read and written are in different
// arrays, so no CTA reads what another writes in the launch, and every value
// takes the operands and the order of the colour-by-colour sweep.
//
// The stencil and the weights are constant over a solve, so they are loaded
// before the wait for the preceding kernel; k_level_up also loads the level's
// right-hand side and iterate there, which k_level_down (or the restriction
// before it) wrote at least one completed kernel before the preceding one.
#include "block_device.cuh"

namespace bmg {
using namespace dev;
namespace {

constexpr int LEVEL_NBX = 32;   // blocks per tile along x: one warp

template <typename T>
constexpr int level_threads() { return sizeof(T) == 8 ? 512 : 1024; }

template <typename T>
struct LevelBlock {
  BlockCoef<T> k;
  BlockPlanes<T> q;
  size_t p;                     // its point A
  int ld, ty;
  bool va, vb, vc, vd;
};

template <typename T, typename S>
__device__ __forceinline__ void level_block(LevelBlock<T>& B, const StencilView<T, S>& v, int bi, int bj, T* planes) {
  const int nb = (v.n + 1) / 2, rows = blockDim.y;
  B.ld = v.ld;
  B.ty = threadIdx.y;
  B.va = bi >= 0 && bi < nb && bj >= 0 && bj < nb;
  B.vb = B.va && bi < nb - 1;
  B.vc = B.va && bj < nb - 1;
  B.vd = B.vb && B.vc;
  const int i = 2 * bi + 1, j = 2 * bj + 1;
  B.p = B.va ? (size_t)j * v.ld + i : 0;
  B.q = block_planes(planes, LEVEL_NBX + 2, rows + 2, (int)threadIdx.x, (int)threadIdx.y);
  const S* const off[5] = {nullptr, v.W, v.S_, v.SW, v.NW};
  block_coef(B.k, i, j, B.va, B.vb, B.vc, B.vd, [&](int plane, int a, int b) -> T {
    const size_t e = (size_t)b * v.ld + a;
    return plane == 5 ? v.D[e] : cvt<T>(off[plane][e]);
  });
}

template <typename T>
__device__ __forceinline__ BlockX<T> level_values(const LevelBlock<T>& B, const T* g) {
  BlockX<T> x{};
  if (B.va) x.a = g[B.p];
  if (B.vb) x.b = g[B.p + 1];
  if (B.vc) x.c = g[B.p + B.ld];
  if (B.vd) x.d = g[B.p + B.ld + 1];
  return x;
}

template <typename T>
__device__ __forceinline__ void level_planes(const LevelBlock<T>& B, const BlockX<T>& x) {
  *B.q.a = x.a;
  *B.q.b = x.b;
  *B.q.c = x.c;
  *B.q.d = x.d;
}

template <typename T>
__device__ __forceinline__ void level_store(const LevelBlock<T>& B, const BlockX<T>& x, T* out) {
  const size_t ext = (size_t)B.ld * B.ld;
  (void)ext;
  if (B.va && BMG_IN(DBG_STRIP_STORE, B.p, ext)) out[B.p] = x.a;
  if (B.vb && BMG_IN(DBG_STRIP_STORE, B.p + 1, ext)) out[B.p + 1] = x.b;
  if (B.vc && BMG_IN(DBG_STRIP_STORE, B.p + B.ld, ext)) out[B.p + B.ld] = x.c;
  if (B.vd && BMG_IN(DBG_STRIP_STORE, B.p + B.ld + 1, ext)) out[B.p + B.ld + 1] = x.d;
}

// One sweep, final on the rows of blocks lo .. hi: A and B also on row hi + 1,
// which C and D of row hi read; in a 5-point sweep (red A, D, then black B, C)
// A on row hi + 1, read by C, and D on row lo - 1, read by B.
template <bool NINE, bool FU, bool ZERO, typename T>
__device__ __forceinline__ void level_sweep(const LevelBlock<T>& B, const BlockX<T>& f, BlockX<T>& x, int lo, int hi) {
  const bool cd = B.ty >= lo && B.ty <= hi, ab = B.ty >= lo && B.ty <= hi + 1;
  auto sync = [] { __syncthreads(); };
  if constexpr (NINE)
    block_sweep<true, FU, ZERO>(B.k, f, x, B.q, B.va && ab, B.vb && ab, B.vc && cd, B.vd && cd, sync);
  else
    block_sweep<false, FU, ZERO>(B.k, f, x, B.q, B.va && ab, B.vb && cd, B.vc && cd,
                                 B.vd && B.ty >= lo - 1 && B.ty <= hi, sync);
}

template <typename T, typename S, bool NINE, bool FU>
__global__ void __launch_bounds__(level_threads<T>())
    k_level_down(StencilView<T, S> v, const T* __restrict__ ci, const T* __restrict__ f, const T* __restrict__ xin,
                 T* __restrict__ xout, T* __restrict__ fc, T* __restrict__ xc, int nu1, const int* done) {
  extern __shared__ __align__(16) unsigned char level_smem[];
  const int hx = 2 * nu1 + 1, hy = nu1 + 1, rows = blockDim.y;
  const int bi = (int)blockIdx.x * (LEVEL_NBX - 2 * hx) + (int)threadIdx.x - hx;
  const int bj = (int)blockIdx.y * (rows - 2 * hy) + (int)threadIdx.y - hy;
  LevelBlock<T> B;
  level_block(B, v, bi, bj, reinterpret_cast<T*>(level_smem));
  BlockX<T> o = level_values(B, v.O);
  pdl_enter();
  if (stopped(done)) return;
  const BlockX<T> fb = level_values(B, f);
  BlockX<T> x{};
  if (xin) x = level_values(B, xin);
  level_planes(B, x);
  __syncthreads();
  for (int s = 0; s < nu1; ++s) {
    const int rem = nu1 - 1 - s, lo = hy - 1 - rem, hi = rows - hy + rem;
    if (s == 0 && !xin)
      level_sweep<NINE, FU, true>(B, fb, x, lo, hi);
    else
      level_sweep<NINE, FU, false>(B, fb, x, lo, hi);
  }
  const bool own = (int)threadIdx.x >= hx && (int)threadIdx.x < LEVEL_NBX - hx && B.ty >= hy && B.ty < rows - hy;
  const int nc = (v.n - 1) / 2, ldc = nc + 2;
  const size_t psc = plane_size(nc), pc = (size_t)(bj + 1) * ldc + bi + 1;
  const bool rab = B.ty >= hy && B.ty <= rows - hy, rcd = B.ty >= hy && B.ty < rows - hy;
  const BlockX<T> r = block_resid<NINE, FU>(B.k, o, fb, x, B.q, B.va && rab, B.vb && rab, B.vc && rcd, B.vd && rcd);
  if (own) level_store(B, x, xout);
  __syncthreads();
  *B.q.a = r.a;
  *B.q.b = r.b;
  *B.q.c = r.c;
  __syncthreads();
  if (own && B.vd && BMG_IN(DBG_RESTRICT_STORE, pc, (size_t)ldc * ldc)) {
    fc[pc] = block_restrict<FU>(r, B.q, [&](int k, int dic, int djc) {
      return ci[k * psc + pc + (size_t)djc * ldc + dic];
    });
    if (xc) xc[pc] = T(0);
  }
}

template <typename T, typename S, bool NINE, bool FU>
__global__ void __launch_bounds__(level_threads<T>())
    k_level_up(StencilView<T, S> v, const T* __restrict__ ci, const T* ec, const T* __restrict__ f,
               const T* __restrict__ xin, T* __restrict__ xout, int nu2, const int* done) {
  extern __shared__ __align__(16) unsigned char level_smem[];
  const int hx = 2 * nu2, hy = nu2, rows = blockDim.y;
  const int bi = (int)blockIdx.x * (LEVEL_NBX - 2 * hx) + (int)threadIdx.x - hx;
  const int bj = (int)blockIdx.y * (rows - 2 * hy) + (int)threadIdx.y - hy;
  LevelBlock<T> B;
  level_block(B, v, bi, bj, reinterpret_cast<T*>(level_smem));
  const int nc = (v.n - 1) / 2, ldc = nc + 2;
  const size_t psc = plane_size(nc), pc = B.va ? (size_t)(bj + 1) * ldc + bi + 1 : (size_t)ldc + 1;
  T w[8];
#pragma unroll
  for (int k = 0; k < 8; ++k) w[k] = ci[k * psc + pc];
  const BlockX<T> fb = level_values(B, f);
  BlockX<T> x = level_values(B, xin);
  pdl_enter();
  if (stopped(done)) return;
  block_interp<FU>(x, ec[pc - ldc - 1], ec[pc - ldc], ec[pc - 1], ec[pc], B.va, B.vb, B.vc, B.vd,
                   [&](int k) { return w[k]; });
  level_planes(B, x);
  __syncthreads();
  for (int s = 0; s < nu2; ++s) {
    const int rem = nu2 - 1 - s;
    level_sweep<NINE, FU, false>(B, fb, x, hy - rem, rows - 1 - hy + rem);
  }
  if ((int)threadIdx.x >= hx && (int)threadIdx.x < LEVEL_NBX - hx && B.ty >= hy && B.ty < rows - hy)
    level_store(B, x, xout);
}

template <typename T>
size_t level_bytes(int rows) { return (size_t)4 * (LEVEL_NBX + 2) * (rows + 2) * sizeof(T); }

dim3 level_grid(int n, int rows, int hx, int hy) {
  const int nb = (n + 1) / 2, ox = LEVEL_NBX - 2 * hx, oy = rows - 2 * hy;
  return dim3((nb + ox - 1) / ox, (nb + oy - 1) / oy);
}

}  // namespace

template <typename T, typename S>
void launch_level_down(const StencilView<T, S>& v, int kind, const T* ci, const T* f, const T* xin, T* xout, T* fc,
                       T* xc, int nu1, int rows, const int* done, cudaStream_t s) {
  const dim3 g = level_grid(v.n, rows, 2 * nu1 + 1, nu1 + 1), b(LEVEL_NBX, rows);
  const size_t bytes = level_bytes<T>(rows);
  auto go = [&](auto kernel) { pdl_launch(kernel, g, b, bytes, s, v, ci, f, xin, xout, fc, xc, nu1, done); };
  if (kind == 9) {
    if (v.fused) go(k_level_down<T, S, true, true>);
    else go(k_level_down<T, S, true, false>);
  } else {
    if (v.fused) go(k_level_down<T, S, false, true>);
    else go(k_level_down<T, S, false, false>);
  }
  count_launch();
}

template <typename T, typename S>
void launch_level_up(const StencilView<T, S>& v, int kind, const T* ci, const T* ec, const T* f, const T* xin,
                     T* xout, int nu2, int rows, const int* done, cudaStream_t s) {
  const dim3 g = level_grid(v.n, rows, 2 * nu2, nu2), b(LEVEL_NBX, rows);
  const size_t bytes = level_bytes<T>(rows);
  auto go = [&](auto kernel) { pdl_launch(kernel, g, b, bytes, s, v, ci, ec, f, xin, xout, nu2, done); };
  if (kind == 9) {
    if (v.fused) go(k_level_up<T, S, true, true>);
    else go(k_level_up<T, S, true, false>);
  } else {
    if (v.fused) go(k_level_up<T, S, false, true>);
    else go(k_level_up<T, S, false, false>);
  }
  count_launch();
}

#define BMG_INST(T, S)                                                                                               \
  template void launch_level_down<T, S>(const StencilView<T, S>&, int, const T*, const T*, const T*, T*, T*, T*, int, \
                                        int, const int*, cudaStream_t);                                              \
  template void launch_level_up<T, S>(const StencilView<T, S>&, int, const T*, const T*, const T*, const T*, T*,      \
                                      int, int, const int*, cudaStream_t);
BMG_INST(double, double)
BMG_INST(float, float)
BMG_INST(float, __nv_bfloat16)
#undef BMG_INST

}  // namespace bmg
