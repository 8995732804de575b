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
// before the wait for the preceding kernel; everything that a cycle writes is
// loaded after it.
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
  int ld, ty, ic, jc;           // ic, jc: its coarse cell
  bool va, vb, vc, vd;
};

// A level's blocks: Dirichlet axes of n = 2 blocks - 1 points, whose last block
// lacks its even points, and (PER) periodic axes of 2 blocks points, whose
// block, point and coarse indexes wrap around; a tile wider than such an axis
// holds copies of its blocks, of which the first is the one that owns.
template <bool PER>
struct LevelMap {
  LevelGrid g;
  int nbx, nby, ncx, ncy;
  __device__ __forceinline__ explicit LevelMap(const LevelGrid& grid) : g(grid) {
    nbx = (g.nx + 1) / 2, nby = (g.ny + 1) / 2;
    ncx = PER && g.px ? g.nx / 2 : (g.nx - 1) / 2, ncy = PER && g.py ? g.ny / 2 : (g.ny - 1) / 2;
  }
  static __device__ __forceinline__ int wrap(int k, int n) { return k < 1 ? k + n : (k > n ? k - n : k); }   // 1 .. n
  __device__ __forceinline__ int bx(int b) const { return PER && g.px ? (b % nbx + nbx) % nbx : b; }
  __device__ __forceinline__ int by(int b) const { return PER && g.py ? (b % nby + nby) % nby : b; }
  __device__ __forceinline__ bool last_x(int b) const { return !(PER && g.px) && b == nbx - 1; }
  __device__ __forceinline__ bool last_y(int b) const { return !(PER && g.py) && b == nby - 1; }
  __device__ __forceinline__ size_t at(int i, int j) const {
    if (PER && g.px) i = wrap(i, g.nx);
    if (PER && g.py) j = wrap(j, g.ny);
    return (size_t)j * (g.nx + 2) + i;
  }
  __device__ __forceinline__ size_t coarse(int ic, int jc) const {
    if (PER && g.px) ic = wrap(ic, ncx);
    if (PER && g.py) jc = wrap(jc, ncy);
    return (size_t)jc * (ncx + 2) + ic;
  }
  __device__ __forceinline__ size_t psc() const { return (size_t)(ncx + 2) * (ncy + 2); }
};

// ux, uy: the thread's block before wrapping.
template <bool PER, typename T, typename S>
__device__ __forceinline__ void level_block(LevelBlock<T>& B, const StencilView<T, S>& v, const LevelMap<PER>& m,
                                            int ux, int uy, T* planes) {
  const int bi = m.bx(ux), bj = m.by(uy);
  B.ld = m.g.nx + 2;
  B.ty = threadIdx.y;
  B.va = bi >= 0 && bi < m.nbx && bj >= 0 && bj < m.nby;
  B.vb = B.va && !m.last_x(bi);
  B.vc = B.va && !m.last_y(bj);
  B.vd = B.vb && B.vc;
  B.ic = bi + 1;
  B.jc = bj + 1;
  const int i = 2 * bi + 1, j = 2 * bj + 1;
  B.p = B.va ? (size_t)j * B.ld + i : 0;
  B.q = block_planes(planes, LEVEL_NBX + 2, (int)blockDim.y + 2, (int)threadIdx.x, (int)threadIdx.y);
  const S* const off[5] = {nullptr, v.W, v.S_, v.SW, v.NW};
  block_coef(B.k, i, j, B.va, B.vb, B.vc, B.vd, [&](int plane, int a, int b) -> T {
    const size_t e = m.at(a, b);
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
__device__ __forceinline__ void level_store(const LevelBlock<T>& B, const BlockX<T>& x, T* out, size_t ext) {
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

template <typename T, typename S, bool NINE, bool FU, bool PER>
__device__ __forceinline__ void down_body(const StencilView<T, S>& v, const LevelGrid& grid, const T* __restrict__ ci,
                                          const T* __restrict__ f, const T* __restrict__ xin, T* __restrict__ xout,
                                          T* __restrict__ fc, T* __restrict__ xc, int nu1, const int* done) {
  extern __shared__ __align__(16) unsigned char level_smem[];
  const LevelMap<PER> m(grid);
  const int hx = 2 * nu1 + 1, hy = nu1 + 1, rows = blockDim.y;
  const int ux = (int)blockIdx.x * (LEVEL_NBX - 2 * hx) + (int)threadIdx.x - hx;
  const int uy = (int)blockIdx.y * (rows - 2 * hy) + (int)threadIdx.y - hy;
  LevelBlock<T> B;
  level_block(B, v, m, ux, uy, reinterpret_cast<T*>(level_smem));
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
  const bool own = (int)threadIdx.x >= hx && (int)threadIdx.x < LEVEL_NBX - hx && B.ty >= hy && B.ty < rows - hy &&
                   ux < m.nbx && uy < m.nby;
  const size_t psc = m.psc(), pc = (size_t)B.jc * (m.ncx + 2) + B.ic;
  const bool rab = B.ty >= hy && B.ty <= rows - hy, rcd = B.ty >= hy && B.ty < rows - hy;
  const BlockX<T> r = block_resid<NINE, FU>(B.k, o, fb, x, B.q, B.va && rab, B.vb && rab, B.vc && rcd, B.vd && rcd);
  if (own) level_store(B, x, xout, (size_t)B.ld * (grid.ny + 2));
  __syncthreads();
  *B.q.a = r.a;
  *B.q.b = r.b;
  *B.q.c = r.c;
  __syncthreads();
  if (own && B.vd && BMG_IN(DBG_RESTRICT_STORE, pc, psc)) {
    fc[pc] = block_restrict<FU>(r, B.q, [&](int k, int dic, int djc) {
      return ci[k * psc + m.coarse(B.ic + dic, B.jc + djc)];
    });
    if (xc) xc[pc] = T(0);
  }
}

template <typename T, typename S, bool NINE, bool FU, bool PER>
__device__ __forceinline__ void up_body(const StencilView<T, S>& v, const LevelGrid& grid, const T* __restrict__ ci,
                                        const T* ec, const T* __restrict__ f, const T* __restrict__ xin,
                                        T* __restrict__ xout, int nu2, const int* done) {
  extern __shared__ __align__(16) unsigned char level_smem[];
  const LevelMap<PER> m(grid);
  const int hx = 2 * nu2, hy = nu2, rows = blockDim.y;
  const int ux = (int)blockIdx.x * (LEVEL_NBX - 2 * hx) + (int)threadIdx.x - hx;
  const int uy = (int)blockIdx.y * (rows - 2 * hy) + (int)threadIdx.y - hy;
  LevelBlock<T> B;
  level_block(B, v, m, ux, uy, reinterpret_cast<T*>(level_smem));
  const int ic = B.va ? B.ic : 1, jc = B.va ? B.jc : 1;
  const size_t psc = m.psc(), pc = (size_t)jc * (m.ncx + 2) + ic;
  T w[8];
#pragma unroll
  for (int k = 0; k < 8; ++k) w[k] = ci[k * psc + pc];
  pdl_enter();
  if (stopped(done)) return;
  const BlockX<T> fb = level_values(B, f);
  BlockX<T> x = level_values(B, xin);
  block_interp<FU>(x, ec[m.coarse(ic - 1, jc - 1)], ec[m.coarse(ic, jc - 1)], ec[m.coarse(ic - 1, jc)],
                   ec[m.coarse(ic, jc)], B.va, B.vb, B.vc, B.vd, [&](int k) { return w[k]; });
  level_planes(B, x);
  __syncthreads();
  for (int s = 0; s < nu2; ++s) {
    const int rem = nu2 - 1 - s;
    level_sweep<NINE, FU, false>(B, fb, x, hy - rem, rows - 1 - hy + rem);
  }
  if ((int)threadIdx.x >= hx && (int)threadIdx.x < LEVEL_NBX - hx && B.ty >= hy && B.ty < rows - hy && ux < m.nbx &&
      uy < m.nby)
    level_store(B, x, xout, (size_t)B.ld * (grid.ny + 2));
}

template <typename T, typename S, bool NINE, bool FU, bool PER>
__global__ void __launch_bounds__(level_threads<T>())
    k_level_down(StencilView<T, S> v, LevelGrid grid, const T* __restrict__ ci, const T* __restrict__ f,
                 const T* __restrict__ xin, T* __restrict__ xout, T* __restrict__ fc, T* __restrict__ xc, int nu1,
                 const int* done) {
  down_body<T, S, NINE, FU, PER>(v, grid, ci, f, xin, xout, fc, xc, nu1, done);
}

template <typename T, typename S, bool NINE, bool FU, bool PER>
__global__ void __launch_bounds__(level_threads<T>())
    k_level_up(StencilView<T, S> v, LevelGrid grid, const T* __restrict__ ci, const T* ec, const T* __restrict__ f,
               const T* __restrict__ xin, T* __restrict__ xout, int nu2, const int* done) {
  up_body<T, S, NINE, FU, PER>(v, grid, ci, ec, f, xin, xout, nu2, done);
}

// One problem of a batched stage per blockIdx.z; the iterate goes x -> x2 -> x.
template <typename T, typename S, bool NINE, bool FU>
__global__ void __launch_bounds__(level_threads<T>()) k_level_down_b(const LevelDesc<T, S>* __restrict__ d, int nu1) {
  const LevelDesc<T, S>& q = d[blockIdx.z];
  down_body<T, S, NINE, FU, false>(q.v, LevelGrid{q.v.n, q.v.n, 0, 0}, q.ci, q.f, q.zero ? nullptr : q.x, q.x2, q.fc,
                                   q.xc, nu1, q.done);
}

template <typename T, typename S, bool NINE, bool FU>
__global__ void __launch_bounds__(level_threads<T>()) k_level_up_b(const LevelDesc<T, S>* __restrict__ d, int nu2) {
  const LevelDesc<T, S>& q = d[blockIdx.z];
  up_body<T, S, NINE, FU, false>(q.v, LevelGrid{q.v.n, q.v.n, 0, 0}, q.ci, q.xc, q.f, q.x2, q.x, nu2, q.done);
}

template <typename T>
size_t level_bytes(int rows) { return (size_t)4 * (LEVEL_NBX + 2) * (rows + 2) * sizeof(T); }

dim3 level_grid(const LevelGrid& g, int rows, int hx, int hy) {
  const int nbx = (g.nx + 1) / 2, nby = (g.ny + 1) / 2, ox = LEVEL_NBX - 2 * hx, oy = rows - 2 * hy;
  return dim3((nbx + ox - 1) / ox, (nby + oy - 1) / oy);
}

template <typename T, typename S, bool PER>
void down(const StencilView<T, S>& v, const LevelGrid& grid, int kind, const T* ci, const T* f, const T* xin, T* xout,
          T* fc, T* xc, int nu1, int rows, const int* done, cudaStream_t s) {
  const dim3 g = level_grid(grid, rows, 2 * nu1 + 1, nu1 + 1), b(LEVEL_NBX, rows);
  const size_t bytes = level_bytes<T>(rows);
  auto go = [&](auto kernel) { pdl_launch(kernel, g, b, bytes, s, v, grid, ci, f, xin, xout, fc, xc, nu1, done); };
  if (kind == 9)
    v.fused ? go(k_level_down<T, S, true, true, PER>) : go(k_level_down<T, S, true, false, PER>);
  else
    v.fused ? go(k_level_down<T, S, false, true, PER>) : go(k_level_down<T, S, false, false, PER>);
  count_launch();
}

template <typename T, typename S, bool PER>
void up(const StencilView<T, S>& v, const LevelGrid& grid, int kind, const T* ci, const T* ec, const T* f,
        const T* xin, T* xout, int nu2, int rows, const int* done, cudaStream_t s) {
  const dim3 g = level_grid(grid, rows, 2 * nu2, nu2), b(LEVEL_NBX, rows);
  const size_t bytes = level_bytes<T>(rows);
  auto go = [&](auto kernel) { pdl_launch(kernel, g, b, bytes, s, v, grid, ci, ec, f, xin, xout, nu2, done); };
  if (kind == 9)
    v.fused ? go(k_level_up<T, S, true, true, PER>) : go(k_level_up<T, S, true, false, PER>);
  else
    v.fused ? go(k_level_up<T, S, false, true, PER>) : go(k_level_up<T, S, false, false, PER>);
  count_launch();
}

}  // namespace

// Block rows per tile of a level whose halves of the cycle run as one launch
// each (0: its steps are launched separately).  The change of a whole cycle
// when one level runs by halves, us, fused arithmetic (8 / 16 / 32 rows):
//   FP64  63: -15 / -6    127: -12 / -4    255: -3 / -10   511: 0 / -17   1023: +121 / +55
//   FP32  127: -11 / -11 / -11   255: -14 / -13 / -11   511: -12 / -15 / -17
//         1023: +4 / -13 / -9    2047: +66 / -2 / +12
// (one rounding per operation: within a few us of these).  Small FP64 levels
// want few warps per SM quarter, each of whose FP64 instructions takes 60
// cycles; larger ones a small halo.  In FP32 32 rows pay while their tiles,
// one to an SM, fit the chip at once.
int level_rows(bool f64, int n) {
  if (f64) return n > 512 ? 0 : n <= 128 ? 8 : 16;
  return n > 1023 ? 0 : n == 511 ? 32 : 16;
}

template <typename T, typename S>
void launch_level_down(const StencilView<T, S>& v, int kind, const T* ci, const T* f, const T* xin, T* xout, T* fc,
                       T* xc, int nu1, int rows, const int* done, cudaStream_t s) {
  down<T, S, false>(v, LevelGrid{v.n, v.n, 0, 0}, kind, ci, f, xin, xout, fc, xc, nu1, rows, done, s);
}

template <typename T, typename S>
void launch_level_up(const StencilView<T, S>& v, int kind, const T* ci, const T* ec, const T* f, const T* xin,
                     T* xout, int nu2, int rows, const int* done, cudaStream_t s) {
  up<T, S, false>(v, LevelGrid{v.n, v.n, 0, 0}, kind, ci, ec, f, xin, xout, nu2, rows, done, s);
}

void launch_level_down_p(const StencilView<double, double>& v, const LevelGrid& grid, int kind, const double* ci,
                         const double* f, const double* xin, double* xout, double* fc, double* xc, int nu1, int rows,
                         const int* done, cudaStream_t s) {
  down<double, double, true>(v, grid, kind, ci, f, xin, xout, fc, xc, nu1, rows, done, s);
}

void launch_level_up_p(const StencilView<double, double>& v, const LevelGrid& grid, int kind, const double* ci,
                       const double* ec, const double* f, const double* xin, double* xout, int nu2, int rows,
                       const int* done, cudaStream_t s) {
  up<double, double, true>(v, grid, kind, ci, ec, f, xin, xout, nu2, rows, done, s);
}

template <typename T, typename S>
void launch_level_down_b(const LevelDesc<T, S>* d, int count, int n, int kind, int nu1, int rows, cudaStream_t s,
                         int fused) {
  dim3 g = level_grid(LevelGrid{n, n, 0, 0}, rows, 2 * nu1 + 1, nu1 + 1);
  g.z = count;
  auto go = [&](auto kernel) { pdl_launch(kernel, g, dim3(LEVEL_NBX, rows), level_bytes<T>(rows), s, d, nu1); };
  if (kind == 9)
    fused ? go(k_level_down_b<T, S, true, true>) : go(k_level_down_b<T, S, true, false>);
  else
    fused ? go(k_level_down_b<T, S, false, true>) : go(k_level_down_b<T, S, false, false>);
  count_launch();
}

template <typename T, typename S>
void launch_level_up_b(const LevelDesc<T, S>* d, int count, int n, int kind, int nu2, int rows, cudaStream_t s,
                       int fused) {
  dim3 g = level_grid(LevelGrid{n, n, 0, 0}, rows, 2 * nu2, nu2);
  g.z = count;
  auto go = [&](auto kernel) { pdl_launch(kernel, g, dim3(LEVEL_NBX, rows), level_bytes<T>(rows), s, d, nu2); };
  if (kind == 9)
    fused ? go(k_level_up_b<T, S, true, true>) : go(k_level_up_b<T, S, true, false>);
  else
    fused ? go(k_level_up_b<T, S, false, true>) : go(k_level_up_b<T, S, false, false>);
  count_launch();
}

#define BMG_INST(T, S)                                                                                               \
  template void launch_level_down<T, S>(const StencilView<T, S>&, int, const T*, const T*, const T*, T*, T*, T*, int, \
                                        int, const int*, cudaStream_t);                                              \
  template void launch_level_up<T, S>(const StencilView<T, S>&, int, const T*, const T*, const T*, const T*, T*,      \
                                      int, int, const int*, cudaStream_t);                                           \
  template void launch_level_down_b<T, S>(const LevelDesc<T, S>*, int, int, int, int, int, cudaStream_t, int);        \
  template void launch_level_up_b<T, S>(const LevelDesc<T, S>*, int, int, int, int, int, cudaStream_t, int);
BMG_INST(double, double)
BMG_INST(float, float)
BMG_INST(float, __nv_bfloat16)
#undef BMG_INST

}  // namespace bmg
