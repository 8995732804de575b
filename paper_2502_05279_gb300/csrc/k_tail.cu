// The level-fused tail: the V-cycle from a small level down to the coarsest and
// back in one CTA per problem.
//
// What bounds it.  A colour phase of a level this small is a dependent chain
// (nine FP64 operations of 63 cycles each, or seventeen with one rounding per
// operation) between two barriers, and only one SM's warps share it, so the
// launch is worth its latency only if a phase waits for little else.  The
// stencils, weights and the Cholesky factor are constant over a solve: they are
// staged in shared memory before the wait for the preceding kernel.  A thread
// owns a 2 x 2 block of points (block_device.cuh), takes the block's
// coefficients into registers once per leg of the cycle, and a phase reads its
// neighbours' values only; barriers span the warps that hold the level's
// blocks and no more.
#include "block_device.cuh"

namespace bmg {
using namespace dev;
namespace {

// Blocks per side of the largest tail level (n = 2 blocks - 1) and its threads.
template <typename T>
constexpr int tail_blocks() { return (tail_max_n<T>() + 1) / 2; }

// Shared memory of one level: the stencil split by parity (plane, parity of j
// and i, (b+1)^2: a block's coefficients then lie at consecutive addresses for
// consecutive threads), the colour planes, and for the levels below the top
// the right-hand side, later the iterate, row-major.
struct TailLevel {
  int n, b, threads;
  int st, ci, x, f;   // offsets in elements of T (f: -1 at the top)
};

// Every offset but those of the f arrays is a multiple of four elements (the
// f arrays, of odd size, come last), so that weights can be copied 16 bytes at a time.
template <typename T>
__host__ __device__ inline int tail_layout(int top_n, int nlev, TailLevel* lv) {
  int off = 0, n = top_n;
  for (int l = 0; l < nlev; ++l, n = (n - 1) / 2) {
    const int b = (n + 1) / 2, nc = (n - 1) / 2;
    TailLevel q{n, b, b * b < 32 ? 32 : b * b, 0, 0, 0, -1};
    if (l + 1 < nlev) {
      q.st = off, off += 24 * (b + 1) * (b + 1);
      q.ci = off, off += 8 * (nc + 2) * (nc + 2);
      q.x = off, off += 4 * (b + 2) * (b + 2);
    }
    if (lv) lv[l] = q;
  }
  n = top_n;
  for (int l = 0; l < nlev; ++l, n = (n - 1) / 2)
    if (l > 0) {
      if (lv) lv[l].f = off;
      off += (n + 2) * (n + 2);
    }
  return off;
}

template <typename T>
struct TailShared {
  TailDesc<T> d;
  TailLevel lv[TAIL_LEVELS];
  double y[COARSE_M_MAX];                                  // substitutions of a larger coarsest level
  double L9[COARSE_LANES * COARSE_LANES], y9[COARSE_LANES], yl9[COARSE_LANES];   // the default one's factor
};

// The warps of a level wait for each other (barrier 1 + level of `threads` threads).
__device__ __forceinline__ void tail_sync(int level, int threads) {
  if (threads <= 32)
    __syncwarp();
  else
    asm volatile("bar.sync %0, %1;\n" ::"r"(1 + level), "r"(threads) : "memory");
}

template <typename T>
struct TailBlock {          // a thread's block of one level
  BlockCoef<T> k;
  BlockPlanes<T> q;
  int i, j;                 // its point A
  bool va, vb, vc, vd;
};

template <typename T>
__device__ __forceinline__ void tail_block(TailBlock<T>& B, const TailLevel& L, T* sm) {
  const int t = threadIdx.x, bi = t % L.b, bj = t / L.b, b1 = L.b + 1;
  B.i = 2 * bi + 1;
  B.j = 2 * bj + 1;
  B.va = t < L.b * L.b;
  B.vb = B.va && B.i < L.n;
  B.vc = B.va && B.j < L.n;
  B.vd = B.vb && B.vc;
  B.q = block_planes(sm + L.x, L.b + 2, L.b + 2, bi, B.va ? bj : 0);
  const T* st = sm + L.st;
  block_coef(B.k, B.i, B.j, B.va, B.vb, B.vc, B.vd, [&](int plane, int i, int j) {
    return st[((plane * 4 + (j & 1) * 2 + (i & 1)) * b1 + (j >> 1)) * b1 + (i >> 1)];
  });
}

// The block's entries of a row-major (n+2)^2 array.
template <typename T>
__device__ __forceinline__ BlockX<T> tail_values(const TailBlock<T>& B, const T* g, int n) {
  const int ld = n + 2, p = B.j * ld + B.i;
  BlockX<T> v{};
  if (B.va) v.a = g[p];
  if (B.vb) v.b = g[p + 1];
  if (B.vc) v.c = g[p + ld];
  if (B.vd) v.d = g[p + ld + 1];
  return v;
}

template <typename T>
__device__ __forceinline__ void put_planes(const TailBlock<T>& B, const BlockX<T>& x) {
  if (B.va) *B.q.a = x.a;
  if (B.vb) *B.q.b = x.b;
  if (B.vc) *B.q.c = x.c;
  if (B.vd) *B.q.d = x.d;
}

// Pre-smoothing, residual and restriction of level l.  The iterate is left in
// the level's planes, the restricted residual in the next level's f.
template <typename T, bool NINE, bool FU>
__device__ __forceinline__ void tail_down(const TailShared<T>& S, T* sm, int l, const T* f_in, const T* x_in,
                                          int nu1) {
  const TailLevel L = S.lv[l];
  const TailLevel C = S.lv[l + 1];
  auto sync = [&] { tail_sync(l, L.threads); };
  TailBlock<T> B;
  tail_block(B, L, sm);
  const BlockX<T> f = tail_values(B, f_in, L.n);
  BlockX<T> x{};
  if (x_in) {
    x = tail_values(B, x_in, L.n);
    put_planes(B, x);
    sync();
  }
  for (int s = 0; s < nu1; ++s) {
    if (s == 0 && !x_in)
      block_sweep<NINE, FU, true>(B.k, f, x, B.q, B.va, B.vb, B.vc, B.vd, sync);
    else
      block_sweep<NINE, FU, false>(B.k, f, x, B.q, B.va, B.vb, B.vc, B.vd, sync);
  }
  const int b1 = L.b + 1;
  const T* st = sm + L.st;   // plane 0: a_O
  BlockX<T> o{};
  {
    const int e = (B.j >> 1) * b1 + (B.i >> 1), pp = b1 * b1;   // parities (j, i): A (1, 1), B (1, 0), C (0, 1), D (0, 0)
    if (B.va) o.a = st[3 * pp + e];
    if (B.vb) o.b = st[2 * pp + e + 1];
    if (B.vc) o.c = st[1 * pp + e + b1];
    if (B.vd) o.d = st[0 * pp + e + b1 + 1];
  }
  const BlockX<T> r = block_resid<NINE, FU>(B.k, o, f, x, B.q, B.va, B.vb, B.vc, B.vd);
  sync();                    // every residual is formed: the planes carry them to the restriction
  put_planes(B, r);
  sync();
  if (B.vd) {
    const int ic = (B.i + 1) / 2, jc = (B.j + 1) / 2, ldc = C.n + 2, psc = ldc * ldc;
    const T* ci = sm + L.ci;
    sm[C.f + jc * ldc + ic] = block_restrict<FU>(r, B.q, [&](int k, int dic, int djc) {
      return ci[k * psc + (jc + djc) * ldc + ic + dic];
    });
  }
  sync();
  put_planes(B, x);          // the iterate again, for the way up
  // (the next level's threads are among this level's: the barrier above orders its f)
}

// Interpolation, correction and post-smoothing of level l; returns the block's iterate.
template <typename T, bool NINE, bool FU>
__device__ __forceinline__ void tail_up(const TailShared<T>& S, T* sm, int l, const T* f_in, T* x_out, int nu2) {
  const TailLevel L = S.lv[l];
  const TailLevel C = S.lv[l + 1];
  auto sync = [&] { tail_sync(l, L.threads); };
  TailBlock<T> B;
  tail_block(B, L, sm);
  const BlockX<T> f = tail_values(B, f_in, L.n);
  BlockX<T> x{};
  if (B.va) x.a = *B.q.a;
  if (B.vb) x.b = *B.q.b;
  if (B.vc) x.c = *B.q.c;
  if (B.vd) x.d = *B.q.d;
  sync();                    // the coarse level's iterate is there
  if (B.va) {
    const int ic = (B.i + 1) / 2, jc = (B.j + 1) / 2, ldc = C.n + 2, psc = ldc * ldc, pc = jc * ldc + ic;
    const T *ci = sm + L.ci + pc, *e = sm + C.f + pc;
    block_interp<FU>(x, e[-ldc - 1], e[-ldc], e[-1], e[0], B.va, B.vb, B.vc, B.vd,
                     [&](int k) { return ci[k * psc]; });
  }
  put_planes(B, x);
  sync();
  for (int s = 0; s < nu2; ++s) block_sweep<NINE, FU, false>(B.k, f, x, B.q, B.va, B.vb, B.vc, B.vd, sync);
  const int ld = L.n + 2, p = B.j * ld + B.i;
  const size_t ext = (size_t)ld * ld;
  if (B.va && BMG_IN(DBG_GS_STORE, p, ext)) x_out[p] = x.a;
  if (B.vb && BMG_IN(DBG_GS_STORE, p + 1, ext)) x_out[p + 1] = x.b;
  if (B.vc && BMG_IN(DBG_GS_STORE, p + ld, ext)) x_out[p + ld] = x.c;
  if (B.vd && BMG_IN(DBG_GS_STORE, p + ld + 1, ext)) x_out[p + ld + 1] = x.d;
}

template <int BYTES>
__device__ __forceinline__ void tail_copy(void* dst, const void* src) {
  if constexpr (BYTES == 16)
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(smem_u32(dst)), "l"(src) : "memory");
  else
    asm volatile("cp.async.ca.shared.global [%0], [%1], %2;\n" ::"r"(smem_u32(dst)), "l"(src), "n"(BYTES)
                 : "memory");
}

template <typename T, bool FU>
__global__ void __launch_bounds__(tail_blocks<T>() * tail_blocks<T>(), 1)
    k_tail(const TailDesc<T>* __restrict__ d, const int* done) {
  extern __shared__ __align__(16) unsigned char tail_smem[];
  __shared__ TailShared<T> S;
  T* sm = reinterpret_cast<T*>(tail_smem);
  const int tid = threadIdx.x, nt = blockDim.x, warp = tid >> 5, lane = tid & 31, warps = nt >> 5;
  // constants of the solve: read before the wait (written no later than the setup)
  for (int k = tid; k < (int)(sizeof(TailDesc<T>) / 4); k += nt)
    reinterpret_cast<int*>(&S.d)[k] = reinterpret_cast<const int*>(d + blockIdx.x)[k];
  __syncthreads();
  const int nlev = S.d.nlev;
  if (tid == 0) tail_layout<T>(S.d.lv[0].v.n, nlev, S.lv);
  __syncthreads();
  // the stencils' rows, one warp each, and the weights: asynchronous copies, all
  // of them in flight together (loads through registers took 19 k cycles)
  int row = warp;
  for (int l = 0; l + 1 < nlev; ++l) {
    const TailLevel L = S.lv[l];
    const StencilView<T, T>& v = S.d.lv[l].v;
    const int ld = L.n + 2, b1 = L.b + 1, pp = b1 * b1;
    const T* const src[6] = {v.O, v.W, v.S_, v.SW, v.NW, v.D};
    for (; row < ld; row += warps)
      for (int i = lane; i < ld; i += 32) {
        T* to = sm + L.st + ((row & 1) * 2 + (i & 1)) * pp + (row >> 1) * b1 + (i >> 1);
#pragma unroll
        for (int k = 0; k < 6; ++k) tail_copy<sizeof(T)>(to + 4 * k * pp, src[k] + row * ld + i);
      }
    row -= ld;               // the next level's rows go to the warps that follow
    const int ldc = S.lv[l + 1].n + 2;
    constexpr int V = 16 / sizeof(T);
    for (int k = V * tid; k < 8 * ldc * ldc; k += V * nt) tail_copy<16>(sm + L.ci + k, S.d.lv[l].ci + k);
    for (int k = tid; k < 4 * (L.b + 2) * (L.b + 2); k += nt) sm[L.x + k] = T(0);
    for (int k = tid; k < ldc * ldc; k += nt) sm[S.lv[l + 1].f + k] = T(0);
  }
  const LevelDesc<T, T>& cd = S.d.lv[nlev - 1];
  const bool nine_unknowns = cd.v.n * cd.v.n == COARSE_LANES;
  if (nine_unknowns) {
    for (int k = tid; k < COARSE_LANES * COARSE_LANES; k += nt) S.L9[k] = cd.L[k];
    if (tid < COARSE_LANES) S.y9[tid] = quot_recip(cd.L[tid * (COARSE_LANES + 1)], &S.yl9[tid]);
  }
  pdl_enter();
  asm volatile("cp.async.wait_all;\n" ::: "memory");
  if (stopped(done) || stopped(S.d.done)) return;
  __syncthreads();
  const LevelDesc<T, T>& top = S.d.lv[0];
  const bool nine = S.d.top_kind == 9;
  auto level_f = [&](int l) -> const T* { return l == 0 ? top.f : sm + S.lv[l].f; };
  int l = 0;
  for (; l + 1 < nlev && tid < S.lv[l].threads; ++l) {
    const T* x_in = l == 0 && !S.d.zero ? top.x : (const T*)nullptr;
    if (l > 0 || nine)
      tail_down<T, true, FU>(S, sm, l, level_f(l), x_in, S.d.nu1);
    else
      tail_down<T, false, FU>(S, sm, l, level_f(l), x_in, S.d.nu1);
  }
  if (l + 1 == nlev && warp == 0) {
    T* f = sm + S.lv[nlev - 1].f;
    __syncwarp();
    if (nine_unknowns) {
      const int p = lane < COARSE_LANES ? (lane / 3 + 1) * 5 + lane % 3 + 1 : 6;
      CoarseFactor<COARSE_LANES> c9;
      coarse_load(c9, S.L9);
      c9.y = S.y9[lane < COARSE_LANES ? lane : 0];
      c9.yl = S.yl9[lane < COARSE_LANES ? lane : 0];
      const T x = (T)coarse_substitute(c9, (double)f[p]);
      __syncwarp();
      if (lane < COARSE_LANES) f[p] = x;
      __syncwarp();
    } else {
      warp_coarse<T>(cd.v.n, cd.L, f, f, S.y);
    }
  }
  for (--l; l >= 0; --l) {   // from the last level this thread took part in
    T* out = l == 0 ? top.x : sm + S.lv[l].f;
    if (l > 0 || nine)
      tail_up<T, true, FU>(S, sm, l, level_f(l), out, S.d.nu2);
    else
      tail_up<T, false, FU>(S, sm, l, level_f(l), out, S.d.nu2);
  }
}

template <typename T, bool FU>
void tail_launch(const TailDesc<T>* d, int count, int top_n, int nlev, const int* done_any, cudaStream_t s) {
  static PerDevice smem;
  allow_smem(smem, k_tail<T, FU>, tail_layout<T>(tail_max_n<T>(), sizeof(T) == 8 ? 4 : 5, nullptr) * sizeof(T));
  const int b = (top_n + 1) / 2;
  pdl_launch(k_tail<T, FU>, count, b * b < 32 ? 32 : b * b, tail_layout<T>(top_n, nlev, nullptr) * sizeof(T), s, d,
             done_any);
  count_launch();
}

}  // namespace

template <typename T>
void launch_tail(const TailDesc<T>* d, int count, int top_n, int nlev, const int* done_any, cudaStream_t s,
                 int fused) {
  if (count <= 0) return;
  if (fused)
    tail_launch<T, true>(d, count, top_n, nlev, done_any, s);
  else
    tail_launch<T, false>(d, count, top_n, nlev, done_any, s);
}
template void launch_tail<double>(const TailDesc<double>*, int, int, int, const int*, cudaStream_t, int);
template void launch_tail<float>(const TailDesc<float>*, int, int, int, const int*, cudaStream_t, int);

}  // namespace bmg
