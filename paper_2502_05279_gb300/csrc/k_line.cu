// Zebra line relaxation with factored lines: the elimination of a line's
// tridiagonal matrix depends on the operator only, so a hierarchy forms it once
// at setup and a sweep only carries right-hand sides through it.
//
// What bounds it.  The Thomas recurrence is a chain along the line, and its
// rounding is fixed, so a half sweep costs at least (line length) x (dependent
// FP64 operations per point).  On GB300 a dependent FP64 operation takes about
// 63 cycles, a warp's FP64 instruction occupies its quarter of the SM for about
// 60 of them whatever the number of active lanes, and an FP64 division takes
// 560 (measured on one warp).  The unfactored form (line_row_body) pays two
// divisions per point and waits for its uncoalesced loads on the same thread:
// 720 us per half sweep at 511^2.
// Layout of the work.  One warp per CTA runs the chains of R lines, one per
// lane, and issues nothing else; the CTA's other warps form the right-hand
// sides g = f - (couplings to the fixed lines) of the next LC positions, fetch
// the factors, and store the previous positions' results, all through shared
// memory, so that their loads coalesce and their FP64 work runs on the other
// three quarters of the SM.  Per point the chain is a product, a difference and
// quot's four operations forward, and two operations backward: 511 x 8 x 63
// cycles, 124 us per half sweep at 511^2; measured 169 (720 unfactored).
#include "cycle_device.cuh"

namespace bmg {
using namespace dev;
namespace {

constexpr int LC = 32;              // positions per stage
constexpr int LINE_THREADS = 256;   // warp 0: the chains; warps 1 .. 7: everything else

// Point of position q (1 .. n) on line w (1 .. n): x-lines run along i, y-lines along j.
template <int AXIS>
__device__ __forceinline__ size_t line_point(int ld, int w, int q) {
  return AXIS == 0 ? (size_t)w * ld + q : (size_t)q * ld + w;
}

// Coupling of p to the previous point of its line.
template <int AXIS, typename T, typename S>
__device__ __forceinline__ T line_prev(const StencilView<T, S>& v, size_t p) {
  return cvt<T>(AXIS == 0 ? v.W[p] : v.S_[p]);
}

// m_1 = a_O, m_q = a_O - a_prev c_{q-1}, c_q = a_next / m_q; one thread per
// line, LF positions read ahead of the chain (about 690 cycles a position, the
// division 560 of them).  blockIdx.y picks the level and axis: the chains of
// all levels run side by side, so a setup waits for the longest line only.
template <typename T, typename S>
__global__ void k_line_factor(LineJobs<T, S> jobs) {
  constexpr int LF = 8;
  const LineJob<T, S> b = jobs.job[blockIdx.y];
  const int w = 1 + blockIdx.x * blockDim.x + threadIdx.x;
  if (w > b.n) return;
  const size_t step = b.axis == 0 ? 1 : (size_t)b.n + 2, line = (size_t)w * (b.axis == 0 ? (size_t)b.n + 2 : 1);
  T cp = T(0);
  for (int q0 = 1; q0 <= b.n; q0 += LF) {
    T o[LF], lo[LF + 1];
#pragma unroll
    for (int k = 0; k <= LF; ++k) {
      const size_t p = line + step * (size_t)(q0 + k <= b.n + 1 ? q0 + k : b.n + 1);
      if (k < LF) o[k] = b.o[p];
      lo[k] = cvt<T>(b.prev[p]);
    }
#pragma unroll
    for (int k = 0; k < LF; ++k) {
      if (q0 + k > b.n) break;
      const size_t p = line + step * (size_t)(q0 + k);
      const T mm = q0 + k == 1 ? o[k] : rsub(o[k], rmul(lo[k], cp));
      cp = rdiv(lo[k + 1], mm);
      if (BMG_IN(DBG_LINE_STORE, p, (size_t)(b.n + 2) * (b.n + 2))) {
        b.c[p] = cp;
        b.m[p] = mm;
      }
    }
  }
}

// m's reciprocal and its remainder for quot.
__global__ void k_line_recip(int n, const double* __restrict__ m, double* __restrict__ y, double* __restrict__ yl) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x + 1, j = blockIdx.y * blockDim.y + threadIdx.y + 1;
  if (i > n || j > n) return;
  const size_t p = (size_t)j * (n + 2) + i;
  if (!BMG_IN(DBG_LINE_STORE, p, (size_t)(n + 2) * (n + 2))) return;
  double rl;
  y[p] = quot_recip(m[p], &rl);
  yl[p] = rl;
}

// Right-hand side of p: f minus the couplings to the two fixed lines, in the
// order of line_row_body (S, N, SW, NE, NW, SE) or line_col_body (W, E, SW, NE, SE, NW).
template <int AXIS, bool NINE, typename T, typename S>
__device__ __forceinline__ T line_rhs(const StencilView<T, S>& v, const T* __restrict__ f, const T* x, size_t p) {
  const int ld = v.ld;
  T g = f[p];
  if (AXIS == 0) {
    g = rsub(g, rmul(cvt<T>(v.S_[p]), x[p - ld]));
    g = rsub(g, rmul(cvt<T>(v.S_[p + ld]), x[p + ld]));
    if (NINE) {
      g = rsub(g, rmul(cvt<T>(v.SW[p]), x[p - ld - 1]));
      g = rsub(g, rmul(cvt<T>(v.SW[p + ld + 1]), x[p + ld + 1]));
      g = rsub(g, rmul(cvt<T>(v.NW[p]), x[p + ld - 1]));
      g = rsub(g, rmul(cvt<T>(v.NW[p + 1 - ld]), x[p + 1 - ld]));
    }
  } else {
    g = rsub(g, rmul(cvt<T>(v.W[p]), x[p - 1]));
    g = rsub(g, rmul(cvt<T>(v.W[p + 1]), x[p + 1]));
    if (NINE) {
      g = rsub(g, rmul(cvt<T>(v.SW[p]), x[p - ld - 1]));
      g = rsub(g, rmul(cvt<T>(v.SW[p + ld + 1]), x[p + ld + 1]));
      g = rsub(g, rmul(cvt<T>(v.NW[p + 1 - ld]), x[p + 1 - ld]));
      g = rsub(g, rmul(cvt<T>(v.NW[p]), x[p + ld - 1]));
    }
  }
  return g;
}

// One stage's inputs and its results, [line][position] with a padded row.
template <typename T, int R>
struct LineStage {
  T g[R][LC + 1], a[R][LC + 1], m[R][LC + 1], y[R][LC + 1], yl[R][LC + 1], out[R][LC + 1];
};

// The lines first, first + 2, ... of one parity, R per CTA, solved in place on
// x.  The lines of the other parity are only read, so every CTA's inputs are
// fixed for the launch; a CTA reads of its own lines only what it wrote itself.
template <typename T, typename S, bool NINE, int AXIS, int R>
__global__ void __launch_bounds__(LINE_THREADS)
    k_line_solve(StencilView<T, S> v, const T* __restrict__ f, T* x, LineFactor<T> fac, int first, const int* done) {
  extern __shared__ __align__(16) unsigned char line_smem[];
  pdl_enter();
  if (stopped(done)) return;
  LineStage<T, R>* st = reinterpret_cast<LineStage<T, R>*>(line_smem);
  const int n = v.n, ld = v.ld, stages = (n + LC - 1) / LC;
  const int w0 = first + 2 * R * (int)blockIdx.x;
  const int tid = threadIdx.x, help = tid - 32;
  // helpers: point (line r, position offset t) number e of a stage; consecutive
  // threads take consecutive addresses
  auto each = [&](int k, auto&& fn) {
#pragma unroll 2
    for (int e = help; e < R * LC; e += LINE_THREADS - 32) {
      const int r = AXIS == 0 ? e / LC : e % R, t = AXIS == 0 ? e % LC : e / R;
      const int w = w0 + 2 * r, q = 1 + k * LC + t;
      if (w <= n && q <= n) fn(r, t, line_point<AXIS>(ld, w, q));
    }
  };
  auto fetch = [&](int k) {
    LineStage<T, R>& b = st[k & 1];
    each(k, [&](int r, int t, size_t p) {
      b.a[r][t] = line_prev<AXIS>(v, p);
      b.m[r][t] = fac.m[p];
      if constexpr (sizeof(T) == 8) {
        b.y[r][t] = fac.y[p];
        b.yl[r][t] = fac.yl[p];
      }
      b.g[r][t] = line_rhs<AXIS, NINE>(v, f, x, p);
    });
  };
  auto fetch_back = [&](int k) {
    LineStage<T, R>& b = st[k & 1];
    each(k, [&](int r, int t, size_t p) {
      b.a[r][t] = fac.c[p];
      b.g[r][t] = x[p];
    });
  };
  auto store = [&](int k) {
    LineStage<T, R>& b = st[k & 1];
    each(k, [&](int r, int t, size_t p) {
      if (BMG_IN(DBG_LINE_STORE, p, (size_t)(n + 2) * ld)) x[p] = b.out[r][t];
    });
  };
  const bool chain = tid < R && w0 + 2 * tid <= n;
  const int r = tid;
  T d = T(0);
  // forward: d_q = (g_q - a_prev d_{q-1}) / m_q
  if (help >= 0) fetch(0);
  __syncthreads();
  for (int k = 0; k < stages; ++k) {
    if (help >= 0) {
      if (k > 0) store(k - 1);
      if (k + 1 < stages) fetch(k + 1);
    } else if (chain) {
      LineStage<T, R>& b = st[k & 1];
      const int cnt = n - k * LC < LC ? n - k * LC : LC;
      // the next position's operands are read before this one's result is stored
      T g = b.g[r][0], a = b.a[r][0], m = b.m[r][0], y = b.y[r][0], yl = b.yl[r][0];
#pragma unroll 4
      for (int t = 0; t < cnt; ++t) {
        const T g1 = b.g[r][t + 1], a1 = b.a[r][t + 1], m1 = b.m[r][t + 1], y1 = b.y[r][t + 1], yl1 = b.yl[r][t + 1];
        const T s = k + t == 0 ? g : rsub(g, rmul(a, d));
        if constexpr (sizeof(T) == 8)
          d = quot(s, m, y, yl);
        else
          d = rdiv(s, m);
        b.out[r][t] = d;
        g = g1, a = a1, m = m1, y = y1, yl = yl1;
      }
    }
    __syncthreads();
  }
  if (help >= 0) store(stages - 1);
  __syncthreads();   // the CTA's forward results are in x
  // backward: x_n = d_n, x_q = d_q - c_q x_{q+1}
  if (help >= 0) fetch_back(stages - 1);
  __syncthreads();
  for (int k = stages - 1; k >= 0; --k) {
    if (help >= 0) {
      if (k + 1 < stages) store(k + 1);
      if (k > 0) fetch_back(k - 1);
    } else if (chain) {
      LineStage<T, R>& b = st[k & 1];
      const int cnt = n - k * LC < LC ? n - k * LC : LC;
      T g = b.g[r][cnt - 1], a = b.a[r][cnt - 1];
#pragma unroll 4
      for (int t = cnt - 1; t >= 0; --t) {
        const int u = t > 0 ? t - 1 : 0;
        const T g1 = b.g[r][u], a1 = b.a[r][u];
        d = 1 + k * LC + t == n ? g : rsub(g, rmul(a, d));
        b.out[r][t] = d;
        g = g1, a = a1;
      }
    }
    __syncthreads();
  }
  if (help >= 0) store(0);
}

template <typename T, typename S, int AXIS, int R>
void half_sweep(const StencilView<T, S>& v, int kind, const T* f, T* x, const LineFactor<T>& fac, int first,
                int lines, const int* done, cudaStream_t s) {
  constexpr size_t bytes = 2 * sizeof(LineStage<T, R>);
  const unsigned g = (unsigned)((lines + R - 1) / R);
  if (kind == 9) {
    static PerDevice smem;
    allow_smem(smem, k_line_solve<T, S, true, AXIS, R>, bytes);
    pdl_launch(k_line_solve<T, S, true, AXIS, R>, g, LINE_THREADS, bytes, s, v, f, x, fac, first, done);
  } else {
    static PerDevice smem;
    allow_smem(smem, k_line_solve<T, S, false, AXIS, R>, bytes);
    pdl_launch(k_line_solve<T, S, false, AXIS, R>, g, LINE_THREADS, bytes, s, v, f, x, fac, first, done);
  }
  count_launch();
}

// Lines per CTA: 8 while that gives at most one CTA per SM (two CTAs on an SM
// may put their chain warps on the same quarter, which runs them at half speed
// each), then 16 and 32 lanes of the same chain warp, which cost it nothing.
template <typename T, typename S, int AXIS>
void sweep_axis(const StencilView<T, S>& v, int kind, const T* f, T* x, const LineFactor<T>& fac, const int* done,
                cudaStream_t s) {
  constexpr int SMS = 152;
  for (int first = 1; first <= 2; ++first) {
    const int lines = first == 1 ? (v.n + 1) / 2 : (v.n - 1) / 2;
    if (lines <= 0) continue;
    if (lines <= 8 * SMS)
      half_sweep<T, S, AXIS, 8>(v, kind, f, x, fac, first, lines, done, s);
    else if (lines <= 16 * SMS)
      half_sweep<T, S, AXIS, 16>(v, kind, f, x, fac, first, lines, done, s);
    else
      half_sweep<T, S, AXIS, 32>(v, kind, f, x, fac, first, lines, done, s);
  }
}

}  // namespace

template <typename T, typename S>
void launch_line_factor(const LineJobs<T, S>& jobs, cudaStream_t s) {
  constexpr int TPB = 32;
  int n = 0;
  for (int k = 0; k < jobs.count; ++k) n = jobs.job[k].n > n ? jobs.job[k].n : n;
  if (n == 0) return;
  k_line_factor<T, S><<<dim3((n + TPB - 1) / TPB, jobs.count), TPB, 0, s>>>(jobs);
  count_launch();
  if constexpr (sizeof(T) == 8)
    for (int k = 0; k < jobs.count; ++k) {
      const LineJob<T, S>& b = jobs.job[k];
      const size_t ps = plane_size(b.n);
      k_line_recip<<<dim3((b.n + 31) / 32, (b.n + 7) / 8), dim3(32, 8), 0, s>>>(b.n, b.m, b.m + ps, b.m + 2 * ps);
      count_launch();
    }
}

template <typename T, typename S>
void launch_line_solve(const StencilView<T, S>& v, int kind, const T* f, T* x, const LineFactor<T>& fx,
                       const LineFactor<T>& fy, int sweeps, int dir, const int* done, cudaStream_t s) {
  for (int k = 0; k < sweeps; ++k) {
    if (dir != LINE_Y) sweep_axis<T, S, 0>(v, kind, f, x, fx, done, s);
    if (dir != LINE_X) sweep_axis<T, S, 1>(v, kind, f, x, fy, done, s);
  }
}

#define BMG_INST(T, S)                                                                                         \
  template void launch_line_factor<T, S>(const LineJobs<T, S>&, cudaStream_t);                                 \
  template void launch_line_solve<T, S>(const StencilView<T, S>&, int, const T*, T*, const LineFactor<T>&,   \
                                        const LineFactor<T>&, int, int, const int*, cudaStream_t);
BMG_INST(double, double)
BMG_INST(float, float)
BMG_INST(float, __nv_bfloat16)
#undef BMG_INST

}  // namespace bmg
