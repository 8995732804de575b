// Two-grid training loss of the learned interpolation and its gradient, on a
// batch of small crops (n = 7, 15 or 31 interior points), one CTA per crop.
//
// For an error vector e the two-grid error propagation of V(2,1) with exact
// coarse solve is
//     E e = S (I - P A_c^{-1} P^T A) S^2 e,   A_c = P^T A P,
// S one four-colour Gauss-Seidel sweep of A e = 0.  The loss of a crop is
// w/K sum_k ||E e_k||_A^2 / e_ref_k (e_ref: Dendy's energies).  Its gradient
// with respect to the weights of P, with u = A_c^{-1} P^T A e1 (e1 = S^2 e),
// e2 = e1 - P u, g2 = S^T (dL/d e3) and the adjoint coarse solve
// v = A_c^{-1} P^T g2, is  dL/dP = (A P v - g2) u^T - (A e2) v^T  on P's
// sparsity pattern; it is chained through Dendy's centre formula and the
// edge split to the network's logits.  Everything is FP64: the crops have
// coefficient jumps of up to 1e6, far beyond what an FP32 coarse solve
// resolves.  A_c keeps the lexicographic band of half-width n_c + 1 and is
// factored as L D L^T; the fine grid operations up to the energies follow the
// oracle's expression orders (sweeps, apply, the Fig. 2 restriction, the
// interpolation), the Galerkin entries are the setup's (bit for bit the
// oracle's), and the coarse solves differ from the oracle's dense solve by
// rounding.
//
// What bounds it: FP64 throughput (a warp's instruction takes 60 cycles of its
// SM quarter) wherever every point has work, and the 63-cycle latency of the
// chains in the factorisation and the substitutions.  So a thread owns a 2 x 2
// block of points with its couplings in registers (block_device.cuh, eight
// warps: two per quarter keep the pipe busy), the adjoint sweep touches a
// colour's neighbours only, the gradient's last two operator products skip the
// coarse points, and the substitutions of four error vectors run side by side,
// a warp each, one fused multiply-add and one shuffle per unknown.  152 crops
// of 31^2 with four vectors: 3300 -> 433 us (one warp factored and solved
// one vector after another, with a division and a five-level sum per unknown).
#include "block_device.cuh"
#include "learned.h"
#include "learned_device.cuh"
#include "rap_device.cuh"

namespace bmg {
using namespace dev;
namespace {

constexpr int TG_VECS = 4;   // error vectors in flight

template <int N>
struct TG {
  static constexpr int LD = N + 2, PS = LD * LD;
  static constexpr int NC = (N - 1) / 2, LDC = NC + 2, PSC = LDC * LDC;
  static constexpr int M = NC * NC, BW = NC + 1, BL = BW + 1;   // coarse unknowns, half band, band row length
  static constexpr int NB = NC + 1, NB2 = NB * NB;              // blocks
  static constexpr int THREADS = NB2 < 64 ? 64 : NB2, WARPS = THREADS / 32;
  static constexpr int PL = 4 * (NB + 2) * (NB + 2);            // the four colour planes
  // shared-memory layout, in doubles
  static constexpr int ST = 0;                   // O, W, S, SW, NW, D = 1/O
  static constexpr int CI = ST + 6 * PS;         // 8 weight planes
  static constexpr int BAND = CI + 8 * PSC;      // lower band of A_c / its factor, M x BL
  static constexpr int RD = BAND + M * BL;       // 1 / D of the factor
  static constexpr int X = RD + M, T = X + PL;   // colour planes
  static constexpr int E = T + PL;               // per vector and thread: the block's e (e2) and g2
  static constexpr int G = E + TG_VECS * 4 * NB2;
  static constexpr int U = G + TG_VECS * 4 * NB2, V = U + TG_VECS * PSC;   // coarse vectors
  static constexpr int RED = V + TG_VECS * PSC;
  static constexpr int TOTAL = RED + WARPS;
  // after the last vector: the eight planes of dL/dw and two of dL/d(edge split)
  static constexpr int DW = X;
  static_assert(DW + 10 * PSC <= U, "gradient planes");
  static constexpr size_t BYTES = (size_t)TOTAL * sizeof(double);
};

__device__ __forceinline__ double warp_sum(double v) {
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// 1/d to about an ulp by Newton's iteration from the hardware's approximation
// (a division would take 560 cycles in the factorisation's chain).  d normal and
// below 2^1022, which the scaled band's pivots are.
__device__ __forceinline__ double recip_newton(double d) {
  double y;
  asm("rcp.approx.ftz.f64 %0, %1;\n" : "=d"(y) : "d"(d));
  y = __fma_rn(y, __fma_rn(-d, y, 1.0), y);
  return __fma_rn(y, __fma_rn(-d, y, 1.0), y);
}

// Scales the band of A_c by the power of two that brings its largest diagonal
// entry into [1, 2), and returns it: band_factor multiplies two entries before it
// divides by a pivot, which over- or underflows for operators beyond 2^+-500 (and
// recip_newton beyond 2^+-1022) if the band is left as it is.  Exact, so results
// scale with the operator bit for bit; the entries set are those of the 9-point
// operator.  scratch: WARPS ints.
template <int N>
__device__ double band_scale(double* band, int* scratch) {
  using L = TG<N>;
  constexpr int M = L::M, NC = L::NC, BL = L::BL;
  int top = 0;
  for (int c = threadIdx.x; c < M; c += L::THREADS)
    top = max(top, (int)(((unsigned)__double2hiint(band[c * BL]) >> 20) & 0x7ffu));
  top = __reduce_max_sync(0xffffffffu, top);
  if ((threadIdx.x & 31) == 0) scratch[threadIdx.x >> 5] = top;
  __syncthreads();
  for (int w = 0; w < L::WARPS; ++w) top = max(top, scratch[w]);
  const int e = top == 2047 ? 1023 : min(max(2046 - top, 1), 2045);   // biased exponent of 2^(1023 - top)
  const double s = __hiloint2double(e << 20, 0);
  constexpr int at[5] = {0, 1, NC - 1, NC, NC + 1};
  for (int c = threadIdx.x; c < M; c += L::THREADS)
#pragma unroll
    for (int q = 0; q < 5; ++q) band[c * BL + at[q]] *= s;
  __syncthreads();
  return s;
}

// Banded L D L^T of the lower band (row i holds A(i, i-d) at d = 0..BW), by the
// whole block: afterwards row i holds L(i, i-d) for d >= 1, rd the reciprocals
// of D.  A step forms its products while the pivot's reciprocal is under way.
// Returns false on a non-positive pivot.
template <int N>
__device__ bool band_factor(double* band, double* rd) {
  using L = TG<N>;
  constexpr int M = L::M, BW = L::BW, BL = L::BL, PAIRS = BW * (BW + 1) / 2;
  constexpr int PER = (PAIRS + L::THREADS - 1) / L::THREADS;
  int pa[PER], pb[PER];                     // pair e: column k + 1 + a, row k + 1 + a + b
#pragma unroll
  for (int q = 0; q < PER; ++q) {
    int a = 0, rem = threadIdx.x + q * L::THREADS;
    if (rem >= PAIRS) a = -1;
    while (a >= 0 && rem >= BW - a) rem -= BW - a, ++a;
    pa[q] = a;
    pb[q] = rem;
  }
  // the last warp forms the pivot's reciprocal while the first ones form the products
  const bool pivot = (int)(threadIdx.x >> 5) == L::WARPS - 1;
  bool ok = true;
  for (int k = 0; k < M; ++k) {
    const double d = band[k * BL];
    // positive and not NaN, on the bit pattern (a comparison would use the FP64 pipe)
    const unsigned long long db = (unsigned long long)__double_as_longlong(d);
    if (db - 1ull >= 0x7ff0000000000000ull) ok = false;
    double prod[PER], cur[PER];
#pragma unroll
    for (int q = 0; q < PER; ++q) {
      const int j = k + 1 + pa[q], i = j + pb[q];
      if (pa[q] >= 0 && i < M) {
        prod[q] = band[i * BL + (i - k)] * band[j * BL + (j - k)];
        cur[q] = band[i * BL + pb[q]];
      }
    }
    if (pivot) {
      const double r = recip_newton(d);
      if ((threadIdx.x & 31) == 0) rd[k] = r;
    }
    __syncthreads();
#pragma unroll
    for (int q = 0; q < PER; ++q) {
      const int j = k + 1 + pa[q], i = j + pb[q];
      if (pa[q] >= 0 && i < M) band[i * BL + pb[q]] = __fma_rn(-prod[q], rd[k], cur[q]);
    }
    __syncthreads();
  }
  for (int e = threadIdx.x; e < M * BW; e += L::THREADS) {
    const int i = e / BW, t = 1 + e % BW;
    if (i - t >= 0) band[i * BL + t] *= rd[i - t];
  }
  __syncthreads();
  return ok;
}

// x <- (L D L^T)^{-1} x for a coarse vector in the (NC+2)^2 layout, by one
// warp: unknown i's partial sum lives in lane i mod 32 while the BW unknowns
// before it (after it, on the way back) are eliminated.
template <int N>
__device__ void band_solve(const double* band, const double* rd, double* x) {
  using L = TG<N>;
  constexpr int M = L::M, NC = L::NC, LDC = L::LDC, BW = L::BW, BL = L::BL;
  const int lane = threadIdx.x & 31;
  auto pos = [](int i) { return (i / NC + 1) * LDC + (i % NC + 1); };
  auto fwd = [&](int j) {   // L(j + d, j) of this lane's unknown j + d
    const int d = (lane - j) & 31;
    return d >= 1 && d <= BW && j + d < M ? band[(j + d) * BL + d] : 0.0;
  };
  double acc = lane < M ? x[pos(lane)] : 0.0, l = fwd(0);
  for (int j = 0; j < M; ++j) {
    const double z = __shfl_sync(0xffffffffu, acc, j & 31);
    const double ln = j + 1 < M ? fwd(j + 1) : 0.0;
    if (lane == (j & 31)) {
      x[pos(j)] = z * rd[j];
      acc = j + 32 < M ? x[pos(j + 32)] : 0.0;
    } else {
      acc = __fma_rn(-l, z, acc);
    }
    l = ln;
  }
  __syncwarp();
  auto bwd = [&](int j) {   // L(j, j - d) of this lane's unknown j - d
    const int d = (j - lane) & 31;
    return d >= 1 && d <= BW && j - d >= 0 ? band[j * BL + d] : 0.0;
  };
  {
    const int i = M - 1 - ((M - 1 - lane) & 31);   // the largest unknown of this lane
    acc = i >= 0 ? x[pos(i)] : 0.0;
  }
  l = bwd(M - 1);
  for (int j = M - 1; j >= 0; --j) {
    const double z = __shfl_sync(0xffffffffu, acc, j & 31);
    const double ln = j > 0 ? bwd(j - 1) : 0.0;
    if (lane == (j & 31)) {
      x[pos(j)] = z;
      acc = j >= 32 ? x[pos(j - 32)] : 0.0;
    } else {
      acc = __fma_rn(-l, z, acc);
    }
    l = ln;
  }
  __syncwarp();
}

// y <- S^T y on the colour planes: for the colours in reverse order, z = d y on
// the colour's points and y = y - A z, whose terms are the couplings to that
// colour only.  y: the block's values; z's planes share q.
template <typename F>
__device__ __forceinline__ void sweep_adjoint(const BlockCoef<double>& k, const BlockX<double>& o, BlockX<double>& y,
                                              const BlockPlanes<double>& q, bool va, bool vb, bool vc, bool vd,
                                              F&& sync) {
  const double zd = vd ? y.d * k.dd : 0.0;
  if (vd) *q.d = zd;
  sync();
  if (va) {
    double s = k.asw * q.d[-q.p - 1];
    s = __fma_rn(k.dsw, zd, s);
    s = __fma_rn(k.anw, q.d[-1], s);
    y.a -= __fma_rn(k.ase, q.d[-q.p], s);
  }
  if (vb) y.b -= __fma_rn(k.ds, zd, k.bs * q.d[-q.p]);
  if (vc) y.c -= __fma_rn(k.dw, zd, k.cw * q.d[-1]);
  if (vd) y.d = __fma_rn(-o.d, zd, y.d);
  const double zc = vc ? y.c * k.cd : 0.0;
  if (vc) *q.c = zc;
  sync();
  if (va) y.a -= __fma_rn(k.cs, zc, k.as * q.c[-q.p]);
  if (vb) {
    double s = k.bsw * q.c[-q.p];
    s = __fma_rn(k.bne, q.c[1], s);
    s = __fma_rn(k.bnw, zc, s);
    y.b -= __fma_rn(k.bse, q.c[1 - q.p], s);
  }
  if (vd) y.d -= __fma_rn(k.dw, zc, k.de * q.c[1]);
  if (vc) y.c = __fma_rn(-o.c, zc, y.c);
  const double zb = vb ? y.b * k.bd : 0.0;
  if (vb) *q.b = zb;
  sync();
  if (va) y.a -= __fma_rn(k.bw, zb, k.aw * q.b[-1]);
  if (vc) {
    double s = k.csw * q.b[-1];
    s = __fma_rn(k.cne, q.b[q.p], s);
    s = __fma_rn(k.cnw, q.b[q.p - 1], s);
    y.c -= __fma_rn(k.bnw, zb, s);
  }
  if (vd) y.d -= __fma_rn(k.ds, zb, k.dn * q.b[q.p]);
  if (vb) y.b = __fma_rn(-o.b, zb, y.b);
  const double za = va ? y.a * k.ad : 0.0;
  if (va) *q.a = za;
  sync();
  if (vb) y.b -= __fma_rn(k.bw, za, k.be * q.a[1]);
  if (vc) y.c -= __fma_rn(k.cs, za, k.cn * q.a[q.p]);
  if (vd) {
    double s = k.dsw * za;
    s = __fma_rn(k.dne, q.a[q.p + 1], s);
    s = __fma_rn(k.dnw, q.a[q.p], s);
    y.d -= __fma_rn(k.dse, q.a[1], s);
  }
  if (va) y.a = __fma_rn(-o.a, za, y.a);
}

template <int N>
__device__ double block_total(double v, double* red) {
  v = warp_sum(v);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = v;
  __syncthreads();
  double s = 0.0;
  if (threadIdx.x == 0)
    for (int w = 0; w < TG<N>::WARPS; ++w) s += red[w];
  __syncthreads();
  return s;   // valid on thread 0
}

// grid: one CTA per crop.  coefs: ncrop x 5 planes (n+2)^2 (ghost ring and
// couplings to it are ignored); vecs: ncrop x K error vectors (n+2)^2;
// delta: ncrop x n_c^2 x 4 logits (NULL: Dendy's weights); eref: ncrop x K
// normalisers, or NULL for energies only; energies: ncrop x K out;
// ddelta: ncrop x n_c^2 x 4 out (with eref); aux: ncrop x 4 coarse planes of
// workspace (with eref); err: set on a non-positive pivot.
template <int N>
__global__ void __launch_bounds__(TG<N>::THREADS, 1)
    k_twogrid(int K, const double* __restrict__ coefs, const double* __restrict__ vecs,
              const float* __restrict__ delta, const double* __restrict__ eref, double weight,
              double* __restrict__ energies, float* __restrict__ ddelta, double* aux, int* __restrict__ err) {
  using L = TG<N>;
  constexpr int LD = L::LD, PS = L::PS, NC = L::NC, LDC = L::LDC, PSC = L::PSC, M = L::M, BL = L::BL, NB = L::NB;
  constexpr int NT = L::THREADS;
  extern __shared__ double sm[];
  const int crop = blockIdx.x, tid = threadIdx.x;
  double *st = sm + L::ST, *ci = sm + L::CI, *band = sm + L::BAND, *rd = sm + L::RD, *red = sm + L::RED;
  if (aux) aux += (size_t)crop * 4 * PSC;
  // stencil, with the ghost ring and every coupling to it zero
  const double* src = coefs + (size_t)crop * 5 * PS;
  for (int e = tid; e < PS; e += NT) {
    const int i = e % LD, j = e / LD;
    const bool in = i >= 1 && i <= N && j >= 1 && j <= N;
    const double o = in ? src[e] : 0.0;
    st[e] = o;
    st[PS + e] = (in && i > 1) ? src[PS + e] : 0.0;
    st[2 * PS + e] = (in && j > 1) ? src[2 * PS + e] : 0.0;
    st[3 * PS + e] = (in && i > 1 && j > 1) ? src[3 * PS + e] : 0.0;
    st[4 * PS + e] = (in && i > 1 && j < N) ? src[4 * PS + e] : 0.0;
    st[5 * PS + e] = in ? rdiv(1.0, o) : 0.0;
  }
  for (int e = tid; e < L::TOTAL - L::CI; e += NT) sm[L::CI + e] = 0.0;
  __syncthreads();
  const Planes<double> A = planes_at(st, PS);
  const float* dl = delta ? delta + (size_t)crop * M * MLP_OUT : nullptr;
  for (int e = tid; e < PSC; e += NT) learned::edge_cell(A, LD, NC, dl, e % LDC, e / LDC, ci, aux);
  __syncthreads();
  for (int e = tid; e < PSC; e += NT) learned::centre_cell(A, LD, NC, e % LDC, e / LDC, ci);
  __syncthreads();
  // Galerkin operator into the lower band: row c holds O; W (d = 1), S (d = NC),
  // SW (d = NC + 1); the NW coupling of c is the SE coupling of row c + NC - 1
  for (int c = tid; c < M; c += NT) {
    const int ic = 1 + c % NC, jc = 1 + c / NC;
    band[c * BL] = rapdev::rap_entry<0, 0>(A, LD, ci, PSC, LDC, NC, ic, jc);
    if (ic > 1) band[c * BL + 1] = rapdev::rap_entry<-1, 0>(A, LD, ci, PSC, LDC, NC, ic, jc);
    if (jc > 1) band[c * BL + NC] = rapdev::rap_entry<0, -1>(A, LD, ci, PSC, LDC, NC, ic, jc);
    if (ic > 1 && jc > 1) band[c * BL + NC + 1] = rapdev::rap_entry<-1, -1>(A, LD, ci, PSC, LDC, NC, ic, jc);
    if (ic > 1 && jc < NC) band[(c + NC - 1) * BL + NC - 1] = rapdev::rap_entry<-1, 1>(A, LD, ci, PSC, LDC, NC, ic, jc);
  }
  __syncthreads();
  const double scale = band_scale<N>(band, reinterpret_cast<int*>(red));
  if (!band_factor<N>(band, rd)) {   // every thread sees every pivot
    if (tid == 0) atomicExch(err, 1);
    return;
  }
  for (int e = tid; e < M; e += NT) rd[e] *= scale;   // 1 / D of the unscaled operator (the first vectors' barriers order it)
  // this thread's block and coarse cell (bi + 1, bj + 1)
  const bool va = tid < L::NB2;
  const int bi = va ? tid % NB : 0, bj = va ? tid / NB : 0, i = 2 * bi + 1, j = 2 * bj + 1;
  const bool vb = va && bi < NB - 1, vc = va && bj < NB - 1, vd = vb && vc;
  const int p = j * LD + i, pc = (bj + 1) * LDC + bi + 1;
  BlockCoef<double> k;
  block_coef(k, i, j, va, vb, vc, vd, [&](int plane, int a, int b) { return st[plane * PS + b * LD + a]; });
  BlockX<double> o{};
  if (va) o.a = st[p];
  if (vb) o.b = st[p + 1];
  if (vc) o.c = st[p + LD];
  if (vd) o.d = st[p + LD + 1];
  const BlockPlanes<double> qx = block_planes(sm + L::X, NB + 2, NB + 2, bi, bj);
  const BlockPlanes<double> qt = block_planes(sm + L::T, NB + 2, NB + 2, bi, bj);
  const BlockX<double> zero{};
  auto sync = [] { __syncthreads(); };
  auto put = [&](const BlockPlanes<double>& q, const BlockX<double>& x) {
    if (va) *q.a = x.a;
    if (vb) *q.b = x.b;
    if (vc) *q.c = x.c;
    if (vd) *q.d = x.d;
  };
  auto keep = [&](int at, int kk, const BlockX<double>& x) {   // per-thread storage of a vector's block
    if (va) {
      double* s = sm + at + kk * 4 * L::NB2 + tid;
      s[0] = x.a, s[L::NB2] = x.b, s[2 * L::NB2] = x.c, s[3 * L::NB2] = x.d;
    }
  };
  auto kept = [&](int at, int kk) {
    BlockX<double> x{};
    if (va) {
      const double* s = sm + at + kk * 4 * L::NB2 + tid;
      x.a = s[0], x.b = s[L::NB2], x.c = s[2 * L::NB2], x.d = s[3 * L::NB2];
    }
    return x;
  };
  auto restrict_to = [&](double* fc, const BlockX<double>& r, const BlockPlanes<double>& q) {
    if (vd)
      fc[pc] = block_restrict<false>(r, q, [&](int w, int dic, int djc) { return ci[w * PSC + pc + djc * LDC + dic]; });
  };
  auto add_p = [&](BlockX<double>& x, const double* ec, double sign) {   // x += sign P ec
    if (va)
      block_interp<false>(x, sign * ec[pc - LDC - 1], sign * ec[pc - LDC], sign * ec[pc - 1], sign * ec[pc], va, vb, vc,
                          vd, [&](int w) { return ci[w * PSC + pc]; });
  };
  double dw[8] = {0, 0, 0, 0, 0, 0, 0, 0};
  auto add_outer = [&](double ga, double gb, double gc, const double* ec) {   // dL/dw of <g, P ec>: g(p) ec(c)
    const double e_sw = ec[pc - LDC - 1], e_se = ec[pc - LDC], e_nw = ec[pc - 1], e_ne = ec[pc];
    dw[CI_LL] += gc * e_nw;
    dw[CI_LR] += gc * e_ne;
    dw[CI_LB] += gb * e_se;
    dw[CI_LA] += gb * e_ne;
    dw[CI_LSW] += ga * e_sw;
    dw[CI_LSE] += ga * e_se;
    dw[CI_LNW] += ga * e_nw;
    dw[CI_LNE] += ga * e_ne;
  };
  const int warp = tid >> 5;
  for (int k0 = 0; k0 < K; k0 += TG_VECS) {
    const int cnt = K - k0 < TG_VECS ? K - k0 : TG_VECS;
    for (int kk = 0; kk < cnt; ++kk) {   // e1 = S^2 e, P^T A e1
      const double* e = vecs + ((size_t)crop * K + k0 + kk) * PS;
      BlockX<double> x{};
      if (va) x.a = e[p];
      if (vb) x.b = e[p + 1];
      if (vc) x.c = e[p + LD];
      if (vd) x.d = e[p + LD + 1];
      put(qx, x);
      sync();
      block_sweep<true, false, false>(k, zero, x, qx, va, vb, vc, vd, sync);
      block_sweep<true, false, false>(k, zero, x, qx, va, vb, vc, vd, sync);
      keep(L::E, kk, x);
      BlockX<double> t = block_resid<true, false>(k, o, zero, x, qx, va, vb, vc, vd);   // -A e1
      t.a = -t.a, t.b = -t.b, t.c = -t.c, t.d = -t.d;
      put(qt, t);
      sync();
      restrict_to(sm + L::U + kk * PSC, t, qt);
      // (the next vector's qt is written after its sweeps' barriers)
    }
    sync();
    for (int kk = warp; kk < cnt; kk += L::WARPS) band_solve<N>(band, rd, sm + L::U + kk * PSC);   // u
    sync();
    for (int kk = 0; kk < cnt; ++kk) {   // e2 = e1 - P u, e3 = S e2, the energy, g2 = S^T dL/d e3
      const size_t at = (size_t)crop * K + k0 + kk;
      BlockX<double> x = kept(L::E, kk);
      add_p(x, sm + L::U + kk * PSC, -1.0);
      keep(L::E, kk, x);
      put(qx, x);
      sync();
      block_sweep<true, false, false>(k, zero, x, qx, va, vb, vc, vd, sync);
      BlockX<double> t = block_resid<true, false>(k, o, zero, x, qx, va, vb, vc, vd);   // -A e3
      double part = 0.0;
      part = rsub(part, rmul(x.a, t.a));
      part = rsub(part, rmul(x.b, t.b));
      part = rsub(part, rmul(x.c, t.c));
      part = rsub(part, rmul(x.d, t.d));
      const double energy = block_total<N>(part, red);
      if (tid == 0) energies[at] = energy;
      if (!eref) continue;
      const double sc = -rdiv(2.0 * weight, rmul((double)K, eref[at]));
      BlockX<double> g{sc * t.a, sc * t.b, sc * t.c, sc * t.d};   // dL/d e3
      sweep_adjoint(k, o, g, qx, va, vb, vc, vd, sync);
      keep(L::G, kk, g);
      put(qt, g);
      sync();
      restrict_to(sm + L::V + kk * PSC, g, qt);
    }
    if (!eref) {
      sync();
      continue;
    }
    sync();
    for (int kk = warp; kk < cnt; kk += L::WARPS) band_solve<N>(band, rd, sm + L::V + kk * PSC);   // v
    sync();
    for (int kk = 0; kk < cnt; ++kk) {   // dL/dP += (A P v - g2) u^T - (A e2) v^T
      const double *u = sm + L::U + kk * PSC, *v = sm + L::V + kk * PSC;
      BlockX<double> t{};
      add_p(t, v, 1.0);
      put(qt, t);
      const BlockX<double> e2 = kept(L::E, kk), g = kept(L::G, kk);
      put(qx, e2);
      sync();
      if (va) {
        // -(A P v) and -(A e2) at the block's A, B, C (its D carries no weight)
        const BlockX<double> pv = block_resid<true, true>(k, o, zero, t, qt, va, vb, vc, false);
        add_outer(-pv.a - g.a, -pv.b - g.b, -pv.c - g.c, u);
        const BlockX<double> ae = block_resid<true, true>(k, o, zero, e2, qx, va, vb, vc, false);
        add_outer(ae.a, ae.b, ae.c, v);
      }
      sync();
    }
  }
  if (!eref) return;
  // dL/dw -> dL/d delta: each edge weight's total derivative (its own term plus
  // the two centre formulas that use it), times S_D q (1 - q)
  double *dW = sm + L::DW, *tx = dW + 8 * PSC, *ty = tx + PSC;
  for (int e = tid; e < 10 * PSC; e += NT) dW[e] = 0.0;
  __syncthreads();
  if (va) {
#pragma unroll
    for (int w = 0; w < 8; ++w) {
      const bool on = w == CI_LL || w == CI_LR ? vc : w == CI_LB || w == CI_LA ? vb : true;
      if (on) dW[w * PSC + pc] = dw[w];
    }
  }
  __syncthreads();
  auto cc = [&](int a, int b, int kk) -> double {   // a_kk / a_O at the centre point of cell (a, b)
    if (a < 1 || b < 1 || a > NC + 1 || b > NC + 1) return 0.0;
    const size_t pp = (size_t)(2 * b - 1) * LD + (2 * a - 1);
    const double oo = A.a<0>(pp, LD);
    const double c = kk == 1 ? A.a<1>(pp, LD) : kk == 2 ? A.a<2>(pp, LD) : kk == 3 ? A.a<3>(pp, LD) : A.a<4>(pp, LD);
    return c / oo;
  };
  auto dwat = [&](int kk, int a, int b) -> double {
    if (a < 0 || b < 0 || a > NC + 1 || b > NC + 1) return 0.0;
    return dW[kk * PSC + (size_t)b * LDC + a];
  };
  for (int e = tid; e < PSC; e += NT) {
    const int ic = e % LDC, jc = e / LDC;
    double t1 = 0.0, t2 = 0.0;
    if (ic >= 1 && jc >= 1 && jc <= NC) {
      const double dll = dwat(CI_LL, ic, jc) - cc(ic, jc + 1, 3) * dwat(CI_LSW, ic, jc + 1) -
                         cc(ic, jc, 4) * dwat(CI_LNW, ic, jc);
      const double dlr = dwat(CI_LR, ic, jc) - cc(ic, jc + 1, 3) * dwat(CI_LSE, ic, jc + 1) -
                         cc(ic, jc, 4) * dwat(CI_LNE, ic, jc);
      const double sd = aux[0 * PSC + e], q = aux[1 * PSC + e];
      t1 = (dll - dlr) * sd * q * (1.0 - q);
    }
    if (ic >= 1 && ic <= NC && jc >= 1) {
      const double dlb = dwat(CI_LB, ic, jc) - cc(ic + 1, jc, 1) * dwat(CI_LSW, ic + 1, jc) -
                         cc(ic, jc, 2) * dwat(CI_LSE, ic, jc);
      const double dla = dwat(CI_LA, ic, jc) - cc(ic + 1, jc, 1) * dwat(CI_LNW, ic + 1, jc) -
                         cc(ic, jc, 2) * dwat(CI_LNE, ic, jc);
      const double sd = aux[2 * PSC + e], q = aux[3 * PSC + e];
      t2 = (dlb - dla) * sd * q * (1.0 - q);
    }
    tx[e] = t1;
    ty[e] = t2;
  }
  __syncthreads();
  float* out = ddelta + (size_t)crop * M * MLP_OUT;
  for (int c = tid; c < M; c += NT) {
    const int ic = 1 + c % NC, jc = 1 + c / NC;
    const size_t q = (size_t)jc * LDC + ic;
    out[c * MLP_OUT + 0] = (float)(-tx[q]);
    out[c * MLP_OUT + 1] = (float)(tx[q + 1]);
    out[c * MLP_OUT + 2] = (float)(-ty[q]);
    out[c * MLP_OUT + 3] = (float)(ty[q + LDC]);
  }
}

// Features of every crop: (a_W + a_E)/a_O and (a_S + a_N)/a_O at the 9 fine
// points of each interior coarse point's 3x3 block; rows crop-major.
__global__ void k_features_crops(int n, const double* __restrict__ coefs, float* __restrict__ X) {
  const int nc = (n - 1) / 2, ld = n + 2;
  const int crop = blockIdx.y;
  const size_t ps = plane_size(n);
  const Planes<double> A = planes_at(coefs + (size_t)crop * 5 * ps, ps);
  for (int c = blockIdx.x * blockDim.x + threadIdx.x; c < nc * nc; c += gridDim.x * blockDim.x) {
    const int ic = 1 + c % nc, jc = 1 + c / nc;
    float* row = X + ((size_t)crop * nc * nc + c) * MLP_IN;
    int k = 0;
    for (int dy = -1; dy <= 1; ++dy)
      for (int dx = -1; dx <= 1; ++dx) {
        const size_t p = (size_t)(2 * jc + dy) * ld + (2 * ic + dx);
        const int i = 2 * ic + dx, j = 2 * jc + dy;
        // couplings to ghost points are not entries of a Dirichlet row
        const double w = i > 1 ? A.a<1>(p, ld) : 0.0, e = i < n ? A.a<2>(p, ld) : 0.0;
        const double s = j > 1 ? A.a<3>(p, ld) : 0.0, nn = j < n ? A.a<4>(p, ld) : 0.0;
        const double o = A.a<0>(p, ld);
        const float2 v = learned::feature_pair(w, e, s, nn, o);
        row[k++] = v.x;
        row[k++] = v.y;
      }
  }
}

template <int N>
int launch_twogrid_n(int ncrop, int K, const double* coefs, const double* vecs, const float* delta, const double* eref,
                     double weight, double* energies, float* ddelta, double* aux, int* err, cudaStream_t s) {
  static PerDevice smem;
  if (int rc = cuda_check(allow_smem(smem, k_twogrid<N>, TG<N>::BYTES), "two-grid kernel shared memory")) return rc;
  k_twogrid<N><<<ncrop, TG<N>::THREADS, TG<N>::BYTES, s>>>(K, coefs, vecs, delta, eref, weight, energies, ddelta,
                                                           eref ? aux : nullptr, err);
  count_launch();
  return cuda_check(cudaGetLastError(), "two-grid kernel launch");
}

}  // namespace

bool twogrid_size_ok(int n) { return n == 7 || n == 15 || n == 31; }

int launch_twogrid(int n, int ncrop, int K, const double* coefs, const double* vecs, const float* delta,
                   const double* eref, double weight, double* energies, float* ddelta, double* aux, int* err,
                   cudaStream_t s) {
  switch (n) {
    case 7: return launch_twogrid_n<7>(ncrop, K, coefs, vecs, delta, eref, weight, energies, ddelta, aux, err, s);
    case 15: return launch_twogrid_n<15>(ncrop, K, coefs, vecs, delta, eref, weight, energies, ddelta, aux, err, s);
    case 31: return launch_twogrid_n<31>(ncrop, K, coefs, vecs, delta, eref, weight, energies, ddelta, aux, err, s);
    default: return set_error(BMG_EINVAL, "two-grid loss: crop size %d is not 7, 15 or 31", n);
  }
}

void launch_features_crops(int n, int ncrop, const double* coefs, float* X, cudaStream_t s) {
  const int nc = (n - 1) / 2;
  k_features_crops<<<dim3((nc * nc + 255) / 256, ncrop), 256, 0, s>>>(n, coefs, X);
  count_launch();
}

}  // namespace bmg
