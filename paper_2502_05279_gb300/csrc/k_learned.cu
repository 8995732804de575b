// Learned interpolation: features, the 18-64-64-4 GELU network (FP32 training
// forward/backward, BF16 tensor-core inference), the learned weights (Dendy's
// edge sums split by the network's logits, Dendy's centre formula) and the
// test-vector training loss with its gradient, plus Adam.  The paper has no
// learned component; the method is the project's extension of Dendy's
// interpolation, with Dendy's weights exactly at zero network output.
#include <cuda_bf16.h>
#include <math.h>

#include "common.cuh"
#include "kernels.h"
#include "learned.h"
#include "learned_device.cuh"

namespace bmg {
namespace {

constexpr int NI = MLP_IN, NH = MLP_HID, NO = MLP_OUT;
constexpr int OFF_W1 = 0, OFF_B1 = OFF_W1 + NI * NH, OFF_W2 = OFF_B1 + NH, OFF_B2 = OFF_W2 + NH * NH,
              OFF_W3 = OFF_B2 + NH, OFF_B3 = OFF_W3 + NH * NO, NPAR = OFF_B3 + NO;
static_assert(NPAR == MLP_PARAMS, "parameter layout");

__device__ __forceinline__ float gelu(float z) { return 0.5f * z * (1.0f + erff(z * 0.70710678118654752f)); }
__device__ __forceinline__ float gelu_grad(float z) {
  return 0.5f * (1.0f + erff(z * 0.70710678118654752f)) + z * expf(-0.5f * z * z) * 0.39894228040143268f;
}

// ---- features: (a_W + a_E)/a_O and (a_S + a_N)/a_O at the 9 fine points of
// the 3x3 block of every interior coarse point (dy outer, dx inner) ------------
// A CTA forms each fine point's pair once (learned::feature_pair) for a tile of
// FX x FY coarse points, into shared memory.
constexpr int FX = 32, FY = 4;                 // coarse tile
constexpr int FPX = 2 * FX + 1, FPY = 2 * FY + 1;   // its fine points
__device__ __forceinline__ void feature_tile(const double* __restrict__ st, int n, int bx, int by,
                                             float2 (*f)[FPX + 1]) {
  const int nc = (n - 1) / 2, ld = n + 2;
  const Planes<double> A = planes_at(st, plane_size(n));
  for (int e = threadIdx.x; e < FPX * FPY; e += blockDim.x) {
    const int a = e % FPX, b = e / FPX;
    const int i = 2 * (bx * FX) + 1 + a, j = 2 * (by * FY) + 1 + b;   // from (2 ic0 - 1, 2 jc0 - 1)
    float2 v = make_float2(0.0f, 0.0f);
    if (i <= 2 * nc + 1 && j <= 2 * nc + 1) {
      const size_t p = (size_t)j * ld + i;
      v = learned::feature_pair(A.a<1>(p, ld), A.a<2>(p, ld), A.a<3>(p, ld), A.a<4>(p, ld), A.a<0>(p, ld));
    }
    f[b][a] = v;
  }
}

__global__ void __launch_bounds__(128) k_features(int n, const double* __restrict__ st, float* __restrict__ X) {
  __shared__ float2 f[FPY][FPX + 1];
  const int nc = (n - 1) / 2;
  feature_tile(st, n, blockIdx.x, blockIdx.y, f);
  __syncthreads();
  for (int e = threadIdx.x; e < FX * FY * NI; e += blockDim.x) {
    const int row = e / (FX * NI), c = e % (FX * NI) / NI, k = e % NI, q = k / 2;
    const int ic = blockIdx.x * FX + c + 1, jc = blockIdx.y * FY + row + 1;
    if (ic > nc || jc > nc) continue;
    const float2 v = f[2 * row + q / 3][2 * c + q % 3];
    X[((size_t)(jc - 1) * nc + (ic - 1)) * NI + k] = k & 1 ? v.y : v.x;
  }
}

// ---- training forward and backward (FP32) --------------------------------------------
// A CTA takes TR rows; thread t owns a 4 x 4 tile of the rows' 64 outputs (rows
// 4 (t / 16) .., columns 4 (t % 16) ..), so that a step of a matrix product
// reads two float4 of shared memory for 16 multiply-adds.  Every sum runs in
// increasing index order.  One row per thread, with its activations in local
// memory, took 60 us forward and 387 us backward (one warp of eight formed the
// deltas, 32 lanes on one bank) on 34200 rows; now 22 and 60 us.
constexpr int TR = 64;          // rows per tile
constexpr int TP = NH + 4;      // row pitch of the 64-wide tiles (float4 aligned)
constexpr int BWD_BLOCKS = 304; // two CTAs per SM

__device__ __forceinline__ float4 ld4(const float* p) { return *reinterpret_cast<const float4*>(p); }

__global__ void __launch_bounds__(256) k_mlp_fwd(const float* __restrict__ X, int M, const float* __restrict__ par,
                                                 float* __restrict__ Z1, float* __restrict__ Z2,
                                                 float* __restrict__ out) {
  __shared__ __align__(16) float w[NPAR];
  __shared__ __align__(16) float sx[TR * NI], sh[TR * TP];
  const int t = threadIdx.x, r0 = blockIdx.x * TR;
  for (int k = t; k < NPAR; k += 256) w[k] = par[k];
  for (int k = t; k < TR * NI; k += 256) sx[k] = r0 + k / NI < M ? X[(size_t)r0 * NI + k] : 0.0f;
  __syncthreads();
  const int j0 = 4 * (t % 16), q0 = 4 * (t / 16);
  float z[4][4];
  auto start = [&](int off) {
#pragma unroll
    for (int a = 0; a < 4; ++a)
#pragma unroll
      for (int b = 0; b < 4; ++b) z[a][b] = w[off + j0 + b];
  };
  auto keep = [&](float* Z) {   // pre-activations to memory, GELU to sh
#pragma unroll
    for (int a = 0; a < 4; ++a) {
      if (r0 + q0 + a < M)
        *reinterpret_cast<float4*>(Z + (size_t)(r0 + q0 + a) * NH + j0) =
            make_float4(z[a][0], z[a][1], z[a][2], z[a][3]);
      *reinterpret_cast<float4*>(sh + (q0 + a) * TP + j0) =
          make_float4(gelu(z[a][0]), gelu(z[a][1]), gelu(z[a][2]), gelu(z[a][3]));
    }
  };
  start(OFF_B1);
  for (int k = 0; k < NI; ++k) {
    const float4 c = ld4(w + OFF_W1 + k * NH + j0);
#pragma unroll
    for (int a = 0; a < 4; ++a) {
      const float x = sx[(q0 + a) * NI + k];
      z[a][0] = fmaf(x, c.x, z[a][0]);
      z[a][1] = fmaf(x, c.y, z[a][1]);
      z[a][2] = fmaf(x, c.z, z[a][2]);
      z[a][3] = fmaf(x, c.w, z[a][3]);
    }
  }
  keep(Z1);
  __syncthreads();
  start(OFF_B2);
#pragma unroll 4
  for (int k = 0; k < NH; ++k) {
    const float4 c = ld4(w + OFF_W2 + k * NH + j0);
#pragma unroll
    for (int a = 0; a < 4; ++a) {
      const float x = sh[(q0 + a) * TP + k];
      z[a][0] = fmaf(x, c.x, z[a][0]);
      z[a][1] = fmaf(x, c.y, z[a][1]);
      z[a][2] = fmaf(x, c.z, z[a][2]);
      z[a][3] = fmaf(x, c.w, z[a][3]);
    }
  }
  __syncthreads();
  keep(Z2);
  __syncthreads();
  const int r = t / NO, j = t % NO;
  static_assert(TR * NO == 256, "one output per thread");
  float s = w[OFF_B3 + j];
  for (int k = 0; k < NH; ++k) s = fmaf(sh[r * TP + k], w[OFF_W3 + k * NO + j], s);
  if (r0 + r < M) out[(size_t)(r0 + r) * NO + j] = s;
}

// Partial weight gradients of a CTA's tiles (tile = blockIdx.x, += gridDim.x),
// no atomics; k_sum_partials adds the CTAs' partials in a fixed order.
struct BwdShared {
  float h1[TR * TP], d1[TR * TP], h2[TR * TP], d2[TR * TP], w2[NH * TP], x[TR * NI], o[TR * NO], w3[NH * NO];
};
__global__ void __launch_bounds__(256) k_mlp_bwd(const float* __restrict__ X, int M, const float* __restrict__ par,
                                                 const float* __restrict__ Z1, const float* __restrict__ Z2,
                                                 const float* __restrict__ dout, float* __restrict__ partial) {
  extern __shared__ __align__(16) unsigned char bwd_smem[];
  BwdShared& S = *reinterpret_cast<BwdShared*>(bwd_smem);
  const int t = threadIdx.x, j0 = 4 * (t % 16), q0 = 4 * (t / 16);
  for (int e = t; e < NH * NH; e += 256) S.w2[(e / NH) * TP + e % NH] = par[OFF_W2 + e];
  for (int e = t; e < NH * NO; e += 256) S.w3[e] = par[OFF_W3 + e];
  constexpr int W1_PER = (NI * NH + 255) / 256;
  float g1[W1_PER] = {}, g2[4][4] = {}, g3 = 0.0f, gb1 = 0.0f, gb2 = 0.0f, gb3 = 0.0f;
  for (int tile = blockIdx.x; tile * TR < M; tile += gridDim.x) {
    const int r0 = tile * TR;
    __syncthreads();
    for (int e = t; e < TR * NI; e += 256) S.x[e] = r0 + e / NI < M ? X[(size_t)r0 * NI + e] : 0.0f;
    S.o[t] = r0 + t / NO < M ? dout[(size_t)r0 * NO + t] : 0.0f;
    __syncthreads();
    // h2 and d2 = (W3 d) gelu'(z2); rows past M have zero deltas
#pragma unroll
    for (int a = 0; a < 4; ++a) {
      const int r = q0 + a;
      const bool ok = r0 + r < M;
      const float4 z = ok ? ld4(Z2 + (size_t)(r0 + r) * NH + j0) : make_float4(0.f, 0.f, 0.f, 0.f);
      const float zz[4] = {z.x, z.y, z.z, z.w};
      float h[4], d[4];
#pragma unroll
      for (int b = 0; b < 4; ++b) {
        float s = 0.0f;
#pragma unroll
        for (int j = 0; j < NO; ++j) s = fmaf(S.w3[(j0 + b) * NO + j], S.o[r * NO + j], s);
        h[b] = gelu(zz[b]);
        d[b] = s * gelu_grad(zz[b]);
      }
      *reinterpret_cast<float4*>(S.h2 + r * TP + j0) = make_float4(h[0], h[1], h[2], h[3]);
      *reinterpret_cast<float4*>(S.d2 + r * TP + j0) = make_float4(d[0], d[1], d[2], d[3]);
    }
    __syncthreads();
    // h1 and d1 = (W2 d2) gelu'(z1)
    float dh[4][4] = {};
#pragma unroll 2
    for (int j = 0; j < NH; j += 4) {
      float4 d[4], c[4];
#pragma unroll
      for (int a = 0; a < 4; ++a) d[a] = ld4(S.d2 + (q0 + a) * TP + j);
#pragma unroll
      for (int b = 0; b < 4; ++b) c[b] = ld4(S.w2 + (j0 + b) * TP + j);
#pragma unroll
      for (int a = 0; a < 4; ++a)
#pragma unroll
        for (int b = 0; b < 4; ++b) {
          dh[a][b] = fmaf(c[b].x, d[a].x, dh[a][b]);
          dh[a][b] = fmaf(c[b].y, d[a].y, dh[a][b]);
          dh[a][b] = fmaf(c[b].z, d[a].z, dh[a][b]);
          dh[a][b] = fmaf(c[b].w, d[a].w, dh[a][b]);
        }
    }
#pragma unroll
    for (int a = 0; a < 4; ++a) {
      const int r = q0 + a;
      const bool ok = r0 + r < M;
      const float4 z = ok ? ld4(Z1 + (size_t)(r0 + r) * NH + j0) : make_float4(0.f, 0.f, 0.f, 0.f);
      *reinterpret_cast<float4*>(S.h1 + r * TP + j0) = make_float4(gelu(z.x), gelu(z.y), gelu(z.z), gelu(z.w));
      *reinterpret_cast<float4*>(S.d1 + r * TP + j0) =
          make_float4(dh[a][0] * gelu_grad(z.x), dh[a][1] * gelu_grad(z.y), dh[a][2] * gelu_grad(z.z),
                      dh[a][3] * gelu_grad(z.w));
    }
    __syncthreads();
#pragma unroll 2
    for (int r = 0; r < TR; ++r) {   // W2: rows q0 .. of h1, columns j0 .. of d2
      const float4 h = ld4(S.h1 + r * TP + q0), d = ld4(S.d2 + r * TP + j0);
      const float hh[4] = {h.x, h.y, h.z, h.w};
#pragma unroll
      for (int a = 0; a < 4; ++a) {
        g2[a][0] = fmaf(hh[a], d.x, g2[a][0]);
        g2[a][1] = fmaf(hh[a], d.y, g2[a][1]);
        g2[a][2] = fmaf(hh[a], d.z, g2[a][2]);
        g2[a][3] = fmaf(hh[a], d.w, g2[a][3]);
      }
    }
#pragma unroll 2
    for (int r = 0; r < TR; ++r) {
#pragma unroll
      for (int q = 0; q < W1_PER; ++q) {
        const int e = t + 256 * q;
        if (e < NI * NH) g1[q] = fmaf(S.x[r * NI + e / NH], S.d1[r * TP + e % NH], g1[q]);
      }
      g3 = fmaf(S.h2[r * TP + t / NO], S.o[r * NO + t % NO], g3);
      if (t < NH) gb1 += S.d1[r * TP + t];
      else if (t < 2 * NH) gb2 += S.d2[r * TP + t - NH];
      else if (t < 2 * NH + NO) gb3 += S.o[r * NO + t - 2 * NH];
    }
  }
  float* out = partial + (size_t)blockIdx.x * NPAR;
#pragma unroll
  for (int q = 0; q < W1_PER; ++q)
    if (t + 256 * q < NI * NH) out[OFF_W1 + t + 256 * q] = g1[q];
#pragma unroll
  for (int a = 0; a < 4; ++a)
#pragma unroll
    for (int b = 0; b < 4; ++b) out[OFF_W2 + (q0 + a) * NH + j0 + b] = g2[a][b];
  out[OFF_W3 + t] = g3;
  if (t < NH) out[OFF_B1 + t] = gb1;
  else if (t < 2 * NH) out[OFF_B2 + t - NH] = gb2;
  else if (t < 2 * NH + NO) out[OFF_B3 + t - 2 * NH] = gb3;
}

// 32 parameters per CTA, eight running sums each, then their sum in order.
__global__ void __launch_bounds__(256) k_sum_partials(const float* __restrict__ partial, int nb,
                                                      float* __restrict__ grad) {
  __shared__ float sum[8][32];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, e = blockIdx.x * 32 + lane;
  float s = 0.0f;
  if (e < NPAR)
    for (int b = w; b < nb; b += 8) s += partial[(size_t)b * NPAR + e];
  sum[w][lane] = s;
  __syncthreads();
  if (w == 0 && e < NPAR) {
    float v = sum[0][lane];
    for (int q = 1; q < 8; ++q) v += sum[q][lane];
    grad[e] = v;
  }
}

__global__ void k_adam(float* __restrict__ par, const float* __restrict__ grad, float* __restrict__ m,
                       float* __restrict__ v, float lr, float b1, float b2, float eps, float c1, float c2) {
  int e = blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= NPAR) return;
  float g = grad[e];
  float mm = b1 * m[e] + (1.0f - b1) * g;
  float vv = b2 * v[e] + (1.0f - b2) * g * g;
  m[e] = mm;
  v[e] = vv;
  par[e] -= lr * (mm / c1) / (sqrtf(vv / c2) + eps);
}

// ---- learned weights (FP64) --------------------------------------------------------------
// delta: (nc*nc, 4) logits (W, E, S, N edge of each interior coarse point);
// the per-cell formulas are in learned_device.cuh.
__global__ void k_learned_edges(int n, const double* __restrict__ st, const float* __restrict__ delta,
                                double* __restrict__ ci, double* __restrict__ aux) {
  int ic = blockIdx.x * blockDim.x + threadIdx.x;
  int jc = blockIdx.y * blockDim.y + threadIdx.y;
  int nc = (n - 1) / 2;
  if (ic > nc + 1 || jc > nc + 1) return;
  learned::edge_cell(planes_at(st, plane_size(n)), n + 2, nc, delta, ic, jc, ci, aux);
}

__global__ void k_learned_centres(int n, const double* __restrict__ st, double* __restrict__ ci) {
  int ic = blockIdx.x * blockDim.x + threadIdx.x;
  int jc = blockIdx.y * blockDim.y + threadIdx.y;
  int nc = (n - 1) / 2;
  if (ic > nc + 1 || jc > nc + 1) return;
  learned::centre_cell(planes_at(st, plane_size(n)), n + 2, nc, ic, jc, ci);
}

// ---- test-vector loss ------------------------------------------------------------------
// err = v - P R v over the interior (R: values at coarse points).
__global__ void k_tv_err(int n, const double* __restrict__ ci, const double* __restrict__ v, double* __restrict__ err) {
  int ic = blockIdx.x * blockDim.x + threadIdx.x + 1;
  int jc = blockIdx.y * blockDim.y + threadIdx.y + 1;
  int nc = (n - 1) / 2, ldc = nc + 2, ld = n + 2;
  if (ic > nc + 1 || jc > nc + 1) return;
  size_t psc = plane_size(nc), pc = (size_t)jc * ldc + ic;
  auto vc = [&](int a, int b) -> double {   // v at coarse point (a, b), 0 on ghosts
    return (a < 1 || b < 1 || a > nc || b > nc) ? 0.0 : v[(size_t)(2 * b) * ld + 2 * a];
  };
  double e_sw = vc(ic - 1, jc - 1), e_se = vc(ic, jc - 1), e_nw = vc(ic - 1, jc), e_ne = vc(ic, jc);
  size_t pf = (size_t)(2 * jc) * ld + 2 * ic;
  if (ic <= nc && jc <= nc) err[pf] = 0.0;
  if (jc <= nc) {
    double t = radd(rmul(ci[CI_LL * psc + pc], e_nw), rmul(ci[CI_LR * psc + pc], e_ne));
    err[pf - 1] = rsub(v[pf - 1], t);
  }
  if (ic <= nc) {
    double t = radd(rmul(ci[CI_LB * psc + pc], e_se), rmul(ci[CI_LA * psc + pc], e_ne));
    err[pf - ld] = rsub(v[pf - ld], t);
  }
  double t = rmul(ci[CI_LSW * psc + pc], e_sw);
  t = radd(t, rmul(ci[CI_LSE * psc + pc], e_se));
  t = radd(t, rmul(ci[CI_LNW * psc + pc], e_nw));
  t = radd(t, rmul(ci[CI_LNE * psc + pc], e_ne));
  err[pf - ld - 1] = rsub(v[pf - ld - 1], t);
}

// Ae = A err and one block partial of err . Ae per 256-thread block (row-strided).
__global__ void __launch_bounds__(256) k_tv_apply(int n, const double* __restrict__ st, const double* __restrict__ err,
                                                  double* __restrict__ Ae, double* __restrict__ partials) {
  __shared__ double red[256];
  int ld = n + 2;
  Planes<double> A = planes_at(st, plane_size(n));
  double acc = 0.0;
  for (int j = 1 + blockIdx.x; j <= n; j += gridDim.x)
    for (int i = 1 + threadIdx.x; i <= n; i += 256) {
      size_t p = (size_t)j * ld + i;
      double s = rmul(A.a<0>(p, ld), err[p]);
      s = radd(s, rmul(A.a<1>(p, ld), err[p - 1]));
      s = radd(s, rmul(A.a<2>(p, ld), err[p + 1]));
      s = radd(s, rmul(A.a<3>(p, ld), err[p - ld]));
      s = radd(s, rmul(A.a<4>(p, ld), err[p + ld]));
      s = radd(s, rmul(A.a<5>(p, ld), err[p - ld - 1]));
      s = radd(s, rmul(A.a<6>(p, ld), err[p + ld + 1]));
      s = radd(s, rmul(A.a<7>(p, ld), err[p + ld - 1]));
      s = radd(s, rmul(A.a<8>(p, ld), err[p + 1 - ld]));
      Ae[p] = s;
      acc = radd(acc, rmul(err[p], s));
    }
  red[threadIdx.x] = acc;
  __syncthreads();
  for (int h = 128; h > 0; h >>= 1) {
    if (threadIdx.x < h) red[threadIdx.x] += red[threadIdx.x + h];
    __syncthreads();
  }
  if (threadIdx.x == 0) partials[blockIdx.x] = red[0];
}

__global__ void k_tv_energy(const double* __restrict__ partials, int np, double* __restrict__ out) {
  if (threadIdx.x != 0) return;
  double s = 0.0;
  for (int k = 0; k < np; ++k) s += partials[k];
  *out = s;
}

// dW (8 planes) += g(p) v(c) over the K vectors, g = -2 Ae / (K E_ref).
__global__ void k_tv_dw(int n, int K, const double* __restrict__ vecs, const double* __restrict__ Aes,
                        const double* __restrict__ scale, double* __restrict__ dW) {
  int ic = blockIdx.x * blockDim.x + threadIdx.x + 1;
  int jc = blockIdx.y * blockDim.y + threadIdx.y + 1;
  int nc = (n - 1) / 2, ldc = nc + 2, ld = n + 2;
  if (ic > nc + 1 || jc > nc + 1) return;
  size_t psc = plane_size(nc), pc = (size_t)jc * ldc + ic, ps = plane_size(n);
  double d[8] = {0, 0, 0, 0, 0, 0, 0, 0};
  size_t pf = (size_t)(2 * jc) * ld + 2 * ic;
  for (int k = 0; k < K; ++k) {
    const double* v = vecs + (size_t)k * ps;
    const double* Ae = Aes + (size_t)k * ps;
    double sc = scale[k];
    auto vc = [&](int a, int b) -> double {
      return (a < 1 || b < 1 || a > nc || b > nc) ? 0.0 : v[(size_t)(2 * b) * ld + 2 * a];
    };
    double e_sw = vc(ic - 1, jc - 1), e_se = vc(ic, jc - 1), e_nw = vc(ic - 1, jc), e_ne = vc(ic, jc);
    if (jc <= nc) {
      double g = sc * Ae[pf - 1];
      d[CI_LL] += g * e_nw;
      d[CI_LR] += g * e_ne;
    }
    if (ic <= nc) {
      double g = sc * Ae[pf - ld];
      d[CI_LB] += g * e_se;
      d[CI_LA] += g * e_ne;
    }
    double g = sc * Ae[pf - ld - 1];
    d[CI_LSW] += g * e_sw;
    d[CI_LSE] += g * e_se;
    d[CI_LNW] += g * e_nw;
    d[CI_LNE] += g * e_ne;
  }
  for (int k = 0; k < 8; ++k) dW[k * psc + pc] = d[k];
}

// Per cell: total derivative of its x-edge and y-edge splits (direct term plus
// the two centres that use each edge weight), as t = (dw1 - dw2) S_D q (1-q).
__global__ void k_tv_edge_t(int n, const double* __restrict__ st, const double* __restrict__ dW,
                            const double* __restrict__ aux, double* __restrict__ tx, double* __restrict__ ty) {
  int ic = blockIdx.x * blockDim.x + threadIdx.x;
  int jc = blockIdx.y * blockDim.y + threadIdx.y;
  int nc = (n - 1) / 2, ldc = nc + 2, ld = n + 2;
  if (ic > nc + 1 || jc > nc + 1) return;
  size_t psc = plane_size(nc), pc = (size_t)jc * ldc + ic;
  Planes<double> A = planes_at(st, plane_size(n));
  // a_x / a_O at the centre point of cell (a, b) = fine (2a-1, 2b-1); 0 outside 1..nc+1
  auto cc = [&](int a, int b, int K) -> double {
    if (a < 1 || b < 1 || a > nc + 1 || b > nc + 1) return 0.0;
    size_t p = (size_t)(2 * b - 1) * ld + (2 * a - 1);
    double o = A.a<0>(p, ld);
    double c = K == 1 ? A.a<1>(p, ld) : K == 2 ? A.a<2>(p, ld) : K == 3 ? A.a<3>(p, ld) : A.a<4>(p, ld);
    return c / o;
  };
  auto dw = [&](int k, int a, int b) -> double {
    if (a < 0 || b < 0 || a > nc + 1 || b > nc + 1) return 0.0;
    return dW[k * psc + (size_t)b * ldc + a];
  };
  double t1 = 0.0, t2 = 0.0;
  if (ic >= 1 && jc >= 1 && jc <= nc) {
    double dll = dw(CI_LL, ic, jc) - cc(ic, jc + 1, 3) * dw(CI_LSW, ic, jc + 1) - cc(ic, jc, 4) * dw(CI_LNW, ic, jc);
    double dlr = dw(CI_LR, ic, jc) - cc(ic, jc + 1, 3) * dw(CI_LSE, ic, jc + 1) - cc(ic, jc, 4) * dw(CI_LNE, ic, jc);
    double sd = aux[0 * psc + pc], q = aux[1 * psc + pc];
    t1 = (dll - dlr) * sd * q * (1.0 - q);
  }
  if (ic >= 1 && ic <= nc && jc >= 1) {
    double dlb = dw(CI_LB, ic, jc) - cc(ic + 1, jc, 1) * dw(CI_LSW, ic + 1, jc) - cc(ic, jc, 2) * dw(CI_LSE, ic, jc);
    double dla = dw(CI_LA, ic, jc) - cc(ic + 1, jc, 1) * dw(CI_LNW, ic + 1, jc) - cc(ic, jc, 2) * dw(CI_LNE, ic, jc);
    double sd = aux[2 * psc + pc], q = aux[3 * psc + pc];
    t2 = (dlb - dla) * sd * q * (1.0 - q);
  }
  tx[pc] = t1;
  ty[pc] = t2;
}

// dL/d delta of interior coarse point (ic, jc): W from its own cell's x-edge,
// E from cell (ic+1, jc), S from its own y-edge, N from cell (ic, jc+1).
__global__ void k_tv_ddelta(int n, const double* __restrict__ tx, const double* __restrict__ ty,
                            float* __restrict__ dd) {
  int ic = blockIdx.x * blockDim.x + threadIdx.x + 1;
  int jc = blockIdx.y * blockDim.y + threadIdx.y + 1;
  int nc = (n - 1) / 2, ldc = nc + 2;
  if (ic > nc || jc > nc) return;
  size_t pc = (size_t)jc * ldc + ic;
  float* o = dd + ((size_t)(jc - 1) * nc + (ic - 1)) * NO;
  o[0] = (float)(-tx[pc]);
  o[1] = (float)(tx[pc + 1]);
  o[2] = (float)(-ty[pc]);
  o[3] = (float)(ty[pc + ldc]);
}

// ---- inference on BF16 tensor cores (mma.sync m16n8k16, FP32 accumulate) ---------------
// A CTA walks over tiles of FX x FY coarse points; the features of a tile go
// from shared memory straight into the first layer's A fragments (a feature
// pair is one packed register), a warp takes the 2 x 16 points of a tile row,
// and layer outputs stay in registers: the accumulator fragments of two
// neighbouring 8-column tiles form the A fragment of the next layer's
// 16-column k-tile.  The weights' B fragments are formed once per CTA, in lane
// order (held in registers instead they left room for 8 warps on an SM: 239
// us).  What bounds it: the 128
// erff of a point (FP32 ALU) and 26 FP64 operations of its features.  At 2047^2
// the features (18 divisions a point, 337 us), the 75 MB array between and the
// network (weights rebuilt by every CTA, activations in local memory, 272 us)
// took 609 us in two launches; now 199 us.
__device__ __forceinline__ unsigned pack_bf16(float lo, float hi) {
  __nv_bfloat162 v = __floats2bfloat162_rn(lo, hi);
  return *reinterpret_cast<unsigned*>(&v);
}

__device__ __forceinline__ void mma_bf16(float (&d)[4], const unsigned (&a)[4], uint2 b) {
  asm volatile(
      "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, "
      "{%0,%1,%2,%3};\n"
      : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b.x), "r"(b.y));
}

// B fragment of a K x N layer at (k0, n0): rows k0 + 2 tg + {0, 1} and + 8 of column n0 + g.
__device__ __forceinline__ unsigned bfrag(const float* w, int K, int N, int k, int c) {
  const float lo = k < K && c < N ? w[k * N + c] : 0.0f, hi = k + 1 < K && c < N ? w[(k + 1) * N + c] : 0.0f;
  return pack_bf16(lo, hi);
}

// The weights' B fragments in lane order: fragment q of lane l at w[q][l];
// q = kt * 8 + nt for layer 1 (kt < 2), 16 + kt * 8 + nt for layer 2, 48 + kt for layer 3.
constexpr int FRAGS = 52;
constexpr int INFER_CTAS = 4;   // per SM
__global__ void __launch_bounds__(32 * FY, INFER_CTAS) k_mlp_infer(int n, const double* __restrict__ st,
                                                                   const float* __restrict__ par,
                                                                   float* __restrict__ out) {
  __shared__ float2 f[FPY][FPX + 1];
  __shared__ uint2 w[FRAGS][32];
  __shared__ float b1[NH], b2[NH], b3[8];
  const int nc = (n - 1) / 2, tx = (nc + FX - 1) / FX, tiles = tx * ((nc + FY - 1) / FY);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, g = lane >> 2, tg = lane & 3;
  for (int e = threadIdx.x; e < NH; e += blockDim.x) {
    b1[e] = par[OFF_B1 + e];
    b2[e] = par[OFF_B2 + e];
  }
  if (threadIdx.x < 8) b3[threadIdx.x] = threadIdx.x < NO ? par[OFF_B3 + threadIdx.x] : 0.0f;
  for (int q = warp; q < FRAGS; q += FY) {
    const int layer = q < 16 ? 0 : q < 48 ? 1 : 2, e = q - (layer == 0 ? 0 : layer == 1 ? 16 : 48);
    const int kt = layer == 2 ? e : e / 8, nt = layer == 2 ? 0 : e % 8;
    const float* src = par + (layer == 0 ? OFF_W1 : layer == 1 ? OFF_W2 : OFF_W3);
    const int K = layer == 0 ? NI : NH, N = layer == 2 ? NO : NH, k = kt * 16 + 2 * tg, c = nt * 8 + g;
    w[q][lane] = make_uint2(bfrag(src, K, N, k, c), bfrag(src, K, N, k + 8, c));
  }
  for (int tile = blockIdx.x; tile < tiles; tile += gridDim.x) {
    const int bx = tile % tx, by = tile / tx, jc = by * FY + warp + 1;
    __syncthreads();                       // the previous tile's features are read
    feature_tile(st, n, bx, by, f);
    __syncthreads();
    if (jc > nc) continue;                 // (the barriers above are the only ones)
#pragma unroll 1
    for (int m = 0; m < 2; ++m) {
      const int c0 = 16 * m + g;           // this lane's points: tile columns c0 and c0 + 8
      if (bx * FX + 16 * m >= nc) break;
      // pair q of a point: fine (dx, dy) = (q % 3 - 1, q / 3 - 1); q > 8 is padding
      auto pair = [&](int c, int q) -> unsigned {
        const float2 v = f[2 * warp + q / 3][2 * c + q % 3];
        return pack_bf16(v.x, v.y);
      };
      float acc[8][4];
#pragma unroll
      for (int nt = 0; nt < 8; ++nt) {
        acc[nt][0] = acc[nt][2] = b1[nt * 8 + 2 * tg];
        acc[nt][1] = acc[nt][3] = b1[nt * 8 + 2 * tg + 1];
      }
      const unsigned a0[4] = {pair(c0, tg), pair(c0 + 8, tg), pair(c0, tg + 4), pair(c0 + 8, tg + 4)};
      const unsigned a1[4] = {tg == 0 ? pair(c0, 8) : 0u, tg == 0 ? pair(c0 + 8, 8) : 0u, 0u, 0u};
#pragma unroll
      for (int nt = 0; nt < 8; ++nt) {
        mma_bf16(acc[nt], a0, w[nt][lane]);
        mma_bf16(acc[nt], a1, w[8 + nt][lane]);
      }
      float acc2[8][4];
#pragma unroll
      for (int nt = 0; nt < 8; ++nt) {
        acc2[nt][0] = acc2[nt][2] = b2[nt * 8 + 2 * tg];
        acc2[nt][1] = acc2[nt][3] = b2[nt * 8 + 2 * tg + 1];
      }
#pragma unroll
      for (int kt = 0; kt < 4; ++kt) {     // A fragments from GELU(layer-1 accumulators)
        const unsigned a[4] = {pack_bf16(gelu(acc[2 * kt][0]), gelu(acc[2 * kt][1])),
                               pack_bf16(gelu(acc[2 * kt][2]), gelu(acc[2 * kt][3])),
                               pack_bf16(gelu(acc[2 * kt + 1][0]), gelu(acc[2 * kt + 1][1])),
                               pack_bf16(gelu(acc[2 * kt + 1][2]), gelu(acc[2 * kt + 1][3]))};
#pragma unroll
        for (int nt = 0; nt < 8; ++nt) mma_bf16(acc2[nt], a, w[16 + kt * 8 + nt][lane]);
      }
      float acc3[4] = {b3[2 * tg], b3[2 * tg + 1], b3[2 * tg], b3[2 * tg + 1]};
#pragma unroll
      for (int kt = 0; kt < 4; ++kt) {
        const unsigned a[4] = {pack_bf16(gelu(acc2[2 * kt][0]), gelu(acc2[2 * kt][1])),
                               pack_bf16(gelu(acc2[2 * kt][2]), gelu(acc2[2 * kt][3])),
                               pack_bf16(gelu(acc2[2 * kt + 1][0]), gelu(acc2[2 * kt + 1][1])),
                               pack_bf16(gelu(acc2[2 * kt + 1][2]), gelu(acc2[2 * kt + 1][3]))};
        mma_bf16(acc3, a, w[48 + kt][lane]);
      }
      if (tg < 2) {                        // columns 2 tg, 2 tg + 1 of the four outputs
        const int ic = bx * FX + c0 + 1;
        float* row = out + ((size_t)(jc - 1) * nc + (ic - 1)) * NO + 2 * tg;
        if (ic <= nc) {
          row[0] = acc3[0];
          row[1] = acc3[1];
        }
        if (ic + 8 <= nc) {
          row[8 * NO] = acc3[2];
          row[8 * NO + 1] = acc3[3];
        }
      }
    }
  }
}

// SplitMix64 (Steele, Lea, Flood 2014) in counter form: interior point number
// k = (j-1) n + (i-1) of stream `seed` gets 2 u - 1, u = (z >> 11) 2^-53.
__global__ void k_uniform_pm1(int n, unsigned long long seed, double* __restrict__ x) {
  int i = blockIdx.x * blockDim.x + threadIdx.x + 1;
  int j = blockIdx.y * blockDim.y + threadIdx.y + 1;
  if (i > n || j > n) return;
  unsigned long long k = (unsigned long long)(j - 1) * n + (i - 1);
  unsigned long long z = seed + (k + 1ull) * 0x9E3779B97F4A7C15ull;
  z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
  z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
  z = z ^ (z >> 31);
  double u = (double)(z >> 11) * 0x1.0p-53;
  x[(size_t)j * (n + 2) + i] = 2.0 * u - 1.0;
}

dim3 grid2(int nx, int ny) { return dim3((nx + 31) / 32, (ny + 7) / 8); }

}  // namespace

void launch_features(int n, const double* st, float* X, cudaStream_t s) {
  int nc = (n - 1) / 2;
  k_features<<<dim3((nc + FX - 1) / FX, (nc + FY - 1) / FY), 128, 0, s>>>(n, st, X);
  count_launch();
}

void launch_mlp_infer(int n, const double* st, const float* par, float* out, cudaStream_t s) {
  const int nc = (n - 1) / 2, tiles = ((nc + FX - 1) / FX) * ((nc + FY - 1) / FY);
  constexpr int RESIDENT = INFER_CTAS * 152;   // a CTA keeps its weights for all of its tiles
  k_mlp_infer<<<tiles < RESIDENT ? tiles : RESIDENT, 32 * FY, 0, s>>>(n, st, par, out);
  count_launch();
}

void launch_learned_ci(int n, const double* st, const float* delta, double* ci, double* aux, cudaStream_t s) {
  int nc = (n - 1) / 2;
  k_learned_edges<<<grid2(nc + 2, nc + 2), dim3(32, 8), 0, s>>>(n, st, delta, ci, aux);
  count_launch();
  k_learned_centres<<<grid2(nc + 2, nc + 2), dim3(32, 8), 0, s>>>(n, st, ci);
  count_launch();
}

void launch_uniform_pm1(int n, unsigned long long seed, double* x, cudaStream_t s) {
  k_uniform_pm1<<<grid2(n, n), dim3(32, 8), 0, s>>>(n, seed, x);
  count_launch();
}

// Test-vector energies E_k = ||v_k - P R v_k||_A^2 (and A err_k kept in Aes).
void launch_tv_energies(int n, const double* st, const double* ci, int K, const double* vecs, double* errs,
                        double* Aes, double* partials, double* energies, cudaStream_t s) {
  int nc = (n - 1) / 2;
  size_t ps = plane_size(n);
  int G = n < 1024 ? n : 1024;
  for (int k = 0; k < K; ++k) {
    k_tv_err<<<grid2(nc + 1, nc + 1), dim3(32, 8), 0, s>>>(n, ci, vecs + k * ps, errs + k * ps);
    k_tv_apply<<<G, 256, 0, s>>>(n, st, errs + k * ps, Aes + k * ps, partials);
    k_tv_energy<<<1, 32, 0, s>>>(partials, G, energies + k);
    count_launch();
    count_launch();
    count_launch();
  }
}

void launch_tv_grad(int n, const double* st, int K, const double* vecs, const double* Aes, const double* scale,
                    const double* aux, double* dW, double* tx, double* ty, float* ddelta, cudaStream_t s) {
  int nc = (n - 1) / 2;
  k_tv_dw<<<grid2(nc + 1, nc + 1), dim3(32, 8), 0, s>>>(n, K, vecs, Aes, scale, dW);
  k_tv_edge_t<<<grid2(nc + 2, nc + 2), dim3(32, 8), 0, s>>>(n, st, dW, aux, tx, ty);
  k_tv_ddelta<<<grid2(nc, nc), dim3(32, 8), 0, s>>>(n, tx, ty, ddelta);
  count_launch();
  count_launch();
  count_launch();
}

void launch_mlp_fwd(const float* X, int M, const float* par, float* Z1, float* Z2, float* out, cudaStream_t s) {
  k_mlp_fwd<<<(M + TR - 1) / TR, 256, 0, s>>>(X, M, par, Z1, Z2, out);
  count_launch();
}

void launch_mlp_bwd(const float* X, int M, const float* par, const float* Z1, const float* Z2, const float* dout,
                    float* partial, float* grad, cudaStream_t s) {
  static PerDevice smem;
  allow_smem(smem, k_mlp_bwd, sizeof(BwdShared));   // a failure shows at the launch
  const int nb = mlp_backward_blocks(M);
  k_mlp_bwd<<<nb, 256, sizeof(BwdShared), s>>>(X, M, par, Z1, Z2, dout, partial);
  k_sum_partials<<<(NPAR + 31) / 32, 256, 0, s>>>(partial, nb, grad);
  count_launch();
  count_launch();
}

void launch_adam(float* par, const float* grad, float* m, float* v, float lr, int step, cudaStream_t s) {
  const float b1 = 0.9f, b2 = 0.999f;
  float c1 = 1.0f - powf(b1, (float)step), c2 = 1.0f - powf(b2, (float)step);
  k_adam<<<(NPAR + 255) / 256, 256, 0, s>>>(par, grad, m, v, lr, b1, b2, 1e-8f, c1, c2);
  count_launch();
}

int mlp_backward_blocks(int M) { return (M + TR - 1) / TR < BWD_BLOCKS ? (M + TR - 1) / TR : BWD_BLOCKS; }

}  // namespace bmg
