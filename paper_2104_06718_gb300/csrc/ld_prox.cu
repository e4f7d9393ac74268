// The proximal solver's elementwise and per-subdomain steps (Sec. 3.3,
// Algorithm 2).  The conditional gradient of block k is the inner
// minimisation of the supergradient method at the Augmented Lagrangian's
// duals lambda' = lambda + (x_hat_B - x_hat_A) / eta (Sec. 3.3.2), so it runs
// on the layerwise transposed and forward passes; the kernels here form
// lambda', take block k's optimal step of Eq. (optimal-gamma-gauss) and move
// the block, and apply the dual update of Eq. (momentum_updates).
// lambda' is kept current instead of re-formed before every block: a block's
// move rewrites lambda' of the two layers it changed, and the dual update
// rewrites all of it with the next iteration's eta (one formula, lam_prime,
// everywhere, so the values are those of re-forming it).
//
// The optimal step of a subdomain is a ratio of two sums over block k's
// neurons; one CTA per subdomain sums them in a fixed order (deterministic)
// before it moves the block, so a run is bitwise reproducible.
#include "ld_common.cuh"

namespace ld {
namespace {

constexpr int NT = 256;

// The weight eta of iteration t's proximal terms: linear from eta0 to eta_end,
// in double, rounded once.
__device__ __forceinline__ float eta_of(const ProxSchedule& c, int t) {
  return (float)__dadd_rn(c.eta0, __ddiv_rn(__dmul_rn(__dsub_rn(c.eta_end, c.eta0), (double)t),
                                            (double)(c.T - 1 > 1 ? c.T - 1 : 1)));
}

// Iteration state at its start (t = 0), or moved on by one iteration.  The
// captured graph holds one iteration and reads the weights from here, so that
// a call launches the same few nodes T times instead of capturing and
// updating T iterations of them.
__global__ void prox_step_kernel(ProxSchedule c, ProxIter* it, int start) {
  const int t = start ? 0 : it->t + 1;
  it->t = t;
  it->eta = eta_of(c, t);
  it->eta_next = eta_of(c, t + 1 < c.T ? t + 1 : t);
}

// lambda' = lambda + (x_hat_B - x_hat_A) / eta, with inv = 1 / eta.
__device__ __forceinline__ float lam_prime(float lam, float xb, float xa, float inv) {
  return __fmaf_rn(__fsub_rn(xb, xa), inv, lam);
}

__global__ void prox_dual_prime_kernel(Problem P, ProxState S) {
  const size_t total = (size_t)P.B * P.N;
  const float inv = 1.f / S.it->eta;
  for (size_t e = blockIdx.x * (size_t)blockDim.x + threadIdx.x; e < total; e += (size_t)gridDim.x * blockDim.x) {
    const int b = (int)(e / P.N), i = (int)(e % P.N);
    S.lp[e] = lam_prime(S.lam[e], S.xB[e], S.xA[(size_t)b * (P.N + 1) + i], inv);
  }
}

__device__ __forceinline__ double block_sum(double v, double* red) {
  for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  __syncthreads();
  if (lane == 0) red[warp] = v;
  __syncthreads();
  double t = 0.0;
  for (int w = 0; w < NT / 32; ++w) t += red[w];
  return t;
}

// One CTA per subdomain: gamma = clip(num / den, 0, 1) with
//   num = grad_B^T (x_hat_B,k - z_B,k) + grad_A^T (x_hat_A,k+1 - z_A,k+1)
//   den = ||z_B,k - x_hat_B,k||^2 / eta + ||z_A,k+1 - x_hat_A,k+1||^2 / eta   (no A term for the output)
// grad_B = lambda'_k, grad_A = -lambda'_{k+1} (1 for the output); with den = 0
// the Augmented Lagrangian is linear along the segment: gamma = 1 if it
// decreases, else 0.  Then x <- gamma z + (1 - gamma) x on both parts.
// Bound by the FP64 pipe (two FMAs a neuron; the operands are widened by
// integer instructions) and by load latency, so kU neurons of a thread load
// together; a thread sums its neurons i, i + NT, ... in that order.
constexpr int kU = 4;
__global__ void __launch_bounds__(NT) prox_block_update_kernel(Problem P, ProxState S, int off_k, int n_k, int off_k1,
                                                               int n_k1, int last) {
  __shared__ double red[NT / 32];
  __shared__ float gam_s;
  const int b = blockIdx.x;
  const float eta = S.it->eta;
  const float inv = 1.f / eta;
  const size_t rb = (size_t)b * P.N, ra = (size_t)b * (P.N + 1);
  float* xB = S.xB + rb + off_k;
  const float* zB = S.zB + rb + off_k;
  const float* lamB = S.lam + rb + off_k;
  const float* xAk = S.xA + ra + off_k;
  float* xA = S.xA + ra + (last ? P.N : off_k1);
  const float* zA = S.zA + ra + (last ? P.N : off_k1);
  float* lp1 = S.lp + rb + off_k1;
  double num = 0.0, den = 0.0;
  for (int i0 = threadIdx.x; i0 < n_k; i0 += kU * NT) {
    float xb[kU], zb[kU], la[kU], xa[kU];
#pragma unroll
    for (int q = 0; q < kU; ++q) {
      const int i = i0 + q * NT;
      const bool in = i < n_k;
      xb[q] = in ? xB[i] : 0.f;
      zb[q] = in ? zB[i] : 0.f;
      la[q] = in ? lamB[i] : 0.f;
      xa[q] = in ? xAk[i] : 0.f;
    }
#pragma unroll
    for (int q = 0; q < kU; ++q) {
      if (i0 + q * NT >= n_k) continue;
      const float lpk = lam_prime(la[q], xb[q], xa[q], inv);
      const double d = widen(zb[q] - xb[q]);
      num -= widen(lpk) * d;
      den += d * d;
    }
  }
  double denA = 0.0;
  for (int i0 = threadIdx.x; i0 < n_k1; i0 += kU * NT) {
    float xa[kU], za[kU], lp[kU];
#pragma unroll
    for (int q = 0; q < kU; ++q) {
      const int i = i0 + q * NT;
      const bool in = i < n_k1;
      xa[q] = in ? xA[i] : 0.f;
      za[q] = in ? zA[i] : 0.f;
      lp[q] = in && !last ? lp1[i] : -1.f;
    }
#pragma unroll
    for (int q = 0; q < kU; ++q) {
      if (i0 + q * NT >= n_k1) continue;
      const double d = widen(za[q] - xa[q]);
      num -= widen(-lp[q]) * d;
      if (!last) denA += d * d;
    }
  }
  num = block_sum(num, red);
  den = block_sum(den + denA, red);
  if (threadIdx.x == 0) {
    den /= (double)eta;
    double g;
    if (den > 0.0) g = fmin(fmax(num / den, 0.0), 1.0);
    else g = num > 0.0 ? 1.0 : 0.0;
    gam_s = (float)g;
  }
  __syncthreads();
  const float g = gam_s, h = 1.f - g;
  if (P.empty[b]) return;
  // move the block, and rewrite lambda' of the layers it changed
  float* lpB = S.lp + rb + off_k;
#pragma unroll kU
  for (int i = threadIdx.x; i < n_k; i += NT) {
    const float xb = fmaf(g, zB[i], h * xB[i]);
    xB[i] = xb;
    lpB[i] = lam_prime(lamB[i], xb, xAk[i], inv);
  }
  const float* lam1 = S.lam + rb + off_k1;
  const float* xB1 = S.xB + rb + off_k1;
#pragma unroll kU
  for (int i = threadIdx.x; i < n_k1; i += NT) {
    const float xa = fmaf(g, zA[i], h * xA[i]);
    xA[i] = xa;
    if (!last) lp1[i] = lam_prime(lam1[i], xB1[i], xa, inv);
  }
}

// The dual update, and lambda' for the next iteration's eta.
__global__ void prox_dual_update_kernel(Problem P, ProxState S, float mu) {
  const size_t total = (size_t)P.B * P.N;
  const float inv = 1.f / S.it->eta, inv_next = 1.f / S.it->eta_next;
  for (size_t e = blockIdx.x * (size_t)blockDim.x + threadIdx.x; e < total; e += (size_t)gridDim.x * blockDim.x) {
    const int b = (int)(e / P.N), i = (int)(e % P.N);
    if (P.empty[b]) continue;
    const float xb = S.xB[e], xa = S.xA[(size_t)b * (P.N + 1) + i];
    const float step = (xb - xa) * inv;
    const float p = fmaf(mu, S.pi[e], step);
    S.pi[e] = p;
    const float lam = S.lam[e] + p;
    S.lam[e] = lam;
    S.lp[e] = lam_prime(lam, xb, xa, inv_next);
  }
}

int grid_of(size_t total) {
  size_t g = (total + NT - 1) / NT;
  if (g > 65535u * 8u) g = 65535u * 8u;
  return (int)(g > 0 ? g : 1);
}

}  // namespace

void launch_prox_step(const ProxSchedule& c, const ProxState& S, int start, cudaStream_t s) {
  count_launch();
  prox_step_kernel<<<1, 1, 0, s>>>(c, S.it, start);
}

void launch_prox_dual_prime(const Problem& P, const ProxState& S, cudaStream_t s) {
  if (P.B == 0) return;
  count_launch();
  prox_dual_prime_kernel<<<grid_of((size_t)P.B * P.N), NT, 0, s>>>(P, S);
}

void launch_prox_block_update(const Problem& P, const ProxState& S, int off_k, int n_k, int off_k1, int n_k1,
                              int last, cudaStream_t s) {
  if (P.B == 0) return;
  count_launch();
  prox_block_update_kernel<<<P.B, NT, 0, s>>>(P, S, off_k, n_k, off_k1, n_k1, last);
}

void launch_prox_dual_update(const Problem& P, const ProxState& S, float mu, cudaStream_t s) {
  if (P.B == 0) return;
  count_launch();
  prox_dual_update_kernel<<<grid_of((size_t)P.B * P.N), NT, 0, s>>>(P, S, mu);
}

}  // namespace ld
