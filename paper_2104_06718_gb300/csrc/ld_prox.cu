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
#include "ld_conv.cuh"

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

// Block k of one subdomain: x_hat_B,k (n_k neurons from flat index off_k; k = 0:
// none) and x_hat_A,k+1 (n_k1 from off_k1; last: the output, column N of xA).
struct ProxBlock {
  int off_k, n_k, off_k1, n_k1, last;
};

// The optimal step of block k and its move: gamma = clip(num / den, 0, 1) with
//   num = grad_B^T (x_hat_B,k - z_B,k) + grad_A^T (x_hat_A,k+1 - z_A,k+1)
//   den = ||z_B,k - x_hat_B,k||^2 / eta + ||z_A,k+1 - x_hat_A,k+1||^2 / eta   (no A term for the output)
// grad_B = lambda'_k, grad_A = -lambda'_{k+1} (1 for the output); with den = 0
// the Augmented Lagrangian is linear along the segment: gamma = 1 if it
// decreases, else 0.  Then x <- gamma z + (1 - gamma) x on both parts, and
// lambda' of the layers the move changed.  zB(i), zA(i): the conditional
// gradient.  The first NT threads of the CTA sum, thread t the neurons t,
// t + NT, ... in that order (kU of them load together; the operands are widened
// by integer instructions, the FP64 pipe does two FMAs a neuron); all nt move.
constexpr int kU = 4;
template <class FB, class FA>
__device__ __forceinline__ void prox_move(const Problem& P, const ProxState& S, const ProxBlock& K, int b, int nt, FB zB,
                                          FA zA) {
  __shared__ double red[2][NT / 32];
  __shared__ float gam_s;
  const float eta = S.it->eta;
  const float inv = 1.f / eta;
  const size_t rb = (size_t)b * P.N, ra = (size_t)b * (P.N + 1);
  float* xB = S.xB + rb + K.off_k;
  const float* lamB = S.lam + rb + K.off_k;
  const float* xAk = S.xA + ra + K.off_k;
  float* xA = S.xA + ra + (K.last ? P.N : K.off_k1);
  float* lp1 = S.lp + rb + K.off_k1;
  if (threadIdx.x < NT) {
    double num = 0.0, den = 0.0, denA = 0.0;
    for (int i0 = threadIdx.x; i0 < K.n_k; i0 += kU * NT) {
      float xb[kU], zb[kU], la[kU], xa[kU];
#pragma unroll
      for (int q = 0; q < kU; ++q) {
        const int i = i0 + q * NT;
        const bool in = i < K.n_k;
        xb[q] = in ? xB[i] : 0.f;
        zb[q] = in ? zB(i) : 0.f;
        la[q] = in ? lamB[i] : 0.f;
        xa[q] = in ? xAk[i] : 0.f;
      }
#pragma unroll
      for (int q = 0; q < kU; ++q) {
        if (i0 + q * NT >= K.n_k) continue;
        const float lpk = lam_prime(la[q], xb[q], xa[q], inv);
        const double d = widen(zb[q] - xb[q]);
        num -= widen(lpk) * d;
        den += d * d;
      }
    }
    for (int i0 = threadIdx.x; i0 < K.n_k1; i0 += kU * NT) {
      float xa[kU], za[kU], lp[kU];
#pragma unroll
      for (int q = 0; q < kU; ++q) {
        const int i = i0 + q * NT;
        const bool in = i < K.n_k1;
        xa[q] = in ? xA[i] : 0.f;
        za[q] = in ? zA(i) : 0.f;
        lp[q] = in && !K.last ? lp1[i] : -1.f;
      }
#pragma unroll
      for (int q = 0; q < kU; ++q) {
        if (i0 + q * NT >= K.n_k1) continue;
        const double d = widen(za[q] - xa[q]);
        num -= widen(-lp[q]) * d;
        if (!K.last) denA += d * d;
      }
    }
    den += denA;
    for (int o = 16; o > 0; o >>= 1) {
      num += __shfl_down_sync(0xffffffffu, num, o);
      den += __shfl_down_sync(0xffffffffu, den, o);
    }
    if ((threadIdx.x & 31) == 0) {
      red[0][threadIdx.x >> 5] = num;
      red[1][threadIdx.x >> 5] = den;
    }
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    double num = 0.0, den = 0.0;
    for (int w = 0; w < NT / 32; ++w) {
      num += red[0][w];
      den += red[1][w];
    }
    den /= (double)eta;
    double g;
    if (den > 0.0) g = fmin(fmax(num / den, 0.0), 1.0);
    else g = num > 0.0 ? 1.0 : 0.0;
    gam_s = (float)g;
  }
  __syncthreads();
  const float g = gam_s, h = 1.f - g;
  if (P.empty[b]) return;
  float* lpB = S.lp + rb + K.off_k;
#pragma unroll 4
  for (int i = threadIdx.x; i < K.n_k; i += nt) {
    const float xb = fmaf(g, zB(i), h * xB[i]);
    xB[i] = xb;
    lpB[i] = lam_prime(lamB[i], xb, xAk[i], inv);
  }
  const float* lam1 = S.lam + rb + K.off_k1;
  const float* xB1 = S.xB + rb + K.off_k1;
#pragma unroll 4
  for (int i = threadIdx.x; i < K.n_k1; i += nt) {
    const float xa = fmaf(g, zA(i), h * xA[i]);
    xA[i] = xa;
    if (!K.last) lp1[i] = lam_prime(lam1[i], xB1[i], xa, inv);
  }
}

// Vertex choice of neuron i of layer k at (lambda'_k, g): z_B, and x_k returned
// (k = 0, off_k < 0: the box argmin).
__device__ __forceinline__ float prox_vertex(const Problem& P, const ProxState& S, int off_k, int b, int i, float g,
                                             float* zB) {
  if (off_k < 0) {
    const int p = prop_of(P, b);
    return g >= 0.f ? P.u0[(size_t)p * P.n0 + i] : P.l0[(size_t)p * P.n0 + i];
  }
  float l, u, xb, xk;
  int code;
  clamped_bounds(P, b, off_k + i, l, u);
  relu_argmin<float>(S.lp[(size_t)b * P.N + off_k + i], g, l, u, xb, xk, code);
  zB[i] = xb;
  return xk;
}

// A whole step of a block whose layer k+1 is a conv of the blocked geometries:
// one CTA per subdomain forms the conditional gradient (transposed pass, vertex
// choice, forward pass, every output one chain of FMAs in the order of the
// layerwise passes) in shared memory and moves the block.  As three launches
// each pass paid its own staging, launch and a round trip of its results
// through L2 (256 Base subdomains, k = 0 and 1: 41 and 44 us in three launches,
// 23 and 27 us in one; a call with T = 100 24.7 -> 16.8 ms with the split-K
// sums added by the move and the top block in one launch too).
constexpr int kBlockNT = 512;
template <int KH, int KW, int ST, int G, int GF>
__global__ void __launch_bounds__(kBlockNT, 2) prox_conv_kernel(LayerDev L, ConvTile TT, ConvTile TF, Problem P,
                                                                ProxState S, ProxBlock K) {
  extern __shared__ __align__(16) float sm[];
  const int b = blockIdx.x, off_k = K.n_k ? K.off_k : -1;
  float* sWt = sm;
  float* sWf = sWt + TT.w_floats;
  float* sR = sWf + TF.w_floats;
  float* sX = sR + ((L.cout * TT.rows * TT.pitch + 3) & ~3);
  float* sB = sX + ((L.cin * TF.rows * TF.pitch + 3) & ~3);
  float* sA = sB + K.n_k;
  conv_t_weights(L, TT, sWt, kBlockNT);
  conv_t_rows(L, TT, sR, S.lp + (size_t)b * P.N + K.off_k1, 0, kBlockNT);
  stage_floats(sWf, L.Wf, L.cout * L.cin * KH * KW, kBlockNT);
  for (int e = threadIdx.x; e < L.cin * TF.rows * TF.pitch; e += kBlockNT) sX[e] = 0.f;
  stage_wait();
  conv_t_items<KH, KW, ST, G>(L, TT, sWt, sR, 0, L.h / ST, kBlockNT, [&](int c, int y, int x, float g) {
    sX[conv_f_at(TF, ST, c, y + L.pad, x + L.pad)] = prox_vertex(P, S, off_k, b, (c * L.h + y) * L.w + x, g, sB);
  });
  __syncthreads();
  conv_f_items<KH, KW, ST, GF>(L, TF, sWf, sX, 0, L.ho, kBlockNT, [&](int o, int y, int x, float acc) {
    sA[(o * L.ho + y) * L.wo + x] = acc + L.b[o];
  });
  __syncthreads();
  prox_move(P, S, K, b, kBlockNT, [&](int i) { return sB[i]; }, [&](int i) { return sA[i]; });
}

// The top block: layer n's one output, g = -W_n.  The dot product's ranges are
// those of the layerwise split-K pass, one chain each, added in order.
__global__ void __launch_bounds__(NT) prox_top_kernel(LayerDev L, Problem P, ProxState S, ProxBlock K, SplitK sk) {
  extern __shared__ float sm[];
  const int b = blockIdx.x, off_k = K.n_k ? K.off_k : -1, n = L.n_in;
  float* sX = sm;
  float* sB = sX + n;
  float* sW = sB + n;
  float* part = sW + n;
  __shared__ float za;
  for (int i = threadIdx.x; i < n; i += NT) {
    const float w = L.W[i];
    sW[i] = w;
    sX[i] = prox_vertex(P, S, off_k, b, i, -w, sB);
  }
  __syncthreads();
  if (threadIdx.x % 32 == 0)
    for (int z = threadIdx.x / 32; z < sk.splits; z += NT / 32) {
      float acc = 0.f;
      const int hi = min(n, (z + 1) * sk.kc);
#pragma unroll 8
      for (int i = z * sk.kc; i < hi; ++i) acc = fmaf(sX[i], sW[i], acc);
      part[z] = acc;
    }
  __syncthreads();
  if (threadIdx.x == 0) {
    float t = 0.f;
    for (int z = 0; z < sk.splits; ++z) t += part[z];
    za = t + L.b[0];
  }
  __syncthreads();
  prox_move(P, S, K, b, NT, [&](int i) { return sB[i]; }, [&](int) { return za; });
}

// The move of a block whose conditional gradient the layerwise passes formed:
// z_B in S.zB, z_A in S.zA, or (part) still as the forward pass's split-K
// partial sums, added here in their order.
__global__ void __launch_bounds__(NT) prox_block_update_kernel(Problem P, ProxState S, ProxBlock K, const float* part,
                                                               int splits, const float* bias) {
  const int b = blockIdx.x;
  float* zA = S.zA + (size_t)b * (P.N + 1) + (K.last ? P.N : K.off_k1);
  const float* zB = S.zB + (size_t)b * P.N + K.off_k;
  if (part) {
    for (int i = threadIdx.x; i < K.n_k1; i += NT) {
      float t = 0.f;
#pragma unroll 4
      for (int z = 0; z < splits; ++z) t += __ldg(part + ((size_t)z * P.B + b) * K.n_k1 + i);
      zA[i] = t + bias[i];
    }
    __syncthreads();
  }
  prox_move(P, S, K, b, NT, [&](int i) { return zB[i]; }, [&](int i) { return zA[i]; });
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

namespace {

template <int KH, int KW, int ST, int G, int GF>
void launch_conv_block(const LayerDev& L, const ConvTile& TT, const ConvTile& TF, size_t smem, int limit, const Problem& P,
                       const ProxState& S, const ProxBlock& K, cudaStream_t s) {
  cudaFuncSetAttribute(prox_conv_kernel<KH, KW, ST, G, GF>, cudaFuncAttributeMaxDynamicSharedMemorySize, limit);
  prox_conv_kernel<KH, KW, ST, G, GF><<<P.B, kBlockNT, smem, s>>>(L, TT, TF, P, S, K);
}

template <int KH, int KW, int ST>
void launch_conv_block(const LayerDev& L, const ConvTile& TT, const ConvTile& TF, size_t smem, int limit, const Problem& P,
                       const ProxState& S, const ProxBlock& K, cudaStream_t s) {
  const bool g3 = L.cin == 3, f4 = L.cout % 4 == 0;
  if (g3 && f4) launch_conv_block<KH, KW, ST, 3, 4>(L, TT, TF, smem, limit, P, S, K, s);
  else if (g3) launch_conv_block<KH, KW, ST, 3, 2>(L, TT, TF, smem, limit, P, S, K, s);
  else if (f4) launch_conv_block<KH, KW, ST, 4, 4>(L, TT, TF, smem, limit, P, S, K, s);
  else launch_conv_block<KH, KW, ST, 4, 2>(L, TT, TF, smem, limit, P, S, K, s);
}

}  // namespace

void launch_prox_block(const LayerDev* Lk, const LayerDev& Lk1, int k, int n, const Problem& P, const ProxState& S,
                       float* x, int x_off, size_t smem_limit, cudaStream_t s) {
  if (P.B == 0) return;
  const int last = k + 1 == n ? 1 : 0;
  const ProxBlock K{Lk ? Lk->r_out_off : 0, Lk ? Lk->n_out : 0, last ? 0 : Lk1.r_out_off, last ? 1 : Lk1.n_out, last};
  if (!last && conv_t_covers(Lk1) && conv_f_covers(Lk1)) {
    const ConvTile TT = conv_t_tile(Lk1, Lk1.h / Lk1.stride), TF = conv_f_tile(Lk1, Lk1.ho);
    const size_t smem = sizeof(float) * ((size_t)TT.w_floats + TF.w_floats + ((Lk1.cout * TT.rows * TT.pitch + 3) & ~3) +
                                         ((Lk1.cin * TF.rows * TF.pitch + 3) & ~3) + (size_t)K.n_k + K.n_k1);
    // two CTAs per SM, or one where the planes need it; else the layerwise passes
    if (smem + 1024 <= smem_limit) {
      count_launch();
      if (conv_geo(Lk1) == 1)
        launch_conv_block<4, 4, 2>(Lk1, TT, TF, smem, (int)smem_limit - 1024, P, S, K, s);
      else
        launch_conv_block<3, 3, 1>(Lk1, TT, TF, smem, (int)smem_limit - 1024, P, S, K, s);
      return;
    }
  }
  if (last) {
    const SplitK sk = forward_split(Lk1, P);
    const size_t smem = sizeof(float) * (3 * (size_t)Lk1.n_in + sk.splits);
    if (smem <= 40 * 1024) {
      count_launch();
      prox_top_kernel<<<P.B, NT, smem, s>>>(Lk1, P, S, K, sk);
      return;
    }
  }
  const EpiArgmin ea{P, k, Lk ? Lk->r_out_off : 0, x_off, S.lp, x, S.zB, nullptr, nullptr};
  if (last)
    launch_top_argmin(Lk1, P, ea, s);
  else
    launch_transposed_argmin(Lk1, nullptr, P, S.lp, ea, s);
  SplitK sk{};
  const bool partials = !last && Lk1.kind == LD_LAYER_FC && launch_forward_partials(Lk1, P, x, sk, s);
  if (!partials) {
    const int plane = Lk1.kind == LD_LAYER_FC ? 1 : Lk1.ho * Lk1.wo;
    const EpiStore es{P, last ? 0 : Lk1.r_out_off, plane, last, Lk1.b, S.zA};
    launch_forward_store(Lk1, P, x, es, s);
  }
  count_launch();
  prox_block_update_kernel<<<P.B, NT, 0, s>>>(P, S, K, partials ? P.splitk_part : nullptr, sk.splits, Lk1.b);
}

void launch_prox_dual_update(const Problem& P, const ProxState& S, float mu, cudaStream_t s) {
  if (P.B == 0) return;
  count_launch();
  prox_dual_update_kernel<<<grid_of((size_t)P.B * P.N), NT, 0, s>>>(P, S, mu);
}

}  // namespace ld
