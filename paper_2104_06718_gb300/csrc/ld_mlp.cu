// The fused FP32 iterations (all T of a launch, state resident) for nets of FC
// layers whose weights fit in shared memory beside one subdomain's state.
//
// The general fused kernel streams FC weights from L2, reads the bounds from
// global memory and runs each FC layer as a pass of its own, with four barriers
// and a chain of memory round trips per iteration: 14k cycles for the 600
// multiply-adds of a 10-20-20-1 net.  Here the weights, the clamped bounds and
// the box sit in shared memory, and an iteration is two phases: every column of
// every transposed pass (one thread each: the passes read only duals of the
// previous iteration), then every row of every forward pass with its Adam
// step (one warp per row, kRows rows in flight).  What bounds an iteration is
// the latency of these two phases: a call on one subdomain, T = 200, went from
// 1.41 to 0.54 ms.
//
// Every value is bitwise that of the general fused kernel: a column sums its
// rows in the order of that kernel's 16-row batches (rotated by the CTA that
// would own the subdomain, in two halves where that kernel splits the rows),
// a row's lanes take the same inputs and add by the same shuffle tree.
#include <algorithm>

#include "ld_common.cuh"

namespace ld {
namespace {

constexpr int NT = 256;
constexpr int kBatch = 16;  // rows of a batch of the general kernel's transposed pass
constexpr int kRows = 4;    // forward rows of a warp in flight

struct MlpLayer {
  int n_in, n_out, vec4, split;
  int w, b;                 // shared-memory offsets (floats) of W and b
  int x, r;                 // of its input x_{k-1} and of its outputs in the flat per-ReLU arrays
};
struct MlpNet {
  int n, N, n0;
  int w_floats, x_floats;   // all weights and biases; all layer inputs
  MlpLayer L[kMaxLayers];
  const float* W[kMaxLayers];
  const float* bias[kMaxLayers];
};

int round4(int x) { return (x + 3) & ~3; }

// code's threads decide whether the general kernel splits a layer's rows.
MlpNet make_mlp(const FusedNet& f, int nt) {
  MlpNet m{};
  m.n = f.n;
  int N = 0;
  for (int k = 0; k < f.n; ++k) {
    const LayerDev& D = f.L[k];
    MlpLayer& L = m.L[k];
    L.n_in = D.n_in;
    L.n_out = D.n_out;
    L.vec4 = f.F[k].vec4;
    L.split = L.vec4 && 2 * (D.n_in / 4) <= nt;
    L.w = m.w_floats;
    L.b = L.w + round4(D.n_in * D.n_out);
    m.w_floats = L.b + round4(D.n_out);
    L.x = m.x_floats;
    m.x_floats += round4(D.n_in);
    L.r = k < f.n - 1 ? D.r_out_off : 0;
    m.W[k] = D.W;
    m.bias[k] = D.b;
    if (k < f.n - 1) N += D.n_out;
  }
  m.N = N;
  m.n0 = f.L[0].n_in;
  return m;
}

// weights, layer inputs; box; bounds, rho, m, v, x_hat_B per ReLU
size_t mlp_smem(const MlpNet& m) {
  return sizeof(float) * ((size_t)m.w_floats + m.x_floats + 2 * (size_t)round4(m.n0) + 6 * (size_t)round4(m.N));
}

__global__ void __launch_bounds__(NT) mlp_kernel(const __grid_constant__ MlpNet net, const __grid_constant__ Problem P,
                                                 float* rho_g, float* m_g, float* v_g,
                                                 const __grid_constant__ FusedIter it, int S) {
  extern __shared__ __align__(16) float sm[];
  __shared__ MlpLayer sL[kMaxLayers];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, b = blockIdx.x, rot = b / S;
  const int n = net.n, N = net.N, n0 = net.n0, n04 = (n0 + 3) & ~3, N4 = (N + 3) & ~3;
  float* sW = sm;
  float* sX = sW + net.w_floats;
  float* sl0 = sX + net.x_floats;
  float* su0 = sl0 + n04;
  float* sl = su0 + n04;
  float* su = sl + N4;
  float* rho = su + N4;
  float* m = rho + N4;
  float* v = m + N4;
  float* xB = v + N4;
  const bool empty = P.empty[b] != 0;
  const int p = prop_of(P, b);
  const size_t gb = (size_t)b * N;
  for (int k = 0; k < n; ++k) {
    const int nw = net.L[k].n_in * net.L[k].n_out;
    for (int e = tid; e < nw; e += NT) sW[net.L[k].w + e] = __ldg(net.W[k] + e);
    for (int e = tid; e < net.L[k].n_out; e += NT) sW[net.L[k].b + e] = __ldg(net.bias[k] + e);
  }
  if (tid < n) sL[tid] = net.L[tid];
  for (int e = tid; e < n0; e += NT) {
    sl0[e] = P.l0[(size_t)p * n0 + e];
    su0[e] = P.u0[(size_t)p * n0 + e];
  }
  for (int j = tid; j < N; j += NT) {
    clamped_bounds(P, b, j, sl[j], su[j]);
    rho[j] = it.crown ? 0.f : rho_g[gb + j];
    m[j] = m_g[gb + j];
    v[j] = v_g[gb + j];
  }
  __syncthreads();

  // g of input i of layer L (index k: into layer k) from the duals of its outputs
  const auto column = [&](const MlpLayer& L, int i) {
    const float* w = sW + L.w + i;
    const float* r = rho + L.r;
    if (!L.vec4) {
      float a = 0.f;
#pragma unroll 4
      for (int o = 0; o < L.n_out; ++o) a = fmaf(w[o * L.n_in], r[o], a);
      return a;
    }
    const int nbat = (L.n_out + kBatch - 1) / kBatch, mid = L.split ? (nbat + 1) / 2 : nbat;
    float part[2] = {0.f, 0.f};
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const int lo = h ? mid : 0, nb = (h ? nbat : mid) - lo;
      float a = 0.f;
      for (int bi = 0; bi < nb; ++bi) {
        const int o0 = kBatch * (lo + (bi + rot) % nb), on = min(kBatch, L.n_out - o0);
#pragma unroll 4
        for (int u = 0; u < on; ++u) a = fmaf(w[(o0 + u) * L.n_in], r[o0 + u], a);
      }
      part[h] = a;
    }
    return L.split ? part[0] + part[1] : part[0];
  };
  // CROWN dual of ReLU j at g (as the general kernel's epilogue)
  const auto crown = [&](int j, float g) {
    const float l = sl[j], u = su[j];
    float a_up, a_lo;
    if (u <= 0.f) {
      a_up = 0.f;
      a_lo = 0.f;
    } else if (l >= 0.f) {
      a_up = 1.f;
      a_lo = 1.f;
    } else {
      a_up = u / (u - l);
      a_lo = (u >= -l) ? 1.f : 0.f;
    }
    rho[j] = a_up * fmaxf(g, 0.f) + a_lo * fminf(g, 0.f);
  };
  if (it.crown) {
    for (int i = tid; i < sL[n - 1].n_in; i += NT) crown(sL[n - 2].r + i, -sW[sL[n - 1].w + i]);
    __syncthreads();
    for (int k = n - 2; k >= 1; --k) {
      for (int i = tid; i < sL[k].n_in; i += NT) crown(sL[k - 1].r + i, column(sL[k], i));
      __syncthreads();
    }
  }
  for (int t = 0; t < it.T; ++t) {
    const AdamStep st = it.step[t];
    // phase 1: the inputs x_k of every layer k+1 (and x_hat_B,k): layers top down
    {
      int i = tid, k = n - 1;
      while (k >= 0) {
        const MlpLayer& L = sL[k];
        if (i >= L.n_in) {
          i -= L.n_in;
          --k;
          continue;
        }
        const float g = k == n - 1 ? -sW[L.w + i] : column(L, i);
        if (k == 0) {
          sX[L.x + i] = g >= 0.f ? su0[i] : sl0[i];
        } else {
          const int j = sL[k - 1].r + i;
          float xb, xv;
          int code;
          relu_argmin<float>(rho[j], g, sl[j], su[j], xb, xv, code);
          sX[L.x + i] = xv;
          xB[j] = xb;
        }
        i += NT;
      }
    }
    __syncthreads();
    // phase 2: rows of the hidden layers, kRows of a warp together
    {
      int j0 = kRows * warp, k = 0;
      while (k < n - 1) {
        const MlpLayer& L = sL[k];
        if (j0 >= L.n_out) {
          j0 -= (L.n_out + kRows - 1) / kRows * kRows;
          ++k;
          continue;
        }
        float acc[kRows];
#pragma unroll
        for (int q = 0; q < kRows; ++q) acc[q] = 0.f;
        const float* x = sX + L.x;
        if (L.vec4) {
          for (int c = lane; c < L.n_in / 4; c += 32) {
            const float4 xv = *reinterpret_cast<const float4*>(x + 4 * c);
#pragma unroll
            for (int q = 0; q < kRows; ++q) {
              const int j = min(j0 + q, L.n_out - 1);
              const float4 a = *reinterpret_cast<const float4*>(sW + L.w + j * L.n_in + 4 * c);
              acc[q] = fmaf(a.x, xv.x, fmaf(a.y, xv.y, fmaf(a.z, xv.z, fmaf(a.w, xv.w, acc[q]))));
            }
          }
        } else {
          for (int c = lane; c < L.n_in; c += 32) {
            const float xv = x[c];
#pragma unroll
            for (int q = 0; q < kRows; ++q) acc[q] = fmaf(sW[L.w + min(j0 + q, L.n_out - 1) * L.n_in + c], xv, acc[q]);
          }
        }
#pragma unroll
        for (int off = 16; off > 0; off >>= 1)
#pragma unroll
          for (int q = 0; q < kRows; ++q) acc[q] += __shfl_xor_sync(0xffffffffu, acc[q], off);
        float a = acc[0];
#pragma unroll
        for (int q = 1; q < kRows; ++q) a = lane == q ? acc[q] : a;
        if (lane < kRows && j0 + lane < L.n_out && !empty) {
          const int jj = j0 + lane, j = L.r + jj;
          const float xa = a + sW[L.b + jj];
          const float sg = xB[j] - xa;
          const float mm = it.beta1 * m[j] + (1.f - it.beta1) * sg;
          const float vv = it.beta2 * v[j] + (1.f - it.beta2) * sg * sg;
          m[j] = mm;
          v[j] = vv;
          rho[j] = rho[j] + st.alpha * (mm * st.inv_bc1) / (sqrtf(vv * st.inv_bc2) + it.eps);
        }
        j0 += kRows * (NT / 32);
      }
    }
    __syncthreads();
  }
  for (int j = tid; j < N; j += NT) {
    rho_g[gb + j] = rho[j];
    m_g[gb + j] = m[j];
    v_g[gb + j] = v[j];
  }
}

}  // namespace

// Whether the net is all FC and its weights and one subdomain's state fit:
// kMlpSmem keeps two CTAs on an SM.
constexpr size_t kMlpSmem = 100 * 1024;
bool mlp_covers(const FusedNet& f) {
  for (int k = 0; k < f.n; ++k)
    if (f.L[k].kind != LD_LAYER_FC || (size_t)f.L[k].n_in * f.L[k].n_out > kMlpSmem) return false;
  return f.n >= 2 && mlp_smem(make_mlp(f, NT)) <= kMlpSmem;
}

// Nets of one hidden layer and many inputs gain little: an iteration is one pass
// over the same W_1 each way, which the general kernel also does in two phases, and
// S >= 2 subdomains of its CTA share each weight it loads.  Its form is taken for
//  * one subdomain an SM and 512 threads, W_1 over 64 KB of more than 640 inputs
//    (784-24-1, T = 100, one subdomain: 478 us, 494 here; 784-10-1 423, 397), and
//  * S >= 2 and 256 threads, more than 256 inputs and 1.5 times the subdomains that
//    the GPU holds of this kernel (784-24-1, 1200 subdomains, T = 200: 2.9 ms, 4.2
//    here; 300-60-1 3.8, 4.2; 300 subdomains of it 1.7, 1.1).
bool mlp_faster(const FusedNet& f, int code, int B) {
  const int S = code & ~kFusedWide, n0 = f.L[0].n_in;
  const bool wide = (code & kFusedWide) != 0;
  if (f.n != 2 || n0 <= 256 || (S > 1 && wide)) return true;
  static int n_sm = 0;
  if (!n_sm) {
    int dev = 0, v = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&v, cudaDevAttrMultiProcessorCount, dev);
    n_sm = v > 0 ? v : 1;
  }
  if (S == 1) return !(wide && n0 > 640 && n0 * f.L[0].n_out > 16384 && B <= n_sm);
  const int per_sm = (int)std::min<size_t>(2048 / NT, (228 * 1024) / (mlp_smem(make_mlp(f, NT)) + 1024));
  return B <= 3 * n_sm * per_sm / 2;
}

cudaError_t launch_mlp(const FusedNet& f, int code, const Problem& P, float* rho, float* m, float* v,
                       const FusedIter& it, cudaStream_t s) {
  const MlpNet net = make_mlp(f, (code & kFusedWide) ? 512 : 256);
  const size_t sm = mlp_smem(net);
  const cudaError_t e = cudaFuncSetAttribute(mlp_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kMlpSmem);
  if (e != cudaSuccess) return e;
  count_launch();
  mlp_kernel<<<P.B, NT, sm, s>>>(net, P, rho, m, v, it, code & ~kFusedWide);
  return cudaGetLastError();
}

}  // namespace ld
