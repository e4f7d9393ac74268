// Interval bound propagation (Sec. 2.2.3; the IBP bounding of Sec. 7.2):
//   l_hat_k = b_k + W_k^+ lo_{k-1} + W_k^- hi_{k-1},  u_hat_k = b_k + W_k^+ hi_{k-1} + W_k^- lo_{k-1}
// with [lo_0, hi_0] = the input box and [lo_k, hi_k] = [relu(l_hat_k), relu(u_hat_k)].
// Every multiply-add is rounded outward (round-down for l_hat, round-up for
// u_hat), so the FP32 results contain the exact interval bounds.  The output
// lower bound of the margin-folded last layer is formed in FP64 from the
// FP64 fold, lowered by the fold's error bound.
// One launch per layer; one warp per (row, output neuron) of a wide FC layer
// and per output bound; 4x4/stride-2 and 3x3/stride-1 convs on operand rows
// staged in shared memory, other layers one thread per (row, output neuron),
// a row being a property (root bounds) or a subdomain
// (bounds recomputed after its splits:
// the first layer reads the box of the subdomain's property, and the split
// clamp of Sec. 2.3.2 is applied to every hidden layer's bounds before they
// feed the next layer through [relu(l), relu(u)]).
#include <algorithm>

#include "ld_common.cuh"

namespace ld {
namespace {

// Input row of row p (the first layer of a subdomain reads its property's box).
__device__ __forceinline__ int ibp_src(const IbpRows& rows, int first, int p) {
  if (!first || rows.n_in_rows <= 0) return p;
  const int src = rows.in_row ? rows.in_row[p] : 0;
  return src < 0 ? 0 : (src >= rows.n_in_rows ? rows.n_in_rows - 1 : src);
}

// Stores the bounds of neuron o of row p, clamped by the row's split mask
// (+1 => l <- max(l,0); -1 => u <- min(u,0)).
__device__ __forceinline__ void ibp_store(const LayerDev& L, const IbpRows& rows, int p, int o, float lo, float hi,
                                          float* lout, float* uout, int out_stride) {
  if (rows.mask) {
    const int m = rows.mask[(size_t)p * rows.mask_stride + L.r_out_off + o];
    if (m > 0) lo = fmaxf(lo, 0.f);
    if (m < 0) hi = fminf(hi, 0.f);
  }
  lout[(size_t)p * out_stride + o] = lo;
  uout[(size_t)p * out_stride + o] = hi;
}

__global__ void ibp_kernel(LayerDev L, int first, int n_rows, const float* __restrict__ lin,
                           const float* __restrict__ uin, int in_stride, float* lout, float* uout,
                           int out_stride, int* status, IbpRows rows) {
  const size_t total = (size_t)n_rows * L.n_out;
  for (size_t e = blockIdx.x * (size_t)blockDim.x + threadIdx.x; e < total; e += (size_t)gridDim.x * blockDim.x) {
    const int p = (int)(e / L.n_out), o = (int)(e % L.n_out);
    const int src = ibp_src(rows, first, p);
    const float* lp = lin + (size_t)src * in_stride;
    const float* up = uin + (size_t)src * in_stride;
    float lo, hi;
    if (L.kind == LD_LAYER_FC) {
      lo = L.b[o];
      hi = L.b[o];
      const float* w = L.W + (size_t)o * L.n_in;
      for (int i = 0; i < L.n_in; ++i) {
        float a = lp[i], c = up[i];
        if (!first) {
          a = fmaxf(a, 0.f);
          c = fmaxf(c, 0.f);
        } else if (!(isfinite(a) && isfinite(c) && a <= c)) {
          atomicCAS(status, 0, (int)LD_ERR_NONFINITE);
        }
        const float wi = w[i];
        lo = __fmaf_rd(wi, wi >= 0.f ? a : c, lo);
        hi = __fmaf_ru(wi, wi >= 0.f ? c : a, hi);
      }
    } else {
      const int hw_o = L.ho * L.wo;
      const int oc = o / hw_o, rem = o % hw_o, y = rem / L.wo, xo = rem % L.wo;
      lo = L.b[oc];
      hi = L.b[oc];
      for (int c = 0; c < L.cin; ++c)
        for (int i = 0; i < L.kh; ++i) {
          const int yy = y * L.stride - L.pad + i;
          if (yy < 0 || yy >= L.h) continue;
          for (int j = 0; j < L.kw; ++j) {
            const int xx = xo * L.stride - L.pad + j;
            if (xx < 0 || xx >= L.w) continue;
            const size_t ii = ((size_t)c * L.h + yy) * L.w + xx;
            float a = lp[ii], cc = up[ii];
            if (!first) {
              a = fmaxf(a, 0.f);
              cc = fmaxf(cc, 0.f);
            } else if (!(isfinite(a) && isfinite(cc) && a <= cc)) {
              atomicCAS(status, 0, (int)LD_ERR_NONFINITE);
            }
            const float wi = L.W[(((size_t)oc * L.cin + c) * L.kh + i) * L.kw + j];
            lo = __fmaf_rd(wi, wi >= 0.f ? a : cc, lo);
            hi = __fmaf_ru(wi, wi >= 0.f ? cc : a, hi);
          }
        }
    }
    ibp_store(L, rows, p, o, lo, hi, lout, uout, out_stride);
  }
}

// 4x4/stride-2 and 3x3/stride-1 convs: a CTA takes one row and a band of bh
// output rows, with the (relu'd) interval ends of the inputs it reads and the
// weights in shared memory; a thread one position and two output channels.
// Each end is one chain of outward-rounded FMAs in the order (c, i, j) from the
// bias, as in ibp_kernel (a tap outside the plane adds an exact zero).  The
// chains are short; what bounds the pass is load latency, paid once per CTA
// here instead of once per product.  With ibp_out_kernel, the call on 32 Deep
// properties went from 107 to 51 us.
struct IbpTile {
  int bands, bh, rows, pitch, cols;  // cols: columns of a padded row that taps read
};
template <int KH, int KW, int ST>
__global__ void __launch_bounds__(256) ibp_conv_kernel(LayerDev L, IbpTile T, int first, const float* __restrict__ lin,
                                                       const float* __restrict__ uin, int in_stride, float* lout,
                                                       float* uout, int out_stride, int* status, IbpRows rows) {
  extern __shared__ __align__(16) float sm[];
  const int p = blockIdx.x / T.bands, y0 = (blockIdx.x % T.bands) * T.bh, ny = min(T.bh, L.ho - y0);
  const int nw = L.cout * L.cin * KH * KW, plane = T.rows * T.pitch, half = T.pitch / ST;
  float* sL = sm + nw;
  float* sU = sL + L.cin * plane;
  const int src = ibp_src(rows, first, p);
  const float* lp = lin + (size_t)src * in_stride;
  const float* up = uin + (size_t)src * in_stride;
  for (int e = threadIdx.x; e < nw; e += 256) sm[e] = __ldg(L.Wf + e);
  bool bad = false;
  for (int e = threadIdx.x; e < L.cin * plane; e += 256) {
    const int c = e / plane, rem = e - c * plane, yy = rem / T.pitch, xx = rem - yy * T.pitch;
    const int y = y0 * ST - L.pad + yy, x = xx - L.pad;
    float a = 0.f, u = 0.f;
    if (y >= 0 && y < L.h && x >= 0 && x < L.w && yy < (ny - 1) * ST + KH && xx < T.cols) {
      a = __ldg(lp + (c * L.h + y) * L.w + x);
      u = __ldg(up + (c * L.h + y) * L.w + x);
      if (!first) {
        a = fmaxf(a, 0.f);
        u = fmaxf(u, 0.f);
      } else if (!(isfinite(a) && isfinite(u) && a <= u)) {
        bad = true;
      }
    }
    const int at = c * plane + yy * T.pitch + (xx % ST) * half + xx / ST;
    sL[at] = a;
    sU[at] = u;
  }
  if (bad) atomicCAS(status, 0, (int)LD_ERR_NONFINITE);
  __syncthreads();
  const int items = L.cout / 2 * ny * L.wo;
  for (int e = threadIdx.x; e < items; e += 256) {
    const int xo = e % L.wo, r = e / L.wo, yo = r % ny, o = r / ny * 2;
    float lo[2], hi[2];
#pragma unroll
    for (int g = 0; g < 2; ++g) lo[g] = hi[g] = __ldg(L.b + o + g);
    const float* xl = sL + yo * ST * T.pitch + xo;
    const float* xu = sU + yo * ST * T.pitch + xo;
    const float* w = sm + o;
    for (int c = 0; c < L.cin; ++c, xl += plane, xu += plane, w += KH * KW * L.cout)
#pragma unroll
      for (int i = 0; i < KH; ++i)
#pragma unroll
        for (int j = 0; j < KW; ++j) {
          const int at = i * T.pitch + (j % ST) * half + j / ST;
          const float a = xl[at], u = xu[at];
#pragma unroll
          for (int g = 0; g < 2; ++g) {
            const float wi = w[(i * KW + j) * L.cout + g];
            lo[g] = __fmaf_rd(wi, wi >= 0.f ? a : u, lo[g]);
            hi[g] = __fmaf_ru(wi, wi >= 0.f ? u : a, hi[g]);
          }
        }
#pragma unroll
    for (int g = 0; g < 2; ++g)
      ibp_store(L, rows, p, ((o + g) * L.ho + y0 + yo) * L.wo + xo, lo[g], hi[g], lout, uout, out_stride);
  }
}

// Output bound of the margin-folded last layer from its FP64 row, one warp per
// row: each weight is within W64_err of the exact fold and the inputs are
// relu'd intervals, so w x >= W64 x - W64_err hi for x in [a, c], c >= 0.
// Lane q takes the inputs q, q + 32, ...; every step rounds down.
__global__ void ibp_out_kernel(LayerDev L, int n_rows, const float* __restrict__ lin, const float* __restrict__ uin,
                               int in_stride, double* out_lb) {
  const int lane = threadIdx.x & 31, p = blockIdx.x * (blockDim.x / 32) + threadIdx.x / 32;
  if (p >= n_rows) return;
  const float* lp = lin + (size_t)p * in_stride;
  const float* up = uin + (size_t)p * in_stride;
  double lod = 0.0;
  for (int i = lane; i < L.n_in; i += 32) {
    const double a = fmax((double)lp[i], 0.0), c = fmax((double)up[i], 0.0);
    const double wi = L.W64[i];
    lod = __fma_rd(wi, wi >= 0.0 ? a : c, lod);
    lod = __dsub_rd(lod, __dmul_ru(L.W64_err[i], c));
  }
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) lod = __dadd_rd(lod, __shfl_xor_sync(0xffffffffu, lod, off));
  if (lane == 0) out_lb[p] = __dadd_rd(lod, __dsub_rd(L.b64[0], L.b64[1]));
}

// FC layers (not the margin-folded last row): one warp per (row, output
// neuron); lane q takes the inputs q, q + 32, ... (coalesced weight reads),
// and the lanes' outward-rounded partial sums are added by a fixed shuffle
// tree, rounding down for l_hat and up for u_hat, then the bias.  A lane waits
// for its loads (weights from HBM or L2, once each), so from 1024 inputs on kAhead
// rounds of them go together: interval bounds of a net with 64 outputs of 16384
// inputs, one subdomain, 152 us with one round at a time, 109 so.  With fewer inputs
// that costs large batches (100-100-100-1, 10000 subdomains 634 -> 818 us).
constexpr int kAhead = 4;
template <bool AHEAD>
__global__ void ibp_fc_warp_kernel(LayerDev L, int first, int n_rows, const float* __restrict__ lin,
                                   const float* __restrict__ uin, int in_stride, float* lout, float* uout,
                                   int out_stride, int* status, IbpRows rows) {
  const int lane = threadIdx.x & 31;
  const size_t total = (size_t)n_rows * L.n_out;
  const size_t nwarp = (size_t)gridDim.x * (blockDim.x / 32);
  for (size_t e = blockIdx.x * (size_t)(blockDim.x / 32) + threadIdx.x / 32; e < total; e += nwarp) {
    const int p = (int)(e / L.n_out), o = (int)(e % L.n_out);
    const int src = ibp_src(rows, first, p);
    const float* lp = lin + (size_t)src * in_stride;
    const float* up = uin + (size_t)src * in_stride;
    const float* w = L.W + (size_t)o * L.n_in;
    float lo = 0.f, hi = 0.f;
    bool bad = false;
    const auto add = [&](float a, float c, float wi) {
      if (!first) {
        a = fmaxf(a, 0.f);
        c = fmaxf(c, 0.f);
      } else if (!(isfinite(a) && isfinite(c) && a <= c)) {
        bad = true;
      }
      lo = __fmaf_rd(wi, wi >= 0.f ? a : c, lo);
      hi = __fmaf_ru(wi, wi >= 0.f ? c : a, hi);
    };
    int i = lane;
    if (AHEAD) {
      const int full = L.n_in / (32 * kAhead) * (32 * kAhead);
      for (; i < full; i += 32 * kAhead) {
        float a[kAhead], c[kAhead], wi[kAhead];
#pragma unroll
        for (int q = 0; q < kAhead; ++q) {
          a[q] = __ldg(lp + i + 32 * q);
          c[q] = __ldg(up + i + 32 * q);
          wi[q] = __ldg(w + i + 32 * q);
        }
#pragma unroll
        for (int q = 0; q < kAhead; ++q) add(a[q], c[q], wi[q]);
      }
    }
    for (; i < L.n_in; i += 32) add(lp[i], up[i], w[i]);
    if (bad) atomicCAS(status, 0, (int)LD_ERR_NONFINITE);
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) {
      lo = __fadd_rd(lo, __shfl_xor_sync(0xffffffffu, lo, off));
      hi = __fadd_ru(hi, __shfl_xor_sync(0xffffffffu, hi, off));
    }
    if (lane == 0) {
      lo = __fadd_rd(lo, L.b[o]);
      hi = __fadd_ru(hi, L.b[o]);
      ibp_store(L, rows, p, o, lo, hi, lout, uout, out_stride);
    }
  }
}

}  // namespace

void launch_ibp_layer(const LayerDev& L, int first, int last, int n_rows, const float* lin, const float* uin,
                      int in_stride, float* lout, float* uout, int out_stride, double* out_lb, int* status,
                      cudaStream_t s, const IbpRows& rows) {
  const size_t total = (size_t)n_rows * L.n_out;
  if (last) {
    if (!out_lb || n_rows < 1) return;
    count_launch();
    ibp_out_kernel<<<(n_rows + 3) / 4, 128, 0, s>>>(L, n_rows, lin, uin, in_stride, out_lb);
    return;
  }
  count_launch();
  if (L.kind == LD_LAYER_FC && L.n_in >= 64) {
    size_t g = (total + 7) / 8;  // 8 warps per block
    if (g > 65535 * 8) g = 65535 * 8;
    const auto k = L.n_in >= 1024 ? ibp_fc_warp_kernel<true> : ibp_fc_warp_kernel<false>;
    k<<<(int)(g < 1 ? 1 : g), 256, 0, s>>>(L, first, n_rows, lin, uin, in_stride, lout, uout, out_stride, status, rows);
    return;
  }
  const int geo = L.kind != LD_LAYER_CONV ? 0 : (L.kh == 4 && L.kw == 4 && L.stride == 2) ? 1
                  : (L.kh == 3 && L.kw == 3 && L.stride == 1)                            ? 2
                                                                                         : 0;
  if (geo && L.cout % 2 == 0 && n_rows > 0) {
    // bands of about one round of items: small calls spread over the SMs
    IbpTile T{};
    T.cols = (L.wo - 1) * L.stride + L.kw;
    T.pitch = (T.cols + L.stride - 1) / L.stride * L.stride;
    T.bh = std::min(L.ho, std::max(1, 256 / (L.cout / 2 * L.wo)));
    T.bands = (L.ho + T.bh - 1) / T.bh;
    T.rows = (T.bh - 1) * L.stride + L.kh;
    const size_t smem = sizeof(float) * ((size_t)L.cout * L.cin * L.kh * L.kw + 2 * (size_t)L.cin * T.rows * T.pitch);
    if (smem <= 96 * 1024) {
      auto k = geo == 1 ? ibp_conv_kernel<4, 4, 2> : ibp_conv_kernel<3, 3, 1>;
      if (smem > 48 * 1024) cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, 96 * 1024);
      k<<<(unsigned)n_rows * T.bands, 256, smem, s>>>(L, T, first, lin, uin, in_stride, lout, uout, out_stride, status,
                                                     rows);
      return;
    }
  }
  int grid = (int)((total + 255) / 256);
  if (grid < 1) grid = 1;
  ibp_kernel<<<grid, 256, 0, s>>>(L, first, n_rows, lin, uin, in_stride, lout, uout, out_stride, status, rows);
}

}  // namespace ld
