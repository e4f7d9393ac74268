// Layerwise FP32 passes of the LD iteration: one launch per pass, each
// spread over the whole batch, with the inner minimisation, CROWN
// initialisation, Adam step and supergradient recording fused into their
// epilogues.
//
// Transposed pass (Sec. 5.2: the same product as a gradient backward pass):
//     g_k = W_{k+1}^T rho_{k+1}                         -> inner minimisation of layer k
// Forward pass (Sec. 5.2: the network's own forward product):
//     x_hat_A,k+1 = W_{k+1} x_k^* + b_{k+1}             -> supergradient, Adam on rho_{k+1}
//
// FC layers are SIMT GEMMs with the subdomain batch as the M dimension in
// 32 x 32 tiles, so one weight tile serves 32 subdomains, with up to 128 of K staged at once; the forward FC pass
// splits K across blocks when the output is small and the last block of a tile
// reduces the partial sums in a fixed order (deterministic) before the
// epilogue.  4x4/stride-2 and 3x3/stride-1 convs take register-blocked kernels
// on operand rows staged in shared memory (several channels per thread,
// compile-time taps, transposed conv split by stride phase); other geometries
// take direct loops.
#include "ld_conv.cuh"

namespace ld {
namespace {

constexpr int TM = 32, TN = 32, NT = 256;
constexpr int kTK = 128;   // K staged at once: the hidden FC widths and the split-K ranges of these nets in one round
constexpr int kNarrow = 16;
constexpr int kSplitStep = 16;  // split-K ranges are multiples of this

// How a launch stages and deals its outputs: TK of K at once, the least of 32, 64
// and 128 that holds its K (loads past K are issued and thrown away), and a
// thread's two columns side by side (the second one's state is in L1 when the first
// one's epilogue is done with it) or, for at most kNarrow outputs, 16 apart, one a
// thread instead of two in a row for half of them.  784-16-16-1, 20 iterations on one
// subdomain: 549 us with 128 and side by side throughout, 486 so; 2400 subdomains:
// 1272, 1095.  (Columns 16 apart throughout: 200-100-1, 2400 subdomains 860 -> 1035 us; the
// choice made in the kernel: a proximal call 16.3 -> 17.7 ms.)
template <int TK_, bool NARROW_>
struct Tile {
  static constexpr int TK = TK_;
  static constexpr bool NARROW = NARROW_;
  static __device__ __forceinline__ int col(int tx, int c) { return NARROW ? tx + 16 * c : 2 * tx + c; }
};

// Accumulates C[m0 + ty + 16r][n0 + T::col(tx, c)] (r, c in {0,1}) over k in [k_lo, k_hi):
//   C[m, n] = sum_k A[m*lda + k] * Bop(k, n)
//   W_KN:  Bop(k, n) = W[k*ldw + n]   (transposed pass: W[o, i], k = o, n = i)
//   !W_KN: Bop(k, n) = W[n*ldw + k]   (forward pass:    W[o, i], k = i, n = o)
// each output one chain of FMAs in the order of k.  The tiles are far too
// small to hide a load behind the products, so what bounds a tile is the
// number of load rounds: all of K (up to TK) is staged in one round, every
// thread's 32 loads in flight together (with 16 per round the 100 rows of the
// Base FC layer took 7 rounds of load, barrier, 16 products).
template <bool W_KN, class T>
__device__ __forceinline__ void gemm_tile(int m0, int n0, int M, int Ncol, int k_lo, int k_hi,
                                          const float* __restrict__ A, int lda, const float* __restrict__ W, int ldw,
                                          float acc[2][2]) {
  constexpr int TK = T::TK;
  __shared__ float As[TM][TK + 1];
  __shared__ __align__(16) float Bs[TK][TN + 2];
  const int t = threadIdx.x, tx = t % 16, ty = t / 16;
  for (int k0 = k_lo; k0 < k_hi; k0 += TK) {
    const int kn = min(TK, k_hi - k0);
    float av[TM * TK / NT], bv[TN * TK / NT];
#pragma unroll
    for (int e = 0; e < TM * TK / NT; ++e) {
      const int idx = t + e * NT, mm = idx / TK, kk = idx % TK;
      av[e] = (m0 + mm < M && kk < kn) ? __ldg(A + (size_t)(m0 + mm) * lda + k0 + kk) : 0.f;
    }
#pragma unroll
    for (int e = 0; e < TN * TK / NT; ++e) {
      const int idx = t + e * NT;
      const int kk = W_KN ? idx / TN : idx % TK, nn = W_KN ? idx % TN : idx / TK;
      bv[e] = (kk < kn && n0 + nn < Ncol)
                  ? (W_KN ? __ldg(W + (size_t)(k0 + kk) * ldw + n0 + nn) : __ldg(W + (size_t)(n0 + nn) * ldw + k0 + kk))
                  : 0.f;
    }
    if (k0 > k_lo) __syncthreads();
#pragma unroll
    for (int e = 0; e < TM * TK / NT; ++e) {
      const int idx = t + e * NT;
      As[idx / TK][idx % TK] = av[e];
    }
#pragma unroll
    for (int e = 0; e < TN * TK / NT; ++e) {
      const int idx = t + e * NT;
      const int nn = W_KN ? idx % TN : idx / TK;  // a thread's two columns side by side
      Bs[W_KN ? idx / TN : idx % TK][T::NARROW ? 2 * (nn % 16) + nn / 16 : nn] = bv[e];
    }
    __syncthreads();
#pragma unroll 8
    for (int kk = 0; kk < kn; ++kk) {
      const float a0 = As[ty][kk], a1 = As[ty + 16][kk];
      const float2 w = *reinterpret_cast<const float2*>(&Bs[kk][2 * tx]);
      acc[0][0] = fmaf(a0, w.x, acc[0][0]);
      acc[0][1] = fmaf(a0, w.y, acc[0][1]);
      acc[1][0] = fmaf(a1, w.x, acc[1][0]);
      acc[1][1] = fmaf(a1, w.y, acc[1][1]);
    }
  }
}

// Applies the epilogue to a thread's outputs of a tile; a reducing epilogue's
// row sums are added over the 16 threads that share a row first.
template <class T, class Epi>
__device__ __forceinline__ void gemm_epilogue(int m0, int n0, int M, int Ncol, const float (&acc)[2][2], const Epi& epi) {
  const int tx = threadIdx.x % 16, ty = threadIdx.x / 16;
#pragma unroll
  for (int r = 0; r < 2; ++r) {
    const int m = m0 + ty + 16 * r;
    double q = 0.0;
#pragma unroll
    for (int c = 0; c < 2; ++c) {
      const int n = n0 + T::col(tx, c);
      if (m < M && n < Ncol) {
        if constexpr (Epi::kReduce)
          q += epi(m, n, acc[r][c]);
        else
          epi(m, n, acc[r][c]);
      }
    }
    if constexpr (Epi::kReduce) {
      for (int o = 8; o > 0; o >>= 1) q += __shfl_down_sync(0xffffffffu, q, o, 16);
      if (tx == 0 && m < M) epi.finish(m, q);
    }
  }
}

// Full-K GEMM with the epilogue applied to every output.
template <bool W_KN, class T, class Epi>
__global__ void __launch_bounds__(NT) gemm_kernel(int M, int Ncol, int K, const float* __restrict__ A, int lda,
                                                  const float* __restrict__ W, int ldw, Epi epi) {
  const int m0 = blockIdx.y * TM, n0 = blockIdx.x * TN;
  float acc[2][2] = {{0.f, 0.f}, {0.f, 0.f}};
  gemm_tile<W_KN, T>(m0, n0, M, Ncol, 0, K, A, lda, W, ldw, acc);
  gemm_epilogue<T>(m0, n0, M, Ncol, acc, epi);
}

// Ranges of the split-K forward pass of FC layer L for B subdomains: `splits`
// ranges of kc inputs each (1: no split).
void split_of(const LayerDev& L, const Problem& P, int& splits, int& kc) {
  const int tiles_n = (L.n_out + TN - 1) / TN, tiles_m = (P.B + TM - 1) / TM;
  // split K until the grid covers the GPU about twice (304 blocks)
  splits = (304 + tiles_n * tiles_m - 1) / (tiles_n * tiles_m);
  const int kmax = (L.n_in + 63) / 64;
  if (splits > kmax) splits = kmax;
  if (splits > 16) splits = 16;
  if (!P.splitk_part || (size_t)splits * P.B * L.n_out > (size_t)P.splitk_part_cap ||
      tiles_n * tiles_m > P.splitk_count_cap)
    splits = 1;
  kc = L.n_in;
  if (splits > 1) {
    kc = ((L.n_in + splits - 1) / splits + kSplitStep - 1) / kSplitStep * kSplitStep;
    splits = (L.n_in + kc - 1) / kc;
  }
}

// The partial sums alone: part[z][m][n] of every range z, for a consumer that
// adds them itself in the order z = 0, 1, ...
template <class T>
__global__ void __launch_bounds__(NT) gemm_partials_kernel(int M, int Ncol, int K, int kc, const float* __restrict__ A,
                                                           int lda, const float* __restrict__ W, int ldw, float* part) {
  const int m0 = blockIdx.y * TM, n0 = blockIdx.x * TN, z = blockIdx.z;
  float acc[2][2] = {{0.f, 0.f}, {0.f, 0.f}};
  gemm_tile<false, T>(m0, n0, M, Ncol, z * kc, min(K, (z + 1) * kc), A, lda, W, ldw, acc);
  const int tx = threadIdx.x % 16, ty = threadIdx.x / 16;
#pragma unroll
  for (int r = 0; r < 2; ++r)
#pragma unroll
    for (int c = 0; c < 2; ++c) {
      const int m = m0 + ty + 16 * r, n = n0 + T::col(tx, c);
      if (m < M && n < Ncol) part[((size_t)z * M + m) * Ncol + n] = acc[r][c];
    }
}

// Split-K forward GEMM: block z covers K range [z*kc, (z+1)*kc); partial sums go
// to part[z][m][n]; the last block to finish a tile sums the partials in the
// order z = 0, 1, ... and applies the epilogue, then re-arms the tile counter.
template <class T, class Epi>
__global__ void __launch_bounds__(NT) gemm_splitk_kernel(int M, int Ncol, int K, int kc, const float* __restrict__ A,
                                                         int lda, const float* __restrict__ W, int ldw, float* part,
                                                         int* count, Epi epi) {
  const int m0 = blockIdx.y * TM, n0 = blockIdx.x * TN, z = blockIdx.z, splits = gridDim.z;
  const int k_lo = z * kc, k_hi = min(K, k_lo + kc);
  float acc[2][2] = {{0.f, 0.f}, {0.f, 0.f}};
  gemm_tile<false, T>(m0, n0, M, Ncol, k_lo, k_hi, A, lda, W, ldw, acc);
  const int tx = threadIdx.x % 16, ty = threadIdx.x / 16;
#pragma unroll
  for (int r = 0; r < 2; ++r)
#pragma unroll
    for (int c = 0; c < 2; ++c) {
      const int m = m0 + ty + 16 * r, n = n0 + T::col(tx, c);
      if (m < M && n < Ncol) part[((size_t)z * M + m) * Ncol + n] = acc[r][c];
    }
  __threadfence();
  __syncthreads();
  __shared__ int last;
  const int tile = blockIdx.y * gridDim.x + blockIdx.x;
  if (threadIdx.x == 0) last = (atomicAdd(&count[tile], 1) == splits - 1);
  __syncthreads();
  if (!last) return;
  __threadfence();
#pragma unroll
  for (int r = 0; r < 2; ++r)
#pragma unroll
    for (int c = 0; c < 2; ++c) {
      const int m = m0 + ty + 16 * r, n = n0 + T::col(tx, c);
      acc[r][c] = 0.f;
      if (m < M && n < Ncol)
        for (int q = 0; q < splits; ++q) acc[r][c] += __ldcg(part + ((size_t)q * M + m) * Ncol + n);
    }
  gemm_epilogue<T>(m0, n0, M, Ncol, acc, epi);
  if (threadIdx.x == 0) count[tile] = 0;
}

// One CTA's outputs of a conv pass belong to one subdomain: adds a reducing
// epilogue's sums over the CTA (fixed order, in the launch's dynamic shared
// memory, whose operands are done with) and hands them over once.
constexpr size_t kFinishSmem = sizeof(double) * NT;
template <class Epi>
__device__ __forceinline__ void cta_finish(int b, double q, float* smem, const Epi& epi) {
  if constexpr (Epi::kReduce) {
    double* red = reinterpret_cast<double*>(smem);
    __syncthreads();
    red[threadIdx.x] = q;
    __syncthreads();
    if (threadIdx.x < 32) {
      double t = 0.0;
      for (int w = 0; w < NT / 32; ++w) t += red[w * 32 + threadIdx.x];
      for (int o = 16; o > 0; o >>= 1) t += __shfl_down_sync(0xffffffffu, t, o);
      if (threadIdx.x == 0) epi.finish(b, t);
    }
  }
}

// Transposed conv, blocked (k4 s2 / k3 s1): a CTA takes one subdomain and a
// band of positions of every stride phase.  Operands come from shared memory
// (direct global reads left each thread waiting for one load per product).
template <int KH, int KW, int ST, int G, class Epi>
__global__ void __launch_bounds__(NT) conv_t_fast_kernel(LayerDev L, ConvTile T, const float* __restrict__ r, int rs,
                                                         Epi epi) {
  extern __shared__ __align__(16) float sm[];
  const int b = blockIdx.x / T.bands, q0 = (blockIdx.x % T.bands) * T.bh, nq = min(T.bh, L.h / ST - q0);
  conv_t_weights(L, T, sm, NT);
  conv_t_rows(L, T, sm + T.w_floats, r + (size_t)b * rs, q0, NT);
  stage_wait();
  conv_t_items<KH, KW, ST, G>(L, T, sm, sm + T.w_floats, q0, nq, NT,
                              [&](int c, int y, int x, float g) { epi(b, (c * L.h + y) * L.w + x, g); });
}

// Forward conv, blocked (k4 s2 / k3 s1): a CTA takes one subdomain and a band
// of output rows.
template <int KH, int KW, int ST, int GF, class Epi>
__global__ void __launch_bounds__(NT) conv_fwd_fast_kernel(LayerDev L, ConvTile T, const float* __restrict__ x, int xs,
                                                           Epi epi) {
  extern __shared__ __align__(16) float sm[];
  float* sX = sm + T.w_floats;
  const int b = blockIdx.x / T.bands, y0 = (blockIdx.x % T.bands) * T.bh, ny = min(T.bh, L.ho - y0);
  stage_floats(sm, L.Wf, L.cout * L.cin * KH * KW, NT);
  const float* xb = x + (size_t)b * xs;
  const int hw_i = L.h * L.w;
  tile_elements(L.cin, T.rows, T.pitch, NT, [&](int, int c, int yy, int xx) {
    const int y = y0 * ST + yy + T.y_off, xi = xx + T.x_off;
    const bool in = y >= 0 && y < L.h && xi >= 0 && xi < L.w;
    stage4(sX + conv_f_at(T, ST, c, yy, xx), xb + (in ? c * hw_i + y * L.w + xi : 0), in);
  });
  stage_wait();
  double q = 0.0;
  conv_f_items<KH, KW, ST, GF>(L, T, sm, sX, y0, ny, NT, [&](int o, int y, int xo, float acc) {
    const int i = (o * L.ho + y) * L.wo + xo;
    if constexpr (Epi::kReduce)
      q += epi(b, i, acc);
    else
      epi(b, i, acc);
  });
  cta_finish(b, q, sm, epi);
}

// Forward conv, direct: out[b, o, y, x] = sum_{c,i,j} W[o,c,i,j] x[b, c, y*s-p+i, x*s-p+j]
template <class Epi>
__global__ void __launch_bounds__(NT) conv_fwd_kernel(LayerDev L, const float* __restrict__ x, int xs, Epi epi) {
  extern __shared__ __align__(16) float sm[];
  float* sW = sm;
  const int nw = L.cout * L.cin * L.kh * L.kw;
  for (int e = threadIdx.x; e < nw; e += blockDim.x) sW[e] = L.W[e];
  __syncthreads();
  const int b = blockIdx.y;
  const float* xb = x + (size_t)b * xs;
  const int hw_o = L.ho * L.wo, plane = L.cout * hw_o;
  double q = 0.0;
  for (int e = blockIdx.x * blockDim.x + threadIdx.x; e < plane; e += gridDim.x * blockDim.x) {
    const int o = e / hw_o, rem = e % hw_o, y = rem / L.wo, xo = rem % L.wo;
    float acc = 0.f;
    for (int c = 0; c < L.cin; ++c) {
      const float* wc = sW + ((size_t)o * L.cin + c) * L.kh * L.kw;
      const float* xc = xb + (size_t)c * L.h * L.w;
      for (int i = 0; i < L.kh; ++i) {
        const int yy = y * L.stride - L.pad + i;
        if (yy < 0 || yy >= L.h) continue;
        for (int j = 0; j < L.kw; ++j) {
          const int xx = xo * L.stride - L.pad + j;
          if (xx < 0 || xx >= L.w) continue;
          acc = fmaf(wc[i * L.kw + j], xc[yy * L.w + xx], acc);
        }
      }
    }
    if constexpr (Epi::kReduce)
      q += epi(b, e, acc);
    else
      epi(b, e, acc);
  }
  cta_finish(b, q, sW, epi);
}

// Transposed conv, direct: g[b, c, yy, xx] = sum_{o,i,j} W[o,c,i,j] r[b, o, y, x] over
// the (y, x) with y*s - p + i = yy and x*s - p + j = xx.
template <class Epi>
__global__ void __launch_bounds__(NT) conv_t_kernel(LayerDev L, const float* __restrict__ r, int rs, Epi epi) {
  extern __shared__ __align__(16) float sm[];
  float* sW = sm;
  const int nw = L.cout * L.cin * L.kh * L.kw;
  for (int e = threadIdx.x; e < nw; e += blockDim.x) sW[e] = L.W[e];
  __syncthreads();
  const int b = blockIdx.y;
  const float* rb = r + (size_t)b * rs;
  const int hw_i = L.h * L.w, plane = L.cin * hw_i, hw_o = L.ho * L.wo;
  for (int e = blockIdx.x * blockDim.x + threadIdx.x; e < plane; e += gridDim.x * blockDim.x) {
    const int c = e / hw_i, rem = e % hw_i, yy = rem / L.w, xx = rem % L.w;
    float acc = 0.f;
    for (int i = 0; i < L.kh; ++i) {
      const int ty = yy + L.pad - i;
      if (ty < 0 || ty % L.stride) continue;
      const int y = ty / L.stride;
      if (y >= L.ho) continue;
      for (int j = 0; j < L.kw; ++j) {
        const int tx = xx + L.pad - j;
        if (tx < 0 || tx % L.stride) continue;
        const int xo = tx / L.stride;
        if (xo >= L.wo) continue;
        const float* wp = sW + ((size_t)c * L.kh + i) * L.kw + j;
        const float* rp = rb + y * L.wo + xo;
        for (int o = 0; o < L.cout; ++o) acc = fmaf(wp[(size_t)o * L.cin * L.kh * L.kw], rp[(size_t)o * hw_o], acc);
      }
    }
    epi(b, e, acc);
  }
}

// Top layer: g_{n-1} = W_n^T rho_n = -W_n (rho_n = -1), no pass needed.
template <class Epi>
__global__ void top_kernel(int B, int n, const float* __restrict__ Wn, Epi epi) {
  const size_t total = (size_t)B * n;
  for (size_t e = blockIdx.x * (size_t)blockDim.x + threadIdx.x; e < total; e += (size_t)gridDim.x * blockDim.x) {
    const int b = (int)(e / n), i = (int)(e % n);
    epi(b, i, -Wn[i]);
  }
}

// Subdomain b is empty when some clamped bound pair crosses (l > u).  One CTA
// per subdomain: bound by the latency of its loads, so they go kE at a time
// (17 us for 128 Deep subdomains with one at a time).
__global__ void __launch_bounds__(NT) empty_kernel(Problem P, int8_t* empty, int* status) {
  constexpr int kE = 8;
  const int b = blockIdx.x;
  if (threadIdx.x == 0 && P.prop && (P.prop[b] < 0 || P.prop[b] >= P.n_props)) atomicCAS(status, 0, (int)LD_ERR_ARG);
  const float* lb = P.lbk + (size_t)prop_of(P, b) * P.N;
  const float* ub = P.ubk + (size_t)prop_of(P, b) * P.N;
  const int8_t* mask = P.mask ? P.mask + (size_t)b * P.N : nullptr;
  int bad = 0;
  for (int j0 = threadIdx.x; j0 < P.N; j0 += kE * NT) {
    float l[kE], u[kE];
    int m[kE];
#pragma unroll
    for (int e = 0; e < kE; ++e) {
      const int j = j0 + e * NT;
      const bool in = j < P.N;
      l[e] = in ? __ldg(lb + j) : 0.f;
      u[e] = in ? __ldg(ub + j) : 0.f;
      m[e] = in && mask ? __ldg(mask + j) : 0;
    }
#pragma unroll
    for (int e = 0; e < kE; ++e)
      bad |= (m[e] > 0 ? fmaxf(l[e], 0.f) : l[e]) > (m[e] < 0 ? fminf(u[e], 0.f) : u[e]) ? 1 : 0;
  }
  bad = __syncthreads_or(bad);
  if (threadIdx.x == 0) empty[b] = (int8_t)(bad ? 1 : 0);
}

// Boxes must be finite with l0 <= u0, ball radii finite and >= 0; bounds
// must not be NaN.
__global__ void box_check_kernel(Problem P, int* status) {
  const size_t total = (size_t)P.n_props * P.n0;
  int bad = 0;
  for (size_t e = blockIdx.x * (size_t)blockDim.x + threadIdx.x; e < total; e += (size_t)gridDim.x * blockDim.x) {
    const float l = P.l0[e], u = P.u0[e];
    if (!(isfinite(l) && isfinite(u) && l <= u)) bad = 1;
  }
  const size_t totk = (size_t)P.n_props * P.N;
  for (size_t e = blockIdx.x * (size_t)blockDim.x + threadIdx.x; e < totk; e += (size_t)gridDim.x * blockDim.x) {
    if (isnan(P.lbk[e]) || isnan(P.ubk[e])) bad = 1;
  }
  if (P.ball_eps)  // l2-ball radii: finite and >= 0
    for (int p = blockIdx.x * blockDim.x + threadIdx.x; p < P.n_props; p += gridDim.x * blockDim.x)
      if (!(isfinite(P.ball_eps[p]) && P.ball_eps[p] >= 0.f)) bad = 1;
  if (bad) atomicCAS(status, 0, (int)LD_ERR_NONFINITE);
}

inline int grid1d(size_t total, int nt = NT) {
  size_t g = (total + nt - 1) / nt;
  return (int)(g > 65535 * 8 ? 65535 * 8 : (g < 1 ? 1 : g));
}

// Shared memory of a blocked conv CTA: two of them still share an SM.
constexpr size_t kConvSmem = 96 * 1024;

// Launches a blocked conv kernel, raising its shared-memory limit where needed.
template <class K, class... A>
void launch_blocked(K kernel, unsigned grid, size_t smem, cudaStream_t s, A... args) {
  if (smem > 44 * 1024) cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kConvSmem);
  kernel<<<grid, NT, smem, s>>>(args...);
}

// Rows per band of a blocked conv pass: the whole plane while the batch alone
// gives each of 152 SMs four CTAs; fewer (at least one round of items per CTA) for
// small batches, and what fits kConvSmem with the weights (row_bytes per
// operand row; a band of bh rows stages bh * st + extra of them).  0: not even
// one row fits.
int conv_band(int rows, int items_per_row, int B, size_t w_bytes, size_t row_bytes, int st, int extra) {
  int bh = rows;
  while (bh > 1 && (size_t)B * ((rows + bh - 1) / bh) < 4 * 152 && (bh + 1) / 2 * items_per_row >= NT) bh = (bh + 1) / 2;
  while (bh > 0 && w_bytes + row_bytes * (size_t)(bh * st + extra) > kConvSmem) bh = bh > 1 ? (bh + 1) / 2 : 0;
  return bh;
}

// Calls f(tile) for the Tile of a GEMM of n outputs over ranges of K inputs.
template <bool NARROW, class F>
void with_tk(int K, F f) {
  if (K <= 32)
    f(Tile<32, NARROW>{});
  else if (K <= 64)
    f(Tile<64, NARROW>{});
  else
    f(Tile<kTK, NARROW>{});
}
template <class F>
void with_tile(int n, int K, F f) {
  if (n <= kNarrow)
    with_tk<true>(K, f);
  else
    with_tk<false>(K, f);
}

template <class Epi>
void transposed(const LayerDev& L, const Problem& P, const float* rho, Epi epi, cudaStream_t s) {
  // g over the inputs of layer L (= the neurons of the layer below it).
  count_launch();
  const float* r = rho + L.r_out_off;
  if (L.kind == LD_LAYER_FC) {
    dim3 grid((L.n_in + TN - 1) / TN, (P.B + TM - 1) / TM);
    with_tile(L.n_in, L.n_out, [&](auto t) {
      gemm_kernel<true, decltype(t), Epi><<<grid, NT, 0, s>>>(P.B, L.n_in, L.n_out, r, P.N, L.W, L.n_in, epi);
    });
    return;
  }
  const size_t smem = sizeof(float) * L.cout * L.cin * L.kh * L.kw;
  if (conv_t_covers(L)) {
    const int geo = conv_geo(L), st = L.stride, G = L.cin == 3 ? 3 : 4;
    const ConvTile T0 = conv_t_tile(L, 0);
    const int bh = conv_band(L.h / st, st * st * (L.cin / G) * (L.w / st), P.B, sizeof(float) * T0.w_floats,
                             sizeof(float) * L.cout * T0.pitch, 1, T0.rows);
    if (bh > 0) {
      const ConvTile T = conv_t_tile(L, bh);
      const unsigned grid = (unsigned)P.B * T.bands;
      if (geo == 1) {
        if (G == 3)
          launch_blocked(conv_t_fast_kernel<4, 4, 2, 3, Epi>, grid, T.smem, s, L, T, r, P.N, epi);
        else
          launch_blocked(conv_t_fast_kernel<4, 4, 2, 4, Epi>, grid, T.smem, s, L, T, r, P.N, epi);
      } else {
        if (G == 3)
          launch_blocked(conv_t_fast_kernel<3, 3, 1, 3, Epi>, grid, T.smem, s, L, T, r, P.N, epi);
        else
          launch_blocked(conv_t_fast_kernel<3, 3, 1, 4, Epi>, grid, T.smem, s, L, T, r, P.N, epi);
      }
      return;
    }
  }
  const int plane = L.cin * L.h * L.w;
  dim3 grid((plane + NT - 1) / NT, P.B);
  conv_t_kernel<Epi><<<grid, NT, smem, s>>>(L, r, P.N, epi);
}

template <class Epi>
void forward(const LayerDev& L, const Problem& P, const float* x, Epi epi, cudaStream_t s) {
  count_launch();
  const float* xin = x + L.x_in_off;
  if (L.kind == LD_LAYER_FC) {
    const int tiles_n = (L.n_out + TN - 1) / TN, tiles_m = (P.B + TM - 1) / TM;
    int splits, kc;
    split_of(L, P, splits, kc);
    if (splits <= 1) {
      dim3 grid(tiles_n, tiles_m);
      with_tile(L.n_out, L.n_in, [&](auto t) {
        gemm_kernel<false, decltype(t), Epi><<<grid, NT, 0, s>>>(P.B, L.n_out, L.n_in, xin, P.XS, L.W, L.n_in, epi);
      });
    } else {
      dim3 grid(tiles_n, tiles_m, splits);
      with_tile(L.n_out, kc, [&](auto t) {
        gemm_splitk_kernel<decltype(t), Epi><<<grid, NT, 0, s>>>(P.B, L.n_out, L.n_in, kc, xin, P.XS, L.W, L.n_in,
                                                                 P.splitk_part, P.splitk_count, epi);
      });
    }
    return;
  }
  const size_t smem = std::max(sizeof(float) * L.cout * L.cin * L.kh * L.kw, Epi::kReduce ? kFinishSmem : 0);
  if (conv_f_covers(L)) {
    const int geo = conv_geo(L), st = L.stride, GF = L.cout % 4 == 0 ? 4 : 2;
    const ConvTile T0 = conv_f_tile(L, 0);
    const int bh = conv_band(L.ho, (L.cout / GF) * L.wo, P.B, sizeof(float) * T0.w_floats,
                             sizeof(float) * L.cin * T0.pitch, st, T0.rows);
    if (bh > 0) {
      ConvTile T = conv_f_tile(L, bh);
      if (Epi::kReduce) T.smem = std::max(T.smem, kFinishSmem);
      const unsigned grid = (unsigned)P.B * T.bands;
      if (geo == 1) {
        if (GF == 4)
          launch_blocked(conv_fwd_fast_kernel<4, 4, 2, 4, Epi>, grid, T.smem, s, L, T, xin, P.XS, epi);
        else
          launch_blocked(conv_fwd_fast_kernel<4, 4, 2, 2, Epi>, grid, T.smem, s, L, T, xin, P.XS, epi);
      } else {
        if (GF == 4)
          launch_blocked(conv_fwd_fast_kernel<3, 3, 1, 4, Epi>, grid, T.smem, s, L, T, xin, P.XS, epi);
        else
          launch_blocked(conv_fwd_fast_kernel<3, 3, 1, 2, Epi>, grid, T.smem, s, L, T, xin, P.XS, epi);
      }
      return;
    }
  }
  const int plane = L.cout * L.ho * L.wo;
  dim3 grid((plane + NT - 1) / NT, P.B);
  conv_fwd_kernel<Epi><<<grid, NT, smem, s>>>(L, xin, P.XS, epi);
}

}  // namespace

void launch_transposed_argmin(const LayerDev& L, const LayerDev*, const Problem& P, const float* rho,
                              EpiArgmin epi, cudaStream_t s) {
  transposed(L, P, rho, epi, s);
}

void launch_transposed_crown(const LayerDev& L, const Problem& P, const float* rho, EpiCrown epi,
                             cudaStream_t s) {
  transposed(L, P, rho, epi, s);
}

void launch_top_argmin(const LayerDev& Ln, const Problem& P, EpiArgmin epi, cudaStream_t s) {
  count_launch();
  top_kernel<EpiArgmin><<<grid1d((size_t)P.B * Ln.n_in), NT, 0, s>>>(P.B, Ln.n_in, Ln.W, epi);
}

void launch_top_crown(const LayerDev& Ln, const Problem& P, EpiCrown epi, cudaStream_t s) {
  count_launch();
  top_kernel<EpiCrown><<<grid1d((size_t)P.B * Ln.n_in), NT, 0, s>>>(P.B, Ln.n_in, Ln.W, epi);
}

void launch_forward_adam(const LayerDev& L, const Problem& P, const float* x, EpiAdam epi, cudaStream_t s) {
  forward(L, P, x, epi, s);
}

void launch_forward_record(const LayerDev& L, const Problem& P, const float* x, EpiRecord epi,
                           cudaStream_t s) {
  forward(L, P, x, epi, s);
}

void launch_forward_store(const LayerDev& L, const Problem& P, const float* x, EpiStore epi, cudaStream_t s) {
  forward(L, P, x, epi, s);
}

SplitK forward_split(const LayerDev& L, const Problem& P) {
  SplitK k{};
  split_of(L, P, k.splits, k.kc);
  return k;
}

bool launch_forward_partials(const LayerDev& L, const Problem& P, const float* x, SplitK& k, cudaStream_t s) {
  k = forward_split(L, P);
  if (!P.splitk_part || (size_t)k.splits * P.B * L.n_out > (size_t)P.splitk_part_cap) return false;
  count_launch();
  dim3 grid((L.n_out + TN - 1) / TN, (P.B + TM - 1) / TM, k.splits);
  with_tile(L.n_out, k.kc, [&](auto t) {
    gemm_partials_kernel<decltype(t)><<<grid, NT, 0, s>>>(P.B, L.n_out, L.n_in, k.kc, x + L.x_in_off, P.XS, L.W, L.n_in,
                                                          P.splitk_part);
  });
  return true;
}

void launch_transposed_scores(const LayerDev& L, const Problem& P, const float* mu, EpiScores epi, cudaStream_t s) {
  transposed(L, P, mu, epi, s);
}

void launch_top_scores(const LayerDev& Ln, const Problem& P, EpiScores epi, cudaStream_t s) {
  count_launch();
  top_kernel<EpiScores><<<grid1d((size_t)P.B * Ln.n_in), NT, 0, s>>>(P.B, Ln.n_in, Ln.W, epi);
}

void launch_forward_eval(const LayerDev& L, const Problem& P, const float* x, EpiEval epi, cudaStream_t s) {
  forward(L, P, x, epi, s);
}

void launch_transposed_dsg(const LayerDev& L, const Problem& P, const float* mu, EpiDsgT epi, cudaStream_t s) {
  transposed(L, P, mu, epi, s);
}

void launch_top_dsg(const LayerDev& Ln, const Problem& P, EpiDsgT epi, cudaStream_t s) {
  count_launch();
  top_kernel<EpiDsgT><<<grid1d((size_t)P.B * Ln.n_in), NT, 0, s>>>(P.B, Ln.n_in, Ln.W, epi);
}

void launch_empty_flags(const Problem& P, int8_t* empty, int* status, cudaStream_t s) {
  if (P.B > 0) {
    count_launch();
    empty_kernel<<<P.B, NT, 0, s>>>(P, empty, status);
  }
  count_launch();
  box_check_kernel<<<grid1d((size_t)P.n_props * (P.n0 > P.N ? P.n0 : P.N)), NT, 0, s>>>(P, status);
}

}  // namespace ld
