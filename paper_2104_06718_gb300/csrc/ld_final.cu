// Final bound in FP64 with outward slack: a sound lower bound q(rho_T).
//
// With rho_n = -1 and g_k = W_{k+1}^T rho_{k+1}, the dual of Eq.
// (nonprox_problem) decomposes over the subproblems (App. A, Eq.
// dual_decomp_vs_dj) into per-neuron minima plus bias terms:
//   q(rho) = sum_j min_{x0_j in [l0_j,u0_j]} (-g_0[j] x0_j)                    (P0)
//          + sum_{k=1}^{n-1} sum_i min_{vertices of P_k} (rho_k[i] xB - g_k[i] x) (Pk)
//          - sum_{k=1}^{n-1} rho_k^T b_k + b_n
// so the final bound needs only the transposed pass.  The FP64 pipe of GB300
// runs 2 operations per clock and SM against 128 FP32 ones, so g_k is summed in
// FP32 to more than FP64 precision: every product is an exact FP32 pair (FMA),
// and the pairs are summed on three levels.  Level 1 starts at 1.5 2^a with
// 2^(a-2) > sum |W||rho| (formed first, rounded up), so that its partial sums
// keep one exponent, every rounding error is exact and at most 2^(a-24)
// (Fast2Sum; the extraction sums of Rump, Ogita and Oishi's AccSum); those
// errors and the products' low parts of a block of k = 64 terms go to level 2,
// started at 1.5 2^b with 2^(b-1) >= (k + 1) 2^(a-24), whose errors, at most
// 2^(b-24) each, level 3 sums plainly; levels 2 and 3 are added in FP64 after
// each block.  So |g - exact| <= delta = (k + k^2) 2^(b-47) a block + 2^-52 |g|,
// at most 1.02 2^-48 sum|W||rho| a block (2^a <= 8 sum), where an FP64 sum has
// the bound gamma_k = 2^-47 sum|W||rho| for 64 terms.  15 FP32 operations a term take the place of
// one FP64 one (64 FP32 slots).  Geometries without a blocked path
// sum in FP64 (the products are exact there) with delta = gamma_K A_i,
// A_i >= sum |W||rho| in FP32 rounded up (Higham, gamma_K = K u / (1 - K u),
// u = 2^-53).  Every term's value t and an upper
// bound e on its error (from delta_i and the rounding of one subtraction and
// one product) are summed per subdomain; the bound returned is
//   S - E - gamma_M * sum|t|   (S = sum t, E = sum e, M = number of terms),
// with t and S in FP64, and E and sum|t| summed rounding upward (per thread and
// warp in FP32) and scaled by 1 + 2 gamma_M as a margin.  A CTA in which a sum
// |W||rho| is below 2^-59 (and not 0) or from 2^117 on, or a sum of errors or |t|
// from 2^100 on, which FP32 does not hold, forms its terms again in FP64.  That
// is one test a CTA and code behind the usual path: FP64 calls within it took the
// conv kernels from 64 to 120 registers (2000 Base subdomains, duals given: 1054 us
// then, 1003 so).  Partial sums go to fixed slots that one kernel adds in a fixed
// order, so the bound does not depend on the order in which blocks run.
#include <cmath>

#include "ld_conv.cuh"

namespace ld {
namespace {

constexpr int BN = 64, NT = 256;
constexpr float kU52 = 2.220446049250313e-16f;  // 2^-52

// Sums of a thread's terms: values, error bounds (up), |values| (up).
struct TermSum {
  double t = 0.0;
  float e = 0.f, a = 0.f;
};
struct WideSum {
  double t = 0.0, e = 0.0, a = 0.0;
};

// |x| rounded up to FP32, by integer instructions (at least 2^-126).
__device__ __forceinline__ float abs_up(double x) {
  const unsigned hi = (unsigned)__double2hiint(x) & 0x7fffffffu, lo = (unsigned)__double2loint(x);
  if (hi < 0x38100000u) return hi | lo ? 1.1754943508222875e-38f : 0.f;
  if (hi >= 0x47e00000u) return x != x ? (float)x : INFINITY;  // beyond FLT_MAX's binade, inf, NaN
  return __uint_as_float(((hi - 0x38000000u) << 3 | lo >> 29) + 1u);
}

constexpr float kHuge = 1.2676506002282294e30f;  // 2^100: FP32 sums of errors and sizes end here
__device__ __forceinline__ bool beyond(const TermSum& s) { return !(s.e < kHuge && s.a < kHuge); }

// Adds t, the minimum of exact values and of the product tx = c x, c within
// delta of its exact value: e = |x| (delta + 2^-52 |c|) + 2^-52 |tx| (none where
// c is exactly 0, also beside an infinite x).
__device__ __forceinline__ void add_term(TermSum& s, double t, double tx, double c, float x, float delta) {
  s.t += t;
  s.e = __fadd_ru(s.e, __fmaf_ru(x, __fmaf_ru(kU52, abs_up(c), delta), __fmul_ru(kU52, abs_up(tx))));
  s.a = __fadd_ru(s.a, abs_up(t));
}
__device__ __forceinline__ void add_term(WideSum& s, double t, double tx, double c, float x, double delta) {
  const double ec = __dadd_ru(delta, __dmul_ru((double)kU52, fabs(c)));
  s.t += t;
  if (ec != 0.0) s.e = __dadd_ru(s.e, __dadd_ru(__dmul_ru((double)x, ec), __dmul_ru((double)kU52, fabs(tx))));
  s.a = __dadd_ru(s.a, fabs(t));
}
// A term without an error.
__device__ __forceinline__ void add_exact(TermSum& s, double t) {
  s.t += t;
  s.a = __fadd_ru(s.a, abs_up(t));
}
__device__ __forceinline__ void add_exact(WideSum& s, double t) {
  s.t += t;
  s.a = __dadd_ru(s.a, fabs(t));
}

__device__ __forceinline__ float add_up(float a, float b) { return __fadd_ru(a, b); }
__device__ __forceinline__ double add_up(double a, double b) { return __dadd_ru(a, b); }
// Sums over the lanes of each group of 2 * top lanes (all 32 lanes take part);
// up: t rounded upward too.
template <class S>
__device__ __forceinline__ void reduce_terms(S& s, int top, int up) {
  for (int off = top; off > 0; off >>= 1) {
    const double t = __shfl_xor_sync(0xffffffffu, s.t, off);
    s.t = up ? __dadd_ru(s.t, t) : s.t + t;
    s.e = add_up(s.e, __shfl_xor_sync(0xffffffffu, s.e, off));
    s.a = add_up(s.a, __shfl_xor_sync(0xffffffffu, s.a, off));
  }
}

// One per-neuron minimum, g within delta of the exact value.  box: P0 term
// with coefficient -g on [l, u]; otherwise the Pk neuron with rho r.
template <class S, class D>
__device__ __forceinline__ void final_term(S& s, bool box, float r, double g, D delta, float l, float u) {
  if (!box && u <= 0.f) {             // blocking: min r*xB over [l,u], exact products (r = 0: 0, also with l = -inf)
    add_exact(s, widen(r) * widen(r > 0.f ? l : u));
    return;
  }
  const double d = box ? -g : widen(r) - g;  // coefficient of xB (and of x) in the box/passing/(u,u) cases
  if (box || l >= 0.f) {              // P0 box, or passing: min d*xB over [l,u]
    // within delta of d the other end may be the minimum: either product is then within |d|_up max|x| of 0
    const double t = d * widen(d >= 0.0 ? l : u);
    add_term(s, t, t, d, fmaxf(fabsf(l), fabsf(u)), delta);
    return;
  }
  // ambiguous: vertices (l,0) -> r*l (exact), (0,0) -> 0, (u,u) -> d*u
  const double tuu = d * widen(u);
  add_term(s, fmin(fmin(widen(r) * widen(l), 0.0), tuu), tuu, d, fabsf(u), delta);
}

struct FinalEpi {
  Problem P;
  int layer;           // k (0 = box)
  int r_off;
  const float* rho;
  double gamma_K;
  int ball_norm;       // layer 0, l2 ball: the term is an upper bound on g_0[i]^2 (for ||g_0||)
  // delta: bound on |g - exact g|
  template <class S, class D>
  __device__ __forceinline__ void term(int b, int i, double g, D delta, S& s) const {
    if (layer == 0) {
      if (ball_norm) {
        // |exact g_0[i]| <= |g| + delta: its square, summed rounding up (in the
        // values: it is the square of the norm itself, not a slack)
        const double a = __dadd_ru(fabs(g), (double)delta);
        s.t = __dadd_ru(s.t, __dmul_ru(a, a));
        return;
      }
      // the box; over an l2 ball l0 = u0 = the centre, which gives the
      // -g_0^T c part of the ball's minimum (the -eps ||g_0|| part is added
      // by the ball pass)
      const int p = prop_of(P, b);
      final_term(s, true, 0.f, g, delta, P.l0[(size_t)p * P.n0 + i], P.u0[(size_t)p * P.n0 + i]);
      return;
    }
    const int j = r_off + i;
    float l, u;
    clamped_bounds(P, b, j, l, u);
    final_term(s, false, rho[(size_t)b * P.N + j], g, delta, l, u);
  }
};

// g of input element (c, yy, xx) of a conv in FP64 (exact products), and the FP32
// sum of their sizes (up); W in its [o][c][i][j] layout, rb one subdomain's duals.
__device__ __forceinline__ double conv_sum64(const LayerDev& L, const float* W, const float* rb, int c, int yy, int xx,
                                             float& abs_sum) {
  const int hw_o = L.ho * L.wo;
  double acc = 0.0;
  float aab = 0.f;
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
      const float* wp = W + ((size_t)c * L.kh + i) * L.kw + j;
      const float* rp = rb + y * L.wo + xo;
      for (int o = 0; o < L.cout; ++o) {
        const float wv = wp[(size_t)o * L.cin * L.kh * L.kw], rv = rp[(size_t)o * hw_o];
        acc = fma((double)wv, (double)rv, acc);
        aab = __fmaf_ru(fabsf(wv), fabsf(rv), aab);
      }
    }
  }
  abs_sum = aab;
  return acc;
}

// ---------------------------------------------------------------- three-level sums
// b - a by one packed instruction (the product with -1 is exact).
__device__ __forceinline__ float2 sub2(float2 b, float2 a) { return __ffma2_rn(a, make_float2(-1.f, -1.f), b); }

// Two sums (packed) of products: start(), size(w, r) for every term, then
// begin(K) and add(w, r) for every term again.
constexpr int kBlk = 64;  // terms between two blocks
struct Sum3x2 {
  float2 p, q, c;      // levels 1 to 3; p holds the sum of sizes until begin()
  double g0, g1;       // finished blocks
  int zero;            // bit h: half h's products are all 0 (or below 2^-150)
  __device__ __forceinline__ void start() { p = make_float2(0.f, 0.f); }
  __device__ __forceinline__ void size(float2 w, float2 r) {
    const float2 h = __fmul2_rn(w, r);
    p = make_float2(__fadd_ru(p.x, fabsf(h.x)), __fadd_ru(p.y, fabsf(h.y)));
  }
  // 2^a from the sum of |rounded products|: 2^(a-1) is more than twice the sum,
  // which leaves room for the products' rounding and the level's own errors;
  // sums below 2^-60 take that a (see result)
  static __device__ __forceinline__ float top(float s) {
    const unsigned e = __float_as_uint(fmaxf(s, 8.673617379884035e-19f)) & 0x7f800000u;
    return __uint_as_float(e) * 8.f;
  }
  static __device__ __forceinline__ float binade(float p) { return __uint_as_float(__float_as_uint(p) & 0x7f800000u); }
  __device__ __forceinline__ void begin(float lvl2) {
    zero = (p.x == 0.f ? 1 : 0) | (p.y == 0.f ? 2 : 0);
    p = make_float2(1.5f * top(p.x), 1.5f * top(p.y));
    q = make_float2(p.x * lvl2, p.y * lvl2);
    c = make_float2(0.f, 0.f);
    g0 = g1 = 0.0;
  }
  // Levels 2 and 3 of a finished block (at most kBlk terms) into FP64; 2^a is
  // recovered from p, which lies in [2^a, 2^(a+1)).
  __device__ __forceinline__ void block(float lvl2) {
    const float2 z = make_float2(1.5f * binade(p.x) * lvl2, 1.5f * binade(p.y) * lvl2);
    g0 += widen(q.x - z.x) + widen(c.x);
    g1 += widen(q.y - z.y) + widen(c.y);
    q = z;
    c = make_float2(0.f, 0.f);
  }
  __device__ __forceinline__ void add(float2 w, float2 r, float2 nr) {
    const float2 nh = __fmul2_rn(w, nr);
    const float2 e = __ffma2_rn(w, r, nh);           // w r = -nh + e exactly
    const float2 t = sub2(p, nh);
    const float2 n1 = __fadd2_rn(nh, sub2(t, p));    // minus the error of t
    p = t;
    const float2 t2 = sub2(q, n1);
    const float2 n2 = __fadd2_rn(n1, sub2(t2, q));   // minus the error of t2
    const float2 t3 = __fadd2_rn(t2, e);
    const float2 e3 = sub2(e, sub2(t3, t2));         // the error of t3
    q = t3;
    c = __fadd2_rn(c, sub2(e3, n2));
  }
  // Value and bound of half h of K products after the last block.  False for
  // sums of sizes below 2^-59 (the bound would be an absolute one, and a product's
  // low part could underflow) but not 0, from 2^117 on, and NaN.
  __device__ __forceinline__ bool result(int h, float kk, int K, double& g, float& delta) const {
    const float ph = h ? p.y : p.x, two_a = binade(ph);
    g = widen(ph - 1.5f * two_a) + (h ? g1 : g0);
    delta = __fmaf_ru(kk, two_a, __fmul_ru(kU52, abs_up(g)));
    if (zero >> h & 1) {
      g = 0.0;
      delta = (float)K * 1.401298464324817e-45f;
      return true;
    }
    return two_a > 6.938893903907228e-18f && two_a < 1.329227995784916e36f;  // 2^-57, 2^120
  }
};
// 2^(b-a) of level 2, 2^(b-1) >= (k + 1) 2^(a-24) for blocks of at most k =
// min(kBlk, K) terms, and blocks times (k + k^2) 2^(b-47-a).
struct Sum3Const {
  float lvl2, kk;
};
inline Sum3Const sum3_const(int blocks, int K) {
  const int k = std::min(kBlk, K);
  int cl = 0;
  while ((1 << cl) < k + 1) ++cl;
  Sum3Const s;
  s.lvl2 = (float)std::ldexp(1.0, cl - 23);
  s.kk = (float)(blocks * std::ldexp((double)k + (double)k * k, cl - 23 - 47) * (1.0 + 1e-6));
  return s;
}
// Blocks of a conv sum: `taps` runs of cout terms (in pieces of kBlk), a new
// block wherever the next run or piece would not fit (as final_conv_fast_kernel).
inline int sum3_blocks(int taps, int cout) {
  int blocks = 1, cnt = 0;
  for (int t = 0; t < taps; ++t)
    for (int o = 0; o < cout; o += kBlk) {
      const int n = std::min(kBlk, cout - o);
      if (cnt + n > kBlk) {
        ++blocks;
        cnt = 0;
      }
      cnt += n;
    }
  return blocks;
}

// Each (subdomain, slot) partial is written exactly once and the slots are
// summed in a fixed order by the combine kernel: the final bound does not
// depend on the order in which blocks run.
__device__ __forceinline__ void acc_add(FinalAcc a, int slot, int b, double t, double e, double at) {
  double* p = a.slots + ((size_t)b * a.n_slots + slot) * 3;
  p[0] = t;
  p[1] = e;
  p[2] = at;
}

// Transposed FC pass (A = rho_{k+1} [B, n_out], W [n_out, n_in]) in three-level
// sums.  Tile: BM = 16 TM subdomains x BN = 64 columns (TM = 4, or 1 when the
// 64-row grid would leave SMs idle; the column blocks, and so the partial-sum
// slots, are the same either way), a thread TM x 4 of it; up to KS rows of K
// staged at once.
constexpr int KS = 128;  // a multiple of kBlk: blocks end where rounds do
// The CTA's outputs in FP64, an output a thread at a time.
template <int TM>
__device__ __noinline__ void fc_wide(int M, int Ncol, int K, const float* A, int lda, const float* W, int ldw,
                                     const FinalEpi& epi, const FinalAcc& acc_out) {
  const int tx = threadIdx.x % 16, ty = threadIdx.x / 16;
  for (int i = 0; i < TM; ++i) {
    const int m = blockIdx.y * 16 * TM + ty + 16 * i;
    WideSum s;
    for (int j = 0; j < 4; ++j) {
      const int n = blockIdx.x * BN + 4 * tx + j;
      if (m >= M || n >= Ncol) continue;
      double g = 0.0;
      float as = 0.f;
#pragma unroll 4
      for (int k = 0; k < K; ++k) {
        const float wv = W[(size_t)k * ldw + n], rv = A[(size_t)m * lda + k];
        g = fma((double)wv, (double)rv, g);
        as = __fmaf_ru(fabsf(wv), fabsf(rv), as);
      }
      epi.term(m, n, g, __dmul_ru(epi.gamma_K, (double)as), s);
    }
    reduce_terms(s, 8, epi.ball_norm);
    if (tx == 0 && m < M) acc_add(acc_out, acc_out.slot + blockIdx.x, m, s.t, s.e, s.a);
  }
}
template <int TM>
__global__ void __launch_bounds__(NT) final_fc_kernel(int M, int Ncol, int K, const float* __restrict__ A, int lda,
                                                      const float* __restrict__ W, int ldw, const __grid_constant__ FinalEpi epi,
                                                      Sum3Const sc, const __grid_constant__ FinalAcc acc_out) {
  constexpr int BMt = 16 * TM;
  extern __shared__ __align__(16) float sm[];
  float* As = sm;                      // [k][BMt + 1]
  float* Bs = As + KS * (BMt + 1) + (4 - (KS * (BMt + 1)) % 4) % 4;  // [k][BN]
  const int t = threadIdx.x, tx = t % 16, ty = t / 16;
  const int m0 = blockIdx.y * BMt, n0 = blockIdx.x * BN;
  Sum3x2 acc[TM][2];
#pragma unroll
  for (int i = 0; i < TM; ++i) {
    acc[i][0].start();
    acc[i][1].start();
  }
#pragma unroll 1
  for (int pass = 0; pass < 2; ++pass) {
    for (int k0 = 0; k0 < K; k0 += KS) {
      const int kn = min(KS, K - k0);
      if (pass == 0 || K > KS) {
        __syncthreads();
        for (int idx = t; idx < BMt * kn; idx += NT) {
          const int mm = idx / kn, kk = idx - mm * kn;
          As[kk * (BMt + 1) + mm] = m0 + mm < M ? __ldg(A + (size_t)(m0 + mm) * lda + k0 + kk) : 0.f;
        }
        for (int idx = t; idx < BN * kn; idx += NT) {
          const int kk = idx / BN, nn = idx % BN;
          Bs[kk * BN + nn] = n0 + nn < Ncol ? __ldg(W + (size_t)(k0 + kk) * ldw + n0 + nn) : 0.f;
        }
        __syncthreads();
      }
      if (pass == 0) {
#pragma unroll 4
        for (int kk = 0; kk < kn; ++kk) {
          const float4 w = *reinterpret_cast<const float4*>(Bs + kk * BN + 4 * tx);
#pragma unroll
          for (int i = 0; i < TM; ++i) {
            const float a = As[kk * (BMt + 1) + ty + 16 * i];
            acc[i][0].size(make_float2(w.x, w.y), make_float2(a, a));
            acc[i][1].size(make_float2(w.z, w.w), make_float2(a, a));
          }
        }
        continue;
      }
      for (int kb = 0; kb < kn; kb += kBlk) {
#pragma unroll 2
        for (int kk = kb; kk < min(kn, kb + kBlk); ++kk) {
          const float4 w = *reinterpret_cast<const float4*>(Bs + kk * BN + 4 * tx);
#pragma unroll
          for (int i = 0; i < TM; ++i) {
            const float a = As[kk * (BMt + 1) + ty + 16 * i];
            acc[i][0].add(make_float2(w.x, w.y), make_float2(a, a), make_float2(-a, -a));
            acc[i][1].add(make_float2(w.z, w.w), make_float2(a, a), make_float2(-a, -a));
          }
        }
#pragma unroll
        for (int i = 0; i < TM; ++i) {
          acc[i][0].block(sc.lvl2);
          acc[i][1].block(sc.lvl2);
        }
      }
    }
    if (pass == 0)
#pragma unroll
      for (int i = 0; i < TM; ++i) {
        acc[i][0].begin(sc.lvl2);
        acc[i][1].begin(sc.lvl2);
      }
  }
  TermSum sum[TM];
  bool bad = false;
#pragma unroll
  for (int i = 0; i < TM; ++i) {
    const int m = m0 + ty + 16 * i;
    if (m >= M) continue;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const int n = n0 + 4 * tx + j;
      if (n >= Ncol) continue;
      double g;
      float delta;
      bad |= !acc[i][j / 2].result(j % 2, sc.kk, K, g, delta);
      epi.term(m, n, g, delta, sum[i]);
    }
    bad |= beyond(sum[i]);
  }
  if (__syncthreads_or(bad)) {
    fc_wide<TM>(M, Ncol, K, A, lda, W, ldw, epi, acc_out);
    return;
  }
#pragma unroll
  for (int i = 0; i < TM; ++i) {
    const int m = m0 + ty + 16 * i;
    reduce_terms(sum[i], 8, epi.ball_norm);
    if (tx == 0 && m < M) acc_add(acc_out, acc_out.slot + blockIdx.x, m, sum[i].t, (double)sum[i].e, (double)sum[i].a);
  }
}

template <class S>
__device__ __forceinline__ void block_reduce_add(FinalAcc a, int slot, int b, S s, int up) {
  __shared__ double red[3][NT / 32];
  reduce_terms(s, 16, up);
  const int w = threadIdx.x / 32, lane = threadIdx.x % 32;
  if (lane == 0) {
    red[0][w] = s.t;
    red[1][w] = (double)s.e;
    red[2][w] = (double)s.a;
  }
  __syncthreads();
  if (threadIdx.x < 3) {  // a thread each for t, e and a
    double v = red[threadIdx.x][0];
    for (int i = 1; i < (int)(blockDim.x / 32); ++i) {
      const double x = red[threadIdx.x][i];
      v = threadIdx.x == 0 && !up ? v + x : __dadd_ru(v, x);
    }
    a.slots[((size_t)b * a.n_slots + slot) * 3 + threadIdx.x] = v;
  }
}

// The elements of CTA blockIdx.x of a conv pass, as WideSum terms: `per` elements
// per item (channels of one position, phase by phase for per > 1).
__device__ __noinline__ WideSum conv_wide(const LayerDev& L, const float* rb, const FinalEpi& epi, int b, int per) {
  WideSum s;
  const int hw = L.h * L.w, ST = per > 1 ? L.stride : 1;
  const int qh = L.h / ST, qw = L.w / ST, ncg = L.cin / per, items = ST * ST * ncg * qh * qw;
  for (int e = blockIdx.x * NT + threadIdx.x; e < items; e += gridDim.x * NT) {
    int q = e;
    const int qx = q % qw;
    q /= qw;
    const int qy = q % qh;
    q /= qh;
    const int cg = q % ncg;
    q /= ncg;
    const int yy = q / ST + ST * qy, xx = q % ST + ST * qx;
    for (int g = 0; g < per; ++g) {
      const int c = cg * per + g;
      float as;
      const double v = conv_sum64(L, L.W, rb, c, yy, xx, as);
      epi.term(b, c * hw + yy * L.w + xx, v, __dmul_ru(epi.gamma_K, (double)as), s);
    }
  }
  return s;
}

// FP64 transposed conv pass; grid row = subdomain.
__global__ void __launch_bounds__(NT) final_conv_kernel(const __grid_constant__ LayerDev L, const float* __restrict__ r,
                                                        int rs, const __grid_constant__ FinalEpi epi, FinalAcc acc_out) {
  extern __shared__ float sW[];
  const int nw = L.cout * L.cin * L.kh * L.kw;
  for (int e = threadIdx.x; e < nw; e += blockDim.x) sW[e] = L.W[e];
  __syncthreads();
  const int b = blockIdx.y;
  const float* rb = r + (size_t)b * rs;
  const int hw_i = L.h * L.w, plane = L.cin * hw_i;
  const float gamma_K = __double2float_ru(epi.gamma_K);
  TermSum s;
  bool bad = false;
  for (int e = blockIdx.x * blockDim.x + threadIdx.x; e < plane; e += gridDim.x * blockDim.x) {
    const int c = e / hw_i, rem = e % hw_i, yy = rem / L.w, xx = rem % L.w;
    float as;
    const double g = conv_sum64(L, sW, rb, c, yy, xx, as);
    bad |= as < 1e-18f && as != 0.f;  // delta too small for FP32
    epi.term(b, e, g, __fmul_ru(gamma_K, as), s);
  }
  if (__syncthreads_or(bad || beyond(s)))
    block_reduce_add(acc_out, acc_out.slot + blockIdx.x, b, conv_wide(L, rb, epi, b, 1), epi.ball_norm);
  else
    block_reduce_add(acc_out, acc_out.slot + blockIdx.x, b, s, epi.ball_norm);
}

// Transposed conv by stride phase (k4 s2 / k3 s1) in three-level sums, G input
// channels per thread (two packed pairs; G = 3: the fourth has zero weights):
// g[b, c, yy, xx] = sum over the phase's taps (i, j) and o of W[o, c, i, j]
// rho[b, o, y, x], weights and the subdomain's rho_{k+1} (with its zero halo) in
// shared memory.  The slots are this grid's blocks.
template <int KH, int KW, int ST, int G>
__global__ void __launch_bounds__(NT, 4) final_conv_fast_kernel(const __grid_constant__ LayerDev L, ConvTile T,
                                                             const float* __restrict__ r, int rs,
                                                             const __grid_constant__ FinalEpi epi, Sum3Const sc,
                                                             FinalAcc acc_out) {
  extern __shared__ __align__(16) float sm[];
  float* sR = sm + T.w_floats;
  const int b = blockIdx.y;
  if (G == 3)
    for (int e = threadIdx.x; e < T.w_floats / 4; e += NT) sm[4 * e + 3] = 0.f;
  conv_t_weights(L, T, sm, NT);
  conv_t_rows(L, T, sR, r + (size_t)b * rs, 0, NT);
  stage_wait();
  const int qh = L.h / ST, qw = L.w / ST, ncg = L.cin / G, plane = T.rows * T.pitch;
  const int items = ST * ST * ncg * qh * qw;
  const int K = L.cout * (KH / ST) * (KW / ST);
  TermSum s;
  bool bad = false;
  for (int e = blockIdx.x * NT + threadIdx.x; e < items; e += gridDim.x * NT) {
    int q = e;
    const int qx = q % qw;
    q /= qw;
    const int qy = q % qh;
    q /= qh;
    const int cg = q % ncg;
    q /= ncg;
    const int rx = q % ST;
    const int ry = q / ST;
    const int i0 = (ry + L.pad) % ST, j0 = (rx + L.pad) % ST;
    const int dy0 = (ry + L.pad - i0) / ST, dx0 = (rx + L.pad - j0) / ST;
    const float* rp = sR + (qy + dy0 - T.y_off) * T.pitch + qx + dx0 - T.x_off;
    const float* wp = sm + (i0 * KW + j0) * T.wc + cg * G;
    Sum3x2 a0, a1;
    a0.start();
    a1.start();
#pragma unroll
    for (int a = 0; a < KH / ST; ++a)
#pragma unroll
      for (int bb = 0; bb < KW / ST; ++bb) {
        const float* ra = rp - a * T.pitch - bb;
        const float* wa = wp + (ST * a * KW + ST * bb) * T.wc;
#pragma unroll 4
        for (int o = 0; o < L.cout; ++o) {
          const float rv = ra[o * plane];
          const float4 w = *reinterpret_cast<const float4*>(wa + o * KH * KW * T.wc);
          a0.size(make_float2(w.x, w.y), make_float2(rv, rv));
          a1.size(make_float2(w.z, w.w), make_float2(rv, rv));
        }
      }
    a0.begin(sc.lvl2);
    a1.begin(sc.lvl2);
    int cnt = 0;
#pragma unroll 1
    for (int a = 0; a < KH / ST; ++a)
#pragma unroll 1
      for (int bb = 0; bb < KW / ST; ++bb) {
        const float* ra = rp - a * T.pitch - bb;
        const float* wa = wp + (ST * a * KW + ST * bb) * T.wc;
        for (int o0 = 0; o0 < L.cout; o0 += kBlk) {
          const int on = min(L.cout, o0 + kBlk);
          if (cnt + on - o0 > kBlk) {
            a0.block(sc.lvl2);
            a1.block(sc.lvl2);
            cnt = 0;
          }
          cnt += on - o0;
#pragma unroll 4
          for (int o = o0; o < on; ++o) {
            const float rv = ra[o * plane];
            const float4 w = *reinterpret_cast<const float4*>(wa + o * KH * KW * T.wc);
            a0.add(make_float2(w.x, w.y), make_float2(rv, rv), make_float2(-rv, -rv));
            a1.add(make_float2(w.z, w.w), make_float2(rv, rv), make_float2(-rv, -rv));
          }
        }
      }
    a0.block(sc.lvl2);
    a1.block(sc.lvl2);
    const int yy = ry + ST * qy, xx = rx + ST * qx;
#pragma unroll
    for (int g = 0; g < G; ++g) {
      double gv;
      float delta;
      const int c = cg * G + g, i = (c * L.h + yy) * L.w + xx;
      bad |= !(g / 2 ? a1 : a0).result(g % 2, sc.kk, K, gv, delta);
      epi.term(b, i, gv, delta, s);
    }
  }
  if (__syncthreads_or(bad || beyond(s)))
    block_reduce_add(acc_out, acc_out.slot + blockIdx.x, b, conv_wide(L, r + (size_t)b * rs, epi, b, G), epi.ball_norm);
  else
    block_reduce_add(acc_out, acc_out.slot + blockIdx.x, b, s, epi.ball_norm);
}

// Geometry and channel blocking of the phase-split transposed conv, or 0.
constexpr size_t kFinalSmem = 160 * 1024;
int final_fast_geo(const LayerDev& L, int& G) {
  G = 0;
  if (!conv_t_covers(L) || conv_t_tile(L, L.h / L.stride).smem > kFinalSmem) return 0;
  G = L.cin == 3 ? 3 : 4;
  return conv_geo(L);
}

int final_fast_blocks(const LayerDev& L, int G) {
  const int items = L.stride * L.stride * (L.cin / G) * (L.h / L.stride) * (L.w / L.stride);
  return (items + NT - 1) / NT;
}

// Top subproblem P_{n-1}: g_{n-1} = -W_n, no product formed.  W_n is the
// margin-folded row summed in FP64 (Wn64) when the net has one, with Wn_err
// bounding the distance of each entry from the exact fold (the error of g
// enters the term's error bound like a summation error); else the FP32 row,
// exact.
__global__ void __launch_bounds__(NT) final_top_kernel(int n, const float* __restrict__ Wn,
                                                       const double* __restrict__ Wn64,
                                                       const double* __restrict__ Wn_err, FinalEpi epi,
                                                       FinalAcc acc_out) {
  const int b = blockIdx.x;
  WideSum s;
  for (int i = threadIdx.x; i < n; i += blockDim.x) {
    if (Wn64)
      epi.term(b, i, -Wn64[i], Wn_err[i], s);
    else
      epi.term(b, i, -widen(Wn[i]), 0.0, s);
  }
  block_reduce_add(acc_out, acc_out.slot, b, s, epi.ball_norm);
}

struct BiasLayers {
  int count;
  int r_off[kMaxLayers];
  int n[kMaxLayers];
  int plane[kMaxLayers];
  const float* bias[kMaxLayers];
};

// Bias terms -rho_k^T b_k, k = 1..n-1 (exact FP64 products).
__global__ void __launch_bounds__(NT) final_bias_kernel(Problem P, BiasLayers BL, const float* __restrict__ rho,
                                                        FinalAcc acc_out) {
  const int b = blockIdx.x;
  const auto terms = [&](auto& s) {
    for (int k = 0; k < BL.count; ++k)
#pragma unroll 4
      for (int i = threadIdx.x; i < BL.n[k]; i += blockDim.x)
        add_exact(s, -widen(rho[(size_t)b * P.N + BL.r_off[k] + i]) * widen(__ldg(BL.bias[k] + i / BL.plane[k])));
  };
  TermSum s;
  terms(s);
  if (__syncthreads_or(beyond(s))) {
    WideSum w;
    terms(w);
    block_reduce_add(acc_out, acc_out.slot, b, w, 0);
    return;
  }
  block_reduce_add(acc_out, acc_out.slot, b, s, 0);
}

// One warp per subdomain: lane i loads slot i of a round, the slots are added in order.
__global__ void final_combine_kernel(Problem P, FinalAcc a, double bn, double bn_err, double gamma_M, double inflate,
                                     double* out) {
  const int lane = threadIdx.x & 31, b = blockIdx.x * (blockDim.x / 32) + threadIdx.x / 32;
  if (b >= P.B) return;
  double S = bn, E = bn_err, A = fabs(bn);
  const double* p = a.slots + (size_t)b * a.n_slots * 3;
  for (int i0 = 0; i0 < a.n_slots; i0 += 32) {
    const bool in = i0 + lane < a.n_slots;
    const double t = in ? p[3 * (i0 + lane)] : 0.0, e = in ? p[3 * (i0 + lane) + 1] : 0.0,
                 at = in ? p[3 * (i0 + lane) + 2] : 0.0;
    const int n = min(32, a.n_slots - i0);
    for (int i = 0; i < n; ++i) {
      S += __shfl_sync(0xffffffffu, t, i);
      E = __dadd_ru(E, __shfl_sync(0xffffffffu, e, i));
      A = __dadd_ru(A, __shfl_sync(0xffffffffu, at, i));
    }
  }
  if (lane == 0) {
    E = __dmul_ru(E, inflate);
    A = __dmul_ru(A, inflate);
    out[b] = P.empty[b] ? __longlong_as_double(0x7ff0000000000000LL)  // +inf: empty subdomain
                        : __dsub_rd(__dsub_rd(S, E), __dmul_ru(gamma_M, A));
  }
}

__global__ void record_finish_kernel(Problem P, const double* q, const double* rest, double* out) {
  for (int b = blockIdx.x * blockDim.x + threadIdx.x; b < P.B; b += gridDim.x * blockDim.x)
    out[b] = P.empty[b] ? __longlong_as_double(0x7ff0000000000000LL) : (rest ? q[b] + rest[b] : q[b]);
}

}  // namespace

static double gamma_of(double K) {
  const double u = 1.1102230246251565e-16;  // 2^-53
  return (K * u) / (1.0 - K * u) * (1.0 + 1e-12);
}

template <int KH, int KW, int ST, int G>
void launch_fast(dim3 grid, const LayerDev& L, const float* r, int rs, FinalEpi epi, FinalAcc acc, cudaStream_t s) {
  const ConvTile T = conv_t_tile(L, L.h / ST);
  if (T.smem > 40 * 1024)
    cudaFuncSetAttribute(final_conv_fast_kernel<KH, KW, ST, G>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                         (int)kFinalSmem);
  final_conv_fast_kernel<KH, KW, ST, G><<<grid, NT, T.smem, s>>>(L, T, r, rs, epi, sum3_const(sum3_blocks((KH / ST) * (KW / ST), L.cout), L.fan_t), acc);
}

template <int TM>
void launch_fc(const LayerDev& L, const Problem& P, const float* r, const FinalEpi& epi, FinalAcc acc, cudaStream_t s) {
  constexpr int BMt = 16 * TM;
  constexpr size_t smem = sizeof(float) * (KS * (BMt + 1) + 4 + KS * BN);
  if (smem > 40 * 1024)
    cudaFuncSetAttribute(final_fc_kernel<TM>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  dim3 grid((L.n_in + BN - 1) / BN, (P.B + BMt - 1) / BMt);
  final_fc_kernel<TM><<<grid, NT, smem, s>>>(P.B, L.n_in, L.n_out, r, P.N, L.W, L.n_in, epi,
                                             sum3_const((L.n_out + kBlk - 1) / kBlk, L.n_out), acc);
}

int sm_count() {
  static int n = 0;
  if (!n) {
    int dev = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev);
    if (n <= 0) n = 1;
  }
  return n;
}

void launch_final_layer(const LayerDev& Lnext, int layer, int r_off, int x_off, const Problem& P,
                        const float* rho, int top, FinalAcc acc, cudaStream_t s, int ball_norm) {
  (void)x_off;
  FinalEpi epi{P, layer, r_off, rho, gamma_of((double)Lnext.fan_t), ball_norm};
  if (P.B == 0) return;
  count_launch();
  if (top) {
    final_top_kernel<<<P.B, NT, 0, s>>>(Lnext.n_in, Lnext.W, Lnext.W64, Lnext.W64_err, epi, acc);
    return;
  }
  const float* r = rho + Lnext.r_out_off;
  if (Lnext.kind == LD_LAYER_FC) {
    const int nb = (Lnext.n_in + BN - 1) / BN;
    if (nb * ((P.B + 63) / 64) >= 2 * sm_count())
      launch_fc<4>(Lnext, P, r, epi, acc, s);
    else
      launch_fc<1>(Lnext, P, r, epi, acc, s);
  } else {
    int G = 0;
    const int geo = final_fast_geo(Lnext, G);
    if (geo) {
      dim3 grid(final_fast_blocks(Lnext, G), P.B);
      if (geo == 1) {
        if (G == 4) launch_fast<4, 4, 2, 4>(grid, Lnext, r, P.N, epi, acc, s);
        else launch_fast<4, 4, 2, 3>(grid, Lnext, r, P.N, epi, acc, s);
      } else {
        if (G == 4) launch_fast<3, 3, 1, 4>(grid, Lnext, r, P.N, epi, acc, s);
        else launch_fast<3, 3, 1, 3>(grid, Lnext, r, P.N, epi, acc, s);
      }
      return;
    }
    const int plane = Lnext.cin * Lnext.h * Lnext.w;
    dim3 grid((plane + NT - 1) / NT, P.B);
    const size_t smem = sizeof(float) * Lnext.cout * Lnext.cin * Lnext.kh * Lnext.kw;
    final_conv_kernel<<<grid, NT, smem, s>>>(Lnext, r, P.N, epi, acc);
  }
}

void launch_final_bias(const std::vector<LayerDev>& Ls, const Problem& P, const float* rho, FinalAcc acc,
                       cudaStream_t s) {
  if (P.B == 0) return;
  BiasLayers BL{};
  BL.count = (int)Ls.size() - 1;
  for (int k = 0; k < BL.count; ++k) {
    const LayerDev& L = Ls[k];
    BL.r_off[k] = L.r_out_off;
    BL.n[k] = L.n_out;
    BL.plane[k] = L.kind == LD_LAYER_FC ? 1 : L.ho * L.wo;
    BL.bias[k] = L.b;
  }
  count_launch();
  final_bias_kernel<<<P.B, NT, 0, s>>>(P, BL, rho, acc);
}

// b_n (the FP64 fold) and the bound on its fold error are read on the host
// once per net and passed here.
void launch_final_combine_bn(const Problem& P, FinalAcc acc, double bn, double bn_err, double gamma_M,
                             double inflate, double* out, cudaStream_t s) {
  if (P.B == 0) return;
  count_launch();
  final_combine_kernel<<<(P.B + 3) / 4, 128, 0, s>>>(P, acc, bn, bn_err, gamma_M, inflate, out);
}

double final_gamma(double K) { return gamma_of(K); }

void launch_record_finish(const Problem& P, const double* q, const double* rest, double* out, cudaStream_t s) {
  if (P.B == 0) return;
  count_launch();
  record_finish_kernel<<<(P.B + 255) / 256, 256, 0, s>>>(P, q, rest, out);
}

// Slots used by the final pass of layer k+1 (transposed pass into layer k).
int final_slots(const LayerDev& Lnext, int top) {
  if (top) return 1;
  if (Lnext.kind == LD_LAYER_FC) return (Lnext.n_in + BN - 1) / BN;
  int G = 0;
  if (final_fast_geo(Lnext, G)) return final_fast_blocks(Lnext, G);
  return (Lnext.cin * Lnext.h * Lnext.w + NT - 1) / NT;
}

}  // namespace ld
