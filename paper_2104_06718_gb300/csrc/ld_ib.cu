// Propagation-based intermediate bounds: CROWN, WK and their layer-wise best
// (Sec. 2.2.1 propagation methods; Sec. 2.2.3 intermediate bounds; the
// experiments take per layer the better of CROWN and WK, Sec. 7.2 and BaDNB's
// root bounds of Sec. 5.1.1).
//
// The bound of neuron i of layer k is the lower bound of the objective
// c^T x_hat_k with c = +e_i (lower) or c = -e_i (minus the upper), obtained by
// substituting c backwards through the layers with each ReLU replaced by a
// linear lower relaxation a_low * x_hat and the upper relaxation
// a_bar * x_hat + b_bar of Eq. (slopes-biases):
//   a_{k-1} = W_k^T c, const = c^T b_k
//   for j = k-1 .. 1:  mu_j = a_low [a_j]_+ + a_bar [a_j]_-
//                      const += [a_j]_-^T b_bar_j + mu_j^T b_j,  a_{j-1} = W_j^T mu_j
//   bound = const + sum_i min(a_0[i] l0[i], a_0[i] u0[i])
// CROWN takes a_low = 1[u >= -l] for an ambiguous ReLU (footnote of Sec. 4.2),
// WK a_low = a_bar (the WK relaxation quoted in Sec. 4.1).  Layer 1 is the
// exact range of an affine map over the box (the interval bound of layer 1).
//
// Rows (owner x rule x sign x neuron) run in groups of 32, one row per lane of
// a warp, with the coefficient vectors of a group stored coefficient-major
// (the 32 rows of a coefficient side by side in 128 bytes).  Every lane of a
// warp then forms the same element of its own row: the weight is one
// broadcast load for 32 rows, the coefficients are one coalesced load shared
// by up to eight channels, and no lane waits for another's sparsity.
//   * Rows of a conv layer: a group is one output position of one owner, its
//     lanes the (rule, sign, channel) combinations, so all 32 rows reach the
//     same window of every layer below; only that window is stored and
//     visited (its size is the same for every position; positions of it
//     outside the plane are skipped).
//   * Rows of an FC layer reach everything: lanes are consecutive rows.
//   * An element whose ReLU is blocking in every row of the group relaxes to a
//     zero coefficient whatever its sum is, so the sum is not formed; a
//     coefficient that is zero in every row is skipped (it would add exact
//     zeros).  Rows of one owner share both patterns, so these tests are
//     uniform and cost one vote.
//
// Each transposed pass a = W^T mu is a compensated FP32 dot product (each
// product split exactly into value and error by an FMA, the running sum by
// TwoSum, the errors summed alongside: Ogita, Rump and Oishi's Dot2), with a
// sum of |w mu| rounded upward beside it.  The result's error is at most
// u |a| + gamma_K^2 sum|W||mu| (u = 2^-24, K = terms per sum), and since a
// multiplies x_{j-1} in the substitution, the bound is lowered by that error
// times max|x_{j-1}|.  (A plain FP32 sum would carry gamma_K sum|W||mu|,
// which over a deep chain of substitutions loosens the bounds by ~1e-3.)
// The relaxation slopes are rounded in the direction that keeps each
// relaxation valid (a_bar upward, b_bar upward; any lower slope in [0,1] is
// valid), and a rounded mu_j product lowers the bound by its rounding error
// times max|x_hat_j|.  The scalar terms of a row (box, bias and intercept
// products) are exact FP32 product pairs summed by the same Dot2 in two halves of
// at most 16 terms, then added in FP64: GB300 runs 2 FP64 operations per clock
// and SM against 128 FP32 ones (64 Base subdomains: 6.1 ms with one FP64 FMA a
// term, 4.7 with a third level of errors, 3.7 with Dot2).  That leaves at
// most 16^2 2^-48 of a block's |terms| beside the gamma_M (FP64) of the sum of
// |terms|; kErrA gives back more than that, so the bounds are no wider than with
// FP64 sums.  Products below 2^-102, which have no exact low part (2^-150 each),
// are covered by 2^-126 a row; a CTA whose terms or errors sum to 2^100 or more
// runs its units again with FP64 terms (a test and a branch a term instead cost
// that call 15 to 20%).  The error bounds are summed in FP32 over a block, in FP64
// over the blocks, the sizes of the terms in FP32 over a thread's units, all
// rounded upward.  So the returned bounds contain the exact CROWN/WK bounds
// (outward), like the interval bounds.
//
// A row's value does not depend on the other rows of a call: the elements of a
// layer are dealt to CTAs and warps by the layer's geometry alone.
#include <algorithm>
#include <cmath>

#include "ld_common.cuh"

namespace ld {
namespace {

constexpr int NW = 8;              // warps per CTA
constexpr int NT = 32 * NW;
constexpr int kUnitC = 8;          // elements per unit (channels of a position / consecutive FC inputs)
// Elements per unit of FC layers with fewer inputs than kWideFc.  Units of 8 leave
// a small call one to three CTAs a group, each a chain of waits (two to five units
// a warp in a row): CROWN/WK bounds of one row of a 400-20-20-20-1 net 203 us, with
// units of 2 and one a warp 106; FSB of 128-128-1 157 and 84 us.  600 rows of such
// nets take up to 1.7 times as long as with units of 8 (300-24-100-1; 80-80-80-80-1 3.0
// -> 3.8 ms, 17.7 with a CTA per row).  The inputs alone decide, so that a row's value
// stays the same in any batch.
constexpr int kUnitFc = 2, kWideFc = 1024;
constexpr int kAdds = 16;          // most scalar terms of each half of a row's sum between two FP64 flushes
constexpr int kMaxChunks = 64;     // CTAs of a group
constexpr int kWarpWork = 1024;    // terms a warp should have (2 to 8 units): its fixed cost is a few hundred instructions
constexpr int kFcRows = 128;       // FC weight rows staged at once (a CTA has one unit per warp)
// Most staged weights of a conv: 12288 of them, one input channel padded to four.
constexpr size_t kStageMost = sizeof(float) * 4 * 12288;
constexpr unsigned kFull = 0xffffffffu;
constexpr float kTwoU = 1.1920928955078125e-07f;  // 2^-23, twice the FP32 unit roundoff
// The rounding of p + c is at most 2^-24 |a|; 2^-23 (1 - 2^-13) is charged for it.
// The 2^-13 is more than the bounds lose by FP32 scalar terms and error sums: a
// box or intercept term is at most |a| times what its error multiplies, so it
// gives back 2^-36 of their sizes (2^-40 are charged) and 2^-13 of the error.
constexpr float kErrA = 1.1920928955078125e-07f * (1.f - 1.220703125e-04f);
constexpr float kHuge = 1.2676506002282294e30f;   // 2^100

// Window of a group's nonzero coefficients on a plane: full, or hh x ww from
// (oy * mul - sub, ox * mul - sub) for the group's position (oy, ox).
struct IbWin {
  int full;
  int hh, ww;
  int mul, sub;
};

struct IbStep {
  LayerDev L;               // layer j: this launch computes a_{j-1} = W_j^T mu_j
  int seed;                 // 1: mu_j is the row's objective (+-e_i, layer k = j): a is a row of W_k, exact
  int box;                  // 1: j == 1, the epilogue adds the box term
  IbWin win, wout;          // windows of mu_j (unused when seed) and of mu_{j-1}
  int in_elems, out_elems;  // coefficients of a group in each
  const float* mu_in;       // [groups of the chunk][in_elems][32]
  float* mu_out;            // [groups of the chunk][out_elems][32] (unused when box)
  const float* bias_prev;   // hidden epilogue: bias of layer j-1 (plane_prev outputs per channel)
  int plane_prev;
  int prev_r_off;           // layer j-1 in the flat ReLU vector
  float g2;                 // upper bound on 2 gamma_K^2 of this pass's sums (0 when seed)
  int chunks, units, units_per_cta;
  int cp;                   // floats of a staged weight row (conv: cin rounded up)
  int flush;                // units between FP64 flushes of the scalar terms
  int slot;                 // this launch's first partial-sum slot
  // bounds of the layers before k, per owner [owners, N], already clamped; boxes
  const float* lbk;
  const float* ubk;
  int N;
  const float* l0;
  const float* u0;
  int n0;
  const int32_t* box_row;   // owner -> box row (nullptr: box_of_owner = owner, or 0 with one box)
  int n_boxes;
  double* part;             // [slots, 32 * groups of the chunk, 3]: value, sum |terms| (up), error bound (up)
};

// Rows of the layer being bounded and their order in groups of 32.
struct IbRowMap {
  int conv;                 // 1: groups are (owner, output position, block of 32 combinations)
  int n_k;                  // neurons of the layer
  int cout, wo, hw;         // conv: channels, output width, positions
  int n_rules, n_signs;
  int rule0;                // rule of rule index 0: 0 CROWN, 1 WK (index 1 is WK)
  int per_pos, gpp;         // conv: combinations of a position, groups of a position
  int64_t rows;             // owners * n_rules * n_signs * n_k
  int64_t group0;           // first group of this chunk
  int n_groups;             // groups of this chunk
};

struct IbRow {
  bool valid;
  int owner, rule, i;
  int oy, ox;               // conv: the group's position (uniform over a warp)
  float sign;
  int64_t acc;              // row index, owner-major: ((owner * rules + rule) * signs + sign) * n_k + i
};

__device__ __forceinline__ IbRow ib_row(const IbRowMap& M, int64_t g, int lane) {
  IbRow r;
  int q, sg;
  r.oy = r.ox = 0;
  if (M.conv) {
    const int64_t per_owner = (int64_t)M.hw * M.gpp;
    r.owner = (int)(g / per_owner);
    const int rem = (int)(g % per_owner);
    const int pos = rem / M.gpp;
    int t = (rem % M.gpp) * 32 + lane;
    r.valid = t < M.per_pos;
    if (!r.valid) t = 0;
    const int o = t % M.cout;
    t /= M.cout;
    sg = t % M.n_signs;
    q = t / M.n_signs;
    r.oy = pos / M.wo;
    r.ox = pos - r.oy * M.wo;
    r.i = o * M.hw + pos;
  } else {
    int64_t e = g * 32 + lane;
    r.valid = e < M.rows;
    if (!r.valid) e = M.rows - 1;
    r.i = (int)(e % M.n_k);
    e /= M.n_k;
    sg = (int)(e % M.n_signs);
    e /= M.n_signs;
    q = (int)(e % M.n_rules);
    r.owner = (int)(e / M.n_rules);
  }
  r.rule = q == 0 ? M.rule0 : 1;
  r.sign = sg == 0 ? 1.f : -1.f;
  r.acc = (((int64_t)r.owner * M.n_rules + q) * M.n_signs + sg) * M.n_k + r.i;
  return r;
}

// Units of ib_box_kernel in one row of a window of ww columns.
__host__ __device__ __forceinline__ int box_units(int stride, int ww) {
  return stride * (((ww + stride - 1) / stride + 1) / 2);
}
// Elements of a unit of a_{j-1}, the inputs of layer L.
inline int unit_elems(const LayerDev& L) { return L.kind == LD_LAYER_FC && L.n_in < kWideFc ? kUnitFc : kUnitC; }
// Whether a_0 of first layer L goes through ib_box_kernel.
inline bool box_pairs(const LayerDev& L) { return L.kind == LD_LAYER_CONV && L.cin <= 4; }

__device__ __forceinline__ int box_of(const IbStep& st, int owner) {
  if (st.box_row) {
    const int p = st.box_row[owner];
    return p < 0 ? 0 : (p >= st.n_boxes ? st.n_boxes - 1 : p);
  }
  return st.n_boxes == 1 ? 0 : owner;
}

// Compensated dot product state: running sum p, accumulated errors c, and
// s >= (sum |w m|) / (1 + u) (the rounded products' sizes, rounded up).
struct Dot2 {
  float p = 0.f, c = 0.f, s = 0.f;
  __device__ __forceinline__ void add(float w, float m) {
    const float h = __fmul_rn(w, m);
    const float r = __fmaf_rn(w, m, -h);           // w m = h + r exactly
    const float t = __fadd_rn(p, h);               // TwoSum(p, h) = t + q exactly
    const float bv = __fsub_rn(t, p);
    const float av = __fsub_rn(t, bv);
    const float q = __fadd_rn(__fsub_rn(p, av), __fsub_rn(h, bv));
    p = t;
    c = __fadd_rn(c, __fadd_rn(q, r));
    s = __fadd_ru(s, fabsf(h));
  }
  __device__ __forceinline__ float value() const { return __fadd_rn(p, c); }
  __device__ __forceinline__ float size() const { return __fmul_ru(s, 1.f + 2.f * kTwoU); }
};

// b - a by one packed instruction (a packed add takes no negated operand; the
// product with -1 is exact, so the rounding is that of the subtraction).
__device__ __forceinline__ float2 sub2(float2 b, float2 a) { return __ffma2_rn(a, make_float2(-1.f, -1.f), b); }

// Two Dot2 in packed form (with nh = -h and nb = -bv of Dot2::add).
struct Pair {
  float2 p = {0.f, 0.f}, c = {0.f, 0.f}, s = {0.f, 0.f};
  __device__ __forceinline__ void add(float2 v, float2 m, float2 nm) {
    const float2 nh = __fmul2_rn(v, nm);
    const float2 r = __ffma2_rn(v, m, nh);
    const float2 t = sub2(p, nh);
    const float2 nb = sub2(p, t);
    const float2 q = __fadd2_rn(sub2(p, __fadd2_rn(t, nb)), sub2(nb, nh));
    p = t;
    c = __fadd2_rn(c, __fadd2_rn(q, r));
    s = make_float2(__fadd_ru(s.x, fabsf(nh.x)), __fadd_ru(s.y, fabsf(nh.y)));
  }
};

// The dot products of a unit's needed elements, two per packed instruction
// (half the issue slots of two Dot2, which leaves them to loads and votes) and
// a last odd one by itself; pairs past np are not touched.
template <int UC>
struct UnitSums {
  static constexpr int kPairs = UC / 2;
  Pair d[kPairs];
  Dot2 one;
  int wa[kPairs], wb[kPairs], w1;    // the elements' places in a staged weight row
  int np;
  bool odd;
  __device__ __forceinline__ void add(const float* ws, float m1) {
    const float2 m = make_float2(m1, m1), nm = make_float2(-m1, -m1);
#pragma unroll
    for (int k = 0; k < kPairs; ++k)
      if (np > k) d[k].add(make_float2(ws[wa[k]], ws[wb[k]]), m, nm);
    if (odd) one.add(ws[w1], m1);
  }
  // Adds n terms: m at mp + k mstep (one coalesced load for all elements), the
  // weights at ws + k CP.  A coefficient that is zero in every row is skipped.
  template <int CP>
  __device__ __forceinline__ void run(const float* __restrict__ mp, int mstep, const float* ws, int cp, int n) {
    const int wstep = CP ? CP : cp;
    constexpr int U = UC == 2 ? 8 : 4;  // coefficients in flight
    int k = 0;
    for (; k + U <= n; k += U, mp += U * (size_t)mstep, ws += U * wstep) {
      float m[U];
#pragma unroll
      for (int q = 0; q < U; ++q) m[q] = __ldg(mp + q * (size_t)mstep);
#pragma unroll
      for (int q = 0; q < U; ++q)
        if (__any_sync(kFull, m[q] != 0.f)) add(ws + q * wstep, m[q]);
    }
    for (; k < n; ++k, mp += mstep, ws += wstep) {
      const float m = __ldg(mp);
      if (__any_sync(kFull, m != 0.f)) add(ws, m);
    }
  }
};

// A row's scalar terms: the current block's sum (d, two halves) and error bound
// e, with sum |terms| in d.s, and the finished blocks (v, ev); WIDE: all in FP64.
template <bool WIDE>
struct RowSum {
  Pair d;
  float e = 0.f;
  double v = 0.0, ev = 0.0, sv = 0.0;
  __device__ __forceinline__ void add(float2 x, float2 a) {
    if (WIDE) {
      const double t0 = (double)x.x * (double)a.x, t1 = (double)x.y * (double)a.y;
      v += t0;
      v += t1;
      sv = __dadd_ru(sv, __dadd_ru(fabs(t0), fabs(t1)));
    } else {
      d.add(x, a, make_float2(-a.x, -a.y));
    }
  }
  // An error of a coefficient times the size of what it multiplies.
  __device__ __forceinline__ void error(float da, float x) {
    if (WIDE)
      ev = __dadd_ru(ev, __dmul_ru((double)da, (double)x));
    else
      e = __fmaf_ru(da, x, e);
  }
  __device__ __forceinline__ void flush() {
    if (WIDE) return;
    v += widen(d.p.x);
    v += widen(d.p.y);
    v += widen(d.c.x) + widen(d.c.y);
    ev = __dadd_ru(ev, widen(e));
    d.p = d.c = make_float2(0.f, 0.f);
    e = 0.f;
  }
  __device__ __forceinline__ double size() const {
    return WIDE ? sv : (double)__fmul_ru(__fadd_ru(d.s.x, d.s.y), 1.f + 2.f * kTwoU);
  }
  // Whether the sums left FP32's range (infinities and NaN among them), after the last flush.
  __device__ __forceinline__ bool beyond() const { return !WIDE && !(size() < (double)kHuge && ev < (double)kHuge); }
};

// Two elements' contribution to the row: coefficients a with error bounds da on
// the input intervals [l, u] (a = da = l = u = 0: none).
template <bool WIDE>
__device__ __forceinline__ void box_terms(RowSum<WIDE>& R, float2 a, float2 da, float2 l, float2 u) {
  R.add(make_float2(a.x >= 0.f ? l.x : u.x, a.y >= 0.f ? l.y : u.y), a);  // min(a l, a u)
  R.error(da.x, fmaxf(fabsf(l.x), fabsf(u.x)));
  R.error(da.y, fmaxf(fabsf(l.y), fabsf(u.y)));
}

// The coefficient of the next pass: a with error bound da through the relaxation
// of a ReLU with bounds [l, u]; ic: the intercept that multiplies a, or 0.
template <bool WIDE>
__device__ __forceinline__ float relu_coeff(RowSum<WIDE>& R, float a, float da, float l, float u, int rule, float& ic) {
  ic = 0.f;
  if (u <= 0.f) return 0.f;                         // blocking: x = 0, nothing to relax
  float m = a;                                      // passing: x = x_hat
  if (l < 0.f) {
    const float ab = __fdiv_ru(u, __fsub_rd(u, l));  // upper slope, rounded up (still a valid relaxation)
    if (a >= 0.f) {
      const float slo = rule == 0 ? (u >= -l ? 1.f : 0.f) : fminf(ab, 1.f);
      m = slo * a;
    } else {
      m = ab * a;
      ic = __fmul_ru(-l, ab);                       // upper intercept, rounded up
    }
    // rounding of the product mu = slope * a, times max |x_hat|
    R.error(__fmul_ru(kTwoU, fabsf(m)), fmaxf(-l, u));
  }
  // the pass's own rounding, times max x_{j-1} = max(u, 0)
  R.error(da, u);
  return m;
}

// A CTA's sums of its rows into the chunk's slot; false (nothing stored): some
// left FP32's range.
template <bool WIDE>
__device__ __forceinline__ bool store_part(const IbStep& st, const IbRowMap& M, int gl, int chunk,
                                           double (*red)[32][3], const RowSum<WIDE>& R) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  if (!WIDE && __syncthreads_or(R.beyond())) return false;
  red[warp][lane][0] = R.v;
  red[warp][lane][1] = R.size();
  red[warp][lane][2] = R.ev;
  __syncthreads();
  if (threadIdx.x < 96) {
    const int q = threadIdx.x / 32;
    double t = red[0][lane][q];
    for (int w = 1; w < NW; ++w) t = q == 0 ? t + red[w][lane][q] : __dadd_ru(t, red[w][lane][q]);
    st.part[(((size_t)st.slot + chunk) * M.n_groups * 32 + (size_t)gl * 32 + lane) * 3 + q] = t;
  }
  return true;
}

// One CTA: units [chunk * units_per_cta, ...) of one group of 32 rows; a unit
// is UC channels of one position (conv) or UC consecutive inputs (FC).
// The elements that some row needs are summed together from one stream of
// coefficients, the weights in shared memory (conv: [tap][o][cp] channels; FC:
// up to kFcRows rows of the CTA's inputs at a time).  Bound by the FP32 pipe:
// 11 operations a term and element; with one or two elements per stream the
// loads, votes and addresses were most of the instructions.
// CP: floats of a staged weight row where it is one of the usual sizes (the
// four rows of an unrolled step are then immediate offsets), else 0.
template <int CP, int UC, bool WIDE>
__device__ __forceinline__ bool ib_step(const IbStep& st, const IbRowMap& M, float* sw, double (*red)[32][3]) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int gl = blockIdx.x / st.chunks, chunk = blockIdx.x % st.chunks;
  const IbRow r = ib_row(M, M.group0 + gl, lane);
  const LayerDev& L = st.L;
  const bool conv = L.kind == LD_LAYER_CONV;
  if (conv && !st.seed) {
    for (int e = threadIdx.x; e < L.cout * L.kh * L.kw * st.cp; e += NT) {
      const int c = e % st.cp, q = e / st.cp, o = q % L.cout, tap = q / L.cout;
      sw[e] = c < L.cin ? __ldg(L.Wt + ((size_t)o * L.kh * L.kw + tap) * L.cin + c) : 0.f;
    }
    __syncthreads();
  }
  const float* mu = st.mu_in + (size_t)gl * st.in_elems * 32 + lane;
  float* out = st.mu_out + (size_t)gl * st.out_elems * 32 + lane;
  const int iy0 = st.win.full ? 0 : r.oy * st.win.mul - st.win.sub;
  const int ix0 = st.win.full ? 0 : r.ox * st.win.mul - st.win.sub;
  const int oy0 = st.wout.full ? 0 : r.oy * st.wout.mul - st.wout.sub;
  const int ox0 = st.wout.full ? 0 : r.ox * st.wout.mul - st.wout.sub;
  const int cb = conv ? (L.cin + UC - 1) / UC : 0;
  const size_t lo_off = st.box ? (size_t)box_of(st, r.owner) * st.n0 : (size_t)r.owner * st.N + st.prev_r_off;
  const float* lp = (st.box ? st.l0 : st.lbk) + lo_off;
  const float* up = (st.box ? st.u0 : st.ubk) + lo_off;
  // seed: the row's output channel and sign (0: a lane without a row)
  const int so = conv ? r.i / (L.ho * L.wo) : 0;
  const float sg = r.valid ? r.sign : 0.f;
  const int hw = conv ? L.h * L.w : 1, ostep = conv ? st.wout.hh * st.wout.ww : 1;
  RowSum<WIDE> R;
  int done = 0;
  const int u_lo = chunk * st.units_per_cta, u_hi = min(st.units, u_lo + st.units_per_cta);
  for (int ub = u_lo; ub < u_hi; ub += NW) {
    const int un = ub + warp;
    // element c (channel / input) of the unit: flat index ib + c hw, coefficient eb + c ostep
    int y = 0, x = 0, c0 = un * UC, nc = min(UC, L.n_in - c0), ib = 0, eb = 0;
    bool in = un < u_hi;
    if (conv) {
      const int pos = un / cb, wy = pos / st.wout.ww, wx = pos - wy * st.wout.ww;
      c0 = (un - pos * cb) * UC;
      nc = min(UC, L.cin - c0);
      y = oy0 + wy;
      x = ox0 + wx;
      in = in && y >= 0 && y < L.h && x >= 0 && x < L.w;
      ib = y * L.w + x;
      eb = pos;
    }
    unsigned act = in ? (1u << nc) - 1u : 0u;
    if (in && !st.box) {
      // elements blocking in every row relax to zero whatever their sum is
      float u[UC];
#pragma unroll
      for (int q = 0; q < UC; ++q) u[q] = q < nc ? __ldg(up + ib + (c0 + q) * hw) : 0.f;
#pragma unroll
      for (int q = 0; q < UC; ++q)
        if (q < nc && !__any_sync(kFull, u[q] > 0.f)) {
          act &= ~(1u << q);
          out[(size_t)(eb + (c0 + q) * ostep) * 32] = 0.f;
        }
    }
    UnitSums<UC> S;
    S.np = __popc(act) / 2;
    S.odd = __popc(act) & 1;
    {
      const int wb = conv ? c0 : warp * UC;   // the unit's first element in a staged weight row
      unsigned rest = act;
#pragma unroll
      for (int k = 0; k < UC / 2; ++k) {
        S.wa[k] = S.wb[k] = 0;
        if (k < S.np) {
          const int a = __ffs(rest) - 1;
          rest &= rest - 1;
          const int b = __ffs(rest) - 1;
          rest &= rest - 1;
          S.wa[k] = wb + a;
          S.wb[k] = wb + b;
        }
      }
      S.w1 = S.odd ? wb + __ffs(rest) - 1 : 0;
    }
    if (!st.seed && conv) {
      const int estep = st.win.hh * st.win.ww * 32, ys = y + L.pad, xs = x + L.pad;
      // taps i0 + t stride read row (y + pad - i0) / stride - t
      const int i0 = ys % L.stride, j0 = xs % L.stride;
      const int oy = ys / L.stride, ox = xs / L.stride;
      if (act)
        for (int i = i0, qy = oy; i < L.kh && qy >= 0; i += L.stride, --qy) {
          const int wy = qy - iy0;
          if (qy >= L.ho || wy < 0 || wy >= st.win.hh) continue;
          for (int j = j0, qx = ox; j < L.kw && qx >= 0; j += L.stride, --qx) {
            const int wx = qx - ix0;
            if (qx >= L.wo || wx < 0 || wx >= st.win.ww) continue;
            S.run<CP>(mu + (wy * st.win.ww + wx) * 32, estep, sw + (i * L.kw + j) * L.cout * st.cp, st.cp, L.cout);
          }
        }
    } else if (!st.seed) {
      constexpr int kCols = NW * UC;
      for (int o0 = 0; o0 < L.n_out; o0 += kFcRows) {
        const int nr = min(kFcRows, L.n_out - o0);
        __syncthreads();
#pragma unroll 4
        for (int e = threadIdx.x; e < nr * kCols; e += NT) {
          const int o = e / kCols, i = ub * UC + e % kCols;
          sw[e] = i < L.n_in ? __ldg(L.W + (size_t)(o0 + o) * L.n_in + i) : 0.f;
        }
        __syncthreads();
        if (act) S.run<CP>(mu + (size_t)o0 * 32, 32, sw, kCols, nr);
      }
    }
    const int ky = y + L.pad - r.oy * L.stride, kx = x + L.pad - r.ox * L.stride;
    // the elements' sums in pairs, the odd one last with an empty second half
    for (int k = 0; act; ++k) {
      const bool two = k < S.np;
      int c[2], ii[2];
      c[0] = c0 + __ffs(act) - 1;
      act &= act - 1;
      c[1] = two ? c0 + __ffs(act) - 1 : c[0];
      act &= act - (two ? 1u : 0u);
      ii[0] = ib + c[0] * hw;
      ii[1] = ib + c[1] * hw;
      Pair D = S.d[0];
#pragma unroll
      for (int q = 1; q < UC / 2; ++q)
        if (k == q) D = S.d[q];
      if (!two) {
        D.p = make_float2(S.one.p, 0.f);
        D.c = make_float2(S.one.c, 0.f);
        D.s = make_float2(S.one.s, 0.f);
      }
      if (st.seed) {
        float w[2];
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          w[h] = 0.f;
          if (h && !two) continue;
          if (!conv) w[h] = sg * __ldg(L.W + (size_t)r.i * L.n_in + c[h]);
          else if (ky >= 0 && ky < L.kh && kx >= 0 && kx < L.kw)
            w[h] = sg * __ldg(L.W + (((size_t)so * L.cin + c[h]) * L.kh + ky) * L.kw + kx);
        }
        D.p = make_float2(w[0], w[1]);
      }
      const float2 l = make_float2(__ldg(lp + ii[0]), two ? __ldg(lp + ii[1]) : 0.f);
      const float2 u = make_float2(__ldg(up + ii[0]), two ? __ldg(up + ii[1]) : 0.f);
      const float2 a = __fadd2_rn(D.p, D.c);
      float2 da = make_float2(0.f, 0.f);
      if (!st.seed) {
        da.x = __fmaf_ru(st.g2, __fmul_ru(D.s.x, 1.f + 2.f * kTwoU), __fmul_ru(kErrA, fabsf(a.x)));
        da.y = __fmaf_ru(st.g2, __fmul_ru(D.s.y, 1.f + 2.f * kTwoU), __fmul_ru(kErrA, fabsf(a.y)));
      }
      if (st.box) {
        box_terms(R, a, da, l, u);
      } else {
        float2 m = make_float2(0.f, 0.f), ic = m, bias = m;
        if (!(a.x == 0.f && D.s.x == 0.f)) {
          m.x = relu_coeff(R, a.x, da.x, l.x, u.x, r.rule, ic.x);
          bias.x = __ldg(st.bias_prev + ii[0] / st.plane_prev);
        }
        if (!(a.y == 0.f && D.s.y == 0.f)) {
          m.y = relu_coeff(R, a.y, da.y, l.y, u.y, r.rule, ic.y);
          bias.y = __ldg(st.bias_prev + ii[1] / st.plane_prev);
        }
        if (ic.x != 0.f || ic.y != 0.f) R.add(ic, a);
        R.add(bias, m);
        out[(size_t)(eb + c[0] * ostep) * 32] = m.x;
        if (two) out[(size_t)(eb + c[1] * ostep) * 32] = m.y;
      }
    }
    if (++done % st.flush == 0) R.flush();
  }
  R.flush();
  return store_part(st, M, gl, chunk, red, R);
}

// The FP64 form, out of line.
template <int CP, int UC>
__device__ __noinline__ void ib_step_wide(const IbStep& st, const IbRowMap& M, float* sw, double (*red)[32][3]) {
  ib_step<CP, UC, true>(st, M, sw, red);
}
template <int CP, int UC>
__global__ void __launch_bounds__(NT, 3) ib_step_kernel(const __grid_constant__ IbStep st,
                                                        const __grid_constant__ IbRowMap M) {
  extern __shared__ __align__(16) float sw[];
  __shared__ double red[NW][32][3];
  if (!ib_step<CP, UC, false>(st, M, sw, red)) ib_step_wide<CP, UC>(st, M, sw, red);
}

// The input box of a conv first layer of C <= 4 channels: a unit is two
// positions of one row and column phase, `stride` columns apart, and all
// channels.  Both positions meet the same weights, so a packed instruction
// holds one channel's two positions and one 16-byte load all its weights; with
// the general kernel's unit (one position, three channels) the units' set-up
// and votes were two thirds of the instructions.  Base, 3 channels: a call of
// 64 subdomains 5.48 -> 3.38 ms, FSB's children of 256 subdomains 1.42 -> 1.09
// ms, Deep's root bounds 0.685 -> 0.542 ms.
template <int C, bool WIDE>
__device__ __forceinline__ bool ib_box(const IbStep& st, const IbRowMap& M, float* sw /* [tap][o][4] */,
                                       double (*red)[32][3]) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int gl = blockIdx.x / st.chunks, chunk = blockIdx.x % st.chunks;
  const IbRow r = ib_row(M, M.group0 + gl, lane);
  const LayerDev& L = st.L;
  for (int e = threadIdx.x; e < L.cout * L.kh * L.kw * 4; e += NT) {
    const int c = e % 4, q = e / 4, o = q % L.cout, tap = q / L.cout;
    sw[e] = c < C ? __ldg(L.Wt + ((size_t)o * L.kh * L.kw + tap) * C + c) : 0.f;
  }
  __syncthreads();
  const float* mu = st.mu_in + (size_t)gl * st.in_elems * 32 + lane;
  const int iy0 = st.win.full ? 0 : r.oy * st.win.mul - st.win.sub;
  const int ix0 = st.win.full ? 0 : r.ox * st.win.mul - st.win.sub;
  const int oy0 = st.wout.full ? 0 : r.oy * st.wout.mul - st.wout.sub;
  const int ox0 = st.wout.full ? 0 : r.ox * st.wout.mul - st.wout.sub;
  const float* lp = st.l0 + (size_t)box_of(st, r.owner) * st.n0;
  const float* up = st.u0 + (size_t)box_of(st, r.owner) * st.n0;
  const int S = L.stride, estep = st.win.hh * st.win.ww * 32, per_row = box_units(S, st.wout.ww);
  RowSum<WIDE> R;
  int done = 0;
  const int u_hi = min(st.units, (chunk + 1) * st.units_per_cta);
  for (int un = chunk * st.units_per_cta + warp; un < u_hi; un += NW) {
    const int wy = un / per_row, k = un - wy * per_row, wx = k % S + 2 * S * (k / S);
    const int y = oy0 + wy, x = ox0 + wx;
    const bool row = y >= 0 && y < L.h;
    const bool in0 = row && wx < st.wout.ww && x >= 0 && x < L.w;
    const bool in1 = row && wx + S < st.wout.ww && x + S >= 0 && x + S < L.w;
    if (!in0 && !in1) continue;
    Pair d[C];
    // taps j0 + t S read column (x + pad - j0) / S - t, and one more for the second position
    const int ys = y + L.pad, xs = x + L.pad;
    const int j0 = (xs % S + S) % S, cx = (xs - j0) / S;
    for (int i = ys % S, qy = ys / S; i < L.kh && qy >= 0; i += S, --qy) {
      const int iy = qy - iy0;
      if (qy >= L.ho || iy < 0 || iy >= st.win.hh) continue;
      for (int j = j0, qx = cx; j < L.kw; j += S, --qx) {
        const int ix = qx - ix0;
        const bool a = in0 && qx >= 0 && qx < L.wo && ix >= 0 && ix < st.win.ww;
        const bool b = in1 && qx + 1 >= 0 && qx + 1 < L.wo && ix + 1 >= 0 && ix + 1 < st.win.ww;
        if (!a && !b) continue;
        const float* mp = mu + (iy * st.win.ww + ix) * 32;
        const float4* w = reinterpret_cast<const float4*>(sw) + (i * L.kw + j) * L.cout;
        for (int o = 0; o < L.cout; o += 4, mp += 4 * (size_t)estep) {
          float2 m[4];
#pragma unroll
          for (int q = 0; q < 4; ++q) {
            const bool on = o + q < L.cout;
            m[q].x = on && a ? __ldg(mp + (size_t)q * estep) : 0.f;
            m[q].y = on && b ? __ldg(mp + (size_t)q * estep + 32) : 0.f;
          }
#pragma unroll
          for (int q = 0; q < 4; ++q) {
            if (!__any_sync(kFull, m[q].x != 0.f || m[q].y != 0.f)) continue;
            const float4 wv = w[o + q];
            const float2 nm = make_float2(-m[q].x, -m[q].y);
            d[0].add(make_float2(wv.x, wv.x), m[q], nm);
            if (C > 1) d[1 % C].add(make_float2(wv.y, wv.y), m[q], nm);
            if (C > 2) d[2 % C].add(make_float2(wv.z, wv.z), m[q], nm);
            if (C > 3) d[3 % C].add(make_float2(wv.w, wv.w), m[q], nm);
          }
        }
      }
    }
#pragma unroll
    for (int c = 0; c < C; ++c) {
      const int i0 = (c * L.h + y) * L.w + x, i1 = i0 + S;
      float2 a = __fadd2_rn(d[c].p, d[c].c), da, l = make_float2(0.f, 0.f), u = l;
      da.x = __fmaf_ru(st.g2, __fmul_ru(d[c].s.x, 1.f + 2.f * kTwoU), __fmul_ru(kErrA, fabsf(a.x)));
      da.y = __fmaf_ru(st.g2, __fmul_ru(d[c].s.y, 1.f + 2.f * kTwoU), __fmul_ru(kErrA, fabsf(a.y)));
      if (in0) {
        l.x = __ldg(lp + i0);
        u.x = __ldg(up + i0);
      } else {
        a.x = da.x = 0.f;
      }
      if (in1) {
        l.y = __ldg(lp + i1);
        u.y = __ldg(up + i1);
      } else {
        a.y = da.y = 0.f;
      }
      box_terms(R, a, da, l, u);
    }
    if (++done % st.flush == 0) R.flush();
  }
  R.flush();
  return store_part(st, M, gl, chunk, red, R);
}

template <int C>
__device__ __noinline__ void ib_box_wide(const IbStep& st, const IbRowMap& M, float* sw, double (*red)[32][3]) {
  ib_box<C, true>(st, M, sw, red);
}
template <int C>
__global__ void __launch_bounds__(NT, 3) ib_box_kernel(const __grid_constant__ IbStep st,
                                                       const __grid_constant__ IbRowMap M) {
  extern __shared__ __align__(16) float sw[];
  __shared__ double red[NW][32][3];
  if (!ib_box<C, false>(st, M, sw, red)) ib_box_wide<C>(st, M, sw, red);
}

// Sums a chunk's slots per row (fixed order), with the objective's bias term.
__global__ void __launch_bounds__(NT) ib_collect_kernel(IbRowMap M, int slots, const double* part, const float* bias,
                                                        int plane, double* acc) {
  const int64_t t = blockIdx.x * (int64_t)NT + threadIdx.x;
  if (t >= (int64_t)M.n_groups * 32) return;
  const IbRow r = ib_row(M, M.group0 + t / 32, (int)(t % 32));
  if (!r.valid) return;
  double v = (double)r.sign * (double)bias[r.i / plane], av = fabs(v), e = 1.1754943508222875e-38;  // 2^-126: see the top
  for (int s = 0; s < slots; ++s) {
    const double* p = part + ((size_t)s * M.n_groups * 32 + t) * 3;
    v += p[0];
    av = __dadd_ru(av, p[1]);
    e = __dadd_ru(e, p[2]);
  }
  double* a = acc + (size_t)r.acc * 3;
  a[0] = v;
  a[1] = av;
  a[2] = e;
}

struct IbFinish {
  int n_owners, n_k, n_rules, n_signs, N, r_off;
  const double* acc;
  double gamma_M;
  const int8_t* mask;       // [owners, N] or nullptr
  float* lbk;
  float* ubk;
  double* out_lb;           // output layer: the lower bound per owner (nullptr: lbk/ubk)
};

// Layer-wise best over the rules: l = max of the lower bounds, u = min of
// the upper bounds (minus the lower bounds of -x_hat); split clamp; stored
// rounded outward to FP32.
__global__ void ib_finish_kernel(IbFinish f) {
  const int64_t total = (int64_t)f.n_owners * f.n_k;
  for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < total; t += (int64_t)gridDim.x * blockDim.x) {
    const int owner = (int)(t / f.n_k), i = (int)(t % f.n_k);
    double lo = -INFINITY, up = INFINITY;
    for (int q = 0; q < f.n_rules; ++q)
      for (int sg = 0; sg < f.n_signs; ++sg) {
        const int64_t r = (((int64_t)owner * f.n_rules + q) * f.n_signs + sg) * f.n_k + i;
        const double* p = f.acc + (size_t)r * 3;
        const double b = __dsub_rd(__dsub_rd(p[0], p[2]), __dmul_ru(f.gamma_M, p[1]));
        if (sg == 0) lo = fmax(lo, b);
        else up = fmin(up, -b);
      }
    if (f.out_lb) {
      f.out_lb[owner] = lo;
      continue;
    }
    float l = __double2float_rd(lo), u = __double2float_ru(up);
    const size_t j = (size_t)owner * f.N + f.r_off + i;
    if (f.mask) {
      const int m = f.mask[j];
      if (m > 0) l = fmaxf(l, 0.f);
      if (m < 0) u = fminf(u, 0.f);
    }
    f.lbk[j] = l;
    f.ubk[j] = u;
  }
}

double gamma32(int K) {
  const double u = 5.9604644775390625e-08;  // 2^-24
  return K * u / (1.0 - K * u) * (1.0 + 1e-6);
}

// Geometry of the substitution of layer k's rows, layer by layer.
struct IbGeo {
  IbWin w[kMaxLayers + 1];   // w[j]: window on layer j's output plane (j < k)
  int elems[kMaxLayers + 1];
  int units[kMaxLayers + 1], chunks[kMaxLayers + 1], per_cta[kMaxLayers + 1];  // of the launch that forms a_j
  int slots, width;          // partial-sum slots of a chunk, widest hidden level
};

IbGeo ib_geo(const std::vector<LayerDev>& Ls, int k) {
  IbGeo g{};
  int mul = 1, sub = 0, hh = 1, ww = 1;
  bool full = Ls[k - 1].kind == LD_LAYER_FC;
  for (int j = k - 1; j >= 0; --j) {
    const LayerDev& up = Ls[j];  // layer j+1, whose input plane this is
    if (up.kind == LD_LAYER_CONV && !full) {
      // positions [y0, y0 + hh) of its output reach [y0 s - p, (y0 + hh - 1) s - p + k) of its input
      hh = (hh - 1) * up.stride + up.kh;
      ww = (ww - 1) * up.stride + up.kw;
      mul *= up.stride;
      sub = sub * up.stride + up.pad;
      // the whole plane once the window is no smaller, or where an FC layer reads it flat
      if (hh >= up.h || ww >= up.w || (j >= 1 && Ls[j - 1].kind == LD_LAYER_FC)) full = true;
    }
    g.w[j] = full ? IbWin{1, up.h, up.w, 0, 0} : IbWin{0, hh, ww, mul, sub};  // full: as layer j+1 sees it
    const bool conv = up.kind == LD_LAYER_CONV;
    g.elems[j] = conv ? up.cin * g.w[j].hh * g.w[j].ww : up.n_in;
    const int uc = unit_elems(up);
    g.units[j] = conv ? g.w[j].hh * g.w[j].ww * ((up.cin + uc - 1) / uc) : (up.n_in + uc - 1) / uc;
    int unit_terms = up.fan_t * std::min(uc, conv ? up.cin : up.n_in);
    if (j == 0 && box_pairs(up)) {
      g.units[j] = g.w[j].hh * box_units(up.stride, g.w[j].ww);
      unit_terms = 2 * up.fan_t * up.cin;
    }
    const int per_warp = uc == kUnitFc ? 1 : std::min(8, std::max(2, kWarpWork / unit_terms));
    g.per_cta[j] = NW * std::max(per_warp, (g.units[j] + NW * kMaxChunks - 1) / (NW * kMaxChunks));
    g.chunks[j] = (g.units[j] + g.per_cta[j] - 1) / g.per_cta[j];
    g.slots += g.chunks[j];
    if (j >= 1) g.width = std::max(g.width, g.elems[j]);
  }
  return g;
}

IbRowMap ib_rows(const LayerDev& Lk, int n_owners, int n_rules, int n_signs, int rule0) {
  IbRowMap M{};
  M.conv = Lk.kind == LD_LAYER_CONV;
  M.n_k = Lk.n_out;
  M.cout = Lk.cout;
  M.wo = Lk.wo;
  M.hw = Lk.ho * Lk.wo;
  M.n_rules = n_rules;
  M.n_signs = n_signs;
  M.rule0 = rule0;
  M.per_pos = n_rules * n_signs * Lk.cout;
  M.gpp = (M.per_pos + 31) / 32;
  M.rows = (int64_t)n_owners * n_rules * n_signs * Lk.n_out;
  return M;
}

int64_t ib_groups(const IbRowMap& M, int n_owners) {
  return M.conv ? (int64_t)n_owners * M.hw * M.gpp : (M.rows + 31) / 32;
}

}  // namespace

// Workspace of layer k's bounds for n_owners: row sums, the partial sums and
// the two coefficient buffers of a chunk of groups (at most kMuCap together).
IbSpace ib_space(const std::vector<LayerDev>& Ls, int k, int n_owners, int n_rules, int n_signs) {
  constexpr size_t kMuCap = (size_t)256 << 20;
  const IbGeo g = ib_geo(Ls, k);
  const IbRowMap M = ib_rows(Ls[k - 1], n_owners, n_rules, n_signs, 0);
  const size_t per_group = sizeof(float) * 32 * (size_t)g.width;
  IbSpace sp;
  const int64_t cap = std::max<int64_t>(1, (int64_t)(kMuCap / (2 * per_group)));
  sp.chunk_groups = std::max<int64_t>(1, std::min<int64_t>({cap, ib_groups(M, n_owners), int64_t(1) << 24}));
  sp.acc = 24 * (size_t)std::max<int64_t>(1, M.rows);
  sp.mu = per_group * (size_t)sp.chunk_groups;
  sp.part = 24 * 32 * (size_t)g.slots * (size_t)sp.chunk_groups;
  return sp;
}

// Bounds of layer k (2 <= k <= n) for every owner, from the bounds of the
// layers before it (already in lbk/ubk, clamped); see IbLayerArgs.
cudaError_t launch_ib_layer(const std::vector<LayerDev>& Ls, int k, const IbLayerArgs& A, cudaStream_t s) {
  const LayerDev& Lk = Ls[k - 1];
  const int n_signs = A.out_lb ? 1 : 2;
  IbRowMap M = ib_rows(Lk, A.n_owners, A.n_rules, n_signs, A.rule0);
  if (M.rows == 0) return cudaSuccess;
  const IbGeo g = ib_geo(Ls, k);
  const int64_t groups = ib_groups(M, A.n_owners);
  IbStep st{};
  st.lbk = A.lbk;
  st.ubk = A.ubk;
  st.N = A.N;
  st.l0 = A.l0;
  st.u0 = A.u0;
  st.n0 = A.n0;
  st.box_row = A.box_row;
  st.n_boxes = A.n_boxes;
  st.part = A.part;
  // FP64 sums, plus Dot2's errors in halves of n = kAdds terms: n^2 2^-48 of their
  // |terms| (its c sums at most n 2^-24 of them in n steps of two roundings)
  const double gamma_M = A.gamma_M + 1.001 * std::ldexp((double)kAdds * kAdds, -48);
  const int plane_k = Lk.kind == LD_LAYER_FC ? 1 : Lk.ho * Lk.wo;
  const int64_t chunk = ib_space(Ls, k, A.n_owners, A.n_rules, n_signs).chunk_groups;
  for (int64_t g0 = 0; g0 < groups; g0 += chunk) {
    M.group0 = g0;
    M.n_groups = (int)std::min(chunk, groups - g0);
    float* cur = A.mu_a;
    float* nxt = A.mu_b;
    st.slot = 0;
    for (int j = k; j >= 1; --j) {
      const LayerDev& L = Ls[j - 1];
      st.L = L;
      st.seed = j == k;
      st.box = j == 1;
      st.win = j == k ? IbWin{1, 1, 1, 0, 0} : g.w[j];
      if (st.win.full) st.win = IbWin{1, L.ho, L.wo, 0, 0};
      st.wout = g.w[j - 1];
      if (st.wout.full) st.wout = IbWin{1, L.h, L.w, 0, 0};
      st.in_elems = st.seed ? 0 : g.elems[j];
      st.out_elems = g.elems[j - 1];
      st.mu_in = cur;
      st.mu_out = nxt;
      if (j >= 2) {
        const LayerDev& Lp = Ls[j - 2];
        st.bias_prev = Lp.b;
        st.plane_prev = Lp.kind == LD_LAYER_FC ? 1 : Lp.ho * Lp.wo;
        st.prev_r_off = Lp.r_out_off;
      } else {
        st.bias_prev = nullptr;
        st.plane_prev = 1;
        st.prev_r_off = 0;
      }
      const double gk = st.seed ? 0.0 : gamma32(L.fan_t);
      st.g2 = (float)(2.0 * gk * gk * (1.0 + 1e-6));
      st.chunks = g.chunks[j - 1];
      st.units = g.units[j - 1];
      st.units_per_cta = g.per_cta[j - 1];
      const bool conv = L.kind == LD_LAYER_CONV;
      const int uc = unit_elems(L);
      st.cp = conv ? (L.cin <= 4 ? 4 : L.cin <= 8 ? 8 : L.cin <= 16 ? 16 : (L.cin + 1) & ~1) : NW * uc;
      const bool pairs = st.box && !st.seed && box_pairs(L);
      if (pairs) st.cp = 4;
      const int adds = pairs ? L.cin : (st.box ? 1 : 2) * ((std::min(uc, conv ? L.cin : L.n_in) + 1) / 2);
      st.flush = std::max(1, kAdds / adds);
      const size_t smem = sizeof(float) * (size_t)st.cp * (st.seed ? 0
                                                           : conv  ? L.cout * L.kh * L.kw
                                                                   : std::min(kFcRows, L.n_out));
      auto kernel = pairs         ? (L.cin == 1   ? ib_box_kernel<1>
                                     : L.cin == 2 ? ib_box_kernel<2>
                                     : L.cin == 3 ? ib_box_kernel<3>
                                                  : ib_box_kernel<4>)
                    : uc == kUnitFc ? ib_step_kernel<NW * kUnitFc, kUnitFc>
                    : st.cp == 4  ? ib_step_kernel<4, kUnitC>
                    : st.cp == 8  ? ib_step_kernel<8, kUnitC>
                    : st.cp == 16 ? ib_step_kernel<16, kUnitC>
                    : st.cp == 64 ? ib_step_kernel<64, kUnitC>
                                  : ib_step_kernel<0, kUnitC>;
      if (smem > 40 * 1024) {
        const cudaError_t ea = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kStageMost);
        if (ea != cudaSuccess) return ea;
      }
      count_launch();
      kernel<<<(unsigned)(M.n_groups * (int64_t)st.chunks), NT, smem, s>>>(st, M);
      cudaError_t e = cudaGetLastError();
      if (e != cudaSuccess) return e;
      st.slot += st.chunks;
      std::swap(cur, nxt);
    }
    count_launch();
    ib_collect_kernel<<<(unsigned)((M.n_groups * 32LL + NT - 1) / NT), NT, 0, s>>>(M, g.slots, A.part, Lk.b, plane_k,
                                                                                 A.acc);
  }
  IbFinish f{A.n_owners, Lk.n_out, A.n_rules, n_signs, A.N, Lk.r_out_off, A.acc, gamma_M, A.mask,
             A.lbk, A.ubk, A.out_lb};
  const int64_t total = (int64_t)A.n_owners * Lk.n_out;
  const int grid = (int)((total + 255) / 256 < 65535 ? (total + 255) / 256 : 65535);
  count_launch();
  ib_finish_kernel<<<grid > 0 ? grid : 1, 256, 0, s>>>(f);
  return cudaGetLastError();
}

}  // namespace ld
