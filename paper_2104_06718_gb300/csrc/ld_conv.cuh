// The blocked conv passes (k4 s2 / k3 s1) on operands staged in shared memory:
// device code shared by the layerwise kernels (ld_passes.cu) and the proximal
// solver's block kernel (ld_prox.cu), and the host's choice of their tiles.
#pragma once
#include <algorithm>

#include "ld_common.cuh"

namespace ld {
namespace {

// Shared-memory tile of the blocked conv passes: the weights, then the rows of
// the operand plane that a band of outputs reads, zero outside the plane (a
// tap there adds an exact zero to the chain), rows split by column phase for a
// stride-2 forward pass so that consecutive outputs read consecutive words.
struct ConvTile {
  int bands, bh;        // bands of bh rows (transposed pass: rows of a stride phase)
  int rows, pitch;      // staged rows per channel and their pitch (floats)
  int y_off, x_off;     // plane row / column of the tile's first, relative to the band's first row * stride
  int w_floats, wc;     // floats of the staged weights; transposed: channels per tap in them (cin padded to 4)
  size_t smem;
};

__device__ __forceinline__ void stage16(float* dst, const float* src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((unsigned)__cvta_generic_to_shared(dst)), "l"(src)
               : "memory");
}
__device__ __forceinline__ void stage4(float* dst, const float* src, bool in) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"((unsigned)__cvta_generic_to_shared(dst)), "l"(src),
               "r"(in ? 4 : 0)
               : "memory");
}
__device__ __forceinline__ void stage_wait() {
  asm volatile("cp.async.wait_all;" ::: "memory");
  __syncthreads();
}
__device__ __forceinline__ void stage_floats(float* dst, const float* src, int n, int nt) {
  for (int e = threadIdx.x; e < n / 4; e += nt) stage16(dst + 4 * e, src + 4 * e);
  for (int e = (n & ~3) + threadIdx.x; e < n; e += nt) stage4(dst + e, src + e, true);
}

// A division by a number the whole launch shares: a shift for a power of two.
struct SharedDiv {
  int d, sh;
  __device__ __forceinline__ int of(int n) const { return sh >= 0 ? n >> sh : n / d; }
};
__device__ __forceinline__ SharedDiv shared_div(int d) { return SharedDiv{d, (d & (d - 1)) == 0 ? __ffs(d) - 1 : -1}; }

// f(e, c, y, x) for the elements e = (c rows + y) pitch + x of a staged tile,
// thread t taking e = t, t + nt, ...: the coordinates move on by those of nt
// with two carries.  Two divisions an element made staging a tile as many
// instructions as its products; with these, shifts in the items' indices and
// pointers that step through the taps, 512 Wide subdomains: a transposed pass
// into the image 27 -> 22 us, the evaluation call 376 -> 354 us; a proximal call
// (256 Base subdomains, T = 100) 16.7 -> 16.3 ms.
template <class F>
__device__ __forceinline__ void tile_elements(int channels, int rows, int pitch, int nt, F f) {
  const int plane = rows * pitch, n = channels * plane;
  const int dc = nt / plane, dr = (nt - dc * plane) / pitch, dx = nt - dc * plane - dr * pitch;
  int e = threadIdx.x, c = e / plane, y = (e - c * plane) / pitch, x = e - c * plane - y * pitch;
  while (e < n) {
    f(e, c, y, x);
    e += nt;
    x += dx;
    y += dr;
    c += dc;
    if (x >= pitch) {
      x -= pitch;
      ++y;
    }
    if (y >= rows) {
      y -= rows;
      ++c;
    }
  }
}

// Weights of the transposed pass: [o][i][j][wc].
__device__ __forceinline__ void conv_t_weights(const LayerDev& L, const ConvTile& T, float* sW, int nt) {
  const int nw = L.cout * L.cin * L.kh * L.kw;
  if (T.wc == L.cin) {
    stage_floats(sW, L.Wt, nw, nt);
  } else {
    for (int e = threadIdx.x; e < nw; e += nt) stage4(sW + e / L.cin * T.wc + e % L.cin, L.Wt + e, true);
  }
}

// The rows of r (one subdomain's [cout, ho, wo]) read by the band from phase row q0.
__device__ __forceinline__ void conv_t_rows(const LayerDev& L, const ConvTile& T, float* sR, const float* rb, int q0,
                                            int nt) {
  const int hw_o = L.ho * L.wo;
  tile_elements(L.cout, T.rows, T.pitch, nt, [&](int e, int o, int yy, int xx) {
    const int y = q0 + yy + T.y_off, x = xx + T.x_off;
    const bool in = y >= 0 && y < L.ho && x >= 0 && x < L.wo;
    stage4(sR + e, rb + (in ? o * hw_o + y * L.wo + x : 0), in);
  });
}

// f(channel, y, x, g) for every output of the band: a thread takes one
// position of one stride phase and G channels; g[c, yy, xx] = sum_{o,i,j}
// W[o,c,i,j] r[o, y, x] over the taps of the phase, one chain of FMAs per
// output in the order (i, j, o).
template <int KH, int KW, int ST, int G, class F>
__device__ __forceinline__ void conv_t_items(const LayerDev& L, const ConvTile& T, const float* sW, const float* sR,
                                             int q0, int nq, int nt, F f) {
  const int qw = L.w / ST, ncg = L.cin / G, plane = T.rows * T.pitch;
  const int items = ST * ST * ncg * nq * qw, wstep = KH * KW * T.wc;
  const SharedDiv d_qw = shared_div(qw), d_nq = shared_div(nq);
  for (int e = threadIdx.x; e < items; e += nt) {
    int q = e / ST, r = d_qw.of(q);
    const int rx = e - q * ST, qx = q - r * qw;
    q = d_nq.of(r);
    const int qy = r - q * nq;
    const int ry = q % ST;
    const int cg = q / ST;
    const int i0 = (ry + L.pad) % ST, j0 = (rx + L.pad) % ST;
    const int dy0 = (ry + L.pad - i0) / ST, dx0 = (rx + L.pad - j0) / ST;
    // channel pairs in packed FMAs (two round-to-nearest FMAs each)
    float2 a01 = make_float2(0.f, 0.f), a23 = a01;
    const float* rp = sR + (qy + dy0 - T.y_off) * T.pitch + qx + dx0 - T.x_off;
    const float* wp = sW + (i0 * KW + j0) * T.wc + cg * G;
#pragma unroll
    for (int a = 0; a < KH / ST; ++a)
#pragma unroll
      for (int bb = 0; bb < KW / ST; ++bb) {
        const float* ra = rp - a * T.pitch - bb;
        const float* wa = wp + (ST * a * KW + ST * bb) * T.wc;
#pragma unroll 8
        for (int o = 0; o < L.cout; ++o, ra += plane, wa += wstep) {
          const float rv = *ra;
          const float4 w = *reinterpret_cast<const float4*>(wa);
          const float2 rr = make_float2(rv, rv);
          a01 = __ffma2_rn(make_float2(w.x, w.y), rr, a01);
          if (G == 4)
            a23 = __ffma2_rn(make_float2(w.z, w.w), rr, a23);
          else
            a23.x = fmaf(w.z, rv, a23.x);
        }
      }
    const int yy = ry + ST * (q0 + qy), xx = rx + ST * qx;
    const float acc[4] = {a01.x, a01.y, a23.x, a23.y};
#pragma unroll
    for (int g = 0; g < G; ++g) f(cg * G + g, yy, xx, acc[g]);
  }
}

// Place of input element (c, row yy of the tile, padded column xx) in the forward tile.
__device__ __forceinline__ int conv_f_at(const ConvTile& T, int st, int c, int yy, int xx) {
  return (c * T.rows + yy) * T.pitch + (st == 2 ? (xx & 1) * (T.pitch / 2) + (xx >> 1) : xx);
}

// f(channel, y, x, acc) for every output of the band of ny rows from y0: a
// thread takes one output position and GF output channels, one chain of FMAs
// per output in the order (c, i, j).
template <int KH, int KW, int ST, int GF, class F>
__device__ __forceinline__ void conv_f_items(const LayerDev& L, const ConvTile& T, const float* sW, const float* sX,
                                             int y0, int ny, int nt, F f) {
  const int nog = L.cout / GF, items = nog * ny * L.wo, plane = T.rows * T.pitch, half = T.pitch / ST;
  const SharedDiv d_wo = shared_div(L.wo), d_ny = shared_div(ny);
  for (int e = threadIdx.x; e < items; e += nt) {
    const int r = d_wo.of(e), xo = e - r * L.wo;
    const int og = d_ny.of(r), yo = r - og * ny;
    float2 a01 = make_float2(0.f, 0.f), a23 = a01;  // channel pairs, as above
    const float* xc = sX + yo * ST * T.pitch + xo;
    const float* wc = sW + og * GF;
#pragma unroll 2
    for (int c = 0; c < L.cin; ++c, xc += plane) {
      const float* xr = xc;
#pragma unroll
      for (int i = 0; i < KH; ++i, xr += T.pitch)
#pragma unroll
        for (int j = 0; j < KW; ++j, wc += L.cout) {
          const float xv = (j % ST ? xr + half : xr)[j / ST];
          if (GF == 4) {
            const float4 w4 = *reinterpret_cast<const float4*>(wc);
            a01 = __ffma2_rn(make_float2(w4.x, w4.y), make_float2(xv, xv), a01);
            a23 = __ffma2_rn(make_float2(w4.z, w4.w), make_float2(xv, xv), a23);
          } else {
            const float2 w2 = *reinterpret_cast<const float2*>(wc);
            a01 = __ffma2_rn(w2, make_float2(xv, xv), a01);
          }
        }
    }
    const float acc[4] = {a01.x, a01.y, a23.x, a23.y};
#pragma unroll
    for (int g = 0; g < GF; ++g) f(og * GF + g, y0 + yo, xo, acc[g]);
  }
}

// 1: 4x4 stride 2, 2: 3x3 stride 1 (the blocked passes), 0: other geometries.
inline int conv_geo(const LayerDev& L) {
  if (L.kh == 4 && L.kw == 4 && L.stride == 2) return 1;
  if (L.kh == 3 && L.kw == 3 && L.stride == 1) return 2;
  return 0;
}
// Whether the blocked transposed / forward pass covers the layer.
inline bool conv_t_covers(const LayerDev& L) {
  return L.kind == LD_LAYER_CONV && conv_geo(L) && L.h % L.stride == 0 && L.w % L.stride == 0 && L.Wt &&
         (L.cin % 4 == 0 || L.cin == 3);
}
inline bool conv_f_covers(const LayerDev& L) {
  return L.kind == LD_LAYER_CONV && conv_geo(L) && L.Wf && L.cout % 2 == 0;
}

// Tiles of the transposed / forward pass with bands of bh rows (bh <= 0: the
// fixed part only).
inline ConvTile conv_t_tile(const LayerDev& L, int bh) {
  const int st = L.stride, dlo = L.pad / st - (L.kh / st - 1), dhi = (st - 1 + L.pad) / st;
  ConvTile T{};
  // rows / columns of r around a position's own: taps reach dy0 - (k/s - 1) .. dy0
  T.wc = (L.cin + 3) & ~3;
  T.w_floats = L.cout * L.kh * L.kw * T.wc;
  T.y_off = T.x_off = dlo;
  T.pitch = L.w / st + dhi - dlo;
  T.bh = bh;
  T.rows = bh + dhi - dlo;
  T.bands = bh > 0 ? (L.h / st + bh - 1) / bh : 0;
  T.smem = sizeof(float) * ((size_t)T.w_floats + (size_t)L.cout * T.rows * T.pitch);
  return T;
}
inline ConvTile conv_f_tile(const LayerDev& L, int bh) {
  const int st = L.stride;
  ConvTile T{};
  T.w_floats = (L.cout * L.cin * L.kh * L.kw + 3) & ~3;
  T.y_off = T.x_off = -L.pad;
  T.pitch = ((L.wo - 1) * st + L.kw + st - 1) / st * st;
  T.bh = bh;
  T.rows = bh * st + L.kh - st;
  T.bands = bh > 0 ? (L.ho + bh - 1) / bh : 0;
  T.smem = sizeof(float) * ((size_t)T.w_floats + (size_t)L.cin * T.rows * T.pitch);
  return T;
}

}  // namespace
}  // namespace ld
