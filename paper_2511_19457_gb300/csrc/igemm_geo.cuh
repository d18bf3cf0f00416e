// Tile geometry of the implicit-GEMM kernels (k_igemm.cu, k_onetile.cu).
#pragma once

#include "sparoa_kernels.h"

namespace sparoa {

constexpr int kBM = 128;  // output rows (pixels) of a tile

// Launch geometry copied out of the kernel parameters into registers once:
// reading IgemmArgs fields through a reference is a memory load, and every
// asm statement with a memory clobber would force it again.
struct Geo {
  int conv, M, N, Nimg, H, W, Cp, Ho, Wo, kh, kw, stride, pad, bw, bh, bn, tw, th, Ktot;
};

__device__ __forceinline__ Geo make_geo(const IgemmArgs& a) {
  Geo g;
  g.conv = a.conv; g.M = a.M; g.N = a.N; g.Nimg = a.Nimg; g.H = a.H; g.W = a.W; g.Cp = a.Cp;
  g.Ho = a.Ho; g.Wo = a.Wo; g.kh = a.kh; g.kw = a.kw; g.stride = a.stride; g.pad = a.pad;
  g.bw = a.bw; g.bh = a.bh; g.bn = a.bn; g.tw = a.tw; g.th = a.th; g.Ktot = a.Ktot;
  return g;
}

struct TileGeo {
  int m0, tn0, th0, tw0, n0;
};

__device__ __forceinline__ TileGeo tile_geo(const Geo& p, int t, int nt, int BN) {
  TileGeo g;
  const int mi = nt == 1 ? t : t / nt;
  g.n0 = (t - mi * nt) * BN;
  g.m0 = 0;
  g.tn0 = g.th0 = g.tw0 = 0;
  if (p.conv == 2) {
    const int per_img = p.th * p.tw;
    g.tn0 = (mi / per_img) * p.bn;
    const int rem = mi - (mi / per_img) * per_img;
    g.th0 = (rem / p.tw) * p.bh;
    g.tw0 = (rem - (rem / p.tw) * p.tw) * p.bw;
  } else {
    g.m0 = mi * kBM;
  }
  return g;
}

// Output pixel / row of tile row r and whether it exists.
__device__ __forceinline__ int64_t tile_row(const Geo& p, const TileGeo& g, int r, bool& valid,
                                            int& img, int& oh, int& ow) {
  if (p.conv == 2) {
    // (the tile's extents are powers of two)
    const int lw = 31 - __clz(p.bw), lh = 31 - __clz(p.bh);
    const int wl = r & (p.bw - 1), hl = (r >> lw) & (p.bh - 1), nl = r >> (lw + lh);
    img = g.tn0 + nl;
    oh = g.th0 + hl;
    ow = g.tw0 + wl;
    valid = img < p.Nimg && oh < p.Ho && ow < p.Wo;
    return ((int64_t)img * p.Ho + oh) * p.Wo + ow;
  }
  const int64_t m = (int64_t)g.m0 + r;
  valid = m < p.M;
  if (p.conv == 1) {
    const int hw = p.Ho * p.Wo;
    img = valid ? (int)(m / hw) : 0;
    const int rem = (int)(m - (int64_t)img * hw);
    oh = valid ? rem / p.Wo : 0;
    ow = valid ? rem - oh * p.Wo : 0;
  } else {
    img = oh = ow = 0;
  }
  return m;
}

}  // namespace sparoa
