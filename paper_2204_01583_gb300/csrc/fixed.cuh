// Fixed-point vectors and the H_W stencil on them.
//
// GB300 issues one FP64 warp instruction per 16 cycles and SM, but one 32 x 32 + 64 bit
// integer multiply-add (IMAD.WIDE) per cycle; a product of two 58-bit numbers costs three of
// those, so a complex 3 x 3 product takes a seventh of its FP64 time.  A Lanczos vector is
// therefore kept as integers of one scale per vector,
//
//     x = hi 2^30 + lo,   lo in [-2^29, 2^29),   |x| <= 2^58,
//
// the largest component just below 2^58 (a power-of-two scale chosen anew for every vector),
// links as integers of unit 2^-58 (carrying the hop factor -1/2 and the time boundary sign).
// Products drop lo * lo only (2^-60 of the full scale), all sums are exact, and one rounding to
// nearest ends each hop: errors of a few 2^-58 of the vector's largest component, zeros exact.
// FP64 rounds every partial sum at 2^-53 of its own size: more where components are of one
// size, less far below the largest.  In norm, S_N b of point and Gaussian sources (8^4 to
// 16^3 x 32) is within 0.7e-15 to 1.1e-15 of FP64 vectors, as two FP64 forms are of one another.
//
// Bounds, for links whose rows and columns have norm at most 1 (kFxRowMax) and
// |4 - m0| <= 4: the real and imaginary parts of a projected component and their sum fit 31
// bits (hi) and 32 bits (lo); a row's cross terms are below 2^62.3; H_W / 4 is at most
// (19.6 + 4) / 4 = 5.9 times the largest component.  The Lanczos coefficients: gam (of X_{i-1})
// is below 2 by the choice of the shift q; a = <X, w> / <X, X> is at most ||H_W|| / 4 <=
// (4 + 4 ||U||) / 4, and ||U|| <= 1.733, the Frobenius norm of such a link (all entries
// 1 / sqrt(3) reach it): |a| <= 2.74, kept in units of 2^-59.  The terms together are at most
// 5.9 + 2 + 2.74 times the largest component, so that every sum stays below 2^62.
#pragma once

#include "common.cuh"

struct FX {
  int hi, lo;
};
template <>
struct Store<FX> {
  using T = int4;  // (re.hi, re.lo, im.hi, im.lo)
};

constexpr int kFxBits = 58;           // vectors: |x| <= 2^58
constexpr double kFxRowMax = 1.0009;  // largest squared norm of a link row or column
// ... and the smallest: products of shorter links are small against the unit that they are
// rounded to (H_W b with m0 = 4, no diagonal term, and 0.3 / 0.01 / 1e-6 of an SU(3) field: off by
// 2.0e-16, 3.9e-15, 3.9e-11; by 1.6e-16 with the whole one)
constexpr double kFxRowMin = 0.25;
constexpr double kFxDiagMax = 4.0;    // largest |4 - m0|

__host__ __device__ __forceinline__ FX fx_split(long long v) {
  // lo: the low 30 bits, sign-extended; hi: the exact rest
  const int lo = (int)((unsigned)v << 2) >> 2;
  return FX{(int)((v - lo) >> 30), lo};
}

// (hh, x) += a b in units of 2^60 and 2^30 (the lo * lo term, below 2^-2, is dropped)
__device__ __forceinline__ void fx_mac(long long& hh, long long& x, int ah, int al, int bh, int bl) {
  hh += (long long)ah * bh;
  x += (long long)ah * bl;
  x += (long long)al * bh;
}
// shifts by less than 32
__device__ __forceinline__ long long fx_shl(long long v, int k) {
  const unsigned lo = (unsigned)v, hi = (unsigned)(v >> 32);
  return (long long)(((unsigned long long)__funnelshift_l(lo, hi, k) << 32) | (lo << k));
}
__device__ __forceinline__ long long fx_shr(long long v, int k) {
  const unsigned lo = (unsigned)v;
  const int hi = (int)(v >> 32);
  return (long long)(((unsigned long long)(unsigned)(hi >> k) << 32) | __funnelshift_r(lo, (unsigned)hi, k));
}
// arithmetic shift right by any k >= 0 (62 at most: the sign is left), in two steps
struct FxShift {
  int a, b;
};
__device__ __forceinline__ FxShift fx_shift(int k) { return {min(k, 31), min(max(k - 31, 0), 31)}; }
__device__ __forceinline__ long long fx_sar(long long v, FxShift k) { return fx_shr(fx_shr(v, k.a), k.b); }
__device__ __forceinline__ long long fx_value(long long hh, long long x) { return hh + (x >> 30); }
constexpr long long kFxHalf30 = 1LL << 29;  // added to x before that shift: rounds to nearest

// The spin projection of a warp's direction and spin, as a selection and sign masks (one
// instruction stream for all warps; as eight predicated cases it took as many instructions
// as a row product):  h = psi_spin + S f q, q the lower component that A_mu maps to this
// spin, f = 1, -1, i, -i:
//   A_x psi_lo = (-i p3, -i p2), A_y psi_lo = (-p3, p2), A_z psi_lo = (-i p2, i p3), A_t = 1,
// S = -1 forward, S = +1 and conjugated backward.  On the (hi, lo) parts without carry:
// |hi| <= 2^29, |lo| <= 2^30.
struct FxProj {
  int lower;       // component of q, and the lower spin that d = u_b - u_f of this spin feeds
  bool swap;       // f = +-i
  int re[2], im;   // 0 or -1: negate q's contribution to re (forward, backward), to im
  int dre, dim;    // 0 or -1: negate the parts of gamma5 A_mu^dag d (after the swap)
};
__device__ __forceinline__ FxProj fx_projection(int mu, int spin) {
  FxProj f;
  f.lower = mu < 2 ? 3 - spin : 2 + spin;
  f.swap = (mu & 1) == 0 && mu < 3;
  const bool neg = mu == 0 || ((mu == 1 || mu == 2) && spin == 0);  // f = -1 or -i
  const bool pr = f.swap ? neg : !neg, pi = !neg;                   // signs of f q: re, im
  f.re[0] = pr ? -1 : 0;
  f.re[1] = ~f.re[0];
  f.im = pi ? -1 : 0;
  // -conj(f) d from (d_re, -d_im): 1: (-d_re, -d_im), -1: (d_re, d_im), i: (-d_im, d_re),
  // -i: (d_im, -d_re)
  f.dre = neg == f.swap ? -1 : 0;
  f.dim = neg ? -1 : 0;
  return f;
}
// v or -v; without EXACT -v - 1
template <bool EXACT>
__device__ __forceinline__ long long fx_neg(long long v, int mask) {
  return EXACT ? (v ^ (long long)mask) - (long long)mask : v ^ (long long)mask;
}

template <int DIR>
__device__ __forceinline__ int4 fx_project(const FxProj& f, int4 p, int4 q) {
  const int ah = f.swap ? q.z : q.x, al = f.swap ? q.w : q.y, bh = f.swap ? q.x : q.z, bl = f.swap ? q.y : q.w;
  const int mr = f.re[DIR], mi = f.im;
  return make_int4(p.x + (ah ^ mr) - mr, p.y + (al ^ mr) - mr, (DIR ? -p.z : p.z) + (bh ^ mi) - mi,
                   (DIR ? -p.w : p.w) + (bl ^ mi) - mi);
}

// Fields of n planes are stored in tiles of 32 consecutive sites: element (k, site) at
// ((site / 32) n + k) 32 + site % 32, so that all components of a site lie at constant
// distances (one address per neighbour; with whole-lattice planes the address arithmetic of 30
// loads took as many instructions as a row product).  The last tile is padded, and the
// padding of a vector is 0.  (Boxes of 4 x 2 x 2 x 2 sites as tiles, with more neighbours in
// the tile's own cache lines, were 3% slower: loads in flight are not shared through L1.)
constexpr int kFxTile = 32;
__host__ __device__ __forceinline__ size_t fx_index(int site, int n) {
  return (size_t)(site >> 5) * (size_t)(n * kFxTile) + (site & 31);
}
__host__ __device__ __forceinline__ size_t fx_padded(size_t v) { return (v + kFxTile - 1) / kFxTile * kFxTile; }

// the neighbours of a site in direction mu
struct FxHops {
  int fwd, bwd;
};
__device__ __forceinline__ FxHops fx_hops(const Geom& g, int s, int mu) {
  const int n = g.L[mu], st = g.st[mu];
  const int q = fast_div(s, g.dst[mu]), c = q - fast_div(q, g.dL[mu]) * n;  // coordinate
  return {c + 1 == n ? s - c * st : s + st, c == 0 ? s + (n - 1) * st : s - st};
}

// Phase 1 of the stencil: a block of 8 warps takes 32 sites, warp 2 mu + spin both hops of
// direction mu for one spin of the half spinor (a whole half spinor per thread needs twice
// the registers, and with half the warps the loads' latency is not covered).  One instruction
// stream serves all warps: eight unrolled hop bodies overflowed the instruction cache.
// The backward hop U^dag h is the conjugate of U^T conj(h), so both hops are the same
// products.  The direction's partials, component by component of gamma5 H_hop x in units of
// the vector / 4 (factor -1/2 in the links): u_f + u_b for the upper spin, -A_mu^dag (u_b -
// u_f) for the lower one.
constexpr int kFxNT = 256;
// Products are rounded to nearest and exact zeros stay: a point source's empty components
// would otherwise collect units of its one large component in every step.
// SCALED (fields with a scale per site, ov_apply_HW): u_f and u_b are shifted right by sf and
// sb before their sums.  Without it negations are to -v - 1, and the reader of the sums over the
// directions adds the units (fx_negations): an addition of 64 bits less per direction and component.
template <bool SCALED = false>
__device__ __forceinline__ void fx_phase1(const int4* __restrict__ in, const int4* __restrict__ U, int mu_spin,
                                          int s, const FxHops& nb, longlong2* out, FxShift sf = {0, 0},
                                          FxShift sb = {0, 0}) {
  const int mu = mu_spin >> 1, spin = mu_spin & 1;
  const FxProj f = fx_projection(mu, spin);
  longlong2* lo = out + 3 * f.lower * kFxTile;
  out += 3 * spin * kFxTile;
#pragma unroll
  for (int dir = 0; dir < 2; ++dir) {
    const int4* pu = in + fx_index(dir == 0 ? nb.fwd : nb.bwd, 12) + 3 * spin * kFxTile;
    const int4* pl = pu + 3 * (f.lower - spin) * kFxTile;
    const int4* Ul = U + fx_index(dir == 0 ? s : nb.bwd, 36) + 9 * mu * kFxTile;
    int4 p[3], q[3], l[9], h[3];
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      p[c] = __ldg(pu + c * kFxTile);
      q[c] = __ldg(pl + c * kFxTile);
    }
#pragma unroll
    for (int e = 0; e < 9; ++e) l[dir == 0 ? e : e % 3 * 3 + e / 3] = __ldg(Ul + e * kFxTile);
#pragma unroll
    for (int c = 0; c < 3; ++c) h[c] = dir == 0 ? fx_project<0>(f, p[c], q[c]) : fx_project<1>(f, p[c], q[c]);
    int2 hs[3];  // re + im
#pragma unroll
    for (int c = 0; c < 3; ++c) hs[c] = make_int2(h[c].x + h[c].z, h[c].y + h[c].w);
#pragma unroll
    for (int i = 0; i < 3; ++i) {
      // a complex product from three real ones: re = a - b, im = c - a - b with a = l_re h_re,
      // b = l_im h_im, c = (l_re + l_im)(h_re + h_im): 27 wide multiply-adds per row, not 36
      // (half a unit in ax rounds re, the second one in cx im)
      long long ah = 0, ax = kFxHalf30, bh = 0, bx = 0, ch = 0, cx = 2 * kFxHalf30;
#pragma unroll
      for (int j = 0; j < 3; ++j) {
        const int4 m = l[3 * i + j];
        fx_mac(ah, ax, m.x, m.y, h[j].x, h[j].y);
        fx_mac(bh, bx, m.z, m.w, h[j].z, h[j].w);
        fx_mac(ch, cx, m.x + m.z, m.y + m.w, hs[j].x, hs[j].y);
      }
      longlong2 u = make_longlong2(fx_value(ah - bh, ax - bx), fx_value(ch - ah - bh, cx - ax - bx));
      if (SCALED) {
        u.x = fx_sar(u.x, dir == 0 ? sf : sb);
        u.y = fx_sar(u.y, dir == 0 ? sf : sb);
      }
      longlong2* o = out + i * kFxTile;
      if (dir == 0) {
        *o = u;
      } else {  // u is conj(u_b)
        const longlong2 uf = *o;
        *o = make_longlong2(uf.x + u.x, uf.y - u.y);
        const long long dr = u.x - uf.x, di = u.y + uf.y;  // d_re, -d_im
        lo[i * kFxTile] = make_longlong2(fx_neg<SCALED>(f.swap ? di : dr, f.dre), fx_neg<SCALED>(f.swap ? dr : di, f.dim));
      }
    }
  }
}

// The directions whose partial of component k is a negation (dre, dim of fx_projection; those
// of a lower spin only).
__device__ __forceinline__ int2 fx_negations(int k) {
  return k < 6 ? make_int2(0, 0) : make_int2(k < 9 ? 4 : 2, 2);
}

// Component k of gamma5 times the hopping part of H_W x / 4: the sum of the partials.
__device__ __forceinline__ longlong2 fx_phase2(const longlong2* sm, int k, int lane) {
  constexpr int D = 12 * kFxTile;
  const longlong2* p = sm + k * kFxTile + lane;
  const longlong2 x = p[0], y = p[D], z = p[2 * D], t = p[3 * D];
  const int2 n = fx_negations(k);
  return make_longlong2((x.x + y.x) + (z.x + t.x) + n.x, (x.y + y.y) + (z.y + t.y) + n.y);
}
// The same with the direction's partials shifted right by k0 .. k3.
__device__ __forceinline__ longlong2 fx_phase2_scaled(const longlong2* sm, int k, int lane, FxShift k0, FxShift k1,
                                                      FxShift k2, FxShift k3) {
  constexpr int D = 12 * kFxTile;
  const longlong2* p = sm + k * kFxTile + lane;
  const longlong2 x = p[0], y = p[D], z = p[2 * D], t = p[3 * D];
  return make_longlong2((fx_sar(x.x, k0) + fx_sar(y.x, k1)) + (fx_sar(z.x, k2) + fx_sar(t.x, k3)),
                        (fx_sar(x.y, k0) + fx_sar(y.y, k1)) + (fx_sar(z.y, k2) + fx_sar(t.y, k3)));
}
