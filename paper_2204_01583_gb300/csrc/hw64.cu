// H_W on FP64 fields in integer arithmetic (fixed.cuh), for ov_apply_HW and the Lanczos bounds.
//
// Each site of the input has a binary scale of its own: its 12 components become 58-bit
// integers relative to the site's largest one, so that an output component is exact to
// about 2^-57 of the largest component of its site and the eight neighbours (FP64 rounds
// every partial sum at 2^-53), however the magnitude varies over the lattice.  A site with a
// non-finite component among these nine is computed in FP64.
//
// 16^3 x 32, 12 right-hand sides, canonical layout: 2655 -> 761 us (packing 134, stencil 627),
// error against 64-bit values 1.9e-16 -> 1.4e-16; 4^4, one right-hand side: 41 -> 10 us.  The
// stencil is bound by instruction issue (53% of cycles; wide multiply-adds on 53% of theirs).
#include <cmath>

#include "fixed.cuh"

namespace {

constexpr int kExpZero = -(1 << 20);  // scale of a site that is zero
constexpr int kExpBad = 1 << 20;      // of a site with a non-finite component
constexpr int kPackNT = 384;          // one warp per component
constexpr int kRow = 13;              // double2 per site of a tile in shared memory (12, padded)

// v 2^(57 - e) rounded, e >= the exponent of v (biased exponents; 1 for subnormal numbers)
__device__ __forceinline__ FX to_fixed(double v, int e) {
  const long long bits = __double_as_longlong(v);
  const int ev = (int)(bits >> 52) & 0x7ff;
  const int d = e - max(ev, 1);
  long long m = ((bits & 0xfffffffffffffLL) | (ev > 0 ? 1LL << 52 : 0)) << 5;
  m = d == 0 ? m : d < 60 ? (m + (1LL << (d - 1))) >> d : 0;
  return fx_split(bits < 0 ? -m : m);
}

// FP64 spinors (canonical, or planes) -> tiles of integers and the scale of every site:
// component = x 2^scale.
template <bool AOS>
__global__ void __launch_bounds__(kPackNT) hw64_pack_kernel(const double2* __restrict__ in, int4* __restrict__ X,
                                                            int* __restrict__ scale, int V) {
  __shared__ double2 sv[AOS ? kFxTile * kRow : 1];
  __shared__ int sm[12][kFxTile];
  const int lane = threadIdx.x & 31, k = threadIdx.x >> 5, s = blockIdx.x * kFxTile + lane;
  const double2* inr = in + (size_t)blockIdx.y * 12 * V;
  double2 v = make_double2(0.0, 0.0);
  if (AOS) {
    const int e = threadIdx.x, site = blockIdx.x * kFxTile + e / 12;
    sv[e / 12 * kRow + e % 12] = site < V ? inr[(size_t)blockIdx.x * (12 * kFxTile) + e] : v;
    __syncthreads();
    v = sv[lane * kRow + k];
  } else if (s < V) {
    v = inr[(size_t)k * V + s];
  }
  sm[k][lane] = max(__double2hiint(v.x) & 0x7fffffff, __double2hiint(v.y) & 0x7fffffff) |
                ((__double2loint(v.x) | __double2loint(v.y)) != 0);  // nonzero for any nonzero component
  __syncthreads();
  int m = 0;
#pragma unroll
  for (int c = 0; c < 12; ++c) m = max(m, sm[c][lane]);
  const int e = max(m >> 20, 1);
  const bool bad = e == 0x7ff;
  const size_t tile = (size_t)blockIdx.y * gridDim.x + blockIdx.x;
  int4 x = make_int4(0, 0, 0, 0);
  if (!bad) {
    const FX re = to_fixed(v.x, e), im = to_fixed(v.y, e);
    x = make_int4(re.hi, re.lo, im.hi, im.lo);
  }
  X[tile * (12 * kFxTile) + threadIdx.x] = x;
  if (k == 0) scale[tile * kFxTile + lane] = bad ? kExpBad : m == 0 ? kExpZero : e - 1023 - 57;
}

// One component in FP64, for sites next to a non-finite component.
__device__ __noinline__ double2 hw64_component(const double2* in, size_t ks, size_t ss, const double2* U, const Geom& g,
                                               int s, int k, double diag) {
  Cx<double> o[12];
  hw_site<double>(in, U, g, s, diag, o, ks, ss);
  double2 r = make_double2(0.0, 0.0);
  for (int c = 0; c < 12; ++c)
    if (c == k) r = make_double2(o[c].re, o[c].im);
  return r;
}

__device__ __forceinline__ double2 hw64_scale(longlong2 w, int e) {
  // (double) w 2^e; inside the normal range by an addition to the exponent
  const double x = (double)w.x, y = (double)w.y;
  if (e >= -900 && e <= 900) {
    const int a = e << 20;
    return make_double2(__hiloint2double(__double2hiint(x) + (w.x != 0 ? a : 0), __double2loint(x)),
                        __hiloint2double(__double2hiint(y) + (w.y != 0 ? a : 0), __double2loint(y)));
  }
  return make_double2(ldexp(x, e), ldexp(y, e));
}

// out = H_W in: phase 1 as in fx_lanczos_hw_kernel, each direction's partials at the larger
// scale of its two neighbours, phase 2 at the largest of the nine.  3 blocks per SM: 761 us for
// 12 right-hand sides at 16^3 x 32, where 4 (64 registers, spills) take 843 and 2 take 938.  With
// the FP64 path of a non-finite site inside the loop over components, 4 took 783.
template <bool AOS>
__global__ void __launch_bounds__(kFxNT, 3) hw64_fx_kernel(const int4* __restrict__ X, const int* __restrict__ scale,
                                                           const int4* __restrict__ U, const double2* __restrict__ in,
                                                           const double2* __restrict__ U64, double2* __restrict__ out,
                                                           const __grid_constant__ Geom g, FX diag, double diag64,
                                                           int nrhs, int per) {
  __shared__ longlong2 sm[4 * 12 * kFxTile];
  __shared__ int se[4][kFxTile];
  __shared__ double2 so[AOS ? kFxTile * kRow : 1];
  const int V = g.V, nb = (V + kFxTile - 1) / kFxTile, ng = gridDim.x / nb;
  const int tb = blockIdx.x / ng, r0 = blockIdx.x % ng * per;
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, mu = wid >> 1;
  const int s = tb * kFxTile + lane;
  const bool on = s < V;
  const FxHops nbr = fx_hops(g, on ? s : 0, mu);
  for (int r = r0; r < min(nrhs, r0 + per); ++r) {
    const int4* Xr = X + (size_t)r * nb * (12 * kFxTile);
    const int* er = scale + (size_t)r * nb * kFxTile;
    if (on) {
      const int ef = er[nbr.fwd], eb = er[nbr.bwd], e = max(ef, eb);
      if ((wid & 1) == 0) se[mu][lane] = e;
      fx_phase1<true>(Xr, U, wid, s, nbr, sm + mu * 12 * kFxTile + lane, fx_shift(e - ef),
                      fx_shift(e - eb));
    }
    __syncthreads();
    if (on && wid < 6) {  // components 2 wid, 2 wid + 1
      const FX d = wid < 3 ? diag : FX{-diag.hi, -diag.lo};
      const int own = er[s], e0 = se[0][lane], e1 = se[1][lane], e2 = se[2][lane], e3 = se[3][lane];
      const int e = max(max(max(e0, e1), max(e2, e3)), own);
      const FxShift k0 = fx_shift(e - e0), k1 = fx_shift(e - e1), k2 = fx_shift(e - e2), k3 = fx_shift(e - e3);
      const FxShift ko = fx_shift(e - own);
#pragma unroll
      for (int j = 0; j < 2; ++j) {
        const int k = 2 * wid + j;
        const int4 x = __ldg(Xr + fx_index(s, 12) + k * kFxTile);
        longlong2 w = fx_phase2_scaled(sm, k, lane, k0, k1, k2, k3);
        long long hh = 0, xx = kFxHalf30;
        fx_mac(hh, xx, d.hi, d.lo, x.x, x.y);
        w.x += fx_sar(fx_value(hh, xx), ko);
        hh = 0;
        xx = kFxHalf30;
        fx_mac(hh, xx, d.hi, d.lo, x.z, x.w);
        w.y += fx_sar(fx_value(hh, xx), ko);
        const double2 v = hw64_scale(w, e + 2);
        if (AOS)
          so[lane * kRow + k] = v;
        else
          out[((size_t)r * 12 + k) * V + s] = v;
      }
      if (e == kExpBad) {  // overwrites the two components
        const double2* inr = in + (size_t)r * 12 * V;
#pragma unroll 1
        for (int k = 2 * wid; k < 2 * wid + 2; ++k) {
          const double2 v = hw64_component(inr, AOS ? 1 : V, AOS ? 12 : 1, U64, g, s, k, diag64);
          if (AOS)
            so[lane * kRow + k] = v;
          else
            out[((size_t)r * 12 + k) * V + s] = v;
        }
      }
    }
    if (!AOS) {
      __syncthreads();
      continue;
    }
    __syncthreads();
    double2* o = out + ((size_t)r * V + (size_t)tb * kFxTile) * 12;
    for (int e = threadIdx.x; e < 12 * kFxTile; e += kFxNT)
      if (tb * kFxTile + e / 12 < V) o[e] = so[e / 12 * kRow + e % 12];
  }
}

}  // namespace

// Bytes moved per site and right-hand side: 192 + 196 packing, 196 + 192 in the stencil, links
// 576 once per block's right-hand sides.
template <bool AOS>
static int hw64_fx(ov_ctx* ctx, const double2* in, double2* out, int nrhs, cudaStream_t s) {
  const int V = ctx->g.V, nb = (V + kFxTile - 1) / kFxTile;
  int st = OV_OK;
  int4* X = (int4*)ws_get(ctx, "hw.fx", sizeof(int4) * 12 * fx_padded(V) * nrhs, &st);
  int* scale = (int*)ws_get(ctx, "hw.fxe", sizeof(int) * fx_padded(V) * nrhs, &st);
  if (st != OV_OK) return st;
  // as many right-hand sides per block as still fill the GPU (their links come from L1)
  int ng = (nrhs + 5) / 6;
  while (ng < nrhs && (size_t)nb * ng < 4 * 4 * 152) ++ng;
  const int per = (nrhs + ng - 1) / ng;
  const size_t grid = (size_t)nb * ((nrhs + per - 1) / per);
  if (grid > 0x7fffffff || nrhs > 65535) return OV_ERR_INVALID_ARG;  // the caller's FP64 kernels
  cudaEvent_t ev;
  kt_begin(ctx, KC_LAYOUT, s, &ev);
  hw64_pack_kernel<AOS><<<dim3(nb, nrhs), kPackNT, 0, s>>>(in, X, scale, V);
  kt_end(ctx, KC_LAYOUT, s, ev);
  const double diag = 4.0 - ctx->m0;
  kt_begin(ctx, KC_DSLASH, s, &ev);
  hw64_fx_kernel<AOS><<<(unsigned)grid, kFxNT, 0, s>>>(X, scale, ctx->Ufx, in, ctx->U64, out, ctx->g,
                                                       fx_split(std::llrint(std::ldexp(diag, 58))), diag, nrhs, per);
  kt_end(ctx, KC_DSLASH, s, ev);
  OV_CHECK_LAUNCH(ctx, "hw64_fx_kernel");
  return OV_OK;
}

int launch_hw64_fx(ov_ctx* ctx, const double2* in, double2* out, int nrhs, bool canonical, cudaStream_t s) {
  return canonical ? hw64_fx<true>(ctx, in, out, nrhs, s) : hw64_fx<false>(ctx, in, out, nrhs, s);
}
