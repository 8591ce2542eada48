// Kernels on the right-hand-side-paired FP32 layout (see pair32.cuh): packing from and
// to the canonical layout, and H_W.
#include <algorithm>

#include "pair32.cuh"

namespace {

// canonical complex64 [rhs][site][12] -> pairs; a missing partner of an odd count is 0.  One
// 32-site tile of a pair at a time through shared memory (as pack_kernel).
constexpr int kTileNT = 384;
constexpr int kTileRow = 13;
__global__ void __launch_bounds__(kTileNT) pack_pair_f32_kernel(const float2* __restrict__ aos, float4* __restrict__ pr,
                                                                int V, int nrhs, size_t ntiles) {
  __shared__ float2 sh[2][32 * kTileRow];
  const int t = threadIdx.x, nt = (V + 31) / 32;
  for (size_t b = blockIdx.x; b < ntiles; b += gridDim.x) {
    const size_t pq = b / nt, s0 = b % nt * 32, r0 = 2 * pq;
    if (s0 + t / 12 < V) {
      const int o = t / 12 * kTileRow + t % 12;
      sh[0][o] = aos[(r0 * V + s0) * 12 + t];
      sh[1][o] = r0 + 1 < nrhs ? aos[((r0 + 1) * V + s0) * 12 + t] : make_float2(0.f, 0.f);
    }
    __syncthreads();
    const size_t s = s0 + t % 32;
    if (s < V) {
      const int o = t % 32 * kTileRow + t / 32;
      const float2 x = sh[0][o], y = sh[1][o];
      pr[(pq * 12 + t / 32) * V + s] = make_float4(x.x, y.x, x.y, y.y);
    }
    __syncthreads();
  }
}

// H_W on the paired layout with 12-real links; the result goes to the canonical layout, one
// right-hand side of the pair at a time through shared memory (16^3 x 32, 12 right-hand sides,
// whole call: 283 -> 150 us; packing 52 us where the strided writes took about 100, the
// stencil 100 us where it and a strided unpacking pass took 190).  grid: x = pair, y = block of
// sites.  At most 128 registers (4 blocks of 128 threads per SM): 12 accumulator pairs, the
// half spinor and the rebuilt link are live together.  The diagonal term is read before
// the hops, so that the x and y neighbours, which share its cache lines, follow it
// through L1.
template <int LK, int NT>
__global__ void __launch_bounds__(NT, 512 / NT) hw_pair12_kernel(const float4* __restrict__ in,
                                                                 float2* __restrict__ out,
                                                                 const float4* __restrict__ L, Geom g, float diag,
                                                                 int nrhs) {
  __shared__ float2 sh[NT * kTileRow];
  const int s0 = blockIdx.y * NT, s = s0 + threadIdx.x, V = g.V;
  P2 o[12];
  if (s < V) {
    int c[4];
    site_coords(g, s, c);
    const float4* inq = in + (size_t)blockIdx.x * 12 * V;
    const float2 d2 = f2(diag, diag), nd2 = f2(-diag, -diag);
#pragma unroll
    for (int k = 0; k < 12; ++k) {
      const P2 v = ldp(inq + k * (size_t)V + s);
      const float2 d = k < 6 ? d2 : nd2;  // lower spins: gamma5 = -1, accumulated negated
      o[k] = {mul2(d, v.re), mul2(d, v.im)};
    }
    hop_pair12<0, LK>(inq, L, g, s, c, o);
    hop_pair12<1, LK>(inq, L, g, s, c, o);
    hop_pair12<2, LK>(inq, L, g, s, c, o);
    hop_pair12<3, LK>(inq, L, g, s, c, o);
  }
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    const int r = 2 * blockIdx.x + h;
    if (r >= nrhs) break;
    if (h > 0) __syncthreads();
    if (s < V)
#pragma unroll
      for (int k = 0; k < 12; ++k)
        sh[threadIdx.x * kTileRow + k] = h == 0 ? f2(o[k].re.x, o[k].im.x) : f2(o[k].re.y, o[k].im.y);
    __syncthreads();
    float2* po = out + ((size_t)r * V + s0) * 12;
    const int n = min(NT, V - s0) * 12;
    for (int e = threadIdx.x; e < n; e += NT) po[e] = sh[e / 12 * kTileRow + e % 12];
  }
}

}  // namespace

int launch_pack_pair32(ov_ctx* ctx, const float2* aos, float4* pr, int nrhs, cudaStream_t s) {
  const size_t n = (size_t)((nrhs + 1) / 2) * ((ctx->g.V + 31) / 32);
  cudaEvent_t ev;
  kt_begin(ctx, KC_LAYOUT, s, &ev);
  pack_pair_f32_kernel<<<(unsigned)std::min<size_t>(n, 152 * 64), kTileNT, 0, s>>>(aos, pr, ctx->g.V, nrhs, n);
  kt_end(ctx, KC_LAYOUT, s, ev);
  OV_CHECK_LAUNCH(ctx, "pack_pair_f32_kernel");
  return OV_OK;
}

// form 2: compact 12-real links (the spin-paired layout's 3 float4 per link, 48 B), the
// centre read first, 128 threads per block; form 6: the same with row 2 rebuilt once in
// scalar arithmetic.
int launch_hw_pair12(ov_ctx* ctx, const float4* in, float2* out, int nrhs, int form, cudaStream_t s) {
  int st = OV_OK;
  const float4* L = s4_links(ctx, s, &st);
  if (st != OV_OK) return st;
  constexpr int NT = 128;
  dim3 grid((nrhs + 1) / 2, (ctx->g.V + NT - 1) / NT);
  const float diag = (float)(4.0 - ctx->m0);
  cudaEvent_t ev;
  kt_begin(ctx, KC_DSLASH, s, &ev);
  if (form == 6)
    hw_pair12_kernel<3, NT><<<grid, NT, 0, s>>>(in, out, L, ctx->g, diag, nrhs);
  else
    hw_pair12_kernel<1, NT><<<grid, NT, 0, s>>>(in, out, L, ctx->g, diag, nrhs);
  kt_end(ctx, KC_DSLASH, s, ev);
  OV_CHECK_LAUNCH(ctx, "hw_pair12_kernel");
  return OV_OK;
}
