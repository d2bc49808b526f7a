// Float-float Dslash, two warps per 32 sites (one per upper spin), hops in loops.
//
// A float-float multiply-add is 12 FP32 instructions, so the eight hops of a
// site unrolled are some 11,000 instructions (180 KB): the kernel that did so
// was 29% issue-active and its warps spent 5 of 6 stalled cycles waiting for
// instructions.  Here one hop body per kind of phase (see fx_hop, dslash_fx.cuh,
// for the spin structure and the split) is looped over the hops' direction and
// the pairs (x, y), (z, t), with the signs, the adjoint and the time boundary as
// run-time factors.  24^3 x 48, 8 systems: 2.50 ms against 5.49 ms; 4^4, 16 systems:
// 17 against 34 us.  Error against complex128 3.1e-15 (was 3.4e-15; with the sums
// of the hops left unnormalised 2.35 ms, but 3.8e-15).
#pragma once

#include "dslash.cuh"

namespace tml {

// a b as an unnormalised pair (exact product of the high parts, cross terms)
__device__ __forceinline__ FF ff_prod(FF a, FF b) {
  const float p = __fmul_rn(a.hi, b.hi);
  float e = __fmaf_rn(a.hi, b.hi, -p);
  e = __fmaf_rn(a.hi, b.lo, e);
  return {p, __fmaf_rn(a.lo, b.hi, e)};
}
// a + s b, s = +-1
__device__ __forceinline__ FF ff_acc(FF a, FF b, float s) { return a + FF{__fmul_rn(s, b.hi), __fmul_rn(s, b.lo)}; }

struct FfSum {
  Cx<FF> up[3], lo[3];
};

// up += w, lo += sf w with w = W h, h = sw (psi_s + sg i^(ODD) psi_{2 + ac}); W = U, or
// U^dag with adj
template <bool ODD>
__device__ __forceinline__ void ff_hop(FfSum& s, const float4* up, const float4* dn, const float4* u, size_t cs,
                                       bool adj, float sg, float sw, float sf) {
  Cx<FF> h[3], m[9];
#pragma unroll
  for (int j = 0; j < 9; ++j) {
    const float4 q = u[(adj ? 3 * (j % 3) + j / 3 : j) * cs];
    m[j] = {FF{q.x, q.y}, adj ? FF{-q.z, -q.w} : FF{q.z, q.w}};
  }
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    const float4 p = up[c * cs], q = dn[c * cs];
    const FF pr = {sw * p.x, sw * p.y}, pi = {sw * p.z, sw * p.w};
    const FF qr = {sg * q.x, sg * q.y}, qi = {sg * q.z, sg * q.w};
    if constexpr (ODD) h[c] = {pr - qi, pi + qr};
    else h[c] = {pr + qr, pi + qi};
  }
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    FF zr = ff_prod(m[3 * a].re, h[0].re), zi = ff_prod(m[3 * a].re, h[0].im);
    zr = ff_fma(-m[3 * a].im, h[0].im, zr);
    zi = ff_fma(m[3 * a].im, h[0].re, zi);
#pragma unroll
    for (int b = 1; b < 3; ++b) {
      const Cx<FF> y = m[3 * a + b];
      zr = ff_fma(y.re, h[b].re, zr);
      zr = ff_fma(-y.im, h[b].im, zr);
      zi = ff_fma(y.re, h[b].im, zi);
      zi = ff_fma(y.im, h[b].re, zi);
    }
    zr = ff_norm(zr);
    zi = ff_norm(zi);
    s.up[a] = {ff_acc(s.up[a].re, zr, 1.0f), ff_acc(s.up[a].im, zi, 1.0f)};
    s.lo[a] = {ff_acc(s.lo[a].re, zr, sf), ff_acc(s.lo[a].im, zi, sf)};
  }
}

// the epilogue (dslash_epilogue) of the components of spins sp and 2 + sp;
// returns their |.|^2
template <int EPI>
__device__ __forceinline__ double ff_epilogue(const DslashArgs& a, int sp, int r, int par, int cb,
                                              const Cx<FF> (&acc)[6]) {
  using O = Ar<FF>;
  const EpiConsts<FF> k = epi_consts<FF>(a);
  const size_t cs = (size_t)a.g.Vh;
  const size_t b0 = ((size_t)(r * 2 + par) * 12 + 3 * sp) * cs + cb;  // chunk q: + (q < 3 ? q : q + 3) cs
  const float4* cf = reinterpret_cast<const float4*>(k.cfield) + b0;
  float4* out = reinterpret_cast<float4*>(a.c.out) + b0;
  const float4* bf = reinterpret_cast<const float4*>(a.c.b) + b0;
  FF part = 0;
#pragma unroll
  for (int q = 0; q < 6; ++q) {
    const size_t i = (q < 3 ? q : q + 3) * cs;
    const FF tw = q < 3 ? k.nu : -k.nu;  // gamma_5 = diag(1, 1, -1, -1)
    Cx<FF> o;
    if (a.c.centre != 0) {
      const float4 c = cf[i];
      o = {FF{c.x, c.y}, FF{c.z, c.w}};
      if (a.c.centre == 2) o = {O::fma(-tw, o.im, o.re), O::fma(tw, o.re, o.im)};
      o = {O::fma(k.shop, acc[q].re, o.re), O::fma(k.shop, acc[q].im, o.im)};
    } else {
      o = {O::mul(k.shop, acc[q].re), O::mul(k.shop, acc[q].im)};
    }
    o = {O::norm(o.re), O::norm(o.im)};
    if (a.c.out_inv) {
      const Cx<FF> v = o;
      o = {O::mul(k.inv, O::norm(O::fma(tw, v.im, v.re))), O::mul(k.inv, O::norm(O::fma(-tw, v.re, v.im)))};
    }
    if constexpr (EPI == EPI_RESID) {
      const float4 b = bf[i];
      o = {O::sub(FF{b.x, b.y}, o.re), O::sub(FF{b.z, b.w}, o.im)};
    } else if (q >= 3 && a.c.g5_out) {
      o = {-o.re, -o.im};
    }
    const FF re = ff_norm(o.re), im = ff_norm(o.im);
    out[i] = make_float4(re.hi, re.lo, im.hi, im.lo);
    if (EPI == EPI_RESID || a.c.partial) part = O::fma(o.re, o.re, O::fma(o.im, o.im, part));
  }
  return (double)part;
}

template <bool DAG, int EPI>
__global__ void __launch_bounds__(128, 4) dslash_ff_kernel(const DslashArgs a, int lgs) {
  __shared__ float4 xch[4][3][32];
  __shared__ double xsum[4];
  const Geom& g = a.g;
  const int rg = blockIdx.x % a.rhs_groups;
  const int sb = blockIdx.x / a.rhs_groups;
  const int par = a.c.parity < 0 ? (sb & 1) : a.c.parity;
  const int gb = a.c.parity < 0 ? (sb >> 1) : sb;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int sp = warp & 1, pair = warp >> 1;
  const int grp = gb * (int)(blockDim.x >> (6 + lgs)) + (pair >> lgs);  // 32-site group
  const int cb = grp * 32 + lane;
  const int r = (rg << lgs) + (pair & ((1 << lgs) - 1));
  const int nrhs = a.c.nrhs;
  const bool act = r < nrhs && (a.c.active == nullptr || a.c.active[r] != 0) && cb < g.Vh;
  if (a.trace_count && blockIdx.x == 0 && threadIdx.x == 0) {
    int n = 0;
    for (int q = 0; q < nrhs; ++q) n += (a.c.active == nullptr || a.c.active[q] != 0) ? 1 : 0;
    *a.trace_count = n;
  }
  constexpr float SF = DAG ? 1.0f : -1.0f;
  FfSum t;
  if (act) {
    const Site s = site_of(g, par, cb);
    const int opar = par ^ 1;
    const size_t cs = (size_t)g.Vh;
    const float4* fup = reinterpret_cast<const float4*>(a.c.in) + ((size_t)(r * 2 + opar) * 12 + 3 * sp) * cs;
    const float4* links = reinterpret_cast<const float4*>(a.links);
#pragma unroll
    for (int c = 0; c < 3; ++c) t.up[c] = {FF(0.0f), FF(0.0f)};
#pragma unroll 1
    for (int it = 0; it < 2; ++it) {
      const float4* fdn = fup + (6 + 3 * (it ? 0 : 1 - 2 * sp)) * (ptrdiff_t)cs;
      const float so = it && sp ? -1.0f : 1.0f, se = it || sp ? 1.0f : -1.0f;  // phase signs: i^ak = so i, se
#pragma unroll
      for (int c = 0; c < 3; ++c) t.lo[c] = {FF(0.0f), FF(0.0f)};
#pragma unroll 1
      for (int back = 0; back < 2; ++back) {
        const int c = it ? s.c[2] : s.c[0], L = it ? g.L[2] : g.L[0], st = it ? g.stride[2] : 1;
        const int step = back ? (c > 0 ? -st : (L - 1) * st) : (c + 1 < L ? st : -(L - 1) * st);
        const int n = (s.lex + step) >> 1;
        const float sb = back ? -1.0f : 1.0f;
        ff_hop<true>(t, fup + n, fdn + n, links + (size_t)(4 * it + (back ? opar : par)) * 9 * cs + (back ? n : cb),
                     cs, back != 0, SF * so * sb, 1.0f, sb);
      }
      // lower row: SF (-so i (w_f - w_b)_odd + se (w_f - w_b)_even); the sums are
      // kept as the bracket times se
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        const Cx<FF> v = t.lo[c];
        const float f = so * se;
        t.lo[c] = {FF{f * v.im.hi, f * v.im.lo}, FF{-f * v.re.hi, -f * v.re.lo}};
      }
#pragma unroll 1
      for (int back = 0; back < 2; ++back) {
        const int c = it ? s.c[3] : s.c[1], L = it ? g.L[3] : g.L[1], st = it ? g.stride[3] : g.stride[1];
        const bool wrap = back ? c == 0 : c + 1 == L;
        const int n = (s.lex + (back ? (wrap ? (L - 1) * st : -st) : (wrap ? -(L - 1) * st : st))) >> 1;
        const float sb = back ? -1.0f : 1.0f, sw = it && g.antiperiodic && wrap ? -1.0f : 1.0f;
        ff_hop<false>(t, fup + n, fdn + n,
                      links + (size_t)(4 * it + 2 + (back ? opar : par)) * 9 * cs + (back ? n : cb), cs, back != 0,
                      SF * se * sb * sw, sw, sb);
      }
      if (it == 0) {  // row 1 - sp
#pragma unroll
        for (int c = 0; c < 3; ++c)
          xch[warp][c][lane] = make_float4(se * t.lo[c].re.hi, se * t.lo[c].re.lo, se * t.lo[c].im.hi, se * t.lo[c].im.lo);
      }
    }
  }
  __syncthreads();
  double part = 0.0;
  if (act) {
    Cx<FF> acc[6];
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      const float4 o = xch[warp ^ 1][c][lane];
      acc[c] = t.up[c];
      const FF re = t.lo[c].re + FF{o.x, o.y}, im = t.lo[c].im + FF{o.z, o.w};
      acc[3 + c] = {FF{SF * re.hi, SF * re.lo}, FF{SF * im.hi, SF * im.lo}};
    }
    part = ff_epilogue<EPI>(a, sp, r, par, cb, acc);
  }
  if (EPI != EPI_OUT || a.c.partial != nullptr) {
    const double ps = warp_sum(part);
    if (lane == 0) xsum[warp] = ps;
    __syncthreads();
    if (lane == 0 && sp == 0 && r < nrhs && grp < a.nwarp)
      a.c.partial[((size_t)r * 2 + par) * a.nwarp + grp] = xsum[warp] + xsum[warp + 1];
  }
}

}  // namespace tml
