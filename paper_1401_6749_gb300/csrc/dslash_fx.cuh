// FP64 Dslash with the hopping sum in 64-bit fixed point on the integer pipes.
//
// GB300 multiplies FP64 at 2 multiply-adds per clock and SM, but does 32
// 32 x 32 -> 64-bit integer multiply-adds (IMAD.WIDE) in the same clock.  The
// hopping sum needs no floating point inside one stencil: every site's 24
// reals are added with factors of modulus <= 1, so a fixed point relative to
// the largest of them keeps more bits than FP64 rounding of the partial sums.
//
// With E at least the biased exponent of the largest component met so far (one
// above it where it was raised), a component x enters as F = trunc(x 2^(1080 - E)),
// |F| < 2^58, split into hi 2^29 + lo (both with the sign of x).  A link's part u is
// round(u 2^58) = ghi 2^29 + glo, |glo| <= 2^28 (pack_links_fx, made with the
// operator, which also says which links the fixed point takes).  Spin projections
// are integer sums of the halves and every product F G is three IMAD.WIDE:
//   hh += ghi hi,   md += ghi lo + glo hi        (glo lo, below the unit, is dropped)
// A hop adds T = hh + (md >> 29) in units of 2^(E - 1080), 2^-58 of the bound
// B = 2^(E - 1022) on the components.  |hi| < 2^30 and |lo| < 2^30 after the
// projection.  Rows of a link have norms of at most 1.5, so by Cauchy and Schwarz the
// sums over a row stay below 1.5 sqrt(6) 2^59 (hh, T) and 2^62 (md), and those over
// four hops below 2^63.
//
// The hops of (x, y) and those of (z, t) are summed apart, each pair of
// directions in a unit of its own, and brought to twice the larger unit at the end:
// so two and four warps per 32 sites (dslash_fx_kernel) compute the same bits, and
// a system's result does not depend on how many share the launch.
//
// Error, in units: per hop 2.5 |row| from the inputs (only those below B / 32 lose
// bits), 6 from the dropped products, 1.5 |row| from the links, 1 from the rounding of T
// and the shifts: at most 125 in all, 3.9 B 2^-53, where FP64 arithmetic errs by up
// to some 50 roundings of the terms that it adds.  These may be far below B: one
// colour small against another with links that hardly mix them, or one neighbour far
// larger than the others.  FP64 keeps the digits of such a component and this sum
// would not, so S, the sum of |re w| + |im w| over the hops, w = W h, is added up beside
// it (FxSum::s) and a site where that is less than B / 4 for any spin and colour takes
// FP64 sums instead (fx_sums_f64).  Replayed in integers against extended precision
// (links exp(i eps H), eps = 0 .. 2; Gaussian fields, steep ones, colours of unlike
// size), the rms error is 0.35 to 0.5 of that of FP64 arithmetic in all, and in the
// components with S between B / 4 and B / 2, the worst, 0.5 to 1.2 of it (B / 8 to B / 4: 0.8 to 2).
// Gaussian fields, CG vectors, Z4 sources and solutions of them have S > B / 4 at every
// site.  M at 16^3 x 32 against complex128: 1.1e-16 (FP64 arithmetic 1.36e-16), of which
// the centre and the last rounding are the most.
//
// Components outside 2^-863 .. 2^878 (infinities and NaN among them) send the
// site to the same FP64 sums, so the kernel's range and special values are those of
// the FP64 arithmetic.
//
// The sums T are converted to FP64 once per output component; centre, twist
// and CG update follow in FP64 (fx_epilogue).
#pragma once


namespace tml {

constexpr unsigned kFxMinExp = 160, kFxMaxExp = 1900;  // biased exponents the fixed point takes
constexpr unsigned kFxBad = 0x7fffu;                   // mark of a site that takes FP64 sums

// right shifts, zero / the sign for counts of the width and more
__device__ __forceinline__ unsigned shr32(unsigned v, unsigned n) {
  unsigned r;
  asm("shr.u32 %0, %1, %2;" : "=r"(r) : "r"(v), "r"(n));
  return r;
}
__device__ __forceinline__ unsigned shr64_lo(unsigned long long v, unsigned n) {
  unsigned long long r;
  asm("shr.u64 %0, %1, %2;" : "=l"(r) : "l"(v), "r"(n));
  return (unsigned)r;
}
__device__ __forceinline__ long long shr64_s(long long v, unsigned n) {
  long long r;
  asm("shr.s64 %0, %1, %2;" : "=l"(r) : "l"(v), "r"(n));
  return r;
}

// |x| 2^(1080 - E) truncated, as unsigned halves (hi, lo < 2^29); z: +-1, x's sign
// times that of the mask nm (0 or -1)
__device__ __forceinline__ int3 fx_of(double x, unsigned E, int nm) {
  const int h = __double2hiint(x);
  const unsigned long long m =
      ((unsigned long long)(((unsigned)h & 0xfffffu) | 0x100000u) << 32 | (unsigned)__double2loint(x)) << 5;
  const unsigned sh = E - (((unsigned)h >> 20) & 0x7ffu);
  return make_int3((int)shr64_lo(m, sh + 29), (int)(shr64_lo(m, sh) & 0x1fffffffu), ((h >> 31) ^ nm) | 1);
}

struct Fx {
  int hi, lo;
};

// a + b of two signed halves pairs: the signs are factors of integer FMAs
__device__ __forceinline__ Fx fx_add(int3 a, int3 b) {
  return {b.x * b.z + a.x * a.z, b.y * b.z + a.y * a.z};
}

__device__ __forceinline__ unsigned abs_hi(double x) { return (unsigned)__double2hiint(x) & 0x7fffffffu; }

// 16-byte words of site cb in a plane of 32-site groups [group][rows][32]
__device__ __forceinline__ unsigned fx_row(int cb, int rows) {
  return (unsigned)(cb >> 5) * (unsigned)(32 * rows) + (unsigned)(cb & 31);
}

// Chunks of a neighbour on their way from memory to the lane's own slots: six
// 16-byte words (three of spin s, three of 2 + ac), 32 lanes apart
struct FxStage {
  double2 w[6][32];
};

__device__ __forceinline__ void fx_copy(FxStage& st, int lane, const double2* up, const double2* dn, size_t cs) {
#pragma unroll
  for (int c = 0; c < 6; ++c) {
    const double2* src = c < 3 ? up + c * cs : dn + (c - 3) * cs;
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((unsigned)__cvta_generic_to_shared(&st.w[c][lane])),
                 "l"(src)
                 : "memory");
  }
}
__device__ __forceinline__ void fx_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
// all copies of this thread but those of the last N commits have arrived
template <int N> __device__ __forceinline__ void fx_arrived() {
  asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}

// The spin structure of a hop, (1 + SGN g_mu) W psi, seen from one upper spin s
// of the output: h = psi_s + SGN i^ak psi_{2 + ac}, w = W h is added to spin s and
// SGN i^-ak w to the lower row ac (B_mu A_mu = 1).  In the DeGrand-Rossi basis
// ac = 1 - s for x, y and s for z, t; i^ak is +-i for x, z (ODD) and +-1 for y, t.
// So one body serves (x, y) and (z, t) and both spins with a run-time sign, the
// mask nd (0 or -1) on psi_{2 + ac}.
struct FxSum {
  long long upr[3], upi[3], lor[3], loi[3];
  unsigned s[3];  // sum of |re w| + |im w| over the hops, in units of 2^-26 B
  unsigned E;     // units of 2^(E - 1080)
  unsigned big;   // largest |high word| met
};

__device__ __forceinline__ long long mad_wide(int a, int b, long long c) { return (long long)a * b + c; }

// one hop: up += w, lo += w (forward) or -= w (backward, W = U^dag), w times -1
// with nm = -1; st holds the neighbour's chunks of spin s and 2 + ac, u points at
// its link
template <bool ODD, bool ADJ>
__device__ __forceinline__ void fx_hop(FxSum& s, const FxStage& st, int lane, const int4* u, int nd, int nm) {
  double2 p[3], q[3];
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    p[c] = st.w[c][lane];
    q[c] = st.w[3 + c][lane];
  }
  unsigned big = 0;
#pragma unroll
  for (int c = 0; c < 3; ++c)
    big = max(max(big, max(abs_hi(p[c].x), abs_hi(p[c].y))), max(abs_hi(q[c].x), abs_hi(q[c].y)));
  if (big == 0) {  // zero, or denormals whose high words vanish (out of range)
    unsigned any = 0;
#pragma unroll
    for (int c = 0; c < 3; ++c)
      any |= (unsigned)(__double2loint(p[c].x) | __double2loint(p[c].y) | __double2loint(q[c].x) |
                        __double2loint(q[c].y));
    big = any ? 1u : 0u;
  }
  s.big = max(s.big, big);
  if ((big >> 20) > s.E) {
    const unsigned E = (big >> 20) + 1, d = E - s.E;
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      s.upr[a] = shr64_s(s.upr[a], d);
      s.upi[a] = shr64_s(s.upi[a], d);
      s.lor[a] = shr64_s(s.lor[a], d);
      s.loi[a] = shr64_s(s.loi[a], d);
      s.s[a] = shr32(s.s[a], d);
    }
    s.E = E;
  }
  const unsigned E = s.E;
  Fx hre[3], him[3];
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    if constexpr (ODD) {  // p + i q
      hre[c] = fx_add(fx_of(p[c].x, E, nm), fx_of(q[c].y, E, ~(nd ^ nm)));
      him[c] = fx_add(fx_of(p[c].y, E, nm), fx_of(q[c].x, E, nd ^ nm));
    } else {
      hre[c] = fx_add(fx_of(p[c].x, E, nm), fx_of(q[c].x, E, nd ^ nm));
      him[c] = fx_add(fx_of(p[c].y, E, nm), fx_of(q[c].y, E, nd ^ nm));
    }
  }
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    // re: u.re h.re - u.im h.im,  im: u.re h.im + u.im h.re  (u.im -> -u.im for the adjoint)
    // md starts at half a unit, so that md >> 29 rounds
    long long hr = 0, hi = 0, mr = 1 << 28, mi = 1 << 28;
#pragma unroll
    for (int b = 0; b < 3; ++b) {
      const int4 w = u[(ADJ ? 3 * b + a : 3 * a + b) * 32];  // (re.hi, re.lo, im.hi, im.lo)
      const Fx xr = hre[b], xi = him[b];
      const Fx si = ADJ ? xi : Fx{-xi.hi, -xi.lo}, sr = ADJ ? Fx{-xr.hi, -xr.lo} : xr;
      hr = mad_wide(w.x, xr.hi, hr);
      mr = mad_wide(w.x, xr.lo, mr);
      hi = mad_wide(w.x, xi.hi, hi);
      mi = mad_wide(w.x, xi.lo, mi);
      hr = mad_wide(w.z, si.hi, hr);
      mr = mad_wide(w.y, xr.hi, mr);
      hi = mad_wide(w.z, sr.hi, hi);
      mi = mad_wide(w.y, xi.hi, mi);
      mr = mad_wide(w.z, si.lo, mr);
      mi = mad_wide(w.z, sr.lo, mi);
      mr = mad_wide(w.w, si.hi, mr);
      mi = mad_wide(w.w, sr.hi, mi);
    }
    const long long tr = hr + (mr >> 29), ti = hi + (mi >> 29);
    s.s[a] += (unsigned)abs((int)(tr >> 32)) + (unsigned)abs((int)(ti >> 32));
    s.upr[a] += tr;
    s.upi[a] += ti;
    s.lor[a] += ADJ ? -tr : tr;
    s.loi[a] += ADJ ? -ti : ti;
  }
}

// One hop in FP64 arithmetic, as fx_hop: up += w, lo +- w; sd and sw (+-1) multiply
// psi_{2 + ac} and w
template <bool ODD, bool ADJ>
__device__ __forceinline__ void f64_hop(Cx<double> (&up)[3], Cx<double> (&lo)[3], const double2* pu, const double2* pd,
                                        const double2* u, size_t cs, double sd, double sw) {
  Cx<double> h[3];
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    const double2 p = pu[c * cs], q = pd[c * cs];
    if constexpr (ODD) h[c] = {sw * __fma_rn(-sd, q.y, p.x), sw * __fma_rn(sd, q.x, p.y)};
    else h[c] = {sw * __fma_rn(sd, q.x, p.x), sw * __fma_rn(sd, q.y, p.y)};
  }
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    double zr = 0.0, zi = 0.0;
#pragma unroll
    for (int b = 0; b < 3; ++b) {
      const double2 v = u[(ADJ ? 3 * b + a : 3 * a + b) * cs];
      const double vi = ADJ ? -v.y : v.y;
      zr = __fma_rn(v.x, h[b].re, zr);
      zr = __fma_rn(-vi, h[b].im, zr);
      zi = __fma_rn(v.x, h[b].im, zi);
      zi = __fma_rn(vi, h[b].re, zi);
    }
    up[a] = {__dadd_rn(up[a].re, zr), __dadd_rn(up[a].im, zi)};
    lo[a] = ADJ ? Cx<double>{__dsub_rn(lo[a].re, zr), __dsub_rn(lo[a].im, zi)}
                : Cx<double>{__dadd_rn(lo[a].re, zr), __dadd_rn(lo[a].im, zi)};
  }
}

// the neighbour of s in direction mu (checkerboard index)
__device__ __forceinline__ int fx_nbr(const Geom& g, const Site& s, int mu, bool bwd) {
  const int c = mu & 2 ? (mu & 1 ? s.c[3] : s.c[2]) : (mu & 1 ? s.c[1] : s.c[0]);
  const int L = g.L[mu], st = g.stride[mu];
  return (bwd ? (c > 0 ? s.lex - st : s.lex + (L - 1) * st) : (c + 1 < L ? s.lex + st : s.lex - (L - 1) * st)) >> 1;
}

// The sums of a site in FP64 arithmetic, where the fixed point does not take it:
// out[0..2] of spin sp and out[3..5] of spin 2 + sp, or only one of the two (rows 1: sp, 2:
// 2 + sp, 3: both), by spin and pair of directions as in the kernel.  Not inlined: it is
// rare.  Each warp of the site calls it for its own rows, so half hops are repeated: M of
// a point source's solution, 16^3 x 32, 4 systems, takes 0.86 ms with links exp(0.3 i H)
// and 1.43 with exp(0.1 i H), where almost every warp has such a site (FP64 kernel 0.81, without
// such sites 0.24).  An exchange of the sums through shared memory takes 0.68 and 1.07, but
// cost the solves 2%, by the registers and the code around it; the whole site in
// each warp took 1.02 and 1.73.
static __device__ __noinline__ void fx_sums_f64(Cx<double>* out, const DslashArgs* ap, int r, int par, int cb, int sp,
                                                int rows) {
  const DslashArgs& a = *ap;
  const Geom& g = a.g;
  const Site s = site_of(g, par, cb);
  const int opar = par ^ 1, SF = a.c.dagger ? +1 : -1;
  const size_t cs = (size_t)g.Vh;
  Cx<double> u[3], l[3];
#pragma unroll
  for (int c = 0; c < 3; ++c) u[c] = l[c] = {0.0, 0.0};
  // spin sp over (x, y) and (z, t); over (x, y) the other upper spin, whose lower row is 2 + sp
#pragma unroll 1
  for (int k = 0; k < 3; ++k) {
    if ((k == 0 && !(rows & 1)) || (k == 2 && !(rows & 2))) continue;
    const int h = k == 2 ? sp ^ 1 : sp, it = k == 1;
    const double2* fup = reinterpret_cast<const double2*>(a.c.in) + ((size_t)(r * 2 + opar) * 12 + 3 * h) * cs;
    const double2* fdn = fup + (6 + 3 * (it ? 0 : 1 - 2 * h)) * (ptrdiff_t)cs;
    const double2* uf = reinterpret_cast<const double2*>(a.links) + (size_t)(4 * it + par) * 9 * cs;  // next direction: + 18 cs
    const double2* ub = reinterpret_cast<const double2*>(a.links) + (size_t)(4 * it + opar) * 9 * cs;
    const int so = it && h ? -1 : 1, se = it || h ? 1 : -1;
    const bool edge = it && g.antiperiodic;
    Cx<double> up[3], lo[3];
#pragma unroll
    for (int c = 0; c < 3; ++c) up[c] = lo[c] = {0.0, 0.0};
    int n = fx_nbr(g, s, 2 * it, false);
    f64_hop<true, false>(up, lo, fup + n, fdn + n, uf + cb, cs, SF * so, 1.0);
    n = fx_nbr(g, s, 2 * it, true);
    f64_hop<true, true>(up, lo, fup + n, fdn + n, ub + n, cs, -SF * so, 1.0);
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      const Cx<double> v = lo[c];
      lo[c] = so == se ? Cx<double>{v.im, -v.re} : Cx<double>{-v.im, v.re};
    }
    n = fx_nbr(g, s, 2 * it + 1, false);
    f64_hop<false, false>(up, lo, fup + n, fdn + n, uf + 18 * cs + cb, cs, SF * se,
                          edge && s.c[3] == g.L[3] - 1 ? -1.0 : 1.0);
    n = fx_nbr(g, s, 2 * it + 1, true);
    f64_hop<false, true>(up, lo, fup + n, fdn + n, ub + 18 * cs + n, cs, -SF * se, edge && s.c[3] == 0 ? -1.0 : 1.0);
    const double f = se * SF;
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      if (k < 2) u[c] = {__dadd_rn(u[c].re, up[c].re), __dadd_rn(u[c].im, up[c].im)};
      if (k > 0) l[c] = {__fma_rn(f, lo[c].re, l[c].re), __fma_rn(f, lo[c].im, l[c].im)};
    }
  }
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    out[c] = u[c];
    out[3 + c] = l[c];
  }
}

// The FP64 epilogue (dslash_epilogue) of spin sp0 (acc[0..2]) and, with NC = 6,
// spin sp0 + 2 (acc[3..5]); acc the hopping sums in units of `unit`.  Returns
// their |.|^2.
template <int EPI, int CENTRE, bool INV, int NC>
__device__ __forceinline__ double fx_epilogue(const DslashArgs& a, int sp0, int r, int par, int cb, double unit,
                                              const Cx<double> (&acc)[NC]) {
  const size_t cs = (size_t)a.g.Vh;
  const size_t b0 = ((size_t)(r * 2 + par) * 12 + 3 * sp0) * cs + cb;  // chunk q: + (q < 3 ? q : q + 3) cs
  const double nu = sp0 < 2 ? a.nu : -a.nu, inv = a.inv;
  const double shop = CENTRE == 0 && INV ? a.hop_scale * unit * inv : a.hop_scale * unit;
  Cx<double> o[NC];
#pragma unroll
  for (int q = 0; q < NC; ++q) {
    const double tw = q < 3 ? nu : -nu;  // gamma_5 = diag(1, 1, -1, -1)
    const Cx<double> v = acc[q];
    if constexpr (CENTRE != 0) {
      const double2 c = reinterpret_cast<const double2*>(a.c.cfield ? a.c.cfield : a.c.in)[b0 + (q < 3 ? q : q + 3) * cs];
      o[q] = {c.x, c.y};
      if constexpr (CENTRE == 2) o[q] = {__fma_rn(-tw, c.y, c.x), __fma_rn(tw, c.x, c.y)};
      o[q] = {__fma_rn(shop, v.re, o[q].re), __fma_rn(shop, v.im, o[q].im)};
      if constexpr (INV) o[q] = {inv * __fma_rn(tw, o[q].im, o[q].re), inv * __fma_rn(-tw, o[q].re, o[q].im)};
    } else if constexpr (INV) {  // A^-1 s_hop h = (s_hop / (1 + nu^2)) (h - i nu g5 h)
      o[q] = {shop * __fma_rn(tw, v.im, v.re), shop * __fma_rn(-tw, v.re, v.im)};
    } else {
      o[q] = {shop * v.re, shop * v.im};
    }
  }
  double part[2] = {0.0, 0.0};  // of the two spins
  if constexpr (EPI == EPI_OUT) {
    double2* out = reinterpret_cast<double2*>(a.c.out) + b0;
#pragma unroll
    for (int q = 0; q < NC; ++q) {
      if ((q >= 3 || sp0 >= 2) && a.c.g5_out) o[q] = {-o[q].re, -o[q].im};
      out[(q < 3 ? q : q + 3) * cs] = make_double2(o[q].re, o[q].im);
    }
    if (a.c.partial) {
#pragma unroll
      for (int q = 0; q < NC; ++q) part[q / 3] = __fma_rn(o[q].re, o[q].re, __fma_rn(o[q].im, o[q].im, part[q / 3]));
    }
  } else if constexpr (EPI == EPI_CGUPD) {
    const double al = a.c.alpha[r];
    double2* rf = reinterpret_cast<double2*>(a.c.r) + b0;
    double2* xf = reinterpret_cast<double2*>(a.c.x) + b0;
    const double2* pf = reinterpret_cast<const double2*>(a.c.p) + b0;
#pragma unroll
    for (int q = 0; q < NC; ++q) {
      const size_t i = (q < 3 ? q : q + 3) * cs;
      const double2 v = rf[i], x = xf[i], p = pf[i];
      const double2 n = make_double2(__fma_rn(-al, o[q].re, v.x), __fma_rn(-al, o[q].im, v.y));
      rf[i] = n;
      xf[i] = make_double2(__fma_rn(al, p.x, x.x), __fma_rn(al, p.y, x.y));
      part[q / 3] = __fma_rn(n.x, n.x, __fma_rn(n.y, n.y, part[q / 3]));
    }
  } else {  // EPI_RESID
    const double2* bf = reinterpret_cast<const double2*>(a.c.b) + b0;
    double2* out = reinterpret_cast<double2*>(a.c.out) + b0;
#pragma unroll
    for (int q = 0; q < NC; ++q) {
      const size_t i = (q < 3 ? q : q + 3) * cs;
      const double2 v = bf[i];
      const double2 n = make_double2(__dsub_rn(v.x, o[q].re), __dsub_rn(v.y, o[q].im));
      out[i] = n;
      part[q / 3] = __fma_rn(n.x, n.x, __fma_rn(n.y, n.y, part[q / 3]));
    }
  }
  return NC == 6 ? __dadd_rn(part[0], part[1]) : part[0];
}

// Does a site need FP64 sums?  m: its (unit << 16 | least s of the rows, in units of
// 2^-10 B) of [upper spin][pair of directions], E the common unit.  Spins that all
// neighbours leave at zero are exact.
__device__ __forceinline__ bool fx_small(const unsigned (&m)[2][2], unsigned E) {
  constexpr unsigned kMin = 1024 / 4;
  unsigned b[2][2];
#pragma unroll
  for (int j = 0; j < 4; ++j) b[j >> 1][j & 1] = shr32(m[j >> 1][j & 1] & 0xffffu, E - (m[j >> 1][j & 1] >> 16));
  bool small = false;
#pragma unroll
  for (int sp = 0; sp < 2; ++sp)
#pragma unroll
    for (int o = 0; o < 2; ++o)  // o = sp: spin sp; else spin 2 + sp, which takes (x, y) from the other upper spin
      small = small || (b[o][0] + b[sp][1] < kMin && (m[o][0] | m[sp][1]) != 0);
  return small;
}

// Two warps take 32 consecutive sites of one system, one for each upper spin
// (with the lower rows it feeds), and exchange the lower row that belongs to
// the other one through shared memory.  The loop over (x, y), (z, t) keeps 12
// sums of 64 bits and the code small; the upper sums of (x, y) wait in shared
// memory too.  The pairs of a block take 2^lgs systems (fastest) of the same sites,
// whose links then come from L1, and the next 32-site groups.
// The neighbours' words come by asynchronous copies to the lane's own slots in
// shared memory, one hop ahead of the one computed: latency is covered without
// registers (24^3 x 48, 12 systems, M: loads at their use 3.45 ms, copies 3.29;
// FP64 arithmetic 12.2; with a unit for each pair of directions and the sums S now 3.40.
// The same copies for the centre's words another 3% longer).  No fences
// or barriers: a lane reads what it copied, and a slot's words are in registers
// before its next copy starts.
// Bound by the integer multiplier (67% busy), fixed latencies of the 64-bit sums and
// issue (53% active): 9,100 instructions per site and system, of which 1,728 products.
// Measured beside it: four blocks per SM 3.79 ms; one thread per site unrolled
// over the hops 3.59; four sets of sites per block 3.89 (spills); projections as
// 64-bit sums 4.8, three products for a complex one 3.38 (the integer pipe is not
// the bound), products forced to IMAD.WIDE by assembly 4.1.
// QUAD: four warps take the 32 sites, one for each spin and pair of directions:
// half the chain of a thread, for lattices that leave SMs idle (4^4, 16 systems:
// 13.9 us, two warps 17.3, FP64 arithmetic 34.9).
template <int EPI, bool QUAD>
__global__ void __launch_bounds__(128, QUAD ? 3 : 5)
    dslash_fx_kernel(const __grid_constant__ DslashArgs a, const int4* links_fx, int lgs) {
  __shared__ FxStage ring[4][2];
  __shared__ longlong2 xu[4][3][32], xl[4][3][32];  // upper and lower sums on their way to another warp or loop
  __shared__ unsigned meta[2][4][32];               // of [pair of warps][2 upper spin + pair of directions], see fx_small
  __shared__ double xsum[4];
  __shared__ double xpart[2][32];
  const Geom& g = a.g;
  const int rg = blockIdx.x % a.rhs_groups;
  const int sb = blockIdx.x / a.rhs_groups;
  const int par = a.c.parity < 0 ? (sb & 1) : a.c.parity;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int sp = warp & 1, pair = QUAD ? 0 : warp >> 1;
  const int it0 = QUAD ? warp >> 1 : 0, it1 = QUAD ? it0 + 1 : 2;  // pairs of directions of this warp
  const int gpb = QUAD ? 1 : (int)(blockDim.x >> (6 + lgs));       // 32-site groups per block
  const int grp = (a.c.parity < 0 ? (sb >> 1) : sb) * gpb + (pair >> lgs);
  const int cb = grp * 32 + lane;
  const int r = (rg << lgs) + (pair & ((1 << lgs) - 1));
  const int nrhs = a.c.nrhs;
  const bool on = r < nrhs && (a.c.active == nullptr || a.c.active[r] != 0);
  const bool sums = EPI != EPI_OUT || a.c.partial != nullptr;
  if (a.trace_count && blockIdx.x == 0 && threadIdx.x == 0) {
    int n = 0;
    for (int q = 0; q < nrhs; ++q) n += (a.c.active == nullptr || a.c.active[q] != 0) ? 1 : 0;
    *a.trace_count = n;
  }
  const int SF = a.c.dagger ? +1 : -1;  // sign of the forward projection; at run time: one code for M and M^dag
  if (!__syncthreads_or(on)) {
    if (sums && lane == 0 && sp == 0 && it0 == 0 && r < nrhs && grp < a.nwarp)
      a.c.partial[((size_t)r * 2 + par) * a.nwarp + grp] = 0.0;
    return;
  }
  const bool act = on && cb < g.Vh;
  FxSum t;
  if (act) {
    const Site s = site_of(g, par, cb);
    const int opar = par ^ 1;
    const size_t cs = (size_t)g.Vh;
    const double2* fup = reinterpret_cast<const double2*>(a.c.in) + ((size_t)(r * 2 + opar) * 12 + 3 * sp) * cs;
    FxStage &s0 = ring[warp][0], &s1 = ring[warp][1];
    auto nbr = [&](int mu, bool bwd) { return fx_nbr(g, s, mu, bwd); };
    // start the copy of neighbour n for a hop of pair it
    auto copy = [&](FxStage& st, int it, int n) {
      fx_copy(st, lane, fup + n, fup + (6 + 3 * (it ? 0 : 1 - 2 * sp)) * (ptrdiff_t)cs + n, cs);
    };
    copy(s0, it0, nbr(2 * it0, false));
    fx_commit();
#pragma unroll 1
    for (int it = it0; it < it1; ++it) {
      const int4* uf = links_fx + (size_t)(4 * it + par) * a.nwarp * 288;  // direction 2 it; the next one: + 576 nwarp
      const int4* ub = links_fx + (size_t)(4 * it + opar) * a.nwarp * 288;
      const int so = it && sp ? -1 : 1, se = it || sp ? 1 : -1;  // phase signs: i^ak = so i, se
      const size_t next = (size_t)a.nwarp * 576;
      const bool ap = it && g.antiperiodic;
#pragma unroll
      for (int c = 0; c < 3; ++c) t.upr[c] = t.upi[c] = t.lor[c] = t.loi[c] = 0;
      t.s[0] = t.s[1] = t.s[2] = 0;
      t.E = kFxMinExp;
      t.big = 0;
      const int nb0 = nbr(2 * it, true);
      copy(s1, it, nb0);
      fx_commit();
      fx_arrived<1>();
      fx_hop<true, false>(t, s0, lane, uf + fx_row(cb, 9), SF * so >> 1, 0);
      copy(s0, it, nbr(2 * it + 1, false));
      fx_commit();
      fx_arrived<1>();
      fx_hop<true, true>(t, s1, lane, ub + fx_row(nb0, 9), -SF * so >> 1, 0);
      // lower row: SF (-so i (w_f - w_b)_odd + se (w_f - w_b)_even); the sums are
      // kept as the bracket times se
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        const long long x = t.lor[c], y = t.loi[c];
        t.lor[c] = so == se ? y : -y;
        t.loi[c] = so == se ? -x : x;
      }
      const int nb1 = nbr(2 * it + 1, true);
      copy(s1, it, nb1);
      fx_commit();
      fx_arrived<1>();
      fx_hop<false, false>(t, s0, lane, uf + next + fx_row(cb, 9), SF * se >> 1, ap && s.c[3] == g.L[3] - 1 ? -1 : 0);
      if (it + 1 < it1) copy(s0, it + 1, nbr(2 * it + 2, false));
      fx_commit();
      fx_arrived<1>();
      fx_hop<false, true>(t, s1, lane, ub + next + fx_row(nb1, 9), -SF * se >> 1, ap && s.c[3] == 0 ? -1 : 0);
      if (it == 0) {  // row 1 - sp
#pragma unroll
        for (int c = 0; c < 3; ++c)
          xl[warp][c][lane] = se > 0 ? make_longlong2(t.lor[c], t.loi[c]) : make_longlong2(-t.lor[c], -t.loi[c]);
      }
      if (QUAD ? it != 0 : it == 0) {
#pragma unroll
        for (int c = 0; c < 3; ++c) xu[warp][c][lane] = make_longlong2(t.upr[c], t.upi[c]);
      }
      if ((t.big >> 20) > kFxMaxExp || (t.big != 0 && (t.big >> 20) < kFxMinExp)) t.E = kFxBad;
      if (t.big == 0) t.E = 0;
      meta[pair][2 * sp + it][lane] = __byte_perm(min(min(t.s[0], t.s[1]), t.s[2]), t.E, 0x5432);
    }
  }
  __syncthreads();
  double part = 0.0;
  if (act) {
    constexpr int NC = QUAD ? 3 : 6;
    // QUAD: the warp of (x, y) finishes spin sp with the upper sums of (z, t), the
    // other one spin 2 + sp with the lower ones of spin 1 - sp's (x, y)
    const int sp0 = QUAD && it0 ? 2 + sp : sp;
    Cx<double> acc[NC];
    // the common unit of the site's sums, the same in all its warps
    unsigned m[2][2], e[2][2];  // [this or the other upper spin][pair of directions]
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      m[j >> 1][j & 1] = meta[pair][2 * (sp ^ (j >> 1)) + (j & 1)][lane];
      e[j >> 1][j & 1] = m[j >> 1][j & 1] >> 16;
    }
    unsigned E = max(max(e[0][0], e[0][1]), max(e[1][0], e[1][1]));
    if (fx_small(m, E)) E = kFxBad;
    E = max(E, kFxMinExp);
    double unit = __hiloint2double((int)(E - 56u) << 20, 0);  // 2^(E - 1079)
    if (E == kFxBad) {
      Cx<double> f[6];
      fx_sums_f64(f, &a, r, par, cb, sp, QUAD ? 1 + it0 : 3);
#pragma unroll
      for (int q = 0; q < NC; ++q) acc[q] = f[QUAD && it0 ? 3 + q : q];
      unit = 1.0;
    } else {
      // one more bit: the sums of four hops may fill 63
      const unsigned d0 = E - e[0][0] + 1, d1 = E - e[0][1] + 1, dx = E - e[1][0] + 1;
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        if (!QUAD || it0 == 0) {
          const longlong2 o = xu[QUAD ? warp ^ 2 : warp][c][lane];  // QUAD: of (z, t), else of (x, y)
          const unsigned dt = QUAD ? d0 : d1, dd = QUAD ? d1 : d0;
          acc[c] = {(double)(shr64_s(t.upr[c], dt) + shr64_s(o.x, dd)), (double)(shr64_s(t.upi[c], dt) + shr64_s(o.y, dd))};
        }
        if (!QUAD || it0) {
          const longlong2 o = xl[QUAD ? warp ^ 3 : warp ^ 1][c][lane];
          const long long lr = shr64_s(t.lor[c], d1) + shr64_s(o.x, dx), li = shr64_s(t.loi[c], d1) + shr64_s(o.y, dx);
          acc[NC - 3 + c] = SF > 0 ? Cx<double>{(double)lr, (double)li} : Cx<double>{(double)-lr, (double)-li};
        }
      }
    }
    if constexpr (EPI == EPI_OUT) {
      switch (2 * a.c.centre + (a.c.out_inv ? 1 : 0)) {
        case 0: part = fx_epilogue<EPI, 0, false>(a, sp0, r, par, cb, unit, acc); break;
        case 1: part = fx_epilogue<EPI, 0, true>(a, sp0, r, par, cb, unit, acc); break;
        case 2: part = fx_epilogue<EPI, 1, false>(a, sp0, r, par, cb, unit, acc); break;
        case 3: part = fx_epilogue<EPI, 1, true>(a, sp0, r, par, cb, unit, acc); break;
        case 4: part = fx_epilogue<EPI, 2, false>(a, sp0, r, par, cb, unit, acc); break;
        default: part = fx_epilogue<EPI, 2, true>(a, sp0, r, par, cb, unit, acc); break;
      }
    } else {  // the solver's operator (launch_nr checks the form)
      part = fx_epilogue<EPI, 2, false>(a, sp0, r, par, cb, unit, acc);
    }
  }
  if (sums) {
    // per site first the upper and the lower spin's terms, then the warp's sites,
    // then the spins: in this order in both forms
    if constexpr (QUAD) {
      if (it0) xpart[sp][lane] = part;
      __syncthreads();
      if (it0 == 0) part += xpart[sp][lane];
    }
    const double ps = __any_sync(0xffffffffu, act) ? warp_sum(part) : 0.0;
    if (lane == 0) xsum[warp] = ps;
    __syncthreads();
    if (lane == 0 && sp == 0 && it0 == 0 && r < nrhs && grp < a.nwarp)
      a.c.partial[((size_t)r * 2 + par) * a.nwarp + grp] = xsum[warp] + xsum[warp + 1];
  }
}

}  // namespace tml
