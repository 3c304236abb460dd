// The FP64 hopping stencil in 64-bit fixed point.
//
// The FP64 pipe of this GPU retires 2 FMAs per clock per SM, the integer
// multiply-add IMAD.WIDE (32 x 32 + 64 bits) 62: a site of the FP64 stencil
// (864 FP64 instructions for the hops, 264 for a clover block pair) takes
// 432-560 clocks of an SM on the FP64 pipe, five to seven times what its
// 1200-2500 bytes take from HBM.  So the products run on integers here:
//
//   * links (|entry| <= 1) are held a second time as integers U 2^60, clover
//     blocks as T 2^59 (2^58 for entries from 2 to 4), each stored as two
//     signed 32-bit limbs;
//   * the spinor read at each neighbour is brought to a common power of two
//     of its 24 components (the largest exponent E, unit 2^(E - 1081): 59
//     bits and sign), projected and multiplied in integers: limbs (ah, al),
//     (bh, bl) give hh += ah bh, mid += ah bl + al bh, three IMAD.WIDE per
//     real product; al bl (2^-58 of the largest product) is left out;
//   * a hop's result hh + mid / 2^32 is rounded to the unit 2^(E - 1077) and
//     added to the site's sum, which is kept at the largest E met so far;
//   * the sum (63 bits) is converted to FP64 once, and the vector part of the
//     epilogue (beta, self, aux, reductions) is FP64.
//
// Accuracy.  With w = 2^-54 times 2^E (E the largest exponent among the site's
// neighbours), a hop's result is off by 0.35 w typically and 2.5 w at most:
// the rounding 0.5, the products al bl left out 6/4, the inputs' truncation
// 0.3, the links' 0.2; a component of the sum of eight by w and 20 w.  That is
// relative to the largest neighbour component, where FP64 arithmetic is
// relative to what the component itself is summed from.  Where the two differ
// (components that do not mix: unit or block-diagonal links, spins and colours
// of very different size), the site is computed in FP64: every real component
// of the sum has to be reached, by at least one of its eight hops, with 2^-5 of
// 2^E (fx_reaches), and the site term's operand must not exceed the neighbours
// by more than 2^6 |beta|.  A component that stays in fixed point is thus off
// by 2^-49 of its own terms typically, the bound of FP64 arithmetic with its
// seventeen roundings in a row.  On Gaussian fields practically no site goes to
// FP64, on the solution of a point source about two in a thousand.  Relative error
// against the exact operator on Gaussian fields 0.97e-16 (FP64 kernel 1.1e-16)
// for Wilson, 1.8e-16 (1.9e-16) for clover.
//
// Measured (full clover D, one parity of 24^3 x 48, one right-hand side): FP64
// kernel 780 us = 0.81 TFLOP/s, its pipe's limit; here 248 us = 3.1 TB/s; the
// FP64 residual of 32^3 x 64 2.46 ms -> 0.83 ms a parity.  Bound by latency: 7100
// instructions a warp of 16 sites at half of the issue slots, because 128
// registers (and 180-420 bytes of spills a thread, 2.6 % of the instructions)
// leave sixteen warps an SM, which wait on loads and on the fixed latency of the
// integer chains; DRAM at 0.42 of the copy rate.
//
// Other sites where fixed point does not apply -- a neighbour component that
// is not finite, or within 2^128 of the ends of the FP64 range -- are computed
// by the FP64 code (fx_site_fp64) too, so infinities and NaN propagate as there.
// Links with an entry above 1 and clover blocks with one of 4 or more have no
// fixed-point form, and their lattice keeps the FP64 kernel: which arithmetic
// runs is a matter of the operator's entries alone.  The copies are a matter of
// memory: where there is none for them the kernel converts as it reads
// (FX_RAW), to the same integers and the same result.
#pragma once

#include "dslash.cuh"

namespace bridge {

constexpr int FX_EMIN = 128, FX_EMAX = 1900;  // biased exponents a spinor may have
constexpr int FX_THREADS = 128;               // block of the stencil: two lanes a site
constexpr int FX_SITES = FX_THREADS / 2;
constexpr uint32_t FX_LINK_TOP = 0x3ff00001u;  // links: at most 1 (+ rounding), unit 2^-60
constexpr int FX_NO_HOP = -2;                  // "exponent" of a hop with phase 0
constexpr int FX_SELF = 6;                     // T x: |x| below 2^FX_SELF |beta| times the largest neighbour
constexpr int FX_CLOV_EMAX = 2;                // clover entries: below 2^e, unit 2^(e - 60), e = 1 or 2
// The exponent e of clover blocks whose largest |entry| has the high word top
// (entries below 2^e); 0: they have no fixed-point form.
BR_HD int fx_clov_exponent(uint32_t top) {
  for (int e = 1; e <= FX_CLOV_EMAX; ++e)
    if (top < ((uint32_t)(1023 + e) << 20)) return e;
  return 0;
}

// x as an integer with unit 2^(E - 1075 - SH), E >= the biased exponent of
// x: |result| < 2^(53 + SH).  Rounds towards zero; neg = -1 changes the sign.
template <int SH>
BR_D long long fx_from_bits(uint32_t lo, uint32_t hi, int E, int neg) {
  const int e = (int)((hi >> 20) & 0x7ffu);
  const uint32_t mh = (hi & 0xfffffu) | 0x100000u;
  unsigned long long m = (((unsigned long long)mh << 32) | lo) << SH;
  m >>= min(E - e, 63);
  const long long s = (long long)(((int)hi >> 31) ^ neg);
  return ((long long)m ^ s) - s;
}

// Two signed 32-bit limbs: x = h 2^32 + l.
struct Fx2 {
  int h, l;
};
BR_D Fx2 fx_split(long long x) { return {(int)(x >> 32) + (int)((uint32_t)x >> 31), (int)x}; }

// The limbs of an operator entry, a double of magnitude up to 2^(e0 - 1023),
// times 2^(60 + 1023 - e0).  The stencil negates limbs: the low one is kept
// off -2^31 (by one unit).
BR_D Fx2 fx_limbs_of(uint32_t lo, uint32_t hi, int e0) {
  Fx2 r = fx_split(fx_from_bits<8>(lo, hi, max(e0, (int)((hi >> 20) & 0x7ffu)), 0));
  r.l = max(r.l, -0x7fffffff);
  return r;
}
// An operator entry as it is read: RAW a double, else its limbs.
template <bool RAW>
BR_D Fx2 fx_limbs(uint32_t w0, uint32_t w1, int e0) {
  if constexpr (RAW) return fx_limbs_of(w0, w1, e0);
  return {(int)w1, (int)w0};
}

// hh += a.h b.h, mid += a.h b.l + a.l b.h.
BR_D void fx_mac(Fx2 a, Fx2 b, long long& hh, long long& mid) {
  asm("mad.wide.s32 %0, %1, %2, %0;" : "+l"(hh) : "r"(a.h), "r"(b.h));
  asm("mad.wide.s32 %0, %1, %2, %0;" : "+l"(mid) : "r"(a.h), "r"(b.l));
  asm("mad.wide.s32 %0, %1, %2, %0;" : "+l"(mid) : "r"(a.l), "r"(b.h));
}
BR_D Fx2 fx_neg(Fx2 a) { return {-a.h, -a.l}; }

// The largest biased exponent of n double2 values held as raw words; 0 when
// all are zero.
template <int N>
BR_D uint32_t fx_max_word(const uint4 w[N]) {
  uint32_t m = 0;
#pragma unroll
  for (int k = 0; k < N; ++k) m = max(m, max(w[k].y & 0x7fffffffu, w[k].w & 0x7fffffffu));
  return m;
}

// What a site's exponent word says for the largest word of its components.
BR_D int fx_site_exponent(uint32_t m) {
  const int E = (int)(m >> 20);
  return m == 0 ? 0 : (E < FX_EMIN || E > FX_EMAX) ? -1 : E;
}

// The fixed-point form of one FP64 spinor, stored at site ih of a block
// (layout: fx_block_bytes).
BR_D void fx_store(char* block, long vh, uint32_t ih, const cx<double> s[12]) {
  uint4 w[12];
#pragma unroll
  for (int k = 0; k < 12; ++k)
    w[k] = make_uint4((uint32_t)__double2loint(s[k].r), (uint32_t)__double2hiint(s[k].r), (uint32_t)__double2loint(s[k].i),
                      (uint32_t)__double2hiint(s[k].i));
  const uint32_t m = fx_max_word<12>(w);
  const int E = (int)(m >> 20);
  uint4* dst = reinterpret_cast<uint4*>(block) + ih;
#pragma unroll
  for (int k = 0; k < 12; ++k) {
    const long long r = fx_from_bits<6>(w[k].x, w[k].y, E, 0), i = fx_from_bits<6>(w[k].z, w[k].w, E, 0);
    dst[k * vh] = make_uint4((uint32_t)r, (uint32_t)(r >> 32), (uint32_t)i, (uint32_t)(i >> 32));
  }
  reinterpret_cast<int*>(block + 192 * vh)[ih] = fx_site_exponent(m);
}

BR_D long long fx_shift_round(long long x, int d) {  // x / 2^d to nearest, d in 0 .. 62
  return (x + ((1ll << d) >> 1)) >> d;
}

// The slots of one site: neighbour index (bit 31: its hop wraps with phase -1)
// and exponent (or FX_NO_HOP), in the order of the directions 2 mu + backward.
struct FxSlots {
  uint2 w[8][FX_SITES];
};

// Bit 0 and bit 3: whether the real and the imaginary part of a hop's result u
// (unit 2^(Ea - 1077)) reach 2^-FX_KEEP times 2^(Ea - 1023).  FX_KEEP: at 4 the
// solution of a point source (24^3 x 48, kappa 0.125) has a site in twenty with
// a component below, in every second warp; at 5 one in 600, at 6 one in 3000.
constexpr int FX_KEEP = 5;
BR_D uint32_t fx_reaches(cx<long long> u) {
  const int r = (int)(u.r >> 32), i = (int)(u.i >> 32);
  constexpr int least = 1 << (54 - FX_KEEP - 32);
  return ((r ^ (r >> 31)) >= least ? 1u : 0u) | ((i ^ (i >> 31)) >= least ? 8u : 0u);
}

// The exponent word of site i of an FP64 block of N planes.
template <int N>
BR_D int fx_exponent(const char* block, long vh, uint32_t i) {
  uint4 w[N];
#pragma unroll
  for (int k = 0; k < N; ++k) w[k] = __ldg(reinterpret_cast<const uint4*>(block) + k * vh + i);
  return fx_site_exponent(fx_max_word<N>(w));
}

template <int MU, bool RAW>
BR_D void fx_neighbours(const HopArgs& a, const char* in, uint32_t ih, const int c[4], uint32_t xh, FxSlots& sh, int site,
                        int& Ea, int& bad) {
  uint32_t f, b;
  bool wf, wb;
  neighbours<MU>(a.g, ih, c, xh, f, b, wf, wb);
  const float bc = a.bcf[MU];
  const int* ex = reinterpret_cast<const int*>(in + 192 * a.g.vh);
  int ef = RAW ? fx_exponent<12>(in, a.g.vh, f) : __ldg(ex + f), eb = RAW ? fx_exponent<12>(in, a.g.vh, b) : __ldg(ex + b);
  bad |= (ef < 0) | (eb < 0);
  if (wf && bc == 0.f) ef = FX_NO_HOP;
  if (wb && bc == 0.f) eb = FX_NO_HOP;
  Ea = max(Ea, max(ef, eb));
  sh.w[2 * MU][site] = make_uint2(f | ((wf && bc < 0.f) ? 0x80000000u : 0u), (uint32_t)ef);
  sh.w[2 * MU + 1][site] = make_uint2(b | ((wb && bc < 0.f) ? 0x80000000u : 0u), (uint32_t)eb);
}

// What one colour of one hop reads: two spin components and a column of the link.
struct FxLoads {
  uint4 p, x, l[3];
};

// A spinor component of a site with exponent word E, as it is read: RAW two
// doubles (E may be below them where the hop has phase 0: any value will do).
template <bool RAW>
BR_D cx<long long> fx_value(uint4 v, int E) {
  if constexpr (RAW) {
    auto one = [&](uint32_t lo, uint32_t hi) { return fx_from_bits<6>(lo, hi, max(E, (int)((hi >> 20) & 0x7ffu)), 0); };
    return {one(v.x, v.y), one(v.z, v.w)};
  }
  return {(long long)(((unsigned long long)v.y << 32) | v.x), (long long)(((unsigned long long)v.w << 32) | v.z)};
}
BR_D long long fx_sign(long long x, int m) { return (x ^ (long long)m) - (long long)m; }  // m = 0 or -1: x or -x
BR_D cx<long long> fx_shfl(cx<long long> v) {
  return {__shfl_xor_sync(0xffffffffu, v.r, 1), __shfl_xor_sync(0xffffffffu, v.i, 1)};
}

// The eight hops of a site for the projected spin component k of this lane.
// With Q = i (mu = 0, 2) or 1 (mu = 1, 3), a sign s and the partner spin
// 3 - k (mu = 0, 1) or 2 + k (mu = 2, 3), every hop reads
//   h = p_k + s Q p_partner,  u = U h,  spin k += u,  partner += s conj(Q) u
// (s = +1 for a forward hop, flipped for a backward one, for k = 1 with mu =
// 1, 2 and for mu = 3).  up: spin k; low[0], low[1]: what goes to the partner
// of mu = 0, 1 and of mu = 2, 3.  Units 2^(Ea - 1077).  Returned: bits 0-5,
// 12-17, 6-11: the components of up, low[0], low[1] that some hop reaches
// (real parts, then imaginary parts; fx_reaches).
//
// A loop over the directions around one body, the loads of the next colour
// issued while one is multiplied: unrolled over the directions the code
// (115 KB) ran out of the instruction cache, and without the early loads the
// kernel took 1.25 times as long.
template <bool RAW>
BR_D uint32_t fx_hops(const HopArgs& a, const char* in, const char* g_out, const char* g_in, long lbb, uint32_t ih, int Ea,
                  const FxSlots& sh, int site, int k, cx<long long> up[3], cx<long long> low[2][3]) {
  const long vs = 16 * a.g.vh;  // bytes of a plane
  const char* pk = in + 3 * k * vs;
  FxLoads b[3];
  auto load = [&](FxLoads& f, int dir, int c) {
    const uint32_t nb = sh.w[dir][site].x & 0x7fffffffu;
    const bool fwd = (dir & 1) == 0;
    const char* px = in + (dir < 4 ? 3 * (3 - k) : 3 * (2 + k)) * vs;
    const unsigned long long at = 16ull * nb;
    f.p = __ldg(reinterpret_cast<const uint4*>(pk + at + c * vs));
    f.x = __ldg(reinterpret_cast<const uint4*>(px + at + c * vs));
    // column c of U, or of U^dagger: entry (r, c) at plane 3 r + c, or 3 c + r
    const char* lp = (fwd ? g_out : g_in) + (dir >> 1) * lbb + 16ull * (fwd ? ih : nb) + (fwd ? c : 3 * c) * vs;
    const long lr = fwd ? 3 * vs : vs;
#pragma unroll
    for (int r = 0; r < 3; ++r) f.l[r] = ldg4<true>(reinterpret_cast<const uint4*>(lp + r * lr));
  };
#pragma unroll
  for (int c = 0; c < 3; ++c) up[c] = low[0][c] = low[1][c] = {0, 0};
  uint32_t reach = 0;
  load(b[0], 0, 0);
#pragma unroll 1
  for (int dir = 0; dir < 8; ++dir) {
    if (dir == 4) {
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        low[0][c] = low[1][c];
        low[1][c] = {0, 0};
      }
      reach = (reach & 0x3fu) | ((reach & 0xfc0u) << 6);
    }
    const uint2 w = sh.w[dir][site];
    const int mu = dir >> 1;
    const bool fwd = (dir & 1) == 0, rot = (mu & 1) == 0;
    // s as a mask, and the sign of Q p's real part
    const int m = (fwd ? 0 : -1) ^ ((k && (mu == 1 || mu == 2)) ? -1 : 0) ^ (mu == 3 ? -1 : 0);
    const int mr = rot ? ~m : m;
    const int s1 = fwd ? 1 : -1;
    long long rh[3] = {0, 0, 0}, rm[3] = {0, 0, 0}, jh[3] = {0, 0, 0}, jm[3] = {0, 0, 0};
    auto mac = [&](const FxLoads& f) {
      const cx<long long> p = fx_value<RAW>(f.p, (int)w.y), x = fx_value<RAW>(f.x, (int)w.y);
      const Fx2 hr = fx_split(p.r + fx_sign(rot ? x.i : x.r, mr)), hi = fx_split(p.i + fx_sign(rot ? x.r : x.i, m));
#pragma unroll
      for (int r = 0; r < 3; ++r) {
        const Fx2 ur = fx_limbs<RAW>(f.l[r].x, f.l[r].y, 1023), li = fx_limbs<RAW>(f.l[r].z, f.l[r].w, 1023);
        const Fx2 ui = {s1 * li.h, s1 * li.l};
        fx_mac(ur, hr, rh[r], rm[r]);
        fx_mac(fx_neg(ui), hi, rh[r], rm[r]);
        fx_mac(ur, hi, jh[r], jm[r]);
        fx_mac(ui, hr, jh[r], jm[r]);
      }
    };
    load(b[1], dir, 1);
    mac(b[0]);
    load(b[2], dir, 2);
    mac(b[1]);
    if (dir < 7) load(b[0], dir + 1, 0);
    mac(b[2]);
    const int d = min(Ea - (int)w.y, 62);  // 62 where there is no contribution: rounds to zero
    const long long half = (1ll << d) >> 1;
    const bool flip = __any_sync(0xffffffffu, w.x >> 31);
    uint32_t hit = 0;
#pragma unroll
    for (int r = 0; r < 3; ++r) {
      cx<long long> u = {(rh[r] + fx_split(rm[r]).h + half) >> d, (jh[r] + fx_split(jm[r]).h + half) >> d};
      hit |= fx_reaches(u) << r;
      if (flip && (w.x >> 31)) u = {-u.r, -u.i};
      up[r] = up[r] + u;
      low[1][r] = low[1][r] + cx<long long>{fx_sign(rot ? u.i : u.r, m), fx_sign(rot ? u.r : u.i, mr)};
    }
    reach |= hit | ((rot ? (hit >> 3) | ((hit & 7u) << 3) : hit) << 6);
  }
  return reach;
}

// y = A x for one packed Hermitian 6x6 block in fixed point (entries below
// 2^e times 2^(60 - e)) and |x| < 2^58 (twelve products then stay below
// 2^63): y in units of 2^e times the unit of x.  RAW: the block in FP64.
template <bool RAW>
BR_D void fx_hermitian6(const char* base, long vh, uint32_t i, int b, int e, const cx<long long> x[6], cx<long long> y[6]) {
  const uint4* p = reinterpret_cast<const uint4*>(base) + 18 * b * vh + i;
  Fx2 xr[6], xi[6];
  long long rh[6], rm[6], ih[6], im[6];
#pragma unroll
  for (int k = 0; k < 6; ++k) {
    xr[k] = fx_split(x[k].r);
    xi[k] = fx_split(x[k].i);
    rh[k] = rm[k] = ih[k] = im[k] = 0;
  }
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    const uint4 w = ldg4<true>(p + k * vh);
    const Fx2 d0 = fx_limbs<RAW>(w.x, w.y, 1023 + e), d1 = fx_limbs<RAW>(w.z, w.w, 1023 + e);
    fx_mac(d0, xr[2 * k], rh[2 * k], rm[2 * k]);
    fx_mac(d0, xi[2 * k], ih[2 * k], im[2 * k]);
    fx_mac(d1, xr[2 * k + 1], rh[2 * k + 1], rm[2 * k + 1]);
    fx_mac(d1, xi[2 * k + 1], ih[2 * k + 1], im[2 * k + 1]);
  }
  int k = 3;
#pragma unroll
  for (int r = 1; r < 6; ++r)
#pragma unroll
    for (int c = 0; c < r; ++c) {
      const uint4 w = ldg4<true>(p + k * vh);
      ++k;
      const Fx2 ar = fx_limbs<RAW>(w.x, w.y, 1023 + e), ai = fx_limbs<RAW>(w.z, w.w, 1023 + e), na = fx_neg(ai);
      fx_mac(ar, xr[c], rh[r], rm[r]);  // y_r += a x_c
      fx_mac(na, xi[c], rh[r], rm[r]);
      fx_mac(ar, xi[c], ih[r], im[r]);
      fx_mac(ai, xr[c], ih[r], im[r]);
      fx_mac(ar, xr[r], rh[c], rm[c]);  // y_c += conj(a) x_r
      fx_mac(ai, xi[r], rh[c], rm[c]);
      fx_mac(ar, xi[r], ih[c], im[c]);
      fx_mac(na, xr[r], ih[c], im[c]);
    }
#pragma unroll
  for (int r = 0; r < 6; ++r) {
    y[r].r = (rh[r] << 4) + ((rm[r] + (1ll << 27)) >> 28);
    y[r].i = (ih[r] << 4) + ((im[r] + (1ll << 27)) >> 28);
  }
}

// 2^(e - 1023) for a biased exponent e in 1 .. 2046.
BR_D double fx_pow2(int e) { return __hiloint2double(e << 20, 0); }

// One hop in FP64 for the projected spin component k of this lane (signs and
// partner spins as in fx_hops): up gets U h, low what goes to the partner.
template <int MU, bool FWD>
BR_D void fx_hop_fp64(const char* in, const char* lb, long vh, uint2 slot, uint32_t ih, int k, cx<double> up[3],
                      cx<double> low[3]) {
  constexpr bool rot = MU == 0 || MU == 2;
  const bool neg = !FWD ^ (k && (MU == 1 || MU == 2)) ^ (MU == 3);
  const uint32_t nb = slot.x & 0x7fffffffu;
  const double phase = (int)slot.y == FX_NO_HOP ? 0.0 : (slot.x >> 31) ? -1.0 : 1.0;
  const double2* pk = reinterpret_cast<const double2*>(in) + 3 * k * vh + nb;
  const double2* px = reinterpret_cast<const double2*>(in) + (MU < 2 ? 3 * (3 - k) : 3 * (2 + k)) * vh + nb;
  cx<double> h[3];
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    const double2 p = __ldg(pk + c * vh), q = __ldg(px + c * vh);
    const cx<double> x = rot ? cx<double>{-q.y, q.x} : cx<double>{q.x, q.y};
    h[c] = neg ? cx<double>{p.x, p.y} - x : cx<double>{p.x, p.y} + x;
    if (phase != 1.0) h[c] = phase * h[c];
  }
  Link<double> U;
  load_link<P_F64, true>(lb, vh, FWD ? ih : nb, U);
#pragma unroll
  for (int r = 0; r < 3; ++r) {
    const cx<double> u = FWD ? crow3(U.m[r][0], U.m[r][1], U.m[r][2], h) : crow3_conj(U.m[0][r], U.m[1][r], U.m[2][r], h);
    const cx<double> w = rot ? times_mi(u) : u;
    up[r] = up[r] + u;
    low[r] = neg ? low[r] - w : low[r] + w;
  }
}
template <int MU>
BR_D void fx_dir_fp64(const HopArgs& a, const char* in, const char* g_out, const char* g_in, long lbb, uint32_t ih,
                      const FxSlots& sh, int site, int k, cx<double> up[3], cx<double> low[3]) {
  fx_hop_fp64<MU, true>(in, g_out + MU * lbb, a.g.vh, sh.w[2 * MU][site], ih, k, up, low);
  fx_hop_fp64<MU, false>(in, g_in + MU * lbb, a.g.vh, sh.w[2 * MU + 1][site], ih, k, up, low);
}

// y = A x for one packed Hermitian 6x6 block in FP64, entry by entry.
BR_D void fx_hermitian6_fp64(const char* base, long vh, uint32_t i, int b, const cx<double> x[6], cx<double> y[6]) {
  const double2* p = reinterpret_cast<const double2*>(base) + 18 * b * vh + i;
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    const double2 d = ldg4<true>(p + k * vh);
    y[2 * k] = d.x * x[2 * k];
    y[2 * k + 1] = d.y * x[2 * k + 1];
  }
  int k = 3;
#pragma unroll
  for (int r = 1; r < 6; ++r)
#pragma unroll
    for (int c = 0; c < r; ++c) {
      const double2 w = ldg4<true>(p + k * vh);
      ++k;
      y[r] = cfma(cx<double>{w.x, w.y}, x[c], y[r]);
      y[c] = cfma_conj(cx<double>{w.x, w.y}, x[r], y[c]);
    }
}

// The site in FP64 by its two lanes (spins 2 k, 2 k + 1 of the output to lane
// k), the sums in the order of the FP64 kernel; called by whole warps (called
// in a divergent branch it cost the other sites a tenth in spills).  Not
// inlined: it runs only where fixed point does not do.  Split over the two
// lanes it costs the FP64 pipe what the FP64 kernel does: full Wilson D on 24^3 x
// 48 with every site here 1650 us, on the FP64 kernel 1421, in fixed point 532.
template <int FL>
__device__ __noinline__ void fx_site_fp64(const HopArgs& a, int rhs, uint32_t ih, int k, const FxSlots& sh,
                                          int site, double2* out) {
  const int p = a.out_parity;
  const long vh = a.g.vh, lbb = link_block_bytes(P_F64, vh), cbb = clover_block_bytes(P_F64, vh);
  auto other = [&](cx<double> z) {
    return cx<double>{__shfl_xor_sync(0xffffffffu, z.r, 1), __shfl_xor_sync(0xffffffffu, z.i, 1)};
  };
  cx<double> v[6];
  {
    const char* g_out = a.gauge + (long)p * 4 * lbb;
    const char* g_in = a.gauge + (long)(1 - p) * 4 * lbb;
    const char* in = a.in + rhs * a.in_rs;
    cx<double> up[3], low[3];  // spin k; the partner's sum: spin 3 - k for mu = 0, 1, then spin 2 + k
#pragma unroll
    for (int r = 0; r < 3; ++r) up[r] = low[r] = czero<double>();
    fx_dir_fp64<0>(a, in, g_out, g_in, lbb, ih, sh, site, k, up, low);
    fx_dir_fp64<1>(a, in, g_out, g_in, lbb, ih, sh, site, k, up, low);
    // each sum goes on where the next directions add to it
#pragma unroll
    for (int r = 0; r < 3; ++r) low[r] = other(low[r]);
    fx_dir_fp64<2>(a, in, g_out, g_in, lbb, ih, sh, site, k, up, low);
    fx_dir_fp64<3>(a, in, g_out, g_in, lbb, ih, sh, site, k, up, low);
#pragma unroll
    for (int r = 0; r < 3; ++r) {
      const cx<double> x = other(k ? up[r] : low[r]);  // spin 1 to lane 0, spin 2 to lane 1
      v[r] = a.beta * (k ? x : up[r]);
      v[3 + r] = a.beta * (k ? low[r] : x);
    }
  }
  auto plane = [&](const char* f, int j) {
    const double2 w = ldg4<true>(reinterpret_cast<const double2*>(f) + (6 * k + j) * vh + ih);
    return cx<double>{w.x, w.y};
  };
  if (FL & F_AUX)
#pragma unroll
    for (int j = 0; j < 6; ++j) v[j] = v[j] + a.caux * plane(a.aux + rhs * a.aux_rs, j);
  if ((FL & F_G5) && k)
#pragma unroll
    for (int j = 0; j < 6; ++j) v[j] = {-v[j].r, -v[j].i};
  if (FL & F_E_CLOV) {
    cx<double> y[6];
    fx_hermitian6_fp64(a.clovE + p * cbb, vh, ih, k, v, y);
#pragma unroll
    for (int j = 0; j < 6; ++j) v[j] = y[j];
  }
  if (FL & F_SELF) {
    const char* self = a.self + rhs * a.self_rs;
    if (FL & F_SELF_CLOV) {
      cx<double> x[6], y[6];
#pragma unroll
      for (int j = 0; j < 6; ++j) x[j] = plane(self, j);
      fx_hermitian6_fp64(a.clovM + p * cbb, vh, ih, k, x, y);
#pragma unroll
      for (int j = 0; j < 6; ++j) v[j] = v[j] + a.s1 * y[j];
    } else {
#pragma unroll
      for (int j = 0; j < 6; ++j) v[j] = v[j] + a.s1 * plane(self, j);
    }
  }
#pragma unroll
  for (int j = 0; j < 6; ++j) out[j] = make_double2(v[j].r, v[j].i);
}

// Two adjacent lanes share an output site: lane k forms the projected spin
// component k of every hop (its products, and its contributions to the two
// lower spins), then the lanes exchange sums and each finishes one chirality
// (spins 2 k, 2 k + 1: one 6x6 clover block).  One lane a site needed 168
// registers and left twelve warps on an SM, a third of the issue slots busy;
// two need 128 (sixteen warps) and read each link as a broadcast.
//
// RAW (FX_RAW: no memory for the copies): operands converted as they are read,
// every neighbour's exponent from its twelve components.  Full D on 24^3 x 48,
// Wilson / clover: FP64 kernel 1421 / 1724 us, RAW 1023 / 1173, from copies 536
// / 641 (staggered, stag.cuh: 528, 406, 238).
template <int FL, int RED, bool RAW>
__global__ void __launch_bounds__(FX_THREADS, RAW ? 2 : 4) hop_kernel_fx(const HopArgs a) {
  const int nrhs = a.nrhs;
  const int rhs = blockIdx.x % nrhs;
  const int sb = blockIdx.x / nrhs;
  const long vh = a.g.vh;
  constexpr int NV = RED == R_NORM ? 1 : RED == R_DOT_A ? 2 : 3;
  __shared__ FxSlots sh;
  PartialSum<double> ps[NV];
  const bool skip = rhs_finished(a.red, rhs);
  if (skip && all_finished(a.red, nrhs)) return;
  if (!skip) {
    const int p = a.out_parity, site = threadIdx.x >> 1, k = threadIdx.x & 1;
    const long lbb = link_block_bytes(P_F64, vh), cbb = clover_block_bytes(P_F64, vh);
    const char* g_out = (RAW ? a.gauge : a.gauge_fx) + (long)p * 4 * lbb;
    const char* g_in = (RAW ? a.gauge : a.gauge_fx) + (long)(1 - p) * 4 * lbb;
    const char* in = RAW ? a.in + rhs * a.in_rs : a.in_fx + rhs * a.in_fx_rs;
    const uint32_t stride = (uint32_t)a.nblk * FX_SITES;
    // whole warps stay in the loop (shuffles): lanes past the end redo the last site
    for (uint32_t i0 = sb * FX_SITES + (site & ~15); i0 < (uint32_t)vh; i0 += stride) {
      const uint32_t want = i0 + (site & 15), ih = min(want, (uint32_t)vh - 1);
      const bool live = want < (uint32_t)vh;
      int Ea = 0, bad = 0;
      {
        int c[4];
        uint32_t xh;
        site_coords(a.g, ih, p, c, xh);
        if (k == 0) {
          fx_neighbours<0, RAW>(a, in, ih, c, xh, sh, site, Ea, bad);
          fx_neighbours<1, RAW>(a, in, ih, c, xh, sh, site, Ea, bad);
        } else {
          fx_neighbours<2, RAW>(a, in, ih, c, xh, sh, site, Ea, bad);
          fx_neighbours<3, RAW>(a, in, ih, c, xh, sh, site, Ea, bad);
        }
      }
      Ea = max(Ea, __shfl_xor_sync(0xffffffffu, Ea, 1));
      __syncwarp();
      cx<long long> q[6];
      {
        cx<long long> up[3], low[2][3];
        const uint32_t mine = fx_hops<RAW>(a, in, g_out, g_in, lbb, ih, Ea, sh, site, k, up, low);
        // spin 0 or 1 from this lane's hops; spin 2 (lane 0) or 3 (lane 1) from both lanes'
        const uint32_t theirs = __shfl_xor_sync(0xffffffffu, mine, 1);
        if (Ea != 0 && ((mine & 0x3fu) != 0x3fu || (((mine >> 6) | (theirs >> 12)) & 0x3fu) != 0x3fu)) bad = 1;
#pragma unroll
        for (int c = 0; c < 3; ++c) {
          const cx<long long> x = fx_shfl(k ? up[c] : low[1][c]);  // spin 1 to lane 0, spin 2's share to lane 1
          const cx<long long> y = fx_shfl(low[0][c]);              // spin 3's share to lane 1
          q[c] = k ? x + low[0][c] : up[c];
          q[3 + c] = k ? y + low[1][c] : x;
        }
      }
      // scale of the sum: beta times its unit (0 for an empty sum)
      int e = Ea - 54;
      if (FL & F_E_CLOV) {
        // T^-1 on the sum, brought below 2^58 first
        unsigned long long m = 0;
#pragma unroll
        for (int j = 0; j < 6; ++j) m |= (unsigned long long)((q[j].r ^ (q[j].r >> 63)) | (q[j].i ^ (q[j].i >> 63)));
        const int d = max(0, 64 - __clzll((long long)m) - 58);
#pragma unroll
        for (int j = 0; j < 6; ++j) q[j] = {fx_shift_round(q[j].r, d), fx_shift_round(q[j].i, d)};
        cx<long long> y[6];
        fx_hermitian6<RAW>((RAW ? a.clovE : a.clovE_fx) + p * cbb, vh, ih, k, a.eE_fx, q, y);
#pragma unroll
        for (int j = 0; j < 6; ++j) q[j] = y[j];
        e += a.eE_fx + d;
      }
      double f = Ea == 0 ? 0.0 : a.beta * fx_pow2(e);
      if ((FL & F_G5) && k) f = -f;
      const long o = 6 * k * vh + ih;  // this lane's planes 6 k .. 6 k + 5
      const double2* self = reinterpret_cast<const double2*>(a.self + rhs * a.self_rs) + o;
      cx<double> v[6], s[6];
      if (FL & F_AUX) {
        const double2* aux = reinterpret_cast<const double2*>(a.aux + rhs * a.aux_rs) + o;
#pragma unroll
        for (int j = 0; j < 6; ++j) {
          const double2 w = ldg4<true>(aux + j * vh);
          v[j] = a.caux == 1.0 ? cx<double>{w.x, w.y} : a.caux * cx<double>{w.x, w.y};
        }
      }
      if ((FL & F_SELF) && !(FL & F_SELF_CLOV))
#pragma unroll
        for (int j = 0; j < 6; ++j) {
          const double2 w = ldg4<true>(self + j * vh);
          s[j] = {w.x, w.y};
        }
#pragma unroll
      for (int j = 0; j < 6; ++j) {
        const cx<double> x = {(double)q[j].r, (double)q[j].i};
        if ((FL & F_SELF) && !(FL & F_SELF_CLOV)) {
          const cx<double> t = a.s1 == 1.0 ? s[j] : a.s1 * s[j];
          v[j] = caxpy(f, x, (FL & F_AUX) ? v[j] + t : t);
        } else {
          v[j] = (FL & F_AUX) ? caxpy(f, x, v[j]) : f * x;
        }
      }
      if (FL & F_SELF_CLOV) {
        uint4 w[6];
#pragma unroll
        for (int j = 0; j < 6; ++j) w[j] = ldg4<true>(reinterpret_cast<const uint4*>(self) + j * vh);
        const uint32_t m = fx_max_word<6>(w);
        const int Es = (int)(m >> 20);
        // the hops must reach the size of what T x is rounded against
        if (m != 0 && (Es < FX_EMIN || Es > FX_EMAX || Ea == 0 || Es > Ea + a.eb_fx + FX_SELF)) bad = 1;
        if (m != 0 && !bad) {
          cx<long long> y[6];
#pragma unroll
          for (int j = 0; j < 6; ++j)
            q[j] = {fx_from_bits<5>(w[j].x, w[j].y, Es, 0), fx_from_bits<5>(w[j].z, w[j].w, Es, 0)};
          fx_hermitian6<RAW>((RAW ? a.clovM : a.clovM_fx) + p * cbb, vh, ih, k, a.eM_fx, q, y);
          // unit of q: 2^(Es - 1080); of y: 2^e times that
          const double fs = a.s1 * fx_pow2(Es - 57 + a.eM_fx);
#pragma unroll
          for (int j = 0; j < 6; ++j) v[j] = caxpy(fs, cx<double>{(double)y[j].r, (double)y[j].i}, v[j]);
        }
      }
      bad |= __shfl_xor_sync(0xffffffffu, bad, 1);
      if (__any_sync(0xffffffffu, bad)) {
        double2 w[6];
        fx_site_fp64<FL>(a, rhs, ih, k, sh, site, w);
        if (bad)
#pragma unroll
          for (int j = 0; j < 6; ++j) v[j] = {w[j].x, w[j].y};
      }
      __syncwarp();  // the slots have been read
      if (live) {
        double2* out = reinterpret_cast<double2*>(a.out + rhs * a.out_rs) + o;
#pragma unroll
        for (int j = 0; j < 6; ++j) out[j * vh] = make_double2(v[j].r, v[j].i);
        if (RED == R_NORM || RED == R_TS) {
          double n = 0;
#pragma unroll
          for (int j = 0; j < 6; ++j) n += v[j].r * v[j].r + v[j].i * v[j].i;
          ps[RED == R_TS ? 2 : 0].add(n);
        }
        if (RED == R_DOT_A || RED == R_TS) {
          const double2* av = reinterpret_cast<const double2*>(a.avec + rhs * a.avec_rs) + o;
          cx<double> d = czero<double>();
#pragma unroll
          for (int j = 0; j < 6; ++j) {
            if (RED == R_DOT_A) {
              const double2 w = ldg4<true>(av + j * vh);
              d = d + cmul_conj(cx<double>{w.x, w.y}, v[j]);
            } else {
              d = d + cmul_conj(v[j], s[j]);
            }
          }
          ps[0].add(d.r);
          ps[NV > 1 ? 1 : 0].add(d.i);
        }
      }
    }
  }
  if (RED != R_NONE) {
    double rv[NV];
#pragma unroll
    for (int k = 0; k < NV; ++k) rv[k] = ps[k].value();
    reduce_finalize<NV>(a.red, rhs, sb, a.nblk, nrhs, rv);
  }
}

// Whether (flags, reduction) has a fixed-point kernel, and its launch (its
// block size is its own; occ as in launch_hop).
bool fx_has(int flags, int red);
bool launch_hop_fx(int flags, int red, const HopArgs& a, int block, cudaStream_t st, int* occ);

}  // namespace bridge
