// Staggered operator kernels.
//
// Operator (Sec. 2 of the paper implements the staggered action and its
// even-odd blocks, Eq. 1; the formula is the textbook Kogut-Susskind one):
//   D chi(x) = m chi(x) + (1/2) sum_mu eta_mu(x) [ U_mu(x) chi(x + mu)
//                                               - U_mu(x - mu)^dagger chi(x - mu) ]
// with eta_0 = 1, eta_1 = (-1)^x, eta_2 = (-1)^(x+y), eta_3 = (-1)^(x+y+z) and
// the boundary phase bc[mu] on every hop that wraps.  The phases are applied
// in the kernel; the links are the same stored links as for Wilson (FP64 18
// reals, FP32 12 reals with row 2 rebuilt in registers).
//
// Field layout: a half-lattice colour vector is three 8-byte (FP32) or
// 16-byte (FP64) planes, one complex colour component each, addressed
// base + (k * Vh + ih) * size, so a warp reads contiguous bytes per plane.
//
// One thread computes one output site of one right-hand side:
//   out = scale * sum_mu eta_mu [U chi(x+mu) - U^dag chi(x-mu)] + s1 self + caux aux
// with an optional fused reduction of |out|^2 or Re <self, out>.
#pragma once

#include "dslash_fx.cuh"
#include "reduce.cuh"

namespace bridge {

BR_HD long stag_site_bytes(int prec) { return prec == P_F64 ? 48 : 24; }
BR_HD long stag_block_bytes(int prec, long vh) { return pad256(stag_site_bytes(prec) * vh); }

template <int P>
BR_D void load_cvec(const char* base, long vh, uint32_t i, cx<typename Tr<P>::R> v[3]) {
  if constexpr (P == P_F64) {
    const double2* p = reinterpret_cast<const double2*>(base);
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      const double2 w = __ldg(p + k * vh + i);
      v[k] = {w.x, w.y};
    }
  } else {
    const float2* p = reinterpret_cast<const float2*>(base);
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      const float2 w = __ldg(p + k * vh + i);
      v[k] = {w.x, w.y};
    }
  }
}

// Plain (coherent) load, for vectors this kernel also writes.
template <int P>
BR_D void load_cvec_rw(const char* base, long vh, uint32_t i, cx<typename Tr<P>::R> v[3]) {
  if constexpr (P == P_F64) {
    const double2* p = reinterpret_cast<const double2*>(base);
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      const double2 w = p[k * vh + i];
      v[k] = {w.x, w.y};
    }
  } else {
    const float2* p = reinterpret_cast<const float2*>(base);
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      const float2 w = p[k * vh + i];
      v[k] = {w.x, w.y};
    }
  }
}

template <int P>
BR_D void store_cvec(char* base, long vh, uint32_t i, const cx<typename Tr<P>::R> v[3]) {
  if constexpr (P == P_F64) {
    double2* p = reinterpret_cast<double2*>(base);
#pragma unroll
    for (int k = 0; k < 3; ++k) p[k * vh + i] = make_double2(v[k].r, v[k].i);
  } else {
    float2* p = reinterpret_cast<float2*>(base);
#pragma unroll
    for (int k = 0; k < 3; ++k) p[k * vh + i] = make_float2(v[k].r, v[k].i);
  }
}

enum StagRed { SR_NONE = 0, SR_NORM = 1, SR_DOT_SELF = 2 };

struct StagArgs {
  Geom g;
  int out_parity, nrhs, nblk;
  double scale, s1, caux;
  float scalef, s1f, cauxf;
  double bc[4];
  float bcf[4];
  char* out;
  long out_rs;
  const char* in;
  long in_rs;
  const char* self;  // may be null
  long self_rs;
  const char* aux;   // may be null
  long aux_rs;
  const char* gauge;  // [parity][mu] link blocks
  int fx;                // FP64: an FxMode, and for FX_COPIES the links and the input in fixed point
  const char* gauge_fx;
  const char* in_fx;
  long in_fx_rs;
  RedArgs red;
};

template <int P, int MU, bool FWD>
BR_D void stag_hop_one(const char* in, const char* lb, long vh, uint32_t nb, uint32_t li, bool wraps,
                       typename Tr<P>::R bc, typename Tr<P>::R eta, cx<typename Tr<P>::R> acc[3]) {
  using R = typename Tr<P>::R;
  cx<R> v[3];
  load_cvec<P>(in, vh, nb, v);
  Link<R> U;
  load_link<P, true>(lb, vh, li, U);
  const R f = (wraps ? bc : R(1)) * (FWD ? eta : -eta);
#pragma unroll
  for (int r = 0; r < 3; ++r) {
    cx<R> w;
    if (FWD)
      w = crow3(U.m[r][0], U.m[r][1], U.m[r][2], v);
    else
      w = crow3_conj(U.m[0][r], U.m[1][r], U.m[2][r], v);
    acc[r] = caxpy(f, w, acc[r]);
  }
}

template <int P, int MU>
BR_D void stag_dir(const StagArgs& a, const char* in, const char* g_out, const char* g_in, long lbb, uint32_t ih,
                   const int c[4], uint32_t xh, typename Tr<P>::R eta, cx<typename Tr<P>::R> acc[3]) {
  using R = typename Tr<P>::R;
  uint32_t f, b;
  bool wf, wb;
  neighbours<MU>(a.g, ih, c, xh, f, b, wf, wb);
  const R bc = pick<R>(a.bc[MU], a.bcf[MU]);
  stag_hop_one<P, MU, true>(in, g_out + MU * lbb, a.g.vh, f, ih, wf, bc, eta, acc);
  stag_hop_one<P, MU, false>(in, g_in + MU * lbb, a.g.vh, b, b, wb, bc, eta, acc);
}

// One output site: v, and s = the self vector (where there is one).
template <int P>
BR_D void stag_site(const StagArgs& a, int rhs, uint32_t ih, cx<typename Tr<P>::R> v[3], cx<typename Tr<P>::R> s[3]) {
  using R = typename Tr<P>::R;
  const int p = a.out_parity;
  const long vh = a.g.vh, lbb = link_block_bytes(P, vh);
  const char* g_out = a.gauge + (long)p * 4 * lbb;
  const char* g_in = a.gauge + (long)(1 - p) * 4 * lbb;
  const char* in = a.in + rhs * a.in_rs;
  const R sc = pick<R>(a.scale, a.scalef), s1 = pick<R>(a.s1, a.s1f), ca = pick<R>(a.caux, a.cauxf);
  int c[4];
  uint32_t xh;
  site_coords(a.g, ih, p, c, xh);
  cx<R> acc[3] = {czero<R>(), czero<R>(), czero<R>()};
  stag_dir<P, 0>(a, in, g_out, g_in, lbb, ih, c, xh, R(1), acc);
  stag_dir<P, 1>(a, in, g_out, g_in, lbb, ih, c, xh, (c[0] & 1) ? R(-1) : R(1), acc);
  stag_dir<P, 2>(a, in, g_out, g_in, lbb, ih, c, xh, ((c[0] + c[1]) & 1) ? R(-1) : R(1), acc);
  stag_dir<P, 3>(a, in, g_out, g_in, lbb, ih, c, xh, ((c[0] + c[1] + c[2]) & 1) ? R(-1) : R(1), acc);
#pragma unroll
  for (int k = 0; k < 3; ++k) v[k] = sc * acc[k];
  if (a.self != nullptr) {
    load_cvec<P>(a.self + rhs * a.self_rs, vh, ih, s);
#pragma unroll
    for (int k = 0; k < 3; ++k) v[k] = v[k] + s1 * s[k];
  }
  if (a.aux != nullptr) {
    cx<R> w[3];
    load_cvec<P>(a.aux + rhs * a.aux_rs, vh, ih, w);
#pragma unroll
    for (int k = 0; k < 3; ++k) v[k] = v[k] + ca * w[k];
  }
}

// One site's contribution to the fused reduction.
template <int RED, class R>
BR_D R stag_red(const cx<R> v[3], const cx<R> s[3]) {
  R n = 0;
#pragma unroll
  for (int k = 0; k < 3; ++k)
    n += RED == SR_NORM ? v[k].r * v[k].r + v[k].i * v[k].i : s[k].r * v[k].r + s[k].i * v[k].i;
  return n;
}

template <int P, int RED>
__global__ void __launch_bounds__(256) stag_hop_kernel(const StagArgs a) {
  using R = typename Tr<P>::R;
  const int nrhs = a.nrhs;
  const int rhs = blockIdx.x % nrhs;
  const int sb = blockIdx.x / nrhs;
  const long vh = a.g.vh;
  PartialSum<R> ps;
  const bool skip = a.red.check_done && a.red.cg != nullptr && a.red.cg[rhs].done != RUNNING;
  if (skip && all_finished(a.red, a.nrhs)) return;
  if (!skip) {
    const uint32_t stride = (uint32_t)a.nblk * blockDim.x;
    for (uint32_t ih = sb * blockDim.x + threadIdx.x; ih < (uint32_t)vh; ih += stride) {
      cx<R> v[3], s[3];
      stag_site<P>(a, rhs, ih, v, s);
      store_cvec<P>(a.out + rhs * a.out_rs, vh, ih, v);
      if (RED != SR_NONE) ps.add(stag_red<RED, R>(v, s));
    }
  }
  if (RED != SR_NONE) {
    double rv[1] = {ps.value()};
    reduce_finalize<1>(a.red, rhs, sb, a.nblk, nrhs, rv);
  }
}

// ------------------------------------------------------------ fixed point
// The FP64 hop in 64-bit fixed point, as dslash_fx.cuh: the same integer links,
// the colour vectors in units of 2^(E - 1081) with one exponent a site (three
// 16-byte planes, then one int a site), one rounding a hop, and the same test
// that every component is reached by a hop.  36 products of
// three IMAD.WIDE a hop; a site has nothing to project or reconstruct, so one
// thread a site keeps its sum, a hop's rows and both hops' loads of a direction
// in 128 registers.  Measured (one parity of 32^4): FP64 kernel 340 us, at the
// FP64 pipe's limit (0.90 TFLOP/s); here 130 us = 5.2 TB/s, 0.77 of the copy rate.
BR_HD long stag_fx_block_bytes(long vh) { return pad256(52 * vh); }
constexpr int SFX_THREADS = 128;

BR_D void stag_fx_store(char* block, long vh, uint32_t ih, const cx<double> v[3]) {
  uint4 w[3];
#pragma unroll
  for (int k = 0; k < 3; ++k)
    w[k] = make_uint4((uint32_t)__double2loint(v[k].r), (uint32_t)__double2hiint(v[k].r), (uint32_t)__double2loint(v[k].i),
                      (uint32_t)__double2hiint(v[k].i));
  const uint32_t m = fx_max_word<3>(w);
  const int E = (int)(m >> 20);
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    const long long r = fx_from_bits<6>(w[k].x, w[k].y, E, 0), i = fx_from_bits<6>(w[k].z, w[k].w, E, 0);
    reinterpret_cast<uint4*>(block)[k * vh + ih] =
        make_uint4((uint32_t)r, (uint32_t)(r >> 32), (uint32_t)i, (uint32_t)(i >> 32));
  }
  reinterpret_cast<int*>(block + 48 * vh)[ih] = fx_site_exponent(m);
}

// Slots of one site (direction 2 mu + backward): neighbour index, bit 31 the
// sign of the hop (staggered and boundary phase, - for backward), exponent.
template <int MU, bool RAW>
BR_D void stag_fx_slots(const StagArgs& a, const char* in, uint32_t ih, const int c[4], uint32_t xh, uint32_t eta_neg,
                        uint2 (*w)[SFX_THREADS], int& Ea, bool& bad) {
  uint32_t f, b;
  bool wf, wb;
  neighbours<MU>(a.g, ih, c, xh, f, b, wf, wb);
  const uint32_t neg = a.bcf[MU] < 0.f;
  const int* ex = reinterpret_cast<const int*>(in + 48 * a.g.vh);
  const int ef = RAW ? fx_exponent<3>(in, a.g.vh, f) : __ldg(ex + f), eb = RAW ? fx_exponent<3>(in, a.g.vh, b) : __ldg(ex + b);
  bad = bad || ef < 0 || eb < 0;
  Ea = max(Ea, max(ef, eb));
  w[2 * MU][threadIdx.x] = make_uint2(f | ((eta_neg ^ (wf & neg)) << 31), (uint32_t)ef);
  w[2 * MU + 1][threadIdx.x] = make_uint2(b | ((eta_neg ^ (wb & neg) ^ 1u) << 31), (uint32_t)eb);
}

struct StagFxLoads {
  uint4 v[3], l[9];
};
BR_D void stag_fx_load(StagFxLoads& f, const char* in, const char* g, long vs, uint32_t nb, uint32_t li) {
#pragma unroll
  for (int k = 0; k < 3; ++k) f.v[k] = __ldg(reinterpret_cast<const uint4*>(in + k * vs) + nb);
#pragma unroll
  for (int k = 0; k < 9; ++k) f.l[k] = ldg4<true>(reinterpret_cast<const uint4*>(g + k * vs) + li);
}

// The hop's result is added to acc; returned: the components it reaches (fx_reaches).
template <bool FWD, bool RAW>
BR_D uint32_t stag_fx_mac(const StagFxLoads& f, uint2 w, int Ea, cx<long long> acc[3]) {
  long long rh[3] = {0, 0, 0}, rm[3] = {0, 0, 0}, jh[3] = {0, 0, 0}, jm[3] = {0, 0, 0};
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    const cx<long long> v = fx_value<RAW>(f.v[c], (int)w.y);
    const Fx2 hr = fx_split(v.r), hi = fx_split(v.i);
#pragma unroll
    for (int r = 0; r < 3; ++r) {
      const uint4 l = f.l[FWD ? 3 * r + c : 3 * c + r];
      const Fx2 ur = fx_limbs<RAW>(l.x, l.y, 1023), ui = fx_limbs<RAW>(l.z, l.w, 1023), nui = fx_neg(ui);
      fx_mac(ur, hr, rh[r], rm[r]);
      fx_mac(FWD ? nui : ui, hi, rh[r], rm[r]);
      fx_mac(ur, hi, jh[r], jm[r]);
      fx_mac(FWD ? ui : nui, hr, jh[r], jm[r]);
    }
  }
  const int d = min(Ea - (int)w.y, 62);  // a zero neighbour (exponent 0): rounds to zero
  const long long half = (1ll << d) >> 1;
  const int m = -(int)(w.x >> 31);
  uint32_t hit = 0;
#pragma unroll
  for (int r = 0; r < 3; ++r) {
    const cx<long long> u = {(rh[r] + fx_split(rm[r]).h + half) >> d, (jh[r] + fx_split(jm[r]).h + half) >> d};
    hit |= fx_reaches(u) << r;
    acc[r].r += fx_sign(u.r, m);
    acc[r].i += fx_sign(u.i, m);
  }
  return hit;
}

// The site in FP64, where a neighbour has no fixed-point form.
__device__ __noinline__ inline void stag_fx_site_fp64(const StagArgs& a, int rhs, uint32_t ih, double2* out) {
  cx<double> v[3], s[3];
  stag_site<P_F64>(a, rhs, ih, v, s);
#pragma unroll
  for (int k = 0; k < 3; ++k) out[k] = make_double2(v[k].r, v[k].i);
}

template <int RED, bool RAW>
__global__ void __launch_bounds__(SFX_THREADS, RAW ? 2 : 4) stag_hop_fx_kernel(const StagArgs a) {
  const int nrhs = a.nrhs;
  const int rhs = blockIdx.x % nrhs;
  const int sb = blockIdx.x / nrhs;
  const long vh = a.g.vh, vs = 16 * vh;
  __shared__ uint2 slot[8][SFX_THREADS];
  PartialSum<double> ps;
  const bool skip = a.red.check_done && a.red.cg != nullptr && a.red.cg[rhs].done != RUNNING;
  if (skip && all_finished(a.red, a.nrhs)) return;
  if (!skip) {
    const int p = a.out_parity;
    const long lbb = link_block_bytes(P_F64, vh);
    const char* g_out = (RAW ? a.gauge : a.gauge_fx) + (long)p * 4 * lbb;
    const char* g_in = (RAW ? a.gauge : a.gauge_fx) + (long)(1 - p) * 4 * lbb;
    const char* in = RAW ? a.in + rhs * a.in_rs : a.in_fx + rhs * a.in_fx_rs;
    const uint32_t stride = (uint32_t)a.nblk * SFX_THREADS;
    for (uint32_t ih = sb * SFX_THREADS + threadIdx.x; ih < (uint32_t)vh; ih += stride) {
      int Ea = 0;
      bool bad = false;
      {
        int c[4];
        uint32_t xh;
        site_coords(a.g, ih, p, c, xh);
        stag_fx_slots<0, RAW>(a, in, ih, c, xh, 0u, slot, Ea, bad);
        stag_fx_slots<1, RAW>(a, in, ih, c, xh, c[0] & 1, slot, Ea, bad);
        stag_fx_slots<2, RAW>(a, in, ih, c, xh, (c[0] + c[1]) & 1, slot, Ea, bad);
        stag_fx_slots<3, RAW>(a, in, ih, c, xh, (c[0] + c[1] + c[2]) & 1, slot, Ea, bad);
      }
      cx<double> v[3], s[3];
      if (a.self != nullptr) load_cvec<P_F64>(a.self + rhs * a.self_rs, vh, ih, s);
      cx<long long> acc[3] = {{0, 0}, {0, 0}, {0, 0}};
      if (!bad) {
        uint32_t reach = 0;
#pragma unroll 1
        for (int mu = 0; mu < 4; ++mu) {
          StagFxLoads f, b;
          const uint2 wf = slot[2 * mu][threadIdx.x], wb = slot[2 * mu + 1][threadIdx.x];
          const uint32_t nf = wf.x & 0x7fffffffu, nb = wb.x & 0x7fffffffu;
          stag_fx_load(f, in, g_out + mu * lbb, vs, nf, ih);
          stag_fx_load(b, in, g_in + mu * lbb, vs, nb, nb);
          reach |= stag_fx_mac<true, RAW>(f, wf, Ea, acc);
          reach |= stag_fx_mac<false, RAW>(b, wb, Ea, acc);
        }
        bad = Ea != 0 && reach != 0x3fu;
      }
      if (bad) {
        double2 w[3];
        stag_fx_site_fp64(a, rhs, ih, w);
#pragma unroll
        for (int k = 0; k < 3; ++k) v[k] = {w[k].x, w[k].y};
      } else {
        const double sc = Ea == 0 ? 0.0 : a.scale * fx_pow2(Ea - 54);
        cx<double> t[3];
#pragma unroll
        for (int k = 0; k < 3; ++k) t[k] = czero<double>();
        if (a.aux != nullptr) {
          load_cvec<P_F64>(a.aux + rhs * a.aux_rs, vh, ih, t);
#pragma unroll
          for (int k = 0; k < 3; ++k) t[k] = a.caux * t[k];
        }
#pragma unroll
        for (int k = 0; k < 3; ++k) {
          if (a.self != nullptr) t[k] = caxpy(a.s1, s[k], t[k]);
          v[k] = caxpy(sc, cx<double>{(double)acc[k].r, (double)acc[k].i}, t[k]);
        }
      }
      store_cvec<P_F64>(a.out + rhs * a.out_rs, vh, ih, v);
      if (RED != SR_NONE) ps.add(stag_red<RED, double>(v, s));
    }
  }
  if (RED != SR_NONE) {
    double rv[1] = {ps.value()};
    reduce_finalize<1>(a.red, rhs, sb, a.nblk, nrhs, rv);
  }
}

// FP64 colour vectors -> their fixed-point form.
__global__ void __launch_bounds__(256) stag_to_fx_kernel(const char* src, long src_rs, char* dst, long dst_rs, uint32_t vh,
                                                         int nrhs, int nblk, RedArgs red) {
  const int rhs = blockIdx.x % nrhs;
  if (rhs_finished(red, rhs)) return;
  for (uint32_t ih = (blockIdx.x / nrhs) * blockDim.x + threadIdx.x; ih < vh; ih += (uint32_t)nblk * blockDim.x) {
    cx<double> v[3];
    load_cvec<P_F64>(src + rhs * src_rs, vh, ih, v);
    stag_fx_store(dst + rhs * dst_rs, vh, ih, v);
  }
}

// ------------------------------------------------------------ vector kernels
enum StagVecOp {
  SV_CGUPD = 0,   // x += alpha p, r -= alpha q, |r|^2 -> FIN_CG_BETA
  SV_CGP = 1,     // p = r + beta p
  SV_NORM = 2,    // |a|^2 -> red.fin
  SV_CONVERT = 3, // b (precision PB) = mask ? a (precision P) : 0
  SV_ACCUM = 4    // b (FP64) += mask ? a : 0
};

struct StagVecArgs {
  uint32_t vh;
  int nrhs, nblk;
  char *a, *b, *c, *d;  // operands (see StagVecOp)
  long a_rs, b_rs, c_rs, d_rs;
  const int* mask;    // per rhs (may be null)
  RedArgs red;
};

template <int P, int PB, int OP>
__global__ void __launch_bounds__(256) stag_vec_kernel(const StagVecArgs a) {
  using R = typename Tr<P>::R;
  using RB = typename Tr<PB>::R;
  const int rhs = blockIdx.x % a.nrhs;
  const int sb = blockIdx.x / a.nrhs;
  PartialSum<R> ps;
  const bool skip = (OP == SV_CGUPD || OP == SV_CGP) && a.red.cg != nullptr && a.red.cg[rhs].done != RUNNING;
  const bool on = a.mask == nullptr || a.mask[rhs] != 0;
  if (skip && all_finished(a.red, a.nrhs)) return;
  if (!skip) {
    const uint32_t stride = (uint32_t)a.nblk * blockDim.x;
    for (uint32_t ih = sb * blockDim.x + threadIdx.x; ih < a.vh; ih += stride) {
      if (OP == SV_CGUPD) {
        const R alpha = (R)a.red.cg[rhs].alpha;
        cx<R> x[3], r[3], p[3], q[3];
        load_cvec_rw<P>(a.a + rhs * a.a_rs, a.vh, ih, x);
        load_cvec_rw<P>(a.b + rhs * a.b_rs, a.vh, ih, r);
        load_cvec<P>(a.c + rhs * a.c_rs, a.vh, ih, p);
        load_cvec<P>(a.d + rhs * a.d_rs, a.vh, ih, q);
        R n = 0;
#pragma unroll
        for (int k = 0; k < 3; ++k) {
          x[k] = x[k] + alpha * p[k];
          r[k] = r[k] - alpha * q[k];
          n += r[k].r * r[k].r + r[k].i * r[k].i;
        }
        store_cvec<P>(a.a + rhs * a.a_rs, a.vh, ih, x);
        store_cvec<P>(a.b + rhs * a.b_rs, a.vh, ih, r);
        ps.add(n);
      } else if (OP == SV_CGP) {
        const R beta = (R)a.red.cg[rhs].beta;
        cx<R> p[3], r[3];
        load_cvec_rw<P>(a.a + rhs * a.a_rs, a.vh, ih, p);
        load_cvec<P>(a.b + rhs * a.b_rs, a.vh, ih, r);
#pragma unroll
        for (int k = 0; k < 3; ++k) p[k] = r[k] + beta * p[k];
        store_cvec<P>(a.a + rhs * a.a_rs, a.vh, ih, p);
      } else if (OP == SV_NORM) {
        cx<R> v[3];
        load_cvec<P>(a.a + rhs * a.a_rs, a.vh, ih, v);
        R n = 0;
#pragma unroll
        for (int k = 0; k < 3; ++k) n += v[k].r * v[k].r + v[k].i * v[k].i;
        ps.add(n);
      } else if (OP == SV_CONVERT) {
        cx<R> v[3];
        cx<RB> w[3];
        load_cvec<P>(a.a + rhs * a.a_rs, a.vh, ih, v);
#pragma unroll
        for (int k = 0; k < 3; ++k) w[k] = on ? cx<RB>{(RB)v[k].r, (RB)v[k].i} : czero<RB>();
        store_cvec<PB>(a.b + rhs * a.b_rs, a.vh, ih, w);
      } else if (OP == SV_ACCUM) {
        if (!on) continue;
        cx<R> v[3];
        cx<double> w[3];
        load_cvec<P>(a.a + rhs * a.a_rs, a.vh, ih, v);
        load_cvec_rw<P_F64>(a.b + rhs * a.b_rs, a.vh, ih, w);
#pragma unroll
        for (int k = 0; k < 3; ++k) w[k] = w[k] + cx<double>{(double)v[k].r, (double)v[k].i};
        store_cvec<P_F64>(a.b + rhs * a.b_rs, a.vh, ih, w);
      }
    }
  }
  if (OP == SV_CGUPD || OP == SV_NORM) {
    double rv[1] = {ps.value()};
    reduce_finalize<1>(a.red, rhs, sb, a.nblk, a.nrhs, rv);
  }
}

// ------------------------------------------------------- canonical layout
// Canonical vectors are one 48-byte record a site; a block moves SC_SITES
// consecutive ones (whole lattices: both parities, which interleave) through
// shared memory, so that both sides are read and written by consecutive
// threads.  One thread a record ran at 2.4 TB/s, this at 4.9 TB/s (FP64, 32^4:
// 85 -> 41 us for both directions).
constexpr int SC_SITES = 256;

struct StagCanonArgs {
  Geom g;
  uint32_t vh;
  int nrhs;
  long V;
  int full;           // 1: canonical full-lattice vectors, 0: half-lattice ones
  double* canon;
  char *even, *odd;   // the parity blocks (half-lattice: `even`)
  long rs;
  char *fx, *fx2;     // from canonical FP64: the fixed-point form too (null: none), as even and odd
  long fx_rs;
};

// Parity block and half-lattice index of canonical site k.
BR_D int stag_where(const StagCanonArgs& a, long k, uint32_t& ih) {
  if (!a.full) {
    ih = (uint32_t)k;
    return 0;
  }
  int c[4];
  uint32_t xh;
  ih = (uint32_t)(k >> 1);
  site_coords(a.g, ih, 0, c, xh);
  return (int)(k & 1) ^ (c[0] & 1);
}

template <int P, bool TO_CANON>
__global__ void __launch_bounds__(SC_SITES) stag_canon_kernel(const StagCanonArgs a) {
  using R = typename Tr<P>::R;
  __shared__ double2 sh[3 * SC_SITES];
  double* flat = reinterpret_cast<double*>(sh);
  const int rhs = blockIdx.x % a.nrhs, t = threadIdx.x;
  const long n_sites = a.full ? a.V : (long)a.vh;
  const long base = (long)(blockIdx.x / a.nrhs) * SC_SITES;
  const int n = (int)min((long)SC_SITES, n_sites - base);
  double* canon = a.canon + ((long)rhs * n_sites + base) * 6;
  if (!TO_CANON) {
#pragma unroll
    for (int k = 0; k < 6; ++k)
      if (t + k * SC_SITES < 6 * n) flat[t + k * SC_SITES] = __ldg(canon + t + k * SC_SITES);
    __syncthreads();
  }
  if (t < n) {
    uint32_t ih;
    const int p = stag_where(a, base + t, ih);
    char* block = (p ? a.odd : a.even) + rhs * a.rs;
    cx<R> v[3];
    if (TO_CANON) {
      load_cvec<P>(block, a.vh, ih, v);
#pragma unroll
      for (int k = 0; k < 3; ++k) sh[3 * t + k] = make_double2((double)v[k].r, (double)v[k].i);
    } else {
#pragma unroll
      for (int k = 0; k < 3; ++k) {
        const double2 w = sh[3 * t + k];
        v[k] = {(R)w.x, (R)w.y};
      }
      store_cvec<P>(block, a.vh, ih, v);
      if constexpr (P == P_F64)
        if (a.fx) stag_fx_store((p ? a.fx2 : a.fx) + rhs * a.fx_rs, a.vh, ih, v);
    }
  }
  if (TO_CANON) {
    __syncthreads();
#pragma unroll
    for (int k = 0; k < 6; ++k)
      if (t + k * SC_SITES < 6 * n) canon[t + k * SC_SITES] = flat[t + k * SC_SITES];
  }
}

}  // namespace bridge
