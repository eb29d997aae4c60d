// Integer form of the Wilson stencil for FP64 and float-float data (A = gamma5 (I - kappa D),
// the operator of wilson_core.cuh).
//
// GB300 issues 2 FP64 operations a clock and SM and 32 wide integer
// multiply-adds (32 x 32 + 64 -> 64 bits; both measured), so a hop's link
// product -- a sum of six real products an output, three multiply-adds a
// product -- costs a fifth as much in 60-bit fixed point as in FP64, and the
// additions almost nothing.  Every product and sum is exact but for the
// low-by-low digit product and two roundings at 2^-58 of the site's largest
// component.  In the norm of a site that is less than FP64's roundings; a
// component far below its site's or its neighbours' largest has fewer bits here
// than FP64 gives it, so that the stand-alone operator looks for such
// components (Witness) and takes their hops in FP64.  The CG loop, whose
// stopping test and solutions are bounded in the norm, does not.
//
// Format.  The 24 reals of a site share one exponent e with every |v| < 2^e;
// a real is the integer X = round(v 2^(59 - e)), |X| <= 2^59, kept as two
// balanced 30-bit digits X = hi 2^30 + lo, |hi| <= 2^29, -2^29 <= lo < 2^29.
// Values within 2^-6 of the site's largest keep all 53 bits; smaller ones
// are rounded at 2^-60 of the largest.  Link entries are X = round(u 2^59)
// (the rows and columns of a usable link have unit length, see
// pack_links_fix_kernel, so |u| <= 1).  A complex number is an int4
// (re.hi, re.lo, im.hi, im.lo): 16 bytes, as in FP64.
//
// One hop.  The spin projection adds digits without carries (|digit| <=
// 2^30).  With h the projected row, each real output is
//   hh = sum u.hi h.hi,  x = sum u.hi h.lo + u.lo h.hi   (|.| < 2^62.6)
//   T  = hh + (x >> 30)          in units 2^(e - 58), |T| <= 4.9 2^58
// (4.9 = sqrt(3) 2 sqrt(2): unit rows of U), then T >> (E - e + 1) with E the
// largest exponent of the eight neighbours, rounded: units 2^(E - 57), and
// the eight hops sum below 2^62.3.  Integer sums do not depend on their
// order, so every split of the hops over warps gives the same bits.
#pragma once

#include "floatfloat.cuh"
#include "internal.h"
#include "wilson_core.cuh"

namespace ssqcd {
namespace wfix {

constexpr int kZeroExp = -3000;      // exponent of a site of zeros
constexpr int kMaxExp = 800;         // sites above 2^800, infinities and NaN: kSpecialExp
constexpr int kSpecialExp = 1 << 20;
constexpr int kFixSites = 16;        // sites a warp covers; half-warp r takes spin row r

// ---- conversion -----------------------------------------------------------------------
__device__ __forceinline__ int exp_field(double v) { return (__double2hiint(v) >> 20) & 0x7ff; }
// key of a real in the site maximum: the IEEE bits of |v| above bit 31
__device__ __forceinline__ int abs_key(double v) { return __double2hiint(v) & 0x7fffffff; }

// exponent of a site from the largest abs_key of its reals and whether any
// real is nonzero
__device__ __forceinline__ int site_exp(int key, bool nonzero) {
  const int ex = key >> 20;
  if (!nonzero) return kZeroExp;
  const int e = max(ex, 1) - 1022;
  return e > kMaxExp ? kSpecialExp : e;
}

// v to digits at exponent field exmax = e + 1022 (>= 1 and >= v's own)
__device__ __forceinline__ int2 to_digits(double v, int exmax) {
  const int hw = __double2hiint(v);
  const int ex = (hw >> 20) & 0x7ff;
  unsigned long long m = (unsigned long long)(((unsigned)hw & 0xfffffu) | (ex ? 0x100000u : 0u)) << 32 |
                         (unsigned)__double2loint(v);
  m <<= 6;
  const int d = min(exmax - max(ex, 1), 63);
  m = (m + ((1ull << d) >> 1)) >> d;
  const long long sg = (long long)(hw >> 31);
  const long long x = ((long long)m ^ sg) - sg + (1ll << 29);
  return make_int2((int)(x >> 30), (int)((unsigned)x & 0x3fffffffu) - (1 << 29));
}
__device__ __forceinline__ int4 to_digits(double2 v, int exmax) {
  const int2 a = to_digits(v.x, exmax), b = to_digits(v.y, exmax);
  return make_int4(a.x, a.y, b.x, b.y);
}

__device__ __forceinline__ int4 to_site_digits(double2 v, int e) { return to_digits(v, e + 1022); }

// Float-float reals (hi + lo): the site exponent from the hi parts, and the
// digits as the sum of both parts' integers (exact above 2^-60 of the site's
// largest).
__device__ __forceinline__ long long float_to_fix(float v, int exmax) {
  const int b = __float_as_int(v), ex = (b >> 23) & 0xff;
  const unsigned long long m = (unsigned long long)((b & 0x7fffff) | (ex ? 0x800000 : 0)) << 35;
  const int d = min(exmax - max(ex, 1), 63);
  const long long x = (long long)((m + ((1ull << d) >> 1)) >> d);
  const long long sg = b >> 31;
  return (x ^ sg) - sg;
}
__device__ __forceinline__ int2 to_digits(float hi, float lo, int exmax) {
  const long long x = float_to_fix(hi, exmax) + float_to_fix(lo, exmax) + (1ll << 29);
  return make_int2((int)(x >> 30), (int)((unsigned)x & 0x3fffffffu) - (1 << 29));
}
__device__ __forceinline__ int4 to_site_digits(float4 v, int e) {
  const int2 a = to_digits(v.x, v.z, e + 126), b = to_digits(v.y, v.w, e + 126);
  return make_int4(a.x, a.y, b.x, b.y);
}

// Four lanes a site (lane = 8 q + j: spin q of site j of eight), three
// components each: the site's word, 16 e + one bit a spin that is not zero
// throughout, the same in its four lanes.
constexpr int kSpinBits = 4;
__device__ __forceinline__ int word_exp(int word) { return word >> kSpinBits; }
__device__ __forceinline__ void site_key(const double2& v, int& key, int& low) {
  key = max(key, max(abs_key(v.x), abs_key(v.y)));
  low |= __double2loint(v.x) | __double2loint(v.y);
}
__device__ __forceinline__ void site_key(const float4& v, int& key, int&) {
  key = max(key, max(__float_as_int(v.x) & 0x7fffffff, __float_as_int(v.y) & 0x7fffffff));
}
__device__ __forceinline__ int key_exp(double2, int key, int nz) { return site_exp(key, nz != 0); }
__device__ __forceinline__ int key_exp(float4, int key, int) {
  const int ex = key >> 23;
  return key == 0 ? kZeroExp : ex == 255 ? kSpecialExp : max(ex, 1) - 126;
}
template <typename V2>
__device__ __forceinline__ int quad_site_word(const V2 (&v)[3], int q) {
  int key = 0, low = 0;
#pragma unroll
  for (int a = 0; a < 3; ++a) site_key(v[a], key, low);
  int nz = (key | low) != 0 ? 1 << q : 0;
#pragma unroll
  for (int o = 8; o <= 16; o <<= 1) {
    key = max(key, __shfl_xor_sync(0xffffffffu, key, o));
    nz |= __shfl_xor_sync(0xffffffffu, nz, o);
  }
  return key_exp(v[0], key, nz) << kSpinBits | nz;
}

// ---- layout -----------------------------------------------------------------------------
// Tiles of 16 consecutive sites, so that every component of a site lies at a
// constant distance from its first one (one address a hop, the loads take
// their offsets as immediates): fields [f][tile][12][16] int4, links
// [mu][tile][9][16] int4, site words (exponents) [f][tile 16].
constexpr int kTile = kFixSites;
__host__ __device__ __forceinline__ int fix_tiles(int V) { return (V + kTile - 1) / kTile; }
__device__ __forceinline__ size_t field_at(int tiles, size_t f, int s) {
  return ((f * tiles + (s >> 4)) * 12) * kTile + (s & 15);
}
__device__ __forceinline__ size_t link_at(int tiles, int mu, int s) {
  return (((size_t)mu * tiles + (s >> 4)) * 9) * kTile + (s & 15);
}

// ---- one hop of one spin row --------------------------------------------------------------
struct Acc3 {
  long long re[3], im[3];
};

__device__ __forceinline__ void mad(long long& acc, int a, int b) { acc += (long long)a * b; }
__device__ __forceinline__ int4 load4(const int4* p) {
  int4 v;
  asm volatile("ld.global.nc.v4.s32 {%0, %1, %2, %3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "l"(p));
  return v;
}

// x + l or x - l for m = 0 or -1
__device__ __forceinline__ int add_signed(int x, int l, int m) { return x + (l ^ m) - m; }
__device__ __forceinline__ void acc_signed(long long& acc, long long x, int m) {
  const long long mm = m;
  acc += (x ^ mm) - mm;
}

// -1 where the entry of B_mu in row r is -1 or -i, else 0
__device__ __forceinline__ int b_sign(int mu, int r) { return (mu == 1 && r == 0) || (mu == 2 && r == 1) ? -1 : 0; }
// -1 where row r's share of the lower spins takes the factor -1 or -i of B^H
__device__ __forceinline__ int eta_sign(int mu, int r) { return mu == 0 || (mu != 3 && r == 0) ? -1 : 0; }

// The operands of one hop of a spin row r: the neighbour's components of spin r
// and of B's column, and the link.
struct HopData {
  int4 p[3], q[3], g[9];
};
template <bool SHARED>
__device__ __forceinline__ void hop_fetch(const int4* u, const int4* x, const int4* l, HopData& d) {
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    d.p[a] = SHARED ? x[a * kTile] : load4(x + a * kTile);
    d.q[a] = SHARED ? l[a * kTile] : load4(l + a * kTile);
  }
#pragma unroll
  for (int e = 0; e < 9; ++e) d.g[e] = SHARED ? u[e * kTile] : load4(u + e * kTile);
}

// w = U h (BACK = false) or U^H h (BACK = true) for spin row r of the projected
// half spinor h = psi_r -+ (B_mu psi_l)_r at the neighbour, negated if neg,
// shifted right by sh (1 .. 62) with rounding.  MU < 0: the direction is the
// run-time value mu_rt (one copy of the code for all four).
template <int MU, bool BACK>
__device__ __forceinline__ void hop_math(const HopData& d, int mu_rt, int r, bool neg, int sh, Acc3& w) {
  const int mu = MU < 0 ? mu_rt : MU;
  const bool swap = (mu & 1) == 0;  // entries +-i (mu = 0, 2), else +-1
  const int m = BACK ? b_sign(mu, r) : ~b_sign(mu, r);
  const int4(&p)[3] = d.p;
  const int4(&q)[3] = d.q;
  const int4(&g)[9] = d.g;
  int4 h[3];
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    h[a].x = add_signed(p[a].x, swap ? q[a].z : q[a].x, swap ? ~m : m);
    h[a].y = add_signed(p[a].y, swap ? q[a].w : q[a].y, swap ? ~m : m);
    h[a].z = add_signed(p[a].z, swap ? q[a].x : q[a].z, m);
    h[a].w = add_signed(p[a].w, swap ? q[a].y : q[a].w, m);
  }
  if (MU < 0 || MU == 3) {
    if (neg) {
#pragma unroll
      for (int a = 0; a < 3; ++a) h[a] = make_int4(-h[a].x, -h[a].y, -h[a].z, -h[a].w);
    }
  }
  // the part of h whose products enter with a minus sign, negated once
  int nh[3], nl[3];
#pragma unroll
  for (int b = 0; b < 3; ++b) {
    nh[b] = BACK ? -h[b].x : -h[b].z;
    nl[b] = BACK ? -h[b].y : -h[b].w;
  }
  const long long half = (1ll << sh) >> 1;
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    long long hr = half, hi = half, xr = 1ll << 29, xi = 1ll << 29;
#pragma unroll
    for (int b = 0; b < 3; ++b) {
      const int4 c = g[BACK ? b * 3 + a : a * 3 + b];
      mad(hr, c.x, h[b].x);
      mad(hi, c.x, h[b].z);
      mad(xr, c.x, h[b].y);
      mad(xi, c.x, h[b].w);
      mad(hr, c.z, BACK ? h[b].z : nh[b]);
      mad(hi, c.z, BACK ? nh[b] : h[b].x);
      mad(xr, c.y, h[b].x);
      mad(xi, c.y, h[b].z);
      mad(xr, c.z, BACK ? h[b].w : nl[b]);
      mad(xi, c.z, BACK ? nl[b] : h[b].y);
      mad(xr, c.w, BACK ? h[b].z : nh[b]);
      mad(xi, c.w, BACK ? nh[b] : h[b].x);
    }
    w.re[a] = (hr + (xr >> 30)) >> sh;
    w.im[a] = (hi + (xi >> 30)) >> sh;
  }
}

// Evidence that the terms of a component's hop sum are not all far below 2^E,
// the scale of the sum's roundings: the largest (as an OR) of its shares from the
// hops, for the three colours of upper spin r and of lower spin 2 + r.  The roundings stay
// below 48 units of 2^(E - 57) (six a hop), ~2 in the root mean square; a share of 2^52
// units and more bounds them by 2^-46, ~2^-51, of the sum of the terms' sizes, where FP64's
// own bound is ~2^-49.  Dense fields always have it: the sixteen reals of a
// component would all have to be below a fourteenth of their spread.
template <bool ON>
struct Witness {
  unsigned up[ON ? 3 : 1] = {}, lo[ON ? 3 : 1] = {};
  // a hop of direction 0 or 1 (both for spin row r: crossed later) or 2 or 3
  template <bool LOWER>
  __device__ __forceinline__ void add(const Acc3& w) {
    if constexpr (ON) {
#pragma unroll
      for (int a = 0; a < 3; ++a) {
        const int re = (int)(w.re[a] >> 32), im = (int)(w.im[a] >> 32);
        const unsigned x = (unsigned)(re ^ (re >> 31)) | (unsigned)(im ^ (im >> 31));
        up[a] |= x;
        if constexpr (LOWER) lo[a] |= x;
      }
    }
  }
  // after directions 0 and 1, which feed lower spin 3 - r: hand over what they gave
  __device__ __forceinline__ void cross() {
    if constexpr (ON) {
#pragma unroll
      for (int a = 0; a < 3; ++a) lo[a] = __shfl_xor_sync(0xffffffffu, up[a], 16);
    }
  }
};
constexpr unsigned kWitnessBits = ~((1u << 20) - 1);  // of the words above: 2^52 and more
// Whether the upper spin r (lower: 2 + r) gets a hop from a spin that is not zero:
// spin row r takes spins r and 2 + r (directions 2 and 3) or 3 - r (0 and 1) and
// feeds spins r and 2 + r, or 3 - r.
__device__ __forceinline__ bool any_hop(const int (&spins)[2], int r, bool lower) {
  const int a = lower ? 1 << (1 - r) | 4 << r : 1 << r | 8 >> r;
  return ((spins[0] & a) | (spins[1] & (5 << r))) != 0;
}

// neighbour of s in direction mu, forward or backward
template <bool BACK>
__device__ __forceinline__ int neighbour_rt(int s, const wcore::Coords& c, const Geometry& g, int mu, bool& twrap) {
  const int x = mu == 0 ? c.x : mu == 1 ? c.y : mu == 2 ? c.z : c.t;
  const int n = mu == 0 ? g.X : mu == 1 ? g.Y : mu == 2 ? g.Z : g.T;
  const int st = mu == 0 ? 1 : mu == 1 ? g.X : mu == 2 ? g.X * g.Y : g.X * g.Y * g.Z;
  const bool wrap = BACK ? x == 0 : x == n - 1;
  twrap = mu == 3 && wrap;
  if (BACK) return wrap ? s + (n - 1) * st : s - st;
  return wrap ? s - (n - 1) * st : s + st;
}

// Neighbour table of a lattice, [tile][8][16]: the site of hop 2 mu + (0
// forward, 1 backward), with kNegBit where the hop crosses an antiperiodic t
// boundary.
constexpr int kNegBit = 1 << 30;
__device__ __forceinline__ const int* nbr_at(const int* __restrict__ nbr, int s) {
  return nbr + (size_t)(s >> 4) * (8 * kTile) + (s & 15);
}

// The integer stencil's view of a lattice and of one field.
struct FixView {
  const int4* __restrict__ u;    // links
  const int* __restrict__ nbr;   // neighbour table
  const int4* __restrict__ dig;  // the field's digits
  const int* __restrict__ ex;    // its site words
  int tiles;
};

// Neighbours of a site, the shifts of their hops and the largest of their
// exponents (special, above kMaxExp, as well when the site's own value is).
struct Hops {
  int nb[8];
  unsigned sh[2];  // eight shifts of a byte
  int E;
  int spins[2];    // bits of the spins that are not zero in the hops of directions 0 and 1, 2 and 3
};
// In two parts: the copies or loads of the hops' operands need the neighbours
// alone, so that they are under way while the exponents come.
__device__ __forceinline__ void load_neighbours(const FixView& v, int s, Hops& h) {
  const int* t = nbr_at(v.nbr, s);
#pragma unroll
  for (int k = 0; k < 8; ++k) h.nb[k] = __ldg(t + k * kTile);
}
__device__ __forceinline__ void load_exponents(const FixView& v, int s, Hops& h) {
  int e[8];
  const int own = word_exp(__ldg(v.ex + s));
#pragma unroll
  for (int k = 0; k < 8; ++k) e[k] = __ldg(v.ex + (h.nb[k] & (kNegBit - 1)));
  h.spins[0] = e[0] | e[1] | e[2] | e[3];
  h.spins[1] = e[4] | e[5] | e[6] | e[7];
#pragma unroll
  for (int k = 0; k < 8; ++k) e[k] = word_exp(e[k]);
  h.E = kZeroExp;
#pragma unroll
  for (int k = 0; k < 8; ++k) h.E = max(h.E, e[k]);
  h.sh[0] = h.sh[1] = 0;
#pragma unroll
  for (int k = 0; k < 8; ++k) h.sh[k >> 2] |= (unsigned)min(h.E - e[k] + 1, 62) << (8 * (k & 3));
  if (own > kMaxExp) h.E = own;
}

// The operands of one hop of direction mu at site s from global memory.
template <bool BACK>
__device__ __forceinline__ void hop_fetch_at(const FixView& v, int s, int nbe, int mu, int r, HopData& d) {
  const int nb = nbe & (kNegBit - 1);
  const int lr = mu < 2 ? 1 - r : r;
  const int4* x = v.dig + (size_t)(nb >> 4) * (12 * kTile) + (nb & 15);
  hop_fetch<false>(v.u + link_at(v.tiles, mu, BACK ? nb : s), x + r * 3 * kTile, x + (6 + lr * 3) * kTile, d);
}

// up += w, d += -+ eta i^swap w (forward, backward): one hop's share of the
// upper spin r and of the lower spin that spin row r feeds
template <bool BACK>
__device__ __forceinline__ void add_hop(const Acc3& w, int mu, int r, Acc3& up, Acc3& d) {
  const bool swap = (mu & 1) == 0;
  const int m = BACK ? eta_sign(mu, r) : ~eta_sign(mu, r);
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    up.re[a] += w.re[a];
    up.im[a] += w.im[a];
    acc_signed(d.re[a], swap ? w.im[a] : w.re[a], swap ? ~m : m);
    acc_signed(d.im[a], swap ? w.re[a] : w.im[a], m);
  }
}

__device__ __forceinline__ void clear(Acc3& x) {
#pragma unroll
  for (int a = 0; a < 3; ++a) x.re[a] = x.im[a] = 0;
}
// directions 0 and 1 of half-warp r feed lower spin 1 - r: hand them over
__device__ __forceinline__ void cross_over(Acc3& d) {
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    d.re[a] = __shfl_xor_sync(0xffffffffu, d.re[a], 16);
    d.im[a] = __shfl_xor_sync(0xffffffffu, d.im[a], 16);
  }
}

// ---- all eight hops in one warp, fed by asynchronous copies ----------------------------------
// The operands of a hop (the neighbour's twelve components, the link's nine
// elements: 21 rows of 16 sites) are copied to shared memory two hops ahead,
// so that the copies' latency is hidden without registers to hold them: with
// the loads in registers a warp waited ~1600 of the ~3700 cycles of a hop.
constexpr int kStageRows = 21;
constexpr int kStageElems = kStageRows * kTile;    // int4 a stage
constexpr int kWarpStages = 2 * kStageElems;       // int4 a warp

__device__ __forceinline__ void copy16(int4* to, const int4* from) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 16;" ::"r"((unsigned)__cvta_generic_to_shared(to)), "l"(from)
               : "memory");
}
__device__ __forceinline__ void copy_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void copy_wait() {
  asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}

// start the copies of hop K (2 mu + backward) of the warp's sites; half-warp r
// takes six components of each site and half of the link's elements
template <int K>
__device__ __forceinline__ void stage_hop(const FixView& v, int s, int nbe, int i, int r, int4* buf) {
  const int nb = nbe & (kNegBit - 1);
  const int4* d = v.dig + (size_t)(nb >> 4) * (12 * kTile) + (nb & 15) + r * 6 * kTile;
  const int4* u = v.u + link_at(v.tiles, K >> 1, (K & 1) ? nb : s) + r * 5 * kTile;
  int4* bd = buf + r * 6 * kTile + i;
  int4* bu = buf + (12 + r * 5) * kTile + i;
#pragma unroll
  for (int a = 0; a < 6; ++a) copy16(bd + a * kTile, d + a * kTile);
#pragma unroll
  for (int e = 0; e < 4; ++e) copy16(bu + e * kTile, u + e * kTile);
  if (r == 0) copy16(bu + 4 * kTile, u + 4 * kTile);
  copy_commit();
}

// the arithmetic of hop K from its stage
template <int K, bool WIT>
__device__ __forceinline__ void staged_hop(const int4* buf, int nbe, int sh, int i, int r, Acc3& up, Acc3& d,
                                           Witness<WIT>& wit) {
  constexpr int MU = K >> 1;
  constexpr bool BACK = (K & 1) != 0;
  const int lr = MU < 2 ? 1 - r : r;
  HopData o;
  Acc3 w;
  hop_fetch<true>(buf + 12 * kTile + i, buf + r * 3 * kTile + i, buf + (6 + lr * 3) * kTile + i, o);
  hop_math<MU, BACK>(o, MU, r, (nbe & kNegBit) != 0, sh, w);
  wit.template add<(MU >= 2)>(w);
  add_hop<BACK>(w, MU, r, up, d);
}

template <int K, bool WIT, typename Last>
__device__ __forceinline__ void pipe_hops(const FixView& v, int s, int i, int r, const Hops& h, int4* buf, Acc3& up,
                                          Acc3& lo, Witness<WIT>& wit, Last last) {
  if constexpr (K < 8) {
    copy_wait<1>();
    __syncwarp();
    staged_hop<K>(buf + (K & 1) * kStageElems, h.nb[K], (int)(h.sh[K >> 2] >> (8 * (K & 3))) & 0xff, i, r, up, lo,
                  wit);
    __syncwarp();
    if constexpr (K + 2 < 8)
      stage_hop<K + 2>(v, s, h.nb[K + 2], i, r, buf + (K & 1) * kStageElems);
    else if constexpr (K + 2 == 8)
      last(buf + (K & 1) * kStageElems);  // commits a group of its own
    else
      copy_commit();
    if constexpr (K == 3) {
      cross_over(lo);
      wit.cross();
    }
    pipe_hops<K + 1>(v, s, i, r, h, buf, up, lo, wit, last);
  }
}

// The eight hops of the warp's 16 sites, whose neighbours are loaded (the
// exponents are loaded here); last(stage) starts the copy of what
// the caller needs after them (committed, complete after copy_wait<1>).
template <bool WIT, typename Last>
__device__ __forceinline__ void hop_sums_piped(const FixView& v, int s, int i, int r, Hops& h, int4* buf,
                                               Acc3& up, Acc3& lo, Witness<WIT>& wit, Last last) {
  clear(up);
  clear(lo);
  stage_hop<0>(v, s, h.nb[0], i, r, buf);
  stage_hop<1>(v, s, h.nb[1], i, r, buf + kStageElems);
  load_exponents(v, s, h);
  pipe_hops<0>(v, s, i, r, h, buf, up, lo, wit, last);
}

// Hop sums of one of four warps (sub: its direction, both hops) for spin row r
// of site s: up = upper output spin r, lo = lower output spin r, both in units
// 2^(E - 57).  The direction is a run-time value, since warps that each run
// their own copy of the code stall on instruction fetches.  All lanes of the
// warp take part.
template <bool WIT>
__device__ __forceinline__ void hop_sums(const FixView& v, int s, int r, int sub, Hops& h, Acc3& up, Acc3& lo,
                                         Witness<WIT>& wit) {
  clear(up);
  clear(lo);
  const int mu = sub;
  const int nf = mu == 0 ? h.nb[0] : mu == 1 ? h.nb[2] : mu == 2 ? h.nb[4] : h.nb[6];
  const int nb = mu == 0 ? h.nb[1] : mu == 1 ? h.nb[3] : mu == 2 ? h.nb[5] : h.nb[7];
  HopData d;
  hop_fetch_at<false>(v, s, nf, mu, r, d);
  load_exponents(v, s, h);
  const unsigned s2 = (mu < 2 ? h.sh[0] : h.sh[1]) >> (16 * (mu & 1));
  const int sf = s2 & 0xff, sb = (s2 >> 8) & 0xff;
  Acc3 w;
  hop_math<-1, false>(d, mu, r, (nf & kNegBit) != 0, sf, w);
  wit.template add<true>(w);
  add_hop<false>(w, mu, r, up, lo);
  hop_fetch_at<true>(v, s, nb, mu, r, d);
  hop_math<-1, true>(d, mu, r, (nb & kNegBit) != 0, sb, w);
  wit.template add<true>(w);
  add_hop<true>(w, mu, r, up, lo);
  if (mu < 2) {
    cross_over(lo);
    wit.cross();
  }
}

// Launch shapes for W = 1 or 4 warps a site group: threads a block, (site group,
// rhs) units a block, and the blocks an SM that the registers are capped for
// (the fastest of those tried: W = 1 at 3, 4, 5 blocks 368, 326, 386 us for 16^3 x
// 32 x 8; W = 4 at 7, 6, 5 24.9, 24.1, 23.7 us an iteration of 8^4 x 2).
constexpr int kFixThreads = 128;
__host__ __device__ constexpr int fix_units(int W) { return kFixThreads / 32 / W; }
__host__ __device__ constexpr int fix_min_blocks(int W) { return W == 1 ? 4 : 5; }

// psi - kappa D psi from a hop sum T in units 2^(E - 57): the sum is made a
// double times 2^-200 (exact up to its rounding: |T| < 2^63) and the factor
// -kappa 2^(E + 143) is a normal number for every E.
__device__ __forceinline__ double hop_factor(int E, double mkappa) {
  const int k = E == kZeroExp || E > kMaxExp ? 0 : E + 143;
  return mkappa * __hiloint2double((k + 1023) << 20, 0);
}
// t 2^-200 rounded to nearest (halves away from zero), put together from
// integers: the conversion instruction takes two of the FP64 pipe's slots, 128
// cycles of a warp, which was half of that pipe's work in the CG loop's stencil.
__device__ __forceinline__ double scaled_double(long long t) {
  const long long sign = t >> 63;
  const unsigned long long a = (unsigned long long)((t ^ sign) - sign);
  unsigned hi = (unsigned)(a >> 32), lo = (unsigned)a;
  const bool low = hi == 0;
  hi = low ? lo : hi;
  lo = low ? 0u : lo;
  const int n = __clz((int)hi);  // 32: t = 0
  const unsigned uh = __funnelshift_l(lo, hi, n), ul = __funnelshift_l(0u, lo, n);
  // the leading one lies at bit 52 and adds one to the exponent field, as does a carry out of the rounding
  const unsigned long long m =
      ((unsigned long long)((uh >> 11) + ((unsigned)((low ? 853 : 885) - n) << 20)) << 32 | __funnelshift_r(ul, uh, 11)) +
      (ul >> 10 & 1);
  const unsigned top = (uh == 0 ? 0u : (unsigned)(m >> 32)) | ((unsigned)sign & 0x80000000u);
  return __hiloint2double((int)top, (int)(unsigned)m);
}
// INT: by integers, else by the conversion instruction and its exponent field lowered
template <bool INT>
__device__ __forceinline__ double hop_finish(double f, long long t, double psi) {
  if (INT) return fma(f, scaled_double(t), psi);
  const double d = (double)t;
  const int hw = __double2hiint(d);
  return fma(f, __hiloint2double(t == 0 ? hw : hw - (200 << 20), __double2loint(d)), psi);
}

// The same for float-float fields: a hop sum T 2^(E - 57) as float-float, from
// its three 21-bit parts (exact in FP32), scaled in two steps.
__device__ __forceinline__ float pow2f(int k) { return __int_as_float((k + 127) << 23); }
__device__ __forceinline__ float2 hop_ff(long long t, float s1, float s2) {
  const float a = (float)(int)(t >> 42) * 0x1p42f, b = (float)((int)(t >> 21) & 0x1fffff) * 0x1p21f;
  const float c = (float)((int)t & 0x1fffff);
  float s, e, h, l;
  ff::fast_two_sum(a, b, s, e);
  ff::fast_two_sum(s, __fadd_rn(e, c), h, l);
  return make_float2(h * s1 * s2, l * s1 * s2);
}
__device__ __forceinline__ float4 hop_cff(longlong2 t, int E) {
  const int k = E == kZeroExp ? 0 : E - 57, k1 = k / 2;
  const float s1 = pow2f(k1), s2 = pow2f(k - k1);
  return ff::make(hop_ff(t.x, s1, s2), hop_ff(t.y, s1, s2));
}

}  // namespace wfix
}  // namespace ssqcd
