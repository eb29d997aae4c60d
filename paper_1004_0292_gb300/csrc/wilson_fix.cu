// Stand-alone application of A = gamma5 (I - kappa D) to FP64 fields with the
// integer stencil (wilson_fix.cuh), its link and spinor conversions, and the
// choice between it and the FP64-pipe kernel (wilson.cu).
#include <algorithm>
#include <type_traits>

#include "wilson_df.cuh"
#include "wilson_fix.cuh"

namespace ssqcd {
namespace {

using namespace wfix;

// FP64 links [4][9][V] -> digits; *bad is set when a link's rows or columns
// are not of unit length to 2^-10 (the bounds of the integer sums, and their
// accuracy, rest on it; every SU(3) field passes) or not finite: such a field
// keeps the FP64 kernel.
__global__ void pack_links_fix_kernel(const double2* __restrict__ u, int4* __restrict__ uf, int V, int* bad) {
  const long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (i >= 4LL * V) return;
  const int mu = (int)(i / V), s = (int)(i % V);
  double row[3] = {0.0, 0.0, 0.0}, col[3] = {0.0, 0.0, 0.0};
#pragma unroll
  for (int e = 0; e < 9; ++e) {
    const double2 z = u[(size_t)(mu * 9 + e) * V + s];
    const double n2 = z.x * z.x + z.y * z.y;
    row[e / 3] += n2;
    col[e % 3] += n2;
    const long long xr = __double2ll_rn(z.x * 0x1p59) + (1ll << 29), xi = __double2ll_rn(z.y * 0x1p59) + (1ll << 29);
    uf[link_at(fix_tiles(V), mu, s) + e * kTile] =
        make_int4((int)(xr >> 30), (int)((unsigned)xr & 0x3fffffffu) - (1 << 29), (int)(xi >> 30),
                  (int)((unsigned)xi & 0x3fffffffu) - (1 << 29));
  }
  bool ok = true;
#pragma unroll
  for (int k = 0; k < 3; ++k)
    ok = ok && fabs(row[k] - 1.0) <= 0x1p-10 && fabs(col[k] - 1.0) <= 0x1p-10;  // false for NaN
  if (!ok) *bad = 1;
}

__global__ void neighbour_table_kernel(Geometry g, int* __restrict__ nbr) {
  const long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  const int k = (int)(t / g.V), s = (int)(t % g.V);
  if (k >= 8) return;
  const wcore::Coords c = wcore::site_coords(s, g);
  bool tw;
  const int nb = k & 1 ? neighbour_rt<true>(s, c, g, k >> 1, tw) : neighbour_rt<false>(s, c, g, k >> 1, tw);
  nbr[(size_t)(s >> 4) * (8 * kTile) + k * kTile + (s & 15)] = nb | (tw && g.bc_t < 0 ? kNegBit : 0);
}

// Fields to digits: four lanes a site (spin q), eight sites a warp.  USER: in
// is [f][V][12] (the caller's layout), else [f][12][V].  Bound by memory: 16 B
// read and 16 B written a component.
template <typename V2, bool USER>
__global__ void __launch_bounds__(256)
pack_fix_kernel(const V2* __restrict__ in, int4* __restrict__ dig, int* __restrict__ ex, int V) {
  const int lane = threadIdx.x & 31, q = lane >> 3;
  const int s = (blockIdx.x * 8 + (threadIdx.x >> 5)) * 8 + (lane & 7);
  const size_t f = blockIdx.y;
  V2 v[3];
#pragma unroll
  for (int a = 0; a < 3; ++a)
    v[a] = s >= V ? V2{} : USER ? __ldg(in + (f * V + s) * 12 + 3 * q + a) : __ldg(in + (f * 12 + 3 * q + a) * V + s);
  const int word = quad_site_word(v, q), e = word_exp(word);
  if (s >= V) return;
  const int tiles = fix_tiles(V);
  if (q == 0) ex[f * tiles * kTile + s] = word;
  const bool none = e == kZeroExp || e == kSpecialExp;
#pragma unroll
  for (int a = 0; a < 3; ++a)
    dig[field_at(tiles, f, s) + (3 * q + a) * kTile] = none ? make_int4(0, 0, 0, 0) : to_site_digits(v[a], e);
}

__device__ __forceinline__ bool is_zero(double2 v) {  // by integers
  return ((unsigned)(__double2hiint(v.x) | __double2hiint(v.y)) << 1 | (unsigned)(__double2loint(v.x) | __double2loint(v.y))) == 0;
}

// (D psi)(s), component comp, in FP64 from the links and the field as they
// are: next to a value the digits cannot hold (above 2^800, not finite), and
// where the digits' roundings may not be small (Witness).  The sums are those of the
// FP64 kernel up to their order.
template <bool USER>
__device__ __noinline__ double2 hop_sum_fp64(const Geometry& g, const double2* __restrict__ u,
                                             const double2* __restrict__ in, size_t f, int s, int comp) {
  const int V = g.V;
  const wcore::Coords c = wcore::site_coords(s, g);
  const int spin = comp / 3, a = comp % 3;
  double2 sum = make_double2(0.0, 0.0);
  for (int hop = 0; hop < 8; ++hop) {
    const int mu = hop >> 1;
    const bool back = (hop & 1) != 0;
    bool tw;
    const int nb = back ? neighbour_rt<true>(s, c, g, mu, tw) : neighbour_rt<false>(s, c, g, mu, tw);
    const bool neg = tw && g.bc_t < 0;
    // the row of the half spinor this output takes, and the unit in front
    const int r = spin < 2 ? spin : (mu < 2 ? 3 - spin : spin - 2);
    const int lr = mu < 2 ? 1 - r : r;
    const bool swap = (mu & 1) == 0;
    const int sb = (mu == 1 && r == 0) || (mu == 2 && r == 1) ? -1 : 1;
    const int sp = back ? sb : -sb;
    double2 x[3], l[3];
#pragma unroll
    for (int b = 0; b < 3; ++b) {
      const int cu = r * 3 + b, cl = 6 + lr * 3 + b;
      x[b] = USER ? in[(f * V + nb) * 12 + cu] : in[(f * 12 + cu) * V + nb];
      l[b] = USER ? in[(f * V + nb) * 12 + cl] : in[(f * 12 + cl) * V + nb];
    }
    double2 t = make_double2(0.0, 0.0);
#pragma unroll
    for (int b = 0; b < 3; ++b) {
      if (is_zero(x[b]) && is_zero(l[b])) continue;
      double2 h = swap ? make_double2(x[b].x - sp * l[b].y, x[b].y + sp * l[b].x)
                       : make_double2(x[b].x + sp * l[b].x, x[b].y + sp * l[b].y);
      if (neg) h = make_double2(-h.x, -h.y);
      const double2 w = u[(size_t)(mu * 9 + (back ? 3 * b + a : 3 * a + b)) * V + (back ? nb : s)];
      if (back)
        wcore::cmac_conj(t, w, h);
      else
        wcore::cmac(t, w, h);
    }
    if (spin >= 2) {
      const int eta = mu == 0 || (mu != 3 && r == 0) ? -1 : 1;
      const double sg = back ? eta : -eta;
      t = swap ? make_double2(-sg * t.y, sg * t.x) : make_double2(sg * t.x, sg * t.y);
    }
    sum.x += t.x;
    sum.y += t.y;
  }
  return sum;
}

// out = A in for all right-hand sides (FP64, or float-float where V2 is
// float4: every part but the integers in float-float).  A warp covers 16 sites of
// one right-hand side (half-warp r: spin row r) and W warps share its hops;
// RB right-hand sides of the same sites sit in one block, so that a link is
// fetched from L2 once for them.  Consecutive blocks take the further
// right-hand sides of the same sites (nrb of them).
template <int W, typename V2, bool USER>
__global__ void __launch_bounds__(kFixThreads, fix_min_blocks(W))
wilson_fix_kernel(Geometry g, FixView v, const double2* __restrict__ u64, const V2* __restrict__ in,
                  V2* __restrict__ out, int nrhs, int RB, int nrb) {
  constexpr bool kFF = std::is_same<V2, float4>::value;  // float-float fields
  static_assert(!(kFF && USER), "the caller's fields are FP64");
  static_assert(W == 1 || W == 4, "one or four warps a site group");
  constexpr int kWarps = kFixThreads / 32;
  constexpr int kUnits = kWarps / W;  // (site group, rhs) units a block
  // W > 1: the warps' hop sums; W = 1: two operand stages a warp
  __shared__ longlong2 part[W > 1 ? kWarps * 6 * 32 : kWarps * kWarpStages];
  __shared__ V2 stage[USER && W > 1 ? kUnits * kFixSites * 13 : 1];
  __shared__ unsigned evidence[W > 1 && !kFF ? kWarps * 6 * 32 : 1];  // the warps' Witness
  const int V = g.V;
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int unit = w / W, sub = w % W;
  const int i = lane & (kFixSites - 1), r = lane >> 4;
  const int blk = blockIdx.x / nrb;
  const int f = (blockIdx.x % nrb) * RB + unit % RB;
  const int s0 = (blk * (kUnits / RB) + unit / RB) * kFixSites;
  const bool work = f < nrhs && s0 < V;
  const int fc = min(f, nrhs - 1);
  const int s = min(s0 + i, V - 1);
  const V2* inf = in + (size_t)fc * 12 * V;
  V2* outf = out + (size_t)fc * 12 * V;
  // the sites' own components (USER): W > 1 an array of their own, W = 1 the
  // stage of hop 6 once that is done
  V2* st = W > 1 ? stage + (USER ? unit * kFixSites * 13 : 0) : reinterpret_cast<V2*>(part + w * kWarpStages);
  if (W == 1 && !work) return;
  const int own = work ? min(kFixSites, V - s0) * 12 : 0;  // components of the group's sites
  auto stage_at = [](int t) { return t + ((unsigned)t * 21846u >> 18); };  // 13 (t / 12) + t % 12 for t < 192
  if (USER && W > 1 && work) {  // the sites' own components, coalesced
    const V2* src = inf + (size_t)s0 * 12;
    for (int t = lane + 32 * sub, at = stage_at(t); t < kFixSites * 12; t += 32 * W, at = stage_at(t))
      if (t < own) st[at] = src[t];
  }
  v.ex += (size_t)fc * v.tiles * kTile;
  v.dig += field_at(v.tiles, fc, 0);
  Hops h;
  load_neighbours(v, s, h);
  Acc3 up, lo;
  Witness<!kFF> wit;
  if constexpr (W == 1) {
    hop_sums_piped(v, s, i, r, h, reinterpret_cast<int4*>(part + w * kWarpStages), up, lo, wit, [&](int4* to) {
      if (USER) {
        const int4* src = reinterpret_cast<const int4*>(inf + (size_t)s0 * 12);
        for (int t = lane; t < own; t += 32) copy16(to + stage_at(t), src + t);
      }
      copy_commit();
    });
    copy_wait<0>();
  } else {
    hop_sums(v, s, r, sub, h, up, lo, wit);
  }
  const double hf = hop_factor(h.E, -g.kappa);
  if (W > 1) {
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      part[(w * 6 + a) * 32 + lane] = make_longlong2(up.re[a], up.im[a]);
      part[(w * 6 + 3 + a) * 32 + lane] = make_longlong2(lo.re[a], lo.im[a]);
      if constexpr (!kFF) {
        evidence[(w * 6 + a) * 32 + lane] = wit.up[a];
        evidence[(w * 6 + 3 + a) * 32 + lane] = wit.lo[a];
      }
    }
    __syncthreads();
  } else {
    __syncwarp();
  }
  unsigned again = 0;  // components whose hops are taken in FP64
  if constexpr (!kFF) {
#pragma unroll
    for (int k = 0; k < 6; ++k) {
      if (W > 1 && k % W != sub) continue;
      unsigned x = k < 3 ? wit.up[k % 3] : wit.lo[k % 3];
      if constexpr (W > 1) {
        x = 0;
#pragma unroll
        for (int q = 0; q < W; ++q) x |= evidence[((unit * W + q) * 6 + k) * 32 + lane];
      }
      if ((x & kWitnessBits) == 0) again |= 1u << k;
    }
    // zero hops, as of a diluted source, are exact
    if (!any_hop(h.spins, r, false)) again &= 56u;
    if (!any_hop(h.spins, r, true)) again &= 7u;
    if (h.E > kMaxExp) again = 63u;
  }
  // component k of this lane: 0..2 spin r, 3..5 spin 2 + r
#pragma unroll
  for (int k = 0; k < 6; ++k) {
    longlong2 t;
    if (W > 1) {
      if (k % W != sub) continue;
      t = part[(unit * W * 6 + k) * 32 + lane];
#pragma unroll
      for (int q = 1; q < W; ++q) {
        const longlong2 p = part[((unit * W + q) * 6 + k) * 32 + lane];
        t.x += p.x;
        t.y += p.y;
      }
    } else {
      t = k < 3 ? make_longlong2(up.re[k % 3], up.im[k % 3]) : make_longlong2(lo.re[k % 3], lo.im[k % 3]);
    }
    const int comp = (k < 3 ? 0 : 6) + r * 3 + k % 3;
    if (!work || s0 + i >= V) continue;
    if constexpr (kFF) {
      float4 d = hop_cff(t, h.E > kMaxExp ? kZeroExp : h.E);
      if (h.E > kMaxExp) d = make_float4(nanf(""), nanf(""), nanf(""), nanf(""));
      wcore::finish_df1(g, inf, outf, make_float2(0.f, 0.f), make_float2(1.f, 0.f), s, comp, d);
    } else {
      const double2 p = USER ? st[i * 13 + comp] : inf[(size_t)comp * V + s];
      double2 o;
      o.x = k < 3 ? hop_finish<false>(hf, t.x, p.x) : hop_finish<true>(hf, t.x, p.x);
      o.y = k < 3 ? hop_finish<false>(hf, t.y, p.y) : hop_finish<true>(hf, t.y, p.y);
      if (k >= 3) o = make_double2(-o.x, -o.y);
      if (USER)
        st[i * 13 + comp] = o;
      else
        outf[(size_t)comp * V + s] = o;
    }
  }
  if constexpr (!kFF) {
    if (work && s0 + i < V && again != 0) {
      const double small = fabs(hf) * 0x1p-148;  // kappa 2^(E - 5)
      for (int k = sub; k < 6; k += W) {
        if ((again >> k & 1) == 0) continue;
        const int comp = (k < 3 ? 0 : 6) + r * 3 + k % 3;
        const double2 p = USER ? in[((size_t)fc * V + s) * 12 + comp] : inf[(size_t)comp * V + s];
        // beside diagonal terms of that size the hops' roundings are as small
        if (h.E <= kMaxExp && fmin(fabs(p.x), fabs(p.y)) >= small) continue;
        const double2 d = hop_sum_fp64<USER>(g, u64, in, fc, s, comp);
        const double sg = k < 3 ? 1.0 : -1.0;
        double2 o;
        o.x = fma(sg, fma(-g.kappa, d.x, p.x), 0.0 * p.x);
        o.y = fma(sg, fma(-g.kappa, d.y, p.y), 0.0 * p.y);
        if (USER)
          st[i * 13 + comp] = o;
        else
          outf[(size_t)comp * V + s] = o;
      }
    }
  }
  if (USER) {
    if (W > 1)
      __syncthreads();
    else
      __syncwarp();
    V2* dst = outf + (size_t)s0 * 12;
    for (int t = lane + 32 * sub; t < own; t += 32 * W) dst[t] = st[stage_at(t)];
  }
}

template <int W, typename V2, bool USER>
void launch_apply(const Geometry& g, const FixView& v, const double2* u64, const V2* in, V2* out, int nrhs,
                  cudaStream_t s) {
  constexpr int kUnits = fix_units(W);
  const int groups = fix_tiles(g.V);
  int RB = 1;
  while (2 * RB <= kUnits && 2 * RB <= nrhs) RB *= 2;
  const int nrb = (nrhs + RB - 1) / RB, gb = (groups + kUnits / RB - 1) / (kUnits / RB);
  const unsigned blocks = (unsigned)gb * nrb;
  wilson_fix_kernel<W, V2, USER><<<blocks, kFixThreads, 0, s>>>(g, v, u64, in, out, nrhs, RB, nrb);
}

template <typename V2, bool USER>
int pack_fields(const V2* in, int nrhs, int V, int4* dig, int* ex, cudaStream_t s) {
  pack_fix_kernel<V2, USER><<<dim3((V + 63) / 64, nrhs), 256, 0, s>>>(in, dig, ex, V);
  count_launches(1);
  SS_CHECK_LAUNCH();
  return SSQCD_OK;
}

// digits of the block of fields, then the stencil
template <typename V2, bool USER>
int apply_block(ssqcd_lattice lat, const V2* in, V2* out, int nrhs, int4* dig, int* ex, cudaStream_t s) {
  const Geometry& g = lat->g;
  const double2* u64 = lat->u64.as<double2>();
  SS_TRY((pack_fields<V2, USER>(in, nrhs, g.V, dig, ex, s)));
  const FixView v{lat->ufix.as<int4>(), lat->fnbr, dig, ex, fix_tiles(g.V)};
  if (fix_split(g.V, nrhs) == 1)
    launch_apply<1, V2, USER>(g, v, u64, in, out, nrhs, s);
  else
    launch_apply<4, V2, USER>(g, v, u64, in, out, nrhs, s);
  count_launches(1);
  SS_CHECK_LAUNCH();
  return SSQCD_OK;
}

// The integer form for all right-hand sides, a block at a time; false in *done
// when there is no room for the digits.
template <typename V2, bool USER>
int apply_fix(ssqcd_lattice lat, const V2* in, V2* out, int nrhs, cudaStream_t s, bool* done, void* work) {
  const int V = lat->g.V, nb = fix_block(V, nrhs);
  const size_t db = fix_field_bytes(V) * nb;
  DevBuf ws;
  *done = false;
  if (work == nullptr && ws.alloc(db + fix_exp_bytes(V) * nb) != SSQCD_OK) return SSQCD_OK;
  char* dig = work != nullptr ? static_cast<char*>(work) : ws.as<char>();
  for (int f = 0; f < nrhs; f += nb) {
    const size_t off = (size_t)f * 12 * V;
    SS_TRY((apply_block<V2, USER>(lat, in + off, out + off, std::min(nb, nrhs - f),
                                  reinterpret_cast<int4*>(dig), reinterpret_cast<int*>(dig + db), s)));
  }
  *done = true;
  return SSQCD_OK;
}

}  // namespace

size_t fix_field_bytes(int V) { return sizeof(int4) * 12 * kTile * (size_t)fix_tiles(V); }
size_t fix_exp_bytes(int V) { return sizeof(int) * kTile * (size_t)fix_tiles(V); }

// Scratch of the integer form for a block of right-hand sides: at most 1 GiB
// at a time (a further block waits for the last one on the stream).
int fix_block(int V, int nrhs) {
  const size_t per = fix_field_bytes(V) + fix_exp_bytes(V);
  const size_t fit = ((size_t)1 << 30) / per;
  return (int)std::max<size_t>(1, std::min<size_t>({fit, (size_t)nrhs, (size_t)65535}));
}

int pack_fix(const double2* in, int nrhs, int V, int4* dig, int* ex, cudaStream_t s) {
  return pack_fields<double2, false>(in, nrhs, V, dig, ex, s);
}
int pack_fix(const float4* in, int nrhs, int V, int4* dig, int* ex, cudaStream_t s) {
  return pack_fields<float4, false>(in, nrhs, V, dig, ex, s);
}

// Warps that share the eight hops of 16 sites: 1 once the groups fill the
// GPU's schedulers (8^4 x 4, 1024 groups: 27.9 us an iteration against 29.6 with
// 4; 16^3 x 32: 48 us an application against 57), 4 below (8^4 x 1, 256 groups:
// 20.0 us an iteration; with eight warps, one hop each, it was 21.4, and 20.9
// against 19.8 for the 64 groups of 4^4 x 4).
int fix_split(int V, int nrhs) { return (long long)fix_tiles(V) * nrhs >= 608 ? 1 : 4; }

int wilson64_lat(ssqcd_lattice lat, const double2* in, bool user, double2* out, int nrhs, cudaStream_t s, void* work) {
  const Geometry& g = lat->g;
  if (nrhs <= 0) return SSQCD_OK;
  AllocStream scope(s);
  if (lat->fix_ok) {
    bool done = false;
    if (user)
      SS_TRY((apply_fix<double2, true>(lat, in, out, nrhs, s, &done, work)));
    else
      SS_TRY((apply_fix<double2, false>(lat, in, out, nrhs, s, &done, work)));
    if (done) return SSQCD_OK;
  }
  if (!user) return wilson64(g, lat->u64.as<double2>(), in, out, nrhs, 0.0, 1.0, nullptr, nullptr, s);
  DevBuf a, b;
  const size_t bytes = sizeof(double2) * 12 * (size_t)g.V * nrhs;
  SS_TRY(a.alloc(bytes));
  SS_TRY(b.alloc(bytes));
  SS_TRY(pack_spinors(in, a.as<double2>(), nrhs, g.V, s));
  SS_TRY(wilson64(g, lat->u64.as<double2>(), a.as<double2>(), b.as<double2>(), nrhs, 0.0, 1.0, nullptr, nullptr, s));
  return unpack_spinors(b.as<double2>(), out, nrhs, g.V, s);
}

int wilson_df_lat(ssqcd_lattice lat, const float4* in, float4* out, int nrhs, cudaStream_t s) {
  if (nrhs <= 0) return SSQCD_OK;
  if (lat->fix_ok) {
    AllocStream scope(s);
    bool done = false;
    SS_TRY((apply_fix<float4, false>(lat, in, out, nrhs, s, &done, nullptr)));
    if (done) return SSQCD_OK;
  }
  {
    AllocStream plain(s, false);  // lattice-owned
    SS_TRY(ensure_df_links(lat));
  }
  return wilson_df(lat->g, lat->udf.as<float4>(), in, out, nrhs, 0.0, 1.0, s);
}

size_t apply_workspace_bytes(ssqcd_lattice lat, int nrhs) {
  if (!lat->fix_ok) return 0;
  const int nb = fix_block(lat->g.V, nrhs);
  return (fix_field_bytes(lat->g.V) + fix_exp_bytes(lat->g.V)) * nb;
}

int take_workspace(ssqcd_lattice lat, size_t bytes, std::unique_ptr<DevBuf>* out) {
  {
    std::lock_guard<std::mutex> lock(lat->ws_mutex);
    for (size_t i = 0; i < lat->ws.size(); ++i)
      if (lat->ws[i]->bytes >= bytes) {
        *out = std::move(lat->ws[i]);
        lat->ws.erase(lat->ws.begin() + i);
        return SSQCD_OK;
      }
  }
  auto b = std::make_unique<DevBuf>();
  // plain allocation: it may be used on any stream and by any thread next
  AllocStream plain(nullptr, false);
  SS_TRY(b->alloc(bytes));
  *out = std::move(b);
  return SSQCD_OK;
}

void give_workspace(ssqcd_lattice lat, std::unique_ptr<DevBuf> ws) {
  if (ws == nullptr || ws->bytes > ((size_t)256 << 20)) return;
  std::unique_ptr<DevBuf> out;  // released outside the lock
  std::lock_guard<std::mutex> lock(lat->ws_mutex);
  lat->ws.push_back(std::move(ws));
  if (lat->ws.size() > 4) {  // the smallest goes
    auto it = std::min_element(lat->ws.begin(), lat->ws.end(),
                               [](const auto& a, const auto& b) { return a->bytes < b->bytes; });
    out = std::move(*it);
    lat->ws.erase(it);
  }
}

int build_fix_links(ssqcd_lattice lat) {
  const int V = lat->g.V;
  lat->fix_ok = false;
  // links, neighbour table and the check's flag in one allocation
  const size_t lb = 3 * fix_field_bytes(V), nb = 8 * fix_exp_bytes(V);
  if (lat->ufix.alloc(lb + nb + sizeof(int)) != SSQCD_OK) return SSQCD_OK;  // no room: the FP64 kernel serves
  int* nbr = reinterpret_cast<int*>(lat->ufix.as<char>() + lb);
  int* bad = reinterpret_cast<int*>(lat->ufix.as<char>() + lb + nb);
  int h = 0;
  SS_CUDA(cudaMemsetAsync(bad, 0, sizeof(int), lat->stream));
  pack_links_fix_kernel<<<grid_for(4LL * V, 256), 256, 0, lat->stream>>>(lat->u64.as<double2>(), lat->ufix.as<int4>(),
                                                                         V, bad);
  neighbour_table_kernel<<<grid_for(8LL * V, 256), 256, 0, lat->stream>>>(lat->g, nbr);
  count_launches(2);
  SS_CHECK_LAUNCH();
  SS_CUDA(cudaMemcpyAsync(&h, bad, sizeof(int), cudaMemcpyDeviceToHost, lat->stream));
  SS_CUDA(cudaStreamSynchronize(lat->stream));
  lat->fix_ok = h == 0;
  // Once links have suited, the memory stays the lattice's: a run in flight
  // (ssqcd_server) may hold it, whatever is uploaded meanwhile.
  if (lat->fix_ok)
    lat->fnbr = nbr;
  else if (lat->fnbr == nullptr)
    lat->ufix.release();
  return SSQCD_OK;
}

}  // namespace ssqcd
