// Combinations of FP64 vectors on the tensor cores (tcgen05), with real or
// complex coefficients:
//
//   out[l][o][e] = sum_{s < count[l]} C[l][o][s] r_s[l][e]
//
// -- the moments of Eq. 2 and the shifted solutions from the stored seed
// residuals (the Krylov-basis identity: every shifted solution is a
// combination of the seed residuals), the moments from solutions in hand, the
// basis combinations of Rayleigh-Ritz.  A complex coefficient is two real ones
// (its real and imaginary part combine the same vectors); the epilogue adds
// the two sums, which sit in neighbouring lanes.
//
// GB300's tensor cores have no fast FP64 rate, so the FP64 products are
// split exactly into fp16 pieces (the error-free splitting of Ozaki et al.,
// "Error-free transformations of matrix multiplication by using fast
// routines of matrix multiplication and its applications", 2012):
//
// * Each residual r_s (real and imaginary parts as separate rows) is scaled
//   by tau_s = 2^e_s >= max |r_s| and rounded to a 56-bit fixed-point
//   integer X = round(|r| 2^(56 - e_s)), whose seven base-256 digits
//   d_0 .. d_6 are the fp16 slices A_p = sign d_p (integers of 8 bits, exact
//   in fp16, which a byte permutation and one paired multiply-add make).
// * Each coefficient column o, B[s][o] = C[l][o][s] tau_s, is scaled by
//   sigma_o = 2^g_o >= max_s |B[s][o]| and split the same way into B_q.
// * A_p B_q sums 16-bit integer products; 256 of them stay below 2^24, so
//   the fp32 accumulator in tensor memory holds the sum of a chunk of 256
//   slots exactly.  The pairs with p + q <= 6 are kept: level l = p + q has
//   weight 2^(-8 (l + 2)), and the dropped levels lie below 2^-64 of the
//   scales.  The chunk sums of the levels I_l are added up exactly in two
//   64-bit integers per output, X_hi = I_0 2^16 +
//   I_1 2^8 + I_2 and X_lo = I_3 2^24 + I_4 2^16 + I_5 2^8 + I_6, and at the
//   end of a tile
//     out = sigma_o 2^-16 (2^-16 X_hi + 2^-48 X_lo)   in FP64.
// The result lies within about 2^-56 of the scales of the exact sum, the
// order of the FP64 sum's own rounding: a CPU emulation of this arithmetic
// on the 8^4 workload puts the moments within 2.3e-16 of the exact ones
// (the FP64 sum: 9.1e-16); on test data whose elements span 4 decades
// within a residual, the fixed-point grid leaves the small ones fewer bits
// (2.4e-15 against 6.5e-16).
//
// Measured (2502 slots of 786,432 complex elements, 31.5 GB, 16 real outputs):
// 15.1 ms, 2.1 TB/s, and 5.0 ms of scale pass.  Before: 34.6 ms -- the scale
// pass compared in FP64 (15 ms; 5 by integers), one lane issued the copies, each
// behind a dependent load of the block table (3200 cycles a K-step), the epilogue
// converted to 64-bit integers on the FP64 pipe, and a digit took twice the
// integer operations.  Those of the slicing warps (~20 an element, the integer
// pipe 58% busy) and the scale pass bound it now.
//
// One persistent CTA per SM (26 warps; wide form 28):
// * warp 25: bulk copies (cp.async.bulk, a lane a slot) of a tile's 16 slots x
//   128 rows of FP64 into a ring of kF64Stages stages;
// * warps 8-23: cut the stage into the seven A slices (core-matrix layout,
//   K-major, no swizzle) in a ring of kSliceStages stages, half of them a K-step
//   in turn; the K-step's B slices (prepared once per launch in the same layout)
//   are copied beside them;
// * warp 24, lane 0: issues seven tcgen05.mma (M = 128, N = 16 (7 - p), K = 16) a
//   K-step into 448 tensor-memory columns, and commits the stage and, every 256
//   slots, the accumulators;
// * warps 0-7: read the accumulators (tcgen05.ld; warp w: lanes 32 (w % 4),
//   outputs 8 (w / 4) ..), add them exactly into X_hi and X_lo, and at the
//   end of a tile form and store the outputs.
// Wide form (more than eight complex outputs; Form): the cut is what a pass costs,
// whatever its outputs, so that 16 complex ones at a time halve it (64 outputs of
// 1000 slots x 4 sources of 12^4: 77 -> 42 ms, then 31 with the rest).  Its 28 pairs
// do not fit tensor memory: the pairs of a level share an accumulator, by rows of
// zeros ahead of B's, for 96 slots; two accumulators, so that the epilogue, with
// registers of the other warps, and the products overlap.
// Every wait is bounded (1 s of device time); past it the kernel sets *err,
// lets its issued copies and MMAs finish, frees its tensor memory and
// returns.
#include <cuda_fp16.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cstdint>
#include <cstdlib>
#include <type_traits>

#include "internal.h"

namespace ssqcd {
namespace {

constexpr int kRows = 128;         // real rows (64 complex elements) per tile
constexpr int kKStep = 16;         // slots per MMA (K of kind::f16)
constexpr int kSlices = 7;         // base-256 digits of the 56-bit fixed point
constexpr int kOut = 16;           // real outputs per launch
constexpr int kWideOut = 32;       // of the wide form
constexpr int kF64Stages = 4;
constexpr int kEpiWarps = 8;       // warps 0 ..
constexpr int kSliceWarps = 16;    // warps 8 ..
constexpr int kMmaWarp = kEpiWarps + kSliceWarps;
constexpr int kLoadWarp = kMmaWarp + 1;
constexpr int kTmemCols = 512;
constexpr int kABytes = kRows * kKStep * 2;       // one fp16 slice: 4096 B
// The two forms of the kernel.  Narrow: 16 real outputs, every pair (p, q) a
// block of 16 accumulator columns of its own.  Wide (more than 8 complex
// outputs): 32 real outputs, the pairs of a level in one block of 32.
template <bool WIDE>
struct Form {
  static constexpr int kO = WIDE ? kWideOut : kOut;
  static constexpr int kBRows = kSlices * kO;         // 112, 224
  static constexpr int kBBytes = kBRows * kKStep * 2;  // 3584, 7168 B
  // wide: rows of zeros ahead of B's, so that every slice's product spans all levels
  static constexpr int kPadBytes = WIDE ? (kSlices - 1) * kO * kKStep * 2 : 0;
  static constexpr int kSliceStages = WIDE ? 3 : 4;
  // K-steps per accumulator flush.  Narrow: 256 products of 16 bits.  Wide: a
  // level's products of signed digits, at most 2 * 2^15 + 5 * 2^14 a slot, of 96 slots.
  static constexpr int kChunkSteps = WIDE ? 6 : 16;
  static constexpr int kBuffers = WIDE ? 2 : 1;  // of accumulators
  static constexpr int kBufferCols = 256;
  static constexpr int kThreads = WIDE ? 896 : 832;  // whole warpgroups where registers move between them
  static constexpr int kEpiOuts = kO / 2;             // real outputs an epilogue thread
  // wide: registers a thread at launch, of the epilogue and of the others
  static constexpr int kRegs = 72, kEpiRegs = 112, kOtherRegs = 56;
  static_assert(kEpiWarps * 32 * kEpiRegs + (896 - kEpiWarps * 32) * kOtherRegs <= 896 * kRegs, "register split");
};
constexpr int kMaxCount = 65535;                  // slots (grid.y of the scale kernel)
constexpr unsigned long long kTcWaitNs = 1000000000ull;
constexpr long long kTcSpin = 1LL << 26;

template <bool WIDE>
struct __align__(1024) SliceStage {
  unsigned char a[kSlices][kABytes];
  unsigned char b[Form<WIDE>::kPadBytes + Form<WIDE>::kBBytes];
};
struct __align__(1024) F64Stage {
  double v[kKStep][kRows];
};
template <bool WIDE>
struct TcShared {
  F64Stage f64[kF64Stages];
  SliceStage<WIDE> sl[Form<WIDE>::kSliceStages];
  unsigned long long full_f[kF64Stages], empty_f[kF64Stages];
  unsigned long long full_s[Form<WIDE>::kSliceStages], full_b[Form<WIDE>::kSliceStages];
  unsigned long long empty_s[Form<WIDE>::kSliceStages];
  unsigned long long tmem_full[2], tmem_empty[2], mma_done;
  unsigned tmem_base;
  int abort;
};

// column of tensor memory where the products of A slice p start (pairs
// (p, q), q = 0 .. 6 - p, 16 columns each)
__host__ __device__ constexpr int col_base(int p) { return 16 * (p * 7 - p * (p - 1) / 2); }

__device__ __forceinline__ unsigned su32(const void* p) { return (unsigned)__cvta_generic_to_shared(p); }
__device__ __forceinline__ void bar_init(unsigned long long* b, unsigned c) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(su32(b)), "r"(c) : "memory");
}
__device__ __forceinline__ void bar_arrive(unsigned long long* b) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(su32(b)) : "memory");
}
__device__ __forceinline__ void bar_arrive_tx(unsigned long long* b, unsigned bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(su32(b)), "r"(bytes) : "memory");
}
__device__ __forceinline__ bool bar_test(unsigned long long* b, unsigned parity) {
  unsigned ok;
  asm volatile(
      "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2, %3;\n selp.u32 %0, 1, 0, p;\n}\n"
      : "=r"(ok)
      : "r"(su32(b)), "r"(parity), "r"(2000u)  // the thread may sleep up to 2 us between tests
      : "memory");
  return ok != 0;
}
__device__ __forceinline__ unsigned long long gtimer() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}
// bounded wait for the phase of the given parity; false after kTcWaitNs or
// when another role has given up (abort)
__device__ __forceinline__ bool bar_wait(unsigned long long* b, unsigned parity, volatile int* abort) {
  if (bar_test(b, parity)) return true;
  const unsigned long long t0 = gtimer();
  for (long long i = 1; i < kTcSpin; ++i) {
    if (bar_test(b, parity)) return true;
    if ((i & 255) == 0) {
      if (*abort) return false;
      if (gtimer() - t0 > kTcWaitNs) return false;
    }
  }
  return false;
}
// the same for all 32 lanes of a warp together: every lane observes the
// phase (so every lane may read what it guards) and all leave together
__device__ __forceinline__ bool bar_wait_warp(unsigned long long* b, unsigned parity, volatile int* abort) {
  if (__all_sync(0xffffffffu, bar_test(b, parity))) return true;
  const unsigned long long t0 = gtimer();
  for (long long i = 0; i < kTcSpin; ++i) {
    if (__all_sync(0xffffffffu, bar_test(b, parity))) return true;
    if ((i & 255) == 255 && __any_sync(0xffffffffu, *abort != 0 || gtimer() - t0 > kTcWaitNs)) return false;
  }
  return false;
}
__device__ __forceinline__ void bulk_copy(void* dst, const void* src, unsigned bytes, unsigned long long* bar) {
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
                   su32(dst)),
               "l"(src), "r"(bytes), "r"(su32(bar))
               : "memory");
}

// ---- tcgen05 ---------------------------------------------------------------------------
// Shared-memory matrix descriptor, K-major without swizzle: core matrices of
// 8 rows x 16 bytes stored as 128 contiguous bytes; `lbo` = byte distance of
// the core matrices adjacent in K, `sbo` = of those adjacent in M (or N).
// Bits: start address >> 4 [0, 14), lbo >> 4 [16, 30), sbo >> 4 [32, 46),
// descriptor version 1 at [46, 48), base offset 0, swizzle mode 0 [61, 64).
__device__ __forceinline__ unsigned long long smem_desc(const void* p, unsigned lbo, unsigned sbo) {
  const unsigned long long a = (su32(p) & 0x3FFFFu) >> 4;
  return a | ((unsigned long long)((lbo >> 4) & 0x3FFFu) << 16) | ((unsigned long long)((sbo >> 4) & 0x3FFFu) << 32) |
         (1ull << 46);
}
// Instruction descriptor of kind::f16: fp32 accumulator (bits [4, 6) = 1),
// A and B fp16 ([7, 10) = 0, [10, 13) = 0), both K-major (bits 15, 16 = 0),
// N >> 3 at [17, 23), M >> 4 at [24, 29).
__host__ __device__ constexpr unsigned idesc_f16(int M, int N) {
  return (1u << 4) | ((unsigned)(N >> 3) << 17) | ((unsigned)(M >> 4) << 24);
}
__device__ __forceinline__ void tc_mma(unsigned d_tmem, unsigned long long a, unsigned long long b, unsigned idesc,
                                       unsigned acc) {
  asm volatile(
      "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
      " tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(d_tmem),
      "l"(a), "l"(b), "r"(idesc), "r"(acc)
      : "memory");
}
// arrive on the mbarrier once the MMAs issued so far by this thread are done
__device__ __forceinline__ void tc_commit(unsigned long long* bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(su32(bar))
               : "memory");
}
__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }
// the 8 consecutive fp32 columns of this thread's lane; load and wait in one
// statement
__device__ __forceinline__ void tc_ld8(unsigned taddr, float (&t)[8]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];\n"
      "tcgen05.wait::ld.sync.aligned;\n"
      : "=f"(t[0]), "=f"(t[1]), "=f"(t[2]), "=f"(t[3]), "=f"(t[4]), "=f"(t[5]), "=f"(t[6]), "=f"(t[7])
      : "r"(taddr)
      : "memory");
}

__device__ __forceinline__ void tc_ld16(unsigned taddr, float (&t)[16]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, "
      "[%16];\n"
      "tcgen05.wait::ld.sync.aligned;\n"
      : "=f"(t[0]), "=f"(t[1]), "=f"(t[2]), "=f"(t[3]), "=f"(t[4]), "=f"(t[5]), "=f"(t[6]), "=f"(t[7]), "=f"(t[8]),
        "=f"(t[9]), "=f"(t[10]), "=f"(t[11]), "=f"(t[12]), "=f"(t[13]), "=f"(t[14]), "=f"(t[15])
      : "r"(taddr)
      : "memory");
}

// byte offset of element (row, k) of a K-major no-swizzle tile of 16 K:
// core matrix (row / 8, k / 8) at (row / 8) * 256 + (k / 8) * 128
__host__ __device__ constexpr int core_off(int row, int k) {
  return (row >> 3) * 256 + (k >> 3) * 128 + (row & 7) * 16 + (k & 7) * 2;
}
constexpr unsigned kLbo = 128, kSbo = 256;

// 57-bit fixed point floor(|x| 2^(57 - e)) for |x| < 2^e: the mantissa at bit
// 4, shifted right by e + 1022 - E >= 0.  Without branches: the lanes of a
// warp hold elements of different exponents.  Zero and subnormals (E = 0)
// give 0: e >= -950 (tc_scales_kernel), so that they are shifted out.
// Whatever x and e are, it is below 2^57.
__device__ __forceinline__ unsigned long long fixed57(double x, int e) {
  const unsigned hw = (unsigned)__double2hiint(x), lw = (unsigned)__double2loint(x);
  const int E = (int)((hw >> 20) & 0x7FF);
  const unsigned k = min((unsigned)(e + 1022 - E), 63u);
  return ((unsigned long long)__funnelshift_l(lw, (hw & 0xFFFFFu) | 0x100000u, 4) << 32 | (lw << 4)) >> k;
}
__device__ __forceinline__ uint2 halves(unsigned long long v) { return make_uint2((unsigned)v, (unsigned)(v >> 32)); }
// X = round(|x| 2^(56 - e)), ties up
__device__ __forceinline__ uint2 fixed56(double x, int e) { return halves((fixed57(x, e) + 1) >> 1); }
// Signed digits (complex and float-float combinations): X with its sign, rounded to nearest,
// plus the bias that makes every base-256 digit d a byte d + 128 and the top
// one (|d| <= 256) a field d + 512 of bits 48 ...  The digits' products then
// average to zero, so that the dropped levels do: with magnitudes and signs
// they add up coherently, the larger part of the error of a short sum.
__device__ __forceinline__ uint2 signed_digits(double x, int e) {
  const unsigned long long t = fixed57(x, e);
  const unsigned sg = (unsigned)(__double2hiint(x) >> 31);
  // a negative x's floor is the complement; twice the bias plus the rounding's one
  constexpr unsigned long long c = 0x0401010101010101ull;
  return halves((((t >> 32 ^ sg) << 32 | ((unsigned)t ^ sg)) + c) >> 1);
}
// The same of a float-float number h + l, |h| < 2^e: both mantissas on the
// 57-bit grid, what is left of them below it cut off.
__device__ __forceinline__ long long float57(float f, int e) {
  const unsigned b = __float_as_uint(f);
  const int E = (int)((b >> 23) & 0xFF);
  const unsigned m = (b & 0x7FFFFFu) | (unsigned)min(E, 1) << 23;
  const unsigned k = min((unsigned)(e + 126 - max(E, 1)), 63u);
  const long long sg = (int)b >> 31;
  return ((long long)(((unsigned long long)m << 33) >> k) ^ sg) - sg;
}
__device__ __forceinline__ uint2 signed_digits(float h, float l, int e) {
  return halves((unsigned long long)(float57(h, e) + float57(l, e) + 0x0401010101010101ll) >> 1);
}
// The digits of two elements side by side, so that a byte permutation with the
// exponent byte of 1024 makes a pair of fp16 numbers 1024 + byte: p[0], p[1]
// from the low words, p[2] the lower half of the high ones.
struct BytePairs {
  unsigned p[3], top;
};
__device__ __forceinline__ BytePairs byte_pairs(uint2 a, uint2 b) {
  BytePairs r;
  r.p[0] = __byte_perm(a.x, b.x, 0x5140);
  r.p[1] = __byte_perm(a.x, b.x, 0x7362);
  r.p[2] = __byte_perm(a.y, b.y, 0x5140);
  r.top = __byte_perm(a.y, b.y, 0x7632);
  return r;
}
// 1024 + byte 6 - P of both (P = 0: 1024 + the top 16 bits)
template <int P>
__device__ __forceinline__ __half2 with_exponent(const BytePairs& r) {
  constexpr int byte = 6 - P;
  const unsigned v = P == 0 ? r.top | 0x64006400u : __byte_perm(r.p[byte >> 1], 0x64646464u, byte & 1 ? 0x4342 : 0x4140);
  return *reinterpret_cast<const __half2*>(&v);
}
template <int P>
__device__ __forceinline__ unsigned signed_pair(const BytePairs& r) {
  const __half2 d = __hadd2(with_exponent<P>(r), __half2half2(__ushort_as_half(P == 0 ? 0xE600 : 0xE480)));  // -1536, -1152
  return *reinterpret_cast<const unsigned*>(&d);
}
// The digits with their signs: the bytes under the exponent of 1024, times the
// signs, less 1024 (exact).  s1: (+-1, +-1), s2: (-+1024, -+1024).
template <int P>
__device__ __forceinline__ unsigned digit_pair(const BytePairs& r, __half2 s1, __half2 s2) {
  const __half2 d = __hfma2(with_exponent<P>(r), s1, s2);
  return *reinterpret_cast<const unsigned*>(&d);
}

// ---- scales and coefficient slices --------------------------------------------------------
// Where the vectors are: slot s of source l in the basis blocks tab[s >> log],
// [slot][L][n] each, or (tab null) at base, [l][slots][n].
struct SlotMap {
  char* const* tab;
  int basis_log, L;
  const double2* base;
  long long slots;
};
__device__ __forceinline__ const double* slot_ptr(const SlotMap& m, long long n, int l, int s) {
  if (m.tab == nullptr) return reinterpret_cast<const double*>(m.base + (l * m.slots + s) * n);
  char* const* tab = m.tab;
  const int basis_log = m.basis_log, L = m.L;
  const int mask = (1 << basis_log) - 1;
  return reinterpret_cast<const double*>(tab[s >> basis_log]) + 2 * (((long long)(s & mask) * L + l) * n);
}

// Real output o of a pass: the part o & 1 of the complex coefficient o / 2
// (cplx), or the real part of coefficient o.
struct CoefView {
  const double2* c;
  long long sl, so, ss;  // strides of source, output, slot
  bool cplx;
  bool sgn;  // signed digits
  __device__ __forceinline__ double get(int l, int o, int s) const {
    const double2 v = c[l * sl + (cplx ? o >> 1 : o) * so + s * ss];
    return cplx && (o & 1) ? v.y : v.x;
  }
};
// slots in whole K-steps: the stride of the slot scales
__host__ __device__ __forceinline__ int padded(int S) { return (S + kKStep - 1) / kKStep * kKStep; }
__device__ __forceinline__ int slots_of(const int* count, int l, int S) { return count != nullptr ? count[l] : S; }

// mx[l'][s] = the largest high word (exponent and leading mantissa bits, sign
// off) of a component of r_s of source l0 + l'; infinities and NaN are at
// least kBadKey; ex[l'][s] (may be null) the sum of the components' exponent
// fields.  By integers: FP64 comparisons run on a pipe of two a clock
// and SM (2.1 TB/s with them).  grid (x: element blocks, y: slot, z: source)
// FF: float-float vectors (re, im, their lower parts), the upper parts' keys and
// exponents as doubles have them.
constexpr unsigned kBadKey = 0x7FF00000u;
template <bool FF>
__global__ void __launch_bounds__(256)
tc_maxabs_kernel(SlotMap map, long long n, int l0, const int* __restrict__ count, int S, unsigned* __restrict__ mx,
                 unsigned long long* __restrict__ ex) {
  const int s = blockIdx.y, lz = blockIdx.z, l = l0 + lz;
  if (s >= slots_of(count, l, S)) return;
  const uint4* r = reinterpret_cast<const uint4*>(slot_ptr(map, n, l, s));
  unsigned m = 0, se = 0;
  const long long stride = (long long)gridDim.x * blockDim.x;
  for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < n; e += 4 * stride) {
    uint4 v[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) v[i] = e + i * stride < n ? __ldg(r + e + i * stride) : make_uint4(0, 0, 0, 0);
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const unsigned a = (FF ? v[i].x : v[i].y) & 0x7FFFFFFFu, b = (FF ? v[i].y : v[i].w) & 0x7FFFFFFFu;
      m = max(m, max(a, b));
      if (FF)
        se += (a >> 23 != 0 ? (a >> 23) + 896 : 0) + (b >> 23 != 0 ? (b >> 23) + 896 : 0);
      else
        se += (a >> 20) + (b >> 20);
    }
    if (se >= 1u << 26) {  // 32 lanes of this still fit 32 bits
      if (ex != nullptr) atomicAdd(ex + (size_t)lz * S + s, (unsigned long long)se);
      se = 0;
    }
  }
  m = __reduce_max_sync(0xffffffffu, m);
  if (FF) m = (unsigned)__double2hiint((double)__uint_as_float(m));
  if ((threadIdx.x & 31) == 0) atomicMax(mx + (size_t)lz * S + s, m);
  if (ex != nullptr) {
    se = __reduce_add_sync(0xffffffffu, se);
    if ((threadIdx.x & 31) == 0) atomicAdd(ex + (size_t)lz * S + s, (unsigned long long)se);
  }
}

// the exponent e with 2^(e - 1) <= x < 2^e (x > 0), 0 for x = 0
__device__ __forceinline__ int exp_above(double x) {
  int e = 0;
  if (x > 0.0) (void)frexp(x, &e);
  return e;
}

// A vector suits the fixed point of its largest component when its components
// are on average at most kMaxSpread binades below it: then max / rms <= 2^5, the
// grid's error, 2^-57 of the largest, is below 2^-52 of the rms, and FP64's own
// rounding of the sum is no smaller (a Gaussian vector: 3 to 4 binades).  A
// point-like vector is far above it.
constexpr int kMaxSpread = 5;
constexpr int kErrWait = 1, kErrSpread = 2;  // bits of the error word

// e[l'][s] (slot scales) and sig[l'][o] = 2^g_o >= max_s |C[l][o][s] 2^e_s|;
// one block of 256 threads per (source, output).  A non-finite residual
// element or coefficient makes sig NaN, so that the outputs of that source
// come out NaN as the FP64 sum's would (the slices themselves stay finite).
template <int OUT>
__global__ void tc_scales_kernel(const unsigned* __restrict__ mx, CoefView C, int O, int S, int l0,
                                 const int* __restrict__ count, int* __restrict__ eslot, double* __restrict__ sig,
                                 const unsigned long long* __restrict__ ex, long long n, int* __restrict__ err) {
  const int lz = blockIdx.x / OUT, o = blockIdx.x % OUT, l = l0 + lz;
  const int cnt = slots_of(count, l, S);
  double m = 0.0;
  bool bad = false;
  for (int s = threadIdx.x; s < cnt; s += blockDim.x) {
    const unsigned key = mx[(size_t)lz * S + s];
    const bool fin = key < kBadKey;
    // 2^(e - 1) <= max < 2^e; a vector of zeros has no share in its outputs' scales
    const int e = !fin ? 0 : key != 0 ? max((int)(key >> 20) - 1022, -950) : -950;
    bad |= !fin;
    if (ex != nullptr && o == 0 && key != 0 &&
        (unsigned long long)(key >> 20) * (unsigned long long)(2 * n) >
            ex[(size_t)lz * S + s] + (unsigned long long)kMaxSpread * (unsigned long long)(2 * n))
      atomicOr(err, kErrSpread);
    if (o == 0) eslot[(size_t)lz * padded(S) + s] = e;
    if (o < O) {
      // the two parts of a complex coefficient share their scale
      for (int k = 0; k < (C.cplx ? 2 : 1); ++k) {
        const double c = C.get(l, o ^ k, s);
        bad |= !isfinite(c);
        if (isfinite(c) && key != 0) m = fmax(m, fabs(ldexp(c, e)));
      }
    }
  }
#pragma unroll
  for (int d = 16; d > 0; d >>= 1) m = fmax(m, __shfl_xor_sync(0xffffffffu, m, d));
  bad = __any_sync(0xffffffffu, bad);
  __shared__ double wm[32];
  __shared__ int wb[32];
  if ((threadIdx.x & 31) == 0) {
    wm[threadIdx.x >> 5] = m;
    wb[threadIdx.x >> 5] = bad ? 1 : 0;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int w = 1; w < (int)(blockDim.x >> 5); ++w) {
      m = fmax(m, wm[w]);
      bad |= wb[w] != 0;
    }
    if (ex != nullptr && (bad || !isfinite(m) || abs(exp_above(m)) > 950)) atomicOr(err, kErrSpread);
    // every output of the source: a bad slot of this source poisons them all
    sig[(size_t)lz * OUT + o] = (bad || !isfinite(m)) ? __longlong_as_double(0x7FF8000000000000ll)
                                                       : ldexp(1.0, exp_above(m));
  }
}

// B image of K-step kk for source l0 + l' (grid (kk, l'), 14 OUT threads): row
// q * OUT + o of the N x 16 operand holds digit q of C[l][o][s] 2^(e_s - g_o)
// for the slots s = 16 kk + k; thread t writes the 8 slots k = 8 (t & 1) ..
// of row t / 2 (16 bytes of one core matrix).
template <int OUT>
__global__ void tc_bslices_kernel(CoefView C, int O, int S, int l0, const int* __restrict__ count,
                                  const int* __restrict__ eslot, const double* __restrict__ sig, int ksteps_cap,
                                  unsigned char* __restrict__ bimg) {
  const int kk = blockIdx.x, lz = blockIdx.y, l = l0 + lz;
  const int t = threadIdx.x, row = t >> 1, h = t & 1;
  const int q = row / OUT, o = row % OUT;
  const int cnt = slots_of(count, l, S);
  __align__(16) __half f[8];
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    const int s = kk * kKStep + 8 * h + i;
    int d = 0;
    if (o < O && s < cnt) {
      const int g = exp_above(sig[(size_t)lz * OUT + o]) - 1;  // sig = 2^g
      double b = ldexp(C.get(l, o, s), eslot[(size_t)lz * padded(S) + s] - g);
      // no share of a vector of zeros, whatever its coefficient (of one that is no number sig tells)
      if (!(fabs(b) <= 1.0)) b = 0.0;
      if (C.sgn) {
        long long X = llrint(ldexp(b, 56));
        for (int k = 6; k >= q; --k) {
          d = k == 0 ? (int)X : (int)((X + 128) & 0xFF) - 128;
          X = (X - d) >> 8;
        }
      } else {
        const unsigned long long X = (unsigned long long)llrint(ldexp(fabs(b), 56));
        d = (int)((X >> (48 - 8 * q)) & 0xFFu);
        if (b < 0.0) d = -d;
      }
    }
    f[i] = __int2half_rn(d);
  }
  unsigned char* dst = bimg + ((size_t)lz * ksteps_cap + kk) * (kSlices * OUT * kKStep * 2) + core_off(row, 8 * h);
  *reinterpret_cast<uint4*>(dst) = *reinterpret_cast<const uint4*>(f);
}

// ---- components far below their vectors' largest ---------------------------------------------
// The roundings of an output are relative to its scale, sig: at most S 2^-53 sig,
// ~sqrt(S) 2^-57 in the root mean square.  A part (real or imaginary) of an output element
// one of whose terms is at least 2^-kTermBits sig is served by that.  The elements with a
// part that has terms, but none such, go on a list (tc_witness_kernel) and take the FP64
// sum behind the pass (tc_rest_kernel); more of them than the list holds, and the
// vectors do not suit.  Dense vectors have next to none, and their elements show it
// by the one to six slots where an output's coefficient is largest: 35 us of the 16^3 x 32
// moments' 1.07 ms.
constexpr int kTermBits = 11;
constexpr int kMaxPass = kWideOut / 2;  // complex outputs a pass
// Words a slot: word d - 1 for components within d binades of the vector's scale,
// the outputs (bits, the real parts of coefficients below, the imaginary ones above)
// whose coefficients make a large term with them; the last but one the coefficients
// that are not zero.
constexpr int kLevels = kTermBits - 1, kMaskWords = kLevels + 2;
struct Components {
  unsigned* mask;               // [l][slot][kMaskWords]
  unsigned long long* largest;  // [l][kMaxPass] coefficient (as float bits) and slot of the largest, per output
  long long* list;              // l' n + element
  unsigned* count;
  unsigned cap;
};
__global__ void tc_masks_kernel(CoefView C, int O, int S, int stride, const unsigned* __restrict__ mx,
                                const int* __restrict__ eslot, const double* __restrict__ sig, Components k) {
  const int lz = blockIdx.y;
  for (int t = blockIdx.x * blockDim.x + threadIdx.x; t < S * O; t += gridDim.x * blockDim.x) {
    const int s = t / O, o = t % O;
    if (mx[(size_t)lz * S + s] == 0) continue;
    const double2 c = C.c[lz * C.sl + o * C.so + s * C.ss];
    const int d = eslot[(size_t)lz * padded(S) + s] - (exp_above(sig[(size_t)lz * stride + 2 * o]) - 1);
    const double re = fabs(ldexp(c.x, d)), im = fabs(ldexp(c.y, d));
    unsigned* m = k.mask + ((size_t)lz * S + s) * kMaskWords;
    const unsigned br = 1u << o, bi = 0x10000u << o;
    for (int v = 1; v <= kLevels; ++v) {
      const double least = ldexp(1.0, v - kTermBits);
      const unsigned bits = (re >= least ? br : 0) | (im >= least ? bi : 0);
      if (bits != 0) atomicOr(m + v - 1, bits);
    }
    atomicOr(m + kLevels, (c.x != 0.0 ? br : 0) | (c.y != 0.0 ? bi : 0));
    atomicMax(k.largest + lz * kMaxPass + o,
              (unsigned long long)__float_as_uint((float)fmax(re, im)) << 32 | (unsigned)s);
  }
}
__global__ void __launch_bounds__(256)
tc_witness_kernel(SlotMap map, long long n, int l0, int O, int S, const int* __restrict__ eslot, Components k,
                  int* __restrict__ err) {
  const int lz = blockIdx.y;
  const unsigned all = (1u << O) - 1;
  // the slots of the outputs' largest coefficients, each once, four to a turn
  // (their loads together: a turn is a pass over four vectors)
  __shared__ int s_slot[kMaxPass];
  __shared__ int s_slots;
  __shared__ bool s_done;  // the whole sum in FP64 already (other blocks of this launch may say so: read once)
  if (threadIdx.x < 32) {
    const int o = threadIdx.x;
    const int s = o < O ? (int)(unsigned)k.largest[lz * kMaxPass + o] : -1 - o;
    const bool first = (int)__ffs(__match_any_sync(0xffffffffu, s)) - 1 == o && o < O;
    const unsigned f = __ballot_sync(0xffffffffu, first);
    if (first) s_slot[__popc(f & ((1u << o) - 1))] = s;
    if (o == 0) {
      s_slots = __popc(f);
      s_done = (*reinterpret_cast<volatile int*>(err) & kErrSpread) != 0;
    }
  }
  __syncthreads();
  if (s_done) return;
  const int slots = s_slots;
  for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < n; e += (long long)gridDim.x * blockDim.x) {
    unsigned fr = 0, fi = 0, nr = 0, ni = 0;  // outputs whose real, imaginary part has a large term, a term
    auto at = [&](int s) { return __ldg(reinterpret_cast<const uint4*>(slot_ptr(map, n, l0 + lz, s)) + e); };
    auto visit = [&](uint4 x, int s) {
      const unsigned* m = k.mask + ((size_t)lz * S + s) * kMaskWords;
      const int top = __ldg(eslot + (size_t)lz * padded(S) + s) + 1023;
      // binades below the scale, at least one; past the levels: none
      const unsigned dr = (unsigned)(top - (int)(x.y >> 20 & 0x7FF)) - 1, di = (unsigned)(top - (int)(x.w >> 20 & 0x7FF)) - 1;
      const unsigned mr = dr < kLevels ? __ldg(m + dr) : 0, mi = di < kLevels ? __ldg(m + di) : 0, nz = __ldg(m + kLevels);
      const unsigned zr = (x.y << 1 | x.x) != 0 ? nz : 0, zi = (x.w << 1 | x.z) != 0 ? nz : 0;
      fr |= mr | mi >> 16;
      fi |= mi | mr >> 16;
      nr |= zr | zi >> 16;
      ni |= zi | zr >> 16;
      return (fr & fi & all) == all;
    };
    bool ok = false;
    for (int o = 0; o < slots && !ok; o += 4) {
      uint4 x[4];
#pragma unroll
      for (int i = 0; i < 4; ++i) x[i] = at(s_slot[min(o + i, slots - 1)]);
#pragma unroll
      for (int i = 0; i < 4; ++i) ok = visit(x[i], s_slot[min(o + i, slots - 1)]);
    }
    for (int s = 0; s < S && !ok; ++s) ok = visit(at(s), s);
    if (!ok && (((nr & ~fr) | (ni & ~fi)) & all) != 0) {
      const unsigned place = atomicAdd(k.count, 1u);
      if (place < k.cap)
        k.list[place] = (long long)lz * n + e;
      else
        atomicOr(err, kErrSpread);
    }
  }
}
// The listed elements' outputs in FP64, a thread each: the outputs of an element
// side by side read its components together.
__global__ void __launch_bounds__(256)
tc_rest_kernel(SlotMap map, long long n, int l0, CoefView C, int O, int S, Components k, long long out_l,
               double2* __restrict__ out, const int* __restrict__ err) {
  if ((*err & kErrSpread) != 0) return;
  const long long work = (long long)min(*k.count, k.cap) * O;
  for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < work; t += (long long)gridDim.x * blockDim.x) {
    const long long at = k.list[t / O], e = at % n;
    const int o = (int)(t % O), lz = (int)(at / n), l = l0 + lz;
    const double2* c = C.c + lz * C.sl + o * C.so;
    double re = 0.0, im = 0.0;
#pragma unroll 4
    for (int s = 0; s < S; ++s) {
      const double2 x = __ldg(reinterpret_cast<const double2*>(slot_ptr(map, n, l, s)) + e), w = c[s * C.ss];
      re = fma(w.x, x.x, fma(-w.y, x.y, re));
      im = fma(w.x, x.y, fma(w.y, x.x, im));
    }
    out[l * out_l + (long long)o * n + e] = make_double2(re, im);
  }
}

// A sum xh 2^32 + xl (|xh| < 2^50) times 2^e as a double, rounded to nearest
// from its leading 64 bits, by integers: the FP64 pipe, two a clock and SM, would
// take a third of the time of a short sum.
__device__ __forceinline__ double sum_to_double(long long xh, long long xl, int e) {
  long long t = xh + (xl >> 32);
  unsigned r = (unsigned)xl;
  const unsigned sg = (unsigned)(t >> 63) & 0x80000000u;
  if (t < 0) {
    t = ~t + (r == 0 ? 1 : 0);
    r = 0u - r;
  }
  const int lz = __clzll(t);
  const int k = 95 - lz + e + 1023;  // biased exponent of the leading bit
  if (t == 0 || k <= 0 || k >= 2046) {
    const double v = ldexp(fma((double)t, 0x1p32, (double)r), e);
    return sg ? -v : v;
  }
  unsigned long long m = (unsigned long long)t << lz;
  m |= lz <= 32 ? (unsigned long long)(r >> (32 - lz)) : (unsigned long long)r << (lz - 32);
  m = (m >> 11) + ((m >> 10) & 1);
  const unsigned long long bits = ((unsigned long long)(k - 1) << 52) + m;
  return __hiloint2double((int)((unsigned)(bits >> 32) | sg), (int)(unsigned)bits);
}

// ---- the combination ------------------------------------------------------------------------
// CPLX: complex coefficients (O real outputs, two for each complex one) and
// signed digits.  FF: float-float vectors, signed digits.  SHORT: at most 64 slots, so that a chunk's sums, below 2^22,
// turn into integers by an FP32 addition instead of a conversion (16 a clock
// and SM).  ACC: the sums are added to out.
template <bool CPLX, bool SHORT, bool ACC, bool WIDE, bool FF>
__global__ void __launch_bounds__(Form<WIDE>::kThreads, 1)
combine_tc_kernel(SlotMap map, long long n, int l0, int nl, const int* __restrict__ count, int S,
                  const int* __restrict__ eslot, const unsigned char* __restrict__ bimg, int ksteps_cap,
                  const double* __restrict__ sig, int O, long long out_l, double2* __restrict__ out,
                  int* __restrict__ err) {
  extern __shared__ unsigned char tc_smem_raw[];
  // vectors that do not suit, known before this launch: the FP64 sum follows
  if ((*err & kErrSpread) != 0) return;
  using F = Form<WIDE>;
  static_assert(CPLX || !WIDE, "the wide form's bound is that of signed digits");
  constexpr int kSliceStages = F::kSliceStages, kChunkSteps = F::kChunkSteps, kBBytes = F::kBBytes;
  constexpr int kE = F::kEpiOuts;
  TcShared<WIDE>* sh = reinterpret_cast<TcShared<WIDE>*>((reinterpret_cast<uintptr_t>(tc_smem_raw) + 1023) & ~(uintptr_t)1023);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const long long tiles_per_src = (2 * n + kRows - 1) / kRows;  // the last one may be short
  const long long tiles = tiles_per_src * nl;
  volatile int* abort = &sh->abort;

  if (threadIdx.x == 0) {
    for (int i = 0; i < kF64Stages; ++i) {
      bar_init(sh->full_f + i, 1);
      bar_init(sh->empty_f + i, kSliceWarps / 2);
    }
    for (int i = 0; i < kSliceStages; ++i) {
      bar_init(sh->full_s + i, kSliceWarps / 2);
      bar_init(sh->full_b + i, 1);
      bar_init(sh->empty_s + i, 1);
    }
    for (int i = 0; i < F::kBuffers; ++i) {
      bar_init(sh->tmem_full + i, 1);
      bar_init(sh->tmem_empty + i, kEpiWarps);
    }
    bar_init(&sh->mma_done, 1);
    sh->abort = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == kMmaWarp) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(su32(&sh->tmem_base)),
                 "r"(kTmemCols)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    tc_fence_before();
  }
  if (WIDE) {  // the zero rows ahead of B's
    constexpr int kPad = F::kPadBytes / 16;
    for (int i = threadIdx.x; i < kSliceStages * kPad; i += F::kThreads)
      reinterpret_cast<uint4*>(sh->sl[i / max(kPad, 1)].b)[i % max(kPad, 1)] = make_uint4(0, 0, 0, 0);
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  }
  __syncthreads();
  tc_fence_after();
  const unsigned tmem = sh->tmem_base;

  auto give_up = [&]() {
    *abort = 1;
    atomicOr(err, kErrWait);
  };

  // Wide: the epilogue's sums take the registers that the others can spare
  // (what they give up is at least what it takes: Form).
  if (warp < kEpiWarps) {
    if (WIDE) asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(F::kEpiRegs));
    // ---- epilogue: warp w reads lanes 32 (w % 4) .., outputs 8 (w / 4) .. ----
    const int quarter = warp & 3, half = warp >> 2;
    const unsigned lane_addr = tmem + ((unsigned)(32 * quarter) << 16);
    long long cc = 0;
    bool ok = true;
    for (long long t = blockIdx.x; t < tiles && ok; t += gridDim.x) {
      const int lz = (int)(t / tiles_per_src), l = l0 + lz;
      const long long row0 = (t % tiles_per_src) * kRows;
      const int cnt = slots_of(count, l, S), ks = (cnt + kKStep - 1) / kKStep;
      const int nch = (ks + kChunkSteps - 1) / kChunkSteps;
      // level sums combined exactly as they arrive: xh = I_0 2^16 + I_1 2^8 +
      // I_2 (< 2^48), xl = I_3 2^24 + I_4 2^16 + I_5 2^8 + I_6 (< 2^56)
      long long xh[kE], xl[kE];
#pragma unroll
      for (int i = 0; i < kE; ++i) xh[i] = xl[i] = 0;
      for (int c = 0; c < nch; ++c, ++cc) {
        if (!bar_wait_warp(sh->tmem_full + cc % F::kBuffers, (unsigned)((cc / F::kBuffers) & 1), abort)) {
          ok = false;
          break;
        }
        tc_fence_after();
        // level by level: the pairs of a level add up in 32 bits
#pragma unroll
        for (int lv = 0; lv < kSlices; ++lv) {
          if constexpr (WIDE) {
            const unsigned at =
                lane_addr + (unsigned)(cc % F::kBuffers * F::kBufferCols + lv * F::kO + kE * half);
            float f[16];
            tc_ld16(at, f);
#pragma unroll
            for (int i = 0; i < kE; ++i) {
              const int v = __float2int_rn(f[i]);
              if (lv <= 2)
                xh[i] += (long long)v * (1 << 8 * (2 - lv));
              else
                xl[i] += (long long)v * (1 << 8 * (6 - lv));
            }
            continue;
          }
          unsigned a[8];
#pragma unroll
          for (int p = 0; p <= lv; ++p) {
            float f[8];
            tc_ld8(lane_addr + (unsigned)(col_base(p) + kOut * (lv - p) + 8 * half), f);
#pragma unroll
            for (int i = 0; i < 8; ++i) {
              const unsigned v = SHORT ? __float_as_uint(f[i] + 12582912.0f) : (unsigned)__float2int_rn(f[i]);
              a[i] = p == 0 ? v : a[i] + v;
            }
          }
#pragma unroll
          for (int i = 0; i < 8; ++i) {
            if (SHORT) a[i] -= (lv + 1) * 0x4B400000u;
            if (lv <= 2)
              xh[i] += (long long)(int)a[i] * (1 << 8 * (2 - lv));
            else
              xl[i] += (long long)(int)a[i] * (1 << 8 * (6 - lv));
          }
        }
        tc_fence_before();
        __syncwarp();
        if (lane == 0) bar_arrive(sh->tmem_empty + cc % F::kBuffers);
      }
      if (!ok) break;
      // the output addresses are formed here, not kept live across the chunks
      long long r = row0 + 32 * quarter + lane;  // real row: element r / 2, part r % 2
      int lo = l, lzo = lz;
      asm volatile("" : "+l"(r), "+r"(lo), "+r"(lzo));
      if constexpr (!CPLX) {
#pragma unroll
        for (int i = 0; i < 8; ++i) {
          const int o = 8 * half + i;
          if (o < O && r < 2 * n) {
            // sum_l I_l 2^(-8 l) = 2^-16 xh + 2^-48 xl
            double v = fma((double)xl[i], 0x1p-48, (double)xh[i] * 0x1p-16);
            v *= sig[(size_t)lzo * kOut + o] * 0x1p-16;
            reinterpret_cast<double*>(out + lo * out_l + (long long)o * n)[r] = v;
          }
        }
      } else {
        // (c x).re = Re c x.re - Im c x.im, (c x).im = Re c x.im + Im c x.re: the
        // element's two parts sit in lanes 2 j and 2 j + 1, the sums with Re c
        // and Im c have one scale and add as integers
#pragma unroll
        for (int i = 0; i < kE; i += 2) {
          const int o = kE * half + i;
          if (o < O) {
            const long long m = lane & 1 ? 0 : -1;
            const long long bh = __shfl_xor_sync(0xffffffffu, xh[i + 1], 1);
            const long long bl = __shfl_xor_sync(0xffffffffu, xl[i + 1], 1);
            const double sc = sig[(size_t)lzo * F::kO + o];
            // sig 2^-64 (2^32 xh + xl); a scale that is no number poisons the sum
            double v = sum_to_double(xh[i] + (bh ^ m) - m, xl[i] + (bl ^ m) - m,
                                     (int)((unsigned)__double2hiint(sc) >> 20) - 1023 - 64);
            if (sc != sc) v = sc;
            if (r < 2 * n) {
              double* at = reinterpret_cast<double*>(out + lo * out_l + (long long)(o / 2) * n) + r;
              *at = ACC ? *at + v : v;
            }
          }
        }
      }
    }
    if (!ok) give_up();
  } else if (warp < kMmaWarp) {
    if (WIDE) asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(F::kOtherRegs));
    // ---- slices: the two halves of the warps take K-steps in turn; thread u
    // of a half <-> row u % 128, slots 8 (u / 128) .. (16-byte stores without
    // conflicts; one half's waits pass while the other works) ----
    constexpr int kPer = 8;
    static_assert(kPer * kSliceWarps / 2 * 32 == kKStep * kRows, "a K-step for half of the warps");
    const int turn = (warp - kEpiWarps) / (kSliceWarps / 2);
    const int u = (threadIdx.x - kEpiWarps * 32) & (kSliceWarps * 16 - 1);
    const int row = u & (kRows - 1), h = u >> 7;
    long long fc = 0, sc = 0, copied = -1;
    bool ok = true;
    for (long long t = blockIdx.x; t < tiles && ok; t += gridDim.x) {
      const int lz = (int)(t / tiles_per_src), l = l0 + lz;
      const int cnt = slots_of(count, l, S), ks = (cnt + kKStep - 1) / kKStep;
      for (int kk = 0; kk < ks; ++kk, ++fc, ++sc) {
        if ((int)(fc & 1) != turn) continue;
        const int fs = (int)(fc % kF64Stages), ss = (int)(sc % kSliceStages);
        // past the last slot: any scale and any numbers, finite digits that meet zeros in B
        const int4* ep = reinterpret_cast<const int4*>(eslot + (size_t)lz * padded(S) + kk * kKStep + kPer * h);
        const int4 e0 = __ldg(ep), e1 = __ldg(ep + 1);
        const int es[kPer] = {e0.x, e0.y, e0.z, e0.w, e1.x, e1.y, e1.z, e1.w};
        if (!bar_wait_warp(sh->full_f + fs, (unsigned)((fc / kF64Stages) & 1), abort)) {
          ok = false;
          break;
        }
        BytePairs X[kPer / 2];
        __half2 s1[kPer / 2], s2[kPer / 2];
#pragma unroll
        for (int i = 0; i < kPer; i += 2) {
          const int j = kPer * h + i;
          const double a = sh->f64[fs].v[j][row], b = sh->f64[fs].v[j + 1][row];
          if constexpr (FF) {
            const float* fa = reinterpret_cast<const float*>(sh->f64[fs].v[j]) + 4 * (row >> 1) + (row & 1);
            const float* fb = fa + 2 * kRows;
            X[i / 2] = byte_pairs(signed_digits(fa[0], fa[2], es[i]), signed_digits(fb[0], fb[2], es[i + 1]));
          } else if constexpr (CPLX) {
            X[i / 2] = byte_pairs(signed_digits(a, es[i]), signed_digits(b, es[i + 1]));
          } else {
            X[i / 2] = byte_pairs(fixed56(a, es[i]), fixed56(b, es[i + 1]));
            const unsigned sg =
                ((unsigned)__double2hiint(a) >> 16 & 0x8000u) | ((unsigned)__double2hiint(b) & 0x80000000u);
            const unsigned o1 = 0x3C003C00u ^ sg, o2 = 0xE400E400u ^ sg;
            s1[i / 2] = *reinterpret_cast<const __half2*>(&o1);
            s2[i / 2] = *reinterpret_cast<const __half2*>(&o2);
          }
        }
        __syncwarp();
        if (lane == 0) bar_arrive(sh->empty_f + fs);
        if (sc >= kSliceStages &&
            !bar_wait_warp(sh->empty_s + ss, (unsigned)((sc / kSliceStages - 1) & 1), abort)) {
          ok = false;
          break;
        }
        if (u == 0) {
          bar_arrive_tx(sh->full_b + ss, kBBytes);
          bulk_copy(sh->sl[ss].b + F::kPadBytes, bimg + ((size_t)lz * ksteps_cap + kk) * kBBytes, kBBytes,
                    sh->full_b + ss);
          copied = sc;
        }
        auto put = [&](auto pc) {
          constexpr int p = decltype(pc)::value;
          unsigned w[kPer / 2];
#pragma unroll
          for (int i = 0; i < kPer / 2; ++i) {
            if constexpr (CPLX || FF)
              w[i] = signed_pair<p>(X[i]);
            else
              w[i] = digit_pair<p>(X[i], s1[i], s2[i]);
          }
          unsigned char* dst = sh->sl[ss].a[p] + core_off(row, kPer * h);
          *reinterpret_cast<uint4*>(dst) = make_uint4(w[0], w[1], w[2], w[3]);
        };
        put(std::integral_constant<int, 0>{});
        put(std::integral_constant<int, 1>{});
        put(std::integral_constant<int, 2>{});
        put(std::integral_constant<int, 3>{});
        put(std::integral_constant<int, 4>{});
        put(std::integral_constant<int, 5>{});
        put(std::integral_constant<int, 6>{});
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        __syncwarp();
        if (lane == 0) bar_arrive(sh->full_s + ss);
      }
    }
    if (!ok) {
      give_up();
      // the copies of coefficients already issued land before the CTA can exit
      for (long long q = copied; q >= 0 && q > copied - kSliceStages; --q) {
        if (((q ^ copied) & 1) != 0) continue;  // the other half's
        const unsigned long long t0 = gtimer();
        while (!bar_test(sh->full_b + q % kSliceStages, (unsigned)((q / kSliceStages) & 1)) &&
               gtimer() - t0 < kTcWaitNs) {
        }
      }
    }
  } else {
    if (WIDE) asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(F::kOtherRegs));
    if (warp == kLoadWarp) {
    // ---- bulk copies of the FP64 residual rows: lane j issues slot j's ----
    // (one lane for all sixteen was the kernel's pace: each copy's address
    // takes a dependent load of the block table, ~3200 cycles a K-step)
    {
      long long fc = 0;
      bool ok = true;
      for (long long t = blockIdx.x; t < tiles && ok; t += gridDim.x) {
        const int lz = (int)(t / tiles_per_src), l = l0 + lz;
        const long long row0 = (t % tiles_per_src) * kRows;
        const int cnt = slots_of(count, l, S), ks = (cnt + kKStep - 1) / kKStep;
        for (int kk = 0; kk < ks; ++kk, ++fc) {
          const int st = (int)(fc % kF64Stages);
          const int nv = min(kKStep, cnt - kk * kKStep);
          const double* src = lane < nv ? slot_ptr(map, n, l, kk * kKStep + lane) + row0 : nullptr;
          // rows of a short tile past the end keep what the stage held: their sums are not stored
          const unsigned bytes = (unsigned)min((long long)kRows, 2 * n - row0) * 8u;
          if (fc >= kF64Stages && !bar_wait_warp(sh->empty_f + st, (unsigned)((fc / kF64Stages - 1) & 1), abort)) {
            ok = false;
            break;
          }
          if (lane == 0) bar_arrive_tx(sh->full_f + st, (unsigned)nv * bytes);
          __syncwarp();
          if (lane < nv) bulk_copy(sh->f64[st].v[lane], src, bytes, sh->full_f + st);
        }
      }
      if (!ok) {
        give_up();
        // the copies already issued land before the CTA can exit
        for (long long q = fc - 1; q >= 0 && q >= fc - kF64Stages; --q) {
          const int st = (int)(q % kF64Stages);
          const unsigned long long t0 = gtimer();
          while (!bar_test(sh->full_f + st, (unsigned)((q / kF64Stages) & 1)) && gtimer() - t0 < kTcWaitNs) {
          }
        }
      }
    }
    } else if (warp == kMmaWarp) {
    // ---- MMA issue (one thread) ----
    if (lane == 0) {
      long long sc = 0, cc = 0;
      bool ok = true;
      for (long long t = blockIdx.x; t < tiles && ok; t += gridDim.x) {
        const int l = l0 + (int)(t / tiles_per_src);
        const int cnt = slots_of(count, l, S), ks = (cnt + kKStep - 1) / kKStep;
        for (int kk = 0; kk < ks; ++kk, ++sc) {
          const int ss = (int)(sc % kSliceStages);
          if (kk % kChunkSteps == 0) {
            if (cc >= F::kBuffers &&
                !bar_wait(sh->tmem_empty + cc % F::kBuffers, (unsigned)((cc / F::kBuffers - 1) & 1), abort)) {
              ok = false;
              break;
            }
            tc_fence_after();
          }
          if (!bar_wait(sh->full_s + ss, (unsigned)((sc / kSliceStages) & 1), abort) ||
              !bar_wait(sh->full_b + ss, (unsigned)((sc / kSliceStages) & 1), abort)) {
            ok = false;
            break;
          }
          tc_fence_after();
          const unsigned acc = (kk % kChunkSteps) != 0 ? 1u : 0u;
#pragma unroll
          for (int p = 0; p < kSlices; ++p) {
            const unsigned long long ad = smem_desc(sh->sl[ss].a[p], kLbo, kSbo);
            if constexpr (WIDE)
              // all levels, the first p times zero rows: products of one shape and place run in order
              tc_mma(tmem + (unsigned)(cc % F::kBuffers * F::kBufferCols), ad,
                     smem_desc(sh->sl[ss].b + F::kPadBytes - p * (F::kO * kKStep * 2), kLbo, kSbo),
                     idesc_f16(kRows, F::kBRows), p > 0 ? 1u : acc);
            else
              tc_mma(tmem + (unsigned)col_base(p), ad, smem_desc(sh->sl[ss].b, kLbo, kSbo),
                     idesc_f16(kRows, kOut * (kSlices - p)), acc);
          }
          tc_commit(sh->empty_s + ss);
          if (kk % kChunkSteps == kChunkSteps - 1 || kk == ks - 1) {
            tc_commit(sh->tmem_full + cc % F::kBuffers);
            ++cc;
          }
        }
      }
      if (!ok) give_up();
      // every MMA issued has completed before the tensor memory is freed
      tc_commit(&sh->mma_done);
      const unsigned long long t0 = gtimer();
      while (!bar_test(&sh->mma_done, 0u) && gtimer() - t0 < kTcWaitNs) {
      }
    }
    }
  }
  __syncthreads();
  if (warp == kMmaWarp) {
    __syncwarp();
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(kTmemCols) : "memory");
  }
}

struct TcWork {
  unsigned long long* ex;
  unsigned* mx;
  int* eslot;
  double* sig;
  unsigned char* bimg;
  int* err;
};
size_t align256(size_t b) { return (b + 255) / 256 * 256; }
TcWork carve(void* w, int nl, int S, int ksteps_cap) {
  char* p = static_cast<char*>(w);
  TcWork t;
  t.ex = reinterpret_cast<unsigned long long*>(p);
  p += align256(sizeof(unsigned long long) * (size_t)nl * S);
  t.mx = reinterpret_cast<unsigned*>(p);
  p += align256(sizeof(unsigned) * (size_t)nl * S);
  t.eslot = reinterpret_cast<int*>(p);
  p += align256(sizeof(int) * (size_t)nl * padded(S));
  t.sig = reinterpret_cast<double*>(p);
  p += align256(sizeof(double) * (size_t)nl * kWideOut);
  t.err = reinterpret_cast<int*>(p);
  p += 256;
  t.bimg = reinterpret_cast<unsigned char*>(p);
  return t;
}

}  // namespace

bool combine_tc_enabled() {
  // SSQCD_MOMENTS_TC=0: the FP64-pipe combination instead (comparison runs)
  static const bool on = [] {
    const char* e = std::getenv("SSQCD_MOMENTS_TC");
    return !(e != nullptr && std::atoi(e) == 0);
  }();
  return on;
}

bool combine_tc_applicable(long long n, int O, int S) {
  return O >= 1 && O <= kOut && n > 0 && S >= 1 && S <= kMaxCount;
}

namespace {
// Elements that the list of tc_witness_kernel holds: a 64th of all, whose FP64
// sums cost a few percent of everyone's.  (Where one slot has an output's only
// large coefficient, 1.3% of a Gaussian vector's elements are on it.)
unsigned rest_cap(long long n, int nl) { return (unsigned)std::min(n * nl / 64 + 64, 1LL << 28); }
}  // namespace

size_t combine_tc_vectors_work_bytes(long long n, int nl, int S) {
  return combine_tc_work_bytes(nl, S) + align256(sizeof(unsigned) * kMaskWords * (size_t)nl * S) +
         align256(sizeof(unsigned long long) * (size_t)nl * kMaxPass) + 256 +
         sizeof(long long) * (size_t)rest_cap(n, nl);
}

size_t combine_tc_work_bytes(int nl, int S) {
  const int ks = (S + kKStep - 1) / kKStep;
  return align256(sizeof(unsigned long long) * (size_t)nl * S) + align256(sizeof(unsigned) * (size_t)nl * S) +
         align256(sizeof(int) * (size_t)nl * padded(S)) +
         align256(sizeof(double) * (size_t)nl * kWideOut) + 256 + (size_t)nl * ks * Form<true>::kBBytes;
}

namespace {

// The scale pass, then a launch for every kOut real (kOut / 2 complex) outputs.
// suits (may be null): set to false, the outputs then not to be used, when a
// vector has too wide a spread (kMaxSpread), an infinity or a NaN; with add
// (complex coefficients: the sums are added to out) that is found out before
// out is touched.  comps (may be null; complex coefficients, not with add):
// elements with small components take the FP64 sum.
int combine_all(const SlotMap& map, long long n, CoefView C, int O, int S, const int* count, double2* out,
                long long out_l, int l0, int nl, void* work, cudaStream_t st, bool* suits, bool add = false,
                bool ff = false, const Components* comps = nullptr) {
  const int ks = (S + kKStep - 1) / kKStep;
  TcWork w = carve(work, nl, S, ks);
  unsigned long long* ex = suits != nullptr ? w.ex : nullptr;
  SS_CUDA(cudaMemsetAsync(w.mx, 0, sizeof(unsigned) * (size_t)nl * S, st));
  if (ex != nullptr) SS_CUDA(cudaMemsetAsync(ex, 0, sizeof(unsigned long long) * (size_t)nl * S, st));
  SS_CUDA(cudaMemsetAsync(w.err, 0, sizeof(int), st));
  // blocks of at least 4 elements a thread
  const unsigned gx = (unsigned)std::max(1LL, std::min(64LL, (n + 1023) / 1024));
  auto* maxabs = ff ? tc_maxabs_kernel<true> : tc_maxabs_kernel<false>;
  maxabs<<<dim3(gx, S, nl), 256, 0, st>>>(map, n, l0, count, S, w.mx, ex);
  SS_CHECK_LAUNCH();
  int dev = 0, sms = 0;
  SS_CUDA(cudaGetDevice(&dev));
  SS_CUDA(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
  const long long tiles = ((2 * n + kRows - 1) / kRows) * nl;
  const int grid = (int)(tiles < sms ? tiles : sms);
  // a pass: its first output, its outputs, and whether it is a wide one
  auto* wide_kern = add ? combine_tc_kernel<true, false, true, true, false> : combine_tc_kernel<true, false, false, true, false>;
  bool wide_ok = C.cplx && O > kOut / 2;
  if (wide_ok) {  // its warps share out the registers of the launch: as many as the shares add up to, or the narrow form
    cudaFuncAttributes at;
    SS_CUDA(cudaFuncGetAttributes(&at, wide_kern));
    wide_ok = at.numRegs >= Form<true>::kRegs;
  }
  auto wide_at = [&](int o0) { return wide_ok && O - o0 > kOut / 2; };
  auto outs_at = [&](int o0) { return std::min(O - o0, !C.cplx ? kOut : wide_at(o0) ? kWideOut / 2 : kOut / 2); };
  auto scales = [&](int o0) {
    CoefView Cp = C;
    Cp.c += o0 * C.so;
    const int Op = (C.cplx ? 2 : 1) * outs_at(o0);
    if (wide_at(o0))
      tc_scales_kernel<kWideOut><<<nl * kWideOut, 256, 0, st>>>(w.mx, Cp, Op, S, l0, count, w.eslot, w.sig, ex, n, w.err);
    else
      tc_scales_kernel<kOut><<<nl * kOut, 256, 0, st>>>(w.mx, Cp, Op, S, l0, count, w.eslot, w.sig, ex, n, w.err);
  };
  int h_err = 0;
  if (add) {  // every output's scales first
    for (int o0 = 0; o0 < O; o0 += outs_at(o0)) {
      scales(o0);
      SS_CHECK_LAUNCH();
      count_launches(1);
    }
    SS_CUDA(cudaMemcpyAsync(&h_err, w.err, sizeof(int), cudaMemcpyDeviceToHost, st));
    SS_CUDA(cudaStreamSynchronize(st));
    if (suits != nullptr) *suits = h_err == 0;
    if (h_err != 0) return SSQCD_OK;
  }
  for (int o0 = 0; o0 < O; o0 += outs_at(o0)) {
    const bool wide = wide_at(o0);
    CoefView Cp = C;
    Cp.c += o0 * C.so;
    const int Op = (C.cplx ? 2 : 1) * outs_at(o0);
    auto* kern = wide    ? wide_kern
                 : add    ? combine_tc_kernel<true, false, true, false, false>
                 : C.cplx ? (S <= 64 ? combine_tc_kernel<true, true, false, false, false>
                                     : combine_tc_kernel<true, false, false, false, false>)
                 : ff     ? combine_tc_kernel<false, false, false, false, true>
                 : S <= 64 ? combine_tc_kernel<false, true, false, false, false>
                           : combine_tc_kernel<false, false, false, false, false>;
    const size_t smem = (wide ? sizeof(TcShared<true>) : sizeof(TcShared<false>)) + 1024;
    SS_CUDA(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));  // the same every time
    scales(o0);
    SS_CHECK_LAUNCH();
    if (comps != nullptr) {
      SS_CUDA(cudaMemsetAsync(comps->mask, 0, (char*)(comps->count + 1) - (char*)comps->mask, st));
      tc_masks_kernel<<<dim3(std::min((S * (Op / 2) + 255) / 256, 64), nl), 256, 0, st>>>(
          Cp, Op / 2, S, wide ? kWideOut : kOut, w.mx, w.eslot, w.sig, *comps);
      SS_CHECK_LAUNCH();
      tc_witness_kernel<<<dim3((unsigned)std::min((n + 255) / 256, 16LL * sms), nl), 256, 0, st>>>(
          map, n, l0, Op / 2, S, w.eslot, *comps, w.err);
      SS_CHECK_LAUNCH();
      count_launches(2);
    }
    if (wide)
      tc_bslices_kernel<kWideOut><<<dim3(ks, nl), 2 * Form<true>::kBRows, 0, st>>>(Cp, Op, S, l0, count, w.eslot, w.sig,
                                                                                   ks, w.bimg);
    else
      tc_bslices_kernel<kOut><<<dim3(ks, nl), 2 * Form<false>::kBRows, 0, st>>>(Cp, Op, S, l0, count, w.eslot, w.sig, ks,
                                                                                w.bimg);
    SS_CHECK_LAUNCH();
    kern<<<grid, wide ? Form<true>::kThreads : Form<false>::kThreads, smem, st>>>(
        map, n, l0, nl, count, S, w.eslot, w.bimg, ks, w.sig, Op, out_l, out + (long long)o0 * n, w.err);
    SS_CHECK_LAUNCH();
    count_launches(3);
    if (comps != nullptr) {
      tc_rest_kernel<<<8 * sms, 256, 0, st>>>(map, n, l0, Cp, Op / 2, S, *comps, out_l, out + (long long)o0 * n,
                                             w.err);
      SS_CHECK_LAUNCH();
      count_launches(1);
    }
  }
  count_launches(1);
  SS_CUDA(cudaMemcpyAsync(&h_err, w.err, sizeof(int), cudaMemcpyDeviceToHost, st));
  SS_CUDA(cudaStreamSynchronize(st));
  if (h_err & kErrWait) return fail(SSQCD_ERR_NOCONV, "combination (tensor cores): a device-side wait hit its limit");
  if (suits != nullptr) *suits = h_err == 0;
  return SSQCD_OK;
}

}  // namespace

int combine_tc(char* const* tab, int basis_log, long long n, int L, const double2* C, int O, int S,
               const int* count, double2* out, int l0, int nl, void* work, cudaStream_t st, bool ff, bool* suits) {
  if (!combine_tc_applicable(n, O, S)) return fail(SSQCD_ERR_ARG, "combine_tc: shape not supported");
  return combine_all(SlotMap{tab, basis_log, L, nullptr, 0}, n, CoefView{C, (long long)O * S, S, 1, false, ff}, O, S, count,
                     out, (long long)O * n, l0, nl, work, st, suits, false, ff);
}

int combine_tc_complex(char* const* tab, int basis_log, long long n, int L, const double2* C, int O, int S,
                       const int* count, double2* out, int l0, int nl, void* work, cudaStream_t st, bool* suits,
                       bool add) {
  if (O < 1 || !combine_tc_applicable(n, 1, S)) return fail(SSQCD_ERR_ARG, "combine_tc: shape not supported");
  return combine_all(SlotMap{tab, basis_log, L, nullptr, 0}, n, CoefView{C, (long long)O * S, S, 1, true, true}, O, S, count,
                     out, (long long)O * n, l0, nl, work, st, suits, add);
}

int combine_tc_vectors(const double2* x, int S, long long n, const double2* C, int O, double2* out, int nl, void* work,
                       cudaStream_t st, bool* suits) {
  if (O < 1 || nl < 1 || !combine_tc_applicable(n, 1, S)) return fail(SSQCD_ERR_ARG, "combine_tc: shape not supported");
  Components k;
  char* p = static_cast<char*>(work) + combine_tc_work_bytes(nl, S);
  k.mask = reinterpret_cast<unsigned*>(p);
  p += align256(sizeof(unsigned) * kMaskWords * (size_t)nl * S);
  k.largest = reinterpret_cast<unsigned long long*>(p);
  p += align256(sizeof(unsigned long long) * (size_t)nl * kMaxPass);
  k.count = reinterpret_cast<unsigned*>(p);  // cleared with the two before it
  k.list = reinterpret_cast<long long*>(p + 256);
  k.cap = rest_cap(n, nl);
  return combine_all(SlotMap{nullptr, 0, 1, x, S}, n, CoefView{C, 0, 1, O, true, true}, O, S, nullptr, out, (long long)O * n,
                     0, nl, work, st, suits, false, false, &k);
}

}  // namespace ssqcd
