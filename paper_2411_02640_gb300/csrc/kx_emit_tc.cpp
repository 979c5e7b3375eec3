// Emitter of the tensor-core transport and thermo kernels (tcgen05, sm_103a).
//
// The mixing sums of the transport properties are products of a state's mass
// fractions with matrices that depend on temperature alone, and those are
// expanded in a few functions of temperature (kx_tc_basis.h), so that
//   R_r = sum_m phi_m(t) sum_j v_j c_rj,m
// with constant c: a matrix product of the states (M = 128 a tile) with
// N_s x rows x (M + 1) constants, and a short sum over m per state and row.
//
// Float64 accuracy from float16 operands: v_j (a state's Y_j 2^ecol_j scaled
// by a power of two to a largest magnitude in [1/2, 1)) and c are each cut
// into digits of 10 bits (integers in [-512, 512], exact in float16); the
// products of digit i of v with digit j of c, i + j = l, are accumulated by
// the tensor cores in one float32 accumulator per level l.  Integer sums
// below 2^24 are exact there, so the levels carry the 50-bit fixed-point
// product without rounding (the splitting scheme of Ozaki et al., Numer.
// Algorithms 59 (2012), on float16 units as in Mukunoki et al., ISC 2020),
// and the kernel adds the levels up in float pairs.  The first level's sum is
// 2^18 sum v c, and those after it add products of lower digits, whose signs
// are as good as random: with sum v c <= kSumMost a level stays below 0.9 x 2^24
// for states of like mass fractions too.  53/325's rows reach sum |c| = 33.7;
// 160/900's 108, and there a state's v are halved until sum v <= kSumMost.  A coefficient set whose
// basis function is scaled by 2^E_m takes (50 + E_m)/10 digits.  Mixed
// precision takes digits up to 2^-27 and adds the levels in float32.
//
// Per tile of 128 states: the 16 compute warps (four groups of four warps, each
// holding the tile's states once and sharing species and rows) turn Y into digits
// straight into tensor memory (operand A), evaluate phi_m, then per stage (16 rows
// x as many sets of accumulator columns as half the free tensor memory holds) read
// the accumulators and add them up.  One warp streams the coefficient digits
// (operand B) into a ring of shared-memory slots with bulk copies, one issues the
// matrix instructions; accumulators are double-buffered, so the tensor cores work
// on the next stage while the compute warps add up this one.  States outside
// 200-4000 K (or with non-finite Y) and rows whose sum is small beside the state's
// largest v (a nearly pure state's own row) are evaluated pair by pair in float
// pairs instead.
//
// Thermo (part 3) is the same with one stage: the mixture's polynomial coefficients,
// per T_mid group and range, as rows of an exact basis (tc_thermo), then c_p and h per
// state.  53/325: 39 -> 12 us up to 16k states (one thread per state took that state's
// 53 x 11 dependent float-pair steps), 49152 states 39 -> 20 us; 160/900 121 -> 14 us.
//
// What bounds it (53/325, GB300): instruction issue and the latencies between the
// stages of a tile (57-66 % of issue slots at four warps per scheduler; the matrix
// products take 24-28 % of the tensor pipe's cycles).  Against the float-pair loops
// over species pairs (one thread per state, 0.75-0.8 of the float32 pipe), per 2^20
// states: viscosity and conductivity 4.17 -> 1.30 ms, diffusion 6.43 -> 1.03 ms,
// mixed 2.06 -> 0.43 and 2.00 -> 0.54 ms; 997 states (few tiles: latency; the blocks
// of a column share a tile's rows) 214 -> 37 and 307 -> 24 us; 160/900 at 2^18 states
// 15.8 -> 2.1 and 16.5 -> 1.4 ms; 9/21 at 2^20 states 0.41 -> 0.37 and 0.49 -> 0.40 ms.
// Errors against 64 bits (rms relative): 1.7e-14 -> 0.8e-14 (viscosity), 1.0e-14 ->
// 1.0e-14 (conductivity), 2.2e-14 -> 1.1e-14 (diffusion).
// Operand A in tensor memory: from shared memory each instruction re-reads its 4 KB
// of A, 32 + N/4 cycles against N/2 here (N = 16 .. 64 columns; measured).  Two
// blocks per SM with half the tensor memory each were no faster (25 against 23 us a
// tile: single stages of 16 columns, and two instruction streams in one cache).
#include <algorithm>
#include <cmath>
#include <cstring>
#include <functional>

#include "kx_emit_text.h"
#include "kx_internal.h"
#include "kx_tc_basis.h"

namespace kx {

extern const char* kTables;

namespace {

const char* kTcPrelude = R"KXTC(
// ---- tensor memory, tcgen05 and mbarrier primitives
#define KX_WAIT_LIMIT (1 << 22)
__device__ __forceinline__ unsigned kx_smem(const void* p) { return (unsigned)__cvta_generic_to_shared(p); }
__device__ __forceinline__ void kx_mb_init(unsigned a, unsigned count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(a), "r"(count) : "memory");
}
__device__ __forceinline__ void kx_mb_arrive(unsigned a) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(a) : "memory");
}
__device__ __forceinline__ void kx_mb_expect(unsigned a, unsigned bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(a), "r"(bytes) : "memory");
}
// Waits for the phase of the given parity to complete; false after KX_WAIT_LIMIT polls.
__device__ __forceinline__ bool kx_mb_wait(unsigned a, unsigned parity) {
  for (int t = 0; t < KX_WAIT_LIMIT; ++t) {
    unsigned ok;
    asm volatile("{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\tselp.u32 %0, 1, 0, p;\n\t}"
                 : "=r"(ok) : "r"(a), "r"(parity) : "memory");
    if (ok) return true;
  }
  return false;
}
// One lane of a converged warp.  The matrix instructions take their operands from uniform registers; behind
// an elected lane they issue in 11 cycles, behind a plain lane == 0 test in 50 (measured, N = 16).
__device__ __forceinline__ bool kx_elect() {
  unsigned p;
  asm volatile("{\n\t.reg .pred P;\n\telect.sync _|P, 0xffffffff;\n\tselp.u32 %0, 1, 0, P;\n\t}" : "=r"(p));
  return p != 0;
}
__device__ __forceinline__ void kx_bulk_load(unsigned dst, const void* src, unsigned bytes, unsigned bar) {
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(dst), "l"(src),
               "r"(bytes), "r"(bar) : "memory");
}
__device__ __forceinline__ void kx_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void kx_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void kx_commit(unsigned bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar) : "memory");
}
// D[128 x N] (+)= A (tensor memory, float16) * B (shared memory descriptor, float16), float32 accumulation
__device__ __forceinline__ void kx_mma(unsigned d, unsigned a, unsigned long long b, unsigned idesc, unsigned acc) {
  asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\ttcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n\t}" ::"r"(d),
               "r"(a), "l"(b), "r"(idesc), "r"(acc) : "memory");
}
__device__ __forceinline__ void kx_ld(unsigned (&r)[4], unsigned a) {
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0, %1, %2, %3}, [%4];" : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(a));
}
__device__ __forceinline__ void kx_ld(unsigned (&r)[8], unsigned a) {
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]) : "r"(a));
}
__device__ __forceinline__ void kx_wait_ld() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }
__device__ __forceinline__ void kx_st2(unsigned a, const unsigned* r) {
  asm volatile("tcgen05.st.sync.aligned.32x32b.x2.b32 [%0], {%1, %2};" ::"r"(a), "r"(r[0]), "r"(r[1]) : "memory");
}
__device__ __forceinline__ void kx_st4(unsigned a, const unsigned* r) {
  asm volatile("tcgen05.st.sync.aligned.32x32b.x4.b32 [%0], {%1, %2, %3, %4};" ::"r"(a), "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3])
               : "memory");
}
__device__ __forceinline__ void kx_st8(unsigned a, const unsigned* r) {
  asm volatile("tcgen05.st.sync.aligned.32x32b.x8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"r"(a), "r"(r[0]), "r"(r[1]), "r"(r[2]),
               "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]) : "memory");
}
__device__ __forceinline__ void kx_wait_st() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }
// two digits 0..1024 in the halves of w, with 0x6400 in each (1024 + n as float16): the float16 integers n - 512
__device__ __forceinline__ unsigned kx_digits(unsigned w) {
  unsigned r;
  asm("sub.rn.f16x2 %0, %1, %2;" : "=r"(r) : "r"(w), "r"(0x66006600u));
  return r;
}
// 10 bits of a in the low half and 10 bits of b in the high half
__device__ __forceinline__ unsigned kx_pack(unsigned a, unsigned b) { return (a & 0x3ffu) | 0x64006400u | (b & 0x3ff0000u); }
__device__ __forceinline__ float kx_rcp(float x) {
  float r;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
  return r;
}
// a / b of float pairs in float32's normal range (kx_df_div without its range handling)
__device__ __forceinline__ kx_df kx_div_n(kx_df a, kx_df b) {
  float rb = kx_rcp(b.hi);
  rb = __fmaf_rn(rb, __fmaf_rn(-b.hi, rb, 1.0f), rb);
  const float q1 = __fmul_rn(a.hi, rb);
  const float p = __fmul_rn(q1, b.hi);
  const float pe = __fmaf_rn(q1, b.hi, -p);
  const float r = __fadd_rn(__fsub_rn(__fsub_rn(a.hi, p), pe), __fmaf_rn(-q1, b.lo, a.lo));
  return kx_qts(q1, __fmul_rn(r, rb));
}
// x 2^s as a float pair, by its bit fields and without branches: 24 bits and the rounded rest; 0 below float32's
// normal range (the result is below 2^100 where it is used)
__device__ __forceinline__ kx_df kx_pair_shift(double x, int s) {
  const unsigned hi = (unsigned)__double2hiint(x), lo = (unsigned)__double2loint(x);
  const int e = (int)((hi >> 20) & 0x7ffu) + s - 896;
  const unsigned sg = hi & 0x80000000u;
  const unsigned h = (__funnelshift_l(lo, hi, 3) & 0x7fffffu) | ((unsigned)e << 23);
  const float l = __fmul_rn(__uint2float_rn(lo & 0x1fffffffu), __int_as_float(max(e - 52, 0) << 23));
  return kx_mk(__uint_as_float(e > 0 ? h | sg : 0u), __uint_as_float(e > 52 ? __float_as_uint(l) | sg : 0u));
}
__device__ __forceinline__ float kx_float_shift(double x, int s) {
  const unsigned hi = (unsigned)__double2hiint(x), lo = (unsigned)__double2loint(x);
  const int e = (int)((hi >> 20) & 0x7ffu) + s - 896;
  const unsigned h = (__funnelshift_l(lo, hi, 3) & 0x7fffffu) | ((unsigned)e << 23);
  return __uint_as_float(e > 0 ? h | (hi & 0x80000000u) : 0u);
}
__device__ __forceinline__ void kx_copy8(unsigned dst, const double* src) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(dst), "l"(src) : "memory");
}
// (hi + lo) 2^x of a normalised float pair as a double, without the float64 pipe: lo in units of hi's last double
// place is an integer below 2^28, added to the bit pattern (doubled where it takes hi below its power of two,
// whose places are half as wide).
__device__ __forceinline__ double kx_df2d_b(kx_df a, int x) {
  const unsigned u = __float_as_uint(a.hi);
  const int e = (int)((u >> 23) & 0xffu);
  int l = __float2int_rn(__fmul_rn(__fmul_rn(a.lo, __int_as_float((254 - e) << 23)), 0x1p52f));   // 2^(52 - (e - 127))
  if ((int)u < 0) l = -l;
  if ((u & 0x7fffffu) == 0u && l < 0) l += l;
  const unsigned long long b = ((unsigned long long)((u & 0x80000000u) | ((unsigned)(e + 896 + x) << 20) | ((u & 0x7fffffu) >> 3)) << 32) | (u << 29);
  return __longlong_as_double((long long)(b + (unsigned long long)(long long)l));
}
)KXTC";

// e^x of a float pair, |x| < 80, to about 2^-47: kx_df_exp with r^2/2 kept as an exact product pair.  For the
// factors that every result of a state carries, where the shorter form's 5e-14 would not average out.
const char* kTcExp = R"KXTC(
__device__ __forceinline__ kx_df kx_df_exp_x(kx_df x) {
  const float tk = __fmaf_rn(x.hi, KX_256_OVER_LN2F, KX_RND_F);
  const int k = __float_as_int(tk) - 0x4b400000;
  const float kf = __fsub_rn(tk, KX_RND_F);
  const float t1 = __fmaf_rn(-kf, KX_C1F, x.hi);
  const float p = __fmul_rn(kf, KX_C2F);
  const float pe = __fmaf_rn(kf, KX_C2F, -p);
  kx_df r = kx_ts(t1, -p);
  r = kx_ts(r.hi, __fadd_rn(r.lo, __fsub_rn(__fsub_rn(x.lo, pe), __fmul_rn(kf, KX_C3F))));
  const float h = __fmul_rn(0.5f, r.hi), h2 = __fmul_rn(h, r.hi), he = __fmaf_rn(h, r.hi, -h2);
  const float tail = __fmul_rn(__fmul_rn(h2, r.hi), __fmaf_rn(__fmaf_rn(r.hi, 1.66666667e-2f, 8.33333333e-2f), r.hi, 0.333333333f));
  const kx_df s = kx_qts(r.hi, h2);
  const kx_df e = kx_mk(s.hi, __fadd_rn(__fadd_rn(s.lo, r.lo), __fadd_rn(tail, __fmaf_rn(r.hi, r.lo, he))));
  const float2 tj = kx_s_dexp[k & 255];
  const kx_df v = kx_df_fma(kx_mk(tj.x, tj.y), e, kx_mk(tj.x, tj.y));
  const float sc = __int_as_float(((k >> 8) + 127) << 23);
  return kx_mk(__fmul_rn(v.hi, sc), __fmul_rn(v.lo, sc));
}
)KXTC";

constexpr int kFloatE = -22;              // a basis function scaled by 2^-22 or less is added up in float32
constexpr int kPhiE = -30;                // ... by 2^-30 or less evaluated in float32: a polynomial of degree 18 in a
                                         // rounded t is off by 2^-16 (t = +-1) to 2^-20 of itself
constexpr int kMidE = -14;                // ... by 2^-14 or less with one exact product
constexpr int kDigit = 10;                 // bits of a digit
constexpr int kSumMost = 40;               // largest sum v c of a row and basis function
constexpr int kStates = 128, kRowsChunk = 16, kGroups = 4;   // states a tile; rows a chunk; groups of 128 compute threads

struct Stage {
  int m0 = 0, m1 = 0;                      // basis functions [m0, m1)
  int units = 0;                           // accumulator groups of 16 columns
  std::vector<int> ubase, count;           // by level 2..6: first unit, basis functions
  std::vector<int> dcount, doff;           // by digit 1..5: basis functions stored, byte offset in the slot
  int tails = 0;                           // basis functions whose level-7 products join level 6
  std::vector<int> toff;                   // by digit 2..5: offset of its copy scaled by 2^-10
  int bytes = 0, offset = 0;               // slot bytes; offset in a chunk's data
};

struct Plan {
  TcBasis b;
  bool mixed = false;
  bool bound_v = false;                    // some row's sum |c| exceeds kSumMost
  int part = 1;
  int nd = 5;                              // digits of v
  std::vector<int> lev;                    // digits (and levels) of basis function m
  std::vector<Stage> st;
  int acols = 0, dcols = 0, nbuf = 2, slots = 0, slot_bytes = 0, chunk_bytes = 0, chunks = 0;
  int smem = 0;
  int red = 24;                            // rows of 128 values exchanged between the compute groups
  std::vector<double> mids;                // thermo: the distinct T_mid
};

std::string hex64(unsigned long long v) { return fmt("0x%llxULL", v); }

bool make_plan(const Mechanism& m, const EmitOptions& opt, Plan& p) {
  p.mixed = opt.mixed;
  p.part = opt.part;
  if (opt.part == 3 ? !tc_thermo(m, p.b, p.mids) : !tc_basis(m, opt.part, opt.mixed, p.b)) return false;
  const TcBasis& b = p.b;
  p.nd = opt.mixed ? 3 : 5;
  for (int r = 0; r < b.rows; ++r)
    for (int q = 0; q <= b.M; ++q) {
      double sum = 0;
      for (int j = 0; j < b.ns; ++j) sum += std::fabs(b.coef[((size_t)r * b.ns + j) * (b.M + 1) + q]);
      p.bound_v |= !opt.mixed && sum > kSumMost;   // (mixed: float32's rounding is what it allows)
    }
  // digits that keep each set's dropped products near 2^-48 of the largest v (mixed: 2^-26)
  const double bits = opt.mixed ? 26.0 : 50.0;
  p.lev.resize(b.M + 1);
  for (int q = 0; q <= b.M; ++q) p.lev[q] = std::min(p.nd, std::max(1, (int)std::ceil((bits + b.E[q]) / kDigit)));
  for (int q = b.M; q > 0; --q) p.lev[q - 1] = std::max(p.lev[q - 1], p.lev[q]);
  // the leading coefficient sets also take the products of level 7 (of 2^-10 the size of level 6's, so a
  // copy of the coefficient digits scaled by 2^-10 adds them to the same accumulators): dropped, they are
  // the largest error of a sum (2^-47 of the largest v, against 2^-49 from the digits' own rounding)
  auto tail = [&](int q) { return !opt.mixed && p.lev[q] == p.nd && b.E[q] >= -2; };
  p.acols = p.nd * b.K / 2;
  const int left = 512 - p.acols;
  p.nbuf = 2;
  int cap = left / 2 / 16;
  if (cap < p.nd + 2) { p.nbuf = 1; cap = left / 16; }
  cap = std::min(cap, 16);
  if (cap < p.nd) return false;
  p.dcols = cap * 16;
  // stages: consecutive basis functions, at most `cap` accumulator groups
  for (int q = 0; q <= b.M;) {
    Stage s;
    s.m0 = q;
    while (q <= b.M && s.units + p.lev[q] <= cap) s.units += p.lev[q++];
    s.m1 = q;
    s.count.assign(p.nd + 2, 0);
    s.ubase.assign(p.nd + 2, 0);
    s.dcount.assign(p.nd + 1, 0);
    s.doff.assign(p.nd + 1, 0);
    int u = 0;
    for (int l = 2; l <= p.nd + 1; ++l) {
      s.ubase[l] = u;
      for (int k = s.m0; k < s.m1; ++k) s.count[l] += p.lev[k] >= l - 1;
      u += s.count[l];
    }
    for (int j = 1; j <= p.nd; ++j) {
      s.dcount[j] = s.count[j + 1];
      s.doff[j] = s.bytes;
      s.bytes += s.dcount[j] * kRowsChunk * b.K * 2;
    }
    s.toff.assign(p.nd + 1, 0);
    for (int k = s.m0; k < s.m1; ++k) s.tails += tail(k);
    for (int j = 2; j <= p.nd && s.tails; ++j) {
      s.toff[j] = s.bytes;
      s.bytes += s.tails * kRowsChunk * b.K * 2;
    }
    s.offset = p.chunk_bytes;
    p.chunk_bytes += s.bytes;
    p.slot_bytes = std::max(p.slot_bytes, s.bytes);
    p.st.push_back(s);
  }
  p.chunks = (b.rows + kRowsChunk - 1) / kRowsChunk;
  if (opt.part == 3) p.red = 8 + kRowsChunk * p.chunks;
  const int fixed = (b.M + 1) * kStates * 8 + p.red * kStates * 8 + (b.M + 1) * 32 * 8 + p.chunks * kRowsChunk * 8 + b.K * 4 + 1024 +
                    (b.K <= 64 ? b.K * kStates * 8 : 0);   // (the next tile's Y, for mechanisms small enough)
  p.slots = std::min(8, (200 * 1024 - fixed) / p.slot_bytes);
  p.slots = std::min(p.slots, std::max(2, (int)p.st.size() * p.chunks));
  if (p.slots < 2) return false;
  p.smem = p.slots * p.slot_bytes + fixed;
  return true;
}

// Coefficient digits of every chunk and stage, in the order and layout that the matrix
// instructions read: per digit a block of (basis function, 16 rows) x K float16 values, in core
// matrices of 8 rows x 16 bytes, K-contiguous (no swizzle).
void emit_digits(std::ostringstream& s, const Plan& p) {
  const TcBasis& b = p.b;
  const size_t bytes = (size_t)p.chunk_bytes * p.chunks;
  std::vector<unsigned short> h(bytes / 2, 0);
  for (int c = 0; c < p.chunks; ++c)
    for (const Stage& st : p.st)
      for (int q = st.m0; q < st.m1; ++q) {
        const int nl = p.lev[q];
        for (int r = 0; r < kRowsChunk; ++r) {
          const int row = c * kRowsChunk + r;
          if (row >= b.rows) continue;
          for (int j = 0; j < b.ns; ++j) {
            const double v = b.coef[((size_t)row * b.ns + j) * (b.M + 1) + q];
            long long Q = (long long)std::nearbyint(std::ldexp(v, kDigit * nl - 1));
            for (int d = nl; d >= 1; --d) {
              long long dig = Q;
              if (d > 1) {
                dig = (((Q + 512) % 1024) + 1024) % 1024 - 512;
                Q = (Q - dig) / 1024;
              }
              // integer to float16 (|dig| <= 512)
              unsigned short bits = 0;
              if (dig != 0) {
                unsigned a = (unsigned)(dig < 0 ? -dig : dig);
                int e = 31 - __builtin_clz(a);
                bits = (unsigned short)((dig < 0 ? 0x8000u : 0u) | ((unsigned)(e + 15) << 10) | ((a << (10 - e)) & 0x3ffu));
              }
              const int n = (q - st.m0) * kRowsChunk + r;
              const size_t at = (size_t)c * p.chunk_bytes + st.offset + st.doff[d] + (size_t)(n / 8) * (b.K * 16) +
                                (size_t)(j / 8) * 128 + (n % 8) * 16 + (j % 8) * 2;
              h[at / 2] = bits;
              if (d >= 2 && q - st.m0 < st.tails) {   // exact: |dig| 2^-10 >= 2^-10
                const unsigned short scaled = bits ? (unsigned short)(bits - (10u << 10)) : 0;
                h[at / 2 - st.doff[d] / 2 + st.toff[d] / 2] = scaled;
              }
            }
          }
        }
      }
  s << "__device__ const unsigned long long kx_dig[" << bytes / 8 << "] __attribute__((aligned(128))) = {";
  for (size_t i = 0; i < bytes / 8; ++i) {
    unsigned long long w = 0;
    for (int k = 3; k >= 0; --k) w = w << 16 | h[4 * i + k];
    if (w) s << hex64(w) << ","; else s << "0,";
  }
  s << "};\n";
}

std::string list(const std::vector<double>& v, bool pair) {
  std::string o;
  for (double x : v) o += pair ? "{" + fpair(x) + "}," : D(x) + ",";
  return o;
}

// Tables and per-state functions of the pairwise evaluation.
void emit_pairwise(std::ostringstream& s, const Mechanism& m, const Plan& p) {
  const int ns = m.ns;
  std::vector<double> iw(ns), w(ns);
  for (int k = 0; k < ns; ++k) { iw[k] = 1.0 / m.W[k]; w[k] = m.W[k]; }
  s << "__device__ const double kx_iw[" << ns << "] = {" << list(iw, false) << "};\n";
  s << "__device__ const double kx_w[" << ns << "] = {" << list(w, false) << "};\n";
  // degree-4 polynomial in L whose coefficient n of a warp's lanes is the expression tab(n)
  auto horner = [](const std::function<std::string(int)>& tab) {
    std::string e = tab(4);
    for (int n = 3; n >= 0; --n) e = fmt("kx_df_fma_u(%s, L, %s)", e.c_str(), tab(n).c_str());
    return e;
  };
  const int SL = (ns + 31) / 32;   // species of a lane: lane, lane + 32, ...
  const std::string last = std::to_string(ns - 1);
  s << "__device__ __forceinline__ kx_df kx_f2(float2 v) { return kx_mk(v.x, v.y); }\n";
  if (p.part != 3)
    s << "__device__ __forceinline__ double kx_lane_sum(double v) {\n"
      << "  for (int d = 16; d > 0; d >>= 1) v += __shfl_xor_sync(0xffffffffu, v, d);\n  return v;\n}\n"
      << "__device__ __forceinline__ kx_df kx_lane_sum(kx_df v) {\n"
      << "  for (int d = 16; d > 0; d >>= 1) v = kx_df_add(v, kx_mk(__shfl_xor_sync(0xffffffffu, v.hi, d), __shfl_xor_sync(0xffffffffu, v.lo, d)));\n"
      << "  return v;\n}\n";
  // chains that a warp of the state functions below has in flight (SL rows of a lane, as many species at a time)
  const int unroll = std::max(1, 4 / SL);
  if (p.part == 2) {
    // -ln D_jk about L_mid, coefficient n of (j, k) at (n ns + j) ns + k: a warp's lanes (k, or j: it is symmetric)
    // read 32 neighbours
    std::vector<unsigned long long> dc(5 * (size_t)ns * ns);
    for (int k = 0; k < ns; ++k)
      for (int j = k; j < ns; ++j) {
        double d[5];
        shift_poly(&m.dif[5 * ((size_t)k * ns + j)], kTcLmid, -1.0, d);
        for (int n = 0; n < 5; ++n) {
          const float h = (float)d[n], l = (float)(d[n] - (double)h);
          unsigned hb, lb;
          std::memcpy(&hb, &h, 4);
          std::memcpy(&lb, &l, 4);
          dc[((size_t)n * ns + j) * ns + k] = dc[((size_t)n * ns + k) * ns + j] = (unsigned long long)lb << 32 | hb;
        }
      }
    s << "__device__ const unsigned long long kx_dcb[" << dc.size() << "] = {";
    for (unsigned long long v : dc) s << hex64(v) << ",";
    s << "};\n";
    s << "__device__ __forceinline__ kx_df kx_dc(int n, int j, int k) {\n"
      << fmt("  const unsigned long long b = kx_dcb[(n * %d + j) * %d + k];\n", ns, ns)
      << "  return kx_mk(__uint_as_float((unsigned)b), __uint_as_float((unsigned)(b >> 32)));\n}\n";
    auto coef = [](const char* j, const char* k) {
      return [=](int n) { return fmt("kx_dc(%d, %s, %s)", n, j, k); };
    };
    // D_k of state i by one warp, its lanes over the partner species: the partners' share of the mass
    // summed directly, so that a nearly pure state keeps its relative accuracy; D_kk where no partner is
    // present.  Every lane returns the value (sums in a fixed order).
    s << "__device__ __noinline__ double kx_diff_row(const double* __restrict__ Y_, long long ld, long long i, int k, float Lh, float Ll, double P) {\n"
      << "  const int lane = threadIdx.x & 31;\n  const kx_df L = kx_mk(Lh, Ll);\n"
      << "  double sy = 0.0, sY = 0.0, so = 0.0;\n"
      << "  for (int j = lane; j < " << ns << "; j += 32) { const double y = Y_[(long long)j * ld + i]; sY += y; if (j != k) so += y; sy = fma(y, kx_iw[j], sy); }\n"
      << "  sy = kx_lane_sum(sy); sY = kx_lane_sum(sY); so = kx_lane_sum(so);\n"
      << "  const double isig = 1.0 / sy;\n"
      << "  kx_df S = kx_mk(0.f, 0.f);\n"
      << "  for (int j = lane; j < " << ns << "; j += 32) {\n"
      << "    if (j == k) continue;\n"
      << "    S = kx_df_fma_u(kx_d2df_i(Y_[(long long)j * ld + i] * kx_iw[j] * isig), kx_df_exp(" << horner(coef("k", "j")) << "), S);\n"
      << "  }\n"
      << "  const double Sd = kx_lane_sum(kx_df2d(kx_df_norm(S))), pr = " << D(P_ATM) << " / P;\n"
      << "  if (Sd > 0.0) return so / sY * pr / Sd;\n"
      << "  const kx_df e = " << horner(coef("k", "k")) << ";\n"
      << "  return kx_df2d(kx_df_exp(kx_mk(-e.hi, -e.lo))) * pr;\n}\n";
    // All D_k of state i by one warp, its lanes over the rows, every species' mole fraction broadcast to them in turn.
    // 2^18 states of 53/325 at 4500 K: 6.5 ms (mixed 2.7), a row at a time as above 58; with 1 % of them there 0.84
    // against 1.82, with none 0.30.  Bound by the coefficients' way from L2 (40 bytes a pair) and the latency of
    // four warps a scheduler; the one-thread-per-state kernel, which a call cannot know to choose, takes 1.8.
    if (p.mixed)   // 1/D_jk to about 2^-22: the polynomial's last sum and the exponential's argument in two parts
      s << "__device__ __forceinline__ float kx_idiff(int j, int k, float L) {\n"
        << "  const float h = fmaf(fmaf(fmaf(kx_dc(4, j, k).hi, L, kx_dc(3, j, k).hi), L, kx_dc(2, j, k).hi), L, kx_dc(1, j, k).hi);\n"
        << "  const kx_df c = kx_dc(0, j, k);\n"
        << "  const float p = __fmul_rn(h, L);\n"
        << "  const kx_df e = kx_ts(c.hi, p);\n"
        << "  const float lo = e.lo + (fmaf(h, L, -p) + c.lo), y = __fmul_rn(e.hi, 1.44269504f);\n"
        << "  const float yl = fmaf(e.hi, 1.44269504f, -y) + fmaf(e.hi, 1.92596303e-8f, lo * 1.44269504f);\n"
        << "  float r;\n  asm(\"ex2.approx.ftz.f32 %0, %1;\" : \"=f\"(r) : \"f\"(y));\n"
        << "  return fmaf(r, yl * 0.693147181f, r);\n}\n";
    s << "__device__ __noinline__ void kx_diff_state(const double* __restrict__ Y_, long long ld, long long i, float Lh, float Ll, double P, double* __restrict__ out) {\n"
      << "  const int lane = threadIdx.x & 31;\n  const kx_df L = kx_mk(Lh, Ll);\n"
      << fmt("  double y[%d], so[%d], sy = 0.0, sY = 0.0;\n", SL, SL)
      << fmt("  #pragma unroll\n  for (int s = 0; s < %d; ++s) {\n", SL)
      << fmt("    const int k = lane + 32 * s;\n    y[s] = k < %d ? Y_[(long long)k * ld + i] : 0.0;\n", ns)
      << "    sY += y[s]; sy = fma(y[s], kx_iw[min(k, " << last << ")], sy);\n  }\n"
      << "  sy = kx_lane_sum(sy); sY = kx_lane_sum(sY);\n"
      << "  const double isig = 1.0 / sy;\n"
      << "  if (!(isig > 0.0 && isig < KX_INF)) {   // outside the domain\n"
      << fmt("    for (int k = lane; k < %d; k += 32) out[(long long)k * ld + i] = KX_NAN;\n", ns)
      << "    if (lane == 0) atomicMin(&kx_bad_first, (unsigned long long)i);\n    return;\n  }\n"
      << (p.mixed ? fmt("  float x[%d], S[%d];\n", SL, SL) : fmt("  kx_df x[%d], S[%d];\n", SL, SL))
      << fmt("  #pragma unroll\n  for (int s = 0; s < %d; ++s) {\n", SL)
      << "    const kx_df X = kx_d2df_i(y[s] * kx_iw[min(lane + 32 * s, " << last << ")] * isig);\n"
      << (p.mixed ? "    x[s] = X.hi; S[s] = 0.0f;\n" : "    x[s] = X; S[s] = kx_mk(0.0f, 0.0f);\n")
      // the partners' share of the mass: the rest of the sum, for a species of more than half of it summed directly
      << "    so[s] = sY - y[s];\n"
      << "    for (unsigned m = __ballot_sync(0xffffffffu, y[s] > 0.5 * sY); m; m &= m - 1) {\n"
      << "      const bool own = lane == __ffs(m) - 1;\n      double d = 0.0;\n"
      << fmt("      #pragma unroll\n      for (int q = 0; q < %d; ++q) if (!own || q != s) d += y[q];\n", SL)
      << "      d = kx_lane_sum(d);\n      if (own) so[s] = d;\n    }\n  }\n"
      << fmt("  #pragma unroll\n  for (int q = 0; q < %d; ++q)\n    #pragma unroll %d\n", SL, unroll)
      << fmt("    for (int jl = 0; jl < min(32, %d - 32 * q); ++jl) {\n      const int j = 32 * q + jl;\n", ns)
      << (p.mixed ? "      const float xj = __shfl_sync(0xffffffffu, x[q], jl);\n"
                  : "      const kx_df xj = kx_mk(__shfl_sync(0xffffffffu, x[q].hi, jl), __shfl_sync(0xffffffffu, x[q].lo, jl));\n")
      << fmt("      #pragma unroll\n      for (int s = 0; s < %d; ++s) {\n", SL)
      << "        const int k = min(lane + 32 * s, " << last << ");\n"
      << (p.mixed ? "        S[s] = fmaf(k == j ? 0.0f : xj, kx_idiff(j, k, Lh), S[s]);\n"
                  : "        S[s] = kx_df_fma_u(k == j ? kx_mk(0.0f, 0.0f) : xj, kx_df_exp(" + horner(coef("j", "k")) + "), S[s]);\n")
      << "      }\n    }\n"
      << "  const double pr = " << D(P_ATM) << " / P;\n"
      << fmt("  #pragma unroll\n  for (int s = 0; s < %d; ++s) {\n", SL)
      << fmt("    const int k = lane + 32 * s;\n    if (k >= %d) break;\n", ns)
      << (p.mixed ? "    const double Sd = kx_f2d(S[s]);\n" : "    const double Sd = kx_df2d(kx_df_norm(S[s]));\n")
      << "    double d = so[s] * pr / (sY * Sd);\n"
      << "    if (!(Sd > 0.0)) {\n      const kx_df e = " << horner(coef("k", "k")) << ";\n"
      << "      d = kx_df2d(kx_df_exp(kx_mk(-e.hi, -e.lo))) * pr;\n    }\n"
      << "    out[(long long)k * ld + i] = d;\n  }\n}\n";
    return;
  }
  if (p.part == 3) {
    std::vector<double> a;
    for (int k = 0; k < ns; ++k)
      for (int rg = 0; rg < 2; ++rg)
        for (int n = 0; n < 6; ++n) a.push_back(rg == 0 ? m.a_lo[7 * k + n] : m.a_hi[7 * k + n]);
    s << "__device__ const double kx_nasa[" << a.size() << "] = {" << list(a, false) << "};\n";
    s << "__device__ const double kx_tmid[" << ns << "] = {" << list(m.Tmid, false) << "};\n";
    s << "__device__ __noinline__ double2 kx_thermo_state(const double* __restrict__ Y_, long long ld, long long i, double T) {\n"
      << "  double cp = 0.0, h = 0.0;\n"
      << "  for (int k = 0; k < " << ns << "; ++k) {\n"
      << "    const double* a = kx_nasa + 12 * k + (T < kx_tmid[k] ? 0 : 6);\n"
      << "    const double y = Y_[(long long)k * ld + i] * (" << D(R_U) << " / kx_w[k]);\n"
      << "    cp = fma(y, fma(fma(fma(fma(a[4], T, a[3]), T, a[2]), T, a[1]), T, a[0]), cp);\n"
      << "    h = fma(y, fma(fma(fma(fma(fma(a[4] * 0.2, T, a[3] * 0.25), T, a[2] / 3.0), T, a[1] * 0.5), T, a[0]), T, a[5]), h);\n"
      << "  }\n  return make_double2(cp, h);\n}\n";
    return;
  }
  // u_k = sqrt(eta_k) W_k^(-1/4), v = 1/u: sum_j X_j phi_kj = sum_j a_kj X_j (1 + u_k v_j)^2, a_kj at j ns + k
  std::vector<double> pv, pl, wa, sq;
  for (int k = 0; k < ns; ++k) {
    double d[5];
    shift_poly(&m.eta[5 * k], kTcLmid, -0.5, d);
    d[0] += 0.25 * std::log(m.W[k]);
    for (int n = 0; n < 5; ++n) pv.push_back(d[n]);
    shift_poly(&m.lam[5 * k], kTcLmid, 1.0, d);
    for (int n = 0; n < 5; ++n) pl.push_back(d[n]);
    for (int j = 0; j < ns; ++j) wa.push_back(1.0 / std::sqrt(8.0 * (1.0 + m.W[j] / m.W[k])));
    sq.push_back(std::sqrt(m.W[k]));
  }
  s << "__device__ const float2 kx_pv[" << pv.size() << "] = {" << list(pv, true) << "};\n";
  s << "__device__ const float2 kx_pl[" << pl.size() << "] = {" << list(pl, true) << "};\n";
  s << "__device__ const float2 kx_wa[" << wa.size() << "] = {" << list(wa, true) << "};\n";
  s << "__device__ const float2 kx_sqw[" << ns << "] = {" << list(sq, true) << "};\n";
  auto of = [](const char* t) { return [=](int n) { return fmt("kx_f2(%s[%d])", t, n); }; };
  // mu and lambda of state i by one warp, its lanes over Wilke's rows, every species' mole fraction and v broadcast
  // to them in turn.  2^18 states of 53/325 at 4500 K: 2.4 ms (mixed 1.6), with a thread for each state 4.4; with 1 %
  // of them there 0.59 against 4.1, with none 0.36; the one-thread-per-state kernel takes 1.3.
  s << "__device__ __noinline__ double2 kx_visc_state(const double* __restrict__ Y_, long long ld, long long i, float Lh, float Ll) {\n"
    << "  const int lane = threadIdx.x & 31;\n  const kx_df L = kx_mk(Lh, Ll);\n"
    << (p.mixed ? fmt("  float x[%d], u[%d], v[%d], S[%d];\n", SL, SL, SL, SL) : fmt("  kx_df x[%d], u[%d], v[%d], S[%d];\n", SL, SL, SL, SL))
    << fmt("  double y[%d], sy = 0.0;\n  kx_df w[%d], sl = kx_mk(0.f, 0.f), sil = kx_mk(0.f, 0.f);\n", SL, SL)
    << fmt("  #pragma unroll\n  for (int s = 0; s < %d; ++s) {\n", SL)
    << "    const int k = min(lane + 32 * s, " << last << ");\n"
    << fmt("    y[s] = lane + 32 * s < %d ? Y_[(long long)k * ld + i] * kx_iw[k] : 0.0;\n    sy += y[s];\n  }\n", ns)
    << "  const double isig = 1.0 / kx_lane_sum(sy);\n"
    << "  if (!(isig > 0.0 && isig < KX_INF)) {   // outside the domain\n"
    << "    if (lane == 0) atomicMin(&kx_bad_first, (unsigned long long)i);\n    return make_double2(KX_NAN, KX_NAN);\n  }\n"
    << fmt("  #pragma unroll\n  for (int s = 0; s < %d; ++s) {\n", SL)
    << "    const int k = min(lane + 32 * s, " << last << ");\n"
    << "    const kx_df X = kx_d2df_i(y[s] * isig);\n"
    << "    const float2* pv = kx_pv + 5 * k; const float2* pl = kx_pl + 5 * k;\n"
    << "    const kx_df e = " << horner(of("pv")) << ", l = " << horner(of("pl")) << ";\n"
    << "    const kx_df ve = kx_df_exp(e), ue = kx_df_exp(kx_mk(-e.hi, -e.lo));\n"
    << (p.mixed ? "    x[s] = X.hi; v[s] = ve.hi; u[s] = ue.hi; S[s] = 0.0f;\n" : "    x[s] = X; v[s] = ve; u[s] = ue; S[s] = kx_mk(0.f, 0.f);\n")
    << "    w[s] = kx_df_mul(X, kx_df_mul(kx_df_mul(ue, ue), kx_f2(kx_sqw[k])));\n"
    << "    sl = kx_df_fma(X, kx_df_exp(l), sl); sil = kx_df_fma(X, kx_df_exp(kx_mk(-l.hi, -l.lo)), sil);\n"
    << "  }\n"
    << fmt("  #pragma unroll\n  for (int q = 0; q < %d; ++q)\n    #pragma unroll %d\n", SL, unroll)
    << fmt("    for (int jl = 0; jl < min(32, %d - 32 * q); ++jl) {\n", ns);
  if (p.mixed)
    s << "      const float xj = __shfl_sync(0xffffffffu, x[q], jl), vj = __shfl_sync(0xffffffffu, v[q], jl);\n";
  else
    s << "      const kx_df xj = kx_mk(__shfl_sync(0xffffffffu, x[q].hi, jl), __shfl_sync(0xffffffffu, x[q].lo, jl));\n"
      << "      const kx_df vj = kx_mk(__shfl_sync(0xffffffffu, v[q].hi, jl), __shfl_sync(0xffffffffu, v[q].lo, jl));\n";
  s << fmt("      #pragma unroll\n      for (int s = 0; s < %d; ++s) {\n", SL)
    << fmt("        const float2 a = kx_wa[(32 * q + jl) * %d + min(lane + 32 * s, %s)];\n", ns, last.c_str());
  if (p.mixed)
    s << "        const float z = fmaf(u[s], vj, 1.0f);\n        S[s] = fmaf(a.x * xj, z * z, S[s]);\n";
  else
    s << "        const kx_df z = kx_df_fma_u(u[s], vj, kx_mk(1.f, 0.f));\n"
      << "        S[s] = kx_df_fma_u(kx_df_mul_u(kx_f2(a), xj), kx_df_mul_u(z, z), S[s]);\n";
  s << "      }\n    }\n  kx_df mu = kx_mk(0.f, 0.f);\n"
    << fmt("  #pragma unroll\n  for (int s = 0; s < %d; ++s) mu = kx_df_add(mu, kx_df_div(w[s], ", SL)
    << (p.mixed ? "kx_mk(S[s], 0.0f)));\n" : "kx_df_norm(S[s])));\n")
    << "  mu = kx_lane_sum(mu); sl = kx_lane_sum(sl); sil = kx_lane_sum(sil);\n"
    << "  return make_double2(kx_df2d(mu), 0.5 * kx_df2d(kx_df_add(sl, kx_df_div(kx_mk(1.0f, 0.0f), sil))));\n}\n";
}

// Matrix instructions of one stage, issued by one thread: level l = i + j of digit i of v and
// digit j of c into the accumulators of that level.
std::string mma_code(const Plan& p, const Stage& st) {
  const int K = p.b.K;
  std::string o;
  for (int l = 2; l <= p.nd + 1; ++l) {
    if (!st.count[l]) continue;
    const int N = 16 * st.count[l];
    const unsigned idesc = (1u << 4) | ((unsigned)(N / 8) << 17) | ((unsigned)(kStates / 16) << 24);
    for (int i = 1; i <= l - 1; ++i) {
      const int j = l - i;
      for (int ks = 0; ks < K / 16; ++ks)
        o += fmt("          kx_mma(dt + %d, ta + %d, bd + %d, 0x%xu, %d);\n", st.ubase[l] * 16, (i - 1) * (K / 2) + 8 * ks,
                 (st.doff[j] + 256 * ks) >> 4, idesc, !(i == 1 && ks == 0));
    }
  }
  if (st.tails) {
    const int N = 16 * st.tails;
    const unsigned idesc = (1u << 4) | ((unsigned)(N / 8) << 17) | ((unsigned)(kStates / 16) << 24);
    for (int i = 2; i <= p.nd; ++i)
      for (int ks = 0; ks < K / 16; ++ks)
        o += fmt("          kx_mma(dt + %d, ta + %d, bd + %d, 0x%xu, 1);\n", st.ubase[p.nd + 1] * 16, (i - 1) * (K / 2) + 8 * ks,
                 (st.toff[p.nd + 2 - i] + 256 * ks) >> 4, idesc);
  }
  return o;
}

// Reads one stage's accumulators and adds phi_m times their sums into the rows' running sums.
std::string sum_code(const Plan& p, const Stage& st) {
  std::string o;
  const int RT = kRowsChunk / kGroups;
  for (int q = st.m0; q < st.m1; ++q) {
    const int nl = p.lev[q];
    o += fmt("      { unsigned r[%d][%d];\n", nl, RT);
    for (int l = 2; l <= nl + 1; ++l) o += fmt("      kx_ld(r[%d], td + %d);\n", l - 2, (st.ubase[l] + q - st.m0) * 16);
    o += "      kx_wait_ld();\n";
    if (q == st.m1 - 1) o += "      kx_fence_before();\n      __syncwarp();\n      if (lane == 0) kx_mb_arrive(dfree + 8 * buf);\n";
    auto L = [&](int l) { return fmt("__uint_as_float(r[%d][a])", l - 2); };
    const bool fl = p.mixed || p.b.E[q] <= kFloatE, mid = !fl && q > 0 && p.b.E[q] <= kMidE;
    if (q > 0) {
      if (fl) o += fmt("      { const float f = sphi[%d * 128 + s].x;\n", q);
      else o += fmt("      { const kx_df f = kx_mk(sphi[%d * 128 + s].x, sphi[%d * 128 + s].y);%s\n", q, q,
                    mid ? " const float fs = __fmul_rn(f.hi, 0x1p-10f);" : "");
    } else {
      o += "      {\n";
    }
    o += fmt("      #pragma unroll\n      for (int a = 0; a < %d; ++a) {\n", RT);
    if (fl) {
      std::string c = L(nl + 1);
      for (int l = nl; l >= 2; --l) c = fmt("__fmaf_rn(%s, 0x1p-10f, %s)", c.c_str(), L(l).c_str());
      if (p.mixed) o += q == 0 ? fmt("        hi[a] = %s;\n", c.c_str()) : fmt("        hi[a] = __fmaf_rn(f, %s, hi[a]);\n", c.c_str());
      else o += fmt("        sm[a] = __fmaf_rn(f, %s, sm[a]);\n", c.c_str());
    } else if (mid) {
      // the first level as an exact product, the rest (2^-8 of it) in float32: 2^-32 of the set's sum
      std::string t = L(nl + 1);
      for (int l = nl; l >= 3; --l) t = fmt("__fmaf_rn(%s, 0x1p-10f, %s)", t.c_str(), L(l).c_str());
      o += fmt("        const float pp = __fmul_rn(f.hi, %s);\n", L(2).c_str());
      o += fmt("        const float pe = __fmaf_rn(f.lo, %s, __fmaf_rn(f.hi, %s, -pp));\n", L(2).c_str(), L(2).c_str());
      o += "        const kx_df w = kx_qts(hi[a], pp);\n";
      o += fmt("        hi[a] = w.hi; lo[a] = __fadd_rn(lo[a], __fadd_rn(w.lo, %s));\n",
               nl >= 2 ? fmt("__fmaf_rn(fs, %s, pe)", t.c_str()).c_str() : "pe");
    } else {
      // the first three levels exactly (two-sums), the rest in float32: 2^-30 of the first
      o += fmt("        const kx_df c2 = kx_ts(%s, %s);\n", L(2).c_str(), nl >= 2 ? fmt("__fmul_rn(%s, 0x1p-10f)", L(3).c_str()).c_str() : "0.0f");
      if (nl >= 3) o += fmt("        const kx_df c3 = kx_qts(c2.hi, __fmul_rn(%s, 0x1p-20f));\n", L(4).c_str());
      std::string lo = nl >= 3 ? "__fadd_rn(c2.lo, c3.lo)" : "c2.lo";
      if (nl >= 4) {
        std::string t = L(nl + 1);
        if (nl == 5) t = fmt("__fmaf_rn(%s, 0x1p-10f, %s)", t.c_str(), L(5).c_str());
        lo = fmt("__fmaf_rn(%s, 0x1p-30f, %s)", t.c_str(), lo.c_str());
      }
      const char* h = nl >= 3 ? "c3.hi" : "c2.hi";
      o += fmt("        const float cl = %s;\n", lo.c_str());
      if (q == 0) {
        o += fmt("        hi[a] = %s; lo[a] = cl; sm[a] = 0.0f;\n", h);
      } else {
        o += fmt("        const float pp = __fmul_rn(f.hi, %s);\n", h);
        o += fmt("        const float pe = __fmaf_rn(f.lo, %s, __fmaf_rn(f.hi, cl, __fmaf_rn(f.hi, %s, -pp)));\n", h, h);
        o += fmt("        const kx_df w = %s(hi[a], pp);\n", q <= 2 ? "kx_ts" : "kx_qts");
        o += "        hi[a] = w.hi; lo[a] = __fadd_rn(lo[a], __fadd_rn(w.lo, pe));\n";
      }
    }
    o += "      } } }\n";
  }
  return o;
}

}  // namespace

std::string emit_transport_tc(const Mechanism& m, const EmitOptions& opt, const std::string& entry, OpCounts* counts,
                              KernelShape* shape) {
  Plan p;
  if (!make_plan(m, opt, p)) return "";
  const TcBasis& b = p.b;
  const int ns = m.ns, K = b.K, G = kGroups, RT = kRowsChunk / G, QW = K / (4 * G);   // QW: groups of four species per compute group
  const int kThreads = 128 * G + 64;
  const bool visc = p.part == 1, diff = p.part == 2, thermo = p.part == 3, mixed = p.mixed;
  const int NST = (int)p.st.size();
  std::ostringstream s;
  s << "// mechanism " << m.name << ": " << m.ns << " species, " << m.nr() << " reactions\n";
  s << "#define P_ATM_R " << D(P_ATM / R_U) << "\n";
  s << "#define KX_T64 0\n#define KX_TDF 1\n#define KX_TDFR 1\n";
  s << kTables << "\n" << kDevicePrelude << "\n" << kTcPrelude << kTcExp << "\n";
  s << "#define KX_COMPUTE_SYNC asm volatile(\"bar.sync 1, " << 128 * G << ";\" ::: \"memory\")\n";
  s << "extern __shared__ __align__(128) unsigned char kx_dyn[];\n";
  s << "__device__ unsigned long long kx_bad_first = 0xffffffffffffffffull;\n";
  emit_digits(s, p);
  emit_pairwise(s, m, p);
  // per row: power of two of its sums (and, viscosity, 2^(18 - rho)/W_k)
  std::string ec;
  for (int j = 0; j < K; ++j) ec += fmt("%d,", j < ns ? b.ecol[j] : 0);
  s << "__device__ const int kx_ecol[" << K << "] = {" << ec << "};\n";
  const int rpad = p.chunks * kRowsChunk;
  std::vector<double> rs(rpad, 0.0);
  for (int r = b.first; r < b.rows; ++r)
    rs[r] = thermo ? std::ldexp(1.0, b.rho[r]) : visc ? std::ldexp(1.0 / m.W[r - b.first], 18 - b.rho[r]) : std::ldexp(1.0, b.rho[0] - b.rho[r]);
  s << "__device__ const float2 kx_rs[" << rpad << "] = {" << list(rs, true) << "};\n";
  // basis functions
  s << "__device__ const float2 kx_phi[" << 32 * (b.M + 1) << "] = {";
  for (int q = 0; q <= b.M; ++q)
    for (int n = 0; n < 32; ++n) {
      const std::vector<double>& c = mixed || b.E[q] <= kPhiE ? b.cheb[q] : b.phi[q];
      s << "{" << fpair(n < (int)c.size() ? c[n] : 0.0) << "},";
    }
  s << "};\n";
  s << "__device__ const float2 kx_g[10] = {" << list(std::vector<double>(b.g0, b.g0 + 5), true)
    << list(std::vector<double>(b.g1, b.g1 + 5), true) << "};\n";
  s << "extern \"C\" __global__ void __launch_bounds__(" << kThreads << ", 1) " << entry
    << "(const double* __restrict__ T_, const double* __restrict__ P_, const double* __restrict__ Y_, long long ld, "
    << "double* __restrict__ out0_, double* __restrict__ out1_, " << (thermo ? "" : "double* __restrict__ out2_, ") << "long long n)\n{\n";
  s << "  __shared__ __align__(8) unsigned long long bars[" << 2 * p.slots + 5 << "];\n";
  s << "  __shared__ unsigned tmem_addr;\n";
  // a compute warp whose wait ran out says so to the groups that read its shared values
  s << "  __shared__ volatile int failed;\n";
  s << "  kx_load_tables();\n";
  s << "  const int warp = __shfl_sync(0xffffffffu, threadIdx.x >> 5, 0), lane = threadIdx.x & 31;\n";
  s << "  unsigned char* const slots = kx_dyn;\n";
  s << fmt("  float2* const sphi = (float2*)(kx_dyn + %d);\n", p.slots * p.slot_bytes);
  s << fmt("  float2* const sred = sphi + %d;   // [][128]: values exchanged between the compute groups\n", (b.M + 1) * kStates);
  s << fmt("  float2* const sph = sred + %d;    // basis polynomials\n", p.red * kStates);
  s << fmt("  float2* const srs = sph + %d;    // row scales\n", 32 * (b.M + 1));
  s << fmt("  int* const sec = (int*)(srs + %d);   // column exponents\n", rpad);
  const bool stage_y = K <= 64;
  if (stage_y) s << fmt("  double* const sy = (double*)(sec + %d);   // [species][128]: Y of the tile, copied ahead by the thread that reads it\n", K);
  s << fmt("  for (int j = threadIdx.x; j < %d; j += %d) sph[j] = kx_phi[j];\n", 32 * (b.M + 1), kThreads);
  s << fmt("  for (int j = threadIdx.x; j < %d; j += %d) srs[j] = kx_rs[j];\n", rpad, kThreads);
  s << fmt("  for (int j = threadIdx.x; j < %d; j += %d) sec[j] = kx_ecol[j];\n", K, kThreads);
  s << "  const unsigned full = kx_smem(bars), empty = full + " << 8 * p.slots << ", dfull = full + " << 16 * p.slots
    << ", dfree = dfull + 16, aready = dfull + 32;\n";
  s << "  if (threadIdx.x == 0) {\n"
    << "    for (int j = 0; j < " << p.slots << "; ++j) { kx_mb_init(full + 8 * j, 1); kx_mb_init(empty + 8 * j, 1); }\n"
    << "    for (int j = 0; j < 2; ++j) { kx_mb_init(dfull + 8 * j, 1); kx_mb_init(dfree + 8 * j, " << 4 * G << "); }\n"
    << "    kx_mb_init(aready, " << 4 * G << ");\n    failed = 0;\n"
    << "    asm volatile(\"fence.mbarrier_init.release.cluster;\" ::: \"memory\");\n"
    << "  }\n";
  s << fmt("  if (warp == %d) {\n", 4 * G)
    << "    asm volatile(\"tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], " << 512 << ";\" ::\"r\"(kx_smem(&tmem_addr)) : \"memory\");\n"
    << "    asm volatile(\"tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;\");\n"
    << "  }\n";
  s << "  kx_fence_before();\n  __syncthreads();\n  kx_fence_after();\n";
  s << "  const unsigned tmem = __shfl_sync(0xffffffffu, tmem_addr, 0);\n";
  s << "  const long long tiles = (n + 127) / 128;\n";
  // chunks of this block: the first (it holds the sums that every row needs) and every gridDim.y-th
  s << "  const int cy = blockIdx.y, gy = gridDim.y, cnext = cy == 0 ? gy : cy;\n";
  s << "  bool ok = true;\n";
  // ---- loader
  s << fmt("  if (warp == %d) {\n", 4 * G + 1) << "    if (lane == 0) {\n      unsigned g = 0;\n"
    << "      for (long long t = blockIdx.x; t < tiles; t += gridDim.x)\n"
    << "        for (int c = 0; c < " << p.chunks << "; c = c == 0 ? cnext : c + gy)\n"
    << "          for (int st = 0; st < " << NST << "; ++st, ++g) {\n"
    << "            const unsigned slot = g % " << p.slots << "u, use = g / " << p.slots << "u;\n"
    << "            if (use > 0) ok = ok && kx_mb_wait(empty + 8 * slot, (use - 1) & 1);\n"
    << "            if (!ok) break;\n";
  {
    std::string off, by;
    for (const Stage& st : p.st) { off += fmt("%d,", st.offset); by += fmt("%d,", st.bytes); }
    s << "            const int offs[" << NST << "] = {" << off << "}, bytes[" << NST << "] = {" << by << "};\n";
  }
  s << "            kx_mb_expect(full + 8 * slot, bytes[st]);\n"
    << "            kx_bulk_load(kx_smem(slots) + slot * " << p.slot_bytes << "u, (const unsigned char*)kx_dig + (size_t)c * " << p.chunk_bytes
    << " + offs[st], bytes[st], full + 8 * slot);\n"
    << "          }\n"
    // every copy has landed before the block ends (the issuing warp waits for each; after a failed wait it does not)
    << "      for (unsigned j = 0; j < " << p.slots << "u && j < g; ++j) {\n"
    << "        const unsigned last = g - 1 - j;\n"
    << "        kx_mb_wait(full + 8 * (last % " << p.slots << "u), (last / " << p.slots << "u) & 1);\n"
    << "      }\n    }\n  }\n";
  // ---- matrix instructions
  s << fmt("  else if (warp == %d) {\n", 4 * G) << "      unsigned g = 0, tt = 0;\n"
    << "      const unsigned ta = tmem;\n"
    << "      for (long long t = blockIdx.x; t < tiles; t += gridDim.x, ++tt) {\n"
    << "        ok = __all_sync(0xffffffffu, ok && kx_mb_wait(aready, tt & 1));\n"
    << "        kx_fence_after();\n"
    << "        for (int c = 0; c < " << p.chunks << "; c = c == 0 ? cnext : c + gy) {\n";
  for (int st = 0; st < NST; ++st) {
    s << "          {\n"
      << "          const unsigned slot = g % " << p.slots << "u, buf = g % " << p.nbuf << "u, use = g / " << p.nbuf << "u;\n"
      << "          ok = ok && kx_mb_wait(full + 8 * slot, (g / " << p.slots << "u) & 1);\n"
      << "          if (use > 0) ok = ok && kx_mb_wait(dfree + 8 * buf, (use - 1) & 1);\n"
      << "          ok = __all_sync(0xffffffffu, ok);\n"
      << "          kx_fence_after();\n"
      << "          if (ok && kx_elect()) {\n"
      << "          const unsigned dt = tmem + " << p.acols << " + buf * " << p.dcols << ";\n"
      << "          const unsigned long long bd = (unsigned long long)((kx_smem(slots) + slot * " << p.slot_bytes << "u) >> 4) | (8ull << 16) | ((unsigned long long)"
      << K << " << 32) | (1ull << 46);\n"
      << mma_code(p, p.st[st])
      << "          kx_commit(dfull + 8 * buf);\n"
      << "          kx_commit(empty + 8 * slot);\n"
      << "          }\n          __syncwarp();\n          ++g;\n          }\n";
  }
  s << "        }\n      }\n  }\n";
  // ---- compute warps
  s << "  else {\n"
    << "    const int s = threadIdx.x & 127, wg = threadIdx.x >> 7;\n"
    << "    const unsigned tl = tmem + ((unsigned)(warp & 3) << 21);\n"
    << "    unsigned g = 0;\n"
    << "    long long i = min((long long)blockIdx.x * 128 + s, n - 1);\n"
    << "    double T = T_[i], P = P_[i];\n";
  auto copy_y = [&](const char* ind, const char* idx) {
    s << ind << "#pragma unroll 4\n" << ind << fmt("for (int q = 0; q < %d; ++q) {\n", 4 * QW)
      << ind << fmt("  const int j = wg * %d + q;\n", 4 * QW)
      << ind << fmt("  if (j < %d) kx_copy8(kx_smem(sy + j * 128 + s), Y_ + (long long)j * ld + %s);\n", ns, idx)
      << ind << "}\n";
  };
  if (stage_y) {
    s << fmt("    for (int j = %d + wg; j < %d; j += %d) sy[j * 128 + s] = 0.0;\n", ns, K, G);
    copy_y("    ", "i");
  }
  s << "    for (long long t = blockIdx.x; t < tiles; t += gridDim.x) {\n"
    << "      const bool in = t * 128 + s < n;\n"
    << "      bool bad = !(T > 0.0 && P > 0.0 && T < KX_INF && P < KX_INF);\n"
    << (thermo ? std::string("      bool gen = false;\n") : fmt("      bool gen = !(T >= %s && T <= %s);\n", D(kTcTlo).c_str(), D(kTcThi).c_str()));
  const char* kShare = "if (!ok) failed = 1;\n      KX_COMPUTE_SYNC;\n      ok = __all_sync(0xffffffffu, ok && !failed);\n";
  auto yval = [&](const std::string& j) {
    return stage_y ? fmt("sy[(%s) * 128 + s]", j.c_str()) : fmt("((%s) < %d ? Y_[(long long)(%s) * ld + i] : 0.0)", j.c_str(), ns, j.c_str());
  };
  if (stage_y) {
    s << "      asm volatile(\"cp.async.wait_all;\" ::: \"memory\");\n";
    if (K > ns) s << "      if (t == blockIdx.x) KX_COMPUTE_SYNC;   // the padding's zeros\n";
  }
  // largest exponent of Y_j 2^ecol_j
  s << "      int mx = 0, raw = 0;\n"
    << "      #pragma unroll 4\n"
    << fmt("      for (int q = 0; q < %d; ++q) {\n", 4 * QW)
    << fmt("        const int j = wg * %d + q;\n", 4 * QW)
    << "        const int e = (__double2hiint(" << yval("j") << ") >> 20) & 0x7ff;\n"
    << "        mx = max(mx, e + sec[j]);\n        raw = max(raw, e);\n      }\n"
    << "      sred[wg * 128 + s].x = __int_as_float(raw == 0x7ff ? 100000 : mx);\n"
    << "      KX_COMPUTE_SYNC;\n"   // (the previous tile's shared values are no longer read)
    << "      #pragma unroll\n"
    << "      for (int q = 0; q < " << G << "; ++q) mx = max(mx, __float_as_int(sred[q * 128 + s].x));\n"
    << "      if (mx >= 100000 || mx < 64) gen = true;\n";
  if (p.bound_v) {
    // sum v in units of 2^-12 from the mantissas' first 12 bits (rounded up), over the compute groups
    s << "      int sv = 0;\n"
      << "      #pragma unroll 4\n"
      << fmt("      for (int q = 0; q < %d; ++q) {\n", 4 * QW)
      << fmt("        const int j = wg * %d + q;\n", 4 * QW)
      << "        const int hi = __double2hiint(" << yval("j") << ");\n"
      << "        sv += (int)((0x801u + (((unsigned)hi >> 9) & 0x7ffu)) >> min((unsigned)(mx - sec[j] - ((hi >> 20) & 0x7ff)), 31u));\n      }\n"
      << "      sred[wg * 128 + s].y = __int_as_float(sv);\n      KX_COMPUTE_SYNC;\n      sv = 0;\n"
      << "      #pragma unroll\n"
      << "      for (int q = 0; q < " << G << "; ++q) sv += __float_as_int(sred[q * 128 + s].y);\n"
      << fmt("      for (int most = %d; sv > most && most < %d; most *= 2) ++mx;\n", kSumMost * 4096, 4096 * ns);
  }
  s
    << "      const bool off = bad || gen;\n"
    << "      const int sc = off ? 0 : 1022 - mx;   // v_j = Y_j 2^(ecol_j + sc), the largest in [1/2, 1)\n"
    << "      if (off) mx = 1 << 20;\n";
  // digits: the integer round(v 2^49) (mixed: 2^29) plus 512 in every base-1024 place, so that the places
  // hold the digits plus 512 (the highest up to 1024)
  int QB = 4;   // quads that one block of digits covers
  while (QW % QB) --QB;
  s << fmt("      #pragma unroll 1\n      for (int b4 = 0; b4 < %d; b4 += %d) {\n", QW, QB)
    << fmt("      unsigned w[%d][%d];\n", p.nd, 2 * QB)
    << "      #pragma unroll\n"
    << fmt("      for (int q2 = 0; q2 < %d; ++q2) {\n", 2 * QB)
    << "        unsigned gl[2], gh[2];\n        #pragma unroll\n        for (int q = 0; q < 2; ++q) {\n"
    << fmt("          const int j = wg * %d + 4 * b4 + 2 * q2 + q;\n", 4 * QW)
    << "          const double yv = " << yval("j") << ";\n"
    << "          const unsigned hi = (unsigned)__double2hiint(yv), lo = (unsigned)__double2loint(yv);\n"
    << "          const int d = mx - sec[j] - (int)((hi >> 20) & 0x7ffu);   // binary orders below the largest\n"
    << "          const unsigned neg = (unsigned)((int)hi >> 31);\n";
  if (!mixed) {
    s << "          const unsigned long long mm = ((unsigned long long)((hi & 0xfffffu) | 0x100000u) << 32) | lo;\n"
      << "          const unsigned long long f = ((mm >> min((unsigned)d + 3u, 63u)) ^ (unsigned long long)(long long)(int)neg) + "
         "(0x4010040100401ull - (unsigned long long)(long long)(int)neg);\n"
      << "          gl[q] = (unsigned)f; gh[q] = (unsigned)(f >> 32);\n"
      << "        }\n"
      << "        w[4][q2] = kx_digits(kx_pack(gl[0] >> 1, gl[1] << 15));\n"
      << "        w[3][q2] = kx_digits(kx_pack(gl[0] >> 11, gl[1] << 5));\n"
      << "        w[2][q2] = kx_digits(kx_pack(gl[0] >> 21, gl[1] >> 5));\n"
      << "        w[1][q2] = kx_digits(kx_pack(__funnelshift_r(gl[0], gh[0], 31), __funnelshift_r(gl[1], gh[1], 15)));\n"
      << "        w[0][q2] = kx_digits((gh[0] >> 9) + ((gh[1] >> 9) << 16) + 0x64006400u);\n";
  } else {
    s << "          const unsigned mm = (((hi & 0xfffffu) | 0x100000u) << 11) | (lo >> 21);\n"
      << "          gl[q] = (__funnelshift_rc(mm, 0u, (unsigned)d + 2u) ^ neg) + (0x40100401u - neg);\n"
      << "        }\n"
      << "        w[2][q2] = kx_digits(kx_pack(gl[0] >> 1, gl[1] << 15));\n"
      << "        w[1][q2] = kx_digits(kx_pack(gl[0] >> 11, gl[1] << 5));\n"
      << "        w[0][q2] = kx_digits((gl[0] >> 21) + ((gl[1] >> 21) << 16) + 0x64006400u);\n";
  }
  s << "      }\n      #pragma unroll\n" << fmt("      for (int k = 0; k < %d; ++k) {\n", p.nd);
  for (int at = 0; at < 2 * QB;) {
    const int x = 2 * QB - at >= 8 ? 8 : 2 * QB - at >= 4 ? 4 : 2;
    s << fmt("        kx_st%d(tl + k * %d + wg * %d + 2 * b4 + %d, &w[k][%d]);\n", x, K / 2, 2 * QW, at, at);
    at += x;
  }
  s << "      } }\n"
    << "      kx_wait_st();\n      kx_fence_before();\n      __syncwarp();\n      if (lane == 0) kx_mb_arrive(aready);\n";
  // the next tile's states on their way
  s << "      const long long in1 = min((t + gridDim.x) * 128 + s, n - 1);\n"
    << "      const double T1 = T_[in1], P1 = P_[in1];\n";
  if (stage_y) copy_y("      ", "in1");
  if (!thermo) {
  // ln T and the basis functions, dealt to the groups, while the first matrix products run
  s << "      const kx_df L = kx_df_log(kx_df_mul(kx_d2df_i(gen ? 1000.0 : T), " << DFc(1.0 / kTcTmid) << "));   // ln T - L_mid\n"
    << "      const kx_df tb = kx_df_mul(L, " << DFc(1.0 / kTcLhalf) << "), t2 = kx_df_mul(tb, tb);\n";
  {
    // cost-balanced deal: float pairs about 12 instructions a degree, float32 one
    std::vector<std::pair<int, int>> jobs;
    for (int q = 1; q <= b.M; ++q) jobs.push_back({-(int)(b.phi[q].size()) * ((mixed || b.E[q] <= kPhiE) ? 2 : 12), q});
    std::sort(jobs.begin(), jobs.end());
    int load[4] = {60, 60, 0, 0};   // the common factors are groups 0 and 1's
    std::vector<int> who[4];
    for (auto& j : jobs) {
      const int w = (int)(std::min_element(load, load + G) - load);
      load[w] -= j.first;
      who[w].push_back(j.second);
    }
    for (int w = 0; w < G; ++w) {
      s << fmt("      %sif (wg == %d) {\n", w ? "else " : "", w);
      for (int q : who[w]) {
        if (mixed || b.E[q] <= kPhiE) continue;
        // even and odd powers side by side
        const int half = ((int)b.phi[q].size() - 1) / 2;
        s << fmt("        { kx_df fe = kx_f2(sph[%d]), fo = kx_f2(sph[%d]);\n", 32 * q + 2 * half, 32 * q + 2 * half + 1)
          << fmt("          #pragma unroll 2\n          for (int k = %d; k >= 0; --k) {\n", half - 1)
          << fmt("            fe = kx_df_fma_u(fe, t2, kx_f2(sph[%d + 2 * k])); fo = kx_df_fma_u(fo, t2, kx_f2(sph[%d + 2 * k + 1]));\n          }\n",
                 32 * q, 32 * q)
          << fmt("          const kx_df f = kx_df_fma(fo, tb, fe); sphi[%d * 128 + s] = make_float2(f.hi, f.lo); }\n", q);
      }
      std::vector<int> floats;
      for (int q : who[w]) if (mixed || b.E[q] <= kPhiE) floats.push_back(q);
      for (size_t at = 0; at < floats.size(); at += 4) {
        const size_t end = std::min(floats.size(), at + 4);
        int deg = 0;
        for (size_t x = at; x < end; ++x) deg = std::max(deg, (int)b.phi[floats[x]].size() - 1);
        s << "        {\n";
        // Clenshaw's recurrence in T_n(t), four side by side
        s << "          const float tt = __fmul_rn(2.0f, tb.hi);\n";
        for (size_t x = at; x < end; ++x) s << fmt("          float f%zu = sph[%d].x, g%zu = 0.0f;\n", x - at, 32 * floats[x] + deg, x - at);
        s << fmt("          #pragma unroll 3\n          for (int k = %d; k >= 1; --k) {\n", deg - 1);
        for (size_t x = at; x < end; ++x)
          s << fmt("            { const float h = __fmaf_rn(tt, f%zu, __fsub_rn(sph[%d + k].x, g%zu)); g%zu = f%zu; f%zu = h; }\n", x - at, 32 * floats[x],
                   x - at, x - at, x - at, x - at);
        s << "          }\n";
        for (size_t x = at; x < end; ++x) s << fmt("          f%zu = __fmaf_rn(tb.hi, f%zu, -g%zu);\n", x - at, x - at, x - at);
        for (size_t x = at; x < end; ++x) s << fmt("          sphi[%d * 128 + s] = make_float2(f%zu, 0.0f);\n", floats[x], x - at);
        s << "        }\n";
      }
      if (w < 2) {   // common factors e^g0, e^g1
        const int o = 5 * w;
        if (w == 0 || visc) {
          s << fmt("        { kx_df f = kx_mk(kx_g[%d].x, kx_g[%d].y);\n          for (int k = 3; k >= 1; --k) f = kx_df_fma_u(f, L, kx_mk(kx_g[%d + k].x, kx_g[%d + k].y));\n"
                   "          f = kx_df_mul(kx_df_exp_x(kx_df_mul(f, L)), %s); sred[%d * 128 + s] = make_float2(f.hi, f.lo); }\n", o + 4, o + 4, o, o,
                   DFc(w ? b.g1c : b.g0c).c_str(), 4 + w);
        }
      }
      s << "      }\n";
    }
  }
  s << "      KX_COMPUTE_SYNC;\n";
  }
  // rows
  if (visc) s << "      kx_df mu = kx_mk(0.0f, 0.0f);\n";
  if (diff) s << (mixed ? "      float fac = 0.0f, sYs = 0.0f;\n" : "      kx_df fac = kx_mk(0.0f, 0.0f), sYs = fac;\n");
  s << "      for (int c = 0; c < " << p.chunks << "; c = c == 0 ? cnext : c + gy) {\n"
    << (mixed ? fmt("      float hi[%d];\n", RT) : fmt("      float hi[%d], lo[%d], sm[%d];\n", RT, RT, RT))
    << (thermo ? std::string() : fmt("      double yr[%d];\n", RT));
  if (!thermo)
    s << fmt("      #pragma unroll\n      for (int a = 0; a < %d; ++a) {\n", RT)
    << fmt("        const int k = c * 16 + wg * %d + a - %d;\n", RT, b.first)
    << fmt("        yr[a] = k >= 0 && k < %d ? Y_[(long long)k * ld + i] : 0.0;\n      }\n", ns);
  for (int st = 0; st < NST; ++st) {
    s << "      {\n"
      << "      const unsigned buf = g % " << p.nbuf << "u;\n"
      << "      ok = __all_sync(0xffffffffu, ok && kx_mb_wait(dfull + 8 * buf, (g / " << p.nbuf << "u) & 1));\n"
      << "      kx_fence_after();\n"
      << "      const unsigned td = tl + " << p.acols << " + buf * " << p.dcols << " + wg * " << RT << ";\n"
      << sum_code(p, p.st[st]) << "      ++g;\n      }\n";
  }
  if (!mixed) {
    s << fmt("      #pragma unroll\n      for (int a = 0; a < %d; ++a)", RT) << " { const kx_df w = kx_ts(hi[a], sm[a]); const kx_df z = kx_ts(w.hi, __fadd_rn(w.lo, lo[a])); hi[a] = z.hi; lo[a] = z.lo; }\n";
  }
  const char* LO = mixed ? "0.0f" : "lo[a]";
  if (thermo) {
    s << fmt("      #pragma unroll\n      for (int a = 0; a < %d; ++a) sred[(8 + c * 16 + wg * %d + a) * 128 + s] = make_float2(hi[a], lo[a]);\n      }\n", RT, RT)
      << "      " << kShare
      // c_p = sum B_n x^n, h = h(x = 0) + T_half x sum B_n/(n + 1) x^n over the T_mid groups
      << "      if (wg < 2 && in && !bad && !gen && ok) {\n"
      << "        const kx_df Td = kx_d2df_i(T);\n        kx_df v = kx_mk(0.0f, 0.0f);\n";
    for (size_t g = 0; g < p.mids.size(); ++g) {
      long long bits;
      std::memcpy(&bits, &p.mids[g], 8);
      s << fmt("        {\n          const bool low = __double_as_longlong(T) < %lldLL;\n", bits)
        << fmt("          const kx_df xc = kx_df_add(Td, kx_mk(low ? %s : %s, 0.0f));\n", F(-kThTc[0]).c_str(), F(-kThTc[1]).c_str())
        << fmt("          const float xs = low ? %s : %s;\n", F(1.0 / kThHalf[0]).c_str(), F(1.0 / kThHalf[1]).c_str())
        << "          const kx_df x = kx_mk(xc.hi * xs, xc.lo * xs);\n"
        << fmt("          const int r0 = low ? %d : %d;\n", 12 * (int)g, 12 * (int)g + 6)
        << "          kx_df B[6];\n          #pragma unroll\n          for (int k = 0; k < 6; ++k) {\n"
        << "            const float2 q = sred[(8 + r0 + k) * 128 + s]; const float f = srs[r0 + k].x;\n"
        << "            B[k] = kx_mk(q.x * f, q.y * f);\n          }\n"
        << "          if (wg == 0) {\n"
        << "            v = kx_df_add(v, kx_df_fma(kx_df_fma(kx_df_fma(kx_df_fma(B[4], x, B[3]), x, B[2]), x, B[1]), x, B[0]));\n"
        << "          } else {\n"
        << fmt("            kx_df q = kx_df_mul(B[4], %s);\n", DFc(0.2).c_str())
        << fmt("            q = kx_df_fma(q, x, kx_df_mul(B[3], %s));\n", DFc(0.25).c_str())
        << fmt("            q = kx_df_fma(q, x, kx_df_mul(B[2], %s));\n", DFc(1.0 / 3.0).c_str())
        << fmt("            q = kx_df_fma(q, x, kx_df_mul(B[1], %s));\n", DFc(0.5).c_str())
        << "            q = kx_df_fma(q, x, B[0]);\n"
        << "            v = kx_df_add(v, kx_df_fma(q, xc, B[5]));\n"
        << "          }\n        }\n";
    }
    s << "        (wg == 0 ? out0_ : out1_)[i] = kx_df2d_s(v, -18 - sc);\n      }\n";
  } else {
  s << "      if (c == 0) {\n"
    << fmt("        #pragma unroll\n        for (int a = 0; a < %d; ++a)\n          if (wg * %d + a < %d) sred[(8 + wg * %d + a) * 128 + s] = make_float2(hi[a], %s);\n", RT, RT, b.first, RT, LO)
    << "        " << kShare
    << "        const float2 c0 = sred[8 * 128 + s], c1 = sred[9 * 128 + s], g0 = sred[4 * 128 + s];\n"
    << "        if (!gen && !(c0.x > 0.0f)) bad = true;\n";
  if (diff) {
    // D_k = (1 - Y_k/sum Y) (p_atm/p) sigma / sum_{j != k} (Y_j/W_j)/D_kj
    if (!mixed)
      s << "        sYs = kx_mk(c1.x, c1.y);\n"
        << "        fac = kx_df_div(kx_df_mul(kx_df_div(kx_mk(c0.x, c0.y), sYs), kx_df_div(" << DFc(P_ATM) << ", kx_d2df_i(P))), kx_mk(g0.x, g0.y));\n";
    else
      s << "        sYs = c1.x;\n        fac = __fdividef(c0.x, c1.x) * __fdividef(" << F(P_ATM) << ", kx_d2f(P)) / g0.x;\n";
  } else {
    s << "        if (wg == 0 && in && !bad && !gen && ok) {\n"
      << "          const float2 c2 = sred[10 * 128 + s], c3 = sred[11 * 128 + s], c4 = sred[12 * 128 + s], g1 = sred[5 * 128 + s];\n";
    // sum X lambda = g1 (c1 + c3)/c0, sum X/lambda = (c2 + c4)/(c0 g1), each row under its own power of two
    auto sum2 = [&](const char* x, int rx, const char* y, int ry) {
      const int top = std::max(b.rho[rx], b.rho[ry]);
      auto sc = [&](const char* v, int r) {
        const std::string f = F(std::ldexp(1.0, b.rho[r] - top));
        return mixed ? fmt("%s.x * %s", v, f.c_str()) : fmt("kx_mk(%s.x * %s, %s.y * %s)", v, f.c_str(), v, f.c_str());
      };
      return mixed ? fmt("(%s + %s)", sc(x, rx).c_str(), sc(y, ry).c_str()) : fmt("kx_df_add(%s, %s)", sc(x, rx).c_str(), sc(y, ry).c_str());
    };
    const int t1 = std::max(b.rho[1], b.rho[3]), t2 = std::max(b.rho[2], b.rho[4]);
    if (!mixed)
      s << "          const kx_df is = kx_df_div(kx_mk(1.0f, 0.0f), kx_mk(c0.x, c0.y)), gl = kx_mk(g1.x, g1.y);\n"
        << "          const kx_df l1 = kx_df_mul(kx_df_mul(" << sum2("c1", 1, "c3", 3) << ", is), gl);\n"
        << "          const kx_df li = kx_df_div(gl, kx_df_mul(" << sum2("c2", 2, "c4", 4) << ", is));\n"
        << fmt("          out1_[i] = 0.5 * (kx_df2d(l1) * %s + kx_df2d(li) * %s);\n", D(std::ldexp(1.0, t1 - b.rho[0])).c_str(),
               D(std::ldexp(1.0, b.rho[0] - t2)).c_str());
    else
      s << fmt("          out1_[i] = kx_f2d(0.5f * g1.x * (__fdividef(%s, c0.x) * %s + __fdividef(c0.x, %s) * %s));\n",
               sum2("c1", 1, "c3", 3).c_str(), F(std::ldexp(1.0, t1 - b.rho[0])).c_str(), sum2("c2", 2, "c4", 4).c_str(),
               F(std::ldexp(1.0, b.rho[0] - t2)).c_str());
    s << "        }\n";
  }
  s << "      }\n";
  // this chunk's rows
  s << "      if (c != 0 || cy == 0) {\n"
    << "        const bool act = in && !bad && !gen && ok;\n"
    << fmt("        const int k0 = c * 16 + wg * %d - %d;   // the first row's species (the same in every lane)\n", RT, b.first);
  if (visc) {
    s << fmt("        #pragma unroll\n        for (int a = 0; a < %d; ++a) {\n", RT)
      << fmt("          if (k0 + a < 0 || k0 + a >= %d || !act) continue;\n", ns)
      << fmt("          const float2 rs = srs[k0 + a + %d];\n", b.first);
    if (!mixed)
      s << "          mu = kx_df_add_u(mu, kx_div_n(kx_df_mul_u(kx_pair_shift(yr[a], sc), kx_mk(rs.x, rs.y)), kx_mk(hi[a], lo[a])));\n";
    else
      s << "          mu.hi = __fmaf_rn(kx_float_shift(yr[a], sc) * rs.x, kx_rcp(hi[a]), mu.hi);\n";
    s << "        }\n";
  } else {
    // every row's value first (independent chains), then the stores, then the rows below 2^-5 sqrt(N_s/64) of the largest v (the sum's error is about
    // 2^-47 sqrt(N_s/64) of it)
    s << fmt("        double dv[%d];\n        #pragma unroll\n        for (int a = 0; a < %d; ++a) {\n", RT, RT)
      << fmt("          const float rs = srs[max(k0 + a, -%d) + %d].x;\n", b.first, b.first);
    if (!mixed)
      s << fmt("          const kx_df ys = kx_pair_shift(yr[a], sc + %d);\n", 18 - b.rho[1])
        << "          const kx_df num = kx_qts(sYs.hi, -ys.hi);   // Y_k <= sum Y, or within a factor of two of it\n"
        << "          const kx_df q = kx_div_n(kx_df_mul_u(kx_mk(num.hi, __fadd_rn(num.lo, __fsub_rn(sYs.lo, ys.lo))), fac), kx_mk(hi[a], lo[a]));\n"
        << "          dv[a] = kx_df2d_b(q, (__float_as_int(rs) >> 23) - 127);\n";
    else
      s << fmt("          const float ys = kx_float_shift(yr[a], sc + %d);\n", 18 - b.rho[1])
        << "          dv[a] = kx_f2d((sYs - ys) * fac * kx_rcp(hi[a]) * rs);\n";
    s << "        }\n"
      << fmt("        unsigned any = 0;\n        #pragma unroll\n        for (int a = 0; a < %d; ++a) {\n", RT)
      << fmt("          if (k0 + a < 0 || k0 + a >= %d) continue;\n", ns)
      << "          const bool low = act && !(hi[a] >= " << F(std::ldexp(std::sqrt(ns / 64.0), 13)) << ");\n"
      << "          if (act && !low) out2_[(long long)(k0 + a) * ld + i] = dv[a];\n"
      << "          if (low) any |= 1u << a;\n        }\n"
      << fmt("        for (int a = 0; a < %d && __any_sync(0xffffffffu, any); ++a)\n", RT)
      << "          for (unsigned w = __ballot_sync(0xffffffffu, (any >> a) & 1u); w; w &= w - 1) {\n"
      << "            const int src = __ffs(w) - 1;\n"
      << "            const double d = kx_diff_row(Y_, ld, __shfl_sync(0xffffffffu, i, src), k0 + a, __shfl_sync(0xffffffffu, L.hi, src),\n"
      << "                                         __shfl_sync(0xffffffffu, L.lo, src), __shfl_sync(0xffffffffu, P, src));\n"
      << "            if (lane == src) out2_[(long long)(k0 + a) * ld + i] = d;\n          }\n";
  }
  s << "      }\n      }\n";
  if (visc) {
    s << "      sred[(16 + wg) * 128 + s] = make_float2(mu.hi, mu.lo);\n      " << kShare
      << "      if (wg == 0 && in && !bad && !gen && ok) {\n"
      << "        const float2 g0 = sred[4 * 128 + s];\n";
    if (!mixed)
      s << "        for (int w = 1; w < " << G << "; ++w) { const float2 v = sred[(16 + w) * 128 + s]; mu = kx_df_add(mu, kx_mk(v.x, v.y)); }\n"
        << "        out0_[i] = kx_df2d(kx_df_mul(mu, kx_mk(g0.x, g0.y)));\n";
    else
      s << "        for (int w = 1; w < " << G << "; ++w) mu.hi += sred[(16 + w) * 128 + s].x;\n"
        << "        out0_[i] = kx_f2d(mu.hi * g0.x);\n";
    s << "      }\n";
  }
  }
  // states outside the domain, outside the basis' temperatures or with non-finite mass fractions
  // A wait that ran out: every block's own results are nan, and the point recorded (diffusion: the rows of this
  // warp's group in the block's chunks; else by the group that writes them, which has seen the others' flag)
  s << "      if (!ok && in) {\n"
    << (diff ? "        atomicMin(&kx_bad_first, (unsigned long long)i);\n" : "        if (wg == 0) atomicMin(&kx_bad_first, (unsigned long long)i);\n");
  if (diff)
    s << fmt("        for (int c = cy; c < %d; c += gy)\n          for (int a = 0; a < %d; ++a) {\n", p.chunks, RT)
      << fmt("            const int k = c * 16 + wg * %d + a - %d;\n", RT, b.first)
      << fmt("            if (k >= 0 && k < %d) out2_[(long long)k * ld + i] = KX_NAN;\n          }\n", ns);
  else
    s << "        if (wg == 0) { out0_[i] = KX_NAN; out1_[i] = KX_NAN; }\n";
  s << "      }\n";
  s << "      if (cy == 0 && ok && __any_sync(0xffffffffu, in && (bad || gen))) {\n";
  s << "        if (in && bad) {\n"
    << "          if (wg == 0) atomicMin(&kx_bad_first, (unsigned long long)i);\n";
  if (thermo) {
    s << "          if (wg == 0) { out0_[i] = KX_NAN; out1_[i] = KX_NAN; }\n        } else if (in && gen && wg == 0) {\n"
      << "          const double2 v = kx_thermo_state(Y_, ld, i, T);\n          out0_[i] = v.x; out1_[i] = v.y;\n        }\n";
  } else {
    if (visc) s << "          if (wg == 0) { out0_[i] = KX_NAN; out1_[i] = KX_NAN; }\n        }\n";
    else s << fmt("          for (int k = wg; k < %d; k += %d) out2_[(long long)k * ld + i] = KX_NAN;\n        }\n", ns, G);
    // the states pair by pair, one after the other by a warp, dealt to the groups
    s << "        const kx_df Lt = kx_d2df(log(gen && !bad ? T : 1000.0) - " << D(kTcLmid) << ");\n"
      << "        int nth = 0;\n"
      << "        for (unsigned w = __ballot_sync(0xffffffffu, in && gen && !bad); w; w &= w - 1, ++nth) {\n"
      << fmt("          if ((nth & %d) != wg) continue;\n", G - 1)
      << "          const int src = __ffs(w) - 1;\n"
      << "          const long long is = __shfl_sync(0xffffffffu, i, src);\n"
      << "          const float Lh = __shfl_sync(0xffffffffu, Lt.hi, src), Ll = __shfl_sync(0xffffffffu, Lt.lo, src);\n";
    if (visc) s << "          const double2 v = kx_visc_state(Y_, ld, is, Lh, Ll);\n"
                << "          if (lane == src) { out0_[i] = v.x; out1_[i] = v.y; }\n        }\n";
    else s << "          kx_diff_state(Y_, ld, is, Lh, Ll, __shfl_sync(0xffffffffu, P, src), out2_);\n        }\n";
  }
  s << "      }\n      i = in1; T = T1; P = P1;\n    }\n    asm volatile(\"cp.async.wait_all;\" ::: \"memory\");\n  }\n";
  s << "  kx_fence_before();\n  __syncthreads();\n"
    << fmt("  if (warp == %d) asm volatile(\"tcgen05.dealloc.cta_group::1.sync.aligned.b32 %%0, %d;\" ::\"r\"(tmem));\n", 4 * G, 512);
  s << "}\n";
  if (counts) {
    // float32-pipe instructions per state: digits, basis functions, level sums, rows
    double f = 25.0 * ns;
    for (int q = 1; q <= b.M; ++q) f += b.phi[q].size() * ((mixed || b.E[q] <= kPhiE) ? 2.0 : 12.0);
    double per = mixed ? 10 : 45;
    for (int q = 0; q <= b.M; ++q) per += (mixed || b.E[q] <= kFloatE) ? p.lev[q] : (6 + 2 + (p.lev[q] >= 3 ? 5 : 0) + (p.lev[q] >= 4 ? 2 : 0) + (q ? 9 : 0));
    counts->fp32 += f + per * b.rows;
    counts->fp64 += diff ? 1 : 3;
  }
  if (shape) {
    shape->threads = kThreads;
    shape->smem = p.smem;
    shape->states_per_block = kStates;
    shape->row_chunks = diff ? p.chunks : 1;
  }
  return s.str();
}

}  // namespace kx
