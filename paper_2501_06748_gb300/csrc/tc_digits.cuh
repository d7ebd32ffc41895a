// FP16 digit splitting of FP64 operands for the tensor-core element kernels (shared by
// the one- and two-row-tile kernels): binary64 fields to fixed point, balanced base-512
// digits, m16n8k16 products per significance level, exact integer recombination, and
// the bulk copies and mbarriers of the operator ring.  The method is described in tc.cu.
#pragma once
#include <cstdint>
#include <cuda_fp16.h>

#include "internal.h"

namespace sbfwi {

namespace tc {

constexpr int kSlices = 6;      // base-512 digits per operand
constexpr int kLevels = 7;      // significance levels kept: k + l = 2..8
constexpr int kTile = 16;       // rows / inner dimension of one mma tile
constexpr int kCols = 8;        // shots of one mma tile

// round(a * 2^(53 - e)) for |a| < 2^e, from the binary64 fields (integer work only)
__device__ __forceinline__ long long to_fixed(double a, int e) {
  const long long bits = __double_as_longlong(a);
  if ((bits & 0x7FFFFFFFFFFFFFFFLL) == 0) return 0;
  const int ex = (int)((bits >> 52) & 0x7FF);
  long long mant = bits & 0x000FFFFFFFFFFFFFLL;
  int ex_eff = ex;
  if (ex == 0) ex_eff = 1;              // subnormal
  else mant |= 0x0010000000000000LL;
  // right shift of the 53-bit significand; |a| < 2^e makes it >= 0
  const int sh = e + 1022 - ex_eff;
  long long v;
  if (sh <= 0) v = mant;
  else if (sh >= 60) v = 0;
  else v = (mant + (1LL << (sh - 1))) >> sh;
  return bits < 0 ? -v : v;
}

// exponent e with |a| < 2^e (for a != 0); very small for a == 0 (integer work only)
__device__ __forceinline__ int exp_bound(double a) {
  const long long bits = __double_as_longlong(a);
  const int ex = (int)((bits >> 52) & 0x7FF);
  if (ex == 0) return (bits & 0x7FFFFFFFFFFFFFFFLL) == 0 ? -1100 : -1021;
  return ex - 1022;
}

// t * 2^E for results outside the normal range (never met by the path's fields): kept
// out of line so that its FP64 conversion is not evaluated speculatively on the hot path
static __device__ __noinline__ double int_to_double_scaled_slow(long long t, int E) { return ldexp((double)t, E); }

// six balanced base-512 digits, most significant first, as FP16 bit patterns of 1536 + d
// The 54-bit recurrence runs on two 32-bit halves: the low 27 bits give the three
// least significant digits and a carry (0 or 1) into the high half, which gives the
// rest -- the same digits as the recurrence on the whole integer.
__device__ __forceinline__ void digits(long long v, unsigned short (&h)[kSlices]) {
  int lo = (int)(v & ((1LL << 27) - 1));      // 0 .. 2^27 - 1
  int hi = (int)(v >> 27);                    // |hi| < 2^26 (arithmetic shift)
#pragma unroll
  for (int k = kSlices - 1; k >= kSlices - 3; --k) {
    const int d = ((lo + 256) & 511) - 256;
    lo = (lo - d) >> 9;
    h[k] = (unsigned short)(0x6600 + d);
  }
  hi += lo;                                   // carry of the low half
#pragma unroll
  for (int k = kSlices - 4; k >= 1; --k) {
    const int d = ((hi + 256) & 511) - 256;
    hi = (hi - d) >> 9;
    h[k] = (unsigned short)(0x6600 + d);
  }
  h[0] = (unsigned short)(0x6600 + hi);
}

// two FP16 patterns of 1536 + d packed in a register -> the pair (d0, d1) as half2
__device__ __forceinline__ unsigned pack_digits(unsigned short lo, unsigned short hi) {
  const unsigned u = (unsigned)lo | ((unsigned)hi << 16);
  __half2 h = *reinterpret_cast<const __half2*>(&u);
  h = __hsub2(h, __halves2half2(__ushort_as_half(0x6600), __ushort_as_half(0x6600)));
  return *reinterpret_cast<const unsigned*>(&h);
}

// ---------------------------------------------------------------------------
// The shot-major product of the element step: y^T = x^T A^T, shots in the rows of the
// mma.  The 16 rows of m16n8k16 hold 8 shots times two consecutive digits of x (row g:
// digit 2p of shot g, row g + 8: digit 2p + 1), its 8 columns 8 rows of the operator, so
// lane (g, t) = (lane / 4, lane % 4) has shot g and vector rows 2t, 2t+1, 2t+8, 2t+9 both
// as the product's operand and as its result: the sweep's next product starts from the
// registers of the last one, without an exchange between lanes, and 28 mma cover the 26
// digit pairs of a 16 x 16 product.
// What bounds it: the number of instructions around the mma (a warp issues them one
// dependent chain at a time, 4 warps per scheduler), so both conversions are cut to
// shifts, byte permutes and 32-bit adds:
//  - the significand is shifted once, with eight fraction bits kept for the rounding; its
//    balanced digits are the 9-bit fields of the integer plus a constant (each field less
//    256), taken for two values at once by byte permutes of 16-bit windows;
//  - accumulators start at 1.5 * 2^23, so the bits of a sum are the constant plus the sum
//    (exact while |sum| <= 2^22: at most four mma of 16 products of |digit| <= 256 per
//    accumulator) and the levels are added as 32-bit integers.
// Measured (64 x 64 elements, n_b 16, N_r 32, 8 shots), with the operator blocks, ring and tiled
// state of tc_step.cuh: fused launch 0.555 -> 0.394 ms, 2124 -> 1500 instructions per warp and
// radial point of both sweeps, DRAM 4.5 -> 6.2 TB/s (6.8 measured copy).
// ---------------------------------------------------------------------------
constexpr int kPairs = kSlices / 2;
constexpr float kMagicF = 12582912.0f;            // 1.5 * 2^23: bits 0x4B400000
constexpr unsigned kMagicBits = 0x4B400000u;
constexpr int kMinExp = 64;                       // least biased exponent of a nonzero column's scale
constexpr int kScaledExp = 128;                   // columns below 2^(128 - 1023) are scaled up first
constexpr int kScaleBits = 256;

struct XDigits {          // A fragments of m16n8k16: digit pairs (0,1), (2,3), (4,5) of one 16-row operand
  uint4 f[kPairs];
};

// |x| as an ordered key: its high word without the sign (0 for |x| < 2^-1042)
__device__ __forceinline__ int mag_key(double x) { return __double2hiint(x) & 0x7FFFFFFF; }
__device__ __forceinline__ int max4(int a, int b, int c, int d) { return max(max(a, b), max(c, d)); }

// 256 * round-half-away(x 2^(53 - f)) in [0.., 8 fraction bits], two's complement, plus the digit
// constants, for E = f + 1022 (f the column's exponent): bits 8 + 9 j .. 16 + 9 j hold digit 5 - j plus
// 256 (j < 5), bits 53..62 digit 0 plus 512
__device__ __forceinline__ uint2 biased_fixed(double x, int E) {
  const unsigned lo = (unsigned)__double2loint(x);
  const int hi = __double2hiint(x);
  const int sgn = hi >> 31;
  const int ex = (hi >> 20) & 0x7FF;
  // the significand with its leading bit at position 60, its bits inverted for x < 0; an arithmetic shift
  // then gives floor(|x| ..) or its complement, and adding half a unit rounds half away from zero
  const int mh = (int)(__funnelshift_l(lo, (unsigned)hi, 8) & 0x0FFFFFFFu) ^ (sgn ^ 0x10000000);
  const unsigned ml = (lo << 8) ^ (unsigned)sgn;
  const int sh = min(max(E - ex, 0), 62);          // 62: the value vanishes (also zeros and subnormals)
  const long long d = (long long)(((unsigned long long)(unsigned)mh << 32) | ml) >> sh;
  constexpr unsigned long long kC =
      256ULL * (1ULL + (1ULL << 9) + (1ULL << 18) + (1ULL << 27) + (1ULL << 36)) + (512ULL << 45);
  const unsigned long long y = (unsigned long long)d + ((kC << 8) + 128ULL);
  return make_uint2((unsigned)y, (unsigned)(y >> 32));
}

__device__ __forceinline__ unsigned unbias(unsigned fields, unsigned bias2) {
  const __half2 h = __hsub2(*reinterpret_cast<const __half2*>(&fields), *reinterpret_cast<const __half2*>(&bias2));
  return *reinterpret_cast<const unsigned*>(&h);
}

// the six digits of two values as half2 (first value in the low half)
__device__ __forceinline__ void digit_pairs(uint2 a, uint2 b, unsigned (&d)[kSlices]) {
  // 16-bit windows of both values: fields at bit offset 0, 1, 0, 3, 4, 5 of each half
  const unsigned w5 = __byte_perm(a.x, b.x, 0x6521), w4 = __byte_perm(a.x, b.x, 0x7632);
  const unsigned w3 = __byte_perm(__funnelshift_r(a.x, a.y, 26), __funnelshift_r(b.x, b.y, 26), 0x5410);
  const unsigned w2 = __byte_perm(a.y, b.y, 0x5410), w1 = __byte_perm(a.y, b.y, 0x6521), w0 = __byte_perm(a.y, b.y, 0x7632);
  constexpr unsigned m9 = 0x01FF01FFu, one = 0x64006400u, b9 = 0x65006500u;   // 1024 + field; 1280
  d[5] = unbias((w5 & m9) | one, b9);
  d[4] = unbias((w4 & 0x03FE03FEu) | 0x60006000u, 0x62006200u);               // 512 + field; 768
  d[3] = unbias((w3 & m9) | one, b9);
  d[2] = unbias(((w2 >> 3) & m9) | one, b9);
  d[1] = unbias(((w1 >> 4) & m9) | one, b9);
  d[0] = unbias(((w0 >> 5) & 0x03FF03FFu) | one, 0x66006600u);                // 1024 + field; 1536
}

__device__ __forceinline__ void split_rows(const double* x, int E, XDigits& d) {   // x: 4 values
  unsigned lo[kSlices], hi[kSlices];
  digit_pairs(biased_fixed(x[0], E), biased_fixed(x[1], E), lo);
  digit_pairs(biased_fixed(x[2], E), biased_fixed(x[3], E), hi);
#pragma unroll
  for (int p = 0; p < kPairs; ++p) d.f[p] = make_uint4(lo[2 * p], lo[2 * p + 1], hi[2 * p], hi[2 * p + 1]);
}

// Biased exponent E of the scale of a column (shot) of 16 rows: |x| < 2^(E - 1022) for its entries, shared
// by the four lanes of the shot.  Columns near the bottom of the range are scaled up by 2^256 first
// (adj = 256, a whole warp's branch that the path's fields rarely take), so that subnormal entries keep
// their bits; then E > 62, which makes the shift of zero entries clear them (a column of zeros takes
// E = 1022, whose results stay inside scaled_double's range).
__device__ __forceinline__ int quad_max(int v) {
  v = max(v, __shfl_xor_sync(0xffffffffu, v, 1));
  return max(v, __shfl_xor_sync(0xffffffffu, v, 2));
}
constexpr int kZeroExp = -8192;                   // a column of zeros (or below 2^-1042)
__device__ __forceinline__ int exp_of_key(int key) { return key > 0 ? max(key >> 20, 1) : kZeroExp; }
__device__ __forceinline__ bool scale_small(int ex) { return ex > kZeroExp / 2 && ex < kScaledExp; }

template <int kV>
__device__ __forceinline__ int key_max(const double (&x)[kV]) {
  int k = 0;
#pragma unroll
  for (int j = 0; j < kV; j += 4) k = max(k, max4(mag_key(x[j]), mag_key(x[j + 1]), mag_key(x[j + 2]), mag_key(x[j + 3])));
  return k;
}

template <int kV>
__device__ __forceinline__ int column_scale(double (&x)[kV], int& adj) {
  auto ex_of = [&] { return exp_of_key(quad_max(key_max(x))); };
  int ex = ex_of();
  adj = 0;
  if (__any_sync(0xffffffffu, scale_small(ex))) {
    if (scale_small(ex)) {
      adj = kScaleBits;
#pragma unroll
      for (int j = 0; j < kV; ++j) x[j] *= 0x1p256;
    }
    ex = ex_of();
  }
  return ex < kMinExp ? 1022 : ex;
}

// The same for the joint operand [v ; q 2^bal], whose q takes its digits at eq = E - bal: the column is small for it
// already where E - bal is, in units where P is far below Q.  Where eq is too small for the conversion even after
// that, q (below 2^-958 then) is scaled up once more and eq with it, which leaves its digits as they are.  (The lift is
// off the chain of the sweep; a test of eq after E took 1.3 % of a session on 24 x 24 elements.)
// ex_of(): the column's exponent.
template <int kV, class ExOf>
__device__ __forceinline__ int joint_scale(double (&v)[kV], double (&q)[kV], int bal, int& adj, int& eq, ExOf ex_of) {
  const int lift = min(max(bal, 0), 1024);
  int ex = ex_of();
  adj = 0;
  int more = 0;
  if (__any_sync(0xffffffffu, scale_small(ex - lift))) {
    if (scale_small(ex - lift)) {
      adj = kScaleBits;
#pragma unroll
      for (int j = 0; j < kV; ++j) { v[j] *= 0x1p256; q[j] *= 0x1p256; }
    }
    ex = ex_of();
    if (ex >= kMinExp && ex - bal < kMinExp) {
      more = kScaleBits;
#pragma unroll
      for (int j = 0; j < kV; ++j) q[j] *= 0x1p256;
    }
  }
  const int E = ex < kMinExp ? 1022 : ex;
  eq = max(E - bal + more, kMinExp);
  return E;
}
template <int kV>
__device__ __forceinline__ int column_scale2(double (&v)[kV], double (&q)[kV], int bal, int& adj, int& eq) {
  return joint_scale<kV>(v, q, bal, adj, eq, [&] { return quad_max(max(exp_of_key(key_max(v)), exp_of_key(key_max(q)) + bal)); });
}

// mma of a digit pair fragment and an operator digit, on top of c (kFirst: of the start value)
template <bool kFirst>
__device__ __forceinline__ void mma_pair(float (&c)[4], const uint4& a, const uint2& b, const float (&start)[4]) {
  if (kFirst) {
    asm volatile(
        "mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%10,%11,%12,%13};\n"
        : "=f"(c[0]), "=f"(c[1]), "=f"(c[2]), "=f"(c[3])
        : "r"(a.x), "r"(a.y), "r"(a.z), "r"(a.w), "r"(b.x), "r"(b.y), "f"(start[0]), "f"(start[1]), "f"(start[2]),
          "f"(start[3]));
  } else {
    asm volatile(
        "mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};\n"
        : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
        : "r"(a.x), "r"(a.y), "r"(a.z), "r"(a.w), "r"(b.x), "r"(b.y));
  }
}

// Digit products of one accumulator row m = k + 2p (k: operator digit, p: pair of x digits) of one
// operand, and their number before operator digit k; m holds level m (even digit of the pair) in the
// results of row g and level m + 1 (odd digit) in those of row g + 8
__host__ __device__ constexpr bool pair_kept(int k, int p) { return k + 2 * p < kLevels; }
__host__ __device__ constexpr int pairs_before(int m, int k) {   // of row m, with an operator digit below k
  int c = 0;
  for (int p = 0; p < kPairs; ++p) c += (m - 2 * p >= 0 && m - 2 * p < k) ? 1 : 0;
  return c;
}
__host__ __device__ constexpr int pairs_of(int m) { return pairs_before(m, kSlices); }
// accumulators of row m for `ops` summed operands: four mma each (exact, see above)
__host__ __device__ constexpr int parts_of(int m, int ops) { return (ops * pairs_of(m) + 3) / 4; }

// The level sums of 8 operator rows (one n-tile), ops operands (16 columns each) summed: add(op, b) gives
// operand op's digits, b[k] the operator's B fragments.  Every (m, part) is a separate accumulator.
template <int kOps>
struct LevelSums {
  static constexpr int kMaxParts = parts_of(4, kOps);
  float acc[kLevels][kMaxParts][4];

  // op: constant after unrolling
  __device__ __forceinline__ void add(int op, const XDigits& x, const uint2* B, const float (&start)[4]) {
#pragma unroll
    for (int k = 0; k < kSlices; ++k) {
      const uint2 b = B[k * 32];
#pragma unroll
      for (int p = 0; p < kPairs; ++p) {
        if (!pair_kept(k, p)) continue;
        const int m = k + 2 * p;
        const int pos = op * pairs_of(m) + pairs_before(m, k);
        if (pos % 4 == 0) mma_pair<true>(acc[m][pos / 4], x.f[p], b, start);
        else mma_pair<false>(acc[m][pos / 4], x.f[p], b, start);
      }
    }
  }

  // column c (0, 1) of this lane's row pair: the sum over the levels as an int64 with weight 2^-52 relative to
  // 2^(e_r + f)
  __device__ __forceinline__ long long total(int c) const {
    int L[kLevels];
#pragma unroll
    for (int l = 0; l < kLevels; ++l) {
      unsigned v = 0, parts = 0;
#pragma unroll
      for (int q = 0; q < parts_of(l, kOps); ++q) { v += __float_as_uint(acc[l][q][c]); ++parts; }
      if (l > 0) {
#pragma unroll
        for (int q = 0; q < parts_of(l - 1, kOps); ++q) { v += __float_as_uint(acc[l - 1][q][c + 2]); ++parts; }
      }
      L[l] = (int)(v - parts * kMagicBits);
    }
    return combine(L);
  }
  static __device__ __forceinline__ long long combine(const int (&L)[kLevels]) {
    // Levels 2..6 are added exactly; levels 7 and 8 are summed exactly apart and rounded once to the nearest
    // unit (floor(floor(x / 2^9) + 2^8) / 2^9 = floor((x + 2^17) / 2^18)); flooring them with shifts biases
    // every product by about -1 unit, which the energy-conserving time loop then accumulates.  Levels 2, 3
    // stay below 2^22 for kOps <= 2, so that their sum fits 32 bits.
    const int low = (L[5] + (L[6] >> 9) + 256) >> 9;
    long long t = (long long)(L[4] + low);
    t += (long long)L[3] * 512;
    t += (long long)L[2] * (1 << 18);
    if constexpr (kOps <= 2) t += (long long)(L[0] * 512 + L[1]) * (1 << 27);
    else t += ((long long)L[0] * 512 + L[1]) * (1 << 27);
    return t;
  }
};

// t * 2^s as a binary64, rounded to nearest-even like a conversion of t, with integer operations (the
// scaling by 2^s is exact unless the result is subnormal): the significand is normalised to bit 62 and a
// carry of the rounding moves into the exponent by itself.  rare: the result may lie outside the normal
// range.  (The conversion instruction takes the FP64 pipe for as long as this takes the integer one: with
// it the fused launch took 0.459 instead of 0.433 ms.)
template <bool kNeg>
__device__ __forceinline__ double scaled_double(long long t, int s, bool& rare) {
  const int hi = (int)(t >> 32), sg = hi >> 31;
  const unsigned long long mag = (unsigned long long)((t ^ (long long)sg) - (long long)sg);
  const int lz = __clzll((long long)mag);
  unsigned long long m = mag << ((lz - 1) & 63);
  m += 0x1FFULL + ((m >> 10) & 1ULL);
  const int be = s - lz + (1023 + 62);            // biased exponent - 1 (t != 0)
  const unsigned blo = (unsigned)(m >> 10), bhi = (unsigned)(m >> 42) + ((unsigned)be << 20);
  const unsigned sgn = (kNeg ? ~(unsigned)hi : (unsigned)hi) & 0x80000000u;
  rare |= (unsigned)be > 2044u;
  return __hiloint2double((int)(lz == 64 ? 0u : bhi | sgn), (int)blo);
}

// kN of them with one branch for the rare ones (one branch each: 0.433 instead of 0.415 ms)
template <int kN, bool kNeg>
__device__ __forceinline__ void scaled_doubles(const long long (&t)[kN], const int (&s)[kN], double (&y)[kN]) {
  bool rare = false;
#pragma unroll
  for (int j = 0; j < kN; ++j) y[j] = scaled_double<kNeg>(t[j], s[j], rare);
  if (rare) {
#pragma unroll
    for (int j = 0; j < kN; ++j) y[j] = int_to_double_scaled_slow(kNeg ? -t[j] : t[j], s[j]);
  }
}

// Bulk global -> shared copies by the TMA engine (cp.async.bulk), completing on an mbarrier
// in shared memory: one thread arms the barrier with the byte count and issues the copies;
// every consumer waits on the barrier's phase.  Addresses and sizes are multiples of 16 bytes.
__device__ __forceinline__ unsigned smem_addr(const void* p) { return (unsigned)__cvta_generic_to_shared(p); }

__device__ __forceinline__ void mbar_init(uint64_t* bar, unsigned count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;\n" ::"r"(smem_addr(bar)), "r"(count) : "memory");
}
// the barrier initialisation visible to the TMA engine before its first use
__device__ __forceinline__ void mbar_fence_init() { asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory"); }

// shared memory that the warp read through ordinary loads may now be overwritten by the TMA engine
__device__ __forceinline__ void fence_proxy_async() { asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory"); }

__device__ __forceinline__ void mbar_expect_tx(uint64_t* bar, unsigned bytes) {
  asm volatile("{\n .reg .b64 st;\n mbarrier.arrive.expect_tx.release.cta.shared::cta.b64 st, [%0], %1;\n}\n"
               ::"r"(smem_addr(bar)), "r"(bytes) : "memory");
}

__device__ __forceinline__ void bulk_g2s(void* smem, const void* gmem, unsigned bytes, uint64_t* bar) {
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];\n"
               ::"r"(smem_addr(smem)), "l"(gmem), "r"(bytes), "r"(smem_addr(bar)) : "memory");
}

// wait until the barrier has completed the phase with this parity; bounded: after about
// 2^24 polls (tens of ms) it records SBFWI_ETIMEOUT in *status and gives up
__device__ __forceinline__ bool mbar_wait(uint64_t* bar, unsigned parity, int* status) {
  const unsigned a = smem_addr(bar);
  for (int it = 0; it < (1 << 24); ++it) {
    unsigned done;
    asm volatile("{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}\n"
                 : "=r"(done) : "r"(a), "r"(parity) : "memory");
    if (done) return true;
  }
  if (status) atomicCAS(status, 0, -4 /* SBFWI_ETIMEOUT */);
  return false;
}

}  // namespace tc

// kernel arguments of the operator slicing and the element step (both tile shapes)
struct SliceArgs {
  int nb, n;
  int64_t E;
  const double* mats;     // [E][n][3][nb][nb]
  const double* rt;       // [E][2][nb][nb]
  unsigned char* ops;     // [E][3 n + 2] operator blocks (tc::OpBlock)
};

struct ElemTcArgs {
  int nb, n;
  int64_t E;
  double a0, a1, a2, c1, c2, dt;
  const unsigned char* ops;
  const int32_t* dofs;
  TcLaunch l;
};

// up to this many elements per SM a launch is short of warps rather than of bandwidth (tc_launch_tiles, tc_state)
constexpr int kFewElements = 13;

// elements padded to 21..32 boundary nodes (tc2.cu)
constexpr int kTwoTileMinNb = 21;
int tc2_prepare(Model& md, cudaStream_t st);
void tc2_element_launch(const ElemTcArgs& a, bool avg_accel, cudaStream_t st);
// one or two shots, one tile (tc_small.cu)
constexpr int kFewShots = 2;
int tc_small_prepare();
void tc_small_launch(const ElemTcArgs& a, bool avg_accel, cudaStream_t st);

}  // namespace sbfwi
