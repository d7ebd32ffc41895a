// The tensor-core element step for one or two shots (n_b <= 16).  With two shots only a quarter
// of the lanes of the 8-shot kernel hold values, but all of them split and recombine, so the
// time does not fall with the shots.  Here a lane holds one value: lane (s, r) = (lane / 16,
// lane % 16) has row r of shot s, and the 16 rows of the mma are the significance levels of the
// two shots: row L (L + 8 for the second shot) of the A fragment for operator digit k holds
// digit L - k of x, so that the accumulators sum whole levels over k: 12 mma per product instead
// of 28, and a quarter of the conversions.  Digits go to the fragments, and levels to the lanes,
// through the warp's shared memory.  Digits, kept levels and roundings are those of the 8-shot
// kernel, so a shot's results do not depend on the shots beside it.
// Measured (fused launch, 8-shot kernel | this one): 64 x 64 elements, n_b 16, N_r 32, 1 shot 0.369 | 0.222 ms
// (1.2 GB of operators: 5.4 TB/s), 1000 polygons, 6 radial points, 2 shots 30 | 18 us, 16 elements, 8 radial
// points, 1 shot 28 | 18 us.
#include "tc_step.cuh"

namespace sbfwi {

namespace tc {

constexpr int kSmallShots = 2;

// digits of one operand [shot][5 zero rows, digits 0..5, zero rows][4 lanes t: rows 2t, 2t+1, 2t+8, 2t+9]; level
// row g of the fragment for operator digit k reads row kZeroRows + g - k, g 0..7 (level 7 is formed and not kept)
constexpr int kZeroRows = kSlices - 1, kDigitRows = kZeroRows + kTile / 2;
static_assert(kZeroRows + kSlices <= kDigitRows && kZeroRows >= kSlices - 1 && kZeroRows + 7 < kDigitRows,
              "a row for every digit and for every level row that is read");
struct SmallDigits {
  __half d[kSmallShots][kDigitRows][kTile];
};
// levels [shot][level][row], strides chosen against bank conflicts
constexpr int kLevelStride = 24, kShotStride = 8 * kLevelStride + 16;

template <bool kDeep>
struct SmallShape {
  static constexpr int kSlots = kDeep ? 4 : 3;
  static constexpr int kWarps = kDeep ? 1 : 4;
  static constexpr int kBlocks = kDeep ? 16 : 4;
};

template <bool kDeep>
struct __align__(16) SmallSmem {
  WarpSmem<1, SmallShape<kDeep>::kSlots> ring;
  SmallDigits dig[2];
  int lev[2 * kShotStride];
};

// x's digits (column exponent E) to the fragment rows of an operand
__device__ __forceinline__ void put_digits(SmallDigits& D, double x, int E, int s, int row) {
  const uint2 y = biased_fixed(x, E);
  const int at = ((row & 7) >> 1) * 4 + (row >> 3) * 2 + (row & 1);
  // digits 5, 4 | 3, 2 | 1, 0 (low, high half): fields less 256 (digit 0 less 512)
  const unsigned w54 = ((y.x >> 8) & 0x1FFu) | ((y.x >> 1) & 0x01FF0000u) | 0x64006400u;
  const unsigned w32 = (__funnelshift_r(y.x, y.y, 26) & 0x1FFu) | ((y.y << 13) & 0x01FF0000u) | 0x64006400u;
  const unsigned w10 = ((y.y >> 12) & 0x1FFu) | ((y.y >> 5) & 0x03FF0000u) | 0x64006400u;
  const unsigned h[3] = {unbias(w54, 0x65006500u), unbias(w32, 0x65006500u), unbias(w10, 0x66006500u)};
#pragma unroll
  for (int p = 0; p < 3; ++p) {
    D.d[s][kZeroRows + 5 - 2 * p][at] = __ushort_as_half((unsigned short)(h[p] & 0xFFFFu));
    D.d[s][kZeroRows + 4 - 2 * p][at] = __ushort_as_half((unsigned short)(h[p] >> 16));
  }
}

// largest over the 16 lanes of a shot
__device__ __forceinline__ int half_max(int v) {
#pragma unroll
  for (int o = 1; o < 16; o <<= 1) v = max(v, __shfl_xor_sync(0xffffffffu, v, o));
  return v;
}

// (A x)(row, s) of this lane (kNeg: its negative) from the operands' digits in D[0..kOps), the operators' in
// b0 (and b1), er the row's exponent, f the column's; last() runs once the digits are read
template <int kOps, bool kNeg, class Last>
__device__ __forceinline__ double small_product(const SmallDigits* D, int* lev, const uint2* b0, const uint2* b1, int er, int f,
                                                int lane, Last last) {
  const int g = lane >> 2, t = lane & 3;
  constexpr int kPer = kOps == 1 ? 3 : 4, kParts = kOps * kSlices / kPer;      // mma per accumulator: at most four
  const float start[4] = {kMagicF, kMagicF, kMagicF, kMagicF};
  float c[2][kParts][4];
  __syncwarp();
#pragma unroll
  for (int op = 0; op < kOps; ++op) {
    const uint2* b = (op == 0 ? b0 : b1) + lane;
#pragma unroll
    for (int k = 0; k < kSlices; ++k) {
      const uint2 x0 = *reinterpret_cast<const uint2*>(&D[op].d[0][kZeroRows + g - k][4 * t]);
      const uint2 x1 = *reinterpret_cast<const uint2*>(&D[op].d[1][kZeroRows + g - k][4 * t]);
      const uint4 x = make_uint4(x0.x, x1.x, x0.y, x1.y);
      const int pos = op * kSlices + k;
#pragma unroll
      for (int nt = 0; nt < 2; ++nt) {
        if (pos % kPer == 0) mma_pair<true>(c[nt][pos / kPer], x, b[(nt * kSlices + k) * 32], start);
        else mma_pair<false>(c[nt][pos / kPer], x, b[(nt * kSlices + k) * 32], start);
      }
    }
  }
  last();
#pragma unroll
  for (int nt = 0; nt < 2; ++nt)
#pragma unroll
    for (int s = 0; s < kSmallShots; ++s) {
      unsigned v0 = 0, v1 = 0;
#pragma unroll
      for (int q = 0; q < kParts; ++q) {
        v0 += __float_as_uint(c[nt][q][2 * s]);
        v1 += __float_as_uint(c[nt][q][2 * s + 1]);
      }
      *reinterpret_cast<int2*>(lev + s * kShotStride + g * kLevelStride + nt * 8 + 2 * t) =
          make_int2((int)(v0 - kParts * kMagicBits), (int)(v1 - kParts * kMagicBits));
    }
  __syncwarp();
  int L[kLevels];
#pragma unroll
  for (int l = 0; l < kLevels; ++l) L[l] = lev[(lane >> 4) * kShotStride + l * kLevelStride + (lane & 15)];
  const long long tt[1] = {LevelSums<kOps>::combine(L)};
  const int sc[1] = {er + f - 52};
  double y[1];
  scaled_doubles<1, kNeg>(tt, sc, y);
  return y[0];
}

// column_scale and column_scale2 for one value per lane
__device__ __forceinline__ int small_scale(double& x, int& adj) {
  int ex = exp_of_key(half_max(mag_key(x)));
  adj = 0;
  if (__any_sync(0xffffffffu, scale_small(ex))) {
    if (scale_small(ex)) { adj = kScaleBits; x *= 0x1p256; }
    ex = exp_of_key(half_max(mag_key(x)));
  }
  return ex < kMinExp ? 1022 : ex;
}
__device__ __forceinline__ int small_scale2(double (&v)[1], double (&q)[1], int bal, int& adj, int& eq) {
  return joint_scale<1>(v, q, bal, adj, eq,
                        [&] { return half_max(max(exp_of_key(mag_key(v[0])), exp_of_key(mag_key(q[0])) + bal)); });
}

}  // namespace tc

template <bool kDeep, bool kAvgAccel>
__global__ void __launch_bounds__(32 * tc::SmallShape<kDeep>::kWarps, tc::SmallShape<kDeep>::kBlocks)
element_step_small_kernel(ElemTcArgs a) {
  using namespace tc;
  constexpr int kSlots = SmallShape<kDeep>::kSlots;
  extern __shared__ __align__(16) unsigned char tc_smem[];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, s = lane >> 4, row = lane & 15;
  SmallSmem<kDeep>& M = reinterpret_cast<SmallSmem<kDeep>*>(tc_smem)[warp];
  const int64_t idx = (int64_t)blockIdx.x * SmallShape<kDeep>::kWarps + warp;
  if (idx >= a.l.n_elems) return;             // whole warp leaves together
  const int64_t e = a.l.elems ? (int64_t)a.l.elems[idx] : idx;
  const int nb = a.nb, n = a.n, B = a.l.B;
  const int per = nb * B;
  Ring<1, kSlots> ring(M.ring, a.ops + e * (3 * n + 2) * (int64_t)OpBlock<1>::kBytes, n, a.l.do_down ? 0 : n,
                       a.l.do_up ? 3 * n + 2 : n);
  if (lane == 0) ring.start();                // constant operators
  for (int k = lane; k < (int)(sizeof(M.dig) / 4); k += 32) reinterpret_cast<unsigned*>(M.dig)[k] = 0u;
  __syncwarp();
  grid_dependency_wait();
  const bool ok = row < nb && s < B;
  const int64_t at = (int64_t)row * B + s;                    // this lane's place in a radial point
  const int64_t st = idx * (int64_t)n * per + at;             // in the state
  const int64_t fi = e * (int64_t)n * per + at;               // in a nodal field
  double x = 0.0;
  if (a.l.do_down) {
    if (ok) x = a.l.ub[(int64_t)a.dofs[e * nb + row] * B + s];
    const bool grad = a.l.grad != nullptr;
    for (int i = n - 1; i >= 0; --i) {
      const int64_t p = st + i * per, o = fi + i * per;
      double zo = 0.0, vo = 0.0, qo = 0.0, fw = 0.0, gr = 0.0;
      if (ok) {
        qo = a.l.q[p];
        vo = a.l.v[p];
        zo = a.l.z[p];
        if (grad) { gr = a.l.grad[p]; fw = a.l.fwd_int[o]; }
      }
      int adj;
      const int E = small_scale(x, adj);
      put_digits(M.dig[0], x, E, s, row);
      const int s0 = ring.slot;
      ring.wait(s0, a.l.status);
      const int er = ring.exps(s0)[row];
      const double hu = small_product<1, false>(M.dig, M.lev, ring.frags(s0), nullptr, er, E - 1022 - adj, lane,
                                                [&] { ring.template release<1>(lane); });
      // the updates of element_step_tc_kernel
      const double u_new = qo - hu;
      const double uddn = fma(a.a0, u_new, -vo);
      const double udn = fma(a.c2, uddn, zo);
      double zn, vn;
      if (kAvgAccel) {
        zn = fma(a.dt, uddn, zo);
        vn = fma(a.a1, zn, vo);
      } else {
        zn = fma(a.c1, uddn, udn);
        vn = fma(a.a0, u_new, fma(a.a1, udn, a.a2 * uddn));
      }
      if (ok) {
        a.l.z[p] = zn;
        a.l.v[p] = vn;
        if (a.l.store_int) a.l.store_int[o] = udn;
        if (grad) a.l.grad[p] = fma(fw, udn, gr);              // dt applied at the end
        if (a.l.u_out) a.l.u_out[o] = u_new;
      }
      x = u_new;
    }
  }
  if (!a.l.do_up) return;
  x = 0.0;                                                     // q of the previous radial point
  double v = ok ? a.l.v[st] : 0.0;
  for (int i = 0; i < n; ++i) {
    const int64_t p = st + i * per;
    const double vnext = ok && i + 1 < n ? a.l.v[p + per] : 0.0;
    const int s0 = ring.slot, s1 = ring.slot_after(1);
    ring.wait(s0, a.l.status);
    ring.wait(s1, a.l.status);
    const int bal = *ring.exps(s1), er = ring.exps(s0)[row];
    int adj, Eq;
    double vs[1] = {v}, qs[1] = {x};
    const int E = small_scale2(vs, qs, bal, adj, Eq);
    put_digits(M.dig[0], vs[0], E, s, row);
    put_digits(M.dig[1], qs[0], Eq, s, row);
    x = small_product<2, true>(M.dig, M.lev, ring.frags(s0), ring.frags(s1), er, E - 1022 - adj, lane,
                               [&] { ring.template release<2>(lane); });
    if (ok) a.l.q[p] = x;
    v = vnext;
  }
  // effective source: f_hat = R q_{n-1} + T v_n, v_n the predictor of the boundary state
  v = 0.0;
  if (ok) {
    const int64_t gi = (int64_t)a.dofs[e * nb + row] * B + s;
    v = fma(a.a0, a.l.ub[gi], fma(a.a1, a.l.udb[gi], a.a2 * a.l.uddb[gi]));
  }
  double f = 0.0;
#pragma unroll
  for (int k = 0; k < 2; ++k) {                                // R q, then T v
    double& y = k ? v : x;
    int adj;
    const int E = small_scale(y, adj);
    put_digits(M.dig[0], y, E, s, row);
    const int sl = ring.slot_after(k);
    ring.wait(sl, a.l.status);
    const double w = small_product<1, false>(M.dig, M.lev, ring.frags(sl), nullptr, ring.exps(sl)[row], E - 1022 - adj, lane,
                                             [] {});
    f = k ? f + w : w;
  }
  if (ok) a.l.fhat[(e * nb + row) * B + s] = f;
}

int tc_small_prepare() {
  const int smem = (int)sizeof(tc::SmallSmem<false>) * tc::SmallShape<false>::kWarps;
  for (const void* f : {(const void*)element_step_small_kernel<false, true>, (const void*)element_step_small_kernel<false, false>})
    SBFWI_CUDA(cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, smem));
  return SBFWI_OK;
}

template <bool kDeep>
static void small_launch(const ElemTcArgs& a, bool avg_accel, cudaStream_t st) {
  constexpr int kWarps = tc::SmallShape<kDeep>::kWarps;
  const int smem = (int)sizeof(tc::SmallSmem<kDeep>) * kWarps;
  const unsigned blocks = (unsigned)((a.l.n_elems + kWarps - 1) / kWarps);
  if (avg_accel) launch_next(element_step_small_kernel<kDeep, true>, blocks, 32 * kWarps, smem, st, a);
  else launch_next(element_step_small_kernel<kDeep, false>, blocks, 32 * kWarps, smem, st, a);
}

void tc_small_launch(const ElemTcArgs& a, bool avg_accel, cudaStream_t st) {
  if (a.l.n_elems <= kFewElements * (int64_t)a.l.sms) small_launch<true>(a, avg_accel, st);
  else small_launch<false>(a, avg_accel, st);
}

}  // namespace sbfwi
