// FP64-accurate element operators on the FP16 tensor cores.
//
// GB300 executes FP64 at ~1.2 TFLOP/s but FP16 mma.sync at ~600 TFLOP/s.  The
// per-step element work is three n_b x n_b matrix products with B shots per radial
// point (q_i = -(P_i v_i + Q_i q_{i-1}), u_i = q_i - H_i u_{i+1}, f_hat = R q_{n-1} + T v_n),
// so it runs here as an error-free splitting of the FP64 operands into FP16 digits
// (the splitting idea of Ozaki, Ogita, Oishi and Rump, "Error-free transformations of
// matrix multiplication", Numer. Algorithms 59 (2012)):
//
//  * every row r of a matrix A is scaled by 2^(53 - e_r), |A[r][.]| < 2^e_r, and
//    rounded to an integer of at most 53 bits; every column (shot) of a vector x the
//    same with its own exponent f; P v + Q q is one product of [P | Q 2^-a] and
//    [v ; q 2^a] with a per-point balancing power a (a shared exponent without it
//    loses ~1e-12 relative near the scaling centre, where |P| << |Q|), H u, R q and
//    T v are scaled on their own;
//  * each integer is written in six balanced base-512 digits (|digit| <= 257, exact
//    in FP16): A_int = sum_k a_k 2^(9(6-k)), x_int = sum_l x_l 2^(9(6-l));
//  * the digit products of one significance level L = k + l are summed by
//    mma.sync.m16n8k16 (FP16 in, FP32 accumulate) into one accumulator per level;
//    every partial sum is an integer below 2^24, so the accumulation is exact;
//  * levels L = 2..8 are kept (the dropped ones weigh < 2^-57 of the scale), turned
//    back into integers, summed in int64 with their weights 2^(9(8-L)), the two lowest
//    levels rounded once to the nearest unit, and converted once to FP64:
//    A x ~ 2^(e_r + f - 52) * T'.
//
// The splitting of the vectors and the recombination are integer work; what stays on
// the FP64 pipe is the conversion of each result and the Newmark arithmetic.
// Shapes: n_b <= 16 (padded to the 16 rows/columns of one m16n8k16 tile) and B <= 8
// shots (padded to its 8 columns); one warp per element.  The joint product sums two
// k-tiles into each level: at most 12 digit products of <= 257^2 times 16 terms,
// 1.3e7 < 2^24, still exact in FP32.
#include <cstdint>
#include <type_traits>
#include <cuda_fp16.h>

#include "internal.h"
#include "prof.h"
#include "tc_digits.cuh"

namespace sbfwi {

// ---------------------------------------------------------------------------
// set-up: slices of the per-step operators in mma fragment layout
// ---------------------------------------------------------------------------
// Operators per element and radial point i: P_i, Q_i, H_i (16 x 16 each after
// padding); per element R and T.  Each is stored as two n-tiles of kSlices B fragments (32
// lanes x uint2, see the shot-major product in tc_digits.cuh) with 16 row exponents.
//
// P_i v_i + Q_i q_{i-1} is formed as ONE product [P_i | Q_i 2^-a][v_i ; q_{i-1} 2^a]
// with shared row exponents (over both halves) and a shared column exponent, where the
// balancing power a_i = e(Q_i) - e(P_i) of the two blocks' largest entries brings them
// to the same scale (P ~ 1e-4 and Q ~ 0.5 near the scaling centre, and q ~ |P| v, so
// q 2^a ~ v).  Without the balancing a shared exponent would cost the smaller block a
// dozen bits.  P's exponent slot holds the joint row exponents, Q's slot holds a_i in
// its first entry.  H, R and T are scaled on their own.

__global__ void slice_operators_kernel(SliceArgs a) {
  using namespace tc;
  // one warp per operator: warps 0..E*n*3-1 are (e, i, P|Q|H), then E*2 warps of (e, R|T)
  const int64_t w = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
  const int nb = a.nb, n = a.n;
  const int64_t nn = (int64_t)nb * nb;
  const int64_t nmat = a.E * n * 3;
  if (w >= nmat + a.E * 2) return;
  const double* h;
  uint2* out;
  int* eout;
  if (w < nmat) {
    h = a.mats + w * nn;
    out = reinterpret_cast<uint2*>(a.frag + w * kSlices * 32);
    eout = a.exps + w * 16;
  } else {
    const int64_t k = w - nmat;
    h = a.rt + k * nn;
    out = reinterpret_cast<uint2*>(a.frag_rt + k * kSlices * 32);
    eout = a.exps_rt + k * 16;
  }
  auto val = [&](int r, int c) { return (r < nb && c < nb) ? h[(int64_t)r * nb + c] : 0.0; };
  int er = -1100;           // lanes 0..15 own one row each
  if (lane < 16)
    for (int c = 0; c < nb; ++c) er = max(er, exp_bound(val(lane, c)));
  // P or Q of a radial point: joint row exponents with the balancing power a
  const int which = w < nmat ? (int)(w % 3) : 2;
  int shift = 0;            // this operator's digits are taken at row exponent + shift
  if (which < 2) {
    const double* hP = which == 0 ? h : h - nn;
    const double* hQ = hP + nn;
    auto vP = [&](int r, int c) { return (r < nb && c < nb) ? hP[(int64_t)r * nb + c] : 0.0; };
    auto vQ = [&](int r, int c) { return (r < nb && c < nb) ? hQ[(int64_t)r * nb + c] : 0.0; };
    int eP = -1100, eQ = -1100;
    if (lane < 16)
      for (int c = 0; c < nb; ++c) { eP = max(eP, exp_bound(vP(lane, c))); eQ = max(eQ, exp_bound(vQ(lane, c))); }
    int mP = eP, mQ = eQ;
    for (int off = 16; off > 0; off >>= 1) {
      mP = max(mP, __shfl_xor_sync(0xffffffffu, mP, off));
      mQ = max(mQ, __shfl_xor_sync(0xffffffffu, mQ, off));
    }
    const int bal = (mP > -1100 && mQ > -1100) ? mQ - mP : 0;
    er = max(eP, eQ > -1100 ? eQ - bal : -1100);
    shift = which == 0 ? 0 : bal;
    if (which == 1 && lane == 0) eout[0] = bal;
    if (which == 1 && lane > 0 && lane < 16) eout[lane] = 0;
  }
  if (lane < 16 && which != 1) eout[lane] = er;
  const int e_lo = __shfl_sync(0xffffffffu, er, g) + shift, e_hi = __shfl_sync(0xffffffffu, er, g + 8) + shift;
  // fragment entries: (g, 2t), (g, 2t+1), (g+8, 2t), (g+8, 2t+1), then columns + 8
  unsigned short dg[8][kSlices];
#pragma unroll
  for (int j = 0; j < 8; ++j) {
    const int r = g + ((j >> 1) & 1) * 8, c = 2 * t + (j & 1) + (j >> 2) * 8;
    digits(to_fixed(val(r, c), r < 8 ? e_lo : e_hi), dg[j]);
  }
  // B fragments of the shot-major product: n-tile 0 holds rows 0..7, n-tile 1 rows 8..15
#pragma unroll
  for (int k = 0; k < kSlices; ++k) {
    out[k * 32 + lane] = make_uint2(pack_digits(dg[0][k], dg[1][k]), pack_digits(dg[4][k], dg[5][k]));
    out[(kSlices + k) * 32 + lane] = make_uint2(pack_digits(dg[2][k], dg[3][k]), pack_digits(dg[6][k], dg[7][k]));
  }
}

// ---------------------------------------------------------------------------
// element step on the tensor cores (one warp per element)
// ---------------------------------------------------------------------------

namespace tc {

// One pipeline stage: the digit fragments of one or two operators and their row
// exponents, brought in by two bulk copies (fragments, exponents) that complete on the
// stage's mbarrier; lane 0 issues them.
constexpr int kStageFrags = 2 * kSlices * 32;     // uint4
struct WarpSmem {
  uint4 frag[2][kStageFrags];
  int exps[2][32];
  uint64_t bar[2];
};
constexpr int kWarpsPerBlock = 4;

__device__ __forceinline__ void stage_ops(WarpSmem& W, int buf, const uint4* src, const int* sexp, int nops,
                                          int lane) {
  if (lane == 0) {
    const unsigned fb = (unsigned)(nops * kSlices * 32 * sizeof(uint4)), eb = (unsigned)(nops * 16 * sizeof(int));
    fence_proxy_async();                  // the warp's earlier reads of this stage come first
    mbar_expect_tx(&W.bar[buf], fb + eb);
    bulk_g2s(W.frag[buf], src, fb, &W.bar[buf]);
    bulk_g2s(W.exps[buf], sexp, eb, &W.bar[buf]);
  }
}

}  // namespace tc

// One warp per element.  The operator digits of the next radial point are copied to
// shared memory (bulk copies on mbarriers, two stages) while the current point computes,
// and each point's state is loaded before its products, so the memory latency overlaps
// the tensor-core and integer work instead of stalling every radial point.
template <bool kAvgAccel>
__global__ void __launch_bounds__(128, 4) element_step_tc_kernel(ElemTcArgs a) {
  using namespace tc;
  extern __shared__ __align__(16) unsigned char tc_smem[];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
  WarpSmem& W = reinterpret_cast<WarpSmem*>(tc_smem)[warp];
  const int64_t idx = (int64_t)blockIdx.x * kWarpsPerBlock + warp;
  if (idx >= a.n_elems) return;               // whole warp leaves together
  const int64_t e = a.elems ? (int64_t)a.elems[idx] : idx;
  if (lane == 0) {
    mbar_init(&W.bar[0], 1);
    mbar_init(&W.bar[1], 1);
    mbar_fence_init();
  }
  __syncwarp();
  unsigned phase = 0;                         // bit b: parity of stage b's next completion
  auto wait_stage = [&](int b) {
    mbar_wait(&W.bar[b], (phase >> b) & 1u, a.status);
    phase ^= 1u << b;
  };
  const int nb = a.nb, n = a.n, B = a.B;
  const int per = nb * B;
  // this lane's vector entries: shot g, rows 2t, 2t+1, 2t+8, 2t+9
  const int row[4] = {2 * t, 2 * t + 1, 2 * t + 8, 2 * t + 9};
  bool ok[4];
  int off[4];
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    ok[j] = row[j] < nb && g < B;
    off[j] = row[j] * B + g;
  }
  const int64_t base = e * (int64_t)n * per;
  const float start[4] = {kMagicF, kMagicF, kMagicF, kMagicF};

  // y = A x over kOps operands (operator digits A[o] in shared memory, row exponents rexp, the
  // operands' digits x[o] at one common column exponent f); kNeg: -y
  auto apply = [&](auto ops, auto neg, const uint4* A, const XDigits* x, const int* rexp, int f, double (&y)[4]) {
    constexpr int kOps = decltype(ops)::value;
    constexpr bool kNeg = decltype(neg)::value;
#pragma unroll
    for (int nt = 0; nt < 2; ++nt) {
      const uint2* b = reinterpret_cast<const uint2*>(A) + nt * kSlices * 32 + lane;
      LevelSums<kOps> s;
      s.template add<0>(x[0], b, start);
      if constexpr (kOps > 1) s.template add<1>(x[1], b + 2 * kSlices * 32, start);
      const int2 er = *reinterpret_cast<const int2*>(rexp + nt * 8 + 2 * t);
      y[2 * nt] = scaled_double<kNeg>(s.total(0), er.x + f - 52);
      y[2 * nt + 1] = scaled_double<kNeg>(s.total(1), er.y + f - 52);
    }
  };
  // one product y = A x, x split here
  auto apply_one = [&](const uint4* A, const int* rexp, double (&x)[4], double (&y)[4]) {
    int adj;
    const int E = column_scale(x, adj);
    XDigits d[1];
    split_rows(x, E, d[0]);
    apply(std::integral_constant<int, 1>{}, std::false_type{}, A, d, rexp, E - 1022 - adj, y);
  };

  double x[4];        // the operand of the next product
  if (a.do_down) {
    const int64_t hop = (int64_t)3 * kSlices * 32;       // uint4 between radial points
    const uint4* Hsrc = a.frag + ((e * n + (n - 1)) * 3 + 2) * kSlices * 32;
    const int* Hexp = a.exps + ((e * n + (n - 1)) * 3 + 2) * 16;
    stage_ops(W, (n - 1) & 1, Hsrc, Hexp, 1, lane);
#pragma unroll
    for (int j = 0; j < 4; ++j) x[j] = ok[j] ? a.ub[(int64_t)a.dofs[e * nb + row[j]] * B + g] : 0.0;
    for (int i = n - 1; i >= 0; --i) {
      const int buf = i & 1;
      if (i > 0) stage_ops(W, buf ^ 1, Hsrc - (int64_t)(n - i) * hop, Hexp - (int64_t)(n - i) * 48, 1, lane);
      // the state of this radial point, loaded ahead of the product
      double zo[4], vo[4], qo[4], fw[4], gr[4];
      const int64_t oi = base + (int64_t)i * per;
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        zo[j] = ok[j] ? a.ud[oi + off[j]] : 0.0;
        vo[j] = ok[j] ? a.v[oi + off[j]] : 0.0;
        qo[j] = ok[j] ? a.q[oi + off[j]] : 0.0;
        fw[j] = (ok[j] && a.grad_int) ? a.fwd_int[oi + off[j]] : 0.0;
        gr[j] = (ok[j] && a.grad_int) ? a.grad_int[oi + off[j]] : 0.0;
      }
      wait_stage(buf);
      double hu[4];
      apply_one(W.frag[buf], W.exps[buf], x, hu);
      __syncwarp();       // the stage just read may be refilled
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const double u_new = qo[j] - hu[j];
        x[j] = ok[j] ? u_new : 0.0;
        if (ok[j]) {
          const int64_t o = oi + off[j];
          const double uddn = fma(a.a0, u_new, -vo[j]);
          const double udn = fma(a.c2, uddn, zo[j]);
          // the interior displacement is not kept: the predictor v carries it
          // the interior u', u'' are not kept either: the Newmark update needs only
          // z = u' + dt (1 - gamma) u'' of the old state, the same value the update
          // would form from u' and u'' (same rounding)
          // average acceleration (beta = 1/4, gamma = 1/2): z' = z + dt u''_new and the new
          // predictor a0 u_new + a1 u'_new + u''_new equals v + a1 z' (one FMA instead of two)
          if (kAvgAccel) {
            const double zn = fma(a.dt, uddn, zo[j]);
            a.ud[o] = zn;
            a.v[o] = fma(a.a1, zn, vo[j]);
          } else {
            a.ud[o] = fma(a.c1, uddn, udn);
            a.v[o] = fma(a.a0, u_new, fma(a.a1, udn, a.a2 * uddn));
          }
          if (a.store_int) a.store_int[o] = udn;
          if (a.grad_int) a.grad_int[o] = fma(fw[j], udn, gr[j]);    // dt applied at the end
          if (a.u_out) a.u_out[o] = u_new;
        }
      }
    }
  }
  if (!a.do_up) return;
  __syncwarp();
  // forward sweep: q_i = -(P_i v_i + Q_i q_{i-1}); stage i holds P_i and Q_i, stage n R and T
  auto stage_up = [&](int i, int buf) {
    if (i < n) stage_ops(W, buf, a.frag + (e * n + i) * 3 * kSlices * 32, a.exps + (e * n + i) * 3 * 16, 2, lane);
    else stage_ops(W, buf, a.frag_rt + e * 2 * kSlices * 32, a.exps_rt + e * 32, 2, lane);
  };
  stage_up(0, 0);
  double vnext[4];
#pragma unroll
  for (int j = 0; j < 4; ++j) vnext[j] = ok[j] ? a.v[base + off[j]] : 0.0;
#pragma unroll
  for (int j = 0; j < 4; ++j) x[j] = 0.0;     // q of the previous radial point
  for (int i = 0; i < n; ++i) {
    const int buf = i & 1;
    stage_up(i + 1, buf ^ 1);
    const int64_t oi = base + (int64_t)i * per;
    double v[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      v[j] = vnext[j];
      vnext[j] = (i + 1 < n && ok[j]) ? a.v[oi + per + off[j]] : 0.0;
    }
    wait_stage(buf);
    // -[P | Q 2^-a][v ; q 2^a] as one product: P's and Q's digits, joint row exponents in P's
    // exponent slot, a in Q's
    const int bal = W.exps[buf][16];
    int adj;
    const int E = column_scale2(v, x, bal, adj);
    XDigits d[2];
    split_rows(v, E, d[0]);
    split_rows(x, max(E - bal, kMinExp), d[1]);
    double qc[4];
    apply(std::integral_constant<int, 2>{}, std::true_type{}, W.frag[buf], d, W.exps[buf], E - 1022 - adj, qc);
    __syncwarp();         // the stage just read may be refilled
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      if (ok[j]) a.q[oi + off[j]] = qc[j];
      x[j] = ok[j] ? qc[j] : 0.0;
    }
  }
  // effective source: f_hat = R q_{n-1} + T v_n, v_n the predictor of the boundary state
  double vb[4];
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    vb[j] = 0.0;
    if (ok[j]) {
      const int64_t gi = (int64_t)a.dofs[e * nb + row[j]] * B + g;
      vb[j] = fma(a.a0, a.ub[gi], fma(a.a1, a.udb[gi], a.a2 * a.uddb[gi]));
    }
  }
  const int bn = n & 1;
  wait_stage(bn);
  double rq[4], tv[4];
  apply_one(W.frag[bn], W.exps[bn], x, rq);
  apply_one(W.frag[bn] + kSlices * 32, W.exps[bn] + 16, vb, tv);
#pragma unroll
  for (int j = 0; j < 4; ++j)
    if (ok[j]) a.fhat[(e * nb + row[j]) * B + g] = rq[j] + tv[j];
}

// ---------------------------------------------------------------------------
// host helpers
// ---------------------------------------------------------------------------
// Padded n_b 17..20 stays on the FP64 kernel: two 16-row tiles then do 4x the digit work
// of one for at most 1.6x the entries, and on the batching meshes the FP64 kernel was
// faster at n_b = 18 (6.6 s against 8.0 s per step of the p = 3 mesh) while the two-tile
// kernel was faster at n_b = 30 (12.5 s against 21.9 s of the p = 5 mesh).
bool tc_supported(int nb, int B) {
  return (nb <= tc::kTile || (nb >= kTwoTileMinNb && nb <= 2 * tc::kTile)) && B <= tc::kCols;
}
bool tc_available(int nb, int B) { return nb <= 2 * tc::kTile && B <= tc::kCols; }

int tc_prepare(Model& md, cudaStream_t st) {
  using namespace tc;
  if (md.nb > kTile) return tc2_prepare(md, st);
  return tc_prepare_one_tile(md, st);
}

// One-tile digits of every element's operators (their top-left 16 x 16 block; for a mesh
// padded beyond 16 this is the whole operator of its elements with n_b <= 16, whose padded
// rows and columns are zero)
int tc_prepare_one_tile(Model& md, cudaStream_t st) {
  using namespace tc;
  const int nb = md.nb, n = md.n;
  const int64_t E = md.E;
  SBFWI_CUDA(md.tc_frag.alloc(sizeof(uint4) * (size_t)E * n * 3 * kSlices * 32));
  SBFWI_CUDA(md.tc_frag_rt.alloc(sizeof(uint4) * (size_t)E * 2 * kSlices * 32));
  SBFWI_CUDA(md.tc_exps.alloc(sizeof(int) * (size_t)E * n * 3 * 16));
  SBFWI_CUDA(md.tc_exps_rt.alloc(sizeof(int) * (size_t)E * 2 * 16));
  SliceArgs a;
  a.nb = nb; a.n = n; a.E = E;
  a.mats = md.mats.as<double>(); a.rt = md.rt.as<double>();
  a.frag = md.tc_frag.as<uint4>(); a.frag_rt = md.tc_frag_rt.as<uint4>();
  a.exps = md.tc_exps.as<int>(); a.exps_rt = md.tc_exps_rt.as<int>();
  const int64_t warps = E * n * 3 + E * 2;
  slice_operators_kernel<<<(unsigned)((warps * 32 + 255) / 256), 256, 0, st>>>(a);
  profiler().count(kPhaseSetup);
  SBFWI_CUDA(cudaGetLastError());
  // the element kernel's two-stage operator pipeline needs more than the default 48 KiB
  for (const void* f : {(const void*)element_step_tc_kernel<true>, (const void*)element_step_tc_kernel<false>})
    SBFWI_CUDA(cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)(sizeof(WarpSmem) * kWarpsPerBlock)));
  md.tc_ready = true;
  md.tc_one_tile = nb > kTile;
  return SBFWI_OK;
}

int tc_element_launch(const Model& md, int B, int down, int up, double* u, double* ud, double* udd, double* v,
                      const double* ub, const double* udb, const double* uddb, double* q, double* fhat,
                      double* store_int, const double* fwd_int, double* grad_int, double* u_out, cudaStream_t st,
                      const int32_t* elems, int64_t n_elems, int* status) {
  ElemTcArgs a;
  a.nb = md.nb; a.n = md.n; a.B = B; a.E = md.E;
  a.a0 = md.a0; a.a1 = md.a1; a.a2 = md.a2; a.c1 = md.c1; a.c2 = md.c2; a.dt = md.dt;
  a.frag = md.tc_frag.as<uint4>(); a.frag_rt = md.tc_frag_rt.as<uint4>();
  a.exps = md.tc_exps.as<int>(); a.exps_rt = md.tc_exps_rt.as<int>();
  a.dofs = md.dev().dofs.as<int32_t>();
  a.u = u; a.ud = ud; a.udd = udd; a.v = v; a.ub = ub; a.udb = udb; a.uddb = uddb; a.q = q; a.fhat = fhat;
  a.do_down = down; a.do_up = up;
  a.store_int = store_int; a.fwd_int = fwd_int; a.grad_int = grad_int; a.u_out = u_out;
  a.elems = elems; a.n_elems = elems ? n_elems : md.E;
  a.status = status;
  if (a.n_elems == 0) return SBFWI_OK;
  // one 16-row tile: n_b <= 16, or the elements of n_b <= 16 of a mesh padded beyond (the
  // one-tile digits of its operators, prepared by tc_prepare_one_tile)
  if (md.nb > tc::kTile && !md.tc_one_tile) return tc2_element_launch(a, md.a2 == 1.0 && md.c1 == md.c2, st);
  const int smem = (int)(sizeof(tc::WarpSmem) * tc::kWarpsPerBlock);   // attribute set by tc_prepare
  const unsigned blocks = (unsigned)((a.n_elems + tc::kWarpsPerBlock - 1) / tc::kWarpsPerBlock);
  // average acceleration (beta = 1/4, gamma = 1/2): the shorter predictor update
  if (md.a2 == 1.0 && md.c1 == md.c2) element_step_tc_kernel<true><<<blocks, 32 * tc::kWarpsPerBlock, smem, st>>>(a);
  else element_step_tc_kernel<false><<<blocks, 32 * tc::kWarpsPerBlock, smem, st>>>(a);
  return SBFWI_OK;
}

}  // namespace sbfwi
