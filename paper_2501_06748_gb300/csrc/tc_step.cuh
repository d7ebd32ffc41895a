// The tensor-core element kernels, for one or two 16-row tiles (kRT): operators of up to 16
// or 32 boundary nodes, up to 8 shots, one warp per element.  Included by tc.cu (kRT = 1)
// and tc2.cu (kRT = 2); the splitting and the products are in tc_digits.cuh.
#pragma once
#include <cstdint>
#include <type_traits>

#include "internal.h"
#include "prof.h"
#include "sync.cuh"
#include "tc_digits.cuh"

namespace sbfwi {

namespace tc {

// One operator in memory: the digits' B fragments [n-tile][k-tile][digit][lane] (uint2), then
// the row exponents; one contiguous block, so that one bulk copy brings it in.  An element's
// operators lie in a row: P_i, Q_i, H_i of radial points 0..n-1, then R, T.
template <int kRT>
struct OpBlock {
  static constexpr int kRows = kTile * kRT;
  static constexpr int kTileFrags = kSlices * 32;                        // uint2 per 8 x 16 tile
  static constexpr int kFragBytes = 2 * kRT * kRT * kTileFrags * 8;
  static constexpr int kBytes = kFragBytes + kRows * 4;
};

// Operator slots per warp, warps (elements) per block and blocks per SM.  Shared memory taken by
// the slots is lost to L1, which joins the two rows of a lane in the nodal fields, and deeper
// rings pay only where few warps share an SM.  Two tiles: 12 KB an operator, so 3 slots and 6
// warps per SM (0.72 ms on the 16^3 cube of n_b 26, 8 shots; 4 slots and 4 warps 0.89 ms).
// One tile: kDeep false for many elements, true (one warp per block, so that the last elements
// spread over the SMs) for few; see tc_launch_tiles for the line between them.
template <int kRT, bool kDeep>
struct Shape {
  static constexpr int kSlots = kRT == 1 && kDeep ? 4 : 3;
  static constexpr int kWarps = kRT == 1 ? (kDeep ? 1 : 4) : 2;
  static constexpr int kBlocks = kRT == 1 ? (kDeep ? 16 : 4) : 3;
};

template <int kRT, int kSlots>
struct __align__(16) WarpSmem {
  unsigned char op[kSlots][OpBlock<kRT>::kBytes];
  uint64_t bar[kSlots + (kSlots & 1)];
};

// A warp's ring of operator slots.  fetch, init: lane 0.
template <int kRT, int kSlots>
struct Ring {
  using Op = OpBlock<kRT>;
  WarpSmem<kRT, kSlots>& W;
  const unsigned char* ops;   // the element's operators
  int n, item, end;           // next item to be read, end of the items
  int slot = 0;               // its slot
  unsigned parity = 0;        // of the ring's current round

  __device__ __forceinline__ Ring(WarpSmem<kRT, kSlots>& w, const unsigned char* o, int n_, int first, int last)
      : W(w), ops(o), n(n_), item(first), end(last) {}
  __device__ __forceinline__ void fetch(int k, int s) {
    const int j = k - n;
    const int blk = j < 0 ? -3 * j - 1 : 3 * (j >> 1) + (j & 1);
    mbar_expect_tx(&W.bar[s], Op::kBytes);
    bulk_g2s(W.op[s], ops + (unsigned)blk * (unsigned)Op::kBytes, Op::kBytes, &W.bar[s]);
  }
  __device__ __forceinline__ void start() {
#pragma unroll
    for (int s = 0; s < kSlots; ++s) mbar_init(&W.bar[s], 1);
    mbar_fence_init();
#pragma unroll
    for (int s = 0; s < kSlots; ++s)
      if (item + s < end) fetch(item + s, s);
  }
  __device__ __forceinline__ int slot_after(int d) const { const int s = slot + d; return s >= kSlots ? s - kSlots : s; }
  __device__ __forceinline__ void wait(int s, int* status) { mbar_wait(&W.bar[s], s < slot ? parity ^ 1u : parity, status); }
  __device__ __forceinline__ const uint2* frags(int s) const { return reinterpret_cast<const uint2*>(W.op[s]); }
  __device__ __forceinline__ const int* exps(int s) const { return reinterpret_cast<const int*>(W.op[s] + Op::kFragBytes); }
  // the warp has read the next kCnt items: refill their slots
  template <int kCnt>
  __device__ __forceinline__ void release(int lane) {
    __syncwarp();
    if (lane == 0) {
      fence_proxy_async();                    // the warp's reads of the slots come before the copies
#pragma unroll
      for (int d = 0; d < kCnt; ++d)
        if (item + kSlots + d < end) fetch(item + kSlots + d, slot_after(d));
    }
    item += kCnt;
    slot += kCnt;
    if (slot >= kSlots) { slot -= kSlots; parity ^= 1u; }
  }
};

// y = A x (kNeg: -y) over kOps operands of kRT k-tiles each: operator digits at b0 (and b1), row
// exponents rexp (of slot 0's operator), the operands' digits x at one common column exponent f.
// last() runs once the digits are read; put(j, y_j, y_{j+1}) takes the lane's results in pairs.
template <int kRT, int kOps, bool kNeg, class Last, class Put>
__device__ __forceinline__ void product(const uint2* b0, const uint2* b1, const int* rexp, const XDigits* x, int f, int lane,
                                        const float (&start)[4], Last last, Put put) {
  constexpr int kTile2 = OpBlock<kRT>::kTileFrags;
  int2 er[2 * kRT];
#pragma unroll
  for (int nt = 0; nt < 2 * kRT; ++nt) er[nt] = *reinterpret_cast<const int2*>(rexp + nt * 8 + 2 * (lane & 3));
#pragma unroll
  for (int nt = 0; nt < 2 * kRT; ++nt) {
    LevelSums<kOps * kRT> sums;
#pragma unroll
    for (int k = 0; k < kRT; ++k) sums.add(k, x[k], b0 + (nt * kRT + k) * kTile2 + lane, start);
    if (kOps > 1) {
#pragma unroll
      for (int k = 0; k < kRT; ++k) sums.add(kRT + k, x[kRT + k], b1 + (nt * kRT + k) * kTile2 + lane, start);
    }
    if (nt == 2 * kRT - 1) last();
    const long long tt[2] = {sums.total(0), sums.total(1)};
    const int sc[2] = {er[nt].x + f - 52, er[nt].y + f - 52};
    double y[2];
    scaled_doubles<2, kNeg>(tt, sc, y);
    put(2 * nt, y[0], y[1]);
  }
}

// This lane's rows 16 r + {2t, 2t+1, 2t+8, 2t+9}, shot g, of the interior state and of nodal fields.
// The interior state of the tensor-core kernels (v, z, q and the gradient accumulators) is kept either
// in whole tiles (kTiles, internal.h): rows and shots beyond n_b and B stay zero, so a lane's two
// neighbouring rows are one 16-byte access at a constant offset, without a bounds check, and a
// warp's are one contiguous range; or as the nodal fields are, [row][shot].
template <int kRT, bool kTiles>
struct LaneRows {
  static constexpr int kV = 4 * kRT;
  int t2, B;
  unsigned o0, p0;            // offsets of the lane's first row in a nodal field and in the state of a point
  bool ok[kV];
  __device__ __forceinline__ LaneRows(int lane, int nb, int b) : t2(2 * (lane & 3)), B(b) {
    const int g = lane >> 2;
    o0 = (unsigned)(t2 * B + g);
    p0 = kTiles ? (unsigned)(t2 * kCols + 2 * g) : o0;
#pragma unroll
    for (int j = 0; j < kV; ++j) ok[j] = row(j) < nb && g < B;
  }
  static __device__ __forceinline__ constexpr int rel(int j) { return (j >> 2) * kTile + ((j >> 1) & 1) * 8 + (j & 1); }
  __device__ __forceinline__ int row(int j) const { return t2 + rel(j); }
  __device__ __forceinline__ unsigned off(int j) const { return o0 + (unsigned)(rel(j) * B); }
  // p: the lane's place in the state of a radial point
  __device__ __forceinline__ void load(const double* p, double (&x)[kV]) const {
#pragma unroll
    for (int j = 0; j < kV; j += 2) {
      if (kTiles) {
        const double2 d = *reinterpret_cast<const double2*>(p + rel(j) * kCols);
        x[j] = d.x;
        x[j + 1] = d.y;
      } else {
        x[j] = ok[j] ? p[rel(j) * B] : 0.0;
        x[j + 1] = ok[j + 1] ? p[rel(j + 1) * B] : 0.0;
      }
    }
  }
  __device__ __forceinline__ void store(double* p, int j, double x0, double x1) const {              // rows of j, j + 1
    if (kTiles) {
      *reinterpret_cast<double2*>(p + rel(j) * kCols) = make_double2(x0, x1);
    } else {
      if (ok[j]) p[rel(j) * B] = x0;
      if (ok[j + 1]) p[rel(j + 1) * B] = x1;
    }
  }
};

}  // namespace tc

// one warp per operator
template <int kRT>
__global__ void slice_operators_kernel(SliceArgs a) {
  using namespace tc;
  using Op = OpBlock<kRT>;
  const int64_t w = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
  const int nb = a.nb, n = a.n, nop = 3 * n + 2;
  const int64_t nn = (int64_t)nb * nb;
  if (w >= a.E * nop) return;
  const int64_t e = w / nop;
  const int b = (int)(w - e * nop);
  const double* h = b < 3 * n ? a.mats + (e * 3 * n + b) * nn : a.rt + (e * 2 + (b - 3 * n)) * nn;
  unsigned char* blk = a.ops + w * Op::kBytes;
  uint2* out = reinterpret_cast<uint2*>(blk);
  int* eout = reinterpret_cast<int*>(blk + Op::kFragBytes);
  auto val = [&](const double* m, int r, int c) { return (r < nb && c < nb) ? m[(int64_t)r * nb + c] : 0.0; };
  auto row_exp = [&](const double* m) {            // lane r < kRows owns row r
    int ex = -1100;
    if (lane < Op::kRows)
      for (int c = 0; c < nb; ++c) ex = max(ex, exp_bound(val(m, lane, c)));
    return ex;
  };
  // P or Q of a radial point: joint row exponents with the balancing power a
  const int which = b < 3 * n ? b % 3 : 2;
  int er, shift = 0;        // this operator's digits are taken at row exponent + shift
  if (which < 2) {
    const double* hP = which == 0 ? h : h - nn;
    const int eP = row_exp(hP), eQ = row_exp(hP + nn);
    int mP = eP, mQ = eQ;
    for (int off = 16; off > 0; off >>= 1) {
      mP = max(mP, __shfl_xor_sync(0xffffffffu, mP, off));
      mQ = max(mQ, __shfl_xor_sync(0xffffffffu, mQ, off));
    }
    const int bal = (mP > -1100 && mQ > -1100) ? mQ - mP : 0;
    er = max(eP, eQ > -1100 ? eQ - bal : -1100);
    shift = which == 0 ? 0 : bal;
    if (which == 1 && lane < Op::kRows) eout[lane] = lane == 0 ? bal : 0;
  } else {
    er = row_exp(h);
  }
  if (which != 1 && lane < Op::kRows) eout[lane] = er > -1100 ? er : 0;
  for (int nt = 0; nt < 2 * kRT; ++nt) {
    const int ex = __shfl_sync(0xffffffffu, er, nt * 8 + g) + shift;
    for (int kt = 0; kt < kRT; ++kt) {
      unsigned short dg[4][kSlices];               // columns 2t, 2t+1, 2t+8, 2t+9 of row g
#pragma unroll
      for (int j = 0; j < 4; ++j)
        digits(to_fixed(val(h, nt * 8 + g, kt * kTile + 2 * t + (j & 1) + (j >> 1) * 8), ex), dg[j]);
#pragma unroll
      for (int k = 0; k < kSlices; ++k)
        out[((nt * kRT + kt) * kSlices + k) * 32 + lane] =
            make_uint2(pack_digits(dg[0][k], dg[1][k]), pack_digits(dg[2][k], dg[3][k]));
    }
  }
}

// One warp per element.  The operators are brought into a ring of shared-memory slots by bulk
// copies on mbarriers, one per operator, in the order of use (H_{n-1}..H_0, then P_0, Q_0, ..,
// P_{n-1}, Q_{n-1}, R, T); a slot is refilled as soon as its last digits are read, so the
// copies of kSlots operators are in flight ahead of the products, across the turn of the
// sweeps.  The state of a radial point is loaded before its product.
template <int kRT, bool kDeep, bool kTiles, bool kAvgAccel>
__global__ void __launch_bounds__(32 * tc::Shape<kRT, kDeep>::kWarps, tc::Shape<kRT, kDeep>::kBlocks)
element_step_tc_kernel(ElemTcArgs a) {
  using namespace tc;
  constexpr int kSlots = Shape<kRT, kDeep>::kSlots;
  constexpr int kV = 4 * kRT;                 // values per lane
  extern __shared__ __align__(16) unsigned char tc_smem[];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, g = lane >> 2;
  const int64_t idx = (int64_t)blockIdx.x * Shape<kRT, kDeep>::kWarps + warp;
  if (idx >= a.l.n_elems) return;               // whole warp leaves together
  const int64_t e = a.l.elems ? (int64_t)a.l.elems[idx] : idx;
  const int nb = a.nb, n = a.n, B = a.l.B;
  const int per = nb * B;
  Ring<kRT, kSlots> ring(reinterpret_cast<WarpSmem<kRT, kSlots>*>(tc_smem)[warp],
                         a.ops + e * (3 * n + 2) * (int64_t)OpBlock<kRT>::kBytes, n, a.l.do_down ? 0 : n,
                         a.l.do_up ? 3 * n + 2 : n);
  if (lane == 0) ring.start();                // constant operators
  __syncwarp();
  grid_dependency_wait();
  const LaneRows<kRT, kTiles> rows(lane, nb, B);
  const int kT = kTiles ? kTile * kRT * kCols : per;          // the state of a radial point
  const int64_t tile = idx * (int64_t)n * kT + rows.p0;       // the lane's place in that of point 0
  const float start[4] = {kMagicF, kMagicF, kMagicF, kMagicF};

  double x[kV];       // the operand of the next product
  if (a.l.do_down) {
#pragma unroll
    for (int j = 0; j < kV; ++j) x[j] = rows.ok[j] ? a.l.ub[(int64_t)a.dofs[e * nb + rows.row(j)] * B + g] : 0.0;
    const bool grad = a.l.grad != nullptr;
    for (int i = n - 1; i >= 0; --i) {
      // the state of this radial point, loaded ahead of the product
      const int64_t p = tile + i * kT;
      const int64_t o = e * (int64_t)n * per + (unsigned)(i * per);
      double zo[kV], vo[kV], qo[kV], fw[kV], gr[kV];
      rows.load(a.l.q + p, qo);
      rows.load(a.l.v + p, vo);
      rows.load(a.l.z + p, zo);
      if (grad) {
        rows.load(a.l.grad + p, gr);
#pragma unroll
        for (int j = 0; j < kV; ++j) fw[j] = rows.ok[j] ? a.l.fwd_int[o + rows.off(j)] : 0.0;
      }
      int adj;
      const int E = column_scale<kV>(x, adj);
      XDigits d[kRT];
#pragma unroll
      for (int r = 0; r < kRT; ++r) split_rows(x + 4 * r, E, d[r]);
      const int s0 = ring.slot;
      ring.wait(s0, a.l.status);
      product<kRT, 1, false>(
          ring.frags(s0), nullptr, ring.exps(s0), d, E - 1022 - adj, lane, start, [&] { ring.template release<1>(lane); },
          [&](int j0, double h0, double h1) {
            double zs[2], vs[2], gs[2];
#pragma unroll
            for (int c = 0; c < 2; ++c) {
              const int j = j0 + c;
              const double u_new = qo[j] - (c ? h1 : h0);
              const double uddn = fma(a.a0, u_new, -vo[j]);
              const double udn = fma(a.c2, uddn, zo[j]);
              // the interior displacement is not kept: the predictor v carries it
              // the interior u', u'' are not kept either: the Newmark update needs only
              // z = u' + dt (1 - gamma) u'' of the old state, the same value the update
              // would form from u' and u'' (same rounding)
              // average acceleration (beta = 1/4, gamma = 1/2): z' = z + dt u''_new and the new
              // predictor a0 u_new + a1 u'_new + u''_new equals v + a1 z' (one FMA instead of two)
              if (kAvgAccel) {
                zs[c] = fma(a.dt, uddn, zo[j]);
                vs[c] = fma(a.a1, zs[c], vo[j]);
              } else {
                zs[c] = fma(a.c1, uddn, udn);
                vs[c] = fma(a.a0, u_new, fma(a.a1, udn, a.a2 * uddn));
              }
              if (a.l.store_int && rows.ok[j]) a.l.store_int[o + rows.off(j)] = udn;
              if (grad) gs[c] = fma(fw[j], udn, gr[j]);    // dt applied at the end
              if (a.l.u_out && rows.ok[j]) a.l.u_out[o + rows.off(j)] = u_new;
              x[j] = u_new;                                // zero beyond n_b and B: the operator's rows and q are
            }
            rows.store(a.l.z + p, j0, zs[0], zs[1]);
            rows.store(a.l.v + p, j0, vs[0], vs[1]);
            if (grad) rows.store(a.l.grad + p, j0, gs[0], gs[1]);
          });
    }
  }
  if (!a.l.do_up) return;
  __syncwarp();
  // forward sweep: q_i = -(P_i v_i + Q_i q_{i-1}), as one product -[P | Q 2^-a][v ; q 2^a]: joint
  // row exponents in P's exponent slot, a in Q's
  double v[kV];
  rows.load(a.l.v + tile, v);
#pragma unroll
  for (int j = 0; j < kV; ++j) x[j] = 0.0;    // q of the previous radial point
  for (int i = 0; i < n; ++i) {
    const int64_t p = tile + i * kT;
    double vnext[kV];
    if (i + 1 < n) rows.load(a.l.v + p + kT, vnext);
    const int s0 = ring.slot, s1 = ring.slot_after(1);
    ring.wait(s0, a.l.status);
    ring.wait(s1, a.l.status);
    const int bal = *ring.exps(s1);
    int adj, Eq;
    const int E = column_scale2<kV>(v, x, bal, adj, Eq);
    XDigits d[2 * kRT];
#pragma unroll
    for (int r = 0; r < kRT; ++r) split_rows(v + 4 * r, E, d[r]);
#pragma unroll
    for (int r = 0; r < kRT; ++r) split_rows(x + 4 * r, Eq, d[kRT + r]);
    product<kRT, 2, true>(
        ring.frags(s0), ring.frags(s1), ring.exps(s0), d, E - 1022 - adj, lane, start,
        [&] { ring.template release<2>(lane); },
        [&](int j0, double q0, double q1) {
          rows.store(a.l.q + p, j0, q0, q1);
          x[j0] = q0;
          x[j0 + 1] = q1;
        });
#pragma unroll
    for (int j = 0; j < kV; ++j) v[j] = vnext[j];
  }
  // effective source: f_hat = R q_{n-1} + T v_n, v_n the predictor of the boundary state
#pragma unroll
  for (int j = 0; j < kV; ++j) {
    v[j] = 0.0;
    if (rows.ok[j]) {
      const int64_t gi = (int64_t)a.dofs[e * nb + rows.row(j)] * B + g;
      v[j] = fma(a.a0, a.l.ub[gi], fma(a.a1, a.l.udb[gi], a.a2 * a.l.uddb[gi]));
    }
  }
  double f[kV];
#pragma unroll
  for (int k = 0; k < 2; ++k) {               // R q, then T v
    double* y = k ? v : x;
    int adj;
    const int E = column_scale<kV>(k ? v : x, adj);
    XDigits d[kRT];
#pragma unroll
    for (int r = 0; r < kRT; ++r) split_rows(y + 4 * r, E, d[r]);
    const int s = ring.slot_after(k);
    ring.wait(s, a.l.status);
    product<kRT, 1, false>(ring.frags(s), nullptr, ring.exps(s), d, E - 1022 - adj, lane, start, [] {},
                           [&](int j0, double y0, double y1) {
                             f[j0] = k ? f[j0] + y0 : y0;
                             f[j0 + 1] = k ? f[j0 + 1] + y1 : y1;
                           });
  }
#pragma unroll
  for (int j = 0; j < kV; ++j)
    if (rows.ok[j]) a.l.fhat[(e * nb + rows.row(j)) * B + g] = f[j];
}

// host side: the digits of every element's operators, and the launch
template <int kRT, bool kDeep>
constexpr int tc_block_smem() {
  using S = tc::Shape<kRT, kDeep>;
  return (int)sizeof(tc::WarpSmem<kRT, S::kSlots>) * S::kWarps;
}

template <int kRT>
int tc_prepare_tiles(Model& md, DevBuf& ops, cudaStream_t st) {
  using namespace tc;
  const int64_t warps = md.E * (3 * (int64_t)md.n + 2);
  SBFWI_CUDA(ops.alloc((size_t)warps * OpBlock<kRT>::kBytes));
  SliceArgs a;
  a.nb = md.nb; a.n = md.n; a.E = md.E;
  a.mats = md.mats.as<double>(); a.rt = md.rt.as<double>();
  a.ops = ops.as<unsigned char>();
  slice_operators_kernel<kRT><<<(unsigned)((warps * 32 + 255) / 256), 256, 0, st>>>(a);
  profiler().count(kPhaseSetup);
  SBFWI_CUDA(cudaGetLastError());
  // the slots need more than the default 48 KiB
  for (const void* f : {(const void*)element_step_tc_kernel<kRT, false, true, true>, (const void*)element_step_tc_kernel<kRT, false, true, false>,
                        (const void*)element_step_tc_kernel<kRT, false, false, true>, (const void*)element_step_tc_kernel<kRT, false, false, false>})
    SBFWI_CUDA(cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, tc_block_smem<kRT, false>()));
  return SBFWI_OK;
}

template <int kRT, bool kDeep>
void tc_launch_shape(const ElemTcArgs& a, bool avg_accel, cudaStream_t st) {
  using S = tc::Shape<kRT, kDeep>;
  const unsigned blocks = (unsigned)((a.l.n_elems + S::kWarps - 1) / S::kWarps);
  auto launch = [&](auto kernel) { launch_next(kernel, blocks, 32 * S::kWarps, tc_block_smem<kRT, kDeep>(), st, a); };
  if (a.l.tiles) avg_accel ? launch(element_step_tc_kernel<kRT, kDeep, true, true>) : launch(element_step_tc_kernel<kRT, kDeep, true, false>);
  else avg_accel ? launch(element_step_tc_kernel<kRT, kDeep, false, true>) : launch(element_step_tc_kernel<kRT, kDeep, false, false>);
}

// One tile: the deep ring up to 13 elements per SM.  Fused launches, shallow | deep, n_b 16, 8 shots, ms:
// 3.8 elements per SM (N_r 16) 0.061 | 0.055, 6.7 (N_r 32) 0.142 | 0.130, 10.5 0.177 | 0.173,
// 12.7 0.215 | 0.210, 15.2 0.224 | 0.240, 20.6 0.348 | 0.371, 27 0.394 | 0.432.
template <int kRT>
void tc_launch_tiles(const ElemTcArgs& a, bool avg_accel, cudaStream_t st) {
  if constexpr (kRT == 1) {
    if (a.l.n_elems <= kFewElements * (int64_t)a.l.sms) return tc_launch_shape<1, true>(a, avg_accel, st);
  }
  tc_launch_shape<kRT, false>(a, avg_accel, st);
}

}  // namespace sbfwi
