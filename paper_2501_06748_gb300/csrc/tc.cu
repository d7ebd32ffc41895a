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
//  * each integer is written in six balanced base-512 digits (-256..255, the first one up
//    to 256 = 2^53 / 2^45, exact in FP16): A_int = sum_k a_k 2^(9(6-k)), x_int = sum_l x_l 2^(9(6-l));
//  * the digit products of one significance level L = k + l are summed by
//    mma.sync.m16n8k16 (FP16 in, FP32 accumulate), at most four products of 16 terms per
//    accumulator: every partial sum is an integer of at most 4 x 16 x 256^2 = 2^22, so the accumulation is exact;
//  * levels L = 2..8 are kept (the dropped ones weigh < 2^-57 of the scale), turned
//    back into integers, summed in int64 with their weights 2^(9(8-L)), the two lowest
//    levels rounded once to the nearest unit, and converted once to FP64:
//    A x ~ 2^(e_r + f - 52) * T'.
//
// The splitting of the vectors and the recombination are integer work; what stays on
// the FP64 pipe is the Newmark arithmetic.
// Shapes: n_b <= 16 (padded to 16) and 3 <= B <= 8 shots (padded to 8) here, n_b 21..32 in
// tc2.cu, one or two shots in tc_small.cu; one warp per element.
#include "tc_step.cuh"

namespace sbfwi {

// Operators per element and radial point i: P_i, Q_i, H_i; per element R and T.
//
// P_i v_i + Q_i q_{i-1} is formed as ONE product [P_i | Q_i 2^-a][v_i ; q_{i-1} 2^a]
// with shared row exponents (over both halves) and a shared column exponent, where the
// balancing power a_i = e(Q_i) - e(P_i) of the two blocks' largest entries brings them
// to the same scale (P ~ 1e-4 and Q ~ 0.5 near the scaling centre, and q ~ |P| v, so
// q 2^a ~ v).  Without the balancing a shared exponent would cost the smaller block a
// dozen bits.  P's exponent slot holds the joint row exponents, Q's slot holds a_i in
// its first entry.  H, R and T are scaled on their own.

// Padded n_b 17..20 stays on the FP64 kernel: two 16-row tiles then do 4x the digit work
// of one for at most 1.6x the entries, and on the batching meshes the FP64 kernel was
// faster at n_b = 18 (6.6 s against 8.0 s per step of the p = 3 mesh) while the two-tile
// kernel was faster at n_b = 30 (12.5 s against 21.9 s of the p = 5 mesh).
bool tc_supported(int nb, int B) {
  return (nb <= tc::kTile || (nb >= kTwoTileMinNb && nb <= 2 * tc::kTile)) && B <= tc::kCols;
}
bool tc_available(int nb, int B) { return nb <= 2 * tc::kTile && B <= tc::kCols; }

static int prepare_one_tile(Model& md, DevBuf& ops, cudaStream_t st) {
  const int rc = tc_prepare_tiles<1>(md, ops, st);
  return rc ? rc : tc_small_prepare();
}

int tc_prepare(Model& md, cudaStream_t st) {
  const int rc = md.nb <= tc::kTile ? prepare_one_tile(md, md.tc_ops, st) : tc2_prepare(md, st);
  md.tc_ready = rc == SBFWI_OK;
  return rc;
}

// One-tile digits of every element's operators (their top-left 16 x 16 block; for a mesh
// padded beyond 16 this is the whole operator of its elements with n_b <= 16, whose padded
// rows and columns are zero)
int tc_prepare_one_tile(Model& md, cudaStream_t st) {
  const int rc = prepare_one_tile(md, md.tc_ops_one, st);
  md.tc_one_ready = rc == SBFWI_OK;
  return rc;
}

static int tc_tile_rows(const Model& md, bool one_tile) {
  return md.nb > tc::kTile && !one_tile ? 2 * tc::kTile : tc::kTile;
}

// Whole tiles save the bounds checks, rows save the traffic of the padding.  Fused launches, tiles | rows, ms:
// 24 x 24 elements, N_r 16: n_b 16, 8 shots 0.055 | 0.060, n_b 8, 3 shots (5.3 times the values) 0.053 | 0.054,
// n_b 4, 3 shots (10.7 times) 0.053 | 0.053, n_b 4, 1 shot 0.053 | 0.051; 64 x 64 elements: n_b 16, 8 shots
// 0.217 | 0.219, 5 shots (1.6 times) 0.212 | 0.203, n_b 8, 8 shots (twice) 0.211 | 0.198.  Two tiles, 32 x 32
// elements: n_b 24, 8 shots 0.243 | 0.254, n_b 32, 4 shots (twice) 0.243 | 0.249.
TcState tc_state(const Model& md, int B, int64_t n_elems, int sms, bool one_tile) {
  TcState t;
  const int rows = tc_tile_rows(md, one_tile), nb = md.nb;
  const double most = n_elems <= kFewElements * (int64_t)sms ? 5.4 : rows > tc::kTile ? 2.0 : 1.1;
  t.tiles = rows * kTileShots <= most * nb * B && !(rows == tc::kTile && B <= kFewShots);
  t.rows = t.tiles ? rows : nb;
  t.doubles = t.tiles ? rows * kTileShots : nb * B;
  return t;
}

int tc_element_launch(const Model& md, const TcLaunch& l, cudaStream_t st) {
  ElemTcArgs a;
  a.l = l;
  a.nb = md.nb; a.n = md.n; a.E = md.E;
  a.a0 = md.a0; a.a1 = md.a1; a.a2 = md.a2; a.c1 = md.c1; a.c2 = md.c2; a.dt = md.dt;
  a.ops = (l.one_tile ? md.tc_ops_one : md.tc_ops).as<unsigned char>();
  a.dofs = md.dev().dofs.as<int32_t>();
  if (!l.elems) a.l.n_elems = md.E;
  if (a.l.n_elems == 0) return SBFWI_OK;
  // average acceleration (beta = 1/4, gamma = 1/2): the shorter predictor update
  const bool avg = md.a2 == 1.0 && md.c1 == md.c2;
  // one 16-row tile: n_b <= 16, or the elements of n_b <= 16 of a mesh padded beyond (the
  // one-tile digits of its operators, prepared by tc_prepare_one_tile)
  if (tc_tile_rows(md, l.one_tile) > tc::kTile) tc2_element_launch(a, avg, st);
  else if (l.B <= kFewShots) tc_small_launch(a, avg, st);
  else tc_launch_tiles<1>(a, avg, st);
  return SBFWI_OK;
}

}  // namespace sbfwi
