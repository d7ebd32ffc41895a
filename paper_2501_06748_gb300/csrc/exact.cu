// The exact discrete adjoint ("Mode X"): the derivative of the discrete misfit with respect
// to the nodal densities, by reverse-mode differentiation of the time loop.
//
// Forward step k (Section 3.3) solves A(rho) x_{k+1} = r_k with r_k = -xi_i^2 M0_i v_k + f_k,
// v_k the Newmark predictor (Eq. (ODE_Newmark)), x_{k+1} = every element's u_{-1}..u_{n+1}
// and the shared boundary u_n; the state is advanced by Eq. (Newmark) and the misfit
// E = 1/2 dt sum (d - u)^2 (Eq. (misfit)) reads the receivers.  The adjoint runs the steps
// backwards.  For step k, with x_bar the adjoint of u_{k+1} (misfit, Newmark update and the
// next step's predictor), mu = A^{-T} x_bar is found with the condensation's own operators
// in reverse (the transposes of the forward sweep, the global solve and the
// back-substitution, in reverse order):
//   up sweep     s_0 = x_bar_0, s_i = x_bar_i - H_{i-1}^T s_{i-1}, element part of the
//                boundary right-hand side -H_{n-1}^T s_{n-1};
//   global       F_bar = A_g^{-T} (x_bar_b + sum_e Z_e^T (-H_{n-1}^T s_{n-1})) = mu_{n+1}
//                (the flux-balance rows), with the transposed multifrontal factors;
//   down sweep   mu_n = -W^T mu_{n+1}, q_{n-1} = s_{n-1} + R^T mu_{n+1},
//                mu_i = G_i^T q_i, v_bar_i = -P_i^T q_i, q_{i-1} = s_{i-1} - Q_i^T q_i,
//                mu_{-1} = -rho_0^T mu_0, v_bar_n(e) = T^T mu_{n+1};
// the predictor's adjoint v_bar flows into the adjoints of u_k, u'_k, u''_k.
// The gradient is dE/drho = -sum_k mu_k^T dR/drho with R the residual of every row
// (rows 0..n: theta u_{i-1} + phi u_i + psi u_{i+1} + xi_i^2 M0_i v_i; rows -1 and n+1:
// the boundary-condition rows).  Every block is a combination of E0, E1, E2, M0 at one
// radial point and of the radial differences of E0, E1 (central inside, one-sided at the
// ends), and these are linear in the densities of the point: E0 = sum_j rho_j E0hat_j with
// E0hat_j = int phi_j c^2 (b1.b1) phi^T phi det J_b d eta (Eq. (Es)).  So each row's share
// is a sum over Gauss points of products of the interpolated mu and u fields (and their eta
// derivatives), bilinear in a line's nodal values: the time loop accumulates the products
// of the nodal values per row and line, which are interpolated and projected onto phi_j
// once at the end.
#include <algorithm>
#include <cstdint>

#include "internal.h"
#include "sync.cuh"

namespace sbfwi {

// ---------------------------------------------------------------------------
// element kernel: down sweep of step k fused with the up sweep of step k-1
// ---------------------------------------------------------------------------
// Bound by the FP64 pipe: four products per radial point and shot.  kStaged: the operators of the next
// point (G, P, Q down; H up) are copied to shared memory while the current one's products run, in two buffers an
// element; read straight from memory, their latency left the pipe 71 % busy: 0.42 -> 0.32 ms a step for 576
// elements of order 4, 32 radial points, 8 shots.
template <bool kStaged>
__global__ void __launch_bounds__(512) exact_element_kernel(ExactElemArgs a) {
  extern __shared__ double sh_all[];
  const int nb = a.nb, n = a.n, B = a.B;
  const int per = nb * B;
  double* sh = sh_all + (kStaged ? (size_t)a.epc * 6 * nb * nb : 0);
  const int tid = threadIdx.x;
  const int le = tid / per, rem = tid - le * per, r = rem / B, s = rem - r * B;
  const int64_t e = (int64_t)blockIdx.x * a.epc + le;
  const bool act = (le < a.epc) && (e < a.E);
  double* tbuf = sh + (size_t)le * n * per;                                  // [n][nb][B]
  double* xb = sh + (size_t)a.epc * n * per + (size_t)le * 4 * per;         // four exchange vectors
  double* xc = xb + per;
  double* xd = xc + per;
  double* xe = xd + per;
  const int64_t nn = (int64_t)nb * nb;
  const int64_t ee = act ? e : 0;
  const double* Me = a.mats + ee * (int64_t)n * 3 * nn;
  const double* Ge = a.xops + ee * (int64_t)n * nn;
  const double* Xe = a.xel + ee * 6 * nn;
  const double* RT = a.rt + ee * 2 * nn;
  const int64_t base = ee * (int64_t)n * per;
  const int64_t mrow = ee * (int64_t)(n + 2) * per;                           // mu rows -1..n of this element
  const int rs = r * B + s;
  const int32_t gnode = act ? a.dofs[ee * nb + r] : 0;
  const bool real_node = act && gnode < a.N;                                  // padding dofs point at node N
  double* ops = kStaged ? sh_all + (size_t)le * 6 * nn : nullptr;            // [2][G P Q] (or H) of this element
  // point i's operators of the down sweep, the H of point i, to buffer i & 1
  auto stage_down = [&](int i) {
    if constexpr (kStaged) {
      if (act && i >= 0) {
        copy_async(ops + (i & 1) * 3 * nn, Ge + (int64_t)i * nn, (int)nn, rem, per, (nb & 1) == 0);
        copy_async(ops + (i & 1) * 3 * nn + nn, Me + (int64_t)i * 3 * nn, (int)(2 * nn), rem, per, (nb & 1) == 0);
      }
      copy_commit();
    }
  };
  auto stage_up = [&](int i) {
    if constexpr (kStaged) {
      if (act && i < n) copy_async(ops + (i & 1) * 3 * nn, Me + ((int64_t)i * 3 + 2) * nn, (int)nn, rem, per, (nb & 1) == 0);
      copy_commit();
    }
  };

  if (a.do_down) {
    stage_down(n - 1);
    xb[rs] = real_node ? a.fbar[(int64_t)gnode * B + s] : 0.0;               // mu_{n+1}
    __syncthreads();
    double qv = 0.0, mu0 = 0.0;
    if (act) {
      const double* W = Xe + nn;
      const double* T = RT + nn;
      double aw = 0.0, at = 0.0, ar = 0.0;
      for (int c = 0; c < nb; ++c) {
        const double x = xb[c * B + s];
        aw = fma(W[c * nb + r], x, aw);
        at = fma(T[c * nb + r], x, at);
        ar = fma(RT[c * nb + r], x, ar);
      }
      a.mu[mrow + (int64_t)(n + 1) * per + rs] = -aw;                        // mu_n
      a.vbn[(ee * nb + r) * B + s] = at;                                      // v_bar_n of this element
      qv = a.s[base + (int64_t)(n - 1) * per + rs] + ar;
    }
    __syncthreads();
    xb[rs] = qv;
    if (!kStaged) __syncthreads();
    for (int i = n - 1; i >= 0; --i) {
      double qn = 0.0;
      if (kStaged) {                     // its buffer was last read before the barrier of the last round
        stage_down(i - 1);
        copy_wait<1>();
        __syncthreads();                 // every thread's copies, and xb
      }
      if (act) {
        const double* G = kStaged ? ops + (i & 1) * 3 * nn : Ge + (int64_t)i * nn;
        const double* P = kStaged ? G + nn : Me + (int64_t)i * 3 * nn;
        const double* Q = P + nn;
        double ag = 0.0, ap = 0.0, aq = 0.0;
        for (int c = 0; c < nb; ++c) {
          const double x = xb[c * B + s];
          ag = fma(G[c * nb + r], x, ag);
          ap = fma(P[c * nb + r], x, ap);
          aq = fma(Q[c * nb + r], x, aq);
        }
        a.mu[mrow + (int64_t)(i + 1) * per + rs] = ag;
        if (i == 0) mu0 = ag;
        const double vbar = -ap;
        // Newmark: adjoints of u, u', u'' at step k from those at k+1 and the predictor's
        const int64_t o = base + (int64_t)i * per + rs;
        const double ud1 = a.uda[o], udd1 = a.udda[o];
        const double uk = fma(a.a0, vbar, fma(-a.cu, ud1, -a.du * udd1));
        const double udk = fma(a.a1, vbar, fma(a.cud, ud1, a.dud * udd1));
        const double uddk = fma(a.a2, vbar, fma(a.cudd, ud1, a.dudd * udd1));
        a.ua[o] = uk; a.uda[o] = udk; a.udda[o] = uddk;
        tbuf[(int64_t)i * per + rs] = fma(a.cu, udk, fma(a.du, uddk, uk));  // x_bar_i of step k-1
        if (i > 0) qn = a.s[base + (int64_t)(i - 1) * per + rs] - aq;
      }
      __syncthreads();
      xb[rs] = qn;
      if (!kStaged) __syncthreads();
    }
    if (kStaged) __syncthreads();
    if (a.do_up) stage_up(0);            // the barriers below separate it from the last reads of its buffer
    // mu_{-1} = -rho_0^T mu_0
    xb[rs] = mu0;
    __syncthreads();
    if (act) {
      double acc = 0.0;
      for (int c = 0; c < nb; ++c) acc = fma(Xe[c * nb + r], xb[c * B + s], acc);
      a.mu[mrow + rs] = -acc;
    }
    // ghosts of the forward solution x_{k+1}: u_{-1} = u_1 + Gamma u_0,
    // u_{n+1} = -(Y_theta u_{n-1} + Y_phi u_n - Y_M u''_n)
    __syncthreads();
    if (act) {
      const int64_t fb = ee * (int64_t)n * per + rs;
      xb[rs] = a.fu_int[fb];                                                  // u_0
      xc[rs] = a.fu_int[fb + (int64_t)(n - 1) * per];                         // u_{n-1}
      xd[rs] = real_node ? a.fu_b[(int64_t)gnode * B + s] : 0.0;              // u_n
      xe[rs] = real_node ? a.fa_b[(int64_t)gnode * B + s] : 0.0;              // u''_n
    }
    __syncthreads();
    if (act) {
      const double* Gam = Xe + 2 * nn + (int64_t)r * nb;
      const double* Yt = Xe + 3 * nn + (int64_t)r * nb;
      const double* Yp = Xe + 4 * nn + (int64_t)r * nb;
      const double* Ym = Xe + 5 * nn + (int64_t)r * nb;
      double g0 = a.fu_int[ee * (int64_t)n * per + (int64_t)(n > 1 ? 1 : 0) * per + rs];   // u_1 (n >= 2)
      double g1 = 0.0;
      for (int c = 0; c < nb; ++c) {
        const int cs = c * B + s;
        g0 = fma(Gam[c], xb[cs], g0);
        g1 = fma(Yt[c], xc[cs], g1);
        g1 = fma(Yp[c], xd[cs], g1);
        g1 = fma(-Ym[c], xe[cs], g1);
      }
      a.ghost[(ee * 2) * per + rs] = g0;
      a.ghost[(ee * 2 + 1) * per + rs] = -g1;
    }
  } else if (a.do_up && (kStaged || act)) {
    stage_up(0);
    for (int i = 0; act && i < n; ++i) {
      const int64_t o = base + (int64_t)i * per + rs;
      tbuf[(int64_t)i * per + rs] = fma(a.cu, a.uda[o], fma(a.du, a.udda[o], a.ua[o]));
    }
  }
  if (!a.do_up) return;
  __syncthreads();
  // up sweep of step k-1: s_0 = x_bar_0, s_i = x_bar_i - H_{i-1}^T s_{i-1}
  for (int i = 0; i < n; ++i) {
    double v = 0.0;
    if (kStaged && i > 0) {
      stage_up(i);
      copy_wait<1>();
      __syncthreads();
    }
    if (act) {
      v = tbuf[(int64_t)i * per + rs];
      if (i > 0) {
        const double* H = kStaged ? ops + ((i - 1) & 1) * 3 * nn : Me + (int64_t)(i - 1) * 3 * nn + 2 * nn;
        for (int c = 0; c < nb; ++c) v = fma(-H[c * nb + r], xb[c * B + s], v);
      }
      a.s[base + (int64_t)i * per + rs] = v;
    }
    __syncthreads();
    xb[rs] = v;
    if (!kStaged) __syncthreads();
  }
  if (kStaged) {
    copy_wait<0>();
    __syncthreads();
  }
  if (act) {
    const double* H = kStaged ? ops + ((n - 1) & 1) * 3 * nn : Me + (int64_t)(n - 1) * 3 * nn + 2 * nn;
    double acc = 0.0;
    for (int c = 0; c < nb; ++c) acc = fma(H[c * nb + r], xb[c * B + s], acc);
    a.fhat[(ee * nb + r) * B + s] = -acc;
  }
}

// ---------------------------------------------------------------------------
// boundary nodes
// ---------------------------------------------------------------------------
// the misfit's share: the adjoint of u at the receivers after step k gets -dt (d - u)
__global__ void exact_misfit_kernel(double* ub, int B, int R, const int64_t* rec, const double* res, int64_t K,
                                    int64_t k, double dt) {
  const int t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= B * R) return;
  const int s = t / R, j = t - s * R;
  ub[rec[j] * B + s] -= dt * res[((int64_t)s * R + j) * K + k];
}

// x_bar of the boundary nodes for the transposed solve, and the Newmark update's share of
// the adjoints of u, u', u'' at step k
__global__ void exact_boundary_pre_kernel(ExactBoundaryArgs a) {
  const int64_t tot = a.N * a.B;
  for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < tot; t += (int64_t)gridDim.x * blockDim.x) {
    const double u1 = a.ub[t], ud1 = a.udb[t], udd1 = a.uddb[t];
    a.ext[t] = fma(a.cu, ud1, fma(a.du, udd1, u1));
    a.ub[t] = fma(-a.cu, ud1, -a.du * udd1);
    a.udb[t] = fma(a.cud, ud1, a.dud * udd1);
    a.uddb[t] = fma(a.cudd, ud1, a.dudd * udd1);
  }
}

// the predictor's share: v_bar of a node is the sum of its elements' T^T mu_{n+1}
__global__ void exact_boundary_post_kernel(ExactBoundaryArgs a) {
  const int64_t tot = a.N * a.B;
  for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < tot; t += (int64_t)gridDim.x * blockDim.x) {
    const int64_t g = t / a.B;
    const int s = (int)(t - g * a.B);
    double v = 0.0;
    for (int64_t l = a.inc_ptr[g]; l < a.inc_ptr[g + 1]; ++l) v += a.vbn[a.inc_list[l] * a.B + s];
    a.ub[t] = fma(a.a0, v, a.ub[t]);
    a.udb[t] = fma(a.a1, v, a.udb[t]);
    a.uddb[t] = fma(a.a2, v, a.uddb[t]);
  }
}

// ---------------------------------------------------------------------------
// gradient: products of one step
// ---------------------------------------------------------------------------
// Row r = -1..n+1 of one element per block: for every line and pair (a, b) of its nodes the
// products sum_shots mu_a w_b, added to the accumulators, with w = u_{r-1} - 2 u_r + u_{r+1},
// u_{r+1} - u_{r-1}, u_r and u'' (rows -1 and n+1: the two in the middle, with the fields of rows
// 0 and n).  The two in the middle are also differentiated along the line: there the values of a line are its
// first node's and the others' differences from it, so that the derivatives lose nothing where a field is
// nearly constant around the element (towards the scaling centre, as xi).
// Why nodal products: interpolating the fields to the Gauss points and multiplying there takes about 70
// FP64 operations per Gauss point, row and shot (seven points a line of order 4), the products 4 (p + 1)^2
// per line, row and shot without a reduction over lanes; the pipe does 2 a clock and SM.  576 elements of
// order 4, 32 radial points, 8 shots: 0.75 -> 0.15 ms a step.
__global__ void __launch_bounds__(128) exact_gradient_kernel(ExactGradArgs a) {
  extern __shared__ double shw[];          // [5][B][nb]: the four w and mu; [3][B][L][pp]: the middle two and mu by line
  const int nb = a.nb, n = a.n, B = a.B, per = nb * B, pp = a.pp, p2 = pp * pp;
  const int64_t e = blockIdx.x / (n + 3);
  const int r = (int)(blockIdx.x - e * (n + 3)) - 1;
  const int rr = min(max(r, 0), n);
  const bool inner = r == rr;
  const int32_t* dofs = a.dofs + e * nb;
  const double* fu = a.fu_int + e * (int64_t)n * per;
  const double* gh = a.ghost + e * 2 * per;
  for (int t = threadIdx.x; t < per; t += blockDim.x) {
    const int j = t / B, s = t - j * B;
    const int32_t gn = dofs[j];
    const bool node = gn < a.N;            // padding dofs point at node N
    // row q of the forward solution: ghosts, interior, boundary nodes
    auto u = [&](int q) {
      if (q < 0) return gh[t];
      if (q < n) return fu[(int64_t)q * per + t];
      if (q == n) return node ? a.fu_b[(int64_t)gn * B + s] : 0.0;
      return gh[per + t];
    };
    const double uA = u(rr - 1), uB = u(rr), uC = u(rr + 1);
    double w3 = 0.0;
    if (inner) w3 = r < n ? a.fa_int[(e * n + r) * (int64_t)per + t] : node ? a.fa_b[(int64_t)gn * B + s] : 0.0;
    const double mu = r <= n ? a.mu[(e * (n + 2) + r + 1) * (int64_t)per + t] : node ? a.fbar[(int64_t)gn * B + s] : 0.0;
    const int o = s * nb + j;
    shw[o] = uA - 2.0 * uB + uC;
    shw[per + o] = uC - uA;
    shw[2 * per + o] = uB;
    shw[3 * per + o] = w3;
    shw[4 * per + o] = mu;
  }
  __syncthreads();
  const int64_t l0 = a.lptr[e];
  const int L = (int)(a.lptr[e + 1] - l0);
  const int lp = L * pp;
  double* line = shw + 5 * per;
  for (int t = threadIdx.x; t < 3 * B * lp; t += blockDim.x) {
    const int v = t / (B * lp), sq = t - v * B * lp, s = sq / lp, q = sq - s * lp;
    const double* f = shw + (v < 2 ? v + 1 : 4) * per + s * nb;
    const int32_t* loc = a.line_local + l0 * pp;
    const double x = f[loc[q]];
    line[t] = q % pp ? x - f[loc[q / pp * pp]] : x;
  }
  __syncthreads();
  double* out = a.prod + (int64_t)blockIdx.x * a.L * 4 * p2;
  for (int o = threadIdx.x; o < L * 4 * p2; o += blockDim.x) {
    const int lk = o / p2, ab = o - lk * p2, l = lk >> 2, k = lk & 3, ia = ab / pp, ib = ab - ia * pp;
    if (!inner && (k == 0 || k == 3)) continue;
    const int32_t* loc = a.line_local + (l0 + l) * pp;
    const bool by_line = k == 1 || k == 2;
    const double* m = by_line ? line + 2 * B * lp + l * pp + ia : shw + 4 * per + loc[ia];
    const double* w = by_line ? line + (k - 1) * B * lp + l * pp + ib : shw + k * per + loc[ib];
    const int stride = by_line ? lp : nb;
    double acc = out[o];
    for (int s = 0; s < B; ++s) acc = fma(m[s * stride], w[s * stride], acc);
    out[o] = acc;
  }
}

// The Gauss-point sums of every station (radial point) from the nodal products of its row and its neighbours:
// a row's terms in E0 and E1 at its own point, and in their radial differences (forward at row 0, backward at
// row n, central inside)
__global__ void exact_collect_kernel(ExactFinalArgs a) {
  const int n = a.n, pp = a.pp, p2 = pp * pp, ng = a.ng;
  const int64_t tot = a.E * (int64_t)(n + 1) * a.L * ng;
  const double inv_2h = 0.5 / a.h;
  for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < tot; t += (int64_t)gridDim.x * blockDim.x) {
    const int g = (int)(t % ng);
    const int64_t tl = t / ng;
    const int l = (int)(tl % a.L);
    const int64_t es = tl / a.L, e = es / (n + 1);
    const int st = (int)(es - e * (n + 1));
    if (l >= (int)(a.lptr[e + 1] - a.lptr[e])) continue;
    const double* ph = a.tab + 2 * (ng + g * pp);                 // double-double pairs: the high parts
    const double* dph = a.tab + 2 * (ng + ng * pp + g * pp);
    auto row = [&](int r, int k) { return a.prod + (((e * (n + 3) + r + 1) * a.L + l) * 4 + k) * p2; };
    // sum_ab x_a y_b prod_ab, with x0 and y0 for the first node's functions
    auto contract = [&](const double* pr, double x0, const double* x, double y0, const double* y) {
      double v = 0.0;
      for (int ia = 0; ia < pp; ++ia) {
        double q = 0.0;
        for (int ib = 0; ib < pp; ++ib) q = fma(ib ? y[2 * ib] : y0, pr[ia * pp + ib], q);
        v = fma(ia ? x[2 * ia] : x0, q, v);
      }
      return v;
    };
    // values and derivatives of the products by line: the first node's value has the functions 1 and 0
    auto vv = [&](int r, int k) { return contract(row(r, k), 1.0, ph, 1.0, ph); };
    auto vd = [&](int r, int k) { return contract(row(r, k), 1.0, ph, 0.0, dph); };
    auto dv = [&](int r, int k) { return contract(row(r, k), 0.0, dph, 1.0, ph); };
    auto nodal = [&](int r, int k) { return contract(row(r, k), ph[0], ph, ph[0], ph); };
    const double xi = a.xi[st];
    double e0 = xi * xi / (a.h * a.h) * nodal(st, 0) + xi * inv_2h * vv(st, 1);
    double e1 = xi * inv_2h * (vd(st, 1) - dv(st, 1));
    const double e2 = -contract(row(st, 2), 0.0, dph, 0.0, dph);
    const double m = -xi * xi * nodal(st, 3);
    // times the weight w that row r's difference gives this station
    auto differences = [&](int r, double w) {
      const double x = a.xi[r];
      e0 = fma(w, x * x * inv_2h * vv(r, 1), e0);
      e1 = fma(w, x * vd(r, 2), e1);
    };
    if (st == 0) differences(0, -1.0 / a.h);
    if (st == n) differences(n, 1.0 / a.h);
    if (st >= 1) differences(st - 1, st == 1 ? 1.0 / a.h : inv_2h);
    if (st < n) differences(st + 1, st + 1 == n ? -1.0 / a.h : -inv_2h);
    // rows -1 and n+1: xi E0 (u_{r+1} - u_{r-1}) / (2h) + E1^T u
    for (int end = 0; end < 2; ++end)
      if (st == (end ? n : 0)) {
        const int r = end ? n + 1 : -1;
        e0 = fma(xi * inv_2h, vv(r, 1), e0);
        e1 += vd(r, 2);
      }
    const int64_t LG = (int64_t)a.L * ng;
    double* acc = a.gacc + es * 4 * LG + (int64_t)l * ng + g;
    acc[0] = e0;
    acc[LG] = e1;
    acc[2 * LG] = e2;
    acc[3 * LG] = m;
  }
}

// dE/drho at every radial point and boundary node of every element from the Gauss-point
// sums: -sum_lines sum_g phi_j(g) (k0 A0 + k1 A1 + k2 A2 + km Am); interior points go to
// the library's nodal layout, the boundary station to a per-element slot (gathered per node)
__global__ void exact_finalize_kernel(ExactFinalArgs a) {
  const int nb = a.nb, n = a.n, pp = a.pp, ng = a.ng;
  const int64_t tot = a.E * (int64_t)(n + 1) * nb;
  const int64_t LG = (int64_t)a.L * ng;
  for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < tot; t += (int64_t)gridDim.x * blockDim.x) {
    const int64_t e = t / ((int64_t)(n + 1) * nb);
    const int rem = (int)(t - e * (int64_t)(n + 1) * nb);
    const int st = rem / nb, j = rem - st * nb;
    const int64_t l0 = a.lptr[e];
    const int Le = (int)(a.lptr[e + 1] - l0);
    const double* acc = a.gacc + ((e * (n + 1) + st) * 4) * LG;
    double sum = 0.0;
    for (int l = 0; l < Le; ++l) {
      for (int q = 0; q < pp; ++q) {
        if (a.line_local[(l0 + l) * pp + q] != j) continue;
        for (int g = 0; g < ng; ++g) {
          const double* k = a.kq + ((e * a.L + l) * ng + g) * 4;
          const int64_t o = (int64_t)l * ng + g;
          const double v = k[0] * acc[o] + k[1] * acc[LG + o] + k[2] * acc[2 * LG + o] + k[3] * acc[3 * LG + o];
          sum = fma(a.tab[2 * (ng + g * pp + q)], v, sum);
        }
      }
    }
    if (st < n) a.g_nodal[(e * n + st) * nb + j] = -sum;
    else a.g_bnd[e * nb + j] = -sum;
  }
}

__global__ void exact_gather_nodes_kernel(const double* g_bnd, const int64_t* inc_ptr, const int64_t* inc_list,
                                          int64_t N, double* g_nodal_b) {
  for (int64_t g = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; g < N; g += (int64_t)gridDim.x * blockDim.x) {
    double v = 0.0;
    for (int64_t l = inc_ptr[g]; l < inc_ptr[g + 1]; ++l) v += g_bnd[inc_list[l]];
    g_nodal_b[g] = v;
  }
}

// ---------------------------------------------------------------------------
// host launchers
// ---------------------------------------------------------------------------
int exact_prepare_launches() {
  for (const void* f : {(const void*)exact_element_kernel<false>, (const void*)exact_element_kernel<true>,
                        (const void*)exact_gradient_kernel}) {
    const int rc = allow_shared_memory(f);
    if (rc) return rc;
  }
  return SBFWI_OK;
}

int exact_element_launch(const ExactElemArgs& a, cudaStream_t st) {
  const int threads = a.epc * a.nb * a.B;
  const unsigned blocks = (unsigned)((a.E + a.epc - 1) / a.epc);
  const size_t smem = exact_element_smem(a.nb, a.n, a.B, a.epc);
  // Staged where the operators leave room for four blocks on an SM (with few shots a block has many elements) and
  // either all blocks are on the SMs at once anyway or a block is one element.  Direct | staged, both element kernels
  // of a step, us: 24 x 24 elements, order 4, 8 shots 389 | 341, order 3, 5 shots 75 | 60; 64 x 64, order 4, 8 shots
  // 2212 | 2148, 3 shots (two elements a block) 1053 | 1072.
  const size_t staged = smem + sizeof(double) * (size_t)a.epc * 6 * a.nb * a.nb;
  if (stage_operators(staged, a.epc, blocks, a.sms)) {
    exact_element_kernel<true><<<blocks, threads, staged, st>>>(a);
  } else {
    exact_element_kernel<false><<<blocks, threads, smem, st>>>(a);
  }
  SBFWI_CUDA(cudaGetLastError());
  return SBFWI_OK;
}

size_t exact_element_smem(int nb, int n, int B, int epc) {
  return sizeof(double) * (size_t)epc * (n + 4) * nb * B;
}

int exact_misfit_launch(double* ub, int B, int R, const int64_t* rec, const double* res, int64_t K, int64_t k, double dt,
                        cudaStream_t st) {
  if (R == 0) return SBFWI_OK;
  exact_misfit_kernel<<<(B * R + 127) / 128, 128, 0, st>>>(ub, B, R, rec, res, K, k, dt);
  SBFWI_CUDA(cudaGetLastError());
  return SBFWI_OK;
}

int exact_boundary_launch(const ExactBoundaryArgs& a, bool post, cudaStream_t st) {
  const unsigned blocks = (unsigned)std::min<int64_t>((a.N * a.B + 255) / 256, 152 * 8);
  if (post) exact_boundary_post_kernel<<<blocks, 256, 0, st>>>(a);
  else exact_boundary_pre_kernel<<<blocks, 256, 0, st>>>(a);
  SBFWI_CUDA(cudaGetLastError());
  return SBFWI_OK;
}

int exact_gradient_launch(const ExactGradArgs& a, cudaStream_t st) {
  if (a.pp < 2 || a.pp > 9) return fail(SBFWI_EUNSUPPORTED, "line order outside 1..8");
  const size_t smem = sizeof(double) * (size_t)a.B * (5 * (size_t)a.nb + 3 * (size_t)a.L * a.pp);
  exact_gradient_kernel<<<(unsigned)(a.E * (a.n + 3)), 128, smem, st>>>(a);
  SBFWI_CUDA(cudaGetLastError());
  return SBFWI_OK;
}

int exact_finalize_launch(const ExactFinalArgs& a, const int64_t* inc_ptr, const int64_t* inc_list, int64_t N,
                          double* g_nodal_b, cudaStream_t st) {
  const int64_t sums = a.E * (int64_t)(a.n + 1) * a.L * a.ng;
  exact_collect_kernel<<<(unsigned)std::min<int64_t>((sums + 127) / 128, 152 * 32), 128, 0, st>>>(a);
  const int64_t tot = a.E * (int64_t)(a.n + 1) * a.nb;
  exact_finalize_kernel<<<(unsigned)std::min<int64_t>((tot + 255) / 256, 152 * 16), 256, 0, st>>>(a);
  exact_gather_nodes_kernel<<<(unsigned)std::min<int64_t>((N + 255) / 256, 152 * 8), 256, 0, st>>>(
      a.g_bnd, inc_ptr, inc_list, N, g_nodal_b);
  SBFWI_CUDA(cudaGetLastError());
  return SBFWI_OK;
}

}  // namespace sbfwi
