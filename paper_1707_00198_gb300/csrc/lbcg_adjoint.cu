// Discrete adjoint (reverse mode) of the colour-gradient LBM step, for gradients of an
// objective of the state at step T with respect to the contact angle (per outermost fluid
// node), the interfacial tension sigma and the two viscosities (Sec. II; Eq. 1-18, 28-36).
//
// One reverse step, from the adjoint lambda' of the stored post-streaming state after the
// step to the adjoint lambda of the state before it, has six stages:
//   fwd_local   : forward intermediates recomputed from the stored state: post-Zou-He
//                 populations, colour densities and rho^N (Eq. 12, 16); clears the scatter
//                 targets of this step;
//   fwd_grad    : raw gradient (Eq. 28, Eq. 29 virtual values evaluated on the fly), the
//                 wetting correction (Eq. 30-36) and n;
//   fwd_dn      : grad n (Eq. 28 on n with Eq. 29 virtual values);
//   adj_collide : transpose of streaming + bounce-back (a gather of lambda'), the
//                 hand-derived reverse of Eq. 14, 1-9, 17, 18, 10 and 13 per node, and the
//                 transpose of Eq. 28/29 applied to n (a scatter onto the n stencil);
//   adj_normal  : reverse of n = g/|g|, of Eq. 30-36 (d|g| and d theta), and the transpose of
//                 Eq. 28/29 applied to rho^N (a scatter);
//   adj_rho     : reverse of Eq. 12 and 16, then of the Zou-He columns -> lambda.
// The three forward stages of step j - 1 have the same neighbour dependencies as the three
// reverse stages of step j, so a reverse step runs as three launches, each with one reverse
// stage of step j and, in separate blocks beside it, one forward stage of step j - 1
// (double-buffered intermediates); only the first reversed step of a checkpoint segment needs
// the three forward kernels alone.
// A value that a stencil reads on a solid neighbour is that node's Eq. 29 virtual value, a
// weighted mean of its own fluid neighbours; the transpose scatters straight through that
// mean onto those fluid nodes.  The kernels are templates on their arithmetic R: double, or
// float for the FP32 reverse sweep (whose chains of dependent operations are several times
// shorter in latency than FP64's); scatters accumulate with atomics in R, the per-node
// parameter adjoints in double.  Node arrays are compact [ny][nx] (index y * nx + x).  The
// lattices are small, so blocks are small (64 threads) to spread a lattice over every SM.
#include <vector>

#include "../../include/lbcg.h"
#include "lbcg_internal.h"
#include "lbcg_wait.cuh"

namespace lbcg {

namespace {

constexpr int kAdjThreads = 64;

template <typename R>
__device__ __forceinline__ bool is_solid(const AdjDevT<R>& A, int x, int y) {
  return A.sol[y * A.L.nx + x] != 0;
}
// bit a-1 of node j's mask: its neighbour in direction a (1..8) is solid
template <typename R>
__device__ __forceinline__ bool nb_solid(const AdjDevT<R>& A, int j, int a) {
  return (A.nbm[j] >> (a - 1)) & 1u;
}
__device__ __forceinline__ bool mask_bit(unsigned m, int a) { return (m >> (a - 1)) & 1u; }
template <typename R>
__device__ __forceinline__ uint8_t flag_at(const AdjDevT<R>& A, int x, int y) {
  return A.flags[A.L.node_off + (long long)y * A.L.pitch + x];
}
template <typename R>
__device__ __forceinline__ int mapx(const AdjDevT<R>& A, int v) { return wrap_or_clamp(v, A.L.nx, A.L.bcx == BC_PERIODIC); }
template <typename R>
__device__ __forceinline__ int mapy(const AdjDevT<R>& A, int v) { return wrap_or_clamp(v, A.L.ny, A.L.bcy == BC_PERIODIC); }

// ------------------------------------------------------------------ forward intermediates
template <typename R, bool kGather>
__device__ __forceinline__ void fwd_local_body(const AdjDevT<R>& A, const void* src, const int i, const int p) {
  const int x = i % A.L.nx, y = i / A.L.nx;
  const int M = A.M;
  // The kernels of the reverse sweep run a few warps per SM, so each memory round trip on a
  // thread's path counts: a node's loads are issued together, before its solid test (the
  // slots of a solid node are read but not used).
  const bool solid = is_solid(A, x, y);
  if constexpr (!kGather) A.lnt_x[i] = A.lnt_y[i] = A.lrnt[i] = R(0.0);
  R fr[9], fb[9], rR, rB;
  if (A.src_fp32) {
    // FP32 forward: its post-Zou-He populations, converted to the reverse arithmetic
    float fr32[9], fb32[9];
    load_node<float>(A.L, static_cast<const float*>(src), x, y, fr32, fb32);
    for (int a = 0; a < 9; ++a) {
      fr[a] = R(fr32[a]);
      fb[a] = R(fb32[a]);
    }
  } else {
    double fr64[9], fb64[9];
    load_node<double>(A.L, static_cast<const double*>(src), x, y, fr64, fb64);
    for (int a = 0; a < 9; ++a) {
      fr[a] = R(fr64[a]);
      fb[a] = R(fb64[a]);
    }
  }
  if (solid) {
    for (int a = 0; a < 9; ++a) A.fr[a * M + p] = A.fb[a * M + p] = R(0.0);
    A.rr[p] = A.rb[p] = A.rn[i] = R(0.0);
    return;
  }
  for (int a = 0; a < 9; ++a) {
    A.fr[a * M + p] = fr[a];
    A.fb[a * M + p] = fb[a];
  }
  A.rn[i] = colour_indicator(fr, fb, rR, rB);
  A.rr[p] = rR;
  A.rb[p] = rB;
}

// Sum of the D2Q9 weights toward the fluid neighbours of a solid node (Eq. 29 denominator)
template <typename R>
__device__ R weight_sum(const AdjDevT<R>& A, int x, int y) {
  const unsigned m = A.nbm[y * A.L.nx + x];
  R den = R(0.0);
  for (int b = 1; b < 9; ++b)
    if (!((m >> (b - 1)) & 1u)) den = radd(den, wgt<R>(b));
  return den;
}

// Value of field v that a stencil reads at (x, y): v itself on a fluid node, the Eq. 29
// virtual value (the same sums in the same order as the step kernels) on a solid node
// (solid: whether (x, y) is a solid node, known from the reading node's neighbour mask)
template <typename R>
__device__ R read_field(const AdjDevT<R>& A, const R* v, int x, int y, bool solid) {
  if (!solid) return v[y * A.L.nx + x];
  const unsigned m = A.nbm[y * A.L.nx + x];
  R num = R(0.0), den = R(0.0);
  for (int b = 1; b < 9; ++b) {
    if (!((m >> (b - 1)) & 1u)) {
      const int x2 = mapx(A, x + ex(b)), y2 = mapy(A, y + ey(b));
      num = radd(num, rmul(wgt<R>(b), v[y2 * A.L.nx + x2]));
      den = radd(den, wgt<R>(b));
    }
  }
  return den > R(0.0) ? rdiv(num, den) : R(0.0);
}

// Transpose of read_field for one or two fields: add `val` to the adjoint of what was read
template <typename R>
__device__ void scatter_field(const AdjDevT<R>& A, R* acc0, R* acc1, int x, int y, bool solid, R v0, R v1) {
  if (!solid) {
    const int j = y * A.L.nx + x;
    atomicAdd(&acc0[j], v0);
    if (acc1) atomicAdd(&acc1[j], v1);
    return;
  }
  const R den = weight_sum(A, x, y);
  if (!(den > R(0.0))) return;
  const R r = R(1.0) / den;
  const unsigned m = A.nbm[y * A.L.nx + x];
  for (int b = 1; b < 9; ++b) {
    if ((m >> (b - 1)) & 1u) continue;
    const int x2 = mapx(A, x + ex(b)), y2 = mapy(A, y + ey(b));
    const int j = y2 * A.L.nx + x2;
    const R c = wgt<R>(b) * r;
    atomicAdd(&acc0[j], c * v0);
    if (acc1) atomicAdd(&acc1[j], c * v1);
  }
}

// field(a): rho^N (of Eq. 28-29's reading) at the neighbour in direction a
template <typename R, typename F>
__device__ __forceinline__ void fwd_grad_body(const AdjDevT<R>& A, const int i, const int p, const uint8_t f, F field) {
  const R nsx = A.nsx[i], nsy = A.nsy[i];
  const R c = A.cos_t[i], s = A.sin_t[i];
  A.pick[p] = 0;
  if (f & F_SOLID) {
    A.grx[p] = A.gry[p] = A.gcx[p] = A.gcy[p] = R(0.0);
    A.nxv[i] = A.nyv[i] = R(0.0);
    return;
  }
  R gx = R(0.0), gy = R(0.0);
#pragma unroll
  for (int a = 1; a < 9; ++a) {
    const R t = rmul(wgt<R>(a), field(a));
    if (ex(a) == 1) gx = radd(gx, t);
    if (ex(a) == -1) gx = radd(gx, -t);
    if (ey(a) == 1) gy = radd(gy, t);
    if (ey(a) == -1) gy = radd(gy, -t);
  }
  gx = rdiv(gx, R(1.0 / 3.0));
  gy = rdiv(gy, R(1.0 / 3.0));
  A.grx[p] = gx;
  A.gry[p] = gy;
  R cgx = gx, cgy = gy;
  const R eps = A.C.grad_eps;
  const R mag = rsqrt_(radd(rmul(gx, gx), rmul(gy, gy)));
  if ((f & F_OFB) && mag > eps) {
    const R esx = rdiv(gx, mag), esy = rdiv(gy, mag);
    const R f1x = rsub(rmul(nsx, c), rmul(nsy, s)), f1y = radd(rmul(nsx, s), rmul(nsy, c));
    const R f2x = radd(rmul(nsx, c), rmul(nsy, s)), f2y = radd(rmul(-nsx, s), rmul(nsy, c));
    const R a1 = rsub(f1x, esx), b1 = rsub(f1y, esy), a2 = rsub(f2x, esx), b2 = rsub(f2y, esy);
    const R d1 = rsqrt_(radd(rmul(a1, a1), rmul(b1, b1)));
    const R d2 = rsqrt_(radd(rmul(a2, a2), rmul(b2, b2)));
    const bool one = d1 <= d2;
    A.pick[p] = one ? 1 : 2;
    cgx = rmul(mag, one ? f1x : f2x);
    cgy = rmul(mag, one ? f1y : f2y);
  }
  A.gcx[p] = cgx;
  A.gcy[p] = cgy;
  const R m2 = sqrt(cgx * cgx + cgy * cgy);
  A.nxv[i] = m2 > eps ? cgx / m2 : R(0.0);
  A.nyv[i] = m2 > eps ? cgy / m2 : R(0.0);
}

template <typename R>
__device__ __forceinline__ void fwd_grad_node(const AdjDevT<R>& A, const int i) {
  const int x = i % A.L.nx, y = i / A.L.nx;
  const unsigned msk = A.nbm[i];
  fwd_grad_body(A, i, i, flag_at(A, x, y), [&](int a) {
    return read_field(A, A.rn, mapx(A, x + ex(a)), mapy(A, y + ey(a)), mask_bit(msk, a));
  });
}

// fx(a), fy(a): n_x and n_y at the neighbour in direction a
template <typename R, typename F, typename G>
__device__ __forceinline__ void fwd_dn_body(const AdjDevT<R>& A, const int p, const bool solid, F fx, G fy) {
  const int M = A.M;
  R d[4] = {0, 0, 0, 0};
  if (!solid) {
#pragma unroll
    for (int a = 1; a < 9; ++a) {
      const R tx = wgt<R>(a) * fx(a);
      const R ty = wgt<R>(a) * fy(a);
      d[0] += ex(a) * tx;
      d[1] += ey(a) * tx;
      d[2] += ex(a) * ty;
      d[3] += ey(a) * ty;
    }
  }
  for (int q = 0; q < 4; ++q) A.dn[q * M + p] = R(3.0) * d[q];
}
template <typename R>
__device__ __forceinline__ void fwd_dn_node(const AdjDevT<R>& A, const int i) {
  const int x = i % A.L.nx, y = i / A.L.nx;
  const unsigned msk = A.nbm[i];
  auto at = [&](const R* v, int a) {
    return read_field(A, v, mapx(A, x + ex(a)), mapy(A, y + ey(a)), mask_bit(msk, a));
  };
  fwd_dn_body(A, i, is_solid(A, x, y), [&](int a) { return at(A.nxv, a); }, [&](int a) { return at(A.nyv, a); });
}

// ------------------------------------------------------------------ reverse kernels
// Transpose of the push (Eq. 15, half-way bounce-back, open edges) and the reverse of the
// node-local part of the step.
// kGather: instead of scattering the transpose of grad n, the adjoints of d_x n_x, d_y n_x (= that
// of d_x n_y) and d_y n_y are stored, and the nodes that were read gather them (k_reverse).
template <typename R, bool kGather>
__device__ __forceinline__ void adj_collide_body(const AdjDevT<R>& A, const R* lam_next, const int i, const int p,
                                                 const bool solid, const unsigned msk, R& d_sigma, R& d_hR, R& d_hB,
                                                 R* src0 = nullptr, R* src1 = nullptr, R* src2 = nullptr) {
  const int x = i % A.L.nx, y = i / A.L.nx;
  const int N = A.N, M = A.M;
  d_sigma = d_hR = d_hB = R(0.0);
  const LatDev& L = A.L;
  const LatConst<R>& C = A.C;
  // the node's forward intermediates, all in flight together before the solid test
  R fr[9], fb[9], f[9];
  for (int a = 0; a < 9; ++a) {
    fr[a] = A.fr[a * M + p];
    fb[a] = A.fb[a * M + p];
    f[a] = fr[a] + fb[a];
  }
  const R rhoR = A.rr[p], rhoB = A.rb[p], rn = A.rn[i];
  const R nxo = A.nxv[i], nyo = A.nyv[i];
  const R gx = A.gcx[p], gy = A.gcy[p];
  const R dxx = A.dn[p], dxy = A.dn[M + p], dyx = A.dn[2 * M + p], dyy = A.dn[3 * M + p];
  if (solid) {
    for (int a = 0; a < 9; ++a) A.lf_r[a * M + p] = A.lf_b[a * M + p] = R(0.0);
    A.ln_x[p] = A.ln_y[p] = A.lg_x[p] = A.lg_y[p] = A.lrn[p] = R(0.0);
    return;
  }
  const bool px = L.bcx == BC_PERIODIC, py = L.bcy == BC_PERIODIC;
  // adjoint of the post-collision, recoloured values (oR_a, oB_a) leaving this node
  R mR[9], mB[9];
  for (int a = 0; a < 9; ++a) {
    mR[a] = mB[a] = R(0.0);
    int j = i, slot = a;
    if (a != 0) {
      const int xr = x + ex(a), yr = y + ey(a);
      if ((!px && (xr < 0 || xr >= L.nx)) || (!py && (yr < 0 || yr >= L.ny))) continue;
      const int xd = mapx(A, xr), yd = mapy(A, yr);
      if (mask_bit(msk, a)) slot = opp(a);
      else j = yd * L.nx + xd;
    }
    mR[a] = lam_next[(2 * slot) * N + j];
    mB[a] = lam_next[(2 * slot + 1) * N + j];
  }
  // forward recomputation of the node-local quantities
  const R rho = rhoR + rhoB, ir = R(1.0) / rho;
  const R kappa = -nxo * nxo * dyy - nyo * nyo * dxx + nxo * nyo * (dxy + dyx);
  const R hsk = R(0.5) * C.sigma * kappa;
  const R Fx = hsk * gx, Fy = hsk * gy;
  const R jx = f[1] - f[3] + f[5] - f[6] - f[7] + f[8];
  const R jy = f[2] - f[4] + f[5] + f[6] - f[7] - f[8];
  const R ux = (jx + R(0.5) * Fx) * ir, uy = (jy + R(0.5) * Fy) * ir;
  const R inv_nu = (1 + rn) * C.h_inv_nuR + (1 - rn) * C.h_inv_nuB;
  const R den_sv = R(3.0) + R(0.5) * inv_nu;
  const R sv = inv_nu / den_sv;
  const R se = C.s_e, seps = C.s_eps, sq = C.s_q, beta = C.beta;
  const R s14 = f[1] + f[2] + f[3] + f[4], s58 = f[5] + f[6] + f[7] + f[8];
  const R me = -4 * f[0] - s14 + 2 * s58;
  const R meps = 4 * f[0] - 2 * s14 + s58;
  const R qx = -2 * (f[1] - f[3]) + (f[5] - f[6] - f[7] + f[8]);
  const R qy = -2 * (f[2] - f[4]) + (f[5] + f[6] - f[7] - f[8]);
  const R pxx = f[1] - f[2] + f[3] - f[4];
  const R pxy = f[5] - f[6] + f[7] - f[8];
  const R u2 = ux * ux + uy * uy, uF = ux * Fx + uy * Fy;
  const R De = se * (me - rho * (-2 + 3 * u2)) - (1 - R(0.5) * se) * (6 * uF);
  const R Deps = seps * (meps - rho * (1 - 3 * u2)) + (1 - R(0.5) * seps) * (6 * uF);
  const R Dqx = sq * (qx + rho * ux) + (1 - R(0.5) * sq) * Fx;
  const R Dqy = sq * (qy + rho * uy) + (1 - R(0.5) * sq) * Fy;
  const R Axx = pxx - rho * (ux * ux - uy * uy), Bxx = 2 * (ux * Fx - uy * Fy);
  const R Dxx = sv * Axx - (1 - R(0.5) * sv) * Bxx;
  const R Axy = pxy - rho * ux * uy, Bxy = ux * Fy + uy * Fx;
  const R Dxy = sv * Axy - (1 - R(0.5) * sv) * Bxy;
  constexpr R k36 = R(1.0) / 36, k12 = R(1.0) / 12, k6 = R(1.0) / 6;
  const R ae = De * k36, aeps = Deps * k36, ajx = -Fx * k6, ajy = -Fy * k6;
  const R aqx = Dqx * k12, aqy = Dqy * k12, axx = Dxx * R(0.25), axy = Dxy * R(0.25);
  R fp[9];
  fp[0] = f[0] - (-4 * ae + 4 * aeps);
  const R c14 = -ae - 2 * aeps;
  fp[1] = f[1] - (c14 + ajx - 2 * aqx + axx);
  fp[2] = f[2] - (c14 + ajy - 2 * aqy - axx);
  fp[3] = f[3] - (c14 - ajx + 2 * aqx + axx);
  fp[4] = f[4] - (c14 - ajy + 2 * aqy - axx);
  const R c58 = 2 * ae + aeps;
  fp[5] = f[5] - (c58 + ajx + aqx + ajy + aqy + axy);
  fp[6] = f[6] - (c58 - ajx - aqx + ajy + aqy - axy);
  fp[7] = f[7] - (c58 - ajx - aqx - ajy - aqy + axy);
  fp[8] = f[8] - (c58 + ajx + aqx - ajy - aqy - axy);
  const R cR = rhoR * ir;
  const R pc = beta * rhoR * rhoB * ir;
  // ---- reverse of Eq. 14: oR = cR fp + pc w (e.n), oB = fp - oR
  R lfp[9], lcR = 0, lpc = 0, lnx = 0, lny = 0;
  for (int a = 0; a < 9; ++a) {
    const R mu = mR[a] - mB[a];        // adjoint of oR through both outputs
    const R en = ex(a) * nxo + ey(a) * nyo;
    lfp[a] = mB[a] + mu * cR;
    lcR += mu * fp[a];
    lpc += mu * wgt<R>(a) * en;
    lnx += mu * pc * wgt<R>(a) * ex(a);
    lny += mu * pc * wgt<R>(a) * ey(a);
  }
  R lrhoR = (lcR + lpc * beta * rhoB) * ir;
  R lrhoB = lpc * beta * rhoR * ir;
  R lrho = -(lcR * rhoR + lpc * beta * rhoR * rhoB) * ir * ir;
  // ---- reverse of fp = f - M^T diag(...) Delta
  R lf[9];
  for (int a = 0; a < 9; ++a) lf[a] = lfp[a];
  // adjoints of the a_k: l_ak = -sum_a M[k][a] lfp[a]
  const R lae = -(-4 * lfp[0] - lfp[1] - lfp[2] - lfp[3] - lfp[4] + 2 * (lfp[5] + lfp[6] + lfp[7] + lfp[8]));
  const R laeps = -(4 * lfp[0] - 2 * (lfp[1] + lfp[2] + lfp[3] + lfp[4]) + lfp[5] + lfp[6] + lfp[7] + lfp[8]);
  const R lajx = -(lfp[1] - lfp[3] + lfp[5] - lfp[6] - lfp[7] + lfp[8]);
  const R lajy = -(lfp[2] - lfp[4] + lfp[5] + lfp[6] - lfp[7] - lfp[8]);
  const R laqx = -(-2 * lfp[1] + 2 * lfp[3] + lfp[5] - lfp[6] - lfp[7] + lfp[8]);
  const R laqy = -(-2 * lfp[2] + 2 * lfp[4] + lfp[5] + lfp[6] - lfp[7] - lfp[8]);
  const R laxx = -(lfp[1] - lfp[2] + lfp[3] - lfp[4]);
  const R laxy = -(lfp[5] - lfp[6] + lfp[7] - lfp[8]);
  const R lDe = lae * k36, lDeps = laeps * k36, lDqx = laqx * k12, lDqy = laqy * k12;
  const R lDxx = laxx * R(0.25), lDxy = laxy * R(0.25);
  R lFx = -lajx * k6, lFy = -lajy * k6;
  R lux = 0, luy = 0, lu2 = 0, luF = 0, lsv = 0;
  R lme = 0, lmeps = 0, lqx = 0, lqy = 0, lpxx = 0, lpxy = 0;
  // De
  lme += se * lDe;
  lrho += -se * (-2 + 3 * u2) * lDe;
  lu2 += -3 * se * rho * lDe;
  luF += -6 * (1 - R(0.5) * se) * lDe;
  // Deps
  lmeps += seps * lDeps;
  lrho += -seps * (1 - 3 * u2) * lDeps;
  lu2 += 3 * seps * rho * lDeps;
  luF += 6 * (1 - R(0.5) * seps) * lDeps;
  // Dqx, Dqy
  lqx += sq * lDqx;
  lrho += sq * ux * lDqx;
  lux += sq * rho * lDqx;
  lFx += (1 - R(0.5) * sq) * lDqx;
  lqy += sq * lDqy;
  lrho += sq * uy * lDqy;
  luy += sq * rho * lDqy;
  lFy += (1 - R(0.5) * sq) * lDqy;
  // Dxx = sv Axx - (1 - sv/2) Bxx
  lsv += (Axx + R(0.5) * Bxx) * lDxx;
  lpxx += sv * lDxx;
  lrho += -sv * (ux * ux - uy * uy) * lDxx;
  lux += -2 * sv * rho * ux * lDxx - (1 - R(0.5) * sv) * 2 * Fx * lDxx;
  luy += 2 * sv * rho * uy * lDxx + (1 - R(0.5) * sv) * 2 * Fy * lDxx;
  lFx += -(1 - R(0.5) * sv) * 2 * ux * lDxx;
  lFy += (1 - R(0.5) * sv) * 2 * uy * lDxx;
  // Dxy = sv Axy - (1 - sv/2) Bxy
  lsv += (Axy + R(0.5) * Bxy) * lDxy;
  lpxy += sv * lDxy;
  lrho += -sv * ux * uy * lDxy;
  lux += -sv * rho * uy * lDxy - (1 - R(0.5) * sv) * Fy * lDxy;
  luy += -sv * rho * ux * lDxy - (1 - R(0.5) * sv) * Fx * lDxy;
  lFy += -(1 - R(0.5) * sv) * ux * lDxy;
  lFx += -(1 - R(0.5) * sv) * uy * lDxy;
  // u2, uF
  lux += 2 * ux * lu2 + Fx * luF;
  luy += 2 * uy * lu2 + Fy * luF;
  lFx += ux * luF;
  lFy += uy * luF;
  // moments -> f
  for (int a = 0; a < 9; ++a) {
    const R r1 = (a == 0) ? -4 : (a <= 4 ? -1 : 2);
    const R r2 = (a == 0) ? 4 : (a <= 4 ? -2 : 1);
    const R rqx = (a == 1) ? -2 : (a == 3) ? 2 : (a >= 5 ? (R)ex(a) : R(0.0));
    const R rqy = (a == 2) ? -2 : (a == 4) ? 2 : (a >= 5 ? (R)ey(a) : R(0.0));
    const R rxx = (a == 1 || a == 3) ? 1 : (a == 2 || a == 4) ? -1 : 0;
    const R rxy = (a >= 5) ? (R)(ex(a) * ey(a)) : R(0.0);
    lf[a] += r1 * lme + r2 * lmeps + rqx * lqx + rqy * lqy + rxx * lpxx + rxy * lpxy;
  }
  // sv = inv_nu / (3 + inv_nu / 2); inv_nu = (1 + rn) hR + (1 - rn) hB
  const R linv = lsv * R(3.0) / (den_sv * den_sv);
  R lrn_loc = (C.h_inv_nuR - C.h_inv_nuB) * linv;
  d_hR = (1 + rn) * linv;
  d_hB = (1 - rn) * linv;
  // u = (j + F/2) / rho
  const R ljx = lux * ir, ljy = luy * ir;
  lFx += R(0.5) * ljx;
  lFy += R(0.5) * ljy;
  lrho += -(ux * lux + uy * luy) * ir;
  for (int a = 0; a < 9; ++a) lf[a] += ex(a) * ljx + ey(a) * ljy;
  // F = (sigma kappa / 2) g
  const R lhsk = gx * lFx + gy * lFy;
  const R lgx = hsk * lFx, lgy = hsk * lFy;
  d_sigma = R(0.5) * kappa * lhsk;
  const R lk = R(0.5) * C.sigma * lhsk;
  // kappa = -nx^2 dyy - ny^2 dxx + nx ny (dxy + dyx)
  lnx += (-2 * nxo * dyy + nyo * (dxy + dyx)) * lk;
  lny += (-2 * nyo * dxx + nxo * (dxy + dyx)) * lk;
  // transpose of grad n = 3 sum_a w_a e_a n~(x + e_a) (Eq. 28 on the Eq. 29-filled n)
  if constexpr (kGather) {
    src0[i] = -nyo * nyo * lk;
    src1[i] = nxo * nyo * lk;
    src2[i] = -nxo * nxo * lk;
  } else if (lk != R(0.0)) {
    const R lxx = -nyo * nyo * lk;   // adjoint of d_x n_x
    const R lxy = nxo * nyo * lk;    // d_y n_x
    const R lyx = nxo * nyo * lk;    // d_x n_y
    const R lyy = -nxo * nxo * lk;   // d_y n_y
    for (int a = 1; a < 9; ++a) {
      const R w = R(3.0) * wgt<R>(a);
      scatter_field(A, A.lnt_x, A.lnt_y, mapx(A, x + ex(a)), mapy(A, y + ey(a)), mask_bit(msk, a),
                    w * (ex(a) * lxx + ey(a) * lxy),
                    w * (ex(a) * lyx + ey(a) * lyy));
    }
  }
  // rho = rhoR + rhoB; f = fr + fb
  lrhoR += lrho;
  lrhoB += lrho;
  for (int a = 0; a < 9; ++a) {
    A.lf_r[a * M + p] = lf[a] + lrhoR;
    A.lf_b[a * M + p] = lf[a] + lrhoB;
  }
  A.lrn[p] = lrn_loc;
  A.ln_x[p] = lnx;
  A.ln_y[p] = lny;
  A.lg_x[p] = lgx;
  A.lg_y[p] = lgy;
}

// d_sigma, d_hR, d_hB: this step's share of the parameter adjoints
template <typename R>
__device__ __forceinline__ void adj_collide_node(const AdjDevT<R>& A, const int i) {
  const double p_hR0 = A.p_hR[i], p_hB0 = A.p_hB[i], p_sigma0 = A.p_sigma[i];
  R ds, dR, dB;
  adj_collide_body<R, false>(A, A.lam_next, i, i, A.sol[i] != 0, A.nbm[i], ds, dR, dB);
  A.p_sigma[i] = p_sigma0 + ds;
  A.p_hR[i] = p_hR0 + dR;
  A.p_hB[i] = p_hB0 + dB;
}

// Reverse of n = g_c / |g_c| (zero below the guard), of Eq. 30-36 (g_c = |g_r| n_f(theta) on
// Omega_Fb, g_c = g_r elsewhere), and the transpose of the raw gradient (Eq. 28 on the
// Eq. 29-filled rho^N), scattered onto rho^N.
// lntx, lnty: the adjoint of n through the neighbours' grad n.  Returns in lrx, lry the adjoint of
// the raw gradient (zero on a solid node), in d_theta this step's share of dJ/d theta.
template <typename R>
__device__ __forceinline__ void adj_normal_body(const AdjDevT<R>& A, const int i, const int p, const bool solid, R lntx,
                                                R lnty, R& lrx, R& lry, R& d_theta) {
  // everything the node reads, in flight together before the solid test
  const R lnx = A.ln_x[p] + lntx, lny = A.ln_y[p] + lnty;
  R lgx = A.lg_x[p], lgy = A.lg_y[p];
  const R gcx = A.gcx[p], gcy = A.gcy[p];
  const int pick = A.pick[p];
  const R grx = A.grx[p], gry = A.gry[p];
  const R nsx = A.nsx[i], nsy = A.nsy[i];
  const R c = A.cos_t[i], s = A.sin_t[i];
  lrx = lry = d_theta = R(0.0);
  if (solid) return;
  {
    const R gx = gcx, gy = gcy;
    const R m = sqrt(gx * gx + gy * gy);
    if (m > A.n_eps) {   // below it n is frozen in the reverse sweep (see AdjDev::n_eps)
      const R im = R(1.0) / m, nx = gx * im, ny = gy * im;
      const R dot = nx * lnx + ny * lny;
      lgx += (lnx - nx * dot) * im;
      lgy += (lny - ny * dot) * im;
    }
  }
  lrx = lgx;
  lry = lgy;
  if (pick != 0) {
    const R gx = grx, gy = gry;
    const R m = sqrt(gx * gx + gy * gy);
    R nfx, nfy, dfx, dfy;
    if (pick == 1) {   // rotation by +theta; d n_f / d theta = (-n_fy, n_fx)
      nfx = nsx * c - nsy * s;
      nfy = nsx * s + nsy * c;
      dfx = -nfy;
      dfy = nfx;
    } else {           // rotation by -theta; d n_f / d theta = (n_fy, -n_fx)
      nfx = nsx * c + nsy * s;
      nfy = -nsx * s + nsy * c;
      dfx = nfy;
      dfy = -nfx;
    }
    const R proj = (nfx * lgx + nfy * lgy) / m;
    lrx = gx * proj;
    lry = gy * proj;
    d_theta = m * (dfx * lgx + dfy * lgy);
  }
}
template <typename R>
__device__ __forceinline__ void adj_normal_node(const AdjDevT<R>& A, const int i) {
  const int x = i % A.L.nx, y = i / A.L.nx;
  const unsigned msk = A.nbm[i];
  const double p_theta0 = A.p_theta[i];
  R lrx, lry, dt;
  adj_normal_body(A, i, i, is_solid(A, x, y), A.lnt_x[i], A.lnt_y[i], lrx, lry, dt);
  if (dt != R(0.0)) A.p_theta[i] = p_theta0 + dt;
  if (lrx != R(0.0) || lry != R(0.0))
    for (int a = 1; a < 9; ++a)
      scatter_field(A, A.lrnt, static_cast<R*>(nullptr), mapx(A, x + ex(a)), mapy(A, y + ey(a)), mask_bit(msk, a),
                    R(3.0) * wgt<R>(a) * (ex(a) * lrx + ey(a) * lry), R(0.0));
}

// reverse of rho^N = (rhoR - rhoB)/(rhoR + rhoB) and of the Zou-He columns
template <typename R>
__device__ __forceinline__ void adj_rho_body(const AdjDevT<R>& A, R* lam, const int i, const int p, const bool solid, R lrnt) {
  const int x = i % A.L.nx, y = i / A.L.nx;
  const int N = A.N, M = A.M;
  // the node's inputs, in flight together before the solid test
  const R lrn = A.lrn[p] + lrnt;
  const R rR = A.rr[p], rB = A.rb[p];
  R lr[9], lb[9];
  for (int a = 0; a < 9; ++a) {
    lr[a] = A.lf_r[a * M + p];
    lb[a] = A.lf_b[a * M + p];
  }
  if (solid) {
    for (int a = 0; a < 18; ++a) lam[a * N + i] = R(0.0);
    return;
  }
  const R rho = rR + rB;
  const R ir2 = R(1.0) / (rho * rho);
  const R cR = 2 * rB * ir2 * lrn, cB = -2 * rR * ir2 * lrn;
  for (int a = 0; a < 9; ++a) {
    lr[a] += cR;
    lb[a] += cB;
  }
  const LatDev& L = A.L;
  R sr[9], sb[9];   // adjoint of the stored values
  if (L.bcx == BC_INOUT && x == 0) {
    // inlet: fr = f (f1, f5, f8 from Zou-He of the known totals), fb = 0
    const R u = inlet_u<R>(L, y);
    const R ck[9] = {1, 0, 1, 2, 1, 0, 2, 2, 0};
    R lt[9];
    for (int a = 0; a < 9; ++a) lt[a] = R(0.0);
    const int known[6] = {0, 2, 3, 4, 6, 7};
    for (int q = 0; q < 6; ++q) {
      const int k = known[q];
      const R drho = ck[k] / (1 - u);
      R v = lr[k];
      v += lr[1] * ((k == 3 ? R(1.0) : R(0.0)) + R(2.0 / 3.0) * u * drho);
      v += lr[5] * ((k == 7 ? R(1.0) : R(0.0)) - (k == 2 ? R(0.5) : R(0.0)) + (k == 4 ? R(0.5) : R(0.0)) + u / 6 * drho);
      v += lr[8] * ((k == 6 ? R(1.0) : R(0.0)) + (k == 2 ? R(0.5) : R(0.0)) - (k == 4 ? R(0.5) : R(0.0)) + u / 6 * drho);
      lt[k] = v;
    }
    for (int a = 0; a < 9; ++a) sr[a] = sb[a] = lt[a];
  } else if (L.bcx == BC_INOUT && x == L.nx - 1) {
    // outlet: known 0,1,2,4,5,8 pass through; f3, f6, f7 from Zou-He, split by frac = kR/kT
    const R* FR = A.fr;
    const R* FB = A.fb;
    const int known[6] = {0, 1, 2, 4, 5, 8};
    R kR = 0, kT = 0;
    for (int q = 0; q < 6; ++q) {
      kR += FR[known[q] * M + p];
      kT += FR[known[q] * M + p] + FB[known[q] * M + p];
    }
    const R frac = kT != 0 ? kR / kT : R(0.0);
    R lt[9], lfrac = 0;
    for (int a = 0; a < 9; ++a) lt[a] = R(0.0);
    const int unk[3] = {3, 6, 7};
    for (int q = 0; q < 3; ++q) {
      const int uu = unk[q];
      const R fu = FR[uu * M + p] + FB[uu * M + p];
      lt[uu] = frac * lr[uu] + (1 - frac) * lb[uu];   // adjoint of the total f_u
      lfrac += fu * (lr[uu] - lb[uu]);
    }
    // f3 = f1 + 2/3 r - 2/3 S, f7 = f5 + (f2 - f4)/2 + r/6 - S/6, f6 = f8 - (f2 - f4)/2 + r/6 - S/6,
    // S = f0 + f2 + f4 + 2 (f1 + f5 + f8)
    const R cs[9] = {1, 2, 1, 0, 1, 2, 0, 0, 2};
    R ltk[9];
    for (int a = 0; a < 9; ++a) ltk[a] = R(0.0);
    for (int q = 0; q < 6; ++q) {
      const int k = known[q];
      ltk[k] += lt[3] * ((k == 1 ? R(1.0) : R(0.0)) - R(2.0 / 3.0) * cs[k]);
      ltk[k] += lt[7] * ((k == 5 ? R(1.0) : R(0.0)) + (k == 2 ? R(0.5) : R(0.0)) - (k == 4 ? R(0.5) : R(0.0)) - cs[k] / 6);
      ltk[k] += lt[6] * ((k == 8 ? R(1.0) : R(0.0)) - (k == 2 ? R(0.5) : R(0.0)) + (k == 4 ? R(0.5) : R(0.0)) - cs[k] / 6);
    }
    for (int a = 0; a < 9; ++a) sr[a] = sb[a] = R(0.0);
    for (int q = 0; q < 6; ++q) {
      const int k = known[q];
      const R dfr = kT != 0 ? (kT - kR) / (kT * kT) : R(0.0);   // d frac / d s_R
      const R dfb = kT != 0 ? -kR / (kT * kT) : R(0.0);         // d frac / d s_B
      sr[k] = lr[k] + ltk[k] + lfrac * dfr;
      sb[k] = lb[k] + ltk[k] + lfrac * dfb;
    }
  } else {
    for (int a = 0; a < 9; ++a) {
      sr[a] = lr[a];
      sb[a] = lb[a];
    }
  }
  for (int a = 0; a < 9; ++a) {
    lam[(2 * a) * N + i] = sr[a];
    lam[(2 * a + 1) * N + i] = sb[a];
  }
}

inline int nblk(int n) { return (n + kAdjThreads - 1) / kAdjThreads; }

// Programmatic dependent launch.  The kernels of a reverse sweep are short, latency-bound
// grids, each depending on the one before it.  A kernel launched by launch_dep may be scheduled
// once every block of the kernel before it has run its dep_trigger (placed after all of a
// block's stores) or exited; its threads wait in dep_wait (the hardware's wait for the full
// completion and memory flush of that kernel) before they read anything.  So the next grid's
// launch overlaps the tail of the last one.  For a kernel launched the ordinary way both
// instructions do nothing.
__device__ __forceinline__ void dep_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void dep_trigger() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
template <typename... P, typename... Q>
cudaError_t launch_dep(void (*k)(P...), int grid, cudaStream_t st, Q... args) {
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3(unsigned(grid));
  cfg.blockDim = dim3(kAdjThreads);
  cfg.stream = st;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, k, args...);
}

// Forward intermediates of one state (the prologue of a segment's reverse sweep).
template <typename R>
__global__ void __launch_bounds__(kAdjThreads) k_fwd_local(AdjDevT<R> A) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < A.N) (fwd_local_body<R, false>(A, A.src, i, i));
}
template <typename R>
__global__ void __launch_bounds__(kAdjThreads) k_fwd_grad(AdjDevT<R> A) {
  dep_wait();
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < A.N) fwd_grad_node(A, i);
  dep_trigger();
}
template <typename R>
__global__ void __launch_bounds__(kAdjThreads) k_fwd_dn(AdjDevT<R> A) {
  dep_wait();
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < A.N) fwd_dn_node(A, i);
  dep_trigger();
}

// The reverse of step j (A) in three stages, each paired in one launch with the stage of the
// forward intermediates of the state before it (B, step j - 1) that has the same dependency on
// the neighbours: (adj_collide, fwd_local), (adj_normal, fwd_grad), (adj_rho, fwd_dn).  A and B
// share the reverse arrays and parameter adjoints but have their own forward intermediates
// and scatter targets, so the two halves of a launch touch disjoint data and run in separate
// blocks side by side: blocks [0, nrev) take the reverse stage, the rest (none for the first
// step of a segment, whose previous state is not recomputed yet) the forward stage.
template <typename R>
__global__ void __launch_bounds__(kAdjThreads) k_rev_collide(AdjDevT<R> A, AdjDevT<R> B, int nrev) {
  const bool rev = int(blockIdx.x) < nrev;
  const int i = (rev ? blockIdx.x : blockIdx.x - nrev) * blockDim.x + threadIdx.x;
  dep_wait();
  if (i < A.N) {
    if (rev) adj_collide_node(A, i);
    else (fwd_local_body<R, false>(B, B.src, i, i));
  }
  dep_trigger();
}
template <typename R>
__global__ void __launch_bounds__(kAdjThreads) k_rev_normal(AdjDevT<R> A, AdjDevT<R> B, int nrev) {
  const bool rev = int(blockIdx.x) < nrev;
  const int i = (rev ? blockIdx.x : blockIdx.x - nrev) * blockDim.x + threadIdx.x;
  dep_wait();
  if (i < A.N) {
    if (rev) adj_normal_node(A, i);
    else fwd_grad_node(B, i);
  }
  dep_trigger();
}
template <typename R>
__global__ void __launch_bounds__(kAdjThreads) k_rev_rho(AdjDevT<R> A, AdjDevT<R> B, int nrev) {
  const bool rev = int(blockIdx.x) < nrev;
  const int i = (rev ? blockIdx.x : blockIdx.x - nrev) * blockDim.x + threadIdx.x;
  dep_wait();
  if (i < A.N) {
    if (rev) adj_rho_body(A, A.lam, i, i, A.sol[i] != 0, A.lrnt[i]);
    else fwd_dn_node(B, i);
  }
  dep_trigger();
}
template <typename R>
__global__ void __launch_bounds__(kAdjThreads) k_adj_rho(AdjDevT<R> A) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < A.N) adj_rho_body(A, A.lam, i, i, A.sol[i] != 0, A.lrnt[i]);
}

// ------------------------------------------------------------------ resident reverse sweep
// A checkpoint segment's whole reverse sweep in one cooperative launch, on lattices that the
// resident step kernel holds: one block per tile of its plan, a thread per node for the reverse
// stages and, in warps of their own beside them, a thread per node for the forward intermediates.
// The stages reach at most two nodes beyond a node, so between two stages a block waits only for
// the tiles around it (the plan's neighbours, a flag per tile), as the step kernel does.
//
// Where the launched stages scatter with atomics and evaluate Eq. 29 on the fly (chains of
// dependent loads on every node next to a wall, which set the pace of the whole lattice: up to
// 20,000 cycles a stage), the tile plus two nodes all round is brought into shared memory in one
// round of loads: the virtual values of its solid nodes are filled in once for all readers, and
// the transposes are gathers (a node from the nodes that read it, a solid node likewise, its fluid
// neighbours their shares of it).  What only a node's own two threads use stays in shared memory.
// 400 x 42, FP32 forward and reverse, us per step of the whole gradient (800 steps): launched
// stages 33.8 (with the resident forward steps), resident with the launched stages' bodies 44.7,
// with tiles in shared memory 26.1, with the node's own values there too 24.0, beside the
// recompute 22.0; FP64 reverse of an FP32 forward 85 -> 57, FP64 both 124 -> 89; without a __threadfence before the
// releases 21.9 -> 20.2, 56.7 -> 55.4 and 81.8 -> 81.1.  What bounds it: three
// waits per reverse step (about 3,300 cycles each with the release before them) and the latency of
// the stages (6,100, 5,300 and 4,100 cycles for one or two warps per scheduler).
__device__ __forceinline__ void half_sync(int id, int n) { asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(n) : "memory"); }

// (FP32: held to 128 registers, so that two blocks of 128 threads fit on an SM beside two of the
// step kernel's that recompute the next segment: 24.0 -> 22.0 us per step on 400 x 42.)
template <typename R>
__global__ void __launch_bounds__(kRevMaxThreads, sizeof(R) == 4 ? 2 : 1) k_reverse(const __grid_constant__ RevRunT<R> P) {
  __shared__ int s_node[kRevMaxSlots];         // node of each slot of tile + 2 (wrapped or clamped)
  __shared__ uint8_t s_mask[kRevMaxSlots];     // its neighbour-solid mask
  __shared__ uint8_t s_kind[kRevMaxSlots];     // bit 0: solid, bit 1: beyond an open or closed edge
  __shared__ uint16_t s_list[kRevMaxSlots];    // solid slots of tile + 1
  __shared__ uint16_t s_ref[kRevMaxSlots];     // and the slot of the node each stands for
  __shared__ R s_den[kRevMaxSlots];            // and its Eq. 29 weight
  __shared__ R s_f[2][kRevMaxSlots];           // forward: the field of the stage (two components)
  __shared__ R s_q[3][kRevMaxSlots];           // reverse: what the stage gathers
  __shared__ R s_acc[2][kRevMaxSlots];         // reverse: a solid node's adjoint over its weight
  __shared__ int s_nlist;
  __shared__ AdjDevT<R> s_V[2];
  // what only the node's own threads use, in shared memory (dynamic): the two sets of forward
  // intermediates and the reverse arrays, M values each
  extern __shared__ __align__(16) unsigned char s_own[];
  const RunTile tl = P.tiles[blockIdx.x];
  const LatDev& L = P.V[0].L;
  const int nx = L.nx, ny = L.ny;
  const bool px = L.bcx == BC_PERIODIC, py = L.bcy == BC_PERIODIC, inout = L.bcx == BC_INOUT;
  const int half = blockDim.x / 2, u = threadIdx.x < half ? threadIdx.x : threadIdx.x - half;
  const bool rev = threadIdx.x < half;   // whole warps
  const bool mine = u < tl.tx * tl.ty;
  const int lx = u % tl.tx, ly = u / tl.tx, x = tl.x0 + lx, y = tl.y0 + ly;
  const int i = y * nx + x;
  const int CW = tl.tx + 4, CH = tl.ty + 4, ns = CW * CH;
  const int c = (ly + 2) * CW + lx + 2;   // this node's slot
  const int M = half;
  if (threadIdx.x == 0) {
    s_nlist = 0;
    R* w = reinterpret_cast<R*>(s_own);
    auto take = [&](int n) {
      R* r = w;
      w += n * M;
      return r;
    };
    for (int q = 0; q < 2; ++q) {
      AdjDevT<R>& V = s_V[q];
      V = P.V[q];
      V.M = M;
      V.fr = take(9);
      V.fb = take(9);
      V.rr = take(1);
      V.rb = take(1);
      V.grx = take(1);
      V.gry = take(1);
      V.gcx = take(1);
      V.gcy = take(1);
      V.dn = take(4);
    }
    R* const lf_r = take(9);
    R* const lf_b = take(9);
    R* const lr = take(5);
    int* const pick = reinterpret_cast<int*>(w);
    for (int q = 0; q < 2; ++q) {
      AdjDevT<R>& V = s_V[q];
      V.lf_r = lf_r;
      V.lf_b = lf_b;
      V.ln_x = lr;
      V.ln_y = lr + M;
      V.lg_x = lr + 2 * M;
      V.lg_y = lr + 3 * M;
      V.lrn = lr + 4 * M;
      V.pick = pick + q * M;
    }
  }
  __syncthreads();
  for (int k = threadIdx.x; k < ns; k += blockDim.x) {
    const int cx = k % CW, cy = k / CW;
    const int xr = tl.x0 + cx - 2, yr = tl.y0 + cy - 2;
    const int xm = wrap_or_clamp(xr, nx, px), ym = wrap_or_clamp(yr, ny, py);
    const int n = ym * nx + xm;
    const bool solid = P.V[0].sol[n] != 0, beyond = (!px && xm != xr) || (!py && ym != yr);
    s_node[k] = n;
    s_mask[k] = P.V[0].nbm[n];
    s_kind[k] = uint8_t((solid ? 1 : 0) | (beyond ? 2 : 0));
    s_f[0][k] = s_f[1][k] = s_q[0][k] = s_q[1][k] = s_q[2][k] = s_acc[0][k] = s_acc[1][k] = R(0.0);
    if (solid && cx >= 1 && cx < CW - 1 && cy >= 1 && cy < CH - 1) {
      const int m = atomicAdd(&s_nlist, 1);
      s_list[m] = uint16_t(k);
      s_ref[m] = uint16_t(k + (py ? 0 : ym - yr) * CW + (px ? 0 : xm - xr));
      R den = R(0.0);
      for (int b = 1; b < 9; ++b)
        if (!mask_bit(s_mask[k], b)) den = radd(den, wgt<R>(b));
      s_den[m] = den;
    }
  }
  __syncthreads();
  const int nlist = s_nlist;
  const bool solid = mine && (s_kind[c] & 1);
  // an open column's nodes are also read through the ghost column beyond it
  const int ghost = !mine || !inout ? 0 : (x == 0 ? -1 : (x == nx - 1 ? 1 : 0));

  unsigned phase = P.base;
  // the end of a stage: false once a wait of some thread of the block ran out
  auto arrive = [&] {
    __syncthreads();
    ++phase;
    if (threadIdx.x == 0) store_release(P.progress + blockIdx.x * kRunFlagStride, phase);
  };
  auto wait = [&]() -> bool {
    bool lost = false;
    for (int j = threadIdx.x; j < tl.nnb && !lost; j += blockDim.x)
      lost = !wait_reached(P.progress + P.nb[tl.nb0 + j] * kRunFlagStride, phase, P.poll_limit, P.err);
    if (__syncthreads_or(lost)) {
      if (threadIdx.x == 0) atomicOr(P.err, ERR_TIMEOUT);
      return false;
    }
    return true;
  };
  auto sync = [&]() -> bool {
    arrive();
    return wait();
  };
  // ---- forward half: a field (nf components) on tile + 2, its virtual values on the solid slots
  // of tile + 1 (the sums of read_field in its order)
  auto fill = [&](const R* v0, const R* v1) {
    for (int k = u; k < ns; k += half)
      if (!(s_kind[k] & 1)) {
        s_f[0][k] = __ldcg(v0 + s_node[k]);
        if (v1) s_f[1][k] = __ldcg(v1 + s_node[k]);
      }
    half_sync(2, half);
    for (int m = u; m < nlist; m += half) {
      const int k = s_list[m], r = s_ref[m];
      const unsigned msk = s_mask[k];
      R n0 = R(0.0), n1 = R(0.0);
#pragma unroll
      for (int b = 1; b < 9; ++b)
        if (!mask_bit(msk, b)) {
          n0 = radd(n0, rmul(wgt<R>(b), s_f[0][r + ey(b) * CW + ex(b)]));
          if (v1) n1 = radd(n1, rmul(wgt<R>(b), s_f[1][r + ey(b) * CW + ex(b)]));
        }
      const R den = s_den[m];
      s_f[0][k] = den > R(0.0) ? rdiv(n0, den) : R(0.0);
      if (v1) s_f[1][k] = den > R(0.0) ? rdiv(n1, den) : R(0.0);
    }
    half_sync(2, half);
  };
  auto fwd_grad = [&](const AdjDevT<R>& A) {
    fill(A.rn, nullptr);
    if (mine)
      fwd_grad_body(A, i, u, A.flags[L.node_off + (long long)y * L.pitch + x],
                    [&](int a) { return s_f[0][c + ey(a) * CW + ex(a)]; });
  };
  auto fwd_dn = [&](const AdjDevT<R>& A) {
    fill(A.nxv, A.nyv);
    if (mine)
      fwd_dn_body(A, u, solid, [&](int a) { return s_f[0][c + ey(a) * CW + ex(a)]; },
                  [&](int a) { return s_f[1][c + ey(a) * CW + ex(a)]; });
  };
  // ---- reverse half: what the readers of slot k (fluid nodes of the lattice) pass to it, of
  // sources (s0, s1) = adjoints of (d_x, d_y); g: only through a ghost beside column x = 0 (-1)
  // or nx - 1 (1), whose readers lie on that column
  auto readers = [&](const R* s0, const R* s1, int k, int g) {
    R v = R(0.0);
#pragma unroll
    for (int a = 1; a < 9; ++a) {
      if (g && ex(a) != g) continue;
      const int r = k - ey(a) * CW - ex(a);
      v += R(3.0) * wgt<R>(a) * (ex(a) * s0[r] + ey(a) * s1[r]);
    }
    return v;
  };
  // sources to shared memory (nq arrays), then the solid nodes' totals for nc components
  auto collect = [&](const R* q0, const R* q1, const R* q2, int nc) {
    for (int k = u; k < ns; k += half)
      if (s_kind[k] == 0) {
        s_q[0][k] = __ldcg(q0 + s_node[k]);
        s_q[1][k] = __ldcg(q1 + s_node[k]);
        if (q2) s_q[2][k] = __ldcg(q2 + s_node[k]);
      }
    half_sync(3, half);
    for (int m = u; m < nlist; m += half) {
      const int k = s_list[m];
      if (s_kind[k] & 2) continue;
      const int xs = s_node[k] % nx;
      const int g = !inout ? 0 : (xs == 0 ? -1 : (xs == nx - 1 ? 1 : 0));
      const R den = s_den[m], r = den > R(0.0) ? R(1.0) / den : R(0.0);
      for (int q = 0; q < nc; ++q) {
        R v = readers(s_q[q], s_q[q + 1], k, 0);
        if (g) v += readers(s_q[q], s_q[q + 1], k + g, g);
        s_acc[q][k] = v * r;
      }
    }
    half_sync(3, half);
  };
  // the adjoint of what this node's neighbours read of it, component q
  auto gather = [&](int q) {
    R v = readers(s_q[q], s_q[q + 1], c, 0);
    if (ghost) v += readers(s_q[q], s_q[q + 1], c + ghost, ghost);
    const unsigned msk = s_mask[c];
    if (msk) {
#pragma unroll
      for (int b = 1; b < 9; ++b) {
        const int k = c - ey(b) * CW - ex(b);
        if (s_kind[k] == 1) v += wgt<R>(b) * s_acc[q][k];
        if (ghost && ex(b) == ghost) {
          const int k2 = c + ghost - ey(b) * CW - ex(b);
          if (s_kind[k2] == 1) v += wgt<R>(b) * s_acc[q][k2];
        }
      }
    }
    return v;
  };

  // the two sets of forward intermediates take turns: step j reverses with set q while the
  // intermediates of state j - 1 go to the other.  Sources of the gathers: set 0's scatter
  // targets hold those of n (three arrays), set 1's those of rho^N (two).
  const char* src = P.states + (P.ns - 1) * P.stride;
  if (!rev && mine) fwd_local_body<R, true>(s_V[0], src, i, u);
  if (!sync()) return;
  if (!rev) fwd_grad(s_V[0]);
  if (!sync()) return;
  if (!rev) fwd_dn(s_V[0]);
  // the node's parameter adjoints, accumulated in double while the block waits
  double p_sigma = 0.0, p_hR = 0.0, p_hB = 0.0, p_theta = 0.0;
  const unsigned msk = mine ? s_mask[c] : 0u;
  __syncthreads();
  const R* lam_next = P.lam_next;
  R* lam = P.lam;
  int q = 0;
#pragma unroll 1
  for (int j = P.ns - 1; j >= 0; --j) {
    const AdjDevT<R>& A = s_V[q];
    const AdjDevT<R>& B = s_V[q ^ 1];
    const bool fwd = !rev && j > 0;
    src -= P.stride;
    R ds = R(0.0), dR = R(0.0), dB = R(0.0), dt = R(0.0);
    if (rev && mine)
      adj_collide_body<R, true>(A, lam_next, i, u, solid, msk, ds, dR, dB, P.V[0].lnt_x, P.V[0].lnt_y, P.V[0].lrnt);
    if (fwd && mine) fwd_local_body<R, true>(B, src, i, u);
    arrive();
    p_sigma += ds;
    p_hR += dR;
    p_hB += dB;
    if (!wait()) return;
    if (rev) {
      collect(P.V[0].lnt_x, P.V[0].lnt_y, P.V[0].lrnt, 2);
      if (mine) {
        R lrx, lry;
        adj_normal_body(A, i, u, solid, gather(0), gather(1), lrx, lry, dt);
        P.V[1].lnt_x[i] = lrx;
        P.V[1].lnt_y[i] = lry;
      }
    }
    if (fwd) fwd_grad(B);
    arrive();
    p_theta += dt;
    if (!wait()) return;
    if (rev) {
      collect(P.V[1].lnt_x, P.V[1].lnt_y, nullptr, 1);
      if (mine) adj_rho_body(A, lam, i, u, solid, gather(0));
    }
    if (fwd) fwd_dn(B);
    if (j > 0 && !sync()) return;
    R* const l = lam;
    lam = const_cast<R*>(lam_next);
    lam_next = l;
    q ^= 1;
  }
  if (rev && mine && !solid) {
    P.V[0].p_sigma[i] += p_sigma;
    P.V[0].p_hR[i] += p_hR;
    P.V[0].p_hB[i] += p_hB;
    P.V[0].p_theta[i] += p_theta;
  }
}

// Seed for an objective J = sum_x c(x) rho^N(x) of the stored state: lam = dJ/d(state).
template <typename R>
__global__ void __launch_bounds__(kAdjThreads) k_seed_weighted(AdjDevT<R> A, const R* c) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= A.N) return;
  const int N = A.N;
  for (int a = 0; a < 9; ++a) A.lf_r[a * N + i] = A.lf_b[a * N + i] = R(0.0);
  const int x = i % A.L.nx, y = i / A.L.nx;
  A.lrn[i] = is_solid(A, x, y) ? R(0.0) : c[i];
}

// Seed for J = sum over fluid nodes of rho_R = sum_a f_a,R (the red mass) of the stored state.
template <typename R>
__global__ void __launch_bounds__(kAdjThreads) k_seed_red_mass(AdjDevT<R> A) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= A.N) return;
  const int N = A.N;
  const int x = i % A.L.nx, y = i / A.L.nx;
  const R one = is_solid(A, x, y) ? R(0.0) : R(1.0);
  for (int a = 0; a < 9; ++a) {
    A.lf_r[a * N + i] = one;
    A.lf_b[a * N + i] = R(0.0);
  }
  A.lrn[i] = R(0.0);
}

}  // namespace

// Forward intermediates of the state A.src (three kernels: the prologue of a segment).
template <typename R>
cudaError_t adjoint_forward(const AdjDevT<R>& A, cudaStream_t st) {
  const int b = nblk(A.N);
  k_fwd_local<R><<<b, kAdjThreads, 0, st>>>(A);
  cudaError_t e = cudaGetLastError();
  if (e == cudaSuccess) e = launch_dep(k_fwd_grad<R>, b, st, A);
  if (e == cudaSuccess) e = launch_dep(k_fwd_dn<R>, b, st, A);
  return e;
}

// One reverse step: lam <- (d step / d state)^T lam_next, parameter adjoints accumulated,
// from the forward intermediates of A's state (computed by the previous call, or by
// adjoint_forward); with B non-null the same three kernels compute B's intermediates.
template <typename R>
cudaError_t adjoint_step(const AdjDevT<R>& A, const AdjDevT<R>* B, cudaStream_t st) {
  const int b = nblk(A.N);
  const AdjDevT<R>& Bv = B ? *B : A;
  const int g = B ? 2 * b : b;
  cudaError_t e = launch_dep(k_rev_collide<R>, g, st, A, Bv, b);
  if (e == cudaSuccess) e = launch_dep(k_rev_normal<R>, g, st, A, Bv, b);
  if (e == cudaSuccess) e = launch_dep(k_rev_rho<R>, g, st, A, Bv, b);
  return e;
}

template <typename R>
cudaError_t adjoint_seed(const AdjDevT<R>& A, const R* c, bool red_mass, cudaStream_t st) {
  const int b = nblk(A.N);
  k_fwd_local<R><<<b, kAdjThreads, 0, st>>>(A);   // also clears lrnt
  if (red_mass) k_seed_red_mass<R><<<b, kAdjThreads, 0, st>>>(A);
  else k_seed_weighted<R><<<b, kAdjThreads, 0, st>>>(A, c);
  k_adj_rho<R><<<b, kAdjThreads, 0, st>>>(A);
  return cudaGetLastError();
}

// 2 sets of 28 intermediates, 23 reverse values and 2 picks per node of the block
template <typename R>
static size_t reverse_smem(int threads) { return size_t(threads / 2) * ((2 * 28 + 23) * sizeof(R) + 2 * sizeof(int)); }

template <typename R>
cudaError_t launch_reverse(const RevRunT<R>& P, int ntiles, int threads, cudaStream_t st) {
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeCooperative;   // every block resident: they wait for one another
  at[0].val.cooperative = 1;
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3(unsigned(ntiles));
  cfg.blockDim = dim3(unsigned(threads));
  cfg.dynamicSmemBytes = reverse_smem<R>(threads);
  cfg.stream = st;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, k_reverse<R>, P);
}
template <typename R>
cudaError_t reverse_blocks(int threads, int* per_sm) {
  const cudaError_t e = allow_max_smem(k_reverse<R>);
  if (e != cudaSuccess) return e;
  return cudaOccupancyMaxActiveBlocksPerMultiprocessor(per_sm, k_reverse<R>, threads, reverse_smem<R>(threads));
}
template cudaError_t launch_reverse<double>(const RevRunT<double>&, int, int, cudaStream_t);
template cudaError_t launch_reverse<float>(const RevRunT<float>&, int, int, cudaStream_t);
template cudaError_t reverse_blocks<double>(int, int*);
template cudaError_t reverse_blocks<float>(int, int*);
template cudaError_t adjoint_forward<double>(const AdjDevT<double>&, cudaStream_t);
template cudaError_t adjoint_forward<float>(const AdjDevT<float>&, cudaStream_t);
template cudaError_t adjoint_step<double>(const AdjDevT<double>&, const AdjDevT<double>*, cudaStream_t);
template cudaError_t adjoint_step<float>(const AdjDevT<float>&, const AdjDevT<float>*, cudaStream_t);
template cudaError_t adjoint_seed<double>(const AdjDevT<double>&, const double*, bool, cudaStream_t);
template cudaError_t adjoint_seed<float>(const AdjDevT<float>&, const float*, bool, cudaStream_t);

}  // namespace lbcg
