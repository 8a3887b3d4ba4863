// The arithmetic of one node of the step (arXiv 1707.00198, Sec. II), shared by the tile kernel
// (one launch per step) and the resident kernel (many steps per launch): the same inlined
// functions, so that both give the same bits.
#pragma once

#include "lbcg_device.cuh"

namespace lbcg {

// Every multiplication, addition and fused multiply-add is written out (rmul, radd, fma_): the
// compiler contracts nothing by itself, so that the kernels that share this code agree bit for
// bit.
//
// On this GPU an FP64 instruction of a warp takes about 19 cycles of its SM (64 if the warp is
// alone on it) whatever its active lanes; a division is 9 of them, a square root 10, a
// reciprocal square root 6 (measured with one block of 1 to 16 warps).  So the FP64 forms below
// are written for few operations: one reciprocal instead of divisions, constants folded on
// entry, and the collision in moment space (back to populations once, from the relaxed
// moments).  FP32 keeps the form f' = f - M^-1 Delta, whose rounding error is the smaller.
// Arithmetic helpers: IEEE reciprocals in FP64; the FP32-arithmetic instantiations use the
// hardware reciprocal and reciprocal square root.
template <typename T>
__device__ __forceinline__ T rcp_(T x) {
  if constexpr (sizeof(T) == 4) return __fdividef(1.0f, x);
  else return __drcp_rn(x);
}

// rho^N (Eq. 12), the colour densities and 1 / rho: exactly +-1 on single-colour nodes
template <typename T>
__device__ __forceinline__ T indicator(const T fr[9], const T fb[9], T& sr, T& sb, T& irho) {
  sr = fr[0];
  sb = fb[0];
#pragma unroll
  for (int a = 1; a < 9; ++a) {
    sr = radd(sr, fr[a]);
    sb = radd(sb, fb[a]);
  }
  irho = rcp_(radd(sr, sb));
  const T v = rmul(rsub(sr, sb), irho);
  return sb == T(0) ? T(1) : (sr == T(0) ? T(-1) : v);
}

// The stencil sums of Eq. 28 of a field, 36 times over in FP64 (fewer operations): c points at
// the node's value in a row-major array whose rows are `w` apart
template <typename T>
__device__ __forceinline__ void stencil(const T* c, int w, T& dx, T& dy) {
  if constexpr (sizeof(T) == 8) {
    const T p = rsub(c[w + 1], c[-w - 1]), q = rsub(c[w - 1], c[-w + 1]);   // along the diagonals
    dx = fma_(T(4), rsub(c[1], c[-1]), rsub(p, q));
    dy = fma_(T(4), rsub(c[w], c[-w]), radd(p, q));
  } else {
    dx = rmul(wgt<T>(1), c[1]);
    dy = rmul(wgt<T>(2), c[w]);
#pragma unroll
    for (int a = 3; a < 9; ++a) {
      const T v = c[ey(a) * w + ex(a)];
      if (ex(a)) dx = fma_(T(ex(a)) * wgt<T>(a), v, dx);
      if (ey(a)) dy = fma_(T(ey(a)) * wgt<T>(a), v, dy);
    }
  }
}
// what `stencil` returns for a unit gradient, times c_s^2
template <typename T>
constexpr T kStencilScale = sizeof(T) == 8 ? T(12) : T(1) / T(3);

// grad rho^N (Eq. 28) and n at a bulk node; eps2 = grad_eps^2
template <typename T>
__device__ __forceinline__ void grad_normal(const T* c, int w, T eps2, T& ax, T& ay, T& nxv, T& nyv) {
  stencil(c, w, ax, ay);
  constexpr T k = sizeof(T) == 8 ? T(1.0 / 12.0) : T(3);
  ax = rmul(ax, k);
  ay = rmul(ay, k);
  nxv = nyv = T(0);
  const T m2 = fma_(ax, ax, rmul(ay, ay));
  if (m2 > eps2) {
    T inv;
    if constexpr (sizeof(T) == 4) inv = rsqrtf(m2);
    else inv = rsqrt(m2);
    nxv = rmul(ax, inv);
    nyv = rmul(ay, inv);
  }
}

// d_x n_x, d_x n_y, d_y n_x, d_y n_y at the scale of `stencil`; cx, cy point at the node's n
template <typename T>
__device__ __forceinline__ void grad_n(const T* cx, const T* cy, int w, T& dxx, T& dyx, T& dxy, T& dyy) {
  stencil(cx, w, dxx, dxy);
  stencil(cy, w, dyx, dyy);
}

// Eq. 48, wetting scheme (b) (lbcg_params.wetting = 1): grad n at an outermost fluid node from
// its fluid neighbours only, d_i n = sum_a w_a (n(x + e_a) - n(x)) e_ai / sum_a w_a e_ai^2 over
// the directions a whose neighbour is fluid (bit a-1 of `solid` clear).  nxs/nys[a] hold n at
// x + e_a (a = 0: the node).  Returned times `scale`, the scale of the caller's Eq. 28 sums.
template <typename T>
__device__ __forceinline__ void grad_n_scheme_b(const T nxs[9], const T nys[9], unsigned solid, T scale, T& dxx, T& dyx,
                                                T& dxy, T& dyy) {
  T sxx = T(0), syx = T(0), sxy = T(0), syy = T(0), wx = T(0), wy = T(0);
#pragma unroll
  for (int a = 1; a < 9; ++a) {
    if ((solid >> (a - 1)) & 1u) continue;
    const T w = wgt<T>(a), ddx = rsub(nxs[a], nxs[0]), ddy = rsub(nys[a], nys[0]);
    if (ex(a)) {
      sxx = fma_(T(ex(a)) * w, ddx, sxx);
      syx = fma_(T(ex(a)) * w, ddy, syx);
      wx = radd(wx, w);
    }
    if (ey(a)) {
      sxy = fma_(T(ey(a)) * w, ddx, sxy);
      syy = fma_(T(ey(a)) * w, ddy, syy);
      wy = radd(wy, w);
    }
  }
  dxx = wx > T(0) ? rmul(rdiv(sxx, wx), scale) : T(0);
  dyx = wx > T(0) ? rmul(rdiv(syx, wx), scale) : T(0);
  dxy = wy > T(0) ? rmul(rdiv(sxy, wy), scale) : T(0);
  dyy = wy > T(0) ? rmul(rdiv(syy, wy), scale) : T(0);
}

// Step constants as the collision uses them (from LatConst, once per thread)
template <typename T>
struct Collide {
  T ks, beta;                 // of the force: see csf_force
  T hlow, hdiff, hsign, hR, hB;   // Eq. 18, see viscous_rate
  T e1, e2, e3, e4, p1, p2, p3, p4, q1, q2, q3;
  __device__ __forceinline__ explicit Collide(const LatConst<T>& c) {
    beta = c.beta;
    hR = c.h_inv_nuR;
    hB = c.h_inv_nuB;
    const T se = c.s_e, sp = c.s_eps, sq = c.s_q;
    const T ce = fma_(T(-0.5), se, T(1)), cp = fma_(T(-0.5), sp, T(1)), cq = fma_(T(-0.5), sq, T(1));
    if constexpr (sizeof(T) == 8) {
      ks = rmul(c.sigma, T(1.0 / 24.0));
      const bool red = c.h_inv_nuR >= c.h_inv_nuB;
      hsign = red ? T(1) : T(-1);
      hlow = rmul(T(2), red ? c.h_inv_nuB : c.h_inv_nuR);
      hdiff = fabs(rsub(c.h_inv_nuR, c.h_inv_nuB));
      // relaxed e, eps and q moments with the weights of M^-1 (1/36, 1/36, 1/12) folded in:
      // e'/36 = e1 e + e2 rho u.u + e3 rho + e4 u.F, and so on
      constexpr T r36 = T(1) / T(36), r12 = T(1) / T(12);
      e1 = rmul(rsub(T(1), se), r36);
      e2 = rmul(rmul(T(3), se), r36);
      e3 = rmul(rmul(T(-2), se), r36);
      e4 = rmul(rmul(T(6), ce), r36);
      p1 = rmul(rsub(T(1), sp), r36);
      p2 = rmul(rmul(T(-3), sp), r36);
      p3 = rmul(sp, r36);
      p4 = rmul(rmul(T(-6), cp), r36);
      q1 = rmul(rsub(T(1), sq), r12);
      q2 = rmul(-sq, r12);
      q3 = rmul(-cq, r12);
    } else {
      ks = rmul(T(0.5), c.sigma);
      e1 = se;
      e4 = ce;
      p1 = sp;
      p4 = cp;
      q1 = sq;
      q3 = cq;
      hlow = hdiff = hsign = e2 = e3 = p2 = p3 = q2 = T(0);   // FP64 form only
    }
  }
};

// Force of a node (Eq. 10, 13) from grad n as grad_n returns it
template <typename T>
__device__ __forceinline__ void csf_force(T gx, T gy, T nx, T ny, T dxx, T dyx, T dxy, T dyy, const Collide<T>& c,
                                          T& Fx, T& Fy) {
  T hsk;
  if constexpr (sizeof(T) == 8) {
    const T u = fma_(-nx, dyy, rmul(ny, radd(dxy, dyx)));
    hsk = rmul(c.ks, fma_(nx, u, rmul(-rmul(ny, ny), dxx)));
  } else {
    const T d = fma_(rmul(-nx, nx), dyy, rmul(-rmul(ny, ny), dxx));
    hsk = rmul(c.ks, rmul(T(3), fma_(rmul(nx, ny), radd(dxy, dyx), d)));
  }
  Fx = rmul(hsk, gx);
  Fy = rmul(hsk, gy);
}

// Moments of the totals f_a (Eq. 3 rows 2-9; the last one read as e_x e_y)
template <typename T>
struct Moments {
  T e, eps, jx, jy, qx, qy, pxx, pxy;
  __device__ __forceinline__ void of(const T f[9]) {
    if constexpr (sizeof(T) == 8) {
      const T p13 = radd(f[1], f[3]), m13 = rsub(f[1], f[3]), p24 = radd(f[2], f[4]), m24 = rsub(f[2], f[4]);
      const T p57 = radd(f[5], f[7]), m57 = rsub(f[5], f[7]), p68 = radd(f[6], f[8]), m68 = rsub(f[6], f[8]);
      const T s14 = radd(p13, p24), s58 = radd(p57, p68), bx = rsub(m57, m68), by = radd(m57, m68);
      pxx = rsub(p13, p24);
      pxy = rsub(p57, p68);
      jx = radd(m13, bx);
      jy = radd(m24, by);
      qx = fma_(T(-2), m13, bx);
      qy = fma_(T(-2), m24, by);
      e = fma_(T(-4), f[0], fma_(T(2), s58, -s14));
      eps = fma_(T(4), f[0], fma_(T(-2), s14, s58));
    } else {
      const T m13 = rsub(f[1], f[3]), m24 = rsub(f[2], f[4]);
      const T s14 = radd(radd(radd(f[1], f[2]), f[3]), f[4]), s58 = radd(radd(radd(f[5], f[6]), f[7]), f[8]);
      const T u = rsub(f[5], f[6]), v = radd(f[5], f[6]);
      jx = radd(rsub(rsub(radd(m13, f[5]), f[6]), f[7]), f[8]);
      jy = rsub(rsub(radd(radd(m24, f[5]), f[6]), f[7]), f[8]);
      qx = fma_(T(-2), m13, radd(rsub(u, f[7]), f[8]));
      qy = fma_(T(-2), m24, rsub(rsub(v, f[7]), f[8]));
      pxx = rsub(radd(rsub(f[1], f[2]), f[3]), f[4]);
      pxy = rsub(radd(u, f[7]), f[8]);
      e = fma_(T(2), s58, fma_(T(-4), f[0], -s14));
      eps = radd(fma_(T(4), f[0], rmul(T(-2), s14)), s58);
    }
  }
};

// FP64: the e and eps moments relaxed towards their values at rest and weighted, what the
// collision needs of them apart from u and F
__device__ __forceinline__ void relax_rest(Moments<double>& m, double rho, const Collide<double>& c) {
  m.e = fma_(c.e1, m.e, rmul(c.e3, rho));
  m.eps = fma_(c.p1, m.eps, rmul(c.p3, rho));
}

// s_v = 1/tau_v = 1/(3 nu + 1/2) (Eq. 5) with the harmonic viscosity of Eq. 18.  FP64: 1 / nu as the
// smaller of the two plus their difference's share, two operations for four, exact in pure fluid on
// that side (as the sum of the halves plus rho^N times half their difference, one operation, pure
// fluid of the smaller 1 / nu was off by the last bits of the larger; 100 x 50 10.57 us per step, now
// 10.64, 1200 x 80 35.2, now 35.4).
template <typename T>
__device__ __forceinline__ T viscous_rate(T rn, const Collide<T>& c) {
  T inv_nu;
  if constexpr (sizeof(T) == 8) inv_nu = fma_(fma_(c.hsign, rn, T(1)), c.hdiff, c.hlow);
  else inv_nu = fma_(radd(T(1), rn), c.hR, rmul(rsub(T(1), rn), c.hB));
  return rmul(inv_nu, rcp_(fma_(T(0.5), inv_nu, T(3))));
}

// Velocity (Eq. 17)
template <typename T>
__device__ __forceinline__ void velocity(const Moments<T>& m, T irho, T Fx, T Fy, T& ux, T& uy) {
  ux = rmul(fma_(T(0.5), Fx, m.jx), irho);
  uy = rmul(fma_(T(0.5), Fy, m.jy), irho);
}

// MRT collision with Guo forcing (Eq. 1-9): f' from the totals f (FP32; unused in FP64) or their
// moments (FP64: after relax_rest).  M^-1 = M^T diag(1/9, 1/36, 1/36, 1/6, 1/12, 1/6, 1/12, 1/4, 1/4); s_rho = s_j = 1
// (Eq. 6), so the momentum changes by exactly F.
template <typename T>
__device__ __forceinline__ void collide_node(const T* f, const Moments<T>& m, T rho, T irho, T sv, T Fx, T Fy,
                                             const Collide<T>& c, T fp[9]) {
  if constexpr (sizeof(T) == 8) {
    const T Jx = fma_(T(0.5), Fx, m.jx), Jy = fma_(T(0.5), Fy, m.jy);   // rho u
    const T ux = rmul(Jx, irho), uy = rmul(Jy, irho);
    const T yy = rmul(Jy, uy), uyF = rmul(uy, Fy);
    const T uu = fma_(Jx, ux, yy), dd = fma_(Jx, ux, -yy);             // rho u.u, rho (ux^2 - uy^2)
    const T uF = fma_(ux, Fx, uyF), dF = fma_(ux, Fx, -uyF), cF = fma_(ux, Fy, rmul(uy, Fx));
    const T ae = fma_(c.e2, uu, fma_(c.e4, uF, m.e));
    const T ap = fma_(c.p2, uu, fma_(c.p4, uF, m.eps));
    const T aqx = fma_(c.q1, m.qx, fma_(c.q2, Jx, rmul(c.q3, Fx)));
    const T aqy = fma_(c.q1, m.qy, fma_(c.q2, Jy, rmul(c.q3, Fy)));
    const T ajx = rmul(radd(m.jx, Fx), T(1.0 / 6.0)), ajy = rmul(radd(m.jy, Fy), T(1.0 / 6.0));
    // p'/4 = (1 - sv)/4 p + sv/4 p_eq + (1 - sv/2)/4 p_F
    const T s4 = rmul(T(0.25), sv), r4 = rsub(T(0.25), s4), c2 = rsub(T(0.5), s4);
    const T axx = fma_(r4, m.pxx, fma_(s4, dd, rmul(c2, dF)));
    const T axy = fma_(r4, m.pxy, fma_(s4, rmul(Jx, uy), rmul(rmul(T(0.5), c2), cF)));
    const T c0 = rmul(rho, T(1.0 / 9.0));
    fp[0] = fma_(T(4), rsub(ap, ae), c0);
    const T c14 = fma_(T(-2), ap, rsub(c0, ae)), c58 = fma_(T(2), ae, radd(c0, ap));
    const T t13 = radd(c14, axx), t24 = rsub(c14, axx), tp = radd(c58, axy), tq = rsub(c58, axy);
    const T U = fma_(T(-2), aqx, ajx), V = fma_(T(-2), aqy, ajy);
    const T X = radd(ajx, aqx), Y = radd(ajy, aqy), P = radd(X, Y), Q = rsub(X, Y);
    fp[1] = radd(t13, U);
    fp[3] = rsub(t13, U);
    fp[2] = radd(t24, V);
    fp[4] = rsub(t24, V);
    fp[5] = radd(tp, P);
    fp[7] = rsub(tp, P);
    fp[6] = rsub(tq, Q);
    fp[8] = radd(tq, Q);
  } else {
    T ux, uy;
    velocity(m, irho, Fx, Fy, ux, uy);
    const T u2 = fma_(ux, ux, rmul(uy, uy)), u6F = rmul(T(6), fma_(ux, Fx, rmul(uy, Fy)));
    const T csv = fma_(T(-0.5), sv, T(1)), jxu = rmul(rho, ux);
    // Delta_k = s_k (m_k - m_k^eq) - (1 - s_k/2) (M F~)_k  with M F~ =
    // (0, 6 u.F, -6 u.F, Fx, -Fx, Fy, -Fy, 2(ux Fx - uy Fy), ux Fy + uy Fx)   (Eq. 8-9)
    const T De = fma_(c.e1, fma_(-rho, fma_(T(3), u2, T(-2)), m.e), rmul(-c.e4, u6F));
    const T Dp = fma_(c.p4, u6F, rmul(c.p1, fma_(-rho, fma_(T(-3), u2, T(1)), m.eps)));
    const T Dqx = fma_(c.q3, Fx, rmul(c.q1, radd(jxu, m.qx)));
    const T Dqy = fma_(c.q3, Fy, rmul(c.q1, fma_(rho, uy, m.qy)));
    const T Dxx = fma_(sv, fma_(-rho, fma_(ux, ux, rmul(-uy, uy)), m.pxx),
                       rmul(-csv, rmul(T(2), fma_(ux, Fx, rmul(-uy, Fy)))));
    const T Dxy = fma_(sv, fma_(-jxu, uy, m.pxy), rmul(-csv, fma_(ux, Fy, rmul(uy, Fx))));
    constexpr T k36 = T(1.0 / 36.0), k6 = T(1.0 / 6.0), k12 = T(1.0 / 12.0);
    const T ae = rmul(De, k36), ap = rmul(Dp, k36), aqx = rmul(Dqx, k12), aqy = rmul(Dqy, k12);
    const T axx = rmul(Dxx, T(0.25)), axy = rmul(Dxy, T(0.25));
    const T c14 = fma_(T(-2), ap, -ae), c58 = fma_(T(2), ae, ap);
    fp[0] = rsub(f[0], fma_(T(-4), ae, rmul(T(4), ap)));
    fp[1] = rsub(f[1], radd(fma_(T(-2), aqx, fma_(-Fx, k6, c14)), axx));
    fp[2] = rsub(f[2], rsub(fma_(T(-2), aqy, fma_(-Fy, k6, c14)), axx));
    fp[3] = rsub(f[3], radd(fma_(T(2), aqx, fma_(Fx, k6, c14)), axx));
    fp[4] = rsub(f[4], rsub(fma_(T(2), aqy, fma_(Fy, k6, c14)), axx));
    const T xp = radd(fma_(-Fx, k6, c58), aqx), xm = rsub(fma_(Fx, k6, c58), aqx);
    fp[5] = rsub(f[5], radd(radd(fma_(-Fy, k6, xp), aqy), axy));
    fp[6] = rsub(f[6], rsub(radd(fma_(-Fy, k6, xm), aqy), axy));
    fp[7] = rsub(f[7], radd(rsub(fma_(Fy, k6, xm), aqy), axy));
    fp[8] = rsub(f[8], rsub(rsub(fma_(Fy, k6, xp), aqy), axy));
  }
}

// Recolouring (Eq. 14; the blue line with the minus sign): oR_a = cR f'_a + w_a pc e_a.n,
// oB_a = cB f'_a - the same
template <typename T>
struct Recolour {
  T cR, cB, c1, c2, nx, ny;
  __device__ __forceinline__ Recolour(T rhoR, T rhoB, T irho, T nx_, T ny_, const Collide<T>& c) : nx(nx_), ny(ny_) {
    cR = rmul(rhoR, irho);
    cB = rmul(rhoB, irho);
    const T pc = rmul(rmul(rmul(c.beta, rhoR), rhoB), irho);
    c1 = rmul(pc, wgt<T>(1));
    c2 = rmul(pc, wgt<T>(5));
  }
  __device__ __forceinline__ void out(int a, const T fp[9], T& oR, T& oB) const {
    if (a == 0) {
      oR = rmul(cR, fp[0]);
      oB = rmul(cB, fp[0]);
      return;
    }
    const T en = a == 1 ? nx : (a == 2 ? ny : (a == 3 ? -nx : (a == 4 ? -ny : (a == 5 ? radd(nx, ny)
                 : (a == 6 ? rsub(ny, nx) : (a == 7 ? -radd(nx, ny) : rsub(nx, ny)))))));
    const T p = rmul(a < 5 ? c1 : c2, en);
    oR = fma_(cR, fp[a], p);
    oB = fma_(cB, fp[a], -p);
  }
};

// Virtual value of Eq. 29 on an outermost solid node: the weighted mean of `val` over its fluid
// neighbours (local indices q, kWallNone where the neighbour is solid); den: virtual_weight(q).  Divided in
// FP64 too: equal neighbours give equal values, and what Eq. 36 picks between can hang on the last bit.
template <typename T>
__device__ __forceinline__ T virtual_weight(const uint16_t q[8]) {
  T den = T(0);
#pragma unroll
  for (int b = 1; b < 9; ++b)
    if (q[b - 1] != kWallNone) den = radd(den, wgt<T>(b));
  return den;
}
// What a sum of n over the fluid neighbours is divided by (FP32) or multiplied with (FP64: the
// reciprocal, 1 operation instead of 9), from the weight
template <typename T>
__device__ __forceinline__ T mean_factor(T den) {
  if constexpr (sizeof(T) == 8) return rcp_(den);
  else return den;
}
template <typename T>
__device__ __forceinline__ T mean_of(T num, T factor) {
  if constexpr (sizeof(T) == 8) return rmul(num, factor);
  else return rdiv(num, factor);
}
template <typename T>
__device__ __forceinline__ T virtual_value(const WallSten& q, const T* val, T den) {
  T num = T(0);
#pragma unroll
  for (int b = 1; b < 9; ++b)
    if (q.i[b - 1] != kWallNone) num = radd(num, rmul(wgt<T>(b), val[q.i[b - 1]]));
  return rdiv(num, den);
}

// The two candidates of Eq. 34 on an outermost fluid node (rotations by +theta and -theta)
template <typename T>
__device__ __forceinline__ void wall_candidates(T nsx, T nsy, T c, T s, T& f1x, T& f1y, T& f2x, T& f2y) {
  f1x = rsub(rmul(nsx, c), rmul(nsy, s));
  f1y = radd(rmul(nsx, s), rmul(nsy, c));
  f2x = radd(rmul(nsx, c), rmul(nsy, s));
  f2y = radd(rmul(-nsx, s), rmul(nsy, c));
}

// FP64: whether two squared distances of Eq. 35 (at most 4) are equal but for their rounding and that of
// the steps before them, a few 1e-15.  The pick of Eq. 36 then follows the operations as the equations
// have them (square roots, divisions), in the oracle's order: next to a wall at 90 degrees a gradient
// along the wall's normal is such a tie, and n would point along the wall one way or the other.
template <typename T>
__device__ __forceinline__ bool near_tie(T d1, T d2) {
  return fabs(rsub(d1, d2)) <= T(1e-13);
}

// wall_normal (below) by two neighbouring lanes, r = 0 for x and r = 1 for y: each takes its
// component's sums, quotients and one of the two distances, the same operations on the same
// values.  (A warp's FP64 operation costs the same for one lane as for 32, and the chain is the
// longest of the step.)  f1, f2: this component of the candidates; d_x, d_y: candidate r + 1.
// All 32 lanes of the warp call it.
template <typename T>
__device__ __forceinline__ void wall_normal_pair(T eps, int wetting, bool unit, T f1, T f2, T cx, T cy, const WallSten& q,
                                                 const T* val, int r, T& cg, T& n) {
  auto v = [&](int a) { return rmul(wgt<T>(a), val[q.i[a - 1]]); };
  T g = rmul(wgt<T>(1), val[q.i[r]]);
  g = radd(g, -rmul(wgt<T>(1), val[q.i[r + 2]]));
  g = radd(g, v(5));
  const T v6 = v(6), v8 = v(8);
  g = radd(g, r ? v6 : -v6);
  g = radd(g, -v(7));
  g = radd(g, r ? -v8 : v8);
  [[maybe_unused]] const T sum = g;
  if constexpr (sizeof(T) == 8) g = rmul(g, T(3));
  else g = rdiv(g, T(1.0 / 3.0));
  auto other = [](T x) { return __shfl_xor_sync(0xFFFFFFFFu, x, 1); };
  T sq = rmul(g, g);
  cg = g;
  n = T(0);
  if constexpr (sizeof(T) == 8) {   // as wall_normal's FP64 form
    const T m2 = radd(sq, other(sq)), inv = rsqrt(m2), mag = rmul(m2, inv);
    const bool on = mag > eps;
    const T es = rmul(g, inv), eo = other(es);
    if (wetting == 2) {
      if (on) n = es;
      return;
    }
    const T a1 = rsub(cx, r ? eo : es), b1 = rsub(cy, r ? es : eo);
    const T d = radd(rmul(a1, a1), rmul(b1, b1)), od = other(d);
    bool one = r ? od <= d : d <= od;
    const bool close = !unit || near_tie(d, od);
    if (__any_sync(0xFFFFFFFFu, close)) {
      const T ge = rdiv(sum, T(1.0 / 3.0)), gge = rmul(ge, ge), mage = rsqrt_(radd(gge, other(gge)));
      const T ese = rdiv(ge, on ? mage : T(1)), eoe = other(ese);
      const T ae = rsub(cx, r ? eoe : ese), be = rsub(cy, r ? ese : eoe);
      const T de = rsqrt_(radd(rmul(ae, ae), rmul(be, be))), ode = other(de);
      if (close) one = r ? ode <= de : de <= ode;
    }
    const T nf = one ? f1 : f2;
    if (on) {
      cg = rmul(mag, nf);
      n = nf;
    }
    if (!unit) {   // uniform over the block
      sq = rmul(cg, cg);
      const T m2 = rsqrt_(radd(sq, other(sq)));
      if (on) n = m2 > eps ? rdiv(cg, m2) : T(0);
    }
  } else {
    const T mag = rsqrt_(radd(sq, other(sq)));
    const bool on = mag > eps;
    const T es = rdiv(g, on ? mag : T(1)), eo = other(es);
    if (wetting == 2) {   // uniform over the block
      if (on) n = es;     // no geometric correction: n from the raw gradient
      return;
    }
    const T a1 = rsub(cx, r ? eo : es), b1 = rsub(cy, r ? es : eo);
    const T d = rsqrt_(radd(rmul(a1, a1), rmul(b1, b1))), od = other(d);
    const bool one = r ? od <= d : d <= od;
    const T cc = rmul(mag, one ? f1 : f2);
    sq = rmul(cc, cc);
    const T m2 = rsqrt_(radd(sq, other(sq)));
    if (on) {
      cg = cc;
      if (m2 > eps) n = rdiv(cc, m2);
    }
  }
}

// Eq. 28 on an outermost fluid node from the shared values of its 8 neighbours, then the
// contact-angle correction of Eq. 30-36 -> corrected gradient and unit normal.  The sums run
// in the oracle's order (directions 1..8, products w*phi then sign), so that a gradient exactly
// along the wall's normal makes Eq. 35-36 an exact tie.  FP64 takes one reciprocal square root in
// place of three square roots and seven divisions: it compares the squared distances (near a tie
// the distances themselves) and takes n = n_f (30 operations against 78).  That holds where the lattice's
// solid normals are of unit length (unit: LatDev::unit_normals); given normals of another length take
// the distances themselves and n = g_c / |g_c|.
template <typename T>
__device__ __forceinline__ void wall_normal(T eps, int wetting, bool unit, T nsx, T nsy, T c, T s, const WallSten& q, const T* val,
                                            T& cgx, T& cgy, T& nx, T& ny) {
  T gx = T(0), gy = T(0);
#pragma unroll
  for (int a = 1; a < 9; ++a) {
    const T tt = rmul(wgt<T>(a), val[q.i[a - 1]]);
    if (ex(a) == 1) gx = radd(gx, tt);
    if (ex(a) == -1) gx = radd(gx, -tt);
    if (ey(a) == 1) gy = radd(gy, tt);
    if (ey(a) == -1) gy = radd(gy, -tt);
  }
  if constexpr (sizeof(T) == 8) {
    const T sx = gx, sy = gy;
    gx = rmul(gx, T(3));
    gy = rmul(gy, T(3));
    const T m2 = radd(rmul(gx, gx), rmul(gy, gy)), inv = rsqrt(m2), mag = rmul(m2, inv);
    cgx = gx;
    cgy = gy;
    nx = ny = T(0);
    if (!(mag > eps)) return;   // (also where m2 = 0)
    const T esx = rmul(gx, inv), esy = rmul(gy, inv);
    if (wetting == 2) {
      nx = esx;
      ny = esy;
      return;
    }
    T f1x, f1y, f2x, f2y;
    wall_candidates<T>(nsx, nsy, c, s, f1x, f1y, f2x, f2y);
    const T a1 = rsub(f1x, esx), b1 = rsub(f1y, esy), a2 = rsub(f2x, esx), b2 = rsub(f2y, esy);
    const T d1 = radd(rmul(a1, a1), rmul(b1, b1)), d2 = radd(rmul(a2, a2), rmul(b2, b2));
    bool one = d1 <= d2;
    if (!unit || near_tie(d1, d2)) {
      const T gex = rdiv(sx, T(1.0 / 3.0)), gey = rdiv(sy, T(1.0 / 3.0));
      const T mage = rsqrt_(radd(rmul(gex, gex), rmul(gey, gey)));
      const T ex_ = rdiv(gex, mage), ey_ = rdiv(gey, mage);
      const T p1 = rsub(f1x, ex_), q1 = rsub(f1y, ey_), p2 = rsub(f2x, ex_), q2 = rsub(f2y, ey_);
      one = rsqrt_(radd(rmul(p1, p1), rmul(q1, q1))) <= rsqrt_(radd(rmul(p2, p2), rmul(q2, q2)));
    }
    nx = one ? f1x : f2x;
    ny = one ? f1y : f2y;
    cgx = rmul(mag, nx);
    cgy = rmul(mag, ny);
    if (!unit) {
      const T m = rsqrt_(radd(rmul(cgx, cgx), rmul(cgy, cgy)));
      nx = m > eps ? rdiv(cgx, m) : T(0);
      ny = m > eps ? rdiv(cgy, m) : T(0);
    }
    return;
  }
  const T cs2 = T(1.0 / 3.0);
  gx = rdiv(gx, cs2);
  gy = rdiv(gy, cs2);
  const T mag = rsqrt_(radd(rmul(gx, gx), rmul(gy, gy)));
  cgx = gx;
  cgy = gy;
  nx = ny = T(0);
  if (mag > eps && wetting == 2) {
    nx = rdiv(gx, mag);   // no geometric correction: n from the raw gradient
    ny = rdiv(gy, mag);
  } else if (mag > eps) {
    const T esx = rdiv(gx, mag), esy = rdiv(gy, mag);                 // Eq. 30
    T f1x, f1y, f2x, f2y;
    wall_candidates<T>(nsx, nsy, c, s, f1x, f1y, f2x, f2y);
    const T a1 = rsub(f1x, esx), b1 = rsub(f1y, esy);
    const T a2 = rsub(f2x, esx), b2 = rsub(f2y, esy);
    const T d1 = rsqrt_(radd(rmul(a1, a1), rmul(b1, b1)));            // Eq. 35
    const T d2 = rsqrt_(radd(rmul(a2, a2), rmul(b2, b2)));
    const T nfx = d1 <= d2 ? f1x : f2x;                               // Eq. 36
    const T nfy = d1 <= d2 ? f1y : f2y;
    cgx = rmul(mag, nfx);                                             // Eq. 31
    cgy = rmul(mag, nfy);
    const T m2 = rsqrt_(radd(rmul(cgx, cgx), rmul(cgy, cgy)));
    if (m2 > eps) {
      nx = rdiv(cgx, m2);
      ny = rdiv(cgy, m2);
    }
  }
}

}  // namespace lbcg
