// position.cuh -- position half of Algorithm 1 on the mixed path, in
// double-float arithmetic on the float32 pipe (df.cuh), for every surface.
//
// Algorithm 1 in multiplier form. The momentum half at x^k and the kick of the
// position half give q = p^{k-1/2} + dt F^k - s n0, s = n0.(p^{k-1/2} + h F^k)
// / |n0|^2, n0 = grad g(x^k); the position half then subtracts h lambda n0.
// Both corrections lie along n0, so with q0 = p^{k-1/2} + dt F^k,
// y = x^k + (dt/m) q0 and mu = (dt/m)(s + h lambda):
//   x^{k+1} = y - mu n0,   p^{k+1/2} = q0 - (m/dt) mu n0,   g(y - mu n0) = 0.
// The projection s only sets where the Newton iteration starts (mu_0 =
// (dt/m) s, formed in float32), not its root. On the first step after a state
// is set there is no momentum half: q0 = p^k + h F^k, mu_0 = 0.
//
// The position-half Newton update lambda += g / (a n1.n0) of Algorithm 1 reads
// mu += g(x(mu)) / (n1.n0) on the line x(mu) = y - mu n0 (mu = a lambda,
// n1 = grad g(x(mu)); n1 = n0 in the frozen-normal variant). g along the line
// is evaluated in double-float; the Newton denominator n1.n0 is float32 (it
// scales the step, not the root):
//   plane, sphere, ellipsoid, cylinder  the exact line form g(y) - b mu +
//     c mu^2 (b = grad g(y).n0, c = n0.H n0 / 2, H the constant Hessian)
//   torus  g at the point
//   Gaussian bump  from its value at x^k: with E = A exp(-rho^2 / 2w^2) at
//     x^k (the one exponential of a step) and the displacement e = x(mu) - x^k,
//     g = g(x^k) + e_z - E expm1(-(2 rho.e + |e_xy|^2) / 2w^2), a short
//     argument (a displacement of 0.1 sigma on a width of 25 sigma: 4e-3); a step
//     over half the box from the bump goes on with the image it comes to
//   thylakoid composite  its piece, chosen at x^k and held for the solve, is a
//     plane, a cylinder or a torus in coordinates mirrored into the block's
//     first quadrant and rotated so that the piece's axis is the third
// The full-step momentum p^k is not needed by the step and is formed only on
// read-out, with the float64 normal.
#pragma once

#include "df.cuh"

namespace surfmd {

// g on the line x(mu) = y - mu n0 in double-float at a point of a torus about
// the third axis, D = y - c, N = n0, keeping rho - R, rho and x(mu) - c in
// float32 for the Newton denominator.
struct DFTorusEval {
  float ttf, rhof, e0, e1, e2;
  __device__ __forceinline__ DF g(DF R, DF gconst, const DF D[3], const DF N[3], DF mu) {
    DF E[3];
#pragma unroll
    for (int d = 0; d < 3; ++d) E[d] = df_sub(D[d], df_mul(N[d], mu));
    const DF rho = df_sqrt(df_add(df_mul(E[0], E[0]), df_mul(E[1], E[1])));
    const DF t = df_sub(rho, R);
    ttf = t.h;
    rhof = rho.h;
    e0 = E[0].h; e1 = E[1].h; e2 = E[2].h;
    return df_add(df_add(df_mul(t, t), df_mul(E[2], E[2])), gconst);
  }
  // n1.n0 = 2 (rho - R)/rho (e_xy . n0_xy) + 2 e_z n0_z
  __device__ __forceinline__ float n1n0(const DF N[3]) const {
    return 2.f * ttf * rcp_approx(rhof) * fmaf(e0, N[0].h, e1 * N[1].h) + 2.f * e2 * N[2].h;
  }
};

// g of the Gaussian bump on the line, from its value at x^k: C = x^k - c (x and
// y at the minimum image), E = A exp(-rho^2 / 2w^2) and g0 = g there, T = the
// displacement to y.
struct DFBumpEval {
  DF E, g0;
  float n1x, n1y;
  __device__ __forceinline__ void at(const SysDev& S, const DF C[3]) {
    E = df_mul(S.bumpA_df, df_exp_neg(df_neg(df_mul(df_add(df_mul(C[0], C[0]), df_mul(C[1], C[1])), S.half_iw2_df))));
    g0 = df_sub(C[2], E);
  }
  __device__ __forceinline__ DF g(const SysDev& S, const DF C[3], const DF T[3], const DF N[3], DF mu) {
    DF e[3];
#pragma unroll
    for (int d = 0; d < 3; ++d) e[d] = df_sub(T[d], df_mul(N[d], mu));
    // -(2 rho.e + |e_xy|^2) / 2w^2
    const DF sx = df_mul(df_add(df_scale2(C[0], 2.f), e[0]), e[0]), sy = df_mul(df_add(df_scale2(C[1], 2.f), e[1]), e[1]);
    const DF ds = df_neg(df_mul(df_add(sx, sy), S.half_iw2_df));
    DF dE;  // E(x(mu)) - E
    if (fabsf(ds.h) <= 0.35f) {
      dE = df_mul(E, df_expm1_small(ds));
    } else {  // a displacement of the order of the bump's width: the exponential anew
      const DF r2 = df_add(df_mul(df_add(C[0], e[0]), df_add(C[0], e[0])), df_mul(df_add(C[1], e[1]), df_add(C[1], e[1])));
      dE = df_sub(df_mul(S.bumpA_df, df_exp_neg(df_neg(df_mul(r2, S.half_iw2_df)))), E);
    }
    const float q = 2.f * S.half_iw2_df.h * (E.h + dE.h);  // E(x(mu)) / w^2
    n1x = q * (C[0].h + e[0].h);
    n1y = q * (C[1].h + e[1].h);
    return df_sub(df_add(g0, e[2]), dE);
  }
  __device__ __forceinline__ float n1n0(const DF N[3]) const {  // n1 = (E dx / w^2, E dy / w^2, 1), n0_z = 1
    return fmaf(n1x, N[0].h, fmaf(n1y, N[1].h, 1.f));
  }
};

// Sign test of a - b (exact to the double-floats' resolution).
__device__ __forceinline__ bool df_less(DF a, DF b) {
  return __fadd_rn(__fsub_rn(a.h, b.h), __fsub_rn(a.l, b.l)) < 0.f;
}

// A thylakoid piece in its local frame: shape kPlane (g = first coordinate),
// kCylinder or kTorus about the third axis; x and y mirrored by (fx, fy), then
// the coordinates rotated (0,1,2) -> (1,2,0) if rot.
struct DFPiece {
  int32_t shape;
  float fx, fy;
  bool rot;
  DF gconst, R;
};

// The piece of a particle at C = x - c (z at its minimum image), as the
// float64 selection thyl_select takes it (the composite is symmetric under x ->
// -x and y -> -y about its centre, so one quadrant serves all); C and T (any
// vector) move into the piece's frame.
__device__ __forceinline__ DFPiece df_thyl_piece(const SysDev& S, DF C[3], DF T[3]) {
  const ThylDF& K = S.thyl_df;
  DFPiece q;
  const DF zero = {0.f, 0.f};
  q.fx = df_less(zero, C[0]) ? 1.f : -1.f;  // x <= c_x: the left block
  q.fy = C[1].h < 0.f ? -1.f : 1.f;
  const DF u = df_scale2(C[0], q.fx), v = df_scale2(C[1], q.fy);
  const DF r2 = df_add(df_mul(v, v), df_mul(C[2], C[2]));
  const bool near_axis = df_less(r2, K.rout2);
  q.R = K.rout;
  q.gconst = K.m_rc2;
  DF cu = zero, cv = zero;  // the piece's centre in u and v
  if (near_axis && df_less(u, K.xf)) {  // between the faces: the bridge, or the connector beyond its end
    q.shape = df_less(K.half_lb, u) ? kTorus : kCylinder;
    q.rot = true;
    cu = K.half_lb;
    if (q.shape == kCylinder) q.gconst = K.m_rb2;
  } else {
    // ex < 0: beyond the inner square towards the bridge, > 0: away from it; ey > 0: beyond it sideways
    int ex = df_less(u, K.inner) ? -1 : (df_less(K.inner_hi, u) ? 1 : 0);
    bool ey = df_less(K.half_lx, v);
    if (ex != 0 && ey) {
      q.shape = kCylinder;
      q.rot = false;
      cu = ex < 0 ? K.inner : K.inner_hi;
      cv = K.half_lx;
    } else {
      if (ex == 0 && !ey) {  // inside the inner square: the nearest side
        const DF dl = df_sub(u, K.xf), dh = df_sub(K.face_hi, u), dv = df_sub(K.side_y, v);
        const bool low = df_less(dl, dh);
        if (!df_less(dv, low ? dl : dh)) ex = low ? -1 : 1;  // the nearer of the two x sides, then against y
      }
      if (ex < 0 && near_axis) {  // the face plane's hole belongs to the connector
        q.shape = kTorus;
        q.rot = true;
        cu = K.half_lb;
      } else {
        q.shape = kPlane;
        q.rot = ex == 0;
        cu = ex < 0 ? K.xf : K.face_hi;
        cv = K.side_y;
        if (ex != 0) cv = zero;
        else cu = zero;
      }
    }
  }
  const DF c[3] = {df_sub(u, cu), df_sub(v, cv), C[2]};
  const DF t[3] = {df_scale2(T[0], q.fx), df_scale2(T[1], q.fy), T[2]};
#pragma unroll
  for (int d = 0; d < 3; ++d) {
    C[d] = q.rot ? c[(d + 1) % 3] : c[d];
    T[d] = q.rot ? t[(d + 1) % 3] : t[d];
  }
  return q;
}

// What bounds it: instruction issue. The bump and the thylakoid went through
// float64 before (two operations per SM and clock): the integrator launch of 128
// thylakoids of 2,500 particles took 179 us (CUDA events) and takes 35, that of
// 100,000 particles on a bump and 900,000 free ones 74.5 us and takes 51.
//
// Position half of a constrained particle: reads x^k, p^{k-1/2} (or p^k on the
// first step) and the combined force F, returns x^{k+1} and p^{k+1/2}. y - c,
// n0 = grad g(x^k) and g in double-float. For the plane, sphere, ellipsoid and
// cylinder forms the Newton iteration runs on the line form first in float32,
// which brings mu to float32 resolution (about 1e-7 of mu n0, itself about
// 1e-4 sigma), then continues in double-float until g, evaluated in
// double-float, meets the tolerance; the torus and the bump iterate in
// double-float throughout. x^{k+1} is rounded once to float64: c + (y - c) - mu
// n0 summed in double-float, or for the bump and the thylakoid (whose centre
// differs from the handle's) x^k + (y - x^k - mu n0) in float64;
// p^{k+1/2} = p + (kick F - (m/dt) mu n0) adds a float32 increment to the
// float64 momentum.
// SURF: the composed surfaces compiled in, bit 0 the bump, bit 1 the thylakoid: a
// handle runs the integrator without the ones it does not have, at fewer
// registers and spills.
template <int SURF>
__device__ __forceinline__ void position_half_df(const SysDev& S, uint32_t ty, int mode, const double xv[3],
                                                 const double pv[3], const DF P[3], const float F[3],
                                                 uint32_t* status, double xo[3], double qo[3]) {
  DF C[3], D[3], N[3], T[3];  // x - c, y - c, n0, y - x
  const DF kick = mode ? S.dt_df : S.half_dt_df;
  df_from3(xv, C);
#pragma unroll
  for (int d = 0; d < 3; ++d) {
    const DF q0 = df_add(P[d], df_mul_f(kick, F[d]));  // q0 = p + kick F
    if (!S.c_zero) C[d] = df_sub(C[d], S.c_df[d]);
    T[d] = df_mul(S.dtm_df[ty], q0);
  }
  float pf[3] = {P[0].h, P[1].h, P[2].h}, Ff[3] = {F[0], F[1], F[2]};
  int32_t shape = S.kind;
  DF gconst = S.gconst_df, R = S.R_df;
  int axis = S.axis;
  const bool moved = ((SURF & 2) && shape == kThylakoid) || ((SURF & 1) && shape == kBump);  // C is not x - c componentwise
  DFPiece piece{};
  if (moved) {
#pragma unroll
    for (int d = 0; d < 3; ++d) {  // minimum images (the bump in x and y, the thylakoid in z), from the float64 master
      if (!(S.periodic[d] && (d < 2 || shape == kThylakoid))) continue;
      const float k = rintf(C[d].h / S.box_len_df[d].h);
      if (k != 0.f) C[d] = df_from(fma(-f2d(k), S.box_len[d], xv[d] - S.c[d]));
    }
    if ((SURF & 2) && shape == kThylakoid) {
      piece = df_thyl_piece(S, C, T);
      shape = piece.shape;
      gconst = piece.gconst;
      R = piece.R;
      axis = 2;
      const float a[3] = {pf[0] * piece.fx, pf[1] * piece.fy, pf[2]}, b[3] = {F[0] * piece.fx, F[1] * piece.fy, F[2]};
#pragma unroll
      for (int d = 0; d < 3; ++d) {
        pf[d] = piece.rot ? a[(d + 1) % 3] : a[d];
        Ff[d] = piece.rot ? b[(d + 1) % 3] : b[d];
      }
    }
  }
#pragma unroll
  for (int d = 0; d < 3; ++d) D[d] = df_add(C[d], T[d]);
  DFBumpEval B;
  DF gy{0.f, 0.f}, b{0.f, 0.f};
  float c = 0.f;
  switch (shape) {
    case kPlane:
#pragma unroll
      for (int d = 0; d < 3; ++d) N[d] = moved ? DF{d == 0 ? 1.f : 0.f, 0.f} : S.pn_df[d];
      gy = moved ? D[0] : df_dot3(S.pn_df, D);
      b = moved ? DF{1.f, 0.f} : df_dot3(S.pn_df, N);
      break;
    case kEllipsoid: {
      DF U[3];
#pragma unroll
      for (int d = 0; d < 3; ++d) {
        N[d] = df_scale2(df_mul(C[d], S.inv_a2_df[d]), 2.f);
        U[d] = df_mul(D[d], S.inv_a2_df[d]);
        c = fmaf(N[d].h * N[d].h, S.inv_a2_df[d].h, c);
      }
      gy = df_add_f(df_dot3(U, D), -1.f);
      b = df_scale2(df_dot3(U, N), 2.f);
      break;
    }
    case kTorus: {
      const DF rho = df_sqrt(df_add(df_mul(C[0], C[0]), df_mul(C[1], C[1])));
      const DF q = df_scale2(df_div(df_sub(rho, R), rho), 2.f);  // 2 (rho - R) / rho
      N[0] = df_mul(q, C[0]);
      N[1] = df_mul(q, C[1]);
      N[2] = df_scale2(C[2], 2.f);
      break;
    }
    case kBump: if constexpr ((SURF & 1) != 0) {
      B.at(S, C);
      const DF q = df_scale2(df_mul(B.E, S.half_iw2_df), 2.f);  // E / w^2
      N[0] = df_mul(q, C[0]);
      N[1] = df_mul(q, C[1]);
      N[2] = {1.f, 0.f};
      break;
    }
    [[fallthrough]];
    default: {  // sphere; cylinder without the axis component (n0 has none)
      DF M[3];
#pragma unroll
      for (int d = 0; d < 3; ++d) {
        const bool off = shape == kCylinder && d == axis;
        M[d] = off ? DF{0.f, 0.f} : D[d];
        N[d] = off ? DF{0.f, 0.f} : df_scale2(C[d], 2.f);
      }
      gy = df_add(df_dot3(M, M), gconst);
      b = df_scale2(df_dot3(M, N), 2.f);
      break;
    }
  }
  const float nnf = fmaf(N[0].h, N[0].h, fmaf(N[1].h, N[1].h, N[2].h * N[2].h));
  if (shape == kSphere || shape == kCylinder) c = nnf;
  float mu0 = 0.f;
  if (mode) {  // mu_0 = (dt/m) n0.(p + h F) / |n0|^2
    float sp = 0.f;
#pragma unroll
    for (int d = 0; d < 3; ++d) sp = fmaf(N[d].h, fmaf(S.half_dt_f, Ff[d], pf[d]), sp);
    mu0 = S.dtm_f[ty] * sp * rcp_approx(nnf);
  }
  const float tol_n = 0.99f * S.tol_f * sqrt_approx(nnf);
  // round-off floor: an update below 4 units of the double-float resolution of the position
  const float dmax = fmaxf(fabsf(D[0].h), fmaxf(fabsf(D[1].h), fabsf(D[2].h)));
  const float floor_mu =
      4.f * 0x1p-47f * dmax * rcp_approx(fmaxf(fabsf(N[0].h), fmaxf(fabsf(N[1].h), fabsf(N[2].h))));
  const bool torus = shape == kTorus, bump = (SURF & 1) && shape == kBump, line = !torus && !bump;
  int it = 0;
  // float32 Newton on the line form g(y) - b mu + c mu^2, whose updates count towards max_newton too: on a thylakoid
  // piece only where that leaves ample for the double-float ones (two or three of each; the frozen normal takes more)
  if (line && !((SURF & 2) && moved && S.max_newton < (S.frozen ? 16 : 8))) {
    for (; it < S.max_newton; ++it) {
      const float gf = fmaf(fmaf(c, mu0, -b.h), mu0, gy.h);
      if (fabsf(gf) < 0.5f * tol_n) break;
      const float dmu = gf * rcp_approx(S.frozen ? nnf : fmaf(-2.f * mu0, c, b.h));
      mu0 += dmu;
      if (fabsf(dmu) <= 0x1p-22f * fabsf(mu0)) {
        ++it;
        break;
      }
    }
  }
  DFTorusEval Q;
  DF mu = {mu0, 0.f};
  bool ok = false;
  for (bool turned = !bump;;) {
    for (;; ++it) {
      const DF g = torus ? Q.g(R, gconst, D, N, mu)
                         : (bump ? B.g(S, C, T, N, mu) : df_add_f(df_sub(gy, df_mul(b, mu)), c * mu.h * mu.h));
      if (fabsf(g.h) < tol_n) { ok = true; break; }
      if (it >= S.max_newton) break;
      const float den = S.frozen ? nnf : (torus ? Q.n1n0(N) : (bump ? B.n1n0(N) : fmaf(-2.f * mu.h, c, b.h)));
      const float dmu = g.h * rcp_approx(den);
      mu = df_add_f(mu, dmu);
      if (it > 0 && fabsf(dmu) <= floor_mu) { ok = true; break; }
    }
    // a step of the bump's over half the box: on from here with the image of the bump that it has come to
    if (turned) break;
    const float px = fmaf(-N[0].h, mu.h, D[0].h), py = fmaf(-N[1].h, mu.h, D[1].h);
    const float near = 0.5f - 0x1p-18f;  // (screened in float32, decided in double-float)
    if (!(fabsf(px) > near * S.box_len_df[0].h || fabsf(py) > near * S.box_len_df[1].h)) break;
    turned = true;
    bool moves = false;
#pragma unroll
    for (int d = 0; d < 2; ++d) {
      const DF L = S.box_len_df[d], e = df_sub(D[d], df_mul(N[d], mu)), half = df_scale2(L, 0.5f);
      const float k = df_less(half, e) ? 1.f : (df_less(e, df_neg(half)) ? -1.f : 0.f);
      if (k != 0.f) {
        C[d] = df_sub(C[d], df_mul_f(L, k));
        moves = true;
      }
    }
    if (!moves) break;
    B.at(S, C);
    it = 0;
    ok = false;
  }
  if (!ok) flag(status, kFlagRattle);
  const float kickf = mode ? S.dt_df.h : S.half_dt_df.h;
  const float cm = mu.h * S.inv_dtm_df[ty].h;  // (m/dt) mu
  if (moved) {
    DF e[3];
    float nf[3] = {N[0].h, N[1].h, N[2].h};
#pragma unroll
    for (int d = 0; d < 3; ++d) e[d] = df_sub(T[d], df_mul(N[d], mu));  // (y - x) - mu n0
    if ((SURF & 2) && S.kind == kThylakoid) {  // back from the piece's frame
      const DF r[3] = {e[0], e[1], e[2]};
      const float nr[3] = {nf[0], nf[1], nf[2]};
      const float s[3] = {piece.fx, piece.fy, 1.f};
#pragma unroll
      for (int d = 0; d < 3; ++d) {
        e[d] = df_scale2(piece.rot ? r[(d + 2) % 3] : r[d], s[d]);
        nf[d] = (piece.rot ? nr[(d + 2) % 3] : nr[d]) * s[d];
      }
    }
#pragma unroll
    for (int d = 0; d < 3; ++d) {
      xo[d] = xv[d] + df_to(e[d]);
      qo[d] = pv[d] + f2d(fmaf(kickf, F[d], -cm * nf[d]));
    }
    return;
  }
#pragma unroll
  for (int d = 0; d < 3; ++d) {
    DF e = df_sub(D[d], df_mul(N[d], mu));  // (y - c) - mu n0
    if (!S.c_zero) e = df_add(e, S.c_df[d]);
    xo[d] = df_to(e);
    qo[d] = pv[d] + f2d(fmaf(kickf, F[d], -cm * N[d].h));  // p + kick F - (m/dt) mu n0
  }
}

}  // namespace surfmd
