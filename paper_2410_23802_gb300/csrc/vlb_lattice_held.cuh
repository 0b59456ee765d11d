// The FP32 cell update of lattices with held particles (vlb_set_fixed_temperature).
//
// A held disk that settles along a channel is turned by almost nothing, so its
// spin is the balance of exchange terms that cancel to their last bits: FP32
// leaves the angle uncertain by about 2e-9 whatever its size, and with a small
// initial spin the angle itself is 1e-6.  Every change of the order of
// operations, here or in the areas of vlb_raster_held.cuh, shows there as 1e-4
// and more of the output, where all other outputs move by 1e-7.  So these
// lattices keep one fixed order of operations, written out below in plain
// scalar form (one distribution after the other, nine moments each, the
// language's divisions); tests/golden/held_spin.json holds what it gives.  The
// order has to come out of the compiler the same in every kernel, alone and
// batched: sums of two products that it contracted now one way, now the other
// are explicit fused operations, and a batched launch of held lattices takes one
// storage type.  The packed form of vlb_lattice_body.cuh is the one for every
// other lattice.
// Cost of the fixed order: 11.8 us per step of an 80 x 1600 channel against
// 9.7 us in the packed form (the areas 0.9 us, the divisions 0.4 us); the lanes'
// exchange terms summed in the warp instead of added one by one made it 12.0.
#pragma once

#include "vlb_lattice_body.cuh"

namespace vlb {

// Owners of cell (tx, ty) of the tile among the np particles of the list:
// ascending particle order, at most MAX_OWNERS, fractions scaled to sum 1 when
// they exceed it (overlap).
__device__ __forceinline__ float held_owners(const PartTile<float>* list, int np, int tx, int ty, int x, int y,
                                             const ParticleArrays& P, int band_off, int band_stamp, int& nown,
                                             int (&own)[MAX_OWNERS], float (&ofs)[MAX_OWNERS], unsigned* err) {
  nown = 0;
#pragma unroll
  for (int k = 0; k < MAX_OWNERS; ++k) { own[k] = -1; ofs[k] = 0.0f; }
  for (int s = 0; s < np; ++s) {
    float f;
    if (particle_share(list[s], tx, ty, x, y, P.band, band_off, band_stamp, f, err) == CELL_FLUID) continue;
    if (nown == MAX_OWNERS) { atomicOr(err, ERR_OWNER_OVERFLOW); break; }
#pragma unroll
    for (int k = 0; k < MAX_OWNERS; ++k)
      if (k == nown) { own[k] = s; ofs[k] = f; }
    ++nown;
  }
  float fs = 0.0f;
#pragma unroll
  for (int k = 0; k < MAX_OWNERS; ++k) fs += ofs[k];
  if (fs > 1.0f) {
    const float inv = 1.0f / fs;
    fs = 0.0f;
#pragma unroll
    for (int k = 0; k < MAX_OWNERS; ++k) { ofs[k] *= inv; fs += ofs[k]; }
  }
  return fs;
}

// As cell_body (vlb_lattice_body.cuh), for FP32 and MODE_INIT, MODE_STEP or
// MODE_MACROS of a lattice with held particles.
template <class S, int MODE>
__device__ __forceinline__ void held_cell_body(const LatticeConst<float>& K, const StepBuffers& B,
                                               const ParticleArrays& P, const CellAt& at, const ListHead& head,
                                               const float2 (&p)[9], const float s_old, PartTile<float>* s_p,
                                               int band_stamp) {
  using C = float;
  constexpr bool HOLD = MODE != MODE_INIT;
  const int tx = at.tx, ty = at.ty;
  const int x = at.tile_x * TILE_X + tx, y = at.tile_y * TILE_Y + ty;
  const bool active = (x < K.nx) && (y < K.ny);
  const int cell = y * K.pitch + x;
  C f[9], g[9];
#pragma unroll
  for (int i = 0; i < 9; ++i) { f[i] = p[i].x; g[i] = p[i].y; }

  // ---- solid fraction and owners (Sec. 2); the loads above are in flight ----
  const int np = load_block_particles<S, C>(P, head, at, true, s_p);
  int nown = 0;
  int own[MAX_OWNERS];
  C ofs[MAX_OWNERS];
  C fs = C(0);
  if (active && np > 0)
    fs = held_owners(s_p, np, tx, ty, x, y, P, K.band_off, band_stamp, nown, own, ofs, B.err);
  else {
#pragma unroll
    for (int k = 0; k < MAX_OWNERS; ++k) { own[k] = -1; ofs[k] = C(0); }
  }

  // ---- flow: volumetric correction (Eq. 8) and the exchange terms (Eq. 28) ---
  // f holds deviations from w_i; rho = 1 + drho.
  // momenta as sums of differences of opposite populations: those differences
  // are exact when the two are close, which keeps j* accurate where it nearly
  // cancels rho u_s in the exchange term below
  C drho = ((f[0] + (f[1] + f[3])) + (f[2] + f[4])) + ((f[5] + f[7]) + (f[6] + f[8]));
  const C d57 = f[5] - f[7], d86 = f[8] - f[6];
  C jx = (f[1] - f[3]) + (d57 + d86);
  C jy = (f[2] - f[4]) + (d57 - d86);
  const C rho = C(1) + drho;
  const C inv_rho = C(1) / rho;
  const C jxs = jx, jys = jy;  // j* before the correction (for the exchange term)
  C lam = mul_rn(C(1) - fs, K.lam_f);
  C dT_init = C(0);  // sum_p f_s,p c_vs (T0_p - T_f): eps^0 - c_v T_f of the mixing rule
  if (nown > 0) {
    const C one_m = C(1) - fs;
    C pf[9];
#pragma unroll
    for (int i = 0; i < 9; ++i) pf[i] = C(0);
    C cjx = one_m * jx, cjy = one_m * jy;
    C hfix = C(0), h0 = C(0), hr = C(0);  // held owners: covered fraction, g^eq deviations
    const C xc = C(tx) + C(0.5), yc = C(ty) + C(0.5);
#pragma unroll
    for (int k = 0; k < MAX_OWNERS; ++k) {
      if (k >= nown) break;
      const PartTile<C>& q = s_p[own[k]];
      const C rx = (xc - q.xh) - q.xl, ry = (yc - q.yh) - q.yl;
      const C rotx = -q.om * ry, roty = q.om * rx;
      const C usx = q.ux + (q.uxl + rotx), usy = q.uy + (q.uyl + roty);  // Eq. 27
      const C w = ofs[k];
      const C u2 = usx * usx + usy * usy;
#pragma unroll
      for (int i = 0; i < 9; ++i) {
        const C eu = C(ex(i)) * usx + C(ey(i)) * usy;
        pf[i] += w * (C(3) * eu + C(4.5) * eu * eu - C(1.5) * u2);
      }
      cjx += w * rho * usx;
      cjy += w * rho * usy;
      lam = fma_rn(w, q.lam_s, lam);
      if (HOLD && q.fixed) {
        // held at T_p = T0: its part of the cell (reading R11), or the whole
        // cell (fixed == 2, reading R11b), takes g^eq(c_vs T_p, T_p), here as
        // the deviation from g^eq(eps_f, T_f)
        const C dTp = q.T0 - K.T_fluid;
        const C wh = q.fixed == 2 ? C(1) : w;
        const C dE = fma_rn(K.cv_s, q.T0, -mul_rn(K.cv_f, K.T_fluid));
        hfix += wh;
        h0 = fma_rn(wh, fma_rn(-mul_rn(C(5.0 / 9.0), K.cref), dTp, dE), h0);
        hr = fma_rn(mul_rn(wh, K.cref), dTp, hr);
      }
      dT_init += w * K.cv_s * (q.T0 - K.T_fluid);
      if (MODE != MODE_MACROS) {
        // momentum exchange (Eq. 28), added to the particle's integer
        // accumulators (a total independent of the order): sum_i e_i f_i^eq(rho, u_s) = rho u_s, so Delta F =
        // -f_s,p (rho u_s - j*), formed as (U_hi - j*) + (U_lo + Omega x r) + drho u_s
        const C v0 = -w * (((q.ux - jxs) + (q.uxl + rotx)) + drho * usx);
        const C v1 = -w * (((q.uy - jys) + (q.uyl + roty)) + drho * usy);
        const C v2 = rx * v1 - ry * v0;
        unsigned long long* acc = P.mes + 6 * (long long)q.id;
        mes_add(acc, v0, B.err);
        mes_add(acc + 2, v1, B.err);
        mes_add(acc + 4, v2, B.err);
      }
    }
#pragma unroll
    for (int i = 0; i < 9; ++i) f[i] = one_m * f[i] + wgt<C>(i) * (fs * drho + rho * pf[i]);
    jx = cjx;
    jy = cjy;
    if (HOLD && hfix > C(0)) {  // g = (1 - f_fix) g + sum over held owners of f_s,p g^eq(c_vs T_p, T_p)
      if (hfix > C(1)) {  // whole-cell holds of several owners: their mean
        const C inv = C(1) / hfix;
        h0 *= inv;
        hr *= inv;
        hfix = C(1);
      }
      const C keep = C(1) - hfix;
      g[0] = fma_rn(keep, g[0], h0);
#pragma unroll
      for (int i = 1; i < 9; ++i) g[i] = fma_rn(wgt<C>(i), hr, mul_rn(keep, g[i]));
    }
  }

  // ---- thermal macroscopics at n+1 (Eqs. 11, 16, 21-25) ----------------------
  // g holds deviations from g^eq(eps_f, T_f) of the initial fluid state
  // (eps_f = c_vf T_f); T, eps and sum g are carried as deviations dT, deps, dG
  // from T_f, eps_f, eps_f so that FP32 rounds the small parts only.
  const C cv = fma_rn(C(1) - fs, K.cv_f, mul_rn(fs, K.cv_s));
  // tau_g from Eq. 22 with alpha_1 = -2; the thermal rates of Eq. 18 (fluid
  // cells use the precomputed values)
  C sj = K.sj_f, se = K.se_f, gk = K.gk_f;
  if (nown > 0) {
    const C tau_g = C(0.5) + lam * K.k3_cref;  // 3 / c_ref
    sj = C(1) / tau_g;
    se = (K.rates_mode == C(0)) ? (tau_g - C(0.5)) / (C(0.5) * (tau_g - C(0.5)) + C(0.25)) : C(1);
    gk = -sj * K.k3_cref;  // Eq. 23: -6/(4 + alpha_1) / (c_ref tau_g)
  }
  C dT, deps, dG, qc, dfs, ux, uy;
  const C half_inv_rho = C(0.5) * inv_rho;
  const C ax = (C(1) - fs) * K.bx * half_inv_rho, ay = (C(1) - fs) * K.by * half_inv_rho;
  if (MODE == MODE_INIT) {
    dT = dT_init / cv;                         // T^0 = eps^0 / c_v
    deps = (cv - K.cv_f) * K.T_fluid + cv * dT;  // eps^0 - eps_f
    dG = deps;
    qc = C(0);
    dfs = C(0);
    // g = g^eq(eps, T) (Eq. 19 with alpha_1 = -2, alpha_2 = 1), as a deviation
    g[0] = deps - C(5) / C(9) * K.cref * dT;
#pragma unroll
    for (int i = 1; i < 9; ++i) g[i] = wgt<C>(i) * K.cref * dT;
    ux = jx * inv_rho + ax * (K.dT_ref + dT);
    uy = jy * inv_rho + ay * (K.dT_ref + dT);
  } else {
    dfs = C(2) * fs - s_old;  // Eq. 24: 2 (f_s^{n+1} - f_s^n) - [df_s/dt]^n
    dG = ((g[0] + (g[1] + g[3])) + (g[2] + g[4])) + ((g[5] + g[7]) + (g[6] + g[8]));
    const C h57 = g[5] - g[7], h86 = g[8] - g[6];
    const C qx = (g[1] - g[3]) + (h57 + h86);
    const C qy = (g[2] - g[4]) + (h57 - h86);
    const C gTx = gk * qx, gTy = gk * qy;
    const C D = cv - C(0.5) * (K.cv_s - K.cv_f) * dfs;
    const C u0x = jx * inv_rho, u0y = jy * inv_rho;
    // Eq. 25 with u = u0 + a (T - T_ref), solved for T - T_f:
    // T - T_f = [(c_vf - D) T_f + dG - c_v/2 (u0.gradT + (T_f - T_ref) a.gradT)] / (D + c_v/2 a.gradT)
    const C agT = ax * gTx + ay * gTy;
    const C num = (K.cv_f - D) * K.T_fluid + dG - C(0.5) * cv * (u0x * gTx + u0y * gTy + K.dT_ref * agT);
    const C den = D + C(0.5) * cv * agT;
    dT = num / den;
    ux = u0x + ax * (K.dT_ref + dT);
    uy = u0y + ay * (K.dT_ref + dT);
    qc = fma_rn((K.cv_s - K.cv_f) * (K.T_fluid + dT), dfs, mul_rn(-cv, ux * gTx + uy * gTy));
    // Eq. 21, eps = sum g + q_c / 2, taken literally (equal to c_v T in exact
    // arithmetic): the conserved moment then carries no rounding of the solve
    deps = dG + C(0.5) * qc;
  }
  const C Fx = (C(1) - fs) * K.bx * (K.dT_ref + dT);
  const C Fy = (C(1) - fs) * K.by * (K.dT_ref + dT);

  if (MODE == MODE_MACROS || MODE == MODE_INIT) {
    if (active && B.macro != nullptr) {
      C* m = static_cast<C*>(B.macro);
      m[0 * K.plane + cell] = rho;
      m[1 * K.plane + cell] = ux;
      m[2 * K.plane + cell] = uy;
      m[3 * K.plane + cell] = K.T_fluid + dT;
      m[4 * K.plane + cell] = fs;
      m[5 * K.plane + cell] = K.cv_f * K.T_fluid + deps;
      m[6 * K.plane + cell] = K.cv_f * K.T_fluid + dG;
    }
  }

  if (MODE != MODE_MACROS) {
    if (!active) return;
    // random key of stochastic rounding (16-bit storage only)
    const unsigned skey = sizeof(S) == 2 ? sr_key(y * K.nx + x, band_stamp) : 0u;
    Pair<C> out[9];

    // ---- MRT collision of f in moment space (Eqs. 3a, 4-7) ------------------
    // Written as f-bar = f + M^-1 (m-bar - m): only the relaxed moments and the
    // forcing change, and M^-1 = M^T diag(1/9, 1/36, 1/36, 1/6, 1/12, 1/6,
    // 1/12, 1/4, 1/4).  The conserved moments get exactly rho and j + F
    // (Eq. 9: rho u = j + F/2); in cells the correction touched, whose f carries
    // FP32-rounded weights, the difference to those targets is put back here
    // so that no rounding bias repeats step after step.
    {
      const C m1 = -C(4) * f[0] - (f[1] + f[2] + f[3] + f[4]) + C(2) * (f[5] + f[6] + f[7] + f[8]);
      const C m2 = C(4) * f[0] - C(2) * (f[1] + f[2] + f[3] + f[4]) + (f[5] + f[6] + f[7] + f[8]);
      const C m4 = -C(2) * f[1] + C(2) * f[3] + f[5] - f[6] - f[7] + f[8];
      const C m6 = -C(2) * f[2] + C(2) * f[4] + f[5] + f[6] - f[7] - f[8];
      const C m7 = f[1] - f[2] + f[3] - f[4];
      const C m8 = f[5] - f[6] + f[7] - f[8];
      // deviations of m^eq(rho, u) from m^eq(1, 0) (Eq. 6), with rho u = j + F/2
      const C e3 = jx + C(0.5) * Fx, e5 = jy + C(0.5) * Fy;
      const C ru2 = e3 * ux + e5 * uy;
      const C e1 = -C(2) * drho + C(3) * ru2;
      const C e2 = drho - C(3) * ru2;
      const C e7 = e3 * ux - e5 * uy, e8 = e3 * uy;
      // forcing moments (Eq. 7)
      const C Fu = Fx * ux + Fy * uy;
      const C F7 = C(2) * (Fx * ux - Fy * uy), F8 = Fx * uy + Fy * ux;
      const C d1 = -K.s_e * (m1 - e1) + (C(1) - C(0.5) * K.s_e) * (C(6) * Fu);
      const C d2 = -K.s_eps * (m2 - e2) + (C(1) - C(0.5) * K.s_eps) * (-C(6) * Fu);
      const C d4 = -K.s_q * (m4 + e3) + (C(1) - C(0.5) * K.s_q) * (-Fx);
      const C d6 = -K.s_q * (m6 + e5) + (C(1) - C(0.5) * K.s_q) * (-Fy);
      const C d7 = -K.s_p * (m7 - e7) + (C(1) - C(0.5) * K.s_p) * F7;
      const C d8 = -K.s_p * (m8 - e8) + (C(1) - C(0.5) * K.s_p) * F8;
      // conserved moments: m-bar_0 = rho, m-bar_3 = j_x + F_x, m-bar_5 = j_y + F_y
      C d0 = C(0), d3 = Fx, d5 = Fy;
      if (nown > 0) {
        const C n0 = ((f[0] + (f[1] + f[3])) + (f[2] + f[4])) + ((f[5] + f[7]) + (f[6] + f[8]));
        const C q57 = f[5] - f[7], q86 = f[8] - f[6];
        d0 = drho - n0;
        d3 = (jx - ((f[1] - f[3]) + (q57 + q86))) + Fx;
        d5 = (jy - ((f[2] - f[4]) + (q57 - q86))) + Fy;
      }
      const C a0 = d0 * C(1.0 / 9.0), a1 = d1 * C(1.0 / 36.0), a2 = d2 * C(1.0 / 36.0);
      const C a3 = d3 * C(1.0 / 6.0), a4 = d4 * C(1.0 / 12.0), a5 = d5 * C(1.0 / 6.0);
      const C a6 = d6 * C(1.0 / 12.0), a7 = d7 * C(0.25), a8 = d8 * C(0.25);
      const C c14 = a0 - a1 - C(2) * a2;
      const C c58 = a0 + C(2) * a1 + a2;
      const C o[9] = {f[0] + (a0 - C(4) * a1 + C(4) * a2), f[1] + (c14 + a3 - C(2) * a4 + a7),
                      f[2] + (c14 + a5 - C(2) * a6 - a7),  f[3] + (c14 - a3 + C(2) * a4 + a7),
                      f[4] + (c14 - a5 + C(2) * a6 - a7),  f[5] + (c58 + a3 + a4 + a5 + a6 + a8),
                      f[6] + (c58 - a3 - a4 + a5 + a6 - a8), f[7] + (c58 - a3 - a4 - a5 - a6 + a8),
                      f[8] + (c58 + a3 + a4 - a5 - a6 - a8)};
#pragma unroll
      for (int i = 0; i < 9; ++i) out[i].x = o[i];
    }

    // ---- MRT collision of g with the source term (Eqs. 17a, 18-20) ----------
    // The same delta form: n-bar - n for the relaxed moments and the source;
    // the conserved moment gets sum g + q_c exactly (sigma_0 = 1 with
    // eps = sum g + q_c / 2, Eq. 21).
    {
      const C n1 = -C(4) * g[0] - (g[1] + g[2] + g[3] + g[4]) + C(2) * (g[5] + g[6] + g[7] + g[8]);
      const C n2 = C(4) * g[0] - C(2) * (g[1] + g[2] + g[3] + g[4]) + (g[5] + g[6] + g[7] + g[8]);
      const C n3 = g[1] - g[3] + g[5] - g[6] - g[7] + g[8];
      const C n4 = -C(2) * g[1] + C(2) * g[3] + g[5] - g[6] - g[7] + g[8];
      const C n5 = g[2] - g[4] + g[5] + g[6] - g[7] - g[8];
      const C n6 = -C(2) * g[2] + C(2) * g[4] + g[5] + g[6] - g[7] - g[8];
      const C n7 = g[1] - g[2] + g[3] - g[4];
      const C n8 = g[5] - g[6] + g[7] - g[8];
      // n^eq = [eps, -4 eps + 2 c_ref T, 4 eps - 3 c_ref T, 0, ...]; q_m = [q, -4q, 4q, 0, ...]
      // (deviations from the moments of g^eq(eps_f, T_f))
      const C ct = K.cref * dT;
      const C d1 = -se * (n1 - (-C(4) * deps + C(2) * ct)) + (C(1) - C(0.5) * se) * (-C(4) * qc);
      const C d2 = -se * (n2 - (C(4) * deps - C(3) * ct)) + (C(1) - C(0.5) * se) * (C(4) * qc);
      const C a0 = qc * C(1.0 / 9.0), a1 = d1 * C(1.0 / 36.0), a2 = d2 * C(1.0 / 36.0);
      const C a3 = -sj * n3 * C(1.0 / 6.0), a4 = -sj * n4 * C(1.0 / 12.0);
      const C a5 = -sj * n5 * C(1.0 / 6.0), a6 = -sj * n6 * C(1.0 / 12.0);
      const C a7 = -se * n7 * C(0.25), a8 = -se * n8 * C(0.25);
      const C c14 = a0 - a1 - C(2) * a2;
      const C c58 = a0 + C(2) * a1 + a2;
      const C o[9] = {g[0] + (a0 - C(4) * a1 + C(4) * a2), g[1] + (c14 + a3 - C(2) * a4 + a7),
                      g[2] + (c14 + a5 - C(2) * a6 - a7),  g[3] + (c14 - a3 + C(2) * a4 + a7),
                      g[4] + (c14 - a5 + C(2) * a6 - a7),  g[5] + (c58 + a3 + a4 + a5 + a6 + a8),
                      g[6] + (c58 - a3 - a4 + a5 + a6 - a8), g[7] + (c58 - a3 - a4 - a5 - a6 + a8),
                      g[8] + (c58 + a3 + a4 - a5 - a6 - a8)};
#pragma unroll
      for (int i = 0; i < 9; ++i) out[i].y = o[i];
    }
    store_pairs<S, C>(B.dst, cell, out, skey);
    static_cast<C*>(B.s_dst)[cell] = C(2) * fs + dfs;
  }
}

// One cell of a lattice pass: the pull, then the update of the lattice's kind.
template <class S, class C, int MODE, bool HOLD>
__device__ __forceinline__ void lattice_cell(const LatticeConst<C>& K, const StepBuffers& B, const ParticleArrays& P,
                                             const CellAt& at, const ListHead& head, PartTile<C>* list,
                                             int band_stamp) {
  constexpr bool HELD = HOLD && sizeof(C) == 4;
  Pair<C> p[9];
  C s_old;
  pull_direct<S, C, MODE, HELD>(K, B, at, p, s_old);
  if constexpr (HELD) held_cell_body<S, MODE>(K, B, P, at, head, p, s_old, list, band_stamp);
  else cell_body<S, C, MODE, HOLD>(K, B, P, at, head, p, s_old, list, band_stamp);
}

}  // namespace vlb
