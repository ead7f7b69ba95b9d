// step_site.cuh -- one collide-and-stream step of one site in scalar FP32: the
// body of the one-site kernel (step.cu) and of its several-step form for small
// lattices (step_multi.cu).
//
// Algebra of the fluid collision.  With S = diag[1,1,1,1,w,w,w,w,w,1,...,1]
// (eq. collision_matrix) every central moment except the five deviatoric
// second-order ones is set to its equilibrium value, so
//     f* = f^mhd(0) + (1 - w) P(f - f^mhd(0)),
// where P(D) is the population whose central moments are zero except the
// second-order ones, which equal dev(Pi_neq) with Pi_neq the raw second
// moment of f - f^mhd(0) (equal to its central moment since that difference
// carries no mass or momentum).  Any basis with the span of the corrected
// T of Sec. 3.1.2 gives this result.  In 1-D, the population with central
// moments (m0, m1, m2) at velocity shift u is
//     f_0 = m0 (1 - u^2) - 2 u m1 - m2,   f_+-1 = (m0 (u^2 +- u) + m1 (2u +- 1) + m2) / 2,
// and the 3-D map is the tensor product over the axes; the 6th-order Hermite
// equilibrium of App. A factors the same way (psi(0,u) = 2/3 - u^2,
// psi(+-1,u) = (1/3 + u^2 +- u)/2).  Everything is evaluated divided by the
// lattice weights w_i = w1(cx) w1(cy) w1(cz), w1 = (2/3, 1/6), and as a
// deviation from the rest equilibrium of (rho0, B_ref), so FP32 keeps the
// relative precision of the dynamic part.
//
// Collision step per site (Sec. 3): a1 load + decode, a2 rho and U
// (eq. LB_moments2), a3 B and Lambda (eqs. mag_field_LB, LB_density_current),
// a4 J from the Hall system (eq. soe_current_density, closed form of its
// 3x3 solve), a5 central-moment fluid collision (eq. cm_collision_step),
// a6 g^Hall(0) (eq. gHall_eq) and BGK (eq. MHD_LBscheme), a7 encode and
// store (eq. stream, AA pattern).
#pragma once

#include "aa.cuh"

namespace flame {
namespace {

// VAR selects the scheme: kVarFlame (the paper's), kVarBgkFluid, kVarEmhd or
// kVarFdCurrent (flame_internal.h); Bfd is the pre-collision B - B_ref field
// (storage type) written by the B pre-pass, read only by kVarFdCurrent.
// L2 reads the populations past L1, for a kernel that takes several steps.
template <bool L2, class T>
__device__ __forceinline__ T load_pop(const T* p) {
  if constexpr (L2) return load_l2(p);
  else return *p;
}

// Reads the populations of P and writes those of O: the state itself, or another
// one (every location is written by the site that read it).
template <class T, bool ODD, int VAR, bool L2>
__device__ __forceinline__ void step_site(const Slots<T>& P, const Slots<T>& O, const Grid& g, const StepConsts& k,
                                          unsigned* __restrict__ flag, const T* __restrict__ Bfd, int x, int y, int z) {
  const int site = (z * g.ny + y) * g.nx + x;
  const Nbr nb = make_nbr(x, y, z, g);

  // a1: load and decode the 48 pre-collision populations.  Fluid values are
  // kept in velocity-cube order s[px + 3 py + 9 pz], p = c + 1.
  float s[kQ];
#pragma unroll
  for (int pz = 0; pz < 3; ++pz)
#pragma unroll
    for (int py = 0; py < 3; ++py)
#pragma unroll
      for (int px = 0; px < 3; ++px) {
        const int i = idx27(px, py, pz);
        const int slot = ODD ? opp27(i) : i;
        s[px + 3 * py + 9 * pz] = Codec<T>::dec(load_pop<L2>(&P.p[slot][site + src_off<ODD>(nb, px - 1, py - 1, pz - 1)]));
      }
  float sg[3][kM];
#pragma unroll
  for (int b = 0; b < 3; ++b)
#pragma unroll
    for (int i = 0; i < kM; ++i) {
      const int slot = mslot(b, ODD ? opp7(i) : i);
      sg[b][i] = Codec<T>::dec(load_pop<L2>(&P.p[slot][site + src_off<ODD>(nb, mx7(i), my7(i), mz7(i))]));
    }

  // a2: rho, momentum and raw second moment (deviations from rest) by three
  // 1-D passes over the velocity cube with the 1-D weights (1, 4, 1) / 6.
  float m0[9], m1[9], m2[9];  // x pass: [py + 3 pz]
#pragma unroll
  for (int q = 0; q < 9; ++q) {
    const float sm = s[3 * q], s0 = s[3 * q + 1], sp = s[3 * q + 2];
    const float t = sp + sm;
    m0[q] = fmaf(4.f, s0, t);
    m1[q] = sp - sm;
    m2[q] = t;
  }
  float M00[3], M10[3], M20[3], M01[3], M11[3], M02[3];  // y pass: [pz]
#pragma unroll
  for (int pz = 0; pz < 3; ++pz) {
    const int q = 3 * pz;
    const float t0 = m0[q + 2] + m0[q];
    M00[pz] = fmaf(4.f, m0[q + 1], t0);
    M02[pz] = t0;
    M01[pz] = m0[q + 2] - m0[q];
    M10[pz] = fmaf(4.f, m1[q + 1], m1[q + 2] + m1[q]);
    M11[pz] = m1[q + 2] - m1[q];
    M20[pz] = fmaf(4.f, m2[q + 1], m2[q + 2] + m2[q]);
  }
  // The density deviation is divided exactly (correct rounding keeps mass
  // unbiased); momentum and stress use the reciprocal of 216 rho / of 216,
  // whose rounding is not one-signed across sites (U) or only rescales the
  // non-conserved stress by 1 + O(1e-8) (Pi).
  const float t00 = M00[2] + M00[0];
  const float drho = fmaf(4.f, M00[1], t00) / 216.f;
  const float rho = k.rho0 + drho;
  const float irho216 = 1.f / (216.f * rho);
  const float U[3] = {fmaf(4.f, M10[1], M10[2] + M10[0]) * irho216, fmaf(4.f, M01[1], M01[2] + M01[0]) * irho216,
                      (M00[2] - M00[0]) * irho216};
  constexpr float k216 = 1.f / 216.f;
  const float pxx = fmaf(4.f, M20[1], M20[2] + M20[0]) * k216;
  const float pyy = fmaf(4.f, M02[1], M02[2] + M02[0]) * k216;
  const float pzz = t00 * k216;
  const float pxy = fmaf(4.f, M11[1], M11[2] + M11[0]) * k216;
  const float pxz = (M10[2] - M10[0]) * k216;
  const float pyz = (M01[2] - M01[0]) * k216;

  // a3: B = sum_i g_i and Lambda_ab = sum_i xi_ia g_ib.
  float dB[3], lam[3][3];
#pragma unroll
  for (int b = 0; b < 3; ++b) {
    dB[b] = 0.25f * sg[b][0] + 0.125f * ((sg[b][1] + sg[b][2]) + (sg[b][3] + sg[b][4]) + (sg[b][5] + sg[b][6]));
    lam[0][b] = 0.125f * (sg[b][1] - sg[b][2]);
    lam[1][b] = 0.125f * (sg[b][3] - sg[b][4]);
    lam[2][b] = 0.125f * (sg[b][5] - sg[b][6]);
  }
  const float B[3] = {k.Bref[0] + dB[0], k.Bref[1] + dB[1], k.Bref[2] + dB[2]};

  // Non-finite guard: one relaxed flag read, and an atomic only while the
  // flag is still clear, so a blown-up field does not serialise on it.
  if (!isfinite(drho + U[0] + U[1] + U[2] + dB[0] + dB[1] + dB[2])) {
    if (*((volatile unsigned*)flag) == 0u) atomicOr(flag, 1u);
  }

  // a4: J + s J x B = y, y = -(omega_B/C^2)(A - 2 U x B), s = 2 alpha_H omega_B / C^2.
  // (Electron MHD: U is neglected against alpha_H J, here and in g^Hall(0).)
  float V[3];
  if constexpr (VAR == kVarFdCurrent) {
    // J = periodic central-difference curl of the pre-collision field
    const long long n3 = g.n3;
    auto Bn = [&](int b, int off) { return Codec<T>::dec(Bfd[b * n3 + site + off]); };
    const float J[3] = {0.5f * ((Bn(2, nb.yp) - Bn(2, nb.ym)) - (Bn(1, nb.zp) - Bn(1, nb.zm))),
                        0.5f * ((Bn(0, nb.zp) - Bn(0, nb.zm)) - (Bn(2, nb.xp) - Bn(2, nb.xm))),
                        0.5f * ((Bn(1, nb.xp) - Bn(1, nb.xm)) - (Bn(0, nb.yp) - Bn(0, nb.ym)))};
#pragma unroll
    for (int a = 0; a < 3; ++a) V[a] = U[a] - k.alphaH * J[a];
  } else {
    const float Ue[3] = {VAR == kVarEmhd ? 0.f : U[0], VAR == kVarEmhd ? 0.f : U[1], VAR == kVarEmhd ? 0.f : U[2]};
    const float gq = 4.f * k.omegaB;
    const float A[3] = {lam[1][2] - lam[2][1], lam[2][0] - lam[0][2], lam[0][1] - lam[1][0]};
    const float uxb[3] = {Ue[1] * B[2] - Ue[2] * B[1], Ue[2] * B[0] - Ue[0] * B[2], Ue[0] * B[1] - Ue[1] * B[0]};
    const float yv[3] = {-gq * (A[0] - 2.f * uxb[0]), -gq * (A[1] - 2.f * uxb[1]), -gq * (A[2] - 2.f * uxb[2])};
    const float sH = 2.f * k.alphaH * gq;
    const float yxb[3] = {yv[1] * B[2] - yv[2] * B[1], yv[2] * B[0] - yv[0] * B[2], yv[0] * B[1] - yv[1] * B[0]};
    const float yb = yv[0] * B[0] + yv[1] * B[1] + yv[2] * B[2];
    const float b2 = B[0] * B[0] + B[1] * B[1] + B[2] * B[2];
    const float iden = 1.f / (1.f + sH * sH * b2);
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      const float J = (yv[a] - sH * yxb[a] + sH * sH * yb * B[a]) * iden;
      V[a] = Ue[a] - k.alphaH * J;
    }
  }

  // a6: magnetic BGK towards g^Hall(0); deviations: rest dB_b, face
  // (axis a, sign +-) dB_b +- Lambda0_ab / C^2, Lambda0_ab = V_a B_b - B_a V_b.
  {
    const float om = k.omegaB, cm = 1.f - k.omegaB;
#pragma unroll
    for (int b = 0; b < 3; ++b) {
      O.p[mslot(b, ODD ? 0 : opp7(0))][site] = Codec<T>::enc(cm * sg[b][0] + om * dB[b]);
#pragma unroll
      for (int a = 0; a < 3; ++a) {
        const float l0 = (a == b) ? 0.f : 4.f * (V[a] * B[b] - B[a] * V[b]);
#pragma unroll
        for (int h = 1; h <= 2; ++h) {
          const int i = 2 * a + h;
          const float v = cm * sg[b][i] + om * (h == 1 ? dB[b] + l0 : dB[b] - l0);
          O.p[mslot(b, ODD ? i : opp7(i))][site + dst_off<ODD>(nb, mx7(i), my7(i), mz7(i))] = Codec<T>::enc(v);
        }
      }
    }
  }

  // a5: fluid.  Dynamic part of the Maxwell stress M(B) - M(B_ref) =
  // miso I - N, N = Bref b + b Bref + b b, miso = Bref.b + |b|^2/2.
  const float bx = dB[0], by = dB[1], bz = dB[2];
  const float Br[3] = {k.Bref[0], k.Bref[1], k.Bref[2]};
  const float Nxx = 2.f * Br[0] * bx + bx * bx, Nyy = 2.f * Br[1] * by + by * by, Nzz = 2.f * Br[2] * bz + bz * bz;
  const float Nxy = Br[0] * by + bx * Br[1] + bx * by;
  const float Nxz = Br[0] * bz + bx * Br[2] + bx * bz;
  const float Nyz = Br[1] * bz + by * Br[2] + by * bz;
  const float miso = Br[0] * bx + Br[1] * by + Br[2] * bz + 0.5f * (bx * bx + by * by + bz * bz);
  // (1 - w) dev(Pi - rho U U - M): the non-equilibrium deviatoric stress.
  const float Sxx = pxx - rho * U[0] * U[0] + Nxx, Syy = pyy - rho * U[1] * U[1] + Nyy,
              Szz = pzz - rho * U[2] * U[2] + Nzz;
  const float r = 1.f - k.omega;
  const float tr3 = (Sxx + Syy + Szz) / 3.f;
  const float Dxx = r * (Sxx - tr3), Dyy = r * (Syy - tr3), Dzz = r * (Szz - tr3);
  const float Dxy = r * (pxy - rho * U[0] * U[1] + Nxy);
  const float Dxz = r * (pxz - rho * U[0] * U[2] + Nxz);
  const float Dyz = r * (pyz - rho * U[1] * U[2] + Nyz);

  // 1-D factors of the x and y axes, divided by the 1-D weight: e = psi/w1 - 1
  // and p0, p1 (p2 is constant), the inverse-moment maps of m0, m1, m2.
  float ex[3], ey[3], p0x[3], p0y[3], p1x[3], p1y[3];
  {
    const float u = U[0], uu = u * u;
    ex[0] = 3.f * uu - 3.f * u, ex[1] = -1.5f * uu, ex[2] = 3.f * uu + 3.f * u;
    p0x[0] = 3.f * (uu - u), p0x[1] = 1.5f * (1.f - uu), p0x[2] = 3.f * (uu + u);
    p1x[0] = 6.f * u - 3.f, p1x[1] = -3.f * u, p1x[2] = 6.f * u + 3.f;
  }
  {
    const float u = U[1], uu = u * u;
    ey[0] = 3.f * uu - 3.f * u, ey[1] = -1.5f * uu, ey[2] = 3.f * uu + 3.f * u;
    p0y[0] = 3.f * (uu - u), p0y[1] = 1.5f * (1.f - uu), p0y[2] = 3.f * (uu + u);
    p1y[0] = 6.f * u - 3.f, p1y[1] = -3.f * u, p1y[2] = 6.f * u + 3.f;
  }
  constexpr float p2[3] = {3.f, -1.5f, 3.f};
  // Along z every term is a quadratic in cz: ez(c) = e0z + e1z c + e2z c^2,
  // p0z(c) = q00 + q10 c + q20 c^2, p1z(c) = q01 + 3 c + q21 c^2,
  // p2z(c) = -1.5 + 4.5 c^2.
  const float uz = U[2], uzz = uz * uz;
  const float e0z = -1.5f * uzz, e1z = 3.f * uz, e2z = 4.5f * uzz;
  const float q00 = 1.5f * (1.f - uzz), q10 = 3.f * uz, q20 = fmaf(4.5f, uzz, -1.5f);
  const float q01 = -3.f * uz, q21 = 9.f * uz;
  // Lorentz term 4.5 (miso (|c|^2 - 1) - c.N.c) + 1.5 tr(N), split as
  // Lxy + Lz1 cz + Lz2 cz^2.
  const float Lbase = 1.5f * (Nxx + Nyy + Nzz) - 4.5f * miso;
  const float LA = 4.5f * (miso - Nxx), LB = 4.5f * (miso - Nyy), LC = 9.f * Nxy;
  const float NX = -9.f * Nxz, NY = -9.f * Nyz, LZ = 4.5f * (miso - Nzz);

  // a7: for each (cx, cy), f*/w - (rest reference) = Z0 + Z1 cz + Z2 cz^2.
#pragma unroll
  for (int py = 0; py < 3; ++py)
#pragma unroll
    for (int px = 0; px < 3; ++px) {
      const int cx = px - 1, cy = py - 1;
      const float exy = ex[px] + ey[py] + ex[px] * ey[py];
      const float g = fmaf(rho, exy, rho);
      // BGK fluid collision: no projected non-equilibrium part; the result is
      // blended with the pre-collision populations below.
      const float A0 = VAR == kVarBgkFluid ? 0.f
                                           : (Dxx * p2[px]) * p0y[py] + (Dyy * p2[py]) * p0x[px] + (Dxy * p1x[px]) * p1y[py];
      const float A1 = VAR == kVarBgkFluid ? 0.f : (Dxz * p1x[px]) * p0y[py] + (Dyz * p1y[py]) * p0x[px];
      const float A2 = VAR == kVarBgkFluid ? 0.f : (Dzz * p0x[px]) * p0y[py];
      float Lxy = Lbase;
      if (cx != 0) Lxy += LA;
      if (cy != 0) Lxy += LB;
      if (cx * cy != 0) Lxy += (cx * cy > 0) ? -LC : LC;
      float Lz1 = 0.f;
      if (cx != 0) Lz1 += (cx > 0) ? NX : -NX;
      if (cy != 0) Lz1 += (cy > 0) ? NY : -NY;
      const float Z0 = fmaf(rho, exy, drho) + g * e0z + A0 * q00 + A1 * q01 - 1.5f * A2 + Lxy;
      const float Z1 = g * e1z + A0 * q10 + 3.f * A1 + Lz1;
      const float Z2 = g * e2z + A0 * q20 + A1 * q21 + 4.5f * A2 + LZ;
      const float tz = Z0 + Z2;
      float vz[3] = {tz - Z1, Z0, tz + Z1};
      if constexpr (VAR == kVarBgkFluid) {
#pragma unroll
        for (int pz = 0; pz < 3; ++pz) vz[pz] = (1.f - k.omega) * s[px + 3 * py + 9 * pz] + k.omega * vz[pz];
      }
#pragma unroll
      for (int pz = 0; pz < 3; ++pz) {
        const int i = idx27(px, py, pz);
        const int slot = ODD ? i : opp27(i);
        O.p[slot][site + dst_off<ODD>(nb, cx, cy, pz - 1)] = Codec<T>::enc(vz[pz]);
      }
    }
}

}  // namespace
}  // namespace flame
