// adjoint.cu -- hand-written vector-Jacobian products of the FLAME step and
// of the initialisation, for gradients of a loss of the final state with
// respect to the initial fields and the Hall length d_i.
//
// Step.  With lambda_{t+1} = dL/df(t+1) (pre-collision populations, natural
// slot order), streaming f(x, q, t+1) = f*(x - c_q, q, t) gives
// dL/df*(x, q) = lambda_{t+1}(x + c_q, q), and the per-site collision's
// transpose Jacobian maps it to lambda_t.  The forward quantities of the
// site (rho, U, Pi, B, Lambda, J, V, D) are recomputed from the state at t.
// Reverse sweep per site (physical populations f, g; gamma = omega_B/C^2,
// s = 2 gamma alpha_H, M = I + s [. x B]):
//   g*  = (1-wB) g + wB g^eq(B, V):   gbar = (1-wB) gbar*; mu = wB W_i gbar*;
//        Bbar += m0 + 4 Q^T V - 4 Q V, Vbar = 4 Q B - 4 Q^T B with
//        m0_b = sum_i mu_bi, Q_ab = sum_i mu_bi xi_ia;
//   V = U - alpha J:  Ubar += Vbar, Jbar = -alpha Vbar, abar -= Vbar.J;
//   J = M^-1 y:       lJ = M^-T Jbar (same closed form with s -> -s),
//        ybar = lJ, sbar = -lJ.(J x B), Bbar -= s lJ x J;
//   s = 2 gamma alpha: abar += 2 gamma sbar;
//   y = -gamma (A - 2 U x B): Abar = -gamma ybar, Ubar += 2 gamma B x ybar,
//        Bbar += 2 gamma ybar x U; Lambdabar_ab = eps_cab Abar_c;
//   f* = rho prod psi(U) + Lorentz(B) + P(D, U), D = (1-w) dev(Pi - rho U U - M(B)):
//        contractions of fbar* with the products of 1-D functions and their
//        U derivatives give rhobar, Ubar, Dbar; Lorentz gives
//        Bbar += 4.5 (tr H B - 2 H B), H = sum_i fbar*_i w_i H2_i;
//        Dbar -> Sbar -> (Pibar, rhobar, Ubar, Bbar);
//   U = j/rho: jbar = Ubar/rho, rhobar -= Ubar.U/rho;
//   moments: fbar_i = rhobar + jbar.c_i + Pibar : c_i c_i,
//            gbar_bi += Bbar_b + sum_a xi_ia Lambdabar_ab.
#include <type_traits>

#include "aa.cuh"
#include "expansion.cuh"
#include "pdl.cuh"

namespace flame {
namespace {

// One site per thread: its 48 state values and the 48 lambda values of x + c_q
// are loaded at once into registers (read-only, with a 256-byte L2 prefetch
// hint), and the whole reverse sweep runs on them.  Bound by memory: with
// the collision left out, these loads and stores alone take 1267 us at 256^3
// FP16 (6.3 TB/s) and 1383 us FP32 (6.9).  What matters is bytes in flight, so
// warps are traded for registers: 64-thread blocks, seven per SM (six for FP32
// storage at odd parity).  us at 256^3, even / odd parity:
//   lambda gathered by 4-byte cp.async into shared memory (bound by those
//   copies: 1483 with the collision left out)       FP32 1572 / 1566, FP16 1512 / 1486
//   lambda loaded after the forward recompute, 128 x 5   1526 / 1706,      1433 / 1724
//   all loads first, 128 threads x 4                     1416 / 1500,      1395 / 1388
//   ... 128 x 3                                          1427 / 1469,      1454 / 1642
//   ... 64 x 7                                           1416 / 1514,      1393 / 1363
//   rows of state and lambda staged by 16-byte cp.async  1661 / 2205,      1540 / 1853
// The d_i contributions are summed per warp in FP64 and the partials added in
// a fixed order by one small kernel.  (Per-warp sums in FP32 gained 0.7 %
// but, where the sites' terms cancel -- a random lambda: sum |a| / |sum a|
// ~ 5000 -- they added ~5x the rounding of the per-site arithmetic to d_i.)
constexpr int kAdjThreads = 64;
template <class T, bool ODD>
constexpr int kAdjMinBlocks = sizeof(T) == 4 && ODD ? 6 : 7;

// The fluid part contracts lambda over the velocity cube with products of 1-D
// functions of the velocity and U: psi (the equilibrium), F0, F1, F2 (the
// inverse-moment maps) and their U derivatives.  On a line (a-, a0, a+) of the
// cube, with h = (a+ - a-)/2 and e = (a- + a+)/2 - a0,
//     F2 = e,  F1 = h + 2 u e,  F0 = a0 + u h + u^2 e,  psi = F0 + e/3,
//     dF0/du = dpsi/du = F1,  dF1/du = 2 e,  and with the 1-D weights
//     w = a0 + e/3,  w c = h/3,  w c^2 = (a0 + e)/3.
// So lambda is first taken into this basis along the three axes (108
// operations, no U), and every contraction is a short polynomial in it.
struct Line {
  float v[3];  // a0, h, e
};
__device__ __forceinline__ Line line(float am, float a0, float ap) {
  return {{a0, 0.5f * (ap - am), fmaf(0.5f, am + ap, -a0)}};
}
__device__ __forceinline__ float f0(float u, float uu, float a, float h, float e) { return fmaf(uu, e, fmaf(u, h, a)); }
__device__ __forceinline__ float f1(float u2, float h, float e) { return fmaf(u2, e, h); }

// The ticket of the sum that follows (sum_partials_kernel), cleared by the kernel
// whose partials it adds: what the memory held before does not matter.
__device__ __forceinline__ void clear_ticket(unsigned* ticket) {
  if ((blockIdx.x | blockIdx.y | blockIdx.z | threadIdx.x | threadIdx.y) == 0) *ticket = 0u;
}

// Per-warp partial sums (no block barrier at the end of the step kernel);
// blocks are whole warps (site_block rounds x to 32).
__device__ __forceinline__ void warp_sum_to(double v, double* out) {
  for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
  if ((threadIdx.x & 31) == 0) *out = v;
}

__device__ __forceinline__ void block_sum_to(double v, double* out) {
  __shared__ double sh[32];
  for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
  const int lane = threadIdx.x & 31, warp = (threadIdx.x + blockDim.x * threadIdx.y) >> 5;
  if (lane == 0) sh[warp] = v;
  __syncthreads();
  if (threadIdx.x == 0 && threadIdx.y == 0) {
    double a = 0.0;
    const int nw = (blockDim.x * blockDim.y + 31) >> 5;
    for (int w = 0; w < nw; ++w) a += sh[w];
    *out = a;
  }
}

// Loads with an L2 prefetch-size hint (the neighbouring warps' segments of the
// same rows arrive with the first request).  Not read-only ones: the kernel may
// have started before the one that writes these buffers ended.
template <class T>
__device__ __forceinline__ float ld_state(const T* p) {
  if constexpr (sizeof(T) == 4) {
    float v;
    asm volatile("ld.global.L2::256B.f32 %0, [%1];" : "=f"(v) : "l"(p));
    return v;
  } else {
    unsigned short h;
    asm volatile("ld.global.L2::256B.b16 %0, [%1];" : "=h"(h) : "l"(p));
    if constexpr (std::is_same_v<T, __half>) return __half2float(__ushort_as_half(h));
    else return __bfloat162float(__ushort_as_bfloat16(h));
  }
}

// Base pointers of lambda_{t+1} (in) and lambda_t (out) per natural slot,
// passed as kernel parameters (as the state's Slots are), so that each of a
// site's 96 lambda accesses is one index computation on a parameter.
struct LamSlots {
  const float* in[kPop];
  float* out[kPop];
};

// The collision's transpose at one site.  sf, sg: the stored pre-collision
// values (deviations over weights); lam: lambda_{t+1} at the site's streamed
// destinations x + c_q, natural slots; out(q, v) takes lambda_t.  Returns the
// site's term of dL/d(d_i).
template <class Out>
__device__ __forceinline__ float adjoint_site(const StepConsts& k, const float (&sf)[kQ], const float (&sg)[3][kM],
                                              const float (&lam)[kPop], const Out& out) {
      // sums of 216 w_i f_i times 1, c_a and c_a c_b, by 1-D passes with (1, 4, 1)
      float drho, jv[3], pv[3][3];
      {
        float m0[9], m1[9], m2[9];
  #pragma unroll
        for (int q = 0; q < 9; ++q) {
          const float am = sf[idx27(0, q % 3, q / 3)], a0 = sf[idx27(1, q % 3, q / 3)], ap = sf[idx27(2, q % 3, q / 3)];
          m2[q] = am + ap;
          m0[q] = fmaf(4.f, a0, m2[q]);
          m1[q] = ap - am;
        }
        float M00[3], M01[3], M02[3], M10[3], M11[3], M20[3];
  #pragma unroll
        for (int pz = 0; pz < 3; ++pz) {
          const int q = 3 * pz;
          M02[pz] = m0[q] + m0[q + 2];
          M00[pz] = fmaf(4.f, m0[q + 1], M02[pz]);
          M01[pz] = m0[q + 2] - m0[q];
          M10[pz] = fmaf(4.f, m1[q + 1], m1[q] + m1[q + 2]);
          M11[pz] = m1[q + 2] - m1[q];
          M20[pz] = fmaf(4.f, m2[q + 1], m2[q] + m2[q + 2]);
        }
        pv[2][2] = M00[0] + M00[2];
        drho = fmaf(4.f, M00[1], pv[2][2]) / 216.f;
        jv[2] = M00[2] - M00[0];
        jv[1] = fmaf(4.f, M01[1], M01[0] + M01[2]);
        pv[1][2] = M01[2] - M01[0];
        pv[1][1] = fmaf(4.f, M02[1], M02[0] + M02[2]);
        jv[0] = fmaf(4.f, M10[1], M10[0] + M10[2]);
        pv[0][2] = M10[2] - M10[0];
        pv[0][1] = fmaf(4.f, M11[1], M11[0] + M11[2]);
        pv[0][0] = fmaf(4.f, M20[1], M20[0] + M20[2]);
      }
      const float rho = k.rho0 + drho;
      const float U[3] = {jv[0] / (216.f * rho), jv[1] / (216.f * rho), jv[2] / (216.f * rho)};
      float dB[3], Lm[3][3];
  #pragma unroll
      for (int b = 0; b < 3; ++b) {
        dB[b] = 0.25f * sg[b][0] + 0.125f * (sg[b][1] + sg[b][2] + sg[b][3] + sg[b][4] + sg[b][5] + sg[b][6]);
        Lm[0][b] = 0.125f * (sg[b][1] - sg[b][2]);
        Lm[1][b] = 0.125f * (sg[b][3] - sg[b][4]);
        Lm[2][b] = 0.125f * (sg[b][5] - sg[b][6]);
      }
      const float B[3] = {k.Bref[0] + dB[0], k.Bref[1] + dB[1], k.Bref[2] + dB[2]};
      const float gam = 4.f * k.omegaB, al = k.alphaH;
      const float Av[3] = {Lm[1][2] - Lm[2][1], Lm[2][0] - Lm[0][2], Lm[0][1] - Lm[1][0]};
      float yv[3];
      {
        const float uxb[3] = {U[1] * B[2] - U[2] * B[1], U[2] * B[0] - U[0] * B[2], U[0] * B[1] - U[1] * B[0]};
  #pragma unroll
        for (int a = 0; a < 3; ++a) yv[a] = -gam * (Av[a] - 2.f * uxb[a]);
      }
      const float s = 2.f * gam * al;
      const float b2 = B[0] * B[0] + B[1] * B[1] + B[2] * B[2];
      const float iden = 1.f / (1.f + s * s * b2);
      float J[3], V[3];
      {
        const float yxb[3] = {yv[1] * B[2] - yv[2] * B[1], yv[2] * B[0] - yv[0] * B[2], yv[0] * B[1] - yv[1] * B[0]};
        const float yb = yv[0] * B[0] + yv[1] * B[1] + yv[2] * B[2];
  #pragma unroll
        for (int a = 0; a < 3; ++a) {
          J[a] = (yv[a] - s * yxb[a] + s * s * yb * B[a]) * iden;
          V[a] = U[a] - al * J[a];
        }
      }
      // D = (1 - w) dev(Pi - rho U U - M(B)); in deviations dev(Pi~ - rho U U + N)
      float D[3][3];
      {
        const float Br[3] = {k.Bref[0], k.Bref[1], k.Bref[2]};
        float S[3][3];
  #pragma unroll
        for (int a = 0; a < 3; ++a)
  #pragma unroll
          for (int b = a; b < 3; ++b) {
            const float N = Br[a] * dB[b] + dB[a] * Br[b] + dB[a] * dB[b];
            S[a][b] = pv[a][b] / 216.f - rho * U[a] * U[b] + N;
          }
        const float r = 1.f - k.omega;
        const float tr3 = (S[0][0] + S[1][1] + S[2][2]) / 3.f;
  #pragma unroll
        for (int a = 0; a < 3; ++a)
  #pragma unroll
          for (int b = a; b < 3; ++b) D[a][b] = r * (a == b ? S[a][b] - tr3 : S[a][b]);
      }

          // ---- magnetic collision
      const float omB = k.omegaB;
      float Bb[3], Vb[3], Q[3][3];  // Q[a][b] = sum_i mu_bi xi_ia
  #pragma unroll
      for (int b = 0; b < 3; ++b) {
        float l[kM];
  #pragma unroll
        for (int i = 0; i < kM; ++i) l[i] = lam[kQ + kM * b + i];
        float m0 = 0.25f * l[0];
  #pragma unroll
        for (int i = 1; i < kM; ++i) m0 += 0.125f * l[i];
        Bb[b] = omB * m0;
  #pragma unroll
        for (int a = 0; a < 3; ++a) Q[a][b] = omB * 0.125f * (l[2 * a + 1] - l[2 * a + 2]);
      }
  #pragma unroll
      for (int c = 0; c < 3; ++c) {
        float qtv = 0.f, qv = 0.f, qb = 0.f, qtb = 0.f;
  #pragma unroll
        for (int a = 0; a < 3; ++a) {
          qtv += Q[a][c] * V[a];
          qv += Q[c][a] * V[a];
          qb += Q[c][a] * B[a];
          qtb += Q[a][c] * B[a];
        }
        Bb[c] += 4.f * (qtv - qv);
        Vb[c] = 4.f * (qb - qtb);
      }
      float Ub[3] = {Vb[0], Vb[1], Vb[2]};
      float Jb[3] = {-al * Vb[0], -al * Vb[1], -al * Vb[2]};
      float abar = -(Vb[0] * J[0] + Vb[1] * J[1] + Vb[2] * J[2]);
      // J = M^-1 y
      float lJ[3];
      {
        const float jxb[3] = {Jb[1] * B[2] - Jb[2] * B[1], Jb[2] * B[0] - Jb[0] * B[2], Jb[0] * B[1] - Jb[1] * B[0]};
        const float jb = Jb[0] * B[0] + Jb[1] * B[1] + Jb[2] * B[2];
  #pragma unroll
        for (int a = 0; a < 3; ++a) lJ[a] = (Jb[a] + s * jxb[a] + s * s * jb * B[a]) * iden;
      }
      {
        const float JxB[3] = {J[1] * B[2] - J[2] * B[1], J[2] * B[0] - J[0] * B[2], J[0] * B[1] - J[1] * B[0]};
        const float sbar = -(lJ[0] * JxB[0] + lJ[1] * JxB[1] + lJ[2] * JxB[2]);
        abar += 2.f * gam * sbar;
        const float lxj[3] = {lJ[1] * J[2] - lJ[2] * J[1], lJ[2] * J[0] - lJ[0] * J[2], lJ[0] * J[1] - lJ[1] * J[0]};
  #pragma unroll
        for (int a = 0; a < 3; ++a) Bb[a] -= s * lxj[a];
      }
      // y = -gamma (A - 2 U x B)
      float Lb[3][3];
      {
        const float* yb = lJ;
        const float bxy[3] = {B[1] * yb[2] - B[2] * yb[1], B[2] * yb[0] - B[0] * yb[2], B[0] * yb[1] - B[1] * yb[0]};
        const float yxu[3] = {yb[1] * U[2] - yb[2] * U[1], yb[2] * U[0] - yb[0] * U[2], yb[0] * U[1] - yb[1] * U[0]};
  #pragma unroll
        for (int a = 0; a < 3; ++a) {
          Ub[a] += 2.f * gam * bxy[a];
          Bb[a] += 2.f * gam * yxu[a];
        }
        const float Ab[3] = {-gam * yb[0], -gam * yb[1], -gam * yb[2]};
        Lb[0][0] = Lb[1][1] = Lb[2][2] = 0.f;
        Lb[1][2] = Ab[0];
        Lb[2][1] = -Ab[0];
        Lb[2][0] = Ab[1];
        Lb[0][2] = -Ab[1];
        Lb[0][1] = Ab[2];
        Lb[1][0] = -Ab[2];
      }

      // ---- fluid collision: contractions of fbar* with products of 1-D functions
      const float Dxx = D[0][0], Dyy = D[1][1], Dzz = D[2][2], Dxy = D[0][1], Dxz = D[0][2], Dyz = D[1][2];
      float rb, Ueq[3], UP[3];
      float Dbxx, Dbyy, Dbzz, Dbxy, Dbxz, Dbyz;
      {
        constexpr float third = 1.f / 3.f;
        float M[3][3][3];  // [z][y][x basis]
  #pragma unroll
        for (int pz = 0; pz < 3; ++pz)
  #pragma unroll
          for (int py = 0; py < 3; ++py) {
            const Line l = line(lam[idx27(0, py, pz)], lam[idx27(1, py, pz)],
                                lam[idx27(2, py, pz)]);
  #pragma unroll
            for (int a = 0; a < 3; ++a) M[pz][py][a] = l.v[a];
          }
  #pragma unroll
        for (int pz = 0; pz < 3; ++pz)
  #pragma unroll
          for (int a = 0; a < 3; ++a) {
            const Line l = line(M[pz][0][a], M[pz][1][a], M[pz][2][a]);
  #pragma unroll
            for (int b = 0; b < 3; ++b) M[pz][b][a] = l.v[b];
          }
  #pragma unroll
        for (int b = 0; b < 3; ++b)
  #pragma unroll
          for (int a = 0; a < 3; ++a) {
            const Line l = line(M[0][b][a], M[1][b][a], M[2][b][a]);
  #pragma unroll
            for (int c = 0; c < 3; ++c) M[c][b][a] = l.v[c];
          }
        // Lorentz: H = sum_i w_i fbar_i H2_i, by w c^2 - w/3 = (2/9) e
        {
          auto w2 = [&](float v0, float v1, float v2, float v3) { return fmaf(third, fmaf(third, v3, v1 + v2), v0); };
          const float Hxx = (2.f / 9.f) * w2(M[0][0][2], M[0][2][2], M[2][0][2], M[2][2][2]);
          const float Hyy = (2.f / 9.f) * w2(M[0][2][0], M[0][2][2], M[2][2][0], M[2][2][2]);
          const float Hzz = (2.f / 9.f) * w2(M[2][0][0], M[2][0][2], M[2][2][0], M[2][2][2]);
          const float Hxy = (1.f / 9.f) * fmaf(third, M[2][1][1], M[0][1][1]);
          const float Hxz = (1.f / 9.f) * fmaf(third, M[1][2][1], M[1][0][1]);
          const float Hyz = (1.f / 9.f) * fmaf(third, M[1][1][2], M[1][1][0]);
          const float trH = Hxx + Hyy + Hzz;
          Bb[0] += 4.5f * (trH * B[0] - 2.f * (Hxx * B[0] + Hxy * B[1] + Hxz * B[2]));
          Bb[1] += 4.5f * (trH * B[1] - 2.f * (Hxy * B[0] + Hyy * B[1] + Hyz * B[2]));
          Bb[2] += 4.5f * (trH * B[2] - 2.f * (Hxz * B[0] + Hyz * B[1] + Hzz * B[2]));
        }
        const float ux = U[0], uy = U[1], uz = U[2], ux2 = 2.f * ux, uy2 = 2.f * uy, uz2 = 2.f * uz;
        const float uxx = ux * ux, uyy = uy * uy, uzz = uz * uz;
        // F0x, F1x and F2x (e), then along y: Bpq[z basis] with x function p and y function q
        float B00[3], B01[3], B02[3], B10[3], B11[3], B12[3], B20[3], B21[3], B22[3];
  #pragma unroll
        for (int c = 0; c < 3; ++c) {
          float A0[3], A1[3], A2[3];
  #pragma unroll
          for (int b = 0; b < 3; ++b) {
            A0[b] = f0(ux, uxx, M[c][b][0], M[c][b][1], M[c][b][2]);
            A1[b] = f1(ux2, M[c][b][1], M[c][b][2]);
            A2[b] = M[c][b][2];
          }
          B00[c] = f0(uy, uyy, A0[0], A0[1], A0[2]);
          B01[c] = f1(uy2, A0[1], A0[2]);
          B02[c] = A0[2];
          B10[c] = f0(uy, uyy, A1[0], A1[1], A1[2]);
          B11[c] = f1(uy2, A1[1], A1[2]);
          B12[c] = A1[2];
          B20[c] = f0(uy, uyy, A2[0], A2[1], A2[2]);
          B21[c] = f1(uy2, A2[1], A2[2]);
          B22[c] = A2[2];
        }
        auto F0z = [&](const float (&v)[3]) { return f0(uz, uzz, v[0], v[1], v[2]); };
        auto F1z = [&](const float (&v)[3]) { return f1(uz2, v[1], v[2]); };
        auto Pz = [&](const float (&v)[3]) { return fmaf(third, v[2], F0z(v)); };
        // equilibrium: rho prod psi and its U derivatives
        {
          float pp[3], dp[3], pd[3];
  #pragma unroll
          for (int c = 0; c < 3; ++c) {
            pp[c] = fmaf(third, fmaf(third, B22[c], B02[c] + B20[c]), B00[c]);
            dp[c] = fmaf(third, B12[c], B10[c]);
            pd[c] = fmaf(third, B21[c], B01[c]);
          }
          rb = Pz(pp);
          Ueq[0] = Pz(dp);
          Ueq[1] = Pz(pd);
          Ueq[2] = F1z(pp);
        }
        // P(D, U): Dbar and the U derivatives
        const float g111 = F1z(B11), g021 = F1z(B02), g120 = F0z(B12), g210 = F0z(B21), g201 = F1z(B20);
        Dbxx = F0z(B20);
        Dbyy = F0z(B02);
        Dbzz = B00[2];
        Dbxy = F0z(B11);
        Dbxz = F1z(B10);
        Dbyz = F1z(B01);
        UP[0] = fmaf(Dyz, g111, fmaf(Dzz, B10[2], fmaf(Dyy, g120, 2.f * fmaf(Dxy, g210, Dxz * g201))));
        UP[1] = fmaf(Dxz, g111, fmaf(Dzz, B01[2], fmaf(Dxx, g210, 2.f * fmaf(Dxy, g120, Dyz * g021))));
        UP[2] = fmaf(Dxy, g111, fmaf(Dyy, g021, fmaf(Dxx, g201, 2.f * fmaf(Dxz, B10[2], Dyz * B01[2]))));
      }
  #pragma unroll
      for (int a = 0; a < 3; ++a) Ub[a] += rho * Ueq[a] + UP[a];
      // D -> S -> (Pi, rho, U, B)
      const float r = 1.f - k.omega;
      const float trD3 = (Dbxx + Dbyy + Dbzz) / 3.f;
      const float Sb[3][3] = {{r * (Dbxx - trD3), r * Dbxy, r * Dbxz},
                              {r * Dbxy, r * (Dbyy - trD3), r * Dbyz},
                              {r * Dbxz, r * Dbyz, r * (Dbzz - trD3)}};
      {
        const float trS = Sb[0][0] + Sb[1][1] + Sb[2][2];
  #pragma unroll
        for (int a = 0; a < 3; ++a) {
          rb -= Sb[a][a] * U[a] * U[a];
          Ub[a] -= 2.f * rho * Sb[a][a] * U[a];
          Bb[a] += -trS * B[a] + 2.f * Sb[a][a] * B[a];
        }
        const int pa[3] = {0, 0, 1}, pb[3] = {1, 2, 2};
  #pragma unroll
        for (int p = 0; p < 3; ++p) {
          const int a = pa[p], b = pb[p];
          rb -= Sb[a][b] * U[a] * U[b];
          Ub[a] -= rho * Sb[a][b] * U[b];
          Ub[b] -= rho * Sb[a][b] * U[a];
          Bb[a] += Sb[a][b] * B[b];
          Bb[b] += Sb[a][b] * B[a];
        }
      }
      // U = j / rho
      const float jb[3] = {Ub[0] / rho, Ub[1] / rho, Ub[2] / rho};
      rb -= (Ub[0] * U[0] + Ub[1] * U[1] + Ub[2] * U[2]) / rho;

      // ---- moments -> populations: fbar_i = rhobar + jbar.c_i + Pibar : c_i c_i,
      // per (c_x, c_y) column as base + lin c_z + Pibar_zz c_z^2
  #pragma unroll
      for (int py = 0; py < 3; ++py)
  #pragma unroll
        for (int px = 0; px < 3; ++px) {
          const int cx = px - 1, cy = py - 1;
          float base = rb, lin = jb[2];
          if (cx != 0) {
            base += (cx > 0 ? jb[0] : -jb[0]) + Sb[0][0];
            lin += cx > 0 ? Sb[0][2] : -Sb[0][2];
          }
          if (cy != 0) {
            base += (cy > 0 ? jb[1] : -jb[1]) + Sb[1][1];
            lin += cy > 0 ? Sb[1][2] : -Sb[1][2];
          }
          if (cx * cy != 0) base += cx * cy > 0 ? Sb[0][1] : -Sb[0][1];
          const float side = base + Sb[2][2];
          out(idx27(px, py, 0), side - lin);
          out(idx27(px, py, 1), base);
          out(idx27(px, py, 2), side + lin);
        }
  #pragma unroll
      for (int b = 0; b < 3; ++b)
  #pragma unroll
        for (int i = 0; i < kM; ++i) {
          float v = (1.f - omB) * lam[kQ + kM * b + i] + Bb[b];
          if (i > 0) {
            const int a = (i - 1) >> 1;
            v += (i & 1) ? Lb[a][b] : -Lb[a][b];
          }
          out(mslot(b, i), v);
        }
  return abar;
}

template <class T, bool ODD>
__global__ void __launch_bounds__(kAdjThreads, (kAdjMinBlocks<T, ODD>))
    adjoint_step_kernel(Slots<T> P, Grid g, StepConsts k, const __grid_constant__ LamSlots L,
                        double* __restrict__ partials, unsigned* __restrict__ ticket) {
  next_kernel_may_come();
  after_previous_kernel();
  clear_ticket(ticket);
  const int x = blockIdx.x * blockDim.x + threadIdx.x;
  const int y = blockIdx.y * blockDim.y + threadIdx.y;
  const int z = blockIdx.z + g.z0;
  double abar_site = 0.0;
  if (x < g.nx && y < g.ny) {
    const int site = (z * g.ny + y) * g.nx + x;
    const Nbr nb = make_nbr(x, y, z, g);
    float sf[kQ], sg[3][kM], lam[kPop];
#pragma unroll
    for (int i = 0; i < kQ; ++i)
      sf[i] = ld_state<T>(P.p[ODD ? opp27(i) : i] + site + src_off<ODD>(nb, cx27(i), cy27(i), cz27(i)));
#pragma unroll
    for (int b = 0; b < 3; ++b)
#pragma unroll
      for (int i = 0; i < kM; ++i)
        sg[b][i] = ld_state<T>(P.p[mslot(b, ODD ? opp7(i) : i)] + site + src_off<ODD>(nb, mx7(i), my7(i), mz7(i)));
    // dL/df* by the streaming transpose: lambda_{t+1} at x + c_q
#pragma unroll
    for (int q = kQ; q < kPop; ++q) {
      const int i = (q - kQ) % kM;
      lam[q] = ld_state<float>(L.in[q] + site + nb(mx7(i), my7(i), mz7(i)));
    }
#pragma unroll
    for (int q = 0; q < kQ; ++q) lam[q] = ld_state<float>(L.in[q] + site + nb(cx27(q), cy27(q), cz27(q)));
    abar_site = (double)adjoint_site(k, sf, sg, lam, [&](int q, float v) { L.out[q][site] = v; });
  }
  const long long blk = ((long long)blockIdx.z * gridDim.y + blockIdx.y) * gridDim.x + blockIdx.x;
  const int warp = (threadIdx.x + blockDim.x * threadIdx.y) >> 5;
  warp_sum_to(abar_site, partials + blk * ((blockDim.x * blockDim.y) >> 5) + warp);
}

// ---------------------------------------------------------------------------
// Initialisation adjoint (FP64), local part: per site the contributions to
// u_bar and B_bar that do not go through a gradient, and the adjoints of the
// central-difference gradients (d_a u_b, d_a B_b at [3a+b]).
//
// Bound by the FP64 pipe (1/64 of the FP32 rate, conversions included):
// per-velocity sums with every product written out took ~1430 operations a
// site, 675 us at 64^3.  Now the sums that do not depend on the fields run
// as three-term FP32 expansions of the FP32 lambda, lambda is widened by its
// bits, and the equilibrium's U derivatives are separable 1-D passes that
// share their partial sums, in FP64 (90 operations of ~175): 100 us.

// The power of two that keeps sums of n values within FP32's range (1 but
// for values near its end).
template <int N>
__device__ __forceinline__ float sum_scale(const float (&l)[N]) {
  float m = 0.f;
#pragma unroll
  for (int i = 0; i < N; ++i) m = fmaxf(m, fabsf(l[i]));
  return m < 0x1p100f ? 1.f : 0x1p-20f;
}

// 216 sum_i w_i l_i times 1, c_a c_b of l in velocity-cube order: r, and
// R = xx, yy, zz, xy, xz, yz.
__device__ __forceinline__ void second_sums(const float (&lam)[kQ], double& r, double (&R)[6]) {
  const float sc = sum_scale(lam);
  float l[kQ];
#pragma unroll
  for (int q = 0; q < kQ; ++q) l[q] = sc * lam[q];
  F3 Y00[3], Y02[3], Y10[3], Y20[3], Y01[3], Y11[3];  // [x function][y function] per pz
#pragma unroll
  for (int pz = 0; pz < 3; ++pz) {
    F3 a0[3];
    F2 a1[3], a2[3];
#pragma unroll
    for (int py = 0; py < 3; ++py) {
      const int q = 3 * (py + 3 * pz);
      a2[py] = two_sum(l[q + 2], l[q]);
      a1[py] = two_diff(l[q + 2], l[q]);
      a0[py] = add3(a2[py], 4.f * l[q + 1]);
    }
    Y02[pz] = add3(a0[2], a0[0]);
    Y00[pz] = add3(Y02[pz], scaled(4.f, a0[1]));
    Y01[pz] = add3(a0[2], -a0[0]);
    Y10[pz] = add3(add3(a1[2], a1[0]), scaled(4.f, a1[1]));
    Y11[pz] = add3(a1[2], -a1[0]);
    Y20[pz] = add3(add3(a2[2], a2[0]), scaled(4.f, a2[1]));
  }
  auto w = [](const F3 (&y)[3]) { return to_double(add3(add3(y[2], y[0]), scaled(4.f, y[1]))); };
  auto c = [](const F3 (&y)[3]) { return to_double(add3(y[2], -y[0])); };
  r = w(Y00);
  R[0] = w(Y20);
  R[1] = w(Y02);
  R[2] = to_double(add3(Y00[2], Y00[0]));
  R[3] = w(Y11);
  R[4] = c(Y10);
  R[5] = c(Y01);
  if (sc != 1.f) {
    r *= 0x1p20;
#pragma unroll
    for (int i = 0; i < 6; ++i) R[i] *= 0x1p20;
  }
}

// psi(u) and its derivative at c = -1, 0, 1 (the undivided 1-D equilibrium).
struct Axis64 {
  double psi[3], dpsi[3];
  __device__ __forceinline__ explicit Axis64(double u) {
    const double h = fma(0.5 * u, u, 1.0 / 6.0), g = 0.5 * u;
    psi[0] = h - g;
    psi[1] = fma(-u, u, 2.0 / 3.0);
    psi[2] = h + g;
    dpsi[0] = u - 0.5;
    dpsi[1] = -2.0 * u;
    dpsi[2] = u + 0.5;
  }
};
__device__ __forceinline__ double dot3(const double (&f)[3], double a, double b, double c) {
  return fma(f[2], c, fma(f[1], b, f[0] * a));
}

__global__ void __launch_bounds__(128, 4)
    init_adjoint_local_kernel(Grid g, StepConsts k, const double* __restrict__ u,
                                          const double* __restrict__ Bf, const float* __restrict__ lam,
                                          double* __restrict__ ubl, double* __restrict__ Bbl,
                                          double* __restrict__ dub, double* __restrict__ dBb,
                                          double* __restrict__ partials, unsigned* __restrict__ ticket) {
  clear_ticket(ticket);
  const int x = blockIdx.x * blockDim.x + threadIdx.x;
  const int y = blockIdx.y * blockDim.y + threadIdx.y;
  const int z = blockIdx.z + g.z0;
  double abar = 0.0;
  if (x < g.nx && y < g.ny) {
    const long long n3 = g.n3;
    const long long site = ((long long)z * g.ny + y) * g.nx + x;
    float l[kQ];
#pragma unroll
    for (int q = 0; q < kQ; ++q) l[q] = lam[(long long)idx27(q % 3, (q / 3) % 3, q / 9) * n3 + site];
    const double U[3] = {u[site], u[n3 + site], u[2 * n3 + site]};

    // equilibrium part of u_bar: sum_i l_i d(psi psi psi)/du_a
    double Ub[3];
    {
      const Axis64 ax(U[0]), ay(U[1]), az(U[2]);
      double P[3], Px[3], Py[3];  // per pz: psi psi, dpsi psi, psi dpsi
#pragma unroll
      for (int pz = 0; pz < 3; ++pz) {
        double X[3], D[3];
#pragma unroll
        for (int py = 0; py < 3; ++py) {
          const int q = 3 * (py + 3 * pz);
          const double a = widened(l[q]), b = widened(l[q + 1]), c = widened(l[q + 2]);
          X[py] = dot3(ax.psi, a, b, c);
          D[py] = dot3(ax.dpsi, a, b, c);
        }
        P[pz] = dot3(ay.psi, X[0], X[1], X[2]);
        Py[pz] = dot3(ay.dpsi, X[0], X[1], X[2]);
        Px[pz] = dot3(ay.psi, D[0], D[1], D[2]);
      }
      Ub[0] = dot3(az.psi, Px[0], Px[1], Px[2]);
      Ub[1] = dot3(az.psi, Py[0], Py[1], Py[2]);
      Ub[2] = dot3(az.dpsi, P[0], P[1], P[2]);
    }
    // H = sum_i l_i w_i H2_i; Lorentz part of B_bar; the gradients of u
    const double B[3] = {Bf[site], Bf[n3 + site], Bf[2 * n3 + site]};
    double Bb[3];
    {
      double r0, R[6];
      second_sums(l, r0, R);
      const double k216 = 1.0 / 216.0, t3 = r0 * (1.0 / 648.0);
      const double Hd[3] = {fma(R[0], k216, -t3), fma(R[1], k216, -t3), fma(R[2], k216, -t3)};
      const double Hxy = R[3] * k216, Hxz = R[4] * k216, Hyz = R[5] * k216;
      const double trH = Hd[0] + Hd[1] + Hd[2];
      Bb[0] = 4.5 * (trH * B[0] - 2.0 * dot3(B, Hd[0], Hxy, Hxz));
      Bb[1] = 4.5 * (trH * B[1] - 2.0 * dot3(B, Hxy, Hd[1], Hyz));
      Bb[2] = 4.5 * (trH * B[2] - 2.0 * dot3(B, Hxz, Hyz, Hd[2]));
      const double cu = -3.0 / (double)k.omega;  // rho = 1 initial density
      const double off[3] = {cu * Hxy, cu * Hxz, cu * Hyz};
#pragma unroll
      for (int a = 0; a < 3; ++a)
#pragma unroll
        for (int b = 0; b < 3; ++b) dub[(3 * a + b) * n3 + site] = a == b ? cu * Hd[a] : off[a + b - 1];
    }
    // Hall equilibrium: mu = W lg, m0, Q[a][b] = sum_i mu_bi xi_ia
    double Q[3][3];
#pragma unroll
    for (int b = 0; b < 3; ++b) {
      float lg[kM];
#pragma unroll
      for (int i = 0; i < kM; ++i) lg[i] = lam[(long long)mslot(b, i) * n3 + site];
      const float sc = sum_scale(lg);
#pragma unroll
      for (int i = 0; i < kM; ++i) lg[i] *= sc;
      const F3 m0 = add3(add3(add3(two_sum(lg[1], lg[2]), two_sum(lg[3], lg[4])), two_sum(lg[5], lg[6])), 2.f * lg[0]);
      double m = to_double(scaled(0.125f, m0));
#pragma unroll
      for (int a = 0; a < 3; ++a) Q[a][b] = to_double(scaled(0.125f, two_diff(lg[2 * a + 1], lg[2 * a + 2])));
      if (sc != 1.f) {
        m *= 0x1p20;
#pragma unroll
        for (int a = 0; a < 3; ++a) Q[a][b] *= 0x1p20;
      }
      Bb[b] += m;
    }
    // central-difference J0 = curl B, V = u - d_i J0
    const double al = (double)k.alphaH;
    double J0[3], V[3];
    {
      const int xp = x + 1 == g.nx ? 0 : x + 1, xm = x == 0 ? g.nx - 1 : x - 1;
      const int yp = y + 1 == g.ny ? 0 : y + 1, ym = y == 0 ? g.ny - 1 : y - 1;
      const int zp = z + 1 == g.nz ? 0 : z + 1, zm = z == 0 ? g.nz - 1 : z - 1;
      auto at = [&](int b, int xx, int yy, int zz) { return Bf[b * n3 + ((long long)zz * g.ny + yy) * g.nx + xx]; };
      auto dx = [&](int b) { return at(b, xp, y, z) - at(b, xm, y, z); };
      auto dy = [&](int b) { return at(b, x, yp, z) - at(b, x, ym, z); };
      auto dz = [&](int b) { return at(b, x, y, zp) - at(b, x, y, zm); };
      J0[0] = 0.5 * (dy(2) - dz(1));
      J0[1] = 0.5 * (dz(0) - dx(2));
      J0[2] = 0.5 * (dx(1) - dy(0));
#pragma unroll
      for (int a = 0; a < 3; ++a) V[a] = fma(-al, J0[a], U[a]);
    }
    // Bbar += 4 (Q^T V - Q V), Vbar = 4 (Q B - Q^T B): by the antisymmetric part of Q
    const double X01 = 4.0 * (Q[0][1] - Q[1][0]), X02 = 4.0 * (Q[0][2] - Q[2][0]), X12 = 4.0 * (Q[1][2] - Q[2][1]);
    Bb[0] -= fma(X01, V[1], X02 * V[2]);
    Bb[1] += fma(X01, V[0], -X12 * V[2]);
    Bb[2] += fma(X02, V[0], X12 * V[1]);
    const double Vb[3] = {fma(X01, B[1], X02 * B[2]), fma(-X01, B[0], X12 * B[2]), -fma(X02, B[0], X12 * B[1])};
    abar = -(Vb[0] * J0[0] + Vb[1] * J0[1] + Vb[2] * J0[2]);
    const double iwB = 1.0 / (double)k.omegaB;
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      ubl[a * n3 + site] = Ub[a] + Vb[a];
      Bbl[a * n3 + site] = Bb[a];
#pragma unroll
      for (int b = 0; b < 3; ++b) {
        // -Q / omega_B, and through J0 = curl B the adjoint -d_i Vbar
        double d = -iwB * Q[a][b];
        if (b == (a + 1) % 3) d = fma(-al, Vb[(a + 2) % 3], d);
        if (b == (a + 2) % 3) d = fma(al, Vb[(a + 1) % 3], d);
        dBb[(3 * a + b) * n3 + site] = d;
      }
    }
  }
  const long long blk = ((long long)blockIdx.z * gridDim.y + blockIdx.y) * gridDim.x + blockIdx.x;
  block_sum_to(abar, partials + blk);
}

// Transpose of the periodic central difference: F_bar(y) += 1/2 (G(y - e_a) - G(y + e_a)).
__global__ void init_adjoint_stencil_kernel(Grid g, const double* __restrict__ ubl, const double* __restrict__ Bbl,
                                            const double* __restrict__ dub, const double* __restrict__ dBb,
                                            double* __restrict__ ubar, double* __restrict__ Bbar) {
  const int x = blockIdx.x * blockDim.x + threadIdx.x;
  const int y = blockIdx.y * blockDim.y + threadIdx.y;
  const int z = blockIdx.z + g.z0;
  if (x >= g.nx || y >= g.ny) return;
  const long long n3 = g.n3;
  const long long site = ((long long)z * g.ny + y) * g.nx + x;
  const int xp = x + 1 == g.nx ? 0 : x + 1, xm = x == 0 ? g.nx - 1 : x - 1;
  const int yp = y + 1 == g.ny ? 0 : y + 1, ym = y == 0 ? g.ny - 1 : y - 1;
  const int zp = z + 1 == g.nz ? 0 : z + 1, zm = z == 0 ? g.nz - 1 : z - 1;
  const long long m[3] = {((long long)z * g.ny + y) * g.nx + xm, ((long long)z * g.ny + ym) * g.nx + x,
                          ((long long)zm * g.ny + y) * g.nx + x};
  const long long p[3] = {((long long)z * g.ny + y) * g.nx + xp, ((long long)z * g.ny + yp) * g.nx + x,
                          ((long long)zp * g.ny + y) * g.nx + x};
  for (int b = 0; b < 3; ++b) {
    double vb = Bbl[b * n3 + site], vu = ubl[b * n3 + site];
    for (int a = 0; a < 3; ++a) {
      const double* G = dBb + (3 * a + b) * n3;
      const double* Gu = dub + (3 * a + b) * n3;
      vb += 0.5 * (G[m[a]] - G[p[a]]);
      vu += 0.5 * (Gu[m[a]] - Gu[p[a]]);
    }
    if (Bbar) Bbar[b * n3 + site] = vb;
    if (ubar) ubar[b * n3 + site] = vu;
  }
}

// Deterministic sum of n partials: up to kSumBlocks blocks sum fixed chunks into
// stage[], and the last of them to finish, by the ticket, adds the stage in a fixed
// order.  (Two kernels had taken 8 us a step.)
constexpr int kSumBlocks = 64;
constexpr int kSumThreads = 256;
__device__ __forceinline__ double sum_of_block(double a) {
  __shared__ double sh[kSumThreads / 32];
  for (int o = 16; o > 0; o >>= 1) a += __shfl_down_sync(0xffffffffu, a, o);
  if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = a;
  __syncthreads();
  a = 0.0;
  if (threadIdx.x == 0)
    for (int w = 0; w < kSumThreads / 32; ++w) a += sh[w];
  return a;
}
__global__ void __launch_bounds__(kSumThreads)
    sum_partials_kernel(const double* partials, long long n, double* stage, unsigned* ticket,
                        double* __restrict__ out) {
  __shared__ bool last;
  next_kernel_may_come();
  after_previous_kernel();
  const long long per = (n + gridDim.x - 1) / gridDim.x;
  const long long lo = per * blockIdx.x, hi = lo + per < n ? lo + per : n;
  double a = 0.0;
  for (long long i = lo + threadIdx.x; i < hi; i += kSumThreads) a += __ldcg(partials + i);
  a = sum_of_block(a);
  if (threadIdx.x == 0) {
    __stcg(stage + blockIdx.x, a);
    __threadfence();
    last = atomicAdd(ticket, 1u) == gridDim.x - 1;
    __threadfence();
  }
  __syncthreads();
  if (!last) return;
  double t = threadIdx.x < gridDim.x ? load_l2(stage + threadIdx.x) : 0.0;
  t = sum_of_block(t);
  if (threadIdx.x == 0) *out = t;
}
// The buffer holds cap partials, kSumBlocks doubles and the ticket.
inline unsigned* ticket_of(double* partials, long long cap) {
  return reinterpret_cast<unsigned*>(partials + cap + kSumBlocks);
}
// Sum of n partials into *out.
inline cudaError_t sum_partials(double* partials, long long cap, long long n, double* out, cudaStream_t s) {
  const long long want = (n + 4 * kSumThreads - 1) / (4 * kSumThreads);
  double* stage = partials + cap;
  return launch_chained(sum_partials_kernel, dim3((unsigned)(want < kSumBlocks ? want : kSumBlocks)), dim3(kSumThreads), 0,
                        s, static_cast<const double*>(partials), n, stage, ticket_of(partials, cap), out);
}

// The partials of either adjoint: one per warp of the step kernel, one per
// block of the initialisation's.
inline long long partials_cap(const Grid& g) {
  const dim3 b = site_block(g, kAdjThreads), gr = site_grid(g, b);
  const dim3 bi = site_block(g, 128), gi = site_grid(g, bi);
  const long long a = (long long)gr.x * gr.y * gr.z * ((b.x * b.y) >> 5), c = (long long)gi.x * gi.y * gi.z;
  return a > c ? a : c;
}

template <class T>
cudaError_t adjoint_t(int odd, const void* pop, Grid g, const StepConsts& k, const float* lin, float* lout,
                      double* partials, double* ddi, cudaStream_t s) {
  const dim3 b = site_block(g, kAdjThreads), gr = site_grid(g, b);
  const long long nblk = (long long)gr.x * gr.y * gr.z;
  const Slots<T> P = make_slots<T>(pop, g);
  LamSlots L;
  for (int q = 0; q < kPop; ++q) {
    L.in[q] = lin + (size_t)q * (size_t)g.n3;
    L.out[q] = lout + (size_t)q * (size_t)g.n3;
  }
  const long long cap = partials_cap(g);
  auto go = [&](auto kern) { return launch_chained(kern, gr, b, 0, s, P, g, k, L, partials, ticket_of(partials, cap)); };
  const cudaError_t e = odd ? go(adjoint_step_kernel<T, true>) : go(adjoint_step_kernel<T, false>);
  if (e != cudaSuccess) return e;
  return sum_partials(partials, cap, nblk * ((b.x * b.y) >> 5), ddi, s);
}

}  // namespace

long long adjoint_partials_needed(Grid g) { return partials_cap(g) + kSumBlocks + 1; }

cudaError_t launch_step_adjoint(int storage, int odd, const void* pop, Grid g, const StepConsts& k, const float* lin,
                                float* lout, double* partials, double* ddi, cudaStream_t s) {
  switch (storage) {
    case 1: return adjoint_t<float>(odd, pop, g, k, lin, lout, partials, ddi, s);
    case 2: return adjoint_t<__half>(odd, pop, g, k, lin, lout, partials, ddi, s);
    case 3: return adjoint_t<__nv_bfloat16>(odd, pop, g, k, lin, lout, partials, ddi, s);
  }
  return cudaErrorInvalidValue;
}

cudaError_t launch_init_adjoint(Grid g, const StepConsts& k, const double* u, const double* B, const float* lam,
                                double* ws, double* partials, double* ubar, double* Bbar, double* ddi,
                                cudaStream_t s) {
  const dim3 b = site_block(g, 128), gr = site_grid(g, b);
  const long long n3 = g.n3;
  double* ubl = ws;
  double* Bbl = ws + 3 * n3;
  double* dub = ws + 6 * n3;
  double* dBb = ws + 15 * n3;
  const long long cap = partials_cap(g);
  init_adjoint_local_kernel<<<gr, b, 0, s>>>(g, k, u, B, lam, ubl, Bbl, dub, dBb, partials, ticket_of(partials, cap));
  init_adjoint_stencil_kernel<<<gr, b, 0, s>>>(g, ubl, Bbl, dub, dBb, ubar, Bbar);
  const cudaError_t e = sum_partials(partials, cap, (long long)gr.x * gr.y * gr.z, ddi, s);
  if (e != cudaSuccess) return e;
  return cudaGetLastError();
}

}  // namespace flame
