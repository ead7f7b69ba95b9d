// diag.cu -- kernels that read or write the population state outside the
// hot path: initialisation from macroscopic fields, moments and
// decoded populations (FP64), and the deterministic FP64 reduction of the
// scalar diagnostics.
#include <type_traits>

#include "aa.cuh"
#include "expansion.cuh"
#include "reduce_final.cuh"

namespace flame {
namespace {

// ---------------------------------------------------------------------------
// Initialisation (once per run).  The arithmetic type R is FP32 for 16-bit
// storage, whose encoding rounds to 2^-11 (FP16) or 2^-8 (BF16) relative, far
// above FP32's 2^-24; the gradients too are taken in R.  FP32 storage takes
// two-term FP32 arithmetic, and FP64 where that does not reach (init_columns).

// Periodic central difference of field f along axis a at (x, y, z), in the
// per-site arithmetic type R (GB300's FP64 pipe is 1/64 of its FP32 rate, so
// 16-bit storage, whose values keep 11 or 8 bits, takes them in FP32).
template <class R, class F>
__device__ __forceinline__ R cdiff(const F* f, int a, int x, int y, int z, const Grid& g) {
  int xp = x, xm = x, yp = y, ym = y, zp = z, zm = z;
  if (a == 0) {
    xp = x + 1 == g.nx ? 0 : x + 1;
    xm = x == 0 ? g.nx - 1 : x - 1;
  } else if (a == 1) {
    yp = y + 1 == g.ny ? 0 : y + 1;
    ym = y == 0 ? g.ny - 1 : y - 1;
  } else {
    zp = z + 1 == g.nz ? 0 : z + 1;
    zm = z == 0 ? g.nz - 1 : z - 1;
  }
  return (R)0.5 * ((R)f[((long long)zp * g.ny + yp) * g.nx + xp] - (R)f[((long long)zm * g.ny + ym) * g.nx + xm]);
}

// F: the element type of the caller's fields (FP64 for flame_init, FP32 for
// flame_init_f32).  Writes the site's populations and returns its speed
// max(|B|/sqrt(rho), |u|).
template <class T, class R, class F>
__device__ __forceinline__ float init_site(T* __restrict__ pop, const Grid& g, const StepConsts& k, int noneq,
                                           const F* __restrict__ rho_f, const F* __restrict__ u,
                                           const F* __restrict__ Bf, const F* __restrict__ gu,
                                           const F* __restrict__ gB, int x, int y, int z) {
      const long long n3 = g.n3;
      const long long site = ((long long)z * g.ny + y) * g.nx + x;
      const R rho = rho_f ? (R)rho_f[site] : (R)1;
      const R U[3] = {(R)u[site], (R)u[n3 + site], (R)u[2 * n3 + site]};
      const R B[3] = {(R)Bf[site], (R)Bf[n3 + site], (R)Bf[2 * n3 + site]};
      R du[9], dB[9];
  #pragma unroll
      for (int a = 0; a < 3; ++a)
  #pragma unroll
        for (int b = 0; b < 3; ++b) {
          du[3 * a + b] = gu ? (R)gu[(3 * a + b) * n3 + site] : cdiff<R>(u + b * n3, a, x, y, z, g);
          dB[3 * a + b] = gB ? (R)gB[(3 * a + b) * n3 + site] : cdiff<R>(Bf + b * n3, a, x, y, z, g);
        }
      const R J0[3] = {dB[5] - dB[7], dB[6] - dB[2], dB[1] - dB[3]};  // curl B
      const R omega = (R)k.omega, omegaB = (R)k.omegaB, aH = (R)k.alphaH;
      const R Br[3] = {(R)k.Bref[0], (R)k.Bref[1], (R)k.Bref[2]};
      const R b[3] = {B[0] - Br[0], B[1] - Br[1], B[2] - Br[2]};
      R N[3][3];
  #pragma unroll
      for (int a = 0; a < 3; ++a)
  #pragma unroll
        for (int c = 0; c < 3; ++c) N[a][c] = Br[a] * b[c] + b[a] * Br[c] + b[a] * b[c];
      const R miso = Br[0] * b[0] + Br[1] * b[1] + Br[2] * b[2] + (R)0.5 * (b[0] * b[0] + b[1] * b[1] + b[2] * b[2]);
      const R trN3 = (N[0][0] + N[1][1] + N[2][2]) / (R)3;
      R Pn[3][3];  // first-order non-equilibrium stress -(rho cs^2/omega)(du + du^T)
  #pragma unroll
      for (int a = 0; a < 3; ++a)
  #pragma unroll
        for (int c = 0; c < 3; ++c) Pn[a][c] = noneq ? -(rho / ((R)3 * omega)) * (du[3 * a + c] + du[3 * c + a]) : (R)0;
      const R trPn3 = (Pn[0][0] + Pn[1][1] + Pn[2][2]) / (R)3;
      const R drho = rho - (R)k.rho0;
  #pragma unroll
      for (int i = 0; i < kQ; ++i) {
        const int c[3] = {cx27(i), cy27(i), cz27(i)};
        R E = 0;  // prod(psi/w1) - 1, accumulated stably
  #pragma unroll
        for (int a = 0; a < 3; ++a) {
          const R uu = U[a] * U[a];
          const R ea = c[a] == 0 ? (R)-1.5 * uu : (R)3 * uu + (R)(3 * c[a]) * U[a];
          E = E + ea + E * ea;
        }
        R cNc = 0, cPc = 0;
  #pragma unroll
        for (int a = 0; a < 3; ++a)
  #pragma unroll
          for (int d = 0; d < 3; ++d) {
            if (c[a] * c[d] == 0) continue;
            cNc += (R)(c[a] * c[d]) * N[a][d];
            cPc += (R)(c[a] * c[d]) * Pn[a][d];
          }
        const R c2 = (R)(c[0] * c[0] + c[1] * c[1] + c[2] * c[2]);
        const R L = (R)4.5 * (miso * (c2 - (R)1) - cNc + trN3);
        const R ne = (R)4.5 * (cPc - trPn3);
        pop[(long long)phys(i) * n3 + site] = Codec<T>::enc((float)(drho + rho * E + L + ne));
      }
      const R V[3] = {U[0] - aH * J0[0], U[1] - aH * J0[1], U[2] - aH * J0[2]};
  #pragma unroll
      for (int bb = 0; bb < 3; ++bb)
  #pragma unroll
        for (int i = 0; i < kM; ++i) {
          const int xi[3] = {mx7(i), my7(i), mz7(i)};
          R l0 = 0, ne = 0;
  #pragma unroll
          for (int a = 0; a < 3; ++a) {
            if (xi[a] == 0) continue;
            l0 += (R)xi[a] * (V[a] * B[bb] - B[a] * V[bb]);
            ne += (R)xi[a] * dB[3 * a + bb];
          }
          const R v = b[bb] + (R)4 * l0 - (noneq ? ne / omegaB : (R)0);
          pop[(long long)phys(mslot(bb, i)) * n3 + site] = Codec<T>::enc((float)v);
        }
      const R va = sqrt((B[0] * B[0] + B[1] * B[1] + B[2] * B[2]) / rho);
      const R um = sqrt(U[0] * U[0] + U[1] * U[1] + U[2] * U[2]);
      return (float)fmax(va, um);
}

// FP32 storage: the populations are FP64 values rounded to FP32.  Their ~770
// FP64 operations a site (and conversions, which cost as much) were all this
// kernel did: 2932 us at 128^3 (23.4 ms at 256^3), where the bytes take 74.
// They are computed in two-term FP32 arithmetic (48 bits) and in the columns of
// the step's collision: for each (c_x, c_y) the three values along c_z are
// Z0 + Z1 c_z + Z2 c_z^2, the Lorentz term's N and the non-equilibrium stress P
// entering as K = N - P.  Differences of the fields and of the reference state
// are taken in FP64, as FP64 would (22 operations a site: the fields' own 48 bits
// would leave less of a small deviation), and split by integer operations.
//
// A value whose rounding the two terms cannot tell (put_rounded) is stored as
// FP64 gives it: its site is done again there, in the same columns (with every
// velocity's products written out that took ~770 operations, now ~330).  So are
// sites with values outside [2^-10, 2^10] (density) or of 2^40 and more (fields).
//
// 128^3 417 us, 256^3 3.2 ms (FP32 fields 302 us and 2.1 ms), bound by FP32 issue
// and the sites done again, one in 1000 to 2000 of random fields: 321 us without
// them.  Where populations cancel at every site (a wave with u = b) all are: 1.4 ms
// (1.6 ms).  Five blocks of 128 threads per SM instead of six, whose 80 registers
// reload some field values: 5 % slower.
struct InitConsts {
  F2 p;    // -1 / (3 omega), or 0 without the non-equilibrium parts
  F2 iwB;  // 1 / omega_B, or 0
  double w3, iw3, wB, iwB64;  // 3 omega, omega_B and their reciprocals
};

// a / b given r = 1 / b: the remainder of the first quotient corrects it.
__device__ __forceinline__ double quotient(double a, double b, double r) {
  const double q = a * r;
  return fma(fma(-q, b, a), r, q);
}

// The two arithmetics of the columns below.
struct TwoTerm {
  using V = F2;
  static __device__ __forceinline__ F2 field(double f) { return from_double(f); }
  static __device__ __forceinline__ F2 field(float f) { return {f, 0.f}; }
  // f - g, rounded to FP64 or exactly
  static __device__ __forceinline__ F2 diff(double f, double g) { return from_double(f - g); }
  static __device__ __forceinline__ F2 diff(float f, float g) { return two_diff(f, g); }
  static __device__ __forceinline__ F2 add(F2 a, F2 b) { return add2(a, b); }
  static __device__ __forceinline__ F2 add(F2 a, float b) { return add2(a, b); }
  static __device__ __forceinline__ F2 addu(F2 a, F2 b) { return add2u(a, b); }
  static __device__ __forceinline__ F2 mul(F2 a, F2 b) { return mul2(a, b); }
  static __device__ __forceinline__ F2 mul(float a, F2 b) { return mul2(a, b); }
  static __device__ __forceinline__ F2 twice(float c, F2 a) { return scaled(c, a); }  // c a power of two
  static __device__ __forceinline__ float head(F2 a) { return a.h; }
  // -rho / (3 omega), d / omega_B
  static __device__ __forceinline__ F2 stress(const InitConsts& ic, int, F2 rho) { return mul2(rho, ic.p); }
  static __device__ __forceinline__ F2 relaxed(const InitConsts& ic, int, F2 d) { return mul2(ic.iwB, d); }
};
struct Fp64 {
  using V = double;
  static __device__ __forceinline__ double field(double f) { return f; }
  static __device__ __forceinline__ double field(float f) { return widened(f); }
  static __device__ __forceinline__ double diff(double f, double g) { return f - g; }
  static __device__ __forceinline__ double diff(float f, float g) { return widened(f) - widened(g); }
  static __device__ __forceinline__ double add(double a, double b) { return a + b; }
  static __device__ __forceinline__ double addu(double a, double b) { return a + b; }
  static __device__ __forceinline__ double mul(double a, double b) { return a * b; }
  static __device__ __forceinline__ double twice(double c, double a) { return c * a; }
  static __device__ __forceinline__ float head(double) { return 0.f; }  // no magnitudes are kept
  static __device__ __forceinline__ double stress(const InitConsts& ic, int noneq, double rho) {
    return noneq ? -quotient(rho, ic.w3, ic.iw3) : 0.0;
  }
  static __device__ __forceinline__ double relaxed(const InitConsts& ic, int noneq, double d) {
    return noneq ? quotient(d, ic.wB, ic.iwB64) : 0.0;
  }
};

// The error of a sum of two-term values whose terms' magnitudes add up to m: 2^-46
// m, and what underflow takes of some tens of products; none where there is no
// term.  Against 113-bit arithmetic (random fields of 1e-9 to 0.3 on mean fields of
// 0 and 0.1, with and without given gradients, 24M values) the error is 2^-45 m at
// most and so seldom above 2^-46 m that 3e-10 values a site round to another FP32
// number than FP64's exact result would, where FP64 arithmetic itself rounds 1e-6
// to 4e-6 a site the other way.
__device__ __forceinline__ float error2(float m) { return fminf(__fmaf_rn(0x1p-46f, m, 0x1p-143f), m); }

__device__ __forceinline__ float diff1(double f, double g) { return (float)(f - g); }
__device__ __forceinline__ float diff1(float f, float g) { return __fsub_rn(f, g); }

// Stores v, which is off by at most e, rounded to FP32; true where e leaves open
// which of two values that is.
__device__ __forceinline__ bool put_rounded(float* out, F2 v, float e) {
  const float r = __fadd_rn(v.h, v.l), rest = __fsub_rn(v.l, __fsub_rn(r, v.h));
  *out = r;
  return __fadd_rn(r, __fadd_rn(rest, copysignf(e, rest))) != r;
}

__device__ __forceinline__ bool put_rounded(float* out, double v, float) {
  *out = (float)v;
  return false;
}

// max(|B|^2 / rho, |u|^2), then its root: a Newton step on the FP32 one.  Small
// fields (top: the largest component) are scaled, so that their squares stay in
// range.
__device__ __forceinline__ float speed2(F2 rho, F2 (&U)[3], F2 (&B)[3], float top) {
  const float sc = top < 0x1p-50f ? 0x1p80f : 1.f;
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    U[a] = scaled(sc, U[a]);
    B[a] = scaled(sc, B[a]);
  }
  const F2 b2 = add2(add2u(mul2(B[0], B[0]), mul2(B[1], B[1])), mul2(B[2], B[2]));
  const F2 u2 = add2(add2u(mul2(U[0], U[0]), mul2(U[1], U[1])), mul2(U[2], U[2]));
  const F2 va = div2(b2, rho, 1.f / rho.h);
  const F2 s2 = va.h > u2.h || (va.h == u2.h && va.l > u2.l) ? va : u2;
  const float r = sqrtf(s2.h);
  return (r > 0.f ? r + __fadd_rn(__fmaf_rn(-r, r, s2.h), s2.l) / (2.f * r) : r) / sc;
}

template <class F>
__device__ __noinline__ float init_site_fp64(float* pop, Grid g, StepConsts k, InitConsts ic, int noneq, const F* rho_f, const F* u,
                                const F* Bf, const F* gu, const F* gB, int x, int y, int z);

// One site's populations, in TwoTerm arithmetic where that does, else in FP64;
// returns its speed max(|B| / sqrt(rho), |u|).
template <class Ar, class F>
__device__ __forceinline__ float init_columns(float* __restrict__ pop, const Grid& g, const StepConsts& k,
                                              const InitConsts& ic, int noneq, const F* __restrict__ rho_f,
                                              const F* __restrict__ u, const F* __restrict__ Bf,
                                              const F* __restrict__ gu, const F* __restrict__ gB, int x, int y, int z) {
  using V = typename Ar::V;
  constexpr bool kTwo = std::is_same_v<Ar, TwoTerm>;
  const long long n3 = g.n3;
  const int site = (z * g.ny + y) * g.nx + x;
  const Nbr nb = make_nbr(x, y, z, g);
  const int fwd[3] = {nb.xp, nb.yp, nb.zp}, back[3] = {nb.xm, nb.ym, nb.zm};
  // d_a F_b
  auto grad = [&](const F* f, const F* gf, int a, int b) -> V {
    if (gf) return Ar::field(gf[(3 * a + b) * n3 + site]);
    return Ar::twice(0.5f, Ar::diff(f[b * n3 + site + fwd[a]], f[b * n3 + site + back[a]]));
  };
  const F rho_v = rho_f ? rho_f[site] : (F)1;
  const V rho = Ar::field(rho_v), drho = Ar::diff(rho_v, (F)k.rho0);
  V U[3], B[3], b[3], dB[9], S[6];
  float mS[6], top = 0.f;  // mS: the magnitudes of the terms of S
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    const F Bv = Bf[a * n3 + site];
    U[a] = Ar::field(u[a * n3 + site]);
    B[a] = Ar::field(Bv);
    b[a] = Ar::diff(Bv, (F)k.Bref[a]);
    top = fmaxf(top, fmaxf(fabsf(Ar::head(U[a])), fabsf(Ar::head(B[a]))));
    if (isnan(Ar::head(U[a])) || isnan(Ar::head(B[a]))) top = __uint_as_float(0x7f800000u);
  }
  const float top_ub = top;
#pragma unroll
  for (int i = 0; i < 9; ++i) {
    dB[i] = grad(Bf, gB, i / 3, i % 3);
    top = isnan(Ar::head(dB[i])) ? __uint_as_float(0x7f800000u) : fmaxf(top, fabsf(Ar::head(dB[i])));
  }
  constexpr int ia[6] = {0, 1, 2, 0, 0, 1}, ib[6] = {0, 1, 2, 1, 2, 2};  // xx yy zz xy xz yz
#pragma unroll
  for (int i = 0; i < 6; ++i) {  // d_a u_b + d_b u_a
    const V s = grad(u, gu, ia[i], ib[i]), t = i < 3 ? s : grad(u, gu, ib[i], ia[i]);
    S[i] = i < 3 ? Ar::twice(2.f, s) : Ar::add(s, t);
    mS[i] = fabsf(Ar::head(s)) + fabsf(Ar::head(t));
    top = isnan(mS[i]) ? __uint_as_float(0x7f800000u) : fmaxf(top, mS[i]);
  }
  if (kTwo && !(top < 0x1p40f && Ar::head(rho) < 0x1p10f && Ar::head(rho) > 0x1p-10f))
    return init_site_fp64<F>(pop, g, k, ic, noneq, rho_f, u, Bf, gu, gB, x, y, z);
  float* out = pop + site;
  bool open = false;
  auto put = [&](int slot, V v, float e) { open |= put_rounded(out + (long long)slot * n3, v, e); };

  // magnetic: b_b + sign (4 (W_a B_b - B_a W_b) - d_a B_b / omega_B), W = U - d_i curl B
  {
    V W[3];
    float mW[3];
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      const int p = (a + 1) % 3, q = (a + 2) % 3;
      W[a] = Ar::add(U[a], Ar::mul(-k.alphaH, Ar::add(dB[3 * p + q], -dB[3 * q + p])));
      mW[a] = fmaf(k.alphaH, fabsf(Ar::head(dB[3 * p + q])) + fabsf(Ar::head(dB[3 * q + p])), fabsf(Ar::head(U[a])));
    }
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      const float mb = fabsf(Ar::head(b[c]));
      out[(long long)(kQ + c) * n3] = diff1(Bf[c * n3 + site], (F)k.Bref[c]);
#pragma unroll
      for (int a = 0; a < 3; ++a) {
        const V ne = -Ar::relaxed(ic, noneq, dB[3 * a + c]);
        const V t = a == c ? ne : Ar::addu(Ar::twice(4.f, Ar::add(Ar::mul(W[a], B[c]), -Ar::mul(B[a], W[c]))), ne);
        const float m = fmaf(ic.iwB.h, fabsf(Ar::head(dB[3 * a + c])), mb);
        const float e = error2(a == c ? m : fmaf(4.f, fmaf(mW[a], fabsf(Ar::head(B[c])), fabsf(Ar::head(B[a])) * mW[c]), m));
        put(kQ + 3 * (2 * a + 1) + c, Ar::addu(b[c], t), e);
        put(kQ + 3 * (2 * a + 2) + c, Ar::addu(b[c], -t), e);
      }
    }
  }

  // fluid; mL: the magnitudes of all terms but those of the equilibrium's velocity part
  V K[6], miso{};
  float mK[6], mI = 0.f;
  const V rp = Ar::stress(ic, noneq, rho);
#pragma unroll
  for (int i = 0; i < 6; ++i) {
    const int a = ia[i], c = ib[i];
    const V N = Ar::addu(Ar::mul(b[c], B[a]), Ar::mul(k.Bref[c], b[a]));
    K[i] = kTwo || noneq ? Ar::add(N, -Ar::mul(rp, S[i])) : N;
    mK[i] = fmaf(fabsf(Ar::head(rp)), mS[i], fmaf(fabsf(Ar::head(b[c])), fabsf(Ar::head(B[a])), fabsf(k.Bref[c]) * fabsf(Ar::head(b[a]))));
  }
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    miso = Ar::addu(miso, Ar::twice(0.5f, Ar::mul(b[a], Ar::add(B[a], k.Bref[a]))));
    mI = fmaf(fabsf(Ar::head(b[a])), fabsf(Ar::head(B[a])) + fabsf(k.Bref[a]), mI);
  }
  const V base0 = Ar::add(drho, Ar::add(Ar::mul(1.5f, Ar::add(Ar::addu(K[0], K[1]), K[2])), Ar::mul(-4.5f, miso)));
  const V LA = Ar::mul(4.5f, Ar::add(miso, -K[0])), LB = Ar::mul(4.5f, Ar::add(miso, -K[1])), LZ = Ar::mul(4.5f, Ar::add(miso, -K[2]));
  const V LC = Ar::mul(9.f, K[3]), NX = Ar::mul(-9.f, K[4]), NY = Ar::mul(-9.f, K[5]);
  const float mL = fmaf(9.f, mI + ((mK[3] + mK[4]) + mK[5]), fmaf(6.f, (mK[0] + mK[1]) + mK[2], fabsf(Ar::head(drho))));
  V ex[3], ey[3];
  float mx[2], my[2];  // of ex, ey at c = 0 and +-1
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    V* e = h ? ey : ex;
    const V uu = Ar::mul(U[h], U[h]), u3 = Ar::mul(3.f, U[h]), q = Ar::mul(3.f, uu);
    e[0] = Ar::add(q, -u3);
    e[1] = Ar::mul(-1.5f, uu);
    e[2] = Ar::add(q, u3);
    float* m = h ? my : mx;
    m[0] = 1.5f * Ar::head(uu);
    m[1] = Ar::head(q) + fabsf(Ar::head(u3));
  }
  const V uzz = Ar::mul(U[2], U[2]);
  const V e0z = Ar::mul(-1.5f, uzz), e1z = Ar::mul(3.f, U[2]), e2z = Ar::mul(4.5f, uzz);
  float eZ[2][2], e0[2][2];  // the errors at c_z = +-1 and 0 by |c_x|, |c_y|
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const float mr = Ar::head(rho) * fmaf(mx[i & 1], my[i >> 1], mx[i & 1] + my[i >> 1]), mg = mr + Ar::head(rho);
    const float m0 = fmaf(mg, 1.5f * Ar::head(uzz), mr + mL);
    e0[i >> 1][i & 1] = error2(m0);
    eZ[i >> 1][i & 1] = error2(fmaf(mg, Ar::head(e2z) + fabsf(Ar::head(e1z)), m0));
  }
#pragma unroll
  for (int py = 0; py < 3; ++py)
#pragma unroll
    for (int px = 0; px < 3; ++px) {
      const int cx = px - 1, cy = py - 1;
      const V rexy = Ar::mul(rho, Ar::add(Ar::mul(ex[px], ey[py]), Ar::add(ex[px], ey[py])));
      const V gg = Ar::add(rexy, rho);
      V L = base0;
      if (cx) L = Ar::addu(L, LA);
      if (cy) L = Ar::addu(L, LB);
      if (cx * cy) L = Ar::addu(L, cx * cy > 0 ? -LC : LC);
      const V Z0 = Ar::addu(Ar::addu(Ar::mul(gg, e0z), rexy), L);
      V Z1 = Ar::mul(gg, e1z);
      if (cx) Z1 = Ar::addu(Z1, cx > 0 ? NX : -NX);
      if (cy) Z1 = Ar::addu(Z1, cy > 0 ? NY : -NY);
      const V tz = Ar::addu(Z0, Ar::addu(Ar::mul(gg, e2z), LZ));
      const float ez = eZ[cy != 0][cx != 0];
      put(px + 3 * py, Ar::addu(tz, -Z1), ez);
      put(px + 3 * py + 9, Z0, e0[cy != 0][cx != 0]);
      put(px + 3 * py + 18, Ar::addu(tz, Z1), ez);
    }

  if constexpr (kTwo) {
    if (open) return init_site_fp64<F>(pop, g, k, ic, noneq, rho_f, u, Bf, gu, gB, x, y, z);
    return speed2(rho, U, B, top_ub);
  } else {
    const double va = sqrt((B[0] * B[0] + B[1] * B[1] + B[2] * B[2]) / rho);
    return (float)fmax(va, sqrt(U[0] * U[0] + U[1] * U[1] + U[2] * U[2]));
  }
}

template <class F>
__device__ __noinline__ float init_site_fp64(float* pop, Grid g, StepConsts k, InitConsts ic, int noneq, const F* rho_f,
                                             const F* u, const F* Bf, const F* gu, const F* gB, int x, int y, int z) {
  return init_columns<Fp64, F>(pop, g, k, ic, noneq, rho_f, u, Bf, gu, gB, x, y, z);
}

template <class T, class R, class F>
__global__ void __launch_bounds__(128, sizeof(T) == 4 ? 6 : 1)
    init_kernel(T* __restrict__ pop, Grid g, StepConsts k, InitConsts ic, int noneq, const F* __restrict__ rho_f,
                const F* __restrict__ u, const F* __restrict__ Bf, const F* __restrict__ gu,
                const F* __restrict__ gB, unsigned* __restrict__ speed_bits) {
  const int x = blockIdx.x * blockDim.x + threadIdx.x;
  const int y = blockIdx.y * blockDim.y + threadIdx.y;
  const int z = blockIdx.z + g.z0;
  const bool in = x < g.nx && y < g.ny;
  float sp = 0.f;
  if (in) {
    if constexpr (sizeof(T) == 4)
      sp = init_columns<TwoTerm, F>(pop, g, k, ic, noneq, rho_f, u, Bf, gu, gB, x, y, z);
    else
      sp = init_site<T, R, F>(pop, g, k, noneq, rho_f, u, Bf, gu, gB, x, y, z);
    if (!isfinite(sp)) sp = __uint_as_float(0x7f800000u);
  }
  // max speed: one atomic per warp (non-negative floats order like their bits)
  const unsigned m = __reduce_max_sync(0xffffffffu, in ? __float_as_uint(sp) : 0u);
  if ((threadIdx.x & 31) == 0 && m) atomicMax(speed_bits, m);
}

// ---------------------------------------------------------------------------
// Moments and decoded populations.  Per-site arithmetic in R: FP64 for FP32
// storage, FP32 for 16-bit storage (whose stored values carry 11 or 8
// significant bits).  Density and field are formed as deviations from the
// reference (rho0, B_ref) and added to it in FP64, so sums over sites keep
// the FP64 reference exact.

template <class T, bool ODD, class R>
__device__ __forceinline__ void load_site(const T* __restrict__ pop, int site, const Nbr& nb, long long n3,
                                          R sf[kQ], R sg[3][kM]) {
#pragma unroll
  for (int i = 0; i < kQ; ++i) sf[i] = (R)Codec<T>::dec(pop[src27<ODD>(i, site, nb, n3)]);
#pragma unroll
  for (int b = 0; b < 3; ++b)
#pragma unroll
    for (int i = 0; i < kM; ++i) sg[b][i] = (R)Codec<T>::dec(pop[src7<ODD>(b, i, site, nb, n3)]);
}

template <class R>
struct SiteMoments {
  R drho, U[3], dB[3], J[3], trlam;  // drho = rho - rho0, dB = B - B_ref
  __device__ __forceinline__ double rho(const StepConsts& k) const { return (double)k.rho0 + (double)drho; }
  __device__ __forceinline__ double B(const StepConsts& k, int a) const { return (double)k.Bref[a] + (double)dB[a]; }
};

template <class R>
__device__ __forceinline__ SiteMoments<R> site_moments(const R sf[kQ], const R sg[3][kM], const StepConsts& k) {
  SiteMoments<R> m;
  R drho = 0, j[3] = {0, 0, 0};
#pragma unroll
  for (int i = 0; i < kQ; ++i) {
    const R t = (R)w27d(i) * sf[i];
    drho += t;
    if (cx27(i)) j[0] += (R)cx27(i) * t;
    if (cy27(i)) j[1] += (R)cy27(i) * t;
    if (cz27(i)) j[2] += (R)cz27(i) * t;
  }
  m.drho = drho;
  const R rho = (R)k.rho0 + drho;
#pragma unroll
  for (int a = 0; a < 3; ++a) m.U[a] = j[a] / rho;
  R lam[3][3];
#pragma unroll
  for (int b = 0; b < 3; ++b) {
    m.dB[b] = (R)0.25 * sg[b][0] + (R)0.125 * (sg[b][1] + sg[b][2] + sg[b][3] + sg[b][4] + sg[b][5] + sg[b][6]);
    lam[0][b] = (R)0.125 * (sg[b][1] - sg[b][2]);
    lam[1][b] = (R)0.125 * (sg[b][3] - sg[b][4]);
    lam[2][b] = (R)0.125 * (sg[b][5] - sg[b][6]);
  }
  m.trlam = lam[0][0] + lam[1][1] + lam[2][2];
  const R gq = (R)4 * (R)k.omegaB;
  const R* U = m.U;
  const R B[3] = {(R)k.Bref[0] + m.dB[0], (R)k.Bref[1] + m.dB[1], (R)k.Bref[2] + m.dB[2]};
  const R A[3] = {lam[1][2] - lam[2][1], lam[2][0] - lam[0][2], lam[0][1] - lam[1][0]};
  const R uxb[3] = {U[1] * B[2] - U[2] * B[1], U[2] * B[0] - U[0] * B[2], U[0] * B[1] - U[1] * B[0]};
  const R yv[3] = {-gq * (A[0] - (R)2 * uxb[0]), -gq * (A[1] - (R)2 * uxb[1]), -gq * (A[2] - (R)2 * uxb[2])};
  const R s = (R)2 * (R)k.alphaH * gq;
  const R yxb[3] = {yv[1] * B[2] - yv[2] * B[1], yv[2] * B[0] - yv[0] * B[2], yv[0] * B[1] - yv[1] * B[0]};
  const R yb = yv[0] * B[0] + yv[1] * B[1] + yv[2] * B[2];
  const R b2 = B[0] * B[0] + B[1] * B[1] + B[2] * B[2];
#pragma unroll
  for (int a = 0; a < 3; ++a) m.J[a] = (yv[a] - s * yxb[a] + s * s * yb * B[a]) / ((R)1 + s * s * b2);
  return m;
}

// per-site arithmetic type of a storage type
template <class T>
struct SiteReal {
  using type = float;
};
template <>
struct SiteReal<float> {
  using type = double;
};

// What a moments launch writes: the density and velocity need the fluid
// populations, the current needs everything (CUR implies FLUID); B comes from
// the magnetic ones alone.  The shell spectra ask for u and B, the band loss
// for B only, and the unused part is neither loaded nor computed.
// O: the element type of the outputs (FP64 for flame_moments, FP32 for
// flame_moments_f32).
template <class O>
struct MomentsOut {
  O *rho, *u, *B, *J;
  long long os;  // stride between the components of u, B and J
  template <class M>
  __device__ __forceinline__ void store(const M& m, const StepConsts& k, long long o) const {
    if (rho) rho[o] = (O)m.rho(k);
    for (int a = 0; a < 3; ++a) {
      if (u) u[a * os + o] = (O)m.U[a];
      if (B) B[a * os + o] = (O)m.B(k, a);
      if (J) J[a * os + o] = (O)m.J[a];
    }
  }
};

// 16-bit storage: FP32 per site.
template <class T, bool ODD, class O, bool FLUID, bool CUR>
__global__ void moments_kernel(const T* __restrict__ pop, Grid g, StepConsts k, MomentsOut<O> out) {
  const int x = blockIdx.x * blockDim.x + threadIdx.x;
  const int y = blockIdx.y * blockDim.y + threadIdx.y;
  const int z = blockIdx.z + g.z0;
  if (x >= g.nx || y >= g.ny) return;
  const int site = (z * g.ny + y) * g.nx + x;
  const Nbr nb = make_nbr(x, y, z, g);
  float sf[kQ], sg[3][kM];
  load_site<T, ODD>(pop, site, nb, g.n3, sf, sg);
  const SiteMoments<float> m = site_moments(sf, sg, k);
  MomentsOut<O> o = out;
  if (!FLUID) o.rho = o.u = nullptr;
  if (!CUR) o.J = nullptr;
  o.store(m, k, site - (long long)g.z0 * g.nx * g.ny);  // index among the updated sites
}

// FP32 storage: FP64 moments.  Bound by the FP64 pipe, which has 1/64 of the
// FP32 rate: the 48 conversions and ~220 operations per site of summing,
// dividing and solving in FP64 took 1012 us at 128^3 (8.0 ms at 256^3).  The
// sums over the populations are linear, so they are taken as three-term FP32
// expansions (72 bits, more than FP64 holds) in the order of the step
// kernel's 1-D passes and turned into FP64 by their bits; the quotients by
// rho and the current's solve stay in FP64: about 20 operations per site
// without the current, 55 with it.  128^3: 298 us for all moments (393 with
// divisions and the constants widened by every thread), 132 us for u and B
// (84 us of HBM traffic).  64 registers, eight blocks per SM: B alone, bound by
// HBM, 46 us against 58 with six blocks; the others do not change.
// The step's FP32 constants widened once on the host (a conversion per thread
// costs as much as an FP64 operation): gq = 4 omega_B, s = 2 d_i gq.
struct Consts64 {
  double rho0, rho0x216, Bref[3], gq2, gq8, s, ss;
  explicit Consts64(const StepConsts& k) {
    rho0 = (double)k.rho0;
    rho0x216 = 216.0 * rho0;
    for (int a = 0; a < 3; ++a) Bref[a] = (double)k.Bref[a];
    const double gq = 4.0 * (double)k.omegaB;
    gq2 = 2.0 * gq;
    gq8 = -0.125 * gq;
    s = 2.0 * (double)k.alphaH * gq;
    ss = s * s;
  }
};

struct SiteMoments64 {
  double rho_, U[3], B_[3], J[3];
  __device__ __forceinline__ double rho(const StepConsts&) const { return rho_; }
  __device__ __forceinline__ double B(const StepConsts&, int a) const { return B_[a]; }
};

// 216 sum_i w_i s_i and 216 sum_i w_i c_ia s_i from the populations in
// velocity-cube order.
__device__ __forceinline__ void fluid_sums(const float (&s)[kQ], F3& r216, F3 (&j216)[3]) {
  F3 M00[3], M10[3], M01[3];
#pragma unroll
  for (int pz = 0; pz < 3; ++pz) {
    F3 m0[3];
    F2 m1[3];
#pragma unroll
    for (int py = 0; py < 3; ++py) {
      const int q = 3 * (py + 3 * pz);
      m0[py] = add3(two_sum(s[q + 2], s[q]), 4.f * s[q + 1]);
      m1[py] = two_diff(s[q + 2], s[q]);
    }
    M00[pz] = add3(add3(m0[2], m0[0]), scaled(4.f, m0[1]));
    M01[pz] = add3(m0[2], -m0[0]);
    M10[pz] = add3(add3(m1[2], m1[0]), scaled(4.f, m1[1]));
  }
  r216 = add3(add3(M00[2], M00[0]), scaled(4.f, M00[1]));
  j216[0] = add3(add3(M10[2], M10[0]), scaled(4.f, M10[1]));
  j216[1] = add3(add3(M01[2], M01[0]), scaled(4.f, M01[1]));
  j216[2] = add3(M00[2], -M00[0]);
}

// 8 dB and 8 Lambda_ab of the magnetic populations.
__device__ __forceinline__ void magnetic_sums(const float (&sg)[3][kM], F3 (&sB)[3], F2 (&d)[3][3]) {
#pragma unroll
  for (int b = 0; b < 3; ++b) {
    F2 f[3];
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      f[a] = two_sum(sg[b][2 * a + 1], sg[b][2 * a + 2]);
      d[a][b] = two_diff(sg[b][2 * a + 1], sg[b][2 * a + 2]);
    }
    sB[b] = add3(add3(add3(f[0], f[1]), f[2]), 2.f * sg[b][0]);
  }
}

// The pre-collision populations of FP32 storage, the fluid ones in
// velocity-cube order.
template <bool ODD>
__device__ __forceinline__ void load_cube(const float* __restrict__ pop, int site, const Nbr& nb, long long n3,
                                          float (&s)[kQ]) {
#pragma unroll
  for (int q = 0; q < kQ; ++q) s[q] = pop[src27<ODD>(idx27(q % 3, (q / 3) % 3, q / 9), site, nb, n3)];
}
template <bool ODD>
__device__ __forceinline__ void load_magnetic(const float* __restrict__ pop, int site, const Nbr& nb, long long n3,
                                              float (&sg)[3][kM]) {
#pragma unroll
  for (int b = 0; b < 3; ++b)
#pragma unroll
    for (int i = 0; i < kM; ++i) sg[b][i] = pop[src7<ODD>(b, i, site, nb, n3)];
}

// A site whose sums overflow FP32 or are not finite.
template <bool ODD>
__device__ __noinline__ void general_moments(const float* pop, int site, Nbr nb, long long n3, StepConsts k,
                                             SiteMoments64* m) {
  double sf[kQ], sg[3][kM];
  load_site<float, ODD, double>(pop, site, nb, n3, sf, sg);
  const SiteMoments<double> d = site_moments(sf, sg, k);
  m->rho_ = d.rho(k);
  for (int a = 0; a < 3; ++a) {
    m->U[a] = d.U[a];
    m->B_[a] = d.B(k, a);
    m->J[a] = d.J[a];
  }
}

// U of 216 rho u and 216 rho.
__device__ __forceinline__ void velocity64(double rho216, const F3 (&j216)[3], double (&U)[3]) {
  const double ir = reciprocal(rho216);
#pragma unroll
  for (int a = 0; a < 3; ++a) U[a] = quotient(to_double(j216[a]), rho216, ir);
}

template <bool ODD, class O, bool FLUID, bool CUR>
__global__ void __launch_bounds__(128, 8)
    moments64_kernel(const float* __restrict__ pop, Grid g, StepConsts k, Consts64 d, MomentsOut<O> out) {
  static_assert(FLUID || !CUR, "the current needs the velocity");
  const int x = blockIdx.x * blockDim.x + threadIdx.x;
  const int y = blockIdx.y * blockDim.y + threadIdx.y;
  const int z = blockIdx.z + g.z0;
  if (x >= g.nx || y >= g.ny) return;
  const int site = (z * g.ny + y) * g.nx + x;
  const Nbr nb = make_nbr(x, y, z, g);
  const long long n3 = g.n3;
  float s[kQ], sg[3][kM];
  if constexpr (FLUID) load_cube<ODD>(pop, site, nb, n3, s);
  load_magnetic<ODD>(pop, site, nb, n3, sg);

  SiteMoments64 m;
  float chk = 0.f;  // the last terms carry a NaN from any overflow or non-finite value
  F3 r216, j216[3], sB[3], A8[3];
  if constexpr (FLUID) {
    fluid_sums(s, r216, j216);
    chk = (r216.l + j216[0].l) + (j216[1].l + j216[2].l);
  }
  F2 lam8[3][3];
  magnetic_sums(sg, sB, lam8);
  chk += (sB[0].l + sB[1].l) + sB[2].l;
  if constexpr (CUR) {
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      A8[a] = add3(lam8[(a + 1) % 3][(a + 2) % 3], -lam8[(a + 2) % 3][(a + 1) % 3]);
      chk += A8[a].l;
    }
  }
  if (isfinite(chk)) {
#pragma unroll
    for (int b = 0; b < 3; ++b) m.B_[b] = d.Bref[b] + to_double(scaled(0.125f, sB[b]));
    if constexpr (FLUID) {
      const double r = to_double(r216);
      m.rho_ = fma(r, 1.0 / 216.0, d.rho0);
      velocity64(d.rho0x216 + r, j216, m.U);
    }
    if constexpr (CUR) {
      const double* B = m.B_;
      double y[3];
#pragma unroll
      for (int a = 0; a < 3; ++a) {
        const int b = (a + 1) % 3, c = (a + 2) % 3;
        y[a] = fma(d.gq2, m.U[b] * B[c] - m.U[c] * B[b], d.gq8 * to_double(A8[a]));
      }
      const double b2 = B[0] * B[0] + B[1] * B[1] + B[2] * B[2];
      const double t = d.ss * (y[0] * B[0] + y[1] * B[1] + y[2] * B[2]);
      const double iden = reciprocal(fma(d.ss, b2, 1.0));
#pragma unroll
      for (int a = 0; a < 3; ++a) {
        const int b = (a + 1) % 3, c = (a + 2) % 3;
        m.J[a] = fma(t, B[a], fma(-d.s, y[b] * B[c] - y[c] * B[b], y[a])) * iden;
      }
    }
  } else {
    general_moments<ODD>(pop, site, nb, n3, k, &m);
  }
  MomentsOut<O> o = out;
  if (!FLUID) o.rho = o.u = nullptr;
  if (!CUR) o.J = nullptr;
  o.store(m, k, site - (long long)g.z0 * g.nx * g.ny);  // index among the updated sites
}

template <class T, bool ODD>
__global__ void populations_kernel(const T* __restrict__ pop, Grid g, StepConsts k, double* __restrict__ f) {
  const int x = blockIdx.x * blockDim.x + threadIdx.x;
  const int y = blockIdx.y * blockDim.y + threadIdx.y;
  const int z = blockIdx.z + g.z0;
  if (x >= g.nx || y >= g.ny) return;
  const int site = (z * g.ny + y) * g.nx + x;
  const Nbr nb = make_nbr(x, y, z, g);
  double sf[kQ], sg[3][kM];
  load_site<T, ODD, double>(pop, site, nb, g.n3, sf, sg);
  const double Br[3] = {(double)k.Bref[0], (double)k.Bref[1], (double)k.Bref[2]};
  const double br2 = Br[0] * Br[0] + Br[1] * Br[1] + Br[2] * Br[2];
  const long long o = site - (long long)g.z0 * g.nx * g.ny;  // index among the updated sites
#pragma unroll 1
  for (int i = 0; i < kQ; ++i) {
    const double c2 = cx27(i) * cx27(i) + cy27(i) * cy27(i) + cz27(i) * cz27(i);
    const double cb = cx27(i) * Br[0] + cy27(i) * Br[1] + cz27(i) * Br[2];
    const double ell = 4.5 * (0.5 * br2 * (c2 - 1.0 / 3.0) - cb * cb);  // rest Lorentz term / w
    f[(long long)i * g.n3i + o] = w27d(i) * ((double)k.rho0 + ell + sf[i]);
  }
  for (int b = 0; b < 3; ++b)
    for (int i = 0; i < kM; ++i) f[(long long)mslot(b, i) * g.n3i + o] = w7d(i) * (Br[b] + sg[b][i]);
}


// Moments at a list of sites (time series): out[j] = rho, u[3], B[3], J[3].
template <class T, bool ODD>
__global__ void probe_kernel(const T* __restrict__ pop, Grid g, StepConsts k, int n, const long long* __restrict__ sites,
                             double* __restrict__ out) {
  const int j = blockIdx.x * blockDim.x + threadIdx.x;
  if (j >= n) return;
  const long long sl = sites[j];
  if (sl < 0 || sl >= g.n3i) {
    for (int v = 0; v < 10; ++v) out[(long long)j * 10 + v] = nan("");
    return;
  }
  const int site = (int)(sl + (long long)g.z0 * g.nx * g.ny);
  const int x = site % g.nx, y = (site / g.nx) % g.ny, z = site / (g.nx * g.ny);
  const Nbr nb = make_nbr(x, y, z, g);
  using R = typename SiteReal<T>::type;
  R sf[kQ], sg[3][kM];
  load_site<T, ODD>(pop, site, nb, g.n3, sf, sg);
  const SiteMoments<R> m = site_moments(sf, sg, k);
  double* o = out + (long long)j * 10;
  o[0] = m.rho(k);
  for (int a = 0; a < 3; ++a) {
    o[1 + a] = (double)m.U[a];
    o[4 + a] = m.B(k, a);
    o[7 + a] = (double)m.J[a];
  }
}

template <class T>
cudaError_t probe_t(int odd, const void* pop, Grid g, const StepConsts& k, int n, const long long* sites, double* out,
                    cudaStream_t s) {
  const int tb = 64, nb = (n + tb - 1) / tb;
  if (odd)
    probe_kernel<T, true><<<nb, tb, 0, s>>>(static_cast<const T*>(pop), g, k, n, sites, out);
  else
    probe_kernel<T, false><<<nb, tb, 0, s>>>(static_cast<const T*>(pop), g, k, n, sites, out);
  return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// FP64 reduction of the scalar diagnostics: per block, then a fixed-order
// final sum (deterministic).  Partial layout (kRedVals):
//   0 sum rho, 1-3 sum rho u, 4-6 sum B, 7 sum |u|^2, 8 sum |B - Bref|^2,
//   9 sum u.(B - Bref), 10-12 sum u, 13 sum |J|^2, 14 max |u|,
//   15 sum ((omega_B/C^2) Tr Lambda)^2, 16 non-finite sites.
//
// Every site's terms in FP64 (16 additions and as many conversions; for FP32
// storage the moments too) bound this kernel by the FP64 pipe.  What is a sum
// or product of FP32 values runs in three-term FP32 expansions instead (72
// bits, more than FP64 holds, for 13 to 22 FP32 operations an addition): the
// sums of 16-bit storage, whose terms come from FP32 arithmetic, and for FP32
// storage the sums over the populations and, over the sites, of density,
// momentum and field.  What is left in FP64 there, the quotients, squares and
// the sums of those, keeps the FP64 pipe busy 79 % of the time.  A block that
// meets a value too large for this, or a non-finite one, sums its sites again
// in FP64 (reduce_general).
//
// A thread's sums become FP64 numbers in shared memory, and a warp sums each
// quantity of the block from there: 13 FP64 additions for a quantity, against 40
// by shuffles in each of the block's warps.
//
// flame_reduce_static, us at 64^3, 128^3, 256^3: FP32 storage 73, 336, 2380 (all in
// FP64 1353 at 128^3, 9767 at 256^3; the moments in two-term FP32 arithmetic took
// 140 and 855, but held 48 bits), FP16 36, 83, 532 (317 and 1435 with FP64 sums; 41,
// 82, 506 with two-term ones).  Blocks per SM, two / three: FP32 341 / 336 at 128^3
// and 2466 / 2380, FP16, whose three spill, 83 / 91 and 532 / 514.

// The FP64 sums of a thread's sites.
template <class T, bool ODD>
__device__ __noinline__ void reduce_general(const T* pop, Grid g, StepConsts k, double* acc) {
  for (int v = 0; v < kRedVals; ++v) acc[v] = 0.0;
  const long long n3 = g.n3;
  const long long off = (long long)g.z0 * g.nx * g.ny;
  for (long long s = (long long)blockIdx.x * blockDim.x + threadIdx.x; s < g.n3i; s += (long long)gridDim.x * blockDim.x) {
    const int site = (int)(s + off);
    const int x = site % g.nx, y = (site / g.nx) % g.ny, z = site / (g.nx * g.ny);
    const Nbr nb = make_nbr(x, y, z, g);
    using R = typename SiteReal<T>::type;
    R sf[kQ], sg[3][kM];
    load_site<T, ODD>(pop, site, nb, n3, sf, sg);
    const SiteMoments<R> m = site_moments(sf, sg, k);
    const R* b = m.dB;
    const R uu = m.U[0] * m.U[0] + m.U[1] * m.U[1] + m.U[2] * m.U[2];
    const R dv = (R)4 * (R)k.omegaB * m.trlam;
    const bool ok = isfinite(m.drho + uu + b[0] + b[1] + b[2] + m.J[0] + m.J[1] + m.J[2]);
    if (!ok) {
      acc[16] += 1.0;
      continue;
    }
    const double rho = m.rho(k);
    acc[0] += rho;
    for (int a = 0; a < 3; ++a) {
      acc[1 + a] += rho * (double)m.U[a];
      acc[4 + a] += m.B(k, a);
      acc[10 + a] += (double)m.U[a];
    }
    acc[7] += (double)uu;
    acc[8] += (double)(b[0] * b[0] + b[1] * b[1] + b[2] * b[2]);
    acc[9] += (double)(m.U[0] * b[0] + m.U[1] * b[1] + m.U[2] * b[2]);
    acc[13] += (double)(m.J[0] * m.J[0] + m.J[1] * m.J[1] + m.J[2] * m.J[2]);
    acc[14] = fmax(acc[14], sqrt((double)uu));
    acc[15] += (double)(dv * dv);
  }
}

constexpr float kRedLimit = 0x1p100f;  // largest term the expansions take

// A thread's sums of the quantities above over its sites, but for 14, the
// maximum of |u|^2, and 16, the number of sites.  add: one site's terms; the
// largest magnitude among them, or NaN for a non-finite site.  finish: the
// block's quantity v from the block's sums r of value().
template <class T>
struct Terms {
  // of rho - rho0, 2^60 (rho - rho0) u (whose second term FP32 holds for all u),
  // B - Bref, ...: FP32 per site
  F3 lin[7], u[3], uu, bb, ub, jj, vv;
  float top;
  int n;
  template <bool ODD>
  __device__ __forceinline__ float add(const T* __restrict__ pop, int site, const Nbr& nb, const Grid& g,
                                       const StepConsts& k, const Consts64&) {
    float sf[kQ], sg[3][kM];
    load_site<T, ODD>(pop, site, nb, g.n3, sf, sg);
    const SiteMoments<float> m = site_moments(sf, sg, k);
    const float* b = m.dB;
    const float u2 = m.U[0] * m.U[0] + m.U[1] * m.U[1] + m.U[2] * m.U[2];
    const float b2 = b[0] * b[0] + b[1] * b[1] + b[2] * b[2];
    const float j2 = m.J[0] * m.J[0] + m.J[1] * m.J[1] + m.J[2] * m.J[2];
    const float dv = 4.f * k.omegaB * m.trlam, r60 = 0x1p60f * m.drho;
    lin[0] = add3(lin[0], m.drho);
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      lin[1 + a] = add3(lin[1 + a], mul2(r60, m.U[a]));
      lin[4 + a] = add3(lin[4 + a], b[a]);
      u[a] = add3(u[a], m.U[a]);
    }
    uu = add3(uu, u2);
    bb = add3(bb, b2);
    ub = add3(ub, m.U[0] * b[0] + m.U[1] * b[1] + m.U[2] * b[2]);
    jj = add3(jj, j2);
    vv = add3(vv, dv * dv);
    top = fmaxf(top, u2);
    ++n;
    return fabsf(r60) * (1.f + u2) + u2 + b2 + j2 + dv * dv + fabsf(b[0]) + fabsf(b[1]) + fabsf(b[2]);
  }
  __device__ __forceinline__ double value(int v) const {
    return v < 7 ? to_double(lin[v]) : v == 7 ? to_double(uu) : v == 8 ? to_double(bb) : v == 9 ? to_double(ub)
         : v < 13 ? to_double(u[v - 10]) : v == 13 ? to_double(jj) : v == 14 ? (double)top
         : v == 15 ? to_double(vv) : (double)n;
  }
  static __device__ __forceinline__ double finish(const double* r, int v, const StepConsts& k, const Consts64&) {
    if (v == 0) return fma(r[16], (double)k.rho0, r[0]);
    if (v < 4) return fma((double)k.rho0, r[9 + v], 0x1p-60 * r[v]);
    if (v < 7) return fma(r[16], (double)k.Bref[v - 4], r[v]);
    return v == 14 ? sqrt(r[14]) : v == 16 ? 0.0 : r[v];
  }
};

// FP32 storage: the sums of 216 (rho - rho0), 216 rho u and 8 (B - Bref), which
// are sums of populations, as expansions; the others in FP64, constant factors
// left to finish.  The current's system J + s J x B = y keeps y's part along B and
// divides the square of the other by 1 + s^2 |B|^2, so that |J|^2 (1 + s^2 |B|^2)
// = |y|^2 + s^2 (y.B)^2: no need of J itself.  y = 2 gq (U x B - A / 2).
template <>
struct Terms<float> {
  F3 lin[7];
  double u[3], uu, bb, ub, jj, vv;  // jj: |y / (2 gq)|^2 ..., vv: (8 Tr Lambda)^2
  long long top;                    // the bits of max |u|^2, which order as the values do
  int n;
  template <bool ODD>
  __device__ __forceinline__ float add(const float* __restrict__ pop, int site, const Nbr& nb, const Grid& g,
                                       const StepConsts& k, const Consts64& d) {
    float s[kQ], sg[3][kM];
    load_cube<ODD>(pop, site, nb, g.n3, s);
    load_magnetic<ODD>(pop, site, nb, g.n3, sg);
    F3 r216, j216[3], sB[3], A8[3];
    F2 lam8[3][3];
    fluid_sums(s, r216, j216);
    double U[3], b[3], B[3], y[3];
    velocity64(to_double(add3(r216, mul2(216.f, k.rho0))), j216, U);
    magnetic_sums(sg, sB, lam8);
    const F3 tr8 = add3(add3(lam8[0][0], lam8[1][1]), lam8[2][2]);
    float big = fabsf(r216.h) + fabsf(r216.l) + fabsf(tr8.h) + fabsf(tr8.l);
    lin[0] = add3(lin[0], r216);
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      A8[a] = add3(lam8[(a + 1) % 3][(a + 2) % 3], -lam8[(a + 2) % 3][(a + 1) % 3]);
      big += fabsf(j216[a].h) + fabsf(j216[a].l) + fabsf(sB[a].h) + fabsf(sB[a].l) + fabsf(A8[a].h) + fabsf(A8[a].l);
      lin[1 + a] = add3(lin[1 + a], j216[a]);
      lin[4 + a] = add3(lin[4 + a], sB[a]);
      const F3 db = scaled(0.125f, sB[a]);
      b[a] = to_double(db);
      B[a] = to_double(add3(db, k.Bref[a]));
    }
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      const int p = (a + 1) % 3, q = (a + 2) % 3;
      y[a] = fma(U[p], B[q], fma(-U[q], B[p], to_double(scaled(-0.0625f, A8[a]))));
      u[a] += U[a];
      bb = fma(b[a], b[a], bb);
      ub = fma(U[a], b[a], ub);
    }
    const double u2 = dot64(U, U), yB = dot64(y, B), dv = to_double(tr8);
    const double j2 = fma(d.ss * yB, yB, dot64(y, y));
    uu += u2;
    jj = fma(j2, reciprocal(fma(d.ss, dot64(B, B), 1.0)), jj);
    vv = fma(dv, dv, vv);
    const long long bits = __double_as_longlong(u2);
    top = bits > top ? bits : top;
    ++n;
    // not finite: a density of zero
    return finite64(u2) && finite64(j2) ? big : __uint_as_float(0x7fc00000u);
  }
  static __device__ __forceinline__ double dot64(const double (&a)[3], const double (&b)[3]) {
    return fma(a[2], b[2], fma(a[1], b[1], a[0] * b[0]));
  }
  static __device__ __forceinline__ bool finite64(double x) { return (__double2hiint(x) & 0x7ff00000) != 0x7ff00000; }
  __device__ __forceinline__ double value(int v) const {
    return v < 7 ? to_double(lin[v]) : v == 7 ? uu : v == 8 ? bb : v == 9 ? ub : v < 13 ? u[v - 10] : v == 13 ? jj
         : v == 14 ? __longlong_as_double(top) : v == 15 ? vv : (double)n;
  }
  static __device__ __forceinline__ double finish(const double* r, int v, const StepConsts& k, const Consts64& d) {
    if (v == 0) return fma(r[16], (double)k.rho0, r[0] / 216.0);
    if (v < 4) return r[v] / 216.0;
    if (v < 7) return fma(r[16], (double)k.Bref[v - 4], 0.125 * r[v]);
    if (v == 13) return d.gq2 * d.gq2 * r[13];
    if (v == 15) return d.gq8 * d.gq8 * r[15];
    return v == 14 ? sqrt(r[14]) : v == 16 ? 0.0 : r[v];
  }
};

constexpr int kRedThreads = 256;
template <class T, bool ODD>
__global__ void __launch_bounds__(kRedThreads, sizeof(T) == 4 ? 3 : 2)
    reduce_kernel(const T* __restrict__ pop, Grid g, StepConsts k, Consts64 d, double* __restrict__ partials) {
  __shared__ double sh[kRedVals][kRedThreads], total[kRedVals];
  Terms<T> terms{};
  bool fits = true;
  const int off = g.z0 * g.nx * g.ny;
  for (long long s = (long long)blockIdx.x * kRedThreads + threadIdx.x; s < g.n3i; s += (long long)gridDim.x * kRedThreads) {
    const int site = (int)s + off;
    const int row = site / g.nx, x = site - row * g.nx, z = row / g.ny, y = row - z * g.ny;
    fits = fits && terms.template add<ODD>(pop, site, make_nbr(x, y, z, g), g, k, d) < kRedLimit;
  }
  const bool general = __syncthreads_or(!fits);
  if (general) {
    double a[kRedVals];
    reduce_general<T, ODD>(pop, g, k, a);
    for (int v = 0; v < kRedVals; ++v) sh[v][threadIdx.x] = a[v];
  } else {
#pragma unroll
    for (int v = 0; v < kRedVals; ++v) sh[v][threadIdx.x] = terms.value(v);
  }
  __syncthreads();
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  for (int v = warp; v < kRedVals; v += kRedThreads / 32) {
    double a = sh[v][lane];
    for (int i = lane + 32; i < kRedThreads; i += 32) a = v == 14 ? fmax(a, sh[v][i]) : a + sh[v][i];
    for (int o = 16; o > 0; o >>= 1) {
      const double t = __shfl_down_sync(0xffffffffu, a, o);
      a = v == 14 ? fmax(a, t) : a + t;
    }
    if (lane == 0) total[v] = a;
  }
  __syncthreads();
  if (threadIdx.x < kRedVals)
    partials[(long long)blockIdx.x * kRedVals + threadIdx.x] =
        general ? total[threadIdx.x] : Terms<T>::finish(total, threadIdx.x, k, d);
}

__global__ void reduce_final_kernel(const double* __restrict__ partials, int nblocks, double* __restrict__ out) {
  const double a = reduce_partials_warp(partials, nblocks, threadIdx.x >> 5);
  if ((threadIdx.x & 31) == 0) out[threadIdx.x >> 5] = a;
}

// Block of `threads` threads: x-rows of up to `threads` sites, several
// rows per block when nx is small.

template <class T, class O, bool FLUID, bool CUR>
void moments_go(int odd, const void* pop, Grid g, const StepConsts& k, const MomentsOut<O>& out, cudaStream_t s) {
  const dim3 b = site_block(g), gr = site_grid(g, b);
  const T* p = static_cast<const T*>(pop);
  if constexpr (sizeof(T) == 4) {
    const Consts64 d(k);
    if (odd) moments64_kernel<true, O, FLUID, CUR><<<gr, b, 0, s>>>(p, g, k, d, out);
    else moments64_kernel<false, O, FLUID, CUR><<<gr, b, 0, s>>>(p, g, k, d, out);
  } else {
    if (odd) moments_kernel<T, true, O, FLUID, CUR><<<gr, b, 0, s>>>(p, g, k, out);
    else moments_kernel<T, false, O, FLUID, CUR><<<gr, b, 0, s>>>(p, g, k, out);
  }
}

template <class T, class O>
cudaError_t moments_t(int odd, const void* pop, Grid g, const StepConsts& k, O* rho, O* u, O* B, O* J,
                      long long os, cudaStream_t s) {
  const MomentsOut<O> out{rho, u, B, J, os};
  if (J) moments_go<T, O, true, true>(odd, pop, g, k, out, s);
  else if (rho || u) moments_go<T, O, true, false>(odd, pop, g, k, out, s);
  else moments_go<T, O, false, false>(odd, pop, g, k, out, s);
  return cudaGetLastError();
}

F2 split(double v) {
  const float h = (float)v;
  return {h, (float)(v - (double)h)};
}

template <class F>
cudaError_t init_t(int storage, void* pop, Grid g, const StepConsts& k, int noneq, const F* rho, const F* u,
                   const F* B, const F* gu, const F* gB, unsigned* speed_bits, cudaStream_t s) {
  const dim3 b = site_block(g), gr = site_grid(g, b);
  const InitConsts ic{noneq ? split(-1.0 / (3.0 * (double)k.omega)) : F2{0.f, 0.f},
                      noneq ? split(1.0 / (double)k.omegaB) : F2{0.f, 0.f},
                      3.0 * (double)k.omega,
                      1.0 / (3.0 * (double)k.omega),
                      (double)k.omegaB,
                      1.0 / (double)k.omegaB};
  switch (storage) {
    case 1:
      init_kernel<float, double, F><<<gr, b, 0, s>>>(static_cast<float*>(pop), g, k, ic, noneq, rho, u, B, gu, gB,
                                                      speed_bits);
      break;
    case 2:
      init_kernel<__half, float, F><<<gr, b, 0, s>>>(static_cast<__half*>(pop), g, k, ic, noneq, rho, u, B, gu, gB,
                                                      speed_bits);
      break;
    case 3:
      init_kernel<__nv_bfloat16, float, F><<<gr, b, 0, s>>>(static_cast<__nv_bfloat16*>(pop), g, k, ic, noneq, rho,
                                                             u, B, gu, gB, speed_bits);
      break;
    default:
      return cudaErrorInvalidValue;
  }
  return cudaGetLastError();
}

template <class O>
cudaError_t moments_any(int storage, int odd, const void* pop, Grid g, const StepConsts& k, O* rho, O* u, O* B,
                        O* J, long long os, cudaStream_t s) {
  if (os == 0) os = g.n3i;
  switch (storage) {
    case 1: return moments_t<float, O>(odd, pop, g, k, rho, u, B, J, os, s);
    case 2: return moments_t<__half, O>(odd, pop, g, k, rho, u, B, J, os, s);
    case 3: return moments_t<__nv_bfloat16, O>(odd, pop, g, k, rho, u, B, J, os, s);
  }
  return cudaErrorInvalidValue;
}

template <class T>
cudaError_t populations_t(int odd, const void* pop, Grid g, const StepConsts& k, double* f, cudaStream_t s) {
  const dim3 b = site_block(g), gr = site_grid(g, b);
  if (odd)
    populations_kernel<T, true><<<gr, b, 0, s>>>(static_cast<const T*>(pop), g, k, f);
  else
    populations_kernel<T, false><<<gr, b, 0, s>>>(static_cast<const T*>(pop), g, k, f);
  return cudaGetLastError();
}

template <class T>
cudaError_t reduce_t(int odd, const void* pop, Grid g, const StepConsts& k, int nblocks, double* partials,
                     double* out, cudaStream_t s) {
  if (odd)
    reduce_kernel<T, true><<<nblocks, kRedThreads, 0, s>>>(static_cast<const T*>(pop), g, k, Consts64(k), partials);
  else
    reduce_kernel<T, false><<<nblocks, kRedThreads, 0, s>>>(static_cast<const T*>(pop), g, k, Consts64(k), partials);
  reduce_final_kernel<<<1, 32 * kRedVals, 0, s>>>(partials, nblocks, out);
  return cudaGetLastError();
}


}  // namespace

cudaError_t launch_init(int storage, void* pop, Grid g, const StepConsts& k, int noneq, const double* rho,
                        const double* u, const double* B, const double* gu, const double* gB,
                        unsigned* speed_bits, cudaStream_t s) {
  return init_t<double>(storage, pop, g, k, noneq, rho, u, B, gu, gB, speed_bits, s);
}

cudaError_t launch_init_f32(int storage, void* pop, Grid g, const StepConsts& k, int noneq, const float* rho,
                            const float* u, const float* B, const float* gu, const float* gB,
                            unsigned* speed_bits, cudaStream_t s) {
  return init_t<float>(storage, pop, g, k, noneq, rho, u, B, gu, gB, speed_bits, s);
}

cudaError_t launch_moments(int storage, int odd, const void* pop, Grid g, const StepConsts& k, double* rho,
                           double* u, double* B, double* J, cudaStream_t s, long long ostride) {
  return moments_any<double>(storage, odd, pop, g, k, rho, u, B, J, ostride, s);
}

cudaError_t launch_moments_f32(int storage, int odd, const void* pop, Grid g, const StepConsts& k, float* rho,
                               float* u, float* B, float* J, cudaStream_t s, long long ostride) {
  return moments_any<float>(storage, odd, pop, g, k, rho, u, B, J, ostride, s);
}

cudaError_t launch_populations(int storage, int odd, const void* pop, Grid g, const StepConsts& k, double* f,
                               cudaStream_t s) {
  switch (storage) {
    case 1: return populations_t<float>(odd, pop, g, k, f, s);
    case 2: return populations_t<__half>(odd, pop, g, k, f, s);
    case 3: return populations_t<__nv_bfloat16>(odd, pop, g, k, f, s);
  }
  return cudaErrorInvalidValue;
}

cudaError_t launch_probe(int storage, int odd, const void* pop, Grid g, const StepConsts& k, int n,
                         const long long* sites, double* out, cudaStream_t s) {
  if (n <= 0) return cudaSuccess;
  switch (storage) {
    case 1: return probe_t<float>(odd, pop, g, k, n, sites, out, s);
    case 2: return probe_t<__half>(odd, pop, g, k, n, sites, out, s);
    case 3: return probe_t<__nv_bfloat16>(odd, pop, g, k, n, sites, out, s);
  }
  return cudaErrorInvalidValue;
}

cudaError_t launch_reduce_partials(int storage, int odd, const void* pop, Grid g, const StepConsts& k, int nblocks,
                                   double* partials, cudaStream_t s) {
  if (nblocks < 1) return cudaErrorInvalidValue;
  switch (storage) {
    case 1:
      if (odd) reduce_kernel<float, true><<<nblocks, kRedThreads, 0, s>>>(static_cast<const float*>(pop), g, k, Consts64(k), partials);
      else reduce_kernel<float, false><<<nblocks, kRedThreads, 0, s>>>(static_cast<const float*>(pop), g, k, Consts64(k), partials);
      break;
    case 2:
      if (odd) reduce_kernel<__half, true><<<nblocks, kRedThreads, 0, s>>>(static_cast<const __half*>(pop), g, k, Consts64(k), partials);
      else reduce_kernel<__half, false><<<nblocks, kRedThreads, 0, s>>>(static_cast<const __half*>(pop), g, k, Consts64(k), partials);
      break;
    case 3:
      if (odd) reduce_kernel<__nv_bfloat16, true><<<nblocks, kRedThreads, 0, s>>>(static_cast<const __nv_bfloat16*>(pop), g, k, Consts64(k), partials);
      else reduce_kernel<__nv_bfloat16, false><<<nblocks, kRedThreads, 0, s>>>(static_cast<const __nv_bfloat16*>(pop), g, k, Consts64(k), partials);
      break;
    default:
      return cudaErrorInvalidValue;
  }
  return cudaGetLastError();
}

cudaError_t launch_reduce(int storage, int odd, const void* pop, Grid g, const StepConsts& k, int nblocks,
                          double* partials, double* out, cudaStream_t s) {
  if (nblocks < 1 || nblocks > kRedBlocksMax) return cudaErrorInvalidValue;
  switch (storage) {
    case 1: return reduce_t<float>(odd, pop, g, k, nblocks, partials, out, s);
    case 2: return reduce_t<__half>(odd, pop, g, k, nblocks, partials, out, s);
    case 3: return reduce_t<__nv_bfloat16>(odd, pop, g, k, nblocks, partials, out, s);
  }
  return cudaErrorInvalidValue;
}


}  // namespace flame
