// FP32 D2Q9 BGK collision, written once over a number type: one node per
// thread (float) or two neighbouring nodes (F2, the packed operations of
// sm_100 and later, which take one issue slot for two results).
//
// What bounds a D2Q9 FP32 pull pass that keeps HBM's reads in flight is
// instruction issue: 350 instructions per 32 nodes with one node per lane, 57 %
// of the slots busy and waiting besides.  Two neighbours share their run
// record, every address (the second is 4 bytes on), their stores (8 bytes) and
// the packed arithmetic.
//
// Every operation is an explicit rounded add, multiply or FMA, so a node has
// the same bits in either form, whatever kernel takes it.
#pragma once
#include <cstdint>

#include "lattice.cuh"

namespace lbm {

#ifdef __CUDACC__

struct F2 {
  unsigned long long v;
};
__device__ __forceinline__ F2 pack2(float a, float b) {
  F2 r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r.v) : "f"(a), "f"(b));
  return r;
}
__device__ __forceinline__ float low(const F2& x) {
  float a;
  asm("mov.b64 {%0, _}, %1;" : "=f"(a) : "l"(x.v));
  return a;
}
__device__ __forceinline__ float high(const F2& x) {
  float b;
  asm("mov.b64 {_, %0}, %1;" : "=f"(b) : "l"(x.v));
  return b;
}

template <class V>
struct Num;
template <>
struct Num<float> {
  static __device__ __forceinline__ float all(float c) { return c; }
  static __device__ __forceinline__ float add(float a, float b) { return __fadd_rn(a, b); }
  static __device__ __forceinline__ float sub(float a, float b) { return __fsub_rn(a, b); }
  static __device__ __forceinline__ float mul(float a, float b) { return __fmul_rn(a, b); }
  static __device__ __forceinline__ float fma(float a, float b, float c) { return __fmaf_rn(a, b, c); }
  static __device__ __forceinline__ float rcp_seed(float a) {
    float r;
    asm("rcp.approx.f32 %0, %1;" : "=f"(r) : "f"(a));
    return r;
  }
};
template <>
struct Num<F2> {
  static __device__ __forceinline__ F2 all(float c) { return pack2(c, c); }
  static __device__ __forceinline__ F2 add(F2 a, F2 b) {
    F2 r;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
    return r;
  }
  static __device__ __forceinline__ F2 mul(F2 a, F2 b) {
    F2 r;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
    return r;
  }
  static __device__ __forceinline__ F2 fma(F2 a, F2 b, F2 c) {
    F2 r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r.v) : "l"(a.v), "l"(b.v), "l"(c.v));
    return r;
  }
  // a - b, rounded once
  static __device__ __forceinline__ F2 sub(F2 a, F2 b) { return fma(b, all(-1.f), a); }
  static __device__ __forceinline__ F2 rcp_seed(F2 a) {
    return pack2(Num<float>::rcp_seed(low(a)), Num<float>::rcp_seed(high(a)));
  }
};

// Run parameters of a node (or of two): rho0, omega, and where a body force
// acts g, g/2 and the folded source constants of the weight classes and of one
// direction of each opposite pair (1, 2, 5, 6).
template <class V>
struct Bgk32 {
  V rho0, om, hx, hy, gx, gy, kf[3], kt[4], ke[4];
};

// f (pre-collision, shifted) becomes f+; r, ux, uy: the node's moments.  Each
// direction keeps its own feq_i = w (r + rho poly_i) and relaxes in the
// difference form f - omega (f - feq), the difference rounded once, so that
// rounding falls on the small non-equilibrium part (rounding feq by itself
// first made the channel's errors a fifth larger); opposite directions share
// e.u, the symmetric part of the polynomial and the source's two parts.
template <class V>
__device__ __forceinline__ void bgk_d2q9(V (&f)[9], const Bgk32<V>& c, bool force, V& r, V& ux, V& uy) {
  using N = Num<V>;
  const V s13 = N::add(f[1], f[3]), s24 = N::add(f[2], f[4]), s57 = N::add(f[5], f[7]), s68 = N::add(f[6], f[8]);
  const V d13 = N::sub(f[1], f[3]), d24 = N::sub(f[2], f[4]), d57 = N::sub(f[5], f[7]), d68 = N::sub(f[6], f[8]);
  r = N::add(f[0], N::add(N::add(s13, s24), N::add(s57, s68)));
  const V jx = N::add(d13, N::sub(d57, d68)), jy = N::add(d24, N::add(d57, d68));
  const V rho = N::add(c.rho0, r);
  // 1/rho: the hardware's reciprocal and a Newton-Raphson step with one rounding
  // at its end, the correctly rounded quotient for every float from 2^-30 to 2^31
  V inv = N::rcp_seed(rho);
  inv = N::fma(inv, N::fma(N::mul(rho, N::all(-1.f)), inv, N::all(1.f)), inv);
  ux = N::mul(force ? N::add(jx, c.hx) : jx, inv);
  uy = N::mul(force ? N::add(jy, c.hy) : jy, inv);
  // - 3/2 u.u
  const V nu = N::mul(N::all(-1.5f), N::fma(ux, ux, N::mul(uy, uy)));
  V ug = nu;
  if (force) ug = N::fma(ux, c.gx, N::mul(uy, c.gy));
  const V mo = N::mul(c.om, N::all(-1.f));
  constexpr float w0 = (float)(4.0 / 9.0), w1 = (float)(1.0 / 9.0), w2 = (float)(1.0 / 36.0);
  {
    V o = N::fma(mo, N::fma(N::all(-w0), N::fma(rho, nu, r), f[0]), f[0]);
    if (force) o = N::sub(o, N::mul(c.kf[0], ug));
    f[0] = o;
  }
  auto pair = [&](int i, int j, int cls, float w, V eu, int n) {
    const V sym = N::fma(N::all(4.5f), N::mul(eu, eu), nu);
    const V pi = N::fma(N::all(3.f), eu, sym), pj = N::fma(N::all(-3.f), eu, sym);
    V oi = N::fma(mo, N::fma(N::all(-w), N::fma(rho, pi, r), f[i]), f[i]);
    V oj = N::fma(mo, N::fma(N::all(-w), N::fma(rho, pj, r), f[j]), f[j]);
    if (force) {
      const V Sc = N::sub(N::mul(c.kt[n], eu), N::mul(c.kf[cls], ug));
      oi = N::add(oi, N::add(Sc, c.ke[n]));
      oj = N::add(oj, N::sub(Sc, c.ke[n]));
    }
    f[i] = oi;
    f[j] = oj;
  };
  pair(1, 3, 1, w1, ux, 0);
  pair(2, 4, 1, w1, uy, 1);
  pair(5, 7, 2, w2, N::add(ux, uy), 2);
  pair(6, 8, 2, w2, N::sub(uy, ux), 3);
}

// Transpose of the collision at one node or two (see collide_adjoint, whose
// moments of d_i = lambda_i - mean lambda these are, with opposite directions
// paired): mu from the pre-collision f and lambda(s+1); returns the node's
// sum_i lambda_i dC_i/dtau.
template <class V>
__device__ __forceinline__ V adjoint_d2q9(const V (&f)[9], const V (&lam)[9], V (&mu)[9], const Bgk32<V>& c,
                                          bool force) {
  using N = Num<V>;
  constexpr float w0 = (float)(4.0 / 9.0), w1 = (float)(1.0 / 9.0), w2 = (float)(1.0 / 36.0);
  const V d13 = N::sub(f[1], f[3]), d24 = N::sub(f[2], f[4]), d57 = N::sub(f[5], f[7]), d68 = N::sub(f[6], f[8]);
  const V r = N::add(f[0], N::add(N::add(N::add(f[1], f[3]), N::add(f[2], f[4])),
                                  N::add(N::add(f[5], f[7]), N::add(f[6], f[8]))));
  const V jx = N::add(d13, N::sub(d57, d68)), jy = N::add(d24, N::add(d57, d68));
  const V rho = N::add(c.rho0, r);
  V ir = N::rcp_seed(rho);
  ir = N::fma(ir, N::fma(N::mul(rho, N::all(-1.f)), ir, N::all(1.f)), ir);
  const V ux = N::mul(force ? N::add(jx, c.hx) : jx, ir), uy = N::mul(force ? N::add(jy, c.hy) : jy, ir);
  const V nu = N::mul(N::all(-1.5f), N::fma(ux, ux, N::mul(uy, uy)));
  const V lbar = N::mul(
      N::all((float)(1.0 / 9.0)),
      N::add(lam[0], N::add(N::add(N::add(lam[1], lam[3]), N::add(lam[2], lam[4])),
                            N::add(N::add(lam[5], lam[7]), N::add(lam[6], lam[8])))));
  V d[9];
#pragma unroll
  for (int i = 0; i < 9; ++i) d[i] = N::sub(lam[i], lbar);
  V lf = N::mul(d[0], f[0]);
#pragma unroll
  for (int i = 1; i < 9; ++i) lf = N::fma(d[i], f[i], lf);
  const V p13 = N::add(d[1], d[3]), p24 = N::add(d[2], d[4]), p57 = N::add(d[5], d[7]), p68 = N::add(d[6], d[8]);
  const V m57 = N::sub(d[5], d[7]), m68 = N::sub(d[6], d[8]);
  const V diag = N::mul(N::all(w2), N::add(p57, p68));
  const V S0 = N::fma(N::all(w0), d[0], N::fma(N::all(w1), N::add(p13, p24), diag));
  const V Sx = N::fma(N::all(w1), N::sub(d[1], d[3]), N::mul(N::all(w2), N::sub(m57, m68)));
  const V Sy = N::fma(N::all(w1), N::sub(d[2], d[4]), N::mul(N::all(w2), N::add(m57, m68)));
  const V Txx = N::fma(N::all(w1), p13, diag), Tyy = N::fma(N::all(w1), p24, diag);
  const V Txy = N::mul(N::all(w2), N::sub(p57, p68));
  const V Tux = N::fma(Txx, ux, N::mul(Txy, uy)), Tuy = N::fma(Txy, ux, N::mul(Tyy, uy));
  const V uS = N::fma(ux, Sx, N::mul(uy, Sy)), uTu = N::fma(ux, Tux, N::mul(uy, Tuy));
  const V dpoly = N::fma(nu, S0, N::fma(N::all(4.5f), uTu, N::mul(N::all(3.f), uS)));
  const V orho = N::mul(c.om, rho), s3 = N::mul(N::all(-3.f), S0);
  V B0 = N::mul(orho, N::fma(s3, ux, N::fma(N::all(9.f), Tux, N::mul(N::all(3.f), Sx))));
  V B1 = N::mul(orho, N::fma(s3, uy, N::fma(N::all(9.f), Tuy, N::mul(N::all(3.f), Sy))));
  V dt = N::sub(lf, N::fma(rho, dpoly, N::mul(r, S0)));
  if (force) {
    const V c2 = N::fma(N::all(-0.5f), c.om, N::all(1.f));
    const V Tgx = N::fma(Txx, c.gx, N::mul(Txy, c.gy)), Tgy = N::fma(Txy, c.gx, N::mul(Tyy, c.gy));
    B0 = N::fma(c2, N::fma(s3, c.gx, N::mul(N::all(9.f), Tgx)), B0);
    B1 = N::fma(c2, N::fma(s3, c.gy, N::mul(N::all(9.f), Tgy)), B1);
    // sum d_i src_i = 3 g.S - 3 (u.g) S0 + 9 u.T.g
    const V ug = N::fma(ux, c.gx, N::mul(uy, c.gy));
    V src = N::mul(N::all(3.f), N::fma(c.gx, Sx, N::mul(c.gy, Sy)));
    src = N::fma(N::all(9.f), N::fma(ux, Tgx, N::mul(uy, Tgy)), N::fma(s3, ug, src));
    dt = N::fma(N::all(0.5f), src, dt);
  }
  // mu_i = lambda_i + (omega (A - lambda_i) + (e_i - u).B/rho), A - lambda_i
  // formed as S0 + dpoly - d_i: the transpose too relaxes in the difference form,
  // so that rounding falls on the small part.  Relative r.m.s. error of the
  // per-link dJ/dq of 40 cylinders over 4000 steps 3.3e-5, 3.4e-5 with
  // (1 - omega) lambda_i + omega A and one addition less a direction.
  const V bx = N::mul(B0, ir), by = N::mul(B1, ir), G = N::add(S0, dpoly);
  const V ub = N::fma(bx, ux, N::mul(by, uy)), C = N::mul(N::all(-1.f), ub);
  auto put = [&](int i, V b) { mu[i] = N::add(lam[i], N::fma(c.om, N::sub(G, d[i]), b)); };
  put(0, C);
  put(1, N::add(C, bx));
  put(3, N::sub(C, bx));
  put(2, N::add(C, by));
  put(4, N::sub(C, by));
  const V s = N::add(bx, by), t = N::sub(bx, by);
  put(5, N::add(C, s));
  put(7, N::sub(C, s));
  put(8, N::add(C, t));
  put(6, N::sub(C, t));
  return N::mul(dt, N::mul(c.om, c.om));
}

#endif  // __CUDACC__

}  // namespace lbm
