// FP64 collision with its sums in 64-bit integers.
//
// What bounds the FP64 step on sm_103a: the FP64 pipe takes 2 operations per
// clock and SM, 32 times fewer than the integer pipes, and a collision written
// in doubles is 70 (D2Q9) to 150 (D3Q19) of them per node.  Most of those are
// additions of populations of the same size, which integers do exactly.  So a
// node's populations become fixed-point numbers on one grid, U = 2^(sc - 62)
// with 2^sc the power of two just above rho0 (a double of at least 2^(sc - 10)
// lands on the grid without rounding; 53 bits are kept of what is smaller):
//   * every sum and difference of populations, and every combination of the
//     relaxed moments back into directions, is an integer addition: exact;
//   * the few products (momentum times velocity, the relaxation rates) stay in
//     doubles, in units of U, with one conversion each way;
//   * D3Q19's (1 - omega) f_i is a 64 x 64-bit integer product, right to about
//     one U;
//   * the result is rounded once, to nearest even, to the double stored.
// U is 2^-3 to 2^-5 of the last place of a population w_i rho0, so the result
// is as near to the exact one as the rounding of the stored double lets it be;
// the same sums in doubles round at the last place of rho.
//
// A node outside the range of the grid (a negative population or one far
// below w_i rho0, rho outside (2^(sc-2), 2^(sc+1)), a velocity near 1/2, not
// a number, ...) is found by integer tests on the way and left to the
// collision in doubles: the function returns false without storing anything.
#pragma once
#include <cmath>
#include <cstdint>

#include "lattice.cuh"

namespace lbm {

// Largest |g| / rho0 the grid takes (its terms must not carry a sum out of
// 64 bits); a stronger force runs the collision in doubles.
constexpr double kFixedMaxForce = 1.0 / 512;

// Fills the constants for stencil L; collision 1 is MRT (D2Q9).
template <class L>
inline void fold_fixed(FixedK& k, double omega, double fpre3, const double g[3], double rho0, int collision) {
  k = FixedK{};
  int e2 = 0;
  std::frexp(rho0, &e2);  // rho0 = m 2^e2, m in [1/2, 1)
  k.sc = e2;
  bool on = e2 > -900 && e2 < 900;
  for (int a = 0; a < 3; ++a) on = on && std::fabs(g[a]) <= kFixedMaxForce * rho0;
  k.on = on ? 1 : 0;
  if (!on) return;
  const double unit = std::ldexp(1.0, 62 - e2);  // grid steps per 1
  k.step = std::ldexp(1.0, e2 - 62);
  for (int a = 0; a < 3; ++a) k.hg[a] = 0.5 * g[a] * unit;
  if (L::Q == 9) {
    // relaxation rates of e, epsilon, q, p (Sec. 2: 1.5, 1.5, 1.2, omega); BGK: omega for all
    const double se = collision == 1 ? 1.5 : omega, sq = collision == 1 ? 1.2 : omega;
    k.c[0] = se / 36.0;
    k.c[1] = 3.0 * se / 36.0;
    k.c[2] = sq / 12.0;
    k.c[3] = omega / 4.0;
    for (int a = 0; a < 2; ++a) {
      k.ge[a] = (1.0 - 0.5 * se) / 6.0 * g[a] * unit;
      k.gp[a] = (1.0 - 0.5 * omega) / 4.0 * g[a] * unit;
      k.gq[a] = g[a] / 12.0 * unit;
      k.gj[a] = (int64_t)std::llrint(g[a] / 6.0 * unit);
    }
  } else {
    k.c[0] = omega / 8.0;
    k.c[1] = omega / 12.0;
    k.c[2] = omega / 36.0;
    k.c[3] = 1.0 / 3.0;
    for (int a = 0; a < 3; ++a) {
      k.ge[a] = fpre3 / 24.0 * g[a] * unit;
      k.gq[a] = fpre3 / 36.0 * g[a] * unit;
    }
    const double om1 = 1.0 - omega;  // in (-1, 1)
    const uint64_t om = (uint64_t)std::ldexp(std::fabs(om1), 63);
    k.oh = (uint32_t)(om >> 32);
    k.oh2 = 2u * k.oh;
    k.ol = (uint32_t)om;
    // centres the two parts a product drops (fl ol and the bits shifted out)
    k.oc = (1ull << 30) + (k.ol >> 1);
    k.neg = om1 < 0.0 ? ~0ull : 0ull;
  }
}

#ifdef __CUDACC__

// f on the grid: the 53-bit significand aligned for an exponent of at most
// sc - 10 + SH (populations below 2^(SH - 9 + sc)), moved down by n places.
// Any n outside 0 .. 31 (which a sign bit, a zero, an infinity and a NaN also
// give) sets bits above the fifth in `bad`.
template <int SH>
__device__ __forceinline__ uint64_t to_grid(double f, int sc, uint32_t& bad) {
  const uint32_t lo = (uint32_t)__double2loint(f), hi = (uint32_t)__double2hiint(f);
  const uint32_t n = (uint32_t)(1013 + SH + sc) - (hi >> 20);
  bad |= n;
  const uint32_t mh = (__funnelshift_l(lo, hi, SH) & ((1u << (20 + SH)) - 1)) | (1u << (20 + SH));
  const uint32_t ml = lo << SH;
  return ((uint64_t)__funnelshift_r(mh, 0u, n) << 32) | __funnelshift_r(ml, mh, n);
}

// The double nearest (ties to even) to v steps of the grid; v in [2^32, 2^63),
// else the sign bit of `bad` is set and the value is meaningless.
__device__ __forceinline__ double from_grid(uint64_t v, int sc, uint32_t& bad) {
  const uint32_t hi = (uint32_t)(v >> 32), lo = (uint32_t)v;
  bad |= hi | (hi - 1u);
  const uint32_t lz = (uint32_t)__clz((int)hi);
  const uint32_t sh = lz - 1u;  // leading bit to place 62
  const uint32_t xh = __funnelshift_l(lo, hi, sh), xl = __funnelshift_l(0u, lo, sh);
  const uint64_t x = (((uint64_t)xh << 32) | xl) + (0x1ffu + ((xl >> 10) & 1u));
  const uint32_t yh = (uint32_t)(x >> 32);
  // the leading bit adds one to the exponent field
  return __hiloint2double((int)((yh >> 10) + ((uint32_t)(1023 + sc) << 20) - (lz << 20)),
                          (int)__funnelshift_r((uint32_t)x, yh, 10));
}

// 1/x by two Newton-Raphson steps on the hardware's approximate reciprocal
// (x positive and normal).
__device__ __forceinline__ double newton_reciprocal(double x) {
  double y;
  asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
  y = fma(fma(-x, y, 1.0), y, y);
  return fma(fma(-x, y, 1.0), y, y);
}

// Whether v, as a signed number, lies in [-2^61, 2^61): 0 if it does.
__device__ __forceinline__ uint32_t beyond61(uint64_t v) { return ((uint32_t)(v >> 32) + 0x20000000u) >> 30; }

// rho, u of the node in the units of the moment cache.
struct NodeMom {
  double rho, ux, uy, uz;
};

// D2Q9, BGK and MRT: f (pre-collision) is replaced by the post-collision
// populations.  In moment space (rows of M, Sec. 2) every moment but rho and j
// relaxes; with X = f0 - Sa and Y = Sa - 4 Sd (Sa, Sd: sums over the axis and
// the diagonal directions) the non-equilibrium moments are
//   e:  -2 X - Y - 3 rho u.u,  epsilon: 3 (X + rho u.u),
//   q_x: -a + 2 b (a = f1 - f3, b = f5 - f6 - f7 + f8),  p: p - rho u u,
// and the Guo source adds (1 - s/2)(6 u.g, -6 u.g, -g, 2 (ux gx - uy gy),
// ux gy + uy gx).  BGK is the case of one rate, so no population is multiplied.
__device__ __forceinline__ bool collide_grid(double (&f)[9], const FixedK& k, bool force, NodeMom& m) {
  uint32_t bad = 0, wide = 0;
  uint64_t F[9];
  F[0] = to_grid<9>(f[0], k.sc, bad);
#pragma unroll
  for (int i = 1; i < 9; ++i) F[i] = to_grid<7>(f[i], k.sc, bad);
  const uint64_t s13 = F[1] + F[3], s24 = F[2] + F[4], s57 = F[5] + F[7], s68 = F[6] + F[8];
  const uint64_t d13 = F[1] - F[3], d24 = F[2] - F[4], d57 = F[5] - F[7], d68 = F[6] - F[8];
  const uint64_t Sa = s13 + s24, Sd = s57 + s68, r = F[0] + Sa + Sd;
  const uint64_t X = F[0] - Sa, Y = Sa - 4 * Sd;
  const uint64_t bx = d57 - d68, by = d57 + d68;
  wide = beyond61(X) | beyond61(Y) | (uint32_t)(Sd >> 61) | (uint32_t)(r >> 63) | ((uint32_t)(r >> 60) == 0u ? 1u : 0u);
  const double rd = __ll2double_rn((long long)r);
  double Jx = __ll2double_rn((long long)(d13 + bx)), Jy = __ll2double_rn((long long)(d24 + by));
  const double Xd = __ll2double_rn((long long)X), Yd = __ll2double_rn((long long)Y);
  const double Qx = __ll2double_rn((long long)(2 * bx - d13)), Qy = __ll2double_rn((long long)(2 * by - d24));
  const double Px = __ll2double_rn((long long)(s13 - s24)), Pxy = __ll2double_rn((long long)(s57 - s68));
  if (force) {
    Jx += k.hg[0];
    Jy += k.hg[1];
  }
  const double inv = newton_reciprocal(rd);
  const double ux = Jx * inv, uy = Jy * inv;
  const double qxx = Jx * ux, qyy = Jy * uy, qxy = Jx * uy;
  const double E = qxx + qyy;
  // rho u.u at most 1/4 (grid units 2^60)
  wide |= (uint32_t)__double2hiint(E) >= 0x43b00000u ? 1u : 0u;
  double De = k.c[0] * fma(-2.0, Xd, fma(-3.0, E, -Yd));
  double Dp = k.c[1] * (Xd + E);
  double Dx = k.c[2] * Qx, Dy = k.c[2] * Qy;
  double Dxx = k.c[3] * ((Px - qxx) + qyy), Dxy = k.c[3] * (Pxy - qxy);
  if (force) {
    const double de = fma(k.ge[0], ux, k.ge[1] * uy);
    De -= de;
    // the same force term with the rate of epsilon (equal to e's)
    Dp += de;
    Dx += k.gq[0];
    Dy += k.gq[1];
    Dxx = fma(-2.0 * k.gp[0], ux, fma(2.0 * k.gp[1], uy, Dxx));
    Dxy = fma(-k.gp[1], ux, fma(-k.gp[0], uy, Dxy));
  }
  const uint64_t ie = (uint64_t)__double2ll_rn(De), ip = (uint64_t)__double2ll_rn(Dp);
  const uint64_t ix = (uint64_t)__double2ll_rn(Dx), iy = (uint64_t)__double2ll_rn(Dy);
  const uint64_t ixx = (uint64_t)__double2ll_rn(Dxx), ixy = (uint64_t)__double2ll_rn(Dxy);
  const uint64_t gx = (uint64_t)k.gj[0], gy = (uint64_t)k.gj[1];
  F[0] += 4 * (ie - ip);
  const uint64_t ax = ie + 2 * ip;                       // axis: + e + 2 epsilon
  const uint64_t tx = 2 * ix + gx, ty = 2 * iy + gy;     // 2 q - j (j's part is -g/6)
  const uint64_t px = ax - ixx, py = ax + ixx;
  F[1] += px + tx;
  F[3] += px - tx;
  F[2] += py + ty;
  F[4] += py - ty;
  const uint64_t dg = 2 * ie + ip;                       // diagonal: - 2 e - epsilon
  const uint64_t vx = gx - ix, vy = gy - iy;             // - j - q
  const uint64_t d0 = 0 - dg - ixy, d1 = ixy - dg;
  F[5] += d0 + (vx + vy);
  F[7] += d0 - (vx + vy);
  F[6] += d1 - (vx - vy);
  F[8] += d1 + (vx - vy);
  uint32_t out = 0;
#pragma unroll
  for (int i = 0; i < 9; ++i) f[i] = from_grid(F[i], k.sc, out);
  m = NodeMom{rd * k.step, ux, uy, 0.0};
  return bad < 32u && wide == 0u && (int32_t)out >= 0;
}

// D3Q19 BGK: f+_i = (1 - omega) f_i + omega feq_i + src_i.  In units of a
// diagonal direction's weight 1/36 the last two are integer combinations of
//   B = omega rho/36 - (T_xx + T_yy + T_zz)/3,
//   T_ab = (omega/8) rho u_a u_b + (pre/24)(g_a u_b + g_b u_a),
//   M_a = (omega/12) rho u_a + (pre/36) g_a       (pre = 3 (1 - omega/2)):
// rest 12 B; axis 2 (B + T_aa +- M_a); diagonal B + T_aa + T_bb +- 2 T_ab +-
// (M_a +- M_b).
__device__ __forceinline__ bool collide_grid(double (&f)[19], const FixedK& k, bool force, NodeMom& m) {
  uint32_t bad = 0, wide = 0;
  uint64_t F[19];
  F[0] = to_grid<9>(f[0], k.sc, bad);
#pragma unroll
  for (int i = 1; i < 19; ++i) F[i] = to_grid<6>(f[i], k.sc, bad);
  uint64_t r = F[0], jx, jy, jz;
#pragma unroll
  for (int i = 1; i < 19; ++i) r += F[i];
  {
    const uint64_t d7 = F[7] - F[8], d9 = F[9] - F[10], d11 = F[11] - F[12], d13 = F[13] - F[14],
                   d15 = F[15] - F[16], d17 = F[17] - F[18];
    jx = (F[1] - F[2]) + (d7 + d9) + (d11 + d13);
    jy = (F[3] - F[4]) + (d7 - d9) + (d15 + d17);
    jz = (F[5] - F[6]) + (d11 - d13) + (d15 - d17);
  }
  wide = (uint32_t)(r >> 63) | ((uint32_t)(r >> 60) == 0u ? 1u : 0u);
  const double rd = __ll2double_rn((long long)r);
  double Jx = __ll2double_rn((long long)jx), Jy = __ll2double_rn((long long)jy), Jz = __ll2double_rn((long long)jz);
  if (force) {
    Jx += k.hg[0];
    Jy += k.hg[1];
    Jz += k.hg[2];
  }
  const double inv = newton_reciprocal(rd);
  const double ux = Jx * inv, uy = Jy * inv, uz = Jz * inv;
  const double Wx = k.c[0] * Jx, Wy = k.c[0] * Jy, Wz = k.c[0] * Jz;
  double Txx = Wx * ux, Tyy = Wy * uy, Tzz = Wz * uz, Txy, Txz, Tyz;
  double Mx = k.c[1] * Jx, My = k.c[1] * Jy, Mz = k.c[1] * Jz;
  if (force) {
    const double vx = Wx + k.ge[0], vy = Wy + k.ge[1];
    Txy = fma(vx, uy, k.ge[1] * ux);
    Txz = fma(vx, uz, k.ge[2] * ux);
    Tyz = fma(vy, uz, k.ge[2] * uy);
    Txx = fma(2.0 * k.ge[0], ux, Txx);
    Tyy = fma(2.0 * k.ge[1], uy, Tyy);
    Tzz = fma(2.0 * k.ge[2], uz, Tzz);
    Mx += k.gq[0];
    My += k.gq[1];
    Mz += k.gq[2];
  } else {
    Txy = Wx * uy;
    Txz = Wx * uz;
    Tyz = Wy * uz;
  }
  const double tr = (Txx + Tyy) + Tzz;
  // (omega/8) rho u.u at most 2^-5 (grid units 2^57); negative only by a force term
  wide |= ((uint32_t)__double2hiint(tr) & 0x7fffffffu) >= 0x43800000u ? 1u : 0u;
  const uint64_t B = (uint64_t)__double2ll_rn(fma(k.c[2], rd, -k.c[3] * tr));
  const uint64_t ixx = (uint64_t)__double2ll_rn(Txx), iyy = (uint64_t)__double2ll_rn(Tyy),
                 izz = (uint64_t)__double2ll_rn(Tzz);
  const uint64_t ixy = 2 * (uint64_t)__double2ll_rn(Txy), ixz = 2 * (uint64_t)__double2ll_rn(Txz),
                 iyz = 2 * (uint64_t)__double2ll_rn(Tyz);
  const uint64_t mx = (uint64_t)__double2ll_rn(Mx), my = (uint64_t)__double2ll_rn(My),
                 mz = (uint64_t)__double2ll_rn(Mz);
  uint32_t out = 0;
  auto put = [&](int i, uint64_t c) {
    // (1 - omega) F_i: |1 - omega| as oh 2^32 + ol over 2^63; F < 2^62
    const uint32_t fh = (uint32_t)(F[i] >> 32), fl = (uint32_t)F[i];
    const uint64_t mid = (uint64_t)fl * k.oh + k.oc + (uint64_t)fh * k.ol;
    const uint64_t R = (uint64_t)fh * k.oh2 + (mid >> 31);
    f[i] = from_grid(c + ((R ^ k.neg) - k.neg), k.sc, out);
  };
  auto pair = [&](int i, uint64_t P, uint64_t M) {
    put(i, P + M);
    put(i + 1, P - M);
  };
  put(0, 12 * B);
  const uint64_t Bx = B + ixx, By = B + iyy, Bz = B + izz;
  pair(1, 2 * Bx, 2 * mx);
  pair(3, 2 * By, 2 * my);
  pair(5, 2 * Bz, 2 * mz);
  const uint64_t Bxy = Bx + iyy, Bxz = Bx + izz, Byz = By + izz;
  pair(7, Bxy + ixy, mx + my);
  pair(9, Bxy - ixy, mx - my);
  pair(11, Bxz + ixz, mx + mz);
  pair(13, Bxz - ixz, mx - mz);
  pair(15, Byz + iyz, my + mz);
  pair(17, Byz - iyz, my - mz);
  m = NodeMom{rd * k.step, ux, uy, uz};
  return bad < 32u && wide == 0u && (int32_t)out >= 0;
}

#endif  // __CUDACC__

}  // namespace lbm
