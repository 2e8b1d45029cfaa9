// FP64 collision in 64-bit integers.
//
// What bounds the FP64 step on sm_103a: the FP64 pipe takes 2 operations per
// clock and SM, 32 times fewer than the integer pipes (a 32 x 32 -> 64-bit
// multiply-add: 16 per clock and SM), and a collision in doubles is 72
// (D2Q9 BGK) to 150 (D3Q19) of them per node, about 400 for MRT.  So a node's
// populations become fixed-point numbers on one grid of step U = 2^(sc - 62),
// with sc such that rho0 is 0.75 .. 1.5 times 2^sc (a double of at least
// 2^(sc - 9) lands on the grid without rounding; 53 bits are kept of what is
// smaller):
//   * every sum and difference of populations, and every combination of the
//     relaxed moments back into directions, is an integer addition: exact;
//   * a product is three 32 x 32 -> 64-bit multiply-adds (the low-by-low term
//     is below the grid), right to about one U;
//   * 1/rho is the one quantity formed in doubles (four FP64 operations);
//   * the result is rounded once, to the double stored.
// U is 2^-4 to 2^-6 of the last place of a population w_i rho0; the same sums
// in doubles round at the last place of rho.  Measured against 64-bit
// references (u after 5 steps): dense D3Q19 7.6e-15 in doubles, 6.1e-15 here;
// the mass of a closed lattice drifts by 3e-17 to 1e-16 a step in doubles and
// not at all over 750 steps here.
//
// A node outside the range of the grid (a negative population or one far
// below w_i rho0, rho outside (2^(sc-1), 1.75 2^sc), a velocity near 1/2, not
// a number, ...) is found by integer tests on the way and left to the
// collision in doubles: the function returns false without storing anything.
// SOON: a node whose populations, density or momentum are out of range returns
// before the products, so that a flow away from rho0 pays for the conversions
// only (2 rho0: D2Q9 2049^2 710 -> 680 us per step, D3Q19 160^3 1205 -> 1175; in
// doubles alone 679 and 1172).  k_inline does without: the branch costs its
// chain 4 % (1000 x 400 channel 21.4 -> 22.3 us), and at 2 rho0 it is no slower
// than doubles were (80 us against 81).
#pragma once
#include <cmath>
#include <cstdint>

#include "lattice.cuh"

namespace lbm {

// Largest |g| / rho0 the grid takes (its terms must not carry a sum out of
// 64 bits); a stronger force runs the collision in doubles.
constexpr double kFixedMaxForce = 1.0 / 512;

__host__ __device__ __forceinline__ Halves halves(int64_t v) {
  const uint32_t lo = (uint32_t)(uint64_t)v;
  return Halves{(int32_t)((uint32_t)((uint64_t)v >> 32) + (lo >> 31)), (int32_t)lo};
}

// Fills the constants for stencil L; collision 1 is MRT (D2Q9).
template <class L>
inline void fold_fixed(FixedK& k, double omega, double fpre3, const double g[3], double rho0, int collision) {
  k = FixedK{};
  int e2 = 0;
  const double m = std::frexp(rho0, &e2);  // rho0 = m 2^e2, m in [1/2, 1)
  k.sc = m < 0.75 ? e2 - 1 : e2;
  bool on = e2 > -900 && e2 < 900;
  k.grid = on ? 1 : 0;
  if (on) k.step = std::ldexp(1.0, k.sc - 62);
  for (int a = 0; a < 3; ++a) on = on && std::fabs(g[a]) <= kFixedMaxForce * rho0;
  k.on = on ? 1 : 0;
  if (!on) return;
  const double unit = std::ldexp(1.0, 62 - k.sc);  // grid steps per 1
  auto steps = [&](double v) { return (int64_t)std::llrint(v * unit); };
  auto rate = [](double v) { return halves((int64_t)std::llrint(std::ldexp(v, 64))); };
  for (int a = 0; a < 3; ++a) k.hg[a] = steps(0.5 * g[a]);
  if (L::Q == 9) {
    // relaxation rates of e, epsilon, q, p (Sec. 2: 1.5, 1.5, 1.2, omega); BGK: omega for all
    const double se = collision == 1 ? 1.5 : omega, sq = collision == 1 ? 1.2 : omega;
    k.c[0] = rate(se / 36.0);
    k.c[1] = rate(se / 12.0);
    k.c[2] = rate(sq / 12.0);
    k.c[3] = rate(omega / 8.0);
    for (int a = 0; a < 2; ++a) {
      k.ge[a] = halves(steps((1.0 - 0.5 * se) / 6.0 * g[a]));
      k.gp[a] = halves(steps((1.0 - 0.5 * omega) / 4.0 * g[a]));
      k.gq[a] = steps(g[a] / 12.0);
      k.gj[a] = steps(g[a] / 6.0);
    }
  } else {
    // omega/36 rounded once; omega/12 and 1 - omega follow from it exactly, so
    // that the collision keeps mass and momentum to its rounding
    const int64_t c36 = (int64_t)std::llrint(std::ldexp(omega / 36.0, 64));
    k.c[0] = rate(omega / 8.0);
    k.c[1] = halves(3 * c36);
    k.c[2] = halves(c36);
    k.c[3] = rate(1.0 / 3.0);
    for (int a = 0; a < 3; ++a) {
      k.ge[a] = halves(steps(fpre3 / 24.0 * g[a]));
      k.gq[a] = steps(fpre3 / 36.0 * g[a]);
    }
    const uint64_t o36 = 18ull * (uint64_t)c36, one = 1ull << 63;  // omega and 1 in 2^-63
    const uint64_t om = o36 <= one ? one - o36 : o36 - one;
    k.oh = (uint32_t)(om >> 32);
    k.oh2 = 2u * k.oh;
    k.ol = (uint32_t)om;
    k.neg = o36 > one ? ~0ull : 0ull;
    // centres a product: + 2^-32 ol/2 for the dropped low-by-low term.  The
    // half step that the shift drops on average stays (subtracted as ~R, one
    // step less than -R, it is half a step the same way): rounding halves up
    // in from_grid adds half a step on average
    k.oc = (uint64_t)(k.ol >> 1);
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

// The double nearest to v steps of the grid (EVEN: ties to even, else up); v
// in [2^32, 2^63), else the sign bit of `bad` is set and the value is
// meaningless.
template <bool EVEN>
__device__ __forceinline__ double from_grid(uint64_t v, int sc, uint32_t& bad) {
  const uint32_t hi = (uint32_t)(v >> 32), lo = (uint32_t)v;
  bad |= hi | (hi - 1u);
  const uint32_t lz = (uint32_t)__clz((int)hi);
  const uint32_t sh = lz - 1u;  // leading bit to place 62
  const uint32_t xh = __funnelshift_l(lo, hi, sh), xl = __funnelshift_l(0u, lo, sh);
  const uint64_t x = (((uint64_t)xh << 32) | xl) + (EVEN ? 0x1ffu + ((xl >> 10) & 1u) : 0x200u);
  const uint32_t yh = (uint32_t)(x >> 32);
  // the leading bit adds one to the exponent field
  return __hiloint2double((int)((yh >> 10) + ((uint32_t)(1023 + sc) << 20) - (lz << 20)),
                          (int)__funnelshift_r((uint32_t)x, yh, 10));
}

// a b / 2^(64 - S), right to about one; the caller keeps |b| below 2^(62 - S).
template <int S>
__device__ __forceinline__ int64_t mul_grid(const Halves& a, const Halves& b) {
  int64_t m = (int64_t)a.l * b.h + (1ll << (31 - S));
  m += (int64_t)a.h * b.l;
  return (int64_t)a.h * (int32_t)((uint32_t)b.h << S) + (m >> (32 - S));
}

// 2^61 / rho for rho = r 2^-62 in [1/2, 2): two Newton-Raphson steps on the
// hardware's approximate reciprocal.
__device__ __forceinline__ int64_t reciprocal_grid(uint64_t r) {
  uint32_t none = 0;
  const double x = from_grid<false>(r, 0, none);  // in [1/2, 2)
  double y;
  asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
  y = fma(fma(-x, y, 1.0), y, y);
  y = fma(fma(-x, y, 1.0), y, y);
  // y in (1/2, 2 + 2^-52]: 53 bits of it at places 61 and below
  const uint32_t lo = (uint32_t)__double2loint(y), hi = (uint32_t)__double2hiint(y);
  const uint32_t n = 1024u - (hi >> 20);
  const uint32_t mh = (__funnelshift_l(lo, hi, 10) & 0x3fffffffu) | 0x40000000u;
  return (int64_t)(((uint64_t)__funnelshift_r(mh, 0u, n) << 32) | __funnelshift_r(lo << 10, mh, n));
}

// Checks that signed numbers lie in [-2^B, 2^B), B > 32: the upper words moved
// into [0, 2^(B - 31)) are or-ed together and looked at once.
template <int B>
struct Within {
  uint32_t seen = 0;
  __device__ __forceinline__ void operator()(uint64_t v) { seen |= (uint32_t)(v >> 32) + (1u << (B - 32)); }
  __device__ __forceinline__ bool broken() const { return (seen >> (B - 31)) != 0u; }
};

// rho and u of a node: r in grid steps, u in 2^-60.
struct NodeMom {
  uint64_t r;
  int64_t ux, uy, uz;
  __device__ __forceinline__ double u(int64_t v) const { return (double)v * 0x1p-60; }
};

// 0 if rho = r 2^-62 lies in [1/2, 1.75).
__device__ __forceinline__ uint32_t beyond_rho(uint64_t r) {
  const uint32_t hi = (uint32_t)(r >> 32);
  return ((hi + 0x10000000u) >> 31) | (hi < 0x20000000u ? 1u : 0u);
}

// D2Q9, BGK and MRT: f (pre-collision) is replaced by the post-collision
// populations.  In moment space (rows of M, Sec. 2) every moment but rho and j
// relaxes; with X = f0 - Sa and Y = Sa - 4 Sd (Sa, Sd: sums over the axis and
// the diagonal directions) the non-equilibrium moments are
//   e:  -2 X - Y - 3 rho u.u,  epsilon: 3 (X + rho u.u),
//   q_x: -a + 2 b (a = f1 - f3, b = f5 - f6 - f7 + f8),  p: p - rho u u,
// and the Guo source adds (1 - s/2)(6 u.g, -6 u.g, -g, 2 (ux gx - uy gy),
// ux gy + uy gx).  BGK is the case of one rate, so no population is multiplied.
template <bool SOON>
__device__ __forceinline__ bool collide_grid(double (&f)[9], const FixedK& k, bool force, NodeMom& m) {
  uint32_t bad = 0, wide = 0;
  uint64_t F[9];
  F[0] = to_grid<9>(f[0], k.sc, bad);
#pragma unroll
  for (int i = 1; i < 9; ++i) F[i] = i < 5 ? to_grid<8>(f[i], k.sc, bad) : to_grid<7>(f[i], k.sc, bad);
  const uint64_t s13 = F[1] + F[3], s24 = F[2] + F[4], s57 = F[5] + F[7], s68 = F[6] + F[8];
  const uint64_t d13 = F[1] - F[3], d24 = F[2] - F[4], d57 = F[5] - F[7], d68 = F[6] - F[8];
  const uint64_t Sa = s13 + s24, Sd = s57 + s68, r = F[0] + Sa + Sd;
  const uint64_t X = F[0] - Sa, Y = Sa - 4 * Sd;
  const uint64_t bx = d57 - d68, by = d57 + d68;
  uint64_t jx = d13 + bx, jy = d24 + by;
  if (force) {
    jx += (uint64_t)k.hg[0];
    jy += (uint64_t)k.hg[1];
  }
  // |X|, |Y| < 1/4, Sd < 1/2, |j| < 1/2
  Within<60> quarter;
  Within<61> half;
  quarter(X);
  quarter(Y);
  half(jx);
  half(jy);
  wide = (uint32_t)(Sd >> 61) | beyond_rho(r);
  if (SOON && (bad >= 32u || wide != 0u || quarter.broken() || half.broken())) return false;
  const Halves inv = halves(reciprocal_grid(r));
  const Halves hx = halves((int64_t)(2 * jx)), hy = halves((int64_t)(2 * jy));
  const int64_t ux = mul_grid<0>(hx, inv), uy = mul_grid<0>(hy, inv);  // 2^-60
  Within<59> slow;  // |u| < 1/2
  slow((uint64_t)ux);
  slow((uint64_t)uy);
  const Halves vx = halves(ux), vy = halves(uy);
  // rho u u in 2^-62: 2 j in 2^-62 times u in 2^-60 over 2^61
  const int64_t qxx = mul_grid<3>(hx, vx), qyy = mul_grid<3>(hy, vy), qxy = mul_grid<3>(hx, vy);
  const int64_t E = qxx + qyy;
  quarter((uint64_t)E);
  const int64_t ne = -(int64_t)(2 * X + Y) - 3 * E;
  int64_t De = mul_grid<0>(halves(ne), k.c[0]), Dp = mul_grid<0>(halves((int64_t)X + E), k.c[1]);
  int64_t Dx = mul_grid<0>(halves((int64_t)(2 * bx - d13)), k.c[2]);
  int64_t Dy = mul_grid<0>(halves((int64_t)(2 * by - d24)), k.c[2]);
  int64_t Dxx = mul_grid<0>(halves((int64_t)(s13 - s24) - qxx + qyy), k.c[3]);
  int64_t Dxy = mul_grid<0>(halves((int64_t)(s57 - s68) - qxy), k.c[3]);
  Dxx += Dxx;
  Dxy += Dxy;
  if (force) {
    // g steps times u in 2^-60
    const int64_t de = mul_grid<4>(vx, k.ge[0]) + mul_grid<4>(vy, k.ge[1]);
    De -= de;
    Dp += de;
    Dx += k.gq[0];
    Dy += k.gq[1];
    Dxx -= 2 * (mul_grid<4>(vx, k.gp[0]) - mul_grid<4>(vy, k.gp[1]));
    Dxy -= mul_grid<4>(vx, k.gp[1]) + mul_grid<4>(vy, k.gp[0]);
  }
  const uint64_t gx = (uint64_t)k.gj[0], gy = (uint64_t)k.gj[1];
  const uint64_t ie = (uint64_t)De, ip = (uint64_t)Dp, ix = (uint64_t)Dx, iy = (uint64_t)Dy;
  F[0] += 4 * (ie - ip);
  const uint64_t ax = ie + 2 * ip;                    // axis: + e + 2 epsilon
  const uint64_t tx = 2 * ix + gx, ty = 2 * iy + gy;  // 2 q - j (j's part is -g/6)
  const uint64_t px = ax - (uint64_t)Dxx, py = ax + (uint64_t)Dxx;
  F[1] += px + tx;
  F[3] += px - tx;
  F[2] += py + ty;
  F[4] += py - ty;
  const uint64_t dg = 2 * ie + ip;                    // diagonal: - 2 e - epsilon
  const uint64_t wx = gx - ix, wy = gy - iy;          // - j - q
  const uint64_t d0 = 0 - dg - (uint64_t)Dxy, d1 = (uint64_t)Dxy - dg;
  F[5] += d0 + (wx + wy);
  F[7] += d0 - (wx + wy);
  F[6] += d1 - (wx - wy);
  F[8] += d1 + (wx - wy);
  uint32_t out = 0;
#pragma unroll
  for (int i = 0; i < 9; ++i) f[i] = from_grid<true>(F[i], k.sc, out);
  m = NodeMom{r, ux, uy, 0};
  return bad < 32u && wide == 0u && !(quarter.broken() || half.broken() || slow.broken()) && (int32_t)out >= 0;
}

// D3Q19 BGK: f+_i = (1 - omega) f_i + omega feq_i + src_i.  In units of a
// diagonal direction's weight 1/36 the last two are integer combinations of
//   B = omega rho/36 - (T_xx + T_yy + T_zz)/3,
//   T_ab = (omega/8) rho u_a u_b + (pre/24)(g_a u_b + g_b u_a),
//   M_a = (omega/12) rho u_a + (pre/36) g_a       (pre = 3 (1 - omega/2)):
// rest 12 B; axis 2 (B + T_aa +- M_a); diagonal B + T_aa + T_bb +- 2 T_ab +-
// (M_a +- M_b).
template <bool SOON>
__device__ __forceinline__ bool collide_grid(double (&f)[19], const FixedK& k, bool force, NodeMom& m) {
  uint32_t bad = 0, wide = 0;
  uint64_t F[19];
  F[0] = to_grid<9>(f[0], k.sc, bad);
#pragma unroll
  for (int i = 1; i < 19; ++i) F[i] = i < 7 ? to_grid<7>(f[i], k.sc, bad) : to_grid<6>(f[i], k.sc, bad);
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
  if (force) {
    jx += (uint64_t)k.hg[0];
    jy += (uint64_t)k.hg[1];
    jz += (uint64_t)k.hg[2];
  }
  wide = beyond_rho(r);
  Within<61> half;  // |j| < 1/2
  half(jx);
  half(jy);
  half(jz);
  if (SOON && (bad >= 32u || wide != 0u || half.broken())) return false;
  const Halves inv = halves(reciprocal_grid(r));
  const Halves hx = halves((int64_t)(2 * jx)), hy = halves((int64_t)(2 * jy)), hz = halves((int64_t)(2 * jz));
  const int64_t ux = mul_grid<0>(hx, inv), uy = mul_grid<0>(hy, inv), uz = mul_grid<0>(hz, inv);  // 2^-60
  Within<59> slow;  // |u| < 1/2
  slow((uint64_t)ux);
  slow((uint64_t)uy);
  slow((uint64_t)uz);
  const Halves vx = halves(ux), vy = halves(uy), vz = halves(uz);
  // 2 (omega/8) j; T in 2^-62: that times u in 2^-60 over 2^61
  int64_t Wx = mul_grid<0>(hx, k.c[0]), Wy = mul_grid<0>(hy, k.c[0]), Wz = mul_grid<0>(hz, k.c[0]);
  const Halves gx = halves(Wx), gy = halves(Wy), gz = halves(Wz);
  int64_t Txx = mul_grid<3>(gx, vx), Tyy = mul_grid<3>(gy, vy), Tzz = mul_grid<3>(gz, vz);
  // 2 T_ab
  int64_t Sxy = 2 * mul_grid<3>(gx, vy), Sxz = 2 * mul_grid<3>(gx, vz), Syz = 2 * mul_grid<3>(gy, vz);
  // M_a: half of 2 j times 2 omega/12 over 2^64
  int64_t Mx = mul_grid<0>(hx, k.c[1]), My = mul_grid<0>(hy, k.c[1]), Mz = mul_grid<0>(hz, k.c[1]);
  if (force) {
    Txx += 2 * mul_grid<4>(vx, k.ge[0]);
    Tyy += 2 * mul_grid<4>(vy, k.ge[1]);
    Tzz += 2 * mul_grid<4>(vz, k.ge[2]);
    Sxy += 2 * (mul_grid<4>(vx, k.ge[1]) + mul_grid<4>(vy, k.ge[0]));
    Sxz += 2 * (mul_grid<4>(vx, k.ge[2]) + mul_grid<4>(vz, k.ge[0]));
    Syz += 2 * (mul_grid<4>(vy, k.ge[2]) + mul_grid<4>(vz, k.ge[1]));
  }
  const int64_t tr = Txx + Tyy + Tzz;
  Within<57> small;  // (omega/8) rho u.u below 2^-5
  small((uint64_t)tr);
  const uint64_t B = (uint64_t)(mul_grid<0>(halves((int64_t)r), k.c[2]) - mul_grid<0>(halves(tr), k.c[3]));
  uint32_t out = 0;
  auto put = [&](int i, uint64_t c) {
    // (1 - omega) F_i: |1 - omega| as oh 2^32 + ol over 2^63; F < 2^62
    const uint32_t fh = (uint32_t)(F[i] >> 32), fl = (uint32_t)F[i];
    const uint64_t mid = (uint64_t)fl * k.oh + k.oc + (uint64_t)fh * k.ol;
    const uint64_t R = (uint64_t)fh * k.oh2 + (mid >> 31);
    f[i] = from_grid<false>(c + (R ^ k.neg), k.sc, out);
  };
  auto pair = [&](int i, uint64_t P, uint64_t M) {
    put(i, P + M);
    put(i + 1, P - M);
  };
  put(0, 12 * B);
  // 2 M_a is what the products above hold (2 j in place of j)
  const uint64_t mx2 = (uint64_t)Mx + 2 * (uint64_t)k.gq[0], my2 = (uint64_t)My + 2 * (uint64_t)k.gq[1],
                 mz2 = (uint64_t)Mz + 2 * (uint64_t)k.gq[2];
  const uint64_t mx = (uint64_t)((int64_t)mx2 >> 1), my = (uint64_t)((int64_t)my2 >> 1),
                 mz = (uint64_t)((int64_t)mz2 >> 1);
  const uint64_t Bx = B + (uint64_t)Txx, By = B + (uint64_t)Tyy, Bz = B + (uint64_t)Tzz;
  pair(1, 2 * Bx, mx2);
  pair(3, 2 * By, my2);
  pair(5, 2 * Bz, mz2);
  const uint64_t Bxy = Bx + (uint64_t)Tyy, Bxz = Bx + (uint64_t)Tzz, Byz = By + (uint64_t)Tzz;
  pair(7, Bxy + (uint64_t)Sxy, mx + my);
  pair(9, Bxy - (uint64_t)Sxy, mx - my);
  pair(11, Bxz + (uint64_t)Sxz, mx + mz);
  pair(13, Bxz - (uint64_t)Sxz, mx - mz);
  pair(15, Byz + (uint64_t)Syz, my + mz);
  pair(17, Byz - (uint64_t)Syz, my - mz);
  m = NodeMom{r, ux, uy, uz};
  return bad < 32u && wide == 0u && !(half.broken() || slow.broken() || small.broken()) && (int32_t)out >= 0;
}

// v (|v| < 1/2, else `wide`) in 2^-60, toward zero.
__device__ __forceinline__ int64_t velocity_grid(double v, uint32_t& wide) {
  const uint32_t lo = (uint32_t)__double2loint(v), hi = (uint32_t)__double2hiint(v);
  const uint32_t e = (hi >> 20) & 0x7ffu;
  wide |= e > 1021u ? 1u : 0u;
  const uint32_t n = 1025u - e;  // places below the 63-bit significand; 0 and denormals vanish
  const uint64_t m = ((uint64_t)((__funnelshift_l(lo, hi, 10) & 0x3fffffffu) | 0x40000000u) << 32) | (lo << 10);
  const int64_t a = (int64_t)(n < 64u ? m >> n : 0ull), s = (int32_t)hi >> 31;
  return (a ^ s) - s;
}

// e . (x, y, z) for a direction given as integers in {-1, 0, 1}.
__device__ __forceinline__ int64_t dot_grid(const int (&e)[3], int64_t x, int64_t y, int64_t z) {
  auto term = [](int c, int64_t v) {
    const int64_t s = c >> 31, on = -(int64_t)(c & 1);
    return ((v ^ s) & on) - s;
  };
  return term(e[0], x) + term(e[1], y) + term(e[2], z);
}

// VIBB link value (Sec. 3.1) on the grid.  With t = rho_d/rho at x_f and x_ff,
// G = t f+_i' there, K(u) = 2 e.u + 3 (e.u)^2 - u.u and Delta the value at x_f
// minus that at x_ff, the rule's feq(rho_d, u_d) + fneq_d is
//   G_ff + 2 q Delta G + 3/2 w rho_d (K(u_d) - K(u_ff) - 2 q Delta K):
// the equilibria's rest parts cancel, and every difference is formed exactly.
// Eight FP64 operations (two reciprocals) in place of about 120, each of which
// holds the FP64 pipe for 64 clocks of a warp's quarter of an SM.
// wq: the link's velocity weights (cf, cff, cw) in 2^-62; diag: the
// direction's weight is 1/36.  False: outside the grid's range, val unset.
template <int SH, bool D3>
__device__ __forceinline__ bool vibb_grid(const int (&e)[3], bool diag, double q, const int64_t (&wq)[3], double fpf,
                                          double fpff, const double (&mf)[4], const double (&mff)[4], bool moving,
                                          const double (&uw)[3], double wall, int local_rho, const FixedK& k,
                                          double& val) {
  constexpr int D = D3 ? 3 : 2;
  uint32_t bad = 0, wide = 0;
  const uint64_t F = to_grid<SH>(fpf, k.sc, bad), FF = to_grid<SH>(fpff, k.sc, bad);
  const uint64_t R = to_grid<10>(mf[0], k.sc, bad), RR = to_grid<10>(mff[0], k.sc, bad);
  const uint64_t Q = to_grid<10>(q, 0, bad);
  const Halves hq = halves((int64_t)Q);
  const uint64_t dR = R - RR;
  Within<59> w59;
  Within<57> w57;
  wide = beyond_rho(R) | beyond_rho(RR);
  w59(dR);
  const uint64_t rd = local_rho && Q > (1ull << 61) ? R : RR + (uint64_t)mul_grid<3>(hq, halves((int64_t)dR));
  const Halves hd = halves((int64_t)rd);
  // t - 1 in 2^-59
  const int64_t tf = mul_grid<0>(hd, halves(reciprocal_grid(R))) - (1ll << 59);
  const int64_t tff = mul_grid<0>(hd, halves(reciprocal_grid(RR))) - (1ll << 59);
  w57((uint64_t)tf);
  w57((uint64_t)tff);
  const int64_t G = (int64_t)F + mul_grid<5>(halves((int64_t)F), halves(tf));
  const int64_t GG = (int64_t)FF + mul_grid<5>(halves((int64_t)FF), halves(tff));
  w59((uint64_t)(G - GG));
  int64_t v = GG + mul_grid<3>(hq, halves(G - GG));
  // K in 2^-59 of a velocity in 2^-60
  auto K = [&](const int64_t (&u)[3]) {
    const int64_t eu = dot_grid(e, u[0], u[1], u[2]);
    w59((uint64_t)eu);
    const Halves he = halves(eu);
    int64_t r = eu + 3 * mul_grid<3>(he, he);
#pragma unroll
    for (int a = 0; a < D; ++a) {
      const Halves h = halves(u[a]);
      r -= mul_grid<3>(h, h);
    }
    return r;
  };
  int64_t u[3] = {0, 0, 0}, uu[3] = {0, 0, 0}, ud[3] = {0, 0, 0};
  const Halves cf = halves(wq[0]), cff = halves(wq[1]), cw = halves(wq[2]);
#pragma unroll
  for (int a = 0; a < D; ++a) {
    u[a] = velocity_grid(mf[1 + a], wide);
    uu[a] = velocity_grid(mff[1 + a], wide);
    ud[a] = mul_grid<2>(cf, halves(u[a])) + mul_grid<2>(cff, halves(uu[a]));
    if (moving) ud[a] += mul_grid<2>(cw, halves(velocity_grid(uw[a], wide)));
    w59((uint64_t)ud[a]);
  }
  const int64_t Kf = K(u), Kff = K(uu), Kd = K(ud);
  w59((uint64_t)(Kf - Kff));
  const int64_t X = Kd - Kff - mul_grid<3>(hq, halves(Kf - Kff));
  w57((uint64_t)X);
  // 3/2 w in 2^-64: 1/24 (diagonal), 1/12 or 1/6 (axis)
  const Halves W = diag ? halves(0x0aaaaaaaaaaaaaabll) : (D3 ? halves(0x1555555555555555ll) : halves(0x2aaaaaaaaaaaaaabll));
  v += mul_grid<5>(halves(mul_grid<0>(hd, W)), halves(X));
  uint32_t out = 0;
  if (moving) {
    const double ws = wall / k.step;  // k.step is a power of two
    wide |= ((uint32_t)__double2hiint(ws) & 0x7fffffffu) >= 0x43b00000u ? 1u : 0u;
    v += __double2ll_rn(ws);
  }
  val = from_grid<true>((uint64_t)v, k.sc, out);
  return bad < 32u && wide == 0u && !(w59.broken() || w57.broken()) && (int32_t)out >= 0;
}

#endif  // __CUDACC__

}  // namespace lbm
