// CUDA kernels of the lattice-Boltzmann step with velocity-interpolation
// bounce-back (arXiv:1903.01111), templated on the velocity set (D2Q9,
// D3Q19) and the storage precision:
//   F64  -- populations f_i stored in double;
//   F32S -- populations stored in float as h_i = f_i - w_i rho0 ("shifted"),
//           so the O(1) rest part w_i rho0 never enters a float rounding.
//
// Storage (compacted): only fluid nodes, open-column nodes and ghost nodes
// (solid nodes that receive a link's missing population) are stored, in
// x-row order; k is the storage index, S their number.  SoA f[i*S + k].
// A fluid run (maximal x-run of fluid nodes in one row) has every node of
// its neighbour rows over [x0 - 1, x_end + 1] stored and contiguous, so one
// run record (the storage index of (x0, row') for each neighbour row)
// addresses every pull; pulls across the periodic x seam use the row's first
// and last storage index.  The buffer read by a step holds f+(t) of every
// fluid node; ghost slots are filled by the link kernel before the bulk
// kernel pulls them.
//
// Every state of a lattice with open columns (D2Q9) holds them filled, by the
// threads of the nodes beside them in the initialisation and in every step
// (open_ends), and by k_open after the caller sets the populations.
//
// Step t -> t+1, on one stream, in one of two forms.  Fused: D3Q19 k_fused
// stages each block's pulls in shared memory, evaluates the block's link rules
// into the staged slots and collides; D2Q9 k_inline does so for the groups of
// nodes that have links and pulls the others straight.  Split (the adjoint's
// recompute, FP64 D3Q19, D2Q9 lattices with links all over, and wherever the
// autotuner finds it faster):
//   k_links: per cut link (x_f, i'), the missing f_i(x_f, t+1), i = opp(i'),
//            from f+ and the moment cache at x_f and x_ff (Sec. 3 and 3.1),
//            written to the ghost slot f[i][k_s] (read only by x_f);
//            momentum exchange force in FP64.
//   k_bulk:  pull streaming f_i(x, t+1) = f+_i(x - e_i, t) (Eq. 1), moments,
//            Guo-forced BGK (Sec. 2, Eq. feq) -> f+(t+1) into the other
//            buffer; rho, u(t+1) into the moment cache where flagged.  Ghost
//            slots of the output get zeros (through the same store
//            instructions as the fluid slots) so that every written sector
//            is complete.  FP64 one-node shapes run k_bulk_list instead, over
//            the fluid nodes alone.
// FP64 collides and evaluates VIBB links in 64-bit integers (fixed64.cuh),
// FP32 D2Q9 BGK in packed pairs (pair32.cuh).
#pragma once
#include <cuda_runtime.h>

#include <cstdint>

#include "fixed64.cuh"
#include "lattice.cuh"
#include "pair32.cuh"

namespace lbm {

struct F64 {
  using T = double;
  static constexpr bool shifted = false;
};
struct F32S {
  using T = float;
  static constexpr bool shifted = true;
};

// One moment-cache record per node: (r, ux, uy, uz) with r = rho (F64) or
// rho - rho0 (F32S); 16 B (FP32) or 32 B (FP64), loaded in one piece.
template <class T>
struct __align__(4 * sizeof(T)) Mom4 {
  T r, ux, uy, uz;
};

// Per stored node word: run id of a fluid node and its cache flag, or the
// open / ghost bit.
constexpr uint32_t W_RUN = (1u << 29) - 1;
constexpr uint32_t W_CACHE = 1u << 29;
constexpr uint32_t W_OPEN = 1u << 30;
constexpr uint32_t W_GHOST = 1u << 31;

// One fluid run starting at x0 with storage index k0: xk = x0 - k0 (so that
// node k of the run sits at x = k + xk), its row (y, z), the domain the row
// belongs to, and for each neighbour row (slot order below) dbase = the
// storage index of (x0, row') minus k0 (so that the pull from (x + dx, row')
// is k + dbase + dx).  48 B.  D2Q9 has two neighbour rows; dbase[2] holds the
// run's open ends instead: bit 0 when it starts next to an open inlet node (at
// x = 1), bit 1 when it ends at x = dbase[2] >> 2 next to an open outlet node.
struct __align__(16) RunRec {
  int32_t xk, y, z, dom;
  int32_t dbase[8];
};

// Run parameters of one domain of a batch (several independent flows
// stacked along the last axis of one lattice, each with its own relaxation
// time, body force and inlet profile; the profiles are in Layout's row_uin).  A
// lattice of one domain reads Params.
struct DomPar {
  double omega, fpre3;    // 1/tau, 3 (1 - 1/(2 tau))
  double g[3];
  int32_t has_force;
  float omega_f, fpre3_f, g_f[3], hg_f[3], omega2_f;  // float copies, as in Params
  Folded kc;              // collision constants, as in Params
  FixedK kx;
};

// Collision parameters of one node, from Params or from its domain.
struct Relax {
  double omega, fpre3, g[3];
  int has_force;
  float omega_f, fpre3_f, g_f[3], hg_f[3], omega2_f;
};

// A run parameter in the storage precision: the double, or its float copy
// rounded on the host (the same value as a conversion on the device).
template <class T>
__host__ __device__ __forceinline__ T par(double d, float f) {
  if constexpr (sizeof(T) == sizeof(float))
    return f;
  else
    return d;
}

// Neighbour-row slots by source-row offset (dy, dz).  D2Q9: (1,0), (-1,0).
// D3Q19: (1,0), (-1,0), (0,1), (0,-1), (1,1), (-1,-1), (1,-1), (-1,1).
__host__ __device__ constexpr int row_slot(int dy, int dz) {
  return dz == 0 ? (dy > 0 ? 0 : 1)
                 : (dy == 0 ? (dz > 0 ? 2 : 3) : (dy == dz ? (dy > 0 ? 4 : 5) : (dy > 0 ? 6 : 7)));
}

struct Layout {
  int64_t S;                   // stored nodes, padded to a multiple of 32
  const uint32_t* word;        // [S]
  const int32_t* node_of;      // [S] dense node index
  const int32_t* tile;         // [ceil(N / MOM_TILE) + 1] first stored node of each tile of dense nodes
  const RunRec* runs;
  const int32_t* row_first;    // [ny*nz] storage index of the row's first stored node (-1: none)
  const int32_t* row_last;     // [ny*nz] ... last stored node
  const int32_t* row_in1;      // [ny*nz] storage index of the fluid node at x = 1 (open inlet rows), else -1
  const int32_t* row_out1;     // [ny*nz] ... at x = width - 2 (open outlet rows), else -1
  const DomPar* dom;           // [ndom] when ndom > 1, else null
  int32_t ndom;
  const uint32_t* fluid;       // [nfluid] storage indices of the fluid nodes (FP64 lattices), else null
  int64_t nfluid;
  const void* row_uin;         // [ny] inlet velocity of each row, storage precision (open inlet)
  const uint32_t* groups;      // D2Q9: 32-node groups with links (nlinked of them), then those without
  int64_t nlinked, ngroups;
  uint32_t ahead;              // nodes ahead that the step kernels prefetch into L2 (0: the state stays there)
};

__device__ __forceinline__ Relax relax_params(const Params& p) {
  return Relax{p.omega,   p.fpre3,   {p.g[0], p.g[1], p.g[2]},          p.has_force,
               p.omega_f, p.fpre3_f, {p.g_f[0], p.g_f[1], p.g_f[2]}, {p.hg_f[0], p.hg_f[1], p.hg_f[2]},
               p.omega2_f};
}

__device__ __forceinline__ Relax relax_domain(const DomPar* __restrict__ dp, int d) {
  const DomPar& q = dp[d];
  return Relax{q.omega,   q.fpre3,   {q.g[0], q.g[1], q.g[2]},          q.has_force,
               q.omega_f, q.fpre3_f, {q.g_f[0], q.g_f[1], q.g_f[2]}, {q.hg_f[0], q.hg_f[1], q.hg_f[2]},
               q.omega2_f};
}

// Relaxation of a node of fluid run `run` (any kernel but the bulk one,
// which resolves the single-domain case at compile time).
__device__ __forceinline__ Relax relax_of_run(const Params& p, const Layout& lay, uint32_t run) {
  return lay.ndom > 1 ? relax_domain(lay.dom, lay.runs[run].dom) : relax_params(p);
}

// One link: storage indices of x_f, x_ff (x_f if no second fluid node) and
// the ghost x_s; meta = dir | rule << 5 | (body + 1) << 7 (25 bits of body).
struct __align__(16) LinkRec {
  uint32_t kf, kff, ks, meta;
};

// --------------------------------------------------------------- helpers --

// Asks L2 for the populations of the N stored nodes from k (a multiple of 32)
// on, `ahead` nodes further, by threads t = 0, 1, ... of nt: one request per
// 128-byte line of a direction.  A block's pulls wait behind its node words and
// runs, so too few of them are in flight to keep HBM busy (D2Q9 FP32 60 %);
// brought into L2 a few microseconds early they wait a third as long.  ahead is
// about 6 MB of state: 8192 x 4096 D2Q9 FP32 468 us per step without, 413 / 402 /
// 399 / 407 at 1.4 / 2.8 / 5.6 / 11 MB; dense 301 x 257 x 259 506 -> 486, 526 at 24 MB
// (the far half of L2 is used up); 384^3 pack 1298 -> 1266.
template <int Q, class T>
__device__ __forceinline__ void prefetch_ahead(const T* f, const Layout& lay, uint64_t k, int N, int t,
                                               int nt) {
  constexpr int per = 128 / (int)sizeof(T);
  const uint64_t from = k + lay.ahead;
  if (lay.ahead == 0u || from + N > (uint64_t)lay.S) return;
  const int lines = N / per;
  for (int j = t; j < lines * Q; j += nt) {
    const int i = j / lines;
    asm volatile("prefetch.global.L2 [%0];" ::"l"(f + (uint64_t)i * lay.S + from + (uint64_t)(j - i * lines) * per));
  }
}

// Clears the force slot of the next step (the grid's first block).
template <int BT>
__device__ __forceinline__ void clear_force(double* force_next, int nbody) {
  if (force_next && blockIdx.x == 0)
    for (int t = threadIdx.x; t < 3 * nbody; t += BT) force_next[t] = 0.0;
}

// Programmatic dependent launch: a step kernel lets its successor start early,
// and the successor reads what no kernel writes (node words, runs, link records)
// before it waits for the predecessor's results.  On lattices that take
// microseconds a step the launch and those loads are a third of it.
//
// Bulk and fused kernels let it start once they have waited themselves, so that
// one successor at most is resident beside a kernel.  At the start of the kernel
// instead, the next five or six steps of a lattice of some 200 blocks take up
// their places at once, each where its predecessors left room, which piles a
// step's blocks onto a few SMs: 32^3 nodes FP32 4.5 us per step, 2.8 so; FP64 28^3
// 7.5 and 4.2.  k_inline and the link kernels, whose chain before the wait is
// longer, do it first (FP32 channel 600 x 500 5.2 us per step, 5.7 the other way).
//
// A kernel started so is resident while its predecessor still writes the
// populations, the moment cache and the multipliers it will read.  Such memory
// is not read-only for the kernel's lifetime, so it is loaded by plain loads
// after the wait, never by __ldg, and never through a __restrict__ pointer
// (which lets the compiler take a non-coherent load, or move a load above the
// wait): the wait makes the predecessor's writes visible to plain loads only.
// __ldg and const __restrict__ are kept for what the host alone writes, and
// __restrict__ for outputs of which a thread reads back no more than its own
// stores.
__device__ __forceinline__ void let_next_start() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void wait_for_previous() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

// Equilibrium of Eq. (feq), C = 1, in storage form: r is rho (F64) or
// rho - rho0 (F32S); rho is the full density.
template <class L, class P>
__device__ __forceinline__ typename P::T equilibrium(int i, typename P::T r, typename P::T rho, typename P::T ux,
                                                      typename P::T uy, typename P::T uz) {
  using T = typename P::T;
  const T eu = (T)L::cx(i) * ux + (T)L::cy(i) * uy + (T)L::cz(i) * uz;
  const T uu = ux * ux + uy * uy + uz * uz;
  const T w = (T)L::w(i);
  const T poly = (T)3 * eu + (T)4.5 * eu * eu - (T)1.5 * uu;
  if (P::shifted) return w * (r + rho * poly);
  return w * rho * ((T)1 + poly);
}

// Pull source coordinate x - c along one axis, with periodic wrap.
__device__ __forceinline__ int src_coord(int c, int x, int xm, int xp) { return c == 0 ? x : (c > 0 ? xm : xp); }

// Moments, collision and store of one fluid node.  f holds the pre-collision
// populations f(x, t+1) in storage form; n < 2^31.  keep == false (a ghost
// or open slot in the bulk pass): the same instructions store zeros and the
// moment cache is not written, so that a warp mixing fluid and ghost slots
// issues one store per direction instead of two divergent store sequences.
// Weight class of direction i: 0 rest, 1 |e| = 1, 2 diagonal.
template <class L>
__host__ __device__ constexpr int weight_class(int i) {
  return i == 0 ? 0 : (L::w(i) == L::w(1) ? 1 : 2);
}

// The node's collision constants folded on the host: the lattice's (Params)
// or its domain's (DomPar), both filled by fold.
template <bool MULTI>
__device__ __forceinline__ const Folded& folded_of(const Params& p, const Layout& lay, int dom) {
  if constexpr (MULTI)
    return lay.dom[dom].kc;
  else
    return p.kc;
}

template <bool MULTI>
__device__ __forceinline__ const FixedK& fixed_of(const Params& p, const Layout& lay, int dom) {
  if constexpr (MULTI)
    return lay.dom[dom].kx;
  else
    return p.kx;
}

// FP32 D2Q9 BGK parameters of one node from its run parameters and folded
// constants, and those of two nodes.
__device__ __forceinline__ Bgk32<float> bgk32_params(float rho0, const Relax& rx, const Folded& kc, bool force) {
  Bgk32<float> c;
  c.rho0 = rho0;
  c.om = rx.omega_f;
  if (force) {
    constexpr int dir[4] = {1, 2, 5, 6};
    c.hx = kc.hg_f[0];
    c.hy = kc.hg_f[1];
    c.gx = rx.g_f[0];
    c.gy = rx.g_f[1];
#pragma unroll
    for (int i = 0; i < 3; ++i) c.kf[i] = kc.kf_f[i];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      c.kt[i] = kc.kt_f[dir[i]];
      c.ke[i] = kc.ke_f[dir[i]];
    }
  }
  return c;
}
__device__ __forceinline__ Bgk32<F2> bgk32_pair(const Bgk32<float>& a, const Bgk32<float>& b, bool force) {
  Bgk32<F2> c;
  c.rho0 = pack2(a.rho0, b.rho0);
  c.om = pack2(a.om, b.om);
  if (force) {
    c.hx = pack2(a.hx, b.hx);
    c.hy = pack2(a.hy, b.hy);
    c.gx = pack2(a.gx, b.gx);
    c.gy = pack2(a.gy, b.gy);
#pragma unroll
    for (int i = 0; i < 3; ++i) c.kf[i] = pack2(a.kf[i], b.kf[i]);
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      c.kt[i] = pack2(a.kt[i], b.kt[i]);
      c.ke[i] = pack2(a.ke[i], b.ke[i]);
    }
  }
  return c;
}

// Collision and store of one node: moments of f, Guo-forced BGK (or D2Q9
// MRT) with the run parameters rx and the folded constants kc, the node's
// moment cache entry when flagged.
#define LBM_K(name) par<T>(kc.name, kc.name##_f)
#define LBM_KI(name, i) par<T>(kc.name[i], kc.name##_f[i])
template <class L, class P>
__device__ __forceinline__ void collide_store(typename P::T (&f)[L::Q], const Params& p, const Relax& rx,
                                              const Folded& kc,
                                              typename P::T* __restrict__ fout, size_t S, uint32_t n_,
                                              Mom4<typename P::T>* __restrict__ mom, bool cache, bool keep = true) {
  using T = typename P::T;
  if constexpr (P::shifted && L::Q == 9) {
    if (p.collision == 0) {
      const bool force = rx.has_force != 0;
      float r, ux, uy;
      bgk_d2q9(f, bgk32_params(p.rho0_f, rx, kc, force), force, r, ux, uy);
      if (cache && keep) mom[n_] = Mom4<float>{r, ux, uy, 0.f};
#pragma unroll
      for (int i = 0; i < 9; ++i) fout[(size_t)i * S + n_] = keep ? f[i] : 0.f;
      return;
    }
  }
  T r = 0, jx = 0, jy = 0, jz = 0;
  if constexpr (!P::shifted) {
    // FP64 (bound by the FP64 pipe, where every add, multiply or FMA takes
    // one issue slot): density and momentum from the sums and differences of
    // opposite directions, Q - 1 operations fewer than summing the
    // directions into each moment
    r = f[0];
#pragma unroll
    for (int i = 1; i < L::Q; ++i) {
      const int j = L::opp(i);
      if (j < i) continue;
      r += f[i] + f[j];
      const T d = f[i] - f[j];
      if (L::cx(i) > 0) jx += d;
      if (L::cx(i) < 0) jx -= d;
      if (L::cy(i) > 0) jy += d;
      if (L::cy(i) < 0) jy -= d;
      if (L::cz(i) > 0) jz += d;
      if (L::cz(i) < 0) jz -= d;
    }
  } else {
#pragma unroll
    for (int i = 0; i < L::Q; ++i) {
      r += f[i];
      if (L::cx(i) > 0) jx += f[i];
      if (L::cx(i) < 0) jx -= f[i];
      if (L::cy(i) > 0) jy += f[i];
      if (L::cy(i) < 0) jy -= f[i];
      if (L::cz(i) > 0) jz += f[i];
      if (L::cz(i) < 0) jz -= f[i];
    }
  }
  const T rho = P::shifted ? par<T>(p.rho0, p.rho0_f) + r : r;
  const T gx = par<T>(rx.g[0], rx.g_f[0]), gy = par<T>(rx.g[1], rx.g_f[1]), gz = par<T>(rx.g[2], rx.g_f[2]);
  const T inv = (T)1 / rho;
  // Guo forcing: velocity shifted by half the body force
  const T hx = LBM_KI(hg, 0), hy = LBM_KI(hg, 1), hz = LBM_KI(hg, 2);
  const T ux = (jx + hx) * inv, uy = (jy + hy) * inv, uz = (jz + hz) * inv;
  if (cache && keep) mom[n_] = Mom4<T>{r, ux, uy, L::D == 3 ? uz : (T)0};
  const T omega = par<T>(rx.omega, rx.omega_f);
  const T uu15 = (T)1.5 * (ux * ux + uy * uy + uz * uz);
  if constexpr (L::Q == 9) {
    if (p.collision == 1) {
      // MRT (Sec. 2, Eq. mrt) on the non-equilibrium part n = f - feq, whose
      // moments are m - meq (meq = M feq, the moments of the BGK
      // equilibrium); Guo source in moment space scaled by (1 - s_k/2).
      const T gx_ = gx, gy_ = gy;
      const T ug2 = ux * gx_ + uy * gy_;
      T n[9], src[9];
#pragma unroll
      for (int i = 0; i < 9; ++i) {
        const T eu = (T)L::cx(i) * ux + (T)L::cy(i) * uy;
        const T w = (T)L::w(i);
        const T poly = (T)3 * eu + (T)4.5 * eu * eu - uu15;
        const T feq = P::shifted ? w * (r + rho * poly) : (w * rho) * ((T)1 + poly);
        n[i] = f[i] - feq;
        const T eg = (T)L::cx(i) * gx_ + (T)L::cy(i) * gy_;
        src[i] = rx.has_force ? w * ((T)3 * (eg - ug2) + (T)9 * eu * eg) : (T)0;
      }
      T dm[9];
#pragma unroll
      for (int k = 0; k < 9; ++k) {
        T mn = 0, ms = 0;
#pragma unroll
        for (int i = 0; i < 9; ++i) {
          if (mrt_m(k, i) != 0) {
            mn += (T)mrt_m(k, i) * n[i];
            ms += (T)mrt_m(k, i) * src[i];
          }
        }
        const T sk = (k == 7 || k == 8) ? omega : (T)((k == 0 || k == 3 || k == 5) ? 0.3 : (k == 1 || k == 2) ? 1.5 : 1.2);
        dm[k] = (sk * mn - ((T)1 - (T)0.5 * sk) * ms) / (T)mrt_norm2(k);
      }
#pragma unroll
      for (int i = 0; i < 9; ++i) {
        T d = 0;
#pragma unroll
        for (int k = 0; k < 9; ++k)
          if (mrt_m(k, i) != 0) d += (T)mrt_m(k, i) * dm[k];
        fout[(size_t)i * S + n_] = keep ? f[i] - d : (T)0;
      }
      return;
    }
  }
  // BGK with the Guo source (1 - 1/(2 tau)) w_i [3 (e_i - u).g + 9 (e_i.u)(e_i.g)]
  //   = 3 (1 - 1/(2 tau)) w_i [(e_i.g)(1 + 3 e_i.u) - u.g].
  const T ug = rx.has_force ? ux * gx + uy * gy + uz * gz : (T)0;
  if constexpr (P::shifted) {
    // Shifted FP32 storage: each direction keeps its own equilibrium
    // feq_i = w (r + rho poly_i) and relaxes in the difference form
    // f + omega (feq - f), so that rounding falls on the small
    // non-equilibrium part; opposite directions (i, j = opp(i), e_j = -e_i)
    // share e.u, the symmetric part 4.5 (e.u)^2 - 1.5 u.u of the polynomial
    // and the two parts of the source, Sc +- So with Sc = kt_i (e_i.u) -
    // kf_c (u.g) and So = ke_i from the folded constants.  (Relaxing the
    // pair's symmetric and antisymmetric parts separately, as FP64 does,
    // measured 5x larger FP32 errors in drag and in the adjoint's dJ/dtau.)
    T sc[3] = {0, 0, 0};
    if (rx.has_force) {
#pragma unroll
      for (int c = 0; c < 3; ++c) sc[c] = LBM_KI(kf, c) * ug;
    }
#pragma unroll
    for (int i = 0; i < L::Q; ++i) {
      const int j = L::opp(i);
      if (i != 0 && j < i) continue;
      const T eu = (T)L::cx(i) * ux + (T)L::cy(i) * uy + (T)L::cz(i) * uz;
      const T w = (T)L::w(i);
      const T sym = (T)4.5 * eu * eu - uu15;
      const T feqi = w * (r + rho * (sym + (T)3 * eu));
      T oi = f[i] + omega * (feqi - f[i]);
      T Sc = 0, So = 0;
      if (rx.has_force) {
        Sc = LBM_KI(kt, i) * eu - sc[weight_class<L>(i)];
        So = LBM_KI(ke, i);
        oi += Sc + So;
      }
      fout[(size_t)i * S + n_] = keep ? oi : (T)0;
      if (i != 0) {
        const T feqj = w * (r + rho * (sym - (T)3 * eu));
        T oj = f[j] + omega * (feqj - f[j]);
        if (rx.has_force) oj += Sc - So;
        fout[(size_t)j * S + n_] = keep ? oj : (T)0;
      }
    }
  } else {
    // FP64 (bound by the FP64 pipe, where every add, multiply or FMA takes
    // one issue slot): per pair of opposite directions (i, j = opp(i)),
    // e_j = -e_i turns the equilibria into A +- B and the sources into
    // Sc +- So, so that with the folded constants
    //   a_c = ko_c rho (1 - 1.5 u.u) - kf_c (u.g),  h_c = kh_c rho,  b_c = kb_c rho,
    //   P = (h_c eu + kt_i) eu + a_c = omega A + Sc,  M = b_c eu + ke_i = omega B + So,
    //   f+_i,j = (1 - omega) f_i,j + (P +- M):
    // the source's symmetric part joins the FMAs of the equilibrium's, its
    // antisymmetric part the FMA of M, and a pair costs an FMA and a multiply
    // for P, an FMA for M and two adds and two FMAs for the outputs.
    const T om1 = LBM_K(om1);
    const T c0 = (T)1 - uu15;
    {
      const T out = om1 * f[0] + ((LBM_KI(ko, 0) * rho) * c0 - LBM_KI(kf, 0) * ug);
      fout[n_] = keep ? out : (T)0;
    }
    T a[3], h[3], b[3];
#pragma unroll
    for (int c = 1; c < 3; ++c) {
      a[c] = (LBM_KI(ko, c) * rho) * c0 - LBM_KI(kf, c) * ug;
      h[c] = LBM_KI(kh, c) * rho;
      b[c] = LBM_KI(kb, c) * rho;
    }
#pragma unroll
    for (int i = 1; i < L::Q; ++i) {
      const int j = L::opp(i);
      if (j < i) continue;
      const int c = weight_class<L>(i);
      const T eu = (T)L::cx(i) * ux + (T)L::cy(i) * uy + (T)L::cz(i) * uz;
      const T Pv = (h[c] * eu + LBM_KI(kt, i)) * eu + a[c];
      const T Mv = b[c] * eu + LBM_KI(ke, i);
      fout[(size_t)i * S + n_] = keep ? om1 * f[i] + (Pv + Mv) : (T)0;
      fout[(size_t)j * S + n_] = keep ? om1 * f[j] + (Pv - Mv) : (T)0;
    }
  }
}

#undef LBM_K
#undef LBM_KI

// Collision and store of one node in the step kernels (SOON: see fixed64.cuh).  FP64 collides on the
// integer grid (fixed64.cuh) and, where a kept node is outside its range,
// takes the populations again (again(f) fills f as it was) and collides in
// doubles.
template <class L, class P, bool MULTI, bool SOON, class Again>
__device__ __forceinline__ void collide_node(typename P::T (&f)[L::Q], const Params& p, const Layout& lay, int dom,
                                             typename P::T* __restrict__ fout, size_t S, uint32_t k,
                                             Mom4<typename P::T>* __restrict__ mom, bool cache, bool keep,
                                             Again&& again) {
  const Relax rx = MULTI ? relax_domain(lay.dom, dom) : relax_params(p);
  if constexpr (!P::shifted) {
    const FixedK& kx = fixed_of<MULTI>(p, lay, dom);
    if (kx.on) {
      NodeMom m;
      // (a slot that is not kept stores zeros whatever comes out)
      if (collide_grid<SOON>(f, kx, rx.has_force != 0, m) || !keep) {
        if (cache && keep) mom[k] = Mom4<double>{(double)m.r * kx.step, m.u(m.ux), m.u(m.uy), m.u(m.uz)};
#pragma unroll
        for (int i = 0; i < L::Q; ++i) fout[(size_t)i * S + k] = keep ? f[i] : 0.0;
        return;
      }
      again(f);
    }
  }
  collide_store<L, P>(f, p, rx, folded_of<MULTI>(p, lay, dom), fout, S, k, mom, cache, keep);
}

// Storage indices of the pull sources x - e_i of fluid node k of run `run`.
template <class L>
__device__ __forceinline__ void pull_sources(uint32_t k, const RunRec& run, const Layout& lay, const Params& p,
                                             uint32_t (&src)[L::Q]) {
  const int nx = p.nx;
  const int x = (int)k + run.xk;
  const bool left = x == 0, right = x == nx - 1;
#pragma unroll
  for (int i = 0; i < L::Q; ++i) {
    // source x - e_i: offsets (dx, dy, dz) = -(cx, cy, cz)
    const int dx = -L::cx(i), dy = -L::cy(i), dz = -L::cz(i);
    if (dy == 0 && dz == 0) {
      if (dx == 0) {
        src[i] = k;
      } else if ((dx < 0 && left) || (dx > 0 && right)) {
        const int row = run.y + p.ny * run.z;
        src[i] = (uint32_t)(dx < 0 ? lay.row_last[row] : lay.row_first[row]);
      } else {
        src[i] = k + dx;
      }
    } else {
      if ((dx < 0 && left) || (dx > 0 && right)) {
        int yy = run.y + dy, zz = run.z + dz;
        yy = yy < 0 ? yy + p.ny : (yy >= p.ny ? yy - p.ny : yy);
        zz = zz < 0 ? zz + p.nz : (zz >= p.nz ? zz - p.nz : zz);
        const int row = yy + p.ny * zz;
        src[i] = (uint32_t)(dx < 0 ? lay.row_last[row] : lay.row_first[row]);
      } else {
        src[i] = (uint32_t)((int)k + run.dbase[row_slot(dy, dz)] + dx);
      }
    }
  }
}

// Offsets src_i - k of the pull sources of fluid node k (run `run`): away
// from the periodic x seam every offset is a per-run constant (dx in the
// node's own row, base - k0 + dx in a neighbour row); at the seam (x = 0 or
// nx - 1 of a periodic row) they come from pull_sources.
template <class L>
__device__ __forceinline__ void pull_offsets(uint32_t k, const RunRec& run, const Layout& lay, const Params& p,
                                             int (&d)[L::Q]) {
  const int x = (int)k + run.xk;
  if (x > 0 && x < p.nx - 1) {
#pragma unroll
    for (int i = 0; i < L::Q; ++i) {
      const int dx = -L::cx(i), dy = -L::cy(i), dz = -L::cz(i);
      d[i] = (dy == 0 && dz == 0) ? dx : run.dbase[row_slot(dy, dz)] + dx;
    }
    return;
  }
  uint32_t src[L::Q];
  pull_sources<L>(k, run, lay, p, src);
#pragma unroll
  for (int i = 0; i < L::Q; ++i) d[i] = (int)(src[i] - k);
}

// The populations f_i(x, t+1) = f+_i(x - e_i, t) of fluid node k of run `run`.
template <class L, class T>
__device__ __forceinline__ void pull_node(const T* fin, size_t S, uint32_t k, const RunRec& run,
                                          const Layout& lay, const Params& p, T (&f)[L::Q]) {
  int d[L::Q];
  pull_offsets<L>(k, run, lay, p, d);
  const T* fk = fin + k;
#pragma unroll
  for (int i = 0; i < L::Q; ++i) f[i] = fk[(ptrdiff_t)i * (ptrdiff_t)S + d[i]];
}

// ------------------------------------------------------------ open sides --

// Sec. 4.3: inlet column x = 0 (storage k0) by non-equilibrium extrapolation
// from x = 1 with the parabolic velocity u_in(y) = 4 u_max (y - y0)(y1 - y)/
// (y1 - y0)^2 (tabulated on the host: in doubles per step it took 30 FP64
// instructions of a warp); f and mom hold the state of the fluid node at x = 1,
// adjacent in storage.
template <class L, class P>
__device__ __forceinline__ void fill_inlet(typename P::T* f, const Mom4<typename P::T>* mom,
                                           size_t S, uint32_t k0, int y, const Layout& lay, const Params& p) {
  using T = typename P::T;
  const T uin = ((const T*)lay.row_uin)[y];
  const uint32_t k1 = k0 + 1;
  const Mom4<T> m1 = mom[k1];
  const T rho1 = P::shifted ? par<T>(p.rho0, p.rho0_f) + m1.r : m1.r;
  T v[L::Q];
#pragma unroll
  for (int i = 0; i < L::Q; ++i) v[i] = f[i * S + k1];
#pragma unroll
  for (int i = 0; i < L::Q; ++i)
    f[i * S + k0] = equilibrium<L, P>(i, m1.r, rho1, uin, (T)0, (T)0) +
                    (v[i] - equilibrium<L, P>(i, m1.r, rho1, m1.ux, m1.uy, (T)0));
}

// Outlet column (storage kl): a copy of the fluid node before it.
template <class L, class P>
__device__ __forceinline__ void fill_outlet(typename P::T* f, size_t S, uint32_t kl) {
  typename P::T v[L::Q];
#pragma unroll
  for (int i = 0; i < L::Q; ++i) v[i] = f[i * S + kl - 1];
#pragma unroll
  for (int i = 0; i < L::Q; ++i) f[i * S + kl] = v[i];
}

// The open columns of a state (f, mom), one thread per row and side (D2Q9):
// the open node is the first (inlet) or last (outlet) stored node of its row.
// Every state of a lattice with open columns holds them filled: by this kernel
// after the caller sets the populations, else by open_ends.
template <class L, class P>
__global__ void k_open(typename P::T* __restrict__ f, const Mom4<typename P::T>* __restrict__ mom, Layout lay,
                       Params p) {
  // threads 0 .. ny-1: inlet rows; ny .. 2 ny - 1: outlet rows
  const int t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= 2 * p.ny) return;
  const size_t S = (size_t)lay.S;
  if (t < p.ny) {
    const int32_t k0 = lay.row_first[t];
    if (p.inlet && k0 >= 0 && (lay.word[k0] & W_OPEN)) fill_inlet<L, P>(f, mom, S, (uint32_t)k0, t, lay, p);
  } else {
    const int32_t kl = lay.row_last[t - p.ny];
    if (p.outlet && kl >= 0 && (lay.word[kl] & W_OPEN)) fill_outlet<L, P>(f, S, (uint32_t)kl);
  }
}

// The open node beside fluid node k of run `run`, written by k's thread after
// it stored k's state: the open columns of the next step cost no launch.  The
// open slots' own threads store nothing.
template <class L, class P>
__device__ __forceinline__ void open_ends(typename P::T* f, const Mom4<typename P::T>* mom,
                                          size_t S, uint32_t k, const RunRec& run, const Layout& lay,
                                          const Params& p) {
  if constexpr (L::D == 2) {
    if (!(p.inlet | p.outlet) || run.dbase[2] == 0) return;
    const int x = (int)k + run.xk;
    if ((run.dbase[2] & 1) && x == 1) fill_inlet<L, P>(f, mom, S, k - 1, run.y, lay, p);
    if ((run.dbase[2] & 2) && x == (run.dbase[2] >> 2)) fill_outlet<L, P>(f, S, k + 1);
  }
}

// ------------------------------------------------------------------ bulk --

// Shapes of the bulk kernel the autotuner chooses from: threads per block,
// nodes per thread in parallel (a thread with two nodes takes k and
// k + ceil(S/2), both ranges coalesced, and has 2Q loads in flight) and nodes
// per thread in sequence (a thread walks k, k + G, k + 2G, ... over the grid
// G and loads the next node's word and run while the current node's pulls
// are in flight).  Two nodes per thread and the sequential walk are built
// for D2Q9 only (D3Q19 threads already have 19 loads in flight).
struct BulkShape {
  int threads, npt, seq;
};
constexpr BulkShape kBulkShapes[] = {{256, 1, 1}, {128, 1, 1}, {512, 1, 1}, {256, 2, 1},
                                     {128, 2, 1}, {512, 2, 1}, {128, 1, 4}, {128, 1, 8}};
constexpr int kNumBulkShapes = 8;

template <class L>
constexpr int bulk_max_npt() {
  return L::Q == 9 ? 2 : 1;
}

// Shapes built for a stencil, one bit per shape.
template <class L>
constexpr unsigned bulk_shape_mask() {
  return L::Q == 9 ? 0xffu : 0x07u;
}

// Default shape, 128-thread blocks: two neighbouring nodes per thread for FP32
// D2Q9 (8192 x 4096 nodes 382 us per step, 388 in 256-thread blocks, 408 with
// one node per thread); one node per thread for D3Q19 (the fused step's best
// block: 1.26 ms per step on a 384^3 pack against 1.33 at 256) and for FP64 D2Q9 (integer collision: 280 us per step on 4097 x 2049 nodes against
// 339 with two nodes per thread, whose registers halve the warps in flight).
template <class L, class P>
constexpr int bulk_default_shape() {
  return L::Q == 9 && P::shifted ? 4 : 1;
}

// Resident blocks per SM a shape is compiled for, from a register budget per
// 256 threads: FP32 D2Q9 6 blocks with one node per thread (40 registers) and
// 4 with two; FP32 D3Q19 5 (48 registers).  Measured: one block more spills
// (D3Q19) or runs slower (D2Q9 two nodes); one fewer leaves too few loads in
// flight.  FP64 (integer collision: bound by instruction issue, 56 % busy at
// 2 blocks, so warps to switch between count): D3Q19 3 blocks (80 registers;
// 192^3 nodes 452 us per step; 521 at 2 without spills, 560 at 4), D2Q9 4 (64
// registers; 4097 x 2049 nodes 280 us; 399 at 2, 321 at 3, 277 at 4.5).
template <class L, class P, int BT, int NPT>
constexpr int bulk_blocks_per_sm() {
  constexpr int base = !P::shifted ? (NPT == 1 ? (L::Q == 9 ? 4 : 3) : 2) : (L::Q == 9 ? (NPT == 1 ? 6 : 4) : 5);
  return base * 256 / BT < 1 ? 1 : base * 256 / BT;
}

// Pull, collision and store of NPT nodes k of a thread, all their pulls issued
// before the first collision.  MULTI: the lattice holds several domains; each
// node's collision reads its run's domain parameters.  ALONE: in a bulk kernel,
// not in k_inline (which has let the next start, and does without SOON).
template <class L, class P, bool MULTI, int NPT, bool ALONE>
__device__ __forceinline__ void bulk_nodes(const uint32_t (&k)[NPT], const bool (&live)[NPT],
                                           const typename P::T* fin, typename P::T* __restrict__ fout,
                                           const Layout& lay, Mom4<typename P::T>* __restrict__ mom, const Params& p) {
  using T = typename P::T;
  const size_t S = (size_t)lay.S;
  uint32_t w[NPT];
  int dom[NPT];
  T f[NPT][L::Q];
#pragma unroll
  for (int j = 0; j < NPT; ++j) w[j] = live[j] ? __ldg(lay.word + k[j]) : W_GHOST;
  if constexpr (NPT == 1) {
    RunRec run{};
    if (live[0] && !(w[0] & (W_GHOST | W_OPEN))) run = lay.runs[w[0] & W_RUN];
    dom[0] = run.dom;
    wait_for_previous();
    if (ALONE) let_next_start();
    if (live[0] && !(w[0] & (W_GHOST | W_OPEN))) pull_node<L>(fin, S, k[0], run, lay, p, f[0]);
  } else {
    wait_for_previous();
    if (ALONE) let_next_start();
#pragma unroll
    for (int j = 0; j < NPT; ++j) {
      dom[j] = 0;
      if (live[j] && !(w[j] & (W_GHOST | W_OPEN))) {
        const RunRec run = lay.runs[w[j] & W_RUN];
        if (MULTI) dom[j] = run.dom;
        pull_node<L>(fin, S, k[j], run, lay, p, f[j]);
      }
    }
  }
#pragma unroll
  for (int j = 0; j < NPT; ++j) {
    if (!live[j] || (w[j] & W_OPEN)) continue;
    // ghost slots: zeros through the same stores (inputs at rest)
    const bool fl = !(w[j] & W_GHOST);
    if (!fl) {
#pragma unroll
      for (int i = 0; i < L::Q; ++i) f[j][i] = P::shifted ? (T)0 : (T)L::w(i);
    }
    collide_node<L, P, MULTI, ALONE>(f[j], p, lay, dom[j], fout, S, k[j], mom, (w[j] & W_CACHE) != 0, fl, [&](T(&g)[L::Q]) {
      pull_node<L>(fin, S, k[j], lay.runs[w[j] & W_RUN], lay, p, g);
    });
    if (L::D == 2 && fl && (p.inlet | p.outlet)) open_ends<L, P>(fout, mom, S, k[j], lay.runs[w[j] & W_RUN], lay, p);
  }
}

// The neighbouring nodes k (even) and k + 1 of one thread, FP32 D2Q9 BGK (see
// pair32.cuh): their words, and the runs of those that are fluid.
struct PairNodes {
  uint2 w;
  RunRec ra, rb;
  __device__ __forceinline__ bool fa() const { return !(w.x & (W_GHOST | W_OPEN)); }
  __device__ __forceinline__ bool fb() const { return !(w.y & (W_GHOST | W_OPEN)); }
  __device__ __forceinline__ bool same() const { return fa() && fb() && ((w.x ^ w.y) & W_RUN) == 0; }
};
__device__ __forceinline__ PairNodes pair_nodes(uint32_t k, bool live, const Layout& lay) {
  PairNodes n{};
  n.w = live ? __ldg((const uint2*)(lay.word + k)) : make_uint2(W_GHOST, W_GHOST);
  if (n.fa()) n.ra = lay.runs[n.w.x & W_RUN];
  if (n.same())
    n.rb = n.ra;
  else if (n.fb())
    n.rb = lay.runs[n.w.y & W_RUN];
  return n;
}

// Their pulls.  Inside one fluid run, away from the periodic seam, the second
// node's sources are those of the first moved by one; any other pair gathers
// its nodes one by one.
__device__ __forceinline__ void pair_pull(uint32_t k, const PairNodes& n, const float* fin,
                                          const Layout& lay, const Params& p, F2 (&f)[9]) {
  using L = D2Q9;
  const size_t S = (size_t)lay.S;
  const int x = (int)k + n.ra.xk;
  if (n.same() && x > 0 && x + 1 < p.nx - 1) {
    const float* fk = fin + k;
    const float2 own = *(const float2*)fk;
    f[0] = pack2(own.x, own.y);
#pragma unroll
    for (int i = 1; i < 9; ++i) {
      const int dx = -L::cx(i), dy = -L::cy(i);
      const float* s =
          fk + ((ptrdiff_t)i * (ptrdiff_t)S + (dy == 0 ? dx : n.ra.dbase[row_slot(dy, 0)] + dx));
      f[i] = pack2(s[0], s[1]);
    }
  } else {
    float a[9] = {0}, b[9] = {0};
    if (n.fa()) pull_node<L>(fin, S, k, n.ra, lay, p, a);
    if (n.fb()) pull_node<L>(fin, S, k + 1, n.rb, lay, p, b);
#pragma unroll
    for (int i = 0; i < 9; ++i) f[i] = pack2(a[i], b[i]);
  }
}

// Their collision and store.
template <bool MULTI>
__device__ __forceinline__ void pair_finish(uint32_t k, bool live, const PairNodes& n, F2 (&f)[9],
                                            float* __restrict__ fout, const Layout& lay,
                                            Mom4<float>* __restrict__ mom, const Params& p) {
  const size_t S = (size_t)lay.S;
  const bool fa = n.fa(), fb = n.fb();
  const int da = n.ra.dom, db = n.rb.dom;
  const Relax xa = MULTI ? relax_domain(lay.dom, da) : relax_params(p);
  bool force = xa.has_force != 0;
  Bgk32<float> ca, cb;
  if (MULTI && da != db) {
    const Relax xb = relax_domain(lay.dom, db);
    force = force || xb.has_force != 0;
    ca = bgk32_params(p.rho0_f, xa, folded_of<MULTI>(p, lay, da), force);
    cb = bgk32_params(p.rho0_f, xb, folded_of<MULTI>(p, lay, db), force);
  } else {
    ca = cb = bgk32_params(p.rho0_f, xa, folded_of<MULTI>(p, lay, da), force);
  }
  F2 r, ux, uy;
  bgk_d2q9(f, bgk32_pair(ca, cb, force), force, r, ux, uy);
  if ((n.w.x & W_CACHE) && fa) mom[k] = Mom4<float>{low(r), low(ux), low(uy), 0.f};
  if ((n.w.y & W_CACHE) && fb) mom[k + 1] = Mom4<float>{high(r), high(ux), high(uy), 0.f};
  float* __restrict__ ok = fout + k;
  if (fa && fb) {
    // (stored as floats: open_ends reads them back as such)
#pragma unroll
    for (int i = 0; i < 9; ++i) *(float2*)(ok + (size_t)i * S) = make_float2(low(f[i]), high(f[i]));
  } else if (live) {
    // ghost slots take zeros (whole sectors), open slots their neighbour's thread
#pragma unroll
    for (int i = 0; i < 9; ++i) {
      if (!(n.w.x & W_OPEN)) ok[(size_t)i * S] = fa ? low(f[i]) : 0.f;
      if (!(n.w.y & W_OPEN)) ok[(size_t)i * S + 1] = fb ? high(f[i]) : 0.f;
    }
  }
  if (p.inlet | p.outlet) {
    if (fa) open_ends<D2Q9, F32S>(fout, mom, S, k, n.ra, lay, p);
    if (fb) open_ends<D2Q9, F32S>(fout, mom, S, k + 1, n.rb, lay, p);
  }
}

template <bool MULTI, bool ALONE>
__device__ __forceinline__ void bulk_pair(uint32_t k, bool live, const float* fin,
                                          float* __restrict__ fout, const Layout& lay, Mom4<float>* __restrict__ mom,
                                          const Params& p) {
  const PairNodes n = pair_nodes(k, live, lay);
  wait_for_previous();
  if (ALONE) let_next_start();
  F2 f[9];
  pair_pull(k, n, fin, lay, p, f);
  pair_finish<MULTI>(k, live, n, f, fout, lay, mom, p);
}

// Block (0) also clears the force slot of the next step.
template <class L, class P, bool MULTI, int BT, int NPT>
__global__ void __launch_bounds__(BT, (bulk_blocks_per_sm<L, P, BT, NPT>())) k_bulk(const typename P::T* fin,
                                                                       typename P::T* __restrict__ fout, Layout lay,
                                                                       Mom4<typename P::T>* __restrict__ mom,
                                                                       double* force_next, Params p) {
  const uint32_t t = blockIdx.x * BT + threadIdx.x;
  if constexpr (NPT == 2 && P::shifted && L::Q == 9) {
    if (p.collision == 0) {
      prefetch_ahead<L::Q>(fin, lay, 2ull * blockIdx.x * BT, 2 * BT, threadIdx.x, BT);
      bulk_pair<MULTI, true>(2 * t, 2ull * t < (uint64_t)lay.S, fin, fout, lay, mom, p);
      clear_force<BT>(force_next, p.nbody);
      return;
    }
  }
  const uint32_t stride = (uint32_t)(((size_t)lay.S + NPT - 1) / NPT);
  uint32_t k[NPT];
  bool live[NPT];
#pragma unroll
  for (int j = 0; j < NPT; ++j) {
    k[j] = t + (uint32_t)j * stride;
    live[j] = t < stride && (uint64_t)k[j] < (uint64_t)lay.S;
    prefetch_ahead<L::Q>(fin, lay, (uint64_t)blockIdx.x * BT + (uint64_t)j * (stride / 32 * 32), BT, threadIdx.x, BT);
  }
  bulk_nodes<L, P, MULTI, NPT, true>(k, live, fin, fout, lay, mom, p);
  clear_force<BT>(force_next, p.nbody);
}

// FP64 bulk pass over the fluid nodes alone, one thread per entry of the
// layout's fluid list, otherwise as k_bulk.  An FP64 warp instruction holds
// the FP64 pipe for the same time whatever its active lanes, so the ghost
// and open slots that k_bulk's warps carry (23 % of a porous pack's storage)
// cost as much as fluid nodes there; this pass has no such lanes.  It leaves
// the ghost and open slots of the output unwritten: a ghost slot is read
// only in its link's direction after the link kernel of the next step has
// written it, and the fluid node beside an open slot writes it.
template <class L, class P, bool MULTI, int BT>
__global__ void __launch_bounds__(BT, (bulk_blocks_per_sm<L, P, BT, 1>())) k_bulk_list(
    const typename P::T* fin, typename P::T* __restrict__ fout, Layout lay,
    Mom4<typename P::T>* __restrict__ mom, double* force_next, Params p) {
  using T = typename P::T;
  const int64_t t = (int64_t)blockIdx.x * BT + threadIdx.x;
  const size_t S = (size_t)lay.S;
  const bool live = t < lay.nfluid;
  const uint32_t k = live ? __ldg(lay.fluid + t) : 0u;
  const uint32_t w = live ? __ldg(lay.word + k) : 0u;
  RunRec run{};
  if (live) run = lay.runs[w & W_RUN];
  wait_for_previous();
  let_next_start();
  clear_force<BT>(force_next, p.nbody);
  if (!live) return;
  // (the block's nodes lie at its share of the storage)
  prefetch_ahead<L::Q>(fin, lay, (uint64_t)k / 32 * 32 - (threadIdx.x & ~31u), BT, threadIdx.x, BT);
  T f[L::Q];
  pull_node<L>(fin, S, k, run, lay, p, f);
  collide_node<L, P, MULTI, true>(f, p, lay, run.dom, fout, S, k, mom, (w & W_CACHE) != 0, true, [&](T(&g)[L::Q]) {
    pull_node<L>(fin, S, k, lay.runs[w & W_RUN], lay, p, g);
  });
  if (L::D == 2 && (p.inlet | p.outlet)) open_ends<L, P>(fout, mom, S, k, lay.runs[w & W_RUN], lay, p);
}

// Resident blocks per SM of the sequential walk (it keeps the next node's
// word and run live): 4 per 256 threads in FP32 (64 registers, no spill;
// at 40 registers the spills cost more than the prefetch wins), 2 in FP64.
template <class P, int BT>
constexpr int bulk_seq_blocks_per_sm() {
  return (P::shifted ? 4 : 2) * 256 / BT;
}

// The fields of a run record that the pull offsets use away from the seam.
template <class L>
struct RunLite {
  int32_t xk, dom;
  int32_t dbase[L::D == 2 ? 2 : 8];
};

template <class L, bool MULTI>
__device__ __forceinline__ RunLite<L> load_run_lite(const RunRec* __restrict__ runs, uint32_t r) {
  RunLite<L> v;
  v.xk = runs[r].xk;
  v.dom = MULTI ? runs[r].dom : 0;
#pragma unroll
  for (int sl = 0; sl < (L::D == 2 ? 2 : 8); ++sl) v.dbase[sl] = runs[r].dbase[sl];
  return v;
}

// Sequential walk over the grid: the word of the node after next is loaded
// while the current node's pulls are in flight, and the next node's run
// record right after the current node's stores (D2Q9).
template <class L, class P, bool MULTI, int BT, int SEQ>
__global__ void __launch_bounds__(BT, (bulk_seq_blocks_per_sm<P, BT>())) k_bulk_seq(
    const typename P::T* fin, typename P::T* __restrict__ fout, Layout lay,
    Mom4<typename P::T>* __restrict__ mom, double* force_next, Params p) {
  using T = typename P::T;
  const size_t S = (size_t)lay.S;
  const uint32_t G = gridDim.x * BT;
  uint32_t k = blockIdx.x * BT + threadIdx.x;
  uint32_t w = k < S ? __ldg(lay.word + k) : W_GHOST;
  RunLite<L> run{};
  if (!(w & (W_GHOST | W_OPEN))) run = load_run_lite<L, MULTI>(lay.runs, w & W_RUN);
  uint32_t w2 = ((uint64_t)k + G < S) ? __ldg(lay.word + k + G) : W_GHOST;
  wait_for_previous();
  let_next_start();
  clear_force<BT>(force_next, p.nbody);
#pragma unroll 1
  for (int it = 0; it < SEQ && (uint64_t)k < S; ++it, k += G) {
    T f[L::Q];
    const bool fluid = !(w & (W_GHOST | W_OPEN));
    if (fluid) {
      int d[L::Q];
      const int x = (int)k + run.xk;
      if (x > 0 && x < p.nx - 1) {
#pragma unroll
        for (int i = 0; i < L::Q; ++i) {
          const int dx = -L::cx(i), dy = -L::cy(i), dz = -L::cz(i);
          d[i] = (dy == 0 && dz == 0) ? dx : run.dbase[row_slot(dy, dz)] + dx;
        }
      } else {
        pull_offsets<L>(k, lay.runs[w & W_RUN], lay, p, d);
      }
      const T* fk = fin + k;
#pragma unroll
      for (int i = 0; i < L::Q; ++i) f[i] = fk[(ptrdiff_t)i * (ptrdiff_t)S + d[i]];
    }
    const uint32_t w3 = ((uint64_t)k + 2ull * G < S) ? __ldg(lay.word + k + 2 * G) : W_GHOST;
    // (a separate zero-store branch here: the walk serves dense lattices,
    // where selecting zeros in every store measured about 2 % slower)
    if (w & W_GHOST) {
#pragma unroll
      for (int i = 0; i < L::Q; ++i) fout[(size_t)i * S + k] = (T)0;
    } else if (fluid) {
      collide_node<L, P, MULTI, true>(f, p, lay, run.dom, fout, S, k, mom, (w & W_CACHE) != 0, true, [&](T(&g)[L::Q]) {
        pull_node<L>(fin, S, k, lay.runs[w & W_RUN], lay, p, g);
      });
      if (p.inlet | p.outlet) open_ends<L, P>(fout, mom, S, k, lay.runs[w & W_RUN], lay, p);
    }
    // the next node's run record, loaded before its pulls are needed
    w = w2;
    if ((uint64_t)k + G < S && !(w & (W_GHOST | W_OPEN))) run = load_run_lite<L, MULTI>(lay.runs, w & W_RUN);
    w2 = w3;
  }
}

// ----------------------------------------------------------------- links --

// Per-direction data of the link kernel, staged in shared memory so that
// lanes holding different directions read it without serialisation.
template <class T, int Q>
struct DirTable {
  int opp[Q];
  T w[Q];
  T e[Q][3];
  int ie[sizeof(T) == 8 ? Q : 1][3];  // the same as integers (FP64)
};

// A direction as values (read from the table); for FP64 as integers too (a
// conversion costs as much as an addition).
template <class T>
struct DirVal {
  T wt, ex, ey, ez;
  __device__ __forceinline__ T w() const { return wt; }
  __device__ __forceinline__ T dot(T x, T y, T z) const { return ex * x + ey * y + ez * z; }
};
template <>
struct DirVal<double> {
  double wt, ex, ey, ez;
  int e[3];
  __device__ __forceinline__ double w() const { return wt; }
  __device__ __forceinline__ double dot(double x, double y, double z) const { return ex * x + ey * y + ez * z; }
};
// Equilibrium of direction `dir` (storage form, see above).
template <class P, class Dir>
__device__ __forceinline__ typename P::T eq_dir(const Dir& dir, typename P::T r, typename P::T rho, typename P::T ux,
                                                typename P::T uy, typename P::T uz) {
  using T = typename P::T;
  const T w = dir.w();
  const T eu = dir.dot(ux, uy, uz);
  const T poly = (T)3 * eu + (T)4.5 * eu * eu - (T)1.5 * (ux * ux + uy * uy + uz * uz);
  return P::shifted ? w * (r + rho * poly) : w * rho * ((T)1 + poly);
}

// Missing population f_i(x_f, t+1) of one link in storage form (see the
// rule list below).  fpf = f+_i'(x_f), fpff = f+_i'(x_ff), fpi = f+_i(x_f)
// (only read by the rule that needs it, through the callbacks' values);
// mf, mff: moments at time t at x_f and x_ff; dir: i'.
template <class P, class Dir>
__device__ __forceinline__ typename P::T link_value(int rule, typename P::T q, const Dir& dir, typename P::T fpf,
                                                    typename P::T fpff, typename P::T fpi, const Mom4<typename P::T>& mf,
                                                    const Mom4<typename P::T>& mff, typename P::T uw0,
                                                    typename P::T uw1, typename P::T uw2, typename P::T rho0,
                                                    int local_rho, bool moving = true) {
  using T = typename P::T;
  // 6 w_i' rho0 (e_i . u_w) with e_i = -e_i'.  FP64 skips it when no wall
  // of the lattice moves (the same for every link of a launch: five FP64
  // instructions of about a hundred per link); FP32 forms it always (the
  // branch moved registers of the fused kernel into spills and cost 2 %)
  const T wall = (P::shifted || moving) ? -(T)6 * dir.w() * rho0 * dir.dot(uw0, uw1, uw2) : (T)0;
  const T two_q = (T)2 * q;
  if (rule == 0) return fpf + wall;
  if (rule == 1) {
    if (q <= (T)0.5) return two_q * fpf + ((T)1 - two_q) * fpff + wall;
    const T inv2q = (T)1 / two_q;
    return (fpf + wall) * inv2q + (two_q - (T)1) * inv2q * fpi;
  }
  if (rule == 3) {
    // Yu: the population reaching the wall, linear between x_f and x_ff at
    // q - 1 along e_i', bounced back; then x_f linear between x_w (at q)
    // and x_ff (at -1), whose f_i(x_ff, t+1) is f+_i(x_f, t) in pull form
    const T i1q = (T)1 / ((T)1 + q);
    return (q * fpf + ((T)1 - q) * fpff + wall) * i1q + q * i1q * fpi;
  }
  const T rhof = P::shifted ? rho0 + mf.r : mf.r;
  const T rhoff = P::shifted ? rho0 + mff.r : mff.r;
  // Eq. (rhod) in storage form; optionally rho_d = rho_f when q > 1/2
  const T rd = (local_rho && q > (T)0.5) ? mf.r : two_q * mf.r + ((T)1 - two_q) * mff.r;
  const T rhod = P::shifted ? rho0 + rd : rd;
  const T neq_f = fpf - eq_dir<P>(dir, mf.r, rhof, mf.ux, mf.uy, mf.uz);
  const T neq_ff = fpff - eq_dir<P>(dir, mff.r, rhoff, mff.ux, mff.uy, mff.uz);
  // every quotient of the rule from one reciprocal, r = 1/(rho_f rho_ff D)
  // with D = q (1 + q) (q > 1/2) or 1 + q: 1/(rho_f rho_ff) = D r,
  // 1/D = rho_f rho_ff r, 1/(1 + q) and 1/q from 1/D
  const bool far = q > (T)0.5;
  const T D = far ? q * ((T)1 + q) : (T)1 + q;
  const T rr = rhof * rhoff;
  const T r = (T)1 / (rr * D);
  const T iD = rr * r;
  const T i1q = far ? q * iD : iD;
  // fneq at d, each term rescaled by its density ratio
  const T nd = rhod * (two_q * neq_f * rhoff + ((T)1 - two_q) * neq_ff * rhof) * (D * r);
  // u*_d (piecewise linear), u**_d (between x_ff and the wall), weighted 1/3 : 2/3
  T af, aff, aw;
  if (!far) {
    af = two_q;
    aff = (T)1 - two_q;
    aw = 0;
  } else {
    const T iq = ((T)1 + q) * iD;
    af = ((T)1 - q) * iq;
    aff = 0;
    aw = (two_q - (T)1) * iq;
  }
  const T bff = ((T)1 - q) * i1q, bw = two_q * i1q;
  const T third = (T)(1.0 / 3.0), two_thirds = (T)(2.0 / 3.0);
  const T cf = third * af, cff = third * aff + two_thirds * bff, cw = third * aw + two_thirds * bw;
  const T udx = cf * mf.ux + cff * mff.ux + cw * uw0;
  const T udy = cf * mf.uy + cff * mff.uy + cw * uw1;
  const T udz = cf * mf.uz + cff * mff.uz + cw * uw2;
  return eq_dir<P>(dir, rd, rhod, udx, udy, udz) + nd + wall;
}

// Direction table of the link kernels in shared memory (filled by the
// block's first Q threads; the caller synchronises).
template <class L, class T>
__device__ __forceinline__ void fill_dir_table(DirTable<T, L::Q>& tab) {
  if (threadIdx.x < L::Q) {
    const int d = threadIdx.x;
    tab.opp[d] = L::opp(d);
    tab.w[d] = (T)L::w(d);
    tab.e[d][0] = (T)L::cx(d);
    tab.e[d][1] = (T)L::cy(d);
    tab.e[d][2] = (T)L::cz(d);
    if constexpr (sizeof(T) == 8) {
      tab.ie[d][0] = L::cx(d);
      tab.ie[d][1] = L::cy(d);
      tab.ie[d][2] = L::cz(d);
    }
  }
}

// Missing population f_i(x_f, t+1) of the link (x_f = node, i' = ip, opposite
// i, as values dir) from the post-collision state (storage form, [Q][N]) and
// the moment cache at time t; x_ff = ff (x_f when there is no second fluid
// node).  fpf receives f+_i'(x_f, t), the link's other term of the momentum
// exchange.  Each rule loads only what it reads.  FP64 VIBB runs on the
// integer grid with the link's velocity weights wq[0], wq[nl], wq[2 nl] (in
// 2^-62; q alone fixes them), in doubles where that says no.
template <class L, class P>
__device__ __forceinline__ typename P::T eval_link(const DirVal<typename P::T>& dir, int ip, int i,
                                                   const typename P::T* f, const Mom4<typename P::T>* mom, size_t N, int rule,
                                                   typename P::T q, uint32_t node, uint32_t ff, typename P::T uw0,
                                                   typename P::T uw1, typename P::T uw2, const Params& p,
                                                   typename P::T& fpf, bool moving, const int64_t* __restrict__ wq,
                                                   int64_t nl) {
  using T = typename P::T;
  fpf = f[(size_t)ip * N + node];
  T fpff = 0, fpi = 0;
  Mom4<T> mf{0, 0, 0, 0}, mff{0, 0, 0, 0};
  if (rule == 1) {
    if (q <= (T)0.5)
      fpff = f[(size_t)ip * N + ff];
    else
      fpi = f[(size_t)i * N + node];
  } else if (rule == 2) {
    fpff = f[(size_t)ip * N + ff];
    mf = mom[node];
    mff = mom[ff];
  } else if (rule == 3) {
    fpff = f[(size_t)ip * N + ff];
    fpi = f[(size_t)i * N + node];
  }
  if constexpr (!P::shifted) {
    // (whatever the lattice's force: a domain alone and in a batch alike)
    if (rule == 2 && p.kx.grid) {
      const int64_t c[3] = {wq[0], wq[nl], moving ? wq[2 * nl] : 0};
      const double m0[4] = {mf.r, mf.ux, mf.uy, mf.uz}, m1[4] = {mff.r, mff.ux, mff.uy, mff.uz};
      const double uw[3] = {uw0, uw1, uw2};
      const double wall = moving ? -6.0 * dir.w() * p.rho0 * dir.dot(uw0, uw1, uw2) : 0.0;
      double val;
      if (vibb_grid<(L::D == 2 ? 8 : 7), L::D == 3>(dir.e, ip >= (L::D == 2 ? 5 : 7), q, c, fpf, fpff, m0, m1, moving, uw,
                                                    wall, p.vibb_local_rho, p.kx, val))
        return val;
    }
  }
  return link_value<P>(rule, q, dir, fpf, fpff, fpi, mf, mff, uw0, uw1, uw2, par<T>(p.rho0, p.rho0_f),
                       p.vibb_local_rho, moving);
}

// Direction ip from the table.
template <class T, int Q>
__device__ __forceinline__ DirVal<T> dir_of(const DirTable<T, Q>& tab, int ip) {
  if constexpr (sizeof(T) == 8)
    return DirVal<T>{tab.w[ip], tab.e[ip][0], tab.e[ip][1], tab.e[ip][2], {tab.ie[ip][0], tab.ie[ip][1], tab.ie[ip][2]}};
  else
    return DirVal<T>{tab.w[ip], tab.e[ip][0], tab.e[ip][1], tab.e[ip][2]};
}

// The link's momentum exchange (f+_i'(x_f,t) + f_i(x_f,t+1)) e_i' without its
// part at rest, 2 w_i' rho0, a geometric constant of the body that the host
// adds in FP64: the sums stay as small as the force (over a closed body the
// rest parts cancel, but not their roundings).  Shifted storage leaves it out
// by itself.
template <class P>
__device__ __forceinline__ typename P::T exchange(typename P::T fpf, typename P::T val, const DirVal<typename P::T>& dir,
                                                  const Params& p) {
  if constexpr (P::shifted) return fpf + val;
  const double c = dir.w() * p.rho0;
  return (fpf - c) + (val - c);
}

// A link's momentum exchange t e added to its body's slot by FP64 atomics.
template <class T>
__device__ __forceinline__ void add_force(double* force, int body, T t, const DirVal<T>& dir) {
  atomicAdd(&force[3 * body + 0], (double)(t * dir.ex));
  atomicAdd(&force[3 * body + 1], (double)(t * dir.ey));
  if (dir.ez != (T)0) atomicAdd(&force[3 * body + 2], (double)(t * dir.ez));
}

// As add_force for the lanes that are here, one atomic per body and component
// (out of line and by values, so that the usual case keeps its registers).
static __device__ __noinline__ void add_force_together(double* force, int body, double t, int ex, int ey, int ez) {
  const unsigned m = __match_any_sync(__activemask(), body);
  const int lane = threadIdx.x & 31;
  double v[3] = {t * ex, t * ey, t * ez};
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    if (m == 0xffffffffu) {
      for (int o = 16; o > 0; o >>= 1) v[a] += __shfl_down_sync(m, v[a], o);
    } else {
      double sum = 0.0;
      for (unsigned r = m; r; r &= r - 1) sum += __shfl_sync(m, v[a], __ffs(r) - 1);
      v[a] = sum;
    }
    if (lane == __ffs(m) - 1) atomicAdd(&force[3 * body + a], v[a]);
  }
}

// Sum of the momentum exchange t e over at most LINKS links of one body in a
// warp.  FP32 adds in FP32; FP64 adds integers in steps of 2^(sc - 57) (a warp's
// reduction of doubles is 15 FP64 instructions), each |t| below 2^(sc + room), so
// that no sum reaches 2^63 steps.  Any other t (the link kernel, a link a lane: a
// density beyond about 9 rho0; 576 links: more than about rho0/4 from rho0; a value
// that is not a number) goes to `far`, which adds it to the body's slot.  128^3
// pack, collisions and links in doubles: 504 us per step at 2 rho0 and 549 at
// 40 rho0; 1214 and 4120 with an atomic per link, 578 with everything in doubles.
template <class T, int LINKS>
struct LinkForce {
  T F[3] = {0, 0, 0};
  template <class Far>
  __device__ __forceinline__ void add(T t, const DirVal<T>& dir, const FixedK&, Far&&) {
    F[0] += t * dir.ex;
    F[1] += t * dir.ey;
    F[2] += t * dir.ez;
  }
  __device__ __forceinline__ void reduce() {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1)
#pragma unroll
      for (int a = 0; a < 3; ++a) F[a] += __shfl_down_sync(0xffffffffu, F[a], o);
  }
  __device__ __forceinline__ double value(int a, const FixedK&) const { return (double)F[a]; }
};
template <int LINKS>
struct LinkForce<double, LINKS> {
  static constexpr int room = LINKS <= 32 ? 1 : (LINKS <= 128 ? -1 : (LINKS <= 256 ? -2 : -4));
  static_assert(LINKS <= 1024, "64-bit sums");
  int64_t F[3] = {0, 0, 0};
  template <class Far>
  __device__ __forceinline__ void add(double t, const DirVal<double>& dir, const FixedK& k, Far&& far) {
    const uint32_t hi = (uint32_t)__double2hiint(t), e = (hi >> 20) & 0x7ffu;
    if (k.grid == 0 || e >= (uint32_t)(1023 + room + k.sc)) return far();
    // t 2^(57 - sc) by its exponent (a t too small for that is none of a step)
    const bool tiny = (int)e < 900 + k.sc || e == 0u;
    const int64_t v = __double2ll_rn(
        __hiloint2double((int)(hi + ((uint32_t)(57 - k.sc) << 20)), __double2loint(t)));
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      const int64_t s = dir.e[a] >> 31, on = tiny ? 0 : -(int64_t)(dir.e[a] & 1);
      F[a] += ((v ^ s) & on) - (s & on);
    }
  }
  __device__ __forceinline__ void reduce() {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1)
#pragma unroll
      for (int a = 0; a < 3; ++a) F[a] += __shfl_down_sync(0xffffffffu, F[a], o);
  }
  __device__ __forceinline__ double value(int a, const FixedK& k) const { return (double)F[a] * (k.step * 32.0); }
};

// One thread per link.  recs: storage indices and metadata; qv: q in
// storage precision; uw: [D][nl] wall velocities or null.  force: the step's
// accumulator slot [MAX_BODIES][3] (FP64).
//
// Rules (storage form; the rest part w rho0 cancels because every rule's
// weights sum to one):
//   half-way  f_i = f+_i'(x_f) + wall
//   Bouzidi   q <= 1/2: 2q f+_i'(x_f) + (1-2q) f+_i'(x_ff) + wall   (Eq. q_less)
//             q >  1/2: (f+_i'(x_f) + wall)/(2q) + (2q-1)/(2q) f+_i(x_f)  (Eq. q_larger)
//   VIBB      feq_i'(rho_d, u_d) + fneq_i'(x_d) + wall                 (Sec. 3.1)
//   Yu        (q f+_i'(x_f) + (1-q) f+_i'(x_ff) + wall)/(1+q) + q/(1+q) f+_i(x_f)  (Sec. 3)
// with wall = 6 w rho0 (e_i . u_w).
template <class L, class P, int SEQ>
__global__ void __launch_bounds__(256, (P::shifted ? 2 : 3)) k_links(typename P::T* f, const Mom4<typename P::T>* mom,
                                               const LinkRec* __restrict__ recs, const typename P::T* __restrict__ qv,
                                               const typename P::T* __restrict__ uwv,
                                               const int64_t* __restrict__ wqv, int64_t nl,
                                               double* force, Params p, int64_t S_) {
  using T = typename P::T;
  let_next_start();
  __shared__ DirTable<T, L::Q> tab;
  fill_dir_table<L>(tab);
  __syncthreads();
  // the block takes SEQ rounds of blockDim consecutive links; the next
  // round's record and q are loaded while the current link is processed
  const int64_t base = (int64_t)blockIdx.x * blockDim.x * SEQ;
  // body of the block's first link: the block's links of that body are
  // summed per lane (storage precision), per warp and per block (FP64);
  // links of any other body (a body boundary inside the block) add their
  // terms with FP64 atomics directly
  const int b0 = (int)(__ldg(&recs[base].meta) >> 7) - 1;
  const size_t N = (size_t)S_;
  LinkForce<T, 32 * SEQ> F;
  int64_t k = base + threadIdx.x;
  bool live = k < nl;
  LinkRec rec{0, 0, 0, 0};
  T q = 0;
  if (live) {
    rec = recs[k];
    q = qv[k];
  }
  wait_for_previous();
#pragma unroll 1
  for (int r = 0; r < SEQ; ++r) {
    const int64_t kn = k + blockDim.x;
    const bool liven = (r + 1 < SEQ) && kn < nl;
    LinkRec recn{0, 0, 0, 0};
    T qn = 0;
    if (liven) {
      recn = recs[kn];
      qn = qv[kn];
    }
    if (live) {
      const int ip = (int)(rec.meta & 31);
      const int rule = (int)((rec.meta >> 5) & 3);
      const int body = (int)(rec.meta >> 7) - 1;
      T uw0 = 0, uw1 = 0, uw2 = 0;
      if (uwv) {
        uw0 = uwv[k];
        uw1 = uwv[nl + k];
        if (L::D == 3) uw2 = uwv[2 * nl + k];
      }
      T fpf;
      const T val = eval_link<L, P>(dir_of(tab, ip), ip, tab.opp[ip], f, mom, N, rule, q, rec.kf, rec.kff, uw0, uw1,
                                    uw2, p, fpf, uwv != nullptr, wqv + k, nl);
      f[(size_t)tab.opp[ip] * N + rec.ks] = val;
      if (body >= 0) {
        const DirVal<T> dir = dir_of(tab, ip);
        const T t = exchange<P>(fpf, val, dir, p);
        auto far = [&] {
          if constexpr (!P::shifted) add_force_together(force, body, t, dir.e[0], dir.e[1], dir.e[2]);
        };
        if (body == b0)
          F.add(t, dir, p.kx, far);
        else
          add_force(force, body, t, dir);
      }
    }
    k = kn;
    rec = recn;
    q = qn;
    live = liven;
  }
  if (b0 < 0) return;
  __shared__ double red[3][32];
  F.reduce();
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  if (lane == 0)
    for (int a = 0; a < 3; ++a) red[a][warp] = F.value(a, p.kx);
  __syncthreads();
  if (threadIdx.x < 3) {
    const int nw = (blockDim.x + 31) >> 5;
    double acc = 0.0;
    for (int wi = 0; wi < nw; ++wi) acc += red[threadIdx.x][wi];
    atomicAdd(&force[3 * b0 + threadIdx.x], acc);
  }
}

// ------------------------------------------------------------ fused step --

// Links of the fused step kernel, in (node, direction) order: the links of
// the stored nodes 32 g .. 32 g + 31 are first[g] .. first[g+1] - 1, and
// mask[k] has bit d set when stored node k has a link in direction d.  One
// 16-B record per link: the storage indices of x_f and x_ff (x_f when there
// is no second fluid node), meta = dir | rule << 5 | (body + 1) << 8, and
// q as FP32 bits (FP32 storage; FP64 keeps q in qd).
struct __align__(16) FusedRec {
  uint32_t kf, kff, meta, q32;
};

template <class T>
struct FusedLinks {
  const int32_t* first;    // [ngroups + 1]
  const uint32_t* mask;    // [S]
  const FusedRec* rec;     // [nl]
  const double* qd;        // [nl] (FP64 storage) or null
  const T* uw;             // [D][nl] wall velocities or null
  const int64_t* wq;       // [3][nl] VIBB velocity weights in 2^-62 (FP64 storage) or null
  int64_t nl;
  int64_t ngroups;         // ceil(S / 32)
};

// Asynchronous global -> shared copies of one real (cp.async, cached in L1;
// no register holds the value while it is in flight).
template <class T>
__device__ __forceinline__ void cp_async_real(T* smem, const T* gmem) {
  const unsigned s = (unsigned)__cvta_generic_to_shared(smem);
  if constexpr (sizeof(T) == 8)
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8;\n" ::"r"(s), "l"(gmem) : "memory");
  else
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;\n" ::"r"(s), "l"(gmem) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;\n" ::: "memory"); }
__device__ __forceinline__ void cp_async_wait_all() { asm volatile("cp.async.wait_all;\n" ::: "memory"); }

// Resident blocks per SM of the step kernels with links, per 256 threads: FP32
// D2Q9 4 (64 registers: the link phase spills at the bulk kernel's 40), FP32
// D3Q19 5 (48), FP64 2 (128; k_fused, 128^3 pack: 214 us per step, 217 and 225 with
// room for 5 and 6 blocks of 128 threads).
template <class L, class P, int BT>
constexpr int fused_blocks_per_sm() {
  constexpr int base = !P::shifted ? 2 : (L::Q == 9 ? 4 : 5);
  return base * 256 / BT < 1 ? 1 : base * 256 / BT;
}

// One time step with the link rules fused into the pull pass, one thread
// per stored node (as k_bulk):
//  1. each fluid node issues the pulls of its non-link directions as
//     asynchronous copies into its column of the block's shared-memory
//     stage (ghost and open slots put the rest state there);
//  2. meanwhile the block evaluates the cut links of its nodes, spread over
//     all its threads (the same rule code as k_links, on f+(t) and the
//     moment cache at t, mom_in), and writes each link value into the
//     stage at its node and direction i = opp(i');
//  3. after one barrier every node collides from its staged column.
// The link values never go through HBM and no ghost slot is read or written
// by the link rules; ghost and open slots of fout get zeros as in k_bulk.
// The moments at t+1 go to mom_out (a second cache buffer: other blocks'
// link phases still read mom_in).  Momentum exchange: per thread in storage
// precision, per warp by shuffles, per block in FP64 and one atomic per
// block and component for the body of the block's first link; links of
// other bodies add their terms with FP64 atomics directly.
template <class L, class P, bool MULTI, int BT>
__global__ void __launch_bounds__(BT, (fused_blocks_per_sm<L, P, BT>())) k_fused(
    const typename P::T* fin, typename P::T* __restrict__ fout, Layout lay,
    FusedLinks<typename P::T> fl, const Mom4<typename P::T>* mom_in,
    Mom4<typename P::T>* __restrict__ mom_out, double* force, double* force_next,
    Params p) {
  using T = typename P::T;
  constexpr int NW = BT / 32;
  __shared__ T stage[NW][L::Q][32];
  __shared__ DirTable<T, L::Q> tab;
  __shared__ double red[3][NW];
  fill_dir_table<L>(tab);
  // (waits before the link records: held back behind them it cost 2 %)
  wait_for_previous();
  let_next_start();
  clear_force<BT>(force_next, p.nbody);
  __syncthreads();  // the direction table (every thread arrives here at once)
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const uint32_t base = blockIdx.x * BT;
  const uint32_t k = base + threadIdx.x;
  const size_t S = (size_t)lay.S;
  const bool live = (uint64_t)k < S;
  const uint32_t w = live ? __ldg(lay.word + k) : W_GHOST;
  const uint32_t mask = live ? __ldg(fl.mask + k) : 0u;
  prefetch_ahead<L::Q>(fin, lay, base, BT, threadIdx.x, BT);
  // the block's range of the link list (the same two words in every thread)
  const int64_t g0 = base >> 5, g1 = g0 + NW < fl.ngroups ? g0 + NW : fl.ngroups;
  const int64_t l0 = __ldg(fl.first + g0), l1 = __ldg(fl.first + g1);
  const int total = (int)(l1 - l0);
  // this thread's first link record, requested before the run record and
  // the pulls so that the link phase does not wait behind them
  FusedRec r_first{0, 0, 0, 0};
  T q_first = 0;
  if ((int)threadIdx.x < total) {
    r_first = fl.rec[l0 + threadIdx.x];
    q_first = P::shifted ? (T)__uint_as_float(r_first.q32) : (T)__ldg(fl.qd + l0 + threadIdx.x);
  }
  const bool fluid = live && !(w & (W_GHOST | W_OPEN));
  T(&col)[L::Q][32] = stage[warp];
  int dom = 0;
  if (fluid) {
    const RunRec run = lay.runs[w & W_RUN];
    if (MULTI) dom = run.dom;
    int d[L::Q];
    pull_offsets<L>(k, run, lay, p, d);
    const T* fk = fin + k;
#pragma unroll
    for (int i = 0; i < L::Q; ++i)
      // direction i comes from the solid side when its opposite is a link
      if (!((mask >> L::opp(i)) & 1u)) cp_async_real(&col[i][lane], fk + ((ptrdiff_t)i * (ptrdiff_t)S + d[i]));
  } else if (live && !P::shifted) {
    // ghost slots store zeros whatever their column holds; FP64 puts the rest
    // state there, which its integer collision takes
#pragma unroll
    for (int i = 0; i < L::Q; ++i) col[i][lane] = (T)L::w(i);
  }
  cp_async_commit();
  const int wb = total > 0 ? (int)(__ldg(&fl.rec[l0].meta) >> 8) - 1 : -1;
  LinkForce<T, 32 * (L::Q - 1)> F;
  for (int j = threadIdx.x; j < total; j += BT) {
    const int64_t li = l0 + j;
    const bool first_round = j == (int)threadIdx.x;
    const FusedRec r = first_round ? r_first : fl.rec[li];
    const T q = first_round ? q_first : (P::shifted ? (T)__uint_as_float(r.q32) : (T)__ldg(fl.qd + li));
    const int ip = (int)(r.meta & 31);
    const int rule = (int)((r.meta >> 5) & 7);
    const int body = (int)(r.meta >> 8) - 1;
    T uw0 = 0, uw1 = 0, uw2 = 0;
    if (fl.uw) {
      uw0 = fl.uw[li];
      uw1 = fl.uw[fl.nl + li];
      if (L::D == 3) uw2 = fl.uw[2 * fl.nl + li];
    }
    T fpf;
    const T val = eval_link<L, P>(dir_of(tab, ip), ip, tab.opp[ip], fin, mom_in, S, rule, q, r.kf, r.kff, uw0, uw1,
                                  uw2, p, fpf, fl.uw != nullptr, fl.wq + li, fl.nl);
    const uint32_t o = r.kf - base;  // the node's place in the block
    stage[o >> 5][tab.opp[ip]][o & 31] = val;
    if (body >= 0) {
      // momentum exchange as in k_links
      const DirVal<T> dir = dir_of(tab, ip);
      const T t = exchange<P>(fpf, val, dir, p);
      auto far = [&] {
        if constexpr (!P::shifted) add_force_together(force, body, t, dir.e[0], dir.e[1], dir.e[2]);
      };
      if (body == wb)
        F.add(t, dir, p.kx, far);
      else
        add_force(force, body, t, dir);
    }
  }
  if (wb >= 0) {
    F.reduce();
    if (lane == 0)
      for (int a = 0; a < 3; ++a) red[a][warp] = F.value(a, p.kx);
  }
  cp_async_wait_all();
  __syncthreads();  // staged pulls, link values and warp sums of the whole block
  if (wb >= 0 && threadIdx.x < 3) {
    double acc = 0.0;
#pragma unroll
    for (int wi = 0; wi < NW; ++wi) acc += red[threadIdx.x][wi];
    atomicAdd(&force[3 * wb + threadIdx.x], acc);
  }
  if (live) {
    T f[L::Q];
#pragma unroll
    for (int i = 0; i < L::Q; ++i) f[i] = col[i][lane];
    collide_node<L, P, MULTI, false>(f, p, lay, dom, fout, S, k, mom_out, (w & W_CACHE) != 0, fluid, [&](T(&g)[L::Q]) {
#pragma unroll
      for (int i = 0; i < L::Q; ++i) g[i] = col[i][lane];
    });
  }
}

// ------------------------------------------------------------ inline step --

// D2Q9 directions in a word each (two bits a direction): cx + 1, cy + 1; the
// opposite of direction i in four bits.  Lanes holding different directions
// unpack them without a table in memory.
constexpr uint32_t d2q9_pack(bool y) {
  uint32_t v = 0;
  for (int i = 0; i < 9; ++i) v |= (uint32_t)((y ? D2Q9::cy(i) : D2Q9::cx(i)) + 1) << (2 * i);
  return v;
}
constexpr uint64_t d2q9_opposites() {
  uint64_t v = 0;
  for (int i = 0; i < 9; ++i) v |= (uint64_t)D2Q9::opp(i) << (4 * i);
  return v;
}

// Nodes a warp without links takes at a time (two groups: 18 FP32 loads in
// flight a thread).
template <class P>
constexpr int inline_free_groups() {
  return P::shifted ? 2 : 1;
}

// One time step of a D2Q9 lattice with its links in the pull pass.  Cut links
// are few in two dimensions (the boundary of an area: 0.06 per node in the
// channel batch), so the groups of 32 stored nodes are listed by whether they
// have any: the first blocks take those with links, a group per warp, the
// others are k_bulk's pass, two groups per warp, with no mask, link range,
// stage or barrier to read or wait for.  A warp with links evaluates them one
// per lane (they are contiguous in the link list) while its pulls are in
// flight, and hands the values to their nodes through its own part of shared
// memory.  Where there are few groups with links, up to two blocks an SM
// (`spread`), a block takes one group and evaluates its links with all its warps: a
// wall row has 96, three rounds of one warp.  Channels of 60 rows, us per step with
// a block and with a warp on each group: 126 groups FP32 3.4 and 6.0, FP64 7.4 and
// 11.5; 284 groups 5.0 and 6.3, 14.2 and 13.4; 564 groups 7.7 and 7.2, 29.9 and 27.5.
constexpr int64_t kInlineSpread = 2 * 152;
__host__ __device__ __forceinline__ bool inline_spread(int64_t nlinked) { return nlinked <= kInlineSpread; }

template <class L, class P, bool MULTI, int BT>
__global__ void __launch_bounds__(BT, (fused_blocks_per_sm<L, P, BT>())) k_inline(
    const typename P::T* fin, typename P::T* __restrict__ fout, Layout lay,
    FusedLinks<typename P::T> fl, const Mom4<typename P::T>* mom_in,
    Mom4<typename P::T>* __restrict__ mom_out, double* force, double* force_next,
    Params p) {
  using T = typename P::T;
  constexpr int NW = BT / 32, NF = inline_free_groups<P>();
  let_next_start();
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const size_t S = (size_t)lay.S;
  const bool spread = inline_spread(lay.nlinked);
  const int64_t nlb = spread ? lay.nlinked : (lay.nlinked + NW - 1) / NW;  // blocks with links
  if ((int64_t)blockIdx.x >= nlb) {
    const int64_t at = lay.nlinked + (((int64_t)blockIdx.x - nlb) * NW + warp) * NF;
    if constexpr (P::shifted) {
      if (p.collision == 0) {
        // two groups a warp, a pair of neighbours a lane
        const int64_t mine = at + (lane >> 4);
        const bool some = mine < lay.ngroups;
        const uint32_t k = (some ? 32u * __ldg(lay.groups + mine) : 0u) + 2u * (lane & 15);
        prefetch_ahead<L::Q>(fin, lay, k & ~31u, 32, lane & 15, 16);
        bulk_pair<MULTI, false>(k, some, fin, fout, lay, mom_out, p);
        clear_force<BT>(force_next, p.nbody);
        return;
      }
    }
    uint32_t k[NF];
    bool live[NF];
#pragma unroll
    for (int j = 0; j < NF; ++j) {
      k[j] = at + j < lay.ngroups ? 32u * __ldg(lay.groups + at + j) + lane : 0u;
      live[j] = at + j < lay.ngroups && (uint64_t)k[j] < S;
    }
    prefetch_ahead<L::Q>(fin, lay, k[0] - lane, 32 * NF, lane, 32);
    bulk_nodes<L, P, MULTI, NF, false>(k, live, fin, fout, lay, mom_out, p);
    clear_force<BT>(force_next, p.nbody);
    return;
  }
  __shared__ T stage[NW][L::Q][32];
  __shared__ double red[2][NW];
  __shared__ int rbody[NW];
  const int64_t at = spread ? (int64_t)blockIdx.x : (int64_t)blockIdx.x * NW + warp;
  const bool some = at < lay.nlinked;
  // spread: the first warp holds the group's nodes, the others its links
  const bool mine = !spread || warp == 0;
  const int first = spread ? (int)threadIdx.x - 32 : lane, step = spread ? BT - 32 : 32;
  const uint32_t g = some ? __ldg(lay.groups + at) : 0u;
  const uint32_t k = 32u * g + lane;
  const bool live = some && (uint64_t)k < S;
  const int64_t l0 = some ? __ldg(fl.first + g) : 0, l1 = some ? __ldg(fl.first + g + 1) : 0;
  FusedRec r{0, 0, 0, 0};
  T q1 = 0;
  if (first >= 0 && l0 + first < l1) {
    r = fl.rec[l0 + first];
    if (!P::shifted) q1 = (T)__ldg(fl.qd + l0 + first);
  }
  const uint32_t w = live ? __ldg(lay.word + k) : W_GHOST;
  const uint32_t mask = live ? __ldg(fl.mask + k) : 0u;
  const bool fluid = !(w & (W_GHOST | W_OPEN));
  T f[L::Q];
  int dom = 0;
  RunRec run{};
  if (fluid && mine) run = lay.runs[w & W_RUN];
  dom = run.dom;
  wait_for_previous();
  clear_force<BT>(force_next, p.nbody);
  auto pull = [&] {
    if (fluid && mine) pull_node<L>(fin, S, k, run, lay, p, f);
  };
  if (P::shifted || spread) pull();  // (else FP64: after the links, whose registers it would spill)
  T(&col)[L::Q][32] = stage[spread ? 0 : warp];
  // forces are summed for the body of the warp's first link
  const int wb = (int)(__shfl_sync(0xffffffffu, r.meta, 0) >> 8) - 1;
  LinkForce<T, 32 * (L::Q - 1)> F;
  for (int64_t li = first < 0 ? l1 : l0 + first; li < l1; li += step) {
    if (li != l0 + first) {
      r = fl.rec[li];
      if (!P::shifted) q1 = (T)__ldg(fl.qd + li);
    }
    const T q = P::shifted ? (T)__uint_as_float(r.q32) : q1;
    const int ip = (int)(r.meta & 31), rule = (int)((r.meta >> 5) & 7), body = (int)(r.meta >> 8) - 1;
    const int i = (int)(d2q9_opposites() >> (4 * ip)) & 15;
    const int ex = (int)((d2q9_pack(false) >> (2 * ip)) & 3) - 1, ey = (int)((d2q9_pack(true) >> (2 * ip)) & 3) - 1;
    auto real = [](int e) { return e == 0 ? (T)0 : (e > 0 ? (T)1 : (T)-1); };
    DirVal<T> dir;
    dir.wt = ip < 5 ? (T)L::w(1) : (T)L::w(5);
    dir.ex = real(ex);
    dir.ey = real(ey);
    dir.ez = (T)0;
    if constexpr (!P::shifted) {
      dir.e[0] = ex;
      dir.e[1] = ey;
      dir.e[2] = 0;
    }
    T uw0 = 0, uw1 = 0;
    if (fl.uw) {
      uw0 = fl.uw[li];
      uw1 = fl.uw[fl.nl + li];
    }
    T fpf;
    const T val = eval_link<L, P>(dir, ip, i, fin, mom_in, S, rule, q, r.kf, r.kff, uw0, uw1, (T)0, p, fpf,
                                  fl.uw != nullptr, fl.wq + li, fl.nl);
    col[i][r.kf & 31] = val;
    if (body >= 0) {
      // momentum exchange as in k_links
      const T t = exchange<P>(fpf, val, dir, p);
      auto far = [&] {
        if constexpr (!P::shifted) add_force_together(force, body, t, dir.e[0], dir.e[1], dir.e[2]);
      };
      if (body == wb)
        F.add(t, dir, p.kx, far);
      else
        add_force(force, body, t, dir);
    }
  }
  if (!P::shifted && !spread) pull();
  if (wb >= 0) F.reduce();
  if (lane == 0) {
    red[0][warp] = F.value(0, p.kx);
    red[1][warp] = F.value(1, p.kx);
    rbody[warp] = wb;
  }
  // the block's force: one atomic per run of warps with one body
  auto add_block_force = [&](int a) {
    double acc = 0.0;
#pragma unroll 1
    for (int wi = 0; wi < NW; ++wi) {
      const int b = rbody[wi];
      acc += red[a][wi];
      if (b >= 0 && (wi == NW - 1 || rbody[wi + 1] != b)) {
        atomicAdd(&force[3 * b + a], acc);
        acc = 0.0;
      }
    }
  };
  if (spread) {
    __syncthreads();
    if (!mine) {  // (the force off the first warp's way)
      if (warp == 1 && lane < 2) add_block_force(lane);
      return;
    }
  } else {
    __syncwarp();
  }
  // the populations of v that come from a wall
  auto take = [&](T(&v)[L::Q]) {
#pragma unroll
    for (int i = 1; i < L::Q; ++i)
      if ((mask >> L::opp(i)) & 1u) v[i] = col[i][lane];
  };
  if (mask) take(f);
  if (live && !(w & W_OPEN)) {
    // ghost slots: zeros through the same stores (inputs at rest)
    if (!fluid) {
#pragma unroll
      for (int i = 0; i < L::Q; ++i) f[i] = P::shifted ? (T)0 : (T)L::w(i);
    }
    collide_node<L, P, MULTI, false>(f, p, lay, dom, fout, S, k, mom_out, (w & W_CACHE) != 0, fluid, [&](T(&v)[L::Q]) {
      pull_node<L>(fin, S, k, lay.runs[w & W_RUN], lay, p, v);
      take(v);
    });
    if (fluid && (p.inlet | p.outlet)) open_ends<L, P>(fout, mom_out, S, k, lay.runs[w & W_RUN], lay, p);
  }
  if (spread) return;
  __syncthreads();
  if (threadIdx.x < 2) add_block_force((int)threadIdx.x);
}

// ------------------------------------------------------- init and fields --

__device__ __forceinline__ bool is_fluid(uint32_t w) { return (w & (W_GHOST | W_OPEN)) == 0; }

// f(x,0) = feq(rho_in, u_in) followed by the collision at t = 0 (fluid
// nodes), and the open columns filled from it; zero elsewhere.  rho_in (N) and
// u_in (N x 3, interleaved), dense indices, may be null for rho0 and rest.
template <class L, class P>
__global__ void k_init(typename P::T* __restrict__ f, Mom4<typename P::T>* __restrict__ mom, Layout lay,
                       const double* __restrict__ rho_in, const double* __restrict__ u_in, Params p) {
  using T = typename P::T;
  const int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (k >= lay.S) return;
  const size_t S = (size_t)lay.S;
  const uint32_t w = lay.word[k];
  if (!is_fluid(w)) {
    if (w & W_OPEN) return;  // (the thread of the fluid node beside it writes it)
#pragma unroll
    for (int i = 0; i < L::Q; ++i) f[(size_t)i * S + k] = (T)0;
    return;
  }
  const int64_t n = lay.node_of[k];
  const Relax rx = relax_of_run(p, lay, w & W_RUN);
  const double rho = rho_in ? rho_in[n] : p.rho0;
  const double ux = u_in ? u_in[3 * n] : 0.0, uy = u_in ? u_in[3 * n + 1] : 0.0;
  const double uz = (u_in && L::D == 3) ? u_in[3 * n + 2] : 0.0;
  T fl[L::Q];
#pragma unroll
  for (int i = 0; i < L::Q; ++i) {
    const double eu = L::cx(i) * ux + L::cy(i) * uy + L::cz(i) * uz;
    const double poly = 3.0 * eu + 4.5 * eu * eu - 1.5 * (ux * ux + uy * uy + uz * uz);
    fl[i] = P::shifted ? (T)(L::w(i) * ((rho - p.rho0) + rho * poly)) : (T)(L::w(i) * rho * (1.0 + poly));
  }
  // one inlined collision for both cases (the lattice's constants or the
  // domain's), so that a domain's initial state has the same bits alone and
  // in a batch
  const Folded* kc = lay.ndom > 1 ? &lay.dom[lay.runs[w & W_RUN].dom].kc : &p.kc;
  collide_store<L, P>(fl, p, rx, *kc, f, S, (uint32_t)k, mom, (w & W_CACHE) != 0);
  open_ends<L, P>(f, mom, S, (uint32_t)k, lay.runs[w & W_RUN], lay, p);
}

// A float as a double by moving its bits: a hardware conversion takes the FP64
// pipe for as long as an FP64 addition.  Denormals, infinities and NaNs
// (`odd`) are not carried over right.
__device__ __forceinline__ double widen(float v, bool& odd) {
  const uint32_t b = __float_as_uint(v), m = b << 1;
  odd |= m - 0x01000000u >= 0xfe000000u && m != 0u;
  return __hiloint2double((int)(m == 0u ? b : ((b & 0x80000000u) | ((m >> 4) + (896u << 20)))), (int)(b << 29));
}

// (1/x) for x in [2^-100, 2^100] (else `odd`) from its float reciprocal by one
// third-order Newton step.
__device__ __forceinline__ double reciprocal_from(double x, float seed, bool& odd) {
  odd |= ((uint32_t)__double2hiint(x) >> 20) - (1023u - 100u) > 200u;
  const double y = widen(seed, odd), d = fma(-x, y, 1.0);
  return fma(y, fma(d, d, d), y);
}

// (rho, u) of a node from its sums in doubles, by divisions: where a value is
// out of the range of the quicker forms.  Out of line, so that its FP64
// instructions are not issued under a predicate in every node's path.
struct RhoU {
  double rho, ux, uy, uz;
};
static __device__ __noinline__ RhoU divided_moments(double rho, double jx, double jy, double jz) {
  return RhoU{rho, jx / rho, jy / rho, jz / rho};
}

// rho = sum f+, u = (sum f+ e - g/2)/rho of fluid node k of the post-collision
// state (the collision conserves mass and adds g to the momentum).  The FP64
// pipe bounds this pass too (2 operations per clock and SM against 28 B read
// and written per clock and SM), so FP64 sums the populations on the integer
// grid and FP32 forms its quotients from one reciprocal: 13 FP64 operations
// per D3Q19 FP64 node (99 with sums and quotients in doubles), 9 per FP32 node
// (41).
template <class L, class P>
__device__ __forceinline__ void node_moments(const typename P::T* __restrict__ f, size_t S, int64_t k,
                                             const Layout& lay, const Params& p, uint32_t w, double (&v)[1 + L::D]) {
  using T = typename P::T;
  T h[L::Q];
#pragma unroll
  for (int i = 0; i < L::Q; ++i) h[i] = f[(size_t)i * S + k];
  if constexpr (!P::shifted) {
    // (a domain whose force is beyond the grid's has no grid constants)
    bool on = p.kx.on != 0;
    if (lay.ndom > 1) on = lay.dom[lay.runs[w & W_RUN].dom].kx.on != 0;
    if (on) {
      uint64_t r = 0, j[3] = {0, 0, 0};
      uint32_t bad = 0;
#pragma unroll
      for (int i = 0; i < L::Q; ++i) {
        const uint64_t F = i == 0    ? to_grid<9>(h[i], p.kx.sc, bad)
                           : L::Q == 9 ? (i < 5 ? to_grid<8>(h[i], p.kx.sc, bad) : to_grid<7>(h[i], p.kx.sc, bad))
                                       : (i < 7 ? to_grid<7>(h[i], p.kx.sc, bad) : to_grid<6>(h[i], p.kx.sc, bad));
        r += F;
        const int c[3] = {L::cx(i), L::cy(i), L::cz(i)};
#pragma unroll
        for (int a = 0; a < L::D; ++a) j[a] += c[a] > 0 ? F : (c[a] < 0 ? 0 - F : 0);
      }
      if (bad < 32u && beyond_rho(r) == 0u) {
        // (half the force in grid steps, value by value: a reference to one of
        // two parameter blocks would copy the kernel's parameters to memory)
        int64_t hg[3] = {p.kx.hg[0], p.kx.hg[1], p.kx.hg[2]};
        if (lay.ndom > 1)
#pragma unroll
          for (int a = 0; a < L::D; ++a) hg[a] = lay.dom[lay.runs[w & W_RUN].dom].kx.hg[a];
        bool odd = false;
        v[0] = from_grid<true>(r, p.kx.sc, bad);
        const float rf = (float)(uint32_t)(r >> 32) * 0x1p-30f;  // rho in units of 2^sc
        const double x = from_grid<true>(r, 0, bad), y = reciprocal_from(x, __frcp_rn(rf), odd) * 0x1p-62;
#pragma unroll
        for (int a = 0; a < L::D; ++a) v[1 + a] = (double)((int64_t)j[a] - hg[a]) * y;
        return;
      }
    }
  }
  T r = 0, jx = 0, jy = 0, jz = 0;
#pragma unroll
  for (int i = 0; i < L::Q; ++i) {
    r += h[i];
    if (L::cx(i) > 0) jx += h[i];
    if (L::cx(i) < 0) jx -= h[i];
    if (L::cy(i) > 0) jy += h[i];
    if (L::cy(i) < 0) jy -= h[i];
    if (L::cz(i) > 0) jz += h[i];
    if (L::cz(i) < 0) jz -= h[i];
  }
  const T j[3] = {jx, jy, jz};
  double hg[3] = {p.kc.hg[0], p.kc.hg[1], p.kc.hg[2]};
  bool force = p.has_force != 0;
  if (lay.ndom > 1) {
    const DomPar& dp = lay.dom[lay.runs[w & W_RUN].dom];
    force = dp.has_force != 0;
#pragma unroll
    for (int a = 0; a < L::D; ++a) hg[a] = dp.kc.hg[a];
  }
  if constexpr (P::shifted) {
    bool odd = false;
    v[0] = p.rho0 + widen(r, odd);
    const double y = reciprocal_from(v[0], __frcp_rn(p.rho0_f + r), odd);
#pragma unroll
    for (int a = 0; a < L::D; ++a) {
      const double ja = widen(j[a], odd);
      v[1 + a] = (force ? ja - hg[a] : ja) * y;
    }
    if (!odd) return;
  }
  const RhoU m = divided_moments((P::shifted ? p.rho0 : 0.0) + (double)r, (double)jx - hg[0], (double)jy - hg[1],
                                    (double)jz - hg[2]);
  v[0] = m.rho;
  v[1] = m.ux;
  v[2] = m.uy;
  if (L::D == 3) v[L::D] = m.uz;
}

// rho and u in FP64 at dense indices, zero at nodes that are not fluid; u:
// [D][N].  A warp takes MOM_TILE dense nodes, whose stored nodes are
// contiguous (lay.tile): where all of them are stored each lane writes its
// own; else the tile is put together in shared memory, so that the outputs are
// written whole and once (clearing them first and writing the fluid nodes'
// scattered runs moved the pack's outputs nearly three times).  A tile per
// warp, since warps that wait for one another between the loads, the FP64 sums
// and the stores overlap none of them.  Blocks per SM: as many as the
// registers allow without spilling the sums (28 % of the warps resident was
// 1.6 times slower).  384^3 pack FP32 2.0 -> 0.79 ms, 8192 x 4096 FP32 0.95 ->
// 0.51 ms (FP64 pipe), 192^3 FP64 1.34 -> 0.22 ms (0.86 of the copy rate).
constexpr int MOM_TILE = 128, MOM_WARPS = 4;
template <class L, class P>
__global__ void __launch_bounds__(32 * MOM_WARPS, (P::shifted ? (L::Q == 9 ? 12 : 10) : 8)) k_moments(
    const typename P::T* __restrict__ f, Layout lay, double* __restrict__ rho_out, double* __restrict__ u_out,
    Params p) {
  __shared__ double tiles[MOM_WARPS][1 + L::D][MOM_TILE];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const size_t S = (size_t)lay.S;
  const int64_t N = p.N, b = (int64_t)blockIdx.x * MOM_WARPS + warp, n0 = b * MOM_TILE;
  if (n0 >= N) return;
  double(&tile)[1 + L::D][MOM_TILE] = tiles[warp];
  const int len = (int)(N - n0 < MOM_TILE ? N - n0 : MOM_TILE);
  const int64_t ka = lay.tile[b], kb = lay.tile[b + 1];
  const bool whole = kb - ka == len;
  if (!whole) {
    for (int t = lane; t < len; t += 32)
#pragma unroll
      for (int a = 0; a <= L::D; ++a) tile[a][t] = 0.0;
    __syncwarp();
  }
  for (int64_t k = ka + lane; k < kb; k += 32) {
    const uint32_t w = lay.word[k];
    double v[1 + L::D] = {};
    if (is_fluid(w)) node_moments<L, P>(f, S, k, lay, p, w, v);
    if (whole) {
      const int64_t n = n0 + (k - ka);
      rho_out[n] = v[0];
#pragma unroll
      for (int a = 0; a < L::D; ++a) u_out[a * N + n] = v[1 + a];
    } else {
      const int t = (int)(lay.node_of[k] - n0);
#pragma unroll
      for (int a = 0; a <= L::D; ++a) tile[a][t] = v[a];
    }
  }
  if (whole) return;
  __syncwarp();
  for (int t = lane; t < len; t += 32) {
    rho_out[n0 + t] = tile[0][t];
#pragma unroll
    for (int a = 0; a < L::D; ++a) u_out[a * N + n0 + t] = tile[1 + a][t];
  }
}

// Moment cache refresh from a post-collision state (after the caller sets
// the populations): same formula as k_moments, storage precision.
template <class L, class P>
__global__ void k_refresh(const typename P::T* __restrict__ f, Layout lay, Mom4<typename P::T>* __restrict__ mom,
                          Params p) {
  using T = typename P::T;
  const int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (k >= lay.S || !(lay.word[k] & W_CACHE) || !is_fluid(lay.word[k])) return;
  const size_t S = (size_t)lay.S;
  const Relax rx = relax_of_run(p, lay, lay.word[k] & W_RUN);
  T r = 0, jx = 0, jy = 0, jz = 0;
#pragma unroll
  for (int i = 0; i < L::Q; ++i) {
    const T v = f[(size_t)i * S + k];
    r += v;
    jx += (T)L::cx(i) * v;
    jy += (T)L::cy(i) * v;
    jz += (T)L::cz(i) * v;
  }
  const T rho = P::shifted ? par<T>(p.rho0, p.rho0_f) + r : r;
  mom[k] = Mom4<T>{r, (jx - par<T>(0.5 * rx.g[0], rx.hg_f[0])) / rho, (jy - par<T>(0.5 * rx.g[1], rx.hg_f[1])) / rho,
                   L::D == 3 ? (jz - par<T>(0.5 * rx.g[2], rx.hg_f[2])) / rho : (T)0};
}

template <class L>
__device__ __forceinline__ double weight_of(int i) {
  double w = 0.0;
#pragma unroll
  for (int k = 0; k < L::Q; ++k)
    if (k == i) w = L::w(k);
  return w;
}

// One direction of the state to (k_get_dir, dense FP64 unshifted output,
// zeroed by the caller) or from (k_set_dir) the caller's layout.
template <class L, class P>
__global__ void k_get_dir(const typename P::T* __restrict__ f, Layout lay, int i, double* __restrict__ out, Params p) {
  const int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (k >= lay.S || !is_fluid(lay.word[k])) return;
  out[lay.node_of[k]] = (double)f[(size_t)i * lay.S + k] + (P::shifted ? weight_of<L>(i) * p.rho0 : 0.0);
}

template <class L, class P>
__global__ void k_set_dir(typename P::T* __restrict__ f, Layout lay, int i, const double* __restrict__ in, Params p) {
  using T = typename P::T;
  const int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (k >= lay.S) return;
  f[(size_t)i * lay.S + k] =
      is_fluid(lay.word[k]) ? (T)(in[lay.node_of[k]] - (P::shifted ? weight_of<L>(i) * p.rho0 : 0.0)) : (T)0;
}

// Populations of listed storage indices (-1: not a fluid node -> 0), FP64
// unshifted, out[k*Q + i].
template <class L, class P>
__global__ void k_gather(const typename P::T* __restrict__ f, Layout lay, const int64_t* __restrict__ sk, int64_t n,
                         double* __restrict__ out, Params p) {
  const int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (k >= n) return;
  const int64_t s = sk[k];
  const bool off = s < 0 || !is_fluid(lay.word[s]);
#pragma unroll
  for (int i = 0; i < L::Q; ++i)
    out[k * L::Q + i] = off ? 0.0 : (double)f[(size_t)i * lay.S + s] + (P::shifted ? L::w(i) * p.rho0 : 0.0);
}

// Failure detection: flag any non-finite population or non-positive density.
template <class L, class P>
__global__ void k_check(const typename P::T* __restrict__ f, Layout lay, int* __restrict__ flag, Params p) {
  using T = typename P::T;
  const int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (k >= lay.S || !is_fluid(lay.word[k])) return;
  T r = 0;
  bool bad = false;
#pragma unroll
  for (int i = 0; i < L::Q; ++i) {
    const T v = f[(size_t)i * lay.S + k];
    bad |= !isfinite(v);
    r += v;
  }
  const double rho = P::shifted ? p.rho0 + (double)r : (double)r;
  if (bad || !(rho > 0.0)) atomicOr(flag, 1);
}

// ------------------------------------------------------------- launchers --

// Link arrays of the fused step kernel without the storage type (the
// launchers cast q and uw).
struct FusedRaw {
  const int32_t* first;
  const uint32_t* mask;
  const FusedRec* rec;
  const double* qd;
  const void* uw;
  const int64_t* wq;
  int64_t nl, ngroups;
};

struct KernelOps {
  int Q, D;
  size_t real_bytes;
  int default_shape;
  unsigned shape_mask;  // bit b: kBulkShapes[b] is built for this stencil
  // shape: index into kBulkShapes; threads: link kernel block size (64, 128 or
  // 256); seq: links per thread of the link kernel (1 or 4)
  void (*bulk)(const void* fin, void* fout, const Layout& lay, void* mom, double* force_next, const Params& p,
               int shape, cudaStream_t s);
  void (*links)(void* f, const void* mom, const LinkRec* recs, const void* q, const void* uw, const int64_t* wq,
                int64_t nl, double* force, const Params& p, int64_t S, int threads, int seq, cudaStream_t s);
  // fused step (threads per block 128, 256 or 512; 512 runs as 256 for
  // FP64 D3Q19, whose link buffer would not fit the static shared memory)
  void (*fused)(const void* fin, void* fout, const Layout& lay, const FusedRaw& fl, const void* mom_in,
                void* mom_out, double* force, double* force_next, const Params& p, int threads, cudaStream_t s);
  void (*open)(void* f, const void* mom, const Layout& lay, const Params& p, cudaStream_t s);
  void (*init)(void* f, void* mom, const Layout& lay, const double* rho, const double* u, const Params& p,
               cudaStream_t s);
  void (*moments)(const void* f, const Layout& lay, double* rho, double* u, const Params& p, cudaStream_t s);
  void (*refresh)(const void* f, const Layout& lay, void* mom, const Params& p, cudaStream_t s);
  void (*get_dir)(const void* f, const Layout& lay, int i, double* out, const Params& p, cudaStream_t s);
  void (*set_dir)(void* f, const Layout& lay, int i, const double* in, const Params& p, cudaStream_t s);
  void (*check)(const void* f, const Layout& lay, int* flag, const Params& p, cudaStream_t s);
  void (*gather)(const void* f, const Layout& lay, const int64_t* sk, int64_t n, double* out, const Params& p,
                 cudaStream_t s);
};

inline unsigned blocks_for(int64_t n, int b) { return (unsigned)((n + b - 1) / b); }

// Launch of a step kernel that may start before its predecessor in the stream
// has ended (it waits by itself).
template <class... K, class... A>
inline void launch_early(void (*kernel)(K...), unsigned grid, int block, cudaStream_t s, A&&... args) {
  cudaLaunchAttribute early;
  early.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  early.val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(grid);
  cfg.blockDim = dim3(block);
  cfg.stream = s;
  cfg.attrs = &early;
  cfg.numAttrs = 1;
  cudaLaunchKernelEx(&cfg, kernel, (K)args...);
}

template <class L, class P>
struct Launch {
  using T = typename P::T;
  template <bool M, int BT, int NPT>
  static void bulk_shape(const void* fin, void* fout, const Layout& lay, void* mom, double* force_next,
                         const Params& p, cudaStream_t s) {
    if constexpr (!P::shifted && NPT == 1) {
      if (lay.fluid) {
        launch_early(k_bulk_list<L, P, M, BT>, blocks_for(lay.nfluid > 0 ? lay.nfluid : 1, BT), BT, s, (const T*)fin,
                     (T*)fout, lay, (Mom4<T>*)mom, force_next, p);
        return;
      }
    }
    launch_early(k_bulk<L, P, M, BT, NPT>, blocks_for((lay.S + NPT - 1) / NPT, BT), BT, s, (const T*)fin, (T*)fout, lay,
                 (Mom4<T>*)mom, force_next, p);
  }
  template <bool M, int BT, int SEQ>
  static void bulk_seq(const void* fin, void* fout, const Layout& lay, void* mom, double* force_next,
                       const Params& p, cudaStream_t s) {
    launch_early(k_bulk_seq<L, P, M, BT, SEQ>, blocks_for((lay.S + SEQ - 1) / SEQ, BT), BT, s, (const T*)fin, (T*)fout,
                 lay, (Mom4<T>*)mom, force_next, p);
  }
  template <bool M>
  static void bulk_m(const void* fin, void* fout, const Layout& lay, void* mom, double* fn, const Params& p,
                     int shape, cudaStream_t s) {
    switch (shape) {
      case 1: return bulk_shape<M, 128, 1>(fin, fout, lay, mom, fn, p, s);
      case 2: return bulk_shape<M, 512, 1>(fin, fout, lay, mom, fn, p, s);
      default: break;
    }
    if constexpr (bulk_max_npt<L>() >= 2) {
      switch (shape) {
        case 3: return bulk_shape<M, 256, 2>(fin, fout, lay, mom, fn, p, s);
        case 4: return bulk_shape<M, 128, 2>(fin, fout, lay, mom, fn, p, s);
        case 5: return bulk_shape<M, 512, 2>(fin, fout, lay, mom, fn, p, s);
        case 6: return bulk_seq<M, 128, 4>(fin, fout, lay, mom, fn, p, s);
        case 7: return bulk_seq<M, 128, 8>(fin, fout, lay, mom, fn, p, s);
        default: break;
      }
    }
    bulk_shape<M, 256, 1>(fin, fout, lay, mom, fn, p, s);
  }
  static void bulk(const void* fin, void* fout, const Layout& lay, void* mom, double* force_next, const Params& p,
                   int shape, cudaStream_t s) {
    if (lay.S == 0) return;
    if (lay.ndom > 1)
      bulk_m<true>(fin, fout, lay, mom, force_next, p, shape, s);
    else
      bulk_m<false>(fin, fout, lay, mom, force_next, p, shape, s);
  }
  static void links(void* f, const void* mom, const LinkRec* recs, const void* q, const void* uw, const int64_t* wq,
                    int64_t nl, double* force, const Params& p, int64_t S, int threads, int seq, cudaStream_t s) {
    if (nl == 0) return;
    const int bt = (threads == 64 || threads == 128) ? threads : 256;
    if (seq == 4)
      launch_early(k_links<L, P, 4>, blocks_for(nl, 4 * bt), bt, s, (T*)f, (const Mom4<T>*)mom, recs, (const T*)q,
                   (const T*)uw, wq, nl, force, p, S);
    else
      launch_early(k_links<L, P, 1>, blocks_for(nl, bt), bt, s, (T*)f, (const Mom4<T>*)mom, recs, (const T*)q,
                   (const T*)uw, wq, nl, force, p, S);
  }
  template <bool M, int BT>
  static void fused_shape(const void* fin, void* fout, const Layout& lay, const FusedRaw& r, const void* mom_in,
                          void* mom_out, double* force, double* force_next, const Params& p, cudaStream_t s) {
    const FusedLinks<T> fl{r.first, r.mask, r.rec, r.qd, (const T*)r.uw, r.wq, r.nl, r.ngroups};
    if constexpr (L::Q == 9) {
      const int64_t nw = BT / 32, nf = inline_free_groups<P>();
      const int64_t nb = (inline_spread(lay.nlinked) ? lay.nlinked : (lay.nlinked + nw - 1) / nw) + (lay.ngroups - lay.nlinked + nw * nf - 1) / (nw * nf);
      launch_early(k_inline<L, P, M, BT>, (unsigned)nb, BT, s, (const T*)fin, (T*)fout, lay, fl,
                   (const Mom4<T>*)mom_in, (Mom4<T>*)mom_out, force, force_next, p);
    } else {
      launch_early(k_fused<L, P, M, BT>, blocks_for(lay.S, BT), BT, s, (const T*)fin, (T*)fout, lay, fl,
                   (const Mom4<T>*)mom_in, (Mom4<T>*)mom_out, force, force_next, p);
    }
  }
  template <bool M>
  static void fused_m(const void* fin, void* fout, const Layout& lay, const FusedRaw& r, const void* mom_in,
                      void* mom_out, double* force, double* force_next, const Params& p, int threads,
                      cudaStream_t s) {
    constexpr bool big_ok = P::shifted || L::Q == 9;
    if (threads == 128) return fused_shape<M, 128>(fin, fout, lay, r, mom_in, mom_out, force, force_next, p, s);
    if (big_ok && threads == 512)
      return fused_shape<M, big_ok ? 512 : 256>(fin, fout, lay, r, mom_in, mom_out, force, force_next, p, s);
    fused_shape<M, 256>(fin, fout, lay, r, mom_in, mom_out, force, force_next, p, s);
  }
  static void fused(const void* fin, void* fout, const Layout& lay, const FusedRaw& r, const void* mom_in,
                    void* mom_out, double* force, double* force_next, const Params& p, int threads,
                    cudaStream_t s) {
    if (lay.S == 0) return;
    if (lay.ndom > 1)
      fused_m<true>(fin, fout, lay, r, mom_in, mom_out, force, force_next, p, threads, s);
    else
      fused_m<false>(fin, fout, lay, r, mom_in, mom_out, force, force_next, p, threads, s);
  }
  static void open(void* f, const void* mom, const Layout& lay, const Params& p, cudaStream_t s) {
    k_open<L, P><<<blocks_for(2 * (int64_t)p.ny, 128), 128, 0, s>>>((T*)f, (const Mom4<T>*)mom, lay, p);
  }
  static void init(void* f, void* mom, const Layout& lay, const double* rho, const double* u, const Params& p,
                   cudaStream_t s) {
    if (lay.S == 0) return;
    k_init<L, P><<<blocks_for(lay.S, 256), 256, 0, s>>>((T*)f, (Mom4<T>*)mom, lay, rho, u, p);
  }
  static void moments(const void* f, const Layout& lay, double* rho, double* u, const Params& p, cudaStream_t s) {
    k_moments<L, P><<<blocks_for(p.N, MOM_TILE * MOM_WARPS), 32 * MOM_WARPS, 0, s>>>((const T*)f, lay, rho, u, p);
  }
  static void refresh(const void* f, const Layout& lay, void* mom, const Params& p, cudaStream_t s) {
    if (lay.S == 0) return;
    k_refresh<L, P><<<blocks_for(lay.S, 256), 256, 0, s>>>((const T*)f, lay, (Mom4<T>*)mom, p);
  }
  static void get_dir(const void* f, const Layout& lay, int i, double* out, const Params& p, cudaStream_t s) {
    if (lay.S == 0) return;
    k_get_dir<L, P><<<blocks_for(lay.S, 256), 256, 0, s>>>((const T*)f, lay, i, out, p);
  }
  static void set_dir(void* f, const Layout& lay, int i, const double* in, const Params& p, cudaStream_t s) {
    if (lay.S == 0) return;
    k_set_dir<L, P><<<blocks_for(lay.S, 256), 256, 0, s>>>((T*)f, lay, i, in, p);
  }
  static void check(const void* f, const Layout& lay, int* flag, const Params& p, cudaStream_t s) {
    if (lay.S == 0) return;
    k_check<L, P><<<blocks_for(lay.S, 256), 256, 0, s>>>((const T*)f, lay, flag, p);
  }
  static void gather(const void* f, const Layout& lay, const int64_t* sk, int64_t n, double* out, const Params& p,
                     cudaStream_t s) {
    if (n == 0) return;
    k_gather<L, P><<<blocks_for(n, 256), 256, 0, s>>>((const T*)f, lay, sk, n, out, p);
  }
  static KernelOps ops() {
    return KernelOps{L::Q,   L::D,    sizeof(T), bulk_default_shape<L, P>(), bulk_shape_mask<L>(), bulk, links, fused,
                     open,   init,    moments,   refresh, get_dir, set_dir, check, gather};
  }
};

KernelOps ops_d2q9_f64();
KernelOps ops_d2q9_f32s();
KernelOps ops_d3q19_f64();
KernelOps ops_d3q19_f32s();

}  // namespace lbm
