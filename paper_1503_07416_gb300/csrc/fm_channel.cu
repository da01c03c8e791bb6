// libfm: the hydrodynamic PFC step in a channel (fm_params.walls = FM_WALLS_Y):
// periodic in x, no-slip walls at y = 0 and y = n_y h (Sec. 6.3), the walls
// moving along x at u_wall[0] (bottom) and u_wall[1] (top).
//
// Grid: the n_y rows are cells j = 0 .. n_y - 1 (centres at (j + 1/2) h), the
// walls half a cell beyond the first and last rows.  A neighbour across a
// wall is a ghost given by the rules of App. E.2: scalars (rho, rho^k, mu,
// kappa) mirror the wall row (no flux), the normal velocity is odd (no
// slip), the tangential velocity is 2 U_wall - u (no slip on a wall moving
// at U_wall); |u|^2 takes the ghosts of its factors.  In the correction form
// of the cycle (M(e) = N(c + e) - N(c)) the corrections carry homogeneous
// ghosts (odd velocity, mirrored scalars) and the coefficient velocity the
// wall speed.
//
// The same scheme and solver as fm_solver.cu otherwise: float64 outer
// residual, FAS V-cycles on the correction equation in precision T, the
// hydrodynamic point block (smooth_point_a) evaluated through an accessor
// that returns the ghost values, the fused level kernels of fm_fused.cuh, the
// coarsest level smoothed ncoarse times; the transfers are nodal in x and
// cell-centred in y (a coarse cell is two fine cells: restriction and
// injection average them, prolongation interpolates linearly between cell
// centres, weights 3/4 and 1/4).  One CUDA graph per step (fm_stepper.cuh).
#include <cuda_runtime.h>
#include <cstring>

#include "fm_state.h"
#include "fm_device.cuh"
#include "fm_stepper.cuh"
#include "fm_fused.cuh"

namespace fm {
namespace ch {

using LY = Layout<KPFC, 2>;  // rho, u, v, mu, kappa

// Neighbours of cell (i, j) of a channel level: x periodic; a neighbour
// across a wall is encoded as -1 - c (bottom) or -1 - c - N (top), c the wall
// row's own cell (the ghost mirrors it).
__device__ __forceinline__ Nb ch_neighbours(int i, int j, const Geo& g) {
  Nb n;
  const int row = j * g.nx;
  n.c = row + i;
  n.m[0] = row + (i == 0 ? g.nx - 1 : i - 1);
  n.p[0] = row + (i == g.nx - 1 ? 0 : i + 1);
  n.m[1] = j == 0 ? -1 - n.c : n.c - g.nx;
  n.p[1] = j == g.ny - 1 ? -1 - n.c - g.N : n.c + g.nx;
  n.m[2] = n.p[2] = n.c;
  return n;
}

__device__ __forceinline__ int cell_of(int i, int N) {
  if (i >= 0) return i;
  const int m = -1 - i;
  return m >= N ? m - N : m;
}

// Ghost of a value: 0 scalar (mirror), 1 tangential velocity (2U - x),
// 2 normal velocity (-x).
template <typename T>
__device__ __forceinline__ T ghost_of(T x, int type, T U) {
  return type == 0 ? x : (type == 2 ? -x : T(2) * U - x);
}

// Accessor of the correction-form point update over a channel level.
template <typename T>
struct ChAcc {
  const Lvl<T>& L;
  T ub, ut;  // wall speeds (of the coefficient velocity)
  __device__ __forceinline__ T e(int q, int i) const {
    const T v = L.e[q][cell_of(i, L.g.N)];
    return (i < 0 && (q == 1 || q == 2)) ? -v : v;  // corrections: odd velocity ghosts
  }
  __device__ __forceinline__ void set_e(int q, int i, T v) const { L.e[q][i] = v; }
  __device__ __forceinline__ T rk(int i) const { return L.rk[cell_of(i, L.g.N)]; }
  __device__ __forceinline__ T cr(int i) const { return L.cr[cell_of(i, L.g.N)]; }
  __device__ __forceinline__ T cv(int d, int i) const {
    const T v = L.cv[d][cell_of(i, L.g.N)];
    if (i >= 0) return v;
    return ghost_of(v, d == 0 ? 1 : 2, i < -L.g.N ? ut : ub);
  }
  __device__ __forceinline__ T f(int q, int i) const { return L.f[q][i]; }
  __device__ __forceinline__ T om(int d, int i) const { return L.om[d][i]; }
};

template <typename T>
struct WallsT {
  T ub, ut;
};

// The injected correction and the coefficients of coarse level C, the
// correction read from the fine level (the mean of rows 2J and 2J + 1 at 2I).
template <typename T>
struct ChInjAcc {
  const Lvl<T>& F;
  ChAcc<T> c;
  __device__ __forceinline__ T e(int q, int i) const {
    const int m = cell_of(i, c.L.g.N), nx = c.L.g.nx;
    const int a = 2 * (m / nx) * F.g.nx + 2 * (m % nx);
    const T v = T(0.5) * (F.e[q][a] + F.e[q][a + F.g.nx]);
    return (i < 0 && (q == 1 || q == 2)) ? -v : v;
  }
  __device__ __forceinline__ T rk(int i) const { return c.rk(i); }
  __device__ __forceinline__ T cr(int i) const { return c.cr(i); }
  __device__ __forceinline__ T cv(int d, int i) const { return c.cv(d, i); }
  __device__ __forceinline__ T om(int d, int i) const { return c.om(d, i); }
};

// M(e) = N(c + e) - N(c) at one cell, through the accessor (App. G.2 operator
// in correction form, as applyM of the periodic solver).
template <typename T, class A>
__device__ __forceinline__ void ch_applyM(const A& a, const Phys<T>& P, T h, const Nb& n, T* M) {
  const T ih = T(1) / h, ih2 = ih * ih;
  const int c = n.c;
  const T rkc = a.rk(c);
  T div = 0;
#pragma unroll
  for (int d = 0; d < 2; ++d) div += a.rk(n.p[d]) * a.e(1 + d, n.p[d]) - a.rk(n.m[d]) * a.e(1 + d, n.m[d]);
  M[0] = a.e(0, c) + P.s * T(0.25) * ih * div;
  auto qc = [&](int idx) {
    T q = 0;
#pragma unroll
    for (int d = 0; d < 2; ++d) {
      const T e = a.e(1 + d, idx);
      q += e * (T(2) * a.cv(d, idx) + e);
    }
    return q;
  };
  const T ec[2] = {a.e(1, c), a.e(2, c)};
  const T w = a.om(0, c);
  const T wx[2] = {-w * ec[1], w * ec[0]};
#pragma unroll
  for (int d = 0; d < 2; ++d) {
    const T dq = qc(n.p[d]) - qc(n.m[d]);
    const T dm = a.e(LY::IMU, n.p[d]) - a.e(LY::IMU, n.m[d]);
    const T nb = a.e(1 + d, n.m[0]) + a.e(1 + d, n.p[0]) + a.e(1 + d, n.m[1]) + a.e(1 + d, n.p[1]);
    const T lapa = (nb - T(4) * ec[d]) * ih2;
    M[1 + d] = rkc * ec[d] + T(0.5) * P.sigma * P.s * rkc * wx[d] + P.s * rkc * ih * (T(0.25) * dq + T(0.5) * dm)
             - T(0.5) * P.s * P.gamma * lapa;
  }
  const T er = a.e(0, c), ek = a.e(LY::IKA, c);
  const T psi = a.cr(c) - T(1.5);
  const T nbk = a.e(LY::IKA, n.m[0]) + a.e(LY::IKA, n.p[0]) + a.e(LY::IKA, n.m[1]) + a.e(LY::IKA, n.p[1]);
  const T nbr = a.e(0, n.m[0]) + a.e(0, n.p[0]) + a.e(0, n.m[1]) + a.e(0, n.p[1]);
  M[LY::IMU] = a.e(LY::IMU, c) - er * (psi * psi + psi * er + er * er * T(1.0 / 3.0)) - P.alpha * er
             - (nbk - T(4) * ek) * ih2;
  M[LY::IKA] = ek - (nbr - T(4) * er) * ih2;
}

// Coarse cell idx of fine rows 2J, 2J + 1: f_C = R(r_F) (x full weighting
// about 2I, y the mean of the two rows), e_C = eh_C = the injection (the
// mean of the two cells at x = 2I).
template <typename T>
__device__ __forceinline__ void ch_restrict(const Lvl<T>& F, const Lvl<T>& C, int idx) {
  const int I = idx % C.g.nx, J = idx / C.g.nx;
  const int x = 2 * I, xm = x == 0 ? F.g.nx - 1 : x - 1, xp = x + 1 == F.g.nx ? 0 : x + 1;
  const int r0 = 2 * J * F.g.nx, r1 = r0 + F.g.nx;
  T fr[LY::NU], ev[LY::NU];
#pragma unroll
  for (int q = 0; q < LY::NU; ++q) {
    const T* r = F.r[q];
    fr[q] = T(0.125) * (r[r0 + xm] + r[r1 + xm] + r[r0 + xp] + r[r1 + xp]) + T(0.25) * (r[r0 + x] + r[r1 + x]);
    ev[q] = T(0.5) * (F.e[q][r0 + x] + F.e[q][r1 + x]);
  }
#pragma unroll
  for (int q = 0; q < LY::NU; ++q) {
    C.f[q][idx] = fr[q];
    C.e[q][idx] = ev[q];
    C.eh[q][idx] = ev[q];
  }
}

// Coefficients of the finest level injected into every coarser level at once: a
// level's value is the mean of the two fine cells of the level
// above at x = 2I, so level l takes the pairwise means over 2^l rows, eight
// rows loaded at a time.
struct InjRows {
  template <typename T>
  static __device__ __forceinline__ void point(const InjAll<T>& A, int t) {
    if (t >= A.off[A.nl]) return;
    int l = 1;
    while (t >= A.off[l + 1]) ++l;
    const int idx = t - A.off[l], I = idx % A.g[l].nx, J = idx / A.g[l].nx;
    const int nx = A.g0.nx, nb = (1 << l) >= 8 ? (1 << l) / 8 : 1, step = (1 << l) >= 8 ? 8 : 1 << l;
    for (int q = 0; q < A.nsrc; ++q) {
      const T* src = A.src[q] + (size_t)(J << l) * nx + (I << l);
      T part[MAXLEV];  // part[k]: the mean of 8 2^k rows waiting for its pair
      T v = T(0);
      for (int b = 0; b < nb; ++b, src += (size_t)8 * nx) {
        T r[8];
  #pragma unroll
        for (int k = 0; k < 8; ++k) r[k] = k < step ? src[(size_t)k * nx] : T(0);
  #pragma unroll
        for (int w = 1; w < 8; w *= 2)
          if (w < step)
  #pragma unroll
            for (int k = 0; k < 8; k += 2 * w) r[k] = T(0.5) * (r[k] + r[k + w]);
        v = r[0];
        int k = 0;
        for (int n = b; n & 1; n >>= 1, ++k) v = T(0.5) * (part[k] + v);
        part[k] = v;
      }
      A.dst[l][q][idx] = v;
    }
  }
};

// Fine cell idx: e_F += P(e_C - eh_C): x linear between nodes, y linear
// between cell centres (3/4 the own coarse cell, 1/4 the next one towards the
// fine cell), the coarse correction's ghost beyond a wall mirrored (scalars)
// or odd (velocity).
template <typename T>
__device__ __forceinline__ void ch_prolong(const Lvl<T>& F, const Lvl<T>& C, int idx) {
  const int i = idx % F.g.nx, j = idx / F.g.nx;
  const int J = j >> 1;
  const int Jn = (j & 1) ? J + 1 : J - 1;
  const bool ghost = Jn < 0 || Jn >= C.g.ny;
  const int Jr = ghost ? J : Jn;
  const int I0 = i >> 1, I1 = (I0 + 1 == C.g.nx) ? 0 : I0 + 1;
  const bool odd = i & 1;
  T ev[LY::NU];
#pragma unroll
  for (int q = 0; q < LY::NU; ++q) {
    const T sg = (ghost && (q == 1 || q == 2)) ? T(-1) : T(1);
    auto dc = [&](int JJ, int II) { return C.e[q][JJ * C.g.nx + II] - C.eh[q][JJ * C.g.nx + II]; };
    T v0 = T(0.75) * dc(J, I0) + T(0.25) * sg * dc(Jr, I0);
    if (odd) v0 = T(0.5) * (v0 + T(0.75) * dc(J, I1) + T(0.25) * sg * dc(Jr, I1));
    ev[q] = F.e[q][idx] + v0;
  }
#pragma unroll
  for (int q = 0; q < LY::NU; ++q) F.e[q][idx] = ev[q];
}
template <typename T>
__global__ void __launch_bounds__(TPB) k_ch_prolong(Lvl<T> F, Lvl<T> C) {
  const int idx = blockIdx.x * blockDim.x + threadIdx.x;
  if (idx < F.g.N) ch_prolong(F, C, idx);
}

// Policy of the fused 2-D kernels (fm_fused.cuh).
template <typename TT>
struct ChPol {
  using T = TT;
  using K = PtK<T>;
  using W = WallsT<T>;
  static constexpr int NU = LY::NU, NC = 4;
  static constexpr bool WALLS = true;
  static constexpr int TILED64 = 1 << 30;  // points a multiprocessor up to which float64 sweeps on tiles (fz_tile)
  __host__ __device__ static K constants(const Phys<T>& P, T h) { return make_ptk<T, 2>(P, h); }
  __device__ static const T* coef(const Lvl<T>& L, int c) {
    return c == 0 ? L.cr : (c == 1 ? L.rk : L.cv[c - 2]);
  }
  // a staged ghost cell, from the wall row's values (p: its element of the first array)
  __device__ static void ghost(T* p, int SN, bool top, const W& w) {
    p[SN] = -p[SN];
    p[2 * SN] = -p[2 * SN];
    p[(NU + 2) * SN] = T(2) * (top ? w.ut : w.ub) - p[(NU + 2) * SN];
    p[(NU + 3) * SN] = -p[(NU + 3) * SN];
  }
  template <class A>
  __device__ static void update(const A& a, const Phys<T>& P, const K& k, const Nb& n, int fc) {
    smooth_point_a<T, KPFC, 2>(a, P, k, n, fc);
  }
  __device__ static void update_lvl(const Lvl<T>& L, const Phys<T>& P, const K& k, const W& w, int i, int j) {
    const Nb n = ch_neighbours(i, j, L.g);
    smooth_point_a<T, KPFC, 2>(ChAcc<T>{L, w.ub, w.ut}, P, k, n, n.c);
  }
  __device__ static void apply(const Lvl<T>& F, const Phys<T>& P, const K&, const W& w, int x, int y, T* M) {
    ch_applyM<T>(ChAcc<T>{F, w.ub, w.ut}, P, F.h, ch_neighbours(x, y, F.g), M);
  }
  __device__ static void apply_coarse(const Lvl<T>& F, const Lvl<T>& C, const Phys<T>& P, const K&, const W& w, int I,
                                      int J, T* M) {
    ch_applyM<T>(ChInjAcc<T>{F, ChAcc<T>{C, w.ub, w.ut}}, P, C.h, ch_neighbours(I, J, C.g), M);
  }
  __device__ static void restrict_lvl(const Lvl<T>& F, const Lvl<T>& C, int i) { ch_restrict(F, C, i); }
  __device__ static void prolong_lvl(const Lvl<T>& F, const Lvl<T>& C, const Phys<T>&, int i) { ch_prolong(F, C, i); }
};

// ---------------------------------------------------------------------------
// float64 kernels of the finest level
// ---------------------------------------------------------------------------
// value of array x at an encoded neighbour index with ghost type `type`
__device__ __forceinline__ double gv(const double* x, int i, int N, int type, const Walls64& W) {
  const double v = x[cell_of(i, N)];
  return i >= 0 ? v : ghost_of(v, type, i < -N ? W.ut : W.ub);
}

// omega^k, S, g^0 (kappa^0 = Lap_h rho^k) with the wall ghosts: 6.9 us at 256^2,
// 10.7 point by point.
template <int TX>
__global__ void __launch_bounds__(TPB) k_ch_prepare(Fields64 F, Geo G, Step64 K, Phys<double> P, Walls64 W) {
  prepare_tile<KPFC, true, TX>(F, G, K, P, blockIdx.x, W);
}

// mu^0 = psi^3/3 + alpha psi + Lap_h kappa^0 + S_mu; the blocks after the last
// point's: rho^k and omega^k down the levels.
template <typename T>
__global__ void __launch_bounds__(TPB) k_ch_prepare_mu(Fields64 F, Geo G, Step64 K, double alpha, Walls64 W,
                                                       const __grid_constant__ InjAll<T> A) {
  const int nb = (G.N + TPB - 1) / TPB;
  if ((int)blockIdx.x >= nb) {
    InjRows::point(A, (blockIdx.x - nb) * TPB + threadIdx.x);
    return;
  }
  const int idx = blockIdx.x * TPB + threadIdx.x;
  if (idx >= G.N) return;
  const int i = idx % G.nx, j = idx / G.nx;
  const Nb n = ch_neighbours(i, j, G);
  const double* ka = F.g[LY::IKA];
  const int N = G.N;
  const double nbk = gv(ka, n.m[0], N, 0, W) + gv(ka, n.p[0], N, 0, W) + gv(ka, n.m[1], N, 0, W) +
                     gv(ka, n.p[1], N, 0, W);
  const double psi = F.rho[idx] - 1.5;
  F.g[LY::IMU][idx] = psi * psi * psi * (1.0 / 3.0) + alpha * psi + (nbk - 4.0 * ka[idx]) * K.ih2 + F.S[LY::IMU][idx];
}

// r = S - N(g) in float64 with the wall ghosts; the level-0 set-up of a
// cycle and the block partial sums of r^2 (15.3 us a launch at 256^2 point by
// point with the wall rows' ghosts chosen at every load, 11.0 on the periodic
// solver's tiles, whose halo rows hold the ghosts).
template <typename T, int TX>
__global__ void __launch_bounds__(TPB, 4) k_ch_resid64(Fields64 F, Resid64Out O, Geo G, Step64 K, Phys<double> P,
                                                       Walls64 W, double* partials) {
  resid64_tile_body<KPFC, T, true, TX>(F, O, G, K, P, partials, blockIdx.x, gridDim.x, W);
}

// rho^{k+1} = S1 - (s/4h) sum_d ([rho^k u_d]_{+d} - [rho^k u_d]_{-d}) with the
// converged velocity (the explicit half is in S1), projected; skipped unless
// the solve succeeded.
__global__ void __launch_bounds__(TPB) k_ch_closure(Fields64 F, Geo G, Step64 K, double delta, Walls64 W, double* out,
                                                    const Ctl* ctl) {
  if (ctl->status != FM_OK) return;
  const int idx = blockIdx.x * blockDim.x + threadIdx.x;
  if (idx >= G.N) return;
  const int i = idx % G.nx, j = idx / G.nx;
  const Nb n = ch_neighbours(i, j, G);
  double div = 0.0;
#pragma unroll
  for (int d = 0; d < 2; ++d)
    div += gv(F.rho, n.p[d], G.N, 0, W) * gv(F.g[1 + d], n.p[d], G.N, d + 1, W) -
           gv(F.rho, n.m[d], G.N, 0, W) * gv(F.g[1 + d], n.m[d], G.N, d + 1, W);
  const double r = F.S[0][idx] - K.c_div * div;
  out[idx] = delta > 0.0 ? proj_rho(r, delta) : fabs(r);
}

// Energy densities of the PFC functional with the Neumann Laplacian, and KE.
__global__ void __launch_bounds__(TPB) k_ch_energy(const double* rho, const double* u, const double* v, Geo G,
                                                   double h, double alpha, double* partials) {
  double acc[5] = {0, 0, 0, 0, 0};
  const double ih2 = 1.0 / (h * h);
  const Walls64 W{0.0, 0.0};
  for (int idx = blockIdx.x * blockDim.x + threadIdx.x; idx < G.N; idx += gridDim.x * blockDim.x) {
    const int i = idx % G.nx, j = idx / G.nx;
    const Nb n = ch_neighbours(i, j, G);
    const double rc = rho[idx];
    acc[0] += 0.5 * rc * (u[idx] * u[idx] + v[idx] * v[idx]);
    const double psi = rc - 1.5;
    const double L = (gv(rho, n.m[0], G.N, 0, W) + gv(rho, n.p[0], G.N, 0, W) + gv(rho, n.m[1], G.N, 0, W) +
                      gv(rho, n.p[1], G.N, 0, W) - 4.0 * rc) * ih2;
    acc[1] += psi * psi * psi * psi / 12.0;
    acc[2] += 0.5 * alpha * psi * psi;
    acc[3] += 0.5 * L * L;
    acc[4] += rc * L;
  }
  block_partials<5>(acc, partials, blockIdx.x);
}

// ---------------------------------------------------------------------------
// Host driver
// ---------------------------------------------------------------------------
template <typename T>
struct ChannelSolver {
  static constexpr int NVEL = 2;

  static Walls64 walls64(const fm_state* st) { return Walls64{st->prm.u_wall[0], st->prm.u_wall[1]}; }
  static WallsT<T> wallsT(const fm_state* st) { return WallsT<T>{(T)st->prm.u_wall[0], (T)st->prm.u_wall[1]}; }
  static Step64 step64(const fm_state* st) { return make_step64(make_phys<double>(st), 1.0 / st->lv[0].h); }

  static Resid64Out out0(fm_state* st, bool cycle, double* const* r64) {
    Resid64Out O;
    memset(&O, 0, sizeof(O));
    for (int q = 0; q < LY::NU; ++q) {
      O.f0[q] = cycle ? st->lv[0].f[q] : nullptr;
      O.e0[q] = cycle ? st->lv[0].e[q] : nullptr;
      O.r64[q] = r64 ? r64[q] : nullptr;
    }
    if (cycle && st->prm.precision == FM_MIXED) {
      O.cr32 = (float*)st->lv[0].cr;
      for (int d = 0; d < 2; ++d) O.cv32[d] = (float*)st->lv[0].cv[d];
    }
    return O;
  }

  // rho^k and omega^k (which = 0) or the coefficient iterate rho, u, v
  // (which = 1) of the finest level down the hierarchy.
  static InjAll<T> injection(fm_state* st, int which) {
    InjAll<T> A;
    memset(&A, 0, sizeof(A));
    A.nl = st->nlev;
    A.g0 = st->lv[0].g;
    A.nsrc = which ? 3 : 2;
    for (int l = 0; l < st->nlev; ++l) {
      const LevelBufs& B = st->lv[l];
      void* v[3] = {which ? B.cr : B.rk, which ? B.cv[0] : B.om[0], B.cv[1]};
      for (int q = 0; q < A.nsrc; ++q) {
        if (l == 0) A.src[q] = (const T*)v[q];
        else A.dst[l][q] = (T*)v[q];
      }
      A.g[l] = B.g;
      A.off[l + 1] = l == 0 ? 0 : A.off[l] + B.g.N;
    }
    return A;
  }

  static int enqueue_prepare(fm_state* st) {
    const Geo G = st->lv[0].g;
    const Fields64 F = make_fields(st);
    if (narrow_tiles(G))
      k_ch_prepare<R64_NARROW><<<prep_tiles<R64_NARROW>(G.nx, G.ny), TPB, 0, st->stream>>>(
          F, G, step64(st), make_phys<double>(st), walls64(st));
    else
      k_ch_prepare<PT_TX><<<prep_tiles(G.nx, G.ny), TPB, 0, st->stream>>>(F, G, step64(st), make_phys<double>(st),
                                                                        walls64(st));
    FM_LAUNCHED();
    const InjAll<T> A = injection(st, 0);
    k_ch_prepare_mu<T><<<nblocks(G.N) + nblocks(A.off[st->nlev]), TPB, 0, st->stream>>>(F, G, step64(st), st->fn.alpha,
                                                                                        walls64(st), A);
    FM_LAUNCHED();
    return FM_OK;
  }

  static int launch_resid64(fm_state* st, const Resid64Out& O) {
    const Geo G = st->lv[0].g;
    const Phys<double> P = make_phys<double>(st);
    if (narrow_tiles(G))
      k_ch_resid64<T, R64_NARROW><<<st->nres, TPB, 0, st->stream>>>(make_fields(st), O, G, step64(st), P, walls64(st),
                                                                    st->partials);
    else
      k_ch_resid64<T, R64_TX><<<st->nres, TPB, 0, st->stream>>>(make_fields(st), O, G, step64(st), P, walls64(st),
                                                               st->partials);
    FM_LAUNCHED();
    return FM_OK;
  }

  static int enqueue_resid_norm(fm_state* st, int in_body, cudaGraphConditionalHandle hdl, int use_handle) {
    int rc = launch_resid64(st, out0(st, true, nullptr));
    if (rc) return rc;
    const double h = st->lv[0].h;
    const InjAll<T> A = injection(st, 1);
    k_norm_ctl<LY::NU, InjRows, T><<<1 + nblocks(A.off[st->nlev]), TPB, 0, st->stream>>>(
        st->partials, st->nres, h * h, (Ctl*)st->ctl, st->prm.tol, st->prm.max_cycles, in_body, hdl, use_handle, A);
    FM_LAUNCHED();
    return FM_OK;
  }

  // *out_in_r: on return the correction of level l is in its r buffer (1) or in e (0).
  static int vcycle(fm_state* st, int l, const Phys<T>& P, int* out_in_r) {
    using Pol = ChPol<T>;
    cudaStream_t s = st->stream;
    const WallsT<T> W = wallsT(st);
    *out_in_r = 0;
    if (l >= fz_small_from<T>(st)) {
      SmallLv<T> S;
      S.count = st->nlev - l;
      for (int q = 0; q < S.count; ++q) S.lv[q] = make_lvl<T>(st, l + q);
      FM_CUDA(fz_small<Pol>(S, P, W, st->prm, &st->launches, s));
      return FM_OK;
    }
    const Lvl<T> L = make_lvl<T>(st, l);
    if (l == st->nlev - 1) {
      FM_CUDA(fz_smooth<Pol>(L, P, W, st->prm.ncoarse, out_in_r, &st->launches, st->sms, s));
      return FM_OK;
    }
    const Lvl<T> C = make_lvl<T>(st, l + 1);
    int c_in_r = 0;
    FM_CUDA(fz_smooth<Pol>(L, P, W, st->prm.nu1, out_in_r, &st->launches, st->sms, s));
    const Lvl<T> F = fz_view(L, *out_in_r);
    FM_CUDA(fz_down<Pol>(F, C, P, W, &st->launches, s));
    const int rc = vcycle(st, l + 1, P, &c_in_r);
    if (rc) return rc;
    k_ch_prolong<T><<<nblocks(F.g.N), TPB, 0, s>>>(F, fz_view(C, c_in_r));
    FM_LAUNCHED();
    FM_CUDA(fz_smooth<Pol>(L, P, W, st->prm.nu2, out_in_r, &st->launches, st->sms, s));
    return FM_OK;
  }

  static int enqueue_body(fm_state* st, cudaGraphConditionalHandle hdl, int use_handle) {
    int in_r = 0;
    int rc = vcycle(st, 0, make_phys<T>(st), &in_r);
    if (rc) return rc;
    const Geo G = st->lv[0].g;
    Resid64Out O = out0(st, true, nullptr);
    if (in_r)  // the correction after an odd number of launches
      for (int q = 0; q < LY::NU; ++q) O.e0[q] = st->lv[0].r[q];
    k_update64<LY::NU, T><<<nblocks(G.N), TPB, 0, st->stream>>>(make_fields(st), O, G.N, st->prm.delta);
    FM_LAUNCHED();
    return enqueue_resid_norm(st, 1, hdl, use_handle);
  }

  static int enqueue_post(fm_state* st) {
    const Geo G = st->lv[0].g;
    const Ctl* ctl = (const Ctl*)st->ctl;
    k_ch_closure<<<nblocks(G.N), TPB, 0, st->stream>>>(make_fields(st), G, step64(st), st->prm.delta, walls64(st),
                                                       st->tmp, ctl);
    FM_LAUNCHED();
    Vel3W vw{{st->vel[0], st->vel[1], nullptr}};
    Vel3 gv3{{st->g[1], st->g[2], nullptr}};
    k_commit<2><<<nblocks(G.N), TPB, 0, st->stream>>>(st->rho, vw, st->tmp, gv3, G.N, (Ctl*)st->ctl);
    FM_LAUNCHED();
    FM_CUDA(cudaMemcpyAsync(st->hscal + 32, st->ctl, sizeof(Ctl), cudaMemcpyDeviceToHost, st->stream));
    return FM_OK;
  }

  static int prepare(fm_state* st) {
    int rc = enqueue_prepare(st);
    if (rc) return rc;
    FM_CUDA(cudaStreamSynchronize(st->stream));
    st->prepared = true;
    return FM_OK;
  }

  static int residual64(fm_state* st, double* const* r64, double* norm_host) {
    int rc = launch_resid64(st, out0(st, false, r64));
    if (rc) return rc;
    const double h = st->lv[0].h;
    k_norm_final<LY::NU><<<1, TPB, 0, st->stream>>>(st->partials, st->nres, h * h, st->dscal);
    FM_LAUNCHED();
    FM_CUDA(cudaMemcpyAsync(st->hscal, st->dscal, sizeof(double), cudaMemcpyDeviceToHost, st->stream));
    FM_CUDA(cudaStreamSynchronize(st->stream));
    *norm_host = st->hscal[0];
    return FM_OK;
  }
};

template <typename T>
static int dispatch(fm_state* st, int what, fm_step_info* info, const double* ri, const double* const* vi,
                    double* ro, double* const* vo, double* const* r64, double* nrm) {
  switch (what) {
    case 0: return Stepper<ChannelSolver<T>>::step(st, info);
    case 1: return Stepper<ChannelSolver<T>>::step_host(st, ri, vi, ro, vo, info);
    case 2: return ChannelSolver<T>::prepare(st);
    default: return ChannelSolver<T>::residual64(st, r64, nrm);
  }
}

static int run(fm_state* st, int what, fm_step_info* info, const double* ri, const double* const* vi, double* ro,
               double* const* vo, double* const* r64, double* nrm) {
  return st->prm.precision == FM_MIXED ? dispatch<float>(st, what, info, ri, vi, ro, vo, r64, nrm)
                                       : dispatch<double>(st, what, info, ri, vi, ro, vo, r64, nrm);
}

}  // namespace ch

int ch_step(fm_state* st, fm_step_info* info) {
  return ch::run(st, 0, info, nullptr, nullptr, nullptr, nullptr, nullptr, nullptr);
}
int ch_step_host(fm_state* st, const double* rho_in, const double* const* vel_in, double* rho_out,
                 double* const* vel_out, fm_step_info* info) {
  return ch::run(st, 1, info, rho_in, vel_in, rho_out, vel_out, nullptr, nullptr);
}
int ch_prepare(fm_state* st) { return ch::run(st, 2, nullptr, nullptr, nullptr, nullptr, nullptr, nullptr, nullptr); }
int ch_residual(fm_state* st, double* const* r64, double* norm) {
  return ch::run(st, 3, nullptr, nullptr, nullptr, nullptr, nullptr, r64, norm);
}
int ch_energy_launch(fm_state* st) {
  const Geo G = st->lv[0].g;
  ch::k_ch_energy<<<st->nblk, TPB, 0, st->stream>>>(st->rho, st->vel[0], st->vel[1], G, st->lv[0].h, st->fn.alpha,
                                                    st->partials);
  return cudaPeekAtLastError() == cudaSuccess ? FM_OK : (cudaGetLastError(), FM_ECUDA);
}

}  // namespace fm
