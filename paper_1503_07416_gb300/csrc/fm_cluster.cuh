// The V-cycle of the coarsest levels (at most SMALL_N points each) in float64
// by one thread-block cluster, used by the single-instance solver: the FP64
// path and the mixed path's float64 coarsest-grid solve.
//
// What bounds it: a warp retires one float64 instruction in 64 clocks on GB300
// however many of its lanes are active and however many are independent, and
// a multiprocessor one in 19 clocks over its four partitions (measured).  A
// point update is ~90 of them.  So
//  * the points of a level are split over the blocks of a cluster of 16 (8
//    where the device does not offer 16), 64 points to a block on the largest
//    level, one warp of each colour;
//  * the rows of the update are split over warps, hence partitions: one warp
//    takes rho (CDFT: and its chemical-potential part), one kappa and mu, one
//    each velocity row; they exchange what they need of one another in shared
//    memory.  The longest chain is then ~23 instead of ~90 instructions a pass;
//    the transfers take one thread per point and component;
//  * the inverse of the velocity block, which depends only on rho^k and
//    omega^k, is formed once per launch.
// A block keeps the records of its points (correction; CDFT: also its
// chemical-potential part), right-hand side and residual in its shared memory;
// neighbours in other blocks are read through distributed shared memory (250
// clocks); the coefficients of all points are in every block's shared memory.
// Phases (a colour pass, a residual, a transfer) are separated by the
// cluster's hardware barrier (400 clocks).  The mixed path's float32 levels are
// widened when they are staged and the correction is rounded on the way out,
// with the integer conversions, so no conversion launch is needed.
//
// Measured (32^2 and 16^2 levels, V(2,2), 4 coarse sweeps, kernel time): PFC
// 42 us, CDFT 58 us; one block on one multiprocessor (the form before) 221 and
// 396 us; points split over the cluster but a whole point update a thread, 92
// and 96 us; kappa and mu finished by the rho role, 46 us.
#pragma once

#include "fm_device.cuh"

namespace fm {

constexpr int CL_TPB = 384;  // twelve warps: two to four sets of the 3 to 5 roles of warps
constexpr int CL_MAX = 16;   // blocks of a cluster
constexpr size_t CL_SMEM_MAX = 128 * 1024;  // the largest plan: PFC 16 x 16 x 4 on 8 blocks, 115,456 bytes

template <int KIND, int DIM>
struct ClDim {
  using LY = Layout<KIND, DIM>;
  static constexpr int NU = LY::NU;
  static constexpr int NR = NU + (KIND == KCDFT ? 1 : 0);  // doubles of a point's record: e, cdft_mc(e)
  static constexpr int NCO = 2 + DIM + LY::NOM;            // coefficients: rho^k, rho, u (DIM), omega^k (NOM)
  static constexpr int NI = DIM == 2 ? 2 : 9;              // the velocity block's inverse: a I + b J, or a matrix
  static constexpr int NV = NI + 1;                        // and s rho^k / (4 h)
  static constexpr int R = 1 + DIM + (KIND == KPFC ? 1 : 0);  // roles: rho, velocities, PFC: kappa and mu
  static constexpr int SETS = CL_TPB / 32 / R;             // warps of each role in a block
};

// --------------------------------------------------------------------------
// The point update by roles
// --------------------------------------------------------------------------
// The point a thread updates: its index, its neighbours' indices and records.
template <int DIM>
struct RolePt {
  int idx;  // -1: none
  int ni[2 * DIM];
  const double* nr[2 * DIM];  // m, p of each direction
};
// What the rho role (a: rho) and the kappa and mu role (a, b: their neighbour
// sums) carry from the first half of an update to the second.
struct RoleRegs {
  double a, b;
};

// smooth_point_a's update of the point t in slot p of a pass, split over the
// roles; a block barrier between the halves.  An accessor A gives rk(i),
// cr(i), cv(d, i), f(q, i), the point's own record recp(i) and velocity-block
// inverse ivp(i), keep_mc(i, e0, ce), and xch(k, p): value k of slot p in the
// exchange area (0 .. DIM - 1 velocity right-hand sides, DIM the new rho,
// DIM + 1 its part of mu).  Every value of another point is loaded before the first
// use, so that remote reads overlap.
template <int KIND, int DIM>
struct RoleUpdate {
  using D = ClDim<KIND, DIM>;
  using LY = Layout<KIND, DIM>;
  static constexpr int AUX = 1 + DIM;

  static __device__ __forceinline__ double sum(const double (&v)[2 * DIM]) {
    double s = v[0] + v[1];
#pragma unroll
    for (int k = 2; k < 2 * DIM; ++k) s += v[k];
    return s;
  }

  template <class A>
  static __device__ __forceinline__ void first(const A& a, const Phys<double>& P, const PtK<double>& K,
                                               const RolePt<DIM>& t, int p, int role, RoleRegs& g) {
    if (role == 0) {
      double u[2 * DIM], r[2 * DIM];
#pragma unroll
      for (int k = 0; k < 2 * DIM; ++k) {
        u[k] = t.nr[k][1 + k / 2];
        r[k] = a.rk(t.ni[k]);
      }
      const double crc = a.cr(t.idx), f0 = a.f(0, t.idx);
      double div = 0;
#pragma unroll
      for (int d = 0; d < DIM; ++d) div += r[2 * d + 1] * u[2 * d + 1] - r[2 * d] * u[2 * d];
      double er = f0 - K.c_div * div;
      const double x = crc + er;
      if (x <= K.proj) er = proj_rho(x, P.delta) - crc;  // Sec. 6 projection
      if constexpr (KIND == KPFC) {
        const double psi = crc - 1.5;
        a.xch(DIM, p) = er;
        a.xch(DIM + 1, p) = er * (psi * psi + psi * er + er * er * (1.0 / 3.0)) + P.alpha * er;
      }
      g.a = er;
    } else if (role == AUX) {
      if constexpr (KIND == KPFC) {
        double v[2 * DIM], k2[2 * DIM];
#pragma unroll
        for (int k = 0; k < 2 * DIM; ++k) {
          v[k] = t.nr[k][0];
          k2[k] = t.nr[k][LY::IKA];
        }
        g.a = a.f(LY::IKA, t.idx) + sum(v) * K.ih2;
        g.b = a.f(LY::IMU, t.idx) + sum(k2) * K.ih2;
      }
    } else {
#pragma unroll
      for (int d = 0; d < DIM; ++d)
        if (role == 1 + d) {
          double v[2 * DIM], q[2], m[2], c[2][DIM], u[2][DIM];
#pragma unroll
          for (int k = 0; k < 2 * DIM; ++k) v[k] = t.nr[k][1 + d];
#pragma unroll
          for (int k = 0; k < 2; ++k) {
            m[k] = t.nr[2 * d + k][KIND == KPFC ? LY::IMU : D::NR - 1];
#pragma unroll
            for (int b = 0; b < DIM; ++b) {
              u[k][b] = t.nr[2 * d + k][1 + b];
              c[k][b] = a.cv(b, t.ni[2 * d + k]);
            }
          }
          const double fd = a.f(1 + d, t.idx), cs = a.ivp(t.idx)[D::NI];
#pragma unroll
          for (int k = 0; k < 2; ++k) {
            q[k] = 0;
#pragma unroll
            for (int b = 0; b < DIM; ++b) q[k] += u[k][b] * (2.0 * c[k][b] + u[k][b]);
          }
          a.xch(d, p) = fd - cs * ((q[1] - q[0]) + 2.0 * (m[1] - m[0])) + K.c_v * sum(v);
        }
    }
  }

  template <class A>
  static __device__ __forceinline__ void second(const A& a, const Phys<double>& P, const PtK<double>& K,
                                                const RolePt<DIM>& t, int p, int role, const RoleRegs& g) {
    const double w = P.w;
    double* eo = a.recp(t.idx);
    if (role == 0) {
      const double er = (1.0 - w) * g.a + w * eo[0];
      eo[0] = er;
      if constexpr (KIND == KCDFT) a.keep_mc(t.idx, er, P.ce);
    } else if (role == AUX) {
      if constexpr (KIND == KPFC) {
        const double c4 = 2.0 * DIM * K.ih2;
        const double ek = g.a - c4 * a.xch(DIM, p);
        const double em = g.b + a.xch(DIM + 1, p) - c4 * ek;
        eo[LY::IKA] = (1.0 - w) * ek + w * eo[LY::IKA];
        eo[LY::IMU] = (1.0 - w) * em + w * eo[LY::IMU];
      }
    } else if (role <= DIM) {
      const double* v = a.ivp(t.idx);
      double eg;
      if constexpr (DIM == 2)
        eg = role == 1 ? v[0] * a.xch(0, p) + v[1] * a.xch(1, p) : v[0] * a.xch(1, p) - v[1] * a.xch(0, p);
      else
        eg = v[3 * role - 3] * a.xch(0, p) + v[3 * role - 2] * a.xch(1, p) + v[3 * role - 1] * a.xch(2, p);
      eo[role] = (1.0 - w) * eg + w * eo[role];
    }
  }
};

// The inverse of the velocity block at a point (see smooth_point_a), and s
// rho^k / (4 h) after it.
template <int DIM>
__device__ __forceinline__ void invert_block(const PtK<double>& K, double rk, const double* om, double* v) {
  const double Ad = rk + K.c_ad, bs = K.c_b * rk;
  if constexpr (DIM == 2) {
    const double b = bs * om[0], inv = 1.0 / (Ad * Ad + b * b);
    v[0] = Ad * inv;
    v[1] = b * inv;
    v[2] = 0.25 * K.c_sih * rk;
  } else {
    v[9] = 0.25 * K.c_sih * rk;
    const double b[3] = {bs * om[0], bs * om[1], bs * om[2]};
    const double inv = 1.0 / (Ad * (Ad * Ad + b[0] * b[0] + b[1] * b[1] + b[2] * b[2]));
#pragma unroll
    for (int r = 0; r < 3; ++r)
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        // Ad^2 I - Ad [b]_x + b b^T, [b]_x rhs = b x rhs
        const double x = r == c ? Ad * Ad : ((c - r + 3) % 3 == 1 ? Ad : -Ad) * b[3 - r - c];
        v[3 * r + c] = (x + b[r] * b[c]) * inv;
      }
  }
}

// --------------------------------------------------------------------------
// The V-cycle of the small levels by a cluster
// --------------------------------------------------------------------------
// Shared-memory offsets (doubles) and constants of the levels; the same in
// every block.  Block r owns the points [r << sh, (r + 1) << sh) of a level.
struct ClPlan {
  int sh[MAXSMALL];
  int rec[MAXSMALL], f[MAXSMALL], r[MAXSMALL], eh[MAXSMALL], iv[MAXSMALL], co[MAXSMALL];
  int rhs;  // values the roles exchange (velocity right-hand sides, kappa and mu sums) at a pass's points
  PtK<double> K[MAXSMALL];
};

template <typename TS, int KIND, int DIM>
static size_t cl_plan(const SmallLv<TS>& S, const Phys<double>& P, const double* h, int nblocks, ClPlan& M) {
  using D = ClDim<KIND, DIM>;
  int off = 0;
  for (int l = 0; l < S.count; ++l) {
    const int N = S.lv[l].g.N;
    int sh = 1;
    while (((long long)nblocks << sh) < N) ++sh;
    M.sh[l] = sh;
    const int n = 1 << sh;
    M.rec[l] = off; off += n * D::NR;
    M.f[l] = off; off += n * D::NU;
    M.r[l] = off; off += n * D::NU;
    M.eh[l] = off; off += n * D::NU;
    M.iv[l] = off; off += n * D::NV;
    M.co[l] = off; off += N * D::NCO;
    M.K[l] = make_ptk<double, DIM>(P, h[l]);
  }
  M.rhs = off;
  off += (DIM + 2) << (M.sh[0] - 1);  // the largest level's points of one colour
  return (size_t)off * sizeof(double);
}

// The address of p (this block's shared memory) in block `rank` of the cluster.
__device__ __forceinline__ const double* cl_map(const double* p, unsigned rank) {
  unsigned long long q;
  asm("mapa.u64 %0, %1, %2;" : "=l"(q) : "l"(p), "r"(rank));
  return reinterpret_cast<const double*>(q);
}
__device__ __forceinline__ unsigned cl_rank() {
  unsigned r;
  asm("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}
__device__ __forceinline__ void cl_sync() {
  asm volatile("barrier.cluster.arrive.release;\nbarrier.cluster.wait.acquire;\n" ::: "memory");
}

// One level: geometry, constants, this block's slabs (record of a point: NR
// values; f, r, eh: component q at q << sh; iv: NV values a point) and the
// coefficients co of all points.
struct ClLvl {
  Geo g;
  int sh;
  double *rec, *f, *r, *eh, *iv, *co;
  double* rhs;
};

// Values of a level by point index: records of any point through the cluster,
// f of this block's points, coefficients from the block's copy.
template <int KIND, int DIM>
struct ClAcc {
  using D = ClDim<KIND, DIM>;
  using LY = Layout<KIND, DIM>;
  const ClLvl& L;
  __device__ __forceinline__ int own(int i) const { return i & ((1 << L.sh) - 1); }
  __device__ __forceinline__ const double* rec(int i) const { return cl_map(L.rec + own(i) * D::NR, i >> L.sh); }
  __device__ __forceinline__ double e(int q, int i) const { return rec(i)[q]; }
  __device__ __forceinline__ double f(int q, int i) const { return L.f[(q << L.sh) + own(i)]; }
  __device__ __forceinline__ double rk(int i) const { return L.co[i]; }
  __device__ __forceinline__ double cr(int i) const { return L.co[L.g.N + i]; }
  __device__ __forceinline__ double cv(int d, int i) const { return L.co[(2 + d) * L.g.N + i]; }
  __device__ __forceinline__ double om(int d, int i) const { return L.co[(2 + DIM + d) * L.g.N + i]; }
  __device__ __forceinline__ double* recp(int i) const { return L.rec + own(i) * D::NR; }
  __device__ __forceinline__ const double* ivp(int i) const { return L.iv + own(i) * D::NV; }
  __device__ __forceinline__ double& xch(int k, int p) const { return L.rhs[(k << (L.sh - 1)) + p]; }
  // the chemical-potential part of point i's current correction (CDFT)
  __device__ __forceinline__ void keep_mc(int i, double e0, double ce) const {
    recp(i)[D::NR - 1] = cdft_mc<double>(e0, cr(i), ce);
  }
  __device__ __forceinline__ double nbs(int q, const Nb& n) const {
    double s = e(q, n.m[0]) + e(q, n.p[0]) + e(q, n.m[1]) + e(q, n.p[1]);
    if constexpr (DIM == 3) s += e(q, n.m[2]) + e(q, n.p[2]);
    return s;
  }
  __device__ __forceinline__ double div(const Nb& n) const {
    double s = 0;
#pragma unroll
    for (int d = 0; d < DIM; ++d) s += rk(n.p[d]) * e(1 + d, n.p[d]) - rk(n.m[d]) * e(1 + d, n.m[d]);
    return s;
  }
  // 1/4 the difference along d of the correction's kinetic part, 1/2 that of
  // its chemical potential (see qcorr, mcorr)
  __device__ __forceinline__ double grad(const Nb& n, int d) const {
    double q[2], m[2];
#pragma unroll
    for (int k = 0; k < 2; ++k) {
      const int i = k ? n.m[d] : n.p[d];
      const double* r = rec(i);
      q[k] = 0;
#pragma unroll
      for (int c = 0; c < DIM; ++c) q[k] += r[1 + c] * (2.0 * cv(c, i) + r[1 + c]);
      m[k] = r[KIND == KPFC ? LY::IMU : D::NR - 1];
    }
    return 0.25 * (q[0] - q[1]) + 0.5 * (m[0] - m[1]);
  }
};

template <typename TS, int KIND, int DIM>
struct ClCycle {
  using D = ClDim<KIND, DIM>;
  using LY = Layout<KIND, DIM>;
  using Acc = ClAcc<KIND, DIM>;
  using Up = RoleUpdate<KIND, DIM>;
  using Pt = RolePt<DIM>;
  static constexpr int NU = D::NU;

  // fn(idx, p, role) for this block's points by the warps of each role; p
  // numbers them within the block.
  template <class F>
  static __device__ __forceinline__ void points(const ClLvl& L, F&& fn) {
    const int n = 1 << L.sh, first = (int)cl_rank() << L.sh;
    const int warp = threadIdx.x >> 5, set = warp / D::R;
    if (set >= D::SETS) return;
    for (int p = set * 32 + (threadIdx.x & 31); p < n && first + p < L.g.N; p += 32 * D::SETS)
      fn(first + p, p, warp - set * D::R);
  }
  // fn(idx, p, q) for this block's points and every component q.
  template <class F>
  static __device__ __forceinline__ void components(const ClLvl& L, F&& fn) {
    const int n = 1 << L.sh, first = (int)cl_rank() << L.sh;
    for (int t = threadIdx.x; t < n * NU; t += CL_TPB) {
      const int p = t & (n - 1);
      if (first + p < L.g.N) fn(first + p, p, t >> L.sh);
    }
  }
  static __device__ __forceinline__ Nb nb(const ClLvl& L, int idx) {
    int i, j, k;
    coords(idx, L.g, i, j, k);
    return neighbours(i, j, k, L.g);
  }

  // The velocity block's inverse at this block's points (see smooth_point_a).
  static __device__ __forceinline__ void invert(const ClLvl& L, const PtK<double>& K) {
    const Acc a{L};
    const int n = 1 << L.sh, first = (int)cl_rank() << L.sh;
    for (int p = threadIdx.x; p < n && first + p < L.g.N; p += CL_TPB) {
      const int i = first + p;
      double om[LY::NOM];
#pragma unroll
      for (int d = 0; d < LY::NOM; ++d) om[d] = a.om(d, i);
      invert_block<DIM>(K, a.rk(i), om, L.iv + p * D::NV);
    }
  }

  static __device__ __forceinline__ Pt point(const ClLvl& L, int p, int c) {
    Pt t;
    t.idx = -1;
    const int first = (int)cl_rank() << L.sh;
    int idx = first + 2 * p;
    if (p < 0 || p >= 1 << (L.sh - 1) || idx >= L.g.N) return t;
    const int row = idx / L.g.nx;  // idx has even x: its row's point of colour c is idx or idx + 1
    idx += (row % L.g.ny + row / L.g.ny + c) & 1;
    t.idx = idx;
    const Nb n = nb(L, idx);
    const Acc a{L};
#pragma unroll
    for (int d = 0; d < DIM; ++d) {
      t.ni[2 * d] = n.m[d];
      t.ni[2 * d + 1] = n.p[d];
    }
#pragma unroll
    for (int k = 0; k < 2 * DIM; ++k) t.nr[k] = a.rec(t.ni[k]);
    return t;
  }
  static __device__ __forceinline__ void pass(const ClLvl& L, const Phys<double>& P, const PtK<double>& K,
                                              const Pt& t, int p, int role) {
    const Acc a{L};
    RoleRegs g;
    if (t.idx >= 0) Up::first(a, P, K, t, p, role, g);
    __syncthreads();
    if (t.idx >= 0) Up::second(a, P, K, t, p, role, g);
    cl_sync();
  }

  // A block has at most 64 points of a colour (1,024 points, 8 blocks): one a
  // thread of each role.
  static __device__ __forceinline__ void smooth(const ClLvl& L, const Phys<double>& P, const PtK<double>& K,
                                                int iters) {
    static_assert(SMALL_N / 8 / 2 <= 32 * D::SETS, "a thread updates one point of a pass");
    const int warp = threadIdx.x >> 5, set = warp / D::R, role = warp - set * D::R;
    const int p = set < D::SETS ? set * 32 + (int)(threadIdx.x & 31) : -1;
    const Pt red = point(L, p, 0), black = point(L, p, 1);
    for (int it = 0; it < iters; ++it) {
      pass(L, P, K, red, p, role);
      pass(L, P, K, black, p, role);
    }
  }

  // out(q, p, M_q) at this block's points: M(e) = N(c + e) - N(c) (see applyM).
  template <class F>
  static __device__ __forceinline__ void apply_M(const ClLvl& L, const Phys<double>& P, const PtK<double>& K, F&& out) {
    const Acc a{L};
    points(L, [&](int idx, int p, int role) {
      const Nb n = nb(L, idx);
      const double* ec = L.rec + p * D::NR;
      if (role == 0) {
        out(0, p, ec[0] + K.c_div * a.div(n));
      } else if (role == 1 + DIM) {
        if constexpr (KIND == KPFC) {
          const double er = ec[0], ek = ec[LY::IKA], psi = a.cr(idx) - 1.5;
          out(LY::IMU, p, ec[LY::IMU] - er * (psi * psi + psi * er + er * er * (1.0 / 3.0)) - P.alpha * er -
                              (a.nbs(LY::IKA, n) - 2.0 * DIM * ek) * K.ih2);
          out(LY::IKA, p, ek - (a.nbs(0, n) - 2.0 * DIM * er) * K.ih2);
        }
      } else {
#pragma unroll
        for (int d = 0; d < DIM; ++d)
          if (role == 1 + d) {
            double wx;
            if constexpr (DIM == 2)
              wx = d == 0 ? -a.om(0, idx) * ec[2] : a.om(0, idx) * ec[1];
            else
              wx = a.om((d + 1) % 3, idx) * ec[1 + (d + 2) % 3] - a.om((d + 2) % 3, idx) * ec[1 + (d + 1) % 3];
            const double rkc = a.rk(idx);
            out(1 + d, p, rkc * ec[1 + d] + K.c_b * rkc * wx + K.c_sih * rkc * a.grad(n, d) -
                              K.c_v * (a.nbs(1 + d, n) - 2.0 * DIM * ec[1 + d]));
          }
      }
    });
  }

  // r = f - M(e); f_C = FW(r), e_C = eh_C = inject(e); f_C += M_C(e_C).
  static __device__ __forceinline__ void down(const ClLvl& L, const ClLvl& C, const Phys<double>& P,
                                              const PtK<double>& K, const PtK<double>& KC) {
    const Acc a{L};
    apply_M(L, P, K, [&](int q, int p, double m) { L.r[(q << L.sh) + p] = L.f[(q << L.sh) + p] - m; });
    cl_sync();
    components(C, [&](int idx, int p, int q) {
      int I, J, Kz;
      coords(idx, C.g, I, J, Kz);
      const int fi = 2 * I, fj = 2 * J, fk = DIM == 3 ? 2 * Kz : 0;
      int xs[3], ys[3], zs[3];  // (sides are even: 2I + 1 does not wrap)
      xs[0] = fi == 0 ? L.g.nx - 1 : fi - 1; xs[1] = fi; xs[2] = fi + 1;
      ys[0] = fj == 0 ? L.g.ny - 1 : fj - 1; ys[1] = fj; ys[2] = fj + 1;
      zs[0] = fk == 0 ? L.g.nz - 1 : fk - 1; zs[1] = fk; zs[2] = fk + 1;
      double acc = 0;
#pragma unroll
      for (int c = 0; c < (DIM == 3 ? 3 : 1); ++c)
#pragma unroll
        for (int b = 0; b < 3; ++b) {
          double row[3];
#pragma unroll
          for (int x = 0; x < 3; ++x) {
            const int g = ((DIM == 3 ? zs[c] : 0) * L.g.ny + ys[b]) * L.g.nx + xs[x];
            row[x] = *cl_map(L.r + (q << L.sh) + a.own(g), g >> L.sh);
          }
          const double w = (DIM == 3 && c == 1 ? 2.0 : 1.0) * (b == 1 ? 2.0 : 1.0);
          acc += w * (row[0] + 2.0 * row[1] + row[2]);
        }
      const double ev = a.e(q, (fk * L.g.ny + fj) * L.g.nx + fi);
      C.f[(q << C.sh) + p] = acc * (DIM == 3 ? 1.0 / 64.0 : 1.0 / 16.0);
      C.eh[(q << C.sh) + p] = ev;
      C.rec[p * D::NR + q] = ev;
      if constexpr (KIND == KCDFT) {
        const Acc ac{C};
        if (q == 0) ac.keep_mc(idx, ev, P.ce);
      }
    });
    cl_sync();
    apply_M(C, P, KC, [&](int q, int p, double m) { C.f[(q << C.sh) + p] += m; });
    cl_sync();  // the first colour pass overwrites corrections M_C reads
  }

  // e += P(e_C - eh_C), with prolong_point's projection.
  static __device__ __forceinline__ void up(const ClLvl& L, const ClLvl& C, const Phys<double>& P) {
    const Acc a{L};
    const Acc ac{C};
    components(L, [&](int idx, int p, int q) {
      int i, j, k;
      coords(idx, L.g, i, j, k);
      double acc = 0;
      for (int c = 0; c <= (DIM == 3 ? (k & 1) : 0); ++c)
        for (int b = 0; b <= (j & 1); ++b)
          for (int x = 0; x <= (i & 1); ++x) {
            const int X = (i >> 1) + x == C.g.nx ? 0 : (i >> 1) + x;
            const int Y = (j >> 1) + b == C.g.ny ? 0 : (j >> 1) + b;
            const int Z = (k >> 1) + c == C.g.nz ? 0 : (k >> 1) + c;
            const int g = (Z * C.g.ny + Y) * C.g.nx + X;
            acc += ac.e(q, g) - *cl_map(C.eh + (q << C.sh) + ac.own(g), g >> C.sh);
          }
      double w = (i & 1) ? 0.5 : 1.0;
      if (j & 1) w *= 0.5;
      if (DIM == 3 && (k & 1)) w *= 0.5;
      double ev = L.rec[p * D::NR + q] + w * acc;
      if (q == 0 && P.delta > 0.0) {
        const double c = a.cr(idx), x = c + ev;
        if (x <= proj_threshold<double>(P.delta)) ev = proj_rho(x, P.delta) - c;
      }
      L.rec[p * D::NR + q] = ev;
      if constexpr (KIND == KCDFT) {
        if (q == 0) a.keep_mc(idx, ev, P.ce);
      }
    });
    cl_sync();
  }
};

template <typename TS, int KIND, int DIM>
__global__ void __launch_bounds__(CL_TPB) k_vcycle_cluster(const __grid_constant__ SmallLv<TS> S,
                                                           const __grid_constant__ ClPlan M, Phys<double> P, int nu1,
                                                           int nu2, int ncoarse) {
  using D = ClDim<KIND, DIM>;
  using C = ClCycle<TS, KIND, DIM>;
  constexpr int NU = D::NU;
  double* sm = reinterpret_cast<double*>(fm_dyn_smem);
  const int nl = S.count;
  auto level = [&](int l) {
    return ClLvl{S.lv[l].g,     M.sh[l],        sm + M.rec[l], sm + M.f[l],  sm + M.r[l],
                 sm + M.eh[l],  sm + M.iv[l],   sm + M.co[l],  sm + M.rhs};
  };
  for (int l = 0; l < nl; ++l) {
    const Lvl<TS>& G = S.lv[l];
    const int N = G.g.N;
    double* co = sm + M.co[l];
    for (int i = threadIdx.x; i < N; i += CL_TPB) {
      TS v[D::NCO];
      v[0] = G.rk[i];
      v[1] = G.cr[i];
#pragma unroll
      for (int d = 0; d < DIM; ++d) v[2 + d] = G.cv[d][i];
#pragma unroll
      for (int d = 0; d < D::LY::NOM; ++d) v[2 + DIM + d] = G.om[d][i];
#pragma unroll
      for (int q = 0; q < D::NCO; ++q) co[q * N + i] = from_t<TS>(v[q]);
    }
  }
  const ClLvl L0 = level(0);
  const int n0 = 1 << L0.sh, first = (int)cl_rank() << L0.sh;
  for (int t = threadIdx.x; t < n0 * NU; t += CL_TPB) {
    const int p = t & (n0 - 1), q = t >> L0.sh;
    if (first + p < L0.g.N) {
      L0.rec[p * D::NR + q] = from_t<TS>(S.lv[0].e[q][first + p]);
      L0.f[t] = from_t<TS>(S.lv[0].f[q][first + p]);
    }
  }
  __syncthreads();
  for (int l = 0; l < nl; ++l) C::invert(level(l), M.K[l]);
  if constexpr (KIND == KCDFT) {
    const ClAcc<KIND, DIM> a{L0};
    for (int p = threadIdx.x; p < n0 && first + p < L0.g.N; p += CL_TPB)
      a.keep_mc(first + p, L0.rec[p * D::NR], P.ce);
  }
  cl_sync();
  for (int l = 0; l + 1 < nl; ++l) {
    C::smooth(level(l), P, M.K[l], nu1);
    C::down(level(l), level(l + 1), P, M.K[l], M.K[l + 1]);
  }
  C::smooth(level(nl - 1), P, M.K[nl - 1], ncoarse);
  for (int l = nl - 2; l >= 0; --l) {
    C::up(level(l), level(l + 1), P);
    C::smooth(level(l), P, M.K[l], nu2);
  }
  // every block has passed a cluster barrier after the last remote read of its memory
  for (int t = threadIdx.x; t < n0 * NU; t += CL_TPB) {
    const int p = t & (n0 - 1), q = t >> L0.sh;
    if (first + p < L0.g.N) S.lv[0].e[q][first + p] = to_t<TS>(L0.rec[p * D::NR + q]);
  }
}

// --------------------------------------------------------------------------
// Sweeps of a larger 2-D coarsest level
// --------------------------------------------------------------------------
// NS (1 or 2) red-black sweeps in float64 of a float32 level on 8 x 4 tiles,
// one tile a block, the point updates by roles: red on the tile and its rings
// 2 NS - 1, black one ring less, and so on, as in the tile form of the fused
// sweeps.  The tile and its halo are widened as they are staged (integer
// conversions); the correction is read from ein (float32 or float64) and the
// tile's is written to eout (another buffer).  The launch is bound by the
// float64 pipe: 70, 48, 30 and 16 points a pass for two sweeps, so 3, 2, 1
// and 1 warps of each role; smaller tiles recompute more than the idle
// multiprocessors give, larger ones leave multiprocessors without a tile (a
// 64^2 level has 128 tiles).  Two sweeps of a 64^2 level, kernel time: 12 us
// (PFC) and 15 us (CDFT) against 32 and 37 us for four colour launches between
// two conversions.
constexpr int CT_TX = 8, CT_TY = 4, CT_SETS = 3;
// Swept on tiles: levels of at most two tiles a multiprocessor.  One block more
// starts a third round, and the recomputed halo (2.6 point updates for one; far
// more on a level narrower than a tile) then costs more than the launches.  A
// cycle of four sweeps of a level of its own, on tiles and as colour launches:
// 128 x 64 (256 tiles) 50.0 / 59.9 us, 128 x 76 (304) 56.2 / 65.0, 110 x 90 (322) 69.1 /
// 66.0, 2 x 1024 (256) 130 / 139, 2 x 4096 (1,024) 194 / 144; CDFT 4096 x 2 (512) 118 / 103.
__host__ __device__ constexpr int ct_tiles(const Geo& g) {
  return ((g.nx + CT_TX - 1) / CT_TX) * ((g.ny + CT_TY - 1) / CT_TY);
}

template <int KIND>
__host__ __device__ constexpr int ct_threads() { return ClDim<KIND, 2>::R * CT_SETS * 32; }

template <int KIND, int NS>
struct CtSmem {
  static constexpr int H = 2 * NS, SW = CT_TX + 2 * H, SN = SW * (CT_TY + 2 * H);
  using D = ClDim<KIND, 2>;
  double rec[SN * D::NR], iv[SN * D::NV], co[4][SN], f[D::NU][SN], x[4][CT_SETS * 32];
};

template <int KIND, int NS>
struct CtAcc {
  using D = ClDim<KIND, 2>;
  CtSmem<KIND, NS>& S;
  __device__ __forceinline__ double rk(int i) const { return S.co[0][i]; }
  __device__ __forceinline__ double cr(int i) const { return S.co[1][i]; }
  __device__ __forceinline__ double cv(int d, int i) const { return S.co[2 + d][i]; }
  __device__ __forceinline__ double f(int q, int i) const { return S.f[q][i]; }
  __device__ __forceinline__ double* recp(int i) const { return S.rec + i * D::NR; }
  __device__ __forceinline__ const double* ivp(int i) const { return S.iv + i * D::NV; }
  __device__ __forceinline__ double& xch(int k, int p) const { return S.x[k][p]; }
  __device__ __forceinline__ void keep_mc(int i, double e0, double ce) const {
    recp(i)[D::NR - 1] = cdft_mc<double>(e0, cr(i), ce);
  }
};

template <typename T>
struct CtPtr {
  T* p[5];
};

template <int KIND, int NS, typename EI, typename EO>
__global__ void __launch_bounds__(ct_threads<KIND>()) k_coarse64_tile(const __grid_constant__ Lvl<float> L,
                                                                      CtPtr<const EI> ein, CtPtr<EO> eout,
                                                                      Phys<double> P, PtK<double> K, int ntx) {
  using D = ClDim<KIND, 2>;
  using SM = CtSmem<KIND, NS>;
  using Up = RoleUpdate<KIND, 2>;
  constexpr int NU = D::NU, H = SM::H, SW = SM::SW, SN = SM::SN, TPBK = ct_threads<KIND>();
  static_assert((CT_TX / 2 + 2 * NS - 1) * (CT_TY + 4 * NS - 2) <= CT_SETS * 32, "a thread updates one point of a pass");
  __shared__ SM S;
  const CtAcc<KIND, NS> a{S};
  const int nx = L.g.nx, ny = L.g.ny;
  const int x0 = (blockIdx.x % ntx) * CT_TX, y0 = (blockIdx.x / ntx) * CT_TY;
  // two threads a cell: the correction and densities, the right-hand side and velocities
  for (int t = threadIdx.x; t < 2 * SN; t += TPBK) {
    const int c = t < SN ? t : t - SN;
    const int g = wrapi(y0 - H + c / SW, ny) * nx + wrapi(x0 - H + c % SW, nx);
    if (t < SN) {
      EI e[NU];
      const float rk = L.rk[g], cr = L.cr[g];
#pragma unroll
      for (int q = 0; q < NU; ++q) e[q] = ein.p[q][g];
#pragma unroll
      for (int q = 0; q < NU; ++q) S.rec[c * D::NR + q] = from_t<EI>(e[q]);
      S.co[0][c] = widen(rk);
      S.co[1][c] = widen(cr);
    } else {
      float f[NU];
      const float u = L.cv[0][g], v = L.cv[1][g], om = L.om[0][g], rk = L.rk[g];
#pragma unroll
      for (int q = 0; q < NU; ++q) f[q] = L.f[q][g];
#pragma unroll
      for (int q = 0; q < NU; ++q) S.f[q][c] = widen(f[q]);
      S.co[2][c] = widen(u);
      S.co[3][c] = widen(v);
      const double w = widen(om);
      invert_block<2>(K, widen(rk), &w, S.iv + c * D::NV);
    }
  }
  __syncthreads();
  if constexpr (KIND == KCDFT) {  // the black cells the first pass reads
    for (int t = threadIdx.x; t < SN / 2; t += TPBK) {
      const int ly = t / (SW / 2), lx = 2 * (t - ly * (SW / 2)) + ((x0 + y0 + ly + 1) & 1);
      const int c = ly * SW + lx;
      a.keep_mc(c, S.rec[c * D::NR], P.ce);
    }
    __syncthreads();
  }
  const int warp = threadIdx.x >> 5, role = warp % D::R;
  const int p = (warp / D::R) * 32 + (threadIdx.x & 31);
#pragma unroll
  for (int pass = 0; pass < 2 * NS; ++pass) {
    const int ring = 2 * NS - 1 - pass, hw = CT_TX / 2 + ring;
    RolePt<2> t;
    RoleRegs g;
    t.idx = -1;
    if (p < hw * (CT_TY + 2 * ring)) {
      const int ry = p / hw;
      const int rx = 2 * (p - ry * hw) + (((pass & 1) + x0 + ring + y0 - ring + ry) & 1);
      t.idx = (H - ring + ry) * SW + H - ring + rx;
      t.ni[0] = t.idx - 1;
      t.ni[1] = t.idx + 1;
      t.ni[2] = t.idx - SW;
      t.ni[3] = t.idx + SW;
#pragma unroll
      for (int k = 0; k < 4; ++k) t.nr[k] = S.rec + t.ni[k] * D::NR;
      Up::first(a, P, K, t, p, role, g);
    }
    __syncthreads();
    if (t.idx >= 0) Up::second(a, P, K, t, p, role, g);
    __syncthreads();
  }
  for (int t = threadIdx.x; t < CT_TX * CT_TY * NU; t += TPBK) {
    const int q = t / (CT_TX * CT_TY), c = t % (CT_TX * CT_TY);
    const int gx = x0 + c % CT_TX, gy = y0 + c / CT_TX;
    if (gx < nx && gy < ny)
      eout.p[q][gy * nx + gx] = to_t<EO>(S.rec[((H + c / CT_TX) * SW + H + c % CT_TX) * D::NR + q]);
  }
}

}  // namespace fm
