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
//    takes rho, kappa and mu (CDFT: rho and its chemical-potential part), one
//    the neighbour sums of kappa and mu, one each velocity row; they exchange
//    what they need of one another in shared memory.  The longest chain is
//    then ~22 instead of ~90 instructions a pass; the transfers take one
//    thread per point and component;
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
// 46 us, CDFT 58 us; one block on one multiprocessor (the form before) 221 and
// 396 us; points split over the cluster but a whole point update a thread, 92
// and 96 us.
#pragma once

#include "fm_device.cuh"

namespace fm {

constexpr int CL_TPB = 384;  // twelve warps: two to four sets of the 3 to 5 roles of warps
constexpr int CL_MAX = 16;   // blocks of a cluster
constexpr size_t CL_SMEM_MAX = 128 * 1024;  // 3-D, 8 blocks: 8 coefficients x ~1,200 points + the slabs, under 110 KB

template <int KIND, int DIM>
struct ClDim {
  using LY = Layout<KIND, DIM>;
  static constexpr int NU = LY::NU;
  static constexpr int NR = NU + (KIND == KCDFT ? 1 : 0);  // doubles of a point's record: e, cdft_mc(e)
  static constexpr int NCO = 2 + DIM + LY::NOM;            // coefficients: rho^k, rho, u (DIM), omega^k (NOM)
  static constexpr int NV = DIM == 2 ? 2 : 9;              // the velocity block's inverse: a I + b J, or a matrix
  static constexpr int R = 1 + DIM + (KIND == KPFC ? 1 : 0);  // roles: rho (kappa, mu), velocities, PFC sums
  static constexpr int SETS = CL_TPB / 32 / R;             // warps of each role in a block
};

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
  // the chemical-potential part of point i's current correction (CDFT)
  __device__ __forceinline__ double keep_mc(int i, double e0, double ce) const {
    const double m = cdft_mc<double>(e0, cr(i), ce);
    L.rec[own(i) * D::NR + D::NR - 1] = m;
    return m;
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
      const double Ad = a.rk(i) + K.c_ad, bs = K.c_b * a.rk(i);
      double* v = L.iv + p * D::NV;
      if constexpr (DIM == 2) {
        const double b = bs * a.om(0, i), inv = 1.0 / (Ad * Ad + b * b);
        v[0] = Ad * inv;
        v[1] = b * inv;
      } else {
        const double b[3] = {bs * a.om(0, i), bs * a.om(1, i), bs * a.om(2, i)};
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
  }

  // The point of one colour a thread updates: neighbours' indices and records.
  struct Pt {
    int idx;  // -1: none
    int ni[2 * DIM];
    const double* nr[2 * DIM];  // m, p of each direction
  };
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
  static __device__ __forceinline__ double sum(const double (&v)[2 * DIM]) {
    double s = v[0] + v[1];
#pragma unroll
    for (int k = 2; k < 2 * DIM; ++k) s += v[k];
    return s;
  }

  // One colour pass over this block's points: slot p of `half` slots, role.
  // Every value of another point is loaded before the first use, so that the
  // remote reads overlap.
  static __device__ __forceinline__ void pass(const ClLvl& L, const Phys<double>& P, const PtK<double>& K,
                                              const Pt& t, int p, int role) {
    constexpr int AUX = 1 + DIM;
    const Acc a{L};
    const int half = L.sh - 1;
    const double w = P.w;
    double* eo = L.rec + (t.idx < 0 ? 0 : a.own(t.idx) * D::NR);
    double er = 0, psi = 0, cub = 0;
    if (t.idx >= 0) {
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
        er = f0 - K.c_div * div;
        const double x = crc + er;
        if (x <= K.proj) er = sqrt(x * x + P.delta * P.delta) - crc;  // Sec. 6 projection
        if constexpr (KIND == KPFC) {
          psi = crc - 1.5;
          cub = er * (psi * psi + psi * er + er * er * (1.0 / 3.0)) + P.alpha * er;
        }
      } else if (KIND == KPFC && role == AUX) {
        double v[2 * DIM], k2[2 * DIM];
#pragma unroll
        for (int k = 0; k < 2 * DIM; ++k) {
          v[k] = t.nr[k][0];
          k2[k] = t.nr[k][LY::IKA];
        }
        L.rhs[(DIM << half) + p] = a.f(LY::IKA, t.idx) + sum(v) * K.ih2;
        L.rhs[((DIM + 1) << half) + p] = a.f(LY::IMU, t.idx) + sum(k2) * K.ih2;
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
            const double fd = a.f(1 + d, t.idx), cs = K.c_sih * a.rk(t.idx);
#pragma unroll
            for (int k = 0; k < 2; ++k) {
              q[k] = 0;
#pragma unroll
              for (int b = 0; b < DIM; ++b) q[k] += u[k][b] * (2.0 * c[k][b] + u[k][b]);
            }
            L.rhs[(d << half) + p] = fd - cs * (0.25 * (q[1] - q[0]) + 0.5 * (m[1] - m[0])) + K.c_v * sum(v);
          }
      }
    }
    __syncthreads();
    if (t.idx >= 0) {
      const double* h = L.rhs + p;
      if (role == 0) {
        if constexpr (KIND == KPFC) {
          const double c4 = 2.0 * DIM * K.ih2;
          const double ek = h[DIM << half] - c4 * er;
          const double em = h[(DIM + 1) << half] + cub - c4 * ek;
          eo[LY::IKA] = (1.0 - w) * ek + w * eo[LY::IKA];
          eo[LY::IMU] = (1.0 - w) * em + w * eo[LY::IMU];
        }
        er = (1.0 - w) * er + w * eo[0];
        eo[0] = er;
        if constexpr (KIND == KCDFT) a.keep_mc(t.idx, er, P.ce);
      } else if (role <= DIM) {
        const double* v = L.iv + a.own(t.idx) * D::NV;
        double eg;
        if constexpr (DIM == 2)
          eg = role == 1 ? v[0] * h[0] + v[1] * h[1 << half] : v[0] * h[1 << half] - v[1] * h[0];
        else
          eg = v[3 * role - 3] * h[0] + v[3 * role - 2] * h[1 << half] + v[3 * role - 1] * h[2 << half];
        eo[role] = (1.0 - w) * eg + w * eo[role];
      }
    }
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
        if (x <= proj_threshold<double>(P.delta)) ev = sqrt(x * x + P.delta * P.delta) - c;
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

}  // namespace fm
