// Fused 2-D level kernels of the gradient-flow and channel solvers: one or
// two red-black sweeps per launch on tiles in shared memory (or a launch per
// colour where that is the better form, see fz_tile), the residual, restriction and
// coarse right-hand side in one launch, and the V-cycle of the smallest levels in
// one block.
//
// Both solvers' levels lie in L2 and their point updates are short, so a
// cycle's time is its number of launches: ~2.6 us each inside the step's
// graph, 44 a cycle for the 512^2 flow (four levels) and 66 for the 256^2
// channel (five levels) with a launch per colour, and 16 with these kernels and the
// injection on the norm launch.  Measured, four steps: 512^2 flow 4,672 -> 2,997 us,
// 256^2 channel 2,463 -> 1,524 us.  A policy M gives the model:
//   T, NU unknowns, NC coefficients read at neighbours, K level constants,
//   W wall speeds, WALLS, TILED64 (see fz_tile); coef(L, c) the c-th of the coefficients;
//   update(a, P, K, n, fc): the point update through an accessor a;
//   apply(F, P, K, W, x, y, M): M(e) at a point of a level in global memory;
//   apply_coarse(F, C, P, KC, W, I, J, M): M_C of the injected correction.
// The sweeps read the correction from one buffer and write it to the other
// (e -> r for dir = 0, r -> e for dir = 1), so a tile's halo always holds
// values from before the launch and the result is exactly NS red-black sweeps.
#pragma once

#include "fm_device.cuh"

namespace fm {

// Walls at y = 0 and y = ny h: a tile's ghost row holds the wall row's
// scalars, its velocity correction negated; a wall point's update writes its
// ghost (mir rows away) too, so the ghost always mirrors the current value.
template <class M, int SN>
struct FzAcc {
  using T = typename M::T;
  static constexpr int NU = M::NU;
  const Lvl<T>& G;
  int mir;
  __device__ __forceinline__ T* sm() const { return reinterpret_cast<T*>(fm_dyn_smem); }
  __device__ __forceinline__ T e(int q, int i) const { return sm()[q * SN + i]; }
  __device__ __forceinline__ void set_e(int q, int i, T v) const {
    sm()[q * SN + i] = v;
    if constexpr (M::WALLS) {
      if (mir) sm()[q * SN + i + mir] = (q == 1 || q == 2) ? -v : v;
    }
  }
  // coefficients in the policy's order: cr first, then rk, cv0, cv1
  __device__ __forceinline__ T cr(int i) const { return sm()[NU * SN + i]; }
  __device__ __forceinline__ T rk(int i) const { return sm()[(NU + 1) * SN + i]; }
  __device__ __forceinline__ T cv(int d, int i) const { return sm()[(NU + 2 + d) * SN + i]; }
  __device__ __forceinline__ T f(int q, int i) const { return G.f[q][i]; }
  __device__ __forceinline__ T om(int d, int i) const { return G.om[d][i]; }
};

template <class M, int TX, int TY, int NS>
__host__ __device__ constexpr size_t fz_smem() {
  return (size_t)(M::NU + M::NC) * RBGeom<TX, TY, NS>::SN * sizeof(typename M::T);
}

template <class M, int TX, int TY, int NS>
__global__ void __launch_bounds__(rb_threads(TX, TY), rb_minb<typename M::T>(TX, TY))
    kf_smooth(const __grid_constant__ Lvl<typename M::T> G, Phys<typename M::T> P, typename M::K K, typename M::W W,
              int ntx, int dir) {
  using T = typename M::T;
  using Gm = RBGeom<TX, TY, NS>;
  constexpr int NU = M::NU, NA = M::NU + M::NC, SN = Gm::SN, SW = Gm::SW, V = 16 / sizeof(T);
  T* buf = reinterpret_cast<T*>(fm_dyn_smem);
  const int nx = G.g.nx, ny = G.g.ny;
  const int x0 = (blockIdx.x % ntx) * TX, y0 = (blockIdx.x / ntx) * TY;
  const T* src[NA];
#pragma unroll
  for (int q = 0; q < NU; ++q) src[q] = dir ? G.r[q] : G.e[q];
#pragma unroll
  for (int c = 0; c < M::NC; ++c) src[NU + c] = M::coef(G, c);
  auto row_of = [&](int y) { return M::WALLS ? min(max(y, 0), ny - 1) : wrapi(y, ny); };
  if (nx % V == 0) {
    constexpr int CPR = SW / V, NCH = CPR * (TY + 2 * Gm::H);
    for (int t = threadIdx.x; t < NCH; t += blockDim.x) {
      const int ly = t / CPR, c = t - ly * CPR;
      const int gi = row_of(y0 + ly - Gm::H) * nx + wrapi(x0 - RB_XO + c * V, nx);
#pragma unroll
      for (int a = 0; a < NA; ++a) cp_async_16(buf + a * SN + ly * SW + c * V, src[a] + gi);
    }
  } else {
    for (int t = threadIdx.x; t < SN; t += blockDim.x) {
      const int ly = t / SW, lx = t - ly * SW;
      const int gi = row_of(y0 + ly - Gm::H) * nx + wrapi(x0 + lx - RB_XO, nx);
#pragma unroll
      for (int a = 0; a < NA; ++a) cp_async_elem(buf + a * SN + t, src[a] + gi);
    }
  }
  cp_async_commit();
  cp_async_wait_all();
  __syncthreads();
  if constexpr (M::WALLS) {
    // ghost rows -1 and ny, where the tile stages them (they hold the wall rows' values)
    const int lb = Gm::H - 1 - y0, lt = ny - y0 + Gm::H;
    const bool hb = lb >= 0, ht = lt < TY + 2 * Gm::H;
    if (hb || ht) {
      for (int t = threadIdx.x; t < 2 * SW; t += blockDim.x) {
        const bool top = t >= SW;
        if (top ? !ht : !hb) continue;
        const int i = (top ? lt : lb) * SW + (top ? t - SW : t);
        M::ghost(buf + i, SN, top, W);
      }
      __syncthreads();
    }
  }
#pragma unroll
  for (int pass = 0; pass < 2 * NS; ++pass) {
    const int color = pass & 1;
    const int ring = 2 * NS - 1 - pass;
    const int hw = (TX + 2 * ring) >> 1;
    const int npts = hw * (TY + 2 * ring);
    for (int t = threadIdx.x; t < npts; t += blockDim.x) {
      const int ry = t / hw;
      const int gy = y0 - ring + ry;
      if (M::WALLS && (gy < 0 || gy >= ny)) continue;
      const int rx = 2 * (t - ry * hw) + ((color + x0 + ring + gy) & 1);
      Nb n;
      n.c = (Gm::H - ring + ry) * SW + RB_XO - ring + rx;
      n.m[0] = n.c - 1;
      n.p[0] = n.c + 1;
      n.m[1] = n.c - SW;
      n.p[1] = n.c + SW;
      n.m[2] = n.p[2] = n.c;
      const FzAcc<M, SN> acc{G, !M::WALLS ? 0 : (gy == 0 ? -SW : (gy == ny - 1 ? SW : 0))};
      M::update(acc, P, K, n, (M::WALLS ? gy : wrapi(gy, ny)) * nx + wrapi(x0 - ring + rx, nx));
    }
    __syncthreads();
  }
  for (int t = threadIdx.x; t < TX * TY; t += blockDim.x) {
    const int ty = t / TX, tx = t - ty * TX;
    const int gx = x0 + tx, gy = y0 + ty;
    if (gx < nx && gy < ny) {
      const int si = (ty + Gm::H) * SW + tx + RB_XO;
#pragma unroll
      for (int q = 0; q < NU; ++q) (dir ? G.e[q] : G.r[q])[gy * nx + gx] = buf[q * SN + si];
    }
  }
}

// One colour of a sweep, in place, a point a thread (see fz_tiled).
template <class M>
__global__ void __launch_bounds__(TPB) kf_colour(const __grid_constant__ Lvl<typename M::T> L, Phys<typename M::T> P,
                                                 typename M::K K, typename M::W W, int color) {
  int i, j, k;
  if (colour_point(blockIdx.x * blockDim.x + threadIdx.x, color, L.g, i, j, k)) M::update_lvl(L, P, K, W, i, j);
}

// f_C = R(f - M(e)) + M_C(e_C), e_C = eh_C = the injection of e, on RR_TX x
// RR_TY coarse points a block (see k_resid_restrict2; between walls the
// restriction and injection average rows 2J and 2J + 1).  The correction is
// read from F.e.
template <class M>
__global__ void __launch_bounds__(TPB) kf_down(const __grid_constant__ Lvl<typename M::T> F,
                                               const __grid_constant__ Lvl<typename M::T> C, Phys<typename M::T> P,
                                               typename M::K KF, typename M::K KC, typename M::W W, int ntx) {
  using T = typename M::T;
  constexpr int NU = M::NU, FW = 2 * RR_TX + 1, FH = M::WALLS ? 2 * RR_TY : 2 * RR_TY + 1, FN = FW * FH;
  __shared__ T sr[NU * FN];
  const int I0 = (blockIdx.x % ntx) * RR_TX, J0 = (blockIdx.x / ntx) * RR_TY;
  const int yb = M::WALLS ? 2 * J0 : 2 * J0 - 1;
  const int nx = F.g.nx, ny = F.g.ny;
  for (int t = threadIdx.x; t < FN; t += blockDim.x) {
    const int ly = t / FW, lx = t - ly * FW;
    const int x = wrapi(2 * I0 - 1 + lx, nx), y = M::WALLS ? yb + ly : wrapi(yb + ly, ny);
    if (M::WALLS && y >= ny) continue;
    T m[NU], fv[NU];
#pragma unroll
    for (int q = 0; q < NU; ++q) fv[q] = F.f[q][y * nx + x];
    M::apply(F, P, KF, W, x, y, m);
#pragma unroll
    for (int q = 0; q < NU; ++q) sr[q * FN + t] = fv[q] - m[q];
  }
  __syncthreads();
  for (int t = threadIdx.x; t < RR_TX * RR_TY; t += blockDim.x) {
    const int ty = t / RR_TX, tx = t - ty * RR_TX;
    const int I = I0 + tx, J = J0 + ty;
    if (I >= C.g.nx || J >= C.g.ny) continue;
    const int ci = J * C.g.nx + I;
    const int ctr = 2 * J * nx + 2 * I;
    T ev[NU], m[NU];
#pragma unroll
    for (int q = 0; q < NU; ++q) ev[q] = M::WALLS ? T(0.5) * (F.e[q][ctr] + F.e[q][ctr + nx]) : F.e[q][ctr];
    M::apply_coarse(F, C, P, KC, W, I, J, m);
#pragma unroll
    for (int q = 0; q < NU; ++q) {
      T acc;
      if constexpr (M::WALLS) {
        const T* r0 = sr + q * FN + 2 * ty * FW + 2 * tx + 1;
        const T* r1 = r0 + FW;
        acc = T(0.125) * (r0[-1] + r1[-1] + r0[1] + r1[1]) + T(0.25) * (r0[0] + r1[0]);
      } else {
        const T* r = sr + q * FN + (2 * ty + 1) * FW + 2 * tx + 1;
        acc = r[-FW - 1] + T(2) * r[-FW] + r[-FW + 1];
        acc += T(2) * (r[-1] + T(2) * r[0] + r[1]);
        acc += r[FW - 1] + T(2) * r[FW] + r[FW + 1];
        acc *= T(1.0 / 16.0);
      }
      C.f[q][ci] = acc + m[q];
      C.e[q][ci] = ev[q];
      C.eh[q][ci] = ev[q];
    }
  }
}

// The V-cycle of the levels S in one block, corrections in global memory
// (L1): a colour pass or transfer between block barriers.  float32 only: a
// float64 point update is ~20 times dearer, and one multiprocessor's float64
// pipe then costs more than the launches it saves.
template <class M>
__global__ void __launch_bounds__(SMALL_TPB) kf_small(const __grid_constant__ SmallLv<typename M::T> S,
                                                      Phys<typename M::T> P, typename M::W W, int nu1, int nu2,
                                                      int ncoarse) {
  using T = typename M::T;
  constexpr int NU = M::NU;
  auto smooth = [&](const Lvl<T>& L, int iters) {
    const typename M::K K = M::constants(P, L.h);
    const int half = L.g.N / 2;
    for (int s = 0; s < 2 * iters; ++s) {
      for (int t = threadIdx.x; t < half; t += SMALL_TPB) {
        int i, j, k;
        colour_point(t, s & 1, L.g, i, j, k);
        M::update_lvl(L, P, K, W, i, j);
      }
      __syncthreads();
    }
  };
  for (int l = 0; l + 1 < S.count; ++l) {
    const Lvl<T>&F = S.lv[l], &C = S.lv[l + 1];
    smooth(F, nu1);
    const typename M::K K = M::constants(P, F.h), KC = M::constants(P, C.h);
    for (int i = threadIdx.x; i < F.g.N; i += SMALL_TPB) {
      T m[NU], fv[NU];
#pragma unroll
      for (int q = 0; q < NU; ++q) fv[q] = F.f[q][i];
      M::apply(F, P, K, W, i % F.g.nx, i / F.g.nx, m);
#pragma unroll
      for (int q = 0; q < NU; ++q) F.r[q][i] = fv[q] - m[q];
    }
    __syncthreads();
    for (int i = threadIdx.x; i < C.g.N; i += SMALL_TPB) {
      T m[NU];
      M::apply_coarse(F, C, P, KC, W, i % C.g.nx, i / C.g.nx, m);
      M::restrict_lvl(F, C, i);
#pragma unroll
      for (int q = 0; q < NU; ++q) C.f[q][i] += m[q];
    }
    __syncthreads();
  }
  smooth(S.lv[S.count - 1], ncoarse);
  for (int l = S.count - 2; l >= 0; --l) {
    const Lvl<T>&F = S.lv[l], &C = S.lv[l + 1];
    for (int i = threadIdx.x; i < F.g.N; i += SMALL_TPB) M::prolong_lvl(F, C, P, i);
    __syncthreads();
    smooth(F, nu2);
  }
}

// Host side ------------------------------------------------------------------

template <class M, int TX, int TY, int NS>
static cudaError_t fz_launch_smooth(const Lvl<typename M::T>& L, const Phys<typename M::T>& P, const typename M::K& K,
                                    const typename M::W& W, int dir, cudaStream_t s) {
  constexpr size_t smem = fz_smem<M, TX, TY, NS>();
  const auto kernel = kf_smooth<M, TX, TY, NS>;
  if constexpr (smem > 48 * 1024) {
    const cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
  }
  const int ntx = (L.g.nx + TX - 1) / TX;
  kernel<<<ntx * ((L.g.ny + TY - 1) / TY), rb_threads(TX, TY), smem, s>>>(L, P, K, W, ntx, dir);
  return cudaPeekAtLastError();
}

// The view of a level whose correction is in r.
template <typename T>
static Lvl<T> fz_view(Lvl<T> L, int in_r) {
  if (in_r)
    for (int q = 0; q < MAXU; ++q) {
      T* t = L.e[q];
      L.e[q] = L.r[q];
      L.r[q] = t;
    }
  return L;
}

// What sweeps a level: 0 a launch per colour, 1 tiles of 16 x 8, 2 of 32 x 16.
// A level of four sweeps, us a cycle, colour / 16 x 8 / 32 x 16:
//  * float32, tiles run two sweeps a launch: channel 128^2 46 / 33 / 35, 512^2 88 / 84 /
//    78, flow 31 / 26 / 27 and 50 / 49 / 46; large tiles from 256^2 points on.  Levels
//    narrower than a tile compute its columns for nothing: they stay on tiles while
//    a few tiles a multiprocessor hold them (channel 8192 x 2, 512 tiles, 48 / 34 / 34;
//    2 x 16384, 2,048 tiles, 56 / 78 / 94) or less than half is added (65536 x 4 92 / 95 / 102).
//  * float64 is bound by the busiest multiprocessor's point updates, a tile's ring
//    among them (562 a sweep for 32 x 16, 154 for 16 x 8): tiles of at most two a
//    multiprocessor (128^2 76 / 59 / 94), or where these are below 1.35 a point
//    (channel 256^2 106 / 104 / 99, 512^2 299 / 300 / 303, 300 x 500 186 / 185 / 229, 150 x 250
//    79 / 87 / 98).  The flow's update reads too little for the tile to
//    pay once the pipe is full (M::TILED64): 128^2 44 / 39 / 55, 512^2 129 / 155 / 150.
template <class M>
static int fz_tile(const Geo& g, int sms) {
  auto tiles = [&](int tx, int ty) { return (long long)((g.nx + tx - 1) / tx) * ((g.ny + ty - 1) / ty); };
  const long long big = tiles(32, 16), small = tiles(16, 8);
  if (sizeof(typename M::T) == 4) {
    if (g.N >= 256 * 256 && 4 * 512 * big <= 5LL * g.N) return 2;
    return small <= 4 * sms || 2 * 128 * small <= 3LL * g.N ? 1 : 0;
  }
  if (g.N > (long long)M::TILED64 * sms) return 0;
  // point updates of a sweep on the busiest multiprocessors, times their number
  auto cost = [&](long long t, int updates) { return (t + sms - 1) / sms * sms * updates; };
  if (g.N >= 256 * 256 && 100 * cost(big, 562) <= 135LL * g.N) return 2;
  return small <= 2 * sms || 100 * cost(small, 154) <= 135LL * g.N ? 1 : 0;
}

// `iters` sweeps of a level (the correction in r if *in_r), on tiles two a launch
// while two are left.  float64 takes one sweep a launch: the two-sweep tile's wider
// halo is 1.3 to 1.7 times the point updates, which are what bounds it.
template <class M>
static cudaError_t fz_smooth(const Lvl<typename M::T>& L, const Phys<typename M::T>& P, const typename M::W& W,
                             int iters, int* in_r, long long* launches, int sms, cudaStream_t s) {
  const typename M::K K = M::constants(P, L.h);
  const int tile = fz_tile<M>(L.g, sms);
  if (!tile) {
    const Lvl<typename M::T> V = fz_view(L, *in_r);
    const int tpb = point_tpb<typename M::T>(L.g.N / 2, sms);
    for (int c = 0; c < 2 * iters; ++c) {
      kf_colour<M><<<blocks_of(L.g.N / 2, tpb), tpb, 0, s>>>(V, P, K, W, c & 1);
      const cudaError_t e = cudaPeekAtLastError();
      if (e != cudaSuccess) return e;
      ++*launches;
    }
    return cudaSuccess;
  }
  const bool big = tile == 2;
  for (int it = 0; it < iters;) {
    cudaError_t e;
    if (sizeof(typename M::T) == 4 && it + 2 <= iters) {
      e = big ? fz_launch_smooth<M, 32, 16, 2>(L, P, K, W, *in_r, s)
              : fz_launch_smooth<M, 16, 8, 2>(L, P, K, W, *in_r, s);
      it += 2;
    } else {
      e = big ? fz_launch_smooth<M, 32, 16, 1>(L, P, K, W, *in_r, s)
              : fz_launch_smooth<M, 16, 8, 1>(L, P, K, W, *in_r, s);
      it += 1;
    }
    if (e != cudaSuccess) return e;
    *in_r ^= 1;
    ++*launches;
  }
  return cudaSuccess;
}

template <class M>
static cudaError_t fz_down(const Lvl<typename M::T>& F, const Lvl<typename M::T>& C, const Phys<typename M::T>& P,
                           const typename M::W& W, long long* launches, cudaStream_t s) {
  const int ntx = (C.g.nx + RR_TX - 1) / RR_TX;
  kf_down<M><<<ntx * ((C.g.ny + RR_TY - 1) / RR_TY), TPB, 0, s>>>(F, C, P, M::constants(P, F.h), M::constants(P, C.h),
                                                                   W, ntx);
  ++*launches;
  return cudaPeekAtLastError();
}

template <class M>
static cudaError_t fz_small(const SmallLv<typename M::T>& S, const Phys<typename M::T>& P, const typename M::W& W,
                            const fm_params& prm, long long* launches, cudaStream_t s) {
  kf_small<M><<<1, SMALL_TPB, 0, s>>>(S, P, W, prm.nu1, prm.nu2, prm.ncoarse);
  ++*launches;
  return cudaPeekAtLastError();
}

// First level of the one-block part: the first of at most SMALL_N points (float32 only).
template <typename T>
static int fz_small_from(const fm_state* st) {
  for (int l = sizeof(T) == 8 ? st->nlev : 0; l < st->nlev; ++l)
    if (st->lv[l].g.N <= SMALL_N && st->nlev - l <= MAXSMALL) return l;
  return st->nlev;
}

}  // namespace fm
