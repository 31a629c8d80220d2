// The FP64 step of a small grid: a tile of SPLIT_X x SPLIT_Y cells, one per
// lane, whose work is divided among four warps.
//
// The FP64 pipe takes 64 clocks a warp instruction on each of an SM's four
// partitions, whatever the number of lanes that hold a cell, so a grid that
// leaves the chip idle is bound by the FP64 instructions one warp issues in a
// row: about 1,100 (40 us a step) where the warp does everything for its cells
// and the ring around them.  Here each partition's warp takes a part:
//   moments   c of the region by three warps, then p and T of the inner region
//             by two each
//   stencils  the unit normals by two warps, grad T and grad p by the third,
//             the Laplacian by the fourth
//   collision each warp the force and u, then two opposite directions of all
//             three lattices; the rest directions go to warps 0, 1, 2
// The operations and their order per value are those of tile_kernel (the same
// functions, the unused results dropped by the compiler): the same bits.
#pragma once

#include "lbe_launch.h"
#include "lbe_tile.cuh"

namespace lbe {

constexpr int SPLIT_X = TILE_SHAPES[SPLIT_TILE].tx, SPLIT_Y = TILE_SHAPES[SPLIT_TILE].ty;
constexpr int SPLIT_THREADS = 128;
static_assert(SPLIT_X * SPLIT_Y == 32, "one cell per lane");

struct SplitTile {
  using S = StF64;
  using C = double;
  static constexpr int RW = SPLIT_X + 4, RH = SPLIT_Y + 4;  // c (ring of 2)
  static constexpr int QW = SPLIT_X + 2, QH = SPLIT_Y + 2;  // p, T, n (ring of 1)
  static_assert(RW * RH <= SPLIT_THREADS && QW * QH <= SPLIT_THREADS / 2, "one value per thread");

  struct Smem {
    C c[RH * RW], p[QH * QW], T[QH * QW], nx[QH * QW], ny[QH * QW];
    C gx[32], gy[32], lapc[32], gTx[32], gTy[32], gpx[32], gpy[32];
  };

  // p or T of a position of the region (see region_values)
  __device__ static C region_one(const InstDev& I, const Phys<C>& P, const char* __restrict__ src,
                                 int gx, int gy, bool wants_T) {
    const int nx = I.nx, ny = I.ny;
    const int y = gy < 0 ? -1 - gy : gy >= ny ? 2 * ny - 1 - gy : gy;
    const Cell<S> q = make_cell<S>(wrapx(gx, nx), y, nx);
    C v[9];
    if (!wants_T) {
      if (nonzero(P.drho)) return I.pcorr[(size_t)y * nx + q.x];
      pull9<S, 0>(I, P, src, q, v);
      return sum9(v);
    }
    C rc = P.rho;
    if (nonzero(P.drho)) {
      pull9<S, 1>(I, P, src, q, v);
      rc = rho_at(P, sum9(v));
    }
    pull9<S, 2, true>(I, P, src, q, v, rc);
    const C T = cell_T(P, sum9(v), rc);
    return gy < 0 || gy >= ny ? ghost_T<S>(I, q.x, gy < 0, T) : T;
  }

  // warp W's part of the collision of the lane's cell
  template <int W>
  __device__ static void part(const InstDev& I, const Phys<C>& P, const char* __restrict__ src,
                              char* __restrict__ dst, const Cell<S>& q, const C f[9], C cc, C pp,
                              C TT, C gpx, C gpy, const Drive<S>& d, const C* wdu) {
    constexpr int A = W == 0 ? 1 : W == 1 ? 2 : W == 2 ? 5 : 6;
    constexpr int B = A < 5 ? A + 2 : A == 5 ? 7 : 8;
    C g[9], h[9];
    pull9<S, 1>(I, P, src, q, g);
    pull9<S, 2, true>(I, P, src, q, h, rho_at(P, cc));
    const size_t rowbase = (size_t)q.y * I.pitch;
    collide<S>(
        P, f, g, h, cc, pp, TT, gpx, gpy, d,
        [&](int k, int i, C v) {
          if (i == 0 ? k == W : (i == A || i == B)) st_cell<S>(I, dst, k, i, rowbase, q.x, v);
        },
        C(0), C(0), nullptr, C(0), wdu);
  }

  __device__ static void run(const InstDev& I, int64_t tile, int parity, Smem& sm) {
    const int t = threadIdx.x, lane = t & 31;
    const int warp = __shfl_sync(0xffffffffu, t >> 5, 0);
    const int nx = I.nx, ny = I.ny;
    const int x0 = (int)(tile % I.tiles_x) * SPLIT_X;
    const int y0 = (int)(tile / I.tiles_x) * SPLIT_Y;
    const char* __restrict__ src = I.buf[parity];
    const Phys<C> P = phys<C>(I);

    // ---- moments: c of the region, then p (first two warps) and T of its
    // inner part; zero beyond the ghost rows
    const int gx = x0 + lane % SPLIT_X, gy = y0 + lane / SPLIT_X;
    const bool active = gx < nx && gy < ny;
    const Cell<S> q = make_cell<S>(active ? gx : 0, active ? gy : 0, nx);
    C f[9];
    pull9<S, 0>(I, P, src, q, f);
    if (t < RW * RH) {
      const int hx = x0 - 2 + t % RW, hy = y0 - 2 + t / RW;
      C c = C(0), p, T;
      if (hy >= -2 && hy <= ny + 1) region_values<S>(I, P, src, hx, hy, false, true, c, p, T);
      sm.c[t] = c;
    }
    const int r = t % (SPLIT_THREADS / 2);
    if (r < QW * QH) {
      const bool wants_T = t >= SPLIT_THREADS / 2;
      const int hx = x0 - 1 + r % QW, hy = y0 - 1 + r / QW;
      C v = C(0);
      if (hy >= -1 && hy <= ny) v = region_one(I, P, src, hx, hy, wants_T);
      (wants_T ? sm.T : sm.p)[r] = v;
    }
    __syncthreads();

    // ---- stencils
    const int tx = lane % SPLIT_X, ty = lane / SPLIT_X;
    const C* c0 = sm.c + (ty + 2) * RW;
    const int qo = (ty + 1) * QW;
    if (warp < 2) {
      const int n = t;
      if (n < QW * QH) {
        const int qx = n % QW, qy = n / QW;
        const C* cq = sm.c + (qy + 1) * RW;
        C gcx, gcy;
        normal3(cq - RW, cq, cq + RW, qx + 1, P.eta_n2, sm.nx[n], sm.ny[n], gcx, gcy);
        if (qx > 0 && qx <= SPLIT_X && qy > 0 && qy <= SPLIT_Y) {
          sm.gx[(qy - 1) * SPLIT_X + qx - 1] = gcx;
          sm.gy[(qy - 1) * SPLIT_X + qx - 1] = gcy;
        }
      }
    } else if (warp == 2) {
      grad3(sm.T + qo - QW, sm.T + qo, sm.T + qo + QW, tx + 1, sm.gTx[lane], sm.gTy[lane]);
      grad3(sm.p + qo - QW, sm.p + qo, sm.p + qo + QW, tx + 1, sm.gpx[lane], sm.gpy[lane]);
    } else {
      sm.lapc[lane] = lap3(c0 - RW, c0, c0 + RW, tx + 2);
    }
    __syncthreads();

    // ---- force, u and the warp's part of the collision
    if (!active) return;
    Stencils<C> st;
    st.gcx = sm.gx[lane];
    st.gcy = sm.gy[lane];
    st.lapc = sm.lapc[lane];
    st.gTx = sm.gTx[lane];
    st.gTy = sm.gTy[lane];
    st.gpx = sm.gpx[lane];
    st.gpy = sm.gpy[lane];
    C d1, d2, dum;
    grad3(sm.nx + qo - QW, sm.nx + qo, sm.nx + qo + QW, tx + 1, d1, dum);
    grad3(sm.ny + qo - QW, sm.ny + qo, sm.ny + qo + QW, tx + 1, dum, d2);
    st.kappa = d1 + d2;
    const C cc = c0[tx + 2], pp = sm.p[qo + tx + 1], TT = sm.T[qo + tx + 1];
    const Drive<S> d = drive<S>(P, gy, f, cc, TT, st);
    C du[4];
    if (I.uvel != nullptr) grad_u(nx, ny, I.uvel, gx, gy, du);
    const C* wdu = I.uvel != nullptr ? du : nullptr;
    char* __restrict__ dst = I.buf[parity ^ 1];
    if (warp == 0)
      part<0>(I, P, src, dst, q, f, cc, pp, TT, st.gpx, st.gpy, d, wdu);
    else if (warp == 1)
      part<1>(I, P, src, dst, q, f, cc, pp, TT, st.gpx, st.gpy, d, wdu);
    else if (warp == 2)
      part<2>(I, P, src, dst, q, f, cc, pp, TT, st.gpx, st.gpy, d, wdu);
    else
      part<3>(I, P, src, dst, q, f, cc, pp, TT, st.gpx, st.gpy, d, wdu);
  }
};

__global__ void __launch_bounds__(SPLIT_THREADS, 1)
split_kernel(const InstDev* __restrict__ insts, int n_inst, int64_t total_tiles, int parity) {
  __shared__ SplitTile::Smem sm;
  grid_wait();
  for (int64_t t = blockIdx.x; t < total_tiles; t += gridDim.x) {
    int lo = 0, hi = n_inst - 1;
    while (lo < hi) {
      const int mid = (lo + hi + 1) >> 1;
      if (insts[mid].tile_begin <= t) lo = mid; else hi = mid - 1;
    }
    const InstDev& I = insts[lo];
    SplitTile::run(I, t - I.tile_begin, parity, sm);
    __syncthreads();
  }
}

}  // namespace lbe
