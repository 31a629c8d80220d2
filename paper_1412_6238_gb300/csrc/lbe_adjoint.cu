// Discrete adjoint (vector-Jacobian product) of one FP64 step, and the
// drop-migration observable.  (The adjoint recomputes the forward step with
// reciprocal products where the step divides, so it differentiates the step
// at a state equal to the FP64 one to rounding, not bitwise.)
//
// The step maps the pre-collision state Q_n (27 planes, [27][ny][nx]) to
// Q_{n+1} = Pull(Post(Q_n; theta)); Post is the collision of every cell,
// which reads its own populations and, through the stencils, c at distance
// <= 2 and p, T at distance 1 (with the wall ghost rows).  Given
// a = dL/dQ_{n+1} the adjoint step returns
//   dL/dQ_n = Post'(Q_n)^T Pull^T a + w dl/dQ_n
// and adds a^T dQ_{n+1}/dtheta (+ w dl/dtheta) to the gradient of
// theta = (sigmaT, eta ratio eta2/eta1, conductivity ratio lam2/lam1), where
// l(Q) = sum_x c u_y / sum_x c is the centroid velocity of phase 1 (the
// migration velocity of Sec. IV.C without the c >= 0.5 threshold) and w the
// loss weight of step n.  Two kernels per step, all deterministic gathers:
//   A   a tile of cells: c, p, T of the tile and its halo and the unit normal
//       (Eq. 3) in shared memory; per cell the forward step (stencils, mu, F,
//       u, the three collisions) recomputed and b = Pull^T a (the transpose of
//       streaming: a permutation with signs, read in place) back-propagated
//       through it; writes the direct population adjoints, the adjoints of
//       the stencil outputs (grad c, lap c, grad T, grad p, kappa) and of the
//       cell's own c, p, T, and adds to the tile's theta sums
//   B   a tile of cells: kappa-bar -> n-bar (transposed divergence) ->
//       grad-c-bar through the normalisation, on the tile, its halo and the
//       ghost rows; then the transposed stencils (ghost images folded back:
//       mirror for c and p, sign flip for T) give p-bar, c-bar, T-bar of the
//       cell, which belong to each of its f, g, hbar.
// An adjoint state is held as the 27 direct adjoints and those three terms of
// the cell: population j of lattice l has a_lj + t_l (the next step's A adds
// them as it reads, the last step's are added in FP64), so B does not rewrite
// 27 planes.
//
// R is the arithmetic type of the states and adjoints: double for an FP64
// handle, float for a handle whose forward step is FP32 or 16-bit arithmetic
// (the adjoint is then linearised about an FP32 trajectory anyway; GB300's
// FP64 rate is 1/64 of its FP32 rate).  The sum of the two FP32 parts of an
// adjoint is formed once, rounded to FP32 where it is used (the value the
// FP64 sum of the parts rounds to) and exact in FP64 in the results.  FP32
// states hold the FP64 state's values rounded to FP32, and c and T as two
// floats (for the normals, which are the FP64 ones rounded, and the observable).
// The theta sums and the observable are FP64.
//
// What bounds it: at 256 x 512 (FP32) a state is 16 MB and a step touches 45
// MB, which the L2 holds but for the states of a segment.  The two kernels take
// 35 us a step (27 and 8).  As seven kernels over FP64 planes (moments, normals,
// permutation, pass A, reduction, B, CD with a read-modify-write of all 27
// planes) it takes 210, much of it conversions between FP64 planes and FP32
// arithmetic at the FP64 pipe's rate.
#include <cstdio>

#include "../../include/lbe.h"
#include "lbe_launch.h"
#include "lbe_tile.cuh"

namespace lbe {
namespace adj {

constexpr int TX = 32, TY = 8, TPB = TX * TY;
constexpr double ICS2 = 3.0;  // 1 / c_s^2: products instead of FP64 divisions

struct Geo {
  int nx, ny, tx, ty;  // cells, tiles
  int64_t N;           // nx * ny
};
Geo make_geo(int nx, int ny) {
  return Geo{nx, ny, (nx + TX - 1) / TX, (ny + TY - 1) / TY, (int64_t)nx * ny};
}

// A state: planes of N values: the populations Q and, in FP32, the moments C, P,
// T and the low parts of c and T.  FP64 states are the populations alone; the
// moments of the one in work are in planes of their own (a segment's states are
// most of the memory of a call, and three planes more in each would be a tenth
// of it; forming them takes 1 % of a reverse step).
template <class R>
struct State {
  const R *Q, *C, *P, *T, *Cl, *Tl;
};
template <class R>
__host__ __device__ constexpr bool two_floats() {
  return sizeof(R) == 4;
}

// Row of the cell whose value (mirrored) a row of the c, p or T halo holds:
// -1 -> 0, -2 -> 1, ny -> ny - 1, ny + 1 -> ny - 2.
__device__ __forceinline__ int mirror_row(int y, int ny) {
  return y < 0 ? -1 - y : (y >= ny ? 2 * ny - 1 - y : y);
}

// Column x of a tile's halo (-2 <= x), wrapped: exact for the columns a cell
// of the tile can reach (up to nx + 1), some column beyond them.
__device__ __forceinline__ int wrap_col(int x, int nx) {
  if (x < 0) x += nx;
  if (x < 0) x += nx;  // nx = 1
  if (x >= nx) x -= nx;
  return x >= nx ? 0 : x;
}
// The thread's cell of the tile; a warp is a row of it (ty is warp-uniform,
// and so are the walls and the planes it selects).
__device__ __forceinline__ int tile_row() {
  static_assert(TX == 32, "a warp per row");
  return __shfl_sync(0xffffffffu, (int)threadIdx.x / TX, 0);
}

// Isotropic gradient at entry k of a tile field whose rows are `w` entries
// apart: the terms i = 1..8 in turn, fused (a change of this order changes
// grad c, off the interface, by more than its own size: there the FP32 values
// of c are equal or one rounding apart, and the derivative of the normal is
// 1/|grad c|).
template <class R>
__device__ __forceinline__ void tgrad(const R* v, int k, int w, R& gx, R& gy) {
  R sx = R(0), sy = R(0);
#pragma unroll
  for (int i = 1; i < 9; i++) {
    const R a = v[k + EY(i) * w + EX(i)];
    if (EX(i) != 0) sx = fma(WGT<R>(i) * R(EX(i)), a, sx);
    if (EY(i) != 0) sy = fma(WGT<R>(i) * R(EY(i)), a, sy);
  }
  gx = sx * R(ICS2);
  gy = sy * R(ICS2);
}
// The unit normal grad c / sqrt(|grad c|^2 + eta_n^2) at entry k of c.
__device__ __forceinline__ void unit_normal(const double* c, int k, int w, double en2, double& nx,
                                            double& ny) {
  const double wa = WGT<double>(1), wd = WGT<double>(5);
  auto diff = [&](int p, int m) { return c[k + p] - c[k + m]; };
  const double d1 = diff(w + 1, -w - 1), d2 = diff(1 - w, w - 1);
  const double gx = ICS2 * (wa * diff(1, -1) + wd * (d1 + d2));
  const double gy = ICS2 * (wa * diff(w, -w) + wd * (d1 - d2));
  const double inv = 1.0 / sqrt(gx * gx + gy * gy + en2);
  nx = gx * inv;
  ny = gy * inv;
}
// (FP32: the same rounded, in two-float arithmetic: lbe_two.cuh.  In FP64 it would
// take half as long as the rest of kernel A.)
template <class R>
__device__ __forceinline__ R tlap(const R* v, int k, int w) {
  const R v0 = v[k];
  R s = R(0);
#pragma unroll
  for (int i = 1; i < 9; i++) s = fma(WGT<R>(i), v[k + EY(i) * w + EX(i)] - v0, s);
  return R(2) * s * R(ICS2);
}

// xi_i . (a, b), without products by the components
template <class R>
__device__ __forceinline__ R xi_dot(int i, R a, R b) {
  const R ea = EX(i) == 0 ? R(0) : (EX(i) > 0 ? a : -a);
  const R eb = EY(i) == 0 ? R(0) : (EY(i) > 0 ? b : -b);
  return EX(i) == 0 ? eb : (EY(i) == 0 ? ea : ea + eb);
}

// ---------------------------------------------------------------- the state
// Sum of 9 FP32 values (and lo0) as hi + lo, hi the sum rounded to FP32.
__device__ __forceinline__ float sum9_exact(const float v[9], float lo0, float& lo) {
  float s = v[0], r = lo0;
#pragma unroll
  for (int i = 1; i < 9; i++) {
    float t, e;
    two_sum(s, v[i], t, e);
    s = t;
    r += e;
  }
  float hi;
  fast_two_sum(s, r, hi, lo);
  return hi;
}

// The state (planes of R: 27 populations, in FP32 C, P, T, Cl and Tl) of the
// buffer `parity`: the pull of every cell and its moments.
template <class S>
__global__ void __launch_bounds__(256)
state_kernel(Geo G, const InstDev* __restrict__ d, int parity, typename S::C* __restrict__ out) {
  using R = typename S::C;
  grid_wait();
  const InstDev& I = *d;
  const int x = blockIdx.x * blockDim.x + threadIdx.x;
  if (x >= G.nx) return;
  const char* buf = I.buf[parity];
  const Phys<R>& P = phys<R>(I);
  for (int y = blockIdx.y; y < G.ny; y += gridDim.y) {
    const int64_t k = (int64_t)y * G.nx + x;
    const Cell<S> q = make_cell<S>(x, y, G.nx);
    R v[9];
    pull9<S, 0>(I, P, buf, q, v);
#pragma unroll
    for (int i = 0; i < 9; i++) out[(int64_t)i * G.N + k] = v[i];
    R lo;
    if constexpr (two_floats<R>()) out[28 * G.N + k] = sum9_exact(v, R(0), lo);
    pull9<S, 1>(I, P, buf, q, v);
#pragma unroll
    for (int i = 0; i < 9; i++) out[(int64_t)(9 + i) * G.N + k] = v[i];
    if constexpr (two_floats<R>()) {
      out[27 * G.N + k] =
          sum9_exact(v, ld_g0lo<S>(I, buf, (size_t)y * I.pitch + XG + x), lo);
      out[30 * G.N + k] = lo;
    }
    pull9<S, 2>(I, P, buf, q, v);
    if constexpr (two_floats<R>()) {
      // hbar_i = v_i + w_i rho c_v T_r(y) and T = sum v / (rho c_v) + T_r(y),
      // the row's constants as two floats
      const double Tr = I.hr0 + I.hr1 * y, hr = I.pd.rho * I.pd.cv * Tr;
      auto add = [](double c, R x, R xl, R& lo) -> R {  // c + x + xl rounded, and the rest
        const R ch = (R)c, cl = (R)(c - (double)ch);
        R s, e;
        two_sum(ch, x, s, e);
        R r;
        fast_two_sum(s, e + (cl + xl), r, lo);
        return r;
      };
      const double w[3] = {WGT<double>(0) * hr, WGT<double>(1) * hr, WGT<double>(5) * hr};
#pragma unroll
      for (int i = 0; i < 9; i++)
        out[(int64_t)(18 + i) * G.N + k] = add(w[i == 0 ? 0 : i < 5 ? 1 : 2], v[i], R(0), lo);
      // sum v / (rho c_v), the sum and the reciprocal as two floats
      R sl;
      const R sh = sum9_exact(v, R(0), sl), q = __fmul_rn(sh, P.yrcv);
      out[29 * G.N + k] =
          add(Tr, q, fmaf(sh, P.yrcv, -q) + (sh * P.krcv + sl * P.yrcv), lo);
      out[31 * G.N + k] = lo;
    } else {
#pragma unroll
      for (int i = 0; i < 9; i++) out[(int64_t)(18 + i) * G.N + k] = v[i];
    }
  }
}

// C, P, T of 27 FP64 planes (an FP64 state, or one handed in by the caller)
__global__ void moments_kernel(Geo G, const InstDev* __restrict__ d, const double* __restrict__ Q,
                               double* __restrict__ C, double* __restrict__ Pp,
                               double* __restrict__ T) {
  const InstDev& I = *d;
  for (int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; k < G.N;
       k += (int64_t)gridDim.x * blockDim.x) {
    double sf = 0, sg = 0, sh = 0;
    for (int i = 0; i < 9; i++) {
      sf += Q[(int64_t)i * G.N + k];
      sg += Q[(int64_t)(9 + i) * G.N + k];
      sh += Q[(int64_t)(18 + i) * G.N + k];
    }
    C[k] = sg;
    Pp[k] = sf;
    T[k] = sh / (I.pd.rho * I.pd.cv);
  }
}

// ---------------------------------------------------------------- tiles
// Tile fields: c (and its low part) on a ring of 2, p, T and the normal on a
// ring of 1 around the TX x TY cells.
constexpr int CW = TX + 4, CH = TY + 4, QW = TX + 2, QH = TY + 2;
template <class R>
struct TileA {
  R c[CH * CW], cl[two_floats<R>() ? CH * CW : 1];
  R p[QH * QW], T[QH * QW], nx[QH * QW], ny[QH * QW];
  Two e;  // FP32: 144 eta_n^2
};

// T of the cell k (row y), or of the ghost row y beyond a wall from its mirror
// cell k
template <class R>
__device__ __forceinline__ R tile_T(const InstDev& I, const Geo& G, const State<R>& st, int64_t k,
                                    int x, int y) {
  const R v = st.T[k];
  if (y >= 0 && y < G.ny) return v;
  double t = (double)v;
  if constexpr (two_floats<R>()) t += (double)st.Tl[k];
  return (R)(2.0 * (y < 0 ? I.Tbot[x] : I.Ttop[x]) - t);
}

// c, p, T and the normals of the tile at (x0, y0) into sm (two barriers).
template <class R>
__device__ __forceinline__ void load_tile(TileA<R>& sm, const Geo& G, const InstDev& I,
                                          const State<R>& st, int x0, int y0) {
  for (int r = threadIdx.x; r < CH * CW; r += TPB) {
    const int rx = r % CW, ry = r / CW;
    const int y = y0 - 2 + ry;
    if (y < -2 || y > G.ny + 1) {
      sm.c[r] = R(0);
      if (two_floats<R>()) sm.cl[r] = R(0);
      continue;
    }
    const int x = wrap_col(x0 - 2 + rx, G.nx);
    const int64_t k = (int64_t)mirror_row(y, G.ny) * G.nx + x;
    sm.c[r] = st.C[k];
    if (two_floats<R>()) sm.cl[r] = st.Cl[k];
    if (rx >= 1 && rx <= TX + 2 && ry >= 1 && ry <= TY + 2) {
      const int q = (ry - 1) * QW + rx - 1;
      const bool in = y >= -1 && y <= G.ny;
      sm.p[q] = in ? st.P[k] : R(0);
      sm.T[q] = in ? tile_T(I, G, st, k, x, y) : R(0);
    }
  }
  if (two_floats<R>() && threadIdx.x == 0) {  // (FP64, by one warp only)
    const double e = 144.0 * I.pd.eta_n2;
    sm.e.h = (float)e;
    sm.e.l = (float)(e - (double)sm.e.h);
  }
  __syncthreads();
  for (int r = threadIdx.x; r < QW * QH; r += TPB) {
    const int k = (r / QW + 1) * CW + r % QW + 1;
    if constexpr (two_floats<R>())
      unit_normal(sm.c, sm.cl, k, CW, sm.e, sm.nx[r], sm.ny[r]);
    else
      unit_normal(sm.c, k, CW, I.pd.eta_n2, sm.nx[r], sm.ny[r]);
  }
  __syncthreads();
}

// Deterministic sum over the block of NV values per thread (FP64); the result
// is valid in thread 0.
template <int NV>
__device__ __forceinline__ void block_sum(double (&v)[NV], double* sh) {
  for (int j = 0; j < NV; j++) sh[j * TPB + threadIdx.x] = v[j];
  __syncthreads();
  for (int s = TPB / 2; s > 0; s >>= 1) {
    if ((int)threadIdx.x < s)
      for (int j = 0; j < NV; j++) sh[j * TPB + threadIdx.x] += sh[j * TPB + threadIdx.x + s];
    __syncthreads();
  }
  for (int j = 0; j < NV; j++) v[j] = sh[j * TPB];
}

// ---------------------------------------------------------------- observable
// Partial sums (sum c u_y, sum c) of each tile, FP64, into part[tile][4].
template <class R>
__global__ void __launch_bounds__(TPB)
observable_kernel(Geo G, const InstDev* __restrict__ d, State<R> st, double* __restrict__ part) {
  __shared__ TileA<double> sm;
  __shared__ double sh[2 * TPB];
  const InstDev& I = *d;
  const Phys<double>& P = I.pd;
  const int x0 = (int)(blockIdx.x % G.tx) * TX, y0 = (int)(blockIdx.x / G.tx) * TY;
  // the tile in FP64: the FP32 state's parts added exactly
  for (int r = threadIdx.x; r < CH * CW; r += TPB) {
    const int rx = r % CW, ry = r / CW;
    const int y = y0 - 2 + ry;
    if (y < -2 || y > G.ny + 1) {
      sm.c[r] = 0.0;
      continue;
    }
    const int x = wrap_col(x0 - 2 + rx, G.nx), ym = mirror_row(y, G.ny);
    const int64_t k = (int64_t)ym * G.nx + x;
    sm.c[r] = (double)st.C[k];
    if constexpr (two_floats<R>()) sm.c[r] += (double)st.Cl[k];
    if (rx >= 1 && rx <= TX + 2 && ry >= 1 && ry <= TY + 2) {
      double T = 0.0;
      if (y >= -1 && y <= G.ny) {
        T = (double)st.T[k];
        if constexpr (two_floats<R>()) T += (double)st.Tl[k];
        if (y != ym) T = 2.0 * (y < 0 ? I.Tbot[x] : I.Ttop[x]) - T;
      }
      sm.T[(ry - 1) * QW + rx - 1] = T;
    }
  }
  __syncthreads();
  for (int r = threadIdx.x; r < QW * QH; r += TPB) {
    const int k = (r / QW + 1) * CW + r % QW + 1;
    unit_normal(sm.c, k, CW, P.eta_n2, sm.nx[r], sm.ny[r]);
  }
  __syncthreads();
  const int tx = threadIdx.x % TX, ty = tile_row();
  const int x = x0 + tx, y = y0 + ty;
  double acc[2] = {0.0, 0.0};
  if (x < G.nx && y < G.ny) {
    const int64_t k = (int64_t)y * G.nx + x;
    const int kc = (ty + 2) * CW + tx + 2, kq = (ty + 1) * QW + tx + 1;
    double gcx, gcy, gTx, gTy, d1, d2, dum;
    tgrad(sm.c, kc, CW, gcx, gcy);
    tgrad(sm.T, kq, QW, gTx, gTy);
    tgrad(sm.nx, kq, QW, d1, dum);
    tgrad(sm.ny, kq, QW, dum, d2);
    const double cc = sm.c[kc];
    const double sigma = P.sigma0 - P.sigmaT * (sm.T[kq] - P.Tref);
    const double g2 = gcx * gcx + gcy * gcy;
    const double cap = -sigma * (d1 + d2) * P.ea * sqrt(g2);
    const double mar = -P.sigmaT * P.ea;
    const double Fy = cap * gcy + mar * (g2 * gTy - (gcx * gTx + gcy * gTy) * gcy) + P.Fby;
    auto f = [&](int i) { return (double)st.Q[(int64_t)i * G.N + k]; };
    const double jy = f(2) - f(4) + f(5) + f(6) - f(7) - f(8);
    const double uy = jy * (3.0 * P.inv_rho) + 0.5 * Fy * P.inv_rho;
    acc[0] = cc * uy;
    acc[1] = cc;
  }
  block_sum(acc, sh);
  if (threadIdx.x == 0) {
    part[blockIdx.x * (int64_t)4] = acc[0];
    part[blockIdx.x * (int64_t)4 + 1] = acc[1];
  }
}

// out[0..3] = the sums of part[n][4] in a fixed order
__global__ void reduce_parts(const double* __restrict__ part, int64_t n, double* __restrict__ out) {
  __shared__ double sh[4 * TPB];
  double v[4] = {0, 0, 0, 0};
  for (int64_t b = threadIdx.x; b < n; b += TPB)
    for (int j = 0; j < 4; j++) v[j] += part[b * 4 + j];
  block_sum(v, sh);
  if (threadIdx.x == 0)
    for (int j = 0; j < 4; j++) out[j] = v[j];
}

// ---------------------------------------------------------------- A
// Stencil-output adjoint planes written by A.
enum { S_GCX = 0, S_GCY, S_LAP, S_GTX, S_GTY, S_GPX, S_GPY, S_KAP, S_C, S_P, S_T, S_NUM };

// FP32: the cell's f, hbar and b and the terms of its neighbourhood come
// through shared memory by asynchronous copies issued before the tile's two
// barriers, so that their latency is paid once and not per direction, without
// the 45 registers that would otherwise hold them (31 -> 27 us at 256 x 512).
template <class R>
struct StageA {  // FP64: unused (that kernel is bound by its arithmetic)
  static constexpr int NB = two_floats<R>() ? 27 : 0, NF = two_floats<R>() ? 18 : 0;
  R b[NB ? NB * TPB : 1], fh[NF ? NF * TPB : 1];
  R t[NB ? 3 * QW * QH : 1];
};
__device__ __forceinline__ void copy_async4(void* dst, const void* src) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(
                   static_cast<uint32_t>(__cvta_generic_to_shared(dst))),
               "l"(src)
               : "memory");
}

// a: the adjoint of the next state (27 planes) and at: its terms of the cell
// (3 planes; NULL: none); a NULL: zero.  part[tile][0..2] gains the tile's
// theta sums.
template <class R>
__global__ void __launch_bounds__(TPB, sizeof(R) == 4 ? 2 : 1)
adjoint_A(Geo G, const InstDev* __restrict__ d, State<R> st, const R* a, const R* at,
          const double* obs, double wl, R* __restrict__ aout, R* __restrict__ S,
          double* __restrict__ part) {
  grid_wait();
  extern __shared__ __align__(16) char smem_raw[];
  TileA<R>& sm = *reinterpret_cast<TileA<R>*>(smem_raw);
  StageA<R>& sg = *reinterpret_cast<StageA<R>*>(smem_raw + sizeof(TileA<R>));
  // (the block sums reuse the tile: 3 TPB doubles)
  double* sh = reinterpret_cast<double*>(smem_raw);
  constexpr bool STAGED = two_floats<R>();
  const InstDev& I = *d;
  const Phys<R>& P = phys<R>(I);
  const R I3 = R(ICS2), H = R(0.5), ONE = R(1), TWO = R(2);
  const int x0 = (int)(blockIdx.x % G.tx) * TX, y0 = (int)(blockIdx.x / G.tx) * TY;
  const int tx = threadIdx.x % TX, ty = tile_row();
  const int x = x0 + tx, y = y0 + ty;
  const uint32_t k = (uint32_t)y * (uint32_t)G.nx + (uint32_t)x;  // (nx ny < 2^31)
  const bool cell = x < G.nx && y < G.ny;
  // b_j(x) = a_j(x + xi_j), or +-a_jbar(x) where x + xi_j is beyond a wall
  auto beyond = [&](int j) { return EY(j) > 0 ? y == G.ny - 1 : (EY(j) < 0 && y == 0); };
  auto b_plane = [&](int l, int j) {
    return a + (int64_t)(l * 9 + (beyond(j) ? OPP(j) : j)) * G.N;
  };
  auto b_cell = [&](int j) -> uint32_t {
    if (beyond(j)) return k;
    const int xs = EX(j) == 0 ? x
                   : EX(j) > 0 ? (x == G.nx - 1 ? 0 : x + 1)
                               : (x == 0 ? G.nx - 1 : x - 1);
    return (uint32_t)(y + EY(j)) * (uint32_t)G.nx + (uint32_t)xs;
  };
  if constexpr (STAGED) {
    if (cell) {
#pragma unroll
      for (int j = 0; j < 9; j++) {
        copy_async4(&sg.fh[j * TPB + threadIdx.x], st.Q + (int64_t)j * G.N + k);
        copy_async4(&sg.fh[(9 + j) * TPB + threadIdx.x], st.Q + (int64_t)(18 + j) * G.N + k);
        if (a != nullptr) {
          const uint32_t kt = b_cell(j);
#pragma unroll
          for (int l = 0; l < 3; l++)
            copy_async4(&sg.b[(9 * l + j) * TPB + threadIdx.x], b_plane(l, j) + kt);
        }
      }
    }
    if (at != nullptr) {
      for (int r = threadIdx.x; r < QW * QH; r += TPB) {
        const int yr = y0 - 1 + r / QW;
        if (yr < 0 || yr >= G.ny) continue;
        const uint32_t kt = (uint32_t)yr * (uint32_t)G.nx +
                            (uint32_t)wrap_col(x0 - 1 + r % QW, G.nx);
#pragma unroll
        for (int l = 0; l < 3; l++)
          copy_async4(&sg.t[l * QW * QH + r], at + (int64_t)l * G.N + kt);
      }
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
  }
  load_tile(sm, G, I, st, x0, y0);
  if constexpr (STAGED) {
    asm volatile("cp.async.wait_group 0;" ::: "memory");
    __syncthreads();  // (the terms are other threads' copies)
  }
  double acc[3] = {0, 0, 0};
  if (cell) {
    auto pull_b = [&](int l, int j) -> R {
      if (a == nullptr) return R(0);
      R v;
      if constexpr (STAGED) {
        v = sg.b[(9 * l + j) * TPB + threadIdx.x];
        if (at != nullptr)
          v += sg.t[l * QW * QH + (beyond(j) ? (ty + 1) * QW + tx + 1
                                             : (ty + 1 + EY(j)) * QW + tx + 1 + EX(j))];
      } else {
        const uint32_t kt = b_cell(j);
        v = b_plane(l, j)[kt];
        if (at != nullptr) v += (at + (int64_t)l * G.N)[kt];
      }
      return (l == 2 && beyond(j)) ? -v : v;
    };
    R f[9], h[9];
#pragma unroll
    for (int i = 0; i < 9; i++) {
      f[i] = STAGED ? sg.fh[i * TPB + threadIdx.x] : (st.Q + (int64_t)i * G.N)[k];
      h[i] = STAGED ? sg.fh[(9 + i) * TPB + threadIdx.x] : (st.Q + (int64_t)(18 + i) * G.N)[k];
    }
    const int kc = (ty + 2) * CW + tx + 2, kq = (ty + 1) * QW + tx + 1;
    const R cc = sm.c[kc], pp = sm.p[kq], TT = sm.T[kq];
    R gcx, gcy, gTx, gTy, gpx, gpy, d1, d2, dum;
    tgrad(sm.c, kc, CW, gcx, gcy);
    const R lapc = tlap(sm.c, kc, CW);
    tgrad(sm.T, kq, QW, gTx, gTy);
    tgrad(sm.p, kq, QW, gpx, gpy);
    tgrad(sm.nx, kq, QW, d1, dum);
    tgrad(sm.ny, kq, QW, dum, d2);
    const R kappa = d1 + d2;
    // forward (same expressions as the FP64 step)
    const R mu = P.beta2 * cc * (cc - ONE) * (TWO * cc - ONE) - P.eps2 * lapc;
    const R sigma = P.sigma0 - P.sigmaT * (TT - P.Tref);
    const R g2 = gcx * gcx + gcy * gcy;
    const R gabs = sqrt(g2);
    const R cdT = gcx * gTx + gcy * gTy;
    const R ea = P.ea;
    const R cap = -sigma * kappa * ea * gabs;
    const R mar = -P.sigmaT * ea;
    const R Fx = cap * gcx + mar * (g2 * gTx - cdT * gcx) + P.Fbx;
    const R Fy = cap * gcy + mar * (g2 * gTy - cdT * gcy) + P.Fby;
    R jx = f[1] - f[3];
    jx = jx + f[5];
    jx = jx - f[6];
    jx = jx - f[7];
    jx = jx + f[8];
    R jy = f[2] - f[4];
    jy = jy + f[5];
    jy = jy + f[6];
    jy = jy - f[7];
    jy = jy - f[8];
    // reciprocal products: FP64 divisions would dominate this kernel
    const R rcs2 = P.rcs2, irho = P.inv_rho, irc = R(ICS2) * irho;
    const R ux = jx * irc + H * Fx * irho;
    const R uy = jy * irc + H * Fy * irho;
    const R eta = P.eta1 + cc * P.deta;
    const R lam = P.lam1 + cc * P.dlam;
    const R tau_f = eta * irc + H;
    const R omega_f = ONE / tau_f;
    const R ircv = R(ICS2) * P.inv_rho_cv;
    const R tau_h = lam * ircv;
    const R omega_T = TWO / (TWO * tau_h + ONE);
    const R omega_g = P.omega_g;
    const R af = ONE - H * omega_f, ag = ONE - H * omega_g, aT = ONE - H * omega_T;
    const R uu = (ux * ux + uy * uy) * I3;
    const R Gm = P.Gm;
    const R W0 = WGT<R>(0);
    const R Gx = Fx - gpx, Gy = Fy - gpy;
    const R rcvT = P.rho * P.cv * TT;

    // ---- reverse through the collisions (unrolled: the directions' components
    // fold, and the loads of b are in flight together)
    R fb[9], gbr[9], hb[9];
    R cb = 0, pb = 0, Tb = 0, uxb = 0, uyb = 0, Fxb = 0, Fyb = 0, Gxb = 0, Gyb = 0;
    R uub = 0, Hib = 0, H0b = 0, rcvTb = 0, wfb = 0, wTb = 0, afb = 0, aTb = 0;
    const R ogf = ONE - omega_g, ohf = ONE - omega_T, off = ONE - omega_f;
#pragma unroll
    for (int i = 0; i < 9; i++) {
      const R W = WGT<R>(i);
      const R xu = xi_dot(i, ux, uy) * I3;
      const R hq = H * (xu * xu - uu);
      const R Gam = W * (ONE + xu + hq);
      const R q = xu + hq;
      const R dx = R(EX(i)) - ux, dy = R(EY(i)) - uy;
      const R fsd = Fx * dx + Fy * dy;
      const R shv = (Gx * dx + Gy * dy) * irc;  // Fbar.(xi - u) / (rho c_s^2)
      const R bf = pull_b(0, i), bg = pull_b(1, i), bh = pull_b(2, i);
      // h: ho = h - wT (h - heq) + aT shv heq, heq = rcvT Gam
      const R heq = rcvT * Gam;
      hb[i] = bh * ohf;
      wTb += bh * (heq - h[i]);
      const R hsb = bh * aT;
      aTb += bh * (shv * heq);
      const R heqb = bh * omega_T + hsb * shv;
      rcvTb += heqb * Gam;
      R Gamb = heqb * rcvT;
      // g: go = g - wg (g - geq) + ag c shv Gam, geq = W (H + c q)
      gbr[i] = bg * ogf;
      const R geqb = bg * omega_g * W;
      const R sgb = bg * ag * Gam;
      Gamb += bg * ag * (cc * shv);
      cb += sgb * shv + geqb * q;
      if (i == 0) H0b += geqb; else Hib += geqb;
      R qb = geqb * cc;
      // the adjoint of shv's numerator, of both
      const R m = (hsb * heq + sgb * cc) * irc;
      Gxb += m * dx;
      Gyb += m * dy;
      // f: fo = f - wf (f - feq) + af fsd Gam, feq = W (p + rcs2 q)
      fb[i] = bf * off;
      wfb += bf * (W * (pp + rcs2 * q) - f[i]);
      const R feqb = bf * omega_f * W;
      const R fsb = bf * af;
      afb += bf * (fsd * Gam);
      const R n = fsb * Gam;
      Fxb += n * dx;
      Fyb += n * dy;
      Gamb += fsb * fsd;
      pb += feqb;
      qb += feqb * rcs2;
      // dx = EX - ux
      uxb -= m * Gx + n * Fx;
      uyb -= m * Gy + n * Fy;
      // Gam = W (1 + xu + hq), q = xu + hq, hq = (xu^2 - uu)/2
      const R hqb = Gamb * W + qb;
      uub -= H * hqb;
      const R xub = (hqb + hqb * xu) * I3;
      if (EX(i) != 0) uxb += EX(i) > 0 ? xub : -xub;
      if (EY(i) != 0) uyb += EY(i) > 0 ? xub : -xub;
    }
    Tb += rcvTb * P.rho * P.cv;
    Fxb += Gxb;
    Fyb += Gyb;
    R gpxb = -Gxb, gpyb = -Gyb;
    R mub = Hib * Gm * I3;
    cb += H0b * (ONE / W0);
    mub -= H0b * (ONE - W0) * Gm * (I3 / W0);
    uxb += uub * TWO * ux * I3;
    uyb += uub * TWO * uy * I3;
    wTb -= H * aTb;
    wfb -= H * afb;
    const R tauhb = -wTb * omega_T * omega_T;
    const R lamb = tauhb * ircv;
    const R taufb = -wfb * omega_f * omega_f;
    const R etab = taufb * irc;
    cb += etab * P.deta + lamb * P.dlam;
    R th_eta = etab * cc * P.eta1;  // d eta / d (eta2/eta1) = c eta1
    R th_lam = lamb * cc * P.lam1;
    // the observable at this step: l = A/B, dl/dc = u_y/B - A/B^2, dl/du_y = c/B
    if (wl != 0.0) {
      const R A = (R)obs[0], B = (R)obs[1], wr = (R)wl;
      cb += wr * (uy / B - A / (B * B));
      uyb += wr * cc / B;
    }
    // u = j/(rho cs2) + F/(2 rho)
    const R jxb = uxb * irc, jyb = uyb * irc;
    Fxb += H * uxb * irho;
    Fyb += H * uyb * irho;
#pragma unroll
    for (int i = 1; i < 9; i++) fb[i] += xi_dot(i, jxb, jyb);
    // F = cap gc + mar (g2 gT - cdT gc) + rho a
    const R capb = Fxb * gcx + Fyb * gcy;
    const R marb = Fxb * (g2 * gTx - cdT * gcx) + Fyb * (g2 * gTy - cdT * gcy);
    R gcxb = Fxb * cap - Fxb * mar * cdT;
    R gcyb = Fyb * cap - Fyb * mar * cdT;
    R g2b = mar * (Fxb * gTx + Fyb * gTy);
    R gTxb = mar * g2 * Fxb, gTyb = mar * g2 * Fyb;
    const R cdTb = -mar * (Fxb * gcx + Fyb * gcy);
    R th_sig = -marb * ea;
    // cap = -sigma kappa ea gabs
    const R sigb = -capb * kappa * ea * gabs;
    const R kapb = -capb * sigma * ea * gabs;
    const R gabsb = -capb * sigma * kappa * ea;
    gcxb += cdTb * gTx;
    gcyb += cdTb * gTy;
    gTxb += cdTb * gcx;
    gTyb += cdTb * gcy;
    if (gabs > R(0)) g2b += gabsb / (TWO * gabs);
    gcxb += TWO * g2b * gcx;
    gcyb += TWO * g2b * gcy;
    // sigma = sigma0 - sigmaT (T - Tref)
    Tb += -sigb * P.sigmaT;
    th_sig += -sigb * (TT - P.Tref);
    // mu = 2 beta c (c-1)(2c-1) - eps^2 lap c
    cb += mub * P.beta2 * (R(6) * cc * cc - R(6) * cc + ONE);
    const R lapb = -mub * P.eps2;

#pragma unroll
    for (int i = 0; i < 9; i++) {
      (aout + (int64_t)i * G.N)[k] = fb[i];
      (aout + (int64_t)(9 + i) * G.N)[k] = gbr[i];
      (aout + (int64_t)(18 + i) * G.N)[k] = hb[i];
    }
    (S + (int64_t)S_GCX * G.N)[k] = gcxb;
    (S + (int64_t)S_GCY * G.N)[k] = gcyb;
    (S + (int64_t)S_LAP * G.N)[k] = lapb;
    (S + (int64_t)S_GTX * G.N)[k] = gTxb;
    (S + (int64_t)S_GTY * G.N)[k] = gTyb;
    (S + (int64_t)S_GPX * G.N)[k] = gpxb;
    (S + (int64_t)S_GPY * G.N)[k] = gpyb;
    (S + (int64_t)S_KAP * G.N)[k] = kapb;
    (S + (int64_t)S_C * G.N)[k] = cb;
    (S + (int64_t)S_P * G.N)[k] = pb;
    (S + (int64_t)S_T * G.N)[k] = Tb;
    acc[0] = (double)th_sig;
    acc[1] = (double)th_eta;
    acc[2] = (double)th_lam;
  }
  __syncthreads();  // the tile is read
  block_sum(acc, sh);
  if (threadIdx.x == 0)
    for (int j = 0; j < 3; j++) part[blockIdx.x * (int64_t)4 + j] += acc[j];
}

// ---------------------------------------------------------------- B
// kappa(X) = sum_i (w_i/cs2) xi_i . n(X + xi_i)  =>  n-bar(Y) = sum_i
// (w_i/cs2) xi_i kappa-bar(Y - xi_i) over cells Y - xi_i; then through
// n = v / s, s = sqrt(|v|^2 + eta_n^2): v-bar = n-bar/s - v (v.n-bar)/s^3.
// v-bar is needed on the tile and its ring of 1, ghost rows -1 and ny
// included, and one row further up (row ny, an image of which row ny - 2
// holds, may lie two rows above the tile); c and kappa-bar one cell further.
template <class R>
struct TileB {
  static constexpr int CH = TY + 5, QH = TY + 3;  // rows y0 - 2 .., y0 - 1 ..
  R c[CH * CW], kap[CH * CW];
  R vx[QH * QW], vy[QH * QW];
  R s[S_KAP][QH * QW];  // S_GCX .. S_GPY
};

template <class R>
__global__ void __launch_bounds__(TPB)
adjoint_B(Geo G, const InstDev* __restrict__ d, State<R> st, const R* S,
          R* __restrict__ tout) {
  grid_wait();
  using Tl = TileB<R>;
  extern __shared__ __align__(16) char smem_raw[];
  Tl& sm = *reinterpret_cast<Tl*>(smem_raw);
  const InstDev& I = *d;
  const int nx = G.nx, ny = G.ny;
  const int x0 = (int)(blockIdx.x % G.tx) * TX, y0 = (int)(blockIdx.x / G.tx) * TY;
  for (int r = threadIdx.x; r < Tl::CH * CW; r += TPB) {
    const int rx = r % CW, ry = r / CW;
    const int y = y0 - 2 + ry, x = wrap_col(x0 - 2 + rx, nx);
    const bool cell = y >= 0 && y < ny;
    const int64_t k = (int64_t)y * nx + x;
    const bool has_c = y >= -2 && y <= ny + 1;
    const int64_t kc = (int64_t)mirror_row(y, ny) * nx + x;
    sm.c[r] = has_c ? st.C[kc] : R(0);
    sm.kap[r] = cell ? S[(int64_t)S_KAP * G.N + k] : R(0);
    if (rx >= 1 && rx <= TX + 2 && ry >= 1 && ry <= Tl::QH) {
      const int q = (ry - 1) * QW + rx - 1;
#pragma unroll
      for (int j = 0; j < S_KAP; j++) sm.s[j][q] = cell ? S[(int64_t)j * G.N + k] : R(0);
    }
  }
  __syncthreads();
  const R en2 = phys<R>(I).eta_n2;
  for (int r = threadIdx.x; r < QW * Tl::QH; r += TPB) {
    const int k = (r / QW + 1) * CW + r % QW + 1, y = y0 - 1 + r / QW;
    R vx = R(0), vy = R(0);
    if (y <= ny) {
      // the transposed divergence: minus the gradient stencil of kappa-bar
      R nbx, nby, gx, gy;
      tgrad(sm.kap, k, CW, nbx, nby);
      tgrad(sm.c, k, CW, gx, gy);
      const R is = R(1) / sqrt(gx * gx + gy * gy + en2);
      const R vn = (gx * nbx + gy * nby) * is * is;
      vx = (gx * vn - nbx) * is;
      vy = (gy * vn - nby) * is;
    }
    sm.vx[r] = vx;
    sm.vy[r] = vy;
  }
  __syncthreads();
  const int tx = threadIdx.x % TX, ty = tile_row();
  const int x = x0 + tx, y = y0 + ty;
  if (x >= nx || y >= ny) return;
  const int64_t k = (int64_t)y * nx + x;
  R cb = S[(int64_t)S_C * G.N + k];
  R pb = S[(int64_t)S_P * G.N + k];
  R Tb = S[(int64_t)S_T * G.N + k];
  // Laplacian centre term
  R sw = R(0);
#pragma unroll
  for (int i = 1; i < 9; i++) sw += WGT<R>(i);
  cb += R(-2) * sw * R(ICS2) * sm.s[S_LAP][(ty + 1) * QW + tx + 1];
  // the transposed stencils at row qy, which holds the cell's value (qy = y)
  // or an image of it (a ghost row); c images reach two rows, p and T one
  auto gather = [&](int qy) {
    const bool depth1 = qy >= -1 && qy <= ny;
    const R tsign = qy == y ? R(1) : R(-1);
#pragma unroll
    for (int i = 1; i < 9; i++) {
      const int Y = qy - EY(i);
      if (Y < -1 || Y > ny) continue;
      const int q = (Y - y0 + 1) * QW + tx + 1 - EX(i);
      const R wa = WGT<R>(i) * R(ICS2);
      const R ex = R(EX(i)), ey = R(EY(i));
      // (the fields are zero off the cells, v-bar lives on the ghost rows too)
      cb += wa * (ex * (sm.s[S_GCX][q] + sm.vx[q]) + ey * (sm.s[S_GCY][q] + sm.vy[q]) +
                  R(2) * sm.s[S_LAP][q]);
      if (depth1) {
        pb += wa * (ex * sm.s[S_GPX][q] + ey * sm.s[S_GPY][q]);
        Tb += tsign * wa * (ex * sm.s[S_GTX][q] + ey * sm.s[S_GTY][q]);
      }
    }
  };
  gather(y);
  if (y < 2) gather(-1 - y);
  if (y >= ny - 2) gather(2 * ny - 1 - y);
  tout[k] = pb;
  tout[G.N + k] = cb;
  tout[2 * G.N + k] = Tb / (phys<R>(I).rho * phys<R>(I).cv);
}

// The adjoint state as 27 FP64 planes (a_lj + t_l).
template <class R>
__global__ void finish_kernel(Geo G, const R* __restrict__ a, const R* __restrict__ at,
                              double* __restrict__ out) {
  for (int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; k < G.N;
       k += (int64_t)gridDim.x * blockDim.x)
    for (int l = 0; l < 3; l++) {
      const double t = (double)at[l * G.N + k];
      for (int i = 0; i < 9; i++)
        out[(int64_t)(9 * l + i) * G.N + k] = (double)a[(int64_t)(9 * l + i) * G.N + k] + t;
    }
}

template <class R>
__global__ void dT0_kernel(Geo G, const InstDev* __restrict__ d, const R* __restrict__ a,
                           const R* __restrict__ at, double* __restrict__ out) {
  const double rcv = d->pd.rho * d->pd.cv;
  for (int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; k < G.N;
       k += (int64_t)gridDim.x * blockDim.x) {
    const double t = (double)at[2 * G.N + k];
    double s = 0.0;
    for (int i = 0; i < 9; i++)
      s += WGT<double>(i) * ((double)a[(int64_t)(18 + i) * G.N + k] + t);
    out[k] = rcv * s;
  }
}

template <class R>
State<R> view(const Geo& G, const void* state) {
  const R* q = static_cast<const R*>(state);
  return State<R>{q, q + 27 * G.N, q + 28 * G.N, q + 29 * G.N, q + 30 * G.N,
                  q + 31 * G.N};
}
int cell_grid(const Geo& G) {
  const int64_t b = (G.N + 255) / 256;
  return (int)(b < 65535 ? b : 65535);
}

template <class S>
cudaError_t state_t(const InstDev* d, const Geo& G, int parity, void* out, cudaStream_t s) {
  const dim3 grid((G.nx + 255) / 256, G.ny < 65535 ? G.ny : 65535);
  return launch_early(state_kernel<S>, grid, 256, 0, s, G, d, parity,
                      static_cast<typename S::C*>(out));
}

template <class R>
cudaError_t step_t(const InstDev* d, const Geo& G, const State<R>& st, const R* a, const R* at,
                   double wl, const double* obs, R* aout, R* tout, R* S, double* part,
                   cudaStream_t s) {
  const unsigned tiles = (unsigned)G.tx * G.ty;
  static_assert(sizeof(TileB<R>) <= 48 * 1024, "shared memory without an opt-in");
  static_assert(sizeof(TileA<R>) >= 3 * TPB * sizeof(double), "the block sums' room");
  constexpr int smem_A = sizeof(TileA<R>) + sizeof(StageA<R>);
  static bool opted[64] = {};  // per device
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (dev < 0 || dev >= 64) return cudaErrorInvalidDevice;
  if (!opted[dev]) {
    e = cudaFuncSetAttribute(adjoint_A<R>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem_A);
    if (e != cudaSuccess) return e;
    opted[dev] = true;
  }
  e = launch_early(adjoint_A<R>, dim3(tiles), TPB, smem_A, s, G, d, st, a, at, obs, wl, aout, S,
                   part);
  if (e != cudaSuccess) return e;
  return launch_early(adjoint_B<R>, dim3(tiles), TPB, sizeof(TileB<R>), s, G, d, st, S, tout);
}

}  // namespace adj

using namespace adj;

size_t adjoint_real_bytes(bool fp32) { return fp32 ? 4 : 8; }
int64_t adjoint_state_planes(bool fp32) { return fp32 ? 32 : 27; }
int64_t adjoint_vector_planes() { return 27 + 3; }
int64_t adjoint_scratch_planes() { return S_NUM; }
int64_t adjoint_part_doubles(int nx, int ny) {
  const Geo G = make_geo(nx, ny);
  return (int64_t)4 * G.tx * G.ty;
}

cudaError_t launch_adjoint_state(int storage, const InstDev* d, int nx, int ny, int parity,
                                 void* state, cudaStream_t s) {
  const Geo G = make_geo(nx, ny);
  switch (storage) {
    case ST_F64: return state_t<StF64>(d, G, parity, state, s);
    case ST_F32: return state_t<StF32>(d, G, parity, state, s);
    case ST_F16DEV: return state_t<StF16>(d, G, parity, state, s);
    case ST_BF16DEV: return state_t<StBF16>(d, G, parity, state, s);
    case ST_F16MIX: return state_t<StMix>(d, G, parity, state, s);
  }
  return cudaErrorInvalidValue;
}

cudaError_t launch_adjoint_moments(const InstDev* d, int nx, int ny, const double* Q, double* cpt,
                                   cudaStream_t s) {
  const Geo G = make_geo(nx, ny);
  moments_kernel<<<cell_grid(G), 256, 0, s>>>(G, d, Q, cpt, cpt + G.N, cpt + 2 * G.N);
  return cudaGetLastError();
}

cudaError_t launch_observable(const InstDev* d, int nx, int ny, bool fp32, const void* Q,
                              const void* cpt, double* part, double* out4, cudaStream_t s) {
  const Geo G = make_geo(nx, ny);
  const unsigned tiles = (unsigned)G.tx * G.ty;
  cudaError_t e = cudaMemsetAsync(part, 0, sizeof(double) * 4 * tiles, s);
  if (e != cudaSuccess) return e;
  if (fp32) {
    observable_kernel<float><<<tiles, TPB, 0, s>>>(G, d, view<float>(G, Q), part);
  } else {
    const double* c = static_cast<const double*>(cpt);
    const State<double> st{static_cast<const double*>(Q), c, c + G.N, c + 2 * G.N, nullptr, nullptr};
    observable_kernel<double><<<tiles, TPB, 0, s>>>(G, d, st, part);
  }
  reduce_parts<<<1, TPB, 0, s>>>(part, tiles, out4);
  return cudaGetLastError();
}

cudaError_t launch_adjoint_step(const InstDev* d, int nx, int ny, bool fp32, const void* Q,
                                const void* cpt, const void* a, const void* at, double wl,
                                const double* obs, void* aout, void* tout, void* scratch,
                                double* part, cudaStream_t s) {
  const Geo G = make_geo(nx, ny);
  if (fp32)
    return step_t<float>(d, G, view<float>(G, Q), static_cast<const float*>(a),
                         static_cast<const float*>(at), wl, obs, static_cast<float*>(aout),
                         static_cast<float*>(tout), static_cast<float*>(scratch), part, s);
  const double* c = static_cast<const double*>(cpt);
  const State<double> st{static_cast<const double*>(Q), c, c + G.N, c + 2 * G.N, nullptr, nullptr};
  return step_t<double>(d, G, st, static_cast<const double*>(a), static_cast<const double*>(at),
                        wl, obs, static_cast<double*>(aout), static_cast<double*>(tout),
                        static_cast<double*>(scratch), part, s);
}

cudaError_t launch_adjoint_sums(const double* part, int nx, int ny, double* out4, cudaStream_t s) {
  const Geo G = make_geo(nx, ny);
  reduce_parts<<<1, TPB, 0, s>>>(part, (int64_t)G.tx * G.ty, out4);
  return cudaGetLastError();
}

cudaError_t launch_adjoint_finish(int nx, int ny, bool fp32, const void* a, const void* at,
                                  double* out, cudaStream_t s) {
  const Geo G = make_geo(nx, ny);
  if (fp32)
    finish_kernel<float><<<cell_grid(G), 256, 0, s>>>(G, static_cast<const float*>(a),
                                                      static_cast<const float*>(at), out);
  else
    finish_kernel<double><<<cell_grid(G), 256, 0, s>>>(G, static_cast<const double*>(a),
                                                       static_cast<const double*>(at), out);
  return cudaGetLastError();
}

cudaError_t launch_adjoint_dT0(const InstDev* d, int nx, int ny, bool fp32, const void* a,
                               const void* at, double* dT0, cudaStream_t s) {
  const Geo G = make_geo(nx, ny);
  if (fp32)
    dT0_kernel<float><<<cell_grid(G), 256, 0, s>>>(G, d, static_cast<const float*>(a),
                                                   static_cast<const float*>(at), dT0);
  else
    dT0_kernel<double><<<cell_grid(G), 256, 0, s>>>(G, d, static_cast<const double*>(a),
                                                    static_cast<const double*>(at), dT0);
  return cudaGetLastError();
}

}  // namespace lbe
