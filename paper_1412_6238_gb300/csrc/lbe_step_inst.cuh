// Instantiation of the step / field kernels for one storage type.  Included
// by lbe_step_<storage>.cu with LBE_ST (policy), LBE_SUFFIX and LBE_ALL_TILES
// defined.
#include <algorithm>

#include "lbe_launch.h"
#include "lbe_tile.cuh"
#if LBE_STASH
#include "lbe_stash.cuh"
#endif
#if !LBE_ALL_TILES  // FP64
#include "lbe_split.cuh"
#endif

#define LBE_CAT2(a, b) a##b
#define LBE_CAT(a, b) LBE_CAT2(a, b)

namespace lbe {

namespace {
template <int TX, int TY>
cudaError_t launch_one(const InstDev* d, int n, int64_t total, int parity, int grid,
                       StepCount seed, cudaStream_t s) {
  if (grid <= 0) grid = 1;
  if ((int64_t)grid > total) grid = (int)total;
  return launch_early(tile_kernel<LBE_ST, TX, TY, 0>, dim3(grid), TX * TY, 0, s, d, n, total,
                      parity, FieldOut{}, seed);
}
template <int TX, int TY>
int occ_one() {
  int b = 0;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&b, tile_kernel<LBE_ST, TX, TY, 0>, TX * TY,
                                                    0) != cudaSuccess)
    return 0;
  return b;
}
}  // namespace

cudaError_t LBE_CAT(launch_step_, LBE_SUFFIX)(int tile, const InstDev* d, int n, int64_t total,
                                               int parity, int grid, StepCount seed,
                                               cudaStream_t s) {
  switch (tile) {
#if LBE_ALL_TILES
    case 0: return launch_one<32, 8>(d, n, total, parity, grid, seed, s);
    case 1: return launch_one<64, 4>(d, n, total, parity, grid, seed, s);
    case 2: return launch_one<32, 16>(d, n, total, parity, grid, seed, s);
    case 3: return launch_one<64, 8>(d, n, total, parity, grid, seed, s);
    case 4: return launch_one<128, 4>(d, n, total, parity, grid, seed, s);
#else
    case SPLIT_TILE:
      grid = (int)std::min<int64_t>(std::max(grid, 1), total);
      return launch_early(split_kernel, dim3(grid), SPLIT_THREADS, 0, s, d, n, total, parity);
    case NARROW_TILE: return launch_one<4, 8>(d, n, total, parity, grid, seed, s);
    case F64_TILE: return launch_one<16, 8>(d, n, total, parity, grid, seed, s);
#endif
    default: return cudaErrorInvalidValue;
  }
}

int LBE_CAT(occupancy_, LBE_SUFFIX)(int tile) {
  switch (tile) {
#if LBE_ALL_TILES
    case 0: return occ_one<32, 8>();
    case 1: return occ_one<64, 4>();
    case 2: return occ_one<32, 16>();
    case 3: return occ_one<64, 8>();
    case 4: return occ_one<128, 4>();
#else
    case SPLIT_TILE: {
      int b = 0;
      return cudaOccupancyMaxActiveBlocksPerMultiprocessor(&b, split_kernel, SPLIT_THREADS, 0) ==
                     cudaSuccess ? b : 0;
    }
    case NARROW_TILE: return occ_one<4, 8>();
    case F64_TILE: return occ_one<16, 8>();
#endif
    default: return 0;
  }
}

#if LBE_PCORR
// The pre-pass of a varying density or the dissipation term, over a work list of
// tiles of PRE_SHAPE, and the pass that collides from what it left in `drive`.
namespace {
constexpr TileShape PRE = TILE_SHAPES[pre_shape(LBE_ST::kind)];
}
cudaError_t LBE_CAT(pcorr_, LBE_SUFFIX)(const InstDev* d, int n, int64_t total, int parity,
                                         int grid, cudaStream_t s) {
  if (grid <= 0) grid = 1;
  if ((int64_t)grid > total) grid = (int)total;
  return launch_early(tile_kernel<LBE_ST, PRE.tx, PRE.ty, 2>, dim3(grid), PRE.tx * PRE.ty, 0, s, d,
                      n, total, parity, FieldOut{}, StepCount{});
}
cudaError_t LBE_CAT(drive_, LBE_SUFFIX)(const InstDev* d, int n, int64_t parts, int parity,
                                         int grid, cudaStream_t s) {
  return launch_early(drive_kernel<LBE_ST, PRE.tx, PRE.ty, DRIVE_THREADS>, dim3((unsigned)grid),
                      DRIVE_THREADS, 0, s, d, n, parts, parity);
}
#endif

cudaError_t LBE_CAT(fields_, LBE_SUFFIX)(const InstDev* d, int64_t tiles, int parity, const FieldOut& out,
                                          cudaStream_t s) {
  if (tiles <= 0) return cudaSuccess;
  const unsigned grid = (unsigned)(tiles < 2147483647 ? tiles : 2147483647);
  tile_kernel<LBE_ST, 32, 8, 1><<<grid, 256, 0, s>>>(d, 1, tiles, parity, out, StepCount{});
  return cudaGetLastError();
}

#if LBE_STASH
namespace {
template <int NC, bool VAR, bool OWN, bool EXPORT = false>
bool stash_attr() {
  static bool done[64] = {};
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return false;
  if (!done[dev]) {
    if (cudaFuncSetAttribute(stash_kernel<LBE_ST, NC, VAR, OWN, EXPORT>,
                             cudaFuncAttributeMaxDynamicSharedMemorySize,
                             StashCfg<LBE_ST, NC, VAR>::SMEM) != cudaSuccess)
      return false;
    done[dev] = true;
  }
  return true;
}
template <int NC, bool VAR, bool OWN>
cudaError_t stash_one(const InstDev* d, int n, int64_t items, int seg, int parity, int grid,
                      int* err, int poll_lim, int withhold, StepCount seed,
                      cudaStream_t s) {
  if (!stash_attr<NC, VAR, OWN>()) return cudaErrorInvalidValue;
  if (grid <= 0) grid = 1;
  if ((int64_t)grid > items) grid = (int)items;
  return launch_early(stash_kernel<LBE_ST, NC, VAR, OWN, false>, dim3(grid),
                      StashCfg<LBE_ST, NC, VAR>::THREADS, StashCfg<LBE_ST, NC, VAR>::SMEM, s, d, n,
                      items, seg, parity, err, poll_lim, withhold, seed, FieldOut{});
}
// the fields of one instance (d), seg rows an item
template <bool VAR>
cudaError_t stash_fields(const InstDev* d, int64_t items, int seg, int parity, int grid, int* err,
                         const FieldOut& out, cudaStream_t s) {
  using Cfg = StashCfg<LBE_ST, 128, VAR>;
  if (!stash_attr<128, VAR, false, true>()) return cudaErrorInvalidValue;
  stash_kernel<LBE_ST, 128, VAR, false, true>
      <<<(int)std::min<int64_t>(grid, items), Cfg::THREADS, Cfg::SMEM, s>>>(
          d, 1, items, seg, parity, err, STASH_POLLS, -1, StepCount{}, out);
  return cudaGetLastError();
}
template <int NC, bool VAR, bool OWN>
int stash_occ() {
  if (!stash_attr<NC, VAR, OWN>()) return 0;
  int b = 0;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&b, stash_kernel<LBE_ST, NC, VAR, OWN, false>,
                                                    StashCfg<LBE_ST, NC, VAR>::THREADS,
                                                    StashCfg<LBE_ST, NC, VAR>::SMEM) != cudaSuccess)
    return 0;
  return b;
}
}  // namespace

cudaError_t LBE_CAT(strip_fields_, LBE_SUFFIX)(const InstDev* d, int64_t items, int seg,
                                                int parity, int grid, int* err, bool var,
                                                const FieldOut& out, cudaStream_t s) {
  return var ? stash_fields<true>(d, items, seg, parity, grid, err, out, s)
             : stash_fields<false>(d, items, seg, parity, grid, err, out, s);
}

cudaError_t LBE_CAT(launch_stash_, LBE_SUFFIX)(const InstDev* d, int n, int64_t items, int seg,
                                                int parity, int grid, int* err, int poll_lim,
                                                int withhold, StepCount seed, bool var,
                                                bool own_ghosts, cudaStream_t s) {
#define LBE_STASH_ONE(V, O) \
  stash_one<128, V, O>(d, n, items, seg, parity, grid, err, poll_lim, withhold, seed, s)
  if (var) return own_ghosts ? LBE_STASH_ONE(true, true) : LBE_STASH_ONE(true, false);
  return own_ghosts ? LBE_STASH_ONE(false, true) : LBE_STASH_ONE(false, false);
#undef LBE_STASH_ONE
}
// resident CTAs per SM (the smaller of the two builds)
int LBE_CAT(stash_occupancy_, LBE_SUFFIX)() {
  const int o[4] = {stash_occ<128, false, false>(), stash_occ<128, true, false>(),
                    stash_occ<128, false, true>(), stash_occ<128, true, true>()};
  int m = o[0];
  for (int j = 1; j < 4; j++) m = o[j] < m ? o[j] : m;
  return m;
}
#endif

}  // namespace lbe
