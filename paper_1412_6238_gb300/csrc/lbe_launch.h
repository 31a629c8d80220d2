// Internal interface between the host API and the kernel translation units.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "lbe_common.cuh"

namespace lbe {

struct TileShape {
  int tx, ty;
};
// Kernel ids: 0..4 tile kernel with these tile shapes; 5, 6 retired (strip
// kernels with a TMA ring of whole source rows, superseded by the stash
// kernel; not built); 7 strip kernel with a per-warp stash of pulled
// populations, 128 output columns (16/32-bit storages; ty = 0: a strip
// marches over its rows), the periodic ghost columns refreshed by
// ghost_kernel after the step; 8 the same kernel writing the ghost columns
// itself (the owner of an edge cell stores it twice).
constexpr int NUM_TILE_SHAPES = 5;
constexpr int NUM_TILES = 9;
constexpr int STRIP_FIRST = 5;
constexpr int STASH_ID = 7;
constexpr int STASH_OWN_ID = 8;
// bytes allocated after an instance's two population buffers, covering the
// widest read past the end of a row of the stash kernel: a stash row of 136
// elements of up to 8 bytes from a strip start x0 <= nx - 1, against a
// pitch of at least nx + 8 elements (at most 127 x 8 bytes)
constexpr size_t ARENA_TAIL = 2048;
// The shapes kernel 0 takes with FP64 storage.  The FP64 pipe takes a warp's
// instruction at the same pace whether 4 lanes hold a cell or 32.
// SPLIT_TILE: 4 x 8 cells, their work divided among four warps (lbe_split.cuh),
// while every SM has at most SPLIT_PER_SM of them.  us a step, 4 x 101 (13
// tiles) 18, one warp a tile 39; 40 x 40 (50 tiles) 18.5, as 16 x 8 40.8; 96 x
// 96 (288) 27, 38; but 128 x 100 (416) 48, 37.5.
// NARROW_TILE: 4 x 8 cells by one warp, when every instance is at most
// NARROW_NX columns wide (4 x 4800 48.5, split 59, as 16 x 8 125; 16 x 1300 51,
// 74, 62).
// F64_TILE: else 16 x 8, of which two run side by side on an SM, so that one
// keeps the pipe busy at the other's barriers (512 x 1024: 842 us a step, 32 x
// 8 896, 8 x 8 867; 128 x 128: 40, 62, 43).
constexpr int NARROW_TILE = NUM_TILES, F64_TILE = NUM_TILES + 1, SPLIT_TILE = NUM_TILES + 2;
constexpr int NARROW_NX = 16;
constexpr int SPLIT_PER_SM = 2;
constexpr TileShape TILE_SHAPES[NUM_TILES + 3] = {{32, 8},  {64, 4},  {32, 16}, {64, 8},
                                                  {128, 4}, {124, 0}, {60, 0},  {128, 0},
                                                  {128, 0}, {4, 8},   {16, 8},  {4, 8}};
// The tiles of the pre-pass (and of the pass that collides after it).
constexpr int pre_shape(int storage) { return storage == ST_F64 ? F64_TILE : 0; }
// CTAs of the pass that collides, per tile of the pre-pass.
constexpr int DRIVE_THREADS = 128;
constexpr int drive_parts(int storage) {
  return TILE_SHAPES[pre_shape(storage)].tx * TILE_SHAPES[pre_shape(storage)].ty / DRIVE_THREADS;
}
inline bool is_strip(int tile) { return tile >= STRIP_FIRST && tile < NUM_TILES; }
inline bool is_stash(int tile) { return tile == STASH_ID || tile == STASH_OWN_ID; }

// Launches a kernel of a step so that it starts while the kernel before it on
// the stream still runs: when that one calls grid_release in every CTA, or as
// its last CTAs end.  It waits for its completion with grid_wait before it
// touches device memory that a step writes or reads.  The launch, the start of
// the CTAs and what comes before grid_wait are then off the critical path, on
// which they are a good part of a small grid's step (us a step without / with
// it: 96 x 64 FP32 8.6 / 7.1, 512 x 256 14.5 / 13.1, dissipation 512 x 256
// 35.0 / 33.8, FP64 128 x 128 37.9 / 37.4; large grids equal).
template <class... P, class... A>
inline cudaError_t launch_early(void (*kernel)(P...), dim3 grid, int threads, size_t smem,
                                cudaStream_t s, A... args) {
  cudaLaunchAttribute attr = {};
  attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr.val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = dim3(threads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cfg.attrs = &attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kernel, static_cast<P>(args)...);
}

// Does the step kernel of this storage exist for this kernel id?
bool tile_available(int storage, int tile);

// Stash strip kernel (16/32-bit storages): one step of every instance over
// `items` work items (strips x segments of seg rows); reads buf[parity],
// writes buf[parity ^ 1]; *err is set if a copy wait runs out of its
// poll_lim polls.  withhold >= 0 (test hook): the copies of that source row
// are not issued, so that the waits for it run out.
constexpr int STASH_POLLS = 1 << 22;       // polls of one bounded copy wait
constexpr int STASH_POLLS_TEST = 1 << 12;  // with the withhold test hook
// seed: the step's number, read for the random bits of the stochastic
// rounding of the 16-bit forms.  var: some instance uses a
// boundary or property variant (the kernel built with them).
cudaError_t launch_stash(int storage, const InstDev* d, int n, int64_t items, int seg, int parity,
                         int grid, int* err, int poll_lim, int withhold, StepCount seed,
                         bool var, bool own_ghosts, cudaStream_t s);
// The same kernel's fields of one instance (d_one, tile_begin 0) over `items`
// work items of seg rows of a strip.
cudaError_t launch_strip_fields(int storage, const InstDev* d_one, int64_t items, int seg,
                                int parity, int grid, int* err, bool var, const FieldOut& out,
                                cudaStream_t s);
int stash_occupancy(int storage);
cudaError_t launch_stash_f32(const InstDev* d, int n, int64_t items, int seg, int parity, int grid,
                             int* err, int poll_lim, int withhold,
                             StepCount seed, bool var,
                             bool own_ghosts, cudaStream_t s);
cudaError_t launch_stash_f16(const InstDev* d, int n, int64_t items, int seg, int parity, int grid,
                             int* err, int poll_lim, int withhold,
                             StepCount seed, bool var,
                             bool own_ghosts, cudaStream_t s);
cudaError_t launch_stash_bf16(const InstDev* d, int n, int64_t items, int seg, int parity,
                              int grid, int* err, int poll_lim, int withhold,
                             StepCount seed, bool var,
                             bool own_ghosts, cudaStream_t s);
cudaError_t launch_stash_mix(const InstDev* d, int n, int64_t items, int seg, int parity,
                             int grid, int* err, int poll_lim, int withhold,
                             StepCount seed, bool var,
                             bool own_ghosts, cudaStream_t s);
cudaError_t strip_fields_f32(const InstDev* d, int64_t items, int seg, int parity, int grid,
                            int* err, bool var, const FieldOut& out, cudaStream_t s);
cudaError_t strip_fields_f16(const InstDev* d, int64_t items, int seg, int parity, int grid,
                            int* err, bool var, const FieldOut& out, cudaStream_t s);
cudaError_t strip_fields_bf16(const InstDev* d, int64_t items, int seg, int parity, int grid,
                            int* err, bool var, const FieldOut& out, cudaStream_t s);
cudaError_t strip_fields_mix(const InstDev* d, int64_t items, int seg, int parity, int grid,
                            int* err, bool var, const FieldOut& out, cudaStream_t s);
int stash_occupancy_f32();
int stash_occupancy_f16();
int stash_occupancy_bf16();
int stash_occupancy_mix();

// One step of every instance in d_inst[0..n_inst): persistent grid of `grid`
// CTAs over total_tiles tiles; reads buf[parity], writes buf[parity ^ 1].
cudaError_t launch_step(int storage, int tile, const InstDev* d_inst, int n_inst,
                        int64_t total_tiles, int parity, int grid, StepCount seed,
                        cudaStream_t s);

// Resident CTAs per SM of the step kernel (0 if unavailable).
int step_occupancy(int storage, int tile);

// Fields c, p, ux, uy, T of one instance (d_one, tiles of shape 0, whose
// tile_begin must be 0) into out.
cudaError_t launch_fields(int storage, const InstDev* d_one, int64_t tiles, int parity,
                          const FieldOut& out, cudaStream_t s);

// Per-storage entry points (defined in lbe_step_<storage>.cu).
cudaError_t launch_step_f64(int tile, const InstDev* d, int n, int64_t total, int parity,
                            int grid, StepCount seed, cudaStream_t s);
cudaError_t launch_step_f32(int tile, const InstDev* d, int n, int64_t total, int parity,
                            int grid, StepCount seed, cudaStream_t s);
cudaError_t launch_step_f16(int tile, const InstDev* d, int n, int64_t total, int parity,
                            int grid, StepCount seed, cudaStream_t s);
cudaError_t launch_step_bf16(int tile, const InstDev* d, int n, int64_t total, int parity,
                             int grid, StepCount seed, cudaStream_t s);
cudaError_t launch_step_mix(int tile, const InstDev* d, int n, int64_t total, int parity,
                            int grid, StepCount seed, cudaStream_t s);
int occupancy_f64(int tile);
int occupancy_f32(int tile);
int occupancy_f16(int tile);
int occupancy_bf16(int tile);
int occupancy_mix(int tile);
cudaError_t fields_f64(const InstDev* d, int64_t tiles, int parity, const FieldOut& out,
                       cudaStream_t s);
// Varying density (FP64 storage only): the corrected p of Eq. 13 of every
// cell into each instance's pcorr (or drive); d is a work list of pre_shape.
cudaError_t pcorr_f64(const InstDev* d, int n, int64_t total, int parity, int grid,
                      cudaStream_t s);
// FP32 storage: the pre-pass of the dissipation term (u of every cell)
cudaError_t pcorr_f32(const InstDev* d, int n, int64_t total, int parity, int grid,
                      cudaStream_t s);
// The pass that collides, after a pre-pass into every instance's `drive`: `parts`
// (drive_parts per tile of the pre-pass) on `grid` CTAs.
cudaError_t drive_f64(const InstDev* d, int n, int64_t parts, int parity, int grid,
                      cudaStream_t s);
cudaError_t drive_f32(const InstDev* d, int n, int64_t parts, int parity, int grid,
                      cudaStream_t s);
cudaError_t fields_f32(const InstDev* d, int64_t tiles, int parity, const FieldOut& out,
                       cudaStream_t s);
cudaError_t fields_f16(const InstDev* d, int64_t tiles, int parity, const FieldOut& out,
                       cudaStream_t s);
cudaError_t fields_bf16(const InstDev* d, int64_t tiles, int parity, const FieldOut& out,
                       cudaStream_t s);
cudaError_t fields_mix(const InstDev* d, int64_t tiles, int parity, const FieldOut& out,
                       cudaStream_t s);

// Auxiliary kernels (lbe_aux.cu).
// The rest state of every cell from c0, T0 (device, [ny][nx]) into
// rest[3][ny][nx]: H_0, H_i (g_i = w_i H_i) and rho c_v T0 (hbar_i = w_i rho
// c_v T0); f = 0.
cudaError_t launch_rest_state(const InstDev* d_one, int nx, int ny, const double* c0,
                              const double* T0, double* rest, cudaStream_t s);
// pre[27][ny][nx] (double, pre-collision) -> buf[parity] (inverse of the
// pull); rest != 0: pre is rest[3][ny][nx] of launch_rest_state.
cudaError_t launch_push(int storage, const InstDev* d_one, int nx, int ny, const double* pre,
                        int parity, int rest, cudaStream_t s);
// buf[parity] -> pre[27][ny][nx] (the pull).
cudaError_t launch_pull(int storage, const InstDev* d_one, int nx, int ny, double* pre,
                        int parity, cudaStream_t s);
// FP64 sums over cur[5][n] and prev[5][n] (or prev = nullptr): out[6] =
// sum c, sum p, sum T, sum |u - u_prev|^2, sum |u|^2, non-finite count.
// partial must hold 6 * sums_blocks() doubles.
int sums_blocks();
cudaError_t launch_sums(const double* cur, const double* prev, int64_t n, double* partial,
                        double* out, cudaStream_t s);
// Periodic ghost columns of buffer `parity` of n_inst instances (16/32-bit
// storages), after a step of the stash kernel.
cudaError_t launch_ghosts(const InstDev* d, int n_inst, int max_ny, int parity, cudaStream_t s);
// The handle's step counter (16-bit storages): advanced after the steps that
// were launched with offsets to it, or set.
cudaError_t launch_seed_add(uint32_t* seed, uint32_t steps, cudaStream_t s);
cudaError_t launch_seed_set(uint32_t* seed, uint32_t value, cudaStream_t s);

// Adjoint kernels (lbe_adjoint.cu), one instance d_one of nx x ny.  fp32:
// states, adjoints and scratch are FP32 (a handle whose arithmetic is), else
// FP64; sizes in planes of nx * ny values of adjoint_real_bytes.
size_t adjoint_real_bytes(bool fp32);
int64_t adjoint_state_planes(bool fp32);  // a state: populations, FP32: and moments
int64_t adjoint_vector_planes();          // an adjoint: 27 planes, then 3 terms of the cell
int64_t adjoint_scratch_planes();
int64_t adjoint_part_doubles(int nx, int ny);  // partial sums of the tiles
// The state of buf[parity].
cudaError_t launch_adjoint_state(int storage, const InstDev* d_one, int nx, int ny, int parity,
                                 void* state, cudaStream_t s);
// c, p, T (cpt[3][N]) of 27 FP64 planes.
cudaError_t launch_adjoint_moments(const InstDev* d_one, int nx, int ny, const double* Q,
                                   double* cpt, cudaStream_t s);
// out4[0..1] = sum c u_y, sum c of a state.  fp32: Q is a state; else Q the 27
// planes and cpt their moments.
cudaError_t launch_observable(const InstDev* d_one, int nx, int ny, bool fp32, const void* Q,
                              const void* cpt, double* part, double* out4, cudaStream_t s);
// One adjoint step at the state (Q, cpt as above): aout (27 planes) and tout
// (3 planes) from a, at (the same of the next state; at may be NULL: zero, a
// NULL: a zero adjoint); part gains the theta sums of its tiles.
cudaError_t launch_adjoint_step(const InstDev* d_one, int nx, int ny, bool fp32, const void* Q,
                                const void* cpt, const void* a, const void* at, double wl,
                                const double* obs, void* aout, void* tout, void* scratch,
                                double* part, cudaStream_t s);
// out4[0..2] = the theta sums.
cudaError_t launch_adjoint_sums(const double* part, int nx, int ny, double* out4, cudaStream_t s);
// 27 FP64 planes, and dL/dT0, of an adjoint.
cudaError_t launch_adjoint_finish(int nx, int ny, bool fp32, const void* a, const void* at,
                                  double* out, cudaStream_t s);
cudaError_t launch_adjoint_dT0(const InstDev* d_one, int nx, int ny, bool fp32, const void* a,
                               const void* at, double* dT0, cudaStream_t s);

// Sets the message lbe_last_error(NULL) returns on this thread (lbe_api.cu).
void set_thread_error(const char* msg);

}  // namespace lbe
