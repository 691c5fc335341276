// Host-side launchers, one set per (order, storage) instantiation (rlb_inst.cu is compiled once
// per pair so that the translation units build in parallel).
#pragma once
#include <cuda_runtime.h>

#include "rlb_common.h"

namespace rlb {
struct StepParams;
struct PipeParams;
struct BatchMember;

struct Launchers {
  cudaError_t (*step)(const void* src, void* dst, const StepParams& p, int* status, bool general, int variant,
                      cudaStream_t s);
  // fields and partial sums of the lattice's kMomThreads-cell blocks [block0, block1)
  cudaError_t (*fields)(const void* src, const StepParams& p, const FieldOut& out, double* partial, int* status,
                        bool pull, int block0, int block1, cudaStream_t s);
  // initial populations of cells [c0, c1)
  cudaError_t (*init)(const double* n, const double* T, const double* u, void* dst, const StepParams& p, int* status,
                      int c0, int c1, cudaStream_t s);
  cudaError_t (*convert)(void* pop, double* dbl, int i0, int i1, bool to_f64, const StepParams& p, cudaStream_t s);
  int step_variants;  // number of step-kernel variants the autotuner may choose from
  // one time step of the persistent batched kernels: a launch over the row tiles [0, row_tiles) and
  // one over the shell tiles [row_tiles, row_tiles + shell_tiles) of the tile -> member table, with
  // counters[2 launch_index] and counters[2 launch_index + 1]; walls != 0 selects the kernels with
  // the bounce-back test (some member has walls)
  cudaError_t (*batch_step)(const BatchMember* members, const int* tile_member, int row_tiles, int shell_tiles,
                            int launch_index, int* counters, int variant, int walls, int grid, cudaStream_t s);
  // resident blocks per SM of the batched step for a variant
  int (*batch_blocks_per_sm)(int variant);
  // one time step of the pipelined kernel with tile width tx (64 or 128), row tiles if rows != 0
  // (tx 96, 128, 160, 192 or 256), float cells split between two warps if split != 0 (float storage)
  cudaError_t (*pipe_step)(const void* src, void* dst, const StepParams& p, const PipeParams& pp, int* status, int tx,
                           int rows, int split, int grid, int threads, int smem, cudaStream_t s);
  // nsteps time steps of the team kernel from buffer a into buffer b and back (one launch; more than
  // one step is a cooperative launch of at most `blocks` blocks, which wait for each other, counted in
  // *arrived)
  cudaError_t (*team_steps)(void* a, void* b, const StepParams& p, int* status, int nsteps, int blocks,
                            unsigned* arrived, cudaStream_t s);
  // blocks of that launch, and of the batched one, that an SM of the current device holds (0: not known)
  int (*team_resident)(int walls);
  int (*team_batch_resident)(int walls);
  // one time step (launch index `launch`) of the batch members' team tiles
  cudaError_t (*team_batch_step)(const BatchMember* members, const int* tile_member, int ntiles, int launch, int walls,
                                 int blocks, cudaStream_t s);
  // one time step of the batched pipelined kernel (launch index `launch`) over the members' tiles;
  // walls != 0 selects the kernel with the bounce-back patch
  cudaError_t (*pipe_batch_step)(const BatchMember* members, const int* tile_member, int launch, const PipeParams& pp,
                                 int* timeout, int tx, int rows, int split, int walls, int grid, int threads, int smem,
                                 cudaStream_t s);
};

// Block layout of pipelined variant v (>= kNumRegVariants) for q populations of `elem` bytes:
// stages (the largest multiple of the consumer-group count that fits the shared memory of one
// block, at least one per group and two in all), groups, threads and shared-memory bytes.  False if the variant
// does not exist for this storage.
struct PipeLayout {
  int tx, nstage, groups, producers, threads, smem, ctas_per_sm, rows, split;
};

// A lattice row of nx cells suits tiles of tx cells when its rows start on 16-byte boundaries and
// the tiles' lanes are at least `eighths` / 8 used.  Two warps per float cell want 7/8 (a 96-cell
// row in 128-cell tiles leaves 1/4 idle and ran slower than the register kernel); one warp per
// float cell 3/4 (200-cell rows in 128-cell tiles ran faster than the register kernel).
inline bool pipe_fits(int nx, int tx, int elem, int eighths = 7) {
  if (nx % (16 / elem) != 0) return false;
  const long long used = (long long)((nx + tx - 1) / tx) * tx;
  return 8LL * nx >= eighths * used;
}

// The fill rule of a layout: 3/4 for one warp per float cell, 7/8 otherwise.
inline int fill_eighths(const PipeLayout& lay, int elem) { return (elem == 4 && !lay.split) ? 6 : 7; }

// Row tiles of tx cells can take a lattice whose x axis is periodic and at least the stencil reach
// vmax_x long (one wrap per pull), with nx <= tx cells per row starting on 16-byte boundaries.
inline bool rows_possible(int nx, int tx, int elem, int bc_x, int vmax_x) {
  return bc_x == kPeriodic && nx <= tx && nx >= vmax_x && nx % (16 / elem) == 0;
}

// ... and suit it when the tile's G = tx / nx rows use at least 3/4 of its lanes (in a batched mix of
// 32- to 128-cell rows every such member stepped faster in row tiles than on the register kernels; a
// 96-cell row per 128-cell tile ran 1.07x faster).
inline bool rows_fit(int nx, int tx, int elem, int bc_x, int vmax_x) {
  return rows_possible(nx, tx, elem, bc_x, vmax_x) && 4 * (tx / nx) * nx >= 3 * tx;
}

// The register-kernel variant of a storage (RLB_F64, RLB_F32, RLB_F16DEV) for lattices that suit neither
// the pipelined kernel nor the team kernel.
inline int register_variant(int storage) { return storage == 1 ? 3 : (storage == 2 ? 2 : 0); }

// Lattices the team kernel is for: at most this many tiles per block that the device holds (float storages 4,
// 116,736 cells; double 1, 14,592).  Measured per step against the register kernels: 1 x 1 x 2613 float 6.7 us
// against 33, 32^3 float 17 against 25, 49 x 48 x 46 48.7 against 59, 48 x 49 x 49 half, open in x, 41.1 against
// 54.2 (only 50 x 50 x 46 half, second order, lost: 26.4 against 24.8), 151 x 93 x 70 512 against 409; 1 x 1 x 800
// double 28 us against 104, 96^3 4.9 ms against 2.3 (there the pipe is busy either way and the team's second and
// third pass through its code cost more).
inline bool small_for_team(long long cells, int elem, int blocks) {
  return (cells + kTeamCells - 1) / kTeamCells <= (elem == 8 ? 1LL : 4LL) * blocks;
}

// Tiles of one lattice: row tiles (groups of tx / nx rows) or tx-cell row segments.
inline long long pipe_tile_count(int nx, int ny, int nz, int tx, int rows) {
  if (rows) {
    const long long g = tx / nx;
    return ((long long)ny * nz + g - 1) / g;
  }
  return (long long)((nx + tx - 1) / tx) * ny * nz;
}

// Tile widths above 128 are built for the float storages, 256 only where two stages of it fit (half
// storage, and the second order's 66 float populations); of double storage's third order only the
// 64-cell tiles (a stage of 96 cells is 100 KB and the shape's four consumer groups want one each).
constexpr bool pipe_built(int tx, int q, int elem) {
  if (q * elem == 128 * 8) return tx == 64;
  return tx <= 128 || (elem < 8 && (tx < 256 || q * elem < 128 * 4));
}

inline bool pipe_layout(int v, int q, int elem, int smem_per_sm, int smem_optin, PipeLayout* out) {
  if (!is_pipe(v)) return false;
  const PipeConfig& cf = pipe_config(v);
  if (!pipe_built(cf.tx, q, elem)) return false;
  const int A = 16 / elem;
  const long long stage = (long long)q * (cf.tx + A) * elem;
  long long budget = smem_per_sm / cf.ctas_per_sm - 1024;
  if (budget > smem_optin) budget = smem_optin;
  const bool split = elem == 4 && cf.split;  // float storage: two consumer warps per cell
  const int wpt = cf.tx / 32 * (split ? 2 : 1);
  const int groups = cf.cons_warps / wpt;
  // The producers that the kernel's warps leave room for: twelve consumer warps leave four in a block of
  // 128 registers a thread.
  const int room = pipe_max_warps(elem, split) - cf.cons_warps;
  const int producers = cf.producers < room ? cf.producers : room;
  if (groups < 1 || cf.cons_warps % wpt != 0 || producers < 1 || producers > q) return false;
  if (producers > kPipeMaxProducerWarps || cf.cons_warps > kPipeMaxConsumerWarps) return false;
  const long long xchg = split ? (long long)cf.cons_warps / 2 * kPipeXchgBytesPerPair : 0;
  long long fit = (budget - kPipeHeaderBytes - xchg) / stage;
  if (fit > kPipeMaxStages) fit = kPipeMaxStages;
  const int nstage = (int)(fit / groups * groups);
  if (nstage < groups || nstage < 2) return false;
  if (out) *out = PipeLayout{cf.tx, nstage, groups, producers, (cf.cons_warps + producers) * 32,
                             (int)(kPipeHeaderBytes + nstage * stage + xchg), cf.ctas_per_sm, cf.rows, split};
  return true;
}

#define RLB_DECLARE_LAUNCHERS(ORDER, STORAGE) extern const Launchers launchers_o##ORDER##_s##STORAGE;
RLB_DECLARE_LAUNCHERS(3, 0)
RLB_DECLARE_LAUNCHERS(3, 1)
RLB_DECLARE_LAUNCHERS(3, 2)
RLB_DECLARE_LAUNCHERS(2, 0)
RLB_DECLARE_LAUNCHERS(2, 1)
RLB_DECLARE_LAUNCHERS(2, 2)
#undef RLB_DECLARE_LAUNCHERS

cudaError_t launch_reduce_partials(const double* partial, int nblocks, double* totals, cudaStream_t s);
}  // namespace rlb
