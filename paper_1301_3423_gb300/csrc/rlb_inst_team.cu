// Team step kernels of one (order, storage): a single step, several steps in a cooperative launch, and
// the batched step.
#include "rlb_inst_select.h"
#include "rlb_team.cuh"

namespace rlb {
using namespace inst;

namespace {
// Blocks of a kernel that an SM of the current device holds; 0 if that cannot be asked.
template <class K>
int ask_resident(K kern) {
  int nb = 0;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, kern, kTeamWarps * 32, 0) == cudaSuccess) return nb;
  cudaGetLastError();
  return 0;
}

template <bool W>
cudaError_t steps_w(void* a, void* b, StepParams p, int* status, int ntiles, int nsteps, int blocks, unsigned* arrived,
                    cudaStream_t s) {
  if (nsteps == 1) {
    k_step_team<L, S, W><<<ntiles, kTeamWarps * 32, 0, s>>>((const T*)a, (T*)b, p, status);
    return cudaGetLastError();
  }
  auto kern = k_steps_team<L, S, W>;
  cudaError_t e = cudaMemsetAsync(arrived, 0, sizeof(unsigned), s);
  if (e != cudaSuccess) return e;
  T *ta = (T*)a, *tb = (T*)b;
  const unsigned grid = blocks < ntiles ? blocks : ntiles;
  unsigned peers = p.debug & kDebugStallTeam ? grid + 1 : grid;
  void* args[] = {&ta, &tb, &p, &status, &ntiles, &nsteps, &arrived, &peers};
  return cudaLaunchCooperativeKernel((const void*)kern, dim3(grid), dim3(kTeamWarps * 32), args, 0, s);
}
}  // namespace

cudaError_t RLB_TFN(steps)(void* a, void* b, const StepParams& p, int* status, int nsteps, int blocks,
                           unsigned* arrived, cudaStream_t s) {
  const int ntiles = (p.cells + kTeamCells - 1) / kTeamCells;
  if (p.has_wall) return steps_w<true>(a, b, p, status, ntiles, nsteps, blocks, arrived, s);
  return steps_w<false>(a, b, p, status, ntiles, nsteps, blocks, arrived, s);
}

int RLB_TFN(resident)(int walls) {
  return walls ? ask_resident(k_steps_team<L, S, true>) : ask_resident(k_steps_team<L, S, false>);
}

int RLB_TFN(batch_resident)(int walls) {
  return walls ? ask_resident(k_step_team_batch<L, S, true>) : ask_resident(k_step_team_batch<L, S, false>);
}

cudaError_t RLB_TFN(batch)(const BatchMember* m, const int* tm, int ntiles, int launch, int walls, int blocks,
                           cudaStream_t s) {
  auto kern = walls ? k_step_team_batch<L, S, true> : k_step_team_batch<L, S, false>;
  kern<<<blocks > 0 && blocks < ntiles ? blocks : ntiles, kTeamWarps * 32, 0, s>>>(m, tm, ntiles, launch);
  return cudaGetLastError();
}
}  // namespace rlb
