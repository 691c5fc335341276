// Team step kernels of one (order, storage): a single step, several steps in a cooperative launch, and
// the batched step.
#include "rlb_inst_select.h"
#include "rlb_team.cuh"

namespace rlb {
using namespace inst;

namespace {
// Resident blocks per SM of a team kernel, asked for once per kernel.
template <class K>
int ask_resident(K kern) {
  int nb = 0;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, kern, kTeamWarps * 32, 0) != cudaSuccess) {
    cudaGetLastError();
    return 1;
  }
  return nb > 0 ? nb : 1;
}
template <bool W>
int resident_steps() {
  static const int nb = ask_resident(k_steps_team<L, S, W>);
  return nb;
}
template <bool W>
int resident_batch() {
  static const int nb = ask_resident(k_step_team_batch<L, S, W>);
  return nb;
}

template <bool W>
cudaError_t steps_w(void* a, void* b, StepParams p, int* status, int ntiles, int nsteps, int sms, unsigned* arrived,
                    cudaStream_t s) {
  if (nsteps == 1) {
    k_step_team<L, S, W><<<ntiles, kTeamWarps * 32, 0, s>>>((const T*)a, (T*)b, p, status);
    return cudaGetLastError();
  }
  auto kern = k_steps_team<L, S, W>;
  int grid = sms * resident_steps<W>();
  if (grid > ntiles) grid = ntiles;
  cudaError_t e = cudaMemsetAsync(arrived, 0, sizeof(unsigned), s);
  if (e != cudaSuccess) return e;
  T *ta = (T*)a, *tb = (T*)b;
  void* args[] = {&ta, &tb, &p, &status, &ntiles, &nsteps, &arrived};
  return cudaLaunchCooperativeKernel((const void*)kern, dim3(grid), dim3(kTeamWarps * 32), args, 0, s);
}
}  // namespace

cudaError_t RLB_TFN(steps)(void* a, void* b, const StepParams& p, int* status, int nsteps, int sms, unsigned* arrived,
                           cudaStream_t s) {
  const int ntiles = (p.cells + kTeamCells - 1) / kTeamCells;
  if (p.has_wall) return steps_w<true>(a, b, p, status, ntiles, nsteps, sms, arrived, s);
  return steps_w<false>(a, b, p, status, ntiles, nsteps, sms, arrived, s);
}

int RLB_TFN(resident)(int walls) {
  return walls ? resident_steps<true>() : resident_steps<false>();
}

cudaError_t RLB_TFN(batch)(const BatchMember* m, const int* tm, int ntiles, int launch, int walls, int sms,
                           cudaStream_t s) {
  auto kern = walls ? k_step_team_batch<L, S, true> : k_step_team_batch<L, S, false>;
  int grid = sms * (walls ? resident_batch<true>() : resident_batch<false>());
  if (grid > ntiles) grid = ntiles;
  kern<<<grid, kTeamWarps * 32, 0, s>>>(m, tm, ntiles, launch);
  return cudaGetLastError();
}
}  // namespace rlb
