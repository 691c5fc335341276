// Team step kernels: the four warps of a block share 32 cells, a quarter of the populations each.
//
// A tile is 32 consecutive cells of the lattice (rows may end inside it), one per lane; warp w of the
// block pulls slice w of their populations, once, into registers (32 floats or doubles at Q = 128),
// adds its partial moments, and collides and stores the same slice after the warps have added the
// partial sums through shared memory.  The pull takes each lane's source offsets from PullTab (one
// offset per axis and velocity component: any boundary, any axis length, rows of any alignment), or,
// where the whole warp is interior, the lattice's constant offsets.
//
// Against one cell per thread with all populations in registers (168 registers, 12 warps an SM) this
// holds a quarter of the state per thread, so more loads are in flight and each cell's serial work is
// a quarter as long: that is what bounds lattices too small to fill the chip, such as 1 x 1 x N tubes,
// and what the register kernels wait for on large ones.  Double storage, bound by the double pipe, has
// one warp solve the Landau frame and the equilibrium's coefficients for the tile (the pipe is shared
// by the SM, so solving it four times would take it from the other blocks); in float all four warps
// solve it, which saves a barrier.
//
// Several steps of a lattice whose tiles (nearly) all fit the chip at once run in one cooperative
// launch with a barrier over the grid after each step (k_steps_team): a small lattice's step is shorter
// than the gap between two launches.
#pragma once

#include "rlb_kernels.cuh"

namespace rlb {

constexpr unsigned long long kTeamWaitNs = 2000000000ull;  // 2 s

// The slice of the populations warp W of a team takes: float arithmetic a range of direction pairs,
// double arithmetic a level slice (Slices).  at(I): position of population I in the warp's registers.
template <class L>
struct TeamDirs {
  // first direction pair of warp w: the boundary nearest to w quarters of the populations
  __host__ __device__ static constexpr int begin(int w) {
    int k = 0, acc = 0;
    while (k < L::NDP && 4 * (acc + L::DP_NPAIR[k]) <= w * L::Q) acc += 2 * L::DP_NPAIR[k++];
    return k;
  }
  __host__ __device__ static constexpr int pop(int k) { return k < L::NDP ? L::DP_FIRST[k] : L::Q; }
  __host__ __device__ static constexpr int size(int w) { return pop(begin(w + 1)) - pop(begin(w)); }
  __host__ __device__ static constexpr int max_size() {
    int m = 0;
    for (int w = 0; w < kTeamWarps; ++w) m = size(w) > m ? size(w) : m;
    return m;
  }
};
template <class L>
__host__ __device__ constexpr int slice_pos(int pair) {  // position of a pair within its double slice
  int n = 0;
  for (int k = 0; k < pair; ++k) n += Slices<L>::slice_of(k) == Slices<L>::slice_of(pair);
  return n;
}

// What the collision of a cell needs once its frame is known, in shared memory: [value][lane].
template <class L, class A>
struct TeamFrame {
  static constexpr int kFloats = 4 * L::NLEV + 6;
};

template <class L, class S>
__host__ __device__ constexpr int team_smem_bytes() {
  using A = typename S::A;
  return (kTeamWarps * 13 + (sizeof(A) == 8 ? TeamFrame<L, A>::kFloats : 0)) * 32 * (int)sizeof(A);
}

template <class A>
__device__ __forceinline__ void put_partial(A* s, const Mom<A>& m) {
  s[0 * 32] = m.N0, s[1 * 32] = m.Nx, s[2 * 32] = m.Ny, s[3 * 32] = m.Nz, s[4 * 32] = m.T00, s[5 * 32] = m.T0x;
  s[6 * 32] = m.T0y, s[7 * 32] = m.T0z, s[8 * 32] = m.Txx, s[9 * 32] = m.Tyy, s[10 * 32] = m.Txy;
  s[11 * 32] = m.Txz, s[12 * 32] = m.Tyz;
}
template <class A>
__device__ __forceinline__ Mom<A> sum_partials(const A* s) {
  A v[13];
#pragma unroll
  for (int k = 0; k < 13; ++k) {
    v[k] = s[k * 32];
#pragma unroll
    for (int w = 1; w < kTeamWarps; ++w) v[k] = v[k] + s[(w * 13 + k) * 32];
  }
  return Mom<A>{v[0], v[1], v[2], v[3], v[4], v[5], v[6], v[7], v[8], v[9], A(0), v[10], v[11], v[12]};
}

// One tile's time step.  OFFS: p.off may be used for interior warps (p in constant memory).
template <class L, class S, bool WALLS, bool OFFS>
__device__ __forceinline__ void team_tile(const typename S::T* src, typename S::T* dst, const StepParams& p,
                                          int* status, int tile, unsigned char* smem) {
  using A = typename S::A;
  using T = typename S::T;
  constexpr bool DBL = std::is_same<A, double>::value;
  constexpr bool DEV = std::is_same<S, StoreF16Dev>::value;
  constexpr int NREG = DBL ? 2 * Slices<L>::PER : TeamDirs<L>::max_size();
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  A* const part = reinterpret_cast<A*>(smem);
  const int c = tile * kTeamCells + lane;
  const bool valid = c < p.cells;
  const Cell cl = make_cell(valid ? c : p.cells - 1, p);

  // population I's place in the registers of the warp that holds it
  auto at = [](auto I) {
    constexpr int i = decltype(I)::value;
    if constexpr (DBL) return ic<2 * slice_pos<L>(i / 2) + (i & 1)>{};
    else {
      constexpr int w = i >= TeamDirs<L>::pop(TeamDirs<L>::begin(3))   ? 3
                        : i >= TeamDirs<L>::pop(TeamDirs<L>::begin(2)) ? 2
                        : i >= TeamDirs<L>::pop(TeamDirs<L>::begin(1)) ? 1
                                                                       : 0;
      return ic<i - TeamDirs<L>::pop(TeamDirs<L>::begin(w))>{};
    }
  };
  // f(I) for every population of warp W's slice
  auto for_slice = [](auto W, auto&& fn) {
    constexpr int w = decltype(W)::value;
    if constexpr (DBL) {
      static_for<Slices<L>::count(w)>([&](auto J) {
        constexpr int i = Slices<L>::pair(w, -1, decltype(J)::value);
        fn(ic<i>{});
        fn(ic<i + 1>{});
      });
    } else {
      static_for<TeamDirs<L>::size(w)>(
          [&](auto J) { fn(ic<TeamDirs<L>::pop(TeamDirs<L>::begin(w)) + decltype(J)::value>{}); });
    }
  };
  auto each_warp = [&](auto&& fn) {
    if (warp == 0) fn(ic<0>{});
    else if (warp == 1) fn(ic<1>{});
    else if (warp == 2) fn(ic<2>{});
    else fn(ic<3>{});
  };

  A f[NREG];
  auto load = [&](const T* q) -> A {
    if constexpr (DEV) return __half2float(__ldcg(q));
    else return (A)__ldcg(q);
  };
  bool fast = false;
  if constexpr (OFFS)
    fast = __all_sync(0xffffffffu, (unsigned)(cl.x - p.ix0) < (unsigned)p.ixn && (unsigned)(cl.y - p.iy0) < (unsigned)p.iyn &&
                                       (unsigned)(cl.z - p.iz0) < (unsigned)p.izn);
  if (fast) {
    const T* base = src + cl.c;
    each_warp([&](auto W) {
      for_slice(W, [&](auto I) { f[at(I).value] = load(base + p.off[decltype(I)::value]); });
    });
  } else {
    PullTab<L> tab(cl, p);
    if constexpr (WALLS) tab.find_walls(cl, p);
    each_warp([&](auto W) {
      for_slice(W, [&](auto I) { f[at(I).value] = load(src + tab.template index<decltype(I)::value, WALLS>(cl, p)); });
    });
  }
  auto get = [&](auto I) -> A { return f[at(I).value]; };
  auto get2 = [&](auto I) -> float2 {
    constexpr int i = decltype(I)::value;
    return make_float2((float)get(ic<i>{}), (float)get(ic<i + 1>{}));
  };

  A* const mine = part + warp * 13 * 32 + lane;
  each_warp([&](auto W) {
    constexpr int w = decltype(W)::value;
    if constexpr (DBL) put_partial<A>(mine, moments_fixed_slice<L, w>(get));
    else put_partial<A>(mine, moments_f2_part<L, DEV, TeamDirs<L>::begin(w), TeamDirs<L>::begin(w + 1)>(get2));
  });
  __syncthreads();

  T* const out = dst + cl.c;
  auto store = [&](auto I, A v) {
    constexpr int i = decltype(I)::value;
    if (valid) {
      if constexpr (DEV) S::template store_dev<L, i>(out + (long long)i * p.cells, v, p);
      else S::template store<L, i>(out + (long long)i * p.cells, v, p);
    }
  };
  bool ok;
  if constexpr (DBL) {
    double* const fr = part + kTeamWarps * 13 * 32 + lane;
    if (warp == 0) {
      Mom<double> m = sum_partials<double>(part + lane);
      finish_fixed<L>(m);
      const Landau<double> lw = landau_step<double>(m, p);
      double inv_tau = 0.0;
      if (lw.ok) {
        const double Tl = lw.eps / (3.0 * lw.n);
        inv_tau = 1.0 / tau_prime<double>(Tl, p);
        const LevCoef<L, double> e = level_coef<L, double>(eq_coef<L::ORDER, double>(lw.n, Tl, lw.U0), 0.0);
#pragma unroll
        for (int l = 0; l < L::NLEV; ++l) {
          fr[(4 * l + 0) * 32] = e.a[l], fr[(4 * l + 1) * 32] = e.b[l];
          fr[(4 * l + 2) * 32] = e.c[l], fr[(4 * l + 3) * 32] = e.d[l];
        }
        fr[(4 * L::NLEV + 0) * 32] = lw.Ux, fr[(4 * L::NLEV + 1) * 32] = lw.Uy, fr[(4 * L::NLEV + 2) * 32] = lw.Uz;
        fr[(4 * L::NLEV + 3) * 32] = lw.U0 * inv_tau;
      } else if (valid) {
        atomicAdd(&status[kStatusNonconv], 1);
      }
      fr[(4 * L::NLEV + 4) * 32] = inv_tau;  // 0: no Landau frame
    }
    __syncthreads();
    const double inv_tau = fr[(4 * L::NLEV + 4) * 32];
    ok = inv_tau != 0.0;
    if (ok) {
      const double Ux = fr[(4 * L::NLEV + 0) * 32], Uy = fr[(4 * L::NLEV + 1) * 32], Uz = fr[(4 * L::NLEV + 2) * 32];
      const double a = fr[(4 * L::NLEV + 3) * 32];
      each_warp([&](auto W) {
        constexpr int w = decltype(W)::value;
        DirTerm<double> dt;
        static_for<Slices<L>::count(w)>([&](auto J) {
          constexpr int j = decltype(J)::value, i = Slices<L>::pair(w, -1, j), l = L::LEV[i];
          constexpr int b = j > 0 ? Slices<L>::pair(w, -1, j > 0 ? j - 1 : 0) : -1;
          if constexpr (b < 0 || L::VX[b < 0 ? 0 : b] != L::VX[i] || L::VY[b < 0 ? 0 : b] != L::VY[i] ||
                        L::VZ[b < 0 ? 0 : b] != L::VZ[i])
            dt = dir_term<L, double, i>(Ux, Uy, Uz, inv_tau, a);
          collide_pair<L, double, false, i>(dt, fr[(4 * l) * 32], fr[(4 * l + 1) * 32], fr[(4 * l + 2) * 32],
                                            fr[(4 * l + 3) * 32], get, store);
        });
      });
    }
  } else {
    const float c_dev = DEV ? p.half_nref : 0.f;
    Mom<float> m = sum_partials<float>(part + lane);
    finish_moments_f2<L, DEV>(m, c_dev);
    const Landau<float> lw = landau_step<float>(m, p);
    ok = lw.ok;
    if (ok) {
      const float Tl = lw.eps / (3.f * lw.n);
      const float inv_tau = 1.f / tau_prime<float>(Tl, p);
      const CollideCoef<L> q = collide_coef<L, DEV>(lw, Tl, inv_tau, c_dev);
      auto put2 = [&](auto I, float2 v) {
        constexpr int i = decltype(I)::value;
        store(ic<i>{}, v.x);
        store(ic<i + 1>{}, v.y);
      };
      each_warp([&](auto W) {
        constexpr int w = decltype(W)::value;
        collide_f2<L, DEV, TeamDirs<L>::begin(w), TeamDirs<L>::begin(w + 1)>(q, get2, put2);
      });
    } else if (valid && warp == 0) {
      atomicAdd(&status[kStatusNonconv], 1);
    }
  }
  // no Landau frame: the populations are streamed without collision
  if (!ok)
    each_warp([&](auto W) { for_slice(W, [&](auto I) { store(I, get(I)); }); });
}

// One time step, one tile per block.
template <class L, class S, bool WALLS>
__global__ void __launch_bounds__(kTeamWarps * 32, kTeamBlocks<typename S::A>)
    k_step_team(const typename S::T* __restrict__ src, typename S::T* __restrict__ dst,
                const __grid_constant__ StepParams p, int* __restrict__ status) {
  __shared__ __align__(16) unsigned char smem[team_smem_bytes<L, S>()];
  team_tile<L, S, WALLS, true>(src, dst, p, status, blockIdx.x, smem);
}

// nsteps time steps in one cooperative launch: block b takes tiles b, b + grid, ...; after each step
// every block adds 1 to *arrived (0 at launch) and waits until all `peers` of the grid have (at most
// kTeamWaitNs; a wait that runs out is counted and ends the block).  A step reads what other SMs wrote
// in the one before: the loads go to L2 (__ldcg).
template <class L, class S, bool WALLS>
__global__ void __launch_bounds__(kTeamWarps * 32, kTeamBlocks<typename S::A>)
    k_steps_team(typename S::T* a, typename S::T* b, const __grid_constant__ StepParams p, int* status, int ntiles,
                 int nsteps, unsigned* arrived, unsigned peers) {
  __shared__ __align__(16) unsigned char smem[team_smem_bytes<L, S>()];
  __shared__ int gone;
  for (int s = 0; s < nsteps; ++s) {
    for (int t = blockIdx.x; t < ntiles; t += gridDim.x) {
      if (t != (int)blockIdx.x) __syncthreads();  // the last tile's shared values are read
      team_tile<L, S, WALLS, true>(s & 1 ? b : a, s & 1 ? a : b, p, status, t, smem);
    }
    if (s + 1 == nsteps) return;
    __syncthreads();
    if (threadIdx.x == 0) {
      __threadfence();
      atomicAdd(arrived, 1u);
      const unsigned want = (unsigned)(s + 1) * peers;
      unsigned long long t0 = 0, now;
      gone = 0;
      for (;;) {
        unsigned v;
        asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(arrived) : "memory");
        if (v >= want) break;
        asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(now));
        if (t0 == 0) t0 = now;
        if (now - t0 > kTeamWaitNs) {
          atomicAdd(&status[kStatusTimeout], 1);
          gone = 1;
          break;
        }
      }
      __threadfence();
    }
    __syncthreads();
    if (gone) return;
  }
}

// One time step of every batch member with steps left: block b takes tiles b, b + grid, ... of the
// members' tiles (tile -> member table).
template <class L, class S, bool WALLS>
__global__ void __launch_bounds__(kTeamWarps * 32, kTeamBlocks<typename S::A>)
    k_step_team_batch(const BatchMember* __restrict__ members, const int* __restrict__ tile_member, int ntiles,
                      int launch) {
  using T = typename S::T;
  __shared__ __align__(16) unsigned char smem[team_smem_bytes<L, S>()];
  bool first = true;
  for (int t = blockIdx.x; t < ntiles; t += gridDim.x) {
    const BatchMember& m = members[__ldg(&tile_member[t])];
    if (launch >= m.steps_left) continue;
    if (!first) __syncthreads();  // the last tile's shared values are read
    first = false;
    const int par = (m.parity0 + launch) & 1;
    team_tile<L, S, WALLS, false>(static_cast<const T*>(m.buf[par]), static_cast<T*>(m.buf[par ^ 1]), m.p, m.status,
                                  t - m.team_tile_begin, smem);
  }
}

}  // namespace rlb
