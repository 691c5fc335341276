// Kernels of the relativistic lattice Boltzmann step (arXiv:1301.3423) for sm_103a.
//
// A step (Eq. (rlb:disc)) is a single fused pass per cell, by one thread per cell in the kernels here
// (rlb_pipe.cuh stages the pull in shared memory, rlb_team.cuh splits a cell between four warps):
//   pull    f~_i(x) = f_i(x - v_i)                     one read per population
//   moments N^mu, T^{mu nu} over mirror pairs         (Sec. II.D)
//   Landau  T^{ab} U_b = eps U^a, n = U.N, T = eps/(3n) (Eq. (eigenproblem))
//   tau'    from eta/s and T                           (Sec. II.D, Sec. III)
//   f^eq    E(p0, t), t = v.U/R, as a cubic in t per energy level (App. B, Eq. (eq:equi3rd) /
//           (eq:equi2nd) regrouped)
//   collide f_i - (U0 - t_i)/tau' (f_i - w_i E_i)      one write per population
// The cells of a step are split over two launches: rows whose y and z are interior (constant
// offsets, or x wrapped only, per 32-aligned warp segment) and the boundary rows (k_step_shell_rows;
// k_step_shell per cell for lattices shorter than the stencil reach).  Batched steps use the same
// split across many lattices (k_step_batch).
//
// The quadrature is a compile-time table (generated rlb_quadrature.h), so every per-population
// constant (velocity components, energy, weight, mirror partner) is an immediate.
#pragma once

#include <cuda_fp16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include <type_traits>
#include <utility>

#include "rlb_common.h"
#include "rlb_quadrature.h"

namespace rlb {

// ---------------------------------------------------------------------------------------------
// compile-time loop
// ---------------------------------------------------------------------------------------------
template <int... Is, class F>
__device__ __forceinline__ void sfor_impl(std::integer_sequence<int, Is...>, F& f) {
  (f(std::integral_constant<int, Is>{}), ...);
}
template <int N, class F>
__device__ __forceinline__ void static_for(F&& f) {
  sfor_impl(std::make_integer_sequence<int, N>{}, f);
}
template <int I>
using ic = std::integral_constant<int, I>;

// ---------------------------------------------------------------------------------------------
// storage formats
// ---------------------------------------------------------------------------------------------
struct StoreF64 {
  using T = double;
  using A = double;                 // arithmetic of the step
  static constexpr bool kKeep = false;  // 128 doubles do not fit the register file: reload
  template <class L, int I>
  __device__ static __forceinline__ A load(const T* p, const StepParams&) { return __ldg(p); }
  template <class L, int I>
  __device__ static __forceinline__ void store(T* p, A v, const StepParams&) { *p = v; }
  template <class L, int I>
  __device__ static __forceinline__ double to_f64(T v, const StepParams&) { return v; }
  template <class L, int I>
  __device__ static __forceinline__ T from_f64(double v, const StepParams&) { return v; }
};

struct StoreF32 {
  using T = float;
  using A = float;
  static constexpr bool kKeep = true;   // all populations of a cell live in registers
  // Each population is read once per step: cached in L2 only, leaving L1 to the register spills
  // (measured 4.7 % faster at 256^3 than loads that also allocate in L1).
  template <class L, int I>
  __device__ static __forceinline__ A load(const T* p, const StepParams&) { return __ldcg(p); }
  template <class L, int I>
  __device__ static __forceinline__ void store(T* p, A v, const StepParams&) { *p = v; }
  template <class L, int I>
  __device__ static __forceinline__ double to_f64(T v, const StepParams&) { return (double)v; }
  template <class L, int I>
  __device__ static __forceinline__ T from_f64(double v, const StepParams&) { return (float)v; }
};

// Half-precision deviation d_i = f_i / w_i - n_ref / 2 from the weight-scaled rest equilibrium.
struct StoreF16Dev {
  using T = __half;
  using A = float;
  static constexpr bool kKeep = true;
  template <class L, int I>
  __device__ static __forceinline__ A load(const T* p, const StepParams& sp) {
    constexpr float w = (float)L::W[I];
    return w * (__half2float(__ldg(p)) + sp.half_nref);
  }
  template <class L, int I>
  __device__ static __forceinline__ void store(T* p, A v, const StepParams& sp) {
    constexpr float iw = (float)(1.0 / L::W[I]);
    *p = __float2half_rn(fmaf(v, iw, -sp.half_nref));
  }
  // the deviation d_i itself (the step kernels work in deviation space)
  template <class L, int I>
  __device__ static __forceinline__ A load_dev(const T* p, const StepParams&) { return __half2float(__ldg(p)); }
  template <class L, int I>
  __device__ static __forceinline__ void store_dev(T* p, A d, const StepParams&) { *p = __float2half_rn(d); }
  template <class L, int I>
  __device__ static __forceinline__ double to_f64(T v, const StepParams& sp) {
    constexpr double w = L::W[I];
    return w * ((double)__half2float(v) + (double)sp.half_nref);
  }
  template <class L, int I>
  __device__ static __forceinline__ T from_f64(double v, const StepParams& sp) {
    constexpr double iw = 1.0 / L::W[I];
    return __float2half_rn((float)(v * iw - (double)sp.half_nref));
  }
};

// ---------------------------------------------------------------------------------------------
// cell geometry and the pull source index
// ---------------------------------------------------------------------------------------------
struct Cell {
  int c, x, y, z;
};

__device__ __forceinline__ Cell make_cell(int c, const StepParams& p) {
  Cell r;
  r.c = c;
  const int yz = c / p.nx;
  r.x = c - yz * p.nx;
  r.z = yz / p.ny;
  r.y = yz - r.z * p.ny;
  return r;
}

// Source coordinate of x - v along an axis of n cells: periodic wrap or copy-out clamp.
// GENERAL handles n < |v| (a full modulo); otherwise one conditional wrap suffices.
template <int V, bool GENERAL>
__device__ __forceinline__ int src_coord(int x, int n, int bc) {
  if constexpr (V == 0) {
    return x;
  } else {
    int s = x - V;
    if (bc) return (V > 0) ? max(s, 0) : min(s, n - 1);
    if constexpr (GENERAL) {
      s %= n;
      return s < 0 ? s + n : s;
    } else {
      if constexpr (V > 0) return s < 0 ? s + n : s;
      else return s >= n ? s - n : s;
    }
  }
}

// src_coord with the shift v known only at run time (one conditional wrap: n >= |v|).
__device__ __forceinline__ int src_coord_rt(int x, int v, int n, int bc) {
  const int s = x - v;
  if ((unsigned)s < (unsigned)n) return s;
  if (bc) return s < 0 ? 0 : n - 1;
  return s < 0 ? s + n : s - n;
}

// The populations' velocities as a table in constant memory, for loops over the populations with
// a run-time index.
template <class L>
struct VelTab {
  signed char v[L::Q][3];
};
template <class L>
constexpr VelTab<L> make_vel_tab() {
  VelTab<L> t{};
  for (int i = 0; i < L::Q; ++i) {
    t.v[i][0] = (signed char)L::VX[i];
    t.v[i][1] = (signed char)L::VY[i];
    t.v[i][2] = (signed char)L::VZ[i];
  }
  return t;
}
template <class L>
__constant__ VelTab<L> kVelTab = make_vel_tab<L>();

// Pull offsets of one shell row (fixed y, z): for every population the constant offset plus the
// row's y and z wrap (or clamp) shifts, worked out once per row by the warp's 32 lanes (four
// populations each) into roff[Q]; the warp's cells then add only their x shift.  A population that
// comes from beyond a wall in y or z does so in the whole row: its offset is that of the cell's own
// reversed population (I ^ 1: mirror pairs are adjacent), to which no x shift is added; bit i % 32 of
// walled[i / 32] marks it.  (151 x 93 x 70 float lattice with walls on y, 28 % shell rows: with the wall
// test per cell and population instead the shell kernel took 178 us beside the interior's 204.)
template <class L, bool WALLS>
__device__ __forceinline__ void shell_row_table(long long* roff, uint32_t (&walled)[4], const Cell& cl,
                                                const StepParams& p) {
  static_assert(L::Q <= 128, "four words of flags");
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    const int i = (threadIdx.x & 31) + 32 * k;
    bool beyond = false;
    if (i < L::Q) {
      const int vy = kVelTab<L>.v[i][1], vz = kVelTab<L>.v[i][2];
      long long o = p.off[i];
      o += (long long)(src_coord_rt(cl.y, vy, p.ny, p.bc[1]) - (cl.y - vy)) * p.nx;
      o += (long long)(src_coord_rt(cl.z, vz, p.nz, p.bc[2]) - (cl.z - vz)) * p.nxy;
      if constexpr (WALLS) {
        beyond = (p.bc[1] == kBounceBack && (unsigned)(cl.y - vy) >= (unsigned)p.ny) ||
                 (p.bc[2] == kBounceBack && (unsigned)(cl.z - vz) >= (unsigned)p.nz);
        if (beyond) o = (long long)(i ^ 1) * p.cells;
      }
      roff[i] = o;
    }
    walled[k] = WALLS ? __ballot_sync(0xffffffffu, beyond) : 0u;
  }
  __syncwarp();
}

// True if the pull source of population I lies beyond a bounce-back wall (then the cell takes its
// own population of the reversed momentum, I ^ 1: mirror pairs are adjacent).
template <class L, int I>
__device__ __forceinline__ bool beyond_wall(const Cell& cl, const StepParams& p) {
  constexpr int vx = L::VX[I], vy = L::VY[I], vz = L::VZ[I];
  bool b = false;
  if constexpr (vx != 0) b = b || (p.bc[0] == kBounceBack && (unsigned)(cl.x - vx) >= (unsigned)p.nx);
  if constexpr (vy != 0) b = b || (p.bc[1] == kBounceBack && (unsigned)(cl.y - vy) >= (unsigned)p.ny);
  if constexpr (vz != 0) b = b || (p.bc[2] == kBounceBack && (unsigned)(cl.z - vz) >= (unsigned)p.nz);
  return b;
}

// WALLS = false compiles the bounce-back test out: kernels for lattices without walls pay nothing.
template <class L, int I, bool GENERAL, bool WALLS>
__device__ __forceinline__ long long pull_index(const Cell& cl, const StepParams& p) {
  constexpr int vx = L::VX[I], vy = L::VY[I], vz = L::VZ[I];
  if constexpr (WALLS) {
    if (p.has_wall && beyond_wall<L, I>(cl, p)) return (long long)(I ^ 1) * p.cells + cl.c;
  }
  const int sx = src_coord<vx, GENERAL>(cl.x, p.nx, p.bc[0]);
  const int sy = src_coord<vy, GENERAL>(cl.y, p.ny, p.bc[1]);
  const int sz = src_coord<vz, GENERAL>(cl.z, p.nz, p.bc[2]);
  return (long long)I * p.cells + (long long)(sz * p.nxy + sy * p.nx + sx);
}


// The in-plane index every pull of one cell needs, as one source offset per axis and velocity
// component (at most 13 values an axis): a population's source is x[vx] + y[vy] + z[vz], two adds,
// whatever the boundary.  Worked out once per cell (wrap, modulo wrap of an axis shorter than the
// reach, or clamp), where pull_index tests and wraps three coordinates for each of the Q
// populations: on a 1 x 1 x N tube, whose x and y take the modulo, that was most of a step.
template <class L>
struct PullTab {
  int x[2 * L::VMAX_X + 1], y[2 * L::VMAX_Y + 1], z[2 * L::VMAX_Z + 1];

  static __device__ __forceinline__ int wrap(int s, int n, int bc) {
    if ((unsigned)s < (unsigned)n) return s;
    if (bc) return s < 0 ? 0 : n - 1;
    s += s < 0 ? n : -n;
    if ((unsigned)s < (unsigned)n) return s;
    s %= n;
    return s < 0 ? s + n : s;
  }
  __device__ __forceinline__ PullTab(const Cell& cl, const StepParams& p) {
#pragma unroll
    for (int j = 0; j <= 2 * L::VMAX_X; ++j) x[j] = wrap(cl.x - (j - L::VMAX_X), p.nx, p.bc[0]);
#pragma unroll
    for (int j = 0; j <= 2 * L::VMAX_Y; ++j) y[j] = wrap(cl.y - (j - L::VMAX_Y), p.ny, p.bc[1]) * p.nx;
#pragma unroll
    for (int j = 0; j <= 2 * L::VMAX_Z; ++j) z[j] = wrap(cl.z - (j - L::VMAX_Z), p.nz, p.bc[2]) * p.nxy;
  }
  // The velocity components that point beyond a wall of each axis, as bits (none on lattices without).
  unsigned wx = 0, wy = 0, wz = 0;
  __device__ __forceinline__ void find_walls(const Cell& cl, const StepParams& p) {
    auto bits = [](int s, int n, int vmax) {  // components v with s - v outside 0 .. n - 1: bit v + vmax
      const int lo = max(s + 1, -vmax), hi = min(s - n, vmax);
      unsigned m = 0;
      if (lo <= vmax) m |= ~0u << (lo + vmax) & ((2u << (2 * vmax)) - 1u);
      if (hi >= -vmax) m |= (2u << (hi + vmax)) - 1u;
      return m;
    };
    if (p.bc[0] == kBounceBack) wx = bits(cl.x, p.nx, L::VMAX_X);
    if (p.bc[1] == kBounceBack) wy = bits(cl.y, p.ny, L::VMAX_Y);
    if (p.bc[2] == kBounceBack) wz = bits(cl.z, p.nz, L::VMAX_Z);
  }
  // index into the population buffer: plane offset of I plus the in-plane index; with WALLS the cell's
  // own value of the mirror partner where I points beyond a wall
  template <int I, bool WALLS>
  __device__ __forceinline__ long long index(const Cell& cl, const StepParams& p) const {
    constexpr int vx = L::VX[I], vy = L::VY[I], vz = L::VZ[I];
    if constexpr (WALLS) {
      unsigned b = 0;
      if constexpr (vx != 0) b |= wx & (1u << (vx + L::VMAX_X));
      if constexpr (vy != 0) b |= wy & (1u << (vy + L::VMAX_Y));
      if constexpr (vz != 0) b |= wz & (1u << (vz + L::VMAX_Z));
      if (b) return (long long)(I ^ 1) * p.cells + cl.c;
    }
    return (long long)I * p.cells + (unsigned)(x[vx + L::VMAX_X] + y[vy + L::VMAX_Y] + z[vz + L::VMAX_Z]);
  }
};

// Pull offset of population I from the cell's own index when only the x coordinate can leave the
// lattice (rows whose y and z are interior): the constant offset with x wrapped or clamped, or the
// cell's own reversed population beyond a bounce-back wall in x.
template <class L, int I, bool WALLS>
__device__ __forceinline__ long long x_row_offset(const Cell& cl, const StepParams& p) {
  constexpr int vx = L::VX[I];
  if constexpr (WALLS && vx != 0) {
    if (p.bc[0] == kBounceBack && (unsigned)(cl.x - vx) >= (unsigned)p.nx) return (long long)(I ^ 1) * p.cells;
  }
  return p.off[I] + (src_coord<vx, false>(cl.x, p.nx, p.bc[0]) - (cl.x - vx));
}

// ---------------------------------------------------------------------------------------------
// moments N^mu, T^{mu nu} (Eqs. (moments:dis1), (moments:dis2)), accumulated over mirror pairs:
// for a pair (v, -v) at energy p0, s1 = p0 (f+ +- f-), s2 = p0^2 (f+ +- f-).
// ---------------------------------------------------------------------------------------------
template <class A>
struct Mom {
  A N0, Nx, Ny, Nz, T00, T0x, T0y, T0z, Txx, Tyy, Tzz, Txy, Txz, Tyz;
};

// Moments of the weights alone, sum_i w_i k_i for the moment kernels k_i of N^0, T^00 and T^ab:
// in deviation space (f_i = w_i (d_i + c)) the constant c contributes c times these.  The odd
// moments cancel exactly between mirror partners.
template <class L>
struct RestSums {
  static constexpr double sum(int e, int a, int b) {  // sum_i w_i p0^e (v_a v_b / R^2 if a >= 0)
    double s = 0.0;
    for (int i = 0; i < L::Q; ++i) {
      const double p = L::P0[L::LEV[i]];
      const double v[3] = {(double)L::VX[i], (double)L::VY[i], (double)L::VZ[i]};
      double t = L::W[i] * (e == 1 ? p : p * p);
      if (a >= 0) t *= v[a] * v[b] * L::INV_R2;
      s += t;
    }
    return s;
  }
  static constexpr double N0 = sum(1, -1, -1), T00 = sum(2, -1, -1), Txx = sum(2, 0, 0), Tyy = sum(2, 1, 1),
                          Txy = sum(2, 0, 1), Txz = sum(2, 0, 2), Tyz = sum(2, 1, 2);
};

template <class L, class A>
__device__ __forceinline__ void add_rest_sums(Mom<A>& m, A c) {
  m.N0 = fma(A(RestSums<L>::N0), c, m.N0);
  m.T00 = fma(A(RestSums<L>::T00), c, m.T00);
  m.Txx = fma(A(RestSums<L>::Txx), c, m.Txx);
  m.Tyy = fma(A(RestSums<L>::Tyy), c, m.Tyy);
  m.Txy = fma(A(RestSums<L>::Txy), c, m.Txy);
  m.Txz = fma(A(RestSums<L>::Txz), c, m.Txz);
  m.Tyz = fma(A(RestSums<L>::Tyz), c, m.Tyz);
}

// DEV = true: get returns deviations d_i = f_i / w_i - c, and the moments are those of
// f_i = w_i (d_i + c).
template <class L, class A, bool DEV = false, class Get>
__device__ __forceinline__ Mom<A> moments(Get&& get, A c = A(0)) {
  Mom<A> m;
  m.N0 = m.Nx = m.Ny = m.Nz = A(0);
  m.T00 = m.T0x = m.T0y = m.T0z = A(0);
  m.Txx = m.Tyy = m.Txy = m.Txz = m.Tyz = A(0);
  static_for<L::NDP>([&](auto K) {
    constexpr int k = decltype(K)::value;
    constexpr int first = L::DP_FIRST[k];
    constexpr int np = L::DP_NPAIR[k];
    A s1p = A(0), s1m = A(0), s2p = A(0), s2m = A(0);
    static_for<np>([&](auto J) {
      constexpr int ip = first + 2 * decltype(J)::value;
      constexpr double wk = DEV ? L::W[ip] : 1.0;  // mirror partners share the weight
      constexpr double p0 = L::P0[L::LEV[ip]];
      const A fa = get(ic<ip>{});
      const A fb = get(ic<ip + 1>{});
      const A sp = fa + fb, sm = fa - fb;
      s1p = fma(A(wk * p0), sp, s1p);
      s1m = fma(A(wk * p0), sm, s1m);
      s2p = fma(A(wk * p0 * p0), sp, s2p);
      s2m = fma(A(wk * p0 * p0), sm, s2m);
    });
    constexpr int vx = L::VX[first], vy = L::VY[first], vz = L::VZ[first];
    constexpr double ir = L::INV_R, ir2 = L::INV_R2;
    m.N0 += s1p;
    m.T00 += s2p;
    if constexpr (vx != 0) {
      m.Nx = fma(A(vx * ir), s1m, m.Nx);
      m.T0x = fma(A(vx * ir), s2m, m.T0x);
      m.Txx = fma(A(vx * vx * ir2), s2p, m.Txx);
    }
    if constexpr (vy != 0) {
      m.Ny = fma(A(vy * ir), s1m, m.Ny);
      m.T0y = fma(A(vy * ir), s2m, m.T0y);
      m.Tyy = fma(A(vy * vy * ir2), s2p, m.Tyy);
    }
    if constexpr (vz != 0) {
      m.Nz = fma(A(vz * ir), s1m, m.Nz);
      m.T0z = fma(A(vz * ir), s2m, m.T0z);
    }
    if constexpr (vx != 0 && vy != 0) m.Txy = fma(A(vx * vy * ir2), s2p, m.Txy);
    if constexpr (vx != 0 && vz != 0) m.Txz = fma(A(vx * vz * ir2), s2p, m.Txz);
    if constexpr (vy != 0 && vz != 0) m.Tyz = fma(A(vy * vz * ir2), s2p, m.Tyz);
  });
  if constexpr (DEV) add_rest_sums<L, A>(m, c);
  // |v|^2 = R^2 for every velocity, so the spatial trace of T equals T^00.
  m.Tzz = m.T00 - m.Txx - m.Tyy;
  return m;
}

// Double arithmetic handles the mirror pairs in four slices: pairs in order of their energy level, a
// quarter each.  A slice's integer sums (below) have their own grid per level, so the slices define
// the rounding, and every double kernel, whether one thread or four share a cell, adds the same four.
template <class L>
struct Slices {
  static constexpr int N = 4, PAIRS = L::Q / 2, PER = (PAIRS + N - 1) / N;
  __host__ __device__ static constexpr int slice_of(int pair) {
    int r = 0;  // the pair's rank by (level, index)
    for (int k = 0; k < PAIRS; ++k)
      r += L::LEV[2 * k] < L::LEV[2 * pair] || (L::LEV[2 * k] == L::LEV[2 * pair] && k < pair);
    return r / PER;
  }
  // pairs of slice s (of level l if l >= 0), and the + population of the j-th of them
  __host__ __device__ static constexpr int count(int s, int l = -1) {
    int n = 0;
    for (int k = 0; k < PAIRS; ++k) n += slice_of(k) == s && (l < 0 || L::LEV[2 * k] == l);
    return n;
  }
  __host__ __device__ static constexpr int pair(int s, int l, int j) {
    for (int k = 0; k < PAIRS; ++k)
      if (slice_of(k) == s && (l < 0 || L::LEV[2 * k] == l) && j-- == 0) return 2 * k;
    return -1;
  }
  // the largest sum of |weights| (1, v_a, v_a v_b) over the populations of slice s and level l
  __host__ __device__ static constexpr int weight(int s, int l) {
    int most = 2 * count(s, l);
    for (int a = 0; a < 3; ++a)
      for (int b = 0; b <= 3; ++b) {
        int r = 0;
        for (int k = 0; k < PAIRS; ++k) {
          const int v[4] = {L::VX[2 * k], L::VY[2 * k], L::VZ[2 * k], 1}, w = v[a] * v[b];
          if (slice_of(k) == s && L::LEV[2 * k] == l) r += 2 * (w < 0 ? -w : w);
        }
        most = r > most ? r : most;
      }
    return most;
  }
  // bits a population may have so that every sum stays below 2^63
  __host__ __device__ static constexpr int bits(int s, int l) {
    int n = 63;
    for (int w = weight(s, l); w > 1; w = (w + 1) / 2) --n;
    return n;
  }
};

// Moments of double populations, summed in 64-bit integers.  GB300's double pipe takes 19 clocks an
// SM for a warp instruction (measured; 64 for a lone warp) and bounds the double step; its integer
// pipe is some 40 times wider.  Per slice and energy level the populations are converted to integers of
// a common grid, 2^-53 to 2^-58 of the power of two above the largest of them, as fine as 63-bit sums allow
// (Slices::bits): the scale goes into the exponent as an integer and the conversion takes 16 clocks.  The
// sums over v with the integer weights 1, v_a, v_a v_b are exact; 9 of them return to double and take p0
// and p0^2.  The grid is per level, so the rare high levels, which p0^2 weights most, are rounded by
// their own size.  The moments' error is below that of adding the 128 terms in double up to a Lorentz
// factor of 4 (third order, r.m.s. of T^00: 4.4e-17 against 8.0e-17 at rest, 7.2e-17 against 1.4e-16 at
// 2).  A grid of 2^-51 from adding 1.5 2^k was two to three times worse from 1.5 on and saved 1 % (96^3,
// ten steps: 25.4 ms against 25.7).
// Double-pipe instructions a cell: 128 conversions there, 63 back, 140 more; 960 when the sums were double.
// Populations that are not finite (or beyond 2^1021, whose moments overflow) give NaN moments.
// Slice SL's part, before the factors 1 / R and 1 / R^2 (finish_fixed).
template <class L, int SL, class Get>
__device__ __forceinline__ Mom<double> moments_fixed_slice(Get&& get) {
  using u64 = unsigned long long;
  using G = Slices<L>;
  Mom<double> m;
  m.N0 = m.Nx = m.Ny = m.Nz = 0.0;
  m.T00 = m.T0x = m.T0y = m.T0z = 0.0;
  m.Txx = m.Tyy = m.Tzz = m.Txy = m.Txz = m.Tyz = 0.0;
  bool finite = true;
  static_for<L::NLEV>([&](auto K) {
    constexpr int l = decltype(K)::value;
    constexpr int n = G::count(SL, l);
    if constexpr (n > 0) {
      constexpr int BITS = G::bits(SL, l);
      static_assert(BITS >= 53 && BITS <= 62, "every double below 2^BITS rounds to an integer below it");
      double f[2 * n];
      unsigned top = 0;
      static_for<n>([&](auto J) {
        constexpr int j = decltype(J)::value, i = G::pair(SL, l, j);
        f[2 * j] = get(ic<i>{});
        f[2 * j + 1] = get(ic<i + 1>{});
        top = max(top, max((unsigned)__double2hiint(f[2 * j]) & 0x7fffffffu,
                           (unsigned)__double2hiint(f[2 * j + 1]) & 0x7fffffffu));
      });
      const int e = max((int)(top >> 20), 64);  // |f| < 2^(e - 1022)
      finite = finite && e < 2045;
      // f 2^(BITS + 1022 - e) as an integer below 2^BITS.  Where the scaled exponent would be negative or
      // 0, the number is less than 1/2 (and stays so when 0 or a subnormal gets an exponent).
      const int shift = (BITS + 1022 - e) * (1 << 20);
      auto grid = [&](double x) -> u64 {
        const int h = __double2hiint(x), t = max((h & 0x7fffffff) + shift, 0);
        return (u64)__double2ll_rn(__hiloint2double(t | (h & (int)0x80000000u), __double2loint(x)));
      };
      u64 s0 = 0, sxx = 0, syy = 0, sxy = 0, sxz = 0, syz = 0, sx = 0, sy = 0, sz = 0;
      static_for<n>([&](auto J) {
        constexpr int j = decltype(J)::value, i = G::pair(SL, l, j);
        constexpr int vx = L::VX[i], vy = L::VY[i], vz = L::VZ[i];
        const u64 a = grid(f[2 * j]), b = grid(f[2 * j + 1]);
        const u64 sp = a + b, sm = a - b;
        s0 += sp;
        if constexpr (vx != 0) sxx += (u64)(long long)(vx * vx) * sp, sx += (u64)(long long)vx * sm;
        if constexpr (vy != 0) syy += (u64)(long long)(vy * vy) * sp, sy += (u64)(long long)vy * sm;
        if constexpr (vz != 0) sz += (u64)(long long)vz * sm;
        if constexpr (vx * vy != 0) sxy += (u64)(long long)(vx * vy) * sp;
        if constexpr (vx * vz != 0) sxz += (u64)(long long)(vx * vz) * sp;
        if constexpr (vy * vz != 0) syz += (u64)(long long)(vy * vz) * sp;
      });
      auto dbl = [](u64 s) { return (double)(long long)s; };
      const double g = __hiloint2double((e + 1 - BITS) << 20, 0);  // the grid, 2^(e - 1022 - BITS)
      const double p1 = L::P0[l] * g, p2 = L::P0[l] * L::P0[l] * g;
      const double d0 = dbl(s0), dx = dbl(sx), dy = dbl(sy), dz = dbl(sz);
      m.N0 = fma(p1, d0, m.N0);
      m.Nx = fma(p1, dx, m.Nx);
      m.Ny = fma(p1, dy, m.Ny);
      m.Nz = fma(p1, dz, m.Nz);
      m.T00 = fma(p2, d0, m.T00);
      m.T0x = fma(p2, dx, m.T0x);
      m.T0y = fma(p2, dy, m.T0y);
      m.T0z = fma(p2, dz, m.T0z);
      m.Txx = fma(p2, dbl(sxx), m.Txx);
      m.Tyy = fma(p2, dbl(syy), m.Tyy);
      m.Txy = fma(p2, dbl(sxy), m.Txy);
      m.Txz = fma(p2, dbl(sxz), m.Txz);
      m.Tyz = fma(p2, dbl(syz), m.Tyz);
    }
  });
  if (!finite) m.N0 = m.T00 = __longlong_as_double(0x7ff8000000000000ll);
  return m;
}
__device__ __forceinline__ void add_moments(Mom<double>& m, const Mom<double>& a) {
  m.N0 = __dadd_rn(m.N0, a.N0), m.Nx = __dadd_rn(m.Nx, a.Nx), m.Ny = __dadd_rn(m.Ny, a.Ny);
  m.Nz = __dadd_rn(m.Nz, a.Nz), m.T00 = __dadd_rn(m.T00, a.T00), m.T0x = __dadd_rn(m.T0x, a.T0x);
  m.T0y = __dadd_rn(m.T0y, a.T0y), m.T0z = __dadd_rn(m.T0z, a.T0z), m.Txx = __dadd_rn(m.Txx, a.Txx);
  m.Tyy = __dadd_rn(m.Tyy, a.Tyy), m.Txy = __dadd_rn(m.Txy, a.Txy), m.Txz = __dadd_rn(m.Txz, a.Txz);
  m.Tyz = __dadd_rn(m.Tyz, a.Tyz);
}
template <class L>
__device__ __forceinline__ void finish_fixed(Mom<double>& m) {
  m.Nx *= L::INV_R, m.Ny *= L::INV_R, m.Nz *= L::INV_R;
  m.T0x *= L::INV_R, m.T0y *= L::INV_R, m.T0z *= L::INV_R;
  m.Txx = __dmul_rn(m.Txx, L::INV_R2), m.Tyy = __dmul_rn(m.Tyy, L::INV_R2);
  m.Txy *= L::INV_R2, m.Txz *= L::INV_R2, m.Tyz *= L::INV_R2;
  // |v|^2 = R^2 for every velocity, so the spatial trace of T equals T^00.
  m.Tzz = m.T00 - m.Txx - m.Tyy;
}
template <class L, class Get>
__device__ __forceinline__ Mom<double> moments_fixed(Get&& get) {
  Mom<double> m = moments_fixed_slice<L, 0>(get);
  static_for<Slices<L>::N - 1>([&](auto K) { add_moments(m, moments_fixed_slice<L, decltype(K)::value + 1>(get)); });
  finish_fixed<L>(m);
  return m;
}

template <class A, class B>
__device__ __forceinline__ Mom<B> convert(const Mom<A>& a) {
  return Mom<B>{B(a.N0),  B(a.Nx),  B(a.Ny),  B(a.Nz),  B(a.T00), B(a.T0x), B(a.T0y),
                B(a.T0z), B(a.Txx), B(a.Tyy), B(a.Tzz), B(a.Txy), B(a.Txz), B(a.Tyz)};
}

__device__ __forceinline__ float rsqrt_(float x) { return rsqrtf(x); }
__device__ __forceinline__ double rsqrt_(double x) { return rsqrt(x); }

// ---------------------------------------------------------------------------------------------
// Landau matching (Eq. (eigenproblem), Sec. II.D).  U is the timelike eigenvector of
// T^a_b = T^{ac} eta_{cb}.  Shifted power iteration started from the Eckart vector N/|N|:
//   V = T.(eta U),  rho = U.V,  W = V + (rho/3) U,  U <- W / |W|.
// The shift rho/3 moves the spacelike eigenvalues -P_k to rho/3 - P_k, which vanish in local
// equilibrium (eps = 3P), so the contraction factor is the relative pressure anisotropy instead
// of P/eps = 1/3.  eps is the Rayleigh quotient U.V, n = U.N.  Each lane stops once converged (a
// warp runs as long as its slowest cell).
// ---------------------------------------------------------------------------------------------
template <class A>
struct Landau {
  A U0, Ux, Uy, Uz, eps, n;
  bool ok;    // a timelike frame with eps > 0 and n > 0
  bool conv;  // the last update moved U by at most tol * U0 (false: stopped at MAXIT)
};

// a.b = a0 b0 - ax bx - ay by - az bz: the product ax bx rounded, the others as multiply-adds.  Written out,
// like the products below that something is subtracted from: which of them the compiler contracts depends on
// the code around, and a cell has to come out the same in every kernel.
__device__ __forceinline__ float mul_rn(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ double mul_rn(double a, double b) { return __dmul_rn(a, b); }
__device__ __forceinline__ float sub_rn(float a, float b) { return __fsub_rn(a, b); }
__device__ __forceinline__ double sub_rn(double a, double b) { return __dsub_rn(a, b); }
template <class A>
__device__ __forceinline__ A minkowski(A a0, A ax, A ay, A az, A b0, A bx, A by, A bz) {
  return fma(-az, bz, fma(-ay, by, fma(a0, b0, -mul_rn(ax, bx))));
}

// Shifted power iteration from the start vector (U0, Ux, Uy, Uz), at most MAXIT updates; a lane
// stops once an update moves U by at most tol * U0.
template <class A, int MAXIT>
__device__ __forceinline__ Landau<A> landau_from(const Mom<A>& m, A U0, A Ux, A Uy, A Uz, const A tol) {
  Landau<A> r;
  r.ok = false;
  r.conv = false;
  for (int it = 0; it < MAXIT; ++it) {
    const A V0 = minkowski(m.T00, m.T0x, m.T0y, m.T0z, U0, Ux, Uy, Uz);
    const A Vx = minkowski(m.T0x, m.Txx, m.Txy, m.Txz, U0, Ux, Uy, Uz);
    const A Vy = minkowski(m.T0y, m.Txy, m.Tyy, m.Tyz, U0, Ux, Uy, Uz);
    const A Vz = minkowski(m.T0z, m.Txz, m.Tyz, m.Tzz, U0, Ux, Uy, Uz);
    const A s = minkowski(U0, Ux, Uy, Uz, V0, Vx, Vy, Vz) * A(1.0 / 3.0);
    const A W0 = fma(s, U0, V0), Wx = fma(s, Ux, Vx), Wy = fma(s, Uy, Vy), Wz = fma(s, Uz, Vz);
    const A WW = minkowski(W0, Wx, Wy, Wz, W0, Wx, Wy, Wz);
    if (!(WW > A(0)) || !(W0 > A(0))) return r;
    const A iw = rsqrt_(WW);
    const A n0 = mul_rn(W0, iw), nx = mul_rn(Wx, iw), ny = mul_rn(Wy, iw), nz = mul_rn(Wz, iw);
    const A d = fmax(fmax(fabs(n0 - U0), fabs(nx - Ux)), fmax(fabs(ny - Uy), fabs(nz - Uz)));
    U0 = n0; Ux = nx; Uy = ny; Uz = nz;
    if (d <= tol * U0) {
      r.conv = true;
      break;
    }
  }
  const A V0 = minkowski(m.T00, m.T0x, m.T0y, m.T0z, U0, Ux, Uy, Uz);
  const A Vx = minkowski(m.T0x, m.Txx, m.Txy, m.Txz, U0, Ux, Uy, Uz);
  const A Vy = minkowski(m.T0y, m.Txy, m.Tyy, m.Tyz, U0, Ux, Uy, Uz);
  const A Vz = minkowski(m.T0z, m.Txz, m.Tyz, m.Tzz, U0, Ux, Uy, Uz);
  r.eps = minkowski(U0, Ux, Uy, Uz, V0, Vx, Vy, Vz);
  r.n = minkowski(U0, Ux, Uy, Uz, m.N0, m.Nx, m.Ny, m.Nz);
  r.U0 = U0; r.Ux = Ux; r.Uy = Uy; r.Uz = Uz;
  r.ok = (r.eps > A(0)) && (r.n > A(0)) && isfinite(r.eps) && isfinite(r.n);
  return r;
}

// Landau matching from the Eckart vector N / |N|; double stops at 8e-16 U0 (a few units in the last
// place), float at 3e-7 U0.
template <class A, int MAXIT>
__device__ __forceinline__ Landau<A> landau(const Mom<A>& m) {
  const A NN = minkowski(m.N0, m.Nx, m.Ny, m.Nz, m.N0, m.Nx, m.Ny, m.Nz);
  if (!(NN > A(0)) || !(m.N0 > A(0))) {
    Landau<A> r;
    r.ok = false;
    r.conv = false;
    return r;
  }
  const A is = rsqrt_(NN);
  const A tol = std::is_same<A, double>::value ? A(8e-16) : A(3e-7);
  return landau_from<A, MAXIT>(m, m.N0 * is, m.Nx * is, m.Ny * is, m.Nz * is, tol);
}

// Landau matching of double moments.  The power iteration gains one to two digits an update at the
// relative anisotropies of a flow, some 16 double updates of 50 operations from the Eckart vector.
// Here the float iteration (whose pipe is 64 times wider) gives U to 1e-7 first; then each correction
// forms the residual r = V - eps U, V = T.(eta U), in double, and solves (T - eps) d = -r in float: on
// the vectors orthogonal to U, where r and d live, T - eps is -4 eps / 3 up to the anisotropy, so d is
// a short Richardson iteration, and U + d is right to the digits that d has (six) beyond the last.
// Two corrections reach the last place of double.  A cell whose Eckart Lorentz factor exceeds 4 or
// whose corrections do not fall below 3e-11 U0 takes the power iteration in double (cut off at MAXIT
// updates).  Out of line: a call keeps the step's code small.
template <int MAXIT>
static __device__ __noinline__ Landau<double> landau_f64(const Mom<double> m) {
  const float N0 = (float)m.N0, Nx = (float)m.Nx, Ny = (float)m.Ny, Nz = (float)m.Nz;
  const float NN = minkowski(N0, Nx, Ny, Nz, N0, Nx, Ny, Nz);
  if (N0 > 0.f && 16.f * NN > N0 * N0 && N0 < 1e15f && N0 > 1e-15f) {
    const Mom<float> t = convert<double, float>(m);
    const Landau<float> lf = landau<float, 8>(t);
    if (lf.ok && lf.conv) {
      double Ux = lf.Ux, Uy = lf.Uy, Uz = lf.Uz;
      double U0 = sqrt(fma(Ux, Ux, fma(Uy, Uy, fma(Uz, Uz, 1.0))));
      const float u0 = (float)U0, e1 = lf.eps, k = 0.75f / e1, tiny = 3e-11f * u0;
      for (int it = 0; it < 4; ++it) {
        const double V0 = minkowski(m.T00, m.T0x, m.T0y, m.T0z, U0, Ux, Uy, Uz);
        const double Vx = minkowski(m.T0x, m.Txx, m.Txy, m.Txz, U0, Ux, Uy, Uz);
        const double Vy = minkowski(m.T0y, m.Txy, m.Tyy, m.Tyz, U0, Ux, Uy, Uz);
        const double Vz = minkowski(m.T0z, m.Txz, m.Tyz, m.Tzz, U0, Ux, Uy, Uz);
        const double eps = minkowski(U0, Ux, Uy, Uz, V0, Vx, Vy, Vz);
        const float r0 = (float)fma(-eps, U0, V0), rx = (float)fma(-eps, Ux, Vx), ry = (float)fma(-eps, Uy, Vy),
                    rz = (float)fma(-eps, Uz, Vz);
        float d0 = k * r0, dx = k * rx, dy = k * ry, dz = k * rz;
        for (int j = 0; j < 12; ++j) {
          const float g0 = fmaf(t.T00, d0, fmaf(-t.T0x, dx, fmaf(-t.T0y, dy, fmaf(-t.T0z, dz, fmaf(-e1, d0, r0)))));
          const float gx = fmaf(t.T0x, d0, fmaf(-t.Txx, dx, fmaf(-t.Txy, dy, fmaf(-t.Txz, dz, fmaf(-e1, dx, rx)))));
          const float gy = fmaf(t.T0y, d0, fmaf(-t.Txy, dx, fmaf(-t.Tyy, dy, fmaf(-t.Tyz, dz, fmaf(-e1, dy, ry)))));
          const float gz = fmaf(t.T0z, d0, fmaf(-t.Txz, dx, fmaf(-t.Tyz, dy, fmaf(-t.Tzz, dz, fmaf(-e1, dz, rz)))));
          d0 = fmaf(k, g0, d0), dx = fmaf(k, gx, dx), dy = fmaf(k, gy, dy), dz = fmaf(k, gz, dz);
          const float step = fmaxf(fmaxf(fabsf(gx), fabsf(gy)), fmaxf(fabsf(gz), fabsf(g0)));
          const float size = fmaxf(fmaxf(fabsf(dx), fabsf(dy)), fmaxf(fabsf(dz), fabsf(d0)));
          if (k * step <= 1e-6f * size) break;
        }
        U0 += d0, Ux += dx, Uy += dy, Uz += dz;
        // back to U.U = 1 (to second order in its deviation)
        const double q = fma(U0, U0, -1.0 - fma(Ux, Ux, fma(Uy, Uy, Uz * Uz)));
        const double h = -0.5 * q;
        U0 = fma(h, U0, U0), Ux = fma(h, Ux, Ux), Uy = fma(h, Uy, Uy), Uz = fma(h, Uz, Uz);
        if (fmaxf(fmaxf(fabsf(dx), fabsf(dy)), fmaxf(fabsf(dz), fabsf(d0))) <= tiny) {
          Landau<double> r;
          r.U0 = U0, r.Ux = Ux, r.Uy = Uy, r.Uz = Uz;
          r.eps = eps;  // of the U before the last correction: second order in it
          r.n = minkowski(U0, Ux, Uy, Uz, m.N0, m.Nx, m.Ny, m.Nz);
          r.ok = r.eps > 0.0 && r.n > 0.0 && isfinite(r.eps) && isfinite(r.n);
          r.conv = true;
          return r;
        }
      }
    }
  }
  return landau<double, MAXIT>(m);
}

// The double-precision solve of a float step, kept out of line: it runs for few cells and would
// otherwise grow the step kernel's hot code (a call keeps the caller's register allocation that of
// the float path).  It starts from the Eckart vector and stops at 1e-12 U0: the populations are
// float, so more digits carry no information, while the double arithmetic still removes the
// gamma^2 cancellation in U.U = 1.
static __device__ __noinline__ Landau<double> landau_fp64_out_of_line(const Mom<double> m) {
  const double NN = minkowski(m.N0, m.Nx, m.Ny, m.Nz, m.N0, m.Nx, m.Ny, m.Nz);
  if (!(NN > 0.0) || !(m.N0 > 0.0)) {
    Landau<double> r;
    r.ok = false;
    r.conv = false;
    return r;
  }
  const double is = rsqrt(NN);
  Landau<double> r = landau_from<double, 40>(m, m.N0 * is, m.Nx * is, m.Ny * is, m.Nz * is, 1e-12);
  r.ok = r.ok && r.conv;  // no frame to 1e-12 in 40 double updates: reported, not used
  return r;
}

// Landau matching in the step's arithmetic A.  Reduced-precision paths switch to double for cells
// whose Eckart Lorentz factor exceeds gamma_thr (or always, if asked): the solve loses about
// gamma^2 digits to cancellation in U.U = 1.
// A double solve that stops at MAXIT without meeting its tolerance is accepted only if the last
// update was below 1e-10 U0 (round-off can keep the last digits moving); a float solve that does
// not converge in 8 updates is redone in double.
template <class A>
__device__ __forceinline__ Landau<A> landau_step(const Mom<A>& m, const StepParams& p) {
  if constexpr (std::is_same<A, double>::value) {
    Landau<double> r = landau_f64<40>(m);
    if (r.ok && !r.conv) {
      const Landau<double> again = landau_from<double, 1>(m, r.U0, r.Ux, r.Uy, r.Uz, 1e-10);
      r.ok = again.ok && again.conv;
    }
    return r;
  } else {
    const float NN = minkowski(m.N0, m.Nx, m.Ny, m.Nz, m.N0, m.Nx, m.Ny, m.Nz);
    Landau<float> r;
    const bool dbl = p.landau_fp64 || m.N0 * m.N0 > p.gamma_thr2 * NN;
    if (!dbl) {
      r = landau<float, 8>(m);
      if (r.conv || !r.ok) return r;
    }
    const Landau<double> d = landau_fp64_out_of_line(convert<A, double>(m));
    return Landau<A>{(A)d.U0, (A)d.Ux, (A)d.Uy, (A)d.Uz, (A)d.eps, (A)d.n, d.ok, d.conv};
  }
}

template <class A>
__device__ __forceinline__ A tau_prime(A T, const StepParams& p) {
  if constexpr (std::is_same<A, double>::value) {
    if (p.tau_is_fixed) return p.tau_fixed;
    const double Tt = p.tau_local ? T : p.T_ref;
    return 0.5 + p.tau_coef / Tt;
  } else {
    if (p.tau_is_fixed) return p.tau_fixed_f;
    const float Tt = p.tau_local ? T : p.T_ref_f;
    return 0.5f + p.tau_coef_f / Tt;
  }
}

// ---------------------------------------------------------------------------------------------
// Equilibrium in factored form.  The projection of the Maxwell-Juttner distribution onto the
// polynomials of degree <= order depends on p only through p0 and s = p.U (rotational symmetry
// about U), so f_i^eq = w_i E(p0_i, t_i) with s = p0 t, t = v.U/R, and, with x = T U0 - 1:
//   order 3:  E = n/(12T) [c00 + p0 (c10 + c01 t) + p0^2 (c20 + c11 t + c02 t^2) + p0^3 (x + T t)^3]
//   order 2:  E = n/(4T)  [c00 + p0 (c10 + c01 t) + p0^2 (x + T t)^2]
// which is App. B's Eq. (eq:equi3rd) / (eq:equi2nd) regrouped.
// ---------------------------------------------------------------------------------------------
template <int ORDER, class A>
struct EqCoef {
  A c00, c10, c01, c20, c11, c02, x, T, pref;
};

template <int ORDER, class A>
__device__ __forceinline__ EqCoef<ORDER, A> eq_coef(A n, A T, A U0) {
  EqCoef<ORDER, A> c;
  const A x = fma(T, U0, A(-1));
  const A x2 = mul_rn(x, x), T2 = mul_rn(T, T);
  c.x = x;
  c.T = T;
  if constexpr (ORDER == 3) {
    const A pref = n / (A(12) * T);
    c.pref = pref;
    c.c00 = A(-6) * pref * fma(T2, fma(A(-4), x, A(1)), fma(x2, fma(A(8), x, A(4)), fma(A(4), x, A(-2))));
    c.c10 = A(6) * pref * fma(T2, fma(A(-6), x, A(1)), fma(x2, fma(A(12), x, A(8)), fma(A(5), x, A(-1))));
    c.c01 = A(6) * pref * T * fma(A(-2), T2, fma(A(12), x2, A(3)));
    c.c20 = A(-3) * pref * x * fma(A(-2), T2, fma(x, fma(A(6), x, A(3)), A(2)));
    c.c11 = A(-6) * pref * T * (fma(x, fma(A(6), x, A(1)), A(1)) - T2);
    c.c02 = A(-3) * pref * T2 * fma(A(6), x, A(-1));
  } else {
    const A pref = n / (A(4) * T);
    c.pref = pref;
    c.c00 = A(2) * pref * (fma(A(4), x2, A(2)) - T2);
    c.c10 = A(-2) * pref * (fma(x, fma(A(4), x, A(1)), A(1)) - T2);
    c.c01 = A(-2) * pref * T * fma(A(4), x, A(-1));
    c.c20 = c.c11 = c.c02 = A(0);
  }
  return c;
}

// The equilibrium as a polynomial in t per energy level l (p0 = p0_l):
//   E(p0_l, t) = a_l + t (b_l + t (c_l + t d_l)),
//   order 3: a = c00 + p0 c10 + p0^2 c20 + pref p0^3 x^3,  b = p0 c01 + p0^2 c11 + 3 pref p0^3 x^2 T,
//            c = p0^2 c02 + 3 pref p0^3 x T^2,             d = pref p0^3 T^3;
//   order 2: a = c00 + p0 c10 + pref p0^2 x^2,  b = p0 c01 + 2 pref p0^2 x T,  c = pref p0^2 T^2,  d = 0.
// The same regrouping of App. B's forms: the per-cell work moves from the 48 (15) directions to
// the 4 (3) energy levels, and each population costs a cubic (quadratic) Horner step in t.
template <class L, class A>
struct LevCoef {
  A a[L::NLEV], b[L::NLEV], c[L::NLEV], d[L::NLEV];
};

// shift: subtracted from every a_l (deviation space evaluates E - c)
template <class L, class A>
__device__ __forceinline__ LevCoef<L, A> level_coef(const EqCoef<L::ORDER, A>& q, A shift = A(0)) {
  LevCoef<L, A> r;
  const A c00 = shift == A(0) ? q.c00 : sub_rn(q.c00, shift);
  static_for<L::NLEV>([&](auto K) {
    constexpr int l = decltype(K)::value;
    constexpr double pd = L::P0[l];
    const A p = A(pd), p2 = A(pd * pd);
    if constexpr (L::ORDER == 3) {
      const A pp3 = A(pd * pd * pd) * q.pref;  // pref p0^3
      const A ppx = pp3 * q.x;
      r.d[l] = pp3 * (q.T * q.T * q.T);
      r.c[l] = fma(A(3) * ppx, q.T * q.T, p2 * q.c02);
      r.b[l] = fma(A(3) * ppx * q.x, q.T, fma(p2, q.c11, p * q.c01));
      r.a[l] = fma(ppx * q.x, q.x, fma(p2, q.c20, fma(p, q.c10, c00)));
    } else {
      const A pp2 = p2 * q.pref;  // pref p0^2
      r.d[l] = A(0);
      r.c[l] = pp2 * (q.T * q.T);
      r.b[l] = fma(A(2) * pp2 * q.x, q.T, p * q.c01);
      r.a[l] = fma(pp2 * q.x, q.x, fma(p, q.c10, c00));
    }
  });
  return r;
}

// Collision of one cell (Eq. (rlb:disc) right-hand side, delta t' = 1):
//   f*_i = f_i + omega_i (w_i E_i - f_i),  omega_i = p_i.U / (tau' p0_i) = (U0 - t_i) / tau'.
// DEV = true: get / put carry deviations d_i = f_i / w_i - c, and the collision is
// d_i + omega_i ((E_i - c) - d_i).
// The part of it that +v (population I) and -v share: t = v.U / R of +v and the two omegas.
template <class A>
struct DirTerm {
  A t, t2, omp, omm;
};
template <class L, class A, int I>
__device__ __forceinline__ DirTerm<A> dir_term(A Ux, A Uy, A Uz, A inv_tau, A a) {
  constexpr int vx = L::VX[I], vy = L::VY[I], vz = L::VZ[I];
  constexpr double ir = L::INV_R;
  A t = A(0);  // direction +v: t; mirror -v: -t
  if constexpr (vx != 0) t = fma(A(vx * ir), Ux, t);
  if constexpr (vy != 0) t = fma(A(vy * ir), Uy, t);
  if constexpr (vz != 0) t = fma(A(vz * ir), Uz, t);
  return DirTerm<A>{t, t * t, fma(-t, inv_tau, a), fma(t, inv_tau, a)};
}
// One mirror pair.  The even part a + c t^2 and the odd part's factor b + d t^2 serve both signs of t.
template <class L, class A, bool DEV, int IP, class Get, class Put>
__device__ __forceinline__ void collide_pair(const DirTerm<A>& k, A ea, A eb, A ec, A ed, Get&& get, Put&& put) {
  const A w = A(L::W[IP]);
  const A even = fma(k.t2, ec, ea);
  A odd = eb;
  if constexpr (L::ORDER == 3) odd = fma(k.t2, ed, odd);
  const A Ep = fma(k.t, odd, even), Em = fma(-k.t, odd, even);
  const A fp = get(ic<IP>{}), fm = get(ic<IP + 1>{});
  if constexpr (DEV) {
    put(ic<IP>{}, fma(k.omp, Ep - fp, fp));
    put(ic<IP + 1>{}, fma(k.omm, Em - fm, fm));
    (void)w;
  } else {
    put(ic<IP>{}, fma(k.omp, fma(w, Ep, -fp), fp));
    put(ic<IP + 1>{}, fma(k.omm, fma(w, Em, -fm), fm));
  }
}
template <class L, class A, bool DEV = false, class Get, class Put>
__device__ __forceinline__ void collide(const Landau<A>& lw, A T, A inv_tau, Get&& get, Put&& put, A c = A(0)) {
  const LevCoef<L, A> e = level_coef<L, A>(eq_coef<L::ORDER, A>(lw.n, T, lw.U0), DEV ? c : A(0));
  const A a = lw.U0 * inv_tau;
  static_for<L::NDP>([&](auto K) {
    constexpr int k = decltype(K)::value;
    constexpr int first = L::DP_FIRST[k];
    const DirTerm<A> dt = dir_term<L, A, first>(lw.Ux, lw.Uy, lw.Uz, inv_tau, a);
    static_for<L::DP_NPAIR[k]>([&](auto J) {
      constexpr int ip = first + 2 * decltype(J)::value;
      constexpr int l = L::LEV[ip];
      collide_pair<L, A, DEV, ip>(dt, e.a[l], e.b[l], e.c[l], e.d[l], get, put);
    });
  });
}

// ---------------------------------------------------------------------------------------------
// Float arithmetic in mirror pairs.  Populations i (direction +v) and i + 1 (direction -v) share
// energy and weight, so their work is one float2 operation (sm_100+ paired FP32 FMA):
// moments accumulate per sign with sign-symmetric constants, and the equilibrium and collision of
// the pair are evaluated together with t2 = (t, -t).
// ---------------------------------------------------------------------------------------------
__device__ __forceinline__ float2 f2(float a, float b) { return make_float2(a, b); }
__device__ __forceinline__ float2 ffma2(float2 a, float2 b, float2 c) { return __ffma2_rn(a, b, c); }
__device__ __forceinline__ float2 fadd2(float2 a, float2 b) { return __fadd2_rn(a, b); }

// Sums of the direction pairs [DPB, DPE) in paired arithmetic: the 13 independent moments before
// the weights' own moments (deviation space) and the trace identity are added (finish_moments_f2).
template <class L, bool DEV = false, int DPB = 0, int DPE = L::NDP, class Get2>
__device__ __forceinline__ Mom<float> moments_f2_part(Get2&& get2) {
  const float2 z = f2(0.f, 0.f);
  float2 N0 = z, Nx = z, Ny = z, Nz = z, T00 = z, T0x = z, T0y = z, T0z = z, Txx = z, Tyy = z, Txy = z, Txz = z, Tyz = z;
  static_for<DPE - DPB>([&](auto K) {
    constexpr int k = DPB + decltype(K)::value;
    constexpr int first = L::DP_FIRST[k];
    constexpr int np = L::DP_NPAIR[k];
    float2 S1 = z, S2 = z;  // (sum over energies for +v, for -v)
    static_for<np>([&](auto J) {
      constexpr int ip = first + 2 * decltype(J)::value;
      constexpr double wk = DEV ? L::W[ip] : 1.0;  // mirror partners share the weight
      constexpr float p0 = (float)(wk * L::P0[L::LEV[ip]]);
      constexpr float p02 = (float)(wk * L::P0[L::LEV[ip]] * L::P0[L::LEV[ip]]);
      const float2 f = get2(ic<ip>{});
      S1 = ffma2(f2(p0, p0), f, S1);
      S2 = ffma2(f2(p02, p02), f, S2);
    });
    constexpr int vx = L::VX[first], vy = L::VY[first], vz = L::VZ[first];
    constexpr double ir = L::INV_R, ir2 = L::INV_R2;
    N0 = fadd2(N0, S1);
    T00 = fadd2(T00, S2);
    if constexpr (vx != 0) {
      constexpr float c = (float)(vx * ir);
      constexpr float cc = (float)(vx * vx * ir2);
      Nx = ffma2(f2(c, -c), S1, Nx);
      T0x = ffma2(f2(c, -c), S2, T0x);
      Txx = ffma2(f2(cc, cc), S2, Txx);
    }
    if constexpr (vy != 0) {
      constexpr float c = (float)(vy * ir);
      constexpr float cc = (float)(vy * vy * ir2);
      Ny = ffma2(f2(c, -c), S1, Ny);
      T0y = ffma2(f2(c, -c), S2, T0y);
      Tyy = ffma2(f2(cc, cc), S2, Tyy);
    }
    if constexpr (vz != 0) {
      constexpr float c = (float)(vz * ir);
      Nz = ffma2(f2(c, -c), S1, Nz);
      T0z = ffma2(f2(c, -c), S2, T0z);
    }
    if constexpr (vx != 0 && vy != 0) {
      constexpr float cc = (float)(vx * vy * ir2);
      Txy = ffma2(f2(cc, cc), S2, Txy);
    }
    if constexpr (vx != 0 && vz != 0) {
      constexpr float cc = (float)(vx * vz * ir2);
      Txz = ffma2(f2(cc, cc), S2, Txz);
    }
    if constexpr (vy != 0 && vz != 0) {
      constexpr float cc = (float)(vy * vz * ir2);
      Tyz = ffma2(f2(cc, cc), S2, Tyz);
    }
  });
  Mom<float> m;
  m.N0 = N0.x + N0.y;
  m.Nx = Nx.x + Nx.y;
  m.Ny = Ny.x + Ny.y;
  m.Nz = Nz.x + Nz.y;
  m.T00 = T00.x + T00.y;
  m.T0x = T0x.x + T0x.y;
  m.T0y = T0y.x + T0y.y;
  m.T0z = T0z.x + T0z.y;
  m.Txx = Txx.x + Txx.y;
  m.Tyy = Tyy.x + Tyy.y;
  m.Txy = Txy.x + Txy.y;
  m.Txz = Txz.x + Txz.y;
  m.Tyz = Tyz.x + Tyz.y;
  m.Tzz = 0.f;
  return m;
}

// The weights' own moments times c (deviation space) and T^zz from the trace identity.
template <class L, bool DEV = false>
__device__ __forceinline__ void finish_moments_f2(Mom<float>& m, float c = 0.f) {
  if constexpr (DEV) add_rest_sums<L, float>(m, c);
  m.Tzz = m.T00 - m.Txx - m.Tyy;
}

template <class L, bool DEV = false, class Get2>
__device__ __forceinline__ Mom<float> moments_f2(Get2&& get2, float c = 0.f) {
  Mom<float> m = moments_f2_part<L, DEV>(get2);
  finish_moments_f2<L, DEV>(m, c);
  return m;
}

// What the paired collision of one cell needs: the level coefficients, U and the relaxation rate.
template <class L>
struct CollideCoef {
  LevCoef<L, float> e;
  float Ux, Uy, Uz, inv_tau, a;  // a = U0 / tau'
};
template <class L, bool DEV>
__device__ __forceinline__ CollideCoef<L> collide_coef(const Landau<float>& lw, float T, float inv_tau, float c) {
  return CollideCoef<L>{level_coef<L, float>(eq_coef<L::ORDER, float>(lw.n, T, lw.U0), DEV ? c : 0.f), lw.Ux, lw.Uy,
                        lw.Uz, inv_tau, lw.U0 * inv_tau};
}

// Collision of the direction pairs [DPB, DPE) (all of them by default).
template <class L, bool DEV = false, int DPB = 0, int DPE = L::NDP, class Get2, class Put2>
__device__ __forceinline__ void collide_f2(const CollideCoef<L>& q, Get2&& get2, Put2&& put2) {
  // the coefficients as (x, x) pairs once per cell, the operands of the paired Horner steps
  struct {
    float2 a[L::NLEV], b[L::NLEV], c[L::NLEV], d[L::NLEV];
  } e;
  static_for<L::NLEV>([&](auto K) {
    constexpr int l = decltype(K)::value;
    e.a[l] = f2(q.e.a[l], q.e.a[l]);
    e.b[l] = f2(q.e.b[l], q.e.b[l]);
    e.c[l] = f2(q.e.c[l], q.e.c[l]);
    e.d[l] = f2(q.e.d[l], q.e.d[l]);
  });
  const float2 Uxp = f2(q.Ux, q.Ux), Uyp = f2(q.Uy, q.Uy), Uzp = f2(q.Uz, q.Uz);
  const float2 itp = f2(q.inv_tau, q.inv_tau), nap = f2(-q.a, -q.a);
  static_for<DPE - DPB>([&](auto K) {
    constexpr int k = DPB + decltype(K)::value;
    constexpr int first = L::DP_FIRST[k];
    constexpr int np = L::DP_NPAIR[k];
    constexpr int vx = L::VX[first], vy = L::VY[first], vz = L::VZ[first];
    constexpr double ir = L::INV_R;
    float2 tt = f2(0.f, 0.f);  // (t, -t), t = v.U / R
    if constexpr (vx != 0) tt = ffma2(f2((float)(vx * ir), (float)(-vx * ir)), Uxp, tt);
    if constexpr (vy != 0) tt = ffma2(f2((float)(vy * ir), (float)(-vy * ir)), Uyp, tt);
    if constexpr (vz != 0) tt = ffma2(f2((float)(vz * ir), (float)(-vz * ir)), Uzp, tt);
    const float2 nom = ffma2(itp, tt, nap);  // -(U0 - t) / tau' for +v, -(U0 + t) / tau' for -v
    static_for<np>([&](auto J) {
      constexpr int ip = first + 2 * decltype(J)::value;
      constexpr int l = L::LEV[ip];
      constexpr float nw = DEV ? -1.f : (float)(-L::W[ip]);
      float2 E;
      if constexpr (L::ORDER == 3)
        E = ffma2(tt, ffma2(tt, ffma2(tt, e.d[l], e.c[l]), e.b[l]), e.a[l]);
      else
        E = ffma2(tt, ffma2(tt, e.c[l], e.b[l]), e.a[l]);
      const float2 f = get2(ic<ip>{});
      const float2 d = ffma2(f2(nw, nw), E, f);  // f - w E (deviation space: d - (E - c))
      put2(ic<ip>{}, ffma2(nom, d, f));        // f - omega (f - w E)
    });
  });
}

// ---------------------------------------------------------------------------------------------
// the fused step kernel
// ---------------------------------------------------------------------------------------------
// Compiler-level barrier: values read from memory before it are read again after it.
__device__ __forceinline__ void reload_barrier() { asm volatile("" ::: "memory"); }

// Moments, Landau matching, relaxation time, equilibrium and collision of one cell (steps a2-a7)
// whose pulled populations get(I) returns (deviations d_i for half-deviation storage); store(I, v)
// writes post-collision population I.  Shared by every step kernel, whatever it pulls from
// (registers, global memory or a shared-memory stage).  RELOAD = true makes the collision read
// every population again through get instead of keeping the moment pass's values in registers
// (for populations staged in shared memory).  A cell without a Landau frame is counted in status
// (valid lanes only) and streamed without collision.
template <class L, class S, bool PACKED, bool RELOAD = false, class Get, class Store>
__device__ __forceinline__ void relax_cell(Get&& get, Store&& store, const StepParams& p, int* __restrict__ status,
                                           const bool valid) {
  using A = typename S::A;
  constexpr bool DEV = std::is_same<S, StoreF16Dev>::value;
  const A c_dev = DEV ? A(p.half_nref) : A(0);
  auto get2 = [&](auto I) -> float2 {
    constexpr int i = decltype(I)::value;
    return make_float2((float)get(ic<i>{}), (float)get(ic<i + 1>{}));
  };
  Mom<A> m;
  if constexpr (PACKED) m = moments_f2<L, DEV>(get2, (float)c_dev);
  else if constexpr (std::is_same<A, double>::value) m = moments_fixed<L>(get);
  else m = moments<L, A, DEV>(get, c_dev);
  if constexpr (RELOAD) reload_barrier();
  const Landau<A> lw = landau_step<A>(m, p);
  if (!lw.ok) {
    // no Landau frame: record it and stream the populations without collision
    if (valid) {
      atomicAdd(&status[kStatusNonconv], 1);
      static_for<L::Q>([&](auto I) { store(I, get(I)); });
    }
    return;
  }
  const A T = lw.eps / (A(3) * lw.n);
  const A inv_tau = A(1) / tau_prime<A>(T, p);
  if constexpr (PACKED) {
    auto put2 = [&](auto I, float2 v) {
      constexpr int i = decltype(I)::value;
      store(ic<i>{}, v.x);
      store(ic<i + 1>{}, v.y);
    };
    collide_f2<L, DEV>(collide_coef<L, DEV>(lw, T, inv_tau, (float)c_dev), get2, put2);
  } else {
    collide<L, A, DEV>(lw, T, inv_tau, get, store, c_dev);
  }
}

// Step-kernel variants for float arithmetic.  Every population is pulled once and all populations
// of a cell stay in registers.
//   bit 0: scalar arithmetic (0) or mirror pairs in float2 with paired FMA (1);
//   bit 1: registers as needed, 2 resident blocks of 128 threads per SM (0), or at most 168
//          registers for 3 resident blocks (1; the compiler spills a little).
// (Also measured slower and not built: keeping half-deviation populations as packed half2 pairs
// at 4 resident blocks (128 registers still spill); staging part of the populations in shared
// memory; a persistent interior kernel that prefetches each thread's next cell into shared memory
// with cp.async while it computes the current one; and two passes over the populations, moments
// then collision, at 64-80 registers and 6-8 resident blocks with L2 evict-last / evict-first
// hints, whose second pass executed about 50% more instructions and still missed L2 on a third
// of its reads.)
// Double arithmetic pulls each population twice (moments, then collision) and has one variant.
enum StepVariant : int { kRegScalar = 0, kRegPacked = 1, kReg3Scalar = 2, kReg3Packed = 3, kNumVariants = 4 };

// The scalar second-order cell asks for 184 registers but fits 168 without spills, so it has 3 blocks either
// way (160 x 70 x 70 float 120 us a step in two blocks, 106 in three).
template <class L, class S, int VARIANT>
struct StepShape {
  static constexpr bool kKeep = std::is_same<typename S::A, float>::value;  // populations in registers
  static constexpr int kMinBlocks = (VARIANT & 2) || (kKeep && L::ORDER == 2 && !(VARIANT & 1)) ? 3 : 1;
};

// How a step kernel pulls: the row kernel's warps lie in rows with interior y and z and are told
// whether their x segment is interior too (constant offsets) or not (only x wraps); the shell row
// kernel's warps lie in boundary rows, whose y and z shifts are the same for the whole warp; the
// per-cell shell kernel (lattices shorter than the stencil reach) wraps every coordinate of every
// cell.
enum PullPath : int { kPathRow = 1, kPathEdge = 2, kPathShellTab = 3 };

// One cell's time step (pull, moments, Landau matching, equilibrium, collision, store).  Invalid
// lanes (valid = false) carry a clamped in-range cell, compute and store nothing.
template <class L, class S, bool GENERAL, int VARIANT, int PATH, bool WALLS>
__device__ __forceinline__ void step_cell(const typename S::T* __restrict__ src, typename S::T* __restrict__ dst,
                                          const StepParams& p, int* __restrict__ status, const Cell cl,
                                          const bool valid, const bool row_fast = false,
                                          const long long* __restrict__ roff = nullptr,
                                          const uint32_t* walled = nullptr) {
  using A = typename S::A;
  using ST = typename S::T;
  constexpr bool PACKED = (VARIANT & 1) && std::is_same<A, float>::value;
  constexpr bool KEEP = StepShape<L, S, VARIANT>::kKeep;
  // Warp-uniform choice: a row warp whose segment is interior pulls with constant offsets; other
  // row warps wrap x only; shell cells resolve wrap / copy-out / bounce-back per population.
  static_assert(PATH == kPathRow || PATH == kPathEdge || PATH == kPathShellTab, "pull path");
  const bool fast = PATH == kPathRow && row_fast;
  const ST* __restrict__ base = src + cl.c;
  ST* __restrict__ out = dst + cl.c;
  // Half-deviation storage works in deviation space: the values in flight are d_i = f_i / w_i - c
  // as stored, and the moments and collision take the weights and c into their constants.
  constexpr bool DEV = std::is_same<S, StoreF16Dev>::value;
  auto ld = [&](auto I, const ST* ptr) -> A {
    constexpr int i = decltype(I)::value;
    if constexpr (DEV) return S::template load_dev<L, i>(ptr, p);
    else return S::template load<L, i>(ptr, p);
  };

  auto load = [&](auto I) -> A {
    constexpr int i = decltype(I)::value;
    if (fast) return ld(I, base + p.off[i]);
    if constexpr (PATH == kPathRow) return ld(I, base + x_row_offset<L, i, WALLS>(cl, p));
    else if constexpr (PATH == kPathShellTab) {
      constexpr int vx = L::VX[i];
      long long o = roff[i];
      if constexpr (vx != 0) {
        bool shift = !row_fast;
        if constexpr (WALLS) shift = shift && !(walled[i / 32] >> (i % 32) & 1u);
        if (shift) {
          if (WALLS && p.bc[0] == kBounceBack && (unsigned)(cl.x - vx) >= (unsigned)p.nx) o = (long long)(i ^ 1) * p.cells;
          else o += src_coord<vx, false>(cl.x, p.nx, p.bc[0]) - (cl.x - vx);
        }
      }
      return ld(I, base + o);
    }
    else return ld(I, src + pull_index<L, i, GENERAL, WALLS>(cl, p));
  };
  auto store = [&](auto I, A v) {
    constexpr int i = decltype(I)::value;
    if (valid) {
      if constexpr (DEV) S::template store_dev<L, i>(out + (long long)i * p.cells, v, p);
      else S::template store<L, i>(out + (long long)i * p.cells, v, p);
    }
  };

  A fk[KEEP ? L::Q : 1];
  if constexpr (KEEP) {
    // one warp-uniform branch around the whole pull, so the fast path is plain constant offsets
    if (fast) static_for<L::Q>([&](auto I) { fk[decltype(I)::value] = ld(I, base + p.off[decltype(I)::value]); });
    else static_for<L::Q>([&](auto I) { fk[decltype(I)::value] = load(I); });
  }
  auto get = [&](auto I) -> A {
    if constexpr (KEEP) return fk[decltype(I)::value];
    else return load(I);
  };
  relax_cell<L, S, PACKED>(get, store, p, status, valid);
}

// Cell of lane `lane` in row-kernel warp w (see k_step_interior).
__device__ __forceinline__ void row_cell(int w, int lane, const StepParams& p, Cell& cl, bool& valid, bool& fast) {
  const int seg = w % p.int_segs, row = w / p.int_segs;
  cl.y = p.iy0 + row % p.iyn;
  cl.z = p.iz0 + row / p.iyn;
  const int x0 = seg * 32, x = x0 + lane;
  valid = x < p.nx;
  cl.x = valid ? x : p.nx - 1;
  cl.c = (cl.z * p.ny + cl.y) * p.nx + cl.x;
  fast = x0 >= p.ix0 && min(x0 + 31, p.nx - 1) < p.ix0 + p.ixn;
}

// Interior rows (y and z inside the interior box, every x): warp w covers the 32-aligned x segment
// w % int_segs of row w / int_segs (the last segment may be partial).  A segment inside the
// interior x range pulls with constant offsets; the others wrap only x.  Whole rows in one kernel
// keep every sector of a row written by neighbouring warps.
template <class L, class S, int VARIANT, bool WALLS>
__global__ void __launch_bounds__(kStepThreads, StepShape<L, S, VARIANT>::kMinBlocks)
    k_step_interior(const typename S::T* __restrict__ src, typename S::T* __restrict__ dst,
                    const __grid_constant__ StepParams p, int* __restrict__ status) {
  const int w = blockIdx.x * (kStepThreads / 32) + (threadIdx.x >> 5);
  if (w >= p.int_warps) return;  // whole warps only
  Cell cl;
  bool valid, fast;
  row_cell(w, threadIdx.x & 31, p, cl, valid, fast);
  step_cell<L, S, false, VARIANT, kPathRow, WALLS>(src, dst, p, status, cl, valid, fast);
}

// Row r of the shell: the rows of the z-boundary planes, then the y-boundary rows of the interior
// planes.
__device__ __forceinline__ void shell_row(int r, const StepParams& p, int& y, int& z) {
  const int A = (p.nz - p.izn) * p.ny;
  if (r < A) {
    const int zz = r / p.ny;
    y = r - zz * p.ny;
    z = zz < p.iz0 ? zz : zz + p.izn;
  } else {
    r -= A;
    const int wy = p.ny - p.iyn;
    const int zz = r / wy, yy = r - zz * wy;
    z = p.iz0 + zz;
    y = yy < p.iy0 ? yy : yy + p.iyn;
  }
}

// Shell rows for lattices whose periodic axes are all at least the stencil reach: warp w covers
// the 32-aligned x segment w % row_segs of shell row w / row_segs, so the y and z shifts of each
// population are the same for the whole warp and x wraps only in segments outside the interior x
// range.
// One warp per block, so that the row (and with it every population's y and z shift) derives from
// blockIdx alone, a value the compiler knows to be the same for the whole warp; as many blocks
// per SM as the four-warp kernels have warps.
template <class L, class S, int VARIANT, bool WALLS>
__global__ void __launch_bounds__(32, 4 * StepShape<L, S, VARIANT>::kMinBlocks)
    k_step_shell_rows(const typename S::T* __restrict__ src, typename S::T* __restrict__ dst,
                      const __grid_constant__ StepParams p, int* __restrict__ status) {
  const int w = blockIdx.x;
  const int seg = w % p.row_segs, r = w / p.row_segs;
  Cell cl;
  shell_row(r, p, cl.y, cl.z);
  const int x0 = seg * 32, x = x0 + (threadIdx.x & 31);
  const bool valid = x < p.nx;
  cl.x = valid ? x : p.nx - 1;
  cl.c = (cl.z * p.ny + cl.y) * p.nx + cl.x;
  const bool xfast = x0 >= p.ix0 && min(x0 + 31, p.nx - 1) < p.ix0 + p.ixn;
  __shared__ long long roff[L::Q];
  uint32_t walled[4];
  shell_row_table<L, WALLS>(roff, walled, cl, p);
  step_cell<L, S, false, VARIANT, kPathShellTab, WALLS>(src, dst, p, status, cl, valid, xfast, roff, walled);
}

// Shell cells (rows whose y or z lies outside the interior box): z-boundary planes, then the
// y-boundary rows of the interior planes; wrapped / clamped pulls.
__device__ __forceinline__ Cell shell_cell(int s, const StepParams& p) {
  Cell cl;
  const int A = (p.nz - p.izn) * p.nxy;
  if (s < A) {
    const int zz = s / p.nxy, r = s - zz * p.nxy;
    cl.z = zz < p.iz0 ? zz : zz + p.izn;
    cl.y = r / p.nx;
    cl.x = r - cl.y * p.nx;
  } else {
    s -= A;
    const int rowy = (p.ny - p.iyn) * p.nx;
    const int zz = s / rowy, r = s - zz * rowy;
    cl.z = p.iz0 + zz;
    const int yy = r / p.nx;
    cl.y = yy < p.iy0 ? yy : yy + p.iyn;
    cl.x = r - yy * p.nx;
  }
  cl.c = (cl.z * p.ny + cl.y) * p.nx + cl.x;
  return cl;
}

template <class L, class S, bool GENERAL, int VARIANT, bool WALLS>
__global__ void __launch_bounds__(kStepThreads, StepShape<L, S, VARIANT>::kMinBlocks)
    k_step_shell(const typename S::T* __restrict__ src, typename S::T* __restrict__ dst,
                 const __grid_constant__ StepParams p, int* __restrict__ status) {
  const int s = blockIdx.x * kStepThreads + threadIdx.x;
  const bool valid = s < p.shell_cells;
  const Cell cl = shell_cell(valid ? s : p.shell_cells - 1, p);
  step_cell<L, S, GENERAL, VARIANT, kPathEdge, WALLS>(src, dst, p, status, cl, valid);
}

// ---------------------------------------------------------------------------------------------
// Batched step: many independent lattices (members) advance together.  Each time step is two
// persistent launches, one over the members' row tiles (four row-kernel warps each: constant
// offsets, or x wrapped only) and one over their shell tiles (four shell-row warps each, or
// kStepThreads shell cells each for members that need the modulo wrap): the decomposition of a
// solo step, so a member's populations are bitwise those
// of the same steps taken alone with the same variant, and each kernel carries one pull path.
// Blocks take tiles from the launch's queue (an atomic counter); a tile's member comes from a
// tile -> member table (row tiles first, then shell tiles), and a block copies a member's
// parameters to shared memory only when its member changes.  Members whose step count is reached
// are skipped.
// ---------------------------------------------------------------------------------------------
template <class L, class S, int VARIANT, bool WALLS, bool ROWS>
__global__ void __launch_bounds__(kStepThreads, StepShape<L, S, VARIANT>::kMinBlocks)
    k_step_batch(const BatchMember* __restrict__ members, const int* __restrict__ tile_member, int tile_begin,
                 int tile_end, int launch_index, int* __restrict__ counter) {
  using ST = typename S::T;
  __shared__ StepParams sp;
  __shared__ int s_tile, s_member;
  __shared__ long long s_roff[kStepThreads / 32][L::Q];  // shell tiles: each warp's row offsets
  int held = -1;  // member whose parameters sp holds (block-uniform)
  for (;;) {
    if (threadIdx.x == 0) {
      const int t = tile_begin + atomicAdd(counter, 1);
      s_tile = t;
      s_member = t < tile_end ? __ldg(&tile_member[t]) : 0;
    }
    __syncthreads();
    const int tile = s_tile;
    const int mi = s_member;
    if (tile >= tile_end) return;
    const BatchMember& m = members[mi];
    const bool active = launch_index < m.steps_left;
    if (active && mi != held) {
      const int* srcw = reinterpret_cast<const int*>(&m.p);
      int* dstw = reinterpret_cast<int*>(&sp);
      for (int k = threadIdx.x; k < (int)(sizeof(StepParams) / sizeof(int)); k += kStepThreads) dstw[k] = srcw[k];
      held = mi;
    }
    __syncthreads();
    if (active) {
      const int par = (m.parity0 + launch_index) & 1;
      const ST* sb = static_cast<const ST*>(m.buf[par]);
      ST* db = static_cast<ST*>(m.buf[par ^ 1]);
      if constexpr (ROWS) {
        const int w = (tile - m.row_tile_begin) * (kStepThreads / 32) + (threadIdx.x >> 5);
        if (w < sp.int_warps) {  // whole warps only
          Cell cl;
          bool valid, fast;
          row_cell(w, threadIdx.x & 31, sp, cl, valid, fast);
          step_cell<L, S, false, VARIANT, kPathRow, WALLS>(sb, db, sp, m.status, cl, valid, fast);
        }
      } else if (sp.general) {
        // per cell, modulo wrap (a periodic axis shorter than the stencil reach)
        const int s = (tile - m.shell_tile_begin) * kStepThreads + threadIdx.x;
        const bool valid = s < sp.shell_cells;
        const Cell cl = shell_cell(valid ? s : sp.shell_cells - 1, sp);
        step_cell<L, S, true, VARIANT, kPathEdge, WALLS>(sb, db, sp, m.status, cl, valid);
      } else {
        // four shell-row warps, as in k_step_shell_rows
        const int w = (tile - m.shell_tile_begin) * (kStepThreads / 32) + (threadIdx.x >> 5);
        if (w < sp.shell_warps) {  // whole warps only
          const int seg = w % sp.row_segs, r = w / sp.row_segs;
          Cell cl;
          shell_row(r, sp, cl.y, cl.z);
          const int x0 = seg * 32, x = x0 + (threadIdx.x & 31);
          const bool valid = x < sp.nx;
          cl.x = valid ? x : sp.nx - 1;
          cl.c = (cl.z * sp.ny + cl.y) * sp.nx + cl.x;
          const bool xfast = x0 >= sp.ix0 && min(x0 + 31, sp.nx - 1) < sp.ix0 + sp.ixn;
          long long* roff = s_roff[threadIdx.x >> 5];
          uint32_t walled[4];
          shell_row_table<L, WALLS>(roff, walled, cl, sp);
          step_cell<L, S, false, VARIANT, kPathShellTab, WALLS>(sb, db, sp, m.status, cl, valid, xfast, roff, walled);
        }
      }
    }
    __syncthreads();  // sp and s_tile are reused by the next tile
  }
}

// ---------------------------------------------------------------------------------------------
// float-float arithmetic: a value as the unevaluated sum hi + lo of two floats (|lo| <= ulp(hi)/2),
// built from the error-free transformations of Dekker and Knuth (two-sum; two-product by FMA).
// About 44 bits of significand, at float-pipe speed: GB300 runs 64 float operations for each double
// one, and a float-float operation takes 7 to 12 of them.
// ---------------------------------------------------------------------------------------------
struct FF {
  float hi, lo;
};

__device__ __forceinline__ FF ff_from(double x) {
  const float hi = (float)x;
  return FF{hi, (float)(x - (double)hi)};
}
__host__ __device__ constexpr FF ff_const(double x) { return FF{(float)x, (float)(x - (double)(float)x)}; }
__device__ __forceinline__ double ff_double(FF a) { return (double)a.hi + (double)a.lo; }

__device__ __forceinline__ FF ff_neg(FF a) { return FF{-a.hi, -a.lo}; }

// hi + lo of a + b exactly (Knuth's two-sum)
__device__ __forceinline__ FF two_sum(float a, float b) {
  const float s = __fadd_rn(a, b);
  const float bb = __fsub_rn(s, a);
  return FF{s, __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb))};
}

__device__ __forceinline__ FF fast_two_sum(float a, float b) {  // |a| >= |b|
  const float s = __fadd_rn(a, b);
  return FF{s, __fsub_rn(b, __fsub_rn(s, a))};
}

// hi + lo of a b exactly
__device__ __forceinline__ FF two_prod(float a, float b) {
  const float p = __fmul_rn(a, b);
  return FF{p, fmaf(a, b, -p)};
}

__device__ __forceinline__ FF ff_add(FF a, FF b) {
  const FF s = two_sum(a.hi, b.hi);
  return fast_two_sum(s.hi, s.lo + (a.lo + b.lo));
}
__device__ __forceinline__ FF ff_add(FF a, float b) {
  const FF s = two_sum(a.hi, b);
  return fast_two_sum(s.hi, s.lo + a.lo);
}
__device__ __forceinline__ FF ff_sub(FF a, FF b) { return ff_add(a, ff_neg(b)); }

__device__ __forceinline__ FF ff_mul(FF a, FF b) {
  const FF p = two_prod(a.hi, b.hi);
  return fast_two_sum(p.hi, p.lo + fmaf(a.hi, b.lo, a.lo * b.hi));
}
__device__ __forceinline__ FF ff_mul(FF a, float b) {
  const FF p = two_prod(a.hi, b);
  return fast_two_sum(p.hi, fmaf(a.lo, b, p.lo));
}
// a times a power of two (exact)
__device__ __forceinline__ FF ff_scale2(FF a, float k) { return FF{a.hi * k, a.lo * k}; }

// acc + m u: the product's error and the sum's error both kept
__device__ __forceinline__ FF ff_mac(FF acc, float m, float u) {
  const FF p = two_prod(m, u);
  const FF s = two_sum(acc.hi, p.hi);
  return FF{s.hi, s.lo + (acc.lo + p.lo)};
}
__device__ __forceinline__ FF ff_mac(FF acc, FF m, FF u) {
  const FF p = two_prod(m.hi, u.hi);
  const FF s = two_sum(acc.hi, p.hi);
  return FF{s.hi, s.lo + (acc.lo + fmaf(m.hi, u.lo, fmaf(m.lo, u.hi, p.lo)))};
}
__device__ __forceinline__ FF ff_mac(FF acc, float m, FF u) {
  const FF p = two_prod(m, u.hi);
  const FF s = two_sum(acc.hi, p.hi);
  return FF{s.hi, s.lo + (acc.lo + fmaf(m, u.lo, p.lo))};
}
__device__ __forceinline__ FF ff_mac(FF acc, FF m, float u) { return ff_mac(acc, u, m); }

// 1 / b and sqrt(b) by one Newton step from the float value
__device__ __forceinline__ FF ff_recip(FF b) {
  const float r = 1.f / b.hi;
  const float e = fmaf(-b.lo, r, fmaf(-b.hi, r, 1.f));
  return fast_two_sum(r, r * e);
}
__device__ __forceinline__ FF ff_sqrt(FF b) {
  const float h = sqrtf(b.hi);
  const float e = fmaf(-h, h, b.hi) + b.lo;
  return fast_two_sum(h, e * (0.5f / h));
}

// The moments of float populations (deviations d_i for half storage) for the fields readout: per
// direction pair, the sums over energies for +v and -v are first combined into their sum P and
// difference D, and the moments accumulate c P (even moments) and c D (odd moments) in float.  The
// odd moments (the velocity) then cancel within each direction pair before they are summed over
// directions, which keeps T^{0a} near float rounding of the populations (about 1e-8 of T^00; summing
// +v and -v over all directions first and subtracting at the end loses an order of magnitude more).
// T^zz is left 0; moments_ext adds it and the weights' own moments.
template <class L, bool DEV, class GetF>
__device__ __forceinline__ Mom<float> moments_pd(GetF&& getf) {
  float N0 = 0.f, Nx = 0.f, Ny = 0.f, Nz = 0.f, T00 = 0.f, T0x = 0.f, T0y = 0.f, T0z = 0.f, Txx = 0.f, Tyy = 0.f,
        Txy = 0.f, Txz = 0.f, Tyz = 0.f;
  static_for<L::NDP>([&](auto K) {
    constexpr int k = decltype(K)::value;
    constexpr int first = L::DP_FIRST[k];
    constexpr int np = L::DP_NPAIR[k];
    float S1p = 0.f, S1m = 0.f, S2p = 0.f, S2m = 0.f;
    static_for<np>([&](auto J) {
      constexpr int ip = first + 2 * decltype(J)::value;
      constexpr double wk = DEV ? L::W[ip] : 1.0;  // mirror partners share the weight
      constexpr float p0 = (float)(wk * L::P0[L::LEV[ip]]);
      constexpr float p02 = (float)(wk * L::P0[L::LEV[ip]] * L::P0[L::LEV[ip]]);
      const float fa = getf(ic<ip>{}), fb = getf(ic<ip + 1>{});
      S1p = fmaf(p0, fa, S1p);
      S1m = fmaf(p0, fb, S1m);
      S2p = fmaf(p02, fa, S2p);
      S2m = fmaf(p02, fb, S2m);
    });
    constexpr int vx = L::VX[first], vy = L::VY[first], vz = L::VZ[first];
    constexpr double ir = L::INV_R, ir2 = L::INV_R2;
    const float P1 = S1p + S1m, D1 = S1p - S1m, P2 = S2p + S2m, D2 = S2p - S2m;
    N0 += P1;
    T00 += P2;
    if constexpr (vx != 0) {
      Nx = fmaf((float)(vx * ir), D1, Nx);
      T0x = fmaf((float)(vx * ir), D2, T0x);
      Txx = fmaf((float)(vx * vx * ir2), P2, Txx);
    }
    if constexpr (vy != 0) {
      Ny = fmaf((float)(vy * ir), D1, Ny);
      T0y = fmaf((float)(vy * ir), D2, T0y);
      Tyy = fmaf((float)(vy * vy * ir2), P2, Tyy);
    }
    if constexpr (vz != 0) {
      Nz = fmaf((float)(vz * ir), D1, Nz);
      T0z = fmaf((float)(vz * ir), D2, T0z);
    }
    if constexpr (vx != 0 && vy != 0) Txy = fmaf((float)(vx * vy * ir2), P2, Txy);
    if constexpr (vx != 0 && vz != 0) Txz = fmaf((float)(vx * vz * ir2), P2, Txz);
    if constexpr (vy != 0 && vz != 0) Tyz = fmaf((float)(vy * vz * ir2), P2, Tyz);
  });
  return Mom<float>{N0, Nx, Ny, Nz, T00, T0x, T0y, T0z, Txx, Tyy, 0.f, Txy, Txz, Tyz};
}

// The float sums completed in float-float: the weights' own moments times c (deviations), and T^zz
// from the trace identity.  Without deviations every moment but T^zz is its float sum exactly.
template <bool DEV>
struct MomExt {
  using M = std::conditional_t<DEV, FF, float>;
  M N0, T00, Txx, Tyy, Txy, Txz, Tyz;
  float Nx, Ny, Nz, T0x, T0y, T0z;  // odd moments: the weights' own vanish
  FF Tzz;
};
template <class L, bool DEV>
__device__ __forceinline__ MomExt<DEV> moments_ext(const Mom<float>& m, float c) {
  MomExt<DEV> r;
  r.Nx = m.Nx, r.Ny = m.Ny, r.Nz = m.Nz, r.T0x = m.T0x, r.T0y = m.T0y, r.T0z = m.T0z;
  if constexpr (DEV) {
    using W = RestSums<L>;
    auto add = [&](double w, float v) { return ff_add(ff_mul(ff_const(w), c), v); };
    r.N0 = add(W::N0, m.N0), r.T00 = add(W::T00, m.T00), r.Txx = add(W::Txx, m.Txx), r.Tyy = add(W::Tyy, m.Tyy);
    r.Txy = add(W::Txy, m.Txy), r.Txz = add(W::Txz, m.Txz), r.Tyz = add(W::Tyz, m.Tyz);
    r.Tzz = ff_sub(r.T00, ff_add(r.Txx, r.Tyy));
  } else {
    r.N0 = m.N0, r.T00 = m.T00, r.Txx = m.Txx, r.Tyy = m.Tyy, r.Txy = m.Txy, r.Txz = m.Txz, r.Tyz = m.Tyz;
    const FF s = two_sum(m.Txx, m.Tyy);
    r.Tzz = ff_add(ff_neg(s), m.T00);
  }
  return r;
}
__device__ __forceinline__ double to_double(float x) { return (double)x; }
__device__ __forceinline__ double to_double(FF x) { return ff_double(x); }
__device__ __forceinline__ float to_float(float x) { return x; }
__device__ __forceinline__ float to_float(FF x) { return x.hi; }
template <class To, bool DEV>
__device__ __forceinline__ Mom<To> mom_of(const MomExt<DEV>& m) {
  auto t = [](auto v) -> To {
    if constexpr (std::is_same<To, double>::value) return to_double(v);
    else return to_float(v);
  };
  return Mom<To>{t(m.N0),  t(m.Nx),  t(m.Ny),  t(m.Nz),  t(m.T00), t(m.T0x), t(m.T0y),
                 t(m.T0z), t(m.Txx), t(m.Tyy), t(m.Tzz), t(m.Txy), t(m.Txz), t(m.Tyz)};
}

// One update of a converged float Landau frame against the float-float moments.  With U made a unit
// vector to float-float precision, V = T.(eta U), eps = U.V and the residual r = V - eps U (orthogonal
// to U), the shifted power update (see landau_from) is U + 3 r / (4 eps) to second order in r: one
// product with T in extended precision, and the update itself, some 1e-7 U, needs float only.  The
// second-order terms of the norm and of the Rayleigh quotient are added (d.d is minus the square of
// the update).  The same update in double took 60 % of the fields kernel at the 1/64-rate double pipe.
struct FrameFF {
  FF U0, Ux, Uy, Uz, eps, n;
  bool ok;
};
template <bool DEV>
__device__ __forceinline__ FrameFF frame_update(const MomExt<DEV>& m, const Landau<float>& lf) {
  const FF z{0.f, 0.f};
  const float x = lf.Ux, y = lf.Uy, w = lf.Uz;
  FF q = ff_mac(ff_mac(ff_mac(FF{1.f, 0.f}, x, x), y, y), w, w);
  const FF U0 = ff_sqrt(fast_two_sum(q.hi, q.lo));
  auto row = [&](auto a, auto b, auto c, auto d) {
    const FF r = ff_mac(ff_mac(ff_mac(ff_mac(z, a, U0), b, -x), c, -y), d, -w);
    return fast_two_sum(r.hi, r.lo);
  };
  const FF V0 = row(m.T00, m.T0x, m.T0y, m.T0z), Vx = row(m.T0x, m.Txx, m.Txy, m.Txz);
  const FF Vy = row(m.T0y, m.Txy, m.Tyy, m.Tyz), Vz = row(m.T0z, m.Txz, m.Tyz, m.Tzz);
  FF e = ff_mac(ff_mac(ff_mac(ff_mac(z, V0, U0), Vx, -x), Vy, -y), Vz, -w);
  e = fast_two_sum(e.hi, e.lo);
  const float k = 0.75f / e.hi;
  auto res = [&](FF V, FF u) {  // k (V - e u): V and e u agree to float rounding, so the difference is exact
    const FF p = ff_mul(e, u);
    return k * ((V.hi - p.hi) + (V.lo - p.lo));
  };
  float d0 = res(V0, U0), dx = res(Vx, FF{x, 0.f}), dy = res(Vy, FF{y, 0.f}), dz = res(Vz, FF{w, 0.f});
  const float dd = d0 * d0 - dx * dx - dy * dy - dz * dz;
  const float h = -0.5f * dd;
  FrameFF r;
  r.U0 = ff_add(U0, fmaf(h, U0.hi, d0));
  r.Ux = two_sum(x, fmaf(h, x, dx));
  r.Uy = two_sum(y, fmaf(h, y, dy));
  r.Uz = two_sum(w, fmaf(h, w, dz));
  r.eps = ff_add(e, (float)(4.0 / 3.0) * dd * e.hi);
  FF nn = ff_mac(z, m.N0, r.U0);
  nn = ff_mac(nn, -m.Nx, r.Ux);
  nn = ff_mac(nn, -m.Ny, r.Uy);
  nn = ff_mac(nn, -m.Nz, r.Uz);
  r.n = fast_two_sum(nn.hi, nn.lo);
  r.ok = r.eps.hi > 0.f && r.n.hi > 0.f && isfinite(r.eps.hi) && isfinite(r.n.hi);
  return r;
}

// Block sums of d[0..4] over kMomThreads threads into out[0..4].  The warps' five sums are reduced
// together: at each of the first three exchanges a lane keeps half of what it holds and hands its
// partner the rest, so a warp adds 8 doubles a lane instead of 25 (the same pairs in the same tree
// as a shuffle reduction of each value).
__device__ __forceinline__ void block_sums(const double (&d)[5], double* __restrict__ out) {
  __shared__ double ws[kMomThreads / 32][8];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const bool b4 = lane & 16, b3 = lane & 8, b2 = lane & 4;
  auto swap = [](double keep, double give, int o) { return keep + __shfl_xor_sync(0xffffffffu, give, o); };
  // lanes with bit 4 clear take values 0, 1, 2, the others 3, 4 (and a zero)
  const double e0 = swap(b4 ? d[3] : d[0], b4 ? d[0] : d[3], 16);
  const double e1 = swap(b4 ? d[4] : d[1], b4 ? d[1] : d[4], 16);
  const double e2 = swap(b4 ? 0.0 : d[2], b4 ? d[2] : 0.0, 16);
  // bit 3 clear: the first two of those, set: the third
  const double g0 = swap(b3 ? e2 : e0, b3 ? e0 : e2, 8);
  const double g1 = swap(b3 ? 0.0 : e1, b3 ? e1 : 0.0, 8);
  // bit 2 clear: the first, set: the second
  double h = swap(b2 ? g1 : g0, b2 ? g0 : g1, 4);
  h += __shfl_xor_sync(0xffffffffu, h, 2);
  h += __shfl_xor_sync(0xffffffffu, h, 1);
  if ((lane & 3) == 0) ws[warp][lane >> 2] = h;  // lane 0, 4, 8, 16, 20: values 0, 1, 2, 3, 4
  __syncthreads();
  if (threadIdx.x < 5) {
    const int k = threadIdx.x < 3 ? threadIdx.x : threadIdx.x + 1;
    double s = 0.0;
#pragma unroll
    for (int w = 0; w < kMomThreads / 32; ++w) s += ws[w][k];
    out[threadIdx.x] = s;
  }
}

// The double solve of a float readout, out of line like the step's (few cells take it).
static __device__ __noinline__ Landau<double> landau_readout_fp64(const Mom<double> m) { return landau<double, 200>(m); }

// ---------------------------------------------------------------------------------------------
// fields and conserved densities of one time level.  Double storage: double moments and Landau solve.
// Float storages: float moments (moments_pd), the step's Landau policy, and one update of a float
// frame in float-float (frame_update).  128^3 float: 357 us, 0.49 of the copy bandwidth, bound by the
// latency of the pulls (issue slots 44 %, 7 of 12 stalled warps on loads); 767 us with the update in
// double and every coordinate of every pull wrapped by itself.  Double: 96^3 876 us against 2563 (integer sums, corrected frame).
//   PULL = true : the pre-collision populations pulled from the previous state
//   PULL = false: the stored populations of each cell
// out.f[k][cell], k = n, eps, U0, U1, U2, U3; partial[block][5] = block sums of
// N^0, T^00, T^0x, T^0y, T^0z, in a fixed order.
// ---------------------------------------------------------------------------------------------
template <class L, class S, bool PULL, bool WALLS>
__global__ void __launch_bounds__(kMomThreads) k_fields(const typename S::T* __restrict__ src,
                                                        const __grid_constant__ StepParams p,
                                                        const FieldOut out,
                                                        double* __restrict__ partial,
                                                        int* __restrict__ status, int block0) {
  // blocks [block0, block0 + gridDim.x) of the lattice's kMomThreads-cell blocks (a launch may cover
  // a chunk of the lattice; the partial sums land in the same slots either way)
  const int blk = block0 + blockIdx.x;
  const int gid = blk * kMomThreads + threadIdx.x;
  const bool valid = gid < p.cells;
  const Cell cl = make_cell(valid ? gid : p.cells - 1, p);
  PullTab<L> tab(cl, p);
  if constexpr (PULL && WALLS) tab.find_walls(cl, p);
  auto index = [&](auto I) -> long long {
    constexpr int i = decltype(I)::value;
    if constexpr (PULL) return tab.template index<i, WALLS>(cl, p);
    else return (long long)i * p.cells + (unsigned)cl.c;
  };
  double d[5];
  bool ok, finite;
  double n, eps, U0, Ux, Uy, Uz;
  auto put = [&](const Landau<double>& lw) {
    ok = lw.ok;
    n = lw.n, eps = lw.eps, U0 = lw.U0, Ux = lw.Ux, Uy = lw.Uy, Uz = lw.Uz;
  };
  auto all_finite = [](const auto& m) {
    return isfinite(m.N0) && isfinite(m.Nx) && isfinite(m.Ny) && isfinite(m.Nz) && isfinite(m.T00) &&
           isfinite(m.T0x) && isfinite(m.T0y) && isfinite(m.T0z) && isfinite(m.Txx) && isfinite(m.Tyy) &&
           isfinite(m.Tzz) && isfinite(m.Txy) && isfinite(m.Txz) && isfinite(m.Tyz);
  };
  if constexpr (std::is_same<typename S::A, double>::value) {
    const Mom<double> m = moments_fixed<L>([&](auto I) -> double { return src[index(I)]; });
    put(landau_f64<200>(m));
    finite = all_finite(m);
    d[0] = m.N0, d[1] = m.T00, d[2] = m.T0x, d[3] = m.T0y, d[4] = m.T0z;
  } else {
    constexpr bool DEV = std::is_same<S, StoreF16Dev>::value;
    const MomExt<DEV> m = moments_ext<L, DEV>(
        moments_pd<L, DEV>([&](auto I) -> float {
          constexpr int i = decltype(I)::value;
          if constexpr (DEV) return S::template load_dev<L, i>(src + index(I), p);
          else return __ldcg(src + index(I));
        }),
        p.half_nref);
    // the step's policy: float solve, double for cells above gamma_thr, for unconverged float
    // solves, or everywhere with landau_fp64
    const Mom<float> mf = mom_of<float>(m);
    finite = all_finite(mf);
    const float NN = minkowski(mf.N0, mf.Nx, mf.Ny, mf.Nz, mf.N0, mf.Nx, mf.Ny, mf.Nz);
    bool dbl = p.landau_fp64 || mf.N0 * mf.N0 > p.gamma_thr2 * NN;
    if (!dbl) {
      const Landau<float> lf = landau<float, 8>(mf);
      dbl = !(lf.ok && lf.conv);
      if (!dbl) {
        const FrameFF r = frame_update<DEV>(m, lf);
        ok = r.ok;
        n = ff_double(r.n), eps = ff_double(r.eps);
        U0 = ff_double(r.U0), Ux = ff_double(r.Ux), Uy = ff_double(r.Uy), Uz = ff_double(r.Uz);
      }
    }
    if (dbl) put(landau_readout_fp64(mom_of<double>(m)));
    d[0] = to_double(m.N0), d[1] = to_double(m.T00), d[2] = m.T0x, d[3] = m.T0y, d[4] = m.T0z;
  }
  if (valid) {
    const double nan = __longlong_as_double(0x7ff8000000000000ll);
    out.f[0][cl.c] = ok ? n : nan;
    out.f[1][cl.c] = ok ? eps : nan;
    out.f[2][cl.c] = ok ? U0 : nan;
    out.f[3][cl.c] = ok ? Ux : nan;
    out.f[4][cl.c] = ok ? Uy : nan;
    out.f[5][cl.c] = ok ? Uz : nan;
    // non-finite populations show as non-finite moments; any other cell without a frame is a
    // Landau failure
    if (!finite) atomicAdd(&status[kStatusNan], 1);
    else if (!ok) atomicAdd(&status[kStatusNonconv], 1);
  } else {
#pragma unroll
    for (int k = 0; k < 5; ++k) d[k] = 0.0;
  }
  block_sums(d, partial + (long long)blk * 5);
}

// Second pass of the conserved-density sums, value blockIdx.x of the five: one block adds the
// per-block partials in a fixed order (thread t takes blocks t, t + 256, ...; then a shuffle and
// shared-memory tree), so the totals are bitwise reproducible.  The adds of a thread are a chain; its
// loads are not, so 16 are kept in flight.
static __global__ void __launch_bounds__(kReduceThreads) k_reduce_partials(const double* __restrict__ partial,
                                                                           int nblocks, double* __restrict__ totals) {
  __shared__ double ws[kReduceThreads / 32];
  const int k = blockIdx.x;
  double d = 0.0;
#pragma unroll 16
  for (int b = threadIdx.x; b < nblocks; b += kReduceThreads) d += partial[(long long)b * 5 + k];
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) d += __shfl_down_sync(0xffffffffu, d, o);
  if ((threadIdx.x & 31) == 0) ws[threadIdx.x >> 5] = d;
  __syncthreads();
  if (threadIdx.x == 0) {
    double s = 0.0;
#pragma unroll
    for (int w = 0; w < kReduceThreads / 32; ++w) s += ws[w];
    totals[k] = s;
  }
}

// ---------------------------------------------------------------------------------------------
// initial state f_i = f_i^eq(n, T, u), and population format conversion
// ---------------------------------------------------------------------------------------------
// The equilibrium's coefficients per energy level (eq_coef and level_coef) in float-float.
template <class L>
__device__ __forceinline__ LevCoef<L, FF> level_coef_ff(FF n, FF T, FF x) {
  LevCoef<L, FF> r;
  const FF x2 = ff_mul(x, x), T2 = ff_mul(T, T);
  const FF nT = ff_mul(n, ff_recip(T));
  auto times = [](FF a, float k) { return ff_mul(a, k); };
  if constexpr (L::ORDER == 3) {
    const FF pref = ff_mul(ff_const(1.0 / 12.0), nT);
    const FF nTh = ff_scale2(nT, 0.5f), nTq = ff_scale2(nT, 0.25f);  // 6 pref, 3 pref
    const FF Tn = ff_mul(nTh, T);                                     // 6 pref T
    // c00 = -6 pref (x2 (8x + 4) + (4x - 2) + T2 (1 - 4x)), ...
    const FF x4 = ff_scale2(x, 4.f), x6 = times(x, 6.f);
    FF c00 = ff_add(ff_mul(x2, ff_add(ff_scale2(x, 8.f), 4.f)), ff_add(x4, -2.f));
    c00 = ff_neg(ff_mul(nTh, ff_add(c00, ff_mul(T2, ff_add(ff_neg(x4), 1.f)))));
    FF c10 = ff_add(ff_mul(x2, ff_add(ff_scale2(x6, 2.f), 8.f)), ff_add(times(x, 5.f), -1.f));
    c10 = ff_mul(nTh, ff_add(c10, ff_mul(T2, ff_add(ff_neg(x6), 1.f))));
    const FF c01 = ff_mul(Tn, ff_sub(ff_add(times(x2, 12.f), 3.f), ff_scale2(T2, 2.f)));
    FF c20 = ff_add(ff_mul(x, ff_add(x6, 3.f)), 2.f);
    c20 = ff_neg(ff_mul(ff_mul(nTq, x), ff_sub(c20, ff_scale2(T2, 2.f))));
    const FF c11 = ff_neg(ff_mul(Tn, ff_sub(ff_add(ff_mul(x, ff_add(x6, 1.f)), 1.f), T2)));
    const FF c02 = ff_neg(ff_mul(ff_mul(nTq, T2), ff_add(x6, -1.f)));
    const FF px = ff_mul(pref, x), px2 = ff_mul(px, x), pT2 = ff_mul(pref, T2);
    const FF a3 = ff_mul(px2, x), b3 = times(ff_mul(px2, T), 3.f), c3 = times(ff_mul(px, T2), 3.f), d3 = ff_mul(pT2, T);
    static_for<L::NLEV>([&](auto K) {
      constexpr int l = decltype(K)::value;
      constexpr double pd = L::P0[l];
      const FF p = ff_const(pd), p2 = ff_const(pd * pd), p3 = ff_const(pd * pd * pd);
      r.a[l] = ff_add(ff_add(c00, ff_mul(p, c10)), ff_add(ff_mul(p2, c20), ff_mul(p3, a3)));
      r.b[l] = ff_add(ff_mul(p, c01), ff_add(ff_mul(p2, c11), ff_mul(p3, b3)));
      r.c[l] = ff_add(ff_mul(p2, c02), ff_mul(p3, c3));
      r.d[l] = ff_mul(p3, d3);
    });
  } else {
    const FF pref = ff_scale2(nT, 0.25f), nTh = ff_scale2(nT, 0.5f), Tn = ff_mul(nTh, T);  // pref, 2 pref, 2 pref T
    const FF x4 = ff_scale2(x, 4.f);
    const FF c00 = ff_mul(nTh, ff_sub(ff_add(ff_scale2(x2, 4.f), 2.f), T2));
    const FF c10 = ff_neg(ff_mul(nTh, ff_sub(ff_add(ff_mul(x, ff_add(x4, 1.f)), 1.f), T2)));
    const FF c01 = ff_neg(ff_mul(Tn, ff_add(x4, -1.f)));
    const FF px = ff_mul(pref, x), a2 = ff_mul(px, x), b2 = ff_scale2(ff_mul(px, T), 2.f), c2 = ff_mul(pref, T2);
    static_for<L::NLEV>([&](auto K) {
      constexpr int l = decltype(K)::value;
      constexpr double pd = L::P0[l];
      const FF p = ff_const(pd), p2 = ff_const(pd * pd);
      r.a[l] = ff_add(c00, ff_add(ff_mul(p, c10), ff_mul(p2, a2)));
      r.b[l] = ff_add(ff_mul(p, c01), ff_mul(p2, b2));
      r.c[l] = ff_mul(p2, c2);
      r.d[l] = FF{0.f, 0.f};
    });
  }
  return r;
}

// The same from double coefficients, for cells whose powers of T or n / T leave the range of a float on the
// way to coefficients that do not (out of line: few cells have such a state).
template <class L>
static __device__ __noinline__ LevCoef<L, FF> level_coef_wide(double n, double T, double g) {
  const LevCoef<L, double> d = level_coef<L, double>(eq_coef<L::ORDER, double>(n, T, g));
  LevCoef<L, FF> r;
  static_for<L::NLEV>([&](auto K) {
    constexpr int l = decltype(K)::value;
    r.a[l] = ff_from(d.a[l]), r.b[l] = ff_from(d.b[l]), r.c[l] = ff_from(d.c[l]), r.d[l] = ff_from(d.d[l]);
  });
  return r;
}

template <class L, class S>
__global__ void __launch_bounds__(128) k_init(const double* __restrict__ n, const double* __restrict__ Tf,
                                              const double* __restrict__ u, typename S::T* __restrict__ dst,
                                              const __grid_constant__ StepParams p, int* __restrict__ status,
                                              int c0, int c1) {
  // cells [c0, c1) (a launch may cover a chunk of the lattice)
  const int c = c0 + blockIdx.x * blockDim.x + threadIdx.x;
  if (c >= c1) return;
  const long long cells = p.cells;
  const double ux = u[c], uy = u[cells + c], uz = u[2 * cells + c];
  const double u2 = ux * ux + uy * uy + uz * uz;
  const double nn = n[c], T = Tf[c];
  if (!(u2 < 1.0) || !(T > 0.0) || !(nn > 0.0)) {
    atomicAdd(&status[kStatusBadInit], 1);
    return;
  }
  const double g = rsqrt(1.0 - u2);
  const double Ux = g * ux, Uy = g * uy, Uz = g * uz;
  if constexpr (std::is_same<typename S::A, double>::value) {
    // the equilibrium per energy level (see level_coef), coefficients in double
    const LevCoef<L, double> ed = level_coef<L, double>(eq_coef<L::ORDER, double>(nn, T, g));
    static_for<L::NDP>([&](auto K) {
      constexpr int k = decltype(K)::value;
      constexpr int first = L::DP_FIRST[k];
      constexpr int np = L::DP_NPAIR[k];
      constexpr int vx = L::VX[first], vy = L::VY[first], vz = L::VZ[first];
      const double t = (vx * Ux + vy * Uy + vz * Uz) * L::INV_R;
      static_for<np>([&](auto J) {
        constexpr int ip = first + 2 * decltype(J)::value;
        constexpr int l = L::LEV[ip];
        constexpr double w = L::W[ip];
        const double Ep = fma(t, fma(t, fma(t, ed.d[l], ed.c[l]), ed.b[l]), ed.a[l]);
        const double Em = fma(-t, fma(-t, fma(-t, ed.d[l], ed.c[l]), ed.b[l]), ed.a[l]);
        S::template store<L, ip>(dst + (long long)ip * cells + c, w * Ep, p);
        S::template store<L, ip + 1>(dst + (long long)(ip + 1) * cells + c, w * Em, p);
      });
    });
  } else {
    // Float storage rounds every population to float.  The cubic in t cancels strongly at the high
    // energy levels (terms up to ~200 times the value at p0 = 10.95, |u| = 0.6), so those levels
    // (p0 > 4) are evaluated with the rounding errors of their products and sums carried along
    // (compensated; the even part a + c t^2 and the odd part t (b + d t^2) shared by +v and -v), the
    // others in float: every population ends within float rounding of the double evaluation.  The
    // inputs are normalised in double (some 40 operations a cell, which the 1/64-rate pipe does
    // beside the float work: 40 % busy); the coefficients, 110 double operations a cell and the bound
    // of this kernel while they were double, are float-float.  128^3 float: 364 us, 876 before; bound
    // by float issue (4660 warp instructions per 32 cells, issue slots 65 %, FMA pipe 62 % used).
    // Their intermediate powers go up to T^3 g^3 and down to T / n: in float up to 1e9 and from 1e-9 on,
    // and with room below for the low parts (1e-25 of 1e-38).
    const FF nf = ff_from(nn), Tf = ff_from(T), xf = ff_from(fma(T, g, -1.0));
    LevCoef<L, FF> e;
    if (Tf.hi > 1e-9f && xf.hi < 1e9f && nf.hi > 1e-25f && nf.hi < 1e25f) e = level_coef_ff<L>(nf, Tf, xf);
    else e = level_coef_wide<L>(nn, T, g);
    // U / R times 1 .. 6 per axis: t = v.U / R is then a sum of at most three of them
    FF m[3][7];
    const double Ua[3] = {Ux * L::INV_R, Uy * L::INV_R, Uz * L::INV_R};
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      m[a][1] = ff_from(Ua[a]);
      m[a][3] = ff_mul(m[a][1], 3.f);
      m[a][5] = ff_mul(m[a][1], 5.f);
      m[a][2] = ff_scale2(m[a][1], 2.f);
      m[a][4] = ff_scale2(m[a][1], 4.f);
      m[a][6] = ff_scale2(m[a][3], 2.f);
    }
    static_for<L::NDP>([&](auto K) {
      constexpr int k = decltype(K)::value;
      constexpr int first = L::DP_FIRST[k];
      constexpr int np = L::DP_NPAIR[k];
      constexpr int v[3] = {L::VX[first], L::VY[first], L::VZ[first]};
      static_assert(L::VMAX_X <= 6 && L::VMAX_Y <= 6 && L::VMAX_Z <= 6, "multiples of U up to 6");
      FF t{0.f, 0.f};
      static_for<3>([&](auto A) {
        constexpr int a = decltype(A)::value, va = v[a] < 0 ? -v[a] : v[a];
        if constexpr (va != 0) {
          const FF x = v[a] < 0 ? ff_neg(m[a][va]) : m[a][va];
          const FF s = two_sum(t.hi, x.hi);
          t = FF{s.hi, s.lo + (t.lo + x.lo)};
        }
      });
      const float t2h = __fmul_rn(t.hi, t.hi);
      const float t2l = fmaf(2.f * t.hi, t.lo, fmaf(t.hi, t.hi, -t2h));
      static_for<np>([&](auto J) {
        constexpr int ip = first + 2 * decltype(J)::value;
        constexpr int l = L::LEV[ip];
        constexpr float w = (float)L::W[ip];
        float Ep, Em;
        if constexpr (L::P0[l] > 4.0) {
          auto lin = [&](FF c0, FF c1) {  // c0 + c1 t^2
            const FF q = two_prod(c1.hi, t2h);
            const FF s = two_sum(c0.hi, q.hi);
            return FF{s.hi, s.lo + fmaf(c1.hi, t2l, fmaf(c1.lo, t2h, c0.lo + q.lo))};
          };
          const FF even = lin(e.a[l], e.c[l]);
          FF b = e.b[l];
          if constexpr (L::ORDER == 3) b = lin(e.b[l], e.d[l]);
          FF odd = two_prod(b.hi, t.hi);
          odd.lo += fmaf(b.hi, t.lo, b.lo * t.hi);
          const FF sp = two_sum(even.hi, odd.hi), sm = two_sum(even.hi, -odd.hi);
          Ep = sp.hi + (sp.lo + (even.lo + odd.lo));
          Em = sm.hi + (sm.lo + (even.lo - odd.lo));
        } else {
          const float tf = t.hi + t.lo;
          Ep = fmaf(tf, fmaf(tf, fmaf(tf, e.d[l].hi, e.c[l].hi), e.b[l].hi), e.a[l].hi);
          Em = fmaf(-tf, fmaf(-tf, fmaf(-tf, e.d[l].hi, e.c[l].hi), e.b[l].hi), e.a[l].hi);
        }
        S::template store<L, ip>(dst + (long long)ip * cells + c, w * Ep, p);
        S::template store<L, ip + 1>(dst + (long long)(ip + 1) * cells + c, w * Em, p);
      });
    });
  }
}

// double[q][cells] <-> half deviations, for populations [i0, i1) (in-range cells only)
template <class L, class S, bool TO_F64>
__global__ void __launch_bounds__(128) k_convert(typename S::T* __restrict__ pop, double* __restrict__ dbl,
                                                 long long dbl_plane_offset, int i0, int i1,
                                                 const __grid_constant__ StepParams p) {
  const int c = blockIdx.x * blockDim.x + threadIdx.x;
  if (c >= p.cells) return;
  const long long cells = p.cells;
  static_for<L::Q>([&](auto I) {
    constexpr int i = decltype(I)::value;
    if (i < i0 || i >= i1) return;
    const long long di = (long long)(i - i0) * cells + c + dbl_plane_offset;
    if constexpr (TO_F64) dbl[di] = S::template to_f64<L, i>(pop[(long long)i * cells + c], p);
    else pop[(long long)i * cells + c] = S::template from_f64<L, i>(dbl[di], p);
  });
}

// The same for float and double storage, whose conversion does not depend on the population: n
// consecutive elements, four a thread, in 16-byte loads and stores where both arrays are aligned for
// them (the library's buffers are; a plane of a host transfer or the caller's pointer need not be).
// 96 x 80 x 112 float, q = 128: 217 us out and 186 in; 271 and 255 with a cell per thread.
constexpr int kConvertThreads = 256;
template <class T, bool TO_F64>
__global__ void __launch_bounds__(kConvertThreads) k_convert_flat(T* __restrict__ pop, double* __restrict__ dbl,
                                                                  long long n) {
  const long long e = ((long long)blockIdx.x * kConvertThreads + threadIdx.x) * 4;
  if (e >= n) return;
  if (e + 4 <= n && ((reinterpret_cast<uintptr_t>(pop) | reinterpret_cast<uintptr_t>(dbl)) & 15) == 0) {
    using V = std::conditional_t<sizeof(T) == 4, float4, double2>;
    union {
      V v[sizeof(T) / 4];
      T x[4];
    } a;
    union {
      double2 v[2];
      double x[4];
    } b;
    if constexpr (TO_F64) {
#pragma unroll
      for (int k = 0; k < (int)sizeof(T) / 4; ++k) a.v[k] = reinterpret_cast<const V*>(pop + e)[k];
#pragma unroll
      for (int k = 0; k < 4; ++k) b.x[k] = (double)a.x[k];
      reinterpret_cast<double2*>(dbl + e)[0] = b.v[0];
      reinterpret_cast<double2*>(dbl + e)[1] = b.v[1];
    } else {
      b.v[0] = reinterpret_cast<const double2*>(dbl + e)[0];
      b.v[1] = reinterpret_cast<const double2*>(dbl + e)[1];
#pragma unroll
      for (int k = 0; k < 4; ++k) a.x[k] = (T)b.x[k];
#pragma unroll
      for (int k = 0; k < (int)sizeof(T) / 4; ++k) reinterpret_cast<V*>(pop + e)[k] = a.v[k];
    }
  } else {
    for (int k = 0; k < 4 && e + k < n; ++k) {
      if constexpr (TO_F64) dbl[e + k] = (double)pop[e + k];
      else pop[e + k] = (T)dbl[e + k];
    }
  }
}

}  // namespace rlb
