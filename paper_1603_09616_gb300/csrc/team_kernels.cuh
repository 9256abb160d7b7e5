// The persistent kernels: teams pull panels from a device counter and run one
// of the two panel solvers (panel_real.cuh, panel.cuh).
#pragma once
#include "panel.cuh"
#include "panel_real.cuh"

namespace gbk {

// The shared state and the panel solver of one of the two recurrences.
template <bool MIX, bool REAL>
struct Team;
template <bool MIX>
struct Team<MIX, false> {
  SeedSmem sm;
  PanelSmemExtra sx;
  __device__ __forceinline__ void solve(const Args& a, char* ws, char* dyn) { solve_panel<MIX>(a, sm, sx, ws, dyn); }
};
template <bool MIX>
struct Team<MIX, true> {
  RealSmem sm;
  __device__ __forceinline__ void solve(const Args& a, char* ws, char* dyn) { solve_panel_real<MIX>(a, sm, ws, dyn); }
};

// 64 registers a thread either way: two teams of TPB threads per SM, or one of TPB_WIDE
template <bool MIX, bool REAL>
constexpr int kMaxThreads = MIX && REAL ? TPB_WIDE : TPB;
template <bool MIX, bool REAL>
constexpr int kMinTeams = MIX && REAL ? MIN_TEAMS_PER_SM / 2 : MIN_TEAMS_PER_SM;

template <bool MIX, bool REAL>
__global__ void __launch_bounds__(kMaxThreads<MIX, REAL>, kMinTeams<MIX, REAL>) team_kernel(const __grid_constant__ Args a) {
  __shared__ Team<MIX, REAL> team;
  auto& sm = team.sm;
  extern __shared__ __align__(16) char dyn_smem[];
  char* ws = a.team_ws + (size_t)blockIdx.x * a.team_bytes;
  team_init(sm, dyn_smem);
  if (a.full_hist) {  // verification: one panel per team, panel = team
    if (threadIdx.x == 0) sm.panel = blockIdx.x;
    __syncthreads();
    if (sm.panel < a.npanels) team.solve(a, ws, dyn_smem);
    return;
  }
  for (;;) {
    if (threadIdx.x == 0) sm.panel = atomicAdd(a.panel_counter, 1);
    __syncthreads();
    if (sm.panel >= a.npanels) return;
    team.solve(a, ws, dyn_smem);
    __syncthreads();
  }
}

// Batched form: many independent systems (each with its own matrix, shifts,
// columns and outputs) in one persistent launch.  Work items are (system,
// panel) pairs numbered through panel_prefix (the host orders the systems,
// largest first); a team copies the item's system descriptor into shared
// memory and runs the same panel solver.  The team workspace is laid out for
// the largest system.
template <bool MIX, bool REAL>
__global__ void __launch_bounds__(kMaxThreads<MIX, REAL>, kMinTeams<MIX, REAL>)
    team_kernel_batched(const Args* __restrict__ sys, const int* __restrict__ panel_prefix, int nsys,
                        int* __restrict__ counter, char* team_ws, size_t team_bytes) {
  __shared__ Team<MIX, REAL> team;
  auto& sm = team.sm;
  __shared__ Args sa;
  __shared__ int s_sys;
  extern __shared__ __align__(16) char dyn_smem[];
  char* ws = team_ws + (size_t)blockIdx.x * team_bytes;
  team_init(sm, dyn_smem);
  const int total = panel_prefix[nsys];
  for (;;) {
    if (threadIdx.x == 0) {
      const int item = atomicAdd(counter, 1);
      int lo = 0;
      if (item < total) {
        int hi = nsys;  // panel_prefix[lo] <= item < panel_prefix[hi]
        while (hi - lo > 1) {
          const int mid = (lo + hi) >> 1;
          if (panel_prefix[mid] <= item) lo = mid;
          else hi = mid;
        }
      }
      s_sys = item < total ? lo : -1;
      sm.panel = item < total ? item - panel_prefix[lo] : 0;
    }
    __syncthreads();
    if (s_sys < 0) return;
    const unsigned* src = reinterpret_cast<const unsigned*>(sys + s_sys);
    unsigned* dst = reinterpret_cast<unsigned*>(&sa);
    for (int i = threadIdx.x; i < (int)(sizeof(Args) / sizeof(unsigned)); i += tpb()) dst[i] = src[i];
    __syncthreads();
    team.solve(sa, ws, dyn_smem);
    __syncthreads();
  }
}

}  // namespace gbk
