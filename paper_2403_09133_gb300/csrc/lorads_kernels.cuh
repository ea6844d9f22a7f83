// Kernel entry points of the solver and of the operator calls, instantiated per element
// type by lorads_f64.cu / lorads_f32.cu.
#pragma once
#include "lorads_geometry.h"
#include "lorads_solver.cuh"

namespace lorads {

// one CTA per problem; CTAs take problems from a queue (batches), or a single problem
template <typename T, int SUB>
__global__ void __launch_bounds__(BLOCK_THREADS_MAX, 1)
solve_block_kernel(const SolverArgs<T>* args, int count, int* queue) {
  __shared__ double red[RED_ROWS * MAXRED];
  __shared__ SolverArgs<T> sa;
  __shared__ int inst;
  for (;;) {
    if (threadIdx.x == 0) inst = atomicAdd(queue, 1);
    __syncthreads();
    const int i = inst;
    if (i >= count) return;
    if (threadIdx.x == 0) sa = args[i];
    __syncthreads();
    BlockScope sc{red};
    run_solver<T, SUB>(sa, sc);
    __syncthreads();
  }
}

// one problem over the whole grid (cooperative launch: all CTAs co-resident)
template <typename T, int SUB>
__global__ void __launch_bounds__(GRID_THREADS_MAX, 1)
solve_grid_kernel(const SolverArgs<T>* args, GridCtl* ctl, Slot* slots, int reps,
                  long long spin) {
  __shared__ double red[RED_ROWS * MAXRED];
  __shared__ SolverArgs<T> sa;
  if (threadIdx.x == 0) sa = *args;
  GridScope sc{red, ctl, slots, reps, spin, 0, (int)gridDim.x};
  sc.init();
  run_solver<T, SUB>(sa, sc);
}

// batches with several CTAs per problem: CTAs [g * group, (g + 1) * group) form group g,
// which takes problems from the queue (largest first) and solves each with a scope spanning
// the group (ctls[g] and its share of the slots are its barrier, picks[g] the index its leader
// fetched).  The launch is
// cooperative, so every CTA of a group is resident and the group's bounded barriers never
// wait on a CTA that has not started.
template <typename T, int SUB>
__global__ void __launch_bounds__(BLOCK_THREADS_MAX, 1)
solve_group_kernel(const SolverArgs<T>* args, int count, int* queue, GridCtl* ctls,
                   Slot* slots, int* picks, int group, long long spin) {
  __shared__ double red[RED_ROWS * MAXRED];
  __shared__ SolverArgs<T> sa;
  const int g = blockIdx.x / group;
  Slot* mine = slots + (size_t)g * group * (SLOT_DOUBLES / 2);
  GroupScope sc{{red, ctls + g, mine, 1, spin, g * group, group}};
  sc.init();
  for (;;) {
    if (sc.is_leader()) picks[g] = atomicAdd(queue, 1);
    if (!sc.sync()) return;
    const int i = __ldcg(picks + g);
    if (i >= count) return;
    if (threadIdx.x == 0) sa = args[i];
    __syncthreads();
    run_solver<T, SUB>(sa, sc);
    __syncthreads();
  }
}

// ---- operators on caller-owned device arrays ----
template <typename T, bool MULTI>
__global__ void op_sddmm_kernel(DevProblem P, int ld, const T* U, const T* V, double* q) {
  const Team t = make_team(ld, blockIdx.x * blockDim.x + threadIdx.x, gridDim.x * blockDim.x);
  for (TeamRows rows(t, P.m); rows.more(); rows.next()) {
    const double v = MULTI ? sddmm_con_multi<T>(P, U, V, ld, rows.j, rows.t)
                           : sddmm_con<T>(P, U, V, ld, rows.j, rows.t);
    if (rows.t.lead) q[rows.j] = v;
  }
}

// Diagonal constraints: one team per row, H of C's entries a round, their rows in flight together.  A
// kernel of its own: beside the form below, which took 72 registers, 2^20 rows of r = 20 took 161 us (FP32),
// here 89.  Few rows wait for their loads and take eight entries a round, many fill the SMs at four.
template <typename T, int H>
__global__ void __launch_bounds__(256, H == 8 ? 2 : 5)
op_spmm_diag_kernel(DevProblem P, int ld, const double* w, double gamma, const T* V, T* out) {
  const Team t = make_team(ld, blockIdx.x * blockDim.x + threadIdx.x, gridDim.x * blockDim.x);
  const T *ra = rowa<T>(P), *cv = cval<T>(P);
  const T g = (T)gamma;
  for (int j = t.id; j < P.n; j += t.count) {
    // the row's own terms from the per-row arrays, asked for before C's entries: through A's rows they
    // wait for four loads in a row after those
    const int con = P.row_con[j];
    const double wj = con >= 0 ? w[con] : 0.0;
    const T a = ra[j];
    Frag<T> Vj, o;
    frag_load(Vj, V, j, ld, t);
    frag_zero(o);
    const int q1 = P.C_rp[j + 1];
    for (int q = P.C_rp[j]; q < q1; q += H) {
      Frag<T> W[H];
      T c[H];
#pragma unroll
      for (int u = 0; u < H; ++u) {
        // an entry past the row's end is neither read nor added
        const bool on = q + u < q1;
        Team tu = t;
        tu.nc = on ? t.nc : 0;
        c[u] = on ? cv[q + u] : T(0);
        frag_load(W[u], V, on ? P.C_col[q + u] : j, ld, tu);
      }
#pragma unroll
      for (int u = 0; u < H; ++u)
        if (q + u < q1) frag_axpy(o, -c[u], W[u]);
    }
    if (con >= 0) frag_axpy(o, (T)(wj * (double)a), Vj);
    if (g != T(0)) frag_axpy(o, g, Vj);
    frag_store(o, out, j, ld, t);
  }
}

// FP32 with the warp's weights: two rows in flight per sub-team (H = 2) leave 48 registers, five CTAs per SM,
// four take 72, three CTAs; four where the rows do not fill the five (r = 20, 200 entries a row, two / four:
// n = 10,000 34.4 / 39.1 us, n = 6,400 31.0 / 26.8) and sub-teams have four of 32 entries
template <typename T, bool OWN, int H>
__global__ void op_spmm_kernel(DevProblem P, int ld, const double* w, double gamma, const T* V,
                               T* out) {
  const WarpRow wr =
      make_warp_row(ld, blockIdx.x * blockDim.x + threadIdx.x, gridDim.x * blockDim.x);
  for (int j = wr.warp; j < P.n; j += wr.nwarps) {
    Frag<T> o;
    spmm_row_warp<T, OWN, H>(P, V, ld, j, w, nullptr, 0.0, 1.0, 0.0, (T)gamma, wr, o);
    if (wr.sub == 0) frag_store(o, out, j, ld, wr.st);
  }
}

// Diagonal constraints: a pass over P, V and the result, bound by HBM.  A kernel of its own: with
// the many-entries form in one kernel it took that form's 72 registers, half the warps.
template <typename T>
__global__ void __launch_bounds__(256, 5)
op_hessian_diag_kernel(DevProblem P, int ld, T rho, T gamma, const T* V, const T* Pm, T* out) {
  const Team t = make_team(ld, blockIdx.x * blockDim.x + threadIdx.x, gridDim.x * blockDim.x);
  const T* ra = rowa<T>(P);
  for (TeamRows rows(t, P.n); rows.more(); rows.next()) {
    Frag<T> Pj, Vj, H;
    frag_load(Pj, Pm, rows.j, ld, rows.t);
    frag_load(Vj, V, rows.j, ld, rows.t);
    hessian_row<T>(ra[rows.j], Vj, Pj, rho, gamma, rows.t, H);
    frag_store(H, out, rows.j, ld, rows.t);
  }
}

// H: entries of a round (hessian_row_warp)
template <typename T, int H>
__global__ void __launch_bounds__(256) op_hessian_kernel(DevProblem P, int ld, T rho, T gamma,
                                                         const T* V, const T* Pm, T* out) {
  const WarpRow wr =
      make_warp_row(ld, blockIdx.x * blockDim.x + threadIdx.x, gridDim.x * blockDim.x);
  for (int j = wr.warp; j < P.n; j += wr.nwarps) {
    Frag<T> Pj, Hj;
    frag_load(Pj, Pm, j, ld, wr.st);
    hessian_row_warp<T, H>(P, V, Pm, ld, j, Pj, rho, gamma, wr, Hj);
    if (wr.sub == 0) frag_store(Hj, out, j, ld, wr.st);
  }
}

// ---- FP64 operators.  FP64 issues one warp instruction per SM every 16 clocks whatever its lanes
// do (1/64 of the FP32 rate), so these kernels are bound by the FP64 instructions they issue, and
// the layout keeps those few: a row of ld doubles is ld / 2 units of 16 bytes, dealt to G lanes (lane
// l: units l, l + G, ...), N <= 8 units per lane (unit_lanes).  The
// solver's layout (4-element chunks, two per lane) leaves a third of the lanes of a ld = 20 row
// without elements in instructions that are issued all the same.
struct UnitRow {
  int G, lane, id, count, units;   // id, count: teams of the grid
};
__device__ inline UnitRow make_unit_row(int ld, int G) {
  UnitRow t;
  const int tid = blockIdx.x * blockDim.x + threadIdx.x;
  t.G = G;
  t.lane = tid & (G - 1);
  t.id = tid / G;
  t.count = gridDim.x * blockDim.x / G;
  t.units = ld / 2;
  return t;
}
__device__ __forceinline__ double2 unit_at(const double* row, int u, int units) {
  return u < units ? *reinterpret_cast<const double2*>(row + 2 * u) : make_double2(0.0, 0.0);
}
__device__ __forceinline__ double team_sum64(double x, int G) {
  for (int off = G >> 1; off > 0; off >>= 1) x += __shfl_xor_sync(0xffffffffu, x, off);
  return x;
}

// <A_i, U V^T>: one team per constraint.  MULTI: constraints of several entries, in as many rounds as
// the longest of the warp's teams has, a team without an entry left empty-handed (see
// sddmm_con_multi; the trace of n = 3,000, r = 9: 2,158 us with repeated entries, 1,671 so)
template <int N, bool MULTI>
__global__ void __launch_bounds__(256) op_sddmm_f64_kernel(DevProblem P, int ld, int G,
                                                           const double* U, const double* V,
                                                           double* q) {
  const UnitRow t = make_unit_row(ld, G);
  const int sub = (threadIdx.x & 31) / G;
  for (int i0 = t.id - sub; i0 < P.m; i0 += t.count) {
    const bool live = i0 + sub < P.m;
    const int i = live ? i0 + sub : P.m - 1;
    // (without the loop of MULTI the compiler keeps fewer loads in flight: 10^6 one-entry constraints,
    // r = 20, 88 us against 85)
    const int e0 = P.con_ptr[i], cnt = live ? P.con_ptr[i + 1] - e0 : 0;
    const int rounds = P.a_multi ? __reduce_max_sync(0xffffffffu, cnt) : 1;
    double s = 0.0;
    for (int k = 0; k < rounds; ++k) {
      const bool on = k < cnt;
      const int e = on ? e0 + k : e0, c = P.con_c[e], r = !MULTI || on ? P.con_r[e] : c;
      const double a = P.con_a[e];
      const int units = !MULTI || on ? t.units : 0;
      const double* Ur = U + (size_t)r * ld;
      const double* Vc = V + (size_t)c * ld;
      const double* Uc = U + (size_t)c * ld;
      const double* Vr = V + (size_t)r * ld;
      double x = 0.0, y = 0.0;
#pragma unroll
      for (int u = 0; u < N; ++u) {
        const double2 p = unit_at(Ur, t.lane + G * u, units);
        const double2 v = unit_at(Vc, t.lane + G * u, units);
        x = fma(p.x, v.x, x);
        y = fma(p.y, v.y, y);
      }
      if (r != c) {
#pragma unroll
        for (int u = 0; u < N; ++u) {
          const double2 p = unit_at(Uc, t.lane + G * u, units);
          const double2 v = unit_at(Vr, t.lane + G * u, units);
          x = fma(p.x, v.x, x);
          y = fma(p.y, v.y, y);
        }
      }
      __syncwarp();
      x = a * team_sum64(x + y, G);
      if (on) s += x;
    }
    if (live && t.lane == 0) q[i] = s;
  }
}

// (A^T(w) - C) V + gamma V with diagonal constraints: one team per row, C's entries two at a time; the
// row's own terms a w + gamma in one product
template <int N>
__global__ void __launch_bounds__(256) op_spmm_f64_diag_kernel(DevProblem P, int ld, int G,
                                                               const double* w, double gamma,
                                                               const double* V, double* out) {
  const UnitRow t = make_unit_row(ld, G);
  for (int j = t.id; j < P.n; j += t.count) {
    const int con = P.row_con[j];
    const double own = con >= 0 ? fma(P.row_a[j], w[con], gamma) : gamma;
    // V_j enters only with a constraint or a gamma (0 times an Inf there would be NaN)
    const int own_units = con >= 0 || gamma != 0.0 ? t.units : 0;
    double2 acc[N];
#pragma unroll
    for (int u = 0; u < N; ++u) acc[u] = make_double2(0.0, 0.0);
    int q = P.C_rp[j];
    const int q1 = P.C_rp[j + 1];
    for (; q + 2 <= q1; q += 2) {
      const double* V0 = V + (size_t)P.C_col[q] * ld;
      const double* V1 = V + (size_t)P.C_col[q + 1] * ld;
      const double c0 = -P.C_val[q], c1 = -P.C_val[q + 1];
#pragma unroll
      for (int u = 0; u < N; ++u) {
        const double2 x = unit_at(V0, t.lane + G * u, t.units);
        const double2 y = unit_at(V1, t.lane + G * u, t.units);
        acc[u].x = fma(c1, y.x, fma(c0, x.x, acc[u].x));
        acc[u].y = fma(c1, y.y, fma(c0, x.y, acc[u].y));
      }
    }
    if (q < q1) {
      const double* V0 = V + (size_t)P.C_col[q] * ld;
      const double c0 = -P.C_val[q];
#pragma unroll
      for (int u = 0; u < N; ++u) {
        const double2 x = unit_at(V0, t.lane + G * u, t.units);
        acc[u].x = fma(c0, x.x, acc[u].x);
        acc[u].y = fma(c0, x.y, acc[u].y);
      }
    }
#pragma unroll
    for (int u = 0; u < N; ++u)
      if (t.lane + G * u < t.units) {
        const double2 x = unit_at(V + (size_t)j * ld, t.lane + G * u, own_units);
        *reinterpret_cast<double2*>(out + (size_t)j * ld + 2 * (t.lane + G * u)) =
            make_double2(fma(own, x.x, acc[u].x), fma(own, x.y, acc[u].y));
      }
  }
}

// eq. linU's matrix with diagonal constraints: gamma P_j + rho a^2 (P_j . V_j) V_j, one team per row
template <int N>
__global__ void __launch_bounds__(256) op_hessian_f64_diag_kernel(DevProblem P, int ld, int G,
                                                                  double rho, double gamma,
                                                                  const double* V,
                                                                  const double* Pm, double* out) {
  const UnitRow t = make_unit_row(ld, G);
  const int sub = (threadIdx.x & 31) / G;
  for (int j0 = t.id - sub; j0 < P.n; j0 += t.count) {
    const bool live = j0 + sub < P.n;
    const int j = live ? j0 + sub : P.n - 1;
    const double a = P.row_a[j];
    double2 p[N], v[N];
    double x = 0.0, y = 0.0;
#pragma unroll
    for (int u = 0; u < N; ++u) {
      p[u] = unit_at(Pm + (size_t)j * ld, t.lane + G * u, t.units);
      v[u] = unit_at(V + (size_t)j * ld, t.lane + G * u, t.units);
      x = fma(p[u].x, v[u].x, x);
      y = fma(p[u].y, v[u].y, y);
    }
    __syncwarp();
    double c = rho * (a * (a * team_sum64(x + y, G)));
    // a row without a constraint takes nothing of V, whatever it holds.  Told from a's bits: an FP64
    // comparison is one more FP64 instruction (2^20 rows of r = 20: 149 us with it)
    const bool none = ((__double2hiint(a) & 0x7fffffff) | __double2loint(a)) == 0;
    if (__any_sync(0xffffffffu, none) && none) {
      c = 0.0;
#pragma unroll
      for (int u = 0; u < N; ++u) v[u] = make_double2(0.0, 0.0);
    }
    if (live) {
#pragma unroll
      for (int u = 0; u < N; ++u)
        if (t.lane + G * u < t.units)
          *reinterpret_cast<double2*>(out + (size_t)j * ld + 2 * (t.lane + G * u)) =
              make_double2(fma(c, v[u].x, gamma * p[u].x), fma(c, v[u].y, gamma * p[u].y));
    }
  }
}

// Hessian of eq. linU for multi-entry constraints from q_i = <A_i, P V^T> (op_sddmm_kernel)
template <typename T>
__global__ void op_hessian_q_kernel(DevProblem P, int ld, T rho, T gamma, const T* V,
                                    const T* Pm, const double* q, T* out) {
  const int tid = blockIdx.x * blockDim.x + threadIdx.x, nt = gridDim.x * blockDim.x;
  const WarpRow wr = make_warp_row(ld, tid, nt);
  for (int j = wr.warp; j < P.n; j += wr.nwarps) {
    Frag<T> Pj, H;
    frag_load(Pj, Pm, j, ld, wr.st);
    hessian_row_q_warp<T>(P, V, ld, j, Pj, q, rho, gamma, wr, H);
    if (wr.sub == 0) frag_store(H, out, j, ld, wr.st);
  }
}

// host-side launchers of the solver kernels, per element type and subproblem solver
// (defined in lorads_f64.cu / lorads_f32.cu for SUB 0 and lorads_f64_direct.cu /
// lorads_f32_direct.cu for SUB 1, compiled in parallel)
template <typename T, int SUB>
struct SolveLaunch {
  static cudaError_t solve_block(const SolverArgs<T>* args, int count, int* queue, int grid,
                                 int threads, cudaStream_t s);
  static cudaError_t block_capacity(int threads, int* blocks_per_sm);
  static cudaError_t solve_grid(const SolverArgs<T>* args, GridCtl* ctl, Slot* slots, int reps,
                                long long spin, int grid, int threads, cudaStream_t s);
  static cudaError_t grid_capacity(int threads, int* blocks_per_sm);
  static cudaError_t solve_group(const SolverArgs<T>* args, int count, int* queue, GridCtl* ctls,
                                 Slot* slots, int* picks, int group, long long spin,
                                 int grid, int threads, cudaStream_t s);
  static cudaError_t group_capacity(int threads, int* blocks_per_sm);
};

#define LORADS_DECLARE_SOLVE_LAUNCH(T, SUB)                                                    \
  template <> cudaError_t SolveLaunch<T, SUB>::solve_block(const SolverArgs<T>*, int, int*,    \
                                                           int, int, cudaStream_t);            \
  template <> cudaError_t SolveLaunch<T, SUB>::block_capacity(int, int*);                      \
  template <> cudaError_t SolveLaunch<T, SUB>::solve_grid(const SolverArgs<T>*, GridCtl*,      \
                                                          Slot*, int, long long, int, int,     \
                                                          cudaStream_t);                       \
  template <> cudaError_t SolveLaunch<T, SUB>::grid_capacity(int, int*);                       \
  template <> cudaError_t SolveLaunch<T, SUB>::solve_group(const SolverArgs<T>*, int, int*,    \
                                                           GridCtl*, Slot*, int*, int,         \
                                                           long long, int, int, cudaStream_t); \
  template <> cudaError_t SolveLaunch<T, SUB>::group_capacity(int, int*);
LORADS_DECLARE_SOLVE_LAUNCH(double, 0)
LORADS_DECLARE_SOLVE_LAUNCH(float, 0)
LORADS_DECLARE_SOLVE_LAUNCH(double, 1)
LORADS_DECLARE_SOLVE_LAUNCH(float, 1)

#define LORADS_DEFINE_SOLVE_LAUNCH_BLOCK(T, SUB)                                               \
  template <>                                                                                  \
  cudaError_t SolveLaunch<T, SUB>::solve_block(const SolverArgs<T>* args, int count,           \
                                               int* queue, int grid, int threads,              \
                                               cudaStream_t s) {                               \
    solve_block_kernel<T, SUB><<<grid, threads, 0, s>>>(args, count, queue);                   \
    return cudaGetLastError();                                                                 \
  }                                                                                            \
  template <>                                                                                  \
  cudaError_t SolveLaunch<T, SUB>::block_capacity(int threads, int* blocks_per_sm) {           \
    return cudaOccupancyMaxActiveBlocksPerMultiprocessor(blocks_per_sm,                        \
                                                         solve_block_kernel<T, SUB>, threads,  \
                                                         0);                                   \
  }

#define LORADS_DEFINE_SOLVE_LAUNCH_MULTI(T, SUB)                                               \
  template <>                                                                                  \
  cudaError_t SolveLaunch<T, SUB>::solve_grid(const SolverArgs<T>* args, GridCtl* ctl,         \
                                              Slot* slots, int reps, long long spin, int grid, \
                                              int threads, cudaStream_t s) {                   \
    void* kargs[] = {(void*)&args, (void*)&ctl, (void*)&slots, (void*)&reps, (void*)&spin};    \
    return cudaLaunchCooperativeKernel((const void*)solve_grid_kernel<T, SUB>, dim3(grid),     \
                                       dim3(threads), kargs, 0, s);                            \
  }                                                                                            \
  template <>                                                                                  \
  cudaError_t SolveLaunch<T, SUB>::grid_capacity(int threads, int* blocks_per_sm) {            \
    return cudaOccupancyMaxActiveBlocksPerMultiprocessor(blocks_per_sm,                        \
                                                         solve_grid_kernel<T, SUB>, threads,   \
                                                         0);                                   \
  }                                                                                            \
  template <>                                                                                  \
  cudaError_t SolveLaunch<T, SUB>::solve_group(const SolverArgs<T>* args, int count,           \
                                               int* queue, GridCtl* ctls, Slot* slots,         \
                                               int* picks, int group, long long spin,          \
                                               int grid, int threads, cudaStream_t s) {        \
    void* kargs[] = {(void*)&args,     (void*)&count, (void*)&queue, (void*)&ctls,             \
                     (void*)&slots,    (void*)&picks, (void*)&group, (void*)&spin};            \
    return cudaLaunchCooperativeKernel((const void*)solve_group_kernel<T, SUB>, dim3(grid),    \
                                       dim3(threads), kargs, 0, s);                            \
  }                                                                                            \
  template <>                                                                                  \
  cudaError_t SolveLaunch<T, SUB>::group_capacity(int threads, int* blocks_per_sm) {           \
    return cudaOccupancyMaxActiveBlocksPerMultiprocessor(blocks_per_sm,                        \
                                                         solve_group_kernel<T, SUB>, threads,  \
                                                         0);                                   \
  }

#define LORADS_DEFINE_SOLVE_LAUNCH(T, SUB) \
  LORADS_DEFINE_SOLVE_LAUNCH_BLOCK(T, SUB) \
  LORADS_DEFINE_SOLVE_LAUNCH_MULTI(T, SUB)

// the solver launchers by run-time subproblem solver, and the operator launchers
template <typename T>
struct Launch {
  static cudaError_t solve_block(int sub, const SolverArgs<T>* args, int count, int* queue,
                                 int grid, int threads, cudaStream_t s) {
    return sub ? SolveLaunch<T, 1>::solve_block(args, count, queue, grid, threads, s)
               : SolveLaunch<T, 0>::solve_block(args, count, queue, grid, threads, s);
  }
  static cudaError_t block_capacity(int sub, int threads, int* blocks_per_sm) {
    return sub ? SolveLaunch<T, 1>::block_capacity(threads, blocks_per_sm)
               : SolveLaunch<T, 0>::block_capacity(threads, blocks_per_sm);
  }
  static cudaError_t solve_grid(int sub, const SolverArgs<T>* args, GridCtl* ctl, Slot* slots,
                                int reps, long long spin, int grid, int threads,
                                cudaStream_t s) {
    return sub ? SolveLaunch<T, 1>::solve_grid(args, ctl, slots, reps, spin, grid, threads, s)
               : SolveLaunch<T, 0>::solve_grid(args, ctl, slots, reps, spin, grid, threads, s);
  }
  static cudaError_t grid_capacity(int sub, int threads, int* blocks_per_sm) {
    return sub ? SolveLaunch<T, 1>::grid_capacity(threads, blocks_per_sm)
               : SolveLaunch<T, 0>::grid_capacity(threads, blocks_per_sm);
  }
  static cudaError_t solve_group(int sub, const SolverArgs<T>* args, int count, int* queue,
                                 GridCtl* ctls, Slot* slots, int* picks, int group,
                                 long long spin, int grid, int threads, cudaStream_t s) {
    return sub ? SolveLaunch<T, 1>::solve_group(args, count, queue, ctls, slots, picks,
                                                group, spin, grid, threads, s)
               : SolveLaunch<T, 0>::solve_group(args, count, queue, ctls, slots, picks,
                                                group, spin, grid, threads, s);
  }
  static cudaError_t group_capacity(int sub, int threads, int* blocks_per_sm) {
    return sub ? SolveLaunch<T, 1>::group_capacity(threads, blocks_per_sm)
               : SolveLaunch<T, 0>::group_capacity(threads, blocks_per_sm);
  }
  static cudaError_t op_sddmm(const DevProblem& P, int ld, const T* U, const T* V, double* q,
                              int grid, cudaStream_t s);
  static cudaError_t op_spmm(const DevProblem& P, int ld, const double* w, double gamma,
                             const T* V, T* out, int grid, cudaStream_t s);
  static cudaError_t op_hessian(const DevProblem& P, int ld, double rho, double gamma, const T* V,
                                const T* Pm, T* out, int grid, cudaStream_t s);
};

#define LORADS_DECLARE_LAUNCH(T)                                                               \
  template <> cudaError_t Launch<T>::op_sddmm(const DevProblem&, int, const T*, const T*,      \
                                              double*, int, cudaStream_t);                      \
  template <> cudaError_t Launch<T>::op_spmm(const DevProblem&, int, const double*, double,    \
                                             const T*, T*, int, cudaStream_t);                  \
  template <> cudaError_t Launch<T>::op_hessian(const DevProblem&, int, double, double,        \
                                                const T*, const T*, T*, int, cudaStream_t);
LORADS_DECLARE_LAUNCH(double)
LORADS_DECLARE_LAUNCH(float)

// (lanes per row: unit_lanes; work: the operator's cost)
template <template <int> class K, class... A>
inline cudaError_t launch_units(UnitWork work, int ld, long long rows, int grid, cudaStream_t s,
                                const A&... args) {
  const int G = unit_lanes(work, ld, rows, grid / OP_CTAS_PER_SM);
  switch (unit_count(ld, G)) {
    case 1: K<1>::go(G, grid, s, args...); break;
    case 2: K<2>::go(G, grid, s, args...); break;
    case 3: K<3>::go(G, grid, s, args...); break;
    case 4: K<4>::go(G, grid, s, args...); break;
    case 5: K<5>::go(G, grid, s, args...); break;
    case 6: K<6>::go(G, grid, s, args...); break;
    case 7: K<7>::go(G, grid, s, args...); break;
    default: K<8>::go(G, grid, s, args...); break;
  }
  return cudaGetLastError();
}
template <int N>
struct SddmmF64 {
  static void go(int G, int grid, cudaStream_t s, const DevProblem& P, int ld, const double* U,
                 const double* V, double* q) {
    if (P.a_multi) op_sddmm_f64_kernel<N, true><<<grid, 256, 0, s>>>(P, ld, G, U, V, q);
    else op_sddmm_f64_kernel<N, false><<<grid, 256, 0, s>>>(P, ld, G, U, V, q);
  }
};
template <int N>
struct SpmmF64Diag {
  static void go(int G, int grid, cudaStream_t s, const DevProblem& P, int ld, const double* w,
                 double gamma, const double* V, double* out) {
    op_spmm_f64_diag_kernel<N><<<grid, 256, 0, s>>>(P, ld, G, w, gamma, V, out);
  }
};
template <int N>
struct HessianF64Diag {
  static void go(int G, int grid, cudaStream_t s, const DevProblem& P, int ld, double rho,
                 double gamma, const double* V, const double* Pm, double* out) {
    op_hessian_f64_diag_kernel<N><<<grid, 256, 0, s>>>(P, ld, G, rho, gamma, V, Pm, out);
  }
};

#define LORADS_DEFINE_LAUNCH(T)                                                                \
  template <>                                                                                  \
  cudaError_t Launch<T>::op_sddmm(const DevProblem& P, int ld, const T* U, const T* V,         \
                                  double* q, int grid, cudaStream_t s) {                       \
    if constexpr (sizeof(T) == 8) return launch_units<SddmmF64>(P.a_diag_only ? UNIT_SDDMM_DIAG : UNIT_SDDMM, \
                                                              ld, P.m, grid, s, P, ld, U, V, q); \
    else if (P.a_multi) op_sddmm_kernel<T, true><<<grid, 256, 0, s>>>(P, ld, U, V, q);         \
    else op_sddmm_kernel<T, false><<<grid, 256, 0, s>>>(P, ld, U, V, q);                       \
    return cudaGetLastError();                                                                 \
  }                                                                                            \
  template <>                                                                                  \
  cudaError_t Launch<T>::op_spmm(const DevProblem& P, int ld, const double* w, double gamma,   \
                                 const T* V, T* out, int grid, cudaStream_t s) {               \
    if (!P.a_diag_only) {                                                                      \
      if (sizeof(T) == 8 || short_rows(P.n, P.a_nnz, team_size_for(ld)))                       \
        op_spmm_kernel<T, true, 2><<<grid, 256, 0, s>>>(P, ld, w, gamma, V, out);              \
      else if (team_size_for(ld) >= 4 && P.n < 48 * (grid / OP_CTAS_PER_SM))                                      \
        op_spmm_kernel<T, sizeof(T) == 8, 4><<<grid, 256, 0, s>>>(P, ld, w, gamma, V, out);    \
      else                                                                                     \
        op_spmm_kernel<T, sizeof(T) == 8, 2><<<grid, 256, 0, s>>>(P, ld, w, gamma, V, out);    \
    } else if constexpr (sizeof(T) == 8) {                                                     \
      return launch_units<SpmmF64Diag>(UNIT_SPMM, ld, P.n, grid, s, P, ld, w, gamma, V, out);  \
    } else if ((long long)P.n * team_size_for(ld) < 512LL * (grid / OP_CTAS_PER_SM)) {         \
      op_spmm_diag_kernel<T, 8><<<grid, 256, 0, s>>>(P, ld, w, gamma, V, out);                 \
    } else {                                                                                   \
      op_spmm_diag_kernel<T, 4><<<grid, 256, 0, s>>>(P, ld, w, gamma, V, out);                 \
    }                                                                                          \
    return cudaGetLastError();                                                                 \
  }                                                                                            \
  template <>                                                                                  \
  cudaError_t Launch<T>::op_hessian(const DevProblem& P, int ld, double rho, double gamma,     \
                                    const T* V, const T* Pm, T* out, int grid,                 \
                                    cudaStream_t s) {                                          \
    if (P.a_multi) {                                                                           \
      const cudaError_t e = op_sddmm(P, ld, Pm, V, P.op_q, grid, s);                           \
      if (e != cudaSuccess) return e;                                                          \
      op_hessian_q_kernel<T><<<grid, 256, 0, s>>>(P, ld, (T)rho, (T)gamma, V, Pm, P.op_q, out); \
    } else if (!P.a_diag_only) {                                                               \
      if (short_rows(P.n, P.a_nnz, team_size_for(ld)))                                         \
        op_hessian_kernel<T, 1><<<grid, 256, 0, s>>>(P, ld, (T)rho, (T)gamma, V, Pm, out);     \
      else                                                                                     \
        op_hessian_kernel<T, 2><<<grid, 256, 0, s>>>(P, ld, (T)rho, (T)gamma, V, Pm, out);     \
    } else if constexpr (sizeof(T) == 8) {                                                     \
      return launch_units<HessianF64Diag>(UNIT_HESSIAN, ld, P.n, grid, s, P, ld, rho, gamma, V,    \
                                          Pm, out);                                            \
    } else {                                                                                   \
      op_hessian_diag_kernel<T><<<grid, 256, 0, s>>>(P, ld, (T)rho, (T)gamma, V, Pm, out);     \
    }                                                                                          \
    return cudaGetLastError();                                                                 \
  }

}  // namespace lorads
