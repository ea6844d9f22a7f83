// Device building blocks of the LoRADS solver (sm_103a).
//
// Layout
//   * Factors are row-major n x ld, ld = 4 * ceil(r / 4); padding columns are kept at 0.
//   * A row is processed by a "team" of G lanes (G a power of two <= 32, aligned inside a
//     warp).  Lane l of a team owns the 4-element chunks c = l, l + G, ... (at most KMAX),
//     loaded as 128-bit accesses (float4, or two double2 for FP64).
//   * A constraint is a list of symmetric entries a (E_rc + E_cr) or a E_rr: one entry for
//     MaxCut (A_i = e_i e_i^T, Section 5.3) and matrix completion (Section 5.4), several for
//     general constraints (tr X = 1) and for the rank-one terms of sensor-network localisation
//     (Section 2.3), which assembly expands into their entries (s a a^T has s a_k a_l at (k, l)).
//     The entries are kept twice: in constraint order (con_ptr, con_r, con_c, con_a) for the
//     products <A_i, X Y^T>, and as a symmetric CSR over rows (both triangles) that carries the
//     constraint id, for the sparse-times-dense products.  Constraints with several entries
//     are also cut into chunks of at most CON_CHUNK entries (chunk_ptr; con_chunk gives each
//     constraint's chunks) so that a long constraint is summed by many teams.
//   * Shuffles always name the whole warp, so every loop over teams runs the same number of
//     rounds in all lanes of a warp (TeamRows): teams past the end take part with empty rows.
//     A shuffle that names only its team's lanes splits the warp: one 8-element dot product with
//     its team sum took 478 clocks in teams of 2 and 552 in teams of 4 (9 warps per SM), 126 and
//     169 with the whole warp named.
//   * Reductions are deterministic: fixed shuffle trees inside warps and over a CTA's warps; over
//     CTAs every CTA adds the same sums in the same order (GridScope).
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

#include "lorads_convert.h"

namespace lorads {

constexpr int KMAX = 2;      // chunks per lane
constexpr int CHUNK = 4;     // elements per chunk (16 B of float, 32 B of double)
constexpr int RED_ROWS = 36;  // rows of a scope's shared array (see BlockScope)
constexpr int MAXRED = 12;   // values per reduction (the last slot carries the barrier status)
constexpr int MAXMEM = 8;    // L-BFGS memory cap
constexpr int CON_CHUNK = 32;  // entries per chunk of a multi-entry constraint

// ------------------------------------------------------------------------------------
// problem view
// ------------------------------------------------------------------------------------
struct DevProblem {
  int n, m;
  // entries in constraint order: constraint i owns entries con_ptr[i] .. con_ptr[i+1]-1
  const int* con_ptr;
  const int* con_r;
  const int* con_c;
  const double* con_a;
  const double* b;
  // some constraint has several entries; then the chunks (chunk_ptr into the entries,
  // con_chunk[i] .. con_chunk[i+1]-1 the chunks of constraint i) are set
  int a_multi;
  int nchunk;
  const int* chunk_ptr;
  const int* con_chunk;
  double* op_q;   // m values of scratch for the operator entry points (multi-entry only)
  // A as symmetric CSR over rows; entry e of row j: column A_col[e], constraint A_con[e]
  const int* A_rp;
  const int* A_col;
  const int* A_con;
  const double* A_val;
  const float* A_valf;
  int64_t a_nnz;   // entries of A_col
  // C as symmetric CSR over rows
  const int* C_rp;
  const int* C_col;
  const double* C_val;
  const float* C_valf;
  // row scaling of U_0 onto diagonal constraints (NULL unless every constraint is a single
  // diagonal entry on its own row with b/a > 0): U_0 row j gets norm row_norm[j] (< 0: keep)
  const double* row_norm;
  double b_inf, C_fro, C_inf;
  double b_one, c_one;   // ||b||_1 and ||vec(C)||_1 (the normalisations of Appendix B)
  // every constraint is a diagonal entry: the Hessian of eq. linU is row-local; then
  // row_con[j] is the constraint on row j (-1: none) and row_a[j] its value (0: none)
  int a_diag_only;
  const int* row_con;
  const double* row_a;
  const float* row_af;
  // every row carries exactly one diagonal constraint with b/a > 0 (n = m, row_norm set): the
  // feasible set of the Burer-Monteiro problem is a product of spheres (Phase III applies)
  int polish_ok;
};

template <typename T> __device__ __forceinline__ const T* cval(const DevProblem& P);
template <> __device__ __forceinline__ const double* cval<double>(const DevProblem& P) { return P.C_val; }
template <> __device__ __forceinline__ const float* cval<float>(const DevProblem& P) { return P.C_valf; }
template <typename T> __device__ __forceinline__ const T* rowa(const DevProblem& P);
template <> __device__ __forceinline__ const double* rowa<double>(const DevProblem& P) { return P.row_a; }
template <> __device__ __forceinline__ const float* rowa<float>(const DevProblem& P) { return P.row_af; }
template <typename T> __device__ __forceinline__ const T* aval(const DevProblem& P);
template <> __device__ __forceinline__ const double* aval<double>(const DevProblem& P) { return P.A_val; }
template <> __device__ __forceinline__ const float* aval<float>(const DevProblem& P) { return P.A_valf; }

// ------------------------------------------------------------------------------------
// teams and fragments
// ------------------------------------------------------------------------------------
struct Team {
  int G;          // lanes per row
  int lane;       // lane inside the team
  int id;         // team index inside the scope
  int count;      // teams in the scope
  int nc;         // chunks per row (ld / 4); 0 for a team past the end of its loop
  int sub;        // team index inside the warp
  int first;      // index of the warp's first team
  bool live;      // false for a team past the end of its loop
  bool lead;      // the first lane of a live team
};

__host__ __device__ inline int team_size_for(int ld) {
  int nc = ld / CHUNK;
  int need = (nc + KMAX - 1) / KMAX;
  int G = 1;
  while (G < need) G <<= 1;
  return G > 32 ? 32 : G;
}

__device__ inline Team make_team(int ld, int tid, int nthreads, int mult = 1) {
  Team t;
  t.G = team_size_for(ld) * (mult > 0 ? mult : 1);
  if (t.G > 32) t.G = 32;
  t.lane = tid & (t.G - 1);
  t.id = tid / t.G;
  t.count = nthreads / t.G;
  t.nc = ld / CHUNK;
  t.sub = (threadIdx.x & 31) / t.G;
  t.first = t.id - t.sub;
  t.live = true;
  t.lead = t.lane == 0;
  return t;
}

// A loop of the teams over rows 0 .. n-1 (row j to team j mod count) in which the lanes of a warp
// stay together: a team whose row lies past the end takes the last round with live = false, an
// empty row (nc = 0: loads give zeros, stores store nothing) and j clamped into range.
struct TeamRows {
  Team t;
  int j;
  int base, n, nc;
  __device__ __forceinline__ TeamRows(const Team& tm, int rows)
      : t(tm), base(tm.first), n(rows), nc(tm.nc) {
    place();
  }
  __device__ __forceinline__ bool more() const { return base < n; }
  __device__ __forceinline__ void next() {
    base += t.count;
    place();
  }
  __device__ __forceinline__ void place() {
    j = base + t.sub;
    t.live = j < n;
    t.nc = t.live ? nc : 0;
    t.lead = t.live && t.lane == 0;
    if (!t.live) j = n - 1;
  }
};

template <typename T>
struct Frag {
  T v[KMAX][CHUNK];
};

template <typename T> __device__ __forceinline__ void load4(const T* p, T* o);
template <> __device__ __forceinline__ void load4<float>(const float* p, float* o) {
  float4 x = *reinterpret_cast<const float4*>(p);
  o[0] = x.x; o[1] = x.y; o[2] = x.z; o[3] = x.w;
}
template <> __device__ __forceinline__ void load4<double>(const double* p, double* o) {
  double2 x = reinterpret_cast<const double2*>(p)[0];
  double2 y = reinterpret_cast<const double2*>(p)[1];
  o[0] = x.x; o[1] = x.y; o[2] = y.x; o[3] = y.y;
}
template <typename T> __device__ __forceinline__ void store4(T* p, const T* o);
template <> __device__ __forceinline__ void store4<float>(float* p, const float* o) {
  *reinterpret_cast<float4*>(p) = make_float4(o[0], o[1], o[2], o[3]);
}
template <> __device__ __forceinline__ void store4<double>(double* p, const double* o) {
  reinterpret_cast<double2*>(p)[0] = make_double2(o[0], o[1]);
  reinterpret_cast<double2*>(p)[1] = make_double2(o[2], o[3]);
}

template <typename T>
__device__ __forceinline__ void frag_zero(Frag<T>& f) {
#pragma unroll
  for (int k = 0; k < KMAX; ++k)
#pragma unroll
    for (int e = 0; e < CHUNK; ++e) f.v[k][e] = T(0);
}

template <typename T>
__device__ __forceinline__ void frag_load(Frag<T>& f, const T* base, long long row, int ld,
                                          const Team& t) {
  const T* p = base + row * (long long)ld;
#pragma unroll
  for (int k = 0; k < KMAX; ++k) {
    int c = t.lane + k * t.G;
    if (c < t.nc) {
      load4<T>(p + c * CHUNK, f.v[k]);
    } else {
#pragma unroll
      for (int e = 0; e < CHUNK; ++e) f.v[k][e] = T(0);
    }
  }
}

template <typename T>
__device__ __forceinline__ void frag_store(const Frag<T>& f, T* base, long long row, int ld,
                                           const Team& t) {
  T* p = base + row * (long long)ld;
#pragma unroll
  for (int k = 0; k < KMAX; ++k) {
    int c = t.lane + k * t.G;
    if (c < t.nc) store4<T>(p + c * CHUNK, f.v[k]);
  }
}

// conversions between element types off the FP64 unit (lorads_convert.h; the same values)
__device__ __forceinline__ double to_double(float x) { return widen(x); }
__device__ __forceinline__ double to_double(double x) { return x; }
template <typename D> __device__ __forceinline__ D from_double(double x);
template <> __device__ __forceinline__ float from_double<float>(double x) { return narrow(x); }
template <> __device__ __forceinline__ double from_double<double>(double x) { return x; }

// convert between element types (FP64 master <-> FP32 shadow)
template <typename D, typename S>
__device__ __forceinline__ void frag_convert(Frag<D>& d, const Frag<S>& s) {
#pragma unroll
  for (int k = 0; k < KMAX; ++k)
#pragma unroll
    for (int e = 0; e < CHUNK; ++e) d.v[k][e] = from_double<D>(to_double(s.v[k][e]));
}

// lane-local partial dot product, accumulated in T
template <typename T>
__device__ __forceinline__ T frag_dot_local(const Frag<T>& a, const Frag<T>& b) {
  T s = T(0);
#pragma unroll
  for (int k = 0; k < KMAX; ++k)
#pragma unroll
    for (int e = 0; e < CHUNK; ++e) s = fma(a.v[k][e], b.v[k][e], s);
  return s;
}

// Sum over the lanes of each team, called by whole warps.  The lanes arrive here from loads that
// only some of them make (a row's last chunks: r = 9, ld = 12, lane 1 of a team has no second one) and
// converge before they exchange.  Builds of the one-CTA FP64 kernel that named only the team's lanes
// and did not converge them diverged on matrix completion, depending on how they were compiled, and
// became exact with a convergence here and nothing else changed.  The shuffle waits for the lanes
// it names by itself, so why that mattered is not known; it has not been seen since.
template <typename T>
__device__ __forceinline__ T team_sum(T x, const Team& t) {
  __syncwarp();
  for (int off = t.G >> 1; off > 0; off >>= 1) x += __shfl_xor_sync(0xffffffffu, x, off);
  return x;
}

template <typename T>
__device__ __forceinline__ T frag_dot(const Frag<T>& a, const Frag<T>& b, const Team& t) {
  return team_sum(frag_dot_local(a, b), t);
}

// y += alpha x
template <typename T>
__device__ __forceinline__ void frag_axpy(Frag<T>& y, T alpha, const Frag<T>& x) {
#pragma unroll
  for (int k = 0; k < KMAX; ++k)
#pragma unroll
    for (int e = 0; e < CHUNK; ++e) y.v[k][e] = fma(alpha, x.v[k][e], y.v[k][e]);
}

// ------------------------------------------------------------------------------------
// counter-based random numbers: SplitMix64 (Steele, Lea and Flood, OOPSLA 2014) and the
// Box-Muller transform (Box and Muller, 1958)
// ------------------------------------------------------------------------------------
__host__ __device__ inline uint64_t splitmix64_mix(uint64_t z) {
  z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ULL;
  z = (z ^ (z >> 27)) * 0x94D049BB133111EBULL;
  return z ^ (z >> 31);
}
// output i (0-based) of the SplitMix64 stream seeded with key
__host__ __device__ inline uint64_t splitmix64_at(uint64_t key, uint64_t i) {
  return splitmix64_mix(key + (i + 1ULL) * 0x9E3779B97F4A7C15ULL);
}
// key of sub-stream s: 0 draws U_0, g >= 1 draws the columns of the g-th rank growth
__host__ __device__ inline uint64_t stream_key(uint64_t seed, uint64_t s) {
  return splitmix64_at(seed, s);
}
__device__ inline double uniform_open01(uint64_t key, uint64_t i) {
  return ((double)(splitmix64_at(key, i) >> 11) + 0.5) * 0x1.0p-53;
}
// standard normal number e of the stream: outputs 2e and 2e+1
__device__ inline double normal_at(uint64_t key, uint64_t e) {
  double u1 = uniform_open01(key, 2 * e);
  double u2 = uniform_open01(key, 2 * e + 1);
  return sqrt(-2.0 * log(u1)) * cospi(2.0 * u2);
}

// ------------------------------------------------------------------------------------
// scopes: one CTA, or the whole grid of a cooperative launch
// ------------------------------------------------------------------------------------
__device__ __forceinline__ int ld_acquire_s32(const int* p) {
  int v;
  asm volatile("ld.acquire.gpu.global.s32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}
struct GridCtl {
  int error;      // a barrier gave up: every CTA of the scope leaves at its next wait
  int pad[3];
};

// Sum over the 32 lanes of a warp of K values (K a power of two, <= 16) by recursive halving:
// each round a lane keeps half of its remaining values and adds the partner's copy of that
// half (the partner keeps the other half), so after log2 K rounds a lane holds one value
// index, completed by a butterfly over the remaining lane offsets.  K - 1 + 5 - log2 K FP64
// adds per lane instead of 5 K (FP64 issues at a small fraction of the FP32 rate here).
// The order of the additions is fixed, so the sums are deterministic; lanes holding the same
// index hold bitwise equal sums.  Returns the index held in w[0].
template <int K>
__device__ __forceinline__ int warp_sum_scatter(double* w) {
  const int lane = threadIdx.x & 31;
  int ix = 0, off = 16;
#pragma unroll
  for (int h = K / 2; h >= 1; h >>= 1) {
    const bool up = (lane & off) != 0;
#pragma unroll
    for (int i = 0; i < h; ++i) {
      const double keep = up ? w[i + h] : w[i];
      const double give = up ? w[i] : w[i + h];
      w[i] = keep + __shfl_xor_sync(0xffffffffu, give, off);
    }
    if (up) ix += h;
    off >>= 1;
  }
#pragma unroll
  for (; off > 0; off >>= 1) w[0] += __shfl_xor_sync(0xffffffffu, w[0], off);
  return ix;
}

// the lane that stores the warp sum of its value index (the first of its group)
template <int K>
__device__ __forceinline__ bool scatter_writer() {
  return ((threadIdx.x & 31) & (32 / K - 1)) == 0;
}

// Stage 1 of a reduction: the warp sums of k values into red[warp * MAXRED + i].
template <int K>
__device__ __forceinline__ void warp_sums_k(const double* v, int k, double* red) {
  const int warp = threadIdx.x >> 5;
  double w[K];
#pragma unroll
  for (int i = 0; i < K; ++i) w[i] = i < k ? v[i] : 0.0;
  const int ix = warp_sum_scatter<K>(w);
  if (scatter_writer<K>() && ix < k) red[warp * MAXRED + ix] = w[0];
}
__device__ __forceinline__ void warp_sums(const double* v, int k, double* red) {
  __syncwarp();
  if (k <= 1) warp_sums_k<1>(v, k, red);
  else if (k <= 2) warp_sums_k<2>(v, k, red);
  else if (k <= 4) warp_sums_k<4>(v, k, red);
  else if (k <= 8) warp_sums_k<8>(v, k, red);
  else warp_sums_k<16>(v, k, red);
}
// Stage 1 for two values carried by teams of G lanes.  G >= 2: value 0 sits in the teams' even
// lanes' x0 and value 1 in their odd lanes' x0, so one butterfly over the lane offsets 16 .. G
// sums both (offsets below G would only add a team's lanes to one another); G = 1: every lane
// carries both.  The additions of each value are those of warp_sum_scatter with the values in
// lane 0 of each team.
__device__ __forceinline__ void warp_sums_pair(double x0, double x1, int G, double* red) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  __syncwarp();
  if (G >= 2) {
    for (int off = 16; off >= G; off >>= 1) x0 += __shfl_xor_sync(0xffffffffu, x0, off);
    if (lane < 2) red[warp * MAXRED + lane] = x0;
  } else {
    const double v[2] = {x0, x1};
    warp_sums_k<2>(v, 2, red);
  }
}

// Stage 2, by one warp: the sum of value i over the CTA's warps (at most 16) in the order of a
// butterfly, in every lane below 16.
__device__ __forceinline__ double block_sum(int i, const double* red) {
  const int lane = threadIdx.x & 31, nw = (blockDim.x + 31) >> 5;
  double x = lane < nw ? red[lane * MAXRED + i] : 0.0;
#pragma unroll
  for (int off = 8; off > 0; off >>= 1) x += __shfl_xor_sync(0xffffffffu, x, off);
  return x;
}

// deterministic CTA-wide sum of k (< MAXRED) values; every thread receives the sums in v.
// Warp i finishes value i, so the second stage takes one chain of four additions whatever k is.
__device__ inline void block_reduce(double* v, int k, double* red /* smem [33*MAXRED] */) {
  const int nw = (blockDim.x + 31) >> 5;
  warp_sums(v, k, red);
  __syncthreads();
  for (int i = threadIdx.x >> 5; i < k; i += nw) {
    const double x = block_sum(i, red);
    if ((threadIdx.x & 31) == 0) red[32 * MAXRED + i] = x;
  }
  __syncthreads();
  for (int i = 0; i < k; ++i) v[i] = red[32 * MAXRED + i];
}

// Scopes: the CTA's shared array `red` holds RED_ROWS rows of MAXRED doubles: rows 0..31 the
// per-warp sums of a reduction, row 32 its results, rows 33..35 per-CTA scalar scratch for the
// solver (no __shared__ variables are declared inside solver functions, which several kernels
// instantiate).
//
// reduce_pair sums two values given in warp_sums_pair's form and calls f(sum 0, sum 1) in thread 0
// of every CTA before the CTA goes on: f evaluates the scalars that follow from the sums (FP64
// divides issue at 1/64 of the FP32 rate here, so one thread per CTA does it) and leaves them in
// the scratch row.  reduce_each<K>(v, f) calls f(i, sum i) for each of K values in one thread of
// the CTA.  EXCHANGE tells whether the scope's CTAs also read one another's memory writes after it;
// without, a reduction orders nothing but its sums.
struct BlockScope {
  double* red;
  __device__ double* scratch() const { return red + 33 * MAXRED; }
  __device__ int tid() const { return threadIdx.x; }
  __device__ int nthreads() const { return blockDim.x; }
  __device__ bool sync() {
    __syncthreads();
    return true;
  }
  template <int K>
  __device__ __forceinline__ bool reduce(double* v) {
    static_assert(K >= 1 && K < MAXRED, "a row of the shared array holds a reduction's values");
    return reduce_any(v, K);
  }
  __device__ bool reduce_any(double* v, int k) {
    block_reduce(v, k, red);
    return true;
  }
  template <bool EXCHANGE, class F>
  __device__ __forceinline__ bool reduce_pair(double x0, double x1, int G, F f) {
    warp_sums_pair(x0, x1, G, red);
    __syncthreads();
    if (threadIdx.x < 32) {
      // lanes 0-15 finish value 0, lanes 16-31 value 1 (block_sum's order)
      const int lane = threadIdx.x, w = lane & 15, nw = (blockDim.x + 31) >> 5;
      double x = w < nw ? red[w * MAXRED + (lane >> 4)] : 0.0;
#pragma unroll
      for (int off = 8; off > 0; off >>= 1) x += __shfl_xor_sync(0xffffffffu, x, off);
      const double o = __shfl_sync(0xffffffffu, x, 16);
      if (lane == 0) f(x, o);
    }
    __syncthreads();
    return true;
  }
  template <int K, class F>
  __device__ __forceinline__ bool reduce_each(const double* v, F f) {
    static_assert(K >= 1 && K < MAXRED, "a row of the shared array holds a reduction's values");
    constexpr int k = K;
    const int nw = (blockDim.x + 31) >> 5;
    warp_sums(v, k, red);
    __syncthreads();
    for (int i = threadIdx.x >> 5; i < k; i += nw) {
      const double x = block_sum(i, red);
      if ((threadIdx.x & 31) == 0) f(i, x);
    }
    __syncthreads();
    return true;
  }
  __device__ bool is_leader() const { return threadIdx.x == 0; }
  __device__ bool leader_cta() const { return true; }
};

// a CTA's partial sum of one value and the number of the barrier it belongs to, stored and
// loaded as one 128-bit access (single-copy atomic as a relaxed .b128 access)
struct alignas(16) Slot {
  double v;
  unsigned long long tag;
};
__device__ __forceinline__ void st_slot(Slot* p, double v, unsigned long long tag) {
  asm volatile(
      "{\n .reg .b128 q;\n mov.b128 q, {%1, %2};\n st.relaxed.gpu.global.b128 [%0], q;\n}\n" ::"l"(p),
      "l"(__double_as_longlong(v)), "l"(tag)
      : "memory");
}
__device__ __forceinline__ void ld_slot(const Slot* p, double& v, unsigned long long& tag) {
  long long a;
  unsigned long long b;
  asm volatile(
      "{\n .reg .b128 q;\n ld.relaxed.gpu.global.b128 q, [%2];\n mov.b128 {%0, %1}, q;\n}\n"
      : "=l"(a), "=l"(b) : "l"(p) : "memory");
  v = __longlong_as_double(a);
  tag = b;
}
__device__ __forceinline__ void fence_release_gpu() {
  asm volatile("fence.release.gpu;" ::: "memory");
}
__device__ __forceinline__ void fence_acquire_gpu() {
  asm volatile("fence.acquire.gpu;" ::: "memory");
}

// One warp: polls the slots of c CTAs until every tag is `bar` and returns the sum of their values:
// lane l adds the CTAs l, l + 32, ... and the lanes combine by a butterfly.  ok turns false when
// the wait is given up: after `limit` polls (which sets *error) or when *error is set.  A function
// of its own: inlined at every reduction its buffers pushed the solver's rows out of registers.
static __device__ __noinline__ double poll_slots(const Slot* from, int c, unsigned bar, int* error,
                                          long long limit, bool& ok) {
  constexpr int TC = 5;            // 160 CTAs per round of loads
  const int lane = threadIdx.x & 31;
  double s = 0.0;
  long long it = 0;
  bool good = true;
  for (int b0 = 0; b0 < c && good; b0 += 32 * TC) {
    double v[TC];
    for (;;) {
      bool all = true;
#pragma unroll
      for (int t = 0; t < TC; ++t) {
        const int b = b0 + lane + 32 * t;
        unsigned long long tag = bar;
        v[t] = 0.0;
        if (b < c) ld_slot(from + b, v[t], tag);
        all = all && tag == bar;
      }
      if (all) break;
      if ((++it & 63) == 0 && ld_acquire_s32(error)) good = false;
      if (good && it > limit) {
        atomicExch(error, 1);
        good = false;
      }
      if (!good) break;
    }
#pragma unroll
    for (int t = 0; t < TC; ++t) s = (b0 == 0 && t == 0) ? v[0] : s + v[t];
  }
  ok = __all_sync(0xffffffffu, good);
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) s += __shfl_xor_sync(0xffffffffu, s, off);
  return s;
}

constexpr int SLOT_VALUES = 9;    // values of one reduction, at most
constexpr int SLOT_REPS = 4;      // copies of every slot, at most (at most 16: one lane stores each)
// doubles of slot memory per CTA of a scope and copy: two barriers x SLOT_VALUES x 16 bytes
constexpr int SLOT_DOUBLES = 2 * SLOT_VALUES * 2;

// A scope of several co-resident CTAs.  A reduction leaves each CTA's sum of every value in a
// slot of its own, tagged with the barrier's number; a CTA polls the slots of all CTAs until
// the tags match and adds the values in CTA order: lane l of a value takes the CTAs l, l + 32, ...
// and the lanes combine by a butterfly, so every CTA forms the same sums.  There is no counter:
// on the critical path are one store's way to L2 and one load's way back, where an arrival on a
// counter, its release, the wait for it and the loads of the partial sums are four such ways.
// Slots are kept in `reps` copies, CTA b polling copy b % reps: one copy polled by 152 CTAs is
// a hot spot that delays the stores behind it.  Measured at 152 x 288 threads, two values,
// memory writes ordered: 5.08 us with a counter, 5.48 / 4.37 / 3.90 / 3.95 / 4.40 / 4.49 us with 1 / 2 /
// 4 / 8 / 16 / 152 copies; 3.32 us (4 copies) when only the sums are exchanged, since the release
// fence is not needed.
// Consecutive barriers use two sets of slots by the parity of their number: a CTA stores for
// barrier g + 2 only after it passed g + 1, where every CTA had stored, that is, had finished
// reading barrier g.  Tags start at 1 and the slots hold no valid tag at launch (the host fills
// them with 0xFF), so stale contents never match.
struct GridScope {
  double* red;             // shared memory (see BlockScope)
  GridCtl* ctl;            // zeroed before launch
  Slot* slots;             // reps copies of 2 x SLOT_VALUES x count() slots
  int reps;
  long long spin_limit;    // polls before a barrier gives up
  int first = 0;           // the scope spans CTAs [first, first + nb) of a cooperative launch
  int nb = 0;              // (0: the whole grid)
  unsigned gen = 0;        // number of the last barrier

  __device__ int count() const { return nb > 0 ? nb : (int)gridDim.x; }
  __device__ double* scratch() const { return red + 33 * MAXRED; }
  __device__ int tid() const { return ((int)blockIdx.x - first) * blockDim.x + threadIdx.x; }
  __device__ int nthreads() const { return count() * blockDim.x; }
  __device__ bool is_leader() const { return (int)blockIdx.x == first && threadIdx.x == 0; }
  __device__ bool leader_cta() const { return (int)blockIdx.x == first; }

  // clears the failure mark; every thread, once, before the scope's first barrier
  __device__ void init() {
    if (threadIdx.x == 0) red[32 * MAXRED + MAXRED - 1] = 0.0;
    __syncthreads();
  }
  __device__ bool failed() const { return red[32 * MAXRED + MAXRED - 1] != 0.0; }

  // One warp: stores the CTA's sum x of value i (the same in every lane below 16) for barrier `bar`
  __device__ __forceinline__ void put(double x, int i, unsigned bar) {
    const int lane = threadIdx.x & 31, c = count(), me = (int)blockIdx.x - first;
    const size_t copy = (size_t)2 * SLOT_VALUES * c;
    Slot* set = slots + ((size_t)(bar & 1u) * SLOT_VALUES + i) * c;
    if (lane < reps) st_slot(set + lane * copy + me, x, bar);
  }
  // One warp: the sum of value i over the scope, in every lane
  __device__ __forceinline__ double take(int i, unsigned bar) {
    const int c = count(), me = (int)blockIdx.x - first;
    const size_t copy = (size_t)2 * SLOT_VALUES * c;
    const Slot* set = slots + ((size_t)(bar & 1u) * SLOT_VALUES + i) * c;
    bool ok = true;
    const double s = poll_slots(set + (me % reps) * copy, c, bar, &ctl->error, spin_limit, ok);
    if (!ok) red[32 * MAXRED + MAXRED - 1] = 1.0;
    return s;
  }
  // both, for a warp with one value
  template <bool EXCHANGE>
  __device__ __forceinline__ double exchange(double x, int i, unsigned bar) {
    if (EXCHANGE) fence_release_gpu();
    put(x, i, bar);
    const double s = take(i, bar);
    if (EXCHANGE) fence_acquire_gpu();
    return s;
  }

  __device__ bool sync() {
    const unsigned bar = ++gen;
    __syncthreads();
    if (threadIdx.x < 32) exchange<true>(0.0, 0, bar);
    __syncthreads();
    return !failed();
  }

  // f(i, sum i) in lane 0 of the warp that finishes value i
  template <int K, class F>
  __device__ __forceinline__ bool reduce_each(const double* v, F f) {
    static_assert(K >= 1 && K <= SLOT_VALUES, "a set of slots holds a reduction's values");
    return each_any(v, K, f);
  }
  template <class F>
  __device__ __forceinline__ bool each_any(const double* v, int k, F f) {
    const int nw = (blockDim.x + 31) >> 5;
    warp_sums(v, k, red);
    const unsigned bar = ++gen;
    __syncthreads();
    // a warp stores all of its values before it waits for any: one trip through L2, and not three, for
    // the line search's 9 values in CTAs of 4 warps (Phase I of ER n = 1,600 5.5 -> 5.2 ms)
    const int warp = threadIdx.x >> 5;
    if (warp < k) fence_release_gpu();
    for (int i = warp; i < k; i += nw) put(block_sum(i, red), i, bar);
    for (int i = warp; i < k; i += nw) {
      const double s = take(i, bar);
      fence_acquire_gpu();
      if ((threadIdx.x & 31) == 0) f(i, s);
    }
    __syncthreads();
    return !failed();
  }
  template <int K>
  __device__ __forceinline__ bool reduce(double* v) {
    static_assert(K >= 1 && K <= SLOT_VALUES, "a set of slots holds a reduction's values");
    return reduce_any(v, K);
  }
  __device__ bool reduce_any(double* v, int k) {
    double* out = red + 32 * MAXRED;
    const bool ok = each_any(v, k, [out](int i, double s) { out[i] = s; });
    for (int i = 0; i < k; ++i) v[i] = out[i];
    return ok;
  }
  template <bool EXCHANGE, class F>
  __device__ __forceinline__ bool reduce_pair(double x0, double x1, int G, F f) {
    warp_sums_pair(x0, x1, G, red);
    const unsigned bar = ++gen;
    __syncthreads();
    const int warp = threadIdx.x >> 5;
    if (warp < 2) {
      const double s = exchange<EXCHANGE>(block_sum(warp, red), warp, bar);
      // warp 1 hands its sum to warp 0 (a named barrier of the two)
      if (warp == 1) {
        if (threadIdx.x == 32) red[32 * MAXRED] = s;
        __syncwarp();
        asm volatile("bar.arrive 1, 64;" ::: "memory");
      } else {
        asm volatile("bar.sync 1, 64;" ::: "memory");
        if (threadIdx.x == 0) f(s, red[32 * MAXRED]);
      }
    }
    __syncthreads();
    return !failed();
  }
};

// The scope of a CTA group inside a batch launch: the grid scope's code, as a type of its own
// so that each kernel instantiates its own solver (no solver instantiation is reached from
// two kernels).
struct GroupScope : GridScope {};

// ------------------------------------------------------------------------------------
// per-row operators (shared by the solver and the operator entry points)
// ------------------------------------------------------------------------------------

// Hessian of eq. linU on row j with fixed factor W:
//   (H P)_j = rho * sum_{entries (j,k) of A_i} a q_i W_k + gamma P_j,
//   q_i = <A_i, P W^T> = a (P_j . W_k + P_k . W_j)   (off-diagonal)   or   a P_j . W_j.
// This form: every constraint is one diagonal entry, at most one per row (a: row j's value, 0
// without a constraint).  Returns the row in out; called by whole warps.
template <typename T>
__device__ __forceinline__ void hessian_row(T a, const Frag<T>& Wj, const Frag<T>& Pj, T rho,
                                            T gamma, const Team& t, Frag<T>& out) {
  const T q = a * frag_dot(Pj, Wj, t);
  const T aq = a * q;
  // a row without a constraint takes no term from W (0 times an Inf there would be NaN)
  const bool on = a != T(0);
#pragma unroll
  for (int kk = 0; kk < KMAX; ++kk)
#pragma unroll
    for (int ee = 0; ee < CHUNK; ++ee)
      out.v[kk][ee] = fma(rho, on ? aq * Wj.v[kk][ee] : T(0), gamma * Pj.v[kk][ee]);
}

// (A^T(w) - C) W on row j, w_i = wb * b_i + wl * lambda_i + we * e_i (e may be NULL),
// plus gamma W_j.  All in T.
template <typename T>
__device__ __forceinline__ void spmm_row(const DevProblem& P, const T* Wm, int ld, int j,
                                         const double* lam, const double* e, double wb, double wl,
                                         double we, T gamma, const Team& t, Frag<T>& out) {
  Frag<T> acc;
  frag_zero(acc);
  const T* cv = cval<T>(P);
  {
    // four rows in flight: the column indices, then the rows, then the sums
    int q = P.C_rp[j];
    const int qe = P.C_rp[j + 1];
    for (; q + 4 <= qe; q += 4) {
      const int k0 = P.C_col[q], k1 = P.C_col[q + 1], k2 = P.C_col[q + 2], k3 = P.C_col[q + 3];
      const T c0 = cv[q], c1 = cv[q + 1], c2 = cv[q + 2], c3 = cv[q + 3];
      Frag<T> W0, W1, W2, W3;
      frag_load(W0, Wm, k0, ld, t);
      frag_load(W1, Wm, k1, ld, t);
      frag_load(W2, Wm, k2, ld, t);
      frag_load(W3, Wm, k3, ld, t);
      frag_axpy(acc, -c0, W0);
      frag_axpy(acc, -c1, W1);
      frag_axpy(acc, -c2, W2);
      frag_axpy(acc, -c3, W3);
    }
    for (; q < qe; ++q) {
      Frag<T> Wk;
      frag_load(Wk, Wm, P.C_col[q], ld, t);
      frag_axpy(acc, -cv[q], Wk);
    }
  }
  const T* av = aval<T>(P);
  const bool a_part = (wb != 0.0) || (lam != nullptr) || (e != nullptr);
  for (int q = a_part ? P.A_rp[j] : 0; q < (a_part ? P.A_rp[j + 1] : 0); ++q) {
    const int i = P.A_con[q];
    double w = wb * P.b[i];
    if (lam) w += wl * lam[i];
    if (e) w += we * e[i];
    Frag<T> Wk;
    frag_load(Wk, Wm, P.A_col[q], ld, t);
    frag_axpy(acc, (T)(w * (double)av[q]), Wk);
  }
  if (gamma != T(0)) {
    Frag<T> Wj;
    frag_load(Wj, Wm, j, ld, t);
    frag_axpy(acc, gamma, Wj);
  }
  out = acc;
}

// <a (E_rc + E_cr), U V^T> = a (U_r . V_c + U_c . V_r), or a U_r . V_r when r = c
// (team-cooperative; the value in every lane)
template <typename T>
__device__ __forceinline__ double sddmm_entry(const T* Um, const T* Vm, int ld, int r, int c,
                                              double a, const Team& t) {
  Frag<T> Ur, Vc;
  frag_load(Ur, Um, r, ld, t);
  frag_load(Vc, Vm, c, ld, t);
  T loc = frag_dot_local(Ur, Vc);
  if (r != c) {
    Frag<T> Uc, Vr;
    frag_load(Uc, Um, c, ld, t);
    frag_load(Vr, Vm, r, ld, t);
    loc += frag_dot_local(Uc, Vr);
  }
  return a * to_double(team_sum(loc, t));
}

// <A_i, U V^T> where every constraint has one entry (the i-th entry is constraint i's)
template <typename T>
__device__ __forceinline__ double sddmm_con(const DevProblem& P, const T* Um, const T* Vm, int ld,
                                            int i, const Team& t) {
  return sddmm_entry<T>(Um, Vm, ld, P.con_r[i], P.con_c[i], P.con_a[i], t);
}

// <A_i, U V^T>: the sum over constraint i's entries (team-cooperative; called by whole warps, whose
// teams take as many rounds as the longest of their constraints), two entries a round, the rows of
// both read before either is summed.  A team that has no entry left takes part empty-handed: repeating
// one of its own cost the warp that entry's loads and, off the diagonal, a second product in every
// round.  Bound by the latency of the rows' loads: the trace of n = 3,000 beside 9,000 constraints of one
// entry, FP32, r = 9, 1,507 us with repeated entries, 975 so.
template <typename T>
__device__ __forceinline__ double sddmm_con_multi(const DevProblem& P, const T* Um, const T* Vm,
                                                  int ld, int i, const Team& t) {
  const int e0 = P.con_ptr[i], cnt = t.live ? P.con_ptr[i + 1] - e0 : 0;
  const int rounds = __reduce_max_sync(0xffffffffu, cnt);
  double s = 0.0;
  for (int k = 0; k < rounds; k += 2) {
    Frag<T> Ur[2], Vc[2];
    int r[2], c[2];
    double a[2];
    T loc[2];
    Team te[2] = {t, t};
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const bool on = k + h < cnt;
      const int e = on ? e0 + k + h : e0;
      c[h] = P.con_c[e];
      r[h] = on ? P.con_r[e] : c[h];
      a[h] = P.con_a[e];
      te[h].nc = on ? t.nc : 0;
    }
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      frag_load(Ur[h], Um, r[h], ld, te[h]);
      frag_load(Vc[h], Vm, c[h], ld, te[h]);
    }
#pragma unroll
    for (int h = 0; h < 2; ++h) loc[h] = frag_dot_local(Ur[h], Vc[h]);
#pragma unroll
    for (int h = 0; h < 2; ++h)
      if (r[h] != c[h]) {
        frag_load(Ur[h], Um, c[h], ld, te[h]);
        frag_load(Vc[h], Vm, r[h], ld, te[h]);
        loc[h] += frag_dot_local(Ur[h], Vc[h]);
      }
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const double x = a[h] * to_double(team_sum(loc[h], t));
      if (k + h < cnt) s += x;
    }
  }
  return s;
}

// ------------------------------------------------------------------------------------
// warp-split rows: one warp per row, S = 32/G sub-teams of G lanes; sub-team s takes the
// row's entries s, s+S, s+2S, ... two at a time (four rows in flight per sub-team), and the
// partial sums are combined over sub-teams with shuffles.  Used where rows carry many
// entries (matrix completion: ~785 per row at n = 40,000), which a single team would walk
// as a chain of dependent loads.
// ------------------------------------------------------------------------------------
struct WarpRow {
  Team st;     // the lane's sub-team
  int sub;     // sub-team index inside the warp
  int S;       // sub-teams per warp
  int warp;    // warp index inside the scope
  int nwarps;  // warps in the scope
};

__device__ inline WarpRow make_warp_row(int ld, int tid, int nthreads, int mult = 1) {
  WarpRow w;
  w.st = make_team(ld, threadIdx.x & 31, 32, mult);   // team ids 0..S-1 inside the warp
  w.sub = w.st.id;
  w.S = 32 / w.st.G;
  w.warp = tid >> 5;
  w.nwarps = nthreads >> 5;
  return w;
}

template <typename T>
__device__ __forceinline__ void frag_warp_combine(Frag<T>& f, int G) {
  __syncwarp();
#pragma unroll
  for (int k = 0; k < KMAX; ++k)
#pragma unroll
    for (int e = 0; e < CHUNK; ++e) {
      T x = f.v[k][e];
      for (int off = G; off < 32; off <<= 1) x += __shfl_xor_sync(0xffffffffu, x, off);
      f.v[k][e] = x;
    }
}

// H entries per sub-team of row j's terms a q W_k, from entry e0 on (all lanes of the warp).  FULL: every
// sub-team has H; else an entry past the row's end e1 reads and adds nothing.  A diagonal entry
// (k = j) has the one product q = a P_j . W_j.  (Adding products with zero rows instead would turn an
// Inf of the other factor into NaN.)
template <typename T, int H, bool FULL>
__device__ __forceinline__ void hessian_entries(const DevProblem& P, const T* Wm, const T* Pm, int ld,
                                                int j, int e0, int e1, const Frag<T>& Pj,
                                                const Frag<T>& Wj, const WarpRow& w,
                                                Frag<T>& acc) {
  const Team& t = w.st;
  const T* av = aval<T>(P);
  Frag<T> Wk[H], Pk[H];
  T a[H], q[H];
  bool on[H], off[H];               // an entry of the row; off the diagonal
#pragma unroll
  for (int h = 0; h < H; ++h) {
    const int e = e0 + w.sub + h * w.S;
    Team tw = t, tp = t;
    int k = j;
    a[h] = T(0);
    on[h] = FULL || e < e1;
    if (on[h]) {
      k = P.A_col[e];
      a[h] = av[e];
    } else {
      tw.nc = 0;
    }
    off[h] = k != j;
    tp.nc = off[h] ? tw.nc : 0;
    frag_load(Wk[h], Wm, k, ld, tw);
    frag_load(Pk[h], Pm, k, ld, tp);
  }
#pragma unroll
  for (int h = 0; h < H; ++h) {
    const T mirror = frag_dot_local(Pk[h], Wj);
    q[h] = a[h] * team_sum(frag_dot_local(Pj, Wk[h]) + (off[h] ? mirror : T(0)), t);
  }
#pragma unroll
  for (int h = 0; h < H; ++h) frag_axpy(acc, on[h] ? a[h] * q[h] : T(0), Wk[h]);
}

// (H P)_j = rho sum a q W_k + gamma P_j with the whole warp; out valid in every lane.  All
// sub-teams take the same number of rounds, H entries each.
template <typename T, int H = 2>
__device__ void hessian_row_warp(const DevProblem& P, const T* Wm, const T* Pm, int ld, int j,
                                 const Frag<T>& Pj, T rho, T gamma, const WarpRow& w,
                                 Frag<T>& out) {
  const Team& t = w.st;
  Frag<T> Wj, acc;
  frag_load(Wj, Wm, j, ld, t);
  frag_zero(acc);
  const int e1 = P.A_rp[j + 1];
  int e0 = P.A_rp[j];
  for (; H == 2 && e0 + 2 * w.S <= e1; e0 += 2 * w.S)
    hessian_entries<T, 2, true>(P, Wm, Pm, ld, j, e0, e1, Pj, Wj, w, acc);
  for (; e0 < e1; e0 += H * w.S)
    hessian_entries<T, H, false>(P, Wm, Pm, ld, j, e0, e1, Pj, Wj, w, acc);
  frag_warp_combine(acc, t.G);
#pragma unroll
  for (int kk = 0; kk < KMAX; ++kk)
#pragma unroll
    for (int ee = 0; ee < CHUNK; ++ee) out.v[kk][ee] = fma(rho, acc.v[kk][ee], gamma * Pj.v[kk][ee]);
}

// H entries per sub-team of a row's sum, from entry s0 of `rounds` on: lane l holds entry l's column and
// weight
template <typename T, int H>
__device__ __forceinline__ void spmm_entries(const T* Wm, int ld, int s0, int rounds, int col, T c,
                                             const WarpRow& w, Frag<T>& acc) {
  Frag<T> Wk[H];
  T ck[H];
#pragma unroll
  for (int u = 0; u < H; ++u) {
    const int src = s0 + u * w.S + w.sub;          // < 32 when it is one of the entries
    const int k = __shfl_sync(0xffffffffu, col, src & 31);
    ck[u] = __shfl_sync(0xffffffffu, c, src & 31);
    Team tw = w.st;
    tw.nc = src < rounds ? w.st.nc : 0;
    frag_load(Wk[u], Wm, k, ld, tw);
  }
#pragma unroll
  for (int u = 0; u < H; ++u)
    if (s0 + u * w.S + w.sub < rounds) frag_axpy(acc, ck[u], Wk[u]);
}

// (A^T(w) - C) W on row j with the whole warp (same weights as spmm_row); out in every lane.  OWN: every
// sub-team forms the weights of its entries, for FP64, whose products outweigh them, and for short
// rows; else the warp forms 32 at once, H rows in flight per sub-team.
template <typename T, bool OWN = sizeof(T) == 8, int H = 2>
__device__ void spmm_row_warp(const DevProblem& P, const T* Wm, int ld, int j, const double* lam,
                              const double* e, double wb, double wl, double we, T gamma,
                              const WarpRow& w, Frag<T>& out) {
  const Team& t = w.st;
  Frag<T> acc;
  frag_zero(acc);
  const T* cv = cval<T>(P);
  {
    const int q1 = P.C_rp[j + 1];
    int q = P.C_rp[j] + w.sub;
    for (; q + w.S < q1; q += 2 * w.S) {
      const int k0 = P.C_col[q], k1 = P.C_col[q + w.S];
      const T c0 = cv[q], c1 = cv[q + w.S];
      Frag<T> W0, W1;
      frag_load(W0, Wm, k0, ld, t);
      frag_load(W1, Wm, k1, ld, t);
      frag_axpy(acc, -c0, W0);
      frag_axpy(acc, -c1, W1);
    }
    if (q < q1) {
      Frag<T> Wk;
      frag_load(Wk, Wm, P.C_col[q], ld, t);
      frag_axpy(acc, -cv[q], Wk);
    }
  }
  const T* av = aval<T>(P);
  const bool a_part = (wb != 0.0) || (lam != nullptr) || (e != nullptr);
  if (a_part && OWN) {
    const int q1 = P.A_rp[j + 1];
    int q = P.A_rp[j] + w.sub;
    for (; q + w.S < q1; q += 2 * w.S) {
      const int i0 = P.A_con[q], i1 = P.A_con[q + w.S];
      const int k0 = P.A_col[q], k1 = P.A_col[q + w.S];
      double c0 = wb * P.b[i0], c1 = wb * P.b[i1];
      if (lam) { c0 += wl * lam[i0]; c1 += wl * lam[i1]; }
      if (e) { c0 += we * e[i0]; c1 += we * e[i1]; }
      Frag<T> W0, W1;
      frag_load(W0, Wm, k0, ld, t);
      frag_load(W1, Wm, k1, ld, t);
      frag_axpy(acc, (T)(c0 * (double)av[q]), W0);
      frag_axpy(acc, (T)(c1 * (double)av[q + w.S]), W1);
    }
    if (q < q1) {
      const int i = P.A_con[q];
      double c = wb * P.b[i];
      if (lam) c += wl * lam[i];
      if (e) c += we * e[i];
      Frag<T> Wk;
      frag_load(Wk, Wm, P.A_col[q], ld, t);
      frag_axpy(acc, (T)(c * (double)av[q]), Wk);
    }
  } else if (a_part) {
    // 32 entries a round: lane l forms the weight of entry l once (FP64, whose instructions take 16
    // clocks of the SM each whatever the lanes do: with every sub-team forming its own, the
    // weights of 8 entries cost as much as those of 32 here), then sub-team s takes the entries
    // s, s + S, ...
    const int lane = threadIdx.x & 31;
    const int q1 = P.A_rp[j + 1];
    __syncwarp();
    for (int q0 = P.A_rp[j]; q0 < q1; q0 += 32) {
      int col = j;
      T c = T(0);
      if (q0 + lane < q1) {
        const int q = q0 + lane, i = P.A_con[q];
        col = P.A_col[q];
        double x = wb * P.b[i];
        if (lam) x += wl * lam[i];
        if (e) x += we * e[i];
        c = from_double<T>(x * to_double(av[q]));
      }
      const int rounds = min(32, q1 - q0);
      int s0 = 0;
      for (; rounds - s0 > w.S; s0 += H * w.S)
        spmm_entries<T, H>(Wm, ld, s0, rounds, col, c, w, acc);
      if (s0 < rounds) spmm_entries<T, 1>(Wm, ld, s0, rounds, col, c, w, acc);
    }
  }
  frag_warp_combine(acc, t.G);
  if (gamma != T(0)) {
    Frag<T> Wj;
    frag_load(Wj, Wm, j, ld, t);
    frag_axpy(acc, gamma, Wj);
  }
  out = acc;
}

// hessian_row_q with the whole warp (entries split across sub-teams); out in every lane
template <typename T>
__device__ void hessian_row_q_warp(const DevProblem& P, const T* Wm, int ld, int j,
                                   const Frag<T>& Pj, const double* q, T rho, T gamma,
                                   const WarpRow& w, Frag<T>& out) {
  const Team& t = w.st;
  Frag<T> acc;
  frag_zero(acc);
  const T* av = aval<T>(P);
  for (int e = P.A_rp[j] + w.sub; e < P.A_rp[j + 1]; e += w.S) {
    Frag<T> Wk;
    frag_load(Wk, Wm, P.A_col[e], ld, t);
    frag_axpy(acc, av[e] * (T)q[P.A_con[e]], Wk);
  }
  frag_warp_combine(acc, t.G);
#pragma unroll
  for (int kk = 0; kk < KMAX; ++kk)
#pragma unroll
    for (int ee = 0; ee < CHUNK; ++ee) out.v[kk][ee] = fma(rho, acc.v[kk][ee], gamma * Pj.v[kk][ee]);
}

}  // namespace lorads
