// bandcg.cuh -- the band solve (-Delta_{S,h}) w = f - mean: conjugate gradients on the compact
// band, preconditioned by one aggregation-multigrid V-cycle, one launch per solve.
//
// What bounds it: latency.  An iteration is some twenty dependent phases over a few thousand to
// a million nodes, so its time is the barriers between the phases, the load latencies inside
// them and, on this part, every FP64 instruction (an SM issues 2 FP64 operations per clock: one
// warp instruction holds its pipe for 64 clocks, a block-wide FP64 shuffle reduction of 1024
// threads takes 1.5 us).  Hence
//   * three engines, the same arithmetic:
//       cluster  one thread-block cluster holds the whole solve in shared memory (matrix,
//                vectors, all levels); neighbours are read through distributed shared memory and
//                phases are separated by the cluster barrier (0.3 us; 0.8 us when global stores
//                have to be flushed, which is why no phase of an iteration stores to global);
//       grid     up to one block per SM, vectors in global memory (L2), each block's share of the
//                matrix cached in shared memory where it fits, a grid barrier (1.2 us) between
//                phases;
//       hybrid   the grid engine on clusters: the finest level(s) as there, and every cluster runs
//                the coarser ones on a copy of its own, as the cluster engine would;
//   * levels of at most kCgLocal nodes run in every block on its own copy in shared memory, so
//     the small levels cost block barriers only and their result needs no broadcast;
//   * reductions over threads and scalars of the FP32 form are double-float (FP32 pipes; solved in
//     units of a power of two where (b,b) would leave FP32's range), and the FP64 form's scalars
//     are formed by one warp and handed to the block through shared memory;
//   * the V-cycle runs in FP32 in both forms.  It only shapes the search directions: in the FP64
//     form the residual, the operator, the iterates and the dot products are FP64, the residual
//     is scaled by a power of two into FP32 range first, and the solve stops on the same FP64
//     residual as before.
// Level l's unknowns are stored compactly (see the multigrid notes in kernels.cuh); block k owns
// nodes [k n, (k + 1) n) of every distributed level.
#pragma once
#include "df32.cuh"
#include "kernels.cuh"

namespace etd {

constexpr int kCgThreads = 1024;
constexpr int kCgLocal = 384;          // largest level that every block solves on its own copy: cluster
constexpr int kCgLocalGrid = 1024;     // engine (0.35 us a phase against 0.5 us distributed), grid engine (against 1.9 us)
constexpr int kCgMaxBlocks = 256;      // stride of the per-block partial sums
constexpr int kCgSmem = 222 * 1024;    // dynamic shared memory of a block (one block per SM)
constexpr int kCgSmemBig = 140 * 1024; // grid engine, bands whose finest matrix does not fit: the rest is L1

__device__ __forceinline__ float2 make_uw(float u, float w) { return make_float2(u, w); }
__device__ __forceinline__ double2 make_uw(double u, double w) { return make_double2(u, w); }

// ---- wide scalars: double-float for FP32 storage, FP64 otherwise ---------------------------
__device__ __forceinline__ double wide_d(double a) { return a; }
__device__ __forceinline__ double wide_d(dfloat a) { return (double)a.hi + (double)a.lo; }
__device__ __forceinline__ double wdiv(double a, double b) { return a / b; }
__device__ __forceinline__ dfloat wdiv(dfloat a, dfloat b) {  // quotient to about 2^-46
  const float q = a.hi / b.hi;
  const dfloat r = a - b * dfloat(q);
  const float q2 = r.hi / b.hi;
  return dfloat(q) + dfloat(q2);
}
__device__ __forceinline__ bool wpos(double a) { return a > 0.0; }
__device__ __forceinline__ bool wpos(dfloat a) { return a.hi > 0.0f; }
__device__ __forceinline__ float wnear(dfloat a) { return to_float(a); }
__device__ __forceinline__ double wnear(double a) { return a; }
__device__ __forceinline__ double shfl_dn(double v, int o) { return __shfl_down_sync(0xffffffffu, v, o); }
__device__ __forceinline__ dfloat shfl_dn(dfloat v, int o) {
  return dfloat(__shfl_down_sync(0xffffffffu, v.hi, o), __shfl_down_sync(0xffffffffu, v.lo, o));
}
template <typename W> __device__ __forceinline__ W warp_sum_w(W v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v = v + shfl_dn(v, o);
  return v;
}

// ---- right-hand sides f of the band solve, in the wide type --------------------------------
enum { RHS_FIELD = 0, RHS_GU = 1, RHS_GF = 2 };
template <typename T> struct Rhs {
  using W = typename WideOf<T>::type;
  int kind;
  const T* a;      // RHS_FIELD: f
  const T* G;      // RHS_GU: G (u - ubar), the coupled nonlocal operand (Eq. (1.2));
  const T* u;      // RHS_GF: G f(u), the fixed-model operand (Eq. (2.16))
  double ubar;
  Ubar<T> ub;      // ubar split into hi + lo in FP32
  __device__ W operator()(long long p) const {
    if (kind == RHS_FIELD) return W(a[p]);
    if constexpr (sizeof(T) == 4) {
      if (kind == RHS_GU) return dfloat(G[p]) * (dfloat(u[p]) - dfloat(ub.hi, ub.lo));
      return dfloat(G[p]) * dfloat(find(u[p]));
    } else {
      if (kind == RHS_GU) return G[p] * (u[p] - ubar);
      return G[p] * find(u[p]);
    }
  }
};

// Initial guess of a band solve, x0 = a + cb b + cc c over the band (b, c may be null), from
// earlier solutions kept on the full grid; the solution is also written to hist (if set).
template <typename T> struct CGGuess {
  const T* a;
  const T* b;
  const T* c;
  T cb, cc;
  T* hist;
};

// One multigrid level (device arrays; level 0 is the band itself).
struct MGL {
  const int* cnt;      // node count (device)
  const float* c;      // couplings c[f * cap + i]
  const int* nb;       // neighbour node of each face (i itself when absent)
  const float* idg;    // inverse diagonal
  int cap;
  const int* agg;      // parent node on level l+1 (l < nlev-1)
  const int* child;    // child[k * cap + I]: node of level l-1 in sub-cell k, -1 if none (l >= 1)
  float *b, *e, *o, *t;
};
struct MGP {
  int nlev;            // 1 = plain Jacobi
  int csweeps;         // Jacobi sweeps on the coarsest level (even)
  int nu;              // pre- and post-smoothing sweeps (1 or 2)
  float w1, w2;        // Jacobi weights of the first and second sweep (one Chebyshev pair)
  float alpha;         // over-correction of the coarse-grid correction
  const __half* c16;   // level-0 couplings in FP16 for the sweeps after the first (FP32 form; else null)
  MGL L[kMGMax];
};

// Shared-memory layout of a block, from the level counts alone (once per band).
// Distributed levels l < lc: block k owns nodes [k n[l], (k + 1) n[l]); local levels l >= lc are
// held whole by every block.
struct CGLayout {
  int cnt[kMGMax];
  int lg;              // levels below lg are spread over all blocks, [lg, lc) over each cluster
  int lc;
  int n[kMGMax];       // nodes per block of a distributed level (a multiple of 32)
  int mat[kMGMax];     // byte offset of the cached matrix (distributed: c, nb code, idg, child code;
                       // local: c, idg, nb, child), -1: read from global memory
  int vec[kMGMax];     // byte offset of b, e, o, t (levels of a cluster, and local levels)
  int cgv;             // byte offset of x, p, q and (FP64) r (cluster engine)
  int c64;             // byte offset of the FP64 couplings, -1: read from global memory
  int agg;             // byte offset of the parents of level lc - 1's own nodes (16-bit), -1: global
  int par;             // hybrid: byte offset of the parent codes of level lg - 1's own nodes
  int lchild;          // byte offset of level lc's child codes
  int bytes;           // what the layout needs; more than `smem`: it does not fit
};
enum { CG_GRID = 0, CG_CLUSTER = 1, CG_HYBRID = 2 };
// Fills y from y.cnt for K blocks in clusters of KC.  Cluster: everything has to fit; hybrid: the
// levels of the clusters have to; matrices of the grid's levels are cached while there is room,
// the finest level first (it takes five of the phases).
__host__ __device__ inline void cg_layout(CGLayout& y, int nlev, int K, int KC, int tsize, int mode, int smem) {
  int at = 0;
  auto take = [&at](int b) {
    const int o = at;
    at += (b + 15) & ~15;
    return o;
  };
  int lc = nlev;
  while (lc > 1 && y.cnt[lc - 1] <= (mode == CG_GRID ? kCgLocalGrid : kCgLocal)) --lc;
  // local levels that would not fit go back to the distributed ones
  for (int b = 0; lc < nlev; ++lc, b = 0) {
    for (int l = lc; l < nlev; ++l) b += 72 * y.cnt[l] + 64;
    if (b + 16 * y.cnt[lc] <= smem) break;
  }
  y.lc = lc;
  y.agg = y.lchild = y.cgv = y.c64 = y.par = -1;
  y.bytes = smem + 1;
  int lg = mode == CG_CLUSTER ? 0 : lc;
  if (mode == CG_HYBRID) {
    // the first level from which a cluster holds all the rest (16 + 84 B a node, local levels and
    // the finer level's parent codes beside them)
    int room = smem - 8192;
    for (int l = lc; l < nlev; ++l) room -= 72 * y.cnt[l] + 64;
    if (lc < nlev) room -= 16 * y.cnt[lc];
    lg = lc;
    for (int l = lc - 1; l >= 1; --l) {
      const int n = ((y.cnt[l] + KC - 1) / KC + 31) & ~31;
      if (n > room / 100) break;
      room -= 100 * n;
      if (4 * ((y.cnt[l - 1] + K - 1) / K + 31) <= room) lg = l;
    }
    if (lg >= lc || lg >= nlev - 1) return;   // nothing for the clusters to do
  }
  y.lg = lg;
  for (int l = 0; l < lc; ++l) {
    const int k = l < lg ? K : KC;
    y.n[l] = ((y.cnt[l] + k - 1) / k + 31) & ~31;
  }
  if (lc < nlev) {
    for (int l = lc; l < nlev; ++l) {
      const int m = y.cnt[l];
      y.vec[l] = take(16 * m);
      y.mat[l] = take((l > lc ? 56 : 40) * m);
    }
    y.lchild = take(32 * y.cnt[lc]);
  }
  for (int l = lg; l < lc; ++l) {
    const int n = y.n[l];
    if (n > smem / 52) return;   // more than a block holds (and no overflow below)
    y.vec[l] = take(16 * n);
    if (l == 0) y.cgv = take((tsize == 4 ? 3 : 4) * tsize * n);
    y.mat[l] = take((l > 0 ? 84 : 52) * n);
    if (l == 0 && tsize == 8) y.c64 = take(48 * n);
  }
  if (mode == CG_HYBRID) y.par = take(4 * y.n[lg - 1]);
  if (lc < nlev && lc > lg && mode != CG_GRID) y.agg = take(2 * y.n[lc - 1]);
  for (int l = 0; l < lg; ++l) {
    const int n = y.n[l], per = l > 0 ? 84 : 52;
    y.mat[l] = y.vec[l] = -1;
    if (n > smem / 52) continue;
    if (at + per * n <= smem) y.mat[l] = take(per * n);
    if (l == 0 && tsize == 8 && at + 48 * n <= smem) y.c64 = take(48 * n);
  }
  if (mode == CG_GRID && lc < nlev && at + 2 * y.n[lc - 1] <= smem) y.agg = take(2 * y.n[lc - 1]);
  y.bytes = at;
}

struct CGCtl2 {
  CGCtl c;
  const CGLayout* lay;   // this engine's layout
  const CGLayout* other; // sel & 2: the layout of the engine that goes first
  double* part;          // per-block partial sums (grid, hybrid), kCgMaxBlocks per slot
  int sel;               // 1: run only if this layout fits; 2: only if the other one does not
  int KC;                // blocks of a cluster
};

// Layouts of a band: [0] the cluster engine's, [1] the grid engine's, [2] the hybrid engine's in
// clusters of kCgCluster.
constexpr int kCgCluster = 16;
struct CGCounts {
  const int* cnt[kMGMax];
};
// One warp per layout (the first three warps of the block).
__device__ inline void cg_layouts(const int* const* cnt, int nlev, int tsize, int clK, int gridK, int hybK, int gsmem,
                                  CGLayout* out) {
  __shared__ CGLayout y[3];
  const int e = threadIdx.x >> 5, l = threadIdx.x & 31;
  if (e >= 3) return;
  if (l < kMGMax) y[e].cnt[l] = l < nlev ? *cnt[l] : 0;
  __syncwarp();
  if (l == 0) {
    if (e == 0) cg_layout(y[e], nlev, clK, clK, tsize, CG_CLUSTER, kCgSmem);
    if (e == 1) cg_layout(y[e], nlev, gridK, 1, tsize, CG_GRID, gsmem);
    if (e == 2) cg_layout(y[e], nlev, hybK, kCgCluster, tsize, CG_HYBRID, kCgSmem);
  }
  __syncwarp();
  for (int k = l; k < (int)(sizeof(CGLayout) / 4); k += 32)
    reinterpret_cast<int*>(out + e)[k] = reinterpret_cast<const int*>(&y[e])[k];
}
static __global__ void k_cg_layout(CGCounts cs, int nlev, int tsize, int clK, int gridK, int hybK, int gsmem,
                                   CGLayout* out) {
  cg_layouts(cs.cnt, nlev, tsize, clK, gridK, hybK, gsmem, out);
}

// ---- shared-memory access by 32-bit address -------------------------------------------------
__device__ __forceinline__ uint32_t mapa_u32(uint32_t a, uint32_t rank) {
  uint32_t r;
  asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(rank));
  return r;
}
__device__ __forceinline__ float lds_f(uint32_t a) {
  float v;
  asm volatile("ld.shared.f32 %0, [%1];" : "=f"(v) : "r"(a));
  return v;
}
__device__ __forceinline__ unsigned lds_u(uint32_t a) {
  unsigned v;
  asm volatile("ld.shared.u32 %0, [%1];" : "=r"(v) : "r"(a));
  return v;
}
__device__ __forceinline__ unsigned lds_h(uint32_t a) {
  unsigned short v;
  asm volatile("ld.shared.u16 %0, [%1];" : "=h"(v) : "r"(a));
  return v;
}
__device__ __forceinline__ void sts_f(uint32_t a, float v) {
  asm volatile("st.shared.f32 [%0], %1;" ::"r"(a), "f"(v) : "memory");
}
__device__ __forceinline__ float ld_dsm(uint32_t a) {
  float v;
  asm volatile("ld.shared::cluster.f32 %0, [%1];" : "=f"(v) : "r"(a));
  return v;
}
__device__ __forceinline__ void st_dsm(uint32_t a, float v) {
  asm volatile("st.shared::cluster.f32 [%0], %1;" ::"r"(a), "f"(v) : "memory");
}
__device__ __forceinline__ double ld_dsm8(uint32_t a) {
  unsigned long long v;
  asm volatile("ld.shared::cluster.u64 %0, [%1];" : "=l"(v) : "r"(a));
  return __longlong_as_double((long long)v);
}

// Vectors of the grid engine: weak loads through L1.  A phase reads nothing that another block
// writes in it, and the acquire of the barrier before it drops what L1 held; the y neighbours
// of a block's nodes are then mostly L1 hits (at 1 M nodes a sweep is bound by L2 traffic).
__device__ __forceinline__ float ldg_w(const float* p) {
  float v;
  asm volatile("ld.global.f32 %0, [%1];" : "=f"(v) : "l"(p));
  return v;
}

enum { V_B = 0, V_E = 1, V_O = 2, V_T = 3 };

// A distributed level as a block sees it: own nodes by local index s, neighbours and children by
// code (cluster: shared::cluster address of the element in the level's first vector; grid: node).
template <bool CL> struct LevD;
template <> struct LevD<true> {   // everything in shared memory
  int n, st;                      // own nodes; bytes of one vector (4 times the allocated nodes)
  uint32_t mat, vec;
  __device__ float c(int f, int s, bool) const { return lds_f(mat + f * st + 4 * s); }
  __device__ unsigned nb(int f, int s) const { return lds_u(mat + (6 + f) * st + 4 * s); }
  __device__ float idg(int s) const { return lds_f(mat + 12 * st + 4 * s); }
  __device__ unsigned child(int k, int s) const { return lds_u(mat + (13 + k) * st + 4 * s); }
  __device__ float own(int v, int s) const { return lds_f(vec + v * st + 4 * s); }
  __device__ void put(int v, int s, float x) const { sts_f(vec + v * st + 4 * s, x); }
  __device__ float nbr(int v, unsigned code) const { return ld_dsm(code + v * st); }
  __device__ void put_nbr(int v, unsigned code, float x) const { st_dsm(code + v * st, x); }
};
template <> struct LevD<false> {  // vectors in global memory, the matrix there or in shared memory
  int n, cs;
  const float* pc;
  const unsigned* pnb;
  const float* pidg;
  const unsigned* pch;
  // streamed level 0 of the FP32 form: couplings of the later sweeps; packed form (null: not)
  const __half* c16;
  const uint4* pk;                // FP16 couplings and the FP32 inverse diagonal
  const short4* nd;               // y and z neighbours as offsets (x neighbours are s - 1, s + 1)
  float* g[4];                    // the whole vectors
  int lb;                         // first own node
  __device__ float c(int f, int s, bool half) const {
    return half && c16 ? __half2float(c16[f * cs + s]) : pc[f * cs + s];
  }
  __device__ unsigned nb(int f, int s) const { return pnb[f * cs + s]; }
  __device__ float idg(int s) const { return pk ? __uint_as_float(pk[s].w) : pidg[s]; }
  __device__ unsigned child(int k, int s) const { return pch[k * cs + s]; }
  __device__ float own(int v, int s) const { return ldg_w(g[v] + lb + s); }
  __device__ void put(int v, int s, float x) const { g[v][lb + s] = x; }
  __device__ float nbr(int v, unsigned code) const { return ldg_w(g[v] + code); }
  __device__ void put_nbr(int v, unsigned code, float x) const { g[v][code] = x; }
};
// Couplings and neighbour codes of node s.
__device__ __forceinline__ void faces(const LevD<true>& A, int s, bool, float (&c)[6], unsigned (&j)[6]) {
#pragma unroll
  for (int f = 0; f < 6; ++f) j[f] = A.nb(f, s);
#pragma unroll
  for (int f = 0; f < 6; ++f) c[f] = A.c(f, s, false);
}
__device__ __forceinline__ void faces(const LevD<false>& A, int s, bool half, float (&c)[6], unsigned (&j)[6]) {
  if (A.nd) {
    const short4 d = A.nd[s];
    const unsigned i = (unsigned)(A.lb + s);
    if (half) {
      const uint4 p = A.pk[s];
      const unsigned w[3] = {p.x, p.y, p.z};
#pragma unroll
      for (int f = 0; f < 3; ++f) {
        const float2 v = __half22float2(*reinterpret_cast<const __half2*>(&w[f]));
        c[2 * f] = v.x;
        c[2 * f + 1] = v.y;
      }
    } else {
#pragma unroll
      for (int f = 0; f < 6; ++f) c[f] = A.pc[f * A.cs + s];
    }
    j[0] = c[0] != 0.0f ? i + 1 : i;
    j[1] = c[1] != 0.0f ? i - 1 : i;
    j[2] = i + d.x;
    j[3] = i + d.y;
    j[4] = i + d.z;
    j[5] = i + d.w;
    return;
  }
#pragma unroll
  for (int f = 0; f < 6; ++f) j[f] = A.nb(f, s);
#pragma unroll
  for (int f = 0; f < 6; ++f) c[f] = A.c(f, s, half);
}
// sum over faces of c (v_i - v_j)
template <class L> __device__ __forceinline__ float lap_d(const L& A, int vec, int s, float vi, bool half) {
  unsigned j[6];   // loads keep their order: all the codes, then all the values
  float c[6], x[6];
  faces(A, s, half, c, j);
#pragma unroll
  for (int f = 0; f < 6; ++f) x[f] = A.nbr(vec, j[f]);
  float a = 0;
#pragma unroll
  for (int f = 0; f < 6; ++f) a += c[f] * (vi - x[f]);
  return a;
}
// sum of a vector over a node's children (codes ~0u: none)
template <class N, class L> __device__ __forceinline__ float child_sum(const N& A, const L& F, int vec, int s) {
  unsigned ch[8];
  float x[8];
#pragma unroll
  for (int k = 0; k < 8; ++k) ch[k] = A.child(k, s);
#pragma unroll
  for (int k = 0; k < 8; ++k) x[k] = ch[k] != ~0u ? F.nbr(vec, ch[k]) : 0.0f;
  return ((x[0] + x[1]) + (x[2] + x[3])) + ((x[4] + x[5]) + (x[6] + x[7]));
}

// A local level: neighbours and children as byte offsets into a vector (0xffff: no child).
struct LevL {
  int n;
  uint32_t mat, vec;
  __device__ uint32_t v(int k, int s) const { return vec + 4 * (k * n + s); }
  __device__ float idg(int s) const { return lds_f(mat + 24 * n + 4 * s); }
  __device__ unsigned child(int k, int s) const { return lds_h(mat + 40 * n + 2 * (k * n + s)); }
  __device__ float lap(int k, int s, float vi) const {
    unsigned j[6];
    float c[6], x[6];
#pragma unroll
    for (int f = 0; f < 6; ++f) j[f] = lds_h(mat + 28 * n + 2 * (f * n + s));
#pragma unroll
    for (int f = 0; f < 6; ++f) c[f] = lds_f(mat + 4 * (f * n + s));
#pragma unroll
    for (int f = 0; f < 6; ++f) x[f] = lds_f(vec + 4 * k * n + j[f]);
    float a = 0;
#pragma unroll
    for (int f = 0; f < 6; ++f) a += c[f] * (vi - x[f]);
    return a;
  }
};

template <typename T> struct CGShared {
  using W = typename WideOf<T>::type;
  CGLayout lay;
  LevD<false> dg[kMGMax];   // levels of the grid
  LevD<true> dc[kMGMax];    // levels of a cluster
  alignas(8) W part[6];   // this block's partial sums (cluster engine)
  W ws[2][32];
  W gamma, alpha;         // written and read by one thread
  double bb, rr, tol2;
  T a, bt, sc;            // sc: FP64, of the residual's FP32 copy; FP32, of the whole solve
  float pre;
  double mean;
  int go, range, zero;
  double csh[kCompShared];
};

// Per-node work of a phase: `load` reads everything node s needs and returns its new values,
// `store` writes them; blocks with more than one node per thread have two nodes' loads in flight.
// `mid` runs once, after the first nodes' loads and before their stores, in every thread.
template <int U, typename Load, typename Mid, typename Store>
__device__ __forceinline__ void nodes_u(int n, Load&& load, Mid&& mid, Store&& store) {
  decltype(load(0)) r[U];
  int s0 = threadIdx.x;
  if (s0 < n) {
#pragma unroll
    for (int u = 0; u < U; ++u) r[u] = load(min(s0 + u * kCgThreads, n - 1));
  }
  mid();
  while (s0 < n) {
#pragma unroll
    for (int u = 0; u < U; ++u)
      if (s0 + u * kCgThreads < n) store(s0 + u * kCgThreads, r[u]);
    s0 += U * kCgThreads;
    if (s0 >= n) break;
#pragma unroll
    for (int u = 0; u < U; ++u) r[u] = load(min(s0 + u * kCgThreads, n - 1));
  }
}
template <typename Load, typename Mid, typename Store>
__device__ __forceinline__ void nodes(int n, Load&& load, Mid&& mid, Store&& store) {
  if (n <= kCgThreads) nodes_u<1>(n, load, mid, store);
  else nodes_u<2>(n, load, mid, store);
}
template <typename Load, typename Store> __device__ __forceinline__ void nodes(int n, Load&& load, Store&& store) {
  nodes(n, load, [] {}, store);
}

__device__ __forceinline__ void cluster_barrier() {
  asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
  asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}

template <typename T, int MODE> struct CGSolve {
  using W = typename WideOf<T>::type;
  static constexpr bool CL = MODE == CG_CLUSTER;
  CGShared<T>& S;
  const CGCtl2& q;
  const MGP& mg;
  int rank, K;
  uint32_t dyn;   // address of the dynamic shared memory

  // Barrier over a cluster: the hardware barrier (it does not spin; in the cluster engine a budget
  // below zero still gives up, at the first one, before anything is read through the cluster).
  __device__ bool cbar() const {
    cluster_barrier();
    if (CL && q.c.budget < 0) {
      if (threadIdx.x == 0) atomicCAS(q.c.status, 0, 6);
      return false;
    }
    return true;
  }
  // Barrier over all blocks of the solve: the arrival counter of grid_sync (a flag per block that
  // every block polls measured 2 to 5 us against its 1.3 us at 152 blocks: the polls' traffic).
  // One that fails has failed in every block.
  __device__ bool bar() const {
    if constexpr (CL) return cbar();
    else return grid_sync(q.c);
  }
  // Block sum of v into this block's partial `slot`; warps from nact on hold zero.  The caller
  // takes a barrier before total(), and between two posts of slots of the same parity.
  __device__ void post(W v, int slot, int nact) const {
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    if (wid < nact) {
      v = warp_sum_w(v);
      if (lane == 0) S.ws[slot & 1][wid] = v;
    }
    __syncthreads();
    if (wid == 0) {
      W t = lane < nact ? S.ws[slot & 1][lane] : W(0);
      t = warp_sum_w(t);
      if (lane == 0) {
        if constexpr (CL) S.part[slot] = t;
        else reinterpret_cast<W*>(q.part)[slot * kCgMaxBlocks + rank] = t;
      }
    }
  }
  // The sum over the blocks, for a whole warp; lane 0 has it.
  __device__ W total(int slot) const {
    W t(0);
    for (int k = threadIdx.x & 31; k < K; k += 32) {
      double raw;
      if constexpr (CL) raw = ld_dsm8(mapa_u32(smem_u32(&S.part[slot]), k));
      else raw = __ldcg(q.part + slot * kCgMaxBlocks + k);
      if constexpr (sizeof(T) == 8) t = t + raw;
      else t = t + dfloat(__int_as_float(__double2loint(raw)), __int_as_float(__double2hiint(raw)));
    }
    return warp_sum_w(t);
  }
  // total() and what follows from it are one warp's work; the last warp has the fewest nodes
  static __device__ bool scalar_warp() { return threadIdx.x >= kCgThreads - 32; }
  static __device__ bool scalar_lane() { return threadIdx.x == kCgThreads - 32; }

  __device__ LevL loc(int l) const {
    return LevL{S.lay.cnt[l], dyn + (uint32_t)S.lay.mat[l], dyn + (uint32_t)S.lay.vec[l]};
  }

  // The V-cycle for the level-0 right-hand side b, with e = w1 D^-1 b already stored and both
  // visible to every block: o = M^-1 b.  Residuals of the pre-sweeps are carried algebraically:
  // r1 = b - A e1, d = w2 D^-1 r1, e2 = e1 + d, r2 = r1 - A d; r2 is gathered into the parent
  // aggregates (the restriction of piecewise-constant P), and a level's correction is added to
  // its children's e by the thread that computed it (or, where the coarser level is this block's
  // or its cluster's own copy, by the child's).  `before` runs before the first phase (the
  // scalar warp forms the stopping test there) and S.go is looked at after the first barrier.
  // `dot` sees every own (node, o).  Returns -1 if a barrier gave up, 1 if the test stopped the
  // solve, 0 with o complete except for the barrier that the caller takes.
  template <typename Before, typename Dot> __device__ int vcycle(Before&& before, Dot&& dot) const {
    const int nlev = mg.nlev, lc = S.lay.lc, last = nlev - 1, ld = lc < last ? lc : last;
    const int lg = MODE == CG_GRID ? lc : (MODE == CG_CLUSTER ? 0 : S.lay.lg);
    const auto gb = [&] { return bar(); };
    const auto cb = [&] { return cbar(); };
    const auto none = [](int, float) {};
    before();
    if (nlev == 1) {
      __syncthreads();
      if (!S.go) return 1;
      auto jac = [&](auto L) {
        nodes(
            L.n, [&](int s) { return L.idg(s) * L.own(V_B, s); },
            [&](int s, float o) {
              L.put(V_O, s, o);
              dot(s, o);
            });
      };
      if constexpr (CL) jac(S.dc[0]);
      else jac(S.dg[0]);
      return 0;
    }
    // down
    if constexpr (MODE != CG_CLUSTER) {
      for (int l = 0; l < ld && l < lg; ++l) {
        const LevD<false> L = S.dg[l];
        if (!sweep1(L, gb)) return -1;
        if (l == 0 && !S.go) return 1;
        if (!sweep2(L, gb)) return -1;
        if (l + 1 < lg && !gather(LevD<false>(S.dg[l + 1]), L, gb)) return -1;
      }
    }
    if constexpr (MODE != CG_GRID) {
      if constexpr (MODE == CG_HYBRID) {
        if (!gather(LevD<true>(S.dc[lg]), LevD<false>(S.dg[lg - 1]), cb)) return -1;
      }
      for (int l = lg; l < ld; ++l) {
        const LevD<true> L = S.dc[l];
        if (!sweep1(L, cb)) return -1;
        if (l == 0 && !S.go) return 1;
        if (!sweep2(L, cb)) return -1;
        if (l + 1 < lc && !gather(LevD<true>(S.dc[l + 1]), L, cb)) return -1;
      }
    }
    // the coarsest levels
    bool ok;
    if constexpr (MODE == CG_GRID) ok = bottom(S.dg, gb);
    else ok = bottom(S.dc, cb);
    if (!ok) return -1;
    // up
    if constexpr (MODE != CG_GRID) {
      for (int l = ld - 1; l >= lg; --l) {
        const LevD<true> L = S.dc[l];
        if (CL && l == 0) {
          if (!post_sweeps(L, cb, dot)) return -1;
          continue;
        }
        if (!post_sweeps(L, cb, none)) return -1;
        if (l > lg) push(L, LevD<true>(S.dc[l - 1]));
        if (!cbar()) return -1;
      }
      if constexpr (MODE == CG_HYBRID) {
        // the cluster's correction to this block's own nodes of level lg - 1
        const LevD<false> L = S.dg[lg - 1];
        const LevD<true> N = S.dc[lg];
        const uint32_t par = dyn + (uint32_t)S.lay.par;
        const float al = mg.alpha;
        nodes(
            L.n, [&](int s) { return L.own(V_E, s) + al * N.nbr(V_O, lds_u(par + 4 * s)); },
            [&](int s, float e) { L.put(V_E, s, e); });
        if (!bar()) return -1;
      }
    }
    if constexpr (MODE != CG_CLUSTER) {
      for (int l = (lg < ld ? lg : ld) - 1; l >= 0; --l) {
        const LevD<false> L = S.dg[l];
        if (l == 0) {
          if (!post_sweeps(L, gb, dot)) return -1;
          continue;
        }
        if (!post_sweeps(L, gb, none)) return -1;
        push(L, LevD<false>(S.dg[l - 1]));
        if (!bar()) return -1;
      }
    }
    return 0;
  }

  // r1 = b - A e into o, d = w2 D^-1 r1 into t.
  template <class L, class B> __device__ __forceinline__ bool sweep1(const L& A, B&& b) const {
    const float w2 = mg.w2;
    nodes(
        A.n,
        [&](int s) {
          const float r1 = A.own(V_B, s) - lap_d(A, V_E, s, A.own(V_E, s), false);
          return make_float2(r1, w2 * A.idg(s) * r1);
        },
        [&](int s, float2 r) {
          A.put(V_O, s, r.x);
          A.put(V_T, s, r.y);
        });
    return b();
  }
  // r2 = r1 - A d into o, e += d.
  template <class L, class B> __device__ __forceinline__ bool sweep2(const L& A, B&& b) const {
    if (mg.nu != 2) return true;
    nodes(
        A.n,
        [&](int s) {
          const float d = A.own(V_T, s);
          return make_float2(A.own(V_O, s) - lap_d(A, V_T, s, d, true), A.own(V_E, s) + d);
        },
        [&](int s, float2 r) {
          A.put(V_O, s, r.x);
          A.put(V_E, s, r.y);
        });
    return b();
  }
  // The residual of level F into the right-hand side of the next level N, and its first sweep.
  template <class N, class L, class B> __device__ __forceinline__ bool gather(const N& A, const L& F, B&& b) const {
    const float w1 = mg.w1;
    nodes(
        A.n,
        [&](int s) {
          const float r = child_sum(A, F, V_O, s);
          return make_float2(r, w1 * A.idg(s) * r);
        },
        [&](int s, float2 r) {
          A.put(V_B, s, r.x);
          A.put(V_E, s, r.y);
        });
    return b();
  }
  // The sweeps after the coarse-grid correction; the barrier after the last is the caller's.
  template <class L, class B, class Dot>
  __device__ __forceinline__ bool post_sweeps(const L& A, B&& b, Dot&& dot) const {
    const bool two = mg.nu == 2;
    const float ws = two ? mg.w2 : mg.w1, w1 = mg.w1;
    const int out = two ? V_T : V_O;
    nodes(
        A.n,
        [&](int s) {
          const float e = A.own(V_E, s);
          return e + ws * A.idg(s) * (A.own(V_B, s) - lap_d(A, V_E, s, e, true));
        },
        [&](int s, float o) {
          A.put(out, s, o);
          if (!two) dot(s, o);
        });
    if (!two) return true;
    if (!b()) return false;
    nodes(
        A.n,
        [&](int s) {
          const float t = A.own(V_T, s);
          return t + w1 * A.idg(s) * (A.own(V_B, s) - lap_d(A, V_T, s, t, true));
        },
        [&](int s, float o) {
          A.put(V_O, s, o);
          dot(s, o);
        });
    return true;
  }
  // The local levels and their correction to level lc - 1, or the sweeps of a coarsest level that
  // is distributed and its push; ends with a barrier.
  template <class L, class B> __device__ bool bottom(const L* d, B&& b) const {
    const int nlev = mg.nlev, lc = S.lay.lc, last = nlev - 1;
    if (lc < nlev) {
      const L A = d[lc - 1];
      local_cycle(A);
      const LevL C = loc(lc);
      const float al = mg.alpha;
      const int a16 = S.lay.agg;
      // blocks of the level's tier: the whole grid, or this cluster
      const int tr = MODE == CG_HYBRID ? rank % q.KC : rank;
      const int* agg = mg.L[lc - 1].agg + (size_t)tr * S.lay.n[lc - 1];
      nodes(
          A.n,
          [&](int s) {
            const int p = a16 >= 0 ? (int)lds_h(dyn + a16 + 2 * s) : agg[s];
            return A.own(V_E, s) + al * lds_f(C.v(V_O, p));
          },
          [&](int s, float e) { A.put(V_E, s, e); });
      return b();
    }
    const L A = d[last];   // e = w1 D^-1 b is the first sweep
    for (int k = 1; k < mg.csweeps; ++k) {
      const int src = (k & 1) ? V_E : V_O, dst = (k & 1) ? V_O : V_E;
      const float w = (k & 1) ? mg.w2 : mg.w1;
      nodes(
          A.n,
          [&](int s) {
            const float v = A.own(src, s);
            return v + w * A.idg(s) * (A.own(V_B, s) - lap_d(A, src, s, v, true));
          },
          [&](int s, float v) { A.put(dst, s, v); });
      if (!b()) return false;
    }
    push(A, d[last - 1]);
    return b();
  }

  // e += alpha o on the children of this block's nodes of level N (each node has one parent).
  template <class N, class L> __device__ void push(const N& A, const L F) const {
    for (int s = threadIdx.x; s < A.n; s += kCgThreads) {
      const float o = mg.alpha * A.own(V_O, s);
      unsigned ch[8];
      float e[8];
#pragma unroll
      for (int k = 0; k < 8; ++k) ch[k] = A.child(k, s);
#pragma unroll
      for (int k = 0; k < 8; ++k) e[k] = ch[k] != ~0u ? F.nbr(V_E, ch[k]) : 0.0f;
#pragma unroll
      for (int k = 0; k < 8; ++k)
        if (ch[k] != ~0u) F.put_nbr(V_E, ch[k], e[k] + o);
    }
  }

  // Levels lc .. nlev-1 on this block's own copy; level lc's right-hand side is gathered from the
  // residual o of level lc - 1.  One node per thread.  Only the warps that hold a node of level lc
  // take part (a named barrier), and from the first level of at most 32 nodes on one warp goes
  // alone: a phase is then a warp barrier and a few shared-memory latencies.  Ends with the
  // result o of level lc visible to the block.
  template <class L> __device__ void local_cycle(const L& F) const {
    const int nlev = mg.nlev, lc = S.lay.lc;
    const int s = threadIdx.x, nthr = (S.lay.cnt[lc] + 31) & ~31;
    if (s < nthr) {
      const LevL N = loc(lc);
      if (s < N.n) {
        const uint32_t lch = dyn + (uint32_t)S.lay.lchild + 4 * s;
        struct {
          uint32_t a;
          int n;
          __device__ unsigned child(int k, int) const { return lds_u(a + 4 * k * n); }
        } codes{lch, N.n};
        const float b = child_sum(codes, F, V_O, s);
        sts_f(N.v(V_B, s), b);
        sts_f(N.v(V_E, s), mg.w1 * N.idg(s) * b);
      }
      int lw = lc;
      while (lw < nlev && S.lay.cnt[lw] > 32) ++lw;
      auto sync = [&](bool blk) {
        if (blk) asm volatile("bar.sync 1, %0;" ::"r"(nthr) : "memory");
        else __syncwarp();
      };
      sync(lw > lc);
      const int lb = lw < nlev - 1 ? lw : nlev - 1;   // levels lc .. lb-1 by all of these warps
      for (int l = lc; l < lb; ++l) local_down(l, s, true, sync);
      if (lw >= nlev) {
        local_coarsest(s, true, sync);
      } else {
        if (s < 32) {
          for (int l = lb; l < nlev - 1; ++l) local_down(l, s, false, sync);
          local_coarsest(s, false, sync);
          for (int l = nlev - 2; l >= lb; --l) local_up(l, s, false, sync);
        }
        if (lb > lc) sync(true);
      }
      for (int l = lb - 1; l >= lc; --l) local_up(l, s, true, sync);
    }
    __syncthreads();
  }
  template <typename Sync> __device__ __forceinline__ void local_down(int l, int s, bool blk, Sync&& sync) const {
    const LevL L = loc(l), N = loc(l + 1);
    if (s < L.n) {
      const float r1 = lds_f(L.v(V_B, s)) - L.lap(V_E, s, lds_f(L.v(V_E, s)));
      sts_f(L.v(V_O, s), r1);
      sts_f(L.v(V_T, s), mg.w2 * L.idg(s) * r1);
    }
    sync(blk);
    if (mg.nu == 2) {
      if (s < L.n) {
        const float d = lds_f(L.v(V_T, s));
        sts_f(L.v(V_O, s), lds_f(L.v(V_O, s)) - L.lap(V_T, s, d));
        sts_f(L.v(V_E, s), lds_f(L.v(V_E, s)) + d);
      }
      sync(blk);
    }
    if (s < N.n) {
      unsigned ch[8];
      float x[8];
#pragma unroll
      for (int k = 0; k < 8; ++k) ch[k] = N.child(k, s);
#pragma unroll
      for (int k = 0; k < 8; ++k) x[k] = ch[k] != 0xffffu ? lds_f(L.v(V_O, 0) + ch[k]) : 0.0f;
      const float b = ((x[0] + x[1]) + (x[2] + x[3])) + ((x[4] + x[5]) + (x[6] + x[7]));
      sts_f(N.v(V_B, s), b);
      sts_f(N.v(V_E, s), mg.w1 * N.idg(s) * b);
    }
    sync(blk);
  }
  template <typename Sync> __device__ __forceinline__ void local_coarsest(int s, bool blk, Sync&& sync) const {
    const LevL L = loc(mg.nlev - 1);
    for (int k = 1; k < mg.csweeps; ++k) {
      const int src = (k & 1) ? V_E : V_O, dst = (k & 1) ? V_O : V_E;
      if (s < L.n) {
        const float v = lds_f(L.v(src, s));
        sts_f(L.v(dst, s), v + ((k & 1) ? mg.w2 : mg.w1) * L.idg(s) * (lds_f(L.v(V_B, s)) - L.lap(src, s, v)));
      }
      sync(blk);
    }
  }
  template <typename Sync> __device__ __forceinline__ void local_up(int l, int s, bool blk, Sync&& sync) const {
    const LevL L = loc(l), N = loc(l + 1);
    if (s < N.n) {
      const float o = mg.alpha * lds_f(N.v(V_O, s));
      unsigned ch[8];
      float e[8];
#pragma unroll
      for (int k = 0; k < 8; ++k) ch[k] = N.child(k, s);
#pragma unroll
      for (int k = 0; k < 8; ++k) e[k] = ch[k] != 0xffffu ? lds_f(L.v(V_E, 0) + ch[k]) : 0.0f;
#pragma unroll
      for (int k = 0; k < 8; ++k)
        if (ch[k] != 0xffffu) sts_f(L.v(V_E, 0) + ch[k], e[k] + o);
    }
    sync(blk);
    const bool two = mg.nu == 2;
    if (s < L.n) {
      const float e = lds_f(L.v(V_E, s));
      sts_f(L.v(two ? V_T : V_O, s), e + (two ? mg.w2 : mg.w1) * L.idg(s) * (lds_f(L.v(V_B, s)) - L.lap(V_E, s, e)));
    }
    sync(blk);
    if (two) {
      if (s < L.n) {
        const float t = lds_f(L.v(V_T, s));
        sts_f(L.v(V_O, s), t + mg.w1 * L.idg(s) * (lds_f(L.v(V_B, s)) - L.lap(V_T, s, t)));
      }
      sync(blk);
    }
  }
};

template <typename T, typename D> struct Trip {
  T p, q;
  D d;
};

enum { A_SUMF = 0, A_BB = 1, A_RR = 2, A_RU = 3, A_DU = 4, A_SUMX = 5, A_SLOTS = 6 };

// Conjugate gradients, Chronopoulos-Gear arrangement (the recurrence s = A p replaces the second
// matrix product of textbook CG), per iteration:
//   x += a p, r -= a s, rr = (r,r), b = r in FP32, e = w1 D^-1 b       | barrier, stop on rr
//   o = M^{-1} b, gamma = (r,o)                                        | barrier
//   w = A o, p = o + beta p, s = w + beta s, delta = (w,o)             | barrier
//   beta = gamma/gamma_old, a = gamma/(delta - beta gamma/a_old)
// Returns early where a barrier failed.
template <typename T, int MODE>
__device__ __forceinline__ void cg_block(const int* __restrict__ idx, const CGVec<T>& v, T* __restrict__ wfull,
                                         const Rhs<T>& rhs, const CGCtl2& q, const MGP& mg, const CGGuess<T>& gs,
                                         unsigned char* cg_dyn, CGShared<T>& S) {
  using W = typename WideOf<T>::type;
  constexpr bool CL = MODE == CG_CLUSTER;
  const int rank = blockIdx.x, K = gridDim.x, t0 = threadIdx.x;
  const CGCtl& c = q.c;
  const int M = S.lay.cnt[0];
  const uint32_t dyn = smem_u32(cg_dyn);
  const int na0 = S.lay.n[0], base = rank * na0;
  const int n0 = max(0, min(na0, M - base));
  const int lc = S.lay.lc, nlev = mg.nlev, lg = MODE == CG_GRID ? lc : (CL ? 0 : S.lay.lg);
  const int crank = MODE == CG_HYBRID ? rank % q.KC : rank;   // rank in the cluster
  if (t0 < lc) {
    const int l = t0, na = S.lay.n[l], lb = (l < lg ? rank : crank) * na, n = max(0, min(na, S.lay.cnt[l] - lb));
    const MGL& G = mg.L[l];
    if (l >= lg) {
      LevD<true>& L = S.dc[l];
      L.n = n;
      L.st = 4 * na;
      L.mat = dyn + (uint32_t)S.lay.mat[l];
      L.vec = dyn + (uint32_t)S.lay.vec[l];
    } else {
      LevD<false>& L = S.dg[l];
      L.n = n;
      L.lb = lb;
      L.c16 = nullptr;
      L.pk = nullptr;
      L.nd = nullptr;
      L.g[0] = G.b;
      L.g[1] = G.e;
      L.g[2] = G.o;
      L.g[3] = G.t;
      if (S.lay.mat[l] >= 0) {
        const unsigned char* m = cg_dyn + S.lay.mat[l];
        L.cs = na;
        L.pc = reinterpret_cast<const float*>(m);
        L.pnb = reinterpret_cast<const unsigned*>(m + 24 * na);
        L.pidg = reinterpret_cast<const float*>(m + 48 * na);
        L.pch = reinterpret_cast<const unsigned*>(m + 52 * na);
      } else {
        L.cs = G.cap;
        L.pc = G.c + lb;
        L.pnb = reinterpret_cast<const unsigned*>(G.nb) + lb;
        L.pidg = G.idg + lb;
        L.pch = l > 0 ? reinterpret_cast<const unsigned*>(G.child) + lb : nullptr;
        if (l == 0 && mg.c16) L.c16 = mg.c16 + lb;
        if (l == 0 && v.pk && *v.wide == 0) {
          L.pk = v.pk + lb;
          L.nd = v.nd + lb;
        }
      }
    }
  }
  __syncthreads();
  // Matrices into shared memory.  Code of node j of a level: the address of its element in the
  // level's first vector where a cluster holds it (j / na by a multiply, exact for the
  // j < 2^32 / na of a level that fits), else j.
  auto code = [&](int l, int j, unsigned mul) -> unsigned {
    if (MODE == CG_GRID || l < lg) return (unsigned)j;
    const unsigned na = (unsigned)S.lay.n[l], r = __umulhi((unsigned)j, mul);
    return mapa_u32(dyn + (uint32_t)S.lay.vec[l], r) + 4u * ((unsigned)j - r * na);
  };
  auto magic = [&](int l) { return 0xffffffffu / (unsigned)S.lay.n[l] + 1u; };
  for (int l = 0; l < lc; ++l) {
    if (S.lay.mat[l] < 0) continue;
    const MGL& G = mg.L[l];
    const int na = S.lay.n[l], lb = (l < lg ? rank : crank) * na, n = max(0, min(na, S.lay.cnt[l] - lb));
    const unsigned mul = magic(l), mulf = l > 0 ? magic(l - 1) : 0;
    unsigned char* m = cg_dyn + S.lay.mat[l];
    for (int s = t0; s < n; s += kCgThreads) {
#pragma unroll
      for (int f = 0; f < 6; ++f) {
        reinterpret_cast<float*>(m)[f * na + s] = G.c[f * G.cap + lb + s];
        reinterpret_cast<unsigned*>(m + 24 * na)[f * na + s] = code(l, G.nb[f * G.cap + lb + s], mul);
      }
      reinterpret_cast<float*>(m + 48 * na)[s] = G.idg[lb + s];
      if (l > 0) {
#pragma unroll
        for (int k = 0; k < 8; ++k) {
          const int ch = G.child[k * G.cap + lb + s];
          reinterpret_cast<unsigned*>(m + 52 * na)[k * na + s] = ch < 0 ? ~0u : code(l - 1, ch, mulf);
        }
      }
    }
  }
  for (int l = lc; l < nlev; ++l) {
    const MGL& G = mg.L[l];
    const int m = S.lay.cnt[l];
    const unsigned mulf = magic(lc - 1);
    unsigned char* p = cg_dyn + S.lay.mat[l];
    for (int s = t0; s < m; s += kCgThreads) {
#pragma unroll
      for (int f = 0; f < 6; ++f) {
        reinterpret_cast<float*>(p)[f * m + s] = G.c[f * G.cap + s];
        reinterpret_cast<unsigned short*>(p + 28 * m)[f * m + s] = (unsigned short)(4 * G.nb[f * G.cap + s]);
      }
      reinterpret_cast<float*>(p + 24 * m)[s] = G.idg[s];
#pragma unroll
      for (int k = 0; k < 8; ++k) {
        const int ch = G.child[k * G.cap + s];
        if (l > lc) reinterpret_cast<unsigned short*>(p + 40 * m)[k * m + s] = ch < 0 ? 0xffff : (unsigned short)(4 * ch);
        else reinterpret_cast<unsigned*>(cg_dyn + S.lay.lchild)[k * m + s] = ch < 0 ? ~0u : code(lc - 1, ch, mulf);
      }
    }
  }
  if (S.lay.agg >= 0) {
    const int na = S.lay.n[lc - 1], lb = (lc - 1 < lg ? rank : crank) * na, n = max(0, min(na, S.lay.cnt[lc - 1] - lb));
    for (int s = t0; s < n; s += kCgThreads)
      reinterpret_cast<unsigned short*>(cg_dyn + S.lay.agg)[s] = (unsigned short)mg.L[lc - 1].agg[lb + s];
  }
  if constexpr (MODE == CG_HYBRID) {
    const unsigned mul = magic(lg);
    const int lb = rank * S.lay.n[lg - 1];
    for (int s = t0; s < S.dg[lg - 1].n; s += kCgThreads)
      reinterpret_cast<unsigned*>(cg_dyn + S.lay.par)[s] = code(lg, mg.L[lg - 1].agg[lb + s], mul);
  }
  // x, r, p, q of the own nodes; the CG operator's couplings
  // (the FP32 form's r is the V-cycle's right-hand side b)
  T *X = v.x + base, *R = v.r + base, *P = v.p + base, *Q = v.q + base;
  if constexpr (CL) {
    X = reinterpret_cast<T*>(cg_dyn + S.lay.cgv);
    P = X + na0;
    Q = P + na0;
    R = sizeof(T) == 4 ? reinterpret_cast<T*>(cg_dyn + S.lay.vec[0]) : Q + na0;
  }
  const T* cA = nullptr;   // FP64 form only; the FP32 form reads the level's own couplings
  int csA = 0;
  if constexpr (sizeof(T) == 8) {
    if (S.lay.c64 >= 0) {
      T* d = reinterpret_cast<T*>(cg_dyn + S.lay.c64);
      for (int s = t0; s < n0; s += kCgThreads)
#pragma unroll
        for (int f = 0; f < 6; ++f) d[f * na0 + s] = v.c[f * v.cap + base + s];
      cA = d;
      csA = na0;
    } else {
      cA = v.c + base;
      csA = v.cap;
    }
  }
  const CGSolve<T, MODE> A{S, q, mg, rank, K, dyn};
  LevD<CL> L0;
  if constexpr (CL) L0 = S.dc[0];
  else L0 = S.dg[0];
  auto cop = [&](int f, int i) -> T {
    if constexpr (sizeof(T) == 4) return L0.c(f, i, false);
    else return cA[f * csA + i];
  };
  const int nact = min(32, (n0 + 31) / 32);
  const float w1 = mg.w1;

  // one band component: the plain mean; several: the mean of each (Sec. 2.1 per component)
  const int C = *c.ncomp;
  CompAcc cacc{S.csh, c.csum, C};
  if (C > 1) {
    if (rank == 0)
      for (int i = t0; i < 2 * kCompCap; i += kCgThreads) c.csum[i] = 0.0;
    if (!A.bar()) return;
    cacc.begin();
  }
  // x0 for the neighbours: the cluster engine's FP32 form keeps it in t, the others in global memory
  constexpr bool kXt = CL && sizeof(T) == 4;
  W s(0);
  for (int i = t0; i < n0; i += kCgThreads) {
    const int p = idx[base + i];
    T x0 = gs.a[p];
    if (gs.b) x0 += gs.cb * gs.b[p];
    if (gs.c) x0 += gs.cc * gs.c[p];
    X[i] = x0;
    if constexpr (kXt) L0.put(V_T, i, x0);
    else if constexpr (CL) v.x[base + i] = x0;
    const W f = rhs(p);
    R[i] = wnear(f);   // f kept for the residual pass
    if (C > 1) cacc.add(c.comp[base + i], (double)wnear(f));
    else s = s + f;
  }
  if (C > 1) cacc.end();
  else A.post(s, A_SUMF, nact);
  if (!A.bar()) return;
  if (A.scalar_warp() && C == 1) {
    const W t = A.total(A_SUMF);
    if (A.scalar_lane()) S.mean = wide_d(t) / M;
  }
  W bb(0), rr(0);
  __syncthreads();
  const auto mean_of = [&](int i) {
    if (C == 1) return W(S.mean);
    const int ci = c.comp[base + i];
    return W(__ldcg(c.csum + ci) / c.csize[ci]);
  };
  {
    for (int i = t0; i < n0; i += kCgThreads) {
      const W mf = mean_of(i);
      const W b = W(R[i]) - mf;
      const T xi = X[i];
      T ax = 0;
#pragma unroll
      for (int f = 0; f < 6; ++f) {
        if constexpr (kXt) ax += cop(f, i) * (xi - L0.nbr(V_T, L0.nb(f, i)));
        else ax += cop(f, i) * (xi - __ldcg(v.x + v.nb[f * v.cap + base + i]));
      }
      const T r = wnear(b - W(ax));
      R[i] = r;
      bb = bb + b * b;
      rr = rr + W(r) * W(r);
      if constexpr (sizeof(T) == 4) {
        L0.put(V_E, i, w1 * L0.idg(i) * r);
      }
    }
  }
  A.post(bb, A_BB, nact);
  A.post(rr, A_RR, nact);
  if (!A.bar()) return;
  const auto first_test = [&] {
    if (!A.scalar_warp()) return;
    const W tb = A.total(A_BB), tr = A.total(A_RR);
    if (!A.scalar_lane()) return;
    const double bbs = wide_d(tb);
    S.bb = bbs;
    S.rr = wide_d(tr);
    S.tol2 = c.rtol * c.rtol * bbs;
    S.go = (bbs == 0.0 || S.rr <= S.tol2) ? 0 : 1;
  };
  first_test();
  if (A.scalar_lane()) {
    S.sc = 1;
    if constexpr (sizeof(T) == 8) {
      // the power of two that takes the larger of |b| and |r| into [1, 2), for the FP32 copy of the
      // residual (a guess far off leaves |r| >> |b|)
      int ex = 0;
      frexp(sqrt(fmax(S.bb, S.rr)), &ex);
      S.sc = ldexp(1.0, max(-1000, min(1000, 1 - ex)));
    } else {
      S.range = !(S.bb < 1e30 && S.rr < 1e30) || S.bb < 1e-20;   // an overflow may read as NaN
      S.zero = S.bb == 0.0;
      S.pre = S.rr < 1.0 && S.bb < 1.0 ? 0x1p60f : 0x1p-30f;
    }
  }
  __syncthreads();
  if constexpr (sizeof(T) == 4) {
    // (b,b) has FP32's range: a right-hand side above some 1e15 or below 1e-10 is solved in units
    // of a power of two near sum |b| + |r| (exact, and undone at the end)
    if (S.range) {
      const float pre = S.pre;
      const auto b_of = [&](int i) { return W(wnear(rhs(idx[base + i]))) - mean_of(i); };
      W l(0);
      for (int i = t0; i < n0; i += kCgThreads) l = l + W(pre * fabsf(wnear(b_of(i)))) + W(pre * fabsf(R[i]));
      A.post(l, A_SUMX, nact);
      if (!A.bar()) return;
      if (A.scalar_warp()) {
        const double t = wide_d(A.total(A_SUMX)) / (double)pre;
        // not finite: left alone; up by 2^60 at most, which leaves room for a large initial guess
        if (A.scalar_lane() && t > 0.0 && t < 1e300) S.sc = ldexpf(1.0f, max(-126, min(60, -ilogb(t))));
      }
      __syncthreads();
      const float sc = S.sc;
      bb = rr = W(0);
      for (int i = t0; i < n0; i += kCgThreads) {
        const W b = b_of(i) * W(sc);
        const float r = R[i] * sc;
        X[i] *= sc;
        R[i] = r;
        bb = bb + b * b;
        rr = rr + W(r) * W(r);
        L0.put(V_E, i, w1 * L0.idg(i) * r);
      }
      A.post(bb, A_BB, nact);
      A.post(rr, A_RR, nact);
      if (!A.bar()) return;
      first_test();
      // a right-hand side that only vanishes beside the residual of a guess far off is not zero
      if (A.scalar_lane() && S.bb == 0.0 && !S.zero) S.go = 1;
      __syncthreads();
    }
  }
  bool conv = !S.go;
  int k = 0;
  if (!conv) {
    T sc = 1;
    if constexpr (sizeof(T) == 8) {
      sc = S.sc;
      for (int i = t0; i < n0; i += kCgThreads) {
        const float b = (float)(R[i] * sc);
        L0.put(V_B, i, b);
        L0.put(V_E, i, w1 * L0.idg(i) * b);
      }
      if (!A.bar()) return;
    }
    for (bool first = true;; first = false) {
      // gamma = (r, o); the FP32 form's thread partial is FP32, as in (w, o) and (r, r) below, then
      // double-float (one to some hundred nodes a thread; compensated partials changed no error
      // against 64 bits and cost up to 0.7%)
      T g = 0;
      const int st = A.vcycle(
          [&] {
            if (first || !A.scalar_warp()) return;
            const W t = A.total(A_RR);
            if (A.scalar_lane()) {
              S.rr = wide_d(t);
              S.go = S.rr <= S.tol2 ? 0 : 1;
            }
          },
          [&](int i, float o) { g += R[i] * (T)o; });
      if (st < 0) return;
      if (st == 1) {
        conv = true;
        break;
      }
      if (k >= c.maxit) break;
      A.post(W(g), A_RU, nact);
      if (!A.bar()) return;
      if (A.scalar_warp()) {
        const W gn = A.total(A_RU);
        if (A.scalar_lane()) {
          const W bt = first ? W(0) : wdiv(gn, S.gamma);
          S.bt = wnear(bt);
          // kept for the step length: (p, A p) = delta - beta gamma / a_old
          S.alpha = first ? W(0) : wdiv(bt * gn, S.alpha);
          S.gamma = gn;
        }
      }
      T du = 0, bt = 0;
      nodes(
          n0,
          [&](int i) {
            const T u = (T)L0.own(V_O, i);
            unsigned j[6];
            float x[6];
            T w = 0;
            if constexpr (sizeof(T) == 4) {
              float cf[6];
              faces(L0, i, false, cf, j);
#pragma unroll
              for (int f = 0; f < 6; ++f) x[f] = L0.nbr(V_O, j[f]);
#pragma unroll
              for (int f = 0; f < 6; ++f) w += cf[f] * (u - x[f]);
            } else {
#pragma unroll
              for (int f = 0; f < 6; ++f) j[f] = L0.nb(f, i);
#pragma unroll
              for (int f = 0; f < 6; ++f) x[f] = L0.nbr(V_O, j[f]);
#pragma unroll
              for (int f = 0; f < 6; ++f) w += cA[f * csA + i] * (u - (T)x[f]);
            }
            return make_uw(u, w);
          },
          [&] {
            __syncthreads();
            bt = S.bt;
          },
          [&](int i, auto r) {
            P[i] = first ? r.x : r.x + bt * P[i];
            Q[i] = first ? r.y : r.y + bt * Q[i];
            du += r.y * r.x;
          });
      A.post(W(du), A_DU, nact);
      if (!A.bar()) return;
      if (A.scalar_warp()) {
        const W dt = A.total(A_DU);
        if (A.scalar_lane()) {
          const W den = dt - S.alpha;
          S.go = wpos(den);
          const W al = wpos(den) ? wdiv(S.gamma, den) : W(0);
          S.alpha = al;
          S.a = wnear(al);
        }
      }
      __syncthreads();
      if (!S.go) {        // (p, A p) <= 0: converged if it is the first direction, else not
        conv = first;
        break;
      }
      const T a = S.a;
      T rn = 0;
      nodes(
          n0,
          [&](int i) {
            const T r = R[i] - a * Q[i];
            return Trip<T, float>{X[i] + a * P[i], r, L0.idg(i)};
          },
          [&](int i, Trip<T, float> t) {
            X[i] = t.p;
            R[i] = t.q;
            rn += t.q * t.q;
            const float b = sizeof(T) == 4 ? (float)t.q : (float)(t.q * sc);
            if constexpr (sizeof(T) == 8) L0.put(V_B, i, b);
            L0.put(V_E, i, w1 * t.d * b);
          });
      A.post(W(rn), A_RR, nact);
      if (!A.bar()) return;
      ++k;
    }
  }
  // zero-mean projection of the solution (per band component)
  __syncthreads();
  if (C > 1) {
    cacc.dst = c.csum + kCompCap;
    cacc.begin();
  }
  W sx(0);
  for (int i = t0; i < n0; i += kCgThreads) {
    if (C > 1) cacc.add(c.comp[base + i], (double)X[i]);
    else sx = sx + W(X[i]);
  }
  if (C > 1) cacc.end();
  else A.post(sx, A_SUMX, nact);
  if (!A.bar()) return;
  if (A.scalar_warp() && C == 1) {
    const W t = A.total(A_SUMX);
    if (A.scalar_lane()) S.mean = wide_d(t) / M;
  }
  __syncthreads();
  const T mx = (T)S.mean, usc = (T)1 / S.sc;
  for (int i = t0; i < n0; i += kCgThreads) {
    const int p = idx[base + i];
    T mi = mx;
    if (C > 1) {
      const int ci = c.comp[base + i];
      mi = (T)(__ldcg(c.csum + kCompCap + ci) / c.csize[ci]);
    }
    T w = X[i] - mi;
    if constexpr (sizeof(T) == 4) w *= usc;
    wfull[p] = w;
    if (gs.hist) gs.hist[p] = w;
  }
  if (rank == 0 && t0 == 0) {
    *c.iters = k;
    *c.resid = S.bb > 0 ? sqrt(S.rr / S.bb) : 0.0;
    if (!conv) atomicCAS(c.status, 0, 5);
    atomicAdd(c.work, (unsigned long long)k * (unsigned long long)M);
  }
}

template <typename T, int MODE>
__global__ void __launch_bounds__(kCgThreads, 1) k_cg(const int* __restrict__ idx, CGVec<T> v, T* __restrict__ wfull,
                                                      Rhs<T> rhs, CGCtl2 q, MGP mg, CGGuess<T> gs) {
  extern __shared__ __align__(16) unsigned char cg_dyn[];
  __shared__ CGShared<T> S;
  const int t0 = threadIdx.x;
  if (t0 < (int)(sizeof(CGLayout) / 4)) reinterpret_cast<int*>(&S.lay)[t0] = reinterpret_cast<const int*>(q.lay)[t0];
  const int skip = (q.sel & 2) ? q.other->bytes <= kCgSmem : 0;
  // An earlier failure (no convergence, a lost copy): no solve.  Nothing sets the word while a
  // cluster's launch runs, so all of its threads read the same.  A block of the other engines may
  // start after another one has given up, and its threads, or the blocks, would read different
  // values: there the first grid barrier looks at it.
  const int st0 = MODE == CG_CLUSTER ? *(volatile int*)q.c.status : 0;
  __syncthreads();
  if (skip || st0 != 0 || ((q.sel & 1) && S.lay.bytes > kCgSmem)) return;
  // A band without usable labels: reported by every solve on it (a frozen band's labels are made
  // once, and the report of that launch is cleared with the call that returns it).
  const int C = *q.c.ncomp;
  if (C > kCompCap || C < 0) {
    if (blockIdx.x == 0 && t0 == 0) atomicCAS(q.c.status, 0, C < 0 ? 6 : 8);
    return;
  }
  if (S.lay.cnt[0] == 0) {
    if (blockIdx.x == 0 && t0 == 0) {
      *q.c.iters = 0;
      *q.c.resid = 0.0;
    }
    return;
  }
  cg_block<T, MODE>(idx, v, wfull, rhs, q, mg, gs, cg_dyn, S);
  // No block leaves while another of its cluster may still read its shared memory, after a failed
  // barrier either: all of them fail at the same one, and one that has yet to arrive there may be
  // reading those that wait.
  if constexpr (MODE != CG_GRID) cluster_barrier();
}

// <w, f>: sum over the band (the nonlocal energy term).
template <typename T>
__global__ void k_band_dot(const int* __restrict__ idx, const int* __restrict__ count, const T* __restrict__ w,
                           Rhs<T> rhs, double* dst) {
  const int M = *count;
  double s = 0;
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < M; i += gridDim.x * blockDim.x) {
    const int p = idx[i];
    s += (double)w[p] * wide_d(rhs(p));
  }
  block_add(s, dst);
}

}  // namespace etd
