// mgsetup.cuh -- set-up of the band solve: the multigrid hierarchy of the current band, its
// connected components and the solve's shared-memory layouts.
//
// What bounds it: latency (the levels shrink by 4 to 8, and every step of a level depends on the
// one before).  Levels of more than 2^15 cells use grid-wide kernels; one cluster of 8 blocks builds
// the rest (k_mg_tail) with the level's cells as a bitmap in shared memory, so that marking, numbering
// and looking up a cell cost shared-memory accesses instead of the three global arrays that the
// larger levels use, and labels the coarsest level.
#pragma once
#include "bandcg.cuh"
#include "kernels.cuh"

namespace etd {

// Extents of one level's grid (any even sizes; level l halves level l-1 along every axis,
// z only in 3D).
struct Ext {
  int x, y, z;
};
// The cell of level l (extents c) holding flat index p of level l-1 (extents f): shifts where f's
// x and y are powers of two, division otherwise.
struct CellOf {
  int lx, ly, mx, my, is3d;
  Ext f, c;
  __device__ CellOf(Ext f_, int is3d_, Ext c_) : is3d(is3d_), f(f_), c(c_) {
    const bool pow2 = !(f.x & (f.x - 1)) && !(f.y & (f.y - 1));
    lx = pow2 ? 31 - __clz(f.x) : -1;
    ly = 31 - __clz(f.y);
    mx = f.x - 1;
    my = f.y - 1;
  }
  __device__ __forceinline__ int operator()(int p) const {
    int X, Y, Z;
    if (lx >= 0) {
      X = p & mx;
      Y = (p >> lx) & my;
      Z = p >> (lx + ly);
    } else {
      const int t = p / f.x;
      X = p - t * f.x;
      Z = t / f.y;
      Y = t - Z * f.y;
    }
    return ((is3d ? Z >> 1 : 0) * c.y + (Y >> 1)) * c.x + (X >> 1);
  }
};

// Mark the cells of level l (extents c) holding nodes of level l-1 (extents f).
static __global__ void k_mg_mark(const int* __restrict__ list, const int* __restrict__ cnt, Ext f, int is3d, Ext c,
                                 unsigned char* __restrict__ mark) {
  const int M = *cnt, t0 = blockIdx.x * blockDim.x + threadIdx.x, ns = gridDim.x * blockDim.x;
  const CellOf cell(f, is3d, c);
#pragma unroll 4
  for (int i = t0; i < M; i += ns) mark[cell(list[i])] = 1;
}

static __global__ void k_mg_parent(const int* __restrict__ list, const int* __restrict__ cnt, Ext f, int is3d, Ext c,
                                   const int* __restrict__ cmap, int* __restrict__ agg) {
  const int M = *cnt, t0 = blockIdx.x * blockDim.x + threadIdx.x, ns = gridDim.x * blockDim.x;
  const CellOf cell(f, is3d, c);
#pragma unroll 4
  for (int i = t0; i < M; i += ns) agg[i] = cmap[cell(list[i])];
}

// Node I of a level, at cell C: its children, its Galerkin couplings (the sums of the finer
// couplings that cross between two cells) and its neighbours; and whether its children are
// connected inside the cell.  If they are in every cell, the components of each level are the
// components of the next coarser one (two nodes are coupled exactly when a finer coupling
// crosses between their cells), so the coarsest level's labels, followed down the parents, are
// the band's components; a cell whose children split inside it sets the fallback flag and the
// union-find over the band runs.  child_at(F): node of the finer level at its cell F, -1 if none;
// node_at(C): node of this level at cell C.  The 8 children, then their couplings and in-cell
// neighbours: rounds of independent loads.
template <typename ChildAt, typename NodeAt>
__device__ __forceinline__ void mg_coarse_node(int I, int C, Ext ec, int is3d, Ext ef, ChildAt&& child_at,
                                               const float* fc, const int* fnb, int fcap,
                                               NodeAt&& node_at, float* __restrict__ c, int* __restrict__ nb,
                                               float* __restrict__ idg, int* __restrict__ child, int cap,
                                               int* fallback) {
  const int X = C % ec.x, tq = C / ec.x, Y = tq % ec.y, Z = tq / ec.y;
  float s[6] = {0, 0, 0, 0, 0, 0};
  int jk[8];
  unsigned pres = 0;
#pragma unroll
  for (int k = 0; k < 8; ++k) {
    const int a = k & 1, b = (k >> 1) & 1, cz = k >> 2;
    jk[k] = (is3d || cz == 0) ? child_at(((2 * Z + cz) * ef.y + (2 * Y + b)) * ef.x + (2 * X + a)) : -1;
    if (jk[k] >= 0) pres |= 1u << k;
  }
  unsigned adj[8] = {};
#pragma unroll
  for (int k = 0; k < 8; ++k) {
    const int a = k & 1, b = (k >> 1) & 1, cz = k >> 2;
    // unconditional loads (node 0 in the place of a missing child): all in flight together
    const int j = jk[k], q = max(j, 0);
    child[k * cap + I] = j;
    const float vx = __ldcg(fc + (a ? 0 : 1) * fcap + q), vy = __ldcg(fc + (b ? 2 : 3) * fcap + q),
                vz = __ldcg(fc + (cz ? 4 : 5) * fcap + q);
    s[a ? 0 : 1] += j >= 0 ? vx : 0.0f;
    s[b ? 2 : 3] += j >= 0 ? vy : 0.0f;
    s[cz ? 4 : 5] += is3d && j >= 0 ? vz : 0.0f;
#pragma unroll
    for (int d = 0; d < 3; ++d) {
      if ((k >> d) & 1) continue;   // the + face of the lower child sees the pair
      const int k2 = k | (1 << d);
      const bool on = __ldcg(fnb + 2 * d * fcap + q) == jk[k2] && j >= 0 && jk[k2] >= 0;
      adj[k] |= on ? 1u << k2 : 0u;
      adj[k2] |= on ? 1u << k : 0u;
    }
  }
  unsigned r = pres & (~pres + 1u);     // lowest present child
#pragma unroll
  for (int it = 0; it < 3; ++it) {      // the cube graph has diameter 3
    unsigned nr = r;
#pragma unroll
    for (int k = 0; k < 8; ++k)
      if ((r >> k) & 1) nr |= adj[k];
    r = nr;
  }
  if (r != pres) atomicExch(fallback, 1);
  const int xp = X + 1 == ec.x ? 0 : X + 1, xm = X == 0 ? ec.x - 1 : X - 1;
  const int yp = Y + 1 == ec.y ? 0 : Y + 1, ym = Y == 0 ? ec.y - 1 : Y - 1;
  const int zp = Z + 1 == ec.z ? 0 : Z + 1, zm = Z == 0 ? ec.z - 1 : Z - 1;
  const int ncell[6] = {(Z * ec.y + Y) * ec.x + xp, (Z * ec.y + Y) * ec.x + xm, (Z * ec.y + yp) * ec.x + X,
                        (Z * ec.y + ym) * ec.x + X, (zp * ec.y + Y) * ec.x + X, (zm * ec.y + Y) * ec.x + X};
  float d = 0;
#pragma unroll
  for (int f = 0; f < 6; ++f) {
    c[f * cap + I] = s[f];
    nb[f * cap + I] = s[f] > 0.0f ? node_at(ncell[f]) : I;
    d += s[f];
  }
  idg[I] = d > 0.0f ? 1.0f / d : 1.0f;
}

static __global__ void k_mg_coarse(const int* __restrict__ clist, const int* __restrict__ ccnt, Ext ec, int is3d,
                                   const unsigned char* __restrict__ fmark, const int* __restrict__ fmap, Ext ef,
                                   const float* __restrict__ fc, const int* __restrict__ fnb, int fcap,
                                   const int* __restrict__ cmap, float* __restrict__ c, int* __restrict__ nb,
                                   float* __restrict__ idg, int* __restrict__ child, int cap, int* fallback) {
  const int M = *ccnt;
  for (int I = blockIdx.x * blockDim.x + threadIdx.x; I < M; I += gridDim.x * blockDim.x)
    mg_coarse_node(
        I, clist[I], ec, is3d, ef, [&](int F) {
          const int m = fmap[F];   // of an unmarked cell: an old entry, not used
          return fmark[F] ? m : -1;
        }, fc, fnb, fcap,
        [&](int C) { return cmap[C]; }, c, nb, idg, child, cap, fallback);
}

// One level's arrays.  The tail's own levels have no list, map or mark in global memory.
struct MGSetLevel {
  Ext e;
  int cap;
  int* cnt;
  const int* list;
  const int* map;
  const unsigned char* mark;
  float* c;
  int* nb;
  float* idg;
  int* agg;
  int* child;
};
constexpr int kTailCells = 1 << 15;
constexpr int kCCCoarse = 1024;   // largest coarsest level that one block labels
struct MGTail {
  int first, nlev, is3d;   // levels first .. nlev-1 are built here (at most kTailCells cells each)
  MGSetLevel L[kMGMax];
  int* ccL;                // labels of the coarsest level
  int* ncomp;              // component count (0 with the fallback flag set)
  int* fallback;
  double* csize;           // component sizes, zeroed here
};
// Shared memory: two bitmaps with their word prefixes, two cell lists (a level has at most half,
// in 3D an eighth, of the cells of the finer one), the scan's warp sums, then the labels.
constexpr int kTailSmem = 2 * 2 * 4 * (kTailCells / 32) + 2 * kTailCells + 2 * kTailCells / 4 + 128;

// Every block of the cluster numbers all the cells (the same bitmap in each); they share the
// marking, the nodes' parents and their couplings, some 70 scattered loads and stores a node.
constexpr int kTailBlocks = 8;
__device__ __forceinline__ void tail_barrier() {   // hardware barrier of the cluster, global writes included
  asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
  asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}
static __global__ void __cluster_dims__(kTailBlocks, 1, 1) __launch_bounds__(1024) k_mg_tail(MGTail a) {
  extern __shared__ __align__(16) unsigned char tail_dyn[];
  constexpr int NW = kTailCells / 32;
  unsigned* const words = reinterpret_cast<unsigned*>(tail_dyn);             // [2][NW]
  unsigned* const pref = words + 2 * NW;                                     // [2][NW]
  unsigned short* const lists = reinterpret_cast<unsigned short*>(pref + 2 * NW);
  int* const wsum = reinterpret_cast<int*>(tail_dyn + kTailSmem - 128);
  __shared__ int cnts[kMGMax];
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
  const int g0 = blockIdx.x * 1024 + tid, gs = kTailBlocks * 1024;
  if (tid < a.nlev && tid < a.first) cnts[tid] = *a.L[tid].cnt;
  for (int k = g0; k < kCompCap; k += gs) a.csize[k] = 0.0;
  __syncthreads();
  for (int l = a.first; l < a.nlev; ++l) {
    const MGSetLevel& F = a.L[l - 1];
    const MGSetLevel& L = a.L[l];
    const int par = (l - a.first) & 1;
    unsigned *W = words + par * NW, *P = pref + par * NW;
    const unsigned *FW = words + (par ^ 1) * NW, *FP = pref + (par ^ 1) * NW;
    unsigned short* lst = lists + par * kTailCells;
    const unsigned short* flst = lists + (par ^ 1) * kTailCells;
    const bool top = l == a.first;
    const int MF = cnts[l - 1];
    const Ext fe = F.e, e = L.e;
    const int* __restrict__ glist = F.list;
    const CellOf cellof(fe, a.is3d, e);
    auto cell = [&](int i) { return cellof(top ? glist[i] : (int)flst[i]); };
    auto rank = [&](int C) { return (int)(P[C >> 5] + __popc(W[C >> 5] & ((1u << (C & 31)) - 1u))); };
    W[tid] = 0;
    __syncthreads();
    // each block marks its share of the finer nodes; the bitmaps are then or-ed together
    for (int i = g0; i < MF; i += gs) {
      const int C = cell(i);
      if (!((W[C >> 5] >> (C & 31)) & 1u)) atomicOr(&W[C >> 5], 1u << (C & 31));
    }
    tail_barrier();
    {
      unsigned w = 0;
      const uint32_t mine = smem_u32(W + tid);
#pragma unroll
      for (int k = 0; k < kTailBlocks; ++k) {
        unsigned x;
        asm volatile("ld.shared::cluster.u32 %0, [%1];" : "=r"(x) : "r"(mapa_u32(mine, k)));
        w |= x;
      }
      tail_barrier();   // every block has read before any overwrites its bitmap
      W[tid] = w;
    }
    __syncthreads();
    {
      const unsigned w = W[tid];
      int inc = __popc(w);
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const int t = __shfl_up_sync(0xffffffffu, inc, o);
        if (lane >= o) inc += t;
      }
      if (lane == 31) wsum[wid] = inc;
      __syncthreads();
      int before = 0, all = 0;
      for (int k = 0; k < 32; ++k) {
        const int v = wsum[k];
        if (k < wid) before += v;
        all += v;
      }
      int pos = before + inc - __popc(w);
      P[tid] = pos;
      for (unsigned m = w; m; m &= m - 1) lst[pos++] = (unsigned short)(32 * tid + __ffs(m) - 1);
      if (tid == 0) {
        cnts[l] = all;
        if (blockIdx.x == 0) *L.cnt = all;
      }
    }
    __syncthreads();
    const int M = cnts[l];
#pragma unroll 4
    for (int i = g0; i < MF; i += gs) F.agg[i] = rank(cell(i));
    if (top) {
      const int* __restrict__ fmap = F.map;
      const unsigned char* __restrict__ fmark = F.mark;
      for (int I = g0; I < M; I += gs)
        mg_coarse_node(
            I, (int)lst[I], e, a.is3d, fe,
            [&](int C) {
              const int m = fmap[C];
              return fmark[C] ? m : -1;
            },
            F.c, F.nb, F.cap, rank, L.c, L.nb, L.idg, L.child, L.cap, a.fallback);
    } else {
      for (int I = g0; I < M; I += gs)
        mg_coarse_node(
            I, (int)lst[I], e, a.is3d, fe,
            [&](int C) {
              const unsigned w = FW[C >> 5];
              return (w >> (C & 31)) & 1u ? (int)(FP[C >> 5] + __popc(w & ((1u << (C & 31)) - 1u))) : -1;
            },
            F.c, F.nb, F.cap, rank, L.c, L.nb, L.idg, L.child, L.cap, a.fallback);
    }
    tail_barrier();
  }
  if (blockIdx.x != 0) return;
  // Label the coarsest level: min-label propagation with pointer jumping (bounded by the node
  // count), compact ids of the roots, the component count.
  int* const lab = reinterpret_cast<int*>(tail_dyn);
  int* const cid = lab + kCCCoarse;
  int* const nroot = cid + kCCCoarse;
  const MGSetLevel& L = a.L[a.nlev - 1];
  const int M = cnts[a.nlev - 1];
  const bool no = *(volatile int*)a.fallback != 0 || M > kCCCoarse;
  __syncthreads();
  if (no) {
    if (tid == 0) {
      *a.ncomp = 0;
      atomicExch(a.fallback, 1);
    }
    return;
  }
  const int i = tid;
  int nbi[6];
  for (int f = 0; f < 6; ++f) nbi[f] = i < M ? __ldcg(L.nb + f * L.cap + i) : i;
  if (i < M) lab[i] = i;
  if (i == 0) *nroot = 0;
  __syncthreads();
  for (int it = 0; it <= M; ++it) {
    int m = i < M ? lab[i] : 0;
    if (i < M) {
      for (int f = 0; f < 6; ++f) m = min(m, lab[nbi[f]]);
      m = min(m, lab[m]);
    }
    __syncthreads();
    const bool ch = i < M && m < lab[i];
    if (ch) lab[i] = m;
    if (!__syncthreads_or(ch)) break;
  }
  if (i < M && lab[i] == i) cid[i] = atomicAdd(nroot, 1);
  __syncthreads();
  if (i < M) a.ccL[i] = cid[lab[i]];
  if (i == 0) *a.ncomp = *nroot;
}

// Each band node's component through its chain of parents; the component sizes.  A band of one
// component needs neither: the solve then removes the plain mean, and only the size is written.
// One more block lays out the solve.
struct CCLevels {
  int nlev;
  const int* cnt[kMGMax];
  const int* agg[kMGMax];
  int tsize, clK, gridK, hybK, gsmem;
  CGLayout* lay;
};
static __global__ void k_cc_down(CCLevels lv, const int* __restrict__ ccL, const int* __restrict__ ncomp,
                                 int* __restrict__ comp, double* __restrict__ csize, const int* fallback) {
  __shared__ double sh[kCompShared];
  if (blockIdx.x == gridDim.x - 1) {
    cg_layouts(lv.cnt, lv.nlev, lv.tsize, lv.clK, lv.gridK, lv.hybK, lv.gsmem, lv.lay);
    return;
  }
  if (*fallback) return;
  const int M = *lv.cnt[0];
  const int C = *ncomp;
  const int nblk = gridDim.x - 1;
  if (C <= 1) {
    if (blockIdx.x == 0 && threadIdx.x == 0) csize[0] = (double)M;
    return;
  }
  CompAcc acc{sh, csize, C};
  acc.begin();
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < M; i += nblk * blockDim.x) {
    int j = i;
    for (int l = 0; l + 1 < lv.nlev; ++l) j = lv.agg[l][j];
    const int c = ccL[j];
    comp[i] = c;
    acc.add(c, 1.0);
  }
  acc.end();
}

// The fallback: a lock-free union-find over the band's neighbour lists, its phases separated by
// grid barriers (cooperative launch; returns at once when the hierarchy gave the components).
// Each node starts as a child of its smallest band neighbour (or of itself), which leaves a
// forest with one tree per local minimum of the index over the band; linking then only has to
// merge those trees; then full compression with a compact id per root (arbitrary order), and the
// nodes' components and the component sizes.
static __global__ void __launch_bounds__(256) k_cc_union(const int* __restrict__ count, const int* __restrict__ nb,
                                                         int cap, int* __restrict__ parent, int* __restrict__ cid,
                                                         int* __restrict__ ncomp, int* __restrict__ comp,
                                                         double* __restrict__ csize, const int* fallback, CGCtl c) {
  __shared__ double sh[kCompShared];
  if (!*fallback) return;
  const int M = *count, t0 = blockIdx.x * blockDim.x + threadIdx.x, ns = gridDim.x * blockDim.x;
  // An earlier failure does not stop the labelling (a frozen band is labelled once, for all the
  // steps after that failure has been reported); a barrier of its own that gives up leaves no
  // component count, which the solves report.
  auto barrier = [&] {
    const bool ok = grid_sync<false>(c);
    if (!ok && t0 == 0) atomicExch(ncomp, kNoComponents);
    return ok;
  };
  for (int i = t0; i < M; i += ns) {
    int m = i;
#pragma unroll
    for (int f = 0; f < 6; ++f) m = min(m, nb[f * cap + i]);
    parent[i] = m;
  }
  if (!barrier()) return;
  for (int i = t0; i < M; i += ns) {
#pragma unroll
    for (int f = 0; f < 6; f += 2) {       // the + faces: every band edge is seen from one end
      const int j = nb[f * cap + i];
      if (j == i) continue;
      int a = cc_root(parent, i), b = cc_root(parent, j);
      for (int tries = 0; a != b; ++tries) {
        if (tries > M) {                   // cannot happen; guards the loop bound
          atomicCAS(c.status, 0, 8);
          break;
        }
        const int hi = a > b ? a : b, lo = a > b ? b : a;
        const int old = atomicCAS(parent + hi, hi, lo);
        if (old == hi) break;
        a = cc_root(parent, old);
        b = lo;
      }
    }
  }
  if (!barrier()) return;
  for (int i = t0; i < M; i += ns) {
    const int r = cc_root(parent, i);
    parent[i] = r;
    if (r == i) cid[i] = atomicAdd(ncomp, 1);
  }
  if (!barrier()) return;
  const int C = *(volatile int*)ncomp;
  if (C > kCompCap) {
    if (t0 == 0) atomicCAS(c.status, 0, 8);
    return;
  }
  if (C <= 1) {
    if (t0 == 0) csize[0] = (double)M;
    return;
  }
  CompAcc acc{sh, csize, C};
  acc.begin();
  for (int i = t0; i < M; i += ns) {
    const int k = __ldcg(cid + __ldcg(parent + i));
    comp[i] = k;
    acc.add(k, 1.0);
  }
  acc.end();
}

}  // namespace etd
