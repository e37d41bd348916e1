// kernels.cuh -- pointwise terms, finite-difference band terms, band compaction, the band
// conjugate-gradient solve and FP64 reductions of the ETD membrane step.
#pragma once
#include <cuda_fp16.h>
#include <cuda_runtime.h>
#include "barrier.h"
#include "fft.cuh"

namespace etd {

// Model coefficients in the working precision (Eq. (1.1)-(1.2), Sec. 3.1) plus grid factors.
template <typename T> struct ModelC {
  T eps_phi, eps_u, mu, lambda_surf, kappa, lambda_line, M_area, alpha, u0;
  T gamma, M, ubar, A1, A2, B1, B2, band_hi, delta, tau;
  T ih2[3];    // 1/h_d^2
  T i2h[3];    // 1/(2 h_d)
  int dim;
  int linear_only;
};

// Slots of the FP64 scalar array shared by the kernels of one plan.
enum Scal {
  S_VOL = 0,      // sum phi (current phi-stage argument)
  S_MASS = 1,     // sum G (u - ubar)  or  sum G (f(u) - ubar)
  S_GRAD = 2, S_WELL = 3, S_NONLOC = 4, S_MASSF = 5, S_VOLE = 6,
  S_MAXB = 7, S_UMIN = 8, S_UMAX = 9,
  S_A0 = 12,      // A0 itself (not a sum); set once
  S_COUNT = 16
};

__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
  return v;
}

// Block-wide sum added atomically to *dst (one atomic per block).  All threads call it.
__device__ __forceinline__ void block_add(double v, double* dst) {
  __shared__ double ws[32];
  v = warp_sum(v);
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  __syncthreads();
  if (lane == 0) ws[wid] = v;
  __syncthreads();
  if (wid == 0) {
    const int nw = (blockDim.x + 31) >> 5;
    double t = (lane < nw) ? ws[lane] : 0.0;
    t = warp_sum(t);
    if (lane == 0) atomicAdd(dst, t);
  }
}

// The same for a double-float partial (FP32 storage): shuffles and additions on the FP32 pipes,
// one FP64 addition per block.  A block's 16 warps need 1.3 k clocks for the FP64 form (an FP64
// warp instruction holds its pipe for 64), 0.3 k for this one; it is a tail of every reduction
// and of every summing pass-A epilogue.
__device__ __forceinline__ void block_add(dfloat v, double* dst) {
  __shared__ dfloat ws[32];
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1)
    v = v + dfloat(__shfl_down_sync(0xffffffffu, v.hi, o), __shfl_down_sync(0xffffffffu, v.lo, o));
  __syncthreads();
  if (lane == 0) ws[wid] = v;
  __syncthreads();
  if (wid == 0) {
    const int nw = (blockDim.x + 31) >> 5;
    dfloat t = lane < nw ? ws[lane] : dfloat(0.0f, 0.0f);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1)
      t = t + dfloat(__shfl_down_sync(0xffffffffu, t.hi, o), __shfl_down_sync(0xffffffffu, t.lo, o));
    if (lane == 0) atomicAdd(dst, (double)t.hi + (double)t.lo);
  }
}

// Wide scalars: double-float for FP32 storage, FP64 otherwise.
template <typename T> struct WideOf;
template <> struct WideOf<float> { using type = dfloat; };
template <> struct WideOf<double> { using type = double; };

// V consecutive values per thread (16-byte loads; V = 1 where a pointer is not 16-byte aligned).
template <typename T, int V> struct __align__(V * sizeof(T)) VecN {
  T v[V];
};

__device__ __forceinline__ void atomic_max_nonneg(double* dst, double v) {
  atomicMax(reinterpret_cast<unsigned long long*>(dst), (unsigned long long)__double_as_longlong(v));
}
__device__ __forceinline__ void atomic_min_d(double* dst, double v) {
  unsigned long long* a = reinterpret_cast<unsigned long long*>(dst);
  unsigned long long old = *a, assumed;
  do {
    assumed = old;
    if (__longlong_as_double((long long)assumed) <= v) break;
    old = atomicCAS(a, assumed, (unsigned long long)__double_as_longlong(v));
  } while (assumed != old);
}
__device__ __forceinline__ void atomic_max_d(double* dst, double v) {
  unsigned long long* a = reinterpret_cast<unsigned long long*>(dst);
  unsigned long long old = *a, assumed;
  do {
    assumed = old;
    if (__longlong_as_double((long long)assumed) >= v) break;
    old = atomicCAS(a, assumed, (unsigned long long)__double_as_longlong(v));
  } while (assumed != old);
}

// Periodic neighbours of flat index p: shifts and masks when every extent is a power of two,
// integer division otherwise.
struct Nb {
  int c, xm, xp, ym, yp, zm, zp;
};
__device__ __forceinline__ Nb neighbours(const Geo& g, int p) {
  if (!g.pow2) {
    const int x = p % g.nx, t = p / g.nx, y = t % g.ny, z = t / g.ny;
    const int sxy = g.nx * g.ny;
    const int rowbase = p - x, planebase = z * sxy, inplane = p - planebase;
    Nb n;
    n.c = p;
    n.xm = rowbase + (x == 0 ? g.nx - 1 : x - 1);
    n.xp = rowbase + (x == g.nx - 1 ? 0 : x + 1);
    n.ym = planebase + (y == 0 ? g.ny - 1 : y - 1) * g.nx + x;
    n.yp = planebase + (y == g.ny - 1 ? 0 : y + 1) * g.nx + x;
    n.zm = (z == 0 ? g.nz - 1 : z - 1) * sxy + inplane;
    n.zp = (z == g.nz - 1 ? 0 : z + 1) * sxy + inplane;
    return n;
  }
  const int mx = g.nx - 1, my = g.ny - 1, mz = g.nz - 1;
  const int sp = g.lx + g.ly;
  const int x = p & mx;
  const int y = (p >> g.lx) & my;
  const int z = p >> sp;
  const int rowbase = p - x;
  const int inplane = p & ((1 << sp) - 1);
  const int planebase = p - inplane;
  Nb n;
  n.c = p;
  n.xm = rowbase + ((x - 1) & mx);
  n.xp = rowbase + ((x + 1) & mx);
  n.ym = planebase + ((((y - 1) & my)) << g.lx) + x;
  n.yp = planebase + ((((y + 1) & my)) << g.lx) + x;
  n.zm = (((z - 1) & mz) << sp) + inplane;
  n.zp = (((z + 1) & mz) << sp) + inplane;
  return n;
}

template <typename T> __device__ __forceinline__ T gloc(T f) {  // g = 18 (f^2 - f)^2
  const T a = f * f - f;
  return (T)18 * a * a;
}
template <typename T> __device__ __forceinline__ T dW(T s) { return (T)36 * s * (s - (T)1) * ((T)2 * s - (T)1); }
template <typename T> __device__ __forceinline__ T d2W(T s) { return (T)36 * ((T)6 * s * s - (T)6 * s + (T)1); }
template <typename T> __device__ __forceinline__ T Wpot(T s) {
  const T a = s * s - s;
  return (T)18 * a * a;
}
template <typename T> __device__ __forceinline__ T find(T u) { return (T)3 * u * u - (T)2 * u * u * u; }
template <typename T> __device__ __forceinline__ T dfind(T u) { return (T)6 * u * ((T)1 - u); }
template <typename T> __device__ __forceinline__ bool in_band(T phi, T hi) {
  return fabs((T)2 * phi - (T)1) < hi;
}

// Delta_{S,h} u at p with face-averaged g (Eq. (2.3)); g evaluated from values gc, g-neighbours.
template <typename T>
__device__ __forceinline__ T surf_lap(const Geo& g, const ModelC<T>& mc, const Nb& n, const T* __restrict__ u,
                                      T gc, T gxm, T gxp, T gym, T gyp, T gzm, T gzp) {
  const T uc = u[n.c];
  T s = (((T)0.5 * (gxp + gc)) * (u[n.xp] - uc) - ((T)0.5 * (gc + gxm)) * (uc - u[n.xm])) * mc.ih2[0] +
        (((T)0.5 * (gyp + gc)) * (u[n.yp] - uc) - ((T)0.5 * (gc + gym)) * (uc - u[n.ym])) * mc.ih2[1];
  if (g.nz > 1)
    s += (((T)0.5 * (gzp + gc)) * (u[n.zp] - uc) - ((T)0.5 * (gc + gzm)) * (uc - u[n.zm])) * mc.ih2[2];
  return s;
}

// ---- pass-A prologues / epilogues ------------------------------------------------------
template <typename T> struct ProLoad {
  const T* a;
  __device__ T operator()(long long i) const { return a[i]; }
};
template <typename T> struct ProMul {
  const T* a;
  const T* b;
  __device__ T operator()(long long i) const { return a[i] * b[i]; }
};
template <typename T> struct EpiStore {
  static constexpr bool kPrefetch = false, kSums = false;
  using Acc = NoAcc;
  using Part = NoAcc;
  __device__ void prefetch(long long) const {}
  __device__ void fold(Part&, Acc&) const {}
  __device__ void finish(Acc&) const {}
  T* out;
  __device__ void operator()(long long i, T v) const { out[i] = v; }
};
// U = GU/G where G > delta, GU elsewhere (Sec. 3.3, recovery after Algorithm 1).
// u from the increment of G u over a stage: the inverse transform delivers
// d = GU_new - G u_base, and on the recovery set {G > delta} u = GU_new / G is formed as
// u_base + d / G (equal in exact arithmetic; the FP32 transform error then scales with the
// increment instead of with G u itself), elsewhere u = GU_new = G u_base + d (Algorithm 1).
__device__ __forceinline__ float div_inc(float a, float b) { return __fdividef(a, b); }
__device__ __forceinline__ double div_inc(double a, double b) { return a / b; }

// Epilogues with inputs of their own (EpiRecover) prefetch their cache lines into L2 before
// the inverse x transform of a row pair, so the loads after it find them on chip.
template <typename T> struct EpiRecover {
  static constexpr bool kPrefetch = true, kSums = false;
  using Acc = NoAcc;
  using Part = NoAcc;
  __device__ void fold(Part&, Acc&) const {}
  __device__ void finish(Acc&) const {}
  __device__ void prefetch(long long i) const {
    asm volatile("prefetch.global.L2 [%0];" ::"l"(G + i));
    asm volatile("prefetch.global.L2 [%0];" ::"l"(base + i));
  }
  T* out;
  const T* G;
  const T* base;
  T delta;
  __device__ void operator()(long long i, T v) const {
    const T gg = G[i];
    const T ub = base[i];
    // the quotient only forms the increment d / G, so the 2-ulp fast division suffices in FP32
    out[i] = gg > delta ? ub + div_inc(v, gg) : gg * ub + v;
  }
};
// phi^{n+1} and G^{n+1} = 18 (phi^2 - phi)^2 (Algorithm 1).
template <typename T> struct EpiPhiG {
  static constexpr bool kPrefetch = false, kSums = false;
  using Acc = NoAcc;
  using Part = NoAcc;
  __device__ void prefetch(long long) const {}
  __device__ void fold(Part&, Acc&) const {}
  __device__ void finish(Acc&) const {}
  T* phi;
  T* G;
  T* zero;   // optional: a field cleared in the same pass (the band-list R2 fills its band later)
  __device__ void operator()(long long i, T v) const {
    phi[i] = v;
    G[i] = gloc(v);
    if (zero) zero[i] = 0;
  }
};

// ---- pointwise / band kernels ----------------------------------------------------------

// R1 without its Laplacian term (Sec. 3.1), and W'(phi) - A1 phi whose spectrum receives
// kappa/(mu eps^2) lambda in pass B.  Delta phi and grad phi are spectral (pass-A outputs).
// V consecutive points per thread (16-byte loads and stores; V = 1 where u is not 16-byte
// aligned), so that six wide loads a thread are in flight: 256^3 FP32 124 -> 88 us for 537 MB.
// The FP64 form is bound by the FP64 pipe (70 instructions a point with its quotients by eps_phi
// and eps_u).  Products with reciprocals formed once would save 47 us a launch (128^3 coupled, three
// steps: 18.80 ms a pass against 19.08), for one rounding more in each quotient: not taken.
template <typename T, int V>
__global__ void __launch_bounds__(256) k_r1(Geo g, ModelC<T> mc, const T* __restrict__ phi, const T* __restrict__ lap,
                     const T* __restrict__ gx, const T* __restrict__ gy, const T* __restrict__ gz,
                     const T* __restrict__ u, const double* __restrict__ scal, double hvol,
                     T* __restrict__ out_rest, T* __restrict__ out_wm) {
  using VT = VecN<T, V>;
  const T e = mc.eps_phi, e2 = e * e;
  const T dvol = (T)(hvol * scal[S_VOL] - scal[S_A0]);
  const T c_a = mc.kappa / (mc.mu * e2);
  const T c_b = mc.kappa / (mc.mu * e2 * e2);
  const T c_c = mc.lambda_surf / (mc.mu * e2);
  const T c_l = mc.lambda_line / mc.mu, c_v = -(mc.M_area / mc.mu) * dvol, c_al = mc.alpha / mc.mu;
  const int nv = (int)(g.n / V);
  for (int q = blockIdx.x * blockDim.x + threadIdx.x; q < nv; q += gridDim.x * blockDim.x) {
    VT rv, wv;
    if (mc.linear_only) {
#pragma unroll
      for (int k = 0; k < V; ++k) rv.v[k] = wv.v[k] = 0;
      reinterpret_cast<VT*>(out_rest)[q] = rv;
      reinterpret_cast<VT*>(out_wm)[q] = wv;
      continue;
    }
    const VT fv = reinterpret_cast<const VT*>(phi)[q], Lv = reinterpret_cast<const VT*>(lap)[q];
    const VT xv = reinterpret_cast<const VT*>(gx)[q], yv = reinterpret_cast<const VT*>(gy)[q];
    VT zv{};
    if (g.nz > 1) zv = reinterpret_cast<const VT*>(gz)[q];
    const VT uv = reinterpret_cast<const VT*>(u)[q];
#pragma unroll
    for (int k = 0; k < V; ++k) {
      const T f = fv.v[k], L = Lv.v[k];
      const T ax = xv.v[k], ay = yv.v[k], az = zv.v[k];
      const T gn = sqrt(ax * ax + ay * ay + az * az);
      const T Wp = dW(f), Wpp = d2W(f);
      const T Wm = Wp - mc.A1 * f;
      const T uu = uv.v[k];
      T r = c_a * (Wpp - mc.A2) * (L - mc.A1 * f / e2) - (c_b * Wpp + c_c) * Wm;
      if (in_band(f, mc.band_hi)) {
        // line-tension term with Delta_{S,h} u (g = g(phi) at the faces), band points only
        const Nb n = neighbours(g, q * V + k);
        const T gzm = g.nz > 1 ? gloc(phi[n.zm]) : (T)0, gzp = g.nz > 1 ? gloc(phi[n.zp]) : (T)0;
        const T lu = surf_lap(g, mc, n, u, gloc(f), gloc(phi[n.xm]), gloc(phi[n.xp]), gloc(phi[n.ym]),
                              gloc(phi[n.yp]), gzm, gzp);
        r += c_l * (mc.eps_u * lu - gloc(f) * dW(uu) / mc.eps_u) * gn;
      }
      r += c_v * gn;
      r += c_al * (uu + mc.u0) * gn * (e * L - Wp / e);
      rv.v[k] = r;
      wv.v[k] = Wm;
    }
    reinterpret_cast<VT*>(out_rest)[q] = rv;
    reinterpret_cast<VT*>(out_wm)[q] = wv;
  }
}

// Membrane-velocity flux component d of g u v at q: v = -d_t phi grad phi / (|grad phi|^2 + 1e-12).
template <typename T>
__device__ __forceinline__ void adv_flux(const Geo& g, const ModelC<T>& mc, const T* __restrict__ phin,
                                         const T* __restrict__ phio, const T* __restrict__ u, int q,
                                         T& Fx, T& Fy, T& Fz) {
  const Nb n = neighbours(g, q);
  const T px = (phin[n.xp] - phin[n.xm]) * mc.i2h[0];
  const T py = (phin[n.yp] - phin[n.ym]) * mc.i2h[1];
  const T pz = g.nz > 1 ? (phin[n.zp] - phin[n.zm]) * mc.i2h[2] : (T)0;
  const T n2 = px * px + py * py + pz * pz + (T)1e-12;
  const T fq = phin[q];
  const T dt = (fq - phio[q]) / mc.tau;
  const T s = -gloc(fq) * u[q] * dt / n2;
  Fx = s * px;
  Fy = s * py;
  Fz = s * pz;
}

// R2 of the coupled OK equation (Sec. 3.1) at a band point p of phin.
template <typename T>
__device__ __forceinline__ T r2_coupled_at(const Geo& g, const ModelC<T>& mc, const T* __restrict__ phin,
                                           const T* __restrict__ phio, const T* __restrict__ u,
                                           const T* __restrict__ w, T mass, int p) {
  const T f = phin[p];
  const Nb n = neighbours(g, p);
  const T gc = gloc(f);
  const T gxm = gloc(phin[n.xm]), gxp = gloc(phin[n.xp]), gym = gloc(phin[n.ym]), gyp = gloc(phin[n.yp]);
  const T gzm = g.nz > 1 ? gloc(phin[n.zm]) : (T)0, gzp = g.nz > 1 ? gloc(phin[n.zp]) : (T)0;
  const T uc = u[p];
  const T sl = surf_lap(g, mc, n, u, gc, gxm, gxp, gym, gyp, gzm, gzp);
  const T guc = gc * uc;
  T lapgu = (gxp * u[n.xp] - (T)2 * guc + gxm * u[n.xm]) * mc.ih2[0] +
            (gyp * u[n.yp] - (T)2 * guc + gym * u[n.ym]) * mc.ih2[1];
  if (g.nz > 1) lapgu += (gzp * u[n.zp] - (T)2 * guc + gzm * u[n.zm]) * mc.ih2[2];
  T ax, ay, az, bx, by, bz;
  adv_flux(g, mc, phin, phio, u, n.xp, ax, ay, az);
  adv_flux(g, mc, phin, phio, u, n.xm, bx, by, bz);
  T div = (ax - bx) * mc.i2h[0];
  adv_flux(g, mc, phin, phio, u, n.yp, ax, ay, az);
  adv_flux(g, mc, phin, phio, u, n.ym, bx, by, bz);
  div += (ay - by) * mc.i2h[1];
  if (g.nz > 1) {
    adv_flux(g, mc, phin, phio, u, n.zp, ax, ay, az);
    adv_flux(g, mc, phin, phio, u, n.zm, bx, by, bz);
    div += (az - bz) * mc.i2h[2];
  }
  return mc.eps_u * (sl - mc.B1 * lapgu) + mc.B2 * guc - gc * dW(uc) / mc.eps_u - mc.gamma * gc * w[p] -
         mc.M * gc * mass - div;
}

// R2 on the band of phin over the whole grid, 0 elsewhere (operator entry point).
template <typename T>
__global__ void k_r2_coupled(Geo g, ModelC<T> mc, const T* __restrict__ phin, const T* __restrict__ phio,
                             const T* __restrict__ u, const T* __restrict__ w, const double* __restrict__ scal,
                             double hvol, T* __restrict__ out) {
  const T mass = (T)(hvol * scal[S_MASS]);
  for (int p = blockIdx.x * blockDim.x + threadIdx.x; p < (int)g.n; p += gridDim.x * blockDim.x) {
    const T f = phin[p];
    out[p] = (mc.linear_only || !in_band(f, mc.band_hi)) ? (T)0 : r2_coupled_at(g, mc, phin, phio, u, w, mass, p);
  }
}

// R2 at the points of the band list of phin only (the step: the rest of `out` was cleared
// when phin was formed).  Consecutive threads take consecutive band points, so the stencil
// work has no idle lanes.
template <typename T>
__global__ void k_r2_coupled_band(Geo g, ModelC<T> mc, const int* __restrict__ idx, const int* __restrict__ count,
                                  const T* __restrict__ phin, const T* __restrict__ phio, const T* __restrict__ u,
                                  const T* __restrict__ w, const double* __restrict__ scal, double hvol,
                                  T* __restrict__ out, unsigned long long* work) {
  const T mass = (T)(hvol * scal[S_MASS]);
  const int M = *count;
  if (work && blockIdx.x == 0 && threadIdx.x == 0) atomicAdd(work, (unsigned long long)M);
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < M; i += gridDim.x * blockDim.x) {
    const int p = idx[i];
    out[p] = mc.linear_only ? (T)0 : r2_coupled_at(g, mc, phin, phio, u, w, mass, p);
  }
}

// R2 of the fixed-membrane model: the Sec. 3 split of Eq. (2.1) with the operands of
// Eq. (2.16) (nonlocal operand g f(u), mass operand g (f(u) - ubar)); band from `mask`.
template <typename T>
__global__ void k_r2_fixed(Geo g, ModelC<T> mc, const T* __restrict__ G, const unsigned char* __restrict__ mask,
                           const T* __restrict__ u, const T* __restrict__ w, const double* __restrict__ scal,
                           double hvol, T* __restrict__ out) {
  const T mass = (T)(hvol * scal[S_MASS]);
  for (int p = blockIdx.x * blockDim.x + threadIdx.x; p < (int)g.n; p += gridDim.x * blockDim.x) {
    if (mc.linear_only || !mask[p]) {
      out[p] = 0;
      continue;
    }
    const Nb n = neighbours(g, p);
    const T gc = G[p];
    const T gxm = G[n.xm], gxp = G[n.xp], gym = G[n.ym], gyp = G[n.yp];
    const T gzm = g.nz > 1 ? G[n.zm] : (T)0, gzp = g.nz > 1 ? G[n.zp] : (T)0;
    const T uc = u[p];
    const T sl = surf_lap(g, mc, n, u, gc, gxm, gxp, gym, gyp, gzm, gzp);
    const T guc = gc * uc;
    T lapgu = (gxp * u[n.xp] - (T)2 * guc + gxm * u[n.xm]) * mc.ih2[0] +
              (gyp * u[n.yp] - (T)2 * guc + gym * u[n.ym]) * mc.ih2[1];
    if (g.nz > 1) lapgu += (gzp * u[n.zp] - (T)2 * guc + gzm * u[n.zm]) * mc.ih2[2];
    const T fp = dfind(uc);
    out[p] = mc.eps_u * (sl - mc.B1 * lapgu) + mc.B2 * guc - gc * dW(uc) / mc.eps_u - mc.gamma * gc * fp * w[p] -
             mc.M * gc * fp * mass;
  }
}

static __global__ void k_zero_off_band(long long n, const unsigned char* __restrict__ mask, void* x, int elem) {
  for (long long p = blockIdx.x * (long long)blockDim.x + threadIdx.x; p < n; p += (long long)gridDim.x * blockDim.x)
    if (!mask[p]) {
      if (elem == 8) reinterpret_cast<double*>(x)[p] = 0.0;
      else reinterpret_cast<float*>(x)[p] = 0.0f;
    }
}

template <typename T>
__global__ void k_axpy(long long n, const T* __restrict__ a, T c, const T* __restrict__ b, T* __restrict__ out) {
  for (long long p = blockIdx.x * (long long)blockDim.x + threadIdx.x; p < n; p += (long long)gridDim.x * blockDim.x)
    out[p] = a[p] + c * b[p];
}

// A0 = <phi^0, 1>_h when the caller left it unset.
static __global__ void k_set_a0(double* scal, double hvol) { scal[S_A0] = hvol * scal[S_VOL]; }

template <typename T> __global__ void k_gloc(long long n, const T* __restrict__ phi, T* __restrict__ G) {
  for (long long p = blockIdx.x * (long long)blockDim.x + threadIdx.x; p < n; p += (long long)gridDim.x * blockDim.x)
    G[p] = gloc(phi[p]);
}

// ---- FP64 reductions ---------------------------------------------------------------------
// Per-thread compensated sum in the storage precision: hi collects the rounded partial sums,
// lo the exact rounding error of each addition (Knuth's two-sum) plus any small parts the
// caller adds.  In FP32 it carries about twice the working precision, so the FP64 sums of
// the few per-thread partials match an FP64 accumulation while the per-element work stays
// on the FP32 pipes (FP64 arithmetic is a small fraction of the FP32 rate on this part).
template <typename T> struct CompSum {
  T hi = 0, lo = 0;
  __device__ __forceinline__ void add(T x) {
    const T s = hi + x;
    const T bp = s - hi;
    lo += (hi - (s - bp)) + (x - bp);
    hi = s;
  }
  __device__ __forceinline__ double value() const { return (double)hi + (double)lo; }
  __device__ __forceinline__ typename WideOf<T>::type wide() const {
    if constexpr (sizeof(T) == 4) return dfloat(hi, lo);
    else return hi + lo;
  }
};

// ubar = hi + lo in the storage precision (lo = 0 in FP64).
template <typename T> struct Ubar {
  T hi, lo;
};
template <typename T> __host__ __device__ inline Ubar<T> split_ubar(double ubar) {
  const T hi = (T)ubar;
  return Ubar<T>{hi, (T)(ubar - (double)hi)};
}

// One term G (x - ubar) of the mass sum.  FP32 forms it to about twice FP32 precision: ubar
// split into hi + lo, d = x - ubar as d_hi + d_lo (two-sum with the high part, then the low
// part), g d = rounded product + its rounding error (an FMA) + g d_lo.
__device__ __forceinline__ void add_mass(CompSum<float>& cs, float x, float g, Ubar<float> ub) {
  const float dh = x - ub.hi;
  const float bp = dh - x;
  const float dl = ((x - (dh - bp)) + (-ub.hi - bp)) - ub.lo;
  const float pr = g * dh;
  const float pe = fmaf(g, dh, -pr);
  cs.add(pr);
  cs.lo += fmaf(g, dl, pe);
}
__device__ __forceinline__ void add_mass(CompSum<double>& cs, double x, double g, Ubar<double> ub) {
  cs.add(g * ((x - ub.hi) - ub.lo));
}

// mode 0: sum a ; 1: sum G (u - ubar) ; 2: sum G (f(u) - ubar).  FP64 storage sums in FP64;
// FP32 storage forms each term to about twice FP32 precision (ubar split into hi + lo, the
// product's rounding error from an FMA) and sums with CompSum.  Four blocks per SM at most: each
// ends in a block sum.
template <typename T, int V>
__global__ void __launch_bounds__(256) k_reduce(long long n, int mode, const T* __restrict__ a,
                                                const T* __restrict__ G, double ubar, double* dst) {
  using VT = VecN<T, V>;
  const long long nv = n / V;
  const Ubar<T> ub = split_ubar<T>(ubar);
  CompSum<T> cs;
  double s = 0.0;
#pragma unroll 2
  for (long long p = blockIdx.x * (long long)blockDim.x + threadIdx.x; p < nv; p += (long long)gridDim.x * blockDim.x) {
    const VT av = reinterpret_cast<const VT*>(a)[p];
    VT gv{};
    if (mode != 0) gv = reinterpret_cast<const VT*>(G)[p];
#pragma unroll
    for (int k = 0; k < V; ++k) {
      const T x = av.v[k], g = gv.v[k];
      if constexpr (sizeof(T) == 8) {
        if (mode == 0) s += x;
        else s += g * ((mode == 1 ? x : find(x)) - ubar);
      } else {
        if (mode == 0) cs.add(x);
        else add_mass(cs, mode == 1 ? x : find(x), g, ub);
      }
    }
  }
  if constexpr (sizeof(T) == 8) block_add(s, dst);
  else block_add(cs.wide(), dst);
}

// ---- inverse-transform epilogues that also form a field sum ------------------------------
// The volume <phi, 1> and the mass sum G (u - ubar) of Sec. 3.3 (k_reduce modes 0 and 1)
// accumulate while pass A stores the field: a compensated sum over each row pair a thread
// stores (Part), folded into wide per-thread sums (Acc), one block sum per CTA added
// atomically at the end; the field is not read back.  The caller zeroes the targets.
template <typename T> struct Sums2 {
  CompSum<T> s0;
};
template <typename T> struct Acc2 {
  typename WideOf<T>::type s0 = typename WideOf<T>::type(0);
};

template <typename T> struct EpiStoreVol {
  static constexpr bool kPrefetch = false, kSums = true;
  using Acc = Acc2<T>;
  using Part = Sums2<T>;
  __device__ void prefetch(long long) const {}
  T* out;
  double* vol;
  __device__ void operator()(long long i, T v, Part& a) const {
    out[i] = v;
    a.s0.add(v);
  }
  __device__ void fold(Part& p, Acc& a) const { a.s0 = a.s0 + p.s0.wide(); }
  __device__ void finish(Acc& a) const { block_add(a.s0, vol); }
};

// EpiPhiG plus the volume of phi^{n+1}.
template <typename T> struct EpiPhiGVol {
  static constexpr bool kPrefetch = false, kSums = true;
  using Acc = Acc2<T>;
  using Part = Sums2<T>;
  __device__ void prefetch(long long) const {}
  T* phi;
  T* G;
  T* zero;
  double* vol;
  __device__ void operator()(long long i, T v, Part& a) const {
    phi[i] = v;
    G[i] = gloc(v);
    if (zero) zero[i] = 0;
    a.s0.add(v);
  }
  __device__ void fold(Part& p, Acc& a) const { a.s0 = a.s0 + p.s0.wide(); }
  __device__ void finish(Acc& a) const { block_add(a.s0, vol); }
};

// EpiRecover plus the mass sum of (G, u~).
template <typename T> struct EpiRecoverMass {
  static constexpr bool kPrefetch = true, kSums = true;
  using Acc = Acc2<T>;
  using Part = Sums2<T>;
  __device__ void prefetch(long long i) const {
    asm volatile("prefetch.global.L2 [%0];" ::"l"(G + i));
    asm volatile("prefetch.global.L2 [%0];" ::"l"(base + i));
  }
  T* out;
  const T* G;
  const T* base;
  T delta;
  Ubar<T> ub;
  double* mass;
  __device__ void operator()(long long i, T v, Part& a) const {
    const T gg = G[i];
    const T b = base[i];
    const T o = gg > delta ? b + div_inc(v, gg) : gg * b + v;
    out[i] = o;
    add_mass(a.s0, o, gg, ub);
  }
  __device__ void fold(Part& p, Acc& a) const { a.s0 = a.s0 + p.s0.wide(); }
  __device__ void finish(Acc& a) const { block_add(a.s0, mass); }
};

// ---- double-float transforms of the membrane state (FP32-mixed form) ----------------------
// Pass-A prologue of the double-float forward transform of an FP32 field.
struct ProWiden {
  const float* a;
  __device__ dfloat operator()(long long i) const { return dfloat(a[i]); }
};

// phi^{n+1} from the inverse transform of the phi-stage increment (FP32-mixed form): the
// real-space phi is carried as hi + lo (hi the FP32 field the other kernels read, lo its
// FP32 remainder), phi^{n+1} = (phi^n_hi + phi^n_lo) + d in double-float; G = 18 (phi (phi -
// 1))^2 is formed from the double-float value with phi - 1 as (hi - 1) + lo (hi - 1 is exact
// for hi in [0.5, 2]), so 1 - phi near the inner edge of the membrane and phi near the outer
// edge both keep their relative accuracy in G.  Also clears the R2 field and forms the volume.
struct EpiPhiIncVol {
  static constexpr bool kPrefetch = true, kSums = true;
  using Acc = Acc2<float>;
  using Part = Sums2<float>;
  __device__ void prefetch(long long i) const {
    asm volatile("prefetch.global.L2 [%0];" ::"l"(cur + i));
    asm volatile("prefetch.global.L2 [%0];" ::"l"(lo + i));
  }
  const float* cur;   // phi^n (high part)
  float* lo;          // low part, phi^n on entry, phi^{n+1} on exit (in place)
  float* nxt;         // phi^{n+1} (high part)
  float* G;
  float* zero;
  double* vol;
  __device__ void operator()(long long i, float d, Part& a) const {
    const dfloat p = add_f(dfloat(cur[i], lo[i]), d);
    const float m1 = __fadd_rn(__fsub_rn(p.hi, 1.0f), p.lo);
    const float q = p.hi * m1;
    nxt[i] = p.hi;
    lo[i] = p.lo;
    G[i] = 18.0f * q * q;
    if (zero) zero[i] = 0.0f;
    a.s0.add(p.hi);
  }
  __device__ void fold(Part& p, Acc& a) const { a.s0 = a.s0 + p.s0.wide(); }
  __device__ void finish(Acc& a) const { block_add(a.s0, vol); }
};

// Energy terms of Eq. (2.16) except the nonlocal one, plus the bound statistics and <phi,1>.
// FP32 storage forms every term to about twice FP32 precision (exact differences and sums by
// two-sum, product errors by FMA) and sums it with CompSum, on the FP32 pipes: the FP64 form of
// the same sums is bound by the FP64 pipe (about 50 FP64 instructions a point; 256^3: 1386 us
// with it and one atomic per thread and statistic, against a 201 MB read).  max |2U - 1| is
// taken at min U or max U, so the two extrema are all that the points keep.
struct EnergySum {   // sum of (a + b) d^2, or of a d, from FP32 values
  CompSum<float> s;
  __device__ __forceinline__ static void two_sum(float a, float b, float& h, float& l) {
    h = __fadd_rn(a, b);
    const float v = __fsub_rn(h, a);
    l = __fadd_rn(__fsub_rn(a, __fsub_rn(h, v)), __fsub_rn(b, v));
  }
  __device__ __forceinline__ void grad(float ga, float gb, float ua, float ub) {
    float gh, gl, dh, dl;
    two_sum(ga, gb, gh, gl);
    two_sum(ub, -ua, dh, dl);
    const float p = __fmul_rn(dh, dh);
    const float e = __fmaf_rn(2.0f * dh, dl, __fmaf_rn(dh, dh, -p));
    const float t = __fmul_rn(gh, p);
    const float te = __fmaf_rn(gl, p, __fmaf_rn(gh, e, __fmaf_rn(gh, p, -t)));
    s.add(t);
    s.lo += te;
  }
  __device__ __forceinline__ void prod(float a, float b) {
    const float t = __fmul_rn(a, b);
    s.add(t);
    s.lo += __fmaf_rn(a, b, -t);
  }
};
// WIDE: FP64 sums also for FP32 storage, where the others left FP32's range (|u| from about 1e9).
template <typename T, bool WIDE>
__global__ void __launch_bounds__(256) k_energy_terms(Geo g, ModelC<T> mc, const T* __restrict__ G,
                                                      const T* __restrict__ U, const T* __restrict__ phi, double* scal) {
  double sg = 0, sw = 0, sm = 0, sv = 0;
  T mn = (T)INFINITY, mx = -(T)INFINITY;
  if constexpr (!WIDE) {
    EnergySum gx{}, gy{}, gz{}, w{};
    CompSum<float> m{}, v{};
    const Ubar<float> ub{mc.ubar, 0.0f};
    for (int p = blockIdx.x * blockDim.x + threadIdx.x; p < (int)g.n; p += gridDim.x * blockDim.x) {
      const Nb n = neighbours(g, p);
      const float gc = G[p], uc = U[p];
      gx.grad(gc, G[n.xp], uc, U[n.xp]);
      gy.grad(gc, G[n.yp], uc, U[n.yp]);
      if (g.nz > 1) gz.grad(gc, G[n.zp], uc, U[n.zp]);
      w.prod(gc, Wpot(uc));
      add_mass(m, find(uc), gc, ub);
      v.add(phi[p]);
      if (gc > mc.delta) {
        mn = fminf(mn, uc);
        mx = fmaxf(mx, uc);
      }
    }
    sg = 0.5 * (gx.s.value() * (double)mc.ih2[0] + gy.s.value() * (double)mc.ih2[1]);
    if (g.nz > 1) sg += 0.5 * gz.s.value() * (double)mc.ih2[2];
    sw = w.s.value();
    sm = m.value();
    sv = v.value();
  } else {
    for (int p = blockIdx.x * blockDim.x + threadIdx.x; p < (int)g.n; p += gridDim.x * blockDim.x) {
      const Nb n = neighbours(g, p);
      const double gc = G[p], uc = U[p];
      const double dx = (double)U[n.xp] - uc, dy = (double)U[n.yp] - uc;
      sg += 0.5 * (gc + (double)G[n.xp]) * dx * dx * (double)mc.ih2[0] +
            0.5 * (gc + (double)G[n.yp]) * dy * dy * (double)mc.ih2[1];
      if (g.nz > 1) {
        const double dz = (double)U[n.zp] - uc;
        sg += 0.5 * (gc + (double)G[n.zp]) * dz * dz * (double)mc.ih2[2];
      }
      sw += gc * (double)Wpot(U[p]);
      sm += gc * ((double)find(U[p]) - (double)mc.ubar);
      sv += (double)phi[p];
      if (gc > (double)mc.delta) {
        mn = fmin(mn, (T)uc);
        mx = fmax(mx, (T)uc);
      }
    }
  }
  block_add(sg, scal + S_GRAD);
  block_add(sw, scal + S_WELL);
  block_add(sm, scal + S_MASSF);
  block_add(sv, scal + S_VOLE);
  // extrema: one warp value, then the first warp's, then one atomic per block
  __shared__ T wmn[32], wmx[32];
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    mn = fmin(mn, __shfl_down_sync(0xffffffffu, mn, o));
    mx = fmax(mx, __shfl_down_sync(0xffffffffu, mx, o));
  }
  if ((threadIdx.x & 31) == 0) {
    wmn[threadIdx.x >> 5] = mn;
    wmx[threadIdx.x >> 5] = mx;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int k = 1; k < (int)(blockDim.x >> 5); ++k) {
      mn = fmin(mn, wmn[k]);
      mx = fmax(mx, wmx[k]);
    }
    if (mn <= mx) {
      const double lo = mn, hi = mx;
      atomic_max_nonneg(scal + S_MAXB, fmax(fabs(2.0 * lo - 1.0), fabs(2.0 * hi - 1.0)));
      atomic_min_d(scal + S_UMIN, lo);
      atomic_max_d(scal + S_UMAX, hi);
    }
  }
}

template <typename T>
__global__ void k_check_finite(long long n, const T* __restrict__ a, int* flag) {
  for (long long p = blockIdx.x * (long long)blockDim.x + threadIdx.x; p < n; p += (long long)gridDim.x * blockDim.x)
    if (!isfinite(a[p])) {
      atomicOr(flag, 1);
      return;
    }
}

// ---- narrow-band compaction: ballot + scan into an ascending index list ----------------
constexpr int kCompactBlock = 1024;

template <typename T>
__global__ void k_band_count(long long n, const T* __restrict__ phi, T hi, unsigned char* __restrict__ mask,
                             int* __restrict__ bcount) {
  const long long p = blockIdx.x * (long long)kCompactBlock + threadIdx.x;
  const bool b = (p < n) && in_band(phi[p], hi);
  if (p < n) mask[p] = b ? 1 : 0;
  const unsigned bal = __ballot_sync(0xffffffffu, b);
  __shared__ int wc[32];
  if ((threadIdx.x & 31) == 0) wc[threadIdx.x >> 5] = __popc(bal);
  __syncthreads();
  if (threadIdx.x < 32) {
    int v = wc[threadIdx.x];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    if (threadIdx.x == 0) bcount[blockIdx.x] = v;
  }
}

// The grid's band, 4 points per thread (one 16-byte load of phi per thread in FP32, one
// 4-byte mask store): a block covers kCompactWide consecutive points.  Needs n % 4 == 0 and
// a 16-byte aligned phi; k_band_scatter4 uses the same blocking.
constexpr int kCompactWide = 4 * kCompactBlock;

__device__ __forceinline__ void load4(const float* p, float (&f)[4]) {
  const float4 v = *reinterpret_cast<const float4*>(p);
  f[0] = v.x; f[1] = v.y; f[2] = v.z; f[3] = v.w;
}
__device__ __forceinline__ void load4(const double* p, double (&f)[4]) {
  const double2 a = *reinterpret_cast<const double2*>(p), b = *reinterpret_cast<const double2*>(p + 2);
  f[0] = a.x; f[1] = a.y; f[2] = b.x; f[3] = b.y;
}

template <typename T>
__global__ void k_band_count4(long long n, const T* __restrict__ phi, T hi, unsigned char* __restrict__ mask,
                              int* __restrict__ bcount) {
  const long long p0 = blockIdx.x * (long long)kCompactWide + 4LL * threadIdx.x;
  int c = 0;
  if (p0 < n) {
    T f[4];
    load4(phi + p0, f);
    uchar4 m;
    m.x = in_band(f[0], hi) ? 1 : 0;
    m.y = in_band(f[1], hi) ? 1 : 0;
    m.z = in_band(f[2], hi) ? 1 : 0;
    m.w = in_band(f[3], hi) ? 1 : 0;
    *reinterpret_cast<uchar4*>(mask + p0) = m;
    c = m.x + m.y + m.z + m.w;
  }
  c = __reduce_add_sync(0xffffffffu, c);
  __shared__ int wc[32];
  if ((threadIdx.x & 31) == 0) wc[threadIdx.x >> 5] = c;
  __syncthreads();
  if (threadIdx.x < 32) {
    int v = (threadIdx.x < (blockDim.x >> 5)) ? wc[threadIdx.x] : 0;
    v = __reduce_add_sync(0xffffffffu, v);
    if (threadIdx.x == 0) bcount[blockIdx.x] = v;
  }
}

// Block counts of a uint8 mask, 4 points per thread (kCompactWide blocking; n % 4 == 0).
static __global__ void k_mask_count4(long long n, const unsigned char* __restrict__ mask, int* __restrict__ bcount) {
  const long long p0 = blockIdx.x * (long long)kCompactWide + 4LL * threadIdx.x;
  int c = 0;
  if (p0 < n) {
    const uchar4 m = *reinterpret_cast<const uchar4*>(mask + p0);
    c = m.x + m.y + m.z + m.w;
  }
  c = __reduce_add_sync(0xffffffffu, c);
  __shared__ int wc[32];
  if ((threadIdx.x & 31) == 0) wc[threadIdx.x >> 5] = c;
  __syncthreads();
  if (threadIdx.x < 32) {
    int v = (threadIdx.x < (blockDim.x >> 5)) ? wc[threadIdx.x] : 0;
    v = __reduce_add_sync(0xffffffffu, v);
    if (threadIdx.x == 0) bcount[blockIdx.x] = v;
  }
}

// Index list and inverse map from the mask, 4 points per thread, ascending (kCompactWide
// blocking, boff = exclusive block offsets).
static __global__ void k_band_scatter4(long long n, const unsigned char* __restrict__ mask,
                                       const int* __restrict__ boff, int* __restrict__ idx, int* __restrict__ bmap) {
  const long long p0 = blockIdx.x * (long long)kCompactWide + 4LL * threadIdx.x;
  uchar4 m = make_uchar4(0, 0, 0, 0);
  if (p0 < n) m = *reinterpret_cast<const uchar4*>(mask + p0);
  const int c = m.x + m.y + m.z + m.w;
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  int inc = c;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int t = __shfl_up_sync(0xffffffffu, inc, o);
    if (lane >= o) inc += t;
  }
  __shared__ int wc[32];
  if (lane == 31) wc[wid] = inc;
  __syncthreads();
  if (threadIdx.x < 32) {
    const int v = (lane < (int)(blockDim.x >> 5)) ? wc[lane] : 0;
    int w = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int t = __shfl_up_sync(0xffffffffu, w, o);
      if (lane >= o) w += t;
    }
    wc[lane] = w - v;
  }
  __syncthreads();
  int i = boff[blockIdx.x] + wc[wid] + inc - c;
  const unsigned char mm[4] = {m.x, m.y, m.z, m.w};
#pragma unroll
  for (int e = 0; e < 4; ++e)
    if (mm[e]) {
      idx[i] = (int)(p0 + e);
      bmap[p0 + e] = i;
      ++i;
    }
}

// Block counts of a uint8 mask (same blocking as k_band_count).
static __global__ void k_mask_count(long long n, const unsigned char* __restrict__ mask, int* __restrict__ bcount) {
  const long long p = blockIdx.x * (long long)kCompactBlock + threadIdx.x;
  const bool b = (p < n) && mask[p];
  const unsigned bal = __ballot_sync(0xffffffffu, b);
  __shared__ int wc[32];
  if ((threadIdx.x & 31) == 0) wc[threadIdx.x >> 5] = __popc(bal);
  __syncthreads();
  if (threadIdx.x < 32) {
    int v = wc[threadIdx.x];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    if (threadIdx.x == 0) bcount[blockIdx.x] = v;
  }
}

// Exclusive scan of nb block counts in place (single block); total -> *count.
static __global__ void k_band_scan(int nb, int* __restrict__ bcount, int* __restrict__ count) {
  __shared__ int part[1024];
  const int per = (nb + blockDim.x - 1) / blockDim.x;
  const int lo = threadIdx.x * per, hi = min(nb, lo + per);
  int s = 0;
  for (int i = lo; i < hi; ++i) s += bcount[i];
  part[threadIdx.x] = s;
  __syncthreads();
  for (int off = 1; off < (int)blockDim.x; off <<= 1) {
    const int v = threadIdx.x >= (unsigned)off ? part[threadIdx.x - off] : 0;
    __syncthreads();
    part[threadIdx.x] += v;
    __syncthreads();
  }
  int run = part[threadIdx.x] - s;
  for (int i = lo; i < hi; ++i) {
    const int c = bcount[i];
    bcount[i] = run;
    run += c;
  }
  if (threadIdx.x == blockDim.x - 1) *count = part[threadIdx.x];
}

static __global__ void k_band_scatter(long long n, const unsigned char* __restrict__ mask, const int* __restrict__ boff,
                               int* __restrict__ idx, int* __restrict__ bmap) {
  const long long p = blockIdx.x * (long long)kCompactBlock + threadIdx.x;
  const bool b = (p < n) && mask[p];
  const unsigned bal = __ballot_sync(0xffffffffu, b);
  __shared__ int wc[32];
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  if (lane == 0) wc[wid] = __popc(bal);
  __syncthreads();
  if (threadIdx.x < 32) {
    int v = wc[lane];
    int inc = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int t = __shfl_up_sync(0xffffffffu, inc, o);
      if (lane >= o) inc += t;
    }
    wc[lane] = inc - v;
  }
  __syncthreads();
  if (b) {
    const int i = boff[blockIdx.x] + wc[wid] + __popc(bal & ((1u << lane) - 1u));
    idx[i] = (int)p;
    bmap[p] = i;
  }
}

// ---- band CG for (-Delta_{S,h}) w = f - mean on the band ---------------------------------
// The band operator in compact form: for band node i (grid point p = idx[i]) and each of its
// 2d faces, c = (G_p + G_q)/(2 h^2) when the neighbour q is also a band node, else 0 (zero
// flux across the band edge); (A v)_i = sum_faces c (v_i - v_q).  Vectors are compact
// (length M, band order), so every CG phase streams contiguous arrays.
template <typename T> struct CGVec {
  T *x, *r, *p, *q;       // compact vectors of the solve
  float *b, *e, *o, *t;   // level-0 vectors of the multigrid cycle
  float* idg;             // inverse diagonal
  T* c;                   // face coefficients, c[d * cap + i], d = x+, x-, y+, y-, z+, z-
  float* c32;             // the same for the multigrid cycle, times csc (FP32 storage: c itself)
  __half* c16;            // the same in FP16 for the multigrid sweeps (FP32 storage only, else null)
  int* nb;                // compact index of the face neighbour (i itself when absent)
  int cap;
  // large FP32 bands, whose matrix is read from memory in every sweep: the FP16 couplings with the
  // inverse diagonal (16 B) and the y and z neighbours as 16-bit offsets (8 B), instead of 12 + 4
  // and 24 B in 13 loads; *wide is set where an offset does not fit or an x neighbour is not next
  // in the list (a band across the periodic boundary), and the full lists are read.  Null: not kept.
  uint4* pk;
  short4* nd;
  int* wide;
  T csc;                  // FP64 storage: a power of two near h^2, which takes c32 to order one
};

template <typename T>
__global__ void k_cg_setup(Geo g, ModelC<T> mc, const int* __restrict__ idx, const int* __restrict__ count,
                           const unsigned char* __restrict__ mask, const int* __restrict__ bmap,
                           const T* __restrict__ G, CGVec<T> v, int* cc_flags) {
  const int M = *count;
  // labelling: component count, fallback flag, the fallback's barrier word
  if (blockIdx.x == 0 && threadIdx.x < 3) cc_flags[threadIdx.x] = 0;
  const int nd = g.nz > 1 ? 6 : 4;
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < M; i += gridDim.x * blockDim.x) {
    const int p = idx[i];
    const Nb n = neighbours(g, p);
    const int q[6] = {n.xp, n.xm, n.yp, n.ym, n.zp, n.zm};
    const T gc = G[p];
    float d = 0;
    int off[6];
    __half hc[6];
#pragma unroll
    for (int f = 0; f < 6; ++f) {
      T c = 0;
      int j = i;
      if (f < nd && mask[q[f]]) {
        c = (T)0.5 * (gc + G[q[f]]) * mc.ih2[f >> 1];
        j = bmap[q[f]];
      }
      v.c[f * v.cap + i] = c;
      const float cf = sizeof(T) == 4 ? (float)c : (float)(c * v.csc);
      if (sizeof(T) == 8) v.c32[f * v.cap + i] = cf;
      if (v.c16) v.c16[f * v.cap + i] = __float2half_rn(cf);
      v.nb[f * v.cap + i] = j;
      off[f] = j - i;
      hc[f] = __float2half_rn(cf);
      d += cf;
    }
    const float di = d > 0.0f ? 1.0f / d : 1.0f;
    v.idg[i] = di;
    if (v.pk) {
      uint4 p;
      unsigned* w = reinterpret_cast<unsigned*>(&p);
#pragma unroll
      for (int f = 0; f < 3; ++f) w[f] = __half_as_ushort(hc[2 * f]) | ((unsigned)__half_as_ushort(hc[2 * f + 1]) << 16);
      w[3] = __float_as_uint(di);
      v.pk[i] = p;
      v.nd[i] = make_short4((short)off[2], (short)off[3], (short)off[4], (short)off[5]);
      bool fits = (off[0] == 0 || off[0] == 1) && (off[1] == 0 || off[1] == -1);
#pragma unroll
      for (int f = 2; f < 6; ++f) fits = fits && off[f] == (int)(short)off[f];
      if (!fits) *v.wide = 1;
    }
  }
}

// Zero the solution on nodes of the previous band that left the band.
static __global__ void k_zero_left(const int* __restrict__ old_idx, const int* __restrict__ old_count,
                            const unsigned char* __restrict__ mask, void* x, int elem) {
  const int M = *old_count;
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < M; i += gridDim.x * blockDim.x) {
    const int p = old_idx[i];
    if (!mask[p]) {
      if (elem == 8) reinterpret_cast<double*>(x)[p] = 0.0;
      else reinterpret_cast<float*>(x)[p] = 0.0f;
    }
  }
}

// ---- connected components of the band (per-component mean removal of the band solve) ----
// The band operator is singular on every connected band component (6-neighbour, periodic),
// so the right-hand side and the solution are projected to zero mean per component (the
// whole-domain mean removal of Sec. 2.1 applied to each component).  Components come from a
// lock-free union-find over the band's neighbour lists: every link points from a larger node
// index to a smaller one, so each chase follows strictly decreasing indices and ends, and a
// failed link means another thread made progress (each loop is bounded by the node count).
constexpr int kCompCap = 4096;   // components the band solve supports (more: status 8)
// Component count of a band whose labelling gave up: negative whatever the blocks that were still
// counting add to it.
constexpr int kNoComponents = -(1 << 30);

__device__ __forceinline__ int cc_root(int* __restrict__ parent, int v) {
  int cur = __ldcg(parent + v);
  if (cur == v) return v;
  int prev = v;
  for (;;) {
    const int next = __ldcg(parent + cur);
    if (next >= cur) break;                // cur is a root (parent[cur] == cur)
    parent[prev] = next;                   // path halving; the value only ever decreases
    prev = cur;
    cur = next;
  }
  return cur;
}

// Per-component sums of one pass over the band: components below kCompShared accumulate in
// shared memory (one global atomic per block and component), others per warp group (lanes
// holding the same component combine their values, one atomic per group).  Every thread of
// the block calls begin() and end(); add() may be called under divergence.
constexpr int kCompShared = 64;
struct CompAcc {
  double* sh;    // kCompShared doubles of shared memory
  double* dst;   // global accumulators, one per component
  int C;
  __device__ void begin() {
    for (int k = threadIdx.x; k < kCompShared; k += blockDim.x) sh[k] = 0.0;
    __syncthreads();
  }
  __device__ void add(int c, double v) {
    if (c < kCompShared) {
      atomicAdd(sh + c, v);
      return;
    }
    const unsigned act = __activemask();
    const unsigned grp = __match_any_sync(act, c);
    double s = 0.0;
    for (unsigned m = grp; m; m &= m - 1) s += __shfl_sync(grp, v, __ffs(m) - 1);
    if ((int)(threadIdx.x & 31) == __ffs(grp) - 1) atomicAdd(dst + c, s);
  }
  __device__ void end() {
    __syncthreads();
    const int n = C < kCompShared ? C : kCompShared;
    for (int k = threadIdx.x; k < n; k += blockDim.x)
      if (sh[k] != 0.0) atomicAdd(dst + k, sh[k]);
    __syncthreads();
  }
};

struct CGCtl {
  unsigned* bar;        // the grid barrier's word
  int* status;          // plan status word
  int* iters;           // out: iterations
  double* resid;        // out: relative residual
  double rtol;
  int maxit;
  long long budget;     // clock cycles a barrier may wait
  unsigned long long* work;  // accumulates band nodes x CG iterations (measurement)
  const int* ncomp;     // connected band components (device)
  const int* comp;      // component of each band node
  const double* csize;  // nodes per component
  double* csum;         // 2 kCompCap FP64 accumulators (zeroed by the solve): f, then x
};

// Inside the band solve every global vector that the kernel itself writes is read with __ldcg:
// an L2 load, never the read-only path that a const __restrict__ pointer would allow, which is
// only valid for data that no thread writes during the launch.  The couplings, neighbour lists
// and level maps are built by earlier launches and are read normally.

// Grid-wide barrier for a cooperative launch on one word (barrier.h; zeroed before the launch):
// each block learns its barrier from the value its own arrival returned, so nothing is reset
// between barriers.  The block's writes are published by the block barrier followed by an
// acquire-release add at GPU scope; blocks that arrive early poll with acquire loads, and
// the last one to arrive takes its acquire from the add itself (without it, its L1 could
// still hold lines that other blocks rewrote during the phase).  The spin has a clock budget: a
// block whose budget runs out, or (HEED) that finds the status word set by an earlier failure,
// closes the word, and the barrier then fails in every block; one that was complete by then
// passes in every block.  Returns false for a failed barrier, with the status word set
// (ETD_ETIMEOUT unless something else was there).
__device__ __forceinline__ unsigned atom_add_acq_rel_gpu(unsigned* p, unsigned v) {
  unsigned old;
  asm volatile("atom.acq_rel.gpu.global.add.u32 %0, [%1], %2;" : "=r"(old) : "l"(p), "r"(v) : "memory");
  return old;
}
__device__ __forceinline__ unsigned ld_acquire_gpu(const unsigned* p) {
  unsigned v;
  asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}

template <bool HEED = true> __device__ __forceinline__ bool grid_sync(const CGCtl& c) {
  __syncthreads();
  __shared__ int ok;
  if (threadIdx.x == 0) {
    const unsigned nb = gridDim.x;
    // the status word is read along with the arrival, not after it (one L2 latency less)
    const int st = HEED ? *(volatile int*)c.status : 0;
    const unsigned old = atom_add_acq_rel_gpu(c.bar, 1u);
    const unsigned target = bar_target(old, nb);
    unsigned w = old + 1u;
    if (!bar_decided(w, target)) {
      const long long t0 = clock64();
      while (!bar_decided(w = ld_acquire_gpu(c.bar), target)) {
        if (st != 0 || clock64() - t0 > c.budget) {
          // the swap fails only where another block arrived or closed the word: look again
          if (atomicCAS(c.bar, w, bar_closed(target)) != w) continue;
          w = bar_closed(target);
          break;
        }
        __nanosleep(32);
      }
    }
    ok = bar_passed(w, target, nb);
    if (!ok) atomicCAS(c.status, 0, 6);
  }
  __syncthreads();
  return ok;
}

// ---- aggregation multigrid preconditioner for the band CG ---------------------------------
// Level l lives on the grid coarsened 2x per axis l times (z only in 3D); its nodes are the
// cells that contain at least one node of level l-1 (an aggregate of up to 2x2x2 nodes).
// With piecewise-constant prolongation P the Galerkin operator P^T A P of a graph Laplacian
// is again a graph Laplacian whose coupling between two neighbouring aggregates is the sum
// of the fine couplings crossing between them, so every level keeps the 7-point compact
// form (c, nb, inverse diagonal).  The preconditioner is one symmetric V(nu,nu) cycle whose
// smoother is weighted Jacobi; with nu = 2 the two sweeps use the weight pair w1, w2 of the
// degree-2 Chebyshev polynomial in D^-1 A (the two sweeps commute, so the cycle stays
// symmetric), and the coarsest level takes an even number of sweeps with the same pair.
constexpr int kMGMax = 7;

}  // namespace etd
