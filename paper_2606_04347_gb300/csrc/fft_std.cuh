// Pass B of the transform entry points: between the two-pass intermediate and the standard half
// spectrum [kz][ky][kx].
#pragma once
#include "fft.cuh"

namespace etd {

// A pencil block holds one kx, 8 bytes of every 32-byte sector of a standard-layout row; KB of
// them side by side are staged in the tile, so that KB consecutive kx go out (or come in) from
// consecutive lanes: 1.6 sectors for three values where passB moves three.
constexpr int kStdThreads = 384;

// Pencil blocks per CTA of passB_std, 0 where passB is taken.  FP32 only (16-byte FP64 values
// already fill half a sector, and those launches are bound by the FP64 pipe), power-of-two nz of 64
// or more, a tile of which two CTAs fit an SM while two CTAs for each SM are left.  Per launch,
// passB -> passB_std:
//   forward, 3 blocks or more: 256^3 92 -> 72 us, 256x256x128 44.7 -> 34.2, 256x128x128
//     22.3 -> 13.0, 256x256x64 22.2 -> 12.6, 128^3 15.2 -> 11.5, 128x256x256 45 -> 43, 256x128x256
//     43 either way; two blocks lose (96x256x256 31.5 -> 39.6);
//   inverse, 6 or more (a whole sector) in a tile of 64 KB: 256x128x128 19.2 -> 13.2, 256x256x64
//     19.8 -> 13.0, 256x32x256 10.8 -> 8.9; beyond, it loses (128^3, 3 blocks: 11.0 -> 12.4;
//     256x128x256, 104 KB: 34.4 -> 45.9; what holds the large tiles' loads up was not found).
inline int std_blocks(const Geo& g, size_t csize, int sms, bool inv) {
  if (csize != 8 || g.nz < 64 || fft_family(g.nz) != 0 || (g.Y1 & (g.Y1 - 1))) return 0;
  for (int kb = 8; kb > g.KB && kb >= (inv ? 6 : 3); --kb)
    if ((g.nxh + kb - 1) / kb * g.Y2 >= 2 * sms && kb * g.Y1 * pitch_b(g.nz) * csize <= 113 * 1024)
      return inv && kb * g.Y1 * pitch_b(g.nz) * csize > 64 * 1024 ? 0 : kb;
  return 0;
}

// Row transforms in place in the tile (Y1 kbn rows, one team each, as many rounds as it takes).
template <typename C, int R, int S, bool INV>
__device__ __forceinline__ void std_rows(int nrows, C* tile, int rs, const C* __restrict__ twz) {
  const int t = threadIdx.x & (S - 1);
  const int nteams = blockDim.x / S, wteam = (int)(threadIdx.x & ~31u) / S;
  for (int r = 0; wteam + r < nrows; r += nteams) {
    const int row = threadIdx.x / S + r;
    const bool ok = row < nrows;
    C* r0 = tile + (ok ? row : 0) * rs;
    C v[R];
#pragma unroll
    for (int j = 0; j < R; ++j) v[j] = ok ? r0[pad16(t + S * j)] : C{0, 0};
    team_fft<C, R, S, INV>(v, t, r0, twz, ok);
    __syncwarp();
    if (ok) {
#pragma unroll
      for (int j = 0; j < R; ++j) r0[pad16(t + S * j)] = v[j];
    }
  }
}

// src: the intermediate (forward) or the standard half spectrum (inverse); dst the other one.
template <typename T, bool INV>
__global__ void __launch_bounds__(kStdThreads, 2) passB_std(Geo g, const typename Cplx<T>::type* __restrict__ src,
                                                           typename Cplx<T>::type* __restrict__ dst,
                                                           const typename Cplx<T>::type* __restrict__ twz, T scale) {
  using C = typename Cplx<T>::type;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  C* tile = reinterpret_cast<C*>(smem_raw);
  const int rs = pitch_b(g.nz);
  // all kx of a ky residue before the next one: the CTAs at work together share whole rows in L2
  const int nkb = (g.nxh + g.KB - 1) / g.KB;
  const int k2 = blockIdx.x / nkb, kx0 = (blockIdx.x % nkb) * g.KB;
  const int kbn = min(g.KB, g.nxh - kx0);
  const long long cb = ((long long)(k2 * g.nxh + kx0) * g.Y1) * g.nz;
  if (!INV) {
    passB_cols_any<T, false>(g, kbn, src, cb, tile, rs, nullptr);
    __syncthreads();
  }
  // standard-layout accesses: a thread keeps its kx, consecutive lanes take kx, then k1, then kz
  const int qs = blockDim.x / kbn, kxl = threadIdx.x % kbn, q0 = threadIdx.x / kbn;
  const int ly = __ffs(g.Y1) - 1, nq = q0 < qs ? g.Y1 * g.nz : 0;
  const auto at_std = [&](int q) {
    const int k1 = q & (g.Y1 - 1), kz = q >> ly;
    return ((long long)kz * g.ny + k2 + g.Y2 * k1) * g.nxh + kx0 + kxl;
  };
  const auto at_tile = [&](int q) { return (kxl * g.Y1 + (q & (g.Y1 - 1))) * rs + pad16(q >> ly); };
  constexpr int U = 8;  // loads in flight
  if (INV) {
    for (int q = q0; q < nq; q += U * qs) {
      C v[U];
#pragma unroll
      for (int j = 0; j < U; ++j)
        if (q + j * qs < nq) v[j] = ldg_c(src + at_std(q + j * qs));
#pragma unroll
      for (int j = 0; j < U; ++j)
        if (q + j * qs < nq) tile[at_tile(q + j * qs)] = cscale(v[j], scale);
    }
    __syncthreads();
  }
  switch (g.nz) {
    case 64: std_rows<C, 16, 4, INV>(kbn * g.Y1, tile, rs, twz); break;
    case 128: std_rows<C, 16, 8, INV>(kbn * g.Y1, tile, rs, twz); break;
    default: std_rows<C, 16, 16, INV>(kbn * g.Y1, tile, rs, twz); break;
  }
  __syncthreads();
  if (INV) {
    passB_cols_any<T, true>(g, kbn, nullptr, cb, tile, rs, dst);
  } else {
    for (int q = q0; q < nq; q += qs) dst[at_std(q)] = tile[at_tile(q)];
  }
}

}  // namespace etd
