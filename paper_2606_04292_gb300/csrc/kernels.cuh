// Grid kernels of one V-cycle level and the coarse tail (one cluster of blocks).
// Included by the FP64 and FP32 translation units, which instantiate them.
#pragma once

#include <algorithm>

#include <cooperative_groups.h>

#include "device.cuh"
#include "launch.h"

namespace rich {

template <typename T>
__device__ __forceinline__ T from_bits(unsigned long long b);
template <>
__device__ __forceinline__ double from_bits<double>(unsigned long long b) {
  return __longlong_as_double((long long)b);
}
template <>
__device__ __forceinline__ float from_bits<float>(unsigned long long b) {
  return __uint_as_float((unsigned)b);
}

// ---------------------------------------------------------------------------
// One colour of a red-black NGS sweep (eq. point-update for every cell of the
// colour; cells of one colour do not couple, so the update is parallel).
// ---------------------------------------------------------------------------
// Launch grid: x = pairs of cells along a row, y = row, z = plane.
// (The bodies of the grid kernels take the block's coordinates explicitly:
// the batched kernels run the same bodies for the blocks of many grids.)
template <typename T, int FORM, int MODEL, int NK = 0>
__device__ __forceinline__ void sweep_body(const Level<T>& L, const Phys<T>& P, int color, int bx, int by, int bz) {
  const int p = bx * blockDim.x + threadIdx.x;
  const int i1 = by, i2 = bz;
  const int i0 = 2 * p + ((color + i1 + i2) & 1);
  if (i0 >= L.n0) return;
  const long long i = (unsigned)(i0 + L.n0 * (i1 + L.n1 * i2));
  point_update<T, FORM, MODEL, NK>(L, P, i, i0, i1, i2);
}

template <typename T, int FORM, int MODEL, int NK = 0>
__global__ void __launch_bounds__(256) k_sweep(Level<T> L, Phys<T> P, int color) {
  sweep_body<T, FORM, MODEL, NK>(L, P, color, blockIdx.x, blockIdx.y, blockIdx.z);
}

// The same half-sweep with ZC planes per thread, software-pipelined: the
// operands of the next plane's cell are loaded before the current cell is
// solved.  Launch grid: x = pairs of cells along a row, y = row, z = chunk
// of ZC planes.
// RESID: the half-sweep also writes the defect d = g - N(u) of each cell it
// updates, at the new value (its neighbours, of the other colour, do not
// change during the half-sweep), and returns the largest |d| (bits)
template <typename T, int FORM, int MODEL, int ZC, int NK, bool YZI, bool RESID>
__device__ __forceinline__ unsigned long long sweep_pipe_body(const Level<T>& L, const Phys<T>& P, int color, int p,
                                                              int i1, int z0) {
  unsigned long long mx = 0;
  CellOps<T> c[2];
  {
    const int i0 = 2 * p + ((color + i1 + z0) & 1);
    c[0].valid = z0 < L.n2 && i0 < L.n0;
    if (c[0].valid) gather<T, FORM, MODEL, YZI>(L, P, i0, i1, z0, c[0]);
  }
#pragma unroll
  for (int k = 0; k < ZC; ++k) {
    if (k + 1 < ZC) {
      const int i2 = z0 + k + 1;
      const int i0 = 2 * p + ((color + i1 + i2) & 1);
      CellOps<T>& nx = c[(k + 1) & 1];
      nx.valid = i2 < L.n2 && i0 < L.n0;
      if (nx.valid) gather<T, FORM, MODEL, YZI>(L, P, i0, i1, i2, nx);
    }
    const CellOps<T>& cur = c[k & 1];
    if (cur.valid) {
      T dg, of;
      cell_sums<T, YZI>(L, cur, dg, of);
      const T x = solve_cell_sums<T, FORM, MODEL, NK, YZI>(L, P, cur, dg, of);
      L.u[cur.i] = x;
      if (RESID) {
        const T di = cell_defect<T, FORM, MODEL>(L, P, cur, dg, of, x);
        L.d[cur.i] = di;
        const unsigned long long b = nbits(di);
        mx = b > mx ? b : mx;
      }
    }
  }
  return mx;
}

template <typename T, int FORM, int MODEL, int ZC, int NK = 0, bool RESID = false>
__global__ void __launch_bounds__(128) k_sweep_pipe(Level<T> L, Phys<T> P, int color, unsigned long long* norm) {
  const int p = blockIdx.x * blockDim.x + threadIdx.x;
  const int i1 = blockIdx.y;
  const int z0 = blockIdx.z * ZC;
  // blocks away from the y and z boundaries (all but a thin shell) skip
  // those boundary tests; the branch is uniform over the block
  // (the deeper pipelines, 4 and 8 planes, keep one body: compile time)
  unsigned long long mx;
  if constexpr (ZC == 2) {
    const bool yzi = L.dim == 3 && i1 > 0 && i1 < L.n1 - 1 && z0 > 0 && z0 + ZC < L.n2;
    mx = yzi ? sweep_pipe_body<T, FORM, MODEL, ZC, NK, true, RESID>(L, P, color, p, i1, z0)
             : sweep_pipe_body<T, FORM, MODEL, ZC, NK, false, RESID>(L, P, color, p, i1, z0);
  } else {
    mx = sweep_pipe_body<T, FORM, MODEL, ZC, NK, false, RESID>(L, P, color, p, i1, z0);
  }
  if (RESID) {
    __shared__ unsigned long long sm[33];
    mx = block_max(mx, sm);
    if (threadIdx.x == 0) atomicMax(norm, mx);
  }
}

// The defect of the cells of one colour (the other colour's defects come
// from a RESID half-sweep).  Launch grid: as k_sweep.
template <typename T, int FORM, int MODEL>
__global__ void __launch_bounds__(256) k_residual_color(Level<T> L, Phys<T> P, int color, unsigned long long* norm) {
  __shared__ unsigned long long sm[33];
  unsigned long long mx = 0;
  const int p = blockIdx.x * blockDim.x + threadIdx.x;
  const int i1 = blockIdx.y, i2 = blockIdx.z;
  const int i0 = 2 * p + ((color + i1 + i2) & 1);
  if (i0 < L.n0) {
    const long long i = (unsigned)(i0 + L.n0 * (i1 + L.n1 * i2));
    const bool yzi = L.dim == 3 && i1 > 0 && i1 < L.n1 - 1 && i2 > 0 && i2 < L.n2 - 1;
    const T di = L.g[pix(L, i, i0, i1, i2)] - (yzi ? apply_N<T, FORM, MODEL, true>(L, P, L.u, i, i0, i1, i2)
                                                    : apply_N<T, FORM, MODEL, false>(L, P, L.u, i, i0, i1, i2));
    L.d[i] = di;
    mx = nbits(di);
  }
  mx = block_max(mx, sm);
  if (threadIdx.x == 0) atomicMax(norm, mx);
}

// One hyperplane i0 + i1 + i2 = s of a lexicographic NGS sweep (the
// paper's ordering, Section 3.1: cells in the order of the flattened index).
// Cells of one hyperplane do not couple; each reads the updated values of its
// lower neighbours (plane s - 1) and the old values of its upper ones (plane
// s + 1), exactly what the sequential sweep reads.  Planes s = 0 .. n0+n1+n2-3
// in turn make one sweep.  Launch grid: x = i1, y = i2 - i2lo.
template <typename T, int FORM, int MODEL, int NK = 0>
__global__ void __launch_bounds__(128) k_sweep_plane(Level<T> L, Phys<T> P, int s, int i2lo) {
  const int i1 = blockIdx.x * blockDim.x + threadIdx.x;
  const int i2 = i2lo + blockIdx.y;
  if (i1 >= L.n1) return;
  const int i0 = s - i1 - i2;
  if (i0 < 0 || i0 >= L.n0) return;
  const long long i = (unsigned)(i0 + L.n0 * (i1 + L.n1 * i2));
  point_update<T, FORM, MODEL, NK>(L, P, i, i0, i1, i2);
}

// d = g - N(u) on a level, with ||d||_inf accumulated into *norm (bit max).
// Launch grid: x = cells along a row, y = row, z = plane.
// (returns |d| of the thread's cell as bits, 0 without one)
template <typename T, int FORM, int MODEL>
__device__ __forceinline__ unsigned long long residual_body(const Level<T>& L, const Phys<T>& P, int bx, int by,
                                                            int bz) {
  const int i0 = bx * blockDim.x + threadIdx.x;
  const int i1 = by, i2 = bz;
  if (i0 >= L.n0) return 0;
  const long long i = (unsigned)(i0 + L.n0 * (i1 + L.n1 * i2));
  // rows away from the y/z boundaries skip those tests (uniform over the block)
  const bool yzi = L.dim == 3 && i1 > 0 && i1 < L.n1 - 1 && i2 > 0 && i2 < L.n2 - 1;
  const T di = L.g[pix(L, i, i0, i1, i2)] - (yzi ? apply_N<T, FORM, MODEL, true>(L, P, L.u, i, i0, i1, i2)
                                                  : apply_N<T, FORM, MODEL, false>(L, P, L.u, i, i0, i1, i2));
  L.d[i] = di;
  return nbits(di);
}

template <typename T, int FORM, int MODEL>
__global__ void __launch_bounds__(256) k_residual(Level<T> L, Phys<T> P, unsigned long long* norm) {
  __shared__ unsigned long long sm[33];
  unsigned long long mx = residual_body<T, FORM, MODEL>(L, P, blockIdx.x, blockIdx.y, blockIdx.z);
  if (norm) {
    mx = block_max(mx, sm);
    if (threadIdx.x == 0) atomicMax(norm, mx);
  }
}

// FAS step 3: psi_bar_H = R psi_h, d_H = R d_h (cb may be null).
// (cs_mask: bit 0 / bit 1 set when fa / fb is a colour-split parameter array)
template <typename T>
__device__ __forceinline__ void restrict_body(const Level<T>& F, const Level<T>& C, const Xfer<T>& X, const T* fa,
                                              const T* fb, T* ca, T* cb, int bx, int by, int bz, int cs_mask = 0) {
  const int J0 = bx * blockDim.x + threadIdx.x;
  const int J1 = by, J2 = bz;
  if (J0 >= C.n0) return;
  const long long J = J0 + (long long)C.n0 * (J1 + C.n1 * J2);
  ca[J] = restrict_at(F, X, fa, J0, J1, J2, (cs_mask & 1) != 0);
  if (cb) cb[J] = restrict_at(F, X, fb, J0, J1, J2, (cs_mask & 2) != 0);
}

template <typename T>
__global__ void __launch_bounds__(256) k_restrict(Level<T> F, Level<T> C, Xfer<T> X, const T* fa, const T* fb,
                                                  T* ca, T* cb, int cs_mask) {
  restrict_body<T>(F, C, X, fa, fb, ca, cb, blockIdx.x, blockIdx.y, blockIdx.z, cs_mask);
}

// FAS step 4 on the coarse level: g_H = N_H(psi_bar_H) + d_H, psi_H = psi_bar_H.
template <typename T, int FORM, int MODEL>
__device__ __forceinline__ void tau_body(const Level<T>& C, const Phys<T>& P, int bx, int by, int bz) {
  const int J0 = bx * blockDim.x + threadIdx.x;
  const int J1 = by, J2 = bz;
  if (J0 >= C.n0) return;
  const long long J = J0 + (long long)C.n0 * (J1 + C.n1 * J2);
  // rows away from the y/z boundaries skip those tests (uniform over the block)
  const bool yzi = C.dim == 3 && J1 > 0 && J1 < C.n1 - 1 && J2 > 0 && J2 < C.n2 - 1;
  C.g[J] = (yzi ? apply_N<T, FORM, MODEL, true>(C, P, C.ubar, J, J0, J1, J2)
                : apply_N<T, FORM, MODEL, false>(C, P, C.ubar, J, J0, J1, J2)) + C.d[J];
  C.u[J] = C.ubar[J];
}

template <typename T, int FORM, int MODEL>
__global__ void __launch_bounds__(256) k_tau(Level<T> C, Phys<T> P) {
  tau_body<T, FORM, MODEL>(C, P, blockIdx.x, blockIdx.y, blockIdx.z);
}

// FAS step 6: u_h += P (u_H - psi_bar_H).
template <typename T>
__device__ __forceinline__ void prolong_body(const Level<T>& F, const Level<T>& C, const Xfer<T>& X, int bx, int by,
                                             int bz) {
  const int i0 = bx * blockDim.x + threadIdx.x;
  const int i1 = by, i2 = bz;
  if (i0 >= F.n0) return;
  const long long i = i0 + (long long)F.n0 * (i1 + F.n1 * i2);
  F.u[i] += prolong_at(C, X, i0, i1, i2);
}

template <typename T>
__global__ void __launch_bounds__(256) k_prolong(Level<T> F, Level<T> C, Xfer<T> X) {
  prolong_body<T>(F, C, X, blockIdx.x, blockIdx.y, blockIdx.z);
}

// ---------------------------------------------------------------------------
// Nested levels (n_fine = 2 n_coarse on every axis the grid has): the same
// transfer operators with their weights written out, so a thread reads no
// tables.  Restriction taps per axis at fine 2J-1 .. 2J+2 with weights
// (1,3,3,1)/8, at the ends (0,4,3,1)/8 and (1,3,4,0)/8 (the normalised
// transpose of the constant-extrapolation interpolation); an axis of one
// cell is a single tap of weight 1.  Interpolation of an interior fine cell
// i: 3/4 of coarse floor(i/2) and 1/4 of the coarse neighbour on i's side;
// fine end cells take their weights from the tables (they fold the ghost).
// ---------------------------------------------------------------------------
template <typename T>
__device__ __forceinline__ void restrict_taps(int J, int nc, int nf, int* idx, T* w) {
  if (nf == 1) {
#pragma unroll
    for (int t = 0; t < 4; ++t) { idx[t] = 0; w[t] = T(0); }
    w[1] = T(1);
    return;
  }
  w[0] = T(0.125); w[1] = T(0.375); w[2] = T(0.375); w[3] = T(0.125);
  if (J == 0) { w[0] = T(0); w[1] = T(0.5); }
  if (J == nc - 1) { w[2] = T(0.5); w[3] = T(0); }
#pragma unroll
  for (int t = 0; t < 4; ++t) {
    const int f = 2 * J - 1 + t;
    idx[t] = f < 0 ? 0 : (f >= nf ? nf - 1 : f);
  }
}

template <typename T>
__device__ __forceinline__ void restrict_nested_body(const Level<T>& F, const Level<T>& C, const T* fa, const T* fb,
                                                     T* ca, T* cb, int bx, int by, int bz, int cs_mask = 0) {
  const int J0 = bx * blockDim.x + threadIdx.x;
  const int J1 = by, J2 = bz;
  if (J0 >= C.n0) return;
  int x[4], y[4], z[4];
  T wx[4], wy[4], wz[4];
  restrict_taps<T>(J0, C.n0, F.n0, x, wx);
  restrict_taps<T>(J1, C.n1, F.n1, y, wy);
  restrict_taps<T>(J2, C.n2, F.n2, z, wz);
  T sa = T(0), sb = T(0);
#pragma unroll
  for (int c = 0; c < 4; ++c) {
    if (wz[c] == T(0)) continue;
    T ya = T(0), yb = T(0);
#pragma unroll
    for (int b = 0; b < 4; ++b) {
      if (wy[b] == T(0)) continue;
      const unsigned row = (unsigned)F.n0 * ((unsigned)y[b] + (unsigned)F.n1 * (unsigned)z[c]);
      unsigned ia[4], ib[4];
#pragma unroll
      for (int a = 0; a < 4; ++a) {
        ia[a] = row + x[a];
        ib[a] = row + x[a];
        if (cs_mask) {
          const unsigned q = pix_of(1, F.n0, F.n1, F.n2, row + x[a], x[a], y[b], z[c]);
          if (cs_mask & 1) ia[a] = q;
          if (cs_mask & 2) ib[a] = q;
        }
      }
      T xa = T(0);
#pragma unroll
      for (int a = 0; a < 4; ++a) xa += wx[a] * fa[ia[a]];
      ya += wy[b] * xa;
      if (fb) {
        T xb = T(0);
#pragma unroll
        for (int a = 0; a < 4; ++a) xb += wx[a] * fb[ib[a]];
        yb += wy[b] * xb;
      }
    }
    sa += wz[c] * ya;
    sb += wz[c] * yb;
  }
  const unsigned J = (unsigned)(J0 + C.n0 * (J1 + C.n1 * J2));
  ca[J] = sa;
  if (cb) cb[J] = sb;
}

template <typename T>
__global__ void __launch_bounds__(256) k_restrict_nested(Level<T> F, Level<T> C, const T* fa, const T* fb, T* ca,
                                                         T* cb, int cs_mask) {
  restrict_nested_body<T>(F, C, fa, fb, ca, cb, blockIdx.x, blockIdx.y, blockIdx.z, cs_mask);
}

template <typename T>
__device__ __forceinline__ void prolong_taps(const Xfer<T>& X, int a, int i, int nf, int* j, T* w) {
  if (i > 0 && i < nf - 1) {
    const int J = i >> 1;
    j[0] = J;
    w[0] = T(0.75);
    j[1] = (i & 1) ? J + 1 : J - 1;
    w[1] = T(0.25);
    return;
  }
  const int c = X.pc[a][i];
  j[0] = X.pj[a][2 * i];
  w[0] = X.pw[a][2 * i];
  j[1] = c > 1 ? X.pj[a][2 * i + 1] : j[0];
  w[1] = c > 1 ? X.pw[a][2 * i + 1] : T(0);
}

// the interpolated coarse correction of fine cell (i0, i1, i2), nested levels
template <typename T>
__device__ __forceinline__ T prolong_nested_at(const Level<T>& F, const Level<T>& C, const Xfer<T>& X, int i0, int i1,
                                               int i2) {
  int jx[2], jy[2], jz[2];
  T wx[2], wy[2], wz[2];
  prolong_taps<T>(X, 0, i0, F.n0, jx, wx);
  prolong_taps<T>(X, 1, i1, F.n1, jy, wy);
  prolong_taps<T>(X, 2, i2, F.n2, jz, wz);
  T s = T(0);
#pragma unroll
  for (int c = 0; c < 2; ++c) {
    if (wz[c] == T(0)) continue;
    T sy = T(0);
#pragma unroll
    for (int b = 0; b < 2; ++b) {
      if (wy[b] == T(0)) continue;
      const unsigned row = (unsigned)C.n0 * ((unsigned)jy[b] + (unsigned)C.n1 * (unsigned)jz[c]);
      T sx = T(0);
#pragma unroll
      for (int a = 0; a < 2; ++a) sx += wx[a] * (C.u[row + jx[a]] - C.ubar[row + jx[a]]);
      sy += wy[b] * sx;
    }
    s += wz[c] * sy;
  }
  return s;
}

template <typename T>
__device__ __forceinline__ void prolong_nested_body(const Level<T>& F, const Level<T>& C, const Xfer<T>& X, int bx,
                                                    int by, int bz) {
  const int i0 = bx * blockDim.x + threadIdx.x;
  const int i1 = by, i2 = bz;
  if (i0 >= F.n0) return;
  const unsigned i = (unsigned)(i0 + F.n0 * (i1 + F.n1 * i2));
  F.u[i] += prolong_nested_at(F, C, X, i0, i1, i2);
}

// one coarse value of the nested full-weighting restriction of a natural
// layout array (the arithmetic of restrict_nested_body, one array)
template <typename T>
__device__ __forceinline__ T restrict_nested_at(const Level<T>& F, const Level<T>& C, const T* fa, int J0, int J1,
                                                int J2) {
  int x[4], y[4], z[4];
  T wx[4], wy[4], wz[4];
  restrict_taps<T>(J0, C.n0, F.n0, x, wx);
  restrict_taps<T>(J1, C.n1, F.n1, y, wy);
  restrict_taps<T>(J2, C.n2, F.n2, z, wz);
  T sa = T(0);
#pragma unroll
  for (int c = 0; c < 4; ++c) {
    if (wz[c] == T(0)) continue;
    T ya = T(0);
#pragma unroll
    for (int b = 0; b < 4; ++b) {
      if (wy[b] == T(0)) continue;
      const unsigned row = (unsigned)F.n0 * ((unsigned)y[b] + (unsigned)F.n1 * (unsigned)z[c]);
      T xa = T(0);
#pragma unroll
      for (int a = 0; a < 4; ++a) xa += wx[a] * fa[row + x[a]];
      ya += wy[b] * xa;
    }
    sa += wz[c] * ya;
  }
  return sa;
}

template <typename T>
__global__ void __launch_bounds__(256) k_prolong_nested(Level<T> F, Level<T> C, Xfer<T> X) {
  prolong_nested_body<T>(F, C, X, blockIdx.x, blockIdx.y, blockIdx.z);
}

// ---------------------------------------------------------------------------
// The interpolation of big 3-d levels through a shared-memory tile: a block
// first stages, in coalesced rows, the coarse corrections u_H - psi_bar_H its
// fine tile reads, with a one-cell halo (out-of-range halo cells repeat the
// edge and are never weighted), then evaluates the taps of
// k_prolong_nested, in the same order, from shared memory: same results,
// fewer L1 requests (16 global loads per fine cell become 8 shared ones).
// (The same staging for the restriction measured slower than its L1-cached
// kernel: 64 taps per coarse cell reuse the cache well.)
// ---------------------------------------------------------------------------
template <typename T>
struct TransferTile {
  static constexpr int PX = 64, PY = 4, PZ = 4;                         // fine tile of the interpolation
};

__device__ __forceinline__ int clampi(int v, int lo, int hi) { return v < lo ? lo : (v > hi ? hi : v); }

template <typename T>
__global__ void __launch_bounds__(TransferTile<T>::PX * TransferTile<T>::PY)
k_prolong_tiled(Level<T> F, Level<T> C, Xfer<T> X) {
  constexpr int PX = TransferTile<T>::PX, PY = TransferTile<T>::PY, PZ = TransferTile<T>::PZ;
  constexpr int CX = PX / 2 + 2, CY = PY / 2 + 2, CZ = PZ / 2 + 2, NT = PX * PY;
  __shared__ T se[CZ][CY][CX];
  const int x0 = blockIdx.x * PX, y0 = blockIdx.y * PY, z0 = blockIdx.z * PZ;
  const int cx0 = x0 / 2 - 1, cy0 = y0 / 2 - 1, cz0 = z0 / 2 - 1;
  for (int t = threadIdx.x; t < CX * CY * CZ; t += NT) {
    const int x = t % CX, y = (t / CX) % CY, z = t / (CX * CY);
    const int gx = clampi(cx0 + x, 0, C.n0 - 1), gy = clampi(cy0 + y, 0, C.n1 - 1), gz = clampi(cz0 + z, 0, C.n2 - 1);
    const unsigned gj = (unsigned)gx + (unsigned)C.n0 * ((unsigned)gy + (unsigned)C.n1 * (unsigned)gz);
    se[z][y][x] = C.u[gj] - C.ubar[gj];
  }
  __syncthreads();
  const int i0 = x0 + threadIdx.x % PX, i1 = y0 + threadIdx.x / PX;
  if (i0 >= F.n0 || i1 >= F.n1) return;
  int jx[2], jy[2];
  T wx[2], wy[2];
  prolong_taps<T>(X, 0, i0, F.n0, jx, wx);
  prolong_taps<T>(X, 1, i1, F.n1, jy, wy);
  // the x-y interpolation of each staged coarse plane, once for the PZ fine
  // cells of the column that share it (the sums of prolong_nested_at)
  T py[CZ];
#pragma unroll
  for (int p = 0; p < CZ; ++p) {
    T sy = T(0);
#pragma unroll
    for (int b = 0; b < 2; ++b) {
      if (wy[b] == T(0)) continue;
      const T* row = &se[p][jy[b] - cy0][0];
      T sx = T(0);
#pragma unroll
      for (int a = 0; a < 2; ++a) sx += wx[a] * row[jx[a] - cx0];
      sy += wy[b] * sx;
    }
    py[p] = sy;
  }
  for (int k = 0; k < PZ; ++k) {
    const int i2 = z0 + k;
    if (i2 >= F.n2) break;
    int jz[2];
    T wz[2];
    prolong_taps<T>(X, 2, i2, F.n2, jz, wz);
    T s = T(0);
#pragma unroll
    for (int c = 0; c < 2; ++c) {
      if (wz[c] == T(0)) continue;
      s += wz[c] * py[jz[c] - cz0];
    }
    const unsigned i = (unsigned)(i0 + F.n0 * (i1 + F.n1 * i2));
    F.u[i] += s;
  }
}

// the tiles pay off on big 3-d levels
inline bool tiled_transfer(int dim, int fn0, int fn1, int fn2) {
  return dim == 3 && fn2 >= 4 && fn1 >= 4 && (long long)fn0 * fn1 * fn2 >= (1LL << 15);
}

__host__ __device__ inline bool nested_levels(int fn0, int fn1, int fn2, int cn0, int cn1, int cn2) {
  const int f[3] = {fn0, fn1, fn2}, c[3] = {cn0, cn1, cn2};
  for (int a = 0; a < 3; ++a)
    if (!(f[a] == 2 * c[a] || (f[a] == 1 && c[a] == 1))) return false;
  return true;
}

// ---------------------------------------------------------------------------
// The coarse tail: the whole cycle from level l0 down in one launch (levels
// small enough that launch latency would dominate a kernel per stage).  Same
// arithmetic as the grid kernels, phase by phase, separated by barriers.
//
// The cycle's loops run over a "team" of threads: one thread block (the
// batched columns), the blocks of one thread-block cluster (the coarse tail,
// the small-grid step), or every block of a cooperative grid.  rank/size index
// the team's threads, sync() is its barrier, max() its max-reduction (every
// thread gets the result).  A team of several blocks can hand the smallest
// levels to its first block alone (solo: block barriers), while the others
// wait at the team's next barrier.
//
// Why a cluster: a phase of a 64^2 level is 2048 point updates, which one SM
// issues in ~5.5 us (FP32) or, bound by its FP64 pipe, ~40 us (FP64); spread
// over 16 SMs it takes the latency of one update, and the hardware barrier of
// a cluster costs a fraction of a launch or of a grid-wide barrier.
// ---------------------------------------------------------------------------
constexpr int SEEN_CELLS = 64;         // the most coarsest cells that revisited() follows
constexpr int TEAM_WORDS = 33 + SEEN_CELLS;
struct BlockTeam {
  static constexpr bool splits = false;
  unsigned long long* sm;              // TEAM_WORDS words: block_max's, revisited()'s
  __device__ unsigned long long* words() const { return sm; }
  __device__ unsigned rank() const { return threadIdx.x; }
  __device__ unsigned size() const { return blockDim.x; }
  __device__ void sync() const { __syncthreads(); }
  __device__ unsigned long long max(unsigned long long v) const { return block_max(v, sm); }
};

// Shared memory of a cluster team: block_max's words and two rotating rows of
// one maximum per block.
struct ClusterShared {
  unsigned long long sm[TEAM_WORDS];
  unsigned long long part[2][CLUSTER_MAX];
};

// The blocks of one cluster (1 to CLUSTER_MAX).  Warps are dealt round robin
// over the blocks, so that a level with few cells uses every SM of the
// cluster.  (barrier.cluster releases and acquires at cluster scope: global
// memory written before it by any block is visible after it to all.)
struct ClusterTeam {
  static constexpr bool splits = true;
  ClusterShared* sh;
  unsigned nct, ct;
  bool solo;
  int parity;
  __device__ explicit ClusterTeam(ClusterShared* s) : sh(s), parity(0) {
    asm("mov.u32 %0, %%cluster_nctarank;" : "=r"(nct));
    asm("mov.u32 %0, %%cluster_ctarank;" : "=r"(ct));
    solo = nct == 1;
  }
  __device__ unsigned long long* words() const { return sh->sm; }
  __device__ bool lead() const { return ct == 0; }
  __device__ unsigned rank() const {
    return solo ? threadIdx.x : (((threadIdx.x >> 5) * nct + ct) << 5) + (threadIdx.x & 31);
  }
  __device__ unsigned size() const { return solo ? blockDim.x : blockDim.x * nct; }
  __device__ void cluster_sync() const {
    asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
    asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
  }
  __device__ void sync() const {
    if (solo) __syncthreads();
    else cluster_sync();
  }
  // (every block writes its maximum into every block's row; the row is next
  // written two reductions, and so at least one cluster barrier, later)
  __device__ unsigned long long max(unsigned long long v) {
    v = block_max(v, sh->sm);
    if (solo) return v;
    if (threadIdx.x < nct) {
      const unsigned a = (unsigned)__cvta_generic_to_shared(&sh->part[parity][ct]);
      unsigned r;
      asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(threadIdx.x));
      asm volatile("st.shared::cluster.u64 [%0], %1;" ::"r"(r), "l"(v) : "memory");
    }
    cluster_sync();
    unsigned long long m = 0;
    for (unsigned k = 0; k < nct; ++k) {
      const unsigned long long w = sh->part[parity][k];
      m = w > m ? w : m;
    }
    parity ^= 1;
    return m;
  }
};

// (three global slots rotate: the slot zeroed at one reduction was last read
// two reductions earlier, with a grid barrier in between)
struct GridTeam {
  static constexpr bool splits = true;
  unsigned long long* slots;
  unsigned long long* sm;
  int round;
  bool solo;
  __device__ unsigned long long* words() const { return sm; }
  __device__ bool lead() const { return blockIdx.x == 0; }
  __device__ unsigned rank() const { return solo ? threadIdx.x : blockIdx.x * blockDim.x + threadIdx.x; }
  __device__ unsigned size() const { return solo ? blockDim.x : gridDim.x * blockDim.x; }
  __device__ void sync() const {
    if (solo) __syncthreads();
    else cooperative_groups::this_grid().sync();
  }
  __device__ unsigned long long max(unsigned long long v) {
    v = block_max(v, sm);
    if (solo) return v;
    unsigned long long* s = slots + round % 3;
    if (threadIdx.x == 0) atomicMax(s, v);
    if (rank() == 0) slots[(round + 1) % 3] = 0ull;
    sync();
    const unsigned long long r = *(volatile unsigned long long*)s;
    ++round;
    return r;
  }
};

// one NGS sweep of a level by a team: red then black half-sweeps (ordering
// 1), or the lexicographic order hyperplane by hyperplane (0).  One copy of
// the point update serves both; the update without a sink is its own (the
// sink's pieces, if-converted, cost the 128-cell column 5%), but in the
// columns, whose second copy would spill (48.1 -> 50.2 ms).
template <typename T, int FORM, int MODEL, typename TM>
__device__ __forceinline__ void team_sweep(const Level<T>& L, const Phys<T>& P, int ordering, TM& tm) {
  const unsigned rows = (unsigned)L.n1 * (unsigned)L.n2;
  const unsigned items = ordering ? (unsigned)((L.n0 + 1) >> 1) * rows : rows;
  const int phases = ordering ? 2 : L.n0 + L.n1 + L.n2 - 2;
  for (int ph = 0; ph < phases; ++ph) {
    for (unsigned t = tm.rank(); t < items; t += tm.size()) {
      int i0, i1, i2;
      unsigned i;
      bool on;
      if (ordering) {
        on = color_cell(L, t, ph, i0, i1, i2, i);
      } else {
        i2 = (int)quick_div(t, (unsigned)L.n1, L.rn1);
        i1 = (int)t - i2 * L.n1;
        i0 = ph - i1 - i2;
        on = i0 >= 0 && i0 < L.n0;
        i = (unsigned)i0 + (unsigned)L.n0 * t;
      }
      if (on) {
        if constexpr (TM::splits) {
          if (P.sink && L.smax) point_update<T, FORM, MODEL, 0, 1>(L, P, i, i0, i1, i2);
          else point_update<T, FORM, MODEL, 0, 0>(L, P, i, i0, i1, i2);
        } else {
          point_update<T, FORM, MODEL>(L, P, i, i0, i1, i2);
        }
      }
    }
    tm.sync();
  }
}

// the defect d = g - N(u) of a level by a team: stored (store), or its
// max-norm (returned to every thread)
template <typename T, int FORM, int MODEL, typename TM>
__device__ __forceinline__ T team_defect(const Level<T>& L, const Phys<T>& P, bool store, TM& tm) {
  unsigned long long mx = 0;
  for (unsigned i = tm.rank(); i < (unsigned)L.ncell; i += tm.size()) {
    int i0, i1, i2;
    cell_coords(L, i, i0, i1, i2);
    const T di = L.g[pix(L, i, i0, i1, i2)] - apply_N<T, FORM, MODEL>(L, P, L.u, i, i0, i1, i2);
    if (store) L.d[i] = di;
    const unsigned long long b = nbits(di);
    mx = b > mx ? b : mx;
  }
  if (store) {
    tm.sync();
    return T(0);
  }
  return from_bits<T>(tm.max(mx));
}

// Whether the coarsest level's iterate is, bit for bit, the kept one (in shared
// memory; first: there is none yet; keep: this one becomes it).  A sweep is a
// function of the iterate, so from then on the sweeps repeat the states since
// the kept one: the stop test has failed at all of them, and after a whole
// number of such periods the iterate is this one.  Kept are the states after 2,
// 4, 8, ... sweeps (Brent's cycle detection, BIT 20, 1980: any period is found
// within twice the sweeps it took to begin).  A defect at round-off need not
// fall to crtol d0, and such a solve otherwise runs all its cmax sweeps.
// GB300, all sweeps / ended at a period of one or two (looked at every second
// sweep) / at any: two steps of the Celia column 3.44 / 2.44 / 2.42 ms, two-layer
// 256^2 13.3 / 11.1 / 10.4, 4096 columns x 4 steps 38.0 / 34.9 / 32.9, Gardner
// 128^2 3.41 / 3.27 / 3.18, 8 served requests 9.94 / 9.82 / 9.55; keeping every
// sixth or twelfth state 33.0 and 33.1 for the columns, 10.6 and 10.75 for the
// two layers.  (Teams of several blocks that share the level, and levels of
// more than SEEN_CELLS cells, do not look.)
template <typename T, typename TM>
__device__ __forceinline__ bool revisited(const Level<T>& L, bool first, bool keep, TM& tm) {
  if constexpr (TM::splits) {
    if (!tm.solo) return false;
  }
  if (L.ncell > SEEN_CELLS) return false;
  bool differs = first;
  for (unsigned i = threadIdx.x; i < (unsigned)L.ncell; i += blockDim.x) {
    const T v = L.u[i];
    unsigned long long b;
    if constexpr (sizeof(T) == 8) b = (unsigned long long)__double_as_longlong(v);
    else b = __float_as_uint(v);
    unsigned long long& kept = tm.words()[33 + i];
    if (b != kept) differs = true;
    if (keep) kept = b;
  }
  return !__syncthreads_or(differs);
}

// Levels l0..nl-1 of one multigrid cycle by one team, with the recursion of
// Section 3.2 unrolled: pre-smoothing, defect, restriction and the FAS right
// side on the way down; gamma visits of each coarser level (1: V-cycle, 2:
// W-cycle); the coarsest level sweeps until its defect drops by crtol or
// cmax sweeps are done; prolongation and post-smoothing on the way up.  LV
// gives the level views (L(l)) and the transfers from level l:
// restrict2(l, fine arrays, coarse coords) and prolong(l, fine coords).
// handoff (teams of several blocks): levels from handoff on run solo.
// One loop, with one copy of the sweep, the defect and the FAS right side:
// the busy warps of a small level fetch each instruction for themselves, and
// a copy per use was a fifth of their stall cycles.
template <typename T, int FORM, int MODEL, typename LV, typename TM>
__device__ __forceinline__ void team_cycle(const LV& lv, int l0, int nl, const Phys<T>& P, int nu1, int nu2, int cmax,
                                           T crtol, int gamma, int gamma_levels, unsigned long long& updates,
                                           int ordering, int handoff, TM& tm) {
  enum { DOWN, COARSEST, POST };
  unsigned long long visits = 0;         // coarse visits done from each level, two bits a level (gamma <= 3)
  int l = l0, solo_at = -1;
  bool arrive = true;                    // at level l from above
  int stage = DOWN, sweeps = 0, done = 0, limit = 0;
  T d0 = T(0);
  for (;;) {
    bool finished = false;
    if (arrive) {
      arrive = false;
      if constexpr (TM::splits) {
        if (!tm.solo && l >= handoff) {
          if (tm.lead()) {
            tm.solo = true;
            solo_at = l;
          } else {
            tm.sync();                   // (the first block's, when it has finished level l)
            finished = true;
          }
        }
      }
      stage = l == nl - 1 ? COARSEST : DOWN;
      sweeps = stage == COARSEST ? (cmax > 1 ? 0 : 1) : nu1;
      done = 0;
      limit = cmax;
    }
    if (!finished) {
      const Level<T>& F = lv.L(l);
      for (int s = 0; s < sweeps; ++s) team_sweep<T, FORM, MODEL, TM>(F, P, ordering, tm);
      updates += (unsigned long long)sweeps * F.ncell;
      finished = true;
      if (stage == COARSEST) {
        done += sweeps;
        if (done < limit) {              // (the last sweep's defect would change nothing)
          if (done > 1 && revisited<T>(F, done == 2, (done & (done - 1)) == 0, tm)) {
            const int p = done - (1 << (31 - __clz(done - 1)));   // sweeps since the kept state
            limit = done + (limit - done) % p;
            finished = done == limit;
          } else {
            const T dn = team_defect<T, FORM, MODEL, TM>(F, P, false, tm);
            if (done == 0) d0 = dn;
            finished = done > 0 && !(dn > crtol * d0);
          }
          sweeps = 1;
        }
        if (!finished) continue;
      } else if (stage == DOWN) {
        team_defect<T, FORM, MODEL, TM>(F, P, true, tm);
        const Level<T>& C = lv.L(l + 1);
        for (unsigned J = tm.rank(); J < (unsigned)C.ncell; J += tm.size()) {
          int J0, J1, J2;
          cell_coords(C, J, J0, J1, J2);
          lv.restrict2(l, F.u, F.d, J0, J1, J2, C.ubar[J], C.d[J]);
        }
        tm.sync();
        for (unsigned J = tm.rank(); J < (unsigned)C.ncell; J += tm.size()) {
          int J0, J1, J2;
          cell_coords(C, J, J0, J1, J2);
          C.g[J] = apply_N<T, FORM, MODEL>(C, P, C.ubar, J, J0, J1, J2) + C.d[J];
          C.u[J] = C.ubar[J];
        }
        tm.sync();
        visits &= ~(3ull << (2 * l));
        ++l;
        arrive = true;
        continue;
      }
    }
    // level l is finished: back to its parent
    if constexpr (TM::splits) {
      if (solo_at == l) {
        solo_at = -1;
        tm.solo = false;
        tm.sync();
      }
    }
    if (l == l0) break;
    const int pl = l - 1;
    const int g = (gamma_levels <= 0 || pl < gamma_levels) ? gamma : 1;
    visits += 1ull << (2 * pl);
    if ((int)((visits >> (2 * pl)) & 3) < g) {           // visit the coarser level again (same right side)
      arrive = true;
      continue;
    }
    const Level<T>& F = lv.L(pl);
    for (unsigned i = tm.rank(); i < (unsigned)F.ncell; i += tm.size()) {
      int i0, i1, i2;
      cell_coords(F, i, i0, i1, i2);
      F.u[i] += lv.prolong(pl, i0, i1, i2);
    }
    tm.sync();
    l = pl;
    stage = POST;
    sweeps = nu2;
  }
}

// The levels of a cycle as the grid kernels treat them: above the coarse
// tail's first level the transfers take the nested formulas where the levels
// nest and the tables otherwise, from it on the tables, so that a launch of
// several levels gives the values of the launches it replaces.
template <typename T>
struct GridLevels {
  const Level<T>* Ls;                  // views and tables of levels base, base + 1, ...
  const Xfer<T>* Xs;
  int base, tail_start;
  __device__ const Level<T>& L(int l) const { return Ls[l - base]; }
  __device__ bool nested(int l) const {
    const Level<T>& F = L(l);
    const Level<T>& C = L(l + 1);
    return l < tail_start && nested_levels(F.n0, F.n1, F.n2, C.n0, C.n1, C.n2);
  }
  __device__ void restrict2(int l, const T* fa, const T* fb, int J0, int J1, int J2, T& a, T& b) const {
    if (nested(l)) {
      a = restrict_nested_at(L(l), L(l + 1), fa, J0, J1, J2);
      b = restrict_nested_at(L(l), L(l + 1), fb, J0, J1, J2);
    } else {
      restrict2_at(L(l), Xs[l - base], fa, fb, J0, J1, J2, a, b);
    }
  }
  __device__ T prolong(int l, int i0, int i1, int i2) const {
    return nested(l) ? prolong_nested_at(L(l), L(l + 1), Xs[l - base], i0, i1, i2)
                     : prolong_at(L(l + 1), Xs[l - base], i0, i1, i2);
  }
};

// copies the descriptors of levels l0 .. nl - 1 to shared memory (the blocks
// read them in every phase; ends without a barrier)
template <typename T>
__device__ __forceinline__ void stage_levels(const Level<T>* Ls, const Xfer<T>* Xs, int l0, int nl, Level<T>* sL,
                                             Xfer<T>* sX) {
  static_assert(sizeof(Level<T>) % 4 == 0 && sizeof(Xfer<T>) % 4 == 0, "copied as words");
  const unsigned* a = reinterpret_cast<const unsigned*>(Ls + l0);
  const unsigned* b = reinterpret_cast<const unsigned*>(Xs + l0);
  const int na = (int)(sizeof(Level<T>) / 4) * (nl - l0), nb = (int)(sizeof(Xfer<T>) / 4) * (nl - l0);
  for (int k = threadIdx.x; k < na; k += blockDim.x) reinterpret_cast<unsigned*>(sL)[k] = a[k];
  for (int k = threadIdx.x; k < nb; k += blockDim.x) reinterpret_cast<unsigned*>(sX)[k] = b[k];
}
constexpr int TEAM_LEVELS = 24;

// one cluster (of 1 to CLUSTER_MAX blocks)
template <typename T, int FORM, int MODEL>
__global__ void __launch_bounds__(TAIL_THREADS, 1) k_tail(const Level<T>* __restrict__ Ls, const Xfer<T>* __restrict__ Xs,
                                                       int l0, int nl, int tail_start, int handoff, Phys<T> P, int nu1,
                                                       int nu2, int cmax, T crtol, int gamma, int gamma_levels,
                                                       unsigned long long* stats, int ordering) {
  __shared__ ClusterShared sh;
  __shared__ Level<T> sL[TEAM_LEVELS];
  __shared__ Xfer<T> sX[TEAM_LEVELS];
  stage_levels(Ls, Xs, l0, nl, sL, sX);
  ClusterTeam tm(&sh);
  tm.sync();
  unsigned long long updates = 0;
  team_cycle<T, FORM, MODEL>(GridLevels<T>{sL, sX, l0, tail_start}, l0, nl, P, nu1, nu2, cmax, crtol, gamma,
                             gamma_levels, updates, ordering, handoff, tm);
  if (threadIdx.x == 0 && tm.lead() && stats) atomicAdd(stats, updates);
  tm.sync();                           // (no block leaves while another may still write to its shared memory)
}

// One coarse cell of a boundary-face array of axis ax: the restriction over the
// face's two in-plane axes.
template <typename T>
__device__ __forceinline__ T restrict_face_at(const int* nF, const int* nC, const Xfer<T>& X, int ax,
                                              const T* __restrict__ fine, int J) {
  const int o0 = ax == 0 ? 1 : 0, o1 = ax == 2 ? 1 : 2;
  const int J1 = J / nC[o0], J0 = J - J1 * nC[o0];
  const int c0 = X.rc[o0][J0], c1 = X.rc[o1][J1];
  T s = T(0);
  for (int a1 = 0; a1 < c1; ++a1)
    for (int a0 = 0; a0 < c0; ++a0)
      s += X.rw[o0][RMAX * J0 + a0] * X.rw[o1][RMAX * J1 + a1] *
           fine[X.ri[o0][RMAX * J0 + a0] + (long long)nF[o0] * X.ri[o1][RMAX * J1 + a1]];
  return s;
}

// FP64 boundary conductances of the finest level whose FP32 copies the FP32
// set-up makes first (null: FP64 levels, or none)
struct FaceSource {
  const double* kb[6];
};

// The per-step set-up of the coarse levels in one cluster: every level's
// boundary conductances and, from level ts on, the lagged conductivity
// (psi0 false), or the frozen state (psi0 true) of the levels from ts on.  One
// launch instead of up to seven per level, each of which takes a launch's ~2
// us whatever its size; the values of the launches it replaces.
template <typename T>
__global__ void __launch_bounds__(TAIL_THREADS, 1) k_team_setup(const Level<T>* __restrict__ Ls,
                                                                const Xfer<T>* __restrict__ Xs, int nl, int ts,
                                                                bool psi0, FaceSource src) {
  __shared__ ClusterShared sh;
  __shared__ Level<T> sL[TEAM_LEVELS];
  __shared__ Xfer<T> sX[TEAM_LEVELS];
  stage_levels(Ls, Xs, 0, nl, sL, sX);
  ClusterTeam tm(&sh);
  tm.sync();
  const int nface = 2 * sL[0].dim;
  if (!psi0 && src.kb[0]) {
    for (int f = 0; f < nface; ++f) {
      const int n[3] = {sL[0].n0, sL[0].n1, sL[0].n2};
      const unsigned cells = (unsigned)(sL[0].ncell / n[f >> 1]);
      for (unsigned i = tm.rank(); i < cells; i += tm.size()) const_cast<T*>(sL[0].kb[f])[i] = (T)src.kb[f][i];
    }
    tm.sync();
  }
  const GridLevels<T> lv{sL, sX, 0, nl};
  for (int l = psi0 ? ts : 0; l + 1 < nl; ++l) {
    const Level<T>& F = sL[l];
    const Level<T>& C = sL[l + 1];
    if (!psi0) {
      const int nF[3] = {F.n0, F.n1, F.n2}, nC[3] = {C.n0, C.n1, C.n2};
      for (int f = 0; f < nface; ++f) {
        const unsigned cells = (unsigned)(C.ncell / nC[f >> 1]);
        for (unsigned J = tm.rank(); J < cells; J += tm.size())
          const_cast<T*>(C.kb[f])[J] = restrict_face_at(nF, nC, sX[l], f >> 1, F.kb[f], (int)J);
      }
    }
    if (l >= ts) {
      const T* from = psi0 ? F.psi0 : F.Kc;
      T* to = const_cast<T*>(psi0 ? C.psi0 : C.Kc);
      for (unsigned J = tm.rank(); J < (unsigned)C.ncell; J += tm.size()) {
        int J0, J1, J2;
        cell_coords(C, J, J0, J1, J2);
        to[J] = lv.nested(l) ? restrict_nested_at(F, C, from, J0, J1, J2) : restrict_at(F, sX[l], from, J0, J1, J2);
      }
    }
    tm.sync();
  }
  tm.sync();
}

// The coarse levels of a big grid as one cooperative launch, a grid barrier
// between phases instead of a launch per stage; block 0 alone takes the
// coarse tail's levels.  slots: three global words for the grid
// reductions; stats: the update count
template <typename T, int FORM, int MODEL>
__global__ void __launch_bounds__(COOP_THREADS) k_coop_cycle(const Level<T>* __restrict__ Ls,
                                                             const Xfer<T>* __restrict__ Xs, int l0, int nl,
                                                             int tail_start, Phys<T> P, int nu1, int nu2, int cmax,
                                                             T crtol, int gamma, int gamma_levels,
                                                             unsigned long long* stats, unsigned long long* slots) {
  __shared__ unsigned long long sm[TEAM_WORDS];
  GridTeam tm{slots, sm, 0, false};
  if (tm.rank() == 0) slots[0] = slots[1] = slots[2] = 0ull;
  tm.sync();
  unsigned long long updates = 0;
  team_cycle<T, FORM, MODEL>(GridLevels<T>{Ls + l0, Xs + l0, l0, tail_start}, l0, nl, P, nu1, nu2, cmax, crtol, gamma,
                             gamma_levels, updates, 1, tail_start, tm);
  if (tm.rank() == 0 && stats) atomicAdd(stats, updates);
}

// ---------------------------------------------------------------------------
// Launchers
// ---------------------------------------------------------------------------
inline int grid_for(long long n, int bs = 256) {
  long long b = (n + bs - 1) / bs;
  const long long cap = 152LL * 32;
  if (b > cap) b = cap;
  if (b < 1) b = 1;
  return (int)b;
}

// 3D launch over (units along x, n1 rows, n2 planes): block x-size is a
// power of two between 32 and 128 covering the row
struct Launch3 {
  dim3 grid, block;
};
// (bx_force > 0: that block x-size, as the autotuner chose it)
inline Launch3 launch3(int nx, int n1, int n2, int bx_force = 0) {
  int bx = 32;
  while (bx < nx && bx < 128) bx <<= 1;
  if (bx_force > 0) bx = bx_force;
  Launch3 L;
  L.block = dim3(bx, 1, 1);
  L.grid = dim3((nx + bx - 1) / bx, n1, n2);
  return L;
}

// what the device says of one kernel's clusters (cluster_fit.h)
template <auto KERN>
struct ClusterQuery {
  int threads;
  bool pending() const { return cudaPeekAtLastError() != cudaSuccess; }
  bool consent() const {
    return cudaFuncSetAttribute(KERN, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) == cudaSuccess;
  }
  int held(int blocks) const {
    cudaLaunchConfig_t cfg{};
    cudaLaunchAttribute at{};
    at.id = cudaLaunchAttributeClusterDimension;
    at.val.clusterDim.x = blocks;
    at.val.clusterDim.y = at.val.clusterDim.z = 1;
    cfg.gridDim = dim3(blocks);
    cfg.blockDim = dim3(threads);
    cfg.attrs = &at;
    cfg.numAttrs = 1;
    int n = 0;
    return cudaOccupancyMaxActiveClusters(&n, KERN, &cfg) == cudaSuccess ? n : -1;
  }
  void clear() const { cudaGetLastError(); }
};
template <auto KERN>
inline int cluster_blocks(int blocks, int clusters, int threads) {
  static ClusterFit fits[16];          // by device; a device beyond them is asked every time
  ClusterFit asked;
  int dev = 0;
  cudaGetDevice(&dev);
  return fit_blocks(dev >= 0 && dev < 16 ? fits[dev] : asked, blocks, clusters, ClusterQuery<KERN>{threads});
}

// launches `clusters` clusters of `blocks` thread blocks each, or of the next
// smaller power of two of which the device holds them all at once
template <auto KERN, typename... KA, typename... A>
inline cudaError_t launch_cluster_as(void (*kern)(KA...), int blocks, int clusters, int threads, cudaStream_t s,
                                     A... args) {
  cudaLaunchConfig_t cfg{};
  cudaLaunchAttribute at{};
  at.id = cudaLaunchAttributeClusterDimension;
  at.val.clusterDim.x = cluster_blocks<KERN>(blocks, clusters, threads);
  at.val.clusterDim.y = at.val.clusterDim.z = 1;
  cfg.gridDim = dim3(at.val.clusterDim.x * clusters);
  cfg.blockDim = dim3(threads);
  cfg.stream = s;
  cfg.attrs = &at;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kern, static_cast<KA>(args)...);
}
template <auto KERN, typename... A>
inline cudaError_t launch_cluster(int blocks, int clusters, int threads, cudaStream_t s, A... args) {
  return launch_cluster_as<KERN>(KERN, blocks, clusters, threads, s, args...);
}

// host: calls fn(LawTag<model>{}) for a runtime law (COMPOSITE included)
template <typename Fn>
inline void by_model(int model, Fn&& fn) {
  if (model == HAVERKAMP) fn(LawTag<HAVERKAMP>{});
  else if (model == GARDNER) fn(LawTag<GARDNER>{});
  else if (model == COMPOSITE) fn(LawTag<COMPOSITE>{});
  else fn(LawTag<VANGENUCHTEN>{});
}

template <typename T, int FORM>
struct Dispatch {
  template <int NK>
  static void sweep_nk(const Level<T>& L, const Phys<T>& P, int model, int color, cudaStream_t s, int bx = 0) {
    const Launch3 g = launch3((L.n0 + 1) >> 1, L.n1, L.n2, bx);
    by_model(model, [&](auto m) {
      k_sweep<T, FORM, decltype(m)::value, NK><<<g.grid, g.block, 0, s>>>(L, P, color);
    });
  }
  // the FP32 increment form compiles the common fixed step counts 1 and 2
  static void sweep(const Level<T>& L, const Phys<T>& P, int model, int color, cudaStream_t s, int bx = 0) {
    if (FORM == FORM_DELTA && P.newton_k == 1) sweep_nk<(FORM == FORM_DELTA ? 1 : 0)>(L, P, model, color, s, bx);
    else if (FORM == FORM_DELTA && P.newton_k == 2)
      sweep_nk<(FORM == FORM_DELTA ? 2 : 0)>(L, P, model, color, s, bx);
    else sweep_nk<0>(L, P, model, color, s, bx);
  }
  template <int ZC, int NK>
  static void sweep_pipe_zk(const Level<T>& L, const Phys<T>& P, int model, int color, cudaStream_t s, int bx) {
    Launch3 g = launch3((L.n0 + 1) >> 1, L.n1, L.n2, bx);
    g.grid.z = (L.n2 + ZC - 1) / ZC;
    by_model(model, [&](auto m) {
      k_sweep_pipe<T, FORM, decltype(m)::value, ZC, NK><<<g.grid, g.block, 0, s>>>(L, P, color, nullptr);
    });
  }
  template <int ZC>
  static void sweep_pipe_z(const Level<T>& L, const Phys<T>& P, int model, int color, cudaStream_t s, int bx) {
    if (FORM == FORM_DELTA && P.newton_k == 1)
      sweep_pipe_zk<ZC, (FORM == FORM_DELTA ? 1 : 0)>(L, P, model, color, s, bx);
    else if (FORM == FORM_DELTA && P.newton_k == 2)
      sweep_pipe_zk<ZC, (FORM == FORM_DELTA ? 2 : 0)>(L, P, model, color, s, bx);
    else sweep_pipe_zk<ZC, 0>(L, P, model, color, s, bx);
  }
  // (levels below 2^20 cells keep one cell per thread unless the autotuner
  // chose otherwise (bx > 0): latency, not load throughput, bounds them.
  // The pipelined kernels take blocks of at most 128 threads.)
  static void sweep_pipe(const Level<T>& L, const Phys<T>& P, int model, int color, int planes, cudaStream_t s,
                         int bx = 0) {
    if (planes <= 1 || L.n2 < 2 || (bx == 0 && L.ncell < (1LL << 20))) sweep(L, P, model, color, s, bx);
    else if (planes == 2) sweep_pipe_z<2>(L, P, model, color, s, bx > 128 ? 128 : bx);
    else if (planes == 4) sweep_pipe_z<4>(L, P, model, color, s, bx > 128 ? 128 : bx);
    else sweep_pipe_z<8>(L, P, model, color, s, bx > 128 ? 128 : bx);
  }
  // one lexicographic sweep: a launch per hyperplane, rows of the plane's
  // i2 range only
  template <int NK>
  static void sweep_lex_nk(const Level<T>& L, const Phys<T>& P, int model, cudaStream_t s) {
    int bx = 32;
    while (bx < L.n1 && bx < 128) bx <<= 1;
    const int nplanes = L.n0 + L.n1 + L.n2 - 2;
    by_model(model, [&](auto m) {
      for (int p = 0; p < nplanes; ++p) {
        const int i2lo = std::max(0, p - (L.n0 - 1) - (L.n1 - 1)), i2hi = std::min(L.n2 - 1, p);
        const dim3 grid((L.n1 + bx - 1) / bx, i2hi - i2lo + 1, 1);
        k_sweep_plane<T, FORM, decltype(m)::value, NK><<<grid, bx, 0, s>>>(L, P, p, i2lo);
      }
    });
  }
  static void sweep_lex(const Level<T>& L, const Phys<T>& P, int model, cudaStream_t s) {
    if (FORM == FORM_DELTA && P.newton_k == 1) sweep_lex_nk<(FORM == FORM_DELTA ? 1 : 0)>(L, P, model, s);
    else if (FORM == FORM_DELTA && P.newton_k == 2) sweep_lex_nk<(FORM == FORM_DELTA ? 2 : 0)>(L, P, model, s);
    else sweep_lex_nk<0>(L, P, model, s);
  }
  // whether sweep_resid applies to a level (the pipelined two-plane kernel)
  static bool fusable(const Level<T>& L, int planes) {
    return FORM == FORM_DELTA && planes == 2 && L.n2 >= 2 && L.ncell >= (1LL << 20);
  }
  // the last half-sweep of a smoothing (colour 1), writing the defects of
  // its cells; residual_color(0) then gives colour 0's: d and ||d||_inf
  // (into *norm) at the end of the smoothing, as one defect pass would
  static void sweep_resid(const Level<T>& L, const Phys<T>& P, int model, unsigned long long* norm, cudaStream_t s) {
    auto sweep_r = [&](auto nk) {
      Launch3 g = launch3((L.n0 + 1) >> 1, L.n1, L.n2);
      g.grid.z = (L.n2 + 1) / 2;
      by_model(model, [&](auto m) {
        k_sweep_pipe<T, FORM, decltype(m)::value, 2, decltype(nk)::value, true><<<g.grid, g.block, 0, s>>>(L, P, 1,
                                                                                                          norm);
      });
    };
    if (FORM == FORM_DELTA && P.newton_k == 1) sweep_r(LawTag<(FORM == FORM_DELTA ? 1 : 0)>{});
    else if (FORM == FORM_DELTA && P.newton_k == 2) sweep_r(LawTag<(FORM == FORM_DELTA ? 2 : 0)>{});
    else sweep_r(LawTag<0>{});
  }
  static void residual_color(const Level<T>& L, const Phys<T>& P, int model, int color, unsigned long long* norm,
                             cudaStream_t s) {
    const Launch3 g = launch3((L.n0 + 1) >> 1, L.n1, L.n2);
    by_model(model, [&](auto m) {
      k_residual_color<T, FORM, decltype(m)::value><<<g.grid, g.block, 0, s>>>(L, P, color, norm);
    });
  }
  static void residual(const Level<T>& L, const Phys<T>& P, int model, unsigned long long* norm,
                       cudaStream_t s, int bx = 0) {
    const Launch3 g = launch3(L.n0, L.n1, L.n2, bx);
    by_model(model, [&](auto m) {
      k_residual<T, FORM, decltype(m)::value><<<g.grid, g.block, 0, s>>>(L, P, norm);
    });
  }
  static void tau(const Level<T>& C, const Phys<T>& P, int model, cudaStream_t s) {
    const Launch3 g = launch3(C.n0, C.n1, C.n2);
    by_model(model, [&](auto m) { k_tau<T, FORM, decltype(m)::value><<<g.grid, g.block, 0, s>>>(C, P); });
  }
  static void restrict2(const Level<T>& F, const Level<T>& C, const Xfer<T>& X, const T* fa, const T* fb,
                        T* ca, T* cb, cudaStream_t s, int cs_mask = 0) {
    const Launch3 g = launch3(C.n0, C.n1, C.n2);
    if (nested_levels(F.n0, F.n1, F.n2, C.n0, C.n1, C.n2))
      k_restrict_nested<T><<<g.grid, g.block, 0, s>>>(F, C, fa, fb, ca, cb, cs_mask);
    else
      k_restrict<T><<<g.grid, g.block, 0, s>>>(F, C, X, fa, fb, ca, cb, cs_mask);
  }
  static void prolong(const Level<T>& F, const Level<T>& C, const Xfer<T>& X, cudaStream_t s) {
    const Launch3 g = launch3(F.n0, F.n1, F.n2);
    if (nested_levels(F.n0, F.n1, F.n2, C.n0, C.n1, C.n2) && tiled_transfer(F.dim, F.n0, F.n1, F.n2)) {
      using TT = TransferTile<T>;
      const dim3 grid((F.n0 + TT::PX - 1) / TT::PX, (F.n1 + TT::PY - 1) / TT::PY, (F.n2 + TT::PZ - 1) / TT::PZ);
      k_prolong_tiled<T><<<grid, TT::PX * TT::PY, 0, s>>>(F, C, X);
    } else if (nested_levels(F.n0, F.n1, F.n2, C.n0, C.n1, C.n2))
      k_prolong_nested<T><<<g.grid, g.block, 0, s>>>(F, C, X);
    else
      k_prolong<T><<<g.grid, g.block, 0, s>>>(F, C, X);
  }
  static void team_setup(const Level<T>* dLs, const Xfer<T>* dXs, int nl, int ts, int blocks, bool psi0,
                         const double* const* kb, cudaStream_t s) {
    FaceSource src{};
    for (int f = 0; kb && f < 6; ++f) src.kb[f] = kb[f];
    launch_cluster<k_team_setup<T>>(blocks, 1, TAIL_THREADS, s, dLs, dXs, nl, ts, psi0, src);
  }
  // the cooperative coarse cycle: the most blocks that can be co-resident
  static int coop_max_blocks(int model) {
    int per_sm = 0, dev = 0, nsm = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
    by_model(model, [&](auto m) {
      cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_coop_cycle<T, FORM, decltype(m)::value>, COOP_THREADS,
                                                    0);
    });
    return per_sm * nsm;
  }
  static cudaError_t coop(const Level<T>* dLs, const Xfer<T>* dXs, int l0, int nl, int tail_start, const Phys<T>& P,
                          int model, int nu1, int nu2, int cmax, T crtol, int gamma, int gamma_levels,
                          unsigned long long* stats, unsigned long long* slots, int blocks, cudaStream_t s) {
    cudaError_t e = cudaSuccess;
    Phys<T> Pv = P;
    void* args[] = {(void*)&dLs, (void*)&dXs, (void*)&l0, (void*)&nl, (void*)&tail_start, (void*)&Pv, (void*)&nu1,
                    (void*)&nu2, (void*)&cmax, (void*)&crtol, (void*)&gamma, (void*)&gamma_levels, (void*)&stats,
                    (void*)&slots};
    by_model(model, [&](auto m) {
      e = cudaLaunchCooperativeKernel((const void*)k_coop_cycle<T, FORM, decltype(m)::value>, dim3(blocks),
                                      dim3(COOP_THREADS), args, 0, s);
    });
    return e;
  }
  // one cluster of `blocks` blocks (a power of two up to CLUSTER_MAX; fewer
  // when the device cannot place that many)
  static void tail(const Level<T>* dLs, const Xfer<T>* dXs, int l0, int nl, const TeamShape& ts, const Phys<T>& P,
                   int model, int nu1, int nu2, int cmax, T crtol, int gamma, int gamma_levels,
                   unsigned long long* stats, int ordering, cudaStream_t s) {
    by_model(model, [&](auto m) {
      launch_cluster<k_tail<T, FORM, decltype(m)::value>>(ts.blocks, 1, TAIL_THREADS, s, dLs, dXs, l0, nl,
                                                          ts.tail_start, ts.handoff, P, nu1, nu2, cmax, crtol, gamma,
                                                          gamma_levels, stats, ordering);
    });
  }
};

}  // namespace rich
