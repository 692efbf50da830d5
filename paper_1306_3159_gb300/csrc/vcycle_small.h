// The coarse end of a V-cycle inside one CTA (device code shared by the
// single-CTA kernel and the cluster kernel).
#pragma once

#include "internal.h"

namespace ibrd {

__device__ __forceinline__ int wrap_small(int i, int n) { return i < 0 ? i + n : (i >= n ? i - n : i); }

// The V-cycle over levels first .. lv.n - 1 in one CTA (at most a few thousand
// cells), x and b of each level in shared memory (X, B: level `first` first, b
// with its shift removed, x the guess of level `first` and zero below);
// smoothing, residual restriction, the exact coarsest solve and prolongation run
// with block-wide barriers between phases. Arithmetic matches the multi-kernel
// levels. The caller has synchronised the block; it is synchronised on return.
template <typename T>
__device__ void vcycle_small_levels(const CoarseLevels& lv, int first, T* X, T* B, const T* __restrict__ table,
                                    int nu1, int nu2) {
  const int tid = threadIdx.x, nt = blockDim.x, base = lv.off[first];
  // cell index -> (i, j, k); shifts when the level's nx, ny are powers of 2
  auto decode = [&](int l, int c, int& i, int& j, int& k) {
    const int lx = lv.lgx[l], ly = lv.lgy[l];
    if (lx >= 0 && ly >= 0) {
      i = c & (lv.nx[l] - 1);
      j = (c >> lx) & (lv.ny[l] - 1);
      k = c >> (lx + ly);
    } else {
      i = c % lv.nx[l];
      j = (c / lv.nx[l]) % lv.ny[l];
      k = c / (lv.nx[l] * lv.ny[l]);
    }
  };
  // one red-black sweep on level l (all sides even): each half-sweep visits
  // only the cells of its colour, enumerated as (i/2, j, k)
  auto sweep = [&](int l) {
    const int nx = lv.nx[l], ny = lv.ny[l], nz = lv.nz[l];
    const int hx = nx >> 1, nh = hx * ny * nz, plane = nx * ny;
    T* x = X + lv.off[l] - base;
    const T* b = B + lv.off[l] - base;
    const T inv = (T)lv.inv[l], off = (T)lv.offd[l];
    const int lx = lv.lgx[l], ly = lv.lgy[l];
    const bool pow2 = lx >= 1 && ly >= 0;
    for (int colour = 0; colour < 2; ++colour) {
      for (int p = tid; p < nh; p += nt) {
        int ih, j, k;
        if (pow2) {
          ih = p & (hx - 1);
          j = (p >> (lx - 1)) & (ny - 1);
          k = p >> (lx - 1 + ly);
        } else {
          ih = p % hx;
          j = (p / hx) % ny;
          k = p / (hx * ny);
        }
        const int i = 2 * ih + ((j + k + colour) & 1);
        const int rowc = k * plane + j * nx;
        const int c = rowc + i;
        const int xw = rowc + (i == 0 ? nx - 1 : i - 1), xe = rowc + (i == nx - 1 ? 0 : i + 1);
        const int ys = c + (j == 0 ? plane - nx : -nx), yn = c + (j == ny - 1 ? nx - plane : nx);
        const int zd = c + (k == 0 ? plane * (nz - 1) : -plane), zu = c + (k == nz - 1 ? -plane * (nz - 1) : plane);
        const T sum = ((x[xw] + x[xe]) + (x[ys] + x[yn])) + (x[zd] + x[zu]);
        x[c] = (b[c] + off * sum) * inv;
      }
      __syncthreads();
    }
  };
  const int last = lv.n - 1;
  for (int l = first; l < last; ++l) {
    for (int sw = 0; sw < nu1; ++sw) sweep(l);
    // residual restriction to level l+1
    const int nx = lv.nx[l], ny = lv.ny[l], nz = lv.nz[l];
    const int nxc = nx >> 1, nyc = ny >> 1, nc = nxc * nyc * (nz >> 1);
    const T* x = X + lv.off[l] - base;
    const T* b = B + lv.off[l] - base;
    T* bc = B + lv.off[l + 1] - base;
    const T diag = (T)lv.diag[l], off = (T)lv.offd[l];
    // one child per thread: entry e = 8 C + (dz, dy, dx) bits, so the 8
    // children of a coarse cell sit in 8 neighbouring lanes and are summed
    // by shuffles (the loop bound is a multiple of 32 so warps stay whole)
    const int nf = 8 * nc, nround = (nf + 31) & ~31;
    for (int e = tid; e < nround; e += nt) {
      T r = 0;
      if (e < nf) {
        int I, J, K;
        decode(l + 1, e >> 3, I, J, K);
        const int i = 2 * I + (e & 1), j = 2 * J + ((e >> 1) & 1), k = 2 * K + (e >> 2 & 1);
        const int c = (k * ny + j) * nx + i;
        const T s = ((x[c - i + wrap_small(i - 1, nx)] + x[c - i + wrap_small(i + 1, nx)]) +
                     (x[c + (wrap_small(j - 1, ny) - j) * nx] + x[c + (wrap_small(j + 1, ny) - j) * nx])) +
                    (x[c + (wrap_small(k - 1, nz) - k) * nx * ny] + x[c + (wrap_small(k + 1, nz) - k) * nx * ny]);
        r = b[c] - (diag * x[c] - off * s);
      }
      r += __shfl_xor_sync(0xffffffffu, r, 1);
      r += __shfl_xor_sync(0xffffffffu, r, 2);
      r += __shfl_xor_sync(0xffffffffu, r, 4);
      if (e < nf && (e & 7) == 0) bc[e >> 3] = r * (T)0.125;
    }
    __syncthreads();
  }
  {
    // exact coarsest solve with the circulant table
    const int nx = lv.nx[last], ny = lv.ny[last], nz = lv.nz[last], n = nx * ny * nz;
    T* x = X + lv.off[last] - base;
    const T* b = B + lv.off[last] - base;
    for (int t = tid; t < n; t += nt) {
      const int ix = t % nx, iy = (t / nx) % ny, iz = t / (nx * ny);
      T acc = 0;
      for (int u = 0; u < n; ++u) {
        const int jx = u % nx, jy = (u / nx) % ny, jz = u / (nx * ny);
        const int dx = ix - jx + (ix < jx ? nx : 0), dy = iy - jy + (iy < jy ? ny : 0), dz = iz - jz + (iz < jz ? nz : 0);
        acc += table[(dz * ny + dy) * nx + dx] * b[u];
      }
      x[t] = acc;
    }
    __syncthreads();
  }
  for (int l = last - 1; l >= first; --l) {
    const int nx = lv.nx[l], ny = lv.ny[l], nz = lv.nz[l], n = nx * ny * nz;
    const int nxc = nx >> 1, nyc = ny >> 1, nzc = nz >> 1;
    T* x = X + lv.off[l] - base;
    const T* xc = X + lv.off[l + 1] - base;
    for (int c = tid; c < n; c += nt) {
      int i, j, k;
      decode(l, c, i, j, k);
      const int I = i >> 1, J = j >> 1, K = k >> 1;
      const int I2 = (i & 1) ? wrap_small(I + 1, nxc) : wrap_small(I - 1, nxc);
      const int J2 = (j & 1) ? wrap_small(J + 1, nyc) : wrap_small(J - 1, nyc);
      const int K2 = (k & 1) ? wrap_small(K + 1, nzc) : wrap_small(K - 1, nzc);
      auto e = [&](int kk, int jj, int ii) { return xc[(kk * nyc + jj) * nxc + ii]; };
      // z, then y, then x (each axis scaled by 4)
      auto zy = [&](int ii) {
        return prolong_axis(prolong_axis(e(K, J, ii), e(K2, J, ii)), prolong_axis(e(K, J2, ii), e(K2, J2, ii)));
      };
      x[c] = prolong_add(x[c], prolong_axis(zy(I), zy(I2)));
    }
    __syncthreads();
    for (int sw = 0; sw < nu2; ++sw) sweep(l);
  }
}

}  // namespace ibrd
