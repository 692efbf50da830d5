// The coarse end of the FP64 V-cycle (Sec. III.E) in one launch of a thread
// block cluster.
//
// One SM of this GPU does two FP64 operations per clock, so a coarse level is
// bound by how many SMs work on it long before memory matters: a 16^3 level
// with two sweeps on each side is about 190000 FP64 operations, 46 us on one SM
// (86 us in the single-CTA kernel of smoother.cu, most of it that). Separate
// launches over the whole chip cost about 3 us for each half-sweep of a level
// this small. Here 16 CTAs of a cluster share the levels of 600 cells and more,
// and its CTA 0 runs the rest in its own shared memory. 32^3 and below: 70 us,
// against 147 us for the separate kernels of the 32^3 level and the single-CTA
// one of the others; 24^3 and below: 51 us, against 95.
//
// * A shared level is cut in z between pairs of planes (2K, 2K + 1), so that a
//   coarse plane's children are one CTA's. A CTA keeps its planes of x with one
//   halo plane on each side, and its planes of b, in shared memory; the cells a
//   half-sweep updates in its outer planes are also stored in the neighbours'
//   halos (distributed shared memory), and a cluster barrier ends the half-sweep.
// * An update is (b + off * neighbours) * inv, with the one rounding of inv = 1 / diag
//   in both terms. (b kept divided by the diagonal and a rounded off / diag save
//   one of its seven instructions, but the sweeps then scale smooth fields: the error of a
//   V-cycle at 64^3 went from 6e-16 to 1e-15 for alpha = 0.01.)
// * After a sweep the residual of the black cells is zero: the restriction forms
//   it in the red cells only (all of them when there was no sweep), together with
//   what the rounding of inv leaves in the black ones (slack x), and the
//   prolongation corrects only the black cells when a sweep follows, which reads
//   no others. Its z-part is formed once per fine plane and coarse cell, also
//   for the halo planes, so that it needs no exchange.
#include <cuda_runtime.h>

#include "internal.h"
#include "vcycle_small.h"

namespace ibrd {
namespace {

constexpr int kClusterThreads = 512;
constexpr int kClusterCells = 3072;  // most cells of a level one CTA takes
constexpr int kSharedCells = 600;    // levels below this many cells are CTA 0's

__device__ __forceinline__ void cluster_sync() {
  asm volatile("barrier.cluster.arrive.release.aligned;\nbarrier.cluster.wait.acquire.aligned;\n" ::: "memory");
}
// the address in CTA `rank`'s shared memory of what p is here
__device__ __forceinline__ unsigned peer(const void* p, int rank) {
  unsigned r;
  asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"((unsigned)__cvta_generic_to_shared(p)), "r"(rank));
  return r;
}
__device__ __forceinline__ void put_peer(unsigned a, double v) {
  asm volatile("st.shared::cluster.f64 [%0], %1;" ::"r"(a), "d"(v) : "memory");
}
__device__ __forceinline__ double get_peer(unsigned a) {
  double v;
  asm volatile("ld.shared::cluster.f64 %0, [%1];" : "=d"(v) : "r"(a) : "memory");
  return v;
}

// The split of a level's nz / 2 plane pairs over C CTAs.
struct Split {
  int pairs, C;
  __host__ __device__ Split(int nz, int C_) : pairs(nz >> 1), C(C_) {}
  __host__ __device__ int start(int r) const { return r * pairs / C; }
  __host__ __device__ int owner(int pair) const { return ((pair + 1) * C + pairs - 1) / pairs - 1; }
  __host__ __device__ int most() const { return (pairs + C - 1) / C; }  // pairs of one CTA
};

// Shared-memory layout, in doubles: per shared level x (2 most + 2 planes) and b
// (2 most planes); the z-interpolated coarse field of the largest one; CTA 0's
// own levels, x and then b.
struct Layout {
  int x[kMaxSmallLevels], b[kMaxSmallLevels], zc, own, total;
  __host__ __device__ Layout(const CoarseLevels& lv, int shared, int C) {
    int o = 0, most_zc = 0;
    for (int l = 0; l < shared; ++l) {
      const int plane = lv.nx[l] * lv.ny[l], m = 2 * Split(lv.nz[l], C).most();
      x[l] = o;
      o += (m + 2) * plane;
      b[l] = o;
      o += m * plane;
      const int z = (m + 2) * (plane >> 2);
      most_zc = z > most_zc ? z : most_zc;
    }
    zc = o;
    o += most_zc;
    own = o;
    o += 2 * (lv.total - lv.off[shared]);
    total = o;
  }
};

__global__ void __launch_bounds__(kClusterThreads) k_vcycle_cluster(const __grid_constant__ CoarseLevels lv, int shared,
                                                                    int C, const double* __restrict__ bg,
                                                                    double* __restrict__ xg,
                                                                    const double* __restrict__ bshift,
                                                                    const double* __restrict__ table, int zero,
                                                                    int nu1, int nu2) {
  extern __shared__ __align__(16) double sm[];
  const Layout L(lv, shared, C);
  const int tid = threadIdx.x, nt = blockDim.x, rank = blockIdx.x;  // the grid is one cluster
  double* own_x = sm + L.own;
  double* own_b = own_x + (lv.total - lv.off[shared]);
  // this CTA's part of shared level l
  struct Part {
    int nx, ny, nz, plane, k0, np, below, above, below_np;  // planes [k0, k0 + np); the ranks next to them in z
    double inv, diag, off;
  };
  auto part = [&](int l) {
    Part p;
    p.nx = lv.nx[l], p.ny = lv.ny[l], p.nz = lv.nz[l];
    p.plane = p.nx * p.ny;
    const Split s(p.nz, C);
    const int a = s.start(rank), e = s.start(rank + 1);
    p.k0 = 2 * a;
    p.np = 2 * (e - a);
    p.below = s.owner(a == 0 ? s.pairs - 1 : a - 1);
    p.above = s.owner(e >= s.pairs ? 0 : e);
    p.below_np = 2 * (s.start(p.below + 1) - s.start(p.below));
    p.diag = lv.diag[l], p.off = lv.offd[l];
    p.inv = lv.inv[l];
    return p;
  };
  // the neighbours' values around cell (i, j) of local plane kk (x planes are shifted by the lower halo)
  auto nbr_sum = [&](const double* X, const Part& p, int i, int j, int kk) {
    const double* c = X + (kk + 1) * p.plane;
    const int row = j * p.nx;
    const double w = c[row + (i == 0 ? p.nx - 1 : i - 1)], e = c[row + (i == p.nx - 1 ? 0 : i + 1)];
    const double s = c[(j == 0 ? p.ny - 1 : j - 1) * p.nx + i], n = c[(j == p.ny - 1 ? 0 : j + 1) * p.nx + i];
    return ((w + e) + (s + n)) + (c[row + i - p.plane] + c[row + i + p.plane]);
  };
  // cells of one colour in the local planes, as (i, j, kk)
  auto for_colour = [&](const Part& p, int colour, auto&& f) {
    const int hx = p.nx >> 1, per = hx * p.ny;
    for (int c = tid; c < per * p.np; c += nt) {
      const int kk = c / per, r = c - kk * per, j = r / hx;
      f(2 * (r - j * hx) + ((j + p.k0 + kk + colour) & 1), j, kk);
    }
  };
  auto sweep = [&](int l, const Part& p) {
    double* X = sm + L.x[l];
    const double* B = sm + L.b[l];
    for (int colour = 0; colour < 2; ++colour) {
      for_colour(p, colour, [&](int i, int j, int kk) {
        const int o = j * p.nx + i;
        const double v = fma(p.off, nbr_sum(X, p, i, j, kk), B[kk * p.plane + o]) * p.inv;
        X[(kk + 1) * p.plane + o] = v;
        if (kk == 0) put_peer(peer(X + (p.below_np + 1) * p.plane + o, p.below), v);
        if (kk == p.np - 1) put_peer(peer(X + o, p.above), v);
      });
      cluster_sync();
    }
  };

  // set-up: x (the guess or zero) and b of the top level, zero x below
  {
    const double sh = bshift ? *bshift : 0.0;
    const Part p = part(0);
    double* X = sm + L.x[0];
    for (int c = tid; c < p.np * p.plane; c += nt) sm[L.b[0] + c] = bg[(size_t)p.k0 * p.plane + c] - sh;
    for (int c = tid; c < (p.np + 2) * p.plane; c += nt) {
      const int kk = c / p.plane, k = p.k0 - 1 + kk;
      X[c] = zero || p.np == 0 ? 0.0
                               : xg[(size_t)(k < 0 ? p.nz - 1 : (k >= p.nz ? 0 : k)) * p.plane + (c - kk * p.plane)];
    }
    for (int l = 1; l < shared; ++l) {
      const Part q = part(l);
      for (int c = tid; c < (q.np + 2) * q.plane; c += nt) sm[L.x[l] + c] = 0.0;
    }
    if (rank == 0)
      for (int c = tid; c < lv.total - lv.off[shared]; c += nt) own_x[c] = 0.0;
  }
  cluster_sync();

  for (int l = 0; l < shared; ++l) {
    const Part p = part(l);
    for (int s = 0; s < nu1; ++s) sweep(l, p);
    // restriction: four entries (dy, dz) per coarse cell in neighbouring lanes,
    // each the red cell of its x-pair (and, without a sweep, the black one)
    const double* X = sm + L.x[l];
    const double* B = sm + L.b[l];
    const int nxc = p.nx >> 1, nyc = p.ny >> 1, cplane = nxc * nyc, nc = cplane * (p.np >> 1);
    const bool next_shared = l + 1 < shared;
    const Split sn(p.nz >> 1, C);  // of the next level, when it is shared
    const double slack = nu1 > 0 ? fma(-p.diag, p.inv, 1.0) * p.diag : 0.0;
    for (int e = tid; e < ((4 * nc + 31) & ~31); e += nt) {
      const int cell = e >> 2, dy = e & 1, dz = (e >> 1) & 1;
      double r = 0.0;
      int K = 0, o = 0;
      if (cell < nc) {
        K = cell / cplane;
        o = cell - K * cplane;
        const int J = o / nxc, I = o - J * nxc, j = 2 * J + dy, kk = 2 * K + dz;
        for (int colour = 0; colour < (nu1 > 0 ? 1 : 2); ++colour) {
          const int i = 2 * I + ((j + p.k0 + kk + colour) & 1), at = j * p.nx + i;
          const double x = X[(kk + 1) * p.plane + at];
          r += fma(slack, x, fma(p.off, nbr_sum(X, p, i, j, kk), fma(-p.diag, x, B[kk * p.plane + at])));
        }
      }
      r += __shfl_xor_sync(0xffffffffu, r, 1);
      r += __shfl_xor_sync(0xffffffffu, r, 2);
      if (cell < nc && (e & 3) == 0) {
        const int Kg = (p.k0 >> 1) + K;
        r *= 0.125;
        if (next_shared) {
          const int to = sn.owner(Kg >> 1);
          put_peer(peer(sm + L.b[l + 1] + (Kg - 2 * sn.start(to)) * cplane + o, to), r);
        } else {
          put_peer(peer(own_b + Kg * cplane + o, 0), r);
        }
      }
    }
    cluster_sync();
  }
  if (rank == 0) vcycle_small_levels<double>(lv, shared, own_x, own_b, table, nu1, nu2);
  cluster_sync();
  for (int l = shared - 1; l >= 0; --l) {
    const Part p = part(l);
    double* X = sm + L.x[l];
    double* Z = sm + L.zc;
    const int nxc = p.nx >> 1, nyc = p.ny >> 1, nzc = p.nz >> 1, cplane = nxc * nyc;
    const bool next_shared = l + 1 < shared;
    const Split sn(p.nz >> 1, C);
    // coarse plane K (periodic), entry o
    auto coarse = [&](int K, int o) {
      K = K < 0 ? nzc - 1 : (K >= nzc ? 0 : K);
      if (!next_shared) return get_peer(peer(own_x + K * cplane + o, 0));
      const int r = sn.owner(K >> 1);
      return get_peer(peer(sm + L.x[l + 1] + (K - 2 * sn.start(r) + 1) * cplane + o, r));
    };
    // z between the parent plane and the one on the fine plane's side, for the local planes and both halos
    if (p.np > 0)
      for (int c = tid; c < (p.np + 2) * cplane; c += nt) {
        const int kk = c / cplane - 1, o = c % cplane, k = p.k0 + kk;  // k = -1 .. nz
        const int K = k >> 1;                                          // (floor)
        Z[c] = prolong_axis(coarse(K, o), coarse((k & 1) ? K + 1 : K - 1, o));
      }
    __syncthreads();
    // y, then x
    if (p.np > 0) {
      const int per = nxc * p.ny;
      for (int c = tid; c < per * (p.np + 2); c += nt) {
        const int kk = c / per, r = c - kk * per, j = r / nxc, I = r - j * nxc, J = j >> 1;
        const int J2 = (j & 1) ? (J == nyc - 1 ? 0 : J + 1) : (J == 0 ? nyc - 1 : J - 1);
        const double *z1 = Z + kk * cplane + J * nxc, *z2 = Z + kk * cplane + J2 * nxc;
        const double mid = prolong_axis(z1[I], z2[I]);
        double* row = X + kk * p.plane + j * p.nx;
        for (int colour = nu2 > 0 ? 1 : 0; colour < 2; ++colour) {
          const int i = 2 * I + ((j + p.k0 + kk - 1 + colour) & 1);
          const int I2 = (i & 1) ? (I == nxc - 1 ? 0 : I + 1) : (I == 0 ? nxc - 1 : I - 1);
          row[i] = prolong_add(row[i], prolong_axis(mid, prolong_axis(z1[I2], z2[I2])));
        }
      }
    }
    cluster_sync();  // the neighbours may store into the halos again
    for (int s = 0; s < nu2; ++s) sweep(l, p);
  }
  const Part p = part(0);
  for (int c = tid; c < p.np * p.plane; c += nt) xg[(size_t)p.k0 * p.plane + c] = sm[L.x[0] + p.plane + c];
  cluster_sync();  // no CTA leaves while another may reach its shared memory
}

// Shared levels of a hierarchy on a cluster of C, 0 if it does not fit one.
int shared_levels(const CoarseLevels& lv, int C) {
  int shared = 0;
  for (; shared < lv.n - 1; ++shared) {
    const int l = shared, n = lv.nx[l] * lv.ny[l] * lv.nz[l];
    if (n < kSharedCells) break;
    if (2 * Split(lv.nz[l], C).most() * lv.nx[l] * lv.ny[l] > kClusterCells) return 0;
  }
  if (shared == 0 || Layout(lv, shared, C).total * (int)sizeof(double) > 200 * 1024) return 0;
  return shared;
}

// CTAs of the cluster this device runs the kernel with: 16, or 8 where the
// larger (non-portable) size is not available; per device.
int cluster_size() {
  static std::atomic<int> size[64];
  int dev = 0;
  IBRD_CUDA(cudaGetDevice(&dev));
  int c = size[dev & 63].load(std::memory_order_acquire);
  if (c) return c;
  const void* f = (const void*)k_vcycle_cluster;
  IBRD_CUDA(cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024));
  c = 8;
  if (cudaFuncSetAttribute(f, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) == cudaSuccess) {
    cudaLaunchConfig_t cfg{};
    cudaLaunchAttribute at{};
    at.id = cudaLaunchAttributeClusterDimension;
    at.val.clusterDim = {16, 1, 1};
    cfg.gridDim = dim3(16);
    cfg.blockDim = dim3(kClusterThreads);
    cfg.dynamicSmemBytes = 200 * 1024;
    cfg.attrs = &at;
    cfg.numAttrs = 1;
    int n = 0;
    if (cudaOccupancyMaxActiveClusters(&n, f, &cfg) == cudaSuccess && n > 0) c = 16;
  }
  cudaGetLastError();
  size[dev & 63].store(c, std::memory_order_release);
  return c;
}

}  // namespace

bool vcycle_cluster_ok(const CoarseLevels& lv) { return lv.n >= 2 && shared_levels(lv, cluster_size()) > 0; }

void launch_vcycle_cluster(const CoarseLevels& lv, const double* b, double* x, const double* bshift,
                           const double* table, bool zero, int nu1, int nu2, cudaStream_t s) {
  const int C = cluster_size(), shared = shared_levels(lv, C);
  if (shared == 0) throw CudaError{cudaErrorInvalidValue, "cluster V-cycle levels"};
  cudaLaunchConfig_t cfg{};
  cudaLaunchAttribute at{};
  at.id = cudaLaunchAttributeClusterDimension;
  at.val.clusterDim = {(unsigned)C, 1, 1};
  cfg.gridDim = dim3(C);
  cfg.blockDim = dim3(kClusterThreads);
  cfg.dynamicSmemBytes = Layout(lv, shared, C).total * sizeof(double);
  cfg.stream = s;
  cfg.attrs = &at;
  cfg.numAttrs = 1;
  prof_begin(P_RBGS64, s);
  IBRD_CUDA(cudaLaunchKernelEx(&cfg, k_vcycle_cluster, lv, shared, C, b, x, bshift, table, zero ? 1 : 0, nu1, nu2));
  prof_end(P_RBGS64, s, "vcycle_cluster", 16.0 * lv.total);
}

}  // namespace ibrd
