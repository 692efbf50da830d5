// Blob kernels: per-blob Peskin weights, tile binning, spreading S and
// averaging J (Sec. II.A, Sec. III.A, Eq. tensor_product).
//
// Each blob touches 4 cells per axis (Peskin 4-point kernel; the 3-point
// kernel uses 3 and a zero fourth weight). Spreading never uses global
// atomics on the field: blobs are binned by the 8x8x8 cell tiles their
// support touches, and one CTA per occupied tile gathers, for each of its
// cells, the contributions of the tile's blobs in increasing blob index, so
// the result is deterministic and each field cell is written once.
#include <algorithm>
#include <climits>
#include <cmath>

#include "internal.h"

namespace ibrd {
namespace {

// Peskin 4-point kernel phi4(r), r in units of h (Peskin, Acta Numerica 2002).
__device__ __forceinline__ double phi4(double r) {
  r = fabs(r);
  if (r < 1.0) return (3.0 - 2.0 * r + sqrt(1.0 + 4.0 * r - 4.0 * r * r)) * 0.125;
  if (r < 2.0) return (5.0 - 2.0 * r - sqrt(-7.0 + 12.0 * r - 4.0 * r * r)) * 0.125;
  return 0.0;
}

// Peskin 3-point kernel phi3(r) (Roma, Peskin and Berger 1999).
__device__ __forceinline__ double phi3(double r) {
  r = fabs(r);
  if (r <= 0.5) return (1.0 + sqrt(1.0 - 3.0 * r * r)) / 3.0;
  if (r < 1.5) {
    const double t = 1.0 - r;
    return (5.0 - 3.0 * r - sqrt(1.0 - 3.0 * t * t)) / 6.0;
  }
  return 0.0;
}

__device__ __forceinline__ int pmod(int a, int n) {
  int r = a % n;
  return r < 0 ? r + n : r;
}

// The distinct tiles under a blob's 4 cells of one axis, in order of appearance;
// -1 where there are fewer. Three only where the last tile of the axis has one
// or two cells and the support crosses all of it.
__device__ __forceinline__ void axis_tiles(int4 ix, int* t) {
  const int a = ix.x / kTile, b = ix.y / kTile, c = ix.z / kTile, d = ix.w / kTile;
  t[0] = a;
  t[1] = b != a ? b : c != a ? c : d != a ? d : -1;
  t[2] = (c != a && c != t[1]) ? c : (d != a && d != t[1]) ? d : -1;
}
int max_axis_tiles(int n, int tiles) { return std::min(tiles, n % kTile == 1 || n % kTile == 2 ? 3 : 2); }

// visit(tile) for the tiles of a blob, shared out over 8 threads: thread c takes
// the ones whose place along (x, y, z) has the parities of c's bits.
template <typename F>
__device__ __forceinline__ void blob_tiles(int4 ix, int4 iy, int4 iz, int c, int ntx, int nty, F&& visit) {
  int tx[3], ty[3], tz[3];
  axis_tiles(ix, tx);
  axis_tiles(iy, ty);
  axis_tiles(iz, tz);
#pragma unroll
  for (int u = 0; u < 8; ++u) {  // first or second place of each axis that the thread has
    const int px = c & 1, py = (c >> 1) & 1, pz = c >> 2;
    const int x = (u & 1) ? (px ? -1 : tx[2]) : (px ? tx[1] : tx[0]);
    const int y = (u & 2) ? (py ? -1 : ty[2]) : (py ? ty[1] : ty[0]);
    const int z = (u & 4) ? (pz ? -1 : tz[2]) : (pz ? tz[1] : tz[0]);
    if (x >= 0 && y >= 0 && z >= 0) visit(x + ntx * (y + nty * z));
  }
}

// Per blob and axis: wrapped position, 4 wrapped cell indices, 4 weights; and the
// number of blobs that touch each tile (count zeroed before). One CTA per 32
// blobs: a thread per blob and axis for the weights, whose divisions and square
// roots are a long FP64 chain, then 8 threads per blob for its tiles. (A thread
// per blob in CTAs of 128 left 4096 blobs on 32 of the SMs: 14.5 us, and 3.4 us
// for the counts in a launch of their own; 7.0 us for both.)
constexpr int kPrepBlobs = 32;
__global__ void __launch_bounds__(8 * kPrepBlobs)
    k_blob_prep(const double* __restrict__ qin, int n, int nx, int ny, int nz, double h, int width,
                double* __restrict__ q, int* __restrict__ idx, double* __restrict__ w64, float* __restrict__ w32,
                int ntx, int nty, int* __restrict__ count) {
  __shared__ int4 cells[3 * kPrepBlobs];
  const int b0 = blockIdx.x * kPrepBlobs, t = threadIdx.x;
  const int g = 3 * b0 + t;  // 3 blob + axis
  if (t < 3 * kPrepBlobs && g < 3 * n) {
    const int a = t % 3;
    const int dim = a == 0 ? nx : a == 1 ? ny : nz;
    const double L = dim * h;
    double p = qin[g];
    p -= floor(p / L) * L;
    if (p >= L) p -= L;
    if (p < 0.0) p = 0.0;
    q[g] = p;
    const double u = p / h - 0.5;  // position in cell-index units (centres at integers)
    int base;
    if (width == 4)
      base = (int)floor(u) - 1;
    else
      base = (int)floor(u + 0.5) - 1;
    double w[4];
#pragma unroll
    for (int s = 0; s < 4; ++s) {
      const double r = u - (double)(base + s);
      if (width == 4)
        w[s] = phi4(r);
      else
        w[s] = (s < 3) ? phi3(r) : 0.0;
    }
    const int4 c = make_int4(pmod(base, dim), pmod(base + 1, dim), pmod(base + 2, dim), pmod(base + 3, dim));
    cells[t] = c;
    reinterpret_cast<int4*>(idx)[g] = c;
    reinterpret_cast<double2*>(w64)[2 * (size_t)g] = make_double2(w[0], w[1]);
    reinterpret_cast<double2*>(w64)[2 * (size_t)g + 1] = make_double2(w[2], w[3]);
    reinterpret_cast<float4*>(w32)[g] = make_float4((float)w[0], (float)w[1], (float)w[2], (float)w[3]);
  }
  __syncthreads();
  const int bl = t >> 3;
  if (b0 + bl < n)
    blob_tiles(cells[3 * bl], cells[3 * bl + 1], cells[3 * bl + 2], t & 7, ntx, nty,
               [&](int tile) { atomicAdd(&count[tile], 1); });
}

// Files each blob under its tiles, in any order; takes the counts back to zero.
__global__ void __launch_bounds__(256) k_tile_fill(const int* __restrict__ idx, int n, int ntx, int nty,
                                                   const int* __restrict__ offset, int* __restrict__ count,
                                                   int* __restrict__ list) {
  const int b = (int)((blockIdx.x * (size_t)blockDim.x + threadIdx.x) >> 3);
  if (b >= n) return;
  const int4* ib = reinterpret_cast<const int4*>(idx) + 3 * (size_t)b;
  blob_tiles(ib[0], ib[1], ib[2], threadIdx.x & 7, ntx, nty, [&](int tile) {
    list[offset[tile] + atomicSub(&count[tile], 1) - 1] = b;
  });
}

// offset[0..n] = exclusive scan of the tiles' counts, active = the tiles with a
// count in increasing order, meta[0] = their number; meta[1], the number of
// covered cells, starts at zero. A CTA has kScanTiles tiles, four a thread, and
// sums the counts before its own itself: 128 KB at most from L2 at 256^3, where
// waiting for its predecessors would be a chain. (One CTA that walked all tiles
// in segments took 19.8 us at 256^3; 7.0 us.)  Both scans run in one 64-bit word, active
// tiles above pairs (each below 2^31).
constexpr int kScanTiles = 4096;
__global__ void __launch_bounds__(1024) k_tile_scan(const int* __restrict__ count, int n, int* __restrict__ offset,
                                                    int* __restrict__ active, int* __restrict__ meta) {
  using u64 = unsigned long long;
  __shared__ u64 wsum[32], wbefore[32];
  const int t = threadIdx.x, lane = t & 31, w = t >> 5;
  const int base = blockIdx.x * kScanTiles;
  auto one = [](int c) { return (u64)(unsigned)c + (c > 0 ? 1ull << 32 : 0ull); };
  const int4* c4 = reinterpret_cast<const int4*>(count);
  u64 before = 0;
#pragma unroll 8
  for (int k = t; k < base / 4; k += 1024) {
    const int4 v = c4[k];
    before += (one(v.x) + one(v.y)) + (one(v.z) + one(v.w));
  }
  const int i0 = base + 4 * t;
  int4 v = make_int4(0, 0, 0, 0);
  if (i0 + 3 < n) {
    v = c4[i0 / 4];
  } else {
    if (i0 < n) v.x = count[i0];
    if (i0 + 1 < n) v.y = count[i0 + 1];
    if (i0 + 2 < n) v.z = count[i0 + 2];
  }
  const u64 sum = (one(v.x) + one(v.y)) + (one(v.z) + one(v.w));
  u64 incl = sum;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const u64 up = __shfl_up_sync(0xffffffffu, incl, o);
    if (lane >= o) incl += up;
    before += __shfl_xor_sync(0xffffffffu, before, o);
  }
  if (lane == 31) wsum[w] = incl, wbefore[w] = before;
  __syncthreads();
  if (w == 0) {
    u64 a = wsum[lane], b = wbefore[lane];
    const u64 own = a;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const u64 up = __shfl_up_sync(0xffffffffu, a, o);
      if (lane >= o) a += up;
      b += __shfl_xor_sync(0xffffffffu, b, o);
    }
    wsum[lane] = b + a - own;  // all before the warp's tiles
  }
  __syncthreads();
  const u64 ex = wsum[w] + incl - sum;
  int ra = (int)(ex >> 32);
  const int o0 = (int)(unsigned)ex, o1 = o0 + v.x, o2 = o1 + v.y, o3 = o2 + v.z;
  if (i0 + 3 < n) {
    reinterpret_cast<int4*>(offset)[i0 / 4] = make_int4(o0, o1, o2, o3);
  } else {
    if (i0 < n) offset[i0] = o0;
    if (i0 + 1 < n) offset[i0 + 1] = o1;
    if (i0 + 2 < n) offset[i0 + 2] = o2;
  }
  if (v.x > 0) active[ra++] = i0;
  if (v.y > 0) active[ra++] = i0 + 1;
  if (v.z > 0) active[ra++] = i0 + 2;
  if (v.w > 0) active[ra++] = i0 + 3;
  if (t == 1023 && blockIdx.x == gridDim.x - 1) {  // (the entries past n count nothing)
    offset[n] = o3 + v.w;
    meta[0] = ra;
    meta[1] = 0;
  }
}

// Bits of the cells start .. start + 7 of an axis of n cells that the 4 cells
// from first on (wrapping) cover.
__device__ __forceinline__ unsigned axis_mask(int first, int start, int n) {
  auto at = [](int v) { return v <= -4 || v >= kTile ? 0u : v >= 0 ? 15u << v : 15u >> -v; };
  const int lo = first - start, rem = n - start;
  return (at(lo) | at(lo - n)) & (rem < kTile ? (1u << rem) - 1u : 0xFFu);
}

// One warp per occupied tile: orders the tile's blobs by index (each finds its
// rank among the others) and lists the cells under any of them. A lane keeps two
// of the tile's 64 rows of 8 cells as bits, so a blob costs the warp one shuffle
// and a few logic instructions; the cells come out tile by tile, in order within
// a tile, at a place taken from meta[1] once per CTA (the order of the tiles
// changes no result: each cell is written once, from its own blobs).  At 4096
// blobs on 256^3 the sort (4.8 us), the count (32.7 us, a thread per cell that
// walked the blobs), the scan (6.7 us) and the fill (40.3 us) were four launches
// with the host waiting for the number of cells between them; now 9.1 us.
__global__ void __launch_bounds__(256) k_tile_cells(const int* __restrict__ active, const int* __restrict__ offset,
                                                    const int* __restrict__ raw, const int* __restrict__ idx,
                                                    int nx, int ny, int nz, int ntx, int nty,
                                                    int* __restrict__ list, int* __restrict__ meta,
                                                    int* __restrict__ cells, int* __restrict__ cell_tile) {
  __shared__ int found[8], place[8];
  const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int na = meta[0];
  if ((int)blockIdx.x * 8 >= na) return;
  const int a = blockIdx.x * 8 + w;
  unsigned rows = 0;  // rows 2 lane (low 8 bits) and 2 lane + 1 of the tile
  int tile = 0, x0 = 0, y0 = 0, z0 = 0;
  if (a < na) {
    tile = active[a];
    const int lo = offset[tile], cnt = offset[tile + 1] - lo;
    x0 = tile % ntx * kTile, y0 = tile / ntx % nty * kTile, z0 = tile / (ntx * nty) * kTile;
    const int j = 2 * (lane & 3), k = lane >> 2;
    for (int p0 = 0; p0 < cnt; p0 += 32) {
      const bool has = p0 + lane < cnt;
      const int b = has ? raw[lo + p0 + lane] : INT_MAX;
      unsigned m = 0;
      if (has) {
        const int* ib = idx + 12 * (size_t)b;
        m = axis_mask(ib[0], x0, nx) | axis_mask(ib[4], y0, ny) << 8 | axis_mask(ib[8], z0, nz) << 16;
      }
      int rank = 0;
      for (int q0 = 0; q0 < cnt; q0 += 32) {
        const int o = q0 == p0 ? b : q0 + lane < cnt ? raw[lo + q0 + lane] : INT_MAX;
        const int nq = min(32, cnt - q0);
        for (int q = 0; q < nq; ++q) rank += __shfl_sync(0xffffffffu, o, q) < b;
      }
      if (has) list[lo + rank] = b;
      const int np = min(32, cnt - p0);
      for (int q = 0; q < np; ++q) {
        const unsigned mq = __shfl_sync(0xffffffffu, m, q);
        if (mq >> (16 + k) & 1u) {
          if (mq >> (8 + j) & 1u) rows |= mq & 0xFFu;
          if (mq >> (9 + j) & 1u) rows |= (mq & 0xFFu) << 8;
        }
      }
    }
    int c = __popc(rows);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) c += __shfl_xor_sync(0xffffffffu, c, o);
    if (lane == 0) found[w] = c;
  } else if (lane == 0) {
    found[w] = 0;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    int total = 0;
    for (int u = 0; u < 8; ++u) place[u] = total, total += found[u];
    const int at = atomicAdd(&meta[1], total);
    for (int u = 0; u < 8; ++u) place[u] += at;
  }
  __syncthreads();
  if (a >= na) return;
  int at = place[w];
#pragma unroll
  for (int u = 0; u < 16; ++u) {  // 32 cells: four rows, from two lanes
    const unsigned m = __shfl_sync(0xffffffffu, rows, 2 * u) | __shfl_sync(0xffffffffu, rows, 2 * u + 1) << 16;
    if (m >> lane & 1u) {
      const int row = 4 * u + (lane >> 3);
      const int r = at + __popc(m & ((1u << lane) - 1u));
      cells[r] = ((z0 + (row >> 3)) * ny + y0 + (row & 7)) * nx + x0 + (lane & 7);
      cell_tile[r] = tile;
    }
    at += __popc(m);
  }
}

// Is cell (i, j, k) inside the support of blob b? (offsets from the blob's
// first support cell, per axis, in [0, 4))
__device__ __forceinline__ bool covers(const int* __restrict__ ib, int i, int j, int k, int nx, int ny, int nz,
                                       int& dx, int& dy, int& dz) {
  dx = i - ib[0];
  dy = j - ib[4];
  dz = k - ib[8];
  dx += dx < 0 ? nx : 0;
  dy += dy < 0 ? ny : 0;
  dz += dz < 0 ? nz : 0;
  return (unsigned)dx < 4u && (unsigned)dy < 4u && (unsigned)dz < 4u;
}

// One thread per covered cell: gathers the contributions of its tile's blobs
// in increasing blob index.
template <typename T, typename W, typename L>
__global__ void __launch_bounds__(256) k_spread(const int* __restrict__ cells, const int* __restrict__ cell_tile,
                                                int n_cells, const int* __restrict__ offset,
                                                const int* __restrict__ list, const int* __restrict__ idx,
                                                const W* __restrict__ wt, const L* __restrict__ lam,
                                                const double* __restrict__ cval, const double* __restrict__ coef,
                                                double scale, T* __restrict__ out, int nx, int ny, int nz) {
  const int t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= n_cells) return;
  const int cell = cells[t], tile = cell_tile[t];
  const int i = cell % nx, j = (cell / nx) % ny, k = cell / (nx * ny);
  W acc = 0;
  for (int p = offset[tile]; p < offset[tile + 1]; ++p) {
    const int b = list[p];
    int dx, dy, dz;
    if (covers(idx + b * 12, i, j, k, nx, ny, nz, dx, dy, dz)) {
      const W* wb = wt + b * 12;
      const double l = lam ? (double)lam[b] : *cval;
      const W amp = (W)(coef ? coef[b] * l : l);
      acc += amp * ((wb[dx] * wb[4 + dy]) * wb[8 + dz]);
    }
  }
  out[cell] += (T)scale * (T)acc;
}

// One warp per blob: lanes cover the 4x4x4 support, two cells each.
template <typename T, typename W, typename O>
__global__ void k_interp(const int* __restrict__ idx, const W* __restrict__ wt, const T* __restrict__ x,
                         double scale, O* __restrict__ out, int n, int nx, int ny) {
  const int warp = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int lane = threadIdx.x & 31;
  if (warp >= n) return;
  const int* ib = idx + warp * 12;
  const W* wb = wt + warp * 12;
  W v = 0;
#pragma unroll
  for (int t = 0; t < 2; ++t) {
    const int s = lane * 2 + t;
    const int sx = s & 3, sy = (s >> 2) & 3, sz = s >> 4;
    const size_t p = ((size_t)ib[8 + sz] * ny + ib[4 + sy]) * nx + ib[sx];
    v += (wb[sx] * wb[4 + sy]) * wb[8 + sz] * (W)x[p];
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  if (lane == 0) out[warp] = (O)(scale * (double)v);
}

}  // namespace

void blobs_setup(BlobSet& b, Dims d, double h, const double* q_in, int n, int* host, cudaStream_t s) {
  // no blobs until everything of the new set is there: an allocation that fails
  // on the way leaves a handle without blobs, whose calls read none of the arrays
  b.n = b.n_cells = 0;
  b.ntx = (d.nx + kTile - 1) / kTile;
  b.nty = (d.ny + kTile - 1) / kTile;
  b.ntz = (d.nz + kTile - 1) / kTile;
  const int nt = b.ntx * b.nty * b.ntz;
  auto room = [](int*& p, size_t entries) {
    cudaFree(p);
    p = nullptr;
    IBRD_CUDA(cudaMalloc(&p, sizeof(int) * entries));
  };
  if (b.ntiles != nt) {
    b.ntiles = 0;
    room(b.tile_count, nt);
    room(b.tile_offset, nt + 1);
    room(b.active, nt);
    b.ntiles = nt;
  }
  if (!b.d_meta) room(b.d_meta, 2);
  if (n > b.cap) {
    b.cap = 0;
    cudaFree(b.q);
    cudaFree(b.idx);
    cudaFree(b.w64);
    cudaFree(b.w32);
    b.q = nullptr;
    b.idx = nullptr;
    b.w64 = nullptr;
    b.w32 = nullptr;
    IBRD_CUDA(cudaMalloc(&b.q, sizeof(double) * 3 * n));
    IBRD_CUDA(cudaMalloc(&b.idx, sizeof(int) * 12 * n));
    IBRD_CUDA(cudaMalloc(&b.w64, sizeof(double) * 12 * n));
    IBRD_CUDA(cudaMalloc(&b.w32, sizeof(float) * 12 * n));
    b.cap = n;
  }
  if (n == 0) return;
  // The lists have room for the most that n blobs can touch, so that the host
  // need not wait for their lengths on the way.
  const size_t pairs = (size_t)n * max_axis_tiles(d.nx, b.ntx) * max_axis_tiles(d.ny, b.nty) *
                       max_axis_tiles(d.nz, b.ntz);
  const size_t most = std::min((size_t)64 * n, d.n());
  if (pairs > b.pair_cap) {
    b.pair_cap = 0;
    room(b.tile_blobs, pairs);
    room(b.tile_raw, pairs);
    b.pair_cap = pairs;
  }
  if (most > b.cell_cap) {
    b.cell_cap = 0;
    room(b.cells, most);
    room(b.cell_tile, most);
    b.cell_cap = most;
  }
  IBRD_CUDA(cudaMemsetAsync(b.tile_count, 0, sizeof(int) * nt, s));
  prof_begin(P_SETUP, s);
  k_blob_prep<<<(n + kPrepBlobs - 1) / kPrepBlobs, 8 * kPrepBlobs, 0, s>>>(
      q_in, n, d.nx, d.ny, d.nz, h, b.width, b.q, b.idx, b.w64, b.w32, b.ntx, b.nty, b.tile_count);
  prof_end(P_SETUP, s, "blob_prep");
  prof_begin(P_SETUP, s);
  k_tile_scan<<<(nt + kScanTiles - 1) / kScanTiles, 1024, 0, s>>>(b.tile_count, nt, b.tile_offset, b.active, b.d_meta);
  prof_end(P_SETUP, s, "tile_scan");
  prof_begin(P_SETUP, s);
  k_tile_fill<<<(n + 31) / 32, 256, 0, s>>>(b.idx, n, b.ntx, b.nty, b.tile_offset, b.tile_count, b.tile_raw);
  prof_end(P_SETUP, s, "tile_fill");
  const int tiles = (int)std::min(pairs, (size_t)nt);  // occupied ones, at most
  prof_begin(P_SETUP, s);
  k_tile_cells<<<(tiles + 7) / 8, 256, 0, s>>>(b.active, b.tile_offset, b.tile_raw, b.idx, d.nx, d.ny, d.nz, b.ntx,
                                               b.nty, b.tile_blobs, b.d_meta, b.cells, b.cell_tile);
  prof_end(P_SETUP, s, "tile_cells");
  IBRD_CUDA(cudaMemcpyAsync(host, b.d_meta, 2 * sizeof(int), cudaMemcpyDeviceToHost, s));
  IBRD_CUDA(cudaStreamSynchronize(s));
  b.n_cells = host[1];
  b.n = n;
}

template <typename T, typename L>
void launch_spread(const BlobSet& b, Dims d, const L* lam, const double* coef, double scale, T* out,
                   int accumulate, cudaStream_t s) {
  if (!accumulate) IBRD_CUDA(cudaMemsetAsync(out, 0, sizeof(T) * d.n(), s));
  if (b.n == 0 || b.n_cells == 0) return;
  const int c = pcls<T>(P_SPREAD64, P_SPREAD32);
  const int blocks = (b.n_cells + 255) / 256;
  prof_begin(c, s);
  if (sizeof(T) == 8)
    k_spread<T, double, L><<<blocks, 256, 0, s>>>(b.cells, b.cell_tile, b.n_cells, b.tile_offset, b.tile_blobs,
                                                  b.idx, b.w64, lam, nullptr, coef, scale, out, d.nx, d.ny, d.nz);
  else
    k_spread<T, float, L><<<blocks, 256, 0, s>>>(b.cells, b.cell_tile, b.n_cells, b.tile_offset, b.tile_blobs,
                                                 b.idx, b.w32, lam, nullptr, coef, scale, out, d.nx, d.ny, d.nz);
  prof_end(c, s, "spread", (double)b.n_cells * (2.0 * sizeof(T) + 8.0) + (double)b.n * (48.0 + 12.0 * sizeof(T) + 16.0));
}

template <typename T>
void launch_spread_const(const BlobSet& b, Dims d, const double* cval, double scale, T* out, cudaStream_t s) {
  if (b.n == 0 || b.n_cells == 0) return;
  const int c = pcls<T>(P_SPREAD64, P_SPREAD32);
  const int blocks = (b.n_cells + 255) / 256;
  prof_begin(c, s);
  if (sizeof(T) == 8)
    k_spread<T, double, double><<<blocks, 256, 0, s>>>(b.cells, b.cell_tile, b.n_cells, b.tile_offset,
                                                       b.tile_blobs, b.idx, b.w64, nullptr, cval, nullptr, scale,
                                                       out, d.nx, d.ny, d.nz);
  else
    k_spread<T, float, double><<<blocks, 256, 0, s>>>(b.cells, b.cell_tile, b.n_cells, b.tile_offset,
                                                      b.tile_blobs, b.idx, b.w32, nullptr, cval, nullptr, scale,
                                                      out, d.nx, d.ny, d.nz);
  prof_end(c, s, "spread_const", (double)b.n_cells * (2.0 * sizeof(T) + 8.0) + (double)b.n * (48.0 + 12.0 * sizeof(T)));
}

template <typename T, typename O>
void launch_interp(const BlobSet& b, Dims d, const T* x, double scale, O* out, cudaStream_t s) {
  if (b.n == 0) return;
  const int threads = 256;
  const int blocks = (int)(((size_t)b.n * 32 + threads - 1) / threads);
  const int c = pcls<T>(P_INTERP64, P_INTERP32);
  prof_begin(c, s);
  if (sizeof(T) == 8)
    k_interp<T, double, O><<<blocks, threads, 0, s>>>(b.idx, b.w64, x, scale, out, b.n, d.nx, d.ny);
  else
    k_interp<T, float, O><<<blocks, threads, 0, s>>>(b.idx, b.w32, x, scale, out, b.n, d.nx, d.ny);
  prof_end(c, s, "interp", (double)b.n * (64.0 * sizeof(T) + 48.0 + 12.0 * sizeof(T) + 8.0));
}

template void launch_spread<double, double>(const BlobSet&, Dims, const double*, const double*, double, double*,
                                            int, cudaStream_t);
template void launch_spread<float, double>(const BlobSet&, Dims, const double*, const double*, double, float*, int,
                                           cudaStream_t);
template void launch_spread<float, float>(const BlobSet&, Dims, const float*, const double*, double, float*, int,
                                          cudaStream_t);
template void launch_spread_const<double>(const BlobSet&, Dims, const double*, double, double*, cudaStream_t);
template void launch_spread_const<float>(const BlobSet&, Dims, const double*, double, float*, cudaStream_t);
template void launch_interp<double, double>(const BlobSet&, Dims, const double*, double, double*, cudaStream_t);
template void launch_interp<float, double>(const BlobSet&, Dims, const float*, double, double*, cudaStream_t);
template void launch_interp<float, float>(const BlobSet&, Dims, const float*, double, float*, cudaStream_t);

}  // namespace ibrd
