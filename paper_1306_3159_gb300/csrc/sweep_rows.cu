// Row-resident red-black Gauss-Seidel kernels for FP32 levels (Sec. III.E: the
// multigrid smoother of the Helmholtz problem A = alpha I - chi L): the sweep
// (with the prolongation of the coarse correction fused in, after a coarse
// solve) and the first sweep from zero with the residual restriction.
//
// One full sweep (red cells from the old black values, then black cells from
// the new red values; red = (i + j + k) even) in one pass over memory.
//
// Only the black values of the old x enter a sweep, and after a sweep the
// residual of every black cell is zero, so between the two half-cycles of a
// V-cycle a level keeps only its black cells: a packed field of nx / 2 values
// per row. In a row of parity a = (j + k) & 1 the red cells are i = 2 m + a
// and the black ones i = 2 m + 1 - a, m = 0 .. nx / 2 - 1. In packed rows the
// six neighbours of entry m of one colour are, of the other colour,
//   y and z: entry m of the adjacent rows and planes,
//   x: entries m - 1, m where the neighbours' parity makes them lie to the
//   left (nbr_sums with right = 0), m, m + 1 where to the right (right = 1);
//   for a red cell right = a, for a black one right = 1 - a.
// The x-pair (2 m, 2 m + 1) of a coarse cell holds one red cell, entry m, so
// the restricted residual is off / 8 times the sum over the coarse cell's four
// rows of the red entries' neighbour sums (the first sweep from zero leaves
// b - diag x = 0 in its red cells), and the correction of a packed row needs
// one interpolated value per coarse cell.
//
// * A warp owns x-rows: lane l holds the 4-cell groups l + 32 s (s < NS) of its
//   row, two packed entries each. x-neighbours come from the neighbouring
//   lanes by shuffles; the periodic wrap of rows of 128 NS cells is the shuffle
//   from lane 31 to lane 0. Rows of other lengths (multiples of 32) leave lanes
//   idle and take one more shuffle for the wrap; rows above 256 cells belong to
//   two warps, whose outermost groups read their neighbour from the published
//   row in shared memory. FP32 V-cycles of one pre- and one post-sweep, which
//   run the sweep from zero and the packed sweep below, against ones of the tiled sweep
//   and separate transfers: 73 and 88 us at 96^3, 117 and 151 at 160^3, 157 and 222 at
//   224^3, 361 and 446 at 320^3, 537 and 1330 at 512^3 (the largest cube a CTA's shared
//   memory holds rows of). Which levels take which form: zero_restrict_rows_ok,
//   rows_plain_ok, rows_prolong_full_ok.
// * A CTA owns TY rows of every plane of a z-chunk, plus one halo row on each
//   side in y whose red cells it also updates (the black cells at the tile's
//   edge rows need them); the neighbouring CTA computes the same red values
//   from the same old data, bit for bit.
// * Planes arrive by TMA: one thread issues tensor-map box copies (the tile's
//   rows plus 2-row halos of x, 1-row halos of b) into a ring of stages, one
//   mbarrier per stage. The periodic wrap in y is the halo boxes' start row,
//   taken modulo ny on the host side of the index (every box starts at x = 0,
//   so the 16-byte rule on the innermost coordinate holds; nx is a multiple of
//   32, which keeps the boxes' shared-memory addresses on 128 bytes).
// * Each thread keeps its row's neighbouring planes in registers (the
//   z-neighbours); every row is published once in shared memory, packed and
//   double-buffered, for the y-neighbours of the next step, so no row is read
//   while it is written and one barrier per plane suffices; thread 0 alone
//   waits on the TMA barriers, one stage ahead.
// * Odd z-chunks march downwards, so that adjacent chunks meet at their
//   common halo planes at the same time (L2 hits, not DRAM re-reads).
//
// What bounds them: the time of one step, that is the instructions of 22 warps
// per SM (issue slots 40 % busy) and the shared-memory round trips between two
// barriers. Three things set it, measured at 256^3 (ncu): the marches are
// compiled for each parity of a row, so that choosing the red or the black half
// of a group costs nothing (14.0 M warp instructions instead of 22.2 M); pairs
// of cells are computed by the two-wide FP32 instructions; and a plane comes in
// as few copies as possible, issued by a warp of its own (with nine copies per
// plane from one of the marching threads every CTA took 40 us, with three 31
// us). Sweep with the prolongation: 34 us for 176 MB (0.77 of the copy
// bandwidth), 51 us for 210 MB when x was a full field. Sweep from zero and
// restriction: 24 us for 109 MB (0.67), 36 us for 143 MB before. At 128^3: 12.6
// and 8.7 us (13.8 and 10.0).
//
// Every mbarrier wait is bounded: a wait that gives up sets *err, drains the
// copies still in flight (again with a bound) and ends the CTA; the host
// turns the flag into IBRD_ERR_TIMEOUT.
#include <cuda.h>
#include <cudaTypedefs.h>

#include <algorithm>
#include <cstring>
#include <mutex>
#include <type_traits>

#include "internal.h"

namespace ibrd {
namespace {

constexpr int kRowsTY = 8;      // tile rows per CTA
constexpr int kSweepRing = 3;   // TMA stages of the sweep (one plane of x and of b each)
constexpr int kZeroRing = 4;    // TMA stages of the sweep from zero (one plane of b each)
constexpr int kCoarseRing = 3;  // coarse planes in the ring of the fused prolongation
constexpr unsigned kDrainLimit = 1u << 26;

__device__ __forceinline__ unsigned smem_u32(const void* p) { return (unsigned)__cvta_generic_to_shared(p); }

__device__ __forceinline__ void mbar_init(unsigned bar, unsigned count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;\n" ::"r"(bar), "r"(count) : "memory");
}
// One lane of the calling (whole) warp: the feeding warp runs its loop in all
// lanes, with uniform addresses, and only the copies themselves are predicated.
__device__ __forceinline__ unsigned elect_lane() {
  unsigned r;
  asm volatile("{\n .reg .pred p;\n elect.sync _|p, 0xffffffff;\n selp.u32 %0, 1, 0, p;\n}\n" : "=r"(r));
  return r;
}
__device__ __forceinline__ void mbar_expect_tx(unsigned bar, unsigned bytes, unsigned lead) {
  asm volatile(
      "{\n .reg .pred p;\n setp.ne.u32 p, %2, 0;\n @p mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;\n}\n" ::"r"(
          bar),
      "r"(bytes), "r"(lead)
      : "memory");
}
// true when the phase with this parity completed within `limit` tries
__device__ __forceinline__ bool mbar_wait(unsigned bar, unsigned parity, unsigned limit) {
  for (unsigned i = 0; i < limit; ++i) {
    unsigned ok;
    asm volatile(
        "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}\n"
        : "=r"(ok)
        : "r"(bar), "r"(parity)
        : "memory");
    if (ok) return true;
  }
  return false;
}
__device__ __forceinline__ void tma_load4(unsigned dst, const CUtensorMap* map, int y, int z, unsigned bar,
                                          unsigned lead) {
  asm volatile(
      "{\n .reg .pred p;\n setp.ne.u32 p, %6, 0;\n"
      " @p cp.async.bulk.tensor.4d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %2, %3, %4}], "
      "[%5];\n}\n" ::"r"(dst),
      "l"(reinterpret_cast<unsigned long long>(map)), "r"(0), "r"(y), "r"(z), "r"(bar), "r"(lead)
      : "memory");
}

// CTA barriers that different warps may reach at different instructions (each
// warp runs its own copy of the march), and one that also ORs a flag.
__device__ __forceinline__ void cta_sync() { asm volatile("barrier.cta.sync.aligned 0;\n" ::: "memory"); }
__device__ __forceinline__ bool cta_sync_or(bool flag) {
  unsigned r;
  asm volatile(
      "{\n .reg .pred p, q;\n setp.ne.u32 p, %1, 0;\n barrier.cta.red.or.pred.aligned q, 0, p;\n"
      " selp.u32 %0, 1, 0, q;\n}\n"
      : "=r"(r)
      : "r"((unsigned)flag)
      : "memory");
  return r != 0;
}

// Tensor maps of a field: boxes of the tile's rows with their halos on both
// sides, with one halo (of the bare rows where the domain is one tile), and of
// one halo.
struct RowMaps {
  CUtensorMap all, part, halo;
};

// Rows y0 - HALO .. y0 + ROWS + HALO - 1 (periodic in ny) of plane z into dst
// (rows of nx values). As few copies as the periodic wrap allows (each costs
// the issuing warp about 90 cycles, and three or six of them per plane decide
// the pace of a march): one box inside the domain, two at one edge of it, three
// when the domain is one tile (with one-halo boxes alone, 16 a plane, a packed sweep
// of 8 x 8 rows took 8.2 us at 128 cells and 11.6 at 320; now 5.9 and 9.4).
template <int ROWS, int HALO>
__device__ __forceinline__ void load_rows(float* dst, int nx, const RowMaps& m, int y0, int ny, int z, unsigned bar,
                                          unsigned lead) {
  const bool low = y0 >= HALO, high = y0 + ROWS + HALO <= ny;
  if (low && high) {
    tma_load4(smem_u32(dst), &m.all, y0 - HALO, z, bar, lead);
  } else if (low) {
    tma_load4(smem_u32(dst), &m.part, y0 - HALO, z, bar, lead);
    tma_load4(smem_u32(dst + (ROWS + HALO) * nx), &m.halo, 0, z, bar, lead);
  } else if (high) {
    tma_load4(smem_u32(dst), &m.halo, ny - HALO, z, bar, lead);
    tma_load4(smem_u32(dst + HALO * nx), &m.part, y0, z, bar, lead);
  } else {
    tma_load4(smem_u32(dst), &m.halo, ny - HALO, z, bar, lead);
    tma_load4(smem_u32(dst + HALO * nx), &m.part, 0, z, bar, lead);
    tma_load4(smem_u32(dst + (ROWS + HALO) * nx), &m.halo, 0, z, bar, lead);
  }
}

// A CTA's warps: WPR for each of the tile's rows and its two halo rows, and one
// that feeds them.
template <int WPR>
constexpr int kRowsThreads = ((kRowsTY + 2) * WPR + 1) * 32;

// The feeding warp of a march over planes 0 .. last: it issues the
// stages' copies (up to `first` before the march, up to i + ahead at step i, when
// the ring slot they take is free) and polls their barriers, stage i + 1 in step
// i; the CTA barrier that ends every step publishes the landed stage. When a
// wait gives up it issues and waits no more (dead), drains the copies in flight
// and sets *err; the CTA learns of it at every sixth step and stops, what it
// wrote since being invalid. The barriers pair with those of the marching warps.
template <typename Issue, typename Wait>
__device__ __forceinline__ void feed_stages(int last, int first, int ahead, Issue&& issue, Wait&& wait_stage,
                                            unsigned limit, int* err) {
  const unsigned lead = elect_lane();
  bool dead = false;
  int issued = -2, landed = -2;
  auto feed = [&](int upto_issue, int upto_wait) {
    if (dead) return;
    while (issued < min(upto_issue, last - 1)) issue(++issued, lead);
    while (!dead && landed < min(upto_wait, last - 1)) {
      if (__all_sync(0xffffffffu, wait_stage(landed + 1, limit)))
        ++landed;
      else
        dead = true;
    }
  };
  bool ok = true;
  for (int i = -1; ok && i < last; ++i) {
    // i = -1: the stages the march starts from; i = 0: they have been read
    if (i) feed(i < 0 ? first : i + ahead, i < 0 ? 1 : i + 1);
    __syncwarp();
    if (i < 0 || (i > 0 && i % 6 == 0))
      ok = !cta_sync_or(dead);
    else
      cta_sync();
  }
  if (dead) {
    while (landed < issued) wait_stage(++landed, kDrainLimit);
    if (lead) atomicOr(err, 1);
  }
}

// Two FP32 operations in one instruction, each rounded as the scalar one is:
// the kernels below are bound by the instructions they issue, and their cells
// come in pairs.
__device__ __forceinline__ unsigned long long bits2(float2 a) {
  return ((unsigned long long)__float_as_uint(a.y) << 32) | __float_as_uint(a.x);
}
__device__ __forceinline__ float2 pair2(unsigned long long a) {
  return make_float2(__uint_as_float((unsigned)a), __uint_as_float((unsigned)(a >> 32)));
}
__device__ __forceinline__ float2 dup2(float a) { return make_float2(a, a); }
__device__ __forceinline__ float2 add2(float2 a, float2 b) {
  unsigned long long r;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(bits2(a)), "l"(bits2(b)));
  return pair2(r);
}
__device__ __forceinline__ float2 mul2(float2 a, float2 b) {
  unsigned long long r;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(bits2(a)), "l"(bits2(b)));
  return pair2(r);
}
__device__ __forceinline__ float2 fma2(float2 a, float2 b, float2 c) {
  unsigned long long r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(bits2(a)), "l"(bits2(b)), "l"(bits2(c)));
  return pair2(r);
}
// prolong_axis and prolong_add on pairs
__device__ __forceinline__ float2 prolong_axis2(float2 n, float2 f) { return fma2(dup2(3.f), n, f); }
__device__ __forceinline__ float2 prolong_add2(float2 x, float2 t64) { return fma2(dup2(0x1p-6f), t64, x); }

// Rows as a kernel sees them. NXT: the row length fixed at compile time (0: taken at
// run time); WPR: warps per row; NS: groups per lane.
template <int NS, int WPR, int NXT>
struct Row {
  static constexpr bool kWrap = NXT == 128 * NS && WPR == 1;  // one full warp holds the whole row
  int nx, lane, g0, gw;  // row length; the warp's first group and its number of groups (at most 32 in all slots but the last)
  __device__ __forceinline__ Row(int nx_, int warp_in_row) {
    nx = NXT ? NXT : nx_;
    lane = threadIdx.x & 31;
    gw = nx / (4 * WPR);
    g0 = WPR == 1 ? 0 : warp_in_row * gw;
  }
  __device__ __forceinline__ bool valid(int s) const { return kWrap || s < NS - 1 || lane + 32 * s < gw; }
  // group of slot s (an idle lane reads the warp's last one)
  __device__ __forceinline__ int group(int s) const {
    if constexpr (kWrap) return lane + 32 * s;
    const int q = lane + 32 * s;
    return g0 + (s < NS - 1 || q < gw ? q : gw - 1);
  }
  __device__ __forceinline__ int last_lane() const { return (gw - 1) & 31; }  // of the warp's last group, in the last slot
};

// The packed pairs v moved by one entry: w = the entries m - 1 or, with right,
// m + 1 of each pair's entries m. Inside a row they are the adjacent lane's, or
// at lane 0 / 31 the adjacent slot's. Beyond the warp's ends: of a row that is
// one warp's, the row's other end (the next shuffle target where the row fills
// the lanes, one more shuffle where it does not); of a row of two warps, edge(m).
template <int NS, int WPR, int NXT, typename F>
__device__ __forceinline__ void shifted(float2 (&w)[NS], const float2 (&v)[NS], bool right,
                                        const Row<NS, WPR, NXT>& r, F&& edge) {
  static_assert(NS <= 2, "the adjacent slot on either side is the other one");
  constexpr bool kWrap = Row<NS, WPR, NXT>::kWrap;
  const int src = (right ? r.lane + 1 : r.lane + 31) & 31;
  float t[NS], e = 0.f;
#pragma unroll
  for (int s = 0; s < NS; ++s) t[s] = __shfl_sync(0xffffffffu, right ? v[s].x : v[s].y, src);
  if constexpr (!kWrap && WPR == 1) e = __shfl_sync(0xffffffffu, right ? v[0].x : v[NS - 1].y, right ? 0 : r.last_lane());
  if constexpr (!kWrap && WPR > 1) {
    const int half = r.nx >> 1, m = right ? 2 * (r.g0 + r.gw) : 2 * r.g0 - 1;
    e = edge(m < 0 ? m + half : (m >= half ? m - half : m));
  }
#pragma unroll
  for (int s = 0; s < NS; ++s) {
    float o = t[s];
    if (NS == 2 && (kWrap || s == (right ? 0 : 1)) && r.lane == (right ? 31 : 0)) o = t[NS - 1 - s];
    if (!kWrap && s == (right ? NS - 1 : 0) && r.lane == (right ? r.last_lane() : 0)) o = e;
    w[s] = right ? make_float2(v[s].y, o) : make_float2(o, v[s].x);
  }
}

// Per entry of the packed pairs v the sum of its two x-neighbours among the
// entries of the same packed row: (m - 1, m) or, with right, (m, m + 1). `row`
// is the published copy of that row.
template <int NS, int WPR, int NXT>
__device__ __forceinline__ void nbr_sums(float2 (&n)[NS], const float2 (&v)[NS], const float* row, bool right,
                                         const Row<NS, WPR, NXT>& r) {
  shifted<NS, WPR, NXT>(n, v, right, r, [&](int m) { return row[m]; });
#pragma unroll
  for (int s = 0; s < NS; ++s) n[s] = add2(v[s], n[s]);
}

// The correction of a packed row: v += (P xc) at its black cells (Sec. III.E,
// cell-centred trilinear prolongation) in the order every prolongation kernel
// uses: z between the row's parent coarse plane cp and the other plane co, then
// y between the parent coarse row cr and its neighbour nr on the row's side
// (coarse rows of nx / 2 floats), then x towards coarse cell m + 1 (right: the
// black cell is the odd one of its pair) or m - 1.
template <int NS, int WPR, int NXT>
__device__ __forceinline__ void add_correction(float2 (&v)[NS], const float* cp, const float* co, int cr, int nr,
                                               bool right, const Row<NS, WPR, NXT>& r) {
  const int nxc = r.nx >> 1;
  const float *pp = cp + cr * nxc, *op = co + cr * nxc, *pn = cp + nr * nxc, *on = co + nr * nxc;
  float2 zy[NS], f[NS];  // the pair after z and y (16 times its value), and its neighbours
#pragma unroll
  for (int s = 0; s < NS; ++s) {
    const int o = 2 * r.group(s);
    const float2 a = *reinterpret_cast<const float2*>(pp + o), b = *reinterpret_cast<const float2*>(op + o);
    const float2 c = *reinterpret_cast<const float2*>(pn + o), d = *reinterpret_cast<const float2*>(on + o);
    zy[s] = prolong_axis2(prolong_axis2(a, b), prolong_axis2(c, d));
  }
  shifted<NS, WPR, NXT>(f, zy, right, r, [&](int m) {
    return prolong_axis(prolong_axis(pp[m], op[m]), prolong_axis(pn[m], on[m]));
  });
#pragma unroll
  for (int s = 0; s < NS; ++s) v[s] = prolong_add2(v[s], prolong_axis2(zy[s], f[s]));
}

// What a sweep reads as the old x.
enum SweepIn {
  IN_FULL = 0,      // a full field
  IN_FULL_PRO = 1,  // a full field plus the prolongation of a coarse field
  IN_PACKED_PRO = 2 // a packed field of black cells plus the prolongation of a coarse field
};

// Shared memory (floats): x ring, b ring, two published planes of corrected
// black rows y0-2 .. y0+TY+1, two planes of red rows y0-1 .. y0+TY, coarse ring.
__host__ __device__ constexpr size_t sweep_rows_floats(int nx, int in) {
  return (size_t)kSweepRing * (kRowsTY + 4) * (in == IN_PACKED_PRO ? nx / 2 : nx) +
         (size_t)kSweepRing * (kRowsTY + 2) * nx + (size_t)(kRowsTY + 4) * nx + (size_t)(kRowsTY + 2) * nx +
         (in == IN_FULL ? 0 : (size_t)kCoarseRing * (kRowsTY / 2 + 4) * (nx / 2));
}

// Grid: (ny / TY, z-chunks). Block: (TY + 2) rows of WPR warps; row w is
// y0 - 1 + w (w = 0 and w = TY + 1 are the halo rows: red cells only; they
// also publish the outer rows y0 - 2 and y0 + TY + 1).
//
// March order: chunk c covers planes [k0, k1) and visits planes k0-2 .. k1+1
// upwards when c is even and k1+1 .. k0-2 downwards when c is odd, so that
// neighbouring chunks start (or end) at their common boundary at the same
// time and the halo planes they share come from L2. The Gauss-Seidel result
// does not depend on the order in which the cells of one colour are updated,
// so both directions give the same sweep. March index i = 0 .. zc + 3 names
// plane mp(i). Step i reads stage i (x of plane i + 1, b of plane i), publishes
// the black cells of plane i + 1, updates the red cells of plane i and the
// black cells of plane i - 1 (when that plane is in the chunk) and stores
// plane i - 1.
//
// With the prolongation fused the x values are corrected as they are read. The
// coarse planes arrive by TMA into a ring of kCoarseRing slots of TY / 2 + 4
// coarse rows (the parents of the tile's rows and their neighbours), riding
// on the stages. Fine planes 2K - 1 and 2K share the coarse pair {K - 1, K}, so
// every second stage brings a new coarse plane (coarse march plane j = i / 2 + 2
// first serves the correction of fine march plane i + 1, i even). Chunks hold
// an even number of planes so that the pairing is the same in both march
// directions.
template <int NS, int WPR, int NXT, int IN>
__global__ void __launch_bounds__(kRowsThreads<WPR>, WPR == 1 ? 2 : 1)
    k_rbgs_rows(const __grid_constant__ RowMaps mx, const __grid_constant__ RowMaps mb,
                const __grid_constant__ RowMaps mc, float* __restrict__ xout, const double* __restrict__ bshift,
                int nx_, int ny, int nz, int zc, float inv, float off, double* __restrict__ part,
                int* __restrict__ err, unsigned wait_limit) {
  constexpr int TY = kRowsTY, R = kSweepRing;
  constexpr bool PRO = IN != IN_FULL, PIN = IN == IN_PACKED_PRO;
  constexpr int XROWS = TY + 4, BROWS = TY + 2, CROWS = TY / 2 + 4;
  const int tid = threadIdx.x, warp = __shfl_sync(0xffffffffu, tid >> 5, 0), w = warp / WPR;
  const Row<NS, WPR, NXT> row(nx_, warp % WPR);
  const int nx = row.nx, nxp = nx >> 1, nxr = PIN ? nxp : nx;  // nxr: row length of the x ring
  extern __shared__ __align__(1024) unsigned char sm_raw[];
  float* XS = reinterpret_cast<float*>(sm_raw);
  float* BS = XS + R * XROWS * nxr;
  float* CP = BS + R * BROWS * nx;
  float* RS = CP + 2 * XROWS * nxp;
  float* CS = RS + 2 * BROWS * nxp;
  unsigned long long* bars = reinterpret_cast<unsigned long long*>(CS + (PRO ? kCoarseRing * CROWS * nxp : 0));

  const int y0 = blockIdx.x * TY;
  const int k0 = blockIdx.y * zc, k1 = min(k0 + zc, nz);
  const bool down = blockIdx.y & 1;
  const float2 msh = dup2(bshift ? -(float)(*bshift) : -0.f), off2 = dup2(off), inv2 = dup2(inv);
  const bool interior = w >= 1 && w <= TY;
  const int last = k1 - k0 + 3;  // march index of the last plane
  auto mp = [&](int i) { return down ? k1 + 1 - i : k0 - 2 + i; };
  auto cmp = [&](int j) { return down ? (k1 >> 1) + 1 - j : (k0 >> 1) - 2 + j; };  // coarse march plane j
  // parity of this warp's row in march plane 1 (ny is even, so the wrap keeps it)
  const bool a1 = (y0 - 1 + w + mp(1)) & 1;
  // coarse rows of this warp's own row: its parent and the parent's neighbour
  const int cr = ((w + 1) >> 1) + 1, nr = (w & 1) ? cr - 1 : cr + 1;

  if (tid == 0) {
    for (int s = 0; s < R; ++s) mbar_init(smem_u32(bars + s), 1);
    asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
  }
  cta_sync();

  // Copies of stage i = -1 .. last - 1 (slot (i + 1) % R): x of march plane
  // i + 1 (rows y0-2 .. y0+TY+1), for i >= 1 b of march plane i (rows y0-1 ..
  // y0+TY), with PRO the coarse march planes 0 and 1 (i = -1) or i / 2 + 2 (even
  // i >= 0; coarse rows y0/2 - 2 .. y0/2 + TY/2 + 1). Planes lie in [-2, nz + 1],
  // coarse ones in [-2, nz / 2 + 1]: one compare wraps them.
  auto wrapz = [](int z, int n) { return z < 0 ? z + n : (z >= n ? z - n : z); };
  auto issue_coarse = [&](int j, unsigned bar, unsigned lead) {
    load_rows<TY / 2, 2>(CS + (j % kCoarseRing) * CROWS * nxp, nxp, mc, y0 >> 1, ny >> 1, wrapz(cmp(j), nz >> 1), bar,
                         lead);
  };
  auto issue = [&](int i, unsigned lead) {
    const unsigned xbytes = XROWS * nxr * 4, bbytes = BROWS * nx * 4, cbytes = CROWS * nxp * 4;
    const int s = (i + 1) % R;
    const unsigned bar = smem_u32(bars + s);
    const bool even = i >= 0 && !(i & 1);
    mbar_expect_tx(bar, xbytes + (i >= 1 ? bbytes : 0u) + (PRO ? (i < 0 ? 2u : (even ? 1u : 0u)) * cbytes : 0u), lead);
    load_rows<TY, 2>(XS + s * XROWS * nxr, nxr, mx, y0, ny, wrapz(mp(i + 1), nz), bar, lead);
    if (i >= 1) load_rows<TY, 1>(BS + s * BROWS * nx, nx, mb, y0, ny, wrapz(mp(i), nz), bar, lead);
    if constexpr (PRO) {
      if (i < 0) {
        issue_coarse(0, bar, lead);
        issue_coarse(1, bar, lead);
      } else if (even) {
        issue_coarse((i >> 1) + 2, bar, lead);
      }
    }
  };
  auto wait_stage = [&](int i, unsigned limit) {
    return mbar_wait(smem_u32(bars + (i + 1) % R), (unsigned)(((i + 1) / R) & 1), limit);
  };
  // rows of the published planes (by the march plane's parity), a coarse plane by its ring slot
  auto cprow = [&](int par, int r) { return CP + (par * XROWS + r) * nxp; };
  auto rsrow = [&](int par, int r) { return RS + (par * BROWS + r) * nxp; };
  auto cslot = [&](int s) -> const float* { return CS + s * CROWS * nxp; };
  // the old black values of row r (0 .. TY + 3) in ring slot `slot`, uncorrected; right: its black cells are the odd ones
  auto load_black = [&](float2 (&v)[NS], int slot, int r, bool right) {
    const float* p = XS + (slot * XROWS + r) * nxr;
#pragma unroll
    for (int s = 0; s < NS; ++s) {
      if constexpr (PIN) {
        v[s] = *reinterpret_cast<const float2*>(p + 2 * row.group(s));
      } else {
        const float4 q = *reinterpret_cast<const float4*>(p + 4 * row.group(s));
        v[s] = right ? make_float2(q.y, q.w) : make_float2(q.x, q.z);
      }
    }
  };
  auto put_row = [&](float* p, const float2 (&v)[NS]) {
#pragma unroll
    for (int s = 0; s < NS; ++s)
      if (row.valid(s)) *reinterpret_cast<float2*>(p + 2 * row.group(s)) = v[s];
  };
  auto get_row = [&](float2 (&v)[NS], const float* p) {
#pragma unroll
    for (int s = 0; s < NS; ++s) v[s] = *reinterpret_cast<const float2*>(p + 2 * row.group(s));
  };
  // the plane in ring slot `slot` (its march index's parity par; right: this
  // row's black cells are the odd ones) into v (this warp's row) and into the
  // published rows; jp / jo: the ring slots of its parent and other coarse planes
  auto take_plane = [&](float2 (&v)[NS], bool right, int slot, int par, int jp, int jo) {
    load_black(v, slot, w + 1, right);
    if constexpr (PRO) add_correction<NS, WPR, NXT>(v, cslot(jp), cslot(jo), cr, nr, right, row);
    put_row(cprow(par, w + 1), v);
    if (!interior) {  // the outer row next to this halo row
      const bool top = w == 0;
      float2 o[NS];
      load_black(o, slot, top ? 0 : TY + 3, !right);
      if constexpr (PRO)
        add_correction<NS, WPR, NXT>(o, cslot(jp), cslot(jo), top ? 1 : CROWS - 2, top ? 0 : CROWS - 1, !right, row);
      put_row(cprow(par, top ? 0 : TY + 3), o);
    }
  };

  bool ok = true;
  float acc = 0.f, comp = 0.f;  // Kahan sum of the new x (tile rows)
  // where the black cells' step stores this row of plane mp(2), mp(3), ...
  const ptrdiff_t plane = (ptrdiff_t)nx * ny;
  float* dst = xout + (ptrdiff_t)mp(2) * plane + (ptrdiff_t)(y0 - 1 + w) * nx;
  const ptrdiff_t dstep = down ? -plane : plane;
  // a warp's march, compiled for each parity of its row in march plane 1
  auto march = [&](auto first_parity) {
    constexpr bool A1 = decltype(first_parity)::value;
    // old black cells of three planes, new red cells of three, b of the black cells of two
    float2 C0[NS], C1[NS], C2[NS], R0[NS], R1[NS], R2[NS], B0[NS], B1[NS];
    ok = !cta_sync_or(false);  // stages -1, 0 and 1 have landed
    if (!ok) return;
    // march planes 0 and 1 have the parent coarse plane 1; the other plane is
    // 0 for plane 0 and 2 for plane 1
    take_plane(C0, A1, 0, 0, 1, 0);
    take_plane(C1, !A1, 1, 1, 1, 2);
    cta_sync();  // the slots of stages -1 and 0 are free

    // Step i: cm, c0, cp = old black cells of march planes i - 1, i, i + 1 (cp is read here); rm2, rm1, r0 = new red
    // cells of planes i - 2, i - 1, i (r0 is formed here); bm1 / b0 = b of the black cells of planes i - 1 / i.
    auto step = [&](float2 (&cm)[NS], float2 (&c0)[NS], float2 (&cp)[NS], float2 (&rm2)[NS], float2 (&rm1)[NS],
                    float2 (&r0)[NS], float2 (&bm1)[NS], float2 (&b0)[NS], int i, auto phase) {
      // i = 1 + phase (mod 6): ring slots and parities are constants
      constexpr int PH = decltype(phase)::value, P0 = (PH + 1) & 1, P1 = PH & 1, S1 = (PH + 2) % R;
      constexpr bool a = A1 != (bool)(PH & 1);  // plane i: red cells at 2 m + a
      static_assert(R == 3 && kCoarseRing == 3, "the unrolling by 6 fixes the slots");
      // coarse planes of plane i + 1: odd i keeps the pair of step i - 1, whose
      // newer plane is the parent; even i brings coarse plane i / 2 + 2 (the
      // other) and the parent is the plane before it
      constexpr int JP = P0 ? (PH / 2 + 2) % 3 : ((PH + 1) / 2 + 1) % 3, JO = (JP + (P0 ? 2 : 1)) % 3;
      take_plane(cp, a, S1, P1, JP, JO);
      float2 br[NS], n[NS], u[NS], d[NS];
      const float* bp = BS + (S1 * BROWS + w) * nx;
#pragma unroll
      for (int s = 0; s < NS; ++s) {
        const float4 t = *reinterpret_cast<const float4*>(bp + 4 * row.group(s));
        br[s] = add2(a ? make_float2(t.y, t.w) : make_float2(t.x, t.z), msh);
        b0[s] = add2(a ? make_float2(t.x, t.z) : make_float2(t.y, t.w), msh);
      }
      // red cells of plane i from the old black cells around them
      nbr_sums<NS, WPR, NXT>(n, c0, cprow(P0, w + 1), a, row);
      get_row(u, cprow(P0, w));
      get_row(d, cprow(P0, w + 2));
#pragma unroll
      for (int s = 0; s < NS; ++s)
        r0[s] = mul2(fma2(off2, add2(add2(n[s], add2(u[s], d[s])), add2(cm[s], cp[s])), br[s]), inv2);
      put_row(rsrow(P0, w), r0);
      if (interior && i >= 3) {
        // black cells of plane i - 1 (there at 2 m + a) from the new red cells around them
        float2 k[NS];
        nbr_sums<NS, WPR, NXT>(n, rm1, rsrow(P1, w), a, row);
        get_row(u, rsrow(P1, w - 1));
        get_row(d, rsrow(P1, w + 1));
        float t = 0.f;
#pragma unroll
        for (int s = 0; s < NS; ++s) {
          k[s] = mul2(fma2(off2, add2(add2(n[s], add2(u[s], d[s])), add2(rm2[s], r0[s])), bm1[s]), inv2);
          if (row.valid(s)) {
            *reinterpret_cast<float4*>(dst + 4 * row.group(s)) =
                a ? make_float4(rm1[s].x, k[s].x, rm1[s].y, k[s].y) : make_float4(k[s].x, rm1[s].x, k[s].y, rm1[s].y);
            t += (rm1[s].x + rm1[s].y) + (k[s].x + k[s].y);
          }
        }
        dst += dstep;
        if (part) {
          const float yk = t - comp, tk = acc + yk;
          comp = (tk - acc) - yk;
          acc = tk;
        }
      }
      if constexpr (PH == 5)
        ok = !cta_sync_or(false);
      else
        cta_sync();
    };
#define IBRD_STEP(c0, c1, c2, r0, r1, r2, b0, b1, ph) \
  if (i + ph >= last) return;                         \
  step(c0, c1, c2, r0, r1, r2, b0, b1, i + ph, std::integral_constant<int, ph>{});
    for (int i = 1; ok; i += 6) {
      IBRD_STEP(C0, C1, C2, R0, R1, R2, B0, B1, 0)
      IBRD_STEP(C1, C2, C0, R1, R2, R0, B1, B0, 1)
      IBRD_STEP(C2, C0, C1, R2, R0, R1, B0, B1, 2)
      IBRD_STEP(C0, C1, C2, R0, R1, R2, B1, B0, 3)
      IBRD_STEP(C1, C2, C0, R1, R2, R0, B0, B1, 4)
      IBRD_STEP(C2, C0, C1, R2, R0, R1, B1, B0, 5)
    }
#undef IBRD_STEP
  };
  if (w == TY + 2) {
    // stage i + 2 takes the slot of stage i - 1, last read before the barrier
    // that ended step i - 1, as was the coarse plane it replaces
    feed_stages(last, 1, 2, issue, wait_stage, wait_limit, err);
  } else if (a1) {
    march(std::true_type{});
  } else {
    march(std::false_type{});
  }
  if (part) {
    double v = (double)acc;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    double* ws = reinterpret_cast<double*>(RS);  // no step reads RS after the last barrier
    if (row.lane == 0 && w < TY + 2) ws[tid >> 5] = v;
    cta_sync();
    if (tid == 0) {
      double sum = 0.0;
      for (int i = 0; i < (TY + 2) * WPR; ++i) sum += ws[i];
      part[blockIdx.x + gridDim.x * blockIdx.y] = sum;
    }
  }
}

// Shared memory (floats): b ring (rows y0-2 .. y0+TY+1), two published planes
// of red rows y0-2 .. y0+TY+1, two planes of black rows y0-1 .. y0+TY, the odd
// rows' restriction sums.
__host__ __device__ constexpr size_t zero_rows_floats(int nx) {
  return (size_t)kZeroRing * (kRowsTY + 4) * nx + (size_t)(kRowsTY + 4) * nx + (size_t)(kRowsTY + 2) * nx +
         (size_t)(kRowsTY / 2) * (nx / 2);
}

// First red-black sweep from x = 0 fused with the residual restriction: red
// cells (b - shift) / diag, black cells from their red neighbours (the
// arithmetic of k_rb_zero_f32v), bc = mean over the 8 children of
// b - shift - A x, in one pass over b (HBM: read b, write the packed black
// cells and bc; the red cells are b / diag and enter no later sweep). FULL: the
// field is written in full, for cycles whose next pass is not the row sweep with
// the prolongation. In exact
// arithmetic the residual is off times the neighbour sum in the red cells and
// zero in the black ones; inv = 1 / diag in FP32 leaves a common relative error
// of up to 3e-8 in every x, which adds (1 - diag inv) diag x to every residual
// (off times slack x): small, but the coarse levels would not average it out.
//
// Layout as in k_rbgs_rows. Step i reads stage i (b of march plane i + 1),
// publishes its red cells, forms the black cells of plane i (all rows: the edge
// rows' neighbours need them) and the restriction sums of plane i - 1. The two
// planes of a coarse cell are summed in registers over two steps, its two rows
// belong to warps w (even y) and the next (odd y): when a plane pair is
// complete the odd row leaves its sums in shared memory (RY) and the even row
// adds them one step later (after the step's barrier) and writes the coarse
// row. Chunks start on even planes and hold an even number of them, so plane
// pairs never straddle chunks.
template <int NS, int WPR, int NXT, bool FULL>
__global__ void __launch_bounds__(kRowsThreads<WPR>, WPR == 1 ? 2 : 1)
    k_zr_rows(const __grid_constant__ RowMaps mb, float* __restrict__ xo, float* __restrict__ bc,
              const double* __restrict__ bshift, int nx_, int ny, int nz, int zc, float inv, float off, float slack,
              int* __restrict__ err, unsigned wait_limit) {
  constexpr int TY = kRowsTY, R = kZeroRing, XROWS = TY + 4, BROWS = TY + 2;
  const int tid = threadIdx.x, warp = __shfl_sync(0xffffffffu, tid >> 5, 0), w = warp / WPR;
  const Row<NS, WPR, NXT> row(nx_, warp % WPR);
  const int nx = row.nx, nxp = nx >> 1;
  extern __shared__ __align__(1024) unsigned char sm_raw[];
  float* BSM = reinterpret_cast<float*>(sm_raw);
  float* RP = BSM + R * XROWS * nx;
  float* XB = RP + 2 * XROWS * nxp;
  float* RY = XB + 2 * BROWS * nxp;
  unsigned long long* bars = reinterpret_cast<unsigned long long*>(RY + (TY / 2) * nxp);

  const int y0 = blockIdx.x * TY;
  const int k0 = blockIdx.y * zc, k1 = min(k0 + zc, nz);  // even
  const bool down = blockIdx.y & 1;
  const float2 msh = dup2(bshift ? -(float)(*bshift) : -0.f), off2 = dup2(off), inv2 = dup2(inv);
  const float2 off8 = dup2(off * 0.125f), slack2 = dup2(slack);
  const bool interior = w >= 1 && w <= TY;
  const int y = y0 - 1 + w;
  const bool odd_row = y & 1;
  const int last = k1 - k0 + 3;
  auto mp = [&](int i) { return down ? k1 + 1 - i : k0 - 2 + i; };
  // parity of this warp's row in march plane 1 (ny is even, so the wrap keeps it)
  const bool a1 = (y + mp(1)) & 1;

  if (tid == 0) {
    for (int s = 0; s < R; ++s) mbar_init(smem_u32(bars + s), 1);
    asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
  }
  cta_sync();
  // stage i = -1 .. last - 1 (slot (i + 1) % R): b of march plane i + 1
  auto issue = [&](int i, unsigned lead) {
    const int s = (i + 1) % R;
    const unsigned bar = smem_u32(bars + s);
    int z = mp(i + 1);
    z += z < 0 ? nz : (z >= nz ? -nz : 0);
    mbar_expect_tx(bar, XROWS * nx * 4, lead);
    load_rows<TY, 2>(BSM + s * XROWS * nx, nx, mb, y0, ny, z, bar, lead);
  };
  auto wait_stage = [&](int i, unsigned limit) {
    return mbar_wait(smem_u32(bars + (i + 1) % R), (unsigned)(((i + 1) / R) & 1), limit);
  };
  auto rprow = [&](int par, int r) { return RP + (par * XROWS + r) * nxp; };
  auto xbrow = [&](int par, int r) { return XB + (par * BROWS + r) * nxp; };
  auto put_row = [&](float* p, const float2 (&v)[NS]) {
#pragma unroll
    for (int s = 0; s < NS; ++s)
      if (row.valid(s)) *reinterpret_cast<float2*>(p + 2 * row.group(s)) = v[s];
  };
  auto get_row = [&](float2 (&v)[NS], const float* p) {
#pragma unroll
    for (int s = 0; s < NS; ++s) v[s] = *reinterpret_cast<const float2*>(p + 2 * row.group(s));
  };
  // the plane in ring slot `slot` (its march index's parity par, this row's
  // parity a): its red cells, (b - shift) / diag, into r (this warp's row) and
  // into the published rows; its black cells' b - shift into bb
  auto take_plane = [&](float2 (&r)[NS], float2 (&bb)[NS], bool a, int slot, int par) {
    const float* p = BSM + (slot * XROWS + w + 1) * nx;
#pragma unroll
    for (int s = 0; s < NS; ++s) {
      const float4 t = *reinterpret_cast<const float4*>(p + 4 * row.group(s));
      r[s] = mul2(add2(a ? make_float2(t.y, t.w) : make_float2(t.x, t.z), msh), inv2);
      bb[s] = add2(a ? make_float2(t.x, t.z) : make_float2(t.y, t.w), msh);
    }
    put_row(rprow(par, w + 1), r);
    if (!interior) {  // the outer row next to this halo row (the other parity)
      const int o = w == 0 ? 0 : TY + 3;
      const float* q = BSM + (slot * XROWS + o) * nx;
      float2 v[NS];
#pragma unroll
      for (int s = 0; s < NS; ++s) {
        const float4 t = *reinterpret_cast<const float4*>(q + 4 * row.group(s));
        v[s] = mul2(add2(a ? make_float2(t.x, t.z) : make_float2(t.y, t.w), msh), inv2);
      }
      put_row(rprow(par, o), v);
    }
  };

  bool ok = true;
  // where this row of plane mp(2), mp(3), ... and the coarse rows go
  const int nxo = FULL ? nx : nxp;  // row length of the output
  const ptrdiff_t pplane = (ptrdiff_t)nxo * ny, cplane = (ptrdiff_t)nxp * (ny >> 1);
  float* dst = xo + (ptrdiff_t)mp(2) * pplane + (ptrdiff_t)y * nxo;
  float* cdst = bc + (ptrdiff_t)(mp(2) >> 1) * cplane + (ptrdiff_t)(y >> 1) * nxp;
  const ptrdiff_t dstep = down ? -pplane : pplane, cstep = down ? -cplane : cplane;
  float2 held[NS];  // restriction sums of a completed plane pair (even rows)
  // coarse row of an even fine row y: its held sums plus the odd row's (RY)
  auto combine = [&]() {
    float2 o[NS];
    get_row(o, RY + ((w - 1) >> 1) * nxp);
#pragma unroll
    for (int s = 0; s < NS; ++s)
      if (row.valid(s)) *reinterpret_cast<float2*>(cdst + 2 * row.group(s)) = mul2(add2(held[s], o[s]), off8);
    cdst += cstep;
  };
  auto march = [&](auto first_parity) {
    constexpr bool A1 = decltype(first_parity)::value;
    // red cells of three planes, b of the black cells of two, black cells of three
    float2 R0[NS], R1[NS], R2[NS], B0[NS], B1[NS], X0[NS], X1[NS], X2[NS];
    float2 acc[NS];  // restriction sums of the plane pair in progress
    ok = !cta_sync_or(false);  // stages -1, 0 and 1 have landed
    if (!ok) return;
    take_plane(R0, B1, !A1, 0, 0);
    take_plane(R1, B0, A1, 1, 1);
    cta_sync();  // the slots of stages -1 and 0 are free

    // Step i: rm, r0, rp = red cells of march planes i - 1, i, i + 1 (rp is read here); b0 / bp = b of the black cells
    // of planes i / i + 1; xm2, xm1, x0 = black cells of planes i - 2, i - 1, i (x0 is formed here).
    auto step = [&](float2 (&rm)[NS], float2 (&r0)[NS], float2 (&rp)[NS], float2 (&b0)[NS], float2 (&bp)[NS],
                    float2 (&xm2)[NS], float2 (&xm1)[NS], float2 (&x0)[NS], int i, auto phase) {
      constexpr int PH = decltype(phase)::value, P0 = (PH + 1) & 1, P1 = PH & 1;
      constexpr bool a = A1 != (bool)(PH & 1);  // plane i: red cells at 2 m + a, black ones at 2 m + 1 - a
      // plane pairs complete at even i; the odd row left its sums in RY before the last barrier
      if (P0 == 1 && interior && !odd_row && i >= 5) combine();
      take_plane(rp, bp, !a, (i + 1) % R, P1);
      float2 n[NS], u[NS], d[NS];
      nbr_sums<NS, WPR, NXT>(n, r0, rprow(P0, w + 1), !a, row);
      get_row(u, rprow(P0, w));
      get_row(d, rprow(P0, w + 2));
#pragma unroll
      for (int s = 0; s < NS; ++s)
        x0[s] = mul2(fma2(off2, add2(add2(n[s], add2(u[s], d[s])), add2(rm[s], rp[s])), b0[s]), inv2);
      put_row(xbrow(P0, w), x0);
      if (interior && i >= 3) {
        if constexpr (FULL) {
#pragma unroll
          for (int s = 0; s < NS; ++s)
            if (row.valid(s))
              *reinterpret_cast<float4*>(dst + 4 * row.group(s)) =
                  a ? make_float4(rm[s].x, xm1[s].x, rm[s].y, xm1[s].y) : make_float4(xm1[s].x, rm[s].x, xm1[s].y, rm[s].y);
        } else {
          put_row(dst, xm1);
        }
        dst += dstep;
        nbr_sums<NS, WPR, NXT>(n, xm1, xbrow(P1, w), !a, row);
        get_row(u, xbrow(P1, w - 1));
        get_row(d, xbrow(P1, w + 1));
        // march order visits a plane pair (2K, 2K + 1) upwards or downwards, its first plane at odd i
#pragma unroll
        for (int s = 0; s < NS; ++s) {
          const float2 p = fma2(slack2, add2(rm[s], xm1[s]), add2(add2(n[s], add2(u[s], d[s])), add2(xm2[s], x0[s])));
          acc[s] = P0 == 1 ? p : add2(acc[s], p);
        }
        if (P0 == 0) {
          if (odd_row) {
            put_row(RY + ((w - 2) >> 1) * nxp, acc);
          } else {
#pragma unroll
            for (int s = 0; s < NS; ++s) held[s] = acc[s];
          }
        }
      }
      if constexpr (PH == 5)
        ok = !cta_sync_or(false);
      else
        cta_sync();
    };
#define IBRD_STEP(r0, r1, r2, b0, b1, x0, x1, x2, ph) \
  if (i + ph >= last) return;                         \
  step(r0, r1, r2, b0, b1, x0, x1, x2, i + ph, std::integral_constant<int, ph>{});
    for (int i = 1; ok; i += 6) {
      IBRD_STEP(R0, R1, R2, B0, B1, X0, X1, X2, 0)
      IBRD_STEP(R1, R2, R0, B1, B0, X1, X2, X0, 1)
      IBRD_STEP(R2, R0, R1, B0, B1, X2, X0, X1, 2)
      IBRD_STEP(R0, R1, R2, B1, B0, X0, X1, X2, 3)
      IBRD_STEP(R1, R2, R0, B0, B1, X1, X2, X0, 4)
      IBRD_STEP(R2, R0, R1, B1, B0, X2, X0, X1, 5)
    }
#undef IBRD_STEP
  };
  if (w == TY + 2) {
    feed_stages(last, 2, 3, issue, wait_stage, wait_limit, err);  // stage i + 3 takes the slot of stage i - 1
  } else if (a1) {
    march(std::true_type{});
  } else {
    march(std::false_type{});
  }
  if (ok && interior && !odd_row) combine();  // the last pair (its RY write preceded the last barrier)
}

PFN_cuTensorMapEncodeTiled_v12000 encode_fn() {
  static PFN_cuTensorMapEncodeTiled_v12000 fn = nullptr;
  static std::once_flag once;
  std::call_once(once, []() {
    void* p = nullptr;
    cudaDriverEntryPointQueryResult q{};
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) ==
            cudaSuccess &&
        q == cudaDriverEntryPointSuccess)
      fn = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(p);
  });
  if (!fn) throw CudaError{cudaErrorNotSupported, "cuTensorMapEncodeTiled entry point"};
  return fn;
}

// Tensor map of an FP32 field of rows of nx values [nz][ny][nx] with boxes of
// one plane of `rows` whole rows. A box side holds at most 256 values: longer
// rows are two halves (a fourth dimension), which land one after the other.
CUtensorMap field_map(const float* f, int nx, int ny, int nz, int rows) {
  CUtensorMap m;
  std::memset(&m, 0, sizeof(m));
  const int parts = nx > 256 ? 2 : 1, w = nx / parts;
  const cuuint64_t dims[4] = {(cuuint64_t)w, (cuuint64_t)parts, (cuuint64_t)ny, (cuuint64_t)nz};
  const cuuint64_t strides[3] = {(cuuint64_t)w * 4, (cuuint64_t)nx * 4, (cuuint64_t)nx * ny * 4};
  const cuuint32_t box[4] = {(cuuint32_t)w, (cuuint32_t)parts, (cuuint32_t)rows, 1};
  const cuuint32_t es[4] = {1, 1, 1, 1};
  const CUresult r = encode_fn()(&m, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 4, const_cast<float*>(f), dims, strides, box,
                                 es, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE,
                                 CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  if (r != CUDA_SUCCESS) throw CudaError{cudaErrorInvalidValue, "cuTensorMapEncodeTiled"};
  return m;
}

// The maps of a field whose tiles have `rows` rows: only those that load_rows
// uses for ny rows (an encoding is most of a microsecond of host time, which
// counts on levels whose kernels take five).
RowMaps row_maps(const float* f, int nx, int ny, int nz, int rows, int halo) {
  RowMaps m{};
  if (ny >= 3 * rows) m.all = field_map(f, nx, ny, nz, rows + 2 * halo);
  m.part = field_map(f, nx, ny, nz, ny >= 2 * rows ? rows + halo : rows);
  m.halo = field_map(f, nx, ny, nz, halo);
  return m;
}

// two CTAs of the sweep and three of the sweep from zero per SM at 256-cell
// rows (228 KB of shared memory, 1 KB reserved per CTA)
static_assert(2 * (4 * sweep_rows_floats(256, IN_FULL_PRO) + 8 * kSweepRing + 1024) <= 228 * 1024, "two CTAs per SM");
static_assert(3 * (4 * zero_rows_floats(256) + 8 * kZeroRing + 1024) <= 228 * 1024, "three CTAs per SM");

template <int NS, int WPR, int NXT, int IN>
void sweep_rows_go(dim3 g, cudaStream_t s, const RowMaps& mx, const RowMaps& mb, const RowMaps& mc, float* xout, const double* bshift, Dims d,
                   int zc, float inv, float off, double* part) {
  const size_t sm = 4 * sweep_rows_floats(d.nx, IN) + 8 * kSweepRing;
  static std::atomic<unsigned long long> attr{0};
  ensure_smem_attr((const void*)k_rbgs_rows<NS, WPR, NXT, IN>,
                   (int)(4 * sweep_rows_floats(NXT ? NXT : 128 * NS * WPR, IN) + 8 * kSweepRing), attr);
  k_rbgs_rows<NS, WPR, NXT, IN><<<g, kRowsThreads<WPR>, sm, s>>>(
      mx, mb, mc, xout, bshift, d.nx, d.ny, d.nz, zc, inv, off, part, wait_error_flag(),
      wait_limit());
}

template <int NS, int WPR, int NXT, bool FULL>
void zero_rows_go(dim3 g, cudaStream_t s, const RowMaps& mb, float* x, float* bc, const double* bshift, Dims d, int zc,
                  float inv, float off, float slack) {
  const size_t sm = 4 * zero_rows_floats(d.nx) + 8 * kZeroRing;
  static std::atomic<unsigned long long> attr{0};
  ensure_smem_attr((const void*)k_zr_rows<NS, WPR, NXT, FULL>,
                   (int)(4 * zero_rows_floats(NXT ? NXT : 128 * NS * WPR) + 8 * kZeroRing), attr);
  k_zr_rows<NS, WPR, NXT, FULL><<<g, kRowsThreads<WPR>, sm, s>>>(mb, x, bc, bshift, d.nx, d.ny, d.nz, zc, inv, off,
                                                                 slack, wait_error_flag(), wait_limit());
}

// Calls f with the kernel shape of rows of nx cells (see rows_sweep_ok).
template <typename F>
void with_row_shape(int nx, F&& f) {
  constexpr std::integral_constant<int, 0> any{};
  constexpr std::integral_constant<int, 1> one{};
  constexpr std::integral_constant<int, 2> two{};
  if (nx == 128)
    f(one, one, std::integral_constant<int, 128>{});
  else if (nx == 256)
    f(two, one, std::integral_constant<int, 256>{});
  else if (nx == 512)
    f(two, two, std::integral_constant<int, 512>{});
  else if (nx < 128)
    f(one, one, any);
  else if (nx < 256)
    f(two, one, any);
  else
    f(two, two, any);
}

// The row sweep of x (in: SweepIn; xc the coarse field of the fused prolongation) into xout.
template <int IN>
int sweep_rows_any(const float* xin, const float* xc, float* xout, const float* b, const double* bshift, Dims d,
                   Stencil st, int zc, double* part, int part_cap, cudaStream_t s) {
  const int nxr = IN == IN_PACKED_PRO ? d.nx / 2 : d.nx;
  const RowMaps mx = row_maps(xin, nxr, d.ny, d.nz, kRowsTY, 2), mb = row_maps(b, d.nx, d.ny, d.nz, kRowsTY, 1);
  const RowMaps mc = xc ? row_maps(xc, d.nx / 2, d.ny / 2, d.nz / 2, kRowsTY / 2, 2) : mx;
  dim3 g(d.ny / kRowsTY, (d.nz + zc - 1) / zc);
  const int nblk = (int)(g.x * g.y);
  if (nblk > part_cap) part = nullptr;
  with_row_shape(d.nx, [&](auto ns, auto wpr, auto nxt) {
    if constexpr (IN != IN_FULL_PRO || wpr.value == 1 || nxt.value == 512)  // (rows_prolong_full_ok)
      sweep_rows_go<ns.value, wpr.value, nxt.value, IN>(g, s, mx, mb, mc, xout, bshift, d, zc,
                                                        (float)(1.0 / st.diag), (float)st.off, part);
  });
  return part ? nblk : 0;
}

int clamp_zc(int zc, int nz, bool even) {
  zc = zc < 2 ? 2 : (zc > nz ? nz : zc);
  return even ? zc + (zc & 1) : zc;
}

}  // namespace

bool rows_sweep_ok(Dims d) {
  return d.nx % 32 == 0 && d.nx <= 512 && d.ny % kRowsTY == 0 && d.ny >= kRowsTY && d.nz % 2 == 0 && d.nz >= 4;
}

// The plain sweep of a full field. A march has a start of four planes and a
// barrier per plane, 5 us at least, which the tiled sweep undercuts on few rows; and
// rows below 96 cells leave lanes idle. Measured (us, row and tiled sweep, data
// in L2) on 16 x 16 rows: 4.9 and 3.6 (96 cells), 5.4 and 4.1 (256), 6.7 and 4.0
// (448); on 32 x 32: 5.0 and 4.4, 5.4 and 4.8, 7.0 and 5.7; on 32 x 64: 5.2 and 4.8,
// 5.7 and 6.7, 7.2 and 7.2; on 64 x 64: 5.8 and 7.1, 6.8 and 8.6, 8.6 and 11.2; on
// 256 x 256: 20.5 and 31.3, 33.1 and 62.4, 63.5 and 93.7. Rows of 32 cells: 5.7 and 4.2
// on 64 x 64, 20.6 and 14.2 on 256 x 256; of 64: 5.3 and 4.9, 20.4 and 17.7. Rows of 128
// and 256 cells, where tuned shapes name the row sweep by their length, keep it on
// every level.
bool rows_plain_ok(Dims d) {
  return rows_sweep_ok(d) && (d.nx == 128 || d.nx == 256 || (d.nx >= 96 && d.ny * (size_t)d.nz >= 2048));
}

// The sweep with the prolongation of a full field, against the prolongation and the
// better of the plain sweeps (us): rows of 96, 160 and 256 cells on 16 x 16: 5.8 and
// 6.5, 7.2 and 6.9, 6.6 and 7.6; on 32 x 32: 5.9 and 7.6, 7.4 and 8.0, 6.8 and 8.0; on
// 256 x 256: 24.6 and 30.2, 47.2 and 47.9, 38.5 and 59.3. Rows of 512: 9.0 and 6.9, 8.7
// and 9.7, 74.4 and 121. Two warps on part of their lanes (rows of 288 to 480), one CTA
// per SM: 9.8 and 7.2, 10.1 and 8.8 (288), 115 and 101 (384 on 256 x 256). Rows of 32:
// 10.6 and 11.6 on 128 x 128, 24.2 and 18.8 on 256 x 256.
bool rows_prolong_full_ok(Dims d) {
  if (!rows_sweep_ok(d) || d.nx == 128 || d.nx == 256) return rows_sweep_ok(d);  // (as for the plain sweep)
  const size_t rows = d.ny * (size_t)d.nz;
  return (d.nx <= 256 || d.nx == 512) && rows >= 1024 && (d.nx >= 64 || rows <= 16384);
}

int rows_sweep_default_zc(Dims d) {
  // about one wave of two resident CTAs per SM (one with two warps per row); an
  // even number of planes, as the sweep with the prolongation fused needs, so
  // that both kernels split a level into the same CTAs (and per-CTA partial sums)
  const int cols = d.ny / kRowsTY;
  int chunks = ((d.nx > 256 ? 1 : 2) * 152) / cols;
  chunks = chunks < 1 ? 1 : chunks;
  int zc = (d.nz + chunks - 1) / chunks;
  zc += zc & 1;
  return zc < 2 ? 2 : zc;
}

int launch_rows_sweep(const float* xin, float* xout, const float* b, const double* bshift, Dims d, Stencil st,
                      int zc, double* part, int part_cap, cudaStream_t s) {
  if (!rows_sweep_ok(d) || !aligned16(xin) || !aligned16(xout) || !aligned16(b) || xin == xout || b == xout)
    throw CudaError{cudaErrorInvalidValue, "row sweep arguments"};
  return sweep_rows_any<IN_FULL>(xin, nullptr, xout, b, bshift, d, st, clamp_zc(zc, d.nz, false), part, part_cap, s);
}

int launch_rows_prolong_sweep(const float* xc, const float* xin, bool packed, float* xout, const float* b,
                              const double* bshift, Dims d, Stencil st, int zc, double* part, int part_cap,
                              cudaStream_t s) {
  if (!rows_sweep_ok(d) || !aligned16(xin) || !aligned16(xout) || !aligned16(b) || !aligned16(xc) || xin == xout ||
      b == xout || xc == xout)
    throw CudaError{cudaErrorInvalidValue, "prolongation + row sweep arguments"};
  // even chunks: fine planes 2K - 1, 2K share their coarse pair in both march directions
  zc = clamp_zc(zc, d.nz, true);
  if (!packed && !rows_prolong_full_ok(d)) throw CudaError{cudaErrorInvalidValue, "prolongation + row sweep level"};
  return packed ? sweep_rows_any<IN_PACKED_PRO>(xin, xc, xout, b, bshift, d, st, zc, part, part_cap, s)
                : sweep_rows_any<IN_FULL_PRO>(xin, xc, xout, b, bshift, d, st, zc, part, part_cap, s);
}

// The sweep from zero and the packed sweep that follows it, against the tiled sweep
// from zero with the restriction, the prolongation and the tiled sweep (us, data in
// L2): rows of 128 cells 10.2 and 9.9 on 8 x 8, 10.0 and 10.9 on 16 x 16; of 224
// 11.9 and 11.5 on 16 x 16, 12.5 and 13.8 on 32 x 32 (and one launch less). Two warps
// per row start later: of 320 15.6 and 12.0 on 16 x 16, 15.7 and 15.1 on 32 x 32, 16.4
// and 18.2 on 32 x 64; of 512 14.2 and 11.5, 14.2 and 17.1, 14.3 and 21.3.
bool zero_restrict_rows_ok(Dims d) {
  return rows_sweep_ok(d) && (d.nx <= 256 || d.ny * (size_t)d.nz >= 1024);
}

int zero_restrict_rows_default_zc(Dims d) {
  return rows_sweep_default_zc(d);  // even: plane pairs of the restriction stay inside a chunk
}

void launch_zero_restrict_rows(const float* b, const double* bshift, float* x, bool full, float* bc, Dims d,
                               Stencil st, int zc, cudaStream_t s) {
  if (!zero_restrict_rows_ok(d) || !aligned16(b) || !aligned16(x) || ((uintptr_t)bc & 7u) || b == x)
    throw CudaError{cudaErrorInvalidValue, "fused zero sweep + restriction arguments"};
  zc = clamp_zc(zc, d.nz, true);
  const RowMaps mb = row_maps(b, d.nx, d.ny, d.nz, kRowsTY, 2);
  dim3 g(d.ny / kRowsTY, (d.nz + zc - 1) / zc);
  const float inv = (float)(1.0 / st.diag), slack = (float)((1.0 - st.diag * (double)inv) * st.diag / st.off);
  with_row_shape(d.nx, [&](auto ns, auto wpr, auto nxt) {
    constexpr int NS = ns.value, WPR = wpr.value, NXT = nxt.value;
    if (full)
      zero_rows_go<NS, WPR, NXT, true>(g, s, mb, x, bc, bshift, d, zc, inv, (float)st.off, slack);
    else
      zero_rows_go<NS, WPR, NXT, false>(g, s, mb, x, bc, bshift, d, zc, inv, (float)st.off, slack);
  });
}

}  // namespace ibrd
