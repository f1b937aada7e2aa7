// Split path, load-first variant: the velocity and stress kernels of
// stencil_split.cu with every global load of a thread issued before any of
// its arithmetic or stores (one round trip to memory per thread instead of
// one per component), and the material lookups from the split tables
// {rho}, {1/mu}, {lambda, lambda + 2 mu}.  Same thread layout (four z cells
// per thread, 16-byte loads, block = 32 x 4 threads, theta fastest across
// blocks), same arithmetic, same in-place update; variants with two z cells
// per thread (8-byte loads, fewer registers), interior / edge split launches
// (a lean-only kernel on the interior tiles), the march along theta
// (hoist_run.cuh) and one launch per half for batches and small grids.
#include <algorithm>

#include "hoist_run.cuh"

namespace cwell {
namespace {

constexpr int HB_X = 32;  // threads along z per block (NV cells each)
constexpr int HB_Y = 4;   // r rows per block

// Block order: ZF = false walks theta fastest (blockIdx.x = theta, y = r tile,
// z = z tile: co-resident blocks share theta-neighbour rows); ZF = true walks
// z fastest (x = z tile, y = r tile, z = theta: co-resident blocks stream
// whole rows, theta neighbours come back from L2).
template <bool ZF, int NV>
__device__ __forceinline__ void block_cell(int &j, int &i, int &k0) {
  const int zt = ZF ? blockIdx.x : blockIdx.z;
  j = ZF ? blockIdx.z : blockIdx.x;
  i = blockIdx.y * HB_Y + threadIdx.y;
  k0 = (zt * HB_X + threadIdx.x) * NV;
}

template <typename T, int NV, int MINB, bool ZF>
__global__ void __launch_bounds__(HB_X *HB_Y, MINB) vel_hoist(const KParams p) {
  int j, i, k0;
  block_cell<ZF, NV>(j, i, k0);
  if (i < p.NR && k0 < p.NZ) hoist_cells<T, NV, true>(p, j, i, k0);
}

template <typename T, int NV, int MINB, bool ZF>
__global__ void __launch_bounds__(HB_X *HB_Y, MINB) str_hoist(const KParams p) {
  int j, i, k0;
  block_cell<ZF, NV>(j, i, k0);
  if (i < p.NR && k0 < p.NZ) hoist_cells<T, NV, false>(p, j, i, k0);
}

// Regions of a half step.  A group of four z cells is lean when its row lies
// outside the radial PML and the group and its +1 z neighbour outside the z
// PML and inside NZ.  The cells fall into
//  * the interior: rows [i_lo, nr), groups [za, zb): the lean body;
//  * the radial layer: rows [nr, NR), groups [za, zb): a body compiled for
//    "radial PML, interior z" (no z memory variable, no z bound check);
//  * the z ends: every row, groups [0, za) and [zb, NZ): the general body.
// Interior and radial tiles are HB_Y rows x 32 threads along z on a 128-byte
// aligned z grid; threads of a tile outside its region do nothing, so a region
// need not start or end on a tile; a first or last interior tile that would
// hold less than a quarter of its cells goes to the z ends instead (8224 cells:
// a 65th tile for 12 of them cost 1.3 % on the refined 20 m well).  The z ends
// are narrow, so their threads are numbered (theta, row, group) with the group
// fastest and no thread idles.  (When a tile belonged to the ends as soon as
// one of its cells did, 128 or 64 cells at each end of every row ran the
// general body instead of pml_z: 16 % of a 1527-cell row, all of a 256-cell
// one.)
struct Regions {
  int r0;            // first row of the radial layer
  int za, zb;        // lean z groups
  int zt0, nzt, nrt; // interior tiles: z tiles zt0 .. zt0 + nzt - 1, r tiles 0 .. nrt - 1 from row i_lo
  int rzt0, rnzt, rnrt;  // radial tiles: the same, r tiles counted from row r0
  int na, nb;        // groups per row of the low and the high z end
  long long interior, radial, ends;  // tiles, tiles, blocks of 128 threads
};

// tiles of the regions r0, za, zb; NV: cells per thread in the interior, NVE:
// in the radial layer and the z ends
template <int NV, int NVE>
Regions region_tiles(const KParams &p, int r0, int za, int zb) {
  Regions q;
  q.r0 = r0;
  q.za = za;
  q.zb = zb;
  const bool any = q.zb > q.za;
  auto tiles = [&](int w, int &t0, int &n) {
    t0 = q.za / w;
    n = any ? (q.zb + w - 1) / w - t0 : 0;
  };
  tiles(NV * HB_X, q.zt0, q.nzt);
  tiles(NVE * HB_X, q.rzt0, q.rnzt);
  q.nrt = (std::max(0, std::min(r0, p.i_hi) - p.i_lo) + HB_Y - 1) / HB_Y;
  q.rnrt = (p.NR - r0 + HB_Y - 1) / HB_Y;
  q.na = q.za / NVE;
  q.nb = (p.NZ - q.zb + NVE - 1) / NVE;
  q.interior = (long long)p.nth * q.nrt * q.nzt;
  q.radial = (long long)p.nth * q.rnrt * q.rnzt;
  q.ends = ((long long)p.nth * (p.i_hi - p.i_lo) * (q.na + q.nb) + HB_X * HB_Y - 1) / (HB_X * HB_Y);
  return q;
}

// first row of the radial layer's tiles.  Stochastic rounding decides by the last
// bits of FP32, so its layer keeps the order of sums that each cell has always had,
// by whole tiles of rows and of 128 z cells (z_sum); the first tile of rows may start
// above the layer.
template <typename T>
int layer_row(const KParams &p) {
  const int r = std::min(p.nr, p.NR);
  return std::is_same<T, half_sr>::value ? r / HB_Y * HB_Y : r;
}

template <typename T, int NV, int NVE>
Regions regions(const KParams &p) {
  int za = (p.pml_z + 3) / 4 * 4, zb = std::max(za, (p.NZ - p.pml_z - 1) / 4 * 4);
  constexpr int W = NV * HB_X;
  if (za % W > W - W / 4) za = (za + W - 1) / W * W;
  if (zb % W < W / 4) zb = zb / W * W;
  return region_tiles<NV, NVE>(p, layer_row<T>(p), za, std::max(za, zb));
}

// cell group of this thread in interior tile t (theta fastest, then r, then z); false: nothing to do
template <int NV>
__device__ __forceinline__ bool interior_cell(const KParams &p, const Regions &q, int t, int &j, int &i, int &k0) {
  j = t % p.nth;
  t /= p.nth;
  i = p.i_lo + (t % q.nrt) * HB_Y + threadIdx.y;
  k0 = ((q.zt0 + t / q.nrt) * HB_X + threadIdx.x) * NV;
  return i < q.r0 && i < p.i_hi && k0 >= q.za && k0 < q.zb && k0 >= p.k_lo && k0 < p.k_hi;
}
template <int NV>
__device__ __forceinline__ bool radial_cell(const KParams &p, const Regions &q, int t, int &j, int &i, int &k0) {
  j = t % p.nth;
  t /= p.nth;
  i = q.r0 + (t % q.rnrt) * HB_Y + threadIdx.y;
  k0 = ((q.rzt0 + t / q.rnrt) * HB_X + threadIdx.x) * NV;
  return i >= p.i_lo && i < p.i_hi && k0 >= q.za && k0 < q.zb && k0 >= p.k_lo && k0 < p.k_hi;
}
template <int NV>
__device__ __forceinline__ bool end_cell(const KParams &p, const Regions &q, int block, int &j, int &i, int &k0) {
  const unsigned n = q.na + q.nb;
  unsigned t = block * (HB_X * HB_Y) + threadIdx.y * HB_X + threadIdx.x;
  const int g = t % n;
  t /= n;
  i = p.i_lo + t % (p.i_hi - p.i_lo);
  j = t / (p.i_hi - p.i_lo);
  k0 = g < q.na ? g * NV : q.zb + (g - q.na) * NV;
  return j < p.nth && k0 >= p.k_lo && k0 < p.k_hi;
}

template <typename T, int NV, bool VEL>
__device__ __forceinline__ void lean_cells_step(const KParams &p, int j, int i, int k0) {
  if (VEL) vel_hoist_body<T, NV, true>(p, j, i, k0);
  else str_hoist_body<T, NV, true>(p, j, i, k0);
}
template <typename T, int NV, bool VEL>
__device__ __forceinline__ void radial_cells_step(const KParams &p, int j, int i, int k0, const OutSet *out = nullptr) {
  if (VEL) vel_hoist_body<T, NV, false, true, true>(p, j, i, k0, out);
  else str_hoist_body<T, NV, false, true, true>(p, j, i, k0, out);
}
// The z ends also hold cells beside the layer that no memory variable touches (up
// to three of a cut group, up to a quarter of a tile): PAIRS gives them the bits of
// the lean body, so that where the cut lies does not show in the fields.
template <typename T, int NV, bool VEL>
__device__ __forceinline__ void end_cells_step(const KParams &p, int j, int i, int k0, const OutSet *out = nullptr) {
  if (VEL) vel_hoist_body<T, NV, false, true, false, true>(p, j, i, k0, out);
  else str_hoist_body<T, NV, false, true, false, false, true>(p, j, i, k0, out);
}

template <typename T, int NV, int MINB, bool VEL>
__global__ void __launch_bounds__(HB_X *HB_Y, MINB) hoist_interior(const KParams p, const Regions q) {
  int j, i, k0;
  if (interior_cell<NV>(p, q, blockIdx.x, j, i, k0)) lean_cells_step<T, NV, VEL>(p, j, i, k0);
}

// Persistent interior kernel with an L2 prefetch of its next tile: one wave
// of resident blocks walks the interior tiles in the order above (theta
// fastest); before computing its tile a block asks L2 for every row its next
// tile will load (one prefetch per 128-byte line), so those loads find their
// lines in L2.  No register or shared memory holds the prefetched data.
template <typename T, int NV, int MINB, bool VEL>
__global__ void __launch_bounds__(HB_X *HB_Y, MINB) hoist_interior_pf(const KParams p, const Regions q) {
  const int n = (int)q.interior;
  for (int t = blockIdx.x; t < n; t += gridDim.x) {
    int j, i, k0;
    if (t + (int)gridDim.x < n && interior_cell<NV>(p, q, t + gridDim.x, j, i, k0)) prefetch_tile<T, NV, VEL>(p, j, i, k0);
    if (interior_cell<NV>(p, q, t, j, i, k0)) lean_cells_step<T, NV, VEL>(p, j, i, k0);
  }
}

// tiles of the interior (RAD: of the radial layer) marched along theta in runs of
// `run` planes (last run shorter); block = one tile of one run, z tiles fastest,
// then r, then the runs; OUT: out of place into `set`
template <typename T, int MINB, bool VEL, bool RAD, bool OUT = false>
__global__ void __launch_bounds__(HB_X *HB_Y, MINB) hoist_run(const KParams p, const Regions q, int run, const OutSet set) {
  extern __shared__ float2 run_tab[];
  run_table<VEL>(p, run_tab);
  const int nzt = RAD ? q.rnzt : q.nzt, nrt = RAD ? q.rnrt : q.nrt;
  int t = blockIdx.x;
  const int k0 = (((RAD ? q.rzt0 : q.zt0) + t % nzt) * HB_X + threadIdx.x) * 4;
  t /= nzt;
  const int i = (RAD ? q.r0 : p.i_lo) + (t % nrt) * HB_Y + threadIdx.y, j0 = t / nrt * run, J = min(run, p.nth - j0);
  const bool in = RAD ? i >= p.i_lo : i < q.r0;
  if (!(in && i < p.i_hi && k0 >= q.za && k0 < q.zb && k0 >= p.k_lo && k0 < p.k_hi)) return;
  void *const *fo = OUT ? set.f : p.f;
  if (VEL) vel_run<T, RAD>(p, fo, (const float *)run_tab, j0, J, i, k0);
  else str_run<T, RAD>(p, fo, run_tab, (const float *)(run_tab + p.n_mat), j0, J, i, k0);
}

// planes per run: the fewest rounds of resident blocks times the planes each
// passes over (a run loads about one plane's worth before its first)
inline int run_planes(long long tiles, int nth, int slots) {
  int best = nth;
  double cost = 1e300;
  for (int d = 1; d <= std::max(1, nth / 4); d++) {
    const int run = (nth + d - 1) / d;
    const long long items = tiles * ((nth + run - 1) / run);
    const double c = (double)((items + slots - 1) / slots) * (run + 1);
    if (c < cost) cost = c, best = run;
  }
  return best;
}

// L2 prefetch of a radial-layer tile: the fields' rows and the memory variables
template <typename T, int NV, bool VEL>
__device__ __forceinline__ void prefetch_radial(const KParams &p, int j, int i, int k0, const OutSet *out = nullptr) {
  constexpr int LANES = 128 / (NV * 4);
  prefetch_tile<T, NV, VEL>(p, j, i, k0, out);
  if (i >= p.nr && (threadIdx.x & (LANES - 1)) == 0) {
    const long long cr = ((long long)j * p.pml_r + (i - p.nr)) * p.NZp + k0;
    const int q0 = VEL ? R_VR : R_ERR, q1 = VEL ? Q_VR : Q_EPP;
    for (int u = 0; u < 3; u++) prefetch_l2(p.psr[q0 + u] + cr), prefetch_l2(p.psr[q1 + u] + cr);
  }
}

// radial layer, walked by one wave of resident blocks that prefetch the next tile
template <typename T, int NV, int MINB, bool VEL>
__global__ void __launch_bounds__(HB_X *HB_Y, MINB) hoist_radial_pf(const KParams p, const Regions q) {
  const int n = (int)q.radial;
  for (int t = blockIdx.x; t < n; t += gridDim.x) {
    int j, i, k0;
    if (t + (int)gridDim.x < n && radial_cell<NV>(p, q, t + gridDim.x, j, i, k0)) prefetch_radial<T, NV, VEL>(p, j, i, k0);
    if (radial_cell<NV>(p, q, t, j, i, k0)) radial_cells_step<T, NV, VEL>(p, j, i, k0);
  }
}

template <typename T, int NV, int MINB, bool VEL>
__global__ void __launch_bounds__(HB_X *HB_Y, MINB) hoist_ends(const KParams p, const Regions q) {
  int j, i, k0;
  if (end_cell<NV>(p, q, blockIdx.x, j, i, k0)) end_cells_step<T, NV, VEL>(p, j, i, k0);
}

// z ends (first blocks) and radial layer in one launch; PF: the radial tiles
// are walked by the blocks left in one wave, prefetching the next tile; OUT:
// out of place into `out`
template <typename T, int NV, int MINB, bool VEL, bool PF, bool OUT = false>
__global__ void __launch_bounds__(HB_X *HB_Y, MINB) hoist_edge(const KParams p, const Regions q, const OutSet set) {
  const OutSet *out = OUT ? &set : nullptr;
  int j, i, k0;
  if (blockIdx.x < q.ends) {
    if (end_cell<NV>(p, q, blockIdx.x, j, i, k0)) end_cells_step<T, NV, VEL>(p, j, i, k0, out);
    return;
  }
  const int n = (int)q.radial, step = gridDim.x - (int)q.ends;
  for (int t = blockIdx.x - (int)q.ends; t < n; t += step) {
    if (PF && t + step < n && radial_cell<NV>(p, q, t + step, j, i, k0)) prefetch_radial<T, NV, VEL>(p, j, i, k0, out);
    if (radial_cell<NV>(p, q, t, j, i, k0)) radial_cells_step<T, NV, VEL>(p, j, i, k0, out);
  }
}

// z ends (first blocks) and the row q.r0 alone, four z tiles per block, out of place
template <typename T, int NV, int MINB, bool VEL>
__global__ void __launch_bounds__(HB_X *HB_Y, MINB) hoist_rim(const KParams p, const Regions q, const OutSet set) {
  int j, i, k0;
  if (blockIdx.x < q.ends) {
    if (end_cell<NV>(p, q, blockIdx.x, j, i, k0)) end_cells_step<T, NV, VEL>(p, j, i, k0, &set);
    return;
  }
  const int t = blockIdx.x - (int)q.ends;
  j = t % p.nth;
  k0 = ((q.rzt0 + t / p.nth * HB_Y + threadIdx.y) * HB_X + threadIdx.x) * NV;
  if (k0 >= q.za && k0 < q.zb) radial_cells_step<T, NV, VEL>(p, j, q.r0, k0, &set);
}

// the whole half step in one launch: z ends, radial layer, interior, in this
// order of blocks (the edge blocks carry the longer bodies)
template <typename T, int NV, int NVE, int MINB, bool VEL>
__global__ void __launch_bounds__(HB_X *HB_Y, MINB) hoist_one(const KParams p, const Regions q) {
  int j, i, k0, t = blockIdx.x;
  if (t < q.ends) {
    if (end_cell<NVE>(p, q, t, j, i, k0)) end_cells_step<T, NVE, VEL>(p, j, i, k0);
  } else if ((t -= (int)q.ends) < q.radial) {
    if (radial_cell<NVE>(p, q, t, j, i, k0)) radial_cells_step<T, NVE, VEL>(p, j, i, k0);
  } else {
    t -= (int)q.radial;
    if (interior_cell<NV>(p, q, t, j, i, k0)) lean_cells_step<T, NV, VEL>(p, j, i, k0);
  }
}

// Batched scenarios and the zones of a refined grid: each half step is one
// launch over up to BATCH_MAX cases, block = one tile (or 128 end threads) of
// one case, all cases' z ends and radial tiles before the interior tiles,
// theta fastest inside a case so that the theta neighbours a block reads are
// read by co-resident blocks too.  The cases' parameters, their regions and
// the prefix sums of their blocks (edge[c] = first z-end or radial block of
// case c, inner[c] = first interior block, counted from 0 each) travel in the
// kernel's parameter space, so a block reads its case's geometry and buffers
// from the constant bank.  Rows outside [i_lo, i_hi) are left alone (as in
// every split kernel: the ghost rows of a refined grid's zones).
struct BatchParams {
  KParams cases[BATCH_MAX];
  Regions q[BATCH_MAX];
  int edge[BATCH_MAX + 1], inner[BATCH_MAX + 1];
  int n;
};
static_assert(sizeof(BatchParams) <= 32000, "batch parameters exceed the kernel parameter space");

constexpr int BATCH_NV = 4, BATCH_NVE = 2, BATCH_MINB = 4;

// the case whose blocks hold block t: start[c] <= t < start[c + 1]
__device__ __forceinline__ int batch_case(const int *start, int n, int t) {
  int lo = 0, hi = n - 1;
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (start[mid] <= t) lo = mid;
    else hi = mid - 1;
  }
  return lo;
}

template <typename T, bool VEL>
__global__ void __launch_bounds__(HB_X *HB_Y, BATCH_MINB) hoist_batch(const __grid_constant__ BatchParams bp) {
  int t = blockIdx.x, j, i, k0;
  const int nedge = bp.edge[bp.n];
  if (t >= nedge) {
    t -= nedge;
    const int c = batch_case(bp.inner, bp.n, t);
    if (interior_cell<BATCH_NV>(bp.cases[c], bp.q[c], t - bp.inner[c], j, i, k0))
      lean_cells_step<T, BATCH_NV, VEL>(bp.cases[c], j, i, k0);
    return;
  }
  const int c = batch_case(bp.edge, bp.n, t);
  const KParams &p = bp.cases[c];
  const Regions &q = bp.q[c];
  t -= bp.edge[c];
  if (t < q.ends) {
    if (end_cell<BATCH_NVE>(p, q, t, j, i, k0)) end_cells_step<T, BATCH_NVE, VEL>(p, j, i, k0);
  } else if (radial_cell<BATCH_NVE>(p, q, t - (int)q.ends, j, i, k0)) {
    radial_cells_step<T, BATCH_NVE, VEL>(p, j, i, k0);
  }
}

template <typename T, bool VEL>
cudaError_t launch_batch_t(const KParams *cases, int n_cases, cudaStream_t s) {
  static thread_local BatchParams bp;  // large: kept off the stack
  for (int c0 = 0; c0 < n_cases; c0 += BATCH_MAX) {
    const int n = std::min(BATCH_MAX, n_cases - c0);
    long long edge = 0, inner = 0;
    bp.n = n;
    for (int c = 0; c <= n; c++) {
      bp.edge[c] = (int)edge;
      bp.inner[c] = (int)inner;
      if (c == n) break;
      bp.cases[c] = cases[c0 + c];
      bp.q[c] = regions<T, BATCH_NV, BATCH_NVE>(cases[c0 + c]);
      edge += bp.q[c].ends + bp.q[c].radial;
      inner += bp.q[c].interior;
      if (edge + inner > 0x7fffffffLL || bp.q[c].ends * (HB_X * HB_Y) > 0x7fffffffLL) return cudaErrorInvalidValue;
    }
    hoist_batch<T, VEL><<<(int)(edge + inner), dim3(HB_X, HB_Y), 0, s>>>(bp);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

int sm_count() {
  static int n = 0;
  if (!n) {
    int dev = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev);
    if (n < 1) n = 1;
  }
  return n;
}

thread_local const SideStream *g_side = nullptr;

// fork / join of the edge launches of a half onto the side stream (when one
// is set and the half has both kinds of tiles); returns the edge stream
inline cudaError_t side_fork(bool fork, cudaStream_t s, cudaStream_t *se) {
  *se = s;
  if (!fork) return cudaSuccess;
  cudaError_t e = cudaEventRecord(g_side->fork, s);
  if (e == cudaSuccess) e = cudaStreamWaitEvent(g_side->side, g_side->fork, 0);
  if (e == cudaSuccess) *se = g_side->side;
  return e;
}
inline cudaError_t side_join(bool fork, cudaStream_t s) {
  if (!fork) return cudaSuccess;
  cudaError_t e = cudaEventRecord(g_side->join, g_side->side);
  if (e == cudaSuccess) e = cudaStreamWaitEvent(s, g_side->join, 0);
  return e;
}

inline int wave(long long tiles, int minb) { return (int)std::min<long long>(tiles, (long long)sm_count() * minb); }

// tables and arrays beyond the march's shared memory and 32-bit offsets go tile by tile
template <typename T>
bool can_run(const KParams &p) {
  const unsigned long long lim = 0xffffffffull - 4096;
  return p.n_mat <= RUN_MATS && (unsigned long long)p.plane * p.nth * sizeof(T) < lim &&
         (unsigned long long)p.pml_r * p.NZp * p.nth * 4 < lim;
}
template <typename T, int MINB, bool VEL, bool RAD, bool OUT>
void launch_run(const KParams &p, const Regions &q, const OutSet &set, cudaStream_t s) {
  const int tiles = RAD ? q.rnrt * q.rnzt : q.nrt * q.nzt, run = run_planes(tiles, p.nth, sm_count() * MINB);
  hoist_run<T, MINB, VEL, RAD, OUT><<<tiles * ((p.nth + run - 1) / run), dim3(HB_X, HB_Y),
                                      run_table_bytes(p.n_mat, VEL), s>>>(p, q, run, set);
}

// MODE 0: one tile per block; 1: persistent with prefetch; 2: marched along theta
template <typename T, int NV, int MINB, int MODE, bool VEL>
void launch_interior(const KParams &p, const Regions &q, cudaStream_t s) {
  dim3 blk(HB_X, HB_Y);
  if constexpr (MODE == 2) {
    static_assert(NV == 4, "four cells per thread");
    constexpr int MB = sizeof(T) == 2 && !VEL ? MINB - 1 : MINB;  // 16 bits: 3 stress, 4 velocity blocks (at most 8 bytes spilled)
    if (can_run<T>(p)) launch_run<T, MB, VEL, false, false>(p, q, OutSet{}, s);
    else hoist_interior<T, NV, 4, VEL><<<(int)q.interior, blk, 0, s>>>(p, q);
  } else if constexpr (MODE == 1) hoist_interior_pf<T, NV, MINB, VEL><<<wave(q.interior, MINB), blk, 0, s>>>(p, q);
  else hoist_interior<T, NV, MINB, VEL><<<(int)q.interior, blk, 0, s>>>(p, q);
}

// Interior launch and edge launch of a half, the latter on the side stream
// (g_side): the regions update disjoint cells from inputs no launch of the half
// writes.  MINB_R = 0: one edge launch (22xx); otherwise the radial layer
// (MINB_R blocks per SM) and the z ends apart (23xx).
template <typename T, int NV, int MINB_IN, int MODE, int NVE, int MINB_R, int MINB_E, int PFE, bool VEL>
cudaError_t launch_split_half(const KParams &p, const Regions &q, cudaStream_t s) {
  dim3 blk(HB_X, HB_Y);
  const bool edge = q.radial > 0 || q.ends > 0;
  const bool fork = g_side && q.interior > 0 && edge;
  cudaStream_t se;  // stream of the edge launches
  cudaError_t e = side_fork(fork, s, &se);
  if (e != cudaSuccess) return e;
  if constexpr (MINB_R == 0) {
    const int rad = PFE ? wave(q.radial, PFE) : (int)q.radial;
    if (edge) hoist_edge<T, NVE, MINB_E, VEL, (PFE > 0)><<<(int)q.ends + rad, blk, 0, se>>>(p, q, OutSet{});
  } else {
    if (q.radial > 0) {
      if constexpr (MODE == 2 && sizeof(T) == 4) {
        if (can_run<T>(p)) launch_run<T, 2, VEL, true, false>(p, q, OutSet{}, se);
        else hoist_radial_pf<T, NVE, MINB_R, VEL><<<wave(q.radial, MINB_R), blk, 0, se>>>(p, q);
      } else {
        hoist_radial_pf<T, NVE, MINB_R, VEL><<<wave(q.radial, MINB_R), blk, 0, se>>>(p, q);
      }
    }
    if (q.ends > 0) hoist_ends<T, NVE, MINB_E, VEL><<<(int)q.ends, blk, 0, se>>>(p, q);
  }
  if (q.interior > 0) launch_interior<T, NV, MINB_IN, MODE, VEL>(p, q, s);
  if ((e = side_join(fork, s)) != cudaSuccess) return e;
  return cudaGetLastError();
}

// block counts and the end threads' numbers are 32-bit
inline bool fits(const Regions &q) { return q.interior + q.radial + q.ends * (HB_X * HB_Y) <= 0x7fffffffLL; }

template <typename T, int NV, int MINB_IN, int MODE, int NVE, int MINB_R, int MINB_E, int PFE = 0>
cudaError_t launch_split_t(const KParams &p, cudaStream_t s, cudaEvent_t *ev, int parts) {
  const Regions q = regions<T, NV, NVE>(p);
  if (!fits(q)) return cudaErrorInvalidValue;
  cudaError_t e = cudaSuccess;
  if (parts & 1) {
    if (ev) cudaEventRecord(ev[0], s);
    e = launch_split_half<T, NV, MINB_IN, MODE, NVE, MINB_R, MINB_E, PFE, true>(p, q, s);
    if (e != cudaSuccess) return e;
    if (ev) cudaEventRecord(ev[1], s);
  }
  if (parts & 2) {
    e = launch_split_half<T, NV, MINB_IN, MODE, NVE, MINB_R, MINB_E, PFE, false>(p, q, s);
    if (ev) cudaEventRecord(ev[2], s);
  }
  return e;
}

template <typename T, int NV, int NVE, int MINB>
cudaError_t launch_one_t(const KParams &p, cudaStream_t s, cudaEvent_t *ev, int parts) {
  const Regions q = regions<T, NV, NVE>(p);
  if (!fits(q)) return cudaErrorInvalidValue;
  const int grid = (int)(q.ends + q.radial + q.interior);
  if (parts & 1) {
    if (ev) cudaEventRecord(ev[0], s);
    hoist_one<T, NV, NVE, MINB, true><<<grid, dim3(HB_X, HB_Y), 0, s>>>(p, q);
    if (ev) cudaEventRecord(ev[1], s);
  }
  if (parts & 2) {
    hoist_one<T, NV, NVE, MINB, false><<<grid, dim3(HB_X, HB_Y), 0, s>>>(p, q);
    if (ev) cudaEventRecord(ev[2], s);
  }
  return cudaGetLastError();
}

template <typename T, int NV, int MINB, bool ZF>
cudaError_t launch_hoist_t(const KParams &p, cudaStream_t s, cudaEvent_t *ev, int parts) {
  dim3 blk(HB_X, HB_Y);
  const int nzt = (p.NZ + NV * HB_X - 1) / (NV * HB_X), nrt = (p.NR + HB_Y - 1) / HB_Y;
  if (nzt > 65535 || p.nth > 65535) return cudaErrorInvalidValue;
  dim3 grd = ZF ? dim3(nzt, nrt, p.nth) : dim3(p.nth, nrt, nzt);
  if (parts & 1) {
    if (ev) cudaEventRecord(ev[0], s);
    vel_hoist<T, NV, MINB, ZF><<<grd, blk, 0, s>>>(p);
    if (ev) cudaEventRecord(ev[1], s);
  }
  if (parts & 2) {
    str_hoist<T, NV, MINB, ZF><<<grd, blk, 0, s>>>(p);
    if (ev) cudaEventRecord(ev[2], s);
  }
  return cudaGetLastError();
}

// the cells beside a one-pass step's: z ends, radial layer and its rim row r1
template <int NV, int MINB, bool RUN>
cudaError_t launch_pass_edges_t(int part, const KParams &p, const OutSet &out, cudaStream_t s) {
  int r1, z0, z1;
  if (!pass_region(p, &r1, &z0, &z1)) return cudaErrorInvalidValue;
  const dim3 blk(HB_X, HB_Y);
  Regions q = region_tiles<4, NV>(p, part == PASS_STR_LAYER ? std::min(r1 + 1, p.NR) : r1, z0, z1);
  if (!fits(q)) return cudaErrorInvalidValue;
  if (part == PASS_STR_RIM) {
    const long long rim = r1 < p.NR ? (long long)p.nth * ((q.rnzt + HB_Y - 1) / HB_Y) : 0;
    if (q.ends + rim > 0) hoist_rim<float, NV, MINB, false><<<(int)(q.ends + rim), blk, 0, s>>>(p, q, out);
    return cudaGetLastError();
  }
  if (part == PASS_STR_LAYER) q.ends = 0;
  const bool march = RUN && q.radial > 0 && can_run<float>(p);
  if (march) {
    if (part == PASS_VEL) launch_run<float, 2, true, true, true>(p, q, out, s);
    else launch_run<float, 2, false, true, true>(p, q, out, s);
  }
  const int grid = (int)q.ends + (march ? 0 : wave(q.radial, MINB));
  if (grid == 0) return cudaGetLastError();
  if (part == PASS_VEL) hoist_edge<float, NV, MINB, true, true, true><<<grid, blk, 0, s>>>(p, q, out);
  else hoist_edge<float, NV, MINB, false, true, true><<<grid, blk, 0, s>>>(p, q, out);
  return cudaGetLastError();
}

// three-way codes (every storage type)
template <typename T>
cudaError_t launch_split3(int code, const KParams &p, cudaStream_t s, cudaEvent_t *ev, int parts) {
  switch (code) {
    case 2304: return launch_split_t<T, 4, 4, 1, 4, 4, 3>(p, s, ev, parts);
    case 2305: return launch_split_t<T, 4, 5, 0, 4, 4, 3>(p, s, ev, parts);
    case 2314: return launch_split_t<T, 4, 4, 1, 2, 5, 4>(p, s, ev, parts);
    case 2315: return launch_split_t<T, 4, 5, 0, 2, 5, 4>(p, s, ev, parts);
    case 2324: return launch_split_t<T, 4, sizeof(T) == 4 ? 3 : 4, 2, 4, 3, 3>(p, s, ev, parts);
    case 2325: return launch_split_t<T, 4, 5, 0, 2, 4, 4>(p, s, ev, parts);
    case 2334: return launch_split_t<T, 4, 4, 1, 4, 3, 3>(p, s, ev, parts);
    case 2335: return launch_split_t<T, 4, 5, 0, 4, 3, 3>(p, s, ev, parts);
  }
  return cudaErrorInvalidValue;
}

template <typename T>
cudaError_t launch_hoist_st(int code, const KParams &p, cudaStream_t s, cudaEvent_t *ev, int parts) {
  switch (code) {
    case 2003: return launch_hoist_t<T, 4, 3, false>(p, s, ev, parts);
    case 2013: return launch_hoist_t<T, 4, 3, true>(p, s, ev, parts);
    case 2004: return launch_hoist_t<T, 4, 4, false>(p, s, ev, parts);
    case 2014: return launch_hoist_t<T, 4, 4, true>(p, s, ev, parts);
    case 2005: return launch_hoist_t<T, 4, 5, false>(p, s, ev, parts);
    case 2106: return launch_hoist_t<T, 2, 6, false>(p, s, ev, parts);
    case 2108: return launch_hoist_t<T, 2, 8, false>(p, s, ev, parts);
    case 2204: return launch_split_t<T, 4, 4, 0, 4, 0, 4>(p, s, ev, parts);
    case 2205: return launch_split_t<T, 4, 5, 0, 4, 0, 4>(p, s, ev, parts);
    case 2216: return launch_split_t<T, 2, 6, 0, 2, 0, 6>(p, s, ev, parts);
    case 2218: return launch_split_t<T, 2, 8, 0, 2, 0, 6>(p, s, ev, parts);
    case 2224: return launch_one_t<T, 4, 2, 4>(p, s, ev, parts);
    case 2225: return launch_one_t<T, 4, 2, 5>(p, s, ev, parts);
    case 2234: return launch_split_t<T, 4, 4, 0, 2, 0, 6>(p, s, ev, parts);
    case 2235: return launch_split_t<T, 4, 5, 0, 2, 0, 6>(p, s, ev, parts);
    case 2244: return launch_split_t<T, 4, 4, 0, 4, 0, 3>(p, s, ev, parts);
    case 2245: return launch_split_t<T, 4, 5, 0, 4, 0, 3>(p, s, ev, parts);
    case 2256: return launch_one_t<T, 2, 2, 5>(p, s, ev, parts);
    case 2258: return launch_split_t<T, 2, 8, 0, 2, 0, 4>(p, s, ev, parts);
    case 2264: return launch_split_t<T, 4, 4, 1, 2, 0, 4>(p, s, ev, parts);
    case 2265: return launch_split_t<T, 4, 5, 1, 2, 0, 4>(p, s, ev, parts);
    case 2274: return launch_split_t<T, 4, 4, 1, 4, 0, 3>(p, s, ev, parts);
    case 2275: return launch_split_t<T, 4, sizeof(T) == 4 ? 3 : 4, 2, 4, 0, 3, 3>(p, s, ev, parts);
    case 2284: return launch_split_t<T, 4, 4, 0, 4, 0, 3, 3>(p, s, ev, parts);
    case 2285: return launch_split_t<T, 4, 5, 0, 4, 0, 3, 3>(p, s, ev, parts);
    case 2294: return launch_split_t<T, 4, 4, 1, 2, 0, 4, 4>(p, s, ev, parts);
    case 2295: return launch_split_t<T, 4, 5, 1, 2, 0, 4, 4>(p, s, ev, parts);
  }
  return launch_split3<T>(code, p, s, ev, parts);
}

}  // namespace

void set_side_stream(const SideStream *ss) { g_side = ss; }

long long batch_blocks(const KParams &p) {
  const Regions q = regions<float, BATCH_NV, BATCH_NVE>(p);
  return q.ends + q.radial + q.interior;
}

cudaError_t launch_batch_split(int storage, bool vel, const KParams *cases, int n_cases, cudaStream_t s) {
  if (n_cases < 1) return cudaErrorInvalidValue;
  switch (storage * 2 + (vel ? 1 : 0)) {
    case 0: return launch_batch_t<float, false>(cases, n_cases, s);
    case 1: return launch_batch_t<float, true>(cases, n_cases, s);
    case 2: return launch_batch_t<__nv_bfloat16, false>(cases, n_cases, s);
    case 3: return launch_batch_t<__nv_bfloat16, true>(cases, n_cases, s);
    case 4: return launch_batch_t<__half, false>(cases, n_cases, s);
    case 5: return launch_batch_t<__half, true>(cases, n_cases, s);
  }
  return cudaErrorInvalidValue;
}

namespace {
// the stochastic rounding of the FP16-SR stores, element by element
__global__ void __launch_bounds__(256) sr_round_kernel(const float *x, const unsigned *dither, unsigned short *out,
                                                       long long n) {
  for (long long q = blockIdx.x * (long long)blockDim.x + threadIdx.x; q < n; q += (long long)gridDim.x * blockDim.x)
    out[q] = __half_as_ushort(sr_round(x[q], dither[q] & 0x1fffu));
}
}  // namespace

cudaError_t launch_sr_round(const float *x, const unsigned *dither, unsigned short *out, long long n, cudaStream_t s) {
  if (n <= 0) return cudaSuccess;
  const int grid = (int)std::min<long long>((n + 255) / 256, 152LL * 8);
  sr_round_kernel<<<grid, 256, 0, s>>>(x, dither, out, n);
  return cudaGetLastError();
}

cudaError_t launch_pass_edges(int code, int part, const KParams &p, const OutSet &out, cudaStream_t s) {
  return pass_edges4(code) ? launch_pass_edges_t<4, 3, true>(part, p, out, s) : launch_pass_edges_t<2, 4, false>(part, p, out, s);
}

cudaError_t launch_hoist(int storage, int code, const KParams &p, cudaStream_t s, cudaEvent_t *ev, int parts) {
  switch (storage) {
    case 0: return launch_hoist_st<float>(code, p, s, ev, parts);
    case 1: return launch_hoist_st<__nv_bfloat16>(code, p, s, ev, parts);
    case 2: return launch_hoist_st<__half>(code, p, s, ev, parts);
    case 3: return launch_split3<half_sr>(code, p, s, ev, parts);  // FP16 with stochastic rounding: 23xx
  }
  return cudaErrorInvalidValue;
}

}  // namespace cwell
