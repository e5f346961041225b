// neighbours.cu -- fixed-radius neighbour search of Eq. Nbd (Sec. 2.2) on a
// cell list: bounding boxes -> cell keys -> stable LSD radix sort (left out for a
// cloud in cell order) -> cell ranges and work queue -> a record per occupied cell
// -> hit bits of its candidates (a warp per cell or part of one) -> exclusive scan
// -> fill from the bits -> (row sort when the input order is not the cell order) ;
// cells that the bits' pool cannot hold are counted and filled a warp per particle.
// Plus the transpose map used by the apply adjoint.
#include <algorithm>
#include <climits>

#include "internal.cuh"

namespace mafp {

// ---------------------------------------------------------------- grid set-up
constexpr int kBoxThreads = 256;
constexpr int kBoxBlocks = 16384;   // bounding-box blocks over all clouds, beside one per cloud

// ------------------------------------------------ several clouds, one grid each
// Cloud b owns particles [off[b], off[b+1]) and cells [cell_base[b], cell_base[b+1])
// of the global cell numbering, with its own bounding box and cell edge, so
// neighbourhoods never cross clouds.  A single cloud is the case nb = 1.
struct CloudGrids {
  const GridDev *grids;      // [nb]
  const long long *cell_base;  // [nb + 1]
  int nb;
  const GridDev *all;        // ok flag and total cell count
};

// First particle of cloud b (off == nullptr: one cloud of n particles).
__device__ __forceinline__ long long cloud_begin(const long long *off, int b, int64_t n) {
  return off ? off[b] : (b == 0 ? 0 : (long long)n);
}

// First bounding-box block of cloud b: a block per cloud and one more per `chunk`
// particles, so that clouds of any sizes get blocks by their own size (by the mean size, a
// cloud of 10^6 particles beside 1000 of 100 had one block, and its search took 2247 us
// for 560).
__device__ __forceinline__ int box_first(const long long *off, int b, int64_t n, int64_t chunk) {
  return b + (int)(max(0LL, min(cloud_begin(off, b, n), (long long)n)) / chunk);
}

// Block box_first(b) + part reduces part `part` of cloud b: min / max of x, y, z, max h,
// count of non-finite entries; also records each particle's cloud.  Min and
// max are exact in the input's own type, so they are taken in it and widened
// once per block.
template <typename T>
__device__ __forceinline__ T lo_of(T a, T b) { return b < a ? b : a; }
template <typename T>
__device__ __forceinline__ T hi_of(T a, T b) { return b > a ? b : a; }

template <typename T>
__global__ void __launch_bounds__(kBoxThreads) k_cloud_bbox(const vec4_t<T> *pos, int64_t n,
                                                            const long long *off, int nb,
                                                            int64_t chunk, double *partial,
                                                            int32_t *cloud_id) {
  pdl_sync();
  int b = 0;   // the last cloud that begins at or before this block, 32 looked at together
  for (int b1 = nb; b1 - b > 1;) {
    const int step = (b1 - b + 31) >> 5, q = b + step * (int)(threadIdx.x & 31);
    const unsigned m = __ballot_sync(
        0xffffffffu, q == b || (q < b1 && box_first(off, q, n, chunk) <= (int)blockIdx.x));
    b += step * (31 - __clz(m));
    b1 = min(b1, b + step);
  }
  const int part = (int)blockIdx.x - box_first(off, b, n, chunk);
  const int parts = box_first(off, b + 1, n, chunk) - box_first(off, b, n, chunk);
  // offsets are checked in k_cloud_grid; clamping keeps every access in [0, n), and a
  // block that offsets out of order leave without a part reads nothing
  const long long lo = max(0LL, min(cloud_begin(off, b, n), (long long)n));
  const long long hi =
      part < 0 || part >= parts ? lo : max(lo, min(cloud_begin(off, b + 1, n), (long long)n));
  const T inf = T(INFINITY);
  T v[7] = {inf, inf, inf, -inf, -inf, -inf, T(0)};
  int bad = 0;
  for (long long i = lo + (long long)part * blockDim.x + threadIdx.x; i < hi;
       i += (long long)parts * blockDim.x) {
    if (nb > 1) cloud_id[i] = b;
    const vec4_t<T> p = ld4(pos + i);
    const bool ok = isfinite(p.x) && isfinite(p.y) && isfinite(p.z) && isfinite(p.w) && p.w > T(0);
    if (!ok) {
      ++bad;
      continue;
    }
    v[0] = lo_of(v[0], p.x); v[1] = lo_of(v[1], p.y); v[2] = lo_of(v[2], p.z);
    v[3] = hi_of(v[3], p.x); v[4] = hi_of(v[4], p.y); v[5] = hi_of(v[5], p.z);
    v[6] = hi_of(v[6], p.w);
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
#pragma unroll
    for (int k = 0; k < 3; ++k) v[k] = lo_of(v[k], __shfl_xor_sync(0xffffffffu, v[k], o));
#pragma unroll
    for (int k = 3; k < 7; ++k) v[k] = hi_of(v[k], __shfl_xor_sync(0xffffffffu, v[k], o));
    bad += __shfl_xor_sync(0xffffffffu, bad, o);
  }
  __shared__ T red[kBoxThreads / 32][7];
  __shared__ int red_bad[kBoxThreads / 32];
  if ((threadIdx.x & 31) == 0) {
    for (int k = 0; k < 7; ++k) red[threadIdx.x >> 5][k] = v[k];
    red_bad[threadIdx.x >> 5] = bad;
  }
  __syncthreads();
  if (threadIdx.x < 8) {
    const int k = threadIdx.x;
    double a;
    if (k < 7) {
      T r = red[0][k];
      for (int w = 1; w < kBoxThreads / 32; ++w)
        r = k < 3 ? lo_of(r, red[w][k]) : hi_of(r, red[w][k]);
      a = (double)r;
    } else {
      int s = 0;
      for (int w = 0; w < kBoxThreads / 32; ++w) s += red_bad[w];
      a = (double)s;
    }
    partial[(long long)blockIdx.x * 8 + k] = a;
  }
}

// One block folds a cloud's `parts` partials into its box.  Thread t takes value t & 7
// of partials t >> 3, + 32, ...: a warp reads 256 consecutive bytes, up to eight reads
// in flight.  (A warp per cloud with a lane per partial took 22 us for 1024 partials, one
// latency after another.)  Every thread of a block of 256 has to call it.
__device__ __forceinline__ void fold_cloud(const double *pb, int parts, double *box) {
  __shared__ double red[8][8];
  const int k = threadIdx.x & 7;
  const double none = k < 3 ? INFINITY : (k < 6 ? -INFINITY : 0.0);
  auto join = [&](double x, double y) { return k < 3 ? fmin(x, y) : (k < 7 ? fmax(x, y) : x + y); };
  double v = none;
#pragma unroll 8
  for (int q = threadIdx.x >> 3; q < parts; q += kBoxThreads / 8) v = join(v, pb[q * 8 + k]);
  v = join(v, __shfl_xor_sync(0xffffffffu, v, 8));
  v = join(v, __shfl_xor_sync(0xffffffffu, v, 16));
  if ((threadIdx.x & 31) < 8) red[threadIdx.x >> 5][k] = v;
  __syncthreads();
  if (threadIdx.x < 8) {
    for (int w = 1; w < kBoxThreads / 32; ++w) v = join(v, red[w][k]);
    box[k] = v;
  }
  __syncthreads();
}

__global__ void __launch_bounds__(kBoxThreads) k_cloud_fold(const double *partial, double *box,
                                                            const long long *off, int64_t n,
                                                            int64_t chunk) {
  pdl_sync();
  const int b = blockIdx.x, first = box_first(off, b, n, chunk);
  const int parts = box_first(off, b + 1, n, chunk) - first;
  partial += (long long)first * 8;
  box += (long long)b * 8;
  if (parts == 1) {
    if (threadIdx.x < 8) box[threadIdx.x] = partial[threadIdx.x];
    return;
  }
  fold_cloud(partial, parts, box);
}

// Cells of cloud b at edge c (>= max h of the cloud); 0 for an empty cloud.
__device__ double cloud_cells(const double v[8], double c, int dim[3]) {
  if (!(v[6] > 0.0)) {
    dim[0] = dim[1] = dim[2] = 1;
    return 0.0;
  }
  double cells = 1.0;
  for (int a = 0; a < 3; ++a) {
    const double d = floor((v[3 + a] - v[a]) / c) + 1.0;
    cells *= d;
    dim[a] = d < 2e9 ? (int)d : INT_MAX;
  }
  return cells;
}

// One block: the box of a single cloud (several are folded before), per-cloud
// grids from the folded boxes, the global cell numbering
// (exclusive scan of the clouds' cell counts) and the all-clouds flag.  The cell
// edge of every cloud starts strictly above its max h times edge_factor >= 1
// (so S_i lies in the 27 cells around i's cell) and grows uniformly when the
// total exceeds cap_cells.
__global__ void __launch_bounds__(kBoxThreads) k_cloud_grid(const double *partial, double *box,
                                                            const long long *off, int64_t n,
                                                            int nb, int64_t chunk,
                                                            GridDev *grids,
                                                            long long *cell_base, GridDev *all,
                                                            DevStatus *st, long long cap_cells,
                                                            double edge_factor) {
  pdl_sync();
  __shared__ double s_nonfinite, s_cells;
  __shared__ double s_scale;
  __shared__ int s_bad;
  __shared__ long long s_sum[kBoxThreads];
  if (threadIdx.x == 0) {
    s_nonfinite = 0.0;
    s_scale = 1.0;
    s_bad = (cloud_begin(off, 0, n) != 0 || cloud_begin(off, nb, n) != n) ? 1 : 0;
  }
  if (nb == 1) fold_cloud(partial, box_first(off, 1, n, chunk), box);
  __syncthreads();
  for (int b = threadIdx.x; b < nb; b += blockDim.x)
    if (cloud_begin(off, b + 1, n) < cloud_begin(off, b, n)) s_bad = 1;
  __syncthreads();
  if (s_bad) {
    // the offsets do not split [0, n) into consecutive ranges
    if (threadIdx.x == 0) {
      all->ok = 0;
      st->cells_identity = st->not_identity ? 0 : 1;
      set_error(st, MAFP_EINVAL, -1);
    }
    return;
  }
  for (int b = threadIdx.x; b < nb; b += blockDim.x) {
    const double bad = box[(long long)b * 8 + 7];
    if (bad > 0.0) atomicAdd(&s_nonfinite, bad);
  }
  __syncthreads();
  if (s_nonfinite > 0.0) {
    if (threadIdx.x == 0) {
      all->ok = 0;
      st->cells_identity = st->not_identity ? 0 : 1;
      st->n_nonfinite += (long long)s_nonfinite;
      set_error(st, MAFP_ENONFINITE, (long long)s_nonfinite);
    }
    return;
  }
  for (int it = 0; it < 64; ++it) {
    if (threadIdx.x == 0) s_cells = 0.0;
    __syncthreads();
    for (int b = threadIdx.x; b < nb; b += blockDim.x) {
      double v[8];
      for (int k = 0; k < 8; ++k) v[k] = box[(long long)b * 8 + k];
      int dim[3];
      const double c = v[6] * (1.0 + 1e-6) * edge_factor * s_scale;
      const double cells = cloud_cells(v, c, dim);
      GridDev &g = grids[b];
      for (int a = 0; a < 3; ++a) g.lo[a] = v[a] < INFINITY ? v[a] : 0.0;
      g.hmax = v[6];
      g.c = c;
      g.inv_c = v[6] > 0.0 ? 1.0 / c : 1.0;
      for (int a = 0; a < 3; ++a) g.dim[a] = dim[a];
      g.ncells = (long long)cells;
      g.ok = 1;
      atomicAdd(&s_cells, cells);
    }
    __syncthreads();
    const bool fits = s_cells <= (double)cap_cells;
    __syncthreads();
    if (fits) break;
    if (threadIdx.x == 0) s_scale *= cbrt(s_cells / (double)cap_cells) * 1.0001;
    __syncthreads();
  }
  // exclusive scan of the cell counts: thread t takes a contiguous span
  const int span = (nb + kBoxThreads - 1) / kBoxThreads;
  const int b0 = threadIdx.x * span, b1 = min(nb, b0 + span);
  long long part_sum = 0;
  for (int b = b0; b < b1; ++b) part_sum += grids[b].ncells;
  s_sum[threadIdx.x] = part_sum;
  __syncthreads();
  if (threadIdx.x == 0) {
    long long acc = 0;
    for (int t = 0; t < kBoxThreads; ++t) {
      const long long v = s_sum[t];
      s_sum[t] = acc;
      acc += v;
    }
  }
  __syncthreads();
  long long run = s_sum[threadIdx.x];
  for (int b = b0; b < b1; ++b) {
    cell_base[b] = run;
    run += grids[b].ncells;
  }
  if (threadIdx.x == 0) {
    long long acc = s_sum[kBoxThreads - 1];
    for (int b = (kBoxThreads - 1) * span; b < nb; ++b) acc += grids[b].ncells;
    cell_base[nb] = acc;
    all->ok = acc <= cap_cells ? 1 : 0;
    all->ncells = acc;
    all->c = grids[0].c;
    if (acc > cap_cells) set_error(st, MAFP_ECAPACITY, cap_cells);
    st->ncells = acc;
    st->cell_size = grids[0].c;
    st->not_identity = 0;     // k_hash clears / sets them when the keys are out of order
    st->cells_identity = 1;
  }
}

// ------------------------------------------------------------- radix sort
constexpr int kRadixThreads = 256;
constexpr int kRadixItems = 8;
constexpr int kRadixTile = kRadixThreads * kRadixItems;

// Cell of coordinate x on one axis, floor((x - lo) inv_c) in FP64 clamped to the grid.
// FP32 decides away from the cell faces: (x - lo) inv_c with the difference, 1/c and
// the product each rounded once is off by at most 3 x 2^-24 of itself (a fourth
// of that is to spare below), so the floor is certain unless a face lies nearer.
// The face at lo is none (x >= lo), nor is the grid's upper one (clamped there).
// The FP64 pipe has 1/64 of the FP32 rate: all particles on it, the kernel took
// 64 us on the 1M jet cloud, 21 us so (its 4.3M cells cleared beside).
template <typename T>
__device__ __forceinline__ uint32_t cell_on_axis(T x, double lo, double inv_c, int dim) {
  const float d = sizeof(T) == 4 ? (float)x - (float)lo : (float)((double)x - lo);
  const float fi = (float)inv_c, v = d * fi, f = floorf(v), err = 2.4e-7f * v + 1e-30f;
  const float top = (float)(dim - 1);
  if ((f > 0.0f && v - f <= err) || (f < top && f + 1.0f - v <= err) || !(v < 4194304.0f) ||
      !(fi > 1e-30f && fi < 1e30f)) {
    const double w = floor(((double)x - lo) * inv_c), t = (double)(dim - 1);
    return (uint32_t)(w < 0.0 ? 0.0 : (w > t ? t : w));
  }
  return (uint32_t)(f > top ? top : f);
}

template <typename T>
__device__ __forceinline__ uint32_t cell_key(const vec4_t<T> &p, int b, const CloudGrids &cg) {
  const GridDev &g = cg.grids[b];
  const uint32_t cx = cell_on_axis<T>(p.x, g.lo[0], g.inv_c, g.dim[0]);
  const uint32_t cy = cell_on_axis<T>(p.y, g.lo[1], g.inv_c, g.dim[1]);
  const uint32_t cz = cell_on_axis<T>(p.z, g.lo[2], g.inv_c, g.dim[2]);
  return (uint32_t)cg.cell_base[b] + (cz * (uint32_t)g.dim[1] + cy) * (uint32_t)g.dim[0] + cx;
}

// One block per radix tile (blocks beyond the tiles only help to clear the cells, of
// which a small sparse cloud has many more): the particles' cell keys, the tile's
// histogram of the first digit, and whether a key is below the one before it.  Clouds that are in
// cell order already (a time loop keeps them so) show it here, and the sort's
// passes and their scans are left out (100 us on the 1M jet cloud).  All blocks
// together also clear the cells and the work counters.
template <typename T>
__global__ void __launch_bounds__(kRadixThreads) k_hash(const vec4_t<T> *pos, int64_t n,
                                                        const int32_t *cloud_id, CloudGrids cg,
                                                        uint32_t *keys, int32_t *vals,
                                                        int32_t *hist, int tiles,
                                                        int32_t *cell_start, int32_t *cell_end,
                                                        int32_t *n_ucell, DevStatus *st) {
  pdl_sync();
  __shared__ int32_t cnt[256];
  __shared__ uint32_t last[kRadixItems + 1][kRadixThreads / 32];
  if (!cg.all->ok) return;
  const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
  cnt[tid] = 0;
  const int64_t base = (int64_t)blockIdx.x * kRadixTile;
  const bool tile = blockIdx.x < tiles;
  uint32_t key[kRadixItems];
#pragma unroll
  for (int c = 0; c < kRadixItems; ++c) {
    const int64_t i = base + c * kRadixThreads + tid;
    key[c] = 0xffffffffu;
    if (i < n) {
      key[c] = cell_key<T>(ld4(pos + i), cg.nb > 1 ? cloud_id[i] : 0, cg);
      keys[i] = key[c];
      vals[i] = (int32_t)i;
    }
    if (lane == 31) last[c][w] = key[c];
  }
  // the key before the tile's first one
  if (tid == 0)
    last[kRadixItems][0] =
        base > 0 && tile ? cell_key<T>(ld4(pos + base - 1), cg.nb > 1 ? cloud_id[base - 1] : 0, cg) : 0u;
  __syncthreads();
  bool out_of_order = false;
#pragma unroll
  for (int c = 0; c < kRadixItems; ++c) {
    uint32_t before = __shfl_up_sync(0xffffffffu, key[c], 1);
    if (lane == 0)
      before = w > 0 ? last[c][w - 1]
                     : (c > 0 ? last[c - 1][kRadixThreads / 32 - 1] : last[kRadixItems][0]);
    out_of_order |= key[c] < before;
    if (base + c * kRadixThreads + tid < n) atomicAdd(&cnt[key[c] & 255u], 1);
  }
  if (__syncthreads_or(out_of_order) && tid == 0) {
    st->not_identity = 1;
    st->cells_identity = 0;
  }
  if (tile) hist[(int64_t)tid * tiles + blockIdx.x] = cnt[tid];
  // the cells and the work counters (cell counts, overflow cells, the tickets of the
  // mask and fill kernels and the mask pool's counter)
  const long long nc = cg.all->ncells;
  if (blockIdx.x == 0 && tid < 8) n_ucell[tid] = 0;
  for (long long k = (long long)blockIdx.x * kRadixThreads + tid; k < nc;
       k += (long long)gridDim.x * kRadixThreads) {
    cell_start[k] = INT_MAX;
    cell_end[k] = 0;
  }
}

__global__ void __launch_bounds__(kRadixThreads) k_radix_hist(const uint32_t *keys, int64_t n,
                                                              int shift, int32_t *hist,
                                                              int tiles, const GridDev *g,
                                                              const DevStatus *st) {
  pdl_sync();
  if (!g->ok || !st->not_identity) return;
  __shared__ int32_t cnt[256];
  cnt[threadIdx.x] = 0;
  __syncthreads();
  const int64_t base = (int64_t)blockIdx.x * kRadixTile;
  for (int k = threadIdx.x; k < kRadixTile; k += kRadixThreads) {
    int64_t idx = base + k;
    if (idx < n) atomicAdd(&cnt[(keys[idx] >> shift) & 255u], 1);
  }
  __syncthreads();
  hist[(int64_t)threadIdx.x * tiles + blockIdx.x] = cnt[threadIdx.x];
}

__global__ void __launch_bounds__(kRadixThreads) k_radix_scatter(
    const uint32_t *kin, const int32_t *vin, uint32_t *kout, int32_t *vout, int64_t n, int shift,
    const long long *offs, int tiles, const GridDev *g, const DevStatus *st) {
  pdl_sync();
  if (!g->ok || !st->not_identity) return;
  __shared__ long long base_d[256];
  __shared__ int32_t wcnt[kRadixThreads / 32][256];
  __shared__ int32_t ctot[256];
  const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
  base_d[tid] = offs[(int64_t)tid * tiles + blockIdx.x];
  const unsigned lt = (1u << lane) - 1u;
  for (int c = 0; c < kRadixItems; ++c) {
    for (int k = tid; k < (kRadixThreads / 32) * 256; k += kRadixThreads) (&wcnt[0][0])[k] = 0;
    __syncthreads();
    const int64_t idx = (int64_t)blockIdx.x * kRadixTile + (int64_t)c * kRadixThreads + tid;
    const bool valid = idx < n;
    uint32_t key = valid ? kin[idx] : 0u;
    int32_t val = valid ? vin[idx] : 0;
    int d = valid ? (int)((key >> shift) & 255u) : 256;
    unsigned peers = __match_any_sync(0xffffffffu, d);
    int rank = __popc(peers & lt);
    if (valid && rank == 0) wcnt[w][d] = __popc(peers);
    __syncthreads();
    {
      int run = 0;
      for (int ww = 0; ww < kRadixThreads / 32; ++ww) {
        int t = wcnt[ww][tid];
        wcnt[ww][tid] = run;
        run += t;
      }
      ctot[tid] = run;
    }
    __syncthreads();
    if (valid) {
      long long p = base_d[d] + wcnt[w][d] + rank;
      kout[p] = key;
      vout[p] = val;
    }
    __syncthreads();
    base_d[tid] += ctot[tid];
    __syncthreads();
  }
}

// The whole sort of a small cloud in one block: the passes that its number of cells
// needs, each a histogram, a scan of it and a stable scatter in chunks of 1024.
// (Eight launches less; a launch costs the host ~3 us, which bounds the step of a
// cloud of a few thousand particles.)  Cell order of an unordered 3D cloud: 4096 particles
// 41 us, 8192 61 us; by passes over the whole GPU 8193 take 68 us, 16384 70 us.  The
// result is in keys_b / vals_b.
constexpr int64_t kSmallSort = 8192;
__global__ void __launch_bounds__(1024) k_sort_small(uint32_t *keys_a, int32_t *vals_a,
                                                     uint32_t *keys_b, int32_t *vals_b, int n,
                                                     const GridDev *g, const DevStatus *st) {
  pdl_sync();
  if (!g->ok || !st->not_identity) return;
  __shared__ int32_t base[256], wcnt[32][256];
  const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
  const unsigned lt = (1u << lane) - 1u;
  const unsigned long long top = (unsigned long long)(g->ncells - 1);
  uint32_t *kin = keys_a, *kout = keys_b;
  int32_t *vin = vals_a, *vout = vals_b;
  for (int shift = 0; shift == 0 || (shift < 32 && (top >> shift) != 0); shift += 8) {
    if (tid < 256) base[tid] = 0;
    __syncthreads();
    for (int k = tid; k < n; k += 1024) atomicAdd(&base[(kin[k] >> shift) & 255u], 1);
    __syncthreads();
    if (w == 0) {   // exclusive scan, eight digits per lane
      int c[8], sum = 0;
      for (int k = 0; k < 8; ++k) {
        c[k] = base[8 * lane + k];
        sum += c[k];
      }
      int inc = sum;
      for (int o = 1; o < 32; o <<= 1) {
        const int u = __shfl_up_sync(0xffffffffu, inc, o);
        if (lane >= o) inc += u;
      }
      int run = inc - sum;
      for (int k = 0; k < 8; ++k) {
        base[8 * lane + k] = run;
        run += c[k];
      }
    }
    for (int k0 = 0; k0 < n; k0 += 1024) {
      for (int k = tid; k < 32 * 256; k += 1024) (&wcnt[0][0])[k] = 0;
      __syncthreads();
      const int k = k0 + tid;
      const bool valid = k < n;
      const uint32_t key = valid ? kin[k] : 0u;
      const int32_t val = valid ? vin[k] : 0;
      const int d = valid ? (int)((key >> shift) & 255u) : 256;
      const unsigned peers = __match_any_sync(0xffffffffu, d);
      const int rank = __popc(peers & lt);
      if (valid && rank == 0) wcnt[w][d] = __popc(peers);
      __syncthreads();
      int total = 0;
      if (tid < 256)
        for (int ww = 0; ww < 32; ++ww) {
          const int t = wcnt[ww][tid];
          wcnt[ww][tid] = total;
          total += t;
        }
      __syncthreads();
      if (valid) {
        const int p = base[d] + wcnt[w][d] + rank;
        kout[p] = key;
        vout[p] = val;
      }
      __syncthreads();
      if (tid < 256) base[tid] += total;
    }
    __syncthreads();   // (the block's own writes are read in the next pass)
    uint32_t *tk = kin; kin = kout; kout = tk;
    int32_t *tv = vin; vin = vout; vout = tv;
  }
  if (kin != keys_b)
    for (int k = tid; k < n; k += 1024) {
      keys_b[k] = kin[k];
      vals_b[k] = vin[k];
    }
}

// --------------------------------------------------------- cell ranges
// Occupied cells go to the work queue in two groups, the ones holding at least
// kBigCell particles (3D cells at the usual h / dx) ahead of the rest, so the
// costly cells are taken first and the kernels end on cheap ones.
constexpr int kBigCell = 24;
// Slot of the cell with ticket t: the first n_ucell[0] tickets are the front
// group, the n_ucell[4] after them the back group (stored from slot n - 1 down).
__device__ __forceinline__ int cell_slot(int t, int nbig, int64_t n) {
  return t < nbig ? t : (int)(n - 1 - (t - nbig));
}
// Cell ranges, sorted positions, the cell order and the work queue.  A cloud in
// cell order is read from the unsorted keys (keys0) and its identity order written
// to svals.  The queue's slots are taken by two atomics per block of particles (one
// per warp, all on one address at 0.75 ns each, took 26 us on the 1M jet cloud).
constexpr int kCellThreads = 512;
template <typename T>
__global__ void __launch_bounds__(kCellThreads) k_cells(
    const uint32_t *keys, const uint32_t *keys0, int32_t *svals, int64_t n,
    const vec4_t<T> *pos, vec4_t<T> *spos, int32_t *cell_start, int32_t *cell_end,
    int32_t *ucell, int32_t *n_ucell, int32_t *order, const DevStatus *st, const GridDev *g) {
  pdl_sync();
  __shared__ int s_cnt[2][kCellThreads / 32 + 1];
  if (!g->ok) return;
  const bool moved = st->not_identity;
  const uint32_t *skeys = moved ? keys : keys0;
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  for (int64_t s0 = (int64_t)blockIdx.x * kCellThreads; s0 < n;
       s0 += (int64_t)gridDim.x * kCellThreads) {
    const int64_t s = s0 + threadIdx.x;
    bool head = false, big = false;
    uint32_t key = 0;
    if (s < n) {
      key = skeys[s];
      const int32_t i = moved ? svals[s] : (int32_t)s;
      if (!moved) svals[s] = i;
      st4(spos + s, ld4(pos + i));
      if (order) order[s] = i;
      head = s == 0 || skeys[s - 1] != key;
      big = head && s + kBigCell - 1 < n && skeys[s + kBigCell - 1] == key;
      if (head) cell_start[key] = (int32_t)s;
      if (s == n - 1 || skeys[s + 1] != key) cell_end[key] = (int32_t)(s + 1);
    }
    // the work queue of the mask and fill kernels, costly cells first: cells
    // of at least kBigCell particles fill the list from the front, the others
    // from the back (slot n - 1 - u; there are at most n cells)
    const unsigned mb = __ballot_sync(0xffffffffu, big);
    const unsigned ml = __ballot_sync(0xffffffffu, head && !big);
    if (lane == 0) {
      s_cnt[0][w] = __popc(mb);
      s_cnt[1][w] = __popc(ml);
    }
    __syncthreads();
    if (threadIdx.x < 2) {   // first slots of the warps' cells in either group
      int *c = s_cnt[threadIdx.x], total = 0;
      for (int k = 0; k < kCellThreads / 32; ++k) {
        const int v = c[k];
        c[k] = total;
        total += v;
      }
      const int first = total ? atomicAdd(n_ucell + 4 * threadIdx.x, total) : 0;
      for (int k = 0; k < kCellThreads / 32; ++k) c[k] += first;
    }
    __syncthreads();
    if (head) {
      const unsigned m = big ? mb : ml;
      const int64_t u0 = s_cnt[big ? 0 : 1][w] + __popc(m & ((1u << lane) - 1u));
      const int64_t u = big ? u0 : n - 1 - u0;
      ucell[2 * u] = (int32_t)key;
      ucell[2 * u + 1] = (int32_t)s;
    }
    __syncthreads();   // the counts are read before the next particles' overwrite them
  }
}

// --------------------------------------------------------- count / fill
__device__ __forceinline__ bool in_support64(double xi, double yi, double zi, double hi,
                                             double xj, double yj, double zj, double hj) {
  double dx = __dsub_rn(xj, xi), dy = __dsub_rn(yj, yi), dz = __dsub_rn(zj, zi);
  double d2 = __dadd_rn(__dadd_rn(__dmul_rn(dx, dx), __dmul_rn(dy, dy)), __dmul_rn(dz, dz));
  double r = __dmul_rn(__dadd_rn(hi, hj), 0.5);
  return d2 <= __dmul_rn(r, r);
}

// FP32 decision, retaken in FP64 within a 1e-5 relative band of the bound.
__device__ __forceinline__ bool in_support(const float4 &a, const float4 &b) {
  float dx = b.x - a.x, dy = b.y - a.y, dz = b.z - a.z;
  float d2 = (dx * dx + dy * dy) + dz * dz;
  float r = (a.w + b.w) * 0.5f;
  float r2 = r * r;
  float diff = d2 - r2;
  if (!(fabsf(diff) > 1e-5f * r2))   // (also where the squares overflow)
    return in_support64(a.x, a.y, a.z, a.w, b.x, b.y, b.z, b.w);
  return diff < 0.0f;
}
__device__ __forceinline__ bool in_support(const double4_16a &a, const double4_16a &b) {
  return in_support64(a.x, a.y, a.z, a.w, b.x, b.y, b.z, b.w);
}

constexpr int kNbrThreads = 128;
constexpr int kNbrSmemBytes = 32768;

// What the search needs of one occupied cell, in the order of the work queue
// (written by k_cell_table): its particles' sorted positions [s0, s0 + P), the
// candidates (the particles of the 27 cells around it, as nr non-empty runs of
// consecutive sorted positions: candidate c of run r, off_r <= c < off_(r+1), is
// sorted position c + delta_r), the power of two 2^-e that takes the cell edge
// into [1/2, 1), and where its hit words start in the mask pool (-1: the cell
// goes to the warp-per-particle kernels).
constexpr int kCellRec = 24;   // ints per record
enum { kRecS0 = 0, kRecP = 1, kRecTotal = 2, kRecRuns = 3, kRecPool = 4, kRecRun = 6 };

// Warp-per-particle count / fill (ballot compaction), for the occupied cells
// listed in sel[0 .. *n_sel): those that the mask kernel below cannot hold.  Few warps
// are at work on few dense cells, and the latency of the candidates' loads is their time:
// four are in flight (50000 particles in 64 cells, whole search: 80.8 ms one at a time,
// 69.2 ms so; the cell's record is in shared memory).
template <typename T, bool FILL>
__global__ void __launch_bounds__(kNbrThreads) k_nbr(
    const GridDev *all, const int32_t *table, const int32_t *sel, const int32_t *n_sel,
    const vec4_t<T> *spos, const int32_t *svals, int32_t *counts, const long long *row_ptr,
    int32_t *col, long long cap_nnz, int64_t n) {
  pdl_wait();
  using V = vec4_t<T>;
  constexpr int CAP = kNbrSmemBytes / sizeof(V);
  extern __shared__ __align__(16) unsigned char smem_raw[];
  V *cand = reinterpret_cast<V *>(smem_raw);
  __shared__ int rec[kCellRec];
  if (!all->ok) return;
  if (FILL && row_ptr[n] > cap_nnz) return;
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, nw = kNbrThreads / 32;
  const unsigned lt = (1u << lane) - 1u;
  const int nu = *n_sel;
  for (int cs = blockIdx.x; cs < nu; cs += gridDim.x) {
    if (threadIdx.x < kCellRec)
      rec[threadIdx.x] = table[(long long)sel[cs] * kCellRec + threadIdx.x];
    __syncthreads();
    const int s0 = rec[kRecS0], s1 = s0 + rec[kRecP], total = rec[kRecTotal];
    const int nr = rec[kRecRuns] & 255;
    const bool staged = total <= CAP;
    if (staged) {
      for (int r = 0; r < nr; ++r) {
        const int off = rec[kRecRun + 2 * r], d = rec[kRecRun + 2 * r + 1];
        const int end = r + 1 < nr ? rec[kRecRun + 2 * r + 2] : total;
        for (int c = off + threadIdx.x; c < end; c += kNbrThreads) cand[c] = ld4(spos + c + d);
      }
    }
    __syncthreads();
    for (int p = s0 + w; p < s1; p += nw) {
      const V xi = ld4(spos + p);
      long long base = 0;
      if (FILL) base = row_ptr[svals[p]];
      int cnt = 0;
      for (int r = 0; r < nr; ++r) {
        const int off = rec[kRecRun + 2 * r], d = rec[kRecRun + 2 * r + 1];
        const int lo = off + d;
        const int len = (r + 1 < nr ? rec[kRecRun + 2 * r + 2] : total) - off;
#pragma unroll 4
        for (int t0 = 0; t0 < len; t0 += 32) {
          const int t = t0 + lane;
          bool hit = false;
          if (t < len) {
            const V xj = staged ? cand[off + t] : ld4(spos + lo + t);
            hit = in_support(xi, xj);
          }
          const unsigned m = __ballot_sync(0xffffffffu, hit);
          if (FILL && hit) col[base + cnt + __popc(m & lt)] = svals[lo + t];
          cnt += __popc(m);
        }
      }
      if (!FILL && lane == 0) counts[svals[p]] = cnt;
    }
    __syncthreads();
  }
}

// ------------------------------------------------ warp-per-cell mask path
// Every particle of a cell shares the candidate set "27 cells around it",
// which is up to 9 runs of consecutive sorted positions (3 x-adjacent cells
// each).  k_cell_table writes each cell's runs once, a thread per cell.  The
// mask and fill kernels then take work items -- a cell, or one of `split` parts
// of its particles -- from a device work queue and handle each by one warp, with
// warp-level synchronisation only: a film cell (a dozen particles, ~4 candidate
// words) and a 3D cell (~40 particles, ~37 words) cost the warp in proportion
// to their work, and no block waits at a barrier for its slowest thread.  The
// mask kernel takes the candidates in windows of kWinWords words: a lane holds
// one candidate of each word in registers, the particles are broadcast one
// after another from shared memory, and a ballot gives the 32 bits of a
// (particle, word).  (With the particles in the lanes and the candidates
// broadcast, 10 floats per two candidates go to every lane: the 128 bytes per
// cycle that shared memory returns bound that form at 0.29 ms on the 1M jet
// cloud, whatever the arithmetic; here 5 floats go out per 256 tests.)  The fill
// kernel turns the bits back into column indices, so the tests run once.
//
// The test is one packed dot product.  With u = (x - x_ref) sc, x_ref a particle
// of the item's cell and sc the power of two that takes the cell edge c into
// [1/2, 1),
//   |u_j - u_i|^2 - (h_i + h_j)^2 / 4
//     = (|u_j|^2 - h_j^2/4) + (|u_i|^2 - h_i^2/4) - 2 u_i.u_j - (h_i/2) h_j,
// a sum and four fused multiply-adds per candidate (two candidates per packed
// FP32 instruction), against eleven operations for the difference form; its
// sign is the bit.
// FP32 evaluates it to 1.3e-5 (|u_i| <= 1, |u_j| <= 2 per axis, partial sums up
// to 28: ten roundings of at most 2^-24 each, and 1.3e-6 from the rounded
// u), so a value within kBand of zero is decided by the FP64 definition on the
// original positions instead -- for FP64 clouds too, whose tests all ran on
// the FP64 pipe before (2138 us against 63 us on the 60k jet cloud).  One word in
// 5000 needs that.  1M jet cloud: 302 us with candidates and differences from
// shared memory, 213 us so.
//
// The bits go to a pool, P rows of nwords (rounded up to 4) per cell (pool_words
// in all, kMaskWords per particle of the context's capacity on average): film
// cells need 4 words per particle, cells of an irregular cloud 60, and only what
// exceeds the pool takes the warp-per-particle kernels.  So does a cell that alone would
// take more than a 64th of the pool (or 1 MB, if that is more): a few such cells (a
// clump, a dense patch) would use it up, and the cells left over would crowd the heavy
// ones in those kernels (80k film particles with 120k in a dense patch, FP64: 584 to 752
// ms, as the cells came, 573 where only the patch's cells take them).
constexpr int kMaskThreads = 128;
constexpr int kMaskWarps = kMaskThreads / 32;
constexpr int kWinWords = 8;
constexpr int kMaskBlock = 64;   // particles prepared at a time
constexpr float kBand = 1.6e-5f;
// Words of a particle's row in the mask pool.
__host__ __device__ constexpr int row_words(int total) { return ((total + 127) >> 7) << 2; }

__host__ __device__ constexpr long long cell_limit(long long pool_words) {
  return pool_words / 64 > (1 << 18) ? pool_words / 64 : (1 << 18);
}

constexpr int kFillThreads = 128;
constexpr int kFillWarps = kFillThreads / 32;
constexpr int kFillWinWords = 16;   // candidate words of one fill window
constexpr int kFillRec = kFillWinWords + 2;   // records of one particle, with pad
// Work items: the cells of the front group in 2^front parts each, then those of
// the back group in 2^back parts.
struct Split {
  int front, back;
};
// Particles [*p0, *p0 + *np) of the cell's P that part `c` of 2^log holds.
__device__ __forceinline__ void item_part(int P, int log, int c, int *p0, int *np) {
  const int q = (P + (1 << log) - 1) >> log;
  *p0 = min(P, c * q);
  *np = min(P, *p0 + q) - *p0;
}

// One thread per occupied cell (queue position t): its record.
__global__ void __launch_bounds__(128) k_cell_table(
    CloudGrids cg, const int32_t *ucell, int32_t *n_ucell, const int32_t *cell_start,
    const int32_t *cell_end, int32_t *table, long long pool_words, int32_t *overflow,
    int64_t n) {
  pdl_sync();
  if (!cg.all->ok) return;
  const int lane = threadIdx.x & 31;
  const int nbig = n_ucell[0], nu = nbig + n_ucell[4];
  unsigned long long *pool = reinterpret_cast<unsigned long long *>(n_ucell + 6);
  for (int t0 = (blockIdx.x * blockDim.x + threadIdx.x) & ~31; t0 < nu;
       t0 += gridDim.x * blockDim.x) {
    const int t = t0 + lane;
    const bool in = t < nu;
    int rec[kCellRec];
#pragma unroll
    for (int k = 0; k < kCellRec; ++k) rec[k] = 0;
    long long need = 0;
    if (in) {
      const int cb = cell_slot(t, nbig, n);
      const int key = ucell[2 * cb], s0 = ucell[2 * cb + 1];
      int b0 = 0, b1 = cg.nb;   // cloud with cell_base[b] <= key < cell_base[b + 1]
      while (b1 - b0 > 1) {
        const int mid = (b0 + b1) >> 1;
        if (cg.cell_base[mid] <= key) b0 = mid; else b1 = mid;
      }
      const GridDev &g = cg.grids[b0];
      const int local = key - (int)cg.cell_base[b0];
      const int dx_ = g.dim[0], dy_ = g.dim[1], dz_ = g.dim[2];
      const int row = local / dx_, cx = local - row * dx_;
      const int cz = row / dy_, cy = row - cz * dy_;
      // run r (dz = r/3-1, dy = r%3-1) covers cells key-1..key+1 of that (y, z)
      // row of the key's own cloud grid, clipped to that grid
      int lo[9], hi[9];
#pragma unroll
      for (int r = 0; r < 9; ++r) {
        const int ddz = r / 3 - 1, ddy = r % 3 - 1;
        lo[r] = INT_MAX;
        hi[r] = 0;
        if (cz + ddz >= 0 && cz + ddz < dz_ && cy + ddy >= 0 && cy + ddy < dy_) {
          const int base = key + (ddz * dy_ + ddy) * dx_;
#pragma unroll
          for (int a = -1; a <= 1; ++a)
            if (cx + a >= 0 && cx + a < dx_) {
              lo[r] = min(lo[r], cell_start[base + a]);
              hi[r] = max(hi[r], cell_end[base + a]);
            }
        }
      }
      int total = 0, nr = 0;
#pragma unroll
      for (int r = 0; r < 9; ++r)
        if (hi[r] > lo[r]) {
#pragma unroll
          for (int k = 0; k <= r; ++k)   // (static indices: rec stays in registers)
            if (k == nr) {
              rec[kRecRun + 2 * k] = total;
              rec[kRecRun + 2 * k + 1] = lo[r] - total;
            }
          total += hi[r] - lo[r];
          ++nr;
        }
      const int P = cell_end[key] - s0;
      int e;   // edges beyond 2^+-120 leave FP32's range: the warp-per-particle kernels
      frexp(g.c, &e);
      rec[kRecS0] = s0;
      rec[kRecP] = P;
      rec[kRecTotal] = total;
      rec[kRecRuns] = nr | ((max(-120, min(120, e)) + 128) << 8);
      need = (long long)row_words(total) * P;
      if (abs(e) > 120 || need > cell_limit(pool_words)) need = 0;
    }
    // the warp's share of the pool, by one atomic
    long long inc = need;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const long long u = __shfl_up_sync(0xffffffffu, inc, o);
      if (lane >= o) inc += u;
    }
    long long base = 0;
    if (lane == 31) base = (long long)atomicAdd(pool, (unsigned long long)inc);
    base = __shfl_sync(0xffffffffu, base, 31) + inc - need;
    if (!in) continue;
    if (need == 0 || base + need > pool_words) {
      // an edge out of range, a cell beyond its share, or the pool is used up
      base = -1;
      overflow[atomicAdd(n_ucell + 1, 1)] = t;
    }
    rec[kRecPool] = (int)(unsigned)(base & 0xffffffffll);
    rec[kRecPool + 1] = (int)(base >> 32);
    int4 *out = reinterpret_cast<int4 *>(table + (long long)t * kCellRec);
#pragma unroll
    for (int k = 0; k < kCellRec / 4; ++k)
      out[k] = make_int4(rec[4 * k], rec[4 * k + 1], rec[4 * k + 2], rec[4 * k + 3]);
  }
}

// The work queue as one warp walks it: an atomic ticket per item; the next
// ticket is drawn and the next item's record loaded (one int per lane) while the
// present item is worked on.
struct ItemWalk {
  const int32_t *table;
  int32_t *ticket;
  Split sp;
  int nfront, items, lane;   // items of the front group, of both
  int at, ahead;             // present item, next ticket (lane 0)
  int rec_next;

  __device__ __forceinline__ int load(int item) const {
    const int cell = item < nfront ? item >> sp.front
                                   : (nfront >> sp.front) + ((item - nfront) >> sp.back);
    return item < items && lane < kCellRec ? table[(long long)cell * kCellRec + lane] : 0;
  }
  __device__ __forceinline__ int draw() const { return lane == 0 ? atomicAdd(ticket, 1) : 0; }
  __device__ __forceinline__ void start(const int32_t *tab, int32_t *tk, int nbig, int nlight,
                                        Split split, int ln) {
    table = tab;
    ticket = tk;
    sp = split;
    lane = ln;
    nfront = nbig << sp.front;
    items = nfront + (nlight << sp.back);
    at = __shfl_sync(0xffffffffu, draw(), 0);
    ahead = draw();
    rec_next = load(at);
  }
  // The present item's record (one int per lane), its first particle's sorted
  // position and count; false at the end.
  __device__ __forceinline__ bool next(int *rec, int *s0, int *p0, int *P) {
    if (at >= items) return false;
    *rec = rec_next;
    const bool f = at < nfront;
    const int log = f ? sp.front : sp.back, part = (f ? at : at - nfront) & ((1 << log) - 1);
    item_part(__shfl_sync(0xffffffffu, *rec, kRecP), log, part, p0, P);
    *s0 = __shfl_sync(0xffffffffu, *rec, kRecS0) + *p0;
    at = __shfl_sync(0xffffffffu, ahead, 0);
    ahead = draw();
    rec_next = load(at);
    return true;
  }
};

// Sorted positions of candidates c0 + lane + 32 u, u = 0..3 (those past the
// last candidate give the last one's); r is the run that holds c0 or an earlier
// one, moved on to c0's.
__device__ __forceinline__ void candidates4(int rec, int nr, int total, int c0, int lane, int *r,
                                            int (&sp)[4]) {
  while (*r + 1 < nr && __shfl_sync(0xffffffffu, rec, kRecRun + 2 * (*r + 1)) <= c0) ++*r;
  const int d0 = __shfl_sync(0xffffffffu, rec, kRecRun + 2 * *r + 1);
  int d[4] = {d0, d0, d0, d0}, c[4];
#pragma unroll
  for (int u = 0; u < 4; ++u) c[u] = min(c0 + lane + 32 * u, total - 1);
  for (int k = *r + 1; k < nr; ++k) {
    const int o = __shfl_sync(0xffffffffu, rec, kRecRun + 2 * k);
    if (o >= c0 + 128) break;
    const int dk = __shfl_sync(0xffffffffu, rec, kRecRun + 2 * k + 1);
#pragma unroll
    for (int u = 0; u < 4; ++u) d[u] = c[u] >= o ? dk : d[u];
  }
#pragma unroll
  for (int u = 0; u < 4; ++u) sp[u] = c[u] + d[u];
}

// (x - ref) sc in FP32: the subtraction in the input's own type, sc exact.
__device__ __forceinline__ float4 local_of(const float4 &v, const float4 &r, float sc) {
  return make_float4((v.x - r.x) * sc, (v.y - r.y) * sc, (v.z - r.z) * sc, v.w * sc);
}
__device__ __forceinline__ float4 local_of(const double4_16a &v, const double4_16a &r, float sc) {
  return make_float4((float)(v.x - r.x) * sc, (float)(v.y - r.y) * sc, (float)(v.z - r.z) * sc,
                     (float)v.w * sc);
}
// |u|^2 - h^2/4
__device__ __forceinline__ float local_c(const float4 &u) {
  return fmaf(u.x, u.x, fmaf(u.y, u.y, fmaf(u.z, u.z, -0.25f * u.w * u.w)));
}

// The tests of particles [0, np) (prepared in part / pcc) against the lanes'
// candidates of NP pairs of words (d = the pairs' staged values), 32 particles at
// a time: their rows' words go to rows (nwp words each) from word w0 on, the
// hits of this lane's particles k = lane, lane + 32 are added to cnt.
template <int NP, typename Retake>
__device__ __forceinline__ void test_window(const float2 (&X)[kWinWords / 2],
                                            const float2 (&Y)[kWinWords / 2],
                                            const float2 (&Z)[kWinWords / 2],
                                            const float2 (&H)[kWinWords / 2],
                                            const float2 (&C)[kWinWords / 2], int np,
                                            const float4 *part, const float *pcc,
                                            uint32_t (*res)[kWinWords + 4], uint32_t *rows,
                                            int nwp, int lane, int (&cnt)[kMaskBlock / 32],
                                            Retake &&retake) {
#pragma unroll
  for (int half = 0; half < kMaskBlock / 32; ++half) {
    if (32 * half >= np) break;
    const int kn = min(32, np - 32 * half);
#pragma unroll 1   // (two particles side by side cost a block per SM: 231 against 214 us)
    for (int k = 0; k < kn; ++k) {
      const float4 f = part[32 * half + k];
      const float cc = pcc[32 * half + k];
      float2 d[NP];
      float near = 1e30f;
      uint32_t b[2 * NP];
#pragma unroll
      for (int i = 0; i < NP; ++i) {
        d[i] = __fadd2_rn(C[i], make_float2(cc, cc));
        d[i] = __ffma2_rn(X[i], make_float2(f.x, f.x), d[i]);
        d[i] = __ffma2_rn(Y[i], make_float2(f.y, f.y), d[i]);
        d[i] = __ffma2_rn(Z[i], make_float2(f.z, f.z), d[i]);
        d[i] = __ffma2_rn(H[i], make_float2(f.w, f.w), d[i]);
        near = fminf(near, fminf(fabsf(d[i].x), fabsf(d[i].y)));
        b[2 * i] = __ballot_sync(0xffffffffu, d[i].x < 0.0f);
        b[2 * i + 1] = __ballot_sync(0xffffffffu, d[i].y < 0.0f);
      }
      if (__any_sync(0xffffffffu, near <= kBand)) retake(32 * half + k, d, b);
      if (lane == 0) {
#pragma unroll
        for (int i = 0; i < NP; i += 2)
          *reinterpret_cast<uint4 *>(&res[k][2 * i]) =
              make_uint4(b[2 * i], b[2 * i + 1], b[2 * i + 2], b[2 * i + 3]);
      }
    }
    __syncwarp();
    if (lane < kn) {
#pragma unroll
      for (int i = 0; i < NP; i += 2) {
        const uint4 v = *reinterpret_cast<const uint4 *>(&res[lane][2 * i]);
        cnt[half] += __popc(v.x) + __popc(v.y) + __popc(v.z) + __popc(v.w);
        *reinterpret_cast<uint4 *>(rows + (long long)(32 * half + lane) * nwp + 2 * i) = v;
      }
    }
    __syncwarp();   // the words are read before the next particles overwrite them
  }
}

template <typename T>
__global__ void __launch_bounds__(kMaskThreads) k_nbr_mask(
    const GridDev *all, const int32_t *table, int32_t *n_ucell, const vec4_t<T> *spos,
    const int32_t *svals, int32_t *counts, uint32_t *mask, Split split) {
  pdl_wait();
  using V = vec4_t<T>;
  // prepared particles (-2 u, -h/2) and |u|^2 - h^2/4; the words of 32 particles
  __shared__ float4 s_part[kMaskWarps][kMaskBlock];
  __shared__ float s_cc[kMaskWarps][kMaskBlock];
  __shared__ __align__(16) uint32_t s_res[kMaskWarps][32][kWinWords + 4];
  const int lane = threadIdx.x & 31, wp = threadIdx.x >> 5;
  if (!all->ok) return;
  ItemWalk walk;
  walk.start(table, n_ucell + 2, n_ucell[0], n_ucell[4], split, lane);
  int rec, s0, p0, P;
  while (walk.next(&rec, &s0, &p0, &P)) {
    const long long pool =
        ((long long)__shfl_sync(0xffffffffu, rec, kRecPool + 1) << 32) |
        (unsigned)__shfl_sync(0xffffffffu, rec, kRecPool);
    if (pool < 0 || P == 0) continue;   // the warp-per-particle kernel's, or no particles
    const int total = __shfl_sync(0xffffffffu, rec, kRecTotal);
    const int nre = __shfl_sync(0xffffffffu, rec, kRecRuns), nr = nre & 255;
    const float sc = __int_as_float((127 + 128 - (nre >> 8)) << 23);
    const int nwp = row_words(total);
    uint32_t *mrow = mask + pool + (long long)nwp * p0;
    const V ref = ld4(spos + s0);
    for (int pb = 0; pb < P; pb += kMaskBlock) {
      const int np = min(kMaskBlock, P - pb);
      __syncwarp();   // the previous particles are read
      for (int q = lane; q < np; q += 32) {
        const float4 u = local_of(ld4(spos + s0 + pb + q), ref, sc);
        s_part[wp][q] = make_float4(-2.0f * u.x, -2.0f * u.y, -2.0f * u.z, -0.5f * u.w);
        s_cc[wp][q] = local_c(u);
      }
      __syncwarp();
      int cnt[kMaskBlock / 32] = {0, 0}, run = 0;
      for (int w0 = 0; w0 < nwp; w0 += kWinWords) {
        float2 X[kWinWords / 2], Y[kWinWords / 2], Z[kWinWords / 2], H[kWinWords / 2],
            C[kWinWords / 2];
        const int run0 = run;
#pragma unroll
        for (int g = 0; g < kWinWords; g += 4) {
          if (w0 + g >= nwp) break;
          int sp[4];
          candidates4(rec, nr, total, (w0 + g) * 32, lane, &run, sp);
          V v[4];
#pragma unroll
          for (int u = 0; u < 4; ++u) v[u] = ld4(spos + sp[u]);
#pragma unroll
          for (int u = 0; u < 4; ++u) {
            const float4 x = local_of(v[u], ref, sc);
            // a slot past the last candidate is far from everything
            const float c = (w0 + g + u) * 32 + lane < total ? local_c(x) : 1e30f;
            const int i = (g + u) / 2;
            if (u % 2 == 0) {
              X[i].x = x.x; Y[i].x = x.y; Z[i].x = x.z; H[i].x = x.w; C[i].x = c;
            } else {
              X[i].y = x.x; Y[i].y = x.y; Z[i].y = x.z; H[i].y = x.w; C[i].y = c;
            }
          }
        }
        // pairs at the bound: the FP64 definition decides
        auto retake = [&](int k, auto &d, auto &b) {
          const V xi = ld4(spos + s0 + pb + k);
          int r = run0;
#pragma unroll
          for (int g = 0; g < kWinWords; g += 4) {
            if (g >= (int)(sizeof(d) / sizeof(float))) break;
            if (w0 + g >= nwp) break;
            int sp[4];
            candidates4(rec, nr, total, (w0 + g) * 32, lane, &r, sp);
#pragma unroll
            for (int u = 0; u < 4; ++u) {
              const float dv = u % 2 ? d[(g + u) / 2].y : d[(g + u) / 2].x;
              bool hit = dv < 0.0f;
              if (fabsf(dv) <= kBand) {
                const V xj = ld4(spos + sp[u]);
                hit = in_support64(xi.x, xi.y, xi.z, xi.w, xj.x, xj.y, xj.z, xj.w);
              }
              b[g + u] = __ballot_sync(0xffffffffu, hit);
            }
          }
        };
        uint32_t *rows = mrow + (long long)nwp * pb + w0;
        if (nwp - w0 > 4)
          test_window<4>(X, Y, Z, H, C, np, s_part[wp], s_cc[wp], s_res[wp], rows, nwp, lane,
                         cnt, retake);
        else
          test_window<2>(X, Y, Z, H, C, np, s_part[wp], s_cc[wp], s_res[wp], rows, nwp, lane,
                         cnt, retake);
      }
#pragma unroll
      for (int half = 0; half < kMaskBlock / 32; ++half)
        if (32 * half + lane < np) counts[svals[s0 + pb + 32 * half + lane]] = cnt[half];
    }
  }
}

// Fill pass for the mask kernel's items, also one warp per item from a work
// queue.  The item's particles go in chunks of 32; for each window of
// kFillWinWords candidate words each lane loads its candidates' original indices
// into registers and, holding one particle, that particle's hit words
// (coalesced) with the place in the row where each word's first hit goes; then
// the chunk's rows are expanded one particle at a time: one candidate per lane,
// its place from a popcount of the lower hits, coalesced stores.  Only that one
// popcount per (particle, word) is left in the expansion (a warp's POPC takes 8
// cycles of the issuing scheduler's unit, measured), and words are walked in
// groups of four up to the window's last one, so film cells (4 words) do not
// pay for a 16-word window: 382 -> 184 us on the 1M jet cloud.  Rows come out ascending when the cloud is in cell
// order (candidates are runs of consecutive sorted positions, ascending).
__global__ void __launch_bounds__(kFillThreads) k_nbr_fill(
    const GridDev *all, const int32_t *table, int32_t *n_ucell, const int32_t *svals,
    const uint32_t *mask, Split split, const long long *row_ptr, int32_t *col, long long cap_nnz,
    int64_t n, int64_t *nnz_dev, DevStatus *st) {
  pdl_wait();
  __shared__ __align__(16) uint2 srec[kFillWarps][32][kFillRec];     // (hit word, place)
  if (!all->ok) return;
  const long long nnz = row_ptr[n];
  if (blockIdx.x == 0 && threadIdx.x == 0) {
    st->nnz = nnz;
    if (nnz_dev) *nnz_dev = nnz;
    if (nnz > cap_nnz) set_error(st, MAFP_ECAPACITY, nnz);
  }
  if (nnz > cap_nnz) return;
  const int lane = threadIdx.x & 31;
  const unsigned lt = (1u << lane) - 1u, bit = 1u << lane;
  uint2(*wr)[kFillRec] = srec[threadIdx.x >> 5];
  ItemWalk walk;
  walk.start(table, n_ucell + 3, n_ucell[0], n_ucell[4], split, lane);
  int rec, s0, part, P;
  while (walk.next(&rec, &s0, &part, &P)) {
    const long long pool =
        ((long long)__shfl_sync(0xffffffffu, rec, kRecPool + 1) << 32) |
        (unsigned)__shfl_sync(0xffffffffu, rec, kRecPool);
    if (pool < 0 || P == 0) continue;
    const int total = __shfl_sync(0xffffffffu, rec, kRecTotal);
    const int nr = __shfl_sync(0xffffffffu, rec, kRecRuns) & 255;
    const int nwp = row_words(total);
    const uint32_t *mrow = mask + pool + (long long)nwp * part;
    for (int p0 = 0; p0 < P; p0 += 32) {
      const int np = min(32, P - p0);
      const int q = p0 + lane;
      const long long rs = lane < np ? row_ptr[svals[s0 + q]] : 0;
      int at = 0, run = 0;
      for (int w0 = 0; w0 < nwp; w0 += kFillWinWords) {
        const int nw = min(nwp - w0, kFillWinWords);
        int32_t cv[kFillWinWords];   // this lane's candidate of every word of the window
        __syncwarp();                // the previous window's reads are done
#pragma unroll
        for (int g = 0; g < kFillWinWords; g += 4) {
          if (g >= nw) break;
          int sp[4];
          const uint4 m4 = lane < np ? *reinterpret_cast<const uint4 *>(
                                           mrow + (long long)q * nwp + w0 + g)
                                     : make_uint4(0u, 0u, 0u, 0u);
          const uint32_t m[4] = {m4.x, m4.y, m4.z, m4.w};
          candidates4(rec, nr, total, (w0 + g) * 32, lane, &run, sp);
#pragma unroll
          for (int u = 0; u < 4; ++u) cv[g + u] = svals[sp[u]];
#pragma unroll
          for (int u = 0; u < 4; ++u) {
            wr[lane][g + u] = make_uint2(m[u], (unsigned)at);
            at += __popc(m[u]);
          }
        }
        __syncwarp();
        for (int k = 0; k < np; ++k) {
          int32_t *crow = col + __shfl_sync(0xffffffffu, rs, k);
          const uint4 *rk = reinterpret_cast<const uint4 *>(wr[k]);
#pragma unroll
          for (int g = 0; g < kFillWinWords / 4; ++g) {
            if (4 * g >= nw) break;
            const uint4 a = rk[2 * g], b = rk[2 * g + 1];
            if (a.x & bit) crow[a.y + __popc(a.x & lt)] = cv[4 * g];
            if (a.z & bit) crow[a.w + __popc(a.z & lt)] = cv[4 * g + 1];
            if (b.x & bit) crow[b.y + __popc(b.x & lt)] = cv[4 * g + 2];
            if (b.z & bit) crow[b.w + __popc(b.z & lt)] = cv[4 * g + 3];
          }
        }
      }
    }
  }
}

// Rows come out ascending in cell order; when the input order differs from the
// cell order each row is sorted, one warp per row, by a bitonic network.  Rows of
// up to 512 entries sort in registers (E consecutive entries per lane: strides
// below E are compare-exchanges between a lane's own registers, the others one
// shuffle per entry; 120 shuffles for 256 entries), longer ones in shared
// memory (36 passes of loads and stores over 256 entries, which all rows used to
// take).  200k random particles, 170 entries per row: 1800 us in shared
// memory, 214 us so.
constexpr int kSortWarps = 4;
constexpr int kSortBuf = kMaxRowSort;
__host__ __device__ constexpr int sort_pad(int i) { return i + (i >> 5); }   // bank of entry i
static_assert(sort_pad(511) < kSortBuf, "register rows leave through the shared buffer");

template <int E>
__device__ __forceinline__ void sort_row(int32_t *row, int len, int lane, int32_t *buf) {
  int v[E];
#pragma unroll
  for (int e = 0; e < E; ++e) v[e] = e * 32 + lane < len ? row[e * 32 + lane] : INT_MAX;
  // entry i = lane E + e (any start order will do)
#pragma unroll
  for (int k = 2; k <= 32 * E; k <<= 1) {
#pragma unroll
    for (int j = k >> 1; j > 0; j >>= 1) {
      if (j >= E) {
        // the pair's lower entry keeps the minimum where bit k of the index is clear
        const bool keep_min = ((lane & (j / E)) == 0) == ((lane & (k / E)) == 0);
#pragma unroll
        for (int e = 0; e < E; ++e) {
          const int o = __shfl_xor_sync(0xffffffffu, v[e], j / E);
          v[e] = keep_min ? min(v[e], o) : max(v[e], o);
        }
      } else {
#pragma unroll
        for (int e = 0; e < E; ++e)
          if ((e & j) == 0) {
            const bool up = k >= E ? (lane & (k / E)) == 0 : (e & k) == 0;
            const int a = v[e], b = v[e + j];
            v[e] = up ? min(a, b) : max(a, b);
            v[e + j] = up ? max(a, b) : min(a, b);
          }
      }
    }
  }
  if constexpr (E > 1) {
    __syncwarp();   // the buffer's previous row is read
#pragma unroll
    for (int e = 0; e < E; ++e) buf[sort_pad(lane * E + e)] = v[e];
    __syncwarp();
#pragma unroll
    for (int e = 0; e < E; ++e) v[e] = buf[sort_pad(e * 32 + lane)];
  }
#pragma unroll
  for (int e = 0; e < E; ++e)
    if (e * 32 + lane < len) row[e * 32 + lane] = v[e];
}

__global__ void __launch_bounds__(kSortWarps * 32) k_rowsort(const long long *row_ptr,
                                                             int32_t *col, int64_t n,
                                                             long long cap_nnz,
                                                             DevStatus *st, const GridDev *g) {
  pdl_sync();
  if (!g->ok || !st->not_identity) return;
  if (row_ptr[n] > cap_nnz) return;
  __shared__ int32_t buf[kSortWarps][kSortBuf];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  int32_t *a = buf[w];
  for (int64_t i = (int64_t)blockIdx.x * kSortWarps + w; i < n;
       i += (int64_t)gridDim.x * kSortWarps) {
    const long long b = row_ptr[i];
    const int len = (int)(row_ptr[i + 1] - b);
    if (len > kMaxRowSort) {
      if (lane == 0) set_error(st, MAFP_ECAPACITY, len);
      continue;
    }
    if (len <= 512) {
      int32_t *row = col + b;
      if (len <= 32) sort_row<1>(row, len, lane, a);
      else if (len <= 64) sort_row<2>(row, len, lane, a);
      else if (len <= 128) sort_row<4>(row, len, lane, a);
      else if (len <= 256) sort_row<8>(row, len, lane, a);
      else sort_row<16>(row, len, lane, a);
      continue;
    }
    int P = 1;
    while (P < len) P <<= 1;
    __syncwarp();
    for (int t = lane; t < P; t += 32) a[t] = t < len ? col[b + t] : INT_MAX;
    __syncwarp();
    for (int k = 2; k <= P; k <<= 1)
      for (int j = k >> 1; j > 0; j >>= 1) {
        for (int t = lane; t < P; t += 32) {
          int u = t ^ j;
          if (u > t) {
            int x = a[t], y = a[u];
            bool asc = (t & k) == 0;
            if ((x > y) == asc) {
              a[t] = y;
              a[u] = x;
            }
          }
        }
        __syncwarp();
      }
    for (int t = lane; t < len; t += 32) col[b + t] = a[t];
    __syncwarp();
  }
}

// tloc[e] = position of i inside row j for the entry e = (i, j).
__global__ void k_tmap(const long long *row_ptr, const int32_t *col, int64_t n, uint16_t *tloc,
                       DevStatus *st) {
  pdl_sync();
  const int lane = threadIdx.x & 31;
  const int64_t wid = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int64_t nwarps = ((int64_t)gridDim.x * blockDim.x) >> 5;
  for (int64_t i = wid; i < n; i += nwarps) {
    const long long b = row_ptr[i], e1 = row_ptr[i + 1];
    for (long long e = b + lane; e < e1; e += 32) {
      const int j = col[e];
      long long lo = row_ptr[j], hi = row_ptr[j + 1];
      const long long rb = lo;
      if (hi - rb > 65535) {
        set_error(st, MAFP_ECAPACITY, hi - rb);
        continue;
      }
      while (lo < hi) {
        long long mid = (lo + hi) >> 1;
        if (col[mid] < i) lo = mid + 1; else hi = mid;
      }
      tloc[e] = (uint16_t)(lo - rb);
    }
  }
}

// ------------------------------------------------------------------ host side
// A1: grids, cell keys, stable radix sort, cell ranges, sorted positions and
// (optionally) the cell order.  On return the sorted indices are in *svals, the
// sorted positions in the context's spos.
template <typename T>
static int sort_into_cells_t(mafp_ctx *ctx, int64_t n, int nb, const long long *cloud_off,
                             const void *pos_h, int32_t *order, const int32_t **svals,
                             cudaStream_t s) {
  using V = vec4_t<T>;
  const V *pos = reinterpret_cast<const V *>(pos_h);
  const int sms = sm_count();
  // particles per bounding-box block: 2048, and at most two blocks per SM of one cloud
  const int64_t chunk = std::max<int64_t>(2048, nb > 1 ? n / kBoxBlocks + 1 : n / (2 * sms) + 1);
  double *box = ctx->cloud_partial + (int64_t)(kMaxClouds + kBoxBlocks) * 8;
  MAFP_TIMED(ctx, s, "k_cloud_bbox",
             launch(k_cloud_bbox<T>, (int)(nb + n / chunk), kBoxThreads, 0, s, pos, n, cloud_off, nb,
                    chunk, ctx->cloud_partial, ctx->cloud_id));
  if (nb > 1)
    MAFP_TIMED(ctx, s, "k_cloud_fold",
               launch(k_cloud_fold, nb, kBoxThreads, 0, s, ctx->cloud_partial, box, cloud_off, n,
                      chunk));
  MAFP_TIMED(ctx, s, "k_cloud_grid",
             launch(k_cloud_grid, 1, kBoxThreads, 0, s, ctx->cloud_partial, box, cloud_off, n, nb,
                    chunk, ctx->d_grids, ctx->cell_base, ctx->d_grid, ctx->d_status,
                    ctx->cap_cells, 0.01 * (double)ctx->tune.cell_edge_pct));
  CloudGrids cg{ctx->d_grids, ctx->cell_base, nb, ctx->d_grid};
  const int tiles = (int)((n + kRadixTile - 1) / kRadixTile);
  MAFP_TIMED(ctx, s, "k_hash",
             launch(k_hash<T>, std::max(tiles, 2 * sms), kRadixThreads, 0, s, pos, n, ctx->cloud_id, cg, ctx->keys_a,
                                                       ctx->vals_a, ctx->radix_hist, tiles,
                                                       ctx->cell_start, ctx->cell_end,
                                                       ctx->n_ucell, ctx->d_status));
  MAFP_LAUNCH_CHECK(ctx);
  uint32_t *kin = ctx->keys_a, *kout = ctx->keys_b;
  int32_t *vin = ctx->vals_a, *vout = ctx->vals_b;
  long long *offs = reinterpret_cast<long long *>(ctx->remap_i64);
  if (n <= kSmallSort) {
    MAFP_TIMED(ctx, s, "k_sort_small",
               launch(k_sort_small, 1, 1024, 0, s, kin, vin, kout, vout, (int)n, ctx->d_grid,
                      ctx->d_status));
    std::swap(kin, kout);
    std::swap(vin, vout);
  }
  for (int p = 0; n > kSmallSort && p < ctx->radix_passes; ++p) {
    if (p > 0)
      MAFP_TIMED(ctx, s, "k_radix_hist",
                 launch(k_radix_hist, tiles, kRadixThreads, 0, s, kin, n, 8 * p, ctx->radix_hist,
                                                              tiles, ctx->d_grid, ctx->d_status));
    int rc = scan_i32_to_i64(ctx, ctx->radix_hist, offs, (int64_t)256 * tiles, s,
                             &ctx->d_status->not_identity);
    if (rc) return rc;
    MAFP_TIMED(ctx, s, "k_radix_scatter",
               launch(k_radix_scatter, tiles, kRadixThreads, 0, s, kin, vin, kout, vout, n, 8 * p,
                                                               offs, tiles, ctx->d_grid,
                                                               ctx->d_status));
    MAFP_LAUNCH_CHECK(ctx);
    // (the unsorted keys and indices stay where they are: a cloud in cell order
    // is read from them)
    std::swap(kin, kout);
    std::swap(vin, vout);
  }
  V *spos = reinterpret_cast<V *>(ctx->spos);
  MAFP_TIMED(ctx, s, "k_cells<T>",
             launch(k_cells<T>, grid_for(n, kCellThreads, sms * 4), kCellThreads, 0, s, 
                 kin, ctx->keys_a, vin, n, pos, spos, ctx->cell_start, ctx->cell_end, ctx->ucell,
                 ctx->n_ucell, order, ctx->d_status, ctx->d_grid));
  MAFP_LAUNCH_CHECK(ctx);
  *svals = vin;
  return MAFP_OK;
}

template <typename T>
static int build_neighbours_t(mafp_ctx *ctx, int64_t n, int nb, const long long *cloud_off,
                              const void *pos_h, int64_t *row_ptr, int32_t *col,
                              int64_t cap_nnz, int64_t *nnz_dev, int32_t *order, cudaStream_t s) {
  const int sms = sm_count();
  const int32_t *vin = nullptr;
  int rc0 = sort_into_cells_t<T>(ctx, n, nb, cloud_off, pos_h, order, &vin, s);
  if (rc0) return rc0;
  const vec4_t<T> *spos = reinterpret_cast<const vec4_t<T> *>(ctx->spos);
  CloudGrids cg{ctx->d_grids, ctx->cell_base, nb, ctx->d_grid};
  const int nbr_blocks = sms * 8;
  int32_t *n_overflow = ctx->n_ucell + 1;
  const long long pool_words = (long long)kMaskWords * ctx->cap_particles;
  // Parts per cell: a small cloud has fewer cells than the GPU has warps (mask and
  // fill at 5650 particles 71 + 134 us unsplit, 24 + 23 us in these parts); in
  // larger ones only the costly cells are split, so that no warp ends late
  // (200k random particles, mask + fill: 535 us unsplit, 438 in halves, 366 in
  // quarters; the 1M jet cloud 423, 398 and 462 us).  The lines follow such uneven
  // clouds; in even ones the parts cost a little just below them (whole search, on
  // either side of 131072: 3D in cell order 228 and 201 us, FP64 471 and 324, film 121
  // and 113; of 524288: 506 and 441, 992 and 667, 188 and 188).
  const Split split = n <= kSplitAll ? Split{3, 1} : n <= kSplitMore ? Split{2, 0} : Split{1, 0};
  const long long *rp = reinterpret_cast<const long long *>(row_ptr);
  MAFP_TIMED(ctx, s, "k_cell_table",
             launch(k_cell_table, grid_for(n, 128, sms * 16), 128, 0, s, 
                 cg, ctx->ucell, ctx->n_ucell, ctx->cell_start, ctx->cell_end, ctx->cell_table,
                 pool_words, ctx->overflow, n));
  MAFP_TIMED(ctx, s, sizeof(T) == 4 ? "k_nbr_mask<float>" : "k_nbr_mask<double>",
             launch(k_nbr_mask<T>, sms * 8, kMaskThreads, 0, s, 
                 ctx->d_grid, ctx->cell_table, ctx->n_ucell, spos, vin, ctx->counts,
                 ctx->nbr_mask, split));
  MAFP_TIMED(ctx, s, "k_nbr<T,false>(overflow cells)",
             launch(k_nbr<T, false>, nbr_blocks, kNbrThreads, kNbrSmemBytes, s, 
                 ctx->d_grid, ctx->cell_table, ctx->overflow, n_overflow, spos, vin, ctx->counts,
                 nullptr, nullptr, 0, n));
  MAFP_LAUNCH_CHECK(ctx);
  int rc = scan_i32_to_i64(ctx, ctx->counts, reinterpret_cast<long long *>(row_ptr), n, s);
  if (rc) return rc;
  // (launched plainly: set up beside the scan's last blocks, the persistent blocks
  // share the SMs out unevenly, 683 against 663 us for the 200k-particle search)
  MAFP_TIMED(ctx, s, "k_nbr_fill",
             k_nbr_fill<<<sms * 8, kFillThreads, 0, s>>>(ctx->d_grid, ctx->cell_table,
                                                         ctx->n_ucell, vin, ctx->nbr_mask, split,
                                                         rp, col, cap_nnz, n, nnz_dev,
                                                         ctx->d_status));
  MAFP_TIMED(ctx, s, "k_nbr<T,true>(overflow cells)",
             launch(k_nbr<T, true>, nbr_blocks, kNbrThreads, kNbrSmemBytes, s, 
                 ctx->d_grid, ctx->cell_table, ctx->overflow, n_overflow, spos, vin, ctx->counts,
                 rp, col, cap_nnz, n));
  MAFP_TIMED(ctx, s, "k_rowsort",
             launch(k_rowsort, grid_for(n, kSortWarps, sms * 8), kSortWarps * 32, 0, s, 
      reinterpret_cast<const long long *>(row_ptr), col, n, cap_nnz, ctx->d_status,
      ctx->d_grid));
  MAFP_LAUNCH_CHECK(ctx);
  return MAFP_OK;
}

int build_neighbours(mafp_ctx *ctx, int64_t n, int32_t dtype, const void *pos_h,
                     int64_t *row_ptr, int32_t *col, int64_t cap_nnz, int64_t *nnz_dev,
                     int32_t *order, cudaStream_t s) {
  if (dtype == MAFP_F64)
    return build_neighbours_t<double>(ctx, n, 1, nullptr, pos_h, row_ptr, col, cap_nnz,
                                      nnz_dev, order, s);
  return build_neighbours_t<float>(ctx, n, 1, nullptr, pos_h, row_ptr, col, cap_nnz,
                                   nnz_dev, order, s);
}

int cell_order(mafp_ctx *ctx, int64_t n, int32_t dtype, const void *pos_h, int32_t *order,
               cudaStream_t s) {
  const int32_t *vin = nullptr;
  if (dtype == MAFP_F64)
    return sort_into_cells_t<double>(ctx, n, 1, nullptr, pos_h, order, &vin, s);
  return sort_into_cells_t<float>(ctx, n, 1, nullptr, pos_h, order, &vin, s);
}

int build_neighbours_batched(mafp_ctx *ctx, int64_t n, int32_t dtype, int32_t nclouds,
                             const int64_t *cloud_offset, const void *pos_h, int64_t *row_ptr,
                             int32_t *col, int64_t cap_nnz, int64_t *nnz_dev, int32_t *order,
                             cudaStream_t s) {
  const long long *off = reinterpret_cast<const long long *>(cloud_offset);
  if (dtype == MAFP_F64)
    return build_neighbours_t<double>(ctx, n, nclouds, off, pos_h, row_ptr, col, cap_nnz,
                                      nnz_dev, order, s);
  return build_neighbours_t<float>(ctx, n, nclouds, off, pos_h, row_ptr, col, cap_nnz, nnz_dev,
                                   order, s);
}

void init_kernel_attributes() {
  cudaFuncSetAttribute(k_nbr<float, false>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                       kNbrSmemBytes);
  cudaFuncSetAttribute(k_nbr<float, true>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                       kNbrSmemBytes);
  cudaFuncSetAttribute(k_nbr<double, false>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                       kNbrSmemBytes);
  cudaFuncSetAttribute(k_nbr<double, true>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                       kNbrSmemBytes);
}

int transpose_map(mafp_ctx *ctx, int64_t n, const int64_t *row_ptr, const int32_t *col,
                  uint16_t *tloc, cudaStream_t s) {
  MAFP_TIMED(ctx, s, "k_tmap",
             launch(k_tmap, grid_for(n * 32, 256, sm_count() * 16), 256, 0, s, 
      reinterpret_cast<const long long *>(row_ptr), col, n, tloc, ctx->d_status));
  MAFP_LAUNCH_CHECK(ctx);
  return MAFP_OK;
}

}  // namespace mafp
