// k_step.cu -- per-particle kernels of the CSPH step (HBM-bound): CFL time
// step, kick-drift-kick updates, the cell mesh of eq. (Dcell) with a
// counting sort into cells, operand packing for the pair kernel, the
// renumbering of Sec. 4.2 and the FP64 conservation sums.
//
// Every per-particle kernel runs on "segmented" blocks: block b covers the
// particles [blk_start[b], blk_end[b]) of one instance, so per-instance
// reductions are fixed-order reductions over whole blocks (no atomics).
#include <algorithm>
#include <cfloat>
#include <climits>

#include "csph_internal.cuh"
#include "step_math.cuh"

namespace csph {

namespace {

__device__ __forceinline__ double ld(const double* a, int64_t i) { return a ? a[i] : 0.0; }

// Return the status of a failed launch from the enclosing launcher.
#define CKL(call)                            \
  do {                                       \
    const cudaError_t ckl_e_ = (call);       \
    if (ckl_e_ != cudaSuccess) return ckl_e_; \
  } while (0)

__device__ __forceinline__ void set_status(int* status, int code) { atomicCAS(status, 0, code); }

// Merge the top-2 multisets (a1 >= a2) and (b1 >= b2).
__device__ __forceinline__ void top2_merge(long long& a1, long long& a2, long long b1, long long b2) {
  if (a1 >= b1) { a2 = a2 > b1 ? a2 : b1; }
  else { a2 = b2 > a1 ? b2 : a1; a1 = b1; }
}

// Order keys of FP32 values (integer order = numeric order), as dkey.
__device__ __forceinline__ int fkey(float x) {
  const int b = __float_as_int(x);
  return b < 0 ? b ^ 0x7fffffff : b;
}
__device__ __forceinline__ float funkey(int k) { return __int_as_float(k < 0 ? k ^ 0x7fffffff : k); }

struct Red {
  long long lo[3], hi[3], d1, d2, viol;
  int dlo[3], dhi[3];
};

__device__ __forceinline__ void red_init(Red& r) {
  for (int a = 0; a < 3; ++a) { r.lo[a] = LLONG_MAX; r.hi[a] = LLONG_MIN; r.dlo[a] = INT_MAX; r.dhi[a] = INT_MIN; }
  r.d1 = 0; r.d2 = 0; r.viol = LLONG_MIN;
}

__device__ __forceinline__ void red_merge(Red& a, const Red& b) {
  for (int k = 0; k < 3; ++k) {
    a.lo[k] = a.lo[k] < b.lo[k] ? a.lo[k] : b.lo[k];
    a.hi[k] = a.hi[k] > b.hi[k] ? a.hi[k] : b.hi[k];
    a.dlo[k] = min(a.dlo[k], b.dlo[k]);
    a.dhi[k] = max(a.dhi[k], b.dhi[k]);
  }
  top2_merge(a.d1, a.d2, b.d1, b.d2);
  a.viol = a.viol > b.viol ? a.viol : b.viol;
}

// Minimum / maximum of a 64-bit key over a full warp: the signed high word,
// then the low word among the lanes that hold it, two redux instructions
// where a butterfly takes ten shuffles and five 64-bit compares.
__device__ __forceinline__ long long warp_min(long long k) {
  const int hi = (int)(k >> 32), m = __reduce_min_sync(0xffffffffu, hi);
  const unsigned lo = __reduce_min_sync(0xffffffffu, hi == m ? (unsigned)k : 0xffffffffu);
  return (long long)(((unsigned long long)(unsigned)m << 32) | lo);
}

__device__ __forceinline__ long long warp_max(long long k) {
  const int hi = (int)(k >> 32), m = __reduce_max_sync(0xffffffffu, hi);
  const unsigned lo = __reduce_max_sync(0xffffffffu, hi == m ? (unsigned)k : 0u);
  return (long long)(((unsigned long long)(unsigned)m << 32) | lo);
}

// The two largest sizes: the largest d1, then that lane's d2 against the other
// lanes' d1.  The Verlet keys stay as they are without `verlet` (a kernel
// without a list handle leaves them at red_init).
__device__ __forceinline__ void warp_reduce(Red& r, int dim, bool verlet) {
#pragma unroll
  for (int a = 0; a < 3; ++a)
    if (a < dim) {
      r.lo[a] = warp_min(r.lo[a]);
      r.hi[a] = warp_max(r.hi[a]);
      if (verlet) {
        r.dlo[a] = __reduce_min_sync(0xffffffffu, r.dlo[a]);
        r.dhi[a] = __reduce_max_sync(0xffffffffu, r.dhi[a]);
      }
    }
  const long long m = warp_max(r.d1);
  const int first = __ffs(__ballot_sync(0xffffffffu, r.d1 == m)) - 1;
  r.d2 = warp_max((int)(threadIdx.x & 31) == first ? r.d2 : r.d1);
  r.d1 = m;
  if (verlet) r.viol = warp_max(r.viol);
}

// Block-wide reduction of Red, once per kernel: each warp, then the first warp
// over the warps' results; result in thread 0.  Every merge is a min / max /
// top-2 of integer keys, so the order does not change the result.  (With
// butterflies and one thread merging the warps it was half of the kick-drift's
// 996 instructions a warp.)
__device__ void block_reduce(Red& r, int dim, bool verlet) {
  __shared__ Red sh[kBlock / 32];
  warp_reduce(r, dim, verlet);
  const int t = threadIdx.x;
  if ((t & 31) == 0) sh[t >> 5] = r;
  __syncthreads();
  if (t < 32) {
    if (t < (int)(blockDim.x >> 5)) r = sh[t];
    else red_init(r);
    warp_reduce(r, dim, verlet);
  }
}

// Block minimum of the dt keys (k_cfl, k_kick2); result in thread 0.
__device__ long long block_min_key(long long k) {
  __shared__ long long sh[kBlock / 32];
  k = warp_min(k);
  if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = k;
  __syncthreads();
  if (threadIdx.x < 32) k = warp_min(threadIdx.x < (blockDim.x >> 5) ? sh[threadIdx.x] : LLONG_MAX);
  return k;
}

__device__ __forceinline__ void write_part(BlockPart* part, const Red& r) {
  BlockPart& b = part[blockIdx.x];
  for (int a = 0; a < 3; ++a) { b.lo[a] = r.lo[a]; b.hi[a] = r.hi[a]; }
  b.d1 = r.d1; b.d2 = r.d2;
}

// ---------------------------------------------------------------------------
// d, P, c and the bounding box of the current state (a mesh build outside the
// step follows).
// ---------------------------------------------------------------------------
__global__ void k_derive(DevParams P, sph_state s, const int64_t* __restrict__ blk_start,
                         const int64_t* __restrict__ blk_end, BlockPart* part) {
  chain_entry();
  int64_t p = blk_start[blockIdx.x] + threadIdx.x;
  Red r;
  red_init(r);
  if (p < blk_end[blockIdx.x]) {
    double vx = ld(s.vx, p), vy = ld(s.vy, p), vz = ld(s.vz, p);
    double v2 = vx * vx + vy * vy + vz * vz;
    double e = s.E[p] - 0.5 * v2;
    int mi = s.mat ? s.mat[p] : 0;
    double Pp, cp;
    eos(P.mat[mi], s.rho[p], e, Pp, cp);
    double d = size_of(P.dim, s.m[p], s.rho[p]);
    s.d[p] = d; s.P[p] = Pp; s.c[p] = cp;
    r.lo[0] = r.hi[0] = dkey(s.x[p]);
    if (P.dim >= 2) r.lo[1] = r.hi[1] = dkey(s.y[p]);
    if (P.dim >= 3) r.lo[2] = r.hi[2] = dkey(s.z[p]);
    r.d1 = dkey(d);
  }
  block_reduce(r, P.dim, false);
  if (threadIdx.x == 0) write_part(part, r);
}

// A step's CFL bound dt_i = eta d_i / (c_i + |v_i|) (cfl_key), min-reduced into
// the instance's dt_key.
__global__ void k_cfl(DevParams P, sph_state s, const int64_t* __restrict__ blk_start,
                      const int64_t* __restrict__ blk_end, const int32_t* __restrict__ blk_inst, long long* dt_key) {
  chain_entry();
  const int64_t p = blk_start[blockIdx.x] + threadIdx.x;
  long long k = LLONG_MAX;
  if (p < blk_end[blockIdx.x]) {
    // every load issued before the arithmetic
    const double vx = ld(s.vx, p), vy = ld(s.vy, p), vz = ld(s.vz, p);
    const double E = s.E[p], rho = s.rho[p], m = s.m[p];
    const int mi = s.mat ? s.mat[p] : 0;
    k = cfl_key(P, vx, vy, vz, E, rho, m, mi);
  }
  k = block_min_key(k);
  if (threadIdx.x == 0) atomicMin(&dt_key[blk_inst[blockIdx.x]], k);
}

// dt = cfl * (the instance's minimum), and the keys ready for the next
// accumulation (sph_cfl_dt; a step's kick-drift forms its own dt).
__global__ void k_reduce_dt(int n_inst, double cfl, double* dt, long long* dt_key) {
  chain_entry();
  const int b = blockIdx.x * blockDim.x + threadIdx.x;
  if (b >= n_inst) return;
  dt[b] = cfl * dunkey(dt_key[b]);
  dt_key[b] = LLONG_MAX;
}

// Arguments of the mesh build.
struct MeshArgs {
  DevParams P;
  const double *x, *y, *z;
  int n_inst, nblk;
  const int64_t *inst_off, *inst_cap, *blk_start, *blk_end;
  const int32_t *blk_inst, *inst_blk;
  const BlockPart* part;
  GridInfo* grid;
  int64_t* total_cells;
  int32_t *cell_count, *cell_start, *scan_sums, *cell_of, *rank, *perm;
  double* slot_org;         // mixed precision: origin of each slot's cell, or NULL
  int* status;
  const int* gate;          // Verlet steps: nothing is built while gate[0] == 0
  const int* vinst;         // Verlet steps of a batched handle: the instances rebuilt, or NULL (all)
};

// One block per instance: the bounding box and the two largest sizes of the
// instance from its block partials, into the grid record.
// vinst (Verlet steps): an instance that keeps its lists keeps its mesh geometry.
__device__ void mesh_reduce_inst(int b, const int32_t* inst_blk, const BlockPart* part, GridInfo* grid, const int* vinst) {
  if (vinst && vinst[b] == 0) return;
  Red r;
  red_init(r);
  for (int k = inst_blk[b] + threadIdx.x; k < inst_blk[b + 1]; k += blockDim.x) {
    Red q;
    for (int a = 0; a < 3; ++a) { q.lo[a] = part[k].lo[a]; q.hi[a] = part[k].hi[a]; }
    q.d1 = part[k].d1; q.d2 = part[k].d2;
    red_merge(r, q);
  }
  block_reduce(r, 3, false);
  if (threadIdx.x == 0) {
    GridInfo& g = grid[b];
    for (int a = 0; a < 3; ++a) { g.x0[a] = dunkey(r.lo[a]); g.hi[a] = dunkey(r.hi[a]); }
    g.dmax1 = dunkey(r.d1);
    g.dmax2 = dunkey(r.d2);
  }
}

// Cell mesh per instance (one block, a thread per instance): D^c of eq.
// (Dcell) with the safety margin, doubled until the instance's share of the
// cell capacity holds the mesh; dims per axis; then the global cell offsets
// in instance order.  Matches the oracle bit for bit.
// vinst (Verlet steps): an instance that keeps its lists keeps its geometry and
// only moves to its new cell offset.
__device__ void mesh_setup(const DevParams& P, int n_inst, const int64_t* inst_off, const int64_t* inst_cap, GridInfo* grid,
                           int64_t* total_cells, int* status, const int* vinst) {
  // the instances' meshes, one thread per instance
  for (int b = threadIdx.x; b < n_inst; b += blockDim.x) {
    GridInfo& g = grid[b];
    if (vinst && vinst[b] == 0) continue;
    double hi[3];
    for (int a = 0; a < 3; ++a) hi[a] = g.hi[a];
    for (int a = P.dim; a < 3; ++a) { g.x0[a] = 0.0; g.hi[a] = 0.0; hi[a] = 0.0; }
    double d1 = g.dmax1, d2 = g.dmax2;
    if (inst_off[b + 1] - inst_off[b] < 2) d2 = d1;
    double dc = __dmul_rn(P.kh, __dadd_rn(d1, d2));
    dc = __dmul_rn(dc, 1.0 + P.cell_beta);
    dc = __dmul_rn(dc, kCellMargin);
    if (!(dc > 0.0) || !isfinite(dc)) { set_status(status, SPH_ERR_NONFINITE); dc = 1.0; }
    int64_t tot;
    double inv;
    int64_t dims[3];
    for (int iter = 0; iter < 2100; ++iter) {
      inv = 1.0 / dc;
      tot = 1;
      for (int a = 0; a < 3; ++a) {
        dims[a] = (a < P.dim) ? (int64_t)floor(__dmul_rn(__dsub_rn(hi[a], g.x0[a]), inv)) + 1 : 1;
        tot *= dims[a];
      }
      if (tot <= inst_cap[b]) break;
      dc = dc * 2.0;
    }
    g.dc = dc;
    g.inv_dc = inv;
    for (int a = 0; a < 3; ++a) g.dims[a] = (int32_t)dims[a];
    g.ncells = tot;
    g.dc_f = (float)dc;
  }
  __syncthreads();
  if (n_inst == 1) {
    if (threadIdx.x == 0) {
      grid[0].cell_off = 0;
      *total_cells = grid[0].ncells;
    }
    return;
  }
  // global cell offsets in instance order (a kept instance only moves): an
  // exclusive scan of the cell counts over the block (warp scans, then the
  // warps' totals), a chunk of instances at a time
  __shared__ long long wsum[32];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, nw = (blockDim.x + 31) >> 5;
  long long carry = 0;
  for (int base = 0; base < n_inst; base += blockDim.x) {
    const int b = base + (int)threadIdx.x;
    const long long v = b < n_inst ? (long long)grid[b].ncells : 0;
    long long x = v;                                   // inclusive scan within the warp
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const long long t = __shfl_up_sync(0xffffffffu, x, o);
      if (lane >= o) x += t;
    }
    if (lane == 31) wsum[w] = x;
    __syncthreads();
    long long before = 0, chunk = 0;                   // the earlier warps' totals, the chunk's total
    for (int k = 0; k < nw; ++k) {
      if (k < w) before += wsum[k];
      chunk += wsum[k];
    }
    if (b < n_inst) grid[b].cell_off = carry + before + x - v;
    carry += chunk;
    __syncthreads();                                   // wsum is rewritten by the next chunk
  }
  if (threadIdx.x == 0) *total_cells = carry;
}

__device__ __forceinline__ int64_t local_cell(const GridInfo& g, int dim, double x, double y, double z,
                                              int32_t c[3]) {
  c[0] = (int32_t)floor(__dmul_rn(__dsub_rn(x, g.x0[0]), g.inv_dc));
  c[1] = dim >= 2 ? (int32_t)floor(__dmul_rn(__dsub_rn(y, g.x0[1]), g.inv_dc)) : 0;
  c[2] = dim >= 3 ? (int32_t)floor(__dmul_rn(__dsub_rn(z, g.x0[2]), g.inv_dc)) : 0;
  return (int64_t)c[0] + (int64_t)g.dims[0] * ((int64_t)c[1] + (int64_t)g.dims[1] * c[2]);
}

// One segmented block's particles (t: the thread's position in the block).
// vinst (Verlet steps): the particles of an instance that keeps its lists are
// counted at their positions of its last build (vref), with its kept
// geometry, which reproduces that build's cells, slots and in-cell order.
__device__ __forceinline__ void mesh_count(const MeshArgs& a, int lb, int t) {
  const int dim = a.P.dim;
  const int64_t p = a.blk_start[lb] + t;
  if (p >= a.blk_end[lb]) return;
  const int b = a.blk_inst[lb];
  const GridInfo& g = a.grid[b];
  const bool kept = a.vinst && a.vinst[b] == 0;
  const double* vref = a.P.vref;
  const double px = kept ? vref[p] : a.x[p];
  const double py = dim >= 2 ? (kept ? vref[a.P.n + p] : a.y[p]) : 0.0;
  const double pz = dim >= 3 ? (kept ? vref[2 * a.P.n + p] : a.z[p]) : 0.0;
  int32_t c[3];
  int64_t lc = local_cell(g, dim, px, py, pz, c);
  bool ok = true;
  for (int k = 0; k < 3; ++k) ok = ok && c[k] >= 0 && c[k] < g.dims[k];
  if (!ok) {  // only a non-finite position can leave the mesh: latch it, stay in bounds
    set_status(a.status, SPH_ERR_NONFINITE);
    lc = 0;
  }
  const int32_t gc = (int32_t)(g.cell_off + lc);
  a.cell_of[p] = gc;
  a.rank[p] = atomicAdd(&a.cell_count[gc], 1);
}

// Exclusive scan of cell_count[0, total) into cell_start, 1024 cells per tile.
constexpr int kScanTile = 1024;

__global__ void k_scan_reduce(const int32_t* __restrict__ cnt, const int64_t* __restrict__ total,
                              int32_t* sums, const int* __restrict__ gate) {
  chain_entry();
  if (gate && gate[0] == 0) return;   // Verlet mode: mesh kept from the last build
  const int64_t tot = *total;
  __shared__ int sh[kBlock];
  // grid-stride over the tiles the current mesh has (the grid is sized for the capacity,
  // capped at a few waves)
  for (int64_t t = blockIdx.x; t * kScanTile < tot; t += gridDim.x) {
    const int64_t base = t * kScanTile;
    int v = 0;
    for (int k = threadIdx.x; k < kScanTile; k += blockDim.x) {
      int64_t c = base + k;
      if (c < tot) v += cnt[c];
    }
    sh[threadIdx.x] = v;
    __syncthreads();
    for (int w = kBlock / 2; w > 0; w >>= 1) {
      if (threadIdx.x < w) sh[threadIdx.x] += sh[threadIdx.x + w];
      __syncthreads();
    }
    if (threadIdx.x == 0) sums[t] = sh[0];
    __syncthreads();
  }
}

// Per tile: exclusive scan plus tile offset; zero the counts for the next use.
// A block adds up the sums of the tiles before its own itself (4 bytes of L2
// per 1024 cells): a one-block scan of them between the two kernels cost a
// launch and its latency per mesh build (400-particle FP64 tube with a mesh per
// step: 1123 -> 1065 us a pass; 32k plate impact with lists: 553 -> 544).
__global__ void k_scan_down(int32_t* cnt, const int64_t* __restrict__ total, const int32_t* __restrict__ sums,
                            int32_t* start, int64_t n_total, const int* __restrict__ gate) {
  chain_entry();
  if (gate && gate[0] == 0) return;   // Verlet mode: mesh kept from the last build
  const int64_t tot = *total;
  constexpr int per = kScanTile / kBlock;  // 4 cells per thread
  __shared__ int sh[kBlock];
  __shared__ int wsum[kBlock / 32];
  int64_t before = 0;                       // tiles whose sums are in `offset`
  int offset = 0;
  for (int64_t t = blockIdx.x; t * kScanTile < tot; t += gridDim.x) {
    const int64_t base = t * kScanTile;
    int part = 0;
    for (int64_t k = before + threadIdx.x; k < t; k += blockDim.x) part += sums[k];
    part = __reduce_add_sync(0xffffffffu, part);
    if ((threadIdx.x & 31) == 0) wsum[threadIdx.x >> 5] = part;
    __syncthreads();
    for (int w = 0; w < kBlock / 32; ++w) offset += wsum[w];
    before = t;
    int vals[per];
    int run = 0;
    for (int k = 0; k < per; ++k) {
      int64_t c = base + threadIdx.x * per + k;
      vals[k] = (c < tot) ? cnt[c] : 0;
      run += vals[k];
    }
    sh[threadIdx.x] = run;
    __syncthreads();
    for (int off = 1; off < kBlock; off <<= 1) {
      int add = threadIdx.x >= (unsigned)off ? sh[threadIdx.x - off] : 0;
      __syncthreads();
      sh[threadIdx.x] += add;
      __syncthreads();
    }
    int acc = offset + sh[threadIdx.x] - run;
    for (int k = 0; k < per; ++k) {
      int64_t c = base + threadIdx.x * per + k;
      if (c < tot) {
        start[c] = acc;
        acc += vals[k];
        cnt[c] = 0;
      }
    }
    if (base + kScanTile >= tot && threadIdx.x == 0) start[tot] = (int32_t)n_total;
    __syncthreads();
  }
}

// vinst (Verlet steps): the slots of an instance that keeps its lists keep
// their particles (its cells' starts come out as before), so its particles
// are not scattered, and its cells are not sorted below.
__device__ __forceinline__ void mesh_scatter(const MeshArgs& a, int64_t p) {
  if (a.vinst) {
    int lo = 0, hi = a.n_inst;                       // the particle's instance
    while (hi - lo > 1) {
      const int mid = (lo + hi) >> 1;
      if (a.inst_off[mid] <= p) lo = mid; else hi = mid;
    }
    if (a.vinst[lo] == 0) return;
  }
  a.perm[a.cell_start[a.cell_of[p]] + a.rank[p]] = (int32_t)p;
}

// Within each cell, order the particles by index (the atomic arrival order is
// not reproducible; this makes the slot order a function of the state only).
// Mixed precision: also the origin of each cell, o = x0 + c dc per axis, for
// every slot of the cell (slot_org; k_pack takes the FP32 offsets from it).
// w0, nw: this warp's index and the number of warps.
__device__ __forceinline__ void mesh_sort(const MeshArgs& a, int64_t tot, int64_t w0, int64_t nw) {
  const int32_t* start = a.cell_start;
  int32_t* perm = a.perm;
  const GridInfo* grid = a.grid;
  const int n_inst = a.n_inst, dim = a.P.dim;
  const int64_t nslots = a.P.n;
  double* slot_org = a.slot_org;
  const int* vinst = a.vinst;
  // One warp per cell: each lane holds up to kSortPer of the cell's particle
  // indices and counts, by broadcasts, the cell's indices smaller than each
  // (indices are distinct), which is its position in ascending order.  Cells
  // above 32 kSortPer particles (never on a sane mesh: the cell code admits
  // 2047) are sorted by one lane.
  constexpr int kSortPer = 4;
  const int lane = threadIdx.x & 31;
  for (int64_t c = w0; c < tot; c += nw) {
    const int b = start[c], e = start[c + 1], n = e - b;
    if (n <= 0) continue;
    int bi = 0;                                      // the cell's instance
    if (n_inst > 1 && (slot_org || vinst)) {
      int lo = 0, hi = n_inst;
      while (hi - lo > 1) {
        const int mid = (lo + hi) >> 1;
        if (grid[mid].cell_off <= c) lo = mid; else hi = mid;
      }
      bi = lo;
    }
    if (vinst && vinst[bi] == 0) continue;          // kept: slots, order and origins as they are
    if (slot_org) {
      const GridInfo& g = grid[bi];
      const int64_t lc = c - g.cell_off;
      const int64_t cc[3] = {lc % g.dims[0], (lc / g.dims[0]) % g.dims[1], lc / ((int64_t)g.dims[0] * g.dims[1])};
#pragma unroll
      for (int a = 0; a < 3; ++a)
        if (a < dim) {
          const double o = __fma_rn((double)cc[a], g.dc, g.x0[a]);
          for (int k = b + lane; k < e; k += 32) slot_org[(int64_t)a * nslots + k] = o;
        }
    }
    if (n <= 1) continue;
    if (n > 32 * kSortPer) {
      if (lane == 0)
        for (int i = b + 1; i < e; ++i) {
          int32_t v = perm[i];
          int j = i - 1;
          while (j >= b && perm[j] > v) { perm[j + 1] = perm[j]; --j; }
          perm[j + 1] = v;
        }
      __syncwarp();
      continue;
    }
    int32_t v[kSortPer];
    int rank[kSortPer];
#pragma unroll
    for (int q = 0; q < kSortPer; ++q) {
      v[q] = lane + 32 * q < n ? perm[b + lane + 32 * q] : INT_MAX;
      rank[q] = 0;
    }
    const int rounds = (n + 31) >> 5;
    for (int r = 0; r < rounds; ++r) {
      const int cnt = min(32, n - 32 * r);
      int32_t mine = INT_MAX;
#pragma unroll
      for (int q = 0; q < kSortPer; ++q)
        if (q == r) mine = v[q];
      for (int k = 0; k < cnt; ++k) {
        const int32_t t = __shfl_sync(0xffffffffu, mine, k);
#pragma unroll
        for (int q = 0; q < kSortPer; ++q) rank[q] += t < v[q] ? 1 : 0;
      }
    }
    __syncwarp();   // every index read before any is written back
#pragma unroll
    for (int q = 0; q < kSortPer; ++q)
      if (lane + 32 * q < n) perm[b + rank[q]] = v[q];
  }
}

// ---------------------------------------------------------------------------
// The mesh build, a kernel per phase, chained (a chained launch that returns at
// once costs 1.5 us).  One kernel for all phases was measured and dropped: with
// a barrier over a cooperative grid a build of 6k particles took 84 us longer,
// with one cluster of 16 CTAs 12 us (30 us at 32k, whose work 16 SMs hold too
// long); the gated steps gained 2 us.
// ---------------------------------------------------------------------------
__global__ void k_mesh_reduce(MeshArgs a) {
  chain_entry();
  if (a.gate && a.gate[0] == 0) return;   // Verlet mode: mesh kept from the last build
  mesh_reduce_inst(blockIdx.x, a.inst_blk, a.part, a.grid, a.vinst);
}

__global__ void k_mesh_setup(MeshArgs a) {
  chain_entry();
  if (a.gate && a.gate[0] == 0) return;
  if (a.n_inst == 1) {                    // one instance: no launch of its own for the reduction
    mesh_reduce_inst(0, a.inst_blk, a.part, a.grid, a.vinst);
    __syncthreads();
  }
  mesh_setup(a.P, a.n_inst, a.inst_off, a.inst_cap, a.grid, a.total_cells, a.status, a.vinst);
}

__global__ void k_cell_count(MeshArgs a) {
  chain_entry();
  if (a.gate && a.gate[0] == 0) return;
  // a capped grid strides over the segmented blocks (cheap to launch when gated)
  for (int lb = blockIdx.x; lb < a.nblk; lb += gridDim.x) mesh_count(a, lb, threadIdx.x);
}

__global__ void k_cell_scatter(MeshArgs a) {
  chain_entry();
  if (a.gate && a.gate[0] == 0) return;
  for (int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; p < a.P.n; p += (int64_t)gridDim.x * blockDim.x)
    mesh_scatter(a, p);
}

__global__ void k_cell_sort(MeshArgs a) {
  chain_entry();
  if (a.gate && a.gate[0] == 0) return;
  mesh_sort(a, *a.total_cells, ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5,
            ((int64_t)gridDim.x * blockDim.x) >> 5);
}

// Verlet lists: vflag[0] = lists invalid (vflag[1]) or the validity criterion
// of k_kick_drift failed for some particle of any instance.
// Also sets, per instance (no pair joins two instances), the frame
// displacement U of the next step's criterion: the midpoint of this step's
// displacement box, which covers k steps since the build, extrapolated to
// k + 1 steps; after a build, one step's worth of it (the new reference is
// this step's state); 0 while the reference is void.  Any U keeps the
// criterion sound; a good one only makes builds rarer.
__global__ void k_verlet_flag(int* vflag, double* vframe, VAcc* vacc, int n_inst, int* vinst, int together) {
  chain_entry();
  // each instance whose criterion failed is rebuilt (its mesh, slots and lists;
  // the other instances keep theirs), or all of them when the lists are void or
  // the instances share an evaluation order (together)
  int fail = 0;
  for (int b = threadIdx.x; b < n_inst; b += blockDim.x) fail |= vacc[b].viol > 0 ? 1 : 0;
  const bool void_ref = vflag[1] != 0;
  const bool any = __syncthreads_or(fail) != 0 || void_ref;
  if (threadIdx.x == 0) vflag[0] = any ? 1 : 0;
  for (int b = threadIdx.x; b < n_inst; b += blockDim.x) {
    const bool rebuild = void_ref || (together ? any : vacc[b].viol > 0);
    vinst[b] = rebuild ? 1 : 0;
    VAcc& va = vacc[b];
    int bx[6];
#pragma unroll
    for (int a = 0; a < 3; ++a) { bx[a] = va.dlo[a]; bx[3 + a] = va.dhi[a]; }
    // reset for the next kick-drift
    va.viol = LLONG_MIN;
#pragma unroll
    for (int a = 0; a < 3; ++a) { va.dlo[a] = INT_MAX; va.dhi[a] = INT_MIN; }
    double* fr = vframe + 6 * b;
    const double ks = fr[3] >= 1.0 ? fr[3] : 1.0;   // steps covered by this step's displacements
    float* Uf = reinterpret_cast<float*>(fr + 4);
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      // midpoint of the box of x - x^b, from that of x - x^b - U
      const double mid = bx[a] <= bx[3 + a] ? 0.5 * ((double)funkey(bx[a]) + (double)funkey(bx[3 + a])) + fr[a]
                                            : fr[a];
      fr[a] = void_ref ? 0.0 : (rebuild ? mid / ks : mid * (ks + 1.0) / ks);
      Uf[a] = (float)fr[a];
    }
    fr[3] = rebuild ? 1.0 : ks + 1.0;
  }
}

// ---------------------------------------------------------------------------
// Kick-drift: v <- v + dt/2 a, x <- x + dt v, rho, E half kicks; predicted
// size d~ from rho~ = rho^h + dt/2 drho; bounding box and sizes for the mesh.
// ---------------------------------------------------------------------------
// The time step: with dt_key, cfl times the instance's minimum, which the
// instance's first block also leaves in dt (k_pack makes the key ready for the
// next accumulation); else the prescribed dt.
// (The rebuild decision of a Verlet step stays a kernel of its own: made by the
// last block of this one, the fence and the ticket of every block added 16 us
// at 1.125M particles, four times that kernel.)
template <bool MIXED>
__global__ void __launch_bounds__(kBlock, 4) k_kick_drift(DevParams P, sph_state s, const int64_t* __restrict__ blk_start,
                             const int64_t* __restrict__ blk_end, const int32_t* __restrict__ blk_inst,
                             const int32_t* __restrict__ inst_blk, double* dt, const long long* __restrict__ dt_key,
                             BlockPart* part, int* status) {
  chain_entry();
  int64_t p = blk_start[blockIdx.x] + threadIdx.x;
  Red r;
  red_init(r);
  const int inst = blk_inst[blockIdx.x];
  if (dt_key && threadIdx.x == 0 && inst_blk[inst] == (int)blockIdx.x) dt[inst] = P.cfl * dunkey(dt_key[inst]);
  if (p < blk_end[blockIdx.x]) {
    const int dim = P.dim;
    const double h = dt_key ? P.cfl * dunkey(dt_key[inst]) : dt[inst];
    const double hdt = 0.5 * h;
    double* X[3] = {s.x, s.y, s.z};
    double* V[3] = {s.vx, s.vy, s.vz};
    const double* A[3] = {s.ax, s.ay, s.az};
    // Every load is issued before the first store: the state arrays may alias
    // as far as the compiler can tell, so a load placed after a store would
    // wait for it, one memory round trip per component.
    double x[3] = {0.0, 0.0, 0.0}, v[3] = {0.0, 0.0, 0.0}, acc[3] = {0.0, 0.0, 0.0}, xb[3] = {0.0, 0.0, 0.0};
#pragma unroll
    for (int a = 0; a < 3; ++a)
      if (a < dim) {
        x[a] = X[a][p];
        v[a] = V[a][p];
        acc[a] = A[a][p];
        if (P.vref) xb[a] = P.vref[(int64_t)a * P.n + p];
      }
    const double rho0 = s.rho[p], drho = s.drho[p], E0 = s.E[p], dE = s.dE[p], m = s.m[p];
    const double db = P.vref ? P.vref[3 * P.n + p] : 0.0;
    bool finite = true;
#pragma unroll
    for (int a = 0; a < 3; ++a)
      if (a < dim) {
        v[a] = axpy<MIXED>(hdt, acc[a], v[a]);
        x[a] = axpy<MIXED>(h, v[a], x[a]);
        r.lo[a] = r.hi[a] = dkey(x[a]);
        finite = finite && finite_bits(x[a]);
      }
    const double rh = axpy<MIXED>(hdt, drho, rho0);
    const double En = axpy<MIXED>(hdt, dE, E0);
    const double rp = axpy<MIXED>(hdt, drho, rh);
    const double d = MIXED ? size_of_mixed(dim, m, rp) : size_of(dim, m, rp);
#pragma unroll
    for (int a = 0; a < 3; ++a)
      if (a < dim) { V[a][p] = v[a]; X[a][p] = x[a]; }
    s.rho[p] = rh;
    s.E[p] = En;
    s.d[p] = d;
    r.d1 = dkey(d);
    if (P.vref) {
      // Verlet-list validity: a listed superset of the pairs within kappa h_ij holds as long
      // as |x_i - x_i^b - U| + kh max(0, d_i - d_i^b) <= beta kh d_i^b for every particle
      // (b: the last build).  U is one displacement shared by all particles, any vector:
      // the separation of a pair changes by (x_j - x_j^b - U) - (x_i - x_i^b - U), so
      // summing the bounds of i and j covers the pair.  U follows the bulk motion (the
      // midpoint of the displacement box, extrapolated from the previous step), so a body
      // in uniform motion keeps its lists.  Kept with a 5 % margin (differences in FP64,
      // the bound itself in FP32: the 5 % margin dwarfs its rounding).
      // (The displacement and U in FP32: their rounding, ~1e-7 of each, is far
      // inside the margin.)  The box is that of x - x^b - U.
      const float* Uf = reinterpret_cast<const float*>(P.vframe + 6 * inst + 4);
      float dsq = 0.0f;
#pragma unroll
      for (int a = 0; a < 3; ++a)
        if (a < dim) {
          const float dx = f32_rn(x[a] - xb[a]) - Uf[a];
          dsq += dx * dx;
          r.dlo[a] = r.dhi[a] = fkey(dx);
        }
      const float kh = P.kh_f;
      const float crit = sqrtf(dsq) + kh * fmaxf(f32_rn(d - db), 0.0f) - 0.95f * P.cell_beta_f * kh * f32_rn(db);
      r.viol = dkey(f64_of(crit));
    }
    if (!finite || !finite_bits(d)) set_status(status, SPH_ERR_NONFINITE);
  }
  block_reduce(r, P.dim, P.vref != nullptr);
  if (threadIdx.x == 0) {
    write_part(part, r);
    if (P.vacc) {                  // the criterion's maximum and displacement box of the instance
      VAcc* va = P.vacc + inst;
      atomicMax(&va->viol, r.viol);
#pragma unroll
      for (int a = 0; a < 3; ++a) {
        atomicMin(&va->dlo[a], r.dlo[a]);
        atomicMax(&va->dhi[a], r.dhi[a]);
      }
    }
  }
}

// Second half kick with the rates of the predicted state; instance time.
// With dt_key, also the instance's minimum of the CFL keys at the new state,
// which the next step of the same sph_step call takes instead of a k_cfl pass.
template <bool MIXED>
__global__ void k_kick2(DevParams P, sph_state s, const int64_t* __restrict__ blk_start,
                        const int64_t* __restrict__ blk_end, const int32_t* __restrict__ blk_inst,
                        const int32_t* __restrict__ inst_blk, const double* __restrict__ dt, double* t_dev,
                        long long* dt_key) {
  chain_entry();
  const int64_t p = blk_start[blockIdx.x] + threadIdx.x;
  const int b = blk_inst[blockIdx.x];
  if (t_dev && threadIdx.x == 0 && inst_blk[b] == (int)blockIdx.x) t_dev[b] += dt[b];
  long long key = LLONG_MAX;
  if (p < blk_end[blockIdx.x]) {
    const int dim = P.dim;
    const double hdt = 0.5 * dt[b];
    double* V[3] = {s.vx, s.vy, s.vz};
    const double* A[3] = {s.ax, s.ay, s.az};
    double v[3] = {0.0, 0.0, 0.0}, acc[3] = {0.0, 0.0, 0.0};
#pragma unroll
    for (int a = 0; a < 3; ++a)
      if (a < dim) { v[a] = V[a][p]; acc[a] = A[a][p]; }
    const double rho0 = s.rho[p], drho = s.drho[p], E0 = s.E[p], dE = s.dE[p];
    double m = 0.0;
    int mi = 0;
    if (dt_key) { m = s.m[p]; mi = s.mat ? s.mat[p] : 0; }
#pragma unroll
    for (int a = 0; a < 3; ++a)
      if (a < dim) v[a] = axpy<MIXED>(hdt, acc[a], v[a]);
    const double rho = axpy<MIXED>(hdt, drho, rho0);
    const double E = axpy<MIXED>(hdt, dE, E0);
#pragma unroll
    for (int a = 0; a < 3; ++a)
      if (a < dim) V[a][p] = v[a];
    s.rho[p] = rho;
    s.E[p] = E;
    if (dt_key) key = cfl_key(P, v[0], v[1], v[2], E, rho, m, mi);
  }
  if (dt_key) {   // uniform over the grid: every thread reaches the block barrier
    const long long k = block_min_key(key);
    if (threadIdx.x == 0) atomicMin(&dt_key[b], k);
  }
}

// ---------------------------------------------------------------------------
// Pack the pair operands in slot order.  With predict, the state holds the
// half-step values q^h and the rates q' of the previous evaluation and the
// operands are the predicted q~ = q^h + dt/2 q'.  P and c of the packed state
// are written back to the particle arrays.
//   mixed: A = {x - o, y - o, z - o, d} (FP32 offsets from the particle's own
//          cell origin o, the local-origin idea of Sec. 3.1), B = {v, m/rho},
//          C = {P, rho c}
//   fp64 : A = {x, y, z, d} (global positions), B, C in FP64
// Bound by the latency of its gathers (FP64 pipe 62 %, DRAM 43 % of peak at
// 1.125M), so mixed runs 6 blocks an SM although that spills a few words: five
// steps of the 1.125M plate impact with lists 5405 / 5376 / 5345 us at 4 / 5 / 6.
// ---------------------------------------------------------------------------
template <bool MIXED>
__global__ void __launch_bounds__(kBlock, MIXED ? 6 : 4) k_pack(DevParams P, sph_state s, const int64_t* __restrict__ blk_start,
                       const int64_t* __restrict__ blk_end, const int32_t* __restrict__ blk_inst,
                       const GridInfo* __restrict__ grid, const double* __restrict__ dt, int predict,
                       const int32_t* __restrict__ perm, const int32_t* __restrict__ cell_of,
                       void* packA, void* packB, void* packC, double* rho_slot, int32_t* slot_cell,
                       int32_t* slot_unit, int n_units, int* status, const int32_t* __restrict__ e_of_c,
                       int32_t* perm_e, void* packAc, const int* __restrict__ gate,
                       unsigned long long* counters, int keep_counts, const int32_t* __restrict__ inst_blk,
                       long long* dt_key) {
  chain_entry();
  // the counters of the pair kernels that follow: the evaluation's pair counts
  // (kept by the reverse mode) and the work counters
  if (counters && blockIdx.x == 0 && threadIdx.x == 0) {
    if (!keep_counts) {
      counters[0] = 0ull;
      counters[1] = 0ull;
      counters[2] = 0ull;
      counters[4] = 0ull;
    }
    counters[5] = 0ull;
    counters[7] = 0ull;
  }
  // the CFL keys, read by the kick-drift, are ready for the next accumulation
  if (dt_key && threadIdx.x == 0 && inst_blk[blk_inst[blockIdx.x]] == (int)blockIdx.x) dt_key[blk_inst[blockIdx.x]] = LLONG_MAX;
  const int64_t sc = blk_start[blockIdx.x] + threadIdx.x;     // cell-order slot
  if (sc >= blk_end[blockIdx.x]) return;
  // the operands go to the slot's evaluation position (unit-major order of the
  // last list build), or to the cell-order slot itself
  const int64_t sl = e_of_c ? (int64_t)e_of_c[sc] : sc;
  const bool build = packAc && gate && gate[0] != 0;          // a list build follows: cell-order copy of A
  int b = blk_inst[blockIdx.x];
  int64_t p = perm[sc];
  if (perm_e) perm_e[sl] = (int32_t)p;
  // every load of the gathered particle first (the stores to P and c below
  // would otherwise hold back the loads placed after them)
  const bool pr = predict != 0;
  double v[3] = {ld(s.vx, p), ld(s.vy, p), ld(s.vz, p)};
  double acc[3] = {0.0, 0.0, 0.0};
  if (pr) {
    acc[0] = s.ax[p];
    if (P.dim >= 2) acc[1] = s.ay[p];
    if (P.dim >= 3) acc[2] = s.az[p];
  }
  const double rho0 = s.rho[p], E0 = s.E[p];
  const double drho = pr ? s.drho[p] : 0.0, dE = pr ? s.dE[p] : 0.0;
  const int mi = s.mat ? s.mat[p] : 0;
  const double d = s.d[p];
  const double m = s.m[p];
  const double X[3] = {s.x[p], P.dim >= 2 ? s.y[p] : 0.0, P.dim >= 3 ? s.z[p] : 0.0};
  const int32_t gc = cell_of[p];
  int32_t u = s.unit ? s.unit[p] : 0;
  const double hdt = pr ? 0.5 * dt[b] : 0.0;
  if (pr) {
    v[0] = axpy<MIXED>(hdt, acc[0], v[0]);
    if (P.dim >= 2) v[1] = axpy<MIXED>(hdt, acc[1], v[1]);
    if (P.dim >= 3) v[2] = axpy<MIXED>(hdt, acc[2], v[2]);
  }
  double rho = pr ? axpy<MIXED>(hdt, drho, rho0) : rho0;
  double E = pr ? axpy<MIXED>(hdt, dE, E0) : E0;
  double e = E - 0.5 * (v[0] * v[0] + v[1] * v[1] + v[2] * v[2]);
  double Pp, cp;
  float cf = 0.0f;
  const Mat& mt = P.mat[mi];
  const bool fast = MIXED && predict &&
                    (mt.eos == SPH_EOS_IDEAL || mt.eos == SPH_EOS_STIFFENED || (mt.eos == SPH_EOS_TAIT && mt.tait_n > 0));
  if (fast) {
    // a mixed step packs FP32 operands: P in FP64 (the stiffened-gas and Tait
    // differences of two large terms, the expressions of eos()), c in FP32
    if (mt.eos == SPH_EOS_TAIT) Pp = mt.tait_B * (ipow(rho / mt.rho0, mt.tait_n) - 1.0);
    else Pp = (mt.gamma - 1.0) * rho * e - (mt.eos == SPH_EOS_STIFFENED ? mt.gamma * mt.p_inf : 0.0);
    cf = sound_speed_f32(mt, f32_rn(rho), f32_rn(e));
    cp = f64_of(cf);
  } else {
    eos(mt, rho, e, Pp, cp);
    cf = (float)cp;
  }
  s.P[p] = Pp;
  s.c[p] = cp;
  slot_cell[sl] = gc;
  if (u < 0 || u >= n_units) { if (n_units > 0) set_status(status, SPH_ERR_INVALID); u = 0; }
  slot_unit[sl] = u;
  rho_slot[sl] = rho;
  if (MIXED) {
    // FP32 offsets from the slot's cell origin (written at the mesh build)
    float off[3] = {0.f, 0.f, 0.f};
#pragma unroll
    for (int a = 0; a < 3; ++a)
      if (a < P.dim) off[a] = f32_rn(X[a] - P.slot_org[(int64_t)a * P.n + sc]);
    const float4 Arec = make_float4(off[0], off[1], off[2], f32_rn(d));
    reinterpret_cast<float4*>(packA)[2 * sl] = Arec;
    if (build) reinterpret_cast<float4*>(packAc)[sc] = Arec;
    const float Vp = fast ? (f32_rn(m) / f32_rn(rho)) * P.vscale_f : (float)((m / rho) * P.vscale);
    // FP32 velocities relative to a reference velocity of whole m/s per
    // particle (k = v truncated, |k| <= 32767): v - k is exact in FP64 and
    // small, so FP32 keeps the velocity differences between neighbours to
    // ~1e-8 m/s instead of one ulp of the bulk velocity.  The references are
    // stored exactly: x and y biased by 32768 in the halves of one word,
    // z as a float.
    int k[3] = {0, 0, 0};
    float vr[3] = {0.f, 0.f, 0.f};
#pragma unroll
    for (int a = 0; a < 3; ++a)
      if (a < P.dim) vr[a] = f32_rn(v[a] - trunc_ref(v[a], k[a]));
    const uint32_t kxy = (uint32_t)(k[0] + 32768) | ((uint32_t)(k[1] + 32768) << 16);
    reinterpret_cast<float4*>(packA)[2 * sl + 1] = make_float4(vr[0], vr[1], vr[2], Vp);
    reinterpret_cast<float4*>(packC)[sl] = make_float4(f32_rn(Pp), fast ? f32_rn(rho) * cf : (float)(rho * cp),
                                                       __uint_as_float(kxy), (float)k[2]);
  } else {
    reinterpret_cast<D4*>(packA)[sl] = D4{X[0], X[1], X[2], d};
    if (build) reinterpret_cast<D4*>(packAc)[sc] = D4{X[0], X[1], X[2], d};
    reinterpret_cast<D4*>(packB)[sl] = D4{v[0], v[1], v[2], m / rho};
    reinterpret_cast<D2*>(packC)[sl] = D2{Pp, rho * cp};
  }
}

// ---------------------------------------------------------------------------
// Renumbering: gather every per-particle array through perm, copy back.
// ---------------------------------------------------------------------------
constexpr int kMaxPermArrays = 24;
struct PermArrays {
  void* ptr[kMaxPermArrays];
  int bytes[kMaxPermArrays];   // element size: 4 or 8
  int count;
};

__global__ void k_gather(int64_t n, const int32_t* __restrict__ perm, PermArrays a, char* scratch) {
  int64_t sl = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (sl >= n) return;
  int64_t p = perm[sl];
  size_t off = 0;
  for (int k = 0; k < a.count; ++k) {
    if (a.bytes[k] == 8) reinterpret_cast<uint64_t*>(scratch + off)[sl] = reinterpret_cast<const uint64_t*>(a.ptr[k])[p];
    else reinterpret_cast<uint32_t*>(scratch + off)[sl] = reinterpret_cast<const uint32_t*>(a.ptr[k])[p];
    off += (size_t)a.bytes[k] * n;
  }
}

// Writes the gathered arrays back; with perm, also makes the slot order the
// identity (particle sl now sits in slot sl).
__global__ void k_scatter_back(int64_t n, PermArrays a, const char* scratch, int32_t* perm) {
  int64_t sl = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (sl >= n) return;
  size_t off = 0;
  for (int k = 0; k < a.count; ++k) {
    if (a.bytes[k] == 8) reinterpret_cast<uint64_t*>(a.ptr[k])[sl] = reinterpret_cast<const uint64_t*>(scratch + off)[sl];
    else reinterpret_cast<uint32_t*>(a.ptr[k])[sl] = reinterpret_cast<const uint32_t*>(scratch + off)[sl];
    off += (size_t)a.bytes[k] * n;
  }
  if (perm) perm[sl] = (int32_t)sl;
}

// ---------------------------------------------------------------------------
// FP64 conservation sums per instance, fixed order: one cluster of CTAs per
// instance, its threads striding over the instance's particles.  The CTAs that
// take part follow from the instance's own size, not from the launch's clusters
// (those past them add zeros), so that an instance's totals are the same bits
// whatever shares its handle.  A single CTA per instance (one SM's FP64 pipe,
// two loads in flight) took 3.3 ms on 1M particles, a cluster of 16 takes 0.1 ms.
// ---------------------------------------------------------------------------
constexpr int64_t kSumEach = 4096;   // particles per CTA of a sum
__global__ void __launch_bounds__(kSumBlock) k_conservation(sph_state s, const int64_t* __restrict__ inst_off, double* out) {
  namespace cg = cooperative_groups;
  const cg::cluster_group cl = cg::this_cluster();
  const int per = (int)cl.num_blocks(), rank = (int)cl.block_rank();
  const int b = blockIdx.x / per;
  double acc[5] = {0, 0, 0, 0, 0};
  const int64_t p0 = inst_off[b], p1 = inst_off[b + 1];
  const int parts = cluster_size_for(per, p1 - p0, kSumEach);   // the largest instance's is per: see the launch
  const int64_t stride = (int64_t)parts * kSumBlock;
#pragma unroll 2
  for (int64_t p = rank < parts ? p0 + (int64_t)rank * kSumBlock + threadIdx.x : p1; p < p1; p += stride) {
    const double m = s.m[p];
    acc[0] += m;
    acc[1] += m * ld(s.vx, p);
    acc[2] += m * ld(s.vy, p);
    acc[3] += m * ld(s.vz, p);
    acc[4] += m * s.E[p];
  }
  if (cluster_sum(acc))
    for (int k = 0; k < 5; ++k) out[b * 5 + k] = acc[k];
}

__global__ void k_check_finite(int dim, sph_state s, int64_t n, int* status) {
  int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (p >= n) return;
  bool ok = isfinite(s.x[p]) && isfinite(s.vx[p]) && isfinite(s.rho[p]) && isfinite(s.E[p]) &&
            isfinite(s.m[p]) && s.rho[p] > 0.0 && s.m[p] > 0.0;
  if (dim >= 2) ok = ok && isfinite(s.y[p]) && isfinite(s.vy[p]);
  if (dim >= 3) ok = ok && isfinite(s.z[p]) && isfinite(s.vz[p]);
  if (!ok) set_status(status, SPH_ERR_NONFINITE);
}

}  // namespace

// ---------------------------------------------------------------------------
// Launchers
// ---------------------------------------------------------------------------
// Grids over the mesh capacity, whose kernels read the live cell count on the
// device and stride over it: at most 8 blocks of kBlock per SM, so a generous
// capacity costs no empty waves.
static int capped_grid(int want) {
  static int cap = 0;
  if (cap == 0) {
    int dev = 0, sms = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    cap = 8 * (sms > 0 ? sms : 1);
  }
  return want < cap ? (want > 0 ? want : 1) : cap;
}

cudaError_t launch_derive(sph_handle* h, const sph_state& s, cudaStream_t st) {
  CKL(launch_chained(k_derive, dim3(h->nblk), dim3(kBlock), st, h->dp, s, h->blk_start, h->blk_end, h->part));
  h->launches += 1;
  return cudaGetLastError();
}

cudaError_t launch_cfl(sph_handle* h, const sph_state& s, cudaStream_t st) {
  CKL(launch_chained(k_cfl, dim3(h->nblk), dim3(kBlock), st, h->dp, s, h->blk_start, h->blk_end, h->blk_inst, h->dt_key));
  h->launches += 1;
  return cudaGetLastError();
}

cudaError_t launch_reduce_dt(sph_handle* h, cudaStream_t st) {
  CKL(launch_chained(k_reduce_dt, dim3(grid_for(h->n_inst, kBlock)), dim3(kBlock), st, h->n_inst, h->dp.cfl, h->dt, h->dt_key));
  h->launches += 1;
  return cudaGetLastError();
}

cudaError_t launch_kick_drift(sph_handle* h, const sph_state& s, cudaStream_t st, bool from_key) {
  const long long* key = from_key ? h->dt_key : nullptr;
  if (h->dp.precision == SPH_PREC_MIXED)
    CKL(launch_chained(k_kick_drift<true>, dim3(h->nblk), dim3(kBlock), st, h->dp, s, h->blk_start, h->blk_end, h->blk_inst,
                       h->inst_blk, h->dt, key, h->part, h->status));
  else
    CKL(launch_chained(k_kick_drift<false>, dim3(h->nblk), dim3(kBlock), st, h->dp, s, h->blk_start, h->blk_end, h->blk_inst,
                       h->inst_blk, h->dt, key, h->part, h->status));
  h->launches += 1;
  return cudaGetLastError();
}

cudaError_t launch_verlet_flag(sph_handle* h, cudaStream_t st) {
  CKL(launch_chained(k_verlet_flag, dim3(1), dim3(h->n_inst < 1024 ? 32 * ((h->n_inst + 31) / 32) : 1024), st,
                     h->vflag, h->vframe, h->vacc, h->n_inst, h->vinst, h->unit_sched != SPH_SCHED_GLOBAL ? 1 : 0));
  h->launches += 1;
  return cudaGetLastError();
}

// Mesh from the block partials left by k_derive or k_kick_drift, then the
// counting sort of particles into cells.
cudaError_t launch_build_grid(sph_handle* h, const sph_state& s, cudaStream_t st, const int* gate) {
  MeshArgs a;
  a.P = h->dp;
  a.x = s.x; a.y = s.y; a.z = s.z;
  a.n_inst = h->n_inst; a.nblk = h->nblk;
  a.inst_off = h->inst_off; a.inst_cap = h->inst_cap; a.blk_start = h->blk_start; a.blk_end = h->blk_end;
  a.blk_inst = h->blk_inst; a.inst_blk = h->inst_blk;
  a.part = h->part; a.grid = h->grid; a.total_cells = h->total_cells;
  a.cell_count = h->cell_count; a.cell_start = h->cell_start; a.scan_sums = h->scan_sums;
  a.cell_of = h->cell_of; a.rank = h->rank; a.perm = h->perm; a.slot_org = h->slot_org;
  a.status = h->status;
  a.gate = gate;
  // per-instance rebuilds only inside the Verlet sequence (gated) of a batched
  // handle; any other build is global (one instance: the same thing)
  a.vinst = gate && h->n_inst > 1 ? h->vinst : nullptr;
  if (h->n_inst > 1) {
    CKL(launch_chained(k_mesh_reduce, dim3(h->n_inst), dim3(kBlock), st, a));
    h->launches += 1;
  }
  CKL(launch_chained(k_mesh_setup, dim3(1), dim3(h->n_inst == 1 ? kBlock : (h->n_inst < 1024 ? 32 * ((h->n_inst + 31) / 32) : 1024)),
                     st, a));
  CKL(launch_chained(k_cell_count, dim3(capped_grid(h->nblk)), dim3(kBlock), st, a));
  int tiles = capped_grid(grid_for(h->cell_cap, kScanTile));
  CKL(launch_chained(k_scan_reduce, dim3(tiles), dim3(kBlock), st, h->cell_count, h->total_cells, h->scan_sums, gate));
  CKL(launch_chained(k_scan_down, dim3(tiles), dim3(kBlock), st, h->cell_count, h->total_cells, h->scan_sums, h->cell_start, h->n, gate));
  CKL(launch_chained(k_cell_scatter, dim3(capped_grid(grid_for(h->n, kBlock))), dim3(kBlock), st, a));
  CKL(launch_chained(k_cell_sort, dim3(capped_grid(grid_for(h->cell_cap * 32, kBlock))), dim3(kBlock), st, a));
  h->launches += 6;
  // a mesh built outside the Verlet sequence changes the slot order under the lists
  if (!gate && h->verlet) return cudaMemsetAsync(&h->vflag[1], 0xff, sizeof(int), st);
  return cudaGetLastError();
}

cudaError_t launch_pack(sph_handle* h, const sph_state& s, bool predict, cudaStream_t st, bool eorder,
                        bool keep_counts) {
  const int kc = keep_counts ? 1 : 0;
  const int32_t* eoc = eorder ? h->e_of_c : nullptr;
  int32_t* pe = eorder ? h->perm_e : nullptr;
  void* Ac = h->packAc;   // written only when a list build follows
  if (h->dp.precision == SPH_PREC_MIXED)
    CKL(launch_chained(k_pack<true>, dim3(h->nblk), dim3(kBlock), st, h->dp, s, h->blk_start, h->blk_end, h->blk_inst, h->grid, h->dt,
                                             predict ? 1 : 0, h->perm, h->cell_of, h->packA, h->packB, h->packC,
                                             h->rho_slot, h->slot_cell, h->slot_unit, h->K, h->status, eoc, pe, Ac,
                                             h->vflag, h->counters, kc, h->inst_blk, h->dt_key));
  else
    CKL(launch_chained(k_pack<false>, dim3(h->nblk), dim3(kBlock), st, h->dp, s, h->blk_start, h->blk_end, h->blk_inst, h->grid, h->dt,
                                              predict ? 1 : 0, h->perm, h->cell_of, h->packA, h->packB, h->packC,
                                              h->rho_slot, h->slot_cell, h->slot_unit, h->K, h->status, eoc, pe, Ac,
                                              h->vflag, h->counters, kc, h->inst_blk, h->dt_key));
  h->launches += 1;
  return cudaGetLastError();
}


// k_pack's FP64 variant into the given operand arrays (the FP64 reverse pass
// of a mixed-precision handle).
cudaError_t launch_pack_fp64(sph_handle* h, const sph_state& s, bool predict, void* A, void* B, void* C,
                             double* rho_out, cudaStream_t st) {
  k_pack<false><<<h->nblk, kBlock, 0, st>>>(h->dp, s, h->blk_start, h->blk_end, h->blk_inst, h->grid, h->dt,
                                            predict ? 1 : 0, h->perm, h->cell_of, A, B, C, rho_out, h->slot_cell,
                                            h->slot_unit, h->K, h->status, nullptr, nullptr, nullptr, nullptr, h->counters, 1,
                                            h->inst_blk, h->dt_key);
  h->launches += 1;
  return cudaGetLastError();
}

cudaError_t launch_kick2(sph_handle* h, const sph_state& s, double* t_dev, cudaStream_t st, bool next_dt) {
  long long* key = next_dt ? h->dt_key : nullptr;
  if (h->dp.precision == SPH_PREC_MIXED)
    CKL(launch_chained(k_kick2<true>, dim3(h->nblk), dim3(kBlock), st, h->dp, s, h->blk_start, h->blk_end, h->blk_inst, h->inst_blk, h->dt,
                                              t_dev, key));
  else
    CKL(launch_chained(k_kick2<false>, dim3(h->nblk), dim3(kBlock), st, h->dp, s, h->blk_start, h->blk_end, h->blk_inst, h->inst_blk, h->dt,
                                               t_dev, key));
  h->launches += 1;
  return cudaGetLastError();
}

cudaError_t launch_renumber(sph_handle* h, sph_state& s, cudaStream_t st, const int32_t* order) {
  PermArrays a;
  a.count = 0;
  auto add = [&](void* ptr, int bytes) {
    if (ptr) { a.ptr[a.count] = ptr; a.bytes[a.count] = bytes; ++a.count; }
  };
  add(s.x, 8); add(s.y, 8); add(s.z, 8);
  add(s.vx, 8); add(s.vy, 8); add(s.vz, 8);
  add(s.rho, 8); add(s.E, 8); add(s.m, 8);
  add(s.ax, 8); add(s.ay, 8); add(s.az, 8); add(s.drho, 8); add(s.dE, 8);
  add(s.d, 8); add(s.P, 8); add(s.c, 8);
  add(s.id, 8);
  add(s.mat, 4); add(s.unit, 4);
  int g = grid_for(h->n, kBlock);
  k_gather<<<g, kBlock, 0, st>>>(h->n, order ? order : h->perm, a, reinterpret_cast<char*>(h->scratch));
  k_scatter_back<<<g, kBlock, 0, st>>>(h->n, a, reinterpret_cast<const char*>(h->scratch), nullptr);
  h->launches += 2;
  if (!h->verlet) return cudaGetLastError();
  // another order than the slot order (the unit-major evaluation order) moves
  // particles between slots under the Verlet lists: rebuild them
  if (order) return cudaMemsetAsync(&h->vflag[1], 0xff, sizeof(int), st);
  // In slot order the mesh, the slots and the lists stay as they are: particle
  // q is now the one in slot q, so the slot permutation becomes the identity,
  // and each particle's cell and the build-time positions and sizes of the
  // validity criterion follow their particles.
  PermArrays b;
  b.count = 0;
  for (int k = 0; k < 4; ++k)
    if (k < h->dp.dim || k == 3) {
      b.ptr[b.count] = h->vref + (size_t)k * h->n;
      b.bytes[b.count] = 8;
      ++b.count;
    }
  b.ptr[b.count] = h->cell_of;
  b.bytes[b.count] = 4;
  ++b.count;
  k_gather<<<g, kBlock, 0, st>>>(h->n, h->perm, b, reinterpret_cast<char*>(h->scratch));
  k_scatter_back<<<g, kBlock, 0, st>>>(h->n, b, reinterpret_cast<const char*>(h->scratch), h->perm);
  h->launches += 2;
  return cudaGetLastError();
}

cudaError_t launch_exclusive_scan(int32_t* cnt, const int64_t* total, int32_t* sums, int32_t* start,
                                  int64_t n_total, int64_t cap, cudaStream_t st, const int* gate) {
  int tiles = capped_grid(grid_for(cap, kScanTile));
  k_scan_reduce<<<tiles, kBlock, 0, st>>>(cnt, total, sums, gate);
  k_scan_down<<<tiles, kBlock, 0, st>>>(cnt, total, sums, start, n_total, gate);
  return cudaGetLastError();
}
// (launch_exclusive_scan's two kernels are counted by its callers)

cudaError_t launch_conservation(sph_handle* h, const sph_state& s, double* out, cudaStream_t st) {
  int64_t most = 0;                    // the largest instance
  for (int b = 0; b < h->n_inst; ++b) most = std::max(most, h->inst_off_h[b + 1] - h->inst_off_h[b]);
  const int per = cluster_size_for(largest_cluster<k_conservation>(kSumBlock), most, kSumEach);
  CKL(launch_clusters(k_conservation, h->n_inst, per, kSumBlock, st, s, h->inst_off, out));
  h->launches += 1;
  return cudaGetLastError();
}

// Largest particle volume m / rho (positive doubles order like their bit patterns).
__global__ void k_max_volume(int64_t n, const double* __restrict__ m, const double* __restrict__ rho,
                             unsigned long long* out) {
  unsigned long long b = 0ull;
  for (int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; p < n; p += (int64_t)gridDim.x * blockDim.x) {
    const double v = m[p] / rho[p];
    if (v > 0.0 && v < 1e300) {
      const unsigned long long q = (unsigned long long)__double_as_longlong(v);
      b = q > b ? q : b;
    }
  }
  for (int o = 16; o > 0; o >>= 1) {
    const unsigned long long q = __shfl_xor_sync(0xffffffffu, b, o);
    b = q > b ? q : b;
  }
  if ((threadIdx.x & 31) == 0 && b) atomicMax(out, b);
}

cudaError_t launch_max_volume(sph_handle* h, const sph_state& s, unsigned long long* out, cudaStream_t st) {
  k_max_volume<<<capped_grid(grid_for(h->n, kBlock)), kBlock, 0, st>>>(h->n, s.m, s.rho, out);
  h->launches += 1;
  return cudaGetLastError();
}

cudaError_t launch_check_finite(sph_handle* h, const sph_state& s, cudaStream_t st) {
  k_check_finite<<<grid_for(h->n, kBlock), kBlock, 0, st>>>(h->dp.dim, s, h->n, h->status);
  h->launches += 1;
  return cudaGetLastError();
}

}  // namespace csph
