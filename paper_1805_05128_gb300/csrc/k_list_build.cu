// k_list_build.cu -- the Verlet list build: every pair within
// (1 + beta) kappa h_ij of the current positions (Sec. 4.2 with the buffered
// horizon of eq. (Dcell)), written as one list per slot for k_pair_lists.
//
// One warp per home cell, lane l owning home particle start_c + chunk + l (a
// cell of edge (1 + beta) D^c holds 27 particles of a lattice, so a warp per
// cell fills its lanes here).  For each neighbour row (the 3 x-consecutive
// cells at (oy, oz), contiguous in slot order) each lane loads one candidate;
// those within reach of the home group's bounding box enter a queue in shared
// memory, in order.  Whenever the queue holds 32, every lane tests its own
// home particle against each (broadcast reads, two candidates per packed FP32
// operation) into a bit mask, and the warp writes, home particle by home
// particle, the entries of the set bits to consecutive places of its row: lane
// c holds candidate c's entry, (slot j << 5) | (ox+1) + 3 (oy+1) + 9 (oz+1).
//
// The test runs in FP32 in both precisions (mixed handles on the packed
// offsets from the cell origins, FP64 handles on offsets from the cell's first
// particle scaled to a cell edge of ~1).  Mixed handles accept r^2 - R^2 < 2^-12
// D^c^2, a superset of the radius: k_pair_lists decides each entry exactly.  FP64
// handles decide the candidates within 2^-17 D^c^2 of R^2 in FP64, so that a row
// holds the radius and nothing beyond it, however far the particle sizes lie
// apart.  (Their FP32 error is below 2^-19 D^c^2: offsets of at most two edges,
// rounded to 2^-23 D^c each, three products of at most D^c^2, and an R of four
// roundings; a superset like the mixed one would hold ten times the radius
// between particles 600 times smaller than the largest.)
// Bound by issue (77 % of the slots) and the latency of its short phases:
// 659 us at 1.125M particles, 768 us at 1M droplet particles.  Rows gathered in
// shared memory, one append per test and lane, and flushed at the end (33 KB a
// block, scalar tests, 68 % of the issue slots): 740 and 854 us.
#include "pair_common.cuh"

namespace csph {

namespace {

constexpr int kQueue = 64;         // under 32 waiting candidates and a chunk of 32

// Minimum / maximum over a full warp (one redux instruction; a NaN loses).
__device__ __forceinline__ float warp_min(float v) {
  float r;
  asm volatile("redux.sync.min.f32 %0, %1, 0xffffffff;" : "=f"(r) : "f"(v));
  return r;
}
__device__ __forceinline__ float warp_max(float v) {
  float r;
  asm volatile("redux.sync.max.f32 %0, %1, 0xffffffff;" : "=f"(r) : "f"(v));
  return r;
}

// The candidates of `mask` (places in `slots`) that lie within R of slot i, in
// FP64 and the oracle's operation order.  A call, because it is rare and its
// code inside the drain cost the whole build 3 %: two steps of the 65k ejecta
// cloud 1657 us without the decision, 1680 inlined, 1656 called.
template <int DIM>
__device__ __noinline__ unsigned decide_exactly(const D4* A, int i, unsigned mask, const int32_t* slots, double kh) {
  unsigned left = mask;
  for (unsigned m = mask; m; m &= m - 1) {
    const int c = __ffs(m) - 1;
    const D4 Ai = A[i], Aj = A[slots[c]];
    const double r2 = Pair<false, DIM>::r2_of(__dsub_rn(Aj.x, Ai.x), DIM >= 2 ? __dsub_rn(Aj.y, Ai.y) : 0.0,
                                              DIM >= 3 ? __dsub_rn(Aj.z, Ai.z) : 0.0);
    const double R = __dmul_rn(kh, __dadd_rn(Ai.w, Aj.w));
    if (!(r2 < __dmul_rn(R, R))) left &= ~(1u << c);
  }
  return left;
}

// Resident blocks: mixed 8 / 7 / 6 took 5305 / 5212 / 5230 us for five steps of
// the 1.125M plate impact; FP64 7 / 6 took 1676 / 1657 us for two of a 65k ejecta cloud.
template <bool MIXED, int DIM>
__global__ void __launch_bounds__(kPairBlock, MIXED ? 7 : 6) k_list_build(PairArgs a) {
  chain_entry();
  using T = typename Ops<MIXED>::T;
  using V4 = typename Ops<MIXED>::V4;
  using F = Pair<true, DIM>;
  // the queue, component by component: x, y, z in the home cell's frame, d
  __shared__ alignas(16) float qx[kWarps][kQueue], qy[kWarps][kQueue], qz[kWarps][kQueue], qd[kWarps][kQueue];
  __shared__ uint32_t qword[kWarps][kQueue];                 // the entry of a row
  __shared__ int32_t qslot[kWarps][kQueue];                  // the candidate's slot in cell order
  __shared__ int32_t nb_start[kWarps][27];                   // start slot of each neighbour cell

  if (a.vflag[0] == 0) return;                               // lists still valid: nothing to build
  if (blockIdx.x == 0 && threadIdx.x == 0) { a.vflag[1] = 0; a.vflag[2] += 1; }
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const unsigned lt = (1u << lane) - 1u;
  const int64_t total = *a.total_cells_dev;
  // positions and sizes in cell order: k_pack's copy (mixed handles, whose packs
  // hold B beside A, and unit-major evaluation orders), else the pack itself
  const V4* __restrict__ A = reinterpret_cast<const V4*>(a.Ac ? a.Ac : a.A);
  // Persistent warps: each takes the next cell from a global counter, so the
  // work spreads evenly whatever the mix of empty and crowded cells.
  for (;;) {
    int64_t cell_g = 0;
    if (lane == 0) cell_g = (int64_t)atomicAdd(a.work_counter, 1ull);
    cell_g = __shfl_sync(0xffffffffu, cell_g, 0);
    if (cell_g >= total) break;
    const int hs = a.cell_start[cell_g], he = a.cell_start[cell_g + 1];
    if (hs == he) continue;                                  // empty cell (warp-uniform)

    int b = 0;
    if (a.n_inst > 1) {  // instance of this cell: binary search of the slot offsets
      int lo = 0, hi = a.n_inst;
      while (hi - lo > 1) {
        int mid = (lo + hi) >> 1;
        if (a.inst_off[mid] <= hs) lo = mid; else hi = mid;
      }
      b = lo;
    }
    if (a.vinst && a.vinst[b] == 0) continue;                // the instance keeps its lists (warp-uniform)
    const GridInfo& g = a.grid[b];
    const int nx = g.dims[0], ny = g.dims[1], nz = g.dims[2];
    const int64_t lc = cell_g - g.cell_off;
    const int cx = (int)(lc % nx), cy = (int)((lc / nx) % ny), cz = (int)(lc / ((int64_t)nx * ny));
    // FP32 frame of the test
    int ex = 0;
    double fx = 0.0, fy = 0.0, fz = 0.0;
    float dct = MIXED ? g.dc_f : 0.f;
    if constexpr (!MIXED) {
      ex = exponent_of(g.dc);
      dct = f32_scaled(g.dc, ex);
      const V4 O = A[hs];
      fx = O.x; fy = O.y; fz = O.z;
    }
    const float band = (MIXED ? 0x1p-12f : 0x1p-17f) * dct * dct;
    auto frame = [&](const V4& R, int ox, int oy, int oz) {
      float4 S;
      if constexpr (MIXED) {
        S = R;
        S.x += (float)ox * dct; S.y += (float)oy * dct; S.z += (float)oz * dct;
      } else {
        S.x = f32_scaled(R.x - fx, ex);
        S.y = DIM >= 2 ? f32_scaled(R.y - fy, ex) : 0.f;
        S.z = DIM >= 3 ? f32_scaled(R.z - fz, ex) : 0.f;
        S.w = f32_scaled(R.w, ex);
      }
      return S;
    };

    // starts of the 27 neighbour cells (index (ox+1) + 3 (oy+1) + 9 (oz+1)); -1 outside the mesh
    if (lane < 27) {
      const int ox = lane % 3 - 1, oy = (lane / 3) % 3 - 1, oz = lane / 9 - 1;
      const int xx = cx + ox, yy = cy + oy, zz = cz + oz;
      const bool in = xx >= 0 && xx < nx && yy >= 0 && yy < ny && zz >= 0 && zz < nz;
      nb_start[warp][lane] = in ? a.cell_start[g.cell_off + xx + (int64_t)nx * (yy + (int64_t)ny * zz)] : -1;
    }
    __syncwarp();

    for (int h0 = hs; h0 < he; h0 += 32) {
      const int i = h0 + lane;
      const bool act = i < he;
      const int nh = min(32, he - h0);
      const int ii = act ? i : hs;
      const float4 H = frame(A[ii], 0, 0, 0);
      const float khdi = a.kh_f * H.w;
      const int row_i = a.e_of_c ? a.e_of_c[ii] : ii;        // the row's slot
      int vc = 0;
      // the home group's bounding box and largest kh d, a warp-wide cull of candidates
      const float bxl = warp_min(H.x), bxh = warp_max(H.x), byl = warp_min(H.y), byh = warp_max(H.y);
      const float bzl = warp_min(H.z), bzh = warp_max(H.z), bkh = warp_max(khdi);
      int head = 0, tail = 0;                                // of the queue (warp-uniform); head a multiple of 32

      // the test of the first nc (at most 32) queued candidates, and their entries
      auto drain = [&](int nc) {
        const int at = head & (kQueue - 1);
        const float2 nx2 = make_float2(-H.x, -H.x), ny2 = make_float2(-H.y, -H.y), nz2 = make_float2(-H.z, -H.z);
        const float2 kh2 = make_float2(a.kh_f, a.kh_f), kd2 = make_float2(khdi, khdi);
        const float2 nk2 = make_float2(-a.kh_f, -a.kh_f), nd2 = make_float2(-khdi, -khdi);
        unsigned mask = 0;
        float near = __int_as_float(0x7f800000);             // the least |r^2 - R^2| (FP64 handles)
#pragma unroll
        for (int c = 0; c < 32; c += 4) {
          if (c >= nc) break;
          const float4 X = *reinterpret_cast<const float4*>(&qx[warp][at + c]);
          const float4 D = *reinterpret_cast<const float4*>(&qd[warp][at + c]);
          float4 Y{}, Z{};
          if (DIM >= 2) Y = *reinterpret_cast<const float4*>(&qy[warp][at + c]);
          if (DIM >= 3) Z = *reinterpret_cast<const float4*>(&qz[warp][at + c]);
#pragma unroll
          for (int k = 0; k < 2; ++k) {
            const float2 dx = add2(k ? make_float2(X.z, X.w) : make_float2(X.x, X.y), nx2);
            float2 r2 = mul2(dx, dx);
            if (DIM >= 2) {
              const float2 dy = add2(k ? make_float2(Y.z, Y.w) : make_float2(Y.x, Y.y), ny2);
              r2 = fma2(dy, dy, r2);
            }
            if (DIM >= 3) {
              const float2 dz = add2(k ? make_float2(Z.z, Z.w) : make_float2(Z.x, Z.y), nz2);
              r2 = fma2(dz, dz, r2);
            }
            const float2 d = k ? make_float2(D.z, D.w) : make_float2(D.x, D.y);
            const float2 diff = fma2(fma2(nk2, d, nd2), fma2(kh2, d, kd2), r2);   // r^2 - R^2
            if (diff.x < band) mask |= 1u << (c + 2 * k);
            if (diff.y < band) mask |= 2u << (c + 2 * k);
            if constexpr (!MIXED) near = fminf(near, fminf(fabsf(diff.x), fabsf(diff.y)));
          }
        }
        if (nc < 32) mask &= (1u << nc) - 1u;
        if (!act) mask = 0;
        const bool mine = lane < nc;
        const int jc = mine ? qslot[warp][at + lane] : -1;
        const uint32_t word = mine ? qword[warp][at + lane] : 0u;
        // no pair with itself: the home particles in this chunk are consecutive candidates
        const unsigned own = __ballot_sync(0xffffffffu, jc >= h0 && jc < h0 + nh);
        if (own) {
          const int first = __ffs(own) - 1;
          const unsigned k = (unsigned)(i - __shfl_sync(0xffffffffu, jc, first));
          if (k < (unsigned)__popc(own)) mask &= ~(1u << (first + k));
        }
        if constexpr (!MIXED) {
          // too close to call in FP32, which is rare: the lane decides its candidates in FP64
          if (near <= band) mask = decide_exactly<DIM>(A, i, mask, &qslot[warp][at], a.kh);
        }
        for (int h8 = 0; h8 < nh; h8 += 8) {   // (the masks of lanes past nh are empty)
#pragma unroll
          for (int k = 0; k < 8; ++k) {
            const int hp = h8 + k;
            const unsigned m = __shfl_sync(0xffffffffu, mask, hp);
            const int v0 = __shfl_sync(0xffffffffu, vc, hp);
            const int row = a.e_of_c ? __shfl_sync(0xffffffffu, row_i, hp) : h0 + hp;
            const int pos = v0 + __popc(m & lt);
            if (((m >> lane) & 1u) && pos < a.vcap) a.vlist[(int64_t)row * a.vcap + pos] = word;
          }
        }
        vc += __popc(mask);
        head += nc;
        __syncwarp();   // the places read are written again by the next chunks
      };

      for (int oz = (DIM >= 3 ? -1 : 0); oz <= (DIM >= 3 ? 1 : 0); ++oz) {
        for (int oy = (DIM >= 2 ? -1 : 0); oy <= (DIM >= 2 ? 1 : 0); ++oy) {
          const int rc = 3 * (oy + 1) + 9 * (oz + 1);     // index of the row's ox = -1 cell
          const int s_m = nb_start[warp][rc], s_0 = nb_start[warp][rc + 1], s_p = nb_start[warp][rc + 2];
          if (s_0 < 0) continue;                           // row outside the mesh
          // contiguous slot range of the row: from the first existing cell to the end of the last
          const int r0 = s_m >= 0 ? s_m : s_0;
          const int xe = s_p >= 0 ? cx + 2 : cx + 1;       // one past the last existing cell in x
          const int64_t rowc = g.cell_off + (int64_t)nx * ((cy + oy) + (int64_t)ny * (cz + oz));
          const int r1 = a.cell_start[rowc + xe];
          const int b1 = a.cell_start[rowc + cx + 1];      // end of the ox = 0 cell
          for (int base = r0; base < r1; base += 32) {
            const int j = base + lane;
            const bool jv = j < r1;
            const V4 R = A[jv ? j : r0];
            float4 S{};
            uint32_t ent = 0;
            if (jv) {
              const int ox = j < s_0 ? -1 : (j < b1 ? 0 : 1);
              S = frame(R, ox, oy, oz);
              const int off = j - (ox < 0 ? s_m : (ox == 0 ? s_0 : b1));
              if (off > 2047) set_status(a.status, SPH_ERR_CAPACITY);   // cell over 2047 particles
              ent = ((uint32_t)(a.e_of_c ? a.e_of_c[j] : j) << 5) | (uint32_t)(rc + ox + 1);
            }
            // keep only the candidates within reach of the home group's box
            // (a superset: every rounding below is monotone in the distance)
            const float gx = fmaxf(0.f, fmaxf(S.x - bxh, bxl - S.x));
            const float gy = DIM >= 2 ? fmaxf(0.f, fmaxf(S.y - byh, byl - S.y)) : 0.f;
            const float gz = DIM >= 3 ? fmaxf(0.f, fmaxf(S.z - bzh, bzl - S.z)) : 0.f;
            const float Rm = fmaf(a.kh_f, S.w, bkh);
            const bool keep = jv && fmaf(-Rm, Rm, F::r2_of(gx, gy, gz)) < band;
            const unsigned km = __ballot_sync(0xffffffffu, keep);
            if (keep) {
              const int c = (tail + __popc(km & lt)) & (kQueue - 1);
              qx[warp][c] = S.x;
              if (DIM >= 2) qy[warp][c] = S.y;
              if (DIM >= 3) qz[warp][c] = S.z;
              qd[warp][c] = S.w;
              qword[warp][c] = ent;
              qslot[warp][c] = j;
            }
            tail += __popc(km);
            __syncwarp();
            if (tail - head >= 32) drain(32);
          }
        }
      }
      if (tail > head) drain(tail - head);
      if (act) {
        if (vc > a.vcap) set_status(a.status, SPH_ERR_CAPACITY);
        a.vcnt[row_i] = vc < a.vcap ? vc : a.vcap;
        const int64_t p = a.perm[i];
        a.vref[p] = a.x[p];
        if (DIM >= 2) a.vref[a.n + p] = a.y[p];
        if (DIM >= 3) a.vref[2 * a.n + p] = a.z[p];
        a.vref[3 * a.n + p] = a.d[p];
      }
      __syncwarp();
    }
    __syncwarp();     // the neighbour-start buffer is rewritten by the next cell
  }
}

template <bool MIXED, int DIM>
cudaError_t launch_one(const PairArgs& args, int blocks_per_sm, cudaStream_t st) {
  const auto [sms, per_sm] = resident_blocks<k_list_build<MIXED, DIM>>(kPairBlock);
  const int b = (blocks_per_sm > 0 && blocks_per_sm < per_sm) ? blocks_per_sm : per_sm;
  return launch_chained(k_list_build<MIXED, DIM>, dim3(sms * b), dim3(kPairBlock), st, args);
}

template <bool MIXED>
cudaError_t launch_dim(sph_handle* h, const PairArgs& args, cudaStream_t st) {
  const int b = h->p.pair_blocks_per_sm;
  switch (h->dp.dim) {
    case 1: return launch_one<MIXED, 1>(args, b, st);
    case 2: return launch_one<MIXED, 2>(args, b, st);
    default: return launch_one<MIXED, 3>(args, b, st);
  }
}

}  // namespace

// Verlet list build over the radius (1 + beta) kappa h_ij; returns at once on
// the device unless vflag[0] is set.
cudaError_t launch_list_build(sph_handle* h, const sph_state& s, cudaStream_t st) {
  PairArgs a = make_args(h, s);
  a.K = 0;
  a.collect_adj = 0;
  a.pair_i = a.pair_j = nullptr;
  const double khl = h->dp.kh * (1.0 + h->dp.cell_beta);
  a.kh = khl;
  a.kh_f = (float)khl;
  if (h->unit_sched != SPH_SCHED_GLOBAL) a.e_of_c = h->e_of_c;   // rows and entries in the unit-major evaluation order
  a.Ac = h->packAc;                                               // A alone, in cell order
  // work counter zeroed by the step's k_pack
  a.work_counter = &h->counters[7];
  a.vinst = h->n_inst > 1 ? h->vinst : nullptr;   // only the instances whose lists are rebuilt
  cudaError_t e = h->dp.precision == SPH_PREC_MIXED ? launch_dim<true>(h, a, st) : launch_dim<false>(h, a, st);
  h->launches += 1;
  return e;
}

}  // namespace csph
