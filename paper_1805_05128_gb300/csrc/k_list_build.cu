// k_list_build.cu -- the Verlet list build: every pair within
// (1 + beta) kappa h_ij of the current positions (Sec. 4.2 with the buffered
// horizon of eq. (Dcell)), written as one list per slot for k_pair_lists.
//
// One warp per home cell, lane l owning home particle start_c + chunk + l (a
// cell of edge (1 + beta) D^c holds 27 particles of a lattice, so a warp per
// cell fills its lanes here).  For each neighbour row (the 3 x-consecutive
// cells at (oy, oz), contiguous in slot order) each lane loads one candidate;
// those within reach of the home group's bounding box are compacted into
// shared memory in order, and every lane tests its own home particle against
// each (a broadcast read) and appends the accepted ones to its row in
// candidate order.  A row entry is 16 bits: the neighbour-cell code (ox+1) +
// 3 (oy+1) + 9 (oz+1) and the offset inside that cell.  The warp then writes
// each home particle's row with 32 consecutive stores.
//
// The test runs in FP32 in both precisions (mixed handles on the packed
// offsets from the cell origins, FP64 handles on offsets from the cell's first
// particle scaled to a cell edge of ~1) and accepts r^2 - R^2 < 2^-12 D^c^2, a
// superset of the radius: k_pair_lists decides each entry exactly.  Bound by
// shared-memory latency and issue.
#include "pair_common.cuh"

namespace csph {

namespace {

// Row capacity between flushes and resident blocks per SM: rows of 64 or 96
// entries with 7-8 resident blocks made the 1.125M plate's step 0.3-3 % slower
// than 128 entries with 6 blocks.  Row stride: cap + 2 16-bit entries, an odd
// number of words, so lane rows fall in distinct banks.
constexpr int kBuildCap = 128;
constexpr int kBuildBlocks = 6;

template <bool MIXED, int DIM>
__global__ void __launch_bounds__(kPairBlock, kBuildBlocks) k_list_build(PairArgs a) {
  chain_entry();
  using T = typename Ops<MIXED>::T;
  using V4 = typename Ops<MIXED>::V4;
  using F = Pair<true, DIM>;
  __shared__ uint16_t list[kWarps][32][kBuildCap + 2];      // [warp][home particle][entry]
  __shared__ float4 cand[kWarps][32];                        // candidates: x, y, z in the home cell's frame, d
  __shared__ uint16_t cand_ent[kWarps][32];                  // their list entries
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
    const float band = 0x1p-12f * dct * dct;
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
      int cnt = 0, vc = 0;
      // the home group's bounding box and largest kh d, a warp-wide cull of candidates
      float bxl = H.x, bxh = H.x, byl = H.y, byh = H.y, bzl = H.z, bzh = H.z, bkh = khdi;
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) {
        bxl = fminf(bxl, __shfl_xor_sync(0xffffffffu, bxl, o)); bxh = fmaxf(bxh, __shfl_xor_sync(0xffffffffu, bxh, o));
        byl = fminf(byl, __shfl_xor_sync(0xffffffffu, byl, o)); byh = fmaxf(byh, __shfl_xor_sync(0xffffffffu, byh, o));
        bzl = fminf(bzl, __shfl_xor_sync(0xffffffffu, bzl, o)); bzh = fmaxf(bzh, __shfl_xor_sync(0xffffffffu, bzh, o));
        bkh = fmaxf(bkh, __shfl_xor_sync(0xffffffffu, bkh, o));
      }

      // The warp writes each home particle's new entries together, 32
      // consecutive entries of one row per store (the self pair dropped by a
      // ballot, list order kept), instead of one entry of 32 rows per store.
      auto flush_lists = [&]() {
        for (int hp = 0; hp < nh; ++hp) {
          const int n = __shfl_sync(0xffffffffu, cnt, hp);
          int v0 = __shfl_sync(0xffffffffu, vc, hp);
          const int64_t ih = a.e_of_c ? (int64_t)a.e_of_c[h0 + hp] : (int64_t)(h0 + hp);   // the row's slot
          const int64_t ihc = h0 + hp;                                                       // cell order
          for (int k0 = 0; k0 < n; k0 += 32) {
            const int k = k0 + lane;
            uint32_t word = 0;
            bool w = false;
            if (k < n) {
              const unsigned ent = list[warp][hp][k];
              const int64_t j = (int64_t)nb_start[warp][ent >> 11] + (ent & 2047u);
              w = j != ihc;
              const int64_t je = a.e_of_c ? (int64_t)a.e_of_c[j] : j;
              word = ((uint32_t)je << 5) | (ent >> 11);
            }
            const unsigned m = __ballot_sync(0xffffffffu, w);
            const int pos = v0 + __popc(m & lt);
            if (w && pos < a.vcap) a.vlist[ih * a.vcap + pos] = word;
            v0 += __popc(m);
          }
          if (lane == hp) vc = v0;
        }
        cnt = 0;
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
            // a chunk adds at most 32 entries to a list: flush first if one could overflow
            if (__any_sync(0xffffffffu, cnt > kBuildCap - 32)) flush_lists();
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
              ent = ((uint32_t)(rc + ox + 1) << 11) | (uint32_t)(off & 2047);
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
              const int c = __popc(km & lt);
              cand[warp][c] = S;
              cand_ent[warp][c] = (uint16_t)ent;
            }
            const int nc = __popc(km);
            __syncwarp();
#pragma unroll 8
            for (int c = 0; c < nc; ++c) {
              const float4 Sc = cand[warp][c];
              const float r2 = F::r2_of(Sc.x - H.x, DIM >= 2 ? Sc.y - H.y : 0.f, DIM >= 3 ? Sc.z - H.z : 0.f);
              const float R = fmaf(a.kh_f, Sc.w, khdi);
              const float diff = fmaf(-R, R, r2);          // r^2 - R^2
              if (diff < band && act) list[warp][lane][cnt++] = cand_ent[warp][c];
            }
            __syncwarp();   // the candidate buffer is rewritten by the next chunk
          }
        }
      }
      flush_lists();
      if (act) {
        if (vc > a.vcap) set_status(a.status, SPH_ERR_CAPACITY);
        a.vcnt[a.e_of_c ? a.e_of_c[i] : i] = vc < a.vcap ? vc : a.vcap;
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
  static int sms = 0, per_sm = 0;
  if (sms == 0) {
    int dev = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_list_build<MIXED, DIM>, kPairBlock, 0);
    if (per_sm < 1) per_sm = 1;
  }
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
