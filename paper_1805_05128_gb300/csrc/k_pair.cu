// k_pair.cu -- the CSPH pair loop (Sec. 4.1-4.2): neighbour search in the
// 3^dim cells of the block B_i, acoustic pair Riemann solver, and the
// per-particle sums of eqs. (SPH:Conti), (SPH:Pulse), (SPH:Energy).
//
// A warp handles a group of up to 32 consecutive slots (cell order), one lane
// per slot.  The part of a group that lies in one x-row of cells is a segment;
// its candidates are the slots of the 3^(dim-1) neighbouring rows from one
// cell before the segment's first cell to one past its last.  Each lane loads
// one candidate, a ballot compacts those that can reach the segment's bounding
// box into shared memory, every lane then tests its own particle against the
// compacted ones (a broadcast read) and appends those that interact to its
// list; after the scan each lane evaluates the fluxes of its own list.
//
// Why groups of slots and not single cells: a cell holds 17.6 particles of a
// lattice (kappa eta = 2.6 spacings), so a warp per cell evaluated the fluxes
// with 55 % of its lanes; a group fills them.  The box cull drops the
// candidates beyond the corners and edges of the block (40 % of them).
// Measured against a warp per cell without the cull, whole passes: 387k plate,
// mixed, 0.97 -> 0.71 ms per step; 203k plate, FP64, 8.16 -> 3.36 ms; 72.9k
// plane, order 2, 0.240 -> 0.138 ms.
//
// Antisymmetry: the momentum flux F_ij e^R that i and j apply are bitwise
// negatives of each other, and so are the energy fluxes Q_ij of FP64
// handles; mixed handles sum the energy flux from velocity differences
// (FwdAcc in pair_common.cuh).
//
// Modes of the kernel: the rates (optionally with order-2 states), the SPH
// gradients of order 2 and the reverse mode; the Verlet list build is
// k_list_build.cu, the evaluation over the lists k_pair_lists.cu.
//
// The candidate test runs in FP32 in both precisions: mixed handles on the
// packed offsets from each particle's own cell origin, FP64 handles on
// offsets from the segment's first particle, scaled by a power of two so that
// the cell edge is ~1 (any length unit stays in FP32's range).  The FP32 test
// decides r^2 < R^2 whenever r^2 lies outside a band of 2^-12 D^c^2 around
// R^2, which bounds the accumulated FP32 error of both sides (<= ~1e-5 D^c^2,
// segments spanning at most kSpan cells included); inside the band the pair is
// decided by the FP64 test on the global positions, with the same operation
// order as the oracle, so the pair set is the FP64 one.  (FP64 handles tested
// every candidate in FP64 before, 12 instructions of a pipe 64 times narrower
// than FP32's: a third of their pair kernel.)  Mixed per-particle sums are
// Kahan-compensated; each slot adds its pairs in candidate order.
#include "pair_common.cuh"

namespace csph {

namespace {

constexpr int kRowCap = 112;   // list entries per slot between flushes (row stride 2 mod 64 bytes: lane rows in
                               // distinct banks); a flush mid-scan is rare (a lattice has 81, the slot itself included)
constexpr int kSegs = 2;       // segments per scan before a flush
constexpr int kSpan = 16;      // cells a segment may span along x (bounds the FP32 frame)

template <bool MIXED, int DIM, int MODE, int G, bool HLL = false, bool EXTRA = true>
__global__ void __launch_bounds__(kPairBlock, (MODE == kModeVjp || MODE == kModeFwd2) ? (MIXED ? 4 : 3)
                                                 : (MODE == kModeGrad ? (MIXED ? 5 : 3) : (MIXED ? 6 : 4)))
    k_pair(PairArgs a) {
  chain_entry();
  constexpr bool VJP = MODE == kModeVjp;
  constexpr bool GRAD = MODE == kModeGrad;
  constexpr int kRows = DIM == 3 ? 9 : (DIM == 2 ? 3 : 1);
  using P = Pair<MIXED, DIM>;
  using T = typename P::T;
  using V4 = typename P::V4;
  using V2 = typename P::V2;
  using VC = typename P::VC;
  constexpr int kHomes = 32 / G;                              // slots per group
  constexpr int kCap = G == 1 ? kRowCap : 2 * kRowCap;
  constexpr bool kOrdered = MIXED && G > 1;                   // the sums take the pairs in candidate order
  __shared__ uint16_t list[kWarps][kHomes][kCap + 2];        // [warp][slot][entry]: cell code << 11 | offset
  __shared__ float4 cand[kWarps][32];                        // candidates that survived the cull: x, y, z, d (FP32)
  __shared__ int2 cand_ent[kWarps][32];                      // their entry in the segment's frame, their slot
  __shared__ float4 nb_tab[kWarps][kSegs][27];               // per segment and cell code: first slot (bits), shift x, y, z

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const unsigned lt = (1u << lane) - 1u;
  const int home = lane / G, hl = lane % G;                   // the lane's slot in the group, its place in the slot
  const V4* __restrict__ A = reinterpret_cast<const V4*>(a.A);
  const VC* __restrict__ C = reinterpret_cast<const VC*>(a.C);
  // Persistent warps: the first group of each is fixed (spread over the CTAs,
  // so that few groups run on many SMs), the following ones come from a
  // global counter, so the work spreads evenly.
  const int n_1 = (int)a.n - 1;
  unsigned long long q = (unsigned long long)warp * gridDim.x + blockIdx.x;
  for (; (int64_t)(q * (unsigned)a.group) < a.n;) {
    const int h0 = (int)(q * (unsigned)a.group);
    const long long t_start = a.load_timed ? clock64() : 0;   // timed unit loads
    const int i = h0 + home;
    const bool act = home < a.group && i < a.n;
    const int ii = act ? i : h0;
    int b = 0;
    if (a.n_inst > 1) {  // instance of this slot: binary search of the slot offsets
      int lo = 0, hi = a.n_inst;
      while (hi - lo > 1) {
        const int mid = (lo + hi) >> 1;
        if (a.inst_off[mid] <= ii) lo = mid; else hi = mid;
      }
      b = lo;
    }
    int cx, row;                                               // the slot's cell along x, its row of cells
    {
      const GridInfo& g = a.grid[b];
      const int lc = a.slot_cell[ii] - (int)g.cell_off;
      row = lc / g.dims[0];
      cx = lc - row * g.dims[0];
    }
    V4 Ai, Bi;
    load_AB(a.A, a.B, (uint32_t)ii, Ai, Bi);
    int cnt = 0, seg_of = 0, cx_seg = 0;
    unsigned nfull = 0, ncand = 0, nexact = 0;
    const int ui = a.K > 0 ? a.slot_unit[ii] : 0;
    const VC Ci = C[ii];
    // reverse mode: i's adjoint operands and the 11 own-side sums
    const V4* __restrict__ Gp = reinterpret_cast<const V4*>(a.G);
    const V2* __restrict__ Rp = reinterpret_cast<const V2*>(a.GR2);
    V4 Gi{};
    V2 Ri{};
    if constexpr (VJP) { Gi = Gp[ii]; Ri = Rp[ii]; }
    const T Vi2 = T(2) * Bi.w, Qi = T(2) * Ri.y;   // FP64 form only
    Kahan<T> s_bx[3], s_bv[3], s_bP, s_bZ, s_bV, s_bd, s_brho;

    FwdAcc<MIXED, DIM, MODE == kModeFwd2, HLL, EXTRA> fw;
    if constexpr (MODE == kModeFwd2) {
      fw.gPi = reinterpret_cast<const V4*>(a.gP)[ii];
      const V4* GV = reinterpret_cast<const V4*>(a.gV);
      fw.gVi[0] = GV[ii];
      if (DIM >= 2) fw.gVi[1] = GV[a.n + ii];
      if (DIM >= 3) fw.gVi[2] = GV[2 * a.n + ii];
    }

    // SPH gradients (GRAD): grad q_i = sum_j V_j (q_j - q_i) (-W'_ij) e^R for q = P, v_x, v_y, v_z
    T gP[3] = {T(0), T(0), T(0)}, gV[3][3] = {{T(0), T(0), T(0)}, {T(0), T(0), T(0)}, {T(0), T(0), T(0)}};
    struct GradTerms { bool live; T fP, fv[3], e[3]; };
    auto grad_terms = [&](int64_t j, T sx, T sy, T sz) -> GradTerms {
      GradTerms q{};
      if (j == i) return q;
      V4 Aj, Bj;
      load_AB(a.A, a.B, (uint32_t)j, Aj, Bj);
      const VC Cj = C[j];
      T dx, dy, dz;
      if (MIXED) {
        dx = (Aj.x - Ai.x) + sx;
        dy = DIM >= 2 ? (Aj.y - Ai.y) + sy : T(0);
        dz = DIM >= 3 ? (Aj.z - Ai.z) + sz : T(0);
      } else {
        dx = __dsub_rn(Aj.x, Ai.x);
        dy = DIM >= 2 ? __dsub_rn(Aj.y, Ai.y) : 0.0;
        dz = DIM >= 3 ? __dsub_rn(Aj.z, Ai.z) : 0.0;
      }
      const T r2 = MIXED ? P::r2_of(dx, dy, dz) : fw.r2_fused(dx, dy, dz);
      if (!positive(r2)) return q;
      T ir, r;
      rsqrt_sqrt(r2, ir, r);
      const T e[3] = {dx * ir, dy * ir, dz * ir};
      T w;
      if constexpr (MIXED) w = -dw_fast<T, DIM>(a.kernel, (T)a.kappa_f, r, (T)a.eta_half_f * (Ai.w + Aj.w), (T)a.wscale_f);
      else w = -dw64<DIM, -1>(a.kernel, a.kappa, a.eta_half, r, Ai.w + Aj.w);
      const T f = Bj.w * w;
      const T dP = Cj.x - Ci.x;
      T dv[3];
      if constexpr (MIXED) {   // relative velocities plus the exact reference difference
        dv[0] = dvel(Bi.x, Bj.x, Ci, Cj, 0);
        dv[1] = dvel(Bi.y, Bj.y, Ci, Cj, 1);
        dv[2] = dvel(Bi.z, Bj.z, Ci, Cj, 2);
      } else {
        dv[0] = Bj.x - Bi.x;
        dv[1] = Bj.y - Bi.y;
        dv[2] = Bj.z - Bi.z;
      }
      q.live = true;
      q.fP = f * dP;
#pragma unroll
      for (int b = 0; b < 3; ++b) { q.fv[b] = f * dv[b]; q.e[b] = e[b]; }
      return q;
    };
    auto add_grad = [&](const GradTerms& q) {
#pragma unroll
      for (int b = 0; b < DIM; ++b) {
        gP[b] = fma_(q.fP, q.e[b], gP[b]);
#pragma unroll
        for (int c = 0; c < DIM; ++c) gV[c][b] = fma_(q.fv[c], q.e[b], gV[c][b]);
      }
    };

    // Reverse mode of the pair's contributions (VJP = true): the derivative of
    // the pair's terms in a, drho, dE of both i and j, contracted with their
    // adjoints, with respect to i's own variables: position (through r, e and
    // W'), v (through v^R), P and Z = rho c (through the acoustic solver),
    // V = m/rho, d (through h_ij) and the rho factor of the continuity term.
    auto pair_vjp = [&](int64_t j, T sx, T sy, T sz) {
      if (j == i) return;
      V4 Aj, Bj;
      load_AB(a.A, a.B, (uint32_t)j, Aj, Bj);
      const VC Cj = C[j];
      const V4 Gj = Gp[j];
      const V2 Rj = Rp[j];
      T dx, dy, dz;
      if (MIXED) {
        dx = (Aj.x - Ai.x) + sx;
        dy = DIM >= 2 ? (Aj.y - Ai.y) + sy : T(0);
        dz = DIM >= 3 ? (Aj.z - Ai.z) + sz : T(0);
      } else {
        dx = __dsub_rn(Aj.x, Ai.x);
        dy = DIM >= 2 ? __dsub_rn(Aj.y, Ai.y) : 0.0;
        dz = DIM >= 3 ? __dsub_rn(Aj.z, Ai.z) : 0.0;
      }
      const T r2 = MIXED ? P::r2_of(dx, dy, dz) : fw.r2_fused(dx, dy, dz);
      if (!positive(r2)) return;
      T ir, r;
      rsqrt_sqrt(r2, ir, r);
      const T e[3] = {dx * ir, dy * ir, dz * ir};
      if constexpr (MIXED) {
        T vi[3] = {Bi.x, Bi.y, Bi.z}, vj[3] = {Bj.x, Bj.y, Bj.z};
#pragma unroll
        for (int q = 0; q < 3; ++q) {   // lab-frame velocities: relative ones plus the references
          vi[q] += ref_v(Ci, q);
          vj[q] += ref_v(Cj, q);
        }
        T vRi = T(0), vRj = T(0);
#pragma unroll
        for (int q = 0; q < DIM; ++q) { vRi += vi[q] * e[q]; vRj += vj[q] * e[q]; }
        const T Zi = Ci.y, Zj = Cj.y, zs = Zi + Zj, Pi = Ci.x, Pj = Cj.x;
        T Ps, vs, izs = T(0);
        if (positive(zs)) {
          izs = rcp_(zs);
          Ps = (Zj * Pi + Zi * Pj + Zi * Zj * (vRi - vRj)) * izs;
          vs = (Zi * vRi + Zj * vRj + Pi - Pj) * izs;
        } else {
          Ps = T(0.5) * (Pi + Pj);
          vs = T(0.5) * (vRi + vRj);
        }
        const T eh = MIXED ? (T)a.eta_half_f : (T)a.eta_half;
        const T hij = eh * (Ai.w + Aj.w);
        T W, Wr, Wh;
        cubic_dw3<T, DIM>(r, hij, W, Wr, Wh);
        const T Vi = Bi.w * (T)a.vinv, Vj = Bj.w * (T)a.vinv;     // the packed volumes are scaled
        const T GRi = Ri.x, rhoi = Ri.y, GRj = Rj.x, rhoj = Rj.y;
        const T F = T(2) * Vi * Vj * Ps * W;
        const T dA[3] = {Gi.x - Gj.x, Gi.y - Gj.y, Gi.z - Gj.z};
        const T dB = Gi.w - Gj.w;
        T gF = dB * vs, ge[3] = {T(0), T(0), T(0)};
#pragma unroll
        for (int q = 0; q < DIM; ++q) { gF += dA[q] * e[q]; ge[q] = F * dA[q]; }
        const T ti = T(2) * W * rhoi * Vj * GRi;          // continuity terms of i and of j
        const T tj = T(2) * W * rhoj * Vi * GRj;
        const T gvs = F * dB + ti - tj;
        T gvRi = -ti, gvRj = tj;
        const T gW = gF * T(2) * Vi * Vj * Ps - GRi * T(2) * rhoi * Vj * (vRi - vs) - GRj * T(2) * rhoj * Vi * (vs - vRj);
        const T gPs = gF * T(2) * Vi * Vj * W;
        s_bV.add(gF * T(2) * Vj * Ps * W - GRj * T(2) * rhoj * (vs - vRj) * W);
        s_brho.add(-(GRi * T(2) * Vj * (vRi - vs) * W));
        T gPi, gZi = T(0);
        if (positive(zs)) {
          gPi = (gPs * Zj + gvs) * izs;
          gvRi += (gPs * Zi * Zj + gvs * Zi) * izs;
          gvRj += (gvs * Zj - gPs * Zi * Zj) * izs;
          gZi = (gPs * ((Pj + Zj * (vRi - vRj)) - Ps) + gvs * (vRi - vs)) * izs;
        } else {
          gPi = T(0.5) * gPs;
          gvRi += T(0.5) * gvs;
          gvRj += T(0.5) * gvs;
        }
        s_bP.add(gPi);
        s_bZ.add(gZi);
        T ede = T(0);
#pragma unroll
        for (int q = 0; q < DIM; ++q) {
          s_bv[q].add(gvRi * e[q]);
          ge[q] += gvRi * vi[q] + gvRj * vj[q];
          ede += ge[q] * e[q];
        }
        const T grr = gW * Wr;
#pragma unroll
        for (int q = 0; q < DIM; ++q) s_bx[q].add(-((ge[q] - ede * e[q]) * ir + grr * e[q]));
        s_bd.add(gW * Wh * eh);
      } else {
        // The same derivatives with fewer instructions of the FP64 pipe (120
        // per pair), which bounds this mode: the factors that belong to i alone
        // (2 V_i, 2 rho_i GR_i, and the constant factors of the sums) are taken
        // out of the loop, GR2.y holds rho GR, and the derivatives of the
        // acoustic state use P* - P_j = Z_j (v* - v_j^R), by which
        // dL/dZ_i = (v_i^R - v*) dL/dP_i.  32k particles: 1.25 -> 0.70 ms a launch.
        const T vi[3] = {Bi.x, Bi.y, Bi.z}, vj[3] = {Bj.x, Bj.y, Bj.z};
        T vRi = vi[0] * e[0], vRj = vj[0] * e[0];
#pragma unroll
        for (int q = 1; q < DIM; ++q) { vRi = fma_(vi[q], e[q], vRi); vRj = fma_(vj[q], e[q], vRj); }
        const T Zi = Ci.y, Zj = Cj.y, zs = Zi + Zj, Pi = Ci.x, Pj = Cj.x;
        const bool zpos = positive(zs);
        T Ps, vs, izs = T(0);
        if (zpos) {
          izs = rcp_(zs);
          Ps = fma_(Zi * Zj, vRi - vRj, fma_(Zi, Pj, Zj * Pi)) * izs;
          vs = (fma_(Zi, vRi, Zj * vRj) + (Pi - Pj)) * izs;
        } else {
          Ps = T(0.5) * (Pi + Pj);
          vs = T(0.5) * (vRi + vRj);
        }
        T W, Wr, Wh;
        cubic_dw3<T, DIM>(r, (T)a.eta_half * (Ai.w + Aj.w), W, Wr, Wh);
        const T Vj = Bj.w, Hj = Rj.y;
        const T VV = Vi2 * Vj, PV = VV * Ps, F = PV * W;
        const T dA[3] = {Gi.x - Gj.x, Gi.y - Gj.y, Gi.z - Gj.z};
        const T dB = Gi.w - Gj.w;
        T gF = dB * vs;
#pragma unroll
        for (int q = 0; q < DIM; ++q) gF = fma_(dA[q], e[q], gF);
        const T ai = vRi - vs, bj = vs - vRj;
        const T ki = Qi * Vj, kj = Hj * Vi2;
        const T ti = ki * W, tj = kj * W;                  // continuity terms of i and of j
        const T gvs = fma_(F, dB, ti - tj);
        const T gW = fma_(-kj, bj, fma_(-ki, ai, gF * PV));
        const T gPs = gF * (VV * W);
        s_bV.add_product(W, fma_(gF * Ps, Vj, -(Hj * bj)));   // x 2
        s_brho.add_product(Vj * ai, W);                        // x -2 GR_i
        T gPi, gvRi, gvRj;
        if (zpos) {
          gPi = fma_(gPs, Zj, gvs) * izs;
          gvRi = fma_(Zi, gPi, -ti);
          gvRj = fma_(Zj, fma_(-gPs, Zi, gvs) * izs, tj);
          s_bZ.add_product(ai, gPi);
        } else {
          gPi = T(0.5) * gPs;
          gvRi = fma_(T(0.5), gvs, -ti);
          gvRj = fma_(T(0.5), gvs, tj);
        }
        s_bP.add(gPi);
        T ge[3], ede = T(0);
#pragma unroll
        for (int q = 0; q < DIM; ++q) {
          s_bv[q].add_product(gvRi, e[q]);
          ge[q] = fma_(gvRi, vi[q], fma_(gvRj, vj[q], F * dA[q]));
          ede = fma_(ge[q], e[q], ede);
        }
        const T along = fma_(-ede, ir, gW * Wr);
#pragma unroll
        for (int q = 0; q < DIM; ++q) {
          s_bx[q].add_product(-ge[q], ir);
          s_bx[q].add_product(-e[q], along);
        }
        s_bd.add_product(gW, Wh);                              // x eta / 2
      }
    };

    auto flush = [&]() {
      [[maybe_unused]] const unsigned flushed = nfull;         // entries of the slot that earlier flushes took
      nfull += (unsigned)cnt;
      if constexpr (kOrdered) {
        // The slot's lanes evaluate consecutive entries; then each of them adds
        // the terms in candidate order, so the sums are those of one lane going
        // through the list.
        const unsigned group = ((1u << G) - 1u) << (home * G);
        for (int k0 = 0; k0 < cnt; k0 += G) {
          const int k = k0 + hl;
          typename FwdAcc<MIXED, DIM, MODE == kModeFwd2, HLL, EXTRA>::Terms q{};
          GradTerms qg{};
          if (k < cnt) {
            const unsigned ent = list[warp][home][k];
            const float4 t = nb_tab[warp][seg_of][min(ent >> 11, 26u)];
            const int64_t j = min(__float_as_int(t.x) + (int)(ent & 2047u), n_1);
            if constexpr (GRAD) qg = grad_terms(j, (T)t.y, (T)t.z, (T)t.w);
            else q = fw.terms(a, i, Ai, Bi, Ci, ui, j, (T)t.y, (T)t.z, (T)t.w);
          }
          const unsigned live = __ballot_sync(group, GRAD ? qg.live : q.live) >> (home * G);
#pragma unroll
          for (int g = 0; g < G; ++g) {
            if constexpr (GRAD) {
              GradTerms r;
              r.fP = __shfl_sync(group, qg.fP, g, G);
#pragma unroll
              for (int c = 0; c < DIM; ++c) {
                r.fv[c] = __shfl_sync(group, qg.fv[c], g, G);
                r.e[c] = __shfl_sync(group, qg.e[c], g, G);
              }
              if ((live >> g) & 1u) add_grad(r);
            } else {
              const auto r = fw.from_lane(q, group, g, G);
              if ((live >> g) & 1u) fw.add(r);
            }
          }
        }
      } else {
        // Lane hl takes the slot's entries hl, hl + G, ... counted over its flushes:
        // when one falls depends on the other slots of the group, the sums do not.
        for (int k = (int)((unsigned)(hl - (int)flushed) % G); k < cnt; k += G) {
          const unsigned ent = list[warp][home][k];
          // (the two minima change nothing on a finite state; on one with infinite
          // sizes, which is latched, they keep the accesses in bounds)
          const float4 t = nb_tab[warp][seg_of][min(ent >> 11, 26u)];
          const int64_t j = min(__float_as_int(t.x) + (int)(ent & 2047u), n_1);
          if constexpr (VJP) {
            pair_vjp(j, (T)t.y, (T)t.z, (T)t.w);
          } else if constexpr (GRAD) {
            const GradTerms q = grad_terms(j, (T)t.y, (T)t.z, (T)t.w);
            if (q.live) add_grad(q);
          } else {
            fw.pair(a, i, Ai, Bi, Ci, ui, j, (T)t.y, (T)t.z, (T)t.w);
          }
        }
      }
      cnt = 0;
    };

    unsigned todo = __ballot_sync(0xffffffffu, act);
    int seg = 0;
    while (todo) {
      if (seg == kSegs) {                                      // the segment tables are full
        flush();
        __syncwarp();
        seg = 0;
      }
      // the next segment: the lanes of one instance and row of cells, within kSpan cells of the first
      const int lead = __ffs(todo) - 1;
      const int b0 = __shfl_sync(0xffffffffu, b, lead), row0 = __shfl_sync(0xffffffffu, row, lead);
      const int cx0 = __shfl_sync(0xffffffffu, cx, lead);
      const bool same = ((todo >> lane) & 1u) && b == b0 && row == row0;
      unsigned members = __ballot_sync(0xffffffffu, same && cx - cx0 < kSpan);
      int cx1 = __shfl_sync(0xffffffffu, cx, 31 - __clz(members));
      const GridInfo& g = a.grid[b0];
      const int nx = g.dims[0], ny = g.dims[1], nz = g.dims[2];
      const int cy0 = row0 % ny, cz0 = row0 / ny;
      // lane r < kRows: first cell of neighbour row r (-1 outside the mesh) and its slot range
      int64_t rbase = -1;
      int rs0 = 0, rs1 = 0;
      if (lane < kRows) {
        const int yy = cy0 + (DIM >= 2 ? lane % 3 - 1 : 0), zz = cz0 + (DIM >= 3 ? lane / 3 - 1 : 0);
        if (yy >= 0 && yy < ny && zz >= 0 && zz < nz) {
          rbase = g.cell_off + (int64_t)nx * (yy + (int64_t)ny * zz);
          rs0 = a.cell_start[rbase + (cx0 > 0 ? cx0 - 1 : 0)];
          rs1 = a.cell_start[rbase + (cx1 + 1 < nx ? cx1 + 2 : nx)];
        }
      }
      // Entries hold an 11-bit offset: from the row's first slot, or, where a
      // crowded row exceeds that, from the cell's (a segment of one cell).
      const bool wide = __any_sync(0xffffffffu, rs1 - rs0 > 2048);
      if (wide && cx1 > cx0) {
        members = __ballot_sync(0xffffffffu, same && cx == cx0);
        cx1 = cx0;
        if (rbase >= 0) rs1 = a.cell_start[rbase + (cx1 + 1 < nx ? cx1 + 2 : nx)];
      }
      const bool mine = (members >> lane) & 1u;
      if (mine) { seg_of = seg; cx_seg = cx - cx0; }
      todo &= ~members;
      const T dcs = MIXED ? (T)g.dc_f : T(0);
      {
        // first slot of the row (or cell) and the exact shift from a home cell's origin, per cell code
        const int ox = lane % 3 - 1, oy = (lane / 3) % 3 - 1, oz = lane / 9 - 1;
        const int r = (DIM >= 2 ? oy + 1 : 0) + (DIM >= 3 ? 3 * (oz + 1) : 0);
        const int src = r < kRows ? r : 0;
        const int st = __shfl_sync(0xffffffffu, rs0, src);
        const int64_t rb = __shfl_sync(0xffffffffu, rbase, src);
        if (lane < 27) {
          int first = st;
          if (wide && rb >= 0 && cx0 + ox >= 0 && cx0 + ox < nx) first = a.cell_start[rb + cx0 + ox];
          nb_tab[warp][seg][lane] = make_float4(__int_as_float(first), MIXED ? (float)ox * (float)dcs : 0.f,
                                                MIXED ? (float)oy * (float)dcs : 0.f, MIXED ? (float)oz * (float)dcs : 0.f);
        }
      }
      // FP32 frame of the test: the origin of cell cx0 (mixed), the segment's first particle (FP64)
      int ex = 0;
      double fx = 0.0, fy = 0.0, fz = 0.0;
      float dct = MIXED ? (float)dcs : 0.f;
      if constexpr (!MIXED) {
        ex = exponent_of(g.dc);
        dct = f32_scaled(g.dc, ex);
        fx = __shfl_sync(0xffffffffu, Ai.x, lead);
        if (DIM >= 2) fy = __shfl_sync(0xffffffffu, Ai.y, lead);
        if (DIM >= 3) fz = __shfl_sync(0xffffffffu, Ai.z, lead);
      }
      const float band = 0x1p-12f * dct * dct;
      auto frame = [&](const V4& R, int relx, int oy, int oz) {
        float4 S;
        if constexpr (MIXED) {
          S.x = R.x + (float)relx * dct;
          S.y = DIM >= 2 ? R.y + (float)oy * dct : 0.f;
          S.z = DIM >= 3 ? R.z + (float)oz * dct : 0.f;
          S.w = R.w;
        } else {
          S.x = f32_scaled(R.x - fx, ex);
          S.y = DIM >= 2 ? f32_scaled(R.y - fy, ex) : 0.f;
          S.z = DIM >= 3 ? f32_scaled(R.z - fz, ex) : 0.f;
          S.w = f32_scaled(R.w, ex);
        }
        return S;
      };
      float4 H = frame(Ai, cx_seg, 0, 0);
      H.w *= a.kh_f;
      // the members' bounding box and largest kh d
      const float inf = __int_as_float(0x7f800000);
      float bxl = mine ? H.x : inf, bxh = mine ? H.x : -inf, byl = mine ? H.y : inf, byh = mine ? H.y : -inf;
      float bzl = mine ? H.z : inf, bzh = mine ? H.z : -inf, bkh = mine ? H.w : 0.f;
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) {
        bxl = fminf(bxl, __shfl_xor_sync(0xffffffffu, bxl, o)); bxh = fmaxf(bxh, __shfl_xor_sync(0xffffffffu, bxh, o));
        if (DIM >= 2) { byl = fminf(byl, __shfl_xor_sync(0xffffffffu, byl, o)); byh = fmaxf(byh, __shfl_xor_sync(0xffffffffu, byh, o)); }
        if (DIM >= 3) { bzl = fminf(bzl, __shfl_xor_sync(0xffffffffu, bzl, o)); bzh = fmaxf(bzh, __shfl_xor_sync(0xffffffffu, bzh, o)); }
        bkh = fmaxf(bkh, __shfl_xor_sync(0xffffffffu, bkh, o));
      }
      if (!mine) H.x = __int_as_float(0x7fc00000);             // NaN: a lane outside the segment accepts nothing
      if (mine) {
        // candidates of the slot's own 3^dim block (sph_pair_counts), and the capacity of its cell
        const int64_t home = a.grid[b0].cell_off + (int64_t)nx * row0 + cx;
        if (a.cell_start[home + 1] - a.cell_start[home] > 2048) set_status(a.status, SPH_ERR_CAPACITY);
      }
      __syncwarp();
      for (int r = 0; r < kRows; ++r) {
        const int64_t rb = __shfl_sync(0xffffffffu, rbase, r);
        if (rb < 0) continue;                                  // row outside the mesh
        const int r0 = __shfl_sync(0xffffffffu, rs0, r), r1 = __shfl_sync(0xffffffffu, rs1, r);
        const int oy = DIM >= 2 ? r % 3 - 1 : 0, oz = DIM >= 3 ? r / 3 - 1 : 0;
        const int rc = 3 * (oy + 1) + 9 * (oz + 1);            // code of the row's ox = -1 cell
        if (mine && hl == 0) ncand += (unsigned)(a.cell_start[rb + (cx + 1 < nx ? cx + 2 : nx)] - a.cell_start[rb + (cx > 0 ? cx - 1 : 0)]);
        for (int base = r0; base < r1; base += 32) {
          const int j = base + lane;
          const bool jv = j < r1;
          const int jl = jv ? j : r0;
          const int relx = a.slot_cell[jl] - (int)rb - cx0;
          const float4 S = frame(load_A(A, jl), relx, oy, oz);
          // keep the candidates within reach of the members' box (a superset:
          // every rounding below is monotone in the distance)
          const float gx = fmaxf(0.f, fmaxf(S.x - bxh, bxl - S.x));
          const float gy = DIM >= 2 ? fmaxf(0.f, fmaxf(S.y - byh, byl - S.y)) : 0.f;
          const float gz = DIM >= 3 ? fmaxf(0.f, fmaxf(S.z - bzh, bzl - S.z)) : 0.f;
          const float Rm = fmaf(a.kh_f, S.w, bkh);
          const bool keep = jv && fmaf(-Rm, Rm, Pair<true, DIM>::r2_of(gx, gy, gz)) <= band;
          const unsigned km = __ballot_sync(0xffffffffu, keep);
          const int nc = __popc(km);
          if (keep) {
            const int c = __popc(km & lt);
            cand[warp][c] = S;
            const int off = j - (wide ? __float_as_int(nb_tab[warp][seg][rc + 1 + relx].x) : r0);
            cand_ent[warp][c] = make_int2(((rc + 1 + relx) << 11) | (off & 2047), j);
          }
          // a chunk adds at most nc entries to a list: flush first if one could overflow
          if (__any_sync(0xffffffffu, cnt > kCap - nc)) flush();
          __syncwarp();
          const int mybase = cx_seg << 11;
#pragma unroll 4
          for (int c0 = 0; c0 < nc; c0 += G) {
            const int c = c0 + hl;                            // G > 1: the slot's lanes test consecutive candidates
            const float4 Sc = cand[warp][c];
            const float r2 = Pair<true, DIM>::r2_of(Sc.x - H.x, DIM >= 2 ? Sc.y - H.y : 0.f, DIM >= 3 ? Sc.z - H.z : 0.f);
            const float R = fmaf(a.kh_f, Sc.w, H.w);
            const float diff = fmaf(-R, R, r2);              // r^2 - R^2
            const bool cv = G == 1 || c < nc;                // (past nc: an old candidate, not used)
            bool acc = cv && diff < 0.f;
            if (cv && fabsf(diff) <= band) {                  // too close to call in FP32: FP64 decides
              const int jc = cand_ent[warp][c].y;
              ++nexact;
              acc = jc == i || exact_accept(a, DIM, a.perm[i], a.perm[jc]);
            }
            if constexpr (G == 1) {
              if (acc) list[warp][home][cnt++] = (uint16_t)(cand_ent[warp][c].x - mybase);
            } else {
              const unsigned took = (__ballot_sync(0xffffffffu, acc) >> (home * G)) & ((1u << G) - 1u);
              if (acc) list[warp][home][cnt + __popc(took & ((1u << hl) - 1u))] = (uint16_t)(cand_ent[warp][c].x - mybase);
              cnt += __popc(took);
            }
          }
          __syncwarp();   // the candidate buffer is rewritten by the next chunk
        }
      }
      ++seg;
    }
    __syncwarp();
    flush();
    // unordered sums: the slot's lanes hold a part each
    [[maybe_unused]] auto lanes_sum = [](T& v) {
#pragma unroll
      for (int o = G / 2; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    };
    const bool owner = act && hl == 0;

    if constexpr (GRAD) {
      if constexpr (G > 1 && !kOrdered) {
#pragma unroll
        for (int b1 = 0; b1 < 3; ++b1) {
          lanes_sum(gP[b1]);
#pragma unroll
          for (int c = 0; c < 3; ++c) lanes_sum(gV[c][b1]);
        }
      }
      if (owner) {
        V4* GP = reinterpret_cast<V4*>(a.gP);
        V4* GV = reinterpret_cast<V4*>(a.gV);
        const T rs = (T)a.rscale;                      // undo the volume and W' scales (powers of two)
        V4 w{};
        w.x = gP[0] * rs; w.y = gP[1] * rs; w.z = gP[2] * rs;
        GP[i] = w;
#pragma unroll
        for (int c = 0; c < DIM; ++c) {
          V4 gr{};
          gr.x = gV[c][0] * rs; gr.y = gV[c][1] * rs; gr.z = gV[c][2] * rs;
          GV[(int64_t)c * a.n + i] = gr;
        }
      }
    } else if constexpr (VJP) {
      if constexpr (G > 1) {
#pragma unroll
        for (int k = 0; k < 3; ++k) { lanes_sum(s_bx[k].s); lanes_sum(s_bv[k].s); }
        lanes_sum(s_bP.s); lanes_sum(s_bZ.s); lanes_sum(s_bV.s); lanes_sum(s_bd.s); lanes_sum(s_brho.s);
      }
      if (owner) {
        double* o = a.vjp_out + 11 * (int64_t)a.perm[i];
#pragma unroll
        for (int k = 0; k < 3; ++k) { o[k] = (double)s_bx[k].s; o[3 + k] = (double)s_bv[k].s; }
        o[6] = (double)s_bP.s;
        o[7] = (double)s_bZ.s;
        o[8] = MIXED ? (double)s_bV.s : 2.0 * (double)s_bV.s;
        o[9] = MIXED ? (double)s_bd.s : a.eta_half * (double)s_bd.s;
        o[10] = MIXED ? (double)s_brho.s : -2.0 * (double)Ri.x * (double)s_brho.s;
      }
    } else {
      fw.fold();
      if constexpr (G > 1) {
        if constexpr (!kOrdered) {
          lanes_sum(fw.s_rho.s); lanes_sum(fw.s_fx.s); lanes_sum(fw.s_fy.s); lanes_sum(fw.s_fz.s); lanes_sum(fw.s_q.s);
        }
        if constexpr (EXTRA) {
#pragma unroll
          for (int o = G / 2; o > 0; o >>= 1) {
            const T other = __shfl_xor_sync(0xffffffffu, fw.dmax, o);
            fw.dmax = other > fw.dmax ? other : fw.dmax;
          }
        }
      }
      if (owner) {
        nfull -= 1;   // the self pair
        fw.write(a, i, nfull);
      }
      warp_counters(a, owner, nfull, ncand, MIXED ? nexact : 0u, ui, lane,
                    a.load_timed ? (unsigned)(clock64() - t_start) : 0u);
    }
    __syncwarp();     // the segment tables and lists are rewritten by the next group
    if (lane == 0) q = atomicAdd(a.work_counter, 1ull) + (unsigned long long)gridDim.x * kWarps;
    q = __shfl_sync(0xffffffffu, q, 0);
  }
}

// Persistent grid: SMs x resident CTAs per SM, capped by the handle's
// pair_blocks_per_sm (0 = as many as fit) and by the number of groups.
template <bool MIXED, int DIM, int MODE, int G, bool HLL, bool EXTRA>
cudaError_t launch_lanes(const PairArgs& args, int blocks_per_sm, cudaStream_t st) {
  const auto [sms, per_sm] = resident_blocks<k_pair<MIXED, DIM, MODE, G, HLL, EXTRA>>(kPairBlock);
  PairArgs a = args;
  a.group = 32 / G;
  // a group of fewer slots while not every SM has four warps at work
  while (a.group > (G == 1 ? 8 : 2) && a.n < (int64_t)4 * sms * a.group) a.group >>= 1;
  const int64_t groups = (a.n + a.group - 1) / a.group;
  const int b = (blocks_per_sm > 0 && blocks_per_sm < per_sm) ? blocks_per_sm : per_sm;
  // few groups: one CTA per SM until each holds a group per warp (a CTA's warps
  // sit on the SM's four schedulers in turn), then as many CTAs as that needs
  const int64_t want = groups < sms ? groups : ((groups + kWarps - 1) / kWarps > sms ? (groups + kWarps - 1) / kWarps : sms);
  const int grid = want < (int64_t)sms * b ? (int)want : sms * b;
  // A plain launch, not chained to the kernel before it: CTAs that become
  // resident while that one still runs are packed onto the SMs with room left
  // instead of being spread over all of them (6k particles in a plane, FP64, a
  // step: 0.30 ms spread, 0.38 ms packed).
  k_pair<MIXED, DIM, MODE, G, HLL, EXTRA><<<grid, kPairBlock, 0, st>>>(a);
  return cudaGetLastError();
}

// Lanes per slot.  One lane per slot does the least work per pair, but a group
// of 32 slots is then one chain of ~600 candidate tests and ~80 fluxes: 147 us
// for 32k particles, whose groups do not fill the chip once.  With four lanes a
// slot's candidates and fluxes are shared out: mixed, pair kernel, 1.5k
// particles 70 -> 41 us, 32k 147 -> 104, 58k 165 -> 141, but 77k 165 -> 185
// (in a plane 24k 40 -> 31, 43k 41 -> 48), with the sums still taken in
// candidate order, the same bits.  FP64 handles, whose fluxes fill the FP64
// pipe from either form, take four lanes at any size, so that their sums'
// rounding does not depend on how many particles share the handle: 1.5k
// 219 -> 101 us, 32k 572 -> 370, 203k 2175 -> 2095; a 97k plane 261 -> 281.
template <bool MIXED, int DIM, int MODE, bool HLL, bool EXTRA = true>
cudaError_t launch_one(const PairArgs& args, int blocks_per_sm, cudaStream_t st) {
  if constexpr (!MIXED) {
    return launch_lanes<MIXED, DIM, MODE, 4, HLL, EXTRA>(args, blocks_per_sm, st);
  } else {
    if constexpr (MODE != kModeVjp) {
      constexpr int64_t few = DIM == 3 ? 65536 : 32768;
      if (args.n <= few) return launch_lanes<MIXED, DIM, MODE, 4, HLL, EXTRA>(args, blocks_per_sm, st);
    }
    return launch_lanes<MIXED, DIM, MODE, 1, HLL, EXTRA>(args, blocks_per_sm, st);
  }
}

template <bool MIXED, int MODE, bool HLL, bool EXTRA>
cudaError_t launch_dim3(sph_handle* h, const PairArgs& args, cudaStream_t st) {
  const int b = h->p.pair_blocks_per_sm;
  switch (h->dp.dim) {
    case 1: return launch_one<MIXED, 1, MODE, HLL, EXTRA>(args, b, st);
    case 2: return launch_one<MIXED, 2, MODE, HLL, EXTRA>(args, b, st);
    default: return launch_one<MIXED, 3, MODE, HLL, EXTRA>(args, b, st);
  }
}

// The pair solver and the side outputs (neighbour sizes, unit adjacency, pair
// output) are template parameters of the flux modes: as run-time branches in
// the pair loop they cost ~1 % and ~10 % of the kernel.
template <bool MIXED, int MODE>
cudaError_t launch_dim(sph_handle* h, const PairArgs& args, cudaStream_t st) {
  constexpr bool kFlux = MODE == kModeFwd || MODE == kModeFwd2;
  if constexpr (!kFlux) {
    return launch_dim3<MIXED, MODE, false, true>(h, args, st);
  } else {
    const bool extra = args.collect_adj || args.pair_i;
    if (h->solver == SPH_SOLVER_HLL)
      return extra ? launch_dim3<MIXED, MODE, true, true>(h, args, st) : launch_dim3<MIXED, MODE, true, false>(h, args, st);
    return extra ? launch_dim3<MIXED, MODE, false, true>(h, args, st) : launch_dim3<MIXED, MODE, false, false>(h, args, st);
  }
}

}  // namespace

// Reverse mode over the same pair set: the mesh and packs of the state s
// (k_pack of the handle's precision) and the adjoint operands G, GR2 (slot
// order, same precision) must be in place; writes 11 doubles per particle.
cudaError_t launch_pair_vjp(sph_handle* h, const sph_state& s, const void* G, const void* GR2, double* out,
                            cudaStream_t st, const void* A64, const void* B64, const void* C64) {
  PairArgs a = make_args(h, s);
  a.K = 0;
  a.collect_adj = 0;
  a.pair_i = a.pair_j = nullptr;
  a.G = G;
  a.GR2 = GR2;
  a.vjp_out = out;
  const bool fp64 = A64 != nullptr || h->dp.precision != SPH_PREC_MIXED;
  if (A64) {                       // FP64 operands of a mixed handle: unscaled volumes
    a.A = A64;
    a.B = B64;
    a.C = C64;
    a.vinv = 1.0;
  }
  const cudaError_t e = fp64 ? launch_dim<false, kModeVjp>(h, a, st) : launch_dim<true, kModeVjp>(h, a, st);
  h->launches += 1;
  return e;
}

cudaError_t launch_pair(sph_handle* h, const sph_state& s, cudaStream_t st) {
  PairArgs a = make_args(h, s);
  cudaError_t e = cudaSuccess;   // counters zeroed by the k_pack before
  if (h->order2) {
    // SPH gradients first (their own pass over the same pair set), then the rates
    a.gP = h->grad_p;
    a.gV = h->grad_v;
    PairArgs ag = a;
    ag.work_counter = &h->counters[7];
    e = h->dp.precision == SPH_PREC_MIXED ? launch_dim<true, kModeGrad>(h, ag, st)
                                          : launch_dim<false, kModeGrad>(h, ag, st);
    h->launches += 1;
    if (e != cudaSuccess) return e;
  }
  if ((e = prof_record(h, true, st)) != cudaSuccess) return e;
  if (h->order2)
    e = h->dp.precision == SPH_PREC_MIXED ? launch_dim<true, kModeFwd2>(h, a, st)
                                          : launch_dim<false, kModeFwd2>(h, a, st);
  else
    e = h->dp.precision == SPH_PREC_MIXED ? launch_dim<true, kModeFwd>(h, a, st)
                                          : launch_dim<false, kModeFwd>(h, a, st);
  h->launches += 1;
  if (e == cudaSuccess) e = prof_record(h, false, st);
  return e;
}

}  // namespace csph
