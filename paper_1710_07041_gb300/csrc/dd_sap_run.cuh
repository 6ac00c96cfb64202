// Host side of the Schwarz smoother for one storage precision: launch
// variants, tuning, graph key (included by dd_sap_<prec>.cu).
#pragma once
#include "dd_sap_fine.cuh"
#include "dd_sap_pair.cuh"

namespace dd {
namespace {

// the kernel specialised for the lattice's block shape when there is one
template <typename S, int STAGE, int MINB, int NT = 256>
int sap_t(const SapLattice *L, int nl, const dd_sap_params &p, const RhsPtrs &rp, const SapWork *ax, int tile,
          bool persistent, bool prepare, cudaStream_t st) {
  constexpr int SH = NT == 256 ? 1 : 2;   // the shape this thread count fits
  if (shape_of(L[0].g) == SH)
    return nl > 1 ? sap_k<S, STAGE, MINB, NT, SH, true>(L, nl, p, rp, ax, tile, persistent, prepare, st)
                  : sap_k<S, STAGE, MINB, NT, SH>(L, nl, p, rp, ax, tile, persistent, prepare, st);
  return nl > 1 ? sap_k<S, STAGE, MINB, NT, 0, true>(L, nl, p, rp, ax, tile, persistent, prepare, st)
                : sap_k<S, STAGE, MINB, NT, 0>(L, nl, p, rp, ax, tile, persistent, prepare, st);
}

// One smoother application in the packed kernel (dd_sap_pair.cuh). From a
// given x each phase of the first sweep works on the residual b - D x of x as
// stored, formed on its colour's blocks as an FP32 field by the operator's
// kernel (so the rounding of x in the first colour's update is seen by the
// second); after that, as from x = 0, every phase takes its residual from the
// stored one and the neighbours' flux. With r0 alone (no e and r) every phase
// but the first from x = 0 does so: the two-level preconditioner's 16-bit
// smoother, whose residual and corrections are not to pass between phases in 16
// bits (dd_mg.cu).
template <typename S, int SHAPE, bool MULTI>
int sap_pair_k(const SapLattice *L, int nl, const dd_sap_params &p, const RhsPtrs &rp, const SapWork &ax, int tile,
               bool prepare, cudaStream_t st) {
  using PG = PairGeom<SHAPE>;
  auto kern = k_sap_pair<S, SHAPE, MULTI>;
  static DeviceOnce once;
  if (int rc = raise_smem(kern, (int)PG::SMEM, once)) return rc;
  if (prepare) return DD_OK;
  const SapGroups G = sap_groups(L, nl, tile);
  // Each CTA requests into L2 the operator of the block that a quarter of the
  // resident CTAs ahead of it starts on (a block's start then waits for L2
  // instead of HBM: 0.412 -> 0.405 ms per FP32 phase at 64x32^3; half of the
  // resident CTAs ahead: 0.428, all of them: 0.445, the requests then push
  // one another out of L2)
  int dev = 0, sms = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  const int ahead = sms * (SHAPE == 1 ? 2 : 1) / 4;
  auto residual = [&](int colour) -> int {   // ax.r0 = b - D x on the blocks of a colour
    RhsPtrs x, b;
    for (int k = 0, r = 0; k < nl; k++) {
      x.n = b.n = L[k].nrhs;
      for (int i = 0; i < L[k].nrhs; i++, r++) {
        x.in[i] = rp.out[r];
        x.out[i] = ax.r0[r];
        b.in[i] = rp.in[r];
        b.out[i] = nullptr;
      }
      if (int rc = launch_residual(L[k].g, L[k].f, x, b, colour, st)) return rc;
    }
    return DD_OK;
  };
  RhsPtrs from_r0 = rp;
  for (int r = 0; r < rp.n; r++) from_r0.in[r] = ax.r0[r];
  const bool incr = ax.e[0] != nullptr;
  if (!incr && p.x_is_zero)   // the second phase's residual reads x on every block
    for (int k = 0, r = 0; k < nl; k++)
      for (int i = 0; i < L[k].nrhs; i++, r++)
        DD_CUDA(cudaMemsetAsync(rp.out[r], 0, (size_t)L[k].g.V * spinor_site_bytes(Store<S>::prec), st));
  for (int sw = 0; sw < p.sweeps; sw++)
    for (int colour = 0; colour < 2; colour++) {
      const bool given = incr ? sw == 0 && !p.x_is_zero : sw || colour || !p.x_is_zero;   // works on b - D x
      int mode = given ? SAP_FROM_B | SAP_B32 : sw ? SAP_HALO_E : SAP_FROM_B | (colour ? SAP_HALO_E : 0);
      if (given)
        if (int rc = residual(colour)) return rc;
      // e is read by the next phase, unless this is the last or that forms b - D x
      if (incr && !(sw == p.sweeps - 1 && colour == 1) && !(given && colour == 0)) mode |= SAP_WRITE_E;
      if (incr && sw + 1 < p.sweeps) mode |= SAP_WRITE_R;   // r by this colour's next one
      // programmatic launch: while the phase before drains a phase's CTAs start,
      // load their clover blocks, ask for the links (a bulk copy in FP32) and
      // for a later block's operator; at the CTA barrier in front of the
      // tensor-memory stores they wait for it (griddepcontrol.wait in the threads
      // that fetch what it wrote), so the rest of the staging does not overlap
      // (64x32^3: 0.388 -> 0.374 ms per phase; 16x8^3: 23.1 -> 20.3 us)
      DD_CUDA(launch_ahead(true, kern, dim3((unsigned)G.nitems), dim3(PG::NT), PG::SMEM, st, G, given ? from_r0 : rp,
                           (const AuxPtrs &)ax, colour, (int)(p.x_is_zero && sw == 0), mode, (int)p.mr_steps, tile,
                           ahead, sap_timeout_counter()));
      DD_LAUNCHED();
    }
  return DD_OK;
}

// one smoother application in the FP64 small-block kernel (dd_sap_fine.cuh)
template <bool MULTI>
int sap_fine_k(const SapLattice *L, int nl, const dd_sap_params &p, const RhsPtrs &rp, const SapWork *ax, int tile,
               bool prepare, cudaStream_t st) {
  static DeviceOnce once;   // 32-site blocks need a little over 48 KB
  if (int rc = raise_smem(k_sap_fine<MULTI>, 64 * 1024, once)) return rc;
  if (prepare) return DD_OK;
  const SapGroups G = sap_groups(L, nl, tile);
  const AuxPtrs none{};
  for (int sw = 0; sw < p.sweeps; sw++)
    for (int colour = 0; colour < 2; colour++) {
      const SapPhase f = sap_phase(p, sw, colour, ax != nullptr);
      k_sap_fine<MULTI><<<G.nitems, fine_threads(L[0].g), fine_smem(L[0].g), st>>>(
          G, rp, ax ? (const AuxPtrs &)*ax : none, colour, f.self_zero, f.halo_zero, f.mode, p.mr_steps, tile);
      DD_LAUNCHED();
    }
  return DD_OK;
}

// Launch variants. The 4^4 and 8 x 4^3 blocks in 32- and 16-bit storage run
// in the packed kernel, whatever the lattice size and right-hand-side count (it
// won from 32 to 8192 blocks: 24.3 -> 19.5 us per phase on 16x8^3, 0.514 -> 0.370
// ms on 64x32^3); only a call without work fields (or DD_SAP_INCR=0) takes the
// general kernel there, whose layouts read the packed links one real at a time
// (four sweeps without work fields, unstaged alone -> the layouts below: FP32
// 16x8^3 273 -> 224 us, 64x32^3 5.52 -> 5.51 ms, FP16 5.47 -> 4.85 ms). FP64 blocks of 16 and 32 sites (a warp or less of
// the general kernel's threads) run in the small-block kernel: 340 -> 43 us per
// phase on 4^4 (blocks of 256 sites fill the general kernel's warps). Everything else runs in the general kernel:
// tiles staged in shared memory with one CTA per SM; tiles staged with two
// CTAs per SM (fits when the storage is 16-bit); only the links staged, with
// two CTAs per SM (when the full staging does not fit twice); tiles read
// through L1/L2 with two CTAs per SM. Variants that do not fit are skipped.
// With several right-hand sides a CTA also solves `tile` of them with one
// staging of its block's operator (rhs_tile; 0 lets the autotuner choose).
template <typename S>
int sap_variants(const SapLattice *L, int nl, const dd_sap_params &p, const RhsPtrs &rp, const SapWork *ax,
                 cudaStream_t st) {
  const Geom &g = L[0].g;
  const bool paired = paired_links(g, L[0].f.prec);
  const bool incr = ax && ax->e[0], r0 = ax && ax->r0[0];
  if (paired ? !r0 && !(incr && p.x_is_zero) : !incr) ax = nullptr;
  const bool pair = paired && ax, fine = Store<S>::prec == DD_F64 && fine_block(g);
  const size_t limit = 227 * 1024, half = 113 * 1024;
  const bool stage1 = SapSmem<S>::bytes(g, 1) <= limit;
  const bool stage2 = SapSmem<S>::bytes(g, 1) <= half;
  const bool links2 = !stage2 && SapSmem<S>::bytes(g, 2) <= half;
  const bool nost2 = SapSmem<S>::bytes(g, 0) <= half;
  if (!stage1 && SapSmem<S>::bytes(g, 0) > limit) {
    set_error("sap: block of %d sites needs more shared memory than available", g.Vb);
    return DD_EINVAL;
  }
  int layouts[4], nlay = 0;
  if (g.Vb > 256) {
    // 512-site blocks (e.g. 8 x 4^3): 512 threads, one CTA per SM
    layouts[nlay++] = stage1 ? 3 : 4;
  } else {
    if (stage1) layouts[nlay++] = 0;
    if (stage2) layouts[nlay++] = 1;
    if (links2) layouts[nlay++] = 5;
    if (nost2 || !stage1) layouts[nlay++] = 2;
  }
  int tiles[6], nt = 0;
  if (p.rhs_tile > 0) {
    tiles[nt++] = p.rhs_tile < rp.n ? p.rhs_tile : rp.n;
  } else {
    const int cand[5] = {1, 2, 4, 8, 12};
    for (int c : cand)
      if (c <= rp.n) tiles[nt++] = c;
  }
  // variant k: layout k % nlay, RHS tile (k / nlay) % nt, persistent grid if
  // k >= nlay * nt; packed and small-block kernels: RHS tile k
  auto variant = [&](int k, bool prepare) {
    if constexpr (Store<S>::prec != DD_F64) {
      if (pair) {
        if (shape_of(g) == 1)
          return nl > 1 ? sap_pair_k<S, 1, true>(L, nl, p, rp, *ax, tiles[k], prepare, st)
                        : sap_pair_k<S, 1, false>(L, nl, p, rp, *ax, tiles[k], prepare, st);
        return nl > 1 ? sap_pair_k<S, 2, true>(L, nl, p, rp, *ax, tiles[k], prepare, st)
                      : sap_pair_k<S, 2, false>(L, nl, p, rp, *ax, tiles[k], prepare, st);
      }
    }
    if constexpr (Store<S>::prec == DD_F64) {
      if (fine)
        return nl > 1 ? sap_fine_k<true>(L, nl, p, rp, ax, tiles[k], prepare, st)
                      : sap_fine_k<false>(L, nl, p, rp, ax, tiles[k], prepare, st);
    }
    const int layout = layouts[k % nlay], tile = tiles[(k / nlay) % nt];
    const bool pers = k >= nlay * nt;
    switch (layout) {
      case 1: return sap_t<S, 1, 2>(L, nl, p, rp, ax, tile, pers, prepare, st);
      case 2: return sap_t<S, 0, 2>(L, nl, p, rp, ax, tile, pers, prepare, st);
      case 3: return sap_t<S, 1, 1, 512>(L, nl, p, rp, ax, tile, pers, prepare, st);
      case 4: return sap_t<S, 0, 1, 512>(L, nl, p, rp, ax, tile, pers, prepare, st);
      case 5: return sap_t<S, 2, 2>(L, nl, p, rp, ax, tile, pers, prepare, st);
      default: return sap_t<S, 1, 1>(L, nl, p, rp, ax, tile, pers, prepare, st);
    }
  };
  auto run = [&](int k) { return variant(k, false); };
  const int nvar = pair || fine ? nt : 2 * nlay * nt;
  int k = 0;
  // the tuner's key: lattice, precision, right-hand-side count, smoother
  // parameters and boundary; a launch over several lattices is tuned once
  // per block shape, precision and total right-hand-side count (a served
  // stream meets ever new mixes of lattices, each would otherwise be tuned)
  const std::string kind = pair ? "sap-pair" : fine ? "sap-fine" : "sap";
  std::string key;
  if (nl == 1) {
    key = tune_key(kind.c_str(), g, L[0].f.prec, rp.n) + "|" + std::to_string(p.sweeps) + "," +
          std::to_string(p.mr_steps) + "," + std::to_string(p.rhs_tile) + "," + std::to_string(g.antiperiodic);
  } else {
    Geom gb = g;   // the block shape only
    for (int mu = 0; mu < 4; mu++) gb.L[mu] = 0;
    key = tune_key((kind + "-lattices").c_str(), gb, L[0].f.prec, rp.n) + "|" + std::to_string(p.sweeps) + "," +
          std::to_string(p.mr_steps) + "," + std::to_string(p.rhs_tile);
  }
  // the graph cache's key adds every lattice's extents, boundary and right-hand sides
  std::string shape;
  for (int k = 0; k < nl; k++)
    shape += "|" + std::to_string(L[k].g.L[0]) + "," + std::to_string(L[k].g.L[1]) + "," +
             std::to_string(L[k].g.L[2]) + "," + std::to_string(L[k].g.L[3]) + "," + std::to_string(L[k].nrhs) + "," +
             std::to_string(L[k].g.antiperiodic);
  // a graph may only replay where a fresh capture records the same arguments:
  // every lattice's field pointers are part of its key
  std::string fields = p.x_is_zero ? "z" : "x";
  for (int k = 0; k < nl; k++)
    fields += std::to_string((uintptr_t)L[k].f.links_full) + "," + std::to_string((uintptr_t)L[k].f.clov) + "," +
              std::to_string((uintptr_t)L[k].f.cinv) + "," + std::to_string((uintptr_t)L[k].f.links) + ";";
  if (pair && r0)
    for (int r = 0; r < rp.n; r++) fields += std::to_string((uintptr_t)ax->r0[r]) + ",";
  // x is pure output when x_is_zero, so trial runs leave the same result
  if (p.x_is_zero) {
    int rc = tuned_variant(key, nvar, run, st, &k);
    if (rc) return rc;
  } else {
    int c = tune_lookup(key);
    k = c >= 0 && c < nvar ? c : 0;
  }
  // (the launches below may be captured: with one variant nothing has run it yet)
  if (int rc = variant(k, true)) return rc;
  // launches of an application: the phases and, in the packed kernel, the residuals formed ahead of them
  const int nres = !pair ? 0 : !incr ? 2 * p.sweeps - (p.x_is_zero ? 1 : 0) : p.x_is_zero ? 0 : 2;
  return sap_launch_as_graph(key + shape + "|" + fields, k, 2 * p.sweeps + nres * nl, rp, ax, [&] { return run(k); },
                             st);
}

}  // namespace
}  // namespace dd
