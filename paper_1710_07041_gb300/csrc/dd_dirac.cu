// Wilson-clover operator y = D x over the whole lattice (Sec. 1's "discretized
// form of the Dirac equation"; the operator every step of the Schwarz method
// of Sec. 3.1 applies):
//   (D x)(n) = A(n) x(n) - 1/2 sum_mu [(1 - g_mu) U_mu(n) x(n+mu) + (1 + g_mu) U_mu(n-mu)^+ x(n-mu)]
// One thread per (site, right-hand side), right-hand side fastest so that the
// threads of one site share its link and clover loads in L1. The kernel is
// HBM-bound: per site it moves 24 (in) + 24 (out) + 72 (links) + 72 (clover)
// reals once, neighbour spinors being re-read from L1/L2.
#include "dd_fine.cuh"
#include "dd_tune.cuh"

namespace dd {
namespace {

// Like load_spinor, but a DD_F16N site comes back unscaled (its 16-bit
// integers as C): the spinor is out times the returned factor, which the
// caller folds into a later coefficient (one multiply instead of 24). The
// other storages return their values and the factor 1.
template <typename S, typename C>
__device__ __forceinline__ C load_spinor_unscaled(const void *field, const Geom &g, int b, int s, Spinor<C> &out) {
  if constexpr (Store<S>::prec == DD_F16N) {
    DD_CHECK_INDEX(b, g.nblocks);
    DD_CHECK_INDEX(s, g.Vb);
    constexpr int NC = spinor_chunks<S>();
    const char *blk = (const char *)field + (size_t)b * g.Vb * spinor_site_bytes(DD_F16N);
    const size_t cstride = (size_t)g.Vb * 16;
#pragma unroll
    for (int c = 0; c < NC; c++) {
      const uint4 v = __ldg((const uint4 *)(blk + c * cstride + (size_t)s * 16));
      const short *q = (const short *)&v;
#pragma unroll
      for (int k = 0; k < 4; k++) out.c[4 * c + k] = {(C)q[2 * k], (C)q[2 * k + 1]};
    }
    // the site's scale row follows the block's NC chunk rows
    return (C)(__ldg((const float *)(blk + NC * cstride) + s) * (1.0f / 32767.0f));
  } else {
    load_spinor<S, C>(field, g, b, s, out);
    return (C)1;
  }
}

// Loads that bypass L1 (the read-only path without allocating a line): for
// the clover tiles, which the Dslash reads once per site, so that L1 keeps
// the spinor and link lines that neighbouring sites read again.
__device__ __forceinline__ uint4 ld_no_l1(const uint4 *p) {
  uint4 v;
  asm("ld.global.nc.L1::no_allocate.v4.u32 {%0, %1, %2, %3}, [%4];"
      : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w)
      : "l"(p));
  return v;
}
__device__ __forceinline__ uint2 ld_no_l1(const uint2 *p) {
  uint2 v;
  asm("ld.global.nc.L1::no_allocate.v2.u32 {%0, %1}, [%2];" : "=r"(v.x), "=r"(v.y) : "l"(p));
  return v;
}

// out = A psi for a full site, as clover_apply, with the tile chunks read by
// ld_no_l1 (the chunked layout of clover_block_chunked: chunk c of site s at
// q[c * n]; with 4 pairs per chunk the last two pairs of both chirality
// blocks share chunk 8)
template <typename S, typename C>
__device__ __forceinline__ void clover_apply_no_l1(const void *clov, size_t n, int b, int s, const Spinor<C> &in,
                                                   Spinor<C> &out) {
  using P = typename Store<S>::pair_t;
  constexpr int CP = chunk_pairs<P>();
  DD_CHECK_INDEX(s, n);
  const uint4 *q = (const uint4 *)((const P *)clov + (size_t)b * 36 * n) + s;
#pragma unroll
  for (int h = 0; h < 2; h++) {
    cpx<C> m[18];
    if constexpr (CP == 4) {
#pragma unroll
      for (int c = 0; c < 4; c++) {
        const uint4 v = ld_no_l1(q + (size_t)(4 * h + c) * n);
        const P *pv = (const P *)&v;
#pragma unroll
        for (int k = 0; k < 4; k++) m[4 * c + k] = from_pair<C, P>(pv[k]);
      }
      const uint2 w = ld_no_l1((const uint2 *)(q + (size_t)8 * n) + h);
      const P *pw = (const P *)&w;
      m[16] = from_pair<C, P>(pw[0]);
      m[17] = from_pair<C, P>(pw[1]);
    } else {
#pragma unroll
      for (int c = 0; c < 18 / CP; c++) {
        const uint4 v = ld_no_l1(q + (size_t)((18 / CP) * h + c) * n);
        const P *pv = (const P *)&v;
#pragma unroll
        for (int k = 0; k < CP; k++) m[CP * c + k] = from_pair<C, P>(pv[k]);
      }
    }
    herm6_mv(m, &in.c[6 * h], &out.c[6 * h]);
  }
}

// PAIRED: links from the smoother's full-link field in the packed order
template <int MU, typename S, typename C, bool PAIRED = false>
__device__ __forceinline__ void dirac_dir(const Geom &g, const Site &t, const void *links, const void *in,
                                          Spinor<C> &acc) {
  int nb, ns;
  float sg;
  bool inside;
  Link<C> u;
  Spinor<C> psi;
  // hop coefficient -1/2 (times the antiperiodic sign; for DD_F16N also the
  // neighbour's site scale, its spinor being loaded unscaled)
  auto coef = [&](C f) {
    if constexpr (Store<S>::prec == DD_F16N) return (C)(-0.5f * sg) * f;
    else return (C)(-0.5f * sg);
  };
  neighbour(g, t, MU, +1, &nb, &ns, &sg, &inside);
  C f = load_spinor_unscaled<S, C>(in, g, nb, ns, psi);
  if constexpr (PAIRED) load_full_link<S, true>(links, g, t.b, t.s, MU, u);
  else load_link<S, C>(links, g, t.b, t.s, MU, u);
  hop<MU, true>(acc, u, psi, coef(f));
  neighbour(g, t, MU, -1, &nb, &ns, &sg, &inside);
  f = load_spinor_unscaled<S, C>(in, g, nb, ns, psi);
  if constexpr (PAIRED) load_full_link<S, true>(links, g, nb, ns, MU, u);
  else load_link<S, C>(links, g, nb, ns, MU, u);
  hop<MU, false>(acc, u, psi, coef(f));
}

// TPB threads per CTA; MINB resident CTAs per SM requested from the compiler
// (caps registers so more warps keep loads in flight).
// SHAPE: the block shape as compile-time constants (see block_shape), or 0.
// SO: storage of the output fields (the input's, or FP64 for double-float inputs).
// NL1: the clover tiles read without allocating L1 lines.
template <typename S, int TPB, int MINB, int SHAPE, bool NL1, typename SO = S>
__global__ void __launch_bounds__(TPB, MINB) k_dirac(Geom g_in, const void *__restrict__ links,
                                                     const void *__restrict__ clov, const RhsPtrs p) {
  using C = typename Store<S>::comp_t;
  const Geom g = block_shape<SHAPE>(g_in);
  const int nrhs = p.n;
  long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (t >= g.V * nrhs) return;
  long long site = t / nrhs;
  int r = (int)(t - site * nrhs);
  int b = (int)(site / g.Vb), s = (int)(site - (long long)b * g.Vb);
  const void *inr = p.in[r];
  Site st = decode(g, b, s);
  Spinor<C> x, acc;
  load_spinor<S, C>(inr, g, b, s, x);
  if constexpr (NL1) clover_apply_no_l1<S, C>(clov, g.Vb, b, s, x, acc);
  else clover_apply<S, C>(clov, g.Vb, b, s, x, acc);
  dirac_dir<0, S, C>(g, st, links, inr, acc);
  dirac_dir<1, S, C>(g, st, links, inr, acc);
  dirac_dir<2, S, C>(g, st, links, inr, acc);
  dirac_dir<3, S, C>(g, st, links, inr, acc);
  store_spinor<SO, C>(p.out[r], g, b, s, acc);
}

// r = b - D x, r as an FP32 field, on the blocks of one colour or on all
// (colour < 0): the residual of the Schwarz smoother's phases from a given
// iterate (the arithmetic of k_dirac, the result not rounded to the storage of
// x and b). PAIRED: with the smoother's own links, all nine entries as rounded
// to the storage (a third row rebuilt from the rounded two is another operator:
// in BF16 the smoothed x then differed by 1.8e-3)
template <typename S, int SHAPE, bool PAIRED>
__global__ void __launch_bounds__(128, 5) k_residual(Geom g_in, const void *__restrict__ links,
                                                     const void *__restrict__ clov, const RhsPtrs px,
                                                     const RhsPtrs pb, int colour) {
  using C = typename Store<S>::comp_t;
  const Geom g = block_shape<SHAPE>(g_in);
  const int nrhs = px.n;
  const long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (t >= (colour < 0 ? g.V : g.V / 2) * nrhs) return;
  const long long site = t / nrhs;
  const int r = (int)(t - site * nrhs);
  const int bi = (int)(site / g.Vb), s = (int)(site - (long long)bi * g.Vb);
  const int b = colour < 0 ? bi : sap_block_of(g, colour, bi);
  const Site st = decode(g, b, s);
  Spinor<C> x, acc;
  if constexpr (PAIRED) {
    // the hops summed apart from the site term, as in the block solves' kernels
    // (onto A x, four times as large as the result, each sum rounds more: FP32
    // from a given x, error against 64 bits 1.43 against 1.41e-7)
    Spinor<C> ax;
#pragma unroll
    for (int i = 0; i < 12; i++) acc.c[i] = {0, 0};
    dirac_dir<0, S, C, PAIRED>(g, st, links, px.in[r], acc);
    dirac_dir<1, S, C, PAIRED>(g, st, links, px.in[r], acc);
    dirac_dir<2, S, C, PAIRED>(g, st, links, px.in[r], acc);
    dirac_dir<3, S, C, PAIRED>(g, st, links, px.in[r], acc);
    load_spinor<S, C>(px.in[r], g, b, s, x);
    clover_apply_no_l1<S, C>(clov, g.Vb, b, s, x, ax);
#pragma unroll
    for (int i = 0; i < 12; i++) acc.c[i] = {ax.c[i].re + acc.c[i].re, ax.c[i].im + acc.c[i].im};
  } else {
    load_spinor<S, C>(px.in[r], g, b, s, x);
    clover_apply_no_l1<S, C>(clov, g.Vb, b, s, x, acc);
    dirac_dir<0, S, C, PAIRED>(g, st, links, px.in[r], acc);
    dirac_dir<1, S, C, PAIRED>(g, st, links, px.in[r], acc);
    dirac_dir<2, S, C, PAIRED>(g, st, links, px.in[r], acc);
    dirac_dir<3, S, C, PAIRED>(g, st, links, px.in[r], acc);
  }
  load_spinor<S, C>(pb.in[r], g, b, s, x);
#pragma unroll
  for (int i = 0; i < 12; i++) acc.c[i] = {x.c[i].re - acc.c[i].re, x.c[i].im - acc.c[i].im};
  store_spinor<float, C>(px.out[r], g, b, s, acc);
}
template <typename S>
int residual_t(const Geom &g, const OpFields &f, const RhsPtrs &x, const RhsPtrs &b, int colour, cudaStream_t st) {
  const unsigned grid = (unsigned)(((colour < 0 ? g.V : g.V / 2) * x.n + 127) / 128);
  auto launch = [&](auto kern, const void *links) { kern<<<grid, 128, 0, st>>>(g, links, f.clov, x, b, colour); };
  if (colour >= 0) {
    if (!paired_links(g, f.prec)) {
      set_error("residual of one colour: packed links only");
      return DD_EINVAL;
    }
    if (shape_of(g) == 1) launch(k_residual<S, 1, true>, f.links_full);
    else launch(k_residual<S, 2, true>, f.links_full);
  } else if (shape_of(g) == 1) {
    launch(k_residual<S, 1, false>, f.links);
  } else {
    launch(k_residual<S, 0, false>, f.links);
  }
  return launched("k_residual");
}

template <typename S, int TPB, int MINB, bool NL1, typename SO = S>
int dirac_v(const Geom &g, const OpFields &f, const RhsPtrs &p, cudaStream_t st) {
  long long n = g.V * p.n;
  const unsigned grid = (unsigned)((n + TPB - 1) / TPB);
  if (shape_of(g) == 1) k_dirac<S, TPB, MINB, 1, NL1, SO><<<grid, TPB, 0, st>>>(g, f.links, f.clov, p);
  else k_dirac<S, TPB, MINB, 0, NL1, SO><<<grid, TPB, 0, st>>>(g, f.links, f.clov, p);
  return launched("k_dirac");
}

// FP64 on small lattices: twelve threads per site (see dd_fine.cuh), 16 sites
// per CTA (of one right-hand side; every block holds a multiple of 16). One or
// two threads a site leave most of the chip's 608 SM sub-partitions (each half
// an FP64 lane per clock) idle here and take the length of one thread's chain,
// ~1130 instructions of 64 clocks: 40.5 us on 4^4 as on 16 x 8^3. A thread of
// this kernel runs ~115: 8.1 us on 4^4.
constexpr int FINE_SITES = 16;
__global__ void __launch_bounds__(12 * FINE_SITES) k_dirac_fine(Geom g, const double2 *__restrict__ links,
                                                               const double2 *__restrict__ clov, const RhsPtrs rp) {
  __shared__ double2 X[24 * FINE_SITES];   // [upper: half 0, half 1; lower: half 0, half 1][6][site]
  const int tiles = g.Vb / FINE_SITES, cta = (int)(blockIdx.x / rp.n), rhs = (int)(blockIdx.x - (unsigned)cta * rp.n);
  const int b = cta / tiles, s0 = (cta - b * tiles) * FINE_SITES;
  FineThread T;
  T.d = threadIdx.x >= 6 * FINE_SITES;
  const int t = threadIdx.x - T.d * 6 * FINE_SITES;
  T.k = t / FINE_SITES;
  T.q = t - T.k * FINE_SITES;
  T.h = T.k / 3;
  T.c = T.k - 3 * T.h;
  T.sh = T.h ? -1.0 : 1.0;
#pragma unroll
  for (int j = 0; j < 6; j++) {
    const int i0 = j < T.k ? j : T.k, j0 = j < T.k ? T.k : j;
    T.off[j] = j == T.k ? T.k >> 1 : herm_off(i0, j0);
  }
  const int s = s0 + T.q;
  const Site st = decode(g, b, s);
  const double2 *in = (const double2 *)rp.in[rhs], *own = in + ((size_t)b * 12 + 6 * T.d) * g.Vb + s;
  const double2 y = fine_row(T, clov + ((size_t)b * 36 + 18 * T.d) * g.Vb + s, g.Vb,
                             [&](int j) { return own[(size_t)j * g.Vb]; });
  FineAcc o;
  fine_global(T, g, st, links, in, false, false, o);
  const int lk = T.d ? T.k : T.c + 3 * (1 - T.h);   // lower component of o.l
  X[(6 * T.d + T.k) * FINE_SITES + T.q] = o.u;
  X[(12 + 6 * T.d + lk) * FINE_SITES + T.q] = o.l;
  __syncthreads();
  const double2 *Xd = X + (12 * T.d + T.k) * FINE_SITES + T.q;
  ((double2 *)rp.out[rhs])[((size_t)b * 12 + 6 * T.d + T.k) * g.Vb + s] = add(y, add(Xd[0], Xd[6 * FINE_SITES]));
}
// Twelve threads run 1.22 times the instructions of one, so the gain ends where
// the chip is full. The line depends on the lattice alone (a right-hand side's
// result must not depend on its batch). Measured, one thread per site -> this
// kernel, in us:
//   sites   1 rhs          4 rhs          12 rhs
//     256   40.5 ->  8.1   41.2 ->  8.1    42.6 ->  14.2
//    1024   40.8 ->  8.3   41.6 -> 14.3    42.6 ->  38.7
//    4096   40.1 -> 14.3   41.3 -> 45.3   115.2 -> 130.8
// (at 1024 sites the two meet at 15 right-hand sides)
inline bool fine_lattice(const Geom &g) { return g.V <= 1024; }

// Launch variants (threads per CTA, CTAs per SM the register budget must
// allow): (128, 5) ~100 registers, (128, 6) ~80, (256, 2) ~128 and (256, 3)
// ~85; for FP64 (128, 4) ~128, (128, 3) ~168, (256, 2) ~128, (256, 1) 255;
// variants 4-7 are 0-3 with the clover tiles read past L1.
// A 256-thread CTA covers one whole 4^4 block, so interior neighbours are
// read by the same SM.
constexpr int DIRAC_VARIANTS = 8;

template <typename S, typename SO = S>
int dirac_t(const Geom &g, const OpFields &f, const RhsPtrs &p, cudaStream_t st) {
  auto shape = [&](int v, auto nl1) {
    constexpr bool N = decltype(nl1)::value;
    if constexpr (Store<S>::prec == DD_F64 || Store<S>::prec == DD_PREC_DF) {
      // FP64 and double-float values take two registers each: looser caps
      switch (v) {
        case 1: return dirac_v<S, 128, 3, N, SO>(g, f, p, st);
        case 2: return dirac_v<S, 256, 2, N, SO>(g, f, p, st);
        case 3: return dirac_v<S, 256, 1, N, SO>(g, f, p, st);
        default: return dirac_v<S, 128, 4, N, SO>(g, f, p, st);
      }
    } else {
      switch (v) {
        case 1: return dirac_v<S, 128, 6, N>(g, f, p, st);
        case 2: return dirac_v<S, 256, 2, N>(g, f, p, st);
        case 3: return dirac_v<S, 256, 3, N>(g, f, p, st);
        default: return dirac_v<S, 128, 5, N>(g, f, p, st);
      }
    }
  };
  auto run = [&](int v) {
    return v >= 4 ? shape(v - 4, std::true_type{}) : shape(v, std::false_type{});
  };
  if constexpr (std::is_same<S, double>::value) {
    if (fine_lattice(g)) {
      k_dirac_fine<<<(unsigned)(g.V / FINE_SITES * p.n), 12 * FINE_SITES, 0, st>>>(
          g, (const double2 *)f.links, (const double2 *)f.clov, p);
      return launched("k_dirac_fine");
    }
  }
  int v = 0;
  const TuneFast fast = tune_fast_key(1, g, f.prec, p.n);
  if (!tune_fast_find(fast, &v)) {
    const std::string key = tune_key("dirac", g, f.prec, p.n);
    if (int rc = tuned_variant(key, DIRAC_VARIANTS, run, st, &v)) return rc;
    if (!getenv("DD_TUNE_VARIANT") && tune_lookup(key) == v) tune_fast_store(fast, v);
  }
  return run(v);
}

}  // namespace

RhsPtrs contiguous(const void *in, void *out, int nrhs, size_t field_bytes) {
  RhsPtrs p;
  p.n = nrhs;
  for (int r = 0; r < nrhs && r < MAX_RHS; r++) {
    p.in[r] = (const char *)in + r * field_bytes;
    p.out[r] = (char *)out + r * field_bytes;
  }
  return p;
}

int launch_dirac(const Geom &g, const OpFields &f, const RhsPtrs &p, cudaStream_t st) {
  NvtxRange range("dd:dirac");
  if (p.n < 1 || p.n > MAX_RHS) {
    set_error("apply_D: 1..%d right-hand sides per launch", MAX_RHS);
    return DD_EINVAL;
  }
  switch (f.prec) {
    case DD_F64: return dirac_t<double>(g, f, p, st);
    case DD_F32: return dirac_t<float>(g, f, p, st);
    case DD_F16: return dirac_t<__half>(g, f, p, st);
    case DD_BF16: return dirac_t<__nv_bfloat16>(g, f, p, st);
    case DD_F16N: return dirac_t<hn16>(g, f, p, st);
  }
  set_error("apply_D: precision %d not available", f.prec);
  return DD_EINVAL;
}

int launch_residual(const Geom &g, const OpFields &f, const RhsPtrs &x, const RhsPtrs &b, int colour, cudaStream_t st) {
  switch (f.prec) {
    case DD_F32: return residual_t<float>(g, f, x, b, colour, st);
    case DD_F16: return residual_t<__half>(g, f, x, b, colour, st);
    case DD_BF16: return residual_t<__nv_bfloat16>(g, f, x, b, colour, st);
    case DD_F16N: return residual_t<hn16>(g, f, x, b, colour, st);
  }
  set_error("residual: precision %d not available", f.prec);
  return DD_EINVAL;
}

int launch_dirac_df(const Geom &g, const OpFields &f, const RhsPtrs &p, cudaStream_t st) {
  if (p.n < 1 || p.n > MAX_RHS || f.prec != DD_PREC_DF || !f.links) {
    set_error("apply_D (double-float): double-float fields and 1..%d right-hand sides", MAX_RHS);
    return DD_EINVAL;
  }
  return dirac_t<dfs, double>(g, f, p, st);
}

int launch_dirac(const Geom &g, const OpFields &f, const void *in, void *out, int nrhs, cudaStream_t st) {
  const size_t fb = (size_t)g.V * spinor_site_bytes(f.prec);
  for (int r0 = 0; r0 < nrhs; r0 += MAX_RHS) {
    int n = nrhs - r0 < MAX_RHS ? nrhs - r0 : MAX_RHS;
    int rc = launch_dirac(g, f, contiguous((const char *)in + r0 * fb, (char *)out + r0 * fb, n, fb), st);
    if (rc) return rc;
  }
  return DD_OK;
}

}  // namespace dd
