// Schwarz colour phase for blocks of 16 and 32 sites in FP64 (the 2^4 block of
// the plain method), six threads per site. The method and the residual modes
// are those of k_sap_phase.
//
// Why. GB300 issues one FP64 instruction of a warp in about 64 clocks per SM
// sub-partition whatever the number of active lanes, and k_sap_phase gives a
// 2^4 block one half-filled warp that runs ~700 of them per half-step: a
// phase on 4^4 (8 blocks) took 340 us with one of four sub-partitions of 8
// SMs at work. Here thread (spin component h, colour c) of a site computes
// one colour of one spin component of every projected hop, and row 3h + c of
// both chirality blocks: ~130 FP64 instructions per half-step in 1.5 warps per
// block. The projections are formed three times over (each by the threads of
// its three colours): 66 instead of 54 FP64 operations per hop and spin.
//
// The even sites' correction is accumulated over the MR steps (e_e = te_0 -
// sum_k alpha_k te_k with te = A_ee^-1 D_eo rho), which saves the last
// half-step. The block's links, A_oo and A_ee^-1 are copied to shared memory.
#pragma once
#include "dd_sap_kernels.cuh"

namespace dd {
namespace {

struct FineThread {
  int h, c, k, q;     // spin, colour, 3 h + c, site of either parity
  int off[6];         // pair of entry (k, j) in a packed Hermitian block
  double sh;          // +1 (h = 0), -1 (h = 1)
};
__device__ __forceinline__ double2 z2(double x, double y) { return make_double2(x, y); }

// the sums of a thread: upper spin h (u), lower spin h (a) and 1 - h (b), colour c
struct FineAcc {
  double2 u, a, b;
};

// one hop: v(i) the source's component i, w(i) the link's entry i; s = -1/2
// times the boundary sign
template <int MU, bool FWD, typename V, typename W>
__device__ __forceinline__ void fine_hop(const FineThread &T, double s, V v, W w, FineAcc &o) {
  const int du = MU < 2 ? 9 - 3 * T.h : 6 + 3 * T.h;   // first colour of the lower spin projected on
  constexpr double F = FWD ? 1.0 : -1.0;
  // chi = u + f d (MU 1, 3) or u + i f d (MU 0, 2)
  const double f = MU == 0 ? F : MU == 3 ? -F : F * T.sh;
  double2 y = z2(0, 0);
#pragma unroll
  for (int k = 0; k < 3; k++) {
    const double2 up = v(3 * T.h + k), d = v(du + k), m = w(FWD ? 3 * T.c + k : 3 * k + T.c);
    const double2 x = (MU == 0 || MU == 2) ? z2(fma(-f, d.y, up.x), fma(f, d.x, up.y))
                                           : z2(fma(f, d.x, up.x), fma(f, d.y, up.y));
    const double mi = FWD ? m.y : -m.y;   // U chi or U^dagger chi
    y.x = fma(m.x, x.x, y.x);
    y.x = fma(-mi, x.y, y.x);
    y.y = fma(m.x, x.y, y.y);
    y.y = fma(mi, x.x, y.y);
  }
  o.u.x = fma(s, y.x, o.u.x);
  o.u.y = fma(s, y.y, o.u.y);
  // the lower spins: the conjugate phase times the hop's sign
  if constexpr (MU == 0) {
    o.b.x = fma(F * s, y.y, o.b.x);
    o.b.y = fma(-F * s, y.x, o.b.y);
  } else if constexpr (MU == 1) {
    o.b.x = fma(f * s, y.x, o.b.x);
    o.b.y = fma(f * s, y.y, o.b.y);
  } else if constexpr (MU == 2) {
    o.a.x = fma(f * s, y.y, o.a.x);
    o.a.y = fma(-f * s, y.x, o.a.y);
  } else {
    o.a.x = fma(-F * s, y.x, o.a.x);
    o.a.y = fma(-F * s, y.y, o.a.y);
  }
}

// row k of a packed Hermitian block (m: its first pair, n sites per pair row)
// times x(j), j = 0..5
template <typename X>
__device__ __forceinline__ double2 fine_row(const FineThread &T, const double2 *m, int n, X x) {
  double2 y = z2(0, 0);
#pragma unroll
  for (int j = 0; j < 6; j++) {
    const double2 e = m[T.off[j] * n], v = x(j);
    const double ar = j == T.k ? (T.k & 1 ? e.y : e.x) : e.x;
    const double ai = j == T.k ? 0.0 : j < T.k ? -e.y : e.y;
    y.x = fma(ar, v.x, y.x);
    y.x = fma(-ai, v.y, y.x);
    y.y = fma(ar, v.y, y.y);
    y.y = fma(ai, v.x, y.y);
  }
  return y;
}

// hops inside the block into the thread's site of parity p, from the shared
// vector v of the other parity; nb: its in-block neighbours (-1: outside)
__device__ __forceinline__ void fine_inner(const FineThread &T, const int *nb, int Vb, int Vh, int p, const double2 *v,
                                           const double2 *L, FineAcc &o) {
  o.u = o.a = o.b = z2(0, 0);
  auto dir = [&](auto mu, auto fwd) {
    constexpr int MU = decltype(mu)::value;
    constexpr bool FWD = decltype(fwd)::value;
    const int n = nb[2 * MU + (FWD ? 0 : 1)];
    if (n < 0) return;
    const double2 *w = L + 9 * MU * Vb + (FWD ? p * Vh + T.q : (1 - p) * Vh + n);
    fine_hop<MU, FWD>(T, -0.5, [&](int i) { return v[i * Vh + n]; }, [&](int i) { return w[i * Vb]; }, o);
  };
  using std::integral_constant;
  dir(integral_constant<int, 0>{}, std::true_type{});
  dir(integral_constant<int, 0>{}, std::false_type{});
  dir(integral_constant<int, 1>{}, std::true_type{});
  dir(integral_constant<int, 1>{}, std::false_type{});
  dir(integral_constant<int, 2>{}, std::true_type{});
  dir(integral_constant<int, 2>{}, std::false_type{});
  dir(integral_constant<int, 3>{}, std::true_type{});
  dir(integral_constant<int, 3>{}, std::false_type{});
}
// hops into site t from the global field x: from neighbours inside the block
// unless self_zero, outside unless halo_zero
__device__ __forceinline__ void fine_global(const FineThread &T, const Geom &g, const Site &t, const double2 *links,
                                            const double2 *x, bool self_zero, bool halo_zero, FineAcc &o) {
  o.u = o.a = o.b = z2(0, 0);
  auto dir = [&](auto mu, auto fwd) {
    constexpr int MU = decltype(mu)::value;
    constexpr bool FWD = decltype(fwd)::value;
    int nb, ns;
    float sg;
    bool inside;
    neighbour(g, t, MU, FWD ? 1 : -1, &nb, &ns, &sg, &inside);
    if (inside ? self_zero : halo_zero) return;
    DD_CHECK_INDEX(nb, g.nblocks);
    DD_CHECK_INDEX(ns, g.Vb);
    const double2 *v = x + (size_t)nb * 12 * g.Vb + ns;
    const double2 *w = links + ((size_t)(FWD ? t.b : nb) * 36 + 9 * MU) * g.Vb + (FWD ? t.s : ns);
    fine_hop<MU, FWD>(T, -0.5 * sg, [&](int i) { return v[(size_t)i * g.Vb]; },
                      [&](int i) { return w[(size_t)i * g.Vb]; }, o);
  };
  using std::integral_constant;
  dir(integral_constant<int, 0>{}, std::true_type{});
  dir(integral_constant<int, 0>{}, std::false_type{});
  dir(integral_constant<int, 1>{}, std::true_type{});
  dir(integral_constant<int, 1>{}, std::false_type{});
  dir(integral_constant<int, 2>{}, std::true_type{});
  dir(integral_constant<int, 2>{}, std::false_type{});
  dir(integral_constant<int, 3>{}, std::true_type{});
  dir(integral_constant<int, 3>{}, std::false_type{});
}
__device__ __forceinline__ double2 add(double2 a, double2 b) { return z2(a.x + b.x, a.y + b.y); }
__device__ __forceinline__ double2 sub(double2 a, double2 b) { return z2(a.x - b.x, a.y - b.y); }

inline bool fine_block(const Geom &g) { return g.Vb == 16 || g.Vb == 32; }
inline int fine_threads(const Geom &g) { return (6 * g.Vh + 31) / 32 * 32; }
// links, A_ee^-1, A_oo, two vectors, the exchange (u, a, b), reduction scratch
inline size_t fine_smem(const Geom &g) {
  return sizeof(double2) * ((size_t)36 * g.Vb + 72 * g.Vh + 24 * g.Vh + 18 * g.Vh) + sizeof(double) * 3 * 8;
}

// MULTI: the launch covers several lattice groups.
template <bool MULTI>
__global__ void __launch_bounds__(96) k_sap_fine(const SapGroups G, const RhsPtrs rp, const AuxPtrs ax, int colour,
                                                 int self_zero, int halo_zero, int mode, int nmr, int tile) {
  extern __shared__ __align__(16) unsigned char smem[];
  const int item = blockIdx.x, grp = MULTI ? sap_group_of(G, item) : 0;
  const Geom g = G.grp[grp].g;
  const int Vb = g.Vb, Vh = g.Vh;
  double2 *L = (double2 *)smem, *Ai = L + 36 * Vb, *Ao = Ai + 36 * Vh, *v0 = Ao + 36 * Vh, *v1 = v0 + 12 * Vh;
  double2 *X = v1 + 12 * Vh;   // [u 6][a 6][b 6][Vh]
  double *red = (double *)(X + 18 * Vh);
  const int nbc = g.nblocks / 2, loc = MULTI ? item - G.grp[grp].item0 : item;
  const int rhs0 = MULTI ? G.grp[grp].rhs0 : 0, nrhs = MULTI ? G.grp[grp].nrhs : rp.n;
  const int b = sap_block_of(g, colour, loc % nbc), rt = loc / nbc;
  const double2 *links = (const double2 *)G.grp[grp].links, *clov = (const double2 *)G.grp[grp].clov;

  // six threads per site; the threads past them repeat the last one's work and write nothing
  const bool act = (int)threadIdx.x < 6 * Vh;
  FineThread T;
  {
    const int t = act ? (int)threadIdx.x : 6 * Vh - 1;
    T.k = t / Vh;
    T.q = t - T.k * Vh;
    T.h = T.k / 3;
    T.c = T.k - 3 * T.h;
    T.sh = T.h ? -1.0 : 1.0;
#pragma unroll
    for (int j = 0; j < 6; j++) {
      const int i0 = j < T.k ? j : T.k, j0 = j < T.k ? T.k : j;
      T.off[j] = j == T.k ? T.k >> 1 : herm_off(i0, j0);
    }
  }
  for (int i = threadIdx.x; i < 36 * Vb; i += blockDim.x) L[i] = links[(size_t)b * 36 * Vb + i];
  for (int i = threadIdx.x; i < 36 * Vh; i += blockDim.x) {
    Ai[i] = ((const double2 *)G.grp[grp].cinv)[(size_t)b * 36 * Vh + i];
    const int r = i / Vh;
    Ao[i] = clov[((size_t)b * 36 + r) * Vb + Vh + (i - r * Vh)];
  }
  const Site se = decode(g, b, T.q), so = decode(g, b, Vh + T.q);
  int ne[8], no[8];   // in-block neighbours of the even and the odd site, (mu, forward / backward)
#pragma unroll
  for (int d = 0; d < 8; d++) {
    int nb, ns;
    float sg;
    bool inside;
    neighbour(g, se, d >> 1, d & 1 ? -1 : 1, &nb, &ns, &sg, &inside);
    ne[d] = inside ? ns - Vh : -1;
    neighbour(g, so, d >> 1, d & 1 ? -1 : 1, &nb, &ns, &sg, &inside);
    no[d] = inside ? ns : -1;
  }
  const int cu = T.k, cl = 6 + T.k;   // the thread's two components
  __syncthreads();
  for (int rr = 0; rr < tile; rr++) {
    if (rt * tile + rr >= nrhs) break;
    const int r = rhs0 + rt * tile + rr;
    double2 *x = (double2 *)rp.out[r] + (size_t)b * 12 * Vb;
    double2 reu = z2(0, 0), rel = z2(0, 0), rou, rol;   // the block residual: even and odd site, upper and lower
    if ((mode & SAP_INCR) && !(mode & SAP_FROM_B)) {
      const double2 *f = (const double2 *)ax.r[r] + (size_t)b * 12 * Vb + Vh + T.q;
      rou = f[cu * Vb];
      rol = f[cl * Vb];
    } else {
      const double2 *f = (const double2 *)rp.in[r] + (size_t)b * 12 * Vb + T.q;
      reu = f[cu * Vb];
      rel = f[cl * Vb];
      rou = f[cu * Vb + Vh];
      rol = f[cl * Vb + Vh];
    }
    const bool incr = mode & SAP_INCR;
    if (incr ? (mode & SAP_HALO_E) : !(self_zero && halo_zero)) {
      const double2 *f = incr ? (const double2 *)ax.e[r] : (const double2 *)rp.out[r];
      FineAcc e, o;
      fine_global(T, g, se, links, f, incr || self_zero, !incr && halo_zero, e);
      fine_global(T, g, so, links, f, incr || self_zero, !incr && halo_zero, o);
      if (!incr && !self_zero) {   // A x on the block's own sites
        const double2 *me = clov + (size_t)b * 36 * Vb + T.q, *mo = me + Vh, *xe = x + T.q, *xo = xe + Vh;
        e.u = add(e.u, fine_row(T, me, Vb, [&](int j) { return xe[j * Vb]; }));
        e.a = add(e.a, fine_row(T, me + 18 * Vb, Vb, [&](int j) { return xe[(6 + j) * Vb]; }));
        o.u = add(o.u, fine_row(T, mo, Vb, [&](int j) { return xo[j * Vb]; }));
        o.a = add(o.a, fine_row(T, mo + 18 * Vb, Vb, [&](int j) { return xo[(6 + j) * Vb]; }));
      }
      const int other = T.c + 3 * (1 - T.h);
      if (act) {
        X[other * Vh + T.q] = e.b;
        X[(6 + other) * Vh + T.q] = o.b;
      }
      __syncthreads();
      reu = sub(reu, e.u);
      rel = sub(rel, add(e.a, X[T.k * Vh + T.q]));
      rou = sub(rou, o.u);
      rol = sub(rol, add(o.a, X[(6 + T.k) * Vh + T.q]));
      __syncthreads();
    }
    // the sums of all threads of the sites to X; after the barrier row(j) is
    // component j of the upper, 6 + j of the lower spins
    auto share = [&](const FineAcc &o) {
      if (act) {
        X[T.k * Vh + T.q] = o.u;
        X[(6 + T.k) * Vh + T.q] = o.a;
        X[(12 + T.c + 3 * (1 - T.h)) * Vh + T.q] = o.b;
      }
      __syncthreads();
    };
    auto put = [&](double2 *v, double2 up, double2 lw) {
      if (act) {
        v[cu * Vh + T.q] = up;
        v[cl * Vh + T.q] = lw;
      }
    };
    // ---- te = A_ee^-1 r_e; rho = r_o - D_oe te; MR steps
    put(v0, reu, rel);
    __syncthreads();
    double2 eeu = fine_row(T, Ai + T.q, Vh, [&](int j) { return v0[j * Vh + T.q]; });
    double2 eel = fine_row(T, Ai + 18 * Vh + T.q, Vh, [&](int j) { return v0[(6 + j) * Vh + T.q]; });
    double2 eou = z2(0, 0), eol = z2(0, 0);
    __syncthreads();
    put(v0, eeu, eel);
    __syncthreads();
    FineAcc o;
    fine_inner(T, no, Vb, Vh, 1, v0, L, o);
    share(o);
    double2 rhu = sub(rou, o.u), rhl = sub(rol, add(o.a, X[(12 + T.k) * Vh + T.q]));
    put(v1, rhu, rhl);
    __syncthreads();
#pragma unroll 1
    for (int step = 0; step < nmr; step++) {
      fine_inner(T, ne, Vb, Vh, 0, v1, L, o);
      share(o);
      const double2 teu = fine_row(T, Ai + T.q, Vh, [&](int j) { return X[j * Vh + T.q]; });
      const double2 tel = fine_row(T, Ai + 18 * Vh + T.q, Vh, [&](int j) {
        return add(X[(6 + j) * Vh + T.q], X[(12 + j) * Vh + T.q]);
      });
      put(v0, teu, tel);
      __syncthreads();
      fine_inner(T, no, Vb, Vh, 1, v0, L, o);
      double2 pu = fine_row(T, Ao + T.q, Vh, [&](int j) { return v1[j * Vh + T.q]; });
      double2 pl = fine_row(T, Ao + 18 * Vh + T.q, Vh, [&](int j) { return v1[(6 + j) * Vh + T.q]; });
      share(o);
      pu = sub(pu, o.u);
      pl = sub(pl, add(o.a, X[(12 + T.k) * Vh + T.q]));
      double pr = 0, pi = 0, pp = 0;
      if (act) {
        pr = pu.x * rhu.x + pu.y * rhu.y + pl.x * rhl.x + pl.y * rhl.y;
        pi = pu.x * rhu.y - pu.y * rhu.x + pl.x * rhl.y - pl.y * rhl.x;
        pp = pu.x * pu.x + pu.y * pu.y + pl.x * pl.x + pl.y * pl.y;
      }
#pragma unroll
      for (int d = 16; d > 0; d >>= 1) {
        pr += __shfl_xor_sync(0xffffffffu, pr, d);
        pi += __shfl_xor_sync(0xffffffffu, pi, d);
        pp += __shfl_xor_sync(0xffffffffu, pp, d);
      }
      const int w = threadIdx.x >> 5, nw = blockDim.x >> 5;
      if ((threadIdx.x & 31) == 0) {
        red[w] = pr;
        red[8 + w] = pi;
        red[16 + w] = pp;
      }
      __syncthreads();
      pr = pi = pp = 0;
      for (int i = 0; i < nw; i++) {
        pr += red[i];
        pi += red[8 + i];
        pp += red[16 + i];
      }
      double ar = 0, ai = 0;
      if (pp > 0) {
        ar = pr / pp;
        ai = pi / pp;
      }
      auto mac = [&](double2 &y, double s, double2 v) {   // y += s alpha v
        y.x += s * (ar * v.x - ai * v.y);
        y.y += s * (ar * v.y + ai * v.x);
      };
      mac(eou, 1, rhu);
      mac(eol, 1, rhl);
      mac(eeu, -1, teu);
      mac(eel, -1, tel);
      mac(rhu, -1, pu);
      mac(rhl, -1, pl);
      put(v1, rhu, rhl);
      __syncthreads();
    }
    // ---- x += e, the correction and the residual for the next phases
    if (act) {
      auto at = [&](int c, int s) { return (size_t)c * Vb + s; };
      if (mode & SAP_WRITE_E) {
        double2 *f = (double2 *)ax.e[r] + (size_t)b * 12 * Vb;
        f[at(cu, T.q)] = eeu;
        f[at(cl, T.q)] = eel;
        f[at(cu, Vh + T.q)] = eou;
        f[at(cl, Vh + T.q)] = eol;
      }
      if (mode & SAP_WRITE_R) {
        double2 *f = (double2 *)ax.r[r] + (size_t)b * 12 * Vb;
        f[at(cu, Vh + T.q)] = rhu;
        f[at(cl, Vh + T.q)] = rhl;
      }
      auto update = [&](int c, int s, double2 e) { x[at(c, s)] = self_zero ? e : add(x[at(c, s)], e); };
      update(cu, T.q, eeu);
      update(cl, T.q, eel);
      update(cu, Vh + T.q, eou);
      update(cl, Vh + T.q, eol);
    }
    __syncthreads();   // the shared vectors are reused by the next right-hand side
  }
}

}  // namespace
}  // namespace dd
