// Schwarz colour phase for blocks of 16 and 32 sites in FP64 (the 2^4 block of
// the plain method), twelve threads per site. The method and the residual modes
// are those of k_sap_phase.
//
// Why. k_sap_phase gives a 2^4 block one half-filled warp that runs ~700 FP64
// instructions per half-step, 64 clocks each: a phase on 4^4 (8 blocks) took
// 340 us with one of four sub-partitions of 8 SMs at work. Here a thread (see
// dd_fine.cuh) runs ~90 per half-step. In a direction of extent 2 a site has
// one neighbour in the block, forward or backward: both kinds run as one hop,
// its direction a sign and a choice of link entries. The phase: 43 us, still the
// FP64 issue rate of one thread's chain (2 x 3 MR half-steps and the first and
// last ones).
//
// The even sites' correction is accumulated over the MR steps (e_e = te_0 -
// sum_k alpha_k te_k with te = A_ee^-1 D_eo rho), which saves the last
// half-step. The block's links, A_oo and A_ee^-1 are copied to shared memory.
#pragma once
#include "dd_fine.cuh"
#include "dd_sap_kernels.cuh"

namespace dd {
namespace {

// hops inside the block into the thread's site of parity p (local coordinates
// lc), from the shared vector v of the other parity; nb: its in-block
// neighbours in the directions {2d, 2d+1} (forward, backward; -1: outside)
template <int MU>
__device__ __forceinline__ void fine_inner_dir(const FineThread &T, const Geom &g, const int *nb, int p,
                                               const double2 *v, const double2 *L, FineAcc &o) {
  const int Vb = g.Vb, Vh = g.Vh;
  auto one = [&](bool fwd, int n) {
    const double2 *w = L + 9 * MU * Vb + (fwd ? p * Vh + T.q : (1 - p) * Vh + n);
    fine_hop<MU>(T, fwd, -0.5, [&](int i) { return v[i * Vh + n]; }, [&](int i) { return w[i * Vb]; }, o);
  };
  const int f = nb[2 * (MU & 1)], b = nb[2 * (MU & 1) + 1];
  if (g.bd[MU] == 2) {   // exactly one of the two
    one(f >= 0, f >= 0 ? f : b);
  } else {
    if (f >= 0) one(true, f);
    if (b >= 0) one(false, b);
  }
}
__device__ __forceinline__ void fine_inner(const FineThread &T, const Geom &g, const int *nb, int p, const double2 *v,
                                           const double2 *L, FineAcc &o) {
  o.u = o.l = z2(0, 0);
  if (T.d == 0) {
    fine_inner_dir<0>(T, g, nb, p, v, L, o);
    fine_inner_dir<1>(T, g, nb, p, v, L, o);
  } else {
    fine_inner_dir<2>(T, g, nb, p, v, L, o);
    fine_inner_dir<3>(T, g, nb, p, v, L, o);
  }
}
inline bool fine_block(const Geom &g) { return g.Vb == 16 || g.Vb == 32; }
inline int fine_threads(const Geom &g) { return 2 * ((6 * g.Vh + 31) / 32 * 32); }   // the halves d in whole warps
// links, A_ee^-1, A_oo, two vectors, the exchange of the sums, reduction scratch
inline size_t fine_smem(const Geom &g) {
  return sizeof(double2) * ((size_t)36 * g.Vb + 72 * g.Vh + 24 * g.Vh + 24 * g.Vh) + sizeof(double) * 3 * 8;
}

// MULTI: the launch covers several lattice groups.
template <bool MULTI>
__global__ void __launch_bounds__(192) k_sap_fine(const SapGroups G, const RhsPtrs rp, const AuxPtrs ax, int colour,
                                                  int self_zero, int halo_zero, int mode, int nmr, int tile) {
  extern __shared__ __align__(16) unsigned char smem[];
  const int item = blockIdx.x, grp = MULTI ? sap_group_of(G, item) : 0;
  const Geom g = G.grp[grp].g;
  const int Vb = g.Vb, Vh = g.Vh;
  double2 *L = (double2 *)smem, *Ai = L + 36 * Vb, *Ao = Ai + 36 * Vh, *v0 = Ao + 36 * Vh, *v1 = v0 + 12 * Vh;
  double2 *X = v1 + 12 * Vh;   // [upper: half 0, half 1; lower: half 0, half 1][6][Vh]
  double *red = (double *)(X + 24 * Vh);
  const int nbc = g.nblocks / 2, loc = MULTI ? item - G.grp[grp].item0 : item;
  const int rhs0 = MULTI ? G.grp[grp].rhs0 : 0, nrhs = MULTI ? G.grp[grp].nrhs : rp.n;
  const int b = sap_block_of(g, colour, loc % nbc), rt = loc / nbc;
  const double2 *links = (const double2 *)G.grp[grp].links, *clov = (const double2 *)G.grp[grp].clov;

  // the threads of a half past its 6 Vh repeat the last one's work and write nothing
  FineThread T;
  bool act;
  {
    const int half = blockDim.x / 2;
    T.d = (int)threadIdx.x >= half;
    int t = (int)threadIdx.x - T.d * half;
    act = t < 6 * Vh;
    if (!act) t = 6 * Vh - 1;
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
  int ne[4], no[4];   // in-block neighbours of the even and the odd site in the thread's directions
#pragma unroll
  for (int e = 0; e < 4; e++) {
    auto at = [&](const Site &t, int mu) {
      int nb, ns;
      float sg;
      bool inside;
      neighbour(g, t, mu, e & 1 ? -1 : 1, &nb, &ns, &sg, &inside);
      return inside ? ns - (t.p ? 0 : Vh) : -1;
    };
    ne[e] = T.d ? at(se, 2 + (e >> 1)) : at(se, e >> 1);
    no[e] = T.d ? at(so, 2 + (e >> 1)) : at(so, e >> 1);
  }
  // the thread's component of a site (chirality d), its row's blocks, and where its sums go
  const int cc = 6 * T.d + T.k;
  const double2 *mi = Ai + 18 * T.d * Vh + T.q, *mo = Ao + 18 * T.d * Vh + T.q;
  const int lk = T.d ? T.k : T.c + 3 * (1 - T.h);   // lower component of o.l
  const double2 *Xd = X + 12 * T.d * Vh + T.q;      // component j of the thread's chirality: Xd[j Vh] + Xd[(6 + j) Vh]
  __syncthreads();
  for (int rr = 0; rr < tile; rr++) {
    if (rt * tile + rr >= nrhs) break;
    const int r = rhs0 + rt * tile + rr;
    double2 *x = (double2 *)rp.out[r] + (size_t)b * 12 * Vb;
    double2 re = z2(0, 0), ro;   // the block residual at the even and the odd site
    if ((mode & SAP_INCR) && !(mode & SAP_FROM_B)) {
      ro = ((const double2 *)ax.r[r] + (size_t)b * 12 * Vb)[cc * Vb + Vh + T.q];
    } else {
      const double2 *f = (const double2 *)rp.in[r] + (size_t)b * 12 * Vb + cc * Vb + T.q;
      re = f[0];
      ro = f[Vh];
    }
    // the hops' sums of all threads to X
    auto share = [&](const FineAcc &o) {
      if (act) {
        X[(6 * T.d + T.k) * Vh + T.q] = o.u;
        X[(12 + 6 * T.d + lk) * Vh + T.q] = o.l;
      }
      __syncthreads();
    };
    auto own = [&] { return add(Xd[T.k * Vh], Xd[(6 + T.k) * Vh]); };
    auto put = [&](double2 *v, double2 a) {
      if (act) v[cc * Vh + T.q] = a;
    };
    const bool incr = mode & SAP_INCR;
    if (incr ? (mode & SAP_HALO_E) : !(self_zero && halo_zero)) {
      const double2 *f = incr ? (const double2 *)ax.e[r] : (const double2 *)rp.out[r];
      FineAcc e, o;
      fine_global(T, g, se, links, f, incr || self_zero, !incr && halo_zero, e);
      fine_global(T, g, so, links, f, incr || self_zero, !incr && halo_zero, o);
      share(e);
      re = sub(re, own());
      __syncthreads();
      share(o);
      ro = sub(ro, own());
      if (!incr && !self_zero) {   // A x on the block's own sites
        const double2 *m = clov + ((size_t)b * 36 + 18 * T.d) * Vb + T.q, *xs = x + 6 * T.d * Vb + T.q;
        re = sub(re, fine_row(T, m, Vb, [&](int j) { return xs[j * Vb]; }));
        ro = sub(ro, fine_row(T, m + Vh, Vb, [&](int j) { return xs[j * Vb + Vh]; }));
      }
      __syncthreads();
    }
    // ---- te = A_ee^-1 r_e; rho = r_o - D_oe te; MR steps
    const double2 *v0d = v0 + 6 * T.d * Vh + T.q, *v1d = v1 + 6 * T.d * Vh + T.q;
    put(v0, re);
    __syncthreads();
    double2 ee = fine_row(T, mi, Vh, [&](int j) { return v0d[j * Vh]; }), eo = z2(0, 0);
    __syncthreads();
    put(v0, ee);
    __syncthreads();
    FineAcc o;
    fine_inner(T, g, no, 1, v0, L, o);
    share(o);
    double2 rh = sub(ro, own());
    put(v1, rh);
    __syncthreads();
#pragma unroll 1
    for (int step = 0; step < nmr; step++) {
      fine_inner(T, g, ne, 0, v1, L, o);
      share(o);
      const double2 te = fine_row(T, mi, Vh, [&](int j) { return add(Xd[j * Vh], Xd[(6 + j) * Vh]); });
      put(v0, te);
      __syncthreads();
      fine_inner(T, g, no, 1, v0, L, o);
      double2 p = fine_row(T, mo, Vh, [&](int j) { return v1d[j * Vh]; });
      share(o);
      p = sub(p, own());
      double pr = 0, pi = 0, pp = 0;
      if (act) {
        pr = p.x * rh.x + p.y * rh.y;
        pi = p.x * rh.y - p.y * rh.x;
        pp = p.x * p.x + p.y * p.y;
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
      mac(eo, 1, rh);
      mac(ee, -1, te);
      mac(rh, -1, p);
      put(v1, rh);
      __syncthreads();
    }
    // ---- x += e, the correction and the residual for the next phases
    if (act) {
      const size_t at = (size_t)cc * Vb + T.q;
      if (mode & SAP_WRITE_E) {
        double2 *f = (double2 *)ax.e[r] + (size_t)b * 12 * Vb;
        f[at] = ee;
        f[at + Vh] = eo;
      }
      if (mode & SAP_WRITE_R) ((double2 *)ax.r[r] + (size_t)b * 12 * Vb)[at + Vh] = rh;
      x[at] = self_zero ? ee : add(x[at], ee);
      x[at + Vh] = self_zero ? eo : add(x[at + Vh], eo);
    }
    __syncthreads();   // the shared vectors are reused by the next right-hand side
  }
}

}  // namespace
}  // namespace dd
