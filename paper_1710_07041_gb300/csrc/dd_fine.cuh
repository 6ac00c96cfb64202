// FP64 operator arithmetic with twelve threads per site, for lattices and
// blocks too small to fill the chip with one or two (dd_sap_fine.cuh and the
// small-lattice FP64 Dslash). GB300 issues one FP64 instruction of a warp in
// about 64 clocks per SM sub-partition whatever the number of active lanes, so
// a small case takes (instructions per thread) x 64 clocks: the work of a site
// is cut into threads. Thread (spin component h, colour c, half d) computes one
// colour of one spin component of the projected hops in the directions {2d,
// 2d+1}, and row 3h + c of chirality block d; the two halves are in different
// warps. The projections are formed three times over (each by the threads of
// its three colours).
#pragma once
#include "dd_internal.cuh"

namespace dd {
namespace {

struct FineThread {
  int h, c, k, q, d;  // spin, colour, 3 h + c, site of either parity, half: directions and chirality
  int off[6];         // pair of entry (k, j) in a packed Hermitian block
  double sh;          // +1 (h = 0), -1 (h = 1)
};
__device__ __forceinline__ double2 z2(double x, double y) { return make_double2(x, y); }

// the sums of a thread, colour c: upper spin h (u); lower spin h (d = 1: z, t)
// or 1 - h (d = 0: x, y)
struct FineAcc {
  double2 u, l;
};
// v with its sign flipped unless pos (an integer operation)
__device__ __forceinline__ double signed_by(bool pos, double v) {
  return pos ? v : __hiloint2double(__double2hiint(v) ^ (int)0x80000000, __double2loint(v));
}

// one hop, forward (fwd) or backward: v(i) the source's component i, w(i) the
// link's entry i; s = -1/2 times the boundary sign
template <int MU, typename V, typename W>
__device__ __forceinline__ void fine_hop(const FineThread &T, bool fwd, double s, V v, W w, FineAcc &o) {
  const int du = MU < 2 ? 9 - 3 * T.h : 6 + 3 * T.h;   // first colour of the lower spin projected on
  // chi = u + f d (MU 1, 3) or u + i f d (MU 0, 2)
  const double f = signed_by(MU == 3 ? !fwd : fwd, MU == 1 || MU == 2 ? T.sh : 1.0);
  double2 y = z2(0, 0);
#pragma unroll
  for (int k = 0; k < 3; k++) {
    const double2 up = v(3 * T.h + k), d = v(du + k), m = w(fwd ? 3 * T.c + k : 3 * k + T.c);
    const double2 x = (MU == 0 || MU == 2) ? z2(fma(-f, d.y, up.x), fma(f, d.x, up.y))
                                           : z2(fma(f, d.x, up.x), fma(f, d.y, up.y));
    const double mi = signed_by(fwd, m.y);   // U chi or U^dagger chi
    y.x = fma(m.x, x.x, y.x);
    y.x = fma(-mi, x.y, y.x);
    y.y = fma(m.x, x.y, y.y);
    y.y = fma(mi, x.x, y.y);
  }
  o.u.x = fma(s, y.x, o.u.x);
  o.u.y = fma(s, y.y, o.u.y);
  // the lower spin takes the conjugate phase of chi's
  const double fs = signed_by(f > 0, s);
  if constexpr (MU == 0 || MU == 2) {
    o.l.x = fma(fs, y.y, o.l.x);
    o.l.y = fma(-fs, y.x, o.l.y);
  } else {
    o.l.x = fma(fs, y.x, o.l.x);
    o.l.y = fma(fs, y.y, o.l.y);
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

// hops into site t from the global field x: from neighbours inside the block
// unless self_zero, outside unless halo_zero
template <int MU>
__device__ __forceinline__ void fine_global_dir(const FineThread &T, const Geom &g, const Site &t, const double2 *links,
                                                const double2 *x, bool self_zero, bool halo_zero, FineAcc &o) {
  int nb[2], ns[2];
  float sg[2];
  bool on[2];
#pragma unroll
  for (int e = 0; e < 2; e++) {
    bool inside;
    neighbour(g, t, MU, e ? -1 : 1, &nb[e], &ns[e], &sg[e], &inside);
    on[e] = !(inside ? self_zero : halo_zero);
  }
  auto one = [&](bool fwd, int b, int s, float sign) {
    DD_CHECK_INDEX(b, g.nblocks);
    DD_CHECK_INDEX(s, g.Vb);
    const double2 *v = x + (size_t)b * 12 * g.Vb + s;
    const double2 *w = links + ((size_t)(fwd ? t.b : b) * 36 + 9 * MU) * g.Vb + (fwd ? t.s : s);
    fine_hop<MU>(T, fwd, -0.5 * sign, [&](int i) { return v[(size_t)i * g.Vb]; },
                 [&](int i) { return w[(size_t)i * g.Vb]; }, o);
  };
  if (g.bd[MU] == 2 && on[0] != on[1]) {   // one hop, whichever it is
    one(on[0], on[0] ? nb[0] : nb[1], on[0] ? ns[0] : ns[1], on[0] ? sg[0] : sg[1]);
  } else {
    if (on[0]) one(true, nb[0], ns[0], sg[0]);
    if (on[1]) one(false, nb[1], ns[1], sg[1]);
  }
}
__device__ __forceinline__ void fine_global(const FineThread &T, const Geom &g, const Site &t, const double2 *links,
                                            const double2 *x, bool self_zero, bool halo_zero, FineAcc &o) {
  o.u = o.l = z2(0, 0);
  if (T.d == 0) {
    fine_global_dir<0>(T, g, t, links, x, self_zero, halo_zero, o);
    fine_global_dir<1>(T, g, t, links, x, self_zero, halo_zero, o);
  } else {
    fine_global_dir<2>(T, g, t, links, x, self_zero, halo_zero, o);
    fine_global_dir<3>(T, g, t, links, x, self_zero, halo_zero, o);
  }
}
__device__ __forceinline__ double2 add(double2 a, double2 b) { return z2(a.x + b.x, a.y + b.y); }
__device__ __forceinline__ double2 sub(double2 a, double2 b) { return z2(a.x - b.x, a.y - b.y); }

}  // namespace
}  // namespace dd
