// Schwarz colour phase for the 4^4 and 8 x 4^3 blocks in 32- and 16-bit
// storage (FP32 arithmetic), two lattice sites per thread in packed
// arithmetic. The method is the one of dd_sap.cu; this file holds the layout.
//
// Packing. GB300 runs FP32 multiply-adds at 128 per SM and clock whether they
// are issued singly or as pairs (fma.rn.f32x2: measured 117 and 124 of 128),
// but a pair takes one issue slot for both, so loads, address arithmetic and
// selects no longer compete with the arithmetic (one integer instruction per
// two multiply-adds cost the single form two thirds of its rate, the packed
// form nothing). The pair is two sites of one x-row of the block: a row
// (y, z, t) has four sites, two of each parity, at x = s and s + 2 ("A" and
// "B"), neighbours in storage. Hops along y, z, t connect A with A and B with
// B. Along x, of the three links inside a row two connect A with A and B with
// B (one packed hop) and one connects A with B (one single hop on the one
// site it reaches): no lane computes a hop that leaves the block in x.
//
// Threads: two per row, thread half h = lane % 2. Half h carries the spin
// component h of every projected hop (three colours), so both halves run the
// same code and read the same link (neighbouring lanes, so that one
// shared-memory wavefront serves both: with the halves 16 lanes apart each
// took its own, measured 4 against 2 wavefronts per 16-byte load),
// and owns chirality block h (spins 2h, 2h+1) of the vectors. After the hops
// one exchange by shuffles turns "spin h" into "chirality h": no shared
// exchange buffer and no barrier. A warp holds 16 rows of one t, so hops that
// leave the block in t are skipped by the whole warp.
//
// Where the operands live, per block of 256 sites: all links as packed pairs
// in shared memory (72 KB, bulk-copied for FP32 storage), both parities' MR
// vectors (24 KB); in tensor memory, per thread, its four clover blocks
// (2 x 72 words) and its row's x-links in the orientation each half-step
// needs (2 x 54 words): 252 of 256 columns. Two CTAs of 128 threads per SM.
//
// The links in shared memory are times -1/2, the hop's coefficient (in the
// operator field as paired_scale says).
//
// Bound and figures (profiles/k_sap_pair_clocks.md). A CTA of FP32 64x32^3 lives
// 55400 clocks at 4 MR steps: 37800 in the half-steps (three quarters of what the
// register ports allow a stream of packed multiply-adds with three distinct
// operands), 5400 taking in residual and flux, 4800 sending the flux, 1500 on x,
// the rest staging. Per phase, general kernel (clover blocks in tensor memory,
// one site pair per two threads) -> this one: 64x32^3 FP32 0.514 -> 0.370 ms; FP16
// 48x24^3 with 12 right-hand sides 1.62 -> 1.26 ms; 16x8^3 FP32, where it is the
// latency of one block, 24.3 -> 19.5 us.
#pragma once
#include "dd_sap_kernels.cuh"

namespace dd {

// SAP_FROM_B with the right-hand side given as an FP32 field (the residual
// b - D x of a given first iterate)
enum { SAP_B32 = 32 };

namespace {

using u64 = unsigned long long;   // two FP32 values: site A in the low word, B in the high
typedef ulonglong2 quad;          // one complex number of both sites: {re A, re B}, {im A, im B}

__device__ __forceinline__ u64 pk(float a, float b) {
  u64 r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
  return r;
}
__device__ __forceinline__ float lo(u64 v) { return __uint_as_float((uint32_t)v); }
__device__ __forceinline__ float hi(u64 v) { return __uint_as_float((uint32_t)(v >> 32)); }
__device__ __forceinline__ u64 fma2(u64 a, u64 b, u64 c) {
  u64 d;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
  return d;
}
__device__ __forceinline__ u64 mul2(u64 a, u64 b) {
  u64 d;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
  return d;
}
__device__ __forceinline__ u64 add2(u64 a, u64 b) {
  u64 d;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
  return d;
}
__device__ __forceinline__ u64 sub2(u64 a, u64 b) {
  u64 d;
  asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
  return d;
}
// (the two sign flips fold into the operands of the instruction that uses them)
__device__ __forceinline__ u64 neg2(u64 a) { return pk(-lo(a), -hi(a)); }
__device__ __forceinline__ u64 sel2(bool c, u64 a, u64 b) { return c ? a : b; }
__device__ __forceinline__ u64 shfl2(u64 v) {   // the other half's value
  return pk(__shfl_xor_sync(0xffffffffu, lo(v), 1), __shfl_xor_sync(0xffffffffu, hi(v), 1));
}

// geometry of the two shapes: BT sites in t, rows (y, z, t), threads
template <int SHAPE> struct PairGeom {
  static constexpr int BT = SHAPE == 2 ? 8 : 4;
  static constexpr int ROWS = 16 * BT, NT = 2 * ROWS, VH = 2 * ROWS, VB = 4 * ROWS;
  static constexpr int TCOLS = 2 * NT;   // TMEM columns (256 per 128 threads)
  // shared memory: links, two vectors (first: the incoming flux), reduction
  // scratch, two barriers, TMEM address
  static constexpr int LINKS = 36 * 2 * ROWS, VEC = 12 * ROWS;   // in quads
  static constexpr size_t SMEM = (size_t)(LINKS + 2 * VEC) * 16 + 3 * 8 * 4 + 32;
};

// ---- tensor memory: N words of this thread's lane from column taddr
template <int N> __device__ __forceinline__ void tm_st(uint32_t a, const uint32_t *u) {
  static_assert(N == 2 || N == 4 || N == 8 || N == 16 || N == 32, "tcgen05.st width");
  __syncwarp();
  if constexpr (N == 2) {
    asm volatile("tcgen05.st.sync.aligned.32x32b.x2.b32 [%0], {%1, %2};\n" ::"r"(a), "r"(u[0]), "r"(u[1]) : "memory");
  } else if constexpr (N == 4) {
    asm volatile("tcgen05.st.sync.aligned.32x32b.x4.b32 [%0], {%1, %2, %3, %4};\n" ::"r"(a), "r"(u[0]), "r"(u[1]),
                 "r"(u[2]), "r"(u[3])
                 : "memory");
  } else if constexpr (N == 8) {
    asm volatile("tcgen05.st.sync.aligned.32x32b.x8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};\n" ::"r"(a), "r"(u[0]),
                 "r"(u[1]), "r"(u[2]), "r"(u[3]), "r"(u[4]), "r"(u[5]), "r"(u[6]), "r"(u[7])
                 : "memory");
  } else if constexpr (N == 16) {
    asm volatile(
        "tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, "
        "%15, %16};\n" ::"r"(a),
        "r"(u[0]), "r"(u[1]), "r"(u[2]), "r"(u[3]), "r"(u[4]), "r"(u[5]), "r"(u[6]), "r"(u[7]), "r"(u[8]), "r"(u[9]),
        "r"(u[10]), "r"(u[11]), "r"(u[12]), "r"(u[13]), "r"(u[14]), "r"(u[15])
        : "memory");
  } else {
    asm volatile(
        "tcgen05.st.sync.aligned.32x32b.x32.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, "
        "%15, %16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31, %32};\n" ::"r"(a),
        "r"(u[0]), "r"(u[1]), "r"(u[2]), "r"(u[3]), "r"(u[4]), "r"(u[5]), "r"(u[6]), "r"(u[7]), "r"(u[8]), "r"(u[9]),
        "r"(u[10]), "r"(u[11]), "r"(u[12]), "r"(u[13]), "r"(u[14]), "r"(u[15]), "r"(u[16]), "r"(u[17]), "r"(u[18]),
        "r"(u[19]), "r"(u[20]), "r"(u[21]), "r"(u[22]), "r"(u[23]), "r"(u[24]), "r"(u[25]), "r"(u[26]), "r"(u[27]),
        "r"(u[28]), "r"(u[29]), "r"(u[30]), "r"(u[31])
        : "memory");
  }
}
// N words of this thread's lane, loaded asynchronously: the registers are
// defined only after tm_wait on the same array, so a load can be issued ahead
// of a barrier or the shuffles before its use.
__device__ __forceinline__ void tm_issue72(uint32_t a, uint32_t *u) {   // a packed clover block
  __syncwarp();
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x32.b32 {"
      "%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, %16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31"
      "}, [%72];\n"
      "tcgen05.ld.sync.aligned.32x32b.x32.b32 {"
      "%32, %33, %34, %35, %36, %37, %38, %39, %40, %41, %42, %43, %44, %45, %46, %47, %48, %49, %50, %51, %52, %53, %54, %55, %56, %57, %58, %59, %60, %61, %62, %63"
      "}, [%73];\n"
      "tcgen05.ld.sync.aligned.32x32b.x8.b32 {"
      "%64, %65, %66, %67, %68, %69, %70, %71"
      "}, [%74];\n"
      : "=r"(u[0]), "=r"(u[1]), "=r"(u[2]), "=r"(u[3]), "=r"(u[4]), "=r"(u[5]), "=r"(u[6]), "=r"(u[7]), "=r"(u[8]),
        "=r"(u[9]), "=r"(u[10]), "=r"(u[11]), "=r"(u[12]), "=r"(u[13]), "=r"(u[14]), "=r"(u[15]), "=r"(u[16]),
        "=r"(u[17]), "=r"(u[18]), "=r"(u[19]), "=r"(u[20]), "=r"(u[21]), "=r"(u[22]), "=r"(u[23]), "=r"(u[24]),
        "=r"(u[25]), "=r"(u[26]), "=r"(u[27]), "=r"(u[28]), "=r"(u[29]), "=r"(u[30]), "=r"(u[31]), "=r"(u[32]),
        "=r"(u[33]), "=r"(u[34]), "=r"(u[35]), "=r"(u[36]), "=r"(u[37]), "=r"(u[38]), "=r"(u[39]), "=r"(u[40]),
        "=r"(u[41]), "=r"(u[42]), "=r"(u[43]), "=r"(u[44]), "=r"(u[45]), "=r"(u[46]), "=r"(u[47]), "=r"(u[48]),
        "=r"(u[49]), "=r"(u[50]), "=r"(u[51]), "=r"(u[52]), "=r"(u[53]), "=r"(u[54]), "=r"(u[55]), "=r"(u[56]),
        "=r"(u[57]), "=r"(u[58]), "=r"(u[59]), "=r"(u[60]), "=r"(u[61]), "=r"(u[62]), "=r"(u[63]), "=r"(u[64]),
        "=r"(u[65]), "=r"(u[66]), "=r"(u[67]), "=r"(u[68]), "=r"(u[69]), "=r"(u[70]), "=r"(u[71])
      : "r"(a), "r"(a + 32), "r"(a + 64)
      : "memory");
}
__device__ __forceinline__ void tm_issue54(uint32_t a, uint32_t *u) {   // a row's packed (36) and single (18) x-link
  __syncwarp();
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x32.b32 {"
      "%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, %16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31"
      "}, [%54];\n"
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 {"
      "%32, %33, %34, %35, %36, %37, %38, %39, %40, %41, %42, %43, %44, %45, %46, %47"
      "}, [%55];\n"
      "tcgen05.ld.sync.aligned.32x32b.x4.b32 {"
      "%48, %49, %50, %51"
      "}, [%56];\n"
      "tcgen05.ld.sync.aligned.32x32b.x2.b32 {"
      "%52, %53"
      "}, [%57];\n"
      : "=r"(u[0]), "=r"(u[1]), "=r"(u[2]), "=r"(u[3]), "=r"(u[4]), "=r"(u[5]), "=r"(u[6]), "=r"(u[7]), "=r"(u[8]),
        "=r"(u[9]), "=r"(u[10]), "=r"(u[11]), "=r"(u[12]), "=r"(u[13]), "=r"(u[14]), "=r"(u[15]), "=r"(u[16]),
        "=r"(u[17]), "=r"(u[18]), "=r"(u[19]), "=r"(u[20]), "=r"(u[21]), "=r"(u[22]), "=r"(u[23]), "=r"(u[24]),
        "=r"(u[25]), "=r"(u[26]), "=r"(u[27]), "=r"(u[28]), "=r"(u[29]), "=r"(u[30]), "=r"(u[31]), "=r"(u[32]),
        "=r"(u[33]), "=r"(u[34]), "=r"(u[35]), "=r"(u[36]), "=r"(u[37]), "=r"(u[38]), "=r"(u[39]), "=r"(u[40]),
        "=r"(u[41]), "=r"(u[42]), "=r"(u[43]), "=r"(u[44]), "=r"(u[45]), "=r"(u[46]), "=r"(u[47]), "=r"(u[48]),
        "=r"(u[49]), "=r"(u[50]), "=r"(u[51]), "=r"(u[52]), "=r"(u[53])
      : "r"(a), "r"(a + 32), "r"(a + 48), "r"(a + 52)
      : "memory");
}
__device__ __forceinline__ void tm_wait72(uint32_t *u) {
  __syncwarp();
  asm volatile("tcgen05.wait::ld.sync.aligned;\n"
      : "+r"(u[0]), "+r"(u[1]), "+r"(u[2]), "+r"(u[3]), "+r"(u[4]), "+r"(u[5]), "+r"(u[6]), "+r"(u[7]), "+r"(u[8]),
        "+r"(u[9]), "+r"(u[10]), "+r"(u[11]), "+r"(u[12]), "+r"(u[13]), "+r"(u[14]), "+r"(u[15]), "+r"(u[16]),
        "+r"(u[17]), "+r"(u[18]), "+r"(u[19]), "+r"(u[20]), "+r"(u[21]), "+r"(u[22]), "+r"(u[23]), "+r"(u[24]),
        "+r"(u[25]), "+r"(u[26]), "+r"(u[27]), "+r"(u[28]), "+r"(u[29]), "+r"(u[30]), "+r"(u[31]), "+r"(u[32]),
        "+r"(u[33]), "+r"(u[34]), "+r"(u[35]), "+r"(u[36]), "+r"(u[37]), "+r"(u[38]), "+r"(u[39]), "+r"(u[40]),
        "+r"(u[41]), "+r"(u[42]), "+r"(u[43]), "+r"(u[44]), "+r"(u[45]), "+r"(u[46]), "+r"(u[47]), "+r"(u[48]),
        "+r"(u[49]), "+r"(u[50]), "+r"(u[51]), "+r"(u[52]), "+r"(u[53]), "+r"(u[54]), "+r"(u[55]), "+r"(u[56]),
        "+r"(u[57]), "+r"(u[58]), "+r"(u[59]), "+r"(u[60]), "+r"(u[61]), "+r"(u[62]), "+r"(u[63]), "+r"(u[64]),
        "+r"(u[65]), "+r"(u[66]), "+r"(u[67]), "+r"(u[68]), "+r"(u[69]), "+r"(u[70]), "+r"(u[71])
      :
      : "memory");
}
__device__ __forceinline__ void tm_wait54(uint32_t *u) {
  __syncwarp();
  asm volatile("tcgen05.wait::ld.sync.aligned;\n"
      : "+r"(u[0]), "+r"(u[1]), "+r"(u[2]), "+r"(u[3]), "+r"(u[4]), "+r"(u[5]), "+r"(u[6]), "+r"(u[7]), "+r"(u[8]),
        "+r"(u[9]), "+r"(u[10]), "+r"(u[11]), "+r"(u[12]), "+r"(u[13]), "+r"(u[14]), "+r"(u[15]), "+r"(u[16]),
        "+r"(u[17]), "+r"(u[18]), "+r"(u[19]), "+r"(u[20]), "+r"(u[21]), "+r"(u[22]), "+r"(u[23]), "+r"(u[24]),
        "+r"(u[25]), "+r"(u[26]), "+r"(u[27]), "+r"(u[28]), "+r"(u[29]), "+r"(u[30]), "+r"(u[31]), "+r"(u[32]),
        "+r"(u[33]), "+r"(u[34]), "+r"(u[35]), "+r"(u[36]), "+r"(u[37]), "+r"(u[38]), "+r"(u[39]), "+r"(u[40]),
        "+r"(u[41]), "+r"(u[42]), "+r"(u[43]), "+r"(u[44]), "+r"(u[45]), "+r"(u[46]), "+r"(u[47]), "+r"(u[48]),
        "+r"(u[49]), "+r"(u[50]), "+r"(u[51]), "+r"(u[52]), "+r"(u[53])
      :
      : "memory");
}
__device__ __forceinline__ u64 word2(const uint32_t *u, int i) {   // packed real i
  return pk(__uint_as_float(u[2 * i]), __uint_as_float(u[2 * i + 1]));
}

// ---- arithmetic on one spin component (three colours: re, im in turn)
// hv = W chi and hv = W^dagger chi, W's entry (r, k) at L[(3 r + k) * stride].
// The column loop is outermost: six independent chains, so that consecutive
// multiply-adds do not wait for one another.
template <bool DAG>
__device__ __forceinline__ void su3_pair(const quad *L, int stride, const u64 *c, u64 *hv) {
#pragma unroll
  for (int k = 0; k < 3; k++) {
    const u64 n = neg2(DAG ? c[2 * k] : c[2 * k + 1]);   // the negated part: -im (W), -re (W^dagger)
    quad u[3];
#pragma unroll
    for (int r = 0; r < 3; r++) u[r] = L[(DAG ? 3 * k + r : 3 * r + k) * stride];
#pragma unroll
    for (int r = 0; r < 3; r++) {
      hv[2 * r] = k ? fma2(u[r].x, c[2 * k], hv[2 * r]) : mul2(u[r].x, c[0]);
      hv[2 * r + 1] = k ? fma2(u[r].x, c[2 * k + 1], hv[2 * r + 1]) : mul2(u[r].x, c[1]);
    }
#pragma unroll
    for (int r = 0; r < 3; r++) {
      hv[2 * r] = fma2(u[r].y, DAG ? c[2 * k + 1] : n, hv[2 * r]);
      hv[2 * r + 1] = fma2(u[r].y, DAG ? n : c[2 * k], hv[2 * r + 1]);
    }
  }
}
// the same for W in registers, packed and single
__device__ __forceinline__ void su3_reg(const u64 *W, const u64 *c, u64 *hv) {
#pragma unroll
  for (int k = 0; k < 3; k++) {
    const u64 n = neg2(c[2 * k + 1]);
#pragma unroll
    for (int r = 0; r < 3; r++) {
      const u64 ur = W[2 * (3 * r + k)];
      hv[2 * r] = k ? fma2(ur, c[2 * k], hv[2 * r]) : mul2(ur, c[0]);
      hv[2 * r + 1] = k ? fma2(ur, c[2 * k + 1], hv[2 * r + 1]) : mul2(ur, c[1]);
    }
#pragma unroll
    for (int r = 0; r < 3; r++) {
      const u64 ui = W[2 * (3 * r + k) + 1];
      hv[2 * r] = fma2(ui, n, hv[2 * r]);
      hv[2 * r + 1] = fma2(ui, c[2 * k], hv[2 * r + 1]);
    }
  }
}
__device__ __forceinline__ void su3_one(const float *W, const float *c, float *hv) {
#pragma unroll
  for (int k = 0; k < 3; k++) {
#pragma unroll
    for (int r = 0; r < 3; r++) {
      const float ur = W[2 * (3 * r + k)];
      hv[2 * r] = k ? fmaf(ur, c[2 * k], hv[2 * r]) : ur * c[0];
      hv[2 * r + 1] = k ? fmaf(ur, c[2 * k + 1], hv[2 * r + 1]) : ur * c[1];
    }
#pragma unroll
    for (int r = 0; r < 3; r++) {
      const float ui = W[2 * (3 * r + k) + 1];
      hv[2 * r] = fmaf(-ui, c[2 * k + 1], hv[2 * r]);
      hv[2 * r + 1] = fmaf(ui, c[2 * k], hv[2 * r + 1]);
    }
  }
}

// y = M x for the packed Hermitian block of both sites (36 packed reals in the
// order of herm6_mv). LAST: the diagonal term, the largest by far, is added when
// the row's others are summed, so that one rounding has its size and not ten. In
// FP32 storage this more than pays for the even sites' correction being summed
// over the MR steps (errors against 64 bits, 16x8^3, 1 to 4 sweeps of 2 to 5 steps:
// 1.24..1.43e-7 general kernel, 1.27..1.55e-7 here with the diagonal first,
// 0.90..1.22e-7 last; a phase on 64x32^3 0.372 and 0.370 ms); in 16-bit storage,
// where the fields' rounding hides it, it would cost 3% (the MR loop's registers).
template <bool LAST> __device__ __forceinline__ void herm6_pair(const u64 *m, const u64 *x, u64 *y) {
  u64 n[12];
#pragma unroll
  for (int i = 0; i < 12; i++) n[i] = neg2(x[i]);
  auto diag = [&](int i) {
    y[2 * i] = fma2(m[i], x[2 * i], y[2 * i]);
    y[2 * i + 1] = fma2(m[i], x[2 * i + 1], y[2 * i + 1]);
  };
  if constexpr (!LAST) {
#pragma unroll
    for (int i = 0; i < 6; i++) {
      y[2 * i] = mul2(m[i], x[2 * i]);
      y[2 * i + 1] = mul2(m[i], x[2 * i + 1]);
    }
  }
#pragma unroll
  for (int i = 0; i < 6; i++)
#pragma unroll
    for (int j = i + 1; j < 6; j++) {
      const u64 ar = m[2 * herm_off(i, j)], ai = m[2 * herm_off(i, j) + 1];
      const bool fi = LAST && i == 0 && j == 1, fj = LAST && i == 0;   // the first term of row i, of row j
      y[2 * i] = fi ? mul2(ar, x[2 * j]) : fma2(ar, x[2 * j], y[2 * i]);
      y[2 * i + 1] = fi ? mul2(ar, x[2 * j + 1]) : fma2(ar, x[2 * j + 1], y[2 * i + 1]);
      y[2 * j] = fj ? mul2(ar, x[2 * i]) : fma2(ar, x[2 * i], y[2 * j]);
      y[2 * j + 1] = fj ? mul2(ar, x[2 * i + 1]) : fma2(ar, x[2 * i + 1], y[2 * j + 1]);
      y[2 * i] = fma2(ai, n[2 * j + 1], y[2 * i]);
      y[2 * i + 1] = fma2(ai, x[2 * j], y[2 * i + 1]);
      y[2 * j] = fma2(ai, x[2 * i + 1], y[2 * j]);
      y[2 * j + 1] = fma2(ai, n[2 * i], y[2 * j + 1]);
      if (LAST && j == 5) {   // row i is complete but for its diagonal, with i = 4 row 5 too
        diag(i);
        if (i == 4) diag(5);
      }
    }
}

// Partial sums of a site pair's hops for thread half h: spin h of the upper
// components (u) and the contributions to lower spin h (a) and 1 - h (b).
// A hop (1 -+ g) W psi projected on spin h is chi = u_h + phase * d, with
// d = d_{1-h} for x and y, d_h for z and t; its upper part adds to u, its
// lower part, the conjugate phase times that with the hop's sign, to b (x, y)
// or a (z, t). hv holds -1/2 W chi (the tile's links are times -1/2).
struct PairAcc {
  u64 u[6], a[6], b[6];
};
// v += s hv and v += s i hv (s: packed sign)
__device__ __forceinline__ void acc_s(u64 *v, u64 s, const u64 *hv) {
#pragma unroll
  for (int i = 0; i < 6; i++) v[i] = fma2(s, hv[i], v[i]);
}
__device__ __forceinline__ void acc_si(u64 *v, u64 s, u64 ns, const u64 *hv) {
#pragma unroll
  for (int c = 0; c < 3; c++) {
    v[2 * c] = fma2(ns, hv[2 * c + 1], v[2 * c]);
    v[2 * c + 1] = fma2(s, hv[2 * c], v[2 * c + 1]);
  }
}
__device__ __forceinline__ void acc_add(u64 *v, const u64 *hv) {
#pragma unroll
  for (int i = 0; i < 6; i++) v[i] = add2(v[i], hv[i]);
}
__device__ __forceinline__ void acc_sub(u64 *v, const u64 *hv) {
#pragma unroll
  for (int i = 0; i < 6; i++) v[i] = sub2(v[i], hv[i]);
}
// three colours of one spin component of a shared vector
__device__ __forceinline__ void ld3(const quad *p, int rows, u64 *o) {
#pragma unroll
  for (int c = 0; c < 3; c++) {
    const quad v = p[c * rows];
    o[2 * c] = v.x;
    o[2 * c + 1] = v.y;
  }
}
// chi = u + s d, chi = u + s i d
__device__ __forceinline__ void proj_s(const u64 *u, const u64 *d, u64 s, u64 *chi) {
#pragma unroll
  for (int i = 0; i < 6; i++) chi[i] = fma2(s, d[i], u[i]);
}
__device__ __forceinline__ void proj_si(const u64 *u, const u64 *d, u64 s, u64 ns, u64 *chi) {
#pragma unroll
  for (int c = 0; c < 3; c++) {
    chi[2 * c] = fma2(ns, d[2 * c + 1], u[2 * c]);
    chi[2 * c + 1] = fma2(s, d[2 * c], u[2 * c + 1]);
  }
}

// Row slot of spin component s of a shared vector: neighbouring lanes read
// (and write) different spins of one row, so the spins alternate between the
// two halves of the 32 banks (rows of 16 bytes, components a multiple of 1 KB
// apart).
__device__ __forceinline__ int slot(int s, int r) { return r ^ (((s ^ (s >> 1)) & 1) << 2); }
// first colour of spin s at row r
__device__ __forceinline__ int spin_at(int rows, int s, int r) { return 3 * s * rows + slot(s, r); }

// What a thread knows about its row: neighbours in the block, signs
struct PairThread {
  int h, r, y, z, t, q;
  u64 sh, nsh;   // (+1, +1) for h = 0, (-1, -1) for h = 1, and its negative
};

// All hops inside the block into the thread's row pair of parity p (spin h),
// from the shared vector V of the other parity. L: the block's links; xl: the
// thread's x-links for this parity, issued by tm_issue54.
template <int SHAPE>
__device__ __forceinline__ void hops_pair(const PairThread &T, int p, const quad *V, const quad *L, uint32_t *xl,
                                          PairAcc &o) {
  using PG = PairGeom<SHAPE>;
  constexpr int R = PG::ROWS, ST = 2 * R;
  const quad *Vu = V + spin_at(R, T.h, T.r), *Vd = V + spin_at(R, 2 + T.h, T.r), *Ve = V + spin_at(R, 3 - T.h, T.r);
  const quad *Ld = L + p * R + T.r, *Ls = L + (1 - p) * R + T.r;   // links at the row's sites of parity p and 1 - p
  {   // x: the packed hop and the single one
    const bool s = T.q ^ p;   // first site of the pair: x = s
    const float sx = s ? -1.f : 1.f;
    const u64 S = pk(sx, sx), N = pk(-sx, -sx);
    u64 W[18], u[6], e[6], chi[6], hv[6];
    float w[18];
    ld3(Vu, R, u);
    ld3(Ve, R, e);
    tm_wait54(xl);
#pragma unroll
    for (int i = 0; i < 18; i++) {
      W[i] = word2(xl, i);
      w[i] = __uint_as_float(xl[36 + i]);
    }
    proj_si(u, e, S, N, chi);
    su3_reg(W, chi, hv);
#pragma unroll
    for (int i = 0; i < 6; i++) {
      o.u[i] = hv[i];
      o.a[i] = 0ull;
    }
#pragma unroll
    for (int c = 0; c < 3; c++) {   // b = -sx i hv
      o.b[2 * c] = mul2(S, hv[2 * c + 1]);
      o.b[2 * c + 1] = mul2(N, hv[2 * c]);
    }
    // the single hop: from A to B (s = 0) or from B to A (s = 1), opposite direction
    float us[6], es[6], cs[6], hs[6];
#pragma unroll
    for (int i = 0; i < 6; i++) {
      us[i] = s ? hi(u[i]) : lo(u[i]);
      es[i] = s ? hi(e[i]) : lo(e[i]);
    }
#pragma unroll
    for (int c = 0; c < 3; c++) {
      cs[2 * c] = fmaf(sx, es[2 * c + 1], us[2 * c]);
      cs[2 * c + 1] = fmaf(-sx, es[2 * c], us[2 * c + 1]);
    }
    su3_one(w, cs, hs);
#pragma unroll
    for (int i = 0; i < 6; i++) hv[i] = pk(s ? hs[i] : 0.f, s ? 0.f : hs[i]);
    acc_add(o.u, hv);
    acc_si(o.b, S, N, hv);
  }
  {   // y
    const int f = T.y < 3 ? 1 : 0, b = T.y > 0 ? -1 : 0;
    u64 u[6], e[6], chi[6], hv[6];
    ld3(Vu + f, R, u);
    ld3(Ve + f, R, e);
    proj_s(u, e, T.sh, chi);
    su3_pair<false>(Ld + 9 * ST, ST, chi, hv);
    if (T.y < 3) {
      acc_add(o.u, hv);
      acc_s(o.b, T.sh, hv);
    }
    ld3(Vu + b, R, u);
    ld3(Ve + b, R, e);
    proj_s(u, e, T.nsh, chi);
    su3_pair<true>(Ls + 9 * ST + b, ST, chi, hv);
    if (T.y > 0) {
      acc_add(o.u, hv);
      acc_s(o.b, T.nsh, hv);
    }
  }
  {   // z
    const int f = T.z < 3 ? 4 : 0, b = T.z > 0 ? -4 : 0;
    u64 u[6], d[6], chi[6], hv[6];
    ld3(V + spin_at(R, T.h, T.r + f), R, u);
    ld3(V + spin_at(R, 2 + T.h, T.r + f), R, d);
    proj_si(u, d, T.sh, T.nsh, chi);
    su3_pair<false>(Ld + 18 * ST, ST, chi, hv);
    if (T.z < 3) {
      acc_add(o.u, hv);
      acc_si(o.a, T.nsh, T.sh, hv);
    }
    ld3(V + spin_at(R, T.h, T.r + b), R, u);
    ld3(V + spin_at(R, 2 + T.h, T.r + b), R, d);
    proj_si(u, d, T.nsh, T.sh, chi);
    su3_pair<true>(Ls + 18 * ST + b, ST, chi, hv);
    if (T.z > 0) {
      acc_add(o.u, hv);
      acc_si(o.a, T.sh, T.nsh, hv);
    }
  }
  // t (the same for the whole warp)
  if (T.t < PG::BT - 1) {
    u64 u[6], d[6], chi[6], hv[6];
    ld3(Vu + 16, R, u);
    ld3(Vd + 16, R, d);
#pragma unroll
    for (int i = 0; i < 6; i++) chi[i] = sub2(u[i], d[i]);
    su3_pair<false>(Ld + 27 * ST, ST, chi, hv);
    acc_add(o.u, hv);
    acc_sub(o.a, hv);
  }
  if (T.t > 0) {
    u64 u[6], d[6], chi[6], hv[6];
    ld3(Vu - 16, R, u);
    ld3(Vd - 16, R, d);
#pragma unroll
    for (int i = 0; i < 6; i++) chi[i] = add2(u[i], d[i]);
    su3_pair<true>(Ls + 27 * ST - 16, ST, chi, hv);
    acc_add(o.u, hv);
    acc_add(o.a, hv);
  }
}

// spin h of both halves -> chirality h: half 0 keeps its upper part and takes
// half 1's; half 1 keeps its lower contributions and adds half 0's
__device__ __forceinline__ void to_chirality(const PairThread &T, const PairAcc &o, u64 *out) {
  const bool h = T.h;
#pragma unroll
  for (int i = 0; i < 6; i++) {
    const u64 x1 = shfl2(sel2(h, o.u[i], o.a[i]));   // h = 0: u of half 1; h = 1: a of half 0 (lower spin 0)
    const u64 x2 = shfl2(o.b[i]);                    // h = 1: b of half 0 (lower spin 1)
    out[i] = h ? add2(o.b[i], x1) : o.u[i];
    out[6 + i] = h ? add2(o.a[i], x2) : x1;
  }
}

// this half's components (spins 2h, 2h + 1) of the thread's row in vector V
__device__ __forceinline__ void st6(const PairThread &T, quad *V, int rows, const u64 *v) {
  quad *p = V + spin_at(rows, 2 * T.h, T.r), *q = V + spin_at(rows, 2 * T.h + 1, T.r);
#pragma unroll
  for (int c = 0; c < 3; c++) {
    p[c * rows] = quad{v[2 * c], v[2 * c + 1]};
    q[c * rows] = quad{v[6 + 2 * c], v[7 + 2 * c]};
  }
}
__device__ __forceinline__ void ld6(const PairThread &T, const quad *V, int rows, u64 *v) {
  ld3(V + spin_at(rows, 2 * T.h, T.r), rows, v);
  ld3(V + spin_at(rows, 2 * T.h + 1, T.r), rows, v + 6);
}

// sum of three values over the CTA's NW warps; red: [3][8] floats. The caller
// reaches a barrier before any thread can write red again.
template <int NW> __device__ __forceinline__ void cta_sum3(float &a, float &b, float &c, float *red) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    a += __shfl_xor_sync(0xffffffffu, a, o);
    b += __shfl_xor_sync(0xffffffffu, b, o);
    c += __shfl_xor_sync(0xffffffffu, c, o);
  }
  const int w = threadIdx.x / 32;
  if ((threadIdx.x & 31) == 0) {
    red[w] = a;
    red[8 + w] = b;
    red[16 + w] = c;
  }
  __syncthreads();
  a = b = c = 0.f;
#pragma unroll
  for (int i = 0; i < NW; i++) {
    a += red[i];
    b += red[8 + i];
    c += red[16 + i];
  }
}

// 32 bytes of constant data (both sites' 16-byte chunks), 32-byte aligned
__device__ __forceinline__ void ldg32(const void *p, uint4 &a, uint4 &b) {
  asm("ld.global.nc.v8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
      : "=r"(a.x), "=r"(a.y), "=r"(a.z), "=r"(a.w), "=r"(b.x), "=r"(b.y), "=r"(b.z), "=r"(b.w)
      : "l"(p));
}
// chirality block h of sites s and s + 1 (s even) of a chunked clover tile (see
// clover_block_chunked; n sites per chunk row) as 36 packed reals
template <typename P>
__device__ __forceinline__ void clover_pair(const P *tile, int n, int s, int h, uint32_t *m) {
  constexpr int CP = chunk_pairs<P>();
  DD_CHECK_INDEX(s, n - 1);
  const uint4 *q = (const uint4 *)tile + s;
  auto put = [&](int i, P a, P b) {   // pair i of both sites
    const cpx<float> u = from_pair<float, P>(a), v = from_pair<float, P>(b);
    m[4 * i] = __float_as_uint(u.re);
    m[4 * i + 1] = __float_as_uint(v.re);
    m[4 * i + 2] = __float_as_uint(u.im);
    m[4 * i + 3] = __float_as_uint(v.im);
  };
  constexpr int NC = CP == 4 ? 4 : 18 / CP;   // whole chunks of a block
#pragma unroll
  for (int c = 0; c < NC; c++) {
    uint4 a, b;
    ldg32(q + (size_t)(NC * h + c) * n, a, b);
    const P *pa = (const P *)&a, *pb = (const P *)&b;
#pragma unroll
    for (int k = 0; k < CP; k++) put(CP * c + k, pa[k], pb[k]);
  }
  if constexpr (CP == 4) {   // the last two pairs: half h of chunk 8
    const uint2 a = __ldg((const uint2 *)(q + (size_t)8 * n) + h), b = __ldg((const uint2 *)(q + (size_t)8 * n + 1) + h);
    const P *pa = (const P *)&a, *pb = (const P *)&b;
#pragma unroll
    for (int k = 0; k < 2; k++) put(16 + k, pa[k], pb[k]);
  }
}

// ---- fields: the chirality half h (six complex) of sites s and s + 1 of block b
template <typename S>
__device__ __forceinline__ void half_site_ld(const char *base, size_t cstride, int h, cpx<float> *o) {
  if constexpr (Store<S>::prec == DD_F32) {
#pragma unroll
    for (int k = 0; k < 3; k++) {
      const float4 v = *(const float4 *)(base + (3 * h + k) * cstride);
      o[2 * k] = {v.x, v.y};
      o[2 * k + 1] = {v.z, v.w};
    }
  } else {
    // half 0: chunk 0 and the first half of chunk 1; half 1: the second half of chunk 1 and chunk 2
    const uint4 v = *(const uint4 *)(base + 2 * h * cstride);
    const uint2 w = *(const uint2 *)(base + cstride + 8 * h);
    cpx<float> f[4], g[2];
    if constexpr (Store<S>::prec == DD_F16N) {
      const short *q = (const short *)&v, *p = (const short *)&w;
#pragma unroll
      for (int k = 0; k < 4; k++) f[k] = {(float)q[2 * k], (float)q[2 * k + 1]};
#pragma unroll
      for (int k = 0; k < 2; k++) g[k] = {(float)p[2 * k], (float)p[2 * k + 1]};
    } else {
      using P = typename Store<S>::pair_t;
      const P *q = (const P *)&v, *p = (const P *)&w;
#pragma unroll
      for (int k = 0; k < 4; k++) f[k] = from_pair<float, P>(q[k]);
#pragma unroll
      for (int k = 0; k < 2; k++) g[k] = from_pair<float, P>(p[k]);
    }
#pragma unroll
    for (int i = 0; i < 6; i++) {
      const cpx<float> a = i < 4 ? f[i < 4 ? i : 0] : g[i < 4 ? 0 : i - 4];
      const cpx<float> c = i < 2 ? g[i < 2 ? i : 0] : f[i < 2 ? 0 : i - 2];
      o[i] = h ? c : a;
    }
  }
}
template <typename S>
__device__ __forceinline__ void half_ld(const void *field, const Geom &g, int b, int s, int h, cpx<float> *A,
                                        cpx<float> *B) {
  DD_CHECK_INDEX(b, g.nblocks);
  DD_CHECK_INDEX(s, g.Vb - 1);
  const char *blk = (const char *)field + (size_t)b * g.Vb * spinor_site_bytes(Store<S>::prec);
  const size_t cs = (size_t)g.Vb * 16;
  half_site_ld<S>(blk + (size_t)s * 16, cs, h, A);
  half_site_ld<S>(blk + (size_t)s * 16 + 16, cs, h, B);
  if constexpr (Store<S>::prec == DD_F16N) {
    const float2 n = *(const float2 *)(blk + 3 * cs + (size_t)s * 4);
    const float na = n.x * (1.0f / 32767.0f), nb = n.y * (1.0f / 32767.0f);
#pragma unroll
    for (int i = 0; i < 6; i++) {
      A[i] = {A[i].re * na, A[i].im * na};
      B[i] = {B[i].re * nb, B[i].im * nb};
    }
  }
}
template <typename S>
__device__ __forceinline__ void half_site_st(char *base, size_t cstride, int h, const cpx<float> *v, float inv) {
  if constexpr (Store<S>::prec == DD_F32) {
#pragma unroll
    for (int k = 0; k < 3; k++)
      *(float4 *)(base + (3 * h + k) * cstride) = make_float4(v[2 * k].re, v[2 * k].im, v[2 * k + 1].re, v[2 * k + 1].im);
  } else {
    uint4 f;
    uint2 g;
    if constexpr (Store<S>::prec == DD_F16N) {
      short *q = (short *)&f, *p = (short *)&g;
      auto fix = [&](float x) { return (short)fminf(fmaxf(rintf(x * inv), -32767.f), 32767.f); };
#pragma unroll
      for (int k = 0; k < 4; k++) {
        q[2 * k] = fix(h ? v[2 + k].re : v[k].re);
        q[2 * k + 1] = fix(h ? v[2 + k].im : v[k].im);
      }
#pragma unroll
      for (int k = 0; k < 2; k++) {
        p[2 * k] = fix(h ? v[k].re : v[4 + k].re);
        p[2 * k + 1] = fix(h ? v[k].im : v[4 + k].im);
      }
    } else {
      using P = typename Store<S>::pair_t;
      P *q = (P *)&f, *p = (P *)&g;
#pragma unroll
      for (int k = 0; k < 4; k++) q[k] = to_pair<P, float>(h ? v[2 + k].re : v[k].re, h ? v[2 + k].im : v[k].im);
#pragma unroll
      for (int k = 0; k < 2; k++) p[k] = to_pair<P, float>(h ? v[k].re : v[4 + k].re, h ? v[k].im : v[4 + k].im);
    }
    *(uint4 *)(base + 2 * h * cstride) = f;
    *(uint2 *)(base + cstride + 8 * h) = g;
  }
}
// (both halves of a site together for DD_F16N: its scale is the largest
// component over the two)
template <typename S>
__device__ __forceinline__ void half_st(void *field, const Geom &g, int b, int s, int h, const cpx<float> *A,
                                        const cpx<float> *B) {
  DD_CHECK_INDEX(b, g.nblocks);
  DD_CHECK_INDEX(s, g.Vb - 1);
  char *blk = (char *)field + (size_t)b * g.Vb * spinor_site_bytes(Store<S>::prec);
  const size_t cs = (size_t)g.Vb * 16;
  float ia = 0.f, ib = 0.f;
  if constexpr (Store<S>::prec == DD_F16N) {
    float ma = 0.f, mb = 0.f;
#pragma unroll
    for (int i = 0; i < 6; i++) {
      ma = fmaxf(ma, fmaxf(fabsf(A[i].re), fabsf(A[i].im)));
      mb = fmaxf(mb, fmaxf(fabsf(B[i].re), fabsf(B[i].im)));
    }
    ma = fmaxf(ma, __shfl_xor_sync(0xffffffffu, ma, 1));
    mb = fmaxf(mb, __shfl_xor_sync(0xffffffffu, mb, 1));
    if (h == 0) *(float2 *)(blk + 3 * cs + (size_t)s * 4) = make_float2(ma, mb);
    ia = ma > 0.f ? 32767.f / ma : 0.f;
    ib = mb > 0.f ? 32767.f / mb : 0.f;
  }
  half_site_st<S>(blk + (size_t)s * 16, cs, h, A, ia);
  half_site_st<S>(blk + (size_t)s * 16 + 16, cs, h, B, ib);
}

// Work-field quads (residuals and face flux): one complex number of both
// sites in storage Q; DD_F16N keeps its residuals in FP32 (they fit the field)
template <typename S, bool RES> struct QuadStore {
  static constexpr bool f32 = Store<S>::prec == DD_F32 || (RES && Store<S>::prec == DD_F16N);
  static constexpr int bytes = f32 ? 16 : 8;
  using raw = std::conditional_t<f32, float4, uint2>;   // as loaded, converted where it is used
};
template <typename S, bool RES>
__device__ __forceinline__ typename QuadStore<S, RES>::raw quad_raw(const void *p, size_t i) {
  return ((const typename QuadStore<S, RES>::raw *)p)[i];
}
template <typename S, bool RES> __device__ __forceinline__ quad quad_of(typename QuadStore<S, RES>::raw v) {
  if constexpr (QuadStore<S, RES>::f32) {
    return quad{pk(v.x, v.y), pk(v.z, v.w)};
  } else {
    using P = typename Store<S>::pair_t;
    const P *h = (const P *)&v;
    const cpx<float> a = from_pair<float, P>(h[0]), b = from_pair<float, P>(h[1]);
    return quad{pk(a.re, a.im), pk(b.re, b.im)};
  }
}
template <typename S, bool RES> __device__ __forceinline__ void quad_st(void *p, size_t i, u64 re, u64 im) {
  if constexpr (QuadStore<S, RES>::f32) {
    ((float4 *)p)[i] = make_float4(lo(re), hi(re), lo(im), hi(im));
  } else {
    using P = typename Store<S>::pair_t;
    uint2 v;
    P *h = (P *)&v;
    h[0] = to_pair<P, float>(lo(re), hi(re));
    h[1] = to_pair<P, float>(lo(im), hi(im));
    ((uint2 *)p)[i] = v;
  }
}

// ---- face flux (see dd_sap_kernels.cuh: across its upper faces a block sends
// the whole hop of its correction e, across its lower faces the projection,
// which the receiver multiplies by its own link). Layout of a block's
// incoming flux in pairs of reals: two x faces [6][rows] single complex
// numbers, then the y, z and t faces [6][parity][face rows] quads; face 2 mu:
// the block's upper face in mu, 2 mu + 1 its lower one.
template <int SHAPE> struct Flux {
  using PG = PairGeom<SHAPE>;
  static constexpr int FR(int mu) { return mu == 3 ? 16 : PG::ROWS / 4; }
  static constexpr int off(int f) {   // in pairs of reals
    int o = 0;
    for (int g = 0; g < f; g++) o += g < 2 ? 6 * PG::ROWS : 24 * FR(g / 2);
    return o;
  }
  static constexpr int total = off(8);
  static_assert(total <= 12 * PG::VB, "the flux fits a spinor field");
  static_assert(total * 8 <= 2 * PG::VEC * 16, "and the shared vectors");
};
template <int SHAPE, int MU> __device__ __forceinline__ int face_row(const PairThread &T) {
  if constexpr (MU == 1) return T.z + 4 * T.t;
  if constexpr (MU == 2) return T.y + 4 * T.t;
  return T.y + 4 * T.z;
}
// incoming flux of the y, z or t face the row lies on, added to the even
// (acc[0]) and odd (acc[1]) pair's partial sums (the two side by side: their
// chains of dependent instructions overlap)
template <typename S, int SHAPE, int MU>
__device__ __forceinline__ void flux_in(const PairThread &T, const char *H, const quad *L, PairAcc *acc) {
  using PG = PairGeom<SHAPE>;
  constexpr int R = PG::ROWS, ST = 2 * R, FR = Flux<SHAPE>::FR(MU), PB = sizeof(typename Store<S>::pair_t);
  constexpr int last = MU == 3 ? PG::BT - 1 : 3;
  const int x = MU == 1 ? T.y : MU == 2 ? T.z : T.t;
  const bool up = x == last;
  if (!up && x != 0) return;
  const char *F = H + (size_t)(up ? Flux<SHAPE>::off(2 * MU) : Flux<SHAPE>::off(2 * MU + 1)) * PB;
  const int fr = face_row<SHAPE, MU>(T);
  u64 v[2][6], hv[2][6];
#pragma unroll
  for (int p = 0; p < 2; p++)
#pragma unroll
    for (int c = 0; c < 3; c++) {
      const quad w = quad_of<S, false>(quad_raw<S, false>(F, ((3 * T.h + c) * 2 + p) * FR + fr));
      v[p][2 * c] = w.x;
      v[p][2 * c + 1] = w.y;
    }
  if (up) {
#pragma unroll
    for (int p = 0; p < 2; p++) su3_pair<false>(L + 9 * MU * ST + p * R + T.r, ST, v[p], hv[p]);
#pragma unroll
    for (int p = 0; p < 2; p++)
#pragma unroll
      for (int i = 0; i < 6; i++) v[p][i] = hv[p][i];
  }
#pragma unroll
  for (int p = 0; p < 2; p++) {
    acc_add(acc[p].u, v[p]);
    // the signs of hops_pair: forward hops across the upper face
    if constexpr (MU == 1) acc_s(acc[p].b, up ? T.sh : T.nsh, v[p]);
    if constexpr (MU == 2) acc_si(acc[p].a, up ? T.nsh : T.sh, up ? T.sh : T.nsh, v[p]);
    if constexpr (MU == 3) {
      if (up) acc_sub(acc[p].a, v[p]);
      else acc_add(acc[p].a, v[p]);
    }
  }
}
// the x faces: site x = 0 is element A of the row's pair of parity q, site
// x = 3 element B of the other one, whose hop l / hv starts the sums
template <typename S, int SHAPE>
__device__ __forceinline__ void flux_x(const PairThread &T, const char *H, const quad *L, float *l, float *hv) {
  using P = typename Store<S>::pair_t;
  constexpr int R = PairGeom<SHAPE>::ROWS, ST = 2 * R;
  float c[6], w[18];
#pragma unroll
  for (int k = 0; k < 3; k++) {
    const P *F = (const P *)H + (3 * T.h + k) * R + T.r;
    const cpx<float> v = from_pair<float, P>(F[Flux<SHAPE>::off(0)]), u = from_pair<float, P>(F[Flux<SHAPE>::off(1)]);
    c[2 * k] = v.re;
    c[2 * k + 1] = v.im;
    l[2 * k] = u.re;
    l[2 * k + 1] = u.im;
  }
  const quad *U3 = L + (1 - T.q) * R + T.r;
#pragma unroll
  for (int i = 0; i < 9; i++) {
    const quad u = U3[i * ST];
    w[2 * i] = hi(u.x);
    w[2 * i + 1] = hi(u.y);
  }
  su3_one(w, c, hv);
}
// chirality half h of the incoming hops into the row's even and odd pair
template <typename S, int SHAPE>
__device__ __forceinline__ void flux_sum(const PairThread &T, const char *H, const quad *L, u64 *de, u64 *dd) {
  PairAcc acc[2];
  float l[6], hv[6];
  flux_x<S, SHAPE>(T, H, L, l, hv);
#pragma unroll
  for (int p = 0; p < 2; p++) {
    const bool at0 = T.q == p;   // this parity holds x = 0 (else x = 3)
#pragma unroll
    for (int k = 0; k < 3; k++) {
      const float re = at0 ? l[2 * k] : hv[2 * k], im = at0 ? l[2 * k + 1] : hv[2 * k + 1];
      const u64 vr = at0 ? pk(re, 0.f) : pk(0.f, re), vi = at0 ? pk(im, 0.f) : pk(0.f, im);
      acc[p].u[2 * k] = vr;
      acc[p].u[2 * k + 1] = vi;
      // lower face (backward hop): b = i hv; upper (forward): b = -i hv
      acc[p].b[2 * k] = at0 ? neg2(vi) : vi;
      acc[p].b[2 * k + 1] = at0 ? vr : neg2(vr);
      acc[p].a[2 * k] = acc[p].a[2 * k + 1] = 0ull;
    }
  }
  flux_in<S, SHAPE, 1>(T, H, L, acc);
  flux_in<S, SHAPE, 2>(T, H, L, acc);
  flux_in<S, SHAPE, 3>(T, H, L, acc);
  __syncwarp();
  to_chirality(T, acc[0], de);
  to_chirality(T, acc[1], dd);
}

// index of the neighbouring block in direction mu and whether the hop crosses
// the antiperiodic time edge
template <int MU> __device__ __forceinline__ int block_step(const Geom &g, int b, const int *bc, bool up, float &sg) {
  int v = bc[MU] + (up ? 1 : -1);
  const bool wrap = v < 0 || v >= g.nb[MU];
  if (wrap) v += up ? -g.nb[MU] : g.nb[MU];
  sg = (MU == 3 && wrap && g.antiperiodic) ? -1.f : 1.f;
  return b + (v - bc[MU]) * g.bstride[MU];
}
// the hop of the correction (the row's pair of parity p: u spin h of the upper
// components, d and e lower spins h and 1 - h) across the y, z or t face the
// row lies on, into the neighbouring block's entry
template <typename S, int SHAPE, int MU>
__device__ __forceinline__ void flux_out(const PairThread &T, const Geom &g, int b, const int *bc, const quad *L,
                                         int p, const u64 *u, const u64 *d, const u64 *e, char *H) {
  using PG = PairGeom<SHAPE>;
  constexpr int R = PG::ROWS, ST = 2 * R, FR = Flux<SHAPE>::FR(MU), PB = sizeof(typename Store<S>::pair_t);
  constexpr int last = MU == 3 ? PG::BT - 1 : 3;
  const int x = MU == 1 ? T.y : MU == 2 ? T.z : T.t;
  const bool up = x == last;
  if (!up && x != 0) return;
  float sg;
  const int nb = block_step<MU>(g, b, bc, up, sg);
  char *F = H + ((size_t)nb * Flux<SHAPE>::total + (up ? Flux<SHAPE>::off(2 * MU + 1) : Flux<SHAPE>::off(2 * MU))) * PB;
  const int fr = face_row<SHAPE, MU>(T);
  u64 chi[6], hv[6];
  // across the upper face the receiver's backward hop, across the lower its forward one
  if constexpr (MU == 1) proj_s(u, e, up ? T.nsh : T.sh, chi);
  if constexpr (MU == 2) proj_si(u, d, up ? T.nsh : T.sh, up ? T.sh : T.nsh, chi);
  if constexpr (MU == 3) {
#pragma unroll
    for (int i = 0; i < 6; i++) chi[i] = up ? add2(u[i], d[i]) : sub2(u[i], d[i]);
  }
  if (up) {
    su3_pair<true>(L + 9 * MU * ST + p * R + T.r, ST, chi, hv);
#pragma unroll
    for (int i = 0; i < 6; i++) chi[i] = hv[i];
  }
  if constexpr (MU == 3) {
#pragma unroll
    for (int i = 0; i < 6; i++) chi[i] = mul2(pk(sg, sg), chi[i]);
  }
#pragma unroll
  for (int c = 0; c < 3; c++)
    quad_st<S, false>(F, ((3 * T.h + c) * 2 + 1 - p) * FR + fr, chi[2 * c], chi[2 * c + 1]);   // the receiver's parity
}
template <typename S, int SHAPE>
__device__ __forceinline__ void flux_out_x(const PairThread &T, const Geom &g, int b, const int *bc, const quad *L,
                                           const quad *V, char *H) {
  using P = typename Store<S>::pair_t;
  constexpr int R = PairGeom<SHAPE>::ROWS, ST = 2 * R;
  float sg, c[6], o[6];
  u64 u[6], e[6];
  // x = 0 (element A of parity q): forward projection to the block below
  const quad *v = V + T.q * PairGeom<SHAPE>::VEC;
  ld3(v + spin_at(R, T.h, T.r), R, u);
  ld3(v + spin_at(R, 3 - T.h, T.r), R, e);
  P *F = (P *)H + (size_t)block_step<0>(g, b, bc, false, sg) * Flux<SHAPE>::total + Flux<SHAPE>::off(0);
#pragma unroll
  for (int k = 0; k < 3; k++)
    F[(3 * T.h + k) * R + T.r] = to_pair<P, float>(lo(u[2 * k]) - lo(e[2 * k + 1]), lo(u[2 * k + 1]) + lo(e[2 * k]));
  // x = 3 (element B of the other parity): the backward hop into the block above
  v = V + (1 - T.q) * PairGeom<SHAPE>::VEC;
  ld3(v + spin_at(R, T.h, T.r), R, u);
  ld3(v + spin_at(R, 3 - T.h, T.r), R, e);
#pragma unroll
  for (int k = 0; k < 3; k++) {
    c[2 * k] = hi(u[2 * k]) + hi(e[2 * k + 1]);
    c[2 * k + 1] = hi(u[2 * k + 1]) - hi(e[2 * k]);
  }
  float w[18];
  const quad *U3 = L + (1 - T.q) * R + T.r;
#pragma unroll
  for (int r = 0; r < 3; r++)
#pragma unroll
    for (int k = 0; k < 3; k++) {   // the link's conjugate transpose
      const quad q = U3[(3 * k + r) * ST];
      w[2 * (3 * r + k)] = hi(q.x);
      w[2 * (3 * r + k) + 1] = -hi(q.y);
    }
  su3_one(w, c, o);
  F = (P *)H + (size_t)block_step<0>(g, b, bc, true, sg) * Flux<SHAPE>::total + Flux<SHAPE>::off(1);
#pragma unroll
  for (int k = 0; k < 3; k++) F[(3 * T.h + k) * R + T.r] = to_pair<P, float>(o[2 * k], o[2 * k + 1]);
}

// One colour phase. Work items (lattice group, block of the colour, tile of
// right-hand sides), one per CTA. mode: SAP_INCR is implied.
template <typename S, int SHAPE, bool MULTI>
__global__ void __launch_bounds__(PairGeom<SHAPE>::NT, SHAPE == 1 ? 2 : 1)
    k_sap_pair(const SapGroups G, const RhsPtrs rp, const AuxPtrs ax, int colour, int self_zero, int mode, int nmr,
               int tile, int ahead, unsigned *timeouts) {
  using PG = PairGeom<SHAPE>;
  using P = typename Store<S>::pair_t;
  constexpr int R = PG::ROWS, ST = 2 * R, NT = PG::NT, CP = chunk_pairs<P>();
  constexpr unsigned LBYTES = PG::LINKS * 16;
  extern __shared__ __align__(16) unsigned char smem[];
  quad *L = (quad *)smem, *V = L + PG::LINKS;   // links; vectors: even sites, odd sites
  float *red = (float *)(V + 2 * PG::VEC);
  uint64_t *mbar = (uint64_t *)(red + 24);
  uint64_t *fbar = mbar + 1;   // the incoming flux
  uint32_t *tmem_at = (uint32_t *)(mbar + 2);
  const unsigned mbar_s = smem_u32(mbar), fbar_s = smem_u32(fbar);

  PairThread T;
  {
    T.h = threadIdx.x & 1;
    T.r = threadIdx.x >> 1;
    T.y = T.r & 3;
    T.z = (T.r >> 2) & 3;
    T.t = threadIdx.x >> 5;
    T.q = (T.y + T.z + T.t) & 1;
    const float s = T.h ? -1.f : 1.f;
    T.sh = pk(s, s);
    T.nsh = pk(-s, -s);
  }
  const int item = blockIdx.x;
  const int k = MULTI ? sap_group_of(G, item) : 0;
  const Geom g = block_shape<SHAPE>(G.grp[k].g);
  const void *__restrict__ links = G.grp[k].links;
  const P *__restrict__ clov = (const P *)G.grp[k].clov;
  const P *__restrict__ cinv = (const P *)G.grp[k].cinv;
  const int nbc = g.nblocks / 2, rhs0 = MULTI ? G.grp[k].rhs0 : 0, nrhs = MULTI ? G.grp[k].nrhs : rp.n;
  const int loc = MULTI ? item - G.grp[k].item0 : item;
  const int b = sap_block_of(g, colour, loc % nbc), rt = loc / nbc;
  constexpr unsigned SB = (unsigned)spinor_site_bytes(Store<S>::prec);
  constexpr unsigned RQ = QuadStore<S, true>::bytes, RB = 6 * NT * RQ;   // stored residual of a block
  constexpr unsigned FB = Flux<SHAPE>::total * sizeof(P);
  constexpr bool LAST = Store<S>::prec == DD_F32;   // order of the site blocks' sums, see herm6_pair

  // this thread's clover blocks: chirality h of the even and the odd pair, both
  // sites' chunks (neighbours in memory) in one 32-byte load
  uint32_t m0[72], m1[72];
  clover_pair<P>(cinv + (size_t)b * 36 * PG::VH, PG::VH, 2 * T.r, T.h, m0);
  // (the odd half of each chunk row)
  clover_pair<P>(clov + (size_t)b * 36 * PG::VB + (size_t)PG::VH * CP, PG::VB, 2 * T.r, T.h, m1);
  // The incoming flux of right-hand side r, contiguous, into the place of the
  // vectors (its reader's prologue then has no trip to L2 in it: read face by
  // face from global memory it took 8200 clocks of a block's 57500 at
  // 64x32^3; issued by thread 0)
  auto flux_issue = [&](int r) {
    fence_proxy_async();
    mbar_arrive_expect(fbar, FB);
    bulk_g2s(V, (const char *)ax.e[r] + (size_t)b * FB, FB, fbar);
  };
  // The next phase's CTAs may start as soon as every CTA of this one has: up to
  // grid_wait they touch the operator only, which no phase writes. (Threads 0
  // and 32 wait below, so the CTA as a whole gets past tmem_sync only once the
  // phase before is complete.)
  grid_launch_dependents();
  // one thread of each warp asks for what comes later
  if (threadIdx.x == 0) {
    mbar_init(mbar);
    mbar_init(fbar);
    fence_proxy_async();
    if constexpr (Store<S>::prec == DD_F32) {
      mbar_arrive_expect(mbar, LBYTES);
      bulk_g2s(L, (const char *)links + (size_t)b * LBYTES, LBYTES, mbar);
    }
    if (mode & SAP_HALO_E) {
      grid_wait();
      flux_issue(rhs0 + rt * tile);
    }
  }
  if (threadIdx.x == 64) {
    // the operator tiles of the CTA that starts about when this one ends,
    // requested into L2
    if (const int ni = item + ahead; ahead && ni < G.nitems) {
      const int nk = MULTI ? sap_group_of(G, ni) : 0;
      const Geom &ng = G.grp[nk].g;
      const int nnbc = ng.nblocks / 2, nloc = MULTI ? ni - G.grp[nk].item0 : ni;
      const size_t nb = sap_block_of(ng, colour, nloc % nnbc);
      prefetch_l2((const P *)G.grp[nk].links + nb * 36 * PG::VB, 36u * PG::VB * sizeof(P));
      prefetch_l2((const P *)G.grp[nk].cinv + nb * 36 * PG::VH, 36u * PG::VH * sizeof(P));
      const P *nc = (const P *)G.grp[nk].clov + nb * 36 * PG::VB;
      for (int c = 0; c < 36 / CP; c++) prefetch_l2(nc + ((size_t)c * PG::VB + PG::VH) * CP, PG::VH * 16u);
    }
  }
  if (threadIdx.x == 32) {
    // fields read later in the block's life, requested into L2 once written
    grid_wait();
    for (int q = 0; q < tile; q++) {
      const int r = rhs0 + rt * tile + q;
      if (rt * tile + q >= nrhs) break;
      if (!self_zero) prefetch_l2((const char *)rp.out[r] + (size_t)b * PG::VB * SB, PG::VB * SB);
      if (!(mode & SAP_FROM_B)) prefetch_l2((const char *)ax.r[r] + (size_t)b * RB, RB);
      if ((mode & SAP_HALO_E) && q) prefetch_l2((const char *)ax.e[r] + (size_t)b * FB, FB);
    }
  }
  if (threadIdx.x < 32) tmem_alloc<PG::TCOLS>(smem_u32(tmem_at));
  tmem_sync();
  // lane threadIdx.x % 128 of the warp's sub-partition, 256 columns per 128 threads
  const uint32_t tm =
      *tmem_at + ((uint32_t)(32 * ((threadIdx.x / 32) % 4)) << 16) + (uint32_t)(threadIdx.x / 128) * 256u;
  constexpr uint32_t TI = 0, TO = 72, TX = 144, TXN = 54;   // A_ee^-1, A_oo, x-links of the even and odd half-step
  tm_st<32>(tm + TI, m0);
  tm_st<32>(tm + TI + 32, m0 + 32);
  tm_st<8>(tm + TI + 64, m0 + 64);
  tm_st<32>(tm + TO, m1);
  tm_st<32>(tm + TO + 32, m1 + 32);
  tm_st<8>(tm + TO + 64, m1 + 64);

  bool quit = false;
  if constexpr (Store<S>::prec == DD_F32) {
    const bool ok = mbar_wait(mbar_s, 0);
    if (__syncthreads_or(!ok)) {   // the staging wait expired: leave as a whole
      wait_expired(timeouts, mbar_s, 0);
      if (threadIdx.x == 0 && (mode & SAP_HALO_E)) mbar_wait(fbar_s, 0);   // its other copy in flight
      quit = true;
    }
  } else {
    // 16-bit links: converted on the way into shared memory, two quads at a time
    const uint4 *src = (const uint4 *)links + (size_t)b * (PG::LINKS / 2);
    for (int i0 = 0; i0 < PG::LINKS / 2; i0 += 6 * NT) {
      uint4 w[6];
#pragma unroll
      for (int i = 0; i < 6; i++) w[i] = __ldg(src + i0 + i * NT + threadIdx.x);
#pragma unroll
      for (int i = 0; i < 6; i++) {
        const P *p = (const P *)&w[i];
        quad *d = L + 2 * (i0 + i * NT + threadIdx.x);
#pragma unroll
        for (int e = 0; e < 2; e++) {
          const cpx<float> a = from_pair<float, P>(p[2 * e]), c = from_pair<float, P>(p[2 * e + 1]);
          constexpr float f = -0.5f / paired_scale<P>();
          d[e] = quad{pk(f * a.re, f * a.im), pk(f * c.re, f * c.im)};
        }
      }
    }
    static_assert(PG::LINKS / 2 == 18 * NT, "whole rounds of the link conversion");
    __syncthreads();
  }
  if (!quit) {
    {   // the row's x-links: the packed one (x = 0 and 2) and the single one (x = 1),
        // U where the half-step's hop is forward, its conjugate transpose where backward
      const quad *D = L + T.q * R + T.r, *E = L + (1 - T.q) * R + T.r;
      const bool q = T.q;
      uint32_t w0[54], w1[54];
#pragma unroll
      for (int r = 0; r < 3; r++)
#pragma unroll
        for (int c = 0; c < 3; c++) {
          const quad u = D[(3 * r + c) * ST], ud = D[(3 * c + r) * ST];
          const quad s = E[(3 * r + c) * ST], sd = E[(3 * c + r) * ST];
          const quad v = quad{ud.x, neg2(ud.y)};
          const quad e = q ? v : u, o = q ? u : v;
          const int i = 3 * r + c;
          w0[4 * i] = __float_as_uint(lo(e.x));
          w0[4 * i + 1] = __float_as_uint(hi(e.x));
          w0[4 * i + 2] = __float_as_uint(lo(e.y));
          w0[4 * i + 3] = __float_as_uint(hi(e.y));
          w1[4 * i] = __float_as_uint(lo(o.x));
          w1[4 * i + 1] = __float_as_uint(hi(o.x));
          w1[4 * i + 2] = __float_as_uint(lo(o.y));
          w1[4 * i + 3] = __float_as_uint(hi(o.y));
          const float fr = lo(s.x), fi = lo(s.y), br = lo(sd.x), bi = -lo(sd.y);
          w0[36 + 2 * i] = __float_as_uint(q ? fr : br);
          w0[37 + 2 * i] = __float_as_uint(q ? fi : bi);
          w1[36 + 2 * i] = __float_as_uint(q ? br : fr);
          w1[37 + 2 * i] = __float_as_uint(q ? bi : fi);
        }
#pragma unroll
      for (int p = 0; p < 2; p++) {
        const uint32_t a = tm + TX + p * TXN;
        const uint32_t *w = p ? w1 : w0;
        tm_st<32>(a, w);
        tm_st<16>(a + 32, w + 32);
        tm_st<4>(a + 48, w + 48);
        tm_st<2>(a + 52, w + 52);
      }
      tmem_wait_st();
    }
    int bc[4];
    block_coords(g, b, bc);
    grid_wait();   // the phases before have written x, the residuals and the flux
#pragma unroll 1
    for (int rr = 0; rr < tile; rr++) {
      if (rt * tile + rr >= nrhs) break;
      const int r = rhs0 + rt * tile + rr;
      // ---- the block residual: b or the stored one (zero on even sites after
      // the first sweep), minus the incoming flux
      u64 r_e[12], r_o[12];
      if (mode & SAP_FROM_B) {
        cpx<float> A[6], B[6];
        auto take = [&](int s, u64 *o) {
          if (mode & SAP_B32) half_ld<float>(rp.in[r], g, b, s, T.h, A, B);
          else half_ld<S>(rp.in[r], g, b, s, T.h, A, B);
#pragma unroll
          for (int i = 0; i < 6; i++) {
            o[2 * i] = pk(A[i].re, B[i].re);
            o[2 * i + 1] = pk(A[i].im, B[i].im);
          }
        };
        take(2 * T.r, r_e);
        take(PG::VH + 2 * T.r, r_o);
      } else {
        const char *res = (const char *)ax.r[r] + (size_t)b * RB;
#pragma unroll
        for (int i = 0; i < 6; i++) {
          const quad v = quad_of<S, true>(quad_raw<S, true>(res, i * NT + threadIdx.x));
          r_o[2 * i] = v.x;
          r_o[2 * i + 1] = v.y;
          r_e[2 * i] = r_e[2 * i + 1] = 0ull;
        }
      }
      if (mode & SAP_HALO_E) {
        // (the same for a warp, whose halves exchange below)
        const bool ok = __all_sync(0xffffffffu, mbar_wait(fbar_s, rr & 1));
        if (ok) {
          const char *H = (const char *)V;
          u64 d[2][12];
          flux_sum<S, SHAPE>(T, H, L, d[0], d[1]);
#pragma unroll
          for (int i = 0; i < 12; i++) {
            r_e[i] = sub2(r_e[i], d[0][i]);
            r_o[i] = sub2(r_o[i], d[1][i]);
          }
        }
        // the flux has been read by all (or a wait expired: leave as a whole)
        if (__syncthreads_or(!ok)) {
          wait_expired(timeouts, fbar_s, rr & 1);
          break;
        }
      }
      // ---- Schur right-hand side, MR steps, reconstruction: half-steps on
      // the even (p = 0) and odd (p = 1) sites in turn, one body of code.
      //   step 0: te = A_ee^-1 r_e; odd: rho = r_o - D_oe te
      //   steps k = 1..n_MR: even: te = A_ee^-1 D_eo rho; odd: p = A_oo rho -
      //     D_oe te, alpha = <p, rho> / <p, p>, e_o += alpha rho, rho -= alpha p
      //   reconstruction: e_e = A_ee^-1 (r_e - D_eo e_o) with e_o = sum_k alpha_k
      //     rho_k is step 0's te minus sum_k alpha_k (step k's te): the steps
      //     accumulate it, and no half-step is spent on D_eo e_o.
      u64 rh[12], eo[12], ee[12];
      uint32_t cl[72], xl[54];
      {
        u64 m[36];
        tm_issue72(tm + TI, cl);
        tm_wait72(cl);
#pragma unroll
        for (int i = 0; i < 36; i++) m[i] = word2(cl, i);
        herm6_pair<LAST>(m, r_e, ee);
        st6(T, V, R, ee);
      }
#pragma unroll
      for (int i = 0; i < 12; i++) {
        eo[i] = 0ull;
        rh[i] = r_o[i];
      }
      const int last = 2 * nmr + 1;
#pragma unroll 1
      for (int step = 1; step <= last; step++) {
        const int p = step & 1;   // 1: odd sites
        tm_issue54(tm + TX + p * TXN, xl);
        __syncthreads();
        PairAcc acc;
        hops_pair<SHAPE>(T, p, V + (1 - p) * PG::VEC, L, xl, acc);
        u64 hv[12], m[36];
        tm_issue72(tm + (p ? TO : TI), cl);
        to_chirality(T, acc, hv);
        tm_wait72(cl);
#pragma unroll
        for (int i = 0; i < 36; i++) m[i] = word2(cl, i);
        if (p) {
          if (step == 1) {
#pragma unroll
            for (int i = 0; i < 12; i++) rh[i] = sub2(rh[i], hv[i]);
          } else {
            u64 w[12];
            herm6_pair<LAST>(m, rh, w);
            u64 a = 0ull, c = 0ull, e = 0ull;
#pragma unroll
            for (int i = 0; i < 12; i++) w[i] = sub2(w[i], hv[i]);
#pragma unroll
            for (int i = 0; i < 6; i++) {   // <p, rho> (re, im) and <p, p>
              a = fma2(w[2 * i], rh[2 * i], a);
              c = fma2(w[2 * i], rh[2 * i + 1], c);
              e = fma2(w[2 * i], w[2 * i], e);
              a = fma2(w[2 * i + 1], rh[2 * i + 1], a);
              c = fma2(neg2(w[2 * i + 1]), rh[2 * i], c);
              e = fma2(w[2 * i + 1], w[2 * i + 1], e);
            }
            float pr = lo(a) + hi(a), pi = lo(c) + hi(c), pp = lo(e) + hi(e);
            cta_sum3<NT / 32>(pr, pi, pp, red);
            float ar = 0.f, ai = 0.f;
            if (pp > 0.f) {
              ar = pr / pp;
              ai = pi / pp;
            }
            const u64 Ar = pk(ar, ar), Ai = pk(ai, ai);
            u64 te[12];   // this thread's part of the step's te
            ld6(T, V, R, te);
#pragma unroll
            for (int i = 0; i < 6; i++) {
              eo[2 * i] = fma2(Ar, rh[2 * i], fma2(neg2(Ai), rh[2 * i + 1], eo[2 * i]));
              eo[2 * i + 1] = fma2(Ar, rh[2 * i + 1], fma2(Ai, rh[2 * i], eo[2 * i + 1]));
              ee[2 * i] = fma2(neg2(Ar), te[2 * i], fma2(Ai, te[2 * i + 1], ee[2 * i]));
              ee[2 * i + 1] = fma2(neg2(Ar), te[2 * i + 1], fma2(neg2(Ai), te[2 * i], ee[2 * i + 1]));
              rh[2 * i] = fma2(neg2(Ar), w[2 * i], fma2(Ai, w[2 * i + 1], rh[2 * i]));
              rh[2 * i + 1] = fma2(neg2(Ar), w[2 * i + 1], fma2(neg2(Ai), w[2 * i], rh[2 * i + 1]));
            }
          }
          if (step < last) st6(T, V + PG::VEC, R, rh);
        } else {
          u64 te[12];
          herm6_pair<LAST>(m, hv, te);
          st6(T, V, R, te);
        }
      }
      // ---- the residual for the block's next phase, the flux of e, x += e (x
      // is read ahead of the flux, whose arithmetic covers the wait)
      // (every thread is past its last hops at the sum's barrier; without MR steps there was none)
      if (nmr == 0) __syncthreads();
      st6(T, V, R, ee);
      st6(T, V + PG::VEC, R, eo);
      cpx<float> xe[2][6], xo[2][6];
      if (!self_zero) {
        half_ld<S>(rp.out[r], g, b, 2 * T.r, T.h, xe[0], xe[1]);
        half_ld<S>(rp.out[r], g, b, PG::VH + 2 * T.r, T.h, xo[0], xo[1]);
      }
      if (mode & SAP_WRITE_R) {
        char *res = (char *)ax.r[r] + (size_t)b * RB;
#pragma unroll
        for (int i = 0; i < 6; i++) quad_st<S, true>(res, i * NT + threadIdx.x, rh[2 * i], rh[2 * i + 1]);
      }
      if (mode & SAP_WRITE_E) {
        __syncthreads();
        char *H = (char *)ax.e[r];
        flux_out_x<S, SHAPE>(T, g, b, bc, L, V, H);
#pragma unroll
        for (int p = 0; p < 2; p++) {
          const quad *v = V + p * PG::VEC;
          u64 u[6], d[6], e[6];
          ld3(v + spin_at(R, T.h, T.r), R, u);
          ld3(v + spin_at(R, 2 + T.h, T.r), R, d);
          ld3(v + spin_at(R, 3 - T.h, T.r), R, e);
          flux_out<S, SHAPE, 1>(T, g, b, bc, L, p, u, d, e, H);
          flux_out<S, SHAPE, 2>(T, g, b, bc, L, p, u, d, e, H);
          flux_out<S, SHAPE, 3>(T, g, b, bc, L, p, u, d, e, H);
        }
        __syncwarp();
      }
      auto update = [&](int s, const quad *v, cpx<float>(*x)[6]) {
        u64 e[12];   // this thread's part of the correction
        ld6(T, v, R, e);
#pragma unroll
        for (int i = 0; i < 6; i++) {
          const cpx<float> a = {lo(e[2 * i]), lo(e[2 * i + 1])}, c = {hi(e[2 * i]), hi(e[2 * i + 1])};
          x[0][i] = self_zero ? a : cpx<float>{x[0][i].re + a.re, x[0][i].im + a.im};
          x[1][i] = self_zero ? c : cpx<float>{x[1][i].re + c.re, x[1][i].im + c.im};
        }
        half_st<S>(rp.out[r], g, b, s, T.h, x[0], x[1]);
      };
      update(2 * T.r, V, xe);
      update(PG::VH + 2 * T.r, V + PG::VEC, xo);
      __syncthreads();   // the shared vectors are reused by the next right-hand side
      if (threadIdx.x == 0 && (mode & SAP_HALO_E) && rr + 1 < tile && rt * tile + rr + 1 < nrhs) flux_issue(r + 1);
    }
  }
  // every thread's TMEM accesses are complete; the allocating warp frees
  tmem_wait_st();
  tmem_sync();
  if (threadIdx.x < 32) tmem_dealloc<PG::TCOLS>(*tmem_at);
}

}  // namespace
}  // namespace dd
