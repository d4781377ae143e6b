// FP32 stage kernel for 3D blocks of 8^3 cells at p = 1..3, written for the
// issue rate of sm_103a.
//
// It computes the same thing as k_stage (Sec. 2, Eqs. (3)-(5): volume
// integral with the contravariant fluxes, Lax-Friedrichs face fluxes, the
// diagonal inverse mass at the Gauss points, the SSP-RK stage combination
// and, on the last stage, the CFL minimum of Sec. 4.3) and the traces across
// same-level and outflow faces of Sec. 3.5, organised so that every
// instruction does twice the work and data stays in registers:
//
//  * Cell pairs.  A thread owns two x-neighbouring cells (i, i+1), i even,
//    and does its floating-point work on float2 pairs with the packed FP32
//    instructions (fma/add/mul .f32x2); shared-memory accesses are 8-byte
//    pairs.
//  * Warp = face point.  Warp w of the CTA handles one face-point index fp
//    (p+1)^2 warps: (q_y, q_z) in the x sweep, (q_x, q_z) in y, (q_x, q_y)
//    in z); its 32 lanes are the 32 cell pairs of a layer (lane = 4 j + m,
//    cells 2m, 2m+1 of row j).  x- and y-neighbour traces and face fluxes
//    move between lanes with warp shuffles; z-face fluxes are carried from
//    layer to layer by the lane that owns the column.
//  * No CTA barrier in the layer sweep.  The y lines at q_z read what the
//    x lines at that q_z wrote, the z lines at q_x what the y lines at that
//    q_x wrote: two barriers among p + 1 warps.  A warp copies the rows of
//    its own z lines two layers ahead (one at p = 3) by TMA as soon as it has
//    finished them, so there is no producer to wait for either.
//  * The block's own faces: their outer traces are read from the neighbours'
//    cells (terms prefetched a phase ahead), one lane per face point, and
//    their fluxes evaluated once, 32 lanes wide, before the x lines.
//
// What bounds it: instruction latency.  It issues on 45 % of the cycles with
// 4 to 5 warps a scheduler; registers and shared memory allow no more.
// Per stage with the traces, before (a guard pass writing all traces, CTA
// barriers; at p = 3 the layer-sweep kernel) and now: 4096 affine blocks,
// p = 1: 326 + 80 -> 274 us; p = 2: 1040 + 258 -> 1130 us; 512 blocks, p = 3:
// 514 + 76 -> 347 us.
//
// Per layer: x lines (volume flux, derivative, x faces, lift) -> residual
// in shared memory; y lines (+= the same along y); z lines (+= along z, the
// z face above against the next layer's trace, 1/J) -> stage combination
// straight to global memory, CFL minimum on the last stage.
#pragma once

#include "dg_device.cuh"

namespace dgf {
namespace pairk {

constexpr int kStatusTimeout = -5;

// ------------------------------------------------------------ float2 math
__device__ __forceinline__ float2 f2(float a) { return make_float2(a, a); }
__device__ __forceinline__ float2 add(float2 a, float2 b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ float2 mul(float2 a, float2 b) { return __fmul2_rn(a, b); }
__device__ __forceinline__ float2 fma2(float2 a, float2 b, float2 c) { return __ffma2_rn(a, b, c); }
__device__ __forceinline__ float2 sub(float2 a, float2 b) { return __ffma2_rn(b, make_float2(-1.f, -1.f), a); }
// The hardware's approximate reciprocal and root, subnormals flushed: a
// density below 1.2e-38 has an infinite reciprocal and the sound speed of a
// subnormal gamma p / rho is 0, so such states are outside what this kernel
// supports (a state that reaches them ends as non-finite).  Us a step without
// the flush and with it: 4096 affine blocks p = 1 878 -> 813, p = 2 3411 ->
// 3390, 512 blocks p = 3 991 -> 954, 71 curved blocks p = 2 170 -> 162.
__device__ __forceinline__ float rcpf(float a) {
  float r;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(a));
  return r;
}
__device__ __forceinline__ float rootf(float a) {
  float r;
  asm("sqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(a));
  return r;
}
// the larger one, NaN if either is
__device__ __forceinline__ float max_nan(float a, float b) {
  float r;
  asm("max.NaN.f32 %0, %1, %2;" : "=f"(r) : "f"(a), "f"(b));
  return r;
}
__device__ __forceinline__ float2 rcp2(float2 a) { return make_float2(rcpf(a.x), rcpf(a.y)); }
__device__ __forceinline__ float2 sqrt2(float2 a) { return make_float2(rootf(a.x), rootf(a.y)); }
__device__ __forceinline__ float2 abs2(float2 a) { return make_float2(fabsf(a.x), fabsf(a.y)); }
__device__ __forceinline__ float2 lds2(const float* p) { return *reinterpret_cast<const float2*>(p); }
__device__ __forceinline__ void sts2(float* p, float2 v) { *reinterpret_cast<float2*>(p) = v; }
__device__ __forceinline__ float2 shfl_up2(float2 v, int d) {
  return make_float2(__shfl_up_sync(0xffffffffu, v.x, d), __shfl_up_sync(0xffffffffu, v.y, d));
}
__device__ __forceinline__ float2 shfl_down2(float2 v, int d) {
  return make_float2(__shfl_down_sync(0xffffffffu, v.x, d), __shfl_down_sync(0xffffffffu, v.y, d));
}

// ------------------------------------------------- TMA bulk copy, mbarrier
__device__ __forceinline__ uint32_t smem_addr(const void* p) {
  return (uint32_t)__cvta_generic_to_shared(p);
}
__device__ __forceinline__ void mbar_init(uint64_t* bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_addr(bar)), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_fence_init() {
  asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}
__device__ __forceinline__ void mbar_arrive_expect(uint64_t* bar, uint32_t bytes) {
  asm volatile("{ .reg .b64 st; mbarrier.arrive.expect_tx.shared::cta.b64 st, [%0], %1; }" ::"r"(smem_addr(bar)),
               "r"(bytes)
               : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint64_t* bar) {
  asm volatile("{ .reg .b64 st; mbarrier.arrive.shared::cta.b64 st, [%0]; }" ::"r"(smem_addr(bar)) : "memory");
}
// one 256-byte row global -> shared, completing on bar (plain, not multicast)
__device__ __forceinline__ void bulk_row(float* dst, const float* src, uint32_t bytes, uint64_t* bar) {
  asm volatile(
      "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
          smem_addr(dst)),
      "l"(src), "r"(bytes), "r"(smem_addr(bar))
      : "memory");
}
// earlier generic-proxy reads of a buffer are ordered before the async
// proxy's writes into it
__device__ __forceinline__ void fence_proxy_async() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }
// bulk prefetch of a global row into L2 (no completion to wait for)
__device__ __forceinline__ void prefetch_row_l2(const float* src, uint32_t bytes) {
  asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(src), "r"(bytes) : "memory");
}
// bounded wait for the phase with the given parity; false if it gave up.
// The retry loop is a single asm statement, so that the compiler keeps its
// register allocation across the wait (a C++ loop around try_wait made it
// spill the live state of the z sweep).
__device__ __forceinline__ bool mbar_wait(uint64_t* bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\t.reg .u32 c;\n\t"
      "mov.u32 c, 0;\n\t"
      "mov.u32 %0, 0;\n"
      "LAB_WAIT:\n\t"
      "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
      "@p bra LAB_DONE;\n\t"
      "add.u32 c, c, 1;\n\t"
      "setp.lt.u32 p, c, %3;\n\t"
      "@p bra LAB_WAIT;\n\t"
      "bra LAB_END;\n"
      "LAB_DONE:\n\t"
      "mov.u32 %0, 1;\n"
      "LAB_END:\n\t"
      "}"
      : "=r"(ok)
      : "r"(smem_addr(bar)), "r"(parity), "r"(1u << 22)
      : "memory");
  return ok != 0;
}

// keeps the compiler from merging two evaluations of the same metric (one
// for the face normals before the face fluxes, one for the volume points
// after them), so the metric is not held in registers across the fluxes
__device__ __forceinline__ void reload_fence() { asm volatile("" ::: "memory"); }

// ------------------------------------------------------------- Euler, x2
// AX >= 0: the area vector a has the one component AX (axis-aligned blocks);
// the terms left out are exact zeros.
template <int AX>
__device__ __forceinline__ float2 dot2(const float2 (&u)[5], const float2 (&a)[3]) {
  if constexpr (AX >= 0) return mul(u[1 + AX], a[AX]);
  return fma2(u[3], a[2], fma2(u[2], a[1], mul(u[1], a[0])));
}
// F . a for a pair of states (Eq. (2))
template <int AX>
__device__ __forceinline__ void flux2(const float2 (&u)[5], const float2 (&a)[3], float2 gm1, float2 (&F)[5]) {
  const float2 ri = rcp2(u[0]);
  const float2 mn = dot2<AX>(u, a);
  const float2 ke = fma2(u[3], u[3], fma2(u[2], u[2], mul(u[1], u[1])));
  const float2 vn = mul(mn, ri);
  const float2 pr = mul(gm1, fma2(mul(ke, ri), f2(-0.5f), u[4]));
  F[0] = mn;
#pragma unroll
  for (int j = 0; j < 3; ++j) F[1 + j] = AX < 0 || AX == j ? fma2(u[1 + j], vn, mul(pr, a[j])) : mul(u[1 + j], vn);
  F[4] = mul(add(u[4], pr), vn);
}

// Lax-Friedrichs flux (Eq. (5), dissipative sign) for two face points at
// once; a = area vector from L to R.  Both physical fluxes are summed into
// the result term by term (fewer live registers than forming F(U_L) and
// F(U_R) first).  A NaN wave speed (negative density or pressure)
// propagates into the flux, as in lf_flux.  an = |a|.
template <int AX>
__device__ __forceinline__ void lf2(const float2 (&uL)[5], const float2 (&uR)[5], const float2 (&a)[3], float2 an,
                                    float2 gam, float2 gm1, float2 (&Fh)[5]) {
  const float2 riL = rcp2(uL[0]), riR = rcp2(uR[0]);
  const float2 mnL = dot2<AX>(uL, a), mnR = dot2<AX>(uR, a);
  const float2 keL = fma2(uL[3], uL[3], fma2(uL[2], uL[2], mul(uL[1], uL[1])));
  const float2 keR = fma2(uR[3], uR[3], fma2(uR[2], uR[2], mul(uR[1], uR[1])));
  const float2 vL = mul(mnL, riL), vR = mul(mnR, riR);
  const float2 pL = mul(gm1, fma2(mul(keL, riL), f2(-0.5f), uL[4]));
  const float2 pR = mul(gm1, fma2(mul(keR, riR), f2(-0.5f), uR[4]));
  const float2 sL = fma2(sqrt2(mul(mul(gam, pL), riL)), an, abs2(vL));
  const float2 sR = fma2(sqrt2(mul(mul(gam, pR), riR)), an, abs2(vR));
  const float2 al = make_float2(max_nan(sL.x, sR.x), max_nan(sL.y, sR.y));
  const float2 h = f2(0.5f);
  const float2 pp = add(pL, pR);
  Fh[0] = mul(h, fma2(al, sub(uL[0], uR[0]), add(mnL, mnR)));
#pragma unroll
  for (int j = 0; j < 3; ++j) {
    const float2 R = AX < 0 || AX == j ? fma2(uR[1 + j], vR, mul(pp, a[j])) : mul(uR[1 + j], vR);
    Fh[1 + j] = mul(h, fma2(al, sub(uL[1 + j], uR[1 + j]), fma2(uL[1 + j], vL, R)));
  }
  Fh[4] = mul(h, fma2(al, sub(uL[4], uR[4]), fma2(add(uL[4], pL), vL, mul(add(uR[4], pR), vR))));
}

__device__ __forceinline__ float2 norm2(const float2 (&a)[3]) {
  return sqrt2(fma2(a[2], a[2], fma2(a[1], a[1], mul(a[0], a[0]))));
}

// The same for one face point.  split: with the two sides' fluxes rounded
// before they are added and 1/2 |m|^2 / rho in one rounding, as lf_flux does;
// the block's upper x face keeps those roundings, so that an affine block's
// states stay the same bit for bit.
__device__ __forceinline__ void lf1(const float (&uL)[5], const float (&uR)[5], const float (&a)[3], float an, float gam,
                                    float gm1, bool split, float (&Fh)[5]) {
  const float riL = rcpf(uL[0]), riR = rcpf(uR[0]);
  const float mnL = fmaf(uL[3], a[2], fmaf(uL[2], a[1], uL[1] * a[0]));
  const float mnR = fmaf(uR[3], a[2], fmaf(uR[2], a[1], uR[1] * a[0]));
  const float keL = fmaf(uL[3], uL[3], fmaf(uL[2], uL[2], uL[1] * uL[1]));
  const float keR = fmaf(uR[3], uR[3], fmaf(uR[2], uR[2], uR[1] * uR[1]));
  const float vL = mnL * riL, vR = mnR * riR;
  const float pL = gm1 * (split ? fmaf(-0.5f * keL, riL, uL[4]) : fmaf(keL * riL, -0.5f, uL[4]));
  const float pR = gm1 * (split ? fmaf(-0.5f * keR, riR, uR[4]) : fmaf(keR * riR, -0.5f, uR[4]));
  const float al = max_nan(fmaf(rootf(gam * pL * riL), an, fabsf(vL)), fmaf(rootf(gam * pR * riR), an, fabsf(vR)));
  const float pp = pL + pR;
  Fh[0] = 0.5f * fmaf(al, uL[0] - uR[0], split ? fmaf(uL[0], vL, __fmul_rn(uR[0], vR)) : mnL + mnR);
#pragma unroll
  for (int j = 0; j < 3; ++j) {
    const float two = __fadd_rn(fmaf(uL[1 + j], vL, __fmul_rn(pL, a[j])), fmaf(uR[1 + j], vR, __fmul_rn(pR, a[j])));
    const float one = fmaf(uL[1 + j], vL, fmaf(uR[1 + j], vR, __fmul_rn(pp, a[j])));
    Fh[1 + j] = 0.5f * fmaf(al, uL[1 + j] - uR[1 + j], split ? two : one);
  }
  Fh[4] = 0.5f * fmaf(al, uL[4] - uR[4], fmaf(uL[4] + pL, vL, __fmul_rn(uR[4] + pR, vR)));
}

// the 1D tables with every entry twice, so that a packed instruction reads
// one as an operand instead of building the pair in registers
template <int N>
struct PairTab {
  float2 lm[N], lp[N], lmw[N], lpwn[N], Sh[N][N];  // lpwn = -l_q(+1) / w_q
};
template <int N>
PairTab<N> pair_tab(const Tab<N, float>& T) {
  PairTab<N> t;
  for (int q = 0; q < N; ++q) {
    t.lm[q] = make_float2(T.lm[q], T.lm[q]);
    t.lp[q] = make_float2(T.lp[q], T.lp[q]);
    t.lmw[q] = make_float2(T.lmw[q], T.lmw[q]);
    t.lpwn[q] = make_float2(-T.lpw[q], -T.lpw[q]);
    for (int j = 0; j < N; ++j) t.Sh[q][j] = make_float2(T.Sh[q][j], T.Sh[q][j]);
  }
  return t;
}

// Metric along a line in direction DIR for a pair of cells (see LineGeo):
// J dxi_DIR/dx (s) = c0 + c1 s + c2 s^2, J(s) = e . (J dxi_DIR/dx)(s), from
// the trilinear coefficients of both cells in shared memory ([21][64]).
template <int DIR>
struct LineGeo2 {
  float2 c0[3], c1[3], c2[3], e[3];
  __device__ __forceinline__ void init(const float* __restrict__ G, int cl, const float (&xi)[3], int stride = 64) {
    float2 al[3][3], be[3][3];
#pragma unroll
    for (int a = 0; a < 3; ++a)
#pragma unroll
      for (int j = 0; j < 3; ++j) al[a][j] = be[a][j] = f2(0.f);
#pragma unroll
    for (int c = 1; c < 8; ++c) {
#pragma unroll
      for (int j = 0; j < 3; ++j) {
        const float2 x = lds2(G + ((c - 1) * 3 + j) * stride + cl);
#pragma unroll
        for (int a = 0; a < 3; ++a) {
          if (!((c >> a) & 1)) continue;
          float fac = 1.f;
          bool has_s = false;
#pragma unroll
          for (int bb = 0; bb < 3; ++bb) {
            if (bb == a || !((c >> bb) & 1)) continue;
            if (bb == DIR) has_s = true;
            else fac *= xi[bb];
          }
          if (has_s) be[a][j] = fma2(x, f2(fac), be[a][j]);
          else al[a][j] = fma2(x, f2(fac), al[a][j]);
        }
      }
    }
#pragma unroll
    for (int j = 0; j < 3; ++j) e[j] = al[DIR][j];
    constexpr int i1 = (DIR + 1) % 3, i2 = (DIR + 2) % 3;
#pragma unroll
    for (int j = 0; j < 3; ++j) {
      const int j1 = (j + 1) % 3, j2 = (j + 2) % 3;
      c0[j] = sub(mul(al[i1][j1], al[i2][j2]), mul(al[i1][j2], al[i2][j1]));
      c1[j] = add(sub(mul(al[i1][j1], be[i2][j2]), mul(al[i1][j2], be[i2][j1])),
                  sub(mul(be[i1][j1], al[i2][j2]), mul(be[i1][j2], al[i2][j1])));
      c2[j] = sub(mul(be[i1][j1], be[i2][j2]), mul(be[i1][j2], be[i2][j1]));
    }
  }
  __device__ __forceinline__ void at(float s, float2 (&Ja)[3]) const {
#pragma unroll
    for (int j = 0; j < 3; ++j) Ja[j] = fma2(f2(s), fma2(f2(s), c2[j], c1[j]), c0[j]);
  }
  __device__ __forceinline__ float2 jac(const float2 (&Ja)[3]) const {
    return fma2(e[2], Ja[2], fma2(e[1], Ja[1], mul(e[0], Ja[0])));
  }
};

// J dxi_DIR/dx of a pair of cells at one point (a face: xi[DIR] = -1 or 1),
// from the tangents along the other two axes; half the work of a LineGeo2.
// The face normals take this and the volume points LineGeo2 afterwards, so
// that a line's metric is not held in registers across the face flux.
template <int DIR>
__device__ __forceinline__ void face_row2(const float* __restrict__ G, int cl, const float (&xi)[3], float2 (&Ja)[3],
                                          int stride = 64) {
  constexpr int i1 = (DIR + 1) % 3, i2 = (DIR + 2) % 3;
  float2 t1[3], t2[3];
#pragma unroll
  for (int j = 0; j < 3; ++j) {
    auto X = [&](int c) { return lds2(G + ((c - 1) * 3 + j) * stride + cl); };
    const float2 mix = fma2(X(7), f2(xi[DIR]), X((1 << i1) | (1 << i2)));
    t1[j] = fma2(mix, f2(xi[i2]), fma2(X((1 << i1) | (1 << DIR)), f2(xi[DIR]), X(1 << i1)));
    t2[j] = fma2(mix, f2(xi[i1]), fma2(X((1 << i2) | (1 << DIR)), f2(xi[DIR]), X(1 << i2)));
  }
#pragma unroll
  for (int j = 0; j < 3; ++j) {
    const int j1 = (j + 1) % 3, j2 = (j + 2) % 3;
    Ja[j] = sub(mul(t1[j1], t2[j2]), mul(t1[j2], t2[j1]));
  }
}

// barrier among the N warps of a group (hardware barriers 1 .. 2 N)
template <int THREADS>
__device__ __forceinline__ void group_sync(int id) {
  asm volatile("bar.sync %0, %1;" ::"r"(id), "n"(THREADS) : "memory");
}

// V selects the CTA shape at p = 1; one shape at p = 2 and 3
template <int P, int V = 0>
struct PairCfg {
  static constexpr int N = P + 1, Q = N * N * N, NFP = N * N, NV = 5;
  static constexpr int NT = 32 * NFP;  // one warp per face point
  static constexpr int ROWS = NV * Q;  // 256-byte state rows of a layer
  static constexpr int OWN = NV * N;   // of them, the rows of one warp's z lines
  static constexpr int NG = 21;        // trilinear coefficient rows of a layer
  // state layers in shared memory: two at p <= 2; at p = 3 a layer is 80 KB
  // and one (with the residual layer) is what fits
  static constexpr int ST = P <= 2 ? 2 : 1;
  // U^n of a z line's points: loaded into registers before the combination
  // (p = 1 with 128 registers), else copied by TMA into the residual rows the
  // warp has read.  Per stage at 4096 blocks (both sides
  // before the axis-aligned instantiation), p = 1: 277 us in registers, 297
  // by TMA; p = 2: 1240 us (spilled registers; spills miss the small L1 that
  // the shared memory leaves), 1143 us by TMA; 512 blocks, p = 3: 406, 361 us.
  static constexpr bool UNREG = P == 1 && V == 0;
  // variables of the carried z-face flux that wait for the z lines in shared
  // memory instead of in registers: what is free beside the layers
  static constexpr int park(bool aff) { return aff && P == 2 ? 4 : 5; }
  // shared memory: ST state layers, the residual layer, 2 geometry layers of
  // a curved block, the parked fluxes
  static constexpr size_t smem(bool aff) {
    return (size_t)((ST + 1) * ROWS * 64 + (aff ? 0 : 2 * NG * 64) + park(aff) * 2 * NT) * sizeof(float);
  }
  // Resident CTAs per SM.  Affine blocks: 2 at p = 2 (about 112 KB of shared
  // memory each, 96 registers), at p = 1 four (128 registers) or five (V = 1,
  // 96 registers, more warps; the autotuner times both), one of 16 warps with
  // 128 registers at p = 3.  Curved blocks hold the metric of a line too and
  // spilled 740 to 1020 bytes in these shapes, so they take fewer CTAs with
  // 168 registers: one at p = 2, three (V = 1: two) at p = 1.  Per stage, 71
  // curved blocks p = 2 59.5 -> 50.2 us, 216 blocks 144 -> 133 us, p = 1 49.4
  // -> 38.8 us.
  static constexpr int minb(bool aff) {
    return P <= 1 ? (aff ? (V ? 5 : 4) : (V ? 2 : 3)) : P == 2 ? (aff ? 2 : 1) : 1;
  }
};

}  // namespace pairk

// GEO: 0 blocks of any shape, 1 every block of the forest affine (no per-cell
// geometry is read, the curved code is not compiled), 2 every block affine
// and axis-aligned (one component of each area vector)
// BATCH: one launch for every forest of a batch (A.members; the tables and
// stage coefficients of A are common to all of them).
template <int P, bool MORTAR, int GEO, bool BATCH = false, int V = 0>
__global__ void __launch_bounds__(pairk::PairCfg<P, V>::NT, pairk::PairCfg<P, V>::minb(GEO != 0))
    k_stage_pair(const __grid_constant__ StageArgs<3, P, float> A, const __grid_constant__ pairk::PairTab<P + 1> T2) {
  static_assert(!(BATCH && MORTAR), "batches run without the mortar repair");
  constexpr bool AFF = GEO != 0, DIAG = GEO == 2;
  constexpr int AX = DIAG ? 0 : -1, AY = DIAG ? 1 : -1, AZ = DIAG ? 2 : -1;
  using namespace pairk;
  using C = PairCfg<P, V>;
  constexpr int N = C::N, Q = C::Q, NFP = C::NFP, NV = 5, ROWS = C::ROWS, NG = C::NG;
  constexpr int n = 8, LAY = 64, nc = 512, nt = 64;
  const auto& T = A.T;
  const int tid = threadIdx.x;
  const int w = tid >> 5, lane = tid & 31;
  const int m = lane & 3, j = lane >> 2;  // cell pair (2m, 2m+1) of row j
  const int i0 = 2 * m;
  const int cl = i0 + n * j;              // first cell of the pair in the layer
  const int fa = w % N, fb = w / N;       // digits of this warp's face point
  if (!BATCH && A.mode == 0 && *A.dtp == 0.0) return;  // t_end reached: identity, nothing evaluated

  constexpr int ST = C::ST, OWN = C::OWN;
  extern __shared__ __align__(128) unsigned char smem_raw[];
  float* Us = reinterpret_cast<float*>(smem_raw);  // [ST][ROWS][64]
  float* Rs = Us + ST * ROWS * LAY;                // [ROWS][64]
  constexpr int PK = C::park(AFF);
  float* Fs = Rs + ROWS * LAY;                     // [PK][NT][2]
  float* Gs = Fs + PK * 2 * C::NT;                 // [2][NG][64], curved blocks
  // unbar[w]: U^n rows of warp w's z lines;
  // full[s][g]: the state rows of z-line owners N g .. N g + N - 1 have
  // arrived in layer buffer s; gfull[s]: the geometry rows; zdone: every
  // warp has finished the z lines of a layer
  __shared__ __align__(8) uint64_t full[ST][N], gfull[2], zdone, unbar[NFP];
  __shared__ float sam[10], san[3];  // affine block: rows of J dxi/dx and 1/J; the rows' norms
  __shared__ int strd[6][8];  // face-trace descriptors of the block
  __shared__ int sdirect;     // faces whose trace is evaluated here (bit f)
  // batch: the item's forest and block.  The layer sweep reads the pointers
  // here where it uses them; kept in registers they spilled (p = 2)
  struct Item {
    const float *U, *Ub, *Unb, *Geo, *Tb, *Hb;
    float* Ob;
    unsigned long long* lam;
    int* status;
    float dt;
  };
  __shared__ Item sit;

  const float2 gam = f2(A.gamma), gm1 = f2(A.gamma - 1.f);
  float2 dt2 = f2(BATCH ? 0.f : (float)*A.dtp);  // per forest of a batch: per item
  const float2 ca2 = f2(A.ca), cb2 = f2(A.cb);
  float xq[N];
#pragma unroll
  for (int q = 0; q < N; ++q) xq[q] = T.x[q];
  // Gauss points of this warp's face-point digits (selected, not indexed, so
  // that nothing lives in local memory)
  float xa = xq[0], xb = xq[0];
#pragma unroll
  for (int q = 1; q < N; ++q) {
    xa = fa == q ? xq[q] : xa;
    xb = fb == q ? xq[q] : xb;
  }

  if (tid == 0) {
    for (int i = 0; i < ST * N; ++i) mbar_init(&full[0][0] + i, N);
    mbar_init(&gfull[0], 1);
    mbar_init(&gfull[1], 1);
    mbar_init(&zdone, NFP);
    for (int i = 0; i < NFP; ++i) mbar_init(&unbar[i], 1);
    mbar_fence_init();
  }
  __syncthreads();
  const int og = w / N;        // owner group of this warp's z lines (its q_y = fb)
  // layers this CTA has finished (geometry buffer L & 1, zdone phase L) and
  // state-buffer uses (buffer F % ST, use F / ST): a chunk below another one
  // also uses a buffer for the layer above it
  uint32_t L = 0, F = 0;
  bool fail = false;           // a bounded wait gave up: wait for nothing more
  auto wait_for = [&](uint64_t* bar, uint32_t parity) {
    if (!fail && !mbar_wait(bar, parity)) fail = true;
  };
  const bool use_un = A.mode == 0 && A.ca != 0.f;
  float lam_min = 3.0e38f;
  bool bad = false;

  const int items = BATCH ? __ldg(&A.istart[A.nmem]) : A.nL * A.nchunks;
  for (int item = blockIdx.x; item < items; item += gridDim.x) {
    // the forest of this item (a batch member, or the one forest)
    const StageArgs<3, P, float>* Mp = &A;
    int li = item;
    if constexpr (BATCH) {
      const int mi = batch_member(A.istart, A.nmem, item);
      Mp = A.members + mi;
      li = item - __ldg(&A.istart[mi]);
      if (A.mode == 0 && *Mp->dtp == 0.0) continue;  // that forest has reached its end time
    }
    const StageArgs<3, P, float>& M = *Mp;
    const int b = li / M.nchunks;
    const int chunk = li - b * M.nchunks;
    const int k0 = chunk * M.zchunk;
    const int k1 = min(n, k0 + M.zchunk);
    const size_t boff = (size_t)b * NV * Q * nc;
    const float* __restrict__ Ub = M.U + boff;
    const float* __restrict__ Unb = M.Un + boff;
    const float* __restrict__ Geo = M.geo + (size_t)b * NG * nc;
    const float* __restrict__ Tb = M.gtr + (size_t)b * 6 * NV * NFP * nt;
    const float* __restrict__ Hb = M.hcell + (size_t)b * nc;
    float* __restrict__ Ob = M.Uout + boff;
    const bool aff = AFF || M.affine[b] != 0;
    const int fmask = MORTAR ? M.fluxmask[b] : 0;
    // A warp copies the state rows of its own z lines of layer k into buffer
    // s: it is the last to read those rows of the layer that was there (the x
    // and y lines that read them come before its z lines through the group
    // barriers).  Warp 0 copies the geometry rows.
    auto issue = [&](int k, int s, const float* u, const float* un) {
      uint64_t* bar = &full[s][og];
      if (lane == 0) mbar_arrive_expect(bar, OWN * LAY * sizeof(float));
      __syncwarp();
      if (lane < OWN) {
        const int r = (lane / N) * Q + w + NFP * (lane % N);
        fence_proxy_async();
        bulk_row(Us + (s * ROWS + r) * LAY, u + (size_t)r * nc + k * LAY, LAY * sizeof(float), bar);
        // U^n of the same layer, read by the stage combination
        if (A.ca != 0.f) prefetch_row_l2(un + (size_t)r * nc + k * LAY, LAY * sizeof(float));
      }
    };
    // An affine block has none to copy, yet completes the phase: buffer and
    // parity are taken from L, which every layer advances, so one that left
    // its phase open would put the curved blocks behind it out of step.
    auto issue_geo = [&](int k, int s, const float* geo) {
      if (AFF || w != 0) return;
      if (aff) {
        if (lane == 0) mbar_arrive(&gfull[s]);
        return;
      }
      if (lane == 0) mbar_arrive_expect(&gfull[s], NG * LAY * sizeof(float));
      __syncwarp();
      if (lane < NG) {
        fence_proxy_async();
        bulk_row(Gs + (s * NG + lane) * LAY, geo + (size_t)lane * nc + k * LAY, LAY * sizeof(float), &gfull[s]);
      }
    };
#define GTR(f, v, fp, t) pTb()[(((size_t)(f) * NV + (v)) * NFP + (fp)) * nt + (t)]

    __syncthreads();  // the previous item is done with every buffer
    if (aff && tid < 10) sam[tid] = M.ameta[(size_t)b * 10 + tid];
    if (aff && tid < 3) {
      const float* r = M.ameta + (size_t)b * 10 + 3 * tid;
      san[tid] = rootf(fmaf(r[2], r[2], fmaf(r[1], r[1], r[0] * r[0])));
    }
    if constexpr (BATCH) {
      if (tid == 97) sit = Item{M.U, Ub, Unb, Geo, Tb, Hb, Ob, M.lam_bits, M.status, (float)*M.dtp};
    }
    auto pU = [&]() { return BATCH ? sit.U : A.U; };
    auto pUb = [&]() { return BATCH ? sit.Ub : Ub; };
    auto pUnb = [&]() { return BATCH ? sit.Unb : Unb; };
    auto pGeo = [&]() { return BATCH ? sit.Geo : Geo; };
    auto pTb = [&]() { return BATCH ? sit.Tb : Tb; };
    if (tid >= 32 && tid < 80) (&strd[0][0])[tid - 32] = __ldg(&M.trd[(size_t)b * 48 + tid - 32]);
    if (tid == 96) {
      int mask = 0;
#pragma unroll
      for (int f = 0; f < 6; ++f) {
        const int kd = __ldg(&M.kind[b * 6 + f]);
        mask |= (kd == 0 || kd == 3) ? 1 << f : 0;
      }
      sdirect = mask;
    }
    // Trace of a same-level or outflow face straight from the neighbour's
    // cells of the stage input (the descriptor of the guard kernel, the same
    // sum in the same order): the guard pass read a whole state copy a stage
    // for them, since a face cell's 32-byte sector holds a row of cells.
    auto face_base = [&](int f, int g0, int g1) -> size_t {
      const int* e = strd[f];
      return (size_t)e[0] * (NV * Q * nc) + (size_t)(e[1] + g0 * e[2] + g1 * e[3] + e[4] + fa * e[5] + fb * e[6]);
    };
    auto face_pair = [&](int f, int g0, int g1, float2 (&t)[NV]) {  // guard cells (g0, g1), (g0 + 1, g1)
      const float* __restrict__ src = pU() + face_base(f, g0, g1);
      const int pn = strd[f][7] >> 1, up = strd[f][7] & 1, d = strd[f][2];
#pragma unroll
      for (int v = 0; v < NV; ++v) {
        float2 acc = f2(0.f);
#pragma unroll
        for (int qn = 0; qn < N; ++qn) {
          const float* x = src + v * (Q * nc) + qn * pn;
          acc = fma2(up ? T2.lp[qn] : T2.lm[qn], make_float2(__ldg(x), __ldg(x + d)), acc);
        }
        t[v] = acc;
      }
    };
    // layers whose rows are wanted: the chunk's, and with two buffers the one
    // above it (its bottom trace; with one buffer that is read from memory)
    const int kend = ST == 2 ? min(n, k1 + 1) : k1;
    for (int i = 0; i < ST; ++i)
      if (k0 + i < kend) issue(k0 + i, (F + i) % ST, Ub, Unb);
    issue_geo(k0, L & 1, Geo);
    if (k0 + 1 < k1) issue_geo(k0 + 1, (L + 1) & 1, Geo);
    __syncthreads();  // the block's tables are there
    if (!aff) wait_for(&gfull[L & 1], (L >> 1) & 1);
    wait_for(&full[F % ST][og], (F / ST) & 1);

    // ------------------------------------ z face below the first layer
    // (the carried flux of an unchunked sweep: the layer below's top trace
    // and metric against this layer's bottom trace, or the guard trace)
    const int fpZ = w;  // (q_x, q_y) = (fa, fb)
    float2 Fbot[NV];
    auto park = [&]() {
#pragma unroll
      for (int v = 0; v < PK; ++v) sts2(Fs + (v * C::NT + tid) * 2, Fbot[v]);
    };
    auto unpark = [&]() {
#pragma unroll
      for (int v = 0; v < PK; ++v) Fbot[v] = lds2(Fs + (v * C::NT + tid) * 2);
    };
    {
      const float* Uc = Us + (F % ST) * ROWS * LAY;
      float2 tm[NV], tl[NV];
#pragma unroll
      for (int v = 0; v < NV; ++v) {
        float2 s = f2(0.f);
#pragma unroll
        for (int qz = 0; qz < N; ++qz) s = fma2(T2.lm[qz], lds2(Uc + (v * Q + fpZ + NFP * qz) * LAY + cl), s);
        tm[v] = s;
      }
      float2 Ja[3];
      if (k0 == 0) {
#pragma unroll
        for (int v = 0; v < NV; ++v) tl[v] = f2(0.f);
        if (sdirect & 16) {
          face_pair(4, i0, j, tl);
        } else {
#pragma unroll
          for (int v = 0; v < NV; ++v) tl[v] = lds2(&GTR(4, v, fpZ, cl));
        }
        if (aff) {
#pragma unroll
          for (int jj = 0; jj < 3; ++jj) Ja[jj] = f2(sam[6 + jj]);
        } else {
          const float xi[3] = {xa, xb, -1.f};
          face_row2<2>(Gs + (L & 1) * NG * LAY, cl, xi, Ja);
        }
      } else {
        const float* Ul = pUb() + (k0 - 1) * LAY + cl;  // the layer below, from memory
#pragma unroll
        for (int v = 0; v < NV; ++v) {
          float2 s = f2(0.f);
#pragma unroll
          for (int qz = 0; qz < N; ++qz)
            s = fma2(T2.lp[qz], __ldg(reinterpret_cast<const float2*>(Ul + (size_t)(v * Q + fpZ + NFP * qz) * nc)), s);
          tl[v] = s;
        }
        if (aff) {
#pragma unroll
          for (int jj = 0; jj < 3; ++jj) Ja[jj] = f2(sam[6 + jj]);
        } else {
          const float xi[3] = {xa, xb, 1.f};
          face_row2<2>(pGeo() + (k0 - 1) * LAY, cl, xi, Ja, nc);
        }
      }
      lf2<AZ>(tl, tm, Ja, aff ? f2(san[2]) : norm2(Ja), gam, gm1, Fbot);
      if (MORTAR && k0 == 0 && (fmask & 16)) {
#pragma unroll
        for (int v = 0; v < NV; ++v) Fbot[v] = tl[v];  // the z- face flux itself
      }
      park();
    }

    // Traces across the block's x and y faces, one guard cell per lane: lane
    // 8 f + g holds face f's at cell g of the layer (g = row for the x faces,
    // column for the y faces) and this warp's face point, sum_q l_q u_q over
    // the N points along the face's axis (a level jump's or a prescribed
    // state's trace comes whole from the guard pass).  A layer's terms are
    // loaded a phase of the layer below apart, each a phase before it is
    // summed, so the loads' latency stays behind the arithmetic (loading them
    // together at the layer's start cost 275 us of 1355 at 4096 blocks, p = 2).
    const int ef = lane >> 3, eg = lane & 7;
    const bool edirect = (sdirect >> ef) & 1;
    float ev[NV], ea[NV], ex[NV], ex2[N == 4 ? NV : 1];
    auto edge_load = [&](int qn, int kk, float (&x)[NV]) {
      if (edirect) {
        const float* __restrict__ src = pU() + face_base(ef, eg, kk) + qn * (strd[ef][7] >> 1);
#pragma unroll
        for (int v = 0; v < NV; ++v) x[v] = __ldg(src + v * (Q * nc));
      } else if (qn == N - 1) {
#pragma unroll
        for (int v = 0; v < NV; ++v) x[v] = GTR(ef, v, w, eg + n * kk);
      } else {
#pragma unroll
        for (int v = 0; v < NV; ++v) x[v] = 0.f;
      }
    };
    auto edge_sum = [&](int qn) {
      const float l = edirect ? ((strd[ef][7] & 1) ? T.lp[qn] : T.lm[qn]) : (qn == N - 1 ? 1.f : 0.f);
#pragma unroll
      for (int v = 0; v < NV; ++v) ea[v] = qn == 0 ? l * ex[v] : fmaf(l, ex[v], ea[v]);
    };
#pragma unroll
    for (int qn = 0; qn < N; ++qn) {
      edge_load(qn, k0, ex);
      edge_sum(qn);
    }
#pragma unroll
    for (int v = 0; v < NV; ++v) ev[v] = ea[v];

    for (int k = k0; k < k1; ++k) {
      const float* Uc = Us + (F % ST) * ROWS * LAY;
      const float* Gc = Gs + (L & 1) * NG * LAY;
      // this warp's x lines read rows of the owners with q_y = fa, its edge
      // traces (and y lines) rows of every owner
#pragma unroll
      for (int g = 0; g < N; ++g) wait_for(&full[F % ST][g], (F / ST) & 1);
      if (!aff) wait_for(&gfull[L & 1], (L >> 1) & 1);
      // the last term of this layer's edge traces, the first of the next one's
      const bool more = k + 1 < k1;
      if (k > k0) {
        if constexpr (N == 3) edge_sum(2);
        if constexpr (N == 4) {
          edge_sum(2);
#pragma unroll
          for (int v = 0; v < NV; ++v) ex[v] = ex2[v];
          edge_sum(3);
        }
#pragma unroll
        for (int v = 0; v < NV; ++v) ev[v] = ea[v];
      }
      // The flux through the block's x and y faces, one face point per lane:
      // the cell's own trace, and the flux in place of the outer trace (the x
      // and y lines below take it instead of evaluating the block's last
      // faces on eight lanes each).
      {
        const int ax = ef >> 1, up = ef & 1, st = ax ? n : 1;
        const int ce = (ax ? eg : n * eg) + (up ? (n - 1) * st : 0);       // cell in the layer
        const float* own = Uc + (ax ? fa + NFP * fb : N * w) * LAY + ce;   // first point of the line
        const int ps = (ax ? N : 1) * LAY;
        float in[NV], Je[3], Fe[NV], an;
#pragma unroll
        for (int v = 0; v < NV; ++v) {
          in[v] = 0.f;
#pragma unroll
          for (int q = 0; q < N; ++q) in[v] = fmaf(up ? T.lp[q] : T.lm[q], own[v * (Q * LAY) + q * ps], in[v]);
        }
        if (aff) {
#pragma unroll
          for (int jj = 0; jj < 3; ++jj) Je[jj] = sam[3 * ax + jj];
          an = san[ax];
        } else {
          const float xi[3] = {ax ? xa : (up ? 1.f : -1.f), ax ? (up ? 1.f : -1.f) : xa, xb};
          float tg[3][3];
          tangents<3, float>(Gc + ce, LAY, xi, tg);
          if (ax) contra_row<3, float>(tg, 1, Je);
          else contra_row<3, float>(tg, 0, Je);
          an = rootf(fmaf(Je[2], Je[2], fmaf(Je[1], Je[1], Je[0] * Je[0])));
        }
        float uL[NV], uR[NV];
#pragma unroll
        for (int v = 0; v < NV; ++v) {
          uL[v] = up ? in[v] : ev[v];
          uR[v] = up ? ev[v] : in[v];
        }
        lf1(uL, uR, Je, an, A.gamma, A.gamma - 1.f, ef == 1, Fe);
        const bool given = MORTAR && ((fmask >> ef) & 1);  // the outer value is the flux itself
#pragma unroll
        for (int v = 0; v < NV; ++v) ev[v] = given ? ev[v] : Fe[v];
      }
      if (more) edge_load(0, k + 1, ex);

      // ----------------------------------------------------- x lines
      // traces -> faces -> lifts -> volume flux and weak derivative, with
      // the state read twice from shared memory rather than held (registers)
      {
        const int fpX = w;  // (q_y, q_z)
        float2 tm[NV], tp[NV];
#pragma unroll
        for (int v = 0; v < NV; ++v) {
          tm[v] = tp[v] = f2(0.f);
#pragma unroll
          for (int qx = 0; qx < N; ++qx) {
            const float2 x = lds2(Uc + (v * Q + qx + N * fpX) * LAY + cl);
            tm[v] = fma2(T2.lm[qx], x, tm[v]);
            tp[v] = fma2(T2.lp[qx], x, tp[v]);
          }
        }
        // face normals at xi_x = -1 (both cells)
        float2 Jm[3];
        if (aff) {
#pragma unroll
          for (int jj = 0; jj < 3; ++jj) Jm[jj] = f2(sam[jj]);
        } else {
          const float xi[3] = {-1.f, xa, xb};
          face_row2<0>(Gc, cl, xi, Jm);
        }
        reload_fence();
        // left face of each cell of the pair: (face i0, face i0+1); the
        // block's x- face is given
        float2 Fl[NV];
        float Fr[NV];
        {
          float2 uL[NV];
#pragma unroll
          for (int v = 0; v < NV; ++v) {
            const float nb = __shfl_up_sync(0xffffffffu, tp[v].y, 1);
            uL[v] = make_float2(m == 0 ? tm[v].x : nb, tp[v].x);
          }
          lf2<AX>(uL, tm, Jm, aff ? f2(san[0]) : norm2(Jm), gam, gm1, Fl);
        }
        // right faces: the next pair's left face; the block's x+ face on m == 3
#pragma unroll
        for (int v = 0; v < NV; ++v) {
          const float e = __shfl_sync(0xffffffffu, ev[v], (m == 3 ? 8 : 0) + j);
          Fl[v].x = m == 0 ? e : Fl[v].x;
          const float nx = __shfl_down_sync(0xffffffffu, Fl[v].x, 1);
          Fr[v] = m == 3 ? e : nx;
        }
        LineGeo2<0> lg;
        if (!aff) {
          const float xi[3] = {0.f, xa, xb};
          lg.init(Gc, cl, xi);
        }
        float2 r[N][NV];
#pragma unroll
        for (int v = 0; v < NV; ++v) {
          const float2 fr = make_float2(Fl[v].y, Fr[v]);
#pragma unroll
          for (int qx = 0; qx < N; ++qx) r[qx][v] = fma2(T2.lmw[qx], Fl[v], mul(T2.lpwn[qx], fr));
        }
#pragma unroll
        for (int jj = 0; jj < N; ++jj) {
          float2 uq[NV], Jq[3], G[NV];
#pragma unroll
          for (int v = 0; v < NV; ++v) uq[v] = lds2(Uc + (v * Q + jj + N * fpX) * LAY + cl);
          if (aff) {
#pragma unroll
            for (int jx = 0; jx < 3; ++jx) Jq[jx] = f2(sam[jx]);
          } else {
            lg.at(xq[jj], Jq);
          }
          flux2<AX>(uq, Jq, gm1, G);
#pragma unroll
          for (int qx = 0; qx < N; ++qx)
#pragma unroll
            for (int v = 0; v < NV; ++v) r[qx][v] = fma2(T2.Sh[qx][jj], G[v], r[qx][v]);
        }
        // the z lines of the layer below have read the residual rows (and its
        // geometry buffer is free)
        if (L > 0) wait_for(&zdone, (L - 1) & 1);
        if (k > k0 && k + 1 < k1) issue_geo(k + 1, (L + 1) & 1, pGeo());
#pragma unroll
        for (int v = 0; v < NV; ++v)
#pragma unroll
          for (int qx = 0; qx < N; ++qx) sts2(Rs + (v * Q + qx + N * fpX) * LAY + cl, r[qx][v]);
      }
      // the y lines at q_z = fb read what the x lines at that q_z wrote
      group_sync<32 * N>(1 + fb);

      // ----------------------------------------------------- y lines
      {
        float2 tm[NV], tp[NV];
#pragma unroll
        for (int v = 0; v < NV; ++v) {
          tm[v] = tp[v] = f2(0.f);
#pragma unroll
          for (int qy = 0; qy < N; ++qy) {
            const float2 x = lds2(Uc + (v * Q + fa + N * qy + NFP * fb) * LAY + cl);
            tm[v] = fma2(T2.lm[qy], x, tm[v]);
            tp[v] = fma2(T2.lp[qy], x, tp[v]);
          }
        }
        float2 Jm[3];
        if (aff) {
#pragma unroll
          for (int jj = 0; jj < 3; ++jj) Jm[jj] = f2(sam[3 + jj]);
        } else {
          const float xi[3] = {xa, -1.f, xb};
          face_row2<1>(Gc, cl, xi, Jm);
        }
        reload_fence();
        // bottom face of my row: against the row below; the block's y- and y+
        // faces are given
        float2 Fb[NV], Ft[NV];
        {
          float2 uL[NV];
#pragma unroll
          for (int v = 0; v < NV; ++v) {
            const float2 nb = shfl_up2(tp[v], 4);
            uL[v] = j == 0 ? tm[v] : nb;
          }
          lf2<AY>(uL, tm, Jm, aff ? f2(san[1]) : norm2(Jm), gam, gm1, Fb);
        }
#pragma unroll
        for (int v = 0; v < NV; ++v) {
          const int from = (j == n - 1 ? 24 : 16) + i0;
          const float2 e = make_float2(__shfl_sync(0xffffffffu, ev[v], from), __shfl_sync(0xffffffffu, ev[v], from + 1));
          Fb[v] = j == 0 ? e : Fb[v];
          const float2 nx = shfl_down2(Fb[v], 4);
          Ft[v] = j == n - 1 ? e : nx;
        }
        if (more) {
          edge_sum(0);
          edge_load(1, k + 1, ex);
        }
        LineGeo2<1> lg;
        if (!aff) {
          const float xi[3] = {xa, 0.f, xb};
          lg.init(Gc, cl, xi);
        }
        float2 r[N][NV];
#pragma unroll
        for (int v = 0; v < NV; ++v)
#pragma unroll
          for (int qy = 0; qy < N; ++qy)
            r[qy][v] = fma2(T2.lmw[qy], Fb[v],
                            fma2(T2.lpwn[qy], Ft[v], lds2(Rs + (v * Q + fa + N * qy + NFP * fb) * LAY + cl)));
#pragma unroll
        for (int jj = 0; jj < N; ++jj) {
          float2 uq[NV], Jq[3], G[NV];
#pragma unroll
          for (int v = 0; v < NV; ++v) uq[v] = lds2(Uc + (v * Q + fa + N * jj + NFP * fb) * LAY + cl);
          if (aff) {
#pragma unroll
            for (int jx = 0; jx < 3; ++jx) Jq[jx] = f2(sam[3 + jx]);
          } else {
            lg.at(xq[jj], Jq);
          }
          flux2<AY>(uq, Jq, gm1, G);
#pragma unroll
          for (int qy = 0; qy < N; ++qy)
#pragma unroll
            for (int v = 0; v < NV; ++v) r[qy][v] = fma2(T2.Sh[qy][jj], G[v], r[qy][v]);
        }
#pragma unroll
        for (int v = 0; v < NV; ++v)
#pragma unroll
          for (int qy = 0; qy < N; ++qy) sts2(Rs + (v * Q + fa + N * qy + NFP * fb) * LAY + cl, r[qy][v]);
      }
      // the z lines at q_x = fa read what the y lines at that q_x wrote
      group_sync<32 * N>(1 + N + fa);

      // ----------------------------------------------------- z lines + stage
      {
        if (more) {
          edge_sum(1);
          if constexpr (N >= 3) edge_load(2, k + 1, ex);
          if constexpr (N == 4) edge_load(3, k + 1, ex2);
        }
        float2 tp[NV], Ft[NV];
#pragma unroll
        for (int v = 0; v < NV; ++v) {
          tp[v] = f2(0.f);
#pragma unroll
          for (int qz = 0; qz < N; ++qz) tp[v] = fma2(T2.lp[qz], lds2(Uc + (v * Q + fpZ + NFP * qz) * LAY + cl), tp[v]);
        }
        {
          // the next layer's bottom trace (same arithmetic as at a chunk start)
          float2 th[NV], Ja[3];
          if (k + 1 < n) {
            if constexpr (ST == 2) {
              const float* Un1 = Us + ((F + 1) % ST) * ROWS * LAY;
              wait_for(&full[(F + 1) % ST][og], ((F + 1) / ST) & 1);
#pragma unroll
              for (int v = 0; v < NV; ++v) {
                float2 s = f2(0.f);
#pragma unroll
                for (int qz = 0; qz < N; ++qz)
                  s = fma2(T2.lm[qz], lds2(Un1 + (v * Q + fpZ + NFP * qz) * LAY + cl), s);
                th[v] = s;
              }
            } else {
              const float* Un1 = pUb() + (k + 1) * LAY + cl;
#pragma unroll
              for (int v = 0; v < NV; ++v) {
                float2 s = f2(0.f);
#pragma unroll
                for (int qz = 0; qz < N; ++qz)
                  s = fma2(T2.lm[qz], __ldg(reinterpret_cast<const float2*>(Un1 + (size_t)(v * Q + fpZ + NFP * qz) * nc)), s);
                th[v] = s;
              }
            }
          } else if (sdirect & 32) {
            face_pair(5, i0, j, th);
          } else {
#pragma unroll
            for (int v = 0; v < NV; ++v) th[v] = lds2(&GTR(5, v, fpZ, cl));
          }
          if (aff) {
#pragma unroll
            for (int jj = 0; jj < 3; ++jj) Ja[jj] = f2(sam[6 + jj]);
          } else {
            const float xi[3] = {xa, xb, 1.f};
            face_row2<2>(Gc, cl, xi, Ja);
          }
          reload_fence();
          lf2<AZ>(tp, th, Ja, aff ? f2(san[2]) : norm2(Ja), gam, gm1, Ft);
          if (MORTAR && k == n - 1 && (fmask & 32)) {
#pragma unroll
            for (int v = 0; v < NV; ++v) Ft[v] = th[v];  // the z+ face flux itself
          }
        }
        LineGeo2<2> lg;
        if (!aff) {
          const float xi[3] = {xa, xb, 0.f};
          lg.init(Gc, cl, xi);
        }
        float2 r[N][NV], iJ[N];
        unpark();
#pragma unroll
        for (int v = 0; v < NV; ++v)
#pragma unroll
          for (int qz = 0; qz < N; ++qz)
            r[qz][v] = fma2(T2.lmw[qz], Fbot[v],
                            fma2(T2.lpwn[qz], Ft[v], lds2(Rs + (v * Q + fpZ + NFP * qz) * LAY + cl)));
#pragma unroll
        for (int v = 0; v < NV; ++v) Fbot[v] = Ft[v];
        park();
        // U^n of the z lines' points into the residual rows this warp has read
        if (!C::UNREG && use_un) {
          __syncwarp();
          if (lane == 0) mbar_arrive_expect(&unbar[w], OWN * LAY * sizeof(float));
          __syncwarp();
          if (lane < OWN) {
            const int rr = (lane / N) * Q + w + NFP * (lane % N);
            fence_proxy_async();
            bulk_row(Rs + rr * LAY, pUnb() + (size_t)rr * nc + k * LAY, LAY * sizeof(float), &unbar[w]);
          }
        }
#pragma unroll
        for (int jj = 0; jj < N; ++jj) {
          float2 uq[NV], Jq[3], G[NV];
#pragma unroll
          for (int v = 0; v < NV; ++v) uq[v] = lds2(Uc + (v * Q + fpZ + NFP * jj) * LAY + cl);
          if (aff) {
#pragma unroll
            for (int jx = 0; jx < 3; ++jx) Jq[jx] = f2(sam[6 + jx]);
            iJ[jj] = f2(sam[9]);
          } else {
            lg.at(xq[jj], Jq);
            iJ[jj] = rcp2(lg.jac(Jq));
          }
          flux2<AZ>(uq, Jq, gm1, G);
#pragma unroll
          for (int qz = 0; qz < N; ++qz)
#pragma unroll
            for (int v = 0; v < NV; ++v) r[qz][v] = fma2(T2.Sh[qz][jj], G[v], r[qz][v]);
        }
        // U^n of the z line's points (prefetched into L2 with the layer), all
        // loads issued before the first use
        float2 un[C::UNREG ? N : 1][NV];
        if (C::UNREG && use_un) {
#pragma unroll
          for (int qz = 0; qz < N; ++qz)
#pragma unroll
            for (int v = 0; v < NV; ++v)
              un[qz][v] = __ldcg(reinterpret_cast<const float2*>(pUnb() + (size_t)(v * Q + fpZ + NFP * qz) * nc + k * LAY + cl));
        }
        // stage combination straight to global memory, CFL on the last stage
        float* const out = (BATCH ? sit.Ob : Ob) + k * LAY + cl;  // (v, q) row offsets added below
        if constexpr (BATCH) dt2 = f2(sit.dt);
        if (!C::UNREG && use_un) wait_for(&unbar[w], L & 1);
        float2 hc = f2(0.f);
        if (A.last) hc = __ldg(reinterpret_cast<const float2*>((BATCH ? sit.Hb : Hb) + k * LAY + cl));
#pragma unroll
        for (int qz = 0; qz < N; ++qz) {
          const int q = fpZ + NFP * qz;
          float2 o[NV];
#pragma unroll
          for (int v = 0; v < NV; ++v) {
            const float2 s = mul(r[qz][v], iJ[qz]);
            float2 val;
            if (A.mode == 1) {
              val = s;
            } else {
              val = mul(cb2, fma2(dt2, s, lds2(Uc + (v * Q + q) * LAY + cl)));
              if (use_un) val = fma2(ca2, C::UNREG ? un[C::UNREG ? qz : 0][v] : lds2(Rs + (v * Q + q) * LAY + cl), val);
            }
            *reinterpret_cast<float2*>(out + (v * Q + q) * nc) = val;
            o[v] = val;
          }
          if (A.last) {
#pragma unroll
            for (int e = 0; e < 2; ++e) {
              const float r0 = e ? o[0].y : o[0].x;
              const float m1 = e ? o[1].y : o[1].x;
              const float m2 = e ? o[2].y : o[2].x;
              const float m3 = e ? o[3].y : o[3].x;
              const float en = e ? o[4].y : o[4].x;
              const float ri = rcpf(r0);
              const float ke = m1 * m1 + m2 * m2 + m3 * m3;
              const float sv = (fabsf(m1) + fabsf(m2) + fabsf(m3)) * ri;
              const float pr = (A.gamma - 1.f) * (en - 0.5f * ke * ri);
              if (!(r0 > 0.f) || !(pr > 0.f) || !(pr < 3.0e38f)) {
                bad = true;
              } else {
                const float lam = sv + 3.f * rootf(A.gamma * pr * ri);
                const float hv = (e ? hc.y : hc.x) / lam;
                lam_min = hv < lam_min ? hv : lam_min;
              }
            }
          }
        }
      }
      // this warp is done with the layer: its residual rows are free, and so
      // are the state rows it owns
      __syncwarp();
      if (lane == 0) mbar_arrive(&zdone);
      if (k + ST < kend) issue(k + ST, F % ST, pUb(), pUnb());
      ++L;
      ++F;
    }
    F += kend - k1;
    if (fail && lane == 0) atomicExch(BATCH ? sit.status : A.status, kStatusTimeout);
    if constexpr (BATCH) {
      // the CFL minimum and the status belong to this item's forest
      if (A.last) {
        cta_min_atomic<C::NT>((double)lam_min, sit.lam);
        lam_min = 3.0e38f;
        if (__syncthreads_or(bad) && tid == 0) atomicExch(sit.status, kStatusNonFinite);
        bad = false;
      }
    }
#undef GTR
  }
  if (fail) {
    // a bounded wait gave up (reported above): wait, bounded, for the copies
    // that may still be in flight into this CTA's buffers
    for (uint32_t i = F > ST ? F - ST : 0; i < F; ++i) mbar_wait(&full[i % ST][og], (i / ST) & 1);
    for (uint32_t i = L > 2 ? L - 2 : 0; !AFF && i < L; ++i) mbar_wait(&gfull[i & 1], (i >> 1) & 1);
    if (!C::UNREG && use_un && L > 0) mbar_wait(&unbar[w], (L - 1) & 1);
  }
  if (!BATCH && A.last) {
    // block min of h/lambda -> one atomic per CTA
    double v = (double)lam_min;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      const double u = __shfl_xor_sync(0xffffffffu, v, o);
      v = u < v ? u : v;
    }
    __shared__ double red[32];
    __syncthreads();
    if (lane == 0) red[w] = v;
    __syncthreads();
    if (w == 0) {
      v = lane < C::NT / 32 ? red[lane] : 3.0e38;
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) {
        const double u = __shfl_xor_sync(0xffffffffu, v, o);
        v = u < v ? u : v;
      }
      if (lane == 0 && v < 3.0e38) atomicMin(A.lam_bits, (unsigned long long)__double_as_longlong(v));
    }
    if (bad) atomicExch(A.status, kStatusNonFinite);
  }
}

// launch (grid = persistent CTAs, or one per work item) and resident CTAs
// per SM, for the launch layer in kernels_inst.cuh; v = the CTA shape
template <int P, int V>
cudaError_t stage_pair_launch_v(const StageArgs<3, P, float>& a, int grid, bool mortar, int shape, cudaStream_t s) {
  using C = pairk::PairCfg<P, V>;
  const pairk::PairTab<P + 1> t2 = pairk::pair_tab<P + 1>(a.T);
  if (mortar) {
    if (shape) k_stage_pair<P, true, 1, false, V><<<grid, C::NT, C::smem(true), s>>>(a, t2);
    else k_stage_pair<P, true, 0, false, V><<<grid, C::NT, C::smem(false), s>>>(a, t2);
  } else {
    if (shape == 2) k_stage_pair<P, false, 2, false, V><<<grid, C::NT, C::smem(true), s>>>(a, t2);
    else if (shape) k_stage_pair<P, false, 1, false, V><<<grid, C::NT, C::smem(true), s>>>(a, t2);
    else k_stage_pair<P, false, 0, false, V><<<grid, C::NT, C::smem(false), s>>>(a, t2);
  }
  return cudaGetLastError();
}

// shape: what every block of the forest is (GEO of k_stage_pair)
template <int P>
cudaError_t stage_pair_launch(const StageArgs<3, P, float>& a, int grid, bool mortar, int shape, cudaStream_t s, int v) {
  if constexpr (P == 1) {
    if (v) return stage_pair_launch_v<P, 1>(a, grid, mortar, shape, s);
  }
  return stage_pair_launch_v<P, 0>(a, grid, mortar, shape, s);
}

// one launch over the forests of a batch (a.members); plain form, no mortar
template <int P>
cudaError_t stage_pair_launch_batch(const StageArgs<3, P, float>& a, int grid, int shape, cudaStream_t s) {
  using C = pairk::PairCfg<P>;
  const pairk::PairTab<P + 1> t2 = pairk::pair_tab<P + 1>(a.T);
  if (shape == 2) k_stage_pair<P, false, 2, true><<<grid, C::NT, C::smem(true), s>>>(a, t2);
  else if (shape) k_stage_pair<P, false, 1, true><<<grid, C::NT, C::smem(true), s>>>(a, t2);
  else k_stage_pair<P, false, 0, true><<<grid, C::NT, C::smem(false), s>>>(a, t2);
  return cudaGetLastError();
}

template <int P, bool MORTAR, int GEO, bool BATCH = false, int V = 0>
int pair_blocks_per_sm_one() {
  using C = pairk::PairCfg<P, V>;
  auto* k = k_stage_pair<P, MORTAR, GEO, BATCH, V>;
  const size_t smem = C::smem(GEO != 0);
  if (cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) != cudaSuccess) return 0;
  int nb = 0;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, k, C::NT, smem) != cudaSuccess) return 0;
  return nb;
}

// the fewest resident CTAs over the instantiations that a forest of this
// shape may launch (CTA shape v; batches have shape 0)
template <int P, int GEO, int V>
int pair_blocks_per_sm() {
  int o = pair_blocks_per_sm_one<P, false, GEO, false, V>();
  auto least = [&](int x) { o = x < o ? x : o; };
  least(pair_blocks_per_sm_one<P, true, GEO != 0, false, V>());
  if constexpr (V == 0) least(pair_blocks_per_sm_one<P, false, GEO, true>());
  return o;
}
template <int P>
int stage_pair_blocks_per_sm(int v, int shape) {
  if constexpr (P == 1) {
    if (v)
      return shape == 2 ? pair_blocks_per_sm<P, 2, 1>() : shape ? pair_blocks_per_sm<P, 1, 1>()
                                                                : pair_blocks_per_sm<P, 0, 1>();
  }
  return shape == 2 ? pair_blocks_per_sm<P, 2, 0>() : shape ? pair_blocks_per_sm<P, 1, 0>()
                                                            : pair_blocks_per_sm<P, 0, 0>();
}

}  // namespace dgf
