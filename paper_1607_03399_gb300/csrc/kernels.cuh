// CUDA kernels of the DG stage (included once per precision; the including
// translation unit defines REAL and the constant-memory table c_ops).
//
// Wedge stage (Sections 3.2, 4.2; one launch per Runge-Kutta stage):
//   CTA = 32 consecutive wedges x (N+1) warps; warp j owns GLL slice j of all
//   32 elements, lane = element.  Per element and slice:
//     geometry from the 6 vertices (Lemma 3.1): r_x, r_y, s_x, s_y, t_zJ = A
//       constant, t_xJ, t_yJ at t_j, J_a = A h_a / 2 at the three columns;
//     W_j = M^tri [ T_j + J_fb ell0_j F_bot + J_ft ellN_j F_top ]
//           + sum_quad M~_e F_e,j                       (lift, weak form)
//       T_j = - sum_c t_cJ(t_j) (D_t u_c)_j  (p),  - t_cJ(t_j) (D_t p)_j  (u_c)
//     X_j = (M^{tri,k})^{-1} W_j, M^{tri,k} = sum_a J_a M_a, by a per-element
//       L D L^T factor, stored or formed in the stage (exact inverse of the
//       Jacobian-weighted wedge mass, Section 4.2);
//     rhs = kappa (-(D_r (r.u) + D_s (s.u))_j + X_p),
//     rhs_u_c = (1/rho) (-(r_c D_r p + s_c D_s p)_j + X_u_c);
//     fused LSRK update res <- a res + dt rhs, q_out <- q_in + b res.
// Tet stage: affine tets, one thread per element (Section 3.2: physical
//   operators are scaled reference operators).
#pragma once
#include <cuda_runtime.h>
#include <type_traits>

#include "dg_internal.hpp"

namespace dgw {
namespace REALNS {

using real = REAL;

template <int N>
__device__ __forceinline__ const AllOps<N, real>& OPS() {
  static_assert(N == NORD, "one order per translation unit");
  return c_ops;
}

__device__ __forceinline__ float rsqrt_r(float x) { return rsqrtf(x); }
__device__ __forceinline__ double rsqrt_r(double x) { return rsqrt(x); }
__device__ __forceinline__ float sqrt_r(float x) { return sqrtf(x); }
__device__ __forceinline__ double sqrt_r(double x) { return sqrt(x); }

// triangle node (a, b) -> index; edge node m of triangle edge ed (from its
// first to its second vertex)
__host__ __device__ constexpr int tri_idx(int N, int a, int b) { return b * (N + 1) - (b * (b - 1)) / 2 + a; }
__host__ __device__ constexpr int edge_node(int N, int ed, int m) {
  return ed == 0 ? tri_idx(N, m, 0) : (ed == 1 ? tri_idx(N, N - m, m) : tri_idx(N, 0, N - m));
}
// Packed state layout: node-major, the four fields innermost, so one thread
// moves a node's (p, u_x, u_y, u_z) with one 16-byte (FP32) access and a warp
// moves 512 contiguous bytes:
//   wedge region [nblk_w][Np][32 lanes][4 fields], tet region likewise.
template <int N>
__device__ __forceinline__ int64_t widx(int blk_e, int node, int lane) {
  constexpr int Np = npw_of(N);
  return ((int64_t(blk_e) * Np + node) * kB + lane) * 4;
}
template <int N>
__device__ __forceinline__ int64_t tidx(int64_t off, int blk_e, int node, int lane) {
  constexpr int Np = npt_of(N);
  return off + ((int64_t(blk_e) * Np + node) * kB + lane) * 4;
}

struct Q4 {
  real p, u, v, w;
};
// shared-memory slab [Np][32][4]
__device__ __forceinline__ Q4 lds4(const real* slab, int node, int lane) {
  const real* a = slab + ((node * kB + lane) << 2);
  if constexpr (sizeof(real) == 4) {
    const float4 t = *reinterpret_cast<const float4*>(a);
    return Q4{real(t.x), real(t.y), real(t.z), real(t.w)};
  } else {
    const double2 t0 = reinterpret_cast<const double2*>(a)[0], t1 = reinterpret_cast<const double2*>(a)[1];
    return Q4{real(t0.x), real(t0.y), real(t1.x), real(t1.y)};
  }
}
// global, read-only for the whole lifetime of the kernel (the non-coherent
// path).  Not for the stage input of a kernel that may be launched as a
// programmatic dependent (k_wedge_stage, k_wedge_wide): the stage that writes
// it may still run when such a kernel starts; they use ld4
__device__ __forceinline__ Q4 ldg4(const real* __restrict__ q, int64_t idx) {
  if constexpr (sizeof(real) == 4) {
    const float4 t = __ldg(reinterpret_cast<const float4*>(q + idx));
    return Q4{real(t.x), real(t.y), real(t.z), real(t.w)};
  } else {
    const double2 t0 = __ldg(reinterpret_cast<const double2*>(q + idx));
    const double2 t1 = __ldg(reinterpret_cast<const double2*>(q + idx) + 1);
    return Q4{real(t0.x), real(t0.y), real(t1.x), real(t1.y)};
  }
}
// global, coherent (the residual, rewritten by the same thread; the stage
// input of a programmatic dependent, after pdl_wait)
__device__ __forceinline__ Q4 ld4(const real* q, int64_t idx) {
  if constexpr (sizeof(real) == 4) {
    const float4 t = *reinterpret_cast<const float4*>(q + idx);
    return Q4{real(t.x), real(t.y), real(t.z), real(t.w)};
  } else {
    const double2 t0 = reinterpret_cast<const double2*>(q + idx)[0], t1 = reinterpret_cast<const double2*>(q + idx)[1];
    return Q4{real(t0.x), real(t0.y), real(t1.x), real(t1.y)};
  }
}
// shared-memory operator records: (a, b, c, d) in natural order -> Q4{a, b, c, d}
__device__ __forceinline__ Q4 ldop4(const real* a) {
  if constexpr (sizeof(real) == 4) {
    const float4 t = *reinterpret_cast<const float4*>(a);
    return Q4{real(t.x), real(t.y), real(t.z), real(t.w)};
  } else {
    const double2 t0 = reinterpret_cast<const double2*>(a)[0], t1 = reinterpret_cast<const double2*>(a)[1];
    return Q4{real(t0.x), real(t0.y), real(t1.x), real(t1.y)};
  }
}
__device__ __forceinline__ void st4(real* q, int64_t idx, const Q4& v) {
  if constexpr (sizeof(real) == 4) {
    *reinterpret_cast<float4*>(q + idx) = make_float4(float(v.p), float(v.u), float(v.v), float(v.w));
  } else {
    reinterpret_cast<double2*>(q + idx)[0] = make_double2(double(v.p), double(v.u));
    reinterpret_cast<double2*>(q + idx)[1] = make_double2(double(v.v), double(v.w));
  }
}

// Packed pairs.  In FP32 one packed FMA instruction (sm_100 family) performs
// two multiply-adds, each rounded as fmaf: half the issue slots of the scalar
// form, same results.  In FP64 a pair is two scalar FMAs.
using real2 = typename std::conditional<sizeof(real) == 4, float2, double2>::type;
__device__ __forceinline__ float2 fma2(const float2 a, const float2 b, const float2 c) { return __ffma2_rn(a, b, c); }
__device__ __forceinline__ double2 fma2(const double2 a, const double2 b, const double2 c) {
  return make_double2(fma(a.x, b.x, c.x), fma(a.y, b.y, c.y));
}
__device__ __forceinline__ float2 add2(const float2 a, const float2 b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ double2 add2(const double2 a, const double2 b) { return make_double2(a.x + b.x, a.y + b.y); }
__device__ __forceinline__ float2 mul2(const float2 a, const float2 b) { return __fmul2_rn(a, b); }
__device__ __forceinline__ double2 mul2(const double2 a, const double2 b) { return make_double2(a.x * b.x, a.y * b.y); }
__device__ __forceinline__ real2 dup2(const real v) {
  real2 r;
  r.x = v;
  r.y = v;
  return r;
}
__device__ __forceinline__ real2 mk2(const real a, const real b) {
  real2 r;
  r.x = a;
  r.y = b;
  return r;
}
// entry (h, l) of an output-pair table (constant memory; an 8-byte operand)
__device__ __forceinline__ real2 cpair(const real* XP, int cols, int h, int l) {
  return *reinterpret_cast<const real2*>(XP + (h * cols + l) * 2);
}
// acc = X x for an NR x NC operator given by output pairs XP (acc[h] holds
// rows 2h, 2h + 1): every output accumulates its products over l in order
template <int NR, int NC>
__device__ __forceinline__ void apply_pairs(const real* XP, const real (&x)[NC], real2 (&acc)[(NR + 1) / 2]) {
  constexpr int NH = (NR + 1) / 2;
#pragma unroll
  for (int h = 0; h < NH; ++h) acc[h] = dup2(real(0));
#pragma unroll
  for (int l = 0; l < NC; ++l) {
    const real2 xx = dup2(x[l]);
#pragma unroll
    for (int h = 0; h < NH; ++h) acc[h] = fma2(cpair(XP, NC, h, l), xx, acc[h]);
  }
}
// row i of a pair-accumulated result
__device__ __forceinline__ real pair_row(const real2* acc, int i) { return (i & 1) ? acc[i >> 1].y : acc[i >> 1].x; }

// a * b + c rounded once (an explicit FMA: the same rounding wherever the
// compiler places the expression, so kernel variants that differ only in when
// they load the operands give the same bits)
__device__ __forceinline__ float fmar(float a, float b, float c) { return fmaf(a, b, c); }
__device__ __forceinline__ double fmar(double a, double b, double c) { return fma(a, b, c); }
// Penalty fluxes of eq. (1): F_p = 1/2 (tau_p [p] - [u_n]), F_u = 1/2 (tau_u [u_n] - [p]).
__device__ __forceinline__ void penalty_flux(real dp, real dun, real tau_p, real tau_u, real& Fp, real& Fu) {
  Fp = real(0.5) * fmar(tau_p, dp, -dun);
  Fu = real(0.5) * fmar(tau_u, dun, -dp);
}
// Boundary ghosts: Dirichlet p+ = -p-, u+ = u-  -> [p] = -2p, [u_n] = 0;
// rigid p+ = p-, u+ = u- - 2 u_n n             -> [p] = 0, [u_n] = -2 u_n.
__device__ __forceinline__ void boundary_jumps(int bc, real pM, real unM, real& dp, real& dun) {
  const bool dir = bc == 0;
  dp = dir ? real(-2) * pM : real(0);
  dun = dir ? real(0) : real(-2) * unM;
}

__device__ __forceinline__ void taus(int flux, real zM, real zP, real& tau_p, real& tau_u) {
  const real zavg = real(0.5) * (zM + zP);
  const real izavg = real(1) / zavg;
  const bool up = flux == 0;
  tau_p = up ? izavg : real(0);
  tau_u = up ? zavg : real(0);
}

// ---------------------------------------------------------------------------
// shared reference operators on the tensor cores (FP32 fields, warp-level
// mma.sync): Out = Op * In with Op an Nt x Nt triangle operator zero-padded
// to 16 x 16 (the A operand, in registers) and In an Nt-row tile in shared
// memory whose columns are (element, field) pairs (the B operand).  TF32 is
// m16n8k8 (two k-steps cover Nt <= 16), BF16 m16n8k16 (one k-step); both
// accumulate in FP32.  3xTF32 splits each operand x = hi + lo into two TF32
// numbers and adds lo*hi + hi*lo + hi*hi (dropping lo*lo), which recovers
// about FP32 accuracy.
// ---------------------------------------------------------------------------
__device__ __forceinline__ uint32_t tf32_of(float x) {
  uint32_t r;
  asm("cvt.rna.tf32.f32 %0, %1;" : "=r"(r) : "f"(x));
  return r;
}
// (lo, hi) -> bf16x2 with lo in the low half (the lower k index of an operand pair)
__device__ __forceinline__ uint32_t bf16x2_of(float lo, float hi) {
  uint32_t r;
  asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(r) : "f"(hi), "f"(lo));
  return r;
}
__device__ __forceinline__ void mma_tf32(float (&d)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
  asm("mma.sync.aligned.m16n8k8.row.col.f32.tf32.tf32.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
      : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}
__device__ __forceinline__ void mma_bf16(float (&d)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
  asm("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
      : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

// A operand registers of one operator: [k-step][4] (hi and, for 3xTF32, lo parts)
template <int OP>
struct AFrag {
  uint32_t h[2][4];
  uint32_t l[OP == kOpTF32x3 ? 2 : 1][4];
};
// Fragment of the row-major Nt x Nt operator Op (rows = outputs), zero-padded.
// m16n8k8 TF32: a0 (g, t), a1 (g + 8, t), a2 (g, t + 4), a3 (g + 8, t + 4) of
// the 16 x 8 slice of k-step ks; m16n8k16 BF16: pairs of columns (2t, 2t + 1)
// and (2t + 8, 2t + 9) of rows g and g + 8 (g = lane / 4, t = lane % 4).
template <int NT, int OP>
__device__ __forceinline__ void afrag_load(const float* Op, int lane, AFrag<OP>& A) {
  const int g = lane >> 2, t = lane & 3;
  auto at = [&](int r, int c) -> float { return (r < NT && c < NT) ? Op[r * NT + c] : 0.f; };
  if constexpr (OP == kOpBF16) {
    A.h[0][0] = bf16x2_of(at(g, 2 * t), at(g, 2 * t + 1));
    A.h[0][1] = bf16x2_of(at(g + 8, 2 * t), at(g + 8, 2 * t + 1));
    A.h[0][2] = bf16x2_of(at(g, 2 * t + 8), at(g, 2 * t + 9));
    A.h[0][3] = bf16x2_of(at(g + 8, 2 * t + 8), at(g + 8, 2 * t + 9));
  } else {
#pragma unroll
    for (int ks = 0; ks < 2; ++ks) {
      const float v[4] = {at(g, t + 8 * ks), at(g + 8, t + 8 * ks), at(g, t + 4 + 8 * ks), at(g + 8, t + 4 + 8 * ks)};
#pragma unroll
      for (int r = 0; r < 4; ++r) {
        A.h[ks][r] = tf32_of(v[r]);
        if constexpr (OP == kOpTF32x3) A.l[ks][r] = tf32_of(v[r] - __uint_as_float(A.h[ks][r]));
      }
    }
  }
}
// B operand of one n-tile: column `col` of the Nt-row operand tile B (layout
// tile_at); rows >= Nt are zero (never read).  TF32: [k-step] (k = t, t + 4)
// per step; BF16: (2t, 2t + 1) and (2t + 8, 2t + 9).
template <int OP>
struct BFrag {
  uint32_t h[2][2];
  uint32_t l[OP == kOpTF32x3 ? 2 : 1][2];
};
template <int NT, int OP>
__device__ __forceinline__ void bfrag_load(const float* B, int col, int lane, BFrag<OP>& F) {
  const int t = lane & 3;
  auto bv = [&](int k) -> float { return k < NT ? B[tile_at(k, col)] : 0.f; };
  if constexpr (OP == kOpBF16) {
    F.h[0][0] = bf16x2_of(bv(2 * t), bv(2 * t + 1));
    F.h[0][1] = bf16x2_of(bv(2 * t + 8), bv(2 * t + 9));
  } else {
#pragma unroll
    for (int ks = 0; ks < (NT + 7) / 8; ++ks) {
      const float x0 = bv(t + 8 * ks), x1 = bv(t + 4 + 8 * ks);
      F.h[ks][0] = tf32_of(x0);
      F.h[ks][1] = tf32_of(x1);
      if constexpr (OP == kOpTF32x3) {
        F.l[ks][0] = tf32_of(x0 - __uint_as_float(F.h[ks][0]));
        F.l[ks][1] = tf32_of(x1 - __uint_as_float(F.h[ks][1]));
      }
    }
  }
}
// d += Op * B for one 16 x 8 output tile
template <int NT, int OP>
__device__ __forceinline__ void op_mma(const AFrag<OP>& A, const BFrag<OP>& F, float (&d)[4]) {
  if constexpr (OP == kOpBF16) {
    mma_bf16(d, A.h[0], F.h[0][0], F.h[0][1]);
  } else {
#pragma unroll
    for (int ks = 0; ks < (NT + 7) / 8; ++ks) {
      if constexpr (OP == kOpTF32x3) {
        mma_tf32(d, A.l[ks], F.h[ks][0], F.h[ks][1]);
        mma_tf32(d, A.h[ks], F.l[ks][0], F.l[ks][1]);
      }
      mma_tf32(d, A.h[ks], F.h[ks][0], F.h[ks][1]);
    }
  }
}

// Ricker wavelet (1 - 2 a) exp(-a), a = (pi f0 (t - t0))^2 (c13 reading).
__device__ __forceinline__ double ricker(double f0, double tau) {
  const double a = (3.14159265358979323846 * f0 * tau) * (3.14159265358979323846 * f0 * tau);
  return (1.0 - 2.0 * a) * exp(-a);
}
// True when a point source lies in element (type, elem): the entries, sorted by
// element, of its 32-element block are scanned.
__device__ __forceinline__ bool has_source(const DevMesh<real>& M, int type, int elem) {
  const int* rng = (type == 6 ? M.w_srng : M.t_srng) + 2 * (elem >> 5);
  const int b = rng[0], e = rng[1];
  for (int s = b; s < e; ++s)
    if (M.src[s].elem == elem) return true;
  return false;
}
// Point-source forcing of element (type, elem) at time t added to the pressure
// accumulators acc[c] of element nodes n0 + c (c < C, n0 + c < np), before the
// kappa scaling: acc += w_s(t) g_s with g_s = (M^k)^{-1} l(x_s) and w_s the
// source's Ricker amplitude.  The time function is evaluated once per source.
template <int C>
__device__ __forceinline__ void add_sources(const DevMesh<real>& M, int type, int elem, int n0, int np, double t,
                                            real (&acc)[C]) {
  const int* rng = (type == 6 ? M.w_srng : M.t_srng) + 2 * (elem >> 5);
  const int sb = rng[0], se = rng[1];
#pragma unroll 1
  for (int s = sb; s < se; ++s) {
    const SourceDev& sd = M.src[s];
    if (sd.elem != elem) continue;
    const real w = real(sd.amp * ricker(sd.f0, t - sd.t0));
    const real* __restrict__ g = M.src_g + sd.goff + n0;
#pragma unroll
    for (int c = 0; c < C; ++c)
      if (n0 + c < np) acc[c] = fmar(w, g[c], acc[c]);
  }
}
// the same on field-pair accumulators whose x component is the pressure
template <int C>
__device__ __forceinline__ void add_sources(const DevMesh<real>& M, int type, int elem, int n0, int np, double t,
                                            real2 (&acc)[C]) {
  const int* rng = (type == 6 ? M.w_srng : M.t_srng) + 2 * (elem >> 5);
  const int sb = rng[0], se = rng[1];
#pragma unroll 1
  for (int s = sb; s < se; ++s) {
    const SourceDev& sd = M.src[s];
    if (sd.elem != elem) continue;
    const real w = real(sd.amp * ricker(sd.f0, t - sd.t0));
    const real* __restrict__ g = M.src_g + sd.goff + n0;
#pragma unroll
    for (int c = 0; c < C; ++c)
      if (n0 + c < np) acc[c].x = fmar(w, g[c], acc[c].x);
  }
}

// Programmatic dependent launch (StageArgs::pdl): the stage after this one may
// be scheduled now; what it does before its own pdl_wait reads mesh tables
// only.  pdl_wait returns when the stage before this one has completed and its
// writes are visible (at once in an ordinary launch); the state and residual
// are read after it, with ordinary loads and bulk copies.
__device__ __forceinline__ void pdl_launch_dependents() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

// advances the time: a step's stages read one slot of the device clock, the
// next step's the other, so in a captured step this runs beside the stages
__global__ void k_clock(const double* from, double* to, double dt) {
  if (threadIdx.x == 0 && blockIdx.x == 0) *to = *from + dt;
}
// sets the device clock (state loads: no host staging, so no synchronisation)
__global__ void k_set_clock(double* clock, double t) {
  if (threadIdx.x == 0 && blockIdx.x == 0) *clock = t;
}

// ---------------------------------------------------------------------------
// wedge stage
// ---------------------------------------------------------------------------
// ---------------------------------------------------------------------------
// bulk asynchronous copies (TMA engine) with mbarrier completion; every wait
// is bounded and reports a timeout through the device error word
// ---------------------------------------------------------------------------
__device__ __forceinline__ uint32_t smem_u32(const void* p) { return uint32_t(__cvta_generic_to_shared(p)); }
__device__ __forceinline__ void mbar_init(uint64_t* bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count) : "memory");
}
__device__ __forceinline__ void fence_mbar_init() { asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory"); }
__device__ __forceinline__ void mbar_expect_tx(uint64_t* bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes) : "memory");
}
__device__ __forceinline__ void bulk_g2s(void* dst, const void* src, uint32_t bytes, uint64_t* bar) {
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
                   smem_u32(dst)),
               "l"(src), "r"(bytes), "r"(smem_u32(bar))
               : "memory");
}
// One poll of the phase; the thread may be suspended for up to the hint
// (1 us) while the phase is incomplete, so waiting threads do not spin.
__device__ __forceinline__ bool mbar_try_wait(uint64_t* bar, uint32_t phase) {
  uint32_t ok;
  asm volatile(
      "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2, %3;\n selp.u32 %0, 1, 0, p;\n}\n"
      : "=r"(ok)
      : "r"(smem_u32(bar)), "r"(phase), "n"(1000)
      : "memory");
  return ok != 0;
}
// About a second of polling at most (each poll suspends for at most ~1 us).
constexpr long long kWaitLimit = 1ll << 20;
template <long long Limit = kWaitLimit>
__device__ __forceinline__ bool mbar_wait_bounded(uint64_t* bar, uint32_t phase) {
  for (long long it = 0; it < Limit; ++it)
    if (mbar_try_wait(bar, phase)) return true;
  return false;
}

// Failure-path check: one warp arms an mbarrier for bytes that no copy will
// ever deliver (no copy is issued), so the stages' bounded wait runs out --
// here after 64 polls instead of the stages' ~1 s budget -- and the kernel
// reports DG_ERR_TIMEOUT through the device error word, exactly as a stage
// whose copy never landed does, then returns.  Nothing is in flight when it
// exits; the GPU and the context stay usable.
__global__ void k_wait_expire(int* err) {
  __shared__ __align__(8) uint64_t bar;
  if (threadIdx.x == 0) {
    mbar_init(&bar, 1);
    fence_mbar_init();
    mbar_expect_tx(&bar, 16u);
  }
  __syncwarp();
  const bool ok = __all_sync(0xffffffffu, mbar_wait_bounded<64>(&bar, 0));
  if (!ok && threadIdx.x == 0) atomicOr(err, kErrTimeout);
}

// per-element geometric factors kept in shared memory ([item][32])
// (the column Jacobians J0..J2 come last: the stage does not use them and
// keeps only the first G_STAGE items)
enum WGeo : int {
  G_RX, G_RY, G_SX, G_SY, G_A, G_NB0, G_NB1, G_NB2, G_NT0, G_NT1, G_NT2, G_JFB, G_JFT,
  G_QNX0, G_QNX1, G_QNX2, G_QNY0, G_QNY1, G_QNY2, G_QCA0, G_QCA1, G_QCA2, G_QCB0, G_QCB1, G_QCB2,
  G_TX0, G_TX1, G_TY0, G_TY1, G_STAGE, G_J0 = G_STAGE, G_J1, G_J2, G_COUNT
};

// Residual slab staged in shared memory by the bulk copy (FP32 up to N = 4,
// FP64 up to N = 3), so that the update reads it there instead of one
// dependent global load per node at the end of the kernel.  At N = 4 the
// stage runs two CTAs per SM (registers), and 103 KB of shared memory per CTA
// still fits two: with the packed-pair arithmetic the staged slab measured
// 1075 -> 820 us per stage on 524,288 wedges (before it, with the scalar
// arithmetic, it had measured slower).  With tensor-core applies the operand
// tiles (Nq x Nt x 128 reals, the size of the residual slab) share the
// residual slab's space: the residual is copied in once the weak-form
// accumulation has released them.
template <int N>
__host__ __device__ constexpr bool stage_res() {
  return sizeof(real) == 4 ? N <= 4 : N <= 3;
}

template <int N, int OP = kOpFFMA>
struct WedgeSmem {
  static constexpr int Nt = nt_of(N), Nq = N + 1, Np = Nt * Nq;
  static constexpr int q = 0;                                            // [4][Np][32]
  static constexpr int r = q + 4 * Np * kB;                              // [4][Np][32] (if staged)
  static constexpr int L = r + (stage_res<N>() ? 4 * Np * kB : 0);       // [NL4][32][4]
  static constexpr int F = L + nl4_of(N) * 4 * kB;                        // [4][Nt][32]
  static constexpr int G = F + 4 * Nt * kB;                              // [G_STAGE][32]
  static constexpr int T = r;  // per-warp operand tiles [Nt][kTP] (tensor cores): the residual slab's space
  static constexpr int reals = G + G_STAGE * kB;
  static_assert(OP == kOpFFMA || (stage_res<N>() && Nq * Nt * kTP <= 4 * Np * kB), "the tiles fit the residual slab's space");
};

template <int N, int OP = kOpFFMA>
__host__ __device__ constexpr int wedge_smem_reals() {
  return WedgeSmem<N, OP>::reals;
}
// Element blocks per CTA of the launch variant with several (a candidate of
// dg_autotune): the warps that work on slice j of the CTA's blocks share an SM
// sub-partition and run the same straight-line code side by side.  One block
// is the default in both mass modes (factor formed in the stage, N = 3,
// 524,288 wedges: 304 us against 401 us with two).
template <int N>
__host__ __device__ constexpr int wedge_bpc_multi() {
  return (sizeof(real) == 4 && N == 3) ? 2 : 1;
}
// bytes: per block two mbarriers and a status word (32 bytes), then per block
// the reals (each block's slabs start 16-byte aligned)
template <int N, int BPC, int OP = kOpFFMA>
__host__ __device__ constexpr int wedge_smem_bytes() {
  return BPC * (32 + wedge_smem_reals<N, OP>() * int(sizeof(real)));
}
constexpr int kHalfSMs = 76;  // half of the 152 SMs
// resident CTAs per SM the stage is compiled for
template <int N, int BPC, int OP>
__host__ __device__ constexpr int wedge_min_ctas() {
  return sizeof(REAL) == 4 ? (N >= 4 ? 2 : 4 / BPC) : 1;
}

// Lemma 3.1 for one wedge: everything the stage needs, from the six vertices
// (bi-unit reference, x = sum_a lambda_a(r,s) [(1-t)/2 X_a + (1+t)/2 X_{a+3}]),
// X = [x_a][y_a][zb_a][zt_a] (a = 0..2, bottom x and y; bottom and top z), in
// six parts: 0 the metric terms (with JAC the column Jacobians too), 1 the
// bottom and 2 the top triangle, 3..5 the quadrilateral faces.
constexpr int kGeoParts = 6;
template <bool JAC>
__device__ __forceinline__ void wedge_geometry_part(int part, const real* sX, real* sG, int lane) {
  auto X = [&](int i) { return sX[i * kB + lane]; };
#define SETG(item, v) sG[(item) * kB + lane] = (v)
  if (part == 0) {
    const real x0 = X(0), y0 = X(3);
    const real xr = real(0.5) * (X(1) - x0), xs = real(0.5) * (X(2) - x0);
    const real yr = real(0.5) * (X(4) - y0), ys = real(0.5) * (X(5) - y0);
    const real A = xr * ys - xs * yr;  // t_z J (constant)
    const real iA = real(1) / A;
    SETG(G_RX, ys * iA);
    SETG(G_RY, -xs * iA);
    SETG(G_SX, -yr * iA);
    SETG(G_SY, xr * iA);
    SETG(G_A, A);
    const real zb0 = X(6), zb1 = X(7), zb2 = X(8), zt0 = X(9), zt1 = X(10), zt2 = X(11);
    if (JAC) {
      SETG(G_J0, real(0.5) * A * (zt0 - zb0));  // J at the three columns (J linear in r, s)
      SETG(G_J1, real(0.5) * A * (zt1 - zb1));
      SETG(G_J2, real(0.5) * A * (zt2 - zb2));
    }
    // z_r, z_s are linear in t: z_r(t) = zr0 + t zr1 (likewise z_s), so
    // t_x J = y_r z_s - z_r y_s and t_y J = z_r x_s - x_r z_s are linear in t
    const real zr0 = real(0.25) * ((zb1 - zb0) + (zt1 - zt0)), zr1 = real(0.25) * ((zt1 - zt0) - (zb1 - zb0));
    const real zs0 = real(0.25) * ((zb2 - zb0) + (zt2 - zt0)), zs1 = real(0.25) * ((zt2 - zt0) - (zb2 - zb0));
    SETG(G_TX0, yr * zs0 - zr0 * ys);
    SETG(G_TX1, yr * zs1 - zr1 * ys);
    SETG(G_TY0, zr0 * xs - xr * zs0);
    SETG(G_TY1, zr1 * xs - xr * zs1);
  } else if (part < 3) {
    // triangle faces: n = c / |c| with c the edge cross product (outward), J_f = |c| / 4
    const bool top = part == 2;
    const real x0 = X(0), y0 = X(3), z0 = X(top ? 9 : 6);
    const real ax = X(1) - x0, ay = X(4) - y0, bx = X(2) - x0, by = X(5) - y0;
    const real az = X(top ? 10 : 7) - z0, bz = X(top ? 11 : 8) - z0;
    const real cx = ay * bz - az * by, cy = az * bx - ax * bz, cz = ax * by - ay * bx;
    const real cc = cx * cx + cy * cy + cz * cz, ic = rsqrt_r(cc), sc = top ? ic : -ic;
    SETG(top ? G_JFT : G_JFB, real(0.25) * cc * ic);
    const int n0 = top ? G_NT0 : G_NB0;
    SETG(n0 + 0, cx * sc);
    SETG(n0 + 1, cy * sc);
    SETG(n0 + 2, cz * sc);
  } else {
    const int ed = part - 3, ia = ed, ib = ed == 2 ? 0 : ed + 1;
    const real dx = X(ib) - X(ia), dy = X(3 + ib) - X(3 + ia);
    const real ll = dx * dx + dy * dy, il = rsqrt_r(ll);
    const real Le = ll * il;
    SETG(G_QNX0 + ed, dy * il);  // horizontal outward normal of the quad face
    SETG(G_QNY0 + ed, -dx * il);
    SETG(G_QCA0 + ed, real(0.25) * Le * (X(9 + ia) - X(6 + ia)));  // M~_e = ca Mea + cb Meb
    SETG(G_QCB0 + ed, real(0.25) * Le * (X(9 + ib) - X(6 + ib)));
  }
#undef SETG
}

// M^{tri,k} = sum_a J_a M_a with J_a = A h_a / 2 (Lemma 3.1) of wedge e from its
// vertices; L D L^T factor row by row into the block's table, in the stored
// factor's form (negated unit lower triangle, 1 / D_i on the diagonal).
template <int N>
__device__ __forceinline__ void factor_wedge(const AllOps<N, real>& O, const DevMesh<real>& M, int e, int lane, real* sL) {
  constexpr int Nt = nt_of(N);
  const int Kp = M.Kw_pad;
#define LQ(q) sL[(((q) >> 2) * kB + lane) * 4 + ((q) & 3)]
  const int v0 = M.w_vid[0 * Kp + e], v1 = M.w_vid[1 * Kp + e], v2 = M.w_vid[2 * Kp + e];
  const int v3 = M.w_vid[3 * Kp + e], v4 = M.w_vid[4 * Kp + e], v5 = M.w_vid[5 * Kp + e];
  const real x0 = M.vx[v0], y0 = M.vy[v0];
  const real Ah = real(0.125) * ((M.vx[v1] - x0) * (M.vy[v2] - y0) - (M.vx[v2] - x0) * (M.vy[v1] - y0));
  const real J0 = Ah * (M.vz[v3] - M.vz[v0]), J1 = Ah * (M.vz[v4] - M.vz[v1]), J2 = Ah * (M.vz[v5] - M.vz[v2]);
  auto mass = [&](int i, int l) {
    return J0 * O.w.Ma[0][i * Nt + l] + J1 * O.w.Ma[1][i * Nt + l] + J2 * O.w.Ma[2][i * Nt + l];
  };
  if constexpr (Nt <= 10) {
    // the whole factor in registers (its latency is what the block waits for), then four entries per store
    constexpr int NL4 = nl4_of(N);
    real F[NL4 * 4];
#pragma unroll
    for (int q = Nt * (Nt + 1) / 2; q < NL4 * 4; ++q) F[q] = real(0);
#pragma unroll
    for (int i = 0; i < Nt; ++i) {
      real row[Nt];  // l_il D_l
#pragma unroll
      for (int l = 0; l < i; ++l) {
        row[l] = mass(i, l);
#pragma unroll
        for (int k = 0; k < l; ++k) row[l] += row[k] * F[l * (l + 1) / 2 + k];
      }
      real d = mass(i, i);
#pragma unroll
      for (int k = 0; k < i; ++k) {
        const real nl = -(row[k] * F[k * (k + 1) / 2 + k]);
        d += row[k] * nl;
        F[i * (i + 1) / 2 + k] = nl;
      }
      F[i * (i + 1) / 2 + i] = real(1) / d;
    }
#pragma unroll
    for (int c = 0; c < NL4; ++c) st4(sL, (c * kB + lane) * 4, Q4{F[c * 4], F[c * 4 + 1], F[c * 4 + 2], F[c * 4 + 3]});
  } else {
#pragma unroll
    for (int i = 0; i < Nt; ++i) {
      real row[Nt];
#pragma unroll
      for (int l = 0; l < i; ++l) {
        row[l] = mass(i, l);
#pragma unroll
        for (int k = 0; k < l; ++k) row[l] += row[k] * LQ(l * (l + 1) / 2 + k);
      }
      real d = mass(i, i);
#pragma unroll
      for (int k = 0; k < i; ++k) {
        const real nl = -(row[k] * LQ(k * (k + 1) / 2 + k));
        d += row[k] * nl;
        LQ(i * (i + 1) / 2 + k) = nl;
      }
      LQ(i * (i + 1) / 2 + i) = real(1) / d;
    }
  }
#undef LQ
}

// X = (M^{tri,k})^{-1} W for the four right-hand sides of a slice (field pairs
// W01, W23) with the L D L^T factor of the block's table sL: forward sweep row
// by row, the diagonal, then the backward sweep in column-update form; four
// entries per shared load.  The table holds the negated unit lower triangle
// and 1 / D_i, so both sweeps are multiply-adds alone.
template <int N>
__device__ __forceinline__ void mass_solve(const real* sL, int lane, real2 (&W01)[nt_of(N)], real2 (&W23)[nt_of(N)]) {
  constexpr int Nt = nt_of(N);
  // row i of the factor, entries q = i (i + 1) / 2 + k, k = 0..i
  auto load_row = [&](int i, real (&Lr)[Nt]) {
    const int a0 = i * (i + 1) / 2;
#pragma unroll
    for (int c4 = a0 >> 2; c4 <= (a0 + i) >> 2; ++c4) {
      const Q4 v = ldop4(sL + (c4 * kB + lane) * 4);
      const real vv[4] = {v.p, v.u, v.v, v.w};
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const int k = c4 * 4 + q - a0;
        if (k >= 0 && k <= i) Lr[k] = vv[q];
      }
    }
  };
#pragma unroll
  for (int i = 1; i < Nt; ++i) {
    real Lr[Nt];
    load_row(i, Lr);
#pragma unroll
    for (int k = 0; k < i; ++k) {
      const real2 nl = dup2(Lr[k]);
      W01[i] = fma2(nl, W01[k], W01[i]);
      W23[i] = fma2(nl, W23[k], W23[i]);
    }
  }
#pragma unroll
  for (int i = 0; i < Nt; ++i) {
    // (read again: held from the sweep, the diagonal would cost Nt registers)
    const real2 d = dup2(sL[((i * (i + 3) / 2 >> 2) * kB + lane) * 4 + (i * (i + 3) / 2 & 3)]);
    W01[i] = mul2(W01[i], d);
    W23[i] = mul2(W23[i], d);
  }
#pragma unroll
  for (int i = Nt - 1; i > 0; --i) {
    real Lr[Nt];
    load_row(i, Lr);
#pragma unroll
    for (int k = 0; k < i; ++k) {
      const real2 nl = dup2(Lr[k]);
      W01[k] = fma2(nl, W01[i], W01[k]);
      W23[k] = fma2(nl, W23[i], W23[k]);
    }
  }
}

// L2 prefetch for block pb, half a wave after the caller's: its neighbour, code
// and material tables, so that the chain neighbour id -> neighbour trace starts
// from L2 instead of DRAM, and its state slab (N <= 4 with the stored factor;
// elsewhere the stage waits on arithmetic and it measured slower).
// 524,288 wedges, us per stage of a step: N = 3 264 without, 249 with the
// tables, 238 with the state too; N = 4 675, 662, 656; N = 2 119, 112, 109; a
// whole wave ahead gains less, the residual slab or the factor nothing.
template <int N>
__device__ __forceinline__ void prefetch_ahead(const DevMesh<real>& M, const real* qin, int pb, int lane, bool state) {
  if (pb >= M.nblk_w) return;
  const int64_t Kp = M.Kw_pad, at = int64_t(pb) * kB;
  if (lane < 13) {
    const void* p = lane < 5    ? static_cast<const void*>(M.w_nbr + lane * Kp + at)
                    : lane < 10 ? static_cast<const void*>(M.w_code + (lane - 5) * Kp + at)
                                : static_cast<const void*>(M.w_mat + (lane - 10) * Kp + at);
    asm volatile("prefetch.global.L2 [%0];" ::"l"(p));
  } else if (lane == 13 && state) {
    asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(qin + widx<N>(pb, 0, 0)),
                 "r"(uint32_t(4 * npw_of(N) * kB * sizeof(real))));
  }
}

// Fused low-storage Runge-Kutta update of a node: res <- a res + dt r, q_out <-
// g q_in + b res, r = kappa X_p, X_u / rho; or the plain right-hand side.  The
// residual is read only where a != 0 and stored only where a later stage reads
// it (StageArgs::res_store): of the five stages of a step the first reads none
// and the last stores none, a tenth of the step's traffic.
struct UpdateCoef {
  real2 s01, s23, dt2, a2, g2, b2;
  __device__ __forceinline__ UpdateCoef(const StageArgs<real>& A, real kappa, real irho)
      : s01(mk2(kappa, irho)), s23(dup2(irho)), dt2(dup2(A.dt)), a2(dup2(A.rk_a)), g2(dup2(A.rk_g)), b2(dup2(A.rk_b)) {}
  // g: packed index of the node; r0 its residual (0 where a = 0), q0 its state.
  // Scaled by the material, then by dt, node by node: a product kappa dt rounded
  // once per element would scale all of the element's updates by the same error,
  // which adds up over nodes and steps where single roundings average out (one
  // c^2 and rho, 1,024 wedges, N = 2, FP32, 1,000 steps: error 1.20e-6 with such
  // a product off by 5e-8, 1.06e-6 so; 1% of the FP64 small-mesh stage).
  __device__ __forceinline__ void node(const StageArgs<real>& A, bool rk, int64_t g, const real2 X01, const real2 X23,
                                       const Q4& r0, const Q4& q0) const {
    const real2 f01 = mul2(X01, s01), f23 = mul2(X23, s23);
    if (!rk || A.rhs_out != nullptr) {
      st4(rk ? A.rhs_out : A.q_out, g, Q4{f01.x, f01.y, f23.x, f23.y});
      if (!rk) return;
    }
    const real2 r01 = fma2(a2, mk2(r0.p, r0.u), mul2(dt2, f01));
    const real2 r23 = fma2(a2, mk2(r0.v, r0.w), mul2(dt2, f23));
    const real2 q01 = fma2(b2, r01, mul2(g2, mk2(q0.p, q0.u)));
    const real2 q23 = fma2(b2, r23, mul2(g2, mk2(q0.v, q0.w)));
    if (A.res_store) st4(A.res, g, Q4{r01.x, r01.y, r23.x, r23.y});
    st4(A.q_out, g, Q4{q01.x, q01.y, q23.x, q23.y});
  }
};
template <int N, bool RES_SMEM>
__device__ __forceinline__ void wedge_update(const StageArgs<real>& A, bool rk, const real* sq, const real* sr, int blk, int j,
                                             int lane, int e, real kappa, real irho, const real2 (&W01)[nt_of(N)],
                                             const real2 (&W23)[nt_of(N)]) {
  constexpr int Nt = nt_of(N);
  if (e >= A.m.Kw) return;
  const UpdateCoef U(A, kappa, irho);
#pragma unroll
  for (int i = 0; i < Nt; ++i) {
    const int n = j * Nt + i;
    const int64_t g = widx<N>(blk, n, lane);
    Q4 r0{0, 0, 0, 0};
    if (rk && A.rk_a != real(0)) r0 = RES_SMEM ? lds4(sr, n, lane) : ld4(A.res, g);
    U.node(A, rk, g, W01[i], W23[i], r0, lds4(sq, n, lane));
  }
}

// ---------------------------------------------------------------------------
// wedge stage on the CUDA cores
// ---------------------------------------------------------------------------
// Entry (m, code) of the neighbour's edge-node table, code = 2 * edge +
// reversed, m-th node of this side: the six candidates packed five bits each
// into one constant, so a lane with its own code extracts its node with a
// shift and a mask instead of an indexed constant load (which is replayed for
// every distinct index of the warp).
// (closed forms and masks throughout, so that they fold to constants in the
// unrolled loops at every order)
__host__ __device__ constexpr uint32_t edge_candidates(int N, int m) {
  return uint32_t(edge_node(N, 0, m)) | uint32_t(edge_node(N, 0, N - m)) << 5 | uint32_t(edge_node(N, 1, m)) << 10 |
         uint32_t(edge_node(N, 1, N - m)) << 15 | uint32_t(edge_node(N, 2, m)) << 20 | uint32_t(edge_node(N, 2, N - m)) << 25;
}
// D_r restricted to the edge b = 0 (rows a = 0..N) differentiates along the
// edge: only its own N + 1 nodes enter; D_s likewise on the edge a = 0.
__host__ __device__ constexpr bool dr_zero(int N, int i, int l) { return i <= N && l > N; }
template <int N>
struct EdgeA0 {
  static constexpr uint32_t nodes() {
    uint32_t m = 0;
    for (int b = 0; b <= N; ++b) m |= 1u << tri_idx(N, 0, b);
    return m;
  }
  static constexpr uint32_t mask = nodes();
};
template <int N>
__host__ __device__ constexpr bool ds_zero(int i, int l) {
  constexpr uint32_t m = EdgeA0<N>::mask;
  return ((m >> i) & 1u) != 0 && ((m >> l) & 1u) == 0;
}
// acc += {X[2h][l], X[2h + 1][l]} * x, leaving out rows known to be zero
// (FP32: the pair is one instruction and is left out when both rows are zero)
template <int NT>
__device__ __forceinline__ real2 fma_rows(const real* XP, int h, int l, real x, real2 acc, bool z0, bool z1) {
  if constexpr (sizeof(real) == 4) {
    if (z0 && (z1 || 2 * h + 1 >= NT)) return acc;
    return fma2(cpair(XP, NT, h, l), dup2(x), acc);
  } else {
    const real2 c = cpair(XP, NT, h, l);
    if (!z0) acc.x = fmar(c.x, x, acc.x);
    if (!z1 && 2 * h + 1 < NT) acc.y = fmar(c.y, x, acc.y);
    return acc;
  }
}
// {-s_p, -s_u}: the ghost state of a boundary face is the own trace with the
// pressure (Dirichlet) or the velocity (rigid) reversed; +1, +1 on interior
// faces.  The negated jump is then own + (-s) * neighbour, one multiply-add
// per component with no branch: rigid -2 u_n, Dirichlet -2 p as before.
__device__ __forceinline__ real2 ghost_signs(bool bnd, int bc) {
  return mk2(bnd && bc == 0 ? real(1) : real(-1), bnd && bc != 0 ? real(1) : real(-1));
}

// Flux pair (F_p, F_u), twice eq. (1)'s, of a triangle-face node with own
// state o, neighbour state v, normal n, -tau_p and -tau_u.  Explicit
// multiply-adds here and in the quadrilateral faces: every form of the stage
// gives the same bits.
__device__ __forceinline__ real2 tri_node_flux(const Q4& o, const Q4& v, real n0, real n1, real n2, const real2 s, real ntp,
                                               real ntu) {
  const real2 d01 = fma2(s, mk2(v.p, v.u), mk2(o.p, o.u));          // negated jumps of p, u_x
  const real2 d23 = fma2(dup2(s.y), mk2(v.v, v.w), mk2(o.v, o.w));  // and of u_y, u_z
  const real dn = fmar(n2, d23.y, fmar(n1, d23.x, n0 * d01.y));
  return mk2(fmar(ntp, d01.x, dn), fmar(ntu, dn, d01.x));
}
// Quadrilateral face ed of slice j: the fluxes along the edge times M~_e =
// (L_e / 4)(h_a Mea + h_b Meb) (ca, cb: half the two factors; identity in t),
// F_p in gp2 and F_u in gu2 by output pairs.
template <int N>
__device__ __forceinline__ void quad_edge(const AllOps<N, real>& O, const real* sq, int j, int lane, int ed,
                                          const Q4 (&tv)[N + 1], real nx, real ny, const real2 s, real tp, real tu, real ca,
                                          real cb, real2 (&gp2)[(N + 2) / 2], real2 (&gu2)[(N + 2) / 2]) {
  constexpr int Nt = nt_of(N), Nq = N + 1, NQH = (N + 2) / 2;
  const real2 ca2 = dup2(ca), cb2 = dup2(cb);
#pragma unroll
  for (int h = 0; h < NQH; ++h) gp2[h] = gu2[h] = dup2(real(0));
#pragma unroll
  for (int m = 0; m < Nq; ++m) {
    const Q4 o = lds4(sq, j * Nt + edge_node(N, ed, m), lane);
    const real2 d01 = fma2(s, mk2(tv[m].p, tv[m].u), mk2(o.p, o.u));
    const real d2 = fmar(s.y, tv[m].v, o.v);
    const real dn = fmar(nx, d01.y, ny * d2);
    const real2 Fp = dup2(fmar(-tp, d01.x, dn)), Fu = dup2(fmar(-tu, dn, d01.x));
#pragma unroll
    for (int h = 0; h < NQH; ++h) {
      const real2 w = fma2(cpair(O.w.MebP, Nq, h, m), cb2, mul2(cpair(O.w.MeaP, Nq, h, m), ca2));
      gp2[h] = fma2(w, Fp, gp2[h]);
      gu2[h] = fma2(w, Fu, gu2[h]);
    }
  }
}

// One stage of a 32-wedge block per N + 1 warps (lane = element, warp j =
// slice j), in the weak-in-t form
//   W_p = M (-(t_xJ D_t u + t_yJ D_t v + A D_t w)) + lifts,  W_u = -t_cJ M D_t p + lifts
// so M^tri is applied per slice to two vectors (the t-divergence and D_t p)
// and, once per element instead of once per slice, to the four triangle-face
// flux vectors: 2 + 4 / (N + 1) applications per slice where forming the four
// right-hand sides first takes 4.  Every lane reads its quadrilateral-face
// neighbours from global memory, also those in its own block (no per-lane
// choice between two address spaces), and a boundary face reads its own trace.
// Bound by memory latency and traffic at N <= 3 (a copy of the slabs and the
// traces alone takes 218 us of the 243 at N = 3), by issue and registers at
// N >= 4.  Instructions per warp, N = 3: 2,769 -> 2,240.  us per stage of a step
// on 524,288 wedges, with the skipped residual traffic and the prefetch: N = 3
// 301 -> 243, N = 4 774 -> 583; 30,118 wedges N = 5 326 -> 125.
// TF: the neighbour nodes of the triangle-face fluxes come from global memory
// and are requested before the slab arrives (meshes where some of them are
// tets or lie in another block, StageArgs::tri_far; two blocks per CTA:
// always); otherwise they are all in this block's slab.
// OTF: the mass factor is formed in the stage, by warp 1 while the slab is in
// flight (the other warps take its part of the geometry, and no traces are
// requested before the slab has arrived, whose registers the factor needs: 322
// us with, 304 without, 332 in an earlier form with two blocks per CTA; N = 3,
// 524,288 wedges).
// OP: M^tri on the CUDA cores, or (precision variants) on the tensor cores: the
// four right-hand sides of a slice are then formed first and pass through the
// warp's operand tile, which shares the residual slab's place.
template <int N, int BPC, bool TF, bool OTF, int OP = kOpFFMA>
__global__ void __launch_bounds__(32 * (N + 1) * BPC, wedge_min_ctas<N, BPC, OP>())
    k_wedge_stage(const StageArgs<real> A, bool rk) {
  constexpr int Nt = nt_of(N), Nq = N + 1, Np = Nt * Nq, NH = (Nt + 1) / 2, NQH = (Nq + 1) / 2;
  // FP32 at N >= 4: the operator products as loops over the input nodes (tables
  // by input node; three nodes unrolled, one, two or five measured slower)
  // instead of straight-line code, which missed the instruction cache and, at
  // N = 5, half of its constant loads: N = 4 622 -> 600 us per stage on 524,288
  // wedges, N = 5 613 -> 438 us on 131,072.  (FP64 waits on its pipe and gains
  // more from leaving out the zeros of D_s: N = 4 1,295 against 1,360 us.)
  constexpr bool rolled = WedgeOps<N, real>::by_input;
  constexpr int NHP = (NH + 1) / 2 * 2;
  static_assert(OP == kOpFFMA || (sizeof(real) == 4 && BPC == 1 && Nt <= 16), "tensor-core applies: FP32, Nt <= 16");
  using SM = WedgeSmem<N, OP>;
  const AllOps<N, real>& O = OPS<N>();
  extern __shared__ __align__(128) unsigned char smem_raw[];
  // block sb of this CTA: warps sb (N+1) .. sb (N+1) + N, one per slice
  const int sb = BPC == 1 ? 0 : threadIdx.x / (32 * Nq);
  const int j = (threadIdx.x >> 5) - sb * Nq;
  const bool leader = int(threadIdx.x) == sb * 32 * Nq;
  // [0] state slab (and stored factor), [1] residual slab, [2] vertex coordinates
  uint64_t* bar = reinterpret_cast<uint64_t*>(smem_raw + 32 * sb);
  int* status = reinterpret_cast<int*>(smem_raw + 32 * sb + 24);
  real* base = reinterpret_cast<real*>(smem_raw + 32 * BPC) + sb * SM::reals;
  real* sq = base + SM::q;
  real* sr = base + SM::r;
  real* sL = base + SM::L;
  real* sF = base + SM::F;  // [face][node][lane] pairs (F_p, F_u), then M^tri applied to each
  real* sG = base + SM::G;
  const DevMesh<real>& M = A.m;
  const real* qin = A.q_in;
  const int lane = threadIdx.x & 31;
  const int blk = blockIdx.x * BPC + sb;
  if (blk >= M.nblk_w) return;  // padding block of the last CTA
  const int e = blk * kB + lane;
  const int Kp = M.Kw_pad;
  constexpr uint32_t slab_bytes = uint32_t(4 * Np * kB * sizeof(real));
  const bool res_async = rk && stage_res<N>() && A.rk_a != real(0);
#define GEO(item) sG[(item) * kB + lane]
  // the warps of one block synchronise among themselves (named barrier 1 + sb)
  auto block_sync = [&]() {
    static_assert(BPC <= 2, "at most two blocks per CTA");
    if (sb == 0) asm volatile("bar.sync 1, %0;" ::"n"(32 * Nq) : "memory");
    else asm volatile("bar.sync 2, %0;" ::"n"(32 * Nq) : "memory");
  };
  // 0. bulk copies of the block's state (and residual) slabs; geometry meanwhile
  constexpr int NL4 = nl4_of(N);
  constexpr uint32_t fac_bytes = uint32_t(NL4 * 4 * kB * sizeof(real));
  constexpr bool stored = !OTF;
  constexpr uint32_t xyz_bytes = uint32_t(12 * kB * sizeof(real));
  if (A.pdl) {
    pdl_launch_dependents();
    pdl_wait();
  }
  if (leader) {
    mbar_init(&bar[0], 1);
    mbar_init(&bar[1], 1);
    mbar_init(&bar[2], 1);
    fence_mbar_init();
    // the block's vertex coordinates first (the geometry waits on them alone), in
    // the flux table's place, which is written after the barrier below
    mbar_expect_tx(&bar[2], xyz_bytes);
    bulk_g2s(sF, M.w_xyz + int64_t(blk) * 12 * kB, xyz_bytes, &bar[2]);
    mbar_expect_tx(&bar[0], slab_bytes + (stored ? fac_bytes : 0u));
    bulk_g2s(sq, qin + int64_t(blk) * 4 * Np * kB, slab_bytes, &bar[0]);
    // stored mass factor: straight into the factor table with the state slab
    if (stored) bulk_g2s(sL, M.w_fac + int64_t(blk) * NL4 * 4 * kB, fac_bytes, &bar[0]);
    if (res_async && OP == kOpFFMA) {
      mbar_expect_tx(&bar[1], slab_bytes);
      bulk_g2s(sr, A.res + int64_t(blk) * 4 * Np * kB, slab_bytes, &bar[1]);
    } else if (!res_async && rk && A.rk_a != real(0)) {
      // not staged: to L2 at least, for the update (N = 5: 438 -> 411 us per stage on 131,072 wedges)
      asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(A.res + int64_t(blk) * 4 * Np * kB), "r"(slab_bytes));
    }
  }
  if (j == N) prefetch_ahead<N>(M, qin, blk + kHalfSMs * wedge_min_ctas<N, BPC, OP>() * BPC, lane, N <= 4 && stored);
  // face neighbours, their impedances and the source flag, loaded while the
  // slabs are in flight; so are (N <= 3) the neighbour traces
  const real kappa = M.w_mat[0 * Kp + e], irho = M.w_mat[1 * Kp + e], zM = M.w_mat[2 * Kp + e];
  int qnbr[3], qcode[3];
#pragma unroll
  for (int ed = 0; ed < 3; ++ed) {
    qnbr[ed] = M.w_nbr[(2 + ed) * Kp + e];
    qcode[ed] = M.w_code[(2 + ed) * Kp + e];
  }
  const int tnbr[2] = {M.w_nbr[0 * Kp + e], M.w_nbr[1 * Kp + e]};
  const int tcode[2] = {M.w_code[0 * Kp + e], M.w_code[1 * Kp + e]};
  // trace of quadrilateral face ed: nodes of slice j of the neighbour (or, on a boundary, of the element itself)
  auto trace = [&](int ed, Q4 (&t)[Nq]) {
    const bool bnd = qnbr[ed] < 0;
    const int nbe = bnd ? e : qnbr[ed], sh = 5 * (bnd ? 2 * ed : qcode[ed]);
    const real* nb = qin + widx<N>(nbe >> 5, j * Nt, nbe & 31);
#pragma unroll
    for (int m = 0; m < Nq; ++m) t[m] = ld4(nb, int((edge_candidates(N, m) >> sh) & 31u) * (kB * 4));
  };
  // requested here at N <= 3, after the slab has arrived at N = 4 (before it they
  // cost spills: 649 against 578 us per stage on 524,288 wedges, 600 face by
  // face), face by face at N = 5
  constexpr bool early = N <= 3 && !OTF, mid = N == 4 || (N <= 3 && OTF);
  Q4 nv[early || mid ? 3 : 1][Nq];
  if constexpr (early) {
#pragma unroll
    for (int ed = 0; ed < 3; ++ed) trace(ed, nv[ed]);
  }
  // the neighbour node of triangle-face flux node t of this warp (round-robin
  // over the warps, bottom then top): a tet's face node, or a wedge's bottom or
  // top node; a boundary face reads its own node
  constexpr int NTT = (2 * Nt + Nq - 1) / Nq;
  auto tri_nbr_node = [&](int t) {
    const int idx = j + t * Nq;
    const int fb = idx >= Nt ? 1 : 0;
    const int k = idx - fb * Nt;
    const int nbr = fb ? tnbr[1] : tnbr[0], code = fb ? tcode[1] : tcode[0];
    const bool bnd = nbr < 0;
    const int nbe = bnd ? e : nbr, nf = bnd ? fb : (code >> 4) & 3;
    const int nk = bnd ? k : O.tab.tri_perm[code & 15][k];
    if constexpr (TF) {
      const bool ntet = !bnd && (code & kCodeTet) != 0;
      const int node = ntet ? O.tab.tet_face[nf][nk] : (nf ? N * Nt : 0) + nk;
      return ld4(qin, ntet ? tidx<N>(M.tet_off, nbe >> 5, node, nbe & 31) : widx<N>(nbe >> 5, node, nbe & 31));
    } else {
      return lds4(sq, (nf ? N * Nt : 0) + nk, nbe & 31);
    }
  };
  Q4 tnv[TF ? NTT : 1];
  if constexpr (TF) {
#pragma unroll
    for (int t = 0; t < NTT; ++t)
      if (j + t * Nq < 2 * Nt) tnv[t] = tri_nbr_node(t);
  }
  real zPq[3], zPt[2];
#pragma unroll
  for (int ed = 0; ed < 3; ++ed) zPq[ed] = qnbr[ed] < 0 ? zM : M.w_mat[2 * Kp + qnbr[ed]];
#pragma unroll
  for (int fb = 0; fb < 2; ++fb)
    zPt[fb] = tnbr[fb] < 0 ? zM
                           : ((tcode[fb] & kCodeTet) ? M.t_mat[2 * M.Kt_pad + tnbr[fb]] : M.w_mat[2 * Kp + tnbr[fb]]);
  const bool src = M.nsrc > 0 && has_source(M, 6, e);
  // the parts of the geometry, round-robin over the warps, each of which waits
  // for the coordinates itself: the barrier's initialisation must be visible first
  block_sync();
  const bool geo_ok = __all_sync(0xffffffffu, mbar_wait_bounded(&bar[2], 0));
  if (geo_ok) {
#pragma unroll 1
    for (int p = OTF ? (j == 1 ? kGeoParts : j - (j > 1)) : j; p < kGeoParts; p += OTF ? Nq - 1 : Nq)
      wedge_geometry_part<false>(p, sF, sG, lane);
  } else if (lane == 0) {
    atomicOr(M.err, kErrTimeout);
  }
  if (OTF && j == 1) {
    factor_wedge<N>(O, M, e, lane, sL);  // while the slabs are in flight
  }
  if (leader) *status = (mbar_wait_bounded(&bar[0], 0) && geo_ok) ? 1 : 0;
  block_sync();
  if (*reinterpret_cast<volatile int*>(status) == 0) {
    // a copy never arrived: report, let any copy in flight drain, leave
    if (leader) {
      atomicOr(M.err, kErrTimeout);
      if (res_async && OP == kOpFFMA) mbar_wait_bounded(&bar[1], 0);
      mbar_wait_bounded(&bar[0], 0);
      mbar_wait_bounded(&bar[2], 0);
    }
    return;
  }

  if constexpr (mid) {
#pragma unroll
    for (int ed = 0; ed < 3; ++ed) trace(ed, nv[ed]);
  }
  // 1. triangle-face node fluxes (bottom then top), spread round-robin over
  //    the warps, without the factor 1/2 (it enters with the lift)
  {
    real ntp[2], ntu[2];
#pragma unroll
    for (int fb = 0; fb < 2; ++fb) {
      real tp, tu;
      taus(A.flux, zM, zPt[fb], tp, tu);
      ntp[fb] = -tp;
      ntu[fb] = -tu;
    }
#pragma unroll
    for (int t = 0; t < NTT; ++t) {
      const int idx = j + t * Nq;
      if (idx >= 2 * Nt) break;
      const int fb = idx >= Nt ? 1 : 0;
      const int k = idx - fb * Nt;
      const real n0 = GEO(fb ? G_NT0 : G_NB0), n1 = GEO(fb ? G_NT1 : G_NB1), n2 = GEO(fb ? G_NT2 : G_NB2);
      const Q4 o = lds4(sq, (fb ? N * Nt : 0) + k, lane);
      Q4 v;
      if constexpr (TF) v = tnv[t];
      else v = tri_nbr_node(t);
      const real2 F = tri_node_flux(o, v, n0, n1, n2, ghost_signs((fb ? tnbr[1] : tnbr[0]) < 0, A.bc), fb ? ntp[1] : ntp[0],
                                    fb ? ntu[1] : ntu[0]);
      *reinterpret_cast<real2*>(sF + ((fb * Nt + k) * kB + lane) * 2) = F;
    }
  }
  block_sync();
  // 2. M^tri applied in place to the four flux vectors (bottom F_p, F_u, top
  //    F_p, F_u), one per warp
#pragma unroll 1
  for (int v = OP == kOpFFMA ? j : 4; v < 4; v += Nq) {
    real* f = sF + ((v >> 1) * Nt * kB + lane) * 2 + (v & 1);
    real2 acc[NH];
    if constexpr (rolled) {
#pragma unroll
      for (int h = 0; h < NH; ++h) acc[h] = dup2(real(0));
#pragma unroll 3
      for (int l = 0; l < Nt; ++l) {
        const real2 xx = dup2(f[l * kB * 2]);
#pragma unroll
        for (int h = 0; h < NH; ++h) acc[h] = fma2(cpair(O.w.MT, NHP, l, h), xx, acc[h]);
      }
    } else {
      real G[Nt];
#pragma unroll
      for (int i = 0; i < Nt; ++i) G[i] = f[i * kB * 2];
      apply_pairs<Nt, Nt>(O.w.MP, G, acc);
    }
#pragma unroll
    for (int i = 0; i < Nt; ++i) f[i * kB * 2] = pair_row(acc, i);
  }

  // 3. quadrilateral faces of slice j: M~_e F_p into W_p (by output pairs), M~_e F_u kept per edge
  real2 Wp[NH];
  real gu[3][Nq];
#pragma unroll
  for (int h = 0; h < NH; ++h) Wp[h] = dup2(real(0));
#pragma unroll
  for (int ed = 0; ed < 3; ++ed) {
    Q4 tv[Nq];
    if constexpr (early || mid) {
#pragma unroll
      for (int m = 0; m < Nq; ++m) tv[m] = nv[ed][m];
    } else {
      trace(ed, tv);
    }
    const real nx = GEO(G_QNX0 + ed), ny = GEO(G_QNY0 + ed);
    real tp, tu;
    taus(A.flux, zM, zPq[ed], tp, tu);
    real2 gp2[NQH], gu2[NQH];
    quad_edge<N>(O, sq, j, lane, ed, tv, nx, ny, ghost_signs(qnbr[ed] < 0, A.bc), tp, tu, real(0.5) * GEO(G_QCA0 + ed),
                 real(0.5) * GEO(G_QCB0 + ed), gp2, gu2);
#pragma unroll
    for (int m = 0; m < Nq; ++m) {
      const int i = edge_node(N, ed, m);
      if (i & 1) Wp[i >> 1].y += pair_row(gp2, m);
      else Wp[i >> 1].x += pair_row(gp2, m);
      gu[ed][m] = pair_row(gu2, m);
    }
  }

  // 4. t-parts of slice j: the t-divergence dd = -(t_xJ D_t u_x + t_yJ D_t u_y
  //    + A D_t u_z) and D_t p; W_p += M^tri dd, Mdp = M^tri D_t p
  const real tj = O.w.gll[j];
  const real ntx = -fmar(tj, GEO(G_TX1), GEO(G_TX0)), nty = -fmar(tj, GEO(G_TY1), GEO(G_TY0)), nA = -GEO(G_A);
  real dtr[Nq];
#pragma unroll
  for (int m = 0; m < Nq; ++m) dtr[m] = O.w.Dt[j * Nq + m];
  // node i: D_t of the four fields as two packed pairs (p, u_x) and (u_y, u_z)
  auto t_part = [&](int i, real& dp, real& dd) {
    real2 dpu = dup2(real(0)), dvw = dup2(real(0));
#pragma unroll
    for (int m = 0; m < Nq; ++m) {
      const Q4 v = lds4(sq, m * Nt + i, lane);
      const real2 d2 = dup2(dtr[m]);
      dpu = fma2(d2, mk2(v.p, v.u), dpu);
      dvw = fma2(d2, mk2(v.v, v.w), dvw);
    }
    dp = dpu.x;
    dd = fmar(ntx, dpu.y, fmar(nty, dvw.x, nA * dvw.y));
  };
  real2 W01[Nt], W23[Nt];
  // the coefficients of the four right-hand sides, and node i's values from the
  // flux pairs, the pressure's (a) and D_t p's (d) part
  struct Lift {
    real2 b01, t01, b23, t23, n23;
    real ntx;
    __device__ __forceinline__ void node(const real2 fb, const real2 ft, real a, real d, real2& w01, real2& w23) const {
      w01 = fma2(fb, b01, fma2(ft, t01, mk2(a, ntx * d)));
      w23 = fma2(dup2(fb.y), b23, fma2(dup2(ft.y), t23, mul2(dup2(d), n23)));
    }
  };
  auto lift_coef = [&]() {
    const real cb = real(0.5) * GEO(G_JFB) * O.w.ell0[j], ct = real(0.5) * GEO(G_JFT) * O.w.ellN[j];
    return Lift{mk2(cb, cb * GEO(G_NB0)), mk2(ct, ct * GEO(G_NT0)), mk2(cb * GEO(G_NB1), cb * GEO(G_NB2)),
                mk2(ct * GEO(G_NT1), ct * GEO(G_NT2)), mk2(nty, nA), ntx};
  };
  auto flux_pair = [&](int fb, int i) { return *reinterpret_cast<const real2*>(sF + ((fb * Nt + i) * kB + lane) * 2); };
  if constexpr (OP == kOpFFMA) {
    real2 Mdp[NH];
    if constexpr (rolled) {
      // a node's two values go into both products at once
#pragma unroll
      for (int h = 0; h < NH; ++h) Mdp[h] = dup2(real(0));
#pragma unroll 3
      for (int l = 0; l < Nt; ++l) {
        real dp, dd;
        t_part(l, dp, dd);
        const real2 xx = dup2(dd), pp = dup2(dp);
#pragma unroll
        for (int h = 0; h < NH; ++h) {
          const real2 c = cpair(O.w.MT, NHP, l, h);
          Wp[h] = fma2(c, xx, Wp[h]);
          Mdp[h] = fma2(c, pp, Mdp[h]);
        }
      }
    } else {
      real dp[Nt], dd[Nt];
#pragma unroll
      for (int i = 0; i < Nt; ++i) t_part(i, dp[i], dd[i]);
#pragma unroll
      for (int l = 0; l < Nt; ++l) {
        const real2 xx = dup2(dd[l]);
#pragma unroll
        for (int h = 0; h < NH; ++h) Wp[h] = fma2(cpair(O.w.MP, Nt, h, l), xx, Wp[h]);
      }
      apply_pairs<Nt, Nt>(O.w.MP, dp, Mdp);
    }
    block_sync();  // M^tri has been applied to the flux vectors
    // 5. right-hand sides of the mass solve by field pairs (p, u_x), (u_y, u_z):
    //    the lifted triangle-face fluxes, -t_cJ M D_t p and the quadrilateral faces
    const Lift C = lift_coef();
#pragma unroll
    for (int i = 0; i < Nt; ++i) C.node(flux_pair(0, i), flux_pair(1, i), pair_row(Wp, i), pair_row(Mdp, i), W01[i], W23[i]);
  } else {
    // 4, 5 on the tensor cores: the four vectors of every element of the block go
    // to this warp's tile (columns lane * 4 + field), M^tri is applied one 16 x 8
    // output tile at a time in place, and each lane reads its element's results back
    real* sT = base + SM::T + j * Nt * kTP;
    const Lift C = lift_coef();
#pragma unroll
    for (int i = 0; i < Nt; ++i) {
      real dp, dd;
      real2 g01, g23;
      t_part(i, dp, dd);
      C.node(flux_pair(0, i), flux_pair(1, i), dd, dp, g01, g23);
      *reinterpret_cast<float4*>(sT + tile_at(i, lane * 4)) = make_float4(g01.x, g01.y, g23.x, g23.y);
    }
    __syncwarp();
    {
      AFrag<OP> Am;
      afrag_load<Nt, OP>(O.w.M, lane, Am);
      const int g = lane >> 2, t = lane & 3;
#pragma unroll 2
      for (int nt = 0; nt < 16; ++nt) {
        BFrag<OP> Bf;
        bfrag_load<Nt, OP>(sT, nt * 8 + g, lane, Bf);
        float d[4] = {0.f, 0.f, 0.f, 0.f};
        op_mma<Nt, OP>(Am, Bf, d);
        if (g < Nt) *reinterpret_cast<float2*>(sT + tile_at(g, nt * 8 + 2 * t)) = make_float2(d[0], d[1]);
        if (g + 8 < Nt) *reinterpret_cast<float2*>(sT + tile_at(g + 8, nt * 8 + 2 * t)) = make_float2(d[2], d[3]);
      }
    }
    __syncwarp();
#pragma unroll
    for (int i = 0; i < Nt; ++i) {
      const float4 w = *reinterpret_cast<const float4*>(sT + tile_at(i, lane * 4));
      W01[i] = mk2(w.x + pair_row(Wp, i), w.y);
      W23[i] = mk2(w.z, w.w);
    }
    if (res_async) {
      // every warp is done with its tile: the residual slab may now land in their space
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
      block_sync();
      if (leader) {
        mbar_expect_tx(&bar[1], slab_bytes);
        bulk_g2s(sr, A.res + int64_t(blk) * 4 * Np * kB, slab_bytes, &bar[1]);
      }
    }
  }
  {
#pragma unroll
    for (int ed = 0; ed < 3; ++ed) {
      const real nx = GEO(G_QNX0 + ed), ny = GEO(G_QNY0 + ed);
#pragma unroll
      for (int m = 0; m < Nq; ++m) {
        const int i = edge_node(N, ed, m);
        W01[i].y = fmar(nx, gu[ed][m], W01[i].y);
        W23[i].x = fmar(ny, gu[ed][m], W23[i].x);
      }
    }
  }
  mass_solve<N>(sL, lane, W01, W23);
  // 6. strong r, s parts of slice j (constant metric terms, Lemma 3.1), D_r and
  //    D_s applied by output pairs, node l of the slice at a time
  {
    const real rx = GEO(G_RX), ry = GEO(G_RY), sx = GEO(G_SX), sy = GEO(G_SY);
    real2 dv[NH], pr[NH], ps[NH];
#pragma unroll
    for (int h = 0; h < NH; ++h) dv[h] = pr[h] = ps[h] = dup2(real(0));
    if constexpr (rolled) {
      // nodes of the edge b = 0, then the others, for which the first pairs of
      // D_r's rows are zero
      constexpr int H0 = (N + 1) / 2;
#pragma unroll 3
      for (int l = 0; l <= N; ++l) {
        const Q4 v = lds4(sq, j * Nt + l, lane);
        const real2 ab = fma2(dup2(v.u), mk2(rx, sx), mul2(dup2(v.v), mk2(ry, sy)));
        const real2 a = dup2(ab.x), b = dup2(ab.y), p = dup2(v.p);
#pragma unroll
        for (int h = 0; h < NH; ++h) {
          const real2 r = cpair(O.w.DrT, NHP, l, h), q = cpair(O.w.DsT, NHP, l, h);
          dv[h] = fma2(q, b, fma2(r, a, dv[h]));
          pr[h] = fma2(r, p, pr[h]);
          ps[h] = fma2(q, p, ps[h]);
        }
      }
#pragma unroll 3
      for (int l = N + 1; l < Nt; ++l) {
        const Q4 v = lds4(sq, j * Nt + l, lane);
        const real2 ab = fma2(dup2(v.u), mk2(rx, sx), mul2(dup2(v.v), mk2(ry, sy)));
        const real2 a = dup2(ab.x), b = dup2(ab.y), p = dup2(v.p);
#pragma unroll
        for (int h = 0; h < NH; ++h) {
          const real2 q = cpair(O.w.DsT, NHP, l, h);
          if (h >= H0) {
            const real2 r = cpair(O.w.DrT, NHP, l, h);
            dv[h] = fma2(r, a, dv[h]);
            pr[h] = fma2(r, p, pr[h]);
          }
          dv[h] = fma2(q, b, dv[h]);
          ps[h] = fma2(q, p, ps[h]);
        }
      }
    } else {
#pragma unroll
      for (int l = 0; l < Nt; ++l) {
        const Q4 v = lds4(sq, j * Nt + l, lane);
        const real2 ab = fma2(dup2(v.u), mk2(rx, sx), mul2(dup2(v.v), mk2(ry, sy)));
#pragma unroll
        for (int h = 0; h < NH; ++h) {
          const bool r0 = dr_zero(N, 2 * h, l), r1 = dr_zero(N, 2 * h + 1, l);
          const bool s0 = ds_zero<N>(2 * h, l), s1 = ds_zero<N>(2 * h + 1, l);
          dv[h] = fma_rows<Nt>(O.w.DrP, h, l, ab.x, dv[h], r0, r1);
          dv[h] = fma_rows<Nt>(O.w.DsP, h, l, ab.y, dv[h], s0, s1);
          pr[h] = fma_rows<Nt>(O.w.DrP, h, l, v.p, pr[h], r0, r1);
          ps[h] = fma_rows<Nt>(O.w.DsP, h, l, v.p, ps[h], s0, s1);
        }
      }
    }
#pragma unroll
    for (int i = 0; i < Nt; ++i) W01[i].x -= pair_row(dv, i);
#pragma unroll
    for (int i = 0; i < Nt; ++i) {
      const real pri = pair_row(pr, i), psi = pair_row(ps, i);
      W01[i].y = fmar(-rx, pri, fmar(-sx, psi, W01[i].y));
      W23[i].x = fmar(-ry, pri, fmar(-sy, psi, W23[i].x));
    }
  }
  // 7. fused low-storage Runge-Kutta update (or plain right-hand side)
  if (res_async && !mbar_wait_bounded(&bar[1], 0)) {
    if (lane == 0) atomicOr(M.err, kErrTimeout);
    mbar_wait_bounded(&bar[1], 0);
    return;
  }
  if (src) add_sources(M, 6, e, j * Nt, Np, M.clock[A.clk] + A.c_stage * double(A.dt), W01);
  wedge_update<N, stage_res<N>()>(A, rk, sq, sr, blk, j, lane, e, kappa, irho, W01, W23);
#undef GEO
}

// Small meshes.  With a block per N + 1 warps a mesh of a few hundred wedges
// leaves most SMs idle and its stage takes as long as one warp's instruction
// chain (and in FP64 as the few busy SMs' FP64 pipes).  Here a CTA takes one
// slice j of a block and its four warps share the slice's work, warp f solving
// for field f: N + 1 times the CTAs and a quarter of the chain, for the
// triangle-face fluxes formed once per slice instead of once per block.  Every
// result is accumulated in k_wedge_stage's order: same bits.
template <int N>
struct WideSmem {
  static constexpr int Nt = nt_of(N), Nq = N + 1, Np = Nt * Nq;
  static constexpr int q = 0;                         // [Np][32][4] state slab
  static constexpr int r = q + 4 * Np * kB;           // [Nt][32][4] the slice's residual
  static constexpr int L = r + 4 * Nt * kB;           // [NL4][32][4] mass factor
  static constexpr int F = L + nl4_of(N) * 4 * kB;    // [2][Nt][32] flux pairs; then the results [4][Nt][32]
  static constexpr int G = F + 4 * Nt * kB;           // [G_STAGE][32] geometry
  static constexpr int D = G + G_STAGE * kB;          // [2][Nt][32] D_t p, t-divergence; then [3][Nt][32] strong parts
  static constexpr int E = D + 3 * Nt * kB;           // [3][Nq][2][32] quadrilateral-face lifts of F_p, F_u
  static constexpr int reals = E + 6 * Nq * kB;
};
template <int N>
__host__ __device__ constexpr int wide_smem_bytes() {
  return 32 + WideSmem<N>::reals * int(sizeof(real));
}
// (FP64 at N = 5 does not fit a CTA's shared memory)
template <int N>
__host__ __device__ constexpr bool wide_fits() {
  return wide_smem_bytes<N>() <= 227 * 1024;
}

// row pairs [H0, H1) of the strong divergence D_r (r.u) + D_s (s.u) of slice j
template <int N, int H0, int H1, int HA>
__device__ __forceinline__ void div_rows(const AllOps<N, real>& O, const real* sq, int j, int lane, real rx, real ry, real sx,
                                         real sy, real2 (&dv)[HA]) {
  constexpr int Nt = nt_of(N);
#pragma unroll
  for (int h = 0; h < HA; ++h) dv[h] = dup2(real(0));
#pragma unroll
  for (int l = 0; l < Nt; ++l) {
    const Q4 v = lds4(sq, j * Nt + l, lane);
    const real2 ab = fma2(dup2(v.u), mk2(rx, sx), mul2(dup2(v.v), mk2(ry, sy)));
#pragma unroll
    for (int h = H0; h < H1; ++h) {
      dv[h - H0] = fma_rows<Nt>(O.w.DrP, h, l, ab.x, dv[h - H0], dr_zero(N, 2 * h, l), dr_zero(N, 2 * h + 1, l));
      dv[h - H0] = fma_rows<Nt>(O.w.DsP, h, l, ab.y, dv[h - H0], ds_zero<N>(2 * h, l), ds_zero<N>(2 * h + 1, l));
    }
  }
}

template <int N>
__global__ void __launch_bounds__(128) k_wedge_wide(const StageArgs<real> A, bool rk) {
  constexpr int Nt = nt_of(N), Nq = N + 1, Np = Nt * Nq, NH = (Nt + 1) / 2, NQH = (Nq + 1) / 2, NL4 = nl4_of(N);
  using SM = WideSmem<N>;
  const AllOps<N, real>& O = OPS<N>();
  extern __shared__ __align__(128) unsigned char smem_raw[];
  // [0] state slab (and stored factor), [1] residual, [2] vertex coordinates
  uint64_t* bar = reinterpret_cast<uint64_t*>(smem_raw);
  int* status = reinterpret_cast<int*>(smem_raw + 24);
  real* base = reinterpret_cast<real*>(smem_raw + 32);
  real* sq = base + SM::q;
  real* sr = base + SM::r;
  real* sL = base + SM::L;
  real* sF = base + SM::F;
  real* sG = base + SM::G;
  real* sD = base + SM::D;
  real* sE = base + SM::E;
  const DevMesh<real>& M = A.m;
  const real* qin = A.q_in;
  const int lane = threadIdx.x & 31, f = threadIdx.x >> 5;
  const int blk = blockIdx.x / Nq, j = blockIdx.x - blk * Nq;
  const int e = blk * kB + lane, Kp = M.Kw_pad;
  constexpr uint32_t slab_bytes = uint32_t(4 * Np * kB * sizeof(real)), res_bytes = uint32_t(4 * Nt * kB * sizeof(real));
  constexpr uint32_t fac_bytes = uint32_t(NL4 * 4 * kB * sizeof(real)), xyz_bytes = uint32_t(12 * kB * sizeof(real));
  const bool stored = M.w_fac != nullptr, res_async = rk && A.rk_a != real(0);
#define GEO(item) sG[(item) * kB + lane]
  if (threadIdx.x == 0) {
    mbar_init(&bar[0], 1);
    mbar_init(&bar[1], 1);
    mbar_init(&bar[2], 1);
    fence_mbar_init();
    mbar_expect_tx(&bar[2], xyz_bytes);
    bulk_g2s(sF, M.w_xyz + int64_t(blk) * 12 * kB, xyz_bytes, &bar[2]);  // in the flux table's place, written later
    mbar_expect_tx(&bar[0], slab_bytes + (stored ? fac_bytes : 0u));
    if (stored) bulk_g2s(sL, M.w_fac + int64_t(blk) * NL4 * 4 * kB, fac_bytes, &bar[0]);
  }
  pdl_launch_dependents();
  // neighbours: warp f < 3 takes quadrilateral face f, all warps share the triangle-face nodes
  const real kappa = M.w_mat[0 * Kp + e], irho = M.w_mat[1 * Kp + e], zM = M.w_mat[2 * Kp + e];
  const int ed = f < 3 ? f : 0;
  const int qnbr = M.w_nbr[(2 + ed) * Kp + e], qcode = M.w_code[(2 + ed) * Kp + e];
  const int tnbr[2] = {M.w_nbr[0 * Kp + e], M.w_nbr[1 * Kp + e]};
  const int tcode[2] = {M.w_code[0 * Kp + e], M.w_code[1 * Kp + e]};
  const real zPq = qnbr < 0 ? zM : M.w_mat[2 * Kp + qnbr];
  real ntp[2], ntu[2];
#pragma unroll
  for (int fb = 0; fb < 2; ++fb) {
    const real zP = tnbr[fb] < 0 ? zM
                                 : ((tcode[fb] & kCodeTet) ? M.t_mat[2 * M.Kt_pad + tnbr[fb]] : M.w_mat[2 * Kp + tnbr[fb]]);
    real tp, tu;
    taus(A.flux, zM, zP, tp, tu);
    ntp[fb] = -tp;
    ntu[fb] = -tu;
  }
  const bool src = f == 0 && M.nsrc > 0 && has_source(M, 6, e);
  // the geometry needs the mesh alone: before the wait for the previous stage
  __syncthreads();  // the mbarriers are initialised
  const bool ok = __all_sync(0xffffffffu, mbar_wait_bounded(&bar[2], 0));
  if (ok) {
#pragma unroll 1
    for (int p = 3 - f; p < kGeoParts; p += 4) wedge_geometry_part<false>(p, sF, sG, lane);
  } else if (lane == 0) {
    atomicOr(M.err, kErrTimeout);
  }
  pdl_wait();
  if (threadIdx.x == 0) {
    bulk_g2s(sq, qin + int64_t(blk) * 4 * Np * kB, slab_bytes, &bar[0]);
    if (res_async) {
      mbar_expect_tx(&bar[1], res_bytes);
      bulk_g2s(sr, A.res + widx<N>(blk, j * Nt, 0), res_bytes, &bar[1]);
    }
  }
  Q4 tv[Nq];
  {
    const bool bnd = qnbr < 0;
    const int nbe = bnd ? e : qnbr, sh = 5 * (bnd ? 2 * ed : qcode);
    const real* nb = qin + widx<N>(nbe >> 5, j * Nt, nbe & 31);
#pragma unroll
    for (int m = 0; m < Nq; ++m) tv[m] = ld4(nb, int((edge_candidates(N, m) >> sh) & 31u) * (kB * 4));
  }
  constexpr int NTT = (2 * Nt + 3) / 4;
  Q4 tnv[NTT];
#pragma unroll
  for (int t = 0; t < NTT; ++t) {
    const int idx = f + 4 * t;
    if (idx >= 2 * Nt) break;
    const int fb = idx >= Nt ? 1 : 0, k = idx - fb * Nt;
    const int nbr = fb ? tnbr[1] : tnbr[0], code = fb ? tcode[1] : tcode[0];
    const bool bnd = nbr < 0, ntet = !bnd && (code & kCodeTet) != 0;
    const int nbe = bnd ? e : nbr, nf = bnd ? fb : (code >> 4) & 3;
    const int nk = bnd ? k : O.tab.tri_perm[code & 15][k];
    const int node = ntet ? O.tab.tet_face[nf][nk] : (nf ? N * Nt : 0) + nk;
    tnv[t] = ld4(qin, ntet ? tidx<N>(M.tet_off, nbe >> 5, node, nbe & 31) : widx<N>(nbe >> 5, node, nbe & 31));
  }
  if (threadIdx.x == 96) *status = (ok && mbar_wait_bounded(&bar[0], 0)) ? 1 : 0;
  if (f == 0 && !stored) factor_wedge<N>(O, M, e, lane, sL);
  __syncthreads();
  if (*reinterpret_cast<volatile int*>(status) == 0) {
    // a copy never arrived: report, let the copies in flight drain, leave
    if (threadIdx.x == 0) {
      atomicOr(M.err, kErrTimeout);
      mbar_wait_bounded(&bar[0], 0);
      if (res_async) mbar_wait_bounded(&bar[1], 0);
      mbar_wait_bounded(&bar[2], 0);
    }
    return;
  }

  // 1. triangle-face node fluxes; the lifts of quadrilateral face f; D_t p and
  //    the t-divergence of the slice's nodes, four warps abreast
#pragma unroll
  for (int t = 0; t < NTT; ++t) {
    const int idx = f + 4 * t;
    if (idx >= 2 * Nt) break;
    const int fb = idx >= Nt ? 1 : 0, k = idx - fb * Nt;
    const real n0 = GEO(fb ? G_NT0 : G_NB0), n1 = GEO(fb ? G_NT1 : G_NB1), n2 = GEO(fb ? G_NT2 : G_NB2);
    const Q4 o = lds4(sq, (fb ? N * Nt : 0) + k, lane);
    const real2 F = tri_node_flux(o, tnv[t], n0, n1, n2, ghost_signs((fb ? tnbr[1] : tnbr[0]) < 0, A.bc),
                                  fb ? ntp[1] : ntp[0], fb ? ntu[1] : ntu[0]);
    *reinterpret_cast<real2*>(sF + ((fb * Nt + k) * kB + lane) * 2) = F;
  }
  if (f < 3) {
    real tp, tu;
    taus(A.flux, zM, zPq, tp, tu);
    const real nx = GEO(G_QNX0 + ed), ny = GEO(G_QNY0 + ed);
    const real ca = real(0.5) * GEO(G_QCA0 + ed), cb = real(0.5) * GEO(G_QCB0 + ed);
    const real2 s = ghost_signs(qnbr < 0, A.bc);
    real2 gp2[NQH], gu2[NQH];
    if (f == 0) quad_edge<N>(O, sq, j, lane, 0, tv, nx, ny, s, tp, tu, ca, cb, gp2, gu2);
    else if (f == 1) quad_edge<N>(O, sq, j, lane, 1, tv, nx, ny, s, tp, tu, ca, cb, gp2, gu2);
    else quad_edge<N>(O, sq, j, lane, 2, tv, nx, ny, s, tp, tu, ca, cb, gp2, gu2);
#pragma unroll
    for (int m = 0; m < Nq; ++m) {
      sE[((f * Nq + m) * 2 + 0) * kB + lane] = pair_row(gp2, m);
      sE[((f * Nq + m) * 2 + 1) * kB + lane] = pair_row(gu2, m);
    }
  }
  const real tj = O.w.gll[j];
  const real ntx = -fmar(tj, GEO(G_TX1), GEO(G_TX0)), nty = -fmar(tj, GEO(G_TY1), GEO(G_TY0)), nA = -GEO(G_A);
  {
    real dtr[Nq];
#pragma unroll
    for (int m = 0; m < Nq; ++m) dtr[m] = O.w.Dt[j * Nq + m];
#pragma unroll
    for (int i = f; i < Nt; i += 4) {
      real2 dpu = dup2(real(0)), dvw = dup2(real(0));
#pragma unroll
      for (int m = 0; m < Nq; ++m) {
        const Q4 v = lds4(sq, m * Nt + i, lane);
        const real2 d2 = dup2(dtr[m]);
        dpu = fma2(d2, mk2(v.p, v.u), dpu);
        dvw = fma2(d2, mk2(v.v, v.w), dvw);
      }
      sD[(0 * Nt + i) * kB + lane] = dpu.x;
      sD[(1 * Nt + i) * kB + lane] = fmar(ntx, dpu.y, fmar(nty, dvw.x, nA * dvw.y));
    }
  }
  __syncthreads();
  // 2. M^tri in place on flux vector f (bottom F_p, F_u, top F_p, F_u); M^tri on
  //    the t-divergence, onto the pressure lifts (warp 0), or on D_t p
  {
    real* v = sF + ((f >> 1) * Nt * kB + lane) * 2 + (f & 1);
    real G[Nt];
#pragma unroll
    for (int i = 0; i < Nt; ++i) G[i] = v[i * kB * 2];
    real2 acc[NH];
    apply_pairs<Nt, Nt>(O.w.MP, G, acc);
#pragma unroll
    for (int i = 0; i < Nt; ++i) v[i * kB * 2] = pair_row(acc, i);
  }
  real2 Wm[NH];
#pragma unroll
  for (int h = 0; h < NH; ++h) Wm[h] = dup2(real(0));
  if (f == 0) {
#pragma unroll
    for (int ec = 0; ec < 3; ++ec)
#pragma unroll
      for (int m = 0; m < Nq; ++m) {
        const int i = edge_node(N, ec, m);
        const real g = sE[((ec * Nq + m) * 2 + 0) * kB + lane];
        if (i & 1) Wm[i >> 1].y += g;
        else Wm[i >> 1].x += g;
      }
  }
  {
    const real* d = sD + (f == 0 ? Nt : 0) * kB + lane;
#pragma unroll
    for (int l = 0; l < Nt; ++l) {
      const real2 xx = dup2(d[l * kB]);
#pragma unroll
      for (int h = 0; h < NH; ++h) Wm[h] = fma2(cpair(O.w.MP, Nt, h, l), xx, Wm[h]);
    }
  }
  __syncthreads();
  // 3. right-hand side of field f and its mass solve
  real W[Nt];
  {
    const real cb = real(0.5) * GEO(G_JFB) * O.w.ell0[j], ct = real(0.5) * GEO(G_JFT) * O.w.ellN[j];
    const real cbf = f == 0 ? cb : cb * GEO(G_NB0 + f - 1), ctf = f == 0 ? ct : ct * GEO(G_NT0 + f - 1);
    const real nf = f == 1 ? ntx : (f == 2 ? nty : nA);
    const real* F = sF + lane * 2 + (f == 0 ? 0 : 1);
#pragma unroll
    for (int i = 0; i < Nt; ++i) {
      const real md = pair_row(Wm, i);
      W[i] = fmar(F[i * kB * 2], cbf, fmar(F[(Nt + i) * kB * 2], ctf, f == 0 ? md : nf * md));
    }
    if (f == 1 || f == 2) {
#pragma unroll
      for (int ec = 0; ec < 3; ++ec) {
        const real n = GEO((f == 1 ? G_QNX0 : G_QNY0) + ec);
#pragma unroll
        for (int m = 0; m < Nq; ++m) {
          const int i = edge_node(N, ec, m);
          W[i] = fmar(n, sE[((ec * Nq + m) * 2 + 1) * kB + lane], W[i]);
        }
      }
    }
  }
  {
    auto load_row = [&](int i, real (&Lr)[Nt]) {
      const int a0 = i * (i + 1) / 2;
#pragma unroll
      for (int c4 = a0 >> 2; c4 <= (a0 + i) >> 2; ++c4) {
        const Q4 v = ldop4(sL + (c4 * kB + lane) * 4);
        const real vv[4] = {v.p, v.u, v.v, v.w};
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          const int k = c4 * 4 + q - a0;
          if (k >= 0 && k <= i) Lr[k] = vv[q];
        }
      }
    };
    real d[Nt];
#pragma unroll
    for (int i = 0; i < Nt; ++i) {
      real Lr[Nt];
      load_row(i, Lr);
#pragma unroll
      for (int k = 0; k < i; ++k) W[i] = fmar(Lr[k], W[k], W[i]);
      d[i] = Lr[i];
    }
#pragma unroll
    for (int i = 0; i < Nt; ++i) W[i] *= d[i];
#pragma unroll
    for (int i = Nt - 1; i > 0; --i) {
      real Lr[Nt];
      load_row(i, Lr);
#pragma unroll
      for (int k = 0; k < i; ++k) W[k] = fmar(Lr[k], W[i], W[k]);
    }
  }
  // 4. strong r, s parts: rows of div u on warps 0 and 2, D_r p on warp 1, D_s p
  //    on warp 3, exchanged through shared memory
  constexpr int HA = (NH + 1) / 2;
  const real rx = GEO(G_RX), ry = GEO(G_RY), sx = GEO(G_SX), sy = GEO(G_SY);
  real2 dv[HA], pd[NH];
  if (f == 0) {
    div_rows<N, 0, HA>(O, sq, j, lane, rx, ry, sx, sy, dv);
  } else if (f == 2) {
    div_rows<N, HA, NH>(O, sq, j, lane, rx, ry, sx, sy, dv);
#pragma unroll
    for (int i = 2 * HA; i < Nt; ++i) sD[i * kB + lane] = pair_row(dv, i - 2 * HA);
  } else {
#pragma unroll
    for (int h = 0; h < NH; ++h) pd[h] = dup2(real(0));
    if (f == 1) {
#pragma unroll
      for (int l = 0; l < Nt; ++l) {
        const real p = sq[((j * Nt + l) * kB + lane) * 4];
#pragma unroll
        for (int h = 0; h < NH; ++h)
          pd[h] = fma_rows<Nt>(O.w.DrP, h, l, p, pd[h], dr_zero(N, 2 * h, l), dr_zero(N, 2 * h + 1, l));
      }
    } else {
#pragma unroll
      for (int l = 0; l < Nt; ++l) {
        const real p = sq[((j * Nt + l) * kB + lane) * 4];
#pragma unroll
        for (int h = 0; h < NH; ++h)
          pd[h] = fma_rows<Nt>(O.w.DsP, h, l, p, pd[h], ds_zero<N>(2 * h, l), ds_zero<N>(2 * h + 1, l));
      }
    }
    real* out = sD + ((f == 1 ? 1 : 2) * Nt) * kB + lane;
#pragma unroll
    for (int i = 0; i < Nt; ++i) out[i * kB] = pair_row(pd, i);
  }
  __syncthreads();
  if (f == 0) {
#pragma unroll
    for (int i = 0; i < Nt; ++i) W[i] -= i < 2 * HA ? pair_row(dv, i < 2 * HA ? i : 0) : sD[i * kB + lane];
    if (src) add_sources(M, 6, e, j * Nt, Np, M.clock[A.clk] + A.c_stage * double(A.dt), W);
  } else if (f < 3) {
    const real nr = f == 1 ? -rx : -ry, ns = f == 1 ? -sx : -sy;
#pragma unroll
    for (int i = 0; i < Nt; ++i)
      W[i] = fmar(nr, sD[(1 * Nt + i) * kB + lane], fmar(ns, sD[(2 * Nt + i) * kB + lane], W[i]));
  }
#pragma unroll
  for (int i = 0; i < Nt; ++i) sF[(f * Nt + i) * kB + lane] = W[i];
  // 5. the update, four fields of a node per thread
  if (!__syncthreads_and(!res_async || mbar_wait_bounded(&bar[1], 0))) {
    // the residual never arrived: report, let the copy drain, leave
    if (threadIdx.x == 0) {
      atomicOr(M.err, kErrTimeout);
      mbar_wait_bounded(&bar[1], 0);
    }
    return;
  }
  if (e < M.Kw) {
    const UpdateCoef U(A, kappa, irho);
#pragma unroll
    for (int i = f; i < Nt; i += 4) {
      const real2 W01 = mk2(sF[(0 * Nt + i) * kB + lane], sF[(1 * Nt + i) * kB + lane]);
      const real2 W23 = mk2(sF[(2 * Nt + i) * kB + lane], sF[(3 * Nt + i) * kB + lane]);
      Q4 r0{0, 0, 0, 0};
      if (res_async) r0 = lds4(sr, i, lane);
      U.node(A, rk, widx<N>(blk, j * Nt + i, lane), W01, W23, r0, lds4(sq, j * Nt + i, lane));
    }
  }
#undef GEO
}

// ---------------------------------------------------------------------------
// tet stage: one 32-tet block per CTA (lane = tet), 4 warps.  Bulk copies move
// the tet operators (laid out per warp chunk by output pairs), the block's
// vertex coordinates and its state slab into shared memory.  Warp f forms the
// normal and the fluxes of face f; warp w forms the volume terms, the lift and
// the update of output nodes [w C, w C + C).  Bound by instruction issue (and
// by the FP64 pipe in FP64), so what the four warps would repeat is done once:
// each face's normal, and (p, -w) with w the reference-direction velocities of
// every node, which the volume terms read (tet_wtab): 2,380 -> 1,919
// instructions per warp at N = 3.  us per stage: 221,184 tets N = 3 FP32 92.3 ->
// 88.1, 41,472 tets N = 4 45.2 -> 41.4 and N = 5 171 -> 99; 27,648 tets N = 3 FP64
// 184 -> 150.
// All warps run the same code.
// ---------------------------------------------------------------------------
template <int N>
__host__ __device__ constexpr int tet_chunk() {  // output nodes per warp
  return (npt_of(N) + 3) / 4;
}
template <int N>
__host__ __device__ constexpr int tet_pairs() {  // output pairs per warp
  return (tet_chunk<N>() + 1) / 2;
}
template <int N>
__host__ __device__ constexpr int tet_rec() {  // reals of a (warp, l) record: D_r, D_s, D_t pairs (a multiple of 4)
  return (6 * tet_pairs<N>() + 3) / 4 * 4;
}
template <int N>
__host__ __device__ constexpr int tet_lrec() {  // reals of a (warp, face node) lift record (a multiple of 4)
  return (2 * tet_pairs<N>() + 3) / 4 * 4;
}
template <int N>
__host__ __device__ constexpr int tet_drecs() {  // reals of all derivative records
  return 4 * npt_of(N) * tet_rec<N>();
}
template <int N>
__host__ __device__ constexpr int tet_ops_image_reals() {  // the global image t_ops: D records, then the lift
  return tet_drecs<N>() + 4 * (4 * nt_of(N)) * tet_lrec<N>();
}
// The table of (p, -w): N <= 3, where it costs no CTA per SM.  In FP32 the
// residual slab is bulk-copied into its place once the volume terms are done
// (elsewhere the update reads the residual from global memory).
template <int N>
__host__ __device__ constexpr bool tet_wtab() {
  return N <= 3;
}
template <int N>
__host__ __device__ constexpr bool tet_stage_res() {
  return sizeof(real) == 4 && tet_wtab<N>();
}
template <int N>
__host__ __device__ constexpr int tet_work_reals() {  // slab, flux pairs, coordinates, normals, (p, -w) table
  return 4 * npt_of(N) * kB + 8 * nt_of(N) * kB + 24 * kB + (tet_wtab<N>() ? 4 * npt_of(N) * kB : 0);
}
// 128-byte header (4 mbarriers), operators, slab [Np][32][4], flux pairs
// [4 faces][Nt][32][2], vertex coordinates [12][32], normals [4][3][32], (p, -w) [Np][32][4]
template <int N>
__host__ __device__ constexpr int tet_smem_bytes() {
  return 128 + (tet_ops_image_reals<N>() + tet_work_reals<N>()) * int(sizeof(real));
}
static_assert(tet_smem_bytes<NORD>() <= 227 * 1024, "the whole operator image fits a CTA at every order and precision");
// acc.x += a.x b, acc.y += a.y b; FP64 leaves out the second where it is padding
template <bool PAD>
__device__ __forceinline__ real2 fma_pair(const real2 a, real b, const real2 acc) {
  if constexpr (sizeof(real) == 8 && PAD) return mk2(fmar(a.x, b, acc.x), acc.y);
  else return fma2(a, dup2(b), acc);
}

template <int N>
__global__ void __launch_bounds__(128, (sizeof(REAL) == 4) ? (N >= 4 ? 3 : 5) : 2)
    k_tet_stage(const StageArgs<real> A, bool rk) {
  constexpr int Np = npt_of(N), Nt = nt_of(N), C = tet_chunk<N>(), CH = tet_pairs<N>(), RS = tet_rec<N>(), LS = tet_lrec<N>();
  const AllOps<N, real>& O = OPS<N>();
  extern __shared__ __align__(128) unsigned char smem_raw[];
  uint64_t* bar = reinterpret_cast<uint64_t*>(smem_raw);  // [0] operators, [1] coordinates, [2] state, [3] residual
  real* sOp = reinterpret_cast<real*>(smem_raw + 128);
  real* sL = sOp + tet_drecs<N>();  // lift [warp][4 Nt][LS]
  real* sq = sOp + tet_ops_image_reals<N>();
  real* sF = sq + 4 * Np * kB;
  real* sX = sF + 8 * Nt * kB;
  real* sN = sX + 12 * kB;
  real* sW = sN + 12 * kB;  // (p, -w), then the residual slab
  constexpr bool stage_res = tet_stage_res<N>();
  const bool res_async = stage_res && rk && A.rk_a != real(0);
  const DevMesh<real>& M = A.m;
  const int lane = threadIdx.x & 31;
  const int w = threadIdx.x >> 5;
  const int blk = blockIdx.x;
  const int e = blk * kB + lane;
  const int Kp = M.Kt_pad;
  constexpr uint32_t slab_bytes = uint32_t(4 * Np * kB * sizeof(real)), xyz_bytes = uint32_t(12 * kB * sizeof(real));
  constexpr uint32_t ops_bytes = uint32_t(tet_ops_image_reals<N>() * sizeof(real));
  if (threadIdx.x == 0) {
    mbar_init(&bar[0], 1);
    mbar_init(&bar[1], 1);
    mbar_init(&bar[2], 1);
    mbar_init(&bar[3], 1);
    fence_mbar_init();
    mbar_expect_tx(&bar[1], xyz_bytes);
    bulk_g2s(sX, M.t_xyz + int64_t(blk) * 12 * kB, xyz_bytes, &bar[1]);
    mbar_expect_tx(&bar[2], slab_bytes);
    bulk_g2s(sq, A.q_in + M.tet_off + int64_t(blk) * 4 * Np * kB, slab_bytes, &bar[2]);
    mbar_expect_tx(&bar[0], ops_bytes);
    bulk_g2s(sOp, M.t_ops, ops_bytes, &bar[0]);
  }
  // face neighbours, impedances, material and the source flag while the copies fly
  const real kappa = M.t_mat[0 * Kp + e], irho = M.t_mat[1 * Kp + e], zM = M.t_mat[2 * Kp + e];
  const int nbr = M.t_nbr[w * Kp + e], code = M.t_code[w * Kp + e];  // this warp's face w
  const real zP = nbr < 0 ? zM : ((code & kCodeTet) ? M.t_mat[2 * Kp + nbr] : M.w_mat[2 * M.Kw_pad + nbr]);
  const bool src = M.nsrc > 0 && has_source(M, 4, e);
  // out-of-block neighbour face nodes of this warp's face, requested before the waits
  Q4 nvs[Nt];
  const bool bnd = nbr < 0;
  const bool ntet = !bnd && (code & kCodeTet) != 0;
  const int nbe = bnd ? e : nbr;
  const bool inblk = bnd || (ntet && (nbe >> 5) == blk);
  const int nfc = (code >> 4) & 3, perm = code & 15;
  if (!inblk) {
    const real* nb = A.q_in + (ntet ? tidx<N>(M.tet_off, nbe >> 5, 0, nbe & 31) : widx<N>(nbe >> 5, 0, nbe & 31));
#pragma unroll
    for (int k = 0; k < Nt; ++k) {
      const int nk = O.tab.tri_perm[perm][k];
      nvs[k] = ldg4(nb, int64_t(ntet ? O.tab.tet_face[nfc][nk] : (nfc ? N * Nt : 0) + nk) * (kB * 4));
    }
  }
  __syncthreads();  // the mbarriers are initialised

  // affine geometry: x = sum_v lambda_v X_v on the bi-unit reference tet
  bool ok = __all_sync(0xffffffffu, mbar_wait_bounded(&bar[1], 0));
  real nR[3][3], n0, n1, n2, sj;  // -d r_m / d x_d; this warp's face: outward unit normal, J_f / J
  {
    auto X = [&](int v, int d) { return sX[(v * 3 + d) * kB + lane]; };
    real G[3][3];  // G[d][m] = d x_d / d r_m
#pragma unroll
    for (int d = 0; d < 3; ++d) {
      const real xd = X(0, d);
#pragma unroll
      for (int m = 0; m < 3; ++m) G[d][m] = real(0.5) * (X(m + 1, d) - xd);
    }
    const real J = G[0][0] * (G[1][1] * G[2][2] - G[1][2] * G[2][1]) -
                   G[0][1] * (G[1][0] * G[2][2] - G[1][2] * G[2][0]) + G[0][2] * (G[1][0] * G[2][1] - G[1][1] * G[2][0]);
    const real iJ = real(1) / J, niJ = -iJ;
    nR[0][0] = (G[1][1] * G[2][2] - G[1][2] * G[2][1]) * niJ;
    nR[0][1] = (G[0][2] * G[2][1] - G[0][1] * G[2][2]) * niJ;
    nR[0][2] = (G[0][1] * G[1][2] - G[0][2] * G[1][1]) * niJ;
    nR[1][0] = (G[1][2] * G[2][0] - G[1][0] * G[2][2]) * niJ;
    nR[1][1] = (G[0][0] * G[2][2] - G[0][2] * G[2][0]) * niJ;
    nR[1][2] = (G[0][2] * G[1][0] - G[0][0] * G[1][2]) * niJ;
    nR[2][0] = (G[1][0] * G[2][1] - G[1][1] * G[2][0]) * niJ;
    nR[2][1] = (G[0][1] * G[2][0] - G[0][0] * G[2][1]) * niJ;
    nR[2][2] = (G[0][0] * G[1][1] - G[0][1] * G[1][0]) * niJ;
    // face w: vertices {0,1,2}, {0,1,3}, {1,2,3}, {0,2,3}, opposite 3, 2, 0, 1
    const int a0 = w == 2 ? 1 : 0, a1 = w < 2 ? 1 : 2, a2 = w == 0 ? 2 : 3, ao = (0x1023 >> (4 * w)) & 3;
    const real px = X(a0, 0), py = X(a0, 1), pz = X(a0, 2);
    const real ax = X(a1, 0) - px, ay = X(a1, 1) - py, az = X(a1, 2) - pz;
    const real bx = X(a2, 0) - px, by = X(a2, 1) - py, bz = X(a2, 2) - pz;
    const real cx = ay * bz - az * by, cy = az * bx - ax * bz, cz = ax * by - ay * bx;
    const real cc = cx * cx + cy * cy + cz * cz, ic = rsqrt_r(cc);
    const real ox = X(ao, 0) - px, oy = X(ao, 1) - py, oz = X(ao, 2) - pz;
    const real sc = (cx * ox + cy * oy + cz * oz > 0) ? -ic : ic;  // away from the opposite vertex
    n0 = sc * cx;
    n1 = sc * cy;
    n2 = sc * cz;
    sj = real(0.25) * cc * ic * iJ;
    sN[(w * 3 + 0) * kB + lane] = n0;
    sN[(w * 3 + 1) * kB + lane] = n1;
    sN[(w * 3 + 2) * kB + lane] = n2;
  }
  ok = __all_sync(0xffffffffu, mbar_wait_bounded(&bar[2], 0)) && ok;

  // fluxes of face w, scaled by J_f / J, into the shared flux table
  {
    real tp, tu;
    taus(A.flux, zM, zP, tp, tu);
    const real2 s = ghost_signs(bnd, A.bc);
    const real hs = real(0.5) * sj;
    // the neighbour's face nodes in this block's own slab (a boundary face reads its own)
    if (inblk) {
#pragma unroll
      for (int k = 0; k < Nt; ++k) {
        const int nk = bnd ? k : O.tab.tri_perm[perm][k];
        nvs[k] = lds4(sq, bnd ? O.tab.tet_face[w][k] : O.tab.tet_face[nfc][nk], nbe & 31);
      }
    }
#pragma unroll
    for (int k = 0; k < Nt; ++k) {
      const Q4 o = lds4(sq, O.tab.tet_face[w][k], lane);
      const real2 F = mul2(tri_node_flux(o, nvs[k], n0, n1, n2, s, -tp, -tu), dup2(hs));
      *reinterpret_cast<real2*>(sF + ((w * Nt + k) * kB + lane) * 2) = F;
    }
  }
  const int I0 = w * C;  // this warp's output nodes
  if constexpr (tet_wtab<N>()) {
    // (p, -w) of this warp's nodes, w_m = sum_d (d r_m / d x_d) u_d
#pragma unroll
    for (int c = 0; c < C; ++c) {
      if (I0 + c < Np) {
        const Q4 v = lds4(sq, I0 + c, lane);
        st4(sW, ((I0 + c) * kB + lane) * 4,
            Q4{v.p, fmar(nR[0][0], v.u, fmar(nR[0][1], v.v, nR[0][2] * v.w)),
               fmar(nR[1][0], v.u, fmar(nR[1][1], v.v, nR[1][2] * v.w)),
               fmar(nR[2][0], v.u, fmar(nR[2][1], v.v, nR[2][2] * v.w))});
      }
    }
  }
  ok = __all_sync(0xffffffffu, mbar_wait_bounded(&bar[0], 0)) && ok;
  if (!__syncthreads_and(ok)) {
    // a copy never arrived: report, let the copies in flight drain, leave
    if (threadIdx.x == 0) {
      atomicOr(M.err, kErrTimeout);
      mbar_wait_bounded(&bar[0], 0);
      mbar_wait_bounded(&bar[1], 0);
      mbar_wait_bounded(&bar[2], 0);
    }
    return;
  }

  // results of the warp's outputs by pairs (c, c + 1): ap the pressure, au[d]
  // the velocity components; first the volume terms
  constexpr bool odd = (C & 1) != 0;  // the last pair's second row is padding
  real2 ap[CH], au[3][CH];
  {
    real2 dr[CH], ds[CH], dt[CH];
#pragma unroll
    for (int h = 0; h < CH; ++h) ap[h] = dr[h] = ds[h] = dt[h] = dup2(real(0));
    const real* rec = sOp + w * Np * RS;
#pragma unroll 4
    for (int l = 0; l < Np; ++l) {
      Q4 v;
      if constexpr (tet_wtab<N>()) {
        v = lds4(sW, l, lane);
      } else {
        const Q4 u = lds4(sq, l, lane);
        v = Q4{u.p, fmar(nR[0][0], u.u, fmar(nR[0][1], u.v, nR[0][2] * u.w)),
               fmar(nR[1][0], u.u, fmar(nR[1][1], u.v, nR[1][2] * u.w)),
               fmar(nR[2][0], u.u, fmar(nR[2][1], u.v, nR[2][2] * u.w))};
      }
      real d[RS];
#pragma unroll
      for (int c4 = 0; c4 < RS; c4 += 4) {
        const Q4 t = ldop4(rec + l * RS + c4);
        d[c4] = t.p;
        d[c4 + 1] = t.u;
        d[c4 + 2] = t.v;
        d[c4 + 3] = t.w;
      }
#pragma unroll
      for (int h = 0; h < CH; ++h) {
        const real2 r2 = mk2(d[2 * h], d[2 * h + 1]), s2 = mk2(d[2 * (CH + h)], d[2 * (CH + h) + 1]),
                    t2 = mk2(d[2 * (2 * CH + h)], d[2 * (2 * CH + h) + 1]);
        if (odd && h == CH - 1) {
          dr[h] = fma_pair<true>(r2, v.p, dr[h]);
          ds[h] = fma_pair<true>(s2, v.p, ds[h]);
          dt[h] = fma_pair<true>(t2, v.p, dt[h]);
          ap[h] = fma_pair<true>(t2, v.w, fma_pair<true>(s2, v.v, fma_pair<true>(r2, v.u, ap[h])));
        } else {
          dr[h] = fma_pair<false>(r2, v.p, dr[h]);
          ds[h] = fma_pair<false>(s2, v.p, ds[h]);
          dt[h] = fma_pair<false>(t2, v.p, dt[h]);
          ap[h] = fma_pair<false>(t2, v.w, fma_pair<false>(s2, v.v, fma_pair<false>(r2, v.u, ap[h])));
        }
      }
    }
#pragma unroll
    for (int d = 0; d < 3; ++d)
#pragma unroll
      for (int h = 0; h < CH; ++h)
        au[d][h] = fma2(dup2(nR[0][d]), dr[h], fma2(dup2(nR[1][d]), ds[h], mul2(dup2(nR[2][d]), dt[h])));
  }
  if (res_async) {
    // every warp is done with the (p, -w) table: the residual slab may land in its place
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    __syncthreads();
    if (threadIdx.x == 0) {
      mbar_expect_tx(&bar[3], slab_bytes);
      bulk_g2s(sW, A.res + M.tet_off + int64_t(blk) * 4 * Np * kB, slab_bytes, &bar[3]);
    }
  }
  // the lift of the four faces: this warp's records [4 Nt][LS]
  {
    const real* lw = sL + w * (4 * Nt) * LS;
#pragma unroll
    for (int f = 0; f < 4; ++f) {
      real2 lu[CH];
#pragma unroll
      for (int h = 0; h < CH; ++h) lu[h] = dup2(real(0));
#pragma unroll 5
      for (int k = 0; k < Nt; ++k) {
        const real2 F = *reinterpret_cast<const real2*>(sF + ((f * Nt + k) * kB + lane) * 2);
        real d[LS];
#pragma unroll
        for (int c4 = 0; c4 < LS; c4 += 4) {
          const Q4 t = ldop4(lw + (f * Nt + k) * LS + c4);
          d[c4] = t.p;
          d[c4 + 1] = t.u;
          d[c4 + 2] = t.v;
          d[c4 + 3] = t.w;
        }
#pragma unroll
        for (int h = 0; h < CH; ++h) {
          const real2 L = mk2(d[2 * h], d[2 * h + 1]);
          if (odd && h == CH - 1) {
            ap[h] = fma_pair<true>(L, F.x, ap[h]);
            lu[h] = fma_pair<true>(L, F.y, lu[h]);
          } else {
            ap[h] = fma_pair<false>(L, F.x, ap[h]);
            lu[h] = fma_pair<false>(L, F.y, lu[h]);
          }
        }
      }
#pragma unroll
      for (int d = 0; d < 3; ++d) {
        const real2 nd = dup2(sN[(f * 3 + d) * kB + lane]);
#pragma unroll
        for (int h = 0; h < CH; ++h) au[d][h] = fma2(nd, lu[h], au[d][h]);
      }
    }
  }
  real p[C];
#pragma unroll
  for (int c = 0; c < C; ++c) p[c] = pair_row(ap, c);
  if (src) add_sources(M, 4, e, I0, Np, M.clock[A.clk] + A.c_stage * double(A.dt), p);
  if (res_async && !__all_sync(0xffffffffu, mbar_wait_bounded(&bar[3], 0))) {
    // the residual slab never arrived: report, let the copy drain, leave
    if (lane == 0) {
      atomicOr(M.err, kErrTimeout);
      mbar_wait_bounded(&bar[3], 0);
    }
    return;
  }
  if (e < M.Kt) {
    const UpdateCoef U(A, kappa, irho);
#pragma unroll
    for (int c = 0; c < C; ++c) {
      if (I0 + c < Np) {
        const int i = I0 + c;
        const int64_t g = tidx<N>(M.tet_off, blk, i, lane);
        Q4 r0{0, 0, 0, 0};
        if (rk && A.rk_a != real(0)) r0 = stage_res ? lds4(sW, i, lane) : ld4(A.res, g);
        U.node(A, rk, g, mk2(p[c], pair_row(au[0], c)), mk2(pair_row(au[1], c), pair_row(au[2], c)), r0, lds4(sq, i, lane));
      }
    }
  }
}

// ---------------------------------------------------------------------------
// canonical <-> packed layout
// ---------------------------------------------------------------------------
// Canonical [shot][field][node] <-> packed [block][node][lane][field] layout.
// One CTA per 32-element block at a time: the block's values pass through a
// [field][node][lane] shared tile (lane pitch 33, so neither phase has bank
// conflicts), the canonical side is read or written one element's contiguous
// node run at a time and the packed side in 16-byte [node][lane] records.
// Padding lanes (e >= K) are neither read nor written.
template <int N>
__host__ __device__ constexpr int pack_smem_bytes() {
  return 4 * npw_of(N) * 33 * int(sizeof(real));
}

template <int N>
__global__ void __launch_bounds__(256) k_pack(const DevMesh<real> M, const real* __restrict__ canon,
                                              real* __restrict__ packed, bool unpack) {
  constexpr int Npw = npw_of(N), Npt = npt_of(N);
  extern __shared__ __align__(128) unsigned char smem_raw[];
  real* tile = reinterpret_cast<real*>(smem_raw);  // [4][Np][33]
  real* cw = const_cast<real*>(canon);
  const int64_t T = M.total_nodes;
  for (int b = blockIdx.x; b < M.nblk_w + M.nblk_t; b += gridDim.x) {
    const bool tet = b >= M.nblk_w;
    const int blk = tet ? b - M.nblk_w : b;
    const int Np = tet ? Npt : Npw, K = tet ? M.Kt : M.Kw;
    const int64_t* cmap = tet ? M.t_canon : M.w_canon;
    real* pk = packed + (tet ? tidx<N>(M.tet_off, blk, 0, 0) : widx<N>(blk, 0, 0));
    const int items = Np * kB;
    if (!unpack) {
      for (int t = threadIdx.x; t < items; t += blockDim.x) {
        const int l = t / Np, n = t - l * Np, e = blk * kB + l;
        if (e < K) {
          const int64_t c = cmap[e] + n;
#pragma unroll
          for (int f = 0; f < 4; ++f) tile[(f * Np + n) * 33 + l] = canon[f * T + c];
        }
      }
      __syncthreads();
      for (int t = threadIdx.x; t < items; t += blockDim.x) {
        const int l = t & 31, n = t >> 5;
        if (blk * kB + l < K)
          st4(pk, int64_t(t) * 4,
              Q4{tile[(0 * Np + n) * 33 + l], tile[(1 * Np + n) * 33 + l], tile[(2 * Np + n) * 33 + l],
                 tile[(3 * Np + n) * 33 + l]});
      }
    } else {
      for (int t = threadIdx.x; t < items; t += blockDim.x) {
        const int l = t & 31, n = t >> 5;
        if (blk * kB + l < K) {
          const Q4 v = ld4(pk, int64_t(t) * 4);
          tile[(0 * Np + n) * 33 + l] = v.p;
          tile[(1 * Np + n) * 33 + l] = v.u;
          tile[(2 * Np + n) * 33 + l] = v.v;
          tile[(3 * Np + n) * 33 + l] = v.w;
        }
      }
      __syncthreads();
      for (int t = threadIdx.x; t < items; t += blockDim.x) {
        const int l = t / Np, n = t - l * Np, e = blk * kB + l;
        if (e < K) {
          const int64_t c = cmap[e] + n;
#pragma unroll
          for (int f = 0; f < 4; ++f) cw[f * T + c] = tile[(f * Np + n) * 33 + l];
        }
      }
    }
    __syncthreads();  // the tile is reused by the next block
  }
}

// ---------------------------------------------------------------------------
// discrete energy (Section 4.1), double accumulation, deterministic order
// ---------------------------------------------------------------------------
// One CTA per 32-element block (lane = element), warp f takes field f.
// Bound by the FP64 pipe (2 multiply-adds per cycle and SM), so the layout
// follows from the operation count: M^1D = C^T C turns the quadratic form of
// M^{tri,k} (x) M^1D into sum_j y_j^T M^{tri,k} y_j with y = (C (x) I) q, each
// of those a symmetric form on its lower triangle (Nt (Nt + 3) / 2 operations
// instead of the Nq Nt^2 of every slice pair), and the block forms the entries
// of M^{tri,k} once in shared memory for its four fields.  At N = 3: 1,605
// FP64 multiply-adds per wedge against 25,600 (each slice pair re-forming the
// mass entries in every thread).  FP32 state, 524,288 wedges, N = 3: 50.3 ms
// -> 2.0 ms (0.63 T multiply-adds/s of FP64 allow 1.3 ms); 128 wedges, FP64: 1.25 ms
// -> 22 us.
template <int N>
__host__ __device__ constexpr int energy_smem_bytes() {
  return nt_of(N) * (nt_of(N) + 1) / 2 * kB * 8;
}

template <int N>
__global__ void __launch_bounds__(128) k_energy(const DevMesh<real> M, const real* __restrict__ q) {
  constexpr int Nt = nt_of(N), Nq = N + 1, Npt = npt_of(N);
  const AllOps<N, real>& O = OPS<N>();
  extern __shared__ __align__(128) unsigned char smem_raw[];
  double* sM = reinterpret_cast<double*>(smem_raw);  // [Nt (Nt + 1) / 2][32]
  __shared__ double red[4];
  const int lane = threadIdx.x & 31, f = threadIdx.x >> 5;
  double E = 0.0;
  if (int(blockIdx.x) < M.nblk_w) {
    const int blk = blockIdx.x, e = blk * kB + lane;
    {
      // J_a = A h_a / 2 at the three columns, from the block's vertex table
      const real* X = M.w_xyz + int64_t(blk) * 12 * kB + lane;
      auto x = [&](int i) { return double(X[i * kB]); };
      const double A = 0.25 * ((x(1) - x(0)) * (x(5) - x(3)) - (x(2) - x(0)) * (x(4) - x(3)));
      const double J0 = 0.5 * A * (x(9) - x(6)), J1 = 0.5 * A * (x(10) - x(7)), J2 = 0.5 * A * (x(11) - x(8));
      // this warp's entries of the packed lower triangle (half the diagonal:
      // the form is twice its lower triangle)
#pragma unroll 1
      for (int at = f; at < Nt * (Nt + 1) / 2; at += 4)
        sM[at * kB + lane] = J0 * O.MaL[0][at] + J1 * O.MaL[1][at] + J2 * O.MaL[2][at];
    }
    __syncthreads();
    if (e < M.Kw) {
      const real* qf = q + widx<N>(blk, 0, lane) + f;
      if constexpr (N <= 3) {
        // all slices at once: a node value is converted to double once (a
        // conversion takes the FP64 pipe as long as a multiply-add)
        double y[Nq][Nt];
#pragma unroll
        for (int i = 0; i < Nt; ++i) {
#pragma unroll
          for (int j = 0; j < Nq; ++j) y[j][i] = 0.0;
#pragma unroll
          for (int m = 0; m < Nq; ++m) {
            const double v = double(qf[(m * Nt + i) * (kB * 4)]);
#pragma unroll
            for (int j = 0; j <= m; ++j) y[j][i] += O.M1C[j * Nq + m] * v;
          }
        }
#pragma unroll
        for (int i = 0; i < Nt; ++i) {
          double s[Nq];
#pragma unroll
          for (int j = 0; j < Nq; ++j) s[j] = 0.0;
#pragma unroll
          for (int l = 0; l <= i; ++l) {
            const double m = sM[(i * (i + 1) / 2 + l) * kB + lane];
#pragma unroll
            for (int j = 0; j < Nq; ++j) s[j] += m * y[j][l];
          }
#pragma unroll
          for (int j = 0; j < Nq; ++j) E += s[j] * y[j][i];
        }
      } else {
        // slice by slice: y of all slices would not fit the registers
#pragma unroll 1
        for (int j = 0; j < Nq; ++j) {
          double y[Nt];
#pragma unroll
          for (int i = 0; i < Nt; ++i) y[i] = 0.0;
#pragma unroll 1
          for (int m = j; m < Nq; ++m) {
            const double cj = O.M1C[j * Nq + m];
#pragma unroll
            for (int i = 0; i < Nt; ++i) y[i] += cj * double(qf[(m * Nt + i) * (kB * 4)]);
          }
          // (the mass entries are read again for every slice: held in registers
          // across the slices they would cost most of the warps in flight)
          asm volatile("" ::: "memory");
#pragma unroll
          for (int i = 0; i < Nt; ++i) {
            double s = 0.0;
#pragma unroll
            for (int l = 0; l <= i; ++l) s += sM[(i * (i + 1) / 2 + l) * kB + lane] * y[l];
            E += s * y[i];
          }
        }
      }
      E = 2.0 * E / double(M.w_mat[(f == 0 ? 0 : 1) * M.Kw_pad + e]);
    }
  } else {
    const int blk = int(blockIdx.x) - M.nblk_w, e = blk * kB + lane;
    if (e < M.Kt) {
      double X[4][3];
#pragma unroll
      for (int v = 0; v < 4; ++v)
#pragma unroll
        for (int d = 0; d < 3; ++d) X[v][d] = double(M.t_xyz[(int64_t(blk) * 12 + v * 3 + d) * kB + lane]);
      double G[3][3];
#pragma unroll
      for (int d = 0; d < 3; ++d)
#pragma unroll
        for (int m = 0; m < 3; ++m) G[d][m] = 0.5 * (X[m + 1][d] - X[0][d]);
      const double J = G[0][0] * (G[1][1] * G[2][2] - G[1][2] * G[2][1]) - G[0][1] * (G[1][0] * G[2][2] - G[1][2] * G[2][0]) +
                       G[0][2] * (G[1][0] * G[2][1] - G[1][1] * G[2][0]);
      // the constant reference mass on its lower triangle, four rows at a time
      const real* qf = q + tidx<N>(M.tet_off, blk, 0, lane) + f;
      double d = 0.0, o = 0.0;
#pragma unroll 1
      for (int i0 = 0; i0 < Npt; i0 += 4) {
        double s[4] = {0.0, 0.0, 0.0, 0.0}, y[4];
#pragma unroll
        for (int r = 0; r < 4; ++r) y[r] = i0 + r < Npt ? double(qf[(i0 + r) * (kB * 4)]) : 0.0;
        const real* m0 = M.tet_mass + i0 * Npt;
#pragma unroll 4
        for (int l = 0; l < i0; ++l) {
          const double ql = double(qf[l * (kB * 4)]);
#pragma unroll
          for (int r = 0; r < 4; ++r) s[r] += double(m0[(i0 + r < Npt ? r : 0) * Npt + l]) * ql;
        }
#pragma unroll
        for (int r = 0; r < 4; ++r) {
          if (i0 + r < Npt) {
#pragma unroll
            for (int c = 0; c < r; ++c) s[r] += double(m0[r * Npt + i0 + c]) * y[c];
            o += s[r] * y[r];
            d += double(m0[r * Npt + i0 + r]) * (y[r] * y[r]);
          }
        }
      }
      E = J * (d + 2.0 * o) / double(M.t_mat[(f == 0 ? 0 : 1) * M.Kt_pad + e]);
    }
  }
  // block reduction in a fixed order
#pragma unroll
  for (int s = 16; s > 0; s >>= 1) E += __shfl_down_sync(0xffffffffu, E, s);
  if (lane == 0) red[f] = E;
  __syncthreads();
  if (threadIdx.x == 0) M.partials[blockIdx.x] = 0.5 * ((red[0] + red[1]) + (red[2] + red[3]));
}

// the block sums in a fixed order: 1024 strided sums, then a tree
__global__ void __launch_bounds__(1024) k_energy_final(const double* __restrict__ partials, int n, double* out, int* err) {
  __shared__ double red[32];
  double s = 0.0;
  for (int i = threadIdx.x; i < n; i += 1024) s += partials[i];
#pragma unroll
  for (int d = 16; d > 0; d >>= 1) s += __shfl_down_sync(0xffffffffu, s, d);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = s;
  __syncthreads();
  if (threadIdx.x < 32) {
    s = red[threadIdx.x];
#pragma unroll
    for (int d = 16; d > 0; d >>= 1) s += __shfl_down_sync(0xffffffffu, s, d);
    if (threadIdx.x == 0) {
      *out = s;
      if (!isfinite(s)) atomicOr(err, kErrNonfinite);
    }
  }
}

}  // namespace REALNS
}  // namespace dgw

#include "adjoint_kernels.cuh"
#include "stage_split.cuh"

namespace dgw {
namespace REALNS {


// ---------------------------------------------------------------------------
// launchers
// ---------------------------------------------------------------------------
// one-time per device: opt in to the dynamic shared memory the stages use
template <int N, int OP>
cudaError_t prepare_op() {
  const cudaError_t err = cudaFuncSetAttribute(k_wedge_stage<N, 1, true, false, OP>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                               wedge_smem_bytes<N, 1, OP>());
  return err != cudaSuccess ? err
                            : cudaFuncSetAttribute(k_wedge_stage<N, 1, true, true, OP>,
                                                   cudaFuncAttributeMaxDynamicSharedMemorySize, wedge_smem_bytes<N, 1, OP>());
}
template <int N>
int prepare_n() {
  constexpr int b2 = wedge_bpc_multi<N>();
  cudaError_t err = cudaFuncSetAttribute(k_wedge_stage<N, 1, false, false>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         wedge_smem_bytes<N, 1>());
  if (err == cudaSuccess)
    err = cudaFuncSetAttribute(k_wedge_stage<N, 1, true, false>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                               wedge_smem_bytes<N, 1>());
  if (err == cudaSuccess)
    err = cudaFuncSetAttribute(k_wedge_stage<N, 1, true, true>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                               wedge_smem_bytes<N, 1>());
  if constexpr (sizeof(real) == 4) {
    if (err == cudaSuccess)
      err = cudaFuncSetAttribute(k_wedge_stage_split<N>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 split_smem_bytes<N>());
    if constexpr (nt_of(N) <= 16) {  // one 16-row tile holds a slice: tensor-core applies
      if (err == cudaSuccess) err = prepare_op<N, kOpTF32x3>();
      if (err == cudaSuccess) err = prepare_op<N, kOpTF32>();
      if (err == cudaSuccess) err = prepare_op<N, kOpBF16>();
    }
  }
  if constexpr (wide_fits<N>()) {
    if (err == cudaSuccess)
      err = cudaFuncSetAttribute(k_wedge_wide<N>, cudaFuncAttributeMaxDynamicSharedMemorySize, wide_smem_bytes<N>());
  }
  if constexpr (b2 != 1) {
    if (err == cudaSuccess)
      err = cudaFuncSetAttribute(k_wedge_stage<N, b2, true, false>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 wedge_smem_bytes<N, b2>());
    if (err == cudaSuccess)
      err = cudaFuncSetAttribute(k_wedge_stage<N, b2, true, true>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 wedge_smem_bytes<N, b2>());
  }
  if (err == cudaSuccess)
    err = cudaFuncSetAttribute(k_tet_stage<N>, cudaFuncAttributeMaxDynamicSharedMemorySize, tet_smem_bytes<N>());
  if (err == cudaSuccess)
    err = cudaFuncSetAttribute(k_pack<N>, cudaFuncAttributeMaxDynamicSharedMemorySize, pack_smem_bytes<N>());
  if (err == cudaSuccess)
    err = cudaFuncSetAttribute(k_energy<N>, cudaFuncAttributeMaxDynamicSharedMemorySize, energy_smem_bytes<N>());
  // the gradient kernels where their shared memory fits one CTA (not FP64 at N = 5,
  // whose adjoint the library refuses)
  if constexpr (grad_smem_bytes<N>() <= 227 * 1024) {
    if (err == cudaSuccess)
      err = cudaFuncSetAttribute(k_wedge_grad<N, false>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 grad_smem_bytes<N>());
    if (err == cudaSuccess)
      err = cudaFuncSetAttribute(k_wedge_grad<N, true>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 grad_smem_bytes<N>());
  }
  if (err == cudaSuccess)
    err = cudaFuncSetAttribute(k_tet_grad<N>, cudaFuncAttributeMaxDynamicSharedMemorySize, tgrad_smem_bytes<N>());
  return int(err);
}

// The small-mesh stage up to this many CTAs (blocks x slices): about one wave.
// us per stage of a step, small-mesh against large-mesh form, by blocks: FP32
// N = 3 1: 4.9 / 6.2, 32: 5.3 / 6.2, 64: 6.2 / 6.6; N = 2 64: 4.3 / 4.9, 128:
// 5.3 / 4.9; N = 4 32: 8.4 / 9.9, 64: 14 / 10; N = 5 4: 9 / 21, 32: 22 / 21;
// FP64 N = 3 1: 32 / 77, 64: 54 / 77, 128: 106 / 78; N = 4 32: 116 / 186.
template <int N>
constexpr int kWideCtas = N <= 3 ? 256 : 160;
constexpr int kPdlBlocks = kHalfSMs;
// Whether the wedge part of a stage takes the small-mesh form.  In FP32 at
// N >= 3 a stage that runs beside other kernels (beside) takes it only up to one
// CTA per SM: past that it gains little by itself, and its N + 1 times as many
// CTAs hold the SMs that the other kernels need.  us, up to kWideCtas / so: reverse
// stage N = 3, 64 blocks 11.3 / 9.7, N = 4, 32 blocks 18.1 / 14.2, 64 + 96 blocks N = 3
// 26.6 / 23.2; stage pair N = 4, 32 + 192 blocks 15.5 / 14.2, N = 3, 64 + 192 9.4 / 8.8.
template <int N>
bool small_mesh_form(int nblk_w, bool beside) {
  const int limit = sizeof(real) == 4 && N >= 3 && beside ? 2 * kHalfSMs : kWideCtas<N>;
  return wide_fits<N>() && nblk_w * (N + 1) <= limit;
}
// Launch attributes of a stage kernel.  dependent: a programmatic dependent of
// the kernel before it on the stream (inside a capture: a programmatic edge).
// carve: the part of an SM's memory to be shared memory, in per cent, or 0 for
// the default, which follows from the kernel's own shared memory and registers.
// Kernels of different carve-outs do not share an SM (its split between L1 and
// shared memory changes only while it is idle): left to the default, two that
// run on two streams queue behind each other on the SMs they meet on, so they
// are given the same.  The two element types' stages ask for all of it: us per
// stage pair of a step, default / all: 100 + 150 blocks FP64 N = 1 47.1 / 24.4,
// N = 2 115.5 / 58.8, N = 3 183.1 / 121.1; 64 + 48 blocks FP32 N = 3 10.1 / 7.8;
// 512 + 768 blocks FP32 N = 1 11.0 / 7.6, N = 3 21.0 / 20.8.  (Of 88 pairs one
// lost by it, whose CTAs happened to find SMs of their own: 64 + 48 blocks FP64
// N = 2 33.0 / 38.3.)
struct LaunchAttrs {
  cudaLaunchAttribute at[2];
  unsigned n = 0;
  LaunchAttrs(bool dependent, int carve) : at{} {
    if (dependent) {
      at[n].id = cudaLaunchAttributeProgrammaticStreamSerialization;
      at[n++].val.programmaticStreamSerializationAllowed = 1;
    }
    if (carve > 0) {
      at[n].id = cudaLaunchAttributePreferredSharedMemoryCarveout;
      at[n++].val.sharedMemCarveout = unsigned(carve);
    }
  }
};
constexpr int kCarveAll = cudaSharedmemCarveoutMaxShared;
// The carve-out of the reverse sweep's kernels, a stage beside its gradient
// kernel.  us per reverse stage, default / this: FP64 N = 2, 128 wedge blocks 149.2 /
// 54.2 and 108 tet blocks 65.2 / 39.6; FP32 N = 1, 512 wedge blocks 12.7 / 7.0.
// FP32 without tets, no more CTAs than SMs: room for one CTA of each, as the
// gradient kernel's gathers and spills live in the L1 that is left (N = 4, 72
// blocks default 18.3, all 18.1, this 15.3).  FP32 with tets: the default, where
// all costs more than it gives (N = 3, 108 tet blocks 9.4 / 11.0).  What lost: FP64
// N = 3, 200 wedge blocks 215 / 247.
template <int N>
int reverse_carve(const DevMesh<real>& m) {
  if (sizeof(real) == 8) return kCarveAll;
  if (m.nblk_t > 0) return 0;
  const bool small = small_mesh_form<N>(m.nblk_w, true);
  if ((small ? m.nblk_w * (N + 1) : m.nblk_w) > 2 * kHalfSMs) return kCarveAll;
  const int stage = small ? wide_smem_bytes<N>() : wedge_smem_bytes<N, 1>();
  const int bytes = stage + grad_smem_bytes<N>() + 2 * 1024, sm = 228 * 1024;  // (1 KB per CTA is the system's)
  return bytes < sm ? int((100ll * bytes + sm - 1) / sm) : kCarveAll;
}
template <typename... P>
cudaError_t launch_kernel(void (*kernel)(P...), int grid, int block, int smem, cudaStream_t s, LaunchAttrs attrs, P... args) {
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3(unsigned(grid));
  cfg.blockDim = dim3(unsigned(block));
  cfg.dynamicSmemBytes = size_t(smem);
  cfg.stream = s;
  cfg.attrs = attrs.at;
  cfg.numAttrs = attrs.n;
  cudaLaunchKernelEx(&cfg, kernel, args...);
  return cudaGetLastError();
}
template <typename... P>
cudaError_t launch_dependent(void (*kernel)(P...), int grid, int block, int smem, cudaStream_t s, bool pdl, int carve,
                             P... args) {
  return launch_kernel(kernel, grid, block, smem, s, LaunchAttrs(pdl, carve), args...);
}
template <int N, int OP>
cudaError_t launch_op(const StageArgs<real>& a, bool rk, cudaStream_t s, int carve) {
  auto kernel = a.m.w_fac == nullptr ? k_wedge_stage<N, 1, true, true, OP> : k_wedge_stage<N, 1, true, false, OP>;
  return launch_kernel(kernel, a.m.nblk_w, 32 * (N + 1), wedge_smem_bytes<N, 1, OP>(), s, LaunchAttrs(false, carve), a, rk);
}
template <int N>
int launch_stage_n(const StageArgs<real>& a, bool rk, cudaStream_t s, cudaStream_t st, cudaEvent_t ev_fork,
                   cudaEvent_t ev_join) {
  // wedges and tets of one stage are independent (each reads the stage input,
  // writes only its own elements): with a second stream the tet stage runs on
  // it, forked from and joined back into s (also inside a graph capture), so
  // the two kernels share the GPU instead of running back to back
  const bool fork = a.m.nblk_w > 0 && a.m.nblk_t > 0 && st != nullptr && ev_fork != nullptr && ev_join != nullptr;
  const int carve = fork ? kCarveAll : (a.reverse ? reverse_carve<N>(a.m) : 0);
  if (fork) {
    cudaError_t err = cudaEventRecord(ev_fork, s);
    if (err == cudaSuccess) err = cudaStreamWaitEvent(st, ev_fork, 0);
    if (err != cudaSuccess) return int(err);
    err = launch_kernel(k_tet_stage<N>, a.m.nblk_t, 128, tet_smem_bytes<N>(), st, LaunchAttrs(false, carve), a, rk);
    if (err == cudaSuccess) err = cudaEventRecord(ev_join, st);
    if (err != cudaSuccess) return int(err);
  }
  if (a.m.nblk_w > 0) {
    constexpr int b2 = wedge_bpc_multi<N>();
    const int want = a.wedge_bpc > 0 ? a.wedge_bpc : 1;
    bool done = false;
    if constexpr (sizeof(real) == 4) {
      // the field-pair split kernel (FP32 CUDA-core applies, stored mass
      // factor): when the autotuner or dg_set_launch_variant chose it
      const bool split = a.op == kOpFFMA && a.m.w_fac != nullptr && a.split > 0;
      if (split) {
        const cudaError_t err = launch_kernel(k_wedge_stage_split<N>, a.m.nblk_w, 64 * (N + 1), split_smem_bytes<N>(), s,
                                              LaunchAttrs(false, carve), a, rk);
        if (err != cudaSuccess) return int(err);
        done = true;
      }
    }
    if constexpr (sizeof(real) == 4 && nt_of(N) <= 16) {
      done = done || a.op != kOpFFMA;
      cudaError_t err = cudaSuccess;
      if (a.op == kOpTF32x3) err = launch_op<N, kOpTF32x3>(a, rk, s, carve);
      else if (a.op == kOpTF32) err = launch_op<N, kOpTF32>(a, rk, s, carve);
      else if (a.op == kOpBF16) err = launch_op<N, kOpBF16>(a, rk, s, carve);
      if (err != cudaSuccess) return int(err);
    }
    if constexpr (wide_fits<N>()) {
      if (!done && a.wedge_bpc <= 1 && small_mesh_form<N>(a.m.nblk_w, fork || a.reverse)) {
        const cudaError_t err = launch_dependent(k_wedge_wide<N>, a.m.nblk_w * (N + 1), 128, wide_smem_bytes<N>(), s,
                                                 a.pdl && a.m.nblk_t == 0, carve, a, rk);
        if (err != cudaSuccess) return int(err);
        done = true;
      }
    }
    if (!done) {
      // as a programmatic dependent only while both stages' CTAs find SMs of
      // their own (64 blocks, N = 3: 7.4 -> 6.6 us; 128 and 256 lose by it)
      const bool otf = a.m.w_fac == nullptr, pdl = a.pdl && a.m.nblk_t == 0 && a.m.nblk_w <= kPdlBlocks;
      StageArgs<real> b = a;
      b.pdl = pdl;
      cudaError_t err = cudaSuccess;
      if (want == 1 || b2 == 1) {
        auto kernel = otf ? k_wedge_stage<N, 1, true, true> : a.tri_far ? k_wedge_stage<N, 1, true, false> : k_wedge_stage<N, 1, false, false>;
        err = launch_dependent(kernel, a.m.nblk_w, 32 * (N + 1), wedge_smem_bytes<N, 1>(), s, pdl, carve, b, rk);
      } else {
        auto kernel = otf ? k_wedge_stage<N, b2, true, true> : k_wedge_stage<N, b2, true, false>;
        err = launch_dependent(kernel, (a.m.nblk_w + b2 - 1) / b2, 32 * (N + 1) * b2, wedge_smem_bytes<N, b2>(), s, pdl, carve, b,
                               rk);
      }
      if (err != cudaSuccess) return int(err);
    }
    cudaError_t err = cudaGetLastError();
    if (err != cudaSuccess) return int(err);
  }
  if (fork) return int(cudaStreamWaitEvent(s, ev_join, 0));
  if (a.m.nblk_t > 0)
    return int(launch_kernel(k_tet_stage<N>, a.m.nblk_t, 128, tet_smem_bytes<N>(), s, LaunchAttrs(false, carve), a, rk));
  return 0;
}

template <int N>
int launch_pack_n(const DevMesh<real>& m, const real* canon, real* packed, bool unpack, cudaStream_t s) {
  int blocks = m.nblk_w + m.nblk_t;
  if (blocks > 152 * 8) blocks = 152 * 8;
  if (blocks < 1) blocks = 1;
  k_pack<N><<<blocks, 256, pack_smem_bytes<N>(), s>>>(m, canon, packed, unpack);
  return int(cudaGetLastError());
}

template <int N>
int launch_energy_n(const DevMesh<real>& m, const real* q, cudaStream_t s) {
  const int grid = m.nblk_w + m.nblk_t;
  if (grid > 0) k_energy<N><<<grid, 128, energy_smem_bytes<N>(), s>>>(m, q);
  k_energy_final<<<1, 1024, 0, s>>>(m.partials, grid, m.energy, m.err);
  return int(cudaGetLastError());
}

}  // namespace REALNS
}  // namespace dgw

// extern launchers of this translation unit (order NORD, precision REAL)
#define DGW_CAT2(a, b) a##b
#define DGW_CAT(a, b) DGW_CAT2(a, b)
namespace dgw {
int DGW_CAT(upload_ops_, REALNS)(const void* host_ops, size_t bytes, void* stream) {
  if (bytes != sizeof(AllOps<NORD, REAL>)) return int(cudaErrorInvalidValue);
  const int rc = REALNS::prepare_n<NORD>();
  if (rc) return rc;
  return int(cudaMemcpyToSymbolAsync(REALNS::c_ops, host_ops, bytes, 0, cudaMemcpyHostToDevice, cudaStream_t(stream)));
}
int DGW_CAT(launch_stage_, REALNS)(const StageArgs<REAL>& a, bool rk, void* stream, void* stream_t, void* ev_fork,
                                   void* ev_join) {
  return REALNS::launch_stage_n<NORD>(a, rk, cudaStream_t(stream), cudaStream_t(stream_t), cudaEvent_t(ev_fork),
                                      cudaEvent_t(ev_join));
}
int DGW_CAT(launch_pack_, REALNS)(const DevMesh<REAL>& m, const REAL* canon, REAL* packed, bool unpack, void* stream) {
  return REALNS::launch_pack_n<NORD>(m, canon, packed, unpack, cudaStream_t(stream));
}
int DGW_CAT(launch_energy_, REALNS)(const DevMesh<REAL>& m, const REAL* q, void* stream) {
  return REALNS::launch_energy_n<NORD>(m, q, cudaStream_t(stream));
}
int DGW_CAT(launch_sample_, REALNS)(const DevMesh<REAL>& m, const REAL* q, REAL* out, int nshots, void* stream) {
  const int n = nshots * m.nrec;
  if (n > 0) REALNS::k_sample<NORD><<<(n + 3) / 4, 128, 0, cudaStream_t(stream)>>>(m, q, out, nshots);
  return int(cudaGetLastError());
}
int DGW_CAT(launch_inject_, REALNS)(const DevMesh<REAL>& m, REAL* muq, REAL* x, const REAL* resid, int nshots, REAL b5,
                                    void* stream) {
  const int n = nshots * m.nrgrp;
  if (n > 0) REALNS::k_inject<NORD><<<(n + 3) / 4, 128, 0, cudaStream_t(stream)>>>(m, muq, x, resid, nshots, b5);
  return int(cudaGetLastError());
}
int DGW_CAT(launch_grad_, REALNS)(const DevMesh<REAL>& m, const REAL* x, const REAL* q, const REAL* r, double dt,
                                  int flux, int bc, double* gk, double* gr, double* gz, void* stream) {
  if (m.nblk_w > 0) {
    constexpr int bytes = REALNS::grad_smem_bytes<NORD>();
    if (bytes > 227 * 1024) return int(cudaErrorInvalidConfiguration);
    constexpr int threads = 32 * (NORD + 1);
    const REALNS::LaunchAttrs attrs(false, REALNS::reverse_carve<NORD>(m));
    const cudaStream_t s = cudaStream_t(stream);
    if (m.nblk_t > 0)
      return int(REALNS::launch_kernel(REALNS::k_wedge_grad<NORD, true>, m.nblk_w, threads, bytes, s, attrs, m, x, q, r, dt, flux,
                                       bc, gk, gr, gz));
    return int(REALNS::launch_kernel(REALNS::k_wedge_grad<NORD, false>, m.nblk_w, threads, bytes, s, attrs, m, x, q, r, dt, flux,
                                     bc, gk, gr, gz));
  }
  return 0;
}
int DGW_CAT(launch_tgrad_, REALNS)(const DevMesh<REAL>& m, const REAL* x, const REAL* q, const REAL* r, double dt,
                                   int flux, int bc, double* gk, double* gr, void* stream) {
  if (m.nblk_t > 0) {
    constexpr int bytes = REALNS::tgrad_smem_bytes<NORD>();
    return int(REALNS::launch_kernel(REALNS::k_tet_grad<NORD>, m.nblk_t, 128, bytes, cudaStream_t(stream),
                                     REALNS::LaunchAttrs(false, REALNS::reverse_carve<NORD>(m)), m, x, q, r, dt, flux, bc, gk, gr));
  }
  return 0;
}
int DGW_CAT(launch_wait_expire_, REALNS)(int* err, void* stream) {
  REALNS::k_wait_expire<<<1, 32, 0, cudaStream_t(stream)>>>(err);
  return int(cudaGetLastError());
}
int DGW_CAT(launch_set_clock_, REALNS)(double* clock, double t, void* stream) {
  REALNS::k_set_clock<<<1, 32, 0, cudaStream_t(stream)>>>(clock, t);
  return int(cudaGetLastError());
}
int DGW_CAT(launch_clock_, REALNS)(const double* from, double* to, double dt, void* stream) {
  REALNS::k_clock<<<1, 32, 0, cudaStream_t(stream)>>>(from, to, dt);
  return int(cudaGetLastError());
}
}  // namespace dgw
