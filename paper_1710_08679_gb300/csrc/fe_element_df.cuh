// Element product in float-float arithmetic (the FP64-accurate products of the
// outer loop, computed on the FP32 pipe), the formulas of elem_apply with the
// sums of products accumulated in compensated form.
//
// A sum of products sum_i a_i b_i of float-float numbers is accumulated as in
// the compensated dot product of Ogita, Rump and Oishi ("Accurate sum and dot
// product", SIAM J. Sci. Comput. 26, 2005): the running sum of the high parts'
// products is kept with its exact rounding errors (TwoProd, TwoSum), and these are
// gathered in one float together with the cross terms hi*lo and lo*hi of each
// product. The result is as accurate as evaluating in float-float throughout, with
// about 11 FP32 operations per term instead of 18 for a float-float multiply and
// add. Multiplications by 4, 2 and 1/4 scale both parts exactly.
#pragma once

#include "fe_df.cuh"
#include "fe_element.cuh"

namespace fe {

// ---------------------------------------------------------------------------
// The product in paired FP32 instructions (ebe_pipe_df_kernel, ebe_pipe_df_lean_kernel). The two
// lanes of every pair are two corners of one element and case: (0, 1) and (2, 3), so the
// corner gradients, the corner stresses and the corner outputs of both come from one
// instruction stream, and the edge outputs
//   y_kl = T_k g_l + T_l g_k
// combine lanes of the two pairs: (02, 13) lane by lane, (03, 12) crosswise, (01) and
// (23) as sums over the lanes of one pair. The register state is that of one case (a
// pair of cases per thread would double it), and the code is half as long: the scalar
// form (5,300 instructions per case) stalled on instruction fetch as often as on
// dependencies. With v_mj = 4 u_mj - u_j and u_mm = u_m (so that v_mm = 3 u_m), every
// corner has the same formula.
//
// A multiply-add term of a compensated sum (pacc_add) takes 10 operations instead of 12: of
// the rounded product p added to s, bb = s' - s reached the new sum s'; the rest of the exact
// product, a b - bb, is one FMA (TwoProd and the second half of TwoSum at once),
// s - (s' - bb) completes the error, and the cross terms are added to it. (Adding the product by
// an FMA, s' = fl(s + a b), would save one more but count part of it twice where s' cancels.)
// That FMA rounds a remainder as large as the sum's own error. Where the sums cancel, which is
// in the gradients sum_j v_mj g_j of displacements that are mostly translation, as a solve's
// are, pacc_add_exact forms both errors without rounding (12 operations), and v_mm = 3 u_m gets
// the one rounding of a product (p4add). Subtractions are FMAs with a factor of -1: paired
// instructions have no negated operands. `pnorm` renormalises where a value becomes an
// operand or a sum goes on.
//
// Mean error of an element product against long double, relative to the scalar form's
// (TwoProd and TwoSum apart, 12 operations a term): random vectors -0.6 %, linear fields
// -2.8 %, translation and a linear field 0.0 %, slip solutions -0.4 %; whole products on
// random vectors 3.1e-15 against 64-bit torch. With pacc_add in the gradients too and 3 u_m
// as 4 u_m - u_m the product takes 1 % less time, and the error of translated fields grows
// by 8 %.
//
// Bound by the FP32 pipe, on which a paired instruction takes two cycles, and by the
// latencies that four warps per scheduler leave uncovered (ncu: FMA pipe 53 %, issue 50 %;
// the scalar form issued half as many instructions again at 65 %). R = 16 on the 41x33x18
// crust block: 750 -> 657 us, R = 4: 283 -> 227 us; R = 16 on the 70x70x35 block: 5.25 -> 4.50 ms.
//
// The element's data: for i = 0, 1, 2 the float4 (g0_i.hi, g1_i.hi, g0_i.lo, g1_i.lo) and
// the same of g2, g3, then (lam'.hi, lam'.lo, mu'.hi, mu'.lo) and (0, 0, 2^e, 0): V/5 =
// f 2^e with 1 <= f < 2, lam' = lam f, mu' = mu f, and the outputs' gradients take the 2^e
// (so that the stresses stay in the range of the moduli; kGeo float-float values in all).
// ---------------------------------------------------------------------------
#ifdef __CUDA_ARCH__
__device__ __forceinline__ float2 q_fma(float2 a, float2 b, float2 c) { return __ffma2_rn(a, b, c); }
__device__ __forceinline__ float2 q_mul(float2 a, float2 b) { return __fmul2_rn(a, b); }
__device__ __forceinline__ float2 q_add(float2 a, float2 b) { return __fadd2_rn(a, b); }
#else   // the same operations on the host, for checks of the arithmetic without a GPU
inline float2 q_fma(float2 a, float2 b, float2 c) { return make_float2(fmaf(a.x, b.x, c.x), fmaf(a.y, b.y, c.y)); }
inline float2 q_mul(float2 a, float2 b) { return make_float2(a.x * b.x, a.y * b.y); }
inline float2 q_add(float2 a, float2 b) { return make_float2(a.x + b.x, a.y + b.y); }
#endif

#define FE_HD __host__ __device__ __forceinline__

FE_HD float2 q_bc(float a) { return make_float2(a, a); }
FE_HD float2 q_sub(float2 a, float2 b) { return q_fma(b, q_bc(-1.f), a); }

// two float-float values (lanes x and y): s + c, c not normalised against s
struct dfp {
  float2 s, c;
};

FE_HD dfp p_pack(const df& a, const df& b) { return {make_float2(a.hi, b.hi), make_float2(a.lo, b.lo)}; }

FE_HD dfp pnorm(const dfp& a) {
  const float2 s = q_add(a.s, a.c);
  return {s, q_add(q_sub(a.s, s), a.c)};
}

// A = a b. z is zero, in a form the compiler cannot see through: it contracts a paired
// multiplication into an addition that follows (whatever the rounding suffix), and the
// error terms here and in padd hold for the rounded product only; an FMA with addend z is
// that product and stays one.
FE_HD void pacc_first(dfp& A, const dfp& a, const dfp& b, float2 z) {
  A.s = q_fma(a.s, b.s, z);
  A.c = q_fma(a.s, b.c, q_fma(a.c, b.s, q_fma(a.s, b.s, q_mul(A.s, q_bc(-1.f)))));
}

// A += a b
FE_HD void pacc_add(dfp& A, const dfp& a, const dfp& b, float2 z) {
  const float2 s = q_add(A.s, q_fma(a.s, b.s, z));
  const float2 nbb = q_sub(A.s, s);                    // -(what a b added to A.s)
  const float2 r = q_sub(A.s, q_add(s, nbb));
  const float2 e = q_add(r, q_fma(a.s, b.s, nbb));     // fl(A.s + p) missed this much of A.s + a b
  A.s = s;
  A.c = q_add(A.c, q_fma(a.s, b.c, q_fma(a.c, b.s, e)));
}

// A += a b for sums that cancel (v_mj g_j of a displacement that is nearly a translation),
// nb = -b.s: the product's and the sum's rounding errors each formed exactly
FE_HD void pacc_add_exact(dfp& A, const dfp& a, const dfp& b, float2 nb, float2 z) {
  const float2 np = q_fma(a.s, nb, z);                 // -p
  const float2 s = q_sub(A.s, np);
  const float2 nbb = q_sub(A.s, s);
  const float2 r = q_sub(A.s, q_add(s, nbb));
  const float2 e = q_add(r, q_sub(nbb, np));           // A.s + p - s
  A.c = q_add(A.c, q_add(e, q_fma(a.s, b.c, q_fma(a.c, b.s, q_fma(a.s, b.s, np)))));
  A.s = s;
}

FE_HD dfp padd(const dfp& a, const dfp& b) {
  const float2 s = q_add(a.s, b.s);
  const float2 nbb = q_sub(a.s, s);
  const float2 e = q_add(q_sub(a.s, q_add(s, nbb)), q_add(b.s, nbb));
  return {s, q_add(e, q_add(a.c, b.c))};
}

// 4 a + b. In lane M (0: x, 1: y, -1: none) b = -a: there the low part 3 a.c + e (e: what
// the sum of the high parts missed) has one rounding, as the product 3 a has.
template <int M>
FE_HD dfp p4add(const dfp& a, const dfp& b) {
  const float2 s = q_fma(a.s, q_bc(4.f), b.s);
  const float2 bb = q_fma(a.s, q_bc(-4.f), s);
  const float2 r = q_fma(a.s, q_bc(4.f), q_sub(bb, s));
  const float2 e = q_add(r, q_sub(b.s, bb));
  const float2 k = make_float2(M == 0 ? 3.f : 4.f, M == 1 ? 3.f : 4.f);
  const float2 t = q_fma(a.c, k, make_float2(M == 0 ? e.x : b.c.x, M == 1 ? e.y : b.c.y));
  return {s, q_add(t, make_float2(M == 0 ? 0.f : e.x, M == 1 ? 0.f : e.y))};
}

FE_HD dfp pscale(const dfp& a, float k) { return {q_mul(a.s, q_bc(k)), q_mul(a.c, q_bc(k))}; }

// g of corner j as a pair of equal lanes, from the element's data
template <int J>
FE_HD dfp geo_both(const float4* gs, int i) {
  const float4 w = gs[2 * i + J / 2];
  return J % 2 == 0 ? dfp{q_bc(w.x), q_bc(w.z)} : dfp{q_bc(w.y), q_bc(w.w)};
}

template <int P, int J>
FE_HD void pair_gradient_term(const float4* gs, const df* xa, const int* off, float2 z, dfp A[3][3]) {
  constexpr int e0 = edge_or_corner(2 * P, J), e1 = edge_or_corner(2 * P + 1, J);
  constexpr int own = J == 2 * P ? 0 : J == 2 * P + 1 ? 1 : -1;   // the lane with 3 u_m
  dfp v[3];
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    const df uj = xa[off[J] + a];
    v[a] = pnorm(p4add<own>(p_pack(xa[off[e0] + a], xa[off[e1] + a]), {q_bc(-uj.hi), q_bc(-uj.lo)}));
  }
#pragma unroll
  for (int b = 0; b < 3; ++b) {
    const dfp g = geo_both<J>(gs, b);
    const float2 ng = q_bc(-g.s.x);
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      if (J == 0)
        pacc_first(A[a][b], v[a], g, z);
      else
        pacc_add_exact(A[a][b], v[a], g, ng, z);
    }
  }
}

// s_m = lam' tr(H_m) I + mu' (H_m + H_m^T) (times 2^e) of corners m = 2P, 2P + 1 (lanes x, y)
template <int P>
FE_HD void pair_stress(const float4* gs, const df* xa, const int* off, float2 z, dfp s[6]) {
  dfp H[3][3];
  pair_gradient_term<P, 0>(gs, xa, off, z, H);
  pair_gradient_term<P, 1>(gs, xa, off, z, H);
  pair_gradient_term<P, 2>(gs, xa, off, z, H);
  pair_gradient_term<P, 3>(gs, xa, off, z, H);
  const float4 w = gs[6];
  const dfp lam = {q_bc(w.x), q_bc(w.y)}, mu = {q_bc(w.z), q_bc(w.w)};
  const dfp two_mu = {q_bc(2.f * w.z), q_bc(2.f * w.w)};
#pragma unroll
  for (int a = 0; a < 3; ++a)
#pragma unroll
    for (int b = 0; b < 3; ++b) H[a][b] = pnorm(H[a][b]);
  dfp lt;
  pacc_first(lt, pnorm(padd(padd(H[0][0], H[1][1]), H[2][2])), lam, z);
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    s[a] = lt;
    pacc_add(s[a], H[a][a], two_mu, z);
    s[a] = pnorm(s[a]);
  }
  pacc_first(s[3], pnorm(padd(H[1][2], H[2][1])), mu, z);
  pacc_first(s[4], pnorm(padd(H[0][2], H[2][0])), mu, z);
  pacc_first(s[5], pnorm(padd(H[0][1], H[1][0])), mu, z);
#pragma unroll
  for (int q = 3; q < 6; ++q) s[q] = pnorm(s[q]);
}

// row c of the symmetric matrix stored (xx, yy, zz, yz, xz, xy)
FE_HD constexpr int sym_at(int c, int b) { return c == b ? c : 6 - c - b; }

// w = (T g)_c
FE_HD dfp row_first(const dfp T[6], int c, const dfp g[3], float2 z) {
  dfp w;
  pacc_first(w, T[sym_at(c, 0)], g[0], z);
  pacc_add(w, T[sym_at(c, 1)], g[1], z);
  pacc_add(w, T[sym_at(c, 2)], g[2], z);
  return w;
}

FE_HD dfp p_swap(const dfp& a) { return {make_float2(a.s.y, a.s.x), make_float2(a.c.y, a.c.x)}; }

FE_HD void store_pair(const dfp& w, df* ox, df* oy) {
  const dfp n = pnorm(w);
  *ox = df(n.s.x, n.c.x);
  *oy = df(n.s.y, n.c.y);
}

// y = K_e u: node values (node a, component c) read at xa[off[a] + c] where they are
// used, outputs stored to o[a VR + c] as they are formed
template <int VR>
FE_HD void elem_apply_df_pair(const float4* gs, const df* xa, const int* off, df* o) {
  dfp s[2][6];   // s[P]: corners 2P (lane x) and 2P + 1 (lane y)
  const float2 z = {gs[7].x, gs[7].y};
  pair_stress<0>(gs, xa, off, z, s[0]);
  pair_stress<1>(gs, xa, off, z, s[1]);
  dfp S[6];      // sum over the four corners, in both lanes
#pragma unroll
  for (int q = 0; q < 6; ++q) {
    const dfp t = pnorm(padd(s[0][q], s[1][q]));
    S[q] = pnorm(padd(t, p_swap(t)));
  }
  dfp g01[3], g23[3];
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    const float4 a = gs[2 * i], b = gs[2 * i + 1];
    g01[i] = pscale({make_float2(a.x, a.y), make_float2(a.z, a.w)}, gs[7].z);
    g23[i] = pscale({make_float2(b.x, b.y), make_float2(b.z, b.w)}, gs[7].z);
  }
  // corners: y_k = (s_k - S/4) g_k
#pragma unroll
  for (int P = 0; P < 2; ++P) {
    dfp A[6];
#pragma unroll
    for (int q = 0; q < 6; ++q) A[q] = pnorm(padd(s[P][q], pscale(S[q], -0.25f)));
#pragma unroll
    for (int c = 0; c < 3; ++c)
      store_pair(row_first(A, c, P == 0 ? g01 : g23, z), o + (2 * P) * VR + c, o + (2 * P + 1) * VR + c);
  }
  // edges, T_k = s_k + S
#pragma unroll
  for (int P = 0; P < 2; ++P)
#pragma unroll
    for (int q = 0; q < 6; ++q) s[P][q] = pnorm(padd(s[P][q], S[q]));
#pragma unroll
  for (int c = 0; c < 3; ++c) {   // (0,2) and (1,3): T01 (g2, g3) + T23 (g0, g1)
    dfp w = row_first(s[0], c, g23, z);
#pragma unroll
    for (int b = 0; b < 3; ++b) pacc_add(w, s[1][sym_at(c, b)], g01[b], z);
    store_pair(w, o + 6 * VR + c, o + 8 * VR + c);
  }
  dfp g10[3], g32[3];
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    g10[i] = p_swap(g01[i]);
    g32[i] = p_swap(g23[i]);
  }
#pragma unroll
  for (int c = 0; c < 3; ++c)     // (0,3) and (1,2): T01 (g3, g2) + swapped T23 (g1, g0)
    store_pair(padd(row_first(s[0], c, g32, z), p_swap(row_first(s[1], c, g10, z))), o + 7 * VR + c, o + 5 * VR + c);
#pragma unroll
  for (int c = 0; c < 3; ++c) {   // (0,1) and (2,3): the two lanes of T01 (g1, g0) and of T23 (g3, g2)
    const dfp a = row_first(s[0], c, g10, z), b = row_first(s[1], c, g32, z);
    const dfp x = {make_float2(a.s.x, b.s.x), make_float2(a.c.x, b.c.x)};
    const dfp y = {make_float2(a.s.y, b.s.y), make_float2(a.c.y, b.c.y)};
    store_pair(padd(x, y), o + 4 * VR + c, o + 9 * VR + c);
  }
}

#undef FE_HD

}  // namespace fe
