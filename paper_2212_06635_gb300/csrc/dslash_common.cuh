// Device helpers shared by the direct and the staged stencil kernels: spin
// projection / colour transport of one hop in the chiral basis, and the 6x6
// chirality-block products of the clover term and its inverses.
#pragma once

#include "tm_internal.h"

namespace tmk {

// ---------------------------------------------------------------------------
// Spin projection / reconstruction of the chiral basis for one hop.
//   S = -1: forward  (1 - g_mu) U_mu(x) psi(x+mu)
//   S = +1: backward (1 + g_mu) U_mu(x-mu)^dagger psi(x-mu)
// With g_mu = [[0, G],[G^+, 0]] (G_x = -i s1, G_y = -i s2, G_z = -i s3, G_t = -1):
//   (1 + S g) psi = (h, S G^+ h),  h = psi_up + S G psi_down,
// so only the two-spin half spinor h is transported by the link.
// ---------------------------------------------------------------------------
// -z where neg, by the sign bits
__device__ __forceinline__ cpx<double> flip_sign(cpx<double> z, bool neg) {
    const long long m = neg ? (long long)0x8000000000000000ull : 0ll;
    return C(__longlong_as_double(__double_as_longlong(z.re) ^ m), __longlong_as_double(__double_as_longlong(z.im) ^ m));
}
__device__ __forceinline__ cpx<float> flip_sign(cpx<float> z, bool neg) { return neg ? -z : z; }
// s a + b with one FMA per part
template <typename R>
__device__ __forceinline__ cpx<R> rfma(R s, cpx<R> a, cpx<R> b) { return C(fma(s, a.re, b.re), fma(s, a.im, b.im)); }

// half spinor h = psi_up + S G psi_down of one hop, times factor: the boundary
// phase of a time hop, times the neighbour's scale for 16-bit spinors (SCALED),
// which are passed unscaled; scaling the 6 projected components costs half of
// scaling the 12 loaded ones.
template <typename R, int MU, int S, bool SCALED, bool RAW = false>
__device__ __forceinline__ void hop_project(cpx<R> (&h0)[3], cpx<R> (&h1)[3], const cpx<R>* psi, R factor) {
    const R s = (R)S;
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        const cpx<R> p0 = psi[c], p1 = psi[3 + c], p2 = psi[6 + c], p3 = psi[9 + c];
        if (MU == 0) {        // h0 = p0 - s i p3, h1 = p1 - s i p2
            h0[c] = p0 - s * mul_i(p3);
            h1[c] = p1 - s * mul_i(p2);
        } else if (MU == 1) { // h0 = p0 - s p3, h1 = p1 + s p2
            h0[c] = p0 - s * p3;
            h1[c] = p1 + s * p2;
        } else if (MU == 2) { // h0 = p0 - s i p2, h1 = p1 + s i p3
            h0[c] = p0 - s * mul_i(p2);
            h1[c] = p1 + s * mul_i(p3);
        } else {              // h0 = p0 - s p2, h1 = p1 - s p3
            h0[c] = p0 - s * p2;
            h1[c] = p1 - s * p3;
        }
        if (RAW) continue;   // the caller applies the factor
        if (SCALED || (MU == 3 && sizeof(R) == 4)) {
            h0[c] = factor * h0[c];
            h1[c] = factor * h1[c];
        } else if (MU == 3) {
            // FP64: the phase is +-1, and a sign flip takes no FP64 instruction
            h0[c] = flip_sign(h0[c], factor < (R)0);
            h1[c] = flip_sign(h1[c], factor < (R)0);
        }
    }
}

// g += U h (DAG: U^dagger h) for both spins of a half spinor
template <typename R, bool DAG>
__device__ __forceinline__ void hop_transport(cpx<R> (&g0)[3], cpx<R> (&g1)[3], const cpx<R> (&u)[9],
                                              const cpx<R> (&h0)[3], const cpx<R> (&h1)[3]) {
#pragma unroll
    for (int a = 0; a < 3; ++a)
#pragma unroll
        for (int b = 0; b < 3; ++b) {
            if (DAG) {
                cfma_cj(g0[a], u[3 * b + a], h0[b]);
                cfma_cj(g1[a], u[3 * b + a], h1[b]);
            } else {
                cfma(g0[a], u[3 * a + b], h0[b]);
                cfma(g1[a], u[3 * a + b], h1[b]);
            }
        }
}

// (x0, x1) = G_mu^+ (g0, g1), the lower spins that a backward hop adds and a forward hop subtracts
template <typename R, int MU>
__device__ __forceinline__ void hop_lower(cpx<R>& x0, cpx<R>& x1, cpx<R> g0, cpx<R> g1) {
    if (MU == 0) { x0 = mul_i(g1); x1 = mul_i(g0); }
    else if (MU == 1) { x0 = g1; x1 = -g0; }
    else if (MU == 2) { x0 = mul_i(g0); x1 = -mul_i(g1); }
    else { x0 = -g0; x1 = -g1; }
}

// One hop added to acc; FIRST: acc is overwritten.  FOLD: a 16-bit spinor's factor
// (SCALED) rides in the FMAs that accumulate instead of multiplying the half spinor
// (12 multiplications fewer).  That takes registers: it pays in the two-flavour
// passes (24^3x48, odd: FP16 61.4 -> 59.5 us, BF16 60.8 -> 59.3 us) and not in the
// light ones (32^3x64, odd, FP16: 101.4 -> 103.8 us).
template <typename R, int MU, int S, bool DAG, bool SCALED = false, bool FIRST = false, bool FOLD = false>
__device__ __forceinline__ void hop_dir(cpx<R> (&acc)[4][3], const cpx<R>* psi,
                                        const cpx<R> (&u)[9], R factor) {
    constexpr bool F = SCALED && FOLD;
    const R s = (R)S;
    cpx<R> h0[3], h1[3], g0[3], g1[3];
    hop_project<R, MU, S, SCALED, F>(h0, h1, psi, factor);
#pragma unroll
    for (int a = 0; a < 3; ++a) g0[a] = g1[a] = C((R)0, (R)0);
    hop_transport<R, DAG>(g0, g1, u, h0, h1);
    const R up = F ? factor : (R)1, dn = F ? s * factor : s;
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        cpx<R> x0, x1;
        hop_lower<R, MU>(x0, x1, g0[a], g1[a]);
        if (FIRST) {
            acc[0][a] = F ? up * g0[a] : g0[a];
            acc[1][a] = F ? up * g1[a] : g1[a];
            acc[2][a] = dn * x0;
            acc[3][a] = dn * x1;
        } else if (F) {
            acc[0][a] = rfma(up, g0[a], acc[0][a]);
            acc[1][a] = rfma(up, g1[a], acc[1][a]);
            acc[2][a] = rfma(dn, x0, acc[2][a]);
            acc[3][a] = rfma(dn, x1, acc[3][a]);
        } else {
            acc[0][a] = acc[0][a] + g0[a];
            acc[1][a] = acc[1][a] + g1[a];
            acc[2][a] = acc[2][a] + dn * x0;
            acc[3][a] = acc[3][a] + dn * x1;
        }
    }
}

// (The two hops of a direction as a pair, the backward transport continuing the forward
// sums to t = gf + gb with t for the upper spins and t - 2 gf for the lower ones, take a
// quarter fewer additions: light FP64 operator at 16^3x32 560 instead of 590 us, at
// 24^3x48 2608 instead of 2748 us.  But t - 2 gf rounds a sum larger than gb - gf, which
// makes the lower spins' error 12 % larger than the upper ones' in FP64, and an infinite
// gf makes NaN of them.  Not used.)

// w = B v (CONJ: B^dagger v) for a full complex 6x6 block stored row major.
template <typename R, bool CONJ>
__device__ __forceinline__ void full6_mv(cpx<R> (&w)[6], const R* m, const cpx<R> (&v)[6]) {
#pragma unroll
    for (int r = 0; r < 6; ++r) w[r] = C((R)0, (R)0);
#pragma unroll
    for (int r = 0; r < 6; ++r)
#pragma unroll
        for (int j = 0; j < 6; ++j) {
            const cpx<R> e = C(m[2 * (6 * r + j)], m[2 * (6 * r + j) + 1]);
            if (CONJ) cfma_cj(w[j], e, v[r]);   // (B^+)_{j r} = conj(B_{r j})
            else cfma(w[r], e, v[j]);
        }
}

// w += H v for a packed hermitian 6x6 block (36 reals).
template <typename R>
__device__ __forceinline__ void herm6_mv_acc(cpx<R> (&w)[6], const R* m, const cpx<R> (&v)[6]) {
#pragma unroll
    for (int r = 0; r < 6; ++r) w[r] = w[r] + m[r] * v[r];
#pragma unroll
    for (int r = 1; r < 6; ++r)
#pragma unroll
        for (int j = 0; j < r; ++j) {
            const cpx<R> e = C(m[herm_off(r, j)], m[herm_off(r, j) + 1]);
            cfma(w[r], e, v[j]);      // lower:  H_rj v_j
            cfma_cj(w[j], e, v[r]);   // upper:  H_jr = conj(H_rj)
        }
}

// out = r - alpha (out + shift p) with the residual and search direction of site i, a
// vector of reals at a time: the update of CG without a stored A p (alpha is known
// before the second factor of the operator is applied).  NR reals from `off` of a site's
// 2 NC.
template <int P, int NC, int NR = 2 * NC>
__device__ __forceinline__ void residual_update(cpx<typename PT<P>::R>* out, const OpProb& pr, long i, int off = 0) {
    using R = typename PT<P>::R;
    constexpr int W = PT<P>::W;
    const long vh = pr.g.vh;
    const R alpha = (R)pr.ctl->alpha, shift = (R)pr.ctl->shift;
    R* o = reinterpret_cast<R*>(out);
    R rs = (R)1, ps = (R)1;
    if constexpr (P == PB16 || P == PF16) {
        const size_t scale = (size_t)vh * NC * 4;
        rs = reinterpret_cast<const float*>(reinterpret_cast<const char*>(pr.r) + scale)[i];
        ps = reinterpret_cast<const float*>(reinterpret_cast<const char*>(pr.p) + scale)[i];
    }
#pragma unroll
    for (int v = 0; v < NR / W; ++v) {
        if (shift != (R)0) {
            R p[W];
            load_reals<P, W>(pr.p, vh, i, off + W * v, p);
#pragma unroll
            for (int e = 0; e < W; ++e) o[W * v + e] += shift * (ps * p[e]);
        }
        R r[W];
        load_reals<P, W>(pr.r, vh, i, off + W * v, r);
#pragma unroll
        for (int e = 0; e < W; ++e) o[W * v + e] = rs * r[e] - alpha * o[W * v + e];
    }
}

}  // namespace tmk
