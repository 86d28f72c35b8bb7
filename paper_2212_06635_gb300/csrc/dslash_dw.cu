// Double-word form of the stencil passes of eq:hQpm (light) and eq:hQh (heavy
// doublet), for the true-residual recomputations of the mixed-precision solvers
// (tm_apply_Mhat_dw).
//
//   K1 (even output):  t_e = M_ee^-1 H_eo psi_o
//   K2 (odd output):   out = g5 [ M_oo psi_o - kappa^2 H_oe t_e ] (+ i rho psi_o)
//
// The heavy passes split the flavours over a thread pair (thread 2 i + f: flavour
// f of site i), as the direct FP32 / 16-bit heavy even pass does, so a thread
// holds one flavour's accumulators; the even inverse takes the partner's D v by
// lane shuffles, the odd pass reads the partner flavour of psi_o directly.
//
// Values are double words (df64.h), held as (hi, lo) FP32 pairs in the FP64
// layouts.  The passes are bound by FP32 issue (17,100-18,700 instructions per
// site, 73-77 % of the issue slots busy), so the code
// - forms every sum of products as a compensated dot product (Ogita, Rump and
//   Oishi, "Accurate sum and dot product", SIAM J. Sci. Comput. 26 (2005), Dot2):
//   the high parts are summed with two_sum, the product errors (two_prod with one
//   FMA), the cross terms and the summation errors go to a second FP32 sum, and
//   the pair is renormalised only where it enters a product;
// - runs the hops, and the rows of the site-local blocks, as loops over one copy of
//   their code, the direction and the row selected at run time: unrolled, the
//   passes (21,000 instructions a site) stall on instruction fetch, and already the
//   blocks' unrolled rows alone cost the odd pass 2.7 warps per issue;
// - copies each hop's spinor and link, and the blocks, into the thread's own
//   shared-memory slots with cp.async while the hop before is computed (a slot is
//   refilled as soon as its words are used): 4 resident blocks are too few warps to
//   hide the loads.
// M_hat^dagger M_hat at 24^3x48 with its conversions 1232 -> 912 us, the heavy
// operator 3022 -> 2264 us against loads at the point of use, rows unrolled, at the
// same errors (8.0e-15 / 8.5e-15).  Pairing the two hops of a direction (dslash_common.cuh;
// 36 compensated additions instead of 48) gives 8.1e-15 and is not used.
// The operator's last pass stores FP64 itself: its conversions (2 per cycle and SM) hide
// behind the FP32 work, as a kernel of their own they took 43 us (light, 905 -> 865 us).
#include "tm_internal.h"
#include "tm_kernels.h"
#include "dslash_common.cuh"

namespace tmk {

// compensated sum: h the running FP32 sum, l the FP32 sum of its errors and of
// the low parts added
struct CSum {
    float h, l;
};
// a += f (xh + xl), f a power of two with sign (f x is exact, so it rides in the FMAs)
__device__ __forceinline__ void cs_add(CSum& a, float xh, float xl, float f = 1.f) {
    const float s = __fmaf_rn(f, xh, a.h);
    const float bb = __fsub_rn(s, a.h);
    const float t = __fadd_rn(__fsub_rn(a.h, __fsub_rn(s, bb)), __fmaf_rn(f, xh, -bb));
    a.h = s;
    a.l = __fadd_rn(a.l, __fmaf_rn(f, xl, t));
}
__device__ __forceinline__ void cs_add(CSum& a, df x, float f = 1.f) { cs_add(a, x.h, x.l, f); }
__device__ __forceinline__ void cs_add(CSum& a, CSum x, float f = 1.f) { cs_add(a, x.h, x.l, f); }
// a += x y (the low-low product, below 2^-48 |x y|, is dropped); cs_fms: a -= x y
__device__ __forceinline__ void cs_fma(CSum& a, df x, df y) {
    const float p = __fmul_rn(x.h, y.h);
    float e = __fmaf_rn(x.h, y.h, -p);
    e = __fmaf_rn(x.h, y.l, e);
    e = __fmaf_rn(x.l, y.h, e);
    cs_add(a, p, e);
}
__device__ __forceinline__ void cs_fms(CSum& a, df x, df y) { cs_fma(a, df(-x.h, -x.l), y); }
__device__ __forceinline__ df cs_get(CSum a) { return df_fast_two_sum(a.h, a.l); }
__device__ __forceinline__ CSum cs_zero() { return CSum{0.f, 0.f}; }

struct CC {   // complex of compensated sums
    CSum re, im;
};
// a += z w, and a += conj(z) w
__device__ __forceinline__ void cc_fma(CC& a, cpx<df> z, cpx<df> w) {
    cs_fma(a.re, z.re, w.re);
    cs_fms(a.re, z.im, w.im);
    cs_fma(a.im, z.re, w.im);
    cs_fma(a.im, z.im, w.re);
}
__device__ __forceinline__ cpx<df> cc_get(CC a) { return C(cs_get(a.re), cs_get(a.im)); }
__device__ __forceinline__ CC cc_zero() { return CC{cs_zero(), cs_zero()}; }

// x + f y, f = +-1, as a double word
__device__ __forceinline__ df df_add(df x, df y, float f) {
    const float s = __fmaf_rn(f, y.h, x.h);
    const float bb = __fsub_rn(s, x.h);
    const float t = __fadd_rn(__fsub_rn(x.h, __fsub_rn(s, bb)), __fmaf_rn(f, y.h, -bb));
    return df_fast_two_sum(s, __fadd_rn(t, __fmaf_rn(f, y.l, x.l)));
}
// ---------------------------------------------------------------------------
// the thread's shared-memory slots: DW_SLOTS vectors (a double-word complex each)
// ---------------------------------------------------------------------------
constexpr int DW_SLOTS = 24;   // spinor of one flavour 12, link 9; the epilogue uses all 24
constexpr int DW_SMEM = DW_SLOTS * DSLASH_BS * 16;

__device__ __forceinline__ void dw_copy(float4* slot, const float4* src) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 16;" ::"r"((unsigned)__cvta_generic_to_shared(slot)), "l"(src)
                 : "memory");
}
__device__ __forceinline__ void dw_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void dw_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory"); }
__device__ __forceinline__ cpx<df> dw_read(const float4* slot) {
    const float4 q = *slot;
    return C(df(q.x, q.y), df(q.z, q.w));
}

__device__ __forceinline__ void dw_write(float4* slot, cpx<df> z) { *slot = make_float4(z.re.h, z.re.l, z.im.h, z.im.l); }

// n vectors from v0 of site i of a double-word array into slots s0 ..
template <int N>
__device__ __forceinline__ void dw_fetch(float4* slots, int s0, const void* base, long vh, int v0, long i) {
    const float4* p = reinterpret_cast<const float4*>(base) + (long)v0 * vh + i;
#pragma unroll
    for (int k = 0; k < N; ++k) dw_copy(slots + (s0 + k) * DSLASH_BS, p + (long)k * vh);
}

// The hops' spin structure (h = psi_up + s G psi_down, lower += s G^+ g;
// dslash_common.cuh) with the direction selected at run time, so that the loop
// over hops holds one copy of it:
//   h0 = p0 + c0 i^k pA, h1 = p1 + c1 i^k pB, k = 1 for mu = 0, 2,
//   (pA, pB) = (p3, p2) for mu = 0, 1 and (p2, p3) for mu = 2, 3,
//   c0 = -s, c1 = s (-, +, +, -);
//   acc2 += d2 i^k x2, acc3 += d3 i^k x3, (x2, x3) = (g1, g0) for mu = 0, 1 and
//   (g0, g1) for mu = 2, 3, d2 = s (+, +, +, -), d3 = s (+, -, -, -).
__device__ __forceinline__ cpx<df> sel(bool c, cpx<df> a, cpx<df> b) {
    return C(df(c ? a.re.h : b.re.h, c ? a.re.l : b.re.l), df(c ? a.im.h : b.im.h, c ? a.im.l : b.im.l));
}
// z + f i^k w (f = +-1; fr = k ? -f : f multiplies the real part's term)
__device__ __forceinline__ cpx<df> df_addc(cpx<df> z, cpx<df> w, bool k, float fr, float f) {
    const cpx<df> x = sel(k, C(w.im, w.re), w);
    return C(df_add(z.re, x.re, fr), df_add(z.im, x.im, f));
}

// The eight hops of flavour f (NF flavours stored) of output site i (parity po).
// Instead of a ninth hop's words, fetch0 fills slots 0 .. 11 and fetch1 slots
// 12 .. 23 for the epilogue (one cp.async group each, both still in flight at the end).
template <typename F0, typename F1>
__device__ __forceinline__ void hops_dw(cpx<df> (&out)[4][3], const OpProb& pr, const Coord& c, long i, int po, int f,
                                        float4* slots, F0 fetch0, F1 fetch1) {
    const Geom& g = pr.g;
    auto neighbour = [&](int hop, bool& wrap) {
        const int mu = hop >> 1;
        const bool fwd = (hop & 1) == 0;
        const int xm = mu == 0 ? c.x : mu == 1 ? c.y : mu == 2 ? c.z : c.t;
        const int lm = mu == 0 ? g.X : mu == 1 ? g.Y : mu == 2 ? g.Z : g.T;
        wrap = fwd ? (xm + 1 == lm) : (xm == 0);
        const int xn = fwd ? (wrap ? 0 : xm + 1) : (wrap ? lm - 1 : xm - 1);
        return cb_index(g, mu == 0 ? xn : c.x, mu == 1 ? xn : c.y, mu == 2 ? xn : c.z, mu == 3 ? xn : c.t);
    };
    CC acc[4][3];
#pragma unroll
    for (int s = 0; s < 4; ++s)
#pragma unroll
        for (int a = 0; a < 3; ++a) acc[s][a] = cc_zero();
    bool wrap;
    dw_fetch<12>(slots, 0, pr.in, g.vh, 12 * f, neighbour(0, wrap));
    dw_commit();
    dw_fetch<9>(slots, 12, pr.gauge[po], g.vh, 0, i);
    dw_commit();
#pragma unroll 1
    for (int hop = 0; hop < 8; ++hop) {
        const int mu = hop >> 1;
        const bool fwd = (hop & 1) == 0;
        const float s = fwd ? -1.f : 1.f;
        const float ph = (mu == 3 && wrap) ? pr.bc_t : 1.f;
        bool nwrap = false;
        const long nn = hop < 7 ? neighbour(hop + 1, nwrap) : 0;
        dw_wait<1>();   // this hop's spinor
        const bool m01 = mu < 2, ik = (mu & 1) == 0;
        const float c0 = -s, c1 = (mu == 1 || mu == 2) ? s : -s;
        const int oa = (m01 ? 9 : 6) * DSLASH_BS, ob = (m01 ? 6 : 9) * DSLASH_BS;
        cpx<df> h0[3], h1[3];
#pragma unroll
        for (int q = 0; q < 3; ++q) {
            h0[q] = df_addc(dw_read(slots + q * DSLASH_BS), dw_read(slots + oa + q * DSLASH_BS), ik, ik ? -c0 : c0, c0);
            h1[q] = df_addc(dw_read(slots + (3 + q) * DSLASH_BS), dw_read(slots + ob + q * DSLASH_BS), ik,
                            ik ? -c1 : c1, c1);
        }
        if (hop < 7) dw_fetch<12>(slots, 0, pr.in, g.vh, 12 * f, nn);
        else fetch0();
        dw_commit();
        dw_wait<1>();   // this hop's link
        // U_ab at slot 12 + 3 a + b; the backward hop takes U^dagger
        const int sa = (fwd ? 3 : 1) * DSLASH_BS, sb = (fwd ? 1 : 3) * DSLASH_BS;
        const float fi = fwd ? ph : -ph;
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            CC t0 = cc_zero(), t1 = cc_zero();
#pragma unroll
            for (int b = 0; b < 3; ++b) {
                cpx<df> e = dw_read(slots + 12 * DSLASH_BS + a * sa + b * sb);
                e = C(df(ph * e.re.h, ph * e.re.l), df(fi * e.im.h, fi * e.im.l));
                cc_fma(t0, e, h0[b]);
                cc_fma(t1, e, h1[b]);
            }
            const cpx<df> g0 = cc_get(t0), g1 = cc_get(t1);
            const cpx<df> x2 = sel(m01, g1, g0), x3 = sel(m01, g0, g1);
            const float d2 = mu == 3 ? -s : s, d3 = mu == 0 ? s : -s;
            cs_add(acc[0][a].re, g0.re);
            cs_add(acc[0][a].im, g0.im);
            cs_add(acc[1][a].re, g1.re);
            cs_add(acc[1][a].im, g1.im);
            const cpx<df> y2 = sel(ik, C(x2.im, x2.re), x2), y3 = sel(ik, C(x3.im, x3.re), x3);
            cs_add(acc[2][a].re, y2.re, ik ? -d2 : d2);
            cs_add(acc[2][a].im, y2.im, d2);
            cs_add(acc[3][a].re, y3.re, ik ? -d3 : d3);
            cs_add(acc[3][a].im, y3.im, d3);
        }
        if (hop < 7) {   // the next hop's link: U_mu(x) forward, U_mu(x - mu) backward
            const int nm = (hop + 1) >> 1;
            const bool nf = !fwd;
            dw_fetch<9>(slots, 12, pr.gauge[nf ? po : 1 - po], g.vh, 9 * nm, nf ? i : nn);
        } else {
            fetch1();
        }
        dw_commit();
        wrap = nwrap;
    }
#pragma unroll
    for (int s = 0; s < 4; ++s)
#pragma unroll
        for (int a = 0; a < 3; ++a) out[s][a] = cc_get(acc[s][a]);
}

// s += (H v)_r for a packed hermitian 6x6 block in slots 0 .. 17 (36 reals), r at run
// time: the rows are a loop (unrolled, the blocks' straight code stalls on instruction fetch)
__device__ __forceinline__ void herm6_row_dw(CC& s, const float4* slots, const cpx<df> (&v)[6], int r) {
    const int tr = 3 + r * (r - 1) / 2;   // slot of entry (r, 0)
#pragma unroll
    for (int j = 0; j < 6; ++j) {
        // H_rj = lower entry (r, j) for r > j, the conjugate of (j, r) for r < j, diagonal r real (two a slot)
        const int k = j < r ? tr + j : (j > r ? 3 + j * (j - 1) / 2 + r : r >> 1);
        cpx<df> e = dw_read(slots + k * DSLASH_BS);
        const bool diag = j == r;
        const float si = j < r ? 1.f : (diag ? 0.f : -1.f);
        if (diag && (r & 1)) e.re = e.im;
        e.im = df(si * e.im.h, si * e.im.l);
        cc_fma(s, e, v[j]);
    }
}

__device__ __forceinline__ df shfl_pair_dw(unsigned mask, df x) {
    return df(__shfl_xor_sync(mask, x.h, 1), __shfl_xor_sync(mask, x.l, 1));
}

template <int NF, int KIND>
__global__ void __launch_bounds__(DSLASH_BS, 4) dslash_dw_kernel(const __grid_constant__ OpBatch<1> b) {
    extern __shared__ __align__(16) float4 dw_smem[];
    const OpProb& pr = b.p[0];
    pdl_wait();
    if (pr.ctl != nullptr && pr.ctl->flag != CTL_RUN) return;
    const long gt = (long)blockIdx.x * DSLASH_BS + threadIdx.x;
    const long i = NF == 2 ? gt >> 1 : gt;
    const int f = NF == 2 ? (int)(gt & 1) : 0;
    const long vh = pr.g.vh;
    const bool valid = i < vh;
    const unsigned mask = __ballot_sync(0xffffffffu, valid);   // both threads of a site agree
    if (!valid) return;
    constexpr int po = (KIND == K1_EO_INV) ? 0 : 1;
    const Coord c = cb_coords(pr.g, i, po);
    float4* slots = dw_smem + threadIdx.x;   // slot k at slots + k * DSLASH_BS; every thread uses its own only
    cpx<df> acc[4][3];
    if constexpr (KIND == K1_EO_INV && NF == 1) {
        // t = B_c v per chirality block c, B_c = (A_c + i s_c mu_t)^-1 stored row
        // major (72 reals); the adjoint sign applies B_c^dagger, whose entry (r, j) is
        // the conjugate of the stored (j, r).  Rows of both blocks pass through the
        // slots in a ring of four.
        const float4* cl = reinterpret_cast<const float4*>(pr.clov) + i;
        const bool plus = pr.sign > 0;
        const long sr = (plus ? 6 : 1) * vh, sj = (plus ? 1 : 6) * vh;
        const float si = plus ? 1.f : -1.f;
        auto fetch_row = [&](int k) {   // row k % 6 of block k / 6
            const float4* p = cl + (k < 6 ? k * sr : 36 * vh + (k - 6) * sr);
#pragma unroll
            for (int j = 0; j < 6; ++j) dw_copy(slots + ((k & 3) * 6 + j) * DSLASH_BS, p + j * sj);
        };
        hops_dw(acc, pr, c, i, po, f, slots, [&] { fetch_row(0); fetch_row(1); }, [&] { fetch_row(2); fetch_row(3); });
        dw_wait<1>();   // rows 0 and 1
#pragma unroll 1
        for (int cb = 0; cb < 2; ++cb) {
            cpx<df> v[6];
#pragma unroll
            for (int j = 0; j < 6; ++j) v[j] = sel(cb == 0, acc[j / 3][j % 3], acc[2 + j / 3][j % 3]);
#pragma unroll 1
            for (int r = 0; r < 6; ++r) {
                const int k = 6 * cb + r;
                dw_wait<2>();   // groups in flight: rows 0-1, 2-3, then one a row: all but the newest two
                CC w = cc_zero();
#pragma unroll
                for (int j = 0; j < 6; ++j) {
                    cpx<df> e = dw_read(slots + ((k & 3) * 6 + j) * DSLASH_BS);
                    e.im = df(si * e.im.h, si * e.im.l);
                    cc_fma(w, e, v[j]);
                }
                if (k + 4 < 12) fetch_row(k + 4);
                dw_commit();
                const cpx<df> o = cc_get(w);
                // out[6 cb + r] without a run-time register index: store directly
                store_reals<PDF, 2>(pr.out, vh, i, 2 * k, reinterpret_cast<const df*>(&o));
            }
        }
    } else if constexpr (KIND == K1_EO_INV) {
        // heavy inverse from A_c - 1 and D_c - 1 (dslash_heavy.cu):
        //   dv = D v, w = A dv, out = w + t i dv + epsbar_t (D v of the partner flavour),
        //   t = (f == 0 ? -1 : 1) (c == 0 ? tw : -tw)
        // (blocks in slots 0 .. 17, v and then dv in slots 18 .. 23)
        hops_dw(acc, pr, c, i, po, f, slots, [&] { dw_fetch<12>(slots, 0, pr.clov, vh, 18, i); },
                [&] { dw_fetch<6>(slots, 12, pr.clov, vh, 30, i); });   // D_0 - 1
        const df tw = df(pr.tw);
        const df eps = df(pr.eps);
#pragma unroll 1
        for (int cb = 0; cb < 2; ++cb) {
            const float ts = (f == 0 ? -1.f : 1.f) * (cb == 0 ? 1.f : -1.f);
            const df t = df(ts * tw.h, ts * tw.l);
            cpx<df> v[6];
#pragma unroll
            for (int j = 0; j < 6; ++j) {
                v[j] = sel(cb == 0, acc[j / 3][j % 3], acc[2 + j / 3][j % 3]);
                dw_write(slots + (18 + j) * DSLASH_BS, v[j]);
            }
            dw_wait<0>();
#pragma unroll 1
            for (int r = 0; r < 6; ++r) {
                float4* own = slots + (18 + r) * DSLASH_BS;
                CC s = cc_zero();
                const cpx<df> v0 = dw_read(own);
                cs_add(s.re, v0.re);
                cs_add(s.im, v0.im);
                herm6_row_dw(s, slots, v, r);
                dw_write(own, cc_get(s));
            }
            dw_fetch<18>(slots, 0, pr.clov, vh, 36 * cb, i);   // A_c - 1
            dw_commit();
#pragma unroll
            for (int j = 0; j < 6; ++j) v[j] = dw_read(slots + (18 + j) * DSLASH_BS);
            dw_wait<0>();
#pragma unroll 1
            for (int r = 0; r < 6; ++r) {
                const cpx<df> dv = dw_read(slots + (18 + r) * DSLASH_BS);
                const cpx<df> dp = C(shfl_pair_dw(mask, dv.re), shfl_pair_dw(mask, dv.im));
                CC s = cc_zero();
                cs_add(s.re, dv.re);
                cs_add(s.im, dv.im);
                herm6_row_dw(s, slots, v, r);
                const cpx<df> w = cc_get(s);
                CC o = cc_zero();
                cs_add(o.re, w.re);
                cs_add(o.im, w.im);
                cs_fms(o.re, t, dv.im);   // t i dv
                cs_fma(o.im, t, dv.re);
                cs_fma(o.re, eps, dp.re);
                cs_fma(o.im, eps, dp.im);
                const cpx<df> q = cc_get(o);
                store_reals<PDF, 2>(pr.out, vh, i, 24 * f + 2 * (6 * cb + r), reinterpret_cast<const df*>(&q));
            }
            if (cb == 0) {
                dw_fetch<18>(slots, 0, pr.clov, vh, 54, i);   // D_1 - 1
                dw_commit();
            }
        }
    } else {
        // out = g5 [ (A + i tw g5 [tau3]) psi - eps tau1 psi - kappa^2 acc ] + i rho psi,
        // A hermitian (36 reals per block); i rho psi = g5 (i rho g5 psi) joins the twist
        // (blocks in slots 0 .. 17, the rest of the sum in slots 18 .. 23)
        hops_dw(acc, pr, c, i, po, f, slots, [&] { dw_fetch<12>(slots, 0, pr.clov, vh, 0, i); },
                [&] { dw_fetch<6>(slots, 12, pr.clov, vh, 12, i); });   // A_0
        const df k2 = df(pr.kappa * pr.kappa);
        const df tr = df(f == 0 ? pr.tw + pr.rho : pr.rho - pr.tw);
        const df eps = df(pr.eps);
#pragma unroll 1
        for (int cb = 0; cb < 2; ++cb) {
            const float sc = cb == 0 ? 1.f : -1.f;   // g5 on the block
            const df t = df(sc * tr.h, sc * tr.l);
            cpx<df> v[6];
            load_reals<PDF, 12>(pr.loc, vh, i, 24 * f + 12 * cb, reinterpret_cast<df*>(v));
#pragma unroll
            for (int r = 0; r < 6; ++r) {
                // i sc (tw t3 + rho) v_r - eps v'_r - kappa^2 acc_r
                const cpx<df> a = sel(cb == 0, acc[r / 3][r % 3], acc[2 + r / 3][r % 3]);
                CC s = cc_zero();
                cs_fms(s.re, t, v[r].im);
                cs_fma(s.im, t, v[r].re);
                if constexpr (NF == 2) {
                    df vp[2];
                    load_reals<PDF, 2>(pr.loc, vh, i, 24 * (1 - f) + 12 * cb + 2 * r, vp);
                    cs_fms(s.re, eps, vp[0]);
                    cs_fms(s.im, eps, vp[1]);
                }
                cs_fms(s.re, k2, a.re);
                cs_fms(s.im, k2, a.im);
                dw_write(slots + (18 + r) * DSLASH_BS, cc_get(s));
            }
            dw_wait<0>();
#pragma unroll 1
            for (int r = 0; r < 6; ++r) {
                const cpx<df> w0 = dw_read(slots + (18 + r) * DSLASH_BS);
                CC s = cc_zero();
                cs_add(s.re, w0.re);
                cs_add(s.im, w0.im);
                herm6_row_dw(s, slots, v, r);
                const cpx<df> w = cc_get(s);
                const cpx<df> o = C(df(sc * w.re.h, sc * w.re.l), df(sc * w.im.h, sc * w.im.l));
                const int off = 24 * f + 2 * (6 * cb + r);
                if constexpr (KIND == K2_OUT64) {
                    const double q[2] = {(double)o.re, (double)o.im};
                    store_reals<P64, 2>(pr.out, vh, i, off, q);
                } else {
                    store_reals<PDF, 2>(pr.out, vh, i, off, reinterpret_cast<const df*>(&o));
                }
            }
            if (cb == 0) {
                dw_fetch<18>(slots, 0, pr.clov, vh, 18, i);   // A_1
                dw_commit();
            }
        }
    }
}

template <int P, int NF, int KIND, int NP>
cudaError_t launch_dslash(const OpBatch<NP>& b, int nblocks, cudaStream_t st);

// the double-word instantiations of launch_dslash (no batch tables, no fused
// norm: the reliable updates use neither); two-flavour passes take 2 vh threads
#define TM_DW_INST(NF, KIND)                                                                       \
    template <>                                                                                    \
    cudaError_t launch_dslash<PDF, NF, KIND, 1>(const OpBatch<1>& b, int nblocks, cudaStream_t st) { \
        if (b.n != 1 || b.p[0].partial != nullptr) return cudaErrorInvalidValue;                    \
        const cudaError_t e = cudaFuncSetAttribute(dslash_dw_kernel<NF, KIND>,                     \
                                                   cudaFuncAttributeMaxDynamicSharedMemorySize, DW_SMEM); \
        if (e != cudaSuccess) return e;                                                            \
        return launch_chained(dslash_dw_kernel<NF, KIND>, nblocks, DSLASH_BS, DW_SMEM, st, b.chained, b); \
    }
TM_DW_INST(1, K1_EO_INV)
TM_DW_INST(1, K2_OE_LOCAL)
TM_DW_INST(2, K1_EO_INV)
TM_DW_INST(2, K2_OE_LOCAL)
TM_DW_INST(1, K2_OUT64)
TM_DW_INST(2, K2_OUT64)

}  // namespace tmk
