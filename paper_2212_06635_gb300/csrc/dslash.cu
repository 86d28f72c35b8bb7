// Even-odd Schur operator kernels of eq:hQpm (light doublet) and the odd pass of
// eq:hQh (heavy doublet; its even pass is in dslash_heavy.cu).
//
//   Q_hat psi_o = g5 [ (M_oo) psi_o - M_oe M_ee^-1 M_eo psi_o ],  M_eo = -kappa H_eo
//
// is applied in two passes, one thread per output site:
//   K1 (even output):  t_e = (M_ee)^-1 H_eo psi_o            hop + site-local 6x6 inverse blocks
//   K2 (odd output):   out = g5 [ M_oo psi_o - kappa^2 H_oe t_e ]   hop + clover/twist + g5
// K2 can fuse ||out||^2 into a deterministic two-level FP64 reduction whose last
// block finalises a solver scalar (CG alpha), so a CG iteration needs no separate
// reduction launch.  Every kernel takes a table of problems (one or a batch of
// lattices of different volumes); a block belongs to exactly one problem.
#include "tm_internal.h"
#include "tm_kernels.h"
#include "dslash_common.cuh"

namespace tmk {

// Whether the first hop writes the accumulators instead of adding to zeros (which
// saves 24 additions a flavour, but moves the register allocation): per pass what
// measured faster.  Adding / writing, us: light FP16 even 106.6 / 110.6, odd 102.3 /
// 100.8; FP32 even 198.7 / 180.4 (with the register cap below), odd 152.3 / 149.4;
// BF16 at 18x22x26x44 30.7 / 31.3 and 28.7 / 29.5; two-flavour odd pass at 24^3x48
// FP16 61.6 / 61.3 (59.5 with the factor folded, hop_dir), FP32 75.0 / 75.9.
template <int P, int NF, int KIND>
constexpr bool hop_first() {
    if (P == P64) return true;
    if (P == P32) return NF == 1;
    return P == PF16 && (NF == 2 || KIND != K1_EO_INV);
}

// All 8 hops for NF flavours into acc[NF][4][3]; output site (c, i) of parity po.
template <int P, int NF, int KIND, int MU>
__device__ __forceinline__ void hop_mu(cpx<typename PT<P>::R> (&acc)[NF][4][3], const OpProb& pr,
                                       const Coord& c, long i, int po) {
    using R = typename PT<P>::R;
    const Geom& g = pr.g;
    int xf = c.x, yf = c.y, zf = c.z, tf = c.t;
    int xb = c.x, yb = c.y, zb = c.z, tb = c.t;
    R ph_f = (R)1, ph_b = (R)1;
    if (MU == 0) { xf = (c.x + 1 == g.X) ? 0 : c.x + 1; xb = (c.x == 0) ? g.X - 1 : c.x - 1; }
    if (MU == 1) { yf = (c.y + 1 == g.Y) ? 0 : c.y + 1; yb = (c.y == 0) ? g.Y - 1 : c.y - 1; }
    if (MU == 2) { zf = (c.z + 1 == g.Z) ? 0 : c.z + 1; zb = (c.z == 0) ? g.Z - 1 : c.z - 1; }
    if (MU == 3) {
        if (c.t + 1 == g.T) { tf = 0; ph_f = (R)pr.bc_t; } else tf = c.t + 1;
        if (c.t == 0) { tb = g.T - 1; ph_b = (R)pr.bc_t; } else tb = c.t - 1;
    }
    const long nf = cb_index(g, xf, yf, zf, tf);
    const long nb = cb_index(g, xb, yb, zb, tb);
    constexpr bool SC = (P == PF16 || P == PB16);   // 16-bit: the scale joins the phase
    constexpr bool FIRST = MU == 0 && hop_first<P, NF, KIND>();
    cpx<R> u[9];
    cpx<R> psi[NF * 12];
    float sc;
    load_spinor_unscaled<P, NF * 12>(pr.in, g.vh, nf, psi, sc);
    load_link<P>(pr.gauge[po], g.vh, MU, i, u);
#pragma unroll
    for (int f = 0; f < NF; ++f)
        hop_dir<R, MU, -1, false, SC, FIRST, NF == 2>(acc[f], psi + 12 * f, u, SC ? ph_f * (R)sc : ph_f);
    load_spinor_unscaled<P, NF * 12>(pr.in, g.vh, nb, psi, sc);
    load_link<P>(pr.gauge[1 - po], g.vh, MU, nb, u);
#pragma unroll
    for (int f = 0; f < NF; ++f)
        hop_dir<R, MU, +1, true, SC, false, NF == 2>(acc[f], psi + 12 * f, u, SC ? ph_b * (R)sc : ph_b);
}

// out = B_c v (CONJ: B_c^dagger v) per chirality block c of the even-site inverse.
// The sign is decided outside: inside the products it made every FMA a pair of
// predicated ones (FP64 even pass at 16^3x32 188.5 -> 149.8 us, light FP16 at
// 32^3x64 112.5 -> 106.6 us).
template <int P, bool CONJ>
__device__ __forceinline__ void inverse_blocks(cpx<typename PT<P>::R>* out, const OpProb& pr, long i,
                                               const cpx<typename PT<P>::R> (&acc)[4][3]) {
    using R = typename PT<P>::R;
#pragma unroll
    for (int cb = 0; cb < 2; ++cb) {
        cpx<R> v[6], w[6];
#pragma unroll
        for (int j = 0; j < 6; ++j) {
            v[j] = acc[2 * cb + j / 3][j % 3];
            w[j] = C((R)0, (R)0);
        }
        // stream the block two rows (24 reals) at a time to bound registers
#pragma unroll
        for (int rr = 0; rr < 3; ++rr) {
            R m[24];
            load_readonly<P, 24>(pr.clov, pr.g.vh, i, 72 * cb + 24 * rr, m);
#pragma unroll
            for (int r2 = 0; r2 < 2; ++r2) {
                const int r = 2 * rr + r2;
#pragma unroll
                for (int j = 0; j < 6; ++j) {
                    const cpx<R> e = C(m[2 * (6 * r2 + j)], m[2 * (6 * r2 + j) + 1]);
                    if (CONJ) cfma_cj(w[j], e, v[r]);
                    else cfma(w[r], e, v[j]);
                }
            }
        }
#pragma unroll
        for (int j = 0; j < 6; ++j) out[6 * cb + j] = w[j];
    }
}

// Resident blocks the compiler must fit per SM (128-thread blocks, FP64 64-thread
// ones; the register cap follows).  Sweeps at 32^3x64 (light) and 24^3x48 (heavy)
// put the optimum at:
//   light 16-bit even pass: 5 blocks (96 registers; the inverse blocks stream two
//     rows at a time for this).  6 blocks: 112.8 -> 133.4 us FP16, 116.6 -> 174.2 us
//     BF16 (before inverse_blocks took its present form: 106.6 us FP16 since);
//   light odd pass: 7 blocks FP16 (72 registers, 16 B spilled) and 6 BF16 (80
//     registers): 5 / 6 / 7 blocks take 112.2 / 104.9 / 103.0 us FP16 and
//     126.9 / 113.2 / 119.0 us BF16 (4 blocks: 108.3 / 113.1 us);
//   light FP32 odd pass: 4 blocks (128 registers, 16 B spilled): 156.5 -> 150.0 us
//     (3 blocks 152.0 us); even pass: 3 blocks (168 registers): 180.4 us against
//     202.8 us at the 188 registers the compiler takes without a bound;
//   two-flavour odd pass: 4 blocks in 16-bit storage (128 registers; 3 / 5
//     blocks: 63.8 -> 67.7 / 75.0 us FP16) and 3 in FP32 (168 registers, 8 B
//     spilled: 94.8 -> 78.1 us at 24^3x48; 2 / 4 blocks: 94.5 / 84.4 us);
//   FP64: 8 blocks of 64 threads (128 registers; 172 B stored to and 176 B loaded from
//     the stack in the even pass, 264 / 300 B in the odd one, 80 / 80 B in the
//     update).  The FP64 units bound the passes, but the waits for operands show at 8
//     warps per SM on lattices of few waves: 4 / 6 / 8 blocks (254 and 168 registers,
//     none spilled) take, even + odd, 320 / 318 / 300 us at 16^3x32, 1377 / 1376 /
//     1378 us at 24^3x48 and 4121 / 4114 / 4116 us at 32^3x64.  4 blocks of 128 threads:
//     320 / 1379 / 4112 us.
// (The two-flavour even pass splits the flavours over a thread pair: dslash_heavy.cu.)
template <int P, int NF, int KIND>
constexpr int dslash_min_blocks() {
    if (P == PF16 || P == PB16) {
        if (NF == 2) return 4;
        if (KIND == K1_EO_INV) return 5;
        return P == PF16 ? 7 : 6;
    }
    if (P == P32) return KIND == K1_EO_INV ? 3 : (NF == 2 ? 3 : 4);
    return 8;   // P64
}

template <int P, int NF, int KIND, int NP, int BS>
__global__ void __launch_bounds__(BS, (dslash_min_blocks<P, NF, KIND>())) dslash_kernel(const __grid_constant__ OpBatch<NP> b) {
    static_assert(NF == 1 || (KIND != K1_EO_INV && P != P64), "two-flavour passes of dslash_heavy.cu");
    using R = typename PT<P>::R;
    __shared__ double sh[BS / 32];
    const int k = find_problem<NP>(b, blockIdx.x);
    const OpProb& pr = b.p[k];
    pdl_wait();
    if (pr.ctl != nullptr && pr.ctl->flag != CTL_RUN) return;
    const int lb = block_in_problem<NP>(b, blockIdx.x, k);
    const long i = (long)lb * BS + threadIdx.x;
    const bool valid = i < pr.g.vh;
    const int po = (KIND == K1_EO_INV) ? 0 : 1;   // output parity
    double nrm = 0.0;
    if (valid) {
        const Coord c = cb_coords(pr.g, i, po);
        cpx<R> acc[NF][4][3];
        if constexpr (!hop_first<P, NF, KIND>()) {
#pragma unroll
            for (int f = 0; f < NF; ++f)
#pragma unroll
                for (int s = 0; s < 4; ++s)
#pragma unroll
                    for (int a = 0; a < 3; ++a) acc[f][s][a] = C((R)0, (R)0);
        }
        hop_mu<P, NF, KIND, 0>(acc, pr, c, i, po);
        hop_mu<P, NF, KIND, 1>(acc, pr, c, i, po);
        hop_mu<P, NF, KIND, 2>(acc, pr, c, i, po);
        hop_mu<P, NF, KIND, 3>(acc, pr, c, i, po);

        cpx<R> out[NF * 12];
        if constexpr (KIND == K1_EO_INV) {
            if constexpr (NF == 1) {
                // t_e = (A_c + i sign s_c mu_t)^-1 (H psi) per chirality block c
                if (pr.sign > 0) inverse_blocks<P, false>(out, pr, i, acc[0]);
                else inverse_blocks<P, true>(out, pr, i, acc[0]);
            }
        } else {
            // out = g5 [ (A + i tw g5 [tau3]) psi - eps tau1 psi - kappa^2 acc ]
            cpx<R> psi[NF * 12];
            load_spinor<P, NF * 12>(pr.loc, pr.g.vh, i, psi);
            R m[72];
            load_readonly<P, 72>(pr.clov, pr.g.vh, i, 0, m);
            const R k2 = (R)(pr.kappa * pr.kappa);
            // W_hat = Q_hat + i rho (eq:hWpm): i rho psi = g5 (i rho g5 psi) joins the twist
            const R tw = (R)pr.tw, rho = (R)pr.rho;
            const R eps = (R)pr.eps;
#pragma unroll
            for (int f = 0; f < NF; ++f) {
                const R t3 = (f == 0) ? (R)1 : (R)-1;
#pragma unroll
                for (int cb = 0; cb < 2; ++cb) {
                    const R sc = (cb == 0) ? (R)1 : (R)-1;
                    cpx<R> v[6], w[6];
#pragma unroll
                    for (int j = 0; j < 6; ++j) {
                        v[j] = psi[12 * f + 6 * cb + j];
                        w[j] = (sc * (tw * t3 + rho)) * mul_i(v[j]);
                        if constexpr (NF == 2) w[j] = w[j] - eps * psi[12 * (1 - f) + 6 * cb + j];
                        w[j] = w[j] - k2 * acc[f][2 * cb + j / 3][j % 3];
                    }
                    herm6_mv_acc<R>(w, m + 36 * cb, v);
#pragma unroll
                    for (int j = 0; j < 6; ++j) out[12 * f + 6 * cb + j] = (cb == 0) ? w[j] : -w[j];
                }
            }
            if constexpr (KIND == K2_UPDATE) residual_update<P, NF * 12>(out, pr, i);
            if (KIND == K2_UPDATE || pr.partial != nullptr) {
                R s = (R)0;
#pragma unroll
                for (int q = 0; q < NF * 12; ++q) s += norm2(out[q]);
                nrm = (double)s;
            }
        }
        store_spinor<P, NF * 12>(pr.out, pr.g.vh, i, out);
    }
    if constexpr (KIND != K1_EO_INV) {
      if (KIND == K2_UPDATE || pr.partial != nullptr) {
        const double bs = block_sum<BS>(nrm, sh);
        reduce_finalize<BS>(pr.partial, pr.counter, pr.nblk, lb, bs, b.fin, pr.ctl, pr.ms,
                            nullptr, sh);
      }
    }
}

template <int P, int NF, int KIND, int NP>
cudaError_t launch_dslash(const OpBatch<NP>& b, int nblocks, cudaStream_t st) {
    return launch_chained(dslash_kernel<P, NF, KIND, NP, dslash_bs(P)>, nblocks, dslash_bs(P), 0, st, b.chained, b);
}

#define TM_INST(P, NF, KIND, NP) \
    template cudaError_t launch_dslash<P, NF, KIND, NP>(const OpBatch<NP>&, int, cudaStream_t);
#define TM_INST_P(P)                                                                      \
    TM_INST(P, 1, K1_EO_INV, 1) TM_INST(P, 1, K2_OE_LOCAL, 1) TM_INST(P, 1, K2_UPDATE, 1) \
    TM_INST(P, 1, K1_EO_INV, MAXP) TM_INST(P, 1, K2_OE_LOCAL, MAXP)
#define TM_INST_TWO(P) TM_INST(P, 2, K2_OE_LOCAL, 1) TM_INST(P, 2, K2_UPDATE, 1)
TM_INST_P(P64)   // (its two-flavour odd pass: dslash_heavy.cu; the double-word passes: dslash_dw.cu)
TM_INST_P(P32) TM_INST_TWO(P32)
TM_INST_P(PB16) TM_INST_TWO(PB16)
TM_INST_P(PF16) TM_INST_TWO(PF16)
#define TM_INST_GROUP(P)                                                                             \
    TM_INST(P, 1, K1_EO_INV, GROUP) TM_INST(P, 1, K2_OE_LOCAL, GROUP) TM_INST(P, 1, K2_UPDATE, GROUP) \
    TM_INST(P, 2, K2_OE_LOCAL, GROUP) TM_INST(P, 2, K2_UPDATE, GROUP)
TM_INST_GROUP(P32)
TM_INST_GROUP(PB16)
TM_INST_GROUP(PF16)

}  // namespace tmk
