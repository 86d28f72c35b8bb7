// Stencil passes of eq:hQpm / eq:hQh for lattices too small to fill the GPU with a
// thread per site: the work of a site is split over 4 threads (8 for two flavours)
// in as many warps.
//
// A small pass is a chain of latencies: one thread's 8 hops and block products are
// 2,700 instructions in a row, and the 32 blocks of an 8^3x16 lattice occupy 32 of 152
// SMs.  Here a block covers 32 sites; warp (mu, flavour) computes the two hops of
// direction mu (no divergence, all loads of a thread in flight at once), the partial
// sums meet in shared memory, and warp (chirality, spin, flavour) forms three rows of
// the site-local product, so that each warp has a quarter of the work in both halves.
// The clover rows are loaded before the wait for the pass before (launch_chained), and
// the next pass may start at once.  Shared memory [warp][real][lane] is free of bank
// conflicts.  M_hat^dagger M_hat at 4^4 as a graph, direct / split: light FP32 17.8 /
// 9.5 us, light FP64 153 / 47 us, heavy FP64 256 / 97 us.  (The four passes as one
// cooperative launch with grid barriers: light FP32 12.9 us, so not used.)
//
// The split costs instructions (each warp of a site computes the coordinates, rows
// are read by 8- or 4-byte pieces), so larger lattices keep the thread per site:
// split_limit (api.cu) holds the line and its measurements.
#include "tm_internal.h"
#include "tm_kernels.h"
#include "dslash_common.cuh"

namespace tmk {

// complex number e (reals 2e, 2e + 1) and real r of a site's native array (RO: load_vec)
template <int P, bool RO>
__device__ __forceinline__ cpx<typename PT<P>::R> load_complex(const void* base, long vh, long i, int e) {
    if constexpr (P == P64) {
        const double2 q = load_vec<RO>(reinterpret_cast<const double2*>(base) + (long)e * vh + i);
        return C(q.x, q.y);
    } else if constexpr (P == P32) {
        const float2 q = load_vec<RO>(reinterpret_cast<const float2*>(base) + ((long)(e >> 1) * vh + i) * 2 + (e & 1));
        return C(q.x, q.y);
    } else {
        const float2 q =
            h2f2<P>(load_vec<RO>(reinterpret_cast<const unsigned int*>(base) + ((long)(e >> 2) * vh + i) * 4 + (e & 3)));
        return C(q.x, q.y);
    }
}
template <int P, bool RO>
__device__ __forceinline__ typename PT<P>::R load_real(const void* base, long vh, long i, int r) {
    constexpr int W = PT<P>::W;
    const long e = ((long)(r / W) * vh + i) * W + r % W;
    if constexpr (P == P64) return load_vec<RO>(reinterpret_cast<const double*>(base) + e);
    else if constexpr (P == P32) return load_vec<RO>(reinterpret_cast<const float*>(base) + e);
    else return h2f<P>(load_vec<RO>(reinterpret_cast<const uint16_t*>(base) + e));
}
template <int P>
__device__ __forceinline__ void store_complex(void* base, long vh, long i, int e, cpx<typename PT<P>::R> z) {
    if constexpr (P == P64) reinterpret_cast<double2*>(base)[(long)e * vh + i] = make_double2(z.re, z.im);
    else if constexpr (P == P32)
        reinterpret_cast<float2*>(base)[((long)(e >> 1) * vh + i) * 2 + (e & 1)] = make_float2(z.re, z.im);
    else reinterpret_cast<unsigned int*>(base)[((long)(e >> 2) * vh + i) * 4 + (e & 3)] = f2h2<P>(z.re, z.im);
}

// entries (r, j), j = 0 .. 5, of a packed hermitian block (clover data) at real offset off
template <int P>
__device__ __forceinline__ void load_herm_row(cpx<typename PT<P>::R> (&m)[6], const void* base, long vh, long i, int off,
                                              int r) {
    using R = typename PT<P>::R;
#pragma unroll
    for (int j = 0; j < 6; ++j) {
        const int hi = r > j ? r : j, lo = r > j ? j : r;
        if (r == j) m[j] = C(load_real<P, true>(base, vh, i, off + r), (R)0);
        else {
            m[j] = load_complex<P, true>(base, vh, i, (off + 6) / 2 + hi * (hi - 1) / 2 + lo);
            if (r < j) m[j].im = -m[j].im;
        }
    }
}

// the two hops of direction MU of flavour f into acc
template <int P, int NF, int MU>
__device__ __forceinline__ void split_hops(cpx<typename PT<P>::R> (&acc)[4][3], const OpProb& pr, const Coord& c, long i,
                                           int po, int f) {
    using R = typename PT<P>::R;
    const Geom& g = pr.g;
    const int x = MU == 0 ? c.x : (MU == 1 ? c.y : (MU == 2 ? c.z : c.t));
    const int L = MU == 0 ? g.X : (MU == 1 ? g.Y : (MU == 2 ? g.Z : g.T));
    const int xf = x + 1 == L ? 0 : x + 1, xb = x == 0 ? L - 1 : x - 1;
    auto at = [&](int q) {
        return cb_index(g, MU == 0 ? q : c.x, MU == 1 ? q : c.y, MU == 2 ? q : c.z, MU == 3 ? q : c.t);
    };
    const long nf = at(xf), nb = at(xb);
    constexpr bool SC = (P == PF16 || P == PB16);
    R ff = MU == 3 && x + 1 == L ? (R)pr.bc_t : (R)1, fb = MU == 3 && x == 0 ? (R)pr.bc_t : (R)1;
    cpx<R> uf[9], ub[9], pf[12], pb[12];
    load_link<P>(pr.gauge[po], g.vh, MU, i, uf);
    load_link<P>(pr.gauge[1 - po], g.vh, MU, nb, ub);
    load_reals<P, 24>(pr.in, g.vh, nf, 24 * f, reinterpret_cast<R*>(pf));
    load_reals<P, 24>(pr.in, g.vh, nb, 24 * f, reinterpret_cast<R*>(pb));
    if constexpr (SC) {
        const float* scale = reinterpret_cast<const float*>(reinterpret_cast<const char*>(pr.in) + (size_t)g.vh * NF * 12 * 4);
        ff *= scale[nf];
        fb *= scale[nb];
    }
    hop_dir<R, MU, -1, false, SC, true>(acc, pf, uf, ff);
    hop_dir<R, MU, +1, true, SC>(acc, pb, ub, fb);
}

template <int P, int NF>
constexpr size_t split_smem() { return (size_t)4 * NF * 24 * 32 * sizeof(typename PT<P>::R); }

template <int P, int NF, int KIND>
__global__ void __launch_bounds__(128 * NF) dslash_split_kernel(const __grid_constant__ OpBatch<1> b) {
    using R = typename PT<P>::R;
    constexpr int NW = 4 * NF, BS = 32 * NW;
    extern __shared__ __align__(16) unsigned char split_mem[];
    R* part = reinterpret_cast<R*>(split_mem);   // [warp][real][lane]
    __shared__ float site_max[NW][32];
    __shared__ double sh[NW];
    const OpProb& pr = b.p[0];
    pdl_trigger();
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const long vh = pr.g.vh, i = (long)blockIdx.x * 32 + lane;
    const bool valid = i < vh;
    constexpr int po = (KIND == K1_EO_INV) ? 0 : 1;
    const int f = w >> 2;
    // the second half's share: rows 3 h + c, c = 0 .. 2, of chirality cb (spin 2 cb + h)
    const int cb = (w >> 1) & 1, h = w & 1;
    cpx<R> m[3][6];    // rows of the first site-local matrix
    cpx<R> v[6];       // odd pass: psi of this chirality; even pass: the summed hops
    if (valid) {
        if constexpr (KIND == K1_EO_INV && NF == 1) {
#pragma unroll
            for (int c = 0; c < 3; ++c)
#pragma unroll
                for (int j = 0; j < 6; ++j) {   // B, or the conjugate of its transpose
                    const int r = 3 * h + c;
                    m[c][j] = load_complex<P, true>(pr.clov, vh, i, 36 * cb + (pr.sign > 0 ? 6 * r + j : 6 * j + r));
                    if (pr.sign < 0) m[c][j].im = -m[c][j].im;
                }
        } else {
            // D_c - 1 (even pass, heavy) or A_c (odd pass)
            const int off = KIND == K1_EO_INV ? 72 * cb + 36 : 36 * cb;
#pragma unroll
            for (int c = 0; c < 3; ++c) load_herm_row<P>(m[c], pr.clov, vh, i, off, 3 * h + c);
        }
    }
    pdl_wait();
    if (pr.ctl != nullptr && pr.ctl->flag != CTL_RUN) return;   // the same for every thread
    if (valid) {
        const Coord x = cb_coords(pr.g, i, po);
        cpx<R> acc[4][3];
        switch (w & 3) {   // warp-uniform
            case 0: split_hops<P, NF, 0>(acc, pr, x, i, po, f); break;
            case 1: split_hops<P, NF, 1>(acc, pr, x, i, po, f); break;
            case 2: split_hops<P, NF, 2>(acc, pr, x, i, po, f); break;
            default: split_hops<P, NF, 3>(acc, pr, x, i, po, f); break;
        }
        R* mine = part + w * 24 * 32 + lane;
#pragma unroll
        for (int s = 0; s < 4; ++s)
#pragma unroll
            for (int c = 0; c < 3; ++c) {
                mine[(2 * (3 * s + c)) * 32] = acc[s][c].re;
                mine[(2 * (3 * s + c) + 1) * 32] = acc[s][c].im;
            }
    }
    __syncthreads();
    // complex component q (0 .. 11) of flavour f, summed over the directions
    auto hops = [&](int q) {
        const R* p = part + (4 * f * 24 + 2 * q) * 32 + lane;
        cpx<R> s = C(p[0], p[32]);
#pragma unroll
        for (int d = 1; d < 4; ++d) s = s + C(p[d * 24 * 32], p[(d * 24 + 1) * 32]);
        return s;
    };
    cpx<R> out[3];
    if constexpr (KIND == K1_EO_INV) {
        if (valid) {
#pragma unroll
            for (int j = 0; j < 6; ++j) v[j] = hops(6 * cb + j);
        }
        if constexpr (NF == 1) {
#pragma unroll
            for (int c = 0; c < 3; ++c) {
                out[c] = C((R)0, (R)0);
#pragma unroll
                for (int j = 0; j < 6; ++j) cfma(out[c], m[c][j], v[j]);
            }
        } else {
            // dv = D v, shared, then out = A dv +- i mubar_t dv + epsbar_t dv of the
            // partner flavour (dslash_heavy.cu)
            cpx<R> dv[3];
#pragma unroll
            for (int c = 0; c < 3; ++c) {
                dv[c] = h == 0 ? v[c] : v[3 + c];
#pragma unroll
                for (int j = 0; j < 6; ++j) cfma(dv[c], m[c][j], v[j]);
            }
            if (valid) {
#pragma unroll
                for (int c = 0; c < 3; ++c) load_herm_row<P>(m[c], pr.clov, vh, i, 72 * cb, 3 * h + c);   // A_c - 1
            }
            __syncthreads();   // every warp has read the partial sums
            R* mine = part + w * 6 * 32 + lane;   // [warp = (flavour, chirality, spin)][real][lane]
#pragma unroll
            for (int c = 0; c < 3; ++c) {
                mine[2 * c * 32] = dv[c].re;
                mine[(2 * c + 1) * 32] = dv[c].im;
            }
            __syncthreads();
            const R* all = part + (w & ~1) * 6 * 32 + lane;     // both spins of this chirality and flavour
            const R* other = part + (w ^ 4) * 6 * 32 + lane;    // the partner flavour's same rows
            const R ts = ((f == 0) == (cb == 0)) ? (R)-pr.tw : (R)pr.tw;
            const R eps = (R)pr.eps;
#pragma unroll
            for (int c = 0; c < 3; ++c) {
                out[c] = dv[c] + ts * mul_i(dv[c]) + eps * C(other[2 * c * 32], other[(2 * c + 1) * 32]);
#pragma unroll
                for (int j = 0; j < 6; ++j) cfma(out[c], m[c][j], C(all[2 * j * 32], all[(2 * j + 1) * 32]));
            }
        }
    } else {
        // out = g5 [ (A + i tw g5 [tau3]) psi - eps tau1 psi - kappa^2 acc ] + i rho psi
        if (valid) {
            R sc = (R)1;
            if constexpr (P == PF16 || P == PB16)
                sc = reinterpret_cast<const float*>(reinterpret_cast<const char*>(pr.loc) + (size_t)vh * NF * 12 * 4)[i];
#pragma unroll
            for (int j = 0; j < 6; ++j) v[j] = sc * load_complex<P, false>(pr.loc, vh, i, 12 * f + 6 * cb + j);
            const R g5 = cb == 0 ? (R)1 : (R)-1, t3 = f == 0 ? (R)1 : (R)-1;
            const R tw = g5 * ((R)pr.tw * t3 + (R)pr.rho), k2 = (R)(pr.kappa * pr.kappa);
#pragma unroll
            for (int c = 0; c < 3; ++c) {
                const cpx<R> p = h == 0 ? v[c] : v[3 + c];
                cpx<R> s = tw * mul_i(p);
                if constexpr (NF == 2)
                    s = s - (R)pr.eps * (sc * load_complex<P, false>(pr.loc, vh, i, 12 * (1 - f) + 6 * cb + 3 * h + c));
                s = s - k2 * hops(6 * cb + 3 * h + c);
#pragma unroll
                for (int j = 0; j < 6; ++j) cfma(s, m[c][j], v[j]);
                out[c] = g5 * s;
            }
            if constexpr (KIND == K2_UPDATE) {   // residual_update of dslash.cu
                const R alpha = (R)pr.ctl->alpha, shift = (R)pr.ctl->shift;
                R rs = (R)1, ps = (R)1;
                if constexpr (P == PF16 || P == PB16) {
                    const size_t off = (size_t)vh * NF * 12 * 4;
                    rs = reinterpret_cast<const float*>(reinterpret_cast<const char*>(pr.r) + off)[i];
                    ps = reinterpret_cast<const float*>(reinterpret_cast<const char*>(pr.p) + off)[i];
                }
                const int e = 12 * f + 6 * cb + 3 * h;
#pragma unroll
                for (int c = 0; c < 3; ++c) {
                    if (shift != (R)0) out[c] = out[c] + shift * (ps * load_complex<P, false>(pr.p, vh, i, e + c));
                    out[c] = rs * load_complex<P, false>(pr.r, vh, i, e + c) - alpha * out[c];
                }
            }
        }
    }
    const int e0 = 12 * f + 6 * cb + 3 * h;
    if constexpr (P == PF16 || P == PB16) {
        // one scale per site: the maximum over its warps
        float a = 0.f;
        if (valid) {
#pragma unroll
            for (int c = 0; c < 3; ++c) a = fmaxf(a, fmaxf(fabsf(out[c].re), fabsf(out[c].im)));
        }
        site_max[w][lane] = a;
        __syncthreads();
#pragma unroll
        for (int k = 0; k < NW; ++k) a = fmaxf(a, site_max[k][lane]);
        const float inv = a > 0.f ? 1.f / a : 0.f;
        if (valid) {
#pragma unroll
            for (int c = 0; c < 3; ++c) store_complex<P>(pr.out, vh, i, e0 + c, inv * out[c]);
            if (w == 0) reinterpret_cast<float*>(reinterpret_cast<char*>(pr.out) + (size_t)vh * NF * 12 * 4)[i] = a;
        }
    } else if (valid) {
#pragma unroll
        for (int c = 0; c < 3; ++c) store_complex<P>(pr.out, vh, i, e0 + c, out[c]);
    }
    if constexpr (KIND != K1_EO_INV) {
        if (KIND == K2_UPDATE || pr.partial != nullptr) {
            R s = (R)0;
            if (valid) {
#pragma unroll
                for (int c = 0; c < 3; ++c) s += norm2(out[c]);
            }
            const double bs = block_sum<BS>((double)s, sh);
            reduce_finalize<BS>(pr.partial, pr.counter, pr.nblk, blockIdx.x, bs, b.fin, pr.ctl, pr.ms, nullptr, sh);
        }
    }
}

template <int P, int NF, int KIND>
cudaError_t launch_dslash_split(const OpBatch<1>& b, int nblocks, cudaStream_t st) {
    constexpr size_t bytes = split_smem<P, NF>();
    if constexpr (bytes + 4096 > 48 * 1024) {
        const cudaError_t e = cudaFuncSetAttribute(dslash_split_kernel<P, NF, KIND>,
                                                   cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
        if (e != cudaSuccess) return e;
    }
    return launch_chained(dslash_split_kernel<P, NF, KIND>, nblocks, 128 * NF, bytes, st, b.chained, b);
}

#define TM_SPLIT_INST(P, NF)                                                                          \
    template cudaError_t launch_dslash_split<P, NF, K1_EO_INV>(const OpBatch<1>&, int, cudaStream_t); \
    template cudaError_t launch_dslash_split<P, NF, K2_OE_LOCAL>(const OpBatch<1>&, int, cudaStream_t); \
    template cudaError_t launch_dslash_split<P, NF, K2_UPDATE>(const OpBatch<1>&, int, cudaStream_t);
#define TM_SPLIT_P(P) TM_SPLIT_INST(P, 1) TM_SPLIT_INST(P, 2)
TM_SPLIT_P(P64)
TM_SPLIT_P(P32)
TM_SPLIT_P(PB16)
TM_SPLIT_P(PF16)

}  // namespace tmk
