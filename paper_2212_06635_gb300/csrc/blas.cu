// BLAS-1 steps of CG / multishift CG (Sec. 4) with fused FP64 reductions, and
// precision conversions between native fields.  One thread per site; each
// thread moves a whole spinor with 16-byte vector accesses.  Reductions: per
// thread in the arithmetic precision, then FP64 warp shuffles, one partial per
// block, and a fixed-order sum by the last block (deterministic).
#include "tm_internal.h"
#include "tm_kernels.h"

namespace tmk {

#define TM_VEC_PROLOGUE(NP)                                 \
    __shared__ double sh[BLAS_BS / 32];                     \
    const int k = find_vproblem<NP>(b, blockIdx.x);         \
    const VecProb& pr = b.p[k];                             \
    const int lb = blockIdx.x - b.blk_start[k];             \
    const long i = (long)lb * BLAS_BS + threadIdx.x;        \
    const bool valid = i < pr.vh;                           \
    (void)sh; (void)valid;

// p = r + beta p
template <int P, int NC, int NP>
__global__ void __launch_bounds__(BLAS_BS) k_cg_pupdate(const __grid_constant__ VecBatch<NP> b) {
    using R = typename PT<P>::R;
    TM_VEC_PROLOGUE(NP)
    if (pr.ctl->flag != CTL_RUN) return;
    const R beta = (R)pr.ctl->beta;
    const bool want = pr.ctl->shift != 0.0;
    double s = 0.0;
    if (valid) {
        cpx<R> p[NC], r[NC];
        load_spinor<P, NC>(pr.v[1], pr.vh, i, r);
        if (beta != (R)0) {
            load_spinor<P, NC>(pr.v[0], pr.vh, i, p);
#pragma unroll
            for (int q = 0; q < NC; ++q) p[q] = r[q] + beta * p[q];
        } else {
#pragma unroll
            for (int q = 0; q < NC; ++q) p[q] = r[q];
        }
        store_spinor<P, NC>(pr.v[0], pr.vh, i, p);
        if (want) {
            R t = (R)0;
#pragma unroll
            for (int q = 0; q < NC; ++q) t += norm2(p[q]);
            s = (double)t;
        }
    }
    if (want) {
        const double bs = block_sum<BLAS_BS>(s, sh);
        reduce_finalize<BLAS_BS>(pr.partial, pr.counter, pr.nblk, lb, bs, FIN_PP, pr.ctl, pr.ms,
                                 nullptr, sh);
    }
}

// x += alpha p;  r -= alpha (Ap + shift p);  ||r||^2
template <int P, int PX, int NC, int NP>
__global__ void __launch_bounds__(BLAS_BS) k_cg_update(const __grid_constant__ VecBatch<NP> b) {
    using R = typename PT<P>::R;
    using RX = typename PT<PX>::R;
    TM_VEC_PROLOGUE(NP)
    if (pr.ctl->flag != CTL_RUN) return;
    const R alpha = (R)pr.ctl->alpha;
    const R sh_ = (R)pr.ctl->shift;
    double s = 0.0;
    if (valid) {
        R t = (R)0;
        // x and r are updated in place, so a step's loads cannot sink below its stores: a
        // few vectors at a time.  All loads of a site first took 114 (FP16) and 252 (FP64)
        // registers; uneven batch of 24, FP16 348.6 -> 343.5 ms, FP32 427.8 -> 421.8, FP64
        // 3823 -> 3790 (a launch in FP32 196 -> 169 us; G = 1, 2, 3 measure the same).
        constexpr int W = PT<PX>::W, NV = 2 * NC / W, G = 2;
        if constexpr (P == PB16 || P == PF16) {   // (the new scale of r needs the whole site)
            cpx<R> p[NC], r[NC], ap[NC];
            load_spinor<P, NC, true>(pr.v[1], pr.vh, i, p);
            const R* pv = reinterpret_cast<const R*>(p);
#pragma unroll
            for (int v = 0; v < NV; v += 3) {
                RX x[3 * W];
#pragma unroll
                for (int g = 0; g < 3; ++g) load_reals<PX, W>(pr.v[0], pr.vh, i, W * (v + g), x + W * g);
#pragma unroll
                for (int k = 0; k < 3 * W; ++k) x[k] += (RX)(alpha * pv[W * v + k]);
#pragma unroll
                for (int g = 0; g < 3; ++g) store_reals<PX, W>(pr.v[0], pr.vh, i, W * (v + g), x + W * g);
            }
            load_spinor<P, NC>(pr.v[2], pr.vh, i, r);
            load_spinor<P, NC, true>(pr.v[3], pr.vh, i, ap);
#pragma unroll
            for (int q = 0; q < NC; ++q) {
                cpx<R> a = ap[q];
                if (sh_ != (R)0) a = a + sh_ * p[q];
                r[q] = r[q] - alpha * a;
                t += norm2(r[q]);
            }
            store_spinor<P, NC>(pr.v[2], pr.vh, i, r);
        } else {
#pragma unroll
            for (int v = 0; v < NV; v += G) {
                R p[G * W], r[G * W], ap[G * W];
                RX x[G * W];
#pragma unroll
                for (int g = 0; g < G; ++g) {
                    load_readonly<P, W>(pr.v[1], pr.vh, i, W * (v + g), p + W * g);
                    load_readonly<P, W>(pr.v[3], pr.vh, i, W * (v + g), ap + W * g);
                    load_reals<P, W>(pr.v[2], pr.vh, i, W * (v + g), r + W * g);
                    load_reals<PX, W>(pr.v[0], pr.vh, i, W * (v + g), x + W * g);
                }
#pragma unroll
                for (int k = 0; k < G * W; ++k) {
                    x[k] += (RX)(alpha * p[k]);
                    if (sh_ != (R)0) ap[k] += sh_ * p[k];
                    r[k] -= alpha * ap[k];
                }
#pragma unroll
                for (int k = 0; k < G * W; k += 2) t += norm2(C(r[k], r[k + 1]));
#pragma unroll
                for (int g = 0; g < G; ++g) {
                    store_reals<PX, W>(pr.v[0], pr.vh, i, W * (v + g), x + W * g);
                    store_reals<P, W>(pr.v[2], pr.vh, i, W * (v + g), r + W * g);
                }
            }
        }
        s = (double)t;
    }
    const double bs = block_sum<BLAS_BS>(s, sh);
    reduce_finalize<BLAS_BS>(pr.partial, pr.counter, pr.nblk, lb, bs, FIN_CG_UPDATE, pr.ctl, pr.ms,
                             nullptr, sh);
}

template <int PD, int PS, int NC, int NP>
__global__ void __launch_bounds__(BLAS_BS) k_convert(const __grid_constant__ VecBatch<NP> b) {
    using RD = typename PT<PD>::R;
    using RS = typename PT<PS>::R;
    TM_VEC_PROLOGUE(NP)
    if (!valid) return;
    cpx<RS> s[NC];
    cpx<RD> d[NC];
    load_spinor<PS, NC, true>(pr.v[1], pr.vh, i, s);
#pragma unroll
    for (int q = 0; q < NC; ++q) d[q] = C((RD)s[q].re, (RD)s[q].im);
    store_spinor<PD, NC>(pr.v[0], pr.vh, i, d);
}

template <int PS, int NC, int NP>
__global__ void __launch_bounds__(BLAS_BS) k_add_to64(const __grid_constant__ VecBatch<NP> b) {
    using RS = typename PT<PS>::R;
    TM_VEC_PROLOGUE(NP)
    if (!valid) return;
    cpx<RS> x[NC];
    cpx<double> y[NC];
    load_spinor<PS, NC, true>(pr.v[1], pr.vh, i, x);
    load_spinor<P64, NC>(pr.v[0], pr.vh, i, y);
#pragma unroll
    for (int q = 0; q < NC; ++q) y[q] = y[q] + C((double)x[q].re, (double)x[q].im);
    store_spinor<P64, NC>(pr.v[0], pr.vh, i, y);
}

// r = b - Ax - shift x (FP64), ||r||^2 -> *dst
template <int NC, int NP>
__global__ void __launch_bounds__(BLAS_BS) k_residual64(const __grid_constant__ VecBatch<NP> b) {
    TM_VEC_PROLOGUE(NP)
    const double shv = pr.ctl ? pr.ctl->shift : 0.0;
    double s = 0.0;
    if (valid) {
        cpx<double> r[NC], bb[NC], ax[NC], x[NC];
        load_spinor<P64, NC, true>(pr.v[1], pr.vh, i, bb);
        load_spinor<P64, NC, true>(pr.v[2], pr.vh, i, ax);
        if (shv != 0.0) load_spinor<P64, NC, true>(pr.v[3], pr.vh, i, x);
#pragma unroll
        for (int q = 0; q < NC; ++q) {
            r[q] = bb[q] - ax[q];
            if (shv != 0.0) r[q] = r[q] - shv * x[q];
            s += norm2(r[q]);
        }
        store_spinor<P64, NC>(pr.v[0], pr.vh, i, r);
    }
    const double bs = block_sum<BLAS_BS>(s, sh);
    reduce_finalize<BLAS_BS>(pr.partial, pr.counter, pr.nblk, lb, bs, FIN_STORE, pr.ctl, pr.ms,
                             pr.dst, sh);
}

template <int P, int NC, int NP>
__global__ void __launch_bounds__(BLAS_BS) k_norm2(const __grid_constant__ VecBatch<NP> b) {
    using R = typename PT<P>::R;
    TM_VEC_PROLOGUE(NP)
    double s = 0.0;
    if (valid) {
        cpx<R> v[NC];
        load_spinor<P, NC, true>(pr.v[0], pr.vh, i, v);
        if constexpr (P == P64) {
#pragma unroll
            for (int q = 0; q < NC; ++q) s += norm2(v[q]);
        } else {
            R t = (R)0;
#pragma unroll
            for (int q = 0; q < NC; ++q) t += norm2(v[q]);
            s = (double)t;
        }
    }
    const double bs = block_sum<BLAS_BS>(s, sh);
    reduce_finalize<BLAS_BS>(pr.partial, pr.counter, pr.nblk, lb, bs, FIN_STORE, pr.ctl, pr.ms,
                             pr.dst, sh);
}

template <int NC>
__global__ void __launch_bounds__(BLAS_BS) k_normalize64(const __grid_constant__ VecBatch<1> b) {
    TM_VEC_PROLOGUE(1)
    if (!valid) return;
    const double sc = 1.0 / sqrt(*pr.dst);
    cpx<double> v[NC];
    load_spinor<P64, NC>(pr.v[0], pr.vh, i, v);
#pragma unroll
    for (int q = 0; q < NC; ++q) v[q] = sc * v[q];
    store_spinor<P64, NC>(pr.v[0], pr.vh, i, v);
}

// ---------------------------------------------------------------------------
// CG with the residual update in the operator's last pass (K2_UPDATE).  The solution
// is touched once per RING iterations: x += sum alpha_i p_i from a ring of search
// directions, so an iteration moves (p, r -> p) here, r once more in the odd pass and
// a quarter of (RING p, x -> x).  Light FP16: 298 B a site instead of 542 with
// x, p, r, A p passing through an update kernel every iteration; two-flavour FP32
// with a shift 1248 instead of 1920 B.
// ---------------------------------------------------------------------------
// p_out = r + beta p_in
template <int P, int NC, int NP>
__global__ void __launch_bounds__(BLAS_BS) k_cg_direction(const __grid_constant__ VecBatch<NP> b) {
    using R = typename PT<P>::R;
    pdl_wait();
    TM_VEC_PROLOGUE(NP)
    if (pr.ctl->flag != CTL_RUN) return;
    const R beta = (R)pr.ctl->beta;
    const bool want = pr.ctl->shift != 0.0;
    double s = 0.0;
    if (valid) {
        cpx<R> p[NC], r[NC];
        load_spinor<P, NC>(pr.v[1], pr.vh, i, r);
        if (beta != (R)0) {
            load_spinor<P, NC>(pr.v[2], pr.vh, i, p);
#pragma unroll
            for (int q = 0; q < NC; ++q) p[q] = r[q] + beta * p[q];
        } else {
#pragma unroll
            for (int q = 0; q < NC; ++q) p[q] = r[q];
        }
        store_spinor<P, NC>(pr.v[0], pr.vh, i, p);
        if (want) {
            R t = (R)0;
#pragma unroll
            for (int q = 0; q < NC; ++q) t += norm2(p[q]);
            s = (double)t;
        }
    }
    if (want) {
        const double bs = block_sum<BLAS_BS>(s, sh);
        reduce_finalize<BLAS_BS>(pr.partial, pr.counter, pr.nblk, lb, bs, FIN_PP, pr.ctl, pr.ms,
                                 nullptr, sh);
    }
}

// x += sum_{i < n} alpha_i p_i, a vector of reals at a time (one thread per site and vector)
template <int P, int PX, int NC, int NP>
__global__ void __launch_bounds__(BLAS_BS) k_cg_xupdate(const __grid_constant__ VecBatch<NP> b, int n, bool always) {
    using R = typename PT<P>::R;
    using RX = typename PT<PX>::R;
    constexpr int W = PT<P>::W;
    pdl_wait();
    const VecProb& pr = b.p[blockIdx.z];
    if (!always && pr.ctl->flag != CTL_RUN) return;
    const long vh = pr.vh, i = (long)blockIdx.x * BLAS_BS + threadIdx.x;
    if (i >= vh) return;
    R alpha[RING];
#pragma unroll
    for (int k = 0; k < RING; ++k) {
        alpha[k] = k < n ? (R)pr.ctl->alpha_ring[k] : (R)0;
        if constexpr (P == PB16 || P == PF16)
            if (k < n) alpha[k] *= reinterpret_cast<const float*>(reinterpret_cast<const char*>(pr.v[2 + k]) + (size_t)vh * NC * 4)[i];
    }
    const int v = blockIdx.y;
    RX x[W];
    load_reals<PX, W>(pr.v[0], vh, i, W * v, x);
#pragma unroll
    for (int k = 0; k < RING; ++k) {
        if (k < n) {
            R p[W];
            load_readonly<P, W>(pr.v[2 + k], vh, i, W * v, p);
#pragma unroll
            for (int e = 0; e < W; ++e) x[e] += (RX)(alpha[k] * p[e]);
        }
    }
    store_reals<PX, W>(pr.v[0], vh, i, W * v, x);
}

// Multishift CG (Sec. 4.2): n iterations of every shift at once.  p_k and x_k pass
// through memory once per RING iterations instead of every one (12 shifts,
// two-flavour FP32: 9.2 KB -> 2.5 KB a site and iteration).  One thread per site and
// vector of reals, with the residuals in registers; 16-bit fields need the maximum
// over a site for p_k's scale, so there one thread per site reads the residuals (from
// L2) for each shift.
template <int P, int PX, int NC>
__global__ void __launch_bounds__(BLAS_BS) k_ms_block(const __grid_constant__ VecBatch<1> b,
                                                      const __grid_constant__ MsVecs mv, int n, bool always) {
    using R = typename PT<P>::R;
    using RX = typename PT<PX>::R;
    constexpr bool H = P == PB16 || P == PF16;
    constexpr int W = H ? 2 * NC : PT<P>::W;   // reals a thread holds
    pdl_wait();
    const VecProb& pr = b.p[0];
    if (!always && pr.ctl->flag != CTL_RUN) return;
    // the coefficients once per block in the vectors' precision: converted from FP64 by
    // every thread they took longer than the vectors' traffic (12 shifts at 24^3x48, mean
    // over a solve: 676 -> 286 us a launch)
    const MsCtl* ms = pr.ms;
    const int ns = ms->nshift;
    __shared__ R coef[MAX_SHIFTS][RING][3];
    __shared__ int live[MAX_SHIFTS], nlive;
    for (int e = threadIdx.x; e < ns * RING; e += BLAS_BS) {
        const int k = e / RING, q = e % RING;
        coef[k][q][0] = q < n ? (R)ms->alpha_ring[q][k] : (R)0;
        coef[k][q][1] = q < n ? (R)ms->zeta_ring[q][k] : (R)0;
        coef[k][q][2] = q < n ? (R)ms->beta_ring[q][k] : (R)0;
    }
    if (threadIdx.x == 0) {
        int m = 0;
        for (int k = 0; k < ns; ++k) {
            bool any = false;   // else frozen before this block of iterations
            for (int q = 0; q < n; ++q) any = any || ms->alpha_ring[q][k] != 0.0;
            if (any) live[m++] = k;
        }
        nlive = m;
    }
    __syncthreads();
    const long vh = pr.vh, i = (long)blockIdx.x * BLAS_BS + threadIdx.x;
    if (i >= vh) return;
    const int off = H ? 0 : W * blockIdx.y;
    R r[H ? 1 : RING][W];
    if constexpr (!H) {
#pragma unroll
        for (int q = 0; q < RING; ++q)
            if (q < n) load_readonly<P, W>(pr.v[2 + q], vh, i, off, r[q]);
    }
    // shifts a thread has in flight: all loads of a step before its stores
    constexpr int G = H ? 1 : 2;
    const int nl = nlive;
#pragma unroll 1
    for (int l = 0; l < nl; l += G) {
        R p[G][W];
        RX x[G][W];
#pragma unroll
        for (int g = 0; g < G; ++g) {
            if (l + g >= nl) continue;
            const int k = live[l + g];
            if constexpr (H) load_spinor<P, NC>(mv.p[k], vh, i, reinterpret_cast<cpx<R>*>(p[g]));
            else load_reals<P, W>(mv.p[k], vh, i, off, p[g]);
            load_reals<PX, W>(mv.x[k], vh, i, off, x[g]);
        }
#pragma unroll
        for (int g = 0; g < G; ++g) {
            if (l + g >= nl) continue;
            const int k = live[l + g];
#pragma unroll
            for (int q = 0; q < RING; ++q) {
                if (q < n) {
                    const R a = coef[k][q][0], z = coef[k][q][1], bt = coef[k][q][2];
                    if constexpr (H) load_spinor<P, NC, true>(pr.v[2 + q], vh, i, reinterpret_cast<cpx<R>*>(r[0]));
                    const R* rq = r[H ? 0 : q];
#pragma unroll
                    for (int e = 0; e < W; ++e) {
                        x[g][e] += (RX)(a * p[g][e]);
                        p[g][e] = z * rq[e] + bt * p[g][e];
                    }
                }
            }
            store_reals<PX, W>(mv.x[k], vh, i, off, x[g]);
            if constexpr (H) store_spinor<P, NC>(mv.p[k], vh, i, reinterpret_cast<const cpx<R>*>(p[g]));
            else store_reals<P, W>(mv.p[k], vh, i, off, p[g]);
        }
    }
}

// ---------------------------------------------------------------------------
// canonical FP64 AoS <-> native
// ---------------------------------------------------------------------------
template <int P, int NC>
__global__ void __launch_bounds__(BLAS_BS) k_import(void* dst, const double* __restrict__ src, long vh) {
    using R = typename PT<P>::R;
    const long i = (long)blockIdx.x * BLAS_BS + threadIdx.x;
    if (i >= vh) return;
    cpx<R> s[NC];
    const double2* p = reinterpret_cast<const double2*>(src) + i * NC;
#pragma unroll
    for (int q = 0; q < NC; ++q) {
        const double2 v = p[q];
        s[q] = C((R)v.x, (R)v.y);
    }
    store_spinor<P, NC>(dst, vh, i, s);
}

template <int P, int NC>
__global__ void __launch_bounds__(BLAS_BS) k_export(double* dst, const void* src, long vh) {
    using R = typename PT<P>::R;
    const long i = (long)blockIdx.x * BLAS_BS + threadIdx.x;
    if (i >= vh) return;
    cpx<R> s[NC];
    load_spinor<P, NC, true>(src, vh, i, s);
    double2* p = reinterpret_cast<double2*>(dst) + i * NC;
#pragma unroll
    for (int q = 0; q < NC; ++q) p[q] = make_double2((double)s[q].re, (double)s[q].im);
}

// ---------------------------------------------------------------------------
// launchers
// ---------------------------------------------------------------------------
template <int P, int NC, int NP>
cudaError_t launch_cg_pupdate(const VecBatch<NP>& b, int nb, cudaStream_t st) {
    k_cg_pupdate<P, NC, NP><<<nb, BLAS_BS, 0, st>>>(b);
    return cudaGetLastError();
}
template <int P, int PX, int NC, int NP>
cudaError_t launch_cg_update(const VecBatch<NP>& b, int nb, cudaStream_t st) {
    k_cg_update<P, PX, NC, NP><<<nb, BLAS_BS, 0, st>>>(b);
    return cudaGetLastError();
}
template <int PD, int PS, int NC, int NP>
cudaError_t launch_convert(const VecBatch<NP>& b, int nb, cudaStream_t st) {
    k_convert<PD, PS, NC, NP><<<nb, BLAS_BS, 0, st>>>(b);
    return cudaGetLastError();
}
template <int PS, int NC, int NP>
cudaError_t launch_add_to64(const VecBatch<NP>& b, int nb, cudaStream_t st) {
    k_add_to64<PS, NC, NP><<<nb, BLAS_BS, 0, st>>>(b);
    return cudaGetLastError();
}
template <int NC, int NP>
cudaError_t launch_residual64(const VecBatch<NP>& b, int nb, cudaStream_t st) {
    k_residual64<NC, NP><<<nb, BLAS_BS, 0, st>>>(b);
    return cudaGetLastError();
}
template <int P, int NC, int NP>
cudaError_t launch_norm2(const VecBatch<NP>& b, int nb, cudaStream_t st) {
    k_norm2<P, NC, NP><<<nb, BLAS_BS, 0, st>>>(b);
    return cudaGetLastError();
}
template <int NC>
cudaError_t launch_normalize64(const VecBatch<1>& b, int nb, cudaStream_t st) {
    k_normalize64<NC><<<nb, BLAS_BS, 0, st>>>(b);
    return cudaGetLastError();
}
template <int P, int NC, int NP>
cudaError_t launch_cg_direction(const VecBatch<NP>& b, int nb, cudaStream_t st) {
    return launch_chained(k_cg_direction<P, NC, NP>, nb, BLAS_BS, 0, st, true, b);
}
template <int P, int PX, int NC, int NP>
cudaError_t launch_cg_xupdate(const VecBatch<NP>& b, int n, bool always, int nb, cudaStream_t st) {
    k_cg_xupdate<P, PX, NC, NP><<<dim3(nb, 2 * NC / PT<P>::W, b.n), BLAS_BS, 0, st>>>(b, n, always);
    return cudaGetLastError();
}
template <int P, int PX, int NC>
cudaError_t launch_ms_block(const VecBatch<1>& b, const MsVecs& mv, int n, bool always, int nb, cudaStream_t st) {
    const int ny = P == PB16 || P == PF16 ? 1 : 2 * NC / PT<P>::W;
    k_ms_block<P, PX, NC><<<dim3(nb, ny), BLAS_BS, 0, st>>>(b, mv, n, always);
    return cudaGetLastError();
}
template <int P, int NC>
cudaError_t launch_import(void* dst, const double* src, long vh, cudaStream_t st) {
    k_import<P, NC><<<(unsigned)((vh + BLAS_BS - 1) / BLAS_BS), BLAS_BS, 0, st>>>(dst, src, vh);
    return cudaGetLastError();
}
template <int P, int NC>
cudaError_t launch_export(double* dst, const void* src, long vh, cudaStream_t st) {
    k_export<P, NC><<<(unsigned)((vh + BLAS_BS - 1) / BLAS_BS), BLAS_BS, 0, st>>>(dst, src, vh);
    return cudaGetLastError();
}

// explicit instantiations
#define TM_PX(P) ((P) == P64 ? P64 : P32)
#define TM_BLAS_P_NC(P, NC)                                                                              \
    template cudaError_t launch_cg_direction<P, NC, 1>(const VecBatch<1>&, int, cudaStream_t);            \
    template cudaError_t launch_cg_xupdate<P, TM_PX(P), NC, 1>(const VecBatch<1>&, int, bool, int, cudaStream_t); \
    template cudaError_t launch_ms_block<P, TM_PX(P), NC>(const VecBatch<1>&, const MsVecs&, int, bool, int, cudaStream_t); \
    template cudaError_t launch_add_to64<P, NC, 1>(const VecBatch<1>&, int, cudaStream_t);               \
    template cudaError_t launch_norm2<P, NC, 1>(const VecBatch<1>&, int, cudaStream_t);                  \
    template cudaError_t launch_import<P, NC>(void*, const double*, long, cudaStream_t);                  \
    template cudaError_t launch_export<P, NC>(double*, const void*, long, cudaStream_t);
#define TM_BLAS_P(P)                                                                                     \
    TM_BLAS_P_NC(P, 12) TM_BLAS_P_NC(P, 24)                                                              \
    template cudaError_t launch_cg_pupdate<P, 12, MAXP>(const VecBatch<MAXP>&, int, cudaStream_t);        \
    template cudaError_t launch_cg_update<P, TM_PX(P), 12, MAXP>(const VecBatch<MAXP>&, int, cudaStream_t);

TM_BLAS_P(P64)
TM_BLAS_P(P32)
TM_BLAS_P(PB16)
TM_BLAS_P(PF16)
#define TM_GROUP(P, NC)                                                                                 \
    template cudaError_t launch_cg_direction<P, NC, GROUP>(const VecBatch<GROUP>&, int, cudaStream_t);   \
    template cudaError_t launch_cg_xupdate<P, P32, NC, GROUP>(const VecBatch<GROUP>&, int, bool, int, cudaStream_t);
TM_GROUP(P32, 12) TM_GROUP(P32, 24)
TM_GROUP(PB16, 12) TM_GROUP(PB16, 24)
TM_GROUP(PF16, 12) TM_GROUP(PF16, 24)
#define TM_CONV2(P, NC, NP)                                                                 \
    template cudaError_t launch_convert<P, P64, NC, NP>(const VecBatch<NP>&, int, cudaStream_t); \
    template cudaError_t launch_convert<P64, P, NC, NP>(const VecBatch<NP>&, int, cudaStream_t);
#define TM_CONV_P(P) TM_CONV2(P, 12, 1) TM_CONV2(P, 24, 1) TM_CONV2(P, 12, MAXP)
TM_CONV_P(P32)
TM_CONV_P(PB16)
TM_CONV_P(PF16)
template cudaError_t launch_convert<P64, P64, 12, 1>(const VecBatch<1>&, int, cudaStream_t);
template cudaError_t launch_convert<P64, P64, 24, 1>(const VecBatch<1>&, int, cudaStream_t);
template cudaError_t launch_convert<P64, P64, 12, MAXP>(const VecBatch<MAXP>&, int, cudaStream_t);
template cudaError_t launch_residual64<12, 1>(const VecBatch<1>&, int, cudaStream_t);
template cudaError_t launch_residual64<24, 1>(const VecBatch<1>&, int, cudaStream_t);
template cudaError_t launch_residual64<12, MAXP>(const VecBatch<MAXP>&, int, cudaStream_t);
template cudaError_t launch_normalize64<12>(const VecBatch<1>&, int, cudaStream_t);
template cudaError_t launch_normalize64<24>(const VecBatch<1>&, int, cudaStream_t);

}  // namespace tmk

// ---------------------------------------------------------------------------
// complex BLAS-1 for flexible CG (FP32 native light fields)
// ---------------------------------------------------------------------------
namespace tmk {

// <a, b> = sum conj(a) b -> dst2[0] (re), dst2[1] (im); deterministic two-level sum
__global__ void __launch_bounds__(BLAS_BS) k_cdot32(const void* a, const void* b, long vh, double* partial,
                                                    unsigned int* counter, double* dst2) {
    __shared__ double sh[BLAS_BS / 32];
    __shared__ int am_last;
    const long i = (long)blockIdx.x * BLAS_BS + threadIdx.x;
    double re = 0.0, im = 0.0;
    if (i < vh) {
        cpx<float> x[12], y[12];
        load_spinor<P32, 12>(a, vh, i, x);
        load_spinor<P32, 12>(b, vh, i, y);
        float r = 0.f, m = 0.f;
#pragma unroll
        for (int q = 0; q < 12; ++q) {
            r += x[q].re * y[q].re + x[q].im * y[q].im;
            m += x[q].re * y[q].im - x[q].im * y[q].re;
        }
        re = r;
        im = m;
    }
    re = block_sum<BLAS_BS>(re, sh);
    im = block_sum<BLAS_BS>(im, sh);
    const int nb = gridDim.x;
    if (threadIdx.x == 0) {
        partial[2 * blockIdx.x] = re;
        partial[2 * blockIdx.x + 1] = im;
        __threadfence();
        am_last = atomicAdd(counter, 1u) == (unsigned)(nb - 1);
    }
    __syncthreads();
    if (!am_last) return;
    __threadfence();
    double tr = 0.0, ti = 0.0;
    for (int k = threadIdx.x; k < nb; k += BLAS_BS) {
        tr += ((volatile double*)partial)[2 * k];
        ti += ((volatile double*)partial)[2 * k + 1];
    }
    tr = block_sum<BLAS_BS>(tr, sh);
    ti = block_sum<BLAS_BS>(ti, sh);
    if (threadIdx.x == 0) {
        *counter = 0u;
        dst2[0] = tr;
        dst2[1] = ti;
    }
}

// y += (ar + i ai) x
__global__ void __launch_bounds__(BLAS_BS) k_caxpy32(void* y, const void* x, float ar, float ai, long vh) {
    const long i = (long)blockIdx.x * BLAS_BS + threadIdx.x;
    if (i >= vh) return;
    cpx<float> a[12], b[12];
    load_spinor<P32, 12>(y, vh, i, a);
    load_spinor<P32, 12>(x, vh, i, b);
    const cpx<float> s = C(ar, ai);
#pragma unroll
    for (int q = 0; q < 12; ++q) cfma(a[q], s, b[q]);
    store_spinor<P32, 12>(y, vh, i, a);
}

// y = x + (br + i bi) y
__global__ void __launch_bounds__(BLAS_BS) k_cxpay32(void* y, const void* x, float br, float bi, long vh) {
    const long i = (long)blockIdx.x * BLAS_BS + threadIdx.x;
    if (i >= vh) return;
    cpx<float> a[12], b[12];
    load_spinor<P32, 12>(y, vh, i, a);
    load_spinor<P32, 12>(x, vh, i, b);
    const cpx<float> s = C(br, bi);
#pragma unroll
    for (int q = 0; q < 12; ++q) a[q] = b[q] + s * a[q];
    store_spinor<P32, 12>(y, vh, i, a);
}

cudaError_t launch_cdot32(const void* a, const void* b, long vh, double* partial, unsigned int* counter,
                          double* dst2, cudaStream_t st) {
    k_cdot32<<<(unsigned)((vh + BLAS_BS - 1) / BLAS_BS), BLAS_BS, 0, st>>>(a, b, vh, partial, counter, dst2);
    return cudaGetLastError();
}
cudaError_t launch_caxpy32(void* y, const void* x, double ar, double ai, long vh, cudaStream_t st) {
    k_caxpy32<<<(unsigned)((vh + BLAS_BS - 1) / BLAS_BS), BLAS_BS, 0, st>>>(y, x, (float)ar, (float)ai, vh);
    return cudaGetLastError();
}
cudaError_t launch_cxpay32(void* y, const void* x, double br, double bi, long vh, cudaStream_t st) {
    k_cxpay32<<<(unsigned)((vh + BLAS_BS - 1) / BLAS_BS), BLAS_BS, 0, st>>>(y, x, (float)br, (float)bi, vh);
    return cudaGetLastError();
}

}  // namespace tmk
