// Kernel-side helpers shared by the translation units (deterministic block/grid
// reductions, solver-scalar finalisers) and the host-visible launcher
// declarations.
#pragma once

#include "tm_internal.h"

namespace tmk {

constexpr int DSLASH_BS = 128;   // direct stencil kernel
// FP64 passes take half-size blocks: their work is even, so the last wave is what
// differs (both light passes at 128 / 64 threads: 16^3x32 320 / 300 us, 24^3x48 1379 /
// 1378 us; both two-flavour ones at 12^3x24 266 / 236 us)
constexpr int dslash_bs(int P) { return P == P64 ? 64 : DSLASH_BS; }
constexpr int STAGED_BS = 64;    // shared-memory staged stencil kernel
constexpr int BLAS_BS = 256;
constexpr int SPLIT_SITES = 32;  // sites per block of the small-lattice stencil kernel
constexpr int MIN_BS = 32;       // fewest sites per block of any reducing kernel (sizes the partials)

// K2_UPDATE: the odd pass of the second factor of a normal operator with the residual
// update in its epilogue, r_out = r - alpha (out + shift p), ||r_out||^2
// K2_OUT64 (double-word passes): K2_OE_LOCAL with the result stored as FP64
enum DslashKind { K1_EO_INV = 0, K2_OE_LOCAL = 1, K2_UPDATE = 2, K2_OUT64 = 3 };

// FinOp codes beyond those in tm_internal.h
enum { FIN_PP = 4, FIN_CG_UPDATE = 5, FIN_MS_UPDATE = 6 };

// ---------------------------------------------------------------------------
// Chained launches (programmatic dependent launch).  A kernel launched with
// `chained` may start while the kernel before it in the stream still runs: until
// pdl_wait() it reads only data that no kernel of the chain writes (links, clover
// blocks); pdl_wait() returns when the kernel before has completed and its writes are
// visible.  The first kernel of a chain is launched without it, so everything
// before the chain has completed by then.  Only the small-lattice kernel lets the
// next one start early (pdl_trigger): on larger grids blocks of the next kernel then
// sit between the last ones of this, and its own blocks end up unevenly spread (heavy
// FP64 at 12^3x24: 484 -> 666 us).  Without it a chained launch follows as this
// kernel's blocks end, which still hides the launch: calls back to back, M_hat^dagger
// M_hat light FP32 at 12^3x24 32.9 -> 20.7 us, light FP16 at 16^3x32 41.2 -> 35.1 us,
// heavy FP16 at 24^3x48 270.5 -> 257.5 us, light FP16 at 32^3x64 419 -> 409 us.
// ---------------------------------------------------------------------------
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void pdl_trigger() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

template <typename... Params, typename... Args>
inline cudaError_t launch_chained(void (*kernel)(Params...), int grid, int block, size_t smem, cudaStream_t st,
                                  bool chained, const Args&... args) {
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3((unsigned)grid);
    cfg.blockDim = dim3((unsigned)block);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute attr{};
    attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr.val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = &attr;
    cfg.numAttrs = chained ? 1 : 0;
    return cudaLaunchKernelEx(&cfg, kernel, args...);
}

// ---------------------------------------------------------------------------
// solver scalar finalisers (run by the first warp of the last block of a reduction)
// ---------------------------------------------------------------------------
// Zeta recurrences of multishift CG for the shifts still active, a lane each: one after
// another their FP64 divisions held the solver's chain up (multishift solves with
// refinement, 10 shifts at 8^2x12x16 19.7 -> 18.4 ms, 12 at 24^3x48 553.4 -> 551.1 ms).
__device__ inline void ms_alpha(MsCtl* ms, double alpha, int k) {
    const double alpha_old = ms->alpha_old, beta_old = ms->beta_old;
    if (k < ms->nshift) {
        if (ms->active[k] != 1) {
            ms->active[k] = 0;
            ms->alpha_s[k] = 0.0;
        } else {
            const double z = ms->zeta[k], zo = ms->zeta_old[k];
            const double den = alpha * beta_old * (zo - z) + zo * alpha_old * (1.0 + ms->dshift[k] * alpha);
            const double zn = z * zo * alpha_old / den;
            ms->alpha_s[k] = alpha * zn / z;
            ms->beta_s[k] = zn / z;            // ratio kept until beta is known
            ms->zeta_old[k] = z;
            ms->zeta[k] = zn;
        }
    }
    __syncwarp();
    if (k == 0) ms->alpha_old = alpha;
}

// After an iteration with ||r||^2 = t: directions and rings of the shifts (a lane each),
// and the end of the solve once all have converged.
__device__ inline void ms_update(SolverCtl* ctl, MsCtl* ms, double t, double beta, int slot, int k) {
    bool running = false;
    if (k < ms->nshift) {
        ms->alpha_ring[slot][k] = ms->active[k] ? ms->alpha_s[k] : 0.0;
        if (ms->active[k]) {
            const double ratio = ms->beta_s[k];
            ms->beta_s[k] = beta * ratio * ratio;
            ms->beta_ring[slot][k] = ms->beta_s[k];
            ms->zeta_ring[slot][k] = ms->zeta[k];
            // shifted residual r_k = zeta_k r
            running = !(ms->zeta[k] * ms->zeta[k] * t < ms->stop_rr);
            if (!running) ms->active[k] = 2;   // converged, last update pending
        }
    }
    const int na = __popc(__ballot_sync(0xffffffffu, running));
    if (k == 0) {
        ms->beta_old = beta;
        ms->n_active = na;
        if (na == 0 && ctl->flag == CTL_RUN) ctl->flag = CTL_STOP;
    }
}

__device__ inline void finalize_scalar(int fin, double t, SolverCtl* ctl, MsCtl* ms, double* dst) {
    const int lane = threadIdx.x;
    switch (fin) {
        case FIN_STORE:
            if (lane == 0) {
                if (dst) *dst = t; else ctl->result = t;
            }
            break;
        case FIN_PP:
            if (lane == 0) ctl->result = t;   // ||p||^2 for shifted systems
            break;
        case FIN_CG_ALPHA:
        case FIN_MS_ALPHA: {
            const double pAp = t + ctl->shift * ctl->result;
            const bool good = pAp > 0.0 && isfinite(pAp);
            const double alpha = good ? ctl->rr / pAp : 0.0;
            if (lane == 0) {
                ctl->pAp = pAp;
                if (good) {
                    ctl->alpha = alpha;
                    ctl->alpha_ring[ctl->slot] = alpha;
                } else {
                    ctl->flag = CTL_BREAKDOWN;
                }
            }
            if (good && fin == FIN_MS_ALPHA) ms_alpha(ms, alpha, lane);
            break;
        }
        case FIN_CG_UPDATE:
        case FIN_MS_UPDATE: {
            const double beta = t / ctl->rr;
            const int slot = ctl->slot;
            __syncwarp();
            if (lane == 0) {
                ctl->rr_old = ctl->rr;
                ctl->rr = t;
                ctl->beta = beta;
                ctl->slot = slot + 1 < ctl->ring ? slot + 1 : 0;
                ctl->iter += 1;
                if (!isfinite(t)) ctl->flag = CTL_BREAKDOWN;
                else if (t < ctl->stop_rr) ctl->flag = CTL_STOP;
                else if (ctl->iter >= ctl->maxiter) ctl->flag = CTL_MAXITER;
            }
            if (fin == FIN_MS_UPDATE) ms_update(ctl, ms, t, beta, slot, lane);
            break;
        }
        default:
            break;
    }
}

template <int BS>
__device__ __forceinline__ double block_sum(double v, double* sh) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    const int w = threadIdx.x >> 5, l = threadIdx.x & 31;
    if (l == 0) sh[w] = v;
    __syncthreads();
    double t = 0.0;
    if (threadIdx.x < 32) {
        t = (threadIdx.x < BS / 32) ? sh[threadIdx.x] : 0.0;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
    }
    __syncthreads();
    return t;
}

// Each block stores its partial; the last block to arrive sums all partials in
// index order (deterministic for a fixed grid) and runs the finaliser.
template <int BS>
__device__ __forceinline__ void reduce_finalize(double* partial, unsigned int* counter, int nblk,
                                                int lb, double bsum, int fin, SolverCtl* ctl,
                                                MsCtl* ms, double* dst, double* sh) {
    __shared__ int am_last;
    if (threadIdx.x == 0) {
        partial[lb] = bsum;
        __threadfence();
        const unsigned prev = atomicAdd(counter, 1u);
        am_last = (prev == (unsigned)(nblk - 1));
    }
    __syncthreads();
    if (!am_last) return;
    __threadfence();
    double t = 0.0;
    for (int k = threadIdx.x; k < nblk; k += BS) t += ((volatile double*)partial)[k];
    t = block_sum<BS>(t, sh);
    if (threadIdx.x == 0) *counter = 0u;
    if (threadIdx.x < 32) finalize_scalar(fin, t, ctl, ms, dst);
}

// ---------------------------------------------------------------------------
// vector (BLAS-1) problem tables
// ---------------------------------------------------------------------------
static_assert(RING >= 2, "VecProb::v");
struct VecProb {
    long vh;
    int nblk;
    void* v[2 + RING];   // (batches use four)
    SolverCtl* ctl;
    MsCtl* ms;
    double* partial;
    unsigned int* counter;
    double* dst;
};

template <int NP>
struct VecBatch {
    int n;
    int fin;
    int blk_start[NP + 1];
    VecProb p[NP];
};

template <int NP>
__device__ __forceinline__ int find_vproblem(const VecBatch<NP>& b, int blk) {
    int k = 0;
#pragma unroll 1
    while (k + 1 < b.n && blk >= b.blk_start[k + 1]) ++k;
    return k;
}

// multishift vectors (single problem)
struct MsVecs {
    void* x[MAX_SHIFTS];
    void* p[MAX_SHIFTS];
};

// ---------------------------------------------------------------------------
// launchers (host)
// ---------------------------------------------------------------------------
template <int P, int NF, int KIND, int NP>
cudaError_t launch_dslash(const OpBatch<NP>& b, int nblocks, cudaStream_t st);
// shared-memory staged variant (FP32 / 16-bit storage), STAGED_BS threads per block
template <int P, int NF, int KIND, int NP>
cudaError_t launch_dslash_staged(const OpBatch<NP>& b, int nblocks, cudaStream_t st);

// several warps per site, for small lattices (dslash_split.cu), SPLIT_SITES sites per block
template <int P, int NF, int KIND>
cudaError_t launch_dslash_split(const OpBatch<1>& b, int nblocks, cudaStream_t st);

// batched solves: p = r + beta p (+ ||p||^2 when the problem has a shift)       v = {p, r}
template <int P, int NC, int NP>
cudaError_t launch_cg_pupdate(const VecBatch<NP>& b, int nblocks, cudaStream_t st);
// batched solves: x += alpha p; r -= alpha (Ap + shift p); ||r||^2 -> FIN_CG_UPDATE   v = {x, p, r, Ap}
template <int P, int PX, int NC, int NP>
cudaError_t launch_cg_update(const VecBatch<NP>& b, int nblocks, cudaStream_t st);
// p_out = r + beta p_in (+ ||p_out||^2 when the problem has a shift)           v = {p_out, r, p_in}
template <int P, int NC, int NP>
cudaError_t launch_cg_direction(const VecBatch<NP>& b, int nblocks, cudaStream_t st);
// x += sum_{i < n} alpha_i p_i, alpha_i = ctl->alpha_ring[i] (n <= RING)         v = {x, -, p_0, ...};
// only while the problem runs, unless `always`; nblocks per problem (all of one size)
template <int P, int PX, int NC, int NP>
cudaError_t launch_cg_xupdate(const VecBatch<NP>& b, int n, bool always, int nblocks, cudaStream_t st);
// dst (precision PD) = src (precision PS)                        v = {dst, src}
template <int PD, int PS, int NC, int NP>
cudaError_t launch_convert(const VecBatch<NP>& b, int nblocks, cudaStream_t st);
// y(F64) += x(PS)                                                v = {y, x}
template <int PS, int NC, int NP>
cudaError_t launch_add_to64(const VecBatch<NP>& b, int nblocks, cudaStream_t st);
// r(F64) = b - Ax - shift x, ||r||^2 -> FIN_STORE(dst)           v = {r, b, Ax, x}
template <int NC, int NP>
cudaError_t launch_residual64(const VecBatch<NP>& b, int nblocks, cudaStream_t st);
// ||v0||^2 -> FIN_STORE(dst)
template <int P, int NC, int NP>
cudaError_t launch_norm2(const VecBatch<NP>& b, int nblocks, cudaStream_t st);
// v0 = v0 * scale (F64 native) where scale = 1/sqrt(*dst)  (power iteration)
template <int NC>
cudaError_t launch_normalize64(const VecBatch<1>& b, int nblocks, cudaStream_t st);

// multishift: for each shift n iterations at once (MsCtl's rings),
//   x_k += alpha_k p_k; p_k = zeta_k r_i + beta_k p_k,  i < n <= RING             v = {-, -, r_1, ...}
// (r_i the residual after the i-th of them); only while the problem runs, unless `always`
template <int P, int PX, int NC>
cudaError_t launch_ms_block(const VecBatch<1>& b, const MsVecs& mv, int n, bool always, int nblocks, cudaStream_t st);

// layout
template <int P, int NC>
cudaError_t launch_import(void* dst, const double* src, long vh, cudaStream_t st);
template <int P, int NC>
cudaError_t launch_export(double* dst, const void* src, long vh, cudaStream_t st);
template <int P>
cudaError_t launch_links_from64(void* dst, const void* src64, long vh, cudaStream_t st);
template <int P>
cudaError_t launch_clover_from64(void* dst, const double* src, long vh, int nreal, cudaStream_t st);
cudaError_t launch_f64_to_df(void* dst, const void* src, long n, cudaStream_t st);

}  // namespace tmk
