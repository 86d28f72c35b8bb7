// Fermion-force outer products of the hopping term on every link.
//
// Sec. 4.3 ("Efficiency") reports that the force of the rational-approximation
// monomials stayed on the CPU, where colour outer products of several
// two-flavour spinors, one pair per shift of the multishift solve, dominated
// its cost.  This kernel computes that step for n field pairs (X_k, Y_k) and
// weights c_k in one pass over the lattice:
//
//   W_mu(x) = ph_mu(x) sum_k c_k sum_flavour [ X_k(x+mu) (x) ((1 - g_mu) Y_k(x))^*
//                                            + ((1 + g_mu) Y_k(x+mu)) (x) X_k(x)^* ]
//   force_mu(x) += T_A[ U_mu(x) W_mu(x) ]    (traceless anti-hermitian part)
//
// so that force_mu(x) is the derivative of S = sum_k c_k Re <Y_k, H[U] X_k>
// along su(3) directions of U_mu(x) (H the hopping term).  Optionally g5 Y_k
// takes the place of Y_k: the Schur operators' hopping force is one such pair
// per shift, X = (M_ee^-1 H_eo b, b) and Y = g5 (M_ee(-s)^-1 H_eo a, a).
//
// Each spin sum reduces to two spin components: in the chiral basis
// g_mu = [[0, G], [G^+, 0]] and (1 + s g_mu) B = (h, s G^+ h) with
// h = B_up + s G B_down, so that
//   sum_spin A (x) ((1 + s g_mu) B)^* = sum_{l=0,1} (A_up + s G A_down)_l (x) h_l^*
// and both terms are sums of two colour outer products of half spinors:
// the forward term pairs the s = -1 halves of X(x+mu) and Y(x), the backward
// term the s = +1 halves of Y(x+mu) and X(x).
//
// Layout and mapping.  Fields are native (structure of arrays over the Vh
// sites of one parity; 32- or 16-bit storage), math is FP32, the force is the
// canonical FP64 link layout and is read, added to and written once.  A block of
// 32 x 2 x 2 threads covers 64 sites: 32 half-site indices of both parities (z),
// directions 0, 1 or 2, 3 of a site per thread (y), so every warp's load of a field
// vector is one contiguous 512-byte span (16 B per site) and its neighbour loads are
// the same span shifted.  Two directions a thread load the site's own X, Y once for
// both (36 vectors instead of 48 per pair); 24^3x48, 12 two-flavour pairs: one
// direction a thread 1609 us FP32 / 1218 us FP16, two 1182 / 981 us, four 1205 / 1178 us.
//
// Site order.  A site's spinors are read for its own links and as the forward
// neighbours of four other sites.  In lexicographic order the +t neighbour is a time
// slice away, and where a slice of all pairs is a good part of the L2 the blocks that
// share it run too far apart (DRAM reads 1.8 x the fields at 64 MB a slice).  Such
// lattices are walked in tiles of up to 8 time slices, t inside z (ForceArgs::tt): 1182 ->
// 1118 us (tiles of 4 / 16 / 48: 1123 / 1177 / 1279 us).  At 33 MB a slice both orders
// take the same time, and below the plain one is faster (12 pairs of one flavour,
// 32 MB: 643 against 670 us), so the line is at 40 MB.
//
// Measured and not used: loads issued one or two terms ahead in registers (168, 3
// blocks: 1144 us), prefetch.global.L2 of the next pair (1117 us), the force added
// through shared memory in contiguous runs (1188 us).
//
// Bytes per launch (algorithmic): each field read once (2 n V spinors), the FP32
// links once (4 V x 12 reals), the force read and written once (2 x 4 V x 18 x 8).
#include "force.h"

namespace tmk {

// half spinor h = (psi_up + S G_mu psi_down), times f:
//   G_x = -i s1, G_y = -i s2, G_z = -i s3, G_t = -1 (chiral basis)
template <int MU, int S>
__device__ __forceinline__ void force_half(cpx<float> (&h)[2][3], const cpx<float>* p, float f) {
    const float s = (float)S;
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        const cpx<float> p0 = p[c], p1 = p[3 + c], p2 = p[6 + c], p3 = p[9 + c];
        cpx<float> a, b;
        if (MU == 0) {          // G psi_dn = -i (p3, p2)
            a = p0 - s * mul_i(p3);
            b = p1 - s * mul_i(p2);
        } else if (MU == 1) {   // G psi_dn = (-p3, p2)
            a = p0 - s * p3;
            b = p1 + s * p2;
        } else if (MU == 2) {   // G psi_dn = (-i p2, i p3)
            a = p0 - s * mul_i(p2);
            b = p1 + s * mul_i(p3);
        } else {                // G psi_dn = -(p2, p3)
            a = p0 - s * p2;
            b = p1 - s * p3;
        }
        h[0][c] = f * a;
        h[1][c] = f * b;
    }
}

// 12 complex components of flavour f at site i, unscaled; sc = the site's
// scale for 16-bit storage (1 for FP32)
template <int P, int NF>
__device__ __forceinline__ void force_load(const void* base, long vh, long i, int f, cpx<float>* p, float& sc) {
    load_readonly<P, 24>(base, vh, i, 24 * f, reinterpret_cast<float*>(p));
    sc = 1.f;
    if constexpr (P == PB16 || P == PF16) {
        const float* nrm = reinterpret_cast<const float*>(reinterpret_cast<const char*>(base) +
                                                          (size_t)vh * NF * 12 * 2 * 2);
        sc = __ldg(nrm + i);
    }
}

// w[3a + b] += sum_l u[l][a] conj(v[l][b])
__device__ __forceinline__ void force_outer2(cpx<float> (&w)[9], const cpx<float> (&u)[2][3],
                                             const cpx<float> (&v)[2][3]) {
#pragma unroll
    for (int a = 0; a < 3; ++a)
#pragma unroll
        for (int b = 0; b < 3; ++b) {
            cfma_cj(w[3 * a + b], v[0][b], u[0][a]);
            cfma_cj(w[3 * a + b], v[1][b], u[1][a]);
        }
}

// Neighbour of site c in direction mu (checkerboard index of the other parity), and
// whether the hop crosses the lattice's edge
template <int MU>
__device__ __forceinline__ long force_neighbour(const Geom& g, const Coord& c, bool& wrap) {
    const int x = MU == 0 ? c.x : (MU == 1 ? c.y : (MU == 2 ? c.z : c.t));
    const int L = MU == 0 ? g.X : (MU == 1 ? g.Y : (MU == 2 ? g.Z : g.T));
    wrap = x + 1 == L;
    const int n = wrap ? 0 : x + 1;
    return cb_index(g, MU == 0 ? n : c.x, MU == 1 ? n : c.y, MU == 2 ? n : c.z, MU == 3 ? n : c.t);
}

// One field pair and flavour f on link (x, MU): w += c_k [ X(x+mu) (x) ((1 - g_mu) Y(x))^*
// + ((1 + g_mu) Y(x+mu)) (x) X(x)^* ], xs, ys the site's own spinors (scales sx, sy),
// xn, yn the fields of the other parity, j the neighbour.
// G5: the Y fields enter as g5 Y.  P_s(g5 B) = B_up - s G B_down = P_-s(B), so
// g5 only flips the projection sign of the Y spinors.
template <int P, int NF, int MU, bool G5>
__device__ __forceinline__ void force_pair(cpx<float> (&w)[9], const void* xn, const void* yn, long vh, long j, int f,
                                           const cpx<float>* xs, float sx, const cpx<float>* ys, float sy, float ck) {
    constexpr int SY1 = G5 ? +1 : -1;   // sign of Y(x) in the forward term
    constexpr int SY2 = G5 ? -1 : +1;   // sign of Y(x+mu) in the backward term
    cpx<float> p[12];
    cpx<float> hu[2][3], hv[2][3];
    float sn;
    // forward hop at x
    force_load<P, NF>(xn, vh, j, f, p, sn);
    force_half<MU, -1>(hu, p, 1.f);
    force_half<MU, SY1>(hv, ys, ck * sn * sy);
    force_outer2(w, hu, hv);
    // backward hop at x+mu (through U_mu(x)^dagger)
    force_load<P, NF>(yn, vh, j, f, p, sn);
    force_half<MU, SY2>(hu, p, 1.f);
    force_half<MU, +1>(hv, xs, ck * sn * sx);
    force_outer2(w, hu, hv);
}

// Z = U W, force += T_A[Z] = (Z - Z^+)/2 - i Im(tr Z)/3 on link (x, MU)
template <int MU>
__device__ __forceinline__ void force_project(const ForceArgs& a, const cpx<float> (&w)[9], float ph, long i, int par,
                                              long lex) {
    cpx<float> u[9];
    load_link<P32>(a.gauge[par], a.g.vh, MU, i, u);
    cpx<float> z[9];
#pragma unroll
    for (int r = 0; r < 3; ++r)
#pragma unroll
        for (int s = 0; s < 3; ++s) {
            cpx<float> acc = C(0.f, 0.f);
#pragma unroll
            for (int m = 0; m < 3; ++m) cfma(acc, u[3 * r + m], w[3 * m + s]);
            z[3 * r + s] = ph * acc;
        }
    const float itr = (z[0].im + z[4].im + z[8].im) * (1.f / 3.f);
    double2* out = reinterpret_cast<double2*>(a.force) + (lex * 4 + MU) * 9;
#pragma unroll
    for (int r = 0; r < 3; ++r)
#pragma unroll
        for (int s = 0; s < 3; ++s) {
            const cpx<float> zrs = z[3 * r + s], zsr = z[3 * s + r];
            float re = 0.5f * (zrs.re - zsr.re);
            float im = 0.5f * (zrs.im + zsr.im);
            if (r == s) im -= itr;
            double2 o = out[3 * r + s];
            o.x += (double)re;
            o.y += (double)im;
            out[3 * r + s] = o;
        }
}

// directions MU and MU + 1 of one site
template <int P, int NF, int MU, bool G5>
__device__ __forceinline__ void force_links(const ForceArgs& a, long i, int par, const Coord& c) {
    const long vh = a.g.vh;
    bool wrap0, wrap1;
    const long j0 = force_neighbour<MU>(a.g, c, wrap0), j1 = force_neighbour<MU + 1>(a.g, c, wrap1);
    cpx<float> w0[9], w1[9];
#pragma unroll
    for (int e = 0; e < 9; ++e) w0[e] = w1[e] = C(0.f, 0.f);
    // pairs and flavours as one loop over one copy of the code: unrolled over the
    // flavours, the variants that share an SM overflow the instruction cache
#pragma unroll 1
    for (int q = 0; q < a.n * NF; ++q) {
        const int k = NF == 2 ? q >> 1 : q, f = NF == 2 ? q & 1 : 0;
        const void* xn = a.x[k][1 - par];
        const void* yn = a.y[k][1 - par];
        const float ck = a.c[k];
        cpx<float> xs[12], ys[12];
        float sx, sy;
        force_load<P, NF>(a.y[k][par], vh, i, f, ys, sy);
        force_load<P, NF>(a.x[k][par], vh, i, f, xs, sx);
        force_pair<P, NF, MU, G5>(w0, xn, yn, vh, j0, f, xs, sx, ys, sy, ck);
        force_pair<P, NF, MU + 1, G5>(w1, xn, yn, vh, j1, f, xs, sx, ys, sy, ck);
    }
    const long lex = 2 * i + (c.x & 1);
    force_project<MU>(a, w0, 1.f, i, par, lex);
    force_project<MU + 1>(a, w1, MU + 1 == 3 && wrap1 ? a.bc_t : 1.f, i, par, lex);
}

// 4 resident blocks per SM (128 registers): 1182 us at 24^3x48, 12 two-flavour FP32
// pairs (before the site order of a.tt); 3 / 5 / 6 blocks 1311 / 1301 / 1524 us.
template <int P, int NF, bool G5>
__global__ void __launch_bounds__(128, 4) force_outer_kernel(const __grid_constant__ ForceArgs a) {
    const int v = blockIdx.x * 32 + threadIdx.x;
    if (v >= a.g.vh) return;
    const int par = threadIdx.z;
    Coord c;
    long i = v;
    if (a.tt == 0) {
        c = cb_coords(a.g, i, par);
    } else {
        // v counts half-sites along x-lines in the order (t / tt, z, y / 2, t % tt, y % 2),
        // slowest first; the last tile of t may be shorter
        const Geom& g = a.g;
        const int hx = g.X / 2;
        const int line = v / hx, xi = v - line * hx;
        const int per = a.tt * g.Z * g.Y, tile = line / per;
        const int st = min(a.tt, g.T - tile * a.tt);
        int r = line - tile * per;
        const int y1 = r & 1;
        r >>= 1;
        c.t = tile * a.tt + r % st;
        r /= st;
        c.y = 2 * (r % (g.Y / 2)) + y1;
        c.z = r / (g.Y / 2);
        c.x = 2 * xi + ((c.y + c.z + c.t + par) & 1);
        i = (long)((c.t * g.Z + c.z) * g.Y + c.y) * hx + xi;
    }
    if (threadIdx.y == 0) force_links<P, NF, 0, G5>(a, i, par, c);   // warp-uniform
    else force_links<P, NF, 2, G5>(a, i, par, c);
}

template <int P, int NF>
static cudaError_t launch_t(const ForceArgs& a, cudaStream_t st) {
    const long nblk = (a.g.vh + 31) / 32;
    if (a.g5y)
        force_outer_kernel<P, NF, true><<<(unsigned)nblk, dim3(32, 2, 2), 0, st>>>(a);
    else
        force_outer_kernel<P, NF, false><<<(unsigned)nblk, dim3(32, 2, 2), 0, st>>>(a);
    return cudaGetLastError();
}

cudaError_t launch_force_outer(int prec, int nf, const ForceArgs& a0, cudaStream_t st) {
    if (a0.n <= 0 || a0.g.vh <= 0) return cudaSuccess;
    ForceArgs a = a0;
    // bytes of all pairs on a plane of constant z, t and on a time slice; in the tiled
    // order the +z neighbour is tt planes away (kept below 24 MB)
    const double plane = (double)a.g.X * a.g.Y * 2 * a.n * 24 * nf * prec_esz(prec);
    if (plane * a.g.Z <= 40e6) a.tt = 0;
    else a.tt = plane * 8 <= 24e6 ? 8 : (plane * 4 <= 24e6 ? 4 : 2);
    switch (prec) {
        case P32: return nf == 1 ? launch_t<P32, 1>(a, st) : launch_t<P32, 2>(a, st);
        case PB16: return nf == 1 ? launch_t<PB16, 1>(a, st) : launch_t<PB16, 2>(a, st);
        case PF16: return nf == 1 ? launch_t<PF16, 1>(a, st) : launch_t<PF16, 2>(a, st);
        default: return cudaErrorInvalidValue;
    }
}

}  // namespace tmk
