// Gauge-field import, low-precision link copies, and the clover term with its
// site-local inverses (Sec. 2: the clover term and the even-site blocks
// (M_ee +- i mu g5)^-1 of eq:hQpm and (M_ee + i mubar g5 tau3 - epsbar tau1)^-1
// of eq:hQh).  All clover arithmetic is FP64; stored copies are converted to the
// requested storage precision afterwards.
#include "tm_internal.h"
#include "dfsplit.h"
#include "tm_kernels.h"

namespace tmk {

// canonical [t][z][y][x][mu][3][3] complex FP64 -> native FP64 [parity][mu*9+k][vh] double2
__global__ void k_gauge_import(void* dst0, void* dst1, const double* __restrict__ src, Geom g) {
    const long V = 2 * g.vh;
    const long idx = (long)blockIdx.x * blockDim.x + threadIdx.x;
    if (idx >= 4 * V) return;
    const long lex = idx >> 2;
    const int mu = (int)(idx & 3);
    long r = lex;
    const int x = (int)(r % g.X); r /= g.X;
    const int y = (int)(r % g.Y); r /= g.Y;
    const int z = (int)(r % g.Z);
    const int t = (int)(r / g.Z);
    const int par = (x + y + z + t) & 1;
    const long cb = lex >> 1;
    double2* d = reinterpret_cast<double2*>(par ? dst1 : dst0);
    const double2* s = reinterpret_cast<const double2*>(src) + idx * 9;
#pragma unroll
    for (int k = 0; k < 9; ++k) d[(long)(mu * 9 + k) * g.vh + cb] = s[k];
}

// native FP64 links of one parity (9 complex per direction) -> native precision P
// (the first LinkStore<P>::N complex per direction; FP32/16-bit keep rows 0, 1)
template <int P>
__global__ void k_links_from64(void* dst, const double2* __restrict__ src, long vh) {
    constexpr int N = LinkStore<P>::N;
    const long e = (long)blockIdx.x * blockDim.x + threadIdx.x;   // destination element
    if (e >= 4 * N * vh) return;
    const long w = e / vh, i = e - w * vh;
    const int mu = (int)(w / N), k = (int)(w % N);
    const double2 v = src[(long)(mu * 9 + k) * vh + i];
    if constexpr (P == P32) {
        reinterpret_cast<float2*>(dst)[e] = make_float2((float)v.x, (float)v.y);
    } else if constexpr (P == P64) {
        reinterpret_cast<double2*>(dst)[e] = v;
    } else {
        const uint32_t w = f2h2<P>((float)v.x, (float)v.y);
        reinterpret_cast<unsigned int*>(dst)[e] = w;
    }
}

// native FP64 clover reals (nreal per site, double2 vectors) -> native precision P
template <int P>
__global__ void k_clover_from64(void* dst, const double* __restrict__ src, long vh, int nreal) {
    constexpr int W = PT<P>::W;
    const long e = (long)blockIdx.x * blockDim.x + threadIdx.x;   // target vector index
    const long nvec = (long)(nreal / W) * vh;
    if (e >= nvec) return;
    const long v = e / vh, i = e - v * vh;
    typename PT<P>::R buf[W];
#pragma unroll
    for (int c = 0; c < W; ++c) {
        const long r = v * W + c;                       // real index within the site
        buf[c] = (typename PT<P>::R)src[((r >> 1) * vh + i) * 2 + (r & 1)];
    }
    store_reals<P, W>(dst, vh, i, (int)(v * W), buf);
}

// ---------------------------------------------------------------------------
// clover term
// ---------------------------------------------------------------------------
using cd = cpx<double>;

// The clover term in three steps, all FP64 and all bound by the FP64 units (about
// 2 lanes per cycle and SM), so the split is the one with the fewest products:
//   k_leaves   one thread per site and plane: the plaquette based at x, once, and
//              its four rotations, which are the leaves of its four corners.  With
//              e = b c^+, f = d^+ a they are  a (e d^+), e f, c^+ (f b), f e:
//              eight 3x3 products, the last of each leaf restricted to the part
//              that survives Q - Q^+ (792 FMAs instead of the 1296 of a site that
//              multiplies out its own four leaves);
//   k_field    one thread per site and plane: sums the corners' contributions,
//              removes the trace: F_munu, 9 reals;
//   k_clover   one thread per site and chirality: A and, on even sites, its inverses.
// The leaves pass through memory: 576 B a site and plane, at 24^3x48 about 0.4 ms
// of the whole.  Two planes at a time fit the (not yet written) array of the light
// even inverse, and F fits the array of A, so nothing is allocated.
// 24^3x48 with both inverses: 16.8 ms as one kernel per parity, each site multiplying out its
// own leaves -> 8.1 ms.
struct M3 {
    cd m[9];
};

// The inner index in the order in which entry (i, j) of a product sums it: links are
// nearer to the identity than to zero, so the terms with a diagonal factor come last,
// when the small ones are summed.  Rounding error of A's off-diagonal entries, against
// each site's own four leaves in the plain order: 1.08 -> 0.96.
__host__ __device__ constexpr int inner(int i, int j, int n) {
    return i == j ? (i + 1 + n) % 3 : (n == 0 ? 3 - i - j : (n == 1 ? i : j));
}

// a b, a b^+, a^+ b
template <bool DA, bool DB>
__device__ __forceinline__ M3 mul3(const M3& a, const M3& b) {
    M3 c;
#pragma unroll
    for (int i = 0; i < 3; ++i)
#pragma unroll
        for (int j = 0; j < 3; ++j) {
            cd s = C(0.0, 0.0);
#pragma unroll
            for (int n = 0; n < 3; ++n) {
                const int k = inner(i, j, n);
                const cd x = DA ? a.m[3 * k + i] : a.m[3 * i + k];
                const cd y = DB ? b.m[3 * j + k] : b.m[3 * k + j];
                if (DA) cfma_cj(s, x, y);
                else if (DB) cfma_cj(s, y, x);
                else cfma(s, x, y);
            }
            c.m[3 * i + j] = s;
        }
    return c;
}

// The anti-hermitian part M - M^+ of M = a b (DA: a^+ b) as 9 reals, one store each
// stride apart: the three diagonal entries' imaginary parts / 2, then the entries
// (1,0), (2,0), (2,1) as (re, im)
template <bool DA>
__device__ __forceinline__ void store_antiherm(double* out, long stride, const M3& a, const M3& b) {
    auto at = [&](int i, int k) { return DA ? a.m[3 * k + i] : a.m[3 * i + k]; };
#pragma unroll
    for (int i = 0; i < 3; ++i) {
        double t = 0.0;
#pragma unroll
        for (int n = 0; n < 3; ++n) {
            const int k = inner(i, i, n);
            const cd x = at(i, k), y = b.m[3 * k + i];
            t = fma(x.re, y.im, t);
            t = DA ? fma(-x.im, y.re, t) : fma(x.im, y.re, t);
        }
        out[i * stride] = t;
    }
#pragma unroll
    for (int i = 1; i < 3; ++i)
#pragma unroll
        for (int j = 0; j < i; ++j) {
            cd s = C(0.0, 0.0), t = C(0.0, 0.0);   // M_ij, M_ji
#pragma unroll
            for (int n = 0; n < 3; ++n) {
                const int k = inner(i, j, n);
                if (DA) {
                    cfma_cj(s, at(i, k), b.m[3 * k + j]);
                    cfma_cj(t, at(j, k), b.m[3 * k + i]);
                } else {
                    cfma(s, at(i, k), b.m[3 * k + j]);
                    cfma(t, at(j, k), b.m[3 * k + i]);
                }
            }
            const int e = 3 + 2 * (i * (i - 1) / 2 + j);
            out[e * stride] = s.re - t.re;
            out[(e + 1) * stride] = s.im + t.im;
        }
}

struct CloverArgs {
    Geom g;
    const void* gauge[2];
    int plane0;          // k_leaves, k_field: planes plane0, plane0 + 1
    double* leaf;        // [parity][plane of the two][corner][9][vh]
    double* F[2];        // per parity [plane][5][vh] pairs (9 reals and one unused); the array of
                         // A, whose pairs of a site k_clover writes over the same site's F
    double kc;           // kappa csw
    double mu_t, mubar_t, epsbar_t;
    double* outB;        // even inverse blocks (may be null)
    double* outH;        // heavy even inverse blocks (may be null)
};

// planes 0 xy, 1 xz, 2 xt, 3 yz, 4 yt, 5 zt
__device__ __forceinline__ void plane_dirs(int plane, int& mu, int& nu) {
    mu = plane < 3 ? 0 : (plane < 5 ? 1 : 2);
    nu = plane < 3 ? plane + 1 : (plane < 5 ? plane - 1 : 3);
}

// checkerboard index of the neighbour d (-1, 0, +1) steps along mu and e along nu
__device__ __forceinline__ long shifted(const Geom& g, const Coord& c, int mu, int d, int nu, int e) {
    int x[4] = {c.x, c.y, c.z, c.t};
    const int L[4] = {g.X, g.Y, g.Z, g.T};
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        x[k] += (k == mu ? d : 0) + (k == nu ? e : 0);
        if (x[k] < 0) x[k] += L[k];
        if (x[k] >= L[k]) x[k] -= L[k];
    }
    return cb_index(g, x[0], x[1], x[2], x[3]);
}

// blockIdx.y = 2 * (plane of the two) + parity
__global__ void __launch_bounds__(64) k_leaves(const __grid_constant__ CloverArgs p) {
    const long vh = p.g.vh, i = (long)blockIdx.x * 64 + threadIdx.x;
    if (i >= vh) return;
    const int par = blockIdx.y & 1, pl = blockIdx.y >> 1;
    int mu, nu;
    plane_dirs(p.plane0 + pl, mu, nu);
    const Coord x = cb_coords(p.g, i, par);
    const long xm = shifted(p.g, x, mu, 1, nu, 0), xn = shifted(p.g, x, mu, 0, nu, 1);
    M3 a, b, c, d;
    load_link<P64>(p.gauge[1 - par], vh, nu, xm, b.m);
    load_link<P64>(p.gauge[1 - par], vh, mu, xn, c.m);
    load_link<P64>(p.gauge[par], vh, mu, i, a.m);
    load_link<P64>(p.gauge[par], vh, nu, i, d.m);
    double* out = p.leaf + (long)(par * 2 + pl) * 36 * vh + i;
    const M3 e = mul3<false, true>(b, c), f = mul3<true, false>(d, a);
    store_antiherm<false>(out + 9 * vh, vh, e, f);                             // corner x + mu
    store_antiherm<false>(out + 27 * vh, vh, f, e);                            // corner x + nu
    store_antiherm<false>(out, vh, a, mul3<false, true>(e, d));                // corner x
    store_antiherm<true>(out + 18 * vh, vh, c, mul3<false, false>(f, b));      // corner x + mu + nu
}

__global__ void __launch_bounds__(128) k_field(const __grid_constant__ CloverArgs p) {
    const long vh = p.g.vh, i = (long)blockIdx.x * 128 + threadIdx.x;
    if (i >= vh) return;
    const int par = blockIdx.y & 1, pl = blockIdx.y >> 1;
    int mu, nu;
    plane_dirs(p.plane0 + pl, mu, nu);
    const Coord x = cb_coords(p.g, i, par);
    const double* same = p.leaf + (long)(par * 2 + pl) * 36 * vh;
    const double* other = p.leaf + (long)((1 - par) * 2 + pl) * 36 * vh;
    const double* src[4] = {same + i, other + 9 * vh + shifted(p.g, x, mu, -1, nu, 0),
                            same + 18 * vh + shifted(p.g, x, mu, -1, nu, -1),
                            other + 27 * vh + shifted(p.g, x, mu, 0, nu, -1)};
    double q[9];
#pragma unroll
    for (int k = 0; k < 9; ++k) q[k] = (src[0][k * vh] + src[1][k * vh]) + (src[2][k * vh] + src[3][k * vh]);
    // F = (Q - Q^+) / 8 less its trace (imaginary; the leaves' diagonal holds half of Q - Q^+)
    const double tr = (q[0] + q[1] + q[2]) * (1.0 / 3.0);
    double2* out = reinterpret_cast<double2*>(p.F[par]) + (long)(p.plane0 + pl) * 5 * vh + i;
#pragma unroll
    for (int k = 0; k < 9; ++k) q[k] = k < 3 ? 0.25 * (q[k] - tr) : 0.125 * q[k];
#pragma unroll
    for (int k = 0; k < 5; ++k) out[k * vh] = make_double2(q[2 * k], k < 4 ? q[2 * k + 1] : 0.0);
}

// hermitian 6x6: real diagonal, strictly lower entries row by row
struct H6 {
    double d[6];
    cd l[15];
    __device__ __forceinline__ cd at(int r, int j) const {   // r != j
        return r > j ? l[r * (r - 1) / 2 + j] : cj(l[j * (j - 1) / 2 + r]);
    }
};

// The 6x6 matrices below (A, A^2, D and their factors) have a diagonal near 1 and small
// entries beside it, so every sum takes the products of small entries first and the one
// with a diagonal factor last: all but its last roundings are then small ones.  Relative
// error of the light inverse blocks 3.7e-16 -> 2.1e-16 (full products in the order of
// the indices: 3.1e-16), of D - 1 3.3e-16 -> 2.2e-16 (2.9e-16), at the same cost.

// the product of two hermitian matrices that commute (hermitian again)
__device__ __forceinline__ H6 mul_commuting(const H6& a, const H6& b) {
    H6 c;
#pragma unroll
    for (int r = 0; r < 6; ++r) {
        double t = 0.0;
#pragma unroll
        for (int k = 0; k < 6; ++k) {
            if (k == r) continue;
            const cd x = a.at(r, k), y = b.at(r, k);   // b_kr = conj(b_rk)
            t = fma(x.re, y.re, t);
            t = fma(x.im, y.im, t);
        }
        c.d[r] = fma(a.d[r], b.d[r], t);
#pragma unroll
        for (int j = 0; j < r; ++j) {
            cd s = C(0.0, 0.0);
#pragma unroll
            for (int k = 0; k < 6; ++k)
                if (k != r && k != j) cfma(s, a.at(r, k), b.at(k, j));
            const cd x = a.at(r, j), y = b.at(r, j);
            s.re = fma(x.re, b.d[j], s.re);
            s.im = fma(x.im, b.d[j], s.im);
            s.re = fma(a.d[r], y.re, s.re);
            s.im = fma(a.d[r], y.im, s.im);
            c.l[r * (r - 1) / 2 + j] = s;
        }
    }
    return c;
}

// (a + shift)^-1 of a hermitian positive definite a + shift, by Cholesky: L, then
// L^-1, then L^-+ L^-1
__device__ __forceinline__ H6 hpd6_inverse(const H6& a, double shift) {
    H6 L;   // L.d: 1 / L_jj
#pragma unroll
    for (int j = 0; j < 6; ++j) {
        double t = -shift;
#pragma unroll
        for (int k = 0; k < j; ++k) {
            const cd x = L.l[j * (j - 1) / 2 + k];
            t = fma(x.re, x.re, t);
            t = fma(x.im, x.im, t);
        }
        L.d[j] = rsqrt(a.d[j] - t);
#pragma unroll
        for (int i = j + 1; i < 6; ++i) {
            cd s = -a.l[i * (i - 1) / 2 + j];
#pragma unroll
            for (int k = 0; k < j; ++k) cfma_cj(s, L.l[j * (j - 1) / 2 + k], L.l[i * (i - 1) / 2 + k]);
            L.l[i * (i - 1) / 2 + j] = -L.d[j] * s;
        }
    }
    // in place, column by column from the right: Li_ij = -Li_ii sum_{j <= k < i} L_ik Li_kj
    H6 D;
#pragma unroll
    for (int j = 0; j < 6; ++j) {
        D.d[j] = L.d[j];
#pragma unroll
        for (int i = j + 1; i < 6; ++i) {
            const cd x = L.l[i * (i - 1) / 2 + j];
            cd s = C(0.0, 0.0);
#pragma unroll
            for (int k = j + 1; k < i; ++k) cfma(s, L.l[i * (i - 1) / 2 + k], D.l[k * (k - 1) / 2 + j]);
            s = C(fma(L.d[j], x.re, s.re), fma(L.d[j], x.im, s.im));
            D.l[i * (i - 1) / 2 + j] = -L.d[i] * s;
        }
    }
    H6 out;
#pragma unroll
    for (int j = 0; j < 6; ++j) {
        double t = 0.0;
#pragma unroll
        for (int k = j + 1; k < 6; ++k) {
            const cd x = D.l[k * (k - 1) / 2 + j];
            t = fma(x.re, x.re, t);
            t = fma(x.im, x.im, t);
        }
        out.d[j] = fma(D.d[j], D.d[j], t);
#pragma unroll
        for (int i = j + 1; i < 6; ++i) {
            const cd x = D.l[i * (i - 1) / 2 + j];
            cd s = C(0.0, 0.0);
#pragma unroll
            for (int k = i + 1; k < 6; ++k) cfma_cj(s, D.l[k * (k - 1) / 2 + i], D.l[k * (k - 1) / 2 + j]);
            out.l[i * (i - 1) / 2 + j] = C(fma(D.d[i], x.re, s.re), fma(D.d[i], x.im, s.im));
        }
    }
    return out;
}

// 36 reals of a packed hermitian block at real offset off, less `one` on the diagonal
__device__ __forceinline__ void store_h6(double* base, long vh, long i, int off, const H6& h, double one) {
    double r[36];
#pragma unroll
    for (int k = 0; k < 6; ++k) r[k] = h.d[k] - one;
#pragma unroll
    for (int k = 0; k < 15; ++k) {
        r[6 + 2 * k] = h.l[k].re;
        r[7 + 2 * k] = h.l[k].im;
    }
    store_reals<P64, 36>(base, vh, i, off, r);
}

// One thread per site of parity PAR and chirality (threadIdx.y):
//   A_c = 1 - kappa csw [ i s1 (x) a1 + i s2 (x) a2 + i s3 (x) a3 ],
//   a1 = F_yz + s F_xt,  a2 = -F_xz + s F_yt,  a3 = F_xy + s F_zt  (s = +1 / -1 per chirality),
// which is the chirality-block form of 1 - kappa csw sum_{mu<nu} g_mu g_nu F_munu:
//   [[ 1 - kc i a3, -kc (i a1 + a2) ], [ -kc (i a1 - a2), 1 + kc i a3 ]].
// Writes A (packed hermitian, 72 reals/site) over F, which both threads of a site
// have read by then; on even sites also the light inverse blocks
// B_c = (A_c + i s mu_t)^-1 = A D - i s mu_t D, D = (A^2 + mu_t^2)^-1 (144 reals),
// and/or the heavy A_c - 1, D_c - 1 (144; the deviation from the identity keeps
// 16-bit rounding relative to it).  A commutes with D, so A D is hermitian and half
// of it is computed.
template <int PAR>
__global__ void __launch_bounds__(128) k_clover(const __grid_constant__ CloverArgs p) {
    const long vh = p.g.vh, i = (long)blockIdx.x * 64 + threadIdx.x;
    const int cb = threadIdx.y;
    const double s = cb == 0 ? 1.0 : -1.0;
    H6 A;
    if (i < vh) {
        auto F = [&](int plane, int k) { return p.F[PAR][2 * ((plane * 5 + (k >> 1)) * vh + i) + (k & 1)]; };
        // per combination: imaginary diagonal, then entries (1,0), (2,0), (2,1)
        double a1[9], a2[9], a3[9];
#pragma unroll
        for (int k = 0; k < 9; ++k) {
            a1[k] = F(3, k) + s * F(2, k);
            a2[k] = s * F(4, k) - F(1, k);
            a3[k] = F(0, k) + s * F(5, k);
        }
        const double kc = p.kc;
#pragma unroll
        for (int r = 0; r < 3; ++r) {
            A.d[r] = 1.0 + kc * a3[r];
            A.d[3 + r] = 1.0 - kc * a3[r];
        }
        auto full = [](const double (&v)[9], int r, int j) {   // entry (r, j) of an antihermitian matrix
            if (r == j) return C(0.0, v[r]);
            const int e = 3 + 2 * (r > j ? r * (r - 1) / 2 + j : j * (j - 1) / 2 + r);
            return r > j ? C(v[e], v[e + 1]) : C(-v[e], v[e + 1]);
        };
#pragma unroll
        for (int r = 0; r < 3; ++r)
#pragma unroll
            for (int j = 0; j < 3; ++j) {
                if (j < r) {
                    const cd z = full(a3, r, j);
                    A.l[r * (r - 1) / 2 + j] = C(kc * z.im, -kc * z.re);             // -kc i z
                    A.l[(r + 3) * (r + 2) / 2 + j + 3] = C(-kc * z.im, kc * z.re);   // +kc i z
                }
                const cd u = full(a1, r, j), v = full(a2, r, j);
                A.l[(r + 3) * (r + 2) / 2 + j] = C(kc * (u.im + v.re), kc * (v.im - u.re));   // -kc (i u - v)
            }
    }
    __syncthreads();
    if (i >= vh) return;
    store_h6(p.F[PAR], vh, i, 36 * cb, A, 0.0);
    if (PAR != 0) return;
    const H6 A2 = mul_commuting(A, A);
    if (p.outB != nullptr) {
        const H6 D = hpd6_inverse(A2, p.mu_t * p.mu_t);
        const H6 AD = mul_commuting(A, D);
        const double m = s * p.mu_t;
        double2* out = reinterpret_cast<double2*>(p.outB) + (long)(36 * cb) * vh + i;
#pragma unroll
        for (int r = 0; r < 6; ++r) {
            out[(7 * r) * vh] = make_double2(AD.d[r], -m * D.d[r]);
#pragma unroll
            for (int j = 0; j < r; ++j) {
                const cd x = AD.l[r * (r - 1) / 2 + j], y = D.l[r * (r - 1) / 2 + j];
                out[(6 * r + j) * vh] = make_double2(fma(m, y.im, x.re), fma(-m, y.re, x.im));
                out[(6 * j + r) * vh] = make_double2(fma(-m, y.im, x.re), fma(-m, y.re, -x.im));
            }
        }
    }
    if (p.outH != nullptr) {
        const H6 D = hpd6_inverse(A2, p.mubar_t * p.mubar_t - p.epsbar_t * p.epsbar_t);
        store_h6(p.outH, vh, i, 72 * cb, A, 1.0);
        store_h6(p.outH, vh, i, 72 * cb + 36, D, 1.0);
    }
}

// unpack the packed hermitian A of one parity to [site][2][6][6] complex (debug export)
__global__ void k_clover_unpack(double2* out, const double* __restrict__ A, long vh) {
    const long i = (long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= vh) return;
    auto get = [&](int r) { return A[((long)(r >> 1) * vh + i) * 2 + (r & 1)]; };
    for (int cb = 0; cb < 2; ++cb)
        for (int r = 0; r < 6; ++r)
            for (int j = 0; j < 6; ++j) {
                double re, im;
                if (r == j) { re = get(36 * cb + r); im = 0.0; }
                else if (r > j) { re = get(36 * cb + herm_off(r, j)); im = get(36 * cb + herm_off(r, j) + 1); }
                else { re = get(36 * cb + herm_off(j, r)); im = -get(36 * cb + herm_off(j, r) + 1); }
                out[((i * 2 + cb) * 6 + r) * 6 + j] = make_double2(re, im);
            }
}

// ---------------------------------------------------------------------------
// launchers
// ---------------------------------------------------------------------------
cudaError_t launch_gauge_import(void* d0, void* d1, const double* src, const Geom& g, cudaStream_t st) {
    const long n = 8 * g.vh;
    k_gauge_import<<<(unsigned)((n + 255) / 256), 256, 0, st>>>(d0, d1, src, g);
    return cudaGetLastError();
}

template <int P>
cudaError_t launch_links_from64(void* dst, const void* src64, long vh, cudaStream_t st) {
    const long n = 4 * LinkStore<P>::N * vh;
    k_links_from64<P><<<(unsigned)((n + 255) / 256), 256, 0, st>>>(dst, reinterpret_cast<const double2*>(src64), vh);
    return cudaGetLastError();
}

template <int P>
cudaError_t launch_clover_from64(void* dst, const double* src, long vh, int nreal, cudaStream_t st) {
    const long n = (long)(nreal / PT<P>::W) * vh;
    k_clover_from64<P><<<(unsigned)((n + 255) / 256), 256, 0, st>>>(dst, src, vh, nreal);
    return cudaGetLastError();
}

cudaError_t launch_clover(const Geom& g, const void* g0, const void* g1, double kappa, double csw, double mu_t,
                          double mubar_t, double epsbar_t, double* outA0, double* outA1, double* outB, double* outH,
                          cudaStream_t st) {
    CloverArgs p{};
    p.g = g;
    p.gauge[0] = g0;
    p.gauge[1] = g1;
    p.leaf = outB;
    p.F[0] = outA0;
    p.F[1] = outA1;
    p.kc = kappa * csw;
    p.mu_t = mu_t;
    p.mubar_t = mubar_t;
    p.epsbar_t = epsbar_t;
    p.outB = outB;
    p.outH = outH;
    const unsigned nb64 = (unsigned)((g.vh + 63) / 64), nb128 = (unsigned)((g.vh + 127) / 128);
    for (p.plane0 = 0; p.plane0 < 6; p.plane0 += 2) {
        k_leaves<<<dim3(nb64, 4), 64, 0, st>>>(p);
        k_field<<<dim3(nb128, 4), 128, 0, st>>>(p);
    }
    k_clover<0><<<nb64, dim3(64, 2), 0, st>>>(p);
    k_clover<1><<<nb64, dim3(64, 2), 0, st>>>(p);
    return cudaGetLastError();
}

cudaError_t launch_clover_unpack(double* out, const double* A, long vh, cudaStream_t st) {
    k_clover_unpack<<<(unsigned)((vh + 127) / 128), 128, 0, st>>>(reinterpret_cast<double2*>(out), A, vh);
    return cudaGetLastError();
}

// FP64 arrays (a double2 per two reals: links, clover blocks, spinors) -> double-word
// arrays (a float4 (h, l, h, l) per two reals), n 16-byte elements
__global__ void k_f64_to_df(float4* dst, const double2* src, long n) {
    const long e = (long)blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= n) return;
    const double2 v = src[e];
    float4 q;
    df_split(v.x, q.x, q.y);
    df_split(v.y, q.z, q.w);
    dst[e] = q;
}
cudaError_t launch_f64_to_df(void* dst, const void* src, long n, cudaStream_t st) {
    if (n <= 0) return cudaSuccess;
    k_f64_to_df<<<(unsigned)((n + 255) / 256), 256, 0, st>>>(reinterpret_cast<float4*>(dst),
                                                              reinterpret_cast<const double2*>(src), n);
    return cudaGetLastError();
}

template cudaError_t launch_links_from64<P32>(void*, const void*, long, cudaStream_t);
template cudaError_t launch_links_from64<PB16>(void*, const void*, long, cudaStream_t);
template cudaError_t launch_links_from64<PF16>(void*, const void*, long, cudaStream_t);
template cudaError_t launch_clover_from64<P32>(void*, const double*, long, int, cudaStream_t);
template cudaError_t launch_clover_from64<PB16>(void*, const double*, long, int, cudaStream_t);
template cudaError_t launch_clover_from64<PF16>(void*, const double*, long, int, cudaStream_t);

}  // namespace tmk
