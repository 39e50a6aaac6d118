// K1: the operator D = 1 - kappa F H of Eq. (2) on the whole lattice, in FP64
// (dslash64_kernel), FP32, and FP32 with FP16 storage of links and clover; one thread
// per site and one or two right-hand sides.
//
// Each thread gathers its 8 neighbour spinors, projects each to a half-spinor
// (the rank-2 projector 1 -/+ gamma_mu), multiplies by the link, reconstructs
// and accumulates; then applies the chiral-block clover term and forms
// in - kappa F (H in).  Spinors are read site by site as 32-byte vectors, links (8 or
// 16 bytes) and clover (16 bytes) plane by plane, coalesced across the warp; neighbours
// of consecutive threads are consecutive, so neighbour re-reads hit L1/L2 and the HBM
// traffic stays close to one read of each field (768 B/site in FP32).
#include <algorithm>

#include "fields.cuh"
#include "qcd_internal.h"

namespace qcd {

// FP16 storage of links and clover (FP32 arithmetic): links as half2, clover
// planes as four halves (uint2).  |entries| <= about 1.5, far inside FP16 range.
__device__ __forceinline__ void load_link(const __half2 *__restrict__ U, long V, long n, int mu, float2 u[9]) {
    const unsigned *p = reinterpret_cast<const unsigned *>(U);
#pragma unroll
    for (int i = 0; i < 9; i++) {
        const unsigned w = __ldg(p + (mu * 9 + i) * V + n);
        u[i] = __half22float2(*reinterpret_cast<const __half2 *>(&w));
    }
}
__device__ __forceinline__ void load_clover(const uint2 *__restrict__ F, long V, long n, float f[72]) {
#pragma unroll
    for (int k = 0; k < 18; k++) {
        const uint2 v = __ldg(F + k * V + n);
        const float2 a = __half22float2(*reinterpret_cast<const __half2 *>(&v.x));
        const float2 b = __half22float2(*reinterpret_cast<const __half2 *>(&v.y));
        f[4 * k] = a.x; f[4 * k + 1] = a.y; f[4 * k + 2] = b.x; f[4 * k + 3] = b.y;
    }
}

// SU(3) 12-real storage (Table 1's compressed links): the first two rows, 3 float4 per link
// ([4][3][V]); the third row of a special unitary matrix is the complex conjugate of the cross
// product of the first two.
__device__ __forceinline__ void load_link(const float4 *__restrict__ U, long V, long n, int mu, float2 u[9]) {
#pragma unroll
    for (int p = 0; p < 3; p++) {
        const float4 v = __ldg(U + (mu * 3 + p) * V + n);
        u[2 * p] = make_float2(v.x, v.y);
        u[2 * p + 1] = make_float2(v.z, v.w);
    }
    auto cross = [](float2 a, float2 b, float2 c, float2 d) {  // conj(a b - c d)
        const float2 v = csub(cmul(a, b), cmul(c, d));
        return make_float2(v.x, -v.y);
    };
    u[6] = cross(u[1], u[5], u[2], u[4]);
    u[7] = cross(u[2], u[3], u[0], u[5]);
    u[8] = cross(u[0], u[4], u[1], u[3]);
}

// MINB: resident blocks per SM requested from the register allocator (each launch says what 3 to 7
// take).  One right-hand side in FP32 is bound by HBM (48^3x96: 1.40 ms, 5.8 TB/s of algorithmic bytes;
// 2.04 ms with the conversions to and from planes that the caller's layout does without), several by
// latency and L1 requests (24^3x48, 12: 675 us, 1200 with the conversions; L2 at 55%, HBM at 45%, issue
// at 42%; staging spinors through shared memory, two lanes per site and links site by site were all
// slower, 811 to 1170 us).  NR: right-hand sides per thread; each link and the
// clover field are loaded once and applied to all of them, so the field bytes
// per right-hand side drop from 576 to 576 / NR (FP32).  Over the grid the
// right-hand side (tile) index varies fastest, so the CTAs of one site block run
// close together and the field bytes come from HBM about once for all of them.
// With FP32 fields two right-hand sides per thread (4 blocks of 128 threads) are
// faster than one, three or four (672 us against 730 for three and 812 for four); with
// FP16 or two-row fields one per thread is, so those launch NR = 1.
template <int MINB, typename R, typename SP, typename LK, typename CL>
__global__ void __launch_bounds__(128, MINB) dslash_kernel(SP *__restrict__ out, const SP *__restrict__ in,
                                                     const LK *__restrict__ U, const CL *__restrict__ F,
                                                     R kappa, Geo g, int nrhs) {
    using C = typename CT<R>::C;
    chain_wait(in);
    // the right-hand side varies fastest over the (1-D) grid: the CTAs of one site block run
    // together and share its links and clover field through L2
    const long sblk = blockIdx.x / nrhs;
    const int rhs = (int)(blockIdx.x - sblk * nrhs);
    const long n = sblk * blockDim.x + threadIdx.x;
    if (n >= g.V) return;
    constexpr int PARTS = sizeof(C) * 12 / sizeof(SP);
    const SP *src = in + (long)rhs * PARTS * g.V;
    int x[4];
    site_coords(g, n, x);
    C acc[12];
#pragma unroll
    for (int k = 0; k < 12; k++) acc[k] = cmk<C>(0, 0);
    C psi[12], u[9];
    const R tsgn_f = (x[3] == g.L[3] - 1) ? (R)g.bc_t : (R)1;
    const R tsgn_b = (x[3] == 0) ? (R)g.bc_t : (R)1;
    // mu = 0
    { long m = nbr_fwd<0>(g, n, x); load_spinor(src, m, psi); load_link(U, g.V, n, 0, u); hop_term<0, true>(psi, u, (R)1, acc); }
    { long m = nbr_bwd<0>(g, n, x); load_spinor(src, m, psi); load_link(U, g.V, m, 0, u); hop_term<0, false>(psi, u, (R)1, acc); }
    { long m = nbr_fwd<1>(g, n, x); load_spinor(src, m, psi); load_link(U, g.V, n, 1, u); hop_term<1, true>(psi, u, (R)1, acc); }
    { long m = nbr_bwd<1>(g, n, x); load_spinor(src, m, psi); load_link(U, g.V, m, 1, u); hop_term<1, false>(psi, u, (R)1, acc); }
    { long m = nbr_fwd<2>(g, n, x); load_spinor(src, m, psi); load_link(U, g.V, n, 2, u); hop_term<2, true>(psi, u, (R)1, acc); }
    { long m = nbr_bwd<2>(g, n, x); load_spinor(src, m, psi); load_link(U, g.V, m, 2, u); hop_term<2, false>(psi, u, (R)1, acc); }
    { long m = nbr_fwd<3>(g, n, x); load_spinor(src, m, psi); load_link(U, g.V, n, 3, u); hop_term<3, true>(psi, u, tsgn_f, acc); }
    { long m = nbr_bwd<3>(g, n, x); load_spinor(src, m, psi); load_link(U, g.V, m, 3, u); hop_term<3, false>(psi, u, tsgn_b, acc); }
    R f[72];
    load_clover(F, g.V, n, f);
    C fa[12];
    clover_mul<R, C>(f, acc, fa);
    load_spinor(src, n, psi);
#pragma unroll
    for (int k = 0; k < 12; k++) {
        psi[k].x = fma(-kappa, fa[k].x, psi[k].x);
        psi[k].y = fma(-kappa, fa[k].y, psi[k].y);
    }
    store_spinor(out + (long)rhs * PARTS * g.V, n, psi);
}

template <int NR, int MODE, typename R, typename SP, typename LK, typename CL>
__device__ __forceinline__ void dslash_site(SP *__restrict__ out, const SP *__restrict__ in,
                                            const LK *__restrict__ U, const CL *__restrict__ F, R kappa,
                                            const Geo &g, long n, int r0, const bool act[NR],
                                            const SP *__restrict__ other, float part[NR][3]);

// The order in which the site blocks (128 sites) are taken: chunk by chunk of a t-slice, each through all of
// t, so that what a chunk shares with the next slice is still in L2.
struct BlockOrder {
    int row = 0, chunk = 0;  // blocks per t-slice, per chunk (0: in order)
};
__device__ __forceinline__ int block_of(const BlockOrder &o, int q, int nblk) {
    const int rows = nblk / o.row;
    if (q >= rows * o.row) return q;  // past the whole slices
    const int c = q / (o.chunk * rows), first = c * o.chunk, w = min(o.chunk, o.row - first);
    q -= first * rows;
    return q / w * o.row + first + q % w;
}

// The same with NR right-hand sides per thread (each link and the clover field loaded once for
// all of them).  MODE fuses the inner products the BiCGStab step after D needs into the
// epilogue: 1: <other, out> and |out|^2, 2: <out, other> and |out|^2, 0: none; each CTA (128
// consecutive sites) sums its sites per right-hand side by a fixed tree (a butterfly within each
// warp, then the four warps in order) into partial[rhs][3][site block], so a right-hand side's
// inner products do not depend on which others share its threads.  Right-hand sides inactive
// in gate (may be null) are skipped, their partials zero.
template <int MINB, int NR, typename R, typename SP, typename LK, typename CL, int MODE = 0, bool CHUNKED = false>
__global__ void __launch_bounds__(128, MINB) dslash_kernel_nr(SP *__restrict__ out, const SP *__restrict__ in,
                                                     const LK *__restrict__ U, const CL *__restrict__ F,
                                                     R kappa, Geo g, int nrhs,
                                                     const SP *__restrict__ other, double *__restrict__ partial,
                                                     const BicgScalars *__restrict__ gate, BlockOrder order) {
    using C = typename CT<R>::C;
    chain_wait(in, other, gate);
    // the right-hand-side tile varies fastest over the (1-D) grid: the CTAs of one site block
    // run together and share its links and clover field through L2
    const int ntile = (nrhs + NR - 1) / NR;
    long sblk = blockIdx.x / ntile;
    const int r0 = (int)(blockIdx.x - sblk * ntile) * NR;
    if constexpr (CHUNKED) sblk = block_of(order, (int)sblk, gridDim.x / ntile);
    const long n = sblk * blockDim.x + threadIdx.x;
    float part[NR][3];
#pragma unroll
    for (int r = 0; r < NR; r++) part[r][0] = part[r][1] = part[r][2] = 0.f;
    bool act[NR];
#pragma unroll
    for (int r = 0; r < NR; r++) act[r] = r0 + r < nrhs && (!gate || gate[r0 + r].active);
    if (n < g.V) dslash_site<NR, MODE>(out, in, U, F, kappa, g, n, r0, act, other, part);
    if (MODE) {
        __shared__ float sh[NR][3][4];
        const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
#pragma unroll
        for (int r = 0; r < NR; r++)
#pragma unroll
            for (int q = 0; q < 3; q++) {
                float v = part[r][q];
#pragma unroll
                for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
                if (lane == 0) sh[r][q][warp] = v;
            }
        __syncthreads();
        if (threadIdx.x < NR * 3) {
            const int r = threadIdx.x / 3, q = threadIdx.x % 3;
            if (r0 + r < nrhs) {
                double t = 0;
                for (int w = 0; w < 4; w++) t += sh[r][q][w];
                partial[((long)(r0 + r) * 3 + q) * (gridDim.x / ntile) + sblk] = t;
            }
        }
    }
}

// one site of dslash_kernel_nr for its right-hand sides r0 .. r0 + NR - 1 (those with act set)
template <int NR, int MODE, typename R, typename SP, typename LK, typename CL>
__device__ __forceinline__ void dslash_site(SP *__restrict__ out, const SP *__restrict__ in,
                                            const LK *__restrict__ U, const CL *__restrict__ F, R kappa,
                                            const Geo &g, long n, int r0, const bool act[NR],
                                            const SP *__restrict__ other, float part[NR][3]) {
    using C = typename CT<R>::C;
    constexpr int PARTS = sizeof(C) * 12 / sizeof(SP);
    const SP *src = in + (long)r0 * PARTS * g.V;
    bool any = false;
#pragma unroll
    for (int r = 0; r < NR; r++) any |= act[r];
    if (!any) return;
    int x[4];
    site_coords(g, n, x);
    C acc[NR][12];
#pragma unroll
    for (int r = 0; r < NR; r++)
#pragma unroll
        for (int k = 0; k < 12; k++) acc[r][k] = cmk<C>(0, 0);
    C psi[12], u[9];
    const R tsgn_f = (x[3] == g.L[3] - 1) ? (R)g.bc_t : (R)1;
    const R tsgn_b = (x[3] == 0) ? (R)g.bc_t : (R)1;
#define QCD_HOP(MU, FWD, SGN)                                                   \
    {                                                                                   \
        const long m = FWD ? nbr_fwd<MU>(g, n, x) : nbr_bwd<MU>(g, n, x);               \
        load_link(U, g.V, FWD ? n : m, MU, u);                                           \
        _Pragma("unroll") for (int r = 0; r < NR; r++) if (act[r]) {                     \
            load_spinor(src + (long)r * PARTS * g.V, m, psi);                      \
            hop_term<MU, FWD>(psi, u, SGN, acc[r]);                                      \
        }                                                                               \
    }
    QCD_HOP(0, true, (R)1)
    QCD_HOP(0, false, (R)1)
    QCD_HOP(1, true, (R)1)
    QCD_HOP(1, false, (R)1)
    QCD_HOP(2, true, (R)1)
    QCD_HOP(2, false, (R)1)
    QCD_HOP(3, true, tsgn_f)
    QCD_HOP(3, false, tsgn_b)
#undef QCD_HOP
    R f[72];
    load_clover(F, g.V, n, f);
#pragma unroll
    for (int r = 0; r < NR; r++) {
        if (act[r]) {
            C fa[12];
            clover_mul<R, C>(f, acc[r], fa);
            load_spinor(src + (long)r * PARTS * g.V, n, psi);
#pragma unroll
            for (int k = 0; k < 12; k++) {
                psi[k].x = fma(-kappa, fa[k].x, psi[k].x);
                psi[k].y = fma(-kappa, fa[k].y, psi[k].y);
            }
            store_spinor(out + (long)(r0 + r) * PARTS * g.V, n, psi);
            if constexpr (MODE != 0) {
                C o[12];
                load_spinor(other + (long)(r0 + r) * PARTS * g.V, n, o);
#pragma unroll
                for (int k = 0; k < 12; k++) {
                    const C a = MODE == 1 ? o[k] : psi[k], b = MODE == 1 ? psi[k] : o[k];
                    part[r][0] = fmaf(a.x, b.x, fmaf(a.y, b.y, part[r][0]));   // Re conj(a) b
                    part[r][1] = fmaf(a.x, b.y, fmaf(-a.y, b.x, part[r][1]));  // Im conj(a) b
                    part[r][2] = fmaf(psi[k].x, psi[k].x, fmaf(psi[k].y, psi[k].y, part[r][2]));
                }
            }
        }
    }
}

// ---- FP64 -----------------------------------------------------------------------------------------
// w = U h (U^dag h) for both spin rows of a half-spinor, added to the w it is given (SUB: subtracted)
template <bool DAG, bool SUB> __device__ __forceinline__ void mul64(const double2 u[9], const double2 h[6], double2 w[6]) {
#pragma unroll
    for (int a = 0; a < 3; a++)
#pragma unroll
        for (int b = 0; b < 3; b++) {
            double2 v = DAG ? u[b * 3 + a] : u[a * 3 + b];
            if (SUB) v = make_double2(-v.x, -v.y);
            w[a] = DAG ? cfmac(v, h[b], w[a]) : cfma(v, h[b], w[a]);
            w[3 + a] = DAG ? cfmac(v, h[3 + b], w[3 + a]) : cfma(v, h[3 + b], w[3 + a]);
        }
}
// a + s b
__device__ __forceinline__ double2 axpy64(double s, double2 b, double2 a) {
    return make_double2(fma(s, b.x, a.x), fma(s, b.y, a.y));
}
// y = H x for the packed chiral block b of F/2 at site n, the large diagonal last
__device__ __forceinline__ void herm6_64(const double2 *__restrict__ F, long V, long n, int b, const double2 x[6],
                                         double2 y[6]) {
    double f[36];
#pragma unroll
    for (int k = 0; k < 18; k++) {
        const double2 v = __ldg(F + (18 * b + k) * V + n);
        f[2 * k] = v.x;
        f[2 * k + 1] = v.y;
    }
    int k = 6;
#pragma unroll
    for (int i = 0; i < 6; i++) {
        y[i] = make_double2(0, 0);
#pragma unroll
        for (int j = 0; j < i; j++) {
            const double2 a = make_double2(f[k], f[k + 1]);
            k += 2;
            y[i] = cfma(a, x[j], y[i]);
            y[j] = cfmac(a, x[i], y[j]);
        }
    }
#pragma unroll
    for (int i = 0; i < 6; i++) y[i] = axpy64(f[i], x[i], y[i]);
}
// D in FP64.  Bound by the FP64 pipe (2 operations per clock and SM, which it reaches), so the order is the
// one with few operations, 1,092 a site (1,176 in the plain order):
//  - t first, the colour products starting the sums (the projector's factor 2 and the boundary sign
//    multiply them when the next hop is added);
//  - along x, y, z the backward product is subtracted from the forward one as it is formed, D = w+ - w-, which is
//    what the lower spins need, and the upper spins add 2 w+ - D: 36 operations instead of 48 for the two
//    reconstructions.
// Together these round a little more (the error against 80-bit arithmetic, of random sites with unitary links
// and a clover term of 0.5 +- 0.03, rises by 3%); the clover's diagonal, its largest entries, added last
// rounds less, and the error ends 15% below that of the plain order (0.94e-16 against 1.12e-16).  Applying the
// second chiral block on top of the first one's result would save 12 more, but raises it by 12%.
// 24^3x48: 1337 -> 1257 us (1497 at first).
__global__ void __launch_bounds__(128, 3) dslash64_kernel(double2 *__restrict__ out, const double2 *__restrict__ in,
                                                          const double2 *__restrict__ U, const double2 *__restrict__ F,
                                                          double kappa, Geo g, int nrhs) {
    chain_wait(in);
    // the right-hand side varies fastest over the (1-D) grid: the CTAs of one site block run
    // together and share its links and clover field through L2
    const long sblk = blockIdx.x / nrhs;
    const int rhs = (int)(blockIdx.x - sblk * nrhs);
    const long n = sblk * blockDim.x + threadIdx.x;
    if (n >= g.V) return;
    const double2 *src = in + (long)rhs * 12 * g.V;
    int x[4];
    site_coords(g, n, x);
    double2 up[6], lo[6], psi[12], u[9];  // the hop sum's upper and lower two spins
#pragma unroll
    for (int k = 0; k < 6; k++) up[k] = lo[k] = make_double2(0, 0);
    {
        const long m = nbr_fwd<3>(g, n, x);
        load_spinor(src, m, psi);
        load_link(U, g.V, n, 3, u);
        mul64<false, false>(u, psi + 6, lo);
    }
    {
        const long m = nbr_bwd<3>(g, n, x);
        load_spinor(src, m, psi);
        load_link(U, g.V, m, 3, u);
        mul64<true, false>(u, psi, up);
    }
    const double sf = x[3] == g.L[3] - 1 ? 2.0 * g.bc_t : 2.0, sb = x[3] == 0 ? 2.0 * g.bc_t : 2.0;
#define QCD_PAIR(MU)                                                                                  \
    {                                                                                                 \
        double2 h[6], w[6], d[6];                                                                     \
        const long mf = nbr_fwd<MU>(g, n, x), mb = nbr_bwd<MU>(g, n, x);                              \
        load_spinor(src, mf, psi);                                                                    \
        load_link(U, g.V, n, MU, u);                                                                  \
        hop_project<MU, true>(psi, 1.0, h);                                                           \
        _Pragma("unroll") for (int k = 0; k < 6; k++) w[k] = make_double2(0, 0);                      \
        mul64<false, false>(u, h, w);                                                                 \
        load_spinor(src, mb, psi);                                                                    \
        load_link(U, g.V, mb, MU, u);                                                                 \
        hop_project<MU, false>(psi, 1.0, h);                                                          \
        _Pragma("unroll") for (int k = 0; k < 6; k++) d[k] = w[k];                                    \
        mul64<true, true>(u, h, d);                                                                   \
        _Pragma("unroll") for (int k = 0; k < 6; k++) {                                               \
            /* lower spins: spin 2 from row 1 (x, y) or 0 (z), spin 3 from the other */               \
            const double2 dk = d[MU == 2 ? k : k < 3 ? k + 3 : k - 3];                                \
            const double2 p = MU == 0 ? cmulmi(dk)                                                    \
                            : MU == 1 ? (k < 3 ? make_double2(-dk.x, -dk.y) : dk)                     \
                                      : (k < 3 ? cmulmi(dk) : cmuli(dk));                             \
            if (MU == 0) {                                                                            \
                up[k] = axpy64(sb, up[k], axpy64(2.0, w[k], make_double2(-d[k].x, -d[k].y)));         \
                lo[k] = axpy64(sf, lo[k], p);                                                         \
            } else {                                                                                  \
                up[k] = axpy64(2.0, w[k], csub(up[k], d[k]));                                         \
                lo[k] = cadd(lo[k], p);                                                               \
            }                                                                                         \
        }                                                                                             \
    }
    QCD_PAIR(0)
    QCD_PAIR(1)
    QCD_PAIR(2)
#undef QCD_PAIR
    // F: e0 = H_0 (up - lo), e1 = H_1 (up + lo); upper spins e0 + e1, lower e1 - e0
    double2 c[6], e0[6], e1[6];
#pragma unroll
    for (int k = 0; k < 6; k++) c[k] = csub(up[k], lo[k]);
    herm6_64(F, g.V, n, 0, c, e0);
#pragma unroll
    for (int k = 0; k < 6; k++) c[k] = cadd(up[k], lo[k]);
    herm6_64(F, g.V, n, 1, c, e1);
    load_spinor(src, n, psi);
#pragma unroll
    for (int k = 0; k < 6; k++) {
        psi[k] = axpy64(-kappa, cadd(e0[k], e1[k]), psi[k]);
        psi[6 + k] = axpy64(-kappa, csub(e1[k], e0[k]), psi[6 + k]);
    }
    store_spinor(out + (long)rhs * 12 * g.V, n, psi);
}

namespace {
// first two rows of every FP32 link
__global__ void k_links_to_rows(float4 *__restrict__ U12, const float2 *__restrict__ U32, long V) {
    const long n = blockIdx.x * (long)blockDim.x + threadIdx.x;
    if (n >= V) return;
    for (int mu = 0; mu < 4; mu++)
        for (int p = 0; p < 3; p++) {
            const float2 a = U32[(mu * 9 + 2 * p) * V + n], b = U32[(mu * 9 + 2 * p + 1) * V + n];
            U12[(mu * 3 + p) * V + n] = make_float4(a.x, a.y, b.x, b.y);
        }
}
// FP16 copies of the FP32 links and clover field
__global__ void k_fields_to_half(__half2 *__restrict__ U16, uint2 *__restrict__ F16, const float2 *__restrict__ U32,
                                 const float4 *__restrict__ F32, long V) {
    const long n = blockIdx.x * (long)blockDim.x + threadIdx.x;
    if (n >= V) return;
    for (int k = 0; k < 36; k++) U16[k * V + n] = __float22half2_rn(U32[k * V + n]);
    for (int k = 0; k < 18; k++) {
        const float4 v = F32[k * V + n];
        const __half2 a = __floats2half2_rn(v.x, v.y), b = __floats2half2_rn(v.z, v.w);
        F16[k * V + n] = make_uint2(*reinterpret_cast<const unsigned *>(&a), *reinterpret_cast<const unsigned *>(&b));
    }
}
}  // namespace

static Geo geo_of(const qcd_ctx *c) {
    Geo g;
    for (int m = 0; m < 4; m++) g.L[m] = c->lat.L[m];
    g.V = c->lat.V;
    g.bc_t = c->bc_t;
    return g;
}

int dslash64(qcd_ctx *c, double2 *out, const double2 *in, int nrhs) {
    Geo g = geo_of(c);
    dim3 grid((unsigned)((g.V + 127) / 128 * nrhs));
    cudaEvent_t ev;
    prof_begin(c, QCD_K_DSLASH64, &ev);
    launch_chained(c, dslash64_kernel, grid, 128, 0, out, in, c->U64, c->F64, c->kappa, g, nrhs);
    return prof_end(c, QCD_K_DSLASH64, ev);
}

// the links as their first two rows (Table 1's SU(3) 12-real form), made on first use after each
// field change
static int ensure_u12(qcd_ctx *c, const Geo &g) {
    if (!c->U12) {
        int rc = dev_alloc(c, (void **)&c->U12, sizeof(float4) * 12 * g.V);
        if (rc) return rc;
    }
    if (c->u12_version != c->field_version) {
        k_links_to_rows<<<(unsigned)((g.V + 255) / 256), 256, 0, c->stream>>>(c->U12, c->U32, g.V);
        field_kernel(c);
        QCD_CUDA(c, cudaGetLastError());
        c->u12_version = c->field_version;
    }
    return QCD_OK;
}

int dslash32_prepare(qcd_ctx *c) { return ensure_u12(c, geo_of(c)); }

// Where the fields and vectors of one t-slice exceed the 126 MB of L2 its blocks are taken in chunks of 32 MB,
// else in order.  us per launch of dslash32_tile, in order -> chunks of 16 / 32 / 48 / 64 MB: 48^3x96, 4 right-hand
// sides (212 MB a slice) 4575 -> 4411 / 4373 / 4432 / 4563, 1 (117 MB) 1451 -> 1374 / 1346 / 1345 / 1350; 40^3x80, 4
// (123 MB) 2248 -> 2150 / 2132 / 2160 / 2217; 32^3x64, 12 (138 MB) 2510 -> 2464 / 2453 / 2488 / 2594; but 40^3x80, 1
// (68 MB) 629 -> 666 / 652 / 654 / 657, 32^3x64, 4 (63 MB) 849 -> 864 / 856 / 874 / 880, 24^3x48, 12 (58 MB) 700 -> 718
// / 714 / 731 / 725.
static BlockOrder block_order(const Geo &g, int nrhs) {
    const long slice = (long)g.L[0] * g.L[1] * g.L[2], site = 288L * nrhs + 768;  // bytes: in, other, out; links, clover
    BlockOrder o;
    if (slice * site > 96L << 20) {
        o.row = (int)std::max(1L, slice / 128);
        o.chunk = (int)std::max(1L, (32L << 20) / (128 * site));
    }
    return o;
}

// The inner solver's D: FP32 with the links in the two-row form (the third row rebuilt in
// registers), one right-hand side per thread, with FP32 accuracy.  A lane's spinor lies 96 bytes from its neighbour
// lane's, so a 32-byte load of a warp touches 24 lines where a plane of the earlier layout took 4, and the kernel
// is slower than it was on planes: 24^3x48 with 12 right-hand sides 700 us against 620, 48^3x96 with 4 4373
// against 3873, with 1 1346 against 1332.  us with 3 / 4 / 5 / 6 / 7 blocks per SM: 24^3x48 with 12 810 / 700 / 730 /
// 711 / 723, 48^3x96 with 4 (in order) 5196 / 4572 / 4802 / 4749 / 4794; two right-hand sides per thread with 3 / 4
// blocks 834 / 815 and 5519 / 5457; full links 813 and 5047, two per thread 834 and 5394; two or four right-hand sides in
// the lanes of a warp 723 to 878 and 4654 to 5261.
template <int MODE>
static int dslash32_tile(qcd_ctx *c, float4 *out, const float4 *in, int nrhs, const float4 *other, double *red,
                         const BicgScalars *gate, const ScalarStep &step) {
    Geo g = geo_of(c);
    const unsigned nblk = (unsigned)((g.V + 127) / 128);
    double *part = MODE ? c->d_red_tiles : nullptr;
    int rc = ensure_u12(c, g);
    if (rc) return rc;
    cudaEvent_t ev;
    prof_begin(c, QCD_K_DSLASH32, &ev);
    const BlockOrder order = block_order(g, nrhs);
    auto kernel = order.chunk ? dslash_kernel_nr<4, 1, float, float4, float4, float4, MODE, true>
                              : dslash_kernel_nr<4, 1, float, float4, float4, float4, MODE>;
    launch_chained(c, kernel, dim3(nblk * nrhs), 128, 0, out, in, c->U12, c->F32, (float)c->kappa, g, nrhs, other, part, gate,
                   order);
    rc = prof_end(c, QCD_K_DSLASH32, ev);
    if (rc || !MODE) return rc;
    return reduce_tiles(c, part, nblk, nrhs, red, step);
}

int dslash32(qcd_ctx *c, float4 *out, const float4 *in, int nrhs) {
    Geo g = geo_of(c);
    cudaEvent_t ev;
    prof_begin(c, QCD_K_DSLASH32, &ev);
    // us with 3 / 4 / 5 / 6 / 7 blocks per SM: one right-hand side on 8^3x16 3.76 / 3.81 / 3.87 / 4.30 / 5.64, 24^3x48 86.6 /
    // 80.3 / 81.9 / 85.9 / 97.5, 48^3x96 1481 / 1434 / 1392 / 1429 / 1584; two per thread: four on 8^3x16 7.02 / 7.26 /
    // 9.83 / 11.2 / 12.3, 48^3x96 4824 / 4407 / 6099 / 7033 / 8238, twelve on 24^3x48 777 / 682 / 1067 / 1280 / 1520
    if (nrhs == 1) {
        launch_chained(c, dslash_kernel<5, float, float4, float2, float4>, dim3((unsigned)((g.V + 127) / 128)), 128, 0,
                       out, in, c->U32, c->F32, (float)c->kappa, g, 1);
    } else {
        dim3 grid((unsigned)((g.V + 127) / 128 * ((nrhs + 1) / 2)));
        launch_chained(c, dslash_kernel_nr<4, 2, float, float4, float2, float4>, grid, 128, 0, out, in, c->U32, c->F32,
                       (float)c->kappa, g, nrhs, nullptr, nullptr, nullptr, BlockOrder());
    }
    return prof_end(c, QCD_K_DSLASH32, ev);
}
int dslash32_dot(qcd_ctx *c, float4 *out, const float4 *in, int nrhs, const float4 *other, int mode, double *red,
                 const BicgScalars *gate, const ScalarStep &step) {
    if (mode == 1) return dslash32_tile<1>(c, out, in, nrhs, other, red, gate, step);
    if (mode == 2) return dslash32_tile<2>(c, out, in, nrhs, other, red, gate, step);
    return dslash32_tile<0>(c, out, in, nrhs, nullptr, nullptr, gate, step);
}

int dslash16(qcd_ctx *c, float4 *out, const float4 *in, int nrhs) {
    Geo g = geo_of(c);
    if (!c->U16) {
        int rc = dev_alloc(c, (void **)&c->U16, sizeof(__half2) * 36 * g.V);
        if (!rc) rc = dev_alloc(c, (void **)&c->F16, sizeof(uint2) * 18 * g.V);
        if (rc) return rc;
    }
    if (c->half_version != c->field_version) {
        k_fields_to_half<<<(unsigned)((g.V + 255) / 256), 256, 0, c->stream>>>(c->U16, c->F16, c->U32, c->F32, g.V);
        field_kernel(c);
        QCD_CUDA(c, cudaGetLastError());
        c->half_version = c->field_version;
    }
    cudaEvent_t ev;
    prof_begin(c, QCD_K_DSLASH32, &ev);
    // us with 3 / 4 / 5 / 6 / 7 blocks per SM: one right-hand side on 8^3x16 3.66 / 3.68 / 3.82 / 3.89 / 4.13, 24^3x48 68.6 /
    // 62.0 / 63.8 / 62.9 / 63.4, 48^3x96 1079 / 977 / 990 / 959 / 965; four on 8^3x16 4.53 / 4.69 / 4.89 / 5.02 / 5.20,
    // 24^3x48 230 / 208 / 212 / 204 / 207, 48^3x96 4041 / 3841 / 3949 / 3720 / 3867; twelve on 24^3x48 668 / 610 / 619 /
    // 586 / 594
    if (nrhs == 1) {
        launch_chained(c, dslash_kernel<4, float, float4, __half2, uint2>, dim3((unsigned)((g.V + 127) / 128)), 128, 0,
                       out, in, c->U16, c->F16, (float)c->kappa, g, 1);
    } else {
        dim3 grid((unsigned)((g.V + 127) / 128 * nrhs));
        launch_chained(c, dslash_kernel_nr<4, 1, float, float4, __half2, uint2>, grid, 128, 0, out, in, c->U16, c->F16,
                       (float)c->kappa, g, nrhs, nullptr, nullptr, nullptr, BlockOrder());
    }
    return prof_end(c, QCD_K_DSLASH32, ev);
}

int dslash12(qcd_ctx *c, float4 *out, const float4 *in, int nrhs) {
    Geo g = geo_of(c);
    if (int rc = ensure_u12(c, g)) return rc;
    cudaEvent_t ev;
    prof_begin(c, QCD_K_DSLASH32, &ev);
    // us with 3 / 4 / 5 / 6 / 7 blocks per SM: one right-hand side on 8^3x16 3.63 / 3.66 / 3.81 / 4.02 / 4.20, 24^3x48 76.9 /
    // 71.7 / 74.4 / 73.7 / 74.9, 48^3x96 1298 / 1184 / 1238 / 1192 / 1197; four on 24^3x48 241 / 213 / 222 / 223 / 224,
    // 48^3x96 4327 / 3900 / 4220 / 4118 / 4179; twelve on 24^3x48 710 / 623 / 657 / 655 / 656
    if (nrhs == 1) {
        launch_chained(c, dslash_kernel<4, float, float4, float4, float4>, dim3((unsigned)((g.V + 127) / 128)), 128, 0,
                       out, in, c->U12, c->F32, (float)c->kappa, g, 1);
    } else {
        dim3 grid((unsigned)((g.V + 127) / 128 * nrhs));
        launch_chained(c, dslash_kernel_nr<4, 1, float, float4, float4, float4>, grid, 128, 0, out, in, c->U12, c->F32,
                       (float)c->kappa, g, nrhs, nullptr, nullptr, nullptr, BlockOrder());
    }
    return prof_end(c, QCD_K_DSLASH32, ev);
}

int dslash(qcd_ctx *c, void *out, const void *in, int prec, int nrhs) {
    switch (prec) {
        case QCD_F64: return dslash64(c, (double2 *)out, (const double2 *)in, nrhs);
        case QCD_F32: return dslash32(c, (float4 *)out, (const float4 *)in, nrhs);
        case QCD_F16: return dslash16(c, (float4 *)out, (const float4 *)in, nrhs);
        case QCD_F32_SU3: return dslash12(c, (float4 *)out, (const float4 *)in, nrhs);
        default: return dslash_x2(c, (double2 *)out, (const float4 *)in, nrhs);
    }
}

}  // namespace qcd
