// K3, right-hand-side tiled thread form of the ll-ordered SSOR block solve (Sec. 3,
// "Inverse of block operator"), for the throughput regime: many SAP blocks and several
// right-hand sides at once.
//
// One CTA per (SAP block, tile of R right-hand sides).  The block spinors of its R right-hand
// sides live in shared memory; two lanes perform one site update for one right-hand side
// (the 8-direction projected hop restricted to the block, the chiral clover product and the
// relaxation), and the dependency levels of the ll order run one after the other with a CTA
// barrier between them (a site's level is one more than the highest level of its earlier
// in-block neighbours, so a level's sites are pairwise non-adjacent and level-by-level
// updating reads exactly the values of the sequential ll sweep).  The R pairs of a site sit
// next to each other in a warp, so the per-site record (transport matrices and clover) they
// share is one set of cache lines for all of them.
//
// What bounds it, and the choices made for it (24^3x48, 4^4 blocks, 4 right-hand sides, FP16, the tuned
// 2 sweeps and one cycle; both colours together):
//  - Of a site's hops only those from the neighbours updated since its last update are formed, half of
//    them; the sum over the others is what the previous pass formed, kept in FP32 in tensor memory, which
//    the kernel has no other use for (12 columns a lane and item; registers and shared memory are full).
//  - Two lanes per site update, one per hop direction and then per chirality and half spinor.  They halve
//    the latency of a level and make its work divide more evenly over the warps: the barrier stalls fell
//    from 2.8 to 0.7 cycles per issued instruction, the issue rate rose from 39% to 49%.  What follows
//    from the warp index is made visibly warp-uniform, which removed a fifth of the instructions.
//  - 926 us against 1098 with one lane per update and all eight hops (243 -> 237 M warp instructions in
//    the first colour's launch at the higher issue rate; FP32, 18x18x12x36, 3^3x6 blocks, 3 right-hand sides:
//    1226 -> 984; FP16, 12^3x24, the same blocks, one right-hand side: 123 -> 109).  Now 60% of
//    the instructions are packed FP32 arithmetic and FP16 conversions at 16 warps per SM (128 registers), the
//    stalls are record loads (2.0) and fixed latencies (1.4).
//
// Records, per block in level order (the order the threads of a level walk), 16-byte aligned:
// the 8 transport matrices W_d (d = 2 mu + backward: U_mu(n) forward, U_mu(n - mu)^dag
// backward) as their first two rows (Table 1's 12-real form; the third row is the conjugate
// cross product of the first two), then the two packed Hermitian chiral blocks of F/2 (72
// reals).  FP32: 672 bytes per site; FP16 storage: 336.  Inside the block a hop that leaves it
// reads an all-zero spinor slot, so D_BB needs no masks; the same matrices serve the hops
// between blocks of opposite colour.
// With FP16 storage the block spinor of each right-hand side, and its source, are kept in
// shared memory in units of the largest |component| of that source on the block (the SSOR
// iteration is linear), so no rescaling is needed inside the sweep; arithmetic is FP32
// throughout.
#include <cuda_fp16.h>

#include <algorithm>
#include <cmath>

#include "fields.cuh"
#include "qcd_internal.h"

namespace qcd {

namespace {

template <bool HALF> struct TileRec {
    static constexpr int link_bytes = HALF ? 24 : 48;             // two rows: 6 complex
    static constexpr int clover_off = 8 * link_bytes;             // 192 / 384
    static constexpr int bytes = clover_off + (HALF ? 144 : 288);  // 336 / 672
    static constexpr int chunks = bytes / 16;
    static constexpr int y_words = HALF ? 12 : 24;  // 4-byte words of one site spinor in shared memory
};
static_assert(TileRec<true>::bytes == kTileRecordBytesHalf && TileRec<false>::bytes == kTileRecordBytes,
              "tile record size");

__device__ __forceinline__ float2 h2f(unsigned w) { return __half22float2(*reinterpret_cast<const __half2 *>(&w)); }
__device__ __forceinline__ unsigned f2h(float2 v) {
    const __half2 h = __float22half2_rn(v);
    return *reinterpret_cast<const unsigned *>(&h);
}

// A site update is shared by the two lanes of a pair (h = 0, 1): in the hops lane h takes the forward or
// the backward neighbours, from the clover term on it takes chirality h, and of the result the upper or
// the lower two spins.

// N words of one spinor in shared memory, as float2 (FP16: half2 words; FP32: two words each)
template <bool HALF, int N> __device__ __forceinline__ void ld_y(const float *p, float2 s[N]) {
    if constexpr (HALF) {
        static_assert(N == 12 || N == 6, "a spinor or half of one");
        if constexpr (N == 12) {
#pragma unroll
            for (int k = 0; k < 3; k++) {
                const uint4 v = reinterpret_cast<const uint4 *>(p)[k];
                s[4 * k] = h2f(v.x); s[4 * k + 1] = h2f(v.y); s[4 * k + 2] = h2f(v.z); s[4 * k + 3] = h2f(v.w);
            }
        } else {
#pragma unroll
            for (int k = 0; k < 3; k++) {
                const uint2 v = reinterpret_cast<const uint2 *>(p)[k];
                s[2 * k] = h2f(v.x); s[2 * k + 1] = h2f(v.y);
            }
        }
    } else {
#pragma unroll
        for (int k = 0; k < N / 2; k++) {
            const float4 v = reinterpret_cast<const float4 *>(p)[k];
            s[2 * k] = make_float2(v.x, v.y);
            s[2 * k + 1] = make_float2(v.z, v.w);
        }
    }
}
// half a spinor into shared memory
template <bool HALF> __device__ __forceinline__ void st_y6(float *p, const float2 s[6]) {
    if constexpr (HALF) {
#pragma unroll
        for (int k = 0; k < 3; k++) reinterpret_cast<uint2 *>(p)[k] = make_uint2(f2h(s[2 * k]), f2h(s[2 * k + 1]));
    } else {
#pragma unroll
        for (int k = 0; k < 3; k++)
            reinterpret_cast<float4 *>(p)[k] = make_float4(s[2 * k].x, s[2 * k].y, s[2 * k + 1].x, s[2 * k + 1].y);
    }
}
// half a spinor in the lattice (48 bytes, 16-byte aligned); data written earlier by the same kernel allowed
__device__ __forceinline__ void ld_half(const float4 *p, float2 s[6]) {
#pragma unroll
    for (int k = 0; k < 3; k++) {
        const float4 v = p[k];
        s[2 * k] = make_float2(v.x, v.y);
        s[2 * k + 1] = make_float2(v.z, v.w);
    }
}
__device__ __forceinline__ void st_half(float4 *p, const float2 s[6]) {
#pragma unroll
    for (int k = 0; k < 3; k++) p[k] = make_float4(s[2 * k].x, s[2 * k].y, s[2 * k + 1].x, s[2 * k + 1].y);
}

// one transport matrix W_d as stored (first two rows), and with the third row rebuilt; d may differ
// between lanes
template <bool HALF> struct LinkRaw {
    unsigned w[HALF ? 6 : 12];
};
template <bool HALF> __device__ __forceinline__ void ld_link(const unsigned char *rec, int d, LinkRaw<HALF> &r) {
    if constexpr (HALF) {
        const uint2 *p = reinterpret_cast<const uint2 *>(rec) + 3 * d;  // 24 bytes, 8-byte aligned
#pragma unroll
        for (int k = 0; k < 3; k++) {
            const uint2 v = __ldg(p + k);
            r.w[2 * k] = v.x; r.w[2 * k + 1] = v.y;
        }
    } else {
        const uint4 *p = reinterpret_cast<const uint4 *>(rec) + 3 * d;
#pragma unroll
        for (int k = 0; k < 3; k++) {
            const uint4 v = __ldg(p + k);
            r.w[4 * k] = v.x; r.w[4 * k + 1] = v.y; r.w[4 * k + 2] = v.z; r.w[4 * k + 3] = v.w;
        }
    }
}
template <bool HALF> __device__ __forceinline__ void link_unpack(const LinkRaw<HALF> &r, float2 W[9]) {
#pragma unroll
    for (int k = 0; k < 6; k++) {
        if constexpr (HALF) W[k] = h2f(r.w[k]);
        else W[k] = make_float2(__uint_as_float(r.w[2 * k]), __uint_as_float(r.w[2 * k + 1]));
    }
    su3_third_row(W);
}

// the packed chiral block h of a record's clover (6 real diagonal entries, then the 15 complex entries
// below the diagonal in row order) as stored.  FP16: 18 half2 words, the first three holding the
// diagonal and each later one a complex entry, converted as they are used
template <bool HALF> struct CloverRaw {
    unsigned w[HALF ? 18 : 36];
};
template <bool HALF> __device__ __forceinline__ void ld_clover(const unsigned char *rec, int h, CloverRaw<HALF> &r) {
    const unsigned char *p = rec + TileRec<HALF>::clover_off;
    if constexpr (HALF) {
        const uint2 *q = reinterpret_cast<const uint2 *>(p + 72 * h);
#pragma unroll
        for (int k = 0; k < 9; k++) {
            const uint2 v = __ldg(q + k);
            r.w[2 * k] = v.x; r.w[2 * k + 1] = v.y;
        }
    } else {
        const uint4 *q = reinterpret_cast<const uint4 *>(p + 144 * h);
#pragma unroll
        for (int k = 0; k < 9; k++) {
            const uint4 v = __ldg(q + k);
            r.w[4 * k] = v.x; r.w[4 * k + 1] = v.y; r.w[4 * k + 2] = v.z; r.w[4 * k + 3] = v.w;
        }
    }
}
// y = H x for that block
template <bool HALF> __device__ __forceinline__ void herm6_rec(const CloverRaw<HALF> &r, const float2 x[6], float2 y[6]) {
    float d[6];
    auto entry = [&](int k) {
        if constexpr (HALF) return h2f(r.w[3 + k]);
        else return make_float2(__uint_as_float(r.w[6 + 2 * k]), __uint_as_float(r.w[7 + 2 * k]));
    };
    if constexpr (HALF) {
#pragma unroll
        for (int k = 0; k < 3; k++) {
            const float2 t = h2f(r.w[k]);
            d[2 * k] = t.x;
            d[2 * k + 1] = t.y;
        }
    } else {
#pragma unroll
        for (int k = 0; k < 6; k++) d[k] = __uint_as_float(r.w[k]);
    }
    // packed FP32 pairs: A_i = sum_j Re(H_ij) x_j, E_i = sum_j s_ij Im(H_ij) x_j with s = +1 below
    // the diagonal (H_ij) and -1 above it (conj(H_ji)); y_i = (A_i.x - E_i.y, A_i.y + E_i.x)
    float2 A[6], E[6];
#pragma unroll
    for (int i = 0; i < 6; i++) {
        A[i] = __fmul2_rn(make_float2(d[i], d[i]), x[i]);
        E[i] = make_float2(0.f, 0.f);
    }
    int k = 0;
#pragma unroll
    for (int i = 1; i < 6; i++) {
#pragma unroll
        for (int j = 0; j < i; j++) {
            const float2 o = entry(k);
            const float2 hr = make_float2(o.x, o.x), hi = make_float2(o.y, o.y);
            A[i] = __ffma2_rn(hr, x[j], A[i]);  // row i gets H_ij x_j
            E[i] = __ffma2_rn(hi, x[j], E[i]);
            A[j] = __ffma2_rn(hr, x[i], A[j]);  // row j gets conj(H_ij) x_i
            E[j] = __ffma2_rn(make_float2(-o.y, -o.y), x[i], E[j]);
            k++;
        }
    }
#pragma unroll
    for (int i = 0; i < 6; i++) y[i] = make_float2(A[i].x - E[i].y, A[i].y + E[i].x);
}

// a + i s b
__device__ __forceinline__ float2 add_is(float2 a, float s, float2 b) {
    return make_float2(fmaf(-s, b.y, a.x), fmaf(s, b.x, a.y));
}
// The hop of fields.cuh along MU with the direction in the lane's sign s (+1: forward, 1 - gamma; -1:
// backward, 1 + gamma), W the transport as it acts.  psi: the neighbour's 12 components; MU = 3: the six
// that the projector keeps (the lower two spins forward, the upper two backward).  The colour multiply
// runs in packed FP32 pairs: for each row a, p = sum_b Re(W_ab) h_b and q = sum_b Im(W_ab) h_b, and
// (W h)_a = (p.x - q.y, p.y + q.x).
template <int MU> __device__ __forceinline__ void hop_pair(const float2 *psi, const float2 W[9], float s, float2 acc[12]) {
    float2 h[6];
    const float2 ss = make_float2(s, s), ms = make_float2(-s, -s);
#pragma unroll
    for (int c = 0; c < 3; c++) {
        if constexpr (MU == 0) {
            h[c] = add_is(psi[c], s, psi[9 + c]);
            h[3 + c] = add_is(psi[3 + c], s, psi[6 + c]);
        } else if constexpr (MU == 1) {
            h[c] = __ffma2_rn(ss, psi[9 + c], psi[c]);
            h[3 + c] = __ffma2_rn(ms, psi[6 + c], psi[3 + c]);
        } else if constexpr (MU == 2) {
            h[c] = add_is(psi[c], s, psi[6 + c]);
            h[3 + c] = add_is(psi[3 + c], -s, psi[9 + c]);
        } else {
            h[c] = cscale(psi[c], 2.f);
            h[3 + c] = cscale(psi[3 + c], 2.f);
        }
    }
#pragma unroll
    for (int a = 0; a < 3; a++) {
        const float2 r0 = make_float2(W[a * 3].x, W[a * 3].x), i0 = make_float2(W[a * 3].y, W[a * 3].y);
        float2 p0 = __fmul2_rn(r0, h[0]), q0 = __fmul2_rn(i0, h[0]);
        float2 p1 = __fmul2_rn(r0, h[3]), q1 = __fmul2_rn(i0, h[3]);
#pragma unroll
        for (int b = 1; b < 3; b++) {
            const float2 rb = make_float2(W[a * 3 + b].x, W[a * 3 + b].x), ib = make_float2(W[a * 3 + b].y, W[a * 3 + b].y);
            p0 = __ffma2_rn(rb, h[b], p0);
            q0 = __ffma2_rn(ib, h[b], q0);
            p1 = __ffma2_rn(rb, h[3 + b], p1);
            q1 = __ffma2_rn(ib, h[3 + b], q1);
        }
        const float2 w0 = make_float2(p0.x - q0.y, p0.y + q0.x), w1 = make_float2(p1.x - q1.y, p1.y + q1.x);
        if constexpr (MU == 3) {
            const float u = s < 0.f ? 1.f : 0.f, l = 1.f - u;
            const float2 uu = make_float2(u, u), ll = make_float2(l, l);
            acc[a] = __ffma2_rn(uu, w0, acc[a]);
            acc[3 + a] = __ffma2_rn(uu, w1, acc[3 + a]);
            acc[6 + a] = __ffma2_rn(ll, w0, acc[6 + a]);
            acc[9 + a] = __ffma2_rn(ll, w1, acc[9 + a]);
            continue;
        }
        acc[a] = cadd(acc[a], w0);
        acc[3 + a] = cadd(acc[3 + a], w1);
        if constexpr (MU == 0) {
            acc[6 + a] = add_is(acc[6 + a], -s, w1);
            acc[9 + a] = add_is(acc[9 + a], -s, w0);
        } else if constexpr (MU == 1) {
            acc[6 + a] = __ffma2_rn(ms, w1, acc[6 + a]);
            acc[9 + a] = __ffma2_rn(ss, w0, acc[9 + a]);
        } else {
            acc[6 + a] = add_is(acc[6 + a], -s, w0);
            acc[9 + a] = add_is(acc[9 + a], s, w1);
        }
    }
}

// The pair's hop sums to chirality h of their total: c = upper -/+ lower (h = 0, 1) of both lanes
__device__ __forceinline__ void pair_chiral(const float2 acc[12], int h, float2 c[6]) {
    const float t = h ? 1.f : -1.f;
    const float2 tt = make_float2(t, t), mt = make_float2(-t, -t);
#pragma unroll
    for (int k = 0; k < 6; k++) {
        const float2 give = __ffma2_rn(mt, acc[k + 6], acc[k]);
        c[k] = __ffma2_rn(tt, acc[k + 6], acc[k]);
        const float2 got = make_float2(__shfl_xor_sync(0xffffffffu, give.x, 1), __shfl_xor_sync(0xffffffffu, give.y, 1));
        c[k] = cadd(c[k], got);
    }
}
// F applied: e = the chiral block on c, then the lane's half of the Dirac spinor, upper = e0 + e1 (h = 0),
// lower = e1 - e0 (h = 1)
template <bool HALF>
__device__ __forceinline__ void pair_clover(const CloverRaw<HALF> &r, const float2 c[6], int h, float2 f[6]) {
    float2 e[6];
    herm6_rec<HALF>(r, c, e);
    const float t = h ? -1.f : 1.f;
    const float2 tt = make_float2(t, t);
#pragma unroll
    for (int k = 0; k < 6; k++) {
        const float2 got = make_float2(__shfl_xor_sync(0xffffffffu, e[k].x, 1), __shfl_xor_sync(0xffffffffu, e[k].y, 1));
        f[k] = __ffma2_rn(tt, got, e[k]);
    }
}

// 12 FP32 columns of this thread's tensor-memory lane (half a spinor)
__device__ __forceinline__ void tmem_st12(uint32_t t, const float2 v[6]) {
    asm volatile("tcgen05.st.sync.aligned.32x32b.x8.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8};" ::"r"(t),
                 "r"(__float_as_uint(v[0].x)), "r"(__float_as_uint(v[0].y)), "r"(__float_as_uint(v[1].x)),
                 "r"(__float_as_uint(v[1].y)), "r"(__float_as_uint(v[2].x)), "r"(__float_as_uint(v[2].y)),
                 "r"(__float_as_uint(v[3].x)), "r"(__float_as_uint(v[3].y))
                 : "memory");
    asm volatile("tcgen05.st.sync.aligned.32x32b.x4.b32 [%0], {%1,%2,%3,%4};" ::"r"(t + 8),
                 "r"(__float_as_uint(v[4].x)), "r"(__float_as_uint(v[4].y)), "r"(__float_as_uint(v[5].x)),
                 "r"(__float_as_uint(v[5].y))
                 : "memory");
    asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ void tmem_ld12(uint32_t t, float2 v[6]) {
    uint32_t r[12];
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
                 : "r"(t));
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0,%1,%2,%3}, [%4];"
                 : "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11])
                 : "r"(t + 8));
    asm volatile("tcgen05.wait::ld.sync.aligned;"
                 : "+r"(r[0]), "+r"(r[1]), "+r"(r[2]), "+r"(r[3]), "+r"(r[4]), "+r"(r[5]), "+r"(r[6]), "+r"(r[7]),
                   "+r"(r[8]), "+r"(r[9]), "+r"(r[10]), "+r"(r[11])::"memory");
#pragma unroll
    for (int k = 0; k < 6; k++) v[k] = make_float2(__uint_as_float(r[2 * k]), __uint_as_float(r[2 * k + 1]));
}

struct TileArgs {
    float4 *x;                 // M_SAP v being accumulated, [nrhs][V][6]
    float4 *r;                 // SAP residual (this colour's sites read and rewritten)
    float4 *y;                 // block solutions: this colour's sites written, the other colour's read
    const float4 *v;           // the SAP input (read in the first cycle)
    const uint4 *rec;          // records of this colour's blocks, [block][vol] x TileRec::bytes
    const int4 *pos;           // [2 passes][vol][2 lanes] per level position (tile_fill_positions): offset from
                               // the block origin; shared-memory slot | mask of the directions mu in which
                               // the lane has a neighbour that the pass updates before the site << 16 | mask
                               // of those leaving the block << 20; slots of the lane's neighbours along
                               // mu = 0 | 1 << 16, 2 | 3 << 16, a zero slot (>= vol) where not in the mask
    const int *coords;         // [vol] block-local coordinates y_mu of a level position, in bytes mu = 0..3
    const int4 *levels;        // [nlev] (first level position, (site, right-hand side) pairs, first warp of the
                               // level's items, its tensor-memory slot)
    const int *origin_site;    // [blocks of this colour] global index of the block origin
    const int *origin;         // [blocks of this colour][4] coordinates of the block origin
    const BicgScalars *gate;   // per right-hand side; inactive ones are skipped (null: all active)
    float kappa, omega;
    long V;
    int L[4], bc_t;
    int vol, nlev, nsweep, nrhs;
    int stride;                // 4-byte words per site in shared memory (the R spinors)
    int zslots;                // zero slots after the vol site slots (hops left out read them)
    int tm_cols;               // tensor-memory columns of the CTA (a power of two)
    int tm_slots;              // slots of 12 columns that a warp has for its items
    int tm_per_warp;           // columns of one warp
    int first;                 // first SAP cycle: the residual starts as v, x as y
    int cross;                 // add the hops from the other colour's last block solutions first
    int store_r;               // the residual is needed by a later cycle
    int store_y;               // the block solutions are needed by the next launch
    // FP16 storage: the block solutions y as FP16 site records [rhs][V] x 48 bytes (the words of
    // the block spinor in shared memory) and their scales [block of either colour][rhs]; the
    // values are y16 x scale, exactly those the kernel holds
    uint4 *y16;
    float *yscale;
    int b[4], nb[4];           // block extents, blocks per direction
    int blk_base, other_base;  // index in yscale of this colour's first block, of the other colour's
};

// N components from k0 on of the other colour's block solution at site mm, in the neighbouring block of rank
// nrank among its colour, for one right-hand side: FP32 in the lattice, or (FP16 storage) the FP16 record
// times its block's scale
template <bool HALF, int N>
__device__ __forceinline__ void load_y_other(const TileArgs &a, int rhs, long mm, int nrank, int k0, float2 psi[N]) {
    if constexpr (HALF) {
        const float sc = a.yscale[(size_t)(a.other_base + nrank) * a.nrhs + rhs];
        const uint2 *q = reinterpret_cast<const uint2 *>(a.y16 + ((size_t)rhs * a.V + mm) * 3) + k0 / 2;
#pragma unroll
        for (int k = 0; k < N / 2; k++) {
            const uint2 v = q[k];
            psi[2 * k] = cscale(h2f(v.x), sc);
            psi[2 * k + 1] = cscale(h2f(v.y), sc);
        }
    } else {
        const float4 *q = a.y + ((size_t)rhs * a.V + mm) * 6 + k0 / 2;
#pragma unroll
        for (int k = 0; k < N / 2; k++) {
            const float4 v = q[k];
            psi[2 * k] = make_float2(v.x, v.y);
            psi[2 * k + 1] = make_float2(v.z, v.w);
        }
    }
}

// One colour of one SAP cycle (Eq. (4), Alg. 1, in residual form) on every block of that colour,
// for the right-hand sides blockIdx.y * R ... + R - 1:
//   prologue  f = r_c (v in the first cycle) + kappa F H_{cc'} y_{c'}   (the hops from the other
//             colour's last block solutions, skipped before any exist)
//   sweeps    y_c = A_cc f: nsweep SSOR sweeps from 0 in ll order, level by level
//   epilogue  x_c += y_c (x_c = y_c in the first cycle), r_c = f - D_cc y_c, y_c stored for the
//             next launch's prologue
// which is Alg. 1's y = K r, w = D y, x += y, r -= w term by term, with the cross hops of each
// colour applied by the launch that next reads them.
//
// A warp item is 16 (site, right-hand side) pairs of one level, two lanes each; the items of a level are
// dealt to the warps in turn, the same in every pass, so a lane meets the same sites throughout and
// keeps what it needs of them in its own tensor-memory columns.  ALL: every item has a slot there.
// FLAT: the prologue and the epilogue take the block in one go, not level by level (tile_flat).
template <bool HALF, int R, bool ALL, bool FLAT = false>
__global__ void __launch_bounds__(kTileMaxThreads, kTileMinBlocks) k_sap_tile(TileArgs a) {
    chain_wait();
    using L = TileRec<HALF>;
    extern __shared__ __align__(16) float sm[];
    __shared__ float scale_s[R];
    __shared__ int act_s[R];
    __shared__ int nrank_s[8];  // rank among its colour of the neighbouring block in direction d
    __shared__ uint32_t tm_base_s;
    const int tid = threadIdx.x, T = blockDim.x;
    const int blk = blockIdx.x, rhs0 = blockIdx.y * R;
    if (tid < R) {
        const int r = rhs0 + tid;
        act_s[tid] = r < a.nrhs && (!a.gate || a.gate[r].active);
        scale_s[tid] = 0.f;
    }
    if (tid < 8) {
        // the block one step along mu = tid / 2, forward for even tid (periodic in the block
        // grid).  Blocks of one colour are listed in lexicographic order (x fastest) and alternate
        // in colour along x, whose block count is even: the rank among its colour is lex / 2.
        const int mu = tid >> 1;
        int cb[4];
        for (int m = 0; m < 4; m++) cb[m] = a.origin[4 * blk + m] / a.b[m];
        if (tid & 1) cb[mu] = cb[mu] == 0 ? a.nb[mu] - 1 : cb[mu] - 1;
        else cb[mu] = cb[mu] + 1 == a.nb[mu] ? 0 : cb[mu] + 1;
        nrank_s[tid] = (cb[0] + a.nb[0] * (cb[1] + a.nb[1] * (cb[2] + a.nb[2] * cb[3]))) >> 1;
    }
    __syncthreads();
    bool any = false;
#pragma unroll
    for (int r = 0; r < R; r++) any |= act_s[r] != 0;
    if (!any) return;  // uniform over the CTA
    // The allocation waits while other CTAs of the SM hold the columns; they give them back without
    // depending on this one.
    if (tid < 32) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                         (uint32_t)__cvta_generic_to_shared(&tm_base_s)),
                     "r"(a.tm_cols)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    const long n0 = a.origin_site[blk];
    const uint4 *recb = a.rec + (size_t)blk * a.vol * L::chunks;
    // [vol + zslots][R spinors]: a site's slot (pa.y) is a permutation of the block-local sites
    // chosen against bank conflicts; slots vol ... vol + zslots - 1 stay zero
    float *ys = sm;
    // FP16 storage: the block's source f in the same units and slots after the spinors
    float *fs = ys + (size_t)(a.vol + a.zslots) * a.stride;
    {
        float4 *y4 = reinterpret_cast<float4 *>(ys);
        const int nz = (a.vol + a.zslots) * a.stride / 4;
        for (int i = tid; i < nz; i += T) y4[i] = make_float4(0.f, 0.f, 0.f, 0.f);
    }
    // (the warp index by shuffle: the compiler then knows what follows from it to be warp-uniform)
    int lane;
    asm volatile("mov.u32 %0, %%laneid;" : "=r"(lane));
    const int warp = __shfl_sync(0xffffffffu, tid >> 5, 0), nwarp = T >> 5;
    const int h = lane & 1;                // the lane's direction, then chirality, then half of the spinor
    const float sgn = h ? -1.f : 1.f;
    const int r_me = (lane >> 1) % R;      // every pair this thread takes has right-hand side r_me
    const bool me_active = act_s[r_me] != 0;
    // this right-hand side's residual, source and solution from the block origin, the lane's half
    const size_t roff = ((size_t)(rhs0 + r_me) * a.V + n0) * 6 + 3 * h;
    float4 *rr = a.r + roff;
    const int *org = a.origin + 4 * blk;
    const int y_me = r_me * L::y_words, half_w = h * (L::y_words / 2);
    const int top = a.nlev - 1;
    __syncthreads();  // the tensor-memory base; the zeroed slots
    // this warp's lane quarter of tensor memory, and its columns there
    const uint32_t tm = tm_base_s + ((uint32_t)(warp & 3) << 21) + (uint32_t)((warp >> 2) * a.tm_per_warp);

    const bool warp_active = __any_sync(0xffffffffu, me_active);
    const int pair = lane >> 1;
    const unsigned char *rech = reinterpret_cast<const unsigned char *>(recb);
    constexpr int LB = L::link_bytes;
    // the link words of the lane's direction along mu, its clover block, in the record of a position
    auto rec_of = [&](int pos) { return rech + (size_t)(unsigned)(pos * L::bytes); };
    auto load_link = [&](const unsigned char *rec, int mu, LinkRaw<HALF> &r) { ld_link<HALF>(rec + LB * h, 2 * mu, r); };

    // the first step of the sweeps, level 0 from y = 0 all around: y = omega f (and again where the block
    // has that one level only)
    auto first_update = [&](float *yp, const float2 fv[6]) {
        const float2 om = make_float2(a.omega, a.omega);
        float2 yo[6];
#pragma unroll
        for (int q = 0; q < 6; q++) yo[q] = __fmul2_rn(om, fv[q]);
        for (int n = 1; top == 0 && n < 2 * a.nsweep; n++)
#pragma unroll
            for (int q = 0; q < 6; q++) {
                if constexpr (HALF) yo[q] = h2f(f2h(yo[q]));  // as stored between the two
                yo[q] = __ffma2_rn(om, __fadd2_rn(fv[q], make_float2(-yo[q].x, -yo[q].y)), yo[q]);
            }
        st_y6<HALF>(yp, yo);
    };
    float *const yh = ys + y_me + half_w, *const fh = fs + y_me + half_w;  // the lane's half in slot 0

    // ---- prologue: f = r (or v) + kappa F H_{cc'} y_{c'} on the block's sites ----
    // FP16: f waits in tensor memory (in r without a slot) until the scale is known; r holds it where the
    // epilogue needs it.  FP32: r holds it
    constexpr bool f_tm = HALF && ALL;
    const bool f_r = !f_tm || a.store_r;
    const float4 *src = a.first ? a.v + roff : rr;
    float m = 0.f;  // largest |component| of f seen by this thread (FP16 scale)
    for (int l = 0; l <= (FLAT ? 0 : top); l++) {
        const int4 lv = FLAT ? make_int4(0, a.vol * R, 0, 0) : __ldg(a.levels + l);
        int slot = lv.w + (warp < lv.z);
        for (int j = warp < lv.z ? warp - lv.z + nwarp : warp - lv.z; j * 16 < lv.y; j += nwarp, slot++) {
            if (!warp_active) continue;
            const int i = j * 16 + pair;
            const bool mine = i < lv.y && me_active;
            const int pos = lv.x + (i < lv.y ? i : 0) / R;
            const int4 pt = __ldg(a.pos + 2 * pos + h);
            float2 f[6], base[6];
            if (mine) ld_half(src + 6 * (long)pt.x, base);
#pragma unroll
            for (int k = 0; k < 6; k++) f[k] = make_float2(0.f, 0.f);
            const unsigned out = mine && a.cross ? (unsigned)pt.y >> 20 : 0u;  // where the lane's hop leaves the block
            if (__any_sync(0xffffffffu, out)) {
                const long st[4] = {1, a.L[0], (long)a.L[0] * a.L[1], (long)a.L[0] * a.L[1] * a.L[2]};
                const int xl = __ldg(a.coords + pos);
                const unsigned char *rec = rec_of(pos);
                CloverRaw<HALF> cl;
                ld_clover<HALF>(rec, h, cl);
                float2 acc[12];
#pragma unroll
                for (int k = 0; k < 12; k++) acc[k] = make_float2(0.f, 0.f);
#define QCD_TILE_CROSS(MU)                                                                                        \
                if (out >> MU & 1) {                                                                              \
                    constexpr int N = MU == 3 ? 6 : 12;                                                           \
                    float2 W[9], psi[N];                                                                          \
                    LinkRaw<HALF> raw;                                                                            \
                    load_link(rec, MU, raw);                                                                      \
                    const int xg = org[MU] + ((xl >> (8 * MU)) & 255); /* global coordinate */                    \
                    const bool wrap = xg == (h ? 0 : a.L[MU] - 1);                                                \
                    const long step = h ? -st[MU] : st[MU];                                                       \
                    const long mm = n0 + pt.x + (wrap ? -step * (a.L[MU] - 1) : step);                            \
                    load_y_other<HALF, N>(a, rhs0 + r_me, mm, nrank_s[2 * MU + h], MU == 3 && !h ? 6 : 0, psi);   \
                    if (MU == 3 && wrap) {                                                                        \
                        _Pragma("unroll") for (int k = 0; k < N; k++) psi[k] = cscale(psi[k], (float)a.bc_t);     \
                    }                                                                                             \
                    link_unpack<HALF>(raw, W);                                                                    \
                    hop_pair<MU>(psi, W, sgn, acc);                                                               \
                }
                QCD_TILE_CROSS(0)
                QCD_TILE_CROSS(1)
                QCD_TILE_CROSS(2)
                QCD_TILE_CROSS(3)
#undef QCD_TILE_CROSS
                __syncwarp();
                float2 c[6];
                pair_chiral(acc, h, c);
                pair_clover<HALF>(cl, c, h, f);  // f = F H_{cc'} y for now
            }
            if (mine) {
#pragma unroll
                for (int k = 0; k < 6; k++) {
                    f[k].x = fmaf(a.kappa, f[k].x, base[k].x);
                    f[k].y = fmaf(a.kappa, f[k].y, base[k].y);
                    if constexpr (HALF) m = fmaxf(m, fmaxf(fabsf(f[k].x), fabsf(f[k].y)));
                }
                if (f_r) st_half(rr + 6 * (long)pt.x, f);
                if constexpr (!HALF)
                    if (FLAT ? pos < __ldg(a.levels).y / R : l == 0) first_update(yh + (pt.y & 0xffff) * a.stride, f);
            }
            __syncwarp();
            if (f_tm) tmem_st12(tm + 12 * slot, f);
        }
    }
    float inv_scale = 1.f, my_scale = 1.f;
    if constexpr (HALF) {
        m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, 1));
#pragma unroll
        for (int o = 16; o >= 2 * R; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
        if (lane < 2 * R && h == 0) atomicMax(reinterpret_cast<int *>(&scale_s[lane >> 1]), __float_as_int(m));
    }
    __syncthreads();  // f is whole (and the FP16 scales are known)
    if constexpr (HALF) {
        my_scale = scale_s[r_me] > 0.f ? scale_s[r_me] : 1.f;
        inv_scale = 1.f / my_scale;
        // the source of the sweeps into shared memory, in the right-hand side's units, by the lanes
        // that hold it
        for (int l = 0; l <= (FLAT ? 0 : top); l++) {
            const int4 lv = FLAT ? make_int4(0, a.vol * R, 0, 0) : __ldg(a.levels + l);
            int slot = lv.w + (warp < lv.z);
            for (int j = warp < lv.z ? warp - lv.z + nwarp : warp - lv.z; j * 16 < lv.y; j += nwarp, slot++) {
                if (!warp_active) continue;
                const int i = j * 16 + pair;
                const bool mine = i < lv.y && me_active;
                const int pos = lv.x + (i < lv.y ? i : 0) / R;
                const int4 pt = __ldg(a.pos + 2 * pos + h);
                float2 f[6];
                if constexpr (f_tm) tmem_ld12(tm + 12 * slot, f);
                else if (mine) ld_half(rr + 6 * (long)pt.x, f);
                if (mine) {
#pragma unroll
                    for (int k = 0; k < 6; k++) f[k] = h2f(f2h(cscale(f[k], inv_scale)));
                    st_y6<true>(fh + (pt.y & 0xffff) * a.stride, f);
                    if (FLAT ? pos < __ldg(a.levels).y / R : l == 0) first_update(yh + (pt.y & 0xffff) * a.stride, f);
                }
                __syncwarp();
            }
        }
    }

    constexpr int NRAW = HALF ? 4 : 2;  // links loaded ahead
    auto load_links = [&](unsigned need, const unsigned char *rec, LinkRaw<HALF> raw[NRAW]) {
#pragma unroll
        for (int mu = 0; mu < NRAW; mu++)
            if (need >> mu & 1) load_link(rec, mu, raw[mu]);
    };
    // the lane's hops of the directions mu in `need` (the warp's; where the lane has none its neighbour is a
    // zero slot), summed over the pair: its chirality
    const float *const yn = ys + y_me;
    auto hops = [&](unsigned need, const unsigned char *rec, const int4 &pt, LinkRaw<HALF> raw[NRAW], float2 c[6]) {
        float2 acc[12];
#pragma unroll
        for (int k = 0; k < 12; k++) acc[k] = make_float2(0.f, 0.f);
#define QCD_TILE_HOP(MU)                                                                       \
        if (need >> MU & 1) {                                                                  \
            constexpr int N = MU == 3 ? 6 : 12;                                                \
            float2 W[9], psi[N];                                                               \
            const int nw_ = MU < 2 ? pt.z : pt.w;                                              \
            const int q = MU & 1 ? (int)((unsigned)nw_ >> 16) : nw_ & 0xffff;                  \
            ld_y<HALF, N>(yn + q * a.stride + (MU == 3 ? L::y_words / 2 - half_w : 0), psi);   \
            link_unpack<HALF>(raw[HALF ? MU : MU & 1], W);                                     \
            if (!HALF && MU < 2 && (need >> (MU + 2) & 1)) load_link(rec, MU + 2, raw[MU & 1]); \
            hop_pair<MU>(psi, W, sgn, acc);                                                    \
        } else if (!HALF && MU < 2 && (need >> (MU + 2) & 1)) {                                \
            load_link(rec, MU + 2, raw[MU & 1]);                                               \
        }
        QCD_TILE_HOP(0)
        QCD_TILE_HOP(1)
        QCD_TILE_HOP(2)
        QCD_TILE_HOP(3)
#undef QCD_TILE_HOP
        pair_chiral(acc, h, c);
    };

    // The timeline: forward over the levels and back, nsweep times, then the epilogue, level by level
    // in one body.  At a site the hop sum is that over the neighbours of one side (the earlier ones in a
    // forward pass, the later ones in a backward pass: those updated since the site was last) plus
    // that over the other side, which is still what the previous pass summed there and is taken
    // from tensor memory where it was kept.  The first forward pass starts from y = 0, where the
    // later neighbours add nothing; at the turn of a sweep a level repeats with the same
    // neighbours, so its hops serve both updates.
    int l = top > 0 ? 1 : 0, sw = 0;
    bool fwd = true, ep = top == 0;
    while (l <= top && (!ep || a.store_r)) {
        const bool more = sw + 1 < a.nsweep;
        const int rep = !ep && (fwd ? l == top : l == 0 && more) ? 2 : 1;
        // (the last level has no later neighbours, the first no earlier ones)
        const bool other = (ep || !fwd || sw > 0) && l != (fwd ? top : 0), keep = !ep && (fwd || more || (!FLAT && a.store_r));
        const int4 lv = FLAT && ep ? make_int4(0, a.vol * R, 0, 0) : __ldg(a.levels + l);
        const int4 *posp = a.pos + (fwd ? 0 : 2 * a.vol) + h;
        int j = warp < lv.z ? warp - lv.z + nwarp : warp - lv.z, slot = lv.w + (warp < lv.z);
        // what does not depend on the other warps is loaded before the barrier
        LinkRaw<HALF> raw[NRAW];
        int4 pt = make_int4(0, 0, 0, 0);
        int pos = 0;
        bool mine = false;
        unsigned need = 0;
        auto fetch = [&]() {
            const int i = j * 16 + pair;
            mine = i < lv.y && me_active;
            pos = lv.x + (i < lv.y ? i : 0) / R;
            pt = __ldg(posp + 2 * pos);
            need = __reduce_or_sync(0xffffffffu, (unsigned)pt.y >> 16 & 15u);
            load_links(need, rec_of(pos), raw);
        };
        bool have = warp_active && j * 16 < lv.y;
        if (have) fetch();
        if (!ep || l == 0) __syncthreads();
        while (have) {
            const unsigned char *rec = rec_of(pos);
            const bool cached = ALL || slot < a.tm_slots;
            const uint32_t tslot = tm + 12 * (cached ? slot : a.tm_slots);
            bool add = other && cached;  // the other side's sum is in tensor memory
            float2 c[6], fa[6];  // fa: F H_BB y (FP16: in the units of the right-hand side's scale)
            bool done = false;
            if constexpr (!ALL || FLAT) {
                // no slot, or the epilogue in one go: sum the other side too, and set it aside
                if (FLAT ? ep : other && !cached) {
                    const int4 po = __ldg(a.pos + (fwd ? 2 * a.vol : 0) + h + 2 * pos);
                    const unsigned no = __reduce_or_sync(0xffffffffu, (unsigned)po.y >> 16 & 15u);
                    if (FLAT || no) {
                        add = done = true;
#pragma unroll 1
                        for (int side = 0; side < 2; side++) {
                            load_links(side ? need : no, rec, raw);
                            hops(side ? need : no, rec, side ? pt : po, raw, c);
                            if (side == 0) tmem_st12(tslot, c);
                        }
                    }
                }
            }
            if (!done) hops(need, rec, pt, raw, c);
            CloverRaw<HALF> cl;
            ld_clover<HALF>(rec, h, cl);
            {
                float2 sum[6];
#pragma unroll
                for (int q = 0; q < 6; q++) sum[q] = make_float2(0.f, 0.f);
                if (add) tmem_ld12(tslot, sum);
                if (keep && cached) tmem_st12(tslot, c);
#pragma unroll
                for (int q = 0; q < 6; q++) sum[q] = cadd(c[q], sum[q]);
                pair_clover<HALF>(cl, sum, h, fa);
            }
            if (mine) {
                const int own = (pt.y & 0xffff) * a.stride;
                float *yp = yh + own;
                float2 fv[6], yo[6];
                ld_y<HALF, 6>(yp, yo);
                const float2 kap = make_float2(a.kappa, a.kappa);
                if (!ep) {
                    // y <- y + omega (f + kappa F H y - y), packed FP32 pairs
                    if constexpr (HALF) ld_y<true, 6>(fh + own, fv);
                    else ld_half(rr + 6 * (long)pt.x, fv);
                    const float2 om = make_float2(a.omega, a.omega);
#pragma unroll
                    for (int q = 0; q < 6; q++) {
                        fv[q] = __ffma2_rn(kap, fa[q], fv[q]);
                        yo[q] = __ffma2_rn(om, __fadd2_rn(fv[q], make_float2(-yo[q].x, -yo[q].y)), yo[q]);
                    }
                    if (rep > 1) {
#pragma unroll
                        for (int q = 0; q < 6; q++) {
                            if constexpr (HALF) yo[q] = h2f(f2h(yo[q]));  // as stored between the two
                            yo[q] = __ffma2_rn(om, __fadd2_rn(fv[q], make_float2(-yo[q].x, -yo[q].y)), yo[q]);
                        }
                    }
                    st_y6<HALF>(yp, yo);
                } else {
                    // ---- epilogue: r = f - D_BB y = f - y + kappa F H_BB y ----
                    ld_half(rr + 6 * (long)pt.x, fv);
#pragma unroll
                    for (int q = 0; q < 6; q++) {
                        if constexpr (HALF) {
                            fa[q] = cscale(fa[q], my_scale);
                            yo[q] = cscale(yo[q], my_scale);
                        }
                        fa[q] = csub(__ffma2_rn(kap, fa[q], fv[q]), yo[q]);
                    }
                    st_half(rr + 6 * (long)pt.x, fa);
                }
            }
            __syncwarp();
            j += nwarp;
            slot++;
            have = j * 16 < lv.y;
            if (have) fetch();
        }
        // the next step
        if (FLAT && ep) break;
        if (ep || (fwd && l < top)) {
            l++;
        } else if (fwd) {
            fwd = false;
            l--;
        } else if (l > 0) {
            l--;
        } else {
            fwd = true;
            if (more) l = 1;
            else ep = true;
            sw++;
        }
    }
    __syncthreads();
    if (warp == 0)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tm_base_s), "r"(a.tm_cols));
    // ---- epilogue: x += y, y to the lattice; a lane takes what it likes ----
    if (me_active)
        for (int i = tid >> 1; i < a.vol * R; i += T / 2) {
            const int4 pt = __ldg(a.pos + 2 * (i / R) + h);
            const float *yp = yh + (pt.y & 0xffff) * a.stride;
            float2 yv[6];
            ld_y<HALF, 6>(yp, yv);
            if constexpr (HALF) {
#pragma unroll
                for (int q = 0; q < 6; q++) yv[q] = cscale(yv[q], my_scale);
            }
            if (a.store_y) {
                if constexpr (HALF) {
                    // the FP16 words as they are; the scale is written once per block below
                    const uint2 *w = reinterpret_cast<const uint2 *>(yp);
                    uint2 *dst = reinterpret_cast<uint2 *>(a.y16 + ((size_t)(rhs0 + r_me) * a.V + n0 + pt.x) * 3) + 3 * h;
                    dst[0] = w[0];
                    dst[1] = w[1];
                    dst[2] = w[2];
                } else {
                    st_half(a.y + roff + 6 * (long)pt.x, yv);
                }
            }
            float4 *xr = a.x + roff + 6 * (long)pt.x;
            if (!a.first) {
                float2 xv[6];
                ld_half(xr, xv);
#pragma unroll
                for (int q = 0; q < 6; q++) yv[q] = cadd(xv[q], yv[q]);
            }
            st_half(xr, yv);
        }
    if constexpr (HALF) {
        if (a.store_y && tid < R && act_s[tid])
            a.yscale[(size_t)(a.blk_base + blk) * a.nrhs + rhs0 + tid] = scale_s[tid] > 0.f ? scale_s[tid] : 1.f;
    }
}

// Records of every block (colour 0 blocks first), one thread per (block, level position).
template <bool HALF>
__global__ void k_tile_records(uint4 *__restrict__ rec, const float2 *__restrict__ U, const float4 *__restrict__ F,
                               Geo g, int4 bdim, int vol, const int *__restrict__ site, const int *__restrict__ org0,
                               const int *__restrict__ org1, int nblk0, long total) {
    using L = TileRec<HALF>;
    const long i = blockIdx.x * (long)blockDim.x + threadIdx.x;
    if (i >= total) return;
    const int gb = (int)(i / vol), p = (int)(i % vol);
    const int *o = gb < nblk0 ? org0 + 4 * gb : org1 + 4 * (gb - nblk0);
    const int b[4] = {bdim.x, bdim.y, bdim.z, bdim.w};
    int y[4], r = __ldg(site + p);  // the block-local site of the position
    for (int m = 0; m < 4; m++) { y[m] = r % b[m]; r /= b[m]; }
    const long gs[4] = {1, g.L[0], (long)g.L[0] * g.L[1], (long)g.L[0] * g.L[1] * g.L[2]};
    long n = 0;
    for (int m = 0; m < 4; m++) n += gs[m] * (o[m] + y[m]);
    unsigned char *R = reinterpret_cast<unsigned char *>(rec + (size_t)i * L::chunks);
    for (int d = 0; d < 8; d++) {
        const int mu = d >> 1;
        const bool fwd = (d & 1) == 0;
        // the backward link of a site on the lattice's lower face wraps around (periodic links)
        const long src = fwd ? n : (o[mu] + y[mu] == 0 ? n + (long)(g.L[mu] - 1) * gs[mu] : n - gs[mu]);
        for (int k = 0; k < 6; k++) {  // rows 0, 1 of W
            const int ra = k / 3, cb = k % 3;
            float2 w;
            if (fwd) {
                w = U[(long)(mu * 9 + ra * 3 + cb) * g.V + src];
            } else {
                w = U[(long)(mu * 9 + cb * 3 + ra) * g.V + src];
                w.y = -w.y;
            }
            if constexpr (HALF) reinterpret_cast<unsigned *>(R + d * L::link_bytes)[k] = f2h(w);
            else reinterpret_cast<float2 *>(R + d * L::link_bytes)[k] = w;
        }
    }
    for (int k = 0; k < 18; k++) {
        const float4 v = F[(long)k * g.V + n];
        if constexpr (HALF) {
            reinterpret_cast<uint2 *>(R + L::clover_off)[k] =
                make_uint2(f2h(make_float2(v.x, v.y)), f2h(make_float2(v.z, v.w)));
        } else {
            reinterpret_cast<float4 *>(R + L::clover_off)[k] = v;
        }
    }
}

template <bool HALF> constexpr int y_bytes_per_site() { return TileRec<HALF>::y_words * 4; }

}  // namespace

size_t tile_smem_bytes(const SapPlan &p, int R) {
    // the block spinors of R right-hand sides and the zero slots; FP16 storage: and the sources
    return p.half ? (size_t)(2 * p.vol + p.tile_zslots) * R * y_bytes_per_site<true>()
                  : (size_t)(p.vol + p.tile_zslots) * R * y_bytes_per_site<false>();
}

namespace {

// Shared-memory wavefronts of the kernel's 16-byte spinor loads with R right-hand sides, for
// the positions and slots in p.h_tile_pos.  The loads of a warp go in four phases of eight
// consecutive lanes: four pairs, the first lane of each reading its site's forward neighbour along mu and
// the second its backward one.  The pairs of a level take its (position, right-hand side) items in
// order; a phase's wavefronts are the most distinct 16-byte addresses that fall on one group of four
// banks.
long tile_bank_cost(const SapPlan &p, int R) {
    const int yw = p.half ? TileRec<true>::y_words : TileRec<false>::y_words, S = R * yw;
    long cost = 0;
    for (int l = 0; l < p.nsteps; l++) {
        const int p0 = p.h_step_ptr[l], n = (p.h_step_ptr[l + 1] - p0) * R;
        for (int i0 = 0; i0 < n; i0 += 4)
            for (int pm = 0; pm < 8; pm++) {
                const int pass = pm >> 2, mu = pm & 3;
                int cnt[8] = {0, 0, 0, 0, 0, 0, 0, 0}, addr[8], na = 0;
                for (int i = i0; i < n && i < i0 + 4; i++) {
                    const int pos = p0 + i / R, r = i % R;
                    for (int h = 0; h < 2; h++) {
                        const int4 pt = p.h_tile_pos[(size_t)(pass * p.vol + pos) * 2 + h];
                        const unsigned w = mu < 2 ? pt.z : pt.w;
                        const int a = (int)(mu & 1 ? w >> 16 : w & 0xffff) * S + r * yw + (mu == 3 && !h ? yw / 2 : 0);
                        bool seen = false;
                        for (int k = 0; k < na; k++) seen = seen || addr[k] == a;
                        if (!seen) {
                            addr[na++] = a;
                            cnt[(a / 4) % 8]++;
                        }
                    }
                }
                cost += *std::max_element(cnt, cnt + 8);
            }
    }
    return cost;
}

// One arrangement of the tile positions: the order of the sites within each level, the slot of
// every site, and the residue (mod 8) that the zero slot of each out-of-block hop should have.
struct TileLayout {
    std::vector<int> order, slot;
    std::vector<int> zres;  // [vol][8]
};

// p.h_tile_pos and p.h_tile_site from a layout.  A neighbour that the pass does not update before the
// site, or that lies outside the block, is replaced by the zero slot vol + k, 0 <= k < zslots, of its own
// bank class (vol + k = its slot, or zres, mod zslots).  A block extent above 255 does not pack:
// tile_positions_valid then rejects the table and the plan takes another form.
void tile_fill_positions(SapPlan &p, const TileLayout &t) {
    const int Z = p.tile_zslots, vol = p.vol;
    p.h_tile_pos.assign(4 * (size_t)vol, make_int4(0, 0, 0, 0));
    p.h_tile_site.assign(2 * (size_t)vol, 0);
    std::vector<int> lev(vol);
    for (int l = 0; l < p.nsteps; l++)
        for (int k = p.h_step_ptr[l]; k < p.h_step_ptr[l + 1]; k++) lev[p.h_step_site[k]] = l;
    auto zero = [&](int c) { return vol + (((c - vol) % Z) + Z) % Z; };
    for (int k = 0; k < vol; k++) {
        const int yl = t.order[k];
        int y[4], r = yl;
        for (int m = 0; m < 4; m++) { y[m] = r % p.b[m]; r /= p.b[m]; }
        p.h_tile_site[k] = yl;
        p.h_tile_site[vol + k] = (int)((unsigned)y[0] | (unsigned)y[1] << 8 | (unsigned)y[2] << 16 | (unsigned)y[3] << 24);
        for (int pass = 0; pass < 2; pass++)
            for (int h = 0; h < 2; h++) {
                unsigned nb[4], fresh = 0, out = 0;
                for (int m = 0, stride = 1; m < 4; stride *= p.b[m], m++) {
                    const bool in = h ? y[m] > 0 : y[m] + 1 < p.b[m];
                    const int q = h ? yl - stride : yl + stride;
                    if (!in) out |= 1u << m;
                    // levels of neighbours differ: earlier ones count in the forward pass
                    const bool count = in && (lev[q] < lev[yl]) == (pass == 0);
                    if (count) fresh |= 1u << m;
                    nb[m] = count ? t.slot[q] : zero(in ? t.slot[q] : t.zres[8 * yl + 2 * m + h]);
                }
                p.h_tile_pos[(size_t)(pass * vol + k) * 2 + h] =
                    make_int4(p.h_site_off[yl], (int)((unsigned)t.slot[yl] | fresh << 16 | out << 20), (int)(nb[0] | nb[1] << 16),
                              (int)(nb[2] | nb[3] << 16));
            }
    }
}

}  // namespace

// The tile kernel reads, for the four pairs of a phase (consecutive items of one level), the slots of
// their sites' forward and backward neighbours along one direction.  A spinor of slot q starts at bank
// group (q R y_words / 4 + 3 r) mod 8 for right-hand side r, which with the FP16 spinor
// (12 words) depends on q mod 2 for R = 4, q mod 4 for R = 2 and q mod 8 for R = 1: the reads of
// a phase are free of conflicts when the slots it reads fall in distinct classes.  Three layouts are
// weighed by the simulated wavefronts:
//  - the ll order itself, slot = block-local site;
//  - two by sub-block class: with Y the sub-block coordinate and z the site's place in its sub-block, a
//    site's class is g = (Y_0 + 2 Y_1 + 4 Y_2) mod 8, or the parity of Y (which tells a site's forward
//    neighbour from its backward one in every direction) with the lowest bits of Y_1 and Y_2, and its slot
//    is 8 times its rank among the sites of its class plus g (when the classes are equally large).  The
//    sites of a level are taken by z, and within one z round-robin over the classes.  Sites of equal
//    z hop alike: within their sub-blocks (class kept) or into the next (class moved alike), so
//    the neighbour reads of a phase stay in distinct classes too, and a hop that is left out reads the
//    zero slot of the class it would have reached.
// The order of the sites within a level is free: no site of a level depends on another of it.
void tile_make_positions(SapPlan &p) {
    const int vol = p.vol;
    p.tile_zslots = p.half ? kTileZeroSlotsHalf : kTileZeroSlots;
    int st[4];
    st[0] = 1;
    for (int m = 1; m < 4; m++) st[m] = st[m - 1] * p.b[m - 1];
    TileLayout ll;
    ll.order.assign(p.h_step_site.begin(), p.h_step_site.end());
    ll.slot.resize(vol);
    ll.zres.resize(8 * (size_t)vol);
    for (int yl = 0; yl < vol; yl++) {
        ll.slot[yl] = yl;
        for (int m = 0; m < 4; m++) {
            ll.zres[8 * yl + 2 * m] = yl + st[m];  // the slot the hop would reach if the block went on
            ll.zres[8 * yl + 2 * m + 1] = yl - st[m];
        }
    }
    tile_fill_positions(p, ll);
    const long cost_ll = tile_bank_cost(p, 1) + tile_bank_cost(p, 2) + tile_bank_cost(p, 4) + tile_bank_cost(p, 8);

    // the classes of a site and of the slots its out-of-block hops would reach
    long best = cost_ll;
    TileLayout chosen = ll;
    for (int scheme = 0; scheme < 2; scheme++) {
        auto cls_of = [&](const int Y[4]) {
            return scheme == 0 ? (Y[0] + 2 * Y[1] + 4 * Y[2]) & 7
                               : ((Y[0] + Y[1] + Y[2] + Y[3]) & 1) | (Y[1] & 1) << 1 | (Y[2] & 1) << 2;
        };
        TileLayout sb;
        std::vector<int> cls(vol), zpos(vol);
        int count[8] = {0, 0, 0, 0, 0, 0, 0, 0};
        sb.zres.resize(8 * (size_t)vol);
        for (int yl = 0; yl < vol; yl++) {
            int y[4], Y[4], r = yl, z = 0, zs = 1;
            for (int m = 0; m < 4; m++) { y[m] = r % p.b[m]; r /= p.b[m]; }
            for (int m = 0; m < 4; m++) {
                Y[m] = y[m] / p.s[m] + 2;  // even offset: the hop below stays non-negative
                z += zs * (y[m] % p.s[m]);
                zs *= p.s[m];
            }
            cls[yl] = cls_of(Y);
            zpos[yl] = z;
            count[cls[yl]]++;
            for (int m = 0; m < 4; m++)
                for (int d = 0; d < 2; d++) {
                    int Z[4] = {Y[0], Y[1], Y[2], Y[3]};
                    Z[m] += d ? -1 : 1;
                    sb.zres[8 * yl + 2 * m + d] = cls_of(Z);
                }
        }
        bool balanced = vol % 8 == 0;
        for (int k = 0; k < 8; k++) balanced = balanced && count[k] == vol / 8;
        if (!balanced) continue;
        sb.slot.resize(vol);
        int rank[8] = {0, 0, 0, 0, 0, 0, 0, 0};
        for (int yl = 0; yl < vol; yl++) sb.slot[yl] = 8 * rank[cls[yl]]++ + cls[yl];
        sb.order.reserve(vol);
        for (int l = 0; l < p.nsteps; l++) {
            // the level's sites grouped by z (groups in order of first appearance), each group
            // round-robin over the classes
            std::vector<int> zorder;
            std::vector<std::vector<int>> groups;
            for (int k = p.h_step_ptr[l]; k < p.h_step_ptr[l + 1]; k++) {
                const int yl = ll.order[k];
                size_t gi = std::find(zorder.begin(), zorder.end(), zpos[yl]) - zorder.begin();
                if (gi == zorder.size()) {
                    zorder.push_back(zpos[yl]);
                    groups.emplace_back();
                }
                groups[gi].push_back(yl);
            }
            for (const auto &grp : groups) {
                std::vector<int> byc[8];
                for (int yl : grp) byc[cls[yl]].push_back(yl);
                size_t taken[8] = {0, 0, 0, 0, 0, 0, 0, 0};
                for (size_t n = 0; n < grp.size();)
                    for (int c = 0; c < 8; c++)
                        if (taken[c] < byc[c].size()) {
                            sb.order.push_back(byc[c][taken[c]++]);
                            n++;
                        }
            }
        }
        tile_fill_positions(p, sb);
        const long cost = tile_bank_cost(p, 1) + tile_bank_cost(p, 2) + tile_bank_cost(p, 4) + tile_bank_cost(p, 8);
        if (cost < best) {
            best = cost;
            chosen = sb;
        }
    }
    tile_fill_positions(p, chosen);
}

bool tile_positions_valid(const SapPlan &p) {
    // every site once, slots a permutation of 0 .. vol - 1, every neighbour slot below vol + zslots
    const size_t vol = p.vol;
    if (p.vol > 0xffff || p.h_tile_pos.size() != 4 * vol || p.h_tile_site.size() != 2 * vol || p.tile_zslots < 1) return false;
    std::vector<char> site(vol, 0), slot(vol, 0);
    for (size_t k = 0; k < vol; k++) {
        const int yl = p.h_tile_site[k];
        if (yl < 0 || yl >= p.vol || site[yl]) return false;
        site[yl] = 1;
        // the packed block-local coordinates are those of the site (x fastest)
        int r = yl;
        for (int m = 0; m < 4; m++) {
            if ((int)((unsigned)p.h_tile_site[vol + k] >> (8 * m) & 255u) != r % p.b[m]) return false;
            r /= p.b[m];
        }
        for (int e = 0; e < 4; e++) {
            const int4 pt = p.h_tile_pos[(size_t)((e >> 1) * p.vol + k) * 2 + (e & 1)];
            const int q = pt.y & 0xffff;
            if (q >= p.vol || pt.x != p.h_site_off[yl] || (e == 0 && slot[q]) || (e > 0 && !slot[q])) return false;
            slot[q] = 1;
            for (unsigned w : {(unsigned)pt.z, (unsigned)pt.w})
                if ((int)(w & 0xffff) >= p.vol + p.tile_zslots || (int)(w >> 16) >= p.vol + p.tile_zslots) return false;
        }
    }
    return true;
}

int tile_build_records(qcd_ctx *c, const SapPlan &p, void *rec) {
    Geo g;
    for (int m = 0; m < 4; m++) g.L[m] = c->lat.L[m];
    g.V = c->lat.V;
    g.bc_t = c->bc_t;
    const long total = (long)(p.nblk[0] + p.nblk[1]) * p.vol;
    const int4 bd = make_int4(p.b[0], p.b[1], p.b[2], p.b[3]);
    const unsigned grid = (unsigned)((total + 127) / 128);
    if (p.half)
        k_tile_records<true><<<grid, 128, 0, c->stream>>>(static_cast<uint4 *>(rec), c->U32, c->F32, g, bd, p.vol,
                                                          p.d_tile_site, p.d_origin[0], p.d_origin[1], p.nblk[0], total);
    else
        k_tile_records<false><<<grid, 128, 0, c->stream>>>(static_cast<uint4 *>(rec), c->U32, c->F32, g, bd, p.vol,
                                                           p.d_tile_site, p.d_origin[0], p.d_origin[1], p.nblk[0], total);
    return check_launch(c, "launch of the tile record kernel");
}

namespace {
using TileKernel = void (*)(TileArgs);
template <bool HALF, bool ALL, bool FLAT = false> TileKernel tile_kernel(int R) {
    switch (R) {
        case 1: return k_sap_tile<HALF, 1, ALL, FLAT>;
        case 2: return k_sap_tile<HALF, 2, ALL, FLAT>;
        case 4: return k_sap_tile<HALF, 4, ALL, FLAT>;
        default: return k_sap_tile<HALF, 8, ALL, FLAT>;
    }
}
TileKernel tile_kernel(bool half, bool all, bool flat, int R) {
    if (!all) return half ? tile_kernel<true, false>(R) : tile_kernel<false, false>(R);
    if (flat) return half ? tile_kernel<true, true, true>(R) : tile_kernel<false, true, true>(R);
    return half ? tile_kernel<true, true>(R) : tile_kernel<false, true>(R);
}
}  // namespace

int tile_set_attributes(qcd_ctx *c) {
    for (int R = 1; R <= kTileMaxRhs; R *= 2)
        for (int k = 0; k < 8; k++)
            QCD_CUDA(c, cudaFuncSetAttribute((const void *)tile_kernel(k & 1, k >> 1 & 1, k >> 2, R),
                                             cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kTileSmemLimit));
    return QCD_OK;
}

namespace {

// warp items (16 (site, right-hand side) pairs) of level l
int tile_level_items(const SapPlan &p, int l, int R) { return ((p.h_step_ptr[l + 1] - p.h_step_ptr[l]) * R + 15) / 16; }
// CTAs of T threads that an SM holds: by registers (128 a thread) and shared memory
long tile_fit(size_t smem, int T) { return std::min<long>(kTileSmemPerSm / (smem + 1024), std::min(512 / T, 16)); }

// Threads of a CTA with R right-hand sides: two per (site, right-hand side) of the largest level, up to
// kTileMaxThreads, and at least two warps, which share a small block's prologue (8^3x16, 2^4 blocks, one
// right-hand side: 92 us per application with one warp, 62 with two, 66 with three; on 24^3x48 1480,
// 1408, 1944).
//  - Two CTAs of 192 or 224 threads leave registers of an SM unused: 256 instead, or 128 where the SMs then take the
//    levels in fewer rounds (its waves times the rounds of a wave).  us with 128 / 192 / 256, FP32, two sweeps of the SAP cycle: 4x2x4^2 blocks, two right-hand
//    sides, 32^3x64 5806 / 7415 / 6836, 16^3x32 439 / 554 / 514, 8^3x16 233 / 191 / 174; 4^4, one, 32^3x64 3512 / 4157 /
//    3782, 16^3x32 357 / 312 / 287; 3^3x6 in natural order, four (224), 30^3x60 14108 / 12619 / 12127.
//  - FP16 blocks of narrow levels whose sums do not fit the tensor memory of eight CTAs of 64 threads (which
//    reach half of its lanes): 96, unless the grid then takes more waves than that loses CTAs.  us with 64 / 96: 3^3x4
//    blocks, 30^3x64 4631 / 4242, 18^3x32 (864 CTAs a colour) 559 / 598; 3^3x6 in natural order 30^3x60 4726 / 4423,
//    18^3x36 855 / 735 (FP32 5089 / 5496 and 947 / 806: left).
int tile_threads(const SapPlan &p, int R) {
    const int t = std::max(64, std::min(((p.max_step * R * 2 + 31) / 32) * 32, kTileMaxThreads));
    const double ctas = std::max(p.nblk[0], p.nblk[1]), sms = std::max(1, p.sms);
    if (t == 192 || t == 224) {
        auto time = [&](int T) {
            int rounds = 0;
            for (int l = 0; l < p.nsteps; l++) rounds += (tile_level_items(p, l, R) + T / 32 - 1) / (T / 32);
            return std::ceil(ctas / (sms * std::max<long>(1, tile_fit(tile_smem_bytes(p, R), T)))) * rounds;
        };
        return time(128) < 0.85 * time(256) ? 128 : 256;
    }
    if (t == 64 && p.half) {
        int items = 0;
        for (int l = 0; l < p.nsteps; l++) items += tile_level_items(p, l, R);
        if ((items + 1) / 2 * 12 > 64 && std::ceil(ctas / (sms * 5)) <= 1.7 * std::ceil(ctas / (sms * 8))) return 96;
    }
    return t;
}

// Relative time of an application with R right-hand sides per CTA: the share of the SMs' warps that its warp
// items take, each costing more the more sites (16 / R) its record loads cover, and the rounds of items that a
// CTA's warps take level by level.  The weights fit measured applications; us with the R that the most
// right-hand sides would give -> with the least cost (R in parentheses): 24^3x48, 4^4 blocks, FP16, 3 right-hand
// sides 1026 (2) -> 892 (4), 5 1704 (4) -> 1501 (2); 16^3x32, 2^4 blocks, FP16, 3 599 (2) -> 367 (4), 5 705 (4)
// -> 523 (8); 8^3x16, 4^4 blocks, FP16, 2 85 (2) -> 65 (1), 8 141 (4) -> 66 (1).
float tile_cost(const SapPlan &p, int R, int nrhs) {
    const int nw = tile_threads(p, R) / 32;
    int items = 0, rounds = 0;
    for (int l = 0; l < p.nsteps; l++) {
        const int n = tile_level_items(p, l, R);
        items += n;
        rounds += (n + nw - 1) / nw;
    }
    const float ctas = (float)std::max(p.nblk[0], p.nblk[1]) * (float)((nrhs + R - 1) / R);
    const float filled = ctas * (float)items * (1.f + 1.12f / (float)R) / ((float)std::max(1, p.sms) * 16.f);
    return filled + 0.73f * (float)rounds;
}

// Whether the prologue and the epilogue take the block's sites in one go instead of level by level: where no
// level has more than 24 (FP16: 12) (site, right-hand side) pairs (and all hop sums have a slot).  The levels' rounds
// would wait for memory one after the other for a few sites each; the epilogue forms all eight hops for it.
// us, level by level -> in one go, one sweep and three cycles (four and two): 2^4 blocks (levels of 1, 4, 6, 4, 1
// sites) on 32^3x64, FP16, one right-hand side 13787 -> 10387 (16851 -> 14779), two 13712 -> 11123 (16680 -> 15481), four
// (24 pairs) 16103 -> 15928 (19915 -> 19926); FP32 10693 -> 8606 (15716 -> 14300), 11485 -> 9442 (16528 -> 15360), 14180 ->
// 13531 (19885 -> 19294); 2^3x4 blocks, FP16, one 6960 -> 5472 (8559 -> 7811), two (24) 8129 -> 8116 (10074 -> 10155);
// FP32, two 7559 -> 7150 (10654 -> 10241), four (48) 12111 -> 12502 (16199 -> 16212).
bool tile_flat(const SapPlan &p, int R) { return p.max_step * R <= (p.half ? 12 : 24); }

// Tensor memory of a CTA: a slot of 12 FP32 columns per warp item, the items dealt to the warps in turn;
// warps four apart share a lane quarter.  As many slots as fit the columns that leave the CTAs resident
// that the other resources allow; if not all do, one more slot is the place where an uncached item holds
// one side's sum while it forms the other's.
// Returns whether every item has a slot.
bool tile_tmem(const SapPlan &p, int R, int T, size_t smem, long grid, TileArgs &a) {
    int items = 0;
    for (int l = 0; l < p.nsteps; l++) items += tile_level_items(p, l, R);
    const int nw = T / 32, share = (nw + 3) / 4, need = (items + nw - 1) / nw;
    // CTAs an SM will hold: what it can and what the grid offers
    const long sms = std::max(1, p.sms);
    const int ctas = (int)std::max<long>(1, std::min(tile_fit(smem, T), (grid + sms - 1) / sms));
    int most = 32;  // columns per CTA
    while (most * 2 <= 512 && most * 2 * ctas <= 512) most *= 2;
    // up to a third of the CTAs is given up for keeping more sums, where the grid's waves grow by no more than
    // a third with it (18^3x32, 3^3x4 blocks, FP32, one right-hand side, 864 CTAs: 903 us with all sums in two waves of
    // four CTAs an SM, 643 with some formed anew in one of six)
    auto waves = [&](int per_sm) { return (grid + sms * per_sm - 1) / (sms * per_sm); };
    while (most < 512 && 12 * need * share > most && most * 2 * (ctas - ctas / 3) <= 512 &&
           3 * waves(512 / (most * 2)) <= 4 * waves(ctas))
        most *= 2;
    int s = need;
    if (12 * s * share > most) s = std::max(0, most / (12 * share) - 1);
    a.tm_slots = s;
    a.tm_per_warp = 12 * (s < need ? s + 1 : s);
    a.tm_cols = 32;
    while (a.tm_cols < a.tm_per_warp * share) a.tm_cols *= 2;
    return s == need;
}

}  // namespace

// first position, pairs, first warp and first slot of every level for each R = 1, 2, 4, 8: [4][nsteps]
void tile_level_table(SapPlan &p) {
    p.h_tile_item.clear();
    for (int R = 1; R <= kTileMaxRhs; R *= 2) {
        const int nw = tile_threads(p, R) / 32;
        int g = 0;
        for (int l = 0; l < p.nsteps; l++) {
            p.h_tile_item.push_back(make_int4(p.h_step_ptr[l], (p.h_step_ptr[l + 1] - p.h_step_ptr[l]) * R, g % nw, g / nw));
            g += tile_level_items(p, l, R);
        }
    }
}

int tile_choose(const SapPlan &p, int nrhs, int *R, int *threads, size_t *smem) {
    // The right-hand sides per CTA, of those that let kTileMinBlocks CTAs share an SM (the registers
    // allow that many of 256 threads): the most that nrhs fills, unless tile_cost finds another at least
    // 5% cheaper.
    const size_t share = kTileSmemPerSm / kTileMinBlocks - 1024;
    int r = 1;
    while (r * 2 <= kTileMaxRhs && r * 2 <= nrhs && tile_smem_bytes(p, r * 2) <= share) r *= 2;
    float least = 0.95f * tile_cost(p, r, nrhs);
    for (int q = 1; q <= kTileMaxRhs && q < 2 * nrhs && (q == 1 || tile_smem_bytes(p, q) <= share); q *= 2) {
        const float cost = tile_cost(p, q, nrhs);
        if (cost < least) {
            least = cost;
            r = q;
        }
    }
    if (tile_smem_bytes(p, r) > kTileSmemLimit) return QCD_ERR_ARG;
    *R = r;
    *threads = tile_threads(p, r);
    *smem = tile_smem_bytes(p, r);
    return QCD_OK;
}

int tile_sap_apply(qcd_ctx *c, const SapPlan &p, float4 *x, const float4 *v, float4 *r, float4 *y, double omega,
                   int nsweep, int nsap, int nrhs, const BicgScalars *gate) {
    int R = 1, T = 32;
    size_t smem = 0;
    if (tile_choose(p, nrhs, &R, &T, &smem)) return fail(c, QCD_ERR_ARG, "SAP block too large for the tile form");
    TileArgs a;
    a.x = x;
    a.r = r;
    a.y = y;
    a.v = v;
    a.pos = p.d_tile_pos;
    a.coords = p.d_tile_site + p.vol;
    a.gate = gate;
    a.kappa = (float)c->kappa;
    a.omega = (float)omega;
    a.V = c->lat.V;
    for (int m = 0; m < 4; m++) a.L[m] = c->lat.L[m];
    a.bc_t = c->bc_t;
    a.vol = p.vol;
    a.nlev = p.nsteps;
    a.nsweep = nsweep;
    a.nrhs = nrhs;
    int lr = 0;
    while ((1 << lr) < R) lr++;
    a.levels = p.d_tile_item + lr * p.nsteps;
    const bool all = tile_tmem(p, R, T, smem, (long)std::max(p.nblk[0], p.nblk[1]) * ((nrhs + R - 1) / R), a);
    a.stride = R * (p.half ? TileRec<true>::y_words : TileRec<false>::y_words);
    a.zslots = p.tile_zslots;
    // FP16 storage: y's FP16 records in the first half of the y field, the scales after them
    a.y16 = reinterpret_cast<uint4 *>(y);
    a.yscale = reinterpret_cast<float *>(a.y16 + (size_t)nrhs * c->lat.V * 3);
    for (int m = 0; m < 4; m++) {
        a.b[m] = p.b[m];
        a.nb[m] = p.nb[m];
    }
    const TileKernel k = tile_kernel(p.half, all, tile_flat(p, R), R);
    const size_t rec_words = (size_t)p.vol * ((p.half ? kTileRecordBytesHalf : kTileRecordBytes) / 16);
    for (int j = 0; j < nsap; j++)
        for (int col = 0; col < 2; col++) {
            const bool last = j == nsap - 1;
            a.rec = reinterpret_cast<const uint4 *>(p.d_rec) + (size_t)(col ? p.nblk[0] : 0) * rec_words;
            a.origin_site = p.d_origin_site[col];
            a.origin = p.d_origin[col];
            a.first = j == 0;
            a.cross = !(j == 0 && col == 0);
            a.store_r = !last;
            a.store_y = !(last && col == 1);
            a.blk_base = col ? p.nblk[0] : 0;
            a.other_base = col ? 0 : p.nblk[0];
            cudaEvent_t ev;
            prof_begin(c, QCD_K_SSOR, &ev);
            launch_chained(c, k, dim3(p.nblk[col], (nrhs + R - 1) / R), T, smem, a);
            int rc = prof_end(c, QCD_K_SSOR, ev);
            if (rc) return rc;
        }
    return QCD_OK;
}

}  // namespace qcd
