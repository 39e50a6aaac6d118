// K3/K4: Luescher's SAP preconditioner (Eq. (4), Alg. 1) with SSOR block
// inverses in locally-lexicographic sub-block order (Sec. 3).
//
// One SAP cycle, for colour c = E then O, in residual form:
//   y_c = A_cc r_c                 (K3: SSOR sweeps on every block of colour c)
//   x  += y_c;  r_c -= D_cc y_c    (K4, in-block hops)
//   r_c' -= D_c'c y_c              (K4, hops that leave the block)
// which equals Alg. 1 (y = K r, w = D y, x += y, r -= w) term by term.
//
// K3 runs a cluster of C CTAs per SAP block (C = 1 when the block fits one
// CTA and the GPU is full of blocks).  The ll order (key = lambda * N_sb +
// sigma, lambda the lexicographic local position inside a sub-block, sigma the
// lexicographic sub-block index) is run as a wavefront of dependency levels:
// a site's level is one more than the highest level of its earlier in-block
// neighbours, so the sites of one level are pairwise non-adjacent and updating
// level after level gives exactly the sequential result.  Each CTA owns an
// equal share of every level (dealt round-robin); barriers (CTA or cluster)
// are placed only where data flows (the paper's OpenMP barriers between
// dependent sites).  Four lanes share a site update (k_ssor_quad).
// Each CTA keeps its sites' spinors in shared memory (neighbours owned by peer
// CTAs are read through distributed shared memory); a lane's part of the next
// site's record and source is loaded into registers while the CTA is on its
// way through the barrier.
#include <cooperative_groups.h>
#include <cuda_fp16.h>

#include <algorithm>
#include <cstring>

#include "fields.cuh"
#include "qcd_internal.h"

namespace qcd {

namespace {

struct BlockGeo {
    int b[4];
    int vol;
};

// adds the hops of site n (global coords x, block-local coords yl) whose
// neighbour lies inside (INB = true) or outside (INB = false) n's block
template <bool INB, bool COHERENT>
__device__ __forceinline__ void masked_hops(const float4 *src, const float2 *__restrict__ U, const Geo &g, long n,
                                            const int x[4], const int yl[4], const BlockGeo &bg, float2 acc[12]) {
    float2 psi[12], u[9];
#define QCD_HOP(MU)                                                                                     \
    {                                                                                                   \
        const bool fin = yl[MU] + 1 < bg.b[MU];                                                         \
        if (fin == INB) {                                                                               \
            long m = nbr_fwd<MU>(g, n, x);                                                              \
            if (COHERENT) load_spinor_rw(src, m, psi); else load_spinor(src, m, psi);         \
            load_link(U, g.V, n, MU, u);                                                                \
            const float sg = (MU == 3 && x[3] == g.L[3] - 1) ? (float)g.bc_t : 1.0f;                    \
            hop_term<MU, true>(psi, u, sg, acc);                                                        \
        }                                                                                               \
        const bool bin = yl[MU] > 0;                                                                    \
        if (bin == INB) {                                                                               \
            long m = nbr_bwd<MU>(g, n, x);                                                              \
            if (COHERENT) load_spinor_rw(src, m, psi); else load_spinor(src, m, psi);         \
            load_link(U, g.V, m, MU, u);                                                                \
            const float sg = (MU == 3 && x[3] == 0) ? (float)g.bc_t : 1.0f;                             \
            hop_term<MU, false>(psi, u, sg, acc);                                                       \
        }                                                                                               \
    }
    QCD_HOP(0)
    QCD_HOP(1)
    QCD_HOP(2)
    QCD_HOP(3)
#undef QCD_HOP
}


namespace cg = cooperative_groups;

// Most sites of one CTA in one step of the kernel: clusters; one CTA per block and per SM; one CTA per block,
// several per SM.  Sites beyond the warps of a step start
// another step without a barrier, but wait for their records then.  Measured, 6^3x12 blocks: 24^3x48 FP16,
// C = 1: 24 sites 6190 us, 48 4122, 64 3342, 96 2919; 12^3x24 FP32, C = 8 (52 sites in the widest level):
// 24 sites 1633 us, 32 1487, 64 1258, and 8^4 blocks FP16: 32 sites 297 us, 48 273, 64 250, 96 327.  Where
// CTAs share an SM the others fill the gaps: 24^3x48, 4^4 blocks FP16: 8 sites 2761 us, 16 1967, 32 2147.
constexpr int kMaxRun = 64;
constexpr int kMaxRunAlone = 96;
constexpr int kMaxRunShared = 16;
constexpr int kMaxCluster = 16;    // CTAs per SAP block (clusters above 8 need the non-portable size)
constexpr size_t kSmemLimit = 200 * 1024;
// most bytes of spinors per CTA of the cluster form where 16 CTAs allow it
constexpr size_t kSlabLimit = 128 * 1024, kSlabLimitHalf = 140 * 1024;

// Per-site record of the SSOR kernel (k_ssor_quad), in 4-byte words: what its four lanes read, 36 complex
// numbers each (2 words in FP32 storage, 1 word, a half2, in FP16).  Lane j has W_d of directions j and
// j + 4 (d = 2 mu + (backward)): U_mu(n) forward, U_mu(n - mu)^dag backward, 3x3 row-major, zero when the
// hop leaves the block; then the rows 3 (j & 1) .. 3 (j & 1) + 2 of chiral block j >> 1 of F/2, six numbers
// each.  Load q of a lane holds its numbers 4 q .. 4 q + 3, and the four lanes' loads lie side by side.
// FP16: the spinors a CTA owns are scaled by one FP32 factor per CTA.
template <bool HALF> struct Rec {
    static constexpr int cw = HALF ? 1 : 2;        // words per complex
    static constexpr int load_words = 4 * cw;      // one lane's load
    static constexpr int words = 4 * 36 * cw;      // 288 (FP32) or 144 (FP16)
    static constexpr int ywords = 12 * cw;         // words of one site's spinor in shared memory
    // word of number e of lane j
    __host__ __device__ static constexpr int at(int j, int e) { return ((e >> 2) * 4 + j) * load_words + (e & 3) * cw; }
};
static_assert(Rec<false>::words * 4 == kSapRecordBytesPerSite, "record size");

// one lane's part of a record, as stored
template <bool HALF> struct QuadRecord {
    uint32_t r[HALF ? 36 : 72];
    __device__ __forceinline__ void load(const float *p) {  // p: the lane's first load
#pragma unroll
        for (int q = 0; q < 9; q++) {
            const float *s = p + q * 4 * Rec<HALF>::load_words;
            if constexpr (HALF)
                asm("ld.global.nc.v4.b32 {%0, %1, %2, %3}, [%4];"
                             : "=r"(r[4 * q]), "=r"(r[4 * q + 1]), "=r"(r[4 * q + 2]), "=r"(r[4 * q + 3]) : "l"(s));
            else
                asm("ld.global.nc.v8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
                             : "=r"(r[8 * q]), "=r"(r[8 * q + 1]), "=r"(r[8 * q + 2]), "=r"(r[8 * q + 3]), "=r"(r[8 * q + 4]),
                               "=r"(r[8 * q + 5]), "=r"(r[8 * q + 6]), "=r"(r[8 * q + 7]) : "l"(s));
        }
    }
    __device__ __forceinline__ float2 at(int e) const {
        if constexpr (HALF) return __half22float2(*reinterpret_cast<const __half2 *>(&r[e]));
        else return make_float2(__uint_as_float(r[2 * e]), __uint_as_float(r[2 * e + 1]));
    }
};

// complex load / store in the storage format (w points at the number's first word)
template <bool HALF> __device__ __forceinline__ float2 ld_c(const float *w) {
    if constexpr (HALF) return __half22float2(*reinterpret_cast<const __half2 *>(w));
    else return *reinterpret_cast<const float2 *>(w);
}
// distributed shared memory: a shared-window address mapped to CTA `rank` of the cluster, and
// loads through it (valid for the executing CTA's own addresses too)
__device__ __forceinline__ uint32_t mapa_u32(uint32_t a, int rank) {
    uint32_t r;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;\n" : "=r"(r) : "r"(a), "r"(rank));
    return r;
}
__device__ __forceinline__ float ld_cluster_f32(uint32_t a) {
    float v;
    asm volatile("ld.shared::cluster.f32 %0, [%1];\n" : "=f"(v) : "r"(a) : "memory");
    return v;
}
// a spinor in the storage format at a shared-window address (CL: of any CTA of the cluster)
template <bool HALF, bool CL> __device__ __forceinline__ void ld_spinor_smem(uint32_t a, float2 q[12]) {
#pragma unroll
    for (int i = 0; i < (HALF ? 3 : 6); i++) {
        uint32_t w[4];
        if constexpr (CL)
            asm volatile("ld.shared::cluster.v4.b32 {%0, %1, %2, %3}, [%4];"
                         : "=r"(w[0]), "=r"(w[1]), "=r"(w[2]), "=r"(w[3]) : "r"(a + 16u * i) : "memory");
        else
            asm volatile("ld.shared.v4.b32 {%0, %1, %2, %3}, [%4];"
                         : "=r"(w[0]), "=r"(w[1]), "=r"(w[2]), "=r"(w[3]) : "r"(a + 16u * i) : "memory");
        if constexpr (HALF) {
#pragma unroll
            for (int k = 0; k < 4; k++) q[4 * i + k] = __half22float2(*reinterpret_cast<const __half2 *>(&w[k]));
        } else {
            q[2 * i] = make_float2(__uint_as_float(w[0]), __uint_as_float(w[1]));
            q[2 * i + 1] = make_float2(__uint_as_float(w[2]), __uint_as_float(w[3]));
        }
    }
}
template <bool HALF> __device__ __forceinline__ void st_c(float *w, float2 v) {
    if constexpr (HALF) *reinterpret_cast<__half2 *>(w) = __float22half2_rn(v);
    else *reinterpret_cast<float2 *>(w) = v;
}

// Builds the per-site records of every block (blocks of colour 0 first), each block's in the order of
// the CTAs' chunk lists: position i % vol holds block-local site list[i % vol].x.
template <bool HALF>
__global__ void k_sap_records(float *__restrict__ rec, const float2 *__restrict__ U, const float4 *__restrict__ F,
                              Geo g, BlockGeo bg, const int2 *__restrict__ list, const int *__restrict__ org0,
                              const int *__restrict__ org1, int nblk0, long total) {
    using L = Rec<HALF>;
    const long i = blockIdx.x * (long)blockDim.x + threadIdx.x;
    if (i >= total) return;
    const int gb = (int)(i / bg.vol), yl = list[i % bg.vol].x;
    const int *o = gb < nblk0 ? org0 + 4 * gb : org1 + 4 * (gb - nblk0);
    int y[4], r = yl;
    for (int m = 0; m < 4; m++) { y[m] = r % bg.b[m]; r /= bg.b[m]; }
    const long gs[4] = {1, g.L[0], (long)g.L[0] * g.L[1], (long)g.L[0] * g.L[1] * g.L[2]};
    long n = 0;
    for (int m = 0; m < 4; m++) n += gs[m] * (o[m] + y[m]);
    float *R = rec + i * L::words;
    for (int d = 0; d < 8; d++) {
        const int mu = d >> 1, e0 = d < 4 ? 0 : 9;
        const bool fwd = (d & 1) == 0;
        const int ym = y[mu] + (fwd ? 1 : -1);
        const bool leaves = ym < 0 || ym >= bg.b[mu];
        const long src = fwd ? n : n - gs[mu];
        for (int a = 0; a < 3; a++)
            for (int bb = 0; bb < 3; bb++) {
                float2 u = make_float2(0.f, 0.f);
                if (!leaves) {
                    u = U[(long)(mu * 9 + (fwd ? a * 3 + bb : bb * 3 + a)) * g.V + src];
                    if (!fwd) u.y = -u.y;
                }
                st_c<HALF>(R + L::at(d & 3, e0 + a * 3 + bb), u);
            }
    }
    float fp[72];
    for (int k = 0; k < 18; k++) {
        const float4 v = F[(long)k * g.V + n];
        fp[4 * k] = v.x; fp[4 * k + 1] = v.y; fp[4 * k + 2] = v.z; fp[4 * k + 3] = v.w;
    }
    // unpack each Hermitian block (6 real diagonal, 15 complex below the diagonal) into full rows
    for (int ch = 0; ch < 2; ch++)
        for (int ii = 0; ii < 6; ii++)
            for (int j = 0; j < 6; j++) {
                float2 e;
                if (ii == j) e = make_float2(fp[36 * ch + ii], 0.f);
                else if (j < ii) { const int q = 36 * ch + 6 + 2 * (ii * (ii - 1) / 2 + j); e = make_float2(fp[q], fp[q + 1]); }
                else { const int q = 36 * ch + 6 + 2 * (j * (j - 1) / 2 + ii); e = make_float2(fp[q], -fp[q + 1]); }
                st_c<HALF>(R + L::at(2 * ch + ii / 3, 18 + 6 * (ii % 3) + j), e);
            }
}

enum { kFormShared, kFormAlone, kFormCluster };  // several CTAs per SM, one CTA per SM, clusters
constexpr int quad_threads(bool half, int form) {
    return form == kFormShared ? 4 * kMaxRunShared : form == kFormCluster && half ? 4 * kMaxRun : 4 * kMaxRunAlone;
}

struct SsorArgs {
    float4 *y;                 // out: the block solutions
    const float4 *f;           // source (the SAP residual)
    const float4 *rec;         // per-site records of this colour's blocks
    float kappa, omega;
    int nsweep;
    long V;
    int vol, C, slab_vol, nchunks, ypitch;  // nchunks: steps; ypitch: words from one spinor to the next in the slab
    const int *chunk_ptr;      // [C][nchunks + 1] the steps, as offsets into the CTA-major list of sites
    const int4 *quad;          // [vol][4] per site of the CTA-major list and lane j: where the neighbours in
                               // directions j and j + 4 lie ((owner CTA << 24) | word in its slab, the zero
                               // spinor when the hop leaves the block), the site's own word in the slab, and
                               // its global offset from the block origin
    const int2 *chunk_site;    // thread form: (block-local site, global offset from the block origin)
    const int *site_off;       // thread form: [vol] global offset of a block-local site from the block origin
    const int *own_off;        // [C][slab_vol] global offset of each site a CTA owns, -1 past the last
    const unsigned char *flags;  // [2 * nchunks] CTA (1) or cluster (2) barrier before a timeline step
    const int *origin_site;    // [blocks of this colour] global index of the block origin
    const BicgScalars *gate;   // blockIdx.y = right-hand side; skipped when inactive (null: all)
    int gb0;                   // thread form: index of this colour's first block in the SoA records
    int b[4];                  // thread form: block extents
};

// K3: y = A_BB f on every block of one colour; blockIdx.x / C enumerates blocks, blockIdx.y is the
// right-hand side.  Four lanes share a site update: lane j forms the hops of directions j and j + 4
// (d = 2 mu + (backward)), the four partial sums meet in a reduce-scatter that leaves lane j with
// spin j, and lane j applies the three clover rows that give spin j (its chirality's, then the sum or
// difference with the other's).
//
// Bound by the chain of levels: about 1.4 us a step in a cluster of 8 with 6^3x12 blocks, 0.6 us of it the
// barrier, the rest one update's latency.  Eight lanes per update shorten no step (the instructions were
// never the chain's longest part) and issue a quarter more per site; a warp per update, with its records
// staged in shared memory, was bound by instruction issue (about 450 per site, 100 here).  Loads wait for
// the arrival at the barrier: issued before it, they delay its release (1313 us instead of 1192).
// 12^3x24, 6^3x12 blocks, 3^3x6 sub-blocks, FP32, 4 sweeps, 4 cycles: 2010 -> 1169 us; 24^3x48, FP16, 2
// sweeps, 4 right-hand sides: 6^3x12 blocks 6098 -> 2708, 4^4 blocks 3619 -> 1873 (before: a warp per update,
// or an octet of lanes where many CTAs shared an SM).
template <bool HALF, int FORM>
__global__ void __launch_bounds__(quad_threads(HALF, FORM), FORM == kFormShared && HALF ? 8 : 0) k_ssor_quad(SsorArgs a) {
    chain_wait();
    constexpr bool CL = FORM == kFormCluster;
    using L = Rec<HALF>;
    extern __shared__ __align__(16) float sm[];
    // the whole cluster shares a right-hand side, so the early exit is uniform
    if (a.gate && !a.gate[blockIdx.y].active) return;
    a.f += (size_t)blockIdx.y * 6 * a.V;
    a.y += (size_t)blockIdx.y * 6 * a.V;
    const int rank = CL ? (int)cg::this_cluster().block_rank() : 0;
    const int nch = a.nchunks;
    int lane;
    asm volatile("mov.u32 %0, %%laneid;" : "=r"(lane));
    const int warp = __shfl_sync(0xffffffffu, threadIdx.x >> 5, 0);
    const int j = lane & 3, grp = lane >> 2;
    const int *cptr_g = a.chunk_ptr + rank * (nch + 1);
    // shared memory: [y slab, then a zero spinor | scales of the cluster's CTAs | chunk pointers];
    // the slab sits at the same offset in every CTA of the cluster (peers read it)
    float *ys = sm;
    float *yscale = ys + (size_t)(a.slab_vol + 1) * a.ypitch;              // [kMaxCluster] + own, being formed
    int *cptr = reinterpret_cast<int *>(yscale + kMaxCluster + 4);         // [nch + 1], from the CTA-major list
    const uint32_t ys_u32 = (uint32_t)__cvta_generic_to_shared(ys);
    const int blk = blockIdx.x / a.C;
    const long n0 = a.origin_site[blk];
    const float *rec = reinterpret_cast<const float *>(a.rec) + (size_t)blk * a.vol * L::words + j * L::load_words;
    const float2 *f2 = reinterpret_cast<const float2 *>(a.f) + n0 * 12 + j * 3;

    // lane constants: half-spinors h0 = psi_a + za psi_b, h1 = psi_c + zc psi_d of directions j (x or y:
    // psi_0, psi_3, psi_1, psi_2) and j + 4 (z: psi_0, psi_2, psi_1, psi_3; t: 2 psi_2, 2 psi_3 forward,
    // 2 psi_0, 2 psi_1 backward), and the factors that rebuild the spins from w = W_d h, in the Dirac
    // representation
    const bool bwd = (j & 1) != 0, up = (j & 2) != 0;
    const float sg = bwd ? -1.f : 1.f;
    const float2 za = up ? make_float2(sg, 0.f) : make_float2(0.f, sg);      // direction j
    const float2 zc = up ? make_float2(-sg, 0.f) : make_float2(0.f, sg);
    const float2 f3a = up ? make_float2(sg, 0.f) : make_float2(0.f, -sg);    // spin 3 gets f3a w0
    const float2 f2a = up ? make_float2(-sg, 0.f) : make_float2(0.f, -sg);   // spin 2 gets f2a w1
    const float2 zA = up ? make_float2(1.f, 0.f) : make_float2(0.f, sg);     // direction j + 4
    const float2 zC = up ? make_float2(1.f, 0.f) : make_float2(0.f, -sg);
    const float f0b = up && !bwd ? 0.f : 1.f;                                // spins 0 and 1: f0b w0, f0b w1
    const float2 f2b = up ? make_float2(bwd ? 0.f : 1.f, 0.f) : make_float2(0.f, -sg);  // spin 2: f2b w0
    const float2 f3b = up ? make_float2(bwd ? 0.f : 1.f, 0.f) : make_float2(0.f, sg);   // spin 3: f3b w1

    // ---- set-up: zero this CTA's slab of y, copy its chunk pointers, FP16: the slab's scale ----
    const int nz = (a.slab_vol + 1) * a.ypitch / 4;
    for (int i = threadIdx.x; i < nz; i += blockDim.x) reinterpret_cast<float4 *>(ys)[i] = make_float4(0.f, 0.f, 0.f, 0.f);
    for (int i = threadIdx.x; i <= nch; i += blockDim.x) cptr[i] = cptr_g[i];
    float inv_scale = 1.f, my_scale = 1.f;
    if constexpr (HALF) {
        // scale = largest |component| of the source on this slab (the block solve is O(1) in it)
        float m = 0.f;
        for (int i = threadIdx.x; i < a.slab_vol * 6; i += blockDim.x) {
            const int sl = i / 6, q = i - 6 * sl;
            const int off = a.own_off[rank * a.slab_vol + sl];
            if (off < 0) continue;
            const float4 v = a.f[(n0 + off) * 6 + q];
            m = fmaxf(m, fmaxf(fmaxf(fabsf(v.x), fabsf(v.y)), fmaxf(fabsf(v.z), fabsf(v.w))));
        }
        for (int off = 16; off > 0; off >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, off));
        if (threadIdx.x == 0) yscale[kMaxCluster] = 0.f;
        __syncthreads();
        if (lane == 0) atomicMax(reinterpret_cast<int *>(yscale + kMaxCluster), __float_as_int(m));  // m >= 0: int order = float order
        __syncthreads();
        my_scale = yscale[kMaxCluster] > 0.f ? yscale[kMaxCluster] : 1.f;
        inv_scale = 1.f / my_scale;
    }
    if (CL) cg::this_cluster().sync();
    else __syncthreads();
    if constexpr (HALF) {
        if (threadIdx.x < a.C) {
            const uint32_t s_u32 = (uint32_t)__cvta_generic_to_shared(yscale + kMaxCluster);
            float v = my_scale;
            if (CL && (int)threadIdx.x != rank) {
                v = ld_cluster_f32(mapa_u32(s_u32, threadIdx.x));
                v = v > 0.f ? v : 1.f;
            }
            yscale[threadIdx.x] = v;
        }
        __syncthreads();
    }

    const int T = a.nsweep * 2 * nch;
    const int slot = warp * 8 + grp;
    // this lane's site of the chunk at sweep position k: its index in the CTA-major list (the last site of
    // the chunk for the lanes past it, whose results are dropped), -1 for a warp past the chunk
    auto position = [&](int k, bool &mine) -> int {
        const int ch = k < nch ? k : 2 * nch - 1 - k;
        const int base = cptr[ch], cnt = cptr[ch + 1] - base;
        mine = slot < cnt;
        return warp * 8 < cnt ? base + (mine ? slot : cnt - 1) : -1;
    };
    auto next = [&](int k) { return k + 1 == 2 * nch ? 0 : k + 1; };
    // the record, source and neighbour codes of the next update wait in registers: they are loaded while
    // the CTA is between two steps, behind the arrival at the barrier
    QuadRecord<HALF> w;
    float2 fv[3];
    int4 code = make_int4(0, 0, 0, 0), code1 = make_int4(0, 0, 0, 0);
    bool mine0, mine1, mine2;
    int k1 = next(0);
    int p0 = position(0, mine0), p1 = position(k1, mine1);
    auto load_source = [&](int off) {
#pragma unroll
        for (int c = 0; c < 3; c++) fv[c] = f2[(size_t)off * 12 + c];
    };
    if (p0 >= 0) {
        code = __ldg(a.quad + (size_t)p0 * 4 + j);
        w.load(rec + (size_t)p0 * L::words);
        load_source(code.w);
    }
    if (p1 >= 0) code1 = __ldg(a.quad + (size_t)p1 * 4 + j);

    int flag = a.flags[k1];
    for (int t = 0; t < T; t++) {
        if (p0 >= 0) {
            float v[24];  // this lane's hops, [spin][colour][re, im]
            {
                float2 q[12], h0[3], h1[3], g0[3], g1[3];
                uint32_t ada = ys_u32 + 4u * (uint32_t)(code.x & 0xffffff), adb = ys_u32 + 4u * (uint32_t)(code.y & 0xffffff);
                if constexpr (CL) {
                    ada = mapa_u32(ada, code.x >> 24);
                    adb = mapa_u32(adb, code.y >> 24);
                }
                ld_spinor_smem<HALF, CL>(ada, q);
                float sca = 1.f, scb = 1.f;
                if constexpr (HALF) {
                    sca = yscale[code.x >> 24];
                    scb = yscale[code.y >> 24];
                }
#pragma unroll
                for (int c = 0; c < 3; c++) {
                    h0[c] = cfma(za, q[9 + c], q[c]);
                    h1[c] = cfma(zc, q[6 + c], q[3 + c]);
                }
                ld_spinor_smem<HALF, CL>(adb, q);
                const bool tf = up && !bwd, tb = up && bwd;
#pragma unroll
                for (int c = 0; c < 3; c++) {
                    const float2 qa = tf ? q[6 + c] : q[c], qb = tb ? q[c] : q[6 + c];
                    const float2 qc = tf ? q[9 + c] : q[3 + c], qd = tb ? q[3 + c] : q[9 + c];
                    g0[c] = cfma(zA, qb, qa);
                    g1[c] = cfma(zC, qd, qc);
                }
#pragma unroll
                for (int r = 0; r < 3; r++) {
                    float2 w0 = make_float2(0.f, 0.f), w1 = make_float2(0.f, 0.f);
#pragma unroll
                    for (int c = 0; c < 3; c++) {
                        const float2 u = w.at(r * 3 + c);
                        w0 = cfma(u, h0[c], w0);
                        w1 = cfma(u, h1[c], w1);
                    }
                    if constexpr (HALF) { w0 = cscale(w0, sca); w1 = cscale(w1, sca); }
                    const float2 e2 = cmul(f2a, w1), e3 = cmul(f3a, w0);
                    v[2 * r] = w0.x; v[2 * r + 1] = w0.y;
                    v[6 + 2 * r] = w1.x; v[6 + 2 * r + 1] = w1.y;
                    v[12 + 2 * r] = e2.x; v[12 + 2 * r + 1] = e2.y;
                    v[18 + 2 * r] = e3.x; v[18 + 2 * r + 1] = e3.y;
                }
#pragma unroll
                for (int r = 0; r < 3; r++) {
                    float2 w0 = make_float2(0.f, 0.f), w1 = make_float2(0.f, 0.f);
#pragma unroll
                    for (int c = 0; c < 3; c++) {
                        const float2 u = w.at(9 + r * 3 + c);
                        w0 = cfma(u, g0[c], w0);
                        w1 = cfma(u, g1[c], w1);
                    }
                    if constexpr (HALF) { w0 = cscale(w0, scb); w1 = cscale(w1, scb); }
                    // one product of each sum is exact, so each is the rounded sum of the two hops
                    v[2 * r] = fmaf(f0b, w0.x, v[2 * r]);
                    v[2 * r + 1] = fmaf(f0b, w0.y, v[2 * r + 1]);
                    v[6 + 2 * r] = fmaf(f0b, w1.x, v[6 + 2 * r]);
                    v[6 + 2 * r + 1] = fmaf(f0b, w1.y, v[6 + 2 * r + 1]);
                    const float2 e2 = cfma(f2b, w0, make_float2(v[12 + 2 * r], v[12 + 2 * r + 1]));
                    const float2 e3 = cfma(f3b, w1, make_float2(v[18 + 2 * r], v[18 + 2 * r + 1]));
                    v[12 + 2 * r] = e2.x; v[12 + 2 * r + 1] = e2.y;
                    v[18 + 2 * r] = e3.x; v[18 + 2 * r + 1] = e3.y;
                }
            }
            // reduce-scatter over the four lanes: lane j ends with spin j of the sum
            float u12[12], A[6];
#pragma unroll
            for (int i = 0; i < 12; i++) {
                const float send = up ? v[i] : v[12 + i], keep = up ? v[12 + i] : v[i];
                u12[i] = keep + __shfl_xor_sync(0xffffffffu, send, 2);
            }
#pragma unroll
            for (int i = 0; i < 6; i++) {
                const float send = bwd ? u12[i] : u12[6 + i], keep = bwd ? u12[6 + i] : u12[i];
                A[i] = keep + __shfl_xor_sync(0xffffffffu, send, 1);
            }
            // chiral components: spins 0, 1 minus and plus spins 2, 3
            float2 x[6];
            {
                float cv[6];
#pragma unroll
                for (int i = 0; i < 6; i++) {
                    const float P = __shfl_xor_sync(0xffffffffu, A[i], 2);
                    cv[i] = up ? P + A[i] : A[i] - P;
                }
#pragma unroll
                for (int c = 0; c < 3; c++) {
                    float2 o;
                    o.x = __shfl_xor_sync(0xffffffffu, cv[2 * c], 1);
                    o.y = __shfl_xor_sync(0xffffffffu, cv[2 * c + 1], 1);
                    const float2 m = make_float2(cv[2 * c], cv[2 * c + 1]);
                    x[c] = bwd ? o : m;
                    x[3 + c] = bwd ? m : o;
                }
            }
            float2 out[3];
#pragma unroll
            for (int r = 0; r < 3; r++) {
                float2 eta = make_float2(0.f, 0.f);
#pragma unroll
                for (int m = 0; m < 6; m++) eta = cfma(w.at(18 + 6 * r + m), x[m], eta);
                float2 Q;
                Q.x = __shfl_xor_sync(0xffffffffu, eta.x, 2);
                Q.y = __shfl_xor_sync(0xffffffffu, eta.y, 2);
                out[r] = up ? csub(eta, Q) : cadd(eta, Q);
            }
            if (mine0) {
                float *yp = ys + code.z + j * 3 * L::cw;
#pragma unroll
                for (int r = 0; r < 3; r++) {
                    float2 yo = ld_c<HALF>(yp + r * L::cw), tt, yn;
                    if constexpr (HALF) yo = cscale(yo, my_scale);
                    tt.x = fmaf(a.kappa, out[r].x, fv[r].x);
                    tt.y = fmaf(a.kappa, out[r].y, fv[r].y);
                    yn.x = fmaf(a.omega, tt.x - yo.x, yo.x);
                    yn.y = fmaf(a.omega, tt.y - yo.y, yo.y);
                    if constexpr (HALF) yn = cscale(yn, inv_scale);
                    st_c<HALF>(yp + r * L::cw, yn);
                }
            }
        }
        if (t + 1 < T) {
            if (CL && flag == 2) {
                __syncwarp();
                cg::this_cluster().barrier_arrive();
            }
            const int k2 = next(k1), nflag = a.flags[k2];
            const int p2 = position(k2, mine2);
            code = code1;
            if (p1 >= 0) {
                w.load(rec + (size_t)p1 * L::words);
                load_source(code.w);
            }
            if (p2 >= 0) {
                code1 = __ldg(a.quad + (size_t)p2 * 4 + j);
                if constexpr (!CL) {  // without a cluster the records of many blocks stream from memory
                    const float *pf = rec + (size_t)p2 * L::words - j * L::load_words;
#pragma unroll
                    for (int i = j * 32; i < L::words; i += 128) asm volatile("prefetch.global.L2 [%0];" ::"l"(pf + i));
                }
            }
            k1 = k2;
            p0 = p1; p1 = p2;
            mine0 = mine1; mine1 = mine2;
            if (CL && flag == 2) cg::this_cluster().barrier_wait();
            else if (flag == 1) __syncthreads();
            flag = nflag;
        }
    }
    // no CTA may leave its slab while a peer can still read it
    if (CL) cg::this_cluster().sync();
    else __syncthreads();
    for (int i = threadIdx.x; i < a.slab_vol * 6; i += blockDim.x) {
        const int sl = i / 6, q = i - 6 * sl;
        const int off = a.own_off[rank * a.slab_vol + sl];
        if (off < 0) continue;
        const float *yp = ys + (size_t)sl * a.ypitch + 2 * q * L::cw;
        float2 lo = ld_c<HALF>(yp), hi = ld_c<HALF>(yp + L::cw);
        if constexpr (HALF) {
            lo = cscale(lo, my_scale);
            hi = cscale(hi, my_scale);
        }
        a.y[(n0 + off) * 6 + q] = make_float4(lo.x, lo.y, hi.x, hi.y);
    }
}

// K3, thread form for the throughput regime (blocks that fit one CTA, many blocks per colour):
// one CTA per block with the block spinor y in shared memory, and every site update of a level
// done by one thread (the 8-direction projected hop, the clover product and the relaxation, as
// in K1), with a CTA barrier between levels.  The links and clover of each block are stored per
// block in level order and structure-of-arrays form ([block][element][level position]), so the
// threads of a level read consecutive addresses: the loads are coalesced and every byte is
// used.  A site update costs about 1,200 thread instructions.  The level order is the cluster
// form's, so the same values are read.
constexpr int kTsY = 28;  // padded words of one site's spinor in shared memory
constexpr int kTsMaxThreads = 256;
constexpr int kSoaLinks = 72;   // float2 per site: 8 hop links (U_mu(n) forward, U_mu(n - mu) backward)
constexpr int kSoaClover = 18;  // float4 per site: the packed clover field
constexpr size_t kSoaBytesPerSite = kSoaLinks * sizeof(float2) + kSoaClover * sizeof(float4);

__global__ void __launch_bounds__(kTsMaxThreads) k_ssor_soa(SsorArgs a) {
    extern __shared__ __align__(16) float sm[];
    if (a.gate && !a.gate[blockIdx.y].active) return;
    a.f += (size_t)blockIdx.y * 6 * a.V;
    a.y += (size_t)blockIdx.y * 6 * a.V;
    const int vol = a.vol, nch = a.nchunks;
    float *ys = sm;                                                // [vol][kTsY]
    int *cptr = reinterpret_cast<int *>(ys + (size_t)vol * kTsY);  // [nch + 1]
    int2 *csite = reinterpret_cast<int2 *>(cptr + ((nch + 1 + 3) & ~3));
    const long n0 = a.origin_site[blockIdx.x];
    const size_t gb = (size_t)a.gb0 + blockIdx.x;
    const float2 *lk = reinterpret_cast<const float2 *>(a.rec) + gb * kSoaLinks * vol;
    const float4 *cl = reinterpret_cast<const float4 *>(reinterpret_cast<const float2 *>(a.rec) +
                                                        (size_t)a.V * kSoaLinks) + gb * kSoaClover * vol;
    for (int i = threadIdx.x; i <= nch; i += blockDim.x) cptr[i] = a.chunk_ptr[i];
    for (int i = threadIdx.x; i < vol; i += blockDim.x) csite[i] = a.chunk_site[i];
    for (int i = threadIdx.x; i < vol * kTsY / 4; i += blockDim.x)
        reinterpret_cast<float4 *>(ys)[i] = make_float4(0.f, 0.f, 0.f, 0.f);
    __syncthreads();
    const int b0 = a.b[0], b1 = a.b[1], b2 = a.b[2], b3 = a.b[3];
    const int st1 = b0, st2 = b0 * b1, st3 = b0 * b1 * b2;
    auto ld_y = [&](int yl, float2 psi[12]) {
        const float4 *p = reinterpret_cast<const float4 *>(ys + yl * kTsY);
#pragma unroll
        for (int q = 0; q < 6; q++) {
            const float4 v = p[q];
            psi[2 * q] = make_float2(v.x, v.y);
            psi[2 * q + 1] = make_float2(v.z, v.w);
        }
    };
    for (int sw = 0; sw < a.nsweep; sw++)
        for (int k = 0; k < 2 * nch; k++) {
            const int ch = k < nch ? k : 2 * nch - 1 - k;
            for (int pos = cptr[ch] + threadIdx.x; pos < cptr[ch + 1]; pos += blockDim.x) {
                const int2 e = csite[pos];
                const int yl = e.x;
                int r = yl;
                const int y0 = r % b0; r /= b0;
                const int y1 = r % b1; r /= b1;
                const int y2 = r % b2;
                const int y3 = r / b2;
                float2 acc[12], psi[12], u[9];
#pragma unroll
                for (int q = 0; q < 12; q++) acc[q] = make_float2(0.f, 0.f);
                auto ld_u = [&](int d) {
#pragma unroll
                    for (int c = 0; c < 9; c++) u[c] = __ldg(lk + (size_t)(d * 9 + c) * vol + pos);
                };
                // in-block hops only (D_BB); a block never wraps around the lattice, so no boundary sign
                if (y0 + 1 < b0) { ld_y(yl + 1, psi); ld_u(0); hop_term<0, true>(psi, u, 1.f, acc); }
                if (y0 > 0) { ld_y(yl - 1, psi); ld_u(1); hop_term<0, false>(psi, u, 1.f, acc); }
                if (y1 + 1 < b1) { ld_y(yl + st1, psi); ld_u(2); hop_term<1, true>(psi, u, 1.f, acc); }
                if (y1 > 0) { ld_y(yl - st1, psi); ld_u(3); hop_term<1, false>(psi, u, 1.f, acc); }
                if (y2 + 1 < b2) { ld_y(yl + st2, psi); ld_u(4); hop_term<2, true>(psi, u, 1.f, acc); }
                if (y2 > 0) { ld_y(yl - st2, psi); ld_u(5); hop_term<2, false>(psi, u, 1.f, acc); }
                if (y3 + 1 < b3) { ld_y(yl + st3, psi); ld_u(6); hop_term<3, true>(psi, u, 1.f, acc); }
                if (y3 > 0) { ld_y(yl - st3, psi); ld_u(7); hop_term<3, false>(psi, u, 1.f, acc); }
                float fc[72];
#pragma unroll
                for (int q = 0; q < 18; q++) {
                    const float4 v = __ldg(cl + (size_t)q * vol + pos);
                    fc[4 * q] = v.x; fc[4 * q + 1] = v.y; fc[4 * q + 2] = v.z; fc[4 * q + 3] = v.w;
                }
                float2 fa[12];
                clover_mul<float, float2>(fc, acc, fa);
                float2 fv[12], yo[12];
                load_spinor(a.f, n0 + e.y, fv);
                ld_y(yl, yo);
                float4 *yp = reinterpret_cast<float4 *>(ys + yl * kTsY);
#pragma unroll
                for (int q = 0; q < 6; q++) {
                    float2 o[2];
#pragma unroll
                    for (int h = 0; h < 2; h++) {
                        const int c = 2 * q + h;
                        const float tx = fmaf(a.kappa, fa[c].x, fv[c].x), ty = fmaf(a.kappa, fa[c].y, fv[c].y);
                        o[h] = make_float2(fmaf(a.omega, tx - yo[c].x, yo[c].x), fmaf(a.omega, ty - yo[c].y, yo[c].y));
                    }
                    yp[q] = make_float4(o[0].x, o[0].y, o[1].x, o[1].y);
                }
            }
            __syncthreads();
        }
    for (int i = threadIdx.x; i < vol * 6; i += blockDim.x) {
        const int yl = i / 6, q = i - 6 * yl;
        a.y[(n0 + a.site_off[yl]) * 6 + q] = reinterpret_cast<const float4 *>(ys + yl * kTsY)[q];
    }
}

// SoA per-block fields of the thread form: links [gb][72][pos] (float2) for all blocks, then the
// clover planes [gb][18][pos] (float4); pos the level position of the site in its block
__global__ void k_sap_soa(float2 *__restrict__ lk, float4 *__restrict__ cl, const float2 *__restrict__ U,
                          const float4 *__restrict__ F, Geo g, BlockGeo bg, const int *__restrict__ pos_of,
                          const int *__restrict__ org0, const int *__restrict__ org1, int nblk0, long total) {
    const long i = blockIdx.x * (long)blockDim.x + threadIdx.x;
    if (i >= total) return;
    const int gb = (int)(i / bg.vol), yl = (int)(i % bg.vol);
    const int *o = gb < nblk0 ? org0 + 4 * gb : org1 + 4 * (gb - nblk0);
    int y[4], r = yl;
    for (int m = 0; m < 4; m++) { y[m] = r % bg.b[m]; r /= bg.b[m]; }
    const long gs[4] = {1, g.L[0], (long)g.L[0] * g.L[1], (long)g.L[0] * g.L[1] * g.L[2]};
    long n = 0;
    for (int m = 0; m < 4; m++) n += gs[m] * (o[m] + y[m]);
    const int pos = pos_of[yl];
    const size_t vol = bg.vol;
    for (int d = 0; d < 8; d++) {
        const int mu = d >> 1;
        const bool fwd = (d & 1) == 0;
        const int ym = y[mu] + (fwd ? 1 : -1);
        const bool in = ym >= 0 && ym < bg.b[mu];
        const long src = fwd ? n : n - gs[mu];
        for (int c = 0; c < 9; c++)
            lk[((size_t)gb * kSoaLinks + d * 9 + c) * vol + pos] =
                in ? U[(long)(mu * 9 + c) * g.V + src] : make_float2(0.f, 0.f);
    }
    for (int q = 0; q < kSoaClover; q++) cl[((size_t)gb * kSoaClover + q) * vol + pos] = F[(long)q * g.V + n];
}

// K4: after the block solve of colour c (y on colour-c sites):
//   colour-c sites:  x += y;  r -= D_cc y          (if upd_in)
//   other sites:     r += kappa F H_{c'c} y        (if upd_cross)
__global__ void __launch_bounds__(128) k_sap_hop(float4 *__restrict__ r, float4 *__restrict__ x,
                                                 const float4 *__restrict__ y, const float2 *__restrict__ U,
                                                 const float4 *__restrict__ F, float kappa, Geo g, BlockGeo bg,
                                                 int colour, int upd_in, int upd_cross,
                                                 const BicgScalars *__restrict__ gate) {
    chain_wait(r, x, y, gate);
    const long n = blockIdx.x * (long)blockDim.x + threadIdx.x;
    if (n >= g.V) return;
    if (gate && !gate[blockIdx.y].active) return;
    r += (size_t)blockIdx.y * 6 * g.V;
    x += (size_t)blockIdx.y * 6 * g.V;
    y += (size_t)blockIdx.y * 6 * g.V;
    int xc[4], yl[4];
    site_coords(g, n, xc);
    int col = 0;
    for (int m = 0; m < 4; m++) {
        col += xc[m] / bg.b[m];
        yl[m] = xc[m] % bg.b[m];
    }
    col &= 1;
    float2 acc[12];
#pragma unroll
    for (int q = 0; q < 12; q++) acc[q] = make_float2(0.f, 0.f);
    if (col == colour) {
        float2 yv[12], xv[12];
        load_spinor(y, n, yv);
        load_spinor_rw(x, n, xv);
#pragma unroll
        for (int q = 0; q < 12; q++) { xv[q].x += yv[q].x; xv[q].y += yv[q].y; }
        store_spinor(x, n, xv);
        if (!upd_in) return;
        masked_hops<true, false>(y, U, g, n, xc, yl, bg, acc);
        float fc[72];
        load_clover(F, g.V, n, fc);
        float2 fa[12], rv[12];
        clover_mul<float, float2>(fc, acc, fa);
        load_spinor_rw(r, n, rv);
#pragma unroll
        for (int q = 0; q < 12; q++) {
            // r -= y - kappa F H_BB y
            rv[q].x = rv[q].x - yv[q].x + kappa * fa[q].x;
            rv[q].y = rv[q].y - yv[q].y + kappa * fa[q].y;
        }
        store_spinor(r, n, rv);
    } else {
        if (!upd_cross) return;
        bool face = false;
        for (int m = 0; m < 4; m++) face |= (yl[m] == 0) || (yl[m] == bg.b[m] - 1);
        if (!face) return;
        masked_hops<false, false>(y, U, g, n, xc, yl, bg, acc);
        float fc[72];
        load_clover(F, g.V, n, fc);
        float2 fa[12], rv[12];
        clover_mul<float, float2>(fc, acc, fa);
        load_spinor_rw(r, n, rv);
#pragma unroll
        for (int q = 0; q < 12; q++) {
            rv[q].x = fmaf(kappa, fa[q].x, rv[q].x);
            rv[q].y = fmaf(kappa, fa[q].y, rv[q].y);
        }
        store_spinor(r, n, rv);
    }
}

// K3, even-odd alternative (block_solver = 1).  Sec. 3 names the even-odd site preconditioning
// of Luescher's SAP as the block solver that the ll-SSOR outperforms at equal cost.  Site parity
// p(n) = (n_0 + n_1 + n_2 + n_3) mod 2; H_BB links opposite parities, so D_BB x = f reduces to
// the Schur complement on the block's even sites,
//   Dhat = 1 - kappa^2 F_e H_eo F_o H_oe,  fhat = f_e + kappa F_e H_eo f_o,
// solved by nmr minimal-residual steps from x_e = 0 (r = fhat; p = Dhat r;
// alpha = <p, r> / <p, p>; x_e += alpha r; r -= alpha p), then x_o = f_o + kappa F_o H_oe x_e.
// One CTA per block (blockIdx.x) and right-hand side (blockIdx.y).  r, p (even sites) and
// t = F_o H_oe r (odd sites) live in lattice-sized scratch that only the block's CTA touches, so
// __syncthreads orders the phases (and L2 holds the block's vectors); values written in this
// launch are read back through coherent loads.
constexpr int kEoThreads = 256;

// out = F(n) sum of the in-block hops of src at site n
template <bool COHERENT>
__device__ __forceinline__ void block_FH(const float4 *src, const float2 *__restrict__ U,
                                         const float4 *__restrict__ F, const Geo &g, long n, const int xc[4],
                                         const int yl[4], const BlockGeo &bg, float2 out[12]) {
    float2 acc[12];
#pragma unroll
    for (int q = 0; q < 12; q++) acc[q] = make_float2(0.f, 0.f);
    masked_hops<true, COHERENT>(src, U, g, n, xc, yl, bg, acc);
    float fc[72];
    load_clover(F, g.V, n, fc);
    clover_mul<float, float2>(fc, acc, out);
}

__global__ void __launch_bounds__(kEoThreads) k_block_eo_mr(float4 *y, const float4 *__restrict__ f, float4 *R,
                                                            float4 *P, float4 *T, const float2 *__restrict__ U,
                                                            const float4 *__restrict__ F, float kappa, Geo g,
                                                            BlockGeo bg, const int *__restrict__ origin, int nmr,
                                                            const BicgScalars *__restrict__ gate) {
    if (gate && !gate[blockIdx.y].active) return;
    const size_t off = (size_t)blockIdx.y * 6 * g.V;
    y += off;
    f += off;
    R += off;
    P += off;
    T += off;
    const int *o = origin + 4 * blockIdx.x;
    const int par0 = (o[0] + o[1] + o[2] + o[3]) & 1;
    __shared__ double red[3][kEoThreads / 32];
    __shared__ float2 alpha_s;
    // block-local site i (lexicographic): global and block-local coordinates, global index, parity
    auto site = [&](int i, int xc[4], int yl[4]) -> long {
        int r = i;
        for (int m = 0; m < 4; m++) {
            yl[m] = r % bg.b[m];
            r /= bg.b[m];
            xc[m] = o[m] + yl[m];
        }
        return xc[0] + (long)g.L[0] * (xc[1] + (long)g.L[1] * (xc[2] + (long)g.L[2] * xc[3]));
    };
    auto odd = [&](const int yl[4]) { return ((par0 + yl[0] + yl[1] + yl[2] + yl[3]) & 1) != 0; };
    const float2 zero = make_float2(0.f, 0.f);
    // r = fhat and x_e = 0 on the even sites
    for (int i = threadIdx.x; i < bg.vol; i += blockDim.x) {
        int xc[4], yl[4];
        const long n = site(i, xc, yl);
        if (odd(yl)) continue;
        float2 h[12], v[12];
        block_FH<false>(f, U, F, g, n, xc, yl, bg, h);
        load_spinor(f, n, v);
#pragma unroll
        for (int q = 0; q < 12; q++) {
            v[q].x = fmaf(kappa, h[q].x, v[q].x);
            v[q].y = fmaf(kappa, h[q].y, v[q].y);
            h[q] = zero;
        }
        store_spinor(R, n, v);
        store_spinor(y, n, h);
    }
    __syncthreads();
    const float k2 = kappa * kappa;
    for (int it = 0; it < nmr; it++) {
        // t = F_o H_oe r on the odd sites
        for (int i = threadIdx.x; i < bg.vol; i += blockDim.x) {
            int xc[4], yl[4];
            const long n = site(i, xc, yl);
            if (!odd(yl)) continue;
            float2 h[12];
            block_FH<true>(R, U, F, g, n, xc, yl, bg, h);
            store_spinor(T, n, h);
        }
        __syncthreads();
        // p = r - kappa^2 F_e H_eo t on the even sites, with <p, r> and <p, p>
        float pr_re = 0.f, pr_im = 0.f, pp = 0.f;
        for (int i = threadIdx.x; i < bg.vol; i += blockDim.x) {
            int xc[4], yl[4];
            const long n = site(i, xc, yl);
            if (odd(yl)) continue;
            float2 h[12], rv[12];
            block_FH<true>(T, U, F, g, n, xc, yl, bg, h);
            load_spinor_rw(R, n, rv);
#pragma unroll
            for (int q = 0; q < 12; q++) {
                const float2 pv = make_float2(fmaf(-k2, h[q].x, rv[q].x), fmaf(-k2, h[q].y, rv[q].y));
                pr_re = fmaf(pv.x, rv[q].x, fmaf(pv.y, rv[q].y, pr_re));
                pr_im = fmaf(pv.x, rv[q].y, fmaf(-pv.y, rv[q].x, pr_im));
                pp = fmaf(pv.x, pv.x, fmaf(pv.y, pv.y, pp));
                h[q] = pv;
            }
            store_spinor(P, n, h);
        }
        double a0 = pr_re, a1 = pr_im, a2 = pp;
        for (int sft = 16; sft > 0; sft >>= 1) {
            a0 += __shfl_xor_sync(0xffffffffu, a0, sft);
            a1 += __shfl_xor_sync(0xffffffffu, a1, sft);
            a2 += __shfl_xor_sync(0xffffffffu, a2, sft);
        }
        const int warp = threadIdx.x >> 5;
        if ((threadIdx.x & 31) == 0) {
            red[0][warp] = a0;
            red[1][warp] = a1;
            red[2][warp] = a2;
        }
        __syncthreads();
        if (threadIdx.x == 0) {
            double s0 = 0, s1 = 0, s2 = 0;
            for (int w = 0; w < (int)(blockDim.x >> 5); w++) {
                s0 += red[0][w];
                s1 += red[1][w];
                s2 += red[2][w];
            }
            alpha_s = s2 > 0 ? make_float2((float)(s0 / s2), (float)(s1 / s2)) : zero;
        }
        __syncthreads();
        const float2 al = alpha_s;
        // x_e += alpha r, r -= alpha p
        for (int i = threadIdx.x; i < bg.vol; i += blockDim.x) {
            int xc[4], yl[4];
            const long n = site(i, xc, yl);
            if (odd(yl)) continue;
            float2 xv[12], rv[12], pv[12];
            load_spinor_rw(y, n, xv);
            load_spinor_rw(R, n, rv);
            load_spinor_rw(P, n, pv);
#pragma unroll
            for (int q = 0; q < 12; q++) {
                xv[q] = cfma(al, rv[q], xv[q]);
                rv[q] = cfma(make_float2(-al.x, -al.y), pv[q], rv[q]);
            }
            store_spinor(y, n, xv);
            store_spinor(R, n, rv);
        }
        __syncthreads();
    }
    // x_o = f_o + kappa F_o H_oe x_e
    for (int i = threadIdx.x; i < bg.vol; i += blockDim.x) {
        int xc[4], yl[4];
        const long n = site(i, xc, yl);
        if (!odd(yl)) continue;
        float2 h[12], v[12];
        block_FH<true>(y, U, F, g, n, xc, yl, bg, h);
        load_spinor(f, n, v);
#pragma unroll
        for (int q = 0; q < 12; q++) {
            v[q].x = fmaf(kappa, h[q].x, v[q].x);
            v[q].y = fmaf(kappa, h[q].y, v[q].y);
        }
        store_spinor(y, n, v);
    }
}

bool geometry_ok(const qcd_ctx *c, const int b[4], const int s[4]) {
    for (int m = 0; m < 4; m++) {
        if (b[m] < 1 || s[m] < 1 || c->lat.L[m] % b[m] != 0 || b[m] % s[m] != 0) return false;
        int nbk = c->lat.L[m] / b[m];
        if (nbk < 2 || nbk % 2 != 0) return false;
    }
    return true;
}

void free_plan(qcd_ctx *c) {
    SapPlan &p = c->plan;
    dev_free(c, p.d_origin[0]);  // one region holds every table
    dev_free(c, p.d_rec);
    p = SapPlan();
}

// Which CTA of the cluster owns (updates and stores) each site of the block.  C = 1: all.
// C > 1: the sites of every level are dealt round-robin over the C CTAs in ll order, so each
// CTA gets an equal share of every level (a t-slab split would give each CTA a band of levels
// and leave most CTAs idle at the ends of the chain); neighbours then mostly sit in other
// CTAs and are read through distributed shared memory.
void assign_owners(SapPlan &np, int C) {
    np.h_own.assign(np.vol, 0);
    std::vector<int> cnt(C, 0);
    if (C == 1) {  // one CTA: the block spinor in natural site order
        for (int yl = 0; yl < np.vol; yl++) np.h_own[yl] = yl;
        cnt[0] = np.vol;
    } else {
        for (int st = 0; st < np.nsteps; st++)
            for (int k = np.h_step_ptr[st]; k < np.h_step_ptr[st + 1]; k++) {
                const int r = (k - np.h_step_ptr[st]) % C;
                np.h_own[np.h_step_site[k]] = (r << 24) | cnt[r]++;
            }
    }
    np.slab_vol = *std::max_element(cnt.begin(), cnt.end());
    np.h_own_off.assign((size_t)C * np.slab_vol, -1);
    for (int yl = 0; yl < np.vol; yl++)
        np.h_own_off[(size_t)(np.h_own[yl] >> 24) * np.slab_vol + (np.h_own[yl] & 0xffffff)] = np.h_site_off[yl];
}

// Deals the block over C CTAs (assign_owners) and cuts every step (level) of each CTA into
// chunks of at most maxslots sites, of equal size: the steps that the kernel runs.
void make_chunks(SapPlan &np, int C, int maxslots) {
    np.C = C;
    assign_owners(np, C);
    std::vector<std::vector<int>> per(C);
    std::vector<std::vector<int>> lists(C);  // chunk lists per CTA
    std::vector<std::vector<int>> ptr(C, std::vector<int>(1, 0));
    int nchunks = 0, nslot = 1;
    for (int st = 0; st < np.nsteps; st++) {
        for (auto &v : per) v.clear();
        for (int k = np.h_step_ptr[st]; k < np.h_step_ptr[st + 1]; k++) {
            const int yl = np.h_step_site[k];
            per[np.h_own[yl] >> 24].push_back(yl);
        }
        size_t most = 1;
        for (auto &v : per) most = std::max(most, v.size());
        const int nc = (int)((most + maxslots - 1) / maxslots);
        for (int j = 0; j < nc; j++) {
            for (int r = 0; r < C; r++) {
                const int sz = (int)per[r].size();
                const int lo = (int)((long)j * sz / nc), hi = (int)((long)(j + 1) * sz / nc);
                for (int q = lo; q < hi; q++) lists[r].push_back(per[r][q]);
                nslot = std::max(nslot, hi - lo);
                ptr[r].push_back((int)lists[r].size());
            }
            nchunks++;
        }
    }
    np.nchunks = nchunks;
    np.nslot = nslot;
    np.h_chunk_ptr.clear();
    np.h_chunk_site.clear();
    for (int r = 0; r < C; r++) {
        const int off = (int)np.h_chunk_site.size();
        for (int v : ptr[r]) np.h_chunk_ptr.push_back(off + v);
        np.h_chunk_site.insert(np.h_chunk_site.end(), lists[r].begin(), lists[r].end());
    }
}

// Barriers of the timeline.  A site reads its in-block neighbours (those owned
// by other CTAs through distributed shared memory).  Each such read must come after the
// neighbour's latest earlier write (barrier in (t_w, t]) and before its next
// write (barrier in (t, t_n]), unless the same warp does both (the own value).
// The intervals are taken over three sweeps and stabbed greedily, first those
// of neighbours owned by other CTAs with cluster barriers (flag 2), then the rest
// with CTA barriers (flag 1) where no barrier stabs them yet; the positions,
// folded modulo one sweep, give a periodic pattern that stabs every interval of
// any number of sweeps (no interval spans a whole sweep, because every site is
// written twice per sweep).  Position 0 is the barrier after the zero fill.
void make_flags(SapPlan &np) {
    const int P = 2 * np.nchunks;
    np.h_flags.assign(P, 0);
    std::vector<int> chunk_of(np.vol, -1);
    for (int r = 0; r < np.C; r++)
        for (int ch = 0; ch < np.nchunks; ch++)
            for (int k = np.h_chunk_ptr[r * (np.nchunks + 1) + ch]; k < np.h_chunk_ptr[r * (np.nchunks + 1) + ch + 1]; k++)
                chunk_of[np.h_chunk_site[k]] = ch;
    auto writes = [&](int yl, std::vector<int> &w) {
        w.clear();
        const int ch = chunk_of[yl];
        for (int sw = 0; sw < 3; sw++) {
            w.push_back(sw * P + ch);
            w.push_back(sw * P + P - 1 - ch);
        }
        std::sort(w.begin(), w.end());
    };
    std::vector<std::pair<int, int>> remote, local;  // (lo, hi]: need a barrier p with lo < p <= hi
    std::vector<int> wi, wj;
    for (int yl = 0; yl < np.vol; yl++) {
        int y[4], r = yl;
        for (int m = 0; m < 4; m++) { y[m] = r % np.b[m]; r /= np.b[m]; }
        int stride = 1;
        for (int m = 0; m < 4; m++) {
            for (int dir = -1; dir <= 1; dir += 2) {
                const int ym = y[m] + dir;
                if (ym < 0 || ym >= np.b[m]) continue;
                const int nb = yl + dir * stride;
                const bool other = (np.h_own[yl] >> 24) != (np.h_own[nb] >> 24);
                auto &iv = other ? remote : local;
                writes(yl, wi);
                writes(nb, wj);
                for (int t : wi) {
                    int prev = -1, next = -1;
                    for (int w : wj) {
                        if (w < t) prev = w;
                        if (w > t && next < 0) next = w;
                    }
                    iv.push_back({prev, t});            // read after the latest write (prev = -1: zero fill)
                    if (next >= 0) iv.push_back({t, next});  // read before the next write
                }
            }
            stride *= np.b[m];
        }
    }
    auto by_hi = [](const std::pair<int, int> &u, const std::pair<int, int> &v) { return u.second < v.second; };
    auto stabbed = [&](const std::pair<int, int> &v) {
        for (int p = v.first + 1; p <= v.second; p++)
            if (p == 0 || np.h_flags[p % P]) return true;
        return false;
    };
    std::sort(remote.begin(), remote.end(), by_hi);
    for (auto &v : remote)
        if (!stabbed(v) && v.second > 0) np.h_flags[v.second % P] = 2;
    std::sort(local.begin(), local.end(), by_hi);
    for (auto &v : local)
        if (!stabbed(v) && v.second > 0) np.h_flags[v.second % P] = 1;
}

// The cluster form with C CTAs per block: the instance of k_ssor_quad, its steps and its shared memory.
// False where the block has fewer sites, a CTA's spinors exceed slab_limit or its shared memory kSmemLimit.
bool make_quad_plan(SapPlan &np, int C, size_t slab_limit) {
    if (C > np.vol) return false;
    const long ctas = (long)(np.nb[0] * np.nb[1]) * (np.nb[2] * np.nb[3]) / 2 * C;  // of one colour
    np.form = C > 1 ? kFormCluster : ctas <= np.sms ? kFormAlone : kFormShared;
    const int most[] = {kMaxRunShared, kMaxRunAlone, kMaxRun};
    make_chunks(np, C, most[np.form]);
    np.nwarps = (np.nslot + 7) / 8;
    const int plain = np.half ? Rec<true>::ywords : Rec<false>::ywords;
    auto bytes = [&](int pitch) {
        return sizeof(float) * ((size_t)(np.slab_vol + 1) * pitch + kMaxCluster + 4) + sizeof(int) * (np.nchunks + 1);
    };
    // FP32: 28 words from spinor to spinor spread 16-byte accesses over all banks (24: over half of them)
    np.ypitch = !np.half && bytes(28) <= kSmemLimit ? 28 : plain;
    np.smem_bytes = bytes(np.ypitch);
    return sizeof(float) * plain * (size_t)np.slab_vol <= slab_limit && np.smem_bytes <= kSmemLimit;
}

// the neighbour codes (SsorArgs::quad) of the cluster form, in the order of the chunks' list of sites
void make_codes(SapPlan &np) {
    np.h_quad.assign(16 * (size_t)np.vol, 0);
    for (int k = 0; k < np.vol; k++) {
        const int yl = np.h_chunk_site[k], own = np.h_own[yl];
        int code[8];
        int y = yl, stride = 1;
        for (int m = 0; m < 4; m++) {
            const int ym = y % np.b[m];
            y /= np.b[m];
            for (int back = 0; back < 2; back++) {
                const bool leaves = back ? ym == 0 : ym + 1 == np.b[m];
                const int o = leaves ? ((own & ~0xffffff) | np.slab_vol) : np.h_own[yl + (back ? -stride : stride)];
                code[2 * m + back] = (o & ~0xffffff) | (o & 0xffffff) * np.ypitch;
            }
            stride *= np.b[m];
        }
        for (int j = 0; j < 4; j++) {
            int *q = &np.h_quad[16 * (size_t)k + 4 * j];
            q[0] = code[j]; q[1] = code[j + 4]; q[2] = (own & 0xffffff) * np.ypitch; q[3] = np.h_site_off[yl];
        }
    }
}

}  // namespace

void sap_plan_flags(SapPlan &p) { make_flags(p); }

bool sap_geometry_ok(const qcd_ctx *c, const int b[4], const int s[4]) { return geometry_ok(c, b, s); }

int sap_plan_host(const qcd_ctx *c, const int b[4], const int s[4], SapPlan &np, int min_ctas, bool half) {
    if (!geometry_ok(c, b, s)) return QCD_ERR_ARG;
    np = SapPlan();
    np.half = half;
    std::memcpy(np.b, b, sizeof(np.b));
    std::memcpy(np.s, s, sizeof(np.s));
    int nq[4];
    for (int m = 0; m < 4; m++) {
        np.nb[m] = c->lat.L[m] / b[m];
        nq[m] = b[m] / s[m];
    }
    np.vol = b[0] * b[1] * b[2] * b[3];
    const int nsb = nq[0] * nq[1] * nq[2] * nq[3];
    // ll order: order[key] = block-local lexicographic site index
    std::vector<int> order(np.vol);
    for (int yl = 0; yl < np.vol; yl++) {
        int y[4], r = yl;
        for (int m = 0; m < 4; m++) { y[m] = r % b[m]; r /= b[m]; }
        int lam = 0, sig = 0;
        for (int m = 3; m >= 0; m--) {
            lam = lam * s[m] + y[m] % s[m];
            sig = sig * nq[m] + y[m] / s[m];
        }
        order[lam * nsb + sig] = yl;
    }
    // Level schedule of the ll order: a site's level is one more than the highest level of its
    // in-block neighbours that come earlier in the order.  Neighbours never share a level, and
    // every earlier neighbour of a site sits on a lower level and every later one on a higher
    // level, so updating the levels one after the other (in any order within a level) reads
    // exactly the values the sequential ll sweep reads: the same result, bit for bit, in as many
    // dependent steps as the longest chain of the order (12 instead of 2592 for 6^3 x 12 blocks
    // with 3^3 x 6 sub-blocks).  The backward sweep runs the levels in reverse.
    std::vector<int> key_of(np.vol), level(np.vol, 0);
    for (int k = 0; k < np.vol; k++) key_of[order[k]] = k;
    int nlev = 0;
    for (int k = 0; k < np.vol; k++) {
        const int yl = order[k];
        int y[4], r = yl;
        for (int m = 0; m < 4; m++) { y[m] = r % b[m]; r /= b[m]; }
        int lv = 0, stride = 1;
        for (int m = 0; m < 4; m++) {
            if (y[m] + 1 < b[m] && key_of[yl + stride] < k) lv = std::max(lv, level[yl + stride] + 1);
            if (y[m] > 0 && key_of[yl - stride] < k) lv = std::max(lv, level[yl - stride] + 1);
            stride *= b[m];
        }
        level[yl] = lv;
        nlev = std::max(nlev, lv + 1);
    }
    np.h_step_ptr.push_back(0);
    for (int lv = 0; lv < nlev; lv++) {
        for (int k = 0; k < np.vol; k++)
            if (level[order[k]] == lv) np.h_step_site.push_back(order[k]);
        if (lv + 1 < nlev) np.h_step_ptr.push_back((int)np.h_step_site.size());
    }
    np.h_step_ptr.push_back(np.vol);
    np.nsteps = (int)np.h_step_ptr.size() - 1;
    for (int k = 0; k < np.nsteps; k++) np.max_step = std::max(np.max_step, np.h_step_ptr[k + 1] - np.h_step_ptr[k]);
    // block origins per colour
    for (int B3 = 0; B3 < np.nb[3]; B3++)
        for (int B2 = 0; B2 < np.nb[2]; B2++)
            for (int B1 = 0; B1 < np.nb[1]; B1++)
                for (int B0 = 0; B0 < np.nb[0]; B0++) {
                    const int col = (B0 + B1 + B2 + B3) & 1;
                    np.h_origin[col].insert(np.h_origin[col].end(), {B0 * b[0], B1 * b[1], B2 * b[2], B3 * b[3]});
                }
    for (int col = 0; col < 2; col++) {
        np.nblk[col] = (int)np.h_origin[col].size() / 4;
        for (int k = 0; k < np.nblk[col]; k++) {
            const int *o = &np.h_origin[col][4 * k];
            np.h_origin_site[col].push_back(o[0] + c->lat.L[0] * (o[1] + c->lat.L[1] * (o[2] + c->lat.L[2] * o[3])));
        }
    }
    np.h_site_off.resize(np.vol);
    for (int yl = 0; yl < np.vol; yl++) {
        int y[4], r = yl;
        for (int m = 0; m < 4; m++) { y[m] = r % b[m]; r /= b[m]; }
        np.h_site_off[yl] = y[0] + c->lat.L[0] * (y[1] + c->lat.L[1] * (y[2] + c->lat.L[2] * y[3]));
    }
    int sms = c->sms_override;
    if (sms < 1 &&
        (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, c->device) != cudaSuccess || sms < 1)) {
        cudaGetLastError();
        sms = 1;
    }
    np.sms = sms;
    // the right-hand-side tiled thread form on request (min_ctas == -2), the block spinor of
    // one right-hand side in one CTA
    if (min_ctas == -2) {
        make_chunks(np, 1, 1 << 20);  // one chunk per level, in level order (diagnostics)
        if (np.vol + kTileZeroSlotsHalf < (1 << 16)) {  // slots are 16-bit
            tile_make_positions(np);
            if (tile_positions_valid(np) && tile_smem_bytes(np, 1) <= kTileSmemLimit) {
                np.tile = true;
                tile_level_table(np);
                np.nwarps = 0;
                np.smem_bytes = tile_smem_bytes(np, 1);
                return QCD_OK;
            }
        }
        // the block spinor does not fit one CTA: the cluster form stands in
        np.h_tile_pos.clear();
    }
    // the thread form on request (min_ctas = -1), FP32 storage, the block spinor in one CTA
    if (min_ctas == -1 && !half) {
        make_chunks(np, 1, 1 << 20);  // one chunk per level, in level order
        const size_t smem = (size_t)np.vol * kTsY * 4 + sizeof(int) * ((np.nchunks + 1 + 3) & ~3) +
                            sizeof(int2) * ((np.vol + 1) & ~1);
        if (smem <= kSmemLimit) {
            np.thread = true;
            np.nwarps = std::min(kTsMaxThreads / 32, (np.nslot + 31) / 32);
            np.smem_bytes = smem;
            np.h_pos.assign(np.vol, 0);
            for (int k = 0; k < np.vol; k++) np.h_pos[np.h_chunk_site[k]] = k;
            make_flags(np);
            return QCD_OK;
        }
    }
    // CTAs per block.  With min_ctas >= 1 the smallest C >= min_ctas whose spinors keep to the slab limit; with
    // min_ctas = 0 the smallest such power of two, and then as many (up to 8, the portable cluster size) as keep
    // one colour's clusters within the SM count.  A block too large for that takes 16 CTAs.
    // Few CTAs with large slabs leave an SM few warps, and a C that is no power of two breaks the dealing of
    // whole sub-blocks to CTAs (two sweeps, one cycle, one right-hand side, us): 32^3x64, 8^4 blocks, FP32: C = 2
    // (192 KB) 2881, 3 3913, 4 (96 KB) 3021, 5 5264, 8 3856; FP16: 1 (192 KB) 6541, 2 (96 KB) 2005, 3 2408, 4 2024;
    // 48^3x32, 8^2x12x4, FP32: 2 (144 KB) 4459, 3 7221, 4 4780; 24^3x48, 6^3x8, FP32: 1 (162 KB) 2002, 2 999, 3 1613,
    // 4 843; 12^4, FP16: 5 1663, 6 1356, 8 (122 KB) 1742, 10 1485, 16 1178, FP32: 10 (194 KB) 2652, 16 (122 KB) 1468.
    // Filling the SMs, 12^3x24, 6^3x12 blocks, 3^3x6 sub-blocks, 4 sweeps and cycles: C = 4 1798 us, 8 1159, 12
    // 1545, 16 1201; natural order 3921, 3161, 2882, 3013; 16^3x32, 8^4 blocks, FP16: 300, 241, 217, 252.
    const int nblk1 = np.nb[0] * np.nb[1] * np.nb[2] * np.nb[3] / 2;
    int Cuse = 0;
    for (int C = std::max(1, min_ctas); C <= kMaxCluster && !Cuse; C += min_ctas >= 1 ? 1 : C)
        if (make_quad_plan(np, C, half ? kSlabLimitHalf : kSlabLimit)) Cuse = C;
    if (!Cuse) Cuse = kMaxCluster;
    if (min_ctas <= 0)
        for (int C = 2; C <= 8; C *= 2)
            if (C > Cuse && C <= np.vol && (long)nblk1 * C <= sms) Cuse = C;  // (a site per CTA at least)
    if (!make_quad_plan(np, Cuse, kSmemLimit)) return QCD_ERR_ARG;
    make_flags(np);
    make_codes(np);
    return QCD_OK;
}

size_t sap_table_bytes(const SapPlan &p) {
    auto up16 = [](size_t x) { return (x + 15) & ~(size_t)15; };
    return up16(sizeof(int) * p.h_origin[0].size()) + up16(sizeof(int) * p.h_origin[1].size()) +
           up16(sizeof(int) * p.h_origin_site[0].size()) + up16(sizeof(int) * p.h_origin_site[1].size()) +
           up16(sizeof(int) * p.h_chunk_ptr.size()) + up16(sizeof(int2) * p.h_chunk_site.size()) +
           up16(sizeof(int) * p.h_site_off.size()) + up16(p.h_flags.size()) + up16(sizeof(int) * p.h_own_off.size()) + up16(sizeof(int) * p.h_pos.size()) +
           up16(sizeof(int4) * p.h_tile_pos.size()) + up16(sizeof(int) * p.h_quad.size()) +
           (p.tile ? up16(sizeof(int) * p.h_tile_site.size()) + up16(sizeof(int4) * p.h_tile_item.size()) : 0);
}

// Copies every table of the plan into one device region (sap_table_bytes long) on the
// context stream and points the plan's device pointers into it.
int sap_upload_tables(qcd_ctx *c, SapPlan &p, void *region) {
    auto up16 = [](size_t x) { return (x + 15) & ~(size_t)15; };
    char *at = static_cast<char *>(region);
    auto put = [&](const void *src, size_t bytes) -> void * {
        void *dst = at;
        if (bytes) {
            cudaError_t e = cudaMemcpyAsync(dst, src, bytes, cudaMemcpyHostToDevice, c->stream);
            if (e != cudaSuccess) return nullptr;
        }
        at += up16(bytes);
        return dst;
    };
    std::vector<int2> cs(p.h_chunk_site.size());
    for (size_t k = 0; k < cs.size(); k++) cs[k] = make_int2(p.h_chunk_site[k], p.h_site_off[p.h_chunk_site[k]]);
    p.d_origin[0] = (int *)put(p.h_origin[0].data(), sizeof(int) * p.h_origin[0].size());
    p.d_origin[1] = (int *)put(p.h_origin[1].data(), sizeof(int) * p.h_origin[1].size());
    p.d_origin_site[0] = (int *)put(p.h_origin_site[0].data(), sizeof(int) * p.h_origin_site[0].size());
    p.d_origin_site[1] = (int *)put(p.h_origin_site[1].data(), sizeof(int) * p.h_origin_site[1].size());
    p.d_chunk_ptr = (int *)put(p.h_chunk_ptr.data(), sizeof(int) * p.h_chunk_ptr.size());
    p.d_chunk_site = (int2 *)put(cs.data(), sizeof(int2) * cs.size());
    p.d_site_off = (int *)put(p.h_site_off.data(), sizeof(int) * p.h_site_off.size());
    p.d_flags = (unsigned char *)put(p.h_flags.data(), p.h_flags.size());
    p.d_own_off = (int *)put(p.h_own_off.data(), sizeof(int) * p.h_own_off.size());
    p.d_pos = p.h_pos.empty() ? nullptr : (int *)put(p.h_pos.data(), sizeof(int) * p.h_pos.size());
    p.d_quad = p.h_quad.empty() ? nullptr : (int4 *)put(p.h_quad.data(), sizeof(int) * p.h_quad.size());
    p.d_tile_pos = p.tile ? (int4 *)put(p.h_tile_pos.data(), sizeof(int4) * p.h_tile_pos.size()) : nullptr;
    p.d_tile_site = p.tile ? (int *)put(p.h_tile_site.data(), sizeof(int) * p.h_tile_site.size()) : nullptr;
    p.d_tile_item = p.tile ? (int4 *)put(p.h_tile_item.data(), sizeof(int4) * p.h_tile_item.size()) : nullptr;
    if (!p.d_origin[0] || !p.d_origin[1] || !p.d_origin_site[0] || !p.d_origin_site[1] || !p.d_chunk_ptr ||
        !p.d_chunk_site || !p.d_site_off || !p.d_flags || !p.d_own_off || (p.thread && !p.d_pos) ||
        (!p.h_quad.empty() && !p.d_quad) ||
        (p.tile && (!p.d_tile_pos || !p.d_tile_site || !p.d_tile_item)))
        return cuda_fail(c, cudaGetLastError(), "cudaMemcpyAsync(SAP tables)");
    // the host vectors may be released only once the copies have consumed them
    QCD_CUDA(c, cudaStreamSynchronize(c->stream));
    return QCD_OK;
}

size_t sap_record_bytes(const SapPlan &p) {
    if (p.tile)
        return (size_t)(p.nblk[0] + p.nblk[1]) * p.vol * (p.half ? kTileRecordBytesHalf : kTileRecordBytes);
    if (p.thread) return (size_t)(p.nblk[0] + p.nblk[1]) * p.vol * kSoaBytesPerSite;
    return (size_t)(p.nblk[0] + p.nblk[1]) * p.vol * (p.half ? Rec<true>::words : Rec<false>::words) * sizeof(float);
}

int sap_build_records(qcd_ctx *c, SapPlan &p, float *rec) {
    Geo g;
    for (int m = 0; m < 4; m++) g.L[m] = c->lat.L[m];
    g.V = c->lat.V;
    g.bc_t = c->bc_t;
    BlockGeo bg;
    for (int m = 0; m < 4; m++) bg.b[m] = p.b[m];
    bg.vol = p.vol;
    const long total = (long)(p.nblk[0] + p.nblk[1]) * p.vol;
    cudaEvent_t ev;
    prof_begin(c, QCD_K_OTHER, &ev);
    field_kernel(c);
    if (p.tile) {
        int trc = tile_build_records(c, p, rec);
        if (trc) return trc;
    } else if (p.thread) {
        float2 *lk = reinterpret_cast<float2 *>(rec);
        float4 *cl = reinterpret_cast<float4 *>(lk + (size_t)total * kSoaLinks);
        k_sap_soa<<<(unsigned)((total + 127) / 128), 128, 0, c->stream>>>(lk, cl, c->U32, c->F32, g, bg, p.d_pos,
                                                                           p.d_origin[0], p.d_origin[1], p.nblk[0], total);
    } else if (p.half)
        k_sap_records<true><<<(unsigned)((total + 127) / 128), 128, 0, c->stream>>>(
            rec, c->U32, c->F32, g, bg, p.d_chunk_site, p.d_origin[0], p.d_origin[1], p.nblk[0], total);
    else
        k_sap_records<false><<<(unsigned)((total + 127) / 128), 128, 0, c->stream>>>(
            rec, c->U32, c->F32, g, bg, p.d_chunk_site, p.d_origin[0], p.d_origin[1], p.nblk[0], total);
    int rc = prof_end(c, QCD_K_OTHER, ev);
    if (rc) return rc;
    p.d_rec = rec;
    p.rec_version = c->field_version;
    return QCD_OK;
}

void sap_invalidate(qcd_ctx *c) { free_plan(c); }

int sap_prepare(qcd_ctx *c, const int b[4], const int s[4], bool half) {
    if (!geometry_ok(c, b, s))
        return fail(c, QCD_ERR_ARG, "SAP geometry: need L % block == 0, L/block even and >= 2, block % subblock == 0");
    SapPlan &p = c->plan;
    if (!(p.vol && std::equal(b, b + 4, p.b) && std::equal(s, s + 4, p.s) && p.half == half)) {
        free_plan(c);
        SapPlan np;
        if (sap_plan_host(c, b, s, np, c->sap_min_ctas, half) != QCD_OK)
            return fail(c, QCD_ERR_ARG, "SAP block too large for the shared memory of a cluster of 16 CTAs");
        void *region = nullptr;
        int rc = dev_alloc(c, &region, sap_table_bytes(np));
        if (rc) return rc;
        if ((rc = sap_upload_tables(c, np, region))) {
            dev_free(c, region);
            return rc;
        }
        float *rec = nullptr;
        if (sap_record_bytes(np) && (rc = dev_alloc(c, (void **)&rec, sap_record_bytes(np)))) {
            dev_free(c, region);
            return rc;
        }
        np.d_rec = rec;
        np.rec_version = -1;
        c->plan = np;
    }
    if (c->plan.rec_version != c->field_version) return sap_build_records(c, c->plan, c->plan.d_rec);
    return QCD_OK;
}

int sap_apply(qcd_ctx *c, float4 *x, const float4 *v, float4 *work, double omega, int nsweep, int nsap, int nrhs,
              const BicgScalars *gate, int block_solver) {
    if (block_solver == 1) return sap_apply_eo(c, c->plan, x, v, work, nsweep, nsap, nrhs, gate);
    return sap_apply_plan(c, c->plan, x, v, work, omega, nsweep, nsap, nrhs, gate);
}

int sap_apply_eo(qcd_ctx *c, const SapPlan &p, float4 *x, const float4 *v, float4 *work, int nmr, int nsap, int nrhs,
                 const BicgScalars *gate) {
    const long V = c->lat.V;
    const size_t vec = 6 * (size_t)V * nrhs;  // float4 per spinor field of nrhs right-hand sides
    float4 *r = work, *y = work + vec, *R = work + 2 * vec, *P = work + 3 * vec, *T = work + 4 * vec;
    Geo g;
    for (int m = 0; m < 4; m++) g.L[m] = c->lat.L[m];
    g.V = V;
    g.bc_t = c->bc_t;
    BlockGeo bg;
    for (int m = 0; m < 4; m++) bg.b[m] = p.b[m];
    bg.vol = p.vol;
    int rc;
    if ((rc = blas_copy(c, r, v, sizeof(float4) * vec))) return rc;
    if ((rc = blas_zero(c, x, sizeof(float4) * vec))) return rc;
    for (int j = 0; j < nsap; j++) {
        for (int col = 0; col < 2; col++) {
            cudaEvent_t ev;
            prof_begin(c, QCD_K_SSOR, &ev);
            k_block_eo_mr<<<dim3(p.nblk[col], nrhs), kEoThreads, 0, c->stream>>>(
                y, r, R, P, T, c->U32, c->F32, (float)c->kappa, g, bg, p.d_origin[col], nmr, gate);
            cudaError_t e = cudaGetLastError();
            if (e != cudaSuccess) return cuda_fail(c, e, "launch of the even-odd block kernel");
            if ((rc = prof_end(c, QCD_K_SSOR, ev))) return rc;
            const int last = (j == nsap - 1);
            prof_begin(c, QCD_K_SAPHOP, &ev);
            launch_chained(c, k_sap_hop, dim3((unsigned)((V + 127) / 128), nrhs), 128, 0, r, x, y, c->U32, c->F32,
                           (float)c->kappa, g, bg, col, !last, !(last && col == 1), gate);
            if ((rc = prof_end(c, QCD_K_SAPHOP, ev))) return rc;
        }
    }
    return QCD_OK;
}

int sap_apply_plan(qcd_ctx *c, const SapPlan &p, float4 *x, const float4 *v, float4 *work, double omega, int nsweep,
                   int nsap, int nrhs, const BicgScalars *gate) {
    const long V = c->lat.V;
    float4 *r = work, *y = work + 6 * V * nrhs;
    Geo g;
    for (int m = 0; m < 4; m++) g.L[m] = c->lat.L[m];
    g.V = V;
    g.bc_t = c->bc_t;
    BlockGeo bg;
    for (int m = 0; m < 4; m++) bg.b[m] = p.b[m];
    bg.vol = p.vol;
    static std::atomic<unsigned long long> attr_done{0};
    static std::mutex attr_mu;
    if (int arc = once_per_device(attr_done, attr_mu, c->device, [&]() -> int {
            const void *ks[] = {(const void *)k_ssor_quad<false, 0>, (const void *)k_ssor_quad<true, 0>,
                                (const void *)k_ssor_quad<false, 1>, (const void *)k_ssor_quad<true, 1>,
                                (const void *)k_ssor_quad<false, 2>, (const void *)k_ssor_quad<true, 2>};
            for (const void *k : ks) {
                QCD_CUDA(c, cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmemLimit));
                QCD_CUDA(c, cudaFuncSetAttribute(k, cudaFuncAttributeNonPortableClusterSizeAllowed, 1));
            }
            QCD_CUDA(c, cudaFuncSetAttribute(k_ssor_soa, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmemLimit));
            return tile_set_attributes(c);
        }))
        return arc;
    SsorArgs a;
    a.y = y;
    a.f = r;
    a.kappa = (float)c->kappa;
    a.omega = (float)omega;
    a.nsweep = nsweep;
    a.V = V;
    a.vol = p.vol;
    a.C = p.C;
    a.slab_vol = p.slab_vol;
    a.nchunks = p.nchunks;
    a.ypitch = p.ypitch;
    a.chunk_ptr = p.d_chunk_ptr;
    a.quad = p.d_quad;
    a.chunk_site = p.d_chunk_site;
    a.site_off = p.d_site_off;
    a.own_off = p.d_own_off;
    a.flags = p.d_flags;
    a.gate = gate;
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute attr[2];  // (the second as in launch_chained)
    attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[1].val.programmaticStreamSerializationAllowed = 1;
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = p.C;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.dynamicSmemBytes = p.smem_bytes;
    cfg.stream = c->stream;
    cfg.attrs = attr;
    int rc;
    if (p.tile) return tile_sap_apply(c, p, x, v, r, y, omega, nsweep, nsap, nrhs, gate);
    if ((rc = blas_copy(c, r, v, sizeof(float4) * 6 * V * nrhs))) return rc;
    if ((rc = blas_zero(c, x, sizeof(float4) * 6 * V * nrhs))) return rc;
    for (int j = 0; j < nsap; j++) {
        for (int col = 0; col < 2; col++) {
            cudaEvent_t ev;
            a.rec = p.d_rec ? reinterpret_cast<const float4 *>(p.d_rec) +
                                  (size_t)(col ? p.nblk[0] : 0) * p.vol * ((p.half ? Rec<true>::words : Rec<false>::words) / 4)
                            : nullptr;
            a.origin_site = p.d_origin_site[col];
            cfg.gridDim = dim3(p.nblk[col] * p.C, nrhs);
            cfg.blockDim = dim3(32 * p.nwarps);
            prof_begin(c, QCD_K_SSOR, &ev);
            cudaError_t e;
            if (p.thread) {
                SsorArgs at = a;
                at.rec = reinterpret_cast<const float4 *>(p.d_rec);
                at.gb0 = col ? p.nblk[0] : 0;
                for (int m = 0; m < 4; m++) at.b[m] = p.b[m];
                k_ssor_soa<<<dim3(p.nblk[col], nrhs), 32 * p.nwarps, p.smem_bytes, c->stream>>>(at);
                e = cudaGetLastError();
            } else {
                static constexpr void (*kKernel[2][3])(SsorArgs) = {
                    {k_ssor_quad<false, 0>, k_ssor_quad<false, 1>, k_ssor_quad<false, 2>},
                    {k_ssor_quad<true, 0>, k_ssor_quad<true, 1>, k_ssor_quad<true, 2>}};
                void (*kern)(SsorArgs) = kKernel[p.half][p.form];
                cfg.numAttrs = c->fields_fresh ? 1 : 2;
                c->fields_fresh = false;
                e = cudaLaunchKernelEx(&cfg, kern, a);
            }
            if (e != cudaSuccess) return cuda_fail(c, e, "launch of the SSOR block kernel");
            if ((rc = prof_end(c, QCD_K_SSOR, ev))) return rc;
            const int last = (j == nsap - 1);
            prof_begin(c, QCD_K_SAPHOP, &ev);
            launch_chained(c, k_sap_hop, dim3((unsigned)((V + 127) / 128), nrhs), 128, 0, r, x, y, c->U32, c->F32,
                           (float)c->kappa, g, bg, col, !last, !(last && col == 1), gate);
            if ((rc = prof_end(c, QCD_K_SAPHOP, ev))) return rc;
        }
    }
    return QCD_OK;
}

}  // namespace qcd
