// K7: the learned correction (a project addition; the paper has none): a
// linear, gauge-covariant network of parallel-transport layers
//   y_c(n) = sum_{d=0..8} sum_{c'} W_d[c][c'] (T_d x_{c'})(n),
// T_0 = 1, T_{2mu} x(n) = U_mu(n) x(n+mu), T_{2mu+1} x(n) = U_mu(n-mu)^dag x(n-mu),
// W_d[c][c'] a 4x4 complex spin matrix.  Because W acts on spin and channel and
// T on colour and site, a layer is, per direction, a dense contraction over
// (input channel, spin) for every (site, colour) row: a GEMM with M = 3V rows,
// K = 9 x Cin x 4 complex, N = Cout x 4 complex.  It runs on the tensor cores
// in BF16 with FP32 accumulation (here mma.sync m16n8k16, the 8 -> 8 layer in
// learned_tc.cu on tcgen05), the weights as real 2x2-block matrices.  A layer
// with one input channel transports that in all directions at once (K = 72);
// the one with one output channel applies the weights first and transports
// the output.  The data gradient is the same with the adjoint weights
// (T_d^dag = T_{opposite d} and W commutes with T); the weight gradient is a
// product with the reduction over the rows.
#include <cuda_bf16.h>

#include <algorithm>
#include <cmath>
#include <cstring>
#include <vector>

#include "fields.cuh"
#include "qcd_internal.h"

namespace qcd {
namespace {

// activation formats
enum { SITE16 = 1, SITE32 = 2 };

template <int FMT> __device__ __forceinline__ void act_st(void *base, long V, int ch, long n, int k, float2 v) {
    if constexpr (FMT == SITE16) {
        static_cast<__nv_bfloat162 *>(base)[((long)ch * V + n) * 12 + k] = __float22bfloat162_rn(v);
    } else {
        static_cast<float2 *>(base)[((long)ch * V + n) * 12 + k] = v;
    }
}

__device__ __forceinline__ uint32_t pack_bf16(float lo, float hi) {
    __nv_bfloat162 h = __floats2bfloat162_rn(lo, hi);
    return *reinterpret_cast<uint32_t *>(&h);
}

__device__ __forceinline__ void mma_bf16(float c[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint32_t b0,
                                         uint32_t b1) {
    asm volatile(
        "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, "
        "{%0,%1,%2,%3};\n"
        : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
        : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}

constexpr int kLayerSites = 64;                 // sites per CTA tile of the layer kernel
constexpr int kLayerRows = 3 * kLayerSites;     // 192 rows = 12 warps x 16 (MMA); threads < 192 gather one row each
constexpr int kLayerWarps = kLayerRows / 16;
static_assert(kLayerWarps * 32 >= kLayerRows, "one gathering thread per row");

__device__ __forceinline__ void cp_async16z(void *smem, const void *gmem, bool valid) {
    const unsigned sa = (unsigned)__cvta_generic_to_shared(smem);
    const int n = valid ? 16 : 0;  // src-size 0: zero fill, nothing read
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;\n" ::"r"(sa), "l"(gmem), "r"(n) : "memory");
}
__device__ __forceinline__ void cp_async8z(void *smem, const void *gmem, bool valid) {
    const unsigned sa = (unsigned)__cvta_generic_to_shared(smem);
    const int n = valid ? 8 : 0;
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8, %2;\n" ::"r"(sa), "l"(gmem), "r"(n) : "memory");
}
__device__ __forceinline__ void cp_commit() { asm volatile("cp.async.commit_group;\n" ::: "memory"); }
template <int N> __device__ __forceinline__ void cp_wait() { asm volatile("cp.async.wait_group %0;\n" ::"n"(N) : "memory"); }

__device__ __forceinline__ void ldsm_x4(const void *p, uint32_t &r0, uint32_t &r1, uint32_t &r2, uint32_t &r3) {
    const unsigned sa = (unsigned)__cvta_generic_to_shared(p);
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];\n"
                 : "=r"(r0), "=r"(r1), "=r"(r2), "=r"(r3)
                 : "r"(sa));
}
__device__ __forceinline__ void ldsm_x2(const void *p, uint32_t &r0, uint32_t &r1) {
    const unsigned sa = (unsigned)__cvta_generic_to_shared(p);
    asm volatile("ldmatrix.sync.aligned.m8n8.x2.shared.b16 {%0,%1}, [%2];\n" : "=r"(r0), "=r"(r1) : "r"(sa));
}

// Shared-memory plan of the layer kernel: two stages (directions d and d+1) of the neighbour
// inputs X[site][ch][12] (site records padded by 16 bytes), the links L[site][9] and the weight
// tile B[N][KDP+8]; the transported A tile [192][KDP+8]; the neighbour table and boundary signs
// of all nine directions.  Row strides of KDP+8 BF16 keep ldmatrix free of bank conflicts.
template <int CIN, int COUT, int FIN> struct LayerSmem {
    static constexpr int KD = CIN * 8, KDP = KD < 16 ? 16 : KD, N = COUT * 8, AS = KDP + 8;
    static constexpr int XC = FIN == SITE16 ? 4 : 8;  // bytes per staged complex input
    static constexpr int XS = CIN * 12 * XC + 16;     // bytes per staged site
    static constexpr size_t x_bytes = (size_t)kLayerSites * XS;
    static constexpr size_t l_bytes = (size_t)kLayerSites * 9 * sizeof(float2);
    static constexpr size_t b_bytes = (size_t)N * AS * sizeof(__nv_bfloat16);
    static constexpr size_t stage = x_bytes + l_bytes + b_bytes;
    static constexpr size_t a_bytes = (size_t)kLayerRows * AS * sizeof(__nv_bfloat16);
    static constexpr size_t total = 2 * stage + a_bytes + (size_t)9 * kLayerSites * (sizeof(int) + sizeof(float));
    static_assert(XS % 16 == 0 && x_bytes % 16 == 0 && l_bytes % 16 == 0 && b_bytes % 16 == 0 && a_bytes % 16 == 0,
                  "16-byte staging");
};

// Neighbour table of a 64-site tile for all nine directions: nbt[d][st] the neighbour site
// (-1 past the end of the lattice), sgt[d][st] the boundary sign of the hop.
__device__ __forceinline__ void layer_neighbours(int *nbt, float *sgt, const Geo &g, int n0, int tid) {
    if (tid >= kLayerSites) return;
    const int V = (int)g.V;
    const int n = n0 + tid;
    int xc0 = 0, xc1 = 0, xc2 = 0, xc3 = 0;
    if (n < V) {
        int r = n;
        xc0 = r % g.L[0]; r /= g.L[0];
        xc1 = r % g.L[1]; r /= g.L[1];
        xc2 = r % g.L[2]; xc3 = r / g.L[2];
    }
    const int xc[4] = {xc0, xc1, xc2, xc3};
    nbt[tid] = n < V ? n : -1;
    sgt[tid] = 1.f;
    int stride = 1;
#pragma unroll
    for (int mu = 0; mu < 4; mu++) {
        const int Lm = g.L[mu];
        const int f = xc[mu] == Lm - 1 ? n - stride * (Lm - 1) : n + stride;
        const int bk = xc[mu] == 0 ? n + stride * (Lm - 1) : n - stride;
        nbt[(1 + 2 * mu) * kLayerSites + tid] = n < V ? f : -1;
        nbt[(2 + 2 * mu) * kLayerSites + tid] = n < V ? bk : -1;
        sgt[(1 + 2 * mu) * kLayerSites + tid] = (mu == 3 && xc[3] == Lm - 1) ? (float)g.bc_t : 1.f;
        sgt[(2 + 2 * mu) * kLayerSites + tid] = (mu == 3 && xc[3] == 0) ? (float)g.bc_t : 1.f;
        stride *= Lm;
    }
}

// Stages direction d of a layer into buffer d & 1 with cp.async (one commit group): the
// neighbour inputs of the tile (all channels), their links (forward U_mu(n), backward
// U_mu(n - mu)) and the direction's weight tile.
template <int CIN, int COUT, int FIN>
__device__ __forceinline__ void layer_issue(unsigned char *smem, const int *nbt, const void *x,
                                            const float2 *__restrict__ U, const __nv_bfloat16 *__restrict__ Bt,
                                            const Geo &g, int n0, int d, int tid, int nth) {
    using S = LayerSmem<CIN, COUT, FIN>;
    constexpr int KDP = S::KDP, N = S::N, AS = S::AS, XS = S::XS;
    const int V = (int)g.V;
    unsigned char *X = smem + (d & 1) * S::stage;
    float2 *L = reinterpret_cast<float2 *>(X + S::x_bytes);
    __nv_bfloat16 *B = reinterpret_cast<__nv_bfloat16 *>(X + S::x_bytes + S::l_bytes);
    const int *nb = nbt + d * kLayerSites;
    // thread -> (site, 16-byte chunk) fixed, channels strided: no index arithmetic in the loop
    constexpr int CH16 = 12 * S::XC / 16;  // 16-byte chunks per site and channel
    constexpr int PAIRS = kLayerSites * CH16;
    static_assert(kLayerWarps * 32 % PAIRS == 0 || PAIRS % (kLayerWarps * 32) == 0, "even split");
    for (int pr = tid; pr < PAIRS; pr += nth) {
        const int st = pr / CH16, k = pr - st * CH16;
        const int m = nb[st];
        const unsigned char *src = static_cast<const unsigned char *>(x) + ((long)(m < 0 ? 0 : m) * 12) * S::XC + k * 16;
        unsigned char *dst = X + st * XS + k * 16;
        const long sstride = (long)V * 12 * S::XC;
#pragma unroll
        for (int ch = 0; ch < CIN; ch++) cp_async16z(dst + ch * CH16 * 16, src + ch * sstride, m >= 0);
    }
    if (d > 0) {
        const int mu = (d - 1) >> 1;
        const bool fwd = ((d - 1) & 1) == 0;
        for (int i = tid; i < kLayerSites * 9; i += nth) {
            const int st = i % kLayerSites, e = i / kLayerSites;
            const int m = nb[st];
            const int ls = fwd ? n0 + st : m;  // U_mu(n) forward, U_mu(n - mu) backward
            cp_async8z(L + st * 9 + e, U + (long)(mu * 9 + e) * V + (m < 0 ? 0 : ls), m >= 0);
        }
    }
    const uint4 *Bd = reinterpret_cast<const uint4 *>(Bt + (long)d * N * KDP);
    for (int i = tid; i < N * KDP / 8; i += nth) {
        const int row = i / (KDP / 8), col = (i % (KDP / 8)) * 8;
        cp_async16z(B + row * AS + col, Bd + i, true);
    }
    cp_commit();
}

// Transport of one (site, channel group) item of the layer kernel: the A rows of the site,
// A[a][8 ch + 2 be (+1)] = sum_b W[a][b] x_ch[be][b] for the CPI channels from cg on.  KIND:
// 0 identity, 1 forward W = U_mu(n), 2 backward W = U_mu(n - mu)^dag, 3 / 4 the same times the
// time-boundary sign.  xs: the staged neighbour site, l: its nine link elements.
template <int CIN, int CPI, int FIN, int KIND>
__device__ __forceinline__ void transport_item(const unsigned char *xs, const float2 *l, float sg, __nv_bfloat16 *arow,
                                               int cg, int as) {
    constexpr bool FWD = KIND == 1 || KIND == 3, SIGN = KIND >= 3;
#pragma unroll
    for (int cc = 0; cc < CPI; cc++) {
        const int ch = cg + cc;
        float2 v[12];
        if constexpr (FIN == SITE16) {
            const uint4 *q = reinterpret_cast<const uint4 *>(xs + ch * 48);
#pragma unroll
            for (int t = 0; t < 3; t++) {
                const uint4 u4 = q[t];
                const uint32_t wds[4] = {u4.x, u4.y, u4.z, u4.w};
#pragma unroll
                for (int e = 0; e < 4; e++)
                    v[t * 4 + e] = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162 *>(&wds[e]));
            }
        } else {
            const float4 *q = reinterpret_cast<const float4 *>(xs + ch * 96);
#pragma unroll
            for (int t = 0; t < 6; t++) {
                const float4 f4 = q[t];
                v[2 * t] = make_float2(f4.x, f4.y);
                v[2 * t + 1] = make_float2(f4.z, f4.w);
            }
        }
#pragma unroll
        for (int a = 0; a < 3; a++) {
            float2 w[3];  // row a of the transport matrix
            if constexpr (KIND > 0) {
#pragma unroll
                for (int b = 0; b < 3; b++) {
                    float2 u = FWD ? l[a * 3 + b] : l[b * 3 + a];
                    if (!FWD) u.y = -u.y;
                    w[b] = SIGN ? cscale(u, sg) : u;
                }
            }
            uint32_t packed[4];
#pragma unroll
            for (int be = 0; be < 4; be++) {
                if constexpr (KIND == 0) {
                    packed[be] = pack_bf16(v[be * 3 + a].x, v[be * 3 + a].y);
                } else {
                    // packed FP32 pairs: p = sum_b Re(w_b) x_b, q = sum_b Im(w_b) x_b; w x = (p.x - q.y, p.y + q.x)
                    float2 pr = __fmul2_rn(make_float2(w[0].x, w[0].x), v[be * 3]);
                    float2 pi = __fmul2_rn(make_float2(w[0].y, w[0].y), v[be * 3]);
#pragma unroll
                    for (int b = 1; b < 3; b++) {
                        pr = __ffma2_rn(make_float2(w[b].x, w[b].x), v[be * 3 + b], pr);
                        pi = __ffma2_rn(make_float2(w[b].y, w[b].y), v[be * 3 + b], pi);
                    }
                    packed[be] = pack_bf16(pr.x - pi.y, pr.y + pi.x);
                }
            }
            *reinterpret_cast<uint4 *>(arow + a * as + ch * 8) = make_uint4(packed[0], packed[1], packed[2], packed[3]);
        }
    }
}

// rows 3 st + a (colour a) of a 12-component site: four spins as BF16 pairs, 16 bytes per row
__device__ __forceinline__ void put_rows(__nv_bfloat16 *row0, int stride, const float2 v[12]) {
#pragma unroll
    for (int a = 0; a < 3; a++)
        *reinterpret_cast<uint4 *>(row0 + a * stride) =
            make_uint4(pack_bf16(v[a].x, v[a].y), pack_bf16(v[3 + a].x, v[3 + a].y), pack_bf16(v[6 + a].x, v[6 + a].y),
                       pack_bf16(v[9 + a].x, v[9 + a].y));
}

// One thread's share of a one-channel field (FP32) of a 64-site tile, transported in every direction:
// thread (st, grp) takes site st and direction grp + 1 (or its opposite, FLIP), and one float4 of the tile's
// own sites for the identity.  The A rows it makes hold the nine directions' four spins side by side,
// 72 columns of a row of kSingleCols BF16 (80 multiplied, the last 8 zero; 88: no ldmatrix bank conflicts).
constexpr int kTileThreads = 512;
constexpr int kSingleCols = 88;
template <bool FLIP> struct SingleField {
    float2 x[12], u[9];
    float4 own;
    float sg;
    int st, mu, d, Lm, stride, V;
    bool fwd;
    __device__ __forceinline__ SingleField(const Geo &g, int tid) {
        const int grp = tid >> 6;
        st = tid & (kLayerSites - 1);
        mu = grp >> 1;
        d = grp + 1;
        fwd = ((grp & 1) == 0) != FLIP;
        Lm = mu == 0 ? g.L[0] : mu == 1 ? g.L[1] : mu == 2 ? g.L[2] : g.L[3];
        stride = mu == 0 ? 1 : mu == 1 ? g.L[0] : mu == 2 ? g.L[0] * g.L[1] : g.L[0] * g.L[1] * g.L[2];
        V = (int)g.V;
    }
    // the loads of a tile; n: the site (0 past the end of the lattice, where `in` is false)
    __device__ __forceinline__ void load(const Geo &g, const float4 *__restrict__ S, const float2 *__restrict__ U, int tile,
                                         int tid, int &n, bool &in) {
        n = tile * kLayerSites + st;
        in = n < V;
        if (!in) n = 0;
        int r = n, xm = 0, xt = 0;
#pragma unroll
        for (int q = 0; q < 4; q++) {
            const int c = q < 3 ? r % g.L[q] : r;
            if (q < 3) r /= g.L[q];
            if (q == mu) xm = c;
            if (q == 3) xt = c;
        }
        const int m = fwd ? (xm == Lm - 1 ? n - stride * (Lm - 1) : n + stride)
                          : (xm == 0 ? n + stride * (Lm - 1) : n - stride);
        sg = !in ? 0.f : (mu == 3 && xt == (fwd ? Lm - 1 : 0)) ? (float)g.bc_t : 1.f;
        load_spinor(S, m, x);
        const int ls = fwd ? n : m;
#pragma unroll
        for (int e = 0; e < 9; e++) u[e] = __ldg(U + (long)(mu * 9 + e) * V + ls);
        const long o = (long)tile * kLayerSites * 6 + tid;
        own = tid < kLayerSites * 6 && o < (long)V * 6 ? __ldg(S + o) : make_float4(0.f, 0.f, 0.f, 0.f);
    }
    __device__ __forceinline__ void put(__nv_bfloat16 *Ss, int tid) const {
        float2 z[12];
#pragma unroll
        for (int a = 0; a < 3; a++) {
            float2 w[3];  // row a of the transport
#pragma unroll
            for (int b = 0; b < 3; b++) {
                w[b] = fwd ? u[a * 3 + b] : make_float2(u[b * 3 + a].x, -u[b * 3 + a].y);
                w[b] = cscale(w[b], sg);
            }
#pragma unroll
            for (int be = 0; be < 4; be++) {
                float2 t = make_float2(0.f, 0.f);
#pragma unroll
                for (int b = 0; b < 3; b++) t = cfma(w[b], x[be * 3 + b], t);
                z[be * 3 + a] = t;
            }
        }
        put_rows(Ss + 3 * st * kSingleCols + d * 8, kSingleCols, z);
        if (tid < kLayerSites * 6) {
            const int os = tid / 6, k0 = 2 * (tid % 6), k1 = k0 + 1;
            *reinterpret_cast<uint32_t *>(Ss + (3 * os + k0 % 3) * kSingleCols + 2 * (k0 / 3)) = pack_bf16(own.x, own.y);
            *reinterpret_cast<uint32_t *>(Ss + (3 * os + k1 % 3) * kSingleCols + 2 * (k1 / 3)) = pack_bf16(own.z, own.w);
        }
    }
    // the zero columns 72 ... 79 of `rows` rows
    static __device__ __forceinline__ void pad(__nv_bfloat16 *Ss, int rows, int tid) {
        for (int i = tid; i < rows; i += kTileThreads)
            *reinterpret_cast<uint4 *>(Ss + i * kSingleCols + 72) = make_uint4(0, 0, 0, 0);
    }
};

// y = layer(x) for one input channel, 1 -> 8.  With one channel to transport, all nine directions'
// A columns of a 64-site tile are made at once, and the layer is one product of 192 rows x 80 by 80 x 64;
// the weights stay in registers as fragments, the next tile's fields are loaded while this one is
// multiplied, and the output leaves through shared memory in whole lines.  Bound by the loads' latency
// at 16 warps per SM.  24^3x48: 0.19 (BF16 out) and 0.23 ms (FP32 out), against 0.57 and 0.60 ms with
// one direction after the other.
template <int FOUT>
__global__ void __launch_bounds__(kTileThreads, 1) k_layer_single(void *y, const float4 *__restrict__ x,
                                                                  const float2 *__restrict__ U,
                                                                  const __nv_bfloat16 *__restrict__ Bt, Geo g, int ntiles,
                                                                  const BicgScalars *__restrict__ gate) {
    if (gate && !gate->active) return;  // a right-hand side that has left the iteration
    extern __shared__ __align__(16) unsigned char l1_smem[];
    __nv_bfloat16 *Sb = reinterpret_cast<__nv_bfloat16 *>(l1_smem);  // two A tiles
    constexpr int OW = FOUT == SITE16 ? 1 : 2;                       // 4-byte words of one complex output
    uint32_t *out = reinterpret_cast<uint32_t *>(l1_smem + 2 * kLayerRows * kSingleCols * sizeof(__nv_bfloat16));
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, gq = lane >> 2, tq = lane & 3;
    SingleField<false> f(g, tid);
    SingleField<false>::pad(Sb, 2 * kLayerRows, tid);
    // warp: three 16-row tiles from mt0 on, two output channels; the weights' fragments
    const int mt0 = 3 * (warp >> 2), c0 = 2 * (warp & 3);
    uint32_t bw[5][2][2];
#pragma unroll
    for (int q = 0; q < 5; q++)
#pragma unroll
        for (int j = 0; j < 2; j++)
#pragma unroll
            for (int h = 0; h < 2; h++) {  // rows k = 16 q + 8 h + 2 tq (+1) = direction 2 q + h, column (c0 + j) 8 + gq
                const int d = 2 * q + h;
                bw[q][j][h] = d < 9 ? *reinterpret_cast<const uint32_t *>(Bt + ((long)d * 64 + (c0 + j) * 8 + gq) * 16 + 2 * tq) : 0u;
            }
    int n;
    bool in;
    if ((int)blockIdx.x < ntiles) f.load(g, x, U, blockIdx.x, tid, n, in);
    int buf = 0;
    for (int tile = blockIdx.x; tile < ntiles; tile += gridDim.x, buf ^= 1) {
        __nv_bfloat16 *Ss = Sb + buf * kLayerRows * kSingleCols;
        f.put(Ss, tid);
        if (tile + (int)gridDim.x < ntiles) f.load(g, x, U, tile + gridDim.x, tid, n, in);
        __syncthreads();  // the A tile is whole; the previous tile's output has left
        float acc[3][2][4];
#pragma unroll
        for (int t = 0; t < 3; t++) {
#pragma unroll
            for (int j = 0; j < 2; j++) acc[t][j][0] = acc[t][j][1] = acc[t][j][2] = acc[t][j][3] = 0.f;
#pragma unroll
            for (int q = 0; q < 5; q++) {
                uint32_t a0, a1, a2, a3;
                ldsm_x4(Ss + ((mt0 + t) * 16 + (lane & 15)) * kSingleCols + q * 16 + (lane >> 4) * 8, a0, a1, a2, a3);
                mma_bf16(acc[t][0], a0, a1, a2, a3, bw[q][0][0], bw[q][0][1]);
                mma_bf16(acc[t][1], a0, a1, a2, a3, bw[q][1][0], bw[q][1][1]);
            }
            // (row, column pair) -> [channel][site][spin 3 + colour], spin tq
#pragma unroll
            for (int j = 0; j < 2; j++)
#pragma unroll
                for (int h = 0; h < 2; h++) {
                    const int r = (mt0 + t) * 16 + gq + 8 * h;
                    uint32_t *o = out + ((c0 + j) * kLayerSites * 12 + (r / 3) * 12 + tq * 3 + r % 3) * OW;
                    if constexpr (FOUT == SITE16) *o = pack_bf16(acc[t][j][2 * h], acc[t][j][2 * h + 1]);
                    else *reinterpret_cast<float2 *>(o) = make_float2(acc[t][j][2 * h], acc[t][j][2 * h + 1]);
                }
        }
        __syncthreads();
        constexpr int W16 = 3 * OW;  // 16-byte words per site and channel
        for (int i = tid; i < 8 * kLayerSites * W16; i += kTileThreads) {
            const int c = i / (kLayerSites * W16), r = i % (kLayerSites * W16);
            const long at = ((long)c * g.V + (long)tile * kLayerSites) * W16 + r;
            if ((long)tile * kLayerSites + r / W16 < g.V)
                static_cast<uint4 *>(y)[at] = reinterpret_cast<const uint4 *>(out)[i];
        }
    }
}

// A layer with one output channel (the last layer), weights first: since W_d acts on spin and
// channel and T_d on colour and site, W_d T_d x = T_d W_d x.  Per direction the staged
// neighbour inputs are only re-laid out as A rows (neighbour site, colour) - no arithmetic -,
// the MMA gives P = W_d x at the neighbours (4 spins), and the 3x3 colour transport is applied
// to P, one output channel instead of CIN input channels.  Output accumulated in registers
// of the thread that owns (site, spin).
template <int CIN, int FIN, int FOUT>
__global__ void __launch_bounds__(kLayerWarps * 32, 2) k_layer_wfirst(void *y, const void *x,
                                                                      const float2 *__restrict__ U,
                                                                      const __nv_bfloat16 *__restrict__ Bt, Geo g,
                                                                      const BicgScalars *__restrict__ gate = nullptr) {
    if (gate && !gate->active) return;  // a right-hand side that has left the iteration
    using S = LayerSmem<CIN, 1, FIN>;
    constexpr int KDP = S::KDP, AS = S::AS, XS = S::XS;
    constexpr int NTH = kLayerWarps * 32;
    static_assert(FIN == SITE16 && CIN * 8 == KDP, "hidden BF16 input of whole 16-column groups");
    extern __shared__ __align__(16) unsigned char ly_smem[];
    __nv_bfloat16 *A = reinterpret_cast<__nv_bfloat16 *>(ly_smem + 2 * S::stage);
    int *nbt = reinterpret_cast<int *>(ly_smem + 2 * S::stage + S::a_bytes);
    float *sgt = reinterpret_cast<float *>(nbt + 9 * kLayerSites);
    float2 *Ps = reinterpret_cast<float2 *>(sgt + 9 * kLayerSites);  // [192 rows][4 spins]
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, gq = lane >> 2, tq = lane & 3;
    const int n0 = blockIdx.x * kLayerSites;
    layer_neighbours(nbt, sgt, g, n0, tid);
    __syncthreads();
    // the output (site, spin) this thread accumulates: 3 colours
    const int ost = tid >> 2, oal = tid & 3;
    float2 yacc[3] = {make_float2(0.f, 0.f), make_float2(0.f, 0.f), make_float2(0.f, 0.f)};
    layer_issue<CIN, 1, FIN>(ly_smem, nbt, x, U, Bt, g, n0, 0, tid, NTH);
#pragma unroll 1
    for (int d = 0; d < 9; d++) {
        cp_wait<0>();
        __syncthreads();  // stage d visible; A and P of the previous direction consumed
        if (d + 1 < 9) layer_issue<CIN, 1, FIN>(ly_smem, nbt, x, U, Bt, g, n0, d + 1, tid, NTH);
        const unsigned char *X = ly_smem + (d & 1) * S::stage;
        const float2 *L = reinterpret_cast<const float2 *>(X + S::x_bytes);
        const __nv_bfloat16 *B = reinterpret_cast<const __nv_bfloat16 *>(X + S::x_bytes + S::l_bytes);
        // A[3 st + b][8 ch + 2 be (+1)] = x_ch(m)[be][b]: a permutation of the staged BF16 words
        for (int it = tid; it < kLayerSites * CIN; it += NTH) {
            const int st = it / CIN, ch = it % CIN;
            const uint4 *q = reinterpret_cast<const uint4 *>(X + st * XS + ch * 48);
            const uint4 q0 = q[0], q1 = q[1], q2 = q[2];
            const uint32_t w[12] = {q0.x, q0.y, q0.z, q0.w, q1.x, q1.y, q1.z, q1.w, q2.x, q2.y, q2.z, q2.w};
#pragma unroll
            for (int b = 0; b < 3; b++)
                *reinterpret_cast<uint4 *>(A + (st * 3 + b) * AS + ch * 8) = make_uint4(w[b], w[3 + b], w[6 + b], w[9 + b]);
        }
        __syncthreads();
        // P = A B: 16 rows per warp, 8 columns (4 spins, re/im)
        float acc[4] = {0.f, 0.f, 0.f, 0.f};
        const int r0 = warp * 16;
#pragma unroll
        for (int k0 = 0; k0 < KDP; k0 += 16) {
            uint32_t a0, a1, a2, a3, b0, b1;
            ldsm_x4(A + (r0 + (lane & 15)) * AS + k0 + (lane >> 4) * 8, a0, a1, a2, a3);
            ldsm_x2(B + (lane & 7) * AS + k0 + ((lane >> 3) & 1) * 8, b0, b1);
            mma_bf16(acc, a0, a1, a2, a3, b0, b1);
        }
        Ps[(r0 + gq) * 4 + tq] = make_float2(acc[0], acc[1]);
        Ps[(r0 + gq + 8) * 4 + tq] = make_float2(acc[2], acc[3]);
        __syncthreads();
        // y(st)[a][al] += sum_b W[a][b] P[(st, b)][al], W = 1, U_mu(n) or U_mu(n - mu)^dag, times the sign
        if (tid < kLayerSites * 4) {
            const float2 p0 = Ps[(ost * 3) * 4 + oal], p1 = Ps[(ost * 3 + 1) * 4 + oal], p2 = Ps[(ost * 3 + 2) * 4 + oal];
            if (d == 0) {
                yacc[0] = cadd(yacc[0], p0);
                yacc[1] = cadd(yacc[1], p1);
                yacc[2] = cadd(yacc[2], p2);
            } else {
                const bool fwd = ((d - 1) & 1) == 0;
                const float sg = sgt[d * kLayerSites + ost];
                const float2 pv[3] = {p0, p1, p2};
#pragma unroll
                for (int a = 0; a < 3; a++) {
                    float2 z = make_float2(0.f, 0.f);
#pragma unroll
                    for (int b = 0; b < 3; b++) {
                        float2 u = fwd ? L[ost * 9 + a * 3 + b] : L[ost * 9 + b * 3 + a];
                        if (!fwd) u.y = -u.y;
                        z = cfma(u, pv[b], z);
                    }
                    yacc[a] = cadd(yacc[a], cscale(z, sg));
                }
            }
        }
    }
    if (tid < kLayerSites * 4) {
        const long n = (long)n0 + ost;
        if (n < g.V)
#pragma unroll
            for (int a = 0; a < 3; a++) act_st<FOUT>(y, g.V, 0, n, oal * 3 + a, yacc[a]);
    }
}

// The weight gradient: P[d][k][j] += sum over rows (site, colour) of A_d[row][k] G[row][j] (real; A_d the
// transported inputs, G the output gradient), of which k_wgrad_finish takes conj(A) G.  Both operands lie
// in shared memory row by row as BF16 and meet in mma.sync with the reduction over the rows, their
// fragments transposed by ldmatrix; a persistent CTA keeps all nine directions' sums in registers
// over its tiles of 64 sites.
__device__ __forceinline__ void ldsm_x4_t(const void *p, uint32_t &r0, uint32_t &r1, uint32_t &r2, uint32_t &r3) {
    const unsigned sa = (unsigned)__cvta_generic_to_shared(p);
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];\n"
                 : "=r"(r0), "=r"(r1), "=r"(r2), "=r"(r3)
                 : "r"(sa)
                 : "memory");
}
__device__ __forceinline__ void ldsm_x2_t(const void *p, uint32_t &r0, uint32_t &r1) {
    const unsigned sa = (unsigned)__cvta_generic_to_shared(p);
    asm volatile("ldmatrix.sync.aligned.m8n8.x2.trans.shared.b16 {%0,%1}, [%2];\n" : "=r"(r0), "=r"(r1) : "r"(sa) : "memory");
}
// The layers with one channel on one side.  Only that side is transported: with T_d^dag = T_e, e the
// opposite direction, sum_n conj(T_d x)(n) G(n) = sum_m conj(x(m)) (T_e G)(m).  S: the one-channel field
// (FP32), transported in all nine directions into 72 columns; H: the eight-channel field, 64 columns, as
// it is.  FLIP = false: S is the layer's input, P[d][16][64]; true: S is the output gradient,
// P[d][64][8], column group d transported by T_e.  The next tile's fields are loaded while this one is
// multiplied.  Bound by those loads' latency at 16 warps per SM.  24^3x48: 0.23 (one input channel) and
// 0.21 ms (one output channel), against 2.5 and 3.2 ms with the operands gathered and transposed anew
// for each direction and, for the latter, all eight inputs transported.
constexpr int kWgHS = 72;  // BF16 per row of H: no ldmatrix bank conflicts
constexpr int kWgTile = kLayerRows * (kSingleCols + kWgHS);
template <bool FLIP, int FH>
__global__ void __launch_bounds__(kTileThreads, 1) k_wgrad_single(float *__restrict__ P, const float4 *__restrict__ S,
                                                                  const void *__restrict__ H,
                                                                  const float2 *__restrict__ U, Geo g, int ntiles) {
    extern __shared__ __align__(16) __nv_bfloat16 ws_smem[];
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, gq = lane >> 2, tq = lane & 3;
    const int st = tid & (kLayerSites - 1), ch = tid >> 6;
    SingleField<FLIP> f(g, tid);
    SingleField<FLIP>::pad(ws_smem, kLayerRows, tid);
    SingleField<FLIP>::pad(ws_smem + kWgTile, kLayerRows, tid);
    float2 hv[12];
    uint4 hw[3];
    auto load = [&](int tile) {
        int n;
        bool in;
        f.load(g, S, U, tile, tid, n, in);
        if constexpr (FH == SITE16) {
            const uint4 *q = reinterpret_cast<const uint4 *>(H) + ((long)ch * g.V + n) * 3;
#pragma unroll
            for (int t = 0; t < 3; t++) hw[t] = in ? __ldg(q + t) : make_uint4(0, 0, 0, 0);
        } else {
            load_spinor(static_cast<const float4 *>(H) + (long)ch * g.V * 6, n, hv);
            if (!in)
#pragma unroll
                for (int k = 0; k < 12; k++) hv[k] = make_float2(0.f, 0.f);
        }
    };
    float acc[5][4];
#pragma unroll
    for (int q = 0; q < 5; q++) acc[q][0] = acc[q][1] = acc[q][2] = acc[q][3] = 0.f;
    if ((int)blockIdx.x < ntiles) load(blockIdx.x);
    int buf = 0;
    for (int tile = blockIdx.x; tile < ntiles; tile += gridDim.x, buf ^= 1) {
        __nv_bfloat16 *Ss = ws_smem + buf * kWgTile, *Hs = Ss + kLayerRows * kSingleCols;
        f.put(Ss, tid);
        if constexpr (FH == SITE16) {
            const uint32_t w[12] = {hw[0].x, hw[0].y, hw[0].z, hw[0].w, hw[1].x, hw[1].y,
                                    hw[1].z, hw[1].w, hw[2].x, hw[2].y, hw[2].z, hw[2].w};
#pragma unroll
            for (int a = 0; a < 3; a++)
                *reinterpret_cast<uint4 *>(Hs + (3 * st + a) * kWgHS + ch * 8) = make_uint4(w[a], w[3 + a], w[6 + a], w[9 + a]);
        } else {
            put_rows(Hs + 3 * st * kWgHS + ch * 8, kWgHS, hv);
        }
        if (tile + (int)gridDim.x < ntiles) load(tile + gridDim.x);
        __syncthreads();  // this buffer is whole; the other one's products are done
        // warp: eight H columns, half of the rows
        const int n0 = (warp & 7) * 8, rb = (warp >> 3) * (kLayerRows / 2);
#pragma unroll
        for (int r0 = rb; r0 < rb + kLayerRows / 2; r0 += 16) {
            uint32_t b0, b1;
            ldsm_x2_t(Hs + (r0 + (lane & 15)) * kWgHS + n0, b0, b1);
#pragma unroll
            for (int q = 0; q < 5; q++) {
                uint32_t a0, a1, a2, a3;
                ldsm_x4_t(Ss + (r0 + (lane & 7) + (lane >> 4) * 8) * kSingleCols + q * 16 + ((lane >> 3) & 1) * 8, a0, a1, a2, a3);
                mma_bf16(acc[q], a0, a1, a2, a3, b0, b1);
            }
        }
    }
#pragma unroll
    for (int q = 0; q < 5; q++)
#pragma unroll
        for (int e = 0; e < 4; e++) {
            const int row = q * 16 + gq + 8 * (e >> 1), h = (warp & 7) * 8 + 2 * tq + (e & 1);
            if (row < 72)
                atomicAdd(FLIP ? &P[(row >> 3) * 512 + h * 8 + (row & 7)] : &P[(row >> 3) * 1024 + (row & 7) * 64 + h], acc[q][e]);
        }
}

// The 8 -> 8 layer: per direction the neighbour inputs and links of a tile are staged with cp.async one
// direction ahead, one thread per (site, channel) transports them into the A rows, and each warp
// multiplies a 16 x 16 piece of P_d.  G is staged once for all nine directions.  24^3x48: 1.5 ms, against
// 4.2 ms with G gathered and both operands transposed in shared memory for every direction.
struct Wg88 {
    static constexpr int XS = 8 * 48 + 16, AS = 72;  // bytes per staged site, BF16 per A or G row
    static constexpr size_t x_bytes = (size_t)kLayerSites * XS, l_bytes = (size_t)kLayerSites * 9 * sizeof(float2);
    static constexpr size_t stage = x_bytes + l_bytes, a_bytes = (size_t)kLayerRows * AS * sizeof(__nv_bfloat16);
    static constexpr size_t total = 2 * stage + 2 * a_bytes + (size_t)9 * kLayerSites * (sizeof(int) + sizeof(float));
};
__global__ void __launch_bounds__(kTileThreads, 1) k_wgrad88(float *__restrict__ P, const void *__restrict__ x,
                                                           const float4 *__restrict__ G, const float2 *__restrict__ U,
                                                           Geo g, int ntiles) {
    extern __shared__ __align__(16) unsigned char wg_smem[];
    __nv_bfloat16 *A = reinterpret_cast<__nv_bfloat16 *>(wg_smem + 2 * Wg88::stage), *Gs = A + kLayerRows * Wg88::AS;
    int *nbt = reinterpret_cast<int *>(wg_smem + 2 * Wg88::stage + 2 * Wg88::a_bytes);
    float *sgt = reinterpret_cast<float *>(nbt + 9 * kLayerSites);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, gq = lane >> 2, tq = lane & 3;
    const int V = (int)g.V, st = tid >> 3, ch = tid & 7;
    const int m0 = (warp & 3) * 16, j0 = (warp >> 2) * 16;
    float acc[9][2][4];
#pragma unroll
    for (int d = 0; d < 9; d++)
#pragma unroll
        for (int q = 0; q < 2; q++) acc[d][q][0] = acc[d][q][1] = acc[d][q][2] = acc[d][q][3] = 0.f;
    for (int tile = blockIdx.x; tile < ntiles; tile += gridDim.x) {
        const int n0 = tile * kLayerSites;
        auto issue = [&](int d) {
            unsigned char *X = wg_smem + (d & 1) * Wg88::stage;
            float2 *L = reinterpret_cast<float2 *>(X + Wg88::x_bytes);
            const int *nb = nbt + d * kLayerSites;
#pragma unroll
            for (int q = 0; q < 3; q++) {  // 64 sites x 8 channels x 3 words of 16 bytes, sites fastest
                const int i = tid + q * kTileThreads, c = i / (3 * kLayerSites), r = i % (3 * kLayerSites), s = r / 3, k = r % 3;
                const int m = nb[s];
                cp_async16z(X + s * Wg88::XS + c * 48 + k * 16,
                            static_cast<const unsigned char *>(x) + ((long)c * V + (m < 0 ? 0 : m)) * 48 + k * 16, m >= 0);
            }
            if (d > 0) {
                const int mu = (d - 1) >> 1;
                const bool fwd = ((d - 1) & 1) == 0;
                for (int i = tid; i < kLayerSites * 9; i += kTileThreads) {
                    const int s = i % kLayerSites, e = i / kLayerSites;
                    const int m = nb[s], ls = fwd ? n0 + s : m;
                    cp_async8z(L + s * 9 + e, U + (long)(mu * 9 + e) * V + (m < 0 ? 0 : ls), m >= 0);
                }
            }
            cp_commit();
        };
        __syncthreads();  // the previous tile's tables and operands are done with
        layer_neighbours(nbt, sgt, g, n0, tid);
        float2 gv[12];
        {
            const int n = n0 + st;
            load_spinor(G + (long)ch * V * 6, n < V ? n : 0, gv);
            if (n >= V)
#pragma unroll
                for (int k = 0; k < 12; k++) gv[k] = make_float2(0.f, 0.f);
        }
        __syncthreads();
        issue(0);
        put_rows(Gs + 3 * st * Wg88::AS + ch * 8, Wg88::AS, gv);
#pragma unroll
        for (int d = 0; d < 9; d++) {
            cp_wait<0>();
            __syncthreads();  // stage d visible; the products of direction d - 1 are done
            if (d + 1 < 9) issue(d + 1);
            const unsigned char *X = wg_smem + (d & 1) * Wg88::stage;
            const float2 *L = reinterpret_cast<const float2 *>(X + Wg88::x_bytes);
            constexpr int kind[9] = {0, 1, 2, 1, 2, 1, 2, 3, 4};
            const float sg = sgt[d * kLayerSites + st];
            __nv_bfloat16 *row = A + 3 * st * Wg88::AS;
            if (kind[d] == 0) transport_item<8, 1, SITE16, 0>(X + st * Wg88::XS, L + st * 9, sg, row, ch, Wg88::AS);
            else if (kind[d] == 1) transport_item<8, 1, SITE16, 1>(X + st * Wg88::XS, L + st * 9, sg, row, ch, Wg88::AS);
            else if (kind[d] == 2) transport_item<8, 1, SITE16, 2>(X + st * Wg88::XS, L + st * 9, sg, row, ch, Wg88::AS);
            else if (kind[d] == 3) transport_item<8, 1, SITE16, 3>(X + st * Wg88::XS, L + st * 9, sg, row, ch, Wg88::AS);
            else transport_item<8, 1, SITE16, 4>(X + st * Wg88::XS, L + st * 9, sg, row, ch, Wg88::AS);
            __syncthreads();
#pragma unroll 4
            for (int r0 = 0; r0 < kLayerRows; r0 += 16) {
                uint32_t a0, a1, a2, a3, b0, b1, b2, b3;
                ldsm_x4_t(A + (r0 + (lane & 7) + (lane >> 4) * 8) * Wg88::AS + m0 + ((lane >> 3) & 1) * 8, a0, a1, a2, a3);
                ldsm_x4_t(Gs + (r0 + (lane & 15)) * Wg88::AS + j0 + (lane >> 4) * 8, b0, b1, b2, b3);
                mma_bf16(acc[d][0], a0, a1, a2, a3, b0, b1);
                mma_bf16(acc[d][1], a0, a1, a2, a3, b2, b3);
            }
        }
    }
#pragma unroll
    for (int d = 0; d < 9; d++)
#pragma unroll
        for (int q = 0; q < 2; q++)
#pragma unroll
            for (int e = 0; e < 4; e++)
                atomicAdd(&P[d * 4096 + (m0 + gq + 8 * (e >> 1)) * 64 + j0 + q * 8 + 2 * tq + (e & 1)], acc[d][q][e]);
}

// B matrices (BF16, [9][N][KDP]) of a layer from its complex weights W [9][cout][cin][4][4];
// adjoint: the layer x -> sum_d W_d^dag T_{opposite d} x (cin and cout swap roles)
__global__ void k_build_B(__nv_bfloat16 *__restrict__ Bt, const float2 *__restrict__ W, int cin, int cout,
                          int adjoint) {
    const int ci = adjoint ? cout : cin, co = adjoint ? cin : cout;  // channels of the layer being built
    const int KD = ci * 8, KDP = KD < 16 ? 16 : KD, N = co * 8;
    const long total = 9L * N * KDP;
    const long i = blockIdx.x * (long)blockDim.x + threadIdx.x;
    if (i >= total) return;
    const int e = (int)(i / ((long)N * KDP));
    const int j = (int)((i / KDP) % N), k = (int)(i % KDP);
    float v = 0.f;
    if (k < KD) {
        const int p = k & 1, be = (k >> 1) & 3, cp = k >> 3;   // input channel, spin, re/im
        const int q = j & 1, al = (j >> 1) & 3, c = j >> 3;     // output channel, spin, re/im
        float2 w;
        if (!adjoint) {
            w = W[(((long)e * cout + c) * cin + cp) * 16 + al * 4 + be];
        } else {
            const int d = e == 0 ? 0 : ((e - 1) ^ 1) + 1;  // W'_e = W_d^dag with d the opposite of e
            const float2 o = W[(((long)d * cout + cp) * cin + c) * 16 + be * 4 + al];
            w = make_float2(o.x, -o.y);
        }
        // complex out = w in as a real 2x2 block [[wr, -wi], [wi, wr]] (rows: out re/im, cols: in re/im)
        v = (p == 0) ? (q == 0 ? w.x : w.y) : (q == 0 ? -w.y : w.x);
    }
    Bt[i] = __float2bfloat16(v);
}

// dW (complex) from P: (P[re][re] + P[im][im]) + i (P[re][im] - P[im][re]); grad += 2 (Re, Im)
__global__ void k_wgrad_finish(float2 *__restrict__ grad, const float *__restrict__ P, int cin, int cout) {
    const int KD = cin * 8, KDP = KD < 16 ? 16 : KD, N = cout * 8;
    const long total = 9L * cout * cin * 16;
    const long i = blockIdx.x * (long)blockDim.x + threadIdx.x;
    if (i >= total) return;
    const int be = i % 4, al = (i / 4) % 4, cp = (int)((i / 16) % cin), c = (int)((i / 16 / cin) % cout);
    const int d = (int)(i / 16 / cin / cout);
    const float *Pd = P + (long)d * KDP * N;
    const int kr = (cp * 4 + be) * 2, jr = (c * 4 + al) * 2;
    const float rr = Pd[kr * N + jr], ii = Pd[(kr + 1) * N + jr + 1];
    const float ri = Pd[kr * N + jr + 1], ir = Pd[(kr + 1) * N + jr];
    grad[i].x += 2.f * (rr + ii);
    grad[i].y += 2.f * (ri - ir);
}

// r = a - b (FP32, 6 float4 per site); r may be b (each element is read and
// written by one thread)
__global__ void k_sub_spinors(float4 *r, const float4 *a, const float4 *b, long n,
                            const BicgScalars *__restrict__ gate = nullptr) {
    const long i = blockIdx.x * (long)blockDim.x + threadIdx.x;
    if (i >= n || (gate && !gate->active)) return;
    const float4 x = a[i], y = b[i];
    r[i] = make_float4(x.x - y.x, x.y - y.y, x.z - y.z, x.w - y.w);
}
// x += y (FP32)
__global__ void k_add_spinors(float4 *__restrict__ x, const float4 *__restrict__ y, long n,
                            const BicgScalars *__restrict__ gate = nullptr) {
    const long i = blockIdx.x * (long)blockDim.x + threadIdx.x;
    if (i >= n || (gate && !gate->active)) return;
    const float4 a = x[i], b = y[i];
    x[i] = make_float4(a.x + b.x, a.y + b.y, a.z + b.z, a.w + b.w);
}

// loss += |y - eps|^2 / en2 over one pair; g = (y - eps) / en2 (FP32)
__global__ void k_loss(float2 *__restrict__ g, double *__restrict__ loss, const float2 *__restrict__ y,
                       const float2 *__restrict__ eps, const double *__restrict__ en2, long V) {
    __shared__ double sh[256];
    const long n = blockIdx.x * (long)blockDim.x + threadIdx.x;
    double acc = 0;
    if (n < V) {
        const float inv = (float)(1.0 / *en2);
#pragma unroll
        for (int k = 0; k < 12; k++) {
            const float2 yk = y[n * 12 + k];
            const float2 e = eps[n * 12 + k];
            const float2 r = make_float2(yk.x - e.x, yk.y - e.y);
            acc += ((double)r.x * r.x + (double)r.y * r.y) * inv;
            g[n * 12 + k] = make_float2(r.x * inv, r.y * inv);
        }
    }
    sh[threadIdx.x] = acc;
    __syncthreads();
    for (int s = 128; s > 0; s >>= 1) {
        if (threadIdx.x < s) sh[threadIdx.x] += sh[threadIdx.x + s];
        __syncthreads();
    }
    if (threadIdx.x == 0) atomicAdd(loss, sh[0]);
}

// |eps|^2 of one pair 
__global__ void k_norm2(double *__restrict__ out, const float2 *__restrict__ e, long n) {
    __shared__ double sh[256];
    double acc = 0;
    for (long i = blockIdx.x * (long)blockDim.x + threadIdx.x; i < n; i += (long)gridDim.x * blockDim.x)
        acc += (double)e[i].x * e[i].x + (double)e[i].y * e[i].y;
    sh[threadIdx.x] = acc;
    __syncthreads();
    for (int s = 128; s > 0; s >>= 1) {
        if (threadIdx.x < s) sh[threadIdx.x] += sh[threadIdx.x + s];
        __syncthreads();
    }
    if (threadIdx.x == 0) atomicAdd(out, sh[0]);
}

// Adam on real parameters: w -= lr mhat / (sqrt(vhat) + eps)
__global__ void k_adam(float *__restrict__ w, const float *__restrict__ g, float *__restrict__ m, float *__restrict__ v,
                       long n, float lr, float b1, float b2, float eps, float c1, float c2) {
    const long i = blockIdx.x * (long)blockDim.x + threadIdx.x;
    if (i >= n) return;
    const float gi = g[i];
    m[i] = b1 * m[i] + (1.f - b1) * gi;
    v[i] = b2 * v[i] + (1.f - b2) * gi * gi;
    w[i] -= lr * (m[i] / c1) / (sqrtf(v[i] / c2) + eps);
}

Geo geo(const qcd_ctx *c) {
    Geo g;
    for (int m = 0; m < 4; m++) g.L[m] = c->lat.L[m];
    g.V = c->lat.V;
    g.bc_t = c->bc_t;
    return g;
}

// CTAs of a persistent kernel: one per SM (fewer tiles: one each)
int tile_grid(const qcd_ctx *c, int tiles) {
    int sms = 0;
    if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, c->device) != cudaSuccess) {
        cudaGetLastError();
        sms = 1;
    }
    return std::min(tiles, std::max(1, sms));
}
template <int FOUT>
int launch_layer_single(qcd_ctx *c, void *y, const float4 *x, const __nv_bfloat16 *Bt, const BicgScalars *gate = nullptr) {
    constexpr size_t smem = 2 * kLayerRows * kSingleCols * sizeof(__nv_bfloat16) + 8 * kLayerSites * (FOUT == SITE16 ? 48 : 96);
    static std::atomic<unsigned long long> attr{0};
    static std::mutex attr_mu;
    if (int arc = once_per_device(attr, attr_mu, c->device, [&]() -> int {
            QCD_CUDA(c, cudaFuncSetAttribute(k_layer_single<FOUT>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
            return QCD_OK;
        }))
        return arc;
    const int tiles = (int)((c->lat.V + kLayerSites - 1) / kLayerSites);
    cudaEvent_t ev;
    prof_begin(c, QCD_K_LEARNED, &ev);
    k_layer_single<FOUT><<<tile_grid(c, tiles), kTileThreads, smem, c->stream>>>(y, x, c->U32, Bt, geo(c), tiles, gate);
    return prof_end(c, QCD_K_LEARNED, ev);
}

template <int CIN, int FIN, int FOUT>
int launch_layer_wfirst(qcd_ctx *c, void *y, const void *x, const __nv_bfloat16 *Bt,
                        const BicgScalars *gate = nullptr) {
    constexpr size_t smem = LayerSmem<CIN, 1, FIN>::total + sizeof(float2) * kLayerRows * 4;
    static std::atomic<unsigned long long> attr{0};
    static std::mutex attr_mu;
    if (int arc = once_per_device(attr, attr_mu, c->device, [&]() -> int {
            QCD_CUDA(c, cudaFuncSetAttribute(k_layer_wfirst<CIN, FIN, FOUT>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                             (int)smem));
            return QCD_OK;
        }))
        return arc;
    const long tiles = (c->lat.V + kLayerSites - 1) / kLayerSites;
    cudaEvent_t ev;
    prof_begin(c, QCD_K_LEARNED, &ev);
    k_layer_wfirst<CIN, FIN, FOUT><<<(unsigned)tiles, kLayerWarps * 32, smem, c->stream>>>(y, x, c->U32, Bt, geo(c),
                                                                                        gate);
    return prof_end(c, QCD_K_LEARNED, ev);
}

// P zeroed by the caller
template <bool FLIP, int FH> int launch_wgrad_single(qcd_ctx *c, float *P, const float4 *S, const void *H) {
    constexpr size_t smem = 2 * kWgTile * sizeof(__nv_bfloat16);
    static std::atomic<unsigned long long> attr{0};
    static std::mutex attr_mu;
    if (int arc = once_per_device(attr, attr_mu, c->device, [&]() -> int {
            QCD_CUDA(c, cudaFuncSetAttribute(k_wgrad_single<FLIP, FH>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
            return QCD_OK;
        }))
        return arc;
    const int tiles = (int)((c->lat.V + kLayerSites - 1) / kLayerSites);
    cudaEvent_t ev;
    prof_begin(c, QCD_K_LEARNED, &ev);
    k_wgrad_single<FLIP, FH><<<tile_grid(c, tiles), kTileThreads, smem, c->stream>>>(P, S, H, c->U32, geo(c), tiles);
    return prof_end(c, QCD_K_LEARNED, ev);
}
int launch_wgrad88(qcd_ctx *c, float *P, const void *x, const float4 *G) {
    static std::atomic<unsigned long long> attr{0};
    static std::mutex attr_mu;
    if (int arc = once_per_device(attr, attr_mu, c->device, [&]() -> int {
            QCD_CUDA(c, cudaFuncSetAttribute(k_wgrad88, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)Wg88::total));
            return QCD_OK;
        }))
        return arc;
    const int tiles = (int)((c->lat.V + kLayerSites - 1) / kLayerSites);
    cudaEvent_t ev;
    prof_begin(c, QCD_K_LEARNED, &ev);
    k_wgrad88<<<tile_grid(c, tiles), kTileThreads, Wg88::total, c->stream>>>(P, x, G, c->U32, geo(c), tiles);
    return prof_end(c, QCD_K_LEARNED, ev);
}

}  // namespace

// ---- network state -----------------------------------------------------------------------

long learned_weight_count() {
    long n = 0;
    for (int l = 0; l < kLearnedLayers; l++) n += 9L * kLearnedChans[l + 1] * kLearnedChans[l] * 16;
    return n;
}

static long layer_woff(int l) {
    long n = 0;
    for (int k = 0; k < l; k++) n += 9L * kLearnedChans[k + 1] * kLearnedChans[k] * 16;
    return n;
}
static long layer_boff(int l, bool adjoint) {
    // B matrices of layers 0..l-1 (forward and adjoint interleaved)
    long n = 0;
    for (int k = 0; k <= l; k++)
        for (int a = 0; a < 2; a++) {
            if (k == l && a == (adjoint ? 1 : 0)) return n;
            const int ci = a ? kLearnedChans[k + 1] : kLearnedChans[k], co = a ? kLearnedChans[k] : kLearnedChans[k + 1];
            const int KD = ci * 8, KDP = KD < 16 ? 16 : KD;
            n += 9L * co * 8 * KDP;
        }
    return n;
}

static int ensure_net(qcd_ctx *c) {
    Learned &L = c->net;
    const long V = c->lat.V;
    if (!L.W) {
        const long nw = learned_weight_count();
        int rc;
        if ((rc = dev_alloc(c, (void **)&L.W, sizeof(float2) * nw))) return rc;
        if ((rc = dev_alloc(c, (void **)&L.grad, sizeof(float2) * nw))) return rc;
        if ((rc = dev_alloc(c, (void **)&L.m, sizeof(float2) * nw))) return rc;
        if ((rc = dev_alloc(c, (void **)&L.v, sizeof(float2) * nw))) return rc;
        if ((rc = dev_alloc(c, (void **)&L.B, sizeof(__nv_bfloat16) * layer_boff(kLearnedLayers, false)))) return rc;
        if ((rc = dev_alloc(c, (void **)&L.P, sizeof(float) * 9 * 64 * 64))) return rc;
        if ((rc = dev_alloc(c, (void **)&L.scal, sizeof(double) * 4))) return rc;
    }
    if (L.V != V) {
        dev_free(c, L.act);
        L.act = nullptr;
        // hidden activations (BF16, 8 channels each), gradients (FP32, 8 channels each), two site spinors
        const size_t bytes = 2 * (sizeof(__nv_bfloat162) * 12 * 8 * V) + 2 * (sizeof(float2) * 12 * 8 * V) +
                             2 * (sizeof(float2) * 12 * V);
        int rc;
        if ((rc = dev_alloc(c, &L.act, bytes))) return rc;
        L.V = V;
        char *p = (char *)L.act;
        L.a1 = p; p += sizeof(__nv_bfloat162) * 12 * 8 * V;
        L.a2 = p; p += sizeof(__nv_bfloat162) * 12 * 8 * V;
        L.g1 = (float2 *)p; p += sizeof(float2) * 12 * 8 * V;
        L.g2 = (float2 *)p; p += sizeof(float2) * 12 * 8 * V;
        L.g3 = (float2 *)p; p += sizeof(float2) * 12 * V;
        L.tmp = (float2 *)p;
    }
    return QCD_OK;
}

// rebuild the BF16 B matrices from the FP32 weights
int learned_sync_B(qcd_ctx *c) {
    Learned &L = c->net;
    for (int l = 0; l < kLearnedLayers; l++)
        for (int a = 0; a < 2; a++) {
            const int ci = a ? kLearnedChans[l + 1] : kLearnedChans[l], co = a ? kLearnedChans[l] : kLearnedChans[l + 1];
            const int KD = ci * 8, KDP = KD < 16 ? 16 : KD;
            const long total = 9L * co * 8 * KDP;
            cudaEvent_t ev;
            prof_begin(c, QCD_K_LEARNED, &ev);
            k_build_B<<<(unsigned)((total + 255) / 256), 256, 0, c->stream>>>(
                L.B + layer_boff(l, a), L.W + layer_woff(l), kLearnedChans[l], kLearnedChans[l + 1], a);
            int rc = prof_end(c, QCD_K_LEARNED, ev);
            if (rc) return rc;
        }
    return QCD_OK;
}

int learned_set_weights(qcd_ctx *c, const float2 *w_host_or_dev, bool on_device) {
    int rc = ensure_net(c);
    if (rc) return rc;
    const size_t bytes = sizeof(float2) * learned_weight_count();
    QCD_CUDA(c, cudaMemcpyAsync(c->net.W, w_host_or_dev, bytes, on_device ? cudaMemcpyDeviceToDevice
                                                                         : cudaMemcpyHostToDevice, c->stream));
    QCD_CUDA(c, cudaMemsetAsync(c->net.m, 0, bytes, c->stream));
    QCD_CUDA(c, cudaMemsetAsync(c->net.v, 0, bytes, c->stream));
    c->net.step = 0;
    c->net.ready = true;
    return learned_sync_B(c);
}

int learned_get_weights(qcd_ctx *c, float2 *w_host) {
    if (!c->net.ready) return fail(c, QCD_ERR_STATE, "no learned weights set");
    QCD_CUDA(c, cudaMemcpyAsync(w_host, c->net.W, sizeof(float2) * learned_weight_count(), cudaMemcpyDeviceToHost,
                                c->stream));
    QCD_CUDA(c, cudaStreamSynchronize(c->stream));
    return QCD_OK;
}

// y = N(x) for one right-hand side in FP32 (layers 1 -> 8 -> 8 -> 1); with
// gate, every kernel returns at once while that right-hand side is inactive
int learned_forward(qcd_ctx *c, float4 *y, const float4 *x, const BicgScalars *gate) {
    Learned &L = c->net;
    if (!L.ready) return fail(c, QCD_ERR_STATE, "no learned weights set");
    int rc = ensure_net(c);
    if (rc) return rc;
    if ((rc = launch_layer_single<SITE16>(c, L.a1, x, L.B + layer_boff(0, false), gate))) return rc;
    if ((rc = learned_layer_tc(c, L.a2, L.a1, L.B + layer_boff(1, false), false, gate))) return rc;
    return launch_layer_wfirst<8, SITE16, SITE32>(c, y, L.a2, L.B + layer_boff(2, false), gate);
}

// loss of one pair (FP32) and, with accumulate,
// its gradient added to the running sum in L.grad (real pairs, 2 (Re, Im) of dL/dW*)
int learned_loss_grad(qcd_ctx *c, const float4 *rho, const float2 *eps, double *loss_out, float4 *ybuf) {
    Learned &L = c->net;
    int rc = learned_forward(c, ybuf, rho);
    if (rc) return rc;
    const long V = c->lat.V;
    QCD_CUDA(c, cudaMemsetAsync(L.scal, 0, sizeof(double) * 2, c->stream));
    cudaEvent_t ev;
    prof_begin(c, QCD_K_LEARNED, &ev);
    k_norm2<<<256, 256, 0, c->stream>>>(L.scal + 1, eps, 12 * V);
    if ((rc = prof_end(c, QCD_K_LEARNED, ev))) return rc;
    prof_begin(c, QCD_K_LEARNED, &ev);
    k_loss<<<(unsigned)((V + 255) / 256), 256, 0, c->stream>>>(L.g3, L.scal, (const float2 *)ybuf, eps, L.scal + 1, V);
    if ((rc = prof_end(c, QCD_K_LEARNED, ev))) return rc;
    // backward: layer 3 (8 -> 1), layer 2 (8 -> 8), layer 1 (1 -> 8)
    auto wgrad_layer = [&](int l, auto launcher) -> int {
        QCD_CUDA(c, cudaMemsetAsync(L.P, 0, sizeof(float) * 9 * 64 * 64, c->stream));
        int r = launcher();
        if (r) return r;
        const long cnt = 9L * kLearnedChans[l + 1] * kLearnedChans[l] * 16;
        cudaEvent_t e2;
        prof_begin(c, QCD_K_LEARNED, &e2);
        k_wgrad_finish<<<(unsigned)((cnt + 255) / 256), 256, 0, c->stream>>>(L.grad + layer_woff(l), L.P,
                                                                            kLearnedChans[l], kLearnedChans[l + 1]);
        return prof_end(c, QCD_K_LEARNED, e2);
    };
    if ((rc = wgrad_layer(2, [&]() { return launch_wgrad_single<true, SITE16>(c, L.P, (const float4 *)L.g3, L.a2); }))) return rc;
    if ((rc = launch_layer_single<SITE32>(c, L.g2, (const float4 *)L.g3, L.B + layer_boff(2, true)))) return rc;
    if ((rc = wgrad_layer(1, [&]() { return launch_wgrad88(c, L.P, L.a1, (const float4 *)L.g2); }))) return rc;
    if ((rc = learned_layer_tc(c, L.g1, L.g2, L.B + layer_boff(1, true), true))) return rc;
    if ((rc = wgrad_layer(0, [&]() { return launch_wgrad_single<false, SITE32>(c, L.P, rho, L.g1); }))) return rc;
    if (loss_out) {
        double h = 0;
        QCD_CUDA(c, cudaMemcpyAsync(&h, L.scal, sizeof(double), cudaMemcpyDeviceToHost, c->stream));
        QCD_CUDA(c, cudaStreamSynchronize(c->stream));
        *loss_out = h;
    }
    return QCD_OK;
}

int learned_adam(qcd_ctx *c, float lr) {
    Learned &L = c->net;
    const long n = 2 * learned_weight_count();
    L.step++;
    const float b1 = 0.9f, b2 = 0.999f;
    const float c1 = 1.f - powf(b1, (float)L.step), c2 = 1.f - powf(b2, (float)L.step);
    cudaEvent_t ev;
    prof_begin(c, QCD_K_LEARNED, &ev);
    k_adam<<<(unsigned)((n + 255) / 256), 256, 0, c->stream>>>((float *)L.W, (const float *)L.grad, (float *)L.m,
                                                                (float *)L.v, n, lr, b1, b2, 1e-8f, c1, c2);
    int rc = prof_end(c, QCD_K_LEARNED, ev);
    if (rc) return rc;
    return learned_sync_B(c);
}

int learned_zero_grad(qcd_ctx *c) {
    QCD_CUDA(c, cudaMemsetAsync(c->net.grad, 0, sizeof(float2) * learned_weight_count(), c->stream));
    return QCD_OK;
}

// out = out + N(v - D out) for nrhs right-hand sides: the learned correction
// applied after SAP; w1, w2: two scratch spinors of nrhs fields each
int learned_correct(qcd_ctx *c, float4 *out, const float4 *v, float4 *w1, float4 *w2, int nrhs,
                    const BicgScalars *gate) {
    const long n4 = 6 * c->lat.V;
    int rc;
    if ((rc = dslash32_dot(c, w1, out, nrhs, nullptr, 0, nullptr, gate, ScalarStep()))) return rc;
    for (int k = 0; k < nrhs; k++) {
        const BicgScalars *gk = gate ? gate + k : nullptr;
        cudaEvent_t ev;
        prof_begin(c, QCD_K_LEARNED, &ev);
        k_sub_spinors<<<(unsigned)((n4 + 255) / 256), 256, 0, c->stream>>>(w1 + k * n4, v + k * n4, w1 + k * n4, n4,
                                                                         gk);
        if ((rc = prof_end(c, QCD_K_LEARNED, ev))) return rc;
        if ((rc = learned_forward(c, w2, w1 + k * n4, gk))) return rc;
        prof_begin(c, QCD_K_LEARNED, &ev);
        k_add_spinors<<<(unsigned)((n4 + 255) / 256), 256, 0, c->stream>>>(out + k * n4, w2, n4, gk);
        if ((rc = prof_end(c, QCD_K_LEARNED, ev))) return rc;
    }
    return QCD_OK;
}

int sub_spinors(qcd_ctx *c, float4 *r, const float4 *a, const float4 *b, int nrhs) {
    const long n4 = 6 * c->lat.V * nrhs;
    cudaEvent_t ev;
    prof_begin(c, QCD_K_LEARNED, &ev);
    k_sub_spinors<<<(unsigned)((n4 + 255) / 256), 256, 0, c->stream>>>(r, a, b, n4);
    return prof_end(c, QCD_K_LEARNED, ev);
}

}  // namespace qcd
