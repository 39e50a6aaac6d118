// K6: the links from the caller's layout to the internal plane-major one (see qcd_internal.h), and
// FP64 <-> FP32 conversion of spinors (the single/double precision conversion at load and store of
// the nested solver, Sec. 3 "SIMDzation").  Spinors keep the caller's layout throughout.
#include <algorithm>

#include "fields.cuh"
#include "qcd_internal.h"

namespace qcd {

namespace {

constexpr int TPB = 256;

// FP64 <-> FP32, two complex numbers per thread
__global__ void k_s64_to_32(float4 *__restrict__ dst, const double2 *__restrict__ src, long n2) {
    for (long i = blockIdx.x * (long)TPB + threadIdx.x; i < n2; i += (long)gridDim.x * TPB) {
        const double2 a = src[2 * i], b = src[2 * i + 1];
        dst[i] = make_float4((float)a.x, (float)a.y, (float)b.x, (float)b.y);
    }
}
__global__ void k_s32_to_64(double2 *__restrict__ dst, const float4 *__restrict__ src, long n2) {
    for (long i = blockIdx.x * (long)TPB + threadIdx.x; i < n2; i += (long)gridDim.x * TPB) {
        const float4 v = src[i];
        dst[2 * i] = make_double2(v.x, v.y);
        dst[2 * i + 1] = make_double2(v.z, v.w);
    }
}
__global__ void k_copy(float4 *__restrict__ dst, const float4 *__restrict__ src, long n) {
    chain_wait(src);
    for (long i = blockIdx.x * (long)TPB + threadIdx.x; i < n; i += (long)gridDim.x * TPB) dst[i] = src[i];
}
// canonical links complex128 [V][4][3][3] -> [4][9][V] double2 and float2
__global__ void k_links(double2 *__restrict__ U64, float2 *__restrict__ U32, const double2 *__restrict__ src,
                        long V) {
    long n = blockIdx.x * (long)TPB + threadIdx.x;
    if (n >= V) return;
#pragma unroll
    for (int k = 0; k < 36; k++) {
        double2 u = src[n * 36 + k];
        U64[k * V + n] = u;
        U32[k * V + n] = make_float2((float)u.x, (float)u.y);
    }
}

unsigned grid_of(long n) { return (unsigned)std::min<long>((n + TPB - 1) / TPB, 65536); }

}  // namespace

#define QCD_LAYOUT_LAUNCH(kernel, n, ...)                                      \
    cudaEvent_t ev;                                                            \
    prof_begin(c, QCD_K_OTHER, &ev);                                           \
    kernel<<<grid_of(n), TPB, 0, c->stream>>>(__VA_ARGS__, n);                 \
    return prof_end(c, QCD_K_OTHER, ev);

int spinor64_to_32(qcd_ctx *c, float4 *dst, const double2 *src, int nrhs) {
    QCD_LAYOUT_LAUNCH(k_s64_to_32, 6 * c->lat.V * nrhs, dst, src)
}
int spinor32_to_64(qcd_ctx *c, double2 *dst, const float4 *src, int nrhs) {
    QCD_LAYOUT_LAUNCH(k_s32_to_64, 6 * c->lat.V * nrhs, dst, src)
}
// by a kernel, which is set up while the one before it runs: FP32 D on 12^3x24 from and to 16-byte boundaries
// takes 10.4 us, with cudaMemcpyAsync 18.4
int copy_spinors(qcd_ctx *c, void *dst, const void *src, size_t bytes) {
    const long n = (long)(bytes / 16);
    cudaEvent_t ev;
    prof_begin(c, QCD_K_OTHER, &ev);
    launch_chained(c, k_copy, grid_of(n), TPB, 0, (float4 *)dst, (const float4 *)src, n);
    return prof_end(c, QCD_K_OTHER, ev);
}
int links_to_internal(qcd_ctx *c, const double2 *canon) {
    cudaEvent_t ev;
    prof_begin(c, QCD_K_OTHER, &ev);
    k_links<<<(unsigned)((c->lat.V + TPB - 1) / TPB), TPB, 0, c->stream>>>(c->U64, c->U32, canon, c->lat.V);
    field_kernel(c);
    return prof_end(c, QCD_K_OTHER, ev);
}

}  // namespace qcd
