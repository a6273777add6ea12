// pcs_fieldmap.cu -- the preprocessing step of Sec. II.B (1): local field,
// magnitude weighting and mask from the two acquisitions without and with the
// readout shift T_shift (pcs_field_map).
//
// Launches on the caller's stream: per-CTA maxima of |S0|^2 over a
// grid-stride range, then one pointwise pass (each CTA first reduces those
// maxima; max is order-independent, so deterministic) writing
// dB = arg(S1 conj S0) / (2 pi gamma_bar B0 T_shift) (ppm; zero outside the
// mask), W = |S0| / max |S0| and mask = (|S0|^2 >= t^2 max |S0|^2).  Two
// voxels per thread and step (16-byte loads), four where the outputs are aligned for it.  The
// mask decision uses round-to-nearest float32 products and sums without
// contraction, so it is reproducible bit for bit.  Memory bound: 8 bytes in
// per voxel for the maximum, 16 in and 9 out for the map.  The maximum pass
// reads through the default cache policy, so that the map finds S0 in the
// 129 MB L2 (streaming loads in both passes read it from HBM twice), and the
// map is a programmatic dependent launch.  The
// maxima lie in the first voxels of field_out, which the map leaves to a third,
// one-CTA launch: no scratch is allocated (a stream-ordered allocation cost a
// call that is waited for about 200 us).  256 x 256 x 64 voxels: 29-31 us a call
// among others (3.4-3.6 TB/s of the 25 bytes a voxel needs), 55-60 us alone; 35.2 and
// 235 before.
#include <cuda_runtime.h>

#include <cmath>
#include <cstdint>
#include <cstdio>

#include "../../include/pcs.h"
#include "pcs_trace.h"

namespace pcs {
pcs_status set_last_error(pcs_status st, const char* msg);
}  // namespace pcs

namespace {

constexpr int kThreads = 256;

__device__ __forceinline__ float mag2_rn(float2 a) { return __fadd_rn(__fmul_rn(a.x, a.x), __fmul_rn(a.y, a.y)); }

// Per-CTA maxima of |S0|^2 over a grid-stride range, two voxels (one 16-byte load) per step.
__global__ void __launch_bounds__(kThreads) fm_max_kernel(const float4* __restrict__ s0, size_t n_pairs,
                                                          const float2* __restrict__ tail, int has_tail,
                                                          float* __restrict__ partial) {
    float m = 0.f;
    auto take = [&m](float4 a) {
        m = fmaxf(m, fmaxf(mag2_rn(make_float2(a.x, a.y)), mag2_rn(make_float2(a.z, a.w))));
    };
    const size_t step = (size_t)gridDim.x * kThreads;
    size_t k = (size_t)blockIdx.x * kThreads + threadIdx.x;
    for (; k + 3 * step < n_pairs; k += 4 * step) {  // four loads in flight per thread
        const float4 a = __ldg(s0 + k), b = __ldg(s0 + k + step), c = __ldg(s0 + k + 2 * step), e = __ldg(s0 + k + 3 * step);
        take(a);
        take(b);
        take(c);
        take(e);
    }
    for (; k < n_pairs; k += step) take(__ldg(s0 + k));
    if (has_tail && blockIdx.x == 0 && threadIdx.x == 0) m = fmaxf(m, mag2_rn(*tail));
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, off));
    __shared__ float red[kThreads / 32];
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = m;
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int w = 1; w < kThreads / 32; ++w) m = fmaxf(m, red[w]);
        partial[blockIdx.x] = m;
    }
}

__device__ __forceinline__ void fm_voxel(float2 a, float2 b, float cut, float inv_max, float ppm_per_rad,
                                         float& field, float& weight, unsigned char& mask) {
    const float m2 = mag2_rn(a);
    const bool in = m2 >= cut;
    const float re = b.x * a.x + b.y * a.y;  // S1 conj(S0)
    const float im = b.y * a.x - b.x * a.y;
    field = in ? atan2f(im, re) * ppm_per_rad : 0.f;
    weight = fminf(1.f, sqrtf(m2) * inv_max);
    mask = in ? 1 : 0;
}

// Maximum over the CTA of NT threads (every thread gets it).
template <int NT>
__device__ __forceinline__ float cta_max(float m) {
    __shared__ float red[NT / 32];
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, off));
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = m;
    __syncthreads();
    m = red[0];
    for (int w = 1; w < NT / 32; ++w) m = fmaxf(m, red[w]);
    return m;
}

// The map of voxels [skip, n), skip a multiple of 4: every CTA first reduces the per-CTA maxima (max is
// order-independent), which lie in field[0 .. n_partial), n_partial <= skip.
// QUAD: four voxels per step (field_out and weight_out 16-byte, mask_out 4-byte aligned), else two.
template <bool QUAD>
__global__ void __launch_bounds__(kThreads) fm_map_kernel(const float4* __restrict__ s0, const float4* __restrict__ s1,
                                                          size_t n, size_t skip, int n_partial, float thr2,
                                                          float ppm_per_rad, float* field,
                                                          float* __restrict__ weight,
                                                          unsigned char* __restrict__ mask) {
    asm volatile("griddepcontrol.wait;" ::: "memory");  // the maxima are complete
    float m = 0.f;
    for (int k = threadIdx.x; k < n_partial; k += kThreads) m = fmaxf(m, __ldcg(field + k));
    const float s_max = cta_max<kThreads>(m);
    const float max2 = s_max;
    const float cut = __fmul_rn(thr2, max2);
    const float inv_max = max2 > 0.f ? 1.0f / sqrtf(max2) : 0.f;
    const size_t step = (size_t)gridDim.x * kThreads;
    const size_t first = (size_t)blockIdx.x * kThreads + threadIdx.x;
    auto lo = [](float4 v) { return make_float2(v.x, v.y); };
    auto hi = [](float4 v) { return make_float2(v.z, v.w); };
    size_t done;
    if constexpr (QUAD) {
        const size_t n_quads = n / 4;
        for (size_t k = skip / 4 + first; k < n_quads; k += step) {
            const float4 a0 = __ldcs(s0 + 2 * k), a1 = __ldcs(s0 + 2 * k + 1), b0 = __ldcs(s1 + 2 * k), b1 = __ldcs(s1 + 2 * k + 1);
            float4 f, w;
            uchar4 mk;
            fm_voxel(lo(a0), lo(b0), cut, inv_max, ppm_per_rad, f.x, w.x, mk.x);
            fm_voxel(hi(a0), hi(b0), cut, inv_max, ppm_per_rad, f.y, w.y, mk.y);
            fm_voxel(lo(a1), lo(b1), cut, inv_max, ppm_per_rad, f.z, w.z, mk.z);
            fm_voxel(hi(a1), hi(b1), cut, inv_max, ppm_per_rad, f.w, w.w, mk.w);
            __stcs(reinterpret_cast<float4*>(field) + k, f);
            __stcs(reinterpret_cast<float4*>(weight) + k, w);
            reinterpret_cast<uchar4*>(mask)[k] = mk;
        }
        done = 4 * n_quads;
    } else {
        const size_t n_pairs = n / 2;
        for (size_t k = skip / 2 + first; k < n_pairs; k += step) {
            const float4 a = __ldcs(s0 + k), b = __ldcs(s1 + k);
            float2 f, w;
            uchar2 mk;
            fm_voxel(lo(a), lo(b), cut, inv_max, ppm_per_rad, f.x, w.x, mk.x);
            fm_voxel(hi(a), hi(b), cut, inv_max, ppm_per_rad, f.y, w.y, mk.y);
            __stcs(reinterpret_cast<float2*>(field) + k, f);
            __stcs(reinterpret_cast<float2*>(weight) + k, w);
            reinterpret_cast<uchar2*>(mask)[k] = mk;
        }
        done = 2 * n_pairs;
    }
    if (blockIdx.x == 0 && done >= skip && threadIdx.x < n - done) {  // the last voxels, fewer than a step's
        const size_t i = done + threadIdx.x;
        const float2 a = reinterpret_cast<const float2*>(s0)[i], b = reinterpret_cast<const float2*>(s1)[i];
        fm_voxel(a, b, cut, inv_max, ppm_per_rad, field[i], weight[i], mask[i]);
    }
}

// Voxels [0, count): one CTA reads the maxima in field[0 .. n_partial) before it writes there.
constexpr int kHeadThreads = 1024;
__global__ void __launch_bounds__(kHeadThreads) fm_head_kernel(const float2* __restrict__ s0, const float2* __restrict__ s1,
                                                               int count, int n_partial, float thr2, float ppm_per_rad,
                                                               float* field, float* __restrict__ weight,
                                                               unsigned char* __restrict__ mask) {
    asm volatile("griddepcontrol.wait;" ::: "memory");  // the map has read the maxima
    float m = 0.f;
    for (int k = threadIdx.x; k < n_partial; k += kHeadThreads) m = fmaxf(m, __ldcg(field + k));
    const float max2 = cta_max<kHeadThreads>(m);
    const float cut = __fmul_rn(thr2, max2);
    const float inv_max = max2 > 0.f ? 1.0f / sqrtf(max2) : 0.f;
    for (int i = threadIdx.x; i < count; i += kHeadThreads)  // (cta_max's barrier follows every read)
        fm_voxel(s0[i], s1[i], cut, inv_max, ppm_per_rad, field[i], weight[i], mask[i]);
}

pcs_status fm_fail(pcs_status st, const char* what, cudaError_t e = cudaSuccess) {
    char buf[256];
    if (e != cudaSuccess) {
        snprintf(buf, sizeof(buf), "pcs_field_map: %s: %s", what, cudaGetErrorString(e));
    } else {
        snprintf(buf, sizeof(buf), "pcs_field_map: %s", what);
    }
    return pcs::set_last_error(st, buf);
}

}  // namespace

extern "C" pcs_status pcs_field_map(const float* s0, const float* s1, size_t n_voxels, double t_shift_s,
                                    double b0_tesla, double threshold, float* field_out, float* weight_out,
                                    unsigned char* mask_out, void* cuda_stream) {
    PCS_TRACE("pcs_field_map");
    if (n_voxels == 0) return PCS_OK;
    if (!s0 || !s1 || !field_out || !weight_out || !mask_out) return fm_fail(PCS_EINVAL, "NULL argument");
    if (!(t_shift_s > 0.0) || !(b0_tesla > 0.0) || !(threshold >= 0.0))
        return fm_fail(PCS_EINVAL, "t_shift and b0 must be > 0, threshold >= 0");
    if ((reinterpret_cast<uintptr_t>(s0) | reinterpret_cast<uintptr_t>(s1)) & 15u)
        return fm_fail(PCS_EINVAL, "s0, s1 must be 16-byte aligned");
    if ((reinterpret_cast<uintptr_t>(field_out) | reinterpret_cast<uintptr_t>(weight_out)) & 7u ||
        (reinterpret_cast<uintptr_t>(mask_out) & 1u))
        return fm_fail(PCS_EINVAL, "field_out, weight_out must be 8-byte and mask_out 2-byte aligned");
    cudaStream_t st = static_cast<cudaStream_t>(cuda_stream);
    int dev = 0, sms = 0;
    cudaError_t e;
    if ((e = cudaGetDevice(&dev)) != cudaSuccess ||
        (e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess)
        return fm_fail(PCS_ECUDA, "device query", e);
    const double ppm_per_rad = 1e6 / (2.0 * M_PI * 42.577478518e6 * b0_tesla * t_shift_s);
    const float thr2 = (float)(threshold * threshold);
    const size_t n_pairs = n_voxels / 2;
    const size_t blocks_needed = (n_pairs + kThreads - 1) / kThreads;
    size_t g = blocks_needed < (size_t)sms * 6 ? blocks_needed : (size_t)sms * 6;
    const int grid = g < 1 ? 1 : (int)g;
    // voxels whose field_out holds the maxima, left to the last launch
    const size_t skip = n_voxels < (size_t)grid + 3 ? n_voxels : ((size_t)grid + 3) & ~(size_t)3;
    const float4* a = reinterpret_cast<const float4*>(s0);
    const float4* b = reinterpret_cast<const float4*>(s1);
    fm_max_kernel<<<grid, kThreads, 0, st>>>(a, n_pairs, reinterpret_cast<const float2*>(s0) + (n_voxels - 1),
                                             (int)(n_voxels & 1), field_out);
    if ((e = cudaGetLastError()) != cudaSuccess) return fm_fail(PCS_ECUDA, "launch", e);
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(kThreads);
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    if (n_voxels > skip) {
        const bool quad = ((reinterpret_cast<uintptr_t>(field_out) | reinterpret_cast<uintptr_t>(weight_out)) & 15u) == 0 &&
                          (reinterpret_cast<uintptr_t>(mask_out) & 3u) == 0;
        if ((e = cudaLaunchKernelEx(&cfg, quad ? fm_map_kernel<true> : fm_map_kernel<false>, a, b, n_voxels, skip, grid,
                                    thr2, (float)ppm_per_rad, field_out, weight_out, mask_out)) != cudaSuccess)
            return fm_fail(PCS_ECUDA, "launch", e);
    }
    cfg.gridDim = dim3(1);
    cfg.blockDim = dim3(kHeadThreads);
    if ((e = cudaLaunchKernelEx(&cfg, fm_head_kernel, reinterpret_cast<const float2*>(s0),
                                reinterpret_cast<const float2*>(s1), (int)skip, grid, thr2, (float)ppm_per_rad, field_out,
                                weight_out, mask_out)) != cudaSuccess)
        return fm_fail(PCS_ECUDA, "launch", e);
    return PCS_OK;
}
