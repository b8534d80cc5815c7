// Adjoint propagator, velocity gradient with checkpointing, FP64 dot product.
//
// Adjoint.  With D = 1 + e, E = 1 - e, C = dt^2 v^2, the transpose of the
// forward map wavelet -> traces runs backward as
//     D mu^n = 2 mu^{n+1} - E mu^{n+2} + L(C mu^{n+1}) + R^T r^{n-1}.
// Multiplying by C shows that psi = C mu obeys the forward recurrence
//     D psi^n = 2 psi^{n+1} - E psi^{n+2} + C L psi^{n+1} + C R^T r^{n-1},
// so the adjoint reuses the forward step kernels run backward in time: the
// receivers become injection points (scale c, no cell volume), the residual
// read backward in time is their wavelet (rows [nt][nrec] as given: one
// contiguous row per step), and the sources are gathered; the
// adjoint source is a[s][n] = psi^{n+1}(x_s) / (hx hy hz).
//
// Gradient.  dJ/dc(x) = sum_n mu^{n+1}(x) g^n(x), g^n = L u^n + s^n, so
// with mu = psi / c the kernels accumulate A = sum_n psi^{n+1} g^n (FP32)
// and dJ/dv = 2 dt^2 v A / c = 2 A / v.  g^n is written by the step kernel that
// advances u^n (the Laplacian it already holds, plus w[n] / (hx hy hz) at the
// sources): no difference of nearly equal wavefields is formed.  The forward
// states are recovered from checkpoints (u^{a-1}, u^a) (FP32, or BF16 / FP16
// with one scale per z plane) by one of two schemes:
//   segments: the first sweep stores a checkpoint at the start of each of S
//     segments of K steps; the backward sweep replays each segment from its
//     checkpoint, in place in two volumes, writing g^n into K more, and runs
//     the segment's adjoint steps against them.  Memory: 2 S checkpoint
//     volumes + K + 2; work: two forward sweeps and one adjoint (with FP32
//     checkpoints the first sweep writes g^n of the last segment itself,
//     which is then not replayed);
//   revolve: the binomial schedule of mmod_revolve.cu over S slots, with the
//     working state in the handle's two buffers, u^{n+1} and g^n of a
//     reversed step in two more volumes; the fewest replayed steps for S slots;
//   segments with S >= nt and FP32 storage keeps g^n of every step (nt + 2
//     volumes, written by the first sweep): no replay.
#include <cooperative_groups.h>
#include <cuda_bf16.h>
#include <cuda_fp16.h>

#include <algorithm>
#include <cfloat>
#include <cstdint>
#include <cstring>

#include "mmod_handle.h"

#define MMOD_API extern "C" __attribute__((visibility("default")))

using namespace mmod;

namespace {

// ---- checkpoint storage: one scale per z plane, 16-bit values ------------

template <class T>
__device__ __forceinline__ T to_store(float v);
template <>
__device__ __forceinline__ __nv_bfloat16 to_store<__nv_bfloat16>(float v) { return __float2bfloat16_rn(v); }
template <>
__device__ __forceinline__ __half to_store<__half>(float v) { return __float2half_rn(v); }
__device__ __forceinline__ float from_store(__nv_bfloat16 v) { return __bfloat162float(v); }
__device__ __forceinline__ float from_store(__half v) { return __half2float(v); }

__device__ __forceinline__ uint32_t pack2(__nv_bfloat16 a, __nv_bfloat16 b) {
    return (uint32_t)__bfloat16_as_ushort(a) | (uint32_t)__bfloat16_as_ushort(b) << 16;
}
__device__ __forceinline__ uint32_t pack2(__half a, __half b) {
    return (uint32_t)__half_as_ushort(a) | (uint32_t)__half_as_ushort(b) << 16;
}
__device__ __forceinline__ uint32_t pack2(short a, short b) {
    return (uint32_t)(unsigned short)a | (uint32_t)(unsigned short)b << 16;
}
template <class T>
__device__ __forceinline__ T stored_half(uint32_t w);
template <>
__device__ __forceinline__ __nv_bfloat16 stored_half<__nv_bfloat16>(uint32_t w) {
    return __ushort_as_bfloat16((unsigned short)w);
}
template <>
__device__ __forceinline__ __half stored_half<__half>(uint32_t w) { return __ushort_as_half((unsigned short)w); }
template <>
__device__ __forceinline__ short stored_half<short>(uint32_t w) { return (short)(unsigned short)w; }

// The two volumes of a checkpoint (u^{a-1}, u^a), handled by one launch
// (blockIdx.y selects the volume): each is a few microseconds of traffic, so
// separate launches would cost as much as the work.
template <class T>
struct CkptPair {
    float *u[2];
    T *q[2];
    float *scale[2];
};

// Scale = max(max |u| over the plane, FLT_MIN), stored = u / scale.  A cluster
// of kPlaneCtas CTAs serves one plane: each takes the maximum of its share,
// the shares meet through distributed shared memory, and the second pass
// reads the plane again from L2.  Bound by memory; one CTA per plane left most
// of the chip idle (a 133 x 144 x 120 volume is 120 planes of 92 KB).  That
// form took 17.7 us per volume there and 15.4 us to restore it, with 4-byte
// accesses; with clusters, 32 bytes per thread and access and one launch per
// state, the gradient of that box (200 steps, binomial schedule, 10 BF16
// slots) went from 24.4 to 18.5 ms.  Padded rows
// are a multiple of 32 floats, so groups of 8 values tile a plane exactly and
// start on 16-byte boundaries.
constexpr int kPlaneCtas = 8;

template <class T>
__global__ void __cluster_dims__(kPlaneCtas, 1, 1) __launch_bounds__(256)
    compress_kernel(const CkptPair<T> p, long long plane) {
    namespace cg = cooperative_groups;
    cg::cluster_group cluster = cg::this_cluster();
    // programmatic dependent launch: the step that follows only reads these volumes before its own wait
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    const int k = blockIdx.x / kPlaneCtas, rank = blockIdx.x % kPlaneCtas, vol = blockIdx.y;
    const float4 *u = reinterpret_cast<const float4 *>(p.u[vol] + (long long)k * plane);
    const long long groups = plane >> 3;
    const int first = rank * 256 + threadIdx.x;
    float m = 0.0f;
#pragma unroll 4
    for (long long g = first; g < groups; g += kPlaneCtas * 256) {
        const float4 a = u[2 * g], b = u[2 * g + 1];
        m = fmaxf(m, fmaxf(fmaxf(fmaxf(fabsf(a.x), fabsf(a.y)), fmaxf(fabsf(a.z), fabsf(a.w))),
                           fmaxf(fmaxf(fabsf(b.x), fabsf(b.y)), fmaxf(fabsf(b.z), fabsf(b.w)))));
    }
    for (int off = 16; off > 0; off >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, off));
    __shared__ float part[8];
    if ((threadIdx.x & 31) == 0) part[threadIdx.x >> 5] = m;
    cluster.sync();
    m = *cluster.map_shared_rank(&part[threadIdx.x & 7], (threadIdx.x >> 3) & (kPlaneCtas - 1));
    for (int off = 16; off > 0; off >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, off));
    __shared__ float half_max[2];   // a warp holds the shares of four CTAs: warps 0 and 1 cover all eight
    if (threadIdx.x < 64 && (threadIdx.x & 31) == 0) half_max[threadIdx.x >> 5] = m;
    cluster.sync();   // also: no CTA leaves while another still reads its shares
    // A plane that holds only zeros and subnormals (the leading edge of a
    // wave, far planes early in a run) gets the smallest normal scale, so
    // 1/scale stays finite.
    const float s = fmaxf(fmaxf(half_max[0], half_max[1]), FLT_MIN);
    if (first == 0) p.scale[vol][k] = s;
    const float inv = 1.0f / s;
    uint4 *out = reinterpret_cast<uint4 *>(p.q[vol] + (long long)k * plane);
#pragma unroll 2
    for (long long g = first; g < groups; g += kPlaneCtas * 256) {
        const float4 a = u[2 * g], b = u[2 * g + 1];
        out[g] = make_uint4(pack2(to_store<T>(a.x * inv), to_store<T>(a.y * inv)),
                            pack2(to_store<T>(a.z * inv), to_store<T>(a.w * inv)),
                            pack2(to_store<T>(b.x * inv), to_store<T>(b.y * inv)),
                            pack2(to_store<T>(b.z * inv), to_store<T>(b.w * inv)));
    }
}

template <class T>
__global__ void __launch_bounds__(256) decompress_kernel(const CkptPair<T> p, long long plane, int ctas) {
    // no early release: the step that follows needs these volumes at once
    asm volatile("griddepcontrol.wait;" ::: "memory");
    const int k = blockIdx.x / ctas, vol = blockIdx.y;   // ctas CTAs per plane
    const uint4 *in = reinterpret_cast<const uint4 *>(p.q[vol] + (long long)k * plane);
    float4 *u = reinterpret_cast<float4 *>(p.u[vol] + (long long)k * plane);
    const float s = p.scale[vol][k];
    const long long groups = plane >> 3;
#pragma unroll 2
    for (long long g = (long long)(blockIdx.x % ctas) * 256 + threadIdx.x; g < groups; g += (long long)ctas * 256) {
        const uint4 v = in[g];
        float4 a, b;
        a.x = from_store(stored_half<T>(v.x)) * s; a.y = from_store(stored_half<T>(v.x >> 16)) * s;
        a.z = from_store(stored_half<T>(v.y)) * s; a.w = from_store(stored_half<T>(v.y >> 16)) * s;
        b.x = from_store(stored_half<T>(v.z)) * s; b.y = from_store(stored_half<T>(v.z >> 16)) * s;
        b.z = from_store(stored_half<T>(v.w)) * s; b.w = from_store(stored_half<T>(v.w >> 16)) * s;
        u[2 * g] = a;
        u[2 * g + 1] = b;
    }
}

// Block floating point (MMOD_CKPT_BFP16): per block of 32 consecutive x
// values of a padded row (rows are padded to 32, so blocks never straddle
// rows), scale s = max |u| over the block and q = round(u * 32767 / s) as
// int16; u is restored as q * (s / 32767), within s / 65534 of the stored
// value.  s is at least kBfpMin, 2^15 times the smallest normal number, so that
// 32767 / s and s / 32767 are finite and normal (below it, the far tail of a wave
// was stored as +-s).  Four threads per block, eight values each (16-byte
// accesses).
constexpr int kBfpBlock = 32;
constexpr float kBfpMax = 32767.0f;
constexpr float kBfpMin = 32768.0f * FLT_MIN;

__device__ __forceinline__ short bfp_value(float v, float s) {
    return (short)max(-32767, min(32767, __float2int_rn(v * (kBfpMax / s))));
}

__global__ void __launch_bounds__(256) compress_bfp_kernel(const CkptPair<short> p, long long nblocks) {
    asm volatile("griddepcontrol.wait;" ::: "memory");   // as compress_kernel
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    const float4 *u = reinterpret_cast<const float4 *>(p.u[blockIdx.y]);
    uint4 *out = reinterpret_cast<uint4 *>(p.q[blockIdx.y]);
    const long long groups = 4 * nblocks, stride = (long long)gridDim.x * 256;
    // a warp's lanes leave the loop together: its base is a multiple of 32
    for (long long base = (long long)blockIdx.x * 256 + (threadIdx.x & ~31); base < groups; base += stride) {
        const long long g = base + (threadIdx.x & 31);
        const bool in = g < groups;
        const float4 z = make_float4(0.0f, 0.0f, 0.0f, 0.0f), a = in ? u[2 * g] : z, b = in ? u[2 * g + 1] : z;
        float m = fmaxf(fmaxf(fmaxf(fabsf(a.x), fabsf(a.y)), fmaxf(fabsf(a.z), fabsf(a.w))),
                        fmaxf(fmaxf(fabsf(b.x), fabsf(b.y)), fmaxf(fabsf(b.z), fabsf(b.w))));
        m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, 1));
        m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, 2));
        if (m < kBfpMin) m = kBfpMin;   // not a block of NaN
        if (!in) continue;
        out[g] = make_uint4(pack2(bfp_value(a.x, m), bfp_value(a.y, m)), pack2(bfp_value(a.z, m), bfp_value(a.w, m)),
                            pack2(bfp_value(b.x, m), bfp_value(b.y, m)), pack2(bfp_value(b.z, m), bfp_value(b.w, m)));
        if ((g & 3) == 0) p.scale[blockIdx.y][g >> 2] = m;
    }
}

__global__ void __launch_bounds__(256) decompress_bfp_kernel(const CkptPair<short> p, long long nblocks) {
    asm volatile("griddepcontrol.wait;" ::: "memory");   // no early release, as decompress_kernel
    const uint4 *in = reinterpret_cast<const uint4 *>(p.q[blockIdx.y]);
    float4 *u = reinterpret_cast<float4 *>(p.u[blockIdx.y]);
    const long long groups = 4 * nblocks, stride = (long long)gridDim.x * 256;
    for (long long g = (long long)blockIdx.x * 256 + threadIdx.x; g < groups; g += stride) {
        const float f = p.scale[blockIdx.y][g >> 2] / kBfpMax;
        const uint4 v = in[g];
        float4 a, b;
        a.x = (float)stored_half<short>(v.x) * f; a.y = (float)stored_half<short>(v.x >> 16) * f;
        a.z = (float)stored_half<short>(v.y) * f; a.w = (float)stored_half<short>(v.y >> 16) * f;
        b.x = (float)stored_half<short>(v.z) * f; b.y = (float)stored_half<short>(v.z >> 16) * f;
        b.z = (float)stored_half<short>(v.w) * f; b.w = (float)stored_half<short>(v.w >> 16) * f;
        u[2 * g] = a;
        u[2 * g + 1] = b;
    }
}

int bfp_grid(long long nblocks) { return (int)std::min<long long>((nblocks + 63) / 64, 152LL * 8); }

size_t ckpt_elem_bytes(int dtype) { return dtype == MMOD_CKPT_FP32 ? 4 : 2; }

// Scales per checkpoint volume: one per z plane (BF16 / FP16), one per
// 32-value block (BFP16), none (FP32).
size_t ckpt_scales(const mmod_handle *h, int dtype) {
    if (dtype == MMOD_CKPT_BFP16) return (size_t)h->vol / kBfpBlock;
    return dtype == MMOD_CKPT_FP32 ? 0 : (size_t)h->cfg.nz;
}

template <class T>
CkptPair<T> ckpt_pair(mmod_handle *h, int slot, float *u_prev, float *u_cur) {
    auto &gw = h->gw;
    CkptPair<T> p;
    p.u[0] = u_prev;
    p.u[1] = u_cur;
    for (int i = 0; i < 2; ++i) {
        p.q[i] = static_cast<T *>(gw.ckpt) + (size_t)(2 * slot + i) * h->vol;
        p.scale[i] = gw.ckpt_scale ? gw.ckpt_scale + (size_t)(2 * slot + i) * ckpt_scales(h, gw.dtype) : nullptr;
    }
    return p;
}

// Launch of a checkpoint kernel, chained to its stream predecessor by
// programmatic dependent launch where the handle uses it.
template <class... P, class... A>
cudaError_t launch_ckpt(const mmod_handle *h, void (*fn)(P...), dim3 grid, cudaStream_t s, A... args) {
    cudaLaunchConfig_t lc = {};
    lc.gridDim = grid;
    lc.blockDim = dim3(256);
    lc.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    lc.attrs = attr;
    lc.numAttrs = h->pdl ? 1 : 0;
    return cudaLaunchKernelEx(&lc, fn, P(args)...);
}

// Save the state (u^{a-1}, u^a) into checkpoint slot (FP32: copies; 16-bit: compress).
cudaError_t save_state(mmod_handle *h, int slot, float *u_prev, float *u_cur, cudaStream_t s) {
    const int dtype = h->gw.dtype;
    const size_t vb = sizeof(float) * (size_t)h->vol;
    const dim3 grid(kPlaneCtas * h->cfg.nz, 2);
    if (dtype == MMOD_CKPT_FP32) {
        const auto p = ckpt_pair<float>(h, slot, u_prev, u_cur);
        for (int i = 0; i < 2; ++i)
            if (cudaError_t e = cudaMemcpyAsync(p.q[i], p.u[i], vb, cudaMemcpyDeviceToDevice, s)) return e;
        return cudaSuccess;
    }
    if (dtype == MMOD_CKPT_BFP16) {
        const long long nb = h->vol / kBfpBlock;
        return launch_ckpt(h, compress_bfp_kernel, dim3(bfp_grid(nb), 2), s, ckpt_pair<short>(h, slot, u_prev, u_cur), nb);
    }
    if (dtype == MMOD_CKPT_BF16)
        return launch_ckpt(h, compress_kernel<__nv_bfloat16>, grid, s,
                           ckpt_pair<__nv_bfloat16>(h, slot, u_prev, u_cur), h->plane);
    return launch_ckpt(h, compress_kernel<__half>, grid, s, ckpt_pair<__half>(h, slot, u_prev, u_cur), h->plane);
}

cudaError_t restore_state(mmod_handle *h, int slot, float *u_prev, float *u_cur, cudaStream_t s) {
    const int dtype = h->gw.dtype;
    const size_t vb = sizeof(float) * (size_t)h->vol;
    const int per = (int)std::min<long long>((h->plane / 8 + 511) / 512, 8);   // CTAs per plane
    const dim3 grid(per * h->cfg.nz, 2);
    if (dtype == MMOD_CKPT_FP32) {
        const auto p = ckpt_pair<float>(h, slot, u_prev, u_cur);
        for (int i = 0; i < 2; ++i)
            if (cudaError_t e = cudaMemcpyAsync(p.u[i], p.q[i], vb, cudaMemcpyDeviceToDevice, s)) return e;
        return cudaSuccess;
    }
    if (dtype == MMOD_CKPT_BFP16) {
        const long long nb = h->vol / kBfpBlock;
        return launch_ckpt(h, decompress_bfp_kernel, dim3(bfp_grid(nb), 2), s, ckpt_pair<short>(h, slot, u_prev, u_cur),
                           nb);
    }
    if (dtype == MMOD_CKPT_BF16)
        return launch_ckpt(h, decompress_kernel<__nv_bfloat16>, grid, s,
                           ckpt_pair<__nv_bfloat16>(h, slot, u_prev, u_cur), h->plane, per);
    return launch_ckpt(h, decompress_kernel<__half>, grid, s, ckpt_pair<__half>(h, slot, u_prev, u_cur), h->plane, per);
}

// Tensor maps of the work volumes for the run's tile shape.
mmod_status encode_grad_maps(mmod_handle *h, int shape) {
    auto &gw = h->gw;
    if (gw.shape == shape || !h->tma_ok) return MMOD_OK;
    gw.shape = -1;   // until every map is one of this shape
    bool ok = true;
    for (int i = 0; i < gw.nwork; ++i) ok = ok && encode_maps(h->cfg, h->nxp, gw.seg[i], shape, &gw.seg_map[i]);
    for (int b = 0; b < 2; ++b) ok = ok && encode_maps(h->cfg, h->nxp, gw.psi[b], shape, &gw.psi_map[b]);
    ok = ok && encode_maps(h->cfg, h->nxp, gw.gradc, shape, &gw.gradc_map);
    if (gw.dtype == MMOD_CKPT_FP32) {
        for (int i = 0; i < 2 * gw.nslot; ++i)
            ok = ok && encode_maps(h->cfg, h->nxp, static_cast<float *>(gw.ckpt) + (size_t)i * h->vol, shape,
                                   &gw.ckpt_map[i]);
    }
    if (!ok) return fail(h, MMOD_ERR_CUDA, "tensor map encoding failed for a work volume");
    gw.shape = shape;
    return MMOD_OK;
}

// Allocate (or keep) the gradient work space: nslot checkpoints of two
// volumes, nwork FP32 work volumes (with tensor maps; cleared on the run's
// stream, in front of the steps that write them), psi, grad_c.
mmod_status ensure_grad_work(mmod_handle *h, int nslot, int nwork, int dtype, int shape, cudaStream_t s) {
    auto &gw = h->gw;
    if (gw.nslot == nslot && gw.nwork == nwork && gw.dtype == dtype) return encode_grad_maps(h, shape);
    free_grad_work(h);
    const size_t vb = sizeof(float) * (size_t)h->vol;
    gw.seg.assign(nwork, nullptr);
    gw.seg_map.resize(nwork);
    gw.ckpt_map.resize(2 * (size_t)nslot);
    for (int i = 0; i < nwork; ++i) {
        MMOD_CK(h, cudaMalloc(&gw.seg[i], vb));
        MMOD_CK(h, cudaMemsetAsync(gw.seg[i], 0, vb, s));
    }
    for (int b = 0; b < 2; ++b) MMOD_CK(h, cudaMalloc(&gw.psi[b], vb));
    MMOD_CK(h, cudaMalloc(&gw.gradc, vb));
    gw.ckpt_bytes = (size_t)nslot * 2 * (size_t)h->vol * ckpt_elem_bytes(dtype);
    if (nslot > 0) MMOD_CK(h, cudaMalloc(&gw.ckpt, gw.ckpt_bytes));
    if (nslot > 0 && dtype != MMOD_CKPT_FP32)
        MMOD_CK(h, cudaMalloc(&gw.ckpt_scale, sizeof(float) * (size_t)nslot * 2 * ckpt_scales(h, dtype)));
    gw.nslot = nslot;
    gw.nwork = nwork;
    gw.dtype = dtype;
    return encode_grad_maps(h, shape);
}

// Checkpoint layout of a gradient call: slots and FP32 work volumes.
// seglen = 0 with nslot = 0: every forward state is kept (FP32 checkpoints,
// ckpt_count >= nt), so nothing is replayed.
void grad_layout(const mmod_handle *h, int ckpt_count, int dtype, int *nslot, int *nwork, int *seglen) {
    const int nt = h->cfg.nt;
    if (h->ckpt_scheme == MMOD_SCHEME_SEGMENTS && dtype == MMOD_CKPT_FP32 && ckpt_count >= nt && nt > 0) {
        *seglen = 0;
        *nslot = 0;
        *nwork = nt + 2;
        return;
    }
    if (h->ckpt_scheme == MMOD_SCHEME_REVOLVE) {
        *seglen = 0;
        *nslot = std::max(1, std::min(ckpt_count, nt - 1));
        *nwork = 2;
    } else {
        *seglen = std::max(1, (nt + ckpt_count - 1) / ckpt_count);
        *nslot = nt > 0 ? (nt + *seglen - 1) / *seglen : 1;
        *nwork = *seglen + 2;
    }
}

// Device copy of an input array: device pointers pass through, host arrays go
// through the staging buffer *stage (allocated on first use, n floats).
mmod_status device_input(mmod_handle *h, const float *p, size_t n, float **stage, const float **out,
                         cudaStream_t s) {
    if (is_device_ptr(p)) {
        *out = p;
        return MMOD_OK;
    }
    if (!*stage) MMOD_CK(h, cudaMalloc(stage, sizeof(float) * std::max<size_t>(n, 1)));
    if (n) MMOD_CK(h, cudaMemcpyAsync(*stage, p, sizeof(float) * n, cudaMemcpyHostToDevice, s));
    *out = *stage;
    return MMOD_OK;
}

// The adjoint sweep's gathers [nt][nsrc] (st_adjg) -> adj_src [nsrc][nt] in time order, host or device.
mmod_status adjoint_output(mmod_handle *h, float *adj_src, cudaStream_t s) {
    const auto &c = h->cfg;
    const size_t nadj = (size_t)c.nt * c.nsrc;
    const bool dev_out = is_device_ptr(adj_src);
    float *dst = adj_src;
    if (!dev_out) {
        if (!h->st_adjo) MMOD_CK(h, cudaMalloc(&h->st_adjo, sizeof(float) * nadj));
        dst = h->st_adjo;
    }
    MMOD_CK(h, launch_unreverse_transpose(h->st_adjg, c.nt, c.nsrc, 1.0 / (c.hx * c.hy * c.hz), dst, s));
    if (!dev_out) {
        MMOD_CK(h, cudaMemcpyAsync(adj_src, dst, sizeof(float) * nadj, cudaMemcpyDeviceToHost, s));
        MMOD_CK(h, cudaStreamSynchronize(s));
    }
    return MMOD_OK;
}

}  // namespace

namespace mmod {

void free_grad_work(mmod_handle *h) {
    auto &gw = h->gw;
    for (float *p : gw.seg)
        if (p) cudaFree(p);
    gw.seg.clear();
    gw.seg_map.clear();
    gw.ckpt_map.clear();
    for (float *&p : gw.psi) {
        if (p) cudaFree(p);
        p = nullptr;
    }
    if (gw.gradc) cudaFree(gw.gradc);
    if (gw.ckpt) cudaFree(gw.ckpt);
    if (gw.ckpt_scale) cudaFree(gw.ckpt_scale);
    gw.gradc = nullptr;
    gw.ckpt = nullptr;
    gw.ckpt_scale = nullptr;
    gw.nslot = gw.nwork = 0;
    gw.dtype = gw.shape = -1;
    gw.ckpt_bytes = 0;
}

}  // namespace mmod

MMOD_API mmod_status mmod_adjoint(mmod_handle *h, const float *resid, float *adj_src, mmod_stream stream) {
    if (!h) return MMOD_ERR_ARG;
    if (mmod_status st = check_latched(h)) return st;
    if (is_cpml(h)) return fail(h, MMOD_ERR_UNSUPPORTED, "the adjoint is built for the damping layers only");
    if (!h->model_set) return fail(h, MMOD_ERR_STATE, "mmod_set_model has not succeeded");
    const auto &c = h->cfg;
    if (c.nrec > 0 && c.nt > 0 && !resid) return fail(h, MMOD_ERR_ARG, "null residual with nrec > 0");
    if (c.nsrc > 0 && c.nt > 0 && !adj_src) return fail(h, MMOD_ERR_ARG, "null adjoint source with nsrc > 0");
    DeviceGuard guard(h->device);
    cudaStream_t s = (cudaStream_t)stream;
    const size_t nres = (size_t)c.nt * c.nrec, nadj = (size_t)c.nt * c.nsrc;
    long long launches = 0;
    const float *dres = nullptr;
    if (mmod_status st = device_input(h, resid, nres, &h->st_tr, &dres, s)) return st;
    if (!h->st_adjw) MMOD_CK(h, cudaMalloc(&h->st_adjw, sizeof(float) * std::max<size_t>(nres, 1)));
    if (!h->st_adjg) MMOD_CK(h, cudaMalloc(&h->st_adjg, sizeof(float) * std::max<size_t>(nadj, 1)));
    if (nres) MMOD_CK(h, cudaMemcpyAsync(h->st_adjw, dres, sizeof(float) * nres, cudaMemcpyDeviceToDevice, s));
    MMOD_CK(h, cudaMemsetAsync(h->u[0], 0, sizeof(float) * (size_t)h->vol, s));
    MMOD_CK(h, cudaMemsetAsync(h->u[1], 0, sizeof(float) * (size_t)h->vol, s));
    h->state_pending = false;
    if (c.nt > 0)
        if (mmod_status st = run_loop_graph(h, h->g_adj, h->adj, h->st_adjw, c.nsrc > 0 ? h->st_adjg : nullptr, s,
                                            &launches))
            return st;
    h->ran = false;   // the wavefield buffers now hold the adjoint state
    if (nadj) {
        if (mmod_status st = adjoint_output(h, adj_src, s)) return st;
        ++launches;
    }
    h->last_launches = launches;
    return check_latched(h);
}

// The velocity gradient and, with adj_src, the adjoint sources of the same
// residual: the gradient's adjoint sweep is mmod_adjoint's, so recording it at
// the sources saves the second sweep.
static mmod_status run_gradient(mmod_handle *h, const float *wavelet, const float *resid, float *grad_v,
                                float *adj_src, int ckpt_count, int ckpt_dtype, mmod_stream stream) {
    if (!h) return MMOD_ERR_ARG;
    if (mmod_status st = check_latched(h)) return st;
    if (is_cpml(h)) return fail(h, MMOD_ERR_UNSUPPORTED, "the gradient is built for the damping layers only");
    if (!h->model_set) return fail(h, MMOD_ERR_STATE, "mmod_set_model has not succeeded");
    const auto &c = h->cfg;
    if (!grad_v) return fail(h, MMOD_ERR_ARG, "null gradient output");
    if (ckpt_count < 1) return fail(h, MMOD_ERR_ARG, "ckpt_count must be >= 1");
    if (ckpt_dtype != MMOD_CKPT_FP32 && ckpt_dtype != MMOD_CKPT_BF16 && ckpt_dtype != MMOD_CKPT_FP16 &&
        ckpt_dtype != MMOD_CKPT_BFP16)
        return fail(h, MMOD_ERR_ARG, "unknown checkpoint type");
    if (c.nsrc > 0 && c.nt > 0 && !wavelet) return fail(h, MMOD_ERR_ARG, "null wavelet with nsrc > 0");
    if (c.nrec > 0 && c.nt > 0 && !resid) return fail(h, MMOD_ERR_ARG, "null residual with nrec > 0");
    DeviceGuard guard(h->device);
    cudaStream_t s = (cudaStream_t)stream;
    const int nt = c.nt;
    int nslot = 0, nwork = 0, seglen = 0;
    grad_layout(h, ckpt_count, ckpt_dtype, &nslot, &nwork, &seglen);
    const int shape = active_shape(h);
    if (mmod_status st = ensure_shape(h, shape)) return st;
    if (mmod_status st = ensure_grad_work(h, nslot, nwork, ckpt_dtype, shape, s)) return st;
    const VolMaps *u_map = h->shapes[shape].u;
    auto &gw = h->gw;
    const bool tma = use_tma(h);
    long long launches = 0;
    const size_t vb = sizeof(float) * (size_t)h->vol;

    const float *dwav = nullptr, *dres = nullptr;
    if (mmod_status st = device_input(h, wavelet, (size_t)c.nsrc * nt, &h->st_wav, &dwav, s)) return st;
    if (mmod_status st = device_input(h, resid, (size_t)c.nrec * nt, &h->st_tr, &dres, s)) return st;
    const size_t nres = (size_t)nt * c.nrec;
    if (!h->st_adjw) MMOD_CK(h, cudaMalloc(&h->st_adjw, sizeof(float) * std::max<size_t>(nres, 1)));
    if (nres) MMOD_CK(h, cudaMemcpyAsync(h->st_adjw, dres, sizeof(float) * nres, cudaMemcpyDeviceToDevice, s));

    // segments with FP32 checkpoints step through the checkpoint volumes themselves
    const bool through = ckpt_dtype == MMOD_CKPT_FP32 && seglen >= 2;
    if (!through)
        for (float *u : h->u) MMOD_CK(h, cudaMemsetAsync(u, 0, vb, s));
    h->state_pending = false;
    StepArgs fa = base_args(h, h->fwd, dwav, shape);
    fa.nrec = 0;   // no receivers in the gradient's forward sweeps
    fa.inv_cell = (float)(1.0 / (c.hx * c.hy * c.hz));
    StepArgs aa = base_args(h, h->adj, h->st_adjw, shape);
    const int nadj = adj_src ? c.nsrc : 0;   // adjoint sources recorded per step
    aa.nrec = nadj;
    if (nadj && !h->st_adjg) MMOD_CK(h, cudaMalloc(&h->st_adjg, sizeof(float) * std::max<size_t>((size_t)nt * nadj, 1)));
    // A step may request c and its u^{n-1} before its wait (pdl 2) where the
    // operation in front of it writes neither.  Steps, imaging and saves never do
    // (the sweeps alternate two volumes; forward and adjoint steps have volumes of
    // their own); a restored checkpoint and a cleared volume may be the u^{n-1} of
    // the next step, whose early copies nothing would order behind those writes:
    // that one step waits first (unsettled).  Not in the binomial schedule, where
    // early requests measured 1 % slower (133 x 144 x 120), against 1-3 % faster
    // in segments.
    const int steady_pdl = h->pdl && h->ckpt_scheme != MMOD_SCHEME_REVOLVE ? 2 : h->pdl;
    bool unsettled = true;   // the last operation on the stream cleared or restored volumes
    auto enqueue = [&](StepArgs &a, const VolMaps &cur, const VolMaps &prev, float *plain_gather_dst) {
        a.pdl = unsettled ? h->pdl : steady_pdl;
        unsettled = false;
        return enqueue_step(h, a, cur, prev, tma, plain_gather_dst, s, &launches);
    };
    auto clear = [&](float *p, size_t bytes) {
        unsettled = true;
        return cudaMemsetAsync(p, 0, bytes, s);
    };
    auto restore = [&](int slot, float *u_prev, float *u_cur) {
        unsettled = true;
        return restore_state(h, slot, u_prev, u_cur, s);
    };
    // forward step n in place on the handle's buffers: u^{n-1} in u[n & 1],
    // u^n in u[(n + 1) & 1], u^{n+1} over u^{n-1}
    auto fwd_step_in_place = [&](int n) {
        fa.n = n;
        fa.ucur = h->u[(n + 1) & 1];
        fa.uprev = h->u[n & 1];
        fa.uout = h->u[n & 1];
        return enqueue(fa, u_map[(n + 1) & 1], u_map[n & 1], nullptr);
    };
    // forward step n from u^{n-1} in prev and u^n in cur into out (prev's
    // volume or another), also writing g^n into gout (null: not)
    struct Vol {
        float *p;
        const VolMaps *m;
    };
    auto seg = [&](int i) { return Vol{gw.seg[i], &gw.seg_map[i]}; };
    auto slot = [&](int sg, int i) {
        return Vol{static_cast<float *>(gw.ckpt) + (size_t)(2 * sg + i) * h->vol, &gw.ckpt_map[2 * sg + i]};
    };
    auto fwd_step = [&](int n, Vol prev, Vol cur, Vol out, float *gout) {
        fa.n = n;
        fa.ucur = cur.p;
        fa.uprev = prev.p;
        fa.uout = out.p;
        fa.gout = gout;
        const cudaError_t e = enqueue(fa, *cur.m, *prev.m, nullptr);
        fa.gout = nullptr;
        return e;
    };
    // forward step n of a replay in the work volumes w0, w1 (u^{n-1} in w0,
    // u^n in w1, u^{n+1} over u^{n-1}), also writing g^n into gout
    auto fwd_step_g = [&](int n, int w0, int w1, float *gout) { return fwd_step(n, seg(w0), seg(w1), seg(w0), gout); };
    // forward steps a0 .. b0-1 from the state in p0 (u^{a0-1}), p1 (u^{a0}),
    // which stay as they are, through q0, q1: u^{a0+1+j} lands in q0, q1 in
    // turn; gof(j): where g of step a0 + j goes (null: not written)
    auto fwd_range = [&](int a0, int b0, Vol p0, Vol p1, Vol q0, Vol q1, auto gof) -> cudaError_t {
        for (int n = a0; n < b0; ++n) {
            const int j = n - a0;
            const Vol out = j & 1 ? q1 : q0, prev = j == 0 ? p0 : j == 1 ? p1 : out, cur = j == 0 ? p1 : j & 1 ? q0 : q1;
            if (cudaError_t e = fwd_step(n, prev, cur, out, gof(j))) return e;
        }
        return cudaSuccess;
    };
    // adjoint step of forward step n: adjoint step m = nt-1-n produces
    // psi^{n+1} in psi[m & 1] (psi^{n+2} stays in the other buffer until the
    // next adjoint step)
    auto adj_step = [&](int n) {
        const int m = nt - 1 - n;
        aa.n = m;
        aa.ucur = gw.psi[(m + 1) & 1];
        aa.uprev = gw.psi[m & 1];
        aa.uout = gw.psi[m & 1];
        // the step kernel records the field it reads (adjoint step m - 1); the plain path the one it writes
        aa.traces = nadj && m >= 1 ? h->st_adjg + (size_t)(m - 1) * nadj : nullptr;
        return enqueue(aa, gw.psi_map[(m + 1) & 1], gw.psi_map[m & 1],
                       nadj ? h->st_adjg + (size_t)m * nadj : nullptr);
    };
    // imaging terms of forward steps n (and n - 1 when ns = 2) from g[t] =
    // g^{n-t}, after their adjoint steps: psi^{n+1} in psi[(nt-1-n) & 1],
    // psi^n in the other buffer
    auto image = [&](int n, const float *const *g, int ns) {
        const int m = nt - 1 - n;
        const float *ps[2] = {gw.psi[m & 1], gw.psi[(m + 1) & 1]};
        ++launches;
        return launch_imaging(ns, ps, g, c.nx, c.ny, c.nz, h->nxp, gw.gradc, s);
    };
    // steps hi down to lo with g^j in gof(j): two adjoint steps, then one
    // imaging pass over both (the same accumulation order as one pass per
    // step, the accumulator read and written once per pair)
    auto backward_range = [&](int hi, int lo, auto gof) -> cudaError_t {
        int n = hi;
        for (; n - 1 >= lo; n -= 2) {
            cudaError_t e = adj_step(n);
            if (e == cudaSuccess) e = adj_step(n - 1);
            if (e != cudaSuccess) return e;
            const float *g[2] = {gof(n), gof(n - 1)};
            if ((e = image(n, g, 2)) != cudaSuccess) return e;
        }
        if (n == lo) {
            cudaError_t e = adj_step(n);
            if (e != cudaSuccess) return e;
            const float *g[1] = {gof(n)};
            return image(n, g, 1);
        }
        return cudaSuccess;
    };

    if (seglen == 0 && nslot == 0) {
        // every step's g^n kept: seg[0], seg[1] hold the stepped state,
        // seg[2 + n] = g^n
        MMOD_CK(h, clear(gw.seg[0], vb));
        MMOD_CK(h, clear(gw.seg[1], vb));
        for (int n = 0; n < nt; ++n) MMOD_CK(h, fwd_step_g(n, n & 1, (n + 1) & 1, gw.seg[2 + n]));
        MMOD_CK(h, clear(gw.psi[0], vb));
        MMOD_CK(h, clear(gw.psi[1], vb));
        MMOD_CK(h, clear(gw.gradc, vb));
        MMOD_CK(h, backward_range(nt - 1, 0, [&](int j) { return gw.seg[2 + j]; }));
    } else if (h->ckpt_scheme == MMOD_SCHEME_REVOLVE) {
        std::vector<RevAction> sched;
        revolve_schedule(nt, nslot, &sched);
        MMOD_CK(h, clear(gw.psi[0], vb));
        MMOD_CK(h, clear(gw.psi[1], vb));
        MMOD_CK(h, clear(gw.gradc, vb));
        float *unext = gw.seg[0], *gn = gw.seg[1];
        // the imaging form of the step kernel: g^n is formed and used in one pass
        const bool one_pass = tma && active_plan(h).has_image && h->claim_planes == 0 &&
                              h->fwd.inj[shape].npts <= kMaxImageSources;
        for (const RevAction &act : sched) {
            switch (act.kind) {
                case MMOD_REV_ADVANCE:
                    for (int n = act.a; n < act.b; ++n) MMOD_CK(h, fwd_step_in_place(n));
                    break;
                case MMOD_REV_SAVE:   // state of step b: u^{b-1} in u[b & 1], u^b in u[(b + 1) & 1]
                    MMOD_CK(h, save_state(h, act.a, h->u[act.b & 1], h->u[(act.b + 1) & 1], s));
                    break;
                case MMOD_REV_RESTORE:
                    if (act.a < 0) {
                        MMOD_CK(h, clear(h->u[0], vb));
                        MMOD_CK(h, clear(h->u[1], vb));
                    } else {
                        MMOD_CK(h, restore(act.a, h->u[act.b & 1], h->u[(act.b + 1) & 1]));
                    }
                    break;
                case MMOD_REV_REVERSE: {   // the adjoint step and its term, g^n from the working state
                    const int n = act.a;
                    if (one_pass) {
                        MMOD_CK(h, adj_step(n));
                        StepArgs ia = fa;
                        ia.n = n;
                        ia.pdl = h->pdl;
                        ia.image = 1;
                        ia.ucur = h->u[(n + 1) & 1];
                        ia.uprev = ia.uout = gw.gradc;
                        ia.c = gw.psi[(nt - 1 - n) & 1];
                        MMOD_CK(h, enqueue_step(h, ia, u_map[(n + 1) & 1], gw.gradc_map, tma, nullptr, s, &launches,
                                                &gw.psi_map[(nt - 1 - n) & 1].own));
                        break;
                    }
                    fa.n = n;
                    fa.ucur = h->u[(n + 1) & 1];
                    fa.uprev = h->u[n & 1];
                    fa.uout = unext;
                    fa.gout = gn;
                    const cudaError_t e = enqueue(fa, u_map[(n + 1) & 1], u_map[n & 1], nullptr);
                    fa.gout = nullptr;
                    MMOD_CK(h, e);
                    MMOD_CK(h, adj_step(n));
                    const float *g[1] = {gn};
                    MMOD_CK(h, image(n, g, 1));
                    break;
                }
                default:
                    return fail(h, MMOD_ERR_CUDA, "invalid checkpoint schedule");
            }
        }
    } else {
        const int nseg = nt > 0 ? nslot : 0;
        // With FP32 checkpoints a replay reproduces the first sweep bit for
        // bit, so the first sweep writes g^n of the last segment straight into
        // the segment buffer and that segment is neither saved nor replayed.
        // (A 16-bit checkpoint would start its replay from the rounded state.)
        // ---- sweep 1: forward with a checkpoint at the start of every segment
        if (through) {
            // no copies: the volumes that hold the state at step a0 are segment
            // sg's checkpoint (slot sg) and the segment steps on into the next
            // slot's; the last segment stays in its own slot.  (Saving and
            // restoring 20 checkpoints of 200^3 took 78 copies of 34 MB, 1 of
            // 42 ms.)  After a full segment u^{b0} is in volume (seglen - 1) & 1.
            MMOD_CK(h, clear(slot(0, 0).p, 2 * vb));
            for (int sg = 0; sg < nseg; ++sg) {
                const int a0 = sg * seglen, b0 = std::min(nt, a0 + seglen), i = sg == 0 ? 0 : seglen & 1;
                if (sg < nseg - 1)
                    MMOD_CK(h, fwd_range(a0, b0, slot(sg, i), slot(sg, 1 - i), slot(sg + 1, 0), slot(sg + 1, 1),
                                         [](int) -> float * { return nullptr; }));
                else
                    MMOD_CK(h, fwd_range(a0, b0, slot(sg, i), slot(sg, 1 - i), slot(sg, i), slot(sg, 1 - i),
                                         [&](int j) { return gw.seg[2 + j]; }));
            }
        } else {
            for (int sg = 0; sg < nseg; ++sg) {
                const int a0 = sg * seglen, b0 = std::min(nt, a0 + seglen);
                // at step a0: u^{a0-1} in u[a0 & 1], u^{a0} in u[(a0 + 1) & 1]
                MMOD_CK(h, save_state(h, sg, h->u[a0 & 1], h->u[(a0 + 1) & 1], s));
                for (int n = a0; n < b0; ++n) MMOD_CK(h, fwd_step_in_place(n));
            }
        }
        // ---- backward: replay each segment (g^n of its steps), then its
        // adjoint steps + imaging
        MMOD_CK(h, clear(gw.psi[0], vb));
        MMOD_CK(h, clear(gw.psi[1], vb));
        MMOD_CK(h, clear(gw.gradc, vb));
        for (int sg = nseg - 1; sg >= 0; --sg) {
            const int a0 = sg * seglen, b0 = std::min(nt, a0 + seglen);
            if (through && sg < nseg - 1) {
                const int i = sg == 0 ? 0 : seglen & 1;
                MMOD_CK(h, fwd_range(a0, b0, slot(sg, i), slot(sg, 1 - i), seg(0), seg(1),
                                     [&](int j) { return gw.seg[2 + j]; }));
            } else if (!through) {
                MMOD_CK(h, restore(sg, gw.seg[0], gw.seg[1]));
                for (int n = a0; n < b0; ++n) {   // seg[2 + n - a0] receives g^n
                    const int j = n - a0;
                    MMOD_CK(h, fwd_step_g(n, j & 1, (j + 1) & 1, gw.seg[2 + j]));
                }
            }
            MMOD_CK(h, backward_range(b0 - 1, a0, [&](int j) { return gw.seg[2 + j - a0]; }));
        }
    }
    h->ran = false;
    // ---- dJ/dv = 2 dt^2 v dJ/dc = 2 A / v (FP32)
    const size_t npts = (size_t)h->npts;
    const bool dev_out = is_device_ptr(grad_v);
    float *dst = grad_v;
    if (!dev_out) {
        if (!h->st_vol) MMOD_CK(h, cudaMalloc(&h->st_vol, sizeof(float) * npts));
        dst = h->st_vol;
    }
    MMOD_CK(h, launch_grad_to_velocity(gw.gradc, h->vel_copy, c.nx, c.ny, c.nz, h->nxp, dst, s));
    ++launches;
    if (!dev_out) {
        MMOD_CK(h, cudaMemcpyAsync(grad_v, dst, sizeof(float) * npts, cudaMemcpyDeviceToHost, s));
        MMOD_CK(h, cudaStreamSynchronize(s));
    }
    if (nadj && nt > 0) {
        if (tma) {   // the last adjoint step had no successor
            MMOD_CK(h, launch_gather(gw.psi[(nt - 1) & 1], h->adj.gather_off, nadj, h->st_adjg + (size_t)(nt - 1) * nadj, s));
            ++launches;
        }
        if (mmod_status st = adjoint_output(h, adj_src, s)) return st;
        ++launches;
    }
    h->last_launches = launches;
    return check_latched(h);
}

MMOD_API mmod_status mmod_gradient(mmod_handle *h, const float *wavelet, const float *resid, float *grad_v,
                                   int ckpt_count, int ckpt_dtype, mmod_stream stream) {
    return run_gradient(h, wavelet, resid, grad_v, nullptr, ckpt_count, ckpt_dtype, stream);
}

MMOD_API mmod_status mmod_gradient_adjoint(mmod_handle *h, const float *wavelet, const float *resid, float *grad_v,
                                           float *adj_src, int ckpt_count, int ckpt_dtype, mmod_stream stream) {
    if (!h) return MMOD_ERR_ARG;
    if (h->cfg.nsrc > 0 && h->cfg.nt > 0 && !adj_src) return fail(h, MMOD_ERR_ARG, "null adjoint source with nsrc > 0");
    return run_gradient(h, wavelet, resid, grad_v, adj_src, ckpt_count, ckpt_dtype, stream);
}

MMOD_API long long mmod_gradient_memory(const mmod_handle *h, int ckpt_count, int ckpt_dtype) {
    if (!h || ckpt_count < 1) return -1;
    if (ckpt_dtype != MMOD_CKPT_FP32 && ckpt_dtype != MMOD_CKPT_BF16 && ckpt_dtype != MMOD_CKPT_FP16 &&
        ckpt_dtype != MMOD_CKPT_BFP16)
        return -1;
    int nslot = 0, nwork = 0, seglen = 0;
    grad_layout(h, ckpt_count, ckpt_dtype, &nslot, &nwork, &seglen);
    const long long vb = 4LL * h->vol;
    const long long eb = ckpt_dtype == MMOD_CKPT_FP32 ? 4 : 2;
    return (long long)(nwork + 3) * vb + (long long)nslot * 2 * h->vol * eb +
           4LL * nslot * 2 * (long long)ckpt_scales(h, ckpt_dtype);
}

MMOD_API mmod_status mmod_dot(const float *a, const float *b, long long n, double *out, mmod_stream stream) {
    if (!a || !b || !out || n < 0) return MMOD_ERR_ARG;
    cudaStream_t s = (cudaStream_t)stream;
    double *d = nullptr;
    if (cudaMallocAsync(&d, sizeof(double), s) != cudaSuccess) return MMOD_ERR_OOM;
    cudaError_t e = cudaMemsetAsync(d, 0, sizeof(double), s);
    if (e == cudaSuccess) e = launch_dot(a, b, n, d, s);
    if (e == cudaSuccess) e = cudaMemcpyAsync(out, d, sizeof(double), cudaMemcpyDeviceToHost, s);
    cudaFreeAsync(d, s);
    if (e == cudaSuccess) e = cudaStreamSynchronize(s);
    return e == cudaSuccess ? MMOD_OK : MMOD_ERR_CUDA;
}
