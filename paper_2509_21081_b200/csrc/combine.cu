// Vector kernels of the path: merge of absorb chunk partials, the final LSE
// combine (Algorithm 1 line 8; Section 3.2 "CombineLSE") and layout helpers
// used once per prefix by the expansion step.
#include <algorithm>

#include "common.cuh"
#include "kernels.h"
#include "sm100.cuh"

namespace tmla {
namespace {

// One block of G x 128 threads per (b, h) (G = 1 for a few chunks, else 4): group g takes chunks g, g+G, ...;
// each thread owns 4 of the 512 latent columns.  The chunk weights are computed once into shared
// memory, so the partial rows are fetched by independent loads (many chunks of few tokens each are
// the rule at small batch sizes, where this kernel would otherwise be a chain of dependent loads).
constexpr int MERGE_MAX_CHUNKS = 1024;
__global__ void __launch_bounds__(512) merge_latent_kernel(const float* __restrict__ o_part,
                                                           const float* __restrict__ lse_part, int n_chunks,
                                                           int BH, __nv_bfloat16* __restrict__ o_lat,
                                                           float* __restrict__ lse) {
    sm100::pdl_trigger();
    sm100::pdl_wait();
    __shared__ float w_s[MERGE_MAX_CHUNKS];
    __shared__ float red[16];
    __shared__ float4 acc_s[3][128];
    const int bh = blockIdx.x, tid = threadIdx.x, grp = tid >> 7, col = tid & 127;
    const int nthr = blockDim.x, G = nthr >> 7, nwarp = nthr >> 5;
    // maximum of the chunk LSEs
    float m = -INFINITY;
    for (int c = tid; c < n_chunks; c += nthr) {
        const float l = lse_part[(int64_t)c * BH + bh];
        w_s[c] = l;
        m = fmaxf(m, l);
    }
    for (int o = 16; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
    if ((tid & 31) == 0) red[tid >> 5] = m;
    __syncthreads();
    m = red[0];
    for (int i = 1; i < nwarp; ++i) m = fmaxf(m, red[i]);
    __syncthreads();
    // weights (0 for an empty chunk, whose O slot was never written) and their sum
    float z = 0.f;
    for (int c = tid; c < n_chunks; c += nthr) {
        const float l = w_s[c];
        const float w = (l == -INFINITY) ? 0.f : __expf(l - m);
        w_s[c] = w;
        z += w;
    }
    for (int o = 16; o > 0; o >>= 1) z += __shfl_xor_sync(0xffffffffu, z, o);
    if ((tid & 31) == 0) red[tid >> 5] = z;
    __syncthreads();
    z = 0.f;
    for (int i = 0; i < nwarp; ++i) z += red[i];
    float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
    if (m != -INFINITY) {
        const float* src = o_part + (int64_t)bh * 512 + col * 4;
        // loads do not wait for the weights (eight in flight per thread); an empty chunk's slot was never
        // written, so its value is dropped by a select
#pragma unroll 8
        for (int c = grp; c < n_chunks; c += G) {
            const float4 v = *reinterpret_cast<const float4*>(src + (int64_t)c * BH * 512);
            const float w = w_s[c];
            const bool live = w != 0.f;
            acc.x += live ? w * v.x : 0.f; acc.y += live ? w * v.y : 0.f;
            acc.z += live ? w * v.z : 0.f; acc.w += live ? w * v.w : 0.f;
        }
    }
    if (grp > 0) acc_s[grp - 1][col] = acc;
    __syncthreads();
    if (grp == 0) {
        for (int g = 0; g < G - 1; ++g) {
            const float4 v = acc_s[g][col];
            acc.x += v.x; acc.y += v.y; acc.z += v.z; acc.w += v.w;
        }
        if (m != -INFINITY) {
            const float inv = 1.f / z;
            acc.x *= inv; acc.y *= inv; acc.z *= inv; acc.w *= inv;
        }
        uint2 pk = make_uint2(pack_bf16(acc.x, acc.y), pack_bf16(acc.z, acc.w));
        *reinterpret_cast<uint2*>(o_lat + (int64_t)bh * 512 + col * 4) = pk;
        if (col == 0) lse[bh] = (m == -INFINITY) ? -INFINITY : m + __logf(z);
    }
}

// Few chunks per request (the common case at larger batch sizes): no shared memory, four (b, h) rows
// per block of 512 threads, each thread owns 4 of a row's 512 latent columns and recomputes the (at most
// NC) chunk weights itself.  The LSEs and the partial rows are all requested before any of them is used
// (one memory round trip per thread); the slot of an empty chunk was never written, so its value is
// dropped by a select, not multiplied by a zero weight.
constexpr int MERGE_FEW = 16;
template <int NC>
__global__ void __launch_bounds__(512) merge_latent_few_kernel(const float* __restrict__ o_part,
                                                               const float* __restrict__ lse_part, int n_chunks,
                                                               int BH, __nv_bfloat16* __restrict__ o_lat,
                                                               float* __restrict__ lse) {
    sm100::pdl_trigger();
    sm100::pdl_wait();
    const int bh = blockIdx.x * 4 + (threadIdx.x >> 7), col = threadIdx.x & 127;
    if (bh >= BH) return;
    float l[NC];
    float4 v[NC];
#pragma unroll
    for (int c = 0; c < NC; ++c) l[c] = c < n_chunks ? lse_part[(int64_t)c * BH + bh] : -INFINITY;
#pragma unroll
    for (int c = 0; c < NC; ++c)
        v[c] = c < n_chunks ? *reinterpret_cast<const float4*>(o_part + ((int64_t)c * BH + bh) * 512 + col * 4)
                            : make_float4(0.f, 0.f, 0.f, 0.f);
    float m = -INFINITY;
#pragma unroll
    for (int c = 0; c < NC; ++c) m = fmaxf(m, l[c]);
    float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
    float z = 0.f;
    if (m != -INFINITY) {
#pragma unroll
        for (int c = 0; c < NC; ++c) {
            const bool live = l[c] != -INFINITY;
            const float w = live ? __expf(l[c] - m) : 0.f;
            acc.x += live ? w * v[c].x : 0.f; acc.y += live ? w * v[c].y : 0.f;
            acc.z += live ? w * v[c].z : 0.f; acc.w += live ? w * v[c].w : 0.f;
            z += w;
        }
        const float inv = 1.f / z;
        acc.x *= inv; acc.y *= inv; acc.z *= inv; acc.w *= inv;
    }
    uint2 pk = make_uint2(pack_bf16(acc.x, acc.y), pack_bf16(acc.z, acc.w));
    *reinterpret_cast<uint2*>(o_lat + (int64_t)bh * 512 + col * 4) = pk;
    if (col == 0) lse[bh] = (m == -INFINITY) ? -INFINITY : m + __logf(z);
}

// Absorb-only step of few (request, head) rows: merge of the chunk partials, output projection O_A W_UV^T (Algorithm 1
// line 7) and the final rounding in one launch.  One block per row, 512 threads: group g of 128 threads takes the chunks g,
// g + 4, ...; the merged latent row stays in fp32 in shared memory; every warp then forms 8 of the 128 outputs as dot
// products over 512 (16 elements per lane, butterfly sum).  What bounds it is latency, so everything is requested at
// once: the warp's 8 KB of weights (64 registers per thread) before the wait for the preceding kernel, which does not write
// them, then the log-sum-exps and the first eight partial rows of the group, before the merge weights are known.
// Each block re-reads its head's weights, so this is for one wave of rows (the rule and both sides measured: api.cu).
constexpr int MP_BATCH = 8;
__device__ __forceinline__ uint4 ldg_nc(const void* p) {   // volatile: stays where it is written
    uint4 v;
    asm volatile("ld.global.nc.v4.u32 {%0, %1, %2, %3}, [%4];\n" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "l"(p));
    return v;
}
__device__ __forceinline__ float4 ldg_f4(const float* p) {
    float4 v;
    asm volatile("ld.global.v4.f32 {%0, %1, %2, %3}, [%4];\n" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "l"(p) : "memory");
    return v;
}
__global__ void __launch_bounds__(512, 1) merge_project_kernel(const float* __restrict__ o_part,
                                                               const float* __restrict__ lse_part, int n_chunks, int B,
                                                               int H, const __nv_bfloat16* __restrict__ w_uv,
                                                               void* __restrict__ out, float* __restrict__ lse_out,
                                                               int out_fp32) {
    __shared__ float w_s[MERGE_MAX_CHUNKS];
    __shared__ float red[16];
    __shared__ float4 acc_s[4][128];
    const int h = blockIdx.x, b = blockIdx.y, BH = B * H, bh = b * H + h;
    const int tid = threadIdx.x, grp = tid >> 7, col = tid & 127, warp = tid >> 5, lane = tid & 31;
    sm100::pdl_trigger();
    uint4 wv[8][2];   // this warp's 8 weight rows, 16 consecutive elements per lane and row
    {
        const __nv_bfloat16* wrow = w_uv + ((int64_t)h * 128 + warp * 8) * 512 + lane * 16;
#pragma unroll
        for (int r = 0; r < 8; ++r) {
            wv[r][0] = ldg_nc(wrow + r * 512);
            wv[r][1] = ldg_nc(wrow + r * 512 + 8);
        }
    }
    sm100::pdl_wait();
    const float* src = o_part + (int64_t)bh * 512 + col * 4;
    const int64_t step = (int64_t)BH * 512;
    const float4 zero = make_float4(0.f, 0.f, 0.f, 0.f);
    float l0 = tid < n_chunks ? lse_part[(int64_t)tid * BH + bh] : -INFINITY;
    float4 v[MP_BATCH];
#pragma unroll
    for (int i = 0; i < MP_BATCH; ++i) {
        const int c = grp + 4 * i;
        v[i] = c < n_chunks ? ldg_f4(src + c * step) : zero;   // (an empty chunk's slot was never written: dropped below)
    }
    float m = l0;
    w_s[tid] = l0;
    for (int c = tid + 512; c < n_chunks; c += 512) {
        const float l = lse_part[(int64_t)c * BH + bh];
        w_s[c] = l;
        m = fmaxf(m, l);
    }
    for (int o = 16; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
    if (lane == 0) red[warp] = m;
    __syncthreads();
    m = red[0];
    for (int i = 1; i < 16; ++i) m = fmaxf(m, red[i]);
    __syncthreads();
    float z = 0.f;
    for (int c = tid; c < n_chunks; c += 512) {
        const float l = w_s[c];
        const float w = (l == -INFINITY) ? 0.f : __expf(l - m);
        w_s[c] = w;
        z += w;
    }
    for (int o = 16; o > 0; o >>= 1) z += __shfl_xor_sync(0xffffffffu, z, o);
    if (lane == 0) red[warp] = z;
    __syncthreads();
    z = 0.f;
    for (int i = 0; i < 16; ++i) z += red[i];
    float4 acc = zero;
    if (m != -INFINITY) {
        for (int c0 = grp; c0 < n_chunks; c0 += 4 * MP_BATCH) {
#pragma unroll
            for (int i = 0; i < MP_BATCH; ++i) {
                const int c = c0 + 4 * i;
                const float w = c < n_chunks ? w_s[c] : 0.f;
                const bool live = w != 0.f;
                acc.x += live ? w * v[i].x : 0.f; acc.y += live ? w * v[i].y : 0.f;
                acc.z += live ? w * v[i].z : 0.f; acc.w += live ? w * v[i].w : 0.f;
            }
#pragma unroll
            for (int i = 0; i < MP_BATCH; ++i) {
                const int c = c0 + 4 * (MP_BATCH + i);
                if (c < n_chunks) v[i] = ldg_f4(src + c * step);
            }
        }
    }
    acc_s[grp][col] = acc;
    __syncthreads();
    // the merged, normalised latent row: this lane's 16 elements (float4 columns 4 lane .. 4 lane + 3)
    const float inv = (m != -INFINITY) ? 1.f / z : 0.f;
    float o[16];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        float4 t = acc_s[0][lane * 4 + q];
#pragma unroll
        for (int g = 1; g < 4; ++g) {
            const float4 u = acc_s[g][lane * 4 + q];
            t.x += u.x; t.y += u.y; t.z += u.z; t.w += u.w;
        }
        o[4 * q] = t.x * inv; o[4 * q + 1] = t.y * inv; o[4 * q + 2] = t.z * inv; o[4 * q + 3] = t.w * inv;
    }
    float res = 0.f;   // lane r < 8 keeps output row warp * 8 + r
#pragma unroll
    for (int r = 0; r < 8; ++r) {
        const uint32_t wr[8] = {wv[r][0].x, wv[r][0].y, wv[r][0].z, wv[r][0].w, wv[r][1].x, wv[r][1].y, wv[r][1].z, wv[r][1].w};
        float d = 0.f;
#pragma unroll
        for (int e = 0; e < 8; ++e) {
            const __nv_bfloat162 p2 = *reinterpret_cast<const __nv_bfloat162*>(&wr[e]);
            d += __low2float(p2) * o[2 * e] + __high2float(p2) * o[2 * e + 1];
        }
        for (int s2 = 16; s2 > 0; s2 >>= 1) d += __shfl_xor_sync(0xffffffffu, d, s2);
        if (lane == r) res = d;
    }
    if (lane < 8) {
        const int64_t idx = (int64_t)bh * 128 + warp * 8 + lane;
        if (out_fp32) reinterpret_cast<float*>(out)[idx] = res;
        else reinterpret_cast<__nv_bfloat16*>(out)[idx] = __float2bfloat16_rn(res);
    }
    if (tid == 0 && lse_out != nullptr) lse_out[bh] = (m == -INFINITY) ? -INFINITY : m + __logf(z);
}

// One warp per (b, h); each lane owns 4 of the 128 output columns.
__global__ void __launch_bounds__(256) combine_kernel(const float* __restrict__ o_naive,
                                                      const float* __restrict__ lse_naive, int n_naive,
                                                      const float* __restrict__ o_abs,
                                                      const float* __restrict__ lse_abs, int BH,
                                                      void* __restrict__ out, float* __restrict__ lse_out, int out_fp32) {
    sm100::pdl_trigger();
    sm100::pdl_wait();
    const int bh = blockIdx.x * 8 + (threadIdx.x >> 5);
    const int lane = threadIdx.x & 31;
    if (bh >= BH) return;
    float m = -INFINITY;
    for (int i = 0; i < n_naive; ++i) m = fmaxf(m, lse_naive[(int64_t)i * BH + bh]);
    float la = -INFINITY;
    if (o_abs != nullptr) {
        la = lse_abs[bh];
        m = fmaxf(m, la);
    }
    float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
    float z = 0.f;
    if (m != -INFINITY) {
        for (int i = 0; i < n_naive; ++i) {
            float l = lse_naive[(int64_t)i * BH + bh];
            if (l == -INFINITY) continue;
            float w = __expf(l - m);
            float4 v = *reinterpret_cast<const float4*>(o_naive + ((int64_t)i * BH + bh) * 128 + lane * 4);
            acc.x += w * v.x; acc.y += w * v.y; acc.z += w * v.z; acc.w += w * v.w;
            z += w;
        }
        if (la != -INFINITY) {
            float w = __expf(la - m);
            float4 v = *reinterpret_cast<const float4*>(o_abs + (int64_t)bh * 128 + lane * 4);
            acc.x += w * v.x; acc.y += w * v.y; acc.z += w * v.z; acc.w += w * v.w;
            z += w;
        }
        float inv = 1.f / z;
        acc.x *= inv; acc.y *= inv; acc.z *= inv; acc.w *= inv;
    }
    if (out_fp32) {
        *reinterpret_cast<float4*>(reinterpret_cast<float*>(out) + (int64_t)bh * 128 + lane * 4) = acc;
    } else {
        uint2 pk = make_uint2(pack_bf16(acc.x, acc.y), pack_bf16(acc.z, acc.w));
        *reinterpret_cast<uint2*>(reinterpret_cast<__nv_bfloat16*>(out) + (int64_t)bh * 128 + lane * 4) = pk;
    }
    if (lse_out != nullptr && lane == 0) lse_out[bh] = (m == -INFINITY) ? -INFINITY : m + __logf(z);
}

// What a prepared prefix keeps besides the expansion (see launch_prepare_layout), one launch of three kinds of blocks.  Bound
// by memory: 16.8 MB of weights each way at 128 heads and 2.3 KB per token.  The transpose moves 16-byte pieces on both
// sides of a 64 x 64 tile (rows of 33 words, so that the 2-byte column reads spread over the banks).
struct LayoutParams {
    const __nv_bfloat16* w; __nv_bfloat16* w_t; int n_w;                         // n_w = H * 16 tiles
    const __nv_bfloat16* ckv; int64_t ld_ckv; uint4* ckv_out; int n_ckv;         // n_*: blocks of each kind
    const __nv_bfloat16* kpe; int64_t ld_kpe; uint4* kpe_out;
    int64_t L, Lp;
    int* status;
};
__global__ void __launch_bounds__(256) prepare_layout_kernel(LayoutParams p) {
    sm100::pdl_wait();   // (must not trigger early: later kernels read what is written here before their own wait, see kernels.h)
    const int tid = threadIdx.x, blk = blockIdx.x;
    if (blk < p.n_w) {
        __shared__ uint32_t tile[64 * 33];
        const int h = blk >> 4, d0 = (blk & 1) * 64, l0 = ((blk >> 1) & 7) * 64;
        const __nv_bfloat16* in = p.w + (int64_t)h * 65536 + (int64_t)d0 * 512 + l0;
        __nv_bfloat16* out = p.w_t + (int64_t)h * 65536 + (int64_t)l0 * 128 + d0;
#pragma unroll
        for (int i = tid; i < 512; i += 256) {
            const uint4 v = *reinterpret_cast<const uint4*>(in + (i >> 3) * 512 + (i & 7) * 8);
            uint32_t* t = tile + (i >> 3) * 33 + (i & 7) * 4;
            t[0] = v.x; t[1] = v.y; t[2] = v.z; t[3] = v.w;
        }
        __syncthreads();
#pragma unroll
        for (int i = tid; i < 512; i += 256) {   // row l of the output tile, dims 8 j .. 8 j + 7
            const int l = i >> 3, j = i & 7, sh = (l & 1) * 16;
            const uint32_t* t = tile + 8 * j * 33 + (l >> 1);
            uint32_t w[4];
#pragma unroll
            for (int k = 0; k < 4; ++k) w[k] = ((t[2 * k * 33] >> sh) & 0xffffu) | ((t[(2 * k + 1) * 33] >> sh) << 16);
            *reinterpret_cast<uint4*>(out + l * 128 + j * 8) = make_uint4(w[0], w[1], w[2], w[3]);
        }
        if (blk == 0 && tid < 64) p.status[tid] = 0;
        return;
    }
    const uint4 zero = make_uint4(0, 0, 0, 0);
    if (blk < p.n_w + p.n_ckv) {                 // 4 latent rows of 64 pieces per pass
        for (int64_t i = (int64_t)(blk - p.n_w) * 256 + tid; i < p.Lp * 64; i += (int64_t)p.n_ckv * 256)
            p.ckv_out[i] = (i >> 6) < p.L ? *reinterpret_cast<const uint4*>(p.ckv + (i >> 6) * p.ld_ckv + (i & 63) * 8) : zero;
    } else {
        const int n = gridDim.x - p.n_w - p.n_ckv;
        for (int64_t i = (int64_t)(blk - p.n_w - p.n_ckv) * 256 + tid; i < p.Lp * 8; i += (int64_t)n * 256)
            p.kpe_out[i] = (i >> 3) < p.L ? *reinterpret_cast<const uint4*>(p.kpe + (i >> 3) * p.ld_kpe + (i & 7) * 8) : zero;
    }
}

// Copies of a step whose tensors live in pinned host memory: up to four arrays, each a whole number of 4-byte words, by
// 16-byte pieces where both ends allow it.  Bound by the host link; eight independent pieces per thread keep it busy.
// Steps on other streams run beside it.  So a block takes no more registers than the attention kernels leave free on an SM
// (384 threads with 128 each: 64 for 256 threads), the launch has the highest priority (behind other steps' waiting CTAs
// a copy took as long as they did), and the kernel behind it is not triggered early, whose CTAs would hold their SMs for
// the length of the transfer.
struct HostCopies {
    const void* src[4];
    void* dst[4];
    int64_t bytes[4];
    int first_block[5];   // blocks [first_block[i], first_block[i + 1]) copy array i
};
__global__ void __launch_bounds__(256, 4) host_copy_kernel(const __grid_constant__ HostCopies c) {
    sm100::pdl_wait();
    int i = 0;
    while (i < 3 && (int)blockIdx.x >= c.first_block[i + 1]) ++i;
    const int n_blk = c.first_block[i + 1] - c.first_block[i];
    const int64_t t = (int64_t)(blockIdx.x - c.first_block[i]) * 256 + threadIdx.x, step = (int64_t)n_blk * 256;
    const bool vec = ((reinterpret_cast<uintptr_t>(c.src[i]) | reinterpret_cast<uintptr_t>(c.dst[i])) & 15) == 0;
    int64_t done = 0;   // bytes copied as 16-byte pieces
    if (vec) {
        const int64_t n = c.bytes[i] / 16;
        const char* src = reinterpret_cast<const char*>(c.src[i]);
        uint4* dst = reinterpret_cast<uint4*>(c.dst[i]);
        for (int64_t k0 = t; k0 < n; k0 += 8 * step) {
            uint4 v[8];
#pragma unroll
            for (int u = 0; u < 8; ++u)
                if (k0 + u * step < n)
                    asm volatile("ld.volatile.global.v4.u32 {%0, %1, %2, %3}, [%4];\n" : "=r"(v[u].x), "=r"(v[u].y), "=r"(v[u].z), "=r"(v[u].w) : "l"(src + (k0 + u * step) * 16) : "memory");
#pragma unroll
            for (int u = 0; u < 8; ++u)
                if (k0 + u * step < n) dst[k0 + u * step] = v[u];
        }
        done = n * 16;
    }
    const int64_t words = c.bytes[i] / 4;
    for (int64_t k = done / 4 + t; k < words; k += step)
        reinterpret_cast<uint32_t*>(c.dst[i])[k] = *(reinterpret_cast<const volatile uint32_t*>(c.src[i]) + k);
}

// Longest-first launch order for ragged suffixes: perm[] = request indices sorted by descending
// suffix length (ties by index, so the order is deterministic).  One block, bitonic sort in
// shared memory of up to 4096 keys.
__global__ void __launch_bounds__(1024) order_by_length_kernel(const int32_t* __restrict__ seq_lens, int B,
                                                               int32_t* __restrict__ perm) {
    __shared__ unsigned long long keys[4096];
    block_order_by_length(seq_lens, B, perm, keys);
}

// -inf into n_slots segments of `count` floats, `stride` floats apart (LSE of partial slots no kernel fills).
__global__ void __launch_bounds__(256) fill_neg_inf_kernel(float* __restrict__ dst, int n_slots, int64_t stride, int64_t count) {
    const int64_t total = (int64_t)n_slots * count;
    for (int64_t i = (int64_t)blockIdx.x * 256 + threadIdx.x; i < total; i += (int64_t)gridDim.x * 256)
        dst[(i / count) * stride + i % count] = -INFINITY;
}

// Row expansion for S_q query tokens per request (Table 1's S_q; causal among the new tokens):
// row b * S_q + j gets request b's page-table row and the suffix length minus the S_q - 1 - j later tokens.
__global__ void __launch_bounds__(256) expand_query_rows_kernel(const int32_t* __restrict__ block_table,
                                                                const int32_t* __restrict__ seq_lens, int B,
                                                                int max_pages, int S_q,
                                                                int32_t* __restrict__ bt_rows,
                                                                int32_t* __restrict__ len_rows) {
    const int64_t n_bt = (int64_t)B * S_q * max_pages;
    for (int64_t i = (int64_t)blockIdx.x * 256 + threadIdx.x; i < n_bt; i += (int64_t)gridDim.x * 256) {
        const int64_t row = i / max_pages;
        bt_rows[i] = block_table[(row / S_q) * max_pages + i % max_pages];
    }
    for (int i = blockIdx.x * 256 + threadIdx.x; i < B * S_q; i += gridDim.x * 256)
        len_rows[i] = max(seq_lens[i / S_q] - (S_q - 1 - i % S_q), 0);
}

}  // namespace

// Test kernel for the bounded wait of the tcgen05 kernels: a barrier on which nothing arrives, the same
// mbar_wait with a short deadline, the same report through the status word, a normal return.
static __global__ void wait_expiry_selftest_kernel(int* status, long long deadline_cycles, int code) {
    __shared__ uint64_t bar;
    __shared__ int abort_flag;
    if (threadIdx.x == 0) {
        sm100::mbar_init(&bar, 1);
        abort_flag = 0;
        sm100::fence_mbar_init();
    }
    __syncthreads();
    const bool ok = sm100::mbar_wait(&bar, 0, &abort_flag, deadline_cycles);   // nobody arrives: runs out
    __syncthreads();
    if (threadIdx.x == 0 && (!ok || abort_flag) && status) atomicOr(status, code);
}
cudaError_t launch_wait_expiry_selftest(int* status, long long deadline_cycles, int code, cudaStream_t s) {
    wait_expiry_selftest_kernel<<<1, 32, 0, s>>>(status, deadline_cycles, code);
    return cudaGetLastError();
}

cudaError_t launch_order_by_length(const int32_t* seq_lens, int B, int32_t* perm, cudaStream_t s) {
    if (B <= 0 || B > 4096) return cudaErrorInvalidValue;
    order_by_length_kernel<<<1, 1024, 0, s>>>(seq_lens, B, perm);
    return cudaGetLastError();
}

cudaError_t launch_fill_neg_inf(float* dst, int n_slots, int64_t stride, int64_t count, cudaStream_t s) {
    if (n_slots <= 0 || count <= 0) return cudaSuccess;
    const int64_t total = (int64_t)n_slots * count;
    fill_neg_inf_kernel<<<(unsigned)std::min<int64_t>((total + 255) / 256, 1184), 256, 0, s>>>(dst, n_slots, stride, count);
    return cudaGetLastError();
}

cudaError_t launch_expand_query_rows(const int32_t* block_table, const int32_t* seq_lens, int B, int max_pages, int S_q,
                                     int32_t* bt_rows, int32_t* len_rows, cudaStream_t s) {
    if (B <= 0 || S_q <= 0) return cudaSuccess;
    const int64_t n = std::max<int64_t>((int64_t)B * S_q * max_pages, (int64_t)B * S_q);
    const unsigned blocks = (unsigned)std::min<int64_t>((n + 255) / 256, 1184);
    expand_query_rows_kernel<<<blocks, 256, 0, s>>>(block_table, seq_lens, B, max_pages, S_q, bt_rows, len_rows);
    return cudaGetLastError();
}

cudaError_t launch_merge_project(const float* o_part, const float* lse_part, int n_chunks, int B, int H, const void* w_uv,
                                 void* out, float* lse_out, bool out_fp32, cudaStream_t s) {
    if (B * H <= 0) return cudaSuccess;
    if (n_chunks > MERGE_MAX_CHUNKS) return cudaErrorInvalidValue;
    return launch_pdl(merge_project_kernel, dim3(H, B), dim3(512), 0, s, o_part, lse_part, n_chunks, B, H,
                      reinterpret_cast<const __nv_bfloat16*>(w_uv), out, lse_out, out_fp32 ? 1 : 0);
}

cudaError_t launch_merge_latent(const float* o_part, const float* lse_part, int n_chunks, int B, int H,
                                void* o_lat_bf16, float* lse, cudaStream_t s) {
    if (B * H <= 0) return cudaSuccess;
    if (n_chunks > MERGE_MAX_CHUNKS) return cudaErrorInvalidValue;
    if (n_chunks <= MERGE_FEW) {
        const dim3 grid((B * H + 3) / 4);
        __nv_bfloat16* o = reinterpret_cast<__nv_bfloat16*>(o_lat_bf16);
        if (n_chunks <= 2) return launch_pdl(merge_latent_few_kernel<2>, grid, dim3(512), 0, s, o_part, lse_part, n_chunks, B * H, o, lse);
        if (n_chunks <= 4) return launch_pdl(merge_latent_few_kernel<4>, grid, dim3(512), 0, s, o_part, lse_part, n_chunks, B * H, o, lse);
        if (n_chunks <= 8) return launch_pdl(merge_latent_few_kernel<8>, grid, dim3(512), 0, s, o_part, lse_part, n_chunks, B * H, o, lse);
        return launch_pdl(merge_latent_few_kernel<MERGE_FEW>, grid, dim3(512), 0, s, o_part, lse_part, n_chunks, B * H, o, lse);
    } else {
        return launch_pdl(merge_latent_kernel, dim3(B * H), dim3(512), 0, s, o_part, lse_part, n_chunks, B * H,
                          reinterpret_cast<__nv_bfloat16*>(o_lat_bf16), lse);
    }
    return cudaGetLastError();
}

cudaError_t launch_combine(const float* o_naive, const float* lse_naive, int n_naive, const float* o_abs,
                           const float* lse_abs, int B, int H, void* out, float* lse_out, cudaStream_t s, bool out_fp32) {
    int BH = B * H;
    if (BH <= 0) return cudaSuccess;
    return launch_pdl(combine_kernel, dim3((BH + 7) / 8), dim3(256), 0, s, o_naive, lse_naive, n_naive, o_abs, lse_abs, BH,
                      out, lse_out, out_fp32 ? 1 : 0);
}

cudaError_t launch_host_copy(const void* const* src, void* const* dst, const int64_t* bytes, int n, cudaStream_t s) {
    HostCopies c{};
    int blocks = 0;
    for (int i = 0; i < 4; ++i) {
        c.first_block[i] = blocks;
        if (i >= n || bytes[i] <= 0) continue;
        if (bytes[i] % 4) return cudaErrorInvalidValue;
        c.src[i] = src[i];
        c.dst[i] = dst[i];
        c.bytes[i] = bytes[i];
        blocks += (int)std::min<int64_t>((bytes[i] + 32767) / 32768, 64);   // 32 KB per block and pass
    }
    c.first_block[4] = blocks;
    if (blocks == 0) return cudaSuccess;
    int lowest = 0, highest = 0;
    const cudaError_t e = cudaDeviceGetStreamPriorityRange(&lowest, &highest);
    return e != cudaSuccess ? e : launch_pdl_at(highest, host_copy_kernel, dim3(blocks), dim3(256), 0, s, c);
}

cudaError_t launch_prepare_layout(const void* w_uk, void* w_uk_t, int H, const void* ckv, int64_t ld_ckv, void* ckv_out, const void* kpe,
                                  int64_t ld_kpe, void* kpe_out, int64_t L, int64_t Lp, int* status, cudaStream_t s) {
    if (H <= 0) return cudaSuccess;
    LayoutParams p{};
    p.w = reinterpret_cast<const __nv_bfloat16*>(w_uk);
    p.w_t = reinterpret_cast<__nv_bfloat16*>(w_uk_t);
    p.n_w = H * 16;
    p.ckv = reinterpret_cast<const __nv_bfloat16*>(ckv);
    p.ld_ckv = ld_ckv;
    p.ckv_out = reinterpret_cast<uint4*>(ckv_out);
    p.n_ckv = (int)std::min<int64_t>((Lp * 64 + 1023) / 1024, 2048);   // (four pieces per thread up to 32768 rows)
    p.kpe = reinterpret_cast<const __nv_bfloat16*>(kpe);
    p.ld_kpe = ld_kpe;
    p.kpe_out = reinterpret_cast<uint4*>(kpe_out);
    p.L = L;
    p.Lp = Lp;
    p.status = status;
    const int n_kpe = (int)std::min<int64_t>((Lp * 8 + 1023) / 1024, 256);
    return launch_pdl(prepare_layout_kernel, dim3(p.n_w + p.n_ckv + n_kpe), dim3(256), 0, s, p);
}

}  // namespace tmla
