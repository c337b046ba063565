// Expansion of a shared prefix (Section 3.1 "Prefill") on tcgen05 / TMEM / TMA: per head h
//     K_nope[h] = ckv [L, 512] * W_UK[h]^T,   V[h] = ckv * W_UV[h]^T   (stored transposed, see below)
// in one pass over the latent tokens.
//
// Work unit = (128 tokens, head), the accumulator [128 tokens][128 dims of K | 128 dims of V].  The units, heads fastest,
// are cut into one contiguous range per SM: a CTA keeps its 128 latent rows (128 KB) in shared memory while it walks
// through the heads, whose weights (256 KB per head, all heads in L2) stream through a ring of three 32 KB stages.
// Bound: the weights' way from L2, 64 bytes per clock and SM at the full tensor rate (a [128 x 128] product of a
// streamed by a streamed operand needs 128).  Two accumulators (all 512 tensor-memory columns): the epilogue of a unit
// runs under the next unit's products.
// Measured (B200, 4864 tokens x 128 heads, both tensors): 125 us = 1.3 PFLOP/s, 93 us without the stores; as two
// products with [128 x 128] tiles, every tile's operands read anew and its epilogue exposed: 346 us.
//
// Output layouts: K_nope [H, L/64, 2 slabs, 64 tokens, 64 dims], V^T [H, L/64, 128 dims, 64 tokens].  An epilogue thread
// holds one token: its 64 dims of a K slab are 128 contiguous bytes, written as four whole 32-byte sectors (with 16-byte
// stores, half sectors, the kernel took 145 us); for V^T the 32 lanes of a warp write 32 consecutive tokens of two dims
// (8-byte stores of four tokens instead of two made no difference).
//
// Warp roles (384 threads): warp 0 = producer of the weight ring, warp 1 = MMA issuer and TMEM owner, warp 2 = producer of
// the latent rows, warps 4-7 = epilogue of K, warps 8-11 = epilogue of V (thread = one token).
#include <algorithm>

#include "kernels.h"
#include "sm100.cuh"

namespace tmla {
namespace {

using namespace sm100;

constexpr int BK = 64, KB = 512 / BK, STAGES = 3;
constexpr int SLAB_BYTES = 128 * 128;             // [128 rows][64 bf16], swizzled
constexpr int C_BYTES = KB * SLAB_BYTES;          // the latent rows
constexpr int STAGE_BYTES = 2 * SLAB_BYTES;       // 128 dims of W_UK, 128 dims of W_UV
constexpr int SMEM_BYTES = C_BYTES + STAGES * STAGE_BYTES + 1024;

struct ExpandParams {
    __nv_bfloat16* k;      // or null: that half is not computed
    __nv_bfloat16* v_t;
    int H, n_blocks;       // n_blocks: 64-token blocks (even)
    int per, rem;          // units per CTA: CTAs [0, rem) take per + 1
    int* status;
};

// PARTS: 1 = K only, 2 = V only, 3 = both (the 8-bit option encodes one tensor before it expands the other)
template <int PARTS>
__global__ void __launch_bounds__(384, 1)
expand_sm100_kernel(const __grid_constant__ CUtensorMap tm_c, const __grid_constant__ CUtensorMap tm_uk,
                    const __grid_constant__ CUtensorMap tm_uv, ExpandParams p) {
    constexpr int N = PARTS == 3 ? 256 : 128;
    constexpr uint32_t FILL = PARTS == 3 ? STAGE_BYTES : SLAB_BYTES;
    extern __shared__ uint8_t smem_raw[];
    uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    uint8_t* sC = smem;
    uint8_t* sW = smem + C_BYTES;
    __shared__ uint64_t w_full[STAGES], w_empty[STAGES], c_full[KB], c_free, acc_full[2], acc_empty[2];
    __shared__ uint32_t tmem_holder;
    __shared__ int abort_word;
    volatile int* abort_flag = &abort_word;

    const int warp = warp_index_uniform(), lane = threadIdx.x & 31;
    // (the trigger must stay behind the wait: what may start now is behind the kernel that wrote w_uk_t and the latent rows, so
    // that a step may read them before its own wait, see kernels.h)
    pdl_wait();
    pdl_trigger();
    const int c = blockIdx.x;
    const int u0 = c * p.per + min(c, p.rem), u1 = u0 + p.per + (c < p.rem ? 1 : 0);

    const uint32_t ld = elect_one() ? 1u : 0u;
    if (warp == 0) {
        if (lane < STAGES) {
            mbar_init(&w_full[lane], 1);
            mbar_init(&w_empty[lane], 1);
        } else if (lane >= 8 && lane < 8 + KB) {
            mbar_init(&c_full[lane - 8], 1);
        } else if (lane >= 16 && lane < 18) {
            mbar_init(&acc_full[lane - 16], 1);
            mbar_init(&acc_empty[lane - 16], PARTS == 3 ? 8 : 4);
        } else if (lane == 18) {
            mbar_init(&c_free, 1);
            *abort_flag = 0;
        }
        fence_mbar_init();
    }
    if (warp == 2 && lane < 3) prefetch_tmap(lane == 0 ? &tm_c : lane == 1 ? &tm_uk : &tm_uv);
    if (warp == 1) tmem_alloc(&tmem_holder, 512);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem_base = __shfl_sync(0xffffffffu, tmem_holder, 0);

    int w_issued = 0, c_issued = 0;   // producer warps: stages and row tiles issued (upper bounds), for the abort path
    if (warp == 0) {
        bool ok = true;
        for (int u = u0; u < u1 && ok; ++u) {
            const int h = u % p.H;
            for (int kb = 0; kb < KB && ok; ++kb) {
                const int s = w_issued % STAGES;
                ok = mbar_wait_warp(&w_empty[s], ((w_issued / STAGES) & 1) ^ 1, abort_flag);
                if (!ok) break;
                uint8_t* dst = sW + s * STAGE_BYTES;
                mbar_arrive_expect_tx_if(ld, &w_full[s], FILL);
                if (PARTS & 1) tma_load_3d_if(ld, dst, &tm_uk, &w_full[s], kb * BK, 0, h);
                if (PARTS & 2) tma_load_3d_if(ld, dst + (PARTS == 3 ? SLAB_BYTES : 0), &tm_uv, &w_full[s], kb * BK, 0, h);
                ++w_issued;
            }
        }
    } else if (warp == 2) {
        for (int t = u0 / p.H; t * p.H < u1; ++t) {
            if (c_issued > 0 && !mbar_wait_warp(&c_free, (c_issued - 1) & 1, abort_flag)) break;   // the previous rows' products
            ++c_issued;
#pragma unroll 1
            for (int kb = 0; kb < KB; ++kb) {
                mbar_arrive_expect_tx_if(ld, &c_full[kb], SLAB_BYTES);
                tma_load_2d_if(ld, sC + kb * SLAB_BYTES, &tm_c, &c_full[kb], kb * BK, t * 128);
            }
        }
    } else if (warp == 1) {
        constexpr uint32_t idesc = idesc_bf16(128, N, false, false);
        bool ok = true;
        int pos = 0, tile = -1;
        for (int u = u0; u < u1 && ok; ++u) {
            const int i = u - u0, buf = i & 1;
            const bool new_rows = i == 0 || u % p.H == 0;
            tile += new_rows ? 1 : 0;
            ok = mbar_wait_warp(&acc_empty[buf], ((i >> 1) & 1) ^ 1, abort_flag);
            for (int kb = 0; kb < KB && ok; ++kb, ++pos) {
                const int s = pos % STAGES;
                ok = new_rows ? mbar_wait2_warp(&c_full[kb], tile & 1, &w_full[s], (pos / STAGES) & 1, abort_flag)
                              : mbar_wait_warp(&w_full[s], (pos / STAGES) & 1, abort_flag);
                if (!ok) break;
                tc_fence_after();
                const uint64_t da = smem_desc_k_sw128(smem_u32(sC + kb * SLAB_BYTES)), db = smem_desc_k_sw128(smem_u32(sW + s * STAGE_BYTES));
#pragma unroll
                for (int k = 0; k < BK / 16; ++k) umma_ss_if(ld, tmem_base + buf * 256, da + 2 * k, db + 2 * k, idesc, (kb | k) != 0);
                umma_commit_if(ld, &w_empty[s]);
            }
            if (!ok) break;
            umma_commit_if(ld, &acc_full[buf]);
            if ((u + 1) % p.H == 0) umma_commit_if(ld, &c_free);   // last head of these rows
        }
    } else if (warp >= 4) {
        const bool is_v = warp >= 8;
        const int lg = (warp & 3) * 32, r = lg + lane;
        const uint32_t col0 = (PARTS == 3 && is_v) ? 128u : 0u;
        bool ok = (PARTS >> (is_v ? 1 : 0)) & 1;                    // (a half that is not computed has no work)
        for (int u = u0; u < u1 && ok; ++u) {
            const int i = u - u0, buf = i & 1, h = u % p.H, blk = u / p.H * 2 + (r >> 6);
            ok = __all_sync(0xffffffffu, mbar_wait(&acc_full[buf], (i >> 1) & 1, abort_flag));
            if (!ok) break;
            tc_fence_after();
            const uint32_t src = tmem_base + ((uint32_t)lg << 16) + buf * 256 + col0;
            const int64_t out0 = ((int64_t)h * p.n_blocks + blk) * 8192;
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                uint32_t t[32];
                tmem_ld32(src + q * 32, t);
                tmem_ld_wait();
                if (q == 3) {
                    tc_fence_before();
                    __syncwarp();
                    if (lane == 0) mbar_arrive(&acc_empty[buf]);
                }
                if (!is_v) {
                    __nv_bfloat16* dst = p.k + out0 + (q >> 1) * 4096 + (r & 63) * 64 + (q & 1) * 32;
#pragma unroll
                    for (int j = 0; j < 2; ++j) {
                        uint32_t w[8];
#pragma unroll
                        for (int e = 0; e < 8; ++e) w[e] = pack_bf16(__uint_as_float(t[j * 16 + 2 * e]), __uint_as_float(t[j * 16 + 2 * e + 1]));
                        asm volatile("st.global.v8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};\n" ::"l"(dst + j * 16), "r"(w[0]),
                                     "r"(w[1]), "r"(w[2]), "r"(w[3]), "r"(w[4]), "r"(w[5]), "r"(w[6]), "r"(w[7]) : "memory");
                    }
                } else {
                    // two lanes exchange halves, so that a lane writes two consecutive tokens of a dim
                    __nv_bfloat16* dst = p.v_t + out0 + q * 32 * 64 + (r & 62);
#pragma unroll
                    for (int d = 0; d < 32; d += 2) {
                        const uint32_t mine = pack_bf16(__uint_as_float(t[d]), __uint_as_float(t[d + 1]));   // this token, dims d and d + 1
                        const uint32_t other = __shfl_xor_sync(0xffffffffu, mine, 1);
                        const uint32_t w = (lane & 1) ? __byte_perm(other, mine, 0x7632) : __byte_perm(mine, other, 0x5410);
                        *reinterpret_cast<uint32_t*>(dst + (d + (lane & 1)) * 64) = w;
                    }
                }
            }
        }
    }
    tc_fence_before();
    __syncthreads();
    if (*abort_flag) {
        // A wait gave up: before the CTA's shared memory is released the producer warps wait (with a limit) for the
        // copies they issued last, the only ones that can still be in flight; then report.
        if (warp == 0)
            for (int q = max(0, w_issued - STAGES); q < w_issued; ++q) mbar_drain(&w_full[q % STAGES], (q / STAGES) & 1);
        if (warp == 2 && c_issued > 0)
            for (int kb = 0; kb < KB; ++kb) mbar_drain(&c_full[kb], (c_issued - 1) & 1);
        if (threadIdx.x == 0 && p.status) atomicOr(p.status, 1);
        __syncthreads();
    }
    if (warp == 1) tmem_dealloc(tmem_base, 512);
}

}  // namespace

cudaError_t set_attrs_expand_sm100() {
    cudaError_t e = cudaFuncSetAttribute(expand_sm100_kernel<1>, cudaFuncAttributeMaxDynamicSharedMemorySize, SMEM_BYTES);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(expand_sm100_kernel<2>, cudaFuncAttributeMaxDynamicSharedMemorySize, SMEM_BYTES);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(expand_sm100_kernel<3>, cudaFuncAttributeMaxDynamicSharedMemorySize, SMEM_BYTES);
    return e;
}

cudaError_t launch_expand_sm100(const void* ckv, int64_t Lp, const void* w_uk, const void* w_uv, int H, void* k_nope, void* v_t,
                                int n_sm, int* status, cudaStream_t s) {
    if (Lp <= 0 || H <= 0 || (!k_nope && !v_t)) return cudaSuccess;
    if (Lp % 128 != 0) return cudaErrorInvalidValue;
    CUtensorMap tm_c, tm_uk, tm_uv;
    {
        uint64_t dims[2] = {512, (uint64_t)Lp};
        uint64_t str[1] = {512 * 2};
        uint32_t box[2] = {BK, 128};
        cudaError_t e = make_tmap_bf16(&tm_c, ckv, 2, dims, str, box);
        if (e != cudaSuccess) return e;
    }
    for (int i = 0; i < 2; ++i) {
        uint64_t dims[3] = {512, 128, (uint64_t)H};
        uint64_t str[2] = {512 * 2, 128 * 512 * 2};
        uint32_t box[3] = {BK, 128, 1};
        cudaError_t e = make_tmap_bf16(i == 0 ? &tm_uk : &tm_uv, i == 0 ? w_uk : w_uv, 3, dims, str, box);
        if (e != cudaSuccess) return e;
    }
    const int64_t units = Lp / 128 * H;   // <= 2^17 x 128
    const int ctas = (int)std::min<int64_t>(std::max(n_sm, 1), units);
    const ExpandParams p{reinterpret_cast<__nv_bfloat16*>(k_nope), reinterpret_cast<__nv_bfloat16*>(v_t), H, (int)(Lp / 64),
                         (int)(units / ctas), (int)(units % ctas), status};
    auto launch = [&](auto* kernel) { return launch_pdl(kernel, dim3(ctas), dim3(384), SMEM_BYTES, s, tm_c, tm_uk, tm_uv, p); };
    if (k_nope && v_t) return launch(expand_sm100_kernel<3>);
    return k_nope ? launch(expand_sm100_kernel<1>) : launch(expand_sm100_kernel<2>);
}

}  // namespace tmla
