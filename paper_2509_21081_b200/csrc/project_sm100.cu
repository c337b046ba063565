// Output projection O_A W_UV^T (Algorithm 1 line 7) with the LSE combine (line 8) as its epilogue, on tcgen05 / TMEM / TMA.
//
// Per head h: acc[b, :] = o_lat[b, h, :] (512) * W_UV[h]^T (512 x 128); out[b, h, :] = the merge of that row (the
// absorb side, already normalised) with the n_slots partials of the shared-prefix kernel by their log-sum-exps.
//
// The product itself is a few hundred clocks; what bounds the step is reading operands and partial slots.  Two forms:
//
// Ring form (several partial slots, or more work than one wave of CTAs).  Work item = (head, 128 requests, BN of the 128
// output columns); a CTA takes every gridDim-th item.  Operands and partials arrive by tiled bulk copies through two
// rings whose producers run ahead of their consumers, also into the next item; a thread that reads its own row of
// every slot from global memory waits once per slot instead.  Measured in a step (B200, before / with the rings): 1024
// requests, 128 heads, 2 slots 84 / 70 us; 128, 128, 3 slots 27.0 / 22.3; 256, 64, 2 slots 20.5 / 18.2; 166, 16, 8
// slots 29.7 / 13.0 (of which BN = 32 instead of 128: 16.5 -> 13.0).
// Warp roles (256 threads): warp 0 = producer of the operand ring, warp 1 = MMA issuer and TMEM owner, warp 2 = producer
// of the partial ring, warps 4-7 = epilogue (thread = one request row).
//
// Latency form (at most one slot, one wave): CTA = (head, 128 requests, 64 columns), two CTAs per SM, the first
// operand tiles requested before the CTA's set-up is complete, the one slot read from global memory meanwhile.
// 64 requests, 128 heads, 4096 tokens: step 84.1 -> 82.1 us; 8 requests without slots: 71.4 -> 69.6 (ring form 72.2).
#include <algorithm>
#include <cstddef>

#include "kernels.h"
#include "sm100.cuh"

namespace tmla {
namespace {

using namespace sm100;

constexpr int BM = 128, BK = 64, KB = 512 / BK;
constexpr int MAX_STAGES = 8;
constexpr int SLAB_BYTES = BM * 128;      // [128 rows][128 bytes], swizzled: 64 bf16 of an operand or 32 fp32 of a partial

template <int BN>
struct Shape {
    static constexpr int OP_BYTES = SLAB_BYTES + BN * BK * 2;                  // A slab + B slab
    static constexpr int PART_SLABS = BN == 128 ? 2 : 1;                        // 32-column slabs per partial stage
    static constexpr int PART_BYTES = PART_SLABS * SLAB_BYTES;
    static constexpr int OP_STAGES = BN == 128 ? 4 : 6, PART_STAGES = BN == 128 ? 3 : 6;
    static constexpr int CHUNKS = BN / (32 * PART_SLABS);                      // partial stages per slot
    static constexpr int SMEM = OP_STAGES * OP_BYTES + PART_STAGES * PART_BYTES + 1024;
    static_assert(OP_STAGES <= MAX_STAGES && PART_STAGES <= MAX_STAGES, "");
};

struct ProjectParams {
    int M, H, n_slots;
    int row_tiles, n_items;
    int early;             // trigger the kernel behind this one at the start (see project_sm100_plan)
    int* status;
    CombineEpilogue ce;
};

struct Barriers {
    uint64_t op_full[MAX_STAGES], op_empty[MAX_STAGES], part_full[MAX_STAGES], part_empty[MAX_STAGES], acc_full[2], acc_empty[2];
    uint32_t tmem_base;
    int abort_flag;
};

// 32 columns of a final row: the weighted partials `acc` plus the absorb side's accumulator columns, normalised, stored at
// element `at` of the output.
__device__ __forceinline__ void store_row32(const CombineEpilogue& ce, int64_t at, const float* acc, const uint32_t (&t)[32], float wa, float inv) {
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        float o[8];
#pragma unroll
        for (int e = 0; e < 8; ++e) {
            const float oa = wa > 0.f ? wa * __uint_as_float(t[j * 8 + e]) : 0.f;
            o[e] = (acc[j * 8 + e] + oa) * inv;
        }
        if (ce.out_fp32) {
            float* dst = reinterpret_cast<float*>(ce.out) + at + j * 8;
            *reinterpret_cast<float4*>(dst) = make_float4(o[0], o[1], o[2], o[3]);
            *reinterpret_cast<float4*>(dst + 4) = make_float4(o[4], o[5], o[6], o[7]);
        } else {
            *reinterpret_cast<uint4*>(reinterpret_cast<__nv_bfloat16*>(ce.out) + at + j * 8) =
                make_uint4(pack_bf16(o[0], o[1]), pack_bf16(o[2], o[3]), pack_bf16(o[4], o[5]), pack_bf16(o[6], o[7]));
        }
    }
}

// ---------------- ring form
template <int BN>
__global__ void __launch_bounds__(256, 1)
project_sm100_kernel(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmB,
                     const __grid_constant__ CUtensorMap tmP, ProjectParams p) {
    using S = Shape<BN>;
    constexpr int N_COL = 128 / BN;
    extern __shared__ uint8_t smem_raw[];
    uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    uint8_t* sOp = smem;
    uint8_t* sPart = smem + S::OP_STAGES * S::OP_BYTES;
    __shared__ Barriers bars;
    Barriers* bar = &bars;
    volatile int* abort_flag = &bar->abort_flag;

    const int warp = warp_index_uniform(), lane = threadIdx.x & 31;
    if (p.early) pdl_trigger();
    pdl_wait();

    const int n_my = (int)blockIdx.x < p.n_items ? (p.n_items - 1 - (int)blockIdx.x) / (int)gridDim.x + 1 : 0;
    struct Item { int n0, m0, h; };
    auto item_of = [&](int k) {   // columns fastest, then row tiles: CTAs that share a head's weights or rows run together
        const int i = (int)blockIdx.x + k * (int)gridDim.x;
        Item it;
        it.n0 = (i % N_COL) * BN;
        it.m0 = (i / N_COL) % p.row_tiles * BM;
        it.h = i / (N_COL * p.row_tiles);
        return it;
    };
    const uint32_t ld = elect_one() ? 1u : 0u;
    auto issue_op = [&](const Item& it, int kb, int pos) {
        const int s = pos % S::OP_STAGES;
        uint8_t* dst = sOp + s * S::OP_BYTES;
        mbar_arrive_expect_tx_if(ld, &bar->op_full[s], S::OP_BYTES);
        tma_load_3d_if(ld, dst, &tmA, &bar->op_full[s], kb * BK, it.h, it.m0);
        tma_load_3d_if(ld, dst + SLAB_BYTES, &tmB, &bar->op_full[s], kb * BK, it.n0, it.h);
    };
    auto issue_part = [&](const Item& it, int slot, int chunk, int pos) {
        const int s = pos % S::PART_STAGES;
        uint8_t* dst = sPart + s * S::PART_BYTES;
        mbar_arrive_expect_tx_if(ld, &bar->part_full[s], S::PART_BYTES);
#pragma unroll
        for (int i = 0; i < S::PART_SLABS; ++i)   // (32 fp32 columns as 64 16-bit elements)
            tma_load_4d_if(ld, dst + i * SLAB_BYTES, &tmP, &bar->part_full[s], 2 * (it.n0 + (chunk * S::PART_SLABS + i) * 32), it.h, it.m0, slot);
    };

    if (warp == 0) {
        if (lane < MAX_STAGES) {
            mbar_init(&bar->op_full[lane], 1);
            mbar_init(&bar->op_empty[lane], 1);
            mbar_init(&bar->part_full[lane], 1);
            mbar_init(&bar->part_empty[lane], 4);
        } else if (lane < MAX_STAGES + 2) {
            mbar_init(&bar->acc_full[lane - MAX_STAGES], 1);
            mbar_init(&bar->acc_empty[lane - MAX_STAGES], 4);
        }
        if (lane == 31) bar->abort_flag = 0;
        fence_mbar_init();
    }
    if (warp == 1) tmem_alloc(&bar->tmem_base, 2 * BN);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem_base = __shfl_sync(0xffffffffu, bar->tmem_base, 0);

    int op_issued = 0, part_issued = 0;   // producer warps: copies issued (upper bounds), for the abort path
    if (warp == 0) {
        bool ok = true;
        for (int k = 0; k < n_my && ok; ++k) {
            const Item it = item_of(k);
            for (int kb = 0; kb < KB && ok; ++kb) {
                const int pos = op_issued;
                ok = mbar_wait_warp(&bar->op_empty[pos % S::OP_STAGES], ((pos / S::OP_STAGES) & 1) ^ 1, abort_flag);
                if (!ok) break;
                issue_op(it, kb, pos);
                ++op_issued;
            }
        }
    } else if (warp == 2) {
        bool ok = true;
        for (int k = 0; k < n_my && ok; ++k) {
            const Item it = item_of(k);
            for (int j = 0; j < p.n_slots * S::CHUNKS && ok; ++j) {
                const int pos = part_issued;
                ok = mbar_wait_warp(&bar->part_empty[pos % S::PART_STAGES], ((pos / S::PART_STAGES) & 1) ^ 1, abort_flag);
                if (!ok) break;
                issue_part(it, j / S::CHUNKS, j % S::CHUNKS, pos);
                ++part_issued;
            }
        }
    } else if (warp == 1) {
        constexpr uint32_t idesc = idesc_bf16(BM, BN, false, false);
        bool ok = true;
        int pos = 0;
        for (int k = 0; k < n_my && ok; ++k) {
            ok = mbar_wait_warp(&bar->acc_empty[k & 1], ((k >> 1) & 1) ^ 1, abort_flag);   // accumulator read by the epilogue
            for (int kb = 0; kb < KB && ok; ++kb, ++pos) {
                const int s = pos % S::OP_STAGES;
                ok = mbar_wait_warp(&bar->op_full[s], (pos / S::OP_STAGES) & 1, abort_flag);
                if (!ok) break;
                tc_fence_after();
                const uint32_t sa = smem_u32(sOp + s * S::OP_BYTES);
                const uint64_t da = smem_desc_k_sw128(sa), db = smem_desc_k_sw128(sa + SLAB_BYTES);
#pragma unroll
                for (int kk = 0; kk < BK / 16; ++kk)
                    umma_ss_if(ld, tmem_base + (k & 1) * BN, da + 2 * kk, db + 2 * kk, idesc, (kb | kk) != 0);
                umma_commit_if(ld, &bar->op_empty[s]);
            }
            if (ok) umma_commit_if(ld, &bar->acc_full[k & 1]);
        }
    } else if (warp >= 4) {
        const CombineEpilogue& ce = p.ce;
        const int lg = (warp & 3) * 32, r = lg + lane;
        const int64_t BH = (int64_t)p.M * p.H;
        bool ok = true;
        int pos = 0;
        for (int k = 0; k < n_my && ok; ++k) {
            const Item it = item_of(k);
            const int row = it.m0 + r;
            const int64_t bh = (int64_t)row * p.H + it.h;
            const bool live = row < p.M;
            // merge weights of this (request, head)
            float la = -INFINITY, m = -INFINITY;
            if (live) {
                la = ce.lse_abs[bh];
                m = la;
#pragma unroll 4
                for (int i = 0; i < p.n_slots; ++i) m = fmaxf(m, ce.lse_naive[i * BH + bh]);
            }
            const float wa = (la == -INFINITY) ? 0.f : __expf(la - m);
            float zsum = wa;
            float acc[BN];
#pragma unroll
            for (int q = 0; q < BN; ++q) acc[q] = 0.f;
            // weighted sum of the slots, while the product is running
#pragma unroll 1
            for (int i = 0; i < p.n_slots && ok; ++i) {
                const float l = live ? ce.lse_naive[i * BH + bh] : -INFINITY;
                const float w = (l == -INFINITY) ? 0.f : __expf(l - m);   // an empty partial's slot was never written
                zsum += w;
#pragma unroll
                for (int c = 0; c < S::CHUNKS; ++c) {
                    const int s = (pos + c) % S::PART_STAGES;
                    ok = __all_sync(0xffffffffu, mbar_wait(&bar->part_full[s], ((pos + c) / S::PART_STAGES) & 1, abort_flag));
                    if (!ok) break;
                    if (w != 0.f) {
#pragma unroll
                        for (int sl = 0; sl < S::PART_SLABS; ++sl) {
                            const uint8_t* src = sPart + s * S::PART_BYTES + sl * SLAB_BYTES + r * 128;
#pragma unroll
                            for (int q = 0; q < 8; ++q) {
                                const float4 v = *reinterpret_cast<const float4*>(src + ((q ^ (r & 7)) << 4));
                                float* a = acc + (c * S::PART_SLABS + sl) * 32 + 4 * q;
                                a[0] += w * v.x; a[1] += w * v.y; a[2] += w * v.z; a[3] += w * v.w;
                            }
                        }
                    }
                    __syncwarp();
                    if (lane == 0) mbar_arrive(&bar->part_empty[s]);
                }
                pos += S::CHUNKS;
            }
            if (!ok) break;
            const float inv = zsum > 0.f ? 1.f / zsum : 0.f;
            ok = __all_sync(0xffffffffu, mbar_wait(&bar->acc_full[k & 1], (k >> 1) & 1, abort_flag));
            if (!ok) break;
            tc_fence_after();
            // the absorb-side row (the accumulator) with its weight, normalise, write the final row
#pragma unroll
            for (int c = 0; c < BN / 32; ++c) {
                uint32_t t[32];
                tmem_ld32(tmem_base + ((uint32_t)lg << 16) + (k & 1) * BN + c * 32, t);
                tmem_ld_wait();
                if (c == BN / 32 - 1) {
                    tc_fence_before();
                    __syncwarp();
                    if (lane == 0) mbar_arrive(&bar->acc_empty[k & 1]);
                }
                if (!live) continue;
                store_row32(ce, bh * 128 + it.n0 + c * 32, acc + c * 32, t, wa, inv);
            }
            if (live && it.n0 == 0 && ce.lse_out) ce.lse_out[bh] = (m == -INFINITY) ? -INFINITY : m + __logf(zsum);
        }
    }
    tc_fence_before();
    __syncthreads();
    if (*abort_flag) {
        // A wait gave up: before the CTA's shared memory is released the producer warps wait (with a limit) for the
        // copies they issued last, the only ones that can still be in flight; then report.
        if (warp == 0)
            for (int q = max(0, op_issued - S::OP_STAGES); q < op_issued; ++q) mbar_drain(&bar->op_full[q % S::OP_STAGES], (q / S::OP_STAGES) & 1);
        if (warp == 2)
            for (int q = max(0, part_issued - S::PART_STAGES); q < part_issued; ++q)
                mbar_drain(&bar->part_full[q % S::PART_STAGES], (q / S::PART_STAGES) & 1);
        if (threadIdx.x == 0 && p.status) atomicOr(p.status, 1);
        __syncthreads();
    }
    if (warp == 1) tmem_dealloc(tmem_base, 2 * BN);
}

// ---------------- latency form
constexpr int LAT_BN = 64, LAT_STAGES = 4, LAT_STAGE_BYTES = SLAB_BYTES + LAT_BN * BK * 2;
constexpr int LAT_SMEM = LAT_STAGES * LAT_STAGE_BYTES + 1024;

__global__ void __launch_bounds__(192, 2)
project_latency_sm100_kernel(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmB, ProjectParams p) {
    extern __shared__ uint8_t smem_raw[];
    uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    __shared__ uint64_t full[LAT_STAGES], empty[LAT_STAGES], acc_full;
    __shared__ uint32_t tmem_holder;
    __shared__ int abort_word;
    volatile int* abort_flag = &abort_word;

    const int warp = warp_index_uniform(), lane = threadIdx.x & 31;
    const int n0 = blockIdx.x * LAT_BN, m0 = blockIdx.y * BM, h = blockIdx.z;
    if (p.early) pdl_trigger();

    const uint32_t ld = elect_one() ? 1u : 0u;
    auto issue_weights = [&](int kb) {
        const int s = kb % LAT_STAGES;
        mbar_arrive_expect_tx_if(ld, &full[s], LAT_STAGE_BYTES);
        tma_load_3d_if(ld, smem + s * LAT_STAGE_BYTES + SLAB_BYTES, &tmB, &full[s], kb * BK, n0, h);
    };
    auto issue_rows = [&](int kb) {
        const int s = kb % LAT_STAGES;
        tma_load_3d_if(ld, smem + s * LAT_STAGE_BYTES, &tmA, &full[s], kb * BK, h, m0);
    };
    // (the weights are the caller's, unchanged while the handle lives: requested before the wait, see kernels.h)
    if (warp == 0) {
        if (lane < LAT_STAGES) {
            mbar_init(&full[lane], 1);
            mbar_init(&empty[lane], 1);
        }
        if (lane == LAT_STAGES) {
            mbar_init(&acc_full, 1);
            *abort_flag = 0;
        }
        fence_mbar_init();
        __syncwarp();
#pragma unroll 1
        for (int kb = 0; kb < LAT_STAGES; ++kb) issue_weights(kb);
        pdl_wait();
#pragma unroll 1
        for (int kb = 0; kb < LAT_STAGES; ++kb) issue_rows(kb);
    }
    pdl_wait();
    if (warp == 1) tmem_alloc(&tmem_holder, LAT_BN);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem_base = __shfl_sync(0xffffffffu, tmem_holder, 0);

    int kb_issued = LAT_STAGES;   // producer warp: operand tiles issued (upper bound), for the abort path
    if (warp == 0) {
        for (int kb = LAT_STAGES; kb < KB; ++kb) {
            if (!mbar_wait_warp(&empty[kb % LAT_STAGES], ((kb / LAT_STAGES) & 1) ^ 1, abort_flag)) break;
            kb_issued = kb + 1;
            issue_weights(kb);
            issue_rows(kb);
        }
    } else if (warp == 1) {
        constexpr uint32_t idesc = idesc_bf16(BM, LAT_BN, false, false);
        bool ok = true;
        for (int kb = 0; kb < KB && ok; ++kb) {
            const int s = kb % LAT_STAGES;
            ok = mbar_wait_warp(&full[s], (kb / LAT_STAGES) & 1, abort_flag);
            if (!ok) break;
            tc_fence_after();
            const uint32_t sa = smem_u32(smem + s * LAT_STAGE_BYTES);
            const uint64_t da = smem_desc_k_sw128(sa), db = smem_desc_k_sw128(sa + SLAB_BYTES);
#pragma unroll
            for (int k = 0; k < BK / 16; ++k) umma_ss_if(ld, tmem_base, da + 2 * k, db + 2 * k, idesc, (kb | k) != 0);
            umma_commit_if(ld, &empty[s]);
        }
        if (ok) umma_commit_if(ld, &acc_full);
    } else {
        const CombineEpilogue& ce = p.ce;
        const int lg = (warp & 3) * 32, row = m0 + lg + lane;
        const int64_t bh = (int64_t)row * p.H + h;
        const bool live = row < p.M;
        // while the operands are in flight: the merge weights of this (request, head) and its row of the slot
        float4 v[LAT_BN / 4];
        float wa = 0.f, wn = 0.f, inv = 0.f, lse = -INFINITY;
        if (live) {
            const float la = ce.lse_abs[bh], ln = p.n_slots > 0 ? ce.lse_naive[bh] : -INFINITY;
            const float m = fmaxf(la, ln);
            wa = (la == -INFINITY) ? 0.f : __expf(la - m);
            wn = (ln == -INFINITY) ? 0.f : __expf(ln - m);      // (an empty partial's slot was never written)
            const float z = wa + wn;
            inv = z > 0.f ? 1.f / z : 0.f;
            if (m != -INFINITY) lse = m + __logf(z);
        }
        const float4* src = reinterpret_cast<const float4*>(ce.o_naive + bh * 128 + n0);
#pragma unroll
        for (int q = 0; q < LAT_BN / 4; ++q) v[q] = wn > 0.f ? src[q] : make_float4(0.f, 0.f, 0.f, 0.f);
        const bool ok = __all_sync(0xffffffffu, mbar_wait(&acc_full, 0, abort_flag));
        tc_fence_after();
        if (ok) {
#pragma unroll
            for (int c = 0; c < LAT_BN / 32; ++c) {
                uint32_t t[32];
                tmem_ld32(tmem_base + ((uint32_t)lg << 16) + c * 32, t);
                tmem_ld_wait();
                float acc[32];
#pragma unroll
                for (int q = 0; q < 8; ++q) {
                    acc[4 * q] = wn * v[8 * c + q].x; acc[4 * q + 1] = wn * v[8 * c + q].y;
                    acc[4 * q + 2] = wn * v[8 * c + q].z; acc[4 * q + 3] = wn * v[8 * c + q].w;
                }
                if (live) store_row32(ce, bh * 128 + n0 + c * 32, acc, t, wa, inv);
            }
            if (live && n0 == 0 && ce.lse_out) ce.lse_out[bh] = lse;
        }
    }
    tc_fence_before();
    __syncthreads();
    if (*abort_flag) {   // as in the ring form
        if (warp == 0)
            for (int kb = max(0, kb_issued - LAT_STAGES); kb < kb_issued; ++kb) mbar_drain(&full[kb % LAT_STAGES], (kb / LAT_STAGES) & 1);
        if (threadIdx.x == 0 && p.status) atomicOr(p.status, 1);
        __syncthreads();
    }
    if (warp == 1) tmem_dealloc(tmem_base, LAT_BN);
}

template <int BN>
cudaError_t launch_columns(const CUtensorMap& tmA, const CUtensorMap& tmB, const CUtensorMap& tmP, ProjectParams p, int n_sm, cudaStream_t s) {
    return launch_pdl(project_sm100_kernel<BN>, dim3(std::min(p.n_items, n_sm)), dim3(256), Shape<BN>::SMEM, s, tmA, tmB, tmP, p);
}

}  // namespace

cudaError_t set_attrs_project_sm100() {
    cudaError_t e = cudaFuncSetAttribute(project_sm100_kernel<32>, cudaFuncAttributeMaxDynamicSharedMemorySize, Shape<32>::SMEM);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(project_latency_sm100_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, LAT_SMEM);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(project_sm100_kernel<128>, cudaFuncAttributeMaxDynamicSharedMemorySize, Shape<128>::SMEM);
    return e;
}

// (the figures at the top of the file: one slot and one wave favour the latency form; with few (head, row tile) pairs the
// ring form's 32-column items keep four times as many SMs reading)
//
// The early trigger lets the next step's shared-prefix kernel start on the SMs this one leaves.  With more (head, row tile)
// pairs than SMs, CTAs that take several are all resident at once, and the trigger would come at the very start: that kernel
// then had every SM before the next step's query absorption, which waits on another stream, and the absorb branch ran
// behind it instead of beside it.  Measured (B200, us per step, with / without the trigger, 128 heads): 198 requests over 5126
// tokens 179 / 167, 140 over 5126 170 / 154, 300 over 2000 204 / 199, 1024 over 4096 644 / 629; with fewer pairs it is worth it:
// 200 requests x 64 heads 87 / 93, and 1 % with two 32-column items per CTA (64 x 64).  The kernel of an 8-bit prefix lasts
// longer and leaves the tensor cores more idle, so that the absorb branch is best beside it from the start: without the
// trigger 128 requests over 700 tokens 67.4 -> 62.0 us, 64 over 4096 93.5 -> 88.5, 40 over 9000 159 -> 130, 200 x 64 heads over
// 4096 111 -> 100 (one shape of fifteen lost: 48 over 2000, 60.5 -> 64.2).
ProjectPlan project_sm100_plan(int B, int H, int n_slots, bool prefix_8bit, int n_sm) {
    const int row_tiles = (B + BM - 1) / BM, tiles = row_tiles * H;
    ProjectPlan p;
    p.latency = n_slots <= 1 && tiles <= n_sm;
    p.columns = p.latency ? LAT_BN : (tiles * 2 <= n_sm ? 32 : 128);
    p.items = 128 / p.columns * tiles;
    p.early = tiles <= n_sm && !prefix_8bit;
    return p;
}

cudaError_t launch_project_sm100(const void* o_lat, const void* w_uv, int B, bool prefix_8bit, int n_sm, int* status, cudaStream_t s,
                                 const CombineEpilogue& ce) {
    if (B <= 0 || ce.H <= 0) return cudaSuccess;
    if (n_sm < 1) n_sm = 1;
    const ProjectPlan pl = project_sm100_plan(B, ce.H, ce.n_naive, prefix_8bit, n_sm);
    const bool latency = pl.latency;
    const int bn = pl.columns, row_tiles = (B + BM - 1) / BM;
    CUtensorMap tmA, tmB, tmP;
    {
        uint64_t dims[3] = {512, (uint64_t)ce.H, (uint64_t)B};
        uint64_t strides[2] = {512 * 2, (uint64_t)ce.H * 512 * 2};
        uint32_t box[3] = {BK, 1, BM};
        cudaError_t e = make_tmap_bf16(&tmA, o_lat, 3, dims, strides, box);
        if (e != cudaSuccess) return e;
    }
    {
        uint64_t dims[3] = {512, 128, (uint64_t)ce.H};
        uint64_t strides[2] = {512 * 2, 128 * 512 * 2};
        uint32_t box[3] = {BK, (uint32_t)bn, 1};
        cudaError_t e = make_tmap_bf16(&tmB, w_uv, 3, dims, strides, box);
        if (e != cudaSuccess) return e;
    }
    const ProjectParams p{B, ce.H, ce.n_naive, row_tiles, pl.items, pl.early, status, ce};
    if (latency) return launch_pdl(project_latency_sm100_kernel, dim3(128 / LAT_BN, row_tiles, ce.H), dim3(192), LAT_SMEM, s, tmA, tmB, p);
    if (ce.n_naive > 0) {   // the partials as rows of 256 16-bit elements (the copies move bytes)
        uint64_t dims[4] = {256, (uint64_t)ce.H, (uint64_t)B, (uint64_t)ce.n_naive};
        uint64_t strides[3] = {512, (uint64_t)ce.H * 512, (uint64_t)B * ce.H * 512};
        uint32_t box[4] = {64, 1, BM, 1};
        cudaError_t e = make_tmap_bf16(&tmP, ce.o_naive, 4, dims, strides, box);
        if (e != cudaSuccess) return e;
    } else {
        tmP = tmA;
    }
    if (bn == 32) return launch_columns<32>(tmA, tmB, tmP, p, n_sm, s);
    return launch_columns<128>(tmA, tmB, tmP, p, n_sm, s);
}

}  // namespace tmla
