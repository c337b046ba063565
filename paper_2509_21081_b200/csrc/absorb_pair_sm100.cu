// Absorb attention over latent tokens (Algorithm 1 line 6) for 128 query rows at a time: a pair of CTAs on one product.
//
// Work item (CTA pair) = (128 query rows, KV chunk).  Over a request's own suffix the rows are the heads of that request (with
// fewer than 128 some rows are nobody's), over the shared prefix 128 consecutive rows of the stacked [B * H] matrix.
//     S [128 rows, 128 tokens] = Q [128, 576] * K_tile [128, 576]^T       (K_tile = latent 512 | rope 64 of 128 tokens)
//     O [128 rows, 512]       += P [128, 128 tokens] * C_tile [128, 512]
// Each CTA holds 64 query rows; with M = 128 over two CTAs the accumulators of its 64 rows fold into all 128 lanes of its tensor
// memory (measured layout: lane l < 64 holds row l of the first half of the N columns, lane 64 + l row l of the second half), so
// O takes 256 columns and S 64, and two S buffers fit beside O.  CTA r supplies tokens [64 r, 64 r + 64) as B of the first
// product (72 KB) and latent dims [256 r, 256 r + 256) of all 128 tokens as B of the second (64 KB): a tile moves 136 KB per CTA
// for 128 tokens x 64 rows, of which the second operand always hits L2.
//
// Why a pair: the 64-row kernel (one CTA, transposed) issues M = 64 products at half rate for S and N = 64 products that take
// 6 KB of shared memory per 32-clock instruction for O: 2580 clocks per 64 tokens x 64 rows, 10 320 SM clocks for what a pair does
// in one tile.  Here the products run at the full rate (measured: 32 and 64 clocks per instruction, 36 * 32 + 16 * 64 = 2176 per
// tile) and a tile takes 2416 clocks, so the tensor core bounds a long chunk.  (B200, us per absorb-only step, the 64-row kernel
// / this one, 128 heads, 16384 + 256 tokens: 1 request 31.3 / 31.2, 8 69.4 / 49.4, 32 247 / 166; hybrid step of 128 requests,
// 4096 + 2048 tokens 184.5 / 145.2.)
//
// The issuing thread elects itself around every group of MMAs: with a predicate that reaches the instructions through other
// data flow (rank, warp and election combined) each took 80 to 100 clocks to issue.
//
// Softmax: thread = (row, 32 tokens of a tile), eight warps.  Every row keeps a reference exponent, the same in the four threads
// that share the row, which is raised only when some logit exceeds it by more than 2^8 (a collective event of the CTA that also
// rescales O).  P (bf16) goes to shared memory as the K-major A operand.
//
// Warp roles (384 threads per CTA): warp 0 loads Q and K tiles, warp 2 the second operand; warp 1 allocates tensor memory and in
// the even CTA issues both products; warps 4-11 softmax and epilogue.
#include <algorithm>
#include <cstddef>

#include "kernels.h"
#include "sm100.cuh"

namespace tmla {
namespace {

using namespace sm100;

constexpr int TOK = 128;
constexpr int SLAB = 64 * 64 * 2;                // [64 rows][64 bf16], 128-byte swizzled rows
constexpr int K_BYTES = 9 * SLAB;                // 64 tokens: 8 latent slabs + 1 rope slab
constexpr int V_BYTES = 8 * SLAB;                // 128 tokens x 256 dims: two blocks of [2 token halves][2 slabs]
constexpr int Q_BYTES = 9 * SLAB;
constexpr int P_BYTES = 2 * SLAB;                // [2 token halves][64 rows][64 tokens]
constexpr float kRescaleThreshold = 8.f;         // log2 units

struct PairParams {
    int B, H;
    int chunk, n_shared_chunks, n_suffix_chunks;
    int shared_groups;     // 128-row groups per shared-prefix chunk
    int stacked;           // ... cut from the stacked [B * H] query matrix (else one per request)
    int Ls_absorb;
    int page_size, max_pages;
    int num_pages;
    const int32_t* block_table;
    const int32_t* seq_lens;
    const int32_t* order;
    const int4* desc;      // optional, per launch position: {request, clamped suffix length, page 0, page 1}
    float scale_log2;
    float* lse_part;       // [n_chunks][B][H]
    __nv_bfloat16* o_lat_direct;   // single chunk: the merged result bf16 [B][H][512], and its LSE
    float* lse_direct;
    int* status;
    const char* l2_base;   // read by the kernel behind this one: requested into L2, l2_bytes per lane of warp 3
    uint32_t l2_total, l2_bytes;
};

struct Shared {
    uint64_t q_full;                  // these four groups count the copies of both CTAs, in the even CTA
    uint64_t k_full[2];               // dims 0..255 | dims 256..511 and rope keys
    uint64_t v_full[2];               // block 0 | 1 of the second operand
    uint64_t p_ready;                 // one arrival per softmax warp of both CTAs
    uint64_t k_empty[2], v_empty[2];  // in both CTAs, by the commits of the even one
    uint64_t s_ready[2];
    uint64_t o_done[2];               // PV product of tile j: o_done[j & 1] (a parity wait tells one completion from none)
    uint64_t v_tail;                  // own copies of the second operand of a ragged last tile
    uint32_t tmem_base;
    int abort_flag;
    float red[4][64];                 // [token quarter][row]
};

constexpr int kPairSmem = K_BYTES + V_BYTES + Q_BYTES + P_BYTES + 1024 + (int)sizeof(Shared);
static_assert(kPairSmem <= 232448, "shared memory of one SM");

constexpr int kSoftmaxBar = 1;
__device__ __forceinline__ bool vote_or(bool pred) {   // over the 256 softmax threads
    uint32_t r;
    asm volatile(
        "{\n.reg .pred p, q;\nsetp.ne.b32 q, %2, 0;\n"
        "bar.red.or.pred p, %1, 256, q;\n"
        "selp.u32 %0, 1, 0, p;\n}\n"
        : "=r"(r) : "n"(kSoftmaxBar), "r"(pred ? 1u : 0u) : "memory");
    return r != 0;
}
__device__ __forceinline__ void softmax_sync() { asm volatile("bar.sync %0, 256;\n" ::"n"(kSoftmaxBar) : "memory"); }

__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(384, 1)
absorb_pair_sm100_kernel(const __grid_constant__ CUtensorMap tm_qa, const __grid_constant__ CUtensorMap tm_qp,
                         const __grid_constant__ CUtensorMap tm_ckv_sh, const __grid_constant__ CUtensorMap tm_kpe_sh,
                         const __grid_constant__ CUtensorMap tm_ckv_pg, const __grid_constant__ CUtensorMap tm_kpe_pg,
                         const __grid_constant__ CUtensorMap tm_o_sh, const __grid_constant__ CUtensorMap tm_o_sf, PairParams p) {
    extern __shared__ uint8_t smem_raw[];
    uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    uint8_t* sK = smem;
    uint8_t* sV = sK + K_BYTES;
    uint8_t* sQ = sV + V_BYTES;
    uint8_t* sP = sQ + Q_BYTES;
    Shared* sh = reinterpret_cast<Shared*>(sP + P_BYTES);
    volatile int* abort_flag = &sh->abort_flag;

    const int warp = warp_index_uniform(), lane = threadIdx.x & 31;
    const uint32_t rank = cluster_cta_rank();
    pdl_trigger();
    // Set-up touches no global memory: it runs before the wait for the preceding kernel.
    if (warp == 0) {
        uint64_t* all = &sh->q_full;
        constexpr int n_bars = (int)(offsetof(Shared, tmem_base) / sizeof(uint64_t));
        if (lane < n_bars) mbar_init(all + lane, all + lane == &sh->p_ready ? 16 : 1);
        if (lane == 0) sh->abort_flag = 0;
        fence_mbar_init();
        __syncwarp();
    }
    if (warp == 1) tmem_alloc_pair(&sh->tmem_base, 512);
    if (warp == 2) {
        if (lane == 0) prefetch_tmap(&tm_qa);
        if (lane == 1) prefetch_tmap(&tm_qp);
        if (lane == 2) prefetch_tmap(&tm_ckv_sh);
        if (lane == 3) prefetch_tmap(&tm_kpe_sh);
        if (lane == 4) prefetch_tmap(&tm_ckv_pg);
        if (lane == 5) prefetch_tmap(&tm_kpe_pg);
    }
    tc_fence_before();
    cluster_sync();
    tc_fence_after();
    const uint32_t tmem_base = __shfl_sync(0xffffffffu, sh->tmem_base, 0);

    // Work items in launch order: the shared-prefix items (chunk fastest, then row group), then the suffix items
    // (chunk fastest, then request position in longest-first order).
    const int item = blockIdx.x >> 1;
    const int n_shared_items = p.n_shared_chunks * p.shared_groups;
    const bool shared_seg = item < n_shared_items;
    // The preceding kernel writes Q_A and the descriptors, the caller's kernels the page table and the lengths: the wait.  The
    // handle's latent rows are older: items over the shared prefix request their first tile before it (below).
    if (!shared_seg) pdl_wait();
    int chunk, row0, n_rows, b = 0, len_b = -1, pg0 = -1, pg1 = -1;
    if (shared_seg) {
        chunk = item % p.n_shared_chunks;
        const int g = item / p.n_shared_chunks;
        row0 = p.stacked ? g * 128 : g * p.H;
        n_rows = p.stacked ? min(128, p.B * p.H - row0) : p.H;
    } else {
        const int i = item - n_shared_items;
        chunk = p.n_shared_chunks + i % p.n_suffix_chunks;
        const int z = i / p.n_suffix_chunks;
        if (p.desc != nullptr) {
            const int4 d = p.desc[z];
            b = d.x; len_b = d.y; pg0 = d.z; pg1 = d.w;
        } else {
            b = p.order ? p.order[z] : z;
        }
        row0 = b * p.H;
        n_rows = p.H;
    }
    int seg_len, tok_begin;
    if (shared_seg) {
        seg_len = p.Ls_absorb;
        tok_begin = chunk * p.chunk;
    } else {
        seg_len = len_b >= 0 ? len_b : min(max(p.seq_lens[b], 0), p.max_pages * p.page_size);
        tok_begin = (chunk - p.n_shared_chunks) * p.chunk;
    }
    // (through a shuffle: the role warps' loops are then known to be uniform)
    const int tok_end = __shfl_sync(0xffffffffu, min(seg_len, tok_begin + p.chunk), 0);
    const int n_tiles = tok_end > tok_begin ? (tok_end - tok_begin + TOK - 1) / TOK : 0;
    const int n_last = tok_end - tok_begin - (n_tiles - 1) * TOK;      // tokens of the last tile
    // Rows of the paged cache past the end may hold anything, NaN included; the PV product takes whole groups of 16 tokens, so the
    // rest of the last group is zeroed in shared memory (the handle's copy of the prefix is padded with zeros).
    const bool zero_tail = !shared_seg && (n_last & 15) != 0;

    const CUtensorMap* tc = shared_seg ? &tm_ckv_sh : &tm_ckv_pg;
    const CUtensorMap* tk = shared_seg ? &tm_kpe_sh : &tm_kpe_pg;
    const int32_t* bt = p.block_table + (int64_t)b * p.max_pages;
    bool bad_page = false;   // producer warps only: a page id of the caller's table was out of range
    // physical page and slot of half `h` (64 tokens) of tile j; a half past the end reads as zeros
    auto page_of = [&](int j, int h, int& page, int& slot) {
        const int t0 = tok_begin + j * TOK + h * 64;
        if (shared_seg) {
            page = t0 / 64;
            slot = 0;
        } else {
            slot = t0 % p.page_size;
            page = p.num_pages;
            if (t0 < tok_end) {
                const int idx = t0 / p.page_size;
                page = (p.desc != nullptr && idx < 2) ? (idx == 0 ? pg0 : pg1) : __shfl_sync(0xffffffffu, bt[idx], 0);
                // The tensor map ends at num_pages: a coordinate at or past it reads as zeros instead of touching memory the
                // caller does not own.  The violation is reported through the status word.
                if ((unsigned)page >= (unsigned)p.num_pages) {
                    bad_page = true;
                    page = p.num_pages;
                }
            }
        }
    };

    int issued = 0;   // producer warps: tiles whose copies were issued, for the abort path
    if (n_tiles > 0) {
        if (warp == 0) {
            // ---------------- Q and K tiles
            const uint32_t ld = elect_one() ? 1u : 0u;
            const uint32_t ld_even = rank == 0 ? ld : 0u;
            const uint32_t kf[2] = {cluster_map(&sh->k_full[0], 0), cluster_map(&sh->k_full[1], 0)};
            auto prefetch_tile = [&](int j) {
                // The ring holds one tile: the paged tiles are requested into L2 two tiles ahead, so that a load into a freed
                // slot takes an L2 round trip.
                if (shared_seg || j >= n_tiles) return;
                int page, slot;
                page_of(j, (int)rank, page, slot);
#pragma unroll 1
                for (int i = 0; i < 4; ++i) tma_prefetch_4d_if(ld, tc, 0, slot, 2 * i, page);
                tma_prefetch_3d_if(ld, tk, 0, slot, page);
            };
            bool ok = true;
            for (int j = 0; j < n_tiles && ok; ++j) {
                int page, slot;
                page_of(j, (int)rank, page, slot);
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    if (j > 0) ok = ok && mbar_wait_warp(&sh->k_empty[h], (j - 1) & 1, abort_flag);
                    if (!ok) break;
                    mbar_arrive_expect_tx_if(ld_even, &sh->k_full[h], 2 * (h == 0 ? 4 : 5) * SLAB);
                    tma_load_4d_pair_if(ld, sK + (4 * h) * SLAB, tc, kf[h], 0, slot, 4 * h, page);
                    tma_load_4d_pair_if(ld, sK + (4 * h + 2) * SLAB, tc, kf[h], 0, slot, 4 * h + 2, page);
                    if (h == 1) tma_load_3d_pair_if(ld, sK + 8 * SLAB, tk, kf[h], 0, slot, page);
                }
                issued = j + 1;
                if (j == 0) {
                    if (shared_seg) pdl_wait();
                    const uint32_t qf = cluster_map(&sh->q_full, 0);
                    const int y = row0 + 64 * (int)rank;
                    mbar_arrive_expect_tx_if(ld_even, &sh->q_full, 2 * Q_BYTES);
#pragma unroll 1
                    for (int sl = 0; sl < 8; ++sl) tma_load_2d_pair_if(ld, sQ + sl * SLAB, &tm_qa, qf, sl * 64, y);
                    tma_load_2d_pair_if(ld, sQ + 8 * SLAB, &tm_qp, qf, 0, y);
                    prefetch_tile(1);
                }
                prefetch_tile(j + 2);
            }
        } else if (warp == 2) {
            // ---------------- second operand: latent dims [256 rank, + 256) of all 128 tokens, two blocks of 128 dims
            const uint32_t ld = elect_one() ? 1u : 0u;
            const uint32_t ld_even = rank == 0 ? ld : 0u;
            const uint32_t vf[2] = {cluster_map(&sh->v_full[0], 0), cluster_map(&sh->v_full[1], 0)};
            const uint32_t vt = cluster_map(&sh->v_tail, rank);
            bool ok = true;
            for (int j = 0; j < n_tiles && ok; ++j) {
                int page[2], slot[2];
                page_of(j, 0, page[0], slot[0]);
                page_of(j, 1, page[1], slot[1]);
                const bool tail = zero_tail && j == n_tiles - 1;     // counted by the CTA's own barrier: its threads zero rows
                if (tail) mbar_arrive_expect_tx_if(ld, &sh->v_tail, V_BYTES);
#pragma unroll
                for (int nb = 0; nb < 2; ++nb) {
                    if (j > 0) ok = ok && mbar_wait_warp(&sh->v_empty[nb], (j - 1) & 1, abort_flag);
                    if (!ok) break;
                    if (!tail) mbar_arrive_expect_tx_if(ld_even, &sh->v_full[nb], V_BYTES);
                    const uint32_t bar = tail ? vt : vf[nb];
                    const int slab = 4 * (int)rank + 2 * nb;
                    tma_load_4d_pair_if(ld, sV + (4 * nb) * SLAB, tc, bar, 0, slot[0], slab, page[0]);
                    tma_load_4d_pair_if(ld, sV + (4 * nb + 2) * SLAB, tc, bar, 0, slot[1], slab, page[1]);
                }
                issued = j + 1;
            }
            if (shared_seg) pdl_wait();
        } else if (warp == 1 && rank == 0) {
            // ---------------- both products (even CTA)
            if (shared_seg) pdl_wait();
            constexpr uint32_t idesc_s = idesc_bf16(128, 128, false, false);
            constexpr uint32_t idesc_o = idesc_bf16(128, 256, false, true);
            const uint32_t qa = smem_u32(sQ), ka = smem_u32(sK), va = smem_u32(sV), pa = smem_u32(sP);
            bool ok = mbar_wait_warp(&sh->q_full, 0, abort_flag);
            for (int j = 0; j <= n_tiles && ok; ++j) {
                if (j < n_tiles) {
                    // S(j) into buffer j & 1: the softmax of tile j - 2 has read it (p_ready of that tile, awaited below)
                    const uint32_t d = tmem_base + 256u + (uint32_t)(j & 1) * 64u;
#pragma unroll
                    for (int h = 0; h < 2; ++h) {
                        ok = ok && mbar_wait_warp(&sh->k_full[h], j & 1, abort_flag);
                        if (!ok) break;
                        tc_fence_after();
                        if (elect_one()) {
#pragma unroll
                            for (int sl = 4 * h; sl < (h == 0 ? 4 : 9); ++sl) {
                                const uint64_t da = smem_desc_k_sw128(qa + sl * SLAB);
                                const uint64_t db = smem_desc_k_sw128(ka + sl * SLAB);
#pragma unroll
                                for (int k = 0; k < 4; ++k) umma_pair_ss(d, da + 2 * k, db + 2 * k, idesc_s, (sl | k) != 0);
                            }
                            umma_pair_commit(&sh->k_empty[h]);
                            if (h == 1) umma_pair_commit(&sh->s_ready[j & 1]);
                        }
                        __syncwarp();
                    }
                    if (!ok) break;
                }
                if (j > 0) {
                    const int t = j - 1;
                    const bool last = t == n_tiles - 1;
                    const int n_k = last ? (n_last + 15) / 16 : 8;
                    ok = mbar_wait_warp(&sh->p_ready, t & 1, abort_flag);
                    if (!ok) break;
#pragma unroll
                    for (int nb = 0; nb < 2; ++nb) {
                        if (!(last && zero_tail)) ok = ok && mbar_wait_warp(&sh->v_full[nb], t & 1, abort_flag);
                        if (!ok) break;
                        tc_fence_after();
                        if (elect_one()) {
                            const uint64_t da0 = smem_desc_k_sw128(pa);
                            const uint64_t db0 = smem_desc_mn_sw128(va + (4 * nb) * SLAB, SLAB, 1024);
                            const uint32_t d = tmem_base + (uint32_t)nb * 128u;
                            auto product = [&](int k) {   // 16 tokens (descriptor addresses count 16-byte units)
                                umma_pair_ss(d, da0 + (k >> 2) * (SLAB / 16) + 2 * (k & 3), db0 + (k >> 2) * (2 * SLAB / 16) + (k & 3) * 128,
                                             idesc_o, (t | k) != 0);
                            };
                            if (n_k == 8) {
#pragma unroll
                                for (int k = 0; k < 8; ++k) product(k);
                            } else {
#pragma unroll 1
                                for (int k = 0; k < n_k; ++k) product(k);
                            }
                            umma_pair_commit(&sh->v_empty[nb]);
                            if (nb == 1) umma_pair_commit(&sh->o_done[t & 1]);
                        }
                        __syncwarp();
                    }
                    if (!ok) break;
                }
            }
        } else if (warp >= 4) {
            // ---------------- softmax: thread = (row, token quarter); the quarter's 32 tokens are half `half`, columns 32 w
            if (shared_seg) pdl_wait();
            const int w = (warp - 4) >> 2, q = warp & 3;
            const int row = 32 * (q & 1) + lane, half = q >> 1;
            const int quarter = 2 * half + w;
            const uint32_t lane_base = (uint32_t)(32 * q) << 16;
            const uint32_t p_bar = cluster_map(&sh->p_ready, 0);
            uint8_t* p_row = sP + half * SLAB + row * 128;
            float m_ref = -INFINITY;      // log2 units
            float l_part[2] = {0.f, 0.f};
            for (int j = 0; j < n_tiles; ++j) {
                const int n_valid = j == n_tiles - 1 ? n_last : TOK;
                const bool ok = __all_sync(0xffffffffu, *abort_flag == 0 && mbar_wait(&sh->s_ready[j & 1], (j >> 1) & 1, abort_flag));
                uint32_t sr[32], pk[16];
                bool exceed = false;
                if (ok) {
                    tc_fence_after();
                    tmem_ld32(tmem_base + lane_base + 256u + (uint32_t)((j & 1) * 64 + 32 * w), sr);
                    tmem_ld_wait();
                    if (n_valid < 32 * quarter + 32) {
#pragma unroll
                        for (int c = 0; c < 32; ++c)
                            if (32 * quarter + c >= n_valid) sr[c] = 0xff800000u;
                    }
                    // probabilities against the current reference: final unless the CTA votes for a rescale
#pragma unroll
                    for (int c = 0; c < 32; c += 2) {
                        const float a0 = fmaf(__uint_as_float(sr[c]), p.scale_log2, -m_ref);
                        const float a1 = fmaf(__uint_as_float(sr[c + 1]), p.scale_log2, -m_ref);
                        exceed |= (a0 > kRescaleThreshold) | (a1 > kRescaleThreshold);
                        pk[c / 2] = pack_bf16(fast_exp2(a0), fast_exp2(a1));
                    }
                }
                if (vote_or(exceed)) {
                    float mx = -INFINITY;
                    if (ok) {
#pragma unroll
                        for (int c = 0; c < 32; ++c) mx = fmaxf(mx, __uint_as_float(sr[c]));
                    }
                    sh->red[quarter][row] = mx * p.scale_log2;
                    softmax_sync();
                    const float cm = fmaxf(fmaxf(sh->red[0][row], sh->red[1][row]), fmaxf(sh->red[2][row], sh->red[3][row]));
                    const float m_new = fmaxf(m_ref, cm);
                    const float f = (m_new == -INFINITY) ? 1.f : fast_exp2(m_ref - m_new);
                    m_ref = m_new;
                    l_part[0] *= f;
                    l_part[1] *= f;
                    if (j > 0) {
                        // this thread's lane of O (the same row), 128 of its 256 columns, once the previous tile's product has
                        // landed
                        if (*abort_flag == 0) mbar_wait(&sh->o_done[(j - 1) & 1], ((j - 1) >> 1) & 1, abort_flag);
                        __syncwarp();
                        tc_fence_after();
#pragma unroll 1
                        for (int i = 0; i < 4; ++i) {
                            uint32_t orr[32];
                            const uint32_t o_addr = tmem_base + lane_base + (uint32_t)(128 * w + 32 * i);
                            tmem_ld32(o_addr, orr);
                            tmem_ld_wait();
#pragma unroll
                            for (int c = 0; c < 32; ++c) orr[c] = __float_as_uint(__uint_as_float(orr[c]) * f);
                            tmem_st32(o_addr, orr);
                        }
                        tmem_st_wait();
                    }
                    if (ok) {
#pragma unroll
                        for (int c = 0; c < 32; c += 2)
                            pk[c / 2] = pack_bf16(fast_exp2(fmaf(__uint_as_float(sr[c]), p.scale_log2, -m_ref)),
                                                  fast_exp2(fmaf(__uint_as_float(sr[c + 1]), p.scale_log2, -m_ref)));
                    }
                }
                if (ok) {
                    // row sums of the rounded values; then P, once the previous tile's product has read its buffer
#pragma unroll
                    for (int c = 0; c < 16; ++c) {
                        l_part[0] += __uint_as_float(pk[c] << 16);
                        l_part[1] += __uint_as_float(pk[c] & 0xffff0000u);
                    }
                    if (j > 0) mbar_wait(&sh->o_done[(j - 1) & 1], ((j - 1) >> 1) & 1, abort_flag);
#pragma unroll
                    for (int c = 0; c < 4; ++c)
                        *reinterpret_cast<uint4*>(p_row + (((4 * w + c) ^ (row & 7)) * 16)) =
                            make_uint4(pk[4 * c], pk[4 * c + 1], pk[4 * c + 2], pk[4 * c + 3]);
                    if (zero_tail && j == n_tiles - 1) {
                        // own half of the second operand: token rows n_last .. next multiple of 16, 4 slabs of 128 bytes each
                        mbar_wait(&sh->v_tail, 0, abort_flag);
                        const int n_rows16 = 16 - (n_last & 15);
                        for (int i = threadIdx.x - 128; i < n_rows16 * 32; i += 256) {
                            const int t = n_last + (i >> 5), sl = (i >> 3) & 3, c16 = i & 7;
                            uint8_t* at = sV + (4 * (sl >> 1) + 2 * (t >> 6) + (sl & 1)) * SLAB + (t & 63) * 128 + c16 * 16;
                            *reinterpret_cast<uint4*>(at) = make_uint4(0, 0, 0, 0);
                        }
                    }
                }
                fence_proxy_async();
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive_cluster(p_bar);
            }

            // ---------------- epilogue: row sums, normalised partial, LSE
            bool staged = false;
            if (!vote_or(*abort_flag != 0)) {
                sh->red[quarter][row] = l_part[0] + l_part[1];
                softmax_sync();
                const float l = sh->red[0][row] + sh->red[1][row] + sh->red[2][row] + sh->red[3][row];
                const float inv = 1.f / l;
                const int r = 64 * (int)rank + row;
                const bool direct = p.o_lat_direct != nullptr;
                if (quarter == 0 && r < n_rows) {
                    const float lse = (m_ref + log2f(l)) * kLn2;
                    if (direct) p.lse_direct[row0 + r] = lse;
                    else p.lse_part[(int64_t)chunk * p.B * p.H + row0 + r] = lse;
                }
                const bool ok = __all_sync(0xffffffffu, mbar_wait(&sh->o_done[(n_tiles - 1) & 1], ((n_tiles - 1) >> 1) & 1, abort_flag));
                tc_fence_after();
                if (ok) {
                    // The normalised rows are staged over the K and V tiles, which no product reads any more, as 128-byte
                    // swizzled boxes of 64 rows and leave with tiled stores (which cut off rows past the tensor's end).
                    // This thread's columns are latent dims 256 half + 128 w + 0 .. 127.
#pragma unroll 1
                    for (int i = 0; i < 4; ++i) {
                        uint32_t orr[32];
                        tmem_ld32(tmem_base + lane_base + (uint32_t)(128 * w + 32 * i), orr);
                        tmem_ld_wait();
                        if (direct) {
                            uint8_t* box = sK + (2 * quarter + (i >> 1)) * SLAB + row * 128;
#pragma unroll
                            for (int c = 0; c < 4; ++c) {
                                uint4 v;
                                uint32_t* vv = reinterpret_cast<uint32_t*>(&v);
#pragma unroll
                                for (int e = 0; e < 4; ++e) {
                                    const uint32_t* x = orr + 8 * c + 2 * e;
                                    vv[e] = pack_bf16(__uint_as_float(x[0]) * inv, __uint_as_float(x[1]) * inv);
                                }
                                *reinterpret_cast<uint4*>(box + (((4 * (i & 1) + c) ^ (row & 7)) * 16)) = v;
                            }
                        } else {
                            uint8_t* box = sK + (4 * quarter + i) * SLAB + row * 128;
#pragma unroll
                            for (int c = 0; c < 8; ++c) {
                                const float4 v = make_float4(__uint_as_float(orr[4 * c]) * inv, __uint_as_float(orr[4 * c + 1]) * inv,
                                                             __uint_as_float(orr[4 * c + 2]) * inv, __uint_as_float(orr[4 * c + 3]) * inv);
                                *reinterpret_cast<float4*>(box + ((c ^ (row & 7)) * 16)) = v;
                            }
                        }
                    }
                    fence_proxy_async();
                    staged = true;
                }
            }
            softmax_sync();
            // one thread issues the stores; a wait that gave up has set the flag, and nothing is stored
            if (threadIdx.x == 128 && staged && !*abort_flag && 64 * (int)rank < n_rows) {
                const CUtensorMap* to = shared_seg ? &tm_o_sh : &tm_o_sf;
                const int y = (shared_seg && p.stacked ? row0 : 0) + 64 * (int)rank;
                const int z = shared_seg && p.stacked ? 0 : row0 / p.H;
                const int n_box = p.o_lat_direct != nullptr ? 8 : 16;
                for (int i = 0; i < n_box; ++i) tma_store_4d(to, sK + i * SLAB, i * 64, y, z, p.o_lat_direct != nullptr ? 0 : chunk);
                bulk_commit();
                bulk_wait_read();   // the staging buffer must outlive the copy; the kernel end publishes the writes
            }
        } else {
            // warp 1 of the odd CTA, warp 3
            if (shared_seg) pdl_wait();
            if (warp == 3) {
                // The output projection behind this kernel reads W_UV (131 KB per head, cold after a long step): every CTA
                // requests its share into L2.
                const uint64_t at = ((uint64_t)blockIdx.x * 32u + (uint32_t)lane) * p.l2_bytes;
                if (at < p.l2_total)
                    asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;\n" ::"l"(p.l2_base + at),
                                 "r"(min(p.l2_bytes, p.l2_total - (uint32_t)at)) : "memory");
            }
        }
    } else {
        if (shared_seg) pdl_wait();
        // empty chunk: weight zero in the merge (a request without any latent token: zero latent output)
        const int r = 64 * (int)rank + (int)threadIdx.x - 128;
        if (warp >= 4 && threadIdx.x < 192 && r < n_rows) {
            if (p.o_lat_direct) {
                p.lse_direct[row0 + r] = -INFINITY;
                for (int l = 0; l < 512; l += 8)
                    *reinterpret_cast<uint4*>(p.o_lat_direct + (int64_t)(row0 + r) * 512 + l) = make_uint4(0, 0, 0, 0);
            } else {
                p.lse_part[(int64_t)chunk * p.B * p.H + row0 + r] = -INFINITY;
            }
        }
    }

    if (bad_page && lane == 0 && p.status) atomicOr(p.status, 0x100);
    tc_fence_before();
    __syncthreads();
    if (*abort_flag) {
        // A wait gave up.  Before the shared memory is released the copies in flight are awaited (with a limit): the even CTA's
        // barriers count those of both CTAs, and neither CTA leaves before the other (the cluster barrier below).
        if ((warp == 0 || warp == 2) && issued > 0) {
            const uint32_t par = (uint32_t)(issued - 1) & 1u;
            if (rank == 0)
                for (int h = 0; h < 2; ++h) mbar_drain(warp == 0 ? &sh->k_full[h] : &sh->v_full[h], par);
            if (rank == 0 && warp == 0) mbar_drain(&sh->q_full, 0);
            if (warp == 2 && zero_tail && issued == n_tiles) mbar_drain(&sh->v_tail, 0);
        }
        if (threadIdx.x == 0 && p.status) atomicOr(p.status, 3);
    }
    __syncwarp();
    cluster_sync();
    if (warp == 1) tmem_dealloc_pair(tmem_base, 512);
}

// [dims 64 | tokens of a page | latent slab | page], so that a box of several slabs is one copy
cudaError_t make_pair_kv_tmaps(const void* ckv, const void* kpe, int64_t ckv_stride, int64_t kpe_stride, int page_size,
                               uint64_t n_pages, CUtensorMap* tm_ckv, CUtensorMap* tm_kpe) {
    {
        uint64_t dims[4] = {64, (uint64_t)page_size, 8, n_pages};
        uint64_t str[3] = {(uint64_t)ckv_stride * 2, 128, (uint64_t)page_size * ckv_stride * 2};
        uint32_t box[4] = {64, 64, 2, 1};
        cudaError_t e = make_tmap_bf16(tm_ckv, ckv, 4, dims, str, box);
        if (e != cudaSuccess) return e;
    }
    uint64_t dims[3] = {64, (uint64_t)page_size, n_pages};
    uint64_t str[2] = {(uint64_t)kpe_stride * 2, (uint64_t)page_size * kpe_stride * 2};
    uint32_t box[3] = {64, 64, 1};
    return make_tmap_bf16(tm_kpe, kpe, 3, dims, str, box);
}
// Output rows as [512 values | rows | groups | chunks]; fp32 values are described as pairs of 16-bit elements.
cudaError_t make_out_tmap(CUtensorMap* tm, const void* base, bool fp32, int64_t rows, int64_t groups, int64_t chunks) {
    const uint64_t w = fp32 ? 1024 : 512;
    uint64_t dims[4] = {w, (uint64_t)rows, (uint64_t)groups, (uint64_t)chunks};
    uint64_t str[3] = {w * 2, (uint64_t)rows * w * 2, (uint64_t)(rows * groups) * w * 2};
    uint32_t box[4] = {64, 64, 1, 1};
    return make_tmap_bf16(tm, base, 4, dims, str, box);
}

}  // namespace

cudaError_t set_attrs_absorb_pair_sm100() {
    return cudaFuncSetAttribute(absorb_pair_sm100_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kPairSmem);
}

cudaError_t launch_absorb_pair_sm100(const AbsorbAttn& a, int64_t Ls_pad, void* o_lat_direct, float* lse_direct, int* status,
                                     cudaStream_t s) {
    const int n_chunks = a.n_shared_chunks + a.n_suffix_chunks;
    if (a.B <= 0 || n_chunks <= 0) return cudaSuccess;
    if (a.chunk % TOK != 0 || a.H > 128) return cudaErrorInvalidValue;
    const int64_t rows = (int64_t)a.B * a.H;
    CUtensorMap tm_qa, tm_qp, tm_ckv_sh, tm_kpe_sh, tm_ckv_pg, tm_kpe_pg, tm_o_sh, tm_o_sf;
    {   // the queries as one [B * H, 512] matrix; rows past the end read as zeros
        uint64_t dims[2] = {512, (uint64_t)rows};
        uint64_t str[1] = {512 * 2};
        uint32_t box[2] = {64, 64};
        cudaError_t e = make_tmap_bf16(&tm_qa, a.q_abs, 2, dims, str, box);
        if (e != cudaSuccess) return e;
        dims[0] = 64;
        str[0] = 64 * 2;
        e = make_tmap_bf16(&tm_qp, a.q_pe, 2, dims, str, box);
        if (e != cudaSuccess) return e;
    }
    if (a.n_shared_chunks > 0) {
        cudaError_t e = make_pair_kv_tmaps(a.ckv_shared, a.kpe_shared, 512, 64, 64, (uint64_t)(Ls_pad / 64), &tm_ckv_sh, &tm_kpe_sh);
        if (e != cudaSuccess) return e;
    }
    if (a.n_suffix_chunks > 0) {
        // the maps end at the caller's last physical page: anything past it reads as zeros
        cudaError_t e = make_pair_kv_tmaps(a.ckv_pages, a.kpe_pages, a.ckv_stride, a.kpe_stride, a.page_size,
                                           (uint64_t)std::max(a.num_pages, 1), &tm_ckv_pg, &tm_kpe_pg);
        if (e != cudaSuccess) return e;
    }
    if (a.n_shared_chunks == 0) { tm_ckv_sh = tm_ckv_pg; tm_kpe_sh = tm_kpe_pg; }
    if (a.n_suffix_chunks == 0) { tm_ckv_pg = tm_ckv_sh; tm_kpe_pg = tm_kpe_sh; }
    const bool direct = n_chunks == 1;
    const void* o = direct ? o_lat_direct : a.o_part;
    cudaError_t e = make_out_tmap(&tm_o_sf, o, !direct, a.H, a.B, n_chunks);
    if (e == cudaSuccess && a.stacked) e = make_out_tmap(&tm_o_sh, o, !direct, rows, 1, n_chunks);
    if (e != cudaSuccess) return e;
    if (!a.stacked) tm_o_sh = tm_o_sf;
    PairParams p{};
    p.B = a.B; p.H = a.H;
    p.chunk = a.chunk; p.n_shared_chunks = a.n_shared_chunks; p.n_suffix_chunks = a.n_suffix_chunks;
    p.stacked = a.stacked ? 1 : 0;
    p.shared_groups = a.stacked ? (int)((rows + 127) / 128) : a.B;
    p.Ls_absorb = a.Ls_absorb;
    p.page_size = a.page_size; p.max_pages = a.max_pages; p.num_pages = a.num_pages;
    p.block_table = a.block_table; p.seq_lens = a.seq_lens; p.order = a.order;
    p.desc = reinterpret_cast<const int4*>(a.desc);
    p.scale_log2 = a.scale * kLog2e;
    p.lse_part = a.lse_part; p.status = status;
    p.o_lat_direct = direct ? reinterpret_cast<__nv_bfloat16*>(o_lat_direct) : nullptr;
    p.lse_direct = lse_direct;
    dim3 grid(2 * (a.n_shared_chunks * p.shared_groups + a.n_suffix_chunks * a.B), 1, 1);
    p.l2_base = reinterpret_cast<const char*>(a.w_uv);
    p.l2_total = a.w_uv ? (uint32_t)a.H * 128u * 512u * 2u : 0u;
    p.l2_bytes = (p.l2_total / (grid.x * 32u) / 16u + 1u) * 16u;
    return launch_pdl(absorb_pair_sm100_kernel, grid, dim3(384), kPairSmem, s, tm_qa, tm_qp, tm_ckv_sh, tm_kpe_sh, tm_ckv_pg,
                      tm_kpe_pg, tm_o_sh, tm_o_sf, p);
}

}  // namespace tmla
