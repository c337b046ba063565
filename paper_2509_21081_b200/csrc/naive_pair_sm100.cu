// Naive shared-prefix attention (Algorithm 1 line 4) for more than 128 query rows: a pair of CTAs on one product.
//
//     S = Q_h [256 rows, 192] * [K_nope_h | k_pe]^T [192, 128 tokens],  O += P [256, 128 tokens] * V_h [128 tokens, 128]
//
// Work item (CTA pair) = (tile range, group of 256 query rows); the ranges, segments and partial slots are those of
// naive_attn_sm100.cu, which takes up to 128 rows and the 8-bit cache.  Each CTA of the pair holds 128 query rows and their
// accumulators (tensor memory: lane = row) and brings half of every tile: 64 tokens of K (24 KB) and 64 dims of V (16 KB).
//
// Why a pair: with both operands in shared memory an SM's 128 B/clock are as busy as its tensor core when it loads whole tiles for
// its own rows; half tiles cut the reads of a tile from 96 to 72 KB for the logits and from 32 to 16 KB for the output, and leave
// room for three tiles in flight (instead of two of K and one of V) and the next segment's query tile.
//
// Why one accumulator and three logits buffers: the two softmax warpgroups take alternate tiles of the SAME rows against one
// reference exponent per row, which the warp with a tile hands to the warp with the next one (lazy: it is raised only when a
// logit exceeds it by more than 2^8, together with O).  S runs up to three tiles ahead of PV, so the chain S -> softmax -> PV of a
// tile overlaps those of its neighbours.  Both products are issued by one thread, in an order that needs no wait between the PV
// product that reads P from a buffer and the S product that overwrites it.  The softmax reads a tile's logits once: the
// probabilities of the first half wait in registers until the tile's maximum and the previous tile's reference are known.
//
// Measured (B200, 1024 rows x 16 heads over 16384 tokens, us per launch, in steps): two accumulators with one logits buffer each (one
// CTA for 256 rows, the form before) 162; this arrangement with two issuing threads and two passes over the logits 143; one pass 143;
// one issuing thread 139; one test for all barriers of a step, PV when all probabilities are there 129 = 1.33 PFLOP/s at the 1.6 GHz
// to which the power cap lowers the clock, which is what cuBLAS sustains: about 1650 clocks per tile, 1280 of them MMAs; the next
// segment's queries requested early and staged stores 126.  All eight
// softmax warps on one tile (64 logits per thread) took 161: nothing then hides the latencies of a tile's barriers and loads.
//
// Warp roles (384 threads per CTA): warp 0 loads Q and K, warp 2 V; in the even CTA warp 1 issues both products; warps 4-7 / 8-11
// softmax of the even / odd tiles (thread = query row).  Tensor memory: O 128 columns, S[b] at 128 + 128 b (P in bf16 overwrites
// its first 64).
#include <algorithm>
#include <cstddef>

#include "kernels.h"
#include "sm100.cuh"

namespace tmla {
namespace {

using namespace sm100;

constexpr int TOK = 128;
constexpr int Q_SLAB = 128 * 128, Q_BYTES = 3 * Q_SLAB;     // 128 rows: two nope slabs, one rope slab
constexpr int SLAB = 64 * 128, K_BYTES = 3 * SLAB;          // 64 tokens
constexpr int V_BYTES = 2 * SLAB;                           // 64 dims, two blocks of 64 tokens
constexpr int STAGES = 3;
constexpr int NQ = 2;                                       // query tiles: this segment's and the next one's
constexpr int NBUF = 3;                                     // logits buffers
// Pairs of exponentials computed on the FMA pipe instead of the special-function unit, by position within a group of eight: one in
// four (with the form before one in eight and three in eight gained less).
constexpr unsigned kPolyExpMask = 0x88u;

struct PairParams {
    int B, H, Ls, Ls_pad;
    int part_rows;
    int m_groups, n_tiles, n_ranges, per, rem, n_seg_max;   // as in naive_attn_sm100.cu
    float scale_log2;
    float* o_part;     // [n_slots][part_rows][H][128]
    float* lse_part;   // [n_slots][part_rows][H]
    int* status;
};

struct Barriers {
    uint64_t q_full[NQ], k_full[STAGES], v_full[STAGES];     // copies of both CTAs, counted in the even one
    uint64_t p_ready[NBUF], o_free;                          // softmax warps of both CTAs, counted in the even one
    uint64_t q_free[NQ];                                     // in both CTAs: the even one's commit, and both warpgroups (staging)
    uint64_t k_empty[STAGES], v_empty[STAGES], s_ready[NBUF];   // in both CTAs, by the even one's commits
    // Completion of PV product u goes to o_done[u & 3]: a waiter knows that product u - 4 has landed (its own latest tile is
    // u or u - 1, whose logits buffer was free), and a parity wait tells one outstanding completion from none.
    uint64_t o_done[4];
    uint32_t tmem_base;
    int abort_flag;
    float m_ref[2][128];                          // [segment & 1][row]: reference exponent (log2 units)
    float m_end[2][2][128], l_end[2][2][128];     // [segment & 1][warpgroup][row]: reference and row sum at the segment's end
};
constexpr int kSmem = NQ * Q_BYTES + STAGES * (K_BYTES + V_BYTES) + 1024 + (int)sizeof(Barriers);
static_assert(kSmem <= 232448, "shared memory of one SM");

struct Segment {
    int t0, cnt, h, slot_seg;
    bool last_of_col;
};

__device__ __forceinline__ void named_sync64(int id) { asm volatile("bar.sync %0, 64;\n" ::"r"(id) : "memory"); }
__device__ __forceinline__ void named_arrive64(int id) { asm volatile("bar.arrive %0, 64;\n" ::"r"(id) : "memory"); }

__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(384, 1)
naive_pair_sm100_kernel(const __grid_constant__ CUtensorMap tm_qn, const __grid_constant__ CUtensorMap tm_qp,
                        const __grid_constant__ CUtensorMap tm_kn, const __grid_constant__ CUtensorMap tm_kp,
                        const __grid_constant__ CUtensorMap tm_vt, const __grid_constant__ CUtensorMap tm_o, PairParams p) {
    extern __shared__ uint8_t smem_raw[];
    uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    uint8_t* sQ = smem;
    uint8_t* sK = sQ + NQ * Q_BYTES;
    uint8_t* sV = sK + STAGES * K_BYTES;
    Barriers* bar = reinterpret_cast<Barriers*>(sV + STAGES * V_BYTES);
    volatile int* abort_flag = &bar->abort_flag;

    const int warp = warp_index_uniform(), lane = threadIdx.x & 31;
    const int rank = (int)cluster_cta_rank();
    const int rng = (int)(blockIdx.x >> 1) / p.m_groups, grp = (int)(blockIdx.x >> 1) % p.m_groups;
    pdl_trigger();
    if (warp == 0) {
        uint64_t* all = &bar->q_full[0];
        constexpr int n_bars = (int)(offsetof(Barriers, tmem_base) / sizeof(uint64_t));
        for (int i = lane; i < n_bars; i += 32) {
            uint64_t* m = all + i;
            const bool probabilities = m >= &bar->p_ready[0] && m < &bar->o_free, queries = m >= &bar->q_free[0] && m < &bar->k_empty[0];
            mbar_init(m, m == &bar->o_free ? 16 : probabilities ? 8 : queries ? 3 : 1);
        }
        if (lane == 0) bar->abort_flag = 0;
        fence_mbar_init();
        __syncwarp();
    }
    if (warp == 1) tmem_alloc_pair(&bar->tmem_base, 512);
    if (warp == 2) {
        if (lane == 0) prefetch_tmap(&tm_qn);
        if (lane == 1) prefetch_tmap(&tm_qp);
        if (lane == 2) prefetch_tmap(&tm_kn);
        if (lane == 3) prefetch_tmap(&tm_kp);
        if (lane == 4) prefetch_tmap(&tm_vt);
    }
    tc_fence_before();
    cluster_sync();
    tc_fence_after();
    const uint32_t tmem_base = __shfl_sync(0xffffffffu, bar->tmem_base, 0);
    pdl_wait();      // nothing above touches global memory

    const int g_begin = rng * p.per + min(rng, p.rem);
    const int g_end = g_begin + p.per + (rng < p.rem ? 1 : 0);
    auto segment_at = [&](int g) {
        Segment s;
        s.h = g / p.n_tiles;
        s.t0 = g - s.h * p.n_tiles;
        s.cnt = min(p.n_tiles - s.t0, g_end - g);
        const int first_tile = s.h * p.n_tiles, big = p.rem * (p.per + 1);
        const int r_first = first_tile < big ? first_tile / (p.per + 1) : p.rem + (first_tile - big) / p.per;
        s.slot_seg = rng - r_first;
        s.last_of_col = s.t0 + s.cnt == p.n_tiles;
        return s;
    };
    // segments of different heads visit their tiles from different starting points (see naive_attn_sm100.cu)
    auto tile_of = [&](const Segment& s, int e) {
        const int rot = (int)(((unsigned)s.h * 37u + (unsigned)s.slot_seg * 11u) % (unsigned)s.cnt);
        const int t = e + rot;
        return s.t0 + (t >= s.cnt ? t - s.cnt : t);
    };
    const int row0 = grp * 256 + rank * 128;

    int issued = 0, q_issued = 0;   // producer warps: copies issued, for the abort path
    if (warp == 0) {
        // ---------------- Q and K: this CTA's rows, tokens [64 rank, + 64) of every tile
        const uint32_t ld = elect_one() ? 1u : 0u, ld_even = rank == 0 ? ld : 0u;
        const uint32_t kf = cluster_map(&bar->k_full[0], 0), qf = cluster_map(&bar->q_full[0], 0);
        int ring = 0, seg = 0;
        bool ok = true;
        auto issue_q = [&](int g, int sg) {   // the query tile of segment sg, which begins at g
            const int h = g / p.n_tiles, buf = sg % NQ;
            uint8_t* dst = sQ + buf * Q_BYTES;
            if (sg >= NQ) ok = mbar_wait_warp(&bar->q_free[buf], ((sg / NQ) & 1) ^ 1, abort_flag);
            if (!ok) return;
            mbar_arrive_expect_tx_if(ld_even, &bar->q_full[buf], 2 * Q_BYTES);
            tma_load_3d_pair_if(ld, dst, &tm_qn, qf + 8u * buf, 0, h, row0);
            tma_load_3d_pair_if(ld, dst + Q_SLAB, &tm_qn, qf + 8u * buf, 64, h, row0);
            tma_load_3d_pair_if(ld, dst + 2 * Q_SLAB, &tm_qp, qf + 8u * buf, 0, h, row0);
            q_issued = sg + 1;
        };
        if (g_begin < g_end) issue_q(g_begin, 0);
        for (int g = g_begin; g < g_end && ok; ++seg) {
            const Segment s = segment_at(g);
            const int at = min(s.cnt - 1, STAGES);   // (by this tile the S products of the segment before are complete, or nearly so)
            for (int e = 0; e < s.cnt && ok; ++e, ++ring) {
                const int st = ring % STAGES;
                if (ring >= STAGES) ok = mbar_wait_warp(&bar->k_empty[st], ((ring / STAGES) & 1) ^ 1, abort_flag);
                if (!ok) break;
                const int blk = 2 * tile_of(s, e) + rank, gb = s.h * (p.Ls_pad / 64) + blk;
                uint8_t* dst = sK + st * K_BYTES;
                if (p.m_groups == 1 && e + STAGES + 1 < s.cnt) {
                    // One row group reads every tile from HBM, at the rate HBM delivers them: the tile after the ring's is
                    // requested into L2.
                    const int pb = s.h * (p.Ls_pad / 64) + 2 * tile_of(s, e + STAGES + 1) + rank;
                    tma_prefetch_3d_if(ld, &tm_kn, 0, 0, pb);
                    tma_prefetch_3d_if(ld, &tm_kn, 0, 64, pb);
                }
                mbar_arrive_expect_tx_if(ld_even, &bar->k_full[st], 2 * K_BYTES);
                tma_load_3d_pair_if(ld, dst, &tm_kn, kf + 8u * st, 0, 0, gb);
                tma_load_3d_pair_if(ld, dst + SLAB, &tm_kn, kf + 8u * st, 0, 64, gb);
                tma_load_2d_pair_if(ld, dst + 2 * SLAB, &tm_kp, kf + 8u * st, 0, blk * 64);
                issued = ring + 1;
                if (e == at && g + s.cnt < g_end) issue_q(g + s.cnt, seg + 1);
            }
            g += s.cnt;
        }
    } else if (warp == 2) {
        // ---------------- V: dims [64 rank, + 64) of every tile
        const uint32_t ld = elect_one() ? 1u : 0u, ld_even = rank == 0 ? ld : 0u;
        const uint32_t vf = cluster_map(&bar->v_full[0], 0);
        int ring = 0;
        bool ok = true;
        for (int g = g_begin; g < g_end && ok;) {
            const Segment s = segment_at(g);
            for (int e = 0; e < s.cnt && ok; ++e, ++ring) {
                const int st = ring % STAGES;
                if (ring >= STAGES) ok = mbar_wait_warp(&bar->v_empty[st], ((ring / STAGES) & 1) ^ 1, abort_flag);
                if (!ok) break;
                if (p.m_groups == 1 && e + STAGES + 1 < s.cnt)   // (see the K producer)
                    tma_prefetch_4d_if(ld, &tm_vt, 0, 64 * rank, 2 * tile_of(s, e + STAGES + 1), s.h);
                mbar_arrive_expect_tx_if(ld_even, &bar->v_full[st], 2 * V_BYTES);
                tma_load_4d_pair_if(ld, sV + st * V_BYTES, &tm_vt, vf + 8u * st, 0, 64 * rank, 2 * tile_of(s, e), s.h);
                issued = ring + 1;
            }
            g += s.cnt;
        }
    } else if (warp == 1 && rank == 0) {
        // ---------------- both products, from one thread: the tensor core runs them in the order of issue, so S of tile e + 3 may
        // follow PV of tile e, which reads P from the same buffer, without a wait for its completion
        constexpr uint32_t idesc_s = idesc_bf16(256, TOK, false, false), idesc_o = idesc_bf16(256, 128, false, false);
        const int n_total = g_end - g_begin;
        Segment ss = segment_at(g_begin), sp = ss;    // segments of the next S product and of the next PV product,
        int seg_s = 0, e_s = 0, seg_p = 0, e_p = 0;   // their numbers, and the tile within the segment
        int un = 0;                                   // next S product
        bool ok = true, k_here = false;               // k_here: the K tile of S product un is known to have landed
        for (int t = 0; t < n_total && ok; ++t) {
            // S up to NBUF tiles ahead of PV, and not into a segment whose query tile takes the place of one that is still in use:
            // segment seg_p's is given back by its epilogue, after its last PV product
            while (un < n_total && un < t + NBUF && seg_s - seg_p < NQ) {
                const int st = un % STAGES, b = un % NBUF;
                if (!k_here) ok = mbar_wait_warp(&bar->k_full[st], (un / STAGES) & 1, abort_flag);
                if (ok && e_s == 0) ok = mbar_wait_warp(&bar->q_full[seg_s % NQ], (seg_s / NQ) & 1, abort_flag);
                if (!ok) break;
                k_here = false;
                tc_fence_after();
                if (elect_one()) {
                    const uint32_t qa = smem_u32(sQ + (seg_s % NQ) * Q_BYTES), ka = smem_u32(sK + st * K_BYTES);
                    const uint32_t d = tmem_base + 128u + (uint32_t)b * 128u;
#pragma unroll
                    for (int sl = 0; sl < 3; ++sl) {
                        const uint64_t da = smem_desc_k_sw128(qa + sl * Q_SLAB), db = smem_desc_k_sw128(ka + sl * SLAB);
#pragma unroll
                        for (int k = 0; k < 4; ++k) umma_pair_ss(d, da + 2 * k, db + 2 * k, idesc_s, (sl | k) != 0);
                    }
                    umma_pair_commit(&bar->s_ready[b]);
                    umma_pair_commit(&bar->k_empty[st]);
                    if (e_s == ss.cnt - 1) umma_pair_commit(&bar->q_free[seg_s % NQ]);   // the Q tile may be replaced
                }
                __syncwarp();
                ++un;
                if (++e_s == ss.cnt) {
                    ++seg_s;
                    e_s = 0;
                    if (un < n_total) ss = segment_at(g_begin + un);
                }
            }
            if (!ok) break;
            // (the barriers of a step are tested together: a test takes some 200 clocks even when its phase is complete.  The next
            // K tile's only where its S product may be issued whatever this PV product does: the K producer stops at a query
            // tile that has no place yet.)
            const int st = t % STAGES, b = t % NBUF;
            uint64_t* const vf = &bar->v_full[st];
            uint64_t* const pr = &bar->p_ready[b];
            if (un < n_total && !k_here && seg_s - seg_p < NQ) {
                ok = mbar_wait3_warp(&bar->k_full[un % STAGES], (un / STAGES) & 1, vf, (t / STAGES) & 1, pr, (t / NBUF) & 1, abort_flag);
                k_here = true;
            } else {
                ok = mbar_wait2_warp(vf, (t / STAGES) & 1, pr, (t / NBUF) & 1, abort_flag);
            }
            if (ok && e_p == 0 && seg_p > 0) ok = mbar_wait_warp(&bar->o_free, (seg_p - 1) & 1, abort_flag);   // epilogue has read O
            if (!ok) break;
            tc_fence_after();
            if (elect_one()) {
                const uint32_t pa = tmem_base + 128u + (uint32_t)b * 128u;
                const uint64_t db = smem_desc_k_sw128(smem_u32(sV + st * V_BYTES));
#pragma unroll
                for (int k = 0; k < 8; ++k)
                    umma_pair_ts(tmem_base, pa + 8 * k, db + (k >> 2) * (SLAB / 16) + 2 * (k & 3), idesc_o, (e_p | k) != 0);
                // o_done last: the odd CTA waits for it before it leaves, not for the v_empty of its last tiles
                umma_pair_commit(&bar->v_empty[st]);
                umma_pair_commit(&bar->o_done[t & 3]);
            }
            __syncwarp();
            if (++e_p == sp.cnt) {
                ++seg_p;
                e_p = 0;
                if (t + 1 < n_total) sp = segment_at(g_begin + t + 1);
            }
        }
    } else if (warp >= 4) {
        // ---------------- softmax.  The loops run to their end whatever happens (a wait that gave up only skips work), so that the
        // named barriers between the two warps of the same rows always match.
        const int i = (warp - 4) >> 2, w = warp & 3;
        const int r = 32 * w + lane;
        const uint32_t lane_base = (uint32_t)(32 * w) << 16;
        const int b_row = row0 + r;
        const bool warp_has_rows = row0 + 32 * w < p.B;
        const uint32_t p_ready = cluster_map(&bar->p_ready[0], 0), o_free = cluster_map(&bar->o_free, 0);
        const uint64_t scale2 = pack_f32x2(p.scale_log2, p.scale_log2);
        int ring_base = 0, segi = 0;
        for (int g = g_begin; g < g_end; ++segi) {
            const Segment s = segment_at(g);
            float m_ref = -INFINITY;
            uint64_t l_a = pack_f32x2(0.f, 0.f), l_b = pack_f32x2(0.f, 0.f);
            for (int e = (ring_base ^ i) & 1; e < s.cnt; e += 2) {
                const int u = ring_base + e, buf = u % NBUF;
                const bool ok = __all_sync(0xffffffffu, *abort_flag == 0 && mbar_wait(&bar->s_ready[buf], (u / NBUF) & 1, abort_flag));
                tc_fence_after();
                if (!warp_has_rows) {   // padding past B: the P rows may hold anything, only keep in step
                    tc_fence_before();
                    __syncwarp();
                    if (lane == 0) mbar_arrive_cluster(p_ready + 8u * buf);
                    continue;
                }
                const uint32_t s_addr = tmem_base + lane_base + 128u + (uint32_t)buf * 128u;
                const int valid = min(TOK, p.Ls - tile_of(s, e) * TOK);
                uint32_t sr[2][32], pk[2][16];
                auto load64 = [&](int col) {   // logits of columns [col, + 64), past the end -inf
                    tmem_ld32(s_addr + (uint32_t)col, sr[0]);
                    tmem_ld32(s_addr + (uint32_t)col + 32u, sr[1]);
                };
                auto mask64 = [&](int col) {
                    if (valid < TOK) {
#pragma unroll
                        for (int c = 0; c < 64; ++c)
                            if (col + c >= valid) sr[c >> 5][c & 31] = 0xff800000u;
                    }
                };
                float mx4[4] = {-INFINITY, -INFINITY, -INFINITY, -INFINITY};   // (four running maxima: short dependent chains)
                auto max32 = [&](const uint32_t (&src)[32]) {
#pragma unroll
                    for (int c = 0; c < 16; ++c)
                        mx4[c & 3] = max3(mx4[c & 3], __uint_as_float(src[2 * c]), __uint_as_float(src[2 * c + 1]));
                };
                // p = 2^(s * scale - m_ref) of 32 logits, packed to bf16, and their sums
                uint64_t sum_a = pack_f32x2(0.f, 0.f), sum_b = pack_f32x2(0.f, 0.f);
                auto probs32 = [&](const uint32_t (&src)[32], uint32_t (&dst)[16]) {
                    const uint64_t neg_m2 = pack_f32x2(-m_ref, -m_ref);
#pragma unroll
                    for (int c = 0; c < 16; ++c) {
                        float x0, x1, p0, p1;
                        const uint64_t logits = pack_f32x2(__uint_as_float(src[2 * c]), __uint_as_float(src[2 * c + 1]));
                        unpack_f32x2(fma_f32x2(logits, scale2, neg_m2), x0, x1);
                        if ((kPolyExpMask >> (c & 7)) & 1) {
                            exp2_poly_x2(x0, x1, p0, p1);
                        } else {
                            p0 = fast_exp2(x0);
                            p1 = fast_exp2(x1);
                        }
                        dst[c] = pack_bf16(p0, p1);
                        if (c & 1) sum_b = add_f32x2(sum_b, pack_f32x2(p0, p1));
                        else sum_a = add_f32x2(sum_a, pack_f32x2(p0, p1));
                    }
                };
                // One pass over the logits, against the reference this warp knows.  The first 64 probabilities stay in registers
                // (they would overwrite logits) until the whole tile's maximum and the previous tile's reference are known.  The
                // segment's first tile sets the reference; the other warpgroup's first tile waits for it.
                load64(0);
                float m_prev = -INFINITY;
                if (e == 1) {
                    named_sync64(1 + 2 * w + (u & 1));
                    m_ref = m_prev = bar->m_ref[segi & 1][r];
                }
                tmem_ld_wait();
                mask64(0);
                max32(sr[0]);
                max32(sr[1]);
                if (e > 0) {
                    probs32(sr[0], pk[0]);
                    tmem_ld32(s_addr + 64u, sr[0]);
                    probs32(sr[1], pk[1]);
                    tmem_ld32(s_addr + 96u, sr[1]);
                } else {
                    load64(64);
                }
                tmem_ld_wait();
                mask64(64);
                max32(sr[0]);
                max32(sr[1]);
                const float mx = fmaxf(fmaxf(mx4[0], mx4[1]), fmaxf(mx4[2], mx4[3])) * p.scale_log2;
                // hand-over of the reference exponent: from the warp with the previous tile, to the one with the next
                if (e > 1) {
                    named_sync64(1 + 2 * w + (u & 1));
                    m_prev = bar->m_ref[segi & 1][r];
                }
                const bool grow = e == 0 || mx > m_prev + 8.f;
                const float m_new = grow ? mx : m_prev;
                const bool redo = __any_sync(0xffffffffu, m_new != m_ref);
                if (redo) bar->m_ref[segi & 1][r] = m_new;
                if (e + 1 < s.cnt) named_arrive64(1 + 2 * w + ((u + 1) & 1));
                if (redo) {
                    if (e > 0 && __any_sync(0xffffffffu, grow)) {
                        // O is rescaled once the previous tile's product has landed; this tile's and later ones wait for p_ready below
                        if (*abort_flag == 0) mbar_wait(&bar->o_done[(u - 1) & 3], ((u - 1) >> 2) & 1, abort_flag);
                        __syncwarp();
                        tc_fence_after();
                        const float f = fast_exp2(m_prev - m_new);
#pragma unroll 1
                        for (int c = 0; c < 4; ++c) {
                            tmem_ld32(tmem_base + lane_base + c * 32, sr[0]);
                            tmem_ld_wait();
#pragma unroll
                            for (int q = 0; q < 32; ++q) sr[0][q] = __float_as_uint(__uint_as_float(sr[0][q]) * f);
                            tmem_st32(tmem_base + lane_base + c * 32, sr[0]);
                        }
                        tmem_st_wait();
                    }
                    // this warpgroup's sums so far are relative to its last reference; the first half again
                    const float f = fast_exp2(m_ref - m_new);
                    l_a = mul_f32x2(l_a, pack_f32x2(f, f));
                    l_b = mul_f32x2(l_b, pack_f32x2(f, f));
                    m_ref = m_new;
                    sum_a = sum_b = pack_f32x2(0.f, 0.f);
                    load64(0);
                    tmem_ld_wait();
                    mask64(0);
                    probs32(sr[0], pk[0]);
                    probs32(sr[1], pk[1]);
                    load64(64);
                    tmem_ld_wait();
                    mask64(64);
                }
                tmem_st16(s_addr, pk[0]);
                tmem_st16(s_addr + 16u, pk[1]);
                probs32(sr[0], pk[0]);
                tmem_st16(s_addr + 32u, pk[0]);
                probs32(sr[1], pk[1]);
                tmem_st16(s_addr + 48u, pk[1]);
                tmem_st_wait();
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive_cluster(p_ready + 8u * buf);
                l_a = add_f32x2(l_a, sum_a);
                l_b = add_f32x2(l_b, sum_b);
            }
            // ---- segment epilogue: normalised partial + LSE into this segment's slot, 64 of the 128 columns per warpgroup
            float la, lc;
            unpack_f32x2(add_f32x2(l_a, l_b), la, lc);
            bar->m_end[segi & 1][i][r] = m_ref;
            bar->l_end[segi & 1][i][r] = la + lc;
            named_sync64(9 + w);
            // (warps without rows wait as well: o_free of this segment must not be reached before that of the last one is complete)
            const int u_last = ring_base + s.cnt - 1;
            const bool ok = __all_sync(0xffffffffu, *abort_flag == 0 && mbar_wait(&bar->o_done[u_last & 3], (u_last >> 2) & 1, abort_flag));
            tc_fence_after();
            float inv = 0.f;
            if (warp_has_rows) {
                const float m0 = bar->m_end[segi & 1][0][r], m1 = bar->m_end[segi & 1][1][r];
                const float m = fmaxf(m0, m1);   // the latest reference, which O is relative to
                const float l = bar->l_end[segi & 1][0][r] * fast_exp2(m0 - m) + bar->l_end[segi & 1][1][r] * fast_exp2(m1 - m);
                inv = 1.f / l;
                const int64_t at = ((int64_t)s.slot_seg * p.part_rows + b_row) * p.H + s.h;
                if (i == 0 && b_row < p.B) {
                    p.lse_part[at] = (m + log2f(l)) * kLn2;
                    if (s.last_of_col)   // the segment that ends a head marks the head's unused slots as empty
                        for (int ss = s.slot_seg + 1; ss < p.n_seg_max; ++ss)
                            p.lse_part[((int64_t)ss * p.part_rows + b_row) * p.H + s.h] = -INFINITY;
                }
            }
            // The rows leave as boxes of 128 rows x 32 values, staged in this segment's query tile (no product reads it any more; q_free
            // waits for this) with 128-byte swizzled rows, and tiled stores, which cut off rows past B.  (A row of a partial is 512
            // bytes, the next one H times as far: the threads' own stores take 16 bytes of 32 rows per instruction.  Expansion-only steps,
            // us, with those / staged: 130 rows x 128 heads over 1000 tokens 47.9 / 35.9, 700 x 128 over 500 86.8 / 75.2, 166 x 16
            // over 7069 30.5 / 26.1.)
#pragma unroll 1
            for (int c = 0; c < 2; ++c) {
                uint8_t* box = sQ + (segi % NQ) * Q_BYTES + i * 16384;
                if (warp_has_rows) {
                    uint32_t orr[32];
                    tmem_ld32(tmem_base + lane_base + (uint32_t)(64 * i + 32 * c), orr);
                    tmem_ld_wait();
#pragma unroll
                    for (int q = 0; q < 8; ++q)
                        *reinterpret_cast<float4*>(box + r * 128 + ((q ^ (r & 7)) * 16)) =
                            make_float4(__uint_as_float(orr[4 * q]) * inv, __uint_as_float(orr[4 * q + 1]) * inv,
                                        __uint_as_float(orr[4 * q + 2]) * inv, __uint_as_float(orr[4 * q + 3]) * inv);
                    fence_proxy_async();
                }
                if (c == 1) {   // O has been read
                    tc_fence_before();
                    __syncwarp();
                    if (lane == 0) mbar_arrive_cluster(o_free);
                }
                asm volatile("bar.sync %0, 128;\n" ::"r"(13 + i) : "memory");
                if (w == 0 && lane == 0) {
                    if (row0 < p.B && *abort_flag == 0) {
                        tma_store_4d(&tm_o, box, 2 * (64 * i + 32 * c), s.h, row0, s.slot_seg);
                        bulk_commit();
                        bulk_wait_read();
                    }
                    if (c == 1) mbar_arrive(&bar->q_free[segi % NQ]);
                }
                if (c == 0) asm volatile("bar.sync %0, 128;\n" ::"r"(13 + i) : "memory");   // the box may be written again
            }
            ring_base += s.cnt;
            g += s.cnt;
        }
    }

    tc_fence_before();
    __syncthreads();
    if (*abort_flag) {
        // A wait gave up.  Before the shared memory is released the copies in flight are awaited (with a limit): the even CTA's
        // barriers count those of both CTAs, and neither CTA leaves before the other (the cluster barrier below).
        if (rank == 0 && (warp == 0 || warp == 2)) {
            for (int pos = max(0, issued - STAGES); pos < issued; ++pos)
                mbar_drain(warp == 0 ? &bar->k_full[pos % STAGES] : &bar->v_full[pos % STAGES], (pos / STAGES) & 1);
            for (int sg = max(0, q_issued - NQ); warp == 0 && sg < q_issued; ++sg) mbar_drain(&bar->q_full[sg % NQ], (sg / NQ) & 1);
        }
        if (threadIdx.x == 0 && p.status) atomicOr(p.status, 2);
    }
    __syncwarp();
    cluster_sync();
    if (warp == 1) tmem_dealloc_pair(tmem_base, 512);
}

}  // namespace

cudaError_t set_attrs_naive_pair_sm100() {
    return cudaFuncSetAttribute(naive_pair_sm100_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmem);
}

cudaError_t launch_naive_pair_sm100(const NaiveAttnSm100& a, cudaStream_t s) {
    if (a.B <= 0 || a.Ls <= 0 || a.n_ranges <= 0) return cudaSuccess;
    PairParams p{};
    p.B = a.B; p.H = a.H; p.Ls = a.Ls; p.Ls_pad = (a.Ls + 127) / 128 * 128;
    p.part_rows = a.part_rows > 0 ? a.part_rows : a.B;
    p.m_groups = (a.B + 255) / 256;
    p.n_tiles = (a.Ls + TOK - 1) / TOK;
    const long long T = (long long)a.H * p.n_tiles;
    if (T >= (1LL << 31) || a.n_ranges > T) return cudaErrorInvalidValue;
    p.n_ranges = a.n_ranges;
    p.per = (int)(T / a.n_ranges);
    p.rem = (int)(T % a.n_ranges);
    p.n_seg_max = a.n_slots;
    p.scale_log2 = a.scale * kLog2e;
    p.o_part = a.o_part; p.lse_part = a.lse_part; p.status = a.status;
    CUtensorMap tm_qn, tm_qp;
    uint64_t dims[3] = {128, (uint64_t)a.H, (uint64_t)a.B};
    uint64_t str[2] = {128 * 2, (uint64_t)a.H * 128 * 2};
    uint32_t box[3] = {64, 1, 128};
    cudaError_t e = make_tmap_bf16(&tm_qn, a.q_nope, 3, dims, str, box);
    if (e != cudaSuccess) return e;
    dims[0] = 64;
    str[0] = 64 * 2;
    str[1] = (uint64_t)a.H * 64 * 2;
    e = make_tmap_bf16(&tm_qp, a.q_pe, 3, dims, str, box);
    if (e != cudaSuccess) return e;
    // partials [values (fp32, as pairs of 16-bit elements) | head | row of this launch | slot]
    CUtensorMap tm_o;
    uint64_t odims[4] = {256, (uint64_t)a.H, (uint64_t)a.B, (uint64_t)std::max(a.n_slots, 1)};
    uint64_t ostr[3] = {512, (uint64_t)a.H * 512, (uint64_t)p.part_rows * a.H * 512};
    uint32_t obox[4] = {64, 1, 128, 1};
    e = make_tmap_bf16(&tm_o, a.o_part, 4, odims, ostr, obox);
    if (e != cudaSuccess) return e;
    return launch_pdl(naive_pair_sm100_kernel, dim3(2 * p.n_ranges * p.m_groups), dim3(384), kSmem, s, tm_qn, tm_qp, *a.tm_kn, *a.tm_kp,
                      *a.tm_vt_half, tm_o, p);
}

cudaError_t make_naive_pair_tmap(const void* v_t, int H, int64_t Ls_pad, CUtensorMap* tm_vt_half) {
    uint64_t dims[4] = {64, 128, (uint64_t)(Ls_pad / 64), (uint64_t)H};
    uint64_t str[3] = {64 * 2, 128 * 64 * 2, (uint64_t)Ls_pad * 128 * 2};
    uint32_t box[4] = {64, 64, 2, 1};
    return make_tmap_bf16(tm_vt_half, v_t, 4, dims, str, box);
}

}  // namespace tmla
