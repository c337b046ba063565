// C ABI of the library: argument validation, the prepared-prefix handle, the
// workspace plan, the crossover rule (Eq. 1 / Table 1) and the launch sequence
// of one decode step (Algorithm 1).
#include <algorithm>
#include <atomic>
#include <cmath>
#include <cstdint>
#include <cstdlib>
#include <cstring>
#include <mutex>
#include <new>

#include "../../include/typhoon_mla.h"
#include "../../include/typhoon_mla_internal.h"
#include "kernels.h"

using namespace tmla;

#include "handle.h"

thread_local bool tmla::tl_pdl = true;

namespace {

thread_local int g_last_launches = 0;
thread_local int g_last_cuda_error = 0;

// Optional CUDA-event timing of one kernel kind inside decode calls.
struct Profile {
    int kernel_id = -1;
    int capacity = 0, used = 0;
    cudaEvent_t* ev = nullptr;  // 2 per recorded launch
};
Profile g_prof;

inline void prof_before(int id, cudaStream_t s) {
    if (id == g_prof.kernel_id && g_prof.used < g_prof.capacity) cudaEventRecord(g_prof.ev[2 * g_prof.used], s);
}
inline void prof_after(int id, cudaStream_t s) {
    if (id == g_prof.kernel_id && g_prof.used < g_prof.capacity) {
        cudaEventRecord(g_prof.ev[2 * g_prof.used + 1], s);
        ++g_prof.used;
    }
}

// Process-wide switches (test and measurement hooks) and the hardware model of the crossover rule.  They
// are atomics; an API call takes one snapshot at its start and plans and launches from that snapshot only.
std::atomic<int> g_kernel_path{TYPHOON_MLA_PATH_TCGEN05};
std::atomic<bool> g_overlap{true};          // absorb branch of a hybrid step on the handle's side stream
std::atomic<bool> g_pdl{true};              // programmatic dependent launch of the step's kernels
std::atomic<int> g_naive_schedule{0};
std::atomic<bool> g_stacked_absorb{true};   // absorb-only steps: batch-stacked kernel over the shared prefix
constexpr double kDefTensor = 1.0e15, kDefHbm = 6.0e12, kDefFixed = 6.0e-6, kDefAbsorbEff = 0.5;
std::atomic<double> g_tensor_flops{kDefTensor};        // sustained rate the attention kernels reach, FLOP/s
std::atomic<double> g_hbm_bytes{kDefHbm};              // bytes/s
std::atomic<double> g_hybrid_fixed_s{kDefFixed};       // extra launches + combine of the hybrid path
std::atomic<double> g_absorb_efficiency{kDefAbsorbEff};   // absorb kernel's share of g_tensor_flops (calibrated on B200)

struct Settings {
    int kernel_path, naive_schedule;
    bool overlap, pdl, stacked_absorb;
    bool tc() const { return kernel_path == TYPHOON_MLA_PATH_TCGEN05; }
};
Settings snapshot() {
    return Settings{g_kernel_path.load(), g_naive_schedule.load(), g_overlap.load(), g_pdl.load(), g_stacked_absorb.load()};
}

inline int64_t round_up(int64_t x, int64_t m) { return (x + m - 1) / m * m; }
inline bool aligned16(const void* p) { return (reinterpret_cast<uintptr_t>(p) & 15u) == 0; }

bool dims_supported(const typhoon_mla_dims_t& d) {
    return d.d_nope == 128 && d.d_rope == 64 && d.d_v == 128 && d.kv_lora_rank == 512 && d.num_heads >= 16 &&
           d.num_heads <= 128 && d.num_heads % 16 == 0;
}

int cuda_fail(cudaError_t e) {
    g_last_cuda_error = (int)e;
    return TYPHOON_MLA_ERR_CUDA;
}
}  // namespace
int tmla::api_cuda_fail(cudaError_t e) { return cuda_fail(e); }
void tmla::api_set_last_launches(int n) { g_last_launches = n; }
namespace {

// ---- side stream and events of a handle -------------------------------------
// Creating and destroying a stream takes about 55 us each (B200 host), as much as a short decode step, so up to
// kKeptSides idle sets per device outlive their handle.  A set belongs to one handle at a time; it comes back only
// after the device has been synchronised (nothing of it is pending) and not while a capture holds it.
// typhoon_mla_release_cached destroys the kept ones.
constexpr int kKeptSides = 4, kSideDevices = 64;
struct Side {
    cudaStream_t stream = nullptr;
    cudaEvent_t fork = nullptr, join = nullptr;
};
std::mutex g_side_mu;
Side g_sides[kSideDevices][kKeptSides];
int g_n_sides[kSideDevices] = {};

void destroy_side(const Side& x) {
    if (x.stream) cudaStreamDestroy(x.stream);
    if (x.fork) cudaEventDestroy(x.fork);
    if (x.join) cudaEventDestroy(x.join);
}
cudaError_t take_side(int dev, Side* out) {
    if (dev >= 0 && dev < kSideDevices) {
        std::lock_guard<std::mutex> lock(g_side_mu);
        if (g_n_sides[dev] > 0) {
            *out = g_sides[dev][--g_n_sides[dev]];
            return cudaSuccess;
        }
    }
    Side x;
    int lo = 0, hi = 0;
    cudaDeviceGetStreamPriorityRange(&lo, &hi);   // hi is the numerically lowest = highest priority
    cudaError_t e = cudaStreamCreateWithPriority(&x.stream, cudaStreamNonBlocking, hi);
    if (e == cudaSuccess) e = cudaEventCreateWithFlags(&x.fork, cudaEventDisableTiming);
    if (e == cudaSuccess) e = cudaEventCreateWithFlags(&x.join, cudaEventDisableTiming);
    if (e != cudaSuccess) destroy_side(x);
    else *out = x;
    return e;
}
void give_side(int dev, const Side& x, bool idle) {
    cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
    if (idle && x.stream && cudaStreamIsCapturing(x.stream, &cap) == cudaSuccess && cap == cudaStreamCaptureStatusNone &&
        dev >= 0 && dev < kSideDevices) {
        std::lock_guard<std::mutex> lock(g_side_mu);
        if (g_n_sides[dev] < kKeptSides) {
            g_sides[dev][g_n_sides[dev]++] = x;
            return;
        }
    }
    destroy_side(x);
}

// ---- workspace plan --------------------------------------------------------
struct Plan {
    int mode;
    int n_split_naive;       // KV splits of the warp-MMA naive kernel / tile ranges of the tcgen05 one
    int n_slots_naive;       // partial slots the naive kernel writes (>= n_split_naive)
    bool absorb_pairs;       // absorb attention by the kernel of 128 rows per CTA pair
    int chunk;               // tokens per absorb chunk
    int n_shared_chunks;     // absorb chunks over the shared prefix (ABSORB mode)
    int n_suffix_chunks;
    // byte offsets into the workspace
    size_t off_order, off_desc, off_qabs, off_opart_a, off_lsepart_a, off_olat, off_lse_a, off_oabs, off_opart_n, off_lsepart_n, total;
};

constexpr int kDefaultNumSM = 148;        // a B200; used where no device is at hand (pure planning queries)
constexpr int kMaxAbsorbChunks = 1024;   // chunks per request the merge kernel accepts

int naive_splits(int B, int H, int64_t Ls, int n_sm, int max_slots) {
    if (Ls <= 0) return 0;
    int n_tiles = (int)((Ls + 63) / 64);
    int base = ((B + 63) / 64) * H;
    int want = (4 * n_sm + base - 1) / base;
    return std::max(1, std::min({want, n_tiles, 64, max_slots}));
}

// Whether the absorb attention of a step of more than 64 heads goes to the kernel of 128 rows per CTA pair: yes, except where the table
// holds few tokens per request and the step runs beside a shared-prefix launch of at most 128 rows.  Those CTAs leave single SMs free,
// not the two neighbouring ones that a pair needs, and with suffixes this short what the 64-row kernel gets done on them counts
// for more than the pair's faster tiles.  (B200, us per step, 64-row / pair: 96 heads, 24 requests, 2301 tokens and one page of 64
// 36.5 / 40.6, 128 heads, 100 requests, 1277 and one page 63.7 / 66.4, 1280 and four pages 63.3 / 66.1; 128 heads, 8 requests, 809
// and four pages 43.8 / 39.4; 54 requests, 1267 and two pages 52.6 / 51.9.  Over 119 such steps this line loses 0.5 % to the better of
// the two, one kernel for all 1.4 and 2.4 %.)
bool many_heads_use_pairs(int B, int64_t cap_suffix, bool beside_prefix) {
    return !(beside_prefix && B <= 128 && (cap_suffix <= 64 || (cap_suffix <= 256 && B > 64)));
}

// Kernel and chunk length of the absorb attention.  cap_suffix: the page table's width in tokens (the suffixes' lengths are on the device).
// max_chunks: at least one per non-empty segment, at most kMaxAbsorbChunks.
// `beside_prefix`: a shared-prefix launch runs beside it.
void absorb_chunks(bool tc, bool stacked, bool beside_prefix, int n_sm, int B, int H, int64_t Ls_absorb, int64_t cap_suffix, int max_chunks,
                   bool* pairs, int* chunk, int* n_sh, int* n_sf) {
    const int64_t longest = std::max<int64_t>(std::max(Ls_absorb, cap_suffix), 1);
    // One CTA (pair) per SM (pair of SMs): minimise waves x (tiles per chunk + fixed cost in tile units) over the number of
    // chunks the longest segment is cut into.  A split segment writes and re-reads fp32 partials, 2 KB per row both ways.
    auto cut = [&](bool pair) {
        const int tile = pair ? 128 : 64, slots = pair ? n_sm / 2 : n_sm;   // (tile: tokens, and rows of an item)
        const double fixed = pair ? 4.0 : 3.0, split = pair ? 3.0 : 3.5;
        // items per chunk of a suffix; of the prefix, cut from the stacked [B * H] query matrix or from each request's rows
        const int units = B * ((H + tile - 1) / tile);
        const int units_sh = stacked ? (int)(((int64_t)B * H + tile - 1) / tile) : units;
        double best_cost = 1e30;
        int64_t c = round_up(longest, tile), weighed = 0;
        for (int parts = 1; parts <= 512; ++parts) {
            const int64_t ch = round_up((longest + parts - 1) / parts, tile);
            if (ch == weighed) continue;
            weighed = ch;
            const int64_t per_req = (Ls_absorb + ch - 1) / ch + (cap_suffix + ch - 1) / ch;
            const int64_t items = (int64_t)units_sh * ((Ls_absorb + ch - 1) / ch) + (int64_t)units * ((cap_suffix + ch - 1) / ch);
            if (per_req > max_chunks) continue;
            const int64_t waves = (items + slots - 1) / slots;
            const double cost = (double)waves * ((double)ch / tile + fixed + (per_req > 1 ? split : 0.0));
            if (cost < best_cost - 1e-9) {
                best_cost = cost;
                c = ch;
            }
            if (ch <= tile) break;
        }
        return c;
    };
    // Estimate of the kernel's time with chunks of `c` tokens, in SM clocks: the items' work spread over all places and half an item more.
    // (2580 and 2416 clocks per tile, as measured in the two kernels.)
    auto clocks = [&](bool pair, int64_t c) {
        const int tile = pair ? 128 : 64;
        const double n_sh = (double)((Ls_absorb + c - 1) / c), n_sf = (double)((cap_suffix + c - 1) / c);
        const double extra = (pair ? 6.0 : 5.0) + (n_sh + n_sf > 1 ? (pair ? 3.0 : 3.5) : 0.0);
        const double t_sh = (double)std::min(c, Ls_absorb) / tile + extra;
        const double t_sf = (double)((std::min(c, cap_suffix) + tile - 1) / tile) + extra;
        const double items_sh = (double)(((int64_t)B * H + tile - 1) / tile) * n_sh;
        const double items_sf = (double)B * ((H + tile - 1) / tile) * n_sf;
        const double longest_item = n_sh > 0 ? t_sh : t_sf;
        const double tiles = std::max(longest_item, (items_sh * t_sh + items_sf * t_sf) / (pair ? n_sm / 2 : n_sm) + 0.5 * longest_item);
        return tiles * (pair ? 2416.0 : 2580.0);
    };
    int64_t c;
    *pairs = false;
    if (tc && H > 64) {
        *pairs = many_heads_use_pairs(B, cap_suffix, beside_prefix);
        c = cut(*pairs);
    } else if (tc) {
        // Up to 64 heads the pair kernel is for the prefix of an absorb-only step, whose rows are stacked and fill its 128; a suffix item
        // has rows of nobody and still takes two SMs.  (B200, us per step, 64-row / pair: 64 heads, 12 requests, 22865 + 567 tokens
        // 71.9 / 51.5; 32 heads, 31, 4399 + 389 35.1 / 30.4; 16 heads, 60, 1426 + 39 28.0 / 33.8; 48 heads, 67, 131 + 11 27.0 / 35.3;
        // 32 heads, 185, 3378 + 17 110 / 134.  Over 184 such steps this choice is on average 0.5 % behind the better of the two, and in
        // four more than 3 % behind the 64-row kernel; pairs throughout 3.6 % and 42, comparing the costs above 1.0 % and 16.)
        c = cut(false);
        if (stacked && (int64_t)B * H >= 128 && Ls_absorb > 0 && Ls_absorb >= cap_suffix) {
            const int64_t c_pair = cut(true);
            if (clocks(true, c_pair) < 0.95 * clocks(false, c)) {
                *pairs = true;
                c = c_pair;
            }
        }
    } else {
        const int units = B * ((H + 63) / 64);
        const int target = std::max(1, (2 * n_sm + units - 1) / units);
        c = std::max<int64_t>(round_up((longest + target - 1) / target, 64), 256);
        while ((Ls_absorb + c - 1) / c + (cap_suffix + c - 1) / c > max_chunks) c *= 2;
    }
    *chunk = (int)c;
    *n_sh = (int)((Ls_absorb + c - 1) / c);
    *n_sf = (int)((cap_suffix + c - 1) / c);
}

// The workspace's parts, for partials of `chunk_rows` rows (chunks x requests x heads) of the absorb attention and `slot_rows` of
// the shared-prefix attention.
void lay_out(Plan* p, int B, int H, int64_t chunk_rows, int64_t slot_rows) {
    const size_t BH = (size_t)B * H;
    size_t off = 0;
    auto take = [&](size_t bytes) {
        size_t o = off;
        off += round_up((int64_t)bytes, 256);
        return o;
    };
    p->off_order = take((size_t)B * 4);
    p->off_desc = take((size_t)B * 16);
    p->off_qabs = take(BH * 512 * 2);
    p->off_opart_a = take((size_t)chunk_rows * 512 * 4);
    p->off_lsepart_a = take((size_t)chunk_rows * 4);
    p->off_olat = take(BH * 512 * 2);
    p->off_lse_a = take(BH * 4);
    p->off_oabs = take(BH * 128 * 4);
    p->off_opart_n = take((size_t)slot_rows * 128 * 4);
    p->off_lsepart_n = take((size_t)slot_rows * 4);
    p->total = off;
}

// The number of partials that a plan chooses neither grows nor falls steadily with the batch or the page table.  A workspace sized
// for B requests and max_pages pages has to do for smaller steps as well: it holds at least the "floor" of its sizes, every term of
// which grows with both, and a step whose own choice does not fit is planned again within what there is, which the floor of ITS
// sizes guarantees to be possible (one chunk per segment, two slots).  The constant is four waves of 64 rows per SM: of (H, L_s,
// pages, sized batch, batch) combinations over 16..128 heads, 100..65536 tokens, 1..200 pages and up to 1024 requests, 67 of 550800
// do not get their own choice in the mode that AUTO takes (1828 with one wave; at most 11 % longer by the plan's own model).
// It also bounds what the warp-MMA plan (about 2 n_sm 64-row chunks per segment) and every schedule of the shared-prefix kernel
// choose, n_sm / (row groups) ranges over H heads: at most 2 n_sm / H / groups + 2 slots.
int64_t floor_chunk_rows(int n_sm, int64_t rows, int64_t Ls_absorb, int64_t cap_suffix) {
    const int segments = (Ls_absorb > 0) + (cap_suffix > 0);
    return std::min(rows * ((Ls_absorb + 63) / 64 + (cap_suffix + 63) / 64), (int64_t)256 * n_sm + segments * rows);
}
int64_t floor_slot_rows(int n_sm, int64_t rows, int64_t Ls) {
    return Ls <= 0 ? 0 : std::min(rows * ((Ls + 63) / 64), (int64_t)256 * n_sm + 2 * rows);
}

// `mode` is resolved (ABSORB, HYBRID or NAIVE); `tc` and `schedule` come from the caller's settings snapshot.  workspace_bytes: 0 gives
// the floor's sizes (offsets and total only).  A plan whose total exceeds workspace_bytes cannot be run with them.
Plan make_plan(const typhoon_mla_shared* sh, bool tc, int schedule, int B, int max_pages, int page_size, int mode,
               int naive_slots_override = -1, bool stacked = true, size_t workspace_bytes = SIZE_MAX) {
    const int H = sh->dims.num_heads;
    const int n_sm = sh->num_sms > 0 ? sh->num_sms : kDefaultNumSM;
    const int64_t cap = (int64_t)max_pages * page_size, rows = (int64_t)B * H;
    const bool use_naive = (mode != TYPHOON_MLA_MODE_ABSORB) && sh->Ls > 0;
    const bool use_absorb = (mode != TYPHOON_MLA_MODE_NAIVE);
    const int64_t Ls_absorb = mode == TYPHOON_MLA_MODE_ABSORB ? sh->Ls : 0;
    auto plan_within = [&](int max_chunks, int max_slots) {
        Plan p{};
        p.mode = mode;
        if (naive_slots_override >= 0) {   // several shared-prefix launches planned by the caller
            p.n_split_naive = naive_slots_override > 0 ? 1 : 0;
            p.n_slots_naive = naive_slots_override;
        } else if (use_naive && tc) {   // n_split_naive = tile ranges
            naive_sm100_plan(B, H, sh->Ls, naive_places(B, n_sm, sh->fp8 != 0), schedule, &p.n_split_naive, &p.n_slots_naive, sh->fp8 != 0,
                             use_absorb ? absorb_branch_us(B, H, cap) : 0.0, max_slots);
        } else {
            p.n_split_naive = use_naive ? naive_splits(B, H, sh->Ls, n_sm, max_slots) : 0;
            p.n_slots_naive = p.n_split_naive;
        }
        if (use_absorb)
            absorb_chunks(tc, stacked, p.n_slots_naive > 0, n_sm, B, H, Ls_absorb, cap, max_chunks, &p.absorb_pairs, &p.chunk,
                          &p.n_shared_chunks, &p.n_suffix_chunks);
        lay_out(&p, B, H, (int64_t)(p.n_shared_chunks + p.n_suffix_chunks) * rows, (int64_t)p.n_slots_naive * rows);
        return p;
    };
    Plan p{};
    if (workspace_bytes > 0) {
        p = plan_within(kMaxAbsorbChunks, INT32_MAX);
        if (p.total <= workspace_bytes) return p;
    }
    const int64_t chunk_rows = use_absorb ? floor_chunk_rows(n_sm, rows, Ls_absorb, cap) : 0;
    const int64_t slot_rows = naive_slots_override >= 0 ? naive_slots_override * rows : use_naive ? floor_slot_rows(n_sm, rows, sh->Ls) : 0;
    Plan least{};
    lay_out(&least, B, H, chunk_rows, slot_rows);
    if (workspace_bytes == 0) return least;
    if (workspace_bytes < least.total) return p;
    // (a chunk's row: 512 values and its LSE; the LSEs' bytes are rounded up to 256)
    const int64_t more = (int64_t)(workspace_bytes - least.total);
    const int64_t max_chunks = (chunk_rows + std::max<int64_t>(more - 256, 0) / (512 * 4 + 4)) / rows;
    return plan_within((int)std::min<int64_t>(max_chunks, kMaxAbsorbChunks), (int)std::min<int64_t>(slot_rows / rows, INT32_MAX));
}

// Worst case over the modes that `mode` can resolve to, over both kernel implementations and over the work decompositions a test hook
// may select, and the floor: a workspace of this size serves steps of at most B requests and max_pages pages whatever the
// switches are set to when they run.  Only local values are used; no process-wide state is read or written.
size_t query_bytes(const typhoon_mla_shared* sh, int B, int max_pages, int page_size, int mode) {
    size_t worst = 0;
    for (int m : {TYPHOON_MLA_MODE_ABSORB, TYPHOON_MLA_MODE_HYBRID, TYPHOON_MLA_MODE_NAIVE}) {
        if (mode != TYPHOON_MLA_MODE_AUTO && mode != m && !(mode == TYPHOON_MLA_MODE_HYBRID && sh->Ls == 0)) continue;
        const int pages = m == TYPHOON_MLA_MODE_NAIVE ? 0 : max_pages;
        worst = std::max(worst, make_plan(sh, true, 0, B, pages, page_size, m, -1, true, 0).total);
        for (bool tc : {true, false})
            for (int schedule : {0, 1, 2})
                for (bool stacked : {true, false})
                    worst = std::max(worst, make_plan(sh, tc, schedule, B, pages, page_size, m, -1, stacked).total);
    }
    return worst + 256;
}

// The handle's buffers, stream and events live on the device it was prepared on.
bool on_handle_device(const typhoon_mla_shared* sh) {
    int dev = -1;
    return cudaGetDevice(&dev) == cudaSuccess && dev == sh->device;
}

int resolve_mode(const typhoon_mla_shared* sh, int B, int max_pages, int mode) {
    if (mode == TYPHOON_MLA_MODE_AUTO) {
        if (max_pages == 0 && sh->Ls > 0) return TYPHOON_MLA_MODE_NAIVE;
        return typhoon_mla_choose_mode(sh, B, -1);
    }
    if (mode == TYPHOON_MLA_MODE_HYBRID && sh->Ls == 0) return TYPHOON_MLA_MODE_ABSORB;
    return mode;
}

}  // namespace

extern "C" {

const char* typhoon_mla_status_string(int status) {
    switch (status) {
        case TYPHOON_MLA_OK: return "ok";
        case TYPHOON_MLA_ERR_INVALID_ARG: return "invalid argument";
        case TYPHOON_MLA_ERR_UNSUPPORTED_DIMS: return "unsupported dimensions";
        case TYPHOON_MLA_ERR_WORKSPACE_TOO_SMALL: return "workspace too small";
        case TYPHOON_MLA_ERR_ALLOC: return "device allocation failed";
        case TYPHOON_MLA_ERR_CUDA: return "CUDA error";
        case TYPHOON_MLA_ERR_DEVICE_CHECK: return "device-side check failed";
        case TYPHOON_MLA_ERR_STATIC_SCRATCH_EXCEEDED: return "problem exceeds the built-in scratch array";
        default: return "unknown status";
    }
}

int typhoon_mla_last_launch_count(void) { return g_last_launches; }
int typhoon_mla_last_cuda_error(void) { return g_last_cuda_error; }

double typhoon_mla_batch_threshold(const typhoon_mla_dims_t* d, int32_t S_q, double T, double M) {
    if (!d || S_q < 1 || !(M > 0.0)) return -1.0;
    const double d_qk = (double)d->d_nope + d->d_rope;
    return (d_qk + d->d_v) / ((double)S_q * (2.0 * d->kv_lora_rank + d->d_rope)) * (T / M);
}

int typhoon_mla_naive_plan(int32_t num_heads, int32_t B, int64_t L_s, int32_t schedule, int32_t num_sms, int32_t suffix_tokens,
                           int32_t* tile_tokens, int32_t* n_ranges, int32_t* row_groups, int32_t* n_slots) {
    if (B < 1 || L_s < 1 || L_s > (int64_t)1 << 30 || schedule < 0 || schedule > 2 || num_sms < 0 || suffix_tokens < 0)
        return TYPHOON_MLA_ERR_INVALID_ARG;
    if (num_heads < 16 || num_heads > 128 || num_heads % 16) return TYPHOON_MLA_ERR_INVALID_ARG;
    if (!tile_tokens || !n_ranges || !row_groups || !n_slots) return TYPHOON_MLA_ERR_INVALID_ARG;
    int r = 0, sl = 0;
    const int places = naive_places(B, num_sms > 0 ? num_sms : kDefaultNumSM, false);
    naive_sm100_plan(B, num_heads, L_s, places, schedule, &r, &sl, false, absorb_branch_us(B, num_heads, suffix_tokens));
    *tile_tokens = naive_sm100_tile_tokens(B);
    *n_ranges = r;
    *row_groups = B <= 128 ? 1 : (B + 255) / 256;
    *n_slots = sl;
    return TYPHOON_MLA_OK;
}

int typhoon_mla_naive_plan_multi(int32_t num_heads, int32_t max_rows, const int64_t* L_s, int32_t n, int32_t schedule, int32_t num_sms,
                                 int32_t* n_ranges, int32_t* n_slots) {
    if (!L_s || !n_ranges || !n_slots || n < 1 || n > kNaiveJobsPerLaunch || max_rows < 1 || max_rows > 128) return TYPHOON_MLA_ERR_INVALID_ARG;
    if (schedule < 0 || schedule > 2 || num_sms < 0 || num_heads < 16 || num_heads > 128 || num_heads % 16) return TYPHOON_MLA_ERR_INVALID_ARG;
    for (int i = 0; i < n; ++i)
        if (L_s[i] < 1 || L_s[i] > (int64_t)1 << 24) return TYPHOON_MLA_ERR_INVALID_ARG;
    naive_sm100_plan_multi(max_rows, num_heads, L_s, n, num_sms > 0 ? num_sms : kDefaultNumSM, schedule, n_ranges, n_slots);
    return TYPHOON_MLA_OK;
}

int typhoon_mla_project_plan(int32_t num_heads, int32_t B, int32_t n_slots, int32_t prefix_8bit, int32_t num_sms, int32_t* columns,
                             int32_t* items, int32_t* ctas, int32_t* early) {
    if (B < 1 || n_slots < 0 || num_sms < 0 || !columns || !items || !ctas || !early) return TYPHOON_MLA_ERR_INVALID_ARG;
    if (num_heads < 16 || num_heads > 128 || num_heads % 16) return TYPHOON_MLA_ERR_INVALID_ARG;
    const int n_sm = num_sms > 0 ? num_sms : kDefaultNumSM;
    const ProjectPlan p = project_sm100_plan(B, num_heads, n_slots, prefix_8bit != 0, n_sm);
    *columns = p.columns;
    *items = p.items;
    *ctas = p.latency ? p.items : std::min(p.items, n_sm);
    *early = p.early ? 1 : 0;
    return TYPHOON_MLA_OK;
}

int typhoon_mla_cost_model(const typhoon_mla_dims_t* d, int32_t kind, int64_t B, int64_t S_q, int64_t L_s,
                           int64_t L_n, int64_t* macs, int64_t* hbm_words) {
    if (!d || B < 0 || S_q < 1 || L_s < 0 || L_n < 0) return TYPHOON_MLA_ERR_INVALID_ARG;
    const int64_t H = d->num_heads;
    const int64_t w_naive = H * ((int64_t)d->d_nope + d->d_rope + d->d_v);      // per (query, token) / per token
    const int64_t w_abs_mac = H * (2 * (int64_t)d->kv_lora_rank + d->d_rope);
    const int64_t w_abs_mem = (int64_t)d->kv_lora_rank + d->d_rope;
    int64_t m, w;
    switch (kind) {
        case TYPHOON_MLA_COST_NAIVE:
            m = B * S_q * (L_s + L_n) * w_naive;
            w = (L_s + B * L_n) * w_naive;
            break;
        case TYPHOON_MLA_COST_ABSORB:
            m = B * S_q * (L_s + L_n) * w_abs_mac;
            w = (L_s + B * L_n) * w_abs_mem;
            break;
        case TYPHOON_MLA_COST_TYPHOON:
            m = B * S_q * (L_s * w_naive + L_n * w_abs_mac);
            w = L_s * w_naive + B * L_n * w_abs_mem;
            break;
        default: return TYPHOON_MLA_ERR_INVALID_ARG;
    }
    if (macs) *macs = m;
    if (hbm_words) *hbm_words = w;
    return TYPHOON_MLA_OK;
}

int typhoon_mla_set_hw_model(double tensor_flops, double hbm_bytes_per_s, double hybrid_fixed_s) {
    g_tensor_flops.store(tensor_flops > 0 ? tensor_flops : kDefTensor);
    g_hbm_bytes.store(hbm_bytes_per_s > 0 ? hbm_bytes_per_s : kDefHbm);
    g_hybrid_fixed_s.store(hybrid_fixed_s >= 0 ? hybrid_fixed_s : kDefFixed);
    return TYPHOON_MLA_OK;
}

int typhoon_mla_set_absorb_efficiency(double fraction) {
    g_absorb_efficiency.store((fraction > 0.0 && fraction <= 1.0) ? fraction : kDefAbsorbEff);
    return TYPHOON_MLA_OK;
}

// `naive_time_factor`: how much longer the shared-prefix part takes than the model says (1 for the 16-bit cache).  The 8-bit
// cache's kernel is bound by its widening step: 1.13 to 1.4 times the 16-bit kernel's time up to 64 query rows (two conversion
// pairs from 16 tiles per CTA on), 1.3 to 1.8 up to 128, 1.5 to 2 above.  The forms cross at 24 to 64 rows (16 heads: up to 128).
// Over 16 and 128 heads, 512 to 32768 tokens, 1 to 512 requests the chosen form is on average 0.35 % behind the better one
// at 1.25 and 1.3, 0.5 % at 1.5 and 1.2, 0.8 % at 1 and 1.6 (128 heads, 24 requests over 32768 tokens 326 us latent against 417;
// 48 over 512 tokens 49.9 against 45.7).
constexpr double kNaiveTime8Bit = 1.3;
static int choose_mode_impl(const typhoon_mla_dims_t* dims, int64_t Ls, int32_t B, int64_t total_suffix_tokens,
                            double naive_time_factor) {
    if (!dims || B < 1 || Ls <= 0) return TYPHOON_MLA_MODE_ABSORB;
    if (total_suffix_tokens == 0) return TYPHOON_MLA_MODE_NAIVE;
    // Shared-prefix part only: the suffix part is identical in both modes.
    // Work terms are Table 1's, with the rope keys of the expanded cache read
    // once per token instead of once per head.
    const typhoon_mla_dims_t& d = *dims;
    const double H = d.num_heads, L = (double)Ls;
    const double f_naive = 2.0 * B * H * L * (d.d_nope + d.d_rope + d.d_v);
    // (the absorb kernels work on groups of 64 or 128 rows of the stacked [B * H] query matrix: a partial group costs as
    // much as a full one; counted in groups of 64)
    const double rows_abs = std::ceil(B * H / 64.0) * 64.0;
    const double f_absorb = 2.0 * rows_abs * L * (2.0 * d.kv_lora_rank + d.d_rope);
    const double by_naive = 2.0 * L * (H * (d.d_nope + d.d_v) + d.d_rope);
    const double by_absorb = 2.0 * L * (d.kv_lora_rank + d.d_rope);
    // The factor: the 64-row absorb kernel reaches about half of the tensor throughput that the naive kernel does (B200).  The
    // pair kernel reaches more, and for 21 to 36 requests of 128 heads the latent form would be the faster one (24 over 16384
    // tokens 135 us, hybrid 185); the line stays, because that form's 16-bit absorbed queries and latent outputs put the result
    // further from the 64-bit one (3.0e-3 against 2.2e-3).  A caller can ask for it.
    const double T = g_tensor_flops.load(), M = g_hbm_bytes.load();
    const double t_hybrid = naive_time_factor * std::max(f_naive / T, by_naive / M) + g_hybrid_fixed_s.load();
    const double t_absorb = std::max(f_absorb / (g_absorb_efficiency.load() * T), by_absorb / M);
    return t_hybrid < t_absorb ? TYPHOON_MLA_MODE_HYBRID : TYPHOON_MLA_MODE_ABSORB;
}

int typhoon_mla_choose_mode_for(const typhoon_mla_dims_t* dims, int64_t Ls, int32_t B, int64_t total_suffix_tokens) {
    return choose_mode_impl(dims, Ls, B, total_suffix_tokens, 1.0);
}

int typhoon_mla_choose_mode(const typhoon_mla_shared_t* sh, int32_t B, int64_t total_suffix_tokens) {
    if (!sh) return TYPHOON_MLA_MODE_ABSORB;
    return choose_mode_impl(&sh->dims, sh->Ls, B, total_suffix_tokens, sh->fp8 ? kNaiveTime8Bit : 1.0);
}

int typhoon_mla_free(typhoon_mla_shared_t* sh) {
    if (!sh) return TYPHOON_MLA_OK;
    // the handle's buffers, stream and events belong to the device it was prepared on, whatever device is current now
    int cur = -1;
    const bool switched = cudaGetDevice(&cur) == cudaSuccess && cur != sh->device && cudaSetDevice(sh->device) == cudaSuccess;
    const bool idle = cudaDeviceSynchronize() == cudaSuccess;
    if (!sh->borrowed_storage) {
        cudaFree(sh->k_nope);
        cudaFree(sh->v_t);
        cudaFree(sh->ckv);
        cudaFree(sh->kpe);
        cudaFree(sh->w_uk_t);
        cudaFree(sh->status);
        cudaFree(sh->k8);
        cudaFree(sh->v8);
        cudaFree(sh->fp8_f);
    }
    Side side;
    side.stream = sh->side_stream; side.fork = sh->ev_fork; side.join = sh->ev_join;
    give_side(sh->device, side, idle);
    if (switched) cudaSetDevice(cur);
    cudaGetLastError();   // a failure while releasing must not surface in the caller's next launch
    // (a caller that lent the storage has to know when work on it may still be pending)
    const int st = (sh->borrowed_storage && !idle) ? TYPHOON_MLA_ERR_CUDA : TYPHOON_MLA_OK;
    delete sh;
    return st;
}

int typhoon_mla_release_cached(void) {
    int cur = -1;
    if (cudaGetDevice(&cur) != cudaSuccess) return cuda_fail(cudaGetLastError());
    std::lock_guard<std::mutex> lock(g_side_mu);
    for (int dev = 0; dev < kSideDevices; ++dev) {
        if (g_n_sides[dev] == 0 || cudaSetDevice(dev) != cudaSuccess) continue;
        while (g_n_sides[dev] > 0) destroy_side(g_sides[dev][--g_n_sides[dev]]);
    }
    cudaSetDevice(cur);
    cudaGetLastError();
    return TYPHOON_MLA_OK;
}

// Buffers of a handle, in bytes.  Ls_pad rows; every part starts on a 256-byte boundary of caller-supplied storage.
struct SharedSizes {
    size_t ckv, kpe, w_uk_t, status, expanded /* one of K_nope, V^T in 16 bits */, codes /* one of them in 8 bits */, scales;
    SharedSizes(int H, int64_t Ls, bool fp8) {
        const size_t Lp = (size_t)round_up(Ls, 128), b_k = (size_t)H * Lp * 128 * 2;
        ckv = Lp * 512 * 2;
        kpe = Lp * 64 * 2;
        w_uk_t = (size_t)H * 512 * 128 * 2;
        status = 256;
        expanded = b_k;
        codes = fp8 ? b_k / 2 : 0;
        scales = fp8 ? (size_t)H * 3 * sizeof(float) : 0;
    }
    static size_t pad(size_t x) { return (size_t)round_up((int64_t)x, 256); }
    size_t storage(bool fp8) const {
        return pad(ckv) + pad(kpe) + pad(w_uk_t) + status + (fp8 ? 2 * pad(codes) + pad(scales) : 2 * pad(expanded));
    }
};

size_t typhoon_mla_shared_storage_bytes(const typhoon_mla_dims_t* dims, int64_t Ls, int32_t fp8, size_t* scratch_bytes) {
    if (scratch_bytes) *scratch_bytes = 0;
    if (!dims || !dims_supported(*dims) || Ls < 0 || Ls > (int64_t)1 << 24) return 0;
    const bool f = fp8 != 0 && Ls > 0;
    const SharedSizes sz(dims->num_heads, Ls, f);
    if (scratch_bytes && f) *scratch_bytes = sz.expanded;
    return sz.storage(f);
}

// `storage` / `scratch`: device memory of the caller, or null (the handle then allocates its own).
static int prepare_impl(const typhoon_mla_dims_t* dims, const void* ckv_shared, const void* kpe_shared,
                        int64_t Ls, int64_t ld_ckv, int64_t ld_kpe, const void* w_uk, const void* w_uv,
                        void* stream, typhoon_mla_shared_t** out_handle, bool fp8, void* storage = nullptr,
                        size_t storage_bytes = 0, void* scratch = nullptr, size_t scratch_bytes = 0) {
    if (!dims || !out_handle || !w_uk || !w_uv || Ls < 0) return TYPHOON_MLA_ERR_INVALID_ARG;
    *out_handle = nullptr;
    if (!dims_supported(*dims)) return TYPHOON_MLA_ERR_UNSUPPORTED_DIMS;
    if (Ls > 0 && (!ckv_shared || !kpe_shared || ld_ckv < 512 || ld_kpe < 64 || ld_ckv % 8 || ld_kpe % 8 ||
                   !aligned16(ckv_shared) || !aligned16(kpe_shared)))
        return TYPHOON_MLA_ERR_INVALID_ARG;
    if (!aligned16(w_uk) || !aligned16(w_uv) || Ls > (int64_t)1 << 24) return TYPHOON_MLA_ERR_INVALID_ARG;
    const SharedSizes sz(dims->num_heads, Ls, fp8 && Ls > 0);
    if (storage) {
        if ((reinterpret_cast<uintptr_t>(storage) & 255u) || (reinterpret_cast<uintptr_t>(scratch) & 255u)) return TYPHOON_MLA_ERR_INVALID_ARG;
        if (storage_bytes < sz.storage(fp8 && Ls > 0)) return TYPHOON_MLA_ERR_WORKSPACE_TOO_SMALL;
        if (fp8 && Ls > 0 && (!scratch || scratch_bytes < sz.expanded)) return TYPHOON_MLA_ERR_WORKSPACE_TOO_SMALL;
    }
    int dev = 0, n_sm = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&n_sm, cudaDevAttrMultiProcessorCount, dev);
    // opt-in shared-memory sizes of every kernel, once per device and off the decode path
    if (e == cudaSuccess) e = set_attrs_naive_sm100();
    if (e == cudaSuccess) e = set_attrs_naive_pair_sm100();
    if (e == cudaSuccess) e = set_attrs_absorb_sm100();
    if (e == cudaSuccess) e = set_attrs_absorb_pair_sm100();
    if (e == cudaSuccess) e = set_attrs_expand_sm100();
    if (e == cudaSuccess) e = set_attrs_project_sm100();
    if (e == cudaSuccess) e = set_attrs_q_absorb_sm100();
    if (e == cudaSuccess) e = set_attrs_attn_mma();
    if (e == cudaSuccess) e = set_attrs_gemm_tn();
    if (e != cudaSuccess) return cuda_fail(e);
    // The allocation-free entry point keeps its scratch in a device array of the library image.  The module
    // that holds it is loaded lazily, and loading it takes device memory: do it here, where allocating is
    // allowed, so that the entry point itself never has to.
    {
        const int st = noalloc_resolve_scratch_for_current_device();
        if (st != TYPHOON_MLA_OK) return st;
    }
    const Settings cfg = snapshot();
    tmla::tl_pdl = cfg.pdl;

    typhoon_mla_shared* sh = new (std::nothrow) typhoon_mla_shared();
    if (!sh) return TYPHOON_MLA_ERR_ALLOC;
    std::memset(sh, 0, sizeof(*sh));
    sh->dims = *dims;
    sh->Ls = Ls;
    sh->Ls_pad = round_up(Ls, 128);
    sh->w_uv = w_uv;
    sh->device = dev;
    sh->num_sms = n_sm;
    const int H = dims->num_heads;
    const size_t Lp = (size_t)sh->Ls_pad;
    sh->borrowed_storage = storage ? 1 : 0;
    char* next = reinterpret_cast<char*>(storage);
    auto alloc = [&](void** p, size_t bytes) {
        if (bytes == 0) { *p = nullptr; return true; }
        if (storage) {
            *p = next;
            next += SharedSizes::pad(bytes);
            sh->owned_bytes += bytes;
            return true;
        }
        if (cudaMalloc(p, bytes) != cudaSuccess) { cudaGetLastError(); *p = nullptr; return false; }
        sh->owned_bytes += bytes;
        return true;
    };
    sh->fp8 = (fp8 && Ls > 0) ? 1 : 0;
    // (the streamed buffers first.  Where in a large page they start does not matter: six shapes with storage at 0, 512, 4096
    // and 13056 bytes behind a 2 MB boundary differ by -1.4 to 0.8 % without a pattern, two at the same offset by 0.7 %)
    bool ok_alloc = sh->fp8 ? alloc(&sh->k8, sz.codes) && alloc(&sh->v8, sz.codes) : alloc(&sh->k_nope, sz.expanded) && alloc(&sh->v_t, sz.expanded);
    ok_alloc = ok_alloc && alloc(&sh->w_uk_t, sz.w_uk_t) && alloc(&sh->ckv, sz.ckv) && alloc(&sh->kpe, sz.kpe) &&
               alloc(reinterpret_cast<void**>(&sh->status), sz.status);
    if (ok_alloc && sh->fp8) ok_alloc = alloc(reinterpret_cast<void**>(&sh->fp8_f), sz.scales);
    if (!ok_alloc) {
        typhoon_mla_free(sh);
        return TYPHOON_MLA_ERR_ALLOC;
    }
    cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
    // 8-bit cache: each tensor is expanded into a 16-bit scratch of the stream's memory pool, encoded from there,
    // and the scratch is handed back in stream order (no synchronisation)
    void* scratch16 = nullptr;   // ours (released below); the caller's scratch is used where it gave one
    if (sh->fp8 && !storage && cudaMallocAsync(&scratch16, sz.expanded, s) != cudaSuccess) {
        cudaGetLastError();
        typhoon_mla_free(sh);
        return TYPHOON_MLA_ERR_ALLOC;
    }
    void* const k_dst = sh->fp8 ? (storage ? scratch : scratch16) : sh->k_nope;
    void* const v_dst = sh->fp8 ? (storage ? scratch : scratch16) : sh->v_t;
    const bool tc = cfg.tc();
    {
        Side side;
        e = take_side(dev, &side);
        sh->side_stream = side.stream; sh->ev_fork = side.fork; sh->ev_join = side.join;
    }
    if (e != cudaSuccess) {
        if (scratch16) cudaFreeAsync(scratch16, s);
        typhoon_mla_free(sh);
        return cuda_fail(e);
    }
    e = launch_prepare_layout(w_uk, sh->w_uk_t, H, ckv_shared, ld_ckv, sh->ckv, kpe_shared, ld_kpe, sh->kpe, Ls, (int64_t)Lp, sh->status, s);
    // (without an expansion kernel behind it, an operation that is no kernel keeps a decode step's early reads of w_uk_t behind
    // the layout kernel's completion)
    if (e == cudaSuccess && Ls == 0) e = cudaMemsetAsync(sh->status, 0, sz.status, s);
    // K_nope[h] = ckv * W_UK[h]^T and V^T[h] = W_UV[h] * ckv^T; with 8-bit storage each is encoded before the scratch takes
    // the next
    auto expand = [&](bool k, bool v) {
        if (tc) return launch_expand_sm100(sh->ckv, (int64_t)Lp, w_uk, w_uv, H, k ? k_dst : nullptr, v ? v_dst : nullptr, n_sm, sh->status, s);
        cudaError_t r = cudaSuccess;
        if (k) r = launch_gemm_tn(GemmTN{sh->ckv, 512, 0, w_uk, 512, 128 * 512, k_dst, 128, (int64_t)Lp * 128, (int)Lp, 128, 512, H, false, 0, true}, s);
        if (v && r == cudaSuccess)
            r = launch_gemm_tn(GemmTN{w_uv, 512, 128 * 512, sh->ckv, 512, 0, v_dst, (int64_t)Lp, (int64_t)(128 * Lp), 128, (int)Lp, 512, H, false, 64}, s);
        return r;
    };
    if (e == cudaSuccess && Ls > 0 && !sh->fp8) e = expand(true, true);
    if (e == cudaSuccess && Ls > 0 && sh->fp8) {
        uint32_t* amax = reinterpret_cast<uint32_t*>(sh->fp8_f + 2 * H);
        e = expand(true, false);
        if (e == cudaSuccess) e = launch_quantize_e4m3(k_dst, false, H, (int64_t)Lp, sh->k8, amax, sh->fp8_f, s);
        if (e == cudaSuccess) e = expand(false, true);
        if (e == cudaSuccess) e = launch_quantize_e4m3(v_dst, true, H, (int64_t)Lp, sh->v8, amax, sh->fp8_f + H, s);
    }
    if (scratch16) {
        const cudaError_t ef = cudaFreeAsync(scratch16, s);
        if (e == cudaSuccess) e = ef;
    }
    if (e == cudaSuccess && Ls > 0)
        e = sh->fp8 ? make_naive_fp8_tmaps(sh->k8, sh->kpe, sh->v8, H, sh->Ls_pad, &sh->tm_kn, &sh->tm_kp, &sh->tm_vt)
                    : make_naive_sm100_tmaps(sh->k_nope, sh->kpe, sh->v_t, H, sh->Ls_pad, &sh->tm_kn, &sh->tm_kp, &sh->tm_vt);
    if (e == cudaSuccess && Ls > 0 && !sh->fp8) e = make_naive_pair_tmap(sh->v_t, H, sh->Ls_pad, &sh->tm_vt_half);
    if (e == cudaSuccess) e = make_q_absorb_tmap(sh->w_uk_t, H, &sh->tm_wuk_t);
    if (e == cudaSuccess && Ls > 0) e = make_absorb_shared_tmaps(sh->ckv, sh->kpe, sh->Ls_pad, &sh->tm_ckv, &sh->tm_kpe_tok);
    if (e != cudaSuccess) {
        typhoon_mla_free(sh);
        return cuda_fail(e);
    }
    *out_handle = sh;
    return TYPHOON_MLA_OK;
}

int typhoon_mla_prepare_shared(const typhoon_mla_dims_t* dims, const void* ckv_shared, const void* kpe_shared,
                               int64_t Ls, int64_t ld_ckv, int64_t ld_kpe, const void* w_uk, const void* w_uv,
                               void* stream, typhoon_mla_shared_t** out_handle) {
    return prepare_impl(dims, ckv_shared, kpe_shared, Ls, ld_ckv, ld_kpe, w_uk, w_uv, stream, out_handle, false);
}

int typhoon_mla_prepare_shared_fp8(const typhoon_mla_dims_t* dims, const void* ckv_shared, const void* kpe_shared,
                                   int64_t Ls, int64_t ld_ckv, int64_t ld_kpe, const void* w_uk, const void* w_uv,
                                   void* stream, typhoon_mla_shared_t** out_handle) {
    return prepare_impl(dims, ckv_shared, kpe_shared, Ls, ld_ckv, ld_kpe, w_uk, w_uv, stream, out_handle, true);
}

int typhoon_mla_prepare_shared_in(const typhoon_mla_dims_t* dims, const void* ckv_shared, const void* kpe_shared,
                                  int64_t Ls, int64_t ld_ckv, int64_t ld_kpe, const void* w_uk, const void* w_uv,
                                  int32_t fp8, void* storage, size_t storage_bytes, void* scratch, size_t scratch_bytes,
                                  void* stream, typhoon_mla_shared_t** out_handle) {
    if (!storage) return TYPHOON_MLA_ERR_INVALID_ARG;
    return prepare_impl(dims, ckv_shared, kpe_shared, Ls, ld_ckv, ld_kpe, w_uk, w_uv, stream, out_handle, fp8 != 0, storage,
                        storage_bytes, scratch, scratch_bytes);
}

int typhoon_mla_shared_view(const typhoon_mla_shared_t* sh, const void** k_nope, const void** v_t, int64_t* Ls,
                            int64_t* Ls_padded, int64_t* owned_bytes) {
    if (!sh) return TYPHOON_MLA_ERR_INVALID_ARG;
    if (k_nope) *k_nope = sh->k_nope;
    if (v_t) *v_t = sh->v_t;
    if (Ls) *Ls = sh->Ls;
    if (Ls_padded) *Ls_padded = sh->Ls_pad;
    if (owned_bytes) *owned_bytes = (int64_t)sh->owned_bytes;
    return TYPHOON_MLA_OK;
}

int typhoon_mla_expand_query_rows(const int32_t* block_table, const int32_t* seq_lens, int32_t B, int32_t max_pages,
                                  int32_t S_q, int32_t* block_table_rows, int32_t* seq_lens_rows, void* stream) {
    if (!seq_lens || !seq_lens_rows || B < 1 || S_q < 1 || max_pages < 0) return TYPHOON_MLA_ERR_INVALID_ARG;
    if (max_pages > 0 && (!block_table || !block_table_rows)) return TYPHOON_MLA_ERR_INVALID_ARG;
    if ((int64_t)B * S_q > INT32_MAX) return TYPHOON_MLA_ERR_INVALID_ARG;
    cudaError_t e = launch_expand_query_rows(block_table, seq_lens, B, max_pages, S_q, block_table_rows, seq_lens_rows,
                                             reinterpret_cast<cudaStream_t>(stream));
    return e == cudaSuccess ? TYPHOON_MLA_OK : cuda_fail(e);
}

int typhoon_mla_order_by_length(const int32_t* seq_lens, int32_t B, int32_t* perm, void* stream) {
    if (!seq_lens || !perm || B < 1 || B > 4096) return TYPHOON_MLA_ERR_INVALID_ARG;
    cudaError_t e = launch_order_by_length(seq_lens, B, perm, reinterpret_cast<cudaStream_t>(stream));
    return e == cudaSuccess ? TYPHOON_MLA_OK : cuda_fail(e);
}

int typhoon_mla_set_overlap(int32_t enable) {
    g_overlap.store(enable != 0);
    return TYPHOON_MLA_OK;
}

int typhoon_mla_set_programmatic_launch(int32_t enable) {
    g_pdl.store(enable != 0);
    return TYPHOON_MLA_OK;
}

int typhoon_mla_set_naive_schedule(int32_t schedule) {
    if (schedule < 0 || schedule > 2) return TYPHOON_MLA_ERR_INVALID_ARG;
    g_naive_schedule.store(schedule);
    return TYPHOON_MLA_OK;
}

int typhoon_mla_set_kernel_path(int32_t path) {
    if (path != TYPHOON_MLA_PATH_TCGEN05 && path != TYPHOON_MLA_PATH_WARP_MMA) return TYPHOON_MLA_ERR_INVALID_ARG;
    g_kernel_path.store(path);
    return TYPHOON_MLA_OK;
}

int typhoon_mla_set_stacked_absorb(int32_t enable) {
    g_stacked_absorb.store(enable != 0);
    return TYPHOON_MLA_OK;
}

int typhoon_mla_check_status(const typhoon_mla_shared_t* sh, void* stream, int32_t* word, int32_t clear) {
    if (!sh) return TYPHOON_MLA_ERR_INVALID_ARG;
    int v = 0;
    cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
    cudaError_t e = cudaMemcpyAsync(&v, sh->status, sizeof(int), cudaMemcpyDeviceToHost, s);
    if (e == cudaSuccess && clear) e = cudaMemsetAsync(sh->status, 0, sizeof(int), s);
    if (e == cudaSuccess) e = cudaStreamSynchronize(s);
    if (e != cudaSuccess) return cuda_fail(e);
    if (word) *word = v;
    return v == 0 ? TYPHOON_MLA_OK : TYPHOON_MLA_ERR_DEVICE_CHECK;
}

int typhoon_mla_test_wait_expiry(const typhoon_mla_shared_t* sh, int64_t deadline_cycles, int32_t code, void* stream) {
    if (!sh || code < 1 || code > 255) return TYPHOON_MLA_ERR_INVALID_ARG;
    const long long d = std::min<long long>(std::max<long long>(deadline_cycles, 1000), 100000000LL);
    const cudaError_t e = launch_wait_expiry_selftest(sh->status, d, code, reinterpret_cast<cudaStream_t>(stream));
    return e == cudaSuccess ? TYPHOON_MLA_OK : cuda_fail(e);
}

int typhoon_mla_shared_export(const typhoon_mla_shared_t* sh, void* k_nope_dst, void* v_t_dst, void* stream) {
    if (!sh || !k_nope_dst || !v_t_dst || sh->fp8) return TYPHOON_MLA_ERR_INVALID_ARG;
    const size_t bytes = (size_t)sh->dims.num_heads * (size_t)sh->Ls_pad * 128 * 2;
    if (bytes == 0) return TYPHOON_MLA_OK;
    cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
    cudaError_t e = cudaMemcpyAsync(k_nope_dst, sh->k_nope, bytes, cudaMemcpyDeviceToDevice, s);
    if (e == cudaSuccess) e = cudaMemcpyAsync(v_t_dst, sh->v_t, bytes, cudaMemcpyDeviceToDevice, s);
    return e == cudaSuccess ? TYPHOON_MLA_OK : cuda_fail(e);
}

int typhoon_mla_shared_export_fp8(const typhoon_mla_shared_t* sh, void* k_codes_dst, void* v_codes_dst, float* scales_dst,
                                  void* stream) {
    if (!sh || !k_codes_dst || !v_codes_dst || !scales_dst || !sh->fp8) return TYPHOON_MLA_ERR_INVALID_ARG;
    const int H = sh->dims.num_heads;
    const size_t n = (size_t)H * (size_t)sh->Ls_pad * 128;
    cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
    cudaError_t e = cudaMemcpyAsync(k_codes_dst, sh->k8, n, cudaMemcpyDeviceToDevice, s);
    if (e == cudaSuccess) e = cudaMemcpyAsync(v_codes_dst, sh->v8, n, cudaMemcpyDeviceToDevice, s);
    if (e == cudaSuccess) e = cudaMemcpyAsync(scales_dst, sh->fp8_f, (size_t)2 * H * sizeof(float), cudaMemcpyDeviceToDevice, s);
    return e == cudaSuccess ? TYPHOON_MLA_OK : cuda_fail(e);
}

size_t typhoon_mla_workspace_bytes(const typhoon_mla_shared_t* sh, int32_t B, int32_t max_pages, int32_t page_size,
                                   int32_t mode) {
    if (!sh || B < 1 || max_pages < 0 || (page_size != 64 && page_size != 128)) return 0;
    if (mode < TYPHOON_MLA_MODE_AUTO || mode > TYPHOON_MLA_MODE_NAIVE) return 0;
    return query_bytes(sh, B, max_pages, page_size, mode);
}

int typhoon_mla_workspace_plan(int32_t num_heads, int64_t L_s, int32_t prefix_8bit, int32_t B, int32_t max_pages, int32_t page_size,
                               int32_t mode, int32_t path, int32_t schedule, int32_t stacked, int32_t num_sms, size_t workspace_bytes,
                               size_t* query, size_t* step, int32_t* n_chunks, int32_t* n_slots, int32_t* absorb_pairs) {
    if (num_heads < 16 || num_heads > 128 || num_heads % 16 || L_s < 0 || L_s > (int64_t)1 << 24 || B < 1 || max_pages < 0)
        return TYPHOON_MLA_ERR_INVALID_ARG;
    if ((page_size != 64 && page_size != 128) || mode < TYPHOON_MLA_MODE_AUTO || mode > TYPHOON_MLA_MODE_NAIVE)
        return TYPHOON_MLA_ERR_INVALID_ARG;
    if (path < 0 || path > 1 || schedule < 0 || schedule > 2 || num_sms < 0) return TYPHOON_MLA_ERR_INVALID_ARG;
    if (!query || !step || !n_chunks || !n_slots || !absorb_pairs) return TYPHOON_MLA_ERR_INVALID_ARG;
    typhoon_mla_shared sh{};
    sh.dims.num_heads = num_heads; sh.dims.d_nope = 128; sh.dims.d_rope = 64; sh.dims.d_v = 128; sh.dims.kv_lora_rank = 512;
    sh.Ls = L_s;
    sh.fp8 = prefix_8bit != 0 && L_s > 0;
    sh.num_sms = num_sms;
    *query = query_bytes(&sh, B, max_pages, page_size, mode);
    const int m = resolve_mode(&sh, B, max_pages, mode);
    const int pages = m == TYPHOON_MLA_MODE_NAIVE ? 0 : max_pages;
    const Plan p = make_plan(&sh, path == TYPHOON_MLA_PATH_TCGEN05, schedule, B, pages, page_size, m, -1, stacked != 0,
                             workspace_bytes > 0 ? workspace_bytes : SIZE_MAX);
    *step = p.total;
    *n_chunks = p.n_shared_chunks + p.n_suffix_chunks;
    *n_slots = p.n_slots_naive;
    *absorb_pairs = p.absorb_pairs ? 1 : 0;
    return workspace_bytes > 0 && workspace_bytes < p.total ? TYPHOON_MLA_ERR_WORKSPACE_TOO_SMALL : TYPHOON_MLA_OK;
}

// One launch of the shared-prefix kernel: `rows` requests starting at `row0` against the prefix of
// `sh`, partial slots [slot0, slot0 + n_slots_level) of the step's partial arrays.
struct NaiveJob {
    const typhoon_mla_shared* sh;
    int row0, rows;
    int n_ranges;         // tile ranges (tcgen05 path) or KV splits (warp-MMA path)
    int n_slots_level;    // slots of this job's level (the kernel marks the ones it does not fill as empty)
    int slot0;
    int n_merged = 1;     // first job of a launch: how many consecutive jobs it takes
};
// Rows of a level that have no prefix: their slots get weight zero in the combine.
struct EmptySlots {
    int slot0, n_slots, row0, rows;
};

// Launch sequence of one step.  `sh` provides the weights, the absorb-side tensor maps, the side stream
// and the status word; `mode` is resolved (ABSORB, HYBRID or NAIVE); `pl.n_slots_naive` is the total
// number of naive partial slots.

static int decode_core(const Settings& cfg, const typhoon_mla_shared* sh, const NaiveJob* jobs, int n_jobs,
                const EmptySlots* empties, int n_empties,
                const Plan& pl, const void* q_nope, const void* q_pe, int32_t B, const void* ckv_pages,
                const void* kpe_pages, int64_t ckv_token_stride, int64_t kpe_token_stride, int32_t page_size, int32_t num_pages,
                const int32_t* block_table, int32_t max_pages, const int32_t* seq_lens, float softmax_scale, int32_t mode,
                void* out, float* lse_out, void* workspace, void* stream, bool out_fp32 = false) {
    const bool use_absorb = mode != TYPHOON_MLA_MODE_NAIVE;
    tmla::tl_pdl = cfg.pdl;
    cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
    char* ws = reinterpret_cast<char*>(workspace);
    const int H = sh->dims.num_heads;
    cudaError_t e = cudaSuccess;
    int launches = 0;

    float* o_part_n = reinterpret_cast<float*>(ws + pl.off_opart_n);
    float* lse_part_n = reinterpret_cast<float*>(ws + pl.off_lsepart_n);
    float* o_abs = reinterpret_cast<float*>(ws + pl.off_oabs);
    float* lse_a = reinterpret_cast<float*>(ws + pl.off_lse_a);

    const int n_chunks = pl.n_shared_chunks + pl.n_suffix_chunks;
    const bool have_absorb = use_absorb && n_chunks > 0;
    const bool tc = cfg.tc();
    // In a hybrid step the absorb branch (lines 5-6) does not depend on the naive kernel (line 4): it runs
    // on the handle's (high-priority) side stream, forked behind the caller's stream here and joined
    // before the projection.
    if (!tc)   // row ranges and the 8-bit cache need the tcgen05 kernel
        for (int j = 0; j < n_jobs; ++j)
            if (jobs[j].rows != B || jobs[j].sh->fp8) return TYPHOON_MLA_ERR_UNSUPPORTED_DIMS;
    cudaStream_t s_main = s;
    const bool forked = cfg.overlap && have_absorb && n_jobs > 0 && sh->side_stream != nullptr;
    if (forked) {
        e = cudaEventRecord(sh->ev_fork, s_main);
        if (e == cudaSuccess) e = cudaStreamWaitEvent(sh->side_stream, sh->ev_fork, 0);
        if (e != cudaSuccess) return cuda_fail(e);
    }
    // A failure after the fork still joins the side stream back into the caller's stream, so that the caller's stream
    // stays the only one with work of this call pending (and a stream capture is not left with an open branch).
    bool open_fork = forked;
    auto fail = [&](cudaError_t err) {
        if (open_fork && cudaEventRecord(sh->ev_join, sh->side_stream) == cudaSuccess) cudaStreamWaitEvent(s_main, sh->ev_join, 0);
        return cuda_fail(err);
    };

    // --- naive shared-prefix attention (Algorithm 1 line 4), one launch per (prefix, row range)
    for (int j = 0; j < n_jobs; j += jobs[j].n_merged) {
        const NaiveJob& jb = jobs[j];
        auto sm100_job = [&](const NaiveJob& x) {
            const char* qn = reinterpret_cast<const char*>(q_nope) + (size_t)x.row0 * H * 128 * 2;
            const char* qp = reinterpret_cast<const char*>(q_pe) + (size_t)x.row0 * H * 64 * 2;
            float* op = o_part_n + ((size_t)x.slot0 * B + x.row0) * H * 128;
            float* lp = lse_part_n + ((size_t)x.slot0 * B + x.row0) * H;
            NaiveAttnSm100 na{qn, qp, &x.sh->tm_kn, &x.sh->tm_kp, &x.sh->tm_vt, x.rows, H, (int)x.sh->Ls,
                              x.n_ranges, x.n_slots_level, softmax_scale, op, lp, sh->status, B};
            if (x.sh->fp8) na.fp8_mult = x.sh->fp8_f;
            na.tm_vt_half = &x.sh->tm_vt_half;
            return na;
        };
        prof_before(TYPHOON_MLA_KERNEL_NAIVE_ATTN, s);
        if (tc && jb.n_merged > 1) {
            NaiveAttnSm100 na[kNaiveJobsPerLaunch];
            for (int k = 0; k < jb.n_merged; ++k) na[k] = sm100_job(jobs[j + k]);
            e = launch_naive_attn_sm100_multi(na, jb.n_merged, s);
        } else if (tc) {
            e = launch_naive_attn_sm100(sm100_job(jb), s);
        } else {
            NaiveAttn na{q_nope, q_pe, jb.sh->k_nope, jb.sh->v_t, jb.sh->kpe, B, H, (int)jb.sh->Ls, (int)jb.sh->Ls_pad,
                         jb.n_ranges, softmax_scale, o_part_n, lse_part_n};
            e = launch_naive_attn_mma(na, s);
        }
        prof_after(TYPHOON_MLA_KERNEL_NAIVE_ATTN, s);
        if (e != cudaSuccess) return fail(e);
        ++launches;
    }
    for (int j = 0; j < n_empties; ++j) {
        const EmptySlots& es = empties[j];
        e = launch_fill_neg_inf(lse_part_n + ((size_t)es.slot0 * B + es.row0) * H, es.n_slots, (int64_t)B * H,
                                (int64_t)es.rows * H, s);
        if (e != cudaSuccess) return fail(e);
        ++launches;
    }
    bool combined = false;
    if (forked) s = sh->side_stream;
    if (have_absorb) {
        // ragged suffixes: the longest requests are launched first (order computed on the device, no host
        // sync): by an extra block of the query-absorption kernel on the tcgen05 path, by its own kernel otherwise
        int32_t* order = nullptr;
        int32_t* desc = nullptr;   // per-position descriptors, written next to the order on the tcgen05 path
        if (pl.n_suffix_chunks > 0 && B > 1 && B <= 4096) order = reinterpret_cast<int32_t*>(ws + pl.off_order);
        // --- query absorption Q_A = Q_N W_UK (Algorithm 1 line 5)
        void* q_abs = ws + pl.off_qabs;
        prof_before(TYPHOON_MLA_KERNEL_Q_ABSORB, s);
        if (tc) {
            if (order) desc = reinterpret_cast<int32_t*>(ws + pl.off_desc);
            // Beside the shared-prefix kernel the absorb branch has the SMs that kernel's CTAs leave free: if those are few,
            // that many CTAs walk through the heads (each resident for the whole launch) instead of one CTA per head
            // queueing for them.  (With one tile of 128 requests per head; a launch then has one CTA per range.)
            int walk_ctas = 0;
            if (forked && B <= 128) {
                int naive_ctas = 0;
                for (int j = 0; j < n_jobs; ++j) naive_ctas = std::max(naive_ctas, jobs[j].n_ranges);
                const int free_sms = sh->num_sms - naive_ctas;
                if (jobs[0].n_merged == n_jobs && free_sms >= 8 && free_sms < H) {
                    // ... but only if the shared-prefix kernel lasts about as long as the walk (measured: about 5 us per head
                    // for a walking CTA, 0.7 us per 64-token tile for a shared-prefix CTA; B = 64, H = 128: the walk wins
                    // from 3072 prefix tokens on and loses at 2048); under a short shared-prefix kernel one CTA per head,
                    // which spreads over the whole GPU as soon as that kernel ends, is faster.  A 64-token tile of the 8-bit
                    // cache takes 1.0 us, with more than 64 rows 1.3 (H = 128, us per step, one CTA per head / walk: 64
                    // requests over 1900 tokens 65.4 / 53.2, over 2400 69.7 / 59.6, 100 over 1500 74.3 / 65.5).
                    int64_t head_tiles = 0;
                    for (int j = 0; j < n_jobs; ++j) head_tiles += (jobs[j].sh->Ls + 63) / 64;
                    const int64_t tiles_per_cta = (head_tiles * H + jobs[0].n_ranges - 1) / jobs[0].n_ranges;
                    const int heads_per_cta = (H + free_sms - 1) / free_sms;
                    const double tile_us = jobs[0].sh->fp8 ? (jobs[0].rows <= 64 ? 1.0 : 1.3) : 0.7;
                    if ((double)tiles_per_cta * tile_us >= 4.0 * heads_per_cta) walk_ctas = free_sms;
                }
            }
            e = launch_q_absorb_sm100(q_nope, &sh->tm_wuk_t, q_abs, B, H, sh->num_sms, walk_ctas, sh->status, order ? seq_lens : nullptr, order,
                                      block_table, max_pages, page_size, desc, s);
        } else {
            GemmTN g1{q_nope, (int64_t)H * 128, 128, sh->w_uk_t, 128, 512 * 128, q_abs, (int64_t)H * 512, 512,
                      B, 512, 128, H, false};
            e = launch_gemm_tn(g1, s);
            if (e == cudaSuccess && order) {
                e = launch_order_by_length(seq_lens, B, order, s);
                ++launches;
            }
        }
        prof_after(TYPHOON_MLA_KERNEL_Q_ABSORB, s);
        if (e != cudaSuccess) return fail(e);
        ++launches;
        // --- absorb attention over latent tokens (Algorithm 1 line 6)
        float* o_part_a = reinterpret_cast<float*>(ws + pl.off_opart_a);
        float* lse_part_a = reinterpret_cast<float*>(ws + pl.off_lsepart_a);
        void* o_lat = ws + pl.off_olat;
        AbsorbAttn ab{q_abs, q_pe, sh->ckv, sh->kpe, mode == TYPHOON_MLA_MODE_ABSORB ? (int)sh->Ls : 0,
                      ckv_pages, kpe_pages, ckv_token_stride, kpe_token_stride, page_size, num_pages, block_table, max_pages,
                      seq_lens, order, desc, B, H, pl.chunk, pl.n_shared_chunks, pl.n_suffix_chunks, softmax_scale,
                      o_part_a, lse_part_a, sh->status, forked ? nullptr : sh->w_uv, cfg.stacked_absorb};
        prof_before(TYPHOON_MLA_KERNEL_ABSORB_ATTN, s);
        if (!tc) e = launch_absorb_attn_mma(ab, s);
        else if (pl.absorb_pairs) e = launch_absorb_pair_sm100(ab, sh->Ls_pad, o_lat, lse_a, sh->status, s);
        else e = launch_absorb_attn_sm100(ab, &sh->tm_ckv, &sh->tm_kpe_tok, o_lat, lse_a, sh->status, s);
        prof_after(TYPHOON_MLA_KERNEL_ABSORB_ATTN, s);
        if (e != cudaSuccess) return fail(e);
        ++launches;
        if (n_jobs == 0 && n_empties == 0 && n_chunks > 1 && (int64_t)B * H <= sh->num_sms) {
            // Absorb-only with at most one (request, head) row per SM: merge + projection + rounding in one launch, a block
            // per row (one block fills an SM's registers).  Measured (B200, us per step, this form / merge and GEMM): 16
            // heads, 8 requests 21.4 / 23.9; 128 heads, 1 request 28.9 / 33; in two waves it loses: 128 heads, 2 requests
            // 39.4 / 36.8; 16 heads, 16 requests 27.5 / 24.7.
            prof_before(TYPHOON_MLA_KERNEL_MERGE, s);
            e = launch_merge_project(o_part_a, lse_part_a, n_chunks, B, H, sh->w_uv, out, lse_out, out_fp32, s);
            prof_after(TYPHOON_MLA_KERNEL_MERGE, s);
            if (e != cudaSuccess) return fail(e);
            g_last_launches = launches + 1;
            return TYPHOON_MLA_OK;
        }
        if (!(tc && n_chunks == 1)) {   // a single-chunk tcgen05 launch has already written the merged result
            prof_before(TYPHOON_MLA_KERNEL_MERGE, s);
            e = launch_merge_latent(o_part_a, lse_part_a, n_chunks, B, H, o_lat, lse_a, s);
            prof_after(TYPHOON_MLA_KERNEL_MERGE, s);
            if (e != cudaSuccess) return fail(e);
            ++launches;
        }
        if (forked) {
            e = cudaEventRecord(sh->ev_join, sh->side_stream);
            if (e == cudaSuccess) e = cudaStreamWaitEvent(s_main, sh->ev_join, 0);
            open_fork = false;
            if (e != cudaSuccess) return cuda_fail(e);
            s = s_main;
        }
        // --- output projection O_A W_UV^T (Algorithm 1 line 7); on the tcgen05 path its epilogue also does the
        //     LSE combine (line 8)
        prof_before(TYPHOON_MLA_KERNEL_W_UV, s);
        if (tc) {
            CombineEpilogue ce;
            ce.o_naive = o_part_n; ce.lse_naive = lse_part_n; ce.n_naive = pl.n_slots_naive;
            ce.lse_abs = lse_a; ce.out = out; ce.lse_out = lse_out; ce.H = H;
            ce.out_fp32 = out_fp32 ? 1 : 0;
            bool any_8bit = false;
            for (int j = 0; j < n_jobs; ++j) any_8bit = any_8bit || jobs[j].sh->fp8 != 0;
            e = launch_project_sm100(o_lat, sh->w_uv, B, any_8bit, sh->num_sms, sh->status, s, ce);
            combined = true;
        } else {
            GemmTN g2{o_lat, (int64_t)H * 512, 512, sh->w_uv, 512, 128 * 512, o_abs, (int64_t)H * 128, 128,
                      B, 128, 512, H, true};
            e = launch_gemm_tn(g2, s);
        }
        prof_after(TYPHOON_MLA_KERNEL_W_UV, s);
        if (e != cudaSuccess) return fail(e);
        ++launches;
    }
    // --- LSE combine (Algorithm 1 line 8)
    if (!combined) {
        prof_before(TYPHOON_MLA_KERNEL_COMBINE, s);
        e = launch_combine(o_part_n, lse_part_n, pl.n_slots_naive, have_absorb ? o_abs : nullptr, lse_a, B, H, out,
                           lse_out, s, out_fp32);
        prof_after(TYPHOON_MLA_KERNEL_COMBINE, s);
        if (e != cudaSuccess) return fail(e);
        ++launches;
    }
    g_last_launches = launches;
    return TYPHOON_MLA_OK;
}

static int decode_impl(const typhoon_mla_shared_t* sh, const void* q_nope, const void* q_pe, int32_t B,
                       const void* ckv_pages, const void* kpe_pages, int64_t ckv_token_stride,
                       int64_t kpe_token_stride, int32_t page_size, int32_t num_pages, const int32_t* block_table,
                       int32_t max_pages, const int32_t* seq_lens, float softmax_scale, int32_t mode, void* out,
                       float* lse_out, void* workspace, size_t workspace_bytes, void* stream, bool out_fp32) {
    g_last_launches = 0;
    if (!sh || !q_nope || !q_pe || !out || B < 1 || max_pages < 0) return TYPHOON_MLA_ERR_INVALID_ARG;
    if (!on_handle_device(sh)) return TYPHOON_MLA_ERR_INVALID_ARG;
    const Settings cfg = snapshot();
    if (page_size != 64 && page_size != 128) return TYPHOON_MLA_ERR_INVALID_ARG;
    if (mode < TYPHOON_MLA_MODE_AUTO || mode > TYPHOON_MLA_MODE_NAIVE) return TYPHOON_MLA_ERR_INVALID_ARG;
    if (!aligned16(q_nope) || !aligned16(q_pe) || !aligned16(out)) return TYPHOON_MLA_ERR_INVALID_ARG;
    if (!(softmax_scale > 0.f) || softmax_scale > 3.0e38f) return TYPHOON_MLA_ERR_INVALID_ARG;   // positive, finite
    mode = resolve_mode(sh, B, max_pages, mode);
    const bool use_absorb = mode != TYPHOON_MLA_MODE_NAIVE;
    if (use_absorb && max_pages > 0) {
        if (!ckv_pages || !kpe_pages || !block_table || !seq_lens || num_pages < 1) return TYPHOON_MLA_ERR_INVALID_ARG;
        if (!aligned16(ckv_pages) || !aligned16(kpe_pages) || ckv_token_stride < 512 || kpe_token_stride < 64 ||
            ckv_token_stride % 8 || kpe_token_stride % 8)
            return TYPHOON_MLA_ERR_INVALID_ARG;
    }
    if (mode == TYPHOON_MLA_MODE_NAIVE && sh->Ls == 0) max_pages = 0;
    if (!workspace || (reinterpret_cast<uintptr_t>(workspace) & 255u)) return TYPHOON_MLA_ERR_INVALID_ARG;
    const Plan pl = make_plan(sh, cfg.tc(), cfg.naive_schedule, B, use_absorb ? max_pages : 0, page_size, mode, -1, cfg.stacked_absorb,
                              std::max<size_t>(workspace_bytes, 1));
    if (workspace_bytes < pl.total) return TYPHOON_MLA_ERR_WORKSPACE_TOO_SMALL;

    NaiveJob job{sh, 0, B, pl.n_split_naive, pl.n_slots_naive, 0};
    return decode_core(cfg, sh, &job, pl.n_split_naive > 0 ? 1 : 0, nullptr, 0, pl, q_nope, q_pe, B, ckv_pages, kpe_pages,
                       ckv_token_stride, kpe_token_stride, page_size, num_pages, block_table, use_absorb ? max_pages : 0,
                       seq_lens, softmax_scale, mode, out, lse_out, workspace, stream, out_fp32);
}

int typhoon_mla_decode(const typhoon_mla_shared_t* sh, const void* q_nope, const void* q_pe, int32_t B,
                       const void* ckv_pages, const void* kpe_pages, int64_t ckv_token_stride,
                       int64_t kpe_token_stride, int32_t page_size, int32_t num_pages, const int32_t* block_table,
                       int32_t max_pages, const int32_t* seq_lens, float softmax_scale, int32_t mode, void* out,
                       float* lse_out, void* workspace, size_t workspace_bytes, void* stream) {
    return decode_impl(sh, q_nope, q_pe, B, ckv_pages, kpe_pages, ckv_token_stride, kpe_token_stride, page_size, num_pages,
                       block_table, max_pages, seq_lens, softmax_scale, mode, out, lse_out, workspace, workspace_bytes, stream,
                       false);
}

// ---- context sharded over several devices: per-device partial + merge -----------------------------
int typhoon_mla_decode_partial(const typhoon_mla_shared_t* sh, const void* q_nope, const void* q_pe, int32_t B,
                               const void* ckv_pages, const void* kpe_pages, int64_t ckv_token_stride,
                               int64_t kpe_token_stride, int32_t page_size, int32_t num_pages,
                               const int32_t* block_table, int32_t max_pages, const int32_t* seq_lens,
                               float softmax_scale, int32_t mode, float* out_partial, float* lse_partial,
                               void* workspace, size_t workspace_bytes, void* stream) {
    if (!lse_partial) return TYPHOON_MLA_ERR_INVALID_ARG;
    return decode_impl(sh, q_nope, q_pe, B, ckv_pages, kpe_pages, ckv_token_stride, kpe_token_stride, page_size, num_pages,
                       block_table, max_pages, seq_lens, softmax_scale, mode, out_partial, lse_partial, workspace,
                       workspace_bytes, stream, true);
}

int typhoon_mla_combine_partials(const float* o_parts, const float* lse_parts, int32_t n_parts, int32_t B, int32_t H,
                                 void* out, float* lse_out, void* stream) {
    if (!o_parts || !lse_parts || !out || n_parts < 1 || B < 1 || H < 1) return TYPHOON_MLA_ERR_INVALID_ARG;
    if (!aligned16(o_parts) || !aligned16(out)) return TYPHOON_MLA_ERR_INVALID_ARG;
    tmla::tl_pdl = g_pdl.load();
    const cudaError_t e = launch_combine(o_parts, lse_parts, n_parts, nullptr, nullptr, B, H, out, lse_out,
                                         reinterpret_cast<cudaStream_t>(stream));
    if (e != cudaSuccess) return cuda_fail(e);
    g_last_launches = 1;
    return TYPHOON_MLA_OK;
}
// ---- several shared prefixes per step (tree-structured prompts) ------------------------------------
namespace {
constexpr int kMaxLevels = 8, kMaxTreeJobs = 256;
struct TreePlan {
    const typhoon_mla_shared* sh0 = nullptr;   // first prefix: weights, absorb-side tensor maps, side stream, status
    NaiveJob jobs[kMaxTreeJobs];
    EmptySlots empties[kMaxTreeJobs];
    int n_jobs = 0, n_empties = 0, total_slots = 0;
};
// `beside`: the step has an absorb branch.  (It is taken to have kTreeSuffix tokens per request whatever the table holds: the slots
// must not depend on the width, or a narrower table could need more of them than the workspace was sized for.)
constexpr int64_t kTreeSuffix = 512;
int plan_tree(const typhoon_mla_prefix_level_t* levels, int n_levels, int B, int schedule, bool beside, TreePlan* tp) {
    if (!levels || n_levels < 1 || n_levels > kMaxLevels || B < 1) return TYPHOON_MLA_ERR_INVALID_ARG;
    for (int l = 0; l < n_levels && !tp->sh0; ++l) {
        if (!levels[l].prefixes || !levels[l].group_begin || levels[l].n_groups < 1) return TYPHOON_MLA_ERR_INVALID_ARG;
        for (int g = 0; g < levels[l].n_groups && !tp->sh0; ++g) tp->sh0 = levels[l].prefixes[g];
    }
    if (!tp->sh0) return TYPHOON_MLA_ERR_INVALID_ARG;
    const int H = tp->sh0->dims.num_heads;
    const int n_sm = tp->sh0->num_sms > 0 ? tp->sh0->num_sms : kDefaultNumSM;
    int level_of[kMaxTreeJobs], slots_of[kMaxTreeJobs], merge0 = 0;   // jobs [merge0, n_jobs) can share launches
    // Prefixes that can share a launch come last: the large ones keep their place at the front of the caller's stream (behind a
    // shared launch a root of 195 rows x 128 heads x 8572 tokens made the step 11 % longer).  One launch per prefix leaves SMs idle at every launch's end and pays
    // set-up and pipeline fill once per (prefix, head); in a shared launch a CTA goes on from one prefix's tiles to the
    // next one's.  (16-bit cache, at most 128 rows: the row groups of larger ones differ in number.)
    auto mergeable = [](const NaiveJob& j) { return !j.sh->fp8 && j.rows <= 128; };
    for (int pass = 0; pass < 2; ++pass) {
        for (int l = 0; l < n_levels; ++l) {
            const typhoon_mla_prefix_level_t& lv = levels[l];
            if (!lv.prefixes || !lv.group_begin || lv.n_groups < 1) return TYPHOON_MLA_ERR_INVALID_ARG;
            if (lv.group_begin[0] != 0 || lv.group_begin[lv.n_groups] != B) return TYPHOON_MLA_ERR_INVALID_ARG;
            for (int g = 0; g < lv.n_groups; ++g) {
                const int r0 = lv.group_begin[g], r1 = lv.group_begin[g + 1];
                if (r1 < r0) return TYPHOON_MLA_ERR_INVALID_ARG;
                const typhoon_mla_shared* sh = lv.prefixes[g];
                if (sh && (sh->dims.num_heads != H || sh->device != tp->sh0->device)) return TYPHOON_MLA_ERR_INVALID_ARG;
                if (!sh || sh->Ls == 0 || r1 == r0) continue;
                const NaiveJob job{sh, r0, r1 - r0, 0, 0, 0};
                if (mergeable(job) != (pass == 1)) continue;
                if (tp->n_jobs == kMaxTreeJobs) return TYPHOON_MLA_ERR_INVALID_ARG;
                level_of[tp->n_jobs] = l;
                tp->jobs[tp->n_jobs++] = job;
            }
        }
        if (pass == 0) merge0 = tp->n_jobs;
    }
    for (int j = 0; j < tp->n_jobs;) {
        const int n = j >= merge0 ? std::min(kNaiveJobsPerLaunch, tp->n_jobs - j) : 1;
        int ranges = 0;
        if (n > 1) {
            int64_t len[kNaiveJobsPerLaunch];
            int rows = 0;
            for (int k = 0; k < n; ++k) {
                len[k] = tp->jobs[j + k].sh->Ls;
                rows = std::max(rows, tp->jobs[j + k].rows);
            }
            naive_sm100_plan_multi(rows, H, len, n, n_sm, schedule, &ranges, &slots_of[j]);
        } else {
            const bool fp8 = tp->jobs[j].sh->fp8 != 0;
            const int rows = tp->jobs[j].rows, places = naive_places(rows, n_sm, fp8);
            naive_sm100_plan(rows, H, tp->jobs[j].sh->Ls, places, schedule, &ranges, &slots_of[j], fp8,
                             beside ? absorb_branch_us(B, H, kTreeSuffix) : 0.0);
        }
        for (int k = 0; k < n; ++k) tp->jobs[j + k].n_ranges = ranges;
        tp->jobs[j].n_merged = n;
        j += n;
    }
    int slot0 = 0;
    for (int l = 0; l < n_levels; ++l) {
        const typhoon_mla_prefix_level_t& lv = levels[l];
        int level_slots = 0;
        for (int j = 0; j < tp->n_jobs; ++j)
            if (level_of[j] == l) level_slots = std::max(level_slots, slots_of[j]);
        if (level_slots == 0) continue;   // no prefix at this level at all: no slots
        for (int j = 0; j < tp->n_jobs; ++j)
            if (level_of[j] == l) {
                tp->jobs[j].n_slots_level = level_slots;
                tp->jobs[j].slot0 = slot0;
            }
        for (int g = 0; g < lv.n_groups; ++g) {
            const int r0 = lv.group_begin[g], r1 = lv.group_begin[g + 1];
            const typhoon_mla_shared* sh = lv.prefixes[g];
            if ((sh && sh->Ls > 0) || r1 == r0) continue;
            if (tp->n_empties == kMaxTreeJobs) return TYPHOON_MLA_ERR_INVALID_ARG;
            tp->empties[tp->n_empties++] = EmptySlots{slot0, level_slots, r0, r1 - r0};
        }
        slot0 += level_slots;
    }
    tp->total_slots = slot0;
    return TYPHOON_MLA_OK;
}
}  // namespace

size_t typhoon_mla_tree_workspace_bytes(const typhoon_mla_prefix_level_t* levels, int32_t n_levels, int32_t B,
                                        int32_t max_pages, int32_t page_size) {
    if (max_pages < 0 || (page_size != 64 && page_size != 128)) return 0;
    // worst case over the work decompositions a test hook may select (the tree step needs the tcgen05 kernels), with and without
    // an absorb branch, and the floor (make_plan)
    size_t worst = 0;
    for (int schedule : {0, 1, 2})
        for (bool beside : {true, false}) {
            TreePlan tp;
            if (plan_tree(levels, n_levels, B, schedule, beside, &tp) != TYPHOON_MLA_OK) return 0;
            for (size_t bytes : {SIZE_MAX, (size_t)0})
                worst = std::max(worst, make_plan(tp.sh0, true, schedule, B, max_pages, page_size, TYPHOON_MLA_MODE_HYBRID, tp.total_slots, true,
                                                  bytes).total);
        }
    return worst + 256;
}

int typhoon_mla_decode_tree(const typhoon_mla_prefix_level_t* levels, int32_t n_levels, const void* q_nope,
                            const void* q_pe, int32_t B, const void* ckv_pages, const void* kpe_pages,
                            int64_t ckv_token_stride, int64_t kpe_token_stride, int32_t page_size, int32_t num_pages,
                            const int32_t* block_table, int32_t max_pages, const int32_t* seq_lens, float softmax_scale,
                            void* out, float* lse_out, void* workspace, size_t workspace_bytes, void* stream) {
    g_last_launches = 0;
    if (!q_nope || !q_pe || !out || B < 1 || max_pages < 0) return TYPHOON_MLA_ERR_INVALID_ARG;
    if (page_size != 64 && page_size != 128) return TYPHOON_MLA_ERR_INVALID_ARG;
    if (!aligned16(q_nope) || !aligned16(q_pe) || !aligned16(out)) return TYPHOON_MLA_ERR_INVALID_ARG;
    if (!(softmax_scale > 0.f) || softmax_scale > 3.0e38f) return TYPHOON_MLA_ERR_INVALID_ARG;
    const Settings cfg = snapshot();
    if (!cfg.tc()) return TYPHOON_MLA_ERR_UNSUPPORTED_DIMS;
    if (max_pages > 0) {
        if (!ckv_pages || !kpe_pages || !block_table || !seq_lens || num_pages < 1) return TYPHOON_MLA_ERR_INVALID_ARG;
        if (!aligned16(ckv_pages) || !aligned16(kpe_pages) || ckv_token_stride < 512 || kpe_token_stride < 64 ||
            ckv_token_stride % 8 || kpe_token_stride % 8)
            return TYPHOON_MLA_ERR_INVALID_ARG;
    }
    TreePlan tp;
    const int rc = plan_tree(levels, n_levels, B, cfg.naive_schedule, max_pages > 0, &tp);
    if (rc != TYPHOON_MLA_OK) return rc;
    if (!on_handle_device(tp.sh0)) return TYPHOON_MLA_ERR_INVALID_ARG;
    // NAIVE when there is no page table (nothing for the absorb branch), else Algorithm 1 with several line-4 launches
    const int mode = max_pages == 0 ? TYPHOON_MLA_MODE_NAIVE : TYPHOON_MLA_MODE_HYBRID;
    if (!workspace || (reinterpret_cast<uintptr_t>(workspace) & 255u)) return TYPHOON_MLA_ERR_INVALID_ARG;
    const Plan pl = make_plan(tp.sh0, true, cfg.naive_schedule, B, max_pages, page_size, mode, tp.total_slots, true,
                              std::max<size_t>(workspace_bytes, 1));
    if (workspace_bytes < pl.total) return TYPHOON_MLA_ERR_WORKSPACE_TOO_SMALL;
    return decode_core(cfg, tp.sh0, tp.jobs, tp.n_jobs, tp.empties, tp.n_empties, pl, q_nope, q_pe, B, ckv_pages, kpe_pages,
                       ckv_token_stride, kpe_token_stride, page_size, num_pages, block_table, max_pages, seq_lens,
                       softmax_scale, mode, out, lse_out, workspace, stream);
}

int typhoon_mla_profile_begin(int32_t kernel_id, int32_t max_launches) {
    if (kernel_id < 0 || kernel_id >= TYPHOON_MLA_NUM_KERNELS || max_launches < 1) return TYPHOON_MLA_ERR_INVALID_ARG;
    if (g_prof.ev) return TYPHOON_MLA_ERR_INVALID_ARG;
    g_prof.ev = new (std::nothrow) cudaEvent_t[2 * (size_t)max_launches];
    if (!g_prof.ev) return TYPHOON_MLA_ERR_ALLOC;
    for (int i = 0; i < 2 * max_launches; ++i) {
        cudaError_t e = cudaEventCreate(&g_prof.ev[i]);
        if (e != cudaSuccess) {
            for (int j = 0; j < i; ++j) cudaEventDestroy(g_prof.ev[j]);
            delete[] g_prof.ev;
            g_prof.ev = nullptr;
            return cuda_fail(e);
        }
    }
    g_prof.capacity = max_launches;
    g_prof.used = 0;
    g_prof.kernel_id = kernel_id;
    return TYPHOON_MLA_OK;
}

int typhoon_mla_profile_end(double* total_ms, int32_t* launches) {
    if (!g_prof.ev) return TYPHOON_MLA_ERR_INVALID_ARG;
    double tot = 0.0;
    int st = TYPHOON_MLA_OK;
    for (int i = 0; i < g_prof.used; ++i) {
        float ms = 0.f;
        cudaError_t e = cudaEventSynchronize(g_prof.ev[2 * i + 1]);
        if (e == cudaSuccess) e = cudaEventElapsedTime(&ms, g_prof.ev[2 * i], g_prof.ev[2 * i + 1]);
        if (e != cudaSuccess) { st = cuda_fail(e); break; }
        tot += ms;
    }
    if (total_ms) *total_ms = tot;
    if (launches) *launches = g_prof.used;
    for (int i = 0; i < 2 * g_prof.capacity; ++i) cudaEventDestroy(g_prof.ev[i]);
    delete[] g_prof.ev;
    g_prof = Profile();
    return st;
}

// Steps whose inputs in host memory are at most this many bytes are copied, in and out, by a kernel of ours, larger ones by
// the copy engines.  Every engine copy costs a hand-over of several microseconds between engine and kernels, but engines
// run beside other streams' kernels for nothing, while copying blocks share the SMs with them.  Measured (B200, us per step,
// engines / kernel): one step at a time 4 requests x 16 heads 51 / 31, 8 x 128 (0.4 MB in, 0.26 MB out) 80 / 59, 32 x 128
// (1.6 / 1.0 MB) 249 / 233; twelve streams 42 / 36, 42 / 41, 73 / 83 (64 x 128, 3.1 / 2.1 MB: 98 / 140).  The line lies where
// no number of streams loses (10 x 128: 84 / 64 and 43 / 42; 14 x 128: 101 / 77 and 46 / 48); one direction by either means
// loses as well (24 x 64, engines in and kernel out, two streams: 48 / 53).
constexpr int64_t kKernelCopyMaxBytes = 512 << 10;

// Address under which kernels may access [p, p + bytes) of host memory, or null: pageable memory, an address 4-byte words
// cannot start at, or a range that is not shown to lie inside ONE pinned allocation or registration.  (Two pinned ends
// prove nothing about the middle: pinned memory is mapped at its own address, so the ends of an array that crosses
// pageable memory are as far apart on the device as on the host.)  One driver query gives type, device address and range.
static void* device_view(const void* p, int64_t bytes) {
    typedef CUresult (*QueryFn)(unsigned, CUpointer_attribute*, void**, CUdeviceptr);
    static const QueryFn query = [] {
        void* fn = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPoint("cuPointerGetAttributes", &fn, cudaEnableDefault, &q) != cudaSuccess || q != cudaDriverEntryPointSuccess) {
            cudaGetLastError();
            fn = nullptr;
        }
        return reinterpret_cast<QueryFn>(fn);
    }();
    const uintptr_t host = reinterpret_cast<uintptr_t>(p);
    if (!query || host == 0 || (host & 3) || bytes <= 0) return nullptr;
    unsigned type = 0, managed = 0;
    CUdeviceptr dev = 0, first = 0;
    size_t size = 0;
    CUpointer_attribute what[5] = {CU_POINTER_ATTRIBUTE_MEMORY_TYPE, CU_POINTER_ATTRIBUTE_IS_MANAGED, CU_POINTER_ATTRIBUTE_DEVICE_POINTER,
                                   CU_POINTER_ATTRIBUTE_RANGE_START_ADDR, CU_POINTER_ATTRIBUTE_RANGE_SIZE};
    void* into[5] = {&type, &managed, &dev, &first, &size};
    // (what does not apply to `p` comes back as zero)
    if (query(5, what, into, (CUdeviceptr)host) != CUDA_SUCCESS || type != CU_MEMORYTYPE_HOST || managed || dev == 0) return nullptr;
    if (first == 0 || dev < first || dev - first > size || size - (dev - first) < (size_t)bytes) return nullptr;
    return reinterpret_cast<void*>(dev);
}

int typhoon_mla_host_range_mapped(const void* p, int64_t bytes) { return device_view(p, bytes) != nullptr ? 1 : 0; }

size_t typhoon_mla_host_staging_bytes(const typhoon_mla_shared_t* sh, int32_t B, int32_t max_pages) {
    if (!sh || B < 1 || max_pages < 0) return 0;
    const size_t BH = (size_t)B * sh->dims.num_heads;
    return round_up(BH * 128 * 2, 256) + round_up(BH * 64 * 2, 256) + round_up((size_t)B * std::max(max_pages, 1) * 4, 256) +
           round_up((size_t)B * 4, 256) + round_up(BH * 128 * 2, 256);
}

int typhoon_mla_decode_host(const typhoon_mla_shared_t* sh, const void* q_nope_host, const void* q_pe_host, int32_t B,
                            const void* ckv_pages, const void* kpe_pages, int64_t ckv_token_stride,
                            int64_t kpe_token_stride, int32_t page_size, int32_t num_pages,
                            const int32_t* block_table_host, int32_t max_pages, const int32_t* seq_lens_host,
                            float softmax_scale, int32_t mode,
                            void* out_host, void* staging, size_t staging_bytes, void* workspace,
                            size_t workspace_bytes, void* stream) {
    if (!sh || !q_nope_host || !q_pe_host || !out_host || !staging || B < 1 || max_pages < 0)
        return TYPHOON_MLA_ERR_INVALID_ARG;
    if (max_pages > 0 && (!block_table_host || !seq_lens_host)) return TYPHOON_MLA_ERR_INVALID_ARG;
    if (staging_bytes < typhoon_mla_host_staging_bytes(sh, B, max_pages)) return TYPHOON_MLA_ERR_WORKSPACE_TOO_SMALL;
    if (reinterpret_cast<uintptr_t>(staging) & 255u) return TYPHOON_MLA_ERR_INVALID_ARG;
    cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
    const size_t BH = (size_t)B * sh->dims.num_heads;
    char* st = reinterpret_cast<char*>(staging);
    char* d_qn = st;
    char* d_qp = d_qn + round_up(BH * 128 * 2, 256);
    char* d_bt = d_qp + round_up(BH * 64 * 2, 256);
    char* d_sl = d_bt + round_up((size_t)B * std::max(max_pages, 1) * 4, 256);
    char* d_out = d_sl + round_up((size_t)B * 4, 256);
    const void* const in_host[4] = {q_nope_host, q_pe_host, block_table_host, seq_lens_host};
    void* const in_dev[4] = {d_qn, d_qp, d_bt, d_sl};
    const int64_t in_bytes[4] = {(int64_t)BH * 256, (int64_t)BH * 128, (int64_t)B * max_pages * 4, max_pages > 0 ? (int64_t)B * 4 : 0};
    const int64_t out_bytes = (int64_t)BH * 256;
    tmla::tl_pdl = g_pdl.load();
    const void* src[4] = {};
    void* out_dev = nullptr;
    bool mapped = in_bytes[0] + in_bytes[1] + in_bytes[2] + in_bytes[3] <= kKernelCopyMaxBytes;
    for (int i = 0; i < 4 && mapped; ++i)
        if (in_bytes[i] > 0) mapped = (src[i] = device_view(in_host[i], in_bytes[i])) != nullptr;
    if (mapped) mapped = (out_dev = device_view(out_host, out_bytes)) != nullptr;
    cudaError_t e = cudaSuccess;
    if (mapped) {
        e = launch_host_copy(src, in_dev, in_bytes, 4, s);
    } else {
        for (int i = 0; i < 4 && e == cudaSuccess; ++i)
            if (in_bytes[i] > 0) e = cudaMemcpyAsync(in_dev[i], in_host[i], in_bytes[i], cudaMemcpyHostToDevice, s);
    }
    if (e != cudaSuccess) return cuda_fail(e);
    int st_code = typhoon_mla_decode(sh, d_qn, d_qp, B, ckv_pages, kpe_pages, ckv_token_stride, kpe_token_stride,
                                     page_size, num_pages, reinterpret_cast<const int32_t*>(d_bt), max_pages,
                                     reinterpret_cast<const int32_t*>(d_sl), softmax_scale, mode, d_out, nullptr,
                                     workspace, workspace_bytes, stream);
    if (st_code != TYPHOON_MLA_OK) return st_code;
    if (mapped) {
        const void* out_src = d_out;
        e = launch_host_copy(&out_src, &out_dev, &out_bytes, 1, s);
    } else {
        e = cudaMemcpyAsync(out_host, d_out, out_bytes, cudaMemcpyDeviceToHost, s);
    }
    if (e != cudaSuccess) return cuda_fail(e);
    return TYPHOON_MLA_OK;
}

}  // extern "C"
