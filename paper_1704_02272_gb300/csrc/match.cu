// Match entry points: kernel selection, workspace layout, the ordering
// kernels, and the C ABI calls pfac_workspace_bytes / pfac_match_async /
// pfac_match (Section 2.3 semantics; see include/pfac.h).
#include <cuda_runtime.h>
#include <math.h>
#include <stdio.h>
#include <string.h>

#include <algorithm>
#include <mutex>

#include "internal.h"
#include "kernels_d.cuh"

namespace pfac {

void *scan_kernel_bps1(int, int, int, int);
void *scan_kernel_bps2(int, int, int, int);
void *scan_kernel_bps3(int, int, int, int);
void *scan_kernel_bps4(int, int, int, int);
void *scan_kernel_bps5(int, int, int, int);
void *scan_kernel_bps6(int, int, int, int);
void *scan_kernel_bps7(int, int, int, int);
void *scan_kernel_bps8(int, int, int, int);
void *scan_kernel_dense();
void *scan_kernel_r8_g0_f(int rep, int nw);
void *scan_kernel_r8_g0_fe(int rep, int nw);
void *scan_kernel_r8_g1_f(int rep, int nw);
void *scan_kernel_r8_g1_fe(int rep, int nw);
void *scan_kernel_r2_g0_f(int rep, int nw);
void *scan_kernel_r2_g0_fe(int rep, int nw);
void *scan_kernel_r2_g1_f(int rep, int nw);
void *scan_kernel_r2_g1_fe(int rep, int nw);

void *resolve_kernel(int w);
void *wresolve_kernel(int w);
void *dresolve_kernel(int w);
void *scan_kernel_d(bool entries_in_smem);
void *scan_kernel_w1(bool packed, uint32_t nb, bool g5, int tb);
void *scan_kernel_w2(bool packed, uint32_t nb, bool g5, int tb);
void *scan_kernel_w4(bool packed, uint32_t nb, bool g5, int tb);
void *scan_kernel_w8(bool packed, uint32_t nb, bool g5, int tb);
void *scan_kernel_w16(bool packed, uint32_t nb, bool g5, int tb);
void *scan_kernel_r8_d0(int rep, int var, int nw);
void *scan_kernel_r8_d1(int rep, int var, int nw);
void *scan_kernel_r2_d0(int rep, int var, int nw);
void *scan_kernel_r2_d1(int rep, int var, int nw);

// the register-staged kernel for 8-bit or 2-bit symbols
static void *scan_kernel_r(uint32_t bps, uint32_t w, int rep, bool gram, int var, int nw) {
    if (w == 3) {  // the dense layout's transition table
        if (bps == 2) return gram ? scan_kernel_r2_d1(rep, var, nw) : scan_kernel_r2_d0(rep, var, nw);
        if (bps == 8) return gram ? scan_kernel_r8_d1(rep, var, nw) : scan_kernel_r8_d0(rep, var, nw);
        return nullptr;
    }
    if (bps == 2) {
        if (w != 0) return nullptr;  // packed records only
        if (gram) return var == VAR_FE ? scan_kernel_r2_g1_fe(rep, nw) : scan_kernel_r2_g1_f(rep, nw);
        return var == VAR_FE ? scan_kernel_r2_g0_fe(rep, nw) : scan_kernel_r2_g0_f(rep, nw);
    }
    if (bps != 8) return nullptr;
    if (gram) return var == VAR_FE ? scan_kernel_r8_g1_fe(rep, nw) : scan_kernel_r8_g1_f(rep, nw);
    return var == VAR_FE ? scan_kernel_r8_g0_fe(rep, nw) : scan_kernel_r8_g0_f(rep, nw);
}

// the window kernel for a table's filter
static void *scan_kernel_w(const DevTable &T, int tb) {
    const bool packed = T.w_packed != 0, g5 = !packed && T.w_gw == 5;
    switch (T.w_stride) {
        case 1: return scan_kernel_w1(packed, T.w_nb, g5, tb);
        case 2: return scan_kernel_w2(packed, T.w_nb, g5, tb);
        case 4: return scan_kernel_w4(packed, T.w_nb, g5, tb);
        case 8: return scan_kernel_w8(packed, T.w_nb, g5, tb);
        case 16: return scan_kernel_w16(packed, T.w_nb, g5, tb);
        default: return nullptr;
    }
}

// chunks of the key-count scan: the fewest units each (a power of two) that
// keep their number within CHUNKS_MAX; fewer than 32 (a unit a warp at least)
// only while all chunks' CTAs run at once.  The expansion walks a full slice
// again with one warp, so in small calls its slices go to as many warps as
// there are (50,000 signatures over printable text, 32 units a chunk / this
// rule: 64 KiB 161 / 85 us, 1 MiB 164 / 92, 9 MB 337 / 302; the kernels before
// the window path took 139, 146 and 318).
constexpr uint32_t CHUNKS_MAX = 2048;
constexpr uint32_t CHUNK_SHIFT_MIN = 3, CHUNK_SHIFT_ADDS = 5;
constexpr uint32_t CHUNKS_AT_ONCE = 1216;  // 152 SMs x 8
static uint32_t chunk_shift(uint64_t n_units) {
    uint32_t s = CHUNK_SHIFT_MIN;
    while (((n_units + (1ull << s) - 1) >> s) > (s < CHUNK_SHIFT_ADDS ? CHUNKS_AT_ONCE : CHUNKS_MAX)) s++;
    return s;
}

// ------------------------------------------------ segment bounds per tile --

// Validates the offsets and lists, per tile, the segment ends that the
// tile's positions can need: every o_s > tile start up to and including the
// first o_s >= tile end (at most SEG_MAXB, else SEG_OVF).
__global__ void k_bounds(const MatchParams P) {
    const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
    const uint64_t gt = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const uint64_t *seg = P.seg;
    for (uint64_t s = gt; s < P.n_seg; s += stride)
        if (__ldg(seg + s + 1) < __ldg(seg + s)) atomicOr(&P.hdr->status, ST_BADSEG);
    if (gt == 0 && (__ldg(seg) != 0 || __ldg(seg + P.n_seg) != P.n))
        atomicOr(&P.hdr->status, ST_BADSEG);
    for (uint64_t t = gt; t < P.n_tiles; t += stride) {
        const uint64_t start = t * TILE, end = start + TILE;
        uint32_t lo = 1, hi = P.n_seg;
        while (lo < hi) {
            const uint32_t mid = (lo + hi) >> 1;
            if (__ldg(seg + mid) > start) hi = mid; else lo = mid + 1;
        }
        uint32_t *B = P.tile_bounds + t * SEGW;
        uint32_t cnt = 0;
        bool ovf = false;
        for (uint32_t s = lo; s <= P.n_seg; s++) {
            const uint64_t o = __ldg(seg + s);
            if (cnt == SEG_MAXB) {
                ovf = true;
                break;
            }
            const uint64_t r = o > start ? o - start : 0;
            B[1 + cnt++] = r < 0xFFFFFFF0ull ? (uint32_t)r : 0xFFFFFFF0u;
            if (o >= end) break;
        }
        B[0] = ovf ? SEG_OVF : cnt;
    }
}

// The segment data of the slice kernels (the window kernel's: k_zero and
// k_wresolve).
__global__ void k_unitseg(const MatchParams P) {
    const uint32_t gt = blockIdx.x * blockDim.x + threadIdx.x;
    unit_segments<true, true>(P, gt >> 5, (gridDim.x * blockDim.x) >> 5, threadIdx.x & 31);
}

// ------------------------------------------------ key-count scan ----------

__device__ __forceinline__ uint64_t block_excl_scan(uint64_t v, uint64_t *sh, uint64_t &total) {
    const uint32_t lane = threadIdx.x & 31, w = threadIdx.x >> 5, nw = blockDim.x >> 5;
    uint64_t inc = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint64_t nb = __shfl_up_sync(0xFFFFFFFFu, inc, o);
        if (lane >= (uint32_t)o) inc += nb;
    }
    if (lane == 31) sh[w] = inc;
    __syncthreads();
    if (w == 0) {
        const uint64_t t = lane < nw ? sh[lane] : 0;
        uint64_t ti = t;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint64_t nb = __shfl_up_sync(0xFFFFFFFFu, ti, o);
            if (lane >= (uint32_t)o) ti += nb;
        }
        if (lane < nw) sh[lane] = ti - t;
        if (lane == nw - 1) sh[32] = ti;
    }
    __syncthreads();
    total = sh[32];
    const uint64_t r = sh[w] + inc - v;
    __syncthreads();
    return r;
}

// Zeroes the head of the workspace (n 16-byte words) and writes the slices'
// first offset indices, which the scan reads where it walks starts itself: a
// kernel rather than a memset, so that the scan's table fill overlaps it.  (The
// resolver checks the offsets: the status is among what is zeroed here.)  With
// the indices written by the scan launch, its own walks could not use them and
// searched all offsets: a request of 9 MB against 50,000 signatures, a fifth of
// whose starts are walked there, 74 us, with them 63; printable text 309 and
// 270.
__global__ void __launch_bounds__(256) k_zero(const __grid_constant__ MatchParams P, uint4 *p, uint64_t n) {
    const uint64_t t = (uint64_t)blockIdx.x * 256 + threadIdx.x, nt = (uint64_t)gridDim.x * 256;
    for (uint64_t i = t; i < n; i += nt) p[i] = make_uint4(0, 0, 0, 0);
    if (P.n_seg > 1) unit_segments<false, true>(P, (uint32_t)(t >> 5), (uint32_t)(nt >> 5), threadIdx.x & 31);
}

// Key counts of the chunks of units, where they are not added up as matches
// are found.
__global__ void __launch_bounds__(256) k_reduce(const MatchParams P) {
    __shared__ uint64_t sh[33];
    dep_wait();
    const uint64_t t0 = (uint64_t)blockIdx.x << P.chunk_shift;
    uint64_t sum = 0;
    for (uint64_t i = threadIdx.x; i < (1ull << P.chunk_shift); i += 256)
        if (t0 + i < P.n_tiles) sum += P.tile_k[t0 + i] & ((1ull << UNIT_KEY_BITS) - 1);
    uint64_t total;
    block_excl_scan(sum, sh, total);
    if (threadIdx.x == 0) P.chunk[blockIdx.x] = total;
}

// Output offsets and keys of one chunk of units per CTA; the last chunk's CTA
// writes the total count.  A CTA adds up the counts of the chunks before its
// own (at most CHUNKS_MAX) and scans its units' counts 8 * span at a time:
// `span` consecutive units per warp, 32, or fewer in small chunks, so that the
// chains of dependent loads run in every warp.  Units whose records were not
// kept get their offset stored for the emit pass.
//
// A warp deals its units that have records out to groups of eight lanes, one record a lane: four units at a
// time, each with one round trip for its records and one for its outputs.
// Units with more records take the whole warp, 32 records at a time.  A
// record's keys follow those of the records at lower positions: the earlier
// lanes' where the records lie in position order, else (the window kernel's
// units, at most 32 records) those found lower by comparing.
constexpr uint32_t EXPAND_GROUP = 8;  // lanes, and most records, of a group's unit

// Keys before this lane's record among the `width` lanes of its group; width
// is the unit's lanes (EXPAND_GROUP or 32).
template <uint32_t WIDTH>
__device__ __forceinline__ uint32_t keys_before(uint32_t pos, uint32_t L, bool unordered, uint32_t lane) {
    if (unordered) {
        uint32_t lower = 0;
#pragma unroll
        for (uint32_t x = 0; x < WIDTH; x++) {
            const uint32_t px = __shfl_sync(0xFFFFFFFFu, pos, x, WIDTH);
            const uint32_t lx = __shfl_sync(0xFFFFFFFFu, L, x, WIDTH);
            if (px < pos) lower += lx;
        }
        return lower;
    }
    uint32_t inc = L;
#pragma unroll
    for (uint32_t s = 1; s < WIDTH; s <<= 1) {
        const uint32_t nb = __shfl_up_sync(0xFFFFFFFFu, inc, s, WIDTH);
        if ((lane & (WIDTH - 1)) >= s) inc += nb;
    }
    return inc - L;
}

__device__ __forceinline__ void write_keys(const MatchParams &P, uint64_t r, uint32_t L, uint64_t t,
                                           uint64_t o) {
    if (!L) return;
    const uint32_t *ids = fin_ids_c(P, (uint32_t)r);
    const uint64_t pk = (P.pos_base + (t << P.unit_shift) + (r >> 32)) << PFAC_ID_BITS;
    for (uint32_t e = 0; e < L; e++, o++)
        if (o < P.cap) P.out[o] = pk | __ldg(ids + e);
}

// The keys of a unit whose records were not kept, where no emit pass follows:
// a warp walks its starts from the root, 32 at a time, in position order.
static __device__ __noinline__ void expand_unit(const MatchParams *PP, uint64_t t, uint64_t o, uint32_t lane) {
    const MatchParams &P = *PP;
    const uint64_t us = t << SLICE_SHIFT;
    for (uint32_t p0 = 0; p0 < (uint32_t)SLICE; p0 += 32) {
        const uint32_t pos = p0 + lane;
        uint32_t fin = 0, L = 0;
        if (us + pos < P.starts_end) {
            fin = w_walk_any(P, us, pos, w_limit(P, (uint32_t)t, us + pos));
            if (fin) L = fin_len_c(P, fin);
        }
        const uint32_t before = keys_before<32>(pos, L, false, lane);
        write_keys(P, ((uint64_t)pos << 32) | fin, L, t, o + before);
        o += __shfl_sync(0xFFFFFFFFu, before + L, 31);
    }
}

__global__ void __launch_bounds__(256, 8) k_expand(const __grid_constant__ MatchParams P, const uint32_t span) {
    __shared__ uint64_t sh[33];
    const uint32_t lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const uint32_t grp = lane / EXPAND_GROUP, gl = lane % EXPAND_GROUP;
    const bool un = P.unordered != 0;
    const uint32_t c = blockIdx.x;
    dep_wait();
    uint64_t base = 0;
    {
        uint64_t v = 0;
        for (uint32_t i = threadIdx.x; i < c; i += 256) v += __ldcg(P.chunk + i);
        block_excl_scan(v, sh, base);
    }
    bool over = false;
    const uint64_t c_end = ((uint64_t)c + 1) << P.chunk_shift;
    const uint64_t t_end = c_end < P.n_tiles ? c_end : P.n_tiles;
    for (uint64_t b0 = (uint64_t)c << P.chunk_shift; b0 < t_end; b0 += 8 * span) {
        const uint64_t t0 = b0 + warp * span, tl = t0 + lane;
        const bool mine = lane < span && tl < t_end;
        const uint64_t kl = mine ? P.tile_k[tl] : 0ull;
        const uint32_t ml = un ? (uint32_t)(kl >> UNIT_KEY_BITS) : (mine ? P.tile_m[tl] : 0u);
        uint64_t tot;
        const uint64_t ol = block_excl_scan(kl & ((1ull << UNIT_KEY_BITS) - 1), sh, tot) + base;
        base += tot;
        if (ml > P.unit_cap) P.key_off[tl] = ol;
        over |= ml > P.unit_cap;
        uint32_t few = __ballot_sync(0xFFFFFFFFu, ml != 0 && ml <= EXPAND_GROUP);
        uint32_t many = __ballot_sync(0xFFFFFFFFu, ml > EXPAND_GROUP && ml <= P.unit_cap);
        // the records of the next four units are loaded while the keys of
        // the current four are written
        uint32_t jn = 0;
        uint64_t rn = 0, on = 0;
        auto next_few = [&]() {
            // the group's unit: the grp-th set bit
            uint32_t f = few;
            for (uint32_t x = 0; x < grp; x++) f &= f - 1;
            jn = f ? __ffs(f) - 1 : 0u;
            const uint32_t m = __shfl_sync(0xFFFFFFFFu, ml, jn);
            on = __shfl_sync(0xFFFFFFFFu, ol, jn);
            rn = f && gl < m ? P.recs[(t0 + jn) * P.unit_cap + gl] : 0ull;
#pragma unroll
            for (uint32_t x = 0; x < 32 / EXPAND_GROUP; x++) few &= few - 1;
        };
        bool more = few != 0;
        if (more) next_few();
        while (more) {
            const uint64_t r = rn, o = on, t = t0 + jn;
            more = few != 0;
            if (more) next_few();
            const uint32_t L = (uint32_t)r ? fin_len_c(P, (uint32_t)r) : 0u;
            write_keys(P, r, L, t, o + keys_before<EXPAND_GROUP>((uint32_t)(r >> 32), L, un, lane));
        }
        // larger units: their rounds of 32 records, each loaded a round ahead
        uint32_t mn = 0, in = 0;
        auto next_many = [&](bool fresh) {
            if (fresh) {
                jn = __ffs(many) - 1;
                many &= many - 1;
                mn = __shfl_sync(0xFFFFFFFFu, ml, jn);
                in = 0;
            }
            rn = in + lane < mn ? P.recs[(t0 + jn) * P.unit_cap + in + lane] : 0ull;
            in += 32;
        };
        more = many != 0;
        if (more) next_many(true);
        uint64_t o = 0;
        while (more) {
            const uint64_t r = rn, t = t0 + jn;
            // the unit's first round starts at its offset
            const uint64_t ob = __shfl_sync(0xFFFFFFFFu, ol, jn);
            if (in == 32) o = ob;
            const bool fresh = in >= mn;
            more = !fresh || many != 0;
            if (more) next_many(fresh);
            const uint32_t L = (uint32_t)r ? fin_len_c(P, (uint32_t)r) : 0u;
            const uint32_t before = keys_before<32>((uint32_t)(r >> 32), L, un, lane);
            write_keys(P, r, L, t, o + before);
            // (unordered units end after one round)
            o += __shfl_sync(0xFFFFFFFFu, before + L, 31);
        }
    }
    if (threadIdx.x == 0 && c == gridDim.x - 1) {
        *P.d_count = base;
        if (P.n_seg <= 1) {
            const bool ok = P.n_seg == 1 ? (P.seg[0] == 0 && P.seg[1] == P.n)
                                         : (P.n == 0 && P.seg[0] == 0);
            if (!ok) atomicOr(&P.hdr->status, ST_BADSEG);
        }
    }
    // where no emit pass follows, this kernel re-walks the units whose records
    // were not kept and publishes the status: its last chunk's CTA can, as no
    // other one changes it (in the checked build every one may)
    if (P.no_emit && __any_sync(0xFFFFFFFFu, over)) {
        __syncwarp();
        for (uint64_t b0 = (uint64_t)c << P.chunk_shift; b0 < t_end; b0 += 8 * span) {
            const uint64_t t0 = b0 + warp * span, tl = t0 + lane;
            const bool full = lane < span && tl < t_end && (P.tile_k[tl] >> UNIT_KEY_BITS) > P.unit_cap;
            uint32_t m = __ballot_sync(0xFFFFFFFFu, full && un);
            while (m) {
                const uint32_t j = __ffs(m) - 1;
                m &= m - 1;
                expand_unit(&P, t0 + j, P.key_off[t0 + j], lane);
            }
        }
    }
    if (P.no_emit || P.n_tiles == 0) {
        if (CHECKED) __syncthreads();
        if (threadIdx.x == 0 && (CHECKED || c == gridDim.x - 1)) publish_status(P, CHECKED ? gridDim.x : 1);
    }
}

// ------------------------------------------------ host side ---------------

struct Plan {
    int var;
    uint32_t k;
    uint32_t tbl_words, tbl_c_words, tbl_e_words, tbl_m_words;
    uint32_t rep_log2;
    uint32_t tbl_g_words, g_rep, g_fold;  // gram filter: words (all copies), copies, fold
    uint32_t tbl_b_words;                 // prefix bytes as the first stage
    uint32_t nw;                          // warps per CTA of the queued kernel
    uint32_t dense_rows;
    uint32_t unit_shift, unit_cap;
    void *kernel;       // scan pass
    void *kernel_emit;  // emit pass
    size_t smem;
    bool queued;
    int kind;           // SCAN_QUEUED or SCAN_REGISTER (compressed layout)
    bool defer;         // the scan hands whole-slice queues to the resolver kernel
    void *kernel_res;
    // emit pass of a register-staged plan: the queued kernel with tables of
    // its own (one bitmap copy, entries through L2)
    size_t smem_emit;
    uint32_t e_tbl_words, e_tbl_m_words;
    // the window kernel takes the scan (the fields above then describe the
    // plan that its options would otherwise run): words of the prefix bitmap
    // in its shared memory
    bool win;
    uint32_t wf_words, wc_words;
    size_t smem_win;
    void *kernel_win, *kernel_win_small;
    // the dense scan kernel takes it: its tables in shared memory
    bool dsc;
    uint32_t d_rep, d_c_words, d_e_words, d_m_words;
    size_t smem_d;
    void *kernel_d;
};

enum { SCAN_QUEUED = PFAC_KERNEL_QUEUED, SCAN_REGISTER = PFAC_KERNEL_REGISTER, SCAN_SERIAL = PFAC_KERNEL_SERIAL };

struct WsLayout {
    uint64_t hdr, tile_m, tile_k, key_off, chunk, ovf, recs, bounds, defer, dbatch, total;
    uint64_t wbuf, wcnt;
    uint32_t n_tiles, defer_cap, dbatch_cap, wsub_cap, wsubs;
};

// entries per slice the resolver kernel's buffer holds (more go to the
// scan kernel's own resolution)
constexpr uint32_t DEFER_PER_UNIT = 8;
// entries per slice of the window kernel's buffer (8 bytes each)
constexpr uint32_t WBUF_PER_UNIT = 16;
// pairs of slices per SM up to which the window kernel reads its filter
// through L2 (more warps over less text, nothing to fill) and not from shared
// memory.  Scan and resolver, always shared memory / this line / 64 pairs:
// 1 MiB, 256 symbols x 1,000 patterns 18.4 / 15.4 / 15.4 us, 52 letters x 100
// 16.4 / 13.3 / 13.3; 4 MiB (27 pairs) 22.5 / 23.6 / 23.6 and 18.4 / 19.5 /
// 17.4; 8 MiB of packets against 20,000 signatures 39.9 / 40.1 / 50.2.
constexpr uint32_t WIN_SMALL_PAIRS = 16;

static inline uint64_t al256(uint64_t x) { return (x + 255) & ~255ull; }

static WsLayout ws_layout(uint64_t n_bytes, uint32_t n_seg, const Plan &pl) {
    WsLayout L{};
    const bool entries = pl.win || pl.dsc;  // the entry buffer in place of the queues
    const uint64_t ub = 1ull << pl.unit_shift;
    const uint64_t nt = (n_bytes + ub - 1) / ub;
    L.n_tiles = (uint32_t)nt;
    uint64_t o = 0;
    auto put = [&](uint64_t sz) {
        const uint64_t at = o;
        o = al256(o + sz);
        return at;
    };
    L.hdr = put(sizeof(WsHeader));
    // the call's first launch zeroes the header and the counts (the record
    // counts only where they are kept apart from the key counts)
    L.wcnt = put(entries ? (uint64_t)WSUB_MAX * WSUB_STRIDE * 4 : 0);
    L.chunk = put((uint64_t)CHUNKS_MAX * 8);
    L.tile_k = put(nt * 8);
    L.tile_m = put(nt * 4);
    L.key_off = put(nt * 8);
    L.ovf = put(nt * 4);
    L.recs = put(nt * pl.unit_cap * 8);
    // segment data: per-tile lists (tile-synchronous kernel) or the first
    // offset index per unit (queued kernel)
    L.bounds = put(n_seg > 1 ? (pl.queued ? nt * 4 : nt * SEGW * 4) : 0);
    // register-staged plans: the queues handed to the resolver kernel (at
    // most one batch per slice, plus each warp's last)
    const bool defer = pl.defer && !entries;
    const uint64_t dcap = defer ? std::min<uint64_t>(nt * DEFER_PER_UNIT, 0xFFFFFF00ull) : 0;
    L.defer_cap = (uint32_t)dcap;
    L.dbatch_cap = defer ? (uint32_t)std::min<uint64_t>(nt + 4096, 0xFFFFFF00ull) : 0u;
    L.defer = put(dcap * 16);
    L.dbatch = put((uint64_t)L.dbatch_cap * 8);
    // the window and dense kernels' entries, in parts that the warps share out between
    // them: at least 512 entries each (a part's counter runs at most one
    // reservation per warp past them)
    L.wsubs = 1;
    while (L.wsubs < WSUB_MAX && nt * WBUF_PER_UNIT >= 1024ull * L.wsubs) L.wsubs *= 2;
    L.wsub_cap = entries ? (uint32_t)std::min<uint64_t>((nt * WBUF_PER_UNIT + L.wsubs - 1) / L.wsubs,
                                                       0xF0000000ull) : 0u;
    L.wbuf = put((uint64_t)L.wsub_cap * L.wsubs * 8);
    L.total = o;
    return L;
}

static void *scan_kernel_for(uint32_t bps, int var, int emit, int nw, int w) {
    switch (bps) {
        case 1: return scan_kernel_bps1(var, emit, nw, w);
        case 2: return scan_kernel_bps2(var, emit, nw, w);
        case 3: return scan_kernel_bps3(var, emit, nw, w);
        case 4: return scan_kernel_bps4(var, emit, nw, w);
        case 5: return scan_kernel_bps5(var, emit, nw, w);
        case 6: return scan_kernel_bps6(var, emit, nw, w);
        case 7: return scan_kernel_bps7(var, emit, nw, w);
        case 8: return scan_kernel_bps8(var, emit, nw, w);
        default: return nullptr;
    }
}

static size_t dense_smem(uint32_t tbl_words) {
    const size_t tbl = ((size_t)tbl_words * 4 + 127) & ~(size_t)127;
    return tbl + STAGES * STAGE_IN + STAGES * SEGW * 4 + 2 * STAGES * 8 + 2 * STAGES * 4 +
           (CW + 1) * 8;
}

constexpr size_t SMEM_LIMIT = 232448;  // per-CTA dynamic shared memory on sm_103a

static size_t queued_smem(uint64_t words, uint32_t nw = QW) {
    const size_t tbl = ((size_t)words * 4 + 127) & ~(size_t)127;
    return tbl + nw * sizeof(WarpArea);
}

static double load_wavefronts(int rep) { return LOAD_WAVEFRONTS[rep < 0 ? 0 : (rep > 5 ? 5 : rep)]; }

// Estimated warp instructions per 512-byte slice of a first stage that
// passes a share `dens` of the positions (measured orders of magnitude:
// ~9 per tested position row, 2 more for hashing, bank-conflict replays,
// ~90 for a slice with any candidate and ~12 per candidate).
static double first_stage_cost(double dens, int rep, bool hashed) {
    const double cand = dens * 512.0;
    return (hashed ? 176.0 : 144.0) + 48.0 * (load_wavefronts(rep) - 1.0) +
           90.0 * (1.0 - exp(-cand)) + 12.0 * cand;
}

// Estimated SM cycles per slice of the register-staged kernel beyond a fixed
// part: the first stage's shared-memory wavefronts (16 lookups a lane) and
// about 10 cycles per candidate for the second stage (a fit to the alphabet-
// 256 cell with 1,000 patterns: 112 cycles a slice with the gram filter at
// 0.1% candidates and 3.7 wavefronts a lookup, 157 with the prefix bitmap in
// 16 copies at 1.5% and 2 wavefronts), plus a little for the gram hash.
static double r_cost(double dens, int rep, bool hashed) {
    return 16.0 * load_wavefronts(rep) + 10.0 * 512.0 * dens + (hashed ? 4.0 : 0.0);
}

static size_t r_smem(uint64_t words, uint32_t nw = RNW) {
    return (((size_t)words * 4 + 127) & ~(size_t)127) + nw * sizeof(RWarpArea);
}

constexpr int R_MAX_REP = 4;  // copies of the first-stage bitmap: 1 .. 16
constexpr bool R_BY_DEFAULT = true;  // the register-staged kernel by default for 8-bit symbols

// Plan of the register-staged kernel (8-bit symbols): the first stage (the
// prefix bitmap, or the gram filter folded to fit) and its copies, entries
// and child masks in shared memory as they fit, chosen by r_cost; the emit
// pass runs the queued kernel with one bitmap copy.
static int make_plan_r(const pfac_table *t, uint32_t k, int var, uint32_t masks, uint32_t gram,
                       int want, uint32_t nw, Plan *pl) {
    const DevTable &T = t->dev;
    const uint64_t ent = 1ull << (k * T.bps);
    const uint32_t fw = (uint32_t)(ent >= 32 ? ent / 32 : 1);
    const uint32_t cw = (fw + (1u << T.c_shift[k]) - 1) >> T.c_shift[k];
    const uint32_t ew = T.n_e[k];
    const bool have_m = T.M[k] != nullptr;
    const uint32_t mw = T.m_words[k];
    const double dens_f = (double)ew / (double)ent;
    double best = 1e30;
    int b_var = 0, b_rep = -1;
    uint32_t b_fold = 0;
    bool b_gram = false, b_m = false;
    for (int vv = VAR_FE; vv >= VAR_F; vv--) {
        if (var != 0 && var != vv) continue;
        for (int mm = 1; mm >= 0; mm--) {
            const bool mon = mm == 1;
            if (mon && !(have_m && masks != 1)) continue;
            if (!mon && masks == 2) continue;
            const uint64_t base = cw + (vv == VAR_FE ? ew : 0u) + (mon ? mw : 0u);
            // a preference for what keeps the walks short: entries in shared
            // memory, and above all the child masks, which drop most candidates
            const double bias = (vv == VAR_FE ? 1.0 : 1.05) * (mon ? 1.0 : 1.3);
            for (int r = 0; r <= R_MAX_REP; r++) {
                if (want >= 0 && r != want) continue;
                if (gram != 2 && r_smem(base + ((uint64_t)fw << r), nw) <= SMEM_LIMIT) {
                    const double c = r_cost(dens_f, r, false) * bias;
                    if (c < best) {
                        best = c;
                        b_var = vv;
                        b_rep = r;
                        b_gram = false;
                        b_m = mon;
                    }
                }
                if (T.g_len && gram != 1) {
                    const uint32_t hb = T.g_bits;
                    const uint64_t gw0 = (1ull << hb) / 32;
                    for (uint32_t f = 0; hb - f >= GRAM_MIN_BITS; f++) {
                        if (r_smem(base + fw + ((gw0 >> f) << r), nw) > SMEM_LIMIT) continue;
                        const double dens = 1.0 - exp(-(double)T.g_set / (double)(1ull << (hb - f)));
                        const double c = r_cost(dens, r, true) * bias;
                        if ((gram == 2 || dens < 0.5) && c < best) {
                            best = c;
                            b_var = vv;
                            b_rep = r;
                            b_gram = true;
                            b_fold = f;
                            b_m = mon;
                        }
                        break;  // the least folding that fits
                    }
                }
            }
        }
    }
    if (b_rep < 0)
        return set_error(PFAC_EINVAL, "pfac_match: no register-staged plan fits in shared memory "
                         "with depth %u%s", k, want >= 0 ? " and these copies" : "");
    pl->var = b_var;
    pl->k = k;
    pl->tbl_c_words = cw;
    pl->tbl_e_words = b_var == VAR_FE ? ew : 0u;
    pl->tbl_m_words = b_m ? mw : 0u;
    pl->tbl_b_words = 0;
    if (b_gram) {
        pl->rep_log2 = 0;
        pl->tbl_words = fw;
        pl->g_rep = (uint32_t)b_rep;
        pl->g_fold = b_fold;
        pl->tbl_g_words = (uint32_t)((((1ull << T.g_bits) / 32) >> b_fold) << b_rep);
    } else {
        pl->rep_log2 = (uint32_t)b_rep;
        pl->tbl_words = fw << b_rep;
    }
    pl->nw = nw;
    pl->kind = SCAN_REGISTER;
    pl->kernel = scan_kernel_r(T.bps, T.W, b_rep, b_gram, b_var, (int)nw);
    pl->defer = true;
    pl->kernel_res = resolve_kernel((int)T.W);
    pl->smem = r_smem((uint64_t)pl->tbl_words + pl->tbl_c_words + pl->tbl_e_words +
                      pl->tbl_m_words + pl->tbl_g_words, nw);
    // the emit pass: the queued kernel, one bitmap copy, entries through L2,
    // child masks when they fit beside its warps' rings
    pl->e_tbl_words = fw;
    pl->e_tbl_m_words = (have_m && queued_smem((uint64_t)fw + cw + mw, QW) <= SMEM_LIMIT) ? mw : 0u;
    pl->smem_emit = queued_smem((uint64_t)fw + cw + pl->e_tbl_m_words, QW);
    pl->kernel_emit = scan_kernel_for(T.bps, VAR_F, 1, QW, (int)T.W);
    pl->unit_shift = SLICE_SHIFT;
    pl->unit_cap = SCAP;
    pl->queued = true;
    if (!pl->kernel || !pl->kernel_emit || !pl->kernel_res)
        return set_error(PFAC_EINVAL, "pfac_match: no register-staged kernel for this table");
    return PFAC_OK;
}

static int make_scan_plan(const pfac_table *t, const pfac_match_opts *opts, Plan *pl) {
    const DevTable &T = t->dev;
    memset(pl, 0, sizeof(*pl));
    // the dense layout runs the compressed layout's kernels over its
    // transition table (record format 3), or on request the thread-serial
    // kernel (scan_kernel 3)
    if (T.layout == PFAC_LAYOUT_DENSE && opts && opts->scan_kernel == SCAN_SERIAL) {
        pl->kind = SCAN_SERIAL;
        pl->var = VAR_DENSE;
        uint32_t rows = (uint32_t)(TABLE_SMEM_MAX / (4ull * T.sigma));
        if (rows > T.n_nodes) rows = T.n_nodes;
        pl->dense_rows = rows;
        pl->tbl_words = rows * T.sigma;
        pl->kernel = pl->kernel_emit = scan_kernel_dense();
        pl->smem = dense_smem(pl->tbl_words);
        pl->unit_shift = 13;
        pl->unit_cap = REC_CAP;
        pl->queued = false;
        return PFAC_OK;
    }
    const uint32_t k = opts && opts->prefix_depth ? opts->prefix_depth
                                                   : (t->tuned_k ? t->tuned_k : T.kdef);
    if (k < t->kmin || k > t->kmax)
        return set_error(PFAC_EINVAL, "pfac_match: prefix depth %u not held (table holds %u..%u)",
                         k, t->kmin, t->kmax);
    const uint64_t ent = 1ull << (k * T.bps);
    const uint32_t fw = (uint32_t)(ent >= 32 ? ent / 32 : 1);
    const uint32_t cw = (fw + (1u << T.c_shift[k]) - 1) >> T.c_shift[k];
    const uint32_t ew = T.n_e[k];
    int var = opts && opts->variant ? (int)opts->variant
                                    : (t->tuned_variant ? (int)t->tuned_variant : 0);
    // the table's tuned choice applies only when the caller picks neither the
    // variant nor the depth
    const bool use_tuned = !(opts && (opts->variant || opts->prefix_depth));
    const uint32_t nwant = opts && opts->warps_per_cta ? opts->warps_per_cta
                                                      : (use_tuned && t->tuned_nw ? t->tuned_nw : QW);
    if (nwant != QW && nwant != QW_WIDE)
        return set_error(PFAC_EINVAL, "pfac_match: warps_per_cta %u (16 or 24)", nwant);
    const uint32_t masks = opts && opts->child_masks ? opts->child_masks
                                                    : (use_tuned ? t->tuned_masks : 0u);
    if (masks > 2) return set_error(PFAC_EINVAL, "pfac_match: child_masks %u", masks);
    const bool have_m = T.M[k] != nullptr;
    const uint32_t mw = T.m_words[k];  // words of the packed child masks
    if (masks == 2 && !have_m)
        return set_error(PFAC_EINVAL, "pfac_match: depth %u keeps no child masks (too many "
                         "entries for shared memory)", k);
    const uint32_t gram = opts && opts->gram_filter ? opts->gram_filter
                                                   : (use_tuned ? t->tuned_gram : 0u);
    if (gram > 2) return set_error(PFAC_EINVAL, "pfac_match: gram_filter %u", gram);
    if (gram == 2 && !T.g_len)
        return set_error(PFAC_EINVAL, "pfac_match: the table has no gram filter");
    const uint32_t pbytes = opts && opts->prefix_bytes ? opts->prefix_bytes
                                                      : (use_tuned ? t->tuned_bytes : 0u);
    if (pbytes > 2) return set_error(PFAC_EINVAL, "pfac_match: prefix_bytes %u", pbytes);
    if (pbytes == 2 && !T.B[k])
        return set_error(PFAC_EINVAL, "pfac_match: depth %u has no prefix bytes (more than %u "
                         "index bits)", k, BYTES_MAX_BITS);
    if (pbytes == 2 && gram == 2)
        return set_error(PFAC_EINVAL, "pfac_match: prefix bytes and the gram filter exclude "
                         "each other");
    const uint32_t copies = opts && opts->bitmap_copies ? opts->bitmap_copies
                                                       : (use_tuned ? t->tuned_copies : 0u);
    int want = -1;
    if (copies) {
        want = 0;
        while ((1u << want) < copies) want++;
        if ((1u << want) != copies || want > 5)
            return set_error(PFAC_EINVAL, "pfac_match: bitmap_copies %u is not 1, 2, 4, .., 32",
                             copies);
    }
    if (pbytes == 2 && copies > 1)
        return set_error(PFAC_EINVAL, "pfac_match: prefix bytes take one bitmap copy (%u asked)",
                         copies);
    if (var != 0 && var != VAR_F && var != VAR_FE)
        return set_error(PFAC_EINVAL, "pfac_match: unknown variant %d", var);
    // a merged trie (reduction step 2) runs the queued kernel's merged-trie
    // instance: entries through L2, the default CTA width
    if (T.dag && var == VAR_FE)
        return set_error(PFAC_EINVAL, "pfac_match: a merged trie takes variant 1 (entries in L2)");
    if (T.dag && nwant != QW)
        return set_error(PFAC_EINVAL, "pfac_match: a merged trie takes %u warps per CTA", QW);
    if (T.dag) var = VAR_F;

    // ---- records kept per slice: 32, or 512 (one per position, so that no
    // slice is scanned twice) where many matches are likely
    const uint32_t recs = opts && opts->records_per_slice
                              ? opts->records_per_slice
                              : (use_tuned && t->tuned_records
                                     ? t->tuned_records
                                     : (t->match_density * SLICE > 8.0 ? (uint32_t)SLICE : SCAP));
    if (recs != (uint32_t)SCAP && recs != (uint32_t)SLICE)
        return set_error(PFAC_EINVAL, "pfac_match: records_per_slice %u (32 or 512)", recs);
    const uint32_t resolver = opts && opts->resolver
                                  ? opts->resolver
                                  : (use_tuned ? t->tuned_resolver : 0u);
    if (resolver > 2) return set_error(PFAC_EINVAL, "pfac_match: resolver %u", resolver);
    if (resolver == 2 && T.dag)
        return set_error(PFAC_EINVAL, "pfac_match: a merged trie resolves its queues in the scan");
    // by default the resolver kernel takes the queues where at least four
    // windows per slice pass the prefix bitmap (uniform text): with fewer,
    // its launch costs more than the scan saves
    const bool defer = !T.dag && (resolver == 2 ||
                                  (resolver == 0 && (double)ew * SLICE >= 4.0 * (double)ent));

    // ---- the register-staged kernel (8-bit symbols): on request, or by
    // default when the caller asks for nothing only the queued kernel has
    const uint32_t want_kind = opts && opts->scan_kernel ? opts->scan_kernel
                                                         : (use_tuned ? t->tuned_kernel : 0u);
    if (want_kind > 2)
        return set_error(PFAC_EINVAL, "pfac_match: scan_kernel %u (3: dense layout only)", want_kind);
    const bool r_usable = (T.bps == 8 || T.bps == 2) && pbytes != 2 && !T.dag;
    if (want_kind == SCAN_REGISTER && !r_usable)
        return set_error(PFAC_EINVAL, "pfac_match: the register-staged kernel needs 8-bit or 2-bit "
                         "symbols (alphabets of 129 to 256, or of up to 4), no prefix bytes and "
                         "no merged trie");
    if (want_kind == SCAN_REGISTER || (want_kind == 0 && r_usable && T.bps == 8 && R_BY_DEFAULT)) {
        const uint32_t rnw = opts && opts->warps_per_cta
                                 ? opts->warps_per_cta
                                 : (use_tuned && t->tuned_nw ? t->tuned_nw : (uint32_t)RNW);
        const int rc = make_plan_r(t, k, var, masks, gram, want, rnw, pl);
        pl->unit_cap = recs;
        pl->defer = defer;
        if (rc == PFAC_OK || want_kind == SCAN_REGISTER) return rc;
        clear_error();
        memset(pl, 0, sizeof(*pl));
    }

    // ---- prefix bitmap as the first stage: largest replication that fits
    auto best_rep = [&](uint64_t extra) -> int {
        int rep = -1;
        for (int r = 0; r <= 5; r++)
            if (queued_smem(((uint64_t)fw << r) + cw + extra, nwant) <= SMEM_LIMIT) rep = r;
        return rep;
    };
    int var_f = var;
    if (var_f == 0) {
        const int rep_f = best_rep(0), rep_fe = best_rep(ew);
        var_f = (rep_fe >= 0 && rep_fe >= rep_f - 1) ? VAR_FE : VAR_F;
    }
    const uint32_t e_f = var_f == VAR_FE ? ew : 0u;
    // child masks: with them if they fit (or on request), then the most copies
    const bool m_f = have_m && (masks == 2 || (masks == 0 && best_rep(e_f + mw) >= 0));
    int rep_f = best_rep(e_f + (m_f ? mw : 0u));
    if (want >= 0 && want <= rep_f) rep_f = want;
    else if (want >= 0) rep_f = -2;  // the requested copies do not fit
    const double dens_f = (double)ew / (double)ent;

    // ---- gram filter as the first stage: the prefix bitmap once (for the
    // exact test of survivors), the filter folded (adjacent words OR-ed)
    // until the chosen copies fit
    bool use_g = false;
    int var_g = 0, rep_g = -1;
    uint32_t fold_g = 0;
    bool m_g = false;
    double cost_g = 1e30;
    if (T.g_len && gram != 1) {
        const uint32_t hb = T.g_bits;
        const uint64_t gw0 = (1ull << hb) / 32;
        // entries and child masks in shared memory compete with the filter's
        // bits: every allowed combination is costed, keeping them when that
        // costs little
        for (int vv = VAR_FE; vv >= VAR_F; vv--) {
            if (var != 0 && var != vv) continue;
            for (int mm = 1; mm >= 0; mm--) {
                const bool mon = mm == 1;
                if (mon && !(have_m && masks != 1)) continue;
                if (!mon && masks == 2) continue;
                const uint64_t base = fw + cw + (vv == VAR_FE ? ew : 0u) + (mon ? mw : 0u);
                // a small preference for what keeps the walks short
                const double bias = (vv == VAR_FE ? 1.0 : 1.05) * (mon ? 1.0 : 1.1);
                for (int r = 0; r <= 5; r++) {
                    if (want >= 0 && r != want) continue;
                    for (uint32_t f = 0; hb - f >= GRAM_MIN_BITS; f++) {
                        if (queued_smem(base + ((gw0 >> f) << r), nwant) > SMEM_LIMIT) continue;
                        // expected share of positions through the first stage
                        const double dens =
                            1.0 - exp(-(double)T.g_set / (double)(1ull << (hb - f)));
                        const double c = first_stage_cost(dens, r, true) * bias;
                        if ((gram == 2 || dens < 0.5) && c < cost_g) {
                            cost_g = c;
                            rep_g = r;
                            fold_g = f;
                            var_g = vv;
                            m_g = mon;
                        }
                        break;  // the least folding that fits
                    }
                }
            }
        }
        if (rep_g >= 0) {
            const double cost_f =
                rep_f >= 0 ? first_stage_cost(dens_f, rep_f, false) * (m_f ? 1.0 : 1.1) : 1e30;
            use_g = gram == 2 || cost_g < cost_f;
        } else if (gram == 2) {
            return set_error(PFAC_EINVAL, "pfac_match: the gram filter does not fit in shared "
                             "memory with depth %u%s", k, want >= 0 ? " and these copies" : "");
        }
    }
    // ---- prefix bytes as the first stage (one copy): the prefix bitmap once
    // for ranks, then entries and child masks as they fit.  By default for
    // prefix nodes whose bitmap passes at least 1% of the positions (where
    // the cheaper second stage pays), unless the gram filter is chosen.
    bool use_b = false;
    int var_b = 0;
    bool m_b = false;
    if (T.B[k] && pbytes != 1 && gram != 2 && (want <= 0)) {
        const uint64_t bw = ent / 4;
        for (int vv = VAR_FE; vv >= VAR_F && !use_b; vv--) {
            if (var != 0 && var != vv) continue;
            for (int mm = 1; mm >= 0; mm--) {
                const bool mon = mm == 1;
                if (mon && !(have_m && masks != 1)) continue;
                if (!mon && masks == 2) continue;
                if (queued_smem(bw + fw + cw + (vv == VAR_FE ? ew : 0u) + (mon ? mw : 0u),
                                nwant) <= SMEM_LIMIT) {
                    var_b = vv;
                    m_b = mon;
                    use_b = pbytes == 2 || (!use_g && dens_f >= 0.01);
                    break;
                }
            }
        }
        if (pbytes == 2 && !use_b)
            return set_error(PFAC_EINVAL, "pfac_match: prefix bytes of depth %u do not fit in "
                             "shared memory", k);
    }
    if (use_b) {
        use_g = false;
        var = var_b;
        pl->rep_log2 = 0;
        pl->tbl_words = fw;
        pl->tbl_e_words = var == VAR_FE ? ew : 0u;
        pl->tbl_m_words = m_b ? mw : 0u;
        pl->tbl_b_words = (uint32_t)(ent / 4);
    } else if (use_g) {
        var = var_g;
        pl->rep_log2 = 0;
        pl->tbl_words = fw;
        pl->tbl_e_words = var == VAR_FE ? ew : 0u;
        pl->tbl_m_words = m_g ? mw : 0u;
        pl->g_rep = (uint32_t)rep_g;
        pl->g_fold = fold_g;
        pl->tbl_g_words = (uint32_t)((((1ull << T.g_bits) / 32) >> fold_g) << rep_g);
    } else {
        if (rep_f == -2)
            return set_error(PFAC_EINVAL, "pfac_match: %u bitmap copies do not fit", copies);
        if (rep_f < 0)
            return set_error(PFAC_EINVAL, "pfac_match: prefix node of depth %u does not fit in "
                             "shared memory with variant %d%s", k, var_f,
                             m_f ? " and child masks" : "");
        var = var_f;
        pl->rep_log2 = (uint32_t)rep_f;
        pl->tbl_words = (uint32_t)((uint64_t)fw << rep_f);
        pl->tbl_e_words = e_f;
        pl->tbl_m_words = m_f ? mw : 0u;
    }
    pl->var = var;
    pl->k = k;
    pl->tbl_c_words = cw;
    // a wider CTA on request, when the tables leave room for its warps
    const uint64_t tw = (uint64_t)pl->tbl_b_words + pl->tbl_words + pl->tbl_c_words +
                        pl->tbl_e_words + pl->tbl_m_words + pl->tbl_g_words;
    if (queued_smem(tw, nwant) > SMEM_LIMIT)
        return set_error(PFAC_EINVAL, "pfac_match: %u warps do not fit next to the tables", nwant);
    pl->nw = nwant;
    pl->kind = SCAN_QUEUED;
    // the resolver kernel takes the plain tries' queues (the merged trie's
    // walk stays in its own instance)
    pl->defer = defer;
    pl->kernel_res = pl->defer ? resolve_kernel((int)T.W) : nullptr;
    const int kvar = T.dag ? (VAR_F | VAR_MERGED) : var;
    pl->kernel = scan_kernel_for(T.bps, kvar, 0, (int)nwant, (int)T.W);
    pl->kernel_emit = scan_kernel_for(T.bps, kvar, 1, (int)nwant, (int)T.W);
    pl->smem = queued_smem(tw, nwant);
    pl->unit_shift = SLICE_SHIFT;
    pl->unit_cap = recs;
    pl->queued = true;
    if (!pl->kernel || !pl->kernel_emit || (pl->defer && !pl->kernel_res))
        return set_error(PFAC_EINVAL, "pfac_match: no kernel for this table");
    return PFAC_OK;
}

// The dense scan kernel for a plan with a record per position: 2-bit symbols,
// one segment.  The counts and the prefix bitmap go to shared memory, then the
// child masks and the entries where they fit, then copies of the bitmap.
static bool plan_dense(const pfac_table *t, Plan *pl) {
    const DevTable &T = t->dev;
    const uint32_t k = pl->k;
    if (T.bps != 2 || (T.W != 0 && T.W != 1 && T.W != 3)) return false;
    const uint32_t fw = ((1u << (2 * k)) + 31) / 32, cw = (fw + (1u << T.c_shift[k]) - 1) >> T.c_shift[k];
    auto al4 = [](uint32_t x) { return (x + 3) & ~3u; };
    auto size = [&](uint32_t rep, uint32_t m, uint32_t e) {
        return ((size_t)(fw << rep) + al4(cw) + al4(m) + al4(e)) * 4 + DNW * sizeof(DWarpArea);
    };
    if (fw % 4 || size(0, 0, 0) > SMEM_LIMIT) return false;
    const uint32_t m = T.M[k] && size(0, T.m_words[k], 0) <= SMEM_LIMIT ? T.m_words[k] : 0u;
    const uint32_t e = size(0, m, T.n_e[k]) <= SMEM_LIMIT ? T.n_e[k] : 0u;
    uint32_t rep = 0;
    while (rep < 4 && size(rep + 1, m, e) <= SMEM_LIMIT) rep++;
    pl->kernel_d = scan_kernel_d(e != 0);
    pl->kernel_res = dresolve_kernel((int)T.W);
    if (!pl->kernel_d || !pl->kernel_res) return false;
    pl->d_rep = rep;
    pl->d_c_words = cw;
    pl->d_m_words = m;
    pl->d_e_words = e;
    pl->smem_d = size(rep, m, e);
    return true;
}

// The plan of a call: the scan plan its options ask for and, when they leave
// every choice to the library and the table has no tuned one, in place of that
// scan the window kernel over the table's filter, or for one segment of
// 2-bit symbols with many matches the dense scan kernel.
static int make_plan(const pfac_table *t, uint32_t n_seg, const pfac_match_opts *opts, Plan *pl) {
    const int rc = make_scan_plan(t, opts, pl);
    if (rc != PFAC_OK) return rc;
    const DevTable &T = t->dev;
    if (T.dag || pl->kind == SCAN_SERIAL) return PFAC_OK;
    if (opts && (opts->variant || opts->prefix_depth || opts->ctas_per_sm || opts->bitmap_copies ||
                 opts->child_masks || opts->gram_filter || opts->prefix_bytes ||
                 opts->warps_per_cta || opts->scan_kernel || opts->test_wait_limit_us ||
                 opts->test_withhold_slice || opts->records_per_slice || opts->resolver))
        return PFAC_OK;
    if (t->tuned_variant || t->tuned_k || t->tuned_nw || t->tuned_kernel) return PFAC_OK;
    if (pl->unit_cap == (uint32_t)SLICE) {
        void *res = pl->kernel_res;
        pl->dsc = n_seg <= 1 && plan_dense(t, pl);
        if (!pl->dsc) pl->kernel_res = res;
        return PFAC_OK;
    }
    if (!T.H || pl->unit_cap != (uint32_t)SCAP) return PFAC_OK;
    // shared memory: the filter's copies, the warps' queues, and the prefix
    // bitmap the candidates are tested against, where it fits beside them
    // (else they are tested through L2: a shallower bitmap that fits lets too
    // many of them through, which cost more in the resolver)
    const size_t fixed = ((size_t)T.w_words << T.w_rep) * 4 + WNW * WQCAP * 4;
    if (fixed > SMEM_LIMIT) return PFAC_OK;
    const uint64_t fw = ((1ull << (pl->k * T.bps)) + 31) / 32;
    const uint64_t cw = (fw + (1ull << T.c_shift[pl->k]) - 1) >> T.c_shift[pl->k];
    if (fw % 4 == 0 && cw % 4 == 0 && fixed + (fw + cw) * 4 <= SMEM_LIMIT) {
        pl->wf_words = (uint32_t)fw;
        pl->wc_words = (uint32_t)cw;
    }
    pl->smem_win = fixed + ((size_t)pl->wf_words + pl->wc_words) * 4;
    pl->kernel_win = scan_kernel_w(T, T.w_rep ? WT_COPIES : WT_ONE);
    pl->kernel_win_small = scan_kernel_w(T, WT_L2);
    pl->kernel_res = wresolve_kernel((int)T.W);
    if (!pl->kernel_win || !pl->kernel_win_small || !pl->kernel_res) {
        pl->kernel_res = pl->defer ? resolve_kernel((int)T.W) : nullptr;
        return PFAC_OK;
    }
    pl->win = true;
    return PFAC_OK;
}

static std::mutex g_attr_mu;

static int prepare_kernel(void *fn, size_t smem) {
    // raise the dynamic shared-memory limit once per kernel, device and size
    static void *done_fn[128];
    static int done_dev[128];
    static size_t done_sz[128];
    static int n_done = 0;
    int dev = 0;
    cudaGetDevice(&dev);
    std::lock_guard<std::mutex> lk(g_attr_mu);
    for (int i = 0; i < n_done; i++)
        if (done_fn[i] == fn && done_dev[i] == dev && done_sz[i] >= smem) return PFAC_OK;
    cudaError_t e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess)
        return set_error(PFAC_ECUDA, "pfac_match: smem attribute: %s", cudaGetErrorString(e));
    if (n_done < 128) {
        done_fn[n_done] = fn;
        done_dev[n_done] = dev;
        done_sz[n_done] = smem;
        n_done++;
    }
    return PFAC_OK;
}

int check_table_device(const pfac_table *t, void *cuda_stream, const char *who) {
    int cur = 0;
    cudaError_t e = cudaGetDevice(&cur);
    if (e != cudaSuccess)
        return set_error(PFAC_ECUDA, "%s: cudaGetDevice: %s", who, cudaGetErrorString(e));
    if (cur != t->device)
        return set_error(PFAC_EINVAL, "%s: the current device is %d but the table lives on "
                         "device %d; make device %d current", who, cur, t->device, t->device);
    cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
    if (cuda_stream && cudaStreamIsCapturing((cudaStream_t)cuda_stream, &cap) != cudaSuccess) {
        cudaGetLastError();
        cap = cudaStreamCaptureStatusNone;
    }
    // the stream's device cannot be queried while the stream captures a graph
    // (the query is not permitted then); the current-device check stands
    if (cuda_stream && cap == cudaStreamCaptureStatusNone) {
        int sd = 0;
        e = cudaStreamGetDevice((cudaStream_t)cuda_stream, &sd);
        if (e != cudaSuccess)
            return set_error(PFAC_ECUDA, "%s: cudaStreamGetDevice: %s", who,
                             cudaGetErrorString(e));
        if (sd != t->device)
            return set_error(PFAC_EINVAL, "%s: the stream belongs to device %d but the table "
                             "lives on device %d", who, sd, t->device);
    }
    return PFAC_OK;
}

// Launches a kernel that may start while the one before it still runs
// (dep_wait in kernels.cuh); with dep == false an ordinary launch.
static cudaError_t launch(const void *fn, uint32_t grid, uint32_t block, void **args, size_t smem,
                          cudaStream_t st, bool dep) {
    cudaLaunchConfig_t c;
    memset(&c, 0, sizeof c);
    c.gridDim = dim3(grid);
    c.blockDim = dim3(block);
    c.dynamicSmemBytes = smem;
    c.stream = st;
    cudaLaunchAttribute a;
    memset(&a, 0, sizeof a);
    a.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    a.val.programmaticStreamSerializationAllowed = 1;
    c.attrs = &a;
    c.numAttrs = dep ? 1 : 0;
    return cudaLaunchKernelExC(&c, fn, args);
}

static int sm_count() {
    int dev = 0, n = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev);
    return n > 0 ? n : 1;
}

}  // namespace pfac

using namespace pfac;

extern "C" int pfac_workspace_bytes(const pfac_table *t, uint64_t n_bytes, uint32_t n_segments,
                                    const pfac_match_opts *opts, uint64_t *bytes) {
    if (!t || !bytes) return set_error(PFAC_EINVAL, "pfac_workspace_bytes: NULL argument");
    if (n_bytes >> (64 - PFAC_ID_BITS))
        return set_error(PFAC_EINVAL, "pfac_workspace_bytes: input longer than 2^%d bytes",
                         64 - PFAC_ID_BITS);
    Plan pl;
    const int rc = make_plan(t, n_segments, opts, &pl);
    if (rc) return rc;
    // enough too for the same call with options that choose its scan (the plan
    // without the window or dense kernel), and for fewer segments (a chunk of
    // a longer text), where another kernel may take it
    auto total = [&](uint32_t n_seg, Plan &p) {
        uint64_t b = ws_layout(n_bytes, n_seg, p).total;
        if (p.win || p.dsc) {
            p.win = p.dsc = false;
            b = std::max(b, ws_layout(n_bytes, n_seg, p).total);
        }
        return b;
    };
    const bool full = pl.unit_cap == (uint32_t)SLICE;
    *bytes = total(n_segments, pl);
    Plan one;
    if (full && n_segments > 1 && make_plan(t, 1, opts, &one) == PFAC_OK)
        *bytes = std::max(*bytes, total(1, one));
    return PFAC_OK;
}

extern "C" int pfac_match_plan(const pfac_table *t, const pfac_match_opts *opts,
                               pfac_plan_info *out) {
    clear_error();
    if (!t || !out) return set_error(PFAC_EINVAL, "pfac_match_plan: NULL argument");
    Plan pl;
    const int rc = make_plan(t, 1, opts, &pl);
    if (rc) return rc;
    memset(out, 0, sizeof *out);
    out->smem_bytes = (uint32_t)pl.smem;
    if (!pl.queued) return PFAC_OK;
    out->variant = (uint32_t)pl.var;
    out->prefix_depth = pl.k;
    const bool g = pl.tbl_g_words != 0;
    out->bitmap_copies = 1u << (g ? pl.g_rep : pl.rep_log2);
    out->child_masks = pl.tbl_m_words ? 2u : 1u;
    out->gram_filter = g ? 2u : 1u;
    out->gram_bits = g ? t->dev.g_bits - pl.g_fold : 0u;
    out->prefix_bytes = pl.tbl_b_words ? 2u : 1u;
    out->warps_per_cta = pl.nw;
    out->scan_kernel = (uint32_t)pl.kind;
    out->records_per_slice = pl.unit_cap;
    out->resolver = pl.kind == SCAN_SERIAL ? 0u : (pl.defer ? 2u : 1u);
    return PFAC_OK;
}

extern "C" int pfac_match_kernel(const pfac_table *t, uint32_t n_segments,
                                 const pfac_match_opts *opts, uint32_t *kernel) {
    clear_error();
    if (!t || !kernel) return set_error(PFAC_EINVAL, "pfac_match_kernel: NULL argument");
    Plan pl;
    const int rc = make_plan(t, n_segments, opts, &pl);
    if (rc) return rc;
    *kernel = pl.win ? PFAC_KERNEL_WINDOW : pl.dsc ? PFAC_KERNEL_DENSE : (uint32_t)pl.kind;
    return PFAC_OK;
}

extern "C" int pfac_match_async(const pfac_table *t, const uint8_t *d_input, uint64_t n_bytes,
                                const uint64_t *d_seg_offsets, uint32_t n_segments,
                                uint64_t *d_out_keys, uint64_t out_capacity, uint64_t *d_count,
                                int32_t *d_status, void *d_workspace, uint64_t workspace_bytes,
                                const pfac_match_opts *opts, void *cuda_stream) {
    if (!t || !d_count || !d_seg_offsets || !d_workspace)
        return set_error(PFAC_EINVAL, "pfac_match: NULL argument");
    if (!t->d_blob) return set_error(PFAC_EINVAL, "pfac_match: table was built host-only");
    {
        const int drc = check_table_device(t, cuda_stream, "pfac_match");
        if (drc) return drc;
    }
    if (n_bytes && !d_input) return set_error(PFAC_EINVAL, "pfac_match: NULL input");
    if (((uintptr_t)d_input & 15) != 0)
        return set_error(PFAC_EINVAL, "pfac_match: input must be 16-byte aligned");
    if (((uintptr_t)d_workspace & 255) != 0)
        return set_error(PFAC_EINVAL, "pfac_match: workspace must be 256-byte aligned");
    if (n_bytes >> (64 - PFAC_ID_BITS))
        return set_error(PFAC_EINVAL, "pfac_match: input longer than 2^%d bytes", 64 - PFAC_ID_BITS);
    if (n_bytes && n_segments == 0)
        return set_error(PFAC_EINVAL, "pfac_match: a non-empty input needs a segment");
    if (out_capacity && !d_out_keys) return set_error(PFAC_EINVAL, "pfac_match: NULL output");
    const uint64_t starts_end = opts && opts->starts_end ? opts->starts_end : n_bytes;
    const uint64_t pos_base = opts ? opts->position_base : 0;
    if (starts_end > n_bytes)
        return set_error(PFAC_EINVAL, "pfac_match: starts_end %llu beyond the input",
                         (unsigned long long)starts_end);
    if ((pos_base + n_bytes) >> (64 - PFAC_ID_BITS) || pos_base + n_bytes < pos_base)
        return set_error(PFAC_EINVAL, "pfac_match: position_base + n_bytes reaches 2^%d",
                         64 - PFAC_ID_BITS);
    Plan pl;
    int rc = make_plan(t, n_segments, opts, &pl);
    if (rc) return rc;
    const WsLayout L = ws_layout(n_bytes, n_segments, pl);
    if (workspace_bytes < L.total)
        return set_error(PFAC_EINVAL, "pfac_match: workspace of %llu bytes, %llu needed",
                         (unsigned long long)workspace_bytes, (unsigned long long)L.total);
    const bool reg = pl.kind == SCAN_REGISTER;
    const size_t smem_emit = reg ? pl.smem_emit : pl.smem;
    rc = pl.win   ? prepare_kernel(pl.kernel_win, pl.smem_win)
         : pl.dsc ? prepare_kernel(pl.kernel_d, pl.smem_d)
                  : prepare_kernel(pl.kernel, pl.smem);
    if (!rc && !pl.win && !pl.dsc && pl.kernel_emit != pl.kernel) rc = prepare_kernel(pl.kernel_emit, smem_emit);
    if (rc) return rc;

    cudaStream_t st = (cudaStream_t)cuda_stream;
    uint8_t *W = (uint8_t *)d_workspace;
    MatchParams P;
    memset(&P, 0, sizeof(P));
    P.T = t->dev;
    P.in = d_input;
    P.n = n_bytes;
    P.seg = d_seg_offsets;
    P.n_seg = n_segments;
    // units holding a start position (the rest of the input is halo)
    const uint64_t ub = 1ull << pl.unit_shift;
    P.n_tiles = (uint32_t)((starts_end + ub - 1) >> pl.unit_shift);
    P.starts_end = starts_end;
    P.pos_base = pos_base;
    P.out = d_out_keys;
    P.cap = out_capacity;
    P.d_count = d_count;
    P.d_status = d_status;
    P.hdr = (WsHeader *)(W + L.hdr);
    P.tile_m = (uint32_t *)(W + L.tile_m);
    P.tile_k = (uint64_t *)(W + L.tile_k);
    P.key_off = (uint64_t *)(W + L.key_off);
    P.chunk = (uint64_t *)(W + L.chunk);
    P.chunk_shift = chunk_shift(P.n_tiles);
    const uint32_t n_chunks = (uint32_t)(((uint64_t)P.n_tiles + (1ull << P.chunk_shift) - 1) >> P.chunk_shift);
    P.ovf_list = (uint32_t *)(W + L.ovf);
    P.recs = (uint64_t *)(W + L.recs);
    P.tile_bounds = (uint32_t *)(W + L.bounds);
    P.unit_seg = (uint32_t *)(W + L.bounds);
    P.unit_shift = pl.unit_shift;
    P.unit_cap = pl.unit_cap;
    P.k = pl.k;
    P.F = pl.k ? t->dev.F[pl.k] : nullptr;
    P.C = pl.k ? t->dev.C[pl.k] : nullptr;
    P.E = pl.k ? t->dev.E[pl.k] : nullptr;
    P.M = pl.k ? t->dev.M[pl.k] : nullptr;
    P.c_shift = pl.k ? t->dev.c_shift[pl.k] : 0u;
    P.tbl_m_words = pl.tbl_m_words;
    P.tbl_g_words = pl.tbl_g_words;
    P.g_rep = pl.g_rep;
    P.g_fold = pl.g_fold;
    P.g_hb = pl.tbl_g_words ? t->dev.g_bits - pl.g_fold : 0u;
    P.kf = pl.tbl_g_words ? t->dev.g_len : pl.k;
    P.Bt = pl.k ? t->dev.B[pl.k] : nullptr;
    P.tbl_b_words = pl.tbl_b_words;
    P.tbl_words = pl.tbl_words;
    P.tbl_c_words = pl.tbl_c_words;
    P.tbl_e_words = pl.tbl_e_words;
    P.rep_log2 = pl.rep_log2;
    P.dense_rows = pl.dense_rows;
    P.wait_limit_ns = opts && opts->test_wait_limit_us ? (uint64_t)opts->test_wait_limit_us * 1000
                                                       : WAIT_LIMIT_NS;
    P.withhold_unit = opts && opts->test_withhold_slice ? opts->test_withhold_slice - 1 : UNIT_NONE;
    if (pl.win || pl.dsc) {
        // the window kernel's re-walks of full slices are the expansion's (the
        // dense kernel has a record for every position)
        P.no_emit = 1;
        P.wbuf = (uint64_t *)(W + L.wbuf);
        P.wcnt = (uint32_t *)(W + L.wcnt);
        P.wsub_cap = L.wsub_cap;
        P.wsub_mask = L.wsubs - 1;
    }
    if (pl.win) {
        const DevTable &T = t->dev;
        const uint32_t bits = T.w_packed ? 2 * T.w_gw : 8 * T.w_gw;
        P.w_words = T.w_words;
        P.w_rep = T.w_rep;
        P.w_gm = gram_mul(bits);
        P.w_glen = T.w_glen;
        P.w_badmask = T.w_short ? 0x01010101u * ((0xFFu << T.bps) & 0xFFu) : 0u;
        P.wf_words = pl.wf_words;
        P.wc_words = pl.wc_words;
        P.unordered = 1;
        P.chunk_adds = P.chunk_shift <= CHUNK_SHIFT_ADDS;
    } else if (pl.defer && !pl.dsc) {
        P.defer = (uint4 *)(W + L.defer);
        P.defer_cap = L.defer_cap;
        P.dbatch = (uint2 *)(W + L.dbatch);
        P.dbatch_cap = L.dbatch_cap;
    }
    const uint32_t nthreads = pl.queued ? pl.nw * 32 : NTHREADS;
    // units a CTA takes in one round: the register-staged kernel's warps
    // take two slices each
    const uint32_t units_per_cta = pl.queued ? (reg ? 2 * pl.nw : pl.nw) : 1;

    // header, and for the slice kernels the per-unit record and key counts
    // (the scan pass writes them only for units with kept survivors)
    const bool ent = pl.win || pl.dsc;
    const uint64_t zero = pl.win ? L.tile_m : (pl.queued ? L.key_off : sizeof(WsHeader));
    const int nsm = sm_count();
    cudaError_t e;
    if (ent) {
        uint4 *zp = (uint4 *)P.hdr;
        uint64_t zn = zero / 16;
        void *args[] = {&P, &zp, &zn};
        // four words a thread, and one slice or offset
        const uint64_t idx = n_segments > 1 ? std::max<uint64_t>(P.n_tiles, n_segments) : 0;
        const uint64_t zb = std::max<uint64_t>((zn + 1023) / 1024, (idx + 255) / 256);
        e = launch((const void *)k_zero, (uint32_t)std::min<uint64_t>(zb ? zb : 1, (uint64_t)nsm * 8), 256, args,
                   0, st, false);
    } else {
        e = cudaMemsetAsync(P.hdr, 0, zero, st);
    }
    const uint32_t cps = opts && opts->ctas_per_sm ? opts->ctas_per_sm : 1;
    if (e == cudaSuccess && n_segments > 1 && P.n_tiles && !pl.win) {
        if (pl.queued) k_unitseg<<<nsm * 4, 256, 0, st>>>(P);
        else k_bounds<<<nsm * 2, 256, 0, st>>>(P);
        e = cudaGetLastError();
    }
    // persistent grid: one CTA per SM (fewer when there are few units)
    const uint64_t want = ((uint64_t)P.n_tiles + units_per_cta - 1) / units_per_cta;
    const uint32_t grid = (uint64_t)nsm * cps < want ? (uint32_t)nsm * cps : (uint32_t)want;
    if (e == cudaSuccess && opts && opts->ev_scan_begin)
        e = cudaEventRecord((cudaEvent_t)opts->ev_scan_begin, st);
    if (e == cudaSuccess && P.n_tiles && pl.win) {
        // few pairs of slices: one warp each, the filter read through L2
        const uint32_t n_pairs = (P.n_tiles + 1) / 2;
        const bool small = n_pairs <= (uint32_t)nsm * WIN_SMALL_PAIRS;
        P.w_ranked = !small && P.wf_words != 0;
        const uint32_t nw = small ? WNW_SMALL : WNW;
        const uint32_t need = (n_pairs + nw - 1) / nw;
        void *args[] = {&P};
        e = launch(small ? pl.kernel_win_small : pl.kernel_win,
                   small || need < (uint32_t)nsm ? need : (uint32_t)nsm, nw * 32, args,
                   small ? (size_t)WNW_SMALL * WQCAP * 4 : pl.smem_win, st, true);
    } else if (e == cudaSuccess && P.n_tiles && pl.dsc) {
        MatchParams PD = P;
        PD.rep_log2 = pl.d_rep;
        PD.tbl_words = (((1u << (2 * pl.k)) + 31) / 32) << pl.d_rep;
        PD.tbl_c_words = pl.d_c_words;
        PD.tbl_m_words = pl.d_m_words;
        PD.tbl_e_words = pl.d_e_words;
        const uint32_t need = ((P.n_tiles + 1) / 2 + DNW - 1) / DNW;
        void *args[] = {&PD};
        e = launch(pl.kernel_d, need < (uint32_t)nsm ? need : (uint32_t)nsm, DNW * 32, args, pl.smem_d, st, true);
    } else if (e == cudaSuccess && P.n_tiles) {
        int emit = 0;
        void *args[] = {&P, &emit};
        e = cudaLaunchKernel(pl.kernel, dim3(grid), dim3(nthreads), args, pl.smem, st);
    }
    if (e == cudaSuccess && P.n_tiles && (pl.win || pl.dsc || pl.defer)) {
        // the handed-over queues (or the window or dense kernel's entries): prefix bitmap, counts and entries through
        // L2 (one bitmap copy)
        MatchParams P3 = P;
        P3.rep_log2 = 0;
        P3.tbl_e_words = 0;
        P3.tbl_m_words = 0;
        void *args[] = {&P3};
        // (small calls: no more warps than their entry buffer has blocks)
        const uint32_t full = (uint32_t)nsm * RES_CTAS;
        const uint64_t blocks = ((uint64_t)P.n_tiles * WBUF_PER_UNIT + 255) / 256;
        e = launch(pl.kernel_res, ent && blocks < full ? (uint32_t)blocks : full, RES_WARPS * 32, args, 0, st, ent);
    }
    if (e == cudaSuccess && opts && opts->ev_scan_end)
        e = cudaEventRecord((cudaEvent_t)opts->ev_scan_end, st);
    if (e == cudaSuccess && P.n_tiles && !P.chunk_adds) {
        void *args[] = {&P};
        e = launch((const void *)k_reduce, n_chunks, 256, args, 0, st, true);
    }
    if (e == cudaSuccess) {
        // a chunk's units over its CTA's eight warps, 32 at most at a time
        const uint32_t span = P.chunk_shift < 8 ? (1u << P.chunk_shift) / 8 : 32u;
        void *args[] = {&P, (void *)&span};
        e = launch((const void *)k_expand, n_chunks ? n_chunks : 1, 256, args, 0, st, true);
    }
    if (e == cudaSuccess && opts && opts->ev_emit_begin)
        e = cudaEventRecord((cudaEvent_t)opts->ev_emit_begin, st);
    if (e == cudaSuccess && P.n_tiles && !P.no_emit) {
        int emit = 1;
        if (reg) {
            // the queued kernel re-scans the overflowing slices with its own
            // tables: one prefix-bitmap copy, entries through L2
            MatchParams P2 = P;
            P2.tbl_words = pl.e_tbl_words;
            P2.rep_log2 = 0;
            P2.tbl_e_words = 0;
            P2.tbl_m_words = pl.e_tbl_m_words;
            P2.tbl_g_words = 0;
            P2.g_rep = P2.g_fold = P2.g_hb = 0;
            P2.tbl_b_words = 0;
            P2.kf = pl.k;
            const uint64_t want_e = ((uint64_t)P.n_tiles + QW - 1) / QW;
            const uint32_t grid_e =
                (uint64_t)nsm * cps < want_e ? (uint32_t)nsm * cps : (uint32_t)want_e;
            void *args[] = {&P2, &emit};
            e = launch(pl.kernel_emit, grid_e, QW * 32, args, smem_emit, st, true);
        } else {
            void *args[] = {&P, &emit};
            e = launch(pl.kernel_emit, grid, nthreads, args, pl.smem, st, pl.queued);
        }
    }
    if (e == cudaSuccess && opts && opts->ev_emit_end)
        e = cudaEventRecord((cudaEvent_t)opts->ev_emit_end, st);
    if (e != cudaSuccess)
        return set_error(PFAC_ECUDA, "pfac_match: launch failed: %s", cudaGetErrorString(e));
    return PFAC_OK;
}

extern "C" int pfac_match(const pfac_table *t, const uint8_t *d_input, uint64_t n_bytes,
                          const uint64_t *d_seg_offsets, uint32_t n_segments, uint64_t *d_out_keys,
                          uint64_t out_capacity, uint64_t *n_out, const pfac_match_opts *opts,
                          void *cuda_stream) {
    clear_error();
    if (!t || !n_out) return set_error(PFAC_EINVAL, "pfac_match: NULL argument");
    if (!t->d_blob) return set_error(PFAC_EINVAL, "pfac_match: table was built host-only");
    int drc = check_table_device(t, cuda_stream, "pfac_match");
    if (drc) return drc;
    cudaStream_t st = (cudaStream_t)cuda_stream;
    uint64_t ws_bytes = 0;
    int rc0 = pfac_workspace_bytes(t, n_bytes, n_segments, opts, &ws_bytes);
    if (rc0) return rc0;
    // the workspace, then the count and the status, read back in one copy
    void *ws = nullptr;
    cudaError_t e = scratch_alloc(&ws, ws_bytes + 256, st);
    if (e != cudaSuccess) {
        cudaGetLastError();
        return set_error(e == cudaErrorMemoryAllocation ? PFAC_ENOMEM : PFAC_ECUDA,
                         "pfac_match: workspace allocation: %s", cudaGetErrorString(e));
    }
    uint64_t *d_cnt = (uint64_t *)((uint8_t *)ws + ws_bytes);
    int32_t *d_st = (int32_t *)(d_cnt + 1);
    int rc = pfac_match_async(t, d_input, n_bytes, d_seg_offsets, n_segments, d_out_keys,
                              out_capacity, d_cnt, d_st, ws, ws_bytes, opts, cuda_stream);
    struct {
        uint64_t cnt;
        int32_t st;
        int32_t pad;
    } h{0, 0, 0};
    if (rc == PFAC_OK) {
        e = cudaMemcpyAsync(&h, d_cnt, sizeof h, cudaMemcpyDeviceToHost, st);
        if (e == cudaSuccess) e = cudaStreamSynchronize(st);
        if (e != cudaSuccess) rc = set_error(PFAC_ECUDA, "pfac_match: %s", cudaGetErrorString(e));
    }
    cudaFreeAsync(ws, st);
    if (rc) return rc;
    *n_out = h.cnt;
    if (h.st != PFAC_OK)
        return set_error(h.st, "pfac_match: device reported %s", pfac_status_str(h.st));
    if (h.cnt > out_capacity)
        return set_error(PFAC_ENOSPC, "pfac_match: %llu matches, capacity %llu",
                         (unsigned long long)h.cnt, (unsigned long long)out_capacity);
    return PFAC_OK;
}
