// Window kernel: the scan pass of the compressed and dense layouts' plain
// tries as one streaming filter over the text, its survivors resolved by a
// second launch (Section 2.3's walks, started only where they can report
// something).
//
// * Filter.  The table holds a window filter H (table.h): a bitmap of 32-bit
//   words over strings of g symbols, filled with every string that can stand
//   at offset 0 .. S-1 of an occurrence of some pattern.  With stride S only
//   every S-th position q is looked up: a start p in [q - S + 1, q] whose
//   pattern has at least g + S - 1 symbols shows one of its g-strings at q,
//   and shorter patterns have every completion of theirs in H.  A lookup
//   reads one word (hash of the window) and tests NB of its bits, each chosen
//   by other symbols of the window.  Segment ends need no attention here: H
//   has no false negatives whatever follows an occurrence.
// * Work split.  A warp takes chunks of 1,024 bytes (two slices of the other
//   scan kernels) round-robin; a lane holds 32 bytes in registers, one load
//   issued a step ahead (and an L2 prefetch WPF steps ahead), and the symbols
//   after them by a shuffle.
// * Candidates (window positions) go to a queue of 128 words per warp.  A
//   full queue is flushed by all lanes: the prefix index of each start is
//   packed from the text (still in L2), tested against a prefix bitmap in
//   shared memory (or through L2) and the passing starts are appended to the
//   call's entry buffer with one atomic.  When the buffer is full the lanes
//   walk their starts from the root instead.
// * k_wresolve then takes the entries in any order: segment limit, exact
//   prefix bit, the batched walks of the queued kernel's resolver, and one
//   record per match at an atomically taken slot of its slice; the key
//   expansion sorts the few records of a slice.
//
// What bounds it: shared-memory lookups (3.7 wavefronts of random banks per
// warp-wide lookup with one copy of H: 59 cycles of an SM's shared memory per
// slice at stride 1) and the ALU instructions around them; S, the bits tested
// and the copies of H are chosen per table to balance both (window.cpp).
// Measured scan pass, before (queued or register-staged kernel) and with this
// one: 20 symbols x 10,000 patterns, 256 MiB: 858 -> 184 us; 64 x 100,000,
// 128 MiB: 569 -> 118 us; 256 x 1,000, 512 MiB: 293 -> 200 us; 52 letters x
// 100, 100 MiB: 111 -> 32 us; 1 GiB of packets against 20,000 signatures:
// 2,773 -> 878 us; DNA x 10,000, 256 MiB: 281 -> 182 us.  The resolver after
// it takes the place of the other kernels' resolver (packets: 374 -> 363 us).
#pragma once
#include "kernels_r.cuh"

namespace pfac {

constexpr int WNW = 24;            // warps per CTA (80 registers a thread, no spills in the loop)
constexpr uint32_t WPF = 4;        // steps ahead of the L2 prefetch
constexpr int WNW_SMALL = 4;   // warps per CTA when the filter is read through L2
constexpr uint32_t WQCAP = 128;          // candidate queue per warp
constexpr uint32_t WX_ROOT = 0xFFFFFFu;  // entry: walk from the root

// How a lookup reaches H: through L2, or from shared memory with one copy or
// with several interleaved word by word.
enum { WT_L2 = 0, WT_ONE = 1, WT_COPIES = 2 };

// 32 bytes of the text in eight registers; the input is 16-byte aligned, and
// one load takes them where it is 32-byte aligned.
struct WChunk {
    uint32_t w[8];
};

__device__ __forceinline__ void w_load32(const uint8_t *p, bool al32, WChunk &c) {
    if (al32) {
        asm volatile(
            "ld.global.nc.L1::no_allocate.v8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
            : "=r"(c.w[0]), "=r"(c.w[1]), "=r"(c.w[2]), "=r"(c.w[3]), "=r"(c.w[4]), "=r"(c.w[5]),
              "=r"(c.w[6]), "=r"(c.w[7])
            : "l"(p));
    } else {
        // two halves of a sector pair: the first load leaves the second's
        // sectors in L1
        const uint4 a = __ldg(reinterpret_cast<const uint4 *>(p));
        const uint4 b = __ldg(reinterpret_cast<const uint4 *>(p + 16));
        c.w[0] = a.x; c.w[1] = a.y; c.w[2] = a.z; c.w[3] = a.w;
        c.w[4] = b.x; c.w[5] = b.y; c.w[6] = b.z; c.w[7] = b.w;
    }
}

// Window starting j symbols after the lane's first (its low bits): raw bytes
// (j <= 34), or 2-bit symbols packed 16 to a word (j <= 37).
template <int PACKED>
__device__ __forceinline__ uint32_t w_twin(const uint32_t (&w)[9], int j) {
    const int per = PACKED ? 16 : 4, bits = PACKED ? 2 : 8, last = PACKED ? 2 : 8;
    const int i = j / per, sh = bits * (j % per);
    if (sh == 0) return w[i];
    return i >= last ? w[i] >> sh : __funnelshift_r(w[i], w[i + 1 <= 8 ? i + 1 : 8], sh);
}

struct WConst {
    uint32_t gm, hm, amask, c4;
    const uint32_t *tbl;  // H in global memory
};

// Bit 0 of the result: whether the window at symbol j of the lane passes.
template <int PACKED, int NB, int G5, int TB>
__device__ __forceinline__ uint32_t w_lookup(const uint32_t (&w)[9], int j, const WConst &K) {
    extern __shared__ __align__(128) uint8_t smem[];
    const uint32_t t = w_twin<PACKED>(w, j);
    uint32_t y = t * K.gm;
    if (G5) y += w_twin<PACKED>(w, j + 1) * WIN_MUL2;
    const uint32_t h = __umulhi(y, K.hm);
    uint32_t x;
    if (TB == WT_L2) x = __ldg(K.tbl + h);
    else if (TB == WT_ONE) x = reinterpret_cast<const uint32_t *>(smem)[h];
    else x = *reinterpret_cast<const uint32_t *>(smem + ((h & K.amask) | K.c4));
    uint32_t r = __funnelshift_r(x, x, w_twin<PACKED>(w, j + (PACKED ? 0 : 2)));
    if (NB >= 2) r &= __funnelshift_r(x, x, w_twin<PACKED>(w, j + (PACKED ? 3 : 0)));
    if (NB >= 3) r &= __funnelshift_r(x, x, w_twin<PACKED>(w, j + (PACKED ? 6 : 1)));
    return r;
}

// All windows of the lane's 32 positions: bit i is set when the one at
// symbol i * S + S - 1 passes.
template <int PACKED, int S, int NB, int G5, int TB>
__device__ __forceinline__ uint32_t w_filter(const uint32_t (&w)[9], const WConst &K) {
    constexpr int NWIN = 32 / S;
    if constexpr (NWIN >= 8) {
        // each test's bit is shifted in at the top of a word: chains of eight
        uint32_t acc[NWIN / 8];
#pragma unroll
        for (int c = 0; c < NWIN / 8; c++) acc[c] = 0;
#pragma unroll
        for (int i = 0; i < 8; i++)
#pragma unroll
            for (int c = 0; c < NWIN / 8; c++)
                acc[c] = __funnelshift_r(
                    acc[c], w_lookup<PACKED, NB, G5, TB>(w, (8 * c + i) * S + S - 1, K), 1);
        // bits 24..31 of each chain
        if (NWIN == 8) return acc[0] >> 24;
        if constexpr (NWIN == 16) return __byte_perm(acc[0], acc[1], 0x0073) & 0xFFFFu;
        if constexpr (NWIN == 32)
            return __byte_perm(__byte_perm(acc[0], acc[1], 0x0073),
                               __byte_perm(acc[2], acc[3], 0x0073), 0x5410);
    } else {
        uint32_t m = 0;
#pragma unroll
        for (int i = 0; i < NWIN; i++)
            m |= (w_lookup<PACKED, NB, G5, TB>(w, i * S + S - 1, K) & 1u) << i;
        return m;
    }
}

// One match: a record in the slice's space while it has room (in any order),
// and the slice's counts: records above bit UNIT_KEY_BITS of its word, keys
// below, so that one atomic takes the slot and counts the keys.  The first
// match past the space lists the slice for the emit pass.  With few slices
// the chunks' key counts are added up here too; with many, neighbouring
// matches would queue on one chunk's word (1 GiB of packets: 0.8 instead of
// 0.36 ms), and k_reduce sums them.
__device__ __forceinline__ void w_emit(const MatchParams &P, uint32_t u, uint32_t pos, uint32_t fin) {
    u = (uint32_t)chk(P, u, P.n_tiles);
    const uint32_t cap = P.unit_cap;
    const unsigned long long keys = fin_len_c(P, fin);
    const uint32_t rank = (uint32_t)(atomicAdd((unsigned long long *)(P.tile_k + u),
                                               (1ull << UNIT_KEY_BITS) | keys) >> UNIT_KEY_BITS);
    if (rank < cap) P.recs[(size_t)u * cap + rank] = ((uint64_t)pos << 32) | fin;
    else if (rank == cap) P.ovf_list[chk(P, atomicAdd(&P.hdr->ovf_count, 1u), P.n_tiles)] = u;
    if (P.chunk_adds) atomicAdd((unsigned long long *)(P.chunk + (u >> P.chunk_shift)), keys);
}

// Walk limit of start p of slice u, relative to the slice start: the first
// offset above p, found between the slice's first offset index and the next
// slice's.
__device__ __forceinline__ uint32_t w_limit(const MatchParams &P, uint32_t u, uint64_t p) {
    const uint64_t ustart = (uint64_t)u << SLICE_SHIFT;
    const uint64_t remain = P.n - ustart;
    const uint32_t rem = remain < LIM_MAX ? (uint32_t)remain : LIM_MAX;
    if (P.n_seg <= 1) return rem;
    // (bounded: offsets out of order leave some indices unwritten)
    uint32_t lo = __ldg(P.unit_seg + u), hi = u + 1 < P.n_tiles ? __ldg(P.unit_seg + u + 1) : P.n_seg;
    lo = lo < P.n_seg ? lo : P.n_seg;
    hi = hi < P.n_seg ? hi : P.n_seg;
    while (lo < hi) {
        const uint32_t mid = (lo + hi) >> 1;
        if (__ldg(P.seg + mid) > p) hi = mid; else lo = mid + 1;
    }
    const uint64_t e = __ldg(P.seg + lo);
    const uint64_t r = e > ustart ? e - ustart : 0;
    return r < rem ? (uint32_t)r : rem;
}

// A lane's walk from the root, for starts the entry buffer has no room for.
template <int W>
__device__ __forceinline__ uint32_t w_walk_fin(const MatchParams &P, uint64_t ub, uint32_t q,
                                               uint32_t lim) {
    const uint32_t sigma = P.T.sigma, psh = W == 3 ? sigma : P.T.pk_shift;
    const uint32_t bmask = W == 0 ? (1u << psh) - 1u : META_BASE_MASK;
    uint32_t s = 0;
    for (;; q++) {
        const uint32_t c = q < lim ? (uint32_t)__ldg(P.in + chk(P, ub + q, P.n)) : 0x100u;
        uint32_t wd, bl, mt, f;
        const uint32_t cur = (uint32_t)chk(P, s, P.T.n_rec);
        load_step<W>(P.T.rec, cur, c, wd, bl, mt, f, psh);
        const int r = take_step(sigma, c, wd, bl, mt, s, bmask);
        if (r == 1) return rec_fin<W>(P, cur, f, mt);
        if (r == 2) return __ldg(P.T.leaf_fin + chk(P, s, P.T.leaf_words));
    }
}

static __device__ __noinline__ void w_walk(const MatchParams *PP, uint64_t p) {
    const MatchParams &P = *PP;
    const uint32_t u = (uint32_t)(p >> SLICE_SHIFT), pos = (uint32_t)p & (SLICE - 1);
    const uint32_t lim = w_limit(P, u, p);
    const uint64_t ub = (uint64_t)u << SLICE_SHIFT;
    uint32_t fin = 0;
    switch (P.T.W) {
        case 0: fin = w_walk_fin<0>(P, ub, pos, lim); break;
        case 1: fin = w_walk_fin<1>(P, ub, pos, lim); break;
        case 2: fin = w_walk_fin<2>(P, ub, pos, lim); break;
        case 3: fin = w_walk_fin<3>(P, ub, pos, lim); break;
        default: fin = w_walk_fin<8>(P, ub, pos, lim); break;
    }
    if (fin) w_emit(P, u, pos, fin);
}

// The text around a start, loaded without branches so that several starts'
// loads overlap: two 16-byte chunks (2-bit symbols) or three words (raw
// bytes) from the aligned address at or below p; zeros where they would pass
// the input's end (ok false).
template <int PACKED>
struct WText {
    uint4 a, b;
    bool ok;
};

template <int PACKED>
__device__ __forceinline__ WText<PACKED> w_text(const MatchParams &P, bool on, uint64_t p) {
    WText<PACKED> t;
    const uint64_t c = p & (PACKED ? ~15ull : ~3ull);
    t.ok = on && c + (PACKED ? 32 : 12) <= P.n;
    const uint8_t *src = P.in + (t.ok ? c : 0ull);
    if (PACKED) {
        t.a = ld_stream16_if(t.ok, src);
        t.b = ld_stream16_if(t.ok, src + 16);
    } else {
        t.a = make_uint4(ld_stream4_if(t.ok, src), ld_stream4_if(t.ok, src + 4),
                         ld_stream4_if(t.ok, src + 8), 0u);
        t.b = make_uint4(0u, 0u, 0u, 0u);
    }
    return t;
}

// Prefix index (k symbols) of the start p that t was loaded for, or WX_ROOT
// where it cannot be formed: too near the input's end, or a byte outside the
// packed range among the symbols read.
template <int PACKED>
__device__ __forceinline__ uint32_t w_prefix(const MatchParams &P, const WText<PACKED> &t, uint64_t p) {
    const uint32_t k = P.k, bps = P.T.bps;
    if (PACKED) {
        const uint32_t bad = (t.a.x | t.a.y | t.a.z | t.a.w | t.b.x | t.b.y | t.b.z | t.b.w) & 0xFCFCFCFCu;
        const uint32_t w = __funnelshift_r(r_pack2(t.a), r_pack2(t.b), 2 * ((uint32_t)p & 15u));
        return !t.ok || bad ? WX_ROOT : (w & ((1u << (2 * k)) - 1u));
    }
    // at most 6 symbols (k * bps <= 20, bps >= 3)
    const uint32_t sh = 8 * ((uint32_t)p & 3u);
    uint32_t lo = __funnelshift_r(t.a.x, t.a.y, sh), hi = __funnelshift_r(t.a.y, t.a.z, sh);
    uint32_t x = 0, bad = 0;
    for (uint32_t i = 0; i < k; i++) {
        const uint32_t s = lo & 0xFFu;
        bad |= s >> bps;
        x |= s << (bps * i);
        lo = __funnelshift_r(lo, hi, 8);
        hi >>= 8;
    }
    return !t.ok || bad ? WX_ROOT : x;
}

// Empties a warp's candidate queue (n <= WQCAP window positions): every start
// a window stands for, one per lane, is tested against a prefix bitmap; the
// survivors go to the entry buffer (position << 24 | prefix index), or are
// walked here when it is full.
template <int PACKED, int S>
__device__ __noinline__ void w_flush(const MatchParams *PP, const uint32_t *q, uint32_t n,
                                     const uint32_t *Fs, uint32_t gw, uint32_t gstride,
                                     uint32_t lane) {
    const MatchParams &P = *PP;
    const uint32_t lt = (1u << lane) - 1u;
    const uint32_t f_mask = (1u << (P.wf_k * P.T.bps)) - 1u;
    constexpr int R = PACKED ? 2 : 4;  // rounds of 32 starts whose loads overlap
    for (uint32_t e0 = 0; e0 < n * S; e0 += 32 * R) {
        uint64_t en[R];
        uint32_t kept[R];
        WText<PACKED> tx[R];
#pragma unroll
        for (int r = 0; r < R; r++) {
            const uint32_t e = e0 + 32 * r + lane;
            const bool in = e < n * S;
            const uint32_t v = q[in ? e / S : 0u];
            const uint64_t pr = gw + (uint64_t)(v >> 10) * gstride;
            const uint64_t p = (pr << (SLICE_SHIFT + 1)) + (v & 1023u) - (S - 1 - e % S);
            const bool on = in && p < P.starts_end;
            en[r] = on ? p : ~0ull;
            tx[r] = w_text<PACKED>(P, on, p);
        }
#pragma unroll
        for (int r = 0; r < R; r++) {
            const uint64_t p = en[r];
            const uint32_t x = w_prefix<PACKED>(P, tx[r], p);
            const uint32_t fx = x & f_mask;
            const uint32_t fw = Fs ? Fs[fx >> 5] : __ldg(P.wf + (fx >> 5));
            const bool keep = p != ~0ull && (x == WX_ROOT || ((fw >> (fx & 31)) & 1u));
            en[r] = (p << 24) | x;
            kept[r] = __ballot_sync(0xFFFFFFFFu, keep);
        }
        uint32_t tot = 0;
#pragma unroll
        for (int r = 0; r < R; r++) tot += __popc(kept[r]);
        if (tot == 0) continue;
        // no reservation once the buffer is full, so that the counter stays
        // within one reservation per warp of its capacity
        uint32_t base = P.wbuf_cap;
        if (lane == 0 && *(volatile uint32_t *)&P.hdr->defer_entries < P.wbuf_cap)
            base = atomicAdd(&P.hdr->defer_entries, tot);
        base = __shfl_sync(0xFFFFFFFFu, base, 0);
#pragma unroll
        for (int r = 0; r < R; r++) {
            if ((kept[r] >> lane) & 1u) {
                const uint32_t at = base + __popc(kept[r] & lt);
                if (at < P.wbuf_cap) P.wbuf[at] = en[r];
                else w_walk(&P, en[r] >> 24);
            }
            base += __popc(kept[r]);
        }
        __syncwarp();
    }
    __syncwarp();
}

// Copies n words (a multiple of 4) of global memory to shared memory, each
// word 2^rep times in a row; `skew` moves the place where a CTA begins, so
// that the SMs do not ask the same L2 slices for the same lines at once.
template <uint32_t NT>
__device__ __forceinline__ void w_fill(uint32_t *dst, const uint32_t *src, uint32_t n, uint32_t rep,
                                       uint32_t skew) {
    constexpr uint32_t U = 8;  // loads in flight per thread
    const uint32_t nv = (n << rep) >> 2;
    uint4 *d = reinterpret_cast<uint4 *>(dst);
    const uint32_t off = nv ? skew % nv : 0u;
    for (uint32_t i0 = threadIdx.x; i0 < nv; i0 += NT * U) {
        uint4 v[U];
        uint32_t at[U];
#pragma unroll
        for (uint32_t u = 0; u < U; u++) {
            const uint32_t i = i0 + u * NT;
            at[u] = i + off < nv ? i + off : i + off - nv;
            if (i >= nv) at[u] = 0;
        }
        if (rep == 0) {
#pragma unroll
            for (uint32_t u = 0; u < U; u++) v[u] = __ldg(reinterpret_cast<const uint4 *>(src) + at[u]);
        } else if (rep == 1) {
#pragma unroll
            for (uint32_t u = 0; u < U; u++) {
                const uint2 x = __ldg(reinterpret_cast<const uint2 *>(src) + at[u]);
                v[u] = make_uint4(x.x, x.x, x.y, x.y);
            }
        } else {
#pragma unroll
            for (uint32_t u = 0; u < U; u++) {
                const uint32_t x = __ldg(src + ((4 * at[u]) >> rep));
                v[u] = make_uint4(x, x, x, x);
            }
        }
#pragma unroll
        for (uint32_t u = 0; u < U; u++)
            if (i0 + u * NT < nv) d[at[u]] = v[u];
    }
}

// The scan pass (TB: where the filter is read from).
template <int PACKED, int S, int NB, int G5, int TB>
__global__ void __launch_bounds__((TB == WT_L2 ? WNW_SMALL : WNW) * 32, 1)
    k_scanw(const __grid_constant__ MatchParams P) {
    constexpr int NW = TB == WT_L2 ? WNW_SMALL : WNW;
    constexpr uint32_t HALO = PACKED ? 16u : 4u;  // bytes of the next chunk a step reads
    constexpr uint32_t NWIN = 32 / S;             // windows of a lane
    extern __shared__ __align__(128) uint8_t smem[];
    const uint32_t lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const uint32_t n_pairs = (P.n_tiles + 1) >> 1;
    const uint32_t gw = blockIdx.x * NW + warp, gstride = gridDim.x * NW;
    if (blockIdx.x * NW >= n_pairs) return;

    if (P.n_seg > 1) unit_segments(P, gw, gstride, lane);

    // shared memory: H (all copies), the prefix bitmap, the queues
    const uint32_t hwords = TB == WT_L2 ? 0u : P.w_words << P.w_rep;
    uint32_t *Fs = reinterpret_cast<uint32_t *>(smem) + hwords;
    uint32_t *q = Fs + (TB == WT_L2 ? 0u : P.wf_words) + warp * WQCAP;
    if (TB != WT_L2) {
        w_fill<NW * 32>(reinterpret_cast<uint32_t *>(smem), P.T.H, P.w_words,
                        TB == WT_ONE ? 0u : P.w_rep, blockIdx.x * 160u);
        w_fill<NW * 32>(Fs, P.wf, P.wf_words, 0u, blockIdx.x * 32u);
        __syncthreads();
    }
    WConst K;
    K.gm = P.w_gm;
    K.tbl = P.T.H;
    K.hm = TB == WT_COPIES ? P.w_words << (2 + P.w_rep) : P.w_words;
    K.amask = ~((4u << P.w_rep) - 1u);
    K.c4 = (lane & ((1u << P.w_rep) - 1u)) << 2;
    const uint32_t *Fq = (TB != WT_L2 && P.wf_words) ? Fs : nullptr;

    const uint64_t N = P.n, N16 = N & ~15ull;
    const uint32_t lt = (1u << lane) - 1u;
    const bool l31 = lane == 31;
    const bool al32 = ((uintptr_t)P.in & 31) == 0;
    uint32_t qn = 0;
    auto load_head = [&](bool on, const uint8_t *a) -> uint4 {
        if (!PACKED) return make_uint4(ld_stream4_if(on, a), 0u, 0u, 0u);
        return ld_stream16_if(on, a);
    };
    // one step: the warp's i-th chunk of 1,024 bytes from registers (h: the
    // next chunk's head, on lane 31); forced = windows that are candidates
    // whatever the filter says
    auto step = [&](uint32_t i, const WChunk &c, const uint4 &h, uint32_t forced) {
        uint32_t w[9];
        if (!PACKED) {
#pragma unroll
            for (int x = 0; x < 8; x++) w[x] = c.w[x];
            const uint32_t nx = __shfl_down_sync(0xFFFFFFFFu, c.w[0], 1);
            w[8] = l31 ? h.x : nx;
        } else {
            w[0] = r_pack2(make_uint4(c.w[0], c.w[1], c.w[2], c.w[3]));
            w[1] = r_pack2(make_uint4(c.w[4], c.w[5], c.w[6], c.w[7]));
            // lane 31 offers the next chunk's head to itself
            const uint32_t nx = __shfl_down_sync(0xFFFFFFFFu, w[0], 1);
            w[2] = l31 ? r_pack2(h) : nx;
#pragma unroll
            for (int x = 3; x < 9; x++) w[x] = 0;
        }
        uint32_t m = w_filter<PACKED, S, NB, G5, TB>(w, K) | forced;
        if (P.w_badmask) {
            // bytes outside the packed symbol range, where H would need
            // completions over them (patterns that end inside a window): the
            // windows that may hold one are candidates (all of a lane's, in
            // the rare steps that have any)
            const uint32_t hm = P.w_badmask;
            const uint32_t ra = (c.w[0] | c.w[1] | c.w[2] | c.w[3] | c.w[4] | c.w[5] | c.w[6] | c.w[7]) & hm;
            const uint32_t rh = (h.x | h.y | h.z | h.w) & hm;
            if (__any_sync(0xFFFFFFFFu, (ra | rh) != 0)) {
                const uint32_t na = __ballot_sync(0xFFFFFFFFu, ra != 0);
                const uint32_t nh = __ballot_sync(0xFFFFFFFFu, rh != 0);
                if (((na >> lane) & 1u) || (l31 ? nh != 0 : ((na >> (lane + 1)) & 1u)))
                    m |= NWIN == 32 ? 0xFFFFFFFFu : (1u << (NWIN & 31)) - 1u;
            }
        }
        uint32_t any = __ballot_sync(0xFFFFFFFFu, m != 0);
        while (any) {
            if (m) {
                const uint32_t j = __ffs(m) - 1;
                m &= m - 1;
                q[qn + __popc(any & lt)] = (i << 10) + (lane * 32 + j * S + S - 1);
            }
            qn += __popc(any);
            if (qn > WQCAP - 32) {
                __syncwarp();
                w_flush<PACKED, S>(&P, q, qn, Fq, gw, gstride, lane);
                qn = 0;
            }
            any = __ballot_sync(0xFFFFFFFFu, m != 0);
        }
    };
    // clean chunks: every load, the next chunk's head included, inside the input
    const uint64_t gc = N >= HALO ? (N - HALO) >> (SLICE_SHIFT + 1) : 0;
    const uint32_t g_clean = gc < n_pairs ? (uint32_t)gc : n_pairs;
    const uint32_t n_it = gw < g_clean ? (g_clean - gw + gstride - 1) / gstride : 0u;
    const uint64_t step_b = (uint64_t)gstride << (SLICE_SHIFT + 1);
    const uint8_t *src = P.in + ((uint64_t)gw << (SLICE_SHIFT + 1)) + lane * 32u;
    uint32_t i = 0;
    if (n_it) {
        for (uint32_t f = 1; f < WPF && f < n_it; f++)
            prefetch_l2_if(lane == 0, src + f * step_b, 2 * SLICE);
        WChunk c0, c1;
        uint4 h0, h1;
        w_load32(src, al32, c0);
        h0 = load_head(l31, src + 32);
        for (;; i++) {
            const bool more = i + 1 < n_it;
            src += step_b;
            if (WPF) prefetch_l2_if(lane == 0 && i + WPF < n_it, src + (WPF - 1) * step_b, 2 * SLICE);
            if (more) {
                w_load32(src, al32, c1);
                h1 = load_head(l31, src + 32);
            }
            step(i, c0, h0, 0u);
            if (!more) break;
            c0 = c1;
            h0 = h1;
        }
        i++;
    }
    // the last chunks: loads as far as the input goes in whole 16-byte pieces;
    // windows that reach past them are candidates (starts at or past
    // starts_end are dropped by the flush)
    for (uint32_t g = gw + i * gstride; g < n_pairs; g += gstride, i++) {
        const uint64_t s0 = (uint64_t)g << (SLICE_SHIFT + 1), o = s0 + lane * 32u;
        uint4 a = make_uint4(0, 0, 0, 0), b = a;
        if (o + 16 <= N) a = ld_stream16(P.in + o);
        if (o + 32 <= N) b = ld_stream16(P.in + o + 16);
        const WChunk c{{a.x, a.y, a.z, a.w, b.x, b.y, b.z, b.w}};
        const uint4 h = load_head(l31 && s0 + 2 * SLICE + HALO <= N, P.in + s0 + 2 * SLICE);
        uint32_t forced = 0;
        for (uint32_t x = 0; x < NWIN; x++)
            if (o + x * S + S - 1 + P.w_glen > N16) forced |= 1u << x;
        step(i, c, h, forced);
    }
    if (qn) {
        __syncwarp();
        w_flush<PACKED, S>(&P, q, qn, Fq, gw, gstride, lane);
    }
}

// Resolves the entries the scan left: each warp takes blocks of up to 128.
template <int W>
__global__ void __launch_bounds__(RES_WARPS * 32, RES_CTAS)
    k_wresolve(const __grid_constant__ MatchParams P) {
    __shared__ RWarpArea areas[RES_WARPS];
    const uint32_t lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const uint32_t lt = (1u << lane) - 1u;
    RWarpArea &A = areas[warp];
    const uint32_t n0 = *(volatile uint32_t *)&P.hdr->defer_entries;
    const uint32_t n = n0 < P.wbuf_cap ? n0 : P.wbuf_cap;
    const uint32_t gw = blockIdx.x * RES_WARPS + warp, gs = gridDim.x * RES_WARPS;
    // few entries: 32 at a time, so that more warps share the latency
    const uint32_t blk = n > gs * QCAP ? (uint32_t)QCAP : 32u;
    const uint32_t k = P.k;
    for (uint64_t b = (uint64_t)gw * blk; b < n; b += (uint64_t)gs * blk) {
        uint32_t qn = 0;
        for (uint32_t r = 0; r < blk; r += 32) {
            const uint64_t e = b + r + lane;
            bool keep = false;
            QEntry en{0u, 0u, 0u, 0u};
            if (e < n) {
                const uint64_t v = P.wbuf[e];
                const uint64_t p = v >> 24;
                const uint32_t x = (uint32_t)v & 0xFFFFFFu;
                en.unit = (uint32_t)chk(P, p >> SLICE_SHIFT, P.n_tiles);
                en.pos = (uint32_t)p & (SLICE - 1);
                en.lim = w_limit(P, en.unit, p);
                en.x = x;
                keep = true;
                if (x == WX_ROOT || en.pos + k > en.lim) {
                    en.x = ROOT_X;
                } else {
                    const uint32_t xx = (uint32_t)chk(P, x, 1ull << (k * P.T.bps));
                    keep = ((__ldg(P.F + (xx >> 5)) >> (xx & 31)) & 1u) != 0;
                }
            }
            const uint32_t bm = __ballot_sync(0xFFFFFFFFu, keep);
            if (keep) A.q[qn + __popc(bm & lt)] = en;
            qn += __popc(bm);
        }
        __syncwarp();
        if (qn == 0) continue;
        resolve_batch_inl<W, VAR_F | VAR_RES>(P, A.q, qn, P.F, P.C, nullptr, lane);
        for (uint32_t e = lane; e < qn; e += 32) {
            const QEntry en = A.q[e];
            if (en.x) w_emit(P, en.unit, en.pos, en.x);
        }
        __syncwarp();
    }
}

}  // namespace pfac
