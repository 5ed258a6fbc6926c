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
//   call's entry buffer with one atomic, on one of up to 64 parts of it so
//   that the warps do not queue on one counter.  When a part is full its
//   warps' lanes walk their starts from the root instead, with the segment
//   indices that the launch before (k_zero) has written.
// * k_wresolve then takes the entries in any order: segment limit, prefix
//   entry, the walk, and one record per match at an atomically taken slot of
//   its slice; the key expansion sorts the few records of a slice.
//
// What bounds it: shared-memory lookups (3.7 wavefronts of random banks per
// warp-wide lookup with one copy of H: 59 cycles of an SM's shared memory per
// slice at stride 1) and the ALU instructions around them; S, the bits tested
// and the copies of H are chosen per table to balance both (window.cpp).  Of the
// L1 data pipe / the ALU pipe: DNA 63 / 71%, packets 60 / 72%, 20 symbols 67 /
// 67%, 64 symbols 59 / 69%, 256 symbols at stride 2 76 / 57%.
// Measured scan pass, before (queued or register-staged kernel) and with this
// one: 20 symbols x 10,000 patterns, 256 MiB: 858 -> 174 us; 64 x 100,000,
// 128 MiB: 569 -> 108 us; 256 x 1,000, 512 MiB: 293 -> 159 us; 52 letters x
// 100, 100 MiB: 111 -> 32 us; 1 GiB of packets against 20,000 signatures:
// 2,773 -> 781 us; DNA x 10,000, 256 MiB: 281 -> 185 us.  The resolver after
// it takes the place of the other kernels' resolver (packets: 374 -> 297 us).
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
__device__ __forceinline__ uint32_t w_lookup(const MatchParams &P, const uint32_t (&w)[9], int j, const WConst &K) {
    extern __shared__ __align__(128) uint8_t smem[];
    const uint32_t t = w_twin<PACKED>(w, j);
    uint32_t y = t * K.gm;
    if (G5) y += w_twin<PACKED>(w, j + 1) * WIN_MUL2;
    const uint32_t h = __umulhi(y, K.hm);
    uint32_t x;
    if (TB == WT_L2) x = __ldg(K.tbl + chk32(P, h, P.w_words));
    else if (TB == WT_ONE) x = reinterpret_cast<const uint32_t *>(smem)[chk32(P, h, P.w_words)];
    else x = *reinterpret_cast<const uint32_t *>(smem + chk32(P, (h & K.amask) | K.c4, (4ull * P.w_words) << P.w_rep));
    uint32_t r = __funnelshift_r(x, x, w_twin<PACKED>(w, j + (PACKED ? 0 : 2)));
    if (NB >= 2) r &= __funnelshift_r(x, x, w_twin<PACKED>(w, j + (PACKED ? 3 : 0)));
    if (NB >= 3) r &= __funnelshift_r(x, x, w_twin<PACKED>(w, j + (PACKED ? 6 : 1)));
    return r;
}

// All windows of the lane's 32 positions: bit i is set when the one at
// symbol i * S + S - 1 passes.
template <int PACKED, int S, int NB, int G5, int TB>
__device__ __forceinline__ uint32_t w_filter(const MatchParams &P, const uint32_t (&w)[9], const WConst &K) {
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
                    acc[c], w_lookup<PACKED, NB, G5, TB>(P, w, (8 * c + i) * S + S - 1, K), 1);
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
            m |= (w_lookup<PACKED, NB, G5, TB>(P, w, i * S + S - 1, K) & 1u) << i;
        return m;
    }
}

// One match: a record in the slice's space while it has room (in any order),
// and the slice's counts: records above bit UNIT_KEY_BITS of its word, keys
// below, so that one atomic takes the slot and counts the keys.  (A slice with
// more matches than its space is walked again by the expansion.)  With few
// slices the chunks' key counts are added up here too; with many, neighbouring
// matches would queue on one chunk's word (1 GiB of packets: 0.8 instead of
// 0.36 ms), and k_reduce sums them.
//
// SHARED: the calling lanes' matches of one slice add once.  For the scan's own
// walks, where most starts may match: 32 adds then queued on one word (8 MiB of
// one symbol that two patterns repeat, apart / shared: 1,074 / 630 us a call; 9
// MB of printable packets against 50,000 signatures 319 / 309).  Not for the
// resolver, whose few matches lie apart: shared there too, 1 GiB of packets
// 1,204 -> 1,249 us.
template <bool SHARED>
__device__ __forceinline__ void w_emit(const MatchParams &P, uint32_t u, uint32_t pos, uint32_t fin) {
    u = (uint32_t)chk(P, u, P.n_tiles);
    const uint32_t cap = P.unit_cap, lane = threadIdx.x & 31;
    const uint32_t same = SHARED ? __match_any_sync(__activemask(), u) : 1u << lane;
    const uint32_t first = __ffs(same) - 1;
    unsigned long long keys = fin_len_c(P, fin);
    if (SHARED) keys = __reduce_add_sync(same, (uint32_t)keys);  // (lists of at most 2^24 ids)
    uint32_t rank = 0;
    if (!SHARED || lane == first) {
        const unsigned long long n = SHARED ? __popc(same) : 1;
        rank = (uint32_t)(atomicAdd((unsigned long long *)(P.tile_k + u), (n << UNIT_KEY_BITS) | keys) >>
                          UNIT_KEY_BITS);
        if (P.chunk_adds) atomicAdd((unsigned long long *)(P.chunk + (u >> P.chunk_shift)), keys);
    }
    if (SHARED) rank = __shfl_sync(same, rank, first) + __popc(same & ((1u << lane) - 1u));
    if (rank < cap) P.recs[(size_t)u * cap + rank] = ((uint64_t)pos << 32) | fin;
}

// Walk limit of start p of slice u, relative to the slice start: the first
// offset above p, found between the slice's first offset index and the next
// slice's (both written by the launch before the scan).
__device__ __forceinline__ uint32_t w_limit(const MatchParams &P, uint32_t u, uint64_t p) {
    const uint64_t ustart = (uint64_t)u << SLICE_SHIFT;
    const uint64_t remain = P.n - ustart;
    const uint32_t rem = remain < LIM_MAX ? (uint32_t)remain : LIM_MAX;
    if (P.n_seg <= 1) return rem;
    // (bounded: offsets out of order leave some indices unwritten)
    uint32_t lo = __ldg(P.unit_seg + chk32(P, u, P.n_tiles));
    uint32_t hi = u + 1 < P.n_tiles ? __ldg(P.unit_seg + u + 1) : P.n_seg;
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

// A lane's walk from the root, for starts the entry buffer has no room for
// (and, after the scan, for slices whose records were not kept).
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

__device__ __forceinline__ uint32_t w_walk_any(const MatchParams &P, uint64_t ub, uint32_t pos,
                                               uint32_t lim) {
    switch (P.T.W) {
        case 0: return w_walk_fin<0>(P, ub, pos, lim);
        case 1: return w_walk_fin<1>(P, ub, pos, lim);
        case 2: return w_walk_fin<2>(P, ub, pos, lim);
        case 3: return w_walk_fin<3>(P, ub, pos, lim);
        default: return w_walk_fin<8>(P, ub, pos, lim);
    }
}

static __device__ __noinline__ void w_walk(const MatchParams *PP, uint64_t p) {
    const MatchParams &P = *PP;
    const uint32_t u = (uint32_t)(p >> SLICE_SHIFT), pos = (uint32_t)p & (SLICE - 1);
    const uint32_t fin = w_walk_any(P, (uint64_t)u << SLICE_SHIFT, pos, w_limit(P, u, p));
    if (fin) w_emit<true>(P, u, pos, fin);
}

// The text around a start, loaded without branches so that several starts'
// loads overlap: the aligned 16-byte (2-bit symbols) or 8-byte piece that
// holds it, and the next one where its k symbols reach into that (every
// scattered load costs its lane a cycle of the SM's L1); zeros where they
// would pass the input's end (ok false).
template <int PACKED>
struct WText {
    uint4 a, b;
    bool ok;
};

template <int PACKED>
__device__ __forceinline__ WText<PACKED> w_text(const MatchParams &P, bool on, uint64_t p) {
    constexpr uint32_t PIECE = PACKED ? 16 : 8;
    WText<PACKED> t;
    const uint64_t c = p & ~(uint64_t)(PIECE - 1);
    t.ok = on && c + 2 * PIECE <= P.n;
    const bool two = t.ok && ((uint32_t)p & (PIECE - 1)) + P.k > PIECE;
    const uint8_t *src = P.in + (t.ok ? c : 0ull);
    if (PACKED) {
        t.a = ld_stream16_if(t.ok, src);
        t.b = ld_stream16_if(two, src + PIECE);
    } else {
        const uint2 a = ld_stream8_if(t.ok, src), b = ld_stream8_if(two, src + PIECE);
        t.a = make_uint4(a.x, a.y, b.x, b.y);
        t.b = make_uint4(0u, 0u, 0u, 0u);
    }
    return t;
}

// The eight bytes from byte s (0 .. 7) of a 16-byte string.
__device__ __forceinline__ uint2 bytes8(const uint4 &v, uint32_t s) {
    const bool up = s >= 4;
    const uint32_t x = up ? v.y : v.x, y = up ? v.z : v.y, z = up ? v.w : v.z, sh = 8 * (s & 3);
    return make_uint2(__funnelshift_r(x, y, sh), __funnelshift_r(y, z, sh));
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
    const uint2 w = bytes8(t.a, (uint32_t)p & 7u);
    uint32_t lo = w.x, hi = w.y;
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
// survivors go to the entry buffer (position << 24 | prefix index, or its rank
// where the bitmap and its counts are in shared memory), or are walked here
// when it is full.
template <int PACKED, int S>
__device__ __forceinline__ void w_flush(const MatchParams &P, const uint32_t *q, uint32_t n,
                                        const uint32_t *Fs, const uint32_t *Cs, uint32_t gw, uint32_t gstride,
                                        uint32_t lane) {
    const uint32_t lt = (1u << lane) - 1u;
    constexpr int R = PACKED ? 2 : 4;  // rounds of 32 starts whose loads overlap
    for (uint32_t e0 = 0; e0 < n * S; e0 += 32 * R) {
        uint64_t en[R];
        uint32_t kept[R];
        WText<PACKED> tx[R];
#pragma unroll
        for (int r = 0; r < R; r++) {
            const uint32_t e = e0 + 32 * r + lane;
            const bool in = e < n * S;
            const uint32_t v = q[in ? chk32(P, e / S, WQCAP) : 0u];
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
            const uint32_t fx = x == WX_ROOT ? 0u : (uint32_t)chk(P, x, 1ull << (P.k * P.T.bps));
            const uint32_t fw = Fs ? Fs[fx >> 5] : __ldg(P.F + (fx >> 5));
            const bool keep = p != ~0ull && (x == WX_ROOT || ((fw >> (fx & 31)) & 1u));
            const uint32_t low = Fs && keep && x != WX_ROOT ? prefix_rank(Fs, 0, Cs, P.c_shift, x) : x;
            en[r] = (p << 24) | low;
            kept[r] = __ballot_sync(0xFFFFFFFFu, keep);
        }
        uint32_t tot = 0;
#pragma unroll
        for (int r = 0; r < R; r++) tot += __popc(kept[r]);
        if (tot == 0) continue;
        // the warp's part of the buffer; no reservation once it is full, so
        // that its counter stays within one reservation per warp of its size
        const uint32_t sub = chk32(P, gw & P.wsub_mask, WSUB_MAX);
        uint32_t *cnt = P.wcnt + sub * WSUB_STRIDE;
        uint64_t *buf = P.wbuf + (size_t)sub * P.wsub_cap;
        uint32_t base = P.wsub_cap;
        if (lane == 0 && *(volatile uint32_t *)cnt < P.wsub_cap) base = atomicAdd(cnt, tot);
        base = __shfl_sync(0xFFFFFFFFu, base, 0);
#pragma unroll
        for (int r = 0; r < R; r++) {
            if ((kept[r] >> lane) & 1u) {
                const uint32_t at = base + __popc(kept[r] & lt);
                if (at < P.wsub_cap) buf[at] = en[r];
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

    // shared memory: H (all copies), the prefix bitmap and its counts, the queues
    const uint32_t hwords = TB == WT_L2 ? 0u : P.w_words << P.w_rep;
    uint32_t *Fs = reinterpret_cast<uint32_t *>(smem) + hwords;
    uint32_t *Cs = Fs + (TB == WT_L2 ? 0u : P.wf_words);
    uint32_t *q = Cs + (TB == WT_L2 ? 0u : P.wc_words) + warp * WQCAP;
    if (TB != WT_L2) {
        w_fill<NW * 32>(reinterpret_cast<uint32_t *>(smem), P.T.H, P.w_words,
                        TB == WT_ONE ? 0u : P.w_rep, blockIdx.x * 160u);
        w_fill<NW * 32>(Fs, P.F, P.wf_words, 0u, blockIdx.x * 32u);
        w_fill<NW * 32>(Cs, P.C, P.wc_words, 0u, 0u);
        __syncthreads();
    }
    // from here on the call's counters are used, zeroed by the kernel before
    dep_wait();
    WConst K;
    K.gm = P.w_gm;
    K.tbl = P.T.H;
    K.hm = TB == WT_COPIES ? P.w_words << (2 + P.w_rep) : P.w_words;
    K.amask = ~((4u << P.w_rep) - 1u);
    K.c4 = (lane & ((1u << P.w_rep) - 1u)) << 2;
    const uint32_t *Fq = (TB != WT_L2 && P.wf_words) ? Fs : nullptr, *Cq = Cs;

    const uint64_t N = P.n, N16 = N & ~15ull;
    const uint32_t lt = (1u << lane) - 1u;
    const bool l31 = lane == 31;
    const bool al32 = ((uintptr_t)P.in & 31) == 0;
    auto load_head = [&](bool on, const uint8_t *a) -> uint4 {
        if (!PACKED) return make_uint4(ld_stream4_if(on, a), 0u, 0u, 0u);
        return ld_stream16_if(on, a);
    };
    // clean chunks: every load, the next chunk's head included, inside the input
    const uint64_t gc = N >= HALO ? (N - HALO) >> (SLICE_SHIFT + 1) : 0;
    const uint32_t g_clean = gc < n_pairs ? (uint32_t)gc : n_pairs;
    const uint32_t n_it = (n_pairs - gw + gstride - 1) / gstride;  // gw < n_pairs or no step
    const uint32_t n_ok = gw < g_clean ? (g_clean - gw + gstride - 1) / gstride : 0u;
    const uint64_t step_b = (uint64_t)gstride << (SLICE_SHIFT + 1);
    const uint8_t *src = P.in + ((uint64_t)gw << (SLICE_SHIFT + 1)) + lane * 32u;
    // the warp's i-th chunk and, on lane 31, the head of the chunk after it;
    // past the clean ones as far as the input goes in whole 16-byte pieces
    auto load = [&](uint32_t i, WChunk &c, uint4 &h) {
        if (i < n_ok) {
            const uint8_t *s = chk_in(P, src, l31 ? 32 + HALO : 32);
            w_load32(s, al32, c);
            h = load_head(l31, s + 32);
            return;
        }
        const uint64_t s0 = (gw + (uint64_t)i * gstride) << (SLICE_SHIFT + 1), o = s0 + lane * 32u;
        const uint4 a = ld_stream16_if(o + 16 <= N, P.in + o);
        const uint4 b = ld_stream16_if(o + 32 <= N, P.in + o + 16);
        c = WChunk{{a.x, a.y, a.z, a.w, b.x, b.y, b.z, b.w}};
        h = load_head(l31 && s0 + 2 * SLICE + HALO <= N, P.in + s0 + 2 * SLICE);
    };
    WChunk c0, c1;
    uint4 h0, h1;
    uint32_t qn = 0;
    if (gw >= n_pairs) return;
    for (uint32_t f = 1; f < WPF && f < n_ok; f++)
        prefetch_l2_if(lane == 0, src + f * step_b, 2 * SLICE);
    load(0, c0, h0);
    for (uint32_t i = 0;; i++) {
        src += step_b;
        prefetch_l2_if(lane == 0 && i + WPF < n_ok, src + (WPF - 1) * step_b, 2 * SLICE);
        if (i + 1 < n_it) load(i + 1, c1, h1);
        uint32_t m = 0;
        if (i < n_it) {
            uint32_t w[9];
            if (!PACKED) {
#pragma unroll
                for (int x = 0; x < 8; x++) w[x] = c0.w[x];
                const uint32_t nx = __shfl_down_sync(0xFFFFFFFFu, c0.w[0], 1);
                w[8] = l31 ? h0.x : nx;
            } else {
                w[0] = r_pack2(make_uint4(c0.w[0], c0.w[1], c0.w[2], c0.w[3]));
                w[1] = r_pack2(make_uint4(c0.w[4], c0.w[5], c0.w[6], c0.w[7]));
                const uint32_t nx = __shfl_down_sync(0xFFFFFFFFu, w[0], 1);
                w[2] = l31 ? r_pack2(h0) : nx;
#pragma unroll
                for (int x = 3; x < 9; x++) w[x] = 0;
            }
            m = w_filter<PACKED, S, NB, G5, TB>(P, w, K);
            if (P.w_badmask) {
                // bytes outside the packed symbol range, where H would need
                // completions over them (patterns that end inside a window):
                // the windows that may hold one are candidates (all of a
                // lane's, in the rare steps that have any)
                const uint32_t hm = P.w_badmask;
                const uint32_t ra = (c0.w[0] | c0.w[1] | c0.w[2] | c0.w[3] | c0.w[4] | c0.w[5] |
                                     c0.w[6] | c0.w[7]) & hm;
                const uint32_t rh = (h0.x | h0.y | h0.z | h0.w) & hm;
                if (__any_sync(0xFFFFFFFFu, (ra | rh) != 0)) {
                    const uint32_t na = __ballot_sync(0xFFFFFFFFu, ra != 0);
                    const uint32_t nh = __ballot_sync(0xFFFFFFFFu, rh != 0);
                    if (((na >> lane) & 1u) || (l31 ? nh != 0 : ((na >> (lane + 1)) & 1u)))
                        m |= NWIN == 32 ? 0xFFFFFFFFu : (1u << (NWIN & 31)) - 1u;
                }
            }
            if (i >= n_ok) {
                // windows that reach past the whole 16-byte pieces are
                // candidates (starts at or past starts_end are dropped by
                // the flush)
                const uint64_t o = ((gw + (uint64_t)i * gstride) << (SLICE_SHIFT + 1)) + lane * 32u;
                for (uint32_t x = 0; x < NWIN; x++)
                    if (o + x * S + S - 1 + P.w_glen > N16) m |= 1u << x;
            }
        }
        // candidates to the queue, a round per lane's next one; a full queue
        // is flushed, and after the last chunk what is left
        uint32_t any = __ballot_sync(0xFFFFFFFFu, m != 0);
        while (any || (i >= n_it && qn)) {
            if (m) {
                const uint32_t j = __ffs(m) - 1;
                m &= m - 1;
                q[chk32(P, qn + __popc(any & lt), WQCAP)] = (i << 10) + (lane * 32 + j * S + S - 1);
            }
            qn += __popc(any);
            if (qn > WQCAP - 32 || i >= n_it) {
                __syncwarp();
                w_flush<PACKED, S>(P, q, qn, Fq, Cq, gw, gstride, lane);
                qn = 0;
            }
            any = __ballot_sync(0xFFFFFFFFu, m != 0);
        }
        if (i >= n_it) break;
        c0 = c1;
        h0 = h1;
    }
}

// Resolves the entries the scan left: each warp takes blocks of up to 64, two
// per lane.  What bounds it is the chain of dependent L2 loads of a walk, so
// the loads that do not depend on each other go out together: the slice's
// first offset indices and the eight symbols after the prefix, then the prefix
// node's words and the segment end, the prefix entry, and one record a round
// with the symbols at hand.  Walks still running after three rounds
// are packed one per lane and advance up to eight records of a chain at a
// time.
constexpr int WRU = 2;                       // entries per lane
constexpr uint32_t WRB = 32 * WRU;           // and per block
struct WTail {
    uint32_t unit[WRB], pos[WRB], q[WRB], lim[WRB], state[WRB], slot[WRB];
};
// pending records of the dense scan kernel (kernels_d.cuh): an entry is the
// record's index, its output word holds the state to walk from
constexpr uint32_t D_PEND = 0x80000000u, D_PEND_ROOT = 0x40000000u, D_PEND_STATE = 0x3FFFFFFFu;

// A resolved walk's output: a match of the window kernel, or the pending
// record's output (0: none) and its keys.
template <int DENSE>
__device__ __forceinline__ void w_result(const MatchParams &P, uint32_t u, uint32_t pos, uint32_t slot,
                                         uint32_t fin) {
    if (!DENSE) {
        if (fin) w_emit<false>(P, u, pos, fin);
        return;
    }
    P.recs[(size_t)u * P.unit_cap + slot] = ((uint64_t)pos << 32) | fin;
    if (fin) atomicAdd((unsigned long long *)(P.tile_k + u), (unsigned long long)fin_len_c(P, fin));
}

template <int W, int DENSE>
__global__ void __launch_bounds__(RES_WARPS * 32, RES_CTAS)
    k_wresolve(const __grid_constant__ MatchParams P) {
    __shared__ WTail tails[RES_WARPS];
    const uint32_t lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const uint32_t lt = (1u << lane) - 1u;
    WTail &T = tails[warp];
    dep_wait();
    const uint32_t gw = blockIdx.x * RES_WARPS + warp, gs = gridDim.x * RES_WARPS;
    // the buffer's parts: lane l counts those of parts l and l + 32
    const uint32_t parts = P.wsub_mask + 1;
    uint32_t n0 = lane < parts ? *(volatile uint32_t *)(P.wcnt + lane * WSUB_STRIDE) : 0u;
    uint32_t n1 = lane + 32 < parts ? *(volatile uint32_t *)(P.wcnt + (lane + 32) * WSUB_STRIDE) : 0u;
    n0 = n0 < P.wsub_cap ? n0 : P.wsub_cap;
    n1 = n1 < P.wsub_cap ? n1 : P.wsub_cap;
    // few entries: blocks of 32, so that more warps share the latency
    const uint32_t all = __reduce_add_sync(0xFFFFFFFFu, (n0 + 31) / 32 + (n1 + 31) / 32);
    const uint32_t blk = all > gs ? WRB : 32u;
    // blocks up to and including each part
    uint32_t i0 = (n0 + blk - 1) / blk, i1 = (n1 + blk - 1) / blk;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t a = __shfl_up_sync(0xFFFFFFFFu, i0, o), c = __shfl_up_sync(0xFFFFFFFFu, i1, o);
        if (lane >= (uint32_t)o) {
            i0 += a;
            i1 += c;
        }
    }
    i1 += __shfl_sync(0xFFFFFFFFu, i0, 31);
    const uint32_t n_blk = __shfl_sync(0xFFFFFFFFu, i1, 31);

    const uint32_t k = P.k, sigma = P.T.sigma, psh = W == 3 ? sigma : P.T.pk_shift;
    const uint32_t bmask = W == 0 ? (1u << psh) - 1u : META_BASE_MASK;
    const uint32_t *__restrict__ rec = P.T.rec;
    for (uint32_t bi = gw; bi < n_blk; bi += gs) {
        // the block's part, its place there and the part's entries
        const uint32_t sub = __popc(__ballot_sync(0xFFFFFFFFu, i0 <= bi)) +
                             __popc(__ballot_sync(0xFFFFFFFFu, i1 <= bi));
        const uint32_t e0 = __shfl_sync(0xFFFFFFFFu, i0, (sub - 1) & 31);
        const uint32_t e1 = __shfl_sync(0xFFFFFFFFu, i1, (sub - 1) & 31);
        const uint32_t before = sub == 0 ? 0u : (sub <= 32 ? e0 : e1);
        const uint32_t s0 = __shfl_sync(0xFFFFFFFFu, n0, sub & 31);
        const uint32_t s1 = __shfl_sync(0xFFFFFFFFu, n1, sub & 31);
        const uint32_t n = sub < 32 ? s0 : s1;
        const uint64_t *buf = P.wbuf + (size_t)sub * P.wsub_cap;
        const uint32_t b = (bi - before) * blk;

        // ---- prefix entry, walk limit and the symbols after the prefix
        // state: -1 nothing to do, 0 walking from st at q, 1 stopped at st,
        // 2 stopped on merged leaf st, 3 output known (fin)
        int state[WRU];
        uint32_t unit[WRU], pos[WRU], lim[WRU], st[WRU], q[WRU], fin[WRU], tq[WRU], t0[WRU], t1[WRU];
        uint32_t slo[WRU], x[WRU], slot[WRU], tn[WRU];
#pragma unroll
        for (int u = 0; u < WRU; u++) {
            const uint32_t e = b + 32 * u + lane;
            const bool on = e < n && (uint32_t)(32 * u) < blk;
            const uint64_t v = on ? buf[e] : 0ull;
            state[u] = on ? 0 : -1;
            st[u] = 0;
            if (DENSE) {
                const uint64_t r = on ? P.recs[chk(P, v, (uint64_t)P.n_tiles << SLICE_SHIFT)] : 0ull;
                unit[u] = (uint32_t)chk(P, v >> SLICE_SHIFT, P.n_tiles ? P.n_tiles : 1);
                slot[u] = (uint32_t)v & (SLICE - 1);
                pos[u] = (uint32_t)(r >> 32);
                st[u] = (uint32_t)r & D_PEND_STATE;
                x[u] = (uint32_t)r & D_PEND_ROOT ? WX_ROOT : 0u;
            } else {
                const uint64_t p = v >> 24;
                unit[u] = (uint32_t)chk(P, p >> SLICE_SHIFT, P.n_tiles ? P.n_tiles : 1);
                slot[u] = 0;
                pos[u] = (uint32_t)p & (SLICE - 1);
                x[u] = (uint32_t)v & 0xFFFFFFu;
            }
            // the slice's first offset indices, the text from p + k on (from
            // p for a walk from the root)
            slo[u] = P.n_seg > 1 ? __ldg(P.unit_seg + unit[u]) : 0u;
            tq[u] = pos[u] + (x[u] == WX_ROOT ? 0u : k);
            // the aligned 8-byte piece, and the next where it holds few of them
            const uint64_t a = ((uint64_t)unit[u] << SLICE_SHIFT) + tq[u], c = a & ~7ull;
            const bool ok = on && c + 16 <= P.n, two = ok && ((uint32_t)a & 7u) > 4;
            const uint8_t *src = P.in + (ok ? c : 0ull);
            const uint2 pa = ld_stream8_if(ok, src), pb = ld_stream8_if(two, src + 8);
            const uint2 s8 = bytes8(make_uint4(pa.x, pa.y, pb.x, pb.y), (uint32_t)a & 7u);
            t0[u] = s8.x;
            t1[u] = s8.y;
            tn[u] = two ? 8u : 8u - ((uint32_t)a & 7u);
            if (!ok) tq[u] = 0xFFFFFF00u;  // no symbol at hand
        }
#pragma unroll
        for (int u = 0; u < WRU; u++) {
            const uint64_t us = (uint64_t)unit[u] << SLICE_SHIFT, p = us + pos[u];
            const uint64_t remain = P.n - us;
            lim[u] = remain < LIM_MAX ? (uint32_t)remain : LIM_MAX;
            if (P.n_seg > 1) {
                // the first offset beyond p, from the slice's first index on:
                // a few steps, then by search up to the next slice's index
                // (bounded: offsets out of order leave some indices unwritten)
                uint32_t lo = slo[u] < P.n_seg ? slo[u] : P.n_seg;
                uint64_t e = __ldg(P.seg + lo);
                for (uint32_t i = 0; i < 3 && e <= p && lo < P.n_seg; i++) e = __ldg(P.seg + ++lo);
                if (e <= p && lo < P.n_seg) {
                    uint32_t hi = unit[u] + 1 < P.n_tiles ? __ldg(P.unit_seg + unit[u] + 1) : P.n_seg;
                    hi = hi < P.n_seg ? hi : P.n_seg;
                    while (lo < hi) {
                        const uint32_t mid = (lo + hi) >> 1;
                        if (__ldg(P.seg + mid) > p) hi = mid; else lo = mid + 1;
                    }
                    e = __ldg(P.seg + lo);
                }
                const uint64_t r = e > us ? e - us : 0;
                lim[u] = r < lim[u] ? (uint32_t)r : lim[u];
            }
            fin[u] = 0;
            q[u] = pos[u];
            if (DENSE) {
                if (x[u] != WX_ROOT) q[u] += k;
            } else if (state[u] == 0 && x[u] != WX_ROOT && pos[u] + k <= lim[u]) {
                // (the scan has tested the index's bit, or ranked it too)
                uint32_t r = x[u];
                if (!P.w_ranked) r = prefix_rank(P.F, 0, P.C, P.c_shift, (uint32_t)chk(P, r, 1ull << (k * P.T.bps)));
                r = (uint32_t)chk(P, r, P.T.n_e[k]);
                const uint32_t ev = __ldg(P.E + r);
                q[u] = pos[u] + k;
                if (ev & D_CONT) {
                    st[u] = ev & D_VAL_MASK;
                } else {
                    state[u] = 3;
                    fin[u] = ev;
                }
            }
        }
        // symbol at slice offset i of walk u
        auto symbol = [&](int u, uint32_t i) -> uint32_t {
            if (i >= lim[u]) return 0x100u;
            const uint32_t d = i - tq[u];
            if (d < tn[u]) return ((d < 4 ? t0[u] : t1[u]) >> (8 * (d & 3))) & 0xFFu;
            return __ldg(P.in + chk(P, ((uint64_t)unit[u] << SLICE_SHIFT) + i, P.n));
        };
        // ---- three rounds, one record of each walk a round
#pragma unroll 1
        for (int round = 0; round < 3; round++) {
            bool any = false;
#pragma unroll
            for (int u = 0; u < WRU; u++) any |= state[u] == 0;
            if (!__any_sync(0xFFFFFFFFu, any)) break;
            uint32_t c[WRU], wd[WRU], bl[WRU], mt[WRU], f1[WRU];
#pragma unroll
            for (int u = 0; u < WRU; u++) {
                if (state[u] != 0) continue;
                c[u] = symbol(u, q[u]);
                load_step<W>(rec, (uint32_t)chk(P, st[u], P.T.n_rec), c[u], wd[u], bl[u], mt[u], f1[u], psh);
            }
#pragma unroll
            for (int u = 0; u < WRU; u++) {
                if (state[u] != 0) continue;
                const uint32_t cur = st[u];
                const int r = take_step(sigma, c[u], wd[u], bl[u], mt[u], st[u], bmask);
                if (r == 0) {
                    q[u]++;
                } else if (r == 2) {
                    state[u] = 2;
                } else if (W == 0 && !(mt[u] & PK_FIN)) {
                    state[u] = 3;
                } else if (W <= 1 || W == 3) {  // outputs in their own array
                    st[u] = cur;
                    state[u] = 1;
                } else {
                    fin[u] = f1[u];
                    state[u] = 3;
                }
            }
        }
        // ---- the walks still running, one per lane
        uint32_t nt = 0;
#pragma unroll
        for (int u = 0; u < WRU; u++) {
            const bool w = state[u] == 0;
            const uint32_t bm = __ballot_sync(0xFFFFFFFFu, w);
            if (w) {
                const uint32_t t = chk32(P, nt + __popc(bm & lt), WRB);
                T.unit[t] = unit[u];
                T.pos[t] = pos[u];
                T.q[t] = q[u];
                T.lim[t] = lim[u];
                T.state[t] = st[u];
                T.slot[t] = slot[u];
            }
            nt += __popc(bm);
        }
        __syncwarp();
        // outputs of the walks that have stopped
#pragma unroll
        for (int u = 0; u < WRU; u++) {
            if (state[u] == 1) fin[u] = rec_fin<W>(P, st[u], 0, PK_FIN);
            else if (state[u] == 2) fin[u] = __ldg(P.T.leaf_fin + chk(P, st[u], P.T.leaf_words));
            if (state[u] >= 1) w_result<DENSE>(P, unit[u], pos[u], slot[u], fin[u]);
        }
        for (uint32_t b0 = 0; b0 < nt; b0 += 32) {
            const uint32_t t = b0 + lane;
            if (t < nt) {
                const uint32_t un = T.unit[t], lm = T.lim[t];
                uint32_t s1 = T.state[t], q1 = T.q[t], f = 0;
                const uint64_t ub = (uint64_t)un << SLICE_SHIFT;
                // each round fetches TS consecutive records from the current
                // state and the next TS symbols; along a single-child chain
                // (placed in consecutive records) it advances up to TS levels
                constexpr int TS = (W == 8 || W == 2) ? 4 : 8;
                const uint32_t n_rec = P.T.n_rec;
                bool done = false;
                while (!done) {
                    uint32_t c[TS], wd[TS], bl[TS], mt[TS], f1[TS];
#pragma unroll
                    for (int i = 0; i < TS; i++) {
                        c[i] = q1 + i < lm ? (uint32_t)__ldg(P.in + chk(P, ub + q1 + i, P.n)) : 0x100u;
                        if (i == 0 || s1 + i < n_rec) {
                            load_step<W>(rec, (uint32_t)chk(P, s1 + i, n_rec), c[i], wd[i], bl[i], mt[i],
                                         f1[i], psh);
                        } else {
                            wd[i] = bl[i] = mt[i] = f1[i] = 0;
                        }
                    }
#pragma unroll
                    for (int i = 0; i < TS; i++) {
                        uint32_t nx = 0;
                        const uint32_t cur = s1 + i;
                        const int r = take_step(sigma, c[i], wd[i], bl[i], mt[i], nx, bmask);
                        if (r == 1) {
                            f = rec_fin<W>(P, cur, f1[i], mt[i]);
                            done = true;
                            break;
                        }
                        if (r == 2) {
                            f = __ldg(P.T.leaf_fin + chk(P, nx, P.T.leaf_words));
                            done = true;
                            break;
                        }
                        if (i + 1 < TS && nx == cur + 1) continue;
                        s1 = nx;
                        q1 += i + 1;
                        break;
                    }
                }
                w_result<DENSE>(P, un, T.pos[t], T.slot[t], f);
            }
        }
        __syncwarp();
    }
    // the offsets are checked here, by the last warps first: they have the
    // fewest entries
    if (!DENSE && P.n_seg > 1) unit_segments<true, false>(P, gs - 1 - gw, gs, lane);
}

}  // namespace pfac
