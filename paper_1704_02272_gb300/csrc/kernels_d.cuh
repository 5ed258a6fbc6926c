// Dense scan kernel: 2-bit symbols and a pattern set so short that several
// positions of every slice match (Section 2.3 over uniform text: more than
// eight expected matches per 512 positions), one segment.
//
// Nearly every candidate is a match here, so what counts is the work per
// match, not the filter.  A warp takes chunks of 1,024 bytes (two slices); a
// lane packs its 32 symbols into two words and tests 32 prefix indices against
// the prefix bitmap F_k (copies over the banks).  The chunk's candidates are
// listed in shared memory in position order, then taken 32 at a time, one per
// lane: rank in F_k, entry E_k (in shared memory where it fits), and the
// record, stored coalesced at the candidate's rank in its slice.  An entry
// that names an output is the match.  One that names a depth-k state whose
// children include the next symbol (child masks M_k) is left pending: its
// record holds D_PEND | state (or the root, for a start whose window leaves
// the input or holds a byte outside the alphabet) and its index goes to the
// entry buffer, and k_wresolve walks it and puts the output, or none, in its
// place.  A record with no output writes no key.
//
// 128 MiB over 4 symbols with 1,000 patterns of 4 to 64 symbols (one position
// in twelve matches): the queued kernel, which resolved every candidate from
// its queue through L2, took 760 us; this one 162 us, and 43 us for the pending
// records (206 us when each slice listed its candidates by itself, with half
// the lanes idle).  It is bound by the instructions per position and per
// candidate (74% issue, 76% of the ALU pipe).
#pragma once
#include "kernels_w.cuh"

namespace pfac {

constexpr int DNW = 24;               // warps per CTA
constexpr uint32_t DQCAP = 64;        // pending records queued per warp
struct DWarpArea {
    uint32_t list[2 * SLICE];         // candidates: position | symbols << 10 | D_LIST_ROOT
    uint32_t pend[DQCAP];             // chunk << 10 | slice << 9 | slot
};
constexpr uint32_t D_LIST_ROOT = 0x80000000u;
constexpr uint32_t D_LIST_SYMS = 10;  // symbols kept with a candidate

// Walks pending record ri from the root (entry buffer full).
static __device__ __noinline__ void d_walk(const MatchParams *PP, uint64_t ri) {
    const MatchParams &P = *PP;
    const uint64_t u = ri >> SLICE_SHIFT, rec = P.recs[ri];
    const uint32_t pos = (uint32_t)(rec >> 32);
    const uint32_t fin = w_walk_any(P, u << SLICE_SHIFT, pos, w_limit(P, (uint32_t)u, (u << SLICE_SHIFT) + pos));
    P.recs[ri] = ((uint64_t)pos << 32) | fin;
    if (fin) atomicAdd((unsigned long long *)(P.tile_k + u), (unsigned long long)fin_len_c(P, fin));
}

// The pending records of a warp to the entry buffer; walked here, one per
// lane, when its part is full.
__device__ __forceinline__ void d_flush(const MatchParams &P, const uint32_t *pend, uint32_t n,
                                        uint32_t gw, uint32_t gstride, uint32_t lane) {
    const uint32_t sub = chk32(P, gw & P.wsub_mask, WSUB_MAX);
    uint32_t *cnt = P.wcnt + sub * WSUB_STRIDE;
    uint64_t *buf = P.wbuf + (size_t)sub * P.wsub_cap;
    uint32_t base = P.wsub_cap;
    if (lane == 0 && *(volatile uint32_t *)cnt < P.wsub_cap) base = atomicAdd(cnt, n);
    base = __shfl_sync(0xFFFFFFFFu, base, 0);
    for (uint32_t e = lane; e < n; e += 32) {
        const uint32_t v = pend[chk32(P, e, DQCAP)];
        const uint64_t u = ((gw + (uint64_t)(v >> 10) * gstride) << 1) + ((v >> 9) & 1u);
        const uint64_t ri = chk(P, (u << SLICE_SHIFT) + (v & (SLICE - 1)), (uint64_t)P.n_tiles << SLICE_SHIFT);
        if (base + e < P.wsub_cap) buf[base + e] = ri;
        else d_walk(&P, ri);
    }
    __syncwarp();
}

template <int ES>
__global__ void __launch_bounds__(DNW * 32, 1) k_scand(const __grid_constant__ MatchParams P) {
    extern __shared__ __align__(128) uint8_t smem[];
    const uint32_t lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const uint32_t n_pairs = (P.n_tiles + 1) >> 1;
    const uint32_t gw = blockIdx.x * DNW + warp, gstride = gridDim.x * DNW;
    if (blockIdx.x * DNW >= n_pairs) return;
    // shared memory: F_k (all copies), counts, child masks, entries, the warps'
    // lists; sections padded to whole vectors
    const uint32_t rep = P.rep_log2;
    const uint32_t fw = P.tbl_words >> rep;
    uint32_t *Fs = reinterpret_cast<uint32_t *>(smem);
    uint32_t *Cs = Fs + P.tbl_words;
    uint32_t *Ms = Cs + ((P.tbl_c_words + 3) & ~3u);
    uint32_t *Es = Ms + ((P.tbl_m_words + 3) & ~3u);
    DWarpArea &A = reinterpret_cast<DWarpArea *>(Es + ((P.tbl_e_words + 3) & ~3u))[warp];
    w_fill<DNW * 32>(Fs, P.F, fw, rep, blockIdx.x * 32u);
    for (uint32_t i = threadIdx.x; i < P.tbl_c_words; i += DNW * 32) Cs[i] = __ldg(P.C + i);
    for (uint32_t i = threadIdx.x; i < P.tbl_m_words; i += DNW * 32) Ms[i] = __ldg(P.M + i);
    if (ES) {
#pragma unroll 8
        for (uint32_t i = threadIdx.x; i < P.tbl_e_words; i += DNW * 32) Es[i] = __ldg(P.E + i);
    }
    __syncthreads();
    // from here on the call's counters are used, zeroed by the kernel before
    dep_wait();
    if (gw >= n_pairs) return;

    const uint64_t N = P.n, N16 = N & ~15ull;
    const uint32_t k = P.k, kmask = (1u << (2 * k)) - 1u, sigma = P.T.sigma;
    // symbols read from a start on: its window, and the next for the masks
    const bool masks = P.tbl_m_words != 0 && k < D_LIST_SYMS;
    const uint32_t k_read = k + (masks ? 1 : 0);
    const uint32_t lt = (1u << lane) - 1u;
    const bool l31 = lane == 31;
    const bool al32 = ((uintptr_t)P.in & 31) == 0;
    // word address of window t in the lane's copy: (((t & kmask) >> 5) << rep
    // | copy) * 4, as one rotate and one and-or (kernels_q.cuh)
    const uint32_t ramt = (3u - rep) & 31u, wmask = (kmask >> 5) << (rep + 2);
    const uint32_t copy = lane & ((1u << rep) - 1u), c4 = copy << 2;
    const uint64_t gc = N >= 16 ? (N - 16) >> (SLICE_SHIFT + 1) : 0;
    const uint32_t g_clean = gc < n_pairs ? (uint32_t)gc : n_pairs;
    const uint32_t n_it = (n_pairs - gw + gstride - 1) / gstride;
    const uint32_t n_ok = gw < g_clean ? (g_clean - gw + gstride - 1) / gstride : 0u;
    const uint64_t step_b = (uint64_t)gstride << (SLICE_SHIFT + 1);
    const uint8_t *src = P.in + ((uint64_t)gw << (SLICE_SHIFT + 1)) + lane * 32u;
    auto load = [&](uint32_t i, WChunk &c, uint4 &h) {
        if (i < n_ok) {
            const uint8_t *s = chk_in(P, src, l31 ? 48 : 32);
            w_load32(s, al32, c);
            h = ld_stream16_if(l31, s + 32);
            return;
        }
        const uint64_t s0 = (gw + (uint64_t)i * gstride) << (SLICE_SHIFT + 1), o = s0 + lane * 32u;
        const uint4 a = ld_stream16_if(o + 16 <= N, P.in + o);
        const uint4 b = ld_stream16_if(o + 32 <= N, P.in + o + 16);
        c = WChunk{{a.x, a.y, a.z, a.w, b.x, b.y, b.z, b.w}};
        h = ld_stream16_if(l31 && s0 + 2 * SLICE + 16 <= N, P.in + s0 + 2 * SLICE);
    };
    WChunk c0, c1;
    uint4 h0, h1;
    uint32_t np = 0;  // pending records queued
    load(0, c0, h0);
    for (uint32_t i = 0; i < n_it; i++) {
        src += step_b;
        if (i + 1 < n_it) load(i + 1, c1, h1);
        const uint64_t g = gw + (uint64_t)i * gstride;
        const uint64_t o = (g << (SLICE_SHIFT + 1)) + lane * 32u;
        const uint4 ca = make_uint4(c0.w[0], c0.w[1], c0.w[2], c0.w[3]);
        const uint4 cb = make_uint4(c0.w[4], c0.w[5], c0.w[6], c0.w[7]);
        const uint32_t w0 = r_pack2(ca), w1 = r_pack2(cb);
        const uint32_t nx = __shfl_down_sync(0xFFFFFFFFu, w0, 1);
        const uint32_t w2 = l31 ? r_pack2(h0) : nx;
        uint32_t acc[4] = {0, 0, 0, 0};
#pragma unroll
        for (int j = 0; j < 32; j++) {
            const uint32_t t = j == 0 ? w0 : (j < 16 ? __funnelshift_r(w0, w1, 2 * j)
                                                    : (j == 16 ? w1 : __funnelshift_r(w1, w2, 2 * (j - 16))));
            const uint32_t x = *reinterpret_cast<const uint32_t *>(
                smem + chk(P, (__funnelshift_r(t, t, ramt) & wmask) | c4, P.tbl_words * 4ull));
            acc[j >> 3] = __funnelshift_r(acc[j >> 3], __funnelshift_r(x, x, t), 1);
        }
        uint32_t m = __byte_perm(__byte_perm(acc[0], acc[1], 0x0073), __byte_perm(acc[2], acc[3], 0x0073), 0x5410);
        // windows that leave the whole 16-byte pieces of the input (with the
        // symbol after them, which the child masks are asked about), or hold
        // a byte outside the 2-bit range: walked from the root
        uint32_t root = 0;
        const uint32_t bad = (ca.x | ca.y | ca.z | ca.w | cb.x | cb.y | cb.z | cb.w) & 0xFCFCFCFCu;
        const uint32_t badh = (h0.x | h0.y | h0.z | h0.w) & 0xFCFCFCFCu;
        if (__any_sync(0xFFFFFFFFu, (bad | badh) != 0)) {
            const uint32_t own = r_bad2(ca) | (r_bad2(cb) << 16);
            const uint32_t nb = __shfl_down_sync(0xFFFFFFFFu, own, 1);
            uint64_t b = (uint64_t)own | ((uint64_t)(l31 ? r_bad2(h0) : nb) << 32);
            for (uint32_t s = 0; s < k; s++, b >>= 1) root |= (uint32_t)b;
        }
        if (i >= n_ok)
            for (uint32_t j = 0; j < 32; j++)
                if (o + j + k_read > N16) root |= 1u << j;
        m |= root;
        if (o + 32 > P.starts_end) {  // starts at or past it start no walk
            const uint64_t left = P.starts_end > o ? P.starts_end - o : 0;
            m &= left >= 32 ? 0xFFFFFFFFu : (1u << (uint32_t)left) - 1u;
        }
        // ---- the chunk's candidates listed in position order
        uint32_t at = __popc(m);
        const uint32_t own_n = at;
#pragma unroll
        for (int s = 1; s < 32; s <<= 1) {
            const uint32_t v = __shfl_up_sync(0xFFFFFFFFu, at, s);
            if (lane >= (uint32_t)s) at += v;
        }
        const uint32_t tot_a = __shfl_sync(0xFFFFFFFFu, at, 15), tot = __shfl_sync(0xFFFFFFFFu, at, 31);
        at -= own_n;
        uint32_t mm = m;
        while (mm) {
            const uint32_t j = __ffs(mm) - 1;
            mm &= mm - 1;
            const uint32_t lo = j < 16 ? w0 : w1, hi = j < 16 ? w1 : w2;
            const uint32_t t = __funnelshift_r(lo, hi, 2 * (j & 15)) & ((1u << (2 * D_LIST_SYMS)) - 1u);
            A.list[chk32(P, at++, 2 * SLICE)] = (lane * 32 + j) | (t << 10) | (((root >> j) & 1u) ? D_LIST_ROOT : 0u);
        }
        __syncwarp();
        // the records of both slices, 32 candidates at a time (no candidate of
        // the second where it lies past the last unit)
        const uint64_t u0 = 2 * g;
        uint32_t keys_a = 0, keys_b = 0;
        for (uint32_t b0 = 0; b0 < tot; b0 += 32) {
            const uint32_t idx = b0 + lane;
            bool pend = false;
            const bool second = idx >= tot_a;
            const uint32_t slot = second ? idx - tot_a : idx;
            if (idx < tot) {
                const uint32_t e = A.list[chk32(P, idx, 2 * SLICE)];
                const uint64_t u = u0 + (second ? 1 : 0);
                uint32_t fin, keys = 0;
                if (e & D_LIST_ROOT) {
                    pend = true;
                    fin = D_PEND | D_PEND_ROOT;
                } else {
                    const uint32_t t = (e & ~D_LIST_ROOT) >> 10;
                    const uint32_t x = t & kmask;
                    const uint32_t r = (uint32_t)chk(
                        P, prefix_rank(Fs + (rep ? copy : 0u), rep, Cs, P.c_shift, x), P.T.n_e[k]);
                    const uint32_t ev = ES ? Es[chk32(P, r, P.tbl_e_words)] : __ldg(P.E + r);
                    if (ev & D_CONT) {
                        pend = true;
                        if (masks) {
                            // four mask bits an entry (all: it reports output)
                            const uint32_t mr = (Ms[chk32(P, r >> 3, P.tbl_m_words)] >> (4 * (r & 7))) & 15u;
                            const uint32_t c = (t >> (2 * k)) & 3u;
                            pend = mr == 15u || (c < sigma && ((mr >> c) & 1u));
                        }
                        fin = pend ? D_PEND | (ev & D_PEND_STATE) : 0u;
                    } else {
                        // (long lists are counted on their own: the sum of
                        // the others stays in 32 bits)
                        fin = ev;
                        if ((ev & FIN_LEN_ESC) != FIN_LEN_ESC) keys = ev & FIN_LEN_ESC;
                        else atomicAdd((unsigned long long *)(P.tile_k + chk(P, u, P.n_tiles)),
                                       (unsigned long long)fin_len_c(P, ev));
                    }
                }
                keys_a += second ? 0u : keys;
                keys_b += second ? keys : 0u;
                P.recs[chk(P, (size_t)u * P.unit_cap + slot, (uint64_t)P.n_tiles * P.unit_cap)] = ((uint64_t)(e & (SLICE - 1)) << 32) | fin;
            }
            const uint32_t pm = __ballot_sync(0xFFFFFFFFu, pend);
            if (pm) {
                if (pend) A.pend[chk32(P, np + __popc(pm & lt), DQCAP)] = (i << 10) | (second ? (uint32_t)SLICE : 0u) | slot;
                np += __popc(pm);
                if (np > DQCAP - 32) {
                    __syncwarp();
                    d_flush(P, A.pend, np, gw, gstride, lane);
                    np = 0;
                }
            }
        }
        keys_a = __reduce_add_sync(0xFFFFFFFFu, keys_a);
        keys_b = __reduce_add_sync(0xFFFFFFFFu, keys_b);
        if (lane < 2) {
            const uint32_t n = lane ? tot - tot_a : tot_a;
            if (n) {
                const uint64_t u = chk(P, u0 + lane, P.n_tiles);
                P.tile_m[u] = n;
                atomicAdd((unsigned long long *)(P.tile_k + u),
                          (unsigned long long)(lane ? keys_b : keys_a));
            }
        }
        __syncwarp();
        c0 = c1;
        h0 = h1;
    }
    if (np) {
        __syncwarp();
        d_flush(P, A.pend, np, gw, gstride, lane);
    }
}

}  // namespace pfac
