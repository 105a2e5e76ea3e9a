// AC refinements of scans with restart intervals.
//
// A refinement scan says for every block which still-zero positions become non-zero and carries one correction bit
// for every non-zero position passed over, so how many bits a symbol takes depends on the block it is in: an interval is
// one chain.  The chain itself is short, though: a symbol's code (a window of the stream, a table entry), the position
// its run of zeros ends at (one entry of the block's list of still-zero positions) and an addition.  Everything else
// a block needs -- its list, the union of the earlier scans' masks, the correction bits in reading order, the new
// positions and their signs -- does not lie on the chain and is done for many blocks at a time.
//
// One CTA per work item (32 restart intervals, see Item).  Warp 0 follows the chains, a lane an interval, for at most
// kRefineSteps symbols; meanwhile the helper warps decode the blocks it finished in the round before once more, a thread a
// block, into side data, and list the still-zero positions of the blocks to come.  Every thread works for its
// own lane's interval, so that shared-memory columns never collide.  At the end of a round the CTA meets once.
//
// Bound by the latency of warp 0's step, 166 cycles a symbol alone on an SM and 200 to 220 beside other CTAs (entropy_kernel's, which
// does all of it in the lane: 700).  What it took: nothing but the chain in the step; one straight line instead of branches
// for block ends and rare cases (350 -> 175); the next symbol's entry requested before anything else that is loaded (-> 166);
// the rings filled by a helper.
// Rounds of 16, 32, 48 and 64 symbols: 233, 177, 157 and 164 k cycles for the busiest CTA of 4 ImageNet-shaped images, whose
// refinement wave took 211 us and takes 84.  1024 such images are better off with entropy_kernel: see refine_in_ctas.
//
// Side data of a block: {mask of the band's non-zero positions after the scan, correction bits in reading order (the last
// one in bit 0), newly non-zero positions, the positive ones among them}; the pixel kernel applies them.
#pragma once
#include <cuda_runtime.h>
#include <stddef.h>
#include <stdint.h>

#include "pcr_entropy.cuh"
#include "pcr_types.h"

namespace pcr {

constexpr int kRefineWarps = 8;               // one that follows the chains, seven helpers
constexpr uint32_t kRefineLists = 16;         // blocks of an interval whose lists are held: being made, being read, or of finished
                                              // blocks whose side data is being made
constexpr uint32_t kRefineRing = 64;          // words of the stream per lane.  A block takes at most 44 (63 symbols of at most 17
                                              // bits, 3 sixteen-zero runs, one run length, 63 correction bits), and its first
                                              // word is held until its side data is made
constexpr int kRefineSteps = 48;              // symbols a round
constexpr uint32_t kRefineAlign = 4096;       // of the structure: a table's place and an index are put together by an OR
struct RefineShared {
    struct { ScanTab t; uint8_t pad[4096 - sizeof(ScanTab)]; } tabs[2];
    uint8_t zpos[64][kRefineLists][32];       // [i][slot][lane]: position of the block's i-th still-zero coefficient of the band, minus
                                              // i; entry nz: Se + 1 - nz (as if position Se + 1 followed)
    uint32_t ring[(kRefineRing + 2) * 32];    // see LaneRing
    uint64_t mask[kRefineLists][32];          // positions of the band that are non-zero before the scan
    uint32_t ends[kRefineLists][32];          // 256 nz + 255, nz = how many still-zero positions there are (at most 63), and, from
                                              // bit 16 on, 256 times the rank that ends the block (nz, or nz - 1 if the last of them is Se)
    uint16_t start[kRefineLists][32];         // where the block began: bit position modulo the ring, kEntEobRefine if inside an
                                              // end-of-band run
    // of the lane's interval: masks of up to four earlier scans (null: none) and their words a block, a byte each;
    // side data of the scan, the first block's row (as a block index) and column, blocks a row in the scan and in the planes
    uint64_t src[4][32], out[32];
    uint32_t range[2][32];                    // ... its bytes
    uint32_t stride[32], row0[32], col0[32], width[32], pitch[32], tab[32];
    // By parity of the round: the blocks whose side data, and those whose lists are to be made: first and number
    uint32_t side_first[2][32], side_count[2][32], list_first[2][32], list_count[2][32], more[2];
    // ... the first bit that is still read, and how far the ring is filled
    uint32_t keep[2][32], filled[2][32];
};
static_assert(offsetof(RefineShared, tabs) == 0 && offsetof(RefineShared, zpos) % 512 == 0 && offsetof(RefineShared, ring) % 16 == 0, "see kRefineAlign");
static_assert(32 * kRefineRing <= kEntEobRefine, "positions modulo the ring fit below the flag");
constexpr size_t kRefineBytes = sizeof(RefineShared) + kRefineAlign;

__device__ __forceinline__ uint32_t refine_slot(uint32_t j) { return j & (kRefineLists - 1u); }
// shared address of the lane's column in slot's list: entry i lies 512 i bytes on
__device__ __forceinline__ uint32_t refine_zpos(const RefineShared& sh, uint32_t slot, uint32_t lane) {
    return (uint32_t)__cvta_generic_to_shared(sh.zpos) + (slot << 5) + lane;
}

// block j of the lane's interval as an index inside its component of its image
__device__ __forceinline__ uint32_t refine_block(const RefineShared& sh, uint32_t lane, uint32_t j) {
    const uint32_t w = sh.width[lane];
    uint32_t x = sh.col0[lane] + j, at = sh.row0[lane];
    if (x >= w) { const uint32_t r = x / w; x -= r * w; at += r * sh.pitch[lane]; }     // (an interval of several rows)
    return at + x;
}

// the masks of block j of the lane's interval
__device__ __forceinline__ uint64_t refine_masks(const RefineShared& sh, uint32_t lane, uint32_t j) {
    const uint32_t bi = refine_block(sh, lane, j), st = sh.stride[lane];
    uint64_t h = 0;
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        const uint64_t* p = reinterpret_cast<const uint64_t*>(sh.src[q][lane]);
        // (through L2: another thread of the CTA may have written it in this launch)
        if (p) h |= __ldcg(p + (uint64_t)bi * ((st >> (8 * q)) & 255u));
    }
    return h;
}

// The list of a block's still-zero positions (see RefineShared::zpos) into its slot.
__device__ __forceinline__ void refine_list(RefineShared& sh, uint32_t lane, uint32_t slot, uint64_t h, uint64_t band, uint32_t Se) {
    h &= band;
    sh.mask[slot][lane] = h;
    const uint64_t z = ~h & band;
    const uint32_t z0 = (uint32_t)z, z1 = (uint32_t)(z >> 32);
    const uint32_t dst0 = refine_zpos(sh, slot, lane);
    uint32_t dst = dst0, v = 0;                                // v: position minus number of still-zero ones before it
    // (straight through all positions, so that lanes with different masks stay together)
#pragma unroll
    for (int pos = 0; pos < 64; ++pos) {
        if (((pos < 32 ? z0 : z1) >> (pos & 31)) & 1u) {
            asm volatile("st.shared.u8 [%0], %1;" : : "r"(dst), "r"(v) : "memory");
            dst += 512u;
        } else ++v;
    }
    const uint32_t n = (dst - dst0) >> 9;
    asm volatile("st.shared.u8 [%0], %1;" : : "r"(dst), "r"(Se + 1u - n) : "memory");      // closing entry: behind the band
    sh.ends[slot][lane] = (256u * n + 255u) | ((256u * ((z >> Se) & 1u ? n - 1u : n)) << 16);
}

using RefineWords = RingWords<kRefineRing>;
// (a table's place and an index are put together by an OR)
__device__ __forceinline__ uint32_t refine_entry(uint32_t tab, uint32_t win) {
    return lds16(tab | ((win >> (31 - kTabBits)) & ((2u << kTabBits) - 2u)));
}
constexpr uint32_t kEntRunSkip = 0x7F1Fu;     // of an entry: the run of zeros (from bit 8 on) and the bits to skip, without the flag
constexpr uint32_t kEntNew = 0x20u;           // the flag: a new coefficient

// One finished block once more -> side data.
__device__ __forceinline__ void refine_side(RefineShared& sh, uint32_t lane, uint32_t j, uint32_t Ss) {
    const uint32_t slot = refine_slot(j);
    const uint32_t st = sh.start[slot][lane], ends = sh.ends[slot][lane], nz = ends & 0xFFFFu, tend = ends >> 16;
    const uint32_t zb = refine_zpos(sh, slot, lane), tab = sh.tab[lane];
    RefineWords W;
    W.col = (uint32_t)__cvta_generic_to_shared(sh.ring) + 4u * lane;
    uint32_t at = st & (kEntEobRefine - 1u), zi = 0, ep = Ss, t;
    uint32_t s0 = 0, s1 = 0, N0 = 0, N1 = 0, G0 = 0, G1 = 0;   // correction bits, new positions, positive ones
    W.load(at);
    uint32_t win = W.window(at);
#pragma unroll 1
    do {
        uint32_t e = refine_entry(tab, win);
        const uint32_t behind = W.behind(at);
        e = st & kEntEobRefine ? kEntEobRefine : e;            // the whole block lies inside an end-of-band run
        if (e == 0) e = long_code(tab, win, kTabAcRefine);   // (there is one: the chain has passed it)
        t = min(zi + (e & kEntRunSkip), nz);                   // 256 times the target's rank, and eight other bits
        const uint32_t e2 = lds8(zb + 2u * (t & 0x3F00u)), skip = e & 31u, n = e2 - ep, k = e2 + (t >> 8);
        const uint32_t isnew = (t | 255u) < nz && (e & kEntNew) ? 1u : 0u, plus = isnew & shr0(win, 32u - skip);
        N0 |= shl0(isnew, k); N1 |= shl0(isnew, k - 32u);
        G0 |= shl0(plus, k); G1 |= shl0(plus, k - 32u);
        const uint32_t corr = __funnelshift_l(behind, win, skip);
        at += skip + n;
        W.load(at);
        if (n > 32u) {
            RefineWords V;
            V.col = W.col;
            V.load(at - n + 32u);
            s1 = shl0(s0, n - 32u) | (corr >> (64u - n));
            s0 = __funnelshift_l(V.window(at - n + 32u), corr, n - 32u);
        } else {
            s1 = __funnelshift_lc(s0, s1, n);
            s0 = shl0(s0, n) | shr0(corr, 32u - n);
        }
        win = skip + n > 31u ? W.window(at) : __funnelshift_l(behind, win, skip + n);
        zi = (t | 255u) + 1u; ep = e2;
    } while (t < tend);
    const uint64_t h = sh.mask[slot][lane];
    uint4* o = reinterpret_cast<uint4*>(sh.out[lane]) + 2ull * refine_block(sh, lane, j);
    o[0] = make_uint4((uint32_t)h | N0, (uint32_t)(h >> 32) | N1, s0, s1);
    o[1] = make_uint4(N0, N1, G0, G1);
}

// Pairs: a refinement that needs nothing but the masks of the refinement before it (same component, same band, same
// restart intervals) does not have to wait for that one's launch.  Lanes 0..15 follow sixteen intervals of the
// earlier scan, lanes 16..31 the same intervals of the later one, whose lists are made as the earlier one's side data gets
// ready.  The chain of a row is then as long as the longer of its two scans instead of their sum.
//
// Blocks from runs.item_blocks on do the wave's DC refinement scans, which touch nothing the others do.
// kRoi: restart intervals outside the MCU rows that the image's crop touches are left out (see entropy_kernel).
template <bool kRoi>
__global__ void __launch_bounds__(32 * kRefineWarps, 3) refine_kernel(Params P, ItemRuns runs) {
    extern __shared__ __align__(16) uint8_t s_refine[];
    const uint32_t over = (uint32_t)__cvta_generic_to_shared(s_refine) & (kRefineAlign - 1u);
    RefineShared& sh = *reinterpret_cast<RefineShared*>(s_refine + (over ? kRefineAlign - over : 0u));
    const uint32_t tid = threadIdx.x, wid = tid >> 5, lane = tid & 31u;
    if (blockIdx.x >= runs.item_blocks) {                     // whole block
        const uint32_t b = blockIdx.x - runs.item_blocks, chunk = b % runs.dc_chunks, i = b / runs.dc_chunks;
        dc_refine_image(P, runs.dc_s[i / runs.dc_images], (int)P.order[runs.dc_pos0 + i % runs.dc_images],
                        chunk * 32u * kRefineWarps + tid, runs.dc_chunks * 32u * kRefineWarps);
        return;
    }
    const unsigned full = 0xffffffffu;
    int run_no = 0;
    while (blockIdx.x >= runs.end[run_no]) ++run_no;
    const Item item = P.items[runs.first[run_no] + blockIdx.x - (run_no ? runs.end[run_no - 1] : 0u)];
    const bool two_images = item.next != 0;                   // (never a pair's item)
    const uint32_t si1 = two_images ? item.next - 1u : item.si + item.pair;
    const uint32_t N = (uint32_t)P.N, s0 = item.si / N, s1 = si1 / N;
    const ScanScript sc = load_entry(P.script + s0);          // (a pair's scans have the same component and band)
    const uint32_t Ss = (uint32_t)sc.Ss, Se = (uint32_t)sc.Se;
    const uint64_t band = low_mask((int)Se + 1) & ~low_mask((int)Ss);

    // what warp 0 keeps of its lane's interval
    const bool half = item.pair && lane >= 16u;               // this lane follows the later scan of the pair
    const uint32_t li = item.pair ? lane & 15u : lane;
    uint32_t n = 0, bstart = 0, bend = 0;                     // blocks, bytes
    int img = 0;
    bool bad = false;
    if (wid == 0) {
        const ScanDesc sd0 = load_entry(P.scans + item.si), sd1 = load_entry(P.scans + si1);
        const ImgDesc im0 = load_entry(P.imgs + item.si % N), im1 = load_entry(P.imgs + si1 % N);
        const ScanAux ax = load_entry(P.saux + (half ? s1 : s0));
        const uint32_t rem0 = sd0.nseg - item.seg0;           // restart intervals left in the first image
        const uint32_t which = half || (two_images && li >= rem0) ? 1u : 0u, si = which ? si1 : item.si;
        uint32_t seg = two_images && li >= rem0 ? li - rem0 : item.seg0 + li;
        const ScanDesc sd = which ? sd1 : sd0;
        img = (int)(si % N);
        const ImgDesc im = which ? im1 : im0;
        const Geometry g = make_geometry(im, P);
        const int c = sc.comp[0];
        bool done = li >= item.count;
        if (seg >= sd.nseg) { done = true; seg = 0; }
        const uint32_t mcu_w = g.ubw[c], total = mcu_w * g.ubh[c];
        const uint32_t m0 = sd.ri ? seg * sd.ri : 0u, m1 = sd.ri ? min(m0 + sd.ri, total) : total;
        if (m0 >= m1) done = true;
        if (kRoi && !done) {
            const CropRect rc = P.roi[img];
            const uint32_t mh = 8u * (uint32_t)P.vs, ph = c != 0 ? mh : 8u;           // pixel rows of an MCU row, of a block row of this scan
            const uint32_t lo = mh * (rc.y0 / mh), hi = mh * ((rc.y0 + rc.h + mh - 1u) / mh);
            const uint32_t r0 = m0 / mcu_w, r1 = (m1 - 1u) / mcu_w;
            if ((r1 + 1u) * ph <= lo || r0 * ph >= hi) done = true;
        }
        const uint32_t* segtab = P.seg_start + sd.seg_base;
        bstart = segtab[seg]; bend = segtab[seg + 1] - 2u;
        if (!done && (bstart < sd.data_off || bend > sd.data_end || bend < bstart)) { bad = true; done = true; }   // a missing marker left a hole
        if (done) { bstart = sd.data_off; bend = sd.data_off; }
        n = done ? 0u : m1 - m0;
        uint32_t strides = 0;
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const ScanAux x = load_entry(P.saux + ax.src[q < ax.nsrc ? q : 0]);
            sh.src[q][lane] = q < ax.nsrc ? reinterpret_cast<uint64_t>(P.aux + x.base + g.loff[c] * x.stride) : 0ull;
            strides |= x.stride << (8 * q);
        }
        sh.stride[lane] = strides;
        sh.out[lane] = reinterpret_cast<uint64_t>(P.aux + ax.base + g.loff[c] * 4ull);
        sh.row0[lane] = m0 / mcu_w * g.bw[c]; sh.col0[lane] = m0 % mcu_w; sh.width[lane] = mcu_w; sh.pitch[lane] = g.bw[c];
        sh.tab[lane] = (uint32_t)__cvta_generic_to_shared(&sh.tabs[which].t);
    } else {
        const ScanAux ax0 = load_entry(P.saux + s0), ax1 = load_entry(P.saux + s1);
        const uint4* a = reinterpret_cast<const uint4*>(P.tabs + ax0.tab0 + item.si % N);      // (an AC scan has one table)
        const uint4* b = reinterpret_cast<const uint4*>(P.tabs + ax1.tab0 + si1 % N);
        constexpr uint32_t words = sizeof(ScanTab) / 16;
        const uint32_t t0 = (uint32_t)__cvta_generic_to_shared(sh.tabs);
        for (uint32_t i = tid - 32u; i < (two_images || item.pair ? 2u : 1u) * words; i += 32u * (kRefineWarps - 1))
            sts128(t0 + (i < words ? 16u * i : 4096u + 16u * (i - words)), __ldg(i < words ? a + i : b + (i - words)));
    }
    const uint32_t ring = (uint32_t)__cvta_generic_to_shared(sh.ring) + 4u * lane;
    if (wid == 0) {
        // the lane's block it stands at, lists that are there, lists that have been asked for, blocks handed on
        uint32_t m = 0, have = 0, asked = half ? 0u : min(n, kRefineLists), handed = 0;
        bool done = n == 0;
        uint32_t pos = 8u * (bstart & 15u);                   // next bit of the lane's chain; the first one behind its interval
        const uint32_t limit = pos + 8u * (bend - bstart);
        uint32_t keep = pos, first = pos;                     // first bit of what is handed on next, of block m
        uint32_t eobrun = 0, zi = 0xFFFFFFFFu, ep = Ss;       // zi: 256 times the still-zero positions passed, minus one
        bool fresh = true;                                    // block m has not been begun
        uint32_t idle = 0, trace = 0;                         // rounds in which nothing moved on
        sh.list_first[0][lane] = 0; sh.list_count[0][lane] = asked; sh.side_first[0][lane] = 0; sh.side_count[0][lane] = 0;
        sh.keep[0][lane] = pos;
        sh.range[0][lane] = bstart; sh.range[1][lane] = bend;
        const bool any = __any_sync(full, n != 0);
        if (lane == 0) sh.more[0] = any;
        const uint32_t tab = sh.tab[lane];
        meet();
        for (uint32_t round = 0;; ++round) {
            const uint32_t b = round & 1u, nb = b ^ 1u;
            if (!sh.more[b]) break;                           // whole CTA
            // ---- the chains
            // a step reads the 64 bits from its start on, and a block's side data up to three words behind its last symbol's
            const uint32_t filled = round ? sh.filled[nb][lane] : 0u;
            uint32_t stop = done ? 0u : min(32u * (filled - min(filled, 3u)), limit + 1u);
            // A block's slot as the number its list, its ends and its start are addressed by: 32 slot + lane, and the place of the lists
            // (a multiple of 512) above.  The next block's ends are loaded ahead.
            const uint32_t lists = (uint32_t)__cvta_generic_to_shared(sh.zpos), to_ends = (uint32_t)__cvta_generic_to_shared(sh.ends) - 4u * lists;
            const uint32_t to_start = (uint32_t)__cvta_generic_to_shared(sh.start) - 2u * lists;
            auto slot_behind = [&](uint32_t at) { return ((at + 32u) & 511u) | lists; };
            uint32_t here = lists + (refine_slot(m) << 5) + lane, next = slot_behind(here);
            uint32_t ends = lds32(to_ends + 4u * here), ends_next = lds32(to_ends + 4u * next);
            RefineWords W;
            W.col = ring;
            if (m >= have) stop = 0;
            if (fresh && stop) sts16(to_start + 2u * here, (pos & (32u * kRefineRing - 1u)) | (eobrun ? kEntEobRefine : 0u));
            W.load(pos);
            uint32_t win = W.window(pos);
            uint32_t only = eobrun ? 0u : kEntRunSkip, force = eobrun ? kEntEobRefine : 0u;   // inside an end-of-band run no symbol is read
            // A step is one straight line: every lane walks it, what does not count is thrown away.  (With block ends and
            // rare cases as branches a step took 340 cycles.)  What is rare (a code longer than the table's index, a step that passed
            // more than 31 bits) makes the lane wait for the end of eight steps.  The chain: win -> e -> t -> e2 -> win.
            bool rare = false;
            uint32_t raw = refine_entry(tab, win);
#pragma unroll 1
            for (int s = 0; s < kRefineSteps; s += 8) {
#pragma unroll 4
                for (int q = 0; q < 8; ++q) {
                    const bool wanted = pos < stop && !rare;
                    const uint32_t behind = W.behind(pos), e = (raw & only) | force;
                    const bool act = wanted && e != 0;
                    rare = rare || (wanted && e == 0);
                    const uint32_t t = min(zi + e + 1u, ends & 0xFFFFu);           // 256 times the target's rank, and eight other bits
                    const uint32_t e2 = lds8(here + 2u * (t & 0x3F00u));          // (where the lane does not act: any byte of the lists)
                    const bool end = act && t >= ends >> 16;
                    // the symbol, and a correction bit for every non-zero position passed
                    const uint32_t skip = e & 31u, d = act ? skip - ep + e2 : 0u;
                    // blocks behind this one that an end of band covers, or that are left of a run of them
                    const uint32_t x = (e >> 8) & 15u, run = __funnelshift_l(shl0(win, skip - x), 1u, x);   // (2^x + the x bits that end the symbol)
                    const uint32_t left = (eobrun ? eobrun : (e >= kEntEobRefine ? run : 1u)) - 1u;
                    eobrun = end ? left : eobrun;
                    only = eobrun ? 0u : kEntRunSkip; force = eobrun ? kEntEobRefine : 0u;
                    win = __funnelshift_l(behind, win, d);
                    raw = refine_entry(tab, win);
                    pos += d;
                    rare = rare || d > 31u;
                    W.load_behind(pos);
                    zi = end ? 0xFFFFFFFFu : (act ? t | 255u : zi);
                    ep = end ? Ss : (act ? e2 : ep);
                    m += end ? 1u : 0u;
                    here = end ? next : here;
                    ends = end ? ends_next : ends;
                    next = slot_behind(here);
                    ends_next = lds32(to_ends + 4u * next);
                    const bool more = m < have;
                    sts16_if(end && more, to_start + 2u * here, (pos & (32u * kRefineRing - 1u)) | force);
                    stop = more ? stop : 0u;                   // also at the interval's end: have is at most n
                }
                if (rare) {
                    rare = false;
                    W.load(pos);
                    win = W.window(pos);
                    raw = refine_entry(tab, win);
                    if (raw == 0 && !eobrun && pos < stop) {
                        raw = long_code(tab, win, kTabAcRefine);
                        if (raw == 0) { bad = true; stop = 0; }        // no such symbol: the lane ends here
                    }
                }
                if (!__any_sync(full, pos < stop)) break;
            }
            fresh = m >= have;
            first = fresh ? pos : pos - ((pos - lds16(to_start + 2u * here)) & (32u * kRefineRing - 1u));
            bad = bad || (!done && pos > limit);
            // ---- what the round left: blocks handed .. m - 1 are finished.  At the meeting the lists asked for so far
            // are there, and the side data of the blocks handed on so far: their slots are free
            const uint32_t pm = __shfl_sync(full, m, (int)li), ph = __shfl_sync(full, handed, (int)li);
            const bool stuck = __shfl_sync(full, (int)((done || bad) && (n == 0 || m < n)), (int)li) != 0;      // the partner gets no further
            done = done || bad || m >= n || (half && stuck && m >= pm);
            have = asked;
            const uint32_t want = done ? asked : max(asked, min(half ? min(ph, n) : n, handed + kRefineLists));
            sh.side_first[nb][lane] = handed; sh.side_count[nb][lane] = m - handed;
            sh.list_first[nb][lane] = asked; sh.list_count[nb][lane] = want - asked;
            // (every round in which a lane has work left moves something on; should none do so for some rounds, the lanes give up)
            const uint32_t moved = pos + filled + m + have + want + handed + keep;
            idle = __any_sync(full, moved != trace) ? 0u : idle + 1u;
            trace = moved;
            if (idle == 8u && !done) bad = done = true;
            const bool more = __any_sync(full, !done || m != handed);
            if (lane == 0) sh.more[nb] = more;
            asked = want; handed = m;
            sh.keep[nb][lane] = keep;
            keep = first;
            meet();
        }
        if (bad) atomicMin(&P.status[img], kErrCorrupt);
        return;
    }
    // the last of the helpers also fills the rings
    constexpr uint32_t helpers = kRefineWarps - 1, filler = kRefineWarps - 1;
    const uint32_t h0 = wid - 1u, h1 = helpers - 1u - h0;
    LaneRing<kRefineRing> fill;
    meet();
    if (wid == filler) fill.init(ring, P.ubuf, sh.range[0][lane], sh.range[1][lane]);
    for (uint32_t round = 0;; ++round) {
        const uint32_t b = round & 1u;
        if (!sh.more[b]) break;
        // ---- the helpers: the lane's finished blocks one after the other from the first helper on, lists from the last one on
        const uint32_t lists = sh.list_count[b][lane], list0 = sh.list_first[b][lane], sides = sh.side_count[b][lane], side0 = sh.side_first[b][lane];
        uint64_t h = 0;                                    // (requested before the side data, used behind it)
        if (wid == filler) fill.request(sh.keep[b][lane]);
        if (h1 < lists) h = refine_masks(sh, lane, list0 + h1);
#pragma unroll 1
        for (uint32_t i = h0; i < sides; i += helpers) refine_side(sh, lane, side0 + i, Ss);
#pragma unroll 1
        for (uint32_t i = h1; i < lists; i += helpers) {
            refine_list(sh, lane, refine_slot(list0 + i), h, band, Se);
            if (i + helpers < lists) h = refine_masks(sh, lane, list0 + i + helpers);
        }
        if (wid == filler) { fill.put(); sh.filled[b][lane] = fill.wr; }
        meet();
    }
}

}  // namespace pcr
