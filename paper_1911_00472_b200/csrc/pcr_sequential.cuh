// Sequential (baseline) scans with restart intervals: one interleaved scan carries, block after block, the DC difference
// and then the AC coefficients up to an end-of-block symbol.
//
// An interval is one chain of symbols, but only two things lie on it: where the next code begins and which table it is
// looked up in.  One CTA per work item (32 restart intervals of one image).  Warp 0 follows the chains, a lane an interval, for
// at most kSeqSteps symbols a round, and leaves behind where every block begins.  Meanwhile the other warps decode the blocks that
// the round before finished: warp 1 their DC differences, a lane an interval, block after block (the predictors run along
// it); the rest their AC coefficients, a thread a block, which go where the progressive first passes put them.
// At the end of a round the CTA meets once.  Every thread works for its own lane's interval, so that shared-memory columns never
// collide.
//
// Bound by warp 0's step: a window, a table entry, and where both lead next, 125 cycles a symbol (a lane that did everything
// itself took 600), then by the warps of four CTAs an SM sharing its schedulers.  1024 ImageNet-shaped images, one stage after the
// other, 742 -> 391 us, 64 such images 713 -> 137 us.  The warps that write count for most of those schedulers' slots: with what a
// symbol needs only in damaged streams or at block ends moved behind the block, and magnitudes by a funnel shift, decode of 1024
// ImageNet-shaped images 688 -> 645 us, of 1024 CelebA-shaped 447 -> 407.  Launches of many images with few intervals keep a lane an
// interval (at the end of the file).
// (Before those two: a step with a predicate for every case 180 cycles; both possible tables looked up and one entry chosen
// afterwards, 64 images 177 -> 189 us; 6 or 12 warps a CTA 183, 181 us, and 1024 images 437 -> 467, 460; rounds of 48 symbols 184,
// of 96 equal.)
#pragma once
#include <cuda_runtime.h>
#include <stddef.h>
#include <stdint.h>

#include "pcr_entropy.cuh"
#include "pcr_types.h"

namespace pcr {

constexpr int kSeqWarps = 8;
constexpr uint32_t kSeqRing = 128;            // words of the stream per lane.  A block takes at most 62 (64 symbols of at most 31
                                              // bits), and its first word is held until it has been written
constexpr uint32_t kSeqSlots = 64;            // blocks of an interval whose beginnings are held
constexpr int kSeqSteps = 64;                 // symbols a round (a block has two at least)
// Blocks a round finishes at most: while warp 0 stores where those behind block m begin, the others read where those of the round
// before began, so the beginnings from m - kSeqRoundBlocks to m + kSeqRoundBlocks are in use at once.
constexpr uint32_t kSeqRoundBlocks = 31;
static_assert(2 * kSeqRoundBlocks + 1 <= kSeqSlots, "a slot is used again while it is read");

struct SeqShared {
    ScanTab tabs[4];                          // DC, DC, AC, AC
    uint32_t ring[(kSeqRing + 2) * 32];       // see LaneRing
    uint32_t start[kSeqSlots][32];            // where a block begins (bit position)
    uint4 head[kSeqWarps - 2][32];            // a block's positions 0..7 while a thread collects them
    uint4 next[8];                            // per block of the MCU: its AC table, the following block's DC table, where that block's entry
                                              // of this array is, the block's own DC table
    uint64_t vals[32];                        // of the lane's interval: where the values of what begins at its position 0 go
    uint32_t mcu0[32];                        // ... its first MCU
    uint32_t range[2][32];                    // ... its bytes
    // by parity of the round: the finished blocks, the first bit that is still read, and how far the ring is filled
    uint32_t first[2][32], count[2][32], more[2], keep[2][32], filled[2][32];
};

template <bool kRoi>
__global__ void __launch_bounds__(32 * kSeqWarps, 4) sequential_kernel(Params P, uint32_t item_begin) {
    __shared__ SeqShared sh;
    const uint32_t tid = threadIdx.x, wid = tid >> 5, lane = tid & 31u;
    const unsigned full = 0xffffffffu;
    const Item item = P.items[item_begin + blockIdx.x];
    const ScanDesc sd = load_entry(P.scans + item.si);
    const int img = (int)(item.si % (uint32_t)P.N);
    const ScanAux ax = load_entry(P.saux + item.si / (uint32_t)P.N);
    const ImgDesc im = load_entry(P.imgs + img);
    const uint32_t mcu_w = im.mx, total = im.mx * im.my;
    const uint32_t hs = (uint32_t)P.hs, vs = (uint32_t)P.vs, bw0 = hs * mcu_w;
    const uint32_t ny = hs * vs, bpm = P.nc == 3 ? ny + 2u : 1u;      // blocks per MCU (a lone component: one block, no padding)
    const uint32_t tabs = (uint32_t)__cvta_generic_to_shared(sh.tabs);

    // what warp 0 keeps of its lane's interval
    uint32_t n = 0, bstart = 0, bend = 0;                     // blocks, bytes
    bool bad = false;
    if (wid == 0) {
        bool done = lane >= item.count;
        uint32_t seg = item.seg0 + lane;
        if (seg >= sd.nseg) { done = true; seg = 0; }
        const uint32_t m0 = sd.ri ? seg * sd.ri : 0, m1 = sd.ri ? min(m0 + sd.ri, total) : total;
        if (m0 >= m1) done = true;
        if (kRoi && !done) {
            const CropRect rc = P.roi[img];
            const uint32_t mh = 8u * vs;                               // pixel rows of an MCU row
            const uint32_t lo = mh * (rc.y0 / mh), hi = mh * ((rc.y0 + rc.h + mh - 1u) / mh);
            const uint32_t r0 = m0 / mcu_w, r1 = (m1 - 1u) / mcu_w;
            if ((r1 + 1u) * mh <= lo || r0 * mh >= hi) done = true;
        }
        const uint32_t* segtab = P.seg_start + sd.seg_base;
        bstart = segtab[seg]; bend = segtab[seg + 1] - 2u;
        if (!done && (bstart < sd.data_off || bend > sd.data_end || bend < bstart)) { bad = true; done = true; }   // a missing marker left a hole
        if (done) { bstart = sd.data_off; bend = sd.data_off; }
        n = done ? 0u : (m1 - m0) * bpm;
        sh.range[0][lane] = bstart; sh.range[1][lane] = bend; sh.keep[0][lane] = 8u * (bstart & 15u);
        sh.mcu0[lane] = m0;
        sh.vals[lane] = reinterpret_cast<uint64_t>(P.vals + 64ull * (bstart >> 4));
        sh.start[0][lane] = 8u * (bstart & 15u);
        sh.count[0][lane] = 0; sh.first[0][lane] = 0;
        const bool any = __any_sync(full, n != 0);
        if (lane == 0) sh.more[0] = any;
    } else {
        const uint4* a = reinterpret_cast<const uint4*>(P.tabs + ax.tab0 + 4u * (uint32_t)img);
        for (uint32_t i = tid - 32u; i < 4u * sizeof(ScanTab) / 16u; i += 32u * (kSeqWarps - 1)) sts128(tabs + 16u * i, __ldg(a + i));
        if (wid == 1 && lane < bpm) {
            auto dc_of = [&](uint32_t j) { return tabs + ((sd.slots >> (2u * (j < ny ? 0u : j - ny + 1u))) & 1u) * (uint32_t)sizeof(ScanTab); };
            const uint32_t c = lane < ny ? 0u : lane - ny + 1u;
            const uint32_t after = lane + 1u == bpm ? 0u : lane + 1u;
            sh.next[lane] = make_uint4(tabs + (2u + ((sd.slots_ac >> (2u * c)) & 1u)) * (uint32_t)sizeof(ScanTab), dc_of(after),
                                       (uint32_t)__cvta_generic_to_shared(sh.next + after), dc_of(lane));
        }
    }
    RingWords<kSeqRing> W;
    W.col = (uint32_t)__cvta_generic_to_shared(sh.ring) + 4u * lane;
    __syncthreads();
    if (wid == 0) {
        // warp 0: blocks finished, blocks handed on, position in the block, entry of the block's place in the MCU
        uint32_t m = 0, handed = 0, k = 0, place = (uint32_t)__cvta_generic_to_shared(sh.next);
        uint32_t pos = 8u * (bstart & 15u);                       // next bit of the lane's chain; the first one behind its interval
        const uint32_t limit = pos + 8u * (bend - bstart);
        uint32_t keep = pos;                                      // first bit of what is handed on next
        uint32_t idle = 0, trace = 0;                             // rounds in which nothing moved on
        bool done = n == 0;
        for (uint32_t round = 0;; ++round) {
            const uint32_t b = round & 1u, nb = b ^ 1u;
            if (!sh.more[b]) break;                           // whole CTA
            // ---- the chains
            const uint32_t filled = round ? sh.filled[nb][lane] : 0u;
            uint32_t stop = done ? 0u : min(32u * (filled - min(filled, 3u)), limit + 1u);
            const uint32_t start = (uint32_t)__cvta_generic_to_shared(sh.start) + 4u * lane, m_end = min(32u * n, 32u * (m + kSeqRoundBlocks));
            uint4 of = lds128(place);                          // see SeqShared::next
            W.load(pos);
            uint32_t tab = k ? of.x : of.w, win = W.window(pos), raw = tab_entry(tab, win), m32 = 32u * m;
            // A step is one straight line that every lane walks.  An entry of zero moves nothing on, so lanes that have arrived
            // somewhere and those that stand at a code longer than the table's index just wait.  The chain: win -> e -> win, and
            // e -> table.  (A coefficient behind the block's end is found where the block is written.)
#pragma unroll 1
            for (int s = 0; s < kSeqSteps; s += 8) {
#pragma unroll 4
                for (int q = 0; q < 8; ++q) {
                    const uint32_t e = pos < stop ? raw : 0u, behind = W.behind(pos), d = e & 31u;
                    k += e >> 9;                               // (an end of block goes beyond 63)
                    const bool end = k > 63u;
                    tab = e ? (end ? of.y : of.x) : tab;
                    win = __funnelshift_l(behind, win, d);
                    raw = tab_entry(tab, win);
                    pos += d;
                    W.load_behind(pos);
                    k = end ? 0u : k;
                    place = end ? of.z : place;
                    of = lds128(place);
                    m32 += end ? 32u : 0u;
                    sts32_if(end, start + 4u * (m32 & (32u * kSeqSlots - 1u)), pos);
                    stop = m32 >= m_end ? 0u : stop;
                }
                if (raw == 0 && pos < stop) {                  // (taken by the next step)
                    raw = long_code(tab, win, k ? kTabAcSeq : kTabDcSeq);
                    if (raw == 0) { bad = true; stop = 0; }    // no such symbol: the lane ends here
                }
                if (!__any_sync(full, pos < stop)) break;
            }
            m = m32 >> 5;
            bad = bad || (!done && pos > limit);
            // ---- what the round left: blocks handed .. m - 1 are finished
            done = done || bad || m >= n;
            sh.first[nb][lane] = handed; sh.count[nb][lane] = m - handed;
            // (every round in which a lane has work left moves something on; should none do so for some rounds, the lanes give up)
            const uint32_t moved = pos + filled + m + handed + keep;
            idle = __any_sync(full, moved != trace) ? 0u : idle + 1u;
            trace = moved;
            if (idle == 8u && !done) bad = done = true;
            const bool more = __any_sync(full, !done || m != handed);
            if (lane == 0) sh.more[nb] = more;
            handed = m;
            sh.keep[nb][lane] = keep;
            keep = sh.start[m & (kSeqSlots - 1u)][lane];
            meet();
        }
        if (bad) atomicMin(&P.status[img], kErrCorrupt);
        return;
    }
    int16_t* const dcp = P.dc + im.blk_base;
    int16_t* const headp = P.head + im.blk_base * 8;
    uint64_t* const auxp = P.aux + ax.base + im.blk_base * 2;
    // block number (in the image) and place in the MCU of block j of the lane's interval
    auto locate = [&](uint32_t j, uint32_t& place) {
        const uint32_t q = j / bpm, m = sh.mcu0[lane] + q;
        place = j - q * bpm;
        if (place >= ny) return (place - ny) * total + ny * total + m;
        const uint32_t row = m / mcu_w, col = m - row * mcu_w;
        return (row * vs + (place >> (hs - 1u))) * bw0 + hs * col + (place & (hs - 1u));
    };
    if (wid == 1) {
        LaneRing<kSeqRing> fill;
        fill.init(W.col, P.ubuf, sh.range[0][lane], sh.range[1][lane]);
        int pred0 = 0, pred1 = 0, pred2 = 0;                  // the predictors
        for (uint32_t round = 0;; ++round) {
            const uint32_t b = round & 1u;
            if (!sh.more[b]) break;
            // ---- the rings, and DC differences
            fill.request(sh.keep[b][lane]);
            const uint32_t count = sh.count[b][lane], first = sh.first[b][lane];
            for (uint32_t i = 0; i < count; ++i) {
                uint32_t place_i;
                const uint32_t blk = locate(first + i, place_i), at = sh.start[(first + i) & (kSeqSlots - 1u)][lane], t = sh.next[place_i].w;
                W.load(at);
                const uint32_t w = W.window(at);
                uint32_t x = tab_entry(t, w);
                if (x == 0) x = long_code(t, w, kTabDcSeq);       // (there is one: the chain has passed it)
                const int d = magnitude(w, x & 31u, (x >> 5) & 15u);
                const int v = d + (place_i < ny ? pred0 : (place_i == ny ? pred1 : pred2));
                if (place_i < ny) pred0 = v; else if (place_i == ny) pred1 = v; else pred2 = v;
                dcp[blk] = (int16_t)v;
            }
            fill.put();
            sh.filled[b][lane] = fill.wr;
            meet();
        }
        return;
    }
    for (uint32_t round = 0;; ++round) {
        const uint32_t b = round & 1u;
        if (!sh.more[b]) break;
        // ---- AC coefficients, the lane's finished blocks one after the other from the first of these warps on
        const uint32_t count = sh.count[b][lane], first = sh.first[b][lane];
        const uint32_t head = (uint32_t)__cvta_generic_to_shared(&sh.head[wid - 2u][lane]);
        for (uint32_t i = wid - 2u; i < count; i += kSeqWarps - 2) {
            uint32_t place_i;
            const uint32_t blk = locate(first + i, place_i), t = sh.next[place_i].x;
            uint32_t at = sh.start[(first + i) & (kSeqSlots - 1u)][lane];
            // (the values of what begins at a bit go to half that bit's number on: a coefficient takes two bits at least)
            int16_t* const vb = reinterpret_cast<int16_t*>(sh.vals[lane]) + ((at + 1u) >> 1);
            int16_t* vp = vb;
            W.load(at);
            uint32_t w = W.window(at), x = tab_entry(sh.next[place_i].w, w);
            if (x == 0) x = long_code(sh.next[place_i].w, w, kTabDcSeq);
            sts128(head, make_uint4(0, 0, 0, 0));
            uint32_t p = 1, M0 = 0, M1 = 0;                // position, mask of those from 8 on
            w = __funnelshift_l(W.behind(at), w, x & 31u);
            at += x & 31u;
            W.load(at);
            x = tab_entry(t, w);
#pragma unroll 1
            for (;;) {                                     // (the next symbol's entry is requested before this one is used)
                if (x == 0) { x = long_code(t, w, kTabAcSeq); if (x == 0) break; }
                const uint32_t skip = x & 31u, sz = (x >> 5) & 15u, w1 = __funnelshift_l(W.behind(at), w, skip), x1 = tab_entry(t, w1);
                at += skip;
                W.load(at);
                p += x >> 9;                                   // (behind the coefficient; an end of block: beyond every position)
                const int v = magnitude(w, skip, sz);
                const bool far = sz && p > 8u;
                sts16_if(sz && !far, head + 2u * p - 2u, (uint32_t)v);
                // (a coefficient behind the block has bits of its own to be stored at, and no place in the masks)
                if (far) *vp = (int16_t)v;
                vp += far ? 1 : 0;
                M0 |= shl0(far ? 1u : 0u, p - 1u); M1 |= shl0(far ? 1u : 0u, p - 33u);
                if (p > 63u) { bad = bad || (sz && p > 64u); break; }
                w = w1; x = x1;
            }
            const uint4 low = lds128(head);                    // (a coefficient is never 0)
            if (low.x | low.y | low.z | low.w) *reinterpret_cast<uint4*>(headp + 8ull * blk) = low;
            if (M0 | M1) *reinterpret_cast<uint4*>(auxp + 2ull * blk) = value_record(M0, M1, vb);
        }
        meet();
    }
    if (bad) atomicMin(&P.status[img], kErrCorrupt);
}

// ---------------------------------------------------------------------------------------
// The same, one lane per restart interval, for launches of many items (see sequential_in_ctas): a warp an item instead of eight, 18
// items an SM instead of four.  Lanes stand at different kinds of symbol in every step, so a block's first symbol goes through the same
// instructions as the others (its value is the difference), stores are predicated, and what changes from block to block comes
// from a small table in shared memory.  Bound by the length of a lane's chain, 600 cycles a symbol: decode of 3072 CelebA-shaped images
// 980 us, with the kernel above 1118; of 1024 480 and 411.
// ---------------------------------------------------------------------------------------
constexpr int kSeqLaneWarps = 2;
constexpr uint32_t kSeqLaneRing = 4 * sizeof(ScanTab), kSeqLanePlaces = kSeqLaneRing + (kRingWords + 2) * 128, kSeqLanePreds = kSeqLanePlaces + 8 * 16;
constexpr uint32_t kSeqLaneBytes = kSeqLanePreds + 3 * 128;

template <bool kRoi>
__global__ void __launch_bounds__(32 * kSeqLaneWarps) sequential_lane_kernel(Params P, uint32_t item_begin, uint32_t item_count) {
    __shared__ __align__(16) uint8_t s_seq[kSeqLaneWarps * kSeqLaneBytes];
    const int wid = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const uint32_t it = blockIdx.x * kSeqLaneWarps + wid;
    if (it >= item_count) return;                             // whole warp
    const Item item = P.items[item_begin + it];
    const ScanDesc sd = load_entry(P.scans + item.si);
    const int img = (int)(item.si % (uint32_t)P.N);
    const ScanAux ax = load_entry(P.saux + item.si / (uint32_t)P.N);
    bool done = (uint32_t)lane >= item.count;
    uint32_t seg = item.seg0 + lane;
    if (seg >= sd.nseg) { done = true; seg = 0; }
    const ImgDesc im = load_entry(P.imgs + img);
    const uint32_t mcu_w = im.mx, total = im.mx * im.my;
    const uint32_t m0 = sd.ri ? seg * sd.ri : 0;
    const uint32_t m1 = sd.ri ? min(m0 + sd.ri, total) : total;
    const unsigned full = 0xffffffffu;
    if (kRoi) {
        if (!done && m1 > m0) {
            const CropRect rc = P.roi[img];
            const uint32_t mh = 8u * (uint32_t)P.vs;                       // pixel rows of an MCU row
            const uint32_t lo = mh * (rc.y0 / mh), hi = mh * ((rc.y0 + rc.h + mh - 1u) / mh);
            const uint32_t r0 = m0 / mcu_w, r1 = (m1 - 1u) / mcu_w;
            if ((r1 + 1u) * mh <= lo || r0 * mh >= hi) done = true;
        }
        if (__all_sync(full, done)) return;
    }
    const uint32_t mem = (uint32_t)__cvta_generic_to_shared(s_seq) + (uint32_t)wid * kSeqLaneBytes;
    const uint32_t hs = (uint32_t)P.hs, vs = (uint32_t)P.vs, bw0 = hs * mcu_w;
    const uint32_t ny = hs * vs, bpm = P.nc == 3 ? ny + 2u : 1u;      // blocks per MCU (a lone component: one block, no padding)
    {
        const uint4* a = reinterpret_cast<const uint4*>(P.tabs + ax.tab0 + 4u * (uint32_t)img);
        for (int i = lane; i < (int)(4 * sizeof(ScanTab) / 16); i += 32) sts128(mem + 16 * i, __ldg(a + i));
        // per block of the MCU: its two tables (shared addresses), where its predictor lies, its block number
        // relative to the MCU's first luminance block or to the MCU's chroma place (bit 31)
        if ((uint32_t)lane < bpm) {
            const uint32_t j = (uint32_t)lane, c = j < ny ? 0u : j - ny + 1u;
            const uint32_t tdc = mem + ((sd.slots >> (2u * c)) & 1u) * (uint32_t)sizeof(ScanTab);
            const uint32_t tac = mem + (2u + ((sd.slots_ac >> (2u * c)) & 1u)) * (uint32_t)sizeof(ScanTab);
            const uint32_t off = c ? (ny * total + (c - 1u) * total) | 0x80000000u : (j >> (hs - 1u)) * bw0 + (j & (hs - 1u));
            sts128(mem + kSeqLanePlaces + 16u * j, make_uint4(tdc, tac, mem + kSeqLanePreds + 128u * c, off));
        }
#pragma unroll
        for (int c = 0; c < 3; ++c) sts32(mem + kSeqLanePreds + 128u * c + 4u * lane, 0u);
    }
    const uint32_t* segtab = P.seg_start + sd.seg_base;
    uint32_t bstart = segtab[seg];
    uint32_t bend = segtab[seg + 1] - 2;
    bool bad = false;
    if (!done && (bstart < sd.data_off || bend > sd.data_end || bend < bstart)) { bad = true; done = true; }
    if (done) { bstart = sd.data_off; bend = sd.data_off; }
    LaneBits br;
    br.init(mem + kSeqLaneRing + 4u * lane, P.ubuf, bstart, bend);
    if (m0 >= m1) done = true;

    uint32_t m = m0, wrap_m = (m0 / mcu_w + 1u) * mcu_w;       // MCU, the first one of the next row
    uint32_t my = (m0 / mcu_w) * vs * bw0 + hs * (m0 % mcu_w); // block number of the MCU's first luminance block (its chroma place is m)
    const uint32_t my_wrap = (vs - 1u) * bw0;                  // what a new row adds beside hs per MCU
    uint32_t place = mem + kSeqLanePlaces;                     // of the current block in the table
    const uint32_t place_end = place + 16u * bpm;
    uint32_t k = 0, M0 = 0, M1 = 0;                            // position (0: the block's DC symbol comes next), mask
    int16_t* vp = P.vals + 4ull * bstart;                      // next value
    int16_t* vb = vp;                                          // the block's first one
    int16_t* dcp = P.dc + im.blk_base;
    int16_t* headp = P.head + im.blk_base * 8;
    uint64_t* auxp = P.aux + ax.base + im.blk_base * 2;
    pin(dcp); pin(headp); pin(auxp);
    uint32_t tdc = 0, tac = 0, pred = 0, blk = 0;
    auto take = [&]() {
        const uint4 v = lds128(place);
        tdc = v.x; tac = v.y; pred = v.z + 4u * lane;
        blk = (v.w & 0x7FFFFFFFu) + ((v.w >> 31) ? m : my);
    };
    bool fresh = true;
    for (;;) {
        br.topup(!done);
        __syncwarp(full);
        if (__all_sync(full, done)) break;
        if (fresh) { take(); fresh = false; }
        uint32_t stop = done ? 0u : min(br.ring_stop(2), br.limit + 1u);
#pragma unroll 1
        for (int t = 0; t < kDecodeSteps; ++t) {
            if (br.pos < stop) {
                const uint32_t win = br.window(br.pos);
                const bool is_dc = k == 0;
                const uint32_t tab = is_dc ? tdc : tac;
                uint32_t e = tab_entry(tab, win);
                if (e == 0) {
                    e = long_code(tab, win, is_dc ? kTabDcSeq : kTabAcSeq);
                    if (e == 0) { bad = true; stop = 0; }
                }
                const uint32_t skip = e & 31u, sz = (e >> 5) & 15u;
                br.pos += skip;
                k += e >> 9;                                               // behind the coefficient (an end of block: beyond every position)
                const uint32_t at = k - 1u;
                int v = magnitude(win, skip, sz);
                if (is_dc) { v += (int)lds32(pred); sts32(pred, (uint32_t)v); }
                const bool far = sz && k > 8u;
                if (is_dc) dcp[blk] = (int16_t)v;                          // (stored even if there was no such symbol: the image is corrupt then)
                if (sz && !far && !is_dc) headp[8u * (uint64_t)blk + at] = (int16_t)v;
                if (far) *vp = (int16_t)v;
                vp += far ? 1 : 0;
                M0 |= shl0(far ? 1u : 0u, at); M1 |= shl0(far ? 1u : 0u, at - 32u);
                if (k > 63u) {                                             // block finished
                    if (sz && k > 64u) { bad = true; stop = 0; }           // (a coefficient behind the block: stored at bits of its own, not in the masks)
                    if (M0 | M1) *reinterpret_cast<uint4*>(auxp + 2ull * blk) = value_record(M0, M1, vb);
                    k = 0; M0 = 0; M1 = 0; vb = vp;
                    place += 16u;
                    if (place == place_end) {
                        place = mem + kSeqLanePlaces;
                        ++m; my += hs;
                        if (m == wrap_m) { wrap_m += mcu_w; my += my_wrap; }
                        if (m >= m1) stop = 0;
                    }
                    take();
                }
            }
        }
        __syncwarp(full);
        bad = bad || br.pos > br.limit;
        done = done || bad || m >= m1;
    }
    if (bad) atomicMin(&P.status[img], kErrCorrupt);
}

}  // namespace pcr
