// Entropy stage for scans that are ONE long restart interval (records written without restart
// markers: one entropy-coded segment per image and scan), and DC refinement scans in waves without AC refinements.
//
// A Huffman stream is a serial chain, so a whole scan on one lane takes tens of thousands of
// dependent steps.  These kernels shorten or remove that chain:
//
//  * dc_refine_kernel: a DC refinement scan carries exactly one raw bit per block, so after
//    unstuffing bit j of a restart interval is block j of the interval in scan order: one thread
//    per MCU, no chain at all (dc_refine_image).  Where the wave has AC refinements in interval warps, extra blocks
//    of their launch do it instead (see entropy_kernel).
//  * first_pass_long_kernel: DC and AC first passes.  One small CTA per (scan, image); the segment is
//    cut into one subsequence of equal bit length per thread.  A thread that starts in the middle of the
//    stream does not know where a code begins nor which coefficient (or which block of the MCU) it is
//    at; it guesses (DC scans some bits ahead of their subsequence), and because Huffman streams
//    re-synchronise, its state at the end of its subsequence is often right.  The threads then hand
//    their end states on: a thread whose predecessor ended in a state other than the one it started
//    from reads again from there, until it is at one of its earlier readings' marked states, where the rest
//    of that reading holds; the rounds stop when nothing changes (thread 0 starts at the true beginning,
//    so after round r threads 0..r are exact).  A counting pass and a prefix sum of the blocks each
//    thread finished (and of the DC differences per component) give every thread its first block
//    and its predictors, and a last pass decodes once more and writes.
//  * sequential_long_kernel: the same scheme for the one scan of a baseline JPEG.
//  * ac_refine_group_kernel: an AC refinement cannot be entered in the middle (how many correction
//    bits follow a symbol depends on which coefficients of the block are already non-zero, i.e. on
//    the block number).  A scan is one chain: one thread follows it, two dependent loads from shared memory a
//    symbol; a helper warp decodes a symbol at EVERY bit position ahead of it, prepares the masks and the
//    lists of zero positions of the next blocks, and decodes the finished blocks once more, one per lane, into
//    side data.  All chains of a record run in one persistent launch that deals them to the SMs' schedulers
//    evenly; the refinements of one component run behind one another, block by block.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

#include "pcr_entropy.cuh"
#include "pcr_types.h"

namespace pcr {

// ---------------------------------------------------------------------------------------
// DC refinement where no launch of interval warps can carry it (see entropy_kernel).  grid = (chunks of MCUs, images of the run).
// ---------------------------------------------------------------------------------------
__global__ void __launch_bounds__(256) dc_refine_kernel(Params P, int s, uint32_t pos0) {
    dc_refine_image(P, s, (int)P.order[pos0 + blockIdx.y], blockIdx.x * 256u + threadIdx.x, gridDim.x * 256u);
}

// ---------------------------------------------------------------------------------------
// First passes and sequential scans that are one restart interval.  The interval is cut into subsequences of equal bit
// length, one per thread of a small CTA.  A position's state is the bit position and a number `st`: DC scans: the
// block's place in its MCU; AC scans: the next zigzag position; sequential scans: 64 times the place plus the next
// zigzag position (0: the block's DC symbol comes next).
//
// Search: every thread follows its subsequence from a guessed state; threads whose predecessor ended in another state than
// they began with follow theirs again, until nothing changes.  A thread leaves its state behind at eight places of
// its subsequence; a later reading that comes by in the same state has met the earlier one and stops there.  (Without
// that every round cost a whole subsequence, and interleaved DC scans take 5 to 9 rounds.)  Count: once more, the blocks
// finished and the DC differences summed; prefix sums give every thread its first block and predictors.  Write: once more.
//
// A step is a window (two loads that hit the L1 cache), a table entry that already holds what the step needs, and an
// addition; bound by that chain, about 110 cycles a symbol (430 with a 64-bit buffer, a canonical table and selects).
// ---------------------------------------------------------------------------------------
// w: the stream's words, in shared memory where they fit, else where they are (the loads are generic ones).
__device__ __forceinline__ uint32_t long_window(const uint32_t* w, uint32_t pos) {
    const uint32_t i = pos >> 5;
    return __funnelshift_l(w[i + 1], w[i], pos);                           // (shift taken mod 32)
}
__device__ __forceinline__ uint32_t long_entry(uint32_t tab, uint32_t win, int kind) {
    const uint32_t e = lds16(tab + ((win >> (32 - kTabBits)) << 1));
    return e ? e : long_code(tab, win, kind);
}
// A position that a writing pass walks along: its 32 bits and the words behind them, requested ahead of their use.
struct LongWalk {
    const uint32_t* base;
    uint32_t p, win, w1, w2;
    __device__ __forceinline__ void load() { const uint32_t* w = base + (p >> 5); w1 = w[1]; w2 = w[2]; }
    __device__ __forceinline__ LongWalk(const uint32_t* b, uint32_t at) : base(b), p(at) { win = __funnelshift_l(b[(at >> 5) + 1], b[at >> 5], at); load(); }
    __device__ __forceinline__ uint32_t behind(uint32_t skip) const { return __funnelshift_l(__funnelshift_l(w2, w1, p), win, skip); }    // the 32 bits `skip` bits on
    __device__ __forceinline__ void go(uint32_t skip, uint32_t next) { win = next; p += skip; load(); }
};
// number of blocks that an end of band covers
__device__ __forceinline__ uint32_t eob_blocks(uint32_t e, uint32_t win) {
    const uint32_t r = (e >> 9) & 15u;
    return (1u << r) + shr0(shl0(win, (e & 31u) - r), 32u - r);
}

// The symbol at a position (its entry as in ScanTab, 0 = none), and what it does to the state: true if a block ends.
struct DcSteps {
    const uint32_t* base;
    uint32_t tabs;                 // shared address of two tables
    uint32_t tbits, bpm;           // bit j: the table of the MCU's block j; blocks per MCU
    __device__ __forceinline__ uint32_t entry(uint32_t pos, uint32_t st) const {
        const uint32_t t = (tbits >> st) & 1u;
        return long_entry(tabs + t * (uint32_t)sizeof(ScanTab), long_window(base, pos), kTabDc);
    }
    __device__ __forceinline__ bool advance(uint32_t, uint32_t& st) const { st = st + 1u == bpm ? 0u : st + 1u; return true; }
};
struct AcSteps {
    const uint32_t* base;
    uint32_t tabs, Ss, Se;
    __device__ __forceinline__ uint32_t entry(uint32_t pos, uint32_t) const {
        return long_entry(tabs, long_window(base, pos), kTabAcFirst);
    }
    __device__ __forceinline__ bool advance(uint32_t e, uint32_t& st) const {
        st += e >> 9;                                                      // (an end of band: beyond every position)
        const bool end = st > Se;
        st = end ? Ss : st;
        return end;
    }
};
struct SeqSteps {
    const uint32_t* base;
    uint32_t tabs, tdc, tac, bpm;  // shared address of the tables DC 0, DC 1, AC 0, AC 1; bit j: which of them block j uses
    __device__ __forceinline__ uint32_t entry(uint32_t pos, uint32_t st) const {
        const uint32_t j = st >> 6;
        const bool dc = (st & 63u) == 0;
        return long_entry(tabs + (dc ? (tdc >> j) & 1u : 2u + ((tac >> j) & 1u)) * (uint32_t)sizeof(ScanTab), long_window(base, pos), dc ? kTabDcSeq : kTabAcSeq);
    }
    __device__ __forceinline__ bool advance(uint32_t e, uint32_t& st) const {
        const uint32_t k = (st & 63u) + ((e >> 9) & 31u), j = st >> 6;
        const bool end = (e & kEntEob) || k > 63u;
        st = end ? (j + 1u == bpm ? 0u : j + 1u) << 6 : (st & ~63u) + k;
        return end;
    }
};

// The symbols that START in [pos, pos_end) from state st.  Every step consumes at least one bit, so the loop ends; an
// undefined code is passed over by one bit (the thread is then reading from a wrong state and only has to arrive
// somewhere).  marks: shared address of this thread's places, one every `every` bits from `begin` on (kPitch bytes apart).
constexpr uint32_t kMarks = 8;
template <class Steps, uint32_t kPitch>
__device__ __forceinline__ void search_span(const Steps& S, uint32_t begin, uint32_t every, uint32_t marks,
                                            uint32_t pos, uint32_t st, uint32_t pos_end, uint32_t& pos_x, uint32_t& st_x) {
    // (from place to place: the lanes of the warp meet there; a loop over the whole subsequence with the comparison inside
    // let them drift apart and ran them one after the other, seven times slower)
    uint32_t stop = begin;
    bool met = pos >= pos_end;             // nothing to read
    const bool idle = met;
#pragma unroll 1
    for (uint32_t i = 0; i < kMarks; ++i) {
        stop += every;                     // (a symbol is at most 31 bits, `every` at least 32: a step passes one place at most)
        const uint32_t bound = met ? 0u : min(stop, pos_end);
        while (pos < bound) {
            const uint32_t e = S.entry(pos, st);
            if (e) S.advance(e, st);
            pos += e ? e & 31u : 1u;
        }
        __syncwarp();
        // (Only places inside the subsequence: every reading passes those or meets an earlier one in front of them, so the keys
        // they hold are the latest reading's throughout, and so is the end state.  A place behind the end of a truncated
        // subsequence is passed by some readings only and would keep an older one's key.)
        if (!met && pos >= stop && stop <= pos_end) {
            const uint32_t key = (pos << 9) + st;                          // (equal keys are equal states: pos stays inside the subsequence)
            met = lds32(marks + i * kPitch) == key;                        // met the reading before: it ends where that one did
            sts32(marks + i * kPitch, key);
        }
        if (__all_sync(0xffffffffu, met || pos >= pos_end)) break;
    }
    if (!met || idle) { pos_x = pos; st_x = st; }
}

// Where the interval of a long scan lies, and this thread's subsequence.
struct LongSpan {
    const uint32_t* base;          // the stream's words
    const uint32_t* origin;        // where they lie in the unstuffed copy
    uint32_t lead, endbit;         // its first bit and the one behind its last, counted from the first word
    uint32_t begin, end, every;
    bool ok;
    // stage: shared memory for `room` words (the caller synchronises behind this)
    // kNarrow, kWords: threads that shorter scans are cut for, and the subsequence's words above which more threads are used
    template <uint32_t kThreads, uint32_t kNarrow, uint32_t kWords>
    __device__ __forceinline__ void init(const Params& P, const ScanDesc& sd, uint32_t tid, uint32_t* stage, uint32_t room) {
        const uint32_t* segtab = P.seg_start + sd.seg_base;
        const uint32_t bstart = segtab[0], bend = segtab[1] - 2u;
        ok = !(bstart < sd.data_off || bend > sd.data_end || bend < bstart);   // (the same for every thread)
        base = origin = reinterpret_cast<const uint32_t*>(P.ubuf) + (bstart >> 2);
        lead = 8u * (bstart & 3u); endbit = ok ? lead + 8u * (bend - bstart) : lead;
        // whole words, at least eight of them: eight places at least 32 bits apart
        // (shorter subsequences mean more rounds: how far a reading takes to fall in does not depend on them)
        const uint32_t all = (endbit + 31u) / 32u, words = max(min(max(8u, (all + kNarrow - 1u) / kNarrow), kWords), (all + kThreads - 1u) / kThreads);
        const uint32_t len = 32u * words;
        every = len / kMarks;
        begin = min(max(tid * len, lead), endbit); end = min((tid + 1u) * len, endbit);
        const uint32_t need = endbit / 32u + 5u;               // (a symbol may begin in the last bit, and the words behind it are looked at)
        if (need <= room) {
            for (uint32_t i = tid; i < need; i += kThreads) stage[i] = __ldg(origin + i);
            base = stage;
        }
    }
};

// Exclusive prefix sum over the CTA's threads in thread order (warp scans, then the warps' totals
// through shared memory); total = the sum over all threads.  Every thread of the CTA calls it.
template <class T>
__device__ __forceinline__ T cta_exclusive_sum(T v, T* s_tmp, int wid, int lane, int warps, T& total) {
    const unsigned full = 0xffffffffu;
    T inc = v;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
        const T o = __shfl_up_sync(full, inc, d);
        if (lane >= d) inc += o;
    }
    __syncthreads();                                           // s_tmp may still be read from the previous call
    if (lane == 31) s_tmp[wid] = inc;
    __syncthreads();
    T before = 0, all = 0;
    for (int w = 0; w < warps; ++w) { const T t = s_tmp[w]; if (w < wid) before += t; all += t; }
    total = all;
    return before + inc - v;
}

// Search of the whole CTA: the true state at the start of every thread's subsequence, in pos and st.
template <class Steps, int kWarps>
__device__ __forceinline__ void search_all(const Steps& S, const LongSpan& L, uint32_t* s_marks, uint32_t* s_pos, uint32_t* s_state, uint32_t st0, uint32_t warm,
                                           uint32_t& pos, uint32_t& st) {
    constexpr uint32_t kThreads = 32 * kWarps;
    const int tid = threadIdx.x, wid = tid >> 5, lane = tid & 31;
    const unsigned full = 0xffffffffu;
#pragma unroll
    for (uint32_t i = 0; i < kMarks; ++i) s_marks[i * kThreads + tid] = 0xFFFFFFFFu;
    const uint32_t marks = (uint32_t)__cvta_generic_to_shared(s_marks + tid);
    // a first guess from `warm` bits in front of the subsequence: most readings have fallen in with the true one by then
    pos = max(L.lead, L.begin - min(L.begin, warm)); st = st0;
    while (__any_sync(full, pos < L.begin)) {
        if (pos < L.begin) {
            const uint32_t e = S.entry(pos, st);
            if (e) S.advance(e, st);
            pos += e ? e & 31u : 1u;
        }
    }
    uint32_t pos_x = pos, st_x = st;
    bool again = true;
    for (uint32_t round = 0; round <= kThreads; ++round) {
        if (__any_sync(full, again)) {
            uint32_t x = pos_x, y = st_x;
            search_span<Steps, 4 * kThreads>(S, L.begin, L.every, marks, pos, st, again ? L.end : 0u, x, y);
            if (again) { pos_x = x; st_x = y; }
        }
        // the state the previous thread ended in (a warp's last lane's through shared memory)
        if (lane == 31) { s_pos[wid] = pos_x; s_state[wid] = st_x; }
        __syncthreads();
        uint32_t ppos = __shfl_up_sync(full, pos_x, 1), pst = __shfl_up_sync(full, st_x, 1);
        if (lane == 0 && wid > 0) { ppos = s_pos[wid - 1]; pst = s_state[wid - 1]; }
        ppos = min(ppos, L.endbit);
        // (behind the interval's end there is nothing to read and nobody to hand a state to: it would wander on a thread a round)
        again = tid > 0 && L.begin < L.end && (ppos != pos || pst != st);
        if (again) { pos = ppos; st = pst; }
        if (!__syncthreads_or(again)) break;
    }
}

// A reading of a DC scan from some state on: blocks and differences per component summed.  An undefined code is passed over by
// one bit.
struct DcReading {
    const DcSteps& S;
    LongWalk w;
    uint32_t st, tab, raw, nb;
    int sum0, sum1, sum2;
    __device__ __forceinline__ uint32_t table(uint32_t place) const { return S.tabs + ((S.tbits >> place) & 1u) * (uint32_t)sizeof(ScanTab); }
    __device__ __forceinline__ DcReading(const DcSteps& s, const uint32_t* base, uint32_t pos, uint32_t place)
        : S(s), w(base, pos), st(place), nb(0), sum0(0), sum1(0), sum2(0) { tab = table(st); raw = tab_entry(tab, w.win); }
    // the symbols that start in front of `end`; j1, j2: the chroma blocks' places
    __device__ __forceinline__ void to(uint32_t end, uint32_t j1, uint32_t j2) {
#pragma unroll 1
        while (w.p < end) {
            const uint32_t e = raw ? raw : long_code(tab, w.win, kTabDc), skip = e ? e & 31u : 1u, win = w.win, next = w.behind(skip);
            const uint32_t at = st;
            st = e ? (st + 1u == S.bpm ? 0u : st + 1u) : st;
            tab = table(st);
            raw = tab_entry(tab, next);
            w.go(skip, next);
            const int d = e ? magnitude(win, skip, e >> 5) : 0;
            sum0 += at < j1 ? d : 0; sum1 += at == j1 ? d : 0; sum2 += at == j2 ? d : 0;
            nb += e ? 1u : 0u;
        }
    }
};

// Interleaved DC scans, wide CTAs.  Bit positions fall in within a few symbols, but a reading can go on for long with the
// wrong place in the MCU (up to 23 rounds of the search above).  So every subsequence is read once from EVERY place, 512 bits ahead of
// it, and one warp follows the true state through the readings.  Where none of them began its subsequence in the true state, that one
// is read once more, and with the first such one the likely cases behind it, all at once: a lone lane took 14 us for each,
// three in an image of 343x562 (DC alone of 16 images of mixed sizes 127 us, by rounds of the search 110, now 95).  On return a thread
// has the start of its subsequence (L.begin, L.end changed to match), its blocks, the number of blocks and the sums of differences in
// front of it.
constexpr uint32_t kDcNone = 0xFFFFFFFFu;
template <uint32_t kThreads> __host__ __device__ constexpr uint32_t dc_words() { return 14 * kThreads + 4; }     // of shared memory at mem
template <uint32_t kThreads>
__device__ __forceinline__ void dc_hypotheses(const DcSteps& S, LongSpan& L, uint32_t* mem, uint32_t j1, uint32_t j2, uint32_t& pos, uint32_t& st,
                                              uint32_t& nb, uint32_t& n, int& pred0, int& pred1, int& pred2, uint32_t& all) {
    const uint32_t tid = threadIdx.x, lane = tid & 31u, H = S.bpm, subs = kThreads / H;
    const unsigned full = 0xffffffffu;
    const uint32_t len = 32u * max(8u, ((L.endbit + 31u) / 32u + subs - 1u) / subs);
    auto begin_of = [&](uint32_t i) { return min(max(i * len, L.lead), L.endbit); };
    auto end_of = [&](uint32_t i) { return min((i + 1u) * len, L.endbit); };
    // by hypothesis and subsequence: the state it begins in (one number: equal ones within a subsequence are equal states), the one
    // it ends in, blocks and sums; behind them the same once more for second readings; in the end, by subsequence, what the caller asks for
    constexpr uint32_t kSet = 7 * kThreads;
    auto store = [&](uint32_t at, const DcReading& R) {
        mem[kThreads + at] = R.w.p; mem[2 * kThreads + at] = R.st; mem[3 * kThreads + at] = R.nb;
        mem[4 * kThreads + at] = (uint32_t)R.sum0; mem[5 * kThreads + at] = (uint32_t)R.sum1; mem[6 * kThreads + at] = (uint32_t)R.sum2;
    };
    const uint32_t h = tid / subs, i = tid - h * subs, b = begin_of(i), e = end_of(i);
    const bool some = h < H && b < e;
    {
        uint32_t k = kDcNone;
        if (some && (i != 0 || h == 0)) {
            const uint32_t from = i == 0 ? L.lead : max(L.lead, b - min(b, 512u));
            DcReading R(S, L.base, from, from == L.lead ? 0u : h);
            R.to(b, j1, j2);
            k = (R.w.p << 3) + R.st;
            R.nb = 0; R.sum0 = R.sum1 = R.sum2 = 0;
            R.to(e, j1, j2);
            store(tid, R);
        }
        mem[tid] = k;
        mem[kSet + tid] = kDcNone;
    }
    // Warp 0 follows the true state from one subsequence to the next, lanes 0..15 looking for it among the first readings, 16..31 among
    // the second ones.  Where it finds none, that subsequence is read once more, and beside it, once, every one behind it from each state that a
    // reading of the one in front of it ended in and that none of its own began in.
    uint32_t p = L.lead, s = 0, blocks = 0, next = 0;          // (warp 0)
    int a0 = 0, a1 = 0, a2 = 0;
    for (bool again = false;; again = true) {
        __syncthreads();
        if (tid < 32u) {
            const uint32_t set = lane < 16u ? 0u : kSet, lh = lane & 15u;
            for (; next < subs; ++next) {
                const uint32_t at = set + lh * subs + next, end = end_of(next);
                const bool live = begin_of(next) < end;
                const unsigned who = __ballot_sync(full, live && lh < H && mem[at] == (p << 3) + s);
                uint32_t q = 0, t = 0, c = 0;
                int d0 = 0, d1 = 0, d2 = 0;
                const uint32_t src = who ? (uint32_t)__ffs((int)who) - 1u : 0u;
                if (who) {
                    if (lane == src) { q = mem[kThreads + at]; t = mem[2 * kThreads + at]; c = mem[3 * kThreads + at]; d0 = (int)mem[4 * kThreads + at]; d1 = (int)mem[5 * kThreads + at]; d2 = (int)mem[6 * kThreads + at]; }
                } else if (live) {
                    if (!again) break;
                    if (lane == 0) {
                        DcReading R(S, L.base, p, s);
                        R.to(end, j1, j2);
                        q = R.w.p; t = R.st; c = R.nb; d0 = R.sum0; d1 = R.sum1; d2 = R.sum2;
                    }
                }
                q = __shfl_sync(full, q, src); t = __shfl_sync(full, t, src); c = __shfl_sync(full, c, src);
                d0 = __shfl_sync(full, d0, src); d1 = __shfl_sync(full, d1, src); d2 = __shfl_sync(full, d2, src);
                __syncwarp(full);
                if (lane == 0) {                               // (no reading of a subsequence passed is looked at again)
                    mem[next] = p; mem[kThreads + next] = s; mem[2 * kThreads + next] = blocks;
                    mem[3 * kThreads + next] = (uint32_t)a0; mem[4 * kThreads + next] = (uint32_t)a1; mem[5 * kThreads + next] = (uint32_t)a2;
                }
                if (live) { p = q; s = t; blocks += c; a0 += d0; a1 += d1; a2 += d2; }
            }
            if (lane == 0) { mem[2 * kSet] = next; mem[2 * kSet + 1] = blocks; mem[2 * kSet + 2] = p; mem[2 * kSet + 3] = s; }
        }
        __syncthreads();
        const uint32_t stop = mem[2 * kSet];
        if (again || stop >= subs) break;
        if (some && (i == stop ? h == 0 : i > stop)) {
            const uint32_t from = i == stop ? mem[2 * kSet + 2] : mem[kThreads + tid - 1u], place = i == stop ? mem[2 * kSet + 3] : mem[2 * kThreads + tid - 1u];
            const uint32_t k = (from << 3) + place;
            bool known = false;
            for (uint32_t j = 0; j < H; ++j) known = known || mem[j * subs + i] == k;
            if (!known) {
                DcReading R(S, L.base, from, place);
                R.to(e, j1, j2);
                store(kSet + tid, R);
                mem[kSet + tid] = k;
            }
        }
    }
    const bool mine = tid < subs;
    L.begin = mine ? begin_of(tid) : L.endbit; L.end = mine ? end_of(tid) : 0u;
    pos = mine ? mem[tid] : L.endbit; st = mine ? mem[kThreads + tid] : 0u; n = mine ? mem[2 * kThreads + tid] : 0u;
    pred0 = mine ? (int)mem[3 * kThreads + tid] : 0; pred1 = mine ? (int)mem[4 * kThreads + tid] : 0; pred2 = mine ? (int)mem[5 * kThreads + tid] : 0;
    all = mem[2 * kSet + 1];
    nb = mine ? (tid + 1u < subs ? mem[2 * kThreads + tid + 1u] : all) - n : 0u;
}

// ---------------------------------------------------------------------------------------
// First passes: one CTA of kWarps warps per listed (scan, image) whose scan is one restart interval.
// Bound by the chain of one subsequence times the rounds until the slowest scan of the record has fallen in: a launch
// waits for that scan; then by the pass that writes.  The stream and the tables are in shared memory because every step of the
// search depends on them.  256 HAM-shaped images at k = 5, decode: 570 us on average over six records when every round read its whole
// subsequence from global memory, 350 us with marks.  Writing passes of straight-line steps and no rounds that only hand a state on
// behind the interval's end (up to 56): 399 and 366 us over three other records.  Four times the warps while most of the machine is
// idle (wide_long_scans), interleaved DC scans then read from every place of the MCU at once (dc_hypotheses; the search took up to 23
// rounds, most of the kernel's time): 345 us of those 366; 64 ImageNet-shaped images 267 -> 156 us, 64 CelebA-shaped 153 -> 100 us.
// ---------------------------------------------------------------------------------------
constexpr int kLongWarps = 2, kLongWideWarps = 8;
// words of a scan that are staged: 8 KB, a 600x450 image's scans have up to 6 (of the luminance 12); 24 KB of a wide CTA
template <int kWarps> __host__ __device__ constexpr uint32_t long_stage() { return kWarps == kLongWarps ? 2048 : 6144; }

// Copies n of the (scan, image)'s tables to shared memory; the CTA's threads together.
__device__ __forceinline__ void load_tabs(uint32_t dst, const ScanTab* src, int n, int tid, int threads) {
    const uint4* a = reinterpret_cast<const uint4*>(src);
    for (int i = tid; i < n * (int)(sizeof(ScanTab) / 16); i += threads) sts128(dst + 16u * i, __ldg(a + i));
}

template <int kWarps>
__global__ void __launch_bounds__(32 * kWarps) first_pass_long_kernel(Params P, const uint32_t* __restrict__ list, uint32_t count) {
    constexpr int kThreads = 32 * kWarps;
    constexpr uint32_t kLongStage = long_stage<kWarps>();
    __shared__ __align__(16) uint8_t s_tabs[2 * sizeof(ScanTab)];
    __shared__ uint32_t s_stage[kLongStage];
    __shared__ uint32_t s_marks[kWarps == kLongWarps ? kMarks * kThreads : dc_words<kThreads>()];
    __shared__ uint32_t s_pos[kWarps], s_state[kWarps], s_u[kWarps];
    __shared__ int s_i[kWarps];
    const int tid = threadIdx.x, wid = tid >> 5, lane = tid & 31;
    const uint32_t it = blockIdx.x;
    if (it >= count) return;                                   // whole CTA
    const uint32_t si = list[it];
    const int s = (int)(si / (uint32_t)P.N), img = (int)(si % (uint32_t)P.N);
    const ScanDesc& sd = P.scans[si];
    const ScanScript sc = P.script[s];
    const ScanAux ax = P.saux[s];
    const Geometry g = make_geometry(P.imgs[img], P);
    const bool dc = sc.Ss == 0, inter = sc.ncomp > 1;
    const uint32_t c0 = (uint32_t)sc.comp[0];
    const uint32_t mcu_w = inter ? g.mx : g.ubw[c0];
    const uint32_t total = mcu_w * (inter ? g.my : g.ubh[c0]);  // MCUs of the scan (one interval)
    const uint32_t tabs = (uint32_t)__cvta_generic_to_shared(s_tabs);
    const bool second = dc && sd.tab_off[1];
    LongSpan L;
    L.init<kThreads, 32 * kLongWarps, 16>(P, sd, (uint32_t)tid, s_stage, kLongStage);
    load_tabs(tabs, P.tabs + ax.tab0 + (uint32_t)img * (uint32_t)ax.ntab, second ? 2 : 1, tid, kThreads);
    __syncthreads();
    if (!L.ok) {
        if (tid == 0) atomicMin(&P.status[img], kErrCorrupt);
        return;
    }
    bool bad = false;
    uint32_t pos, st, all, nb = 0;
    if (dc) {
        const uint32_t ny = (uint32_t)(P.hs * P.vs), bpm = inter ? ny + 2u : 1u, hs = (uint32_t)P.hs;
        DcSteps S;
        S.base = L.base; S.tabs = tabs; S.bpm = bpm; S.tbits = 0;
        for (uint32_t j = 0; j < bpm; ++j) S.tbits |= ((sd.slots >> (2u * (inter && j >= ny ? j - ny + 1u : 0u))) & 1u) << j;
        const uint32_t j1 = inter ? ny : 6u, j2 = inter ? ny + 1u : 6u;          // the chroma blocks' places
        uint32_t n;
        int pred0, pred1, pred2;
        if (kWarps != kLongWarps && bpm > 1u) {
            dc_hypotheses<32 * kWarps>(S, L, s_marks, j1, j2, pos, st, nb, n, pred0, pred1, pred2, all);
        } else {
            search_all<DcSteps, kWarps>(S, L, s_marks, s_pos, s_state, 0u, 512u, pos, st);
            int sum0 = 0, sum1 = 0, sum2 = 0, t;
            DcReading R(S, L.base, pos, st);
            R.to(L.end, j1, j2);
            nb = R.nb; sum0 = R.sum0; sum1 = R.sum1; sum2 = R.sum2;
            n = cta_exclusive_sum(nb, s_u, wid, lane, kWarps, all);
            pred0 = cta_exclusive_sum(sum0, s_i, wid, lane, kWarps, t);
            pred1 = cta_exclusive_sum(sum1, s_i, wid, lane, kWarps, t);
            pred2 = cta_exclusive_sum(sum2, s_i, wid, lane, kWarps, t);
        }
        const uint32_t n1 = total * bpm;
        n = min(n, n1);
        // the place inside the MCU follows from the block number (equal to the handed-on state unless
        // the stream is damaged; taking it from the block number keeps every store inside the image)
        if (nb && st != n % bpm) bad = true;
        uint32_t j = n % bpm, m = n / bpm, mcol = m % mcu_w;
        uint32_t yb = inter ? (uint32_t)P.vs * (m / mcu_w) * g.bw[0] + hs * mcol : (m / mcu_w) * g.bw[c0] + mcol;
        int16_t* const yp = P.dc + g.coff[inter ? 0 : c0];
        int16_t* const cp = P.dc + g.coff[1];
        const uint32_t c_step = g.mx * g.my, step = inter ? hs : 1u;
        const uint32_t wrap = (inter ? (uint32_t)P.vs * g.bw[0] : g.bw[c0]) - step * mcu_w;
        for (uint32_t p = pos; p < L.end && n < n1; ++n) {
            const uint32_t win = long_window(L.base, p), e = S.entry(p, j);
            if (!e) { bad = true; break; }
            const int d = magnitude(win, e & 31u, e >> 5);
            p += e & 31u;
            if (j < j1) {
                pred0 += d;
                yp[yb + (inter ? (j >> (hs - 1u)) * g.bw[0] + (j & (hs - 1u)) : 0u)] = (int16_t)(pred0 << sc.Al);
            } else {
                const bool first = j == j1;
                const int v = d + (first ? pred1 : pred2);
                if (first) pred1 = v; else pred2 = v;
                cp[m + (first ? 0u : c_step)] = (int16_t)(v << sc.Al);
            }
            if (++j == bpm) {
                j = 0; ++m;
                yb += step;
                if (++mcol == mcu_w) { mcol = 0; yb += wrap; }
            }
        }
        if (all < n1) bad = true;                              // the stream ends before the last block
    } else {
        AcSteps S;
        S.base = L.base; S.tabs = tabs; S.Ss = (uint32_t)sc.Ss; S.Se = (uint32_t)sc.Se;
        search_all<AcSteps, kWarps>(S, L, s_marks, s_pos, s_state, S.Ss, 0u, pos, st);
        for (uint32_t p = pos, k = st; p < L.end;) {
            const uint32_t e = S.entry(p, k);
            const uint32_t n = e & kEntEob ? eob_blocks(e, long_window(L.base, p)) : 1u;
            if (e) nb += S.advance(e, k) ? n : 0u;
            p += e ? e & 31u : 1u;
        }
        uint32_t m = min(cta_exclusive_sum(nb, s_u, wid, lane, kWarps, all), total);
        if (all < total) bad = true;                           // the stream ends before the last block
        // The blocks that BEGIN in this subsequence, the last one to its end; a block that began before it is passed over
        // (the thread before writes it).  So every block has one writer and its values one run in the value
        // array.  What the state at `pos` says is true: an undefined code or a coefficient beyond the band means a
        // corrupt stream.
        const uint32_t Ss = S.Ss, Se = S.Se, bw = g.bw[c0];
        int16_t* const headp = P.head + g.coff[c0] * 8;
        int16_t* const vals = P.vals + 16ll * (L.origin - reinterpret_cast<const uint32_t*>(P.ubuf));
        uint64_t* const auxp = P.aux + ax.base + g.loff[c0] * ax.stride;
        const bool lists = ax.stride == 2u;                    // the band reaches beyond position 7
        // (A step is one straight line that every lane of the warp walks, as in entropy_kernel: an entry of zero moves nothing on.)
        uint32_t k = st, M0 = 0, M1 = 0, lim = m < total ? L.end : 0u;      // lim: the first bit at which no symbol is read
        bool own = k == Ss;
        uint32_t nv = (pos + 1u) >> 1, nv0 = nv;               // next value, the block's first one
        uint32_t bcol = m % mcu_w, bi = (m / mcu_w) * bw + bcol;
        LongWalk w(L.base, pos);
        uint32_t raw = tab_entry(S.tabs, w.win);
        while (__any_sync(0xffffffffu, w.p < lim)) {
#pragma unroll 4
            for (int q = 0; q < 8; ++q) {
                const uint32_t e = w.p < lim ? raw : 0u, skip = e & 31u, sz = (e >> 5) & 15u, win = w.win, next = w.behind(skip);
                raw = tab_entry(S.tabs, next);
                w.go(skip, next);
                k += e >> 9;                                   // behind the coefficient (an end of band: beyond every position)
                const uint32_t at = k - 1u;
                const bool over = sz && k > Se + 1u, coef = sz && own && !over, far = coef && k > 8u, end = k > Se;
                const int val = magnitude(win, skip, sz) << sc.Al;
                stg16_if(coef && !far, headp + 8u * (uint64_t)bi + at, (uint32_t)val);
                stg16_if(far, vals + nv, (uint32_t)val);
                nv += far ? 1u : 0u;
                M0 |= shl0(coef ? 1u : 0u, at); M1 |= shl0(coef ? 1u : 0u, at - 32u);
                const bool some = end && (M0 | M1) != 0;
                if (lists) stg128_if(some, auxp + (uint64_t)bi * 2, value_record(M0, M1, vals + nv0));
                else stg64_if(some, auxp + bi, M0, M1);
                lim = own && e ? L.endbit : lim;
                // the block ends, an end-of-band run skips more
                const uint32_t r = (e >> 9) & 15u, adv = end ? (e & kEntEob ? __funnelshift_l(shl0(win, skip - r), 1u, r) : 1u) : 0u;   // 2^r + the r bits that end the symbol
                lim = end ? (adv >= total - m ? 0u : L.end) : lim;
                nv = end && !own ? (w.p + 1u) >> 1 : nv;       // this thread's values begin where its first block does
                nv0 = end ? nv : nv0;
                k = end ? Ss : k; own = own || end;
                M0 = end ? 0u : M0; M1 = end ? 0u : M1;
                if (over) { bad = true; lim = 0; }
                m += adv; bcol += adv; bi += adv;
                if (bcol >= mcu_w) { bcol = m % mcu_w; bi = (m / mcu_w) * bw + bcol; }
            }
            if (raw == 0 && w.p < lim) {                       // (taken by the next step)
                raw = long_code(S.tabs, w.win, kTabAcFirst);
                if (raw == 0) { bad = true; lim = 0; }
            }
        }
    }
    if (__syncthreads_or(bad) && tid == 0) atomicMin(&P.status[img], kErrCorrupt);
}

// ---------------------------------------------------------------------------------------
// A sequential (baseline) scan that is one restart interval: one CTA of kSeqLongWarps warps per listed image.  Bound like
// the kernel above.
// ---------------------------------------------------------------------------------------
constexpr int kSeqLongWarps = 4, kSeqLongWideWarps = 16;
template <int kWarps> __host__ __device__ constexpr uint32_t seq_long_stage() { return kWarps == kSeqLongWarps ? 6144 : 4096; }      // words

template <int kWarps>
__global__ void __launch_bounds__(32 * kWarps) sequential_long_kernel(Params P, const uint32_t* __restrict__ list, uint32_t count) {
    constexpr int kThreads = 32 * kWarps;
    constexpr uint32_t kSeqLongStage = seq_long_stage<kWarps>();
    __shared__ __align__(16) uint8_t s_tabs[4 * sizeof(ScanTab)];
    __shared__ uint32_t s_stage[kSeqLongStage];
    __shared__ uint32_t s_marks[kMarks * kThreads];
    __shared__ uint32_t s_pos[kWarps], s_state[kWarps], s_u[kWarps];
    __shared__ int s_i[kWarps];
    const int tid = threadIdx.x, wid = tid >> 5, lane = tid & 31;
    const uint32_t it = blockIdx.x;
    if (it >= count) return;                                   // whole CTA
    const uint32_t si = list[it];
    const int img = (int)(si % (uint32_t)P.N);
    const ScanDesc& sd = P.scans[si];
    const ScanAux ax = P.saux[si / (uint32_t)P.N];
    const Geometry g = make_geometry(P.imgs[img], P);
    const uint32_t mcu_w = g.mx, total = g.mx * g.my, ny = (uint32_t)(P.hs * P.vs), hs = (uint32_t)P.hs, vs = (uint32_t)P.vs;
    const uint32_t bpm = P.nc == 3 ? ny + 2u : 1u;
    SeqSteps S;
    S.tabs = (uint32_t)__cvta_generic_to_shared(s_tabs); S.bpm = bpm; S.tdc = 0; S.tac = 0;
    for (uint32_t j = 0; j < bpm; ++j) {
        const uint32_t c = j < ny ? 0u : j - ny + 1u;
        S.tdc |= ((sd.slots >> (2u * c)) & 1u) << j; S.tac |= ((sd.slots_ac >> (2u * c)) & 1u) << j;
    }
    load_tabs(S.tabs, P.tabs + ax.tab0 + 4u * (uint32_t)img, 4, tid, kThreads);
    LongSpan L;
    L.init<kThreads, 32 * kSeqLongWarps, 32>(P, sd, (uint32_t)tid, s_stage, kSeqLongStage);
    S.base = L.base;
    __syncthreads();
    if (!L.ok) {
        if (tid == 0) atomicMin(&P.status[img], kErrCorrupt);
        return;
    }
    bool bad = false;
    uint32_t pos, st, all, nb = 0;
    search_all<SeqSteps, kWarps>(S, L, s_marks, s_pos, s_state, 0u, 0u, pos, st);
    int sum0 = 0, sum1 = 0, sum2 = 0;
    for (uint32_t p = pos, q = st; p < L.end;) {
        const uint32_t e = S.entry(p, q), j = q >> 6;
        const int d = (q & 63u) == 0 ? magnitude(long_window(L.base, p), e & 31u, (e >> 5) & 15u) : 0;      // (no symbol: 0)
        sum0 += j < ny ? d : 0; sum1 += j == ny ? d : 0; sum2 += j > ny ? d : 0;
        if (e) nb += S.advance(e, q) ? 1u : 0u;
        p += e ? e & 31u : 1u;
    }
    int t;
    uint32_t n = cta_exclusive_sum(nb, s_u, wid, lane, kWarps, all);
    int pred0 = cta_exclusive_sum(sum0, s_i, wid, lane, kWarps, t);
    int pred1 = cta_exclusive_sum(sum1, s_i, wid, lane, kWarps, t);
    int pred2 = cta_exclusive_sum(sum2, s_i, wid, lane, kWarps, t);
    const uint32_t n1 = total * bpm;
    n = min(n, n1);
    // (as for the DC scans above)
    if ((nb || (st & 63u)) && (st >> 6) != n % bpm) bad = true;
    if (all < n1) bad = true;                                  // the stream ends before the last block
    // the blocks that BEGIN in this subsequence (see above); a DC symbol is written by the thread that has it
    int16_t* const dcp = P.dc + g.coff[0];
    int16_t* const headp = P.head + g.coff[0] * 8;
    int16_t* const vals = P.vals + 16ll * (L.origin - reinterpret_cast<const uint32_t*>(P.ubuf));
    uint64_t* const auxp = P.aux + ax.base + 2 * g.coff[0];
    uint32_t j = n % bpm, k = st & 63u, m = n / bpm, mcol = m % mcu_w, M0 = 0, M1 = 0, lim = n < n1 ? L.end : 0u;
    uint32_t yb = vs * (m / mcu_w) * g.bw[0] + hs * mcol;
    const uint32_t wrap = (vs - 1u) * g.bw[0];
    bool own = k == 0;
    uint32_t nv = (pos + 1u) >> 1, nv0 = nv;                   // next value, the block's first one
    LongWalk w(L.base, pos);
    auto dc_tab = [&](uint32_t place) { return S.tabs + ((S.tdc >> place) & 1u) * (uint32_t)sizeof(ScanTab); };
    auto ac_tab = [&](uint32_t place) { return S.tabs + (2u + ((S.tac >> place) & 1u)) * (uint32_t)sizeof(ScanTab); };
    uint32_t raw = tab_entry(k ? ac_tab(j) : dc_tab(j), w.win);
    while (__any_sync(0xffffffffu, w.p < lim)) {
#pragma unroll 4
        for (int q = 0; q < 8; ++q) {
            const uint32_t e = w.p < lim ? raw : 0u, skip = e & 31u, sz = (e >> 5) & 15u, win = w.win, next = w.behind(skip);
            const bool is_dc = k == 0;
            const uint32_t kk = k + (e >> 9), after = j + 1u == bpm ? 0u : j + 1u;     // (an end of block goes beyond 63)
            const bool over = sz && kk > 64u && !is_dc, end = kk > 63u;
            raw = e ? tab_entry(end ? dc_tab(after) : ac_tab(j), next) : raw;
            w.go(skip, next);
            const uint32_t blk = j < ny ? yb + (j >> (hs - 1u)) * g.bw[0] + (j & (hs - 1u)) : j * total + m;
            int v = magnitude(win, skip, sz);
            v += is_dc ? (j < ny ? pred0 : (j == ny ? pred1 : pred2)) : 0;
            const bool dc_now = is_dc && e;
            pred0 = dc_now && j < ny ? v : pred0; pred1 = dc_now && j == ny ? v : pred1; pred2 = dc_now && j > ny ? v : pred2;
            stg16_if(dc_now, dcp + blk, (uint32_t)v);
            const bool coef = sz && own && !is_dc && !over, far = coef && kk > 8u;
            stg16_if(coef && !far, headp + 8ull * blk + kk - 1u, (uint32_t)v);
            stg16_if(far, vals + nv, (uint32_t)v);
            nv += far ? 1u : 0u;
            M0 |= shl0(far ? 1u : 0u, kk - 1u); M1 |= shl0(far ? 1u : 0u, kk - 33u);
            stg128_if(end && (M0 | M1) != 0, auxp + 2ull * blk, value_record(M0, M1, vals + nv0));
            lim = own && e ? L.endbit : lim;
            n += end ? 1u : 0u;
            lim = end ? (n < n1 ? L.end : 0u) : lim;
            nv = end && !own ? (w.p + 1u) >> 1 : nv;
            nv0 = end ? nv : nv0;
            k = end ? 0u : kk; own = own || end;
            M0 = end ? 0u : M0; M1 = end ? 0u : M1;
            if (over) { bad = true; lim = 0; }
            const bool mcu = end && after == 0;
            j = end ? after : j;
            m += mcu ? 1u : 0u; mcol += mcu ? 1u : 0u; yb += mcu ? hs : 0u;
            if (mcol == mcu_w) { mcol = 0; yb += wrap; }
        }
        if (raw == 0 && w.p < lim) {                           // (taken by the next step)
            raw = long_code(k ? ac_tab(j) : dc_tab(j), w.win, k ? kTabAcSeq : kTabDcSeq);
            if (raw == 0) { bad = true; lim = 0; }
        }
    }
    if (__syncthreads_or(bad) && tid == 0) atomicMin(&P.status[img], kErrCorrupt);
}

// ---------------------------------------------------------------------------------------
// AC refinements of scans that are one restart interval.  The unit of work is a chain: one
// refinement scan of one (image, component) group; a group has at most four (its "levels", in
// scan order).  Side data written per block is that of entropy_kernel's refinement branch:
// {non-zero mask of the band after the scan, correction bits in reading order, the last one in bit 0,
// newly non-zero positions, the positive ones among them}.
//
// The time of a chain is the latency of what one thread does per symbol, so the decoding thread only follows
// the chain, through two shared-memory tables that the chain's helper warp prepares:
//   q[bit]       what the symbol that begins at this bit of the stream is (skip, run, flags): every bit position is
//                decoded in advance, 32 at a time, so the thread neither assembles a window nor looks up a code;
//   zpos[b][i]   non-zero positions in front of the i-th still-zero coefficient of block b: by differences the number of
//                correction bits passed; and whether the block ends there.
// A symbol is two dependent loads and a handful of additions, and what a block that ends takes beyond that does not ask how many
// still-zero positions there are: the list says where the block ends, and its entries beyond that are all closing ones.  Per block the
// thread leaves the bit position where the next one begins; the helper warp decodes the 32 blocks of a finished batch once more, one
// lane per block, to make the side data.
// A lone thread takes about four cycles an instruction whatever it waits for, so the count of instructions decides.  The launch in us
// with 16 instructions a symbol and a block change that carried the next block's bounds along (clock64 in a copy that took most symbols
// by one load: 45 cycles a symbol and 370 a block); with lists that say where a block ends; and now, with runs counted from the entry
// reached, the flag of the ending entry taken out once a block instead of in every symbol, and the chain's place in shared memory in a
// uniform register:
//   HAM-shaped, 1024 / 512 / 128 images   1728 -> 1565 -> 1414, 1468 -> 1285 -> 1181, 1412 -> 1230 -> 1127
//   mixed sizes, 200                      3281 -> 2846 -> 2656
//   ImageNet-shaped, 1024 / 256           2843 -> 2483 -> 2289, 2768 -> 2409 -> 2241
//   CelebA-shaped, 256 at k = 8           268 -> 237 -> 221
// Not kept (HAM-shaped 1024, 512, 128, mixed sizes; of the second form): block change by selects in the symbol's line (1785, 1349,
// 1279, 2890); a loop of one load a symbol behind a block's last non-zero position (1599, 1335, 1273, 2786); the entries behind the
// symbol's own bits requested before the number of correction bits is known (2331, 1754, 1652, 3628); the loop unrolled (1869).
// Codes longer than the quick table's index are looked up where the thread meets one, since few records have many of them; with the
// helper looking them up at every bit position, filling q was 28 % of its time.  128 HAM-shaped images whose refinement tables have
// longer codes than they need (us: looked up by the helper; by the thread, the block again for every one; and now): all 10 bits 9829,
// 11333, 8344; all longer by the same number, the shortest 10 bits 14354, 13878, 10181; those of three bits and more by seven 6616,
// 8105, 7314; those of five and more by six 3271, 3170, 3434.  (All of a block's long codes looked up from the first one on: 7224,
// 8890, 5986, 3465, but 1 to 2 % on the mixed sizes and ImageNet-shaped records above.)
//
// A later refinement of the same component needs the masks the earlier one leaves, block by
// block.  Both walk the same block grid in the same order, so the later chain runs behind the
// earlier one instead of after it: every chain publishes the number of blocks whose side data it
// has written (global memory, after a fence), and a helper that depends on it waits, with a
// bounded number of polls, until the blocks it is about to read are there.  A chain is only
// started after the chains it depends on (queue order), so its producer is running or done.
// ---------------------------------------------------------------------------------------
constexpr int kChainPairs = 16;          // chains per CTA of the persistent refinement launch (four per scheduler), two warps each
constexpr uint32_t kChainRing = 128;     // words of bitstream per chain in shared memory
constexpr uint32_t kChainBits = 32 * kChainRing;
constexpr int kChainLutBits = 9;         // refinement alphabets are small (runs 0..15 with size 0 or 1): short codes
constexpr uint32_t kChainBlockWords = 44;   // a block never needs more: 63 symbols of at most 17 bits, 3 sixteen-zero runs, one run length, 63 correction bits
constexpr uint32_t kSpinLimit = 1u << 22;   // polls (of at least 64 ns) before a wait gives up
constexpr int kErrTimeout = -4;

// Polls *flag until it reaches `need`, sleeping `ns` nanoseconds between polls; false after `limit` polls.
__device__ __forceinline__ bool wait_at_least(const volatile uint32_t* flag, uint32_t need, uint32_t limit, uint32_t ns = 64) {
#pragma unroll 1
    for (uint32_t i = 0; i < limit; ++i) {
        if (*flag >= need) return true;
        __nanosleep(ns);
    }
    return false;
}

// Entry of q: twice the bits to skip (code, sign bit, run-length bits) in bits 0..5, 6 = a new coefficient, 7 = more than
// a plain step (an end-of-band run that covers further blocks, or no symbol: the rest but bit 15 is zero),
// 9..15 = run of zeros plus one (from 64 on: the rest of the band; 64 + the exponent of an end-of-band run).  kQLong: a code longer than the quick
// table's index (an exponent that no run has); the decoding thread looks it up where it meets one, and leaves the entry there.
constexpr uint32_t kQNew = 0x40u, kQSpecial = 0x80u, kQRest = 64u << 9, kQBad = kQSpecial | kQRest, kQLong = kQBad | (15u << 9);
__device__ __forceinline__ uint32_t chain_entry(uint32_t len, uint32_t rs) {
    const uint32_t r = rs >> 4, newc = rs & 1u;
    if (rs & 14u) return kQBad;                                        // a refinement symbol has size 0 or 1
    if (newc || r == 15u) return (2u * (len + newc)) | (newc ? kQNew : 0u) | ((r + 1u) << 9);
    return (2u * (len + r)) | (r ? kQSpecial : 0u) | kQRest | (r << 9);
}

constexpr uint32_t kChainList = 68;          // bytes of a block's list (64 entries; blocks side by side fall on different banks)

struct ChainMail {                     // what the two warps of a chain tell each other at a meeting point
    uint32_t nd, rd, err_c;            // decoder: blocks it decoded, the word it stands at, error
    uint32_t wr, err_h;                // helper: the ring is filled up to this word, error
};
struct ChainShared {
    uint16_t q[kChainBits];            // by bit position modulo kChainBits
    uint8_t zpos[2][32][kChainList];   // [batch][block][i]: twice the number of the band's non-zero positions in front of the block's i-th still-zero
                                       // one; from the number of still-zero positions on, twice all of them.  Bit 7: the block ends there
                                       // (those entries, and the one of a still-zero position Se)
    uint32_t start[2][33];             // per block, and behind the last: where it began (bit position; bit 31: inside an end-of-band run)
    uint32_t ring[kChainRing];
    const uint8_t* dht;                         // the table's body: 16 length counts, then the values
    uint16_t quick[1 << kChainLutBits];         // q entries of the codes of at most kChainLutBits bits, kQLong: longer
    uint16_t first[8], cnt[8], idx[8];          // the longer codes: first code, how many, index of the first value
    ChainMail mail[2];                 // by parity of the meeting point
    uint32_t job_gi, job_level;        // the pair's job (job_gi = 0xFFFFFFFF: none left)
    uint32_t total, lead, limit;                // of the job, for the decoder (bits counted from the interval's first word)
    uint32_t once;                              // where the block began whose long code was looked up last (a bit position)
    volatile uint32_t phase_c, phase_h;         // meeting points each side has reached
};
static_assert(kChainPairs * sizeof(ChainShared) <= 227 * 1024, "one CTA per SM holds all its chains");

// the n bits (1..32) at bit position p of the ring
__device__ __forceinline__ uint32_t ring_bits(const uint32_t* ring, uint32_t p, uint32_t n) {
    const uint32_t a = ring[(p >> 5) & (kChainRing - 1)], b = ring[((p >> 5) + 1u) & (kChainRing - 1)];
    return __funnelshift_l(b, a, p & 31u) >> (32u - n);
}

// The entry of the code longer than kChainLutBits bits at pos2 (twice its bit position), left in q too.
template <int kUnroll>
__device__ __forceinline__ uint32_t chain_long(uint32_t base, uint32_t pos2) {
    constexpr uint32_t kRing = offsetof(ChainShared, ring), kFirst = offsetof(ChainShared, first), kCnt = offsetof(ChainShared, cnt), kIdx = offsetof(ChainShared, idx);
    const uint32_t p = pos2 >> 1, w = base + kRing;
    const uint32_t x = __funnelshift_l(lds32(w + 4u * (((p >> 5) + 1u) & (kChainRing - 1u))), lds32(w + 4u * ((p >> 5) & (kChainRing - 1u))), p & 31u);
    uint32_t e = kQBad;
#pragma unroll kUnroll
    for (uint32_t j = 0; j < 16u - kChainLutBits; ++j) {
        const uint32_t l = kChainLutBits + 1u + j, d = (x >> (32u - l)) - lds16(base + kFirst + 2u * j);
        if (d < lds16(base + kCnt + 2u * j)) {
            const uint2 a = lds64(base + (uint32_t)offsetof(ChainShared, dht));
            e = chain_entry(l, reinterpret_cast<const uint8_t*>(((uint64_t)a.y << 32) | a.x)[16u + ((lds16(base + kIdx + 2u * j) + d) & 255u)]);
            break;
        }
    }
    sts16(base + (pos2 & (2u * kChainBits - 1u)), e);
    return e;
}

// A block with several long codes, from its beginning (pos2: twice the bit position; last: its list's last entry): every one is looked up where it
// stands.  -> where the decoder goes on, in front of the block's last symbol: r (or what leads to the same target), passed2 and pos2 there.
// (Not inlined, and back into the decoder's own loop: with this loop, or another end of a block, beside it that one takes 2 to 5 % longer.)
__device__ __noinline__ uint3 chain_long_codes(uint32_t base, uint32_t pos2, uint32_t last) {
    uint32_t r = last - 64u, entry = 0, passed2, e, d2;
#pragma unroll 1
    do {
        e = lds16(base + (pos2 & (2u * kChainBits - 1u)));
        if (e == kQLong) e = chain_long<16 - kChainLutBits>(base, pos2);
        r = __viaddmin_u32(r, e >> 9, last);
        passed2 = entry;
        entry = lds8(r);
        d2 = (e & 63u) + entry - passed2;
        pos2 += d2;
    } while (entry < 128u);
    return make_uint3(r - (e >> 9), passed2, pos2 - d2);
}

// Polls *flag (another warp's progress word in global memory) until it reaches `need`; `seen` keeps
// the last value read, so that a consumer that is behind anyway polls once per many batches.
__device__ __forceinline__ bool wait_progress(const volatile uint32_t* flag, uint32_t need, uint32_t& seen, uint32_t limit) {
    if (seen >= need) return true;
#pragma unroll 1
    for (uint32_t i = 0; i < limit; ++i) {
        seen = *flag;
        if (seen >= need) return true;
        __nanosleep(500);
    }
    return false;
}

// Meeting point k of a chain's two warps: each side announces that it has arrived (everything it
// wrote to shared memory before is visible to the other behind the meeting) and waits, with a
// bounded number of polls, for the other.  false: the partner never came.
__device__ __forceinline__ bool meet_decoder(ChainShared& sh, uint32_t k) {          // one thread
    __threadfence_block();
    sh.phase_c = k;
    const bool ok = wait_at_least(&sh.phase_h, k, kSpinLimit, 300);
    __threadfence_block();
    return ok;
}
__device__ __forceinline__ bool meet_helper(ChainShared& sh, uint32_t k, int lane) {  // a whole warp
    __syncwarp();
    if (lane == 0) { __threadfence_block(); sh.phase_h = k; }
    // (long sleeps: the helper is far ahead of the decoder, and its polls would take issue slots from the chains)
    bool ok = true;
    if (lane == 0) ok = wait_at_least(&sh.phase_c, k, kSpinLimit, 1000);
    ok = __shfl_sync(0xffffffffu, (int)ok, 0) != 0;
    __threadfence_block();
    return ok;
}

// The decoding side of a chain: one thread.  It takes the pair's jobs (first the statically assigned
// one, then tickets of its scheduler's queue), and per job follows the bit stream batch by batch.
// `base`: the shared address of sh, the same in the whole warp.
__device__ __forceinline__ void chain_decoder(const RefineList& fl, ChainShared& sh, uint32_t base, const uint32_t* __restrict__ list, uint32_t n_groups,
                                              uint32_t* sync, uint32_t levels, uint32_t rounds, uint32_t q, uint32_t slot) {
    const uint32_t per_round = 4u * gridDim.x, statics = per_round * rounds;
    const uint32_t a_q = base, a_zpos = base + (uint32_t)offsetof(ChainShared, zpos), a_start = base + (uint32_t)offsetof(ChainShared, start);
    uint32_t mk = 0;                                           // meeting points so far
    bool first_job = true;
    for (;;) {
        uint32_t gi, level;
        for (;;) {
            if (first_job) {
                first_job = false;
                gi = (slot / levels) * per_round + 4u * blockIdx.x + q;
                level = slot % levels;
            } else {
                const uint32_t t = atomicAdd(&sync[q], 1u);
                gi = statics + 4u * (t / levels) + q;
                level = t % levels;
            }
            if (gi >= n_groups) { gi = 0xFFFFFFFFu; break; }  // the queue is empty (entries only grow)
            if ((int)level < fl.n[list[gi] >> 28]) break;      // (a component with fewer refinements has no such level)
        }
        sh.job_gi = gi; sh.job_level = level;
        if (!meet_decoder(sh, ++mk)) return;                   // the helper has the job
        if (gi == 0xFFFFFFFFu) return;
        if (!meet_decoder(sh, ++mk)) return;                   // tables, first lists and ring are ready
        if (sh.mail[mk & 1u].err_h) continue;                  // a scan whose bounds are off: the helper reports it
        uint32_t wr = sh.mail[mk & 1u].wr;
        const uint32_t total = sh.total, limit = sh.limit;
        sh.once = 0xFFFFFFFFu;
        uint32_t pos2 = 2u * sh.lead;                          // twice the bit position (the tables' entries are two bytes)
        uint32_t eobrun = 0, m = 0, p = 0;
        for (;;) {
            const uint32_t nblk = min(32u, total - m);
            // A block is only begun while kChainBlockWords words lie ahead (q ends one word before the ring) and, the
            // batch's first one, while the interval has not ended (reading on behind it is found below; zeros follow).
            const uint32_t lead2 = 64u * (wr - min(wr, kChainBlockWords + 3u));
            const uint32_t start = a_start + 132u * p;
            // (addresses) the block's last entry, and the one its last symbol reached
            uint32_t last = a_zpos + 32u * kChainList * p + 63u, r = last - 64u;
            uint32_t nd = 0, passed2 = 0;                      // blocks done; twice the non-zero positions passed in this one
            int err = 0;
            sts32(start, pos2 >> 1);
            bool go = pos2 < lead2 && (pos2 >> 1) <= limit;
            while (go) {
                if (eobrun == 0) {
                    uint32_t e, raw = lds16(a_q + (pos2 & (2u * kChainBits - 1u))), corr2;     // (raw: the next symbol's entry)
                    do {
                        uint32_t entry;
#pragma unroll 1
                        do {
                            e = raw;
                            // the target: the (r+1)-th still-zero position from here; a run past the last one (an end
                            // of band is one too) ends at a closing entry
                            const uint32_t t = __viaddmin_u32(r, e >> 9, last);
                            entry = lds8(t);
                            corr2 = entry - passed2;           // one correction bit for each non-zero position passed
                            pos2 += (e & 63u) + corr2;         // code, sign and correction bits in one step
                            raw = lds16(a_q + (pos2 & (2u * kChainBits - 1u)));
                            r = t;
                            passed2 = entry;
                        } while (entry < 128u);
                        // (the flag of the ending entry, counted along until here)
                        pos2 -= 128u; corr2 -= 128u;
                        raw = lds16(a_q + (pos2 & (2u * kChainBits - 1u)));
                        r = last + (kChainList - 64u);
                        last += kChainList;
                        passed2 = 0;
                        ++nd;
                        sts32(start + 4u * nd, pos2 >> 1);
                    } while (!(e & kQSpecial) && nd != nblk && pos2 < lead2);
                    if (e & kQSpecial) {
                        if (e == kQLong) {
                            // A long code: its entry looked up, and the block once more from its beginning; where that happens a second
                            // time, all of its long codes are, so that a block's symbols are walked three times at most.
                            --nd; last -= kChainList;
                            const uint32_t from = lds32(start + 4u * nd);
                            if (sh.once != from) {
                                sh.once = from;
                                chain_long<1>(base, pos2 - corr2);
                                r = last - 64u; pos2 = 2u * from;
                                continue;
                            }
                            const uint3 at = chain_long_codes(base, 2u * from, last);
                            r = at.x; passed2 = at.y; pos2 = at.z;
                            continue;
                        }
                        if (e == kQBad) { err = kErrCorrupt; --nd; break; }
                        // the band also ends for the next eobrun blocks
                        const uint32_t x = (e >> 9) & 15u;
                        eobrun = (1u << x) + ring_bits(sh.ring, ((pos2 - corr2) >> 1) - x, x) - 1u;
                    }
                } else {
#pragma unroll 1
                    do {
                        sts32(start + 4u * nd, (pos2 >> 1) | 0x80000000u);
                        pos2 += lds8(last) & 127u;             // inside an end-of-band run: corrections for the whole band
                        --eobrun;
                        ++nd; last += kChainList;
                    } while (eobrun && nd < nblk && pos2 < lead2);
                    r = last - 64u;
                    sts32(start + 4u * nd, pos2 >> 1);
                }
                go = nd < nblk && pos2 < lead2;
            }
            if (!err && (pos2 >> 1) > limit) err = kErrCorrupt;    // read past the end of the interval
            ++mk;
            sh.mail[mk & 1u].nd = nd; sh.mail[mk & 1u].rd = pos2 >> 6; sh.mail[mk & 1u].err_c = (uint32_t)err;
            if (!meet_decoder(sh, mk)) return;
            wr = sh.mail[mk & 1u].wr;
            if (err || sh.mail[mk & 1u].err_h) break;
            m += nd;
            if (nd == nblk) {
                p ^= 1u;
                if (m >= total) break;
            } else {                                           // stopped early: the helper lists the blocks from m again
                if (!meet_decoder(sh, ++mk)) return;
                wr = sh.mail[mk & 1u].wr;
                if (sh.mail[mk & 1u].err_h) break;
                p ^= 1u;
            }
        }
    }
}

// The helper side of a chain: a whole warp.  Per job it builds the tables, then stays one batch ahead
// of the decoder with the lists of still-zero positions (waiting, with bounded polls, for
// an earlier refinement of the same blocks when this launch decodes that too), keeps the ring of
// bitstream words and their symbols filled, and one batch behind it makes the side data.
__device__ __forceinline__ void chain_helper(const Params& P, const RefineList& fl, ChainShared& sh, const uint32_t* __restrict__ list,
                                             uint32_t* progress_all, int lane) {
    const unsigned full = 0xffffffffu;
    uint32_t mk = 0;
    for (;;) {
        if (!meet_helper(sh, ++mk, lane)) return;
        const uint32_t gi = sh.job_gi;
        const int level = (int)sh.job_level;
        if (gi == 0xFFFFFFFFu) return;
        const uint32_t entry = list[gi];
        const int c = (int)(entry >> 28), img = (int)(entry & 0x0FFFFFFFu);
        uint32_t* progress = progress_all + 4ull * gi;
        volatile uint32_t* my_progress = progress + level;
        const int s = fl.scan[c][level];
        const ScanDesc& sd = P.scans[(uint32_t)s * (uint32_t)P.N + (uint32_t)img];
        const ScanScript sc = P.script[s];
        const Geometry g = make_geometry(P.imgs[img], P);
        const uint32_t Ss = (uint32_t)sc.Ss, Se = (uint32_t)sc.Se;
        const uint32_t mcu_w = g.ubw[c], total = g.ubw[c] * g.ubh[c], bw = g.bw[c];
        // the code tables: q entries of the short codes, the canonical description of the longer ones
        const uint8_t* dht = P.rec + sd.tab_off[0];
        {
            uint32_t* s_code = &sh.start[0][0];                // scratch (51 words): first code, first index, end of the codes
            const uint32_t my = lane < 16 ? dht[lane] : 0u;
            uint32_t code = 0, idx = 0;
            for (int l = 1; l <= 16; ++l) {
                const uint32_t n = __shfl_sync(full, my, l - 1);
                if (lane == 0) {
                    s_code[l] = code; s_code[17 + l] = idx;
                    if (l <= kChainLutBits) s_code[34 + l] = (code + n) << (kChainLutBits - l);
                    else { const int j = l - kChainLutBits - 1; sh.first[j] = (uint16_t)code; sh.cnt[j] = (uint16_t)n; sh.idx[j] = (uint16_t)idx; }
                }
                code = (code + n) << 1;
                idx += n;
            }
            __syncwarp(full);
            int l = 1;
            for (int e = 0; e < (1 << kChainLutBits) / 32; ++e) {      // consecutive entries: the code length only grows
                const uint32_t x = (uint32_t)lane * ((1u << kChainLutBits) / 32u) + (uint32_t)e;
                while (l <= kChainLutBits && x >= s_code[34 + l]) ++l;
                uint32_t v = kQLong;
                if (l <= kChainLutBits) v = chain_entry((uint32_t)l, dht[16u + ((s_code[17 + l] + (x >> (kChainLutBits - l)) - s_code[l]) & 255u)]);
                sh.quick[x] = (uint16_t)v;
            }
            __syncwarp(full);
        }
        const uint32_t* segtab = P.seg_start + sd.seg_base;
        const uint32_t bstart = segtab[0], bend = segtab[1] - 2u;
        const bool bad = bstart < sd.data_off || bend > sd.data_end || bend < bstart;
        const uint32_t rd0 = bstart >> 2, lead = 8u * (bstart & 3u);
        const uint32_t* words = reinterpret_cast<const uint32_t*>(P.ubuf) + rd0;
        const uint32_t wlim = ((bend + 3u) >> 2) + 2u - rd0;   // words beyond are not read (zeros instead)
        if (lane == 0) {
            sh.total = total; sh.lead = lead;
            sh.limit = lead + 8u * (bend - bstart);            // first bit behind the interval
            sh.dht = dht;
        }
        // masks of the positions that are already non-zero: the union of up to four earlier scans; a
        // source that this launch decodes itself (an earlier level of the group) is waited for
        // (prod* = its progress word)
        const ScanAux ax = P.saux[s];
        const uint64_t band = low_mask((int)Se + 1) & ~low_mask((int)Ss);
        const uint64_t* src0 = nullptr; const uint64_t* src1 = nullptr; const uint64_t* src2 = nullptr; const uint64_t* src3 = nullptr;
        uint32_t st0 = 0, st1 = 0, st2 = 0, st3 = 0;
        const volatile uint32_t* prod0 = nullptr; const volatile uint32_t* prod1 = nullptr; const volatile uint32_t* prod2 = nullptr;
        {
            auto producer = [&](int scan) -> const volatile uint32_t* {
                for (int w = 0; w < level; ++w) if (fl.scan[c][w] == scan) return progress + w;
                return nullptr;
            };
            auto note = [&](const volatile uint32_t* q) { if (q) { if (!prod0) prod0 = q; else if (!prod1) prod1 = q; else prod2 = q; } };
            const ScanAux x0 = P.saux[ax.src[0]];
            src0 = P.aux + x0.base + g.loff[c] * x0.stride; st0 = x0.stride; note(producer(ax.src[0]));
            if (ax.nsrc > 1) { const ScanAux x = P.saux[ax.src[1]]; src1 = P.aux + x.base + g.loff[c] * x.stride; st1 = x.stride; note(producer(ax.src[1])); }
            if (ax.nsrc > 2) { const ScanAux x = P.saux[ax.src[2]]; src2 = P.aux + x.base + g.loff[c] * x.stride; st2 = x.stride; note(producer(ax.src[2])); }
            if (ax.nsrc > 3) { const ScanAux x = P.saux[ax.src[3]]; src3 = P.aux + x.base + g.loff[c] * x.stride; st3 = x.stride; note(producer(ax.src[3])); }
        }
        uint64_t* outp = P.aux + ax.base + g.loff[c] * 4ull;
        uint32_t* ring = sh.ring;
        uint32_t wr = 0, seen0 = 0, seen1 = 0, seen2 = 0;
        const bool watched = level + 1 < fl.n[c];              // a later level of the group reads the side data
        int err = bad ? kErrCorrupt : 0;
        auto block_index = [&](uint32_t x) { const uint32_t row = x / mcu_w; return row * bw + (x - row * mcu_w); };
        // the masks of blocks m0 .. m0 + 31, one per lane (requested: nothing waits for the loads yet)
        auto masks = [&](uint32_t m0, uint64_t& h) -> int {
            const uint32_t nblk = min(32u, total - m0), need = m0 + nblk;
            const bool polls = (prod0 && seen0 < need) || (prod1 && seen1 < need) || (prod2 && seen2 < need);
            if (polls) {
                if (prod0 && !wait_progress(prod0, need, seen0, kSpinLimit)) return kErrTimeout;
                if (prod1 && !wait_progress(prod1, need, seen1, kSpinLimit)) return kErrTimeout;
                if (prod2 && !wait_progress(prod2, need, seen2, kSpinLimit)) return kErrTimeout;
                __threadfence();
            }
            h = 0;
            if ((uint32_t)lane < nblk) {
                const uint32_t bi = block_index(m0 + lane);
                uint64_t v = __ldcg(src0 + (uint64_t)bi * st0);    // not through L1: a line may hold blocks written later
                if (src1) v |= __ldcg(src1 + (uint64_t)bi * st1);
                if (src2) v |= __ldcg(src2 + (uint64_t)bi * st2);
                if (src3) v |= __ldcg(src3 + (uint64_t)bi * st3);
                h = v;
            }
            return 0;
        };
        // the blocks' lists of still-zero positions into batch buffer b
        auto lists = [&](uint32_t m0, uint32_t b, uint64_t& h) {
            const uint32_t nblk = min(32u, total - m0);
            if ((uint32_t)lane < nblk) {
                h &= band;
                const uint64_t v = h;
                // the positions of the band that are still zero, in order: the target of a run r is then one
                // table look-up for the decoder (the (r+1)-th of those not yet passed)
                const uint64_t z = ~v & band;
                const uint32_t n = (uint32_t)__popcll(z), row = (uint32_t)__cvta_generic_to_shared(&sh.zpos[b][lane][0]);
                const uint32_t closing = (2u * (Se + 1u - Ss - n) | 128u) * 0x01010101u;
#pragma unroll
                for (uint32_t w = 0; w < kChainList; w += 4u) sts32(row + w, closing);
                uint32_t dst = row, v2 = 0u - 2u * Ss;             // v2: twice the non-zero positions so far
                // (straight through all positions, lanes with different masks stay together; a position outside the band
                // counts as non-zero)
#pragma unroll
                for (int pos = 0; pos < 64; ++pos) {
                    const uint32_t zw = pos < 32 ? (uint32_t)z : (uint32_t)(z >> 32);
                    if ((zw >> (pos & 31)) & 1u) {
                        asm volatile("st.shared.u8 [%0], %1;" : : "r"(dst), "r"(v2) : "memory");
                        ++dst;
                    } else v2 += 2u;
                }
                if ((z >> Se) & 1u)                                // the block also ends at a still-zero position Se
                    asm volatile("st.shared.u8 [%0], %1;" : : "r"(dst - 1u), "r"(closing) : "memory");
            }
        };
        // The ring and q filled as far as they go while word `oldest` is still needed.  The symbol at a word's bits
        // needs the word behind it, so q ends one word before the ring.  The next words are requested ahead.
        uint32_t ahead = 0;
        auto request = [&]() { ahead = wr + lane < wlim ? __ldg(words + wr + lane) : 0u; };
        auto top_up = [&](uint32_t oldest) {
            while (wr - oldest + 32u <= kChainRing) {
                ring[(wr + lane) & (kChainRing - 1)] = ahead;
                __syncwarp(full);
#pragma unroll 1
                for (uint32_t w = wr - 1u; w != wr + 31u; w += 8u) {   // (word -1 at first: never looked at)
                    uint32_t x[9], e[8];
#pragma unroll
                    for (uint32_t i = 0; i < 9; ++i) x[i] = ring[(w + i) & (kChainRing - 1)];
#pragma unroll
                    for (uint32_t i = 0; i < 8; ++i) e[i] = sh.quick[__funnelshift_l(x[i + 1], x[i], (uint32_t)lane) >> (32 - kChainLutBits)];
#pragma unroll
                    for (uint32_t i = 0; i < 8; ++i) sh.q[(32u * (w + i) + lane) & (kChainBits - 1u)] = (uint16_t)e[i];
                }
                wr += 32u;
                request();
                __syncwarp(full);
            }
        };
        // the blocks m0 .. m0 + nd - 1 of batch buffer b once more, one per lane -> side data; then the count
        auto side_data = [&](uint32_t m0, uint32_t nd, uint32_t b, uint64_t h) {
            bool over = false;
            if ((uint32_t)lane < nd) {
                const uint32_t st = sh.start[b][lane], nz = Se + 1u - Ss - (uint32_t)__popcll(h);
                const uint8_t* zp = &sh.zpos[b][lane][0];
                uint32_t at = st & 0x7FFFFFFFu, zi = 0xFFFFFFFFu, ep = 0, k = 0;     // zi: the entry reached
                uint32_t s0 = 0, s1 = 0, N0 = 0, N1 = 0, G0 = 0, G1 = 0, isnew = 0;
                // a block inside an end-of-band run is one step over the rest of the band that takes no symbol
                uint32_t e = st >> 31 ? kQRest : (uint32_t)sh.q[at & (kChainBits - 1u)];
#pragma unroll 1
                for (int i = 0; i < 80 && k < Se; ++i) {       // (bounded: more symbols than a block can have)
                    const uint32_t skip = (e & 63u) >> 1, sign_at = at + skip - 1u;
                    const uint32_t t = __viaddmin_u32(zi, e >> 9, nz), e2 = zp[t] & 127u, n = (e2 - ep) >> 1;
                    k = (e2 >> 1) + t + Ss;
                    isnew = e & kQNew ? 1u : 0u;
                    const uint32_t plus = isnew & (ring[(sign_at >> 5) & (kChainRing - 1)] >> (~sign_at & 31u));
                    N0 |= shl0(isnew, k); N1 |= shl0(isnew, k - 32u);
                    G0 |= shl0(plus, k); G1 |= shl0(plus, k - 32u);
                    at += skip;
                    if (n) {
                        const uint32_t w = ring_bits(ring, at, 32u);
                        if (n > 32u) {
                            s1 = (w >> (64u - n)) | (s0 << (n - 32u));
                            s0 = __funnelshift_l(ring_bits(ring, at + 32u, 32u), w, n - 32u);
                        } else {
                            s1 = __funnelshift_lc(s0, s1, n);
                            s0 = shl0(s0, n) | (w >> (32u - n));
                        }
                        at += n;
                    }
                    ep = e2; zi = t;
                    e = sh.q[at & (kChainBits - 1u)];
                }
                over = isnew && k > Se;                        // a new coefficient behind the band
                uint4* o = reinterpret_cast<uint4*>(outp + (uint64_t)block_index(m0 + lane) * 4);
                o[0] = make_uint4((uint32_t)h | N0, (uint32_t)(h >> 32) | N1, s0, s1);
                o[1] = make_uint4(N0, N1, G0, G1);
            }
            if (__any_sync(full, over)) err = kErrCorrupt;
            if (watched) {
                __threadfence();                               // the side data before the count
                __syncwarp(full);
                if (lane == 0) *my_progress = m0 + nd;
            }
        };
        uint64_t h_now = 0, h_next = 0, h_pend = 0;            // masks of the batch being decoded, the one after it, the one before it
        if (!bad) {
            err = masks(0, h_now);
            request();
            top_up(0);
            lists(0, 0, h_now);
        }
        ++mk;
        if (lane == 0) { sh.mail[mk & 1u].wr = wr; sh.mail[mk & 1u].err_h = (uint32_t)err; }
        if (!meet_helper(sh, mk, lane)) return;
        uint32_t m = 0, p = 0, rd_c = 0, pend_m = 0, pend_n = 0, pend_p = 0;
        while (!err) {
            const uint32_t nblk = min(32u, total - m);
            const bool more = m + nblk < total;
            if (more) { const int e = masks(m + nblk, h_next); if (!err) err = e; }
            if (pend_n) { side_data(pend_m, pend_n, pend_p, h_pend); pend_n = 0; }
            top_up(rd_c);
            if (more) lists(m + nblk, p ^ 1u, h_next);
            ++mk;
            if (lane == 0) { sh.mail[mk & 1u].wr = wr; sh.mail[mk & 1u].err_h = (uint32_t)err; }
            if (!meet_helper(sh, mk, lane)) return;
            const uint32_t nd = sh.mail[mk & 1u].nd;
            const int err_c = (int)sh.mail[mk & 1u].err_c;
            rd_c = sh.mail[mk & 1u].rd;
            if (err || err_c) { if (!err) err = err_c; break; }
            if (nd == nblk) {
                pend_m = m; pend_n = nd; pend_p = p; h_pend = h_now;
                h_now = h_next;
                p ^= 1u;
                m += nd;
                if (m >= total) { side_data(pend_m, pend_n, pend_p, h_pend); break; }
            } else {                                           // the decoder stopped early: its blocks now, the lists from m again
                if (nd) side_data(m, nd, p, h_now);
                m += nd;
                top_up(rd_c);
                { const int e = masks(m, h_now); if (!err) err = e; }
                lists(m, p ^ 1u, h_now);
                ++mk;
                if (lane == 0) { sh.mail[mk & 1u].wr = wr; sh.mail[mk & 1u].err_h = (uint32_t)err; }
                if (!meet_helper(sh, mk, lane)) return;
                p ^= 1u;
            }
        }
        __syncwarp(full);
        if (lane == 0) {
            __threadfence();
            *my_progress = 0xFFFFFFFFu;                        // a scan that failed must not keep a later one waiting
            if (err) atomicMin(&P.status[img], err);
        }
    }
}

// Persistent launch: one CTA per SM with `pairs` chains, each a decoding warp (one thread of it
// works) and a helper warp; warp w and its helper w + pairs sit on scheduler w % 4.  The groups
// ((image, component) pairs, luminance first, most bytes first) are dealt to four queues, one per
// scheduler (group gi is in queue gi % 4); within a queue every group is followed through its levels
// (the refinement scans of the component that this call decodes, in script order), so a producer is
// always taken before its consumer.  The first `rounds` groups of each CTA's schedulers are assigned
// statically (group r * 4 * CTAs + 4 * CTA + q in round r: every scheduler of the device gets one
// long luminance chain before any gets a second, and a group's levels start together in one CTA);
// after that a decoder that has finished takes the next entry of its queue from a counter in global
// memory.  sync: four queue counters, then four progress words per group, all zero before the launch.
__global__ void __launch_bounds__(64 * kChainPairs, 1) ac_refine_group_kernel(Params P, RefineList fl, const uint32_t* __restrict__ list,
                                                                              uint32_t n_groups, uint32_t* __restrict__ sync, int levels, int rounds) {
    extern __shared__ __align__(16) unsigned char s_dyn[];     // one ChainShared per chain
    ChainShared* s_sh = reinterpret_cast<ChainShared*>(s_dyn);
    const int pairs = (int)(blockDim.x >> 6);
    const int wid = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if ((int)threadIdx.x < pairs) { s_sh[threadIdx.x].phase_c = 0; s_sh[threadIdx.x].phase_h = 0; }
    __syncthreads();
    if (wid < pairs) {
        // (a reduction leaves its result in a uniform register, which loads and stores add for nothing: 5 % of the launch)
        const uint32_t base = __reduce_max_sync(0xffffffffu, (uint32_t)__cvta_generic_to_shared(&s_sh[wid]));
        if (lane == 0) chain_decoder(fl, s_sh[wid], base, list, n_groups, sync, (uint32_t)levels, (uint32_t)rounds, (uint32_t)wid & 3u, (uint32_t)wid >> 2);
    } else {
        chain_helper(P, fl, s_sh[wid - pairs], list, sync + 4, lane);
    }
}

// Test hook: the bounded wait on a flag that nothing sets; *result = 1 if it gave up as it should.
__global__ void bounded_wait_probe_kernel(uint32_t limit, int* result) {
    __shared__ uint32_t s_flag;
    if (threadIdx.x == 0) s_flag = 0;
    __syncthreads();
    const bool ok = wait_at_least(&s_flag, 1u, limit);
    if (threadIdx.x == 0) *result = ok ? 0 : 1;
}

}  // namespace pcr
