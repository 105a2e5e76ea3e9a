// Entropy stage of the PCR decoder: restart-interval index with the symbol tables, and the Huffman decode of
// one wave of scans.  (Baseline images: pcr_sequential.cuh.)
//
// Parallel decomposition: one LANE per restart interval.  A warp takes up to 32 consecutive
// restart intervals of one (scan, image) pair, so its lanes share the scan's Huffman tables
// (lookup tables in shared memory).  Every lane runs ONE flat loop whose iteration decodes one
// Huffman symbol (or one block of an end-of-band run); block changes are a few predicated
// instructions inside that loop, so lanes that sit in different blocks stay converged.
//
// First passes leave a block's coefficients as DC value, dense values of positions 1..7, and for the positions
// behind them a mask and a packed list of values: nothing has to be zeroed before a decode, and a block's part
// of a scan is a few bytes instead of a 128-byte line.  An AC refinement needs, per block, only WHICH band
// positions are already non-zero: a 64-bit mask.  A refinement lane decodes with bit operations by rank (the
// mask's zero positions are counted per byte; a run of r zeros looks up the byte that holds the r-th and selects
// inside it; one correction bit per set bit of the mask passed over) and leaves {new mask, correction bits, new
// positions, their signs} as side data, which the pixel kernel applies when it expands the block.
//
// (AC refinements of records that do not fill the machine: pcr_refine.cuh.)
// Bound by the latency of a lane's chain and, with the machine full, by the issue rate that the resident warps allow: a
// refinement step is about 155 warp instructions (276 with masks searched for the r-th zero and a bit reader that carries its
// state) in one straight line; with branches for block ends and rare cases the two refinement waves of 1024 ImageNet-shaped images
// took 226 + 270 us, now 183 + 216.  (Registers held down to 112 for a sixth CTA an SM: 255 + 254.)  The three waves were 217 + 332 + 511
// us with coefficient planes; now 165 + 183 + 216.
#pragma once
#include <cuda_runtime.h>
#include <stddef.h>
#include <stdint.h>

#include "pcr_types.h"

namespace pcr {

constexpr int kErrCorrupt = -3;

#ifndef PCR_ENTROPY_WARPS
#define PCR_ENTROPY_WARPS 3
#endif
constexpr int kEntropyWarps = PCR_ENTROPY_WARPS;

constexpr int kRingWords = 16;       // words of the bitstream a lane of the interval kernels holds in shared memory

// A table entry as 16-byte loads: what a warp needs of several tables is requested before the first of it is used (a kernel's
// start is a chain of dependent loads).
template <class T> __device__ __forceinline__ T load_entry(const T* p) {
    static_assert(sizeof(T) % 16 == 0 && alignof(T) >= 16, "whole vectors");
    union U { uint4 v[sizeof(T) / 16]; T t; __device__ U() {} } u;
#pragma unroll
    for (size_t i = 0; i < sizeof(T) / 16; ++i) u.v[i] = __ldg(reinterpret_cast<const uint4*>(p) + i);
    return u.t;
}

struct ScanList { int32_t n; int32_t s[64]; };      // the scans one launch covers

// ---------------------------------------------------------------------------------------
// Tables of the interval kernels: one ScanTab per (scan, image, table), built once per decode beside the
// restart-interval index (the entropy warps then only copy 2.3 KB; building the table in every entropy
// warp took about 1000 instructions in front of a few hundred symbols).  An entry already holds what the
// scan's decode loop needs of a symbol:
//   bits 0..4   bits to skip: the code plus its extra bits (magnitude, sign, or run length)
//   AC refinement: bit 5 a new coefficient, bits 8..14 run of zeros, or 64 + run-length exponent for an end
//               of band (as a run it passes over every position there can be)
//   otherwise:  bits 5..8 magnitude size, bits 9..13 positions that the symbol moves on by (sequential DC: 1; an end of band of an
//               AC first pass: its run-length exponent), bit 15 end of band or block (beyond every position)
// 0 = a code longer than kTabBits bits, or no valid symbol of this kind of scan.
// ---------------------------------------------------------------------------------------
constexpr int kTabBits = 10;
struct __align__(16) ScanTab {
    uint16_t lut[1 << kTabBits];
    uint16_t first[8], cnt[8], idx[8];      // codes of kTabBits + 1 + j bits: first code, how many, index of the first value
                                            // (first[7]: the greatest 16 bits that begin with a code)
    uint8_t vals[256];
};
static_assert(sizeof(ScanTab) % 16 == 0, "tables are copied as 16-byte vectors");
enum { kTabDc = 0, kTabAcFirst = 1, kTabAcRefine = 2, kTabAcSeq = 3, kTabDcSeq = 4 };
constexpr uint32_t kEntEob = 0x8000u;         // first passes and sequential scans
constexpr uint32_t kEntEobRefine = 0x4000u;   // end of band of one block in a refinement

__device__ __forceinline__ uint32_t sym_entry(int kind, uint32_t len, uint32_t sym) {
    const uint32_t r = (sym >> 4) & 15u, sz = sym & 15u;
    if (kind == kTabDc) return sym > 15u ? 0u : ((len + sz) | (sz << 5));
    if (kind == kTabDcSeq) return sym > 15u ? 0u : ((len + sz) | (sz << 5) | (1u << 9));
    if (kind == kTabAcRefine) {
        if (sz > 1u) return 0u;
        if (sz || r == 15u) return (len + sz) | (sz << 5) | (r << 8);
        return (len + r) | ((64u + r) << 8);
    }
    if (sz || r == 15u) return (len + sz) | (sz << 5) | ((r + 1u) << 9);
    if (kind == kTabAcSeq) return r ? 0u : len | (1u << 9) | kEntEob;
    return (len + r) | (r << 9) | kEntEob;
}

// One warp builds one table in device memory from a DHT body (16 length counts, then the values in code order).
__device__ __forceinline__ void build_scan_tab(ScanTab* __restrict__ t, const uint8_t* __restrict__ dht, int kind, int lane,
                                               uint32_t* s_code, uint8_t* s_vals) {
    // s_code: [3][17] words of the warp: first code, first index, one past the last code left-aligned to kTabBits
    const uint32_t my = lane < 16 ? dht[lane] : 0u;
    uint32_t code = 0, p = 0;
    for (int l = 1; l <= 16; ++l) {
        const uint32_t c = __shfl_sync(0xffffffffu, my, l - 1);
        if (lane == 0) {
            s_code[l] = code; s_code[17 + l] = p;
            s_code[34 + l] = l <= kTabBits ? (code + c) << (kTabBits - l) : 0u;
            if (l > kTabBits) { const int j = l - kTabBits - 1; t->first[j] = (uint16_t)code; t->cnt[j] = (uint16_t)c; t->idx[j] = (uint16_t)p; }
        }
        code = (code + c) << 1;
        p += c;
    }
    if (lane == 0) t->first[7] = (uint16_t)((code >> 1) - 1u);
    const uint32_t nvals = min(p, 256u);
    for (uint32_t j = lane; j < 256u; j += 32) { const uint8_t v = j < nvals ? dht[16 + j] : 0; s_vals[j] = v; t->vals[j] = v; }
    __syncwarp();
    // every lane fills 32 consecutive entries; the code length only grows along them
    int l = 1;
    for (int g = 0; g < 4; ++g) {
        uint32_t w[4];
#pragma unroll
        for (int h = 0; h < 4; ++h) {
            uint32_t pair = 0;
#pragma unroll
            for (int b = 0; b < 2; ++b) {
                const uint32_t x = 32u * (uint32_t)lane + 8u * (uint32_t)g + 2u * (uint32_t)h + (uint32_t)b;
                while (l <= kTabBits && x >= s_code[34 + l]) ++l;
                uint32_t e = 0;
                if (l <= kTabBits) e = sym_entry(kind, (uint32_t)l, s_vals[(s_code[17 + l] + (x >> (kTabBits - l)) - s_code[l]) & 255u]);
                pair |= e << (16 * b);
            }
            w[h] = pair;
        }
        reinterpret_cast<uint4*>(t->lut)[4 * lane + g] = make_uint4(w[0], w[1], w[2], w[3]);
    }
}

// One table per warp: the tables of the listed scans of images img0 .. img0 + nimg - 1 of the processing order,
// slot by slot.  Follows the index warps of the same launch (see unstuff_index_kernel).
__device__ __forceinline__ void tables_warp(const Params& P, const ScanList& sl, int img0, int nimg, uint32_t w, int lane,
                                            uint32_t* s_code, uint8_t* s_vals) {
    const int slot = (int)(w & 3u);
    const uint32_t pair = w >> 2;
    const int s = sl.s[pair / (uint32_t)nimg];
    const ScanAux ax = P.saux[s];
    if (slot >= ax.ntab) return;
    const int img = (int)P.order[img0 + pair % (uint32_t)nimg];
    const ScanDesc& sd = P.scans[(size_t)s * P.N + img];
    const ScanScript sc = P.script[s];
    const bool seq = sc.Ss == 0 && sc.Se == 63;
    const uint32_t off = seq && slot >= 2 ? sd.tab_ac[slot - 2] : sd.tab_off[slot];
    if (!off) return;
    const int kind = seq ? (slot < 2 ? kTabDcSeq : kTabAcSeq) : (sc.Ss == 0 ? kTabDc : (sc.Ah == 0 ? kTabAcFirst : kTabAcRefine));
    build_scan_tab(P.tabs + ax.tab0 + (uint32_t)img * (uint32_t)ax.ntab + (uint32_t)slot, P.rec + off, kind, lane, s_code, s_vals);
}

// ---------------------------------------------------------------------------------------
// Restart-interval index and unstuffing, one warp per (listed scan, image).
// Copies the pair's entropy-coded bytes into P.ubuf with the zero byte after every 0xFF
// removed, bytes of each aligned group of four stored in reverse (big-endian words), at the
// same start offset as in the record.  Records, in offsets of that copy, the first byte of every
// restart interval (the byte after each RSTn marker) plus one final entry = end of data + 2, so
// interval j spans [seg[j], seg[j+1] - 2).
// Tile by tile of 512 bytes, lanes take 16-byte slices.  Stuffed zeros and markers are found four bytes at
// a time; one warp prefix sum places the slices; a lane writes the output words that begin in its slice,
// taking up to three bytes of the last one from its neighbour, so nothing goes through shared memory.  (The
// byte-by-byte form with a staging row took 680 warp instructions a tile, this one about 300; bound by the
// latency of one warp's tiles, up to 50 for a baseline JPEG of 25 KB.  1024 ImageNet-shaped images at k = 10 125 -> 68 us.)
// Blocks from index_blocks on build the lookup tables of the same scans and images (one warp per table).
// ---------------------------------------------------------------------------------------

// bit 7 of every byte that is zero
__device__ __forceinline__ uint32_t zero_bytes(uint32_t x) { return ~(((x & 0x7F7F7F7Fu) + 0x7F7F7F7Fu) | x) & 0x80808080u; }
// the bit 7s of four words' bytes as a 16-bit mask
__device__ __forceinline__ uint32_t byte_mask(uint32_t a, uint32_t b, uint32_t c, uint32_t d) {
    constexpr uint32_t k = 0x00204081u;
    return ((a * k) >> 28) | (((b * k) >> 28) << 4) | (((c * k) >> 28) << 8) | (((d * k) >> 28) << 12);
}
// removes byte i (0..15) of the sixteen in k[0..3] (later bytes move down)
__device__ __forceinline__ void drop_byte(uint32_t (&k)[4], uint32_t i) {
#pragma unroll
    for (uint32_t w = 0; w < 4; ++w) {
        const uint32_t moved = __funnelshift_r(k[w], w < 3 ? k[w + 1] : 0u, 8);
        const uint32_t m = i < 4u * w ? 0u : (i >= 4u * w + 4u ? 0xFFFFFFFFu : (1u << (8u * (i & 3u))) - 1u);   // bytes that stay
        k[w] = (k[w] & m) | (moved & ~m);
    }
}

// What a lane finds in its slice of a tile: its sixteen bytes at p, the word in front of them (its last byte counts) and the one behind.
// drop: stuffed zeros; mark: first bytes of restart markers; range: the bytes that lie inside the data [a, b).
struct SliceMarks { uint32_t range, drop, mark; };
__device__ __forceinline__ SliceMarks slice_marks(const uint4& v, uint32_t prev, uint32_t next, uint32_t p, uint32_t a, uint32_t b) {
    SliceMarks s;
    s.range = 0xFFFFu;
    if (p < a) s.range &= 0xFFFFu << (a - p);                        // (only the first slice)
    if (p + 16u > b) s.range &= p < b ? (1u << (b - p)) - 1u : 0u;
    const uint32_t k[4] = {v.x, v.y, v.z, v.w};
    uint32_t ff[4], rst[5];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        ff[i] = zero_bytes(~k[i]);
        rst[i] = zero_bytes((k[i] ^ 0xD0D0D0D0u) & 0xF8F8F8F8u);
    }
    rst[4] = zero_bytes((next ^ 0xD0D0D0D0u) & 0xF8F8F8F8u);
    const uint32_t pff = zero_bytes(~prev);
    s.drop = byte_mask(zero_bytes(k[0]) & __funnelshift_l(pff, ff[0], 8), zero_bytes(k[1]) & __funnelshift_l(ff[0], ff[1], 8),
                       zero_bytes(k[2]) & __funnelshift_l(ff[1], ff[2], 8), zero_bytes(k[3]) & __funnelshift_l(ff[2], ff[3], 8));
    s.mark = byte_mask(ff[0] & __funnelshift_r(rst[0], rst[1], 8), ff[1] & __funnelshift_r(rst[1], rst[2], 8),
                       ff[2] & __funnelshift_r(rst[2], rst[3], 8), ff[3] & __funnelshift_r(rst[3], rst[4], 8));
    // a zero in front of the data's first byte does not count; a marker's second byte has to lie inside the data
    if (p < a) s.drop &= ~(1u << (a - p));
    s.mark &= s.range & (p + 16u >= b ? s.range >> 1 : 0xFFFFu);
    return s;
}

// kSplit: a CTA takes a pair, its warps runs of the pair's tiles: they count what their run keeps and finds first, and meet; a word
// that two runs share is written byte by byte.  For launches of few pairs, whose time is that of the longest scan: all scans
// of 64 ImageNet-shaped images 38 -> 19 us, 1024 baseline JPEGs 124 -> 54 us.  The bytes are read twice, so launches that fill the
// machine, and short scans, keep a warp a pair (see launch_index_kernel): 1024 ImageNet-shaped images at k = 10 72 us, split 95.
constexpr int kIndexWarps = 8;
template <bool kSplit>
__global__ void __launch_bounds__(32 * kIndexWarps) unstuff_index_kernel(Params P, ScanList sl, int img0, int nimg, uint32_t index_blocks) {
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    if (blockIdx.x >= index_blocks) {
        __shared__ uint32_t s_code[kIndexWarps][51];
        __shared__ uint8_t s_vals[kIndexWarps][256];
        const uint32_t w = ((blockIdx.x - index_blocks) * blockDim.x + threadIdx.x) >> 5;
        if (w < 4u * (uint32_t)(sl.n * nimg)) tables_warp(P, sl, img0, nimg, w, lane, s_code[wid], s_vals[wid]);
        return;
    }
    const unsigned full = 0xffffffffu;
    const int pair = kSplit ? (int)blockIdx.x : (int)((blockIdx.x * blockDim.x + threadIdx.x) >> 5);
    if (pair >= sl.n * nimg) return;
    const int img = (int)P.order[img0 + pair % nimg];      // img0, nimg: a run of the processing order
    const ScanDesc& sd = P.scans[sl.s[pair / nimg] * P.N + img];
    const uint32_t a = sd.data_off, b = sd.data_end, nseg = sd.nseg;
    uint32_t* seg = P.seg_start + sd.seg_base;
    uint32_t* out = reinterpret_cast<uint32_t*>(P.ubuf);
    const uint4 zero4 = make_uint4(0, 0, 0, 0);
    uint32_t begin = a & ~15u, end_run = b;  // the run of tiles
    uint32_t found = 0, kept = 0;            // markers seen, bytes written so far (warp uniform)
    uint32_t held = 0, nheld = a & 3u;       // the bytes of an output word that the previous tile left incomplete (at first: that precede the data)
    uint32_t before = 0;                     // last byte of the previous tile, in the top byte
    bool shared_word = false;                // the run begins inside an output word that another run began
    bool last_run = true, first_run = true;
    if (kSplit) {
        const uint32_t tiles = (b - begin + 511u) / 512u, each = (tiles + kIndexWarps - 1) / kIndexWarps;
        begin = min(begin + 512u * each * (uint32_t)wid, b);
        if (begin < b) end_run = min(begin + 512u * each, b);        // (an empty run keeps end_run = begin = b)
        first_run = wid == 0;
        last_run = begin < b ? end_run == b : first_run;             // (no bytes at all: the first one)
        if (!first_run && begin < b) before = (uint32_t)P.rec[begin - 1u] << 24;
        uint32_t sum = 0, marks = 0, carry = before;                 // what the run keeps, the markers it finds
        uint4 ahead = zero4;
        if (begin + 16u * lane < b && begin < end_run) ahead = __ldg(reinterpret_cast<const uint4*>(P.rec + begin + 16u * lane));
        for (uint32_t p0 = begin; p0 < end_run; p0 += 512) {
            const uint32_t p = p0 + 16u * lane;
            const uint4 v = ahead;
            ahead = zero4;
            if (p + 512 < b) ahead = __ldg(reinterpret_cast<const uint4*>(P.rec + p + 512));
            uint32_t prev = __shfl_up_sync(full, v.w, 1), next = __shfl_down_sync(full, v.x, 1);
            const uint32_t next_tile = __shfl_sync(full, ahead.x, 0);
            if (lane == 0) prev = carry;
            if (lane == 31) next = next_tile;
            carry = __shfl_sync(full, v.w, 31);
            if (p < a && lane == 0) prev = 0;
            const SliceMarks s = slice_marks(v, prev, next, p, a, b);
            sum += (uint32_t)__popc(s.range & ~s.drop);
            marks += (uint32_t)__popc(s.mark);
        }
        __shared__ uint32_t s_kept[kIndexWarps], s_found[kIndexWarps];
        sum = __reduce_add_sync(full, sum); marks = __reduce_add_sync(full, marks);
        if (lane == 0) { s_kept[wid] = sum; s_found[wid] = marks; }
        __syncthreads();
        for (int w = 0; w < wid; ++w) { kept += s_kept[w]; found += s_found[w]; }
        if (begin >= b && !last_run) return;                         // whole warp
        if (!first_run) { nheld = 0; shared_word = ((a + kept) & 3u) != 0; }
    }
    if (lane == 0 && first_run) seg[0] = a;
    uint4 ahead = zero4;                     // the next tile is loaded while this one is worked on
    {
        const uint32_t p = begin + 16u * lane;
        if (p < b) ahead = __ldg(reinterpret_cast<const uint4*>(P.rec + p));   // chunks are padded to 16 bytes
    }
    for (uint32_t p0 = begin; p0 < end_run; p0 += 512) {
        const uint32_t p = p0 + 16u * lane;
        const uint4 v = ahead;
        ahead = zero4;
        if (p + 512 < b) ahead = __ldg(reinterpret_cast<const uint4*>(P.rec + p + 512));
        const bool last_tile = p0 + 512 >= b;
        uint32_t prev = __shfl_up_sync(full, v.w, 1), next = __shfl_down_sync(full, v.x, 1);
        const uint32_t next_tile = __shfl_sync(full, ahead.x, 0);
        if (lane == 0) prev = before;
        if (lane == 31) next = next_tile;
        before = __shfl_sync(full, v.w, 31);
        if (p < a && lane == 0) prev = 0;                            // (only the first slice; nothing precedes the data)
        uint32_t k[4] = {v.x, v.y, v.z, v.w};
        const SliceMarks sm = slice_marks(v, prev, next, p, a, b);
        uint32_t drop = sm.drop, mark = sm.mark;
        const uint32_t keep = sm.range & ~drop, c = (uint32_t)__popc(keep);
        uint32_t sum = c | ((uint32_t)__popc(mark) << 16);
        const uint32_t own = sum;
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            const uint32_t o = __shfl_up_sync(full, sum, d);
            if (lane >= d) sum += o;
        }
        const uint32_t tile = __shfl_sync(full, sum, 31);
        const uint32_t o = a + kept + ((sum - own) & 0xFFFFu);       // where the slice's first kept byte goes
        uint32_t ord = found + ((sum - own) >> 16);
        while (mark) {
            const uint32_t i = (uint32_t)__ffs((int)mark) - 1u;
            mark &= mark - 1u;
            ++ord;
            if (ord < nseg) seg[ord] = o + (uint32_t)__popc(keep & ((1u << i) - 1u)) + 2u;
        }
        // the kept bytes to the front
        if (p < a) {                                                 // bytes in front of the data
            const uint32_t n = a - p;
            if (n & 8u) { k[0] = k[2]; k[1] = k[3]; }
            if (n & 4u) { k[0] = k[1]; k[1] = k[2]; k[2] = k[3]; }
#pragma unroll
            for (int i = 0; i < 4; ++i) k[i] = __funnelshift_r(k[i], i < 3 ? k[i + 1] : 0u, 8u * (n & 3u));
            drop >>= n;
        }
        for (uint32_t m = drop & 0xFFFFu, n = 0; m; ++n) {
            const uint32_t i = (uint32_t)__ffs((int)m) - 1u;
            m &= m - 1u;
            drop_byte(k, i - n);
        }
        // and the neighbour's first bytes behind them (a slice that ends the data has none; what lies there is never decoded)
        const uint32_t follow = __shfl_down_sync(full, k[0], 1);
        uint32_t k4 = follow;
        if (c < 16u) {
            const uint32_t sh = 8u * (c & 3u), lo = follow << sh, hi = sh ? follow >> (32u - sh) : 0u, m = (1u << sh) - 1u;
#pragma unroll
            for (uint32_t w = 0; w < 4; ++w) k[w] = (c >> 2) == w ? (k[w] & m) | lo : (c >> 2) + 1u == w ? hi : k[w];
            k4 = hi;
        }
        // output words that begin in [o, o + c); one that the tile's end cuts off is held back for the next tile
        const uint32_t s = (0u - o) & 3u, w0 = (o + 3u) >> 2, end = o + c;
        const bool cut = lane == 31 && !last_tile && (end & 3u) != 0;
        const uint32_t w1 = cut ? end >> 2 : (end + 3u) >> 2;
        uint32_t word = 0;
#pragma unroll
        for (uint32_t j = 0; j < 4; ++j) {
            const uint32_t x = __funnelshift_r(k[j], j < 3 ? k[j + 1] : k4, 8u * s);
            if (w0 + j < w1) out[w0 + j] = __byte_perm(x, 0, 0x0123);
            if (w0 + j == w1) word = x;
        }
        if (kSplit && shared_word && p0 == begin && lane == 0)       // the bytes up to the first word that begins in this run
            for (uint32_t i = 0; i < min(s, c); ++i) P.ubuf[(o + i) ^ 3u] = (uint8_t)(k[0] >> (8u * i));
        if (lane == 0 && nheld) out[(o - nheld) >> 2] = __byte_perm(held | (k[0] << (8u * nheld)), 0, 0x0123);
        const uint32_t q = __shfl_sync(full, cut ? end & 3u : 0u, 31);
        held = __shfl_sync(full, word, 31) & ((1u << (8u * q)) - 1u);
        nheld = q;
        kept += tile & 0xFFFFu;
        found += tile >> 16;
    }
    if (kSplit && !last_run) {                                       // the bytes of the word that the next run goes on with
        if (lane == 0)
            for (uint32_t i = 0; i < nheld; ++i) P.ubuf[(a + kept - nheld + i) ^ 3u] = (uint8_t)(held >> (8u * i));
        return;
    }
    if (lane == 0) {
        seg[nseg] = a + kept + 2;
        if (found != nseg - 1) atomicMin(&P.status[img], kErrCorrupt);
    }
}

// ---------------------------------------------------------------------------------------
// One wave of scans.  Each warp takes one item; each lane one restart interval.
// ---------------------------------------------------------------------------------------
struct Geometry {
    uint32_t mx, my;          // MCU grid
    uint32_t bw[3], ubw[3], ubh[3];
    uint64_t coff[3];         // first block of each component (global block index)
    uint64_t loff[3];         // first block of each component counted inside its component
};

__device__ __forceinline__ Geometry make_geometry(const ImgDesc& im, const Params& P) {
    Geometry g;
    const uint32_t hs = (uint32_t)P.hs, vs = (uint32_t)P.vs, ny = hs * vs;      // luminance blocks per MCU
    g.mx = im.mx; g.my = im.my;
    g.bw[0] = hs * im.mx; g.bw[1] = g.bw[2] = im.mx;
    g.ubw[0] = (im.W + 7) / 8; g.ubh[0] = (im.H + 7) / 8;
    uint32_t cw = (im.W + hs - 1) / hs, ch = (im.H + vs - 1) / vs;
    g.ubw[1] = g.ubw[2] = (cw + 7) / 8; g.ubh[1] = g.ubh[2] = (ch + 7) / 8;
    g.coff[0] = im.blk_base;
    g.coff[1] = im.blk_base + (uint64_t)ny * im.mx * im.my;
    g.coff[2] = g.coff[1] + (uint64_t)im.mx * im.my;
    const uint64_t mcus_before = im.blk_base / (ny + (P.nc == 3 ? 2u : 0u));   // every image holds the same blocks per MCU
    g.loff[0] = ny * mcus_before; g.loff[1] = g.loff[2] = mcus_before;
    return g;
}

// Block number (in the planes) of block j of MCU (mrow, mcol) in an interleaved scan: the luminance
// blocks of the MCU row by row, then Cb, then Cr.  *comp = its component.
__device__ __forceinline__ uint64_t mcu_block(const Geometry& g, const Params& P, uint32_t mrow, uint32_t mcol, int j, int* comp) {
    const int ny = P.hs * P.vs;
    if (j < ny) {
        const uint32_t r = (uint32_t)j >> (P.hs - 1), c = (uint32_t)j & (uint32_t)(P.hs - 1);
        *comp = 0;
        return g.coff[0] + (uint64_t)((uint32_t)P.vs * mrow + r) * g.bw[0] + (uint32_t)P.hs * mcol + c;
    }
    const int cc = j - ny + 1;
    *comp = cc;
    return g.coff[cc] + (uint64_t)mrow * g.bw[cc] + mcol;
}

__device__ __forceinline__ uint64_t low_mask(int p) { return p >= 64 ? ~0ull : ((1ull << p) - 1ull); }

// ---------------------------------------------------------------------------------------
// Bit reader of the interval kernels.  The position is one number: bits counted from the first bit of a
// 16-byte group of the unstuffed copy.  The words around it lie in the lane's column of a ring in shared
// memory (two rows more than the ring: they repeat rows 0 and 1), so the window of the next 32 bits is two shared
// loads and a funnel shift, and skipping is an addition: no buffer, no refill branch.  All lanes top their
// columns up together.  `stop` is the first position at which a step may not begin (the ring runs out, the
// interval has ended, the lane has nothing to do): one comparison per step.
// Shared memory is addressed by 32-bit addresses (a generic pointer's window base was recomputed per access).
// ---------------------------------------------------------------------------------------
__device__ __forceinline__ uint32_t lds32(uint32_t a) { uint32_t v; asm volatile("ld.shared.u32 %0, [%1];" : "=r"(v) : "r"(a) : "memory"); return v; }
__device__ __forceinline__ uint32_t lds16(uint32_t a) { uint32_t v; asm volatile("ld.shared.u16 %0, [%1];" : "=r"(v) : "r"(a) : "memory"); return v; }
__device__ __forceinline__ uint32_t lds8(uint32_t a) { uint32_t v; asm volatile("ld.shared.u8 %0, [%1];" : "=r"(v) : "r"(a) : "memory"); return v; }
// nothing where `on` is false, without a branch
__device__ __forceinline__ void sts16_if(bool on, uint32_t a, uint32_t v) {
    asm volatile("{ .reg .pred p; setp.ne.u32 p, %2, 0; @p st.shared.u16 [%0], %1; }" : : "r"(a), "h"((uint16_t)v), "r"((uint32_t)on) : "memory");
}
__device__ __forceinline__ void lds128_if(bool on, uint32_t a, uint4& v) {
    asm volatile("{ .reg .pred p; setp.ne.u32 p, %5, 0; @p ld.shared.v4.u32 {%0, %1, %2, %3}, [%4]; }" : "+r"(v.x), "+r"(v.y), "+r"(v.z), "+r"(v.w) : "r"(a), "r"((uint32_t)on) : "memory");
}
__device__ __forceinline__ void sts32_if(bool on, uint32_t a, uint32_t v) {
    asm volatile("{ .reg .pred p; setp.ne.u32 p, %2, 0; @p st.shared.u32 [%0], %1; }" : : "r"(a), "r"(v), "r"((uint32_t)on) : "memory");
}
__device__ __forceinline__ void sts128_if(bool on, uint32_t a, const uint4& v) {
    asm volatile("{ .reg .pred p; setp.ne.u32 p, %5, 0; @p st.shared.v4.u32 [%0], {%1, %2, %3, %4}; }" : : "r"(a), "r"(v.x), "r"(v.y), "r"(v.z), "r"(v.w), "r"((uint32_t)on) : "memory");
}
__device__ __forceinline__ void stg16_if(bool on, void* a, uint32_t v) {
    asm volatile("{ .reg .pred p; setp.ne.u32 p, %2, 0; @p st.global.u16 [%0], %1; }" : : "l"(a), "h"((uint16_t)v), "r"((uint32_t)on) : "memory");
}
__device__ __forceinline__ void stg32_if(bool on, void* a, uint32_t v) {
    asm volatile("{ .reg .pred p; setp.ne.u32 p, %2, 0; @p st.global.u32 [%0], %1; }" : : "l"(a), "r"(v), "r"((uint32_t)on) : "memory");
}
__device__ __forceinline__ void stg64_if(bool on, void* a, uint32_t x, uint32_t y) {
    asm volatile("{ .reg .pred p; setp.ne.u32 p, %3, 0; @p st.global.v2.u32 [%0], {%1, %2}; }" : : "l"(a), "r"(x), "r"(y), "r"((uint32_t)on) : "memory");
}
__device__ __forceinline__ void stg128_if(bool on, void* a, const uint4& v) {
    asm volatile("{ .reg .pred p; setp.ne.u32 p, %5, 0; @p st.global.v4.u32 [%0], {%1, %2, %3, %4}; }" : : "l"(a), "r"(v.x), "r"(v.y), "r"(v.z), "r"(v.w), "r"((uint32_t)on) : "memory");
}
__device__ __forceinline__ uint2 lds64(uint32_t a) { uint2 v; asm volatile("ld.shared.v2.u32 {%0, %1}, [%2];" : "=r"(v.x), "=r"(v.y) : "r"(a) : "memory"); return v; }
__device__ __forceinline__ uint4 lds128(uint32_t a) { uint4 v; asm volatile("ld.shared.v4.u32 {%0, %1, %2, %3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "r"(a) : "memory"); return v; }
__device__ __forceinline__ void sts32(uint32_t a, uint32_t v) { asm volatile("st.shared.u32 [%0], %1;" : : "r"(a), "r"(v) : "memory"); }
__device__ __forceinline__ void sts16(uint32_t a, uint32_t v) { asm volatile("st.shared.u16 [%0], %1;" : : "r"(a), "h"((uint16_t)v) : "memory"); }
__device__ __forceinline__ void sts128(uint32_t a, const uint4& v) { asm volatile("st.shared.v4.u32 [%0], {%1, %2, %3, %4};" : : "r"(a), "r"(v.x), "r"(v.y), "r"(v.z), "r"(v.w) : "memory"); }
// shifts that give 0 for counts of as many bits as the word has, and more
__device__ __forceinline__ uint32_t shl0(uint32_t x, uint32_t n) { uint32_t y; asm("shl.b32 %0, %1, %2;" : "=r"(y) : "r"(x), "r"(n)); return y; }
__device__ __forceinline__ uint64_t shl0(uint64_t x, uint32_t n) { uint64_t y; asm("shl.b64 %0, %1, %2;" : "=l"(y) : "l"(x), "r"(n)); return y; }
__device__ __forceinline__ uint32_t shr0(uint32_t x, uint32_t n) { uint32_t y; asm("shr.u32 %0, %1, %2;" : "=r"(y) : "r"(x), "r"(n)); return y; }
// byte permutation with the selector's sign form (__byte_perm masks it out)
__device__ __forceinline__ uint32_t prmt(uint32_t a, uint32_t b, uint32_t s) { uint32_t y; asm("prmt.b32 %0, %1, %2, %3;" : "=r"(y) : "r"(a), "r"(b), "r"(s)); return y; }

// keeps a pointer in registers (instead of being put together from the kernel's parameters at every use)
template <class T> __device__ __forceinline__ void pin(T*& p) {
    size_t a = __cvta_generic_to_global(p);
    asm volatile("" : "+l"(a));
    p = static_cast<T*>(__cvta_global_to_generic(a));
}

struct LaneBits {
    uint32_t col;          // shared address of this lane's column: row r at col + 128 r
    const uint4* g4;       // the 16-byte group that position 0 lies in
    uint32_t pos, wr;      // next bit; next word to fetch (a multiple of 4)
    uint32_t limit;        // first bit behind the interval

    __device__ __forceinline__ void init(uint32_t column, const uint8_t* ubuf, uint32_t bstart, uint32_t bend) {
        col = column;
        g4 = reinterpret_cast<const uint4*>(ubuf) + (bstart >> 4);
        pos = 8u * (bstart & 15u);
        limit = pos + 8u * (bend - bstart);
        wr = 0;
        request();
    }
    __device__ __forceinline__ void put(uint32_t w, const uint4& v) {
        const uint32_t p = col + (w & (kRingWords - 1)) * 128u;
        sts32(p, v.x); sts32(p + 128u, v.y); sts32(p + 256u, v.z); sts32(p + 384u, v.w);
        if ((w & (kRingWords - 1)) == 0) { sts32(p + kRingWords * 128u, v.x); sts32(p + kRingWords * 128u + 128u, v.y); }
    }
    // Top-up (all lanes of the warp together): what the next one will store first is requested right after
    // the previous one, so that its latency passes beside the decode steps.
    uint4 va, vb;
    __device__ __forceinline__ void request() {
        const uint4* g = g4 + (wr >> 2);
        va = __ldg(g); vb = __ldg(g + 1);
    }
    __device__ __forceinline__ void topup(bool on) {
        const uint32_t room = on ? (kRingWords - (wr - (pos >> 5))) >> 2 : 0u;
        if (room > 0) put(wr, va);
        if (room > 1) put(wr + 4, vb);
        if (room > 2) put(wr + 8, __ldg(g4 + (wr >> 2) + 2));
        if (room > 3) put(wr + 12, __ldg(g4 + (wr >> 2) + 3));
        wr += 4u * room;
        if (on) request();
    }
    // steps may begin below this position: `words` words from the one the position lies in are in the ring
    __device__ __forceinline__ uint32_t ring_stop(uint32_t words) const { return 32u * (wr - min(wr, words - 1u)); }
    __device__ __forceinline__ uint32_t window(uint32_t at) const {
        const uint32_t p = col + ((at << 2) & ((kRingWords - 1) * 128u));
        return __funnelshift_l(lds32(p + 128u), lds32(p), at);    // (shift taken mod 32)
    }
};

// The same for the kernels whose CTAs follow 32 intervals at a time (pcr_refine.cuh, pcr_sequential.cuh): one warp reads along
// the columns while another fills them, for the round after; the ring is larger because the blocks of the round before
// are still read.  Two rows more than the ring repeat rows 0 and 1.
template <uint32_t kWords>
struct LaneRing {
    uint32_t col;          // shared address of this lane's column: row r at col + 128 r
    const uint4* g4;       // the 16-byte group that position 0 lies in
    uint32_t wr, last;     // next word to fetch (a multiple of 4); words from this one on are not needed
    uint4 v[4];
    uint32_t room;

    __device__ __forceinline__ void init(uint32_t column, const uint8_t* ubuf, uint32_t bstart, uint32_t bend) {
        col = column;
        g4 = reinterpret_cast<const uint4*>(ubuf) + (bstart >> 4);
        wr = 0;
        // (a step that begins at the end of the interval looks at four words; nothing is read far beyond)
        last = bend > bstart ? (8u * (bstart & 15u) + 8u * (bend - bstart)) / 32u + 8u : 0u;
    }
    // up to sixteen words are requested; those from bit `keep` on are still read
    __device__ __forceinline__ void request(uint32_t keep) {
        room = wr < last ? min((kWords - (wr - (keep >> 5))) >> 2, 4u) : 0u;
#pragma unroll
        for (uint32_t i = 0; i < 4; ++i)
            if (i < room) v[i] = __ldg(g4 + (wr >> 2) + i);
    }
    __device__ __forceinline__ void put() {
#pragma unroll
        for (uint32_t i = 0; i < 4; ++i) {
            if (i >= room) continue;
            const uint32_t w = (wr + 4u * i) & (kWords - 1), p = col + w * 128u;
            sts32(p, v[i].x); sts32(p + 128u, v[i].y); sts32(p + 256u, v[i].z); sts32(p + 384u, v[i].w);
            if (w == 0) { sts32(p + kWords * 128u, v[i].x); sts32(p + kWords * 128u + 128u, v[i].y); }
        }
        wr += 4u * room;
    }
};
// A position in such a column: the words it lies in and the one behind them, requested ahead of their use.
template <uint32_t kWords>
struct RingWords {
    uint32_t col, wa, wb, wc;
    __device__ __forceinline__ void load(uint32_t pos) {
        const uint32_t p = col + ((pos << 2) & ((kWords - 1) * 128u));
        wa = lds32(p); wb = lds32(p + 128u); wc = lds32(p + 256u);
    }
    __device__ __forceinline__ void load_behind(uint32_t pos) {
        const uint32_t p = col + ((pos << 2) & ((kWords - 1) * 128u));
        wb = lds32(p + 128u); wc = lds32(p + 256u);
    }
    __device__ __forceinline__ uint32_t window(uint32_t pos) const { return __funnelshift_l(wb, wa, pos); }     // its 32 bits (shifts taken mod 32)
    __device__ __forceinline__ uint32_t behind(uint32_t pos) const { return __funnelshift_l(wc, wb, pos); }     // the 32 after them
};
// Where the roles of a CTA's warps meet, each in a loop of its own (one loop with branches keeps every role's registers
// alive in all of them).
__device__ __forceinline__ void meet() { __syncwarp(); asm volatile("bar.sync 0;" : : : "memory"); }
// entry of a table for the code at the front of a window
__device__ __forceinline__ uint32_t tab_entry(uint32_t tab, uint32_t win) { return lds16(tab + ((win >> (31 - kTabBits)) & ((2u << kTabBits) - 2u))); }

// The signed value of the sz-bit magnitude field that ends bit `skip` of the window.
__device__ __forceinline__ int magnitude(uint32_t win, uint32_t skip, uint32_t sz) {
    // a leading 1: the field itself; a leading 0: one more than the field with ones in front of it
    const uint32_t x = shl0(win, skip - sz), ones = (uint32_t)~((int)x >> 31);
    return (int)(__funnelshift_l(x, ones, sz) - ones);        // (sz = 0: 0)
}

// A code longer than kTabBits bits (or an undefined one) of the table at shared address t: entry as above, 0 if
// there is no such symbol.
__device__ __forceinline__ uint32_t long_code(uint32_t t, uint32_t win, int kind) {
    const uint32_t w16 = win >> 16;
    if (w16 > lds16(t + (uint32_t)offsetof(ScanTab, first) + 14u)) return 0;      // (the usual case of a reading from a wrong position)
#pragma unroll 1
    for (uint32_t j = 0; j < 16 - kTabBits; ++j) {
        const uint32_t l = kTabBits + 1u + j, d = (w16 >> (16u - l)) - lds16(t + (uint32_t)offsetof(ScanTab, first) + 2u * j);
        if (d < lds16(t + (uint32_t)offsetof(ScanTab, cnt) + 2u * j))    // (index masked: damaged tables stay in bounds)
            return sym_entry(kind, l, lds8(t + (uint32_t)offsetof(ScanTab, vals) + ((lds16(t + (uint32_t)offsetof(ScanTab, idx) + 2u * j) + d) & 255u)));
    }
    return 0;
}

// select_in_byte.at[8 * b + r] = position of the (r+1)-th set bit of byte b
struct SelectTable {
    uint8_t at[2048 + 16];
    constexpr SelectTable() : at() {
        for (int b = 0; b < 256; ++b) {
            int r = 0;
            for (int i = 0; i < 8; ++i)
                if ((b >> i) & 1) at[8 * b + r++] = (uint8_t)i;
        }
    }
};
__device__ const __align__(16) SelectTable kSelect{};

// Still-zero positions of a refinement's band in a block, prepared for rank queries: the mask and, byte by
// byte, how many set bits lie in this byte and those below (at most 63, so that bytes can be compared with a
// rank by one subtraction per word; the last one is the number of set bits).
__device__ __forceinline__ uint4 rank_index(uint64_t z) {
    const uint32_t z0 = (uint32_t)z, z1 = (uint32_t)(z >> 32);
    auto bytes = [](uint32_t x) {
        x = x - ((x >> 1) & 0x55555555u);
        x = (x & 0x33333333u) + ((x >> 2) & 0x33333333u);
        return (x + (x >> 4)) & 0x0F0F0F0Fu;
    };
    const uint32_t c0 = bytes(z0), c1 = bytes(z1);
    const uint32_t low = (c0 * 0x01010101u) >> 24;
    return make_uint4(z0, z1, c0 * 0x01010101u, (c1 + low) * 0x01010101u);
}

// side data of a block of a first pass that reaches beyond position 7: the mask of its positions and where its
// values for positions 8..63 begin
__device__ __forceinline__ uint4 value_record(uint32_t m0, uint32_t m1, const int16_t* first) {
    const uint64_t a = reinterpret_cast<uint64_t>(first);
    return make_uint4(m0, m1, (uint32_t)a, (uint32_t)(a >> 32));
}

constexpr int kDecodeSteps = 16;     // decode steps between two top-ups of the rings
constexpr int kMaskQueue = 8;        // blocks whose masks a refinement lane holds ahead

// Shared memory of one warp (dynamic): two tables, the ring, a block's positions 0..7 per lane, and for waves with AC refinements the mask queue.
constexpr uint32_t kWarpRing = 2 * sizeof(ScanTab), kWarpHead = kWarpRing + (kRingWords + 2) * 128, kWarpQueue = kWarpHead + 512;
template <bool kRefine> __host__ __device__ constexpr uint32_t warp_bytes() { return kWarpQueue + (kRefine ? kMaskQueue * 512 : 0); }

// DC refinement scan s of one image: a bit per block, so bit j of a restart interval is block j in scan order and a thread
// does an MCU without a chain.  MCUs first, first + step, ...
__device__ __forceinline__ void dc_refine_image(const Params& P, int s, int img, uint32_t first, uint32_t step) {
    const ScanDesc sd = P.scans[(size_t)s * P.N + img];
    const ScanScript sc = P.script[s];
    const ImgDesc im = P.imgs[img];
    const Geometry g = make_geometry(im, P);
    const bool inter = sc.ncomp > 1;
    const int c0 = sc.comp[0];
    const uint32_t mcu_w = inter ? g.mx : g.ubw[c0];
    const uint32_t mcu_h = inter ? g.my : g.ubh[c0];
    const uint32_t total = mcu_w * mcu_h;
    const uint32_t bpm = inter ? (uint32_t)(P.hs * P.vs + 2) : 1u;   // blocks (= bits) per MCU
    const uint32_t* segtab = P.seg_start + sd.seg_base;
    const uint32_t* words = reinterpret_cast<const uint32_t*>(P.ubuf);
    const int p1 = 1 << sc.Al;
    bool bad = false;
    for (uint32_t m = first; m < total; m += step) {
        const uint32_t seg = sd.ri ? m / sd.ri : 0u;
        if (seg >= sd.nseg) { bad = true; continue; }
        const uint32_t m0 = seg * sd.ri;                       // 0 without restart markers
        const uint32_t bstart = segtab[seg], bend = segtab[seg + 1] - 2u;
        if (bstart < sd.data_off || bend > sd.data_end || bend < bstart) { bad = true; continue; }   // a missing marker left a hole
        const uint32_t bit = bpm * (m - m0);
        if (bit + bpm > 8u * (bend - bstart)) { bad = true; continue; }                             // the interval is too short
        const uint32_t p = 8u * (bstart & 3u) + bit;           // from the first bit of word bstart >> 2
        const uint32_t wi = (bstart >> 2) + (p >> 5);
        const uint32_t w0 = __ldg(words + wi), w1 = __ldg(words + wi + 1);   // the copy has spare bytes behind its end
        const uint32_t v = __funnelshift_l(w1, w0, p & 31u) >> (32u - bpm);  // the MCU's bits, first block in the top bit
        const uint32_t mrow = m / mcu_w, mcol = m - mrow * mcu_w;
#pragma unroll
        for (uint32_t j = 0; j < 6; ++j) {
            if (j >= bpm) break;
            if (!((v >> (bpm - 1u - j)) & 1u)) continue;
            uint64_t blk;
            int comp;
            if (!inter) blk = g.coff[c0] + (uint64_t)mrow * g.bw[c0] + mcol;
            else blk = mcu_block(g, P, mrow, mcol, (int)j, &comp);
            int16_t* dcv = P.dc + blk;                        // (no other scan of the wave writes it)
            *dcv = (int16_t)(*dcv | p1);
        }
    }
    if (bad) atomicMin(&P.status[img], kErrCorrupt);
}

// kRoi: restart intervals whose MCU rows lie wholly outside the MCU rows that the image's crop
// rectangle (P.roi) touches are not decoded (their blocks are never transformed).
// kRefine: the wave holds AC refinements (its warps then need a mask queue; the other waves run with less
// shared memory and fewer registers).
//
// A refinement step of a full machine is bound by its instructions (about 150): with the byte of the target counted in one word, rank and clamping in
// one instruction and the signs masked out of the positions, 1024 ImageNet-shaped images' last wave 217 -> 211 us.
//
// Pairs: a refinement that needs nothing but the masks of the refinement before it (same component, same band, same
// restart intervals) does not have to wait for that one's launch.  Lanes 0..15 of a warp decode sixteen intervals of the
// earlier scan, lanes 16..31 the same intervals of the later one, never further than the blocks their partner
// has finished; what is there is agreed upon at every top-up, where the warp meets anyway.  The chain of a
// row is then as long as the longer of its two scans instead of their sum.  (No rule chooses pairs in lanes, see pairs_pay; the overrides
// do.  Without the code for them the compiler allocates the step worse: last wave of 1024 ImageNet-shaped images 211 -> 215 us.)
//
// Blocks from runs.item_blocks on (kRefine) do the wave's DC refinement scans, which touch nothing the others do, in the
// shadow of the chains instead of in a launch behind them: 32 images of 32x32 at k = 10 72 -> 66 us, 96 mixed 4:4:4 images
// 457 -> 437 us, 1024 CelebA-shaped 498 -> 491 us.
//
// First passes: a step is one straight line of predicated instructions (with branches for block ends and long codes 300
// cycles an AC symbol alone on an SM, now 230), and what a warp needs of the tables is loaded at once (the start of a warp 6 to 10 k cycles,
// now 3.5 k).  After eight steps a warp whose lanes have all arrived tops up at once: with short intervals (32x32 images) it stands
// still for half of the steps otherwise.  DC alone of 1024 images 55 -> 40 us (pairs of luminance blocks stored together, MCUs
// without a branch inside).
// Three forms (which: first_pass_form).  kFirstFull packs the stores (see below): those of 1024 ImageNet-shaped images at k = 5 took
// half of the load/store units' time, 197 us against 172 (before: 206); 64 images 44 us without packing, 66 with it.  kFirstShort is held
// to registers for eight CTAs an SM instead of five: where intervals are short, what counts is how many warps start side by side.  Decode of
// 32x32 images at k = 5, five and eight CTAs: 1024 73.4 and 71.5 us, 2048 110 and 104, 4096 178 and 167; of ImageNet-shaped images 64 80
// and 80, 256 118 and 123, 1024 352 and 379.
enum { kFirstFew = 0, kFirstFull = 1, kFirstShort = 2 };     // (see first_pass_form)
template <bool kRoi, bool kRefine, int kForm>
__global__ void __launch_bounds__(32 * kEntropyWarps, kRefine ? 4 : (kForm == kFirstShort ? 8 : 1)) entropy_kernel(Params P, ItemRuns runs) {
    constexpr bool kPack = kForm == kFirstFull;
    extern __shared__ __align__(16) uint8_t s_entropy[];
    __shared__ __align__(16) uint8_t s_sel[kRefine ? sizeof(SelectTable) : 16];
    const int wid = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const uint32_t it = blockIdx.x * kEntropyWarps + wid;
    if (kRefine && blockIdx.x >= runs.item_blocks) {          // whole block
        const uint32_t b = blockIdx.x - runs.item_blocks, chunk = b % runs.dc_chunks, i = b / runs.dc_chunks;
        dc_refine_image(P, runs.dc_s[i / runs.dc_images], (int)P.order[runs.dc_pos0 + i % runs.dc_images],
                        chunk * 32u * kEntropyWarps + threadIdx.x, runs.dc_chunks * 32u * kEntropyWarps);
        return;
    }
    if (kRefine) {
        for (int i = threadIdx.x; i < (int)sizeof(SelectTable) / 16; i += 32 * kEntropyWarps)
            reinterpret_cast<uint4*>(s_sel)[i] = __ldg(reinterpret_cast<const uint4*>(kSelect.at) + i);
        __syncthreads();
    }
    if (it >= runs.end[runs.n - 1]) return;                   // whole warp
    int run_no = 0;
    while (it >= runs.end[run_no]) ++run_no;
    const Item item = P.items[runs.first[run_no] + it - (run_no ? runs.end[run_no - 1] : 0u)];
    const bool half = kRefine && item.pair && lane >= 16;     // this lane decodes the later scan of the pair
    const uint32_t li = kRefine && item.pair ? (uint32_t)lane & 15u : (uint32_t)lane;
    // tables: a DC scan may use two tables of one image; an AC item may span two images
    const bool two_images = item.next != 0;
    const uint32_t si1 = two_images ? item.next - 1u : item.si + item.pair;
    const uint32_t N = (uint32_t)P.N, s0 = item.si / N, s1 = si1 / N;
    const int s = (int)(half ? s1 : s0);
    const ScanDesc sd0 = load_entry(P.scans + item.si), sd1 = load_entry(P.scans + si1);
    const ScanAux ax0 = load_entry(P.saux + s0), ax1 = load_entry(P.saux + s1);
    const ScanScript sc = load_entry(P.script + s);
    const ImgDesc im0 = load_entry(P.imgs + item.si % N), im1 = load_entry(P.imgs + si1 % N);
    const bool dc = sc.Ss == 0;              // a DC first pass (DC refinement scans have no items)
    const ScanAux ax = half ? ax1 : ax0;
    // From here on no lane leaves before the warp does: lanes without work just stay `done`.
    bool done = li >= item.count;
    const uint32_t rem0 = sd0.nseg - item.seg0;               // restart intervals left in the first image
    const uint32_t which = half || (two_images && li >= rem0) ? 1u : 0u;
    uint32_t seg = two_images && li >= rem0 ? li - rem0 : item.seg0 + li;
    const ScanDesc sd = which ? sd1 : sd0;
    const int img = (int)((which ? si1 : item.si) % N);
    if (seg >= sd.nseg) { done = true; seg = 0; }
    const ImgDesc im = which ? im1 : im0;
    const Geometry g = make_geometry(im, P);

    const bool inter = sc.ncomp > 1;
    const int c0 = sc.comp[0];
    const uint32_t mcu_w = inter ? g.mx : g.ubw[c0];
    const uint32_t mcu_h = inter ? g.my : g.ubh[c0];
    const uint32_t total = mcu_w * mcu_h;
    const uint32_t m0 = sd.ri ? seg * sd.ri : 0;
    const uint32_t m1 = sd.ri ? min(m0 + sd.ri, total) : total;
    const unsigned full = 0xffffffffu;
    if (kRoi) {
        if (!done && m1 > m0) {
            const CropRect rc = P.roi[img];
            const uint32_t mh = 8u * (uint32_t)P.vs;                       // pixel rows of an MCU row
            const uint32_t ph = (inter || c0 != 0) ? mh : 8u;              // pixel rows per MCU row of this scan
            const uint32_t lo = mh * (rc.y0 / mh), hi = mh * ((rc.y0 + rc.h + mh - 1u) / mh);
            const uint32_t r0 = m0 / mcu_w, r1 = (m1 - 1u) / mcu_w;
            if ((r1 + 1u) * ph <= lo || r0 * ph >= hi) done = true;
        }
        if (__all_sync(full, done)) return;                               // nothing of this item is wanted
    }
    const uint32_t mem = (uint32_t)__cvta_generic_to_shared(s_entropy) + (uint32_t)wid * warp_bytes<kRefine>();
    const uint32_t* segtab = P.seg_start + sd.seg_base;
    uint32_t bstart = __ldg(segtab + seg);
    uint32_t bend = __ldg(segtab + seg + 1) - 2;
    {
        const uint32_t t0 = ax0.tab0 + (item.si % N) * (uint32_t)ax0.ntab;
        const uint32_t t1 = dc ? t0 + 1u : ax1.tab0 + (si1 % N) * (uint32_t)ax1.ntab;
        const bool second = two_images || item.pair || (dc && sd0.tab_off[1]);
        const uint4* a = reinterpret_cast<const uint4*>(P.tabs + t0);
        const uint4* b = reinterpret_cast<const uint4*>(P.tabs + t1);
        constexpr int n = (int)(sizeof(ScanTab) / 16);
        uint4 v[(n + 31) / 32];
#pragma unroll
        for (int i = 0; i < (n + 31) / 32; ++i) if (lane + 32 * i < n) v[i] = __ldg(a + lane + 32 * i);
#pragma unroll
        for (int i = 0; i < (n + 31) / 32; ++i) if (lane + 32 * i < n) sts128(mem + 16 * (lane + 32 * i), v[i]);
        if (second) {
#pragma unroll
            for (int i = 0; i < (n + 31) / 32; ++i) if (lane + 32 * i < n) v[i] = __ldg(b + lane + 32 * i);
#pragma unroll
            for (int i = 0; i < (n + 31) / 32; ++i) if (lane + 32 * i < n) sts128(mem + 16 * (n + lane + 32 * i), v[i]);
        }
    }
    bool bad = false;
    if (!done && (bstart < sd.data_off || bend > sd.data_end || bend < bstart)) {   // a missing marker left a hole
        bad = true; done = true;
    }
    if (done) { bstart = sd.data_off; bend = sd.data_off; }
    LaneBits br;
    br.init(mem + kWarpRing + 4u * lane, P.ubuf, bstart, bend);
    const int Al = sc.Al;
    if (m0 >= m1) done = true;
    RingWords<kRingWords> W;
    W.col = br.col;

    if (dc) {
        // ---- DC first pass: one MCU per step, its blocks unrolled
        const int ny = P.hs * P.vs, bpm = inter ? ny + 2 : 1;       // blocks per MCU
        uint32_t m = m0, mrow = m0 / mcu_w, mcol = m0 % mcu_w;
        int pred0 = 0, pred1 = 0, pred2 = 0;
        // block numbers inside the image: the MCU's first luminance block (or the scan's own component) and its chroma blocks
        const uint32_t hs = inter ? (uint32_t)P.hs : 1u, vs = inter ? (uint32_t)P.vs : 1u, bw0 = g.bw[inter ? 0 : c0];
        const uint32_t y_off = inter ? 0u : (uint32_t)(g.coff[c0] - im.blk_base), c_off = (uint32_t)(g.coff[1] - im.blk_base), c_step = g.mx * g.my;
        int16_t* dcp = P.dc + im.blk_base;
        pin(dcp);
        const uint32_t t0 = mem + (sd.slots & 1u) * (uint32_t)sizeof(ScanTab), t1 = mem + ((sd.slots >> 2) & 1u) * (uint32_t)sizeof(ScanTab),
                       t2 = mem + ((sd.slots >> 4) & 1u) * (uint32_t)sizeof(ScanTab);      // tables of the luminance (or the scan's own) and the chroma blocks
        for (;;) {
            br.topup(!done);
            __syncwarp(full);
            if (__all_sync(full, done)) break;
            // an MCU's symbols need at most 6 * 31 bits: seven words and the windows' second and third one
            const uint32_t stop = done ? 0u : min(br.ring_stop(9), br.limit + 1u);
            // (The chain: entry -> next window -> next entry; everything else is requested or done beside it.)
            W.load(br.pos);
            uint32_t win = W.window(br.pos), e = tab_entry(t0, win);
#pragma unroll 1
            for (int t = 0; t < kDecodeSteps / 4; ++t) {
                if (br.pos >= stop || m >= m1 || bad) continue;
                const uint32_t yb = y_off + (vs * mrow) * bw0 + hs * mcol, cb = c_off + mrow * g.mx + mcol;
                // Straight through the MCU; one that holds a code longer than the table's index is gone over again (long codes
                // looked up), so that nothing branches inside.
                const uint32_t pos0 = br.pos, win0 = win, e0 = e;
                const int was0 = pred0, was1 = pred1, was2 = pred2;
                bool again = false, longs = false;
                do {
                    if (again) {
                        longs = true; again = false;
                        br.pos = pos0; win = win0; e = e0; pred0 = was0; pred1 = was1; pred2 = was2;
                        W.load_behind(br.pos);
                    }
                    int before = 0;
#pragma unroll
                    for (int j = 0; j < 6; ++j) {
                        if (j >= bpm) break;
                        const bool luma = j < ny || !inter, cbl = !luma && j == ny;
                        if (longs && e == 0) { e = long_code(luma ? t0 : (cbl ? t1 : t2), win, kTabDc); bad = bad || e == 0; }      // (then nothing moves on)
                        again = again || e == 0;
                        const uint32_t skip = e & 31u, sz = e >> 5, behind = W.behind(br.pos), after = j + 1 >= bpm || j + 1 < ny ? t0 : (j + 1 == ny ? t1 : t2);
                        const uint32_t next = __funnelshift_l(behind, win, skip);
                        e = tab_entry(after, next);
                        br.pos += skip;
                        W.load_behind(br.pos);
                        const int d = magnitude(win, skip, sz);
                        win = next;
                        if (luma) {
                            pred0 += d;
                            if (hs == 1u) dcp[yb + (uint32_t)j * bw0] = (int16_t)(pred0 << Al);
                            else if (j & 1) *reinterpret_cast<uint32_t*>(dcp + yb + (uint32_t)(j >> 1) * bw0) = __byte_perm((uint32_t)(before << Al), (uint32_t)(pred0 << Al), 0x5410);
                            before = pred0;
                        } else if (cbl) dcp[cb] = (int16_t)((pred1 += d) << Al);
                        else dcp[cb + c_step] = (int16_t)((pred2 += d) << Al);
                    }
                } while (again && !longs);
                ++m;
                if (++mcol == mcu_w) { mcol = 0; ++mrow; }
            }
            __syncwarp(full);
            bad = bad || br.pos > br.limit;
            done = done || bad || m >= m1;
        }
    } else {
        const uint32_t tab = mem + which * (uint32_t)sizeof(ScanTab);
        const uint32_t c = (uint32_t)c0, Ss = (uint32_t)sc.Ss, Se = (uint32_t)sc.Se;
        const uint32_t bw = g.bw[c];
        const uint32_t wrap = bw - mcu_w + 1;              // step of the block index at the end of a block row
        uint32_t m = m0, bcol = m0 % mcu_w;
        uint32_t bi = (m0 / mcu_w) * bw + bcol;            // block index inside the image's component
        if (!kRefine || sc.Ah == 0) {
            // ---- AC first pass: one Huffman symbol per step
            uint64_t* auxp = P.aux + ax.base + g.loff[c] * ax.stride;
            int16_t* headp = P.head + g.coff[c] * 8;
            pin(auxp); pin(headp);
            const bool lists = ax.stride == 2u;            // the band reaches beyond position 7
            // kPack: values leave four at a time (the list is one run per interval), a block's positions 1..7 in whole words where
            // the band holds whole words of them: a lane's store is a sector of its own, and the stores of five scans are
            // what a full machine waits for.
            int16_t* const vlist = P.vals + 4ull * bstart;
            uint32_t nv = 0, nv0 = 0, v01 = 0, v23 = 0;     // values so far, those before the block, the last four
            const uint32_t hlo = max(Ss, 1u), hhi = min(Se, 7u);
            // how the head leaves: 0 by coefficient, 1 all of it, 2 its first six positions, 3 its last two
            const int heads = !kPack ? 0 : (hlo == 1u && hhi == 7u ? 1 : (hlo == 1u && hhi == 5u ? 2 : (hlo == 6u && hhi == 7u ? 3 : 0)));
            const uint32_t slot = mem + kWarpHead + 16u * lane;
            sts128(slot, make_uint4(0, 0, 0, 0));
            uint32_t wrap_m = m + mcu_w - bcol;             // the first block of the next block row
            uint32_t M0 = 0, M1 = 0, k = Ss;
            for (;;) {
                br.topup(!done);
                __syncwarp(full);
                if (__all_sync(full, done)) break;
                uint32_t stop = done ? 0u : min(br.ring_stop(3), br.limit + 1u);
                W.load(br.pos);
                uint32_t win = W.window(br.pos), raw = tab_entry(tab, win);
                // A step is one straight line but for block rows that end.  An entry of zero moves nothing on: lanes that have
                // arrived somewhere, and those that stand at a code longer than the table's index, wait.
#pragma unroll 1
                for (int t = 0; t < kDecodeSteps; t += 8) {
#pragma unroll 4
                    for (int q = 0; q < 8; ++q) {
                        const uint32_t e = br.pos < stop ? raw : 0u, behind = W.behind(br.pos);
                        const uint32_t skip = e & 31u, sz = (e >> 5) & 15u, next = __funnelshift_l(behind, win, skip);
                        raw = tab_entry(tab, next);
                        br.pos += skip;
                        W.load_behind(br.pos);
                        k += e >> 9;                           // behind the coefficient (an end of band: beyond every position)
                        const uint32_t at = k - 1u;
                        const bool coef = sz && k <= Se + 1u, far = coef && k > 8u;
                        const int val = magnitude(win, skip, sz) << Al;
                        const bool end = k > Se;               // the block is finished (also where nothing of the band is left)
                        int16_t* const h = headp + 8u * (uint64_t)bi;
                        M0 |= shl0(coef ? 1u : 0u, at); M1 |= shl0(coef ? 1u : 0u, at - 32u);
                        nv += far ? 1u : 0u;
                        if (kPack) {
                            v01 = far ? __byte_perm(v01, v23, 0x5432) : v01;
                            v23 = far ? __byte_perm(v23, (uint32_t)val, 0x5432) : v23;
                            stg64_if(far && (nv & 3u) == 0, vlist + nv - 4u, v01, v23);
                        } else stg16_if(far, vlist + nv - 1u, (uint32_t)val);
                        if (heads == 0) stg16_if(coef && !far, h + at, (uint32_t)val);
                        else {
                            sts16_if(coef && !far, slot + 2u * at, (uint32_t)val);
                            const uint4 v = lds128(slot);
                            if (heads == 1) stg128_if(end && (M0 & 0xFEu), h, v);
                            else if (heads == 2) { stg64_if(end && (v.x | v.y), h, v.x, v.y); stg32_if(end && v.z, h + 4, v.z); }
                            else stg32_if(end && v.w, h + 6, v.w);
                            sts128_if(end, slot, make_uint4(0, 0, 0, 0));
                        }
                        const bool some = end && (M0 | M1) != 0;
                        if (lists) stg128_if(some, auxp + (uint64_t)bi * 2, value_record(M0, M1, vlist + nv0));
                        else stg64_if(some, auxp + bi, M0, M1);
                        if (sz && k > Se + 1u) { bad = true; stop = 0; }           // a coefficient behind the band
                        // an end of band may leave the following blocks empty too
                        const uint32_t r = (e >> 9) & 15u, adv = e & kEntEob ? __funnelshift_l(shl0(win, skip - r), 1u, r) : 1u;   // 2^r + the r bits that end the symbol
                        m += end ? adv : 0u; bi += end ? adv : 0u;
                        k = end ? Ss : k; nv0 = end ? nv : nv0;
                        M0 = end ? 0u : M0; M1 = end ? 0u : M1;
                        if (m >= wrap_m && m < m1) {           // (only where an interval holds several rows)
                            const uint32_t row = m / mcu_w;
                            bi = row * bw + (m - row * mcu_w); wrap_m = (row + 1u) * mcu_w;
                        }
                        stop = m >= m1 ? 0u : stop;
                        win = next;
                    }
                    if (raw == 0 && br.pos < stop) {           // (taken by the next step)
                        raw = long_code(tab, win, kTabAcFirst);
                        if (raw == 0) { bad = true; stop = 0; }        // no such symbol: the lane ends here
                    }
                    if (!kRefine && !__any_sync(full, br.pos < stop)) break;      // (in the other form it costs registers that the refinements need)
                }
                __syncwarp(full);
                bad = bad || br.pos > br.limit;
                done = done || bad || m >= m1;
            }
            // the last values (what lies behind them up to the group of four belongs to this interval too)
            if (kPack && (nv & 3u)) {
                for (uint32_t p = nv & 3u; p < 4u; ++p) { v01 = __byte_perm(v01, v23, 0x5432); v23 >>= 16; }
                *reinterpret_cast<uint2*>(vlist + (nv & ~3u)) = make_uint2(v01, v23);
            }
        } else {
            // ---- AC refinement: one Huffman symbol, or one block of an end-of-band run, per step.
            // A run of r zeros ends at the (r+1)-th still-zero position not yet passed.  Positions are
            // therefore counted by rank: T = rank of the target among the block's still-zero positions; its
            // position comes from the byte counts (how many are at most T tells the byte, a table the bit
            // inside it), with no search whose length depends on the data.  Position minus rank counts the
            // non-zero positions below, so the number of correction bits that follow a symbol is the
            // difference of two such values.
            const uint64_t band = low_mask((int)Se + 1) & ~low_mask((int)Ss);
            const uint32_t band0 = (uint32_t)band, band1 = (uint32_t)(band >> 32);
            // history masks: the union of up to four earlier scans' (one or two in most scripts)
            const uint64_t* src[4];
            uint32_t st[4];
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const ScanAux x = P.saux[ax.src[q < ax.nsrc ? q : 0]];
                src[q] = P.aux + x.base + g.loff[c] * x.stride; st[q] = x.stride;
            }
            const bool two = ax.nsrc > 1, more = ax.nsrc > 2;
            uint64_t* outp = P.aux + ax.base + g.loff[c] * 4ull;
            pin(outp);
            const uint32_t queue = mem + kWarpQueue + 16u * lane;       // block m at queue + 512 (m % kMaskQueue)
            uint32_t sel = (uint32_t)__cvta_generic_to_shared(s_sel);
            asm volatile("" : "+r"(sel));                              // (kept in a register)
            uint32_t hm = m, hbi = bi;                                 // fetch cursor of the queue
            uint32_t wrap_m = m + mcu_w - bcol, hwrap_m = wrap_m;      // the first block of the next block row
            uint32_t eobrun = 0;
            uint4 Z = make_uint4(0, 0, 0, 0);                          // the block's still-zero positions (see rank_index)
            uint32_t zi = 0, ep = Ss;                                  // zero positions passed; position minus rank of the last
            uint32_t s0 = 0, s1 = 0, N0 = 0, N1 = 0, G0 = 0, G1 = 0;   // correction bits, new positions, positive ones
            bool fresh = true;                                         // the block's entry has not been taken from the queue yet
            auto take = [&]() { Z = lds128(queue + ((m & (kMaskQueue - 1)) << 9)); };
            // (the masks are requested ahead like the words of the stream)
            uint64_t ha[4], hb[4];
            uint32_t hlimit = half ? m : m1;                           // blocks whose masks are there
            uint32_t asked = hm;                                       // one past the blocks whose masks have been requested
            auto request = [&]() {
                uint32_t b = hbi, mm = hm, wm = hwrap_m;
                asked = min(hm + 4u, hlimit);
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    ha[q] = hb[q] = 0;
                    if (mm < hlimit) {
                        ha[q] = src[0][(uint64_t)b * st[0]];
                        if (two) hb[q] = src[1][(uint64_t)b * st[1]];
                    }
                    ++b; ++mm;
                    if (mm == wm) { b += wrap - 1u; wm += mcu_w; }
                }
            };
            if (!done) request();
            for (;;) {
                br.topup(!done);
                uint32_t want = done ? 0u : min((uint32_t)kMaskQueue - (hm - m), hlimit - hm);
                if (half) want = min(want, asked - hm);                // (what the partner finished since is requested below)
#pragma unroll
                for (int q = 0; q < kMaskQueue; ++q) {
                    if (q == 4 && !__any_sync(full, want > 4u)) break;
                    if (q < (int)want) {
                        uint64_t x;
                        if (q < 4) x = ha[q] | hb[q];
                        else { x = src[0][(uint64_t)hbi * st[0]]; if (two) x |= src[1][(uint64_t)hbi * st[1]]; }
                        if (more) x |= src[2][(uint64_t)hbi * st[2]] | src[3][(uint64_t)hbi * st[3]];
                        sts128(queue + ((hm & (kMaskQueue - 1)) << 9), rank_index(~x & band));
                        ++hm; ++hbi;
                        if (hm == hwrap_m) { hbi += wrap - 1u; hwrap_m += mcu_w; }
                    }
                }
                __syncwarp(full);
                if (item.pair) {                                       // how far the partner is (all lanes take part)
                    const uint32_t pm = __shfl_sync(full, m, (int)li);
                    const bool stuck = __shfl_sync(full, (int)(done && m < m1), (int)li) != 0;     // ... and that it will get no further
                    if (half) {
                        hlimit = min(pm, m1);
                        if (stuck && m >= hlimit) done = true;
                    }
                }
                if (__all_sync(full, done)) break;
                if (!done) {
                    request();
                    if (fresh && m < hm) take();
                }
                // a step reads the window at its start and, at most 31 bits on, two words (three for more than
                // 32 correction bits)
                uint32_t stop = done || m >= hm ? 0u : min(br.ring_stop(4), br.limit + 1u);
                W.load(br.pos);
                uint32_t win = W.window(br.pos), raw = tab_entry(tab, win);
                bool late = false, rare = false;               // the step before passed more than 31 bits; a long code, or more than 32 correction bits
                auto target = [&](uint32_t e, uint32_t nz, uint32_t& T, uint32_t& k, uint32_t& n) {
                    T = __viaddmin_u32(zi, e >> 8, nz);        // the rank of the target; nz = behind the band
                    const uint32_t tt = T * 0x01010101u + 0x80808080u;
                    const uint32_t j = (uint32_t)__popc(((tt - Z.z) & 0x80808080u) | (((tt - Z.w) >> 1) & 0x40404040u));
                    const uint32_t zb = __byte_perm(Z.x, Z.y, j) & 255u, cj = prmt(Z.z, Z.w, j - 1u) & 255u;   // (j = 0: no byte below, the selector's sign form gives 0)
                    k = 8u * j + lds8(sel + 8u * zb + T - cj);
                    k = T < nz ? k : Se + 1u;
                    n = k - T - ep;                            // correction bits behind the symbol
                };
                // what a symbol does once it is known how many correction bits it has
                auto apply = [&](bool act, uint32_t e, uint32_t nz, uint32_t T, uint32_t k, uint32_t n) {
                    const uint32_t skip = e & 31u, d = act ? skip + n : 0u;
                    const uint32_t isnew = act && T < nz ? (e >> 5) & 1u : 0u, n0 = shl0(isnew, k), n1 = shl0(isnew, k - 32u);
                    const uint32_t plus = (uint32_t)((int)shl0(win, skip - 1u) >> 31);     // the sign that ends the symbol (a new coefficient's)
                    N0 |= n0; N1 |= n1;
                    G0 |= n0 & plus; G1 |= n1 & plus;
                    const bool end = act && k >= Se;           // block finished
                    const uint32_t x = (e >> 8) & 15u, run = __funnelshift_l(shl0(win, skip - x), 1u, x);   // of an end of band: blocks it covers (2^x + the x bits that end it)
                    const uint32_t left = (eobrun ? eobrun : (e >= kEntEobRefine ? run : 1u)) - 1u;
                    uint64_t* const o = outp + (uint64_t)bi * 4;
                    stg128_if(end, o, make_uint4((~Z.x & band0) | N0, (~Z.y & band1) | N1, s0, s1));
                    stg128_if(end, o + 2, make_uint4(N0, N1, G0, G1));
                    eobrun = end ? left : eobrun;
                    m += end ? 1u : 0u;
                    const bool row = end && m == wrap_m;
                    bi += row ? wrap : (end ? 1u : 0u); wrap_m += row ? mcu_w : 0u;
                    zi = end ? 0u : (act ? T + 1u : zi); ep = end ? Ss : (act ? ep + n : ep);
                    s0 = end ? 0u : s0; s1 = end ? 0u : s1; N0 = end ? 0u : N0; N1 = end ? 0u : N1; G0 = end ? 0u : G0; G1 = end ? 0u : G1;
                    // (only an entry that is there: waiting lanes look ranks up in their Z too, and a slot's old contents may lead
                    // outside the table; the finished block's entry does not)
                    lds128_if(end && m < hm, queue + ((m & (kMaskQueue - 1)) << 9), Z);
                    stop = m < hm ? stop : 0u;                 // also at the interval's end: hm is at most m1
                    return d;
                };
                // A step is one straight line that every lane walks; what is rare waits for the end of eight.
#pragma unroll 1
                for (int t = 0; t < kDecodeSteps; t += 8) {
#pragma unroll 1
                    for (int q = 0; q < 8; ++q) {
                        const bool wanted = br.pos < stop && !late && !rare;
                        const uint32_t nz = Z.w >> 24, e = eobrun ? kEntEobRefine : raw;    // (this block lies inside an end-of-band run)
                        const uint32_t behind = W.behind(br.pos);
                        if (late) win = W.window(br.pos);
                        uint32_t T, k, n;
                        target(e, nz, T, k, n);
                        const bool act = wanted && e != 0 && n <= 32u;
                        rare = rare || (wanted && !act);
                        const uint32_t bits = act ? n : 0u, corr = __funnelshift_l(behind, win, e & 31u);
                        s1 = __funnelshift_lc(s0, s1, bits);
                        s0 = shl0(s0, bits) | shr0(corr, 32u - bits);
                        const uint32_t d = apply(act, e, nz, T, k, n);
                        win = __funnelshift_l(behind, win, d);
                        raw = tab_entry(tab, win);
                        br.pos += d;
                        late = d > 31u;
                        W.load(br.pos);
                    }
                    if (late) { win = W.window(br.pos); raw = tab_entry(tab, win); late = false; }
                    if (rare) {
                        rare = false;
                        const uint32_t nz = Z.w >> 24;
                        uint32_t e = eobrun ? kEntEobRefine : raw, T, k, n;
                        if (e == 0) e = long_code(tab, win, kTabAcRefine);
                        target(e, nz, T, k, n);
                        if (e == 0) { bad = true; stop = 0; }  // no such symbol: the lane ends here
                        else {
                            const uint32_t at = br.pos + (e & 31u), cw = br.window(at);
                            if (n > 32u) {
                                s1 = (cw >> (64u - n)) | (s0 << (n - 32u));
                                s0 = __funnelshift_l(br.window(at + 32u), cw, n - 32u);
                            } else {
                                s1 = __funnelshift_lc(s0, s1, n);
                                s0 = shl0(s0, n) | shr0(cw, 32u - n);
                            }
                            br.pos += apply(true, e, nz, T, k, n);
                            W.load(br.pos);
                            win = W.window(br.pos); raw = tab_entry(tab, win);
                        }
                    }
                    if (t == 0 && __ballot_sync(full, br.pos < stop) == 0) break;
                }
                __syncwarp(full);
                fresh = m >= hm;
                bad = bad || br.pos > br.limit;
                done = done || bad || m >= m1;
            }
        }
    }
    if (bad) atomicMin(&P.status[img], kErrCorrupt);
}

}  // namespace pcr
