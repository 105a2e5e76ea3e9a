// Pixel stage of the PCR decoder: dequantise -> 8x8 inverse DCT -> 2x2 chroma replication ->
// YCbCr to RGB -> crop -> packed uint8 store, fused in one kernel.
//
// Integer specification (the CPU oracle implements the same function from its definition):
//   F = coef * Q                                              (int32)
//   pass 1, columns:  T(y,u) = (sum_v M[y][v] F(v,u) + 2^11) >> 12
//   pass 2, rows:     s(y,x) = (sum_u M[x][u] T(y,u) + 2^15) >> 16,  sample = clamp(s + 128)
//   M[n][k] = round(8192 * c_k * cos((2n+1) k pi / 16)), c_0 = 1/sqrt 2, i.e. +-K_j with
//   K_j = round(8192 cos(j pi / 16)); all sums modulo 2^32, shifts arithmetic.
//   The sums are evaluated here by an even/odd butterfly, which is exact integer algebra on
//   the same matrix, so the result is identical to the plain matrix product.
//   R = clamp(Y + ((91881 cr + 32768) >> 16)), G = clamp(Y + ((-22553 cb - 46802 cr + 32768) >> 16)),
//   B = clamp(Y + ((116130 cb + 32768) >> 16)) with cb, cr = sample - 128 of chroma (x>>1, y>>1).
#pragma once
#include <cuda_bf16.h>
#include <cuda_fp16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include "pcr_types.h"

namespace pcr {

constexpr int kStagePitch = 3 * 128 + 16;     // bytes per staged RGB row (+ spare, keeps rows 16-byte aligned)

// Chroma sampling of a record as a template code: luminance blocks per MCU (horizontal, vertical),
// components, and the MCUs (across) and MCU rows of one work unit.  A unit is 128 pixels wide and its blocks
// fill whole warps, each of one kind (4:2:0: two warps of luminance, one of chroma): one thread per block.
enum { kSamp420 = 0, kSamp422 = 1, kSamp440 = 2, kSamp444 = 3, kSampGrey = 4 };
template <int kSamp> struct Sampling;
template <> struct Sampling<kSamp420> { static constexpr int HS = 2, VS = 2, NC = 3, U = 8, R = 2; };
template <> struct Sampling<kSamp422> { static constexpr int HS = 2, VS = 1, NC = 3, U = 8, R = 2; };
template <> struct Sampling<kSamp440> { static constexpr int HS = 1, VS = 2, NC = 3, U = 16, R = 1; };
template <> struct Sampling<kSamp444> { static constexpr int HS = 1, VS = 1, NC = 3, U = 16, R = 2; };
template <> struct Sampling<kSampGrey> { static constexpr int HS = 1, VS = 1, NC = 1, U = 16, R = 4; };
template <int kSamp> __host__ __device__ constexpr int unit_threads() {
    using S = Sampling<kSamp>;
    return S::U * S::R * (S::HS * S::VS + (S::NC == 3 ? 2 : 0));
}
constexpr int sampling_code(int hs, int vs, int nc) {
    return nc == 1 ? kSampGrey : (hs == 2 ? (vs == 2 ? kSamp420 : kSamp422) : (vs == 2 ? kSamp440 : kSamp444));
}
constexpr uint32_t kUnitMcus[5] = {8, 8, 16, 16, 16}, kUnitRows[5] = {2, 2, 1, 2, 4};

// zigzag position -> natural index, by walking the anti-diagonals
struct ZigzagTable {
    uint8_t nat[64];
    constexpr ZigzagTable() : nat() {
        int r = 0, c = 0;
        for (int k = 0; k < 64; ++k) {
            nat[k] = (uint8_t)(r * 8 + c);
            if (((r + c) & 1) == 0) {
                if (c == 7) ++r; else if (r == 0) ++c; else { --r; ++c; }
            } else {
                if (r == 7) ++c; else if (c == 0) ++r; else { ++r; --c; }
            }
        }
    }
};
__device__ constexpr ZigzagTable kZigzag{};

// One 8-point pass on the integer matrix M (see the header comment) of a vector with x[N] .. x[7] = 0:
// out[n] = (sum_k M[n][k] x[k] + rnd) >> kShift.  The compiler drops the terms of zeros.
template <int kShift, int N>
__device__ __forceinline__ void idct(const uint32_t (&x)[N], uint32_t rnd, uint32_t (&o)[8]) {
    constexpr uint32_t K1 = 8035, K2 = 7568, K3 = 6811, K4 = 5793, K5 = 4551, K6 = 3135, K7 = 1598;
    const uint32_t x4 = N > 4 ? x[N > 4 ? 4 : 0] : 0u, x5 = N > 5 ? x[N > 5 ? 5 : 0] : 0u, x6 = N > 6 ? x[N > 6 ? 6 : 0] : 0u, x7 = N > 7 ? x[N > 7 ? 7 : 0] : 0u;
    const uint32_t a0 = K4 * (x[0] + x4) + rnd, a1 = K4 * (x[0] - x4) + rnd;
    const uint32_t b0 = K2 * x[2] + K6 * x6, b1 = K6 * x[2] - K2 * x6;
    const uint32_t e0 = a0 + b0, e3 = a0 - b0, e1 = a1 + b1, e2 = a1 - b1;
    const uint32_t o0 = K1 * x[1] + K3 * x[3] + K5 * x5 + K7 * x7;
    const uint32_t o1 = K3 * x[1] - K7 * x[3] - K1 * x5 - K5 * x7;
    const uint32_t o2 = K5 * x[1] - K1 * x[3] + K7 * x5 + K3 * x7;
    const uint32_t o3 = K7 * x[1] - K5 * x[3] + K3 * x5 - K1 * x7;
    o[0] = (uint32_t)((int)(e0 + o0) >> kShift); o[7] = (uint32_t)((int)(e0 - o0) >> kShift);
    o[1] = (uint32_t)((int)(e1 + o1) >> kShift); o[6] = (uint32_t)((int)(e1 - o1) >> kShift);
    o[2] = (uint32_t)((int)(e2 + o2) >> kShift); o[5] = (uint32_t)((int)(e2 - o2) >> kShift);
    o[3] = (uint32_t)((int)(e3 + o3) >> kShift); o[4] = (uint32_t)((int)(e3 - o3) >> kShift);
}

// Zigzag positions whose row and column are both below n, as a 64-bit mask, and the words of four positions that hold them.
constexpr uint64_t corner_mask(int n) {
    ZigzagTable z{};
    uint64_t m = 0;
    for (int k = 0; k < 64; ++k)
        if ((z.nat[k] >> 3) < n && (z.nat[k] & 7) < n) m |= 1ull << k;
    return m;
}
constexpr int corner_words(int n) {
    int w = 0;
    for (int k = 0; k < 64; ++k)
        if ((corner_mask(n) >> k) & 1u) w = k / 4 + 1;
    return w;
}
template <int N> struct Corner {
    static constexpr int n = N, words = corner_words(N);
    static constexpr uint64_t mask = corner_mask(N);
};
static_assert((corner_mask(4) & 0xFFu) == 0xFFu, "positions 0..7 lie in the smallest corner");

// Two samples as a pair of 16-bit numbers, {clamp((a >> 16) + 128), clamp((b >> 16) + 128)} with clamp to 0..255: the
// upper halves by one permutation, then two packed operations.  The upper end is cut before 128 is added, so
// nothing wraps for sums near the ends of the 32-bit range.
__device__ __forceinline__ uint32_t sample_pair(uint32_t a, uint32_t b) {
    return __viaddmax_s16x2(__vmins2(__byte_perm(a, b, 0x7632), 0x007F007Fu), 0x00800080u, 0u);
}
// bytes {lo(a), hi(a), lo(b), hi(b)} of two pairs
__device__ __forceinline__ uint32_t pair_bytes(uint32_t a, uint32_t b) { return __byte_perm(a, b, 0x6420); }

struct Image { uint32_t W, H, mx, my; uint64_t blk_base, out_off; };
template <int kBpm> __device__ __forceinline__ Image image_of(const Unit& u) { return Image{u.W, u.H, u.mx, u.my, kBpm * u.mcus, u.out_off}; }

// Where a decode's coefficients lie (built per call for the chosen k, see CoefLists in pcr_types.h): the
// DC plane, the head plane (positions 1..7), and per first pass and component the masks and values of the rest.
// The refinements' side data is folded in here, in scan order.  Nothing of this is written back: the
// lists of all decoded scans stay as they are, and whoever needs blocks expands them again.
//
// Expands block `blk` of the planes (number `local` inside its component) into this thread's line in shared
// memory: position p is the int16 at line + (p >> 2) * 8 * kT + 2 * (p & 3) (kT threads' lines interleaved by
// eight bytes: every thread keeps to its own banks, whatever position it addresses).
// A correction moves a non-zero coefficient away from zero by 2^Al if its bit Al is still clear; a
// new coefficient is +-2^Al.
// Returns (for the whole warp, which calls it together) whether every coefficient lies in the low kCorner x kCorner
// corner; then only the words of the line that hold the corner are written.  kCorner = 8: not asked for.
template <int kT, bool kRefine, int kCorner>
__device__ __forceinline__ bool expand_block(const Params& P, const CoefLists& cl, int comp, uint64_t blk, uint64_t local, uint8_t* line, bool valid) {
    constexpr int kPitch = 8 * kT;
    auto at = [&](int pos) { return reinterpret_cast<int16_t*>(line + 2 * pos + (pos >> 2) * (kPitch - 8)); };
    const int nfirst = cl.n_first[comp], nref = kRefine ? cl.n_refine[comp] : 0;
    // all of the block's loads are requested before the first is used
    const uint4 zero4 = make_uint4(0, 0, 0, 0);
    uint4 head = zero4, rec = zero4;
    uint32_t dc = 0;
    const uint64_t at_rec = cl.sequential ? blk : local;
    uint4 a0 = zero4, b0 = zero4, a1 = zero4, b1 = zero4;
    if (valid) {
        head = __ldg(reinterpret_cast<const uint4*>(P.head + blk * 8));
        dc = __ldg(reinterpret_cast<const uint16_t*>(P.dc) + blk) & cl.dc_mask[comp];
        if (nfirst > 0) rec = __ldg(reinterpret_cast<const uint4*>(P.aux + cl.first[comp][0]) + at_rec);
        if (kRefine) {
            if (nref > 0) { const uint4* o = reinterpret_cast<const uint4*>(P.aux + cl.refine[comp][0]) + 2 * local; a0 = __ldg(o); b0 = __ldg(o + 1); }
            if (nref > 1) { const uint4* o = reinterpret_cast<const uint4*>(P.aux + cl.refine[comp][1]) + 2 * local; a1 = __ldg(o); b1 = __ldg(o + 1); }
        }
    }
    bool small = false;
    constexpr int kCornerWords = Corner<kCorner>::words;
    if (kCorner < 8) {
        // positions that are non-zero (a refinement's mask holds those before it too)
        constexpr uint64_t kMask = Corner<kCorner>::mask;
        uint32_t n0 = rec.x | a0.x | a1.x, n1 = rec.y | a0.y | a1.y;
        if (valid) {
            for (int i = 1; i < nfirst; ++i) { const uint2 r = __ldg(reinterpret_cast<const uint2*>(reinterpret_cast<const uint4*>(P.aux + cl.first[comp][i]) + at_rec)); n0 |= r.x; n1 |= r.y; }
            if (kRefine)
                for (int i = 2; i < nref; ++i) { const uint2 r = __ldg(reinterpret_cast<const uint2*>(reinterpret_cast<const uint4*>(P.aux + cl.refine[comp][i]) + 2 * local)); n0 |= r.x; n1 |= r.y; }
        }
        small = !__any_sync(0xffffffffu, ((n0 & ~(uint32_t)kMask) | (n1 & ~(uint32_t)(kMask >> 32))) != 0);
    }
    if (!valid) return small;
#pragma unroll
    for (int w = 2; w < kCornerWords; ++w) *reinterpret_cast<uint2*>(line + w * kPitch) = make_uint2(0, 0);
    if (!small) {
#pragma unroll
        for (int w = kCornerWords; w < 16; ++w) *reinterpret_cast<uint2*>(line + w * kPitch) = make_uint2(0, 0);
    }
    const uint4 hm = cl.head_mask[comp];           // positions that no decoded scan covers may hold a later scan's values
    *reinterpret_cast<uint2*>(line) = make_uint2((head.x & hm.x) | dc, head.y & hm.y);
    *reinterpret_cast<uint2*>(line + kPitch) = make_uint2(head.z & hm.z, head.w & hm.w);
    for (int i = 0; i < nfirst; ++i) {
        if (i) rec = __ldg(reinterpret_cast<const uint4*>(P.aux + cl.first[comp][i]) + at_rec);
        const int16_t* v = reinterpret_cast<const int16_t*>(((uint64_t)rec.w << 32) | rec.z);
#pragma unroll
        for (int half = 0; half < 2; ++half) {
            uint32_t m = half ? rec.y : rec.x & ~0xFFu;
            uint8_t* const lh = line + half * 8 * kPitch;
            while (m) {                            // four at a time, so that their loads are in flight together
                int pos[4], x[4];
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    pos[e] = m ? __ffs((int)m) - 1 : -1;
                    m &= m - 1u;                   // (0 stays 0)
                    if (pos[e] >= 0) x[e] = __ldg(v++);
                }
#pragma unroll
                for (int e = 0; e < 4; ++e)
                    if (pos[e] >= 0) *reinterpret_cast<int16_t*>(lh + (pos[e] >> 2) * kPitch + 2 * (pos[e] & 3)) = (int16_t)x[e];
            }
        }
    }
    if (kRefine) {
        for (int i = 0; i < nref; ++i) {
            const int p1 = cl.p1[comp][i];
            uint4 a = i == 0 ? a0 : a1, b = i == 0 ? b0 : b1;    // {mask, corrections}, {new, signs}
            if (i > 1) { const uint4* o = reinterpret_cast<const uint4*>(P.aux + cl.refine[comp][i]) + 2 * local; a = __ldg(o); b = __ldg(o + 1); }
            // corrections: the coefficients that were non-zero before the scan, in zigzag order, take the
            // correction bits in reading order (as many as there are such positions, the last one in bit 0);
            // the walk through each half ends with its last set bit (in 32 bits, and without a branch around a correction: 1024 ImageNet-shaped
            // images at k = 10 347 -> 334 us)
            const uint32_t h0 = a.x & ~b.x, h1 = a.y & ~b.y;
            // (none of them: a shift by 64, which gives 0; the side data of a damaged image may have bits all the same)
            const int n0 = __popc(h0);
            const uint64_t cc = shl0(((uint64_t)a.w << 32) | a.z, 64u - (uint32_t)(n0 + __popc(h1)));
#pragma unroll
            for (int half = 0; half < 2; ++half) {
                uint32_t h = half ? h1 : h0, c = half ? (uint32_t)((cc << n0) >> 32) : (uint32_t)(cc >> 32) & (n0 ? ~0u << (32 - n0) : 0u);
                while (c) {
                    const int pos = 32 * half + __ffs((int)h) - 1;
                    h &= h - 1u;
                    int16_t* e = at(pos);
                    const int v = *e;
                    if ((int)c < 0 && (v & p1) == 0) *e = (int16_t)(v >= 0 ? v + p1 : v - p1);
                    c += c;
                }
            }
#pragma unroll
            for (int half = 0; half < 2; ++half) {
                uint32_t nw = half ? b.y : b.x;
                const uint32_t sg = half ? b.w : b.z;
                while (nw) {
                    const int bit = __ffs((int)nw) - 1;
                    nw &= nw - 1u;
                    *at(32 * half + bit) = (int16_t)(((sg >> bit) & 1u) ? p1 : -p1);
                }
            }
        }
    }
    return small;
}

// kMode: 0 = all 64 coefficients sit in the block's 128-byte line (pcr_pixels_noalloc); 1 = coefficient lists
// (expand_block); 3 = no decoded scan reaches beyond position 7 and none is a refinement: the head plane and
// the DC plane are all there is.
// kRefine: AC refinements among the decoded scans (kMode 1).
// kRoi: only work units, and in them MCU rows, that touch their image's crop rectangle (P.roi) are processed.
//
// kStage serves triangle chroma upsampling, which needs chroma samples of neighbouring work
// units: 0 = everything in one launch (2x2 replication); 1 = chroma pass: the chroma blocks are
// transformed and their samples stored in P.chroma, nothing else; 2 = pixel pass: luminance blocks
// as in 0, chroma samples with a one-sample border read back from P.chroma, every pixel's chroma = (9 own +
// 3 horizontally nearer + 3 vertically nearer + 1 diagonal + 8) >> 4, neighbours clamped to the MCU-padded
// planes.  3 = no pixels: the expanded blocks are written to P.planes (pcr_coeffs).
// kCoarse: every AC scan so far left low bits out (or kMode 3), so nearly all coefficients sit in the low 4x4 corner: warps
// whose blocks have none outside it take a transform of that corner, which needs fewer registers, and the
// kernel is compiled for more CTAs an SM (the full transform spills then).  1024 ImageNet-shaped images at
// k = 5: 240 -> 166 us; for a record at full precision both would cost time (baseline 281 -> 418 us, k = 10 348 -> 478).
// kSamp: the record's chroma sampling (see Sampling); the triangle filter (kStage 1, 2) exists for
// 4:2:0 only.  A greyscale record has no chroma: every pixel is (Y, Y, Y).
//
// One thread per block through the whole transform; the chroma samples go through shared memory, the luminance
// samples stay in the registers of the thread that made them and meet the chroma there, two pixels
// per instruction (16-bit pairs).  Bound by instruction issue (integer multiplications and additions of the transform, about
// 0.65 of the slots, 0.73 with kCoarse).  Pixel stage of 1024 ImageNet-shaped images, before (lines of 128 bytes per block, colour as a
// step of its own) and now: k = 5 348 -> 164 us, k = 10 562 -> 334 us, baseline 351 -> 272 us.
template <bool kRefine, int kMode, bool kRoi = false, int kStage = 0, int kSamp = kSamp420, bool kCoarse = false>
__global__ void __launch_bounds__(unit_threads<kSamp>(), (kCoarse ? 1152 : 672) / unit_threads<kSamp>())
pixel_kernel(Params P, CoefLists cl, uint8_t* __restrict__ out) {
    using S = Sampling<kSamp>;
    constexpr int HS = S::HS, VS = S::VS, NC = S::NC, U = S::U, R = S::R, kT = unit_threads<kSamp>();
    constexpr int kYCols = HS * U;                            // luminance blocks per block row of a unit
    constexpr int kYBlocks = R * VS * kYCols;                  // luminance blocks of a unit
    constexpr int kBpm = HS * VS + (NC == 3 ? 2 : 0);          // blocks per MCU
    constexpr int kPxW = 8 * HS, kPxH = 8 * VS, kRows = R * kPxH;   // pixels per MCU, pixel rows of a unit
    static_assert(kPxW * U == 128 && kT % 32 == 0 && kYBlocks % 32 == 0, "a unit is 128 pixels wide, its warps are of one kind");
    static_assert(kStage == 0 || kStage == 3 || kSamp == kSamp420, "triangle upsampling is built for 4:2:0");
    constexpr int kLineBytes = kMode == 1 ? 128 * kT : 16, kStageBytes = kRows * kStagePitch;
    // the lines are read before, the staged rows written after the barrier behind the transform
    __shared__ __align__(16) uint8_t s_mem[kStage == 3 || kLineBytes > kStageBytes ? kLineBytes : kStageBytes];
    __shared__ __align__(16) uint8_t s_c[2][8 * R][8 * U];
    __shared__ __align__(16) int32_t s_q[3][64];
    __shared__ uint8_t s_ct[kStage == 2 ? 2 : 1][kStage == 2 ? 8 * R + 2 : 1][kStage == 2 ? 8 * U + 2 : 1];   // chroma tile + border
    uint8_t* const s_stage = s_mem;

    const int tid = threadIdx.x;
    const Unit un = P.units[blockIdx.x];
    const Image im = image_of<kBpm>(un);
    const int nm = min(U, (int)im.mx - (int)un.mcol0);                // MCUs across in this unit
    int r_lo = 0, r_hi = min(R, (int)im.my - (int)un.mrow);           // its MCU rows that are wanted
    if (kRoi) {
        const CropRect r = P.roi[un.img];
        const int ux0 = kPxW * un.mcol0, y0 = (int)(r.y0 / kPxH) - (int)un.mrow, y1 = (int)((r.y0 + r.h - 1u) / kPxH) + 1 - (int)un.mrow;
        r_lo = max(r_lo, y0); r_hi = min(r_hi, y1);
        if (r_lo >= r_hi || ux0 >= (int)(r.x0 + r.w) || ux0 + kPxW * nm <= (int)r.x0) return;      // whole CTA: nothing of this unit is wanted
    }
    // (the quantisers are requested before the block's loads and stored behind them)
    constexpr int kQLoads = (96 + kT - 1) / kT;
    uint32_t q2[kQLoads];
    if (kStage != 3) {
#pragma unroll
        for (int i = 0; i < kQLoads; ++i)
            if (tid + i * kT < 96) q2[i] = __ldg(reinterpret_cast<const uint32_t*>(P.qtab + (size_t)un.img * 192) + tid + i * kT);
    }
    // ---- thread j owns block j: the unit's luminance block rows, then its Cb rows, then its Cr rows
    int comp = 0, yr, yc;                 // component, block row / column inside the unit
    uint64_t blk, local;                  // block number in the planes / inside its component
    bool valid;
    if (NC == 1 || tid < kYBlocks) {
        yr = tid / kYCols; yc = tid % kYCols;
        valid = yc < HS * nm && yr >= VS * r_lo && yr < VS * r_hi && kStage != 1;
        local = (uint64_t)(VS * un.mrow + yr) * (HS * im.mx) + HS * un.mcol0 + yc;
        blk = im.blk_base + local;
        local += (uint64_t)(HS * VS) * (un.mcus);
    } else {
        const int i = tid - kYBlocks;
        comp = 1 + i / (U * R);
        yr = i % (U * R) / U; yc = i % U;
        valid = yc < nm && yr >= r_lo && yr < r_hi && kStage != 2;
        local = (uint64_t)(un.mrow + yr) * im.mx + un.mcol0 + yc;
        blk = im.blk_base + (uint64_t)(HS * VS + comp - 1) * im.mx * im.my + local;
        local += un.mcus;
    }
    uint8_t* const line = s_mem + 8 * tid;
    constexpr int kCorner = kCoarse ? 4 : 8;          // the corner that a shorter transform is made for
    bool small = kMode == 3;              // every coefficient of the warp's blocks lies in it
    if (kMode == 1) small = expand_block<kT, kRefine, kCorner>(P, cl, comp, blk, local, line, valid);
    if (kStage == 3) {
        if (valid) {
            uint4* dst = reinterpret_cast<uint4*>(P.planes + blk * 64);
#pragma unroll
            for (int q = 0; q < 8; ++q) {
                if (small && 2 * q >= Corner<kCorner>::words) { dst[q] = make_uint4(0, 0, 0, 0); continue; }
                const uint2 lo = *reinterpret_cast<const uint2*>(line + (2 * q) * 8 * kT), hi = small && 2 * q + 1 >= Corner<kCorner>::words ? make_uint2(0, 0) : *reinterpret_cast<const uint2*>(line + (2 * q + 1) * 8 * kT);
                dst[q] = make_uint4(lo.x, lo.y, hi.x, hi.y);
            }
        }
        return;
    }
#pragma unroll
    for (int i = 0; i < kQLoads; ++i)
        if (tid + i * kT < 96) *reinterpret_cast<int2*>(&s_q[0][0] + 2 * (tid + i * kT)) = make_int2((int)(q2[i] & 0xFFFFu), (int)(q2[i] >> 16));
    __syncthreads();                  // the quantisers are there
    uint32_t yp[32];                      // a luminance block's samples, two per word (row y: words 4y .. 4y + 3)
    if (valid) {
        const int4* q4 = reinterpret_cast<const int4*>(&s_q[comp][0]);
        uint4 head = make_uint4(0, 0, 0, 0);
        if (kMode == 3) {
            const uint4 hm = cl.head_mask[comp];
            head = __ldg(reinterpret_cast<const uint4*>(P.head + blk * 8));
            head = make_uint4((head.x & hm.x) | (__ldg(reinterpret_cast<const uint16_t*>(P.dc) + blk) & cl.dc_mask[comp]), head.y & hm.y, head.z & hm.z, head.w & hm.w);
        }
        const uint4* dense = reinterpret_cast<const uint4*>(P.planes + blk * 64);
        auto word = [&](int w) {                                      // zigzag positions 4w .. 4w + 3
            if (kMode == 3) return w == 0 ? make_uint2(head.x, head.y) : (w == 1 ? make_uint2(head.z, head.w) : make_uint2(0, 0));
            if (kMode == 0) return __ldg(reinterpret_cast<const uint2*>(dense) + w);
            return *reinterpret_cast<const uint2*>(line + w * 8 * kT);
        };
        auto dequantise = [&](uint2 c2, const int4& q, uint32_t (&f)[4]) {
            f[0] = (uint32_t)((int)(short)(c2.x & 0xFFFFu) * q.x); f[1] = (uint32_t)(((int)c2.x >> 16) * q.y);
            f[2] = (uint32_t)((int)(short)(c2.y & 0xFFFFu) * q.z); f[3] = (uint32_t)(((int)c2.y >> 16) * q.w);
        };
        // Pass 1: columns (two fraction bits kept).  Pass 2: rows; the final shift by 16 takes the upper halves, the
        // level shift is part of the clamping.  A warp whose blocks have nothing outside the low N x N corner takes N of the
        // columns and N terms of each sum.
        auto transform = [&](auto corner) {
            constexpr int N = decltype(corner)::n, kWords = kMode == 3 ? 2 : Corner<N>::words;
            constexpr uint64_t kIn = Corner<N>::mask;
            uint32_t v[N][N];                                         // [column][row]
#pragma unroll
            for (int k = 0; k < 64; ++k)
                if (k >= 4 * kWords && ((kIn >> k) & 1u)) v[kZigzag.nat[k] & 7][kZigzag.nat[k] >> 3] = 0;
#pragma unroll
            for (int w = 0; w < kWords; ++w) {
                uint32_t f[4];
                dequantise(word(w), q4[w], f);
#pragma unroll
                for (int e = 0; e < 4; ++e)
                    if ((kIn >> (4 * w + e)) & 1u) v[kZigzag.nat[4 * w + e] & 7][kZigzag.nat[4 * w + e] >> 3] = f[e];
            }
            uint32_t t[8][N];
#pragma unroll
            for (int u = 0; u < N; ++u) {
                uint32_t o[8];
                idct<12, N>(v[u], 1u << 11, o);
#pragma unroll
                for (int y = 0; y < 8; ++y) t[y][u] = o[y];
            }
#pragma unroll
            for (int y = 0; y < 8; ++y) {
                uint32_t r[8];
                idct<0, N>(t[y], 1u << 15, r);
#pragma unroll
                for (int p = 0; p < 4; ++p) yp[4 * y + p] = sample_pair(r[2 * p], r[2 * p + 1]);
            }
        };
        if (kMode == 3 || (kCorner < 8 && kMode == 1 && small)) transform(Corner<kCorner>{});
        else if (kMode != 3) transform(Corner<8>{});
        if (NC == 3 && comp != 0) {
            uint8_t* dst;
            int pitch;
            if (kStage == 1) {
                pitch = 8 * (int)im.mx;
                dst = P.chroma + (un.mcus) * 128 + (comp == 2 ? 64ull * im.mx * im.my : 0ull) +
                      (size_t)(8 * (un.mrow + yr)) * pitch + 8 * (un.mcol0 + yc);
            } else { dst = &s_c[comp - 1][8 * yr][8 * yc]; pitch = 8 * U; }
#pragma unroll
            for (int y = 0; y < 8; ++y)
                *reinterpret_cast<uint2*>(dst + y * pitch) = make_uint2(pair_bytes(yp[4 * y], yp[4 * y + 1]), pair_bytes(yp[4 * y + 2], yp[4 * y + 3]));
        }
    }
    if (kStage == 1) return;                                          // chroma pass: no pixels
    if (kStage == 2) {
        // chroma tile of the unit with a one-sample border, clamped to the padded planes
        const int cw = 8 * (int)im.mx, chh = 8 * (int)im.my, tw = 8 * nm + 2;
        const uint8_t* cbase = P.chroma + (un.mcus) * 128;
        for (int i = tid; i < 2 * (8 * R + 2) * tw; i += kT) {
            const int c = i / ((8 * R + 2) * tw), rem2 = i - c * (8 * R + 2) * tw, r = rem2 / tw, x = rem2 - r * tw;
            const int gy = min(max(8 * (int)un.mrow + r - 1, 0), chh - 1), gx2 = min(max(8 * (int)un.mcol0 + x - 1, 0), cw - 1);
            s_ct[c][r][x] = cbase[(size_t)c * cw * chh + (size_t)gy * cw + gx2];
        }
    }
    __syncthreads();

    // ---- colour, staged as the output's byte layout: 8 pixels of a row = 24 bytes
    if (valid && (NC == 1 || comp == 0)) {
        // chroma terms of a sample c (0..255): the upper halves of kR * c + rR and so on
        constexpr int kRr = 91881, kGb = -22553, kGr = -46802, kBb = 116130, kRnd = 32768;
        auto red = [&](int cr) { return (uint32_t)(kRr * cr + (kRnd - 128 * kRr)); };
        auto green = [&](int cb, int cr) { return (uint32_t)(kGb * cb + kGr * cr + (kRnd - 128 * (kGb + kGr))); };
        auto blue = [&](int cb) { return (uint32_t)(kBb * cb + (kRnd - 128 * kBb)); };
#pragma unroll
        for (int y = 0; y < 8; ++y) {
            uint32_t dr[4], dg[4], db[4];                             // per pixel pair
            if (kStage == 2) {
                const int row = 8 * yr + y, ry = 1 + (row >> 1), rn = ry + ((row & 1) ? 1 : -1);   // own / vertically nearer tile row
#pragma unroll
                for (int p = 0; p < 4; ++p) {
                    uint32_t x2[3][2];
#pragma unroll
                    for (int e = 0; e < 2; ++e) {
                        const int cx = 1 + 4 * yc + p, cn = cx + (e ? 1 : -1);
                        int m[2];
#pragma unroll
                        for (int c = 0; c < 2; ++c)
                            m[c] = (9 * s_ct[c][ry][cx] + 3 * s_ct[c][ry][cn] + 3 * s_ct[c][rn][cx] + s_ct[c][rn][cn] + 8) >> 4;
                        x2[0][e] = red(m[1]); x2[1][e] = green(m[0], m[1]); x2[2][e] = blue(m[0]);
                    }
                    dr[p] = __byte_perm(x2[0][0], x2[0][1], 0x7632); dg[p] = __byte_perm(x2[1][0], x2[1][1], 0x7632); db[p] = __byte_perm(x2[2][0], x2[2][1], 0x7632);
                }
            } else if (NC == 3 && HS == 2) {
                if (y % VS == 0) {
                    const uint32_t cbw = *reinterpret_cast<const uint32_t*>(&s_c[0][(8 * yr + y) / VS][4 * yc]);
                    const uint32_t crw = *reinterpret_cast<const uint32_t*>(&s_c[1][(8 * yr + y) / VS][4 * yc]);
#pragma unroll
                    for (int p = 0; p < 4; ++p) {                     // two pixels share a sample
                        const int cb = (int)((cbw >> (8 * p)) & 255u), cr = (int)((crw >> (8 * p)) & 255u);
                        dr[p] = __byte_perm(red(cr), 0, 0x3232); dg[p] = __byte_perm(green(cb, cr), 0, 0x3232); db[p] = __byte_perm(blue(cb), 0, 0x3232);
                    }
                }
            } else if (NC == 3) {
                if (y % VS == 0) {
                    const uint2 cb2 = *reinterpret_cast<const uint2*>(&s_c[0][(8 * yr + y) / VS][8 * yc]);
                    const uint2 cr2 = *reinterpret_cast<const uint2*>(&s_c[1][(8 * yr + y) / VS][8 * yc]);
#pragma unroll
                    for (int p = 0; p < 4; ++p) {
                        const uint32_t cbw = (p < 2 ? cb2.x : cb2.y) >> (16 * (p & 1)), crw = (p < 2 ? cr2.x : cr2.y) >> (16 * (p & 1));
                        const int cb0 = (int)(cbw & 255u), cb1 = (int)((cbw >> 8) & 255u), cr0 = (int)(crw & 255u), cr1 = (int)((crw >> 8) & 255u);
                        dr[p] = __byte_perm(red(cr0), red(cr1), 0x7632); dg[p] = __byte_perm(green(cb0, cr0), green(cb1, cr1), 0x7632);
                        db[p] = __byte_perm(blue(cb0), blue(cb1), 0x7632);
                    }
                }
            }
            uint32_t w[6];
#pragma unroll
            for (int h = 0; h < 2; ++h) {                             // four pixels: RGBR GBRG BRGB
                uint32_t rg[2], b[2];
#pragma unroll
                for (int e = 0; e < 2; ++e) {
                    const uint32_t Y = yp[4 * y + 2 * h + e];
                    if (NC == 1) { rg[e] = __byte_perm(Y, Y, 0x6240); b[e] = Y; }
                    else {
                        const uint32_t r2 = __viaddmin_s16x2_relu(Y, dr[2 * h + e], 0x00FF00FFu), g2 = __viaddmin_s16x2_relu(Y, dg[2 * h + e], 0x00FF00FFu);
                        b[e] = __viaddmin_s16x2_relu(Y, db[2 * h + e], 0x00FF00FFu);
                        rg[e] = __byte_perm(r2, g2, 0x6240);          // R0 G0 R1 G1
                    }
                }
                w[3 * h] = __byte_perm(rg[0], b[0], 0x2410);          // R0 G0 B0 R1
                w[3 * h + 1] = __byte_perm(__byte_perm(rg[0], b[0], 0x0063), rg[1], 0x5410);   // G1 B1 R2 G2
                w[3 * h + 2] = __byte_perm(rg[1], b[1], 0x6324);      // B2 R3 G3 B3
            }
            uint2* d = reinterpret_cast<uint2*>(s_stage + (8 * yr + y) * kStagePitch + 24 * yc);
            d[0] = make_uint2(w[0], w[1]); d[1] = make_uint2(w[2], w[3]); d[2] = make_uint2(w[4], w[5]);
        }
    }
    __syncthreads();

    // ---- store: each staged row is a contiguous byte run of the output
    const int x0 = kPxW * (int)un.mcol0;
    const int npx = min(kPxW * nm, (int)im.W - x0);
    const int row0 = kPxH * r_lo;                                     // first staged row that is wanted
    const int nrows = min(kPxH * r_hi, (int)im.H - kPxH * (int)un.mrow) - row0;
    const int nbytes = 3 * npx;
    const uint8_t* const stage0 = s_stage + row0 * kStagePitch;
    uint8_t* gbase = out + im.out_off + ((uint64_t)(kPxH * un.mrow + row0) * im.W + x0) * 3;
    const size_t gpitch = (size_t)im.W * 3;
    if (((reinterpret_cast<uintptr_t>(gbase) | gpitch | (uintptr_t)nbytes) & 15u) == 0) {
        // rows start and end on 16-byte boundaries: whole 16-byte vectors
        const int vec = nbytes >> 4;
        for (int i = tid; i < nrows * 24; i += kT) {                   // (24 vectors in a full row)
            const int row = i / 24, c = i - 24 * row;
            if (c < vec) *reinterpret_cast<uint4*>(gbase + row * gpitch + 16 * c) = *reinterpret_cast<const uint4*>(stage0 + row * kStagePitch + 16 * c);
        }
    } else {
        // rows at any byte address.  The 16-byte-aligned chunks of global memory that lie inside a row:
        // five staged words shifted into place, one 16-byte store
        constexpr int kInner = (3 * 128) / 16 - 1;
        for (int i = tid; i < nrows * kInner; i += kT) {
            const int row = i / kInner, slot = 1 + (i - row * kInner);
            uint8_t* gp = gbase + row * gpitch;
            const int lead = (int)(reinterpret_cast<uintptr_t>(gp) & 15u);
            if (16 * slot + 16 > lead + nbytes) continue;     // the row's last chunk, or behind it
            const int o0 = 16 * slot - lead;                  // the chunk's first byte, counted from the row's first
            const uint32_t* q = reinterpret_cast<const uint32_t*>(stage0 + row * kStagePitch) + (o0 >> 2);
            const int sh = 8 * (o0 & 3);
            const uint32_t p0 = q[0], p1 = q[1], p2 = q[2], p3 = q[3], p4 = q[4];   // (the spare bytes keep p4 in bounds)
            *reinterpret_cast<uint4*>(gp + o0) = make_uint4(__funnelshift_r(p0, p1, sh), __funnelshift_r(p1, p2, sh),
                                                            __funnelshift_r(p2, p3, sh), __funnelshift_r(p3, p4, sh));
        }
        // the first and the last chunk of every row: whole words where they lie inside the row, else bytes
        if (tid < 2 * nrows) {
            const int row = tid >> 1;
            uint8_t* gp = gbase + row * gpitch;
            const int lead = (int)(reinterpret_cast<uintptr_t>(gp) & 15u);
            const int nch = (lead + nbytes + 15) >> 4;
            if (!(tid & 1) || nch > 1) {
                const int o0 = 16 * ((tid & 1) ? nch - 1 : 0) - lead;
                const uint8_t* srow = stage0 + row * kStagePitch;
                const uint32_t* sw = reinterpret_cast<const uint32_t*>(srow);
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    const int sb = o0 + 4 * j;                // first staged byte of this output word
                    if (sb >= 0 && sb + 4 <= nbytes) {
                        const uint32_t lo = sw[sb >> 2], hi = sw[(sb >> 2) + 1];   // the spare bytes keep hi in bounds
                        *reinterpret_cast<uint32_t*>(gp + sb) = __funnelshift_r(lo, hi, 8 * (sb & 3));
                    } else {
                        for (int b = max(sb, 0); b < min(sb + 4, nbytes); ++b) gp[b] = srow[b];
                    }
                }
            }
        }
    }
}

// Pixel stage when nothing but DC coefficients has been decoded and every image is a multiple of
// 16 pixels wide: each 8x8 luminance block is one constant sample, each MCU one chroma pair, so
// an MCU row of the output is runs of eight equal pixels.  A CTA takes one work unit (8 MCUs of
// two MCU rows): 64 threads turn the unit's luminance blocks into RGB triples (the same
// arithmetic as the general kernel: the transform collapses to its k = 0 term, samples clamp to
// 0..255), then every thread writes 16-byte vectors whose bytes are picked from the two triples
// of the vector's MCU half-row.  48 bytes per MCU row = 3 vectors, so a vector never leaves its MCU.
// kAligned = false: images of any width.  A row of the unit then starts at any byte address: every
// thread takes one 16-byte-aligned chunk of global memory that the row touches, builds its four
// words from the triples of the (at most two) pixels each word covers, and stores the chunk whole
// when it lies inside the row, byte by byte at the row's two ends.
template <bool kRoi, bool kAligned = true>
__global__ void __launch_bounds__(128) dc_pixel_kernel(Params P, uint3 dc_mask, uint8_t* __restrict__ out) {
    constexpr int U = Sampling<kSamp420>::U, R = Sampling<kSamp420>::R;
    __shared__ uint32_t s_tri[2 * R][2 * U];           // [block row of the unit][block column]: R | G << 8 | B << 16
    const int tid = threadIdx.x;
    const Unit un = P.units[blockIdx.x];
    const Image im = image_of<6>(un);
    const int nm = min(U, (int)im.mx - (int)un.mcol0);
    int r_lo = 0, r_hi = min(R, (int)im.my - (int)un.mrow);
    if (kRoi) {
        const CropRect r = P.roi[un.img];
        const int ux0 = 16 * un.mcol0;
        r_lo = max(r_lo, (int)(r.y0 / 16u) - (int)un.mrow); r_hi = min(r_hi, (int)((r.y0 + r.h - 1u) / 16u) + 1 - (int)un.mrow);
        if (r_lo >= r_hi || ux0 >= (int)(r.x0 + r.w) || ux0 + 16 * nm <= (int)r.x0) return;
    }
    {
        constexpr uint32_t K4 = 5793;
        const int brow = tid / (2 * U), bcol = tid % (2 * U);
        if (brow >= 2 * r_lo && brow < 2 * r_hi && bcol < 2 * nm) {
            const uint16_t* q = P.qtab + (size_t)un.img * 192;
            auto sample = [&](uint64_t blk, int comp) {
                const int F = (int)(short)((uint32_t)__ldg(P.dc + blk) & (comp == 0 ? dc_mask.x : (comp == 1 ? dc_mask.y : dc_mask.z))) * (int)q[64 * comp];
                const int T = (int)(K4 * (uint32_t)F + (1u << 11)) >> 12;
                const int smp = ((int)(K4 * (uint32_t)T + (1u << 15)) >> 16) + 128;
                return min(max(smp, 0), 255);
            };
            const uint64_t mcus = (uint64_t)im.mx * im.my;
            const uint64_t yb = im.blk_base + (uint64_t)(2 * un.mrow + brow) * (2 * im.mx) + 2 * un.mcol0 + bcol;
            const uint64_t cbk = im.blk_base + 4 * mcus + (uint64_t)(un.mrow + (brow >> 1)) * im.mx + un.mcol0 + (bcol >> 1);
            const int Y = sample(yb, 0), cb = sample(cbk, 1) - 128, cr = sample(cbk + mcus, 2) - 128;
            const int Rv = Y + ((91881 * cr + 32768) >> 16);
            const int G = Y + ((-22553 * cb - 46802 * cr + 32768) >> 16);
            const int B = Y + ((116130 * cb + 32768) >> 16);
            s_tri[brow][bcol] = (uint32_t)min(max(Rv, 0), 255) | ((uint32_t)min(max(G, 0), 255) << 8) | ((uint32_t)min(max(B, 0), 255) << 16);
        }
    }
    __syncthreads();
    const int row0 = 16 * r_lo, nrows = min(16 * r_hi, (int)im.H - 16 * (int)un.mrow) - row0;
    const size_t gpitch = (size_t)im.W * 3;
    uint8_t* gbase = out + im.out_off + ((uint64_t)(16 * un.mrow + row0) * im.W + 16 * (uint64_t)un.mcol0) * 3;
    if (!kAligned) {
        const int len = 3 * min(16 * nm, (int)im.W - 16 * (int)un.mcol0);      // bytes of the unit in one output row
        // the four bytes at offset o of a row (o may lie up to 15 bytes before the row or behind its end:
        // those bytes are not stored, their pixels are clamped into the unit): pixel px from channel ph
        // on, then pixel px + 1
        auto word_at = [&](const uint32_t* tri, int o) {
            const int oo = o + 24;
            const int px = (int)(((uint32_t)oo * 0xAAABu) >> 17) - 8, ph = oo - 3 * (px + 8);
            const uint32_t A = tri[min(max(px, 0), 16 * nm - 1) >> 3], Bt = tri[min(max(px + 1, 0), 16 * nm - 1) >> 3];
            return __byte_perm(A, Bt, ph == 0 ? 0x4210u : (ph == 1 ? 0x5421u : 0x6542u));
        };
        // the bytes of one output row of the unit, once per block row (the eight pixel rows of a block row are
        // equal), with 16 bytes of margin on either side so that a chunk may begin before the row or end behind it
        constexpr int kPatWords = (16 + 3 * 16 * U + 16) / 4;
        __shared__ __align__(16) uint32_t s_pat[2 * R][kPatWords];
        for (int i = tid; i < 2 * R * kPatWords; i += 128) {
            const int br = i / kPatWords, wi = i - br * kPatWords;
            s_pat[br][wi] = word_at(s_tri[br], 4 * wi - 16);
        }
        __syncthreads();
        // the 16 bytes of a row from offset o on (o >= -16): five pattern words, shifted into place
        auto chunk_at = [&](const uint32_t* pat, int o) {
            const int sb = o + 16, a = 8 * (sb & 3);
            const uint32_t* q = pat + (sb >> 2);
            const uint32_t p0 = q[0], p1 = q[1], p2 = q[2], p3 = q[3], p4 = q[4];
            return make_uint4(__funnelshift_r(p0, p1, a), __funnelshift_r(p1, p2, a), __funnelshift_r(p2, p3, a), __funnelshift_r(p3, p4, a));
        };
        // chunks that lie inside the row: whole 16-byte stores
        constexpr int kInner = (3 * 16 * U) / 16 - 1;
        for (int i = tid; i < nrows * kInner; i += 128) {
            const int row = i / kInner, slot = 1 + (i - row * kInner);
            uint8_t* g = gbase + row * gpitch;                                  // first byte of the row
            const int lead = (int)(reinterpret_cast<uintptr_t>(g) & 15u);
            if (16 * slot + 16 > lead + len) continue;                          // the row's last chunk, or behind it
            const int o0 = 16 * slot - lead;                                    // the chunk's first byte, counted from g
            *reinterpret_cast<uint4*>(g + o0) = chunk_at(s_pat[(row0 + row) >> 3], o0);
        }
        // the first and the last chunk of every row: whole words where they lie inside, else bytes
        if (tid < 2 * nrows) {
            const int row = tid >> 1;
            uint8_t* g = gbase + row * gpitch;
            const int lead = (int)(reinterpret_cast<uintptr_t>(g) & 15u);
            const int nch = (lead + len + 15) >> 4;
            const int slot = (tid & 1) ? nch - 1 : 0;
            if (!(tid & 1) || nch > 1) {
                const int o0 = 16 * slot - lead;
                const uint4 v = chunk_at(s_pat[(row0 + row) >> 3], o0);
                const uint32_t w4[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    const int o = o0 + 4 * j;
                    if (o >= 0 && o + 4 <= len) {
                        *reinterpret_cast<uint32_t*>(g + o) = w4[j];
                    } else {
#pragma unroll
                        for (int b = 0; b < 4; ++b)
                            if (o + b >= 0 && o + b < len) g[o + b] = (uint8_t)(w4[j] >> (8 * b));
                    }
                }
            }
        }
        return;
    }
    const int vec = 3 * nm;                                 // 16-byte vectors per output row of this unit
    for (int i = tid; i < nrows * 3 * U; i += 128) {        // (as if the unit were full: the division is by a constant)
        const int row = i / (3 * U), v = i - row * (3 * U), mcu = v / 3, kk = v - 3 * mcu, br = (row0 + row) >> 3;
        if (v >= vec) continue;
        const uint32_t A = s_tri[br][2 * mcu], Bt = s_tri[br][2 * mcu + 1];
        // four-byte words of a run of equal pixels repeat with period three: RGBR GBRG BRGB
        const uint32_t aw0 = __byte_perm(A, 0, 0x0210), aw1 = __byte_perm(A, 0, 0x1021), aw2 = __byte_perm(A, 0, 0x2102);
        const uint32_t bw0 = __byte_perm(Bt, 0, 0x0210), bw1 = __byte_perm(Bt, 0, 0x1021), bw2 = __byte_perm(Bt, 0, 0x2102);
        uint4 o;
        if (kk == 0) o = make_uint4(aw0, aw1, aw2, aw0);           // bytes 0..15: left pixels
        else if (kk == 1) o = make_uint4(aw1, aw2, bw0, bw1);      // bytes 16..23 left, 24..31 right
        else o = make_uint4(bw2, bw0, bw1, bw2);                   // bytes 32..47: right pixels
        *reinterpret_cast<uint4*>(gbase + row * gpitch + 16 * v) = o;
    }
}

// Training-tensor epilogue: crop, optional mirror, bilinear resize to size x size with half-pixel
// centres (the crop's edge pixels repeated, no low-pass filter), (v / 255 - mean) / std, planar
// output [image][channel][row][column].  Images pos0 .. pos0 + gridDim.y - 1 of the processing order.
struct TensorArgs {
    const CropRect* crops;     // [N], by image index
    void* out;                 // [N][3][size][size]
    int32_t size;
    int32_t f32;               // output type: 0 half precision, 1 single precision, 2 bfloat16
    float mean[3], inv_std[3];
};

__device__ __forceinline__ void tensor_store(float* p, float v) { *p = v; }
__device__ __forceinline__ void tensor_store(__half* p, float v) { *p = __float2half_rn(v); }
__device__ __forceinline__ void tensor_store(__nv_bfloat16* p, float v) { *p = __float2bfloat16_rn(v); }
__device__ __forceinline__ void tensor_store2(float* p, float v, float w) { *reinterpret_cast<float2*>(p) = make_float2(v, w); }
__device__ __forceinline__ void tensor_store2(__half* p, float v, float w) { *reinterpret_cast<__half2*>(p) = __floats2half2_rn(v, w); }
__device__ __forceinline__ void tensor_store2(__nv_bfloat16* p, float v, float w) { *reinterpret_cast<__nv_bfloat162*>(p) = __floats2bfloat162_rn(v, w); }

// Two horizontally adjacent RGB pixels (six bytes from byte `off` on, at any alignment) as floats, read as aligned
// words: the word holding the first byte, the next one, and a third only when the six bytes reach
// into it.
__device__ __forceinline__ void load_rgb_pair(const uint32_t* base, uint32_t off, float& r0, float& g0, float& b0,
                                              float& r1, float& g1, float& b1) {
    const uint32_t* w = base + (off >> 2);
    const uint32_t w0 = __ldg(w), w1 = __ldg(w + 1);
    const uint32_t w2 = (off & 3u) == 3u ? __ldg(w + 2) : 0u;
    const uint32_t lo = __funnelshift_r(w0, w1, 8 * off), hi = __funnelshift_r(w1, w2, 8 * off);   // bytes 0..3, 4..7 (shifts taken mod 32)
    r0 = __uint_as_float(__byte_perm(lo, 0x4B000000u, 0x7540)) - 8388608.f;      // byte into the mantissa of 2^23
    g0 = __uint_as_float(__byte_perm(lo, 0x4B000000u, 0x7541)) - 8388608.f;
    b0 = __uint_as_float(__byte_perm(lo, 0x4B000000u, 0x7542)) - 8388608.f;
    r1 = __uint_as_float(__byte_perm(lo, 0x4B000000u, 0x7543)) - 8388608.f;
    g1 = __uint_as_float(__byte_perm(hi, 0x4B000000u, 0x7540)) - 8388608.f;
    b1 = __uint_as_float(__byte_perm(hi, 0x4B000000u, 0x7541)) - 8388608.f;
}

#ifndef PCR_TENSOR_ROWS
#define PCR_TENSOR_ROWS 16
#endif
constexpr int kTensorRows = PCR_TENSOR_ROWS;      // output rows per CTA

// One CTA per band of kTensorRows output rows of one image, kCols neighbouring output columns per thread (their
// horizontal taps and weights are computed once for the band).  Two for even sizes: pairs of values are stored
// together.  The taps are read from global memory through the read-only path: neighbouring threads and rows hit the same
// cache lines (staging the band's source rows in shared memory first was 40 % slower: it costs the
// L1 capacity that these reads live on).  A source row that the previous output row used, as the lower or the upper one, is
// not interpolated again: a usual crop is about as large as the output, so one new source row per output row.
// Neither the issue slots (71 % used) nor DRAM (33 %) are full: of 13.0 cycles that a warp takes an instruction it waits 7.8 for
// its taps, with 58 % of the warps an SM could hold (48 registers).  1024 images cropped to 224x224 fp16 (51 M output pixels): 220 us
// with a column a thread, 195 us with two and rows used again, 184 us with the normalisation as one multiplication and addition a
// value.
template <typename OutT, int kCols>
__global__ void __launch_bounds__(256 / kCols) tensor_kernel(Params P, TensorArgs T, const uint8_t* __restrict__ rgb, uint32_t pos0) {
    __shared__ int s_off0[kTensorRows], s_off1[kTensorRows];       // byte offsets of a row's upper / lower source row in the crop
    __shared__ float s_ay[kTensorRows];
    const uint32_t img = P.order[pos0 + blockIdx.y];
    const int S = T.size;
    const int oy0 = blockIdx.x * kTensorRows;
    const int nrows = min(kTensorRows, S - oy0);
    const ImgDesc im = P.imgs[img];
    const CropRect r = T.crops[img];
    const float sx = (float)r.w / (float)S, sy = (float)r.h / (float)S;
    const uint32_t pitch = im.W * 3u;
    const uint32_t* const image = reinterpret_cast<const uint32_t*>(rgb + im.out_off);   // (images start at multiples of 128)
    const uint32_t crop0 = r.y0 * pitch + r.x0 * 3u;          // first byte of the crop
    if ((int)threadIdx.x < nrows) {
        float fy = ((float)(oy0 + (int)threadIdx.x) + 0.5f) * sy - 0.5f;
        fy = fminf(fmaxf(fy, 0.f), (float)(r.h - 1));
        const int iy = (int)floorf(fy), iy1 = min(iy + 1, (int)r.h - 1);
        s_ay[threadIdx.x] = fy - (float)iy;
        s_off0[threadIdx.x] = iy * (int)pitch; s_off1[threadIdx.x] = iy1 * (int)pitch;   // an image stays below 2 GiB
    }
    __syncthreads();
    const uint32_t plane = (uint32_t)S * (uint32_t)S;
    const float w0 = T.inv_std[0] / 255.f, w1 = T.inv_std[1] / 255.f, w2 = T.inv_std[2] / 255.f;
    const float z0 = -T.mean[0] * T.inv_std[0], z1 = -T.mean[1] * T.inv_std[1], z2 = -T.mean[2] * T.inv_std[2];
    OutT* const obase = static_cast<OutT*>(T.out) + (size_t)img * 3 * plane + (size_t)oy0 * S;
    for (int ox = kCols * (int)threadIdx.x; ox < S; ox += 256) {
        uint32_t p0[kCols];                                 // byte of the left tap in the crop's first row, from the image's first byte
        float ax[kCols], bx[kCols];
#pragma unroll
        for (int c = 0; c < kCols; ++c) {
            const int u = r.flip ? S - 1 - (ox + c) : ox + c;
            float fx = ((float)u + 0.5f) * sx - 0.5f;
            fx = fminf(fmaxf(fx, 0.f), (float)(r.w - 1));
            const int ix = (int)floorf(fx);
            ax[c] = fx - (float)ix; bx[c] = 1.f - ax[c];
            // (at the crop's right edge the right tap has weight 0: whatever byte lies there does not count)
            p0[c] = crop0 + 3u * (uint32_t)ix;
        }
        float t[kCols][3], h[kCols][3];                     // the upper / lower source row at these columns
        auto source_row = [&](int q, float (&v)[kCols][3]) {
#pragma unroll
            for (int c = 0; c < kCols; ++c) {
                float r0, g0, b0, r1, g1, b1;
                load_rgb_pair(image, p0[c] + (uint32_t)q, r0, g0, b0, r1, g1, b1);
                v[c][0] = bx[c] * r0 + ax[c] * r1; v[c][1] = bx[c] * g0 + ax[c] * g1; v[c][2] = bx[c] * b0 + ax[c] * b1;
            }
        };
        auto copy_row = [&](float (&a)[kCols][3], const float (&b)[kCols][3]) {
#pragma unroll
            for (int c = 0; c < kCols; ++c) { a[c][0] = b[c][0]; a[c][1] = b[c][1]; a[c][2] = b[c][2]; }
        };
        int tq = -1, hq = -1;                               // their offsets
        OutT* o = obase + ox;
        for (int dy = 0; dy < nrows; ++dy, o += S) {
            const int q0 = s_off0[dy], q1 = s_off1[dy];
            const float ay = s_ay[dy], by = 1.f - ay;
            if (q0 != tq) { if (q0 == hq) copy_row(t, h); else source_row(q0, t); tq = q0; }
            if (q1 != hq) { if (q1 == tq) copy_row(h, t); else source_row(q1, h); hq = q1; }
            float v[3][kCols];
#pragma unroll
            for (int c = 0; c < kCols; ++c) {
                // (v / 255 - mean) / std as one multiplication and one addition
                v[0][c] = (by * t[c][0] + ay * h[c][0]) * w0 + z0;
                v[1][c] = (by * t[c][1] + ay * h[c][1]) * w1 + z1;
                v[2][c] = (by * t[c][2] + ay * h[c][2]) * w2 + z2;
            }
#pragma unroll
            for (int e = 0; e < 3; ++e) {
                if (kCols == 2) tensor_store2(o + e * plane, v[e][0], v[e][kCols - 1]);
                else tensor_store(o + e * plane, v[e][0]);
            }
        }
    }
}

}  // namespace pcr
