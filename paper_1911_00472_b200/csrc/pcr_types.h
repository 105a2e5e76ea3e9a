// Structures shared by the host side and the kernels of the PCR decoder.
#pragma once
#include <stdint.h>
#include <vector_types.h>

namespace pcr {

// One scan of the (record-wide) scan script: which components, which band, which bit.
struct __align__(16) ScanScript {
    int32_t ncomp;
    int32_t comp[3];
    int32_t Ss, Se, Ah, Al;
};

// Where an AC scan keeps its per-block side data in the auxiliary array (units of uint64,
// indexed by the block's number inside its component across the whole record):
//  - a first-pass AC scan writes the mask of zigzag positions it made non-zero and, if its band reaches beyond
//    position 7, a second word: where the block's values for those positions begin in the value array;
//  - an AC refinement scan writes four words per block: {mask of non-zero positions of its band
//    after the scan, correction bits in reading order (last bit at bit 0), mask of newly
//    non-zero positions, mask of those that are positive}.  The pixel kernel applies them to a block
//    when it expands it.
//  - a sequential scan writes the same for positions 8..63 of the blocks of all components, indexed by the
//    block's number in the planes.
// A refinement scan finds the positions that were non-zero before it by OR-ing the masks of up
// to four earlier scans (src), each read with its own stride.
struct __align__(16) ScanAux {
    uint64_t base;        // first word of this scan's side data
    uint32_t stride;      // words per block: 1 or 2 (first passes), 4 (refinements)
    int32_t nsrc;
    int32_t src[4];       // scan indices
    uint32_t tab0;        // first of the scan's lookup tables (see ScanTab): image i has ntab of them from tab0 + i * ntab on
    int32_t ntab;         // 2 for a DC first pass, 1 for an AC scan, 4 for a sequential scan, 0 for a DC refinement
};

// Where the coefficients of the decoded scans lie, per component (built per call for the chosen k).
constexpr int kMaxFirst = 56;      // first passes of a component that reach beyond position 7: at most one for each of 8..63
                                   // (pcr_open refuses a position that is sent twice)
struct CoefLists {
    uint4 head_mask[3];            // positions 1..7 that a decoded scan covers, as 16-bit lanes of the head plane's entries
    uint32_t dc_mask[3];           // bits of the DC coefficient that a decoded scan covers (a refinement of an earlier
                                   // decode may have left others in blocks that a damaged stream no longer reaches)
    int32_t n_first[3], n_refine[3];
    int32_t sequential;            // side data indexed by the block's number in the planes, not inside its component
    uint64_t first[3][kMaxFirst];  // first word of the scan's side data (two words per block)
    uint64_t refine[3][4];         // the refinement scans in scan order: first word of the side data (four words per block)
    int32_t p1[3][4];              // 1 << Al of the scan
};

// The AC refinements one call decodes, per component in scan order (for the chain launch).
struct RefineList {
    int32_t n[3];
    int32_t scan[3][4];
};

// One (scan, image) pair: where its entropy-coded bytes and Huffman tables live.
struct __align__(16) ScanDesc {
    uint32_t data_off;    // first entropy-coded byte (offset in the record)
    uint32_t data_end;    // one past the last byte of the chunk
    uint32_t seg_base;    // first entry of this pair in the segment table
    uint32_t nseg;        // restart intervals in the scan
    uint32_t ri;          // restart interval in MCUs (0 = none)
    uint32_t tab_off[2];  // offsets of up to two DHT table bodies (16 counts, then values)
    uint32_t slots;       // 2 bits per scan component: which of tab_off it uses
    uint32_t tab_ac[2];   // sequential scans only: up to two AC table bodies (tab_off then holds the DC tables)
    uint32_t slots_ac;    // 2 bits per scan component: which of tab_ac it uses
};

struct __align__(16) ImgDesc {
    uint32_t W, H, mx, my;
    uint64_t blk_base;    // first block of the image in the coefficient planes
    uint64_t out_off;     // first byte of the image in the output buffer
};

// Restart intervals one warp takes (one lane each).  Fewer than 32 leaves lanes idle but
// gives more warps to hide the latency of the serial decode chains.
#ifndef PCR_SEGS_PER_ITEM
#define PCR_SEGS_PER_ITEM 32
#endif
constexpr int kSegsPerItem = PCR_SEGS_PER_ITEM;

// Entropy work item: up to kSegsPerItem consecutive restart intervals of one (scan, image); or up to half as many of
// two AC refinements of the same band that follow one another (see entropy_kernel).
struct Item {
    uint32_t si;          // scan * N + image
    uint32_t seg0;        // first restart interval of the item
    uint32_t count;       // restart intervals in the item (<= kSegsPerItem)
    uint32_t next;        // 0, or 1 + (scan * N + image) of the image whose first intervals the item runs on into
    uint32_t pair;        // 0, or the distance to the later refinement of the pair (in scan * N + image)
};
// The runs of the item list that one launch covers.
constexpr int kMaxRuns = 24;
struct ItemRuns {
    int32_t n;
    uint32_t first[kMaxRuns], end[kMaxRuns];   // first item of the run; items in this run and those before it
    // DC refinement scans in blocks behind those of the items: of the images order[dc_pos0 ..], dc_chunks blocks an image
    uint32_t item_blocks;
    int32_t dc_s[3];
    uint32_t dc_pos0, dc_images, dc_chunks;
};

// Crop rectangle of one image (pixels) and whether its columns are mirrored; the pixel kernel
// skips work units that lie outside it when one is given.
struct CropRect {
    uint32_t x0, y0, w, h, flip;
};

// Pixel work unit: a run of MCUs in one MCU row of one image.
// With what a CTA needs of its image, so that one load tells it everything.
struct __align__(16) Unit {
    uint32_t img;
    uint16_t mrow, mcol0, mx, my, W, H;
    uint64_t mcus;        // MCUs of the images before this one
    uint64_t out_off;     // first byte of the image in the output buffer
};

struct ScanTab;             // lookup table of one Huffman table (pcr_entropy.cuh)

struct Params {
    const uint8_t* rec;         // record bytes on the device
    uint8_t* ubuf;              // entropy-coded bytes without stuffing, big-endian words
    int16_t* planes;            // coefficient planes, 64 int16 per block, zigzag order: only written when somebody asks
                                // for them (pcr_coeffs); the decode itself keeps coefficients as
    int16_t* dc;                //  - the DC coefficient of every block, dense (same block numbering),
    int16_t* head;              //  - zigzag positions 1..7 of every block, dense (8 int16 = 16 bytes per block, the first
                                //    one unused),
    int16_t* vals;              //  - the non-zero values of positions 8..63, block after block in reading order; their
                                //    positions are the masks of the scan's side data.  A coefficient takes at least two
                                //    bits of the stream, so the values of whatever begins at byte b of the
                                //    unstuffed copy begin at index 4 b and nothing overlaps.
                                //    (Eight bytes per record byte: more than planes would take from about 0.4 bytes a
                                //    pixel on in 4:2:0.)
                                // Every decode of a record's bytes writes the same values to the same places, so none of this
                                // is cleared between decodes
    const ScanScript* script;   // [G]
    const ScanAux* saux;        // [G]
    uint64_t* aux;              // side data of the AC scans
    const ScanDesc* scans;      // [G][N]
    const ImgDesc* imgs;        // [N]
    uint32_t* seg_start;        // segment table: first byte of every restart interval
    const Item* items;
    const Unit* units;
    const uint16_t* qtab;       // [N][3][64] quantisers, zigzag order
    uint8_t* chroma;            // chroma sample planes (triangle upsampling only): per image, at 128 bytes
                                // per MCU in front of it, a Cb plane then a Cr plane of 8*my rows x 8*mx bytes
    ScanTab* tabs;              // lookup tables of the decoded scans, by ScanAux::tab0
    const uint32_t* order;      // [N] processing order of the images
    const CropRect* roi;        // [N] or null: only work units that touch the image's rectangle are transformed
    int* status;                // [N]
    int32_t N;
    // chroma sampling of the record's images: the luminance component has hs x vs blocks per MCU
    // (1 or 2 each), every chroma component one; nc = 3, or 1 for greyscale (then hs = vs = 1 and
    // the block grid has no MCU padding)
    int32_t hs, vs, nc;
};

}  // namespace pcr
