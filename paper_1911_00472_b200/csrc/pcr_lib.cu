// Host side of the PCR decoder and its C ABI (see include/pcr.h).
//
// pcr_open walks the record's metadata and every image's JPEG marker segments once, on the
// host, and turns them into flat device tables (per (scan, image) byte ranges and Huffman
// table positions, per image geometry, work lists).  pcr_decode only enqueues work: the
// prefix copy, the restart-interval index, one entropy kernel per dependency wave of the
// scan script, and the fused pixel kernel.
#include <cuda_runtime.h>
#include <stdint.h>
#include <stdio.h>
#include <stdlib.h>
#include <string.h>

#include <algorithm>
#include <atomic>
#include <map>
#include <memory>
#include <mutex>
#include <new>
#include <system_error>
#include <thread>
#include <utility>
#include <vector>

#include "../../include/pcr.h"
#include "pcr_entropy.cuh"
#include "pcr_long.cuh"
#include "pcr_msssim.cuh"
#include "pcr_pixels.cuh"
#include "pcr_refine.cuh"
#include "pcr_sequential.cuh"
#include "pcr_types.h"

using namespace pcr;

static std::atomic<uint64_t> g_launches{0};

// Device buffers of closed records are kept for the next pcr_open instead of going back to the
// driver: cudaMalloc and cudaFree cost milliseconds and cudaFree waits for the whole device, which
// a loader that opens and closes one record after the other cannot afford.  Sizes are rounded up
// to classes with three mantissa bits (at most 12.5 % slack) so that records of similar size
// reuse each other's buffers.
namespace {
struct DeviceCache {
    std::mutex mu;
    std::multimap<std::pair<int, size_t>, void*> free_;
    size_t cached = 0;
    static constexpr size_t kLimit = 24ull << 30;
} g_cache;

size_t size_class(size_t n) {
    if (n < 4096) return 4096;
    int top = 63 - __builtin_clzll((unsigned long long)n);
    const size_t step = (size_t)1 << (top - 3);
    return (n + step - 1) & ~(step - 1);
}

void* dev_alloc(size_t n, int device) {
    const size_t cls = size_class(n);
    {
        std::lock_guard<std::mutex> lk(g_cache.mu);
        auto it = g_cache.free_.find({device, cls});
        if (it != g_cache.free_.end()) {
            void* p = it->second;
            g_cache.free_.erase(it);
            g_cache.cached -= cls;
            return p;
        }
    }
    void* p = nullptr;
    if (cudaMalloc(&p, cls) != cudaSuccess) {
        cudaGetLastError();
        // give cached buffers back and try once more
        std::lock_guard<std::mutex> lk(g_cache.mu);
        for (auto& kv : g_cache.free_) cudaFree(kv.second);
        g_cache.free_.clear();
        g_cache.cached = 0;
        if (cudaMalloc(&p, cls) != cudaSuccess) { cudaGetLastError(); return nullptr; }
    }
    return p;
}

// Page-locked host blocks in which pcr_open builds a record's tables: one asynchronous copy takes them to the
// device, and a block that has been used before costs no page faults.  Kept for later opens up to kHostLimit bytes.
struct HostCache {
    std::mutex mu;
    std::multimap<size_t, void*> free_;
    size_t cached = 0;
    static constexpr size_t kLimit = 256ull << 20;
} g_host;

void* host_alloc(size_t n) {
    const size_t cls = size_class(n);
    {
        std::lock_guard<std::mutex> lk(g_host.mu);
        auto it = g_host.free_.find(cls);
        if (it != g_host.free_.end()) {
            void* p = it->second;
            g_host.free_.erase(it);
            g_host.cached -= cls;
            return p;
        }
    }
    void* p = nullptr;
    if (cudaHostAlloc(&p, cls, cudaHostAllocPortable) != cudaSuccess) { cudaGetLastError(); return nullptr; }
    return p;
}
void host_release(void* p, size_t n) {
    if (!p) return;
    const size_t cls = size_class(n);
    std::lock_guard<std::mutex> lk(g_host.mu);
    if (g_host.cached + cls <= HostCache::kLimit) {
        g_host.free_.insert({cls, p});
        g_host.cached += cls;
    } else {
        cudaFreeHost(p);
    }
}

// internal streams and (non-timing) events are pooled the same way
struct HandlePool {
    std::mutex mu;
    std::multimap<int, cudaStream_t> streams;
    std::multimap<int, cudaEvent_t> events;
} g_handles;

cudaStream_t pool_stream_get(int device) {
    {
        std::lock_guard<std::mutex> lk(g_handles.mu);
        auto it = g_handles.streams.find(device);
        if (it != g_handles.streams.end()) { cudaStream_t q = it->second; g_handles.streams.erase(it); return q; }
    }
    cudaStream_t q = nullptr;
    if (cudaStreamCreateWithFlags(&q, cudaStreamNonBlocking) != cudaSuccess) { cudaGetLastError(); return nullptr; }
    return q;
}
void pool_stream_put(cudaStream_t q, int device) {
    if (!q) return;
    std::lock_guard<std::mutex> lk(g_handles.mu);
    g_handles.streams.insert({device, q});
}
cudaEvent_t pool_event_get(int device) {
    {
        std::lock_guard<std::mutex> lk(g_handles.mu);
        auto it = g_handles.events.find(device);
        if (it != g_handles.events.end()) { cudaEvent_t e = it->second; g_handles.events.erase(it); return e; }
    }
    cudaEvent_t e = nullptr;
    if (cudaEventCreateWithFlags(&e, cudaEventDisableTiming) != cudaSuccess) { cudaGetLastError(); return nullptr; }
    return e;
}
void pool_event_put(cudaEvent_t e, int device) {
    if (!e) return;
    std::lock_guard<std::mutex> lk(g_handles.mu);
    g_handles.events.insert({device, e});
}

void dev_release(void* p, size_t n, int device) {
    if (!p) return;
    const size_t cls = size_class(n);
    std::lock_guard<std::mutex> lk(g_cache.mu);
    if (g_cache.cached + cls <= DeviceCache::kLimit) {
        g_cache.free_.insert({{device, cls}, p});
        g_cache.cached += cls;
    } else {
        cudaFree(p);
    }
}
}  // namespace

struct pcr_record {
    const uint8_t* host = nullptr;
    size_t len = 0;
    int N = 0, G = 0;
    std::vector<uint64_t> group_end;
    std::vector<pcr_image_info> info;
    std::vector<uint64_t> blk_base, nblk;
    uint64_t total_blocks = 0, total_segs = 0;
    int hs = 2, vs = 2, nc = 3;     // chroma sampling, the same for every image of the record
    uint32_t unit_mcus = 8, unit_rows = 2;   // MCUs across and MCU rows of a pixel work unit
    unsigned dc_refine_chunks = 1;  // 256-MCU chunks of the largest image, at most 8 (dc_refine_kernel's grid)
    bool widths_mult16 = true;    // every image is a multiple of 16 pixels wide (the DC-only pixel kernel's condition)
    size_t out_bytes = 0;
    // scan script analysis
    std::vector<ScanScript> script;
    std::vector<int> wave_of_scan;
    int n_waves = 0;
    // images are cut into slices that run as independent pipelines on their own streams;
    // items are sorted by (slice, wave, scan), units by image
    int n_slices = 1;
    std::vector<uint32_t> slice_img;                            // [n_slices + 1] first image of each slice
    std::vector<uint32_t> slice_unit;                           // [n_slices + 1] first pixel unit of each slice
    std::vector<uint32_t> item_begin, item_count;               // [n_slices][G]
    std::vector<uint32_t> longest, longest_chain;               // by scan: entropy-coded bytes, and bytes of an interval, of the image that has most
    std::vector<uint64_t> intervals, long_bytes;                // by scan: intervals; entropy-coded bytes that kernels for long intervals read
    std::vector<uint64_t> first_bytes;                          // of AC first passes: entropy-coded bytes that items stand for
    // Scans that are one long restart interval take kernels of their own (pcr_long.cuh): first passes
    // as (scan, image) pairs sorted by (slice, wave, scan); AC refinements as (component, image)
    // groups sorted by slice (all refinement scans of the component that a call decodes, in one CTA)
    std::vector<uint32_t> long_begin, long_count;               // [n_slices][G]
    uint32_t* d_long = nullptr;
    uint32_t n_groups = 0;                                      // (image, component) pairs whose AC refinements are chains
    uint32_t* d_group = nullptr;                                // luminance first, most bytes first
    uint32_t* d_chain_sync = nullptr;                           // queue counters and progress words of the chain launch
    int n_sms = 1;
    cudaEvent_t ev_chain = nullptr;
    std::vector<cudaStream_t> streams;                          // one per slice
    std::vector<cudaEvent_t> ev_index;                          // [n_waves] index of wave w done (side stream)
    cudaEvent_t ev_start = nullptr;                             // index of the first wave done
    cudaEvent_t ev_fork = nullptr;
    cudaStream_t copy_stream = nullptr;                         // host-to-device copies of later scan groups
    cudaStream_t side_stream = nullptr;                         // index of the later waves, beside the first entropy wave
    cudaEvent_t ev_side = nullptr;
    std::vector<cudaEvent_t> ev_copy;                           // [n_waves] bytes of wave w have arrived
    std::vector<cudaEvent_t> ev_join;
    std::vector<std::vector<int>> wave_scans;
    // The same with pairs of AC refinements in one wave (see entropy_kernel); pair_of[s] = the earlier refinement that
    // scan s follows, or -1.  Empty when the script has no such pair.
    std::vector<std::vector<int>> paired_waves;
    std::vector<int> pair_of;
    int pairs = -1;                                             // see pairs_pay (PCR_PAIRS overrides: 0 never, 1 always)
    double refine_ctas = 3.4;                                   // see refine_in_ctas (PCR_REFINE_CTAS overrides)
    int64_t long_ctas = -1;                                     // see wide_long_scans (PCR_LONG_CTAS: a line in CTAs an SM instead)
    int64_t seq_ctas = -1;                                      // see sequential_in_ctas (PCR_SEQ_CTAS: a line in items an SM instead)
    int64_t index_ctas = -1;                                    // see launch_index_kernel (PCR_INDEX_CTAS: a line in pairs an SM instead)
    int64_t pack_warps = -1;                                    // see first_pass_form (PCR_PACK_WARPS: a line in warps an SM instead)
    uint32_t short_warps = 20;                                  // see first_pass_form (PCR_SHORT_WARPS overrides)
    // Items of the AC refinements (and of a sequential scan): the sum of their chains' bytes, an item counting with its longest.
    // By scan; by the pair's later scan.  And the sum of their squares
    std::vector<uint64_t> chain_bytes, pair_chain_bytes;
    std::vector<double> chain_squares, pair_chain_squares;
    std::vector<uint32_t> pair_begin, pair_count;               // [n_slices][G] items of the pair, by its later scan
    uint32_t n_units = 0;
    // device state
    int device = 0;
    uint8_t* d_rec = nullptr;
    uint8_t* d_ubuf = nullptr;
    size_t resident = 0;
    int16_t* d_planes = nullptr;  // canonical planes (allocated when pcr_coeffs first asks for them)
    int16_t* d_dc = nullptr;
    int16_t* d_head = nullptr;
    int16_t* d_vals = nullptr;
    int decoded_k = 0;            // fidelity of the state the coefficient lists and side data hold (0: none)
    int lists_k = 0;              // fidelity of the last decode, whatever rows it decoded
    bool planes_current = false;  // d_planes holds the coefficients of the last decode
    ScanTab* d_tabs = nullptr;
    ScanScript* d_script = nullptr;
    ScanAux* d_saux = nullptr;
    uint64_t* d_aux = nullptr;
    std::vector<ScanAux> saux;
    ScanDesc* d_scans = nullptr;
    ImgDesc* d_imgs = nullptr;
    uint32_t* d_seg = nullptr;
    Item* d_items = nullptr;
    Unit* d_units = nullptr;
    uint32_t* d_unit_prefix = nullptr;
    uint16_t* d_qtab = nullptr;
    uint32_t* d_order = nullptr;  // processing order of the images (slices are runs of it)
    MsDesc* d_ms = nullptr;       // per-image table of pcr_msssim (built on first use)
    size_t ms_scratch = 0;        // bytes of scratch pcr_msssim needs
    uint64_t ms_floats = 0;       // floats of all pyramids (the sums follow them)
    int upsampling = PCR_UPSAMPLE_REPLICATE;
    uint8_t* d_chroma = nullptr;  // chroma sample planes between the two passes of triangle upsampling
    CropRect* d_crops = nullptr;  // crop rectangles of the last pcr_decode_tensor (allocated on first use)
    int* d_status = nullptr;
    std::vector<int> h_status;
    std::vector<std::pair<void*, size_t>> bufs;   // every device buffer of the record with its size
    std::vector<std::pair<void*, size_t>> stages; // host blocks the tables were built in (their copies may be in flight)
    cudaStream_t up_stream = nullptr;             // pcr_open's uploads and memsets (never the default stream:
                                                  // that one would wait for every other record's decode)
    cudaEvent_t ev_ready = nullptr;               // the record's device state is set up
    cudaEvent_t ev_done = nullptr;                // end of the last decode enqueued
    bool decode_enqueued = false;
    // identity of the record for the cache of closed records (pcr_set_record_cache): valid when key_len != 0
    uint64_t key_hash = 0;
    size_t key_len = 0;
    uint32_t key_env = 0;                         // the tuning variables read when it was opened
    size_t device_bytes = 0;                      // what its device buffers add up to
    // optional stage timing
    bool profiling = false;
    std::vector<cudaEvent_t> events;
    std::vector<pcr_stage_time> profile;  // names and launch counts of the last decode
};

static const int kMaxStages = 16;

static inline uint32_t rd32(const uint8_t* p) { return (uint32_t)p[0] | ((uint32_t)p[1] << 8) | ((uint32_t)p[2] << 16) | ((uint32_t)p[3] << 24); }
static inline uint64_t rd64(const uint8_t* p) { return (uint64_t)rd32(p) | ((uint64_t)rd32(p + 4) << 32); }

// Writes the list of pixel work units at set-up, and every (scan, image)'s place in the segment table into its
// descriptor (the host has the places in an array of their own: the descriptors' cache lines belong to the threads that
// made them): block = position of the processing order.
__global__ void __launch_bounds__(128) units_kernel(const ImgDesc* __restrict__ imgs, const uint32_t* __restrict__ order,
                                                    const uint32_t* __restrict__ prefix, Unit* __restrict__ units, uint32_t unit_mcus, uint32_t unit_rows,
                                                    ScanDesc* __restrict__ scans, const uint32_t* __restrict__ seg_base, uint32_t G, uint32_t bpm) {
    const uint32_t img = order[blockIdx.x];
    const ImgDesc im = imgs[img];
    for (uint32_t g = threadIdx.x; g < G; g += 128) scans[(size_t)g * gridDim.x + img].seg_base = seg_base[(size_t)g * gridDim.x + img];
    const uint32_t per_row = (im.mx + unit_mcus - 1) / unit_mcus, n = per_row * ((im.my + unit_rows - 1) / unit_rows);
    Unit* dst = units + prefix[blockIdx.x];
    for (uint32_t j = threadIdx.x; j < n; j += 128) {
        Unit un;
        un.img = img; un.mrow = (uint16_t)(j / per_row * unit_rows); un.mcol0 = (uint16_t)((j % per_row) * unit_mcus);
        un.mx = (uint16_t)im.mx; un.my = (uint16_t)im.my; un.W = (uint16_t)im.W; un.H = (uint16_t)im.H;
        un.mcus = im.blk_base / bpm; un.out_off = im.out_off;
        dst[j] = un;
    }
}

namespace {

struct TableRef { uint32_t off = 0; };   // offset of the 16 length counts of a DHT table body; 0 = undefined

struct ImageParse {
    uint32_t W = 0, H = 0;
    int cid[3] = {0, 0, 0}, tq[3] = {0, 0, 0};
    uint16_t q[4][64];
    bool qdef[4] = {false, false, false, false};
    TableRef dc[4], ac[4];
    uint32_t ri = 0;
    bool have_frame = false;
    bool sequential = false;      // SOF0: one interleaved scan carries whole blocks
    int hs = 2, vs = 2, nc = 3;   // luminance blocks per MCU, components
};

struct ScanParse {
    ScanScript sc;
    uint32_t tab[3];       // table body offset per scan component (0 when the scan uses none)
    uint32_t tab_ac[3];    // sequential scans: the AC table per component (tab then holds the DC tables)
    uint32_t data_off, data_end, ri;
};

// Validate one DHT table body at p (inside [p, end)): returns its length or 0.
size_t check_dht_body(const uint8_t* p, size_t avail) {
    if (avail < 16) return 0;
    uint32_t code = 0, n = 0;
    for (int l = 1; l <= 16; ++l) {
        code += p[l - 1];
        n += p[l - 1];
        if (code > (1u << l)) return 0;
        code <<= 1;
    }
    if (n > 256 || 16 + (size_t)n > avail) return 0;
    return 16 + n;
}

// Walk the marker segments of chunk [off, off+len) of one image up to and including its SOS.
int parse_chunk(const uint8_t* rec, uint64_t off, uint32_t len, bool first, ImageParse& im, ScanParse& out) {
    uint64_t p = off, end = off + len;
    if (first) {
        if (len < 4 || rec[p] != 0xFF || rec[p + 1] != 0xD8) return PCR_E_FORMAT;
        p += 2;
    }
    for (;;) {
        if (p + 4 > end || rec[p] != 0xFF) return PCR_E_FORMAT;
        while (p < end && rec[p] == 0xFF) ++p;
        if (p >= end) return PCR_E_FORMAT;
        int mk = rec[p++];
        if (p + 2 > end) return PCR_E_FORMAT;
        uint32_t L = ((uint32_t)rec[p] << 8) | rec[p + 1];
        if (L < 2 || p + L > end) return PCR_E_FORMAT;
        const uint8_t* s = rec + p + 2;
        uint32_t sl = L - 2;
        if (mk == 0xDB) {
            uint32_t q = 0;
            while (q < sl) {
                int pq = s[q] >> 4, tq = s[q] & 15;
                ++q;
                if (tq > 3 || pq > 1 || q + (pq ? 128u : 64u) > sl) return PCR_E_FORMAT;
                for (int k = 0; k < 64; ++k) {
                    im.q[tq][k] = pq ? (uint16_t)((s[q] << 8) | s[q + 1]) : s[q];
                    q += pq ? 2 : 1;
                }
                im.qdef[tq] = true;
            }
        } else if (mk == 0xC2 || mk == 0xC0) {            // progressive / baseline sequential, Huffman
            if (im.have_frame || sl < 9 || s[0] != 8 || (s[5] != 3 && s[5] != 1) || sl < 6u + 3u * s[5]) return PCR_E_FORMAT;
            im.sequential = mk == 0xC0;
            im.H = ((uint32_t)s[1] << 8) | s[2];
            im.W = ((uint32_t)s[3] << 8) | s[4];
            im.nc = s[5];
            for (int c = 0; c < im.nc; ++c) {
                im.cid[c] = s[6 + 3 * c];
                int hv = s[7 + 3 * c];
                im.tq[c] = s[8 + 3 * c];
                if (im.tq[c] > 3) return PCR_E_FORMAT;
                // luminance 1 or 2 blocks per MCU in each direction, chroma one: 4:4:4, 4:2:2, 4:4:0, 4:2:0
                if (c == 0) { im.hs = hv >> 4; im.vs = hv & 15; if (im.hs < 1 || im.hs > 2 || im.vs < 1 || im.vs > 2) return PCR_E_FORMAT; }
                else if (hv != 0x11) return PCR_E_FORMAT;
            }
            if (im.nc == 1) im.hs = im.vs = 1;                // a lone component is never interleaved: no MCU padding
            if (im.W == 0 || im.H == 0) return PCR_E_FORMAT;
            im.have_frame = true;
        } else if (mk == 0xC4) {
            uint32_t q = 0;
            while (q < sl) {
                int tc = s[q] >> 4, th = s[q] & 15;
                if (tc > 1 || th > 3) return PCR_E_FORMAT;
                size_t n = check_dht_body(s + q + 1, sl - q - 1);
                if (!n) return PCR_E_FORMAT;
                (tc ? im.ac[th] : im.dc[th]).off = (uint32_t)(p + 2 + q + 1);
                q += 1 + (uint32_t)n;
            }
        } else if (mk == 0xDD) {
            if (sl != 2) return PCR_E_FORMAT;
            im.ri = ((uint32_t)s[0] << 8) | s[1];
        } else if (mk == 0xDA) {
            if (!im.have_frame || sl < 1) return PCR_E_FORMAT;
            int ns = s[0];
            if (ns < 1 || ns > 3 || sl != (uint32_t)(4 + 2 * ns)) return PCR_E_FORMAT;
            ScanScript& sc = out.sc;
            memset(&sc, 0, sizeof sc);
            sc.ncomp = ns;
            int td[3] = {0, 0, 0}, ta[3] = {0, 0, 0};
            for (int i = 0; i < ns; ++i) {
                int id = s[1 + 2 * i], found = -1;
                for (int c = 0; c < im.nc; ++c) if (im.cid[c] == id) found = c;
                if (found < 0) return PCR_E_FORMAT;
                for (int j = 0; j < i; ++j) if (sc.comp[j] >= found) return PCR_E_FORMAT;   // frame order
                sc.comp[i] = found;
                td[i] = s[2 + 2 * i] >> 4;
                ta[i] = s[2 + 2 * i] & 15;
                if (td[i] > 3 || ta[i] > 3) return PCR_E_FORMAT;
            }
            sc.Ss = s[1 + 2 * ns]; sc.Se = s[2 + 2 * ns];
            sc.Ah = s[3 + 2 * ns] >> 4; sc.Al = s[3 + 2 * ns] & 15;
            if (sc.Ss > sc.Se || sc.Se > 63 || sc.Al > 13) return PCR_E_FORMAT;
            if (im.sequential) {
                if (sc.Ss != 0 || sc.Se != 63 || sc.Ah != 0 || sc.Al != 0 || ns != im.nc) return PCR_E_FORMAT;
            } else if (sc.Ss == 0 && sc.Se != 0) return PCR_E_FORMAT;
            if (sc.Ss > 0 && ns != 1) return PCR_E_FORMAT;
            if (ns > 1 && ns != im.nc) return PCR_E_FORMAT; // interleaved scans hold all three components
            if (sc.Ah != 0 && sc.Ah != sc.Al + 1) return PCR_E_FORMAT;
            for (int i = 0; i < 3; ++i) out.tab[i] = out.tab_ac[i] = 0;
            for (int i = 0; i < ns && im.sequential; ++i) {
                out.tab_ac[i] = im.ac[ta[i]].off;
                if (!out.tab_ac[i]) return PCR_E_FORMAT;
            }
            for (int i = 0; i < ns; ++i) {
                if (sc.Ss == 0 && sc.Ah == 0) { out.tab[i] = im.dc[td[i]].off; if (!out.tab[i]) return PCR_E_FORMAT; }
                if (sc.Ss > 0) { out.tab[i] = im.ac[ta[i]].off; if (!out.tab[i]) return PCR_E_FORMAT; }
            }
            out.data_off = (uint32_t)(p + L);
            out.data_end = (uint32_t)end;
            out.ri = im.ri;
            return PCR_OK;
        } else if ((mk >= 0xC0 && mk <= 0xCF) || (mk >= 0xD0 && mk <= 0xD9)) {
            return PCR_E_FORMAT;     // other frame types, stray restart / SOI / EOI markers
        }
        p += L;
    }
}

void free_device(pcr_record* r) {
    // nothing is handed on before the record's set-up and its last decode have finished
    if (r->up_stream) cudaStreamSynchronize(r->up_stream);
    if (r->ev_done && r->decode_enqueued) cudaEventSynchronize(r->ev_done);
    if (r->ev_ready) pool_event_put(r->ev_ready, r->device);
    r->ev_ready = nullptr;
    if (r->up_stream) pool_stream_put(r->up_stream, r->device);
    r->up_stream = nullptr;
    r->decode_enqueued = false;
    for (cudaStream_t q : r->streams) pool_stream_put(q, r->device);
    r->streams.clear();
    if (r->ev_start) pool_event_put(r->ev_start, r->device);
    r->ev_start = nullptr;
    if (r->ev_chain) pool_event_put(r->ev_chain, r->device);
    r->ev_chain = nullptr;
    for (cudaEvent_t e : r->ev_index) pool_event_put(e, r->device);
    r->ev_index.clear();
    if (r->ev_fork) pool_event_put(r->ev_fork, r->device);
    r->ev_fork = nullptr;
    if (r->copy_stream) pool_stream_put(r->copy_stream, r->device);
    r->copy_stream = nullptr;
    if (r->side_stream) pool_stream_put(r->side_stream, r->device);
    r->side_stream = nullptr;
    if (r->ev_side) pool_event_put(r->ev_side, r->device);
    r->ev_side = nullptr;
    for (cudaEvent_t e : r->ev_copy) pool_event_put(e, r->device);
    r->ev_copy.clear();
    for (cudaEvent_t e : r->ev_join) pool_event_put(e, r->device);
    r->ev_join.clear();
    for (cudaEvent_t e : r->events) cudaEventDestroy(e);
    r->events.clear();
    // buffers go back to the cache once the record's last decode has finished
    if (r->ev_done) {
        if (r->decode_enqueued) cudaEventSynchronize(r->ev_done);
        pool_event_put(r->ev_done, r->device);
        r->ev_done = nullptr;
    }
    for (auto& b : r->bufs) dev_release(b.first, b.second, r->device);
    r->bufs.clear();
    for (auto& b : r->stages) host_release(b.first, b.second);
    r->stages.clear();
}

template <class T>
int take(pcr_record* r, T** dst, size_t bytes) {
    *dst = static_cast<T*>(dev_alloc(bytes, r->device));
    if (!*dst) return PCR_E_NOMEM;
    r->bufs.push_back({*dst, bytes});
    return PCR_OK;
}

// A run of tables laid out one behind the other, alike in a page-locked host block and on the device.
struct Tables {
    size_t bytes = 0;
    uint8_t *host = nullptr, *dev = nullptr;
    size_t add(size_t n) { const size_t at = bytes; bytes = (bytes + std::max<size_t>(n, 1) + 15) & ~(size_t)15; return at; }
    template <class T> T* h(size_t at) const { return reinterpret_cast<T*>(host + at); }
    template <class T> T* d(size_t at) const { return reinterpret_cast<T*>(dev + at); }
    std::unique_ptr<uint8_t[]> pageable;              // (no device: the record is still validated)
    int allocate(pcr_record* r, bool on_device = true) {
        if (!on_device) {
            pageable.reset(new uint8_t[bytes]);
            host = pageable.get();
            return PCR_OK;
        }
        host = static_cast<uint8_t*>(host_alloc(bytes));
        if (!host) return PCR_E_NOMEM;
        r->stages.push_back({host, bytes});
        return take(r, &dev, bytes);
    }
    int copy(pcr_record* r, size_t n) const {
        return !n || cudaMemcpyAsync(dev, host, n, cudaMemcpyHostToDevice, r->up_stream) == cudaSuccess ? PCR_OK : PCR_E_CUDA;
    }
};

int open_impl(const uint8_t* rec, size_t len, pcr_record* r) {
    if (len < 64 || len >= (1ull << 32)) return PCR_E_FORMAT;
    if (memcmp(rec, "PCR1", 4) != 0 || rd32(rec + 4) != 1) return PCR_E_FORMAT;
    uint32_t N = rd32(rec + 8), G = rd32(rec + 12);
    uint64_t meta_off = rd64(rec + 24), index_off = rd64(rec + 32), data_off = rd64(rec + 40), total = rd64(rec + 48);
    if (N == 0 || G == 0 || G > 64 || N > (1u << 24)) return PCR_E_FORMAT;
    if (total != len) return PCR_E_FORMAT;
    // (offsets are compared with what is left behind them: a sum with one near 2^64 would wrap)
    const uint64_t index_len = 8ull * (G + 1) + 16ull * G * N;
    if (meta_off < 64 || meta_off > len || 16ull * N > len - meta_off) return PCR_E_FORMAT;
    if (index_off < 64 || index_off > len || index_len > len - index_off) return PCR_E_FORMAT;
    if (data_off > len || data_off < index_off + index_len) return PCR_E_FORMAT;
    r->host = rec; r->len = len; r->N = (int)N; r->G = (int)G;
    r->group_end.resize(G + 1);
    for (uint32_t g = 0; g <= G; ++g) r->group_end[g] = rd64(rec + index_off + 8ull * g);
    if (r->group_end[0] != data_off) return PCR_E_FORMAT;
    for (uint32_t g = 1; g <= G; ++g)
        if (r->group_end[g] < r->group_end[g - 1] || r->group_end[g] > len) return PCR_E_FORMAT;
    const uint8_t* chunk = rec + index_off + 8ull * (G + 1);

    const bool on_device = cudaGetDevice(&r->device) == cudaSuccess;
    if (on_device && !(r->up_stream = pool_stream_get(r->device))) return PCR_E_CUDA;
    Tables T;
    const size_t at_script = T.add(sizeof(ScanScript) * G), at_saux = T.add(sizeof(ScanAux) * G), at_scans = T.add(sizeof(ScanDesc) * G * N),
                 at_imgs = T.add(sizeof(ImgDesc) * N), at_qtab = T.add(384ull * N), at_prefix = T.add(4ull * (N + 1)), at_order = T.add(4ull * N),
                 at_base = T.add(4ull * G * N), at_group = T.add(12ull * N), at_long = T.add(4ull * G * N);
    if (int rc = T.allocate(r, on_device)) return rc;
    ScanDesc* const scans = T.h<ScanDesc>(at_scans);
    ImgDesc* const imgs = T.h<ImgDesc>(at_imgs);
    uint16_t* const qtab = T.h<uint16_t>(at_qtab);
    r->info.resize(N); r->blk_base.resize(N); r->nblk.resize(N);
    r->script.resize(G);
    // every image's chunks are walked independently (a few host threads for large records); the
    // running sums over images follow in one serial pass
    struct Counts {                                                  // of a (scan, image)
        uint32_t nseg, bytes;                                        // restart intervals, entropy-coded bytes
        uint32_t chain() const { return (uint32_t)((float)bytes / (float)nseg); }      // bytes of an interval, on average
    };
    std::vector<Counts> counts((size_t)G * N);
    std::vector<uint32_t> image_bytes(N);                            // entropy-coded bytes
    std::vector<uint8_t> one_interval(N, 0);                         // some scan of the image is one restart interval
    uint8_t sampling0 = 0;
    auto parse_image = [&](uint32_t i) -> int {
        ImageParse im;
        ScanScript script[64];
        uint32_t sum = 0;
        const uint8_t* m = rec + meta_off + 16ull * i;
        for (uint32_t g = 0; g < G; ++g) {
            const uint8_t* c = chunk + 16ull * ((uint64_t)g * N + i);
            uint64_t off = rd64(c);
            uint32_t clen = rd32(c + 8);
            uint64_t padded = ((uint64_t)clen + 15) & ~15ull;
            if ((off & 15) || off < r->group_end[g] || off > r->group_end[g + 1] || padded > r->group_end[g + 1] - off) return PCR_E_FORMAT;
            if (clen >= (1u << 28)) return PCR_E_FORMAT;        // bit positions inside a scan are 32-bit
            ScanParse sp;
            int rc = parse_chunk(rec, off, clen, g == 0, im, sp);
            if (rc) return rc;
            script[g] = sp.sc;
            ScanDesc& sd = scans[(size_t)g * N + i];
            sd.data_off = sp.data_off; sd.data_end = sp.data_end; sd.ri = sp.ri;
            // up to two distinct tables per scan
            sd.tab_ac[0] = sp.tab_ac[0]; sd.tab_ac[1] = 0; sd.slots_ac = 0;
            for (int ci = 1; ci < sp.sc.ncomp && sp.tab_ac[0]; ++ci) {
                if (sp.tab_ac[ci] == sd.tab_ac[0]) continue;
                if (sd.tab_ac[1] == 0) sd.tab_ac[1] = sp.tab_ac[ci];
                if (sp.tab_ac[ci] != sd.tab_ac[1]) return PCR_E_FORMAT;
                sd.slots_ac |= 1u << (2 * ci);
            }
            sd.tab_off[0] = sp.tab[0]; sd.tab_off[1] = 0; sd.slots = 0;
            for (int ci = 1; ci < sp.sc.ncomp; ++ci) {
                if (sp.tab[ci] == sd.tab_off[0]) continue;
                if (sd.tab_off[1] == 0) sd.tab_off[1] = sp.tab[ci];
                if (sp.tab[ci] != sd.tab_off[1]) return PCR_E_FORMAT;
                sd.slots |= 1u << (2 * ci);
            }
            uint32_t mx = (im.W + 8 * im.hs - 1) / (8 * im.hs), my = (im.H + 8 * im.vs - 1) / (8 * im.vs);
            uint64_t total_mcu;
            if (sp.sc.ncomp > 1) total_mcu = (uint64_t)mx * my;
            else {
                uint32_t wc = sp.sc.comp[0] == 0 ? im.W : (im.W + im.hs - 1) / im.hs, hc = sp.sc.comp[0] == 0 ? im.H : (im.H + im.vs - 1) / im.vs;
                total_mcu = (uint64_t)((wc + 7) / 8) * ((hc + 7) / 8);
            }
            sd.nseg = sd.ri ? (uint32_t)((total_mcu + sd.ri - 1) / sd.ri) : 1u;
            counts[(size_t)g * N + i] = Counts{sd.nseg, sd.data_end - sd.data_off};
            if (sd.nseg == 1) one_interval[i] = 1;
            sum += sd.data_end - sd.data_off;
        }
        image_bytes[i] = sum;
        if (!im.have_frame) return PCR_E_FORMAT;
        if (rd32(m + 4) != im.W || rd32(m + 8) != im.H) return PCR_E_FORMAT;   // metadata and frame header agree
        for (int c = 0; c < im.nc; ++c) {
            if (!im.qdef[im.tq[c]]) return PCR_E_FORMAT;
            memcpy(&qtab[(size_t)i * 192 + 64 * c], im.q[im.tq[c]], 128);
        }
        // one script and one sampling per record: the first image's
        const uint8_t samp = (uint8_t)(im.hs | (im.vs << 2) | (im.nc << 4));
        if (i == 0) { sampling0 = samp; std::copy(script, script + G, r->script.begin()); }
        else if (samp != sampling0 || memcmp(script, r->script.data(), sizeof(ScanScript) * G) != 0) return PCR_E_FORMAT;
        pcr_image_info& inf = r->info[i];
        inf.width = im.W; inf.height = im.H; inf.label = (int32_t)rd32(m); inf.rsvd = 0;
        inf.out_bytes = 3ull * im.W * im.H;
        imgs[i].W = im.W; imgs[i].H = im.H;
        imgs[i].mx = (im.W + 8 * im.hs - 1) / (8 * im.hs); imgs[i].my = (im.H + 8 * im.vs - 1) / (8 * im.vs);
        return PCR_OK;
    };
    {
        const unsigned hw = std::max(1u, std::thread::hardware_concurrency());
        const unsigned nthreads = std::min({8u, hw, N / 64 + 1u});
        std::vector<int> rcs(nthreads, PCR_OK);
        // The heads of an image's chunks lie all over the record: those of the next image are requested while
        // one is walked (the walk waited for memory most of its time).
        auto request = [&](uint32_t i) {
            for (uint32_t g = 0; g < G; ++g) {
                const uint64_t off = rd64(chunk + 16ull * ((uint64_t)g * N + i));
                if (off >= len) continue;
                const uint8_t* p = rec + off;
                for (size_t b = 0; b < (g == 0 ? 384u : 128u) && off + b < len; b += 64) __builtin_prefetch(p + b);
            }
        };
        std::atomic<uint32_t> next_image{1};
        auto work = [&](unsigned t) {                    // (runs of images: the first threads work while the others start)
            for (;;) {
                const uint32_t i0 = next_image.fetch_add(16), i1 = std::min(N, i0 + 16);
                if (i0 >= N) return;
                request(i0);
                for (uint32_t i = i0; i < i1; ++i) {
                    if (i + 1 < i1) request(i + 1);
                    const int rc = parse_image(i);
                    if (rc != PCR_OK) { rcs[t] = rc; return; }
                }
            }
        };
        if (const int rc = parse_image(0)) return rc;
        std::vector<std::thread> pool;
        pool.reserve(nthreads);
        try {
            for (unsigned t = 1; t < nthreads; ++t) pool.emplace_back(work, t);
        } catch (const std::system_error&) {}            // (no more threads to be had: those there are and this one do it)
        work(0);
        for (auto& th : pool) th.join();
        for (int rc : rcs) if (rc != PCR_OK) return rc;
    }
    uint64_t blocks = 0, out_off = 0, segs = 0;
    r->hs = sampling0 & 3; r->vs = (sampling0 >> 2) & 3; r->nc = sampling0 >> 4;
    const uint32_t bpm = (uint32_t)(r->hs * r->vs + (r->nc == 3 ? 2 : 0));      // blocks per MCU
    r->unit_mcus = kUnitMcus[sampling_code(r->hs, r->vs, r->nc)];
    r->unit_rows = kUnitRows[sampling_code(r->hs, r->vs, r->nc)];
    uint64_t max_items = 1;
    uint32_t* const seg_base = T.h<uint32_t>(at_base);
    for (size_t j = 0; j < (size_t)G * N; ++j) {
        seg_base[j] = (uint32_t)segs;
        segs += (uint64_t)counts[j].nseg + 1;               // one closing entry per (scan, image)
        if (segs >= (1ull << 32)) return PCR_E_FORMAT;
        max_items += counts[j].nseg / kSegsPerItem + 1 + counts[j].nseg / (kSegsPerItem / 2) + 1;     // (the pairs' items too)
    }
    bool single = false;                              // any scan of any image is one restart interval
    for (uint32_t i = 0; i < N; ++i) {
        single = single || one_interval[i];
        pcr_image_info& inf = r->info[i];
        inf.out_offset = out_off;
        out_off += (inf.out_bytes + 127) & ~127ull;
        if (imgs[i].W & 15u) r->widths_mult16 = false;
        r->dc_refine_chunks = std::max(r->dc_refine_chunks, std::min(8u, (imgs[i].mx * imgs[i].my + 255u) / 256u));
        r->blk_base[i] = blocks; r->nblk[i] = (uint64_t)bpm * imgs[i].mx * imgs[i].my;
        imgs[i].blk_base = blocks; imgs[i].out_off = inf.out_offset;
        blocks += r->nblk[i];
    }
    // 16 spare bytes behind the last image: the tensor epilogue reads pixels as aligned words and may
    // touch up to 8 bytes past a pixel pair
    r->total_blocks = blocks; r->out_bytes = out_off + 16; r->total_segs = segs;

    // side data of the AC scans: one or two words per block for a first pass, four for a refinement
    const uint64_t total_mcus = blocks / bpm;
    uint64_t aux_words = 0;
    r->saux.assign(G, ScanAux{});
    int n_refine[3] = {0, 0, 0};
    for (uint32_t s = 0; s < G; ++s)
        if (r->script[s].Ss > 0 && r->script[s].Ah > 0 && ++n_refine[r->script[s].comp[0]] > 4) return PCR_E_FORMAT;
    // An AC position is sent by one first pass, before any refinement of it (T.81 B.2.3: only the first scan of a band has
    // Ah = 0).  The lists rely on it: at most kMaxFirst first passes of a component reach beyond position 7, first
    // passes are expanded before refinements, and no two scans write the same values.
    uint64_t sent[3] = {0, 0, 0};
    for (const ScanScript& sc : r->script) {
        const uint64_t band = (sc.Se == 63 ? ~0ull : (1ull << (sc.Se + 1)) - 1ull) & ~((1ull << std::max(1, sc.Ss)) - 1ull);
        for (int i = 0; i < sc.ncomp; ++i) {
            if (sc.Ah == 0 && (sent[sc.comp[i]] & band)) return PCR_E_FORMAT;
            sent[sc.comp[i]] |= band;
        }
    }
    uint64_t n_tabs = 0;
    for (uint32_t s = 0; s < G; ++s) {
        const ScanScript& sc = r->script[s];
        ScanAux& ax = r->saux[s];
        ax.ntab = sc.Ss > 0 ? 1 : (sc.Se == 63 ? 4 : (sc.Ah == 0 ? 2 : 0));
        ax.tab0 = (uint32_t)n_tabs;
        n_tabs += (uint64_t)N * (uint64_t)ax.ntab;
        if (sc.Ss == 0 && sc.Se != 63) continue;
        ax.stride = sc.Ah ? 4u : (sc.Se >= 8 ? 2u : 1u);
        ax.base = aux_words;
        if (sc.Ss == 0) { aux_words += 2 * blocks; continue; }
        aux_words += (sc.comp[0] == 0 ? (uint64_t)(r->hs * r->vs) : 1ull) * total_mcus * ax.stride;
        aux_words = (aux_words + 1) & ~1ull;      // 16-byte alignment of every scan's area
        if (sc.Ah) {
            // positions already non-zero = union of the masks of earlier scans on this band; an
            // earlier scan is covered by a later refinement whose band contains its own
            std::vector<int> src;
            for (uint32_t t = 0; t < s; ++t) {
                const ScanScript& st = r->script[t];
                if (st.Ss == 0 || st.comp[0] != sc.comp[0] || st.Ss > sc.Se || sc.Ss > st.Se) continue;
                src.push_back((int)t);
            }
            std::vector<int> keep;
            for (int t : src) {
                bool covered = false;
                for (int u : src)
                    if (u > t && r->script[u].Ah && r->script[u].Ss <= r->script[t].Ss && r->script[u].Se >= r->script[t].Se) covered = true;
                if (!covered) keep.push_back(t);
            }
            if (keep.empty() || keep.size() > 4) return PCR_E_FORMAT;
            ax.nsrc = (int)keep.size();
            for (size_t i = 0; i < keep.size(); ++i) ax.src[i] = keep[i];
        }
    }

    // What has to be zero lies together; zeroing it (0.1 ms for 1024 ImageNet-shaped images) passes beside the rest of this call.
    Tables Z;
    const size_t at_aux = Z.add((size_t)aux_words * 8), at_ubuf = Z.add(len + 256), at_dc = Z.add((size_t)blocks * 2), at_head = Z.add((size_t)blocks * 16),
                 at_seg = Z.add((size_t)(segs + 1) * 4), at_status = Z.add((size_t)N * 4), at_sync = Z.add((4 + 12 * (size_t)N) * 4);
    if (on_device) {
        if (int rc = take(r, &Z.dev, Z.bytes)) return rc;
        r->d_aux = Z.d<uint64_t>(at_aux); r->d_ubuf = Z.d<uint8_t>(at_ubuf); r->d_dc = Z.d<int16_t>(at_dc); r->d_head = Z.d<int16_t>(at_head);
        r->d_seg = Z.d<uint32_t>(at_seg); r->d_status = Z.d<int>(at_status); r->d_chain_sync = Z.d<uint32_t>(at_sync);
        if (cudaMemsetAsync(Z.dev, 0, Z.bytes, r->up_stream) != cudaSuccess) return PCR_E_CUDA;
    }

    // dependency waves of the script: a scan waits for every earlier scan that touches an
    // overlapping coefficient band of one of its components
    r->wave_of_scan.assign(G, 0);
    for (uint32_t s = 0; s < G; ++s) {
        int w = 0;
        for (uint32_t t = 0; t < s; ++t) {
            bool share = false;
            for (int a = 0; a < r->script[s].ncomp; ++a)
                for (int b = 0; b < r->script[t].ncomp; ++b)
                    if (r->script[s].comp[a] == r->script[t].comp[b]) share = true;
            if (share && r->script[s].Ss <= r->script[t].Se && r->script[t].Ss <= r->script[s].Se)
                w = std::max(w, r->wave_of_scan[t] + 1);
        }
        r->wave_of_scan[s] = w;
        r->n_waves = std::max(r->n_waves, w + 1);
    }
    r->wave_scans.assign(r->n_waves, {});
    for (uint32_t s = 0; s < G; ++s) r->wave_scans[r->wave_of_scan[s]].push_back((int)s);
    // pairs of AC refinements
    r->pair_of.assign(G, -1);
    {
        std::vector<int> wave(G, 0);
        bool any = false;
        for (uint32_t s = 0; s < G; ++s) {
            const ScanScript& sc = r->script[s];
            int w = 0, prev = -1, before = 0;     // the last earlier scan that touches the band; the wave all others allow
            for (uint32_t t = 0; t < s; ++t) {
                const ScanScript& st = r->script[t];
                bool share = false;
                for (int a = 0; a < sc.ncomp; ++a)
                    for (int b = 0; b < st.ncomp; ++b)
                        if (sc.comp[a] == st.comp[b]) share = true;
                if (!share || sc.Ss > st.Se || st.Ss > sc.Se) continue;
                if (prev >= 0) before = std::max(before, wave[prev] + 1);
                prev = (int)t;
                w = std::max(w, wave[t] + 1);
            }
            const ScanScript* sp = prev >= 0 ? &r->script[prev] : nullptr;
            bool pair = sp && sc.Ss > 0 && sc.Ah && sp->Ss == sc.Ss && sp->Se == sc.Se && sp->Ah && r->pair_of[prev] < 0 && before <= wave[prev];
            for (uint32_t i = 0; pair && i < N; ++i) {
                const ScanDesc &x = scans[(size_t)prev * N + i], &y = scans[(size_t)s * N + i];
                pair = x.nseg == y.nseg && x.ri == y.ri;
            }
            if (pair) { r->pair_of[s] = prev; w = wave[prev]; any = true; }
            wave[s] = w;
        }
        int n = 0;
        for (uint32_t s = 0; s < G; ++s) {
            n = std::max(n, wave[s] + 1);
            if (r->script[s].Ah == 0 && wave[s] != r->wave_of_scan[s]) any = false;    // (first passes keep their place)
        }
        if (any) {
            r->paired_waves.assign(n, {});
            for (uint32_t s = 0; s < G; ++s) r->paired_waves[wave[s]].push_back((int)s);
        } else r->pair_of.assign(G, -1);
    }
    if (const char* e = getenv("PCR_REFINE_CTAS")) r->refine_ctas = atof(e);
    if (const char* e = getenv("PCR_PAIRS")) r->pairs = atoi(e) != 0;
    if (const char* e = getenv("PCR_SEQ_CTAS")) r->seq_ctas = std::max(0, atoi(e));
    if (const char* e = getenv("PCR_INDEX_CTAS")) r->index_ctas = std::max(0, atoi(e));
    if (const char* e = getenv("PCR_LONG_CTAS")) r->long_ctas = std::max(0, atoi(e));
    if (const char* e = getenv("PCR_PACK_WARPS")) r->pack_warps = std::max(0, atoi(e));
    if (const char* e = getenv("PCR_SHORT_WARPS")) r->short_warps = (uint32_t)std::max(0, atoi(e));
    // slices: enough images each to fill the machine, few enough to keep launches cheap
    {
        // four at most: one record decodes as fast with four slices as with eight, and two records
        // in flight then stay close to the eight hardware queues that streams are mapped onto
        int want = (int)std::min<uint32_t>(4, std::max<uint32_t>(1, N / 128));
        if (const char* e = getenv("PCR_SLICES")) want = std::max(1, std::min(64, atoi(e)));
        r->n_slices = (int)std::min<uint32_t>((uint32_t)want, N);
        r->slice_img.resize(r->n_slices + 1);
        for (int g = 0; g <= r->n_slices; ++g) r->slice_img[g] = (uint32_t)((uint64_t)N * g / r->n_slices);
    }
    // Processing order of the images: a slice is a run of this order.  The time a slice needs for
    // its entropy waves is set by its longest restart intervals, so the images are sorted by their
    // entropy-coded bytes per MCU row, most first: the slice of the heaviest rows starts first, slices
    // of light images finish their waves early and their pixel stage overlaps the waves of the heavy
    // ones.  (By width alone, the first version of this order: 2 % slower on the ImageNet-shaped record.)
    uint32_t* const order = T.h<uint32_t>(at_order);
    for (uint32_t i = 0; i < N; ++i) order[i] = i;
    if (r->n_slices > 1) {
        std::vector<double> key(N);
        for (uint32_t i = 0; i < N; ++i) key[i] = (double)image_bytes[i] / (double)std::max<uint32_t>(1, imgs[i].my);
        std::stable_sort(order, order + N, [&](uint32_t a, uint32_t b) { return key[a] > key[b]; });
    }
    Tables TI;
    TI.add(sizeof(Item) * max_items);
    if (int rc = TI.allocate(r, on_device)) return rc;
    Item* const items = TI.h<Item>(0);
    uint32_t n_items = 0;
    r->chain_bytes.assign(G, 0); r->chain_squares.assign(G, 0); r->item_begin.assign((size_t)r->n_slices * G, 0); r->item_count.assign((size_t)r->n_slices * G, 0);
    // A scan that is one restart interval of at least this many bytes goes to the kernels for long
    // intervals; DC refinement scans have no items at all (see dc_refine_image).
    uint32_t long_min = 64;
    if (const char* e = getenv("PCR_LONG_MIN_BYTES")) long_min = (uint32_t)std::max(0, atoi(e));
    auto is_long = [&](int s, uint32_t i) {
        const ScanDesc& sd = scans[(size_t)s * N + i];
        return sd.nseg == 1 && sd.data_end - sd.data_off >= long_min && sd.data_end - sd.data_off < (1u << 27);   // (the chains count half bits)
    };
    // the AC refinements of one component of one image go together: all of them one interval each,
    // at least one of them long
    std::vector<uint8_t> grouped((size_t)N * 3, 0);
    for (uint32_t i = 0; single && i < N; ++i)
        for (int c = 0; c < 3; ++c) {
            bool any = false, one_interval = true, big = false;
            for (uint32_t s = 0; s < G; ++s) {
                const ScanScript& sc = r->script[s];
                if (sc.Ss == 0 || sc.Ah == 0 || sc.comp[0] != c) continue;
                any = true;
                const ScanDesc& sd = scans[(size_t)s * N + i];
                one_interval = one_interval && sd.nseg == 1 && sd.data_end - sd.data_off < (1u << 27);
                big = big || is_long((int)s, i);
            }
            grouped[(size_t)i * 3 + c] = any && one_interval && big;
        }
    auto takes_long_kernel = [&](int s, uint32_t i) {
        const ScanScript& sc = r->script[s];
        if (sc.Ss > 0 && sc.Ah != 0) return grouped[(size_t)i * 3 + sc.comp[0]] != 0;
        return is_long(s, i);
    };
    uint32_t *const longs = T.h<uint32_t>(at_long), *const groups = T.h<uint32_t>(at_group);
    uint32_t n_longs = 0, n_groups = 0;
    r->long_begin.assign((size_t)r->n_slices * G, 0); r->long_count.assign((size_t)r->n_slices * G, 0);
    for (int g = 0; g < r->n_slices; ++g) {
        for (int w = 0; w < r->n_waves; ++w)
            for (int s : r->wave_scans[w]) {
                const ScanScript& sc = r->script[s];
                if (sc.Ah != 0) continue;                      // first passes only
                r->long_begin[(size_t)g * G + s] = n_longs;
                for (uint32_t pos = r->slice_img[g]; single && pos < r->slice_img[g + 1]; ++pos)
                    if (is_long(s, order[pos])) longs[n_longs++] = (uint32_t)(s * N + order[pos]);
                r->long_count[(size_t)g * G + s] = n_longs - r->long_begin[(size_t)g * G + s];
            }
    }
    // one list for the whole record: luminance first (its chains are the longest), within a
    // component the images with the most refinement bytes first
    for (int c = 0; single && c < 3; ++c) {
        std::vector<std::pair<uint64_t, uint32_t>> byw;
        for (uint32_t i = 0; i < N; ++i) {
            if (!grouped[(size_t)i * 3 + c]) continue;
            uint64_t bytes = 0;
            for (uint32_t s = 0; s < G; ++s) {
                const ScanScript& sc = r->script[s];
                if (sc.Ss > 0 && sc.Ah != 0 && sc.comp[0] == c) bytes += scans[(size_t)s * N + i].data_end - scans[(size_t)s * N + i].data_off;
            }
            byw.push_back({bytes, i});
        }
        std::stable_sort(byw.begin(), byw.end(), [](const std::pair<uint64_t, uint32_t>& a, const std::pair<uint64_t, uint32_t>& b) { return a.first > b.first; });
        for (auto& e : byw) groups[n_groups++] = ((uint32_t)c << 28) | e.second;
    }
    r->n_groups = n_groups;
    for (int g = 0; g < r->n_slices; ++g)
        for (int w = 0; w < r->n_waves; ++w)
            for (int s : r->wave_scans[w]) {
                const uint32_t begin = n_items;
                const Counts* const of = &counts[(size_t)s * N];
                const bool ac = r->script[s].Ss > 0;
                const bool dc_refine = r->script[s].Ss == 0 && r->script[s].Ah != 0, chains = ac ? r->script[s].Ah != 0 : r->script[s].Se == 63;
                Item* open = nullptr;                         // an unfilled last item that the next image may extend
                uint32_t last = 0;                            // the longest chain of the last item
                uint64_t load = 0;
                double squares = 0;
                for (uint32_t pos = r->slice_img[g]; pos < r->slice_img[g + 1] && !dc_refine; ++pos) {
                    const uint32_t i = order[pos];
                    if (single && takes_long_kernel((int)s, i)) continue;
                    const uint32_t nseg = of[i].nseg, si = (uint32_t)(s * N + i), chain = chains ? of[i].chain() : 0u;
                    // full warps of 32 restart intervals; in AC scans the last warp of an image
                    // runs on into the first intervals of the next image (two tables per warp)
                    uint32_t j = 0;
                    if (open) {                               // continued from the previous image
                        j = std::min<uint32_t>(kSegsPerItem - open->count, nseg);
                        open->count += j; open->next = si + 1u;
                        open = nullptr;
                        if (chain > last) { load += chain - last; squares += (double)chain * chain - (double)last * last; }
                    }
                    for (; j < nseg; j += kSegsPerItem) {
                        const uint32_t cnt = std::min<uint32_t>(kSegsPerItem, nseg - j);
                        items[n_items] = Item{si, j, cnt, 0u, 0u};
                        open = ac && cnt < (uint32_t)kSegsPerItem ? &items[n_items] : nullptr;
                        ++n_items;
                        load += last = chain;
                        squares += (double)chain * chain;
                    }
                }
                r->chain_bytes[s] += load;
                r->chain_squares[s] += squares;
                r->item_begin[(size_t)g * G + s] = begin;
                r->item_count[(size_t)g * G + s] = n_items - begin;
            }
    r->first_bytes.assign(G, 0); r->longest.assign(G, 0); r->longest_chain.assign(G, 0); r->long_bytes.assign(G, 0); r->intervals.assign(G, 0);
    for (uint32_t s = 0; s < G; ++s) {
        const Counts* const of = &counts[(size_t)s * N];
        const bool first = r->script[s].Ah == 0, ac = r->script[s].Ss > 0;
        uint32_t most = 0;
        uint64_t sum = 0, long_sum = 0;
        for (uint32_t i = 0; i < N; ++i) { most = std::max(most, of[i].bytes); sum += of[i].bytes; }
        for (uint32_t i = 0; single && first && i < N; ++i) long_sum += takes_long_kernel((int)s, i) ? of[i].bytes : 0u;
        r->longest[s] = most;
        if (first) r->long_bytes[s] = long_sum;
        if (first && ac) r->first_bytes[s] = sum - long_sum;
        for (uint32_t i = 0; first && !ac && r->script[s].Se == 63 && i < N; ++i) {      // (sequential)
            r->longest_chain[s] = std::max(r->longest_chain[s], of[i].chain());
            r->intervals[s] += of[i].nseg;
        }
    }
    // the pairs' items: sixteen intervals of one image
    r->pair_chain_bytes.assign(G, 0); r->pair_chain_squares.assign(G, 0); r->pair_begin.assign((size_t)r->n_slices * G, 0); r->pair_count.assign((size_t)r->n_slices * G, 0);
    for (int g = 0; g < r->n_slices; ++g)
        for (uint32_t s = 0; s < G; ++s) {
            const uint32_t begin = n_items;
            uint64_t load = 0;
            for (uint32_t pos = r->slice_img[g]; r->pair_of[s] >= 0 && pos < r->slice_img[g + 1]; ++pos) {
                const uint32_t i = order[pos], a = (uint32_t)r->pair_of[s];
                if (single && takes_long_kernel((int)s, i)) continue;
                const uint32_t nseg = counts[(size_t)s * N + i].nseg, longer = std::max(counts[(size_t)s * N + i].chain(), counts[(size_t)a * N + i].chain());
                for (uint32_t j = 0; j < nseg; j += kSegsPerItem / 2) {
                    items[n_items++] = Item{a * N + i, j, std::min<uint32_t>(kSegsPerItem / 2, nseg - j), 0u, (s - a) * N};
                    load += longer;
                    r->pair_chain_squares[s] += (double)longer * longer;
                }
            }
            r->pair_chain_bytes[s] += load;
            r->pair_begin[(size_t)g * G + s] = begin;
            r->pair_count[(size_t)g * G + s] = n_items - begin;
        }
    if (on_device && cudaDeviceGetAttribute(&r->n_sms, cudaDevAttrMultiProcessorCount, r->device) != cudaSuccess) return PCR_E_CUDA;
    // pixel work units (see Sampling in pcr_pixels.cuh), image by image in processing order, inside an image
    // MCU row by MCU row.  The host only counts them; a small kernel writes the list at set-up.
    uint32_t* const unit_prefix = T.h<uint32_t>(at_prefix);
    unit_prefix[0] = 0;
    for (uint32_t pos = 0; pos < N; ++pos) {
        const ImgDesc& im = imgs[order[pos]];
        if (im.my > 65535 || im.mx > 65535) return PCR_E_FORMAT;
        const uint64_t nu = (uint64_t)((im.mx + r->unit_mcus - 1) / r->unit_mcus) * ((im.my + r->unit_rows - 1) / r->unit_rows);
        if (unit_prefix[pos] + nu >= (1ull << 32)) return PCR_E_FORMAT;
        unit_prefix[pos + 1] = unit_prefix[pos] + (uint32_t)nu;
    }
    r->slice_unit.assign(r->n_slices + 1, 0);
    for (int g = 0; g <= r->n_slices; ++g) r->slice_unit[g] = unit_prefix[r->slice_img[g]];
    r->n_units = unit_prefix[N];

    if (!on_device) return PCR_E_CUDA;
    // the rest of the device state
    std::copy(r->script.begin(), r->script.end(), T.h<ScanScript>(at_script));
    std::copy(r->saux.begin(), r->saux.end(), T.h<ScanAux>(at_saux));
    if (int rc = take(r, &r->d_rec, (size_t)(len + 64))) return rc;
    if (int rc = take(r, &r->d_tabs, (size_t)(std::max<uint64_t>(n_tabs, 1) * sizeof(ScanTab)))) return rc;
    if (int rc = take(r, &r->d_vals, (size_t)(8 * (len + 256)))) return rc;      // four values per byte, two bytes each
    if (int rc = take(r, &r->d_units, (size_t)std::max<uint32_t>(r->n_units, 1) * sizeof(Unit))) return rc;
    r->d_script = T.d<ScanScript>(at_script); r->d_saux = T.d<ScanAux>(at_saux); r->d_scans = T.d<ScanDesc>(at_scans); r->d_imgs = T.d<ImgDesc>(at_imgs);
    r->d_qtab = T.d<uint16_t>(at_qtab); r->d_unit_prefix = T.d<uint32_t>(at_prefix); r->d_order = T.d<uint32_t>(at_order);
    r->d_group = T.d<uint32_t>(at_group); r->d_long = T.d<uint32_t>(at_long); r->d_items = TI.d<Item>(0);
    if (int rc = T.copy(r, at_long + 4ull * n_longs)) return rc;
    if (int rc = TI.copy(r, sizeof(Item) * (size_t)n_items)) return rc;
    units_kernel<<<N, 128, 0, r->up_stream>>>(r->d_imgs, r->d_order, r->d_unit_prefix, r->d_units, r->unit_mcus, r->unit_rows,
                                              r->d_scans, T.d<uint32_t>(at_base), G, bpm);
    ++g_launches;
    if (n_groups && cudaFuncSetAttribute(ac_refine_group_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)(kChainPairs * sizeof(ChainShared))) != cudaSuccess) return PCR_E_CUDA;
    r->h_status.assign(N, 0);
    r->resident = 0;
    if (!(r->ev_done = pool_event_get(r->device))) return PCR_E_CUDA;
    // the set-up above runs on the record's own stream; every decode waits for this event first
    if (!(r->ev_ready = pool_event_get(r->device))) return PCR_E_CUDA;
    if (cudaEventRecord(r->ev_ready, r->up_stream) != cudaSuccess) return PCR_E_CUDA;
    if (r->n_slices > 1) {
        if (!(r->ev_fork = pool_event_get(r->device))) return PCR_E_CUDA;
        if (!(r->copy_stream = pool_stream_get(r->device))) return PCR_E_CUDA;
        if (!(r->side_stream = pool_stream_get(r->device))) return PCR_E_CUDA;
        if (!(r->ev_side = pool_event_get(r->device))) return PCR_E_CUDA;
        if (!(r->ev_start = pool_event_get(r->device))) return PCR_E_CUDA;
        if (!(r->ev_chain = pool_event_get(r->device))) return PCR_E_CUDA;
        for (int w = 0; w < r->n_waves; ++w) {
            cudaEvent_t e;
            if (!(e = pool_event_get(r->device))) return PCR_E_CUDA;
            r->ev_copy.push_back(e);
            if (!(e = pool_event_get(r->device))) return PCR_E_CUDA;
            r->ev_index.push_back(e);
        }
        for (int g = 0; g < r->n_slices; ++g) {
            cudaStream_t q; cudaEvent_t e;
            if (!(q = pool_stream_get(r->device))) return PCR_E_CUDA;
            r->streams.push_back(q);
            if (!(e = pool_event_get(r->device))) return PCR_E_CUDA;
            r->ev_join.push_back(e);
        }
    }
    return PCR_OK;
}

}  // namespace

// ---------------------------------------------------------------------------------------
// Cache of closed records.  A loader reads the same records epoch after epoch; with the cache
// on, pcr_close parks the whole record (parse results, device tables and buffers) and a later
// pcr_open of the same bytes takes it back instead of walking every image's marker segments and
// uploading the tables again.  A record is recognised by its address, its length, the tuning
// variables in force and a hash of its header, sample metadata, index (position and length of every
// chunk) and the head of every image's first chunk (frame header and tables).
// ---------------------------------------------------------------------------------------
namespace {
struct RecordCache {
    std::mutex mu;
    std::vector<pcr_record*> lru;     // most recently closed last
    size_t bytes = 0, limit = 0;
} g_rcache;

inline uint64_t mix64(uint64_t h, uint64_t v) {
    h ^= v + 0x9E3779B97F4A7C15ull + (h << 6) + (h >> 2);
    h *= 0xFF51AFD7ED558CCDull;
    return h ^ (h >> 29);
}
uint64_t hash_bytes(uint64_t h, const uint8_t* p, size_t n) {
    size_t i = 0;
    for (; i + 8 <= n; i += 8) { uint64_t v; memcpy(&v, p + i, 8); h = mix64(h, v); }
    uint64_t tail = 0;
    if (i < n) { memcpy(&tail, p + i, n - i); h = mix64(h, tail ^ ((uint64_t)(n - i) << 56)); }
    return h;
}
uint32_t env_key() {
    uint32_t h = 0;
    for (const char* name : {"PCR_SLICES", "PCR_LONG_MIN_BYTES", "PCR_PAIRS", "PCR_REFINE_CTAS", "PCR_PACK_WARPS", "PCR_SHORT_WARPS", "PCR_SEQ_CTAS", "PCR_INDEX_CTAS", "PCR_LONG_CTAS"}) {
        const char* v = getenv(name);
        for (h = h * 1000003u + (v ? 1u : 0u); v && *v; ++v) h = h * 1000003u + (uint8_t)*v;
    }
    return h;
}
// 0 when the bytes do not even look like a record (pcr_open then reports the error)
uint64_t record_identity(const uint8_t* rec, size_t len) {
    if (len < 64 || len >= (1ull << 32) || memcmp(rec, "PCR1", 4) != 0) return 0;
    const uint32_t N = rd32(rec + 8), G = rd32(rec + 12);
    const uint64_t index_off = rd64(rec + 32), data_off = rd64(rec + 40);
    if (N == 0 || G == 0 || G > 64 || N > (1u << 24) || data_off > len) return 0;
    if (index_off < 64 || index_off > data_off || 8ull * (G + 1) + 16ull * G * N > data_off - index_off) return 0;
    uint64_t h = hash_bytes(len, rec, (size_t)data_off);        // header, sample metadata, index
    const uint8_t* chunk = rec + index_off + 8ull * (G + 1);
    for (uint64_t j = 0; j < (uint64_t)N; ++j) {              // the chunks of scan group 1: frame header and tables of every image
        const uint64_t off = rd64(chunk + 16 * j);
        const uint32_t clen = rd32(chunk + 16 * j + 8);
        if (off > len || clen > len - off) return 0;
        h = hash_bytes(h, rec + off, std::min<size_t>(clen, 256));
    }
    return h ? h : 1;
}
void evict_records_locked(std::vector<pcr_record*>* out) {
    while (g_rcache.bytes > g_rcache.limit && !g_rcache.lru.empty()) {
        pcr_record* r = g_rcache.lru.front();
        g_rcache.lru.erase(g_rcache.lru.begin());
        g_rcache.bytes -= r->device_bytes;
        out->push_back(r);
    }
}
}  // namespace

extern "C" {

int pcr_set_record_cache(size_t max_device_bytes) {
    std::vector<pcr_record*> gone;
    {
        std::lock_guard<std::mutex> lk(g_rcache.mu);
        g_rcache.limit = max_device_bytes;
        evict_records_locked(&gone);
    }
    for (pcr_record* r : gone) { free_device(r); delete r; }
    return PCR_OK;
}

// Bound by the host's cache misses on the chunk heads (each chunk's head is a line of its own in the record), then by the
// start of the copies.  1024 ImageNet-shaped images, ten scans: 740 -> 350 us with the next image's heads prefetched, the
// tables built in reused page-locked blocks that go over in one copy each, and the zeroing beside the walk.
int pcr_open(const void* bytes, size_t len, pcr_record** rec) {
    if (rec) *rec = nullptr;
    if (!bytes || !rec) return PCR_E_ARG;
    uint64_t key = 0;
    const uint32_t ekey = env_key();
    if (g_rcache.limit) {
        key = record_identity(static_cast<const uint8_t*>(bytes), len);
        int dev = -1;
        cudaGetDevice(&dev);
        std::lock_guard<std::mutex> lk(g_rcache.mu);
        for (size_t i = g_rcache.lru.size(); key && i-- > 0;) {
            pcr_record* c = g_rcache.lru[i];
            if (c->host != bytes || c->key_len != len || c->key_hash != key || c->key_env != ekey || c->device != dev) continue;
            g_rcache.lru.erase(g_rcache.lru.begin() + (long)i);
            g_rcache.bytes -= c->device_bytes;
            // a fresh handle: nothing resident, nothing decoded, default settings
            c->resident = 0; c->decoded_k = 0; c->lists_k = 0; c->planes_current = false; c->upsampling = PCR_UPSAMPLE_REPLICATE; c->profiling = false;
            c->decode_enqueued = false;
            *rec = c;
            return PCR_OK;
        }
    }
    pcr_record* r = new (std::nothrow) pcr_record();
    if (!r) return PCR_E_NOMEM;
    int rc;
    try {
        rc = open_impl(static_cast<const uint8_t*>(bytes), len, r);
    } catch (const std::bad_alloc&) {
        rc = PCR_E_NOMEM;
    }
    if (rc != PCR_OK) {
        free_device(r);
        delete r;
        return rc;
    }
    r->key_hash = key; r->key_len = key ? len : 0; r->key_env = ekey;
    for (auto& b : r->bufs) r->device_bytes += size_class(b.second);
    *rec = r;
    return PCR_OK;
}

int pcr_num_images(const pcr_record* rec) { return rec ? rec->N : PCR_E_ARG; }
int pcr_num_groups(const pcr_record* rec) { return rec ? rec->G : PCR_E_ARG; }

int pcr_get_image(const pcr_record* rec, int i, pcr_image_info* info) {
    if (!rec || !info || i < 0 || i >= rec->N) return PCR_E_ARG;
    *info = rec->info[i];
    return PCR_OK;
}

int pcr_get_images(const pcr_record* rec, int first, int count, pcr_image_info* info) {
    if (!rec || !info || first < 0 || count < 0 || first > rec->N || count > rec->N - first) return PCR_E_ARG;
    memcpy(info, rec->info.data() + first, (size_t)count * sizeof *info);
    return PCR_OK;
}

size_t pcr_out_bytes(const pcr_record* rec) { return rec ? rec->out_bytes : 0; }

size_t pcr_prefix_bytes(const pcr_record* rec, int k) {
    if (!rec || k < 1 || k > rec->G) return 0;
    return (size_t)rec->group_end[k];
}

int pcr_evict(pcr_record* rec) {
    if (!rec) return PCR_E_ARG;
    rec->resident = 0;
    return PCR_OK;
}

}  // extern "C"

// The pixel kernels of one slice at one fidelity (see pcr_pixels.cuh for what the template arguments choose).
struct PixelPlan { bool dc_only, head_only, refine, coarse, widths_mult16, triangle, roi; int samp; };

template <int kSamp>
static void launch_pixels_sampled(const PixelPlan& pl, unsigned grid, cudaStream_t q, const Params& Q, const CoefLists& cl, uint8_t* o8) {
    constexpr int T = unit_threads<kSamp>();
    if (pl.refine) pixel_kernel<true, 1, false, 0, kSamp><<<grid, T, 0, q>>>(Q, cl, o8);
    else if (pl.coarse) pixel_kernel<false, 1, false, 0, kSamp, true><<<grid, T, 0, q>>>(Q, cl, o8);
    else pixel_kernel<false, 1, false, 0, kSamp><<<grid, T, 0, q>>>(Q, cl, o8);
}

template <bool kRoi>
static void launch_pixels_420(const PixelPlan& pl, unsigned grid, cudaStream_t q, const Params& Q, const CoefLists& cl, uint8_t* o8) {
    constexpr int T = unit_threads<kSamp420>();
    if (pl.dc_only && pl.widths_mult16) dc_pixel_kernel<kRoi><<<grid, 128, 0, q>>>(Q, make_uint3(cl.dc_mask[0], cl.dc_mask[1], cl.dc_mask[2]), o8);
    else if (pl.dc_only) dc_pixel_kernel<kRoi, false><<<grid, 128, 0, q>>>(Q, make_uint3(cl.dc_mask[0], cl.dc_mask[1], cl.dc_mask[2]), o8);
    else if (pl.head_only) pixel_kernel<false, 3, kRoi, 0, kSamp420, true><<<grid, T, 0, q>>>(Q, cl, o8);
    else if (pl.refine) pixel_kernel<true, 1, kRoi><<<grid, T, 0, q>>>(Q, cl, o8);
    else if (pl.coarse) pixel_kernel<false, 1, kRoi, 0, kSamp420, true><<<grid, T, 0, q>>>(Q, cl, o8);
    else pixel_kernel<false, 1, kRoi><<<grid, T, 0, q>>>(Q, cl, o8);
}

static void launch_pixels(const PixelPlan& pl, unsigned grid, cudaStream_t q, const Params& Q, const CoefLists& cl, uint8_t* o8) {
    constexpr int T = unit_threads<kSamp420>();
    if (pl.samp == kSamp422) launch_pixels_sampled<kSamp422>(pl, grid, q, Q, cl, o8);
    else if (pl.samp == kSamp440) launch_pixels_sampled<kSamp440>(pl, grid, q, Q, cl, o8);
    else if (pl.samp == kSamp444) launch_pixels_sampled<kSamp444>(pl, grid, q, Q, cl, o8);
    else if (pl.samp == kSampGrey) launch_pixels_sampled<kSampGrey>(pl, grid, q, Q, cl, o8);
    else if (pl.roi) launch_pixels_420<true>(pl, grid, q, Q, cl, o8);
    else if (pl.triangle) {
        // chroma pass (samples of every chroma block into the sample planes), then the pixel pass
        pixel_kernel<true, 1, false, 1><<<grid, T, 0, q>>>(Q, cl, o8);
        pixel_kernel<true, 1, false, 2><<<grid, T, 0, q>>>(Q, cl, o8);
        ++g_launches;
    } else launch_pixels_420<false>(pl, grid, q, Q, cl, o8);
    ++g_launches;
}

template <typename OutT>
static void launch_tensor(dim3 grid, cudaStream_t q, const Params& P, const TensorArgs& T, const uint8_t* rgb, uint32_t pos0) {
    // pairs of columns where a pair never straddles rows and its store is aligned
    const bool pairs = T.size % 2 == 0 && (reinterpret_cast<uintptr_t>(T.out) & (2 * sizeof(OutT) - 1)) == 0;
    if (pairs) tensor_kernel<OutT, 2><<<grid, 128, 0, q>>>(P, T, rgb, pos0);
    else tensor_kernel<OutT, 1><<<grid, 256, 0, q>>>(P, T, rgb, pos0);
}

// The expanded blocks of the whole record into the canonical planes.
static void launch_planes(int samp, unsigned grid, const Params& Q, const CoefLists& cl) {
    if (samp == kSamp422) pixel_kernel<true, 1, false, 3, kSamp422><<<grid, unit_threads<kSamp422>()>>>(Q, cl, nullptr);
    else if (samp == kSamp440) pixel_kernel<true, 1, false, 3, kSamp440><<<grid, unit_threads<kSamp440>()>>>(Q, cl, nullptr);
    else if (samp == kSamp444) pixel_kernel<true, 1, false, 3, kSamp444><<<grid, unit_threads<kSamp444>()>>>(Q, cl, nullptr);
    else if (samp == kSampGrey) pixel_kernel<true, 1, false, 3, kSampGrey><<<grid, unit_threads<kSampGrey>()>>>(Q, cl, nullptr);
    else pixel_kernel<true, 1, false, 3, kSamp420><<<grid, unit_threads<kSamp420>()>>>(Q, cl, nullptr);
    ++g_launches;
}

static Params record_params(const pcr_record* rec) {
    Params P;
    memset(&P, 0, sizeof P);
    P.rec = rec->d_rec; P.ubuf = rec->d_ubuf; P.planes = rec->d_planes; P.dc = rec->d_dc; P.head = rec->d_head; P.vals = rec->d_vals;
    P.script = rec->d_script; P.scans = rec->d_scans;
    P.saux = rec->d_saux; P.aux = rec->d_aux;
    P.imgs = rec->d_imgs; P.seg_start = rec->d_seg; P.items = rec->d_items; P.units = rec->d_units;
    P.tabs = rec->d_tabs;
    P.qtab = rec->d_qtab; P.order = rec->d_order; P.status = rec->d_status; P.N = rec->N;
    P.hs = rec->hs; P.vs = rec->vs; P.nc = rec->nc;
    P.chroma = rec->d_chroma;
    return P;
}

// Where the coefficients of scans 0 .. k-1 lie.
static void coef_lists(const pcr_record* rec, int k, CoefLists* cl) {
    memset(cl, 0, sizeof *cl);
    uint16_t mask[3][8] = {};
    for (int s = 0; s < k; ++s) {
        const ScanScript& sc = rec->script[s];
        const ScanAux& ax = rec->saux[s];
        if (sc.Ss == 0)                                            // the DC plane
            for (int q = 0; q < sc.ncomp; ++q) cl->dc_mask[sc.comp[q]] = 0xFFFFu & ~((1u << sc.Al) - 1u);
        if (sc.Ss == 0 && sc.Se != 63) continue;
        for (int i = 0; i < sc.ncomp; ++i) {
            const int c = sc.comp[i];
            for (int p = std::max(1, sc.Ss); p <= std::min(7, sc.Se); ++p) mask[c][p] = 0xFFFFu;
            if (sc.Ah) {
                cl->p1[c][cl->n_refine[c]] = 1 << sc.Al;
                cl->refine[c][cl->n_refine[c]++] = ax.base;
            } else if (sc.Se >= 8) {
                cl->first[c][cl->n_first[c]++] = ax.base;
                cl->sequential = sc.Ss == 0;
            }
        }
    }
    for (int c = 0; c < 3; ++c) memcpy(&cl->head_mask[c], mask[c], 16);
}

// refine_kernel's shared memory is beyond what a launch may take unasked; asked for once per device and kernel (asking loads the kernel,
// which records without refinements have no use for).
template <bool kRoi>
static bool allow_refine_smem(int device) {
    static std::atomic<uint64_t> asked{0};
    const uint64_t bit = 1ull << (device & 63);
    if (device < 64 && (asked.load(std::memory_order_acquire) & bit)) return true;
    if (cudaFuncSetAttribute(refine_kernel<kRoi>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kRefineBytes) != cudaSuccess) return false;
    if (device < 64) asked.fetch_or(bit, std::memory_order_release);
    return true;
}

// The AC refinements among scans k0 .. k-1 of a wave in items an SM, an item counting by its longest chain beside the chain that a byte of the
// scan lies in on average (of the scan where that is longest; a chroma scan's are a third of luminance's).  Not the average item's chain: a
// launch waits for the long ones, and with that unit records of mixed sizes changed sides at 1.4 times the number of others.
static double refine_load(const pcr_record* rec, const std::vector<int>& wave, bool paired, int k0, int k, double* chain = nullptr) {
    double sum = 0, longest = 0;
    std::vector<char> counted(rec->G, 0);                     // scans that a pair's items stand for
    for (int s : wave)
        if (paired && s < k && rec->pair_of[s] >= k0) counted[rec->pair_of[s]] = 1;
    for (int s : wave) {
        if (s < k0 || s >= k || rec->script[s].Ss == 0 || rec->script[s].Ah == 0 || counted[s]) continue;
        const bool pair = paired && rec->pair_of[s] >= k0;
        uint64_t items = 0;
        for (int g = 0; g < rec->n_slices; ++g) items += (pair ? rec->pair_count : rec->item_count)[(size_t)g * rec->G + s];
        const double bytes = (double)std::max<uint64_t>(items, (pair ? rec->pair_chain_bytes : rec->chain_bytes)[s]);
        sum += bytes;
        if (items) longest = std::max(longest, std::max(bytes, (pair ? rec->pair_chain_squares : rec->chain_squares)[s]) / bytes);
    }
    if (chain) *chain = longest;
    return sum > 0 ? sum / longest / rec->n_sms : 0;
}

// refine_kernel's CTAs take a wave's refinements up to rec->refine_ctas by refine_load, lane-per-interval warps of entropy_kernel beyond.  A CTA's
// chains are several times as fast (170 to 220 cycles a symbol), but three CTAs are all an SM holds, 96 chains against 480.
// Decode in us, CTAs and warps, by refine_load, means over two or three contents.  k = 9, one wave: ImageNet-shaped images 3.0 242
// and 248, 3.3 229 and 237, 3.8 262 and 259, 4.0 283 and 277; in 4:4:4 2.5 216 and 228, 3.0 255 and 236, 3.4 282 and 261; in 4:2:2 2.4 213 and 220,
// 2.8 238 and 240, 3.4 276 and 265; CelebA-shaped 3.2 172 and 176, 3.4 183 and 182, 3.7 191 and 186, 4.2 223 and 214; HAM-shaped 2.5 242 and 243,
// 3.0 280 and 267, 3.5 316 and 296; mixed sizes 2.7 228 and 246, 3.1 240 and 259, 3.7 247 and 247, 4.2 261 and 257; 128x128 2.3 107 and 110, 2.9 118
// and 119.  k = 6, luminance alone: ImageNet-shaped 3.0 257 and 264, 3.7 292 and 281, 4.2 322 and 303; CelebA-shaped 3.0 198 and 201, 3.8 221
// and 219, 4.5 249 and 243.  Short chains gain from fewer steps outside the loop: 32x32 at k = 9 3.7 106 and 110, 4.4 109 and 113, 5.0 114 and 117,
// 6.3 111 and 99, at k = 6 2.7 87 and 96; 64x64 2.9 107 and 106, 3.5 118 and 120.
//
// Behind another wave of refinements the line lies further out: the slices of the record get there one after the other.  Decode at k = 10
// with the later wave (luminance alone) in CTAs and in warps: ImageNet-shaped 5.0 552 and 556, 5.5 586 and 588, 5.9 601 and 600, 6.8 675 and 664,
// 7.4 721 and 705; CelebA-shaped 4.5 359 and 359, 5.3 405 and 397, 6.0 442 and 429, 6.8 498 and 475; HAM-shaped 3.9 534 and 531, 4.6 602 and 585, 5.4
// 677 and 644; greyscale 4.9 486 and 508, 5.4 508 and 530, 5.9 518 and 543; mixed sizes 3.4 438 and 503, 4.0 502 and 550.
//
// With pairs the line is where pairs cease to pay (see pairs_pay).
static bool refine_in_ctas(const pcr_record* rec, const std::vector<int>& wave, bool paired, bool later, int k0, int k) {
    double chain = 0, first = 0;                              // `first`: of the wave that would hold the pairs' earlier scans
    const double load = refine_load(rec, wave, paired, k0, k, &chain);
    bool pairs = false;
    for (int s : wave) {
        if (!paired || s >= k || rec->pair_of[s] < k0) continue;
        pairs = true;
        for (const std::vector<int>& w : rec->wave_scans)
            if (std::find(w.begin(), w.end(), rec->pair_of[s]) != w.end()) first = std::max(first, refine_load(rec, w, false, k0, k));
    }
    double line = chain < 48.0 ? 1.32 : (pairs ? 0.91 + 0.22 * std::min(std::max(first - 1.85, 0.0), 1.45) : 1.0);
    if (later && !pairs) line = 1.8;
    return load <= rec->refine_ctas * line;
}

// Whether refinements that follow one another are decoded in pairs (see refine_kernel).  Pairs shorten the chain but leave the lanes
// of the shorter scan idle.  They pay in CTAs, while an SM's three hold them all at once; beyond, two waves take no longer than
// the pairs' second round.  Decode at k = 10 in us by refine_load with pairs, pairs in CTAs and no pairs, means over two or three contents:
// ImageNet-shaped images 2.2 232 and 255, 3.0 283 and 306, 3.3 314 and 306, 3.8 338 and 319; CelebA-shaped 2.8 185 and 193, 3.3 219 and 203, 3.8 225
// and 203; HAM-shaped 2.7 252 and 285, 3.2 318 and 298, 3.6 356 and 321; greyscale 3.2 279 and 273, 3.6 298 and 270, 4.3 328 and 289; mixed sizes 2.7
// 261 and 318, 3.4 300 and 314, 4.3 347 and 376; 128x128 1.6 112 and 117, 2.4 133 and 132, 2.8 140 and 136.
// Chroma scans beside the earlier scan fill the first wave without pairs too (`first`), which then takes a second round itself: 4:2:2
// ImageNet-shaped (first 1.9) 3.0 292 and 322, (2.1) 3.2 308 and 331, (2.4) 3.5 344 and 341, CelebA-shaped (2.1) 3.2 205 and 215, (2.4) 3.7 249 and
// 231; 4:4:4 ImageNet-shaped (3.0) 3.3 314 and 353, (3.1) 3.5 351 and 387, (3.7) 4.1 390 and 416, (4.2) 4.7 432 and 406, CelebA-shaped (3.2) 3.6 223
// and 238, (3.7) 4.2 257 and 262, HAM-shaped (3.2) 3.2 344 and 380, (3.7) 3.7 392 and 417, (4.3) 4.2 455 and 414, mixed sizes (3.5) 3.3 342 and 385.
// Where chains are short, a wave less counts for more: 32x32 2.6 82 and 99, 3.7 109 and 121, 4.4 115 and 123, 5.2 121 and 140, 8.8 149 and 149;
// 64x64 2.9 102 and 106, 3.5 115 and 128, 4.2 123 and 132, 5.9 148 and 141.
// Pairs in warps and no pairs: ImageNet-shaped 10 526 and 484, 13 601 and 581, 18 747 and 697; CelebA-shaped 10 343 and 348, 13 399 and 402, 17 490
// and 474; HAM-shaped 9 496 and 529, 11 565 and 586, 14 725 and 719, 18 877 and 847; greyscale 14 570 and 523, 17 670 and 602; mixed sizes 10 589 and 549:
// never chosen, since what gains (HAM-shaped) gains less than the others lose.
static bool pairs_pay(const pcr_record* rec, int k0, int k) {
    for (const std::vector<int>& wave : rec->paired_waves)
        for (int s : wave)
            if (s < k && rec->pair_of[s] >= k0 && !refine_in_ctas(rec, wave, true, false, k0, k)) return false;
    return true;
}

// Form of entropy_kernel for the first passes among scans k0 .. k-1 of a wave: kFirstFull where there is so much to store that stores are
// what the machine waits for, which is a matter of how much data an SM has, not of how many warps it comes in; elsewhere a step
// without the packing is the shorter chain.  Decode in us without and with packing, by entropy-coded kilobytes of AC scans an SM: k = 5
// ImageNet-shaped images 5 102 and 134, 9 120 and 141, 13 157 and 165, 16 194 and 185, 18 213 and 209, 27 294 and 270, 34 357 and
// 335; CelebA-shaped 9 120 and 126, 12 145 and 142, 18 185 and 180, 23 251 and 225; HAM-shaped 6 191 and 199, 9 266 and 270, 12 346 and
// 324; 1024 of 96x96 5 85 and 93, 4096 of 32x32 4 167 and 188 (these two fill the machine with warps, 15 and 83 an SM).
// kFirstShort for many warps of little data (see entropy_kernel).
static int first_pass_form(const pcr_record* rec, const std::vector<int>& wave, int k0, int k) {
    uint64_t warps = 0, bytes = 0;
    for (int s : wave)
        if (s >= k0 && s < k && rec->script[s].Ah == 0) {
            for (int g = 0; g < rec->n_slices; ++g) warps += rec->item_count[(size_t)g * rec->G + s];
            bytes += rec->first_bytes[s];
        }
    const uint64_t sms = (uint64_t)rec->n_sms;
    if (rec->pack_warps >= 0 ? warps > (uint64_t)rec->pack_warps * sms : bytes > 11000ull * sms) return kFirstFull;
    return warps > (uint64_t)rec->short_warps * sms ? kFirstShort : kFirstFew;
}

// Whether sequential_kernel's CTAs take the sequential scan's items or sequential_lane_kernel's warps.  A CTA's chains are five times as fast,
// but an SM holds four CTAs and eighteen warps, and a CTA costs the same whether its lanes are in use or not: the warps are better where
// images have few intervals and there are many images, by the items an SM in units of the longest chain.  Decode in us, CTAs and warps, two
// contents each: CelebA-shaped images (14 lanes in use) 5.1 411 and 481, 7.0 556 and 576, 7.7 597 and 595, 8.9 680 and 642, 10.2 766 and 694, 15 1118
// and 980; 64x64 (4) 7.9 169 and 173, 10.1 200 and 193; 96x96 (6) 4.9 157 and 203, 7.4 217 and 230; mixed sizes (13) 1.7 305 and 750, 2.2 439 and
// 870; HAM-shaped (29) 5.4 958 and 1048; ImageNet-shaped (23) 8.9 1268 and 1406.
static bool sequential_in_ctas(const pcr_record* rec, int s) {
    uint64_t items = 0;
    for (int g = 0; g < rec->n_slices; ++g) items += rec->item_count[(size_t)g * rec->G + s];
    if (rec->seq_ctas >= 0) return items <= (uint64_t)rec->seq_ctas * (uint64_t)rec->n_sms;
    return rec->intervals[s] >= 20 * items || (double)rec->chain_bytes[s] <= 8.0 * rec->n_sms * rec->longest_chain[s];
}

// Whether the long scans of a wave that are first passes (or sequential) get CTAs of four times as many warps: while most of the
// machine is idle, by the number of CTAs an SM or by what there is to read in units of the longest scan (an SM holds few wide CTAs, but those of
// chroma scans are soon gone); beyond, the narrow ones do less in all.  Decode in us, narrow and wide, means over two or three contents.
// k = 5, by longest scans an SM: ImageNet-shaped 0.3 232 and 155, 0.9 221 and 201, 1.4 253 and 236, 1.8 291 and 264, 2.5 330 and 381; CelebA-shaped
// 1.0 163 and 112, 1.5 173 and 145, 2.3 196 and 182, 2.9 202 and 205; HAM-shaped 0.4 283 and 255, 1.6 366 and 345, 3 437 and 435; greyscale 1.2
// 214 and 170, 2.4 212 and 238; mixed sizes 0.4 396 and 196.  k = 1, by CTAs an SM: ImageNet-shaped 0.4 178 and 105, 1.3 160 and 122, 2.6 171 and
// 143, 4.3 181 and 176, 6.9 225 and 246; HAM-shaped 1.7 215 and 194, 3.0 255 and 263; 128x128 2.6 95 and 77.  Scans below a kilobyte gain only
// side by side with few others: 128x128 k = 5 4.3 CTAs an SM 106 and 108, 6.5 110 and 120; 64x64 8.6 100 and 120.
// Baseline, by CTAs an SM: ImageNet-shaped 0.4 654 and 615, 0.9 638 and 595, 1.1 676 and 758; HAM-shaped 0.4 465 and 448, 1.1 593 and 615; mixed
// sizes 1.7 719 and 632; 1024x1024 0.4 2031 and 1126.  Scans that a narrow CTA's threads read in 32 words each gain nothing: CelebA-shaped
// 0.4 436 and 448, 1.3 562 and 577, 32x32 142 and 148.
static bool wide_long_scans(const pcr_record* rec, const std::vector<int>& wave, bool sequential, int k0, int k) {
    uint64_t ctas = 0, bytes = 0, longest = 0;
    for (int s : wave) {
        if (s < k0 || s >= k || rec->script[s].Ah != 0) continue;
        for (int g = 0; g < rec->n_slices; ++g) ctas += rec->long_count[(size_t)g * rec->G + s];
        bytes += rec->long_bytes[s];
        longest = std::max<uint64_t>(longest, rec->longest[s]);
    }
    const uint64_t sms = (uint64_t)rec->n_sms;
    if (rec->long_ctas >= 0) return ctas * (sequential ? 4u : 1u) <= (uint64_t)rec->long_ctas * sms;
    if (sequential) return longest > 128u * kSeqLongWarps * 32u && (4u * ctas <= 3u * sms || (double)bytes <= 0.55 * sms * longest);
    return ctas <= 3u * sms || (longest >= 1000u && (double)bytes <= 2.2 * sms * longest);
}

// Decode scans k0 .. k-1 on top of the state scans 0 .. k0-1 left behind (k0 = 0: from scratch),
// then produce the pixels of fidelity k.
static int decode_range(pcr_record* rec, int k0, int k, void* out, void* stream, const TensorArgs* targs = nullptr) {
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    const size_t need = (size_t)rec->group_end[k];
    const bool prof = rec->profiling;
    rec->profile.clear();
    auto mark = [&](const char* name, int launches) {
        if (!prof || rec->profile.size() + 1 >= rec->events.size()) return;
        pcr_stage_time t;
        memset(&t, 0, sizeof t);
        strncpy(t.name, name, sizeof t.name - 1);
        t.launches = launches;
        rec->profile.push_back(t);
        cudaEventRecord(rec->events[rec->profile.size()], st);
    };
    const bool pipelined = rec->n_slices > 1 && !prof;
    // (the copy of missing bytes, on a stream of its own, need not wait for pcr_open's uploads)
    if (pipelined && rec->resident < need && (cudaEventRecord(rec->ev_fork, st) != cudaSuccess ||
                                              cudaStreamWaitEvent(rec->copy_stream, rec->ev_fork, 0) != cudaSuccess)) return PCR_E_CUDA;
    if (cudaStreamWaitEvent(st, rec->ev_ready, 0) != cudaSuccess) return PCR_E_CUDA;      // pcr_open's uploads
    if (prof) cudaEventRecord(rec->events[0], st);
    if (!pipelined && rec->resident < need) {
        size_t from = rec->resident & ~(size_t)15;
        if (cudaMemcpyAsync(rec->d_rec + from, rec->host + from, need - from, cudaMemcpyHostToDevice, st) != cudaSuccess) return PCR_E_CUDA;
        rec->resident = need;
    }
    mark("h2d", 0);
    if (k0 == 0 && cudaMemsetAsync(rec->d_status, 0, (size_t)rec->N * 4, st) != cudaSuccess) return PCR_E_CUDA;
    Params P = record_params(rec);
    P.roi = targs ? targs->crops : nullptr;          // (only read by the crop-restricted kernels)
    RefineList fl;                                    // the AC refinements this call decodes
    memset(&fl, 0, sizeof fl);
    for (int s = k0; s < k; ++s) {
        const ScanScript& sc = rec->script[s];
        if (sc.Ss == 0 || sc.Ah == 0) continue;
        const int c = sc.comp[0];
        if (fl.n[c] < 4) fl.scan[c][fl.n[c]++] = s;
    }
    CoefLists cl;                                     // everything the pixel stage shows, earlier calls' scans included
    coef_lists(rec, k, &cl);
    // the waves of this call: with pairs of refinements when both scans of a pair are to be decoded
    bool paired = false;
    for (int s = 0; s < k; ++s) paired = paired || (rec->pair_of[s] >= k0);
    if (paired) paired = rec->pairs < 0 ? pairs_pay(rec, k0, k) : rec->pairs != 0;
    const std::vector<std::vector<int>>& waves = paired ? rec->paired_waves : rec->wave_scans;
    const bool chains = fl.n[0] + fl.n[1] + fl.n[2] > 0 && rec->n_groups > 0;
    const int chain_depth = kChainPairs / 4;    // chains per scheduler of the chain launch
    PixelPlan plan;
    plan.samp = sampling_code(rec->hs, rec->vs, rec->nc);
    const bool s420 = plan.samp == kSamp420;
    plan.dc_only = plan.head_only = s420;             // no AC scan at all / no scan beyond zigzag position 7, no refinement
    plan.refine = false;
    plan.coarse = true;                               // every AC scan leaves low bits out (first passes ahead of refinements)
    for (int s = 0; s < k; ++s) {
        const ScanScript& sc = rec->script[s];
        if (sc.Ss > 0 || sc.Se > 0) plan.dc_only = false;
        if (sc.Se > 7 || (sc.Ss > 0 && sc.Ah > 0)) plan.head_only = false;
        if (sc.Ss > 0 && sc.Ah > 0) plan.refine = true;
        if (sc.Se > 0 && sc.Al == 0) plan.coarse = false;
    }
    plan.widths_mult16 = rec->widths_mult16;
    plan.triangle = !targs && rec->upsampling == PCR_UPSAMPLE_TRIANGLE;
    const bool roi = targs && s420;                   // decode only the MCU rows the crops touch (built for 4:2:0)
    plan.roi = roi;
    rec->planes_current = false;
    rec->decoded_k = rec->lists_k = k;
    const int G = rec->G;
    std::vector<char> copied(rec->n_waves, 0);      // wave w has to wait for its copy event
    // the stages of one slice; stage numbers: 0 nothing (in the profile: the status words' memset), 1 index, 2+w entropy wave w,
    // 2+W chains, 3+W pixels
    const int W = (int)waves.size();
    std::vector<char> indexed(rec->n_waves, 0);     // wave w of the current slice has an index launch to wait for
    // index (and lookup tables, where the interval kernels will want them) of the listed scans, all images
    auto launch_index_kernel = [&](const ScanList& sl, cudaStream_t q) {
        const uint32_t pairs = (uint32_t)sl.n * (uint32_t)rec->N;
        bool tables = false;
        for (int i = 0; i < sl.n; ++i)
            for (int g = 0; g < rec->n_slices; ++g) tables = tables || rec->item_count[(size_t)g * rec->G + sl.s[i]] + rec->long_count[(size_t)g * rec->G + sl.s[i]] > 0;
        // A CTA a pair while an SM has few of them (it holds eight) and the longest scan of the launch is long enough for eight warps.  Decode in us
        // with a warp and with a CTA a pair, by pairs an SM and bytes of the longest scan: 64 ImageNet-shaped images at k = 10 4.3 5 k 227 and
        // 199, 256 (two waves side by side) 8.6 5 k 425 and 459, baseline 128 0.9 30 k 293 and 219, 1024 6.9 753 and 682, k = 1 768 5.2
        // 4 k equal, 1024 (no markers) 6.9 226 and 228; CelebA-shaped k = 1 512 3.5 1.2 k 62 and 64, 1024 6.9 87 and 92, k = 5 (no
        // markers) 128 4.3 2 k 180 and 182; 96 of mixed sizes (no markers) 3.2 8 k 180 and 162; 512 of 64x64 k = 1 3.5 0.3 k 36 and 39; 1024 of
        // 32x32 6.9 0.3 k 38 and 41.
        uint64_t bytes = 0;
        for (int i = 0; i < sl.n; ++i) bytes = std::max<uint64_t>(bytes, rec->longest[sl.s[i]]);
        const uint64_t sms = (uint64_t)rec->n_sms;
        const bool split = rec->index_ctas >= 0 ? pairs <= (uint64_t)rec->index_ctas * sms : pairs <= 8 * sms && pairs <= bytes * sms / 700;
        const uint32_t nb = split ? pairs : (pairs + kIndexWarps - 1) / kIndexWarps, nt = tables ? (4 * pairs + kIndexWarps - 1) / kIndexWarps : 0;
        if (split) unstuff_index_kernel<true><<<nb + nt, 32 * kIndexWarps, 0, q>>>(P, sl, 0, rec->N, nb);
        else unstuff_index_kernel<false><<<nb + nt, 32 * kIndexWarps, 0, q>>>(P, sl, 0, rec->N, nb);
        ++g_launches;
    };
    // restart-interval index of wave w of slice g on stream q: 1 launched, 0 nothing to do, -1 error
    auto launch_index = [&](int w, cudaStream_t q) -> int {
        ScanList sl;
        sl.n = 0;
        for (int s : waves[w]) if (s >= k0 && s < k) sl.s[sl.n++] = s;
        if (!sl.n) return 0;
        if (copied[w] && cudaStreamWaitEvent(q, rec->ev_copy[w], 0) != cudaSuccess) return -1;
        launch_index_kernel(sl, q);
        return 1;
    };
    auto run_stage = [&](int stage, int g, cudaStream_t q) -> bool {
        const uint32_t i0 = rec->slice_img[g], i1 = rec->slice_img[g + 1];
        const uint32_t u0 = rec->slice_unit[g], nu = rec->slice_unit[g + 1] - u0;
        if (stage == 0) return true;             // (coefficients need no clearing: every decode writes the same values to the same places)
        if (stage == 1) {
            if (pipelined || g != 0) return true;   // done wave by wave, as the bytes arrive; one launch covers every slice
            ScanList sl;
            sl.n = 0;
            for (int s = k0; s < k; ++s) sl.s[sl.n++] = s;
            launch_index_kernel(sl, q);
            return true;
        }
        if (stage < 2 + W) {
            const int w = stage - 2;
            if (pipelined) {
                if (w > 0 && indexed[w]) {
                    // the later waves were indexed on the side stream, beside the first wave
                    if (cudaStreamWaitEvent(q, rec->ev_index[w], 0) != cudaSuccess) return false;
                }
            }
            const ScanScript& first = rec->script[waves[w][0]];
            const bool sequential = first.Ss == 0 && first.Se == 63;   // a baseline record: its one scan is sequential
            // The runs of items of the wave's scans, pairs (the longest chains) first: those of lane-per-interval warps, and
            // those of refine_kernel's CTAs.
            ItemRuns runs, refs;
            runs.n = refs.n = 0;
            uint32_t count = 0, ref_count = 0;
            bool refine = false, failed = false;           // waves without AC refinements need no mask queues
            int dc_n = 0, dc_s[3];                         // the wave's DC refinements, at most one per component
            for (int s : waves[w])
                if (s >= k0 && s < k && rec->script[s].Ss == 0 && rec->script[s].Ah != 0 && dc_n < 3) dc_s[dc_n++] = s;
            bool dc_done = dc_n == 0;
            auto carry_dc = [&](ItemRuns& with, unsigned chunks) -> unsigned {      // the DC refinements in extra blocks of a launch
                with.dc_pos0 = i0; with.dc_images = i1 - i0; with.dc_chunks = chunks;
                for (int j = 0; j < dc_n; ++j) with.dc_s[j] = dc_s[j];
                dc_done = true;
                return dc_n * with.dc_images * chunks;
            };
            auto launch_items = [&](bool last) {
                if (!count) return;
                unsigned nb = (count + kEntropyWarps - 1) / kEntropyWarps;
                const uint32_t smem = kEntropyWarps * (refine ? warp_bytes<true>() : warp_bytes<false>());
                runs.item_blocks = nb;
                if (last && refine && !dc_done) nb += carry_dc(runs, (rec->dc_refine_chunks + 1) / 2);      // about five MCUs a thread (waves without AC refinements are compiled without this)
                const int form = first_pass_form(rec, waves[w], k0, k);
                if (refine) {
                    if (roi) entropy_kernel<true, true, kFirstFull><<<nb, 32 * kEntropyWarps, smem, q>>>(P, runs);
                    else entropy_kernel<false, true, kFirstFull><<<nb, 32 * kEntropyWarps, smem, q>>>(P, runs);
                } else if (form == kFirstFull) {
                    if (roi) entropy_kernel<true, false, kFirstFull><<<nb, 32 * kEntropyWarps, smem, q>>>(P, runs);
                    else entropy_kernel<false, false, kFirstFull><<<nb, 32 * kEntropyWarps, smem, q>>>(P, runs);
                } else if (form == kFirstShort) {
                    if (roi) entropy_kernel<true, false, kFirstShort><<<nb, 32 * kEntropyWarps, smem, q>>>(P, runs);
                    else entropy_kernel<false, false, kFirstShort><<<nb, 32 * kEntropyWarps, smem, q>>>(P, runs);
                } else {
                    if (roi) entropy_kernel<true, false, kFirstFew><<<nb, 32 * kEntropyWarps, smem, q>>>(P, runs);
                    else entropy_kernel<false, false, kFirstFew><<<nb, 32 * kEntropyWarps, smem, q>>>(P, runs);
                }
                ++g_launches;
                runs.n = 0; count = 0;
            };
            auto launch_refinements = [&](bool last) {
                if (!ref_count) return;
                if (!(roi ? allow_refine_smem<true>(rec->device) : allow_refine_smem<false>(rec->device))) failed = true;
                unsigned nb = ref_count;
                refs.item_blocks = nb;
                if (last && !dc_done) nb += carry_dc(refs, (rec->dc_refine_chunks + 1) / 2);      // about two MCUs a thread
                if (roi) refine_kernel<true><<<nb, 32 * kRefineWarps, kRefineBytes, q>>>(P, refs);
                else refine_kernel<false><<<nb, 32 * kRefineWarps, kRefineBytes, q>>>(P, refs);
                ++g_launches;
                refs.n = 0; ref_count = 0;
            };
            bool later = false;                            // a wave before this one holds refinements too
            for (int v = 0; v < w; ++v)
                for (int s : waves[v]) later = later || (s >= k0 && s < k && rec->script[s].Ss > 0 && rec->script[s].Ah != 0);
            const bool ctas = refine_in_ctas(rec, waves[w], paired, later, k0, k);
            auto add_run = [&](bool to_ctas, uint32_t first, uint32_t n) {
                if (!n) return;
                ItemRuns& to = to_ctas ? refs : runs;
                uint32_t& n_to = to_ctas ? ref_count : count;
                if (to.n == kMaxRuns) { if (to_ctas) launch_refinements(false); else launch_items(false); }
                n_to += n;
                if (to.n && to.first[to.n - 1] + (to.end[to.n - 1] - (to.n > 1 ? to.end[to.n - 2] : 0u)) == first) { to.end[to.n - 1] = n_to; return; }
                to.first[to.n] = first; to.end[to.n] = n_to;
                ++to.n;
            };
            std::vector<char> in_pair(rec->G, 0);
            for (int s : waves[w]) {
                if (s < k0 || s >= k) continue;
                refine = refine || (!ctas && rec->script[s].Ss > 0 && rec->script[s].Ah != 0);
                if (!paired || rec->pair_of[s] < k0) continue;
                in_pair[s] = in_pair[rec->pair_of[s]] = 1;
                if (!sequential) add_run(ctas, rec->pair_begin[(size_t)g * G + s], rec->pair_count[(size_t)g * G + s]);
            }
            for (int s : waves[w]) {
                if (s < k0 || s >= k || in_pair[s]) continue;
                add_run(ctas && rec->script[s].Ss > 0 && rec->script[s].Ah != 0, rec->item_begin[(size_t)g * G + s], rec->item_count[(size_t)g * G + s]);
            }
            const uint32_t begin = runs.n ? runs.first[0] : 0u;
            if (sequential) {
                if (count) {
                    const unsigned nl = (count + kSeqLaneWarps - 1) / kSeqLaneWarps;
                    if (sequential_in_ctas(rec, waves[w][0])) {
                        if (roi) sequential_kernel<true><<<count, 32 * kSeqWarps, 0, q>>>(P, begin);
                        else sequential_kernel<false><<<count, 32 * kSeqWarps, 0, q>>>(P, begin);
                    } else if (roi) sequential_lane_kernel<true><<<nl, 32 * kSeqLaneWarps, 0, q>>>(P, begin, count);
                    else sequential_lane_kernel<false><<<nl, 32 * kSeqLaneWarps, 0, q>>>(P, begin, count);
                    ++g_launches;
                }
                const int s0 = waves[w][0];      // the record's one scan
                const uint32_t lc = (s0 >= k0 && s0 < k) ? rec->long_count[(size_t)g * G + s0] : 0u;
                if (lc) {                                  // images whose scan is one long restart interval
                    const uint32_t* list = rec->d_long + rec->long_begin[(size_t)g * G + s0];
                    if (wide_long_scans(rec, waves[w], true, k0, k)) sequential_long_kernel<kSeqLongWideWarps><<<lc, 32 * kSeqLongWideWarps, 0, q>>>(P, list, lc);
                    else sequential_long_kernel<kSeqLongWarps><<<lc, 32 * kSeqLongWarps, 0, q>>>(P, list, lc);
                    ++g_launches;
                }
                return true;
            }
            launch_refinements(true);
            launch_items(true);
            if (failed) return false;
            // scans that are one long restart interval: the first passes of the wave (a contiguous run
            // of the list) ...
            {
                uint32_t lb = 0, lc = 0;
                bool lany = false;
                for (int s : waves[w]) {
                    if (s >= k) break;
                    if (s < k0 || rec->script[s].Ah != 0) continue;
                    if (!lany) { lb = rec->long_begin[(size_t)g * G + s]; lany = true; }
                    lc += rec->long_count[(size_t)g * G + s];
                }
                if (lc) {
                    if (wide_long_scans(rec, waves[w], false, k0, k)) first_pass_long_kernel<kLongWideWarps><<<lc, 32 * kLongWideWarps, 0, q>>>(P, rec->d_long + lb, lc);
                    else first_pass_long_kernel<kLongWarps><<<lc, 32 * kLongWarps, 0, q>>>(P, rec->d_long + lb, lc);
                    ++g_launches;
                }
            }
            // ... (their AC refinements follow in one launch for the whole record, once every slice
            // has finished its waves) and the DC refinement scans that the interval kernel did not take
            for (int j = 0; j < dc_n && !dc_done; ++j) {
                const int s = dc_s[j];
                for (uint32_t p0 = i0; p0 < i1; p0 += 65535u) {
                    dc_refine_kernel<<<dim3(rec->dc_refine_chunks, std::min(i1 - p0, 65535u)), 256, 0, q>>>(P, s, p0);
                    ++g_launches;
                }
            }
            return true;
        }
        Params Q = P;
        Q.units = P.units + u0;
        if (stage == 2 + W) {
            // the AC refinements of scans that are one long restart interval: one persistent launch
            // for all slices (the first slice's stream carries it; the caller has joined the others)
            if (g != 0 || !chains) return true;
            const int levels = std::max(fl.n[0], std::max(fl.n[1], fl.n[2]));
            const int rounds = std::max(1, chain_depth / levels);
            const int pairs = 4 * rounds * levels;          // chains per CTA: a decoding and a helper warp each
            if (cudaMemsetAsync(rec->d_chain_sync, 0, (size_t)(4 + 4 * (size_t)rec->n_groups) * 4, q) != cudaSuccess) return false;
            const unsigned grid = std::min<unsigned>((unsigned)rec->n_sms, (rec->n_groups + 3u) / 4u);
            ac_refine_group_kernel<<<grid, 64 * pairs, (size_t)pairs * sizeof(ChainShared), q>>>(P, fl, rec->d_group, rec->n_groups, rec->d_chain_sync, levels, rounds);
            ++g_launches;
            return true;
        }
        if (nu) {
            launch_pixels(plan, nu, q, Q, cl, static_cast<uint8_t*>(out));
            // the grid's second dimension (one image each) holds at most 65535 entries
            for (uint32_t p0 = i0; targs && p0 < i1; p0 += 65535u) {
                const dim3 tg((unsigned)((targs->size + kTensorRows - 1) / kTensorRows), std::min(i1 - p0, 65535u));
                if (targs->f32 == 2) launch_tensor<__nv_bfloat16>(tg, q, P, *targs, static_cast<const uint8_t*>(out), p0);
                else if (targs->f32) launch_tensor<float>(tg, q, P, *targs, static_cast<const uint8_t*>(out), p0);
                else launch_tensor<__half>(tg, q, P, *targs, static_cast<const uint8_t*>(out), p0);
                ++g_launches;
            }
        }
        return true;
    };
    auto launched_in = [&](int stage) -> int {      // kernel launches of a stage over all slices (for the profile)
        if (stage == 0) return 0;
        if (stage == 2 + W) return chains ? 1 : 0;
        if (stage >= 2 && stage < 2 + W) {
            bool any = false;
            for (int s : waves[stage - 2]) if (s >= k0 && s < k) any = true;
            if (!any) return 0;
        }
        return rec->n_slices;
    };
    const int n_stages = 4 + W;
    if (rec->n_slices == 1 || prof) {
        // one stage after the other (also the timed layout of the stage profile); with several
        // slices the slices of a stage run side by side on their streams, between two joins
        for (int stage = 0; stage < n_stages; ++stage) {
            if (rec->n_slices == 1) {
                if (!run_stage(stage, 0, st)) return PCR_E_CUDA;
            } else {
                if (cudaEventRecord(rec->ev_fork, st) != cudaSuccess) return PCR_E_CUDA;
                for (int g = 0; g < rec->n_slices; ++g) {
                    cudaStream_t q = rec->streams[g];
                    if (cudaStreamWaitEvent(q, rec->ev_fork, 0) != cudaSuccess) return PCR_E_CUDA;
                    if (!run_stage(stage, g, q)) return PCR_E_CUDA;
                    if (cudaEventRecord(rec->ev_join[g], q) != cudaSuccess) return PCR_E_CUDA;
                    if (cudaStreamWaitEvent(st, rec->ev_join[g], 0) != cudaSuccess) return PCR_E_CUDA;
                }
            }
            char name[24];
            if (stage == 0) snprintf(name, sizeof name, "clear");
            else if (stage == 1) snprintf(name, sizeof name, "index");
            else if (stage < 2 + W) snprintf(name, sizeof name, "entropy%d", stage - 2);
            else if (stage == 2 + W) snprintf(name, sizeof name, "chains");
            else snprintf(name, sizeof name, "pixels");
            const int nl = launched_in(stage);
            if (stage <= 1 || stage == n_stages - 1 || nl) mark(name, nl);
        }
    } else {
        // every slice is its own pipeline on its own stream, forked from and joined to the caller's;
        // missing record bytes arrive on a copy stream, the scan groups of each wave behind an event
        if (cudaEventRecord(rec->ev_fork, st) != cudaSuccess) return PCR_E_CUDA;
        if (cudaStreamWaitEvent(rec->side_stream, rec->ev_fork, 0) != cudaSuccess) return PCR_E_CUDA;
        if (rec->resident < need) {
            bool any = false;
            for (int w = 0; w < W; ++w) {
                size_t upto = 0;
                for (int s : waves[w]) if (s < k) upto = std::max(upto, (size_t)rec->group_end[s + 1]);
                if (upto > rec->resident) {
                    const size_t from = rec->resident & ~(size_t)15;
                    if (cudaMemcpyAsync(rec->d_rec + from, rec->host + from, upto - from, cudaMemcpyHostToDevice, rec->copy_stream) != cudaSuccess) return PCR_E_CUDA;
                    rec->resident = upto;
                    any = true;
                }
                if (any) {
                    if (cudaEventRecord(rec->ev_copy[w], rec->copy_stream) != cudaSuccess) return PCR_E_CUDA;
                    copied[w] = true;
                }
            }
        }
        // restart-interval index, one launch per wave for all slices: the first wave's on the caller's
        // stream, the later waves' on the side stream, beside the first entropy wave
        if (launch_index(0, st) < 0) return PCR_E_CUDA;
        if (cudaEventRecord(rec->ev_start, st) != cudaSuccess) return PCR_E_CUDA;
        for (int w = 1; w < W; ++w) {
            const int li = launch_index(w, rec->side_stream);
            if (li < 0) return PCR_E_CUDA;
            indexed[w] = li > 0;
            if (li > 0 && cudaEventRecord(rec->ev_index[w], rec->side_stream) != cudaSuccess) return PCR_E_CUDA;
        }
        // with a chain launch the slices meet once: it follows the entropy waves of all of them
        const int meet = chains ? 2 + W : n_stages;
        for (int g = 0; g < rec->n_slices; ++g) {
            cudaStream_t q = rec->streams[g];
            if (cudaStreamWaitEvent(q, rec->ev_start, 0) != cudaSuccess) return PCR_E_CUDA;
            for (int stage = 0; stage < meet; ++stage)
                if (!run_stage(stage, g, q)) return PCR_E_CUDA;
            if (cudaEventRecord(rec->ev_join[g], q) != cudaSuccess) return PCR_E_CUDA;
            if (!chains && cudaStreamWaitEvent(st, rec->ev_join[g], 0) != cudaSuccess) return PCR_E_CUDA;
        }
        if (chains) {
            cudaStream_t q0 = rec->streams[0];
            for (int g = 1; g < rec->n_slices; ++g)
                if (cudaStreamWaitEvent(q0, rec->ev_join[g], 0) != cudaSuccess) return PCR_E_CUDA;
            if (!run_stage(2 + W, 0, q0)) return PCR_E_CUDA;
            if (cudaEventRecord(rec->ev_chain, q0) != cudaSuccess) return PCR_E_CUDA;
            for (int g = 0; g < rec->n_slices; ++g) {
                cudaStream_t q = rec->streams[g];
                if (g && cudaStreamWaitEvent(q, rec->ev_chain, 0) != cudaSuccess) return PCR_E_CUDA;
                for (int stage = 3 + W; stage < n_stages; ++stage)
                    if (!run_stage(stage, g, q)) return PCR_E_CUDA;
                if (cudaEventRecord(rec->ev_join[g], q) != cudaSuccess) return PCR_E_CUDA;
                if (cudaStreamWaitEvent(st, rec->ev_join[g], 0) != cudaSuccess) return PCR_E_CUDA;
            }
        }
        // the side and copy streams rejoin the caller's stream too (implied by the slices' waits
        // whenever they carried work; stated so that every fork is joined)
        if (cudaEventRecord(rec->ev_side, rec->side_stream) != cudaSuccess) return PCR_E_CUDA;
        if (cudaStreamWaitEvent(st, rec->ev_side, 0) != cudaSuccess) return PCR_E_CUDA;
        if (copied[W - 1] && cudaStreamWaitEvent(st, rec->ev_copy[W - 1], 0) != cudaSuccess) return PCR_E_CUDA;
    }
    if (cudaEventRecord(rec->ev_done, st) != cudaSuccess) return PCR_E_CUDA;
    rec->decode_enqueued = true;
    if (cudaGetLastError() != cudaSuccess) return PCR_E_CUDA;
    return PCR_OK;
}

extern "C" {

void pcr_release_cached_memory(void) {
    {
        std::vector<pcr_record*> gone;
        {
            std::lock_guard<std::mutex> lk(g_rcache.mu);
            gone.swap(g_rcache.lru);
            g_rcache.bytes = 0;
        }
        for (pcr_record* r : gone) { free_device(r); delete r; }
    }
    std::lock_guard<std::mutex> lk(g_cache.mu);
    for (auto& kv : g_cache.free_) cudaFree(kv.second);
    g_cache.free_.clear();
    g_cache.cached = 0;
    std::lock_guard<std::mutex> lh(g_host.mu);
    for (auto& kv : g_host.free_) cudaFreeHost(kv.second);
    g_host.free_.clear();
    g_host.cached = 0;
}

int pcr_decode(pcr_record* rec, int k, void* out, void* stream) {
    if (!rec || !out || k < 1 || k > rec->G) return PCR_E_ARG;
    if (reinterpret_cast<uintptr_t>(out) & 15u) return PCR_E_ARG;
    return decode_range(rec, 0, k, out, stream);
}

int pcr_decode_more(pcr_record* rec, int k, void* out, void* stream) {
    if (!rec || !out || k < 1 || k > rec->G) return PCR_E_ARG;
    if (reinterpret_cast<uintptr_t>(out) & 15u) return PCR_E_ARG;
    if (rec->decoded_k < 1 || k <= rec->decoded_k) return PCR_E_ARG;
    return decode_range(rec, rec->decoded_k, k, out, stream);
}

int pcr_decode_tensor(pcr_record* rec, int k, const pcr_crop* crops, int size, const float* mean, const float* std_,
                      int dtype, void* rgb, void* tensor, void* stream) {
    if (!rec || !crops || !mean || !std_ || !rgb || !tensor || k < 1 || k > rec->G) return PCR_E_ARG;
    if (rec->upsampling != PCR_UPSAMPLE_REPLICATE) return PCR_E_ARG;      // the tensor path resamples replicated chroma only
    if (size < 1 || size > 4096 || (dtype != PCR_F16 && dtype != PCR_F32 && dtype != PCR_BF16)) return PCR_E_ARG;
    if (reinterpret_cast<uintptr_t>(rgb) & 15u) return PCR_E_ARG;
    if (reinterpret_cast<uintptr_t>(tensor) & (dtype == PCR_F32 ? 3u : 1u)) return PCR_E_ARG;
    static_assert(sizeof(pcr_crop) == sizeof(CropRect), "pcr_crop and CropRect have the same layout");
    for (int i = 0; i < rec->N; ++i) {
        const pcr_crop& c = crops[i];
        const pcr_image_info& inf = rec->info[i];
        if (inf.out_bytes >= (1ull << 31)) return PCR_E_ARG;      // the epilogue indexes an image's bytes with 32 bits
        if (c.w < 1 || c.h < 1 || c.flip > 1 || c.x0 > inf.width || c.y0 > inf.height || c.w > inf.width - c.x0 ||
            c.h > inf.height - c.y0) return PCR_E_ARG;
        if (!(std_[0] > 0.f) || !(std_[1] > 0.f) || !(std_[2] > 0.f)) return PCR_E_ARG;
    }
    if (!rec->d_crops) {
        if (int rc = take(rec, &rec->d_crops, (size_t)rec->N * sizeof(CropRect))) return rc;
    }
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    if (cudaMemcpyAsync(rec->d_crops, crops, (size_t)rec->N * sizeof(CropRect), cudaMemcpyHostToDevice, st) != cudaSuccess) return PCR_E_CUDA;
    TensorArgs T;
    T.crops = rec->d_crops; T.out = tensor; T.size = size; T.f32 = dtype == PCR_F32 ? 1 : (dtype == PCR_BF16 ? 2 : 0);
    for (int c = 0; c < 3; ++c) { T.mean[c] = mean[c]; T.inv_std[c] = 1.0f / std_[c]; }
    const int rc = decode_range(rec, 0, k, rgb, stream, &T);
    rec->decoded_k = 0;          // rows outside the crops were not decoded: nothing to raise the fidelity of
    return rc;
}

static void msssim_layout(pcr_record* rec, std::vector<MsDesc>* table) {
    uint64_t floats = 0;
    if (table) table->resize(rec->N);
    for (int i = 0; i < rec->N; ++i) {
        const uint32_t W = rec->info[i].width, H = rec->info[i].height;
        uint32_t M = 0;
        while (M < (uint32_t)kMsMaxScales && (std::min(W, H) >> M) >= (uint32_t)kMsWin) ++M;
        uint64_t len = 0;
        for (uint32_t j = 0; j < M; ++j) len += (uint64_t)(W >> j) * (H >> j);
        if (table) {
            MsDesc& d = (*table)[i];
            d.W = W; d.H = H; d.M = M; d.rsvd = 0;
            d.rgb_off = rec->info[i].out_offset; d.plane_off = floats; d.plane_len = len;
        }
        floats += 2 * len;
    }
    floats = (floats + 1) & ~1ull;                      // the double-precision sums start 8-byte aligned
    rec->ms_floats = floats;
    rec->ms_scratch = (size_t)(floats * 4 + (uint64_t)rec->N * kMsMaxScales * 2 * 8);
}

size_t pcr_msssim_scratch_bytes(pcr_record* rec) {
    if (!rec) return 0;
    if (!rec->ms_scratch) msssim_layout(rec, nullptr);
    return rec->ms_scratch;
}

int pcr_msssim(pcr_record* rec, const void* rgb_a, const void* rgb_b, void* scratch, float* dev_scores, void* stream) {
    if (!rec || !rgb_a || !rgb_b || !scratch || !dev_scores) return PCR_E_ARG;
    if ((reinterpret_cast<uintptr_t>(scratch) & 15u) || (reinterpret_cast<uintptr_t>(dev_scores) & 3u)) return PCR_E_ARG;
    if (rec->N > 65535) return PCR_E_ARG;       // one grid row per image
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    if (!rec->d_ms) {
        std::vector<MsDesc> table;
        msssim_layout(rec, &table);
        Tables T;
        T.add(table.size() * sizeof(MsDesc));
        if (int rc = T.allocate(rec)) return rc;
        std::copy(table.begin(), table.end(), T.h<MsDesc>(0));
        if (int rc = T.copy(rec, T.bytes)) return rc;
        rec->d_ms = T.d<MsDesc>(0);
        if (cudaEventRecord(rec->ev_ready, rec->up_stream) != cudaSuccess) return PCR_E_CUDA;
    }
    if (cudaStreamWaitEvent(st, rec->ev_ready, 0) != cudaSuccess) return PCR_E_CUDA;
    float* planes = static_cast<float*>(scratch);
    double* sums = reinterpret_cast<double*>(planes + rec->ms_floats);
    if (cudaMemsetAsync(sums, 0, (size_t)rec->N * kMsMaxScales * 2 * 8, st) != cudaSuccess) return PCR_E_CUDA;
    MsWindow win;
    {
        double g[kMsWin], tot = 0.0;
        for (int k = 0; k < kMsWin; ++k) { const double x = k - (kMsWin - 1) / 2.0; g[k] = exp(-(x * x) / (2.0 * 1.5 * 1.5)); tot += g[k]; }
        for (int k = 0; k < kMsWin; ++k) win.g[k] = (float)(g[k] / tot);
    }
    const unsigned N = (unsigned)rec->N;
    ms_luma_kernel<<<dim3(64, N), 256, 0, st>>>(rec->d_ms, static_cast<const uint8_t*>(rgb_a), static_cast<const uint8_t*>(rgb_b), planes);
    ++g_launches;
    for (int j = 0; j < kMsMaxScales; ++j) {
        ms_scale_kernel<<<dim3(j == 0 ? 32 : (j == 1 ? 8 : 2), N), kMsTile * kMsTile, 0, st>>>(rec->d_ms, planes, sums, j, win);
        ++g_launches;
        if (j + 1 < kMsMaxScales) {
            ms_pool_kernel<<<dim3(j == 0 ? 32 : 8, N), 256, 0, st>>>(rec->d_ms, planes, j);
            ++g_launches;
        }
    }
    ms_final_kernel<<<(N + 255) / 256, 256, 0, st>>>(rec->d_ms, sums, dev_scores, (int)N);
    ++g_launches;
    // pcr_close waits for this event before it hands the record's buffers (the table above among them) on
    if (cudaEventRecord(rec->ev_done, st) != cudaSuccess) return PCR_E_CUDA;
    rec->decode_enqueued = true;
    if (cudaGetLastError() != cudaSuccess) return PCR_E_CUDA;
    return PCR_OK;
}

int pcr_set_upsampling(pcr_record* rec, int mode) {
    if (!rec || (mode != PCR_UPSAMPLE_REPLICATE && mode != PCR_UPSAMPLE_TRIANGLE)) return PCR_E_ARG;
    if (mode == PCR_UPSAMPLE_TRIANGLE && !(rec->hs == 2 && rec->vs == 2 && rec->nc == 3)) return PCR_E_ARG;   // built for 4:2:0
    if (mode == PCR_UPSAMPLE_TRIANGLE && !rec->d_chroma) {
        if (int rc = take(rec, &rec->d_chroma, (size_t)(std::max<uint64_t>(rec->total_blocks / 6, 1) * 128)   /* 4:2:0: six blocks per MCU */)) return rc;
    }
    rec->upsampling = mode;
    return PCR_OK;
}

int pcr_status(pcr_record* rec, int* first_bad_image, int* code) {
    if (!rec || !first_bad_image || !code) return PCR_E_ARG;
    if (cudaMemcpy(rec->h_status.data(), rec->d_status, (size_t)rec->N * 4, cudaMemcpyDeviceToHost) != cudaSuccess) return PCR_E_CUDA;
    *first_bad_image = -1; *code = PCR_OK;
    for (int i = 0; i < rec->N; ++i)
        if (rec->h_status[i] != 0) { *first_bad_image = i; *code = rec->h_status[i]; break; }
    return PCR_OK;
}

int pcr_coeffs(pcr_record* rec, const int16_t** dev_planes, size_t* bytes) {
    if (!rec || !dev_planes || !bytes) return PCR_E_ARG;
    // the decode keeps coefficients as lists: expand them into the canonical layout now
    if (!rec->d_planes)
        if (int rc = take(rec, &rec->d_planes, (size_t)(std::max<uint64_t>(rec->total_blocks, 1) * 128))) return rc;
    if (!rec->planes_current && rec->total_blocks) {
        CoefLists cl;
        coef_lists(rec, rec->lists_k, &cl);
        launch_planes(sampling_code(rec->hs, rec->vs, rec->nc), rec->n_units, record_params(rec), cl);
        if (cudaDeviceSynchronize() != cudaSuccess) return PCR_E_CUDA;
        rec->planes_current = true;
    }
    *dev_planes = rec->d_planes;
    *bytes = (size_t)rec->total_blocks * 128;
    return PCR_OK;
}

int pcr_image_blocks(const pcr_record* rec, int i, uint64_t* first_block, uint64_t* n_blocks) {
    if (!rec || !first_block || !n_blocks || i < 0 || i >= rec->N) return PCR_E_ARG;
    *first_block = rec->blk_base[i];
    *n_blocks = rec->nblk[i];
    return PCR_OK;
}

int pcr_get_scan(const pcr_record* rec, int s, pcr_scan_info* info) {
    if (!rec || !info || s < 0 || s >= rec->G) return PCR_E_ARG;
    const ScanScript& sc = rec->script[s];
    info->ncomp = sc.ncomp;
    for (int i = 0; i < 3; ++i) info->comp[i] = sc.comp[i];
    info->Ss = sc.Ss; info->Se = sc.Se; info->Ah = sc.Ah; info->Al = sc.Al;
    info->wave = rec->wave_of_scan[s];
    info->rsvd = 0;
    info->bytes = rec->group_end[s + 1] - rec->group_end[s];
    return PCR_OK;
}

int pcr_get_sampling(const pcr_record* rec, int* hs, int* vs, int* ncomp) {
    if (!rec || !hs || !vs || !ncomp) return PCR_E_ARG;
    *hs = rec->hs; *vs = rec->vs; *ncomp = rec->nc;
    return PCR_OK;
}

int pcr_set_profiling(pcr_record* rec, int enable) {
    if (!rec) return PCR_E_ARG;
    if (enable && rec->events.empty()) {
        for (int i = 0; i <= kMaxStages; ++i) {
            cudaEvent_t e;
            if (cudaEventCreate(&e) != cudaSuccess) return PCR_E_CUDA;
            rec->events.push_back(e);
        }
    }
    rec->profiling = enable != 0;
    return PCR_OK;
}

int pcr_get_profile(pcr_record* rec, pcr_stage_time* out, int cap, int* n) {
    if (!rec || !out || !n || cap < 0) return PCR_E_ARG;
    *n = 0;
    for (size_t i = 0; i < rec->profile.size() && (int)i < cap; ++i) {
        out[i] = rec->profile[i];
        if (cudaEventElapsedTime(&out[i].ms, rec->events[i], rec->events[i + 1]) != cudaSuccess) return PCR_E_CUDA;
        ++*n;
    }
    return PCR_OK;
}

uint64_t pcr_launch_count(void) { return g_launches.load(); }

int pcr_selftest_bounded_wait(int* gave_up) {
    if (!gave_up) return PCR_E_ARG;
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return PCR_E_CUDA;
    int* d = static_cast<int*>(dev_alloc(sizeof(int), dev));
    if (!d) return PCR_E_NOMEM;
    int rc = PCR_OK;
    if (cudaMemset(d, 0xFF, sizeof(int)) != cudaSuccess) rc = PCR_E_CUDA;
    if (rc == PCR_OK) {
        bounded_wait_probe_kernel<<<1, 32>>>(2000u, d);      // 2000 polls of about 64 ns: the wait ends by itself
        ++g_launches;
        if (cudaMemcpy(gave_up, d, sizeof(int), cudaMemcpyDeviceToHost) != cudaSuccess) rc = PCR_E_CUDA;
    }
    dev_release(d, sizeof(int), dev);
    return rc;
}

const char* pcr_strerror(int code) {
    switch (code) {
    case PCR_OK: return "ok";
    case PCR_E_ARG: return "invalid argument";
    case PCR_E_FORMAT: return "not a valid or supported record";
    case PCR_E_CORRUPT: return "corrupt entropy-coded data";
    case PCR_E_TIMEOUT: return "device-side wait timed out";
    case PCR_E_CUDA: return "CUDA runtime error";
    case PCR_E_NOMEM: return "out of memory";
    default: return "unknown error";
    }
}

// ---------------------------------------------------------------------------------------
// pcr_pixels_noalloc: the pixel stage for one image, for callers that may not allocate.
// The pixel kernel reads an image descriptor, a work-unit list and the quantisers from
// global memory; pcr_open puts those in cudaMalloc'd tables.  Here they live in one
// file-scope device array that a small kernel fills on every call.
// ---------------------------------------------------------------------------------------
namespace {

constexpr uint32_t kNoAllocMaxDim = 4096;                                         // pixels per side
constexpr uint32_t kNoAllocMcus = kUnitMcus[kSamp420], kNoAllocRows = kUnitRows[kSamp420];
constexpr uint32_t kNoAllocMaxUnits = (kNoAllocMaxDim / 16 / kNoAllocRows) * (kNoAllocMaxDim / 16 / kNoAllocMcus);
struct NoAllocScratch {
    uint16_t qtab[192];
    Unit units[kNoAllocMaxUnits];
};
static __device__ __align__(256) unsigned char g_noalloc_scratch[sizeof(NoAllocScratch)];

struct QuantArg { uint16_t q[192]; };

__global__ void noalloc_fill_kernel(uint32_t W, uint32_t H, QuantArg qa) {
    NoAllocScratch* s = reinterpret_cast<NoAllocScratch*>(g_noalloc_scratch);   // device code may name the array
    const uint32_t mx = (W + 15) / 16, my = (H + 15) / 16;
    const uint32_t per_row = (mx + kNoAllocMcus - 1) / kNoAllocMcus;
    const uint32_t tid = blockIdx.x * blockDim.x + threadIdx.x, nth = gridDim.x * blockDim.x;
    if (tid < 192) s->qtab[tid] = qa.q[tid];
    for (uint32_t u = tid; u < per_row * ((my + kNoAllocRows - 1) / kNoAllocRows); u += nth) {
        Unit un;
        un.img = 0; un.mrow = (uint16_t)(u / per_row * kNoAllocRows); un.mcol0 = (uint16_t)((u % per_row) * kNoAllocMcus);
        un.mx = (uint16_t)mx; un.my = (uint16_t)my; un.W = (uint16_t)W; un.H = (uint16_t)H; un.mcus = 0; un.out_off = 0;
        s->units[u] = un;
    }
}

constexpr int kMaxDevices = 64;
void* g_noalloc_ptr[kMaxDevices];          // device address of the array, per device
std::atomic<int> g_noalloc_ready[kMaxDevices];

}  // namespace

int pcr_pixels_noalloc(const int16_t* dev_coeffs, uint32_t width, uint32_t height, const uint16_t* host_qtab,
                       uint8_t* dev_rgb, void* stream) {
    if (!dev_coeffs || !host_qtab || !dev_rgb || width == 0 || height == 0) return PCR_E_ARG;
    if (width > kNoAllocMaxDim || height > kNoAllocMaxDim) return PCR_E_ARG;   // beyond the fixed scratch
    // the pixel kernel reads every block as eight 16-byte vectors
    if (reinterpret_cast<uintptr_t>(dev_coeffs) & 15u) return PCR_E_ARG;
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return PCR_E_CUDA;
    if (dev < 0 || dev >= kMaxDevices) return PCR_E_ARG;
    if (!g_noalloc_ready[dev].load(std::memory_order_acquire)) {
        // In host code the array's name is only a handle; its device address has to be asked for,
        // once per device, with that device current.
        void* p = nullptr;
        if (cudaGetSymbolAddress(&p, g_noalloc_scratch) != cudaSuccess || !p) { cudaGetLastError(); return PCR_E_CUDA; }
        g_noalloc_ptr[dev] = p;
        g_noalloc_ready[dev].store(1, std::memory_order_release);
    }
    NoAllocScratch* s = static_cast<NoAllocScratch*>(g_noalloc_ptr[dev]);
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    const uint32_t mx = (width + 15) / 16, my = (height + 15) / 16;
    const uint32_t n_units = ((mx + kNoAllocMcus - 1) / kNoAllocMcus) * ((my + kNoAllocRows - 1) / kNoAllocRows);
    QuantArg qa;
    memcpy(qa.q, host_qtab, sizeof qa.q);
    noalloc_fill_kernel<<<(n_units + 255) / 256, 256, 0, st>>>(width, height, qa);
    ++g_launches;
    Params P;
    memset(&P, 0, sizeof P);
    P.planes = const_cast<int16_t*>(dev_coeffs);     // read only by the pixel kernel
    P.units = s->units; P.qtab = s->qtab; P.N = 1;
    CoefLists none;
    memset(&none, 0, sizeof none);
    pixel_kernel<false, 0><<<n_units, unit_threads<kSamp420>(), 0, st>>>(P, none, dev_rgb);
    ++g_launches;
    if (cudaGetLastError() != cudaSuccess) return PCR_E_CUDA;
    return PCR_OK;
}

void pcr_close(pcr_record* rec) {
    if (!rec) return;
    if (g_rcache.limit && rec->key_len) {
        // park it: its set-up and its last decode have to be complete before another handle may use it
        if (rec->up_stream) cudaStreamSynchronize(rec->up_stream);
        if (rec->ev_done && rec->decode_enqueued) cudaEventSynchronize(rec->ev_done);
        rec->device_bytes = 0;
        for (auto& b : rec->bufs) rec->device_bytes += size_class(b.second);
        std::vector<pcr_record*> gone;
        {
            std::lock_guard<std::mutex> lk(g_rcache.mu);
            if (rec->device_bytes <= g_rcache.limit) {
                g_rcache.lru.push_back(rec);
                g_rcache.bytes += rec->device_bytes;
                rec = nullptr;
                evict_records_locked(&gone);
            }
        }
        for (pcr_record* r : gone) { free_device(r); delete r; }
        if (!rec) return;
    }
    free_device(rec);
    delete rec;
}

}  // extern "C"
