// fvv_internal.h -- device-side data layout and kernel launchers of libfvv.
//
// Everything a kernel needs about the rig travels by value in kernel
// parameters (cameras, grid, per-slot arena layout); everything per frame
// lives in the slot's part of the arena.  Launchers enqueue on a stream and
// never synchronise.
#pragma once

#include <algorithm>
#include <cstddef>
#include <cstdint>

#include <cuda_runtime.h>

#include "../../include/fvv.h"

namespace fvv {

constexpr int kMaxComponents = 8192;  // raw components sortable by one block
// int32 from one component's statistics to the next: a 128-byte line each, as
// atomics to one line wait for one another (the labelling of a court frame,
// whose ten or so components take 2,700 words x 7 atomics: 42.2 us with 7
// int32 each, 40.6 with 8, 38.4 with 32).
constexpr int kStatStride = 32;
// Words of the slab the MC compaction stages per chunk: the chunk
// and the neighbours its cells reach (a word in +x, a row in +y, a plane in
// +z).  Chunks whose ROIs reach further read global memory instead.
constexpr uint32_t kSlabWords = 6144;
constexpr int kMaxRois = 4096;
constexpr uint32_t kChunkRoi = 8192;  // a chunk's slab words + kChunkRoi * the ROI of its first word
static_assert(kSlabWords < kChunkRoi && (unsigned long long)kChunkRoi * kMaxRois < 1ull << 32, "chunk_len");
constexpr int kChunk = 256;           // threads of a block of k_mc_compact, fine words per turn of its chunks
constexpr int kMaxTurns = 4;          // turns per chunk, by the words in the launch (launch_filter):
constexpr int kTurnChunks = 4;
constexpr int kMcBlocksPerSm = 4;     // resident blocks of k_mc_compact
constexpr uint32_t kEmptyDepth = 0xFFFFFFFFu;  // depth-buffer bits meaning +inf
constexpr int kMaxTriPerCell = 12;

struct Cam {
    float P[12];
    float C[3];
    int W, H, Wq;        // Wq = 32-bit words per silhouette row
    float Wf, Hf;        // W and H as floats
    uint32_t bit_off;    // first silhouette word of this camera in a slot
    uint32_t blk_off;    // first tile of its blocked silhouette (Layout::silb), kBlkWords words each
    uint64_t pix_off;    // first pixel of this camera in per-slot pixel arrays
    // Bound (pixels) on how far the computed image position of any point the
    // bisection of a grid edge can test lies from the box of the edge ends'
    // approximate image positions; negative: no bound (the camera can see
    // part of the volume at w' <= 0).  See segment_margins in fvv_api.cu.
    float seg_du, seg_dv;
};

struct CamSet {
    int n;
    int oob;             // FVV_OOB_*
    uint64_t cells;      // bit n: camera n's pixel cells (Layout::vcell) decide (see cell_cameras in fvv_api.cu)
    Cam c[FVV_MAX_CAMS];
};

struct Grid {
    float o[3];          // volume origin (vol_min)
    float sc, sf;        // coarse and fine steps
    int nx, ny, nz, nxw; // coarse dims, words per coarse row
    long long coarse_um, fine_um;
    int steps;           // bisection steps
    int rule;            // FVV_SURFACE_*
    int t_np, t_nb;
    float t_v;
    int max_comp, max_rois;
    uint32_t max_fine_words, max_chunks;
    uint32_t max_verts, max_tris;
    int tile_y, tile_z;  // fine-carve tile shape of this launch sequence (kFineTiles)
};

// Fine-carve tiles: kTileX x tile_y x tile_z interior samples, classified
// per camera once and tested in sub-tiles of 4 x kSubY x kSubZ samples, one
// per lane.  The autotuner picks the shape among kFineTiles (FVV_TILE_*).
constexpr int kTileX = 4;
constexpr int kSubY = 2, kSubZ = 4;
constexpr int kFineTiles[FVV_N_TILES][2] = {{4, 8}, {4, 4}, {8, 8}};   // (tile_y, tile_z)

// Per-slot device bookkeeping (zeroed at the start of each reconstruction).
struct SlotInfo {
    unsigned int flags;
    int n_roots;
    int n_rois;
    uint32_t n_words;           // fine words in use
    uint32_t n_chunks;
    uint32_t n_tiles;           // fine-carve tiles of all ROIs
    uint32_t next_tile;         // the fine carve's next unclaimed tile
    uint32_t next_chunk;        // the compaction's next unclaimed chunk
    uint32_t n_verts, n_tris;
    uint32_t n_on;
    uint32_t chunk_words;       // fine words per scan chunk
    uint32_t n_front;           // coarse words that camera 0 does not empty
    unsigned long long tests_coarse, tests_fine, tests_bisect;
    unsigned long long look_fine, look_bisect;   // silhouette words read
};

// Device ROI record (one per kept component).
struct DRoi {
    int cmin[3], cmax[3], gmin[3], gmax[3], fdim[3];
    float fo[3];
    int count;
    int nxw;                    // words per padded fine row
    uint32_t word_off;          // first fine word of this ROI in the slot
    uint32_t n_words;
    uint32_t tile_off;          // first fine-carve tile of this ROI in the slot
    uint32_t vert_off, tri_off; // filled after the scans (for fvv_roi)
};

// Offsets (bytes) of each per-slot array from the slot base.  All 256-aligned.
struct Layout {
    char* base;                 // arena + slots region
    size_t stride;              // bytes per slot
    size_t info;                // SlotInfo
    size_t sil;                 // uint32 silhouette bits
    size_t silb;                // uint32 silhouette bits again, blocked: per camera, tiles of 32 x 32 pixels (row-major,
                                // Wq a row), in a tile 8 x 4 words of 8 x 4 pixels (row-major, bit 8 (y % 4) + x % 8),
                                // so that a 128-byte line holds a square of pixels
    size_t coarse;              // uint32 coarse bits (nz*ny*nxw)
    size_t front;               // uint4 per word that camera 0 leaves voxels of: the word, voxels left, their
                                // foreground votes, first voxel
    size_t parent;              // int32 union-find parents, nx*ny*nz
    size_t roots;               // int32 root linear indices, max_comp
    size_t cstat;               // int32 per component: count, min xyz, max xyz (7 of kStatStride)
    size_t rois;                // DRoi, max_rois
    size_t roi_label;           // int32 label per sorted component (0 = removed)
    size_t fine;                // uint32 fine bits, max_fine_words
    size_t emask;               // uint4 per fine word with a bipolar edge: masks in x, y, z, vertices of earlier words
    size_t chunk_st;            // uint64 x2 per chunk: look-back states (vertices, triangles)
    size_t chunk_len;           // uint32 per chunk: kChunkRoi * the ROI of its first word + words of its staged slab (a multiple of 4; 0: not staged)
    size_t vrec;                // uint64 vertex records, max_verts
    size_t verts;               // float x3, max_verts
    size_t vcell;               // uint2 per vertex and four cameras: its pixel cells (write_cells), max_verts
    size_t tris;                // uint32 x3, max_tris
    size_t tsoup;               // float4 x3 per triangle: its vertices and centroid
                                // (v0 xyz, v1 xyz, v2 xyz, centroid xyz), max_tris
    size_t trec;                // uint64 triangle records (word, cell, case, triangle, ROI), max_tris
    size_t vrgb;                // uint8 x3, max_verts
    size_t vcam;                // int32, max_verts
    size_t depth;               // uint32 per pixel of all cameras
    size_t dbox;                // int32 x4 per camera and ROI: boxes that hold the depth pixels the last z-buffer wrote
    size_t dcount;              // int32 per camera: its boxes
    size_t mask_stage;          // uint8 per pixel (host uploads), or 0
    size_t rgb_stage;           // uint8 x3 per pixel (host uploads), or 0
};

// FVV_FLAG_* bits that say that a slot has no results.
constexpr unsigned kOverCapacity =
    FVV_FLAG_ROOTS | FVV_FLAG_ROIS | FVV_FLAG_FINE | FVV_FLAG_VERTS | FVV_FLAG_TRIS | FVV_FLAG_LOOP;

template <typename T>
__host__ __device__ inline T* slot_ptr(const Layout& L, int slot, size_t off) {
    return reinterpret_cast<T*>(L.base + (size_t)slot * L.stride + off);
}

constexpr uint32_t kBlkWords = 32;      // words of a tile of a blocked silhouette

// Bit (word * 32 + bit, see Layout::silb) of pixel (px, py) in the blocked
// silhouette of an image of Wq words a row.
__host__ __device__ constexpr uint32_t blocked_bit(uint32_t px, uint32_t py, uint32_t Wq) {
    const uint32_t tile = (py >> 5) * Wq + (px >> 5);
    return (tile * kBlkWords + (py & 28u) + (px >> 3 & 3u)) * 32u + (py & 3u) * 8u + (px & 7u);
}

// Where the coarse voxels fall in the first n cameras' silhouettes: the cameras
// are static and so is the grid, so this is laid out once, when the rig is
// created.  e[c * voxels + L]: blocked_bit of voxel L's pixel in camera c, or
// kNoPixel where the voxel is not in front of the camera or not inside its image.
constexpr int kMaxSide = 65535;         // pixels of an image's side
constexpr uint32_t kNoPixel = 0xFFFFFFFFu;
static_assert(blocked_bit(kMaxSide - 1, kMaxSide - 1, (kMaxSide + 31) / 32) < kNoPixel &&
                  (unsigned long long)((kMaxSide + 31) / 32) * ((kMaxSide + 31) / 32) * 1024u <= 1ull << 32,
              "every pixel of the largest image has a bit of its own below kNoPixel");
constexpr int kTableCams = 8;
static_assert(kTableCams * (unsigned long long)((kMaxSide + 31) / 32) * ((kMaxSide + 31) / 32) * kBlkWords < 1ull << 32,
              "the words of the blocked silhouettes of the table's cameras have 32-bit offsets");
struct CoarseTable {
    const uint32_t* e;
    int n;                      // 1 to kTableCams (see coarse_table_cams in fvv_api.cu)
    uint32_t word[kTableCams];  // first words of its cameras' blocked silhouettes
};

struct SlotList {
    int n;
    int s[FVV_MAX_BATCH];
};

// Marching-cubes table in device memory.
struct McTable {
    const uint8_t* ntri;        // [256]
    const uint8_t* edges;       // [256][12][3]
};

// Blocks per slot for a grid-stride kernel: enough for the work, at most
// about 8 blocks per SM over the whole batch.
inline int grid_x(int sms, int n_slots, long long work_items, int per_block) {
    const long long want = (work_items + per_block - 1) / per_block;
    const long long cap = std::max(1LL, (long long)sms * 8 / std::max(1, n_slots));
    return (int)std::max(1LL, std::min(want, cap));
}

// Launch shape of the tunable kernels (index FVV_TUNE_*): threads per block
// (a multiple of 32, <= 256) and resident blocks per SM over the whole batch.
struct Tuning {
    int threads[FVV_N_TUNE];
    int waves[FVV_N_TUNE];
    int fine_tile;       // index into kFineTiles
    int zb_cams;         // groups of four cameras a z-buffer warp takes its triangles through: 1, 2 or 4
};

// The grid with the tuned fine-carve tile shape.
inline Grid tuned_grid_params(const Grid& g, const Tuning& tu) {
    Grid out = g;
    out.tile_y = kFineTiles[tu.fine_tile][0];
    out.tile_z = kFineTiles[tu.fine_tile][1];
    return out;
}

inline Tuning default_tuning() {
    Tuning t;
    for (int k = 0; k < FVV_N_TUNE; ++k) {
        t.threads[k] = 256;
        t.waves[k] = 8;
    }
    t.waves[FVV_TUNE_ZBUFFER] = 16;
    t.waves[FVV_TUNE_COARSE] = 16;
    t.waves[FVV_TUNE_BISECT] = 16;
    t.waves[FVV_TUNE_FINE] = 16;
    t.fine_tile = FVV_TILE_4x4x8;
    t.zb_cams = 4;
    return t;
}

// Blocks per slot of a tuned grid-stride kernel: the tuned blocks per SM
// spread over the launch's slots, but never more than kMaxWavesPerSlot per
// SM for one slot (one frame's work is too little for more: with the
// shapes tuned on a 64-frame batch at 64 blocks per SM, one frame took
// 0.561 ms at p50 uncapped and 0.531 ms capped at 16).
constexpr int kMaxWavesPerSlot = 16;
inline int tuned_grid(const Tuning& tu, int knob, int sms, int n_slots, long long work_items, int parts = 1) {
    const long long per_block = tu.threads[knob];
    const long long want = (work_items + per_block - 1) / per_block;
    const long long cap = std::max(1LL, (long long)sms * std::min(tu.waves[knob], kMaxWavesPerSlot * n_slots) /
                                            std::max(1, n_slots * parts));
    return (int)std::max(1LL, std::min(want, cap));
}

// Blocks per slot of k_clear_fine (256 threads): by the words, and by the images'
// rows (`rows` of all cameras, a warp each, four blocks per SM at most), which the
// depth boxes take however few words a slot holds: eight mat frames in slots of
// twice their words 227 -> 218 us the reconstruction, one such frame 168 -> 150.
inline int clear_blocks(int sms, int n_slots, uint32_t max_fine_words, long long rows) {
    return std::max(grid_x(sms, n_slots, (long long)max_fine_words, 256), grid_x(sms / 2, n_slots, rows, 8));
}

// Blocks per slot of the fine hull, whose warps claim tiles until none is left:
// the slot's share of the blocks that the GPU holds at a time, whatever its
// capacity.  More of them delay the next slot (four 4K court frames 104 us with all
// 608 each, 88 with 152; four court frames 231 and 208).  From 16 slots on the
// launch has a round of resident blocks for every eight (fewer, and more frames'
// silhouettes are in work than the L2 holds: 64 court frames 2964 us with four
// rounds, 3072 with one; 16 of them 762 with two, 772 with one), in whole rounds
// (12 court frames 570 us with one, 627 with one and a half; 24 of them 1133 with
// three, 1218 with one and a half).  One block per 2048 words of capacity starved
// slots fitted to their frames (the clear and the hull of one small frame 84 us
// instead of 22, of one court frame 142 instead of 74) and is a little better only
// where a frame has a few hundred tiles (eight mat frames at 4 cm: 40.4, now 44).
inline int fine_blocks(const Tuning& tu, int sms, int n_slots, uint32_t max_fine_words) {
    const long long resident = (long long)sms * 1024 / tu.threads[FVV_TUNE_FINE];   // at the kernel's 64 registers
    const long long share = resident * std::max(1, n_slots / 8) / n_slots;
    return (int)std::max(1LL, std::min<long long>(share, tuned_grid(tu, FVV_TUNE_FINE, sms, n_slots,
                                                                   (long long)max_fine_words * 32)));
}

// Builds the 256-case table from the face rule (host).
void build_mc_table(uint8_t ntri[256], uint8_t edges[256 * kMaxTriPerCell * 3]);

// ---- launchers (all enqueue on `st`)
// Packs frame j's masks (src[j * cams.n + n]) into slots[j], j < n_frames;
// host_src: the sources are mapped page-locked host memory.
cudaError_t launch_pack(const CamSet& cams, const Layout& L, int n_frames, const int* slots,
                        const uint8_t* const* src, bool host_src, int sms, cudaStream_t st);
cudaError_t launch_coarse_table(const CamSet& cams, const Grid& g, uint32_t* e, int n, cudaStream_t st);
// The coarse hull; the slots' n_front must be zero (k_zero_info, or launch_reset_coarse to run it again).
cudaError_t launch_reset_coarse(const Layout& L, const SlotList& sl, cudaStream_t st);
cudaError_t launch_coarse_carve(const CamSet& cams, const Grid& g, const Layout& L, const SlotList& sl,
                                const CoarseTable& tab, int sms, const Tuning& tu, cudaStream_t st);
// The labelling's and the compaction's kernels made ready on the current device (once, when a rig is created).
cudaError_t prepare_ccl();
cudaError_t prepare_mc();
cudaError_t launch_ccl(const Grid& g, const Layout& L, const SlotList& sl, int sms, cudaStream_t st);
// The filter and ROI table alone (k_filter), e.g. again for another fine-carve tile shape.
cudaError_t launch_filter(const Grid& g, const Layout& L, const SlotList& sl, int sms, cudaStream_t st);
cudaError_t launch_fine_carve(const CamSet& cams, const Grid& g, const Layout& L, const SlotList& sl,
                              int sms, const Tuning& tu, cudaStream_t st);
cudaError_t launch_mc_prefix(const CamSet& cams, const Grid& g, const Layout& L, const SlotList& sl, const McTable& mc, int sms,
                             cudaStream_t st);
cudaError_t launch_bisect(const CamSet& cams, const Grid& g, const Layout& L, const SlotList& sl, int sms,
                          const Tuning& tu, cudaStream_t st);
cudaError_t launch_mc_triangles(const Grid& g, const Layout& L, const SlotList& sl, const McTable& mc, int sms,
                                const Tuning& tu, cudaStream_t st);
// Depth images of every slot to empty and their written boxes to none (once,
// when a rig is created).  They are cleared again where the last z-buffer wrote
// by launch_fine_carve, and launch_mc_prefix lists the next one's boxes.
cudaError_t launch_init_depth(const CamSet& cams, const Layout& L, int n_slots, int sms, cudaStream_t st);
cudaError_t launch_depth(const CamSet& cams, const Grid& g, const Layout& L, const SlotList& sl,
                         int sms, const Tuning& tu, cudaStream_t st);
// Colour-call arguments of up to kColourBatch slots, passed by value as a
// kernel parameter (so nothing is copied from host memory).
constexpr int kColourBatch = 48;
struct ColourBatch {
    int n;
    int slot[kColourBatch];
    float view[kColourBatch][3];
    const uint8_t* rgb[kColourBatch][FVV_MAX_CAMS];
};

cudaError_t launch_colour(const CamSet& cams, const Grid& g, const Layout& L, const ColourBatch& cb, int sms,
                          int total_slots, cudaStream_t st);

// Where the results of a call's slots go (device memory; any may be NULL).
struct GatherSlots {
    int n;
    int slot[FVV_MAX_BATCH];
    char* dst[FVV_MAX_BATCH][4];        // vertices, triangles, colours, cameras
};

// Copies every slot's results to their destinations and its SlotInfo to infos[i]
// (page-locked host memory, device address); slots over a capacity only the latter.
cudaError_t launch_gather_results(const Layout& L, const GatherSlots& gs, SlotInfo* infos, int sms, cudaStream_t st);

// A novel view (step E) of one reconstructed slot: the virtual camera as a
// Cam (P, C, W, H, Wf, Hf; the other fields unused) and the capture RGB.
struct ViewArgs {
    Cam v;
    int slot;
    const uint8_t* rgb[FVV_MAX_CAMS];
};

cudaError_t launch_render_view(const CamSet& cams, const Grid& g, const Layout& L, const ViewArgs& va,
                              unsigned long long* key, uint8_t* out_rgb, int32_t* out_cam, int sms, cudaStream_t st);
cudaError_t launch_debug_pixels(const CamSet& cams, int cam, long long n, const float* pts, int32_t* px,
                                int32_t* py, cudaStream_t st);
cudaError_t launch_debug_labels(const Grid& g, const Layout& L, int slot, int32_t* dst, cudaStream_t st);
// Writes a given coarse grid into slot and seeds its union-find forest as the
// coarse hull does (the slot's SlotInfo must be zeroed first).
cudaError_t launch_debug_seed(const Grid& g, const Layout& L, int slot, const uint32_t* src, cudaStream_t st);
cudaError_t launch_debug_depth(const CamSet& cams, const Layout& L, int slot, float* dst, size_t npix,
                               cudaStream_t st);

}  // namespace fvv
