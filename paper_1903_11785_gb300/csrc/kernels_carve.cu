// kernels_carve.cu -- silhouette packing (step a0) and the coarse and fine
// visual hulls (Sec. II-B-1 and II-B-3).
//
// Silhouettes are kept as 1 bit per pixel (a 1080p camera is 260 KB, a
// 16-camera frame 4 MB, so a frame's silhouettes stay in L2), row by row for
// the fine hull and the surface, which scan short rows of them, and once more in
// square blocks for the coarse hull, whose gathers run across them.
#include <climits>

#include "fvv_device.cuh"

namespace fvv {
namespace {

// The masks of up to kPackFrames frames (frame j: slot[j], camera n:
// src[j * n_cams + n]) packed by one launch.
constexpr int kPackPtrs = 2048;
struct PackSrc {
    const uint8_t* src[kPackPtrs];
    int slot[kPackPtrs / 4];
};

// High bit of each nonzero byte of w, gathered into 4 bits (byte k -> bit k).
__device__ __forceinline__ uint32_t nonzero_bytes4(uint32_t w) {
    uint32_t t = (((w & 0x7F7F7F7Fu) + 0x7F7F7F7Fu) | w) & 0x80808080u;
    return ((t >> 7) & 1u) | ((t >> 14) & 2u) | ((t >> 21) & 4u) | ((t >> 28) & 8u);
}

// Step a0: uint8 mask (nonzero = foreground) -> 1 bit per pixel, 32 pixels per
// word, bit x%32 of word x/32 of its row; and the same bits blocked
// (Layout::silb), whose words are the transposed bytes of four rows' words.
// One thread per 32 x 4 pixels; grid (blocks, cameras, frames).  Bound by
// HBM: eight 16-byte loads are in flight per thread.
// Rows of a width that 32 does not divide, or that do not start at 16 bytes, are
// read by the aligned 4-byte words that hold them: a byte at a time, 8 court
// frames of 1917 x 1079 took 2140 us instead of 2003 a call, four 4K ones of 3838
// pixels 1023 instead of 837.
__global__ void __launch_bounds__(256) k_pack(const __grid_constant__ CamSet cams, const __grid_constant__ PackSrc a,
                                              const __grid_constant__ Layout L) {
    pdl_begin();
    const Cam& c = cams.c[blockIdx.y];
    const uint8_t* src = a.src[blockIdx.z * (unsigned)cams.n + blockIdx.y];
    uint32_t* __restrict__ sil = slot_ptr<uint32_t>(L, a.slot[blockIdx.z], L.sil) + c.bit_off;
    uint32_t* __restrict__ silb = slot_ptr<uint32_t>(L, a.slot[blockIdx.z], L.silb) + (size_t)c.blk_off * kBlkWords;
    const unsigned Wq = (unsigned)c.Wq;
    const size_t units = (size_t)((c.H + 3) >> 2) * Wq;
    const bool vec = (c.W % 32 == 0) && ((reinterpret_cast<uintptr_t>(src) & 15u) == 0);
    for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < units; i += (size_t)gridDim.x * blockDim.x) {
        const size_t r4 = i / Wq;
        const unsigned wq = (unsigned)(i - r4 * Wq);
        const int rows = min(4, c.H - (int)(4 * r4));
        const uint8_t* p = src + 4 * r4 * (unsigned)c.W + (size_t)wq * 32;
        uint32_t bits[4] = {0u, 0u, 0u, 0u};
        if (vec) {
            uint4 v[8];
#pragma unroll
            for (int r = 0; r < 4; ++r) {
                const uint4* q = reinterpret_cast<const uint4*>(p + (size_t)min(r, rows - 1) * (unsigned)c.W);
                v[2 * r] = __ldcs(q);
                v[2 * r + 1] = __ldcs(q + 1);
            }
#pragma unroll
            for (int r = 0; r < 4; ++r) {
                const uint4 a0 = v[2 * r], a1 = v[2 * r + 1];
                bits[r] = nonzero_bytes4(a0.x) | nonzero_bytes4(a0.y) << 4 | nonzero_bytes4(a0.z) << 8 |
                          nonzero_bytes4(a0.w) << 12 | nonzero_bytes4(a1.x) << 16 | nonzero_bytes4(a1.y) << 20 |
                          nonzero_bytes4(a1.z) << 24 | nonzero_bytes4(a1.w) << 28;
            }
        } else {
            // any width and address: the words that hold the rows' 32 bytes,
            // shifted into place; bytes where such a word reaches past the image.
            // (Kept in L1: a thread's last word is the next one's first, and a
            // sector is read by several loads; evict-first, twelve unaligned 4K
            // masks read in place took 529 us instead of 512.)
            const int nb = min(32, c.W - (int)wq * 32);
            const uintptr_t first = reinterpret_cast<uintptr_t>(src), end = first + (size_t)c.W * (unsigned)c.H;
            uintptr_t q[4];
#pragma unroll
            for (int r = 0; r < 4; ++r) q[r] = reinterpret_cast<uintptr_t>(p) + (size_t)min(r, rows - 1) * (unsigned)c.W;
            if ((q[0] & ~(uintptr_t)3) >= first && (q[3] & ~(uintptr_t)3) + 36 <= end) {
                uint32_t v[4][9];
#pragma unroll
                for (int r = 0; r < 4; ++r)
#pragma unroll
                    for (int k = 0; k < 9; ++k) v[r][k] = __ldg(reinterpret_cast<const uint32_t*>(q[r] & ~(uintptr_t)3) + k);
#pragma unroll
                for (int r = 0; r < 4; ++r) {
                    const uint32_t sh = 8u * (uint32_t)(q[r] & 3u);
#pragma unroll
                    for (int k = 0; k < 8; ++k)
                        bits[r] |= nonzero_bytes4(__funnelshift_r(v[r][k], v[r][k + 1], sh)) << (4 * k);
                    bits[r] &= 0xFFFFFFFFu >> (32 - nb);
                }
            } else {
#pragma unroll 1
                for (int b = 0; b < nb; ++b)
#pragma unroll
                    for (int r = 0; r < 4; ++r)
                        bits[r] |= (uint32_t)(reinterpret_cast<const uint8_t*>(q[r])[b] != 0) << b;
            }
        }
#pragma unroll
        for (int r = 0; r < 4; ++r) {
            if (r < rows) sil[(4 * r4 + r) * Wq + wq] = bits[r];
            else bits[r] = 0u;
        }
        // byte k of the four rows' words: the blocked word of columns 8k .. 8k + 7
        const uint32_t lo01 = __byte_perm(bits[0], bits[1], 0x5140), hi01 = __byte_perm(bits[0], bits[1], 0x7362);
        const uint32_t lo23 = __byte_perm(bits[2], bits[3], 0x5140), hi23 = __byte_perm(bits[2], bits[3], 0x7362);
        const size_t at = ((r4 >> 3) * Wq + wq) * 32 + (r4 & 7) * 4;
        *reinterpret_cast<uint4*>(silb + at) =
            make_uint4(__byte_perm(lo01, lo23, 0x5410), __byte_perm(lo01, lo23, 0x7632),
                       __byte_perm(hi01, hi23, 0x5410), __byte_perm(hi01, hi23, 0x7632));
    }
}

// The coarse table (see CoarseTable), one thread per voxel.
__global__ void __launch_bounds__(256) k_coarse_table(const __grid_constant__ CamSet cams, const __grid_constant__ Grid g,
                                                      uint32_t* __restrict__ table, int ncams) {
    const size_t nvox = (size_t)g.nx * g.ny * g.nz;
    for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < nvox; i += (size_t)gridDim.x * blockDim.x) {
        const uint32_t row = (uint32_t)(i / (uint32_t)g.nx);
        const int x = (int)(i - (size_t)row * (uint32_t)g.nx);
        const float X = fadd(g.o[0], fmul(fadd((float)x, 0.5f), g.sc));
        const float Y = fadd(g.o[1], fmul(fadd((float)(int)(row % (uint32_t)g.ny), 0.5f), g.sc));
        const float Z = fadd(g.o[2], fmul(fadd((float)(int)(row / (uint32_t)g.ny), 0.5f), g.sc));
        for (int n = 0; n < ncams; ++n) {
            int px, py;
            cam_pixel(cams.c[n], X, Y, Z, px, py);
            table[n * nvox + i] =
                px < 0 ? kNoPixel : blocked_bit((uint32_t)px, (uint32_t)py, (uint32_t)cams.c[n].Wq);
        }
    }
}

// Sec. II-B-1: the coarse hull over the whole volume, a 32-voxel word of the
// occupancy bitset at a time, a voxel per lane, in two passes.  Occupied voxels
// also start the union-find forest of Sec. II-B-2: each run of consecutive
// occupied voxels within a word is one tree, rooted at the run's first voxel
// (in this word), which is its smallest linear index.
//
// The pixels are read from the coarse table.  A camera's test of a 32-voxel word is then a coalesced load of
// the table, a gather from the blocked silhouette and a ballot, about 14
// instructions instead of 55.  The gather bounds the row-major layout:
// 32 voxels project to a line of some 100 pixels, and unless the line is level
// each lane reads another row, so another 128-byte line (7 million voxels x
// 1.4 tests at the 312 G gathers/s measured for the L2 are 31 us a court
// frame); blocked, the line crosses 4 to 8 lines.
//
// The first pass takes every word through the first `levels` cameras, kWords
// words of a warp in flight together, writes the empty ones and lists the
// others; the second takes the listed words through the other cameras, one at a
// time per warp.  In one pass, the warps whose words cross a player's outline
// held the launch up: 48 to 60 us a court frame however the words were grouped.
// Court frames (229,000 words, 16 cameras): 52 -> 37 us for one, 1960 -> 1070 us
// for 64; four 4K court frames (10 abstaining cameras, 23 million voxels each)
// 453 -> 235 us, against every voxel projected.
constexpr int kWords = 8;
template <bool ABSTAIN, bool MORE>            // MORE: levels > 1
__global__ void __launch_bounds__(256) k_coarse_first(const __grid_constant__ CamSet cams, const __grid_constant__ Grid g,
                                                      const __grid_constant__ Layout L,
                                                      const __grid_constant__ SlotList sl,
                                                      const __grid_constant__ CoarseTable tab, int levels) {
    pdl_begin();
    __shared__ unsigned long long sh[32];
    __shared__ uint32_t s_at[2][8];           // per turn and warp: words it lists, then where they go
    const int slot = sl.s[blockIdx.y];
    const uint32_t* __restrict__ silb = slot_ptr<uint32_t>(L, slot, L.silb);
    uint32_t* bits = slot_ptr<uint32_t>(L, slot, L.coarse);
    uint4* front = slot_ptr<uint4>(L, slot, L.front);
    SlotInfo* info = slot_ptr<SlotInfo>(L, slot, L.info);
    const int lane = threadIdx.x & 31;
    const int wid = threadIdx.x >> 5, bw = blockDim.x >> 5;
    const uint32_t nwords = (uint32_t)g.nz * (uint32_t)g.ny * (uint32_t)g.nxw;
    const size_t nvox = (size_t)g.nz * g.ny * g.nx;
    const uint32_t turn = (uint32_t)bw * (uint32_t)kWords;   // words of the block in a turn
    uint32_t tests = 0;                       // of this lane's words
    int buf = 0;
    for (uint32_t b0 = blockIdx.x * turn; b0 < nwords; b0 += gridDim.x * turn, buf ^= 1) {
        const uint32_t w0 = b0 + (uint32_t)wid * (uint32_t)kWords;
        // lane q < kWords answers for word w0 + q
        const uint32_t w = min(w0 + (uint32_t)(lane % kWords), nwords - 1u);
        const uint32_t row = w / (uint32_t)g.nxw;
        const int x0 = (int)(w - row * (uint32_t)g.nxw) * 32;
        const uint32_t first = row * (uint32_t)g.nx + (uint32_t)x0;
        const int nv = w0 + (uint32_t)(lane % kWords) < nwords ? min(32, g.nx - x0) : 0;
        uint32_t m[kWords];                   // voxels left of each word (the same in every lane)
        uint32_t voted = 0u;                  // foreground votes of this lane's word
        uint32_t any = 0u;
        {   // camera 0
            uint32_t e[kWords], word[kWords];
#pragma unroll
            for (int q = 0; q < kWords; ++q) {
                const uint32_t f = __shfl_sync(kFull, first, q);
                e[q] = lane < __shfl_sync(kFull, nv, q) ? __ldg(tab.e + f + lane) : kNoPixel;
            }
#pragma unroll
            for (int q = 0; q < kWords; ++q) word[q] = e[q] != kNoPixel ? __ldg(silb + tab.word[0] + (e[q] >> 5)) : 0u;
#pragma unroll
            for (int q = 0; q < kWords; ++q) {
                const bool bit = (word[q] >> (e[q] & 31u)) & 1u;
                m[q] = __ballot_sync(kFull, bit);
                if (ABSTAIN) {
                    if (lane == q) voted = m[q];
                    const int n = __shfl_sync(kFull, nv, q);
                    m[q] |= __ballot_sync(kFull, e[q] == kNoPixel) & (n > 0 ? kFull >> (32 - n) : 0u);
                }
                any |= m[q];
            }
            if (lane < kWords) tests += (uint32_t)nv;
        }
        const uint32_t* te = tab.e + nvox + lane;
#pragma unroll 1
        for (int c = 1; MORE && c < levels && any; ++c, te += nvox) {
            const uint32_t* __restrict__ sb = silb + tab.word[c];
            uint32_t e[kWords], word[kWords];
#pragma unroll
            for (int q = 0; q < kWords; ++q) {
                const uint32_t f = __shfl_sync(kFull, first, q);
                e[q] = (m[q] >> lane) & 1u ? __ldg(te + f) : kNoPixel;
            }
#pragma unroll
            for (int q = 0; q < kWords; ++q) word[q] = e[q] != kNoPixel ? __ldg(sb + (e[q] >> 5)) : 0u;
            any = 0u;
#pragma unroll
            for (int q = 0; q < kWords; ++q) {
                tests += lane == q ? (uint32_t)__popc(m[q]) : 0u;
                const bool bit = (word[q] >> (e[q] & 31u)) & 1u;
                const uint32_t v = __ballot_sync(kFull, bit);
                if (ABSTAIN) {
                    if (lane == q) voted |= v;
                    m[q] &= v | __ballot_sync(kFull, e[q] == kNoPixel);
                } else {
                    m[q] = v;
                }
                any |= m[q];
            }
        }
        uint32_t left = 0u;
#pragma unroll
        for (int q = 0; q < kWords; ++q) left = lane == q ? m[q] : left;
        const bool own = lane < kWords && nv > 0;
        if (own && !left) bits[w] = 0u;
        // places in the list, one atomic a block and turn (one a warp took 20 us
        // of a single frame: a counter serves about one atomic a nanosecond)
        const uint32_t who = __ballot_sync(kFull, own && left != 0u);
        if (lane == 0) s_at[buf][wid] = (uint32_t)__popc(who);
        __syncthreads();
        if (wid == 0) {
            const uint32_t n = lane < bw ? s_at[buf][lane] : 0u;
            uint32_t incl = n;
#pragma unroll
            for (int o = 1; o < 8; o <<= 1) {
                const uint32_t y = __shfl_up_sync(kFull, incl, o);
                if (lane >= o) incl += y;
            }
            const uint32_t all = __shfl_sync(kFull, incl, 7);
            uint32_t at = 0;
            if (lane == 0 && all) at = atomicAdd(&info->n_front, all);
            at = __shfl_sync(kFull, at, 0);
            if (lane < bw) s_at[buf][lane] = at + incl - n;
        }
        __syncthreads();
        // (a word is listed once, so the places stay below nwords from a counter that started at zero)
        const uint32_t at = s_at[buf][wid] + (uint32_t)__popc(who & ((1u << lane) - 1u));
        if (((who >> lane) & 1u) && at < nwords) front[at] = make_uint4(w, left, voted, first);
    }
    const unsigned long long t = block_sum<unsigned long long>(tests, sh);
    if (threadIdx.x == 0 && t) atomicAdd(&info->tests_coarse, t);
}

template <bool ABSTAIN>
__global__ void __launch_bounds__(256) k_coarse_rest(const __grid_constant__ CamSet cams, const __grid_constant__ Grid g,
                                                     const __grid_constant__ Layout L,
                                                     const __grid_constant__ SlotList sl,
                                                     const __grid_constant__ CoarseTable tab, int levels) {
    pdl_begin();
    __shared__ uint32_t s_blk[kTableCams];
    __shared__ unsigned long long sh[32];
    const int slot = sl.s[blockIdx.y];
    SlotInfo* info = slot_ptr<SlotInfo>(L, slot, L.info);
    const uint32_t nfront = min(info->n_front, (uint32_t)g.nz * (uint32_t)g.ny * (uint32_t)g.nxw);
    if (((blockIdx.x * blockDim.x) >> 5) >= nfront) return;   // the whole block
    for (int n = threadIdx.x; n < tab.n; n += blockDim.x) s_blk[n] = tab.word[n];
    __syncthreads();
    const uint32_t* __restrict__ silb = slot_ptr<uint32_t>(L, slot, L.silb);
    const uint32_t* __restrict__ sil = slot_ptr<uint32_t>(L, slot, L.sil);
    uint32_t* bits = slot_ptr<uint32_t>(L, slot, L.coarse);
    int* parent = slot_ptr<int>(L, slot, L.parent);
    const uint4* front = slot_ptr<uint4>(L, slot, L.front);
    const int lane = threadIdx.x & 31;
    const size_t nvox = (size_t)g.nz * g.ny * g.nx;
    const uint32_t nwarps = (gridDim.x * blockDim.x) >> 5;
    uint32_t i = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    unsigned long long tests = 0;             // (the same in every lane)
    uint32_t on_count = 0;
    uint4 f = i < nfront ? __ldcg(front + i) : make_uint4(0u, 0u, 0u, 0u);
    for (; i < nfront; i += nwarps) {
        const uint4 cur = f;
        if (i + nwarps < nfront) f = __ldcg(front + i + nwarps);
        uint32_t m = cur.y;                   // voxels left (the same in every lane)
        bool voted = (cur.z >> lane) & 1u;
        const uint32_t* te = tab.e + levels * nvox + cur.w + (uint32_t)lane;
        int n = levels;
        uint32_t e = n < tab.n && ((m >> lane) & 1u) ? __ldg(te) : kNoPixel;
        for (; n < tab.n && m; ++n) {
            const bool live = (m >> lane) & 1u;
            const uint32_t word = live && e != kNoPixel ? __ldg(silb + s_blk[n] + (e >> 5)) : 0u;
            // the next camera's entries are on their way while this one's gather is
            te += nvox;
            const uint32_t next = live && n + 1 < tab.n ? __ldg(te) : kNoPixel;
            tests += (unsigned)__popc(m);
            const bool bit = (word >> (e & 31u)) & 1u;
            if (ABSTAIN) voted |= bit;
            m = __ballot_sync(kFull, live && (bit || (ABSTAIN && e == kNoPixel)));
            e = next;
        }
        if (m && n < cams.n) {                // cameras past the table
            const uint32_t row = cur.w / (uint32_t)g.nx;
            const int x = (int)(cur.w - row * (uint32_t)g.nx) + lane;
            const float X = fadd(g.o[0], fmul(fadd((float)x, 0.5f), g.sc));
            const float Y = fadd(g.o[1], fmul(fadd((float)(int)(row % (uint32_t)g.ny), 0.5f), g.sc));
            const float Z = fadd(g.o[2], fmul(fadd((float)(int)(row / (uint32_t)g.ny), 0.5f), g.sc));
#pragma unroll 1
            for (; n < cams.n && m; ++n) {
                bool live = (m >> lane) & 1u;
                tests += (unsigned)__popc(m);
                if (live) test_cam<ABSTAIN>(cams.c[n], sil, X, Y, Z, live, voted);
                m = __ballot_sync(kFull, live);
            }
        }
        if (ABSTAIN) m = __ballot_sync(kFull, ((m >> lane) & 1u) && voted);
        // occupied voxels start the union-find forest: each run one tree
        if ((m >> lane) & 1u) {
            const uint32_t starts = m & ~(m << 1);   // first voxel of each run
            const int run0 = 31 - __clz(starts & (0xFFFFFFFFu >> (31 - lane)));
            parent[cur.w + (uint32_t)lane] = (int)cur.w + run0;
        }
        if (lane == 0) {
            bits[cur.x] = m;
            on_count += __popc(m);
        }
    }
    const unsigned long long t = block_sum<unsigned long long>(lane == 0 ? tests : 0ull, sh);
    const unsigned long long c = block_sum<unsigned long long>((unsigned long long)on_count, sh);
    if (threadIdx.x == 0) {
        if (t) atomicAdd(&info->tests_coarse, t);
        if (c) atomicAdd(&info->n_on, (uint32_t)c);
    }
}

// Clears the fine grids, the compaction's chunk states and the depth pixels
// that the slot's last z-buffer may have written, and resets the fine carve's
// tile counter.
__global__ void __launch_bounds__(256) k_clear_fine(const __grid_constant__ CamSet cams, const __grid_constant__ Grid g,
                                                    const __grid_constant__ Layout L,
                                                    const __grid_constant__ SlotList sl) {
    pdl_begin();
    const int slot = sl.s[blockIdx.y];
    SlotInfo* info = slot_ptr<SlotInfo>(L, slot, L.info);
    const uint32_t nwords = info->n_words;
    // the first camera's depth boxes (below) are on their way meanwhile
    const int lane = threadIdx.x & 31, bw = blockDim.x >> 5;
    const int blocks = (int)gridDim.x, block = (int)blockIdx.x, n0 = block % cams.n;
    const int* counts = slot_ptr<int>(L, slot, L.dcount);
    const int4* boxes = slot_ptr<int4>(L, slot, L.dbox);
    const int count0 = counts[n0];
    const int4 first0 = boxes[(size_t)n0 * (unsigned)g.max_rois + (unsigned)min(lane, g.max_rois - 1)];
    uint32_t* fine = slot_ptr<uint32_t>(L, slot, L.fine);
    for (uint32_t w = blockIdx.x * blockDim.x + threadIdx.x; w < nwords; w += gridDim.x * blockDim.x) fine[w] = 0u;
    // the compaction's look-back states of this reconstruction's chunks, and
    // each chunk's slab: words lo .. hi-1, hi past the farthest neighbour of
    // its words, in whole 16-byte units (the fine array is padded to 256
    // bytes), or 0 when that is more than kSlabWords; with it the ROI of word lo
    const uint32_t nchunks = info->n_chunks, cw = info->chunk_words;
    const int nrois = info->n_rois;
    const DRoi* rois = slot_ptr<DRoi>(L, slot, L.rois);
    unsigned long long* cst = slot_ptr<unsigned long long>(L, slot, L.chunk_st);
    uint32_t* clen = slot_ptr<uint32_t>(L, slot, L.chunk_len);
    for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < nchunks; i += gridDim.x * blockDim.x) {
        cst[2 * (size_t)i] = 0ull;
        cst[2 * (size_t)i + 1] = 0ull;
        const uint32_t lo = i * cw, last = min(lo + cw, nwords) - 1u;
        const int k0 = roi_of_word(rois, nrois, lo), k1 = roi_of_word(rois, nrois, last);
        uint32_t reach = 0;
        for (int k = k0; k <= k1; ++k) {
            const uint32_t rs = (uint32_t)rois[k].nxw;
            reach = max(reach, 1u + rs + rs * (uint32_t)(rois[k].fdim[1] + 2));
        }
        const uint32_t n4 = (min(nwords, last + 1u + reach) - lo + 3u) & ~3u;
        clen[i] = (n4 <= kSlabWords ? n4 : 0u) + (uint32_t)k0 * kChunkRoi;
    }
    if (blockIdx.x == 0 && threadIdx.x == 0) info->next_tile = 0u;
    // Depth boxes: a camera's rows, counted through all its boxes, are dealt out
    // to the warps of its blocks (blocks i, i + cameras, ...; fewer blocks than
    // cameras take several cameras each).  Where the boxes overlap so much that
    // their union's box has fewer pixels, its rows are taken instead.  A warp goes
    // from one of its rows to the next (box by box, each warp walked through all
    // boxes: a frame of 500 ROIs 114 us for this kernel and the hull, now 69).
    const bool many = blocks >= cams.n;
    const int sub = many ? block / cams.n : 0;
    const int subs = many ? (blocks - n0 + cams.n - 1) / cams.n : 1;
    const int nw = subs * bw, me = sub * bw + (int)(threadIdx.x >> 5);
    const int4 none = make_int4(0, -1, 0, -1);
    for (int n = n0; n < cams.n; n += many ? cams.n : blocks) {
        const int W = cams.c[n].W, count = n == n0 ? count0 : counts[n];
        const int4* box = boxes + (size_t)n * (unsigned)g.max_rois;
        uint32_t* D = slot_ptr<uint32_t>(L, slot, L.depth) + cams.c[n].pix_off;
        auto clear = [&](int x0, int x1, int y) {
            uint32_t* row = D + (size_t)y * (unsigned)W;
            for (int x = x0 + lane; x <= x1; x += 32) __stcs(row + x, kEmptyDepth);
        };
        int4 mine = lane < count ? (n == n0 ? first0 : box[lane]) : none;
        int4 u = make_int4(INT_MAX, -1, INT_MAX, -1);
        float area = 0.0f;
        for (int k = lane; k < count; k += 32) {
            const int4 b = k < 32 ? mine : box[k];
            if (b.y < 0) continue;             // none
            area += (float)(b.y - b.x + 1) * (float)(b.w - b.z + 1);
            u = make_int4(min(u.x, b.x), max(u.y, b.y), min(u.z, b.z), max(u.w, b.w));
        }
        for (int o = 16; o > 0; o >>= 1) area += __shfl_xor_sync(kFull, area, o);
        u = make_int4(__reduce_min_sync(kFull, u.x), __reduce_max_sync(kFull, u.y), __reduce_min_sync(kFull, u.z),
                      __reduce_max_sync(kFull, u.w));
        if (u.y < 0) continue;                 // no box
        if (area > (float)(u.y - u.x + 1) * (float)(u.w - u.z + 1)) {
            for (int y = u.z + me; y <= u.w; y += nw) clear(u.x, u.y, y);
            continue;
        }
        int at = me;                           // this warp's next row, counted from the boxes at hand
        for (int k0 = 0;;) {
            int end = mine.w - mine.z + 1;     // rows of the boxes of lanes 0 .. this one
            for (int o = 1; o < 32; o <<= 1) {
                const int e = __shfl_up_sync(kFull, end, o);
                if (lane >= o) end += e;
            }
            const int rows = __shfl_sync(kFull, end, 31);
            for (; at < rows; at += nw) {
                const int k = __ffs(__ballot_sync(kFull, end > at)) - 1;
                clear(__shfl_sync(kFull, mine.x, k), __shfl_sync(kFull, mine.y, k), __shfl_sync(kFull, mine.w + 1 - end, k) + at);
            }
            at -= rows;
            k0 += 32;
            if (k0 >= count) break;
            mine = k0 + lane < count ? box[k0 + lane] : none;
        }
    }
}

// The ROI holding fine-carve tile t: the last ROI whose first tile is <= t.
__device__ __forceinline__ int roi_of_tile(const DRoi* rois, int n, uint32_t t) {
    int lo = 0, hi = n - 1;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (rois[mid].tile_off <= t) lo = mid;
        else hi = mid - 1;
    }
    return lo;
}

// What every sample of a fine-carve tile sees in camera c, one camera per
// lane.  m is the centre of the box of the tile's samples and h its half
// sides.  With u = x'/w' at m, a point m + d of the box lies at
// u + sum (p_0j - u p_2j) d_j / w', so within sum |p_0j - u p_2j| h_j /
// (w'_m - sum |p_2j| h_j) of u (rows alike): one projection bounds the tile
// as tightly as the box of its eight corners' projections does, but for the
// change of w' inside the tile (below 1%), at a third of the instructions.
// The bound is widened by 0.2% and 2^-10 pixels for its own roundings and by
// the camera's error margin (Cam::seg_du, seg_dv; its allowance of 2^-19 |X|
// for a point's deviation covers the half-ulp roundings of m and h) and then
// holds the pixel of every sample.  fg_all: the box is inside the image and every
// pixel of it is set, so every sample votes foreground.  bg_all: no pixel of
// the box inside the image is set and (under STRICT, where a point outside
// the image votes background) the rest lies outside it, or (under ABSTAIN)
// the box is inside the image: every sample votes background.  `inside`: the
// box is inside the image.  A margin also says that every point of the
// volume has w' > 0.
template <bool ABSTAIN>
__device__ __forceinline__ void classify_tile_camera(const SmemCam& c, const uint32_t* __restrict__ sil,
                                                     const float* m, const float* h, bool& fg_all, bool& bg_all,
                                                     bool& inside, uint32_t& reads) {
    fg_all = bg_all = inside = false;
    float xh, yh, wh;
    project(c.P, m[0], m[1], m[2], xh, yh, wh);
    const float ew = __fmaf_rn(fabsf(c.P[8]), h[0], __fmaf_rn(fabsf(c.P[9]), h[1], fmul(fabsf(c.P[10]), h[2])));
    if (!(wh > ew) || !(c.du >= 0.0f)) return;
    const float r = rcp_approx(wh), rw = fmul(rcp_approx(fsub(wh, ew)), 1.002f);
    const float u = fmul(xh, r), v = fmul(yh, r);
    float eu = fmul(fabsf(__fmaf_rn(-u, c.P[10], c.P[2])), h[2]), ev = fmul(fabsf(__fmaf_rn(-v, c.P[10], c.P[6])), h[2]);
    eu = __fmaf_rn(fabsf(__fmaf_rn(-u, c.P[9], c.P[1])), h[1], eu);
    ev = __fmaf_rn(fabsf(__fmaf_rn(-v, c.P[9], c.P[5])), h[1], ev);
    eu = __fmaf_rn(fabsf(__fmaf_rn(-u, c.P[8], c.P[0])), h[0], eu);
    ev = __fmaf_rn(fabsf(__fmaf_rn(-v, c.P[8], c.P[4])), h[0], ev);
    eu = __fmaf_rn(eu, rw, fadd(c.du, 0x1p-10f));
    ev = __fmaf_rn(ev, rw, fadd(c.dv, 0x1p-10f));
    const float u0 = fsub(u, eu), u1 = fadd(u, eu), v0 = fsub(v, ev), v1 = fadd(v, ev);
    if (!(u0 > -1.0e6f && u1 < 1.0e6f && v0 > -1.0e6f && v1 < 1.0e6f)) return;   // also NaN
    // floors: a sum rounded down to kMagic + floor
    auto floor_int = [](float t) { return __float_as_int(__fadd_rd(t, kMagic)) - 0x4B400000; };
    const int bx0 = floor_int(u0), bx1 = floor_int(u1), by0 = floor_int(v0), by1 = floor_int(v1);
    inside = bx0 >= 0 && by0 >= 0 && bx1 < c.W && by1 < c.H;
    // the part of the box inside the image
    const int x0 = max(bx0, 0), x1 = min(bx1, c.W - 1), y0 = max(by0, 0), y1 = min(by1, c.H - 1);
    if (x0 > x1 || y0 > y1) {            // entirely outside the image
        bg_all = !ABSTAIN;
        return;
    }
    if (x1 - x0 > 31 || y1 - y0 > 31) return;   // too large to scan: undecided
    const int w0 = x0 >> 5, dw = (x1 >> 5) - w0;                             // dw: 0 or 1
    uint32_t m0 = ~0u << (x0 & 31), m1 = ~0u >> (31 - (x1 & 31));
    if (dw == 0) {
        m0 &= m1;
        m1 = 0u;
    }
    const uint32_t* row = sil + c.bit_off + (unsigned)y0 * (unsigned)c.Wq + (unsigned)w0;
    uint32_t miss = 0u, hit = 0u;
    for (int y = y0; y <= y1; y += 2) {     // two rows a turn, the last one twice if they are odd in number
        const uint32_t a0 = __ldg(row), a1 = __ldg(row + dw);
        row += y < y1 ? c.Wq : 0;
        const uint32_t b0 = __ldg(row), b1 = __ldg(row + dw);
        row += c.Wq;
        miss |= (~(a0 & b0) & m0) | (~(a1 & b1) & m1);
        hit |= ((a0 | b0) & m0) | ((a1 | b1) & m1);
    }
    reads += (unsigned)((y1 - y0 + 1) * (dw + 1));
    fg_all = inside && miss == 0u;
    bg_all = hit == 0u && (inside || !ABSTAIN);
}

// Sec. II-B-3: the fine hull of every ROI, each treated as its own volume.
// Fine grids are stored padded by one unoccupied sample per side (index 0
// and fdim+1), rows of ceil((fdim_x+2)/32) words, cleared beforehand; only
// occupied samples are written, by OR into their word.
//
// A warp takes 32 / CG tiles of 4 x TY x TZ interior samples (x, y, z) at a
// time, CG lanes each (CG = 8 for up to 8 cameras, else 16), and first
// decides, per camera, whether all of a tile's samples vote foreground or
// all vote background there (classify_tile_camera).  A
// sample's first background camera in index order is then either an
// undecided camera before the tile's first all-background camera, where it
// is tested, or that camera; so each sample projects and looks its pixel up
// only at those undecided cameras, and its test count (first background
// camera + 1, or N when occupied) and occupancy are those of the plain
// per-sample loop.  Tiles whose samples are all decided are counted (and,
// where occupied, written) without walking them; the others are walked by the
// whole warp, one after the other, 4 x 2 x 4 samples at a time, one per lane,
// each camera for the whole tile before the next.
//
// Bound by instruction issue.  Of a court frame's 55,000 tiles (16 cameras)
// 43% end in closed form, and 7.5 of its 28.8 million sample tests are made.
// 64 court frames: 4498 us with two lanes a camera projecting a tile's eight
// corners, one tile a warp, and four sub-tiles walked one after the other;
// 2700 us now.  One frame: 89 -> 71 us.
template <int CG, bool ABSTAIN, int TY, int TZ>
__device__ __forceinline__ void fine_tiles(const Grid& g, const SmemCam* sc, int ncam, uint32_t ntiles, int nrois,
                                           const DRoi* rois, const uint32_t* __restrict__ sil, uint32_t* fine,
                                           uint32_t* next_tile, uint32_t claim, unsigned long long& tests,
                                           uint32_t& reads) {
    constexpr int kSubsY = TY / kSubY, kSubs = kSubsY * (TZ / kSubZ);
    constexpr uint64_t kGroup = (1ull << CG) - 1ull;
    const int lane = threadIdx.x & 31, own = lane % CG;
    const int xi = lane & 3, yi = (lane >> 2) & 1, zi = lane >> 3;
    // the ROI of this lane's tile
    uint32_t lo = 0, hi = 0, woff = 0;
    int fx = 1, fy = 1, fz = 1, nxw = 1, ntx = 1, nty = 1;
    float fo0 = 0.f, fo1 = 0.f, fo2 = 0.f;
    // Tiles differ a lot in cost (a surface tile tests many cameras, an empty
    // one few), so the warps claim them from a counter.  Claims are small and
    // of neighbouring tiles: costly tiles lie together (one warp would work a
    // long claim of them off alone), and the tiles in work at a time then
    // read the same silhouette rows.
    uint32_t t0 = 0;
    if (lane == 0) t0 = atomicAdd(next_tile, claim);
    t0 = __shfl_sync(kFull, t0, 0);
    while (t0 < ntiles) {
        const bool mine = (uint32_t)(lane / CG) < claim && t0 + (uint32_t)(lane / CG) < ntiles;
        const uint32_t t = t0 + (mine ? (uint32_t)(lane / CG) : 0u);
        if (t >= hi || t < lo) {
            const DRoi& r = rois[roi_of_tile(rois, nrois, t)];
            lo = r.tile_off;
            fx = r.fdim[0];
            fy = r.fdim[1];
            fz = r.fdim[2];
            ntx = (fx + kTileX - 1) / kTileX;
            nty = (fy + TY - 1) / TY;
            hi = lo + (uint32_t)ntx * (uint32_t)nty * (uint32_t)((fz + TZ - 1) / TZ);
            woff = r.word_off;
            nxw = r.nxw;
            fo0 = r.fo[0];
            fo1 = r.fo[1];
            fo2 = r.fo[2];
        }
        const uint32_t lt = t - lo;
        const uint32_t r1 = lt / (uint32_t)ntx;
        const int tz = (int)(r1 / (uint32_t)nty);
        const int x0 = (int)(lt - r1 * (uint32_t)ntx) * kTileX, y0 = (int)(r1 - (uint32_t)tz * (uint32_t)nty) * TY,
                  z0 = tz * TZ;
        // bit n: every sample votes foreground (fgm) / background (bgm) in camera n;
        // inm: the tile's box is inside camera n's image
        uint64_t fgm = 0, bgm = 0, inm = 0;
        {
            const float a0 = fadd(fo0, fmul(fadd((float)x0, 0.5f), g.sf));
            const float a1 = fadd(fo1, fmul(fadd((float)y0, 0.5f), g.sf));
            const float a2 = fadd(fo2, fmul(fadd((float)z0, 0.5f), g.sf));
            const float b0 = fadd(fo0, fmul(fadd((float)min(x0 + kTileX - 1, fx - 1), 0.5f), g.sf));
            const float b1 = fadd(fo1, fmul(fadd((float)min(y0 + TY - 1, fy - 1), 0.5f), g.sf));
            const float b2 = fadd(fo2, fmul(fadd((float)min(z0 + TZ - 1, fz - 1), 0.5f), g.sf));
            const float m[3] = {fmul(fadd(a0, b0), 0.5f), fmul(fadd(a1, b1), 0.5f), fmul(fadd(a2, b2), 0.5f)};
            const float h[3] = {fmul(fsub(b0, a0), 0.5f), fmul(fsub(b1, a1), 0.5f), fmul(fsub(b2, a2), 0.5f)};
            for (int cg = 0; cg < ncam; cg += CG) {
                const int cam = cg + own;
                bool fg = false, bg = false, in = false;
                uint32_t rd = 0;
                if (mine && cam < ncam) classify_tile_camera<ABSTAIN>(sc[cam], sil, m, h, fg, bg, in, rd);
                reads += rd;
                const int sh = lane & ~(CG - 1);
                fgm |= ((uint64_t)(__ballot_sync(kFull, fg) >> sh) & kGroup) << cg;
                bgm |= ((uint64_t)(__ballot_sync(kFull, bg) >> sh) & kGroup) << cg;
                inm |= ((uint64_t)(__ballot_sync(kFull, in) >> sh) & kGroup) << cg;
            }
        }
        const int nb = bgm ? __ffsll((long long)bgm) - 1 : ncam;
        const uint64_t before = nb >= 64 ? ~0ull : (1ull << nb) - 1ull;
        const uint64_t undecided = ~(fgm | bgm) & before;
        // every camera before nb sees the whole tile as foreground: its
        // samples stop at camera nb (nb + 1 tests), or are all occupied
        if (mine && own == 0 && undecided == 0ull)
            tests += (unsigned)(min(kTileX, fx - x0) * min(TY, fy - y0) * min(TZ, fz - z0)) *
                     (unsigned)(nb < ncam ? nb + 1 : ncam);
        // tiles left: those with undecided cameras, and the occupied ones to write
        uint32_t todo_tiles = __ballot_sync(kFull, mine && own == 0 && (undecided != 0ull || nb >= ncam));
        while (todo_tiles) {
            const int src = __ffs(todo_tiles) - 1;
            todo_tiles &= todo_tiles - 1u;
            uint64_t todo = __shfl_sync(kFull, undecided, src);
            const int tnb = __shfl_sync(kFull, nb, src);
            const int tx0 = __shfl_sync(kFull, x0, src), ty0 = __shfl_sync(kFull, y0, src),
                      tz0 = __shfl_sync(kFull, z0, src);
            const int tfx = __shfl_sync(kFull, fx, src), tfy = __shfl_sync(kFull, fy, src),
                      tfz = __shfl_sync(kFull, fz, src);
            // this lane's samples: bit s of `act` for sub-tile s
            uint32_t act = 0u;
#pragma unroll
            for (int s = 0; s < kSubs; ++s) {
                const int y = ty0 + (s % kSubsY) * kSubY + yi, z = tz0 + (s / kSubsY) * kSubZ + zi;
                if (tx0 + xi < tfx && y < tfy && z < tfz) act |= 1u << s;
            }
            uint32_t alive = act;
            if (todo) {
                const uint64_t tin = __shfl_sync(kFull, inm, src), tfg = __shfl_sync(kFull, fgm, src);
                const float tf0 = __shfl_sync(kFull, fo0, src), tf1 = __shfl_sync(kFull, fo1, src),
                            tf2 = __shfl_sync(kFull, fo2, src);
                const float X = fadd(tf0, fmul(fadd((float)(tx0 + xi), 0.5f), g.sf));
                float Y[kSubsY], Z[kSubs / kSubsY];
#pragma unroll
                for (int e = 0; e < kSubsY; ++e)
                    Y[e] = fadd(tf1, fmul(fadd((float)(ty0 + e * kSubY + yi), 0.5f), g.sf));
#pragma unroll
                for (int e = 0; e < kSubs / kSubsY; ++e)
                    Z[e] = fadd(tf2, fmul(fadd((float)(tz0 + e * kSubZ + zi), 0.5f), g.sf));
                const uint64_t tbefore = tnb >= 64 ? ~0ull : (1ull << tnb) - 1ull;
                uint32_t voted = (!ABSTAIN || (tfg & tbefore) != 0ull) ? ~0u : 0u;
                // In camera order: the first all-background camera tnb stops
                // every sample still alive there; before it, all-foreground
                // cameras pass every sample and only the undecided ones are
                // tested, per lane.
                while (todo && __any_sync(kFull, alive != 0u)) {
                    const int n = __ffsll((long long)todo) - 1;
                    todo &= todo - 1ull;
                    const SmemCam& c = sc[n];
                    if ((tin >> n) & 1ull) {
#pragma unroll
                        for (int s = 0; s < kSubs; ++s) {
                            if ((alive >> s) & 1u) {
                                const uint32_t bit = cam_bit_inside(c, sil, X, Y[s % kSubsY], Z[s / kSubsY], true);
                                ++reads;
                                if (!bit) {
                                    alive &= ~(1u << s);
                                    tests += (unsigned)(n + 1);
                                }
                                if (ABSTAIN) voted |= bit << s;
                            }
                        }
                    } else {
#pragma unroll 1
                        for (int s = 0; s < kSubs; ++s) {
                            if ((alive >> s) & 1u) {
                                bool in;
                                const float Ys = fadd(tf1, fmul(fadd((float)(ty0 + (s % kSubsY) * kSubY + yi), 0.5f), g.sf));
                                const float Zs = fadd(tf2, fmul(fadd((float)(tz0 + (s / kSubsY) * kSubZ + zi), 0.5f), g.sf));
                                const uint32_t bit = cam_bit(c, sil, X, Ys, Zs, in);
                                reads += in ? 1u : 0u;
                                if (ABSTAIN ? (in && !bit) : !bit) {
                                    alive &= ~(1u << s);
                                    tests += (unsigned)(n + 1);
                                }
                                if (ABSTAIN) voted |= bit << s;
                            }
                        }
                    }
                }
                tests += (unsigned)__popc(alive) * (unsigned)(tnb < ncam ? tnb + 1 : ncam);
                alive = tnb >= ncam ? alive & voted : 0u;
            }
            // OR the occupied samples into their words: the four lanes of one
            // (y, z) row, a nibble of a sub-tile's ballot, span at most two
            // words; lane l writes row l of the tile's kSubs * 8 rows
            if (__any_sync(kFull, alive != 0u)) {
                const uint32_t tw = __shfl_sync(kFull, woff, src);
                const int tn = __shfl_sync(kFull, nxw, src);
#pragma unroll
                for (int r0 = 0; r0 < kSubs * 8; r0 += 32) {
                    uint32_t bal = 0u;
#pragma unroll
                    for (int s = r0 / 8; s < min(kSubs, r0 / 8 + 4); ++s) {
                        const uint32_t b = __ballot_sync(kFull, (alive >> s) & 1u);
                        if ((lane >> 3) == s - r0 / 8) bal = b;
                    }
                    const int row = r0 + lane;               // sub-tile row / 8, its row row % 8: (zi, yi)
                    const uint32_t nib = row < kSubs * 8 ? (bal >> (4 * (row & 7))) & 15u : 0u;
                    if (nib) {
                        const int s = row >> 3;
                        const int y = ty0 + (s % kSubsY) * kSubY + (row & 1), z = tz0 + (s / kSubsY) * kSubZ + ((row >> 1) & 3);
                        const uint32_t word = tw + ((uint32_t)(z + 1) * (uint32_t)(tfy + 2) + (uint32_t)(y + 1)) * (uint32_t)tn +
                                              (uint32_t)((tx0 + 1) >> 5);
                        const int p = (tx0 + 1) & 31;        // 1, 5, ..., 29
                        atomicOr(fine + word, nib << p);
                        if (p == 29 && (nib >> 3)) atomicOr(fine + word + 1, 1u);
                    }
                }
            }
        }
        if (lane == 0) t0 = atomicAdd(next_tile, claim);
        t0 = __shfl_sync(kFull, t0, 0);
    }
}

template <int CG, int TY, int TZ>
__global__ void __launch_bounds__(256) k_fine_carve(const __grid_constant__ CamSet cams,
                                                    const __grid_constant__ Grid g,
                                                    const __grid_constant__ Layout L,
                                                    const __grid_constant__ SlotList sl, uint32_t resident) {
    pdl_begin();
    __shared__ unsigned long long sh_t[32];
    __shared__ SmemCam sc[FVV_MAX_CAMS];
    const int slot = sl.s[blockIdx.y];
    const SlotInfo* info = slot_ptr<SlotInfo>(L, slot, L.info);
    const uint32_t ntiles = info->n_words ? info->n_tiles : 0u;
    // a block that comes too late for any tile leaves at once
    if (__syncthreads_and(__ldcg(&info->next_tile) >= ntiles)) return;
    load_smem_cams(cams, cams.n, sc);
    __syncthreads();
    const int nrois = info->n_rois;
    const DRoi* rois = slot_ptr<DRoi>(L, slot, L.rois);
    const uint32_t* __restrict__ sil = slot_ptr<uint32_t>(L, slot, L.sil);
    uint32_t* fine = slot_ptr<uint32_t>(L, slot, L.fine);
    uint32_t* next_tile = &slot_ptr<SlotInfo>(L, slot, L.info)->next_tile;
    // Tiles a warp takes at a time: one for each of its lane groups, but at
    // least two claims for every warp that can be resident (`resident`).  One
    // counter serves about one claim a nanosecond: a court frame's 55,000 tiles
    // took 80 us claimed one by one, 70 two by two, and 95 in claims of 5 or
    // with the first claims dealt out.
    const uint32_t nwarps = min((gridDim.x * blockDim.x) >> 5, resident);
    const uint32_t claim = max(1u, min(32u / CG, ntiles / (2u * nwarps)));
    unsigned long long tests = 0;
    uint32_t reads = 0;
    if (cams.oob == FVV_OOB_ABSTAIN)
        fine_tiles<CG, true, TY, TZ>(g, sc, cams.n, ntiles, nrois, rois, sil, fine, next_tile, claim, tests,
                                       reads);
    else
        fine_tiles<CG, false, TY, TZ>(g, sc, cams.n, ntiles, nrois, rois, sil, fine, next_tile, claim, tests,
                                       reads);
    const unsigned long long t = block_sum<unsigned long long>(tests, sh_t);
    const unsigned long long rd = block_sum<unsigned long long>((unsigned long long)reads, sh_t);
    if (threadIdx.x == 0 && t) atomicAdd(&slot_ptr<SlotInfo>(L, slot, L.info)->tests_fine, t);
    if (threadIdx.x == 0 && rd) atomicAdd(&slot_ptr<SlotInfo>(L, slot, L.info)->look_fine, rd);
}

// Test hook: the pixel each point falls in for one camera (-1, -1 if none).
__global__ void k_debug_pixels(const __grid_constant__ CamSet cams, int cam, long long n,
                               const float* __restrict__ pts, int32_t* px, int32_t* py) {
    const Cam& c = cams.c[cam];
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
        int u, v;
        cam_pixel(c, pts[3 * i], pts[3 * i + 1], pts[3 * i + 2], u, v);
        px[i] = u;
        py[i] = v;
    }
}

}  // namespace

cudaError_t launch_debug_pixels(const CamSet& cams, int cam, long long n, const float* pts, int32_t* px,
                                int32_t* py, cudaStream_t st) {
    const unsigned g = (unsigned)std::min<long long>((n + 255) / 256, 8192);
    k_debug_pixels<<<g, 256, 0, st>>>(cams, cam, n, pts, px, py);
    return cudaGetLastError();
}

cudaError_t launch_pack(const CamSet& cams, const Layout& L, int n_frames, const int* slots,
                        const uint8_t* const* src, bool host_src, int sms, cudaStream_t st) {
    size_t max_words = 0;
    for (int n = 0; n < cams.n; ++n)
        max_words = std::max(max_words, (size_t)((cams.c[n].H + 3) / 4) * (unsigned)cams.c[n].Wq);   // a thread per 4 rows
    const int per_launch = std::min(kPackPtrs / 4, kPackPtrs / std::max(1, cams.n));
    // Device sources: enough blocks to stream HBM at full rate.  Masks read in
    // place from host memory are bound by the host link, which some megabyte
    // of loads in flight keeps busy (128 bytes a thread); more of them only
    // wait longer, and hold up the other streams' work.  Blocks of 32 threads,
    // three per SM in all, a block per image at least: 48 court frames 168 GB/s
    // with 256 threads, 195 with 32; 20 judo frames 190 and 202; four rigs
    // served at saturation 2200 frames/s with 256 threads, 2370 with 128, 2580
    // with 64 and 2760 with 32 (eight such blocks per SM: 2460; two: 2820, but 20
    // 720p frames 165 GB/s instead of 183).  With the link to itself a call on large
    // masks takes up to 3% longer than by two blocks of 256 per SM (twelve 4K masks
    // 482 -> 497 us).
    const size_t cap = host_src ? (size_t)std::max(1, 3 * sms / std::max(1, cams.n * std::min(n_frames, per_launch)))
                                : (size_t)2048;
    const unsigned th = host_src ? 32 : 256;
    const unsigned gx = (unsigned)std::max<size_t>(1, std::min<size_t>((max_words + th - 1) / th, cap));
    static_assert(sizeof(CamSet) + sizeof(PackSrc) + sizeof(Layout) <= 32764, "k_pack parameters");
    thread_local PackSrc a;   // 18 KB: kept off the stack
    for (int j0 = 0; j0 < n_frames; j0 += per_launch) {
        const int nf = std::min(per_launch, n_frames - j0);
        for (int j = 0; j < nf; ++j) {
            a.slot[j] = slots[j0 + j];
            for (int n = 0; n < cams.n; ++n) a.src[j * cams.n + n] = src[(size_t)(j0 + j) * cams.n + n];
        }
        const cudaError_t e = launch_pdl(k_pack, dim3(gx, cams.n, nf), dim3(th), 0, st, cams, a, L);
        if (e != cudaSuccess) return e;
    }
    return cudaGetLastError();
}

cudaError_t launch_coarse_table(const CamSet& cams, const Grid& g, uint32_t* e, int n, cudaStream_t st) {
    const size_t nvox = (size_t)g.nx * g.ny * g.nz;
    k_coarse_table<<<(unsigned)std::min<size_t>((nvox + 255) / 256, 16384), 256, 0, st>>>(cams, g, e, n);
    return cudaGetLastError();
}

namespace {
__global__ void k_reset_coarse(const __grid_constant__ Layout L, const __grid_constant__ SlotList sl) {
    pdl_begin();
    if (threadIdx.x == 0) slot_ptr<SlotInfo>(L, sl.s[blockIdx.x], L.info)->n_front = 0u;
}
}  // namespace

cudaError_t launch_reset_coarse(const Layout& L, const SlotList& sl, cudaStream_t st) {
    return launch_pdl(k_reset_coarse, dim3(sl.n), dim3(32), 0, st, L, sl);
}

cudaError_t launch_coarse_carve(const CamSet& cams, const Grid& g, const Layout& L, const SlotList& sl,
                                const CoarseTable& tab, int sms, const Tuning& tu, cudaStream_t st) {
    const int th = tu.threads[FVV_TUNE_COARSE];
    const long long words = (long long)g.nz * g.ny * g.nxw;
    const int g1 = tuned_grid(tu, FVV_TUNE_COARSE, sms, sl.n, (words + kWords - 1) / kWords * 32);
    const int g2 = tuned_grid(tu, FVV_TUNE_COARSE, sms, sl.n, words * 32);
    // Cameras of the first pass: three where the launch is too small to hide the
    // second pass's chains of loads (one court frame, 229,000 words: 46 us with one
    // camera, 34 with three; two, 458,000: 67 and 57), else one (64 frames: 988 and
    // 1085).  Where the two cross depends on the rig: below 0.8 million words for
    // one 4K court frame of abstaining cameras (81 and 89 us, twice that 133 and
    // 159), at 0.9 for 720p frames (640,000: 62.5 and 61; 960,000: 83 and 85), above
    // 1.8 for court frames (1.8 million: 168 and 165), so the line lies below the
    // first, and the others lose a tenth at most (three court frames: 84 and 76).
    const int levels = std::min(tab.n, words * sl.n < 600000 ? 3 : 1);
#define FVV_LAUNCH(A, M) launch_pdl(k_coarse_first<A, M>, dim3(g1, sl.n), dim3(th), 0, st, cams, g, L, sl, tab, levels)
    if (cams.oob == FVV_OOB_ABSTAIN) {
        if (levels > 1) FVV_LAUNCH(true, true);
        else FVV_LAUNCH(true, false);
        launch_pdl(k_coarse_rest<true>, dim3(g2, sl.n), dim3(th), 0, st, cams, g, L, sl, tab, levels);
    } else {
        if (levels > 1) FVV_LAUNCH(false, true);
        else FVV_LAUNCH(false, false);
        launch_pdl(k_coarse_rest<false>, dim3(g2, sl.n), dim3(th), 0, st, cams, g, L, sl, tab, levels);
    }
#undef FVV_LAUNCH
    return cudaGetLastError();
}

cudaError_t launch_fine_carve(const CamSet& cams, const Grid& g, const Layout& L, const SlotList& sl, int sms,
                              const Tuning& tu, cudaStream_t st) {
    long long rows = 0;
    for (int n = 0; n < cams.n; ++n) rows += cams.c[n].H;
    const int gc = clear_blocks(sms, sl.n, g.max_fine_words, rows);
    launch_pdl(k_clear_fine, dim3(gc, sl.n), dim3(256), 0, st, cams, g, L, sl);
    const int th = tu.threads[FVV_TUNE_FINE];
    const int gx = fine_blocks(tu, sms, sl.n, g.max_fine_words);
    // the tile shape (tile_y, tile_z) the k_filter of this sequence counted tiles with
    const uint32_t resident = (uint32_t)sms * 32u;   // 1024 threads per SM at the kernel's 64 registers
#define FVV_LAUNCH(CG, TY, TZ) \
    launch_pdl(k_fine_carve<CG, TY, TZ>, dim3(gx, sl.n), dim3(th), 0, st, cams, g, L, sl, resident)
#define FVV_LAUNCH_CG(TY, TZ)                       \
    if (cams.n <= 8) FVV_LAUNCH(8, TY, TZ);         \
    else FVV_LAUNCH(16, TY, TZ)
    if (g.tile_y == 4 && g.tile_z == 4) {
        FVV_LAUNCH_CG(4, 4);
    } else if (g.tile_y == 8 && g.tile_z == 8) {
        FVV_LAUNCH_CG(8, 8);
    } else {
        FVV_LAUNCH_CG(4, 8);
    }
#undef FVV_LAUNCH_CG
#undef FVV_LAUNCH
    return cudaGetLastError();
}

}  // namespace fvv
