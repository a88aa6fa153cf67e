// kernels_mc.cu -- Sec. II-C: surface polygonisation of every fine grid.
//
// Each fine grid is padded by one unoccupied sample per side and stored as
// rows of 32-bit words, so one thread owns 32 cells (or 32 samples) and works
// with word-wide bit operations:
//   compact   bipolar-edge masks (x: w ^ w>>1, y: w ^ w(y+1), z: w ^ w(z+1)),
//             vertices = popcounts, triangles = table counts of mixed cells;
//             exclusive prefix per word (sums over the block + a look-back
//             over the earlier chunks, of 256 to 1024 words) and one record per
//             bipolar edge, in edge-key order (3*Lpad + axis), and one per triangle; the
//             grid slab a chunk reads is staged in shared memory by a bulk
//             copy.
//   bisect    one thread per vertex: fixed-count bisection of its edge
//             against the silhouettes (the exact intersection of Eqs. (2)-(3)
//             read as the hull crossing on the edge).
//   triangles table triangles of each mixed cell, vertex ids = word prefix +
//             rank of the edge inside its word.
// Vertex and triangle order is therefore (ROI, key) and (ROI, cell, table
// order): independent of scheduling, identical to a serial scan.
#include <atomic>

#include "fvv_device.cuh"

namespace fvv {

// ------------------------------------------------------------ MC table (host)
//
// Corners are numbered x + 2y + 4z.  Cube edge e runs along axis e/4 from its
// lower corner, whose other two coordinates, in increasing axis order, are
// (e & 1, e >> 1 & 1).  On every face the bipolar edges are joined by
// segments (two bipolar edges: one segment; four, i.e. two diagonal ON
// corners: one segment around each ON corner, keeping ON corners apart), each
// directed so that the ON side is on its right seen from outside the cube;
// chaining them gives loops whose normals point from ON to OFF.  Loops are
// taken in order of their smallest edge, walked from it, and fanned from the
// first vertex that shares no face with a vertex it is not adjacent to.
namespace {

void edge_ends(int e, int& lo, int& hi) {
    const int axis = e >> 2;
    int other[2], k = 0;
    for (int b = 0; b < 3; ++b)
        if (b != axis) other[k++] = b;
    lo = ((e & 1) << other[0]) | (((e >> 1) & 1) << other[1]);
    hi = lo | (1 << axis);
}

int edge_of(int c0, int c1) {
    for (int e = 0; e < 12; ++e) {
        int lo, hi;
        edge_ends(e, lo, hi);
        if ((lo == c0 && hi == c1) || (lo == c1 && hi == c0)) return e;
    }
    return -1;
}

}  // namespace

void build_mc_table(uint8_t ntri[256], uint8_t edges[256 * kMaxTriPerCell * 3]) {
    // face membership of every edge, and each face's corner cycle
    int face_mask[12] = {0};
    int cyc[6][4];
    for (int f = 0; f < 6; ++f) {
        const int b = f >> 1, t = f & 1;
        const int p = b == 0 ? 1 : 0, q = b == 2 ? 1 : 2;
        const int uv[4][2] = {{0, 0}, {1, 0}, {1, 1}, {0, 1}};
        for (int i = 0; i < 4; ++i) cyc[f][i] = (t << b) | (uv[i][0] << p) | (uv[i][1] << q);
        for (int i = 0; i < 4; ++i) face_mask[edge_of(cyc[f][i], cyc[f][(i + 1) & 3])] |= 1 << f;
    }
    for (int cs = 0; cs < 256; ++cs) {
        int nxt[12];
        for (int e = 0; e < 12; ++e) nxt[e] = -1;
        for (int f = 0; f < 6; ++f) {
            const int b = f >> 1, t = f & 1;
            const int hand = b == 1 ? -1 : 1;       // (p, q, b) right-handed?
            const int side = t ? 1 : -1;            // outward normal along b
            const int uv[4][2] = {{0, 0}, {1, 0}, {1, 1}, {0, 1}};
            int s[4], fe[4], nb = 0;
            for (int i = 0; i < 4; ++i) s[i] = (cs >> cyc[f][i]) & 1;
            for (int i = 0; i < 4; ++i)
                if (s[i] != s[(i + 1) & 3]) fe[nb++] = i;  // face edge i joins corners i, i+1
            int seg[2][3], ns = 0;                          // (face edge, face edge, ON corner)
            if (nb == 2) {
                int on = 0;
                while (!s[on]) ++on;
                seg[0][0] = fe[0]; seg[0][1] = fe[1]; seg[0][2] = on;
                ns = 1;
            } else if (nb == 4) {
                for (int i = 0; i < 4; ++i)
                    if (s[i]) {
                        seg[ns][0] = (i + 3) & 3; seg[ns][1] = i; seg[ns][2] = i;
                        ++ns;
                    }
            }
            for (int k = 0; k < ns; ++k) {
                const int i0 = seg[k][0], i1 = seg[k][1], a = seg[k][2];
                // doubled face-plane coordinates of the two midpoints and the ON corner
                const int P[2] = {uv[i0][0] + uv[(i0 + 1) & 3][0], uv[i0][1] + uv[(i0 + 1) & 3][1]};
                const int Q[2] = {uv[i1][0] + uv[(i1 + 1) & 3][0], uv[i1][1] + uv[(i1 + 1) & 3][1]};
                const int A[2] = {2 * uv[a][0], 2 * uv[a][1]};
                const int cr = (Q[0] - P[0]) * (A[1] - P[1]) - (Q[1] - P[1]) * (A[0] - P[0]);
                const int ep = edge_of(cyc[f][i0], cyc[f][(i0 + 1) & 3]);
                const int eq = edge_of(cyc[f][i1], cyc[f][(i1 + 1) & 3]);
                if (cr * hand * side < 0) nxt[ep] = eq;
                else nxt[eq] = ep;
            }
        }
        int done = 0, nt = 0;
        for (int e0 = 0; e0 < 12; ++e0) {
            if (nxt[e0] < 0 || (done >> e0 & 1)) continue;
            int loop[12], n = 0;
            for (int e = e0; !(done >> e & 1); e = nxt[e]) {
                done |= 1 << e;
                loop[n++] = e;
            }
            int apex = 0;
            for (int i = 0; i < n; ++i) {
                bool ok = true;
                for (int d = 2; d + 1 < n && ok; ++d)
                    if (face_mask[loop[i]] & face_mask[loop[(i + d) % n]]) ok = false;
                if (ok) {
                    apex = i;
                    break;
                }
            }
            for (int d = 1; d + 1 < n; ++d) {
                uint8_t* o = edges + ((size_t)cs * kMaxTriPerCell + nt) * 3;
                o[0] = (uint8_t)loop[apex];
                o[1] = (uint8_t)loop[(apex + d) % n];
                o[2] = (uint8_t)loop[(apex + d + 1) % n];
                ++nt;
            }
        }
        ntri[cs] = (uint8_t)nt;
    }
}

// ------------------------------------------------------------------ kernels
namespace {

// The 8 words around fine word w (rows y, y+1 and planes z, z+1; this word
// and the next in x) as "samples at xp" (c*) and "samples at xp+1" (s*),
// indexed by corner bits (dy + 2dz).
struct Nbhd {
    uint32_t w[4];   // sample xp, corner dy + 2 dz
    uint32_t s[4];   // sample xp + 1
};

__device__ __forceinline__ void load_nbhd(const uint32_t* fine, const RoiCursor& r, uint32_t w, Nbhd& n) {
    const uint32_t rs = (uint32_t)r.nxw, ps = (uint32_t)r.nxw * (uint32_t)(r.fdim[1] + 2);
    const bool hx = r.wx + 1 < r.nxw, hy = r.yp + 1 < r.fdim[1] + 2, hz = r.zp + 1 < r.fdim[2] + 2;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        const bool dy = k & 1, dz = k >> 1;
        const bool ok = (!dy || hy) && (!dz || hz);
        const uint32_t base = w + (dy ? rs : 0u) + (dz ? ps : 0u);
        const uint32_t a = ok ? __ldg(fine + base) : 0u;
        const uint32_t b = (ok && hx) ? __ldg(fine + base + 1) : 0u;
        n.w[k] = a;
        n.s[k] = (a >> 1) | (b << 31);
    }
}

__device__ __forceinline__ uint32_t mixed_cells(const Nbhd& n) {
    const uint32_t a = n.w[0];
    return (a ^ n.s[0]) | (a ^ n.w[1]) | (a ^ n.s[1]) | (a ^ n.w[2]) | (a ^ n.s[2]) | (a ^ n.w[3]) | (a ^ n.s[3]);
}

// The cases of all 32 cells of a word (bit 2k: w[k], bit 2k + 1: s[k]), a byte
// each, cell b's in byte b % 4 of out[b / 4 * kChunk]: four 8 x 8 bit
// transposes by swaps of bits, pairs and nibbles, some 100 instructions for
// what costs 24 a cell when its bits are picked out of the eight words.
__device__ __forceinline__ void cell_cases(const Nbhd& n, uint32_t* out) {
    uint32_t lo[4], hi[4];   // [g]: byte g of w0 s0 w1 s1, and of w2 s2 w3 s3
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        const uint32_t a = n.w[2 * h], b = n.s[2 * h], c = n.w[2 * h + 1], d = n.s[2 * h + 1];
        const uint32_t ab = __byte_perm(a, b, 0x5140), ab2 = __byte_perm(a, b, 0x7362);
        const uint32_t cd = __byte_perm(c, d, 0x5140), cd2 = __byte_perm(c, d, 0x7362);
        uint32_t* o = h ? hi : lo;
        o[0] = __byte_perm(ab, cd, 0x5410);
        o[1] = __byte_perm(ab, cd, 0x7632);
        o[2] = __byte_perm(ab2, cd2, 0x5410);
        o[3] = __byte_perm(ab2, cd2, 0x7632);
    }
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        uint32_t x = lo[q], y = hi[q], t;
        t = (x ^ (x >> 7)) & 0x00AA00AAu;
        x ^= t ^ (t << 7);
        t = (y ^ (y >> 7)) & 0x00AA00AAu;
        y ^= t ^ (t << 7);
        t = (x ^ (x >> 14)) & 0x0000CCCCu;
        x ^= t ^ (t << 14);
        t = (y ^ (y >> 14)) & 0x0000CCCCu;
        y ^= t ^ (t << 14);
        t = (x ^ (y << 4)) & 0xF0F0F0F0u;
        out[2 * q * kChunk] = x ^ t;
        out[(2 * q + 1) * kChunk] = y ^ (t >> 4);
    }
}

// The 8 words of load_nbhd, read from a slab of the slot's fine words
// staged in shared memory (slab[i] = fine word lo + i).
__device__ __forceinline__ void load_nbhd_slab(const uint32_t* slab, uint32_t lo, const RoiCursor& r, uint32_t w,
                                               Nbhd& n) {
    const uint32_t rs = (uint32_t)r.nxw, ps = (uint32_t)r.nxw * (uint32_t)(r.fdim[1] + 2);
    const bool hx = r.wx + 1 < r.nxw, hy = r.yp + 1 < r.fdim[1] + 2, hz = r.zp + 1 < r.fdim[2] + 2;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        const bool dy = k & 1, dz = k >> 1;
        const bool ok = (!dy || hy) && (!dz || hz);
        const uint32_t i = w - lo + (dy ? rs : 0u) + (dz ? ps : 0u);
        const uint32_t a = ok ? slab[i] : 0u;
        const uint32_t b = (ok && hx) ? slab[i + 1] : 0u;
        n.w[k] = a;
        n.s[k] = (a >> 1) | (b << 31);
    }
}

// ---- staging through the tensor memory accelerator (1-D bulk copies into
// shared memory, completion counted on an mbarrier)
__device__ __forceinline__ uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ void mbar_init(uint64_t* bar) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_u32(bar)) : "memory");
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}

// One arrival that also expects `bytes` of copies to complete on the barrier.
__device__ __forceinline__ void mbar_expect_tx(uint64_t* bar, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes)
                 : "memory");
}

__device__ __forceinline__ bool mbar_try_wait(uint64_t* bar, uint32_t parity) {
    uint32_t done;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(done)
        : "r"(smem_u32(bar)), "r"(parity)
        : "memory");
    return done != 0u;
}

// Copy `bytes` (a multiple of 16; both addresses 16-byte aligned) from
// global to shared memory; completes on `bar`.  Shared memory that generic
// loads read before must be ordered before the copy (fence_proxy_async).
__device__ __forceinline__ void bulk_copy_g2s(void* dst, const void* src, uint32_t bytes, uint64_t* bar) {
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
                     smem_u32(dst)),
                 "l"(src), "r"(bytes), "r"(smem_u32(bar))
                 : "memory");
}

__device__ __forceinline__ void fence_proxy_async() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }

// Decoupled look-back state of a chunk, one word per count (vertices,
// triangles): bits 62-63 say what bits 0-61 hold -- 0 nothing yet, 1 the
// chunk's own count, 2 the count of chunks 0..c together.
constexpr unsigned long long kStAgg = 1ull << 62, kStInc = 2ull << 62, kStVal = (1ull << 62) - 1ull;

__device__ __forceinline__ void st_state(unsigned long long* p, unsigned long long v) {
    asm volatile("st.relaxed.gpu.global.b64 [%0], %1;" ::"l"(p), "l"(v) : "memory");
}

__device__ __forceinline__ unsigned long long ld_state(const unsigned long long* p) {
    unsigned long long v;
    asm volatile("ld.relaxed.gpu.global.b64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
    return v;
}

// Polls of a bounded wait (the slab copy, or the states of earlier chunks)
// before the kernel gives up on it and sets FVV_FLAG_LOOP.
constexpr int kMaxPolls = 1 << 22;

// Counts (vertices, triangles) of the chunks before chunk c, by warp 0: the
// lanes read the states of 32 earlier chunks at a time (lane i: chunk
// top - i), wait until all 32 are published, and add the values from the
// nearest chunk back to the first inclusive one; without an inclusive one
// in the window, all 32 and the window before.  False if the polls ran out.
__device__ __forceinline__ bool look_back_warp(const unsigned long long* st, uint32_t c, unsigned long long& sv,
                                               unsigned long long& stt) {
    const int lane = threadIdx.x & 31;
    sv = stt = 0;
    bool need_v = true, need_t = true;
    int polls = 0;
    for (long long top = (long long)c - 1; top >= 0 && (need_v || need_t);) {
        const long long q = top - lane;
        // chunks before chunk 0 read as an inclusive zero, which ends the walk
        const unsigned long long a = q >= 0 ? ld_state(st + 2 * q) : kStInc;
        const unsigned long long b = q >= 0 ? ld_state(st + 2 * q + 1) : kStInc;
        if (__any_sync(kFull, (a >> 62) == 0ull || (b >> 62) == 0ull)) {
            if (++polls > kMaxPolls) return false;
            continue;
        }
        const unsigned iv = __ballot_sync(kFull, (a >> 62) == 2ull), it = __ballot_sync(kFull, (b >> 62) == 2ull);
        const int lv = iv ? __ffs(iv) - 1 : 31, lt = it ? __ffs(it) - 1 : 31;
        unsigned long long xv = (need_v && lane <= lv) ? (a & kStVal) : 0ull;
        unsigned long long xt = (need_t && lane <= lt) ? (b & kStVal) : 0ull;
        for (int o = 16; o > 0; o >>= 1) {
            xv += __shfl_xor_sync(kFull, xv, o);
            xt += __shfl_xor_sync(kFull, xt, o);
        }
        sv += xv;
        stt += xt;
        need_v = need_v && !iv;
        need_t = need_t && !it;
        top -= 32;
    }
    return true;
}

// Vertex record: ROI (14 bits) | axis (2) | ON at lower sample (1) | xp, yp, zp (15 bits each).
__device__ __forceinline__ uint64_t pack_vrec(int k, int axis, int s0on, int xp, int yp, int zp) {
    return (uint64_t)k | (uint64_t)axis << 14 | (uint64_t)s0on << 16 | (uint64_t)xp << 17 | (uint64_t)yp << 32 |
           (uint64_t)zp << 47;
}

// Triangle record: fine word (26 bits) | cell bit (5) | triangle of the cell
// (4) | cell case (8) | ROI (14).
__device__ __forceinline__ uint64_t pack_trec(uint32_t w, int b, int j, int cs, int k) {
    return (uint64_t)w | (uint64_t)b << 26 | (uint64_t)j << 31 | (uint64_t)cs << 35 | (uint64_t)k << 43;
}

// The boxes that hold every pixel this frame's z-buffer can write, for the clear
// of the slot's next frame: every mesh vertex lies
// in its ROI's fine grid box grown by one fine voxel (padding samples and
// surface points), so every covered pixel centre lies in the convex hull
// of the projections of that box's eight corners, widened by two pixels and
// clamped to the image; the whole image if a corner is not in front of the
// camera.  One box per ROI and camera, (0, -1, 0, -1) for none, whether or not a
// capacity turns out to be exceeded and nothing is drawn in them; eight lanes, a
// corner each, work a box out, from the launch's last block on.  (By one block, a
// thread per box, a frame of 500 ROIs and 16 cameras waited 130 us for it, one of
// 3,000 a millisecond; now some microseconds.  In k_mc_triangles, which has no
// registers to spare, 64 court frames took 190 us more; in k_zbuffer a 720p frame
// one and a half.)
__device__ __forceinline__ void list_depth_boxes(const CamSet& cams, const Grid& g, const Layout& L, int slot,
                                                 const DRoi* rois, int nrois) {
    int4* box = slot_ptr<int4>(L, slot, L.dbox);
    int* count = slot_ptr<int>(L, slot, L.dcount);
    if (blockIdx.x == 0)
        for (int n = threadIdx.x; n < cams.n; n += blockDim.x) count[n] = nrois;
    const int boxes = cams.n * nrois, lane = threadIdx.x & 31, q = lane & 7;
    const int step = (int)(gridDim.x * blockDim.x >> 5) * 4;
    for (int i0 = (int)(((gridDim.x - 1u - blockIdx.x) * blockDim.x + threadIdx.x) >> 5) * 4; i0 < boxes; i0 += step) {
        const int i = min(i0 + (lane >> 3), boxes - 1);       // (the last ones once more)
        const int n = i / nrois, k = i - n * nrois;
        const Cam& c = cams.c[n];
        const DRoi& r = rois[k];
        float X[3];
#pragma unroll
        for (int a = 0; a < 3; ++a)
            X[a] = (q >> a) & 1 ? r.fo[a] + (float)(r.fdim[a] + 1) * g.sf : r.fo[a] - g.sf;
        float xh, yh, wh;
        project(c.P, X[0], X[1], X[2], xh, yh, wh);
        const bool front = (__ballot_sync(kFull, wh > 0.0f) >> (lane & 24) & 0xFFu) == 0xFFu;
        float umin = __fdiv_rn(xh, wh), vmin = __fdiv_rn(yh, wh), umax = umin, vmax = vmin;
#pragma unroll
        for (int o = 1; o < 8; o <<= 1) {
            umin = fminf(umin, __shfl_xor_sync(kFull, umin, o));
            umax = fmaxf(umax, __shfl_xor_sync(kFull, umax, o));
            vmin = fminf(vmin, __shfl_xor_sync(kFull, vmin, o));
            vmax = fmaxf(vmax, __shfl_xor_sync(kFull, vmax, o));
        }
        int x0 = 0, x1 = c.W - 1, y0 = 0, y1 = c.H - 1;
        if (front && umin > -1.0e6f && umax < 1.0e6f && vmin > -1.0e6f && vmax < 1.0e6f) {
            x0 = max(0, (int)floorf(umin) - 2);
            x1 = min(c.W - 1, (int)floorf(umax) + 2);
            y0 = max(0, (int)floorf(vmin) - 2);
            y1 = min(c.H - 1, (int)floorf(vmax) + 2);
        }
        if (q == 0)
            box[(size_t)n * (unsigned)g.max_rois + (unsigned)k] =
                x0 > x1 || y0 > y1 ? make_int4(0, -1, 0, -1) : make_int4(x0, x1, y0, y1);
    }
}

// Sec. II-C classify and compact, in one pass over each slot's fine words:
// chunks of one to kMaxTurns turns of 256 words are claimed in order from a
// per-slot counter; a chunk's words and the neighbours its cells reach (a slab)
// are copied into shared memory by one bulk copy; each warp takes its words 32 at
// a time, a lane each: their bipolar-edge masks (x: w ^ w>>1, y: w ^ w(y+1), z:
// w ^ w(z+1)), vertex counts (the masks' popcounts) and triangle counts (table
// counts of the mixed cells).  Sums over the block give the counts of the chunk,
// and a decoupled look-back over the earlier chunks' published counts gives its
// base, so vertex ids follow the edge-key order (3*Lpad + axis) and triangles
// (ROI, cell, table order) of a serial scan.  Then each turn's words write their
// masks and prefix, and its mixed cells, listed in order in shared memory, are
// taken a lane each to write one record per vertex and one per triangle; the last
// chunk sets the totals and the capacity flags.  A chunk waits only on chunks
// claimed before it, whose blocks are running, so the look-back always ends.
//
// What bounds it is not the memory (some 15 MB for a court frame of 0.29 M words,
// 0.38 M vertices and 0.77 M triangles) but the claim, copy, counts and look-back
// that follow one another in every chunk, and, written by the lane that has the
// word, the records: a word of a level surface has 32 mixed cells, its neighbours
// none, and 12 of 32 lanes were at work.  A lane per listed cell, one store per
// word with a crossed edge and none for the others, no look-back for chunks
// without a mixed cell, and the ROI of a chunk's first word found beforehand
// (k_clear_fine): one court frame 39.4 -> 29.4 us, 64 of them 1341 -> 815.  Longer
// chunks share the chain out over more words where there are enough (the stage's
// kernels for 64 court frames, 118 chunks of one turn for each resident block: 2009
// us with one turn, 1877 with two, 1707 with four, the same with eight), and leave
// the chip idle where there are not (a frame of 28,640 vertices, 0.1 chunks, with
// one, two and four turns: 28, 34 and 43 us; four 4K court frames, 1.2 chunks: 54,
// 58 and 75).  In between it matters little (court, 1.9 chunks, one and two turns:
// 54 and 51; 4K mat, 3.3 chunks, one and three: 68 and 71), so launch_filter gives a
// turn for every kTurnChunks = 4.  Tried without gain: claiming a chunk ahead, with
// its copy (six times the time: a claimed chunk's counts then come only after the
// look-back before them), looking back over 64 to 512 chunks at a time (the same to
// half as much again), pauses between polls (the same).
__global__ void __launch_bounds__(kChunk, kMcBlocksPerSm) k_mc_compact(const __grid_constant__ CamSet cams,
                                                       const __grid_constant__ Grid g,
                                                       const __grid_constant__ Layout L,
                                                       const __grid_constant__ SlotList sl,
                                                       const __grid_constant__ McTable mc) {
    pdl_begin();
    extern __shared__ __align__(128) uint32_t slab[];   // kSlabWords
    __shared__ uint8_t s_ntri[256];
    __shared__ uint32_t s_turn[kChunk / 32][kMaxTurns], s_tot[kChunk / 32];
    __shared__ uint32_t s_word[kChunk / 32][4][32];        // a turn's words: masks, vertices before
    __shared__ uint16_t s_cell[kChunk / 32][32 * 32];      // a turn's mixed cells: word * 32 + cell
    __shared__ uint32_t s_case[8][kChunk];   // (cell_cases)
    __shared__ __align__(8) uint64_t bar;
    __shared__ uint32_t s_c, s_len, s_fail;
    __shared__ unsigned long long s_base[2];
    const int slot = sl.s[blockIdx.y];
    SlotInfo* info = slot_ptr<SlotInfo>(L, slot, L.info);
    // (n_words is set to zero where a capacity is exceeded, by the block with the
    // slot's last chunk, when every other chunk is claimed: a block that may still
    // read that finds no chunk left)
    const uint32_t nwords = info->n_words, nchunks = info->n_chunks, cw = info->chunk_words;
    const int nrois = info->n_rois;
    if (threadIdx.x == 0) {
        mbar_init(&bar);
        s_fail = 0u;
    }
    for (int i = threadIdx.x; i < 256; i += blockDim.x) s_ntri[i] = mc.ntri[i];
    __syncthreads();
    DRoi* rois = slot_ptr<DRoi>(L, slot, L.rois);
    const uint32_t* fine = slot_ptr<uint32_t>(L, slot, L.fine);
    uint4* emask = slot_ptr<uint4>(L, slot, L.emask);
    uint64_t* vrec = slot_ptr<uint64_t>(L, slot, L.vrec);
    uint64_t* trec = slot_ptr<uint64_t>(L, slot, L.trec);
    unsigned long long* cst = slot_ptr<unsigned long long>(L, slot, L.chunk_st);
    const uint32_t* clen = slot_ptr<uint32_t>(L, slot, L.chunk_len);
    list_depth_boxes(cams, g, L, slot, rois, nrois);
    bool pending = false;   // the wait for a copy ran out, and it may still be in flight
    const uint32_t turns = cw / kChunk, warp = threadIdx.x >> 5;
    const int lane = threadIdx.x & 31;
    // A warp's counts in one word: under 2^15 vertices (3 x 32 x 256) and 2^17 triangles
    constexpr int kVertBits = 15;
    constexpr uint32_t kVertMask = (1u << kVertBits) - 1u;
    static_assert(3 * 32 * 32 * kMaxTurns < 1 << kVertBits && kMaxTriPerCell * 32 * 32 * kMaxTurns < 1 << (32 - kVertBits),
                  "a warp's counts");
    const uint8_t* my_case = reinterpret_cast<const uint8_t*>(&s_case[0][threadIdx.x]);
    auto case_of = [&](int b) { return (int)my_case[(b >> 2) * (kChunk * 4) + (b & 3)]; };
    uint32_t parity = 0;
    RoiCursor p;
    for (;;) {
        if (threadIdx.x == 0) {
            const uint32_t c = nchunks ? atomicAdd(&info->next_chunk, 1u) : 0u;
            const uint32_t len = c < nchunks ? __ldcg(clen + c) : 0u;   // (k_clear_fine)
            s_c = c;
            s_len = s_fail ? len & ~(kChunkRoi - 1u) : len;
        }
        __syncthreads();                                   // the chunk is claimed, and the slab's last one written
        const uint32_t c = s_c;
        if (c >= nchunks) break;
        const uint32_t len = s_len, n4 = len & (kChunkRoi - 1u);
        bool use = n4 != 0u;
        if (use) {
            if (threadIdx.x == 0) {
                fence_proxy_async();
                mbar_expect_tx(&bar, n4 * 4u);
                bulk_copy_g2s(slab, fine + c * cw, n4 * 4u, &bar);
            }
            bool done = false;
            for (int it = 0; it < kMaxPolls && !done; ++it) done = mbar_try_wait(&bar, parity);
            // a copy that does not complete in time: this chunk and the later
            // ones read global memory, and the slot is flagged
            if (done) {
                parity ^= 1u;
            } else {
                s_fail = 1u;
                pending = true;
                atomicOr(&info->flags, (unsigned)FVV_FLAG_LOOP);
            }
            use = done;
        }
        const uint32_t lo = c * cw;
        auto nbhd = [&](uint32_t w, Nbhd& n) {
            if (use) load_nbhd_slab(slab, lo, p, w, n);
            else load_nbhd(fine, p, w, n);
        };
        // counts, 32 words at a time, in a warp's order of words
        uint32_t run = 0, passes = 0;         // counts of the warp's words so far; bit j: turn j has anything to write
        const uint32_t wlo = lo + warp * 32u * turns + lane;
        for (uint32_t j = 0; j < turns; ++j) {
            const uint32_t w = wlo + 32u * j;
            uint32_t mixed = 0;
            bool start = false;
            Nbhd n;
            if (w < nwords) {
                p.seek_from(rois, nrois, w, j ? p.k : (int)(len / kChunkRoi));
                nbhd(w, n);
                mixed = mixed_cells(n);
                start = w == p.lo;
            }
            if (!__any_sync(kFull, mixed || start)) continue;
            passes |= 1u << j;
            if (lane == 0) s_turn[warp][j] = run;
            uint32_t v = 0;
            if (mixed) {
                cell_cases(n, &s_case[0][threadIdx.x]);
                uint32_t t = 0;
                for (uint32_t m = mixed; m; m &= m - 1u) t += s_ntri[case_of(__ffs(m) - 1)];
                v = t << kVertBits |
                    (uint32_t)(__popc(n.w[0] ^ n.s[0]) + __popc(n.w[0] ^ n.w[1]) + __popc(n.w[0] ^ n.w[2]));
            }
            run += __reduce_add_sync(kFull, v);
        }
        if (lane == 0) s_tot[warp] = run;
        // A chunk without a mixed cell has neither vertices nor triangles; without
        // a ROI's first word and not the last, nothing else wants its base either.
        const bool full = __syncthreads_or(passes || c == nchunks - 1u);
        if (threadIdx.x == 0) {
            if (!full) {
                st_state(cst + 2 * (size_t)c, c ? kStAgg : kStInc);
                st_state(cst + 2 * (size_t)c + 1, c ? kStAgg : kStInc);
            }
        }
        if (!full) continue;
        uint32_t ev = 0, et = 0, tv = 0, tt = 0;
#pragma unroll
        for (int k = 0; k < kChunk / 32; ++k) {
            const uint32_t t = s_tot[k];
            if (k == (int)warp) ev = tv, et = tt;
            tv += t & kVertMask;
            tt += t >> kVertBits;
        }
        if (threadIdx.x < 32) {
            unsigned long long bv = 0, bt = 0;
            bool ok = true;
            if (c > 0) {
                if (threadIdx.x == 0) {
                    st_state(cst + 2 * (size_t)c, kStAgg | tv);
                    st_state(cst + 2 * (size_t)c + 1, kStAgg | tt);
                }
                ok = look_back_warp(cst, c, bv, bt);
            }
            if (threadIdx.x == 0) {
                st_state(cst + 2 * (size_t)c, kStInc | ((bv + tv) & kStVal));
                st_state(cst + 2 * (size_t)c + 1, kStInc | ((bt + tt) & kStVal));
                if (!ok) atomicOr(&info->flags, (unsigned)FVV_FLAG_LOOP);
                s_base[0] = bv;
                s_base[1] = bt;
                if (c == nchunks - 1u) {
                    // totals and capacities (the records past a capacity were not written)
                    const unsigned long long nv = bv + tv, nt = bt + tt;
                    unsigned fl = 0;
                    if (nv > g.max_verts) fl |= FVV_FLAG_VERTS;
                    if (nt > g.max_tris) fl |= FVV_FLAG_TRIS;
                    if (fl) atomicOr(&info->flags, fl);
                    info->n_verts = fl ? 0u : (uint32_t)nv;
                    info->n_tris = fl ? 0u : (uint32_t)nt;
                    if (fl) info->n_words = 0;   // nothing downstream runs on this frame
                }
            }
        }
        __syncthreads();
        for (; passes; passes &= passes - 1u) {
            const uint32_t j = __ffs(passes) - 1, w = wlo + 32u * j;
            const uint32_t before = s_turn[warp][j];
            const unsigned long long vb = s_base[0] + ev + (before & kVertMask), tb = s_base[1] + et + (before >> kVertBits);
            Nbhd n;
            uint32_t mixed = 0, xm = 0, ym = 0, zm = 0;
            bool start = false;
            if (w < nwords) {
                p.seek_from(rois, nrois, w, (int)(len / kChunkRoi));
                nbhd(w, n);
                mixed = mixed_cells(n);
                xm = n.w[0] ^ n.s[0];
                ym = n.w[0] ^ n.w[1];
                zm = n.w[0] ^ n.w[2];
                start = w == p.lo;
                if (turns > 1u && mixed) cell_cases(n, &s_case[0][threadIdx.x]);
            }
            // vertices and mixed cells of the words before this lane's
            uint32_t x = (uint32_t)(__popc(xm) + __popc(ym) + __popc(zm)) | (uint32_t)__popc(mixed) << 16;
            const uint32_t own = x;
            for (int o = 1; o < 32; o <<= 1) {
                const uint32_t y = __shfl_up_sync(kFull, x, o);
                if (lane >= o) x += y;
            }
            const uint32_t cells = __shfl_sync(kFull, x, 31) >> 16;
            x -= own;
            const uint32_t vfirst = x & 0xFFFFu;
            if (__any_sync(kFull, start)) {
                uint32_t t = 0;
                for (uint32_t m = mixed; m; m &= m - 1u) t += s_ntri[case_of(__ffs(m) - 1)];
                uint32_t y = t;
                for (int o = 1; o < 32; o <<= 1) {
                    const uint32_t z = __shfl_up_sync(kFull, y, o);
                    if (lane >= o) y += z;
                }
                if (start) {
                    rois[p.k].vert_off = (uint32_t)(vb + vfirst);
                    rois[p.k].tri_off = (uint32_t)(tb + y - t);
                }
            }
            // (read only for words with a crossed edge)
            if (xm | ym | zm) emask[w] = make_uint4(xm, ym, zm, (uint32_t)(vb + vfirst));
            // the turn's mixed cells in order, for a lane each
            s_word[warp][0][lane] = xm;
            s_word[warp][1][lane] = ym;
            s_word[warp][2][lane] = zm;
            s_word[warp][3][lane] = vfirst;
            uint16_t* put = s_cell[warp] + (x >> 16);
            for (uint32_t m = mixed; m; m &= m - 1u) *put++ = (uint16_t)(lane * 32 + __ffs(m) - 1);
            const uint64_t rec = pack_vrec(p.k, 0, 0, p.wx * 32, p.yp, p.zp);
            __syncwarp();
            unsigned long long t = tb;
            for (uint32_t i = 0; i < cells; i += 32u) {
                const bool has = i + lane < cells;
                const uint32_t cell = has ? s_cell[warp][i + lane] : 0u, src = cell >> 5, b = cell & 31u;
                const uint32_t cs = has ? reinterpret_cast<const uint8_t*>(&s_case[b >> 2][warp * 32u + src])[b & 3u] : 0u;
                const uint32_t nt = s_ntri[cs];                       // (none for case 0)
                uint32_t y = nt;
                for (int o = 1; o < 32; o <<= 1) {
                    const uint32_t z = __shfl_up_sync(kFull, y, o);
                    if (lane >= o) y += z;
                }
                const uint64_t r = __shfl_sync(kFull, rec, (int)src) + ((uint64_t)b << 17 | (uint64_t)(cs & 1u) << 16);
                if (has) {
                    const uint32_t lm = (1u << b) - 1u;
                    unsigned long long id = vb + s_word[warp][3][src] + __popc(s_word[warp][0][src] & lm) +
                                            __popc(s_word[warp][1][src] & lm) + __popc(s_word[warp][2][src] & lm);
                    // the cell's own sample (case bit 0) against the next in x, y and z (bits 1, 2 and 4)
                    const bool fx = (cs ^ cs >> 1) & 1u, fy = (cs ^ cs >> 2) & 1u, fz = (cs ^ cs >> 4) & 1u;
                    if (fx && id < g.max_verts) vrec[id] = r;
                    id += fx;
                    if (fy && id < g.max_verts) vrec[id] = r + (1u << 14);
                    id += fy;
                    if (fz && id < g.max_verts) vrec[id] = r + (2u << 14);
                    const unsigned long long first = t + y - nt;
                    const uint64_t tr = pack_trec(w - lane + src, (int)b, 0, (int)cs, (int)(r & 0x3FFFu));
                    for (uint32_t q = 0; q < nt; ++q)
                        if (first + q < g.max_tris) trec[first + q] = tr + ((uint64_t)q << 31);
                }
                t += __shfl_sync(kFull, y, 31);
            }
            __syncwarp();
        }
    }
    if (threadIdx.x == 0 && pending) {
        // a copy whose wait ran out: wait (bounded) before the block's shared memory goes
        for (int it = 0; it < kMaxPolls && !mbar_try_wait(&bar, parity); ++it) {
        }
    }
}

// What camera c sees of the grid edge m - h .. m + h, that is of every point
// its bisection can test.  h is `half` along the axis, so (dx, dy, dw), the
// rows of P applied to it, are one product each (as nine multiply-adds with h's
// zeros: 3636 instead of 3590 us for 64 court frames).  With u = x'/w' at m the
// ends lie at u +- (dx - u dw) / (w' +- dw), so within
// |dx - u dw| / (w' - |dw|) of u, and 1 / (w' - |dw|) <= (1 + 2 |dw| / w') / w'
// where |dw| <= w' / 2.  The box of that, widened by 0.2% and 2^-10 pixels for
// the bound's own roundings and by the camera's margins (segment_margins on the
// host; its allowance of 32 half ulps for a point's deviation holds 30
// midpoints and m), holds every tested point's pixel.  all_fg: the box's pixels
// are all inside the image and set.  inside: they are all inside the image.
// Boxes wider than 32 or taller than 8 pixels are not scanned.
__device__ __forceinline__ void check_edge(const SmemCam& c, const uint32_t* __restrict__ sil, const float* m, int axis,
                                           float half, bool& all_fg, bool& inside, uint32_t& reads) {
    all_fg = inside = false;
    float xh, yh, wh;
    project(c.P, m[0], m[1], m[2], xh, yh, wh);
    const float dx = fmul(c.P[axis], half);
    const float dy = fmul(c.P[4 + axis], half);
    const float dw = fmul(c.P[8 + axis], half);
    const float r = rcp_approx(wh), u = fmul(xh, r), v = fmul(yh, r);
    const float rw = fmul(r, __fmaf_rn(fmul(fabsf(dw), r), 2.0f, 1.002f));
    const float eu = __fmaf_rn(fabsf(__fmaf_rn(-u, dw, dx)), rw, fadd(c.du, 0x1p-10f));
    const float ev = __fmaf_rn(fabsf(__fmaf_rn(-v, dw, dy)), rw, fadd(c.dv, 0x1p-10f));
    const float u0 = fsub(u, eu), u1 = fadd(u, eu), v0 = fsub(v, ev), v1 = fadd(v, ev);
    inside = wh > fmul(2.0f, fabsf(dw)) && c.du >= 0.0f && u0 >= 0.0f && v0 >= 0.0f && u1 < c.Wf && v1 < c.Hf;
    if (!inside) return;
    // floors on the FMA pipe: kMagic + floor, and differences of the bits
    const int x0 = __float_as_int(__fadd_rd(u0, kMagic)) - 0x4B400000, y0 = __float_as_int(__fadd_rd(v0, kMagic)) - 0x4B400000;
    const int nx = __float_as_int(__fadd_rd(u1, kMagic)) - 0x4B400000 - x0, ny = __float_as_int(__fadd_rd(v1, kMagic)) - 0x4B400000 - y0;
    if (nx > 31 || ny > 7) return;
    const uint32_t want = (2u << nx) - 1u;           // nx + 1 pixels from x0 on
    const int sh = x0 & 31, two = sh + nx > 31 ? 1 : 0;
    const uint32_t* row = sil + c.bit_off + (unsigned)y0 * (unsigned)c.Wq + ((unsigned)x0 >> 5);
    uint32_t miss = 0u;
    for (int y = 0; y <= ny; y += 2) {               // two rows a turn, the last one twice if they are odd in number
        const uint32_t* next = row + (y < ny ? c.Wq : 0);
        const uint32_t a0 = __ldg(row), b0 = __ldg(next);
        uint32_t a1 = 0u, b1 = 0u;
        if (two) {
            a1 = __ldg(row + 1);
            b1 = __ldg(next + 1);
        }
        miss |= ~(__funnelshift_r(a0, a1, sh) & __funnelshift_r(b0, b1, sh)) & want;
        row = next + c.Wq;
    }
    reads += (unsigned)((ny + 1) << two);
    all_fg = miss == 0u;
}

// Sec. II-C, exact intersection: between the ON end a and the OFF end b of a
// bipolar edge, `steps` times m = (a+b)/2, a = m if m is occupied else b = m;
// the vertex is the final midpoint.
//
// Every point tested lies on the edge (up to rounding), so a camera that sees
// the whole edge inside its silhouette (check_edge) votes foreground for
// all of them: it is decided once per edge, and only the other cameras are
// tested at each midpoint, from the vertex's list.  A midpoint's first
// background camera in index order is then the first listed camera that votes
// background, so the occupancy and the test count (that camera's index + 1,
// or N when the midpoint is occupied) are those of the plain early-exit loop
// over all cameras.

// A grid edge: its point X with coordinate `axis` running from a, the ON
// sample's, to b, the OFF one's.
struct Edge {
    float X[3], a, b;
    int axis;
};

__device__ __forceinline__ Edge edge_of_record(uint64_t rec, const DRoi* rois, const Grid& g) {
    const int k = (int)(rec & 0x3FFFu), s0 = (int)(rec >> 16 & 1u);
    const int q[3] = {(int)(rec >> 17 & 0x7FFFu), (int)(rec >> 32 & 0x7FFFu), (int)(rec >> 47 & 0x7FFFu)};
    const DRoi& r = rois[k];
    Edge e;
    e.axis = (int)(rec >> 14 & 3u);
#pragma unroll
    for (int d = 0; d < 3; ++d) e.X[d] = fadd(r.fo[d], fmul(fadd((float)(q[d] - 1), 0.5f), g.sf));
    const int qa = e.axis == 0 ? q[0] : e.axis == 1 ? q[1] : q[2];
    const float c0 = e.axis == 0 ? e.X[0] : e.axis == 1 ? e.X[1] : e.X[2];
    const float c1 = fadd(r.fo[e.axis], fmul(fadd((float)qa, 0.5f), g.sf));
    e.a = s0 ? c0 : c1;
    e.b = s0 ? c1 : c0;
    return e;
}

// The point of edge e whose running coordinate is t.
__device__ __forceinline__ void edge_point(const Edge& e, float t, float* p) {
#pragma unroll
    for (int d = 0; d < 3; ++d) p[d] = e.axis == d ? t : e.X[d];
}

// The cameras that must be tested at each midpoint of edge e (bit n: camera
// n); seen_fg: some camera votes foreground on the whole edge; inside: the edge
// is inside the image of every camera to be tested.
template <class Mask>
__device__ __forceinline__ Mask edge_undecided(const SmemCam* sc, int ncam, const uint32_t* __restrict__ sil,
                                               const Edge& e, bool& seen_fg, bool& inside, uint32_t& reads) {
    Mask undecided = 0;
    seen_fg = false;
    inside = true;
    float m[3];
    edge_point(e, fmul(fadd(e.a, e.b), 0.5f), m);
    const float half = fmul(fsub(e.b, e.a), 0.5f);
    // the cameras' fields come from shared memory (the camera is the same in
    // every lane); four checks at a time overlap their loads (one at a time: 3772
    // instead of 3636 us for 64 court frames), 16 inlined copies with constant
    // operands cost more in instruction-cache misses than the loads
#pragma unroll 4
    for (int n = 0; n < ncam; ++n) {
        bool fg, in;
        check_edge(sc[n], sil, m, e.axis, half, fg, in, reads);
        undecided |= fg ? (Mask)0 : (Mask)1 << n;
        seen_fg |= fg;
        inside &= in;                        // (a camera that is not inside is never decided)
    }
    return undecided;
}

__device__ __forceinline__ int first_bit(uint32_t m) { return __ffs((int)m) - 1; }
__device__ __forceinline__ int first_bit(uint64_t m) { return __ffsll((long long)m) - 1; }

// The `steps` bisection steps of edge e with the cameras of `undecided` tested at
// each midpoint; e.a and e.b end as the last bracket.  INSIDE: the edge is
// inside every such camera's image (no clamps, no tests of the pixel).
template <bool INSIDE, class Mask>
__device__ __forceinline__ void edge_bisect(const SmemCam* sc, int ncam, const uint32_t* __restrict__ sil, int steps,
                                            bool abstain, Mask undecided, bool seen_fg, Edge& e, uint32_t& tests,
                                            uint32_t& reads) {
    for (int it = 0; it < steps; ++it) {
        const float t = fmul(fadd(e.a, e.b), 0.5f);
        float m[3];
        edge_point(e, t, m);
        int stop = -1;
        bool voted = !abstain || seen_fg;
        for (Mask u = undecided; u; u &= u - 1) {
            const int n = first_bit(u);
            bool in = true;
            uint32_t bit;
            if constexpr (INSIDE) bit = cam_bit_inside(sc[n], sil, m[0], m[1], m[2], true);
            else bit = cam_bit(sc[n], sil, m[0], m[1], m[2], in);
            reads += in ? 1u : 0u;
            if (abstain ? (in && !bit) : !bit) {
                stop = n;
                break;
            }
            voted |= bit != 0u;
        }
        tests += stop < 0 ? (unsigned)ncam : (unsigned)(stop + 1);
        const bool on = stop < 0 && voted;
        e.a = on ? t : e.a;
        e.b = on ? e.b : t;
    }
}

// Vertex i of a slot: its position and its pixel cells for the z-buffer.
__device__ __forceinline__ void store_vertex(float* verts, uint2* vcell, uint32_t i, const float* v,
                                             const SmemCam* sc, const CellCam* cc, int ncam) {
#pragma unroll
    for (int d = 0; d < 3; ++d) verts[3 * (size_t)i + d] = v[d];
    write_cells(sc, cc, ncam, v[0], v[1], v[2], vcell + (size_t)i * (unsigned)((ncam + 3) >> 2));
}

// Vertices a warp sorts at once, per lane, and the bucket of the sort that
// holds every list of kSortCap - 1 or more cameras (one more bucket, the
// last, holds the window's empty places).
constexpr int kBisectWin = 4;
constexpr int kSortCap = 7;
constexpr int kSortBuckets = kSortCap + 1;
constexpr int kSortPerLane = kSortBuckets * kBisectWin / 32;   // sort counters per lane
static_assert(kSortBuckets * kBisectWin % 32 == 0 && kBisectWin <= 8, "sort counters");

// Per-warp shared memory of the sorted path (dynamic shared memory, one per
// warp of the block).
template <class Mask>
struct BisectWarpSmem {
    Mask und[32 * kBisectWin];                 // undecided cameras of the window's vertices
    uint8_t seen[32 * kBisectWin];             // inside | seen_fg << 1
    uint8_t perm[32 * kBisectWin];             // window places in sorted order
    int cnt[kSortBuckets * kBisectWin];        // bucket-major counts, then their exclusive prefix
};

// One vertex per thread.  Lanes whose undecided lists differ in length idle in
// the midpoint loop while the longest list is walked (about 42% of the lanes
// busy there in vertex order, on a CPU model of a volleyball-shaped frame).
// When a slot has enough vertices for every warp of the launch that can be
// resident for it (`resident_warps`) to take two windows of 32 * kv
// consecutive vertices (kv = 2 or 4), each warp takes such windows instead:
// it finds every vertex's undecided cameras, sorts the window's vertices by
// the length of that list (a counting sort in the warp's shared memory, no
// block barrier) and then bisects them 32 at a time in that order, so that a
// warp's lanes walk lists of about the same length.  Each vertex's
// arithmetic is the same in both orders; only the lane that does it changes.
//
// Bound by instruction issue.  Mask is uint32_t for up to 32 cameras.  64 court
// frames 4655 -> 3590 us, one 109 -> 82 us, four 4K court frames 126 -> 77 us
// against projecting both ends of an edge in every camera and all three
// coordinates of every midpoint with the tests a point anywhere needs.
template <class Mask>
__global__ void __launch_bounds__(256) k_bisect(const __grid_constant__ CamSet cams, const __grid_constant__ Grid g,
                                                const __grid_constant__ Layout L, const __grid_constant__ SlotList sl,
                                                uint32_t resident_warps) {
    pdl_begin();
    __shared__ unsigned long long sh_t[32];
    __shared__ SmemCam sc[FVV_MAX_CAMS];
    __shared__ CellCam cc[FVV_MAX_CAMS];
    extern __shared__ __align__(16) unsigned char bisect_smem[];   // BisectWarpSmem per warp
    BisectWarpSmem<Mask>* wsm = reinterpret_cast<BisectWarpSmem<Mask>*>(bisect_smem);
    const int ncam = cams.n;
    load_smem_cams(cams, ncam, sc);
    load_cell_cams(cams, ncam, cc);
    __syncthreads();
    const bool abstain = cams.oob == FVV_OOB_ABSTAIN;
    const int slot = sl.s[blockIdx.y];
    const SlotInfo* info = slot_ptr<SlotInfo>(L, slot, L.info);
    const uint32_t nv = info->n_words ? info->n_verts : 0u;
    const DRoi* rois = slot_ptr<DRoi>(L, slot, L.rois);
    const uint32_t* __restrict__ sil = slot_ptr<uint32_t>(L, slot, L.sil);
    const uint64_t* vrec = slot_ptr<uint64_t>(L, slot, L.vrec);
    float* verts = slot_ptr<float>(L, slot, L.verts);
    uint2* vcell = slot_ptr<uint2>(L, slot, L.vcell);
    unsigned long long tests = 0, reads = 0;
    const uint32_t nthreads = gridDim.x * blockDim.x;
    int kv = 1;                                    // the same in every block of the slot
    for (int k = kBisectWin; k >= 2; k >>= 1)
        if (kv == 1 && (unsigned long long)nv >= 64ull * resident_warps * (unsigned)k) kv = k;
    // the steps of vertex i (edge e, undecided cameras `und`; where `have`), and
    // its results; all lanes of a warp call it together and take the same form
    auto finish = [&](bool have, uint32_t i, Edge& e, Mask und, bool seen_fg, bool inside) {
        const bool all_inside = __all_sync(kFull, inside || !have);
        if (!have) return;
        uint32_t t = 0, rd = 0;
        if (all_inside) edge_bisect<true>(sc, ncam, sil, g.steps, abstain, und, seen_fg, e, t, rd);
        else edge_bisect<false>(sc, ncam, sil, g.steps, abstain, und, seen_fg, e, t, rd);
        tests += t;
        reads += rd;
        float v[3];
        edge_point(e, fmul(fadd(e.a, e.b), 0.5f), v);
        store_vertex(verts, vcell, i, v, sc, cc, ncam);
    };
    if (kv == 1 || g.steps == 0) {
        const uint32_t lane = threadIdx.x & 31;
        for (uint32_t base = blockIdx.x * blockDim.x + (threadIdx.x & ~31u); base < nv; base += nthreads) {
            const uint32_t i = base + lane;
            const bool have = i < nv;
            Edge e{};
            Mask und = 0;
            bool seen_fg = false, inside = true;
            if (have) {
                e = edge_of_record(vrec[i], rois, g);
                uint32_t rd = 0;
                if (g.steps > 0) und = edge_undecided<Mask>(sc, ncam, sil, e, seen_fg, inside, rd);
                reads += rd;
            }
            finish(have, i, e, und, seen_fg, inside);
        }
    } else {
        const int lane = threadIdx.x & 31;
        BisectWarpSmem<Mask>& w = wsm[threadIdx.x >> 5];
        const uint32_t win = 32u * (uint32_t)kv;
        const uint32_t nwarps = nthreads >> 5;
        // windows of the slot's vertices, taken by the warps in turn (the loop
        // condition is the same in every lane)
        for (uint32_t base = ((blockIdx.x * blockDim.x + threadIdx.x) >> 5) * win; base < nv;
             base += nwarps * win) {
            // (1) each lane's kv vertices (place p of the window: vertex
            // base + p, empty from nv on): their undecided cameras
            for (int j = 0; j < kv; ++j) {
                const int p = j * 32 + lane;
                if (base + (uint32_t)p >= nv) break;
                const Edge e = edge_of_record(vrec[base + (uint32_t)p], rois, g);
                bool seen_fg, inside;
                uint32_t rd = 0;
                w.und[p] = edge_undecided<Mask>(sc, ncam, sil, e, seen_fg, inside, rd);
                w.seen[p] = (uint8_t)((inside ? 1u : 0u) | (seen_fg ? 2u : 0u));
                reads += rd;
            }
            // (2) counting sort of the window's places by list length
#pragma unroll
            for (int e = 0; e < kSortPerLane; ++e) w.cnt[kSortPerLane * lane + e] = 0;
            __syncwarp();
            // a place's key and its rank among the lanes of its window row with
            // that key (worked out twice, so that nothing stays in registers)
            auto place = [&](int j, int& key, int& rank) {
                const int p = j * 32 + lane;
                key = base + (uint32_t)p >= nv ? kSortCap : min(__popcll((unsigned long long)w.und[p]), kSortCap - 1);
                const unsigned same = __match_any_sync(kFull, key);
                rank = __popc(same & ((1u << lane) - 1u));
                return __popc(same);
            };
            for (int j = 0; j < kv; ++j) {
                int key, rank;
                const int n = place(j, key, rank);
                if (rank == 0) w.cnt[key * kBisectWin + j] = n;
            }
            __syncwarp();
            {   // exclusive prefix of the counts (bucket-major, then window row)
                int c[kSortPerLane], incl = 0;
#pragma unroll
                for (int e = 0; e < kSortPerLane; ++e) incl += c[e] = w.cnt[kSortPerLane * lane + e];
#pragma unroll
                for (int o = 1; o < 32; o <<= 1) {
                    const int t = __shfl_up_sync(kFull, incl, o);
                    if (lane >= o) incl += t;
                }
#pragma unroll
                for (int e = kSortPerLane - 1; e >= 0; --e) w.cnt[kSortPerLane * lane + e] = incl -= c[e];
            }
            __syncwarp();
            for (int j = 0; j < kv; ++j) {
                int key, rank;
                place(j, key, rank);
                w.perm[w.cnt[key * kBisectWin + j] + rank] = (uint8_t)(j * 32 + lane);
            }
            __syncwarp();
            // (3) the bisections, 32 at a time in sorted order (empty places last)
            for (int j = 0; j < kv; ++j) {
                const int p = w.perm[j * 32 + lane];
                const uint32_t i = base + (uint32_t)p;
                const bool have = i < nv;
                if (!__any_sync(kFull, have)) break;
                Edge e{};
                if (have) e = edge_of_record(vrec[i], rois, g);
                const uint32_t seen = w.seen[p];
                finish(have, i, e, w.und[p], (seen & 2u) != 0u, (seen & 1u) != 0u);
            }
            __syncwarp();   // the window's shared memory is read before the next one writes it
        }
    }
    const unsigned long long t = block_sum<unsigned long long>(tests, sh_t);
    const unsigned long long rd = block_sum<unsigned long long>(reads, sh_t);
    if (threadIdx.x == 0 && t) atomicAdd(&slot_ptr<SlotInfo>(L, slot, L.info)->tests_bisect, t);
    if (threadIdx.x == 0 && rd) atomicAdd(&slot_ptr<SlotInfo>(L, slot, L.info)->look_bisect, rd);
}

// Sec. II-C, Eq. (2), camera c, for the edge from the occupied end a to the
// unoccupied end b: walk the pixels of the line between their pixels in
// Bresenham order from a's end and stop at the first one outside the image
// or not in the silhouette; lambda = |centre of the last silhouette pixel -
// p_a| / |p_b - p_a| in the image plane, at most 1.  Cameras that bound
// nothing (an end behind the camera, the walk reaching b's pixel, a not
// seen, p_a = p_b) give 1.  `tests` counts the pixels visited.
__device__ __forceinline__ float cam_lambda(const Cam& c, const uint32_t* __restrict__ sil, const float* a,
                                           const float* b, uint32_t& tests) {
    float xa, ya, wa, xb, yb, wb;
    project(c.P, a[0], a[1], a[2], xa, ya, wa);
    project(c.P, b[0], b[1], b[2], xb, yb, wb);
    if (!(wa > 0.0f && wb > 0.0f)) return 1.0f;
    // end pixels: floor of the exact quotient, clamped to [-1, n + 1]
    const float ra = rcp_approx(wa), rb = rcp_approx(wb);
    int x = pixel_floor(xa, wa, ra, c.Wf), y = pixel_floor(ya, wa, ra, c.Hf);
    const int x1 = pixel_floor(xb, wb, rb, c.Wf), y1 = pixel_floor(yb, wb, rb, c.Hf);
    const int dx = abs(x1 - x), dy = -abs(y1 - y);
    const int sx = x < x1 ? 1 : -1, sy = y < y1 ? 1 : -1;
    int err = dx + dy;
    bool have = false;
    int lx = 0, ly = 0;
    for (;;) {   // at most max(dx, -dy) + 1 <= 65537 pixels
        ++tests;
        const bool in = (unsigned)x < (unsigned)c.W && (unsigned)y < (unsigned)c.H;
        const uint32_t word = in ? __ldg(sil + c.bit_off + (unsigned)y * (unsigned)c.Wq + ((unsigned)x >> 5)) : 0u;
        if (!((word >> (x & 31)) & 1u)) break;
        have = true;
        lx = x;
        ly = y;
        if (x == x1 && y == y1) return 1.0f;
        const int e2 = 2 * err;
        if (e2 >= dy) {
            err += dy;
            x += sx;
        }
        if (e2 <= dx) {
            err += dx;
            y += sy;
        }
    }
    if (!have) return 1.0f;
    const float ua = __fdiv_rn(xa, wa), va = __fdiv_rn(ya, wa), ub = __fdiv_rn(xb, wb), vb = __fdiv_rn(yb, wb);
    const float ex = fsub(fadd((float)lx, 0.5f), ua), ey = fsub(fadd((float)ly, 0.5f), va);
    const float fx = fsub(ub, ua), fy = fsub(vb, va);
    const float num = __fsqrt_rn(fadd(fmul(ex, ex), fmul(ey, ey)));
    const float den = __fsqrt_rn(fadd(fmul(fx, fx), fmul(fy, fy)));
    if (!(den > 0.0f)) return 1.0f;
    const float l = __fdiv_rn(num, den);
    return l < 1.0f ? l : 1.0f;
}

// Sec. II-C, Eq. (3): lambda = the minimum of Eq. (2) over the cameras; the
// vertex is a + lambda (b - a).  One vertex per thread.
template <int NC>
__global__ void __launch_bounds__(256) k_lambda(const __grid_constant__ CamSet cams, const __grid_constant__ Grid g,
                                                const __grid_constant__ Layout L, const __grid_constant__ SlotList sl) {
    pdl_begin();
    __shared__ unsigned long long sh_t[32];
    __shared__ SmemCam sc[FVV_MAX_CAMS];
    __shared__ CellCam cc[FVV_MAX_CAMS];
    const int ncam = NC > 0 ? NC : cams.n;
    load_smem_cams(cams, ncam, sc);
    load_cell_cams(cams, ncam, cc);
    __syncthreads();
    const int slot = sl.s[blockIdx.y];
    const SlotInfo* info = slot_ptr<SlotInfo>(L, slot, L.info);
    const uint32_t nv = info->n_words ? info->n_verts : 0u;
    const DRoi* rois = slot_ptr<DRoi>(L, slot, L.rois);
    const uint32_t* __restrict__ sil = slot_ptr<uint32_t>(L, slot, L.sil);
    const uint64_t* vrec = slot_ptr<uint64_t>(L, slot, L.vrec);
    float* verts = slot_ptr<float>(L, slot, L.verts);
    uint2* vcell = slot_ptr<uint2>(L, slot, L.vcell);
    uint32_t tests = 0;
    for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < nv; i += gridDim.x * blockDim.x) {
        const uint64_t rec = vrec[i];
        const int k = (int)(rec & 0x3FFFu), axis = (int)(rec >> 14 & 3u), s0 = (int)(rec >> 16 & 1u);
        const int q[3] = {(int)(rec >> 17 & 0x7FFFu), (int)(rec >> 32 & 0x7FFFu), (int)(rec >> 47 & 0x7FFFu)};
        const DRoi& r = rois[k];
        float a[3], b[3];
#pragma unroll
        for (int d = 0; d < 3; ++d) {
            const float c0 = fadd(r.fo[d], fmul(fadd((float)(q[d] - 1), 0.5f), g.sf));
            const float c1 = fadd(r.fo[d], fmul(fadd((float)(q[d] - 1 + (d == axis)), 0.5f), g.sf));
            a[d] = s0 ? c0 : c1;
            b[d] = s0 ? c1 : c0;
        }
        float lam = 1.0f;
        if constexpr (NC > 0) {
#pragma unroll
            for (int n = 0; n < NC; ++n) {
                const float l = cam_lambda(cams.c[n], sil, a, b, tests);
                if (l < lam) lam = l;
            }
        } else {
            for (int n = 0; n < cams.n; ++n) {
                const float l = cam_lambda(cams.c[n], sil, a, b, tests);
                if (l < lam) lam = l;
            }
        }
#pragma unroll
        for (int d = 0; d < 3; ++d) a[d] = fadd(a[d], fmul(lam, fsub(b[d], a[d])));
        store_vertex(verts, vcell, i, a, sc, cc, ncam);
    }
    // every pixel visited is one silhouette word read
    const unsigned long long t = block_sum<unsigned long long>(tests, sh_t);
    if (threadIdx.x == 0 && t) {
        atomicAdd(&slot_ptr<SlotInfo>(L, slot, L.info)->tests_bisect, t);
        atomicAdd(&slot_ptr<SlotInfo>(L, slot, L.info)->look_bisect, t);
    }
}

// Sec. II-C: the triangles, one per thread from the triangle records: the
// table gives the triangle's three cube edges, and each edge's vertex id is
// its word's vertex offset plus the rank of the edge among the word's
// bipolar edges (x, y, z masks in canonical order).  Also the centroid
// ((v0 + v1) + v2) / 3 of each triangle, for the depth images (Sec. II-D-1).
// Near the memory's rate with many frames: 68 bytes of records a triangle and the
// vertices, 64 court frames (49 M triangles) 810 us.  A word's masks and offset are
// one 16-byte load (four of 4 bytes: 897), the table 16 bytes a load (a court frame
// 21.2 -> 17.1 us).
__global__ void __launch_bounds__(256) k_mc_triangles(const __grid_constant__ Layout L,
                                                      const __grid_constant__ SlotList sl,
                                                      const __grid_constant__ McTable mc) {
    pdl_begin();
    __shared__ __align__(16) uint8_t s_edges[256 * kMaxTriPerCell * 3];
    for (int i = threadIdx.x; i < 256 * kMaxTriPerCell * 3 / 16; i += blockDim.x)
        reinterpret_cast<uint4*>(s_edges)[i] = reinterpret_cast<const uint4*>(mc.edges)[i];   // (256-byte aligned in the arena)
    __syncthreads();
    const int slot = sl.s[blockIdx.y];
    const SlotInfo* info = slot_ptr<SlotInfo>(L, slot, L.info);
    const uint32_t nt = info->n_words ? info->n_tris : 0u;
    const DRoi* rois = slot_ptr<DRoi>(L, slot, L.rois);
    const uint4* emask = slot_ptr<uint4>(L, slot, L.emask);
    const uint64_t* trec = slot_ptr<uint64_t>(L, slot, L.trec);
    uint32_t* tris = slot_ptr<uint32_t>(L, slot, L.tris);
    const float* verts = slot_ptr<float>(L, slot, L.verts);
    float4* tsoup = slot_ptr<float4>(L, slot, L.tsoup);
    for (uint32_t t = blockIdx.x * blockDim.x + threadIdx.x; t < nt; t += gridDim.x * blockDim.x) {
        const uint64_t rec = trec[t];
        const uint32_t w = (uint32_t)(rec & 0x3FFFFFFu);
        const int b = (int)(rec >> 26 & 31u), j = (int)(rec >> 31 & 15u), cs = (int)(rec >> 35 & 255u);
        const int k = (int)(rec >> 43 & 0x3FFFu);
        const uint32_t rs = (uint32_t)rois[k].nxw, ps = rs * (uint32_t)(rois[k].fdim[1] + 2);
        uint32_t id[3];
#pragma unroll
        for (int v = 0; v < 3; ++v) {
            const int e = s_edges[(cs * kMaxTriPerCell + j) * 3 + v];
            const int axis = e >> 2;
            // offsets of the edge's lower corner (same convention as the table)
            const int o0 = e & 1, o1 = (e >> 1) & 1;
            const int dx = axis == 0 ? 0 : o0;
            const int dy = axis == 1 ? 0 : (axis == 0 ? o0 : o1);
            const int dz = axis == 2 ? 0 : o1;
            const uint32_t wi = w + (uint32_t)((b + dx) >> 5) + (dy ? rs : 0u) + (dz ? ps : 0u);
            const int bb = (b + dx) & 31;
            const uint32_t lm = (1u << bb) - 1u;
            const uint4 m = emask[wi];
            uint32_t rank = __popc(m.x & lm) + __popc(m.y & lm) + __popc(m.z & lm);
            if (axis >= 1) rank += (m.x >> bb) & 1u;
            if (axis >= 2) rank += (m.y >> bb) & 1u;
            id[v] = m.w + rank;
        }
        tris[3 * (size_t)t + 0] = id[0];
        tris[3 * (size_t)t + 1] = id[1];
        tris[3 * (size_t)t + 2] = id[2];
        // the triangle's vertices and centroid ((v0 + v1) + v2) / 3, stored
        // together for the kernels that draw it
        float v[12];
#pragma unroll
        for (int q = 0; q < 3; ++q)
#pragma unroll
            for (int d = 0; d < 3; ++d) v[3 * q + d] = verts[3 * (size_t)id[q] + d];
#pragma unroll
        for (int d = 0; d < 3; ++d) v[9 + d] = __fdiv_rn(fadd(fadd(v[d], v[3 + d]), v[6 + d]), 3.0f);
        tsoup[3 * (size_t)t + 0] = make_float4(v[0], v[1], v[2], v[3]);
        tsoup[3 * (size_t)t + 1] = make_float4(v[4], v[5], v[6], v[7]);
        tsoup[3 * (size_t)t + 2] = make_float4(v[8], v[9], v[10], v[11]);
    }
}

}  // namespace

cudaError_t prepare_mc() {
    return cudaFuncSetAttribute(k_mc_compact, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                (int)(kSlabWords * sizeof(uint32_t)));
}

cudaError_t launch_mc_prefix(const CamSet& cams, const Grid& g, const Layout& L, const SlotList& sl, const McTable& mc, int sms,
                             cudaStream_t st) {
    const int gc = grid_x(sms, sl.n, g.max_chunks, 1);
    const cudaError_t e = launch_pdl(k_mc_compact, dim3(gc, sl.n), dim3(kChunk), kSlabWords * sizeof(uint32_t), st,
                                     cams, g, L, sl, mc);
    return e != cudaSuccess ? e : cudaGetLastError();
}

// Resident blocks per SM of a k_bisect instantiation (index: 0 for up to 32
// cameras, else 1) with `threads` threads and `smem` bytes of
// dynamic shared memory, asked of the runtime once per shape and kept.  The
// figure is that of the GPU current at the first call; on a host that mixes
// GPU models it may not fit the others, which changes only how the
// vertices are grouped into windows, never a result.
template <class K>
int bisect_blocks_per_sm(K kernel, int which, int threads, size_t smem) {
    static std::atomic<int> known[2][9];   // [which][threads / 32]; 0: not asked yet
    std::atomic<int>& slot = known[which][threads / 32];
    int n = slot.load(std::memory_order_relaxed);
    if (n == 0) {
        if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, kernel, threads, smem) != cudaSuccess || n < 1) {
            (void)cudaGetLastError();
            n = 1;
        }
        slot.store(n, std::memory_order_relaxed);
    }
    return n;
}

template <class Mask>
cudaError_t launch_bisect_mask(const CamSet& cams, const Grid& g, const Layout& L, const SlotList& sl, int sms, int th,
                               int gv, cudaStream_t st) {
    // the warps that can be resident for each slot: those launched, or the
    // slot's share of what the GPU holds if that is fewer
    const size_t smem = (size_t)(th / 32) * sizeof(BisectWarpSmem<Mask>);
    const int per_sm = bisect_blocks_per_sm(k_bisect<Mask>, sizeof(Mask) == 8, th, smem);
    const long long launched = (long long)gv * (th / 32);
    const long long fit = (long long)std::max(per_sm, 1) * sms * (th / 32) / std::max(sl.n, 1);
    const uint32_t resident = (uint32_t)std::max(1LL, std::min(launched, fit));
    return launch_pdl(k_bisect<Mask>, dim3(gv, sl.n), dim3(th), smem, st, cams, g, L, sl, resident);
}

cudaError_t launch_bisect(const CamSet& cams, const Grid& g, const Layout& L, const SlotList& sl, int sms,
                          const Tuning& tu, cudaStream_t st) {
    const int th = tu.threads[FVV_TUNE_BISECT];
    const int gv = tuned_grid(tu, FVV_TUNE_BISECT, sms, sl.n, g.max_verts);
    if (g.rule == FVV_SURFACE_LAMBDA) {
#define FVV_LAUNCH(NC) launch_pdl(k_lambda<NC>, dim3(gv, sl.n), dim3(th), 0, st, cams, g, L, sl)
        FVV_DISPATCH_NC(cams.n, FVV_LAUNCH)
#undef FVV_LAUNCH
        return cudaGetLastError();
    }
    const cudaError_t e = cams.n <= 32 ? launch_bisect_mask<uint32_t>(cams, g, L, sl, sms, th, gv, st)
                                       : launch_bisect_mask<uint64_t>(cams, g, L, sl, sms, th, gv, st);
    return e != cudaSuccess ? e : cudaGetLastError();
}

cudaError_t launch_mc_triangles(const Grid& g, const Layout& L, const SlotList& sl, const McTable& mc, int sms,
                                const Tuning& tu, cudaStream_t st) {
    const int gw = tuned_grid(tu, FVV_TUNE_TRIANGLES, sms, sl.n, g.max_tris);
    launch_pdl(k_mc_triangles, dim3(gw, sl.n), dim3(tu.threads[FVV_TUNE_TRIANGLES]), 0, st, L, sl, mc);
    return cudaGetLastError();
}

}  // namespace fvv
