// kernels_render.cu -- Sec. II-D: per-camera depth images (Eq. (4)) and the
// per-vertex visibility test and colour choice of Sec. II-D-2 and II-E.
//
// Depth images hold the binary32 bits of the squared distance (non-negative,
// so the unsigned order of the bits is the order of the values) and are
// merged with atomicMin; 0xFFFFFFFF means no triangle covered the pixel
// (+infinity).  Readers take the square root.
#include "fvv_device.cuh"

namespace fvv {
namespace {

// The depth images only ever hold values inside each camera's boxes
// (Layout::dbox), which contain every pixel the slot's last z-buffer could
// write: a reconstruction clears them (k_clear_fine) and lists its own
// (list_depth_boxes), so every pixel outside them is empty (+infinity)
// without clearing whole images each frame.
__global__ void __launch_bounds__(256) k_init_depth(const __grid_constant__ Layout L, size_t n16,
                                                    int n_cams) {
    const int slot = blockIdx.y;
    uint4* d = slot_ptr<uint4>(L, slot, L.depth);
    const uint4 v = make_uint4(kEmptyDepth, kEmptyDepth, kEmptyDepth, kEmptyDepth);
    for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < n16; i += (size_t)gridDim.x * blockDim.x)
        d[i] = v;
    if (blockIdx.x == 0 && threadIdx.x < (unsigned)n_cams) slot_ptr<int>(L, slot, L.dcount)[threadIdx.x] = 0;
}

// Eq. (4) coverage of one triangle (world vertices X, Y, Z) in camera c, in
// two parts, raster_setup and raster_pixels (below).
// The first part: the homogeneous image points of the vertices
// and the candidate pixels (centres within 1/64 px of the box of the
// approximate projections; their error is below 1e-3 px for images up to
// 65535 px, and the exact box test in raster_pixels decides).  False if a
// vertex is not in front of the camera or no pixel centre is a candidate.
//
// The candidate columns are ceil(umin - 1/2 - 1/64) .. floor((umax + 1/64)
// - 1/2), clamped to the image (rows alike).  They are rounded on the FMA
// pipe: for |t| < 2^22, t + 1.5 * 2^23 rounded down (up) is 1.5 * 2^23 +
// floor(t) (ceil(t)) exactly, since floats in [2^23, 2^24) are the
// integers; the box ends are kept in that form (kMagic + integer), so that
// comparing them compares the integers.  A clamped end is always in that range; an end
// outside it only arises for an empty box, which the comparison then shows.
struct TriSetup {
    float xh[3], yh[3], wh[3];
    float x0, x1, y0, y1;                    // kMagic + first/last candidate column and row
};

template <class CamT>
__device__ __forceinline__ bool raster_setup(const CamT& c, const float* X, const float* Y, const float* Z,
                                             TriSetup& s) {
    bool ok = true;
    float u[3], v[3];
#pragma unroll
    for (int j = 0; j < 3; ++j) {
        project(c.P, X[j], Y[j], Z[j], s.xh[j], s.yh[j], s.wh[j]);
        ok &= s.wh[j] > 0.0f;
        const float r = rcp_approx(s.wh[j]);
        u[j] = fmul(s.xh[j], r);
        v[j] = fmul(s.yh[j], r);
    }
    const float umin = fminf(u[0], fminf(u[1], u[2])), umax = fmaxf(u[0], fmaxf(u[1], u[2]));
    const float vmin = fminf(v[0], fminf(v[1], v[2])), vmax = fmaxf(v[0], fmaxf(v[1], v[2]));
    constexpr float kSlack = 0.5f + 1.0f / 64.0f;
    s.x0 = __fadd_ru(fmaxf(fsub(umin, kSlack), 0.0f), kMagic);
    s.y0 = __fadd_ru(fmaxf(fsub(vmin, kSlack), 0.0f), kMagic);
    s.x1 = __fadd_rd(fminf(fsub(fadd(umax, 1.0f / 64.0f), 0.5f), fsub(c.Wf, 1.0f)), kMagic);
    s.y1 = __fadd_rd(fminf(fsub(fadd(vmax, 1.0f / 64.0f), 0.5f), fsub(c.Hf, 1.0f)), kMagic);
    // (umax >= 0 and vmax >= 0 also turn away all-NaN image positions)
    return ok && umax >= 0.0f && vmax >= 0.0f && s.x0 <= s.x1 && s.y0 <= s.y1;
}

// The second part: the triangle is skipped if its projected area is zero;
// `sink(pixel)` is called for each candidate pixel (row-major index in an
// image W pixels wide) whose centre p lies in the closed box of the projection and on the
// inner side of (or on) all three edges, either winding.  Everything is
// decided on the homogeneous image points (x', y', w') without dividing: the
// edge function of edge (i, j) at p is (p_x a - p_y b) + c with
// a = y_i w_j - w_i y_j, b = x_i w_j - w_i x_j, c = x_i y_j - y_i x_j (its sign
// is the image-plane one for w > 0), the area is zero iff
// (x_0 a_12 - y_0 b_12) + w_0 c_12 is, and the box test uses the exact signs
// of p w_j - x_j from one FMA each.  A centre is in the box iff it is at or
// right of some vertex and at or left of some vertex, in x and in y; the first
// holds for all columns from some one on and the second up to some one, so
// the candidate rectangle is trimmed at its ends (at most one column or row
// each, as a rule none) instead of testing every pixel.
template <class Sink>
__device__ __forceinline__ void raster_pixels(unsigned W, const TriSetup& s, Sink&& sink) {
    const float* xh = s.xh;
    const float* yh = s.yh;
    const float* wh = s.wh;
    float ea[3], eb[3], ec[3];
#pragma unroll
    for (int e = 0; e < 3; ++e) {
        const int i = e, j = (e + 1) % 3;
        ea[e] = fsub(fmul(yh[i], wh[j]), fmul(wh[i], yh[j]));
        eb[e] = fsub(fmul(xh[i], wh[j]), fmul(wh[i], xh[j]));
        ec[e] = fsub(fmul(xh[i], yh[j]), fmul(yh[i], xh[j]));
    }
    const float det = fadd(fsub(fmul(xh[0], ea[1]), fmul(yh[0], eb[1])), fmul(wh[0], ec[1]));
    if (!(det > 0.0f || det < 0.0f)) return;
    // pixel centres, exact in binary32 (below 2^22)
    float x0 = fadd(fsub(s.x0, kMagic), 0.5f), x1 = fadd(fsub(s.x1, kMagic), 0.5f);
    float y0 = fadd(fsub(s.y0, kMagic), 0.5f), y1 = fadd(fsub(s.y1, kMagic), 0.5f);
    auto right_of = [&](float p, const float* h) {   // at or right of (below) some vertex
        return __fmaf_rn(p, wh[0], -h[0]) >= 0.0f || __fmaf_rn(p, wh[1], -h[1]) >= 0.0f ||
               __fmaf_rn(p, wh[2], -h[2]) >= 0.0f;
    };
    auto left_of = [&](float p, const float* h) {
        return __fmaf_rn(p, wh[0], -h[0]) <= 0.0f || __fmaf_rn(p, wh[1], -h[1]) <= 0.0f ||
               __fmaf_rn(p, wh[2], -h[2]) <= 0.0f;
    };
    while (x0 <= x1 && !right_of(x0, xh)) x0 = fadd(x0, 1.0f);
    while (x0 <= x1 && !left_of(x1, xh)) x1 = fsub(x1, 1.0f);
    while (y0 <= y1 && !right_of(y0, yh)) y0 = fadd(y0, 1.0f);
    while (y0 <= y1 && !left_of(y1, yh)) y1 = fsub(y1, 1.0f);
    if (!(x0 <= x1 && y0 <= y1)) return;
    size_t row = (size_t)(unsigned)__float2int_rz(y0) * W + (unsigned)__float2int_rz(x0);
    for (float py = y0; py <= y1; py = fadd(py, 1.0f), row += W) {
        const float b0 = fmul(py, eb[0]), b1 = fmul(py, eb[1]), b2 = fmul(py, eb[2]);
        size_t pix = row;
        for (float px = x0; px <= x1; px = fadd(px, 1.0f), ++pix) {
            const float e0 = fadd(fsub(fmul(px, ea[0]), b0), ec[0]);
            const float e1 = fadd(fsub(fmul(px, ea[1]), b1), ec[1]);
            const float e2 = fadd(fsub(fmul(px, ea[2]), b2), ec[2]);
            const bool in = (e0 >= 0.0f && e1 >= 0.0f && e2 >= 0.0f) || (e0 <= 0.0f && e1 <= 0.0f && e2 <= 0.0f);
            if (in) sink(pix);
        }
    }
}

// Eq. (4) coverage of one triangle (world vertices X, Y, Z) in camera c.
template <class Sink>
__device__ __forceinline__ void raster_tri(const Cam& c, const float* X, const float* Y, const float* Z,
                                           Sink&& sink) {
    TriSetup s;
    if (raster_setup(c, X, Y, Z, s)) raster_pixels((unsigned)c.W, s, sink);
}

// A camera's fields for drawing, kept in shared memory: lanes draw in
// different cameras (80 bytes: eight lanes' 16-byte reads of eight
// consecutive cameras fall in different banks).
struct __align__(16) ZCam {
    float P[12];
    float C[3];
    int W;
    float Wf, Hf;
    unsigned long long pix_off;
};
static_assert(sizeof(ZCam) == 80, "ZCam");

// Entries of a warp's queue: 31 left from before and 4 cameras of 32 triangles.
constexpr int kZQueue = 160;

// Draws queue entry q (triangle, camera) of this lane: the triangle is set up
// from its record and its covered pixels keep the minimum of the squared
// centroid distance (sqrt is monotone, so the square root of that minimum is
// the minimum distance itself, taken where the depth is read).  The minimum
// is an atomic whose result nobody waits for: reading the pixel first, to
// skip the atomics that lose, made each pixel wait for a read from L2 (court
// frame 66 -> 58 us, batch of 64 frames 3.31 -> 2.94 ms, large triangles of
// the 4K court 413 -> 273 us a batch without it).
__device__ __forceinline__ void zdraw(const ZCam* zc, uint2 q, const float4* tsoup, uint32_t* D) {
    const ZCam& c = zc[q.y];
    const uint32_t t = q.x;
    const float4 r0 = __ldg(tsoup + 3 * (size_t)t), r1 = __ldg(tsoup + 3 * (size_t)t + 1),
                 r2 = __ldg(tsoup + 3 * (size_t)t + 2);
    const float X[3] = {r0.x, r0.w, r1.z}, Y[3] = {r0.y, r1.x, r1.w}, Z[3] = {r0.z, r1.y, r2.x};
    const float dx = fsub(r2.y, c.C[0]);
    const float dy = fsub(r2.z, c.C[1]);
    const float dz = fsub(r2.w, c.C[2]);
    const uint32_t d2 = __float_as_uint(fadd(fadd(fmul(dx, dx), fmul(dy, dy)), fmul(dz, dz)));
    TriSetup s;
    if (!raster_setup(c, X, Y, Z, s)) return;
    uint32_t* img = D + c.pix_off;
    raster_pixels((unsigned)c.W, s, [&](size_t pix) { atomicMin(img + pix, d2); });
}

// 0x80 in every byte of v that is not zero.
__device__ __forceinline__ uint32_t nonzero_bytes(uint32_t v) {
    return (((v & 0x7F7F7F7Fu) + 0x7F7F7F7Fu) | v) & 0x80808080u;
}

// Eq. (4) depth images.  Grid (blocks, slots), issued slot by slot, so one
// frame's depth images are worked on together.  A warp takes 32 triangles at
// a time, one per lane, reads the pixel cells of their vertices (write_cells,
// 8 bytes per vertex and four cameras) and compares them bytewise: about 30
// instructions for four cameras' pairs, instead of three projections and a
// box each (about 100 a pair).  About 70% of the (triangle, camera) pairs of
// a one-pixel mesh are turned away; the warp queues the others and draws them
// 32 at a time, one per lane (zdraw), whatever their cameras.  It takes the
// triangles through `quads` groups of four cameras (1, 2 or 4, the
// autotuner's choice), so that their indices are read once for all of them;
// a frame with too few triangles to give every warp that can be resident for
// it (`resident`) two such units is cut into units of one group each.
// Court-shaped frames (800,000 triangles, 16 cameras): 72 -> 40 us a frame in
// a batch of 64; 4K court (180,000 triangles of 9 pixels): 82 -> 40 us.
__global__ void __launch_bounds__(256) k_zbuffer(const __grid_constant__ CamSet cams,
                                                    const __grid_constant__ Layout L,
                                                    const __grid_constant__ SlotList sl, int quads,
                                                    uint32_t resident) {
    pdl_begin();
    __shared__ ZCam zc[FVV_MAX_CAMS];
    __shared__ uint2 zq[8][kZQueue];          // per warp (at most 256 threads)
    const int slot = sl.s[blockIdx.y];
    const SlotInfo* info = slot_ptr<SlotInfo>(L, slot, L.info);
    const uint32_t nt = info->n_words ? info->n_tris : 0u;
    const int lane = threadIdx.x & 31;
    const uint32_t nwarps = (gridDim.x * blockDim.x) >> 5, batches = (nt + 31u) >> 5;
    const uint32_t warp = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const unsigned ng = (unsigned)(cams.n + 3) >> 2;   // groups of four cameras
    unsigned per = (unsigned)quads;           // groups a unit covers
    if ((unsigned long long)batches * ((ng + per - 1u) / per) < 2ull * resident) per = 1u;
    const uint32_t parts = (ng + per - 1u) / per;      // units per batch
    const unsigned long long units = (unsigned long long)batches * parts;
    if (((unsigned long long)blockIdx.x * blockDim.x >> 5) >= units) return;   // the whole block
    for (int k = threadIdx.x; k < cams.n; k += blockDim.x) {
        const Cam& c = cams.c[k];
        for (int j = 0; j < 12; ++j) zc[k].P[j] = c.P[j];
        for (int j = 0; j < 3; ++j) zc[k].C[j] = c.C[j];
        zc[k].W = c.W;
        zc[k].Wf = c.Wf;
        zc[k].Hf = c.Hf;
        zc[k].pix_off = c.pix_off;
    }
    __syncthreads();
    const uint32_t* tris = slot_ptr<uint32_t>(L, slot, L.tris);
    const uint2* vcell = slot_ptr<uint2>(L, slot, L.vcell);
    const float4* tsoup = slot_ptr<float4>(L, slot, L.tsoup);
    uint32_t* D = slot_ptr<uint32_t>(L, slot, L.depth);
    const unsigned lt = (1u << lane) - 1u;
    uint2* q = zq[threadIdx.x >> 5];
    int qn = 0;                               // queued pairs (the same in every lane)
    for (unsigned long long u = warp; u < units; u += nwarps) {
        const uint32_t batch = parts == 1u ? (uint32_t)u : (uint32_t)(u / parts);
        const unsigned g0 = ((uint32_t)u - batch * parts) * per, g1 = min(g0 + per, ng);
        const uint32_t t = batch * 32u + (uint32_t)lane;
        const bool have = t < nt;
        const uint2* v[3];
#pragma unroll
        for (int j = 0; j < 3; ++j) v[j] = vcell + (have ? (size_t)__ldg(tris + 3 * (size_t)t + j) * ng : 0u);
#pragma unroll 1
        for (unsigned g = g0; g < g1; ++g) {
            const uint2 a = __ldg(v[0] + g), b = __ldg(v[1] + g), c = __ldg(v[2] + g);
            const uint32_t dx = (a.x ^ b.x) | (a.x ^ c.x) | ((a.x | b.x | c.x) & 0x80808080u);
            const uint32_t dy = (a.y ^ b.y) | (a.y ^ c.y) | ((a.y | b.y | c.y) & 0x80808080u);
            const uint32_t m = have ? nonzero_bytes(dx) & nonzero_bytes(dy) : 0u;
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                const bool on = (m >> (8 * k + 7)) & 1u;
                const unsigned who = __ballot_sync(kFull, on);
                if (on) q[qn + __popc(who & lt)] = make_uint2(t, 4u * g + k);
                qn += __popc(who);
            }
            __syncwarp();
#pragma unroll 1
            while (qn >= 32) {
                qn -= 32;
                zdraw(zc, q[qn + lane], tsoup, D);
                __syncwarp();                 // read before the entries are reused
            }
        }
    }
    if (lane < qn) zdraw(zc, q[lane], tsoup, D);
}

// Stored squared distance -> distance (+infinity for an empty pixel).
__device__ __forceinline__ float depth_of(uint32_t bits) {
    return bits == kEmptyDepth ? __int_as_float(0x7f800000) : __fsqrt_rn(__uint_as_float(bits));
}

// Sec. II-D-2 and II-E: the capture cameras ranked by squared distance of
// their centre to the viewpoint vp, ties to the lower index (thread m <
// cams.n places camera m; the caller synchronises).
__device__ __forceinline__ void rank_cameras(const CamSet& cams, const float* vp, int* rank_cam) {
    if (threadIdx.x < (unsigned)cams.n) {
        float d2[FVV_MAX_CAMS];
        const int me = threadIdx.x;
        int r = 0;
        for (int m = 0; m < cams.n; ++m) {
            const float ax = fsub(cams.c[m].C[0], vp[0]), ay = fsub(cams.c[m].C[1], vp[1]),
                        az = fsub(cams.c[m].C[2], vp[2]);
            d2[m] = fadd(fadd(fmul(ax, ax), fmul(ay, ay)), fmul(az, az));
        }
        for (int m = 0; m < cams.n; ++m) r += (d2[m] < d2[me]) || (d2[m] == d2[me] && m < me);
        rank_cam[r] = me;
    }
}

// The colour of world point (X,Y,Z): the first camera in rank order that has
// it in front, inside the image and with |X - C| - depth <= t_v, and that
// camera's RGB at the point's pixel.  Returns the camera, or -1 with (0,0,0).
__device__ __forceinline__ int colour_point(const CamSet& cams, const int* rank_cam,
                                            const uint32_t* __restrict__ depth, const uint8_t* const* rgb, float t_v,
                                            float X, float Y, float Z, uint8_t* col) {
    col[0] = col[1] = col[2] = 0;
    for (int k = 0; k < cams.n; ++k) {
        const int n = rank_cam[k];
        const Cam& c = cams.c[n];
        int px, py;
        cam_pixel(c, X, Y, Z, px, py);
        if (px < 0) continue;
        const size_t pix = (size_t)py * (unsigned)c.W + (size_t)px;
        const float dx = fsub(X, c.C[0]), dy = fsub(Y, c.C[1]), dz = fsub(Z, c.C[2]);
        const float dist = __fsqrt_rn(fadd(fadd(fmul(dx, dx), fmul(dy, dy)), fmul(dz, dz)));
        const float dep = depth_of(__ldg(depth + c.pix_off + pix));
        if (!(fsub(dist, dep) <= t_v)) continue;
        const uint8_t* src = rgb[n] + 3 * pix;
        col[0] = __ldg(src);
        col[1] = __ldg(src + 1);
        col[2] = __ldg(src + 2);
        return n;
    }
    return -1;
}

// Per vertex: colour_point with the cameras ranked for the slot's viewpoint.
__global__ void __launch_bounds__(256) k_colour(const __grid_constant__ CamSet cams, const __grid_constant__ Grid g,
                                                const __grid_constant__ Layout L,
                                                const __grid_constant__ ColourBatch cb) {
    pdl_begin();
    __shared__ int rank_cam[FVV_MAX_CAMS];
    const int slot = cb.slot[blockIdx.y];
    rank_cameras(cams, cb.view[blockIdx.y], rank_cam);
    __syncthreads();
    const SlotInfo* info = slot_ptr<SlotInfo>(L, slot, L.info);
    const uint32_t nv = info->n_words ? info->n_verts : 0u;
    const float* verts = slot_ptr<float>(L, slot, L.verts);
    const uint32_t* depth = slot_ptr<uint32_t>(L, slot, L.depth);
    const uint8_t* const* rgb = cb.rgb[blockIdx.y];
    uint8_t* out = slot_ptr<uint8_t>(L, slot, L.vrgb);
    int* ocam = slot_ptr<int>(L, slot, L.vcam);
    for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < nv; i += gridDim.x * blockDim.x) {
        uint8_t col[3];
        const int chosen = colour_point(cams, rank_cam, depth, rgb, g.t_v, verts[3 * (size_t)i],
                                        verts[3 * (size_t)i + 1], verts[3 * (size_t)i + 2], col);
        out[3 * (size_t)i] = col[0];
        out[3 * (size_t)i + 1] = col[1];
        out[3 * (size_t)i + 2] = col[2];
        ocam[i] = chosen;
    }
}

// ---- results

// Copies n bytes, 16, 4 or 1 at a time as the destination's alignment allows
// (the sources are 256-byte aligned), by all threads of the `blocks` blocks.
__device__ __forceinline__ void copy_bytes(char* __restrict__ dst, const char* __restrict__ src, size_t n,
                                           unsigned block, unsigned blocks) {
    const size_t i0 = (size_t)block * blockDim.x + threadIdx.x, step = (size_t)blocks * blockDim.x;
    const uintptr_t a = reinterpret_cast<uintptr_t>(dst);
    size_t done = 0;
    if ((a & 15u) == 0) {
        const size_t m = n >> 4;
        const uint4* s = reinterpret_cast<const uint4*>(src);
        uint4* d = reinterpret_cast<uint4*>(dst);
        size_t i = i0;
        for (; i + 3 * step < m; i += 4 * step) {     // four loads in flight
            const uint4 v0 = __ldcs(s + i), v1 = __ldcs(s + i + step), v2 = __ldcs(s + i + 2 * step),
                        v3 = __ldcs(s + i + 3 * step);
            __stcs(d + i, v0);
            __stcs(d + i + step, v1);
            __stcs(d + i + 2 * step, v2);
            __stcs(d + i + 3 * step, v3);
        }
        for (; i < m; i += step) __stcs(d + i, __ldcs(s + i));
        done = m << 4;
    } else if ((a & 3u) == 0) {
        const size_t m = n >> 2;
        for (size_t i = i0; i < m; i += step)
            __stcs(reinterpret_cast<uint32_t*>(dst) + i, __ldcs(reinterpret_cast<const uint32_t*>(src) + i));
        done = m << 2;
    }
    for (size_t i = done + i0; i < n; i += step) dst[i] = src[i];
}

// The results of several slots in one launch, as long as the device's own
// counts say, so that nobody waits for them first; the counts go to the host with
// them.  Grid (blocks, slots).  Bound by HBM: 64 court frames (1.1 GB read and
// written) 474 us, of a call of 733; with 64 + 256 copies and a wait between them
// the call took 2520.
__global__ void __launch_bounds__(256) k_gather_results(const __grid_constant__ Layout L,
                                                        const __grid_constant__ GatherSlots gs, SlotInfo* infos) {
    pdl_begin();
    const int slot = gs.slot[blockIdx.y];
    const SlotInfo* info = slot_ptr<SlotInfo>(L, slot, L.info);
    if (blockIdx.x == 0 && threadIdx.x < sizeof(SlotInfo) / 4)
        reinterpret_cast<uint32_t*>(infos + blockIdx.y)[threadIdx.x] = reinterpret_cast<const uint32_t*>(info)[threadIdx.x];
    if (info->n_words == 0u || (info->flags & kOverCapacity)) return;
    const size_t nv = info->n_verts, nt = info->n_tris;
#pragma unroll 1
    for (int k = 0; k < 4; ++k) {
        char* dst = gs.dst[blockIdx.y][k];
        const size_t off = k == 0 ? L.verts : k == 1 ? L.tris : k == 2 ? L.vrgb : L.vcam;
        const size_t n = k == 0 ? 12 * nv : k == 1 ? 12 * nt : k == 2 ? 3 * nv : 4 * nv;
        if (dst) copy_bytes(dst, slot_ptr<char>(L, slot, off), n, blockIdx.x, gridDim.x);
    }
}
static_assert(sizeof(SlotInfo) % 4 == 0 && sizeof(SlotInfo) / 4 <= 256, "SlotInfo copy");
static_assert(sizeof(GatherSlots) + sizeof(Layout) <= 32000, "k_gather_results parameters");

// ---- Sec. II-E, step E: a novel view of the coloured mesh

__global__ void __launch_bounds__(256) k_view_clear(unsigned long long* __restrict__ key, size_t npix) {
    for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < npix; i += (size_t)gridDim.x * blockDim.x)
        key[i] = ~0ull;
}

// Visibility in the virtual view: every covered pixel keeps the minimum of
// (squared distance from the triangle's centroid to the view centre, as float
// bits) << 32 | triangle index -- the nearest triangle, ties to the lower
// index.  One thread per triangle; nobody waits for the atomics (reading each
// pixel first to skip those that lose took 20.1 us instead of 11.7 for a
// full-HD view of 800,000 triangles).
__global__ void __launch_bounds__(256) k_view_raster(const __grid_constant__ Layout L,
                                                     const __grid_constant__ ViewArgs va,
                                                     unsigned long long* __restrict__ key) {
    const Cam& v = va.v;
    const SlotInfo* info = slot_ptr<SlotInfo>(L, va.slot, L.info);
    const uint32_t nt = info->n_words ? info->n_tris : 0u;
    const float4* tsoup = slot_ptr<float4>(L, va.slot, L.tsoup);
    for (uint32_t t = blockIdx.x * blockDim.x + threadIdx.x; t < nt; t += gridDim.x * blockDim.x) {
        const float4 r0 = __ldg(tsoup + 3 * (size_t)t), r1 = __ldg(tsoup + 3 * (size_t)t + 1),
                     r2 = __ldg(tsoup + 3 * (size_t)t + 2);
        const float X[3] = {r0.x, r0.w, r1.z}, Y[3] = {r0.y, r1.x, r1.w}, Z[3] = {r0.z, r1.y, r2.x};
        const float dx = fsub(r2.y, v.C[0]);
        const float dy = fsub(r2.z, v.C[1]);
        const float dz = fsub(r2.w, v.C[2]);
        const unsigned long long k =
            (unsigned long long)__float_as_uint(fadd(fadd(fmul(dx, dx), fmul(dy, dy)), fmul(dz, dz))) << 32 | t;
        raster_tri(v, X, Y, Z, [&](size_t pix) { atomicMin(key + pix, k); });
    }
}

// Colour of every pixel of the view: colour_point of its triangle's
// centroid, with the capture cameras ranked for the view centre, so the
// camera is chosen per pixel (Sec. II-E: the nearest camera where it sees
// the surface, its neighbours where it is occluded).
__global__ void __launch_bounds__(256) k_view_shade(const __grid_constant__ CamSet cams,
                                                    const __grid_constant__ Grid g, const __grid_constant__ Layout L,
                                                    const __grid_constant__ ViewArgs va,
                                                    const unsigned long long* __restrict__ key,
                                                    uint8_t* __restrict__ out_rgb, int32_t* __restrict__ out_cam) {
    __shared__ int rank_cam[FVV_MAX_CAMS];
    rank_cameras(cams, va.v.C, rank_cam);
    __syncthreads();
    const uint32_t* depth = slot_ptr<uint32_t>(L, va.slot, L.depth);
    const float4* tsoup = slot_ptr<float4>(L, va.slot, L.tsoup);
    const size_t npix = (size_t)va.v.W * (unsigned)va.v.H;
    for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < npix; i += (size_t)gridDim.x * blockDim.x) {
        const unsigned long long k = key[i];
        uint8_t col[3] = {0, 0, 0};
        int chosen = -1;
        if (k != ~0ull) {
            const float4 r2 = __ldg(tsoup + 3 * (size_t)(uint32_t)k + 2);   // (v2 z, centroid xyz)
            chosen = colour_point(cams, rank_cam, depth, va.rgb, g.t_v, r2.y, r2.z, r2.w, col);
        }
        out_rgb[3 * i] = col[0];
        out_rgb[3 * i + 1] = col[1];
        out_rgb[3 * i + 2] = col[2];
        if (out_cam) out_cam[i] = chosen;
    }
}

__global__ void k_debug_depth(const __grid_constant__ Layout L, int slot, float* dst, size_t npix) {
    const uint32_t* d = slot_ptr<uint32_t>(L, slot, L.depth);
    for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < npix; i += (size_t)gridDim.x * blockDim.x) {
        const uint32_t b = d[i];
        dst[i] = depth_of(b);
    }
}

}  // namespace

cudaError_t launch_init_depth(const CamSet& cams, const Layout& L, int n_slots, int sms, cudaStream_t st) {
    size_t pix = 0;
    for (int n = 0; n < cams.n; ++n) pix += (size_t)cams.c[n].W * cams.c[n].H;
    const size_t n16 = (pix * 4 + 15) / 16;
    const unsigned gx = (unsigned)std::max<size_t>(1, std::min<size_t>((n16 + 255) / 256, (size_t)sms * 4));
    for (int s0 = 0; s0 < n_slots; s0 += 65535) {
        // slots s0.. in one launch (blockIdx.y is at most 65535)
        Layout Ls = L;
        Ls.base = L.base + (size_t)s0 * L.stride;
        k_init_depth<<<dim3(gx, std::min(65535, n_slots - s0)), 256, 0, st>>>(Ls, n16, cams.n);
    }
    return cudaGetLastError();
}

cudaError_t launch_depth(const CamSet& cams, const Grid& g, const Layout& L, const SlotList& sl, int sms,
                         const Tuning& tu, cudaStream_t st) {
    const int gz = tuned_grid(tu, FVV_TUNE_ZBUFFER, sms, sl.n, (long long)g.max_tris);
    const int th = tu.threads[FVV_TUNE_ZBUFFER];
    // warps that the GPU can hold for a slot: 1024 threads per SM at the kernel's 64 registers
    const uint32_t resident = (uint32_t)std::max(1LL, (long long)sms * 32 / std::max(1, sl.n));
    const cudaError_t e = launch_pdl(k_zbuffer, dim3(gz, sl.n), dim3(th), 0, st, cams, L, sl, tu.zb_cams, resident);
    return e != cudaSuccess ? e : cudaGetLastError();
}

cudaError_t launch_colour(const CamSet& cams, const Grid& g, const Layout& L, const ColourBatch& cb, int sms,
                          int total_slots, cudaStream_t st) {
    const int gv = grid_x(sms, total_slots, g.max_verts, 256);
    launch_pdl(k_colour, dim3(gv, cb.n), dim3(256), 0, st, cams, g, L, cb);
    return cudaGetLastError();
}

cudaError_t launch_gather_results(const Layout& L, const GatherSlots& gs, SlotInfo* infos, int sms, cudaStream_t st) {
    const int gx = std::max(1, sms * 8 / std::max(1, gs.n));
    const cudaError_t e = launch_pdl(k_gather_results, dim3(gx, gs.n), dim3(256), 0, st, L, gs, infos);
    return e != cudaSuccess ? e : cudaGetLastError();
}

cudaError_t launch_render_view(const CamSet& cams, const Grid& g, const Layout& L, const ViewArgs& va,
                              unsigned long long* key, uint8_t* out_rgb, int32_t* out_cam, int sms, cudaStream_t st) {
    const size_t npix = (size_t)va.v.W * (unsigned)va.v.H;
    const unsigned gp = (unsigned)std::max<size_t>(1, std::min<size_t>((npix + 255) / 256, (size_t)sms * 8));
    k_view_clear<<<gp, 256, 0, st>>>(key, npix);
    const unsigned gt = (unsigned)std::max<long long>(1, std::min<long long>((g.max_tris + 255) / 256, (long long)sms * 8));
    k_view_raster<<<gt, 256, 0, st>>>(L, va, key);
    k_view_shade<<<gp, 256, 0, st>>>(cams, g, L, va, key, out_rgb, out_cam);
    return cudaGetLastError();
}

cudaError_t launch_debug_depth(const CamSet& cams, const Layout& L, int slot, float* dst, size_t npix,
                               cudaStream_t st) {
    (void)cams;
    k_debug_depth<<<(unsigned)std::min<size_t>((npix + 255) / 256, 8192), 256, 0, st>>>(L, slot, dst, npix);
    return cudaGetLastError();
}

}  // namespace fvv
