// fvv_device.cuh -- device helpers shared by the kernels of libfvv: the
// silhouette predicate of Sec. II-B-1 and small warp/block reductions.
//
// All floating point uses the explicit round-to-nearest intrinsics
// (__fmul_rn, __fadd_rn, __fdiv_rn, __fsqrt_rn), which the compiler never
// fuses into an FMA, and explicit __fmaf_rn where a fused step is meant, so
// every result has one fixed binary32 value.
#pragma once

#include "fvv_internal.h"

namespace fvv {

constexpr unsigned kFull = 0xFFFFFFFFu;

// Programmatic dependent launch.  The kernels of a call are launched with
// launch_pdl, so that a kernel's blocks can be scheduled while the kernel
// before it in the stream is still finishing.  Every such kernel calls
// pdl_begin() first: it waits until the kernel before it has completed and
// its memory is visible (a no-op when the kernel was launched without the
// attribute), then lets the kernel after it be scheduled.
__device__ __forceinline__ void pdl_begin() {
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}

template <typename... KArgs, typename... Args>
inline cudaError_t launch_pdl(void (*kernel)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t st,
                              Args... args) {
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kernel, args...);
}

__device__ __forceinline__ float fadd(float a, float b) { return __fadd_rn(a, b); }
__device__ __forceinline__ float fsub(float a, float b) { return __fsub_rn(a, b); }
__device__ __forceinline__ float fmul(float a, float b) { return __fmul_rn(a, b); }

// (x', y', w') = P (X, Y, Z, 1), each row evaluated as ((p3 + p2 Z) + p1 Y) + p0 X
// with three fused multiply-adds (one rounding per step).
__device__ __forceinline__ void project(const float* p, float X, float Y, float Z, float& xp, float& yp,
                                        float& wp) {
    xp = __fmaf_rn(p[0], X, __fmaf_rn(p[1], Y, __fmaf_rn(p[2], Z, p[3])));
    yp = __fmaf_rn(p[4], X, __fmaf_rn(p[5], Y, __fmaf_rn(p[6], Z, p[7])));
    wp = __fmaf_rn(p[8], X, __fmaf_rn(p[9], Y, __fmaf_rn(p[10], Z, p[11])));
}

// Approximate reciprocal (PTX rcp.approx.ftz.f32: at most 1 ulp of error).
__device__ __forceinline__ float rcp_approx(float w) {
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(w));
    return r;
}

// floor(x / w) of the exact quotient, clamped to [-1, n + 1] (w > 0,
// n < 2^22): k0 = trunc(clamp(x * rcp(w), 0, n)) is within one of the answer
// whenever the answer is in [0, n]; the residual r0 = x - k0 w, formed by one
// FMA, is exact when |r0| < w and rounds monotonically otherwise, so r0 < 0
// means k0 is one too big and r0 >= w means one too small (or the quotient
// is outside [0, n), which the result then shows).  No branch and no
// conversion instruction: the integer part comes from a round-toward-zero
// add of 2^23.
__device__ __forceinline__ int pixel_floor(float x, float w, float r, float n) {
    const float q = fminf(fmaxf(fmul(x, r), 0.0f), n);
    const float t = __fadd_rz(q, 8388608.0f);   // 2^23 + trunc(q)
    const float k0 = fsub(t, 8388608.0f);
    const float r0 = __fmaf_rn(-k0, w, x);
    return (__float_as_int(t) - 0x4B000000) - (r0 < 0.0f ? 1 : 0) + (r0 >= w ? 1 : 0);
}

// Silhouette bit of camera c at the pixel holding world point (X,Y,Z)
// (Sec. II-B-1: project the voxel onto the silhouette): the pixel is
// (floor(x'/w'), floor(y'/w')) of the exact quotients of the binary32
// homogeneous coordinates.  `in` says whether the point is in front of the
// camera and inside its image; the bit is 0 when it is not.
template <class CamT>
__device__ __forceinline__ uint32_t cam_bit(const CamT& c, const uint32_t* __restrict__ sil, float X, float Y,
                                            float Z, bool& in) {
    float xp, yp, wp;
    project(c.P, X, Y, Z, xp, yp, wp);
    const float r = rcp_approx(wp);
    const int px = pixel_floor(xp, wp, r, c.Wf);
    const int py = pixel_floor(yp, wp, r, c.Hf);
    in = wp > 0.0f && (unsigned)px < (unsigned)c.W && (unsigned)py < (unsigned)c.H;
    const uint32_t word = in ? __ldg(sil + c.bit_off + (unsigned)py * (unsigned)c.Wq + ((unsigned)px >> 5)) : 0u;
    return (word >> (px & 31)) & 1u;
}

// The pixel a point falls in for camera c, or -1 in px/py if none (behind the
// camera or outside the image).  Same arithmetic as cam_bit.
__device__ __forceinline__ void cam_pixel(const Cam& c, float X, float Y, float Z, int& px, int& py) {
    float xp, yp, wp;
    project(c.P, X, Y, Z, xp, yp, wp);
    const float r = rcp_approx(wp);
    px = pixel_floor(xp, wp, r, c.Wf);
    py = pixel_floor(yp, wp, r, c.Hf);
    if (!(wp > 0.0f && (unsigned)px < (unsigned)c.W && (unsigned)py < (unsigned)c.H)) px = py = -1;
}

// One camera's test of a live lane.  STRICT: a camera that does not see the
// point votes background, so the lane stays alive only on a foreground bit.
// ABSTAIN: such a camera does not vote; the lane must see one foreground vote.
template <bool ABSTAIN>
__device__ __forceinline__ void test_cam(const Cam& c, const uint32_t* __restrict__ sil, float X, float Y, float Z,
                                         bool& alive, bool& voted) {
    bool in;
    const uint32_t bit = cam_bit(c, sil, X, Y, Z, in);
    if constexpr (ABSTAIN) {
        alive = !in || bit;
        voted |= in && bit;
    } else {
        alive = bit != 0u;
    }
}

// Camera counts with an unrolled instantiation of k_lambda (anything else runs its
// generic loop), so that the camera matrices are read as constant-bank operands
// instead of indexed constant loads.
#define FVV_DISPATCH_NC(n, F)   \
    switch (n) {                \
        case 4: F(4); break;    \
        case 6: F(6); break;    \
        case 8: F(8); break;    \
        case 10: F(10); break;  \
        case 12: F(12); break;  \
        case 16: F(16); break;  \
        default: F(0); break;   \
    }

// A camera's fields for tests where lanes use different cameras, kept in
// shared memory (80 bytes: consecutive cameras fall in different banks).
struct __align__(16) SmemCam {
    float P[12];
    float Wf, Hf;
    int W, H, Wq;
    uint32_t bit_off;
    float du, dv;            // Cam::seg_du, seg_dv
};

// Copy the first n cameras into sc (all threads of the block; the caller
// synchronises).
__device__ __forceinline__ void load_smem_cams(const CamSet& cams, int n, SmemCam* sc) {
    for (int i = threadIdx.x; i < n; i += blockDim.x) {
        const Cam& c = cams.c[i];
        for (int k = 0; k < 12; ++k) sc[i].P[k] = c.P[k];
        sc[i].Wf = c.Wf;
        sc[i].Hf = c.Hf;
        sc[i].W = c.W;
        sc[i].H = c.H;
        sc[i].Wq = c.Wq;
        sc[i].bit_off = c.bit_off;
        sc[i].du = c.seg_du;
        sc[i].dv = c.seg_dv;
    }
}

// Silhouette bit of a point that is known to be in front of camera c and
// inside its image (where `on`; 0 elsewhere): cam_bit without the clamps and
// the tests.
__device__ __forceinline__ uint32_t cam_bit_inside(const SmemCam& c, const uint32_t* __restrict__ sil, float X, float Y,
                                                   float Z, bool on) {
    float xp, yp, wp;
    project(c.P, X, Y, Z, xp, yp, wp);
    const float r = rcp_approx(wp);
    const float tx = __fadd_rz(fmul(xp, r), 8388608.0f), ty = __fadd_rz(fmul(yp, r), 8388608.0f);
    const float rx = __fmaf_rn(-fsub(tx, 8388608.0f), wp, xp), ry = __fmaf_rn(-fsub(ty, 8388608.0f), wp, yp);
    const unsigned px = (__float_as_uint(tx) & 0x7FFFFFu) + (rx >= wp ? 1u : 0u) - (rx < 0.0f ? 1u : 0u);
    const unsigned py = (__float_as_uint(ty) & 0x7FFFFFu) + (ry >= wp ? 1u : 0u) - (ry < 0.0f ? 1u : 0u);
    const uint32_t word = on ? __ldg(sil + c.bit_off + py * (unsigned)c.Wq + (px >> 5)) : 0u;
    return (word >> (px & 31u)) & 1u;
}

// ---- pixel cells: which pixel centres a vertex lies between, per camera
//
// A triangle covers no pixel centre of a camera if no column of centres, or
// no row, lies between its vertices' image positions; for meshes of one-pixel
// triangles that turns away two pairs (triangle, camera) out of three.  The
// cell of an image position u is floor(u - 1/2): the centres (integers plus
// 1/2) at or left of it.  Per vertex and camera the low 7 bits of its column
// and of its row cell are kept, one byte each, four cameras to a uint2 (x:
// columns, y: rows), with bit 7 set where the cell is not certain: u - 1/2 is
// within a slack of an integer, or the camera's cells do not decide
// (CamSet::cells; it then may have points that are not in front of it).
// Positions outside the image count as the cell before the first centre or
// at the last one.  Three
// equal bytes without bit 7 then mean that no column (row) of centres lies
// between the vertices: their cells are equal modulo 128 and, where
// CamSet::cells says so, less than 128 apart.
constexpr float kMagic = 12582912.0f;        // 1.5 * 2^23: floats within 2^22 of it are integers

// What a camera's cells take beside its matrix.
struct __align__(16) CellCam {
    float iW, iH;            // 1 / W, 1 / H
    float certain;           // 1/2 - slack: a position nearer than that to its cell's middle is certain; -1: never
    float pad_;
};

// The slack bounds, twice over, the error of an image position formed as in
// cell_at: seven roundings of at most 2^-23 relative to a position of at most W.
__device__ __forceinline__ void load_cell_cams(const CamSet& cams, int n, CellCam* cc) {
    for (int i = threadIdx.x; i < n; i += blockDim.x) {
        const float W = cams.c[i].Wf, H = cams.c[i].Hf;
        const float slack = __fmaf_rn(fadd(fmaxf(W, H), 2.0f), 0x1p-19f, 0x1p-12f);
        cc[i].iW = __frcp_rn(W);
        cc[i].iH = __frcp_rn(H);
        cc[i].certain = (cams.cells >> i) & 1u ? fsub(0.5f, slack) : -1.0f;
        cc[i].pad_ = 0.0f;
    }
}

// The cell of u = n s, s = x iw clamped to [0, 1] (all on the FMA pipe: the
// integer ALU is the busier one in the kernels that call this): floor(u - 1/2)
// is u - 1 rounded to the nearest integer, in the low bits of the result,
// unless u - 1/2 is near an integer, which the distance to it shows.
__device__ __forceinline__ uint32_t cell_at(float x, float iw, float n, float certain, bool& sure) {
    float s;
    asm("mul.rn.sat.f32 %0, %1, %2;" : "=f"(s) : "f"(x), "f"(iw));
    const float a = __fmaf_rn(s, n, kMagic - 1.0f);
    const float e = __fmaf_rn(s, n, fsub(kMagic - 1.0f, a));   // u - 1 - cell
    sure = fabsf(e) < certain;
    return __float_as_uint(a);
}

// The pixel cells of vertex (X, Y, Z) in the ncam cameras of sc and cc (all
// lanes use the same camera at a time), out[g] for cameras 4g .. 4g + 3.
__device__ __forceinline__ void write_cells(const SmemCam* sc, const CellCam* cc, int ncam, float X, float Y, float Z,
                                            uint2* out) {
#pragma unroll 1
    for (int g = 0; 4 * g < ncam; ++g) {
        uint32_t cx[4] = {0u, 0u, 0u, 0u}, cy[4] = {0u, 0u, 0u, 0u};
        uint32_t fx = 0, fy = 0;
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const int n = 4 * g + k;
            if (n >= ncam) break;
            float xp, yp, wp;
            project(sc[n].P, X, Y, Z, xp, yp, wp);
            const float r = rcp_approx(wp);
            bool sx, sy;
            cx[k] = cell_at(xp, fmul(r, cc[n].iW), sc[n].Wf, cc[n].certain, sx);
            cy[k] = cell_at(yp, fmul(r, cc[n].iH), sc[n].Hf, cc[n].certain, sy);
            if (!sx) fx |= 0x80u << (8 * k);
            if (!sy) fy |= 0x80u << (8 * k);
        }
        const uint32_t bx = __byte_perm(__byte_perm(cx[0], cx[1], 0x0040), __byte_perm(cx[2], cx[3], 0x0040), 0x5410);
        const uint32_t by = __byte_perm(__byte_perm(cy[0], cy[1], 0x0040), __byte_perm(cy[2], cy[3], 0x0040), 0x5410);
        out[g] = make_uint2((bx & 0x7F7F7F7Fu) | fx, (by & 0x7F7F7F7Fu) | fy);
    }
}

// The ROI holding fine word w: the last ROI whose first word is <= w.
__device__ __forceinline__ int roi_of_word(const DRoi* rois, int n, uint32_t w) {
    int lo = 0, hi = n - 1;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (rois[mid].word_off <= w) lo = mid;
        else hi = mid - 1;
    }
    return lo;
}

// Position of fine word w in its ROI's padded grid, with the ROI fields that the
// compaction needs kept in registers; another ROI is read only when w leaves
// the current one (a chunk's words are visited in increasing order, a few ROIs at
// most, from the chunk's first one on).
struct RoiCursor {
    int k = -1;
    uint32_t lo = 0, hi = 0;
    int fdim[3];
    int nxw;
    // word position
    int wx, yp, zp;

    __device__ __forceinline__ void take(const DRoi& r) {
        lo = r.word_off;
        hi = lo + r.n_words;
        nxw = r.nxw;
#pragma unroll
        for (int a = 0; a < 3; ++a) fdim[a] = r.fdim[a];
    }

    // (w: at or after the first word of ROI k0)
    __device__ __forceinline__ void seek_from(const DRoi* rois, int n, uint32_t w, int k0) {
        if (w >= hi || w < lo) {
            k = k0;
            take(rois[k]);
            while (w >= hi && k + 1 < n) take(rois[++k]);
        }
        place(w);
    }

    __device__ __forceinline__ void place(uint32_t w) {
        const uint32_t lw = w - lo;
        const uint32_t row = lw / (uint32_t)nxw;
        wx = (int)(lw - row * (uint32_t)nxw);
        yp = (int)(row % (uint32_t)(fdim[1] + 2));
        zp = (int)(row / (uint32_t)(fdim[1] + 2));
    }
};

// Sum over the block (blockDim.x a multiple of 32, <= 1024); result valid in
// thread 0.  `sh` needs 32 entries.
template <typename T>
__device__ __forceinline__ T block_sum(T v, T* sh) {
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(kFull, v, o);
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    __syncthreads();
    if (lane == 0) sh[wid] = v;
    __syncthreads();
    T s = 0;
    if (threadIdx.x == 0)
        for (int i = 0; i < (int)(blockDim.x >> 5); ++i) s += sh[i];
    return s;
}

// Exclusive prefix over the block of one uint32 per thread; `total` gets the
// block sum in every thread.  `sh` needs 33 entries.
__device__ __forceinline__ uint32_t block_exclusive_scan(uint32_t v, uint32_t* sh, uint32_t& total) {
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = blockDim.x >> 5;
    uint32_t x = v;
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t y = __shfl_up_sync(kFull, x, o);
        if (lane >= o) x += y;
    }
    __syncthreads();
    if (lane == 31) sh[wid] = x;
    __syncthreads();
    if (wid == 0) {
        uint32_t s = lane < nw ? sh[lane] : 0u;
        uint32_t t = s;
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t y = __shfl_up_sync(kFull, t, o);
            if (lane >= o) t += y;
        }
        if (lane < nw) sh[lane] = t - s;
        if (lane == 31) sh[32] = t;
    }
    __syncthreads();
    total = sh[32];
    return sh[wid] + x - v;
}

// 64-bit version of block_exclusive_scan; `sh` needs 33 entries.
__device__ __forceinline__ unsigned long long block_exclusive_scan64(unsigned long long v, unsigned long long* sh,
                                                                     unsigned long long& total) {
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = blockDim.x >> 5;
    unsigned long long x = v;
    for (int o = 1; o < 32; o <<= 1) {
        const unsigned long long y = __shfl_up_sync(kFull, x, o);
        if (lane >= o) x += y;
    }
    __syncthreads();
    if (lane == 31) sh[wid] = x;
    __syncthreads();
    if (wid == 0) {
        const unsigned long long s = lane < nw ? sh[lane] : 0ull;
        unsigned long long t = s;
        for (int o = 1; o < 32; o <<= 1) {
            const unsigned long long y = __shfl_up_sync(kFull, t, o);
            if (lane >= o) t += y;
        }
        if (lane < nw) sh[lane] = t - s;
        if (lane == 31) sh[32] = t;
    }
    __syncthreads();
    total = sh[32];
    return sh[wid] + x - v;
}

}  // namespace fvv
