// noalloc.cu -- fvv_label_components_noalloc: 26-connected labelling of a
// coarse occupancy bitset with the size filter, for callers that cannot
// allocate device memory.
//
// Its scratch (union-find parents and the component list; the components' voxel
// counts are kept in the labels' array until the labels are written) lives in
// one file-scope static __device__ array, so the call
// allocates nothing: no cudaMalloc, no cudaFree, no allocating library call.
// The array is part of the library image, so every GPU that loads the
// library holds it (kScratchInts ints, about 33.6 MB) until the process exits.
//
// Host code cannot use the array's name as a device address (in host code it
// names a host-side stand-in), so the first call on each device, with that
// device current, asks cudaGetSymbolAddress for the real address and keeps it.
// That first call should therefore come before any stream capture.
//
// Every call shares the one array: calls that overlap on the GPU (on
// different streams, or from different threads) race on it.  Each call
// clears what must start at zero; the rest is written before it is read.
#include <mutex>

#include "ccl_device.cuh"

namespace fvv {
namespace {

constexpr int kNaMaxVoxels = 8 * 1024 * 1024;       // 8,388,608 coarse voxels
constexpr int kNaMaxComponents = kMaxComponents;    // 8192 raw components
// layout, in ints: [0] root count, [1] flags, [64 ..) roots, then parents per voxel
constexpr int kNaRoots = 64;
constexpr int kNaParent = (kNaRoots + kNaMaxComponents + 63) / 64 * 64;
constexpr int kScratchInts = kNaParent + kNaMaxVoxels;

static __device__ __align__(256) int g_na_scratch[kScratchInts];

struct NaGrid {
    const uint32_t* bits;
    int nx, ny, nz, nxw;
    int t_np, t_nb;
};

// Word w of the grid with the bits past nx cleared.
__device__ __forceinline__ uint32_t na_word(const NaGrid& g, uint32_t w) {
    const uint32_t word = __ldg(g.bits + w);
    const bool last = (g.nx & 31) && w % (uint32_t)g.nxw == (uint32_t)g.nxw - 1u;
    return last ? word & ((1u << (g.nx & 31)) - 1u) : word;
}

// The word at (wx, y, z), 0 outside the grid.
__device__ __forceinline__ uint32_t na_word_at(const NaGrid& g, int y, int z, int wx) {
    if (y < 0 || z < 0 || y >= g.ny || z >= g.nz || wx < 0 || wx >= g.nxw) return 0u;
    const uint32_t word = __ldg(g.bits + ((uint32_t)z * (uint32_t)g.ny + (uint32_t)y) * (uint32_t)g.nxw + (uint32_t)wx);
    return (g.nx & 31) && wx == g.nxw - 1 ? word & ((1u << (g.nx & 31)) - 1u) : word;
}

// Calls f(word, row, wx) for the words of the grid that are not empty, G lanes
// to a word, so that a lane can take a voxel (number lane % G of its word): a warp
// reads 32 words, a lane each, interleaved over the warps (lane l of warp k
// reads word base + l * nwarps + k), so that neighbouring words, which often
// belong to one object, are worked on by different warps.  G = 32 takes the words
// one at a time, the same in every lane; G < 32 is for rows of one word, of at
// most G voxels: 32 / G words at a time, some of which may be empty.
template <int G, class F>
__device__ __forceinline__ void na_for_words(const NaGrid& g, F&& f) {
    const uint32_t nwords = (uint32_t)g.nz * (uint32_t)g.ny * (uint32_t)g.nxw;
    const int lane = threadIdx.x & 31;
    const uint32_t nwarps = (gridDim.x * blockDim.x) >> 5, gw = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    for (uint32_t base = 0; base < nwords; base += nwarps * 32u) {
        const uint32_t mw = base + (uint32_t)lane * nwarps + gw;
        const uint32_t mine = mw < nwords ? na_word(g, mw) : 0u;
        uint32_t pending = __ballot_sync(kFull, mine != 0u);
        if constexpr (G < 32) {
            constexpr int kAtOnce = 32 / G;
#pragma unroll 1
            for (int q = 0; q < G && pending >> (q * kAtOnce); ++q) {
                const int src = q * kAtOnce + lane / G;
                const uint32_t word = __shfl_sync(kFull, mine, src);
                if (pending >> (q * kAtOnce) & (kFull >> (32 - kAtOnce))) f(word, base + (uint32_t)src * nwarps + gw, 0);
            }
        } else {
            for (; pending; pending &= pending - 1u) {
                const int src = __ffs(pending) - 1;
                const uint32_t w = base + (uint32_t)src * nwarps + gw;
                const uint32_t row = w / (uint32_t)g.nxw;
                f(__shfl_sync(kFull, mine, src), row, (int)(w - row * (uint32_t)g.nxw));
            }
        }
    }
}

// First voxel (bit) of the run of `word` that voxel b belongs to.
__device__ __forceinline__ int run_start(uint32_t word, int b) {
    const uint32_t starts = word & ~(word << 1);
    return 31 - __clz(starts & (0xFFFFFFFFu >> (31 - b)));
}

// Zero the counters, start a tree at each run of consecutive occupied voxels of
// a word, and a count at its first voxel.  `count` (the labels' array, written in
// full at the end) holds a component's voxels at its root.
template <int G>
__global__ void __launch_bounds__(256) k_na_seed(NaGrid g, int* sc, int32_t* __restrict__ count) {
    pdl_begin();
    if (blockIdx.x == 0 && threadIdx.x < 64) sc[threadIdx.x] = 0;
    int* parent = sc + kNaParent;
    const int b = threadIdx.x % G;
    na_for_words<G>(g, [&](uint32_t word, uint32_t row, int wx) {
        if (!((word >> b) & 1u)) return;
        const int first = (int)row * g.nx + wx * 32, run = run_start(word, b);
        parent[first + b] = first + run;
        if (run == b) count[first + b] = 0;
    });
}

// The unions of k_union (kernels_ccl.cu, where the rule is): runs across a word
// boundary, and with the four rows before that touch the row; a lane per voxel.
// A thread that walked 32 voxels through 13 neighbours each, one union after
// the other, took 318 us on a court-sized grid (400 x 220 x 80, 12 players and
// 2,000 stray voxels), this takes 24; the call 496 -> 63 us, and 10.1 ms -> 0.7
// on that grid with a quarter of its voxels occupied at random.
template <int G>
__global__ void __launch_bounds__(256) k_na_union(NaGrid g, int* sc) {
    pdl_begin();
    int* parent = sc + kNaParent;
    const int b = threadIdx.x % G;
    int budget = kStepBudget;
    na_for_words<G>(g, [&](uint32_t word, uint32_t row, int wx) {
        if (!((word >> b) & 1u) || budget <= 0) return;
        const int y = (int)(row % (uint32_t)g.ny), z = (int)(row / (uint32_t)g.ny);
        const int run = run_start(word, b), run0 = (int)row * g.nx + wx * 32 + run;
        if (b == 0 && (na_word_at(g, y, z, wx - 1) >> 31)) unite(parent, run0, run0 - 1, budget);
        for (int k = 0; k < 4; ++k) {
            const int dy = k == 0 ? -1 : k - 2, dz = k == 0 ? 0 : -1;
            const uint32_t n = na_word_at(g, y + dy, z + dz, wx);
            const bool left = b > 0 ? (n >> (b - 1)) & 1u : na_word_at(g, y + dy, z + dz, wx - 1) >> 31;
            const bool mid = (n >> b) & 1u;
            const bool right = b < 31 ? (n >> (b + 1)) & 1u : na_word_at(g, y + dy, z + dz, wx + 1) & 1u;
            const int nrow = ((z + dz) * g.ny + (y + dy)) * g.nx + wx * 32;
            if (run == b && (left || mid)) unite(parent, run0, nrow + (left ? b - 1 : b), budget);
            if (!mid && right) unite(parent, run0, nrow + b + 1, budget);
        }
    });
    if (budget <= 0) atomicOr(sc + 1, (int)FVV_FLAG_LOOP);
}

// Point every voxel at its root, list the roots and count each component's
// voxels.  A warp keeps the count of the component it met last, so that a
// large one costs it one atomic and not one a word.
template <int G>
__global__ void __launch_bounds__(256) k_na_compress(NaGrid g, int* sc, int32_t* __restrict__ count) {
    pdl_begin();
    int* parent = sc + kNaParent;
    const int lane = threadIdx.x & 31, b = threadIdx.x % G;
    int budget = kStepBudget, cur = -1, held = 0;   // cur, held: the same in every lane
    na_for_words<G>(g, [&](uint32_t word, uint32_t row, int wx) {
        const int L = (int)row * g.nx + wx * 32 + b;
        int r = -1;
        if (((word >> b) & 1u) && budget > 0) {
            r = find_root_readonly(parent, L, budget);
            if (r != L) parent[L] = r;
        }
        const uint32_t roots = __ballot_sync(kFull, r == L);
        if (roots) {
            int at = 0;
            if (lane == 0) at = atomicAdd(sc, __popc(roots));
            at = __shfl_sync(kFull, at, 0) + __popc(roots & ((1u << lane) - 1u));
            if (r == L && at < kNaMaxComponents) sc[kNaRoots + at] = L;
        }
        const uint32_t any = __ballot_sync(kFull, r >= 0);
        if (!any) return;
        const int lead = __shfl_sync(kFull, r, __ffs(any) - 1);
        const int n = __popc(__ballot_sync(kFull, r == lead));
        if (lead != cur) {
            if (lane == 0 && cur >= 0) atomicAdd(count + cur, held);
            cur = lead;
            held = 0;
        }
        held += n;
        const uint32_t same = __match_any_sync(kFull, r);
        if (r >= 0 && r != lead && lane == __ffs(same) - 1) atomicAdd(count + r, __popc(same));
    });
    if (lane == 0 && cur >= 0) atomicAdd(count + cur, held);
    if (budget <= 0) atomicOr(sc + 1, (int)FVV_FLAG_LOOP);
}

// Canonical labels: a kept component (t_np <= voxels <= t_nb) has label 1 + the
// number of kept ones with a smaller root, which is left in its root's parent
// entry as -(label + 1), a removed one's as -1.  Four lanes count for a root, a
// quarter of all kept roots each (8192 at most), 64 roots a block; a block that
// has none leaves.  (A bitonic sort in one block took 40 us for 2,200 roots.)
constexpr int kNaRankRoots = 64;
__global__ void __launch_bounds__(256) k_na_rank(NaGrid g, int* sc, const int32_t* __restrict__ count,
                                                 int32_t* __restrict__ counts) {
    pdl_begin();
    __shared__ __align__(16) int key[2048];
    __shared__ int sh[32];
    const int n = sc[0];
    const bool over = n > kNaMaxComponents;
    if (blockIdx.x > 0 && (over || (int)blockIdx.x * kNaRankRoots >= n)) return;   // the whole block
    int* parent = sc + kNaParent;
    const int i = blockIdx.x * kNaRankRoots + threadIdx.x / 4;
    const int root = !over && i < n ? sc[kNaRoots + i] : -1;
    int before = 0, kept = 0;
    bool keep = false;
    if (root >= 0) {
        const int c = __ldcg(count + root);
        keep = c >= g.t_np && c <= g.t_nb;
    }
    for (int t0 = 0; t0 < (over ? 0 : n); t0 += 2048) {
#pragma unroll
        for (int q = 0; q < 8; ++q) {
            const int k = (int)threadIdx.x + 256 * q;
            int v = 0x7FFFFFFF;                     // past the end, or removed: before nobody
            if (t0 + k < n) {
                const int r = sc[kNaRoots + t0 + k], c = __ldcg(count + r);
                if (c >= g.t_np && c <= g.t_nb) v = r;
            }
            key[k] = v;
            kept += v != 0x7FFFFFFF;
        }
        __syncthreads();
        const int m = min(2048, (n - t0 + 15) & ~15);
        for (int k = 4 * (threadIdx.x & 3); k < m; k += 16) {
            const int4 v = *reinterpret_cast<const int4*>(key + k);
            before += (v.x < root) + (v.y < root) + (v.z < root) + (v.w < root);
        }
        __syncthreads();
    }
    before += __shfl_xor_sync(kFull, before, 1);
    before += __shfl_xor_sync(kFull, before, 2);
    if (root >= 0 && (threadIdx.x & 3) == 0) parent[root] = keep ? -(before + 2) : -1;
    const int total = block_sum<int>(kept, sh);
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        counts[0] = n;
        counts[1] = total;
        counts[2] = sc[1] | (over ? (int)FVV_FLAG_ROOTS : 0);
    }
}

// Every voxel of the output: its canonical label, 0 for empty or removed.  A
// warp takes 32 words, a lane per voxel of each, so that a word's labels go out
// in one piece; of rows of one word (G < 32) a lane per voxel of all of them,
// whose labels follow one another.
template <int G>
__global__ void __launch_bounds__(256) k_na_labels(NaGrid g, const int* sc, int32_t* __restrict__ labels) {
    pdl_begin();
    const int* parent = sc + kNaParent;
    const uint32_t nwords = (uint32_t)g.nz * (uint32_t)g.ny * (uint32_t)g.nxw;
    const int lane = threadIdx.x & 31;
    const uint32_t nwarps = (gridDim.x * blockDim.x) >> 5;
    for (uint32_t base = ((blockIdx.x * blockDim.x + threadIdx.x) >> 5) * 32u; base < nwords; base += nwarps * 32u) {
        const uint32_t mw = base + (uint32_t)lane;
        const uint32_t mine = mw < nwords ? na_word(g, mw) : 0u;
        auto put = [&](uint32_t word, int b, int L) {
            int lab = 0;
            if ((word >> b) & 1u) {
                const int r = __ldg(parent + L), t = r < 0 ? r : __ldg(parent + r);
                lab = t < 0 ? -t - 1 : 0;           // else: roots were not tagged (too many components)
            }
            __stcs(labels + L, lab);
        };
        const int m = (int)min(32u, nwords - base);
        if constexpr (G < 32) {
            for (int i0 = 0; i0 < m * g.nx; i0 += 32) {
                const int i = i0 + lane, k = min(i / g.nx, 31);
                const uint32_t word = __shfl_sync(kFull, mine, k);
                if (i < m * g.nx) put(word, i - k * g.nx, (int)base * g.nx + i);
            }
            continue;
        }
        const uint32_t row = min(mw, nwords - 1u) / (uint32_t)g.nxw;
        const int x0 = (int)(min(mw, nwords - 1u) - row * (uint32_t)g.nxw) * 32;
        const int first = (int)row * g.nx + x0, nv = min(32, g.nx - x0);
#pragma unroll 4
        for (int k = 0; k < m; ++k) {
            const uint32_t word = __shfl_sync(kFull, mine, k);
            const int L = __shfl_sync(kFull, first, k) + lane;
            if (lane < __shfl_sync(kFull, nv, k)) put(word, lane, L);
        }
    }
}

// The call's five kernels, G lanes to a word.
template <int G>
void na_launch(const NaGrid& g, int* sc, int32_t* labels, int32_t* counts, unsigned blocks, cudaStream_t st) {
    const dim3 ranks(kNaMaxComponents / kNaRankRoots);
    // Dependent launch hides the gaps between a small grid's kernels (3,600 words: 44
    // us without and 35 with it; 39,000: 38 and 30; 84,000: 45 and 42); a large
    // one's run slower with it, as the next kernel's waiting blocks take room on the
    // SMs (140,000: 44 and 46; 229,000: 51 and 61).  They are even at some 130,000
    // words; the line lies at 65,536, where the blocks stop growing with the grid.
    if (blocks < 2048) {
        launch_pdl(k_na_seed<G>, dim3(blocks), dim3(256), 0, st, g, sc, labels);
        launch_pdl(k_na_union<G>, dim3(blocks), dim3(256), 0, st, g, sc);
        launch_pdl(k_na_compress<G>, dim3(blocks), dim3(256), 0, st, g, sc, labels);
        launch_pdl(k_na_rank, ranks, dim3(256), 0, st, g, sc, labels, counts);
        launch_pdl(k_na_labels<G>, dim3(blocks), dim3(256), 0, st, g, sc, labels);
    } else {
        k_na_seed<G><<<blocks, 256, 0, st>>>(g, sc, labels);
        k_na_union<G><<<blocks, 256, 0, st>>>(g, sc);
        k_na_compress<G><<<blocks, 256, 0, st>>>(g, sc, labels);
        k_na_rank<<<ranks, 256, 0, st>>>(g, sc, labels, counts);
        k_na_labels<G><<<blocks, 256, 0, st>>>(g, sc, labels);
    }
}

std::mutex g_na_mutex;
int* g_na_ptr[256] = {};   // device address of g_na_scratch, per device ordinal

}  // namespace
}  // namespace fvv

using namespace fvv;

extern "C" fvv_status fvv_label_components_noalloc(const uint32_t* coarse_bits, int nx, int ny, int nz, int t_np,
                                                   int t_nb, int32_t* labels, int32_t* counts, void* stream) {
    if (!coarse_bits || !labels || !counts) return FVV_ERR_INVALID_ARG;
    if (nx < 1 || ny < 1 || nz < 1) return FVV_ERR_INVALID_ARG;
    if ((long long)nx * ny * nz > kNaMaxVoxels) return FVV_ERR_INVALID_ARG;   // beyond the static scratch
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 256) return FVV_ERR_CUDA;
    int* sc = nullptr;
    {
        std::lock_guard<std::mutex> lock(g_na_mutex);
        if (!g_na_ptr[dev]) {
            void* p = nullptr;
            if (cudaGetSymbolAddress(&p, g_na_scratch) != cudaSuccess || !p) return FVV_ERR_CUDA;
            g_na_ptr[dev] = static_cast<int*>(p);
        }
        sc = g_na_ptr[dev];
    }
    const cudaStream_t st = static_cast<cudaStream_t>(stream);
    NaGrid g{coarse_bits, nx, ny, nz, (nx + 31) / 32, t_np, t_nb};
    const long long words = (long long)nz * ny * g.nxw;
    // four words a warp, so that a small grid's objects are spread over many, up to 2048 blocks
    const unsigned blocks = (unsigned)std::max(1LL, std::min((words + 31) / 32, 2048LL));
    // Rows of up to four voxels are taken several words at a time: one at a time, a
    // warp has one to four lanes at work, where a thread per word had them all
    // (nx = 1, 7.8 million words, 30% occupied: 859 us with a thread per word, 2120
    // one word at a time, 601 with a lane a word; 0.04% occupied: 142, 281 and 146;
    // nx = 4, 2 million words, 2%: 202, 246 and 165).  From five voxels on a warp on
    // one word is the faster of the first two everywhere (nx = 6: 263 and 211 us).
    if (nx == 1) na_launch<1>(g, sc, labels, counts, blocks, st);
    else if (nx == 2) na_launch<2>(g, sc, labels, counts, blocks, st);
    else if (nx <= 4) na_launch<4>(g, sc, labels, counts, blocks, st);
    else na_launch<32>(g, sc, labels, counts, blocks, st);
    return cudaGetLastError() == cudaSuccess ? FVV_OK : FVV_ERR_CUDA;
}
