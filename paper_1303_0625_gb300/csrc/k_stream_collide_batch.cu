// The fused kernel over a batch of independent domains (cases): the tiles of every
// active case in one launch, each with its own case's parameters.  A tile is a run of
// row segments (32 lanes x V nodes, rows in order), one per warp, tile_h per warp: a
// block works on as many rows as its warps need.  With tiles of one row and 128 threads
// half of a block had no nodes on rows of 256 (V = 4), and part of the last block of
// every row elsewhere: 96 open channels of 256 x 128, FP32, one launch 58 us, now 47
// (its bytes at the copy rate: 34); 512 channels of 128 to 1024 x 64 to 512, 1125 us,
// now 1099 (972).  What is left between a launch and its bytes: the two dependent loads
// (tile, case) before a block's populations.  The device code is in
// k_stream_collide.cuh.
#include "k_stream_collide.cuh"

namespace gbm {

namespace {

constexpr int SC_WARPS = SC_BLOCK_X / 32;

// This warp's row segments of one tile {case, first segment, its row, segments per row}.
// The force kernel of the step has swapped the buffers: f1 holds the current populations,
// f0 takes the next.
template <int P, int V, bool FORCE, bool LOCAL>
__device__ __forceinline__ void tile_segments(const StepParams &p, const int4 &tl, int tile_h) {
    using R = typename Raw<P>::R;
    int seg = tl.y + (threadIdx.x >> 5), y = tl.z;
    for (int h = 0; h < tile_h; h++, seg += SC_WARPS) {
        for (; seg >= tl.w; seg -= tl.w) y++;
        if (y >= p.L.ny) return;
        const R *fin = static_cast<const R *>(p.f1);
        R *fout = static_cast<R *>(p.f0);
        const int x0 = (seg * 32 + (threadIdx.x & 31)) * V;
        if constexpr (P == LBM_FP16_DEV) sc_tile<V, FORCE, LOCAL, true>(p, fin, fout, x0, y);
        else if (p.L.bc_x == LBM_OPEN) sc_row<P, V, FORCE, true, 0>(p, fin, fout, x0, y);
        else sc_row<P, V, FORCE, false, 0>(p, fin, fout, x0, y);
    }
}

// Persistent blocks walk the list of the active tiles of all cases (case-major).
template <int P, int V, bool FORCE, bool LOCAL>
__global__ void __launch_bounds__(SC_BLOCK_X, 6)
    k_stream_collide_batch(const StepParams *__restrict__ cases, const int4 *__restrict__ tiles,
                           const int *__restrict__ ntiles, int tile_h) {
    const int n = *ntiles;
    for (int k = blockIdx.x; k < n; k += gridDim.x) {
        const int4 tl = tiles[k];
        tile_segments<P, V, FORCE, LOCAL>(cases[tl.x], tl, tile_h);
    }
}

// The same tiles with one block per tile (grid = capacity of the list).
// FP32 with 4- or 8-byte words: at most 48 registers (10 blocks per SM), at the
// cost of a few bytes of spills.
template <int P, int V>
constexpr int tiles_min_blocks() { return (P == LBM_FP32_DEV && V <= 2) ? 10 : 6; }

template <int P, int V, bool FORCE, bool LOCAL, bool ROWS>
__global__ void __launch_bounds__(SC_BLOCK_X, (tiles_min_blocks<P, V>()))
    k_stream_collide_tiles(const StepParams *__restrict__ cases, const int4 *__restrict__ tiles,
                           const int *__restrict__ ntiles, int tile_h) {
    if ((int)blockIdx.x >= *ntiles) return;
    const int4 tl = tiles[blockIdx.x];
    tile_segments<P, V, FORCE, LOCAL>(cases[tl.x], tl, ROWS ? tile_h : 1);
}

template <int P, int V, bool FORCE, bool LOCAL>
cudaError_t launch_scb(const BatchLaunch &b, cudaStream_t st) {
    static int per_sm = -1, sms = 0;
    if (per_sm < 0) {
        int dev = 0;
        cudaError_t e = cudaGetDevice(&dev);
        if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
        if (e == cudaSuccess)
            e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(
                &per_sm, k_stream_collide_batch<P, V, FORCE, LOCAL>, SC_BLOCK_X, 0);
        if (e != cudaSuccess) return e;
    }
    if (b.persistent)
        k_stream_collide_batch<P, V, FORCE, LOCAL>
            <<<per_sm * sms, SC_BLOCK_X, 0, st>>>(b.cases, b.tiles, b.ntiles, b.tile_h);
    else if (b.max_tiles > 0 && b.tile_h == 1)
        k_stream_collide_tiles<P, V, FORCE, LOCAL, false>
            <<<b.max_tiles, SC_BLOCK_X, 0, st>>>(b.cases, b.tiles, b.ntiles, 1);
    else if (b.max_tiles > 0)
        k_stream_collide_tiles<P, V, FORCE, LOCAL, true>
            <<<b.max_tiles, SC_BLOCK_X, 0, st>>>(b.cases, b.tiles, b.ntiles, b.tile_h);
    return cudaGetLastError();
}

template <int P, int V>
cudaError_t launch_scb_v(const BatchLaunch &b, cudaStream_t st) {
    // FP64 and FP32 need rho_w only in wall rows (a run-time branch of sc_row)
    const bool local = P == LBM_FP16_DEV && b.local;
    if (b.force)
        return local ? launch_scb<P, V, true, P == LBM_FP16_DEV>(b, st) : launch_scb<P, V, true, false>(b, st);
    return local ? launch_scb<P, V, false, P == LBM_FP16_DEV>(b, st) : launch_scb<P, V, false, false>(b, st);
}

template <int P>
cudaError_t launch_scb_p(const BatchLaunch &b, cudaStream_t st) {
    constexpr int V16 = 16 / (int)sizeof(typename Raw<P>::R);
    switch (b.variant) {
        case 1: return launch_scb_v<P, V16 / 2>(b, st);
        case 2: return launch_scb_v<P, (V16 / 4 > 0 ? V16 / 4 : 1)>(b, st);
        default: return launch_scb_v<P, V16>(b, st);
    }
}

}  // namespace

int segment_nodes(int precision, int variant) {
    const int v16 = precision == LBM_FP64 ? 2 : (precision == LBM_FP32_DEV ? 4 : 8);
    const int v = variant == 1 ? v16 / 2 : (variant == 2 ? (v16 / 4 > 0 ? v16 / 4 : 1) : v16);
    return 32 * v;
}

int tile_segments(int tile_h) { return SC_WARPS * tile_h; }

cudaError_t launch_stream_collide_batch(const BatchLaunch &b, cudaStream_t st) {
    switch (b.precision) {
        case LBM_FP64: return launch_scb_p<LBM_FP64>(b, st);
        case LBM_FP32_DEV: return launch_scb_p<LBM_FP32_DEV>(b, st);
        default: return launch_scb_p<LBM_FP16_DEV>(b, st);
    }
}

}  // namespace gbm
