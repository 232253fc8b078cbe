// Fused pull-advection + bounce-back + collision (Eq. 1-3, Eq. 8) on one domain.
// The device code is in k_stream_collide.cuh: sc_row for FP64 and FP32 storage
// (after the force kernel, which leaves the returned populations in the solid
// nodes' slots), sc_tile for FP16.
#include "k_stream_collide.cuh"

namespace gbm {

namespace {

// Blocks on an SM, of BGK without a body force: for at most 80 registers a thread with
// 16-byte words, 56 (FP64) or 48 with 8, 32 with 4.  (With 84 and 94, one block less: a
// step of the FP64 channel of 1200 x 120 nodes 38.1 us, now 35.2; 2048 x 1024 nodes in
// FP32 24.7, now 23.5.)
template <int P, int V, bool FORCE, bool OPEN, int COLL>
constexpr int row_blocks() {
    constexpr int bytes = V * (int)sizeof(typename Raw<P>::R);
    return FORCE || OPEN || COLL ? 0 : (bytes == 16 ? 6 : (bytes == 4 ? 16 : (P == LBM_FP64 ? 9 : 10)));
}

// One block per SC_BLOCK_X * V nodes of a row.
template <int P, int V, bool FORCE, bool OPEN, int COLL>
__global__ void __launch_bounds__(SC_BLOCK_X, (row_blocks<P, V, FORCE, OPEN, COLL>())) k_stream_collide(const StepParams p) {
    early_start();
    using R = typename Raw<P>::R;
    const long long t = *p.t;
    sc_row<P, V, FORCE, OPEN, COLL>(p, static_cast<const R *>((t & 1) ? p.f1 : p.f0),
                                    static_cast<R *>((t & 1) ? p.f0 : p.f1),
                                    (blockIdx.x * SC_BLOCK_X + threadIdx.x) * V, blockIdx.y);
    if (P == LBM_FP32_DEV && p.sc_last) end_of_step(p, t, gridDim.x * gridDim.y);
}

template <int V, bool FORCE, bool LOCAL, bool DEFER, int COLL = 0, bool BND = false>
__global__ void __launch_bounds__(SC_BLOCK_X) k_stream_collide16(const StepParams p) {
    using R = Raw<LBM_FP16_DEV>::R;
    const long long t = *p.t;
    sc_tile<V, FORCE, LOCAL, false, DEFER, COLL, BND>(
        p, static_cast<const R *>((t & 1) ? p.f1 : p.f0), static_cast<R *>((t & 1) ? p.f0 : p.f1),
        (blockIdx.x * SC_BLOCK_X + threadIdx.x) * V, blockIdx.y);
}

// FP16 with the per-node path deferred (variants 3-5): the nodes that
// k_stream_collide16 leaves to the per-node update (update_node) are computed
// from the same populations after it, by k_boundary_update: one thread per node
// of the step's list of fluid nodes next to solids, then of the first and last
// columns and of the wall rows.  The force kernel of the step fills the list: it
// visits every fluid node with a link into its solid (one atomic per warp and
// list chunk).  The list's length is kept per step parity; the update kernel of
// step t clears the slot of step t + 1.  A node next to two disks is computed
// twice, with identical results.  Inline in the vector path these nodes run with
// one or two active lanes per warp; which way is faster depends on the workload
// (the autotuner measures both).
constexpr int BN_BLOCK = 256;

__host__ __device__ inline long long boundary_edge_nodes(const Lattice &L) {
    long long n = L.nx > 1 ? 2LL * L.ny : (long long)L.ny;
    if (L.bc_y == LBM_WALL && L.nx > 2) n += 2LL * (L.nx - 2);
    return n;
}

template <bool FORCE, bool LOCAL, bool BND>
__global__ void __launch_bounds__(BN_BLOCK) k_boundary_update(const StepParams p) {
    using R = Raw<LBM_FP16_DEV>::R;
    const Lattice &L = p.L;
    const long long t = *p.t;
    const R *fin = static_cast<const R *>((t & 1) ? p.f1 : p.f0);
    R *fout = static_cast<R *>((t & 1) ? p.f0 : p.f1);
    const int nlist = (p.nsolid > 0 && p.bnd) ? min(p.bnd[t & 1], p.bnd_cap) : 0;
    const int ncol = L.nx > 1 ? 2 * L.ny : L.ny;
    const long long total = nlist + boundary_edge_nodes(L);
    for (long long e = (long long)blockIdx.x * BN_BLOCK + threadIdx.x; e < total;
         e += (long long)gridDim.x * BN_BLOCK) {
        int x, y;
        if (e < nlist) {
            const int k = p.bnd[2 + e];
            x = k % L.pitch;
            y = k / L.pitch;
        } else if (e < nlist + ncol) {
            const int c = (int)(e - nlist);
            y = L.nx > 1 ? c >> 1 : c;
            x = (L.nx > 1 && (c & 1)) ? L.nx - 1 : 0;
        } else {
            const int c = (int)(e - nlist - ncol), w = L.nx - 2;
            y = c < w ? 0 : L.ny - 1;
            x = 1 + (c < w ? c : c - w);
        }
        if (!(p.flags[cell_of(L, x, y)] & 1u))
            update_node<FORCE, LOCAL, false, 0, BND>(p, fin, fout, x, y);
    }
    if (blockIdx.x == 0 && threadIdx.x == 0 && p.bnd) p.bnd[(t + 1) & 1] = 0;
}

// FP16: open-channel columns of every row, on the populations of t+1.
template <bool FORCE>
__global__ void k_open_columns(const StepParams p) {
    using R = Raw<LBM_FP16_DEV>::R;
    const int y = blockIdx.x * blockDim.x + threadIdx.x;
    if (y >= p.L.ny) return;
    const long long t = *p.t;
    open_row<FORCE>(p, static_cast<R *>((t & 1) ? p.f0 : p.f1), y);
}

// ------------------------------------------------------------ FP64, FP32

template <int P, int V, bool FORCE, int COLL>
cudaError_t launch_row(const StepParams &p, cudaStream_t st) {
    const dim3 grid((p.L.nx + SC_BLOCK_X * V - 1) / (SC_BLOCK_X * V), p.L.ny);
    if (p.L.bc_x == LBM_OPEN)
        return launch_step(p, k_stream_collide<P, V, FORCE, true, COLL>, grid, SC_BLOCK_X, st, p);
    return launch_step(p, k_stream_collide<P, V, FORCE, false, COLL>, grid, SC_BLOCK_X, st, p);
}

template <int P, int V>
cudaError_t launch_row_v(const StepParams &p, cudaStream_t st) {
    if (p.body_x != 0.0 || p.body_y != 0.0) return launch_row<P, V, true, 0>(p, st);
    return launch_row<P, V, false, 0>(p, st);
}

// Node widths per thread: variants 0 and 3 one 16-byte word per population,
// 1 and 4 8 bytes, 2 and 5 4 bytes (FP64: one node).  MRT: 8-byte words.
template <int P>
cudaError_t launch_row_p(const StepParams &p, cudaStream_t st) {
    constexpr int V16 = 16 / (int)sizeof(typename Raw<P>::R);
    constexpr int V4 = V16 / 4 > 0 ? V16 / 4 : 1;
    if (p.collision == LBM_MRT) return launch_row<P, V16 / 2, false, 1>(p, st);
    switch (p.sc_variant % 3) {
        case 1: return launch_row_v<P, V16 / 2>(p, st);
        case 2: return launch_row_v<P, V4>(p, st);
        default: return launch_row_v<P, V16>(p, st);
    }
}

// ------------------------------------------------------------------ FP16

// The update kernel of the deferred per-node path, over the list of step t.
template <bool FORCE, bool LOCAL>
cudaError_t launch_update(const StepParams &p, cudaStream_t st) {
    cudaError_t e = cudaSuccess;
    static int sms = 0;
    if (!sms) {
        int dev = 0;
        e = cudaGetDevice(&dev);
        if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
        if (e != cudaSuccess) return e;
    }
    const long long most = (p.nsolid > 0 ? p.bnd_cap : 0) + boundary_edge_nodes(p.L);
    long long blocks = (most + BN_BLOCK - 1) / BN_BLOCK;
    if (blocks > 8LL * sms) blocks = 8LL * sms;
    if (blocks < 1) blocks = 1;
    if (p.boundary == LBM_INTERPOLATED)
        k_boundary_update<FORCE, LOCAL, true><<<(unsigned)blocks, BN_BLOCK, 0, st>>>(p);
    else
        k_boundary_update<FORCE, LOCAL, false><<<(unsigned)blocks, BN_BLOCK, 0, st>>>(p);
    return cudaGetLastError();
}

template <int V, bool FORCE, bool LOCAL, bool DEFER>
cudaError_t launch_sc(const StepParams &p, cudaStream_t st) {
    const dim3 grid((p.L.nx + SC_BLOCK_X * V - 1) / (SC_BLOCK_X * V), p.L.ny);
    k_stream_collide16<V, FORCE, LOCAL, DEFER><<<grid, SC_BLOCK_X, 0, st>>>(p);
    cudaError_t e = cudaGetLastError();
    // with solids, the force kernel lists the nodes next to them and the
    // host launches the update after it (launch_deferred_update)
    if (e != cudaSuccess || !DEFER || p.list_by_forces) return e;
    return launch_update<FORCE, LOCAL>(p, st);
}

template <int V, bool DEFER>
cudaError_t launch_sc_v(const StepParams &p, cudaStream_t st) {
    const bool force = p.body_x != 0.0 || p.body_y != 0.0;
    const bool local = p.rho_w_mode == LBM_RHOW_LOCAL;
    if (force)
        return local ? launch_sc<V, true, true, DEFER>(p, st) : launch_sc<V, true, false, DEFER>(p, st);
    return local ? launch_sc<V, false, true, DEFER>(p, st) : launch_sc<V, false, false, DEFER>(p, st);
}

// MRT: one launch shape, 8-byte words per population plane, slow nodes inline.
template <bool LOCAL, bool BND>
cudaError_t launch_mrt16(const StepParams &p, cudaStream_t st) {
    constexpr int V = 4;
    const dim3 grid((p.L.nx + SC_BLOCK_X * V - 1) / (SC_BLOCK_X * V), p.L.ny);
    k_stream_collide16<V, false, LOCAL, false, 1, BND><<<grid, SC_BLOCK_X, 0, st>>>(p);
    return cudaGetLastError();
}

// Node widths as for FP32; variants 3-5 with the per-node path deferred to
// k_boundary_update (always, with the interpolated boundary).
cudaError_t launch_sc16(const StepParams &p, cudaStream_t st) {
    if (p.collision == LBM_MRT) {
        const bool local = p.rho_w_mode == LBM_RHOW_LOCAL;
        if (p.boundary == LBM_INTERPOLATED)
            return local ? launch_mrt16<true, true>(p, st) : launch_mrt16<false, true>(p, st);
        return local ? launch_mrt16<true, false>(p, st) : launch_mrt16<false, false>(p, st);
    }
    switch (p.boundary == LBM_INTERPOLATED && p.sc_variant < 3 ? p.sc_variant + 3 : p.sc_variant) {
        case 1: return launch_sc_v<4, false>(p, st);
        case 2: return launch_sc_v<2, false>(p, st);
        case 3: return launch_sc_v<8, true>(p, st);
        case 4: return launch_sc_v<4, true>(p, st);
        case 5: return launch_sc_v<2, true>(p, st);
        default: return launch_sc_v<8, false>(p, st);
    }
}

}  // namespace

cudaError_t launch_stream_collide(const StepParams &p, cudaStream_t st) {
    switch (p.precision) {
        case LBM_FP64: return launch_row_p<LBM_FP64>(p, st);
        case LBM_FP32_DEV: return launch_row_p<LBM_FP32_DEV>(p, st);
        default: return launch_sc16(p, st);
    }
}

cudaError_t launch_deferred_update(const StepParams &p, cudaStream_t st) {
    const bool force = p.body_x != 0.0 || p.body_y != 0.0;
    const bool local = p.rho_w_mode == LBM_RHOW_LOCAL;
    if (force) return local ? launch_update<true, true>(p, st) : launch_update<true, false>(p, st);
    return local ? launch_update<false, true>(p, st) : launch_update<false, false>(p, st);
}

cudaError_t launch_open_columns(const StepParams &p, cudaStream_t st) {
    const dim3 grid((p.L.ny + 127) / 128);
    if (p.body_x != 0.0 || p.body_y != 0.0) k_open_columns<true><<<grid, 128, 0, st>>>(p);
    else k_open_columns<false><<<grid, 128, 0, st>>>(p);
    return cudaGetLastError();
}

}  // namespace gbm
