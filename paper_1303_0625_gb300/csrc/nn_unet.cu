// The warm-start U-Net on the GPU: forward, backward and Adam, with every 3x3
// convolution an implicit GEMM on the tensor cores (tcgen05, BF16 operands, FP32
// accumulation in tensor memory).  The remaining layers (pooling, the 1x1 head, the
// loss, Adam) are small kernels of their own.
//
// Layout: activations and their gradients are planes of 8 channels,
// X[C / 8][B][H + 2][W + 2][8] in BF16, with a border of zeros that is written once
// (a plane's image stride is rounded up to 128 pixels).  A pixel of a plane is 16
// bytes and pixels are consecutive, so a run of pixels is one bulk copy, and in
// shared memory it is, as it stands, the no-swizzle core-matrix layout of
// tcgen05.mma: 8 pixels x 8 channels = 128 bytes, the next 8 pixels behind them.  A
// tap's displacement is then a shift of the operand's start address by (dy (W + 2)
// + dx) pixels of 16 bytes, borders included, and no operand is gathered: the
// convolutions copy each input pixel once per output tile instead of once per tap
// (with NHWC and one 16-byte cp.async per pixel, tap and 8 channels, they ran at 6%
// of the tensor cores' rate).
//
// Convolutions as GEMMs over the padded pixels Q = (b, y, x) of all images (rows
// that are border pixels are computed and not stored):
//   forward      out[Q][co]  = sum_{tap,ci} x[Q + s(tap)][ci] w[co][tap][ci]      M=Q  N=Cout K=9 Cin
//   data grad    dx[Q][ci]   = sum_{tap,co} dz[Q - s(tap)][co] w[co][tap][ci]     M=Q  N=Cin  K=9 Cout
//   weight grad  dw[tap][ci][co] = sum_Q x[Q + s(tap)][ci] dz[Q][co]  M=(dy, ci)  N=Cout K=Q, one per dx
// s(tap) = (tap / 3 - 1, tap % 3 - 1).  The weight gradient splits K over blocks, whose
// FP32 partial sums are added in a fixed order (k_sum_parts): nothing in a training step
// depends on the order in which blocks come to an end, so that it can be repeated bit
// for bit.
//
// Weights: FP32 masters, gradients and Adam moments [tap][Cin][Cout]; BF16 copies
// packed as the B operands of the forward and data-gradient convolutions (packed_at).
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <cmath>
#include <cstdarg>
#include <cstddef>
#include <cstdio>
#include <cstring>
#include <random>
#include <string>
#include <vector>

#include "lbm_nn.h"

namespace nn {

using bf16 = __nv_bfloat16;

// ------------------------------------------------------------- layout

// One level's images: H x W pixels with a border of one, PSI pixels per image.
struct Geo {
    int H, W, Wp, PSI;
    __host__ __device__ Geo() : H(0), W(0), Wp(0), PSI(0) {}
    __host__ __device__ Geo(int h, int w) : H(h), W(w), Wp(w + 2), PSI(((h + 2) * (w + 2) + 127) / 128 * 128) {}
    // pixel (n, y, x)
    __host__ __device__ long long at(int n, int y, int x) const {
        return (long long)n * PSI + (long long)(y + 1) * Wp + x + 1;
    }
    // interior pixel of Q, or false
    __device__ __forceinline__ bool where(int Q, int B, int &n, int &y, int &x) const {
        n = Q / PSI;
        const int r = Q - n * PSI;
        y = r / Wp - 1;
        x = r - (y + 1) * Wp - 1;
        return n < B && (unsigned)y < (unsigned)H && (unsigned)x < (unsigned)W;
    }
};

// 8-channel groups of the K axis of a convolution with G source groups: taps come in
// pairs of groups (K = 16 an instruction), so an odd G gets one more group of zeros,
// unless one group is all (the input layer): there two taps share a pair, the last with
// zeros.  Zeros on both sides: an infinity times a zero weight is not a number.
__host__ __device__ inline int k_groups(int G, bool pair_taps) {
    return pair_taps ? 10 : 9 * (G + (G & 1));
}
// N tile of a convolution with N outputs, and their number
__host__ __device__ inline int n_tiles(int N) { return (N + 127) / 128; }
__host__ __device__ inline int n_tile(int N) {
    return ((N + n_tiles(N) - 1) / n_tiles(N) + 31) / 32 * 32;
}
// Element of the packed B operand [N tile][K group][n][8]: output n, tap, source
// channel c; KG groups, Ge of them per tap.
__host__ __device__ inline long long packed_at(int n, int tap, int c, int BN, int KG, int Ge) {
    return (((long long)(n / BN) * KG + tap * Ge + c / 8) * BN + n % BN) * 8 + c % 8;
}

// 8 channels of a pixel
__device__ __forceinline__ void unpack8(const uint4 &v, float (&f)[8]) {
    const __nv_bfloat162 *h = reinterpret_cast<const __nv_bfloat162 *>(&v);
#pragma unroll
    for (int j = 0; j < 4; j++) {
        const float2 t = __bfloat1622float2(h[j]);
        f[2 * j] = t.x;
        f[2 * j + 1] = t.y;
    }
}
__device__ __forceinline__ uint4 pack8(const float (&f)[8]) {
    uint4 v;
    __nv_bfloat162 *h = reinterpret_cast<__nv_bfloat162 *>(&v);
#pragma unroll
    for (int j = 0; j < 4; j++) h[j] = __floats2bfloat162_rn(f[2 * j], f[2 * j + 1]);
    return v;
}

// The forward pass is a chain of about twenty kernels of 6 to 45 us.  Each but the first
// is launched early: once all blocks of a convolution have issued their last copies, the
// next kernel's blocks take the places that fall free, set up their barriers and TMEM and
// fetch their weights, and early_wait holds what reads or writes the layers until the one
// ahead has ended.  (What the first kernel waits for, as any launch, is complete for the
// chain: the weights too.)  16 images of 128 x 256: a pass 292 -> 290 us behind other
// work, 417 -> 367 from an idle GPU, four training steps 5.30 -> 5.10 ms; with the next
// kernel let in at a convolution's start the weights' copies got in the way (296 us).
__device__ __forceinline__ void early_next() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void early_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

// ------------------------------------------------ tcgen05 convolution

constexpr int TC_M = 128;
constexpr int TC_THREADS = 224;  // warps: A, MMA, four for the epilogue, B
constexpr int WG_THREADS = 192;  // copies, MMA, four for the bias gradient and the epilogue
constexpr int TC_MAX_STAGES = 10, TC_MAX_A = 12;
constexpr int TC_KB = 24;                // K groups of 8 channels per stage of B, at most
constexpr long long TC_SPIN = 1 << 24;

__device__ __forceinline__ uint32_t smem_u32(const void *p) {
    return (uint32_t)__cvta_generic_to_shared(p);
}

// Shared-memory matrix descriptor without swizzle: `lead` bytes between K groups
// (8 channels, or 8 pixels when K is the pixels), `stride` bytes between groups of 8
// rows (pixels, outputs, or channels).
__device__ __forceinline__ uint32_t desc_lo(uint32_t addr, uint32_t lead) { return addr >> 4 | lead >> 4 << 16; }
__host__ __device__ constexpr uint32_t desc_hi(uint32_t stride) { return stride >> 4 | 1u << 14; }

// Waits for phase `parity` of an mbarrier, at most `limit` polls.
__device__ __forceinline__ bool tc_wait(uint32_t mbar, uint32_t parity, long long limit) {
    uint32_t done = 0;
    for (long long it = 0; it < limit && !done; it++)
        asm volatile(
            "{\n.reg .pred p;\nmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n"
            "selp.u32 %0, 1, 0, p;\n}\n"
            : "=r"(done)
            : "r"(mbar), "r"(parity)
            : "memory");
    return done != 0;
}

__device__ __forceinline__ void mbar_init(uint32_t mbar, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;\n" ::"r"(mbar), "r"(count));
}
__device__ __forceinline__ void mbar_expect(uint32_t mbar, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;\n" ::"r"(mbar), "r"(bytes)
                 : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint32_t mbar) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];\n" ::"r"(mbar) : "memory");
}
// contiguous global -> shared copy (16-byte aligned, a multiple of 16 bytes)
__device__ __forceinline__ void bulk_copy(uint32_t dst, const void *src, uint32_t bytes, uint32_t mbar) {
    asm volatile(
        "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];\n" ::"r"(dst),
        "l"(src), "r"(bytes), "r"(mbar)
        : "memory");
}
// the mbarrier completes a phase when every MMA this thread issued has
__device__ __forceinline__ void tc_commit(uint32_t mbar) {
    asm volatile(
        "tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n" ::"r"(mbar)
        : "memory");
}
__device__ __forceinline__ void tc_alloc(uint32_t *slot, int ncols) {  // one warp
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;\n" ::"r"(smem_u32(slot)),
                 "r"(ncols));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;\n");
}
__device__ __forceinline__ void tc_free(uint32_t tmem, int ncols, int warp) {
    asm volatile("tcgen05.fence::before_thread_sync;\n");
    __syncthreads();
    if (warp == 0)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;\n" ::"r"(tmem), "r"(ncols));
}

// 32 consecutive FP32 accumulator columns of this warp's 32 TMEM lanes
__device__ __forceinline__ void tc_ld32(uint32_t addr, float (&f)[32]) {
    uint32_t v[32];
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,"
        "%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];\n"
        "tcgen05.wait::ld.sync.aligned;\n"
        : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]),
          "=r"(v[8]), "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]), "=r"(v[14]),
          "=r"(v[15]), "=r"(v[16]), "=r"(v[17]), "=r"(v[18]), "=r"(v[19]), "=r"(v[20]), "=r"(v[21]),
          "=r"(v[22]), "=r"(v[23]), "=r"(v[24]), "=r"(v[25]), "=r"(v[26]), "=r"(v[27]), "=r"(v[28]),
          "=r"(v[29]), "=r"(v[30]), "=r"(v[31])
        : "r"(addr));
#pragma unroll
    for (int j = 0; j < 32; j++) f[j] = __uint_as_float(v[j]);
}

// one lane of the calling warp
__device__ __forceinline__ bool elect_one() {
    uint32_t p;
    asm volatile("{\n.reg .pred p;\nelect.sync _|p, 0xffffffff;\nselp.u32 %0, 1, 0, p;\n}\n" : "=r"(p));
    return p != 0;
}

// One MMA from the low words of its descriptors (address and leading stride) and their
// common high words (stride between row groups).  The issuing warp's own instructions
// are in series, and the MMA takes its operands from uniform registers: the whole warp
// runs the loops, on values that are uniform by construction, and one lane issues.
// (One thread, with tap offsets from shared memory, issued an MMA in 200 cycles, where
// one takes 50 to 64.)
__device__ __forceinline__ void tc_mma(uint32_t tmem, uint32_t alo, uint32_t ahi, uint32_t blo, uint32_t bhi,
                                       uint32_t idesc, uint32_t acc) {
    asm volatile(
        "{\n.reg .pred p;\n.reg .b64 a, b;\nsetp.ne.u32 p, %6, 0;\nmov.b64 a, {%1, %2};\nmov.b64 b, {%3, %4};\n"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], a, b, %5, p;\n}\n" ::"r"(tmem),
        "r"(alo), "r"(ahi), "r"(blo), "r"(bhi), "r"(idesc), "r"(acc));
}

// The barriers and flags of a kernel's pipeline.  A producer warp fills shared-memory
// stages with bulk copies, one thread issues MMAs, further warps read.  full[s]
// completes when a fill's bytes have arrived, empty[s] when the stage's readers are
// done.  A wait that gives up (`limit` polls) in any role raises `abort`: the other
// roles stop at their next wait, and before the CTA frees its tensor memory the
// producer waits for the copies it has in flight and the issuer for its MMAs (at most
// TC_SPIN polls each).
struct Pipe {
    uint64_t full[TC_MAX_STAGES], empty[TC_MAX_STAGES];    // the stages
    uint64_t afull[TC_MAX_A], aempty[TC_MAX_A];            // convolution: tiles of A
    uint64_t tfull[2], tempty[2];                          // accumulators
    uint64_t once, drain;
    uint32_t tmem;
    int abort;
};

__device__ __forceinline__ void pipe_init(Pipe &pp, int readers, int ncols, int warp, int tid) {
    if (warp == 0) tc_alloc(&pp.tmem, ncols);
    if (warp == 1) {
        constexpr int N = offsetof(Pipe, tmem) / 8;  // all barriers, a lane each
        static_assert(N <= 64, "two per lane");
        for (int k = tid & 31; k < N; k += 32) {
            uint64_t *b = pp.full + k;
            mbar_init(smem_u32(b), b >= pp.empty && b < pp.afull ? readers : (b >= pp.tempty && b < &pp.once ? 4 : 1));
        }
        if ((tid & 31) == 0) pp.abort = 0;
        asm volatile("fence.mbarrier_init.release.cluster;\n");
    }
    asm volatile("tcgen05.fence::before_thread_sync;\n");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;\n");
}

// Wait of one role; raises abort when it gives up, and stops when another role has.
__device__ __forceinline__ bool pipe_wait(Pipe &pp, uint64_t &bar, uint32_t parity, long long limit) {
    for (long long it = 0; it < limit; it++) {
        if (tc_wait(smem_u32(&bar), parity, 1)) return true;
        if (*(volatile int *)&pp.abort) return false;
    }
    *(volatile int *)&pp.abort = 1;
    return false;
}
// The same for a whole warp; every lane sees the completed phase.
__device__ __forceinline__ bool pipe_wait_warp(Pipe &pp, uint64_t &bar, uint32_t parity, long long limit) {
    const bool go = pipe_wait(pp, bar, parity, limit);
    return __all_sync(0xffffffffu, go);
}
// Position in a ring of n stages: the stage, and the parity of its phase (no divisions:
// the roles' own instructions are in series, and a division is as long as an MMA).
struct Ring {
    int s = 0;
    uint32_t phase = 0;
    bool first = true;  // not all stages used yet
    __device__ __forceinline__ void next(int n) {
        if (++s == n) {
            s = 0;
            phase ^= 1;
            first = false;
        }
    }
};
// After an abort: the last fills of a ring of n stages, `fills` of them issued.
__device__ __forceinline__ void drain_fills(uint64_t *full, int n, int fills) {
    for (int c = max(fills - n, 0); c < fills; c++) tc_wait(smem_u32(&full[c % n]), (c / n) & 1, TC_SPIN);
}
// After an abort: the MMAs this thread has issued.
__device__ __forceinline__ void drain_mmas(Pipe &pp) {
    tc_commit(smem_u32(&pp.drain));
    tc_wait(smem_u32(&pp.drain), 0, TC_SPIN);
}

// Forward convolution (sign = +1), or the gradient with respect to its input (sign =
// -1, w the transposed weights): out[Q][n] = act(bias + sum over taps and source
// channels of src[Q + sign s(tap)][c] w[n][tap][c]), times (mask > 0) when a mask is
// given; with up, stored to the 2 x 2 pixels of the next finer level.
struct ConvOp {
    const bf16 *src;    // planes, sstr pixels each
    const bf16 *zero;   // zeros, as many pixels as a copy takes: the group after an odd G
    const bf16 *w;      // packed, [N tile][KG][BN][8]
    const float *bias;  // [N] or null
    const bf16 *mask;   // planes as out, or null
    bf16 *out;          // planes, ostr pixels each
    long long sstr, ostr;
    Geo geo, fine;
    int B, G, N, Ge, KG, sign, relu, up;
    // Shared memory, either (stages = 0) all of B and na tiles of A: a tile's pixels with
    // their neighbours for all taps, nseg row segments of segpx pixels per group, rowpx
    // between rows; or stages of gb K groups of B (gb divides Ge) and na units of A: gb
    // groups of one of the three rows of taps, 130 pixels each, for that row's taps.
    int nseg, segpx, rowpx, gb, na, stages;
    int ntile;   // tiles of 128 padded pixels
};

// Persistent CTAs, tiles of 128 consecutive padded pixels x BN outputs.  Warp 0 copies A
// (once for all taps, or once for the three taps of a row), warp 6 the weights (once,
// where they fit beside two tiles of A, else in stages), warp 1 issues the MMAs in the
// order of K (tap by tap, channels ascending) into one of two accumulators, warps 2 to 5
// store the other.  What bounds it: the operands' shared-memory reads at N = 32 and 64
// (4 KB of A for 16 or 32 cycles of tensor work), the streamed weights' way through L2
// on the coarse levels.  One CTA per tile, with everything in turn, left each CTA
// waiting for its own copies (8 to 14 us per tile, tensor pipe 6 to 17% active).  At 4
// levels of 32 to 256 channels, 16 images of 128 x 256: 1297 us a forward pass then, 303
// now; with all of a tile's A in one buffer (or, where two do not fit, each tap's A
// beside its weights) instead of units of a row, 330; with units of a row throughout,
// 437 (the waits of each row and tap are longer than the few MMAs between them).
template <int BN>
__global__ void __launch_bounds__(TC_THREADS) k_conv_tc(const ConvOp op, long long limit, int *err) {
    extern __shared__ __align__(1024) unsigned char smem[];
    __shared__ __align__(8) Pipe pp;
    __shared__ __align__(16) float bias[BN];
    constexpr uint32_t HI = desc_hi(128);
    constexpr int ACC = BN <= 32 ? 32 : (BN <= 64 ? 64 : 128), NCOLS = 2 * ACC;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, nt = blockIdx.y;
    const bool bstays = op.stages == 0;
    const int S = op.stages, nblk = bstays ? 1 : op.Ge / op.gb;
    constexpr int SEG = TC_M + 2;                                                // pixels of a unit's group
    const uint32_t gs = (bstays ? (uint32_t)(op.nseg * op.segpx) : SEG) * 16;    // K group stride
    const uint32_t unit = (bstays ? op.Ge : op.gb) * gs;
    const uint32_t a0 = smem_u32(smem), b0 = a0 + op.na * unit, stage = op.gb * BN * 16;
    const uint32_t none = b0 + op.KG * BN * 16;  // the input layer: a tile of zeros
    const bf16 *w = op.w + (long long)nt * op.KG * BN * 8;
    if (tid < BN) bias[tid] = op.bias && nt * BN + tid < op.N ? op.bias[nt * BN + tid] : 0.f;
    if (op.Ge == 1 && tid < TC_M) {
        *reinterpret_cast<uint4 *>(smem + (none - a0) + tid * 16) = make_uint4(0, 0, 0, 0);
        asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");
    }
    pipe_init(pp, 1, NCOLS, warp, tid);
    const uint32_t tmem = pp.tmem;
    if (warp == 0) {
        early_wait();
        int fills = 0;
        Ring ar;  // an empty[] of an earlier use: the other parity
        bool go = true;
        for (int tile = blockIdx.x; tile < op.ntile && go; tile += gridDim.x) {
            const long long q0 = op.geo.Wp + (long long)tile * TC_M - 1;
            for (int u = 0; u < (bstays ? 1 : 3 * nblk); u++) {
                if (!ar.first) go = pipe_wait_warp(pp, pp.aempty[ar.s], ar.phase ^ 1, limit);
                if (!go) break;
                const uint32_t bar = smem_u32(&pp.afull[ar.s]), to = a0 + ar.s * unit;
                if (lane == 0) mbar_expect(bar, unit);
                __syncwarp();
                if (bstays) {
                    for (int c = lane; c < op.Ge * op.nseg; c += 32) {
                        const int g = op.nseg == 3 ? c / 3 : c, row = op.nseg == 3 ? c - 3 * g - 1 : -1;
                        bulk_copy(to + c * op.segpx * 16,
                                  g < op.G ? op.src + (g * op.sstr + q0 + row * op.geo.Wp) * 8 : op.zero, op.segpx * 16, bar);
                    }
                } else if (lane < op.gb) {
                    const int row = u / nblk - 1, g = u % nblk * op.gb + lane;
                    bulk_copy(to + lane * SEG * 16,
                              g < op.G ? op.src + (g * op.sstr + q0 + op.sign * row * op.geo.Wp) * 8 : op.zero, SEG * 16, bar);
                }
                ar.next(op.na);
                fills++;
            }
        }
        early_next();
        __syncwarp();
        if (lane == 0 && *(volatile int *)&pp.abort) drain_fills(pp.afull, op.na, fills);
    } else if (warp == 6) {
        int fills = 0;
        if (lane == 0 && bstays) {
            mbar_expect(smem_u32(&pp.once), op.KG * BN * 16);
            for (int k = 0; k < op.KG; k += TC_KB)
                bulk_copy(b0 + k * BN * 16, w + (long long)k * BN * 8, min(TC_KB, op.KG - k) * BN * 16,
                          smem_u32(&pp.once));
        } else if (lane == 0) {
            Ring br;
            bool go = true;
            for (int tile = blockIdx.x; tile < op.ntile && go; tile += gridDim.x)
                for (int k = 0; k < 9 * nblk; k++) {
                    if (!br.first && !(go = pipe_wait(pp, pp.empty[br.s], br.phase ^ 1, limit))) break;
                    const uint32_t bar = smem_u32(&pp.full[br.s]);
                    mbar_expect(bar, stage);
                    bulk_copy(b0 + br.s * stage, w + (long long)k * op.gb * BN * 8, stage, bar);
                    br.next(S);
                    fills++;
                }
        }
        __syncwarp();
        if (lane == 0 && *(volatile int *)&pp.abort) {
            if (bstays) tc_wait(smem_u32(&pp.once), 0, TC_SPIN);
            else drain_fills(pp.full, S, fills);
        }
    } else if (warp == 1) {
        // kind::f16: D FP32, A and B BF16, both K-major, M = 128, N = BN
        constexpr uint32_t idesc = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(BN >> 3) << 17) |
                                   ((uint32_t)(TC_M >> 4) << 24);
        const bool leader = elect_one();
        bool go = !bstays || pipe_wait_warp(pp, pp.once, 0, limit), issued = false;
        Ring br, ar, acr;  // stages of B, units of A, accumulators
        for (int tile = blockIdx.x; tile < op.ntile && go; tile += gridDim.x) {
            if (!acr.first) go = pipe_wait_warp(pp, pp.tempty[acr.s], acr.phase ^ 1, limit);
            if (!go) break;
            const uint32_t d = tmem + acr.s * ACC;
            uint32_t blo = desc_lo(b0, BN * 16), acc = 0;
            issued = true;
            if (bstays) {
                if (!(go = pipe_wait_warp(pp, pp.afull[ar.s], ar.phase, limit))) break;
                asm volatile("tcgen05.fence::after_thread_sync;\n");
                const uint32_t abuf = a0 + ar.s * unit;
                if (op.Ge == 1) {
                    // two taps each, the distance between them the stride of K groups; the
                    // last one's partner is the tile of zeros
#pragma unroll
                    for (int t = 0; t < 10; t += 2) {
                        const uint32_t o0 = abuf + (t / 3 * op.rowpx + t % 3) * 16;
                        const uint32_t o1 = t < 8 ? abuf + ((t + 1) / 3 * op.rowpx + (t + 1) % 3) * 16 : none;
                        if (leader) tc_mma(d, desc_lo(o0, o1 - o0), HI, blo, HI, idesc, t > 0);
                        blo += 2 * BN;
                    }
                } else {
                    const uint32_t alo = desc_lo(abuf, gs) + (op.sign > 0 ? 0 : 2 * op.rowpx + 2);
                    for (int dy = 0; dy < 3; dy++)
                        for (int dx = 0; dx < 3; dx++) {
                            uint32_t an = alo + op.sign * (dy * op.rowpx + dx);
#pragma unroll 2
                            for (int g = 0; g < op.Ge; g += 2) {
                                if (leader) tc_mma(d, an, HI, blo, HI, idesc, acc);
                                acc = 1;
                                an += gs >> 3;
                                blo += 2 * BN;
                            }
                        }
                }
                if (leader) tc_commit(smem_u32(&pp.aempty[ar.s]));
                ar.next(op.na);
            } else {
                // no way out of these loops: a branch on a wait's outcome would make their
                // values non-uniform.  After a wait that gave up the MMAs left read what
                // is there, and nothing is stored.
                for (int row = 0; row < 3; row++) {
                    const int as0 = ar.s;
                    const uint32_t ap0 = ar.phase;
                    for (int dx = 0; dx < 3; dx++) {
                        ar.s = as0;
                        ar.phase = ap0;
                        for (int blk = 0; blk < nblk; blk++) {
                            if (dx == 0) pipe_wait_warp(pp, pp.afull[ar.s], ar.phase, limit);
                            pipe_wait_warp(pp, pp.full[br.s], br.phase, limit);
                            asm volatile("tcgen05.fence::after_thread_sync;\n");
                            uint32_t an = desc_lo(a0 + ar.s * unit, SEG * 16) + (op.sign > 0 ? dx : 2 - dx);
                            blo = desc_lo(b0 + br.s * stage, BN * 16);
#pragma unroll 2
                            for (int k = 0; k < op.gb; k += 2) {
                                if (leader) tc_mma(d, an, HI, blo, HI, idesc, acc);
                                acc = 1;
                                an += 2 * SEG;
                                blo += 2 * BN;
                            }
                            if (leader) {
                                tc_commit(smem_u32(&pp.empty[br.s]));
                                if (dx == 2) tc_commit(smem_u32(&pp.aempty[ar.s]));
                            }
                            br.next(S);
                            ar.next(op.na);
                        }
                    }
                }
                go = __all_sync(0xffffffffu, *(volatile int *)&pp.abort == 0);
            }
            if (go && leader) tc_commit(smem_u32(&pp.tfull[acr.s]));
            acr.next(2);
        }
        if (issued && leader && *(volatile int *)&pp.abort) drain_mmas(pp);
        __syncwarp();
    } else {
        // epilogue: warp w reads TMEM lanes 32 (w % 4) .. + 31, a pixel per lane; the
        // mask (one bit per channel) is fetched while the MMAs run
        early_wait();
        const int part = warp & 3, ng = (min(BN, op.N - nt * BN) + 7) >> 3;
        const uint4 *mask = reinterpret_cast<const uint4 *>(op.mask) + (long long)(nt * BN >> 3) * op.ostr;
        uint4 *out = reinterpret_cast<uint4 *>(op.out) + (long long)(nt * BN >> 3) * op.ostr;
        int i = 0;
        for (int tile = blockIdx.x; tile < op.ntile; tile += gridDim.x, i++) {
            const int Q = op.geo.Wp + tile * TC_M + part * 32 + lane;
            int n_, y, x;
            const bool in = op.geo.where(Q, op.B, n_, y, x);
            uint32_t keep[BN / 32];
#pragma unroll
            for (int c = 0; c < BN / 32; c++) {
                keep[c] = 0xffffffffu;
                if (!op.mask) continue;
                uint4 mk[4];
#pragma unroll
                for (int h = 0; h < 4; h++)
                    mk[h] = in && 4 * c + h < ng ? mask[(4 * c + h) * op.ostr + Q] : make_uint4(0, 0, 0, 0);
                keep[c] = 0;
#pragma unroll
                for (int h = 0; h < 4; h++) {
                    float m[8];
                    unpack8(mk[h], m);
#pragma unroll
                    for (int j = 0; j < 8; j++) keep[c] |= m[j] > 0.f ? 1u << (8 * h + j) : 0u;
                }
            }
            long long at = Q;
            if (op.up && in) at = op.fine.at(n_, 2 * y, 2 * x);
            if (!pipe_wait_warp(pp, pp.tfull[i & 1], (i / 2) & 1, limit)) break;
            asm volatile("tcgen05.fence::after_thread_sync;\n");
#pragma unroll
            for (int c = 0; c < BN / 32; c++) {
                float f[32];
                __syncwarp();
                tc_ld32(tmem + ((uint32_t)(part * 32) << 16) + (i & 1) * ACC + 32 * c, f);
                if (c == BN / 32 - 1) {  // the accumulator is read
                    asm volatile("tcgen05.fence::before_thread_sync;\n");
                    __syncwarp();
                    if (lane == 0) mbar_arrive(smem_u32(&pp.tempty[i & 1]));
                }
#pragma unroll
                for (int h = 0; h < 4; h++) {
                    float o[8];
#pragma unroll
                    for (int j = 0; j < 8; j++) {
                        o[j] = f[8 * h + j] + bias[32 * c + 8 * h + j];
                        if (op.relu) o[j] = fmaxf(o[j], 0.f);
                        if (!(keep[c] >> (8 * h + j) & 1u)) o[j] = 0.f;
                    }
                    if (!in || 4 * c + h >= ng) continue;
                    const uint4 pk = pack8(o);
                    uint4 *to = out + (4 * c + h) * op.ostr + at;
                    to[0] = pk;
                    if (op.up) {
                        to[1] = pk;
                        to[op.fine.Wp] = pk;
                        to[op.fine.Wp + 1] = pk;
                    }
                }
            }
        }
    }
    __syncthreads();
    if (tid == 0 && pp.abort) atomicOr(err, 1);
    tc_free(tmem, NCOLS, warp);
}

// Weight gradient: for each dx a GEMM D[(dy, ci)][co] over the pixels, both operands
// MN-major (8 consecutive channels of a pixel are a core-matrix row), so the planes are
// copied as they are: 8-channel groups (dy, g) of a run of pixels, from (dy, -1) on, and
// dz's groups.  dx shifts A's start address by a pixel.  A CTA takes 16 groups (128
// rows) x BN outputs and a range of pixels, in runs of up to 128 (Runs); its sums go to
// the range's partial result, four outputs at a time.  The bias gradient, the sum of dz,
// is taken from the staged dz by the epilogue warps.
struct WgradOp {
    const bf16 *x, *dz;  // planes, xstr and zstr pixels each
    float *part;         // of every range of pixels: [tap][Ci][Co], then [Co] for the bias
    long long xstr, zstr;
    int Wp, Ci, Co, G, stages;
    // the sum over pixels: rows of W pixels, H of them PSI apart, the first at q0; npix
    // in all, perz to a CTA, runpx at most to a stage
    long long W, npix, perz;
    int H, PSI, q0, runpx;
};
constexpr int WG_PX = 128, WG_SPLIT = 64;  // a CTA has a multiple of 64 pixels

// A CTA's pixels, in runs of up to 128 for one stage: part of a row, or as many whole
// rows as fit (with the border pixels between them copied along and left out).
struct Runs {
    long long x, rem;  // column of the next pixel; pixels left
    int y, n;
    int rows, len;     // this run: rows of len pixels
    __device__ __forceinline__ Runs(const WgradOp &op) {
        const long long p = (long long)blockIdx.z * op.perz, r = p / op.W;
        rem = min(op.perz, op.npix - p);
        x = p - r * op.W;
        n = (int)(r / op.H);
        y = (int)(r - (long long)n * op.H);
    }
    __device__ __forceinline__ bool next(const WgradOp &op) {
        if (rem <= 0) return false;
        rows = 1;
        len = (int)min(min(op.W - x, rem), (long long)WG_PX);
        if (x == 0 && len == op.W)
            while (rows * len + len <= min(rem, (long long)WG_PX) && y + rows < op.H) rows++;
        return true;
    }
    __device__ __forceinline__ long long at(const WgradOp &op) const {
        return op.q0 + (long long)n * op.PSI + (long long)y * op.Wp + x;
    }
    __device__ __forceinline__ int span(const WgradOp &op) const { return (rows - 1) * op.Wp + len; }
    __device__ __forceinline__ void advance(const WgradOp &op) {
        rem -= rows * len;
        x += len;
        if (x < op.W) return;
        x = 0;
        if ((y += rows) < op.H) return;
        y = 0;
        n++;
    }
};

template <int BN>
__global__ void __launch_bounds__(WG_THREADS) k_wgrad_tc(const WgradOp op, long long limit, int *err) {
    extern __shared__ __align__(1024) unsigned char smem[];
    __shared__ __align__(8) Pipe pp;
    constexpr int COLS = 3 * BN, NCOLS = COLS <= 128 ? 128 : (COLS <= 256 ? 256 : 512);
    const uint32_t AG = (op.runpx + 2) * 16, ZG = op.runpx * 16;  // bytes of a group of A, of dz
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int m0 = blockIdx.x * 16;                       // first (dy, g) group
    const int ng = min(16, 3 * op.G - m0);                // groups that exist
    const int n0 = blockIdx.y * BN, zg = min(BN, op.Co - n0) / 8;
    const int S = op.stages;
    const uint32_t base = smem_u32(smem), stage = 16 * AG + BN / 8 * ZG;
    const bool bias = blockIdx.x == 0;
    Runs run(op);
    float *sum = op.part + (long long)blockIdx.z * (9 * op.Ci + 1) * op.Co;  // of this range
    pipe_init(pp, bias ? 5 : 1, NCOLS, warp, tid);
    const uint32_t tmem = pp.tmem;
    if (warp == 0) {
        int fills = 0;
        Ring r;
        for (; run.next(op); run.advance(op), r.next(S)) {
            if (!r.first && !pipe_wait_warp(pp, pp.empty[r.s], r.phase ^ 1, limit)) break;
            const uint32_t at = base + r.s * stage, bar = smem_u32(&pp.full[r.s]);
            const uint32_t zb = run.span(op) * 16, ab = zb + 32;
            if (lane == 0) mbar_expect(bar, ng * ab + zg * zb);
            __syncwarp();
            const long long q = run.at(op);
            for (int c = lane; c < ng + zg; c += 32) {
                if (c < ng) {
                    const int m = m0 + c, dy = m / op.G, g = m - dy * op.G;
                    bulk_copy(at + c * AG, op.x + (g * op.xstr + q + (dy - 1) * op.Wp - 1) * 8, ab, bar);
                } else {
                    bulk_copy(at + 16 * AG + (c - ng) * ZG,
                              op.dz + ((long long)(n0 / 8 + c - ng) * op.zstr + q) * 8, zb, bar);
                }
            }
            fills++;
        }
        __syncwarp();
        if (lane == 0 && *(volatile int *)&pp.abort) drain_fills(pp.full, S, fills);
    } else if (warp == 1) {
        // kind::f16: D FP32, A and B BF16, both MN-major, M = 128, N = BN
        constexpr uint32_t idesc = (1u << 4) | (1u << 7) | (1u << 10) | (1u << 15) | (1u << 16) |
                                   ((uint32_t)(BN >> 3) << 17) | ((uint32_t)(TC_M >> 4) << 24);
        const bool leader = elect_one();
        bool go = true, issued = false;
        Ring r;
        uint32_t acc = 0;
        const uint32_t ahi = desc_hi(AG), zhi = desc_hi(ZG);
        for (; run.next(op); run.advance(op), r.next(S)) {
            if (!(go = pipe_wait_warp(pp, pp.full[r.s], r.phase, limit))) break;
            asm volatile("tcgen05.fence::after_thread_sync;\n");
            const uint32_t at = base + r.s * stage;
            uint32_t arow = desc_lo(at, 128), zrow = desc_lo(at + 16 * AG, 128);
            for (int y = 0; y < run.rows; y++, arow += op.Wp, zrow += op.Wp)
                for (int k = 0; k < run.len; k += 16) {
                    if (leader) {
#pragma unroll
                        for (int dx = 0; dx < 3; dx++)
                            tc_mma(tmem + dx * BN, arow + k + dx, ahi, zrow + k, zhi, idesc, acc);
                    }
                    acc = 1;
                }
            if (leader) tc_commit(smem_u32(&pp.empty[r.s]));
            issued = true;
        }
        if (go && leader) tc_commit(smem_u32(&pp.tfull[0]));
        if (issued && leader && *(volatile int *)&pp.abort) drain_mmas(pp);
        __syncwarp();
    } else {
        // 128 threads: channel group g, every np-th pixel
        const int t = tid - 64, g = t % zg, np = 128 / zg, p0 = t / zg;
        float a[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
        if (bias) {
            Ring r;
            for (; run.next(op); run.advance(op), r.next(S)) {
                if (!pipe_wait_warp(pp, pp.full[r.s], r.phase, limit)) break;
                const int span = run.span(op);
                const uint4 *z = reinterpret_cast<const uint4 *>(smem + r.s * stage + 16 * AG + g * ZG);
                if (p0 < np)
                    for (int px = p0; px < span; px += np) {
                        const uint4 v = z[px];
                        const __nv_bfloat162 *h = reinterpret_cast<const __nv_bfloat162 *>(&v);
#pragma unroll
                        for (int j = 0; j < 4; j++) {
                            const float2 f = __bfloat1622float2(h[j]);
                            a[2 * j] += f.x;
                            a[2 * j + 1] += f.y;
                        }
                    }
                __syncwarp();
                if (lane == 0) mbar_arrive(smem_u32(&pp.empty[r.s]));
            }
        }
        const bool done = pipe_wait_warp(pp, pp.tfull[0], 0, limit);
        if (bias) {
            // every MMA has read its stages, and after the barrier every thread its dz:
            // the first stage takes the threads' sums, added in the order of the pixels
            // (the four warps come to the barriers whatever their waits' outcome)
            float *sums = reinterpret_cast<float *>(smem);
            asm volatile("bar.sync 1, 128;\n" ::: "memory");
            if (done && p0 < np)
#pragma unroll
                for (int j = 0; j < 8; j++) sums[t * 8 + j] = a[j];
            asm volatile("bar.sync 1, 128;\n" ::: "memory");
            if (done && t < zg * 8) {
                float b = 0.f;
                for (int p = 0; p < np; p++) b += sums[(p * zg + (t >> 3)) * 8 + (t & 7)];
                sum[(long long)9 * op.Ci * op.Co + n0 + t] = b;
            }
        }
        if (done) {
            asm volatile("tcgen05.fence::after_thread_sync;\n");
            const int part = warp & 3;
            const int m = m0 + part * 4 + (lane >> 3);  // this lane's (dy, g)
            const bool mine = m < 3 * op.G;
            const int dy = m / op.G, ci = (m - dy * op.G) * 8 + (lane & 7);
#pragma unroll
            for (int dx = 0; dx < 3; dx++) {
                float *row = sum + ((long long)(dy * 3 + dx) * op.Ci + ci) * op.Co + n0;
#pragma unroll
                for (int c0 = 0; c0 < BN; c0 += 32) {
                    float f[32];
                    __syncwarp();
                    tc_ld32(tmem + ((uint32_t)(part * 32) << 16) + dx * BN + c0, f);
#pragma unroll
                    for (int j = 0; j < 32; j += 4)
                        if (mine && n0 + c0 + j < op.Co)
                            *reinterpret_cast<float4 *>(row + c0 + j) =
                                make_float4(f[j], f[j + 1], f[j + 2], f[j + 3]);
                }
            }
        }
    }
    __syncthreads();
    if (tid == 0 && pp.abort) atomicOr(err, 1);
    tc_free(tmem, NCOLS, warp);
}

// s + c, c the rounding errors, plus x (Knuth's two-sum)
__device__ __forceinline__ void add_comp(float &s, float &c, float x) {
    const float t = s + x, b = t - s;
    c += (s - (t - b)) + (x - b);
    s = t;
}

// The sum of nz partial results of n4 + m4 float4 each, into dst and dst2 (m4 of them): a
// thread of SP_Z takes every SP_Z-th, in order, and the first thread adds theirs, in
// order; the additions' rounding errors are added up beside them, so that the sum is
// rounded once.  What bounds it is the reads, from L2 (up to 40 MB a layer).
constexpr int SP_X = 32, SP_Z = 8;
__global__ void __launch_bounds__(SP_X *SP_Z) k_sum_parts(const float4 *part, int nz, int n4, int m4, float4 *dst,
                                                          float4 *dst2) {
    __shared__ float4 ss[SP_Z][SP_X], sc[SP_Z][SP_X];
    const int x = threadIdx.x % SP_X, z0 = threadIdx.x / SP_X, i = blockIdx.x * SP_X + x;
    const long long str = n4 + m4;
    float4 s = make_float4(0.f, 0.f, 0.f, 0.f), c = s;
    if (i < str)
#pragma unroll 4
        for (int z = z0; z < nz; z += SP_Z) {
            const float4 v = part[z * str + i];
            add_comp(s.x, c.x, v.x);
            add_comp(s.y, c.y, v.y);
            add_comp(s.z, c.z, v.z);
            add_comp(s.w, c.w, v.w);
        }
    ss[z0][x] = s;
    sc[z0][x] = c;
    __syncthreads();
    if (z0 != 0 || i >= str) return;
    for (int z = 1; z < SP_Z; z++) {
        const float4 v = ss[z][x], d = sc[z][x];
        add_comp(s.x, c.x, v.x);
        add_comp(s.y, c.y, v.y);
        add_comp(s.z, c.z, v.z);
        add_comp(s.w, c.w, v.w);
        c = make_float4(c.x + d.x, c.y + d.y, c.z + d.z, c.w + d.w);
    }
    (i < n4 ? dst[i] : dst2[i - n4]) = make_float4(s.x + c.x, s.y + c.y, s.z + c.z, s.w + c.w);
}

// ------------------------------------------------------ other layers

constexpr int EW = 256;  // threads of the elementwise kernels

inline unsigned blocks(long long n) { return (unsigned)((n + EW - 1) / EW); }

// NCHW float input [B][8][H][W] -> one plane
__global__ void k_pack_input(const float *in, bf16 *x, int B, Geo geo) {
    early_next();
    const int HW = geo.H * geo.W;
    const long long i = (long long)blockIdx.x * EW + threadIdx.x;
    if (i >= (long long)B * HW) return;
    const int n = (int)(i / HW), r = (int)(i - (long long)n * HW), y = r / geo.W;
    float f[8];
#pragma unroll
    for (int c = 0; c < 8; c++) f[c] = in[((long long)n * 8 + c) * HW + r];
    reinterpret_cast<uint4 *>(x)[geo.at(n, y, r - y * geo.W)] = pack8(f);
}

// The layers below take a group of 8 channels (blockIdx.y) of one pixel per thread:
// neighbouring threads have neighbouring pixels, 16 bytes each.
__device__ __forceinline__ bool pixel_of(long long i, int B, const Geo &geo, int &n, int &y, int &x) {
    const int HW = geo.H * geo.W;
    if (i >= (long long)B * HW) return false;
    n = (int)(i / HW);
    const int r = (int)(i - (long long)n * HW);
    y = r / geo.W;
    x = r - y * geo.W;
    return true;
}

// 2x2 average pooling of planes on `fine` into planes on `geo`
__global__ void k_pool(const bf16 *in, long long istr, bf16 *out, long long ostr, int B, Geo fine, Geo geo) {
    early_next();
    early_wait();
    int n, y, x;
    if (!pixel_of((long long)blockIdx.x * EW + threadIdx.x, B, geo, n, y, x)) return;
    const uint4 *p = reinterpret_cast<const uint4 *>(in) + blockIdx.y * istr + fine.at(n, 2 * y, 2 * x);
    const uint4 v[4] = {p[0], p[1], p[fine.Wp], p[fine.Wp + 1]};
    float a[8], t[8];
    unpack8(v[0], a);
#pragma unroll
    for (int k = 1; k < 4; k++) {
        unpack8(v[k], t);
#pragma unroll
        for (int j = 0; j < 8; j++) a[j] += t[j];
    }
#pragma unroll
    for (int j = 0; j < 8; j++) a[j] *= 0.25f;
    reinterpret_cast<uint4 *>(out)[blockIdx.y * ostr + geo.at(n, y, x)] = pack8(a);
}

// de = (e > 0) * dpool / 4 + dskip on `geo`, dpool on the next coarser level (dskip:
// already masked)
__global__ void k_pool_back(const bf16 *dpool, long long pstr, const bf16 *e, const bf16 *dskip, bf16 *de,
                            long long str, int B, Geo coarse, Geo geo) {
    int n, y, x;
    if (!pixel_of((long long)blockIdx.x * EW + threadIdx.x, B, geo, n, y, x)) return;
    const long long q = blockIdx.y * str + geo.at(n, y, x);
    float dp[8], ev[8], ds[8], o[8];
    unpack8(reinterpret_cast<const uint4 *>(dpool)[blockIdx.y * pstr + coarse.at(n, y / 2, x / 2)], dp);
    unpack8(reinterpret_cast<const uint4 *>(e)[q], ev);
    unpack8(reinterpret_cast<const uint4 *>(dskip)[q], ds);
#pragma unroll
    for (int j = 0; j < 8; j++) o[j] = (ev[j] > 0.f ? 0.25f * dp[j] : 0.f) + ds[j];
    reinterpret_cast<uint4 *>(de)[q] = pack8(o);
}

// dd on `geo` = sum over the 2x2 children of dcat on `fine`
__global__ void k_up_back(const bf16 *dcat, long long cstr, bf16 *dd, long long str, int B, Geo fine, Geo geo) {
    int n, y, x;
    if (!pixel_of((long long)blockIdx.x * EW + threadIdx.x, B, geo, n, y, x)) return;
    const uint4 *p = reinterpret_cast<const uint4 *>(dcat) + blockIdx.y * cstr + fine.at(n, 2 * y, 2 * x);
    const uint4 v[4] = {p[0], p[1], p[fine.Wp], p[fine.Wp + 1]};
    float a[8] = {0, 0, 0, 0, 0, 0, 0, 0}, t[8];
#pragma unroll
    for (int k = 0; k < 4; k++) {
        unpack8(v[k], t);
#pragma unroll
        for (int j = 0; j < 8; j++) a[j] += t[j];
    }
    reinterpret_cast<uint4 *>(dd)[blockIdx.y * str + geo.at(n, y, x)] = pack8(a);
}

// 1x1 head: out[n][o][y][x] = b[o] + sum_c w[o][c] d[c] (FP32), NCHW output
__global__ void k_head(const bf16 *d, long long dstr, const float *w, const float *b, float *out, int B,
                       Geo geo, int C) {
    early_wait();
    const long long i = (long long)blockIdx.x * EW + threadIdx.x;
    int n, y, x;
    if (!pixel_of(i, B, geo, n, y, x)) return;
    const uint4 *p = reinterpret_cast<const uint4 *>(d) + geo.at(n, y, x);
    float acc[3] = {b[0], b[1], b[2]};
    for (int c = 0; c < C; c += 8) {
        float v[8];
        unpack8(p[(c >> 3) * dstr], v);
#pragma unroll
        for (int j = 0; j < 8; j++)
#pragma unroll
            for (int o = 0; o < 3; o++) acc[o] += w[o * C + c + j] * v[j];
    }
    const long long HW = (long long)geo.H * geo.W, r = i - n * HW;
#pragma unroll
    for (int o = 0; o < 3; o++) out[(n * 3 + o) * HW + r] = acc[o];
}

// a block's sum of one value per thread, in a fixed order, in thread 0
__device__ __forceinline__ float block_sum(float (&s)[EW], float a) {
    s[threadIdx.x] = a;
    __syncthreads();
    for (int o = EW / 2; o > 0; o >>= 1) {
        if (threadIdx.x < o) s[threadIdx.x] += s[threadIdx.x + o];
        __syncthreads();
    }
    return s[0];
}

// fluid-node count (for the loss normalisation), a part per block
__global__ void k_count(const float *fluid, long long n, float *cnt) {
    __shared__ float s[EW];
    float a = 0.f;
    for (long long i = (long long)blockIdx.x * EW + threadIdx.x; i < n; i += (long long)gridDim.x * EW)
        a += fluid[i];
    a = block_sum(s, a);
    if (threadIdx.x == 0) cnt[blockIdx.x] = a;
}

// loss = sum (out - t)^2 m / (3 count), a part per block; dout = 2 (out - t) m / (3 count)
__global__ void k_loss(const float *out, const float *tgt, const float *fluid, const float *cnt,
                       float *dout, double *loss, int B, int HW) {
    __shared__ float s[EW];
    const long long n3 = (long long)B * 3 * HW;
    const float count = block_sum(s, cnt[threadIdx.x]);
    __syncthreads();
    const float inv = 1.f / (3.f * fmaxf(count, 1.f));
    float a = 0.f;
    for (long long i = (long long)blockIdx.x * EW + threadIdx.x; i < n3; i += (long long)gridDim.x * EW) {
        const long long n = i / (3 * HW), r = i % HW;
        const float m = fluid[n * HW + r];
        const float d = (out[i] - tgt[i]) * m;
        a += d * d;
        dout[i] = 2.f * d * inv;
    }
    a = block_sum(s, a);
    if (threadIdx.x == 0) loss[1 + blockIdx.x] = (double)(a * inv);
}
constexpr int CNT_BLOCKS = EW, LOSS_BLOCKS = 1024;

// the loss's parts, in order
__global__ void __launch_bounds__(32) k_loss_sum(double *loss) {
    double a = 0.0;
    for (int i = threadIdx.x; i < LOSS_BLOCKS; i += 32) a += loss[1 + i];
    for (int o = 16; o > 0; o >>= 1) a += __shfl_down_sync(0xffffffffu, a, o);
    if (threadIdx.x == 0) loss[0] = a;
}

// head backward: dd[c] = (d[c] > 0) sum_o dout[o] w[o][c]; of the block's pixels, into
// its partial result: dw[o][c] = sum of dout[o] d[c], db[o] = sum of dout[o].  A thread takes every
// gridDim.x EW-th pixel of one group of 8 channels and keeps its 24 sums in registers
// to the end (one pixel per thread and 96 warp sums for it took 220 us at 0.5 M
// pixels, the memory traffic 12).
__global__ void __launch_bounds__(EW) k_head_back(const float *dout, const bf16 *d, long long dstr,
                                                  const float *w, bf16 *dd, float *part, int B, Geo geo,
                                                  int C) {
    __shared__ float red[EW / 32][28];
    const int c0 = blockIdx.y * 8;
    const long long HW = (long long)geo.H * geo.W;
    float wv[3][8], s[3][8], sb[3] = {0.f, 0.f, 0.f};
#pragma unroll
    for (int o = 0; o < 3; o++)
#pragma unroll
        for (int j = 0; j < 8; j++) {
            wv[o][j] = w[o * C + c0 + j];
            s[o][j] = 0.f;
        }
    for (long long i = (long long)blockIdx.x * EW + threadIdx.x; i < B * HW; i += (long long)gridDim.x * EW) {
        int n, y, x;
        pixel_of(i, B, geo, n, y, x);
        const long long q = blockIdx.y * dstr + geo.at(n, y, x), r = i - n * HW;
        float g[3], v[8], o8[8];
#pragma unroll
        for (int o = 0; o < 3; o++) g[o] = dout[(n * 3 + o) * HW + r];
        unpack8(reinterpret_cast<const uint4 *>(d)[q], v);
#pragma unroll
        for (int j = 0; j < 8; j++) {
            const float t = g[0] * wv[0][j] + g[1] * wv[1][j] + g[2] * wv[2][j];
            o8[j] = v[j] > 0.f ? t : 0.f;
#pragma unroll
            for (int o = 0; o < 3; o++) s[o][j] += g[o] * v[j];
        }
#pragma unroll
        for (int o = 0; o < 3; o++) sb[o] += g[o];
        reinterpret_cast<uint4 *>(dd)[q] = pack8(o8);
    }
    auto sum = [&](float v, int k) {
        for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
        if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5][k] = v;
    };
#pragma unroll
    for (int o = 0; o < 3; o++) {
#pragma unroll
        for (int j = 0; j < 8; j++) sum(s[o][j], o * 8 + j);
        sum(sb[o], 24 + o);
    }
    __syncthreads();
    if (threadIdx.x >= 28) return;
    float v = 0.f;  // the last of the four for the bias stays zero
    if (threadIdx.x < 27)
        for (int k = 0; k < EW / 32; k++) v += red[k][threadIdx.x];
    float *p = part + (long long)blockIdx.x * (3 * C + 4);
    if (threadIdx.x < 24) p[(threadIdx.x >> 3) * C + c0 + (threadIdx.x & 7)] = v;
    else if (blockIdx.y == 0) p[3 * C + threadIdx.x - 24] = v;
}

// Where a parameter sits: the vector of all convolutions, weights [tap][Cin][Cout] (the
// 1x1 head: [Cout][Cin]) then biases, both padded to 8; in the caller's order
// [Cout][Cin][k][k] then biases, from abi; and the packed BF16 copies.
constexpr int MAX_CONVS = 16;
struct ConvTab {
    struct E {
        int w_off, b_off, abi, ci, co, taps;
        bf16 *fwd, *bwd;  // null: none
        int fBN, fKG, fGe, bBN, bKG, bGe;
    } e[MAX_CONVS];
    int n;
    // caller's index of parameter i, or -1 (padding); the weight's (co, tap, ci) or co = -1
    __device__ __forceinline__ long long abi_of(long long i, int &k, int &co, int &tap, int &ci) const {
        k = 0;
        while (k + 1 < n && i >= e[k + 1].w_off) k++;
        const E &c = e[k];
        co = -1;
        if (i >= c.b_off) {
            const int j = (int)(i - c.b_off);
            return j < c.co ? c.abi + (long long)c.co * c.ci * c.taps + j : -1;
        }
        const int j = (int)(i - c.w_off);
        if (j >= c.co * c.ci * c.taps) return -1;
        if (c.taps == 1) {
            co = j / c.ci;
            ci = j - co * c.ci;
            tap = 0;
        } else {
            co = j % c.co;
            const int r = j / c.co;
            tap = r / c.ci;
            ci = r - tap * c.ci;
        }
        return c.abi + ((long long)co * c.ci + ci) * c.taps + tap;
    }
    __device__ __forceinline__ void pack(int k, int co, int tap, int ci, float v) const {
        const E &c = e[k];
        const bf16 b = __float2bfloat16(v);
        if (c.fwd) c.fwd[packed_at(co, tap, ci, c.fBN, c.fKG, c.fGe)] = b;
        if (c.bwd) c.bwd[packed_at(ci, tap, co, c.bBN, c.bKG, c.bGe)] = b;
    }
};

// Adam on the flat FP32 master vector; refreshes the BF16 copies.
__global__ void k_adam(ConvTab tab, float *w, const float *g, float *m, float *v, long long n, float lr,
                       float c1, float c2) {
    const long long i = (long long)blockIdx.x * EW + threadIdx.x;
    if (i >= n) return;
    const float gi = g[i];
    const float mi = 0.9f * m[i] + 0.1f * gi, vi = 0.999f * v[i] + 0.001f * gi * gi;
    m[i] = mi;
    v[i] = vi;
    const float wi = w[i] - lr * (mi / c1) / (sqrtf(vi / c2) + 1e-8f);
    w[i] = wi;
    int k, co, tap, ci;
    if (tab.abi_of(i, k, co, tap, ci) >= 0 && co >= 0) tab.pack(k, co, tap, ci, wi);
}

// The caller's parameter vector into the masters and BF16 copies
__global__ void k_from_abi(ConvTab tab, const float *abi, float *w, long long n) {
    const long long i = (long long)blockIdx.x * EW + threadIdx.x;
    if (i >= n) return;
    int k, co, tap, ci;
    const long long a = tab.abi_of(i, k, co, tap, ci);
    const float v = a >= 0 ? abi[a] : 0.f;
    w[i] = v;
    if (a >= 0 && co >= 0) tab.pack(k, co, tap, ci, v);
}

// A vector in the masters' layout into the caller's order
__global__ void k_to_abi(ConvTab tab, const float *w, float *abi, long long n) {
    const long long i = (long long)blockIdx.x * EW + threadIdx.x;
    if (i >= n) return;
    int k, co, tap, ci;
    const long long a = tab.abi_of(i, k, co, tap, ci);
    if (a >= 0) abi[a] = w[i];
}

// network input of one case: mask (owner >= 0) and Re / 100, zero elsewhere
__global__ void k_case_input(const int32_t *owner, float re100, float *in, int HW) {
    const int i = blockIdx.x * EW + threadIdx.x;
    if (i >= HW) return;
    in[i] = owner[i] >= 0 ? 1.f : 0.f;
    in[HW + i] = re100;
    for (int c = 2; c < 8; c++) in[c * HW + i] = 0.f;
}

}  // namespace nn

// ================================================================ network

using nn::bf16;

namespace {

struct Conv {
    int ci, co, k;            // k = 3 or 1
    size_t w_off, b_off;      // into the flat parameter vector
    bf16 *fwd = nullptr;      // packed BF16 weights of the forward convolution
    bf16 *bwd = nullptr;      // and of the data gradient
};

// planes of 8 channels on one level's pixels
struct Planes {
    bf16 *p = nullptr;        // pixel 0 of the first plane
    long long str = 0;        // pixels per plane
    Planes group(int g) const { return Planes{p + (long long)g * str * 8, str}; }
};

struct Level {
    nn::Geo geo;
    int C;
    Planes inp;               // pooled input (l > 0)
    Planes ea;                // encoder: relu(conv a)
    Planes cat;               // decoder (l < L-1): {upsampled output of level l + 1, e}
    Planes e;                 // level output: the last C channels of cat (l < L-1)
    Planes da, d;             // decoder: relu(conv a); relu(conv b) (l = 0: for the head)
    Planes g1, g2, gcat, gin; // gradients
};

}  // namespace

struct lbm_unet {
    lbm_unet_config cfg{};
    cudaStream_t stream = nullptr;
    bool own_stream = false;
    cudaStream_t side[2] = {};    // weight gradients (backward), in turn
    cudaEvent_t fork = nullptr, join[2] = {};
    int turn = 0;
    std::vector<Conv> convs;  // parameter order
    std::vector<Level> lv;
    nn::ConvTab tab{};
    long long nparam = 0, nabi = 0;
    float *w = nullptr, *g = nullptr, *m = nullptr, *v = nullptr;
    Planes x;                // packed input
    bf16 *zero = nullptr;    // ConvOp::zero
    float *out = nullptr, *dout = nullptr;
    float *io_in = nullptr, *io_tgt = nullptr, *io_fl = nullptr;  // staging
    float *abi = nullptr;    // parameters or gradients in the caller's order
    float *part[2] = {};     // partial sums of a layer's gradient, one for each side stream
    float *cnt = nullptr;    // fluid nodes, by block
    double *loss = nullptr;  // the loss, then its parts by block
    int *err_d = nullptr;    // bit 0: a bounded wait of a tensor-core kernel ran out
    long long wait_limit = nn::TC_SPIN;  // polls of an mbarrier before a wait gives up
    int sms = 0;             // streaming multiprocessors of the device
    bool early = false;      // launch_tc in the forward pass
    long long adam_t = 0;
    std::string err;
    std::vector<void *> allocs;
};

namespace {

thread_local std::string g_nn_error;

lbm_status nfail(lbm_unet *n, lbm_status st, const char *fmt, ...) __attribute__((format(printf, 3, 4)));
lbm_status nfail(lbm_unet *n, lbm_status st, const char *fmt, ...) {
    char buf[512];
    va_list ap;
    va_start(ap, fmt);
    vsnprintf(buf, sizeof buf, fmt, ap);
    va_end(ap);
    if (n) n->err = buf;
    else g_nn_error = buf;
    return st;
}

#define NCK(n, call)                                                                        \
    do {                                                                                    \
        cudaError_t e_ = (call);                                                            \
        if (e_ != cudaSuccess)                                                              \
            return nfail((n), e_ == cudaErrorMemoryAllocation ? LBM_ENOMEM : LBM_ECUDA,     \
                         "%s failed: %s", #call, cudaGetErrorString(e_));                  \
    } while (0)

// after a synchronisation: a tensor-core kernel that gave up waiting
lbm_status check_err(lbm_unet *n) {
    int e = 0;
    NCK(n, cudaMemcpyAsync(&e, n->err_d, sizeof(int), cudaMemcpyDeviceToHost, n->stream));
    NCK(n, cudaStreamSynchronize(n->stream));
    if (e) {
        cudaMemsetAsync(n->err_d, 0, sizeof(int), n->stream);
        return nfail(n, LBM_ETIMEOUT, "a bounded wait of the tensor-core convolution ran out");
    }
    return LBM_OK;
}

template <class T>
cudaError_t nalloc(lbm_unet *n, T **p, size_t count) {
    cudaError_t e = cudaMalloc(reinterpret_cast<void **>(p), count * sizeof(T) + 16);
    if (e == cudaSuccess) n->allocs.push_back(*p);
    return e;
}

template <class... K, class... A>
cudaError_t launch(lbm_unet *n, bool early, void (*kernel)(K...), dim3 grid, int threads, int smem, A... args) {
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = grid;
    cfg.blockDim = dim3(threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = n->stream;
    cudaLaunchAttribute at{};
    at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at.val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = &at;
    cfg.numAttrs = early ? 1 : 0;
    return cudaLaunchKernelEx(&cfg, kernel, static_cast<K>(args)...);
}

// C channels of planes for max_batch images, all zero, with room before and after
// them that the convolutions' halos may read (zero as well)
cudaError_t palloc(lbm_unet *n, Planes *q, const nn::Geo &geo, int C) {
    const size_t front = (size_t)(geo.Wp + 16) / 8 * 8 + 8, back = nn::TC_M + geo.Wp + 32;
    q->str = (long long)n->cfg.max_batch * geo.PSI;
    const size_t px = front + (size_t)(C / 8) * q->str + back;
    bf16 *base = nullptr;
    cudaError_t e = nalloc(n, &base, px * 8);
    if (e == cudaSuccess) e = cudaMemsetAsync(base, 0, px * 8 * sizeof(bf16), n->stream);
    q->p = base + front * 8;
    return e;
}

void nrelease(lbm_unet *n) {
    if (!n) return;
    for (void *p : n->allocs) cudaFree(p);
    for (cudaStream_t s : n->side)
        if (s) cudaStreamDestroy(s);
    if (n->fork) cudaEventDestroy(n->fork);
    for (cudaEvent_t v : n->join)
        if (v) cudaEventDestroy(v);
    if (n->own_stream && n->stream) cudaStreamDestroy(n->stream);
    delete n;
}

int conv_index(const lbm_unet *n, const char kind, int l, int ab) {
    // order: enc0a enc0b ... enc{L-1}b, dec{L-2}a dec{L-2}b ... dec0b, head
    const int L = n->cfg.levels;
    if (kind == 'e') return 2 * l + ab;
    if (kind == 'd') return 2 * L + 2 * (L - 2 - l) + ab;
    return 2 * L + 2 * (L - 1);
}

constexpr int SMEM_MAX = 225 * 1024, SMEM_TWO = 111 * 1024;  // of one CTA; of each of two on an SM

template <int BN>
cudaError_t launch_tc(lbm_unet *n, nn::ConvOp &op) {
    using namespace nn;
    static bool attr = false;
    if (!attr) {
        cudaError_t e = cudaFuncSetAttribute(k_conv_tc<BN>, cudaFuncAttributeMaxDynamicSharedMemorySize, SMEM_MAX);
        if (e != cudaSuccess) return e;
        attr = true;
    }
    // A tile of A once for all taps: three row segments where a tile is shorter than a
    // row, else the run of pixels from the row above to the row below
    op.nseg = op.geo.Wp >= TC_M + 2 ? 3 : 1;
    op.segpx = op.nseg == 3 ? TC_M + 2 : TC_M + 2 * op.geo.Wp + 2;
    op.rowpx = op.nseg == 3 ? op.segpx : op.geo.Wp;
    const int a = op.Ge * op.nseg * op.segpx * 16;
    const int wall = op.KG * BN * 16 + (op.Ge == 1 ? TC_M * 16 : 0);  // and the tile of zeros
    int smem = 0;
    if (2 * a + wall <= SMEM_MAX) {  // all weights beside two tiles or more, two CTAs if they fit
        op.stages = 0;
        op.na = (2 * a + wall <= SMEM_TWO ? SMEM_TWO - wall : SMEM_MAX - wall) / a;
        if (op.na > 4) op.na = 4;
        smem = op.na * a + wall;
    } else {
        // the units of a row and two to come, and stages of weights (a copy is 2000 to
        // 3000 cycles on its way, a stage of 16 groups 400 to 512 of MMAs)
        // (24 groups, where that leaves three stages: a layer of 192 channels to 64 at 64 x
        // 128, 16 images: 57 -> 47 us)
        int unit = 0, wstage = 0;
        for (op.gb = op.Ge < TC_KB ? op.Ge : TC_KB;; op.gb -= 2) {
            if (op.Ge % op.gb) continue;
            unit = op.gb * (TC_M + 2) * 16, wstage = op.gb * BN * 16;
            op.na = op.Ge / op.gb + 2;
            if (op.na * unit + 3 * wstage > SMEM_MAX) op.na--;
            if (op.gb <= 16 || op.na * unit + 3 * wstage <= SMEM_MAX) break;
        }
        op.stages = (SMEM_MAX - op.na * unit) / wstage;
        if (op.stages > TC_MAX_STAGES) op.stages = TC_MAX_STAGES;
        smem = op.na * unit + op.stages * wstage;
    }
    const long long rows = (long long)op.B * op.geo.PSI - op.geo.Wp;
    op.ntile = (int)((rows + TC_M - 1) / TC_M);
    const int ny = n_tiles(op.N);
    int ctas = (smem <= SMEM_TWO ? 2 : 1) * n->sms / ny;
    if (ctas > op.ntile) ctas = op.ntile;
    if (ctas < 1) ctas = 1;
    return launch(n, n->early, k_conv_tc<BN>, dim3(ctas, ny), TC_THREADS, smem, op, n->wait_limit, n->err_d);
}

// src, out, mask: planes on geo (up: out on fine)
cudaError_t conv(lbm_unet *n, const bf16 *w, int Cs, int N, int sign, const float *bias, bool relu,
                 const Planes &src, const Planes *mask, const Planes &out, const nn::Geo &geo,
                 const nn::Geo *fine, int B) {
    nn::ConvOp op{};
    op.src = src.p;
    op.sstr = src.str;
    op.zero = n->zero;
    op.w = w;
    op.bias = bias;
    op.mask = mask ? mask->p : nullptr;
    op.out = out.p;
    op.ostr = out.str;
    op.geo = geo;
    op.up = fine ? 1 : 0;
    if (fine) op.fine = *fine;
    op.B = B;
    op.G = Cs / 8;
    op.N = N;
    const bool pairs = op.G == 1 && sign > 0;
    op.Ge = pairs ? 1 : op.G + (op.G & 1);
    op.KG = nn::k_groups(op.G, pairs);
    op.sign = sign;
    op.relu = relu;
    switch (nn::n_tile(N)) {
        case 32: return launch_tc<32>(n, op);
        case 64: return launch_tc<64>(n, op);
        case 96: return launch_tc<96>(n, op);
        default: return launch_tc<128>(n, op);
    }
}

cudaError_t conv_fwd(lbm_unet *n, const Conv &cv, const Planes &src, const Planes &out, const nn::Geo &geo,
                     const nn::Geo *fine, int B) {
    return conv(n, cv.fwd, cv.ci, cv.co, 1, n->w + cv.b_off, true, src, nullptr, out, geo, fine, B);
}

// gradient with respect to the conv's input (masked by mask > 0 when given)
cudaError_t conv_dgrad(lbm_unet *n, const Conv &cv, const Planes &dz, const Planes *mask, const Planes &dx,
                       const nn::Geo &geo, int B) {
    return conv(n, cv.bwd, cv.co, cv.ci, -1, nullptr, false, dz, mask, dx, geo, nullptr, B);
}

// K splits of a weight gradient: four per SM and tile of 128 (tap, ci) rows, at most one
// per 64 pixels (`blocks`).  An accumulator adds one split's pixels in series, each
// addition rounded towards zero in the tensor core, so the length of a split is part of
// the gradient's rounding, not only of its time.
int wg_splits(const lbm_unet *n, int ci, int co, long long blocks) {
    const int bn = co <= 32 ? 32 : (co <= 64 ? 64 : 128);
    const int z = 4 * n->sms / ((9 * ci + 127) / 128 * ((co + bn - 1) / bn));
    return z < 1 ? 1 : (z > blocks ? (int)blocks : z);
}

// Floats of the partial sums of any layer's gradient.
size_t part_size(const lbm_unet *n) {
    const nn::Geo g(n->cfg.height, n->cfg.width);
    const long long blocks = ((long long)n->cfg.max_batch * g.PSI + nn::WG_SPLIT - 1) / nn::WG_SPLIT;
    size_t most = (size_t)2 * n->sms * (3 * n->cfg.base + 4);  // the head
    for (const Conv &c : n->convs) {
        const size_t s = c.k == 1 ? 0 : (size_t)wg_splits(n, c.ci, c.co, blocks) * (9 * c.ci + 1) * c.co;
        if (s > most) most = s;
    }
    return most;
}

// dst = the sum of nz partial results' first cnt floats, dst2 that of the rest (cnt2)
cudaError_t sum_parts(const float *part, int nz, int cnt, int cnt2, float *dst, float *dst2, cudaStream_t st) {
    const int n4 = cnt / 4, m4 = cnt2 / 4;
    nn::k_sum_parts<<<(n4 + m4 + nn::SP_X - 1) / nn::SP_X, nn::SP_X * nn::SP_Z, 0, st>>>(
        reinterpret_cast<const float4 *>(part), nz, n4, m4, reinterpret_cast<float4 *>(dst),
        reinterpret_cast<float4 *>(dst2));
    return cudaGetLastError();
}

// The next side stream and its partial sums, once what the main stream has so far is done.
cudaError_t next_side(lbm_unet *n, cudaStream_t *st, float **part) {
    *st = n->side[n->turn];
    *part = n->part[n->turn];
    n->turn ^= 1;
    const cudaError_t e = cudaEventRecord(n->fork, n->stream);
    return e == cudaSuccess ? cudaStreamWaitEvent(*st, n->fork, 0) : e;
}

template <int BN>
cudaError_t launch_wg(lbm_unet *n, nn::WgradOp &op, float *dw, float *db, cudaStream_t st) {
    using namespace nn;
    static bool attr = false;
    if (!attr) {
        cudaError_t e = cudaFuncSetAttribute(k_wgrad_tc<BN>, cudaFuncAttributeMaxDynamicSharedMemorySize, SMEM_MAX);
        if (e != cudaSuccess) return e;
        attr = true;
    }
    const int stage = 16 * (op.runpx + 2) * 16 + BN / 8 * op.runpx * 16;
    const bool two = 2 * stage <= SMEM_TWO && 3 * BN <= 256;  // CTAs on an SM
    op.stages = (two ? SMEM_TWO : SMEM_MAX) / stage;
    if (op.stages > 4) op.stages = 4;
    const int gx = (3 * op.G + 15) / 16, gy = (op.Co + BN - 1) / BN;
    const long long blocks = (op.npix + WG_SPLIT - 1) / WG_SPLIT;
    int z = wg_splits(n, op.Ci, op.Co, blocks);
    op.perz = (blocks + z - 1) / z * WG_SPLIT;
    z = (int)((op.npix + op.perz - 1) / op.perz);
    k_wgrad_tc<BN><<<dim3(gx, gy, z), WG_THREADS, op.stages * stage, st>>>(op, n->wait_limit, n->err_d);
    cudaError_t e = cudaGetLastError();
    return e == cudaSuccess ? sum_parts(op.part, z, 9 * op.Ci * op.Co, op.Co, dw, db, st) : e;
}

cudaError_t conv_wgrad(lbm_unet *n, const Conv &cv, const Planes &dz, const Planes &x, const nn::Geo &geo, int B) {
    nn::WgradOp op{};
    op.x = x.p;
    op.xstr = x.str;
    op.dz = dz.p;
    op.zstr = dz.str;
    float *dw = n->g + cv.w_off, *db = n->g + cv.b_off;
    op.Wp = geo.Wp;
    op.PSI = geo.PSI;
    if (geo.W % 16 == 0) {
        // the pixels inside, an MMA's 16 from one row: no work for the borders, and a
        // sum in the order of the pixels of the images (four training steps of 16
        // images of 128 x 256: 6.25 -> 6.17 ms)
        op.W = geo.W;
        op.H = geo.H;
        op.npix = (long long)B * geo.H * geo.W;
        op.q0 = geo.Wp + 1;
        const int rows = geo.W < nn::WG_PX ? nn::WG_PX / geo.W : 1;
        op.runpx = (rows - 1) * geo.Wp + (geo.W < nn::WG_PX ? geo.W : nn::WG_PX);
    } else {
        // rows that are no multiple of 16: the planes as one row, borders and all
        op.W = op.npix = (long long)B * geo.PSI;
        op.H = 1;
        op.runpx = nn::WG_PX;
    }
    op.Ci = cv.ci;
    op.Co = cv.co;
    op.G = cv.ci / 8;
    cudaStream_t st;
    cudaError_t e = next_side(n, &st, &op.part);
    if (e != cudaSuccess) return e;
    return cv.co <= 32 ? launch_wg<32>(n, op, dw, db, st)
                       : (cv.co <= 64 ? launch_wg<64>(n, op, dw, db, st) : launch_wg<128>(n, op, dw, db, st));
}

lbm_status forward_chain(lbm_unet *n, const float *in_dev, float *out_dev, int B) {
    const int L = n->cfg.levels;
    const nn::Geo &g0 = n->lv[0].geo;
    const unsigned pixels = nn::blocks((long long)B * g0.H * g0.W);
    NCK(n, (nn::k_pack_input<<<pixels, nn::EW, 0, n->stream>>>(in_dev, n->x.p, B, g0), cudaGetLastError()));
    for (int l = 0; l < L; l++) {
        Level &v = n->lv[l];
        if (l > 0) {
            const Level &u = n->lv[l - 1];
            const dim3 grid(nn::blocks((long long)B * v.geo.H * v.geo.W), u.C / 8);
            NCK(n, launch(n, true, nn::k_pool, grid, nn::EW, 0, u.e.p, u.e.str, v.inp.p, v.inp.str, B, u.geo, v.geo));
        }
        NCK(n, conv_fwd(n, n->convs[conv_index(n, 'e', l, 0)], l > 0 ? v.inp : n->x, v.ea, v.geo, nullptr, B));
        // the deepest level's output is only used upsampled, as the channels before
        // the skip's in the level above
        const Level *u = l == L - 1 ? &n->lv[l - 1] : nullptr;
        NCK(n, conv_fwd(n, n->convs[conv_index(n, 'e', l, 1)], v.ea, u ? u->cat : v.e, v.geo,
                        u ? &u->geo : nullptr, B));
    }
    for (int l = L - 2; l >= 0; l--) {
        Level &v = n->lv[l];
        NCK(n, conv_fwd(n, n->convs[conv_index(n, 'd', l, 0)], v.cat, v.da, v.geo, nullptr, B));
        const Level *u = l > 0 ? &n->lv[l - 1] : nullptr;
        NCK(n, conv_fwd(n, n->convs[conv_index(n, 'd', l, 1)], v.da, u ? u->cat : v.d, v.geo,
                        u ? &u->geo : nullptr, B));
    }
    const Conv &hd = n->convs[conv_index(n, 'h', 0, 0)];
    const Planes &d = n->lv[0].d;
    NCK(n, launch(n, true, nn::k_head, pixels, nn::EW, 0, d.p, d.str, n->w + hd.w_off, n->w + hd.b_off, out_dev, B, g0,
                  n->lv[0].C));
    return LBM_OK;
}

lbm_status forward(lbm_unet *n, const float *in_dev, float *out_dev, int B) {
    n->early = true;
    const lbm_status st = forward_chain(n, in_dev, out_dev, B);
    n->early = false;
    return st;
}

// The main stream waits for the weight gradients so far.
cudaError_t join_side(lbm_unet *n) {
    for (int k = 0; k < 2; k++) {
        cudaError_t e = cudaEventRecord(n->join[k], n->side[k]);
        if (e == cudaSuccess) e = cudaStreamWaitEvent(n->stream, n->join[k], 0);
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

// The weight gradients run on two streams of their own in turn, each from the dz it sums
// on, so that the sums over one layer's splits are not in the way of the next layer:
// nothing before the optimizer needs them, and neither they nor the convolutions that
// carry the gradient on fill the chip (four training steps of 16 images of 128 x 256:
// 6.15 ms in one stream, 5.32 with one beside it, when the splits were added atomically).
// A level's g1 and g2 are written twice, by the decoder's and by the encoder's half: the
// second writes wait for the first half's weight gradients.
lbm_status backward_side(lbm_unet *n, const float *tgt_dev, const float *fl_dev, int B) {
    const int L = n->cfg.levels;
    const nn::Geo &g0 = n->lv[0].geo;
    const long long HW = (long long)g0.H * g0.W;
    NCK(n, (nn::k_count<<<nn::CNT_BLOCKS, nn::EW, 0, n->stream>>>(fl_dev, B * HW, n->cnt), cudaGetLastError()));
    NCK(n, (nn::k_loss<<<nn::LOSS_BLOCKS, nn::EW, 0, n->stream>>>(n->out, tgt_dev, fl_dev, n->cnt, n->dout,
                                                                  n->loss, B, (int)HW),
           cudaGetLastError()));
    // head: gradient of d0 (masked by d0 > 0) into lv[0].g1
    Level &v0 = n->lv[0];
    const Conv &hd = n->convs[conv_index(n, 'h', 0, 0)];
    unsigned hb = nn::blocks(B * HW);
    if (hb > 2u * n->sms) hb = 2u * n->sms;
    NCK(n, (nn::k_head_back<<<dim3(hb, v0.C / 8), nn::EW, 0, n->stream>>>(
               n->dout, v0.d.p, v0.d.str, n->w + hd.w_off, v0.g1.p, n->part[n->turn], B, g0, v0.C),
            cudaGetLastError()));
    cudaStream_t st;
    float *part;
    NCK(n, next_side(n, &st, &part));
    NCK(n, (nn::k_loss_sum<<<1, 32, 0, st>>>(n->loss), cudaGetLastError()));
    NCK(n, sum_parts(part, (int)hb, 3 * v0.C, 4, n->g + hd.w_off, n->g + hd.b_off, st));
    // decoder: g1 of level l holds d(d_l) (masked)
    for (int l = 0; l < L - 1; l++) {
        Level &v = n->lv[l];
        const Conv &cb = n->convs[conv_index(n, 'd', l, 1)], &ca = n->convs[conv_index(n, 'd', l, 0)];
        NCK(n, conv_wgrad(n, cb, v.g1, v.da, v.geo, B));
        NCK(n, conv_dgrad(n, cb, v.g1, &v.da, v.g2, v.geo, B));
        NCK(n, conv_wgrad(n, ca, v.g2, v.cat, v.geo, B));
        NCK(n, conv_dgrad(n, ca, v.g2, &v.cat, v.gcat, v.geo, B));
        Level &u = n->lv[l + 1];
        const dim3 grid(nn::blocks((long long)B * u.geo.H * u.geo.W), u.C / 8);
        NCK(n, (nn::k_up_back<<<grid, nn::EW, 0, n->stream>>>(v.gcat.p, v.gcat.str, u.g1.p, u.g1.str, B, v.geo, u.geo),
                cudaGetLastError()));
    }
    NCK(n, join_side(n));
    // encoder: g1 of level l holds d(e_l) (masked)
    for (int l = L - 1; l >= 0; l--) {
        Level &v = n->lv[l];
        const Conv &cb = n->convs[conv_index(n, 'e', l, 1)], &ca = n->convs[conv_index(n, 'e', l, 0)];
        NCK(n, conv_wgrad(n, cb, v.g1, v.ea, v.geo, B));
        NCK(n, conv_dgrad(n, cb, v.g1, &v.ea, v.g2, v.geo, B));
        NCK(n, conv_wgrad(n, ca, v.g2, l > 0 ? v.inp : n->x, v.geo, B));
        if (l == 0) break;
        NCK(n, conv_dgrad(n, ca, v.g2, nullptr, v.gin, v.geo, B));
        Level &u = n->lv[l - 1];
        const Planes skip = u.gcat.group(v.C / 8);
        const dim3 grid(nn::blocks((long long)B * u.geo.H * u.geo.W), u.C / 8);
        NCK(n, (nn::k_pool_back<<<grid, nn::EW, 0, n->stream>>>(v.gin.p, v.gin.str, u.e.p, skip.p, u.g1.p, u.g1.str, B,
                                                                v.geo, u.geo),
                cudaGetLastError()));
    }
    return LBM_OK;
}

lbm_status backward(lbm_unet *n, const float *tgt_dev, const float *fl_dev, int B) {
    const lbm_status st = backward_side(n, tgt_dev, fl_dev, B);
    NCK(n, join_side(n));  // also after an error: nothing is left behind on the side stream
    return st;
}

lbm_status stage_inputs(lbm_unet *n, const float *in, const float *tgt, const float *fl, int B,
                        int on_device, const float **din, const float **dtgt, const float **dfl) {
    const size_t HW = (size_t)n->cfg.height * n->cfg.width;
    if (on_device) {
        *din = in;
        if (dtgt) *dtgt = tgt;
        if (dfl) *dfl = fl;
        return LBM_OK;
    }
    NCK(n, cudaMemcpyAsync(n->io_in, in, (size_t)B * 8 * HW * sizeof(float), cudaMemcpyHostToDevice,
                           n->stream));
    *din = n->io_in;
    if (dtgt) {
        NCK(n, cudaMemcpyAsync(n->io_tgt, tgt, (size_t)B * 3 * HW * sizeof(float),
                               cudaMemcpyHostToDevice, n->stream));
        *dtgt = n->io_tgt;
    }
    if (dfl) {
        NCK(n, cudaMemcpyAsync(n->io_fl, fl, (size_t)B * HW * sizeof(float), cudaMemcpyHostToDevice,
                               n->stream));
        *dfl = n->io_fl;
    }
    return LBM_OK;
}

}  // namespace

extern "C" {

lbm_status lbm_unet_create(const lbm_unet_config *cfg, lbm_unet **out) {
    if (!cfg || !out) return nfail(nullptr, LBM_EINVAL, "null argument");
    *out = nullptr;
    const lbm_unet_config &c = *cfg;
    if (c.levels < 2 || c.levels > 4 || c.base < 8 || c.base % 8 || c.base > 64)
        return nfail(nullptr, LBM_EINVAL, "levels must be 2..4 and base a multiple of 8 up to 64");
    const int div = 1 << (c.levels - 1);
    if (c.height < div || c.width < div || c.height % div || c.width % div)
        return nfail(nullptr, LBM_EINVAL, "height and width must be multiples of %d", div);
    if (c.max_batch < 1 || (long long)c.max_batch * c.height * c.width >= (1ll << 31))
        return nfail(nullptr, LBM_EINVAL, "max_batch out of range");
    if (c.base != 8 && c.base != 16 && c.base != 32)
        return nfail(nullptr, LBM_EINVAL, "base must be 8, 16 or 32");
    if (cudaSetDevice(c.device) != cudaSuccess)
        return nfail(nullptr, LBM_ECUDA, "cannot select device %d", c.device);
    lbm_unet *n = new (std::nothrow) lbm_unet;
    if (!n) return nfail(nullptr, LBM_ENOMEM, "host allocation failed");
    n->cfg = c;
    if (cudaDeviceGetAttribute(&n->sms, cudaDevAttrMultiProcessorCount, c.device) != cudaSuccess ||
        n->sms < 1)
        n->sms = 1;
    if (c.stream) {
        n->stream = static_cast<cudaStream_t>(c.stream);
    } else {
        if (cudaStreamCreateWithFlags(&n->stream, cudaStreamNonBlocking) != cudaSuccess) {
            nrelease(n);
            return nfail(nullptr, LBM_ECUDA, "stream creation failed");
        }
        n->own_stream = true;
    }
    const int L = c.levels;
    // parameter layout
    std::vector<int> ch(L);
    for (int l = 0; l < L; l++) ch[l] = c.base << l;
    size_t off = 0;
    auto add = [&](int ci, int co, int k) {
        Conv cv;
        cv.ci = ci;
        cv.co = co;
        cv.k = k;
        cv.w_off = off;
        off += (size_t)co * ci * k * k;
        off = (off + 7) & ~size_t(7);  // keep every weight block 16-byte aligned in BF16
        cv.b_off = off;
        off += (co + 7) & ~7;
        n->nabi += (long long)co * ci * k * k + co;
        n->convs.push_back(cv);
    };
    int cin = 8;
    for (int l = 0; l < L; l++) {
        add(cin, ch[l], 3);
        add(ch[l], ch[l], 3);
        cin = ch[l];
    }
    for (int l = L - 2; l >= 0; l--) {
        add(ch[l + 1] + ch[l], ch[l], 3);
        add(ch[l], ch[l], 3);
    }
    add(ch[0], 3, 1);
    n->nparam = (long long)off;
    cudaError_t e = cudaSuccess;
    const size_t B = c.max_batch;
    e = nalloc(n, &n->w, off);
    if (e == cudaSuccess) e = nalloc(n, &n->g, off);
    if (e == cudaSuccess) e = nalloc(n, &n->m, off);
    if (e == cudaSuccess) e = nalloc(n, &n->v, off);
    // packed BF16 weights (zero where a tile or a pair of groups is padded) and the
    // table of the parameters' places
    long long abi = 0;
    for (Conv &cv : n->convs) {
        nn::ConvTab::E &t = n->tab.e[n->tab.n++];
        t = {(int)cv.w_off, (int)cv.b_off, (int)abi, cv.ci, cv.co, cv.k * cv.k, nullptr, nullptr, 0, 0, 0, 0, 0, 0};
        abi += (long long)cv.co * cv.ci * cv.k * cv.k + cv.co;
        if (cv.k == 1) continue;
        auto pack = [&](int N, int Cs, bool pairs, bf16 **p, int &BN, int &KG, int &Ge) {
            const int G = Cs / 8;
            BN = nn::n_tile(N);
            KG = nn::k_groups(G, pairs);
            Ge = pairs ? 1 : G + (G & 1);
            const size_t cnt = (size_t)nn::n_tiles(N) * KG * BN * 8;
            if (e == cudaSuccess) e = nalloc(n, p, cnt);
            if (e == cudaSuccess) e = cudaMemsetAsync(*p, 0, cnt * sizeof(bf16), n->stream);
        };
        pack(cv.co, cv.ci, cv.ci == 8, &cv.fwd, t.fBN, t.fKG, t.fGe);
        pack(cv.ci, cv.co, false, &cv.bwd, t.bBN, t.bKG, t.bGe);
        t.fwd = cv.fwd;
        t.bwd = cv.bwd;
    }
    const size_t HW = (size_t)c.height * c.width;
    if (e == cudaSuccess) e = cudaEventCreateWithFlags(&n->fork, cudaEventDisableTiming);
    for (int k = 0; k < 2 && e == cudaSuccess; k++) {
        e = cudaStreamCreateWithFlags(&n->side[k], cudaStreamNonBlocking);
        if (e == cudaSuccess) e = cudaEventCreateWithFlags(&n->join[k], cudaEventDisableTiming);
    }
    if (e == cudaSuccess) e = palloc(n, &n->x, nn::Geo(c.height, c.width), 8);
    const size_t zeros = (nn::TC_M + 2 * (c.width + 2) + 2) * 8;  // the longest copy of a convolution
    if (e == cudaSuccess) e = nalloc(n, &n->zero, zeros);
    if (e == cudaSuccess) e = cudaMemsetAsync(n->zero, 0, zeros * sizeof(bf16), n->stream);
    if (e == cudaSuccess) e = nalloc(n, &n->abi, (size_t)n->nabi);
    if (e == cudaSuccess) e = nalloc(n, &n->out, B * HW * 3);
    if (e == cudaSuccess) e = nalloc(n, &n->dout, B * HW * 3);
    if (e == cudaSuccess) e = nalloc(n, &n->io_in, B * HW * 8);
    if (e == cudaSuccess) e = nalloc(n, &n->io_tgt, B * HW * 3);
    if (e == cudaSuccess) e = nalloc(n, &n->io_fl, B * HW);
    for (int k = 0; k < 2 && e == cudaSuccess; k++) e = nalloc(n, &n->part[k], part_size(n));
    if (e == cudaSuccess) e = nalloc(n, &n->cnt, nn::CNT_BLOCKS);
    if (e == cudaSuccess) e = nalloc(n, &n->loss, 1 + nn::LOSS_BLOCKS);
    if (e == cudaSuccess) e = nalloc(n, &n->err_d, 1);
    if (e == cudaSuccess) e = cudaMemsetAsync(n->err_d, 0, sizeof(int), n->stream);
    n->lv.resize(L);
    for (int l = 0; l < L && e == cudaSuccess; l++) {
        Level &v = n->lv[l];
        v.geo = nn::Geo(c.height >> l, c.width >> l);
        v.C = ch[l];
        const int cprev = l > 0 ? ch[l - 1] : 8, cnext = l + 1 < L ? ch[l + 1] : 0;
        if (l > 0) e = palloc(n, &v.inp, v.geo, cprev);
        if (e == cudaSuccess) e = palloc(n, &v.ea, v.geo, v.C);
        if (l < L - 1) {
            if (e == cudaSuccess) e = palloc(n, &v.cat, v.geo, v.C + cnext);
            v.e = v.cat.group(cnext / 8);
            if (e == cudaSuccess) e = palloc(n, &v.da, v.geo, v.C);
            if (e == cudaSuccess && l == 0) e = palloc(n, &v.d, v.geo, v.C);
            if (e == cudaSuccess) e = palloc(n, &v.gcat, v.geo, v.C + cnext);
        }
        if (e == cudaSuccess) e = palloc(n, &v.g1, v.geo, v.C);
        if (e == cudaSuccess) e = palloc(n, &v.g2, v.geo, v.C);
        if (e == cudaSuccess && l > 0) e = palloc(n, &v.gin, v.geo, cprev);
    }
    if (e == cudaSuccess) e = cudaMemsetAsync(n->g, 0, off * sizeof(float), n->stream);  // the padding
    if (e == cudaSuccess) e = cudaMemsetAsync(n->m, 0, off * sizeof(float), n->stream);
    if (e == cudaSuccess) e = cudaMemsetAsync(n->v, 0, off * sizeof(float), n->stream);
    if (e != cudaSuccess) {
        lbm_status st = e == cudaErrorMemoryAllocation ? LBM_ENOMEM : LBM_ECUDA;
        nfail(nullptr, st, "lbm_unet_create: %s", cudaGetErrorString(e));
        nrelease(n);
        return st;
    }
    // He-normal weights (std sqrt(2 / fan_in)), zero biases, seeded: drawn in the order
    // [Cout][tap][Cin] of each convolution
    std::vector<float> w(n->nabi, 0.f);
    std::mt19937_64 rng(c.seed);
    std::normal_distribution<double> nd(0.0, 1.0);
    for (int k = 0; k < n->tab.n; k++) {
        const nn::ConvTab::E &t = n->tab.e[k];
        const double sd = std::sqrt(2.0 / (t.ci * t.taps));
        for (int co = 0; co < t.co; co++)
            for (int tap = 0; tap < t.taps; tap++)
                for (int ci = 0; ci < t.ci; ci++)
                    w[t.abi + ((size_t)co * t.ci + ci) * t.taps + tap] = (float)(sd * nd(rng));
    }
    e = cudaMemcpyAsync(n->abi, w.data(), w.size() * sizeof(float), cudaMemcpyHostToDevice, n->stream);
    if (e == cudaSuccess) {
        nn::k_from_abi<<<nn::blocks(n->nparam), nn::EW, 0, n->stream>>>(n->tab, n->abi, n->w, n->nparam);
        e = cudaGetLastError();
    }
    if (e == cudaSuccess) e = cudaStreamSynchronize(n->stream);
    if (e != cudaSuccess) {
        nfail(nullptr, LBM_ECUDA, "lbm_unet_create: %s", cudaGetErrorString(e));
        nrelease(n);
        return LBM_ECUDA;
    }
    *out = n;
    return LBM_OK;
}

lbm_status lbm_unet_destroy(lbm_unet *n) {
    if (!n) return LBM_OK;
    cudaSetDevice(n->cfg.device);
    cudaStreamSynchronize(n->stream);
    nrelease(n);
    return LBM_OK;
}

const char *lbm_unet_last_error(const lbm_unet *n) { return n ? n->err.c_str() : g_nn_error.c_str(); }

lbm_status lbm_unet_set_wait_limit(lbm_unet *n, int64_t polls) {
    if (!n || polls < 0) return LBM_EINVAL;
    n->wait_limit = (long long)polls;
    return LBM_OK;
}

int64_t lbm_unet_param_count(const lbm_unet *n) { return n ? n->nabi : -1; }

// a vector in the masters' layout to the caller, in the caller's order
static lbm_status export_abi(lbm_unet *n, const float *w, float *a, int32_t on_device) {
    float *to = on_device ? a : n->abi;
    NCK(n, (nn::k_to_abi<<<nn::blocks(n->nparam), nn::EW, 0, n->stream>>>(n->tab, w, to, n->nparam),
            cudaGetLastError()));
    if (!on_device)
        NCK(n, cudaMemcpyAsync(a, to, n->nabi * sizeof(float), cudaMemcpyDeviceToHost, n->stream));
    NCK(n, cudaStreamSynchronize(n->stream));
    return LBM_OK;
}

lbm_status lbm_unet_get_params(lbm_unet *n, float *a, int32_t on_device) {
    if (!n || !a) return LBM_EINVAL;
    NCK(n, cudaSetDevice(n->cfg.device));
    return export_abi(n, n->w, a, on_device);
}

lbm_status lbm_unet_set_params(lbm_unet *n, const float *a, int32_t on_device) {
    if (!n || !a) return LBM_EINVAL;
    NCK(n, cudaSetDevice(n->cfg.device));
    std::vector<float> h;
    if (on_device) {
        h.resize(n->nabi);
        NCK(n, cudaMemcpyAsync(h.data(), a, h.size() * sizeof(float), cudaMemcpyDeviceToHost, n->stream));
        NCK(n, cudaStreamSynchronize(n->stream));
    }
    const float *v = on_device ? h.data() : a;
    for (int64_t i = 0; i < n->nabi; i++)
        if (!std::isfinite(v[i])) return nfail(n, LBM_EINVAL, "non-finite parameter");
    NCK(n, cudaMemcpyAsync(n->abi, v, n->nabi * sizeof(float), cudaMemcpyHostToDevice, n->stream));
    NCK(n, (nn::k_from_abi<<<nn::blocks(n->nparam), nn::EW, 0, n->stream>>>(n->tab, n->abi, n->w, n->nparam),
            cudaGetLastError()));
    NCK(n, cudaMemsetAsync(n->m, 0, n->nparam * sizeof(float), n->stream));
    NCK(n, cudaMemsetAsync(n->v, 0, n->nparam * sizeof(float), n->stream));
    n->adam_t = 0;
    NCK(n, cudaStreamSynchronize(n->stream));
    return LBM_OK;
}

lbm_status lbm_unet_forward(lbm_unet *n, const float *in, float *out, int32_t B, int32_t on_device) {
    if (!n || !in || !out || B < 1 || B > n->cfg.max_batch) return LBM_EINVAL;
    NCK(n, cudaSetDevice(n->cfg.device));
    const float *din = nullptr;
    lbm_status st = stage_inputs(n, in, nullptr, nullptr, B, on_device, &din, nullptr, nullptr);
    if (st == LBM_OK) st = forward(n, din, on_device ? out : n->out, B);
    if (st != LBM_OK || on_device) return st;
    const size_t bytes = (size_t)B * 3 * n->cfg.height * n->cfg.width * sizeof(float);
    NCK(n, cudaMemcpyAsync(out, n->out, bytes, cudaMemcpyDeviceToHost, n->stream));
    return check_err(n);
}

lbm_status lbm_unet_gradients(lbm_unet *n, const float *in, const float *tgt, const float *fl,
                              int32_t B, float *grads, double *loss, int32_t on_device) {
    if (!n || !in || !tgt || !fl || !grads || B < 1 || B > n->cfg.max_batch) return LBM_EINVAL;
    NCK(n, cudaSetDevice(n->cfg.device));
    const float *din, *dt, *df;
    lbm_status st = stage_inputs(n, in, tgt, fl, B, on_device, &din, &dt, &df);
    if (st == LBM_OK) st = forward(n, din, n->out, B);
    if (st == LBM_OK) st = backward(n, dt, df, B);
    if (st != LBM_OK) return st;
    double l = 0.0;
    NCK(n, cudaMemcpyAsync(&l, n->loss, sizeof(double), cudaMemcpyDeviceToHost, n->stream));
    NCK(n, cudaStreamSynchronize(n->stream));
    st = check_err(n);
    if (st == LBM_OK) st = export_abi(n, n->g, grads, on_device);
    if (st != LBM_OK) return st;
    if (loss) *loss = l;
    return LBM_OK;
}

lbm_status lbm_unet_train_step(lbm_unet *n, const float *in, const float *tgt, const float *fl,
                               int32_t B, float lr, double *loss, int32_t on_device) {
    if (!n || !in || !tgt || !fl || B < 1 || B > n->cfg.max_batch || !(lr > 0.f)) return LBM_EINVAL;
    NCK(n, cudaSetDevice(n->cfg.device));
    const float *din, *dt, *df;
    lbm_status st = stage_inputs(n, in, tgt, fl, B, on_device, &din, &dt, &df);
    if (st == LBM_OK) st = forward(n, din, n->out, B);
    if (st == LBM_OK) st = backward(n, dt, df, B);
    if (st != LBM_OK) return st;
    n->adam_t++;
    const float c1 = (float)(1.0 - std::pow(0.9, (double)n->adam_t));
    const float c2 = (float)(1.0 - std::pow(0.999, (double)n->adam_t));
    NCK(n, (nn::k_adam<<<nn::blocks(n->nparam), nn::EW, 0, n->stream>>>(n->tab, n->w, n->g, n->m, n->v,
                                                                       n->nparam, lr, c1, c2),
           cudaGetLastError()));
    if (loss) {
        NCK(n, cudaMemcpyAsync(loss, n->loss, sizeof(double), cudaMemcpyDeviceToHost, n->stream));
        return check_err(n);
    }
    return LBM_OK;
}

lbm_status lbm_unet_input(lbm_unet *n, const int32_t *owner, double re, float *in) {
    if (!n || !owner || !in || !std::isfinite(re)) return LBM_EINVAL;
    NCK(n, cudaSetDevice(n->cfg.device));
    const int HW = n->cfg.height * n->cfg.width;
    NCK(n, (nn::k_case_input<<<nn::blocks(HW), nn::EW, 0, n->stream>>>(owner, (float)(re / 100.0), in, HW),
           cudaGetLastError()));
    return LBM_OK;
}

}  // extern "C"
