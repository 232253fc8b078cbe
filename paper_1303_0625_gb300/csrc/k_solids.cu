// Set-up and export kernels: initial populations, node flags, rasterising an
// added disk, and copies of the state in FP64 for the caller.  The per-step
// work of the solids lives in k_solid_step.cu.
#include "lbm_internal.cuh"

#include <cmath>

namespace gbm {

namespace {

// bit 0: the node is solid; bit i (1..8): the node x - e_i is solid or
// beyond a non-periodic edge, i.e. population i arrives by bounce-back.
__device__ __forceinline__ uint16_t node_flags(const Lattice &L, const uint16_t *owner, int x,
                                               int y) {
    uint16_t f = owner[cell_of(L, x, y)] != FLUID ? 1u : 0u;
#pragma unroll
    for (int i = 1; i < 9; i++) {
        int xs, ys;
        if (!locate(L, x - cx(i), y - cy(i), xs, ys) || owner[cell_of(L, xs, ys)] != FLUID)
            f |= (uint16_t)(1u << i);
    }
    return f;
}

// Rasterise solid s at (X, Y): lowest id wins.
__device__ __forceinline__ void stamp(const StepParams &p, int s, double X, double Y, double r) {
    const Box bx = disk_box(X, Y, r, 0);
    const DiskTest inside(X, Y, r);
    for (int c = threadIdx.x; c < bx.w * bx.h; c += blockDim.x) {
        const int iu = bx.x0 + c % bx.w, ju = bx.y0 + c / bx.w;
        if (!inside(iu, ju)) continue;
        int x, y;
        if (!locate(p.L, iu, ju, x, y)) continue;
        atomic_min_u16(p.owner + cell_of(p.L, x, y), (uint16_t)s);
    }
}

__global__ void k_tick(const StepParams p) { early_start(); *p.t += 1; }

// --------------------------------------------------------- initialisation

template <int P>
__global__ void k_init_populations(const StepParams p) {
    const Lattice &L = p.L;
    const int x = blockIdx.x * blockDim.x + threadIdx.x, y = blockIdx.y;
    if (x >= L.nx) return;
    double ux = p.u0x, uy = p.u0y;
    if (L.bc_x == LBM_OPEN) {
        const double h = (double)L.ny, yy = (double)y + 0.5;
        ux = 4.0 * p.umax * yy * (h - yy) / (h * h);
        uy = 0.0;
    }
    const double uu = ux * ux + uy * uy;
    const long long k = cell_of(L, x, y);
    for (int i = 0; i < 9; i++) {
        const double eu = cx(i) * ux + cy(i) * uy;
        const double f = p.rho0 * wgt<double>(i) * (1.0 + 3.0 * eu + 4.5 * eu * eu - 1.5 * uu);
        put64<P>(p.f0, L.plane, i, k, f);
        put64<P>(p.f1, L.plane, i, k, f);
    }
}

// Flags of every node; the row padding (nx <= x < pitch) is marked solid, so
// that the advection-collision kernel stores zeros there and never sends a
// padding node down the per-node path.
__global__ void k_flags_all(const StepParams p) {
    const int x = blockIdx.x * blockDim.x + threadIdx.x, y = blockIdx.y;
    if (x >= p.L.pitch) return;
    p.flags[cell_of(p.L, x, y)] = x < p.L.nx ? node_flags(p.L, p.owner, x, y) : (uint16_t)1u;
}

__global__ void __launch_bounds__(SOLID_BLOCK) k_stamp(const StepParams p, int s) {
    const DSolid &b = p.S[s];
    if (!solid_ok(b)) {
        if (threadIdx.x == 0) atomicOr(p.status, 2);
        return;
    }
    stamp(p, s, b.x, b.y, b.r);
}

__global__ void __launch_bounds__(SOLID_BLOCK) k_stamp_finish(const StepParams p, int s) {
    const DSolid &b = p.S[s];
    if (!solid_ok(b)) {
        if (threadIdx.x == 0) atomicOr(p.status, 2);
        return;
    }
    const Box bx = disk_box(b.x, b.y, b.r, 1);
    for (int c = threadIdx.x; c < bx.w * bx.h; c += blockDim.x) {
        int x, y;
        if (!locate(p.L, bx.x0 + c % bx.w, bx.y0 + c / bx.w, x, y)) continue;
        const long long k = cell_of(p.L, x, y);
        p.flags[k] = node_flags(p.L, p.owner, x, y);
    }
}

// ----------------------------------------------------------------- export

template <int P>
__global__ void k_export_populations(const StepParams p, double *out) {
    const Lattice &L = p.L;
    const int x = blockIdx.x * blockDim.x + threadIdx.x, y = blockIdx.y;
    if (x >= L.nx) return;
    const long long t = *p.t;
    const void *f = (t & 1) ? p.f1 : p.f0;
    const long long k = cell_of(L, x, y), n = (long long)L.nx * L.ny, o = (long long)y * L.nx + x;
    for (int i = 0; i < 9; i++) out[i * n + o] = f64<P>(f, L.plane, i, k);
}

template <int P>
__global__ void k_import_populations(const StepParams p, const double *in) {
    const Lattice &L = p.L;
    const int x = blockIdx.x * blockDim.x + threadIdx.x, y = blockIdx.y;
    if (x >= L.nx) return;
    const long long t = *p.t;
    void *f = (t & 1) ? p.f1 : p.f0;
    const long long k = cell_of(L, x, y), n = (long long)L.nx * L.ny, o = (long long)y * L.nx + x;
    for (int i = 0; i < 9; i++) put64<P>(f, L.plane, i, k, in[i * n + o]);
}

// Equilibrium initial state from a network prediction pred [3][ny][nx]
// (FP32): rho = 1 + R p0, u = U (p1, p2) at every fluid node (Eq. 8).
// With base, relative to the channel's Poiseuille flow (see lbm_nn.h).
template <int P>
__global__ void k_warm_start(const StepParams p, const float *pred, double U, double R, int base) {
    const Lattice &L = p.L;
    const int x = blockIdx.x * blockDim.x + threadIdx.x, y = blockIdx.y;
    if (x >= L.nx) return;
    const long long k = cell_of(L, x, y), n = (long long)L.nx * L.ny, o = (long long)y * L.nx + x;
    if (p.flags[k] & 1u) return;
    const long long t = *p.t;
    void *f = (t & 1) ? p.f1 : p.f0;
    double rho = 1.0 + R * (double)pred[o];
    double ux = U * (double)pred[n + o];
    const double uy = U * (double)pred[2 * n + o];
    if (base) {
        const double h = (double)L.ny, yy = (double)y + 0.5, nu = (p.tau - 0.5) / 3.0;
        ux += 4.0 * p.umax * yy * (h - yy) / (h * h);
        rho += p.rho0 - 1.0 + 24.0 * nu * p.umax * (double)(L.nx - 1 - x) / (h * h);
    }
    const double uu = ux * ux + uy * uy;
    for (int i = 0; i < 9; i++) {
        const double eu = cx(i) * ux + cy(i) * uy;
        put64<P>(f, L.plane, i, k, rho * wgt<double>(i) * (1.0 + 3.0 * eu + 4.5 * eu * eu - 1.5 * uu));
    }
}

// The same with the mass flux of every column made equal to the inlet's
// (open channel, walls in y): the steady flow carries the inlet's flux
// sum_y rho u_x through every column, and an error in it relaxes on the
// slowest scales of the channel.  One block per column x: rho and u_x of its
// fluid nodes as above (Poiseuille base), Q(x) = sum rho u_x and the inlet's
// Q_in = sum over column 0 of rho u_P (FP64, fixed tree), then
// u_x -> u_x Q_in / Q(x) and f = f^eq.
constexpr int WS_BLOCK = 128;

__device__ double block_sum_ws(double v, double *sh) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    __syncthreads();
    if (lane == 0) sh[w] = v;
    __syncthreads();
    double t = 0.0;
    for (int k = 0; k < WS_BLOCK / 32; k++) t += sh[k];
    return t;
}

template <int P>
__global__ void __launch_bounds__(WS_BLOCK) k_warm_start_flux(const StepParams p, const float *pred,
                                                              double U, double R) {
    __shared__ double sh[WS_BLOCK / 32];
    const Lattice &L = p.L;
    const int x = blockIdx.x;
    const long long n = (long long)L.nx * L.ny;
    const long long t = *p.t;
    void *f = (t & 1) ? p.f1 : p.f0;
    const double h = (double)L.ny, nu = (p.tau - 0.5) / 3.0;
    auto rho_at = [&](int xx, int y) {
        return p.rho0 + R * (double)pred[(long long)y * L.nx + xx] +
               24.0 * nu * p.umax * (double)(L.nx - 1 - xx) / (h * h);
    };
    auto up_at = [&](int y) {
        const double yy = (double)y + 0.5;
        return 4.0 * p.umax * yy * (h - yy) / (h * h);
    };
    double q = 0.0, qin = 0.0;
    for (int y = threadIdx.x; y < L.ny; y += WS_BLOCK) {
        if (!(p.flags[cell_of(L, 0, y)] & 1u)) qin += rho_at(0, y) * up_at(y);
        if (!(p.flags[cell_of(L, x, y)] & 1u))
            q += rho_at(x, y) * (up_at(y) + U * (double)pred[n + (long long)y * L.nx + x]);
    }
    q = block_sum_ws(q, sh);
    qin = block_sum_ws(qin, sh);
    const double scale = q > 0.0 ? qin / q : 1.0;
    for (int y = threadIdx.x; y < L.ny; y += WS_BLOCK) {
        const long long k = cell_of(L, x, y), o = (long long)y * L.nx + x;
        if (p.flags[k] & 1u) continue;
        const double rho = rho_at(x, y);
        const double ux = (up_at(y) + U * (double)pred[n + o]) * scale;
        const double uy = U * (double)pred[2 * n + o];
        const double uu = ux * ux + uy * uy;
        for (int i = 0; i < 9; i++) {
            const double eu = cx(i) * ux + cy(i) * uy;
            put64<P>(f, L.plane, i, k, rho * wgt<double>(i) * (1.0 + 3.0 * eu + 4.5 * eu * eu - 1.5 * uu));
        }
    }
}

// Network input of a case, [8][ny][nx] floats: 0 the solid mask, 1 Re / 100,
// 2 log10(Re) / 2, 3 the signed distance to the nearest disk surface / 16
// (clipped to [-1, 4]), 4 the axial distance from that disk's centre in its
// radii / 8 (clipped to [-1, 4]; positive downstream), 5 the channel's
// parabola 4 y'(ny - y') / ny^2 (y' = y + 1/2), 6 x / nx, 7 y' / ny - 1/2.
// Geometry from the solid table, centres at the current time.
__global__ void k_case_features(const StepParams p, float re, float *in) {
    const Lattice &L = p.L;
    const int x = blockIdx.x * blockDim.x + threadIdx.x, y = blockIdx.y;
    if (x >= L.nx) return;
    const long long n = (long long)L.nx * L.ny, o = (long long)y * L.nx + x;
    float dmin = 1e30f, ax = 0.f;
    for (int s = 0; s < p.nsolid; s++) {
        const DSolid &b = p.S[s];
        const float dx = (float)((double)x - b.x), dy = (float)((double)y - b.y);
        const float r = sqrtf(b.r2f);
        const float d = sqrtf(dx * dx + dy * dy) - r;
        if (d < dmin) {
            dmin = d;
            ax = dx / (8.f * r);
        }
    }
    if (p.nsolid == 0) dmin = 64.f;
    const float h = (float)L.ny, yy = (float)y + 0.5f;
    in[o] = p.owner[cell_of(L, x, y)] != FLUID ? 1.f : 0.f;
    in[n + o] = re / 100.f;
    in[2 * n + o] = log10f(re) / 2.f;
    in[3 * n + o] = fminf(fmaxf(dmin / 16.f, -1.f), 4.f);
    in[4 * n + o] = fminf(fmaxf(ax, -1.f), 4.f);
    in[5 * n + o] = 4.f * yy * (h - yy) / (h * h);
    in[6 * n + o] = (float)x / (float)L.nx;
    in[7 * n + o] = yy / h - 0.5f;
}

// Four nodes a thread: rows of 8192 nodes, 4096 of them: 38 us, with one 134.
__global__ void k_export_owner(const StepParams p, int32_t *out) {
    const Lattice &L = p.L;
    const int x = 4 * (blockIdx.x * blockDim.x + threadIdx.x), y = blockIdx.y;
    if (x >= L.nx) return;
    // the pitch is a multiple of 64; out is the caller's, its rows not padded
    const ushort4 s = *reinterpret_cast<const ushort4 *>(p.owner + cell_of(L, x, y));
    const uint16_t v[4] = {s.x, s.y, s.z, s.w};
    int32_t o[4];
#pragma unroll
    for (int j = 0; j < 4; j++) o[j] = v[j] == FLUID ? -1 : (int32_t)v[j];
    int32_t *to = out + (long long)y * L.nx + x;
    if ((reinterpret_cast<uintptr_t>(to) & 15) == 0 && x + 4 <= L.nx) {
        *reinterpret_cast<int4 *>(to) = make_int4(o[0], o[1], o[2], o[3]);
        return;
    }
#pragma unroll
    for (int j = 0; j < 4; j++)
        if (x + j < L.nx) to[j] = o[j];
}

// Density and velocity: r = sum f_i, u = (sum e_i f_i - F / 2) / r, in 64 bits without
// FP64 arithmetic, of which GB300 issues about two lanes per clock and SM: one FP64
// operation of a warp takes as long as 32 or more of its integer operations.  Sums: the
// populations (in the deviation modes d_i = f_i - w_i) as 64-bit integers in units of
// 2^-60 (FP64: 2^-58; bits below, 1e-18, are cut off, less than an FP64 addition
// rounds), so exact.  Division: a fixed-point reciprocal of r and one product each,
// rounded once: 0.63 units in the last place at most, half of one and the reciprocal's
// 2^-56, an eighth of one for a mantissa close to 2.  8192 x 4096 nodes, FP32 and
// FP16: 0.50 ms (its bytes at the copy rate: 0.30 and 0.21; the integer units bound it);
// with the sums alone in integers 1.01, all in FP64 3.79.  FP64, 2048 x 1024: 42 us (28),
// before 172.
template <int P> struct Fixed;
template <> struct Fixed<LBM_FP32_DEV> {
    static constexpr int BITS = 60;
    static constexpr long long ONE = 1ll << BITS;  // added to the sum of the d_i
    // false: |d| >= 1/2 or not a number
    static __device__ __forceinline__ bool from(float d, long long &q) {
        const int b = __float_as_int(d), e = (b >> 23) & 0xFF, sh = e - 90;
        const unsigned m = (b & 0x7FFFFF) | 0x800000;  // subnormals and zeros: shifted out
        const unsigned long long v =
            sh >= 0 ? (unsigned long long)m << sh : (unsigned long long)(m >> min(-sh, 31));
        q = b < 0 ? -(long long)v : (long long)v;
        return e < 126;
    }
};
template <> struct Fixed<LBM_FP16_DEV> : Fixed<LBM_FP32_DEV> {};
template <> struct Fixed<LBM_FP64> {
    static constexpr int BITS = 58;
    static constexpr long long ONE = 0;
    // false: |f| >= 1 or not a number
    static __device__ __forceinline__ bool from(double f, long long &q) {
        const long long b = __double_as_longlong(f);
        const int e = (int)(b >> 52) & 0x7FF, sh = e - 1017;
        const unsigned long long m = (b & 0xFFFFFFFFFFFFFll) | 0x10000000000000ll;
        const unsigned long long v = sh >= 0 ? m << min(sh, 5) : m >> min(-sh, 63);
        q = b < 0 ? -(long long)v : (long long)v;
        return e < 1023;
    }
};

// p 2^(e - 64), p > 0, rounded to nearest (the exponent far from the ends of its range).
__device__ __forceinline__ double packed64(unsigned long long p, int e, bool negative) {
    const int n = __clzll((long long)p);
    p <<= n;
    const long long m = (long long)(p >> 11) + (long long)(p >> 10 & 1);
    const long long b = ((long long)(e - n + 1021) << 52) + m;
    return __longlong_as_double(negative ? b | 0x8000000000000000ll : b);
}

// 2^122 / r for r in [2^59, 2^61), to 2^-56 of it: FP32's approximation of 1 / r to about
// 22 bits, y, then y (1 + e + e^2) with e = 1 - r y in fixed point.  (Two units in the last
// place of y, the bound of __fdividef, leave |e| below 2^-21; the square from e's upper 16
// bits is then within 2^-56.3.)
__device__ __forceinline__ unsigned long long reciprocal62(unsigned long long r) {
    const unsigned rh = (unsigned)(r >> 32), rl = (unsigned)r;
    const unsigned y = (unsigned)(__fdividef(1.f, (float)rh * 0x1p-28f) * 0x1p30f);
    const long long ry = (long long)((unsigned long long)rh * y + ((unsigned long long)rl * y >> 32));
    const long long e = (1ll << 58) - ry;  // below 2^37
    const int es = (int)(e >> 22);
    const long long t = e + (long long)(es * es >> 14);
    return ((unsigned long long)y << 32) + ((unsigned long long)y * (unsigned)t >> 26) +
           (unsigned long long)(((long long)y * (int)(t >> 32)) * 64);
}

// j / r from y = reciprocal62(r): j in units of 2^-BITS.
template <int BITS>
__device__ __forceinline__ double quotient62(long long j, unsigned long long y) {
    if (j == 0) return 0.0;
    unsigned long long a = j < 0 ? -(unsigned long long)j : (unsigned long long)j;
    const int n = __clzll((long long)a);
    a <<= n;
    const unsigned ah = (unsigned)(a >> 32), al = (unsigned)a, yh = (unsigned)(y >> 32), yl = (unsigned)y;
    const unsigned long long q = (unsigned long long)ah * yh + ((unsigned long long)ah * yl >> 32) +
                                 ((unsigned long long)al * yh >> 32);
    return packed64(q, 66 - n - BITS, j < 0);
}

// half_x, half_y: F / 2 in units of 2^-BITS, or fixed = false.  Nodes outside the range
// of the fixed-point form (1/2 <= r < 2) take FP64 arithmetic.
template <int P>
__global__ void k_fields(const StepParams p, bool fixed, long long half_x, long long half_y, double *rho, double *ux,
                         double *uy) {
    using S = typename Prec<P>::S;
    using X = Fixed<P>;
    const Lattice &L = p.L;
    const int x = blockIdx.x * blockDim.x + threadIdx.x, y = blockIdx.y;
    if (x >= L.nx) return;
    const long long t = *p.t;
    const S *f = static_cast<const S *>((t & 1) ? p.f1 : p.f0);
    const long long k = cell_of(L, x, y), o = (long long)y * L.nx + x;
    if (p.owner[k] != FLUID) {
        rho[o] = ux[o] = uy[o] = __longlong_as_double(0x7ff8000000000000ll);
        return;
    }
    typename Prec<P>::C d[9];
#pragma unroll
    for (int i = 0; i < 9; i++) d[i] = ldc(f + i * L.plane + k);
    long long q[9];
#pragma unroll
    for (int i = 0; i < 9; i++) fixed &= X::from(d[i], q[i]);
    const long long a = q[5] - q[7], b = q[6] - q[8];
    const long long r60 = (((q[0] + q[1]) + (q[2] + q[3])) + ((q[4] + q[5]) + (q[6] + q[7])) + q[8] + X::ONE)
                          << (60 - X::BITS);
    if (fixed && r60 >= 1ll << 59 && r60 < 1ll << 61) {
        const unsigned long long inv = reciprocal62((unsigned long long)r60);
        rho[o] = packed64((unsigned long long)r60, 4, false);
        ux[o] = quotient62<X::BITS>(q[1] - q[3] + a - b - half_x, inv);
        uy[o] = quotient62<X::BITS>(q[2] - q[4] + a + b - half_y, inv);
        return;
    }
    double v[9];
#pragma unroll
    for (int i = 0; i < 9; i++) v[i] = Prec<P>::dev ? (double)d[i] + wgt<double>(i) : (double)d[i];
    const double c = v[5] - v[7], e = v[6] - v[8];
    const double r = ((v[0] + v[1]) + (v[2] + v[3])) + ((v[4] + v[5]) + (v[6] + v[7])) + v[8];
    rho[o] = r;
    ux[o] = ((v[1] - v[3]) + (c - e) - 0.5 * p.body_x) / r;
    uy[o] = ((v[2] - v[4]) + (c + e) - 0.5 * p.body_y) / r;
}

// bit i of mask[y][x]: fluid node x has a link along e_i (x + e_i solid).
__global__ void k_link_masks(const StepParams p, uint8_t *mask) {
    const Lattice &L = p.L;
    const int x = blockIdx.x * blockDim.x + threadIdx.x, y = blockIdx.y;
    if (x >= L.nx) return;
    uint8_t m = 0;
    if (p.owner[cell_of(L, x, y)] == FLUID) {
        for (int i = 1; i < 9; i++) {
            int xb, yb;
            if (locate(L, x + cx(i), y + cy(i), xb, yb) && p.owner[cell_of(L, xb, yb)] != FLUID)
                m |= (uint8_t)(1u << (i - 1));
        }
    }
    mask[(long long)y * L.nx + x] = m;
}

// covers the row padding too: (nx + 127) / 128 * 128 >= pitch = (nx + 63) / 64 * 64
dim3 cell_grid(const Lattice &L) { return dim3((L.nx + 127) / 128, L.ny); }

}  // namespace

// ------------------------------------------------------------ launchers

cudaError_t launch_tick(const StepParams &p, cudaStream_t st) {
    return launch_step(p, k_tick, dim3(1), 1, st, p);
}

cudaError_t launch_init_populations(const StepParams &p, cudaStream_t st) {
    switch (p.precision) {
        case LBM_FP64: k_init_populations<LBM_FP64><<<cell_grid(p.L), 128, 0, st>>>(p); break;
        case LBM_FP32_DEV: k_init_populations<LBM_FP32_DEV><<<cell_grid(p.L), 128, 0, st>>>(p); break;
        default: k_init_populations<LBM_FP16_DEV><<<cell_grid(p.L), 128, 0, st>>>(p);
    }
    return cudaGetLastError();
}

cudaError_t launch_flags_all(const StepParams &p, cudaStream_t st) {
    k_flags_all<<<cell_grid(p.L), 128, 0, st>>>(p);
    return cudaGetLastError();
}

cudaError_t launch_stamp_solid(const StepParams &p, int id, cudaStream_t st) {
    k_stamp<<<1, SOLID_BLOCK, 0, st>>>(p, id);
    k_stamp_finish<<<1, SOLID_BLOCK, 0, st>>>(p, id);
    return cudaGetLastError();
}

cudaError_t launch_export_populations(const StepParams &p, double *out, cudaStream_t st) {
    switch (p.precision) {
        case LBM_FP64: k_export_populations<LBM_FP64><<<cell_grid(p.L), 128, 0, st>>>(p, out); break;
        case LBM_FP32_DEV: k_export_populations<LBM_FP32_DEV><<<cell_grid(p.L), 128, 0, st>>>(p, out); break;
        default: k_export_populations<LBM_FP16_DEV><<<cell_grid(p.L), 128, 0, st>>>(p, out);
    }
    return cudaGetLastError();
}

cudaError_t launch_import_populations(const StepParams &p, const double *in, cudaStream_t st) {
    switch (p.precision) {
        case LBM_FP64: k_import_populations<LBM_FP64><<<cell_grid(p.L), 128, 0, st>>>(p, in); break;
        case LBM_FP32_DEV: k_import_populations<LBM_FP32_DEV><<<cell_grid(p.L), 128, 0, st>>>(p, in); break;
        default: k_import_populations<LBM_FP16_DEV><<<cell_grid(p.L), 128, 0, st>>>(p, in);
    }
    return cudaGetLastError();
}

cudaError_t launch_warm_start(const StepParams &p, const float *pred, double u_scale,
                              double rho_scale, int base, cudaStream_t st) {
    if (base & 2) {  // the column flux made equal to the inlet's (with the Poiseuille base)
        switch (p.precision) {
            case LBM_FP64: k_warm_start_flux<LBM_FP64><<<p.L.nx, WS_BLOCK, 0, st>>>(p, pred, u_scale, rho_scale); break;
            case LBM_FP32_DEV: k_warm_start_flux<LBM_FP32_DEV><<<p.L.nx, WS_BLOCK, 0, st>>>(p, pred, u_scale, rho_scale); break;
            default: k_warm_start_flux<LBM_FP16_DEV><<<p.L.nx, WS_BLOCK, 0, st>>>(p, pred, u_scale, rho_scale);
        }
        return cudaGetLastError();
    }
    const dim3 g = cell_grid(p.L);
    switch (p.precision) {
        case LBM_FP64: k_warm_start<LBM_FP64><<<g, 128, 0, st>>>(p, pred, u_scale, rho_scale, base); break;
        case LBM_FP32_DEV: k_warm_start<LBM_FP32_DEV><<<g, 128, 0, st>>>(p, pred, u_scale, rho_scale, base); break;
        default: k_warm_start<LBM_FP16_DEV><<<g, 128, 0, st>>>(p, pred, u_scale, rho_scale, base);
    }
    return cudaGetLastError();
}

cudaError_t launch_case_features(const StepParams &p, double re, float *in, cudaStream_t st) {
    k_case_features<<<cell_grid(p.L), 128, 0, st>>>(p, (float)re, in);
    return cudaGetLastError();
}

cudaError_t launch_export_owner(const StepParams &p, int32_t *out, cudaStream_t st) {
    k_export_owner<<<dim3((p.L.nx + 511) / 512, p.L.ny), 128, 0, st>>>(p, out);
    return cudaGetLastError();
}

template <int P>
cudaError_t launch_fields_p(const StepParams &p, double *rho, double *ux, double *uy, cudaStream_t st) {
    const bool fixed = std::fabs(p.body_x) < 0.5 && std::fabs(p.body_y) < 0.5;
    auto half = [&](double f) { return fixed ? std::llrint(std::ldexp(0.5 * f, Fixed<P>::BITS)) : 0ll; };
    k_fields<P><<<cell_grid(p.L), 128, 0, st>>>(p, fixed, half(p.body_x), half(p.body_y), rho, ux, uy);
    return cudaGetLastError();
}

cudaError_t launch_fields(const StepParams &p, double *rho, double *ux, double *uy,
                          cudaStream_t st) {
    switch (p.precision) {
        case LBM_FP64: return launch_fields_p<LBM_FP64>(p, rho, ux, uy, st);
        case LBM_FP32_DEV: return launch_fields_p<LBM_FP32_DEV>(p, rho, ux, uy, st);
        default: return launch_fields_p<LBM_FP16_DEV>(p, rho, ux, uy, st);
    }
}

cudaError_t launch_link_masks(const StepParams &p, uint8_t *mask, cudaStream_t st) {
    k_link_masks<<<cell_grid(p.L), 128, 0, st>>>(p, mask);
    return cudaGetLastError();
}

}  // namespace gbm
