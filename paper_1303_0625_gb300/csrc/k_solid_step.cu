// Per-solid work of one step t -> t+1.
//
// k_forces, one block per solid (or k_links, one or several blocks per solid, and
// k_record, one warp per solid, which may run beside the advection-collision kernel or
// after it), comes first:
//   the link sums of Eq. 4 and Eq. 5 over every fluid-solid link of time t (Eq. 6
//   and Eq. 7), and in the FP64 and FP32 modes the population each link returns,
//   left in the solid node's slot for the advection-collision kernel to pull;
//   the momentum booked by the node-type changes of the previous step (the
//   solid's segment of the event list) -> the force record of t; the motion
//   t -> t+1 (prescribed, or Newton-Euler on the Eq. 5 force; Eq. 4 when the
//   context selects it for comparison); the largest displacement of any solid
//   since the last pair test.
// k_ring, one warp per moving solid, reads no population and writes nothing that
// the advection-collision kernel reads: it may run beside it.
//   P  only when some solid may have come within reach of another one since
//      the last test: the solid's near list, the solids whose centres are
//      closer than r_s + r_q + NEAR_REACH + NEAR_MARGIN at t or t+1
//   R  on the ring (old disk XOR new disk): the owner at t and at t+1 from
//      the geometry of the solid and of its near list (lowest id where disks
//      overlap), so that no map of the old owners is kept; every node whose
//      owner changes goes to the step's change list; covered and fresh nodes
//      are queued per warp in lane order and published as the solid's
//      segment of the step's event list.
// k_changes and k_events follow all three (few moving solids: k_remask_few, one launch):
//   A  the change list into the owner map and the node flags (a node on the
//      rings of several solids is listed by each with the same owner; flag
//      bits are set and cleared atomically); the clock advances
//   E  after that: every warp of the grid takes events from the list: a fresh
//      node is refilled by extrapolation (Sec. IV.B) from nodes fluid at t and
//      at t+1; each event's momentum and torque go to its own slot; the moving
//      solids' state becomes t+1.
//
// Work per solid follows its perimeter: the nodes near the ends of the disk's
// chord in every row (FP32 bounds with a one-node margin) are dealt out to the
// threads; every decision is taken by the exact test.
//
// Precision: per-link products and a candidate's sum over its links (up to eight) are in
// the arithmetic precision of the storage mode (FP32 in the deviation modes), and so is
// the sum over the 32 candidates that a warp takes at once (in a batch: FP64); the sums
// of these, the booked momenta and the motion are FP64, in a fixed order.
#include "lbm_internal.cuh"

#include <algorithm>
#include <atomic>

namespace gbm {

namespace {

constexpr int SW_BLOCK = 256;
constexpr int WARPS = SW_BLOCK / 32;
constexpr double PI = 3.14159265358979323846;
constexpr unsigned FULL = 0xffffffffu;

// ------------------------------------------------------------- barrier

// Barrier of a grid that is one cluster (few moving solids): the hardware's, which no
// block can fail to reach.  A limit of 0 polls gives up at once (the time-out path's
// test): false, and status bit 2 raised; the caller's block then returns.
__device__ bool cluster_sync(const StepParams &p) {
    if (p.spin_limit <= 0) {
        if (threadIdx.x == 0) atomicOr(p.status, 4);
        return false;
    }
    __threadfence();
    asm volatile("barrier.cluster.arrive.release;\nbarrier.cluster.wait.acquire;\n" ::: "memory");
    return true;
}

// ------------------------------------------------------------- helpers

template <class T, int N>
__device__ __forceinline__ void warp_sum(T (&v)[N]) {
#pragma unroll
    for (int k = 0; k < N; k++)
        for (int o = 16; o > 0; o >>= 1) v[k] += __shfl_down_sync(FULL, v[k], o);
}

// The warp's sums of the lanes' six values: component sum_of(lane) in each lane whose
// sum_of is below 6.  Halves of the values go to the other lane of a pair at each step, so
// that a warp issues 9 additions instead of 30, over the same tree (FP64: two lanes per
// clock and SM).
__device__ __forceinline__ int sum_of(int lane) { return lane & 3 ? 6 : lane >> 2; }
template <class T>
__device__ __forceinline__ T warp_sum6(const T (&v)[6], int lane) {
    const bool a = lane & 16, b = lane & 8, c = lane & 4;
    T h[4], q[2];
#pragma unroll
    for (int k = 0; k < 4; k++) {
        const T up = k < 2 ? v[4 + (k & 1)] : T(0);
        h[k] = (a ? up : v[k]) + __shfl_xor_sync(FULL, a ? v[k] : up, 16);
    }
#pragma unroll
    for (int k = 0; k < 2; k++) q[k] = (b ? h[k + 2] : h[k]) + __shfl_xor_sync(FULL, b ? h[k] : h[k + 2], 8);
    T s = (c ? q[1] : q[0]) + __shfl_xor_sync(FULL, c ? q[0] : q[1], 4);
    s += __shfl_xor_sync(FULL, s, 2);
    return s + __shfl_xor_sync(FULL, s, 1);
}
// The same, WIDE: added in FP64, else in the type they come in.
template <bool WIDE, class T>
__device__ __forceinline__ double chunk_sum(const T (&v)[6], int lane) {
    if constexpr (!WIDE) return (double)warp_sum6(v, lane);
    const double w[6] = {(double)v[0], (double)v[1], (double)v[2], (double)v[3], (double)v[4], (double)v[5]};
    return warp_sum6(w, lane);
}

// Set or clear one bit of a 16-bit flags word atomically.
__device__ __forceinline__ void flag_bit(uint16_t *flags, long long k, int bit, bool on) {
    const uintptr_t a = reinterpret_cast<uintptr_t>(flags + k);
    unsigned int *w = reinterpret_cast<unsigned int *>(a & ~uintptr_t(3));
    const unsigned int m = (1u << bit) << ((a & 2) ? 16 : 0);
    if (on) atomicOr(w, m);
    else atomicAnd(w, ~m);
}

__device__ __forceinline__ double cvt_s(double v) { return v; }
__device__ __forceinline__ float cvt_s(float v) { return v; }
__device__ __forceinline__ float cvt_s(__half v) { return __half2float(v); }

// Centre split into an integer part and an FP32 fraction, for FP32 bounds
// on the nodes of a row that lie within some radius of it.
struct Centre {
    int xi, yi;
    float fx, fy;
    __device__ __forceinline__ Centre(int xi_, int yi_, float fx_, float fy_)
        : xi(xi_), yi(yi_), fx(fx_), fy(fy_) {}
    __device__ __forceinline__ Centre(double X, double Y) {
        const double a = floor(X), b = floor(Y);
        xi = (int)a;
        yi = (int)b;
        fx = (float)(X - a);
        fy = (float)(Y - b);
    }
    // The integers of row j within rr of the centre, [a, b] (a > b: none),
    // from the FP32 chord; false when the row misses the circle.
    __device__ __forceinline__ bool chord(int j, float rr, int &a, int &b) const {
        const float dy = (float)(j - yi) - fy;
        const float h2 = rr * rr - dy * dy;
        if (h2 < 0.f) return false;
        const float h = sqrtf(h2);
        a = xi + (int)ceilf(fx - h);
        b = xi + (int)floorf(fx + h);
        return true;
    }
};

// Cell of the neighbour (x + dx, y + dy) of an in-domain node (|dx|, |dy|
// <= 3), or -1 beyond a non-periodic edge.
__device__ __forceinline__ int neighbour(const Lattice &L, int x, int y, int dx, int dy) {
    x += dx;
    y += dy;
    if (x < 0 || x >= L.nx) {
        if (L.bc_x != LBM_PERIODIC) return -1;
        x += x < 0 ? L.nx : -L.nx;
    }
    if (y < 0 || y >= L.ny) {
        if (L.bc_y != LBM_PERIODIC) return -1;
        y += y < 0 ? L.ny : -L.ny;
    }
    return y * L.pitch + x;
}

// Unwrapped node coordinates near one disk -> domain nodes, without integer
// division: along a periodic axis the nodes within WRAP_REACH of the centre
// lie within one period of the image offset taken once per disk (the domain
// is wider than 2 r + 8).
constexpr int WRAP_REACH = 8;
__host__ __device__ __forceinline__ int floor_div(int a, int n) {
    return a >= 0 ? a / n : -((n - 1 - a) / n);
}
struct Wrap {
    int ox, oy, nx, ny;
    bool px, py;
    // ix, iy = floor of the centre, rc = ceil(r)
    __device__ __forceinline__ Wrap(const Lattice &L, int ix, int iy, int rc) {
        nx = L.nx;
        ny = L.ny;
        px = L.bc_x == LBM_PERIODIC;
        py = L.bc_y == LBM_PERIODIC;
        ox = px ? nx * floor_div(ix - rc - WRAP_REACH, nx) : 0;
        oy = py ? ny * floor_div(iy - rc - WRAP_REACH, ny) : 0;
    }
    __device__ __forceinline__ bool operator()(int i, int j, int &x, int &y) const {
        x = i - ox;
        y = j - oy;
        if (px) {
            while (x >= nx) x -= nx;  // at most twice
        } else if ((unsigned)x >= (unsigned)nx) {
            return false;
        }
        if (py) {
            while (y >= ny) y -= ny;
        } else if ((unsigned)y >= (unsigned)ny) {
            return false;
        }
        return true;
    }
};

// Up to two x-ranges of a row; the second is empty when a1 > b1.
struct Ranges {
    int a0, b0, a1, b1;
};

// Nodes of row j that can lie inside exactly one of two disks of radius r
// centred at c0 and c1: between the chord ends of radius r + RING_EPS (a
// superset of each disk's nodes in the row) and those of r - RING_EPS (a
// subset), at the left and at the right.  RING_EPS is far above the FP32
// rounding of a chord end (a few 1e-3 where the chord is short), so the exact
// boundary node of each disk lies between the two; the exact test decides.
constexpr float RING_EPS = 0.05f;
__device__ __forceinline__ bool ring_ranges(const Centre &c0, const Centre &c1, float r, int j,
                                            Ranges &R) {
    int a0, b0, a1, b1, p0, q0, p1, q1;
    bool h0 = c0.chord(j, r + RING_EPS, a0, b0), h1 = c1.chord(j, r + RING_EPS, a1, b1);
    h0 = h0 && a0 <= b0;
    h1 = h1 && a1 <= b1;
    if (!h0 && !h1) return false;
    R.a1 = 1;
    R.b1 = 0;
    const bool i0 = h0 && c0.chord(j, r - RING_EPS, p0, q0) && p0 <= q0;
    const bool i1 = h1 && c1.chord(j, r - RING_EPS, p1, q1) && p1 <= q1;
    if (!i0 || !i1) {  // the row is near the top or bottom of a disk: the whole union
        R.a0 = h0 ? (h1 ? min(a0, a1) : a0) : a1;
        R.b0 = h0 ? (h1 ? max(b0, b1) : b0) : b1;
        return true;
    }
    R.a0 = min(a0, a1);
    R.b0 = max(p0, p1) - 1;  // left: first node of the outer chords .. last before the inner
    R.a1 = min(q0, q1) + 1;  // right: after the inner chords .. last of the outer
    R.b1 = max(b0, b1);
    if (R.a1 <= R.b0 + 1) {  // the two ends meet: one range
        R.b0 = R.b1;
        R.a1 = 1;
        R.b1 = 0;
    }
    return true;
}

// Rows a disk can touch at either of two centres (floor iy0, iy1; rc =
// ceil(r)), with a margin of g: a superset of rows_of's.
__device__ __forceinline__ void rows_of_i(int iy0, int iy1, int rc, int g, int &j0, int &j1) {
    j0 = min(iy0, iy1) - rc - g;
    j1 = max(iy0, iy1) + rc + 1 + g;
}

// Deals the nodes of rows j0..j1 (the ranges that rng(j, R) gives for each
// row) to the lanes of the warp, NB nodes per lane at a time: fetch(i, j, u)
// is called for all NB nodes of a lane first, then process(u, ok) for each, on
// every lane of the warp together (ok is false for items past the end and for
// nodes fetch rejected).  Rows come in blocks of 32, one to a lane.
template <int NB, class RF, class FF, class PF>
__device__ __forceinline__ void warp_nodes_n(int j0, int j1, int lane, RF &&rng, FF &&fetch, PF &&process) {
    for (int jb = j0; jb <= j1; jb += 32) {
        const int j = jb + lane;
        Ranges R;
        R.a0 = R.a1 = 0;
        int n0 = 0, n1 = 0;
        if (j <= j1 && rng(j, R)) {
            n0 = R.b0 >= R.a0 ? R.b0 - R.a0 + 1 : 0;
            n1 = R.b1 >= R.a1 ? R.b1 - R.a1 + 1 : 0;
        }
        int inc = n0 + n1;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int v = __shfl_up_sync(FULL, inc, o);
            if (lane >= o) inc += v;
        }
        const int total = __shfl_sync(FULL, inc, 31);
        const int excl = inc - (n0 + n1);
        for (int e0 = 0; e0 < total; e0 += 32 * NB) {
            bool ok[NB];
#pragma unroll
            for (int u = 0; u < NB; u++) {
                const int e = e0 + u * 32 + lane;
                // lane q holding item e: the last lane whose prefix is <= e
                int q = 0;
#pragma unroll
                for (int step = 16; step > 0; step >>= 1) {
                    const int c = q + step;
                    const int ex = __shfl_sync(FULL, excl, c & 31);
                    if (c < 32 && ex <= e) q = c;
                }
                const int qa0 = __shfl_sync(FULL, R.a0, q), qa1 = __shfl_sync(FULL, R.a1, q);
                const int qn0 = __shfl_sync(FULL, n0, q), qex = __shfl_sync(FULL, excl, q);
                const int tt = e - qex;
                const int i = tt < qn0 ? qa0 + tt : qa1 + (tt - qn0);
                ok[u] = e < total && fetch(i, jb + q, u);
            }
#pragma unroll
            for (int u = 0; u < NB; u++) process(u, ok[u]);
        }
    }
}


// ------------------------------------------------------------- forces

__device__ __forceinline__ double net_weight(const StepParams &p, const DSolid &b) {
    const double M = b.rho_s * PI * b.r * b.r;
    const double g = sqrt(p.grav_x * p.grav_x + p.grav_y * p.grav_y);
    return fabs(1.0 - p.rho0 / b.rho_s) * M * g;
}

__device__ __forceinline__ double lub_mag(double kappa, double zeta, double gap) {
    if (gap >= zeta) return 0.0;
    const double q = (zeta - gap) / zeta;
    return kappa * q * q;
}

// R(t+1) split, reduced into the domain (through the integer part: no FP64
// division) and in FP32.
__device__ __forceinline__ void set_next_centre(const Lattice &L, DSolid &b) {
    split_coord(b.xn, b.ix1, b.fx1);
    split_coord(b.yn, b.iy1, b.fy1);
    b.xnw = L.bc_x == LBM_PERIODIC ? b.xn - (double)(L.nx * floor_div(b.ix1, L.nx)) : b.xn;
    b.ynw = L.bc_y == LBM_PERIODIC ? b.yn - (double)(L.ny * floor_div(b.iy1, L.ny)) : b.yn;
    b.xnf = (float)b.xn;
    b.ynf = (float)b.yn;
}

// Motion t -> t+1 of solid s; fg = force and torque at t (lane 0): Eq. 5,
// or Eq. 4 when the context asks for the conventional form.
// The lubrication sum runs over the lanes of the warp.
__device__ void move_solid(const StepParams &p, int s, int lane, long long t, const double *fg) {
    DSolid &b = p.S[s];
    const Lattice &L = p.L;
    if (b.motion == LBM_PRESCRIBED) {
        if (lane == 0) {
            const double dt = (double)(t + 1 - b.ta);
            b.xn = __dadd_rn(b.xa, __dmul_rn(b.vx, dt));
            b.yn = __dadd_rn(b.ya, __dmul_rn(b.vy, dt));
            set_next_centre(L, b);
            b.vxn = b.vx;
            b.vyn = b.vy;
            b.omn = b.om;
        }
        return;
    }
    double fl[2] = {0.0, 0.0};
    if (p.lub > 0.0) {
        const double ka = net_weight(p, b);
        const float zf = (float)p.lub + 0.01f * (float)b.r + 1.f;
        for (int q = lane; q < p.nsolid; q += 32) {
            if (q == s) continue;
            const DSolid &B = p.S[q];
            // FP32 first, with a slack far above its rounding: out of range for most
            float ddx = (float)(b.ix0 - B.ix0) + (b.fx0 - B.fx0);
            float ddy = (float)(b.iy0 - B.iy0) + (b.fy0 - B.fy0);
            if (L.bc_x == LBM_PERIODIC) ddx -= (float)L.nx * rintf(ddx / (float)L.nx);
            if (L.bc_y == LBM_PERIODIC) ddy -= (float)L.ny * rintf(ddy / (float)L.ny);
            const float reach = (sqrtf(b.r2f) + sqrtf(B.r2f)) * 1.001f + zf;
            if (ddx * ddx + ddy * ddy > reach * reach) continue;
            const double dx = min_image(b.x - B.x, L.nx, L.bc_x == LBM_PERIODIC);
            const double dy = min_image(b.y - B.y, L.ny, L.bc_y == LBM_PERIODIC);
            const double d = sqrt(dx * dx + dy * dy);
            const double kb = net_weight(p, B);
            const double m = lub_mag(ka > kb ? ka : kb, p.lub, d - b.r - B.r);
            if (m > 0.0 && d > 0.0) {
                fl[0] += m * dx / d;
                fl[1] += m * dy / d;
            }
        }
        warp_sum(fl);
        if (lane == 0) {
            if (L.bc_y == LBM_WALL) {
                fl[1] += lub_mag(ka, p.lub, (b.y - b.r) + 0.5);
                fl[1] -= lub_mag(ka, p.lub, ((double)L.ny - 0.5) - (b.y + b.r));
            }
            if (L.bc_x == LBM_WALL) {
                fl[0] += lub_mag(ka, p.lub, (b.x - b.r) + 0.5);
                fl[0] -= lub_mag(ka, p.lub, ((double)L.nx - 0.5) - (b.x + b.r));
            }
        }
    }
    if (lane != 0) return;
    const double M = b.rho_s * PI * b.r * b.r;
    const double I = 0.5 * M * b.r * b.r;
    const double buoy = 1.0 - p.rho0 / b.rho_s;
    const double Fx = fg[0] + buoy * M * p.grav_x + fl[0];
    const double Fy = fg[1] + buoy * M * p.grav_y + fl[1];
    const double vx1 = b.vx + Fx / M, vy1 = b.vy + Fy / M;
    b.xn = b.x + 0.5 * (b.vx + vx1);
    b.yn = b.y + 0.5 * (b.vy + vy1);
    set_next_centre(L, b);
    b.vxn = vx1;
    b.vyn = vy1;
    b.omn = b.om + fg[2] / I;
}

// Force record of time t of solid s from its link sums acc and the momentum
// booked into t by the node-type changes of the previous step (lane 0: Eq. 4
// force and torque, then Eq. 5); then its motion to t+1.
__device__ void record_forces(const StepParams &p, int s, int lane, long long t,
                              const double (&acc)[6], const double (&booked)[6]) {
    double fg[3] = {0.0, 0.0, 0.0};
    if (lane == 0) {
        const long long slot = t % p.ring_len;
        double *rc = p.ring + (slot * 2 + 0) * p.nsolid * 3 + (long long)s * 3;
        double *rg = p.ring + (slot * 2 + 1) * p.nsolid * 3 + (long long)s * 3;
        for (int q = 0; q < 3; q++) {
            rc[q] = acc[q] + booked[q];
            rg[q] = acc[3 + q] + booked[3 + q];
            fg[q] = p.motion_cme ? rc[q] : rg[q];  // the form that drives a free solid
        }
    }
    move_solid(p, s, lane, t, fg);
}

// ------------------------------------------------- fluid-solid links

// A block of FB threads walks the links of one solid.  Candidates: a node x_f can have a
// link into the disk when r - eps < |x_f - R| <= r + sqrt 2 + eps, between the outer chord
// of each row and the inner one; thread t reads the flags of candidate t, t + FB ...
// FP32 arithmetic, half-way: a candidate's thread takes its links itself (direction i with
// x_f + e_i solid).  FP64, and with the interpolated boundary: it lists them in shared
// memory, in candidate order, and every thread takes links t, t + FB ... of that list, so
// that all lanes work: with a thread per candidate, the lanes of a warp have one to five
// links each in different directions, and the warp goes through the link's arithmetic up
// to eight times, which in FP64 (two lanes per clock and SM) was most of the kernel's
// time.  In FP32 the list costs more than it saves (a step of 768 x 512 nodes with six
// disks of r 51, FP16, the links before the fused kernel: 46.4 us with it, 43.5 without),
// and with its 11 KB of shared memory a block, SMs beside FP16's fused kernel had to
// change their split of L1 and shared memory, which they do only when empty.
// A link reads its own population, its solid's owner only when the near list is
// not empty, and with the interpolated boundary one population more.  Sums: a
// candidate's links in the order of the directions (the list's terms go through shared
// memory to the candidate's thread); then over the tree of its warp's 32, both in the
// arithmetic precision of the storage mode; then in FP64 over the turns of each of four
// warps (one block of 128 threads) and over these four, in order, so that a solid's
// candidates may go to several blocks.  (A force is a small difference of large link
// terms, so another order of the FP32 sums would change it in the fifth digit.)
constexpr int FB = 128;                  // threads per solid (batches: or twice as many)
constexpr int LU = 2;                    // links a thread loads before it works on them
constexpr float ANN_EPS = 0.05f;         // above the FP32 rounding of a chord end

// Do candidates' own threads take their links (above)?
template <int P, bool BND>
__host__ __device__ constexpr bool direct() {
    return P != LBM_FP64 && !BND;
}

template <int P, bool BND, int NT = FB> struct LinkShared {
    using C = typename Prec<P>::C;
    static constexpr int LIST = direct<P, BND>() ? 0 : 1;
    int wsum[NT / 32];
    int cnt[NT];                  // the turn's rows: exclusive prefix of their candidates
    int lo[NT], i0[NT], i1[NT];   // row: [lo, hi] minus the inner chord [i0, i1]
    double part[NT / 32][6];      // the warps' sums
    int4 cand[LIST * NT + 1];     // candidate: {cell, x - floor X, y - floor Y, flags}
    uint16_t link[LIST * 8 * NT + 1];  // direction | candidate << 4
    C rho[LIST * NT + 1];         // local density of the candidates (rho_w local)
    C term[6][LIST * LU * NT + 1];     // the terms of the links in hand
};

// Exclusive prefix of n over the block, and its total (whole blocks call it).
template <int P, bool BND, int NT>
__device__ __forceinline__ int block_scan(int n, LinkShared<P, BND, NT> &sh, int &total) {
    const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
    int inc = n;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int v = __shfl_up_sync(FULL, inc, o);
        if (lane >= o) inc += v;
    }
    __syncthreads();  // wsum's last use, and the tables' the caller rewrites after this
    if (lane == 31) sh.wsum[wib] = inc;
    __syncthreads();
    int before = 0;
    total = 0;
#pragma unroll
    for (int w = 0; w < NT / 32; w++) {
        if (w < wib) before += sh.wsum[w];
        total += sh.wsum[w];
    }
    return before + inc - n;
}

// Terms of a link along e_i whose middle is (dx, dy) from R: Eq. 4 force and torque, then
// Eq. 5, from f_i and the returned f_bb, at the solid's velocity (ux, uy) there.
template <class C>
__device__ __forceinline__ void link_terms(C ex, C ey, C dx, C dy, C ux, C uy, C fi, C fbb, C (&v)[6]) {
    const C cmx = ex * fi + ex * fbb, cmy = ey * fi + ey * fbb;
    const C gmx = (ex - ux) * fi - (-ex - ux) * fbb;
    const C gmy = (ey - uy) * fi - (-ey - uy) * fbb;
    v[0] = cmx;
    v[1] = cmy;
    v[2] = dx * cmy - dy * cmx;
    v[3] = gmx;
    v[4] = gmy;
    v[5] = dx * gmy - dy * gmx;
}

// The links of solid s: their sums added to acc (its warp's: component sum_of(l) of the
// Eq. 4 force and torque, then of Eq. 5, in lane l), and with GHOST the returned
// populations into the solid nodes' slots of fs.
// The solid's candidates are taken chunk by chunk of `chunk` <= NT; this block takes the chunks part, part + nparts ...  With
// slots (chunks of a warp) each chunk's sums are left there instead, six to a slot, with
// slots of zeros after the chunks of each turn of rows up to a multiple of LINK_PARTS and
// to LEAD_SLOTS, and their number in the last slot.
//   per link  f_i = f~_i(x_f), the returned f_bb = f_i - 6 w_i rho_w (e_i . v) with
//   v the solid's velocity at x_s = x_f + e_i / 2 (BND: interpolated from the cut
//   of the link, v and the lever there); Eq. 4 = e_i f_i - e_opp f_bb, Eq. 5 =
//   (e_i - v) f_i - (e_opp - v) f_bb, torque (x_s - R) x F (Eq. 7).
template <int P, bool LOCAL, bool BND, bool GHOST, bool WIDE, int NT>
__device__ __forceinline__ void solid_links(const StepParams &p, const DSolid &b, int s,
                                            typename Prec<P>::S *fs, bool owners, bool list,
                                            long long t, int chunk, int part, int nparts,
                                            LinkShared<P, BND, NT> &sh, double &acc,
                                            double *slots = nullptr) {
    using C = typename Prec<P>::C;
    using S = typename Prec<P>::S;
    const int tid = threadIdx.x, lane = tid & 31;
    const Lattice &L = p.L;
    const int plane = (int)L.plane;
    const Centre c(b.ix0, b.iy0, b.fx0, b.fy0);
    const Wrap wrap(L, b.ix0, b.iy0, b.rc);
    const float r = sqrtf(b.r2f);
    const C vx = pick<C>(b.vx, b.vxf), vy = pick<C>(b.vy, b.vyf), om = pick<C>(b.om, b.omf);
    const C rho0 = pick<C>(p.rho0, p.rho0_f);
    int j0, j1, nslot = 0;
    rows_of_i(b.iy0, b.iy0, b.rc, 3, j0, j1);
    for (int jc = j0; jc <= j1; jc += FB) {  // rows in turns of FB
        // candidates of row jc + tid
        int lo = 1, hi = 0, i0 = 1, i1 = 0, n = 0;
        const int j = jc + tid;
        if (tid < FB && j <= j1 && c.chord(j, r + 1.4143f + ANN_EPS, lo, hi) && lo <= hi) {
            n = hi - lo + 1;
            if (c.chord(j, r - ANN_EPS, i0, i1) && i0 <= i1) n -= i1 - i0 + 1;
        }
        int total;
        const int excl = block_scan(n, sh, total);
        sh.cnt[tid] = excl;
        sh.lo[tid] = lo;
        sh.i0[tid] = i0 <= i1 ? i0 : 1;  // an empty inner chord: i0 > i1
        sh.i1[tid] = i0 <= i1 ? i1 : 0;
        __syncthreads();
        for (int base = part * chunk; base < total; base += nparts * chunk) {
            // candidate e -> row (binary search over the prefix) and column
            const int e = base + tid;
            int q = 0;
#pragma unroll
            for (int step = NT / 2; step > 0; step >>= 1)
                if (q + step < NT && sh.cnt[q + step] <= e) q += step;
            const int jj = jc + q;
            int iu = sh.lo[q] + (e - sh.cnt[q]);
            const int a = sh.i0[q], bb = sh.i1[q];
            if (a <= bb && iu >= a) iu += bb - a + 1;  // step over the inner chord
            int x = 0, y = 0;
            const bool here = tid < chunk && e < total && wrap(iu, jj, x, y);
            const int k = here ? (int)cell_of(L, x, y) : 0;
            const unsigned m = here ? p.flags[k] : 1u;
            const bool bounced_node = !(m & 1u) && (m & 0x1FEu);
            if (!GHOST && list) {
                // FP16: the node goes to the deferred per-node path's list of step t
                const unsigned want = __ballot_sync(FULL, bounced_node);
                if (want) {
                    int at = 0;
                    if (lane == 0) at = atomicAdd(p.bnd + (t & 1), __popc(want));
                    at = __shfl_sync(FULL, at, 0) + __popc(want & ((1u << lane) - 1u));
                    if (bounced_node) {
                        if (at < p.bnd_cap) p.bnd[2 + at] = k;
                        else atomicOr(p.status, 16);
                    }
                }
            }
            // bit i: x_f + e_i is solid or beyond a wall (bit opp(i) of the flags)
            unsigned dirs = bounced_node ? ((m & 0x66u) << 2 | (m >> 2 & 0x66u)) : 0u;
            C sum[6] = {0, 0, 0, 0, 0, 0};  // of this candidate's links
            const bool any = dirs != 0;
            if constexpr (direct<P, BND>()) {
                S fv[9];
                int kb[9];
                uint16_t own[9];
#pragma unroll
                for (int i = 1; i < 9; i++) {
                    kb[i] = -1;
                    int xb, yb;
                    if (!(dirs >> i & 1u) || !wrap(iu + cx(i), jj + cy(i), xb, yb)) continue;
                    kb[i] = (int)cell_of(L, xb, yb);  // else beyond a wall
                    fv[i] = fs[i * plane + k];
                    if (owners) own[i] = p.owner[kb[i]];
                }
                C rho_w = rho0;
                if (LOCAL && any) {
                    C a9 = 0;
#pragma unroll
                    for (int q9 = 0; q9 < 9; q9++) a9 += (C)cvt_s(fs[q9 * plane + k]);
                    rho_w = (C)1 + a9;
                }
                const C px = (C)(iu - c.xi), py = (C)(jj - c.yi);
#pragma unroll
                for (int i = 1; i < 9; i++) {
                    if (kb[i] < 0 || (owners && own[i] != (uint16_t)s)) continue;
                    const C ex = (C)cx(i), ey = (C)cy(i), w = wgt<C>(i);
                    const C back = (C)cvt_s(fv[i]), fi = back + w;
                    const C dx = px + (C)0.5 * ex - (C)c.fx, dy = py + (C)0.5 * ey - (C)c.fy;
                    const C ux = vx - om * dy, uy = vy + om * dx;
                    const C a6 = (C)6 * w * rho_w, eu = ex * ux + ey * uy;
                    C v[6];
                    if (GHOST) st(fs + opp(i) * plane + kb[i], fma(-a6, eu, back));
                    link_terms(ex, ey, dx, dy, ux, uy, fi, fma(-a6, eu, fi), v);
#pragma unroll
                    for (int q6 = 0; q6 < 6; q6++) sum[q6] += v[q6];
                }
            } else {
                int nlink;
                const int mine0 = block_scan(__popc(dirs), sh, nlink), mine1 = mine0 + __popc(dirs);
                if (LOCAL) {
                    C a9 = 0;
                    if (dirs) {
                        S fv[9];
#pragma unroll
                        for (int q9 = 0; q9 < 9; q9++) fv[q9] = fs[q9 * plane + k];
#pragma unroll
                        for (int q9 = 0; q9 < 9; q9++) a9 += (C)cvt_s(fv[q9]);
                    }
                    sh.rho[tid] = Prec<P>::dev ? (C)1 + a9 : a9;
                }
                sh.cand[tid] = make_int4(k, iu - c.xi, jj - c.yi, (int)m);
                for (int at = mine0; dirs; dirs &= dirs - 1)
                    sh.link[at++] = (uint16_t)((__ffs(dirs) - 1) | tid << 4);
                __syncthreads();
                for (int l0 = 0; l0 < nlink; l0 += LU * NT) {
                    int4 cd[LU];
                    int kb[LU], dir[LU];
                    S fi_s[LU], fo_s[LU], fn_s[LU];
                    C rho_w[LU];
                    uint16_t own[LU];
                    bool inner[LU];  // BND: x_f - e_i is a fluid node of the domain
#pragma unroll
                    for (int u = 0; u < LU; u++) {
                        kb[u] = -1;
                        const int l = l0 + u * NT + tid;
                        if (l >= nlink) continue;
                        const int lk = sh.link[l], i = lk & 15;
                        const int4 cc = cd[u] = sh.cand[lk >> 4];
                        dir[u] = i;
                        rho_w[u] = LOCAL ? sh.rho[lk >> 4] : rho0;
                        int xb, yb;
                        if (!wrap(c.xi + cc.y + cx(i), c.yi + cc.z + cy(i), xb, yb)) continue;
                        kb[u] = (int)cell_of(L, xb, yb);  // else beyond a wall
                        fi_s[u] = fs[i * plane + cc.x];
                        if (owners) own[u] = p.owner[kb[u]];
                        if (BND) {
                            inner[u] = !((cc.w >> i) & 1);
                            fo_s[u] = fs[opp(i) * plane + cc.x];
                            fn_s[u] = fi_s[u];
                            int xn, yn;
                            if (inner[u] && wrap(c.xi + cc.y - cx(i), c.yi + cc.z - cy(i), xn, yn))
                                fn_s[u] = fs[i * plane + (int)cell_of(L, xn, yn)];
                        }
                    }
#pragma unroll
                    for (int u = 0; u < LU; u++) {
                        C v[6] = {0, 0, 0, 0, 0, 0};
                        if (kb[u] >= 0 && !(owners && own[u] != (uint16_t)s)) {
                            const int i = dir[u], di = cd[u].y, dj = cd[u].z;
                            const C ex = (C)cx(i), ey = (C)cy(i), w = wgt<C>(i);
                            const C back = (C)cvt_s(fi_s[u]);  // as stored
                            const C fi = Prec<P>::dev ? back + w : back;
                            C dx, dy, ux, uy, fbb, ret = 0;  // ret: f_bb as stored
                            if (BND) {
                                C q;  // the link is cut at this fraction
                                if (Prec<P>::dev) {
                                    q = (C)link_fraction_split(di, dj, c.fx, c.fy, b.r, cx(i), cy(i));
                                    dx = ((C)di - (C)c.fx) + q * ex;
                                    dy = ((C)dj - (C)c.fy) + q * ey;
                                } else {
                                    // the unwrapped node is at the centre's nearest image
                                    const double px = (double)(c.xi + di) - b.x;
                                    const double py = (double)(c.yi + dj) - b.y;
                                    q = (C)link_fraction_at(px, py, b.r, cx(i), cy(i));
                                    dx = (C)px + q * ex;
                                    dy = (C)py + q * ey;
                                }
                                ux = vx - om * dy;
                                uy = vy + om * dx;
                                const C mw = -(C)6 * w * rho_w[u] * (ex * ux + ey * uy);
                                const C q2 = (C)2 * q;
                                const C fo = (C)cvt_s(fo_s[u]), fn = (C)cvt_s(fn_s[u]);
                                auto returned = [&](C f, C o, C nb) {
                                    if (q2 >= (C)1) return (f + mw) / q2 + ((q2 - (C)1) / q2) * o;
                                    if (inner[u]) return q2 * f + ((C)1 - q2) * nb + mw;
                                    return f + mw;
                                };
                                // full populations for the force; as stored for the pull
                                // (the interpolation's weights sum to one)
                                if (Prec<P>::dev) fbb = returned(fi, fo + w, fn + w);
                                if (GHOST || !Prec<P>::dev) ret = returned(back, fo, fn);
                                if (!Prec<P>::dev) fbb = ret;
                            } else {
                                // x_s = x_f + e_i / 2 relative to R, from the unwrapped coordinate
                                if (Prec<P>::dev) {
                                    dx = (C)di + (C)0.5 * ex - (C)c.fx;
                                    dy = (C)dj + (C)0.5 * ey - (C)c.fy;
                                } else {
                                    dx = (C)(((double)(c.xi + di) + 0.5 * (double)ex) - b.x);
                                    dy = (C)(((double)(c.yi + dj) + 0.5 * (double)ey) - b.y);
                                }
                                ux = vx - om * dy;
                                uy = vy + om * dx;
                                const C a6 = (C)6 * w * rho_w[u], eu = ex * ux + ey * uy;
                                fbb = fma(-a6, eu, fi);
                                ret = fma(-a6, eu, back);
                            }
                            if (GHOST) st(fs + opp(i) * plane + kb[u], ret);
                            link_terms(ex, ey, dx, dy, ux, uy, fi, fbb, v);
                        }
#pragma unroll
                        for (int q6 = 0; q6 < 6; q6++) sh.term[q6][u * NT + tid] = v[q6];
                    }
                    __syncthreads();
                    // the candidate's thread adds its links' terms
                    for (int l = max(mine0, l0); l < min(mine1, l0 + LU * NT); l++)
#pragma unroll
                        for (int q6 = 0; q6 < 6; q6++) sum[q6] += sh.term[q6][l - l0];
                    __syncthreads();  // the terms (and the list) are reused
                }
            }
            const int e32 = base + (tid & ~31);  // this warp's first candidate
            if ((tid & ~31) < chunk && e32 < total) {
                double v = 0.0;
                if (__any_sync(FULL, any)) v = chunk_sum<WIDE>(sum, lane);
                if (!slots) acc += v;
                else if (sum_of(lane) < 6 && nslot + e32 / 32 < p.link_slots - 1)
                    slots[(nslot + e32 / 32) * 6 + sum_of(lane)] = v;
            }
        }
        if (slots) {
            int k = (total + 31) / 32;
            for (; k % LINK_PARTS || nslot + k < LEAD_SLOTS; k++)
                if (k % nparts == part && tid < 6 && nslot + k < p.link_slots - 1) slots[(nslot + k) * 6 + tid] = 0.0;
            nslot += k;
            if (part == 0 && tid == 0) slots[(p.link_slots - 1) * 6] = (double)nslot;
        }
    }
}

// Sums over the block's warps (whose sums solid_links has left in w), in order, to all
// lanes of warp 0: warps LINK_PARTS apart first, as one that takes their chunks in turn.
template <int P, bool BND, int NT>
__device__ __forceinline__ void block_sums(LinkShared<P, BND, NT> &sh, double w, double (&acc)[6]) {
    const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
    if (sum_of(lane) < 6) sh.part[wib][sum_of(lane)] = w;
    __syncthreads();
    if (wib != 0) return;
    double aq = 0.0;
    if (lane < 6)
#pragma unroll
        for (int c = 0; c < LINK_PARTS; c++) {
            double a = sh.part[c][lane];
#pragma unroll
            for (int k = c + LINK_PARTS; k < NT / 32; k += LINK_PARTS) a += sh.part[k][lane];
            aq += a;
        }
#pragma unroll
    for (int q = 0; q < 6; q++) acc[q] = __shfl_sync(FULL, aq, q);
}

// The momenta booked into the record of t by the node-type changes of the step
// before: component q of the solid's event segment, in order, in lane q < 6.
__device__ __forceinline__ void booked_events(const StepParams &p, const DSolid &b, long long t,
                                              int lane, double (&booked)[6]) {
    double bq = 0.0;
    if (lane < 6 && b.ev_t == t)
        for (int e0 = 0; e0 < b.ev_n; e0 += 8) {  // eight loads in flight, added in order
            double v[8];
#pragma unroll
            for (int k = 0; k < 8; k++)
                v[k] = e0 + k < b.ev_n ? p.ev_mom[6 * (b.ev_off + e0 + k) + lane] : 0.0;
#pragma unroll
            for (int k = 0; k < 8; k++)
                if (e0 + k < b.ev_n) bq += v[k];
        }
#pragma unroll
    for (int q = 0; q < 6; q++) booked[q] = __shfl_sync(FULL, bq, q);
}

// Distance of the solid's centre at t and t+1 from that at the last pair test
// (FP32 from the split centres, with a slack above its rounding).
__device__ __forceinline__ float displacement(const DSolid &b) {
    const float d0 = hypotf((float)(b.ix0 - b.ixt) + (b.fx0 - b.fxt),
                            (float)(b.iy0 - b.iyt) + (b.fy0 - b.fyt));
    const float d1 = hypotf((float)(b.ix1 - b.ixt) + (b.fx1 - b.fxt),
                            (float)(b.iy1 - b.iyt) + (b.fy1 - b.fyt));
    return fmaxf(d0, d1) + 1e-3f;
}

// FP64 sums over a warp's lanes: in FP64, and in batches.  (In FP32 they would cost the
// force kernel of 2000 disks tens of microseconds: GB300 issues FP64 for about two lanes
// per clock and SM.)
template <int P>
__host__ __device__ constexpr bool wide() {
    return P == LBM_FP64;
}

// FP16 rounds a returned population: it stays in registers there (sc_tile).
template <int P>
__host__ __device__ constexpr bool ghosts() {
    return P != LBM_FP16_DEV;
}

// The near lists hold at t unless a solid was added or changed since the last
// pair test; without them (or with solids in reach) a link's owner is read.
__device__ __forceinline__ bool need_owners(const StepParams &p, const DSolid &b) {
    const bool lists_ok = p.near_id && ((volatile unsigned int *)p.bar)[3] == 0u;
    return !lists_ok || b.near_n != 0;
}

// The half-way boundary: links, record and motion of one solid per block.
template <int P, bool LOCAL, int NT>
__global__ void __launch_bounds__(NT, 896 / NT) k_forces(const StepParams p) {
    early_start();
    using S = typename Prec<P>::S;
    __shared__ LinkShared<P, false, NT> sh;
    const int tid = threadIdx.x, lane = tid & 31;
    const long long t = *p.t;
    S *fs = static_cast<S *>((t & 1) ? p.f1 : p.f0);  // populations of time t
    // the previous step's events are reached through the solids' segments;
    // the list fills again in this step's re-rasterisation
    if (blockIdx.x == 0 && tid == 0 && p.ev_len) {
        *p.ev_len = 0;
        *p.chg_len = 0;
    }
    float disp = 0.f;
    for (int s = blockIdx.x; s < p.nsolid; s += gridDim.x) {
        DSolid &b = p.S[s];
        if (!solid_ok(b)) {
            if (tid == 0) atomicOr(p.status, 2);
            continue;
        }
        double sum = 0.0, acc[6];
        solid_links<P, LOCAL, false, ghosts<P>(), wide<P>()>(p, b, s, fs, need_owners(p, b), p.list_by_forces, t,
                                                             NT, 0, 1, sh, sum);
        block_sums(sh, sum, acc);
        if (tid < 32) {
            double booked[6];
            booked_events(p, b, t, lane, booked);
            record_forces(p, s, lane, t, acc, booked);
            if (lane == 0) disp = fmaxf(disp, displacement(b));
        }
        __syncthreads();  // sh.part is reused
    }
    if (tid == 0 && disp > 0.f)  // non-negative: bits order as values
        atomicMax(p.bar + 2, __float_as_uint(disp));
}

// The same in two kernels: k_links, after which the advection-collision kernel can
// run, and k_record (records and motion), beside it, or after it as the step's last.  A solid's links go to
// gridDim.y blocks: one, or several that take its candidates 32 at a time in turn:
// LINK_PARTS, each the share of one warp of the single block, or more, which leave every
// turn's sums to k_record.  The sums are the same bit for bit, whichever way.  (With the interpolated boundary one 30-node disk in FP64 took
// 68 us in one block with a thread per candidate: one SM's FP64 unit.)
constexpr int LINK_CHUNK = FB / LINK_PARTS;

// BLOCKS: registers for so many blocks on an SM, at the cost of a few bytes of spills.
template <int P, bool LOCAL, bool BND, int BLOCKS>
__global__ void __launch_bounds__(FB, BLOCKS) k_links(const StepParams p) {
    early_start();
    using S = typename Prec<P>::S;
    __shared__ LinkShared<P, BND> sh;
    const long long t = *p.t;
    S *fs = static_cast<S *>((t & 1) ? p.f1 : p.f0);
    for (int s = blockIdx.x; s < p.nsolid; s += gridDim.x) {
        const DSolid &b = p.S[s];
        if (!solid_ok(b)) continue;  // k_record reports it
        double *slots = p.link_slots ? p.part + (long long)s * p.link_slots * 6 : nullptr;
        double sum = 0.0, acc[6];
        solid_links<P, LOCAL, BND, ghosts<P>(), wide<P>()>(p, b, s, fs, need_owners(p, b), p.list_by_forces, t,
                                                           gridDim.y > 1 ? LINK_CHUNK : FB, blockIdx.y, gridDim.y,
                                                           sh, sum, slots);
        if (slots) continue;
        block_sums(sh, sum, acc);
        if (threadIdx.x == 0)
            for (int q = 0; q < 6; q++) p.part[((long long)s * LINK_PARTS + blockIdx.y) * 6 + q] = acc[q];
        __syncthreads();  // sh.part is reused
    }
}

// Record and motion of solid s, by one warp.
__device__ __forceinline__ void record_solid(const StepParams &p, int s, int lane, long long t) {
    DSolid &b = p.S[s];
    if (!solid_ok(b)) {
        if (lane == 0) atomicOr(p.status, 2);
        return;
    }
    double aq = 0.0, acc[6], booked[6];
    if (p.link_slots) {  // as the warps of one block would have added them
        const double *part = p.part + (long long)s * p.link_slots * 6 + lane;
        if (lane < 6) {
            double a[LINK_PARTS] = {0.0, 0.0, 0.0, 0.0};
#pragma unroll
            for (int c = 0; c < LEAD_SLOTS; c++) a[c % LINK_PARTS] += part[c * 6];
            const int n = min((int)part[(p.link_slots - 1) * 6 - lane], p.link_slots - LINK_PARTS);
            for (int c = LEAD_SLOTS; c < n; c += LINK_PARTS)
#pragma unroll
                for (int w = 0; w < LINK_PARTS; w++) a[w] += part[(c + w) * 6];
            aq = ((a[0] + a[1]) + a[2]) + a[3];
        }
    } else if (lane < 6) {
        for (int c = 0; c < p.link_parts; c++) aq += p.part[((long long)s * LINK_PARTS + c) * 6 + lane];
    }
#pragma unroll
    for (int q = 0; q < 6; q++) acc[q] = __shfl_sync(FULL, aq, q);
    booked_events(p, b, t, lane, booked);
    record_forces(p, s, lane, t, acc, booked);
    if (lane == 0) atomicMax(p.bar + 2, __float_as_uint(displacement(b)));
}

__global__ void __launch_bounds__(SW_BLOCK) k_record(const StepParams p) {
    early_start();
    const int lane = threadIdx.x & 31;
    const long long t = *p.t;
    if (blockIdx.x == 0 && threadIdx.x == 0 && p.ev_len) {
        *p.ev_len = 0;
        *p.chg_len = 0;
    }
    const int s = blockIdx.x * WARPS + (threadIdx.x >> 5);
    if (s < p.nsolid) record_solid(p, s, lane, t);
    if (p.record_last) end_of_step(p, t, gridDim.x);
}

// ----------------------------------------------------- re-rasterisation

// Pair test: the near list of the moving solid moving[base + warp index]
// (whole blocks call it; base + warp index may be >= nmoving).  The centres
// at t and t+1 of every solid are staged in shared memory one tile at a time.
// FP32 distances with a slack far above their rounding.
constexpr int NEAR_TILE = 512;
__device__ void phase_pairs_block(const StepParams &p, int base, int4 *ipos, float4 *fpos,
                                  float *rad) {
    const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
    const int m = base + wib;
    const bool mine = m < p.nmoving;
    const int s = mine ? p.moving[m] : -1;
    const Lattice &L = p.L;
    const bool px = L.bc_x == LBM_PERIODIC, py = L.bc_y == LBM_PERIODIC;
    const float nxf = (float)L.nx, nyf = (float)L.ny;
    int4 bi = make_int4(0, 0, 0, 0);
    float4 bf = make_float4(0.f, 0.f, 0.f, 0.f);
    float rb = 0.f;
    if (mine) {
        const DSolid &b = p.S[s];
        rb = sqrtf(b.r2f);
        bi = make_int4(b.ix0, b.iy0, b.ix1, b.iy1);
        bf = make_float4(b.fx0, b.fy0, b.fx1, b.fy1);
    }
    uint16_t *out = mine ? p.near_id + (long long)s * NEAR_CAP : nullptr;
    int cnt = 0;
    for (int t0 = 0; t0 < p.nsolid; t0 += NEAR_TILE) {
        const int n = min(NEAR_TILE, p.nsolid - t0);
        __syncthreads();
        for (int q = threadIdx.x; q < n; q += blockDim.x) {
            const DSolid &B = p.S[t0 + q];
            ipos[q] = make_int4(B.ix0, B.iy0, B.ix1, B.iy1);
            fpos[q] = make_float4(B.fx0, B.fy0, B.fx1, B.fy1);
            rad[q] = sqrtf(B.r2f);
        }
        __syncthreads();
        if (!mine) continue;
        for (int q0 = 0; q0 < n; q0 += 32) {
            const int q = q0 + lane;
            bool hit = false;
            if (q < n && t0 + q != s) {
                const int4 ci = ipos[q];
                const float4 cf = fpos[q];
                const float lim = rb + rad[q] + NEAR_REACH + NEAR_MARGIN + 0.05f;
                float dx = (float)(bi.x - ci.x) + (bf.x - cf.x);
                float dy = (float)(bi.y - ci.y) + (bf.y - cf.y);
                float ex = (float)(bi.z - ci.z) + (bf.z - cf.z);
                float ey = (float)(bi.w - ci.w) + (bf.w - cf.w);
                if (px) {
                    dx -= nxf * rintf(dx / nxf);
                    ex -= nxf * rintf(ex / nxf);
                }
                if (py) {
                    dy -= nyf * rintf(dy / nyf);
                    ey -= nyf * rintf(ey / nyf);
                }
                hit = dx * dx + dy * dy < lim * lim || ex * ex + ey * ey < lim * lim;
            }
            const unsigned h = __ballot_sync(FULL, hit);
            if (hit) {
                const int at = cnt + __popc(h & ((1u << lane) - 1u));
                if (at < NEAR_CAP) out[at] = (uint16_t)(t0 + q);
            }
            cnt += __popc(h);
        }
    }
    if (mine && lane == 0) p.S[s].near_n = cnt <= NEAR_CAP ? cnt : -1;
}

// Is the domain node (x, y) inside the disk (X, Y, r)?  Decided at the
// node's periodic image nearest to the centre, by the exact test, as the
// rasterisation of the disk decides it.
__device__ __forceinline__ bool inside_at(const Lattice &L, int x, int y, double X, double Y,
                                          double r) {
    // the image shift in FP32: it only has to be right for nodes within r + 1
    // of the centre, far from the half-period where it could round either way
    int i = x, j = y;
    if (L.bc_x == LBM_PERIODIC) i += L.nx * (int)rintf((float)(X - (double)x) / (float)L.nx);
    if (L.bc_y == LBM_PERIODIC) j += L.ny * (int)rintf((float)(Y - (double)y) / (float)L.ny);
    const float dx = (float)((double)i - X), dy = (float)((double)j - Y), rr = (float)r + 1.0f;
    if (dx * dx + dy * dy > rr * rr) return false;
    return inside_disk(i, j, X, Y, r);
}

// Lowest-id owners of the domain node (x, y) at t (was) and t+1 (now), given
// those of solid s alone: the solids of s's near list (every solid when the
// list overflowed) that hold the node.  Centres at t: x, y (phase R only).
__device__ void near_owners(const StepParams &p, const DSolid &b, int s, int x, int y,
                            uint16_t &was, uint16_t &now) {
    const int nn = b.near_n;
    if (nn == 0) return;
    const uint16_t *nl = p.near_id + (long long)s * NEAR_CAP;
    const int n = nn < 0 ? p.nsolid : nn;
    for (int k = 0; k < n; k++) {
        const int q = nn < 0 ? k : (int)nl[k];
        if (q == s || (q >= (int)was && q >= (int)now)) continue;
        const DSolid &B = p.S[q];
        if (q < (int)was && inside_at(p.L, x, y, B.x, B.y, B.r)) was = (uint16_t)q;
        if (q < (int)now && inside_at(p.L, x, y, B.xn, B.yn, B.r)) now = (uint16_t)q;
    }
}

// Was the domain node (x, y) inside a solid of s's near list at t?  Only
// those (and s itself, tested by the caller) can have held a node within
// NEAR_REACH of s's surface.  Centres at t: xo, yo (phase E).
__device__ bool near_at_t(const StepParams &p, const DSolid &b, int s, int x, int y) {
    const int nn = b.near_n;
    if (nn == 0) return false;
    const uint16_t *nl = p.near_id + (long long)s * NEAR_CAP;
    const int n = nn < 0 ? p.nsolid : nn;
    for (int k = 0; k < n; k++) {
        const int q = nn < 0 ? k : (int)nl[k];
        if (q == s) continue;
        const DSolid &B = p.S[q];
        if (inside_at(p.L, x, y, B.xo, B.yo, B.r)) return true;
    }
    return false;
}

constexpr int EVENTS = SOLID_EVENTS;

// Ring of solid s (phase R): every node whose owner changes, into the
// step's change list, and the covered and fresh nodes of s, queued per warp
// in lane order and published as the solid's segment of the step's event
// list (to be booked into the force record of t+1), each with its unwrapped
// coordinates in the solid's frame.  No memory is read per node: the owners
// come from the geometry.
__device__ void phase_ring(const StepParams &p, int s, int lane, long long t, int2 *queue,
                           int &qn) {
    DSolid &b = p.S[s];
    const Lattice &L = p.L;
    const DiskTest in0(b.x, b.y, b.r, b.ix0, b.iy0, b.fx0, b.fy0, b.r2f, b.rmf);
    const DiskTest in1(b.xn, b.yn, b.r, b.ix1, b.iy1, b.fx1, b.fy1, b.r2f, b.rmf);
    const Centre c0(b.ix0, b.iy0, b.fx0, b.fy0), c1(b.ix1, b.iy1, b.fx1, b.fy1);
    const Wrap wrap(L, b.ix0, b.iy0, b.rc);
    const float rf = sqrtf(b.r2f);
    int j0, j1;
    rows_of_i(b.iy0, b.iy1, b.rc, 1, j0, j1);
    if (lane == 0) qn = 0;
    __syncwarp();
    constexpr int UR = 2;  // nothing is loaded per node: a short batch suffices
    int kk[UR], iu[UR], ju[UR];
    bool w0[UR];  // on the ring the node is inside s at t (true) or at t+1 (false)
    warp_nodes_n<UR>(
        j0, j1, lane, [&](int j, Ranges &R) { return ring_ranges(c0, c1, rf, j, R); },
        [&](int i, int j, int u) {
            const bool a = in0(i, j);
            if (a == in1(i, j)) return false;
            int x, y;
            if (!wrap(i, j, x, y)) return false;
            kk[u] = (int)cell_of(L, x, y);
            iu[u] = i;
            ju[u] = j;
            w0[u] = a;
            return true;
        },
        [&](int u, bool ok) {
            bool covered = false, fresh = false, changed = false;
            int2 chg;
            const int k = kk[u];
            if (ok) {
                uint16_t was = w0[u] ? (uint16_t)s : FLUID, now = w0[u] ? FLUID : (uint16_t)s;
                const int x = k % L.pitch, y = k / L.pitch;
                near_owners(p, b, s, x, y, was, now);
                if (was != now) {
                    // the new owner; bit 16: the node's solidity flips, bit 17: to solid
                    const bool sn = now != FLUID;
                    chg = make_int2(k, (int)now | (sn != (was != FLUID) ? (sn ? 0x30000 : 0x10000)
                                                                         : 0));
                    changed = true;
                }
                covered = was == FLUID && now == (uint16_t)s;
                fresh = was == (uint16_t)s && now == FLUID;
            }
            // the change list, one atomic per warp
            const unsigned cm = __ballot_sync(FULL, changed);
            if (cm) {
                int cb = 0;
                if (lane == 0) cb = atomicAdd(p.chg_len, __popc(cm));
                cb = __shfl_sync(FULL, cb, 0);
                if (changed) {
                    const int at = cb + __popc(cm & ((1u << lane) - 1u));
                    if (at < p.chg_cap) p.chg[at] = chg;
                    else atomicOr(p.status, 8);
                }
            }
            // queue the covered and fresh nodes in lane order
            __syncwarp();
            const unsigned want = __ballot_sync(FULL, covered || fresh);
            if (!want) return;
            const int base = qn;
            __syncwarp();
            if (lane == 0) qn = base + __popc(want);
            if (covered || fresh) {
                const int pos = base + __popc(want & ((1u << lane) - 1u));
                // node code, and its unwrapped coordinates relative to floor(R)
                if (pos < EVENTS)
                    queue[pos] = make_int2(
                        (k << 1) | (fresh ? 1 : 0),
                        (int)((unsigned)(iu[u] - c0.xi + 32768) |
                              ((unsigned)(ju[u] - c0.yi + 32768) << 16)));
                else atomicOr(p.status, 8);
            }
            __syncwarp();
        });
    __syncwarp();
    const int n = min(qn, EVENTS);
    // publish the events: one segment of the step's event list per solid
    int off = 0;
    if (lane == 0 && n) off = atomicAdd(p.ev_len, n);
    off = __shfl_sync(FULL, off, 0);
    const bool fits = off + n <= p.ev_cap;
    for (int e = lane; e < n; e += 32) {
        if (fits) {
            const int2 q = queue[e];
            const unsigned d = (unsigned)q.y;
            p.ev[off + e] = make_int4(q.x, s, c0.xi + (int)(d & 0xFFFFu) - 32768,
                                      c0.yi + (int)(d >> 16) - 32768);
        }
    }
    if (lane == 0) {
        if (!fits) atomicOr(p.status, 8);
        b.ev_off = off;
        b.ev_n = fits ? n : 0;
        b.ev_t = t + 1;
        b.xo = b.x;
        b.yo = b.y;
        b.ixo = b.ix0;
        b.iyo = b.iy0;
        b.fxo = b.fx0;
        b.fyo = b.fy0;
    }
    __syncwarp();
}

// One covered or fresh node of the step's event list, with the whole warp
// (phase E): the refill of a fresh node (Sec. IV.B), then the node's momentum
// (covered: post-collision, into the solid; fresh: refilled, out of it) and
// its torque about the solid's new centre, into the event's slot of ev_mom.
// Events are independent: a refill reads only nodes that are fluid at t and
// at t+1, which no event writes.
template <int P>
__device__ void phase_event(const StepParams &p, int e, int lane, void *fnew) {
    using C = typename Prec<P>::C;
    using S = typename Prec<P>::S;
    const Lattice &L = p.L;
    const S *fsn = static_cast<const S *>(fnew);
    const int pl = (int)L.plane;
    const int4 ev = p.ev[e];
    const int code = ev.x, s = ev.y;
    const DSolid &b = p.S[s];
    double acc[6] = {0.0, 0.0, 0.0, 0.0, 0.0, 0.0};
    {
        const int k = code >> 1;
        const int x = k % L.pitch, y = k / L.pitch;
        C fj = 0;  // lane j < 9: population j of the node (a fresh node's as stored)
        if (code & 1) {
            // fresh: refill (Sec. IV.B).  Lane 3(i-1)+(d-1) tests x + d e_i: a
            // node fluid at t+1 (owner map) that no solid held at t (the
            // solid's own disk at t in its frame, and its near list)
            bool use = false;
            if (lane < 24) {
                const int i = lane / 3 + 1, d = lane % 3 + 1;
                const int kp = neighbour(L, x, y, d * cx(i), d * cy(i));
                if (kp >= 0 && p.owner[kp] == FLUID) {
                    const DiskTest old(b.xo, b.yo, b.r, b.ixo, b.iyo, b.fxo, b.fyo, b.r2f,
                                       b.rmf);
                    use = !old(ev.z + d * cx(i), ev.w + d * cy(i)) &&
                          !near_at_t(p, b, s, kp % L.pitch, kp / L.pitch);
                }
            }
            const unsigned um = __ballot_sync(FULL, use);
            unsigned d3 = 0, d2 = 0, d1 = 0;  // directions old-fluid up to distance 3, 2, 1
#pragma unroll
            for (int i = 1; i < 9; i++) {
                const unsigned bits = (um >> (3 * (i - 1))) & 7u;
                if (bits == 7u) d3 |= 1u << (i - 1);
                if ((bits & 3u) == 3u) d2 |= 1u << (i - 1);
                if (bits & 1u) d1 |= 1u << (i - 1);
            }
            unsigned dirs = 0;
            int scheme = 0;  // 1: A1, 2: A2, 3: A3, 0: equilibrium
            if (p.refill <= LBM_REFILL_A1 && d3) {
                dirs = d3;
                scheme = 1;
            } else if (p.refill <= LBM_REFILL_A2 && d2) {
                dirs = d2;
                scheme = 2;
            } else if (d1) {
                dirs = d1;
                scheme = 3;
            }
            if (scheme) {
                // lane 3j + (d-1) sums f_j(x + d e_i) over the chosen directions
                const int j = lane / 3, d = lane % 3 + 1;
                const C wd = scheme == 1 ? (d == 1 ? (C)3 : (d == 2 ? (C)-3 : (C)1))
                                         : (scheme == 2 ? (d == 1 ? (C)2 : (d == 2 ? (C)-1 : (C)0))
                                                        : (d == 1 ? (C)1 : (C)0));
                C sum = 0;
                if (lane < 27 && wd != (C)0) {
#pragma unroll
                    for (int i = 1; i < 9; i++) {
                        if (!((dirs >> (i - 1)) & 1u)) continue;
                        sum += (C)ldc(fsn + j * pl + neighbour(L, x, y, d * cx(i), d * cy(i)));
                    }
                }
                C v = wd * sum;
                v += __shfl_down_sync(FULL, v, 1) + __shfl_down_sync(FULL, v, 2);
                v = stored(fsn, v / (C)__popc(dirs));
                if (lane < 27 && lane % 3 == 0) st(static_cast<S *>(fnew) + j * pl + k, v);
                fj = __shfl_sync(FULL, v, 3 * (lane < 9 ? lane : 0));  // lane j <- lane 3j
            } else if (lane < 9) {
                // no old-fluid neighbour: equilibrium at rho0 and the solid's velocity
                double ux, uy, ddx, ddy;
                point_velocity(L, b.xn, b.yn, b.vxn, b.vyn, b.omn, (double)x, (double)y, ux, uy,
                               ddx, ddy);
                const double eu = cx(lane) * ux + cy(lane) * uy, uu = ux * ux + uy * uy;
                const double fe =
                    p.rho0 * wgt<double>(lane) * (1.0 + 3.0 * eu + 4.5 * eu * eu - 1.5 * uu);
                fj = stored(fsn, (C)(Prec<P>::dev ? fe - wgt<double>(lane) : fe));
                st(static_cast<S *>(fnew) + lane * pl + k, fj);
            }
            __syncwarp();
        } else if (lane < 9) {
            fj = (C)ldc(fsn + lane * pl + k);  // covered: its post-collision populations
        }
        // momentum and mass of the node (post-collision if covered, refilled if
        // fresh), summed in the arithmetic precision of the storage mode
        C jm[3] = {0, 0, 0};
        if (lane < 9) {
            C v = fj;
            if (Prec<P>::dev) v += wgt<C>(lane);
            jm[0] = (C)cx(lane) * v;
            jm[1] = (C)cy(lane) * v;
            jm[2] = v;
        }
        warp_sum(jm);
        if (lane == 0) {
            // fresh: from the solid; covered: to it.  The node's momentum, its
            // velocity relative to the boundary and its lever about the new
            // centre in the arithmetic precision C (the FP64 mode from the
            // domain node at the nearest periodic image; the deviation modes
            // from the node's unwrapped coordinates and the split centre)
            const C sgn = (code & 1) ? (C)-1 : (C)1;
            const C mx = jm[0], my = jm[1], mm = jm[2];
            C ux, uy, dx, dy;
            if (P == LBM_FP64) {
                double vx, vy, ddx, ddy;
                point_velocity(L, b.xn, b.yn, b.vxn, b.vyn, b.omn, (double)x, (double)y, vx, vy,
                               ddx, ddy);
                ux = (C)vx;
                uy = (C)vy;
                dx = (C)ddx;
                dy = (C)ddy;
            } else {
                dx = (C)(ev.z - b.ix1) - (C)b.fx1;
                dy = (C)(ev.w - b.iy1) - (C)b.fy1;
                const C vxn = (C)b.vxn, vyn = (C)b.vyn, omn = (C)b.omn;
                ux = vxn - omn * dy;
                uy = vyn + omn * dx;
            }
            // the Eq. 5 record's booking: the same, or relative to the boundary, m (u - v)
            const C rx = p.relative_changes ? mx - mm * ux : mx;
            const C ry = p.relative_changes ? my - mm * uy : my;
            acc[0] = (double)(sgn * mx);
            acc[1] = (double)(sgn * my);
            acc[2] = (double)(sgn * (dx * my - dy * mx));
            acc[3] = (double)(sgn * rx);
            acc[4] = (double)(sgn * ry);
            acc[5] = (double)(sgn * (dx * ry - dy * rx));
        }
    }
    if (lane == 0)
        for (int q = 0; q < 6; q++) p.ev_mom[6 * e + q] = acc[q];
    __syncwarp();
}

// The state of a moving solid becomes that of t+1 (xo, yo keep R(t) for the
// events of the step).
__device__ __forceinline__ void advance_solid(const Lattice &L, DSolid &b) {
    b.x = b.xn;
    b.y = b.yn;
    b.xw = b.xnw;
    b.yw = b.ynw;
    b.ix0 = b.ix1;
    b.iy0 = b.iy1;
    b.fx0 = b.fx1;
    b.fy0 = b.fy1;
    b.xwi = L.bc_x == LBM_PERIODIC ? b.ix1 - L.nx * floor_div(b.ix1, L.nx) : b.ix1;
    b.ywi = L.bc_y == LBM_PERIODIC ? b.iy1 - L.ny * floor_div(b.iy1, L.ny) : b.iy1;
    b.xwr = b.fx1;
    b.ywr = b.fy1;
    b.vx = b.vxn;
    b.vy = b.vyn;
    b.om = b.omn;
    b.vxf = (float)b.vxn;
    b.vyf = (float)b.vyn;
    b.omf = (float)b.omn;
    b.xf = b.xnf;
    b.yf = b.ynf;
}

// P and R, one warp per moving solid (whole blocks call it).
struct RingShared {
    int2 queue[WARPS][EVENTS];
    int qn[WARPS];
    int4 ipos[NEAR_TILE];
    float4 fpos[NEAR_TILE];
    float rad[NEAR_TILE];
};
__device__ __forceinline__ void rings(const StepParams &p, RingShared &sh) {
    const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
    const long long t = *p.t;
    const volatile unsigned int *ctl = p.bar;
    // nothing changes the control words between the force kernel and the events
    const bool pairs = ctl[3] != 0u || __uint_as_float(ctl[2]) >= 0.5f * NEAR_MARGIN;
    if (pairs) phase_pairs_block(p, blockIdx.x * WARPS, sh.ipos, sh.fpos, sh.rad);
    const int m = blockIdx.x * WARPS + wib;
    if (m >= p.nmoving) return;
    const int s = p.moving[m];
    DSolid &b = p.S[s];
    if (pairs && lane == 0) {  // the centres the near list was taken at
        b.ixt = b.ix0;
        b.iyt = b.iy0;
        b.fxt = b.fx0;
        b.fyt = b.fy0;
    }
    __syncwarp();
    if (solid_ok(b)) phase_ring(p, s, lane, t, sh.queue[wib], sh.qn[wib]);
    else if (lane == 0) atomicOr(p.status, 2);
}

// Beside the advection-collision kernel.
__global__ void __launch_bounds__(SW_BLOCK, 4) k_ring(const StepParams p) {
    __shared__ RingShared sh;
    // the re-rasterisation of an earlier step gave up: the state is not the method's
    // any more, and this launch does nothing (the host reports the time-out)
    if (*(volatile int *)p.status & 4) return;
    rings(p, sh);
}

// A: owners and flags of t+1.
__device__ __forceinline__ void changes(const StepParams &p) {
    const int gt = blockIdx.x * SW_BLOCK + threadIdx.x, nt = gridDim.x * SW_BLOCK;
    const Lattice &L = p.L;
    const int nchg = min(*(volatile int *)p.chg_len, p.chg_cap);
    for (int c = gt; c < nchg; c += nt) {
        const int2 q = p.chg[c];
        const int k = q.x;
        p.owner[k] = (uint16_t)(q.y & 0xFFFF);
        if (q.y & 0x10000) {
            // bit 0 of the node, bit d of the neighbour x + e_d
            const bool sn = (q.y & 0x20000) != 0;
            const int x = k % L.pitch, y = k / L.pitch;
            flag_bit(p.flags, k, 0, sn);
#pragma unroll
            for (int d = 1; d < 9; d++) {
                const int kn = neighbour(L, x, y, cx(d), cy(d));
                if (kn >= 0) flag_bit(p.flags, kn, d, sn);
            }
        }
    }
}

// The clock, and the pair test's control words, once nothing of the step t reads them.
__device__ __forceinline__ void advance_clock(const StepParams &p, long long t) {
    *p.t = t + 1;
    volatile unsigned int *ctl = p.bar;
    if (ctl[3] != 0u || __uint_as_float(ctl[2]) >= 0.5f * NEAR_MARGIN) {
        ctl[2] = 0u;  // the pair test of this step has run
        ctl[3] = 0u;
    }
}

// E: the covered and fresh nodes of step t, dealt to every warp of the grid.
template <int P>
__device__ __forceinline__ void events(const StepParams &p, long long t) {
    const int gt = blockIdx.x * SW_BLOCK + threadIdx.x, nt = gridDim.x * SW_BLOCK;
    void *fnew = ((t + 1) & 1) ? p.f1 : p.f0;  // populations of time t+1
    const int nev = min(*(volatile int *)p.ev_len, p.ev_cap);
    for (int e = gt >> 5; e < nev; e += nt >> 5) phase_event<P>(p, e, threadIdx.x & 31, fnew);
    for (int m = gt; m < p.nmoving; m += nt) advance_solid(p.L, p.S[p.moving[m]]);
}

// A and E (after the advection-collision kernel and k_ring).  Two launches, the second
// set up while the first runs: as one, with a barrier across the grid, it had to be
// launched cooperatively, which waits for an idle GPU.  A step of 2048 x 1024 nodes with
// 125 disks, FP64: 13 us less; 8192 x 4096, 2000 disks, FP32: 3.4; 500 disks on a
// quarter of that: 1.5.  (Without the early start of the second: 1.8 us more there.)
__global__ void __launch_bounds__(SW_BLOCK) k_changes(const StepParams p) {
    // k_events' blocks may take their places; they wait for the end of this launch
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    if (*(volatile int *)p.status & 4) return;
    changes(p);
    if (blockIdx.x != 0 || threadIdx.x != 0) return;
    if (p.spin_limit <= 0) atomicOr(p.status, 4);  // as cluster_sync
    else advance_clock(p, *p.t);
}
template <int P>
__global__ void __launch_bounds__(SW_BLOCK, 4) k_events(const StepParams p) {
    asm volatile("griddepcontrol.wait;" ::: "memory");
    if (*(volatile int *)p.status & 4) return;
    events<P>(p, *p.t - 1);
}

// The same for few moving solids, in one cluster; RING: after P and R in the same
// launch, where they do not run beside the advection-collision kernel.
template <int P, bool RING>
__global__ void __launch_bounds__(SW_BLOCK, 4) k_remask_few(const StepParams p) {
    early_start();
    __shared__ RingShared sh;
    if (*(volatile int *)p.status & 4) return;
    const long long t = *p.t;
    if constexpr (RING) {
        rings(p, sh);
        if (!cluster_sync(p)) return;
    }
    changes(p);
    if (!cluster_sync(p)) return;
    if (blockIdx.x == 0 && threadIdx.x == 0) advance_clock(p, t);  // every block has read t
    events<P>(p, t);
}

cudaError_t sm_count(int &sms) {
    static std::atomic<int> known{0};
    cudaError_t e = cudaSuccess;
    if (!(sms = known.load())) {
        int dev = 0;
        e = cudaGetDevice(&dev);
        if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
        if (e == cudaSuccess) known = sms;
    }
    return e;
}

template <int P, bool LOCAL, int NT>
cudaError_t launch_f_n(const StepParams &p, cudaStream_t st, int sms) {
    static int per_sm = -1;
    if (per_sm < 0) {
        const cudaError_t e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_forces<P, LOCAL, NT>, NT, 0);
        if (e != cudaSuccess) return e;
    }
    // one solid per block, looped beyond the resident blocks
    return launch_step(p, k_forces<P, LOCAL, NT>, dim3(std::min(p.nsolid, 8 * per_sm * sms)), NT, st, p);
}

// k_links with the interpolated boundary: 96 registers in FP32, five blocks on an SM; seven
// with 72 are 1.5 us slower at 500 disks of r 20 (115 us a step), but take 1000 in one
// wave instead of two (228 -> 216).
template <int P, bool LOCAL>
cudaError_t launch_f(const StepParams &p, cudaStream_t st) {
    int sms = 0;
    const cudaError_t e = sm_count(sms);
    if (e != cudaSuccess) return e;
    if (!p.link_parts)
        return launch_f_n<P, LOCAL, FB>(p, st, sms);
    const dim3 grid(std::min(p.nsolid, 64 * sms), p.link_parts);
    constexpr bool fp64 = P == LBM_FP64;
    if (p.boundary != LBM_INTERPOLATED) return launch_step(p, k_links<P, LOCAL, false, fp64 ? 5 : 7>, grid, FB, st, p);
    if (!fp64 && p.nsolid * p.link_parts > 5 * sms)
        return launch_step(p, k_links<P, LOCAL, true, fp64 ? 4 : 7>, grid, FB, st, p);
    return launch_step(p, k_links<P, LOCAL, true, fp64 ? 4 : 5>, grid, FB, st, p);
}

// Re-rasterisation of up to FEW_MOVING solids: one cluster of 8 blocks (one solid: 4)
// and its barrier, instead of a cooperative launch (which waits for an idle GPU) and a
// barrier in memory.  A step of 321 x 197 nodes with 6 moving disks, FP32: 41.6 -> 35.9
// us launched one by one, 32.0 -> 29.7 in a graph; 500 x 300 with 16: 42.7 -> 38.6, 34.8
// -> 31.9.  16: 64 warps have about as many events to do as a step of that many solids
// lists, and the cluster no more blocks to give.
template <int P>
cudaError_t launch_few(const StepParams &p, bool ring, cudaStream_t st) {
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(p.nmoving > 1 ? 8 : 4);
    cfg.blockDim = dim3(SW_BLOCK);
    cfg.stream = st;
    cudaLaunchAttribute at[2] = {};
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = cfg.gridDim.x;
    at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
    at[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = at;
    cfg.numAttrs = p.early ? 2 : 1;
    return ring ? cudaLaunchKernelEx(&cfg, k_remask_few<P, true>, p) : cudaLaunchKernelEx(&cfg, k_remask_few<P, false>, p);
}

template <int P>
cudaError_t launch_r(const StepParams &p, bool ring, cudaStream_t st) {
    if (p.nmoving <= FEW_MOVING) return launch_few<P>(p, ring, st);
    static int per_sm = -1, sms = 0;
    if (per_sm < 0) {
        int dev = 0;
        cudaError_t e = cudaGetDevice(&dev);
        if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
        if (e == cudaSuccess)
            e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_events<P>, SW_BLOCK, 0);
        if (e != cudaSuccess) return e;
    }
    // the changes go to every thread, the events to every warp: not many more than a
    // step has of them (tens per moving solid), up to every resident block
    const int blocks = std::min(per_sm * sms, 4 * p.nmoving);
    k_changes<<<std::min(2 * sms, p.nmoving), SW_BLOCK, 0, st>>>(p);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(blocks);
    cfg.blockDim = dim3(SW_BLOCK);
    cfg.stream = st;
    cudaLaunchAttribute at{};
    at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at.val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = &at;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, k_events<P>, p);
}

// ------------------------------------------------------------- batch

// Force records of a batch of independent domains whose solids rest, the first
// kernel of a step: one block per (case, solid) item of the active list (the links
// and the record, as k_forces).  The last block to finish (a ticket, no waiting)
// advances the step counter of every active case and swaps its population
// buffers, after every block has read them.  Batch convention: between steps f0
// holds the current populations; the fused kernel, which comes after this swap,
// reads f1 and writes f0.
// BLOCKS: on an SM.
template <int P, bool LOCAL, int NT, int BLOCKS>
__global__ void __launch_bounds__(NT, BLOCKS)
    k_solids_batch(StepParams *cases, const int2 *__restrict__ items,
                   const int *__restrict__ nitems, const int *__restrict__ active,
                   const int *__restrict__ nactive, unsigned int *ticket) {
    using S = typename Prec<P>::S;
    __shared__ bool last;
    __shared__ LinkShared<P, false, NT> sh;
    const int n = *nitems;
    for (int k = blockIdx.x; k < n; k += gridDim.x) {
        const int2 it = items[k];
        const StepParams &p = cases[it.x];
        const long long t = *p.t;
        const DSolid &b = p.S[it.y];
        if (!solid_ok(b)) {
            if (threadIdx.x == 0) atomicOr(p.status, 2);
            continue;
        }
        // FP64 sums throughout: the drags decide when a case has converged
        double sum = 0.0, acc[6];
        solid_links<P, LOCAL, false, ghosts<P>(), true>(p, b, it.y, static_cast<S *>(p.f0), true, false, t, NT, 0,
                                                        1, sh, sum);
        block_sums(sh, sum, acc);
        if (threadIdx.x < 32) {
            const double none[6] = {0.0, 0.0, 0.0, 0.0, 0.0, 0.0};  // resting: no node changes type
            record_forces(p, it.y, threadIdx.x, t, acc, none);
        }
        __syncthreads();  // sh.part is reused
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        __threadfence();
        last = atomicAdd(ticket, 1u) == gridDim.x - 1;
    }
    __syncthreads();
    if (!last) return;
    __threadfence();
    const int na = *nactive;
    for (int a = threadIdx.x; a < na; a += blockDim.x) {
        StepParams &p = cases[active[a]];
        *p.t += 1;
        void *f = p.f0;  // the buffer that the step fills becomes the current one
        p.f0 = p.f1;
        p.f1 = f;
    }
    if (threadIdx.x == 0) *ticket = 0;
}

template <int P, bool LOCAL, int NT, int BLOCKS>
cudaError_t launch_sb_b(const BatchLaunch &b, cudaStream_t st, int sms) {
    const int blocks = std::max(1, std::min(b.max_items, BLOCKS * sms));
    k_solids_batch<P, LOCAL, NT, BLOCKS><<<blocks, NT, 0, st>>>(b.cases, b.items, b.nitems, b.active,
                                                                b.nactive, b.ticket);
    return cudaGetLastError();
}

// 80 registers a thread, or 64 and some spills where that makes room for all items at once
// (96 channels of 256 x 128: 58.8 us a step with 80, 59.8 with 64; 512 of 128 to 1024 x 64
// to 512, in two waves with 80: 1130, with 64 1115).
template <int P, bool LOCAL, int NT>
cudaError_t launch_sb_n(const BatchLaunch &b, cudaStream_t st, int sms) {
    return b.max_items <= 768 / NT * sms ? launch_sb_b<P, LOCAL, NT, 768 / NT>(b, st, sms)
                                         : launch_sb_b<P, LOCAL, NT, 1024 / NT>(b, st, sms);
}

// A disk has about 9.5 r + 7 candidates.  Up to 128, one turn of 128 threads; more take
// another turn, a chain of loads, where 256 threads need one: 96 open channels of 256 x
// 128 with disks of up to 16, 68.1 -> 65.9 us a step; two of 1024 x 512, r 51, 34.3 ->
// 28.0; but 8 of 64 x 48, r 4.8, 13.9 -> 14.5.  More items than find room at 256 threads
// go to 128.
template <int P, bool LOCAL>
cudaError_t launch_sb(const BatchLaunch &b, cudaStream_t st) {
    int sms = 0;
    const cudaError_t e = sm_count(sms);
    if (e != cudaSuccess) return e;
    return b.rmax > 12.5 && b.max_items <= 4 * sms ? launch_sb_n<P, LOCAL, 256>(b, st, sms)
                                                   : launch_sb_n<P, LOCAL, FB>(b, st, sms);
}

// Convergence test and list rebuild, one block.  Case states: 0 active,
// 1 converged, 2 step cap reached, 3 unstable (a status bit raised, or a
// non-finite drag).  The drag of a case is the x component of the Eq. 5
// force summed over its solids in the latest record; it has converged when
// it moved by less than tol relative since the previous test.  Modes:
// BATCH_TEST tests and rebuilds the lists if a case retired; BATCH_REBUILD
// keeps the states, clears the drag history and rebuilds the lists;
// BATCH_GATHER only copies the step counters.  Every mode copies them.
constexpr int CV_BLOCK = 1024;
__global__ void __launch_bounds__(CV_BLOCK)
    k_batch_converge(BatchLaunch b, int ncase, double tol, long long max_steps, int window,
                     int mode, int *state, double *drag, int *calm, double *anchor,
                     long long *steps, int *toff, int *ioff, int seg_w, int tile_n) {
    __shared__ int changed;
    __shared__ int wsum[3][CV_BLOCK / 32];
    __shared__ int carry[3];
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    if (tid == 0) {
        changed = mode == BATCH_REBUILD;
        carry[0] = carry[1] = carry[2] = 0;
    }
    __syncthreads();
    for (int c = tid; c < ncase; c += CV_BLOCK) {
        const StepParams &p = b.cases[c];
        const long long t = *p.t;
        steps[c] = t;
        if (mode == BATCH_GATHER) continue;
        if (mode == BATCH_REBUILD) {
            drag[c] = __longlong_as_double(0x7ff8000000000000ll);  // no history
            anchor[c] = drag[c];
            calm[c] = 0;
            continue;
        }
        if (state[c] != 0) continue;
        int ns = 0;
        if (*p.status != 0) ns = 3;
        double D = 0.0;
        if (ns == 0 && p.nsolid > 0 && t >= 1) {
            const long long slot = (t - 1) % p.ring_len;
            const double *rg = p.ring + (slot * 2 + 1) * p.nsolid * 3;
            for (int s = 0; s < p.nsolid; s++) D += rg[s * 3];
            // converged once the drag has stayed within tol of the drag at the
            // start of `window` tests in a row (window 1: of the previous test)
            const double a = anchor[c];
            drag[c] = D;
            if (!isfinite(D)) ns = 3;
            else if (isfinite(a) && fabs(D - a) < tol * fabs(D)) {
                if (++calm[c] >= window) ns = 1;
            } else {
                anchor[c] = D;
                calm[c] = 0;
            }
        }
        if (ns == 0 && t >= max_steps) ns = 2;
        if (ns != 0) {
            state[c] = ns;
            changed = 1;
        }
    }
    __syncthreads();
    if (!changed) return;
    // exclusive scans of (active, tiles, items) over the cases, in chunks
    for (int base = 0; base < ncase; base += CV_BLOCK) {
        const int c = base + tid;
        int v[3] = {0, 0, 0};
        if (c < ncase && state[c] == 0) {
            const Lattice &L = b.cases[c].L;
            v[0] = 1;
            v[1] = ((L.nx + seg_w - 1) / seg_w * L.ny + tile_n - 1) / tile_n;
            v[2] = b.cases[c].nsolid;
        }
        int inc[3];
#pragma unroll
        for (int q = 0; q < 3; q++) {
            inc[q] = v[q];
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int u = __shfl_up_sync(FULL, inc[q], o);
                if (lane >= o) inc[q] += u;
            }
            if (lane == 31) wsum[q][wid] = inc[q];
        }
        __syncthreads();
        if (wid == 0) {
#pragma unroll
            for (int q = 0; q < 3; q++) {
                int w = wsum[q][lane];
#pragma unroll
                for (int o = 1; o < 32; o <<= 1) {
                    const int u = __shfl_up_sync(FULL, w, o);
                    if (lane >= o) w += u;
                }
                wsum[q][lane] = w;  // inclusive over warps
            }
        }
        __syncthreads();
        int ex[3];
#pragma unroll
        for (int q = 0; q < 3; q++) ex[q] = carry[q] + (wid ? wsum[q][wid - 1] : 0) + inc[q] - v[q];
        if (v[0]) {
            b.active[ex[0]] = c;
            toff[c] = ex[1];
            ioff[c] = ex[2];
        }
        __syncthreads();
        if (tid == 0)
            for (int q = 0; q < 3; q++) carry[q] += wsum[q][CV_BLOCK / 32 - 1];
        __syncthreads();
    }
    const int na = carry[0];
    if (tid == 0) {
        *b.nactive = na;
        *b.ntiles = carry[1];
        *b.nitems = carry[2];
    }
    int4 *tiles = b.tiles;
    int2 *items = b.items;
    for (int a = 0; a < na; a++) {
        const int c = b.active[a];
        const Lattice &L = b.cases[c].L;
        const int nseg = (L.nx + seg_w - 1) / seg_w;
        const int nt = (nseg * L.ny + tile_n - 1) / tile_n, o = toff[c];
        for (int k = tid; k < nt; k += CV_BLOCK)
            tiles[o + k] = make_int4(c, k * tile_n % nseg, k * tile_n / nseg, nseg);
        const int ns = b.cases[c].nsolid, oi = ioff[c];
        for (int s = tid; s < ns; s += CV_BLOCK) items[oi + s] = make_int2(c, s);
    }
}

}  // namespace

cudaError_t launch_solids_batch(const BatchLaunch &b, cudaStream_t st) {
    if (b.precision == LBM_FP64)
        return b.local ? launch_sb<LBM_FP64, true>(b, st) : launch_sb<LBM_FP64, false>(b, st);
    if (b.precision == LBM_FP32_DEV)
        return b.local ? launch_sb<LBM_FP32_DEV, true>(b, st) : launch_sb<LBM_FP32_DEV, false>(b, st);
    return b.local ? launch_sb<LBM_FP16_DEV, true>(b, st) : launch_sb<LBM_FP16_DEV, false>(b, st);
}

cudaError_t launch_batch_converge(const BatchLaunch &b, const BatchState &s, int mode,
                                  cudaStream_t st) {
    k_batch_converge<<<1, CV_BLOCK, 0, st>>>(b, s.ncase, s.tol, s.max_steps, s.window, mode,
                                             s.state, s.drag, s.calm, s.anchor, s.steps, s.toff,
                                             s.ioff, segment_nodes(b.precision, b.variant),
                                             tile_segments(b.tile_h));
    return cudaGetLastError();
}

cudaError_t launch_forces(const StepParams &p, cudaStream_t st) {
    if (p.nsolid == 0) return cudaSuccess;
    const bool local = p.rho_w_mode == LBM_RHOW_LOCAL;
    switch (p.precision) {
        case LBM_FP64: return local ? launch_f<LBM_FP64, true>(p, st) : launch_f<LBM_FP64, false>(p, st);
        case LBM_FP32_DEV:
            return local ? launch_f<LBM_FP32_DEV, true>(p, st) : launch_f<LBM_FP32_DEV, false>(p, st);
        default: return local ? launch_f<LBM_FP16_DEV, true>(p, st) : launch_f<LBM_FP16_DEV, false>(p, st);
    }
}

cudaError_t launch_record(const StepParams &p, cudaStream_t st) {
    if (p.nsolid == 0 || !p.link_parts) return cudaSuccess;
    return launch_step(p, k_record, dim3((p.nsolid + WARPS - 1) / WARPS), SW_BLOCK, st, p);
}

cudaError_t launch_ring(const StepParams &p, cudaStream_t st) {
    if (p.nmoving == 0) return cudaSuccess;
    k_ring<<<(p.nmoving + WARPS - 1) / WARPS, SW_BLOCK, 0, st>>>(p);
    return cudaGetLastError();
}

cudaError_t launch_remask(const StepParams &p, bool ring, cudaStream_t st) {
    if (p.nmoving == 0) return cudaSuccess;
    switch (p.precision) {
        case LBM_FP64: return launch_r<LBM_FP64>(p, ring, st);
        case LBM_FP32_DEV: return launch_r<LBM_FP32_DEV>(p, ring, st);
        default: return launch_r<LBM_FP16_DEV>(p, ring, st);
    }
}

}  // namespace gbm
