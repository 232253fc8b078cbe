// Device code of the fused pull-advection + half-way bounce-back + BGK
// collision (Eq. 1-3, Eq. 8), shared by the single-domain kernel
// (k_stream_collide.cu) and the batch kernels (k_stream_collide_batch.cu).
// Each translation unit compiles its own copy, so that the register budget of
// one kernel family does not constrain the other's per-node path.
//
// Layout: SoA planes f_i[ny][pitch], x fastest, pitch a multiple of 64.
// Every thread owns V consecutive nodes of one row, V chosen so that one
// population of those nodes is 16, 8 or 4 bytes.  Each of the nine pulls is one
// aligned vector load from the source row (y - c_y); the x-shifted pulls (c_x =
// +-1) take the missing neighbour element from the adjacent lane with a warp
// shuffle (lanes 0 and 31 load it directly), so DRAM sees each population plane
// read once, fully coalesced.  Results go out as nine vector stores (solid nodes
// and nodes in the row padding store zeros).
//
// Bounce-back in the FP64 and FP32 modes (sc_row): a population that comes back
// from a solid, f~_opp(x) + 6 w_i rho_w (e_i . v), is found by the force kernel
// of the step, which visits every fluid-solid link anyway, and left where the
// pull reads it: in slot i of the solid node x - e_i, which holds no state.  So
// the vector path treats a node next to a solid as any other.  Walls, periodic
// edges and open columns are put in place in registers by the threads that hold
// them.  No node takes a per-node path: next to the solids one ran with one or
// two active lanes per warp through a chain of dependent loads (flags, owner,
// solid record), which cost 0.05 ms of 0.41 on 8192 x 4096 nodes with 2000 disks
// in FP32 (and held the MRT kernel with the interpolated boundary at 0.31 ms on
// a quarter of that).
//
// FP16 storage (sc_tile) would round such a value once more than arithmetic in
// registers does, so there the nodes next to a solid or a wall and the first and
// last column take a per-node path (update_node), in the vector kernel itself or
// in a pass after it.
//
// Storage: FP64 stores f_i; the deviation modes store f_i - w_i (FP32 or
// FP16) and compute in FP32 entirely in deviation form, so that the small
// deviations keep their relative precision:
//   drho = sum d_i,  rho = 1 + drho,  rho u = sum e_i d_i,
//   deq_i = w_i (drho + rho (3 e.u + 4.5 (e.u)^2 - 1.5 u.u)).
#pragma once
#include "lbm_internal.cuh"

namespace gbm {

namespace {

template <int P> struct Raw;
template <> struct Raw<LBM_FP64> { using R = double; };
template <> struct Raw<LBM_FP32_DEV> { using R = float; };
template <> struct Raw<LBM_FP16_DEV> { using R = unsigned short; };

template <int BYTES> struct Word;
template <> struct Word<2> { using T = uint16_t; };
template <> struct Word<4> { using T = uint32_t; };
template <> struct Word<8> { using T = uint2; };
template <> struct Word<16> { using T = uint4; };

// V consecutive values of one population plane, loaded as one word
template <class R, int V> union Pack {
    typename Word<sizeof(R) * V>::T u;
    R r[V];
};
template <int V> union FlagPack {
    typename Word<2 * V>::T u;
    uint16_t f[V];
};

__device__ __forceinline__ double cvt(double v) { return v; }
__device__ __forceinline__ float cvt(float v) { return v; }
__device__ __forceinline__ float cvt(unsigned short v) { return __half2float(__ushort_as_half(v)); }
__device__ __forceinline__ void put(double &d, double v) { d = v; }
__device__ __forceinline__ void put(float &d, float v) { d = v; }
__device__ __forceinline__ void put(unsigned short &d, float v) {
    d = __half_as_ushort(__float2half_rn(v));
}

// two adjacent values of a population plane at once
__device__ __forceinline__ void put2(unsigned short *d, float a, float b) {
    *reinterpret_cast<__half2 *>(d) = __floats2half2_rn(a, b);
}

// Paired FP32 arithmetic: one instruction for the same operation on two nodes.
__device__ __forceinline__ float2 add2(float2 a, float2 b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ float2 sub2(float2 a, float2 b) {
    return __fadd2_rn(a, make_float2(-b.x, -b.y));
}
__device__ __forceinline__ float2 mul2(float2 a, float2 b) { return __fmul2_rn(a, b); }
__device__ __forceinline__ float2 fma2(float2 a, float2 b, float2 c) { return __ffma2_rn(a, b, c); }
__device__ __forceinline__ float2 dup2(float a) { return make_float2(a, a); }

__device__ __forceinline__ double shfl_up1(double v) { return __shfl_up_sync(0xffffffffu, v, 1); }
__device__ __forceinline__ float shfl_up1(float v) { return __shfl_up_sync(0xffffffffu, v, 1); }
__device__ __forceinline__ unsigned short shfl_up1(unsigned short v) {
    return (unsigned short)__shfl_up_sync(0xffffffffu, (int)v, 1);
}
__device__ __forceinline__ double shfl_dn1(double v) { return __shfl_down_sync(0xffffffffu, v, 1); }
__device__ __forceinline__ float shfl_dn1(float v) { return __shfl_down_sync(0xffffffffu, v, 1); }
__device__ __forceinline__ unsigned short shfl_dn1(unsigned short v) {
    return (unsigned short)__shfl_down_sync(0xffffffffu, (int)v, 1);
}

// FP16: replace the bounced populations of node (x, y) (rare path): population i,
// whose source x - e_i is a wall or a solid, becomes f~_opp(x) + 6 w_i rho_w
// (e_i . v) with v the wall's or solid's velocity at x - e_i / 2 (Sec. III.A;
// the moving-wall term).
// BND: disks with the interpolated boundary (LBM_INTERPOLATED), compiled only
// into the kernels that run the per-node path outside the vector path.
template <bool LOCAL, bool BND = false>
__device__ __forceinline__ void bounce(const StepParams &p, const Raw<LBM_FP16_DEV>::R *fin, int x,
                                       int y, uint16_t fl, float (&g)[9]) {
    using C = float;
    const Lattice &L = p.L;
    const int k = y * L.pitch + x;
    const int plane = (int)L.plane;
    C rho_w = p.rho0_f;
    if (LOCAL) {
        C s = 0;
#pragma unroll
        for (int j = 0; j < 9; j++) s += cvt(fin[j * plane + k]);
        rho_w = 1.f + s;
    }
#pragma unroll
    for (int i = 1; i < 9; i++) {
        if (!((fl >> i) & 1u)) continue;
        const int sx = x - cx(i), sy = y - cy(i);
        C vx = 0, vy = 0;
        int xs, ys;
        if (L.bc_y == LBM_WALL && (sy < 0 || sy >= L.ny)) {
            vx = sy < 0 ? p.wall_ux0_f : p.wall_ux1_f;
        } else if (locate(L, sx, sy, xs, ys)) {
            const uint16_t o = p.owner[cell_of(L, xs, ys)];
            if (BND && o != FLUID) {
                // the cut at fraction q of the link towards the wall; linear
                // interpolation of the returned population (deviation form
                // as well: the weights sum to one):
                //   q < 1/2:  2q f~_opp(x) + (1 - 2q) f~_opp(x + e_i) + M
                //   q >= 1/2: (f~_opp(x) + M) / (2q) + (2q - 1) / (2q) f~_i(x)
                // M = 6 w_i rho_w (e_i . v), v at the cut x - q e_i; half-way
                // value where x + e_i is not a fluid node
                const DSolid &b = p.S[o];
                // the offset from the centre's nearest image, split
                int di = x - b.xwi, dj = y - b.ywi;
                if (L.bc_x == LBM_PERIODIC) {
                    if (2 * di > L.nx) di -= L.nx;
                    else if (2 * di < -L.nx) di += L.nx;
                }
                if (L.bc_y == LBM_PERIODIC) {
                    if (2 * dj > L.ny) dj -= L.ny;
                    else if (2 * dj < -L.ny) dj += L.ny;
                }
                const C q = (C)link_fraction_split(di, dj, b.xwr, b.ywr, b.r, -cx(i), -cy(i));
                const C ddx = ((C)di - (C)b.xwr) - q * (C)cx(i);
                const C ddy = ((C)dj - (C)b.ywr) - q * (C)cy(i);
                const C ux = (C)b.vxf - (C)b.omf * ddy, uy = (C)b.vyf + (C)b.omf * ddx;
                const C m = (C)6 * wgt<C>(i) * rho_w * ((C)cx(i) * ux + (C)cy(i) * uy);
                const C back = cvt(fin[opp(i) * plane + k]);
                const C q2 = (C)2 * q;
                if (q2 >= (C)1) {
                    g[i] = (back + m) / q2 + ((q2 - (C)1) / q2) * cvt(fin[i * plane + k]);
                } else if (!((fl >> opp(i)) & 1u)) {
                    int xn, yn;
                    locate(L, x + cx(i), y + cy(i), xn, yn);
                    g[i] = q2 * back +
                           ((C)1 - q2) * cvt(fin[opp(i) * plane + yn * L.pitch + xn]) + m;
                } else {
                    g[i] = back + m;
                }
                continue;
            }
            if (o != FLUID) {
                const DSolid &b = p.S[o];
                vx = b.vxf;
                vy = b.vyf;
                if (b.omf != 0.0f) {
                    // x - e_i / 2 relative to R, nearest periodic image
                    C dx = (C)(x - b.xwi) - (C)(0.5f * cx(i)) - (C)b.xwr;
                    C dy = (C)(y - b.ywi) - (C)(0.5f * cy(i)) - (C)b.ywr;
                    if (L.bc_x == LBM_PERIODIC) {
                        if (dx > (C)(0.5 * L.nx)) dx -= (C)L.nx;
                        else if (dx < (C)(-0.5 * L.nx)) dx += (C)L.nx;
                    }
                    if (L.bc_y == LBM_PERIODIC) {
                        if (dy > (C)(0.5 * L.ny)) dy -= (C)L.ny;
                        else if (dy < (C)(-0.5 * L.ny)) dy += (C)L.ny;
                    }
                    const C om = b.omf;
                    vx -= om * dy;
                    vy += om * dx;
                }
            }
        }
        const C back = cvt(fin[opp(i) * plane + k]);
        g[i] = back + (C)6 * wgt<C>(i) * rho_w * ((C)cx(i) * vx + (C)cy(i) * vy);
    }
}

// Is (rho, ux, uy) not a physical state?  FP64: from the high words (the FP64
// unit is what bounds the FP64 kernel, and a comparison occupies it too).
__device__ __forceinline__ bool unphysical(float r, float vx, float vy) {
    return !(r > 0.f) || !(fabsf(vx) < 1e30f) || !(fabsf(vy) < 1e30f);
}
__device__ __forceinline__ bool unphysical(double r, double vx, double vy) {
    constexpr int BIG = 0x46293E59;  // high word of 1e30
    const int h = __double2hiint(r);
    return h <= 0 || h >= 0x7FF00000 || (__double2hiint(vx) & 0x7FFFFFFF) > BIG ||
           (__double2hiint(vy) & 0x7FFFFFFF) > BIG;
}

// BGK collision (with Guo forcing when FORCE) of one node in place; check(rho, ux, uy)
// sees its density and velocity.
template <int P, bool FORCE, class Check>
__device__ __forceinline__ void collide(const StepParams &p, typename Prec<P>::C (&g)[9], Check &&check) {
    using C = typename Prec<P>::C;
    C s0 = 0, jx = 0, jy = 0;
#pragma unroll
    for (int i = 0; i < 9; i++) {
        s0 += g[i];
        jx += (C)cx(i) * g[i];
        jy += (C)cy(i) * g[i];
    }
    const C rho = Prec<P>::dev ? (C)1 + s0 : s0;
    const C Fx = pick<C>(p.body_x, p.body_xf), Fy = pick<C>(p.body_y, p.body_yf);
    const C inv = reciprocal(rho);
    const C ux = FORCE ? (jx + (C)0.5 * Fx) * inv : jx * inv;
    const C uy = FORCE ? (jy + (C)0.5 * Fy) * inv : jy * inv;
    const C uu = ux * ux + uy * uy;
    const C om = pick<C>(p.omega, p.omega_f);
    check(rho, ux, uy);
#pragma unroll
    for (int i = 0; i < 9; i++) {
        const C eu = (C)cx(i) * ux + (C)cy(i) * uy;
        const C poly = (C)3 * eu + (C)4.5 * eu * eu - (C)1.5 * uu;
        C eq;
        if (Prec<P>::dev) eq = wgt<C>(i) * (s0 + rho * poly);  // f_eq - w_i
        else eq = rho * wgt<C>(i) * ((C)1 + poly);
        C o = g[i] - (g[i] - eq) * om;
        if (FORCE) {
            o += ((C)1 - (C)0.5 * om) * wgt<C>(i) *
                 ((C)3 * (((C)cx(i) - ux) * Fx + ((C)cy(i) - uy) * Fy) +
                  (C)9 * eu * ((C)cx(i) * Fx + (C)cy(i) * Fy));
        }
        g[i] = o;
    }
}

// MRT collision of one node in place (Sec. IV names the model and its rates
// S = diag(0, 1.64, 1.54, 0, 1.9, 0, 1.9, 1/tau, 1/tau)): the moments of the
// basis (rho, e, eps, j_x, q_x, j_y, q_y, p_xx, p_xy) relax towards those of
// the Eq. 8 equilibrium, -2 rho + 3 j^2 / rho, rho - 3 j^2 / rho, -j,
// (j_x^2 - j_y^2) / rho and j_x j_y / rho (in the deviation modes minus the
// moments of the weights, which are 1, -2, 1 and zeros), and the change goes
// back to the populations through the transposed basis over the squared row
// norms (36, 36, 12, 12, 4, 4).  No body force.  check(rho, ux, uy) sees the
// node's density and velocity.
template <int P, class Check>
__device__ __forceinline__ void collide_mrt(const StepParams &p, typename Prec<P>::C (&g)[9], Check &&check) {
    using C = typename Prec<P>::C;
    const C ax = g[1] + g[2] + g[3] + g[4], dg = g[5] + g[6] + g[7] + g[8];
    const C s0 = g[0] + ax + dg;
    const C jx = g[1] - g[3] + g[5] - g[6] - g[7] + g[8];
    const C jy = g[2] - g[4] + g[5] + g[6] - g[7] - g[8];
    const C rho = Prec<P>::dev ? (C)1 + s0 : s0;
    const C inv = reciprocal(rho);
    check(rho, jx * inv, jy * inv);
    const C jj = (jx * jx + jy * jy) * inv;
    const C e = (C)-4 * g[0] - ax + (C)2 * dg;
    const C eps = (C)4 * g[0] - (C)2 * ax + dg;
    const C qx = (C)2 * (g[3] - g[1]) + g[5] - g[6] - g[7] + g[8];
    const C qy = (C)2 * (g[4] - g[2]) + g[5] + g[6] - g[7] - g[8];
    const C pxx = g[1] - g[2] + g[3] - g[4];
    const C pxy = g[5] - g[6] + g[7] - g[8];
    const C eeq = Prec<P>::dev ? (C)-2 * s0 + (C)3 * jj : (C)-2 * rho + (C)3 * jj;
    const C epseq = Prec<P>::dev ? s0 - (C)3 * jj : rho - (C)3 * jj;
    const C om = pick<C>(p.omega, p.omega_f);
    const C de = (C)(1.64 / 36.0) * (e - eeq);
    const C dp = (C)(1.54 / 36.0) * (eps - epseq);
    const C dqx = (C)(1.9 / 12.0) * (qx + jx);
    const C dqy = (C)(1.9 / 12.0) * (qy + jy);
    const C dxx = (C)0.25 * om * (pxx - (jx * jx - jy * jy) * inv);
    const C dxy = (C)0.25 * om * (pxy - jx * jy * inv);
    const C a = -de - (C)2 * dp, b = (C)2 * de + dp;
    g[0] -= (C)4 * (dp - de);
    g[1] -= a - (C)2 * dqx + dxx;
    g[2] -= a - (C)2 * dqy - dxx;
    g[3] -= a + (C)2 * dqx + dxx;
    g[4] -= a + (C)2 * dqy - dxx;
    g[5] -= b + dqx + dqy + dxy;
    g[6] -= b - dqx + dqy - dxy;
    g[7] -= b - dqx - dqy + dxy;
    g[8] -= b + dqx - dqy - dxy;
}

// Inlet profile of an open channel at row y: u_in = 4 umax y' (ny - y') / ny^2,
// y' = y + 1/2 (walls at y = -1/2 and ny - 1/2); in the precision C of the
// kernel (no FP64 arithmetic in the FP32 kernels).
template <class C>
__device__ __forceinline__ C inlet_ux(const StepParams &p, int y) {
    const C h = (C)p.L.ny, yy = (C)y + (C)0.5;
    return (C)4 * pick<C>(p.umax, p.umax_f) * yy * (h - yy) / (h * h);
}

// feq(rho0, (u_in, 0)) into g (deviation form in the deviation modes).
template <int P>
__device__ __forceinline__ void inlet_equilibrium(const StepParams &p, typename Prec<P>::C u_in,
                                                  typename Prec<P>::C (&g)[9]) {
    using C = typename Prec<P>::C;
    const C r = pick<C>(p.rho0, p.rho0_f);
#pragma unroll
    for (int i = 0; i < 9; i++) {
        const C eu = (C)cx(i) * u_in;
        const C poly = (C)3 * eu + (C)4.5 * eu * eu - (C)1.5 * u_in * u_in;
        g[i] = Prec<P>::dev ? wgt<C>(i) * ((r - (C)1) + r * poly) : r * wgt<C>(i) * ((C)1 + poly);
    }
}

// Non-equilibrium extrapolation onto an open column from the post-collision
// populations g of its inner neighbour n, in place: g + feq(rho_b, u_b) -
// feq(rho_n, u_n), with rho_n, u_n the neighbour's density and velocity (BGK
// keeps rho and rho u; Guo forcing adds F to rho u).  Inlet: u_b = (u_in, 0),
// rho_b = rho_n; outlet: rho_b = rho0, u_b = u_n.
template <int P, bool FORCE>
__device__ __forceinline__ void extrapolate_open(const StepParams &p, bool inlet,
                                                 typename Prec<P>::C u_in,
                                                 typename Prec<P>::C (&g)[9]) {
    using C = typename Prec<P>::C;
    C s0 = 0, jx = 0, jy = 0;
#pragma unroll
    for (int i = 0; i < 9; i++) {
        s0 += g[i];
        jx += (C)cx(i) * g[i];
        jy += (C)cy(i) * g[i];
    }
    const C rn = Prec<P>::dev ? (C)1 + s0 : s0;
    if (FORCE) {
        jx -= (C)0.5 * pick<C>(p.body_x, p.body_xf);
        jy -= (C)0.5 * pick<C>(p.body_y, p.body_yf);
    }
    const C uxn = jx / rn, uyn = jy / rn;
    const C ub = inlet ? u_in : uxn, vb = inlet ? (C)0 : uyn;
    const C rb = inlet ? rn : pick<C>(p.rho0, p.rho0_f);
    const C uun = uxn * uxn + uyn * uyn, uub = ub * ub + vb * vb;
#pragma unroll
    for (int i = 0; i < 9; i++) {
        const C en = (C)cx(i) * uxn + (C)cy(i) * uyn, eb = (C)cx(i) * ub + (C)cy(i) * vb;
        const C pn = (C)3 * en + (C)4.5 * en * en - (C)1.5 * uun;
        const C pb = (C)3 * eb + (C)4.5 * eb * eb - (C)1.5 * uub;
        g[i] += wgt<C>(i) * ((rb - rn) + rb * pb - rn * pn);
    }
}

// FP16: complete update of one node, with periodic wrap, bounce-back and walls
// (beyond a non-periodic edge: a resting wall): used for the nodes the vector
// path leaves out (fluid nodes next to a solid or wall, the first and last
// column).  With OPEN, the columns of an open channel are computed here too:
// the update of the inner neighbour (x = 1 or nx - 2, recomputed from fin)
// followed by the non-equilibrium extrapolation; next to a solid neighbour
// the inlet is feq(rho0, u_in) and the outlet updates as a walled node.
// Without OPEN they update as walled nodes and a later pass (open_col)
// replaces them.
template <bool FORCE, bool LOCAL, bool OPEN, int COLL = 0, bool BND = false>
__device__ __noinline__ void update_node(const StepParams &p, const Raw<LBM_FP16_DEV>::R *fin,
                                         Raw<LBM_FP16_DEV>::R *fout, int x, int y) {
    constexpr int P = LBM_FP16_DEV;
    using C = float;
    using R = Raw<P>::R;
    const Lattice &L = p.L;
    const int plane = (int)L.plane;
    const int k = y * L.pitch + x;
    const uint16_t fl = p.flags[k];
    C g[9];
    if (fl & 1u) {
#pragma unroll
        for (int i = 0; i < 9; i++) put(fout[i * plane + k], (C)0);
        return;
    }
    int xu = x;  // node whose update is computed
    uint16_t flu = fl;
    bool open = false;
    C u_in = 0;
    if (OPEN && L.bc_x == LBM_OPEN && (x == 0 || x == L.nx - 1)) {
        const uint16_t fln = p.flags[x == 0 ? k + 1 : k - 1];
        if (x == 0) u_in = inlet_ux<C>(p, y);
        if (!(fln & 1u)) {
            open = true;
            xu = x == 0 ? 1 : x - 1;
            flu = fln;
        } else if (x == 0) {
            inlet_equilibrium<P>(p, u_in, g);
#pragma unroll
            for (int i = 0; i < 9; i++) put(fout[i * plane + k], g[i]);
            return;
        }
    }
    const bool per_x = L.bc_x == LBM_PERIODIC, per_y = L.bc_y == LBM_PERIODIC;
#pragma unroll
    for (int i = 0; i < 9; i++) {
        int xs = xu - cx(i), ys = y - cy(i);
        // wrap along periodic axes; clamp elsewhere (the value is then bounced)
        if (xs < 0) xs = per_x ? xs + L.nx : 0;
        if (xs >= L.nx) xs = per_x ? xs - L.nx : L.nx - 1;
        if (ys < 0) ys = per_y ? ys + L.ny : 0;
        if (ys >= L.ny) ys = per_y ? ys - L.ny : L.ny - 1;
        g[i] = cvt(fin[i * plane + ys * L.pitch + xs]);
    }
    if (flu & 0x1FEu) bounce<LOCAL, BND>(p, fin, xu, y, flu, g);
    auto check = [&](C rho, C ux, C uy) {
        if (unphysical(rho, ux, uy)) atomicOr(p.status, 1);
    };
    if constexpr (COLL == 1) collide_mrt<P>(p, g, check);
    else collide<P, FORCE>(p, g, check);
    if (OPEN && open) extrapolate_open<P, FORCE>(p, x == 0, u_in, g);
#pragma unroll
    for (int i = 0; i < 9; i++) {
        R v;
        put(v, g[i]);
        fout[i * plane + k] = v;
    }
}

// FP16: one row segment, V nodes a lane from x0 on (the whole warp works on the
// same row), nodes next to a solid or a wall and the first and last column left
// to the per-node path.
// DEFER: the per-node path is a later pass over those nodes (k_boundary_update);
// otherwise each thread runs it for its own nodes at the end of the segment.
// COLL: 0 = BGK, 1 = MRT (no body force, slow nodes inline).
template <int V, bool FORCE, bool LOCAL, bool OPEN, bool DEFER = false, int COLL = 0, bool BND = false>
__device__ __forceinline__ void sc_tile(const StepParams &p, const Raw<LBM_FP16_DEV>::R *__restrict__ fin,
                                        Raw<LBM_FP16_DEV>::R *__restrict__ fout, int x0, int y) {
    constexpr int P = LBM_FP16_DEV;
    using R = Raw<P>::R;
    using C = float;
    const Lattice &L = p.L;
    const int lane = threadIdx.x & 31;
    const int plane = (int)L.plane;
    const int xl = min(x0, L.pitch - V);  // in-bounds load position for every lane
    int ym = y - 1, yp = y + 1;
    if (ym < 0) ym = L.bc_y == LBM_PERIODIC ? L.ny - 1 : 0;
    if (yp >= L.ny) yp = L.bc_y == LBM_PERIODIC ? 0 : L.ny - 1;
    const int rm = ym * L.pitch, r0 = y * L.pitch, rp = yp * L.pitch;
#define SROW(i) (cy(i) == 1 ? rm : (cy(i) == -1 ? rp : r0))

    Pack<R, V> raw[9];
#pragma unroll
    for (int i = 0; i < 9; i++)
        raw[i].u = __ldg(reinterpret_cast<const typename Word<sizeof(R) * V>::T *>(
            fin + i * plane + SROW(i) + xl));
    FlagPack<V> fl;
    fl.u = *reinterpret_cast<const typename Word<2 * V>::T *>(p.flags + r0 + xl);
    // neighbour elements of the x-shifted pulls at the warp's ends; at the
    // row ends they are wrong, but those columns take the per-node path
    R hl[3] = {R(0), R(0), R(0)};
    if (lane == 0) {
        const int xh = max(x0 - 1, 0);
        hl[0] = fin[1 * plane + SROW(1) + xh];
        hl[1] = fin[5 * plane + SROW(5) + xh];
        hl[2] = fin[8 * plane + SROW(8) + xh];
    } else if (lane == 31) {
        const int xh = min(x0 + V, L.pitch - 1);
        hl[0] = fin[3 * plane + SROW(3) + xh];
        hl[1] = fin[6 * plane + SROW(6) + xh];
        hl[2] = fin[7 * plane + SROW(7) + xh];
    }
    R halo[9];
#pragma unroll
    for (int i = 0; i < 9; i++) {
        halo[i] = R(0);
        if (cx(i) == 1) halo[i] = shfl_up1(raw[i].r[V - 1]);
        else if (cx(i) == -1) halo[i] = shfl_dn1(raw[i].r[0]);
    }
#undef SROW
    if (x0 >= L.nx) return;
    if (lane == 0) {
        halo[1] = hl[0];
        halo[5] = hl[1];
        halo[8] = hl[2];
    } else if (lane == 31) {
        halo[3] = hl[0];
        halo[6] = hl[1];
        halo[7] = hl[2];
    }
#define PULL(i, j) \
    cvt(cx(i) == 0 ? raw[i].r[j] \
                   : (cx(i) == 1 ? ((j) == 0 ? halo[i] : raw[i].r[(j) - 1]) \
                                 : ((j) == V - 1 ? halo[i] : raw[i].r[(j) + 1])))
    uint32_t slow = 0;  // bit j: node j needs the per-node path
    // node j needs the per-node path, or has a non-physical state (flagged)
    auto classify = [&](int j, C r, C vx, C vy) {
        const uint16_t f = fl.f[j];
        const int x = x0 + j;
        if (!(f & 1u) && ((f & 0x1FEu) || x == 0 || x == L.nx - 1)) slow |= 1u << j;
        else if (!(f & 1u) && x < L.nx &&
                 (!(r > (C)0) || !(fabs(vx) < (C)1e30) || !(fabs(vy) < (C)1e30)))
            atomicOr(p.status, 1);
    };
    if constexpr (COLL == 1) {
        // MRT, one node at a time
        static_assert(!FORCE && !DEFER, "MRT runs without body force and with inline slow nodes");
        Pack<R, V> o[9];
#pragma unroll
        for (int j = 0; j < V; j++) {
            C g[9];
            C a = 0, jx = 0, jy = 0;
#pragma unroll
            for (int i = 0; i < 9; i++) {
                g[i] = PULL(i, j);
                a += g[i];
                jx += (C)cx(i) * g[i];
                jy += (C)cy(i) * g[i];
            }
            const C r = (C)1 + a;
            classify(j, r, jx / r, jy / r);
            collide_mrt<P>(p, g, [](C, C, C) {});
#pragma unroll
            for (int i = 0; i < 9; i++) put(o[i].r[j], (fl.f[j] & 1u) ? (C)0 : g[i]);
        }
#pragma unroll
        for (int i = 0; i < 9; i++)
            *reinterpret_cast<typename Word<sizeof(R) * V>::T *>(fout + i * plane + r0 + x0) = o[i].u;
    } else if constexpr (!FORCE) {
        // Deviation form, two nodes per instruction (FADD2 / FMUL2 / FFMA2).
        // With E_i = s0 + rho (3 e_i.u + 4.5 (e_i.u)^2 - 1.5 u.u) the
        // equilibrium deviation is w_i E_i, and BGK gives
        // (1 - omega) g_i + omega w_i E_i.  Opposite populations share
        // A = s0 - 1.5 rho u.u and the even part 4.5 rho (e.u)^2; the odd part
        // 3 rho e.u changes sign.  (bgk32x2 is exact to FP32's rounding, which the
        // storage rounds ten thousand times as much.)
        static_assert(V % 2 == 0, "two nodes at a time");
        const float om = p.omega_f;
        const float2 omc = dup2(1.f - om);
        Pack<R, V> o[9];
#pragma unroll
        for (int j = 0; j < V; j += 2) {
            float2 g[9];
#pragma unroll
            for (int i = 0; i < 9; i++) g[i] = make_float2(PULL(i, j), PULL(i, j + 1));
            const float2 s0 = add2(add2(add2(g[0], g[1]), add2(g[2], g[3])),
                                   add2(add2(g[4], g[5]), add2(add2(g[6], g[7]), g[8])));
            const float2 jx = sub2(add2(add2(g[1], g[5]), g[8]), add2(add2(g[3], g[6]), g[7]));
            const float2 jy = sub2(add2(add2(g[2], g[5]), g[6]), add2(add2(g[4], g[7]), g[8]));
            const float2 rho = add2(dup2(1.f), s0);
            const float2 inv = make_float2(1.f / rho.x, 1.f / rho.y);
            const float2 ux = mul2(jx, inv), uy = mul2(jy, inv);
            classify(j, rho.x, ux.x, uy.x);
            classify(j + 1, rho.y, ux.y, uy.y);
            const float2 A = fma2(mul2(dup2(-1.5f), rho), fma2(ux, ux, mul2(uy, uy)), s0);
            float2 out[9];
            out[0] = fma2(dup2(om * wgt<float>(0)), A, mul2(omc, g[0]));
            // (i, opp(i)) with e_i.u = eu: (1, 3) ux, (2, 4) uy, (5, 7) ux + uy, (6, 8) uy - ux
            auto pair = [&](int i, int k, float2 eu) {
                const float2 q = mul2(rho, eu);
                const float2 sym = fma2(q, mul2(dup2(4.5f), eu), A);
                const float2 ow = dup2(om * wgt<float>(i));
                out[i] = fma2(ow, fma2(dup2(3.f), q, sym), mul2(omc, g[i]));
                out[k] = fma2(ow, fma2(dup2(-3.f), q, sym), mul2(omc, g[k]));
            };
            pair(1, 3, ux);
            pair(2, 4, uy);
            pair(5, 7, add2(ux, uy));
            pair(6, 8, sub2(uy, ux));
            const bool s_a = fl.f[j] & 1u, s_b = fl.f[j + 1] & 1u;  // solid nodes store zeros
#pragma unroll
            for (int i = 0; i < 9; i++)
                put2(&o[i].r[j], s_a ? 0.f : out[i].x, s_b ? 0.f : out[i].y);
        }
#pragma unroll
        for (int i = 0; i < 9; i++)
            *reinterpret_cast<typename Word<sizeof(R) * V>::T *>(fout + i * plane + r0 + x0) = o[i].u;
    } else {
    // moments of every node from the pulled populations
    C s0[V], ux[V], uy[V], rho[V];
#pragma unroll
    for (int j = 0; j < V; j++) {
        C a = 0, jx = 0, jy = 0;
#pragma unroll
        for (int i = 0; i < 9; i++) {
            const C g = PULL(i, j);
            a += g;
            jx += (C)cx(i) * g;
            jy += (C)cy(i) * g;
        }
        const C r = (C)1 + a, inv = (C)1 / r;
        s0[j] = a;
        rho[j] = r;
        ux[j] = (jx + 0.5f * p.body_xf) * inv;
        uy[j] = (jy + 0.5f * p.body_yf) * inv;
        classify(j, r, ux[j], uy[j]);
    }
    // relax towards equilibrium, one population plane at a time
    const C om = p.omega_f;
#pragma unroll
    for (int i = 0; i < 9; i++) {
        Pack<R, V> o;
#pragma unroll
        for (int j = 0; j < V; j++) {
            const C g = PULL(i, j);
            const C eu = (C)cx(i) * ux[j] + (C)cy(i) * uy[j];
            const C uu = ux[j] * ux[j] + uy[j] * uy[j];
            const C poly = (C)3 * eu + (C)4.5 * eu * eu - (C)1.5 * uu;
            const C eq = wgt<C>(i) * (s0[j] + rho[j] * poly);
            C v = g - (g - eq) * om;
            const C Fx = p.body_xf, Fy = p.body_yf;
            v += ((C)1 - (C)0.5 * om) * wgt<C>(i) *
                 ((C)3 * (((C)cx(i) - ux[j]) * Fx + ((C)cy(i) - uy[j]) * Fy) +
                  (C)9 * eu * ((C)cx(i) * Fx + (C)cy(i) * Fy));
            put(o.r[j], (fl.f[j] & 1u) ? (C)0 : v);  // solid nodes store zeros
        }
        *reinterpret_cast<typename Word<sizeof(R) * V>::T *>(fout + i * plane + r0 + x0) = o.u;
    }
    }
#undef PULL
    // nodes next to a solid or a wall and the first/last column
    if constexpr (!DEFER) {
        while (slow) {
            const int j = __ffs(slow) - 1;
            slow &= slow - 1;
            update_node<FORCE, LOCAL, OPEN, COLL, BND>(p, fin, fout, x0 + j, y);
        }
    }
}

// FP16 open channel (bc_x = LBM_OPEN), after the fused kernel of step t has
// written the populations of t+1 into f: column x = 0 (inlet) or x = nx - 1
// (outlet) of row y takes the non-equilibrium extrapolation of its inner
// neighbour's post-collision populations (extrapolate_open); next to a solid
// neighbour the inlet takes feq(rho0, u_in) and the outlet keeps its own
// update (a resting wall beyond the edge).  open_row does both columns.
template <bool FORCE>
__device__ __forceinline__ void open_col(const StepParams &p, Raw<LBM_FP16_DEV>::R *f, int y, bool inlet) {
    constexpr int P = LBM_FP16_DEV;
    using C = float;
    const Lattice &L = p.L;
    const int plane = (int)L.plane;
    const int x = inlet ? 0 : L.nx - 1;
    const int k = y * L.pitch + x, kn = inlet ? k + 1 : k - 1;
    if (p.flags[k] & 1u) return;
    const C u_in = inlet ? inlet_ux<C>(p, y) : (C)0;
    C g[9];
    if (p.flags[kn] & 1u) {
        if (!inlet) return;
        inlet_equilibrium<P>(p, u_in, g);
    } else {
#pragma unroll
        for (int i = 0; i < 9; i++) g[i] = cvt(f[i * plane + kn]);
        extrapolate_open<P, FORCE>(p, inlet, u_in, g);
    }
#pragma unroll
    for (int i = 0; i < 9; i++) put(f[i * plane + k], g[i]);
}

template <bool FORCE>
__device__ __forceinline__ void open_row(const StepParams &p, Raw<LBM_FP16_DEV>::R *f, int y) {
    open_col<FORCE>(p, f, y, true);
    open_col<FORCE>(p, f, y, false);
}


// ------------------------------------------------ FP64 and FP32: sc_row

// BGK collision of one FP64 node, no body force.  GB300 issues about two FP64
// lanes per clock and SM, so the number of FP64 operations is the kernel's time:
// about 57 here, against about 154 with nine separate equilibria and a division
// (2048 x 1024 nodes: 246 us a step against 484).
// The even and the odd part of two opposite populations relax on their own, each by
// omega times its distance from equilibrium, so that what is rounded is small:
//   E_i = rho - 1.5 j.u + 4.5 (e_i.j)(e_i.u)   (rho u = j)
//   s = 2 w_i E_i - (f_i + f_opp),  m = 6 w_i (e_i.j) - (f_i - f_opp)
//   f_i, f_opp  +=  omega / 2 (s +- m)
// (As (1 - omega) f + omega (...) it took 60 operations, 263 us, and the error against
// 64-bit arithmetic in another order was 1.1 times that of nine equilibria, in the density
// of a channel after 100 steps up to 4.8 times: mass drifted by up to 1.2 times the
// weights' own rounding, 9 fl(1/9) - 1.)
__device__ __forceinline__ void bgk64(double om, double (&g)[9], double &rho, double &ux,
                                      double &uy) {
    const double a1 = g[1] + g[3], d1 = g[1] - g[3], a2 = g[2] + g[4], d2 = g[2] - g[4];
    const double a5 = g[5] + g[7], d5 = g[5] - g[7], a6 = g[6] + g[8], d6 = g[6] - g[8];
    rho = (g[0] + (a1 + a2)) + (a5 + a6);
    const double jx = d1 + (d5 - d6), jy = d2 + (d5 + d6);
    const double inv = reciprocal(rho);
    ux = jx * inv;
    uy = jy * inv;
    const double pxx = jx * ux, pyy = jy * uy, pxy = jx * uy, t = pxx + pyy;
    const double A = fma(-1.5, t, rho), B = fma(4.5, t, A);
    const double oh = 0.5 * om;  // uniform over the launch
    g[0] = fma(om, fma(wgt<double>(0), A, -g[0]), g[0]);
    auto pair = [&](int i, int k, double E, double ej, double a, double d) {
        const double s = fma(2.0 * wgt<double>(i), E, -a), m = fma(6.0 * wgt<double>(i), ej, -d);
        g[i] = fma(oh, s + m, g[i]);
        g[k] = fma(oh, s - m, g[k]);
    };
    pair(1, 3, fma(4.5, pxx, A), jx, a1, d1);
    pair(2, 4, fma(4.5, pyy, A), jy, a2, d2);
    pair(5, 7, fma(9.0, pxy, B), jx + jy, a5, d5);
    pair(6, 8, fma(-9.0, pxy, B), jy - jx, a6, d6);
}

// Two FP32 nodes per instruction: BGK in deviation form, j = rho u,
//   d_i  <-  d_i - omega (d_i - w_i (E_i +- 3 e_i.j))   for e_i and its opposite
//   E_i = s0 + 4.5 (e_i.j)(e_i.u) - 1.5 j.u
// Every product with a weight is inside a fused multiply-add whose result is the small
// distance from equilibrium, and the constants' own rounding is taken out of the sums that
// make up mass and momentum: the weights add up to 1 + 2^-27, which the population at rest
// gives back, and 3 w_i is 1/3 and 1/12 less one unit in the last place, 1 over e_i e_i.
// (In (1 - omega) d_i + omega w_i (...) the rounded omega w_i let mass drift by up to 7e-8
// of the deviation a step; with as many operations.)
__host__ __device__ constexpr float odd32(int i) { return i <= 4 ? 1.f / 3.f : 0x1.555554p-4f; }
static_assert((double)wgt<float>(0) + 4.0 * (double)wgt<float>(1) + 4.0 * (double)wgt<float>(5) == 1.0 + 0x1p-27, "mass");
static_assert(2.0 * (double)odd32(1) + 4.0 * (double)odd32(5) == 1.0, "momentum");
__device__ __forceinline__ void bgk32x2(float om, float2 (&g)[9], float2 &rho, float2 &ux,
                                        float2 &uy) {
    const float2 s0 = add2(add2(add2(g[0], g[1]), add2(g[2], g[3])),
                           add2(add2(g[4], g[5]), add2(add2(g[6], g[7]), g[8])));
    const float2 jx = sub2(add2(add2(g[1], g[5]), g[8]), add2(add2(g[3], g[6]), g[7]));
    const float2 jy = sub2(add2(add2(g[2], g[5]), g[6]), add2(add2(g[4], g[7]), g[8]));
    rho = add2(dup2(1.f), s0);
    const float2 inv = make_float2(1.f / rho.x, 1.f / rho.y);
    ux = mul2(jx, inv);
    uy = mul2(jy, inv);
    const float2 xx = mul2(jx, ux), yy = mul2(jy, uy), xy = mul2(jx, uy), t = add2(xx, yy);
    const float2 A = fma2(dup2(-1.5f), t, s0), B = fma2(dup2(4.5f), t, A);
    g[0] = fma2(dup2(-om), fma2(dup2(0x1p-27f), s0, fma2(dup2(-wgt<float>(0)), A, g[0])), g[0]);
    auto pair = [&](int i, int k, float2 E, float2 j) {
        const float2 w = dup2(-wgt<float>(i));
        g[i] = fma2(dup2(-om), fma2(dup2(-odd32(i)), j, fma2(w, E, g[i])), g[i]);
        g[k] = fma2(dup2(-om), fma2(dup2(odd32(i)), j, fma2(w, E, g[k])), g[k]);
    };
    pair(1, 3, fma2(dup2(4.5f), xx, A), jx);
    pair(2, 4, fma2(dup2(4.5f), yy, A), jy);
    pair(5, 7, fma2(dup2(9.f), xy, B), add2(jx, jy));
    pair(6, 8, fma2(dup2(-9.f), xy, B), sub2(jy, jx));
}

// Collision of V nodes in place; check(j, rho, ux, uy) for each of them.
template <int P, int V, bool FORCE, int COLL, class Check>
__device__ __forceinline__ void collide_nodes(const StepParams &p, typename Prec<P>::C (&g)[V][9],
                                              Check &&check) {
    using C = typename Prec<P>::C;
    if constexpr (COLL == 0 && !FORCE && P == LBM_FP32_DEV && V % 2 == 0) {
#pragma unroll
        for (int j = 0; j < V; j += 2) {
            float2 h[9], r, ux, uy;
#pragma unroll
            for (int i = 0; i < 9; i++) h[i] = make_float2(g[j][i], g[j + 1][i]);
            bgk32x2(p.omega_f, h, r, ux, uy);
            check(j, r.x, ux.x, uy.x);
            check(j + 1, r.y, ux.y, uy.y);
#pragma unroll
            for (int i = 0; i < 9; i++) {
                g[j][i] = h[i].x;
                g[j + 1][i] = h[i].y;
            }
        }
    } else {
#pragma unroll
        for (int j = 0; j < V; j++) {
            auto check_j = [&](C rho, C ux, C uy) { check(j, rho, ux, uy); };
            if constexpr (COLL == 1) {
                collide_mrt<P>(p, g[j], check_j);
            } else if constexpr (!FORCE && P == LBM_FP64) {
                C rho, ux, uy;
                bgk64(p.omega, g[j], rho, ux, uy);
                check_j(rho, ux, uy);
            } else {
                collide<P, FORCE>(p, g[j], check_j);
            }
        }
    }
}

// Update (advection, walls, collision) of the inner node (x, y) of an open
// channel, 0 < x < nx - 1, into g: for the outlet column's lane when the node
// before it belongs to another warp.  Returned populations come from the solid
// nodes' slots, as in sc_row.
template <int P, bool FORCE, int COLL>
__device__ __noinline__ void inner_update(const StepParams &p, const typename Raw<P>::R *fin, int x,
                                          int y, typename Prec<P>::C (&g)[9]) {
    using C = typename Prec<P>::C;
    const Lattice &L = p.L;
    const int plane = (int)L.plane, k = y * L.pitch + x;
    C rho_w = pick<C>(p.rho0, p.rho0_f);
    if (p.rho_w_mode == LBM_RHOW_LOCAL) {
        C s = 0;
#pragma unroll
        for (int i = 0; i < 9; i++) s += cvt(fin[i * plane + k]);
        rho_w = Prec<P>::dev ? (C)1 + s : s;
    }
#pragma unroll
    for (int i = 0; i < 9; i++) {
        const int ys = y - cy(i);
        if (ys < 0 || ys >= L.ny) {  // open channels are walled in y
            const C uw = ys < 0 ? pick<C>(p.wall_ux0, p.wall_ux0_f) : pick<C>(p.wall_ux1, p.wall_ux1_f);
            g[i] = cvt(fin[opp(i) * plane + k]) + (C)6 * wgt<C>(i) * rho_w * ((C)cx(i) * uw);
        } else {
            g[i] = cvt(fin[i * plane + ys * L.pitch + x - cx(i)]);
        }
    }
    auto unchecked = [](C, C, C) {};  // the node's own lane checks it
    if constexpr (COLL == 1) collide_mrt<P>(p, g, unchecked);
    else collide<P, FORCE>(p, g, unchecked);
}

// One row segment: nodes x0 .. x0 + V - 1 of row y in each lane, x0 = 32 V times
// the segment's index plus V times the lane (whole warps call it, with the same
// y in every lane).  fin: populations of t with the returned populations in the
// solid nodes' slots; fout: of t + 1.
//   edges  periodic: the first column's pulls from column nx - 1 come through
//          lane 0's halo load, the last column's from column 0 through one
//          predicated load in the lane that holds it;
//          walls (half-way, at rest in x): the node's own opposite populations;
//          y walls (first and last row): the same plus the moving-wall term
//          6 w_i rho_w (e_i . u_wall), over whichever is there already;
//          open columns (OPEN): the collided inner neighbour extrapolated
//          (extrapolate_open), from this lane's registers or the lane before.
template <int P, int V, bool FORCE, bool OPEN, int COLL>
__device__ __forceinline__ void sc_row(const StepParams &p, const typename Raw<P>::R *fin,
                                       typename Raw<P>::R *fout, int x0, int y) {
    using R = typename Raw<P>::R;
    using C = typename Prec<P>::C;
    using W = typename Word<sizeof(R) * V>::T;
    static_assert(P != LBM_FP16_DEV, "FP16 rounds the returned populations: sc_tile");
    const Lattice &L = p.L;
    const int lane = threadIdx.x & 31;
    const int plane = (int)L.plane;
    const int xl = min(x0, L.pitch - V);  // in-bounds load position for every lane
    const bool per_x = L.bc_x == LBM_PERIODIC;
    int ym = y - 1, yp = y + 1;
    if (ym < 0) ym = L.bc_y == LBM_PERIODIC ? L.ny - 1 : 0;
    if (yp >= L.ny) yp = L.bc_y == LBM_PERIODIC ? 0 : L.ny - 1;
    const int rm = ym * L.pitch, r0 = y * L.pitch, rp = yp * L.pitch;
#define SROW(i) (cy(i) == 1 ? rm : (cy(i) == -1 ? rp : r0))
    Pack<R, V> raw[9];
#pragma unroll
    for (int i = 0; i < 9; i++)
        raw[i].u = *reinterpret_cast<const W *>(fin + i * plane + SROW(i) + xl);
    FlagPack<V> fl;
    fl.u = *reinterpret_cast<const typename Word<2 * V>::T *>(p.flags + r0 + xl);
    R hl[3] = {R(0), R(0), R(0)};
    if (lane == 0) {
        const int xh = x0 > 0 ? min(x0, L.pitch) - 1 : (per_x ? L.nx - 1 : 0);
        hl[0] = fin[1 * plane + SROW(1) + xh];
        hl[1] = fin[5 * plane + SROW(5) + xh];
        hl[2] = fin[8 * plane + SROW(8) + xh];
    } else if (lane == 31) {
        const int xh = min(x0 + V, L.pitch - 1);
        hl[0] = fin[3 * plane + SROW(3) + xh];
        hl[1] = fin[6 * plane + SROW(6) + xh];
        hl[2] = fin[7 * plane + SROW(7) + xh];
    }
    R halo[9];
#pragma unroll
    for (int i = 0; i < 9; i++) {
        halo[i] = R(0);
        if (cx(i) == 1) halo[i] = shfl_up1(raw[i].r[V - 1]);
        else if (cx(i) == -1) halo[i] = shfl_dn1(raw[i].r[0]);
    }
    if (lane == 0) {
        halo[1] = hl[0];
        halo[5] = hl[1];
        halo[8] = hl[2];
    } else if (lane == 31) {
        halo[3] = hl[0];
        halo[6] = hl[1];
        halo[7] = hl[2];
    }
    // pulled populations of every node
    C g[V][9];
#pragma unroll
    for (int j = 0; j < V; j++)
#pragma unroll
        for (int i = 0; i < 9; i++)
            g[j][i] = cvt(cx(i) == 0 ? raw[i].r[j]
                                     : (cx(i) == 1 ? (j == 0 ? halo[i] : raw[i].r[j == 0 ? 0 : j - 1])
                                                   : (j == V - 1 ? halo[i]
                                                                 : raw[i].r[j == V - 1 ? j : j + 1])));
    const int jl = L.nx - 1 - x0;  // this lane's node in the last column, if 0 <= jl < V
    if (jl >= 0 && jl < V) {
        C e[3];
        if (per_x) {
            e[0] = cvt(fin[3 * plane + SROW(3)]);
            e[1] = cvt(fin[6 * plane + SROW(6)]);
            e[2] = cvt(fin[7 * plane + SROW(7)]);
        } else {
            const int k = r0 + L.nx - 1;
            e[0] = cvt(fin[1 * plane + k]);
            e[1] = cvt(fin[8 * plane + k]);
            e[2] = cvt(fin[5 * plane + k]);
        }
#pragma unroll
        for (int j = 0; j < V; j++)
            if (j == jl) {
                g[j][3] = e[0];
                g[j][6] = e[1];
                g[j][7] = e[2];
            }
    }
    if (x0 == 0 && !per_x) {
        g[0][1] = cvt(fin[3 * plane + r0]);
        g[0][5] = cvt(fin[7 * plane + r0]);
        g[0][8] = cvt(fin[6 * plane + r0]);
    }
#undef SROW
    if (L.bc_y == LBM_WALL && (y == 0 || y == L.ny - 1)) {
        const bool lo = y == 0;
        const C uw = lo ? pick<C>(p.wall_ux0, p.wall_ux0_f) : pick<C>(p.wall_ux1, p.wall_ux1_f);
        Pack<R, V> own[9];  // the node's own populations (rho_w = rho0 needs three of them)
#pragma unroll
        for (int i = 0; i < 9; i++) {
            own[i].u = W{};
            if (p.rho_w_mode == LBM_RHOW_LOCAL || cy(i) == (lo ? -1 : 1))
                own[i].u = *reinterpret_cast<const W *>(fin + i * plane + r0 + xl);
        }
#pragma unroll
        for (int j = 0; j < V; j++) {
            C rho_w = pick<C>(p.rho0, p.rho0_f);
            if (p.rho_w_mode == LBM_RHOW_LOCAL) {
                C s = 0;
#pragma unroll
                for (int i = 0; i < 9; i++) s += cvt(own[i].r[j]);
                rho_w = Prec<P>::dev ? (C)1 + s : s;
            }
#pragma unroll
            for (int i = 1; i < 9; i++)
                if (cy(i) != 0 && (cy(i) == 1) == lo)
                    g[j][i] = cvt(own[opp(i)].r[j]) + (C)6 * wgt<C>(i) * rho_w * ((C)cx(i) * uw);
        }
    }
    collide_nodes<P, V, FORCE, COLL>(p, g, [&](int j, C r, C vx, C vy) {
        if (!(fl.f[j] & 1u) && x0 + j < L.nx && unphysical(r, vx, vy)) atomicOr(p.status, 1);
    });
    if constexpr (OPEN) {
        // whole warps, uniform branches: the collided inner neighbour of column 0 is
        // node 1 (this lane, or the next with one node per lane), of column nx - 1
        // node nx - 2 (this lane, the lane before, or the warp before: recomputed)
        const bool first = x0 == 0, last = jl >= 0 && jl < V;
        if (__any_sync(0xffffffffu, first)) {
            C n[9];
            uint16_t fn = 1u;
            if constexpr (V > 1) {
#pragma unroll
                for (int i = 0; i < 9; i++) n[i] = g[1][i];
                fn = fl.f[1];
            } else {
#pragma unroll
                for (int i = 0; i < 9; i++) n[i] = __shfl_down_sync(0xffffffffu, g[0][i], 1);
                fn = (uint16_t)__shfl_down_sync(0xffffffffu, (int)fl.f[0], 1);
            }
            if (first) {
                const C u_in = inlet_ux<C>(p, y);
                if (fn & 1u) inlet_equilibrium<P>(p, u_in, n);
                else extrapolate_open<P, FORCE>(p, true, u_in, n);
#pragma unroll
                for (int i = 0; i < 9; i++) g[0][i] = n[i];
            }
        }
        if (__any_sync(0xffffffffu, last)) {
            C n[9];
            uint16_t fn;
#pragma unroll
            for (int i = 0; i < 9; i++) n[i] = __shfl_up_sync(0xffffffffu, g[V - 1][i], 1);
            fn = (uint16_t)__shfl_up_sync(0xffffffffu, (int)fl.f[V - 1], 1);
            if (last) {
                if (jl > 0) {
#pragma unroll
                    for (int j = 1; j < V; j++)
                        if (j == jl) {
#pragma unroll
                            for (int i = 0; i < 9; i++) n[i] = g[j - 1][i];
                            fn = fl.f[j - 1];
                        }
                } else if (lane == 0) {
                    fn = p.flags[r0 + L.nx - 2];
                    if (!(fn & 1u)) inner_update<P, FORCE, COLL>(p, fin, L.nx - 2, y, n);
                }
                if (!(fn & 1u)) {
                    extrapolate_open<P, FORCE>(p, false, (C)0, n);
#pragma unroll
                    for (int j = 0; j < V; j++)
                        if (j == jl) {
#pragma unroll
                            for (int i = 0; i < 9; i++) g[j][i] = n[i];
                        }
                }
            }
        }
    }
    if (x0 >= L.nx) return;
#pragma unroll
    for (int i = 0; i < 9; i++) {
        Pack<R, V> o;
#pragma unroll
        for (int j = 0; j < V; j++) put(o.r[j], (fl.f[j] & 1u) ? (C)0 : g[j][i]);
        *reinterpret_cast<W *>(fout + i * plane + r0 + x0) = o.u;
    }
}

}  // namespace

}  // namespace gbm
