// The FP64 T2S2-FDLBM1 step in two launches per step, one node per thread, for any
// boundary combination: each quantity of Sec. 2D is formed once per node, with
// no halo recomputed.
//
//   k_split_prepare  first launch of a call: f~ -> P = fbar^{+,h} (Eqs. 2.19,
//                    2.34), written over f~, and Q = f~+ (Eq. 2.20)
//   k_split_star     P -> S = f* (Eqs. 2.32-2.35; Eq. 3.10 at wall nodes)
//   k_split_update   Q, S -> f~ of the next step (Eq. 2.23; Eq. 3.10 at wall
//                    nodes) and, in registers, its P and Q; the last step of a
//                    call stores f~ instead
//
// A wall node's thread works at its nearest interior node x_j and extrapolates
// from there, so that walls need no launch of their own; it reads Q of another
// node, so on walled grids Q alternates between two buffers.
//
// The difference weights come from tables with the metric, the time step and
// the sign folded in (split_tables.h): one multiply-add per tap, and next to
// a wall, where the second-order upwind tap would leave the domain, the entry
// of that sign holds the central difference.  The weights of each axis sum to
// exactly zero, and stay so in the kernels: the centre weights of a diagonal are
// added into one only where that sum is exact (MERGE: uniform periodic grids).
//
// What bounds it: the FP64 units, 227 FP64 instructions per node (prepare
// 79, star 104, update 44): 1024^2 periodic 431 us per step, 0.87 of the rate at
// which a warp's FP64 instruction takes 64 cycles of its scheduler; the 576
// bytes per node that pass between the launches are hidden behind them.  The
// sweep it replaced there recomputed 8 halo rows and columns per tile and spent
// 239 instructions per node: 718 us.  Small grids wait for launches and for one
// warp's chain of instructions: 64^2 7.1 us per step (sweep 59.6), 257^2 cavity
// 34.6 (five staged launches with a thread per wall node 81).
#include <algorithm>
#include <cmath>
#include <type_traits>
#include <vector>

#include "chain.cuh"
#include "internal.h"
#include "split_tables.h"
#include "walls_nodes.cuh"

namespace fdlbm {
namespace {

// Threads per block: one warp.  A warp's FP64 instruction holds its
// scheduler's FP64 unit for 64 cycles, so a launch lasts as long as the
// scheduler with the most warps; single warps spread most evenly (257^2 cavity:
// 35.1 us per step, 45.5 in blocks of 128, 1024^2: the same either way).
constexpr int kThreads = 32;

// The launches of a call are chained (chain.cuh).  Letting the next one's blocks
// in at the start of the kernel instead of after a warp's arithmetic made them
// take SM slots unevenly (257^2 periodic FP64: 51.6 us per step against 31.4;
// without the chain attribute 35.2).

template <class R>
struct SplitArgs {
    R *P, *S;                // [9][ny][pitch]; S: planes 1 to 8 (population 0 does not move)
    const R *Qin;            // f~+ of this step
    R *Qout;                 // f~+ of the next step (k_split_update), or f~ (its last launch)
    const R *force;
    const R *tx, *ty;        // weight tables of the stage: [n][2][4] (sign +, sign -)
    int nx, ny, pitch;
    size_t plane;
    int wx, wy;
    int x0, y0, w, h;        // rectangle of the launch: all nodes, or the interior ones
    int strip, strip_blocks; // strip width (threads run along rows of a strip), blocks per strip
    int wall_blocks;         // leading blocks that take the wall nodes
    R wall_u[4][2];
    Coeffs<R> c;
    R keep_star, w_star[3], l_star[2];  // (1 - b*)/2, b* w_i, b* c_i of the linear terms
};

template <class R>
struct Taps {
    R m1, c, p1, p2;         // at k + s, k, k - s, k - 2s for velocity sign s
};

template <class R>
__device__ __forceinline__ Taps<R> load_taps(const R *t)
{
    const double2 u = __ldg(reinterpret_cast<const double2 *>(t));
    const double2 v = __ldg(reinterpret_cast<const double2 *>(t) + 1);
    return {u.x, u.y, v.x, v.y};
}

// A node, its neighbours (wrapped on a periodic axis; on a walled axis clamped,
// where the weights are zero) and the weights of its differences.
template <class R, bool WALLS, bool MERGE>
struct Site {
    int x[5], y[5];          // k - 2 .. k + 2
    Taps<R> xp, xn, yp, yn;  // weights for the signs of each axis

    __device__ __forceinline__ void set(const SplitArgs<R> &a, int xc, int yc)
    {
#pragma unroll
        for (int d = -2; d <= 2; ++d) {
            int u = xc + d, v = yc + d;
            if (WALLS && a.wx) u = min(max(u, 0), a.nx - 1);
            else u = u < 0 ? u + a.nx : (u >= a.nx ? u - a.nx : u);
            if (WALLS && a.wy) v = min(max(v, 0), a.ny - 1);
            else v = v < 0 ? v + a.ny : (v >= a.ny ? v - a.ny : v);
            x[d + 2] = u;
            y[d + 2] = v * a.pitch;
        }
        xp = load_taps(a.tx + 8 * xc);
        yp = load_taps(a.ty + 8 * yc);
        xn = WALLS ? load_taps(a.tx + 8 * xc + 4) : xp;
        yn = WALLS ? load_taps(a.ty + 8 * yc + 4) : yp;
    }

    // acc plus the weighted taps of population i of plane f around the node
    __device__ __forceinline__ R advance(const R *f, int i, R v0, R acc) const
    {
        const int r0 = y[2];
        if (MERGE && cx(i) != 0 && cy(i) != 0) acc = fma(xp.c + yp.c, v0, acc);
        else {
            if (cx(i) != 0) acc = fma(cx(i) > 0 ? xp.c : xn.c, v0, acc);
            if (cy(i) != 0) acc = fma(cy(i) > 0 ? yp.c : yn.c, v0, acc);
        }
        if (cx(i) != 0) {
            const Taps<R> &w = cx(i) > 0 ? xp : xn;
            const int s = cx(i);
            acc = fma(w.m1, f[r0 + x[2 + s]], acc);
            acc = fma(w.p1, f[r0 + x[2 - s]], acc);
            acc = fma(w.p2, f[r0 + x[2 - 2 * s]], acc);
        }
        if (cy(i) != 0) {
            const Taps<R> &w = cy(i) > 0 ? yp : yn;
            const int s = cy(i);
            acc = fma(w.m1, f[y[2 + s] + x[2]], acc);
            acc = fma(w.p1, f[y[2 - s] + x[2]], acc);
            acc = fma(w.p2, f[y[2 - 2 * s] + x[2]], acc);
        }
        return acc;
    }
};

// Node coordinates of this thread.  Wall nodes come first, in blocks of their
// own (a warp that holds both kinds would run Eq. 3.10 for its interior lanes
// too); then the rectangle, linear over strips of `strip` columns, so that
// every warp is full on any width.  LANES threads share a node.  False past the
// end.
template <class R, bool WALLS, int LANES = 1>
__device__ __forceinline__ bool my_node(const SplitArgs<R> &a, int &x, int &y)
{
    const int per_block = blockDim.x / LANES, t = threadIdx.x / LANES;
    if (WALLS && blockIdx.x < a.wall_blocks) {
        const int k = blockIdx.x * per_block + t;
        const int rows = a.wy ? 2 * a.nx : 0;  // S and N rows, corners included
        if (k < rows) {
            x = k < a.nx ? k : k - a.nx;
            y = k < a.nx ? 0 : a.ny - 1;
            return true;
        }
        const int len = a.wy ? a.ny - 2 : a.ny, m = k - rows;  // W and E columns
        x = m < len ? 0 : a.nx - 1;
        y = (m < len ? m : m - len) + (a.wy ? 1 : 0);
        return a.wx && m < 2 * len;
    }
    const int b = blockIdx.x - (WALLS ? a.wall_blocks : 0);
    const int strip = b / a.strip_blocks;
    const unsigned k = (b - strip * a.strip_blocks) * per_block + t;
    const int xs = strip * a.strip;
    const unsigned w = min(a.strip, a.w - xs);
    const unsigned row = k / w;
    x = a.x0 + xs + (int)(k - row * w);
    y = a.y0 + (int)row;
    return row < (unsigned)a.h;
}

// The wall that owns node (x, y) and its interior neighbour x_j along the
// inward normal (diagonal at corners; the W/E walls own the corners); -1 at an
// interior node, whose x_j is itself.
template <class R>
__device__ __forceinline__ int wall_side(const SplitArgs<R> &a, int x, int y, int &jx, int &jy)
{
    jx = a.wx ? min(max(x, 1), a.nx - 2) : x;
    jy = a.wy ? min(max(y, 1), a.ny - 2) : y;
    if (jx != x) return x == 0 ? FDLBM_WALL_W : FDLBM_WALL_E;
    if (jy != y) return y == 0 ? FDLBM_WALL_S : FDLBM_WALL_N;
    return -1;
}

template <class R>
__device__ __forceinline__ void wall_velocity(const SplitArgs<R> &a, int side, R &u, R &v)
{
    u = v = R(0);
#pragma unroll
    for (int s = 0; s < 4; ++s)
        if (s == side) {
            u = a.wall_u[s][0];
            v = a.wall_u[s][1];
        }
}

// Sums and differences of opposite populations, and the moments from them:
// pairs (1,3), (2,4), (5,7), (6,8).
template <class R>
struct Node {
    R s[4], d[4], drho, jx, jy, inv, base, h45, e[4];

    __device__ __forceinline__ void moments(const R g[9])
    {
        const int a[4] = {1, 2, 5, 6}, b[4] = {3, 4, 7, 8};
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            s[k] = g[a[k]] + g[b[k]];
            d[k] = g[a[k]] - g[b[k]];
        }
        drho = g[0] + ((s[0] + s[1]) + (s[2] + s[3]));
        jx = d[0] + (d[2] - d[3]);
        jy = d[1] + (d[2] + d[3]);
    }
    // Eq. 3.2 in pairs: f^eq - w rho0 = w t +- c e with t = drho + (4.5 e^2 -
    // 1.5 j.j)/rho (see equilibrium_dev_j); t of the rest population is base
    __device__ __forceinline__ void equilibrium(const Coeffs<R> &c)
    {
        inv = node_reciprocal(macro_density(c, drho));
        const R q = jx * jx + jy * jy;
        h45 = R(4.5) * inv;
        base = fma(q, R(-1.5) * inv, drho);
        e[0] = jx;
        e[1] = jy;
        e[2] = jx + jy;
        e[3] = jy - jx;
    }
    __device__ __forceinline__ R t(int k) const { return fma(e[k] * e[k], h45, base); }
    __device__ __forceinline__ static R w(int k) { return k < 2 ? wq<R>(1) : wq<R>(5); }
    __device__ __forceinline__ static R lin(int k) { return k < 2 ? LinearCoef<R>::c1 : LinearCoef<R>::c2; }
};

// P and Q of one node from its f~ (g): g + b (f^eq - g) + c F.
template <class R, bool FORCE>
__device__ __forceinline__ void prepare(const SplitArgs<R> &a, const R g[9], R Fx, R Fy, R P[9], R Q[9])
{
    const Coeffs<R> &c = a.c;
    if constexpr (FORCE) {
        R drho, rho, ux, uy, geq[9], F[9];
        node_eq<R, true>(c, g, Fx, Fy, c.half_dt, drho, rho, ux, uy, geq);
        force_terms(c.rho0, geq, ux, uy, Fx, Fy, F, force_dshift(c, drho));
#pragma unroll
        for (int i = 0; i < 9; ++i) {
            const R neq = geq[i] - g[i];
            P[i] = g[i] + c.b_bar * neq + c.c_bar * F[i];
            Q[i] = g[i] + c.b_til * neq + c.c_til * F[i];
        }
    } else {
        Node<R> n;
        n.moments(g);
        n.equilibrium(c);
        const R neq0 = fma(wq<R>(0), n.base, -g[0]);
        P[0] = fma(c.b_bar, neq0, g[0]);
        Q[0] = fma(c.b_til, neq0, g[0]);
        const int ia[4] = {1, 2, 5, 6}, ib[4] = {3, 4, 7, 8};
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            // halving is exact, so each difference is rounded once; a product lin e
            // rounded by itself was off alike at every step of a nearly uniform flow
            // (192^2 Taylor vortex in a mean flow, 1000 steps, against 80-bit
            // arithmetic: momentum 8.4e-15 off, 3.7e-16 so, the sweep 7.1e-16)
            const R sym = fma(n.w(k), n.t(k), R(-0.5) * n.s[k]);
            const R asym = fma(n.lin(k), n.e[k], R(-0.5) * n.d[k]);
            const R na = sym + asym, nb = sym - asym;
            P[ia[k]] = fma(c.b_bar, na, g[ia[k]]);
            P[ib[k]] = fma(c.b_bar, nb, g[ib[k]]);
            Q[ia[k]] = fma(c.b_til, na, g[ia[k]]);
            Q[ib[k]] = fma(c.b_til, nb, g[ib[k]]);
        }
    }
}

// f* of populations 1 to 8 (and 0 if REST) from fbar* (gs): gs + b* (f^eq - gs) + c* F.
template <class R, bool FORCE, bool REST>
__device__ __forceinline__ void relax_star(const SplitArgs<R> &a, const R gs[9], R Fx, R Fy, R st[9])
{
    const Coeffs<R> &c = a.c;
    if constexpr (FORCE) {
        R drho, rho, ux, uy, geq[9], F[9];
        node_eq<R, true>(c, gs, Fx, Fy, c.half_h, drho, rho, ux, uy, geq);
        force_terms(c.rho0, geq, ux, uy, Fx, Fy, F, force_dshift(c, drho));
#pragma unroll
        for (int i = REST ? 0 : 1; i < 9; ++i) st[i] = gs[i] + c.b_star * (geq[i] - gs[i]) + c.c_star * F[i];
    } else {
        Node<R> n;
        n.moments(gs);
        n.equilibrium(c);
        if (REST) st[0] = fma(a.w_star[0], n.base, (a.keep_star + a.keep_star) * gs[0]);
        const int ia[4] = {1, 2, 5, 6}, ib[4] = {3, 4, 7, 8};
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const R sym = fma(a.keep_star, n.s[k], a.w_star[k < 2 ? 1 : 2] * n.t(k));
            const R asym = fma(a.keep_star, n.d[k], a.l_star[k < 2 ? 0 : 1] * n.e[k]);
            st[ia[k]] = sym + asym;
            st[ib[k]] = sym - asym;
        }
    }
}

template <class R, bool FORCE>
__device__ __forceinline__ void load_force(const SplitArgs<R> &a, int x, int y, R &Fx, R &Fy)
{
    Fx = Fy = R(0);
    if (FORCE) {
        const size_t o = (size_t)y * a.pitch + x;
        Fx = __ldg(a.force + o);
        Fy = __ldg(a.force + a.plane + o);
    }
}

// Four threads per node, for grids and wall nodes that leave schedulers idle: a
// node's chain of FP64 instructions (48 in the star kernel, 55 in the update,
// against 104 and 123) is what such a launch waits for.  Thread q of a node takes
// the axis velocity 1 + q and the diagonal one 5 + q, whose differences run along
// the same half axes; the moments are summed over the four by shuffles, and the
// rest population is everybody's.  Every thread of the warp takes part in the
// shuffles: those past the last node work on a copy of the first.  (129^2 cavity,
// whose wall nodes alone are split: 20.9 -> 14.2 us per step; 64^2 periodic 11.6 ->
// 7.1.)
template <class R, bool FORCE, bool MERGE>
struct Quad {
    const SplitArgs<R> &a;
    const int q;
    const R ax, ay, dx, dy;  // velocities
    Taps<R> wx, wy;
    R wxy;                   // MERGE: the centre weight of the diagonal population
    int o0, x[3], y[3];      // offsets at k, and at k + s, k - s, k - 2s in x and in y
    R drho, jx, jy, rm, inv, h45, base;

    __device__ __forceinline__ explicit Quad(const SplitArgs<R> &a_)
        : a(a_), q(threadIdx.x & 3), ax(R(q == 0) - R(q == 2)), ay(R(q == 1) - R(q == 3)),
          dx(q == 0 || q == 3 ? R(1) : R(-1)), dy(q < 2 ? R(1) : R(-1))
    {
    }

    __device__ __forceinline__ static int index(int k, int n, bool wall)
    {
        return wall ? min(max(k, 0), n - 1) : k < 0 ? k + n : (k >= n ? k - n : k);
    }

    __device__ __forceinline__ void set(int xc, int yc)
    {
        const int sx = q == 0 || q == 3 ? 1 : -1, sy = q < 2 ? 1 : -1;
        const int at[3] = {1, -1, -2};
        const int row = yc * a.pitch;
        o0 = row + xc;
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            x[k] = row + index(xc + at[k] * sx, a.nx, a.wx);
            y[k] = index(yc + at[k] * sy, a.ny, a.wy) * a.pitch + xc;
        }
        wx = load_taps(a.tx + 8 * xc + (sx > 0 ? 0 : 4));
        wy = load_taps(a.ty + 8 * yc + (sy > 0 ? 0 : 4));
        if (MERGE) wxy = wx.c + wy.c;
    }

    // acc plus the weighted taps of the axis and of the diagonal population
    __device__ __forceinline__ R axis(const R *f, R acc) const
    {
        const bool h = !(q & 1);
        acc = fma(h ? wx.c : wy.c, f[o0], acc);
        acc = fma(h ? wx.m1 : wy.m1, f[h ? x[0] : y[0]], acc);
        acc = fma(h ? wx.p1 : wy.p1, f[h ? x[1] : y[1]], acc);
        return fma(h ? wx.p2 : wy.p2, f[h ? x[2] : y[2]], acc);
    }
    __device__ __forceinline__ R diagonal(const R *f, R acc) const
    {
        const R v0 = f[o0];
        if (MERGE) acc = fma(wxy, v0, acc);
        else acc = fma(wy.c, v0, fma(wx.c, v0, acc));
        acc = fma(wx.m1, f[x[0]], acc);
        acc = fma(wy.m1, f[y[0]], acc);
        acc = fma(wx.p1, f[x[1]], acc);
        acc = fma(wy.p1, f[y[1]], acc);
        acc = fma(wx.p2, f[x[2]], acc);
        return fma(wy.p2, f[y[2]], acc);
    }

    __device__ __forceinline__ static R sum4(R v)
    {
        v += __shfl_xor_sync(0xffffffffu, v, 1);
        return v + __shfl_xor_sync(0xffffffffu, v, 2);
    }

    // Eq. 3.3 (force shift `shift`) and the common terms of Eq. 3.2
    __device__ __forceinline__ void macro(R g0, R ga, R gd, R Fx, R Fy, R shift)
    {
        drho = sum4(ga + gd) + g0;
        jx = sum4(fma(dx, gd, ax * ga));
        jy = sum4(fma(dy, gd, ay * ga));
        rm = macro_density(a.c, drho);
        if (FORCE) {
            jx += shift * rm * Fx;
            jy += shift * rm * Fy;
        }
        inv = node_reciprocal(rm);
        const R jj = jx * jx + jy * jy;
        h45 = R(4.5) * inv;
        base = fma(jj, R(-1.5) * inv, drho);
    }
    __device__ __forceinline__ void equilibrium(R &e0, R &ea, R &ed) const
    {
        const R ja = fma(ax, jx, ay * jy), jd = fma(dx, jx, dy * jy);
        e0 = wq<R>(0) * base;
        ea = fma(LinearCoef<R>::c1, ja, wq<R>(1) * fma(ja * ja, h45, base));
        ed = fma(LinearCoef<R>::c2, jd, wq<R>(5) * fma(jd * jd, h45, base));
    }
    // Eq. 3.12 at the equilibrium (e0, ea, ed)
    __device__ __forceinline__ void force_term(R e0, R ea, R ed, R Fx, R Fy, R &f0, R &fa, R &fd) const
    {
        const R nuF = -(jx * Fx + jy * Fy) * inv, r0 = a.c.rho0 - force_dshift(a.c, drho);
        f0 = R(3) * nuF * fma(wq<R>(0), r0, e0);
        fa = R(3) * (nuF + fma(ax, Fx, ay * Fy)) * fma(wq<R>(1), r0, ea);
        fd = R(3) * (nuF + fma(dx, Fx, dy * Fy)) * fma(wq<R>(5), r0, ed);
    }
    // Eq. 3.10 from x_j's values
    __device__ __forceinline__ void extrapolate(int side, R Fx, R Fy, R shift, R &g0, R &ga, R &gd)
    {
        R u, v, e0, ea, ed;
        wall_velocity(a, side, u, v);
        macro(g0, ga, gd, Fx, Fy, shift);
        equilibrium(e0, ea, ed);
        const R ua = fma(ax, u, ay * v), ud = fma(dx, u, dy * v), uu = R(1.5) * (u * u + v * v);
        g0 = wq<R>(0) * (drho - rm * uu) + (g0 - e0);
        ga = wq<R>(1) * (drho + rm * (ua * (R(3) + R(4.5) * ua) - uu)) + (ga - ea);
        gd = wq<R>(5) * (drho + rm * (ud * (R(3) + R(4.5) * ud) - uu)) + (gd - ed);
    }
};

template <class R, bool FORCE, bool WALLS, bool MERGE>
__device__ __forceinline__ void star_quad(const SplitArgs<R> &a)
{
    int x, y;
    const bool valid = my_node<R, WALLS, 4>(a, x, y);
    const bool walls = WALLS && blockIdx.x < a.wall_blocks;
    if (!valid) {
        x = walls ? 0 : a.x0;
        y = walls ? 0 : a.y0;
    }
    int jx = x, jy = y, side = -1;
    if (WALLS) side = wall_side(a, x, y, jx, jy);  // a wall for the whole block, or for none of it
    Quad<R, FORCE, MERGE> n(a);
    n.set(jx, jy);
    R Fx, Fy;
    load_force<R, FORCE>(a, jx, jy, Fx, Fy);
    chain_wait();
    const size_t pa = (1 + n.q) * a.plane, pd = (5 + n.q) * a.plane;
    R g0 = a.P[n.o0], ga = n.axis(a.P + pa, a.P[pa + n.o0]), gd = n.diagonal(a.P + pd, a.P[pd + n.o0]);
    n.macro(g0, ga, gd, Fx, Fy, a.c.half_h);
    R e0, ea, ed;
    n.equilibrium(e0, ea, ed);
    const R b = a.c.b_star;
    g0 = fma(b, e0 - g0, g0);
    ga = fma(b, ea - ga, ga);
    gd = fma(b, ed - gd, gd);
    if (FORCE) {
        R f0, fa, fd;
        n.force_term(e0, ea, ed, Fx, Fy, f0, fa, fd);
        g0 = fma(a.c.c_star, f0, g0);
        ga = fma(a.c.c_star, fa, ga);
        gd = fma(a.c.c_star, fd, gd);
    }
    if (WALLS && walls) n.extrapolate(side, R(0), R(0), R(0), g0, ga, gd);
    chain_next();
    if (!valid) return;
    const size_t o = (size_t)y * a.pitch + x;
    a.S[pa + o] = ga;
    a.S[pd + o] = gd;
}

// P and Q of node o from its f~, four threads per node.  The first launch of a call
// and the update both come here (and to prepare), so that a state does not depend
// on how its steps are divided into calls.
template <class R, bool FORCE, bool MERGE>
__device__ __forceinline__ void prepare_quad(const SplitArgs<R> &a, Quad<R, FORCE, MERGE> &n, size_t o, bool valid, R g0,
                                             R ga, R gd, R Fx, R Fy)
{
    const size_t pa = (1 + n.q) * a.plane, pd = (5 + n.q) * a.plane;
    n.macro(g0, ga, gd, Fx, Fy, a.c.half_dt);
    R e0, ea, ed, f0 = R(0), fa = R(0), fd = R(0);
    n.equilibrium(e0, ea, ed);
    if (FORCE) n.force_term(e0, ea, ed, Fx, Fy, f0, fa, fd);
    auto relax = [&](R g, R e, R f, R &P, R &Q) {
        const R neq = e - g;
        P = fma(a.c.b_bar, neq, g);
        Q = fma(a.c.b_til, neq, g);
        if (FORCE) {
            P = fma(a.c.c_bar, f, P);
            Q = fma(a.c.c_til, f, Q);
        }
    };
    R P0, Q0, Pa, Qa, Pd, Qd;
    relax(g0, e0, f0, P0, Q0);
    relax(ga, ea, fa, Pa, Qa);
    relax(gd, ed, fd, Pd, Qd);
    // P lies over f~, and on a periodic grid Qout is Qin: all four threads have read
    // the rest population that one of them now writes (a shuffle orders no memory)
    __syncwarp();
    chain_next();
    if (!valid) return;
    if (n.q == 0) {
        a.P[o] = P0;
        a.Qout[o] = Q0;
    }
    a.P[pa + o] = Pa;
    a.P[pd + o] = Pd;
    a.Qout[pa + o] = Qa;
    a.Qout[pd + o] = Qd;
}

template <class R, bool FORCE, bool WALLS, bool MERGE, bool LAST>
__device__ __forceinline__ void update_quad(const SplitArgs<R> &a)
{
    int x, y;
    const bool valid = my_node<R, WALLS, 4>(a, x, y);
    const bool walls = WALLS && blockIdx.x < a.wall_blocks;
    if (!valid) {
        x = walls ? 0 : a.x0;
        y = walls ? 0 : a.y0;
    }
    int jx = x, jy = y, side = -1;
    if (WALLS) side = wall_side(a, x, y, jx, jy);
    Quad<R, FORCE, MERGE> n(a);
    n.set(jx, jy);
    chain_wait();
    const size_t pa = (1 + n.q) * a.plane, pd = (5 + n.q) * a.plane;
    R g0 = a.Qin[n.o0], ga = n.axis(a.S + pa, a.Qin[pa + n.o0]), gd = n.diagonal(a.S + pd, a.Qin[pd + n.o0]);
    R Fx, Fy;
    if (WALLS && walls) {
        load_force<R, FORCE>(a, jx, jy, Fx, Fy);
        n.extrapolate(side, Fx, Fy, a.c.half_dt, g0, ga, gd);
    }
    const size_t o = (size_t)y * a.pitch + x;
    if (LAST) {
        if (!valid) return;
        if (n.q == 0) a.Qout[o] = g0;
        a.Qout[pa + o] = ga;
        a.Qout[pd + o] = gd;
        return;
    }
    load_force<R, FORCE>(a, x, y, Fx, Fy);
    prepare_quad<R, FORCE, MERGE>(a, n, o, valid, g0, ga, gd, Fx, Fy);
}

// QUAD, here and below: four threads per node for every node; else for the wall
// nodes.
template <class R, bool FORCE, bool WALLS, bool QUAD>
__global__ void __launch_bounds__(kThreads) k_split_prepare(const SplitArgs<R> a)
{
    int x, y;
    R Fx, Fy;
    if (QUAD || (WALLS && blockIdx.x < a.wall_blocks)) {
        const bool valid = my_node<R, WALLS, 4>(a, x, y);
        if (!valid) x = y = 0;
        const size_t o = (size_t)y * a.pitch + x;
        Quad<R, FORCE, false> n(a);
        load_force<R, FORCE>(a, x, y, Fx, Fy);
        prepare_quad<R, FORCE, false>(a, n, o, valid, a.P[o], a.P[(1 + n.q) * a.plane + o],
                                      a.P[(5 + n.q) * a.plane + o], Fx, Fy);
        return;
    }
    if (!my_node<R, WALLS>(a, x, y)) return;
    const size_t o = (size_t)y * a.pitch + x;
    R g[9], P[9], Q[9];
#pragma unroll
    for (int i = 0; i < 9; ++i) g[i] = a.P[i * a.plane + o];
    load_force<R, FORCE>(a, x, y, Fx, Fy);
    prepare<R, FORCE>(a, g, Fx, Fy, P, Q);
    chain_next();
#pragma unroll
    for (int i = 0; i < 9; ++i) {
        a.P[i * a.plane + o] = P[i];
        a.Qout[i * a.plane + o] = Q[i];
    }
}

template <class R, bool FORCE, bool WALLS, bool QUAD, bool MERGE>
__global__ void __launch_bounds__(kThreads) k_split_star(const SplitArgs<R> a)
{
    if (QUAD || (WALLS && blockIdx.x < a.wall_blocks)) {
        star_quad<R, FORCE, WALLS, MERGE>(a);
        return;
    }
    int x, y;
    if (!my_node<R, WALLS>(a, x, y)) return;
    int jx = x, jy = y, side = -1;
    if (WALLS) side = wall_side(a, x, y, jx, jy);
    Site<R, WALLS, MERGE> n;
    n.set(a, jx, jy);
    R Fx, Fy;
    load_force<R, FORCE>(a, jx, jy, Fx, Fy);
    chain_wait();
    R gs[9], st[9];
#pragma unroll
    for (int i = 0; i < 9; ++i) {
        const R *f = a.P + i * a.plane;
        const R v0 = f[n.y[2] + n.x[2]];
        gs[i] = i == 0 ? v0 : n.advance(f, i, v0, v0);
    }
    relax_star<R, FORCE, WALLS>(a, gs, Fx, Fy, st);
    if (WALLS && side >= 0) {  // Eq. 3.10 for f* (no force shift)
        R u, v, wv[9];
        wall_velocity(a, side, u, v);
        nee<R, false>(a.c, st, R(0), R(0), R(0), u, v, wv);
#pragma unroll
        for (int i = 1; i < 9; ++i) st[i] = wv[i];
    }
    chain_next();
    const size_t o = (size_t)y * a.pitch + x;
#pragma unroll
    for (int i = 1; i < 9; ++i) a.S[i * a.plane + o] = st[i];
}

template <class R, bool FORCE, bool WALLS, bool QUAD, bool MERGE, bool LAST>
__global__ void __launch_bounds__(kThreads) k_split_update(const SplitArgs<R> a)
{
    if (QUAD || (WALLS && blockIdx.x < a.wall_blocks)) {
        update_quad<R, FORCE, WALLS, MERGE, LAST>(a);
        return;
    }
    int x, y;
    if (!my_node<R, WALLS>(a, x, y)) return;
    int jx = x, jy = y, side = -1;
    if (WALLS) side = wall_side(a, x, y, jx, jy);
    Site<R, WALLS, MERGE> n;
    n.set(a, jx, jy);
    chain_wait();
    R g[9];
#pragma unroll
    for (int i = 0; i < 9; ++i) {
        const int o0 = n.y[2] + n.x[2];
        const R q = a.Qin[i * a.plane + o0];
        const R *f = a.S + i * a.plane;
        g[i] = i == 0 ? q : n.advance(f, i, f[o0], q);
    }
    R Fx, Fy;
    if (WALLS && side >= 0) {  // Eq. 3.10 for the new f~ (force shift dt/2)
        R u, v, wv[9];
        wall_velocity(a, side, u, v);
        load_force<R, FORCE>(a, jx, jy, Fx, Fy);
        nee<R, FORCE>(a.c, g, Fx, Fy, a.c.half_dt, u, v, wv);
#pragma unroll
        for (int i = 0; i < 9; ++i) g[i] = wv[i];
    }
    const size_t o = (size_t)y * a.pitch + x;
    if (LAST) {
#pragma unroll
        for (int i = 0; i < 9; ++i) a.Qout[i * a.plane + o] = g[i];
        return;
    }
    load_force<R, FORCE>(a, x, y, Fx, Fy);
    R P[9], Q[9];
    prepare<R, FORCE>(a, g, Fx, Fy, P, Q);
    chain_next();
#pragma unroll
    for (int i = 0; i < 9; ++i) {
        a.P[i * a.plane + o] = P[i];
        a.Qout[i * a.plane + o] = Q[i];
    }
}

// One launch over all nodes; split_walls: the wall nodes in blocks of their
// own.  lanes: threads per node (1 or 4).  chained: scheduled while the previous launch of the chain still runs.
template <class R, class K>
cudaError_t launch(K kernel, SplitArgs<R> a, int lanes, bool split_walls, bool chained, cudaStream_t s)
{
    constexpr int nt = kThreads;
    const int nodes = nt / lanes, wall_nodes = nt / 4;  // per block
    const int wx = split_walls && a.wx, wy = split_walls && a.wy;
    a.x0 = wx;
    a.y0 = wy;
    a.w = a.nx - 2 * wx;
    a.h = a.ny - 2 * wy;
    const int strips = (a.w + 63) / 64;
    a.strip = (a.w + strips - 1) / strips;
    a.strip_blocks = (int)(((long long)a.strip * a.h + nodes - 1) / nodes);
    const long long walls = (wy ? 2ll * a.nx : 0) + (wx ? 2ll * a.h : 0);
    a.wall_blocks = (int)((walls + wall_nodes - 1) / wall_nodes);
    const dim3 grid((unsigned)(a.wall_blocks + a.strip_blocks * ((a.w + a.strip - 1) / a.strip)));
    if (chained) return chained_launch(kernel, grid, nt, 0, s, a);
    kernel<<<grid, nt, 0, s>>>(a);
    return cudaGetLastError();
}

template <class R, bool FORCE, bool WALLS, bool QUAD, bool MERGE>
cudaError_t run(SplitArgs<R> a, R *Q0, R *Q1, const R *tabs, int nsteps, cudaStream_t s)
{
    const R *bx = tabs, *by = tabs + 8 * (size_t)a.nx;                     // stage B (scale -h m)
    const R *cxs = by + 8 * (size_t)a.ny, *cys = cxs + 8 * (size_t)a.nx;   // stage C (scale -dt m)
    R *q[2] = {Q0, Q1};
    a.Qout = q[0];
    cudaError_t e = launch<R>(k_split_prepare<R, FORCE, WALLS, QUAD>, a, QUAD ? 4 : 1, WALLS, false, s);
    for (int k = 0; k < nsteps && e == cudaSuccess; ++k) {
        const bool last = k + 1 == nsteps;
        a.tx = bx;
        a.ty = by;
        e = launch<R>(k_split_star<R, FORCE, WALLS, QUAD, MERGE>, a, QUAD ? 4 : 1, WALLS, true, s);
        if (e != cudaSuccess) break;
        a.tx = cxs;
        a.ty = cys;
        a.Qin = q[k & 1];
        a.Qout = last ? a.P : q[(k + 1) & 1];
        e = last ? launch<R>(k_split_update<R, FORCE, WALLS, QUAD, MERGE, true>, a, QUAD ? 4 : 1, WALLS, true, s)
                 : launch<R>(k_split_update<R, FORCE, WALLS, QUAD, MERGE, false>, a, QUAD ? 4 : 1, WALLS, true, s);
    }
    return e;
}

}  // namespace

size_t split_table_bytes(int nx, int ny) { return 16 * (size_t)(nx + ny) * sizeof(double); }

// Grids of at most so many nodes take four threads per node throughout: up to two
// such warps per scheduler of 152 SMs on a periodic grid, one on a walled one
// (us per step, four threads against one: 24^2 6.4 / 11.7, 64^2 7.1 / 11.6, 96^2
// 10.9 / 12.5, 120^2 15.1 / 13.0; walled 65^2 10.6 / 13.2, 97^2 14.2 / 13.6).
constexpr long long kQuadNodes = 9728, kQuadWalledNodes = 4864;

// nsteps steps of the state in s.gin, in place.
cudaError_t launch_split(const StepArgs<double> &s, double *Q0, double *Q1, const double *tables, bool merge,
                         int nsteps, cudaStream_t stream)
{
    using R = double;
    if (nsteps <= 0) return cudaSuccess;
    SplitArgs<R> a{};
    a.P = const_cast<R *>(s.gin);
    a.S = s.gout;
    a.force = s.force;
    a.nx = s.nx;
    a.ny = s.ny;
    a.pitch = s.pitch;
    a.plane = s.plane;
    a.wx = s.bc_x == FDLBM_WALL;
    a.wy = s.bc_y == FDLBM_WALL;
    for (int k = 0; k < 4; ++k)
        for (int j = 0; j < 2; ++j) a.wall_u[k][j] = s.wall_u[k][j];
    a.c = s.c;
    a.keep_star = (R(1) - s.c.b_star) * R(0.5);
    a.w_star[0] = s.c.b_star * wq<R>(0);
    a.w_star[1] = s.c.b_star * wq<R>(1);
    a.w_star[2] = s.c.b_star * wq<R>(5);
    a.l_star[0] = s.c.b_star * LinearCoef<R>::c1;
    a.l_star[1] = s.c.b_star * LinearCoef<R>::c2;
    const bool walls = a.wx || a.wy;
    const std::true_type y{};
    const std::false_type n{};
    auto go = [&](auto wl, auto quad, auto mg) {
        constexpr bool W = decltype(wl)::value, Q = decltype(quad)::value, M = decltype(mg)::value;
        return s.force ? run<R, true, W, Q, M>(a, Q0, Q1, tables, nsteps, stream)
                       : run<R, false, W, Q, M>(a, Q0, Q1, tables, nsteps, stream);
    };
    const bool quad = (long long)a.nx * a.ny <= (walls ? kQuadWalledNodes : kQuadNodes);
    if (walls) return quad ? go(y, y, n) : go(y, n, n);
    if (quad) return merge ? go(n, y, y) : go(n, y, n);
    return merge ? go(n, n, y) : go(n, n, n);
}

}  // namespace fdlbm
