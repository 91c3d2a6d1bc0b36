// The FP32 T2S2-FDLBM1 step on small and medium grids, one launch per step: a
// block of 256 threads takes a tile of 32 x 16 nodes through the three stages
// of Sec. 2D in shared memory, for any boundary combination.
//
//   A  all nodes of the tile and 4 around it: P = fbar^{+,h} (Eqs. 2.19, 2.34)
//      into shared memory, Q = f~+ (Eq. 2.20) of the tile in registers
//   B  the tile and 2 around it: f* (Eqs. 2.32-2.35)
//   C  the tile: f~ of the next step (Eq. 2.23)
//
// Every thread works on pairs of neighbouring columns in packed FP32x2
// arithmetic (packed.cuh): its own pair of the tile, then one of the ring
// around it.
//
// Walls: wall nodes belong to the tile of their interior neighbour x_j.  In
// tiles that touch a wall, Eq. 3.10 runs for all their wall nodes together
// after stage B (f*) and after stage C (the new f~), one thread per wall node,
// and columns and rows next to a wall, where the upwind difference would leave
// the domain, select the central one.  Outside a walled domain, loads read the
// nearest node; no stored value depends on those.
//
// What bounds it: at 1025^2 (cavity, 29 us per step, 36 GLUPS) the shared-memory
// pipe, 60 % busy with 38 64-bit loads per pair and stage; issue slots 42 % busy.
// The tile's halo costs 1.9 times stage A and 1.4 times stage B.  On small grids
// it is one tile's latency: 64^2 3.5 us per step, 257^2 cavity 4.9 (walls sweep
// 9.8).  Tried: two rows per thread (tile 32 x 32, 128 registers) 2048^2 122 us
// against 110; more threads for the ring (384, 512) 1024^2 30 and 42 against 27.
#include <algorithm>

#include "internal.h"
#include "packed.cuh"
#include "tile.cuh"
#include "walls_nodes.cuh"

namespace fdlbm {
namespace {

using namespace packed;

template <bool FORCE>
struct TileSmem {
    f2 P[9][kAP * kAR];  // plane 0, read by its own pair only, takes f* of population 0 in
                         // stage B; after stage B the planes hold the tile's new f~ (walls)
    f2 S[8][kBP * kBR];  // f* of populations 1 to 8
    f2 F[FORCE ? 2 : 1][FORCE ? kAP * kAR : 1];
    float mx[2 * kAP], my[kAR];  // metrics of stage A's region
};

// Scale -s m of the difference in one axis for the columns of the pair (or one
// row, twice), and the columns where the difference of a sign is the central one
// alone (edge tiles).
struct Diff {
    f2 k;
    bool p0, p1, n0, n1;
};

// An output rectangle [x0, x1) x [y0, y1) that another launch writes.
struct Rect {
    int x0, x1, y0, y1;
};

// MASK: the frame of a walled grid around the warp-tile kernel's interior.
template <bool FORCE, bool MASK = false>
struct Tile {
    using Smem = TileSmem<FORCE>;
    const StepArgs<float> &a;
    Smem &sm;
    const int x0, y0, t;
    const bool wx, wy;
    const bool inside;  // no column of stage A's region lies outside [0, nx)
    Rect skip;          // MASK: nodes that are not stored
    f2 w[4];  // mixed weights at +1, 0, -1, -2
    f2 rho0;

    __device__ Tile(const StepArgs<float> &a_, Smem &sm_, int bx, int by)
        : a(a_), sm(sm_), x0(bx * kTX), y0(by * kTY), t(threadIdx.x), wx(a_.bc_x == FDLBM_WALL),
          wy(a_.bc_y == FDLBM_WALL), inside(x0 >= 4 && x0 + kTX + 4 <= a_.nx), w{bc(a_.st.wm1), bc(a_.st.w0), bc(a_.st.w1), bc(a_.st.w2)}, rho0(bc(a_.c.rho0))
    {
    }

    // The nine (or, with a force field, eleven) values of a pair: g and F.
    // (Plain loads: the read-only path is for data that no running kernel
    // writes, and a chained launch starts while the previous step still runs.)
    struct Pair {
        f2 g[9], Fx, Fy;
    };
    __device__ __forceinline__ void load(int c, int r, Pair &v) const
    {
        const int x = x0 - 4 + 2 * c;
        const size_t row = (size_t)axis_index(y0 - 4 + r, a.ny, wy) * a.pitch;
        if (inside) {  // uniform over the block; x is even: aligned pairs
            const float *p = a.gin + row + x;
#pragma unroll
            for (int i = 0; i < 9; ++i) v.g[i] = *reinterpret_cast<const f2 *>(p + i * a.plane);
            if (FORCE) {
                v.Fx = *reinterpret_cast<const f2 *>(a.force + row + x);
                v.Fy = *reinterpret_cast<const f2 *>(a.force + a.plane + row + x);
            }
        } else {
            const size_t g0 = row + axis_index(x, a.nx, wx), g1 = row + axis_index(x + 1, a.nx, wx);
#pragma unroll
            for (int i = 0; i < 9; ++i) v.g[i] = make_float2(a.gin[i * a.plane + g0], a.gin[i * a.plane + g1]);
            if (FORCE) {
                v.Fx = make_float2(a.force[g0], a.force[g1]);
                v.Fy = make_float2(a.force[a.plane + g0], a.force[a.plane + g1]);
            }
        }
    }

    // Moments with the force shift, and the equilibrium's 1/rho.  The momentum is
    // summed along each axis in the same way: the axis populations, then the two
    // diagonal ones that move forward, then the two that move back.  Near a steady
    // state every step rounds alike, and the order decides how far the state
    // settles from FP64: a 257^2 cavity at Re 1000 1.36e-4 (relative L2 of u) with
    // the lid on the N or the E wall, 6.9e-4 in the order of moments2_j, 3.4e-4 and
    // 5.3e-4 in that of moments_dev.
    __device__ __forceinline__ MacroJ macro(const f2 g[9], f2 Fx, f2 Fy, float shift) const
    {
        MacroJ m;
        const f2 east = add2(g[5], g[8]), west = add2(g[6], g[7]);
        m.jx = sub2(add2(sub2(g[1], g[3]), east), west);
        m.jy = sub2(add2(sub2(g[2], g[4]), add2(g[5], g[6])), add2(g[7], g[8]));
        m.drho = add2(add2(add2(add2(g[1], g[3]), add2(g[2], g[4])), g[0]), add2(east, west));
        const f2 rho = add2(rho0, m.drho);
        m.inv = make_float2(rcp_approx(rho.x), rcp_approx(rho.y));
        if (a.c.incomp) m.inv = bc(1.f / a.c.rho0);
        if (FORCE) {
            const f2 hr = mul2(bc(shift), a.c.incomp ? rho0 : add2(rho0, m.drho));
            m.jx = fma2(hr, Fx, m.jx);
            m.jy = fma2(hr, Fy, m.jy);
        }
        return m;
    }

    // Stage A at pair c, row r of its region; Q kept for the tile's own pairs.
    template <bool OWN>
    __device__ __forceinline__ void stage_a(int c, int r, const Pair &v, f2 Q[9])
    {
        f2 geq[9], P[9];
        const f2(&g)[9] = v.g;
        const f2 Fx = v.Fx, Fy = v.Fy;
        const MacroJ m = macro(g, Fx, Fy, a.c.half_dt);
        equilibrium2_j(m, geq);
        const f2 bb = bc(a.c.b_bar), bt = bc(a.c.b_til);
#pragma unroll
        for (int i = 0; i < 9; ++i) {
            const f2 neq = sub2(geq[i], g[i]);
            P[i] = fma2(bb, neq, g[i]);
            if (OWN) Q[i] = fma2(bt, neq, g[i]);
        }
        if (FORCE) {
            const f2 uF = mul2(fma2(m.jx, Fx, mul2(m.jy, Fy)), m.inv);
            const f2 rf = a.c.incomp ? sub2(rho0, m.drho) : rho0;
            if (OWN) force_add2(geq, rf, Fx, Fy, uF, bc(3.f * a.c.c_bar), bc(3.f * a.c.c_til), P, Q);
            else force_add1(geq, rf, Fx, Fy, uF, bc(3.f * a.c.c_bar), P);
        }
#pragma unroll
        for (int i = 0; i < 9; ++i) sm.P[i][r * kAP + c] = P[i];
        if (FORCE) {
            sm.F[0][r * kAP + c] = Fx;
            sm.F[1][r * kAP + c] = Fy;
        }
    }

    template <bool EDGE>
    __device__ __forceinline__ void weights(int x, int y, float s, Diff &dx, Diff &dy) const
    {
        const f2 mx = *reinterpret_cast<const f2 *>(&sm.mx[x - x0 + 4]);
        const float my = sm.my[y - y0 + 4];
        dx.k = mul2(bc(-s), mx);
        dy.k = bc(-s * my);
        if (EDGE) {
            dx.p0 = wx && x <= 1;
            dx.p1 = wx && x + 1 <= 1;
            dx.n0 = wx && x >= a.nx - 2;
            dx.n1 = wx && x + 1 >= a.nx - 2;
            dy.p0 = dy.p1 = wy && y <= 1;
            dy.n0 = dy.n1 = wy && y >= a.ny - 2;
        }
    }

    // acc - s xi_a d/dx_a of one axis, from the taps at 0, +1, -1, -2 along the
    // velocity: the difference first, so that the sum rounds to acc's size once.
    // Edge tiles take the same weights as the others (a central part and an upwind
    // correction with weights of their own settled the 257^2 cavity alike).
    template <bool EDGE>
    __device__ __forceinline__ f2 axis(f2 v0, f2 up, f2 dn, f2 dn2, f2 k, bool c0, bool c1, f2 acc) const
    {
        f2 d = fma2(w[3], dn2, fma2(w[2], dn, fma2(w[0], up, mul2(w[1], v0))));
        if (EDGE) {
            const f2 c = mul2(bc(0.5f), sub2(up, dn));
            d = make_float2(c0 ? c.x : d.x, c1 ? c.y : d.y);
        }
        return fma2(k, d, acc);
    }

    // acc - s xi.grad of population i from its plane f at o (row stride W).
    template <bool EDGE, int W>
    __device__ __forceinline__ f2 advance(const f2 *f, int o, int i, f2 v0, f2 acc, const Diff &dx, const Diff &dy) const
    {
        if (cx(i) != 0) {
            const f2 L = f[o - 1], R = f[o + 1];
            const f2 lo = make_float2(L.y, v0.x), hi = make_float2(v0.y, R.x);
            if (cx(i) > 0) acc = axis<EDGE>(v0, hi, lo, L, dx.k, dx.p0, dx.p1, acc);
            else acc = axis<EDGE>(v0, lo, hi, R, dx.k, dx.n0, dx.n1, acc);
        }
        if (cy(i) > 0) acc = axis<EDGE>(v0, f[o + W], f[o - W], f[o - 2 * W], dy.k, dy.p0, dy.p1, acc);
        if (cy(i) < 0) acc = axis<EDGE>(v0, f[o - W], f[o + W], f[o + 2 * W], dy.k, dy.n0, dy.n1, acc);
        return acc;
    }

    // f* of one pair from fbar* (gs).
    __device__ __forceinline__ void relax(const f2 gs[9], f2 Fx, f2 Fy, f2 st[9]) const
    {
        const MacroJ m = macro(gs, Fx, Fy, a.c.half_h);
        if (!FORCE) {
            // (1 - b') g + b' f^eq, b' = 1 - fl(1 - b) (make_relax)
            RelaxK k;
            const float omb = 1.f - a.c.b_star, bp = 1.f - omb, bc1 = bp * (1.f / 3.f), bc2 = (bp - 2.f * bc1) * 0.25f;
            k.omb = bc(omb);
            k.bw0 = bc(bp * (4.f / 9.f));
            k.bw1 = bc(bp * (1.f / 9.f));
            k.bw2 = bc(bp * (1.f / 36.f));
            k.bc1 = bc(bc1);
            k.bc2 = bc(bc2);
            k.nbc1 = bc(-bc1);
            k.nbc2 = bc(-bc2);
            relax2_j(m, gs, k, st);
        } else {
            f2 geq[9];
            equilibrium2_j(m, geq);
            const f2 bs = bc(a.c.b_star);
#pragma unroll
            for (int i = 0; i < 9; ++i) st[i] = fma2(bs, sub2(geq[i], gs[i]), gs[i]);
            const f2 uF = mul2(fma2(m.jx, Fx, mul2(m.jy, Fy)), m.inv);
            force_add1(geq, a.c.incomp ? sub2(rho0, m.drho) : rho0, Fx, Fy, uF, bc(3.f * a.c.c_star), st);
        }
    }

    // Stage B at pair c, row r of its region.
    template <bool EDGE>
    __device__ __forceinline__ void stage_b(int c, int r)
    {
        const int o = (r + 2) * kAP + c + 1;
        Diff dx, dy;
        weights<EDGE>(x0 - 2 + 2 * c, y0 - 2 + r, a.c.h, dx, dy);
        f2 gs[9], st[9], Fx = bc(0.f), Fy = bc(0.f);
        if (FORCE) {
            Fx = sm.F[0][o];
            Fy = sm.F[1][o];
        }
#pragma unroll
        for (int i = 0; i < 9; ++i) {
            const f2 v0 = sm.P[i][o];
            gs[i] = i == 0 ? v0 : advance<EDGE, kAP>(sm.P[i], o, i, v0, v0, dx, dy);
        }
        relax(gs, Fx, Fy, st);
        if (EDGE) sm.P[0][o] = st[0];
#pragma unroll
        for (int i = 1; i < 9; ++i) sm.S[i - 1][r * kBP + c] = st[i];
    }

    // Eq. 3.10 for f* of the wall nodes in stage B's region (corners are never read).
    __device__ __forceinline__ void walls_star()
    {
        constexpr int BX = 2 * kBP;
        int x, y, jx, jy;
        float u, v;
        if (t < 2 * BX) {  // S and N rows
            const bool south = t < BX;
            x = jx = x0 - 2 + (south ? t : t - BX);
            y = south ? 0 : a.ny - 1;
            jy = south ? 1 : a.ny - 2;
            u = south ? a.wall_u[FDLBM_WALL_S][0] : a.wall_u[FDLBM_WALL_N][0];
            v = south ? a.wall_u[FDLBM_WALL_S][1] : a.wall_u[FDLBM_WALL_N][1];
            if (!wy || (wx && (x < 1 || x > a.nx - 2))) return;
        } else {  // W and E columns
            const int q = t - 2 * BX;
            const bool west = q < kBR;
            y = jy = y0 - 2 + (west ? q : q - kBR);
            x = west ? 0 : a.nx - 1;
            jx = west ? 1 : a.nx - 2;
            u = west ? a.wall_u[FDLBM_WALL_W][0] : a.wall_u[FDLBM_WALL_E][0];
            v = west ? a.wall_u[FDLBM_WALL_W][1] : a.wall_u[FDLBM_WALL_E][1];
            if (q >= 2 * kBR || !wx || (wy && (y < 1 || y > a.ny - 2))) return;
        }
        // both nodes in the region?
        const int xl = x0 - 2, yl = y0 - 2;
        if (min(x, jx) < xl || max(x, jx) >= xl + BX || min(y, jy) < yl || max(y, jy) >= yl + kBR) return;
        float g[9], wv[9];
        float *s = reinterpret_cast<float *>(&sm.S[0][0]);
        const int oj = (jy - yl) * BX + (jx - xl), ob = (y - yl) * BX + (x - xl);
        g[0] = reinterpret_cast<const float *>(&sm.P[0][0])[(jy - yl + 2) * (2 * kAP) + (jx - xl + 2)];
#pragma unroll
        for (int i = 1; i < 9; ++i) g[i] = s[(i - 1) * (2 * kBP * kBR) + oj];
        nee<float, false>(a.c, g, 0.f, 0.f, 0.f, u, v, wv);
#pragma unroll
        for (int i = 1; i < 9; ++i) s[(i - 1) * (2 * kBP * kBR) + ob] = wv[i];
    }

    // Stage C at the thread's own pair; Q becomes the new f~.
    template <bool EDGE>
    __device__ __forceinline__ void stage_c(int p, int r, f2 Q[9])
    {
        const int o = (r + 2) * kBP + p + 1;
        Diff dx, dy;
        weights<EDGE>(x0 + 2 * p, y0 + r, a.c.dt, dx, dy);
#pragma unroll
        for (int i = 1; i < 9; ++i) Q[i] = advance<EDGE, kBP>(sm.S[i - 1], o, i, sm.S[i - 1][o], Q[i], dx, dy);
    }

    // Eq. 3.10 for the new f~ of the wall nodes whose x_j is in the tile.
    __device__ __forceinline__ void walls_out()
    {
        int x, y, jx, jy, side;
        if (t < 2 * kTX) {  // S and N rows
            const bool south = t < kTX;
            x = jx = x0 + (south ? t : t - kTX);
            y = south ? 0 : a.ny - 1;
            jy = south ? 1 : a.ny - 2;
            side = south ? FDLBM_WALL_S : FDLBM_WALL_N;
            if (!wy || x >= a.nx || (wx && (x < 1 || x > a.nx - 2))) return;
        } else if (t < 2 * kTX + 2 * kTY) {  // W and E columns
            const int q = t - 2 * kTX;
            const bool west = q < kTY;
            y = jy = y0 + (west ? q : q - kTY);
            x = west ? 0 : a.nx - 1;
            jx = west ? 1 : a.nx - 2;
            side = west ? FDLBM_WALL_W : FDLBM_WALL_E;
            if (!wx || y >= a.ny || (wy && (y < 1 || y > a.ny - 2))) return;
        } else {  // corners: diagonal x_j, the velocity of the W and E walls
            const int q = t - 2 * kTX - 2 * kTY;
            if (q >= 4 || !wx || !wy) return;
            x = q & 1 ? a.nx - 1 : 0;
            jx = q & 1 ? a.nx - 2 : 1;
            y = q & 2 ? a.ny - 1 : 0;
            jy = q & 2 ? a.ny - 2 : 1;
            side = q & 1 ? FDLBM_WALL_E : FDLBM_WALL_W;
        }
        if (jx < x0 || jx >= x0 + kTX || jy < y0 || jy >= y0 + kTY) return;
        float u = 0.f, v = 0.f;
#pragma unroll
        for (int s = 0; s < 4; ++s)
            if (s == side) {
                u = a.wall_u[s][0];
                v = a.wall_u[s][1];
            }
        float g[9], wv[9], Fx = 0.f, Fy = 0.f;
        const float *s = reinterpret_cast<const float *>(&sm.P[0][0]);
#pragma unroll
        for (int i = 0; i < 9; ++i) g[i] = s[i * (2 * kAP * kAR) + (jy - y0) * kTX + (jx - x0)];
        if (FORCE) {
            const size_t fo = (size_t)jy * a.pitch + jx;
            Fx = __ldg(a.force + fo);
            Fy = __ldg(a.force + a.plane + fo);
        }
        nee<float, FORCE>(a.c, g, Fx, Fy, a.c.half_dt, u, v, wv);
        const size_t ob = (size_t)y * a.pitch + x;
#pragma unroll
        for (int i = 0; i < 9; ++i) a.gout[i * a.plane + ob] = wv[i];
    }

    template <bool EDGE>
    __device__ __forceinline__ void run()
    {
        const int p = t % kTP, r = t / kTP;
        int c, rr;
        f2 Q[9];
        {
            // both loads first: the ring's is in flight during the work on the own pair
            Pair own, ring;
            load(p + 2, r + 4, own);
            ring_site<4>(min(t, kARing - 1), c, rr);
            if (t < kARing) load(c, rr, ring);
            stage_a<true>(p + 2, r + 4, own, Q);
            f2 unused[9];
            if (t < kARing) stage_a<false>(c, rr, ring, unused);
        }
        __syncthreads();
        stage_b<EDGE>(p + 1, r + 2);
        if (t < kBRing) {
            ring_site<2>(t, c, rr);
            stage_b<EDGE>(c, rr);
        }
        __syncthreads();
        if (EDGE) {
            walls_star();
            __syncthreads();
        }
        stage_c<EDGE>(p, r, Q);
        const int x = x0 + 2 * p, y = y0 + r;
        const bool row = wy ? y >= 1 && y <= a.ny - 2 : y < a.ny;
        bool lo = wx ? x >= 1 && x <= a.nx - 2 : x < a.nx;
        bool hi = wx ? x + 1 <= a.nx - 2 : x + 1 < a.nx;
        if (MASK && y >= skip.y0 && y < skip.y1) {
            lo = lo && (x < skip.x0 || x >= skip.x1);
            hi = hi && (x + 1 < skip.x0 || x + 1 >= skip.x1);
        }
        float *dst = a.gout + (size_t)y * a.pitch + x;
        if (row && lo && hi) {
#pragma unroll
            for (int i = 0; i < 9; ++i) *reinterpret_cast<f2 *>(dst + i * a.plane) = Q[i];
        } else if (row) {
#pragma unroll
            for (int i = 0; i < 9; ++i) {
                if (lo) dst[i * a.plane] = Q[i].x;
                if (hi) dst[i * a.plane + 1] = Q[i].y;
            }
        }
        if (EDGE) {
#pragma unroll
            for (int i = 0; i < 9; ++i) sm.P[i][t] = Q[i];
            __syncthreads();
            walls_out();
        }
    }

    __device__ __forceinline__ void metrics()
    {
        if (t < 2 * kAP) sm.mx[t] = __ldg(a.mx + axis_index(x0 - 4 + t, a.nx, wx));
        else if (t < 2 * kAP + kAR) sm.my[t - 2 * kAP] = __ldg(a.my + axis_index(y0 - 4 + t - 2 * kAP, a.ny, wy));
    }

    // A tile whose stages B and C meet a wall or the weights next to one.
    __device__ __forceinline__ bool edge() const
    {
        return (wx && (x0 <= 3 || x0 + kTX + 1 >= a.nx - 2)) || (wy && (y0 <= 3 || y0 + kTY + 1 >= a.ny - 2));
    }

    template <bool WALLS>
    __device__ __forceinline__ void go()
    {
        if (WALLS && edge()) run<true>();
        else run<false>();
    }
};

constexpr int kMinBlocks = 3;  // 80 registers, 58 KB (66 KB with a force field) of shared memory

// The metrics are fetched before the previous step's results are needed.
template <bool FORCE, bool WALLS>
__device__ __forceinline__ void tile_step(const StepArgs<float> &a, unsigned char *smem_raw, int bx, int by)
{
    Tile<FORCE> tile(a, *reinterpret_cast<TileSmem<FORCE> *>(smem_raw), bx, by);
    tile.metrics();
    chain_wait();
    tile.template go<WALLS>();
    chain_next();
}

// TALL: a launch for the rows of tiles from row0 on.
template <bool FORCE, bool WALLS, bool TALL>
__global__ void __launch_bounds__(kNT, kMinBlocks)
    k_step_tile(const __grid_constant__ StepArgs<float> a, const int row0)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    tile_step<FORCE, WALLS>(a, smem_raw, blockIdx.x, blockIdx.y + (TALL ? row0 : 0));
}

// The frame of a walled grid: the tiles that hold nodes outside `skip`, the
// interior rectangle of the warp-tile kernel.  One wave of blocks lasts about
// 10 us, where the walls sweep in blocks of one warp walks a chain of twelve rows
// and more in 25 us (2049^2 cavity 95 -> 81 us per step, 4097^2 279 -> 265, forced
// 2048 x 2049 channel 137 -> 113).  On a walled x axis those are the
// first column of tiles and the ones from `east` on, then on a walled y axis the
// first row and the ones from `north` on.
struct FrameTiles {
    Rect skip;
    int tx, ty, east, north;  // tiles of the grid; first frame column and row on the far sides
    int cols, rows;           // frame columns (ty tiles each) and rows (of the other columns)
};

template <bool FORCE>
__global__ void __launch_bounds__(kNT, kMinBlocks)
    k_frame_tile(const __grid_constant__ StepArgs<float> a, const __grid_constant__ FrameTiles f)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    int b = blockIdx.x, bx, by;
    if (b < f.cols * f.ty) {
        bx = b / f.ty;
        by = b - bx * f.ty;
        if (bx > 0) bx += f.east - 1;
    } else {
        b -= f.cols * f.ty;
        const int w = f.tx - f.cols;  // the columns that are not in the frame
        by = b / w;
        bx = b - by * w + (f.cols > 0 ? 1 : 0);
        if (by > 0) by += f.north - 1;
    }
    Tile<FORCE, true> tile(a, *reinterpret_cast<TileSmem<FORCE> *>(smem_raw), bx, by);
    tile.skip = f.skip;
    tile.metrics();
    chain_wait();
    tile.template go<true>();
    chain_next();
}

// Batched: block b is tile (b - blk_start[c]) of case c = blk_case[b], tiles_x[c]
// tiles per row; the case's arguments are copied into shared memory first.
constexpr size_t kArgsOff = (sizeof(TileSmem<true>) + 15) / 16 * 16;

__global__ void __launch_bounds__(kNT, kMinBlocks)
    kb_step_tile(const StepArgs<float> *cases, const int *blk_case, const int *blk_start, const int *tiles_x,
                 int blk_off)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    StepArgs<float> *s = reinterpret_cast<StepArgs<float> *>(smem_raw + kArgsOff);
    static_assert(sizeof(StepArgs<float>) % 4 == 0 && sizeof(StepArgs<float>) / 4 <= kNT, "copied as 32-bit words");
    const int bid = blk_off + blockIdx.x;
    const int c = blk_case[bid];
    if (threadIdx.x < sizeof(StepArgs<float>) / 4)
        reinterpret_cast<int *>(s)[threadIdx.x] = reinterpret_cast<const int *>(cases + c)[threadIdx.x];
    const int u = bid - blk_start[c], nt = tiles_x[c];
    __syncthreads();
    if (s->force) tile_step<true, true>(*s, smem_raw, u % nt, u / nt);
    else tile_step<false, true>(*s, smem_raw, u % nt, u / nt);
}

}  // namespace

void tile_counts(int nx, int ny, bool wall_x, bool wall_y, int *tx, int *ty)
{
    *tx = tiles_along(nx, wall_x, kTX);
    *ty = tiles_along(ny, wall_y, kTY);
}

int tile_launches(int nx, int ny, bool wall_x, bool wall_y)
{
    int tx, ty;
    tile_counts(nx, ny, wall_x, wall_y, &tx, &ty);
    return (ty + kMaxTileRows - 1) / kMaxTileRows;
}

cudaError_t launch_tile(const StepArgs<float> &a, cudaStream_t s)
{
    const bool walls = a.bc_x == FDLBM_WALL || a.bc_y == FDLBM_WALL;
    const size_t smem = a.force ? sizeof(TileSmem<true>) : sizeof(TileSmem<false>);
    int tx, ty;
    tile_counts(a.nx, a.ny, a.bc_x == FDLBM_WALL, a.bc_y == FDLBM_WALL, &tx, &ty);
    auto kern = a.force ? (walls ? k_step_tile<true, true, false> : k_step_tile<true, false, false>)
                        : (walls ? k_step_tile<false, true, false> : k_step_tile<false, false, false>);
    if (ty > kMaxTileRows) kern = a.force ? k_step_tile<true, true, true> : k_step_tile<false, true, true>;
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    for (int row0 = 0; row0 < ty && e == cudaSuccess; row0 += kMaxTileRows)
        e = chained_launch(kern, dim3(tx, std::min(ty - row0, kMaxTileRows)), kNT, smem, s, a, row0);
    return e;
}

// The nodes of a walled grid outside the rectangle [x0, x1) x [y0, y1).
cudaError_t launch_frame_tile(const StepArgs<float> &a, int x0, int x1, int y0, int y1, cudaStream_t s)
{
    const bool wx = a.bc_x == FDLBM_WALL, wy = a.bc_y == FDLBM_WALL;
    FrameTiles f{{x0, x1, y0, y1}};
    tile_counts(a.nx, a.ny, wx, wy, &f.tx, &f.ty);
    // (a rectangle that is empty, or ends in the first tile: every tile is frame)
    const bool none = x1 <= x0 || y1 <= y0;
    f.east = none ? 1 : std::min(f.tx, std::max(1, x1 / kTX));
    f.north = none ? 1 : std::min(f.ty, std::max(1, y1 / kTY));
    f.cols = wx || none ? 1 + f.tx - f.east : 0;
    f.rows = wy && f.cols < f.tx ? 1 + f.ty - f.north : 0;
    const size_t smem = a.force ? sizeof(TileSmem<true>) : sizeof(TileSmem<false>);
    auto kern = a.force ? k_frame_tile<true> : k_frame_tile<false>;
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    return chained_launch(kern, dim3(f.cols * f.ty + f.rows * (f.tx - f.cols)), kNT, smem, s, a, f);
}

// Tiles [blk_off, blk_off + nblocks) of the batch's tables.
cudaError_t launch_batched_tile(const BatchTables &t, int parity, int blk_off, int nblocks, cudaStream_t s)
{
    if (nblocks <= 0) return cudaSuccess;
    constexpr size_t smem = kArgsOff + sizeof(StepArgs<float>);
    cudaError_t e = cudaFuncSetAttribute(kb_step_tile, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    return chained_launch(kb_step_tile, dim3(nblocks), kNT, smem, s,
                          static_cast<const StepArgs<float> *>(t.args[parity]), t.blk_case, t.blk_start, t.tiles_x,
                          blk_off);
}

}  // namespace fdlbm
