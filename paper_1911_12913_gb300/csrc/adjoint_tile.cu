// One FP32 adjoint step (adjoint.cu has the formulas) in one launch: a block
// takes a tile of 32 x 16 nodes through the three stages in shared memory, on
// pairs of neighbouring columns in packed FP32x2 arithmetic, as the forward
// tile kernel (step_tile.cu) does.
//
//   A'  the tile and 4 around it: g, F -> P = fbar^{+,h}; lam' and F into shared memory
//   B'  the tile and 2 around it: gs = P - h D(P), lam_S = -dt D^T lam', the node
//       map's VJP at gs -> lam_gs, and the force cotangent of stage B
//   C'  the tile: lam_P = lam_gs - h D^T lam_gs, the node maps' VJP at g -> lam,
//       and the force cotangent, added in FP64
//
// The node maps are polynomials of second degree in the lattice velocity, so
// their VJPs need only the lattice moments of the incoming cotangents (six, eight
// with the forcing term of Eq. 3.12): no per-population derivative is formed.
//
// What bounds it: latency at two blocks per SM (98 KB of shared memory, 124
// registers): shared-memory pipe 65 %, issue slots 42 % busy, waits for global
// loads and for dependent arithmetic first; so the loads of stage C' (g, the rest
// population of lam', the FP64 force gradient) are issued before the barrier that
// precedes it (2048^2 274 -> 252 us), and the
// metrics before the previous step's results are needed.  Persistent blocks that
// copied the next tile during stage C' were slower (278 us: 76 small copies per
// thread and tile).  Against the sweep of adjoint.cu, which walks a chain of
// rows in scalar arithmetic, us per step on GB300, with a force field: 256^2
// 18.4 -> 7.4, 512^2 19.6, 2048^2 360 -> 254, 4096^2 1288 -> 1007.
#include <algorithm>
#include <cstdint>

#include "internal.h"
#include "packed.cuh"
#include "tile.cuh"

namespace fdlbm {
namespace {

using namespace packed;

struct AdjSmem {
    f2 P[9][kAP * kAR];
    f2 L[8][kAP * kAR];  // lam' of populations 1 to 8
    f2 G[8][kBP * kBR];  // lam_gs of populations 1 to 8
    f2 F[2][kAP * kAR];
    float mx[2 * kAP], my[kAR];
};

struct AdjTileArgs {
    StepArgs<float> a;
    const float *lam_next;
    float *lam_prev;
    double *dforce;
    int row0;  // first row of tiles of the launch (TALL)
};

// Lattice moments sum w_i (1, 3x, 3y, xx, xy, yy, xxy, xyy) v_i of a cotangent.
// The cotangents of density and momentum pass through every collision, so the
// rounding of the first three adds up over a rollout.  They are written as the
// value that one population (or one opposite pair) gives plus the departures of
// the others from it: v_i = c0 + xi_i . c returns c0 and c with no error from the
// weights, and a cotangent near that form with few roundings of full size (force
// gradient of a 100-step rollout on 256^2: 2.7e-7 off the 64-bit one, with the plain
// sums 9e-7, with the sweep of adjoint.cu 6e-7).
struct Moments {
    f2 m0, x3, y3, xx, xy, yy, xxy, xyy;
    __device__ __forceinline__ void set(const f2 v[9])
    {
        const f2 w1 = bc(1.f / 9.f), w2 = bc(1.f / 36.f), c2 = bc(1.f / 12.f);
        const f2 s13 = add2(v[1], v[3]), d13 = sub2(v[1], v[3]), s24 = add2(v[2], v[4]), d24 = sub2(v[2], v[4]);
        const f2 s57 = add2(v[5], v[7]), d57 = sub2(v[5], v[7]), s68 = add2(v[6], v[8]), d68 = sub2(v[6], v[8]);
        const f2 sd = add2(s57, s68), dy = add2(d57, d68), dx = sub2(d57, d68), q = mul2(w2, sd);
        const f2 n4 = mul2(bc(-4.f), v[0]);
        m0 = add2(v[0], fma2(w1, add2(add2(s13, s24), n4), mul2(w2, add2(sd, n4))));
        x3 = fma2(bc(0.5f), d13, mul2(c2, fma2(bc(-2.f), d13, dx)));
        y3 = fma2(bc(0.5f), d24, mul2(c2, fma2(bc(-2.f), d24, dy)));
        xx = fma2(w1, s13, q);
        yy = fma2(w1, s24, q);
        xy = mul2(w2, sub2(s57, s68));
        xxy = mul2(w2, dy);
        xyy = mul2(w2, dx);
    }
};

// a p + b q, per moment.
__device__ __forceinline__ Moments combine(f2 a, const Moments &p, f2 b, const Moments &q)
{
    return {fma2(a, p.m0, mul2(b, q.m0)), fma2(a, p.x3, mul2(b, q.x3)),   fma2(a, p.y3, mul2(b, q.y3)),
            fma2(a, p.xx, mul2(b, q.xx)), fma2(a, p.xy, mul2(b, q.xy)),   fma2(a, p.yy, mul2(b, q.yy)),
            fma2(a, p.xxy, mul2(b, q.xxy)), fma2(a, p.xyy, mul2(b, q.xyy))};
}

__device__ __forceinline__ Moments scaled(f2 a, const Moments &p)
{
    return {mul2(a, p.m0), mul2(a, p.x3), mul2(a, p.y3),  mul2(a, p.xx),
            mul2(a, p.xy), mul2(a, p.yy), mul2(a, p.xxy), mul2(a, p.xyy)};
}

// The node map at g (moments with the force shift sh, Eqs. 3.2, 3.3, 3.12) and
// its vector-Jacobian product.
struct NodeVjp {
    f2 rho, ux, uy;
    __device__ __forceinline__ void eval(const f2 g[9], f2 rho0, f2 Fx, f2 Fy, float sh)
    {
        const MacroJ m = moments2_j(g, rho0);
        rho = add2(rho0, m.drho);
        const f2 hr = mul2(bc(sh), rho);
        ux = mul2(fma2(hr, Fx, m.jx), m.inv);
        uy = mul2(fma2(hr, Fy, m.jy), m.inv);
    }

    // B: moments of the cotangents of f^eq, C: of the F_i.  With e = xi.u, s =
    // (xi - u).F, Phi = 3e + 4.5e^2 - 1.5u.u the map is f^eq_i = w_i [drho + rho
    // Phi_i] (minus w_i rho0), F_i = 3 s_i w_i rho (1 + Phi_i), and
    //   T, Tx, Ty = sum (1 + Phi_i) (1, x, y) w_i lam_F,i
    //   a_i = lam_eq,i + 3 s_i lam_F,i    the cotangent of f^eq_i
    // The cotangent of u is rho times sum (3 + 9 e_i) xi_i w_i a_i - 3 u sum w_i
    // a_i - 3 F T, and j = rho u - sh rho F takes it over rho, so rho cancels.
    // Returns what the cotangents of the zeroth moment and of the first of g have
    // beyond B's own (d0, dx, dy: terms in u and F), and adds those of the force
    // to lFx, lFy.
    __device__ __forceinline__ void vjp(const Moments &B, const Moments &C, f2 Fx, f2 Fy, float sh, f2 &d0, f2 &dx,
                                        f2 &dy, f2 &lFx, f2 &lFy) const
    {
        const f2 three = bc(3.f);
        const f2 ux3 = mul2(three, ux), uy3 = mul2(three, uy), ux9 = mul2(three, ux3), uy9 = mul2(three, uy3);
        const f2 qx = mul2(mul2(bc(1.5f), ux), ux3), qy = mul2(mul2(bc(1.5f), uy), uy3);  // 4.5 u^2
        const f2 qxy = mul2(ux3, uy3);                                                    // 9 ux uy
        const f2 nk = mul2(bc(-1.f / 3.f), add2(qx, qy));                                 // -1.5 u.u
        const f2 k = add2(bc(1.f), nk);
        f2 t = fma2(qx, C.xx, fma2(qy, C.yy, mul2(qxy, C.xy)));
        const f2 T = fma2(k, C.m0, fma2(ux, C.x3, fma2(uy, C.y3, t)));
        t = mul2(three, fma2(qxy, C.xxy, mul2(qy, C.xyy)));
        const f2 Tx3 = fma2(add2(k, qx), C.x3, fma2(ux9, C.xx, fma2(uy9, C.xy, t)));
        t = mul2(three, fma2(qxy, C.xyy, mul2(qx, C.xxy)));
        const f2 Ty3 = fma2(add2(k, qy), C.y3, fma2(ux9, C.xy, fma2(uy9, C.yy, t)));
        // w_i a_i, in moments
        const f2 fx3 = mul2(three, Fx), fy3 = mul2(three, Fy), fx9 = mul2(three, fx3), fy9 = mul2(three, fy3);
        const f2 nuf = mul2(bc(-1.f), fma2(ux, fx3, mul2(uy, fy3)));
        const f2 b0 = fma2(nuf, C.m0, fma2(Fx, C.x3, mul2(Fy, C.y3)));
        const f2 bx3 = fma2(nuf, C.x3, fma2(fx9, C.xx, mul2(fy9, C.xy)));
        const f2 by3 = fma2(nuf, C.y3, fma2(fx9, C.xy, mul2(fy9, C.yy)));
        const f2 a0 = add2(B.m0, b0), ax3 = add2(B.x3, bx3), ay3 = add2(B.y3, by3);
        const f2 axx = fma2(nuf, C.xx, fma2(Fx, C.x3, fma2(fy3, C.xxy, B.xx)));
        const f2 axy = fma2(nuf, C.xy, fma2(fx3, C.xxy, fma2(fy3, C.xyy, B.xy)));
        const f2 ayy = fma2(nuf, C.yy, fma2(fx3, C.xyy, fma2(Fy, C.y3, B.yy)));
        t = fma2(qx, axx, fma2(qy, ayy, mul2(qxy, axy)));
        f2 lrho = fma2(nk, a0, fma2(ux, ax3, fma2(uy, ay3, t)));
        const f2 na0 = mul2(bc(-1.f), a0), nT = mul2(bc(-1.f), T);
        dx = add2(bx3, fma2(ux9, axx, fma2(uy9, axy, fma2(ux3, na0, mul2(fx3, nT)))));
        dy = add2(by3, fma2(ux9, axy, fma2(uy9, ayy, fma2(uy3, na0, mul2(fy3, nT)))));
        const f2 s = bc(sh), cx = add2(B.x3, dx), cy = add2(B.y3, dy);
        lrho = fma2(cx, fma2(s, Fx, mul2(bc(-1.f), ux)), fma2(cy, fma2(s, Fy, mul2(bc(-1.f), uy)), lrho));
        lFx = fma2(rho, fma2(ux3, nT, fma2(s, cx, Tx3)), lFx);
        lFy = fma2(rho, fma2(uy3, nT, fma2(s, cy, Ty3)), lFy);
        d0 = add2(b0, lrho);
    }
};

// c0 + xi_i . c for the nine populations.
__device__ __forceinline__ void linear(f2 c0, f2 cx, f2 cy, f2 v[9])
{
    v[0] = c0;
    v[1] = add2(c0, cx);
    v[3] = sub2(c0, cx);
    v[2] = add2(c0, cy);
    v[4] = sub2(c0, cy);
    v[5] = add2(v[1], cy);
    v[8] = sub2(v[1], cy);
    v[6] = add2(v[3], cy);
    v[7] = sub2(v[3], cy);
}

// Metrics around a pair, for the transposed differences: of the pairs to the
// left, here and to the right, and of the rows k - 2 .. k + 2.  The weights of
// Eq. 2.36 sum to zero exactly and multiply m lam, so that on a uniform grid the
// transposed difference of a constant vanishes (weights that carried the metric,
// rounded tap by tap, would scale the cotangent by about 1e-8 a step).  UNI: one
// metric value on each axis, which multiplies the sum instead.
template <bool UNI>
struct Around {
    f2 x[UNI ? 1 : 3], y[UNI ? 1 : 5];
};

// Asynchronous copies global -> shared of a pair (8 bytes) or one value (4).
__device__ __forceinline__ void copy8(void *dst, const float *src)
{
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"((unsigned)__cvta_generic_to_shared(dst)), "l"(src)
                 : "memory");
}
__device__ __forceinline__ void copy4(void *dst, const float *src)
{
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"((unsigned)__cvta_generic_to_shared(dst)), "l"(src)
                 : "memory");
}

template <bool FORCE, bool UNI>
struct AdjTile {
    const AdjTileArgs &q;
    const StepArgs<float> &a;
    AdjSmem &sm;
    const int x0, y0, t;
    const bool inside;  // no column of stage A's region lies outside [0, nx)
    f2 w[4];            // mixed weights at +1, 0, -1, -2
    f2 rho0;

    __device__ AdjTile(const AdjTileArgs &q_, AdjSmem &sm_, int bx, int by)
        : q(q_), a(q_.a), sm(sm_), x0(bx * kTX), y0(by * kTY), t(threadIdx.x),
          inside(x0 >= 4 && x0 + kTX + 4 <= q_.a.nx),
          w{bc(q_.a.st.wm1), bc(q_.a.st.w0), bc(q_.a.st.w1), bc(q_.a.st.w2)}, rho0(bc(q_.a.c.rho0))
    {
    }

    // Offsets of the pair c, row r of stage A's region.
    __device__ __forceinline__ void site(int c, int r, size_t &g0, size_t &g1) const
    {
        const int x = x0 - 4 + 2 * c;
        const size_t row = (size_t)axis_index(y0 - 4 + r, a.ny, false) * a.pitch;
        g0 = row + (inside ? x : axis_index(x, a.nx, false));
        g1 = inside ? g0 + 1 : row + axis_index(x + 1, a.nx, false);
    }

    __device__ __forceinline__ f2 pair(const float *p, size_t g0, size_t g1) const
    {
        return inside ? *reinterpret_cast<const f2 *>(p + g0) : make_float2(p[g0], p[g1]);
    }

    // lam' (populations 1 to 8) into shared memory, in flight during stage A'.
    __device__ __forceinline__ void fetch(int o, size_t g0, size_t g1)
    {
#pragma unroll
        for (int i = 1; i < 9; ++i) {
            const float *p = q.lam_next + i * a.plane;
            if (inside) {
                copy8(&sm.L[i - 1][o], p + g0);
            } else {
                copy4(&sm.L[i - 1][o].x, p + g0);
                copy4(&sm.L[i - 1][o].y, p + g1);
            }
        }
    }

    __device__ __forceinline__ void load_g(size_t g0, size_t g1, f2 g[9]) const
    {
#pragma unroll
        for (int i = 0; i < 9; ++i) g[i] = pair(a.gin + i * a.plane, g0, g1);
    }

    // Stage A': P from g and F, as the forward step forms it.
    __device__ __forceinline__ void stage_a(int o, const f2 g[9], f2 Fx, f2 Fy)
    {
        MacroJ m = moments2_j(g, rho0);
        if (FORCE) {
            const f2 hr = mul2(bc(a.c.half_dt), add2(rho0, m.drho));
            m.jx = fma2(hr, Fx, m.jx);
            m.jy = fma2(hr, Fy, m.jy);
        }
        f2 geq[9], P[9];
        equilibrium2_j(m, geq);
#pragma unroll
        for (int i = 0; i < 9; ++i) P[i] = fma2(bc(a.c.b_bar), sub2(geq[i], g[i]), g[i]);
        if (FORCE) {
            const f2 uF = mul2(fma2(m.jx, Fx, mul2(m.jy, Fy)), m.inv);
            force_add1(geq, rho0, Fx, Fy, uF, bc(3.f * a.c.c_bar), P);
            sm.F[0][o] = Fx;
            sm.F[1][o] = Fy;
        }
#pragma unroll
        for (int i = 0; i < 9; ++i) sm.P[i][o] = P[i];
    }

    // sum_j w_j (m lam)(k + s j) over both axes for population i from its plane
    // f at o (row stride W), v0 the value there.
    template <int W>
    __device__ __forceinline__ f2 gather(const f2 *f, int o, int i, f2 v0, const Around<UNI> &m) const
    {
        f2 sum = bc(0.f);
        // values at -1, 0, +1, +2 along the velocity
        auto axis = [&](f2 dn, f2 at, f2 up, f2 up2) {
            return fma2(w[3], up2, fma2(w[2], up, fma2(w[0], dn, mul2(w[1], at))));
        };
        if (cx(i) != 0) {
            f2 L = f[o - 1], C = v0, R = f[o + 1];
            if (!UNI) {
                L = mul2(L, m.x[0]);
                C = mul2(C, m.x[UNI ? 0 : 1]);
                R = mul2(R, m.x[UNI ? 0 : 2]);
            }
            const f2 lo = make_float2(L.y, C.x), hi = make_float2(C.y, R.x);
            sum = cx(i) > 0 ? axis(lo, C, hi, R) : axis(hi, C, lo, L);
            if (UNI) sum = mul2(m.x[0], sum);
        }
        if (cy(i) != 0) {
            const int s = cy(i) > 0 ? 1 : -1;
            f2 dn = f[o - s * W], at = v0, up = f[o + s * W], up2 = f[o + 2 * s * W];
            if (!UNI) {
                dn = mul2(dn, m.y[UNI ? 0 : 2 - s]);
                at = mul2(at, m.y[UNI ? 0 : 2]);
                up = mul2(up, m.y[UNI ? 0 : 2 + s]);
                up2 = mul2(up2, m.y[UNI ? 0 : 2 + 2 * s]);
            }
            const f2 ys = axis(dn, at, up, up2);
            if (UNI) sum = cx(i) != 0 ? fma2(m.y[0], ys, sum) : mul2(m.y[0], ys);
            else sum = cx(i) != 0 ? add2(sum, ys) : ys;
        }
        return sum;
    }

    // The metrics around column pair cA, row rA of stage A's region.
    __device__ __forceinline__ Around<UNI> around(int cA, int rA) const
    {
        Around<UNI> m;
        const f2 *x = reinterpret_cast<const f2 *>(sm.mx) + cA;
        const float *y = sm.my + rA;
        if (UNI) {
            m.x[0] = x[0];
            m.y[0] = bc(y[0]);
        } else {
#pragma unroll
            for (int k = 0; k < (UNI ? 1 : 3); ++k) m.x[k] = x[k - 1];
#pragma unroll
            for (int k = 0; k < (UNI ? 1 : 5); ++k) m.y[k] = bc(y[k - 2]);
        }
        return m;
    }

    // Stage B' at pair c, row r of its region: lam_gs (lg) and the force cotangent.
    __device__ __forceinline__ void stage_b(int c, int r, f2 lg[9], f2 &fBx, f2 &fBy)
    {
        const int o = (r + 2) * kAP + c + 1;
        f2 Fx = bc(0.f), Fy = bc(0.f);
        if (FORCE) {
            Fx = sm.F[0][o];
            Fy = sm.F[1][o];
        }
        NodeVjp n;
        {
            const f2 mxc = reinterpret_cast<const f2 *>(sm.mx)[c + 1];
            const f2 kx = mul2(bc(-a.c.h), mxc), ky = bc(-a.c.h * sm.my[r + 2]);
            f2 gs[9];
#pragma unroll
            for (int i = 0; i < 9; ++i) {
                const f2 *f = sm.P[i];
                const f2 v0 = f[o];
                f2 acc = v0;
                auto axis = [&](f2 up, f2 dn, f2 dn2, f2 k) {
                    acc = fma2(k, fma2(w[3], dn2, fma2(w[2], dn, fma2(w[0], up, mul2(w[1], v0)))), acc);
                };
                if (cx(i) != 0) {
                    const f2 L = f[o - 1], R = f[o + 1];
                    const f2 lo = make_float2(L.y, v0.x), hi = make_float2(v0.y, R.x);
                    if (cx(i) > 0) axis(hi, lo, L, kx);
                    else axis(lo, hi, R, kx);
                }
                if (cy(i) > 0) axis(f[o + kAP], f[o - kAP], f[o - 2 * kAP], ky);
                if (cy(i) < 0) axis(f[o - kAP], f[o + kAP], f[o + 2 * kAP], ky);
                gs[i] = acc;
            }
            n.eval(gs, rho0, Fx, Fy, a.c.half_h);
        }
        f2 lS[9];
        {
            const Around<UNI> m = around(c + 1, r + 2);
            const f2 ndt = bc(-a.c.dt);
            lS[0] = bc(0.f);
#pragma unroll
            for (int i = 1; i < 9; ++i) lS[i] = mul2(ndt, gather<kAP>(sm.L[i - 1], o, i, sm.L[i - 1][o], m));
        }
        Moments V;
        V.set(lS);
        f2 d0, d1, d2, lin[9];
        fBx = fBy = bc(0.f);
        const Moments B = scaled(bc(a.c.b_star), V);
        n.vjp(B, scaled(bc(a.c.c_star), V), Fx, Fy, a.c.half_h, d0, d1, d2, fBx, fBy);
        linear(add2(B.m0, d0), add2(B.x3, d1), add2(B.y3, d2), lin);
        const f2 keep = bc(1.f - a.c.b_star);
#pragma unroll
        for (int i = 0; i < 9; ++i) lg[i] = fma2(keep, lS[i], lin[i]);
#pragma unroll
        for (int i = 1; i < 9; ++i) sm.G[i - 1][r * kBP + c] = lg[i];
    }

    __device__ __forceinline__ void run()
    {
        const int p = t % kTP, r = t / kTP;
        size_t g0, g1;
        site(p + 2, r + 4, g0, g1);
        if (t < 2 * kAP) sm.mx[t] = __ldg(a.mx + axis_index(x0 - 4 + t, a.nx, false));
        else if (t < 2 * kAP + kAR) sm.my[t - 2 * kAP] = __ldg(a.my + axis_index(y0 - 4 + t - 2 * kAP, a.ny, false));
        chain_wait();
        {
            int c, rr;
            size_t h0, h1;
            fetch((r + 4) * kAP + p + 2, g0, g1);
            ring_site<4>(min(t, kARing - 1), c, rr);
            site(c, rr, h0, h1);
            if (t < kARing) fetch(rr * kAP + c, h0, h1);
            f2 g[9], k[9], Fx = bc(0.f), Fy = bc(0.f), Hx = bc(0.f), Hy = bc(0.f);
            load_g(g0, g1, g);
            if (FORCE) {
                Fx = pair(a.force, g0, g1);
                Fy = pair(a.force + a.plane, g0, g1);
            }
            if (t < kARing) {
                load_g(h0, h1, k);
                if (FORCE) {
                    Hx = pair(a.force, h0, h1);
                    Hy = pair(a.force + a.plane, h0, h1);
                }
            }
            stage_a((r + 4) * kAP + p + 2, g, Fx, Fy);
            if (t < kARing) stage_a(rr * kAP + c, k, Hx, Hy);
        }
        asm volatile("cp.async.wait_all;" ::: "memory");
        __syncthreads();
        f2 lg0, fBx, fBy;
        {
            f2 lg[9];
            stage_b(p + 1, r + 2, lg, fBx, fBy);
            lg0 = lg[0];
        }
        if (t < kBRing) {
            int c, rr;
            ring_site<2>(t, c, rr);
            f2 lg[9], ux, uy;
            stage_b(c, rr, lg, ux, uy);
        }
        // ---------------------------------------------------------------- C'
        const int x = x0 + 2 * p, y = y0 + r, oA = (r + 4) * kAP + p + 2, oB = (r + 2) * kBP + p + 1;
        const bool lo = y < a.ny && x < a.nx, hi = y < a.ny && x + 1 < a.nx;
        f2 lP[9], lQ[9], g[9];
        // in flight over the barrier and the gathers
        lQ[0] = pair(q.lam_next, g0, g1);
        load_g(g0, g1, g);
        double *d = q.dforce + (size_t)y * a.nx + x;
        const size_t N = (size_t)a.nx * a.ny;
        double df0 = 0.0, df1 = 0.0, df2 = 0.0, df3 = 0.0;
        if (q.dforce && lo) {
            df0 = d[0];
            df1 = d[N];
        }
        if (q.dforce && hi) {
            df2 = d[1];
            df3 = d[N + 1];
        }
        __syncthreads();
        {
            const Around<UNI> m = around(p + 2, r + 4);
            const f2 nh = bc(-a.c.h);
            lP[0] = lg0;
#pragma unroll
            for (int i = 1; i < 9; ++i) {
                const f2 v0 = sm.G[i - 1][oB];
                lP[i] = fma2(nh, gather<kBP>(sm.G[i - 1], oB, i, v0, m), v0);
                lQ[i] = sm.L[i - 1][oA];
            }
        }
        f2 Fx = bc(0.f), Fy = bc(0.f);
        if (FORCE) {
            Fx = sm.F[0][oA];
            Fy = sm.F[1][oA];
        }
        NodeVjp n;
        n.eval(g, rho0, Fx, Fy, a.c.half_dt);
        Moments VP, VQ;
        VP.set(lP);
        VQ.set(lQ);
        f2 d0, d1, d2, lFx = bc(0.f), lFy = bc(0.f);
        const f2 bP = bc(a.c.b_bar), bQ = bc(a.c.b_til);
        n.vjp(combine(bP, VP, bQ, VQ), combine(bc(a.c.c_bar), VP, bc(a.c.c_til), VQ), Fx, Fy, a.c.half_dt, d0, d1, d2,
              lFx, lFy);
        {
            // lam = lQ + b~ (c0 + xi.c - lQ) for the moments of lQ, and the smaller
            // terms: (1 - b) lP + b (moments of lP), those in u and F
            f2 lin[9], rest[9];
            linear(VQ.m0, VQ.x3, VQ.y3, lin);
            linear(fma2(bP, VP.m0, d0), fma2(bP, VP.x3, d1), fma2(bP, VP.y3, d2), rest);
            const f2 kP = bc(1.f - a.c.b_bar);
#pragma unroll
            for (int i = 0; i < 9; ++i)
                lP[i] = add2(lQ[i], fma2(bQ, sub2(lin[i], lQ[i]), fma2(kP, lP[i], rest[i])));
        }
        float *dst = q.lam_prev + (size_t)y * a.pitch + x;
        if (lo && hi) {
#pragma unroll
            for (int i = 0; i < 9; ++i) *reinterpret_cast<f2 *>(dst + i * a.plane) = lP[i];
        } else if (lo) {
#pragma unroll
            for (int i = 0; i < 9; ++i) dst[i * a.plane] = lP[i].x;
        }
        if (q.dforce) {
            if (lo) {
                d[0] = df0 + (double(lFx.x) + double(fBx.x));
                d[N] = df1 + (double(lFy.x) + double(fBy.x));
            }
            if (hi) {
                d[1] = df2 + (double(lFx.y) + double(fBx.y));
                d[N + 1] = df3 + (double(lFy.y) + double(fBy.y));
            }
        }
    }
};

// TALL: a launch for the rows of tiles from row0 on.
template <bool FORCE, bool UNI, bool TALL>
__global__ void __launch_bounds__(kNT, 2) k_adj_tile(const __grid_constant__ AdjTileArgs q)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int by = blockIdx.y + (TALL ? q.row0 : 0);
    AdjTile<FORCE, UNI>(q, *reinterpret_cast<AdjSmem *>(smem_raw), blockIdx.x, by).run();
    chain_next();
}

}  // namespace

// Whether the kernel takes these buffers: it reads and writes column pairs (the
// rows of the storage layout keep a buffer's own alignment).
bool adjoint_tile_ok(const void *state, const void *lam_next, const void *lam_prev)
{
    return ((reinterpret_cast<uintptr_t>(state) | reinterpret_cast<uintptr_t>(lam_next) |
             reinterpret_cast<uintptr_t>(lam_prev)) & 7) == 0;
}

cudaError_t launch_adjoint_tile(const StepArgs<float> &a, bool uniform, const float *lam_next, float *lam_prev,
                                double *dforce, cudaStream_t s)
{
    AdjTileArgs q{a, lam_next, lam_prev, dforce, 0};
    const int tx = tiles_along(a.nx, false, kTX), ty = tiles_along(a.ny, false, kTY);
    auto kern = a.force ? (uniform ? k_adj_tile<true, true, false> : k_adj_tile<true, false, false>)
                        : (uniform ? k_adj_tile<false, true, false> : k_adj_tile<false, false, false>);
    if (ty > kMaxTileRows) kern = a.force ? k_adj_tile<true, false, true> : k_adj_tile<false, false, true>;
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(AdjSmem));
    if (e != cudaSuccess) return e;
    for (; q.row0 < ty && e == cudaSuccess; q.row0 += kMaxTileRows)
        e = chained_launch(kern, dim3(tx, std::min(ty - q.row0, kMaxTileRows)), kNT, sizeof(AdjSmem), s, q);
    return e;
}

}  // namespace fdlbm
