// D3Q19 update by warps that march along z, for domains of any size: the moment form of
// Eq. ACM2.0 (lwacm_core.cuh) with walls and forcing.
//
// A warp takes an item: a strip of 30 columns, a tile of four rows and a run of planes.
// Lane l holds column x0 + l - 1 (lanes 0 and 31 are the strip's neighbours) of the four
// rows and of the rows below and above them. Rows 1 and 3 of the tile are one FP32x2 pair,
// rows 2 and 4 the other, rows 0 and 5 (the neighbours, which only send) a third: every
// operation issues once for two nodes, and since rows 1 and 3 send up what rows 2 and 4
// receive (and those down what the first pair receives), half the exchange along y moves
// nothing at all. Each plane's link values are formed once (pre-combine, Eq. ACM2.0b(a))
// and handed on without shared memory or a barrier (stream, Eq. ACM2.0b(b)): along x by
// warp shuffles, along y within a lane's rows, along z through the sums of three planes,
// the oldest complete once the next plane has been read (post-combine, Eq. ACM2.0b(c)).
// The loads of the next plane are in flight meanwhile.
//
// What bounds it, FP32 256^3 (128 GLUPS, 131 us a step): instructions, 153 a node (85 of them
// FP32, most packed), issue slots 51% and the FMA pipe 58% busy with 16 warps a SM; DRAM 47%.
// Measured and left out: the next planes in a ring in shared memory by asynchronous copies
// (no waits for memory, but 180 instructions a node: 138 us), 20 warps at 96 registers (135
// us), 12 warps at 168 (141 us).
//
// Lanes read and write single elements, so no alignment of rows, planes or storage types
// is asked for, and a node's sums are formed in the same order whatever the item.
#include "dev_cache.h"
#include "launch.h"
#include "lwacm_core.cuh"
#include "rows2.cuh"

namespace lwacm {
namespace {

using rows2::add;
using rows2::bc;
using rows2::byte_at;
using rows2::fma;
using rows2::from_left;
using rows2::from_right;
using rows2::mul;
using rows2::sub;
using rows2::widen;
using F2 = float2;

constexpr int kStrip = 30;  // columns of a strip (lanes 1 to 30)
constexpr int kTile = 4;    // rows of a tile
constexpr int kWarps = 4;   // warps per CTA: tiles one above the other

struct Dom3 {
    int nx, ny, nz;
    long long fstride;
    float a;  // 1 - 6 nu
    // 4 nu, and -6 nu as am1 + am1l = -3/2 odd exactly: the links give a momentum j back 3/2 odd j and
    // the post-combine 1 + am1 of it, so that rounded apart every step changed the momentum (by 6e-8
    // of 6 nu: 3e-7 of u after 24 steps at nu = 0.06)
    float odd, am1, am1l;
    float g[3];       // constant acceleration (Eq. force)
    int forced;
    const float *field;  // per-node acceleration
    // half-way walls (Eqs. ACM2.0cccbb2 / ACM2.0ccccbb) on both ends of x, y, z; the top of the lid
    // axis (1 or 2) moves with the lid velocity; wall = 36 nu rho0
    int wx, wy, wz, lid_axis;
    float wall, lid[3];
};

enum { FIRST = 0, START = 1, MID = 2, LAST = 3 };

// the links with one c_y of two rows: s = the three with c_z = 0, t = their x-momentum,
// p / m the ones with c_z = +1 / -1
struct Send {
    F2 s, t, p, m;
};
// sums of a plane for two rows
struct Sum3 {
    F2 D, X, Y, Z;
};

template <typename T, bool FIELD, bool WALLS>
struct March3 {
    const T *in;
    T *out;
    const Dom3 &dm;
    long long plane;
    float odd;
    unsigned off, lo, hi;  // bytes to row y0 at the lane's column in a plane; to the rows below and above the tile
    bool st;
    // WALLS: the lane's column lies at an x wall; the tile's first / last row at a y wall
    bool e0 = false, eN = false, low = false, top = false, edge = false;

    __device__ __forceinline__ March3(const T *in_, T *out_, const Dom3 &dm_, int x0, int y0)
        : in(in_), out(out_), dm(dm_), plane((long long)dm_.nx * dm_.ny), odd(dm_.odd) {
        const int lane = threadIdx.x & 31, x = x0 + lane - 1;
        const unsigned xw = (unsigned)(x < 0 ? x + dm.nx : (x < dm.nx ? x : x % dm.nx)), nx = (unsigned)dm.nx;
        off = ((unsigned)y0 * nx + xw) * (unsigned)sizeof(T);
        lo = ((unsigned)(y0 > 0 ? y0 - 1 : dm.ny - 1) * nx + xw) * (unsigned)sizeof(T);
        hi = ((unsigned)(y0 + kTile < dm.ny ? y0 + kTile : 0) * nx + xw) * (unsigned)sizeof(T);
        st = lane >= 1 && lane <= kStrip && x < dm.nx;
        if (WALLS) {
            e0 = dm.wx && x == 0;
            eN = dm.wx && x == dm.nx - 1;
            edge = dm.wx && (x0 == 0 || x0 + kStrip >= dm.nx);
            low = dm.wy && y0 == 0;
            top = dm.wy && y0 + kTile == dm.ny;
        }
    }
    // from x - 1 / x + 1; nothing comes through a wall
    __device__ __forceinline__ F2 left(F2 v) const {
        const F2 t = from_left(v);
        return WALLS && e0 ? bc<F2>(0.f) : t;
    }
    __device__ __forceinline__ F2 right(F2 v) const {
        const F2 t = from_right(v);
        return WALLS && eN ? bc<F2>(0.f) : t;
    }

    struct Raw {
        T f[4][6];
    };
    // ordinary loads: the grid before may still write what this one reads until
    // griddepcontrol.wait (ldraw, rows2.cuh)
    __device__ __forceinline__ void load(int z, Raw &r) const {
        z = z < 0 ? z + dm.nz : (z >= dm.nz ? z - dm.nz : z);
#pragma unroll
        for (int f = 0; f < 4; ++f) {
            const T *p = in + (z * plane + f * dm.fstride);
            r.f[f][0] = *byte_at(p, lo);
#pragma unroll
            for (int j = 0; j < kTile; ++j) r.f[f][1 + j] = *byte_at(p + (long long)j * dm.nx, off);
            r.f[f][5] = *byte_at(p, hi);
        }
    }

    struct Node {
        // w K, K = d - 3/2 rho |u|^2, and w 9/2 rho of the axis (w = 1/18) and the diagonal links (1/36);
        // K itself is not kept (K / 3 of the rest link is 12 K2), which takes 116 registers instead
        // of 146 and so four CTAs a SM instead of three (384 x 256 x 256 178 us instead of 199)
        F2 u, v, w, rho, K1, K2, B1, B2;
    };
    __device__ __forceinline__ Node consts(F2 d, F2 u, F2 v, F2 w) const {
        Node n;
        n.u = u;
        n.v = v;
        n.w = w;
        n.rho = add(d, 1.f);
        const F2 K = fma(n.rho, mul(fma(u, u, fma(v, v, mul(w, w))), -1.5f), d);
        n.K2 = mul(K, 1.f / 36.f);
        n.K1 = add(n.K2, n.K2);
        n.B2 = mul(n.rho, 0.125f);
        n.B1 = add(n.B2, n.B2);
        return n;
    }
    // w (K + 9/2 rho e^2) +- w rho s e; with t = w 9/2 rho e the odd part is (2 s / 9) t
    __device__ __forceinline__ void pair(const Node &n, F2 e, bool dg, F2 &gp, F2 &gm) const {
        const F2 t = mul(dg ? n.B2 : n.B1, e), c = fma(t, e, dg ? n.K2 : n.K1);
        gp = fma(odd, t, c);
        gm = fma(-odd, t, c);
    }
    __device__ __forceinline__ F2 plus(const Node &n, F2 e, bool dg) const {
        const F2 t = mul(dg ? n.B2 : n.B1, e);
        return fma(odd, t, fma(t, e, dg ? n.K2 : n.K1));
    }

    // the in-row links and the own terms of two rows (plane behind P, own C, ahead N)
    template <int MODE>
    __device__ __forceinline__ void in_row(const Node &n, F2 d, Sum3 &P, Sum3 &C, Sum3 &N, F2 gx, F2 gy, F2 gz) const {
        constexpr bool OWN = MODE == START || MODE == MID, DOWN = MODE == MID || MODE == LAST, UP = MODE != LAST;
        F2 zp, zm, pp, mm, pm, mp;
        pair(n, n.w, false, zp, zm);
        pair(n, add(n.u, n.w), true, pp, mm);  // (1,0,1) (-1,0,-1)
        pair(n, sub(n.u, n.w), true, pm, mp);  // (1,0,-1) (-1,0,1)
        if (OWN) {
            F2 xp, xm;
            pair(n, n.u, false, xp, xm);
            const F2 l = left(xp), r = right(xm);
            const F2 m = add(fma(dm.a, d, bc<F2>(dm.am1l)), dm.am1);  // a rho u = u + m u (post_combine)
            C.Z = add(fma(m, n.w, C.D), n.w);           // so far every link came with c_z = +1
            C.X = add(fma(m, n.u, add(C.X, sub(l, r))), n.u);
            C.Y = add(fma(m, n.v, C.Y), n.v);
            C.D = fma(12.f, n.K2, add(C.D, add(l, r)));
            if (dm.forced) {  // Eq. force: the odd part of f^(e)(rho(x,t), g) adds rho g to j
                C.X = fma(dm.g[0], n.rho, C.X);
                C.Y = fma(dm.g[1], n.rho, C.Y);
                C.Z = fma(dm.g[2], n.rho, C.Z);
                if (FIELD) {
                    C.X = fma(n.rho, gx, C.X);
                    C.Y = fma(n.rho, gy, C.Y);
                    C.Z = fma(n.rho, gz, C.Z);
                }
            }
        }
        if (DOWN) {
            const F2 l = left(pm), r = right(mm), s = add(zm, add(l, r));
            P.D = add(P.D, s);
            P.X = add(P.X, sub(l, r));
            P.Z = sub(P.Z, s);
        }
        if (UP) {
            const F2 l = left(pp), r = right(mp);
            N.D = add(zp, add(l, r));
            N.X = sub(l, r);
        }
    }
    template <int MODE>
    __device__ __forceinline__ void to_rows(const Node &n, Send &up, Send &dn) const {
        if (MODE == START || MODE == MID) {
            F2 yp, ym, pp, mm, pm, mp;
            pair(n, n.v, false, yp, ym);
            pair(n, add(n.u, n.v), true, pp, mm);  // (1,1,0) (-1,-1,0)
            pair(n, sub(n.u, n.v), true, pm, mp);  // (1,-1,0) (-1,1,0)
            F2 l = left(pp), r = right(mp);
            up.s = add(yp, add(l, r));
            up.t = sub(l, r);
            l = left(pm), r = right(mm);
            dn.s = add(ym, add(l, r));
            dn.t = sub(l, r);
        }
        pair(n, add(n.v, n.w), true, up.p, dn.m);  // (0,1,1) (0,-1,-1)
        pair(n, sub(n.v, n.w), true, up.m, dn.p);  // (0,1,-1) (0,-1,1)
    }
    // rows 0 (up) and 5 (down, its v negated): what they send to the tile
    template <int MODE>
    __device__ __forceinline__ void halo(const Node &n, Send &h) const {
        if (MODE == START || MODE == MID) {
            const F2 l = left(plus(n, add(n.v, n.u), true)), r = right(plus(n, sub(n.v, n.u), true));
            h.s = add(plus(n, n.v, false), add(l, r));
            h.t = sub(l, r);
        }
        if (MODE != LAST) h.p = plus(n, add(n.v, n.w), true);
        if (MODE == MID || MODE == LAST) h.m = plus(n, sub(n.v, n.w), true);
        if (WALLS && low) h.s.x = h.t.x = h.p.x = h.m.x = 0.f;
        if (WALLS && top) h.s.y = h.t.y = h.p.y = h.m.y = 0.f;
    }
    // WALLS: what the walls send back to plane z of the row pair k (tile rows k and k + 2): for each
    // link whose source lies beyond a wall the node's own value of the opposite link, plus the lid
    // term at the top of the lid axis; a link that leaves through two walls is taken at the z wall,
    // else at the y wall
    __device__ __forceinline__ void bounce(const Node &n, int k, int z, Sum3 &C) const {
        const bool z0 = dm.wz && z == 0, zN = dm.wz && z == dm.nz - 1;
        const bool y0 = low && k == 0, yN = top && k == 1;  // the pair's first / second row
        if (!(z0 || zN || y0 || yN || edge)) return;
        F2 zp, zm, xzp, xzm, zxp, zxm, yzp, yzm, zyp, zym;
        pair(n, add(n.u, n.w), true, xzp, xzm);  // (1,0,1) (-1,0,-1)
        pair(n, sub(n.u, n.w), true, zxp, zxm);  // (1,0,-1) (-1,0,1)
        pair(n, add(n.v, n.w), true, yzp, yzm);  // (0,1,1) (0,-1,-1)
        pair(n, sub(n.v, n.w), true, zyp, zym);  // (0,1,-1) (0,-1,1)
        if (z0 || zN) pair(n, n.w, false, zp, zm);
        if (z0) {
            const F2 s = add(zm, add(add(xzm, zxp), add(yzm, zyp)));
            C.D = add(C.D, s);
            C.Z = add(C.Z, s);
            C.X = add(C.X, sub(xzm, zxp));
            C.Y = add(C.Y, sub(yzm, zyp));
        }
        if (zN) {
            const float w = dm.lid_axis == 2 ? dm.wall * (1.f / 36.f) : 0.f;
            const F2 a = add(zp, -2.f * w * dm.lid[2]);
            const F2 b = add(zxm, w * (dm.lid[0] - dm.lid[2])), c = add(xzp, w * (-dm.lid[0] - dm.lid[2]));
            const F2 d = add(zym, w * (dm.lid[1] - dm.lid[2])), e = add(yzp, w * (-dm.lid[1] - dm.lid[2]));
            const F2 s = add(a, add(add(b, c), add(d, e)));
            C.D = add(C.D, s);
            C.Z = sub(C.Z, s);
            C.X = add(C.X, sub(b, c));
            C.Y = add(C.Y, sub(d, e));
        }
        F2 yp, ym, xyp, xym, yxp, yxm;
        if (y0 || yN || edge) {
            pair(n, n.v, false, yp, ym);
            pair(n, add(n.u, n.v), true, xyp, xym);  // (1,1,0) (-1,-1,0)
            pair(n, sub(n.u, n.v), true, yxp, yxm);  // (1,-1,0) (-1,1,0)
        }
        if (y0) {
            const float b = z0 ? 0.f : yzm.x, c = zN ? 0.f : zym.x, s = ym.x + (xym.x + yxp.x) + (b + c);
            C.D.x += s;
            C.Y.x += s;
            C.X.x += xym.x - yxp.x;
            C.Z.x += b - c;
        }
        if (yN) {
            const float w = dm.lid_axis == 1 ? dm.wall * (1.f / 36.f) : 0.f;
            const float a = yp.y - 2.f * w * dm.lid[1];
            const float b = yxm.y + w * (dm.lid[0] - dm.lid[1]), c = xyp.y + w * (-dm.lid[0] - dm.lid[1]);
            const float d = z0 ? 0.f : zyp.y + w * (dm.lid[2] - dm.lid[1]);
            const float e = zN ? 0.f : yzp.y + w * (-dm.lid[2] - dm.lid[1]);
            const float s = a + (b + c) + (d + e);
            C.D.y += s;
            C.Y.y -= s;
            C.X.y += b - c;
            C.Z.y += d - e;
        }
        if (edge) {
            F2 xp, xm;
            pair(n, n.u, false, xp, xm);
            if (e0 || eN) {
                const F2 zero = bc<F2>(0.f), a = e0 ? xm : xp;
                F2 b = e0 ? xzm : zxp, c = e0 ? zxm : xzp, d = e0 ? xym : yxp, e = e0 ? yxm : xyp;
                if (z0) b = zero;
                if (zN) c = zero;
                if (y0) d.x = 0.f;
                if (yN) e.y = 0.f;
                const F2 s = add(a, add(add(b, c), add(d, e)));
                C.D = add(C.D, s);
                C.X = e0 ? add(C.X, s) : sub(C.X, s);
                C.Z = add(C.Z, sub(b, c));
                C.Y = add(C.Y, sub(d, e));
            }
        }
    }
    template <int MODE>
    __device__ __forceinline__ void receive(const Send &up, const Send &dn, Sum3 &P, Sum3 &C, Sum3 &N) const {
        if (MODE == START || MODE == MID) {
            C.D = add(C.D, add(up.s, dn.s));
            C.X = add(C.X, add(up.t, dn.t));
            C.Y = add(C.Y, sub(up.s, dn.s));
        }
        if (MODE == MID || MODE == LAST) {
            const F2 s = add(up.m, dn.m);
            P.D = add(P.D, s);
            P.Y = add(P.Y, sub(up.m, dn.m));
            P.Z = sub(P.Z, s);
        }
        if (MODE != LAST) {
            N.D = add(N.D, add(up.p, dn.p));
            N.Y = sub(up.p, dn.p);
        }
    }
    // the finished plane z: density and, as the IEEE quotient, the velocity (branch-free for the
    // values of a flow, CUDA's division for any other, as velocity() of rows2.cuh)
    __device__ __forceinline__ void finish(int z, const Sum3 (&P)[2]) const {
        F2 b[2], f[2][4];
        float jm = 0.f;
#pragma unroll
        for (int p = 0; p < 2; ++p) {
            b[p] = add(P[p].D, 1.f);
            f[p][0] = P[p].D;
            const F2 j[3] = {P[p].X, P[p].Y, P[p].Z};
#pragma unroll
            for (int c = 0; c < 3; ++c) jm = fmaxf(jm, fmaxf(fabsf(j[c].x), fabsf(j[c].y)));
        }
        const float least = fminf(fminf(b[0].x, b[0].y), fminf(b[1].x, b[1].y));
        const float most = fmaxf(fmaxf(b[0].x, b[0].y), fmaxf(b[1].x, b[1].y));
        if (least >= 0.25f && most <= 4.f && jm <= 1e30f) {
#pragma unroll
            for (int p = 0; p < 2; ++p) {
                const tile::Div2 q = tile::div_prep2(b[p]);
                f[p][1] = tile::div_apply2(P[p].X, q);
                f[p][2] = tile::div_apply2(P[p].Y, q);
                f[p][3] = tile::div_apply2(P[p].Z, q);
            }
        } else {
#pragma unroll
            for (int p = 0; p < 2; ++p) {
                f[p][1] = rows2::quotient(P[p].X, b[p]);
                f[p][2] = rows2::quotient(P[p].Y, b[p]);
                f[p][3] = rows2::quotient(P[p].Z, b[p]);
            }
        }
        if (st)
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                T *o = out + (z * plane + k * dm.fstride);
                const long long nx = dm.nx;
                stf(byte_at(o, off), f[0][k].x);
                stf(byte_at(o + nx, off), f[1][k].x);
                stf(byte_at(o + 2 * nx, off), f[0][k].y);
                stf(byte_at(o + 3 * nx, off), f[1][k].y);
            }
    }

    // source plane z: completes the plane behind (P, stored), adds to its own (C) and leaves
    // the first sums of the plane ahead in P
    template <int MODE>
    __device__ __forceinline__ void source(int z, Raw &r, Sum3 (&P)[2], Sum3 (&C)[2], bool more) const {
        const F2 d0 = make_float2(widen(r.f[0][1]), widen(r.f[0][3])), d1 = make_float2(widen(r.f[0][2]), widen(r.f[0][4]));
        const Node n0 = consts(d0, make_float2(widen(r.f[1][1]), widen(r.f[1][3])),
                               make_float2(widen(r.f[2][1]), widen(r.f[2][3])),
                               make_float2(widen(r.f[3][1]), widen(r.f[3][3])));
        const Node n1 = consts(d1, make_float2(widen(r.f[1][2]), widen(r.f[1][4])),
                               make_float2(widen(r.f[2][2]), widen(r.f[2][4])),
                               make_float2(widen(r.f[3][2]), widen(r.f[3][4])));
        const Node nh = consts(make_float2(widen(r.f[0][0]), widen(r.f[0][5])),
                               make_float2(widen(r.f[1][0]), widen(r.f[1][5])),
                               make_float2(widen(r.f[2][0]), -widen(r.f[2][5])),
                               make_float2(widen(r.f[3][0]), widen(r.f[3][5])));
        if (more) load(z + 1, r);
        F2 g[2][3];
        if (FIELD && (MODE == START || MODE == MID)) {
            constexpr unsigned K = 4 / sizeof(T);  // the field is FP32 whatever the storage
#pragma unroll
            for (int c = 0; c < 3; ++c) {
                const float *q = dm.field + (z * plane + c * dm.fstride);
                const long long nx = dm.nx;
                g[0][c] = make_float2(*byte_at(q, off * K), *byte_at(q + 2 * nx, off * K));
                g[1][c] = make_float2(*byte_at(q + nx, off * K), *byte_at(q + 3 * nx, off * K));
            }
        }
        Sum3 N[2];
        in_row<MODE>(n0, d0, P[0], C[0], N[0], g[0][0], g[0][1], g[0][2]);
        in_row<MODE>(n1, d1, P[1], C[1], N[1], g[1][0], g[1][1], g[1][2]);
        if (WALLS && (MODE == START || MODE == MID)) {
            bounce(n0, 0, z, C[0]);
            bounce(n1, 1, z, C[1]);
        }
        Send up0, dn0, up1, dn1, h;
        halo<MODE>(nh, h);
        to_rows<MODE>(n0, up0, dn0);
        to_rows<MODE>(n1, up1, dn1);
        // rows 1, 3 receive from below (rows 0, 2) and above (2, 4); rows 2, 4 from (1, 3) and (3, 5)
        auto lo = [](F2 a, F2 b) { return make_float2(a.x, b.x); };
        auto hi = [](F2 a, F2 b) { return make_float2(a.y, b.y); };
        const Send ua = {lo(h.s, up1.s), lo(h.t, up1.t), lo(h.p, up1.p), lo(h.m, up1.m)};
        const Send db = {hi(dn0.s, h.s), hi(dn0.t, h.t), hi(dn0.p, h.p), hi(dn0.m, h.m)};
        receive<MODE>(ua, dn1, P[0], C[0], N[0]);
        receive<MODE>(up0, db, P[1], C[1], N[1]);
        if (MODE == MID || MODE == LAST) {
            finish(z - 1, P);
        }
        if (MODE != LAST) {
            P[0] = N[0];
            P[1] = N[1];
        }
    }

    __device__ __forceinline__ void planes(int za, int zb) const {
        Raw r;
        Sum3 pa[2], pb[2];
        const bool floor = WALLS && dm.wz && za == 0, roof = WALLS && dm.wz && zb == dm.nz;
        if (floor) {  // nothing comes through a z wall
#pragma unroll
            for (int p = 0; p < 2; ++p) pa[p].D = pa[p].X = pa[p].Y = bc<F2>(0.f);
            load(za, r);
        } else {
            load(za - 1, r);
            source<FIRST>(za - 1, r, pa, pb, true);
        }
        source<START>(za, r, pb, pa, true);
        int z = za + 1;
        for (; z + 1 < zb; z += 2) {
            source<MID>(z, r, pa, pb, true);
            source<MID>(z + 1, r, pb, pa, true);
        }
        if (z < zb) {
            source<MID>(z, r, pa, pb, true);
            if (roof)
                finish(z, pb);
            else
                source<LAST>(z + 1, r, pb, pa, false);
        } else if (roof) {
            finish(z - 1, pa);
        } else {
            source<LAST>(z, r, pa, pb, false);
        }
    }
};

// items numbered strips first, then groups of kWarps tiles, then runs of planes, so that
// the neighbours of a strip pass each plane together and share its lines in L2 (runs of
// equal length that cross from column to column, out of step, took 235 us on 256^3)
template <typename T, bool FIELD, bool WALLS>
__global__ void __launch_bounds__(32 * kWarps) k_d3q19_rows(const T *in, T *out, Dom3 dm, int strips, int groups, int runs) {
    // the next step's CTAs may take their SMs as this step's leave them; none touches
    // global memory before this grid is complete
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    const int rest = (int)(blockIdx.x / (unsigned)strips), strip = (int)blockIdx.x - rest * strips;
    const int run = rest / groups, group = rest - run * groups;
    int y0 = (group * kWarps + (int)(threadIdx.x >> 5)) * kTile;
    if (y0 >= dm.ny) return;
    // the last tile ends with the domain: rows that two tiles update get the same values twice
    y0 = min(y0, dm.ny - kTile);
    const March3<T, FIELD, WALLS> m(in, out, dm, strip * kStrip, y0);
    asm volatile("griddepcontrol.wait;" ::: "memory");
    m.planes((int)((long long)dm.nz * run / runs), (int)((long long)dm.nz * (run + 1) / runs));
}

// CTAs of the kernel that the GPU holds (-1 when it cannot be determined)
template <typename T, bool FIELD, bool WALLS>
int room() {
    static DevSlots cap;
    return per_device(cap, [] {
        int per = 0;
        if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, k_d3q19_rows<T, FIELD, WALLS>, 32 * kWarps, 0) !=
                cudaSuccess || per < 1)
            return -1;
        return per * device_sms();
    });
}

// Runs of planes per column: `cols` columns of nz planes on a GPU that holds `room` CTAs.
// The least planes on the busiest place, a run costing 1.3 planes more than its own (its two
// neighbours, each in part), one wave counted 4% dearer (CTAs that follow each other even out:
// 256^3 in runs of 64 planes, one wave, 133.8 us, of 32 planes 129.3, of 16 129.2).
int plan_runs(long long cols, int nz, int room) {
    int best = 1;
    double least = 1e300;
    for (int r = 1; r <= nz && (r == 1 || cols * r <= 4LL * room); ++r) {
        const long long waves = (cols * r + room - 1) / room;
        const double c = (double)waves * ((nz + r - 1) / r + 1.3) * (waves == 1 ? 1.04 : 1.0);
        if (c < least - 1e-9) {
            least = c;
            best = r;
        }
    }
    return best;
}

template <typename T, bool FIELD, bool WALLS>
cudaError_t launch_t(const void *in, void *out, const Dom3 &dm, int strips, int groups, int runs, cudaStream_t st) {
    const long long ctas = (long long)strips * groups * runs;
    if (ctas > 0x7fffffffLL) return cudaErrorInvalidValue;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)ctas);
    cfg.blockDim = dim3(32 * kWarps);
    cfg.stream = st;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, k_d3q19_rows<T, FIELD, WALLS>, (const T *)in, (T *)out, dm, strips, groups, runs);
}

template <typename T, bool FIELD, bool WALLS>
cudaError_t launch_t(const void *in, void *out, const StepParams &p, cudaStream_t st) {
    const int places = room<T, FIELD, WALLS>();
    if (places < 1) return cudaErrorNotSupported;
    Dom3 dm;
    dm.nx = p.nx;
    dm.ny = p.ny;
    dm.nz = p.nz;
    dm.fstride = p.fstride;
    dm.a = p.a;
    dm.odd = p.s * (2.f / 9.f);
    dm.am1 = -1.5f * dm.odd;
    dm.am1l = (float)(-1.5 * (double)dm.odd - (double)dm.am1);
    for (int c = 0; c < 3; ++c) dm.g[c] = p.has_force ? p.force[c] : 0.f;
    dm.forced = p.has_force || p.gfield;
    dm.field = p.gfield;
    dm.wx = p.walled[0];
    dm.wy = p.walled[1];
    dm.wz = p.walled[2];
    dm.lid_axis = p.lid_axis;
    dm.wall = p.wallc;
    for (int c = 0; c < 3; ++c) dm.lid[c] = p.lid[c];
    const int strips = (p.nx - 1) / kStrip + 1, groups = (p.ny - 1) / (kTile * kWarps) + 1;
    return launch_t<T, FIELD, WALLS>(in, out, dm, strips, groups, plan_runs((long long)strips * groups, p.nz, places), st);
}

}  // namespace

int rows3d_runs(long long cols, int nz, int room) { return plan_runs(cols, nz, room); }

bool rows3d_supported(const StepParams &p) {
    // a whole tile; a byte offset within a plane fits 32 bits; the plain scheme
    return p.ny >= kTile && (long long)p.nx * p.ny < (1LL << 30) && p.sdelta == 0.f && !p.scalar && !p.bulk;
}

// Whether the march takes less than the gather (with the scalar: its two kernels less than the
// gather's one). A warp works on 30 columns and a CTA on 16 rows whatever the domain has, so a
// narrow one pays for `slots` nodes and a gather only for its own: picoseconds a step, fitted to 200
// shapes of 1 to 95 columns and 5 to 1000 rows (us a step, gather / march: 2 x 256 x 256 8.4 /
// 15.5, 4 x 256 x 256 13.7 / 15.5, 5 x 256 x 256 16.3 / 15.5, 6 x 6 x 10000 18.1 / 33.8, 14 x 6 x
// 10000 36.4 / 33.8, 1 x 64 x 64 4.7 / 3.6; with the scalar 4 x 256 x 256 15.3 / 28.0, 8 x 256 x 256
// 27.6 / 28.1, 2 x 24 x 24 5.4 / 5.1). The gather of a walled domain has the wall pass after it, the
// march not (a channel of 2 x 256 x 256 15.4 / 19.8, of 4 x 256 x 256 19.8 / 20.0, of 8 x 6 x 10000
// 34.7 / 41.9; a cavity of 3 x 256 x 256 20.1 / 23.1, of 6 x 6 x 10000 76.7 / 50.1).
bool rows3d_pays(const StepParams &p) {
    const double n = (double)p.N, cols = (double)((p.nx - 1) / kStrip + 1) * kStrip;
    const double slots = cols * ((p.ny - 1) / (kTile * kWarps) + 1) * (kTile * kWarps) * p.nz;
    if (p.scalar) return 13.0 * cols * ((p.ny - 1) / kTile + 1) * kTile * p.nz < 45.0 * n + 0.4e6;
    if (rows3d_walls(p))
        return (p.bc == BC_CAVITY ? 11.0 * slots - 2000.0 * n / p.ny : 9.0 * slots - 140.0 * n / p.ny) <
               38.0 * n + 9.5e6;
    return (p.gfield ? 8.0 : 7.0) * slots < 38.0 * n + 2.8e6;
}

// Walls applied in the kernel (no wall pass after it), without a force field, up to 2^20 nodes:
// the bounces take registers (232: two CTAs a SM instead of four) and instructions in every
// boundary warp, a wall pass 5 to 8 us a step (kernel and pass / walls in the kernel: the 60^3
// cavity 9.7 / 5.2, 125 x 74 x 37 11.1 / 8.1, 100^3 18.6 / 18.1, 200^3 81 / 104).
bool rows3d_walls(const StepParams &p) {
    return p.bc != BC_PERIODIC && !p.gfield && p.N <= (1LL << 20) && rows3d_supported(p);
}

template <typename T>
static cudaError_t rows3d_t(const void *in, void *out, const StepParams &p, cudaStream_t st) {
    if (p.gfield) return launch_t<T, true, false>(in, out, p, st);
    return rows3d_walls(p) ? launch_t<T, false, true>(in, out, p, st) : launch_t<T, false, false>(in, out, p, st);
}

cudaError_t launch_step_rows3d(int storage, const void *in, void *out, const StepParams &p, cudaStream_t st) {
    switch (storage) {
        case STORE_F32: return rows3d_t<float>(in, out, p, st);
        case STORE_BF16: return rows3d_t<__nv_bfloat16>(in, out, p, st);
        case STORE_F16: return rows3d_t<__half>(in, out, p, st);
    }
    return cudaErrorInvalidValue;
}

}  // namespace lwacm
