// The D2Q9 update of a strip of columns and a run of rows by one warp, shared by the
// single-domain kernel (kernels_rows2.cu) and the ensemble kernels
// (kernels_batch.cu).
#pragma once

#include "lwacm_core.cuh"
#include "tile_common.cuh"

namespace lwacm {
namespace rows2 {

using F2 = float2;

constexpr int kHalf = 30;  // columns of a strip (lanes 1 to 30)

// one D2Q9 domain: its node (0,0) at packed index base; s = 18 nu, a = 1 - 6 nu
struct Dom2 {
    int nx, ny;
    long long base, fstride;
    float s, a;
};
// half-way walls (Eqs. ACM2.0cccbb2 / ACM2.0ccccbb) on both ends of x / y; the top y
// wall moves with the lid velocity
struct Walls2 {
    int wx, wy;
    float wallc;       // 36 nu rho0
    float lidx, lidy;
};
// forcing (Eq. force): rho(x,t) (g + g(x)) added to j, g(x) two FP32 fields
struct Force2 {
    int on;
    float gx, gy;
    const float *field;
};

constexpr int kMaxWarps = 16;  // per CTA (one strip a warp; one warp with two strips)
// warps of a CTA of the one-strip form: the strips of a row in as few CTAs as possible
inline int cta_warps(int nx) {
    const int s = (nx - 1) / kHalf + 1, parts = (s - 1) / kMaxWarps + 1;
    return (s - 1) / parts + 1;
}
// How a domain is cut: strips per warp and rows per item, given the warps the GPU holds
// of each form (room1, room2).
//
// An item reads two rows more than it updates, and a warp alone takes 0.2 to 0.25 us (one
// strip) or 0.3 to 0.4 us (two) a row, so short items win until the GPU is full, and then
// whole waves of items: the best rows per item measured over 256^2 to 2048^2 (plain,
// cavity, bulk viscosity) are those that fill the GPU just once, one strip a warp up to 5
// rows (724^2: 5 rows 4.2 us, two strips 4.7; 1024^2: 8 rows 7.3, two strips 6.5), two up
// to 8 (1024^2: 6 rows 6.5, 4 rows 7.3; the cavity 8 rows 7.4, 6 rows 8.9). Larger domains
// take 8 to 16 rows, whichever wastes least of the last wave (2048^2: 10 rows 18.1, 16 rows
// 19.5), 16 where there are more than 4 waves (4096^2: 70.8, 64 rows 84) and 32 where there
// are more than 9 (8192^2: 262, 24 rows 266). Two strips a warp only where they are mostly
// there: in domains of up to 30 columns the second one is empty (30 x 65536 nodes, one strip /
// two: 11.3 / 15.3, bulk viscosity 18.8 / 30.3, the 2D tiles 25.7; 1000 domains of 20 x 300
// 47.6 / 67.4).
struct Cut {
    int ns, rows;
};
// w1, w2: strips (of one, of two) times rows in all
inline Cut cut_rows(long long w1, long long w2, long long room1, long long room2) {
    const long long once1 = (w1 - 1) / room1 + 1, once2 = (w2 - 1) / room2 + 1;
    Cut c{1, (int)once1};
    if (once1 > 5) {
        const bool two = 4 * w2 <= 3 * w1;
        const long long w = two ? w2 : w1, room = two ? room2 : room1, once = two ? once2 : once1;
        c.ns = two ? 2 : 1;
        c.rows = 16;
        if (once <= 8)
            c.rows = (int)once;
        else if (w > 9 * 16 * room)
            c.rows = 32;
        else if (w <= 4 * 16 * room)
            for (int h = 16, best = 1 << 30; h >= 8; --h) {
                const int cost = (int)((w / h + room) / room) * (2 * h + 3);
                if (cost < best) best = cost, c.rows = h;
            }
    }
    return c;
}
inline Cut cut_domain(int nx, int ny, long long room1, long long room2) {
    Cut c = cut_rows((long long)((nx - 1) / kHalf + 1) * ny, (long long)((nx - 1) / (2 * kHalf) + 1) * ny, room1, room2);
    if (c.rows > ny) c.rows = ny;
    return c;
}

// ---- arithmetic on one node (float) or a pair of nodes (FP32x2): explicit roundings, so
// that both forms give a node the same values
template <int NS>
struct Pack;
template <>
struct Pack<1> {
    using F = float;
};
template <>
struct Pack<2> {
    using F = float2;
};
template <typename F>
__device__ __forceinline__ F bc(float v);
template <>
__device__ __forceinline__ float bc<float>(float v) { return v; }
template <>
__device__ __forceinline__ F2 bc<F2>(float v) { return make_float2(v, v); }
__device__ __forceinline__ float add(float a, float b) { return __fadd_rn(a, b); }
__device__ __forceinline__ float mul(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ float fma(float a, float b, float c) { return __fmaf_rn(a, b, c); }
__device__ __forceinline__ float sub(float a, float b) { return __fsub_rn(a, b); }
__device__ __forceinline__ F2 add(F2 a, F2 b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ F2 mul(F2 a, F2 b) { return __fmul2_rn(a, b); }
__device__ __forceinline__ F2 fma(F2 a, F2 b, F2 c) { return __ffma2_rn(a, b, c); }
__device__ __forceinline__ F2 sub(F2 a, F2 b) { return __ffma2_rn(b, make_float2(-1.f, -1.f), a); }
__device__ __forceinline__ float neg(float a) { return -a; }
__device__ __forceinline__ F2 neg(F2 a) { return make_float2(-a.x, -a.y); }
template <typename F>
__device__ __forceinline__ F add(F a, float b) { return add(a, bc<F>(b)); }
template <typename F>
__device__ __forceinline__ F mul(F a, float b) { return mul(a, bc<F>(b)); }
template <typename F>
__device__ __forceinline__ F fma(float a, F b, F c) { return fma(bc<F>(a), b, c); }
// the h-th node of a pack
__device__ __forceinline__ float &at(float &v, int) { return v; }
__device__ __forceinline__ float &at(F2 &v, int h) { return h ? v.y : v.x; }

// value from the neighbour at x - 1 / x + 1 (lane 0 / 31: unused)
__device__ __forceinline__ float from_left(float v) { return __shfl_up_sync(tile::FULL, v, 1); }
__device__ __forceinline__ float from_right(float v) { return __shfl_down_sync(tile::FULL, v, 1); }
__device__ __forceinline__ F2 from_left(F2 v) { return make_float2(from_left(v.x), from_left(v.y)); }
__device__ __forceinline__ F2 from_right(F2 v) { return make_float2(from_right(v.x), from_right(v.y)); }

// an element some bytes from a pointer that is uniform over the warp: a 32-bit offset of the
// lane's own costs no address arithmetic
template <typename T>
__device__ __forceinline__ T *byte_at(T *p, unsigned bytes) {
    return (T *)((char *)p + bytes);
}
template <typename T>
__device__ __forceinline__ const T *byte_at(const T *p, unsigned bytes) {
    return (const T *)((const char *)p + bytes);
}
// stored elements as loaded: widened when used, so that a load in flight holds nothing up.
// Ordinary loads and not __ldg: a grid launched with programmatic stream serialization is
// alive while the grid before it still writes what this one reads, and the read-only path is
// defined only for data that nobody writes during the kernel (griddepcontrol.wait orders
// ordinary loads). COHERENT: past L1, for what other CTAs of the same launch write.
template <bool COHERENT, typename T>
__device__ __forceinline__ T ldraw(const T *p) {
    return COHERENT ? __ldcg(p) : *p;
}
__device__ __forceinline__ float widen(float v) { return v; }
__device__ __forceinline__ float widen(__nv_bfloat16 v) { return __bfloat162float(v); }
__device__ __forceinline__ float widen(__half v) { return __half2float(v); }

// u = j / rho, the IEEE quotient: branch-free (tile_common.cuh, div_apply) for the
// values of a flow, CUDA's division for any other (a state that has blown up)
__device__ __forceinline__ void velocity(float rn, float X, float Y, float &u, float &v) {
    if (rn >= 0.25f && rn <= 4.f && fmaxf(fabsf(X), fabsf(Y)) <= 1e30f) {
        const tile::Div1 r = tile::div_prep(rn);
        u = tile::div_apply(X, r);
        v = tile::div_apply(Y, r);
    } else {
        u = X / rn;
        v = Y / rn;
    }
}
__device__ __forceinline__ void velocity(F2 rn, F2 X, F2 Y, F2 &u, F2 &v) {
    const float lo = fminf(rn.x, rn.y), hi = fmaxf(rn.x, rn.y);
    const float j = fmaxf(fmaxf(fabsf(X.x), fabsf(X.y)), fmaxf(fabsf(Y.x), fabsf(Y.y)));
    if (lo >= 0.25f && hi <= 4.f && j <= 1e30f) {
        const tile::Div2 r = tile::div_prep2(rn);
        u = tile::div_apply2(X, r);
        v = tile::div_apply2(Y, r);
    } else {
        u = make_float2(X.x / rn.x, X.y / rn.y);
        v = make_float2(Y.x / rn.x, Y.y / rn.y);
    }
}
__device__ __forceinline__ float quotient(float a, float b) { return a / b; }
__device__ __forceinline__ F2 quotient(F2 a, F2 b) { return make_float2(a.x / b.x, a.y / b.y); }

// What a row has received until its update is complete. Plain: the sums D, X, Y of the
// density and momentum; S the density term of omega_p. BULK: the values themselves, g3, g5,
// g8 the links with c_y = +1 from the row below, ax = g1 + g2 and dx = g1 - g2 of its own
// row, g0 its rest value, o0 .. o3 the density terms of omega_p. u, v, d its own fields.
template <typename F>
struct Part {
    F D, X, Y, S, u, v;
    F g3, g5, g8, ax, dx, d, g0, gx, gy, o0, o1, o2, o3;
};

// One source row of a march: FIRST sends to the row above only, START also adds to its
// own, MID completes the row below as well, LAST completes the row below only.
enum { FIRST = 0, START = 1, MID = 2, LAST = 3 };

// Rows [ya, yb) of the NS strips from column x0. Without WALLS every axis wraps.
//
// BULK (periodic): the source's equilibrium is the quasi-equilibrium f^(e*) of Appendix
// "Computing derivatives locally"; with h = gamma (Tr^(+) - Tr^(e)) / 2, P = Pxx + Pyy
// = |u|^2 + 2/3 and T = rho h (1 - a) / 4 the pre-combined increment of the pair (c, -c)
// with e = c.u is  axis: rho h (1 - P - h) / 2 -+ 2 T e;  diagonal: rho h (h + P) / 4
// +- T e;  rest: rho h (h - 2 + P). The node stores Tr^(+) - Tr^(e) = sum_i (|c_i|^2 -
// 2/3) g_i / rho_a - |u+|^2, rho_a the zeroth moment built with a.
// NUP (periodic; omega_p, Section 2.2 item 3): the density gains sdelta sum_i W_i(x -
// c_i), W_i = w_i rho e (the odd part with s_p = s + sdelta), and with BULK a third of the
// increment's odd part, -rho h / 2 (axis) or rho h / 4 (diagonal) times e.
template <int NS, typename T, bool COHERENT, bool WALLS, bool FIELD, bool BULK, bool NUP>
struct March {
    using F = typename Pack<NS>::F;
    using A = Part<F>;
    static constexpr int NF = BULK ? 4 : 3;
    struct Raw {
        T f[NF][NS];
        float g[FIELD ? 2 : 1][NS];
    };
    const T *in;
    T *out;
    const Dom2 &dm;
    const Walls2 &wl;
    const Force2 &fc;
    // The links give a momentum j back 3/2 odd j and the post-combine 1 + am1 of it: 3/2 odd + am1
    // has to vanish, or every step changes the momentum by the rest (rounded apart it was 6e-8 of
    // 6 nu, 3e-7 of u after 24 steps at nu = 0.06), so am1 + am1l is -3/2 odd exactly
    const float gamma, sdelta, nu, odd, am1, am1l;
    unsigned xo[NS];  // the lane's columns, wrapped
    bool st[NS], e0[NS], eN[NS];
    bool edge;  // the strips hold a column at an x wall

    __device__ __forceinline__ March(const T *in_, T *out_, const Dom2 &dm_, int x0, const Walls2 &wl_,
                                     const Force2 &fc_, float gamma_, float sdelta_)
        : in(in_ + dm_.base), out(out_ + dm_.base), dm(dm_), wl(wl_), fc(fc_), gamma(gamma_), sdelta(sdelta_),
          nu(dm_.s * (1.f / 18.f)), odd(dm_.s * (2.f / 9.f)),
          am1(BULK ? dm_.s * (-1.f / 3.f) : odd * -1.5f), am1l(fmaf(odd, -1.5f, -am1)) {
        const int lane = threadIdx.x & 31;
        edge = WALLS && wl.wx && (x0 == 0 || x0 + NS * kHalf >= dm.nx);
#pragma unroll
        for (int h = 0; h < NS; ++h) {
            const int x = x0 + h * kHalf + lane - 1;
            st[h] = lane >= 1 && lane <= kHalf && x < dm.nx;
            e0[h] = WALLS && wl.wx && x == 0;
            eN[h] = WALLS && wl.wx && x == dm.nx - 1;
            xo[h] = (unsigned)(x < 0 ? x + dm.nx : (x < dm.nx ? x : x % dm.nx));
        }
    }

    __device__ __forceinline__ void load(int y, Raw &r) const {
        if (WALLS && wl.wy)
            y = max(0, min(y, dm.ny - 1));
        else
            y = y < 0 ? y + dm.ny : (y >= dm.ny ? y - dm.ny : y);
        const long long row = (long long)y * dm.nx;
#pragma unroll
        for (int f = 0; f < NF; ++f)
#pragma unroll
            for (int h = 0; h < NS; ++h) r.f[f][h] = ldraw<COHERENT>(in + (row + f * dm.fstride) + xo[h]);
        if (FIELD)
#pragma unroll
            for (int f = 0; f < 2; ++f)
#pragma unroll
                for (int h = 0; h < NS; ++h) r.g[f][h] = fc.field[(row + f * dm.fstride) + xo[h]];
    }
    static __device__ __forceinline__ float pick(const T (&v)[1]) { return widen(v[0]); }
    static __device__ __forceinline__ F2 pick(const T (&v)[2]) { return make_float2(widen(v[0]), widen(v[1])); }
    static __device__ __forceinline__ float pickg(const float (&v)[1], float) { return v[0]; }
    static __device__ __forceinline__ F2 pickg(const float (&v)[2], F2) { return make_float2(v[0], v[1]); }

    __device__ __forceinline__ void store(int y, F D, F u, F v, F tr) const {
        T *o = out + (long long)y * dm.nx;
#pragma unroll
        for (int h = 0; h < NS; ++h)
            if (st[h]) {
                stf(o + xo[h], at(D, h));
                stf(o + dm.fstride + xo[h], at(u, h));
                stf(o + 2 * dm.fstride + xo[h], at(v, h));
                if (BULK) stf(o + 3 * dm.fstride + xo[h], at(tr, h));
            }
    }

    // Source row y with the fields r: completes the row below (P, stored), adds to its
    // own (C) and leaves the first sums of the row above in P. The fields of row y + 4 (up
    // to row yb) are loaded into r meanwhile. A row beyond a y wall holds the fields of the
    // wall's own row (load), whose opposite links it sends back.
    template <int MODE>
    __device__ __forceinline__ void source(int y, Raw &r, A &P, A &C, int yb) const {
        constexpr bool OWN = MODE == START || MODE == MID, DOWN = MODE == MID || MODE == LAST, UP = MODE != LAST;
        const F d = pick(r.f[0]), u = pick(r.f[1]), v = pick(r.f[2]);
        F gx = bc<F>(0.f), gy = bc<F>(0.f);
        if (FIELD) {
            gx = pickg(r.g[0], F{});
            gy = pickg(r.g[FIELD ? 1 : 0], F{});
        }
        const F rho = add(d, 1.f);
        const F K = fma(mul(rho, -1.5f), fma(u, u, mul(v, v)), d);  // d - 3/2 rho |u|^2
        if constexpr (BULK) {
            const F tr = pick(r.f[NF - 1]);
            if (MODE != LAST && y + 4 <= yb) load(y + 4, r);
            source_bulk<MODE>(y, d, u, v, rho, K, tr, gx, gy, P, C);
            return;
        }
        if (MODE != LAST && y + 4 <= yb) load(y + 4, r);
        const F k9 = mul(K, 1.f / 9.f), k36 = mul(K, 1.f / 36.f), b9 = mul(rho, 0.5f), b36 = mul(rho, 0.125f);
        F W[4];
        // w (K + 9/2 rho e^2) +- w rho s e; with t = b e, w rho s e = (2 s / 9) t
        auto pair = [&](int p, F e, bool dg, F &gp, F &gm) {
            const F t = mul(dg ? b36 : b9, e), c = fma(t, e, dg ? k36 : k9);
            gp = fma(odd, t, c);
            gm = fma(-odd, t, c);
            if (NUP) W[p] = mul(t, 2.f / 9.f);  // w rho e
        };
        F g1, g2, g3, g4, g5, g6, g7, g8;  // (1,0) (-1,0) (0,1) (0,-1) (1,1) (-1,-1) (1,-1) (-1,1)
        pair(0, u, false, g1, g2);
        pair(1, v, false, g3, g4);
        pair(2, add(u, v), true, g5, g6);
        pair(3, sub(u, v), true, g7, g8);
        // what arrives from the left (links with c_x = +1) and from the right
        F l1 = bc<F>(0.f), l5 = l1, l7 = l1, r2 = l1, r6 = l1, r8 = l1;
        if (OWN) l1 = from_left(g1), r2 = from_right(g2);
        if (UP) l5 = from_left(g5), r8 = from_right(g8);
        if (DOWN) l7 = from_left(g7), r6 = from_right(g6);
        if (WALLS && edge)
            // nothing comes through an x wall: a node there takes its own value of the
            // opposite link (the diagonal links below, with the row's own sums)
#pragma unroll
            for (int h = 0; h < NS; ++h) {
                if (e0[h]) at(l1, h) = at(g2, h), at(l5, h) = at(l7, h) = 0.f;
                if (eN[h]) at(r2, h) = at(g1, h), at(r6, h) = at(r8, h) = 0.f;
            }
        if (DOWN) {  // the row below: links with c_y = -1
            if (WALLS && wl.wy && y >= dm.ny) {  // bounced, from the moving wall
                g4 = add(g3, -(wl.wallc * (1.f / 9.f)) * wl.lidy);
                l7 = add(g8, (wl.wallc * (1.f / 36.f)) * (wl.lidx - wl.lidy));
                r6 = add(g5, (wl.wallc * (1.f / 36.f)) * (-wl.lidx - wl.lidy));
            }
            const F all = add(g4, add(l7, r6));
            F D = add(P.D, all);
            const F X = add(add(P.X, sub(l7, r6)), P.u), Y = add(sub(P.Y, all), P.v);
            if (NUP) {  // (-1,-1), (1,-1) and (0,-1), W_-c = -W_c
                const F w = sub(from_right(W[2]), from_left(W[3]));
                D = fma(sdelta, sub(P.S, add(w, W[1])), D);
            }
            F un, vn;
            velocity(add(D, 1.f), X, Y, un, vn);
            store(y - 1, D, un, vn, D);
        }
        if (OWN) {  // the row itself: rest and c_y = 0 links, and a rho u = u + m u (u added last)
            C.D = fma(4.f / 9.f, K, add(C.D, add(l1, r2)));
            if (NUP) C.S = add(C.S, sub(from_left(W[0]), from_right(W[0])));
            const F m = add(fma(dm.a, d, bc<F>(am1l)), am1);
            C.X = fma(m, u, add(C.X, sub(l1, r2)));
            C.Y = fma(m, v, C.Y);
            if (WALLS && edge) {  // the diagonal links (in a row at a y wall the row beyond it has them)
                const bool low = wl.wy && y == 0, top = wl.wy && y == dm.ny - 1;
#pragma unroll
                for (int h = 0; h < NS; ++h) {
                    float &D = at(C.D, h), &X = at(C.X, h), &Y = at(C.Y, h);
                    const float v5 = at(g5, h), v6 = at(g6, h), v7 = at(g7, h), v8 = at(g8, h);
                    if (e0[h] && !low) D += v6, X += v6, Y += v6;  // (1,1)
                    if (e0[h] && !top) D += v8, X += v8, Y -= v8;  // (1,-1)
                    if (eN[h] && !top) D += v5, X -= v5, Y -= v5;  // (-1,-1)
                    if (eN[h] && !low) D += v7, X -= v7, Y += v7;  // (-1,1)
                }
            }
            if (fc.on) {  // Eq. force: the odd part of f^(e)(rho(x,t), g) adds rho g to j
                C.X = fma(fc.gx, rho, C.X);
                C.Y = fma(fc.gy, rho, C.Y);
                if (FIELD) {
                    C.X = fma(rho, gx, C.X);
                    C.Y = fma(rho, gy, C.Y);
                }
            }
            C.u = u;
            C.v = v;
        }
        if (UP) {  // the row above: links with c_y = +1
            if (WALLS && wl.wy && y < 0) g3 = g4, l5 = g6, r8 = g7;  // bounced
            P.D = P.Y = add(g3, add(l5, r8));
            P.X = sub(l5, r8);
            if (NUP) P.S = add(W[1], sub(from_left(W[2]), from_right(W[3])));
        }
    }

    // The same for the bulk-viscosity variant, whose trace is the small difference of
    // large sums: the node's values are added in one order once all are there, as the
    // 2D-tile kernel adds them (bit for bit the same fields).
    template <int MODE>
    __device__ __forceinline__ void source_bulk(int y, F d, F u, F v, F rho, F K, F tr, F gx, F gy, A &P, A &C) const {
        constexpr bool OWN = MODE == START || MODE == MID, DOWN = MODE == MID || MODE == LAST, UP = MODE != LAST;
        const F k9 = mul(K, 1.f / 9.f), k36 = mul(K, 1.f / 36.f), b9 = mul(rho, 0.5f), b36 = mul(rho, 0.125f);
        const F h = mul(tr, 0.5f * gamma), rh = mul(rho, h), Pt = fma(u, u, fma(v, v, bc<F>(2.f / 3.f)));
        const F bax = mul(rh, 0.5f), bdg = mul(rh, 0.25f), cax = sub(sub(bc<F>(1.f), Pt), h), cdg = add(h, Pt);
        const F odg = mul(bdg, 1.f - dm.a), rn = mul(rho, nu);
        const F a9 = add(mul(rn, 2.f), mul(odg, -2.f)), a36 = add(mul(rn, 0.5f), odg);
        F w9, w36, W[4];
        if (NUP) {
            w9 = fma(1.f / 3.f, mul(rh, -0.5f), mul(rho, 1.f / 9.f));
            w36 = fma(1.f / 3.f, mul(rh, 0.25f), mul(rho, 1.f / 36.f));
        }
        auto pair = [&](int p, F e, bool dg, F &gp, F &gm) {
            const F c = fma(dg ? bdg : bax, dg ? cdg : cax, fma(mul(dg ? b36 : b9, e), e, dg ? k36 : k9));
            const F o = dg ? a36 : a9;
            gp = fma(o, e, c);
            gm = fma(neg(o), e, c);
            if (NUP) W[p] = mul(dg ? w36 : w9, e);
        };
        F g1, g2, g3, g4, g5, g6, g7, g8;
        pair(0, u, false, g1, g2);
        pair(1, v, false, g3, g4);
        pair(2, add(u, v), true, g5, g6);
        pair(3, sub(u, v), true, g7, g8);
        if (DOWN) {  // complete the row below
            const F l7 = from_left(g7), r6 = from_right(g6);
            const F axs = add(P.ax, add(P.g3, g4)), dgs = add(add(P.g5, r6), add(l7, P.g8));
            F D = add(P.g0, add(axs, dgs));
            const F rna = add(D, 1.f);
            if (NUP) {
                const F n2 = sub(P.o2, from_right(W[2])), n3 = sub(from_left(W[3]), P.o3);
                D = fma(sdelta, add(add(P.o0, sub(P.o1, W[1])), add(n2, n3)), D);
            }
            const F m = fma(dm.a, P.d, bc<F>(am1)), d5 = sub(P.g5, r6), d7 = sub(l7, P.g8);
            F X = add(fma(m, P.u, add(P.dx, add(d5, d7))), P.u);
            F Y = add(fma(m, P.v, add(sub(P.g3, g4), sub(d5, d7))), P.v);
            if (fc.on) {
                const F rp = add(P.d, 1.f);
                X = fma(fc.gx, rp, X);
                Y = fma(fc.gy, rp, Y);
                if (FIELD) {
                    X = fma(rp, P.gx, X);
                    Y = fma(rp, P.gy, Y);
                }
            }
            F un, vn;
            velocity(NUP ? add(D, 1.f) : rna, X, Y, un, vn);
            // |c|^2 - 2/3: rest -2/3, axis 1/3, diagonal 4/3
            const F tn = fma(-2.f / 3.f, P.g0, fma(1.f / 3.f, axs, mul(dgs, 4.f / 3.f)));
            store(y - 1, D, un, vn, sub(quotient(tn, rna), fma(un, un, mul(vn, vn))));
        }
        if (OWN) {
            const F l1 = from_left(g1), r2 = from_right(g2);
            C.ax = add(l1, r2);
            C.dx = sub(l1, r2);
            C.g0 = fma(4.f / 9.f, K, mul(rh, add(add(h, -2.f), Pt)));
            if (NUP) C.o0 = sub(from_left(W[0]), from_right(W[0]));
            C.d = d;
            C.u = u;
            C.v = v;
            C.gx = gx;
            C.gy = gy;
        }
        if (UP) {  // to the row above
            P.g3 = g3;
            P.g5 = from_left(g5);
            P.g8 = from_right(g8);
            if (NUP) {
                P.o1 = W[1];
                P.o2 = from_left(W[2]);
                P.o3 = from_right(W[3]);
            }
        }
    }

    // a march over rows ya - 1 .. yb: four rows of loads in flight
    __device__ __forceinline__ void rows(int ya, int yb) const {
        Raw r0, r1, r2, r3;
        A pa, pb;
        load(ya - 1, r0);
        load(ya, r1);
        load(ya + 1, r2);
        if (ya + 2 <= yb) load(ya + 2, r3);
        source<FIRST>(ya - 1, r0, pa, pb, yb);
        source<START>(ya, r1, pb, pa, yb);
        int y = ya + 1;
        for (; y + 3 < yb; y += 4) {
            source<MID>(y, r2, pa, pb, yb);
            source<MID>(y + 1, r3, pb, pa, yb);
            source<MID>(y + 2, r0, pa, pb, yb);
            source<MID>(y + 3, r1, pb, pa, yb);
        }
        if (y == yb) {
            source<LAST>(y, r2, pa, pb, yb);
            return;
        }
        source<MID>(y, r2, pa, pb, yb);
        if (y + 1 == yb) {
            source<LAST>(y + 1, r3, pb, pa, yb);
            return;
        }
        source<MID>(y + 1, r3, pb, pa, yb);
        if (y + 2 == yb) {
            source<LAST>(y + 2, r0, pa, pb, yb);
            return;
        }
        source<MID>(y + 2, r0, pa, pb, yb);
        source<LAST>(y + 3, r1, pb, pa, yb);
    }
};

}  // namespace rows2
}  // namespace lwacm
