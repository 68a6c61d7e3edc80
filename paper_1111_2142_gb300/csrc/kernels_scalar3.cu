// The passive scalar of Eq. ACM2.0t on D3Q19 (periodic) by warps that march along z, any size,
// run after the flow kernel on the same state at t:
//   T+(x) = a_t T(x) + sum_i w_i [(1 - a_t)(T + 9/2 e^2 - 3/2 |u|^2) + 3 T e](x - c_i).
//
// The strips, tiles, row pairs and runs of planes are those of kernels_rows3.cu: a lane holds a
// column of four rows and their two neighbours, values move along x by shuffles, along y within
// the lane, along z through the sums of three planes, here one number a node. 20 bytes a node
// (T, u, v, w in, T out).
//
// What bounds it, FP32 256 x 256 x 128 (48 us, 3.5 TB/s at 20 bytes a node): instructions and
// their latency with 24 warps a SM, as the flow kernel's. The row-tiled kernel (kernels_scalar.cu)
// took 52 us there and 46.6 against 51.6 on 128 x 256 x 256, the gather, flow and scalar in one,
// 78 on 200 x 100 x 90 (this kernel and the flow's 30.5) and 321 with BF16 storage on 256 x 256 x
// 128 (116).
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
using rows2::neg;
using rows2::sub;
using rows2::widen;
using F2 = float2;

constexpr int kStrip = 30, kTile = 4, kWarps = 4;  // as kernels_rows3.cu

struct Dom3 {
    int nx, ny, nz;
    long long fstride;
    float at;  // a_t = 1 - 6 alpha
};

enum { FIRST = 0, START = 1, MID = 2, LAST = 3 };

// what two rows send along y: the links with c_z = 0, +1, -1
struct Send {
    F2 s, p, m;
};

template <typename T>
struct March3 {
    const T *in;  // the fields u, v, w, T, fstride apart
    T *out;       // the scalar's field of the new state
    const Dom3 &dm;
    long long plane;
    float b1, b2;  // w 9/2 (1 - a_t) of the axis and the diagonal links
    unsigned off, lo, hi;
    bool st;

    __device__ __forceinline__ March3(const T *in_, T *out_, const Dom3 &dm_, int x0, int y0)
        : in(in_), out(out_), dm(dm_), plane((long long)dm_.nx * dm_.ny), b1((1.f - dm_.at) * 0.25f),
          b2((1.f - dm_.at) * 0.125f) {
        const int lane = threadIdx.x & 31, x = x0 + lane - 1;
        const unsigned xw = (unsigned)(x < 0 ? x + dm.nx : (x < dm.nx ? x : x % dm.nx)), nx = (unsigned)dm.nx;
        off = ((unsigned)y0 * nx + xw) * (unsigned)sizeof(T);
        lo = ((unsigned)(y0 > 0 ? y0 - 1 : dm.ny - 1) * nx + xw) * (unsigned)sizeof(T);
        hi = ((unsigned)(y0 + kTile < dm.ny ? y0 + kTile : 0) * nx + xw) * (unsigned)sizeof(T);
        st = lane >= 1 && lane <= kStrip && x < dm.nx;
    }
    struct Raw {
        T f[4][6];  // u, v, w, T
    };
    __device__ __forceinline__ void load(int z, Raw &r) const {
        z = z < 0 ? z + dm.nz : (z >= dm.nz ? z - dm.nz : z);
#pragma unroll
        for (int f = 0; f < 4; ++f) {
            const T *p = in + (z * plane + f * dm.fstride);
            r.f[f][0] = __ldg(byte_at(p, lo));
#pragma unroll
            for (int j = 0; j < kTile; ++j) r.f[f][1 + j] = __ldg(byte_at(p + (long long)j * dm.nx, off));
            r.f[f][5] = __ldg(byte_at(p, hi));
        }
    }
    struct Node {
        F2 u, v, w, K1, K2, O1, O2;  // w (1 - a_t)(T - 3/2 |u|^2) and 3 w T of both kinds of links
    };
    __device__ __forceinline__ Node consts(F2 u, F2 v, F2 w, F2 t) const {
        Node n;
        n.u = u;
        n.v = v;
        n.w = w;
        const F2 K = fma(bc<F2>(-1.5f), fma(u, u, fma(v, v, mul(w, w))), t);
        n.K2 = mul(K, (1.f - dm.at) * (1.f / 36.f));
        n.K1 = add(n.K2, n.K2);
        n.O2 = mul(t, 1.f / 12.f);
        n.O1 = add(n.O2, n.O2);
        return n;
    }
    __device__ __forceinline__ void pair(const Node &n, F2 e, bool dg, F2 &gp, F2 &gm) const {
        const F2 c = fma(mul(e, dg ? b2 : b1), e, dg ? n.K2 : n.K1), o = mul(dg ? n.O2 : n.O1, e);
        gp = add(c, o);
        gm = sub(c, o);
    }
    __device__ __forceinline__ F2 plus(const Node &n, F2 e, bool dg) const {
        const F2 c = fma(mul(e, dg ? b2 : b1), e, dg ? n.K2 : n.K1);
        return add(c, mul(dg ? n.O2 : n.O1, e));
    }
    template <int MODE>
    __device__ __forceinline__ void in_row(const Node &n, F2 t, F2 &P, F2 &C, F2 &N) const {
        F2 zp, zm, pp, mm, pm, mp;
        pair(n, n.w, false, zp, zm);
        pair(n, add(n.u, n.w), true, pp, mm);  // (1,0,1) (-1,0,-1)
        pair(n, sub(n.u, n.w), true, pm, mp);  // (1,0,-1) (-1,0,1)
        if (MODE == START || MODE == MID) {
            F2 xp, xm;
            pair(n, n.u, false, xp, xm);
            C = add(C, add(from_left(xp), from_right(xm)));
            C = fma(dm.at, t, fma(12.f, n.K2, C));  // the rest link, w_0 = 12 / 36, and the own term
        }
        if (MODE == MID || MODE == LAST) P = add(P, add(zm, add(from_left(pm), from_right(mm))));
        if (MODE != LAST) N = add(zp, add(from_left(pp), from_right(mp)));
    }
    template <int MODE>
    __device__ __forceinline__ void to_rows(const Node &n, Send &up, Send &dn) const {
        if (MODE == START || MODE == MID) {
            F2 yp, ym, pp, mm, pm, mp;
            pair(n, n.v, false, yp, ym);
            pair(n, add(n.u, n.v), true, pp, mm);  // (1,1,0) (-1,-1,0)
            pair(n, sub(n.u, n.v), true, pm, mp);  // (1,-1,0) (-1,1,0)
            up.s = add(yp, add(from_left(pp), from_right(mp)));
            dn.s = add(ym, add(from_left(pm), from_right(mm)));
        }
        pair(n, add(n.v, n.w), true, up.p, dn.m);  // (0,1,1) (0,-1,-1)
        pair(n, sub(n.v, n.w), true, up.m, dn.p);  // (0,1,-1) (0,-1,1)
    }
    template <int MODE>
    __device__ __forceinline__ void halo(const Node &n, Send &h) const {
        if (MODE == START || MODE == MID)
            h.s = add(plus(n, n.v, false),
                      add(from_left(plus(n, add(n.v, n.u), true)), from_right(plus(n, sub(n.v, n.u), true))));
        if (MODE != LAST) h.p = plus(n, add(n.v, n.w), true);
        if (MODE == MID || MODE == LAST) h.m = plus(n, sub(n.v, n.w), true);
    }
    template <int MODE>
    __device__ __forceinline__ void receive(const Send &up, const Send &dn, F2 &P, F2 &C, F2 &N) const {
        if (MODE == START || MODE == MID) C = add(C, add(up.s, dn.s));
        if (MODE == MID || MODE == LAST) P = add(P, add(up.m, dn.m));
        if (MODE != LAST) N = add(N, add(up.p, dn.p));
    }
    __device__ __forceinline__ Node node(const Raw &r, int a, int b, float sign, F2 &t) const {
        t = make_float2(widen(r.f[3][a]), widen(r.f[3][b]));
        return consts(make_float2(widen(r.f[0][a]), widen(r.f[0][b])),
                      make_float2(widen(r.f[1][a]), sign * widen(r.f[1][b])),
                      make_float2(widen(r.f[2][a]), widen(r.f[2][b])), t);
    }
    template <int MODE>
    __device__ __forceinline__ void source(int z, Raw &r, F2 (&P)[2], F2 (&C)[2], bool more) const {
        F2 t0, t1, th;
        const Node n0 = node(r, 1, 3, 1.f, t0), n1 = node(r, 2, 4, 1.f, t1), nh = node(r, 0, 5, -1.f, th);
        if (more) load(z + 1, r);
        F2 N[2];
        in_row<MODE>(n0, t0, P[0], C[0], N[0]);
        in_row<MODE>(n1, t1, P[1], C[1], N[1]);
        Send up0, dn0, up1, dn1, h;
        halo<MODE>(nh, h);
        to_rows<MODE>(n0, up0, dn0);
        to_rows<MODE>(n1, up1, dn1);
        auto lo2 = [](F2 a, F2 b) { return make_float2(a.x, b.x); };
        auto hi2 = [](F2 a, F2 b) { return make_float2(a.y, b.y); };
        const Send ua = {lo2(h.s, up1.s), lo2(h.p, up1.p), lo2(h.m, up1.m)};
        const Send db = {hi2(dn0.s, h.s), hi2(dn0.p, h.p), hi2(dn0.m, h.m)};
        receive<MODE>(ua, dn1, P[0], C[0], N[0]);
        receive<MODE>(up0, db, P[1], C[1], N[1]);
        if ((MODE == MID || MODE == LAST) && st) {
            T *o = out + (z - 1) * plane;
            const long long nx = dm.nx;
            stf(byte_at(o, off), P[0].x);
            stf(byte_at(o + nx, off), P[1].x);
            stf(byte_at(o + 2 * nx, off), P[0].y);
            stf(byte_at(o + 3 * nx, off), P[1].y);
        }
        if (MODE != LAST) {
            P[0] = N[0];
            P[1] = N[1];
        }
    }
    __device__ __forceinline__ void planes(int za, int zb) const {
        Raw r;
        F2 pa[2], pb[2];
        load(za - 1, r);
        source<FIRST>(za - 1, r, pa, pb, true);
        source<START>(za, r, pb, pa, true);
        int z = za + 1;
        for (; z + 1 < zb; z += 2) {
            source<MID>(z, r, pa, pb, true);
            source<MID>(z + 1, r, pb, pa, true);
        }
        if (z < zb) {
            source<MID>(z, r, pa, pb, true);
            source<LAST>(z + 1, r, pb, pa, false);
        } else {
            source<LAST>(z, r, pa, pb, false);
        }
    }
};

template <typename T>
__global__ void __launch_bounds__(32 * kWarps) k_scalar_march(const T *__restrict__ in, T *__restrict__ out, Dom3 dm,
                                                              int strips, int groups, int runs) {
    // (an ordinary launch: with its CTAs set up ahead of the flow kernel's end, as the flow kernels
    // do among themselves, a step of 256 x 256 x 128 took 150 us instead of 120)
    const int rest = (int)(blockIdx.x / (unsigned)strips), strip = (int)blockIdx.x - rest * strips;
    const int run = rest / groups, group = rest - run * groups;
    int y0 = (group * kWarps + (int)(threadIdx.x >> 5)) * kTile;
    if (y0 >= dm.ny) return;
    y0 = min(y0, dm.ny - kTile);  // the last tile ends with the domain
    const March3<T> m(in, out, dm, strip * kStrip, y0);
    m.planes((int)((long long)dm.nz * run / runs), (int)((long long)dm.nz * (run + 1) / runs));
}

template <typename T>
cudaError_t launch_t(const void *in, void *out, const StepParams &p, cudaStream_t st) {
    static DevSlots cap;
    const int places = per_device(cap, [] {
        int per = 0;
        if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, k_scalar_march<T>, 32 * kWarps, 0) != cudaSuccess ||
            per < 1)
            return -1;
        return per * device_sms();
    });
    if (places < 1) return cudaErrorNotSupported;
    Dom3 dm;
    dm.nx = p.nx;
    dm.ny = p.ny;
    dm.nz = p.nz;
    dm.fstride = p.fstride;
    dm.at = p.at;
    const int strips = (p.nx - 1) / kStrip + 1, groups = (p.ny - 1) / (kTile * kWarps) + 1;
    const int runs = rows3d_runs((long long)strips * groups, p.nz, places);
    const long long ctas = (long long)strips * groups * runs;
    if (ctas > 0x7fffffffLL) return cudaErrorInvalidValue;
    k_scalar_march<T><<<(unsigned)ctas, 32 * kWarps, 0, st>>>((const T *)in + p.fstride, (T *)out + 4 * p.fstride, dm,
                                                              strips, groups, runs);
    return cudaGetLastError();
}

}  // namespace

cudaError_t launch_scalar_march(int storage, const void *in, void *out, const StepParams &p, cudaStream_t st) {
    switch (storage) {
        case STORE_F32: return launch_t<float>(in, out, p, st);
        case STORE_BF16: return launch_t<__nv_bfloat16>(in, out, p, st);
        case STORE_F16: return launch_t<__half>(in, out, p, st);
    }
    return cudaErrorInvalidValue;
}

}  // namespace lwacm
