// Many steps of one small D2Q9 domain in one launch, by one thread-block cluster.
//
// A step of a small domain takes about as long as its launch (64^2: 1.25 us replayed from a
// graph). Here up to 16 CTAs, one to an SM, each hold a run of whole rows for as many steps as
// asked: a thread keeps its nodes' fields in registers, leaves their eight link values (and
// the density terms of omega_p) in shared memory, those of a first or last row in the shared
// memory of the CTA that holds the next row as well, and gathers what arrives at its nodes
// after a barrier of the cluster. Two sets of link arrays alternate, so one barrier a step is
// enough: a CTA writes a set again only after every CTA has passed the barrier of the step
// between. The barrier is the hardware's, and every thread of every CTA takes part in it the
// same number of times.
//
// A thread reads its own nodes' fields at the start and writes them at the end, so `in` and
// `out` may be one buffer.
//
// The values and sums are formed as the marching kernel forms them (rows2.cuh), in the same
// order, so the fields do not depend on how many steps a launch takes (the bulk-viscosity
// variant as there, in the 2D-tile kernel's order).
//
// What bounds it: the barrier and the chain of a node's update behind it (0.5 us a step with one
// warp a CTA), and with 1024 nodes a CTA the instructions of 32 warps on one SM (128^2 1.05 us,
// with bulk viscosity 1.24; replayed launches 1.46 and 1.89).
#include "dev_cache.h"
#include "launch.h"
#include "lwacm_core.cuh"
#include "rows2.cuh"

namespace lwacm {
namespace {

using rows2::Walls2;

constexpr int kCtas = 16;       // CTAs of the cluster
constexpr int kThreads = 1024;  // threads of a CTA at most
constexpr int kMaxSmem = 227 * 1024;
constexpr int kNodes = 1664;    // nodes of a CTA at most, one or two a thread: the marching kernel in
                                // graphs catches up there (us a step over 256 steps, cluster / march:
                                // 64^2 0.62 / 1.26, 128^2 1.05 / 1.46, 160^2 1.43 / 1.89, its cavity
                                // 1.87 / 1.91, 176^2 cavity 2.10 / 2.03)

struct Small2 {
    int nx, ny;
    int nrows;  // rows of a CTA at most
    long long fstride;
    float s, a, gamma, sdelta;
    int forced;
    float gx, gy;
    Walls2 wl;
};

// address of a shared variable of this CTA in CTA `rank` of the cluster
__device__ __forceinline__ uint32_t map_rank(uint32_t addr, int rank) {
    uint32_t r;
    asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(addr), "r"(rank));
    return r;
}
__device__ __forceinline__ void st_cluster(uint32_t addr, float v) {
    asm volatile("st.shared::cluster.f32 [%0], %1;" ::"r"(addr), "f"(v) : "memory");
}
__device__ __forceinline__ void cluster_barrier() {
    asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
    asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}

template <int PER, typename T, bool WALLS, bool BULK, bool NUP>
__global__ void __launch_bounds__(kThreads) k_d2q9_cluster(const T *in, T *out, Small2 p, int steps) {
    constexpr int NV = NUP ? 12 : 8;  // values a node leaves: links 1 to 8, then W_0 to W_3
    constexpr int NF = BULK ? 4 : 3;
    extern __shared__ float sm[];
    const int ctas = (int)gridDim.x, rank = (int)blockIdx.x, nt = (int)blockDim.x;
    const int ya = (int)((long long)p.ny * rank / ctas), rows = (int)((long long)p.ny * (rank + 1) / ctas) - ya;
    const int up = rank + 1 == ctas ? 0 : rank + 1, dn = rank == 0 ? ctas - 1 : rank - 1;
    const int dn_rows = (int)((long long)p.ny * (dn + 1) / ctas) - (int)((long long)p.ny * dn / ctas);
    // link arrays [set][value][row -1 .. rows][x], the same places in every CTA
    const int pitch = (p.nrows + 2) * p.nx, set = NV * pitch;
    const uint32_t base = tile::sa(sm);
    const uint32_t base_up = map_rank(base, up), base_dn = map_rank(base, dn);
    const float nu = p.s * (1.f / 18.f), odd = __fmul_rn(p.s, 2.f / 9.f);
    const float am1 = BULK ? p.s * (-1.f / 3.f) : __fmul_rn(odd, -1.5f), am1l = fmaf(odd, -1.5f, -am1);  // as March's
    // the thread's nodes
    int at[PER], xl[PER], xr[PER];  // place in a value's array; the places of x - 1 and x + 1 less this one
    int y[PER], xs[PER];
    bool on[PER], first[PER], last[PER];  // in use; in the CTA's first, last row
    float d[PER], u[PER], v[PER], tr[PER];
#pragma unroll
    for (int k = 0; k < PER; ++k) {
        const int i = (int)threadIdx.x + k * nt;
        on[k] = i < rows * p.nx;
        const int r = on[k] ? i / p.nx : 0, x = on[k] ? i - r * p.nx : 0;
        at[k] = (r + 1) * p.nx + x;
        xl[k] = x == 0 ? p.nx - 1 : -1;
        xr[k] = x == p.nx - 1 ? 1 - p.nx : 1;
        y[k] = ya + r;
        first[k] = r == 0;
        last[k] = r == rows - 1;
        xs[k] = x;
        const long long g = (long long)y[k] * p.nx + x;
        d[k] = u[k] = v[k] = tr[k] = 0.f;
        if (on[k]) {
            d[k] = rows2::widen(rows2::ldraw<true>(in + g));
            u[k] = rows2::widen(rows2::ldraw<true>(in + p.fstride + g));
            v[k] = rows2::widen(rows2::ldraw<true>(in + 2 * p.fstride + g));
            if (BULK) tr[k] = rows2::widen(rows2::ldraw<true>(in + (NF - 1) * p.fstride + g));
        }
    }
    cluster_barrier();  // every CTA runs before any writes to its shared memory
    for (int s = 0; s < steps; ++s) {
        const int so = (s & 1) * set;
        float *G = sm + so;
        float own[PER][8], df0[PER];
#pragma unroll
        for (int k = 0; k < PER; ++k) {
            if (!on[k]) continue;
            const float rho = __fadd_rn(d[k], 1.f);
            const float K = fmaf(__fmul_rn(rho, -1.5f), fmaf(u[k], u[k], __fmul_rn(v[k], v[k])), d[k]);
            const float k9 = __fmul_rn(K, 1.f / 9.f), k36 = __fmul_rn(K, 1.f / 36.f);
            const float b9 = __fmul_rn(rho, 0.5f), b36 = __fmul_rn(rho, 0.125f);
            const float e[4] = {u[k], v[k], __fadd_rn(u[k], v[k]), __fsub_rn(u[k], v[k])};
            float val[NV];
            if (BULK) {
                const float h = __fmul_rn(tr[k], 0.5f * p.gamma), rh = __fmul_rn(rho, h);
                const float Pt = fmaf(u[k], u[k], fmaf(v[k], v[k], 2.f / 3.f));
                const float bax = __fmul_rn(rh, 0.5f), bdg = __fmul_rn(rh, 0.25f);
                const float cax = __fsub_rn(__fsub_rn(1.f, Pt), h), cdg = __fadd_rn(h, Pt);
                const float odg = __fmul_rn(bdg, 1.f - p.a), rn = __fmul_rn(rho, nu);
                const float a9 = __fadd_rn(__fmul_rn(rn, 2.f), __fmul_rn(odg, -2.f));
                const float a36 = __fadd_rn(__fmul_rn(rn, 0.5f), odg);
                df0[k] = __fmul_rn(rh, __fadd_rn(__fadd_rn(h, -2.f), Pt));
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    const bool dg = q >= 2;
                    const float c = fmaf(dg ? bdg : bax, dg ? cdg : cax,
                                         fmaf(__fmul_rn(dg ? b36 : b9, e[q]), e[q], dg ? k36 : k9));
                    val[2 * q] = fmaf(dg ? a36 : a9, e[q], c);
                    val[2 * q + 1] = fmaf(-(dg ? a36 : a9), e[q], c);
                    if (NUP)
                        val[NUP ? 8 + q : 0] =
                            __fmul_rn(fmaf(1.f / 3.f, dg ? __fmul_rn(rh, 0.25f) : __fmul_rn(rh, -0.5f),
                                           __fmul_rn(rho, dg ? 1.f / 36.f : 1.f / 9.f)),
                                      e[q]);
                }
            } else {
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    const float t = __fmul_rn(q >= 2 ? b36 : b9, e[q]), c = fmaf(t, e[q], q >= 2 ? k36 : k9);
                    val[2 * q] = fmaf(odd, t, c);
                    val[2 * q + 1] = fmaf(-odd, t, c);
                    if (NUP) val[NUP ? 8 + q : 0] = __fmul_rn(t, 2.f / 9.f);
                }
            }
            // links (1,0) (-1,0) (0,1) (0,-1) (1,1) (-1,-1) (1,-1) (-1,1)
#pragma unroll
            for (int q = 0; q < NV; ++q) G[q * pitch + at[k]] = val[q];
#pragma unroll
            for (int q = 0; q < 8; ++q) own[k][q] = val[q];
            if (first[k]) {  // to the row after the last of the CTA below: links with c_y = -1
                const uint32_t to = base_dn + 4u * (uint32_t)(so + (dn_rows + 1) * p.nx + xs[k]);
                const int q[6] = {3, 5, 6, 9, 10, 11};
#pragma unroll
                for (int j = 0; j < (NUP ? 6 : 3); ++j) st_cluster(to + 4u * (uint32_t)(q[j] * pitch), val[q[j]]);
            }
            if (last[k]) {  // to the row before the first of the CTA above: links with c_y = +1
                const uint32_t to = base_up + 4u * (uint32_t)(so + xs[k]);
                const int q[6] = {2, 4, 7, 9, 10, 11};
#pragma unroll
                for (int j = 0; j < (NUP ? 6 : 3); ++j) st_cluster(to + 4u * (uint32_t)(q[j] * pitch), val[q[j]]);
            }
        }
        cluster_barrier();
#pragma unroll
        for (int k = 0; k < PER; ++k) {
            if (!on[k]) continue;
            const int c = at[k], l = c + xl[k], r = c + xr[k], nx = p.nx;
            auto g = [&](int q, int i) { return G[q * pitch + i]; };
            float l1 = g(0, l), r2 = g(1, r), g3 = g(2, c - nx), g4 = g(3, c + nx);
            float l5 = g(4, l - nx), r6 = g(5, r + nx), l7 = g(6, l + nx), r8 = g(7, r - nx);
            const float rho = __fadd_rn(d[k], 1.f);
            const float K = fmaf(__fmul_rn(rho, -1.5f), fmaf(u[k], u[k], __fmul_rn(v[k], v[k])), d[k]);
            const float m = BULK ? fmaf(p.a, d[k], am1) : __fadd_rn(fmaf(p.a, d[k], am1l), am1);
            float D, X, Y, un, vn, tn = 0.f;
            if (BULK) {
                const float axs = __fadd_rn(__fadd_rn(l1, r2), __fadd_rn(g3, g4));
                const float dgs = __fadd_rn(__fadd_rn(l5, r6), __fadd_rn(l7, r8));
                const float g0 = fmaf(4.f / 9.f, K, df0[k]);
                D = __fadd_rn(g0, __fadd_rn(axs, dgs));
                const float rna = __fadd_rn(D, 1.f);
                if (NUP) {
                    const float o0 = __fsub_rn(g(NV - 4, l), g(NV - 4, r)), o1 = __fsub_rn(g(NV - 3, c - nx), g(NV - 3, c + nx));
                    const float n2 = __fsub_rn(g(NV - 2, l - nx), g(NV - 2, r + nx));
                    const float n3 = __fsub_rn(g(NV - 1, l + nx), g(NV - 1, r - nx));
                    D = fmaf(p.sdelta, __fadd_rn(__fadd_rn(o0, o1), __fadd_rn(n2, n3)), D);
                }
                const float d5 = __fsub_rn(l5, r6), d7 = __fsub_rn(l7, r8);
                X = __fadd_rn(fmaf(m, u[k], __fadd_rn(__fsub_rn(l1, r2), __fadd_rn(d5, d7))), u[k]);
                Y = __fadd_rn(fmaf(m, v[k], __fadd_rn(__fsub_rn(g3, g4), __fsub_rn(d5, d7))), v[k]);
                if (p.forced) {
                    X = fmaf(p.gx, rho, X);
                    Y = fmaf(p.gy, rho, Y);
                }
                rows2::velocity(NUP ? __fadd_rn(D, 1.f) : rna, X, Y, un, vn);
                const float ts = fmaf(-2.f / 3.f, g0, fmaf(1.f / 3.f, axs, __fmul_rn(dgs, 4.f / 3.f)));
                tn = __fsub_rn(ts / rna, fmaf(un, un, __fmul_rn(vn, vn)));
            } else {
                const bool e0 = WALLS && p.wl.wx && xs[k] == 0, eN = WALLS && p.wl.wx && xs[k] == nx - 1;
                const bool low = WALLS && p.wl.wy && y[k] == 0, top = WALLS && p.wl.wy && y[k] == p.ny - 1;
                const float *o = own[k];
                if (WALLS) {  // as March::source
                    if (e0) l1 = o[1], l5 = l7 = 0.f;
                    if (eN) r2 = o[0], r6 = r8 = 0.f;
                    if (low) g3 = o[3], l5 = o[5], r8 = o[6];
                    if (top) {
                        g4 = __fadd_rn(o[2], -(p.wl.wallc * (1.f / 9.f)) * p.wl.lidy);
                        l7 = __fadd_rn(o[7], (p.wl.wallc * (1.f / 36.f)) * (p.wl.lidx - p.wl.lidy));
                        r6 = __fadd_rn(o[4], (p.wl.wallc * (1.f / 36.f)) * (-p.wl.lidx - p.wl.lidy));
                    }
                }
                const float below = __fadd_rn(g3, __fadd_rn(l5, r8));
                D = fmaf(4.f / 9.f, K, __fadd_rn(below, __fadd_rn(l1, r2)));
                X = fmaf(m, u[k], __fadd_rn(__fsub_rn(l5, r8), __fsub_rn(l1, r2)));
                Y = fmaf(m, v[k], below);
                if (WALLS) {
                    if (e0 && !low) D = __fadd_rn(D, o[5]), X = __fadd_rn(X, o[5]), Y = __fadd_rn(Y, o[5]);
                    if (e0 && !top) D = __fadd_rn(D, o[7]), X = __fadd_rn(X, o[7]), Y = __fsub_rn(Y, o[7]);
                    if (eN && !top) D = __fadd_rn(D, o[4]), X = __fsub_rn(X, o[4]), Y = __fsub_rn(Y, o[4]);
                    if (eN && !low) D = __fadd_rn(D, o[6]), X = __fsub_rn(X, o[6]), Y = __fadd_rn(Y, o[6]);
                }
                if (p.forced) {
                    X = fmaf(p.gx, rho, X);
                    Y = fmaf(p.gy, rho, Y);
                }
                const float all = __fadd_rn(g4, __fadd_rn(l7, r6));
                D = __fadd_rn(D, all);
                if (NUP) {
                    const float sb = __fadd_rn(g(NV - 3, c - nx), __fsub_rn(g(NV - 2, l - nx), g(NV - 1, r - nx)));
                    const float so2 = __fadd_rn(sb, __fsub_rn(g(NV - 4, l), g(NV - 4, r)));
                    const float w = __fsub_rn(g(NV - 2, r + nx), g(NV - 1, l + nx));
                    D = fmaf(p.sdelta, __fsub_rn(so2, __fadd_rn(w, g(NV - 3, c + nx))), D);
                }
                X = __fadd_rn(__fadd_rn(X, __fsub_rn(l7, r6)), u[k]);
                Y = __fadd_rn(__fsub_rn(Y, all), v[k]);
                rows2::velocity(__fadd_rn(D, 1.f), X, Y, un, vn);
            }
            // as stored and read again
            T t;
            stf(&t, D);
            d[k] = rows2::widen(t);
            stf(&t, un);
            u[k] = rows2::widen(t);
            stf(&t, vn);
            v[k] = rows2::widen(t);
            if (BULK) {
                stf(&t, tn);
                tr[k] = rows2::widen(t);
            }
        }
    }
#pragma unroll
    for (int k = 0; k < PER; ++k) {
        if (!on[k]) continue;
        const long long g = (long long)y[k] * p.nx + xs[k];
        stf(out + g, d[k]);
        stf(out + p.fstride + g, u[k]);
        stf(out + 2 * p.fstride + g, v[k]);
        if (BULK) stf(out + (NF - 1) * p.fstride + g, tr[k]);
    }
}

// the cluster's shape for a domain: CTAs, rows of one at most, threads, nodes of a thread
struct Shape {
    int ctas, nrows, threads, per;
};
Shape shape_of(int nx, int ny) {
    Shape s;
    s.ctas = ny < kCtas ? ny : kCtas;
    s.nrows = (ny - 1) / s.ctas + 1;
    const long long nodes = (long long)s.nrows * nx;
    s.per = nodes <= kThreads ? 1 : (nodes <= kNodes ? 2 : 0);
    const int t = s.per ? (int)((nodes - 1) / s.per + 1) : 0;
    s.threads = (t + 31) / 32 * 32;
    return s;
}
size_t link_bytes(int nx, int nrows, bool nup) { return 2 * (size_t)(nup ? 12 : 8) * (nrows + 2) * nx * sizeof(float); }

template <int PER, typename T, bool WALLS, bool BULK, bool NUP>
cudaError_t launch_k(const void *in, void *out, const Small2 &q, const Shape &s, int steps, cudaStream_t st) {
    auto kern = k_d2q9_cluster<PER, T, WALLS, BULK, NUP>;
    const size_t bytes = link_bytes(q.nx, s.nrows, NUP);
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = kCtas;
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.attrs = at;
    cfg.numAttrs = 1;
    // once per device: opt in to clusters of 16 and to the largest shared memory this kernel asks for,
    // and see whether the device has room for such a cluster
    static DevSlots set;
    const int ok = per_device(set, [&] {
        cfg.gridDim = dim3(kCtas);
        cfg.blockDim = dim3(kThreads);
        cfg.dynamicSmemBytes = kMaxSmem;
        int clusters = 0;
        const bool fits =
            cudaFuncSetAttribute(kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) == cudaSuccess &&
            cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, kMaxSmem) == cudaSuccess &&
            cudaOccupancyMaxActiveClusters(&clusters, kern, &cfg) == cudaSuccess && clusters > 0;
        if (!fits) cudaGetLastError();
        return fits ? 1 : -1;
    });
    if (ok < 1) return cudaErrorNotSupported;
    cfg.gridDim = dim3((unsigned)s.ctas);
    cfg.blockDim = dim3((unsigned)s.threads);
    cfg.dynamicSmemBytes = bytes;
    cfg.stream = st;
    at[0].val.clusterDim.x = (unsigned)s.ctas;
    return cudaLaunchKernelEx(&cfg, kern, (const T *)in, (T *)out, q, steps);
}
template <int PER, typename T>
cudaError_t launch_v(const void *in, void *out, const Small2 &q, const Shape &s, int bc, bool bulk, int steps,
                     cudaStream_t st) {
    if (bulk && q.sdelta != 0.f) return launch_k<PER, T, false, true, true>(in, out, q, s, steps, st);
    if (bulk) return launch_k<PER, T, false, true, false>(in, out, q, s, steps, st);
    if (q.sdelta != 0.f) return launch_k<PER, T, false, false, true>(in, out, q, s, steps, st);
    if (bc == BC_PERIODIC) return launch_k<PER, T, false, false, false>(in, out, q, s, steps, st);
    return launch_k<PER, T, true, false, false>(in, out, q, s, steps, st);
}
template <typename T>
cudaError_t launch_t(const void *in, void *out, const Small2 &q, const Shape &s, int bc, bool bulk, int steps,
                     cudaStream_t st) {
    return s.per == 1 ? launch_v<1, T>(in, out, q, s, bc, bulk, steps, st)
                      : launch_v<2, T>(in, out, q, s, bc, bulk, steps, st);
}

}  // namespace

bool cluster2d_supported(const StepParams &p) {
    const Shape s = shape_of(p.nx, p.ny);
    return !p.gfield && s.per > 0 && link_bytes(p.nx, s.nrows, p.sdelta != 0.f) <= kMaxSmem;
}

cudaError_t launch_cluster2d(int storage, const void *in, void *out, const StepParams &p, int steps, cudaStream_t st) {
    if (!cluster2d_supported(p)) return cudaErrorInvalidValue;
    const Shape s = shape_of(p.nx, p.ny);
    Small2 q;
    q.nx = p.nx;
    q.ny = p.ny;
    q.nrows = s.nrows;
    q.fstride = p.fstride;
    q.s = p.s;
    q.a = p.a;
    q.gamma = p.gamma;
    q.sdelta = p.sdelta;
    q.forced = p.has_force;
    q.gx = p.force[0];
    q.gy = p.force[1];
    q.wl.wx = p.walled[0];
    q.wl.wy = p.walled[1];
    q.wl.wallc = p.wallc;
    q.wl.lidx = p.lid[0];
    q.wl.lidy = p.lid[1];
    switch (storage) {
        case STORE_F32: return launch_t<float>(in, out, q, s, p.bc, p.bulk, steps, st);
        case STORE_BF16: return launch_t<__nv_bfloat16>(in, out, q, s, p.bc, p.bulk, steps, st);
        case STORE_F16: return launch_t<__half>(in, out, q, s, p.bc, p.bulk, steps, st);
    }
    return cudaErrorInvalidValue;
}

}  // namespace lwacm
