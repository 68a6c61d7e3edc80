// D2Q9 update by warps that march along y (single domains and ensembles): the moment
// form of Eq. ACM2.0 (lwacm_core.cuh) with walls, forcing, omega_p and the
// bulk-viscosity variant in the kernel.
//
// A warp takes an item: one or two strips of 30 columns and a run of rows. Lane l holds
// node x0 + l - 1 of a row (lanes 0 and 31 are the strip's neighbours), and with two
// strips node x0 + 30 + l - 1 as well, both in one FP32x2 pair: every operation on link
// values issues once for two nodes and no value moves between the halves of a pair. The warp reads each row
// of its strip once, forms the row's eight link values once (pre-combine, Eq.
// ACM2.0b(a)) and hands them on without shared memory or a barrier (stream, Eq.
// ACM2.0b(b)): along x by warp shuffles, along y through the sums of three rows kept in
// registers, of which the oldest is complete once the next row has been read
// (post-combine, Eq. ACM2.0b(c)). The loads of the next four rows are in flight
// meanwhile.
//
// What bounds it, FP32 periodic: at 8192^2 memory (262 us a step, 6.1 TB/s, 91% of a copy's
// rate; the 2D-tile kernel 490 us), at 4096^2 the same with the tail of the last wave (70.1
// us; 123 us), at 1024^2, where the state stays in L2, the latency of the rows of a warp (6.6
// us; 8.9 us) and at 64^2 the launch (1.25 us; 1.8 us). With two rows of loads in flight
// instead of four, 4096^2 took 82.8 us.
//
// A lane reads and writes single elements, 32 neighbours per warp access, so no
// alignment of rows, domains or storage types is asked for. The sums of a node are
// formed in the same order whatever the item, so results do not depend on how a
// domain is cut.
#include "dev_cache.h"
#include "launch.h"
#include "lwacm_core.cuh"
#include "rows2.cuh"
#include "tile_common.cuh"

namespace lwacm {
namespace {

using namespace rows2;

// One domain. The warps of a CTA (one, with two strips a warp) take neighbouring strips
// of one run of rows, so that all row arithmetic is uniform over the CTA; CTAs are
// numbered along x first, so that neighbours read the same rows at the same time.
template <int NS, typename T, bool WALLS, bool FIELD, bool BULK, bool NUP>
__global__ void __launch_bounds__(32 * (NS == 1 ? kMaxWarps : 1))
    k_d2q9_rows(const T *in, T *out, Dom2 dm, int ctasx, int rows, Walls2 wl, Force2 fc,
                float gamma, float sdelta) {
    // the next step's CTAs may take their SMs as this step's leave them; none touches
    // global memory before this grid is complete
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    const int run = (int)(blockIdx.x / (unsigned)ctasx), cx = (int)blockIdx.x - run * ctasx;
    int x0 = cx * (NS * kHalf);
    if (NS == 1) {
        x0 = (cx * (int)(blockDim.x >> 5) + (int)(threadIdx.x >> 5)) * kHalf;
        if (x0 >= dm.nx) return;
    }
    const March<NS, T, false, WALLS, FIELD, BULK, NUP> m(in, out, dm, x0, wl, fc, gamma, sdelta);
    asm volatile("griddepcontrol.wait;" ::: "memory");
    const int ya = run * rows;
    m.rows(ya, min(ya + rows, dm.ny));
}

// warps of the kernel that the GPU holds (-1 when it cannot be determined)
template <int NS, typename T, bool WALLS, bool FIELD, bool BULK, bool NUP>
int room(int warps) {
    static DevSlots slots[kMaxWarps + 1];
    return per_device(slots[warps], [&] {
        int per = 0;
        if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, k_d2q9_rows<NS, T, WALLS, FIELD, BULK, NUP>,
                                                          32 * warps, 0) != cudaSuccess || per < 1)
            return -1;
        return per * warps * device_sms();
    });
}

template <int NS, typename T, bool WALLS, bool FIELD, bool BULK, bool NUP>
cudaError_t launch_rows(const void *in, void *out, const StepParams &p, int warps, int rows, const Walls2 &wl,
                        const Force2 &fc, cudaStream_t st) {
    Dom2 dm;
    dm.nx = p.nx;
    dm.ny = p.ny;
    dm.base = 0;
    dm.fstride = p.fstride;
    dm.s = p.s;
    dm.a = p.a;
    const int strips = (p.nx - 1) / (NS * kHalf) + 1, ctasx = (strips - 1) / warps + 1;
    const long long ctas = (long long)ctasx * ((p.ny - 1) / rows + 1);
    if (ctas > 0x7fffffffLL) return cudaErrorInvalidValue;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)ctas);
    cfg.blockDim = dim3(32 * warps);
    cfg.stream = st;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, k_d2q9_rows<NS, T, WALLS, FIELD, BULK, NUP>, (const T *)in, (T *)out, dm, ctasx,
                              rows, wl, fc, p.gamma, p.sdelta);
}
template <typename T, bool WALLS, bool FIELD, bool BULK, bool NUP>
cudaError_t launch_rows(const void *in, void *out, const StepParams &p, const Walls2 &wl, const Force2 &fc,
                        cudaStream_t st) {
    const int warps = cta_warps(p.nx);
    const int room1 = room<1, T, WALLS, FIELD, BULK, NUP>(warps), room2 = room<2, T, WALLS, FIELD, BULK, NUP>(1);
    if (room1 < 1 || room2 < 1) return cudaErrorNotSupported;
    const Cut c = cut_domain(p.nx, p.ny, room1, room2);
    return c.ns == 1 ? launch_rows<1, T, WALLS, FIELD, BULK, NUP>(in, out, p, warps, c.rows, wl, fc, st)
                     : launch_rows<2, T, WALLS, FIELD, BULK, NUP>(in, out, p, 1, c.rows, wl, fc, st);
}

template <typename T, bool FIELD>
cudaError_t rows_variant(const void *in, void *out, const StepParams &p, const Force2 &fc, cudaStream_t st) {
    const Walls2 none{};
    if (p.bulk && p.sdelta != 0.f) return launch_rows<T, false, FIELD, true, true>(in, out, p, none, fc, st);
    if (p.bulk) return launch_rows<T, false, FIELD, true, false>(in, out, p, none, fc, st);
    if (p.sdelta != 0.f) return launch_rows<T, false, FIELD, false, true>(in, out, p, none, fc, st);
    if (p.bc == BC_PERIODIC) return launch_rows<T, false, FIELD, false, false>(in, out, p, none, fc, st);
    Walls2 wl;
    wl.wx = p.walled[0];
    wl.wy = p.walled[1];
    wl.wallc = p.wallc;
    wl.lidx = p.lid[0];
    wl.lidy = p.lid[1];
    return launch_rows<T, true, FIELD, false, false>(in, out, p, wl, fc, st);
}

template <typename T>
cudaError_t rows_t(const void *in, void *out, const StepParams &p, cudaStream_t st) {
    Force2 fc;
    fc.on = p.has_force || p.gfield;
    fc.gx = p.has_force ? p.force[0] : 0.f;
    fc.gy = p.has_force ? p.force[1] : 0.f;
    fc.field = p.gfield;
    return p.gfield ? rows_variant<T, true>(in, out, p, fc, st) : rows_variant<T, false>(in, out, p, fc, st);
}

}  // namespace

cudaError_t launch_step_rows2d(int storage, const void *in, void *out, const StepParams &p, cudaStream_t st) {
    switch (storage) {
        case STORE_F32: return rows_t<float>(in, out, p, st);
        case STORE_BF16: return rows_t<__nv_bfloat16>(in, out, p, st);
        case STORE_F16: return rows_t<__half>(in, out, p, st);
    }
    return cudaErrorInvalidValue;
}

}  // namespace lwacm
