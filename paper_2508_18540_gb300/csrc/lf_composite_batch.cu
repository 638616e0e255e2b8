// lf_composite_batch.cu -- the swizzle blending of several scenes in one launch.
#include "lf_composite.cuh"

namespace lf {

namespace {

// The tiles of several scenes in one grid (same plane type, sampling and
// views per thread). Item li of a scene: chunk group li % groups (a
// contiguous share of the non-empty planes), then view group, column tile,
// row band.
template <int DT, bool BILINEAR, int VG>
__global__ void __launch_bounds__(kCompBlock, comp_ctas(VG, BILINEAR, DT)) k_composite_batched(const CompScene* __restrict__ scs,
                                                                                 int n_sc)
{
    const long long it = blockIdx.x;
    int si = 0;
    while (si + 1 < n_sc && it >= scs[si + 1].base) ++si;
    const CompScene& sc = scs[si];
    const CompParams p = sc.p;
    const CompGeom G = sc.G;
    const CompWs w = sc.w;
    const long long li0 = it - sc.base;
    const int cgs = sc.groups, cg = (int)(li0 % cgs);
    const int nvg = G.groups_x * p.Vy;
    const long long li = li0 / cgs, rest = li / nvg;
    const int by = (int)(rest / sc.nbx), nby = (p.Ny + G.BY - 1) / G.BY;
    const int band = (by & 1) ? nby - 1 - (by >> 1) : (by >> 1);
    const int P = *w.np;
    const int q0 = (int)((long long)P * cg / cgs), q1 = (int)((long long)P * (cg + 1) / cgs);
    // partial (Q, T) of a chunk group: group 0 in the view buffer, group c > 0 in partial buffer c - 1
    float4* part = cg > 0 ? sc.part + (size_t)(cg - 1) * p.Vx * p.Vy * p.Ny * p.Nx : nullptr;
    composite_tile<DT, BILINEAR, VG, false>(p, G, sc.planes, w, sc.out, nullptr, part, cgs > 1, (int)(li % nvg),
                                            (int)(rest % sc.nbx) * G.TX, band * G.BY, q0, q1 - q0);
}

template <int DT, bool BILINEAR, int VG>
void launch_batched(const CompScene* scs, int n_sc, long long total, size_t smem, cudaStream_t s)
{
    auto kern = k_composite_batched<DT, BILINEAR, VG>;
    cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kCompSmemMax);
    kern<<<(unsigned)total, kCompBlock, smem, s>>>(scs, n_sc);
}

struct BatchLaunch {
    const CompScene* scs;
    int n_sc;
    long long total;
    int VG;
    size_t smem;
    cudaStream_t s;
    template <int DT, bool BILINEAR>
    void operator()() const
    {
        switch (VG) {
        case 15: launch_batched<DT, BILINEAR, 15>(scs, n_sc, total, smem, s); break;
        case 9: launch_batched<DT, BILINEAR, 9>(scs, n_sc, total, smem, s); break;
        case 5: launch_batched<DT, BILINEAR, 5>(scs, n_sc, total, smem, s); break;
        default: launch_batched<DT, BILINEAR, 3>(scs, n_sc, total, smem, s); break;
        }
    }
};

}  // namespace

void launch_composite_batched(const CompScene* scenes_dev, int n_sc, long long total, int dtype, bool bilinear,
                              int VG, size_t smem, cudaStream_t s)
{
    if (total <= 0) return;
    dispatch(dtype, bilinear, BatchLaunch{scenes_dev, n_sc, total, VG, smem, s});
    note_launches(1);
}

}  // namespace lf
