// lf_bin.cuh -- depths by rank and the plane distances (see lf_bin.cu).
#pragma once

#include "lf_internal.cuh"

namespace lf {

__device__ __forceinline__ double rank_depth(const BuildWs& w, long long r)
{
    return __longlong_as_double((long long)w.keyA[w.valA[r]]);
}

// member count and distance of plane k
__device__ __forceinline__ void median_plane(const BuildWs& w, const BinParams& p, int k, double* d_out,
                                             int32_t* count_out)
{
    if (w.hdr->timeout) {   // the order is not valid: no plane
        count_out[k] = 0;
        d_out[k] = 0.0;
        return;
    }
    const long long M = (long long)w.hdr->M;
    const int lo = w.chunk_start[k], hi = w.chunk_start[k + 1];
    const int c = hi - lo;
    count_out[k] = c;
    double d = 0.0;
    if (p.binning == LF_BIN_QUANTILE) {
        if (c > 0) {
            double med;
            if (c & 1)
                med = rank_depth(w, lo + c / 2);
            else
                med = __dmul_rn(__dadd_rn(rank_depth(w, lo + c / 2 - 1), rank_depth(w, lo + c / 2)), 0.5);
            d = __dadd_rn(med, p.D_forward);
        }
    } else if (M > 0) {
        const double izmin = __ddiv_rn(1.0, rank_depth(w, 0));
        const double izmax = __ddiv_rn(1.0, rank_depth(w, M - 1));
        const double span = __dsub_rn(izmin, izmax);
        const double disp = __dsub_rn(izmin, __dmul_rn(__ddiv_rn(__dadd_rn((double)k, 0.5), (double)p.N), span));
        d = __dadd_rn(__ddiv_rn(1.0, disp), p.D_forward);
    }
    d_out[k] = d;
}

}  // namespace lf
