// lf_tiles.cu -- 3D tiling (Sec. 4.4), two levels: lists are built per
// (32x32 super-tile, chunk) and every raster CTA (16x16 tile, chunk) filters
// its super-tile's list down to the primitives whose footprint meets its
// tile, keeping the order.
//
//  k_bin_emit (lf_bin.cu)
//      one (super-tile id, rank) pair per super-tile a primitive's footprint
//      touches, written in rank (depth) order;
//  sort_tile_keys (lf_sort.cu)
//      stable radix sort of the pairs by super-tile id: every list stays in
//      depth order, and chunks (monotone in rank) form contiguous runs;
//  k_ranges
//      [start, end) of every (super-tile, chunk) run; the plane distances.
#include "lf_internal.cuh"
#include "lf_bin.cuh"

namespace lf {

namespace {

// Entry i starts a (super-tile, chunk) list when its super-tile or chunk
// differs from entry i - 1's; it then also ends the list of entry i - 1. A
// warp takes 32 consecutive entries: the chunk of an entry's rank comes from
// the rank-ordered chunk array, the previous entry's from the lane below.
// The first med_blocks blocks take the plane distances instead.
__global__ void __launch_bounds__(256) k_ranges(BuildWs w, BinParams p, const uint32_t* __restrict__ keys,
                                                const uint32_t* __restrict__ ranks, int med_blocks,
                                                double* __restrict__ d_out, int32_t* __restrict__ count_out)
{
    pdl_wait();
    pdl_trigger();
    const int N = p.N;
    if ((int)blockIdx.x < med_blocks) {
        const int k = blockIdx.x * blockDim.x + threadIdx.x;
        if (k < N) median_plane(w, p, k, d_out, count_out);
        return;
    }
    const long long n = w.hdr->timeout ? 0 : (long long)w.hdr->tile_n;   // after a wait gave up: no list
    const int lane = threadIdx.x & 31;
    const long long stride = (long long)(gridDim.x - med_blocks) * blockDim.x;
    for (long long i0 = (long long)(blockIdx.x - med_blocks) * blockDim.x + (threadIdx.x - lane); i0 < n; i0 += stride) {
        const long long i = i0 + lane;
        const bool in = i < n;
        const uint32_t t = in ? keys[i] : 0u;
        const int c = in ? w.r_chunk[ranks[i]] : 0;
        uint32_t tp = __shfl_up_sync(0xffffffffu, t, 1);
        int cp = __shfl_up_sync(0xffffffffu, c, 1);
        if (lane == 0 && in && i > 0) {
            tp = keys[i - 1];
            cp = w.r_chunk[ranks[i - 1]];
        }
        if (!in) continue;
        const bool first = i == 0 || tp != t || cp != c;
        if (first) {
            w.seg[(long long)t * N + c].x = (int)i;
            if (i > 0) w.seg[(long long)tp * N + cp].y = (int)i;
        }
        if (i == n - 1) w.seg[(long long)t * N + c].y = (int)n;
    }
}

}  // namespace

int tile_bits_for(long long tiles)
{
    int b = 1;
    while ((1ll << b) < tiles) ++b;
    return b;
}

const uint32_t* launch_tile_lists(const BuildWs& ws, const BinParams& p, long long cap, int supers_x, int n_supers,
                                  double* d, int32_t* count, cudaStream_t s)
{
    uint32_t* keys = nullptr;
    uint32_t* ranks = nullptr;
    sort_tile_keys(ws, cap, tile_bits_for(n_supers), s, &keys, &ranks);
    const long long want = (cap + 255) / 256;
    const int med = (p.N + 255) / 256;
    const unsigned blocks = (unsigned)(med + (want < 152 * 16 ? want : 152 * 16));
    launch_pdl(k_ranges, dim3(blocks), dim3(256), 0, s, ws, p, keys, ranks, med, d, count);
    note_launches(1);
    return ranks;
}

}  // namespace lf
