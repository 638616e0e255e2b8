// lf_bin.cu -- depth binning (the chunking step of Algorithm 1; Sec. 4.4) and
// the pairs of the 3D tiling (Sec. 4.4).
//
//  k_bin_emit  rank r of the (depth, index) order -> chunk:
//               quantile:  floor(r N / M)   (equal-count chunks)
//               disparity: min(N-1, floor(N (1/z_min - 1/z) / (1/z_min - 1/z_max)))
//             records the first rank of every chunk (chunks are monotone in
//             rank), copies the primitive's footprint, colour and projection
//             into rank order for the raster kernels, and writes one
//             (super-tile id, rank) pair per 32x32 super-tile that the
//             footprint touches, in rank (depth) order, with the totals of
//             the pairs' radix digits. A block's place among the pairs comes
//             from decoupled look-back (separate kernels for the copies, the
//             block totals, their scan and the pairs before).
//  median_plane  d_k = median member depth + D_forward (quantile; mean of the
//             two middle depths for an even count) or the bin's disparity
//             midpoint; run by the kernel after the pairs' sort.
// All FP64 operations use explicit round-to-nearest intrinsics in the order
// of the definitions above. The depth of rank r is the FP64 whose IEEE bits
// are the depth key of primitive valA[r] (keyA, by primitive). The gathers
// bound the binning (52 to 84 bytes at random per rank).
#include "lf_internal.cuh"
#include "lf_bin.cuh"

namespace lf {

namespace {

constexpr int kT = 256;

// 1 / z_min, 1 / z_min - 1 / z_max of the disparity bins, and in FP32 what
// decides a bin away from its edges
struct DispRange {
    double izmin, span;
    float izminf, scale, margin;   // N / span; error bound of the FP32 bin position
};

__device__ __forceinline__ int chunk_of_rank(const BuildWs& w, const BinParams& p, const DispRange& dr, long long r,
                                             long long M)
{
    if (p.binning == LF_BIN_QUANTILE) return (int)((r * (long long)p.N) / M);
    if (!(dr.span > 0.0)) return 0;
    const double z = rank_depth(w, r);
    // FP64 divisions run at two lanes a clock and SM, so the position is taken
    // in FP32 first; its error is at most 4 ulp of 1/z_min times N / span and
    // 4 ulp of N, and only positions within twice that of a bin edge need the
    // definition itself
    const float f32 = __fmul_rn(dr.scale, __fsub_rn(dr.izminf, __frcp_rn(__double2float_rn(z))));
    const float fl = floorf(f32), in = f32 - fl;
    if (in > dr.margin && in < 1.0f - dr.margin) return fl >= (float)(p.N - 1) ? p.N - 1 : (int)fl;
    const double f = floor(__ddiv_rn(__dmul_rn((double)p.N, __dsub_rn(dr.izmin, __ddiv_rn(1.0, z))), dr.span));
    return f >= (double)(p.N - 1) ? p.N - 1 : (int)f;
}

__device__ __forceinline__ uint32_t tile_count(int4 rc)
{
    if (rc.z < rc.x || rc.w < rc.y) return 0u;
    return (uint32_t)((rc.z / kSuper - rc.x / kSuper + 1) * (rc.w / kSuper - rc.y / kSuper + 1));
}

// The block's pairs are written to shared memory at their block-local
// offsets and copied out contiguously (coalesced): all at once while they fit
// into the staging area, else the pairs of 256 ranks at a time, and pairs of
// 256 ranks that don't fit directly.
constexpr int kEmitStage = 4096;   // pairs
// Up to this many super-tiles, a block with at least two pairs per super-tile
// counts its pairs per super-tile and folds the counts into the totals of the
// two digits at its end: the top digit of a 10-bit id has four values, and an
// atomic per pair on four words serialises (with the staging above: 48 -> 25 us
// for 5M pairs on 1024 super-tiles; with fewer pairs the folding costs more).
constexpr int kFoldSupers = 1024;

// Chunks and copies (BIN) and pairs (EMIT) of PER ranks per thread, kT apart.
// One kernel does both for few primitives, where launches and latencies
// count; for many, one kernel of one rank per thread gathers (it needs all the
// loads in flight that the registers allow) and another one emits from the
// rank-ordered footprints (both at once, 4 ranks per thread: 97 us at 943k
// voxels against 52 + 17).
template <int PER, bool BIN, bool EMIT>
__global__ void __launch_bounds__(kT, EMIT ? 4 : 6) k_bin_emit(BuildWs w, BinParams p, int32_t* chunk_out,
                                                 const int4* __restrict__ rect, const float* __restrict__ rgb,
                                                 const float* __restrict__ dens8, int kind, int supers_x,
                                                 int n_supers, int tile_passes)
{
    pdl_wait();
    pdl_trigger();
    __shared__ uint32_t s_key[EMIT ? kEmitStage : 1];
    __shared__ uint32_t s_rank[EMIT ? kEmitStage : 1];
    __shared__ uint32_t s_hist[EMIT ? kTilePassesMax : 1][kSortDigits];
    __shared__ uint32_t s_super[EMIT ? kFoldSupers : 1];
    __shared__ int s_chunk[BIN ? PER * kT : 1];
    __shared__ uint32_t s_warp[kT / 32];
    __shared__ uint32_t s_block;
    __shared__ unsigned long long s_base;
    __shared__ DispRange s_dr;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const long long M = (long long)w.hdr->M;
    if (tid == 0) {
        // After a wait gave up (of the sort, or in an earlier block here) valA is
        // no order: no block does anything. (Depths out of order give bins below
        // zero, and chunk_start would be written there.)
        s_block = EMIT ? atomicAdd(&w.hdr->ticket[kDepthPasses + kTilePassesMax], 1u)
                       : w.hdr->timeout ? kNoTicket : blockIdx.x;
        if (BIN && p.binning != LF_BIN_QUANTILE && M > 0) {
            // (read in bounds without waiting for the ticket, in order or not)
            const uint32_t last_prim = (uint32_t)(w.hdr->n - 1);
            const double zmin = __longlong_as_double((long long)w.keyA[min(w.valA[0], last_prim)]);
            const double zmax = __longlong_as_double((long long)w.keyA[min(w.valA[M - 1], last_prim)]);
            DispRange d;
            d.izmin = __ddiv_rn(1.0, zmin);
            d.span = __dsub_rn(d.izmin, __ddiv_rn(1.0, zmax));
            d.izminf = __double2float_rn(d.izmin);
            d.scale = (float)p.N / __double2float_rn(d.span);
            d.margin = 4.76837158e-7f * (d.scale * d.izminf + 2.0f * (float)p.N);   // 2^-21
            s_dr = d;
        }
    }
    const bool may_fold = tile_passes == 2 && n_supers <= kFoldSupers;
    if (EMIT) {
        for (int i = tid; i < kTilePassesMax * kSortDigits; i += kT) (&s_hist[0][0])[i] = 0u;
        if (may_fold)
            for (int i = tid; i < n_supers; i += kT) s_super[i] = 0u;
    }
    __syncthreads();
    const long long b = s_block, r0 = b * (PER * kT);
    if (s_block >= kNoTicket) return;
    if (M == 0) {
        if (BIN && b == 0)
            for (int k = tid; k <= p.N; k += kT) w.chunk_start[k] = 0;
        return;
    }
    if (r0 >= M) return;
    const DispRange dr = s_dr;

    int4 rc[PER];
    if (!BIN) {
#pragma unroll
        for (int j = 0; j < PER; ++j) {
            const long long r = r0 + j * kT + tid;
            rc[j] = r < M ? w.r_rect[r] : make_int4(0, 0, -1, -1);
        }
    } else {
        uint32_t g[PER];
#pragma unroll
        for (int j = 0; j < PER; ++j) {
            const long long r = r0 + j * kT + tid;
            g[j] = r < M ? w.valA[r] : 0u;
            rc[j] = r < M ? rect[g[j]] : make_int4(0, 0, -1, -1);
        }
#pragma unroll
        for (int j = 0; j < PER; ++j) {
            const long long r = r0 + j * kT + tid;
            if (r >= M) continue;
            const int c = chunk_of_rank(w, p, dr, r, M);
            s_chunk[j * kT + tid] = c;
            chunk_out[g[j]] = c;
            // rank-ordered copies
            w.r_chunk[r] = c;
            w.r_rect[r] = rc[j];
            const size_t gg = g[j];
            w.r_rgb[r] = make_float4(rgb[3 * gg], rgb[3 * gg + 1], rgb[3 * gg + 2], 0.f);
            if (kind == 0) {
                const float2 m = w.mean2d[gg];
                w.r_geo[r] = make_float4(m.x, m.y, 0.f, 0.f);
                w.r_con[r] = w.conic_o[gg];
            } else {
                w.r_geo[r] = w.conic_o[gg];
                const float4* d4 = reinterpret_cast<const float4*>(dens8 + 8 * gg);
                w.r_den[2 * r] = d4[0];
                w.r_den[2 * r + 1] = d4[1];
            }
        }
        __syncthreads();
        // first rank of every chunk
#pragma unroll
        for (int j = 0; j < PER; ++j) {
            const int i = j * kT + tid;
            const long long r = r0 + i;
            if (r >= M) continue;
            const int c = s_chunk[i], cp = r == 0 ? -1 : i > 0 ? s_chunk[i - 1] : chunk_of_rank(w, p, dr, r - 1, M);
            for (int k = cp + 1; k <= c; ++k) w.chunk_start[k] = (int32_t)r;
            if (r == M - 1)
                for (int k = c + 1; k <= p.N; ++k) w.chunk_start[k] = (int32_t)M;
        }
    }
    if (!EMIT) return;

    // block-local places of the pairs, in rank order
    uint32_t off[PER], start[PER + 1], total = 0;   // start: of all pairs of one j
#pragma unroll
    for (int j = 0; j < PER; ++j) {
        const uint32_t c = tile_count(rc[j]);
        uint32_t x = c;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t u = __shfl_up_sync(0xffffffffu, x, o);
            if (lane >= o) x += u;
        }
        __syncthreads();
        if (lane == 31) s_warp[warp] = x;
        __syncthreads();
        uint32_t before = 0, sum = 0;
#pragma unroll
        for (int q = 0; q < kT / 32; ++q) {
            before += q < warp ? s_warp[q] : 0u;
            sum += s_warp[q];
        }
        off[j] = total + before + x - c;
        start[j] = total;
        total += sum;
    }
    start[PER] = total;
    if (tid == 0) st_word(w.bstat + b, (b == 0 ? kSumAll : kSumOwn) | total);

    const bool staged = total <= (uint32_t)kEmitStage;
    const bool fold = may_fold && total >= 2u * (uint32_t)n_supers;
    auto emit = [&](int j, uint32_t* keys, uint32_t* ranks, uint32_t at) {
        if (rc[j].z < rc[j].x || rc[j].w < rc[j].y) return;
        const int sx0 = rc[j].x / kSuper, sx1 = rc[j].z / kSuper, sy0 = rc[j].y / kSuper, sy1 = rc[j].w / kSuper;
        uint32_t o = off[j] - at;
        for (int sy = sy0; sy <= sy1; ++sy)
            for (int sx = sx0; sx <= sx1; ++sx, ++o) {
                const uint32_t key = (uint32_t)(sy * supers_x + sx);
                keys[o] = key;
                ranks[o] = (uint32_t)(r0 + j * kT + tid);
                if (fold)
                    atomicAdd(&s_super[key], 1u);
                else
                    for (int q = 0; q < tile_passes; ++q) atomicAdd(&s_hist[q][(key >> (8 * q)) & 255u], 1u);
            }
    };
    auto copy_out = [&](unsigned long long to, uint32_t n) {
        for (uint32_t i = tid; i < n; i += kT) {
            w.tkeyA[to + i] = s_key[i];
            w.entA[to + i] = s_rank[i];
        }
    };
    if (staged) {
#pragma unroll
        for (int j = 0; j < PER; ++j) emit(j, s_key, s_rank, 0u);
    }

    // pairs of the blocks before this one (warp 0, 32 words per round trip)
    if (warp == 0) {
        unsigned long long base = 0;
        long long t = b - 1;
        int idle = 0;
        bool done = b == 0;
        while (!done) {
            const unsigned long long v = t - lane >= 0 ? ld_word(w.bstat + (t - lane)) : kSumAll;
            const unsigned missing = __ballot_sync(0xffffffffu, v < kSumOwn);
            const unsigned all = __ballot_sync(0xffffffffu, v >= kSumAll);
            const int nm = missing ? __ffs(missing) - 1 : 32, na = all ? __ffs(all) - 1 : 32;
            done = na < nm;
            const int use = done ? na + 1 : nm;
            unsigned long long x = lane < use ? v & kSumMask : 0ull;
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
            base += x;
            t -= use;
            idle = use ? 0 : idle + 1;
            if (idle > w.look_tries) {
                if (lane == 0) give_up(w.hdr);
                done = true;
            }
        }
        if (lane == 0) {
            if (b > 0) st_word(w.bstat + b, kSumAll | (base + total));
            s_base = base;
            if (r0 + (PER * kT) >= M) {   // the last block
                const unsigned long long all_pairs = base + total;
                const int over = all_pairs > (unsigned long long)w.hdr->dup_capacity;
                w.hdr->total_dups = all_pairs;
                w.hdr->overflow = over;
                w.hdr->tile_n = over ? 0ull : all_pairs;
            }
        }
    }
    __syncthreads();
    const unsigned long long base = s_base;
    if (base + total > (unsigned long long)w.hdr->dup_capacity) return;   // the last block reports the overflow
    if (staged) {
        copy_out(base, total);
    } else {   // the ranks of one j at a time, through the staging area where they fit
#pragma unroll
        for (int j = 0; j < PER; ++j) {
            const uint32_t cnt = start[j + 1] - start[j];
            if (cnt > (uint32_t)kEmitStage) {
                emit(j, w.tkeyA + base, w.entA + base, 0u);
                continue;
            }
            __syncthreads();
            emit(j, s_key, s_rank, start[j]);
            __syncthreads();
            copy_out(base + start[j], cnt);
        }
        __syncthreads();
    }
    if (fold) {
        for (int i = tid; i < n_supers; i += kT) {
            const uint32_t c = s_super[i];
            if (c) {
                atomicAdd(&s_hist[0][i & 255], c);
                atomicAdd(&s_hist[1][i >> 8], c);
            }
        }
        __syncthreads();
    }
    for (int i = tid; i < tile_passes * kSortDigits; i += kT) {
        const uint32_t c = (&s_hist[0][0])[i];
        if (c) atomicAdd(&w.dhist[kDepthPasses * kSortDigits + i], c);
    }
}

}  // namespace

void launch_bin(const BuildWs& ws, const BinParams& p, long long n, int32_t* chunk, const int32_t* rect,
                const float* rgb, const float* dens8, int kind, int supers_x, int n_supers, cudaStream_t s)
{
    const long long nn = n > 0 ? n : 1;
    const int tile_passes = tile_sort_passes(tile_bits_for(n_supers));
    const dim3 blocks((unsigned)((nn + ws.dup_block - 1) / ws.dup_block));
    const int4* rc = reinterpret_cast<const int4*>(rect);
    if (ws.dup_block == kT) {
        launch_pdl(k_bin_emit<1, true, true>, blocks, dim3(kT), 0, s, ws, p, chunk, rc, rgb, dens8, kind, supers_x,
                   n_supers, tile_passes);
        note_launches(1);
        return;
    }
    launch_pdl(k_bin_emit<1, true, false>, dim3((unsigned)((nn + kT - 1) / kT)), dim3(kT), 0, s, ws, p, chunk, rc, rgb,
               dens8, kind, supers_x, n_supers, tile_passes);
    launch_pdl(k_bin_emit<4, false, true>, blocks, dim3(kT), 0, s, ws, p, chunk, rc, rgb, dens8, kind, supers_x,
               n_supers, tile_passes);
    note_launches(2);
}

}  // namespace lf
