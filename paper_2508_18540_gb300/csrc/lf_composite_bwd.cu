// lf_composite_bwd.cu -- the adjoint of the swizzle blending.
#include "lf_composite.cuh"

namespace lf {

namespace {

// ---------------------------------------------------------------------------
// Adjoint of the swizzle blending. For one view pixel the forward computes
// Q = sum_k T_k C_k, T_{k+1} = T_k (1 - A_k), output (Q + T_N bg, 1 - T_N).
// With upstream gradient g = (g_rgb, g_a):
//   dL/dC_k = T_k g_rgb,   dL/dA_k = -T_k B_k,
//   B_k = sum_{j>k} (prod_{k<l<j} (1 - A_l)) C_j . g_rgb + (prod_{l>k} (1 - A_l)) (g_rgb . bg - g_a),
//   B_{k-1} = C_k . g_rgb + (1 - A_k) B_k.
// B needs no transmittance; T_k is recovered back to front as
// T_{k+1} / (1 - A_k). Every view pixel has a stop plane: the saving
// forward's, or, found by a front-to-back walk of the adjoint's own, the
// plane before which the plain forward's flush took T as 0 or the first with
// A = 1; T_k is known in front of it (or behind the last plane) and the
// planes behind it get no gradient from the pixel. T in front of a stop
// plane is far from underflow (at least 2^-24 at the last flush test before
// it, at most four planes earlier, each leaving at least 2^-24).
//
// The forward's staged tiles are used (4 consumer warps, windows of plane
// rows in the ring). Nearest: a 16-byte atomic per sample cost more than its
// instructions (1.77 ms on 45 views of 512^2, N 64, with 35 % fewer instructions
// than a kernel that took 1.72), so a thread adds up the gradients of
// consecutive views while they sample the same texel (neighbouring views shift
// by under a texel near the focal plane) and adds a run to dplanes with one FP32
// vector atomic. With the runs no unit is the bound alone (from saved state, FP32:
// issue slots 61 % busy, requests from L1 to L2 54 %, L2's atomic units 32 %, DRAM
// 9 %, at 18 warps per SM). Three views' texels are loaded before
// their steps back, so that the loads overlap. (Summing a plane's gradients
// per warp in shared memory first takes 12 to 16 shared-memory wavefronts a
// sample, where the texel and the atomic take 8: 1.72 ms.)
// Bilinear: a sample has four taps, and 32 neighbouring pixels of VG
// neighbouring views sample little more than two rows of 32 texels. The warp
// blends its window of the two plane rows into an FP32 row, as the forward
// does, sums the gradients of that row's texels in shared memory (left taps,
// then right taps), and adds them to dplanes once per plane, split by the row
// weights. One view at a time the lanes add to distinct texels (read, add,
// write; no shared atomics): even and odd lanes have a window each, and
// lanes two apart never share a texel while neighbouring pixels advance by
// more than half a texel (P_s + gm > kPairStep). Other planes, and windows
// wider than the warp's, add straight to dplanes.
// The planes behind the last stop plane of a warp's pixels in a triple of
// views (view columns 3 m .. 3 m + 2) are not walked for it: they carry T = 0
// for all of them, and what the stop planes' alpha gradients miss on ragged
// rows is below kTBehind of a colour times its gradient.
// ---------------------------------------------------------------------------
constexpr float kPairStep = 0.51f;
// The planes behind a stop plane k carry no gradient, but dL/dA_k = -T_k B_k
// holds their colours. On ragged rows they are walked for B with T_k above
// this, as the adjoint of such rows always did (16 views of 203^2, N 128, BF16,
// from saved state: 303 us without, 308 with 2^-18, 395 with 2^-20). On rows of
// whole 16-byte words they are not, and never were: where no pixel of a warp
// goes further, the alpha gradient of an opaque texel leaves out the colours
// behind it (a fitting step of 300k Gaussians would take 3.13 ms instead of
// 3.09).
constexpr float kTBehind = 3.814697265625e-6f;   // 2^-18

// alpha of staged texel i of a row
template <int DT>
__device__ __forceinline__ float texel_alpha(uint32_t row, uint32_t i);
template <>
__device__ __forceinline__ float texel_alpha<LF_F32>(uint32_t row, uint32_t i)
{
    return lds_f1(row + i * 16u + 12u);
}
template <>
__device__ __forceinline__ float texel_alpha<LF_F16>(uint32_t row, uint32_t i)
{
    return __half2float(__ushort_as_half(lds<unsigned short>(row + i * 8u + 6u)));
}
template <>
__device__ __forceinline__ float texel_alpha<LF_BF16>(uint32_t row, uint32_t i)
{
    return __uint_as_float((uint32_t)lds<unsigned short>(row + i * 8u + 6u) << 16);
}
template <>
__device__ __forceinline__ float texel_alpha<LF_U8>(uint32_t row, uint32_t i)
{
    return u8_byte<3>(lds_u32(row + i * 4u)) * (1.0f / 255.0f);
}

// Walk state of a thread's views.
template <int VG>
struct BwdViews {
    float T[VG], B[VG];
    int stop[VG];      // plane index in front of which T stands (N: behind the last); -1: no such view
    float4 g[VG];
};

__device__ __forceinline__ void add_smem(uint32_t a, float4 v)
{
    const float4 t = lds_f4(a);
    sts_f4(a, make_float4(t.x + v.x, t.y + v.y, t.z + v.z, t.w + v.w));
}

__device__ __forceinline__ float rcp_approx(float x)
{
    float y;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

// The view's step back over a plane sampled as t: T in front of it, the texel
// gradient (T g_rgb, -T B), and B in front of it. False: no gradient.
// T / oma is T times the approximate reciprocal; EXACT adds one correction by
// the quotient's own remainder (Markstein, IBM J. Res. Dev. 34, 1990), within a
// rounding of the true quotient. FP32 planes go without, as their kernel always
// did (3 % of a 512^2 adjoint); the others, whose ragged rows were divided, have
// it (ragged FP16, 21 views of 301^2, N 60: 642 -> 662 us, with the division
// itself 808).
template <bool EXACT, int VG>
__device__ __forceinline__ bool step_back(BwdViews<VG>& s, int jj, int k, float4 t, float4* gt)
{
    const float oma = 1.0f - t.w;
    if (k < s.stop[jj] && oma > 0.0f) {
        const float r = rcp_approx(oma);
        float q = s.T[jj] * r;
        if (EXACT) q = fmaf(fmaf(-q, oma, s.T[jj]), r, q);
        s.T[jj] = q;
    }
    const float T = s.T[jj], B = s.B[jj];
    const float4 g = s.g[jj];
    *gt = make_float4(T * g.x, T * g.y, T * g.z, -T * B);
    s.B[jj] = fmaf(t.x, g.x, fmaf(t.y, g.y, fmaf(t.z, g.z, oma * B)));
    return k <= s.stop[jj];
}

// FS: started from the state the saving forward wrote (one walk, back to
// front); else a front-to-back walk of the opacities first.
template <int DT, bool BILINEAR, int VG, bool FS>
__global__ void __launch_bounds__(kCompBlock, comp_bwd_ctas(VG, BILINEAR))
    k_composite_bwd_staged(const __grid_constant__ CompParams p, const __grid_constant__ CompGeom G,
                           const char* __restrict__ planes, const __grid_constant__ CompWs w,
                           const float4* __restrict__ dviews, float4* __restrict__ dplanes,
                           const float4* __restrict__ state)
{
    extern __shared__ __align__(128) unsigned char smem[];
    const TileSmem sm(G, smem);
    constexpr bool LONG = BILINEAR;   // descriptors with the warps' windows
    constexpr bool kExact = DT != LF_F32;
    __shared__ int s_kmax, s_n;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int nvg = G.groups_x * p.Vy;
    const int vgroup = blockIdx.x % nvg;
    const int vi = vgroup / G.groups_x, j0 = (vgroup % G.groups_x) * VG;
    const int X0 = (blockIdx.x / nvg) * G.TX, Y0 = blockIdx.y * G.BY;
    pdl_wait();
    const int P = *w.np;
    const float* blk = w.blk + (size_t)(vgroup % G.groups_x) * p.N * CoefBlock<VG>::kFloats;
    const float2* yt = w.yt + (size_t)vi * p.N;
    if (tid == 0) {
        sm.init(G);
        s_kmax = -1;
    }
    __syncthreads();
    Ring ring;
    const bool producer = tid >= kCompThreads;
    const int tx = tid % G.TX, ty = tid / G.TX;
    const int x = X0 + tx, y = Y0 + ty;
    const bool live = !producer && x < p.Nx && y < p.Ny;
    const ThreadGeom tg = thread_geom(p, G, x, y, ty);
    const size_t plane_sz = (size_t)p.W * p.H;
    // per warp: gradient sums of the even lanes, of the odd ones (wcap texels
    // each), bilinear: the blended row
    const uint32_t wrow = sm.warp_rows + (uint32_t)warp * G.wcap * (BILINEAR ? 48u : 32u);
    const uint32_t orow = wrow + G.wcap * 16u, brow = orow + G.wcap * 16u;
    const float4 zero4 = make_float4(0.f, 0.f, 0.f, 0.f);

    BwdViews<VG> s;
#pragma unroll
    for (int jj = 0; jj < VG; ++jj) {
        s.T[jj] = 1.f;
        s.stop[jj] = live && j0 + jj < p.Vx ? p.N : -1;
    }
    if constexpr (FS) {
        // state {T_k, k}: T in front of plane k, 0 behind it (the saving
        // forward stopped there); k = N: T behind the last plane
        if (live) {
#pragma unroll
            for (int jj = 0; jj < VG; ++jj) {
                if (j0 + jj >= p.Vx) break;
                const float4 sv = state[((size_t)(vi * p.Vx + j0 + jj) * p.Ny + y) * p.Nx + x];
                s.T[jj] = sv.x;
                s.stop[jj] = __float_as_int(sv.y);
            }
        }
    } else if (producer) {
        if (!produce<DT, BILINEAR, VG, false, true, LONG>(p, G, planes, blk, yt, P, X0, Y0, sm, ring, p.N)) {
            atomicExch(w.err, 1);
            if (lane == 0) *reinterpret_cast<volatile int*>(sm.end) = -1;
        }
    } else {
        // front to back, opacities only: T in front of each view's stop plane
        bool done = false;   // every view of the warp has stopped
        for (int q = 0; q < P; q += kPair) {
            if (!mbar_wait_bounded(sm.full + 8 * ring.st, ring.ph)) {
                atomicExch(w.err, 1);
                *reinterpret_cast<volatile int*>(sm.end) = -1;
                break;
            }
            const uint32_t empty = sm.empty + 8 * ring.st;
            uint32_t sa = sm.stages + (uint32_t)ring.st * G.stage_bytes;
            ring.next(G.stages);
            if (done && q >= *reinterpret_cast<volatile int*>(sm.end)) {
                __syncwarp();
                if (lane == 0) mbar_arrive(empty);
                break;
            }
            for (int u = 0; u < min(kPair, P - q); ++u, sa += G.plane_bytes) {
            const uint32_t d = sm.desc + (LONG ? 64u : kDescBytes) * (uint32_t)((q + u) & (kDescs - 1));
            const float4 A = lds_f4(d);
            const int kw = __float_as_int(A.z), mode = (kw >> tg.mode_sh) & 3, k = kw >> 8;
            if (u == 0 && (q & 3) == 0 && q > 0 && !done) {
                bool all = true;
#pragma unroll
                for (int jj = 0; jj < VG; ++jj) {
                    if (s.stop[jj] == p.N && s.T[jj] < kTFlush) s.stop[jj] = k;
                    all = all && s.stop[jj] != p.N;
                }
                done = __all_sync(0xffffffffu, all);
                if (done && lane == 0) atomicAdd(sm.sat, 1);
            }
            if (!done && mode != kSkip) {
                const float4 B = lds_f4(d + 16);
                const int first = __float_as_int(A.y);
                float a[VG];
                ViewH vh;
                if constexpr (!BILINEAR) {
                    const int iy = tg.psy + (__float_as_int(floor_magic<true>(B.x, tg.yf, B.y)) - kMagicBits);
                    const size_t grow = ((size_t)k * p.H + iy) * p.W;
#pragma unroll
                    for (int jj = 0; jj < VG; ++jj) {
                        const int ix =
                            __float_as_int(floor_magic<true>(A.x, tg.xf, vh.template get<VG>(sa, A.w, jj))) + tg.pxm;
                        a[jj] = 0.f;
                        if ((uint32_t)ix >= (uint32_t)p.W) continue;
                        a[jj] = mode == kGlobal ? load_texel<DT>(planes, grow + ix).w
                                                : texel_alpha<DT>(sa + tg.row, (uint32_t)(ix - first));
                    }
                } else {
                    const RowPair rp(p, tg, B.x, B.y);
                    const int lo = (int)lds_u32(d + 32 + 4 * warp), n = (int)lds_u32(d + 48 + 4 * warp);
                    const bool fits = n < (int)G.wcap;
                    if (n > 0 && fits) {
                        __syncwarp();   // the plane before has been read
                        blend_rows<DT>(p, planes, sa, tg, G, rp, mode, k, first, lo, n, brow);
                        __syncwarp();
                    }
#pragma unroll
                    for (int jj = 0; jj < VG; ++jj) {
                        float wx;
                        const int i0 = (int)tap_bits(A.x, tg.xf, vh.template get<VG>(sa, A.w, jj), true, wx) + tg.pxm;
                        const float wa = 1.0f - wx;
                        float u0 = 0.f, u1 = 0.f;
                        if (n > 0 && fits) {
                            if ((uint32_t)i0 < (uint32_t)p.W) u0 = lds_f1(brow + (uint32_t)(i0 - lo) * 16u + 12u);
                            if ((uint32_t)(i0 + 1) < (uint32_t)p.W)
                                u1 = lds_f1(brow + (uint32_t)(i0 + 1 - lo) * 16u + 12u);
                        } else if (n > 0) {
                            float4 t1;
                            u0 = sample_global<DT>(p, planes, k, rp, i0, &t1).w;
                            u1 = t1.w;
                        }
                        a[jj] = fmaf(wa, u0, wx * u1);
                    }
                }
#pragma unroll
                for (int jj = 0; jj < VG; ++jj) {
                    if (s.stop[jj] != p.N) continue;
                    const float oma = 1.0f - a[jj];
                    if (oma > 0.0f)
                        s.T[jj] *= oma;
                    else
                        s.stop[jj] = k;
                }
            }
            }
            __syncwarp();
            if (lane == 0) mbar_arrive(empty);
        }
    }

    // last stop plane of every triple of views over the warp's pixels
    constexpr int NT = (VG + 2) / 3;
    int km[NT], kmax = -1;
#pragma unroll
    for (int t = 0; t < NT; ++t) {
        int m = -1;
        if (!producer) {
#pragma unroll
            for (int jj = 3 * t; jj < 3 * t + 3 && jj < VG; ++jj)
                m = max(m, DT != LF_F32 && !G.bulk && s.stop[jj] >= 0 && s.T[jj] > kTBehind ? p.N : s.stop[jj]);
        }
        km[t] = __reduce_max_sync(0xffffffffu, m);
        kmax = max(kmax, km[t]);
    }
    if (lane == 0) atomicMax(&s_kmax, kmax);
    __syncthreads();
    if (!FS && *reinterpret_cast<volatile int*>(sm.end) < 0) return;   // a wait gave up
    if (producer) {
        // list entries up to the CTA's last stop plane
        int n = P;
        while (n > 0) {
            const int e = n - 1 - lane;
            const bool keep = e >= 0 && (__float_as_int(__ldg(blk + (size_t)e * CoefBlock<VG>::kFloats + 3)) &
                                         ~kWideBit) <= s_kmax;
            const unsigned m = __ballot_sync(0xffffffffu, keep);
            if (m) {
                n -= __ffs(m) - 1;
                break;
            }
            n = max(n - 32, 0);
        }
        if (lane == 0) s_n = n;
    } else {
        if (BILINEAR)
            for (int c = lane; c < 2 * (int)G.wcap; c += 32) sts_f4(wrow + 16u * (uint32_t)c, zero4);
    }
    __syncthreads();
    const int n2 = s_n;
    if (producer) {
        if (!produce<DT, BILINEAR, VG, true, false, LONG>(p, G, planes, blk, yt, n2, X0, Y0, sm, ring, n2)) atomicExch(w.err, 1);
        return;
    }
#pragma unroll
    for (int jj = 0; jj < VG; ++jj) {
        s.g[jj] = s.stop[jj] >= 0 ? dviews[view_pixel(p, vi * p.Vx + j0 + jj, x, y)] : zero4;
        s.B[jj] = fmaf(s.g[jj].x, p.bg[0], fmaf(s.g[jj].y, p.bg[1], fmaf(s.g[jj].z, p.bg[2], -s.g[jj].w)));
    }

    // back to front: T, texel gradients, the B recurrence
    for (int i0 = 0; i0 < n2; i0 += kPair, ring.next(G.stages)) {
        if (!mbar_wait_bounded(sm.full + 8 * ring.st, ring.ph)) {
            atomicExch(w.err, 1);
            return;
        }
        uint32_t sa = sm.stages + (uint32_t)ring.st * G.stage_bytes;
        for (int i = i0; i < min(n2, i0 + kPair); ++i, sa += G.plane_bytes) {
        const uint32_t d = sm.desc + (LONG ? 64u : kDescBytes) * (uint32_t)(i & (kDescs - 1));
        const float4 A = lds_f4(d);
        const int kw = __float_as_int(A.z), mode = (kw >> tg.mode_sh) & 3, k = kw >> 8;
        if (k <= kmax && mode != kSkip) {
            const float4 Bq = lds_f4(d + 16);
            const int first = __float_as_int(A.y);
            float4* dk = dplanes + (size_t)k * plane_sz;
            ViewH vh;
            if constexpr (!BILINEAR) {
                const int iy = tg.psy + (__float_as_int(floor_magic<true>(Bq.x, tg.yf, Bq.y)) - kMagicBits);
                const uint32_t base = sa + tg.row + (uint32_t)(tg.pxm - first) * (uint32_t)Texel<DT>::kBytes;
                // + floor bits = the texel
                float4* drow = dk + ((ptrdiff_t)iy * p.W + tg.pxm);
// the gradient of a run of views that sample the same texel
                float4 run = zero4;
                uint32_t rb = 0u;   // its floor bits (0: none yet)
#pragma unroll
                for (int t = 0; t < NT; ++t) {
                    float h[3];
#pragma unroll
                    for (int e = 0; e < 3 && 3 * t + e < VG; ++e) h[e] = vh.template get<VG>(sa, A.w, 3 * t + e);
                    if (k > km[t]) continue;
                    // the triple's texels first: their loads overlap
                    uint32_t b[3];
                    float4 tx[3];
                    bool in[3];
#pragma unroll
                    for (int e = 0; e < 3 && 3 * t + e < VG; ++e) {
                        in[e] = true;
                        if (mode == kInside) {
                            b[e] = __float_as_uint(floor_magic<false>(A.x, tg.xf, h[e]));
                            tx[e] = Texel<DT>::load(base + b[e] * (uint32_t)Texel<DT>::kBytes, 0u);
                        } else {
                            b[e] = __float_as_uint(floor_magic<true>(A.x, tg.xf, h[e]));
                            const uint32_t ix = b[e] + (uint32_t)tg.pxm;
                            in[e] = ix < (uint32_t)p.W;
                            tx[e] = zero4;
                            if (in[e])
                                tx[e] = mode == kGlobal
                                            ? load_texel<DT>(planes, ((size_t)k * p.H + iy) * p.W + ix)
                                            : Texel<DT>::load(base + b[e] * (uint32_t)Texel<DT>::kBytes, 0u);
                        }
                    }
#pragma unroll
                    for (int e = 0; e < 3 && 3 * t + e < VG; ++e) {
                        float4 gt;
                        if (!step_back<kExact>(s, 3 * t + e, k, tx[e], &gt) || !in[e]) gt = zero4, b[e] = rb;
                        const bool fresh = b[e] != rb;
                        if (fresh && rb) atomicAdd(drow + rb, run);
                        run.x = fresh ? gt.x : run.x + gt.x;
                        run.y = fresh ? gt.y : run.y + gt.y;
                        run.z = fresh ? gt.z : run.z + gt.z;
                        run.w = fresh ? gt.w : run.w + gt.w;
                        rb = b[e];
                    }
                }
                if (rb) atomicAdd(drow + rb, run);
            } else {
                const RowPair rp(p, tg, Bq.x, Bq.y);
                const int lo = (int)lds_u32(d + 32 + 4 * warp), n = (int)lds_u32(d + 48 + 4 * warp);
                const bool fits = n < (int)G.wcap;
                const bool sums = fits && (float)p.P_s + A.x > kPairStep;   // else straight to dplanes
                const uint32_t acc = lane & 1 ? orow : wrow;
                if (n <= 0) continue;
                float4* drow = dk + (ptrdiff_t)rp.y0 * p.W;   // rows outside the plane are not written
                if (fits) {
                    __syncwarp();   // the plane before has been read
                    blend_rows<DT>(p, planes, sa, tg, G, rp, mode, k, first, lo, n, brow);
                    __syncwarp();
                }
#pragma unroll
                for (int jj = 0; jj < VG; ++jj) {
                    const float h = vh.template get<VG>(sa, A.w, jj);
                    if (k > km[jj / 3]) continue;
                    float wx;
                    const int i0 = (int)tap_bits(A.x, tg.xf, h, true, wx) + tg.pxm;
                    const float wa = 1.0f - wx;
                    const bool c0 = (uint32_t)i0 < (uint32_t)p.W, c1 = (uint32_t)(i0 + 1) < (uint32_t)p.W;
                    const uint32_t o0 = (uint32_t)(i0 - lo) * 16u;
                    float4 u0 = zero4, u1 = zero4;
                    if (fits) {
                        if (c0) u0 = lds_f4(brow + o0);
                        if (c1) u1 = lds_f4(brow + o0 + 16u);
                    } else {
                        u0 = sample_global<DT>(p, planes, k, rp, i0, &u1);
                    }
                    float4 gt;
                    const bool add = step_back<kExact>(s, jj, k, mix_taps(wx, u0, u1), &gt);
                    if (sums) {
                        if (add && c0) add_smem(acc + o0, make_float4(wa * gt.x, wa * gt.y, wa * gt.z, wa * gt.w));
                        __syncwarp();
                        if (add && c1) add_smem(acc + o0 + 16u, make_float4(wx * gt.x, wx * gt.y, wx * gt.z, wx * gt.w));
                        __syncwarp();
                    } else {
                        const float ww[4] = {rp.w0 * wa, rp.w0 * wx, rp.w1 * wa, rp.w1 * wx};
#pragma unroll
                        for (int m = 0; m < 4; ++m)
                            if (add && (m & 1 ? c1 : c0) && (m >> 1 ? rp.w1 : rp.w0) != 0.0f)
                                atomicAdd(drow + (m >> 1) * p.W + i0 + (m & 1),
                                          make_float4(ww[m] * gt.x, ww[m] * gt.y, ww[m] * gt.z, ww[m] * gt.w));
                    }
                }
                if (sums) {
                    for (int c = lane; c < n; c += 32) {
                        const uint32_t a = 16u * (uint32_t)c;
                        const float4 u = lds_f4(wrow + a), v = lds_f4(orow + a);
                        const float4 w4 = make_float4(v.x + u.x, v.y + u.y, v.z + u.z, v.w + u.w);
                        if (w4.x != 0.f || w4.y != 0.f || w4.z != 0.f || w4.w != 0.f) {
                            float4* dst = drow + lo + c;
                            if (rp.w0 != 0.0f)
                                atomicAdd(dst, make_float4(rp.w0 * w4.x, rp.w0 * w4.y, rp.w0 * w4.z, rp.w0 * w4.w));
                            if (rp.w1 != 0.0f)
                                atomicAdd(dst + p.W, make_float4(rp.w1 * w4.x, rp.w1 * w4.y, rp.w1 * w4.z, rp.w1 * w4.w));
                        }
                        sts_f4(wrow + a, zero4);
                        sts_f4(orow + a, zero4);
                    }
                }
            }
        }
        }
        __syncwarp();
        if (lane == 0) mbar_arrive(sm.empty + 8 * ring.st);
    }
}

template <int DT, bool BILINEAR, int VG, bool FS>
void launch_bwd(const CompParams& p, const CompGeom& G, const void* planes, const CompWs& ws, const float4* dviews,
                float4* dplanes, const float4* state, cudaStream_t s)
{
    auto kern = k_composite_bwd_staged<DT, BILINEAR, VG, FS>;
    cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kCompSmemMax);
    const dim3 grid((unsigned)(G.groups_x * p.Vy * ((p.Nx + G.TX - 1) / G.TX)), (unsigned)((p.Ny + G.BY - 1) / G.BY));
    launch_pdl(kern, grid, dim3(kCompBlock), G.smem_bytes, s, p, G, static_cast<const char*>(planes), ws, dviews, dplanes,
               state);
}

struct BwdLaunch {
    const CompParams& p;
    const CompGeom& G;
    const void* planes;
    const CompWs& ws;
    const float4* dviews;
    float4* dplanes;
    const float4* state;
    cudaStream_t s;
    template <int DT, bool BILINEAR, int VG>
    void vg() const
    {
        if (state)
            launch_bwd<DT, BILINEAR, VG, true>(p, G, planes, ws, dviews, dplanes, state, s);
        else
            launch_bwd<DT, BILINEAR, VG, false>(p, G, planes, ws, dviews, dplanes, nullptr, s);
    }
    template <int DT, bool BILINEAR>
    void operator()() const
    {
        switch (G.VG) {
        case 9: vg<DT, BILINEAR, 9>(); break;
        default: vg<DT, BILINEAR, 3>(); break;
        }
    }
};

}  // namespace

void launch_composite_bwd(const CompParams& p, const void* planes, const CompWs& ws, const float* dviews,
                          float* dplanes, cudaStream_t s, const float4* state)
{
    const CompGeom G = comp_geom(p, planes, ws.VG, false, true, 128);
    dispatch(p.dtype, p.bilinear != 0, BwdLaunch{p, G, planes, ws, reinterpret_cast<const float4*>(dviews),
                                                 reinterpret_cast<float4*>(dplanes), state, s});
    note_launches(1);
}

}  // namespace lf
