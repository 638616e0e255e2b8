// lf_filter.cu -- the V2LF low-pass plane filter (Sec. 4.5), in place.
//
// SVR's supersampling is replaced by a Gaussian low-pass filter on the
// sweeping planes, done in place with no extra memory. Separable: a normalised
// discrete Gaussian w[-r..r] (standard deviation sigma, in plane pixels) over
// the rows, then over the columns, every RGBA channel, transparent zero
// padding outside the plane, FP32 arithmetic, result stored in the plane type.
//  k_filter_fused both passes in one walk, a cluster of CTAs per plane: every
//                 texel is read once (and a halo) and written once; many
//                 planes of up to 512 columns.
//  The other planes take two passes:
//  k_filter_rows  one CTA per (plane, row): the row is walked in segments;
//                 each segment and its right halo are read into shared
//                 memory, the left halo is the previous segment's tail of
//                 original texels carried in shared memory, so writing the
//                 segment back never destroys an input still needed.
//  k_filter_cols  one CTA per (plane, strip of 32 columns), 8 threads per
//                 column: walks down the strip in bands of 32 rows; each
//                 band and the r rows below it are read into shared memory
//                 (the r rows above are the previous band's tail of original
//                 texels, carried with the look-ahead), so writing the band
//                 back never destroys an input still needed. Every texel is
//                 read once and written once.
#include <cuda_bf16.h>
#include <cuda_fp16.h>

#include <type_traits>

#include "lf_internal.cuh"

namespace lf {

namespace {

constexpr int kRowThreads = 256;
constexpr int kSeg = 1024;          // texels per row segment
constexpr int kColStrip = 32;   // columns per CTA of the column pass
constexpr int kColLanes = 8;    // threads per column
constexpr int kColBand = 32;    // output rows per step (>= 2 * kFilterMaxRadius: the carry never overlaps)
static_assert(kColBand >= 2 * kFilterMaxRadius, "column carry would overlap");

// a stored texel, and its FP32 channels
template <int DT>
using Stored = std::conditional_t<DT == LF_F32, float4, std::conditional_t<DT == LF_U8, uint32_t, uint2>>;

template <int DT>
__device__ __forceinline__ float4 widen(Stored<DT> u)
{
    if constexpr (DT == LF_F32) {
        return u;
    } else if constexpr (DT == LF_U8) {
        return u8_unpack(u);
    } else if constexpr (DT == LF_F16) {
        const float2 a = __half22float2(*reinterpret_cast<const __half2*>(&u.x));
        const float2 b = __half22float2(*reinterpret_cast<const __half2*>(&u.y));
        return make_float4(a.x, a.y, b.x, b.y);
    } else {
        const float2 a = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&u.x));
        const float2 b = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&u.y));
        return make_float4(a.x, a.y, b.x, b.y);
    }
}

template <int DT>
__device__ __forceinline__ float4 ld(const void* p, size_t i)
{
    return widen<DT>(reinterpret_cast<const Stored<DT>*>(p)[i]);
}

template <int DT>
__device__ __forceinline__ void st(void* p, size_t i, float4 v)
{
    if (DT == LF_F32) {
        reinterpret_cast<float4*>(p)[i] = v;
    } else if (DT == LF_U8) {
        reinterpret_cast<uint32_t*>(p)[i] = u8_pack(v.x, v.y, v.z, v.w);
    } else if (DT == LF_F16) {
        const __half2 lo = __floats2half2_rn(v.x, v.y), hi = __floats2half2_rn(v.z, v.w);
        uint2 u;
        u.x = *reinterpret_cast<const uint32_t*>(&lo);
        u.y = *reinterpret_cast<const uint32_t*>(&hi);
        reinterpret_cast<uint2*>(p)[i] = u;
    } else {
        const __nv_bfloat162 lo = __floats2bfloat162_rn(v.x, v.y), hi = __floats2bfloat162_rn(v.z, v.w);
        uint2 u;
        u.x = *reinterpret_cast<const uint32_t*>(&lo);
        u.y = *reinterpret_cast<const uint32_t*>(&hi);
        reinterpret_cast<uint2*>(p)[i] = u;
    }
}

__device__ __forceinline__ void fma4(float4& a, float w, float4 v)
{
    a.x = fmaf(w, v.x, a.x);
    a.y = fmaf(w, v.y, a.y);
    a.z = fmaf(w, v.z, a.z);
    a.w = fmaf(w, v.w, a.w);
}

template <int DT>
__global__ void __launch_bounds__(kRowThreads) k_filter_rows(void* planes, int W, int H, FilterParams f)
{
    extern __shared__ float4 buf[];   // [r + kSeg + r]: left halo, segment, right halo
    const int r = f.radius;
    const size_t row = (size_t)blockIdx.x;          // plane * H + y
    const size_t base = row * (size_t)W;
    for (int i = threadIdx.x; i < r; i += kRowThreads) buf[i] = make_float4(0.f, 0.f, 0.f, 0.f);
    for (int x0 = 0; x0 < W; x0 += kSeg) {
        const int n = min(kSeg, W - x0);
        for (int i = threadIdx.x; i < n + r; i += kRowThreads) {
            const int x = x0 + i;
            buf[r + i] = x < W ? ld<DT>(planes, base + x) : make_float4(0.f, 0.f, 0.f, 0.f);
        }
        __syncthreads();
        float4 out[kSeg / kRowThreads];
#pragma unroll
        for (int q = 0; q < kSeg / kRowThreads; ++q) {
            const int i = threadIdx.x + q * kRowThreads;
            float4 a = make_float4(0.f, 0.f, 0.f, 0.f);
            if (i < n)
                for (int t = -r; t <= r; ++t) fma4(a, f.w[t + r], buf[r + i + t]);
            out[q] = a;
        }
        __syncthreads();
        // carry the segment's last r original texels as the next left halo
        if (n == kSeg)
            for (int i = threadIdx.x; i < r; i += kRowThreads) buf[i] = buf[kSeg + i];
#pragma unroll
        for (int q = 0; q < kSeg / kRowThreads; ++q) {
            const int i = threadIdx.x + q * kRowThreads;
            if (i < n) st<DT>(planes, base + x0 + i, out[q]);
        }
        __syncthreads();
    }
}

template <int DT>
__global__ void __launch_bounds__(kColStrip* kColLanes) k_filter_cols(void* planes, int W, int H, FilterParams f)
{
    extern __shared__ float4 cbuf[];   // rows [r + kColBand + r][kColStrip]: top halo, band, look-ahead
    const int r = f.radius;
    const int tx = threadIdx.x % kColStrip, ty = threadIdx.x / kColStrip;
    const int x = blockIdx.x * kColStrip + tx;
    const bool col = x < W;
    const size_t plane = (size_t)blockIdx.y * (size_t)W * H;
    const float4 zero = make_float4(0.f, 0.f, 0.f, 0.f);
    // rows -r .. r - 1 of the first band: zero padding above, then originals
    for (int i = ty; i < 2 * r; i += kColLanes) {
        const int y = i - r;
        cbuf[i * kColStrip + tx] = (col && y >= 0 && y < H) ? ld<DT>(planes, plane + (size_t)y * W + x) : zero;
    }
    for (int y0 = 0; y0 < H; y0 += kColBand) {
        const int n = min(kColBand, H - y0);
        // rows y0 + r .. y0 + n + r - 1 (originals; zero below the plane);
        // rows y0 - r .. y0 + r - 1 are already in place
        for (int i = 2 * r + ty; i < n + 2 * r; i += kColLanes) {
            const int y = y0 + i - r;
            cbuf[i * kColStrip + tx] = (col && y < H) ? ld<DT>(planes, plane + (size_t)y * W + x) : zero;
        }
        __syncthreads();
        float4 out[kColBand / kColLanes];
#pragma unroll
        for (int q = 0; q < kColBand / kColLanes; ++q) {
            const int i = ty + q * kColLanes;
            float4 a = zero;
            if (i < n)
                for (int t = -r; t <= r; ++t) fma4(a, f.w[t + r], cbuf[(r + i + t) * kColStrip + tx]);
            out[q] = a;
        }
        __syncthreads();
        // the band's last r rows and the look-ahead become the next band's
        // top halo and first rows (originals: nothing below y0 + n is written yet)
        if (n == kColBand)
            for (int i = threadIdx.x; i < 2 * r * kColStrip; i += blockDim.x) cbuf[i] = cbuf[kColBand * kColStrip + i];
#pragma unroll
        for (int q = 0; q < kColBand / kColLanes; ++q) {
            const int i = ty + q * kColLanes;
            if (col && i < n) st<DT>(planes, plane + (size_t)(y0 + i) * W + x, out[q]);
        }
        __syncthreads();
    }
}

// ---------------------------------------------------------------------------
// Both passes in one walk over a plane.
// ---------------------------------------------------------------------------
constexpr int kStrip = 64;            // columns per CTA
constexpr int kBand = 16;             // rows per step
constexpr int kFusedThreads = 256;    // 4 outputs per thread and pass: of one row, then of one column
constexpr int kStripsMax = 8;         // CTAs per cluster (portable size)
// One walk or two passes: a cluster takes a plane, so few planes leave SMs
// idle and the two-pass kernels, with a CTA per row, win. 512^2 FP32, radius 3:
// 24 planes 97 us (two passes 99), 32 99 (126), 64 164 (237); 256^2: 16 planes
// 38 (36), 24 38 (44); 128^2: 32 planes 23 (23), 64 23 (33); FP16 64 planes of
// 512^2 142 (208). Planes wider than eight strips don't fit a cluster.
constexpr int kFusedPlanes = 32, kFusedCtas = 64;

// the value that a store in the plane's type and a load back give
template <int DT>
__device__ __forceinline__ float4 as_stored(float4 v)
{
    if (DT == LF_F32) return v;
    if (DT == LF_U8) return u8_unpack(u8_pack(v.x, v.y, v.z, v.w));
    if (DT == LF_F16) {
        const float2 a = __half22float2(__floats2half2_rn(v.x, v.y)), b = __half22float2(__floats2half2_rn(v.z, v.w));
        return make_float4(a.x, a.y, b.x, b.y);
    }
    const float2 a = __bfloat1622float2(__floats2bfloat162_rn(v.x, v.y));
    const float2 b = __bfloat1622float2(__floats2bfloat162_rn(v.z, v.w));
    return make_float4(a.x, a.y, b.x, b.y);
}

// Four neighbouring outputs: out[q] = sum_t w[t] at(q + t), t = 0 .. 2 r in
// order, each texel read once (2 r + 4 reads instead of 4 (2 r + 1)).
template <typename At>
__device__ __forceinline__ void slide4(const FilterParams& f, float4 (&out)[4], At at)
{
    const int n = 2 * f.radius;   // at least 2
#pragma unroll
    for (int q = 0; q < 4; ++q) out[q] = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
    for (int t = 0; t < 3; ++t) {
        const float4 v = at(t);
#pragma unroll
        for (int q = 0; q <= t; ++q) fma4(out[q], f.w[t - q], v);
    }
    for (int t = 3; t <= n; ++t) {
        const float4 v = at(t);
#pragma unroll
        for (int q = 0; q < 4; ++q) fma4(out[q], f.w[t - q], v);
    }
#pragma unroll
    for (int t = 1; t <= 3; ++t) {
        const float4 v = at(n + t);
#pragma unroll
        for (int q = t; q < 4; ++q)
            if (n + t >= q) fma4(out[q], f.w[n + t - q], v);
    }
}

// 16-byte slot of texel u of a row: eight lanes that read every fourth texel
// hit eight different bank groups
__device__ __forceinline__ int swz(int u) { return u ^ ((u >> 3) & 3); }

// One cluster per plane, one CTA per strip of 64 columns, all of them walking
// down in steps of 16 rows. A step puts the band's original texels (with r
// columns on either side) into shared memory, filters its rows into a ring of
// row-filtered rows, rounded to the plane's type as a stored row pass would
// be, and filters the ring's columns into the output rows r above the band.
// In place: a step writes only rows whose originals every CTA of the cluster
// has read, its own and its neighbours' columns: the cluster barrier's arrive
// follows the step's loads and its wait precedes the step's stores. The next
// band's texels load into registers meanwhile.
// The passes read 2 r + 4 texels of shared memory per four outputs (2 r + 1
// per output in k_filter_rows and k_filter_cols). Bound by the latency of a
// step at three or four CTAs per SM: 64 planes of 512^2 FP32, radius 3, take
// 164 us (two passes 237; one read and one write of every texel at copy speed
// 79).
template <int DT>
__global__ void __launch_bounds__(kFusedThreads, 4) k_filter_fused(void* planes, int W, int H, FilterParams f, int pitch,
                                                                 int ring)
{
    extern __shared__ float4 fbuf[];
    float4* raw = fbuf;                        // [kBand][pitch]
    float4* rows = fbuf + kBand * pitch;       // [ring][kStrip], row y at y & (ring - 1)
    // texels of a band: thread t loads columns t % 16 + 16 q of row t / 16
    constexpr int kLoads = (kStrip + 2 * kFilterMaxRadius) / 16;
    static_assert(kFusedThreads == 16 * kBand, "sixteen threads per row of a band");
    const int tid = threadIdx.x, r = f.radius, lrow = tid / 16, lu = tid % 16;
    const int x0 = (int)blockIdx.x * kStrip, span = kStrip + 2 * r;
    const size_t plane = (size_t)blockIdx.y * (size_t)W * H;
    const float4 zero = make_float4(0.f, 0.f, 0.f, 0.f);
    for (int i = tid; i < ring * kStrip; i += kFusedThreads) rows[i] = zero;   // rows above the plane
    Stored<DT> next[kLoads];   // as stored: a conversion would wait for the load
    auto load = [&](int y) {
        const Stored<DT>* src = reinterpret_cast<const Stored<DT>*>(planes) + (plane + (size_t)y * W);
#pragma unroll
        for (int q = 0; q < kLoads; ++q) {
            const int x = x0 - r + lu + 16 * q;
            next[q] = Stored<DT>{};   // all types: 0
            if (y < H && lu + 16 * q < span && x >= 0 && x < W) next[q] = src[x];
        }
    };
    load(lrow);
    for (int y0 = 0; y0 < H + r; y0 += kBand) {
#pragma unroll
        for (int q = 0; q < kLoads; ++q)
            if (lu + 16 * q < span) raw[lrow * pitch + swz(lu + 16 * q)] = widen<DT>(next[q]);
        asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
        __syncthreads();
        if (y0 + kBand < H + r) load(y0 + kBand + lrow);
        float4 out[4];
        {
            const int row = tid / (kStrip / 4), c = tid % (kStrip / 4) * 4;
            const float4* src = raw + row * pitch;
            slide4(f, out, [&](int t) { return src[swz(c + t)]; });
            float4* dst = rows + ((y0 + row) & (ring - 1)) * kStrip;
#pragma unroll
            for (int q = 0; q < 4; ++q) dst[swz(c + q)] = as_stored<DT>(out[q]);
        }
        __syncthreads();
        {
            const int c = tid % kStrip, y = y0 - r + tid / kStrip * 4;   // first output row
            slide4(f, out, [&](int t) { return rows[((y - r + t) & (ring - 1)) * kStrip + swz(c)]; });
            asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
#pragma unroll
            for (int q = 0; q < 4; ++q)
                if (y + q >= 0 && y + q < H && x0 + c < W) st<DT>(planes, plane + (size_t)(y + q) * W + x0 + c, out[q]);
        }
    }
}

constexpr int fused_pitch(int radius) { return (kStrip + 2 * radius + 31) / 32 * 32; }

template <int DT>
void launch_fused(void* planes, int N, int W, int H, const FilterParams& f, cudaStream_t s)
{
    const int strips = (W + kStrip - 1) / kStrip;
    const int pitch = fused_pitch(f.radius), ring = kBand + 2 * f.radius <= 32 ? 32 : 64;
    const size_t smem = sizeof(float4) * (size_t)(kBand * pitch + ring * kStrip);
    auto kern = k_filter_fused<DT>;
    // (the limit of the widest filter: one set to this launch's own size would
    // refuse a wider filter that another thread launches at the same time)
    constexpr size_t smem_max = sizeof(float4) * (size_t)(kBand * fused_pitch(kFilterMaxRadius) + 64 * kStrip);
    cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem_max);
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)strips, (unsigned)N);
    cfg.blockDim = dim3(kFusedThreads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute at;
    at.id = cudaLaunchAttributeClusterDimension;
    at.val.clusterDim.x = (unsigned)strips;
    at.val.clusterDim.y = at.val.clusterDim.z = 1;
    cfg.attrs = &at;
    cfg.numAttrs = 1;
    cudaLaunchKernelEx(&cfg, kern, planes, W, H, f, pitch, ring);
    note_launches(1);
}

template <int DT>
void launch_filter_t(void* planes, int N, int W, int H, const FilterParams& f, cudaStream_t s)
{
    const int strips = (W + kStrip - 1) / kStrip;
    if (f.radius >= 1 && strips <= kStripsMax && N >= kFusedPlanes && N <= 65535 && strips * N >= kFusedCtas) {
        launch_fused<DT>(planes, N, W, H, f, s);
        return;
    }
    k_filter_rows<DT><<<(unsigned)((size_t)N * H), kRowThreads, sizeof(float4) * (kSeg + 2 * f.radius), s>>>(
        planes, W, H, f);
    const dim3 grid((unsigned)((W + kColStrip - 1) / kColStrip), (unsigned)N);
    k_filter_cols<DT><<<grid, kColStrip * kColLanes, sizeof(float4) * (kColBand + 2 * f.radius) * kColStrip, s>>>(
        planes, W, H, f);
    note_launches(2);
}

}  // namespace

void launch_filter_planes(void* planes, int dtype, int N, int W, int H, const FilterParams& f, cudaStream_t s)
{
    switch (dtype) {
    case LF_F32: launch_filter_t<LF_F32>(planes, N, W, H, f, s); break;
    case LF_F16: launch_filter_t<LF_F16>(planes, N, W, H, f, s); break;
    case LF_U8: launch_filter_t<LF_U8>(planes, N, W, H, f, s); break;
    default: launch_filter_t<LF_BF16>(planes, N, W, H, f, s); break;
    }
}

}  // namespace lf
