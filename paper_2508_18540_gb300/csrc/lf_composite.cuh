// lf_composite.cuh -- device code shared by the composite's translation
// units: the staged tile walk of the swizzle blending (Sec. 4.3). See
// lf_composite.cu for the method.
#pragma once

#include <cuda_bf16.h>
#include <cuda_fp16.h>

#include "lf_internal.cuh"

namespace lf {

namespace {

// |fma(gm, x, h)| below this bound for every x of a row keeps the exact floor
// below valid without a clamp.
constexpr float kNarrow = 1048576.0f;    // 2^20
constexpr float kClamp = 2097152.0f;     // 2^21

// Floats of one plane's entry in a view group's table: {gm, smallest h,
// largest h, plane index | wide flag << 31}, then h of the VG views (one view:
// h is the smallest).
template <int VG>
struct CoefBlock {
    static constexpr int kViews = VG == 1 ? 0 : 4 * ((VG + 3) / 4);
    static constexpr int kFloats = 4 + kViews;
};
constexpr int kWideBit = (int)0x80000000u;
constexpr int kTabPlanes = 4, kTabViews = 16;   // planes x views of one table CTA

// Four BF16 channels -> FP32, exactly: the mixed-precision add of each BF16
// operand and -0.0 (x + -0 = x, signed zeros included). It widens on the
// floating-point pipe; the shift-and-mask widening takes integer-pipe slots
// that the composite's index arithmetic needs (BF16 composite 0.425 ->
// 0.411 ms on the display frame, views bit for bit the same).
__device__ __forceinline__ float4 bf16x4_to_f32(uint2 u)
{
    float4 r;
    asm("{\n\t.reg .b16 a, b, c, d;\n\tmov.b32 {a, b}, %4;\n\tmov.b32 {c, d}, %5;\n\t"
        "add.rn.f32.bf16 %0, a, 0f80000000;\n\tadd.rn.f32.bf16 %1, b, 0f80000000;\n\t"
        "add.rn.f32.bf16 %2, c, 0f80000000;\n\tadd.rn.f32.bf16 %3, d, 0f80000000;\n\t}"
        : "=f"(r.x), "=f"(r.y), "=f"(r.z), "=f"(r.w) : "r"(u.x), "r"(u.y));
    return r;
}

template <int DT>
__device__ __forceinline__ float4 load_texel(const void* planes, size_t idx)
{
    if (DT == LF_F32) {
        return __ldg(reinterpret_cast<const float4*>(planes) + idx);
    } else if (DT == LF_U8) {
        return u8_unpack(__ldg(reinterpret_cast<const uint32_t*>(planes) + idx));
    } else {
        const uint2 u = __ldg(reinterpret_cast<const uint2*>(planes) + idx);
        if (DT == LF_F16) {
            const float2 a = __half22float2(*reinterpret_cast<const __half2*>(&u.x));
            const float2 b = __half22float2(*reinterpret_cast<const __half2*>(&u.y));
            return make_float4(a.x, a.y, b.x, b.y);
        } else {
            return bf16x4_to_f32(u);
        }
    }
}

// index of view v's pixel (x, y) in the output: separate views, or the
// quilt atlas (tile row v / c, tile column v % c)
__device__ __forceinline__ size_t view_pixel(const CompParams& p, int v, int x, int y)
{
    if (p.atlas_cols <= 0) return ((size_t)v * p.Ny + y) * p.Nx + x;
    const int c = p.atlas_cols;
    return ((size_t)(v / c) * p.Ny + y) * ((size_t)c * p.Nx) + (size_t)(v % c) * p.Nx + x;
}

// plain forms: T below this is taken as 0 at every fourth non-empty plane
constexpr float kTFlush = 5.9604644775390625e-8f;   // 2^-24
// saving forms: a walk stops once T would fall below this (taken as 0), the
// plain forms' flush threshold
constexpr float kTStop = kTFlush;

// ---------------------------------------------------------------------------
// Staged composite. All views of one view row i sample plane k on the same
// plane rows (their vertical map depends on (i, k) only), and neighbouring
// views read horizontally shifted copies of those rows. A CTA of 4 consumer
// warps and one producer warp owns a tile of TX output columns x BY output
// rows (128 x 1, 64 x 2 or 32 x 4) for a group of VG views of one view row.
// Per list entry (non-empty plane) the producer warp finds the window of
// texel columns that the tile's views sample on it (the affine map's values
// at the tile's ends for the smallest and the largest h) and the plane rows,
// 32 entries at a time, one per lane, into descriptors in shared memory; then
// it stages only that window of the BY (bilinear: 2 BY) plane rows and the
// views' h in a ring in shared memory. Rows that start on 16-byte boundaries
// come by bulk asynchronous copies of one lane (cp.async.bulk, byte count on
// the stage's "full" mbarrier); other rows (FP16 / BF16 / RGBA8 planes of odd
// widths) by 4- or 8-byte cp.async of all lanes, which arrive on the same
// barrier.
// A stage holds kPair consecutive entries, so a warp waits, releases and
// counts once per pair. Warps release a stage through an "empty" mbarrier;
// there is no CTA-wide barrier in the plane loop.
// Modes of a plane in a CTA: kInside -- every sampled texel lies in the
// plane, so a texel's shared address is one multiply-add on the floor's bits;
// kBorder -- some lie outside: the staged window is followed by a zero texel,
// and an unsigned minimum takes every index off the window there (the edge
// tiles of the outer view groups touch the plane's edges, so this is no rare
// case); kSkip -- none lies in the plane; kGlobal -- the window is wider than
// the stage or the indices need clamping, texels are read through L1.
// Small CTAs of their own rings, four (VG > 9) to seven per SM, leave an SM
// less idle than two of 8 warps: the warps of a CTA wait for its slowest one
// at the ring, and a CTA whose views have all reached T = 0 ends (the
// producer sees every warp's note, signals the end through the ring and
// stages no more) and gives its place to the next tile.
// Bilinear: the vertical tap pair depends on (i, k, y) only, so each warp
// first blends its window of the two staged rows into an FP32 row of its own,
// and each view then takes its two horizontal taps from that row.
// The floor of the FP32 index uses the exact round-toward-minus-infinity add
// of 1.5 * 2^23 (valid for |value| < 2^22) instead of a conversion unit op.
// All waits are bounded; a wait that gives up sets the error word.
// ---------------------------------------------------------------------------

constexpr float kMagic = 12582912.0f;          // 1.5 * 2^23
constexpr int kMagicBits = 0x4B400000;

__device__ __forceinline__ void bulk_copy_g2s(uint32_t dst, const void* src, uint32_t bytes, uint32_t bar)
{
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                 ::"r"(dst), "l"(src), "r"(bytes), "r"(bar)
                 : "memory");
}

__device__ __forceinline__ void fence_proxy_async() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }

// loads at 32-bit shared addresses: ordinary loads to the compiler (ordered by
// the barriers' memory clobbers, free to overlap otherwise)
template <typename T>
__device__ __forceinline__ T lds(uint32_t a)
{
    return *static_cast<const T*>(__cvta_shared_to_generic(a));
}
__device__ __forceinline__ float4 lds_f4(uint32_t a) { return lds<float4>(a); }
__device__ __forceinline__ uint2 lds_u2(uint32_t a) { return lds<uint2>(a); }
__device__ __forceinline__ float lds_f1(uint32_t a) { return lds<float>(a); }
__device__ __forceinline__ uint32_t lds_u32(uint32_t a) { return lds<uint32_t>(a); }

template <int DT>
struct Texel;
template <>
struct Texel<LF_F32> {
    static constexpr int kBytes = 16;
    static __device__ __forceinline__ float4 load(uint32_t row, uint32_t i) { return lds_f4(row + i * 16u); }
};
template <>
struct Texel<LF_F16> {
    static constexpr int kBytes = 8;
    static __device__ __forceinline__ float4 load(uint32_t row, uint32_t i)
    {
        const uint2 u = lds_u2(row + i * 8u);
        const float2 a = __half22float2(*reinterpret_cast<const __half2*>(&u.x));
        const float2 b = __half22float2(*reinterpret_cast<const __half2*>(&u.y));
        return make_float4(a.x, a.y, b.x, b.y);
    }
};
template <>
struct Texel<LF_U8> {
    static constexpr int kBytes = 4;
    static __device__ __forceinline__ float4 load(uint32_t row, uint32_t i) { return u8_unpack(lds_u32(row + i * 4u)); }
};
template <>
struct Texel<LF_BF16> {
    static constexpr int kBytes = 8;
    static __device__ __forceinline__ float4 load(uint32_t row, uint32_t i)
    {
        const uint2 u = lds_u2(row + i * 8u);
        return bf16x4_to_f32(u);
    }
};


// floor(fma(g, x, h)) as the bit pattern of (value + 1.5 * 2^23) rounded
// toward minus infinity; callers add base - kMagicBits to get an index.
template <bool CLAMP>
__device__ __forceinline__ float floor_magic(float g, float x, float h)
{
    float f = __fmaf_rn(g, x, h);
    if (CLAMP) f = fminf(fmaxf(f, -kClamp), kClamp);
    return __fadd_rd(f, kMagic);
}

// plane texel (row or column) sampled by output pixel x along one axis
// (nearest), or its lower bilinear tap
__device__ __forceinline__ int plane_index(int P_s, int x, float gm, float h)
{
    return P_s * x + (__float_as_int(floor_magic<true>(gm, (float)x, h)) - kMagicBits);
}

constexpr int kWarps = kCompThreads / 32;        // consumer warps
constexpr int kCompBlock = kCompThreads + 32;    // + one producer warp
constexpr int kPair = 2;                         // list steps per stage
constexpr int kDescs = 64;                       // descriptors in shared memory (two producer batches)
enum { kInside = 0, kBorder = 1, kSkip = 2, kGlobal = 3 };   // modes

// Descriptor of one list step, kDescBytes (short form) or 64 bytes:
//  {gm, first staged texel column, plane << 8 | modes, smallest h},
//  {gm_y, h_y, smallest h, largest h},
//  long form (bilinear, adjoint): per warp the first texel column of its own
//  window, clipped to the plane, and the window's texel count.
// modes: bits 2 r, 2 r + 1 the mode of output row r (kSkip also where its
// plane rows lie outside the plane).
// Copy record of a step (the producer's): {byte offset of the first texel of
// plane row 0 of output row 0 (64 bits), window bytes (0: nothing staged),
// rows}; rows: bit r * RPY + t set where plane row t of output row r lies in
// the plane.
constexpr uint32_t kDescBytes = 32;

__device__ __forceinline__ void sts_f4(uint32_t a, float4 v)
{
    asm volatile("st.shared.v4.f32 [%0], {%1, %2, %3, %4};" ::"r"(a), "f"(v.x), "f"(v.y), "f"(v.z), "f"(v.w) : "memory");
}

__device__ __forceinline__ void sts_f1(uint32_t a, float v)
{
    asm volatile("st.shared.f32 [%0], %1;" ::"r"(a), "f"(v) : "memory");
}

template <int BYTES>
__device__ __forceinline__ void cp_async(uint32_t dst, const void* src)
{
    asm volatile("cp.async.ca.shared.global [%0], [%1], %2;" ::"r"(dst), "l"(src), "n"(BYTES) : "memory");
}

// the thread's arrival on bar once its earlier cp.async have landed
__device__ __forceinline__ void cp_async_arrive(uint32_t bar)
{
    asm volatile("cp.async.mbarrier.arrive.noinc.shared.b64 [%0];" ::"r"(bar) : "memory");
}

inline size_t round16(size_t v) { return (v + 15) / 16 * 16; }

// Position in the stage ring, counted by the producer and by every consumer.
struct Ring {
    int st = 0;
    uint32_t ph = 0;      // phase parity of the entry about to be filled or read
    bool wrapped = false; // from the second round on the producer waits for releases
    __device__ __forceinline__ void next(int stages)
    {
        if (++st == stages) st = 0, ph ^= 1u, wrapped = true;
    }
};

// Shared-memory addresses of one CTA.
struct TileSmem {
    uint32_t stages, full, empty, warp_rows, desc, copies;
    int* sat;   // consumer warps whose views have all stopped
    int* end;   // first list step that is not staged
    __device__ __forceinline__ TileSmem(const CompGeom& G, unsigned char* smem)
    {
        stages = smem_addr(smem);
        warp_rows = stages + G.rows_off;
        full = stages + G.bar_off;
        empty = full + 8 * kStages;
        sat = reinterpret_cast<int*>(smem + G.bar_off + 16 * kStages);
        end = sat + 1;
        copies = empty + 8 * kStages + 16;
        desc = copies + 16 * kDescs;
    }
    // one thread, before the CTA's first barrier
    __device__ __forceinline__ void init(const CompGeom& G) const
    {
        for (int s = 0; s < G.stages; ++s) {
            mbar_init(full + 8 * s, G.bulk ? 1 : 33);
            mbar_init(empty + 8 * s, kWarps);
        }
        *sat = 0;
        *end = 0x7fffffff;
        fence_proxy_async();
    }
};

// The producer warp: stages steps 0 .. n - 1, step i being list entry
// (REV ? n - 1 - i : i) of the tables blk, yt. EARLY: once every consumer warp
// has noted that it needs no more, *sm.end is set to the step reached and that
// step's "full" barrier completed without data. LONG: long descriptors.
// n_tab: entries that the tables have room for (n itself if REV), so that the
// first ones load while n does. Returns false if a wait gave up.
template <int DT, bool BILINEAR, int VG, bool REV, bool EARLY, bool LONG>
__device__ __forceinline__ bool produce(const CompParams& p, const CompGeom& G, const char* __restrict__ planes,
                                        const float* __restrict__ blk, const float2* __restrict__ yt, int n, int X0,
                                        int Y0, const TileSmem& sm, Ring& ring, int n_tab)
{
    constexpr int CW = CoefBlock<VG>::kFloats, KV = CoefBlock<VG>::kViews;
    constexpr int TB = Texel<DT>::kBytes;
    constexpr int RPY = BILINEAR ? 2 : 1;
    constexpr int AL = 16 / TB;               // texels per 16 bytes
    constexpr uint32_t DB = LONG ? 64u : kDescBytes;
    const int lane = threadIdx.x & 31;
    const int X1 = min(X0 + G.TX, p.Nx) - 1;
    auto entry = [&](int i) { return REV ? n - 1 - i : i; };
    float4 nh = make_float4(0.f, 0.f, 0.f, 0.f);
    float2 ny = make_float2(0.f, 0.f);
    auto fetch = [&](int i) {
        if (i >= n_tab) return;
        nh = __ldg(reinterpret_cast<const float4*>(blk + (size_t)entry(i) * CW));
        ny = __ldg(yt + entry(i));
    };
    // waits for the stage's release; 1: every warp has stopped, 2: gave up
    auto acquire = [&](int i) -> int {
        if (!ring.wrapped) return 0;
        if (!mbar_wait_bounded(sm.empty + 8 * ring.st, ring.ph ^ 1u)) return 2;
        return EARLY && *reinterpret_cast<volatile int*>(sm.sat) == kWarps ? 1 : 0;
    };
    fetch(lane);
    for (int i0 = 0; i0 < n; i0 += 32) {
        const float4 hd = nh;
        const float2 hy = ny;
        const int il = i0 + lane;
        fetch(il + 32);
        if (il < n) {
            const float gm = hd.x, h0 = hd.y, h1 = hd.z;
            const int kw = __float_as_int(hd.w), k = kw & ~kWideBit;
            // texel columns the tile samples: the affine map's ends (a NaN h clamps to the far left, outside)
            const int lo = min(plane_index(p.P_s, X0, gm, h0), plane_index(p.P_s, X1, gm, h0));
            const int hi = max(plane_index(p.P_s, X0, gm, h1), plane_index(p.P_s, X1, gm, h1)) + (RPY - 1);
            const int first = max(lo, 0) / AL * AL;
            const int last = min(min(hi, p.W - 1) / AL * AL + AL, p.W);   // one past
            int mode = lo >= 0 && hi < p.W ? kInside : kBorder;
            if (hi < 0 || lo >= p.W)
                mode = kSkip;
            else if (last - first > G.cap || kw < 0)
                mode = kGlobal;
            int rows = 0, modes = 0;
            const int iy0 = plane_index(p.P_s, Y0, hy.x, hy.y);
            for (int r = 0; r < G.BY; ++r) {
                const int y = Y0 + r, iy = r == 0 ? iy0 : plane_index(p.P_s, y, hy.x, hy.y);
                int m = 0;
#pragma unroll
                for (int t = 0; t < RPY; ++t)
                    if (y < p.Ny && iy + t >= 0 && iy + t < p.H) m |= 1 << t;
                rows |= m << (r * RPY);
                modes |= (m ? mode : (int)kSkip) << (2 * r);
            }
            const uint32_t slot = (uint32_t)(il & (kDescs - 1)), d = sm.desc + slot * DB;
            sts_f4(d, make_float4(gm, __int_as_float(first), __int_as_float(k << 8 | modes), h0));
            sts_f4(d + 16, make_float4(hy.x, hy.y, h0, h1));
            const long long off = (((long long)k * p.H + iy0) * p.W + first) * TB;
            sts_f4(sm.copies + 16 * slot, make_float4(__int_as_float((int)off), __int_as_float((int)(off >> 32)),
                                                      __int_as_float(mode <= kBorder ? (last - first) * TB : 0),
                                                      __int_as_float(rows)));
            if (LONG) {
#pragma unroll
                for (int w = 0; w < kWarps; ++w) {
                    const int xa = X0 + 32 * w % G.TX, xb = min(xa + 31, p.Nx - 1);
                    const int wl = max(0, min(plane_index(p.P_s, xa, gm, h0), plane_index(p.P_s, xb, gm, h0)));
                    const int wh = min(p.W - 1, max(plane_index(p.P_s, xa, gm, h1), plane_index(p.P_s, xb, gm, h1)) +
                                                    (RPY - 1));
                    sts_f1(d + 32 + 4 * w, __int_as_float(wl));
                    sts_f1(d + 48 + 4 * w, __int_as_float(xa < p.Nx ? wh - wl + 1 : 0));
                }
            }
        }
        __syncwarp();
        const int cnt = min(32, n - i0);
        int stop = 0;
        const int R = G.BY * RPY, u = lane >> 4, j = lane & 15;
        if (G.bulk) {
            // lane 16 u + j copies row j of the stage's step u, j = R the
            // step's h: issued by one lane, the copies of four-row tiles took
            // half a microsecond a step, more than a small grid's blending
            for (int e = 0; e < cnt; e += kPair) {
                const int i = i0 + e;
                const uint32_t full = sm.full + 8 * ring.st;
                if (lane == 0) stop = acquire(i);
                __syncwarp();
                stop = __shfl_sync(0xffffffffu, stop, 0);
                if (stop) {
                    if (stop == 1 && lane == 0) {
                        *reinterpret_cast<volatile int*>(sm.end) = i;
                        mbar_arrive(full);
                    }
                    if (stop == 1) ring.next(G.stages);
                    break;
                }
                const bool has = e + u < cnt;
                const uint32_t slot = (uint32_t)((i + u) & (kDescs - 1));
                const uint32_t sa = sm.stages + (uint32_t)ring.st * G.stage_bytes + (u ? G.plane_bytes : 0u);
                const uint32_t dst = sa + G.hdr_bytes + (uint32_t)j * G.win_bytes;
                const float4 c = has ? lds_f4(sm.copies + 16 * slot) : make_float4(0.f, 0.f, 0.f, 0.f);
                const uint32_t bytes = __float_as_uint(c.z), rows = __float_as_uint(c.w);
                // the zero texel behind the row's window (read in mode kBorder)
                if (!BILINEAR && has && j < R) sts_f4(dst + bytes, make_float4(0.f, 0.f, 0.f, 0.f));
                fence_proxy_async();
                const uint32_t tx = has ? 4u * KV + (uint32_t)__popc(rows) * bytes : 0u;
                const uint32_t both = tx + __shfl_xor_sync(0xffffffffu, tx, 16);
                __syncwarp();   // lane 0's arrival orders the zero texels too
                if (lane == 0) mbar_arrive_expect_tx(full, both);
                __syncwarp();
                if (has && j == R && VG > 1) bulk_copy_g2s(sa, blk + (size_t)entry(i + u) * CW + 4, 4u * KV, full);
                if (bytes && j < R && ((rows >> j) & 1u)) {
                    const char* src = planes + ((unsigned long long)__float_as_uint(c.y) << 32 | __float_as_uint(c.x));
                    int down = j % RPY;
                    if (j >= RPY) {
                        const float4 B = lds_f4(sm.desc + slot * DB + 16);
                        down += plane_index(p.P_s, Y0 + j / RPY, B.x, B.y) - plane_index(p.P_s, Y0, B.x, B.y);
                    }
                    bulk_copy_g2s(dst, src + (ptrdiff_t)down * (ptrdiff_t)((size_t)p.W * TB), bytes, full);
                }
                ring.next(G.stages);
            }
        } else {
            for (int e = 0; e < cnt; e += kPair) {
                const int i = i0 + e;
                const uint32_t full = sm.full + 8 * ring.st;
                stop = __reduce_max_sync(0xffffffffu, acquire(i));
                if (stop) {
                    if (stop == 1) {
                        if (lane == 0) *reinterpret_cast<volatile int*>(sm.end) = i;
                        __syncwarp();
                        mbar_arrive(full);
                        if (lane == 0) mbar_arrive(full);
                        ring.next(G.stages);
                    }
                    break;
                }
                // lane 16 u + j finds row j of step u, then all lanes copy row by row
                const bool has = e + u < cnt;
                const uint32_t slot = (uint32_t)((i + u) & (kDescs - 1));
                const uint32_t sa = sm.stages + (uint32_t)ring.st * G.stage_bytes + (u ? G.plane_bytes : 0u);
                const uint32_t dst = sa + G.hdr_bytes + (uint32_t)j * G.win_bytes;
                const float4 c4 = has ? lds_f4(sm.copies + 16 * slot) : make_float4(0.f, 0.f, 0.f, 0.f);
                if (VG > 1 && has && j < KV / 4)
                    cp_async<16>(sa + 16u * (uint32_t)j, blk + (size_t)entry(i + u) * CW + 4 + 4 * j);
                const int texels = (int)(__float_as_uint(c4.z) / TB);
                const bool on = texels && j < R && ((__float_as_uint(c4.w) >> j) & 1u);
                unsigned long long src = 0;
                if (on) {
                    int down = j % RPY;
                    if (j >= RPY) {
                        const float4 B = lds_f4(sm.desc + slot * DB + 16);
                        down += plane_index(p.P_s, Y0 + j / RPY, B.x, B.y) - plane_index(p.P_s, Y0, B.x, B.y);
                    }
                    src = (unsigned long long)planes +
                          ((unsigned long long)__float_as_uint(c4.y) << 32 | __float_as_uint(c4.x)) +
                          (unsigned long long)((long long)down * (long long)((size_t)p.W * TB));
                    // the zero texel behind the window
                    if (!BILINEAR) {
#pragma unroll
                        for (int t = 0; t < TB / 4; ++t) sts_f1(dst + (uint32_t)texels * TB + 4u * t, 0.f);
                    }
                }
                for (uint32_t m = __ballot_sync(0xffffffffu, on); m; m &= m - 1) {
                    const int l = __ffs(m) - 1;
                    const char* from = reinterpret_cast<const char*>(__shfl_sync(0xffffffffu, src, l));
                    const uint32_t to = __shfl_sync(0xffffffffu, dst, l);
                    const int n_tex = __shfl_sync(0xffffffffu, texels, l);
                    for (int c = lane; c < n_tex; c += 32) cp_async<TB>(to + (uint32_t)c * TB, from + (size_t)c * TB);
                }
                cp_async_arrive(full);
                __syncwarp();   // lane 0's arrival orders the zero texels too
                if (lane == 0) mbar_arrive(full);
                ring.next(G.stages);
            }
        }
        if (stop) return stop == 1;
        __syncwarp();
    }
    return true;
}

// Per-thread constants of one tile. Threads past the view's right edge take
// its last column (their addresses stay in the staged window).
struct ThreadGeom {
    float xf, yf;          // output pixel
    int pxm;               // P_s x - magic bits: + floor bits = texel index
    int psy;               // P_s y
    uint32_t row;          // offset of the thread's (first) staged row in a stage
    int mode_sh;           // its output row's bits in a descriptor's modes
};

__device__ __forceinline__ ThreadGeom thread_geom(const CompParams& p, const CompGeom& G, int x, int y, int ty)
{
    ThreadGeom t;
    x = min(x, p.Nx - 1);
    t.xf = (float)x;
    t.yf = (float)y;
    t.pxm = p.P_s * x - kMagicBits;
    t.psy = p.P_s * y;
    t.row = G.hdr_bytes + (uint32_t)(ty * (p.bilinear ? 2 : 1)) * G.win_bytes;
    t.mode_sh = 2 * ty;
    return t;
}

// h of views 4 e .. 4 e + 3 of a staged plane, loaded as the unrolled view
// loop reaches them
struct ViewH {
    float4 v;
    template <int VG>
    __device__ __forceinline__ float get(uint32_t sa, float h0, int jj)
    {
        if (VG == 1) return h0;
        if (jj % 4 == 0) v = lds_f4(sa + 4u * (uint32_t)jj);
        return jj % 4 == 0 ? v.x : jj % 4 == 1 ? v.y : jj % 4 == 2 ? v.z : v.w;
    }
};

// Bilinear rows of output row y: upper plane row and the weights of it and
// the row below (0 outside the plane).
struct RowPair {
    int y0;
    float w0, w1;
    __device__ __forceinline__ RowPair(const CompParams& p, const ThreadGeom& tg, float gmy, float hy)
    {
        float fy = __fmaf_rn(gmy, tg.yf, hy);
        fy = fminf(fmaxf(fy, -kClamp), kClamp);
        const float m = __fadd_rd(fy, kMagic);
        const float wy = fy - (m - kMagic);
        y0 = tg.psy + (__float_as_int(m) - kMagicBits);
        w0 = (y0 >= 0 && y0 < p.H) ? 1.0f - wy : 0.0f;
        w1 = (y0 + 1 >= 0 && y0 + 1 < p.H) ? wy : 0.0f;
    }
};

__device__ __forceinline__ float4 mix_rows(float4 a, float4 b, const RowPair& rp)
{
    // a row outside the plane was not read (zeros) and has weight 0
    return make_float4(fmaf(rp.w1, b.x, rp.w0 * a.x), fmaf(rp.w1, b.y, rp.w0 * a.y), fmaf(rp.w1, b.z, rp.w0 * a.z),
                       fmaf(rp.w1, b.w, rp.w0 * a.w));
}

// Blends texels lo .. lo + n - 1 of the warp's two plane rows into its FP32
// row at shared address dst (all lanes; the caller orders the accesses).
template <int DT>
__device__ __forceinline__ void blend_rows(const CompParams& p, const void* __restrict__ planes, uint32_t sa,
                                           const ThreadGeom& tg, const CompGeom& G, const RowPair& rp, int mode, int k,
                                           int first, int lo, int n, uint32_t dst)
{
    const float4 z = make_float4(0.f, 0.f, 0.f, 0.f);
    const uint32_t r0 = sa + tg.row, r1 = r0 + G.win_bytes;
    for (int c = threadIdx.x & 31; c < n; c += 32) {
        float4 a = z, b = z;
        if (mode != kGlobal) {
            if (rp.w0 != 0.0f) a = Texel<DT>::load(r0, (uint32_t)(lo + c - first));
            if (rp.w1 != 0.0f) b = Texel<DT>::load(r1, (uint32_t)(lo + c - first));
        } else {
            const size_t at = ((size_t)k * p.H + rp.y0) * p.W + lo + c;   // read only where the row exists
            if (rp.w0 != 0.0f) a = load_texel<DT>(planes, at);
            if (rp.w1 != 0.0f) b = load_texel<DT>(planes, at + p.W);
        }
        sts_f4(dst + 16u * (uint32_t)c, mix_rows(a, b, rp));
    }
    if ((threadIdx.x & 31) == 0) sts_f4(dst + 16u * (uint32_t)n, z);   // read for columns off the plane
}

// One bilinear sample from the two staged rows (slots of columns i0, i0 + 1 in
// window slots s0, s1; an off slot reads as zero), same rounding order.
template <int DT>
__device__ __forceinline__ void sample_staged(uint32_t r0, uint32_t r1, const RowPair& rp, uint32_t s0, uint32_t s1,
                                              bool in0, bool in1, float4& u0, float4& u1)
{
    const float4 z = make_float4(0.f, 0.f, 0.f, 0.f);
    const bool v0 = rp.w0 != 0.0f, v1 = rp.w1 != 0.0f;
    const float4 a0 = in0 && v0 ? Texel<DT>::load(r0, s0) : z, a1 = in1 && v0 ? Texel<DT>::load(r0, s1) : z;
    const float4 b0 = in0 && v1 ? Texel<DT>::load(r1, s0) : z, b1 = in1 && v1 ? Texel<DT>::load(r1, s1) : z;
    u0 = mix_rows(a0, b0, rp);
    u1 = mix_rows(a1, b1, rp);
}

// One bilinear sample at columns i0, i0 + 1 read straight from the plane,
// in the same rounding order (vertical pairs, then the horizontal pair).
template <int DT>
__device__ __forceinline__ float4 sample_global(const CompParams& p, const void* __restrict__ planes, int k,
                                                const RowPair& rp, int i0, float4* u1)
{
    const float4 z = make_float4(0.f, 0.f, 0.f, 0.f);
    float4 u[2];
#pragma unroll
    for (int t = 0; t < 2; ++t) {
        const bool in = (uint32_t)(i0 + t) < (uint32_t)p.W;
        const size_t at = ((size_t)k * p.H + rp.y0) * p.W + i0 + t;
        const float4 a = in && rp.w0 != 0.0f ? load_texel<DT>(planes, at) : z;
        const float4 b = in && rp.w1 != 0.0f ? load_texel<DT>(planes, at + p.W) : z;
        u[t] = mix_rows(a, b, rp);
    }
    *u1 = u[1];
    return u[0];
}

// Saving form, view J (a: its carried T, negated once it has stopped): nt, the
// transmittance behind plane q, or -|a| where it is below kTStop; there, if
// a > 0 (the view's stop plane), q goes to the view's stop slot. Branch-free:
// a predicated store at [stop + immediate]. (One store, T kept in a
// register: each costs a shared-memory slot whether or not a lane stops.)
template <int J>
__device__ __forceinline__ float stop_below(uint32_t stop, float a, float nt, int q)
{
    float r;
    asm volatile(
        "{\n\t.reg .pred l, s;\n\t.reg .f32 n;\n\tsetp.lt.f32 l, %3, 0f33800000;\n\t"
        "setp.gt.and.f32 s, %2, 0f00000000, l;\n\t@s st.shared.u32 [%1+%5], %4;\n\t"
        "abs.f32 n, %2;\n\tneg.f32 n, n;\n\tselp.f32 %0, n, %3, l;\n\t}"
        : "=f"(r)
        : "r"(stop), "f"(a), "f"(nt), "r"(q), "n"(4 * J));
    return r;
}
static_assert(kTStop == 5.9604644775390625e-8f, "0f33800000 above is 2^-24");

// One view's blend of one texel t of plane q (view jj of the thread's group).
// Plain form: Q += T c, T <- T - T A. Saving form: the view's walk stops at
// the first plane q behind which T would fall below kTStop (0 behind a plane
// with A = 1): plane q still blends with its T_q, q goes to the view's stop
// slot in shared memory (stop + 4 jj, the thread's VG slots), and a[3] = -T_q
// marks the view as stopped (T = 0 from there on, the colour the plain form
// would still add being below 2^-24 per plane). The kernel stores the state
// at the end of its walk.
template <bool SAVE>
__device__ __forceinline__ void blend_texel(float (&a)[4], float4 t, uint32_t stop, int jj, int q)
{
    const float T = SAVE ? fmaxf(a[3], 0.0f) : a[3];
    a[0] = fmaf(T, t.x, a[0]);
    a[1] = fmaf(T, t.y, a[1]);
    a[2] = fmaf(T, t.z, a[2]);
    const float nt = fmaf(-T, t.w, T);
    if (!SAVE) {
        a[3] = nt;
        return;
    }
    switch (jj) {   // jj is a constant in every (unrolled) caller
    case 0: a[3] = stop_below<0>(stop, a[3], nt, q); break;
    case 1: a[3] = stop_below<1>(stop, a[3], nt, q); break;
    case 2: a[3] = stop_below<2>(stop, a[3], nt, q); break;
    case 3: a[3] = stop_below<3>(stop, a[3], nt, q); break;
    case 4: a[3] = stop_below<4>(stop, a[3], nt, q); break;
    case 5: a[3] = stop_below<5>(stop, a[3], nt, q); break;
    case 6: a[3] = stop_below<6>(stop, a[3], nt, q); break;
    case 7: a[3] = stop_below<7>(stop, a[3], nt, q); break;
    case 8: a[3] = stop_below<8>(stop, a[3], nt, q); break;
    case 9: a[3] = stop_below<9>(stop, a[3], nt, q); break;
    case 10: a[3] = stop_below<10>(stop, a[3], nt, q); break;
    case 11: a[3] = stop_below<11>(stop, a[3], nt, q); break;
    case 12: a[3] = stop_below<12>(stop, a[3], nt, q); break;
    case 13: a[3] = stop_below<13>(stop, a[3], nt, q); break;
    default: a[3] = stop_below<14>(stop, a[3], nt, q); break;
    }
}

// Plain form, before every fourth non-empty plane of the list: a view whose
// transmittance has fallen below kTFlush = 2^-24 (the FP32 spacing at 1)
// takes T = 0, so the planes behind it add nothing; what they would still
// add is below 2^-24 of a colour's range per channel, and the output's
// 1 - T moves by less than 2^-24. The decision depends on the view pixel's
// own walk and the list position only, so every layout of the work
// (views per thread, tiles, batch plans) gives the same bits.
// Returns whether every view of this thread has T == 0 exactly (saving form:
// has stopped). T never leaves 0 (T <- T - T A), and behind it a plane adds
// T c = 0 to Q, so skipping such planes changes no bit of the output.
template <int VG, bool SAVE>
__device__ __forceinline__ bool flush_tiny(float (&acc)[VG][4])
{
    if (SAVE) {
        int most = __float_as_int(acc[0][3]);   // negative: stopped (a NaN keeps its warp walking)
#pragma unroll
        for (int jj = 1; jj < VG; ++jj) most = max(most, __float_as_int(acc[jj][3]));
        return most < 0;
    }
    uint32_t most = 0u;   // largest bit pattern: 0 only if every T is +0 (a NaN keeps its warp walking)
#pragma unroll
    for (int jj = 0; jj < VG; ++jj) {
        acc[jj][3] = acc[jj][3] < kTFlush ? 0.0f : acc[jj][3];
        most = max(most, __float_as_uint(acc[jj][3]));
    }
    return most == 0u;
}

// a += T x of two views
__device__ __forceinline__ void blend2(float& a0, float& a1, f32x2 T, f32x2 x)
{
    const float2 r = unpack2(fma2(T, x, pack2(a0, a1)));
    a0 = r.x, a1 = r.y;
}

// bytes K of two RGBA8 texels
template <int K>
__device__ __forceinline__ f32x2 u8_bytes(uint32_t u0, uint32_t u1)
{
    constexpr uint32_t sel = 0x7440u | (uint32_t)K;
    return add2(pack2(__uint_as_float(__byte_perm(u0, 0x4B000000u, sel)), __uint_as_float(__byte_perm(u1, 0x4B000000u, sel))),
                pack2(-8388608.0f, -8388608.0f));
}

// One plane of a nearest tile: every view of the thread's pixel. A, d: the
// plane's descriptor and its shared address; sa: its stage; Y0: the tile's
// first output row.
template <int DT, int VG, bool SAVE, int MODE>
__device__ __forceinline__ void blend_nearest(const CompParams& p, const CompGeom& G, const void* __restrict__ planes,
                                              float (&acc)[VG][4], float4 A, uint32_t d, uint32_t sa,
                                              const ThreadGeom& tg, const TileSmem& sm, uint32_t stop, int Y0)
{
    using TX_ = Texel<DT>;
    constexpr uint32_t TB = TX_::kBytes;
    const int k = __float_as_int(A.z) >> 8;
    // window slot of the texel whose floor bits are b: c + b
    const uint32_t c = (uint32_t)(tg.pxm - __float_as_int(A.y)), row = sa + tg.row;
    const uint32_t base = row + c * TB;
    uint32_t last = 0;
    const char* grow = nullptr;
    if (MODE == kBorder) last = lds_u32(sm.copies + (d - sm.desc) / kDescBytes * 16u + 8u) / TB;
    if (MODE == kGlobal) {
        const float4 B = lds_f4(d + 16);
        const int iy = plane_index(p.P_s, Y0 + (int)threadIdx.x / G.TX, B.x, B.y);
        grow = static_cast<const char*>(planes) + ((size_t)k * p.H + iy) * p.W * TB;
    }
    ViewH vh;
    // RGBA8, two views at a time in packed FP32 pairs (the same roundings): a
    // sample was 14 instructions of unpacking and blending around its load, a
    // pair of samples is 18 (2.02 -> 1.90 ms for 90 views of 512^2 from 256
    // planes of 1024^2). The other types gain nothing: FP32 texels arrive as
    // {r, g, b, a} and are bound by shared-memory wavefronts (0.37 -> 0.39 ms
    // with packed positions), 16-bit ones spill at 9 views per thread.
    constexpr int kTwo = DT != LF_U8 || SAVE || MODE == kGlobal ? 0 : VG / 2 * 2;
    const f32x2 gm2 = pack2(A.x, A.x), x2 = pack2(tg.xf, tg.xf), magic2 = pack2(kMagic, kMagic);
#pragma unroll
    for (int jj = 0; jj < kTwo; jj += 2) {
        constexpr float s = 1.0f / 255.0f;
        const float ha = vh.template get<VG>(sa, A.w, jj), hb = vh.template get<VG>(sa, A.w, jj + 1);
        const float2 m = unpack2(add2_down(fma2(gm2, x2, pack2(ha, hb)), magic2));   // floor_magic of both
        const uint32_t b0 = __float_as_uint(m.x), b1 = __float_as_uint(m.y);
        const uint32_t u0 = lds_u32(MODE == kBorder ? row + min(b0 + c, last) * TB : base + b0 * TB);
        const uint32_t u1 = lds_u32(MODE == kBorder ? row + min(b1 + c, last) * TB : base + b1 * TB);
        // colour bytes scale by 1/255 through T, as below; alpha keeps byte / 255
        const f32x2 T = pack2(acc[jj][3], acc[jj + 1][3]), Ts = mul2(T, pack2(s, s));
        blend2(acc[jj][0], acc[jj + 1][0], Ts, u8_bytes<0>(u0, u1));
        blend2(acc[jj][1], acc[jj + 1][1], Ts, u8_bytes<1>(u0, u1));
        blend2(acc[jj][2], acc[jj + 1][2], Ts, u8_bytes<2>(u0, u1));
        blend2(acc[jj][3], acc[jj + 1][3], T, mul2(u8_bytes<3>(u0, u1), pack2(-s, -s)));
    }
#pragma unroll
    for (int jj = kTwo; jj < VG; ++jj) {
        const float h = vh.template get<VG>(sa, A.w, jj);
        const uint32_t b = __float_as_uint(floor_magic<MODE == kGlobal>(A.x, tg.xf, h));
        const uint32_t a = MODE == kBorder ? row + min(b + c, last) * TB : base + b * TB;
        if (MODE == kGlobal) {
            float4 t = make_float4(0.f, 0.f, 0.f, 0.f);
            if (b + (uint32_t)tg.pxm < (uint32_t)p.W) t = load_texel<DT>(grow, b + (uint32_t)tg.pxm);
            blend_texel<SAVE>(acc[jj], t, stop, jj, k);
        } else if constexpr (DT == LF_U8 && !SAVE) {
            // colour bytes scale by 1/255 through T (one multiply per
            // texel instead of three); alpha keeps A = byte / 255
            constexpr float s = 1.0f / 255.0f;
            const uint32_t u = lds_u32(a);
            const float T = acc[jj][3], Ts = T * s;
            acc[jj][0] = fmaf(Ts, u8_byte<0>(u), acc[jj][0]);
            acc[jj][1] = fmaf(Ts, u8_byte<1>(u), acc[jj][1]);
            acc[jj][2] = fmaf(Ts, u8_byte<2>(u), acc[jj][2]);
            acc[jj][3] = fmaf(-T, u8_byte<3>(u) * s, T);
        } else {
            blend_texel<SAVE>(acc[jj], TX_::load(a, 0u), stop, jj, k);
        }
    }
}

// Bilinear sample position along x: floor bits, weight of the right tap.
__device__ __forceinline__ uint32_t tap_bits(float gm, float x, float h, bool clamp, float& wx)
{
    float f = __fmaf_rn(gm, x, h);
    if (clamp) f = fminf(fmaxf(f, -kClamp), kClamp);
    const float m = __fadd_rd(f, kMagic);
    wx = f - (m - kMagic);
    return __float_as_uint(m);
}

__device__ __forceinline__ float4 mix_taps(float wx, float4 a, float4 b)
{
    const float wa = 1.0f - wx;
    return make_float4(fmaf(wa, a.x, wx * b.x), fmaf(wa, a.y, wx * b.y), fmaf(wa, a.z, wx * b.z), fmaf(wa, a.w, wx * b.w));
}

// Horizontal taps of every view from the warp's blended row (shared address
// row, n texels from lo on, then a zero texel that takes every index off them
// unless INSIDE). clamp: positions past kNarrow occur.
template <int VG, bool SAVE, bool INSIDE>
__device__ __forceinline__ void blend_taps(float (&acc)[VG][4], float4 A, uint32_t sa, uint32_t row, int lo, int n,
                                           const ThreadGeom& tg, uint32_t stop, bool clamp)
{
    const int k = __float_as_int(A.z) >> 8;
    const uint32_t c = (uint32_t)(tg.pxm - lo), base = row + c * 16u;
    ViewH vh;
#pragma unroll
    for (int jj = 0; jj < VG; ++jj) {
        float wx;
        const uint32_t b = tap_bits(A.x, tg.xf, vh.template get<VG>(sa, A.w, jj), !INSIDE && clamp, wx);
        uint32_t a0 = base + b * 16u, a1 = a0 + 16u;
        if (!INSIDE) {
            a0 = row + min(b + c, (uint32_t)n) * 16u;
            a1 = row + min(b + c + 1u, (uint32_t)n) * 16u;
        }
        blend_texel<SAVE>(acc[jj], mix_taps(wx, lds_f4(a0), lds_f4(a1)), stop, jj, k);
    }
}

// One tile of one view group over the list entries [q0, q0 + P): output
// columns X0 .., rows Y0 .., view group vgroup (view row vgroup / groups_x).
// part == nullptr: final views in out (SAVE: and the adjoint's state, {T_k,
// k}: k the plane behind which T falls below 2^-24 (and is taken as 0), T_k
// the transmittance in front of it; or k = N and the transmittance behind the
// last plane, see blend_texel); else the partial (Q, T) in part, separate
// views order.
template <int DT, bool BILINEAR, int VG, bool SAVE>
__device__ __forceinline__ void composite_tile(const CompParams& p, const CompGeom& G, const char* __restrict__ planes,
                                               const CompWs& w, float* __restrict__ out, float4* __restrict__ state,
                                               float4* __restrict__ part, bool partial, int vgroup, int X0, int Y0,
                                               int q0, int P)
{
    extern __shared__ __align__(128) unsigned char smem[];
    const TileSmem sm(G, smem);
    const int tid = threadIdx.x, lane = tid & 31;
    const int vi = vgroup / G.groups_x;            // view row
    const int j0 = (vgroup % G.groups_x) * VG;     // first view column of the group
    if (tid == 0) sm.init(G);
    __syncthreads();
    Ring ring;
    if (tid >= kCompThreads) {
        const float* blk = w.blk + ((size_t)(vgroup % G.groups_x) * p.N + q0) * CoefBlock<VG>::kFloats;
        if (!produce<DT, BILINEAR, VG, false, true, BILINEAR>(p, G, planes, blk, w.yt + (size_t)vi * p.N + q0, P, X0, Y0, sm,
                                                    ring, p.N - q0))
            atomicExch(w.err, 1);
        return;
    }
    const int tx = tid % G.TX, ty = tid / G.TX;
    const int x = X0 + tx, y = Y0 + ty;
    const bool live = x < p.Nx && y < p.Ny;
    const ThreadGeom tg = thread_geom(p, G, x, y, ty);
    float acc[VG][4];
#pragma unroll
    for (int jj = 0; jj < VG; ++jj) acc[jj][0] = acc[jj][1] = acc[jj][2] = 0.f, acc[jj][3] = 1.f;
    // saving form: the thread's stop slots
    const uint32_t stop = sm.stages + G.stop_off + 4u * (uint32_t)(tid * VG);
    const uint32_t wrow = sm.warp_rows + (uint32_t)(tid >> 5) * G.wcap * 16u;   // bilinear: the warp's blended row
    bool warp_sat = false;   // every view of every lane of this warp has T == 0
    constexpr uint32_t DB = BILINEAR ? 64u : kDescBytes;
    for (int q = 0; q < P; q += kPair, ring.next(G.stages)) {
        if (!mbar_wait_bounded(sm.full + 8 * ring.st, ring.ph)) {
            atomicExch(w.err, 1);
            return;
        }
        if (warp_sat && q >= *reinterpret_cast<volatile int*>(sm.end)) break;
        if ((q & 3) == 0 && q > 0 && !warp_sat) {
            const bool dark = flush_tiny<VG, SAVE>(acc);
            warp_sat = __all_sync(0xffffffffu, dark || !live);
            if (warp_sat && lane == 0) atomicAdd(sm.sat, 1);
        }
        const uint32_t empty = sm.empty + 8 * ring.st;
        uint32_t sa = sm.stages + (uint32_t)ring.st * G.stage_bytes;
        uint32_t d = sm.desc + (uint32_t)(q & (kDescs - 1)) * DB;
        const uint32_t d_end = warp_sat ? d : d + (uint32_t)min(kPair, P - q) * DB;
        for (; d != d_end; d += DB, sa += G.plane_bytes) {
            const float4 A = lds_f4(d);
            const int mode = (__float_as_int(A.z) >> tg.mode_sh) & 3;
            if (!BILINEAR) {
                if (mode == kInside)
                    blend_nearest<DT, VG, SAVE, kInside>(p, G, planes, acc, A, d, sa, tg, sm, stop, Y0);
                else if (mode == kBorder)
                    blend_nearest<DT, VG, SAVE, kBorder>(p, G, planes, acc, A, d, sa, tg, sm, stop, Y0);
                else if (mode == kGlobal)
                    blend_nearest<DT, VG, SAVE, kGlobal>(p, G, planes, acc, A, d, sa, tg, sm, stop, Y0);
            } else if (mode != kSkip) {
                const int kw = __float_as_int(A.z);
                const float4 B = lds_f4(d + 16);
                const RowPair rp(p, tg, B.x, B.y);
                const int lo = (int)lds_u32(d + 32 + 4 * (tid >> 5)), n = (int)lds_u32(d + 48 + 4 * (tid >> 5));
                // blending a warp's window first pays while it is read more often than it is
                // made, some 2 accesses per 32 texels against one saved per view (few views
                // that lie far apart have wide windows): 3 views of 512^2, N 64, FP32 162 us
                // with a line at 2/3, 152 at 1/2; RGBA8 texels, which need unpacking, 197 and 262
                const bool direct = VG <= 5 && mode != kGlobal &&
                                    (DT == LF_U8 ? 3 * ((n + 31) / 32) > 2 * VG : 2 * ((n + 31) / 32) > VG);
                if (n > 0 && direct) {
                    const uint32_t r0 = sa + tg.row, c = (uint32_t)(tg.pxm - __float_as_int(A.y));
                    ViewH vh;
#pragma unroll
                    for (int jj = 0; jj < VG; ++jj) {
                        float wx;
                        const uint32_t b = tap_bits(A.x, tg.xf, vh.template get<VG>(sa, A.w, jj), false, wx);
                        const uint32_t i0 = b + (uint32_t)tg.pxm;
                        float4 u0, u1;
                        sample_staged<DT>(r0, r0 + G.win_bytes, rp, b + c, b + c + 1u, i0 < (uint32_t)p.W,
                                          i0 + 1u < (uint32_t)p.W, u0, u1);
                        blend_texel<SAVE>(acc[jj], mix_taps(wx, u0, u1), stop, jj, kw >> 8);
                    }
                } else if (n > 0 && n < (int)G.wcap) {
                    __syncwarp();   // the plane before has been read
                    blend_rows<DT>(p, planes, sa, tg, G, rp, mode, kw >> 8, __float_as_int(A.y), lo, n, wrow);
                    __syncwarp();
                    if (mode == kInside)
                        blend_taps<VG, SAVE, true>(acc, A, sa, wrow, lo, n, tg, stop, false);
                    else
                        blend_taps<VG, SAVE, false>(acc, A, sa, wrow, lo, n, tg, stop, mode == kGlobal);
                } else if (n > 0) {
                    // window wider than the warp's row (a plane far nearer than the rest)
                    ViewH vh;
#pragma unroll
                    for (int jj = 0; jj < VG; ++jj) {
                        float wx;
                        const int i0 = (int)tap_bits(A.x, tg.xf, vh.template get<VG>(sa, A.w, jj), true, wx) + tg.pxm;
                        float4 tb;
                        const float4 ta = sample_global<DT>(p, planes, kw >> 8, rp, i0, &tb);
                        blend_texel<SAVE>(acc[jj], mix_taps(wx, ta, tb), stop, jj, kw >> 8);
                    }
                }
            }
        }
        __syncwarp();
        if (lane == 0) mbar_arrive(empty);
    }
    if (!live) return;
#pragma unroll
    for (int jj = 0; jj < VG; ++jj) {
        const int j = j0 + jj;
        if (j >= p.Vx) break;
        const int v = vi * p.Vx + j;
        const float T = SAVE ? fmaxf(acc[jj][3], 0.0f) : acc[jj][3];
        if (partial) {
            const float4 qt = make_float4(acc[jj][0], acc[jj][1], acc[jj][2], T);
            if (part)
                part[((size_t)v * p.Ny + y) * p.Nx + x] = qt;
            else
                reinterpret_cast<float4*>(out)[view_pixel(p, v, x, y)] = qt;
            continue;
        }
        reinterpret_cast<float4*>(out)[view_pixel(p, v, x, y)] = make_float4(
            fmaf(T, p.bg[0], acc[jj][0]), fmaf(T, p.bg[1], acc[jj][1]), fmaf(T, p.bg[2], acc[jj][2]), 1.0f - T);
        if (SAVE) {
            // stopped: {T_k, k} of the stop plane; else {T behind the last plane, N}
            const int k = acc[jj][3] < 0.0f ? (int)lds_u32(stop + 4u * jj) : p.N;
            state[((size_t)v * p.Ny + y) * p.Nx + x] = make_float4(fabsf(acc[jj][3]), __int_as_float(k), 0.0f, 0.0f);
        }
    }
}

// Most dynamic shared memory of a layout. Every launch sets its kernel's limit
// to this, whatever it needs: the limit is the kernel's, and one set to a
// launch's own size would refuse a larger launch of another thread.
constexpr size_t kCompSmemMax = 200 * 1024;

// CTAs per SM that the adjoint's registers leave room for: nearest 9 views at 96
// registers and 3 at 64 (9 at 128: 3.22 ms a fitting step of 300k Gaussians
// instead of 3.10, with fewer spills but fewer warps); bilinear 9 at 128 and 3 at 96,
// without spills (fitting steps of 256^2, N 64, 12 views: 1.32 ms with 96 and
// 64, 0.95 now; 45 views 2.72 and 2.29).
__host__ __device__ constexpr int comp_bwd_ctas(int VG, bool bilinear)
{
    return bilinear ? (VG > 3 ? 3 : 4) : (VG > 3 ? 4 : 6);
}

// CTAs per SM of the forward, that is, registers per thread: nearest 15 views
// at 96, 9 at 72 (FP32 planes; the others, whose texels take fewer registers,
// at 64), bilinear 15 at 128 (three CTAs: 0.91 ms on FP16 planes, 45 views of
// 512^2, N 64; at 96 registers spills take it to 1.03), fewer at 96 (FP32, 5
// views of 256^2, N 64: 92 us at six CTAs and 64 registers, with spills, 65
// now; 2 views 72 and 52), but RGBA8, 3 views and fewer, which has the shortest
// windows, at five CTAs (2 x 2 views of 400^2, N 50: 214 us at four, 197 now).
__host__ __device__ constexpr int comp_ctas(int VG, bool bilinear, int dtype)
{
    return bilinear ? (VG > 9 ? 3 : VG > 3 || dtype != LF_U8 ? 4 : 5) : (VG > 9 ? 4 : VG > 5 ? (dtype == LF_F32 ? 5 : 6) : 7);
}

// f.template operator()<DT, BILINEAR>() for the run-time plane type and sampling
template <typename F>
void dispatch(int dtype, bool bilinear, F f)
{
    switch (dtype) {
    case LF_F32: bilinear ? f.template operator()<LF_F32, true>() : f.template operator()<LF_F32, false>(); break;
    case LF_F16: bilinear ? f.template operator()<LF_F16, true>() : f.template operator()<LF_F16, false>(); break;
    case LF_U8: bilinear ? f.template operator()<LF_U8, true>() : f.template operator()<LF_U8, false>(); break;
    default: bilinear ? f.template operator()<LF_BF16, true>() : f.template operator()<LF_BF16, false>(); break;
    }
}

}  // namespace

}  // namespace lf
