// lf_composite.cu -- swizzle blending of the sweeping planes into the quilt
// views (Sec. 4.3; the compositing steps of Algorithm 1), and its adjoint.
//
// k_comp_tables evaluates, per (view column j, plane k) and (view row i,
// plane k), the affine form of Eq. (u_prime) in plane pixels,
//   X(x) = P_s x + (gm x + hb),  X(x) + 1/2 = P_s x + (gm x + hn),
// from the FP64 display set-up (Delta x_j = 2 D_focal s_j tan(phi_x/2),
// den = (d_k - D_forward) tan(theta'/2), a = d_k tan(theta/2),
// g = W a / (Nx den), h = (W/2)((Delta (D_focal - d_k)/D_focal + a (1-Nx)/Nx)/den + 1) - 1/2,
// gm = g - P_s), rounded once to FP32.
// The composite kernels walk the planes front to back for every view pixel:
// nearest texel index P_s x + floor(fma(gm, x, hn)) (FP32 decision), or
// bilinear taps around X with zero padding; Q += T c_k, T *= 1 - A_k
// (Eq. (alpha_blend)); empty planes skipped; output (Q + T bg, 1 - T).
#include <cmath>
#include <cstring>
#include <initializer_list>

#include "lf_composite.cuh"

namespace lf {

namespace {

__device__ __forceinline__ double view_offset(int j, int V, double Df, double tphi)
{
    const double s = V <= 1 ? 0.0 : __dsub_rn(__ddiv_rn((double)j, (double)(V - 1)), 0.5);
    return __dmul_rn(__dmul_rn(__dmul_rn(2.0, Df), s), tphi);
}

__device__ __forceinline__ void axis_coeffs(double delta, double dk, double Df, double Dfwd, double tth, double tthp,
                                            int n, int Wp, int P_s, float* out)
{
    const double den = __dmul_rn(__dsub_rn(dk, Dfwd), tthp);
    const double a = __dmul_rn(dk, tth);
    const double g = __ddiv_rn(__dmul_rn((double)Wp, a), __dmul_rn((double)n, den));
    const double A = __ddiv_rn(__dmul_rn(delta, __dsub_rn(Df, dk)), Df);
    const double c0 = __ddiv_rn(__dmul_rn(a, (double)(1 - n)), (double)n);
    const double hw = __dmul_rn(0.5, (double)Wp);
    const double hn = __dmul_rn(hw, __dadd_rn(__ddiv_rn(__dadd_rn(A, c0), den), 1.0));
    out[0] = __double2float_rn(__dsub_rn(g, (double)P_s));
    out[1] = __double2float_rn(hn);
    out[2] = __double2float_rn(__dsub_rn(hn, 0.5));
}

// Tables of one composite, non-empty planes only, in order ("list entries"):
// w.blk[group][entry][CoefBlock] per group of VG view columns, w.yt[view
// row][entry] = (gm, h) along y, *w.np entries. CTA (x, y): planes 4 x ..
// 4 x + 3, view group y (or, past the groups, 16 view rows). The staged
// kernels stream an entry's block with its plane rows, so their CTAs start
// without loading a table. The work is FP64 divisions at two lanes a clock
// and SM, so the CTAs are small: 64 threads, one plane pair a warp (512
// threads on a tenth of the SMs: 14 us for 45 views of 64 planes).
__device__ __forceinline__ void comp_tables(const CompParams& p, const double* __restrict__ d,
                                            const int32_t* __restrict__ count, const CompWs& w, int VG)
{
    __shared__ float s_h[kTabViews][kTabPlanes];
    __shared__ int s_wide[kTabPlanes];
    const int tx = threadIdx.x, ty = threadIdx.y, tid = ty * kTabPlanes + tx;
    const int k0 = blockIdx.x * kTabPlanes, k = k0 + tx;
    const int groups = (p.Vx + VG - 1) / VG;
    const int row = blockIdx.y;
    if (k0 >= p.N || row >= groups + (p.Vy + kTabViews - 1) / kTabViews) return;
    // list entry of plane k: non-empty planes before it
    int q = 0;
    for (int b = 0; b < k0; b += kTabPlanes * kTabViews) q += __syncthreads_count(b + tid < k0 && count[b + tid] != 0);
    const bool ne = k < p.N && count[k] != 0;
    int total = q;
#pragma unroll
    for (int e = 0; e < kTabPlanes; ++e) {
        const int c = k0 + e < p.N && count[k0 + e] != 0;
        q += e < tx ? c : 0;
        total += c;
    }
    if (row == 0 && tid == 0) {
        if (k0 == 0) *w.err = 0;
        if (k0 + kTabPlanes >= p.N) *w.np = total;
    }
    float o[3];
    if (row >= groups) {
        const int i = (row - groups) * kTabViews + ty;
        if (ne && i < p.Vy) {
            axis_coeffs(view_offset(i, p.Vy, p.D_focal, p.tphi_y), d[k], p.D_focal, p.D_forward, p.tth_y, p.tthp_y, p.Ny,
                        p.H, p.P_s, o);
            w.yt[(size_t)i * p.N + q] = make_float2(o[0], p.bilinear ? o[2] : o[1]);
        }
        return;
    }
    const int CW = VG == 1 ? 4 : 4 + 4 * ((VG + 3) / 4);
    float* blk = w.blk + ((size_t)row * p.N + q) * CW;
    if (ty == 0) s_wide[tx] = 0;
    __syncthreads();
    if (ne && ty < VG) {
        const int j = min(row * VG + ty, p.Vx - 1);
        axis_coeffs(view_offset(j, p.Vx, p.D_focal, p.tphi_x), d[k], p.D_focal, p.D_forward, p.tth_x, p.tthp_x, p.Nx,
                    p.W, p.P_s, o);
        const float h = p.bilinear ? o[2] : o[1];
        s_h[ty][tx] = h;
        if (VG > 1) blk[4 + ty] = h;
        // the row's range of gm x + h (affine in x): flag planes that may leave kNarrow
        const float lo = fminf(o[2], o[1]), hi = fmaxf(o[2], o[1]);
        const float span = fabsf(o[0]) * (float)(p.Nx - 1);
        if (!(fmaxf(fabsf(lo), fabsf(hi)) + span + 2.0f < 0.99f * kNarrow)) s_wide[tx] = 1;
    }
    __syncthreads();
    if (ne && ty == 0) {
        float mn = s_h[0][tx], mx = mn;
        for (int v = 1; v < VG; ++v) mn = fminf(mn, s_h[v][tx]), mx = fmaxf(mx, s_h[v][tx]);
        *reinterpret_cast<float4*>(blk) = make_float4(o[0], mn, mx, __int_as_float(k | (s_wide[tx] ? kWideBit : 0)));
    }
}

__global__ void __launch_bounds__(kTabPlanes* kTabViews) k_comp_tables(CompParams p, const double* __restrict__ d,
                                                                       const int32_t* __restrict__ count, CompWs w,
                                                                       int VG)
{
    pdl_wait();
    pdl_trigger();
    comp_tables(p, d, count, w, VG);
}

// every scene of a batch: scene blockIdx.z
__global__ void __launch_bounds__(kTabPlanes* kTabViews) k_comp_tables_batched(const CompScene* __restrict__ scs)
{
    const CompScene& sc = scs[blockIdx.z];
    const CompParams p = sc.p;
    comp_tables(p, sc.d, sc.count, sc.w, sc.G.VG);
}

template <int DT, bool BILINEAR, int VG, bool SAVE>
__global__ void __launch_bounds__(kCompBlock, comp_ctas(VG, BILINEAR, DT))
    k_composite_staged(const __grid_constant__ CompParams p, const __grid_constant__ CompGeom G,
                       const char* __restrict__ planes, const __grid_constant__ CompWs w, float* __restrict__ out,
                       float4* __restrict__ state)
{
    pdl_wait();
    // fastest: the view groups, then the column tiles of one row band, so
    // that the CTAs reading the same plane rows run together (rows read from
    // DRAM once, then from L2)
    const int nvg = G.groups_x * p.Vy;
    // row bands from both edges inward: the bands whose views rarely reach
    // T = 0 (the scene's borders) start first, the cheap centre ones last
    const int by = (int)blockIdx.y;
    const int band = (by & 1) ? (int)gridDim.y - 1 - (by >> 1) : (by >> 1);
    composite_tile<DT, BILINEAR, VG, SAVE>(p, G, planes, w, out, state, nullptr, false, blockIdx.x % nvg,
                                           (blockIdx.x / nvg) * G.TX, band * G.BY, 0, *w.np);
}

// Failure-detection self-test: one thread waits on an mbarrier of expected
// count 1 that nothing arrives on, with the wait limit given; the bounded
// wait gives up and the kernel records how (1: gave up, 2: the phase
// completed, which cannot happen) and exits normally.
__global__ void k_wait_selftest(unsigned long long limit_ns, int* result)
{
    __shared__ uint64_t bar;
    const uint32_t b = smem_addr(&bar);
    mbar_init(b, 1);
    fence_proxy_async();
    *result = mbar_wait_for(b, 0u, limit_ns) ? 2 : 1;
}

// Texels that a group of VG views spreads over on the planes from nearest times
// the focal distance (from the reference camera) on.
constexpr double kNearest = 0.25;
double view_spread(const CompParams& p, int VG, double nearest = kNearest)
{
    if (p.Vx < 2) return 0.0;
    const double near = nearest * p.D_focal, views = (VG < p.Vx ? VG : p.Vx) - 1;
    const double near_shift = std::fabs(p.D_focal - p.D_forward - near) / (near * p.tthp_x), far_shift = 1.0 / p.tthp_x;
    return 0.5 * p.W * views * 2.0 * p.tphi_x / (p.Vx - 1) * (near_shift > far_shift ? near_shift : far_shift);
}

constexpr double kAdvance = 1.3;   // most texels (over P_s) between neighbouring pixels

// Columns of a tile, at most `most`: 128, 64 or 32, whichever pads and stages
// least: a narrower tile pads the view's width less and stages relatively
// wider windows (a staged texel costs about 0.4 of a sample). Ragged rows are
// copied texel by texel, row after row, by the producer warp, which a tile of
// several rows of the forward waits for (the adjoint has more to do): with 128, 64 and 32 columns, 10 views of 251^2, N 150,
// FP16, take 93, 107 and 144 us, 16 views of 151 x 110, N 128, BF16, 94, 82 and
// 108, 16 views of 203 x 150, N 128, BF16, 105, 114 and 127.
int tile_columns(const CompParams& p, int VG, int most, bool bwd)
{
    const bool ragged = !bwd && (size_t)p.W * texel_bytes(p.dtype) % 16 != 0;
    const double by_64 = ragged ? 1.1 : 1.02, by_32 = ragged ? 1.5 : 1.05;
    int best = 32;
    double best_cost = 1e300;
    for (int tx : {128, 64, 32}) {
        if (tx > most) continue;
        const double window = tx * kAdvance * p.P_s + view_spread(p, VG, p.bilinear ? 0.5 : kNearest);
        const double cost = (double)((p.Nx + tx - 1) / tx * tx) * (tx == 128 ? 1.0 : tx == 64 ? by_64 : by_32) *
                            (1.0 + 0.4 * (p.bilinear ? 2.0 : 1.0) * window / ((double)tx * VG));
        if (cost < best_cost) best_cost = cost, best = tx;
    }
    return best;
}

constexpr double kSMs = 152.0;

// Views per thread: the least waves of CTAs times (VG + fixed) per CTA and CTAs
// per SM. The fixed cost of a view group (staging every plane's window) is
// worth about three views. A last, partly filled wave counts half a wave and
// half of what fills it (its CTAs have the SM to fewer): it decides where the
// grid is small -- 9 views of 128^2, N 16: 3 views per thread run 2 % faster
// than 9 (0.142 against 0.146 ms a frame); 9 of 256^2 bilinear: 9 run 7 %
// faster than 3; 45 of 512^2: 15 run 6 % faster than 9.
// The bilinear adjoint's cost goes almost by the sample, a group's fixed cost
// is about 0.6 views: 45 views of 256^2, 9 per thread 2.29 ms a fitting step, 3
// per thread 2.49; 12 views 1.26 and 0.95.
template <typename Ctas>
int views_per_thread(const CompParams& p, std::initializer_list<int> options, bool bwd, double fixed, Ctas ctas)
{
    int best = 1;
    double best_cost = 1e300;
    for (int vg : options) {
        const int tx = tile_columns(p, vg, 128, bwd), by = kCompThreads / tx;
        const double tiles = (double)((p.Nx + tx - 1) / tx) * ((p.Ny + by - 1) / by) * p.Vy;
        const double waves = tiles * ((p.Vx + vg - 1) / vg) / (kSMs * ctas(vg)), whole = std::floor(waves);
        const double part = waves - whole;
        const double cost = (whole + (part > 0.0 ? 0.5 + 0.5 * part : 0.0)) * (vg + fixed) * ctas(vg);
        if (cost < best_cost) best_cost = cost, best = vg;
    }
    return best;
}

template <int DT, bool BILINEAR, int VG, bool SAVE>
void launch_fwd(const CompParams& p, const CompGeom& G, const void* planes, const CompWs& ws, float* out, float4* state,
                cudaStream_t s)
{
    auto kern = k_composite_staged<DT, BILINEAR, VG, SAVE>;
    cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kCompSmemMax);
    const dim3 grid((unsigned)(G.groups_x * p.Vy * ((p.Nx + G.TX - 1) / G.TX)), (unsigned)((p.Ny + G.BY - 1) / G.BY));
    launch_pdl(kern, grid, dim3(kCompBlock), G.smem_bytes, s, p, G, static_cast<const char*>(planes), ws, out, state);
}

struct FwdLaunch {
    const CompParams& p;
    const CompGeom& G;
    const void* planes;
    const CompWs& ws;
    float* out;
    float4* state;
    cudaStream_t s;
    template <int DT, bool BILINEAR, int VG>
    void vg() const
    {
        if (state)
            launch_fwd<DT, BILINEAR, VG, true>(p, G, planes, ws, out, state, s);
        else
            launch_fwd<DT, BILINEAR, VG, false>(p, G, planes, ws, out, nullptr, s);
    }
    template <int DT, bool BILINEAR>
    void operator()() const
    {
        switch (G.VG) {
        case 15: vg<DT, BILINEAR, 15>(); break;
        case 9: vg<DT, BILINEAR, 9>(); break;
        case 5: vg<DT, BILINEAR, 5>(); break;
        case 3: vg<DT, BILINEAR, 3>(); break;
        default: vg<DT, BILINEAR, 1>(); break;
        }
    }
};

}  // namespace

int comp_views_fwd(const CompParams& p)
{
    return views_per_thread(p, {15, 9, 5, 3, 1}, false, 3.0, [&](int vg) { return comp_ctas(vg, p.bilinear != 0, p.dtype); });
}

int comp_views_bwd(const CompParams& p)
{
    const bool bilinear = p.bilinear != 0;
    return views_per_thread(p, {9, 3}, true, bilinear ? 0.6 : 3.0, [&](int vg) { return comp_bwd_ctas(vg, bilinear); });
}

// Staged layout of one composite (see CompGeom). The stage holds the window
// that a tile needs on the planes from a quarter of the focal distance on, or
// the whole plane row where that fits the shared memory the CTAs of an SM can
// share; wider windows (planes nearer still) are read through L1 (kGlobal).
// Where two stages do not fit the shared memory at all, the windows are cut to
// what does (FP32, 9 views of 256 x 200 at P_s = 8, N 24, bilinear: 118 us; 496
// with windows of half that, which most planes' do not fit).
CompGeom comp_geom(const CompParams& p, const void* planes, int VG, bool save, bool bwd, int tile_x)
{
    CompGeom G;
    std::memset(&G, 0, sizeof(G));
    const size_t TB = (size_t)texel_bytes(p.dtype);
    const int rpy = p.bilinear ? 2 : 1;
    G.TX = tile_columns(p, VG, tile_x, bwd);
    G.BY = kCompThreads / G.TX;
    G.VG = VG;
    G.groups_x = (p.Vx + VG - 1) / VG;
    G.bulk = ((uintptr_t)planes) % 16 == 0 && ((size_t)p.W * TB) % 16 == 0;
    G.hdr_bytes = (uint32_t)(VG == 1 ? 0 : 16 * ((VG + 3) / 4));
    const double advance = kAdvance * p.P_s;
    const size_t stop = save ? 4 * (size_t)kCompThreads * VG : 0;
    const size_t ctrl = 16 * kStages + 16 + 16 * kDescs + (size_t)kDescs * (p.bilinear ? 64 : kDescBytes);
    const int ctas = bwd ? comp_bwd_ctas(VG, p.bilinear != 0) : comp_ctas(VG, p.bilinear != 0, p.dtype);
    const size_t budget = (size_t)(227 * 1024) / ctas - 1024;
    const size_t full = round16((size_t)p.W * TB) + 16;   // and the zero texel
    auto stage = [&](size_t win) { return kPair * (G.hdr_bytes + win * G.BY * rpy); };
    size_t rows = 0, fixed = 0, need = 0;
    // Bilinear, few views far apart: the windows of near planes alone can take
    // so much shared memory that fewer CTAs run than the registers allow, with
    // two stages each (FP32, 3 x 2 views of 323^2, N 69, a fitting step: 1.19 ms
    // with windows from a quarter of the focal distance on, 1.08 from 0.35 on;
    // 3 views of 512^2: 185 and 162 us from half of it on). Then only planes
    // further away get windows, up to half the focal distance: a display
    // focused at the middle disparity of its scene has no nearer ones.
    for (double nearest : {kNearest, 0.35, 0.5}) {
        const double spread = view_spread(p, VG, nearest);
        // per-warp rows, bilinear: the blended row; the adjoint's gradient sums
        const double warp_tex = 32.0 * advance + spread + 4.0;
        G.wcap = (uint32_t)(warp_tex < 512.0 ? warp_tex : 512.0) / 8 * 8;
        rows = p.bilinear ? (size_t)kWarps * G.wcap * 16 * (bwd ? 3 : 1) : 0;
        fixed = rows + ctrl + stop + 128;
        const double tile_tex = G.TX * advance + spread + 4.0 + 48.0 / (double)TB;
        need = tile_tex * (double)TB < (double)full ? round16((size_t)tile_tex * TB) : full;
        if (!p.bilinear || fixed + 3 * stage(need) <= budget) break;
    }
    G.stages = kStages;
    while (G.stages > 2 && fixed + G.stages * stage(need) > budget) --G.stages;
    while (G.stages > 2 && fixed + G.stages * stage(need) > kCompSmemMax) --G.stages;
    size_t win = need;
    if (fixed + G.stages * stage(full) <= budget)
        win = full;
    else if (fixed + G.stages * stage(need) > kCompSmemMax)
        win = ((kCompSmemMax - fixed) / G.stages / kPair - G.hdr_bytes) / (G.BY * rpy) / 16 * 16;
    G.win_bytes = (uint32_t)win;
    G.cap = (int)((win - 16) / TB);
    G.stage_bytes = (uint32_t)stage(win);
    G.plane_bytes = G.stage_bytes / kPair;
    G.rows_off = (uint32_t)(((size_t)G.stages * G.stage_bytes + 127) / 128 * 128);
    G.bar_off = (uint32_t)(G.rows_off + rows);
    G.stop_off = (uint32_t)(G.bar_off + ctrl);
    G.smem_bytes = (uint32_t)(G.stop_off + stop);
    return G;
}

void launch_comp_tables(const CompParams& p, const double* d, const int32_t* count, const CompWs& ws, cudaStream_t s)
{
    int chunks = 0, rows = 0;
    comp_tables_grid(p, ws.VG, &chunks, &rows);
    launch_pdl(k_comp_tables, dim3((unsigned)chunks, (unsigned)rows), dim3(kTabPlanes, kTabViews), 0, s, p, d, count, ws,
               ws.VG);
    note_launches(1);
}

void launch_comp_tables_batched(const CompScene* scenes_dev, int n_sc, int max_chunks, int max_rows, cudaStream_t s)
{
    k_comp_tables_batched<<<dim3((unsigned)max_chunks, (unsigned)max_rows, (unsigned)n_sc),
                            dim3(kTabPlanes, kTabViews), 0, s>>>(scenes_dev);
    note_launches(1);
}

void comp_tables_grid(const CompParams& p, int VG, int* chunks, int* rows)
{
    *chunks = (p.N + kTabPlanes - 1) / kTabPlanes;
    *rows = (p.Vx + VG - 1) / VG + (p.Vy + kTabViews - 1) / kTabViews;
}

void launch_composite(const CompParams& p, const void* planes, const CompWs& ws, float* out, cudaStream_t s,
                      float4* state)
{
    const CompGeom G = comp_geom(p, planes, ws.VG, state != nullptr, false, 128);
    dispatch(p.dtype, p.bilinear != 0, FwdLaunch{p, G, planes, ws, out, state, s});
    note_launches(1);
}

namespace {

// Composition of a batch scene's chunk groups, front to back (the "over"
// operator is associative): Q = Q_0 + T_0 Q_1 + T_0 T_1 Q_2 ..., T = T_0 T_1
// ...; then the views (Q + T bg, 1 - T).
__global__ void k_merge_chunk_groups(CompParams p, int groups, const float4* __restrict__ part, float* out)
{
    const long long per = (long long)p.Nx * p.Ny;
    const long long total = per * p.Vx * p.Vy;
    for (long long e = (long long)blockIdx.x * blockDim.x + threadIdx.x; e < total;
         e += (long long)gridDim.x * blockDim.x) {
        const int v = (int)(e / per);
        const long long pix = e - (long long)v * per;
        const int y = (int)(pix / p.Nx), x = (int)(pix - (long long)y * p.Nx);
        float4* dst = reinterpret_cast<float4*>(out) + view_pixel(p, v, x, y);
        float4 a = *dst;
        for (int c = 1; c < groups; ++c) {
            const float4 b = __ldcs(part + ((size_t)(c - 1) * p.Vx * p.Vy * per + e));
            a.x = fmaf(a.w, b.x, a.x);
            a.y = fmaf(a.w, b.y, a.y);
            a.z = fmaf(a.w, b.z, a.z);
            a.w *= b.w;
        }
        *dst = make_float4(fmaf(a.w, p.bg[0], a.x), fmaf(a.w, p.bg[1], a.y), fmaf(a.w, p.bg[2], a.z), 1.0f - a.w);
    }
}

}  // namespace

void launch_merge_chunk_groups(const CompParams& p, int groups, const float4* part, float* out, cudaStream_t s)
{
    const long long total = (long long)p.Nx * p.Ny * p.Vx * p.Vy;
    const long long want = (total + 255) / 256;
    const unsigned blocks = (unsigned)(want < 152 * 32 ? want : 152 * 32);
    k_merge_chunk_groups<<<blocks, 256, 0, s>>>(p, groups, part, out);
    note_launches(1);
}

void launch_wait_selftest(unsigned long long limit_ns, int* result, cudaStream_t s)
{
    k_wait_selftest<<<1, 1, 0, s>>>(limit_ns, result);
    note_launches(1);
}

}  // namespace lf
