// lf_sort.cu -- stable LSD radix sort (8-bit digits) of (key, value) pairs,
// and the depth order built on it.
//
// Used twice per build:
//  - the depth sort of Algorithm 1 (its sort-and-chunk step): the order of
//    the culled-in primitives by (FP64 depth, index). The IEEE bits of a
//    positive FP64 depth order like the depth; relative to the smallest valid
//    key they span up to ~55 bits. The sort takes their top 24 varying bits
//    (an order-preserving truncation) as a 32-bit key, drops culled
//    primitives in the first pass and sorts stably in three passes (the
//    first pass takes each key's index as its value, so equal keys stay in
//    index order). Keys that share the truncated value form runs that are
//    then put in (full key, index) order: every member of a run of up to 32
//    counts the members before it, longer runs that are out of order go to
//    one CTA each (Batcher's odd-even merge network, in shared memory up to
//    2048 keys, in global memory beyond). The run pass keeps the order exact
//    for any input; 24 bits trade a fourth pass for short runs (1M Gaussians
//    over depths 1.5..10: runs of at most 5 keys, 12k pairs to reorder;
//    grid-aligned voxels: runs of equal full keys, already in order).
//  - the 3D tiling (Sec. 4.4): 32-bit keys = super-tile id of every
//    (super-tile, rank) pair emitted in rank order; the stable sort groups the
//    pairs by super-tile and keeps each one's pairs in depth order.
//
// One kernel per pass (k_sweep), by decoupled look-back (Merrill and Garland,
// Single-pass Parallel Prefix Scan with Decoupled Look-back, 2016), with the
// digit totals of all passes known beforehand (k_depth_hist; the pair
// emission): a block of 512 threads ranks
// its 2048 or 4096 keys stably (ballot-based digit matching, per-warp
// counters, warps own contiguous key ranges), publishes its digit counts,
// exchanges the keys through shared memory into digit order, adds up the
// counts of the blocks before it by decoupled look-back (one thread per
// digit, 16 predecessors per round trip), and writes every digit run
// contiguously. Blocks of 2048 keys while those make one wave of the chip's
// 152 SMs, else 4096 (two blocks of 64 registers a thread per SM; 8192 keys
// at one block per SM left too few warps for the ranking: 33 us a pass at 1M
// keys). A pass is bound by the ranking's instructions and the look-back's
// latency. (Three
// kernels per pass over 2048-key blocks -- counts, one scan per digit,
// scatter -- took 83 us for the three passes of 1M keys and some 40 us for
// 10k, where launches dominate.)
// Item counts may live on the device (culled-in count, pair count), so grids
// are sized for the capacity and blocks past the count exit early.
#include "lf_internal.cuh"

namespace lf {

namespace {

constexpr int kBits = 8;
constexpr int kDigits = 1 << kBits;
constexpr int kWarps = kSweepThreads / 32;
constexpr int kDepthKeyBits = 24;                // truncated depth key width
constexpr uint32_t kDepthKeyMask = (1u << kDepthKeyBits) - 1u;
static_assert(kDepthPasses * kBits == kDepthKeyBits, "digits of the truncated depth key");

// Right shift that keeps the top kDepthKeyBits varying bits of a depth key
// relative to the smallest valid key (0 if the range already fits).
__device__ __forceinline__ int depth_shift(unsigned long long lo, unsigned long long hi)
{
    if (lo > hi) return 0;
    const int bits = 64 - __clzll((long long)(hi - lo));
    return bits > kDepthKeyBits ? bits - kDepthKeyBits : 0;
}

// lanes holding the same digit (ballot per digit bit); valid lanes only
__device__ __forceinline__ uint32_t match_digit(uint32_t d, bool ok)
{
    uint32_t peers = __ballot_sync(0xffffffffu, ok);
#pragma unroll
    for (int b = 0; b < kBits; ++b) {
        const bool bit = (d >> b) & 1u;
        const uint32_t m = __ballot_sync(0xffffffffu, bit);
        peers &= bit ? m : ~m;
    }
    return peers;
}

// exclusive scan of one value per thread over the block; every thread calls it
__device__ __forceinline__ uint32_t block_exscan(uint32_t v, uint32_t* warp_tmp)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    uint32_t x = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t u = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += u;
    }
    __syncthreads();
    if (lane == 31) warp_tmp[warp] = x;
    __syncthreads();
    uint32_t before = 0;
#pragma unroll
    for (int w = 0; w < kWarps; ++w) before += w < warp ? warp_tmp[w] : 0u;
    return before + x - v;
}

// Digit totals of the three depth passes over the culled-in keys.
constexpr int kHistKeys = 16;   // keys per thread
__global__ void __launch_bounds__(kSweepThreads) k_depth_hist(BuildWs w, long long n)
{
    pdl_wait();
    pdl_trigger();
    __shared__ uint32_t h[kDepthPasses][kDigits];
    for (int i = threadIdx.x; i < kDepthPasses * kDigits; i += kSweepThreads) (&h[0][0])[i] = 0u;
    const unsigned long long lo = w.hdr->kmin;
    const int shift = depth_shift(lo, w.hdr->kmax);
    __syncthreads();
    const long long base = (long long)blockIdx.x * (kSweepThreads * kHistKeys);
    unsigned long long k[kHistKeys];
#pragma unroll
    for (int r = 0; r < kHistKeys; ++r) {
        const long long i = base + r * kSweepThreads + threadIdx.x;
        k[r] = i < n ? w.keyA[i] : kInvalidKey;
    }
#pragma unroll
    for (int r = 0; r < kHistKeys; ++r) {
        if (k[r] == kInvalidKey) continue;
        const uint32_t t = (uint32_t)((k[r] - lo) >> shift);
#pragma unroll
        for (int q = 0; q < kDepthPasses; ++q) atomicAdd(&h[q][(t >> (q * kBits)) & (kDigits - 1)], 1u);
    }
    __syncthreads();
    for (int i = threadIdx.x; i < kDepthPasses * kDigits; i += kSweepThreads) {
        const uint32_t c = (&h[0][0])[i];
        if (c) atomicAdd(&w.dhist[i], c);
    }
}

struct SweepArgs {
    WsHeader* hdr;
    long long n_static;                    // number of keys, unless n_dev
    const unsigned long long* n_dev;       // device count (or null)
    int shift;
    int pass;                              // ticket
    int look_tries;
    const uint32_t* tot;                   // digit totals of this pass
    unsigned long long* stat;              // look-back words [blocks][kDigits]
};

constexpr int kLook = 16;   // predecessors per round trip of the look-back

template <int KPT>
struct SweepSmem {
    uint32_t wcnt[kWarps][kDigits];       // per-warp digit counts, then per-warp offsets
    uint32_t blk_start[kDigits];          // block-local start of every digit run
    uint32_t glob_base[kDigits];          // global destination of every digit run
    uint32_t xkey[kSweepThreads * KPT];   // exchange buffer in block-local digit order
    uint32_t xval[kSweepThreads * KPT];
    uint32_t warp_tmp[kWarps];
    uint32_t tile, placed;
};

// One pass. FIRST (depth): the keys are the truncated forms of the 64-bit
// keys at kin, culled ones dropped; a key's value is its index.
template <int KPT, bool FIRST>
__global__ void __launch_bounds__(kSweepThreads, 2) k_sweep(const void* __restrict__ kin, const uint32_t* __restrict__ vin,
                                                         uint32_t* __restrict__ kout, uint32_t* __restrict__ vout,
                                                         SweepArgs a)
{
    pdl_wait();
    pdl_trigger();
    extern __shared__ __align__(16) unsigned char sweep_raw[];
    SweepSmem<KPT>& S = *reinterpret_cast<SweepSmem<KPT>*>(sweep_raw);
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const long long n = a.n_dev ? (long long)*a.n_dev : a.n_static;
    // After a wait gave up (in a pass before, or in an earlier block of this one)
    // no block does anything: the tickets lie past any count of keys. (The keys
    // may hold stale ones then, which the digit totals don't count, and their
    // places could lie past the arrays.)
    if (tid == 0) S.tile = atomicAdd(&a.hdr->ticket[a.pass], 1u);
    for (int i = tid; i < kWarps * kDigits; i += kSweepThreads) (&S.wcnt[0][0])[i] = 0u;
    __syncthreads();
    const long long tile = S.tile, blk = tile * (kSweepThreads * KPT);
    if (blk >= n) return;

    // warp w owns keys [32 KPT w, 32 KPT (w + 1)) of the block, visited in
    // order round by round, so equal digits keep their order
    uint32_t key[KPT], val[KPT], pos[KPT];
    uint32_t okm = 0;
    const long long wbase = blk + warp * (32 * KPT);
    unsigned long long lo = 0;
    int dshift = 0;
    if (FIRST) {
        lo = a.hdr->kmin;
        dshift = depth_shift(lo, a.hdr->kmax);
    }
#pragma unroll
    for (int r = 0; r < KPT; ++r) {
        const long long idx = wbase + r * 32 + lane;
        bool ok = idx < n;
        if (FIRST) {
            const unsigned long long k = ok ? static_cast<const unsigned long long*>(kin)[idx] : kInvalidKey;
            ok = k != kInvalidKey;
            key[r] = (uint32_t)((k - lo) >> dshift);
            val[r] = (uint32_t)idx;
        } else {
            key[r] = ok ? static_cast<const uint32_t*>(kin)[idx] : 0u;
            val[r] = ok ? vin[idx] : 0u;
        }
        okm |= ok ? (1u << r) : 0u;
    }
    const uint32_t lt = (1u << lane) - 1u;
#pragma unroll
    for (int r = 0; r < KPT; ++r) {
        const bool ok = (okm >> r) & 1u;
        const uint32_t d = ok ? (key[r] >> a.shift) & (kDigits - 1u) : 0u;
        const uint32_t peers = match_digit(d, ok);
        const uint32_t before = ok ? S.wcnt[warp][d] : 0u;
        __syncwarp();
        pos[r] = before + __popc(peers & lt);
        if (ok && (__ffs(peers) - 1) == lane) S.wcnt[warp][d] = before + __popc(peers);
        __syncwarp();
    }
    __syncthreads();
    // per digit: exclusive offsets over warps and the block's count, published at once
    uint32_t run = 0;
    if (tid < kDigits) {
#pragma unroll
        for (int w = 0; w < kWarps; ++w) {
            const uint32_t c = S.wcnt[w][tid];
            S.wcnt[w][tid] = run;
            run += c;
        }
        st_word(a.stat + (size_t)tile * kDigits + tid, (tile == 0 ? kSumAll : kSumOwn) | run);
    }
    const uint32_t start = block_exscan(tid < kDigits ? run : 0u, S.warp_tmp);
    if (tid < kDigits) S.blk_start[tid] = start;
    if (tid == kDigits - 1) S.placed = start + run;
    const uint32_t dbase = block_exscan(tid < kDigits ? a.tot[tid] : 0u, S.warp_tmp);   // orders blk_start, too
    // exchange into block-local digit order
#pragma unroll
    for (int r = 0; r < KPT; ++r) {
        if (!((okm >> r) & 1u)) continue;
        const uint32_t d = (key[r] >> a.shift) & (kDigits - 1u);
        const uint32_t l = S.blk_start[d] + S.wcnt[warp][d] + pos[r];
        S.xkey[l] = key[r];
        S.xval[l] = val[r];
    }
    if (tid < kDigits) {
        unsigned long long sum = 0;
        long long t = tile - 1;
        int idle = 0;
        bool done = tile == 0;
        while (!done) {
            unsigned long long v[kLook];
#pragma unroll
            for (int u = 0; u < kLook; ++u)
                v[u] = t - u >= 0 ? ld_word(a.stat + (size_t)(t - u) * kDigits + tid) : kSumAll;
            int u = 0;
#pragma unroll
            for (int e = 0; e < kLook; ++e) {
                if (u != e || done || v[e] < kSumOwn) continue;   // in order, up to the first word not there yet
                sum += v[e] & kSumMask;
                done = v[e] >= kSumAll;
                ++u;
            }
            t -= u;
            idle = u ? 0 : idle + 1;
            if (idle > a.look_tries) {
                give_up(a.hdr);
                done = true;
            }
        }
        if (tile > 0) st_word(a.stat + (size_t)tile * kDigits + tid, kSumAll | (sum + run));
        S.glob_base[tid] = dbase + (uint32_t)sum;
    }
    __syncthreads();
    // coalesced write-out: item l of digit d goes to glob_base[d] + (l - blk_start[d])
    for (uint32_t l = tid; l < S.placed; l += kSweepThreads) {
        const uint32_t k = S.xkey[l], d = (k >> a.shift) & (kDigits - 1u);
        const uint32_t dst = S.glob_base[d] + (l - S.blk_start[d]);
        kout[dst] = k;
        vout[dst] = S.xval[l];
    }
}

// ---- depth order ---------------------------------------------------------

// (full key, index) order of two ranks' primitives
__device__ __forceinline__ bool depth_less(unsigned long long ka, uint32_t va, unsigned long long kb, uint32_t vb)
{
    return ka < kb || (ka == kb && va < vb);
}

constexpr int kShortRun = 32;
constexpr uint32_t kListed = 0x80000000u;   // on the first key of a long run that is out of order
constexpr int kLongRunCtas = 152;
constexpr int kLongRunThreads = 1024;
constexpr int kSmemRun = 2048;

// The sorted ranks (tkeyB, valB) into (full key, index) order (valA). A rank
// alone with its truncated key is copied. The members of a run of up to
// kShortRun equal truncated keys each count the members before them. Longer
// runs are copied (the sort is stable: they are in index order, which is right
// unless some neighbour pair has a larger full key first); a member that finds
// such a pair claims its run (top bit of the run's first key) and the first
// claim lists it in tkeyA for k_depth_long_runs. (Out of place: no rank reads
// what another one writes.)
__global__ void __launch_bounds__(256) k_depth_runs(BuildWs w)
{
    pdl_wait();
    pdl_trigger();
    const long long M = (long long)w.hdr->M;
    const long long r = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (r >= M || w.hdr->timeout) return;   // after a wait gave up valB is not an order
    const uint32_t* key = w.tkeyB;
    auto same = [&](long long i, uint32_t k) { return i >= 0 && i < M && ((key[i] ^ k) & kDepthKeyMask) == 0u; };
    const uint32_t k = key[r], v = w.valB[r];
    const bool left = same(r - 1, k), right = same(r + 1, k);
    if (!left && !right) {
        w.valA[r] = v;
        return;
    }
    long long s = r, e = r + 1;   // the run, as far as kShortRun from here
    bool longer = same(r - kShortRun, k) || same(r + kShortRun, k);
    if (!longer) {
        while (same(s - 1, k)) --s;
        while (same(e, k)) ++e;
        longer = e - s > kShortRun;
    }
    const unsigned long long full = w.keyA[v];
    if (!longer) {
        int before = 0;
        for (long long i = s; i < e; ++i) {
            const uint32_t u = w.valB[i];
            before += i != r && depth_less(w.keyA[u], u, full, v) ? 1 : 0;
        }
        w.valA[s + before] = v;
        return;
    }
    w.valA[r] = v;
    if (!left || w.keyA[w.valB[r - 1]] <= full) return;
    // the run's ends by bisection (the truncated keys are in order): half the
    // members of a shuffled run come here, and walking to its start they took a
    // quarter of its length squared in loads (a build of 400k near-equal depths:
    // 91.6 -> 46.8 ms, the rest in k_depth_long_runs)
    const uint32_t kt = k & kDepthKeyMask;
    auto first = [&](long long lo, long long hi, uint32_t t) {   // first rank in [lo, hi) of a key >= t, else hi
        while (lo < hi) {
            const long long mid = lo + (hi - lo) / 2;
            if ((key[mid] & kDepthKeyMask) < t)
                lo = mid + 1;
            else
                hi = mid;
        }
        return lo;
    };
    s = first(0, r, kt);
    if ((key[s] & kListed) || (atomicOr(&w.tkeyB[s], kListed) & kListed)) return;
    e = first(r + 1, M, kt + 1u);
    const unsigned long long q = atomicAdd(&w.hdr->long_runs, 1ull);
    w.tkeyA[2 * q] = (uint32_t)s;
    w.tkeyA[2 * q + 1] = (uint32_t)(e - s);
}

// Batcher's odd-even merge network over P = 2^m slots: every comparator puts
// the smaller element at the lower slot, so slots past the run length L act
// as +infinity and are never touched. Stage (p, k) compares slot a with
// a + k when a >= k mod p, (a - k mod p) mod 2k < k and a, a + k lie in the
// same block of 2p slots.
__device__ __forceinline__ bool oem_pair(long long a, long long p, long long k)
{
    const long long j0 = k % p;
    return a >= j0 && ((a - j0) % (2 * k)) < k && (a / (2 * p)) == ((a + k) / (2 * p));
}

// Runs longer than kShortRun: one CTA per run (grid-stride over the list).
__global__ void __launch_bounds__(kLongRunThreads) k_depth_long_runs(BuildWs w)
{
    pdl_wait();
    pdl_trigger();
    __shared__ unsigned long long sk[kSmemRun];
    __shared__ uint32_t sv[kSmemRun];
    const unsigned long long nr = w.hdr->long_runs;
    for (unsigned long long q = blockIdx.x; q < nr; q += gridDim.x) {
        const long long r = w.tkeyA[2 * q];
        const long long L = w.tkeyA[2 * q + 1];
        long long P = 1;
        while (P < L) P <<= 1;
        if (P <= kSmemRun) {
            for (long long i = threadIdx.x; i < L; i += blockDim.x) {
                const uint32_t v = w.valA[r + i];
                sv[i] = v;
                sk[i] = w.keyA[v];
            }
            __syncthreads();
            for (long long p = 1; p < P; p <<= 1)
                for (long long k = p; k >= 1; k >>= 1) {
                    for (long long a = threadIdx.x; a + k < L; a += blockDim.x) {
                        if (!oem_pair(a, p, k)) continue;
                        const long long b = a + k;
                        if (depth_less(sk[b], sv[b], sk[a], sv[a])) {
                            const unsigned long long tk = sk[a];
                            const uint32_t tv = sv[a];
                            sk[a] = sk[b], sv[a] = sv[b];
                            sk[b] = tk, sv[b] = tv;
                        }
                    }
                    __syncthreads();
                }
            for (long long i = threadIdx.x; i < L; i += blockDim.x) w.valA[r + i] = sv[i];
            __syncthreads();
        } else {
            unsigned long long* gk = w.keyB + r;
            uint32_t* gv = w.valA + r;
            for (long long i = threadIdx.x; i < L; i += blockDim.x) gk[i] = w.keyA[gv[i]];
            __syncthreads();
            for (long long p = 1; p < P; p <<= 1)
                for (long long k = p; k >= 1; k >>= 1) {
                    for (long long a = threadIdx.x; a + k < L; a += blockDim.x) {
                        if (!oem_pair(a, p, k)) continue;
                        const long long b = a + k;
                        if (depth_less(gk[b], gv[b], gk[a], gv[a])) {
                            const unsigned long long tk = gk[a];
                            const uint32_t tv = gv[a];
                            gk[a] = gk[b], gv[a] = gv[b];
                            gk[b] = tk, gv[b] = tv;
                        }
                    }
                    __syncthreads();
                }
        }
    }
}

template <int KPT, bool FIRST>
void sweep_kpt_launch(const void* kin, const uint32_t* vin, uint32_t* kout, uint32_t* vout, const SweepArgs& a,
                      long long blocks, cudaStream_t s)
{
    cudaFuncSetAttribute(k_sweep<KPT, FIRST>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(SweepSmem<KPT>));
    launch_pdl(k_sweep<KPT, FIRST>, dim3((unsigned)blocks), dim3(kSweepThreads), sizeof(SweepSmem<KPT>), s, kin, vin, kout,
               vout, a);
    note_launches(1);
}

template <bool FIRST>
void sweep(int kpt, const void* kin, const uint32_t* vin, uint32_t* kout, uint32_t* vout, const SweepArgs& a,
           long long blocks, cudaStream_t s)
{
    if (kpt == 4)
        sweep_kpt_launch<4, FIRST>(kin, vin, kout, vout, a, blocks, s);
    else
        sweep_kpt_launch<8, FIRST>(kin, vin, kout, vout, a, blocks, s);
}

}  // namespace

int sweep_kpt(long long n)
{
    return n <= 152ll * kSweepThreads * 4 ? 4 : 8;
}

void sort_depth_keys(const BuildWs& ws, long long n, cudaStream_t s)
{
    if (n <= 0) return;
    const long long per = kSweepThreads * kHistKeys;
    launch_pdl(k_depth_hist, dim3((unsigned)((n + per - 1) / per)), dim3(kSweepThreads), 0, s, ws, n);
    // the passes end in tkeyB / valB
    uint32_t* kb[2] = {ws.tkeyB, ws.tkeyA};
    uint32_t* vb[2] = {ws.valB, ws.valA};
    for (int pass = 0; pass < kDepthPasses; ++pass) {
        SweepArgs a;
        a.hdr = ws.hdr;
        a.n_static = n;
        a.n_dev = pass == 0 ? nullptr : &ws.hdr->M;
        a.shift = pass * kBits;
        a.pass = pass;
        a.look_tries = ws.look_tries;
        a.tot = ws.dhist + pass * kDigits;
        a.stat = ws.sstat + (size_t)pass * ws.nb_depth * kDigits;
        const int in = (pass + 1) & 1, out = pass & 1;
        if (pass == 0)
            sweep<true>(ws.kpt_depth, ws.keyA, nullptr, kb[out], vb[out], a, ws.nb_depth, s);
        else
            sweep<false>(ws.kpt_depth, kb[in], vb[in], kb[out], vb[out], a, ws.nb_depth, s);
    }
    launch_pdl(k_depth_runs, dim3((unsigned)((n + 255) / 256)), dim3(256), 0, s, ws);
    launch_pdl(k_depth_long_runs, dim3(kLongRunCtas), dim3(kLongRunThreads), 0, s, ws);
    note_launches(3);
}

int tile_sort_passes(int tile_bits) { return (tile_bits + kBits - 1) / kBits; }

void sort_tile_keys(const BuildWs& ws, long long cap, int tile_bits, cudaStream_t s, uint32_t** keys_out,
                    uint32_t** vals_out)
{
    uint32_t* kb[2] = {ws.tkeyA, ws.tkeyB};
    uint32_t* vb[2] = {ws.entA, ws.entB};
    int cur = 0;
    for (int pass = 0; cap > 0 && pass < tile_sort_passes(tile_bits); ++pass) {
        SweepArgs a;
        a.hdr = ws.hdr;
        a.n_static = cap;
        a.n_dev = &ws.hdr->tile_n;
        a.shift = pass * kBits;
        a.pass = kDepthPasses + pass;
        a.look_tries = ws.look_tries;
        a.tot = ws.dhist + (kDepthPasses + pass) * kDigits;
        a.stat = ws.sstat + ((size_t)kDepthPasses * ws.nb_depth + (size_t)pass * ws.nb_tile) * kDigits;
        sweep<false>(ws.kpt_tile, kb[cur], vb[cur], kb[cur ^ 1], vb[cur ^ 1], a, ws.nb_tile, s);
        cur ^= 1;
    }
    *keys_out = kb[cur];
    *vals_out = vb[cur];
}

}  // namespace lf
