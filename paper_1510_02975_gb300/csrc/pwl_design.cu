// pwl_design.cu -- knot placement for the nearly optimal partition T*
// (Section III-B): the local knot density |f''|^{2/5} (Eq. 16) on M uniform
// cells, its FP64 cumulative sum (the numerator of Eq. 18 by the midpoint
// rule) and the inversion F(x_i) = i/N (Eq. 17).
//
// Every kernel is batched over F functions described by device arrays
// (descriptors and CSR offsets of knots, cells and 256-cell chunks, the
// chunks of a function padded to whole tiles of 8); a single function is a
// batch of one.  Three launches:
//   densities       d_k = |f''(t_k)|^{2/5} and one partial sum per chunk, or per
//                   tile (FP32 mode of a batch, and of one function of many cells)
//   scan            exclusive FP64 scan of the partial sums, per function
//   knots           per tile of 2048 cells: the in-tile prefix of the
//                   densities and the knots whose targets tau_i = i G_M / N
//                   fall into the tile
// No CTA waits for another tile of its function: a batch designed by one CTA
// per function waits for its largest function and for the barriers of every
// tile in turn.  40 functions of up to 4095 intervals at 64 cells per
// interval, FP64: 25.2 ms that way (which also computed the densities twice),
// 0.82 ms this way (density 0.755).
#include <math.h>

#include <algorithm>

#include "pwl_design.cuh"

namespace pwl {

namespace {

constexpr int kDesignThreads = 256;
constexpr int kChunk = kDesignThreads;         // density cells per chunk
constexpr int kTileChunks = 8;                 // chunks per tile (every function holds whole tiles)
constexpr int kTile = kChunk * kTileChunks;    // cells per tile
constexpr int kTilePer = kTile / kDesignThreads;  // cells per thread of a tile

__device__ __forceinline__ double warp_sum(double v)
{
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

// Block-wide exclusive scan of one double per thread (kDesignThreads
// threads).  Returns the exclusive prefix; *total receives the block sum.
__device__ __forceinline__ double block_exclusive_scan(double v, double* s_warp, double* total)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    constexpr int W = kDesignThreads / 32;
    double incl = v;
    for (int o = 1; o < 32; o <<= 1) {
        double t = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += t;
    }
    double excl = __shfl_up_sync(0xffffffffu, incl, 1);
    if (lane == 0) excl = 0.0;
    if (lane == 31) s_warp[warp] = incl;
    __syncthreads();
    if (warp == 0) {
        double ws = (lane < W) ? s_warp[lane] : 0.0;
        double wi = ws;
        for (int o = 1; o < 32; o <<= 1) {
            double t = __shfl_up_sync(0xffffffffu, wi, o);
            if (lane >= o) wi += t;
        }
        double we = __shfl_up_sync(0xffffffffu, wi, 1);
        if (lane == 0) we = 0.0;
        if (lane < W) s_warp[lane] = we;
        if (lane == W - 1) s_warp[W] = wi;
    }
    __syncthreads();
    double r = s_warp[warp] + excl;
    *total = s_warp[W];
    __syncthreads();
    return r;
}

// Density of one cell: d_k = |f''(t_k)|^{2/5}, f'' and the power in T
template <typename T, bool SAMPLED>
__device__ __forceinline__ double cell_density(const pwl_func& F, double delta, int64_t k)
{
    // t_k = a + (k + 1/2) delta, rounded as written (no fused multiply-add)
    const double t = __dadd_rn(F.a, __dmul_rn((double)k + 0.5, delta));
    return (double)FMath<T>::dens(func_second_derivative_k<SAMPLED, T>(F, (T)t));
}

// One CTA per chunk, one cell per thread: d_k, the chunk's FP64 sum and its
// last cell of positive density.  The kernel is bound by the FP64 pipe (about
// one lane-operation per SM and clock, which 8 warps keep busy), so a chunk is
// as small as a 256-thread CTA: one N = 1024 design (65536 cells) then fills
// 256 CTAs, where 2048-cell chunks left it on 32 of the 152 SMs (J0, from f to
// a table and 2^20 evaluations: 493 -> 416 us).
template <typename T, bool SAMPLED>
__global__ void __launch_bounds__(kDesignThreads, 2) density_chunks_kernel(DesignPlan p)
{
    __shared__ double s_red[kDesignThreads / 32];
    __shared__ int s_last[kDesignThreads / 32];
    for (int64_t ch = blockIdx.x; ch < p.total_chunks; ch += gridDim.x) {
        const int f = p.tile_func ? p.tile_func[ch / kTileChunks] : 0;
        const pwl_func F = p.funcs[f];
        if ((F.kind == PWL_F_SAMPLED) != SAMPLED) continue;  // the other launch's (uniform per CTA)
        const int64_t M = p.moff[f + 1] - p.moff[f];
        const int64_t k = (ch - p.choff[f]) * kChunk + threadIdx.x;
        const double delta = p.delta[f];  // (a division here is a tenth of a Gaussian density's FP64 operations)
        double acc = 0.0;
        if (k < M) {
            acc = cell_density<T, SAMPLED>(F, delta, k);
            p.d[p.moff[f] + k] = acc;
        }
        const unsigned pos = __ballot_sync(0xffffffffu, acc > 0.0);
        acc = warp_sum(acc);
        if ((threadIdx.x & 31) == 0) {
            s_red[threadIdx.x >> 5] = acc;
            s_last[threadIdx.x >> 5] = pos ? (int)threadIdx.x + 31 - __clz(pos) : -1;
        }
        __syncthreads();
        if (threadIdx.x == 0) {
            double sum = 0.0;
            int last = -1;
            for (int w = 0; w < kDesignThreads / 32; ++w) {
                sum += s_red[w];
                last = max(last, s_last[w]);
            }
            p.csum[ch] = sum;
            p.plast[ch] = last < 0 ? -1 : k + last;  // k: the chunk's first cell (thread 0)
        }
        __syncthreads();
    }
}

// The same by whole tiles, one function, 8 cells per thread: one partial per tile (in
// its first chunk; the others' are 0).  A chunk's sum takes 5 additions per lane, which
// FP64 densities hardly notice but FP32 ones do, and so they do the parameters'
// conversions in every cell: a whole FP32 design on 2^24 cells 614 us, by chunks 855.
// For tiles enough to fill the chip.
template <typename T, bool SAMPLED>
__global__ void __launch_bounds__(kDesignThreads) density_tiles_kernel(DesignPlan p)
{
    __shared__ double s_red[kDesignThreads / 32];
    __shared__ int s_last[kDesignThreads / 32];
    const pwl_func F = p.funcs[0];
    const double delta = p.delta[0];
    const int64_t M = p.moff[1];
    const int t = threadIdx.x;
    for (int64_t tile = blockIdx.x; tile < p.total_chunks / kTileChunks; tile += gridDim.x) {
        const int64_t c0 = tile * kTile, ch = tile * kTileChunks;
        double acc = 0.0;
        int last = -1;
#pragma unroll 2
        for (int r = 0; r < kTilePer; ++r) {
            const int64_t k = c0 + r * kDesignThreads + t;
            if (k >= M) break;
            const double v = cell_density<T, SAMPLED>(F, delta, k);
            p.d[k] = v;
            acc += v;
            if (v > 0.0) last = r * kDesignThreads + t;
        }
        acc = warp_sum(acc);
        last = __reduce_max_sync(0xffffffffu, last);
        if ((t & 31) == 0) {
            s_red[t >> 5] = acc;
            s_last[t >> 5] = last;
        }
        __syncthreads();
        if (t < kTileChunks) {
            double sum = 0.0;
            int m = -1;
            for (int w = 0; w < kDesignThreads / 32; ++w) {
                sum += s_red[w];
                m = max(m, s_last[w]);
            }
            p.csum[ch + t] = t == 0 ? sum : 0.0;
            p.plast[ch + t] = t > 0 || m < 0 ? -1 : c0 + m;
        }
        __syncthreads();
    }
}

// smallest i in [1, N] with tau_i = i G_M / N >= G (N if none below N)
__device__ __forceinline__ int64_t first_target_at_or_above(double G, double GM, int64_t N)
{
    auto tau = [&](int64_t i) { return (double)i * GM / (double)N; };
    const double e = floor(G / GM * (double)N);
    int64_t i = (int64_t)fmin(fmax(e, 1.0), (double)N);
    while (i > 1 && tau(i - 1) >= G) --i;
    while (i < N && tau(i) < G) ++i;
    return i;
}

// Per function: the exclusive FP64 scan of the chunk sums (cbase), the last
// cell of positive density before every chunk (plast, in place), G_M (stot),
// and every tile's first target (in its first chunk's csum, which is spent by
// then): one lane per tile, where two lanes of every tile's CTA held the FP64
// pipe for as long as whole warps would.
// kScanPer consecutive chunks per thread, 2048 chunks a round.
constexpr int kScanPer = 8;

__global__ void __launch_bounds__(kDesignThreads) chunk_scan_kernel(DesignPlan p)
{
    __shared__ double s_warp[kDesignThreads / 32 + 1];
    __shared__ long long s_max[kDesignThreads / 32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    for (int f = blockIdx.x; f < p.F; f += gridDim.x) {
        const int64_t c0 = p.choff[f], c1 = p.choff[f + 1];
        double carry = 0.0;
        long long before = -1;  // last positive cell of the rounds before
        for (int64_t base = c0; base < c1; base += kDesignThreads * kScanPer) {
            const int64_t c = base + (int64_t)threadIdx.x * kScanPer;
            double v[kScanPer], run = 0.0;
            long long l[kScanPer], mine = -1;
#pragma unroll
            for (int r = 0; r < kScanPer; ++r) {
                v[r] = c + r < c1 ? p.csum[c + r] : 0.0;
                l[r] = c + r < c1 ? p.plast[c + r] : -1;
                run += v[r];
                mine = max(mine, l[r]);
            }
            double tot;
            double ex = carry + block_exclusive_scan(run, s_warp, &tot);
            long long incl = mine;
            for (int o = 1; o < 32; o <<= 1) {
                const long long t = __shfl_up_sync(0xffffffffu, incl, o);
                if (lane >= o) incl = max(incl, t);
            }
            if (lane == 31) s_max[warp] = incl;
            __syncthreads();
            long long prev = __shfl_up_sync(0xffffffffu, incl, 1);
            prev = max(lane == 0 ? -1ll : prev, before);
            for (int w = 0; w < kDesignThreads / 32; ++w) {
                if (w < warp) prev = max(prev, s_max[w]);
                before = max(before, s_max[w]);
            }
#pragma unroll
            for (int r = 0; r < kScanPer; ++r) {
                if (c + r < c1) {
                    p.cbase[c + r] = ex;
                    p.plast[c + r] = prev;
                }
                ex += v[r];
                prev = max(prev, l[r]);
            }
            carry += tot;
            __syncthreads();  // s_max is rewritten in the next round
        }
        const int64_t N = p.koff[f + 1] - p.koff[f] - 1;
        const double delta = p.delta[f], GM = delta * carry;
        if (threadIdx.x == 0) p.stot[f] = GM;
        __syncthreads();  // cbase complete, csum read
        for (int64_t ch = c0 + (int64_t)threadIdx.x * kTileChunks; ch < c1; ch += kDesignThreads * kTileChunks)
            reinterpret_cast<int64_t*>(p.csum)[ch] = GM > 0.0 ? first_target_at_or_above(delta * p.cbase[ch], GM, N) : 1;
    }
}

// The knots whose targets fall into a tile of kTileChunks chunks (tau_i at or
// above G at the tile's start and below G at the next tile's): the tile's
// densities and the FP64 prefix of its thread partials in shared memory,
// then per knot the largest cell k with G_k <= tau_i (binary search over the
// thread prefixes, then the thread's cells), the walk back to a cell of
// positive density, and x_i = a + k delta + (tau_i - G_k) / d_k.  It reads 8
// bytes per cell; writing G to memory and searching it there took 24 bytes
// per cell and a chain of ~17 dependent L2 reads per knot.
//
// Targets can crowd (few cells per knot, or a peak that a fraction of the cells
// holds), so a tile's knots go to `slices` CTAs, 256 at a time in turn; slices
// without a knot are passed over, 256 at a time, without reading their tile.
// 2^20 intervals on 2048 cells 0.18 ms (18.1 with one CTA per tile), 100000 with a
// peak of 1e-4 of the domain 0.76 ms (2.31).
struct TileItem {
    int64_t tile, i0, i1;  // the tile and its knots (i0 <= i < i1)
    int f, slice;
    __device__ __forceinline__ TileItem(const DesignPlan& p, int64_t item)
    {
        const int64_t tiles = p.total_chunks / kTileChunks, ch = (tile = item % tiles) * kTileChunks;
        slice = (int)(item / tiles);
        f = p.tile_func ? p.tile_func[tile] : 0;
        const int64_t c0 = (ch - p.choff[f]) * kChunk, N = p.koff[f + 1] - p.koff[f] - 1;
        if (p.stot[f] > 0.0) {
            // the next tile's first target ends this one's, so every knot has exactly one tile
            const int64_t* first = reinterpret_cast<const int64_t*>(p.csum + ch);
            i0 = first[0];
            i1 = c0 + kTile < p.moff[f + 1] - p.moff[f] ? first[kTileChunks] : N;
        } else {  // f linear on I (or no finite density): the uniform partition, by the first tile
            i0 = 1;
            i1 = c0 == 0 ? N : 1;
        }
    }
    // whether the item has anything to write (the first one of a function the end knots)
    __device__ __forceinline__ bool any(const DesignPlan& p) const
    {
        return i0 + slice * kDesignThreads < i1 || (slice == 0 && tile * kTileChunks == p.choff[f]);
    }
};

__global__ void __launch_bounds__(kDesignThreads) invert_tiles_kernel(DesignPlan p, int slices)
{
    __shared__ double s_d[kTile];
    __shared__ double s_S[kDesignThreads];  // tile base + exclusive prefix of the thread partials
    __shared__ double s_warp[kDesignThreads / 32 + 1];
    __shared__ int s_items[kDesignThreads];
    __shared__ int s_count;
    const int t = threadIdx.x;
    const int64_t items = p.total_chunks / kTileChunks * slices, step = (int64_t)gridDim.x * kDesignThreads;
    for (int64_t base_item = blockIdx.x; base_item < items; base_item += step) {
        const bool list = items > gridDim.x;  // (else one item per CTA)
        if (list) {
            if (t == 0) s_count = 0;
            __syncthreads();
            const int64_t mine = base_item + (int64_t)t * gridDim.x;
            if (mine < items && TileItem(p, mine).any(p)) s_items[atomicAdd(&s_count, 1)] = t;
            __syncthreads();
        }
        for (int n = 0; n < (list ? s_count : 1); ++n) {
            const TileItem it(p, list ? base_item + (int64_t)s_items[n] * gridDim.x : base_item);
            if (!list && !it.any(p)) continue;
            const int64_t ch = it.tile * kTileChunks;  // the tile's first chunk
            const int f = it.f;
            const int64_t M = p.moff[f + 1] - p.moff[f];
            const int64_t N = p.koff[f + 1] - p.koff[f] - 1;
            const int64_t c0 = (ch - p.choff[f]) * kChunk;
            const int64_t i_first = it.i0 + it.slice * kDesignThreads + t, i_step = (int64_t)slices * kDesignThreads;
            const double a = p.funcs[f].a, b = p.funcs[f].b;
            const double delta = p.delta[f];
            const double GM = p.stot[f];
            double* __restrict__ knots = p.knots + p.koff[f];
            if (t == 0 && c0 == 0 && it.slice == 0) {
                knots[0] = a;
                knots[N] = b;
            }
            if (!(GM > 0.0)) {
                for (int64_t i = i_first; i < it.i1; i += i_step) knots[i] = a + (double)i * (b - a) / (double)N;
                continue;
            }
            const double base = p.cbase[ch];
            if (it.i0 >= it.i1) continue;  // (only the end knots)
            const int cnt = (int)min((int64_t)kTile, M - c0);
            const double* __restrict__ d = p.d + p.moff[f] + c0;
            for (int i = t; i < kTile; i += kDesignThreads) s_d[i] = i < cnt ? d[i] : 0.0;
            __syncthreads();
            double run = 0.0;
            for (int r = 0; r < kTilePer; ++r) run += s_d[t * kTilePer + r];
            double tot;
            s_S[t] = base + block_exclusive_scan(run, s_warp, &tot);
            __syncthreads();
            const int U = (cnt + kTilePer - 1) / kTilePer;  // threads holding cells
            for (int64_t i = i_first; i < it.i1; i += i_step) {
                const double tau = (double)i * GM / (double)N;
                int lo = 0, hi = U - 1;  // largest u with G at its first cell <= tau (u = 0 is)
                while (lo < hi) {
                    const int mid = (lo + hi + 1) >> 1;
                    if (delta * s_S[mid] <= tau) lo = mid; else hi = mid - 1;
                }
                const int nr = min(kTilePer, cnt - lo * kTilePer);
                double acc = 0.0, Gk = delta * s_S[lo];
                int kl = lo * kTilePer;
                for (int r = 1; r < nr; ++r) {  // the thread's last cell with G <= tau (G does not decrease)
                    acc += s_d[lo * kTilePer + r - 1];
                    const double Gr = delta * (s_S[lo] + acc);
                    if (!(Gr <= tau)) break;
                    kl = lo * kTilePer + r;
                    Gk = Gr;
                }
                int kk = kl;  // largest cell <= kl of positive density
                while (kk >= 0 && !(s_d[kk] > 0.0)) --kk;
                double x;
                if (kk == kl) {
                    x = __dadd_rn(a, __dmul_rn((double)(c0 + kk), delta));
                    x = __dadd_rn(x, fmin(fmax((tau - Gk) / s_d[kk], 0.0), delta));
                } else {
                    // no density between the last positive cell (in the tile or before
                    // it) and here, so tau is at or past G at that cell's end: its
                    // right edge
                    const int64_t e = kk >= 0 ? c0 + kk : p.plast[ch];
                    x = e < 0 ? a : __dadd_rn(__dadd_rn(a, __dmul_rn((double)e, delta)), delta);
                }
                knots[i] = x;
            }
            __syncthreads();  // the shared arrays are rewritten for the next tile
        }
        __syncthreads();  // (nobody reads the list any more)
    }
}

// FP32 density from the function's FP32 constants: |f''|^{2/5} by the
// hardware exp2/log2 pair (__powf), a few ulp (the FP32 mode's knot bound
// allows a relative density error near 1e-6), for a third of the
// instructions of powf
template <bool SAMPLED>
__device__ __forceinline__ float fused_density_f(const FuncF& G, const pwl_func& F, float t0f, float deltaf,
                                                 int local)
{
    const float t = __fmaf_rn((float)local + 0.5f, deltaf, t0f);
    float f2;
    if constexpr (SAMPLED) f2 = (float)sampled_second_derivative(F, (double)t);
    else f2 = func_second_derivative_f(G, t);
    return __powf(fabsf(f2), 0.4f);
}

// ---- FP32 mode of a batch -----------------------------------------------------
// The same three launches with almost no FP64 operation per density cell
// (GB300 runs about one FP64 operation per SM and cycle):
//   - what needs FP64 once per function or tile (constants, cell width, tile
//     start, the first target of every tile) comes from launches with one
//     thread per tile: an FP64 instruction occupies the pipe for the whole warp
//     however few of its lanes run it, and done by one lane, or by every thread,
//     of each tile's CTA these took most of the time (design of 4096 functions
//     1.79 ms, 1.25 ms by one CTA per function, 0.94 ms now; 40 functions
//     209 -> 36 us);
//   - the densities go to scratch and come back in 16-byte vectors; cell
//     midpoints are formed in FP32 from the tile start (the FP32 f'' rounds its
//     argument to FP32 anyway);
//   - sums inside a tile are float-float (a compensated pair hi + lo, about
//     48 significant bits): thread partials, the block scan and the tile
//     total; the tile totals, their scan and G_M are FP64;
//   - the knot search compares float-float values in FP32, in units of the
//     density sum (G / delta): the target tau_i / delta = i G_M / (N delta)
//     minus the tile base is formed in FP64 once per knot and split into a
//     float-float pair;
//   - the step inside the cell, (tau_i - G_k) / d_k, is FP32 (it is at most
//     delta, so its rounding is below 1e-7 delta), and x = a + k delta + step
//     is FP64.
struct FF {
    float hi, lo;
};
__device__ __forceinline__ FF ff_add(FF x, FF y)
{
    const float s = __fadd_rn(x.hi, y.hi);
    const float bp = __fsub_rn(s, x.hi);
    const float e = __fadd_rn(__fsub_rn(x.hi, __fsub_rn(s, bp)), __fsub_rn(y.hi, bp));
    const float t = __fadd_rn(e, __fadd_rn(x.lo, y.lo));
    const float hi = __fadd_rn(s, t);
    return FF{hi, __fsub_rn(t, __fsub_rn(hi, s))};
}
// x + v without the renormalisation: lo gathers the rounding errors of a few
// additions (each below 2^-24 hi, so its own rounding is below 2^-47 hi);
// ff_norm brings the pair back into rounded form.  7 operations instead of 11 for
// each cell of a thread's partial sum (both tile kernels are bound by issue): 4096
// functions, densities 521 -> 509 us, knots 414 -> 398 us with a barrier less.
__device__ __forceinline__ FF ff_acc(FF x, float v)
{
    const float s = __fadd_rn(x.hi, v);
    const float bp = __fsub_rn(s, x.hi);
    const float e = __fadd_rn(__fsub_rn(x.hi, __fsub_rn(s, bp)), __fsub_rn(v, bp));
    return FF{s, __fadd_rn(x.lo, e)};
}
__device__ __forceinline__ FF ff_norm(FF x)
{
    const float hi = __fadd_rn(x.hi, x.lo);
    return FF{hi, __fsub_rn(x.lo, __fsub_rn(hi, x.hi))};
}
__device__ __forceinline__ FF ff_neg(FF x) { return FF{-x.hi, -x.lo}; }
__device__ __forceinline__ bool ff_le(FF x, FF y) { return x.hi < y.hi || (x.hi == y.hi && x.lo <= y.lo); }
__device__ __forceinline__ FF ff_from_double(double v)
{
    const float hi = __double2float_rn(v);
    return FF{hi, __double2float_rn(v - (double)hi)};
}
// The same pair without FP64 operations, for v of normal FP32 magnitude (else by
// the conversions): the top 24 significant bits, the 29 below them, and a
// compensated sum that brings them into rounded form.
__device__ __forceinline__ FF ff_from_double_bits(double v)
{
    const uint32_t h = (uint32_t)__double2hiint(v), l = (uint32_t)__double2loint(v);
    const uint32_t e = h >> 20 & 0x7ffu;
    if (e < 1023 - 60 || e > 1023 + 120) return ff_from_double(v);
    // (sign, exponent, upper 23 mantissa bits) as FP32; the lower 29 bits are
    // worth l' 2^(e - 52), exact in FP32 but for the last few
    const uint32_t top = (h & 0x80000000u) | (e - 896) << 23 | (h << 3 & 0x7ffff8u) | l >> 29;
    const float hi = __uint_as_float(top);
    const float ulp = __uint_as_float((h & 0x80000000u) | (e - 896 - 52) << 23);  // +-2^(e - 52)
    const float lo = __uint2float_rn(l & 0x1fffffffu) * ulp;
    const float s = __fadd_rn(hi, lo);
    return FF{s, __fsub_rn(lo, __fsub_rn(s, hi))};
}
__device__ __forceinline__ double ff_to_double(FF x) { return (double)x.hi + (double)x.lo; }

// Block-wide exclusive scan of one float-float per thread (kDesignThreads).  The
// caller has a barrier between its return and the next use of s_w.
__device__ __forceinline__ FF ff_block_exclusive_scan(FF v, FF* s_w)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    constexpr int W = kDesignThreads / 32;
    FF incl = v;
    for (int o = 1; o < 32; o <<= 1) {
        const FF n{__shfl_up_sync(0xffffffffu, incl.hi, o), __shfl_up_sync(0xffffffffu, incl.lo, o)};
        if (lane >= o) incl = ff_add(n, incl);
    }
    FF excl{__shfl_up_sync(0xffffffffu, incl.hi, 1), __shfl_up_sync(0xffffffffu, incl.lo, 1)};
    if (lane == 0) excl = FF{0.0f, 0.0f};
    if (lane == 31) s_w[warp] = incl;
    __syncthreads();
    if (warp == 0) {
        FF ws = lane < W ? s_w[lane] : FF{0.0f, 0.0f};
        FF wi = ws;
        for (int o = 1; o < W; o <<= 1) {
            const FF n{__shfl_up_sync(0xffffffffu, wi.hi, o), __shfl_up_sync(0xffffffffu, wi.lo, o)};
            if (lane >= o) wi = ff_add(n, wi);
        }
        FF we{__shfl_up_sync(0xffffffffu, wi.hi, 1), __shfl_up_sync(0xffffffffu, wi.lo, 1)};
        if (lane == 0) we = FF{0.0f, 0.0f};
        if (lane < W) s_w[lane] = we;
    }
    __syncthreads();
    return ff_add(s_w[warp], excl);
}

// smallest i in [1, N] with i c >= S (N if none below N), c = G_M / (N delta)
__device__ __forceinline__ int64_t first_target_at_or_above_units(double S, double c, int64_t N)
{
    const double e = floor(S / c);
    int64_t i = (int64_t)fmin(fmax(e, 1.0), (double)N);
    while (i > 1 && (double)(i - 1) * c >= S) --i;
    while (i < N && (double)i * c < S) ++i;
    return i;
}

// One thread per tile: the tile's start in FP32 (in its first chunk's cbase,
// which the scan overwrites), and each function's constants.
__global__ void __launch_bounds__(128) tile_setup_f_kernel(DesignPlan p)
{
    const int64_t tile = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (tile >= p.total_chunks / kTileChunks) return;
    const int f = p.tile_func[tile];
    const int64_t ch = tile * kTileChunks, c0 = (ch - p.choff[f]) * kChunk;
    const double a = p.funcs[f].a, delta = p.delta[f];
    *reinterpret_cast<float*>(p.cbase + ch) = (float)(a + (double)c0 * delta);
    if (c0 == 0) {
        const pwl_func F = p.funcs[f];
        DesignFunc d{};
        d.g = make_funcf(F);
        d.deltaf = (float)delta;
        d.a = a;
        d.delta = delta;
        p.ffuncs[f] = d;
    }
}

// One warp per function: the exclusive FP64 scan of the tile sums (cbase), the
// last cell of positive density before every tile (plast, in place), and, from
// the total, cunit = G_M / (N delta) (0: the uniform partition) and every
// tile's first target (smallest i in [1, N] with i cunit >= the tile's base, N
// if none; in its first chunk's csum, which is spent by then).
__global__ void __launch_bounds__(128) tile_scan_f_kernel(DesignPlan p)
{
    const int lane = threadIdx.x & 31;
    for (int f = blockIdx.x * 4 + (threadIdx.x >> 5); f < p.F; f += gridDim.x * 4) {
        const int64_t c0 = p.choff[f], tiles = (p.choff[f + 1] - c0) / kTileChunks;
        const int64_t N = p.koff[f + 1] - p.koff[f] - 1;
        double carry = 0.0;
        long long before = -1;
        for (int64_t base = 0; base < tiles; base += 32) {
            const int64_t ch = c0 + (base + lane) * kTileChunks;
            const bool in = base + lane < tiles;
            double incl = in ? p.csum[ch] : 0.0;
            long long last = in ? p.plast[ch] : -1;
            for (int o = 1; o < 32; o <<= 1) {
                const double v = __shfl_up_sync(0xffffffffu, incl, o);
                const long long l = __shfl_up_sync(0xffffffffu, last, o);
                if (lane >= o) {
                    incl += v;
                    last = max(last, l);
                }
            }
            double ex = __shfl_up_sync(0xffffffffu, incl, 1);
            long long prev = __shfl_up_sync(0xffffffffu, last, 1);
            if (lane == 0) {
                ex = 0.0;
                prev = -1;
            }
            if (in) {
                p.cbase[ch] = carry + ex;
                p.plast[ch] = max(prev, before);
            }
            carry += __shfl_sync(0xffffffffu, incl, 31);
            before = max(before, __shfl_sync(0xffffffffu, last, 31));
        }
        const double cunit = carry / (double)N;
        const bool linear = !(p.ffuncs[f].delta * carry > 0.0);  // f linear on I, or no finite density
        for (int64_t tile = lane; tile < tiles; tile += 32) {
            const int64_t ch = c0 + tile * kTileChunks;
            reinterpret_cast<int64_t*>(p.csum)[ch] =
                linear ? 1 : first_target_at_or_above_units(p.cbase[ch], cunit, N);
        }
        if (lane == 0) p.ffuncs[f].cunit = linear ? 0.0 : cunit;
    }
}

// FP32 densities of function f from its cell c0 on: every function starts
// 16-byte aligned, with room for the last vector's padding (float index
// moff + 4 f rounded down to a multiple of 4)
__device__ __forceinline__ float* tile_densities(const DesignPlan& p, int f, int64_t c0)
{
    return reinterpret_cast<float*>(p.d) + (p.moff[f] + 4 * (int64_t)f) / 4 * 4 + c0;
}

template <bool SAMPLED>
__global__ void __launch_bounds__(kDesignThreads, SAMPLED ? 4 : 8) density_tiles_f_kernel(DesignPlan p)
{
    __shared__ FF s_w[kDesignThreads / 32];
    __shared__ int s_last[kDesignThreads / 32];
    const int t = threadIdx.x;
    for (int64_t tile = blockIdx.x; tile < p.total_chunks / kTileChunks; tile += gridDim.x) {
        const int f = p.tile_func[tile];
        const DesignFunc& D = p.ffuncs[f];
        if ((D.g.kind == PWL_F_SAMPLED) != SAMPLED) continue;  // the other launch's (uniform per CTA)
        const int64_t ch = tile * kTileChunks, c0 = (ch - p.choff[f]) * kChunk, M = p.moff[f + 1] - p.moff[f];
        const FuncF G = D.g;
        const float deltaf = D.deltaf, t0f = *reinterpret_cast<const float*>(p.cbase + ch);
        const int cnt = (int)min((int64_t)kTile, M - c0);
        FF part{0.0f, 0.0f};
        int last = -1;
        float* __restrict__ out = tile_densities(p, f, c0);
        // cells strided over the threads, one copy of the loop's body (unrolled,
        // the Bessel functions overflow the instruction cache)
#pragma unroll 1
        for (int l = t; l < cnt; l += kDesignThreads) {
            float v;
            if constexpr (SAMPLED) v = fused_density_f<true>(G, p.funcs[f], t0f, deltaf, l);
            else v = fused_density_f<false>(G, pwl_func{}, t0f, deltaf, l);
            out[l] = v;
            part = ff_acc(part, v);
            if (v > 0.0f) last = l;
        }
        part = ff_norm(part);
        for (int o = 16; o > 0; o >>= 1)
            part = ff_add(part, FF{__shfl_down_sync(0xffffffffu, part.hi, o), __shfl_down_sync(0xffffffffu, part.lo, o)});
        last = __reduce_max_sync(0xffffffffu, last);
        if ((t & 31) == 0) {
            s_w[t >> 5] = part;
            s_last[t >> 5] = last;
        }
        __syncthreads();
        if (t == 0) {  // (the first of the tile's chunks stands for the tile)
            FF r{0.0f, 0.0f};
            int m = -1;
            for (int w = 0; w < kDesignThreads / 32; ++w) {
                r = ff_add(r, s_w[w]);
                m = max(m, s_last[w]);
            }
            p.csum[ch] = ff_to_double(r);
            p.plast[ch] = m < 0 ? -1 : c0 + m;
        }
        __syncthreads();
    }
}

// 8 CTAs per SM: the kernel waits on the chain of loads that starts a tile and
// on the scan's barriers (4 CTAs per SM 586 us, 6 480 us, 8 414 us, and 398 us since
// the thread sums do without renormalising).
__global__ void __launch_bounds__(kDesignThreads, 8) invert_tiles_f_kernel(DesignPlan p)
{
    __shared__ float4 s_d4[kTile / 4];
    __shared__ FF s_ex[kDesignThreads];  // exclusive float-float prefix of the thread partials
    __shared__ FF s_w[kDesignThreads / 32];
    float* s_d = reinterpret_cast<float*>(s_d4);
    const int t = threadIdx.x;
    for (int64_t tile = blockIdx.x; tile < p.total_chunks / kTileChunks; tile += gridDim.x) {
        const int f = p.tile_func[tile];
        const int64_t ch = tile * kTileChunks, c0 = (ch - p.choff[f]) * kChunk, M = p.moff[f + 1] - p.moff[f];
        const int64_t N = p.koff[f + 1] - p.koff[f] - 1;
        const double a = p.ffuncs[f].a, delta = p.ffuncs[f].delta, cunit = p.ffuncs[f].cunit;
        double* __restrict__ knots = p.knots + p.koff[f];
        if (t == 0 && c0 == 0) {
            knots[0] = a;
            knots[N] = p.funcs[f].b;
        }
        if (cunit == 0.0) {
            if (c0 == 0) {
                const double b = p.funcs[f].b;
                for (int64_t i = 1 + t; i < N; i += kDesignThreads) knots[i] = a + (double)i * (b - a) / (double)N;
            }
            continue;
        }
        // tau_i / delta = i * cunit; the next tile's first target ends this one's
        const int64_t* first = reinterpret_cast<const int64_t*>(p.csum + ch);
        const int64_t i0 = first[0], i1 = c0 + kTile < M ? first[kTileChunks] : N;
        if (i0 >= i1) continue;
        const int cnt = (int)min((int64_t)kTile, M - c0);
        const float4* in = reinterpret_cast<const float4*>(tile_densities(p, f, c0));
        FF part{0.0f, 0.0f};
#pragma unroll
        for (int q = 0; q < kTilePer / 4; ++q) {  // zero past the function's last cell: adds nothing
            const int i = t * (kTilePer / 4) + q;
            float4 v = 4 * i < cnt ? in[i] : make_float4(0.0f, 0.0f, 0.0f, 0.0f);
            if (4 * i + 3 >= cnt) {  // the padding of the last vector is not written
                v.w = 0.0f;
                if (4 * i + 2 >= cnt) v.z = 0.0f;
                if (4 * i + 1 >= cnt) v.y = 0.0f;
            }
            s_d4[t * (kTilePer / 4) + q] = v;
            part = ff_acc(part, v.x);
            part = ff_acc(part, v.y);
            part = ff_acc(part, v.z);
            part = ff_acc(part, v.w);
        }
        s_ex[t] = ff_block_exclusive_scan(ff_norm(part), s_w);
        __syncthreads();
        {
            const int U = (cnt + kTilePer - 1) / kTilePer;
            const double cb = p.cbase[ch];
            const float deltaf = p.ffuncs[f].deltaf;
            // float-float prefix of local cell l: S_u + the thread's cells before l
            auto ff_at = [&](int l) {
                const int u = l / kTilePer;
                FF q = s_ex[u];
                for (int r = u * kTilePer; r < l; ++r) q = ff_add(q, FF{s_d[r], 0.0f});
                return q;
            };
            // (i < 2^16 and c0 < 2^28 in a batch: 32-bit conversions)
            for (int64_t i = i0 + t; i < i1; i += kDesignThreads) {
                const FF tl = ff_from_double_bits((double)(int)i * cunit - cb);  // target in the tile
                int lo = 0, hi = U - 1;  // largest u with S_u <= target (u = 0 is)
                while (lo < hi) {
                    const int mid = (lo + hi + 1) >> 1;
                    if (ff_le(s_ex[mid], tl)) lo = mid; else hi = mid - 1;
                }
                const int nr = min(kTilePer, cnt - lo * kTilePer);
                FF q = s_ex[lo], Sk = q;
                int kl = lo * kTilePer;
                for (int r = 1; r < nr; ++r) {
                    q = ff_add(q, FF{s_d[lo * kTilePer + r - 1], 0.0f});
                    if (!ff_le(q, tl)) break;
                    kl = lo * kTilePer + r;
                    Sk = q;
                }
                int kk = kl;
                while (kk >= 0 && !(s_d[kk] > 0.0f)) --kk;
                double x;
                if (kk >= 0) {
                    if (kk != kl) Sk = ff_at(kk);
                    const FF diff = ff_add(tl, ff_neg(Sk));  // (tau - G_k) / delta
                    const float step = fminf(fmaxf((diff.hi + diff.lo) * deltaf / s_d[kk], 0.0f), deltaf);
                    x = __dadd_rn(__fma_rn((double)((int)c0 + kk), delta, a), widen_bits(step));
                } else {
                    const int64_t e = p.plast[ch];
                    x = e < 0 ? a : __dadd_rn(__dadd_rn(a, __dmul_rn((double)e, delta)), delta);
                }
                knots[i] = x;
            }
        }
        __syncthreads();  // the shared arrays are rewritten for the next tile
    }
}

// Writes the descriptor and offsets of a one-function batch into the
// workspace (kernel parameters, so the call needs no host-to-device copy).
__global__ void single_setup_kernel(pwl_func F, int64_t N, int64_t M, int64_t chunks, pwl_func* funcs,
                                    int64_t* koff, int64_t* moff, int64_t* choff, double* delta)
{
    if (threadIdx.x == 0 && blockIdx.x == 0) {
        funcs[0] = F;
        delta[0] = (F.b - F.a) / (double)M;
        koff[0] = 0;
        koff[1] = N + 1;
        moff[0] = 0;
        moff[1] = M;
        choff[0] = 0;
        choff[1] = chunks;
    }
}

inline size_t align256(size_t x) { return (x + 255) & ~(size_t)255; }

}  // namespace

int64_t design_chunks(int64_t M) { return (M + kTile - 1) / kTile * kTileChunks; }

// FP64 per cell, or (FP32 mode of a batch) floats with 4 more per function
static size_t density_bytes(int64_t F, int64_t total_cells)
{
    return align256(std::max(sizeof(double) * (size_t)total_cells, sizeof(float) * (size_t)(total_cells + 4 * F + 4)));
}

size_t design_scratch_bytes(int64_t F, int64_t total_cells, int64_t total_chunks)
{
    return density_bytes(F, total_cells) + align256(sizeof(double) * (size_t)total_chunks) * 2 +
           align256(sizeof(int64_t) * (size_t)total_chunks) + align256(sizeof(double) * (size_t)F);
}

void design_carve_scratch(DesignPlan& p, void* scratch)
{
    char* w = static_cast<char*>(scratch);
    p.d = reinterpret_cast<double*>(w);
    w += density_bytes(p.F, p.total_cells);
    p.csum = reinterpret_cast<double*>(w);
    w += align256(sizeof(double) * (size_t)p.total_chunks);
    p.cbase = reinterpret_cast<double*>(w);
    w += align256(sizeof(double) * (size_t)p.total_chunks);
    p.plast = reinterpret_cast<int64_t*>(w);
    w += align256(sizeof(int64_t) * (size_t)p.total_chunks);
    p.stot = reinterpret_cast<double*>(w);
}

pwl_status design_launch(const DesignPlan& p, cudaStream_t s)
{
    const DeviceInfo& di = device_info();
    const int64_t tiles = p.total_chunks / kTileChunks;
    const int grid_chunks = (int)std::min<int64_t>(p.total_chunks, (int64_t)di.sms * 16);
    const int grid_tiles = (int)std::min<int64_t>(tiles, (int64_t)di.sms * 16);
    const bool by_tiles = p.precision == PWL_PREC_FP32 && p.F == 1 && tiles >= (int64_t)di.sms * 8;
    const int kinds = plan_kinds(p.kinds);
    if (kinds & kKindsAnalytic) {
        if (by_tiles)
            density_tiles_kernel<float, false><<<grid_tiles, kDesignThreads, 0, s>>>(p);
        else if (p.precision == PWL_PREC_FP32)
            density_chunks_kernel<float, false><<<grid_chunks, kDesignThreads, 0, s>>>(p);
        else
            density_chunks_kernel<double, false><<<grid_chunks, kDesignThreads, 0, s>>>(p);
        PWL_CHECK_LAUNCH("density_chunks_kernel");
    }
    if (kinds & kKindsSampled) {
        if (by_tiles)
            density_tiles_kernel<float, true><<<grid_tiles, kDesignThreads, 0, s>>>(p);
        else if (p.precision == PWL_PREC_FP32)
            density_chunks_kernel<float, true><<<grid_chunks, kDesignThreads, 0, s>>>(p);
        else
            density_chunks_kernel<double, true><<<grid_chunks, kDesignThreads, 0, s>>>(p);
        PWL_CHECK_LAUNCH("density_chunks_kernel");
    }
    chunk_scan_kernel<<<(int)std::min<int64_t>(p.F, 65535), kDesignThreads, 0, s>>>(p);
    PWL_CHECK_LAUNCH("chunk_scan_kernel");
    // enough slices that a tile holding every knot is done in two rounds of its
    // CTAs, as far as a CTA passes over a few batches of empty ones
    const int64_t slices = std::max<int64_t>(
        1, std::min<int64_t>(p.n_max / (2 * kDesignThreads), (int64_t)di.sms * 8 * kDesignThreads * 8 / tiles));
    const int grid_items = (int)std::min<int64_t>(tiles * slices, (int64_t)di.sms * 16);
    invert_tiles_kernel<<<grid_items, kDesignThreads, 0, s>>>(p, (int)slices);
    PWL_CHECK_LAUNCH("invert_tiles_kernel");
    return PWL_OK;
}

pwl_status design_batch_f_launch(const DesignPlan& p, cudaStream_t s)
{
    const DeviceInfo& di = device_info();
    const int grid = (int)std::min<int64_t>(p.total_chunks / kTileChunks, (int64_t)di.sms * 16);
    const int kinds = plan_kinds(p.kinds);
    const int grid_setup = (int)((p.total_chunks / kTileChunks + 127) / 128);
    tile_setup_f_kernel<<<grid_setup, 128, 0, s>>>(p);
    PWL_CHECK_LAUNCH("tile_setup_f_kernel");
    if (kinds & kKindsAnalytic) {
        density_tiles_f_kernel<false><<<grid, kDesignThreads, 0, s>>>(p);
        PWL_CHECK_LAUNCH("density_tiles_f_kernel");
    }
    if (kinds & kKindsSampled) {
        density_tiles_f_kernel<true><<<grid, kDesignThreads, 0, s>>>(p);
        PWL_CHECK_LAUNCH("density_tiles_f_kernel");
    }
    tile_scan_f_kernel<<<(int)std::min<int64_t>((p.F + 3) / 4, 65535), 128, 0, s>>>(p);
    PWL_CHECK_LAUNCH("tile_scan_f_kernel");
    invert_tiles_f_kernel<<<grid, kDesignThreads, 0, s>>>(p);
    PWL_CHECK_LAUNCH("invert_tiles_f_kernel");
    return PWL_OK;
}

}  // namespace pwl

using namespace pwl;

namespace {
constexpr size_t kMetaBytes = 512;  // descriptor, three offset pairs, cell width
int64_t resolve_cells(int64_t n, int64_t m) { return m > 0 ? m : 64 * n; }
}  // namespace

extern "C" {

size_t pwl_design_workspace_size(int64_t n_intervals, int64_t m_cells)
{
    if (n_intervals < 1) return 0;
    const int64_t M = resolve_cells(n_intervals, m_cells);
    // the size stays two doubles per cell, which the call's contract has had
    // callers provide; the kernels use about half of it
    return kMetaBytes + std::max(design_scratch_bytes(1, M, design_chunks(M)), align256(2 * sizeof(double) * (size_t)M));
}

pwl_status pwl_design(const pwl_func* f, int64_t n_intervals, int64_t m_cells, int32_t precision,
                      double* d_knots, void* d_workspace, size_t workspace_bytes, void* stream)
{
    clear_error();
    pwl_status st = validate_func(f);
    if (st != PWL_OK) return st;
    if (n_intervals < 1 || n_intervals > kMaxIntervals)
        return fail(PWL_EINVAL, "n_intervals must be in [1, %d] (got %lld)", kMaxIntervals,
                    (long long)n_intervals);
    if (m_cells < 0 || m_cells > (int64_t)1 << 32)
        return fail(PWL_EINVAL, "m_cells must be in [0, 2^32] (got %lld)", (long long)m_cells);
    if (precision != PWL_PREC_FP64 && precision != PWL_PREC_FP32)
        return fail(PWL_EINVAL, "unknown precision %d", precision);
    if (!d_knots) return fail(PWL_EINVAL, "d_knots is NULL");
    const int64_t M = resolve_cells(n_intervals, m_cells);
    const size_t need = pwl_design_workspace_size(n_intervals, m_cells);
    if (!d_workspace || workspace_bytes < need)
        return fail(PWL_EINVAL, "workspace of %zu bytes needed (got %zu)", need, workspace_bytes);
    if (reinterpret_cast<uintptr_t>(d_workspace) % 256 != 0)
        return fail(PWL_EINVAL, "workspace must be 256-byte aligned");

    char* w = static_cast<char*>(d_workspace);
    DesignPlan p{};
    p.F = 1;
    p.kinds = kinds_of(f, 1);
    p.funcs = reinterpret_cast<pwl_func*>(w);
    p.koff = reinterpret_cast<int64_t*>(w + 128);
    p.moff = reinterpret_cast<int64_t*>(w + 160);
    p.choff = reinterpret_cast<int64_t*>(w + 192);
    p.delta = reinterpret_cast<double*>(w + 224);
    p.n_max = n_intervals;
    p.total_knots = n_intervals + 1;
    p.total_cells = M;
    p.total_chunks = design_chunks(M);
    p.precision = precision;
    p.knots = d_knots;
    design_carve_scratch(p, w + kMetaBytes);
    cudaStream_t s = as_stream(stream);
    single_setup_kernel<<<1, 1, 0, s>>>(prepared(*f), n_intervals, M, p.total_chunks, const_cast<pwl_func*>(p.funcs),
                                        const_cast<int64_t*>(p.koff), const_cast<int64_t*>(p.moff),
                                        const_cast<int64_t*>(p.choff), const_cast<double*>(p.delta));
    PWL_CHECK_LAUNCH("single_setup_kernel");
    return design_launch(p, s);
}

}  // extern "C"
