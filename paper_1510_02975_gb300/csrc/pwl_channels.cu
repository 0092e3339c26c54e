// pwl_channels.cu -- channel-wise CPWL map: y[r, c] = v_c(x[r, c]) for a
// row-major x[R, C] with one CPWL function per channel (Algorithm 1 per
// element), and its backward (gradients w.r.t. x, the vertex values and the
// knots of every channel).  The knots and values are plain FP32 device
// arrays [C, N+1] (learnable parameters that change every step), so each CTA
// builds the cell index of its channels in shared memory when it starts.
//
// Both directions: a CTA owns a tile of CH consecutive channels (a lane keeps
// one of them) and holds, per channel, K uniform cells and one 16-byte record
// per interval, channel-interleaved ([e * CH + ch]) so that the lanes of a
// quarter- or half-warp read different banks whatever they look up.
//   cell       {x_k of the first knot in the cell (+inf if none), the interval
//              at the cell's left end | the distance to the next knot}
//   interval i {x_{i-1}, v_{i-1}, s_i, x_i} (forward),
//              {x_{i-1}, 1/h_i, s_i, x_i} (backward); record N + 1 serves
//              x = x_N
// An element takes the cell's interval, from x_k on the next one and from the
// knot after it on the one after that: two shared loads, two compares and no
// side selects.  The second distance is a BF16 number rounded up, so a point
// between a knot and its rounded place, or past a third knot of the cell, walks
// on while it is at or beyond the interval's right end.
//
// The CTAs of a cluster own adjacent tiles, 128 bytes of a row together (64
// for two 16-channel BF16 tiles), and walk the same rows: a row segment of
// less than a line that one CTA alone reads costs the whole line (a copy of
// [65536, 4096] FP32 in 64-byte segments: 640 us, by pairs 360 us).  What a
// copy of that access pattern reaches also depends on the L1 the index
// leaves: 16-channel tiles 360 us up to 132 KB of shared memory, 370 at 164
// KB, 500 at 198 KB and beyond; 8-channel tiles 503, 578 and 665.  So tiles
// are wide and, where that allows it, the index below kIndexBytes.
//
// Measured, [65536, 4096] x 257 knots: forward 532 -> 377 us (FP32; 5.70 TB/s),
// backward 1042 -> 780 us (4.1 TB/s); [16384, 4096] in BF16: forward 196 ->
// 110 us, backward 695 -> 238 us, 388 us of the 695 FP32 copies of the streams,
// which the BF16 kernel does without.  Before, the forward had 8-channel
// tiles (16-byte cells), the backward two compare-and-swap adds
// and side selects per element (103 instructions), and four CTAs a
// cluster left 8 SMs idle.  What bounds them now: the forward the access
// pattern (350-370 us as a plain copy), the backward instruction issue.
// A range costs ~5 us (forward) to ~15 us (backward) besides its rows: the
// index build and, backward, the reductions into the global gradients.
//
// Work: the tile groups (one per cluster) x passes of the CTA's rows, cut
// into one contiguous range per cluster, equal to a pass; a CTA rebuilds its
// index only where its range enters another group.
#include <math.h>

#include <algorithm>
#include <map>
#include <mutex>
#include <tuple>

#include "pwl_channels.cuh"

namespace pwl {

namespace {

constexpr int kChThreads = 1024;  // threads per CTA, both directions
constexpr int kFwdUnroll = 16;    // rows in flight per thread (64 KB per SM in FP32)
constexpr int kFwdTail = 4;       // rows per predicated batch of a range's tail
constexpr int kBwdUnroll = 8;     // rows of x and gy in flight per thread (64 KB per SM in FP32)
constexpr int kBwdTail = 2;
constexpr int kFwdGroup = 4;      // elements looked up together (their shared loads overlap, one chain test)
constexpr int kBwdGroup = 2;      // (fixed-point sums)
constexpr int kFloatGroup = 4;    // (FP32 sums; 2: 880 instead of 940 us, but 1181 instead of 862 at one point)
constexpr int kStage = 4;         // knots and values in flight per thread while a tile is staged

template <typename IO>
__device__ __forceinline__ float to_f32(IO v);
template <>
__device__ __forceinline__ float to_f32<float>(float v) { return v; }
template <>
__device__ __forceinline__ float to_f32<__nv_bfloat16>(__nv_bfloat16 v) { return __bfloat162float(v); }
template <typename IO>
__device__ __forceinline__ IO from_f32(float v);
template <>
__device__ __forceinline__ float from_f32<float>(float v) { return v; }
template <>
__device__ __forceinline__ __nv_bfloat16 from_f32<__nv_bfloat16>(float v) { return __float2bfloat16_rn(v); }

__device__ __forceinline__ void st_cs(float* p, float v) { __stcs(p, v); }
__device__ __forceinline__ void st_cs(__nv_bfloat16* p, __nv_bfloat16 v) { *p = v; }

// Cell of a point in [a, b]: cell_of with the clamp at 0 done by the unsigned
// conversion (negative and NaN give 0).  Monotone in x; the builder applies it
// to the knots.
__device__ __forceinline__ int chan_cell(float xc, float inv_w, float off, int K)
{
    return (int)min(__float2uint_rz(__fmaf_rn(xc, inv_w, off)), (unsigned)(K - 1));
}

// odd pitch of the staged knots and values ([ch][j]): the linear copy from
// global memory and the [j][ch] reads of the build are both nearly free of
// bank conflicts
__host__ __device__ __forceinline__ int stage_pitch(int N) { return (N + 1) | 1; }

// A cell's second word: interval i (16 bits) and, in the upper half, a BF16
// number strictly above d (the distance from the cell's first knot to the next
// one; an FP32 difference at or above it is of a point at or beyond that knot
// whatever the roundings).
__device__ __forceinline__ float make_cell(int i, float d)
{
    return __uint_as_float((unsigned)i | (min(__float_as_uint(fmaxf(d, 0.0f)) >> 16, 0x7f7fu) + 1) << 16);
}

// Builds the index of channels [c0, c0 + CH): interval records rec[i * CH + ch]
// (i = 0..N+1) and cell records cells[c * CH + ch].  The staged knots and
// values live where the cell records go, which are written last, from the
// interval records.  Every cell gets a record in range whatever the knots are,
// so that knots that do not increase (*bad is set) give unspecified results
// but no stray access.  staged() runs after the first barrier; the caller has
// a barrier before (nobody reads the previous tile) and gets one after.
// Measured (16 channels of 257 knots, clocks): staging 3000, interval records
// 2300, cells 4500.
template <int CH, bool BWD, class Staged>
__device__ __forceinline__ void build_tile(const ChanArgs& p, int64_t c0, float2* cells, float4* rec, int* bad,
                                           const Staged& staged)
{
    const int N = p.N, K = p.K, n1 = N + 1, P = stage_pitch(N);
    const int nch = (int)min((int64_t)CH, p.C - c0);
    float* xs = reinterpret_cast<float*>(cells);
    float* vs = xs + (size_t)CH * P;
    {
        constexpr int per_ch = kChThreads / CH;
        const int ch = threadIdx.x / per_ch;
        if (ch < nch) {
            const float* kx = p.knots + (c0 + ch) * (int64_t)n1;
            const float* kv = p.values + (c0 + ch) * (int64_t)n1;
            for (int j = threadIdx.x % per_ch; j < n1; j += kStage * per_ch) {
                float a[kStage], b[kStage];
#pragma unroll
                for (int u = 0; u < kStage; ++u)
                    if (j + u * per_ch < n1) {
                        a[u] = kx[j + u * per_ch];
                        b[u] = kv[j + u * per_ch];
                    }
#pragma unroll
                for (int u = 0; u < kStage; ++u)
                    if (j + u * per_ch < n1) {
                        xs[ch * P + j + u * per_ch] = a[u];
                        vs[ch * P + j + u * per_ch] = b[u];
                    }
            }
        }
        if (threadIdx.x == 0) *bad = 0;
    }
    __syncthreads();
    staged();
    // from here on a thread keeps one channel
    constexpr int RP = kChThreads / CH;
    const int ch = threadIdx.x % CH, row = threadIdx.x / CH;
    const float inf = __int_as_float(0x7f800000);
    if (ch < nch) {
        bool ok = true;
        for (int i = 1 + row; i <= N; i += RP) {
            const float xl = xs[ch * P + i - 1], vl = vs[ch * P + i - 1];
            const float xr = xs[ch * P + i], vr = vs[ch * P + i];
            // slopes and reciprocal lengths by FP32 IEEE division of the FP32
            // differences: at most ~2 ulp from the exact slope of the FP32 table
            const float h = __fsub_rn(xr, xl), s = __fdiv_rn(__fsub_rn(vr, vl), h);
            rec[i * CH + ch] = make_float4(xl, BWD ? __frcp_rn(h) : vl, s, xr);
            ok = ok && xr > xl;
            if (i == N) {
                // x = x_N.  Forward: v_N exactly.  Backward: delta = 0 from x_N to
                // a right end one spacing above it, so that its sums reach knot N;
                // gx = gy s_N
                const float up = fabsf(xr) < 0x1p-100f ? xr + 0x1p-100f : nextafterf(xr, inf);
                rec[(N + 1) * CH + ch] = BWD ? make_float4(xr, 1.0f / (up - xr), s, up) : make_float4(xr, vr, 0.0f, inf);
            }
        }
        if (row == RP - 1) rec[ch] = make_float4(xs[ch * P], 0.0f, 0.0f, xs[ch * P]);
        if (!ok) *bad = 1;
    }
    __syncthreads();
    if (ch < nch) {
        // a few consecutive knots per thread: knot j names the cells after knot
        // j - 1's up to its own, which is a knot cell of knot j if it is the
        // first there (and x_N the cells past its own, which no point reaches)
        const float4* knot = rec + CH + ch;  // x_j = knot[j * CH].x, j = 0..N
        const float a = knot[0].x, b = knot[N * CH].x;
        const float inv_w = (float)K / (b - a), off = -a * inv_w;
        const int per = (n1 + RP - 1) / RP, je = min(n1, (row + 1) * per);
        int j = row * per;
        if (j < je) {
            int c = j > 0 ? chan_cell(knot[(j - 1) * CH].x, inv_w, off, K) + 1 : 0;
            float xj = knot[j * CH].x;
            for (; j < je; ++j) {
                const float xn = j < N ? knot[(j + 1) * CH].x : inf;
                const int cj = chan_cell(xj, inv_w, off, K);
                const float2 free = make_float2(inf, make_cell(j, inf));
#pragma unroll 4
                for (; c < cj; ++c) cells[c * CH + ch] = free;
                if (c == cj) cells[c * CH + ch] = make_float2(xj, make_cell(j, xn - xj));
                if (j == N)
                    for (c = cj + 1; c < K; ++c) cells[c * CH + ch] = free;
                c = cj + 1;
                xj = xn;
            }
        }
    }
    __syncthreads();
}

// Shared memory by 32-bit address.  A pointer into extern shared memory is
// rebuilt from special registers at each use in a cluster launch (about six
// instructions per element of the backward); these addresses are formed once.
__device__ __forceinline__ uint32_t smem_addr(const void* p)
{
    uint32_t a = (uint32_t)__cvta_generic_to_shared(p);
    asm volatile("" : "+r"(a));  // keeps the compiler from forming it again
    return a;
}
__device__ __forceinline__ float2 lds2(uint32_t a)
{
    float2 v;
    asm("ld.shared.v2.f32 {%0, %1}, [%2];" : "=f"(v.x), "=f"(v.y) : "r"(a) : "memory");
    return v;
}
__device__ __forceinline__ float4 lds4(uint32_t a)
{
    float4 v;
    asm("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "r"(a) : "memory");
    return v;
}
template <int OFF>
__device__ __forceinline__ void red_add(uint32_t a, int v)
{
    asm volatile("red.shared.add.s32 [%0+%2], %1;" ::"r"(a), "r"(v), "n"(OFF) : "memory");
}

// A thread's channel is fixed for a tile: its constants live in registers.
template <int CH>
struct ChanConst {
    uint32_t cells, rec;  // shared addresses of the channel's first cell and record
    uint32_t last;        // of record N + 1
    float a, b, inv_w, off;
    int K;
    __device__ __forceinline__ ChanConst(const ChanArgs& p, const float2* cells0, const float4* rec0, int ch)
        : cells(smem_addr(cells0 + ch)), rec(smem_addr(rec0 + ch)), last(rec + (uint32_t)(p.N + 1) * (16 * CH)),
          a(rec0[CH + ch].x), b(rec0[p.N * CH + ch].w), inv_w((float)p.K / (b - a)), off(-a * inv_w), K(p.K)
    {
    }
};

// The records of the intervals of G points in [a, b], and their addresses.
template <int CH, int G>
__device__ __forceinline__ void chan_lookup(const float (&xc)[G], const ChanConst<CH>& cc, float4 (&r)[G],
                                            uint32_t (&at)[G])
{
    float2 c[G];
#pragma unroll
    for (int g = 0; g < G; ++g) c[g] = lds2(cc.cells + chan_cell(xc[g], cc.inv_w, cc.off, cc.K) * (8 * CH));
    bool more = false;
#pragma unroll
    for (int g = 0; g < G; ++g) {
        const unsigned w = __float_as_uint(c[g].y);
        int i = (int)(w & 0xffffu);
        if (xc[g] >= c[g].x) ++i;
        if (xc[g] - c[g].x >= __uint_as_float(w & 0xffff0000u)) ++i;
        at[g] = cc.rec + i * (16 * CH);
        r[g] = lds4(at[g]);
    }
#pragma unroll
    for (int g = 0; g < G; ++g) more = more || xc[g] >= r[g].w;
    if (more) {
#pragma unroll
        for (int g = 0; g < G; ++g)
            while (xc[g] >= r[g].w && at[g] < cc.last) {
                at[g] += 16 * CH;
                r[g] = lds4(at[g]);
            }
    }
}

// ---- forward -----------------------------------------------------------------
template <int CH, int G>
__device__ __forceinline__ void chan_fwd(float (&v)[G], const ChanConst<CH>& cc)
{
    float xc[G];
    float4 r[G];
    uint32_t at[G];
#pragma unroll
    for (int g = 0; g < G; ++g) xc[g] = clamp_nan(v[g], cc.a, cc.b);
    chan_lookup<CH, G>(xc, cc, r, at);
#pragma unroll
    for (int g = 0; g < G; ++g) v[g] = __fmaf_rn(xc[g] - r[g].x, r[g].z, r[g].y);
}

template <typename IO, int CH>
__device__ __forceinline__ void chan_fwd_rows(const ChanArgs& p, int64_t c0, int64_t r0, int64_t r1,
                                              const float2* cells, const float4* rec, const IO* __restrict__ x,
                                              IO* __restrict__ y)
{
    constexpr int RP = kChThreads / CH, U = kFwdUnroll, G = kFwdGroup;
    const int ch = threadIdx.x % CH, row = threadIdx.x / CH;
    if (c0 + ch >= p.C) return;
    const ChanConst<CH> cc(p, cells, rec, ch);
    int64_t r = r0 + row;
    const int64_t step = (int64_t)RP * p.C;  // elements between a thread's consecutive rows
    const IO* px = x + r * p.C + c0 + ch;
    IO* py = y + r * p.C + c0 + ch;
    for (; r + (U - 1) * RP < r1; r += U * RP) {
        // x is read at the L2 only (ld.global.cg)
        float v[U];
#pragma unroll
        for (int u = 0; u < U; ++u) v[u] = to_f32<IO>(__ldcg(px + u * step));
#pragma unroll
        for (int u = 0; u < U; u += G) {
            float w[G];
#pragma unroll
            for (int g = 0; g < G; ++g) w[g] = v[u + g];
            chan_fwd<CH, G>(w, cc);
#pragma unroll
            for (int g = 0; g < G; ++g) st_cs(py + (u + g) * step, from_f32<IO>(w[g]));
        }
        px += U * step;
        py += U * step;
    }
    // the rest (fewer than U rows per thread) in predicated batches: a few load
    // latencies instead of one per row
    for (; r < r1; r += (int64_t)kFwdTail * RP) {
        const int64_t left = (r1 - r + RP - 1) / RP;
        const int rem = left < kFwdTail ? (int)left : kFwdTail;
        float v[kFwdTail];
#pragma unroll
        for (int u = 0; u < kFwdTail; ++u) v[u] = u < rem ? to_f32<IO>(__ldcg(px + u * step)) : cc.a;
        chan_fwd<CH, kFwdTail>(v, cc);
#pragma unroll
        for (int u = 0; u < kFwdTail; ++u)
            if (u < rem) st_cs(py + u * step, from_f32<IO>(v[u]));
        px += kFwdTail * step;
        py += kFwdTail * step;
    }
}

// Calls body(tile, r0, r1) for the row ranges of this CTA's share of the work.
template <int CH, class Body>
__device__ __forceinline__ void for_each_range(const ChanArgs& p, const Body& body)
{
    constexpr int RP = kChThreads / CH;
    const int64_t cluster = blockIdx.x / p.cluster, nclusters = gridDim.x / p.cluster;
    const int64_t w1 = p.work * (cluster + 1) / nclusters;
    for (int64_t w = p.work * cluster / nclusters; w < w1;) {
        const int64_t group = w / p.passes, end = min(w1, (group + 1) * p.passes);
        const int64_t tile = group * p.cluster + blockIdx.x % p.cluster;
        const int64_t r0 = (w - group * p.passes) * RP, r1 = min(p.R, (end - group * p.passes) * RP);
        w = end;
        if (tile * CH < p.C) body(tile, r0, r1);  // no tile past the last one of a partial group
    }
}

template <typename IO, int CH>
__global__ void __launch_bounds__(kChThreads, 1) channels_forward_kernel(const ChanArgs p, const IO* x, IO* y)
{
    extern __shared__ float4 s_ch[];
    __shared__ int s_bad;
    float4* rec = s_ch;
    float2* cells = reinterpret_cast<float2*>(rec + (size_t)(p.N + 2) * CH);
    for_each_range<CH>(p, [&](int64_t tile, int64_t r0, int64_t r1) {
        __syncthreads();  // nobody reads the previous tile any more
        build_tile<CH, false>(p, tile * CH, cells, rec, &s_bad, [] {});
        if (threadIdx.x == 0 && s_bad) atomicOr(p.status, 1);
        chan_fwd_rows<IO, CH>(p, tile * CH, r0, r1, cells, rec, x, y);
    });
}

// ---- backward ----------------------------------------------------------------
// gx = gy * s_i; per (channel, interval) the sums A_i = sum gy (x_i - x)/h_i and
// B_i = sum gy (x - x_{i-1})/h_i accumulate in shared memory; at the end of a
// tile's rows they become g_v[j] += A_{j+1} + B_j (+ clamped terms) and
// g_x[j] += -s_{j+1} A_{j+1} - s_j B_j, added to the global gradients.
//
// An FP32 shared-memory add is a compare-and-swap loop in software (about 10
// instructions, 2.6 adds per clock and SM against more than 9 for int32), so a
// range of rows takes one of two forms of the sums:
//
//   fixed point, two 32-bit words per sum: a term v in units of 2^-F is
//     h 2^19 + l + rest with h = rint(v 2^-19) (by adding 1.5 2^23, which needs
//     no conversion) and l = rint(v - h 2^19), both added with native integer
//     atomics that return nothing.  |v| < 2^37 keeps h and l within 2^18, so
//     6144 rows add less than 2^31 - 2^28 to a word; every 6144 rows the words
//     are looked over and the tile's sums flushed where one has passed 2^28.
//     A term of 2^17 units or more is rounded at 2^-18 of itself or finer (from
//     2^23 on it is exact).  The rest of a smaller one, which the words do not
//     hold, goes to the global gradients in FP32, and so does a term beyond 2^37
//     (taken out of the words again): every sum is accurate relative to its own
//     terms, however small they are beside the channel's other gradients.
//   FP32, one word per sum: where more than kSlowSamples of the range's 1024
//     sampled elements have such a term, or none is nonzero.
//
// F comes, per channel, from 64 (128) sampled |gy|, spread over the range's rows at
// irregular distances (the first rows of sequences and the like are not typical);
// terms of up to 4 to 8 times their largest fit (see fix_exponent).
//
// [65536, 4096] x 257 knots, us (the FP32 atomics before; one unit from the mean exponent
// of the rows R k / 64 and four global adds for every element above it; now):
//   normal gradients                                    1009    694    785
//   log-normal, sigma 1 / 1.6 / 2 / 3                   1009   1858+   870 / 1110 / 940 / 940
//   every 1024th row zero                               1010   6315    785
//   half / 97% / 99.9% zero                         917-968    695    785 / 785 / 842
//   0.1% / 1% of them 2^10 as large                     1009           874 / 1344
//   over 10 decades along x, one interval's 2^-26       1010   2820+   940
//   a third of the points outside                        943   1490    912
//   all points of a channel / half of all in an interval 3090   690    784 / 785
//   half of them within 2^-10 of a knot in some channels 2416          1250
// In FP32 alone: 850-895 for every distribution, but 2860 where all points of a channel
// fall into one interval, 1565 with 7 intervals (740), and 5 to 27 times the rounding error
// (6e-8).  Of the 785, the test for small terms takes 20 and the look at the words 30
// (the barriers' waits).
constexpr int kDigitBits = 19;
constexpr int kRangeBits = 37;                                // terms below 2^37 units
constexpr float kFixLimit = 0x1p37f;
constexpr unsigned kSmallKey = 2u * ((127 + 17) << 23) - 2u;  // small_key of 2^17
constexpr int kSegRows = 6144;                                // whole unrolled passes of every tile width
constexpr int kFullWord = 1 << 28;
constexpr int kSlowSamples = 4;  // (log-normal, sigma 2: 940 us, with 6 1356; with 3 some normal ranges take FP32 sums)
constexpr float kMagic = 0x1.8p23f;
constexpr unsigned kMagicBits = 0x4B400000u;
constexpr float kDigit = 0x1p19f, kPerDigit = 0x1p-19f;

// What a range's setup shares, and what the rare paths need (in registers it would
// weigh on the loop that hardly ever takes them).
struct BwdShared {
    int bad;
    // per channel, of the nonzero finite samples: the largest binary exponent (kNoSample
    // if none), the exponents' sum, their number
    int emax[16], esum[16], ecnt[16];
    float unit[16];  // per channel: 2^-F
    float *gv, *gk;  // the tile's rows of the global gradients (or NULL)
    uint32_t rec;    // shared address of the tile's first record
    int N;
};
__shared__ BwdShared s_bwd;
constexpr int kNoSample = -1000;

// This thread's sampled element: its channel, a row of its stratum of [r0, r1).
// The rows are the CTA's own, so that gx may overwrite gy.
template <typename IO, int CH>
__device__ __forceinline__ void sample(const ChanArgs& p, int64_t c0, int64_t r0, int64_t r1, const IO* x,
                                       const IO* gy, float& xs, float& gs)
{
    constexpr int S = kChThreads / CH;
    const int64_t c = c0 + threadIdx.x % CH, n = r1 - r0, s = threadIdx.x / CH;
    xs = gs = 0.0f;
    if (c >= p.C) return;
    // multiples of the golden ratio mod 1; one row for the tile's channels (a row each
    // read 16 times the sectors, 0.08 of the 0.66 GB of a call at 16384 rows)
    const unsigned h = (unsigned)(c0 / CH * S + s) * 0x9E3779B9u;
    const int64_t lo = n * s / S, w = min(n * (s + 1) / S - lo, (int64_t)0x7fffffff);
    const int64_t at = (r0 + lo + (int64_t)((uint64_t)h * (uint64_t)w >> 32)) * p.C + c;
    xs = to_f32<IO>(__ldcg(x + at));
    gs = to_f32<IO>(__ldcg(gy + at));
}
// the samples' binary exponents (nonzero finite ones) into the channels' figures
template <int CH>
__device__ __forceinline__ void add_exponents(float g)
{
    const int ex = (int)(__float_as_uint(g) >> 23 & 0xffu);
    const bool ok = ex != 0 && ex != 0xff;
    int top = ok ? ex - 127 : kNoSample, sum = ok ? ex - 127 : 0, cnt = ok ? 1 : 0;
    for (int o = CH; o < 32; o <<= 1) {
        top = max(top, __shfl_xor_sync(0xffffffffu, top, o));
        sum += __shfl_xor_sync(0xffffffffu, sum, o);
        cnt += __shfl_xor_sync(0xffffffffu, cnt, o);
    }
    if ((threadIdx.x & 31) < CH && cnt) {
        atomicMax(&s_bwd.emax[threadIdx.x % CH], top);
        atomicAdd(&s_bwd.esum[threadIdx.x % CH], sum);
        atomicAdd(&s_bwd.ecnt[threadIdx.x % CH], cnt);
    }
}

// F of a channel, from its largest sample, but no more than 2^7 of the mean (a single
// outlier would leave the others few bits).  Few samples say little: with less than 8
// nonzero ones the tile's largest counts too, up to 2^10 above the channel's own, and
// with none it stands alone (where it is far too coarse, the channel's terms count as
// small).  2^F and 2^-F are normal FP32 numbers.  kNoSample if the tile has no nonzero
// sample.
template <int CH>
__device__ __forceinline__ int fix_exponent(int ch)
{
    const int n = s_bwd.ecnt[ch];
    int e = n > 0 ? min(s_bwd.emax[ch], (int)floorf((float)s_bwd.esum[ch] / (float)n) + 7) : kNoSample;
    if (n < 8) {
        int top = kNoSample;
        for (int q = 0; q < CH; ++q) top = max(top, s_bwd.emax[q]);
        e = n > 0 ? max(e, min(top, e + 10)) : top;
    }
    return e == kNoSample ? kNoSample : min(max(kRangeBits - (n < 16 ? 4 : 3) - e, -100), 126);
}
__device__ __forceinline__ float exp2_int(int e) { return __int_as_float((e + 127) << 23); }

// orders terms by magnitude, 0 (which is exact) above all
__device__ __forceinline__ unsigned small_key(float v) { return 2u * __float_as_uint(v) - 2u; }

// h 2^19 of a term, and the rest of it
__device__ __forceinline__ float fix_high(float v, float& m)
{
    m = __fmaf_rn(v, kPerDigit, kMagic);
    return __fmaf_rn(__fsub_rn(m, kMagic), -kDigit, v);
}
// one term into its two words (h at byte offset 0, l at byte offset L)
template <int L, int SIGN = 1>
__device__ __forceinline__ void fix_add(uint32_t at, float v)
{
    float m;
    const float low = fix_high(v, m);
    red_add<0>(at, (int)(SIGN * (__float_as_uint(m) - kMagicBits)));
    red_add<L>(at, (int)(SIGN * (unsigned)__float2int_rn(low)));
}
// what fix_add's words leave out
__device__ __forceinline__ float fix_rest(float v)
{
    float m;
    const float low = fix_high(v, m);
    return low - __int2float_rn(__float2int_rn(low));
}
__device__ __forceinline__ void float_add(uint32_t at, float v)
{
    if (v != 0.0f) asm volatile("red.shared.add.f32 [%0], %1;" ::"r"(at), "f"(v) : "memory");
}

// FP32 sums of the gradients w.r.t. the end values of clamped elements
struct EndSums {
    float left, right;
};

// What the backward of one channel needs besides its lookup: record address ->
// address of the interval's A words and B words (odd rows: B and A).
struct BwdOut {
    uint32_t first, second;
    float scale;
    bool odd;
};
template <int CH>
__device__ __forceinline__ bool odd_row()
{
    return CH == 16 && threadIdx.x / CH % 2;
}

// Two terms (in the order of this thread's row) of an element whose record is at
// `at`, to the global gradients in FP32; s: the interval's slope.
template <int CH>
__device__ __noinline__ void add_global_terms(float t1, float t2, uint32_t at, float s)
{
    const int e = (int)(at - s_bwd.rec) / (16 * CH), i = max(e, 1);  // 0 only where x_0 is NaN
    const int64_t k = (int64_t)(threadIdx.x % CH) * (s_bwd.N + 1) + i;
    const float l = odd_row<CH>() ? t2 : t1;                        // at the interval's left knot
    const float r = e > s_bwd.N ? 0.0f : odd_row<CH>() ? t1 : t2;  // at its right one (none past x_N)
    if (s_bwd.gv) {
        if (l != 0.0f) atomicAdd(s_bwd.gv + k - 1, l);
        if (r != 0.0f) atomicAdd(s_bwd.gv + k, r);
    }
    if (s_bwd.gk) {
        if (l != 0.0f) atomicAdd(s_bwd.gk + k - 1, -s * l);
        if (r != 0.0f) atomicAdd(s_bwd.gk + k, -s * r);
    }
}
// The same for what the words of two terms leave out.
template <int CH>
__device__ __noinline__ void add_rests(float t1, float t2, uint32_t at, float s)
{
    const float unit = s_bwd.unit[threadIdx.x % CH];
    const float e1 = fix_rest(t1) * unit, e2 = fix_rest(t2) * unit;
    if (e1 != 0.0f || e2 != 0.0f) add_global_terms<CH>(e1, e2, at, s);
}

// Two terms out of range, whose words hold nonsense: out of the words again (integer
// adds are exact modulo 2^32) and to the global gradients.
template <int CH>
__device__ __noinline__ void add_instead(float v1, float v2, float t1, float t2, uint32_t at, float s, uint32_t first,
                                         uint32_t second)
{
    fix_add<8 * CH, -1>(at + first, v1);  // (as they were added, in units)
    fix_add<8 * CH, -1>(at + second, v2);
    add_global_terms<CH>(t1, t2, at, s);
}

// G elements: gx in place of g.  One branch per group: what elements outside the
// domain, small terms and terms out of range need comes after the adds (a branch for
// each of the three, two of them before the adds: 840 us instead of 800).
template <int CH, int G, bool FLOAT>
__device__ __forceinline__ void chan_bwd(const float (&x)[G], float (&g)[G], const ChanConst<CH>& cc, const BwdOut& o,
                                         EndSums& ends)
{
    float xc[G], gs[G];
    float4 r[G];
    uint32_t at[G];
    bool inside = true, fits = true;
#pragma unroll
    for (int q = 0; q < G; ++q) {
        xc[q] = fminf(fmaxf(x[q], cc.a), cc.b);  // NaN -> a
        inside = inside && x[q] == xc[q];
        gs[q] = x[q] == xc[q] ? (FLOAT ? g[q] : g[q] * o.scale) : 0.0f;
    }
    chan_lookup<CH, G>(xc, cc, r, at);
    // 1 - delta and delta, each from the interval's other end and so accurate
    // where it is small; odd rows take them in the other order
    auto terms = [&](int q, float gq, float& t1, float& t2) {
        const float p1 = o.odd ? r[q].x : r[q].w, p2 = o.odd ? r[q].w : r[q].x;
        t1 = gq * (fabsf(p1 - xc[q]) * r[q].y);
        t2 = gq * (fabsf(p2 - xc[q]) * r[q].y);
    };
    unsigned small = ~0u;
    if constexpr (FLOAT) {
        // elements of one interval added up first: adds to one address wait for each other
        float t1[G], t2[G];
#pragma unroll
        for (int q = 0; q < G; ++q) terms(q, gs[q], t1[q], t2[q]);
#pragma unroll
        for (int q = 1; q < G; ++q)
            if (at[q] == at[0]) {
                t1[0] += t1[q];
                t2[0] += t2[q];
                t1[q] = t2[q] = 0.0f;
            }
#pragma unroll
        for (int q = 0; q < G; ++q) {
            float_add(at[q] + o.first, t1[q]);
            float_add(at[q] + o.second, t2[q]);
        }
    } else {
#pragma unroll
        for (int q = 0; q < G; ++q) {
            float t1, t2;
            terms(q, gs[q], t1, t2);
            fix_add<8 * CH>(at[q] + o.first, t1);
            fix_add<8 * CH>(at[q] + o.second, t2);
            small = min(small, min(small_key(t1), small_key(t2)));
            fits = fits && fabsf(gs[q]) < kFixLimit;
        }
    }
    if (!inside || !fits || small < kSmallKey) {
        if (!fits || small < kSmallKey) {
#pragma unroll
            for (int q = 0; q < G; ++q) {
                float t1, t2;
                terms(q, gs[q], t1, t2);
                if (fabsf(gs[q]) < kFixLimit) {
                    if (min(small_key(t1), small_key(t2)) < kSmallKey) add_rests<CH>(t1, t2, at[q], r[q].z);
                } else {
                    float u1, u2;
                    terms(q, g[q], u1, u2);
                    add_instead<CH>(t1, t2, u1, u2, at[q], r[q].z, o.first, o.second);
                }
            }
        }
#pragma unroll
        for (int q = 0; q < G; ++q) {
            const bool in = x[q] == xc[q];
            ends.left += x[q] < cc.a ? g[q] : 0.0f;
            ends.right += x[q] > cc.b ? g[q] : 0.0f;
            g[q] = in ? g[q] * r[q].z : x[q] != x[q] ? x[q] : 0.0f;
        }
        return;
    }
#pragma unroll
    for (int q = 0; q < G; ++q) g[q] *= r[q].z;
}

// Whether the fixed-point form of a sampled element needs a global add.
template <int CH>
__device__ __forceinline__ bool slow_sample(float x, float g, const ChanConst<CH>& cc, float scale)
{
    float xc[1] = {fminf(fmaxf(x, cc.a), cc.b)};
    float4 r[1];
    uint32_t at[1];
    chan_lookup<CH, 1>(xc, cc, r, at);
    const float gs = g * scale, t1 = gs * (fabsf(r[0].w - xc[0]) * r[0].y), t2 = gs * (fabsf(r[0].x - xc[0]) * r[0].y);
    return x == xc[0] && (!(fabsf(gs) < kFixLimit) || min(small_key(t1), small_key(t2)) < kSmallKey);
}

template <typename IO, int CH, bool FLOAT>
__device__ __forceinline__ void chan_bwd_rows(const ChanArgs& p, int64_t c0, int64_t r0, int64_t r1,
                                              const float2* cells, const float4* rec, int* acc, float scale,
                                              const IO* __restrict__ x, const IO* __restrict__ gy,
                                              IO* __restrict__ gx)
{
    constexpr int RP = kChThreads / CH, U = kBwdUnroll, G = FLOAT ? kFloatGroup : kBwdGroup;
    const int ch = threadIdx.x % CH, row = threadIdx.x / CH;
    const int64_t c = c0 + ch;
    if (c >= p.C) return;
    const ChanConst<CH> cc(p, cells, rec, ch);
    const bool odd = odd_row<CH>();
    const uint32_t words = smem_addr(acc + ch) - cc.rec;
    const BwdOut out{words + (odd ? 4 * CH : 0), words + (odd ? 0 : 4 * CH), scale, odd};
    EndSums ends{0.0f, 0.0f};
    int64_t r = r0 + row;
    const int64_t step = (int64_t)RP * p.C;
    const IO* px = x + r * p.C + c;
    const IO* pg = gy + r * p.C + c;
    IO* po = gx + r * p.C + c;
    for (; r + (U - 1) * RP < r1; r += U * RP) {
        IO xv[U], gv[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
            xv[u] = __ldcg(px + u * step);
            gv[u] = __ldcg(pg + u * step);
        }
#pragma unroll
        for (int u = 0; u < U; u += G) {
            float xf[G], gf[G];
#pragma unroll
            for (int q = 0; q < G; ++q) {
                xf[q] = to_f32<IO>(xv[u + q]);
                gf[q] = to_f32<IO>(gv[u + q]);
            }
            chan_bwd<CH, G, FLOAT>(xf, gf, cc, out, ends);
#pragma unroll
            for (int q = 0; q < G; ++q) st_cs(po + (u + q) * step, from_f32<IO>(gf[q]));
        }
        px += U * step;
        pg += U * step;
        po += U * step;
    }
    for (; r < r1; r += (int64_t)kBwdTail * RP) {
        const int64_t left = (r1 - r + RP - 1) / RP;
        const int rem = left < kBwdTail ? (int)left : kBwdTail;
        float xf[kBwdTail], gf[kBwdTail];
#pragma unroll
        for (int u = 0; u < kBwdTail; ++u) {
            xf[u] = u < rem ? to_f32<IO>(__ldcg(px + u * step)) : cc.a;
            gf[u] = u < rem ? to_f32<IO>(__ldcg(pg + u * step)) : 0.0f;
        }
        chan_bwd<CH, kBwdTail, FLOAT>(xf, gf, cc, out, ends);
#pragma unroll
        for (int u = 0; u < kBwdTail; ++u)
            if (u < rem) st_cs(po + u * step, from_f32<IO>(gf[u]));
        px += kBwdTail * step;
        pg += kBwdTail * step;
        po += kBwdTail * step;
    }
    if (s_bwd.gv) {
        float* gv = s_bwd.gv + ch * (p.N + 1);
        if (ends.left != 0.0f) atomicAdd(gv, ends.left);
        if (ends.right != 0.0f) atomicAdd(gv + p.N, ends.right);
    }
}

// (out of line: inlined, it costs the fixed-point loop registers)
template <typename IO, int CH>
__device__ __noinline__ void chan_bwd_rows_float(const ChanArgs& p, int64_t c0, int64_t r0, int64_t r1,
                                                 const float2* cells, const float4* rec, int* acc, const IO* x,
                                                 const IO* gy, IO* gx)
{
    chan_bwd_rows<IO, CH, true>(p, c0, r0, r1, cells, rec, acc, 1.0f, x, gy, gx);
}

// n floats from shared memory (16-byte aligned) added to global ones, whole
// 16-byte vectors where dst allows.
__device__ __forceinline__ void add_global(float* dst, const float* src, int n)
{
    const int nv = reinterpret_cast<uintptr_t>(dst) % 16 == 0 ? n / 4 : 0;
    for (int i = threadIdx.x; i < nv; i += kChThreads)
        atomicAdd(reinterpret_cast<float4*>(dst) + i, reinterpret_cast<const float4*>(src)[i]);
    for (int i = 4 * nv + threadIdx.x; i < n; i += kChThreads)
        if (src[i] != 0.0f) atomicAdd(dst + i, src[i]);
}

// Adds a tile's sums to the global gradients and clears them.  With the tile's
// last rows done (`stage`: the cell records' memory) the gradients pass
// through shared memory, laid out as in global memory, and are added 16 bytes
// at a time (one reduction per lane and address, to 32 different lines per
// warp, took 15000 clocks for 16 channels of 257 knots).
template <int CH>
__device__ __forceinline__ void flush_tile(const ChanArgs& p, int64_t c0, const float4* rec, int* acc, bool flt,
                                           float* stage, float* g_values, float* g_knots)
{
    __syncthreads();
    const int N = p.N, n1 = N + 1;
    const int ch = threadIdx.x % CH, nch = (int)min((int64_t)CH, p.C - c0);
    const float unit = s_bwd.unit[ch];
    float* stage_k = stage + (CH * n1 + 3) / 4 * 4;
    // a sum, cleared: its FP32 word, or h 2^19 + l of its two words (with l's carry
    // moved to h, one conversion is exact, or rounds below half an ulp, and nothing
    // cancels)
    auto take = [&](int i, int w) {
        int *ph = acc + (i * 4 + w) * CH + ch, *pl = ph + 2 * CH;
        const int hi = *ph, l = *pl, h = hi + (l >> kDigitBits);
        *ph = 0;
        *pl = 0;
        if (flt) return __int_as_float(hi);
        return __fmaf_rn((float)h, kDigit, (float)(l & ((1 << kDigitBits) - 1))) * unit;
    };
    if (ch < nch)
        for (int j = threadIdx.x / CH; j <= N; j += kChThreads / CH) {
            // A of interval j + 1 (of the elements at x_N for j = N), B of interval j
            const float A = take(j + 1, 0), B = j > 0 ? take(j, 1) : 0.0f;
            const float gv = A + B, gk = -rec[(j + 1) * CH + ch].z * A - rec[j * CH + ch].z * B;
            if (stage) {
                stage[ch * n1 + j] = gv;
                stage_k[ch * n1 + j] = gk;
            } else {
                const int64_t at = (c0 + ch) * n1 + j;
                if (g_values && gv != 0.0f) atomicAdd(g_values + at, gv);
                if (g_knots && gk != 0.0f) atomicAdd(g_knots + at, gk);
            }
        }
    __syncthreads();
    if (stage && g_values) add_global(g_values + c0 * n1, stage, nch * n1);
    if (stage && g_knots) add_global(g_knots + c0 * n1, stage_k, nch * n1);
}

// Whether a word of the tile's sums could wrap in the next kSegRows rows.
template <int CH>
__device__ __forceinline__ bool near_full(const ChanArgs& p, const int* acc)
{
    __syncthreads();
    bool full = false;
    for (int i = threadIdx.x; i < (p.N + 2) * CH; i += kChThreads) {
        const int4 v = reinterpret_cast<const int4*>(acc)[i];
        for (const int w : {v.x, v.y, v.z, v.w}) full = full || (unsigned)(w + kFullWord) > 2u * kFullWord;
    }
    return __syncthreads_or(full);
}

template <typename IO, int CH>
__global__ void __launch_bounds__(kChThreads, 1) channels_backward_kernel(const ChanArgs p, const IO* x, const IO* gy,
                                                                          IO* gx, float* g_values, float* g_knots)
{
    extern __shared__ float4 s_ch[];
    float4* rec = s_ch;
    int* acc = reinterpret_cast<int*>(rec + (size_t)(p.N + 2) * CH);
    float2* cells = reinterpret_cast<float2*>(acc + (size_t)(p.N + 2) * 4 * CH);
    for (int i = threadIdx.x; i < (p.N + 2) * 4 * CH; i += kChThreads) acc[i] = 0;
    if (threadIdx.x == 0) {
        s_bwd.rec = smem_addr(rec);
        s_bwd.N = p.N;
    }
    for_each_range<CH>(p, [&](int64_t tile, int64_t r0, int64_t r1) {
        const int64_t c0 = tile * CH;
        const int ch = threadIdx.x % CH;
        __syncthreads();  // nobody reads the previous tile any more
        if (threadIdx.x < CH) {
            s_bwd.emax[threadIdx.x] = kNoSample;
            s_bwd.esum[threadIdx.x] = s_bwd.ecnt[threadIdx.x] = 0;
        }
        if (threadIdx.x == 0) {
            s_bwd.gv = g_values ? g_values + c0 * (p.N + 1) : nullptr;
            s_bwd.gk = g_knots ? g_knots + c0 * (p.N + 1) : nullptr;
        }
        float xs, gs;
        sample<IO, CH>(p, c0, r0, r1, x, gy, xs, gs);
        build_tile<CH, true>(p, c0, cells, rec, &s_bwd.bad, [&] { add_exponents<CH>(gs); });
        if (threadIdx.x == 0 && s_bwd.bad) atomicOr(p.status, 1);
        const int F = fix_exponent<CH>(ch);
        bool slow = F == kNoSample;
        const float scale = slow ? 1.0f : exp2_int(F);
        if (threadIdx.x < CH) s_bwd.unit[ch] = slow ? 1.0f : exp2_int(-F);
        if (c0 + ch < p.C && !slow) slow = slow_sample<CH>(xs, gs, ChanConst<CH>(p, cells, rec, ch), scale);
        const bool flt = __syncthreads_count(slow) > kSlowSamples;
        for (int64_t r = r0; r < r1;) {
            const int64_t from = r;
            r = flt ? r1 : min(r1, r + kSegRows);
            if (flt)
                chan_bwd_rows_float<IO, CH>(p, c0, from, r, cells, rec, acc, x, gy, gx);
            else
                chan_bwd_rows<IO, CH, false>(p, c0, from, r, cells, rec, acc, scale, x, gy, gx);
            if (r == r1 || near_full<CH>(p, acc))
                flush_tile<CH>(p, c0, rec, acc, flt, r < r1 ? nullptr : reinterpret_cast<float*>(cells), g_values,
                               g_knots);
        }
    });
}

// ---- launch shapes -------------------------------------------------------------
// The sizes the calls accept are those of one CTA holding 8 channels' 16-byte
// cells, knots, values and slopes (forward) or 16 channels' 8-byte cells,
// 8-byte interval records, two sums and knots (backward), plus a little for
// scalars; every accepted size fits the tiles below (4 channels forward and 8
// backward take less for the same N and K).  Without k_cells, that index may shrink to
// its remainder of 16 cells.
size_t accepted_bytes(int64_t N, int64_t K, bool backward)
{
    const size_t n1 = (size_t)(N + 1), n2 = (size_t)(N + 2);
    if (!backward) return 128 * ((size_t)K + n1) + 200;
    return 128 * ((size_t)K + n2) + 128 * n2 + 64 * n1 + 392;
}

size_t tile_bytes(int64_t N, int64_t K, int CH, bool backward)
{
    const size_t recs = 16 * (size_t)(N + 2) * (size_t)CH * (backward ? 2 : 1);
    return recs + 8 * (size_t)std::max<int64_t>(K, stage_pitch((int)N)) * (size_t)CH;
}

// Shared memory of a CTA that leaves the L1 at least ~60 KB (a carve-out of
// 196 KB) for the rows in flight.
constexpr size_t kIndexBytes = 196 * 1024 - 1024 - 512;
constexpr int64_t kCells = 2;  // cells per knot where they fit

struct ChanShape {
    int CH, K;
    size_t smem;
};

// The widest tile whose index holds at least one cell per knot (or what the caller
// asked for) within kIndexBytes or, before the tile is narrowed, the whole shared
// memory: few cells and little L1 cost less than 32-byte row segments.
//   Forward, [65536, 2048] FP32: 16 channels up to N = 517 205-226 us, with all of the
//   shared memory up to 602 279, 8 channels up to 1036 313-318, with all up to 1206 374,
//   then 4 channels 666-726.  (With 2 cells per knot as the least: 288 from 388 on, 614
//   from 777.)
//   Backward, [65536, 4096]: 16 channels up to N = 309 780-798, with all up to 360 943,
//   8 channels up to 620 1258-1318, then with all 1540 (1245 from 258 on, 2530 from 518).
ChanShape choose_shape(int64_t N, int64_t k_cells, bool backward)
{
    const int64_t want = k_cells > 0 ? k_cells : kCells * (N + 1);
    const int64_t need = k_cells > 0 ? k_cells : N + 1;
    const size_t optin = device_info().smem_optin - 512, part = std::min(kIndexBytes, optin);
    const struct {
        int CH;
        size_t budget;
    } candidates[] = {{16, part}, {16, optin}, {8, part}, {8, optin}, {4, optin}};
    ChanShape s{};
    for (int i = 0; i < (backward ? 4 : 5); ++i) {  // (no accepted backward needs 4 channels)
        const auto& c = candidates[i];
        const size_t recs = 16 * (size_t)(N + 2) * (size_t)c.CH * (backward ? 2 : 1);
        const int64_t room = c.budget > recs ? (int64_t)((c.budget - recs) / (8 * (size_t)c.CH)) : 0;
        s.CH = c.CH;
        s.K = (int)std::min(want, std::max<int64_t>(room, 1));
        if (room >= std::max<int64_t>(need, stage_pitch((int)N))) break;
    }
    s.smem = tile_bytes(N, s.K, s.CH, backward);
    return s;
}

std::mutex g_cluster_mu;
std::map<std::tuple<int, const void*, int, size_t>, int> g_clusters;

// resident clusters of a kernel (a host call of several microseconds, cached)
cudaError_t cluster_count(const void* fn, const cudaLaunchConfig_t& cfg, int ctas, int* n)
{
    std::lock_guard<std::mutex> lk(g_cluster_mu);
    const auto key = std::make_tuple(device_info().device, fn, ctas, (size_t)cfg.dynamicSmemBytes);
    const auto it = g_clusters.find(key);
    if (it != g_clusters.end()) {
        *n = it->second;
        return cudaSuccess;
    }
    const cudaError_t e = cudaOccupancyMaxActiveClusters(n, fn, &cfg);
    if (e != cudaSuccess) return e;
    *n = std::max(*n, 1);
    g_clusters[key] = *n;
    return cudaSuccess;
}

template <typename... Args>
pwl_status launch(ChanArgs p, int CH, size_t smem, void (*kern)(const ChanArgs, Args...), cudaStream_t s,
                  Args... args)
{
    const void* fn = reinterpret_cast<const void*>(kern);
    PWL_CUDA_TRY(ensure_smem_limit(fn, smem));
    // a cluster covers a 128-byte line of a row (two CTAs for 16-channel BF16
    // tiles: four leave 8 of the 152 SMs without a cluster)
    p.cluster = CH == 16 ? 2 : (CH == 8 ? 4 : 8);
    cudaLaunchConfig_t cfg{};
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = p.cluster;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.blockDim = dim3(kChThreads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    cfg.gridDim = dim3(p.cluster);
    int clusters = 0;
    PWL_CUDA_TRY(cluster_count(fn, cfg, p.cluster, &clusters));
    const int64_t tiles = (p.C + CH - 1) / CH, groups = (tiles + p.cluster - 1) / p.cluster;
    p.passes = (p.R + kChThreads / CH - 1) / (kChThreads / CH);
    p.work = groups * p.passes;
    cfg.gridDim = dim3(p.cluster * (unsigned)std::min<int64_t>(clusters, p.work));
    PWL_CUDA_TRY(cudaLaunchKernelEx(&cfg, kern, p, args...));
    PWL_CHECK_LAUNCH("channels kernel");
    return PWL_OK;
}

template <typename IO>
pwl_status launch_forward(ChanArgs p, const ChanShape& sh, const void* x, void* y, cudaStream_t s)
{
    const IO* xi = static_cast<const IO*>(x);
    IO* yo = static_cast<IO*>(y);
    switch (sh.CH) {
    case 16: return launch(p, 16, sh.smem, channels_forward_kernel<IO, 16>, s, xi, yo);
    case 8: return launch(p, 8, sh.smem, channels_forward_kernel<IO, 8>, s, xi, yo);
    default: return launch(p, 4, sh.smem, channels_forward_kernel<IO, 4>, s, xi, yo);
    }
}

template <typename IO>
pwl_status launch_backward(ChanArgs p, const ChanShape& sh, const void* x, const void* gy, void* gx, float* g_values,
                           float* g_knots, cudaStream_t s)
{
    const IO *xi = static_cast<const IO*>(x), *gi = static_cast<const IO*>(gy);
    IO* go = static_cast<IO*>(gx);
    switch (sh.CH) {
    case 16:
        return launch(p, 16, sh.smem, channels_backward_kernel<IO, 16>, s, xi, gi, go, g_values, g_knots);
    default:
        return launch(p, 8, sh.smem, channels_backward_kernel<IO, 8>, s, xi, gi, go, g_values, g_knots);
    }
}

// Validates the arguments shared by both directions and fills p and the shape.
pwl_status setup(const float* knots, const float* values, int64_t C, int64_t N, int64_t R, int64_t k_cells,
                 int32_t* d_status, int32_t io_dtype, bool backward, ChanArgs& p, ChanShape& sh)
{
    if (!knots || !values) return fail(PWL_EINVAL, "knots / values is NULL");
    if (C < 1 || N < 1 || N > 65535) return fail(PWL_EINVAL, "need C >= 1 channels and 1 <= N <= 65535 intervals");
    if (R < 0) return fail(PWL_EINVAL, "rows must be >= 0");
    if (k_cells < 0 || k_cells > (1 << 20)) return fail(PWL_EINVAL, "k_cells must be in [0, 2^20]");
    if (!d_status) return fail(PWL_EINVAL, "status word is NULL");
    if (io_dtype != PWL_FP32 && io_dtype != PWL_BF16) return fail(PWL_EINVAL, "io dtype must be FP32 or BF16");
    if (R == 0) return PWL_OK;
    const size_t optin = device_info().smem_optin;
    const int64_t least = k_cells > 0 ? k_cells : ((backward ? 2 : 4) * (N + 1) - 1) % 16 + 1;
    if (accepted_bytes(N, least, backward) > optin)
        return fail(PWL_ENOTSUP, "a channel index of N = %lld intervals and %lld cells does not fit one CTA",
                    (long long)N, (long long)least);
    sh = choose_shape(N, k_cells, backward);
    p.knots = knots;
    p.values = values;
    p.C = C;
    p.R = R;
    p.N = (int)N;
    p.K = sh.K;
    p.status = d_status;
    return PWL_OK;
}

pwl_status backward(const float* knots, const float* values, int64_t C, int64_t N, int64_t k_cells, const void* x,
                    const void* gy, void* gx, float* g_values, float* g_knots, int64_t R, int32_t io_dtype,
                    int32_t* d_status, void* stream)
{
    ChanArgs p{};
    ChanShape sh{};
    const pwl_status st = setup(knots, values, C, N, R, k_cells, d_status, io_dtype, true, p, sh);
    if (st != PWL_OK || R == 0) return st;
    if (!x || !gy || !gx) return fail(PWL_EINVAL, "x / gy / gx is NULL");
    if (io_dtype == PWL_BF16)
        return launch_backward<__nv_bfloat16>(p, sh, x, gy, gx, g_values, g_knots, as_stream(stream));
    return launch_backward<float>(p, sh, x, gy, gx, g_values, g_knots, as_stream(stream));
}

}  // namespace

}  // namespace pwl

using namespace pwl;

extern "C" {

pwl_status pwl_channels_forward(const float* d_knots, const float* d_values, int64_t n_channels,
                                int64_t n_intervals, int64_t k_cells, const void* d_x, void* d_y, int64_t rows,
                                int32_t io_dtype, int32_t* d_status, void* stream)
{
    clear_error();
    ChanArgs p{};
    ChanShape sh{};
    const pwl_status st =
        setup(d_knots, d_values, n_channels, n_intervals, rows, k_cells, d_status, io_dtype, false, p, sh);
    if (st != PWL_OK || rows == 0) return st;
    if (!d_x || !d_y) return fail(PWL_EINVAL, "x / y is NULL");
    if (io_dtype == PWL_BF16) return launch_forward<__nv_bfloat16>(p, sh, d_x, d_y, as_stream(stream));
    return launch_forward<float>(p, sh, d_x, d_y, as_stream(stream));
}

pwl_status pwl_channels_backward(const float* d_knots, const float* d_values, int64_t n_channels,
                                 int64_t n_intervals, int64_t k_cells, const float* d_x, const float* d_gy,
                                 float* d_gx, float* d_g_values, float* d_g_knots, int64_t rows, int32_t* d_status,
                                 void* stream)
{
    clear_error();
    return backward(d_knots, d_values, n_channels, n_intervals, k_cells, d_x, d_gy, d_gx, d_g_values, d_g_knots, rows,
                    PWL_FP32, d_status, stream);
}

pwl_status pwl_channels_backward_bf16(const float* d_knots, const float* d_values, int64_t n_channels,
                                      int64_t n_intervals, int64_t k_cells, const void* d_x, const void* d_gy,
                                      void* d_gx, float* d_g_values, float* d_g_knots, int64_t rows,
                                      int32_t* d_status, void* stream)
{
    clear_error();
    return backward(d_knots, d_values, n_channels, n_intervals, k_cells, d_x, d_gy, d_gx, d_g_values, d_g_knots, rows,
                    PWL_BF16, d_status, stream);
}

}  // extern "C"
