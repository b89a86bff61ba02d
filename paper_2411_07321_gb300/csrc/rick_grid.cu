// rick_grid.cu -- convolutional gridding (Eq. 3 of De Rubeis et al.) and its
// adjoint, degridding.
//
// Plain gridding: one warp per work item = (subtile of one w-plane, chunk of at
// most sub_cap records).  The warp sums the footprints of its records -- every
// corner in the 16 x 16 cells of the subtile -- into (16 + W - 1)^2 cells of its
// own in shared memory, with plain loads and stores (up to W = 3 with adds), and adds
// the cells it reached to the planes (16-byte reductions in L2) onto tiles cleared
// before.  Eight chunks of a subtile are a CTA's, summed over its warps first; a dense
// subtile's sums meet in slots of its own.
//
// Compensated and deterministic gridding: one CTA per work item = (uv-tile of
// one w-plane, chunk of at most chunk_cap records).  The CTA owns the T x T
// output cells of its tile: it sums
// into a shared-memory accumulator the records binned at the tile (footprint
// corner inside it) and the records of the west / north / north-west tiles
// whose footprints reach into it (their edge classes), each clipped to the
// tile, then writes the tile once with plain coalesced stores.  The
// checkerboard (-1)^(i+j) of the centred FFT is applied in that write.  A tile
// with more than one chunk is zeroed first and its chunks add their sums with
// float2 atomics.  Tiles without records are not gridding items: the
// persistent gridding CTAs clear them in groups between their gridding items,
// so the stores of zeros overlap the gridding of the other tiles.
//
// Degridding: one CTA per chunk of a non-empty tile's own bin; the CTA stages
// the (T + W - 1)^2 plane region its records can touch into shared memory and
// each thread gathers one record's W x W footprint.
#include "rick_common.cuh"

struct GridArgs {
    TileArgs t;
    float2 *planes;
    int log2T;
    int accumulate;  // add into the planes instead of overwriting them
    const uint8_t *touched;  // per tile: add into it (tiles an earlier chunk gridded), or NULL
    uint32_t nzero;  // tile-clearing items (RICK_ZERO_GROUP tiles each) where every tile has
                     // to be written, else 0 (plain sums: only whether)
    SubShape sub;            // plain sums: subtiles, their record offsets, the work items
    const uint32_t *suboff;
    const uint2 *items;
    const uint4 *groups;
    float2 *slots;  // sums of dense subtiles
    uint32_t *arrived;
    uint32_t nslots;
    const uint32_t *mcslot;     // deterministic mode: slot of each multi-item tile
    unsigned long long *mcacc;  // deterministic mode: the slots' int64 (re, im) sums
};

// Accumulation modes: FP32 sums (one warp per subtile), FP32 rounds
// folded by compensated summation, or 64-bit fixed point (deterministic: the
// sums do not depend on the order of the atomics).
#define GM_PLAIN 0
#define GM_COMP 1
#define GM_DET 2

// Tiles per clearing item of the grid kernel.
#define RICK_ZERO_GROUP 8

struct DegridArgs {
    TileArgs t;
    const float2 *planes;
    const float *weight;
    float2 *vis_out;
    int log2T;
};

// Largest t in [0, ntiles) with base[t] <= b (base non-decreasing).
__device__ __forceinline__ uint32_t find_tile(const uint32_t *base, uint32_t ntiles, uint32_t b)
{
    uint32_t lo = 0, hi = ntiles;
    while (hi - lo > 1) {
        uint32_t mid = (lo + hi) >> 1;
        if (base[mid] <= b)
            lo = mid;
        else
            hi = mid;
    }
    return lo;
}

// Neumaier's compensated summation of a into (s, c).
__device__ __forceinline__ void neumaier(float &s, float &c, float a)
{
    float t = s + a;
    if (fabsf(s) >= fabsf(a))
        c += (s - t) + a;
    else
        c += (a - t) + s;
    s = t;
}

// ------------------------------------------------------------------------
// Record streams.  A group of W consecutive lanes walks a contiguous run of
// records; lane j of the group owns footprint row j (W cells).  Per record,
// lane j evaluates kernel segment j at both offsets -- gx[j] = G((j - h) - fx)
// and gy[j] = G((j - h) - fy), one Horner chain on (x, y) pairs with packed
// two-wide FP32 FMAs and the segment's coefficients held (duplicated) in the
// lane's registers -- so it already has its row's v weight, scales the
// visibility by it, and takes the W u weights from its group with shuffles:
// W shuffles and W packed FMAs per record and lane (re and im of two cells per
// instruction pair).  While consecutive records share
// the footprint corner (the channels of one baseline-time land on the same
// cells) the row sums stay in registers; when the corner changes the group
// adds its rows to the tile accumulator at once -- one row per lane, so the
// group's atomics never collide.

// A record stream is a group of G consecutive lanes, lane j owning footprint
// row j < W.  G is the power of two next to W when that packs as many groups
// into a warp as W lanes would (W = 7: four groups either way, and the lane
// arithmetic is shifts), else W itself (W = 9: three groups of nine instead of
// two of sixteen).  A warp holds NG = 32 / G groups; its last 32 - NG G lanes
// stay idle.
template <int W>
struct StreamShape {
    static constexpr int P2 = W <= 1 ? 1 : W <= 2 ? 2 : W <= 4 ? 4 : W <= 8 ? 8 : 16;
    static constexpr int G = (32 / P2 == 32 / W) ? P2 : W;
    static constexpr int NG = 32 / G;
    static constexpr int LIVE = NG * G;  // lanes of a warp that carry a stream
};

// The cells a subtile's footprints reach, and the stride of their rows in shared
// memory: odd, so that the lanes of a group, one row each, access 8-byte cells in
// distinct bank pairs.
template <int W>
struct SubCells {
    static constexpr int ROWS = (1 << RICK_SUB_LOG) + W - 1, STRIDE = ROWS | 1;
    static constexpr int CELLS = ROWS * STRIDE;
};

// Warps of a gridding CTA (256 threads).
#define RICK_GRID_WARPS 8

// The lane's row sums into the tile accumulator: fb is the index of the row's
// first cell, bit jx of fv says whether column jx lies inside the tile (fv = 0
// when the row is outside it or the lane carries no row).  Both are set once
// per footprint corner, so the loop over records carries two registers for
// the flush instead of the corner's geometry.
template <int W>
__device__ __forceinline__ void group_flush(float *acc_re, float *acc_im, int fb, uint32_t fv,
                                            const float *ar, const float *ai)
{
    if (!fv) return;
#pragma unroll
    for (int jx = 0; jx < W; ++jx) {
        if ((fv >> jx) & 1u) {
            atomicAdd(&acc_re[fb + jx], ar[jx]);
            atomicAdd(&acc_im[fb + jx], ai[jx]);
        }
    }
}

// The lane's row sums into its warp's cells, fb the index of the row's first one.
// No other warp writes them, and the groups of the warp take turns.
template <int W>
__device__ __forceinline__ void warp_flush(float2 *cells, int fb, const float *ar, const float *ai)
{
    float2 *p = cells + fb;
    float2 o[W];
#pragma unroll
    for (int jx = 0; jx < W; ++jx) o[jx] = p[jx];
#pragma unroll
    for (int jx = 0; jx < W; ++jx) p[jx] = make_float2(o[jx].x + ar[jx], o[jx].y + ai[jx]);
}

// The same while the other groups add theirs, two float adds a cell.
template <int W>
__device__ __forceinline__ void warp_flush_atomic(float2 *cells, int fb, const float *ar,
                                                  const float *ai)
{
    float *p = (float *)(cells + fb);
#pragma unroll
    for (int jx = 0; jx < W; ++jx) {
        atomicAdd(p + 2 * jx, ar[jx]);
        atomicAdd(p + 2 * jx + 1, ai[jx]);
    }
}

// The same into the 64-bit fixed-point tile: each row sum scaled by 2^k and
// rounded to an integer, then added with integer atomics (exact, so the tile
// does not depend on the order in which the groups flush).
template <int W>
__device__ __forceinline__ void group_flush_det(unsigned long long *acc64, float fx, int T, int TP,
                                                int lx, int row, bool live, const float *ar,
                                                const float *ai)
{
    if (!live || (unsigned)row >= (unsigned)T) return;
#pragma unroll
    for (int jx = 0; jx < W; ++jx) {
        int col = lx + jx;
        if ((unsigned)col < (unsigned)T) {
            int i = 2 * (row * TP + col);
            atomicAdd(&acc64[i], (unsigned long long)__float2ll_rn(ar[jx] * fx));
            atomicAdd(&acc64[i + 1], (unsigned long long)__float2ll_rn(ai[jx] * fx));
        }
    }
}

// Asynchronous copies global -> shared (cp.async): 16 or 4 bytes, both
// addresses aligned to the size.
__device__ __forceinline__ void cp_async16(void *sdst, const void *gsrc)
{
    const unsigned d = (unsigned)__cvta_generic_to_shared(sdst);
    asm volatile("cp.async.ca.shared.global [%0], [%1], 16;\n" ::"r"(d), "l"(gsrc) : "memory");
}
__device__ __forceinline__ void cp_async4(void *sdst, const void *gsrc)
{
    const unsigned d = (unsigned)__cvta_generic_to_shared(sdst);
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;\n" ::"r"(d), "l"(gsrc) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;\n" ::: "memory"); }
// all but the most recently committed group have landed (for this thread)
__device__ __forceinline__ void cp_async_wait1() { asm volatile("cp.async.wait_group 1;\n" ::: "memory"); }
__device__ __forceinline__ void cp_async_wait0() { asm volatile("cp.async.wait_group 0;\n" ::: "memory"); }

// Record ring of a warp: where a warp carries at most three record streams
// (W >= 9), the streams' next records are staged in shared memory by the whole
// warp, RICK_GRID_RB records per stream per chunk, two chunks in flight, so that
// the record loop reads them from shared memory instead of waiting on global
// loads one record ahead.  With four streams (W = 7) the loads that the ring
// would save are shared by more records a step, and it measured slower (5e7
// visibilities: 1.16 -> 1.24 ms; plain loads two records ahead: 1.34).
#define RICK_GRID_RB 16

template <int W>
struct RecRing {
    static constexpr bool ON = W > 1 && StreamShape<W>::NG <= 3;
    static constexpr int NG = StreamShape<W>::NG;
    static constexpr int SLOTS = ON ? NG * RICK_GRID_RB : 1;  // records per chunk and warp
};

// Copy chunk c of the warp's streams (iterations c RB ... c RB + RB - 1; past
// a stream's end its last record again) into buffer c & 1 of the ring.  Slot
// e = lane + 32 h holds record e % RB of stream e / RB, whose first record and
// last index are cr0[h] and clast[h].
template <int W>
__device__ __forceinline__ void ring_issue(const TileArgs &ta, float4 *wrec, uint32_t *wcel,
                                           uint32_t c, const uint32_t *cr0, const uint32_t *clast)
{
    constexpr int RB = RICK_GRID_RB, SLOTS = RecRing<W>::SLOTS;
#pragma unroll
    for (int h = 0; h < (SLOTS + 31) / 32; ++h) {
        const int e = (threadIdx.x & 31) + 32 * h;
        if (e < SLOTS) {
            const uint32_t idx = cr0[h] + min(c * RB + (uint32_t)(e % RB), clast[h]);
            const int slot = (int)(c & 1u) * SLOTS + e;
            cp_async16(wrec + slot, ta.rec + idx);
            cp_async4(wcel + slot, ta.rcell + idx);
        }
    }
    cp_async_commit();
}

// n records of one segment of the tile's record list, starting at record r0.
// DET: the flushes go to the 64-bit fixed-point tile acc64 (scale fx).
template <int W, bool DET>
__device__ __forceinline__ void grid_stream(const TileArgs &ta, uint32_t r0, uint32_t n,
                                            uint32_t ntrip, int x0,
                                            int y0, float *acc_re, float *acc_im, int T, int TP,
                                            const float2 *coef2, unsigned long long *acc64,
                                            float fx)
{
    constexpr int G = StreamShape<W>::G;
    const int lane = threadIdx.x & 31, grp = lane / G;
    const int j = lane - grp * G;  // this lane's row / kernel segment
    const bool live = lane < StreamShape<W>::LIVE && j < W && n > 0;
    if (ntrip == 0) return;
    const uint32_t last = n > 0 ? n - 1 : 0;
    float ar[W], ai[W];
#pragma unroll
    for (int jx = 0; jx < W; ++jx) ar[jx] = ai[jx] = 0.0f;
    const float4 *rec = ta.rec + r0;
    const uint32_t *rcell = ta.rcell + r0;
    // the warp's record ring: chunk c of every stream of the warp in buffer c & 1
    using Ring = RecRing<W>;
    constexpr int RB = RICK_GRID_RB, NGR = Ring::NG;
    __shared__ __align__(16) float4 s_rrec[Ring::ON ? RICK_GRID_WARPS * 2 * Ring::SLOTS : 1];
    __shared__ uint32_t s_rcel[Ring::ON ? RICK_GRID_WARPS * 2 * Ring::SLOTS : 1];
    float4 *wrec = s_rrec + (Ring::ON ? (threadIdx.x >> 5) * 2 * Ring::SLOTS : 0);
    uint32_t *wcel = s_rcel + (Ring::ON ? (threadIdx.x >> 5) * 2 * Ring::SLOTS : 0);
    const int rg = grp < NGR ? grp : NGR - 1;  // the stream this lane reads (idle lanes: any)
    // this lane's slots of a chunk (e = lane + 32 h): record rr of stream g,
    // whose first record and last index come from the stream's first lane
    constexpr int NH = (Ring::SLOTS + 31) / 32;
    uint32_t cr0[NH], clast[NH];
#pragma unroll
    for (int h = 0; h < NH; ++h) {
        const int e = (threadIdx.x & 31) + 32 * h, g = min(e / RB, NGR - 1);
        cr0[h] = Ring::ON ? __shfl_sync(0xffffffffu, r0, g * G) : 0u;
        clast[h] = Ring::ON ? __shfl_sync(0xffffffffu, last, g * G) : 0u;
    }
    auto ring_at = [&](uint32_t i) { return (int)((i / RB) & 1u) * Ring::SLOTS + rg * RB + (int)(i % RB); };
    uint32_t cur;
    float4 q;
    int ri = 0;  // ring slot of the record being read (running: reset at chunk starts)
    if constexpr (Ring::ON) {
        ring_issue<W>(ta, wrec, wcel, 0, cr0, clast);
        ring_issue<W>(ta, wrec, wcel, 1, cr0, clast);
        cp_async_wait1();
        __syncwarp();
        ri = ring_at(0);
        q = wrec[ri];
        cur = wcel[ri];
    } else {
        cur = rcell[0];
        q = rec[0];
    }
    uint32_t cell = cur;
    // the flush target of corner cur (group_flush)
    int fb;
    uint32_t fv;
    auto target = [&](uint32_t c) {
        const int lx = (int)(c & 0xFFFFu) - x0, row = (int)(c >> 16) - y0 + j;
        fb = row * TP + lx;
        uint32_t m = 0;
#pragma unroll
        for (int jx = 0; jx < W; ++jx) m |= ((unsigned)(lx + jx) < (unsigned)T ? 1u : 0u) << jx;
        fv = (live && (unsigned)row < (unsigned)T) ? m : 0u;
    };
    target(cur);
    for (uint32_t i = 0; i < ntrip; ++i) {
        // the next record; past the stream's end the last one again
        float4 nq;
        uint32_t ncell;
        if constexpr (Ring::ON) {
            const uint32_t i1 = i + 1;
            if (i1 % RB == 0) {
                if (i1 < ntrip) {
                    // entering chunk c = i1 / RB: the warp is done with chunk c - 1
                    // (record i was read last iteration), so its buffer takes chunk
                    // c + 1; chunk c has landed once only that copy is pending
                    __syncwarp();
                    ring_issue<W>(ta, wrec, wcel, i1 / RB + 1, cr0, clast);
                    cp_async_wait1();
                    __syncwarp();
                }
                ri = ring_at(i1);
            } else {
                ++ri;
            }
            nq = wrec[ri];
            ncell = wcel[ri];
        } else {
            const uint32_t ln = min(i + 1, last);
            nq = rec[ln];
            ncell = rcell[ln];
        }
        if (cell != cur) {
            if (DET)
                group_flush_det<W>(acc64, fx, T, TP, (int)(cur & 0xFFFFu) - x0,
                                   (int)(cur >> 16) - y0 + j, live, ar, ai);
            else
                group_flush<W>(acc_re, acc_im, fb, fv, ar, ai);
#pragma unroll
            for (int jx = 0; jx < W; ++jx) ar[jx] = ai[jx] = 0.0f;
            cur = cell;
            target(cur);
        }
        float gx = 1.0f, gy = 1.0f;
        if (W > 1) {
            const float2 s2 = make_float2(2.0f * (q.z - ta.kp.fc), 2.0f * (q.w - ta.kp.fc));
            float2 g2 = coef2[RICK_POLY_DEG];
#pragma unroll
            for (int k = RICK_POLY_DEG - 1; k >= 0; --k) g2 = __ffma2_rn(g2, s2, coef2[k]);
            gx = g2.x;
            gy = g2.y;
        }
        const float gz = i < n ? gy : 0.0f;
        const float2 vv = __fmul2_rn(make_float2(q.x, q.y), make_float2(gz, gz));
        const float2 vr2 = make_float2(vv.x, vv.x), vi2 = make_float2(vv.y, vv.y);
        float wv[W];
#pragma unroll
        for (int jx = 0; jx < W; ++jx) {
            // power-of-two groups: the lane inside the group is an immediate
            // (width form); groups of W lanes: the absolute lane
            wv[jx] = W == 1 ? gx
                   : (G & (G - 1)) == 0 ? __shfl_sync(0xffffffffu, gx, jx, G)
                                        : __shfl_sync(0xffffffffu, gx, grp * G + jx);
        }
#pragma unroll
        for (int jx = 0; jx + 1 < W; jx += 2) {
            const float2 w2 = make_float2(wv[jx], wv[jx + 1]);
            const float2 a2 = __ffma2_rn(vr2, w2, make_float2(ar[jx], ar[jx + 1]));
            const float2 b2 = __ffma2_rn(vi2, w2, make_float2(ai[jx], ai[jx + 1]));
            ar[jx] = a2.x; ar[jx + 1] = a2.y;
            ai[jx] = b2.x; ai[jx + 1] = b2.y;
        }
        if (W & 1) {
            ar[W - 1] = __fmaf_rn(vv.x, wv[W - 1], ar[W - 1]);
            ai[W - 1] = __fmaf_rn(vv.y, wv[W - 1], ai[W - 1]);
        }
        q = nq;
        cell = ncell;
    }
    if (DET)
        group_flush_det<W>(acc64, fx, T, TP, (int)(cur & 0xFFFFu) - x0, (int)(cur >> 16) - y0 + j,
                           live, ar, ai);
    else
        group_flush<W>(acc_re, acc_im, fb, fv, ar, ai);
    if constexpr (Ring::ON) {
        // the copies still in flight land before the ring is used again
        cp_async_wait0();
        __syncwarp();
    }
}

template <int W, int MODE>
__device__ __forceinline__ void tile_item(const GridArgs &a, uint32_t b, uint32_t t, float *sm,
                                          const float2 *coef2)
{
    constexpr bool COMP = MODE == GM_COMP, DET = MODE == GM_DET;
    const TileArgs &ta = a.t;
    const uint32_t chunk = b - ta.base[t], nch = ta.base[t + 1] - ta.base[t];
    const int T = 1 << a.log2T, TP = T + 1, TT = T * TP, nt = ta.nt;
    const uint32_t tx = t % nt, ty = (t / nt) % nt, k = t / (nt * nt);
    const int x0 = tx << a.log2T, y0 = ty << a.log2T;
    const uint32_t *off = ta.offsets;

    // the four record ranges that can touch this tile: its own bin, and the
    // edge classes of the west, north and north-west bins that reach into it
    uint32_t rs[4], rl[4];
    rs[0] = off[4 * t];
    rl[0] = off[4 * t + 4] - rs[0];
    rs[1] = rl[1] = rs[2] = rl[2] = rs[3] = rl[3] = 0;
    if (tx > 0) {
        rs[1] = off[4 * (t - 1) + 1];
        rl[1] = off[4 * (t - 1) + 3] - rs[1];
    }
    if (ty > 0) {
        rs[2] = off[4 * (t - nt) + 2];
        rl[2] = off[4 * (t - nt) + 4] - rs[2];
    }
    if (tx > 0 && ty > 0) {
        rs[3] = off[4 * (t - nt - 1) + 2];
        rl[3] = off[4 * (t - nt - 1) + 3] - rs[3];
    }
    const uint32_t Ltot = rl[0] + rl[1] + rl[2] + rl[3];
    // the ranges in shared memory, for a loop over them that is not unrolled
    // (one copy of the record loop keeps the kernel small)
    __shared__ uint32_t s_rs[4], s_rl[4];
    if (threadIdx.x < 4) {
        s_rs[threadIdx.x] = rs[threadIdx.x];
        s_rl[threadIdx.x] = rl[threadIdx.x];
    }
    const uint32_t cap = ta.hdr->chunk_cap;
    const uint32_t vbeg = chunk * cap;
    const uint32_t vend = min(Ltot, vbeg + cap);

    // accumulators with padded rows (stride T + 1): the lanes of a group own
    // different rows, which then fall in different banks
    float *acc_re = sm, *acc_im = sm + TT;
    float *sum_re = sm + 2 * TT, *sum_im = sm + 3 * TT, *cmp_re = sm + 4 * TT, *cmp_im = sm + 5 * TT;
    unsigned long long *acc64 = (unsigned long long *)sm;  // DET: (re, im) pairs
    const float fx = DET ? ta.hdr->fx_scale : 0.0f;
    for (int i = threadIdx.x; i < TT; i += blockDim.x) {
        if (DET) {
            acc64[2 * i] = 0ull;
            acc64[2 * i + 1] = 0ull;
        } else {
            acc_re[i] = 0.0f;
            acc_im[i] = 0.0f;
        }
        if (COMP) sum_re[i] = sum_im[i] = cmp_re[i] = cmp_im[i] = 0.0f;
    }
    __syncthreads();

    // deterministic: one round over the chunk; compensated: rounds of 4096 records,
    // each folded into the (sum, compensation) pair of every cell.  The
    // round's piece of each of the four ranges is split evenly into one
    // contiguous run per record stream, so the streams of a warp always walk
    // the same range with runs of equal length (a split of the whole round
    // would let a warp's streams straddle a range boundary, and the warp then
    // walks both ranges one after the other).
    constexpr int NG = StreamShape<W>::NG;
    const int lane = threadIdx.x & 31;
    const bool streaming = lane < StreamShape<W>::LIVE;
    const uint32_t nstreams = (blockDim.x >> 5) * NG;
    const uint32_t stream = (threadIdx.x >> 5) * NG + (streaming ? lane / StreamShape<W>::G : 0);
    const uint32_t round = COMP ? 4096u : max(vend - vbeg, 1u);
    for (uint32_t rb = vbeg; rb < vend; rb += round) {
        const uint32_t re = min(vend, rb + round);
        uint32_t base = 0;
#pragma unroll 1
        for (int g = 0; g < 4; ++g) {
            const uint32_t lg = s_rl[g];
            const uint32_t a0 = max(rb, base), a1 = min(re, base + lg);
            if (a0 < a1) {
                const uint32_t per = (a1 - a0 + nstreams - 1) / nstreams;
                const uint32_t v0 = min(a0 + stream * per, a1), v1 = min(v0 + per, a1);
                const uint32_t nv = streaming ? v1 - v0 : 0u;
                grid_stream<W, DET>(ta, s_rs[g] + ((nv ? v0 : a0) - base), nv, per, x0, y0,
                                     acc_re, acc_im, T, TP, coef2, acc64, fx);
            }
            base += lg;
        }
        if (COMP) {
            __syncthreads();
            for (int i = threadIdx.x; i < TT; i += blockDim.x) {
                neumaier(sum_re[i], cmp_re[i], acc_re[i]);
                neumaier(sum_im[i], cmp_im[i], acc_im[i]);
                acc_re[i] = 0.0f;
                acc_im[i] = 0.0f;
            }
            __syncthreads();
        }
    }
    if (!COMP) __syncthreads();

    // flush: (-1)^(i+j) folded in; plain stores unless the tile has several chunks
    const int n = ta.n;
    float2 *plane = a.planes + (size_t)k * n * n;
    if (DET && nch > 1) {  // several work items: exact integer sums in the tile's slot
        unsigned long long *slot = a.mcacc + (size_t)a.mcslot[t] * 2 * T * T;
        for (int i = threadIdx.x; i < T * T; i += blockDim.x) {
            const int ip = (i >> a.log2T) * TP + (i & (T - 1));
            const unsigned long long re = acc64[2 * ip], im = acc64[2 * ip + 1];
            if (re) atomicAdd(&slot[2 * i], re);
            if (im) atomicAdd(&slot[2 * i + 1], im);
        }
        return;
    }
    const float fxi = DET ? ta.hdr->fx_inv : 0.0f;
    const bool acc = a.accumulate || (a.touched && a.touched[t]);
    for (int i = threadIdx.x; i < T * T; i += blockDim.x) {
        int row = i >> a.log2T, col = i & (T - 1), ip = row * TP + col;
        int gi = x0 + col, gj = y0 + row;
        float re = DET ? __ll2float_rn((long long)acc64[2 * ip]) * fxi
                 : COMP ? sum_re[ip] + cmp_re[ip] : acc_re[ip];
        float im = DET ? __ll2float_rn((long long)acc64[2 * ip + 1]) * fxi
                 : COMP ? sum_im[ip] + cmp_im[ip] : acc_im[ip];
        if ((gi + gj) & 1) {
            re = -re;
            im = -im;
        }
        float2 *dst = plane + (size_t)gj * n + gi;
        if (nch == 1 && !acc) {
            *dst = make_float2(re, im);
        } else if (nch == 1) {  // the only writer of this tile in this launch
            float2 o = *dst;
            *dst = make_float2(o.x + re, o.y + im);
        } else if (re != 0.0f || im != 0.0f) {
            atomicAdd(dst, make_float2(re, im));
        }
    }
}

// Clear the tiles of group z that have no work item (no records reach them):
// 16-byte stores, the CTA's threads striding over the tile.
__device__ __forceinline__ void zero_group(const GridArgs &a, uint32_t z)
{
    const TileArgs &ta = a.t;
    const int T = 1 << a.log2T, half = T >> 1, nt = ta.nt, n = ta.n;
    const uint32_t t1 = min(ta.ntiles, (z + 1) * RICK_ZERO_GROUP);
    for (uint32_t t = z * RICK_ZERO_GROUP; t < t1; ++t) {
        if (ta.base[t + 1] != ta.base[t]) continue;
        const uint32_t tx = t % nt, ty = (t / nt) % nt, k = t / (nt * nt);
        float4 *plane = (float4 *)(a.planes + (size_t)k * n * n);
        for (int i = threadIdx.x; i < T * half; i += blockDim.x) {
            const int row = i / half, col2 = i - row * half;
            plane[((size_t)((ty << a.log2T) + row) * n + (tx << a.log2T)) / 2 + col2] =
                make_float4(0.f, 0.f, 0.f, 0.f);
        }
    }
}

// This lane's kernel segment (= its footprint row within its group).
template <int W, bool PIN = true>
__device__ __forceinline__ void load_coef(const KernelPoly &kp, float2 *coef2)
{
    const int seg = min((int)((threadIdx.x & 31) % StreamShape<W>::G), W - 1);
#pragma unroll
    for (int k = 0; k < RICK_POLY_N; ++k) {
        coef2[k] = make_float2(kp.c[seg][k], kp.c[seg][k]);
        // opaque from here on: the compiler would rather read them again in every
        // step than keep them, and a lane-indexed constant load is a replay per row
        if (PIN) asm volatile("" : "+f"(coef2[k].x), "+f"(coef2[k].y));
    }
}

// Persistent: one wave of CTAs takes work items (tile, chunk) from a counter
// in the workspace header (reset by zero_tiles_kernel, launched just before),
// and with each a clearing item for a group of tiles without records, so that
// the HBM-bound clearing of the empty tiles runs under the issue-bound
// gridding of the others.
template <int W, int MODE>
__global__ void __launch_bounds__(32 * RICK_GRID_WARPS, 3) grid_kernel(GridArgs a)
{
    extern __shared__ float sm[];
    __shared__ uint32_t s_b, s_tile, s_z;
    const uint32_t total = a.t.base[a.t.ntiles];
    float2 coef2[RICK_POLY_N];
    load_coef<W, false>(a.t.kp, coef2);
    for (;;) {
        if (threadIdx.x == 0) {
            const uint32_t b = atomicAdd(&a.t.hdr->grid_next, 1u);
            s_b = b;
            s_tile = b < total ? find_tile(a.t.base, a.t.ntiles, b) : 0u;
            s_z = a.nzero ? atomicAdd(&a.t.hdr->zero_next, 1u) : 0u;
        }
        __syncthreads();
        const uint32_t b = s_b, t = s_tile, z = s_z;
        __syncthreads();  // everyone has the item before thread 0 takes the next
        if (b >= total && z >= a.nzero) break;
        if (b < total) {
            tile_item<W, MODE>(a, b, t, sm, coef2);
            __syncthreads();  // the accumulator is reused by the next item
        }
        if (z < a.nzero) zero_group(a, z);
    }
}

// Plane and first cell of a subtile.
struct SubOrigin {
    int k, x0, y0;
};
__device__ __forceinline__ SubOrigin sub_origin(const GridArgs &a, uint32_t id)
{
    const SubShape &sub = a.sub;
    const uint32_t q = 1u << sub.lq, tile = id >> (2 * sub.lq), nt = a.t.nt, row = tile / nt;
    return {(int)(row / nt), (int)(((tile - row * nt) << sub.log2T) + ((id & (q - 1)) << sub.ls)),
            (int)((row % nt << sub.log2T) + ((id >> sub.lq & (q - 1)) << sub.ls))};
}

// n records, r0 ... r0 + n - 1, in ntrip >= n steps (the same for every lane of the
// warp) into the warp's cells; fbase: index of this lane's footprint row for a
// corner at (0, 0).  As grid_stream, but for the flush.
template <int W>
__device__ __forceinline__ void warp_stream(const TileArgs &ta, uint32_t r0, uint32_t n,
                                            uint32_t ntrip, int fbase, const float2 *coef2,
                                            float2 *cells)
{
    constexpr int G = StreamShape<W>::G, NGR = StreamShape<W>::NG, ST = SubCells<W>::STRIDE;
    // Up to W = 3 a warp has ten groups and more, and taking turns costs more than the few
    // compare-and-swap loops of a row.  Gridding of 4e6 visibilities of one channel /
    // 1e7 of 16, adds against turns: W = 3 218 / 192 against 236 / 182 us, W = 4 290 / 209
    // against 259 / 185, W = 5 398 / 292 against 310 / 238, W = 6 507 / 346 against 358 /
    // 271.
    constexpr bool ATOMIC = NGR > 8;
    using Ring = RecRing<W>;
    constexpr int RB = RICK_GRID_RB, NH = (Ring::SLOTS + 31) / 32;
    __shared__ __align__(16) float4 s_rrec[Ring::ON ? RICK_GRID_WARPS * 2 * Ring::SLOTS : 1];
    __shared__ uint32_t s_rcel[Ring::ON ? RICK_GRID_WARPS * 2 * Ring::SLOTS : 1];
    const int lane = threadIdx.x & 31;
    const int grp = lane / G, j = lane - grp * G, rg = grp < NGR ? grp : NGR - 1;
    const int lead = grp * G;
    const bool live = lane < StreamShape<W>::LIVE && j < W && n > 0;
    const uint32_t last = r0 + (n > 0 ? n - 1 : 0);  // absolute, as is r
    float ar[W], ai[W];
#pragma unroll
    for (int jx = 0; jx < W; ++jx) ar[jx] = ai[jx] = 0.0f;
    float4 *wrec = s_rrec + (Ring::ON ? (threadIdx.x >> 5) * 2 * Ring::SLOTS : 0);
    uint32_t *wcel = s_rcel + (Ring::ON ? (threadIdx.x >> 5) * 2 * Ring::SLOTS : 0);
    uint32_t cr0[NH], clast[NH];
#pragma unroll
    for (int h = 0; h < NH; ++h) {
        const int g = min((lane + 32 * h) / RB, NGR - 1);
        cr0[h] = Ring::ON ? __shfl_sync(0xffffffffu, r0, g * G) : 0u;
        clast[h] = Ring::ON ? __shfl_sync(0xffffffffu, last - r0, g * G) : 0u;
    }
    // ring slot of the stream's record i (idle lanes read any stream)
    auto ring_at = [&](uint32_t i) {
        return (int)((i / RB) & 1u) * Ring::SLOTS + rg * RB + (int)(i % RB);
    };
    uint32_t r = r0, cur;
    float4 q;
    int ri = 0;
    if constexpr (Ring::ON) {
        ring_issue<W>(ta, wrec, wcel, 0, cr0, clast);
        ring_issue<W>(ta, wrec, wcel, 1, cr0, clast);
        cp_async_wait1();
        __syncwarp();
        ri = ring_at(0);
        q = wrec[ri];
        cur = wcel[ri];
    } else {
        q = ta.rec[r];
        cur = ta.rcell[r];
    }
    uint32_t cell = cur;
    // (unrolled by two, the ring's loop gains 3.5 % at W = 9, the other loses as much)
#pragma unroll(Ring::ON ? 2 : 1)
    for (uint32_t i = 0; i < ntrip; ++i) {
        // the next record; past the stream's end the last one again
        float4 nq;
        uint32_t ncell;
        const bool in = i < n;
        if constexpr (Ring::ON) {
            const uint32_t i1 = i + 1;
            if (i1 % RB == 0) {
                if (i1 < ntrip) {
                    // entering chunk c = i1 / RB: the warp is done with chunk c - 1
                    // (record i was read last iteration), so its buffer takes chunk
                    // c + 1; chunk c has landed once only that copy is pending
                    __syncwarp();
                    ring_issue<W>(ta, wrec, wcel, i1 / RB + 1, cr0, clast);
                    cp_async_wait1();
                    __syncwarp();
                }
                ri = ring_at(i1);
            } else {
                ++ri;
            }
            nq = wrec[ri];
            ncell = wcel[ri];
        } else {
            r = min(r + 1, last);
            nq = __ldg(ta.rec + r);
            ncell = __ldg(ta.rcell + r);
        }
        const bool turn = cell != cur;
        if (ATOMIC) {
            if (turn) {
                if (live) warp_flush_atomic<W>(cells, (int)((cur >> 16) * ST + (cur & 0xFFFFu)) + fbase, ar, ai);
#pragma unroll
                for (int jx = 0; jx < W; ++jx) ar[jx] = ai[jx] = 0.0f;
                cur = cell;
            }
        } else if (__any_sync(0xffffffffu, turn)) {
            // the groups that change corner, one after the other: footprints of two
            // groups may overlap
            unsigned m = __ballot_sync(0xffffffffu, turn && live && j == 0);
            while (m) {
                if (live && grp * G == __ffs(m) - 1)
                    warp_flush<W>(cells, (int)((cur >> 16) * ST + (cur & 0xFFFFu)) + fbase, ar, ai);
                __syncwarp();
                m &= m - 1;
            }
            if (turn) {
#pragma unroll
                for (int jx = 0; jx < W; ++jx) ar[jx] = ai[jx] = 0.0f;
                cur = cell;
            }
        }
        float gx = 1.0f, gy = 1.0f;
        if (W > 1) {
            const float2 s2 = make_float2(2.0f * (q.z - ta.kp.fc), 2.0f * (q.w - ta.kp.fc));
            float2 g2 = coef2[RICK_POLY_DEG];
#pragma unroll
            for (int k = RICK_POLY_DEG - 1; k >= 0; --k) g2 = __ffma2_rn(g2, s2, coef2[k]);
            gx = g2.x;
            gy = g2.y;
        }
        const float gz = in ? gy : 0.0f;
        const float2 vv = __fmul2_rn(make_float2(q.x, q.y), make_float2(gz, gz));
        const float2 vr2 = make_float2(vv.x, vv.x), vi2 = make_float2(vv.y, vv.y);
        float wv[W];
#pragma unroll
        for (int jx = 0; jx < W; ++jx) {
            // power-of-two groups: the lane inside the group is an immediate
            // (width form); groups of W lanes: the absolute lane
            wv[jx] = W == 1 ? gx
                   : (G & (G - 1)) == 0 ? __shfl_sync(0xffffffffu, gx, jx, G)
                                        : __shfl_sync(0xffffffffu, gx, grp * G + jx);
        }
#pragma unroll
        for (int jx = 0; jx + 1 < W; jx += 2) {
            const float2 w2 = make_float2(wv[jx], wv[jx + 1]);
            const float2 a2 = __ffma2_rn(vr2, w2, make_float2(ar[jx], ar[jx + 1]));
            const float2 b2 = __ffma2_rn(vi2, w2, make_float2(ai[jx], ai[jx + 1]));
            ar[jx] = a2.x; ar[jx + 1] = a2.y;
            ai[jx] = b2.x; ai[jx + 1] = b2.y;
        }
        if (W & 1) {
            ar[W - 1] = __fmaf_rn(vv.x, wv[W - 1], ar[W - 1]);
            ai[W - 1] = __fmaf_rn(vv.y, wv[W - 1], ai[W - 1]);
        }
        q = nq;
        cell = ncell;
    }
#pragma unroll 1
    for (int h = 0; h < (ATOMIC ? 1 : NGR); ++h) {
        if (ATOMIC && live)
            warp_flush_atomic<W>(cells, (int)((cur >> 16) * ST + (cur & 0xFFFFu)) + fbase, ar, ai);
        if (!ATOMIC && live && grp == h)
            warp_flush<W>(cells, (int)((cur >> 16) * ST + (cur & 0xFFFFu)) + fbase, ar, ai);
        __syncwarp();
    }
    if constexpr (Ring::ON) {
        // the copies still in flight land before the ring is used again
        cp_async_wait0();
        __syncwarp();
    }
}

// Chunk `chunk` of a subtile's records into the warp's cells.
template <int W>
__device__ __forceinline__ void grid_chunk(const GridArgs &a, uint32_t id, uint32_t chunk,
                                           float2 *cells, const float2 *coef2)
{
    constexpr int NG = StreamShape<W>::NG;
    const SubShape &sub = a.sub;
    const int lane = threadIdx.x & 31;
    // the subtile's up to four record ranges, lane g holding range g
    uint32_t rs = 0, rl = 0;
    if (lane < 4) {
        const int64_t rid = rick_subtile_range(sub, id, lane);
        if (rid >= 0) {
            rs = a.suboff[rid];
            rl = a.suboff[rid + 1] - rs;
        }
    }
    uint32_t n = rl + __shfl_xor_sync(0xffffffffu, rl, 1);
    n += __shfl_xor_sync(0xffffffffu, n, 2);
    n = __shfl_sync(0xffffffffu, n, 0);
    const uint32_t nch = rick_sub_chunks(n, a.t.hdr->sub_cap), len = (n + nch - 1) / nch;
    const uint32_t vbeg = chunk * len, vend = min(vbeg + len, n);
    const SubOrigin so = sub_origin(a, id);
    const int fbase = (lane % StreamShape<W>::G - so.y0) * SubCells<W>::STRIDE - so.x0;
    const bool streaming = lane < StreamShape<W>::LIVE;
    const uint32_t stream = streaming ? lane / StreamShape<W>::G : 0;
    uint32_t base = 0;
#pragma unroll 1
    for (int g = 0; g < 4; ++g) {
        const uint32_t s = __shfl_sync(0xffffffffu, rs, g), l = __shfl_sync(0xffffffffu, rl, g);
        const uint32_t a0 = max(vbeg, base), a1 = min(vend, base + l);
        if (a0 < a1) {
            // split evenly into one run per stream
            const uint32_t per = (a1 - a0 + NG - 1) / NG;
            const uint32_t v0 = min(a0 + stream * per, a1), v1 = min(v0 + per, a1);
            const uint32_t nv = streaming ? v1 - v0 : 0u;
            warp_stream<W>(a.t, s + ((nv ? v0 : a0) - base), nv, per, fbase, coef2, cells);
        }
        base += l;
    }
}

// Tile t of the planes zeroed by threads i of n_threads, 16 bytes a store.
__device__ __forceinline__ void clear_tile(float2 *planes, uint32_t t, int nt, int log2T, int n,
                                           int i, int n_threads)
{
    const uint32_t tx = t % nt, ty = t / nt % nt, k = t / nt / nt;
    float4 *tile = (float4 *)(planes + ((size_t)k * n + (ty << log2T)) * n + (tx << log2T));
    const int lh = log2T - 1;  // float4 = two cells
    for (; i < 1 << (log2T + lh); i += n_threads)
        tile[(size_t)(i >> lh) * (n / 2) + (i & ((1 << lh) - 1))] = make_float4(0.f, 0.f, 0.f, 0.f);
}

// The tiles of [t0, t1) without records zeroed by the warp.
__device__ __forceinline__ void clear_empty(const GridArgs &a, uint32_t t0, uint32_t t1)
{
    for (uint32_t t = t0; t < min(t1, a.t.ntiles); ++t)
        if (a.t.base[t + 1] == a.t.base[t])
            clear_tile(a.planes, t, a.t.nt, a.log2T, a.t.n, threadIdx.x & 31, 32);
}

// Two cells of a subtile's row, col even, added to its cells in the planes or a slot (row
// stride n) -- the checkerboard (-1)^(i+j) folded in (the subtile's first row and column
// are even); nothing where both are zero, as cells are that no footprint reached, those
// off the grid among them.
__device__ __forceinline__ void add_cells(float2 *out, int n, int row, int col, float2 u, float2 v)
{
    if (u.x != 0.0f || u.y != 0.0f || v.x != 0.0f || v.y != 0.0f) {
        if (row & 1) {
            u.x = -u.x;
            u.y = -u.y;
        } else {
            v.x = -v.x;
            v.y = -v.y;
        }
        atomicAdd((float4 *)(out + (size_t)row * n + col), make_float4(u.x, u.y, v.x, v.y));
    }
}

__device__ __forceinline__ float2 *sub_cells(const GridArgs &a, uint32_t id)
{
    const SubOrigin so = sub_origin(a, id);
    return a.planes + ((size_t)so.k * a.t.n + so.y0) * a.t.n + so.x0;
}

// The sums of nc sets of a subtile's cells (strides of SubCells::CELLS) added to
// out and the cells zeroed, by threads t of nt: two cells of a row at a time.
template <int W>
__device__ __forceinline__ void cells_out(float2 *out, int n, float2 *cells, int nc, int t, int nt)
{
    constexpr int ROWS = SubCells<W>::ROWS, ST = SubCells<W>::STRIDE, HP = (ROWS + 1) / 2;
    // (By two, items of a few records take a fifth less -- 1e6 visibilities spread over
    // 1e5 subtiles, W = 4 / 9: 247 -> 201, 432 -> 396 us -- but at W = 7 the record loop
    // comes out 3 to 5 % slower: 4e6 visibilities of one channel, 339 -> 356.)
#pragma unroll(W == 7 ? 1 : 2)
    for (int i = t; i < ROWS * HP; i += nt) {
        const int row = i / HP, col = 2 * (i - row * HP);
        const bool two = ROWS % 2 == 0 || col + 1 < ROWS;
        float2 u = make_float2(0.0f, 0.0f), v = u;
#pragma unroll 2
        for (int c = 0; c < nc; ++c) {
            float2 *p = cells + c * SubCells<W>::CELLS + row * ST + col;
            u = __fadd2_rn(u, p[0]);
            p[0] = make_float2(0.0f, 0.0f);
            if (two) {
                v = __fadd2_rn(v, p[1]);
                p[1] = make_float2(0.0f, 0.0f);
            }
        }
        add_cells(out, n, row, col, u, v);
    }
}

// The work of the plain kernels: groups, a CTA each, then single items, a warp each,
// `take` at a time.  A CTA begins with the group of its own number, and the warps of a
// CTA beyond the groups with single items of their own; only what is left is handed out
// by counters, whose atomics pass one by one (3.5 ns each: with one counter that every
// warp asks, 1e5 items of a few records took 380 us, and the last requests of 4864 warps
// 17 us).  A warp asks one of RICK_ITEM_COUNTERS, each for every RICK_ITEM_COUNTERS-th
// `take` items.
//
// And the CTA's group: the subtile, its slot (~0: the planes), the subtile's first slot
// and number of groups, its job of a batch; and whether it was the last of its subtile's
// to arrive.
struct PlainWork {
    uint32_t total[2];  // groups and single items of all jobs
    uint32_t take, idle;  // idle: CTAs without a group
    uint32_t clear;       // tiles to look at per warp and item
    uint32_t index, id, slot, first, all;
    int job;
    bool last;
};

__device__ __forceinline__ void start_work(volatile PlainWork &w, uint32_t groups, uint32_t singles)
{
    const uint32_t share = singles / (gridDim.x * RICK_GRID_WARPS);
    w.total[0] = groups;
    w.total[1] = singles;
    w.take = share >= 64 ? 8u : share >= 16 ? 4u : 1u;
    w.idle = groups < gridDim.x ? gridDim.x - groups : 0u;
    w.index = ~0u;
    w.slot = ~0u;
}

// The slots of a subtile whose groups have all arrived added up and to the planes.
template <int W>
__device__ __forceinline__ void slots_out(const GridArgs &a, const volatile PlainWork &g)
{
    constexpr int ROWS = SubCells<W>::ROWS, HP = (ROWS + 1) / 2;
    const uint32_t ns = rick_sub_slots(g.all);
    const float2 *first = a.slots + (size_t)g.first * RICK_SLOT_CELLS;
    float2 *out = sub_cells(a, g.id);
    for (int i = threadIdx.x; i < ROWS * HP; i += 32 * RICK_GRID_WARPS) {
        const int row = i / HP, col = 2 * (i - row * HP);
        const float4 *p = (const float4 *)(first + row * RICK_SLOT_STRIDE + col);
        double s[4] = {0.0, 0.0, 0.0, 0.0};
#pragma unroll 4
        for (uint32_t k = 0; k < ns; ++k) {
            const float4 v = __ldcg(p + k * (RICK_SLOT_CELLS / 2));
            s[0] += v.x;
            s[1] += v.y;
            s[2] += v.z;
            s[3] += v.w;
        }
        // (signed for the checkerboard already; no footprint reaches a zero cell)
        if (s[0] != 0.0 || s[1] != 0.0 || s[2] != 0.0 || s[3] != 0.0)
            atomicAdd((float4 *)(out + (size_t)row * a.t.n + col),
                      make_float4((float)s[0], (float)s[1], (float)s[2], (float)s[3]));
    }
}

// The next group, for the whole CTA; total[0] or more after the last.  Counts the one
// before in at its subtile's slots, and sends them to the planes if it was the last.
template <int W, typename Jobs>
__device__ __forceinline__ uint32_t next_group(const Jobs &jobs, volatile PlainWork &g)
{
    __syncthreads();  // the cells are zero again, the last item has been read
    if (threadIdx.x == 0) {
        g.index = g.index == ~0u ? blockIdx.x
                : g.idle == 0 ? gridDim.x + atomicAdd(&jobs.hdr()->group_next, 1u) : ~0u - 1;
        g.last = false;
        if (g.slot != ~0u) {
            __threadfence();  // the CTA's sums before its count
            g.last = atomicAdd(&jobs.args(g.job).arrived[g.first], 1u) == g.all - 1;
        }
    }
    __syncthreads();
    if (g.last) {
        __threadfence();
        slots_out<W>(jobs.args(g.job), g);
        __syncthreads();
    }
    return g.index;
}

// The warp's next single item after its last one (~0: none yet); ~0 after the last.
__device__ __forceinline__ uint32_t next_single(WsHeader *hdr, const volatile PlainWork &w,
                                                uint32_t last)
{
    const uint32_t total = w.total[1], take = w.take, idle = w.idle, wid = threadIdx.x >> 5;
    uint32_t b = last + 1;
    if (last == ~0u && gridDim.x - blockIdx.x <= idle) {
        b = (wid * idle + gridDim.x - 1 - blockIdx.x) * take;
    } else if (last == ~0u || b % take == 0) {
        const uint32_t first = RICK_GRID_WARPS * idle;
        if (first * take >= total) return ~0u;
        const uint32_t k = (blockIdx.x * RICK_GRID_WARPS + wid) % RICK_ITEM_COUNTERS;
        if ((threadIdx.x & 31) == 0)
            b = (first + k + RICK_ITEM_COUNTERS * atomicAdd(&hdr->item_next[k][0], 1u)) * take;
        b = __shfl_sync(0xffffffffu, b, 0);
    }
    return b < total ? b : ~0u;
}

// The counters are in the workspace header (reset by zero_tiles_kernel, launched just
// before).
//
// CLEAR: also zero the tiles without records, a share of them with every item, so that
// the HBM-bound clearing runs under the issue-bound gridding (as a launch of its own / so:
// 5e7 visibilities on 32 planes of 8192^2, W = 9, 4.48 / 3.56 ms; 2e7 on 16 of 4096^2,
// W = 7, 869 / 762 us); at the start where there are fewer items than would keep every
// warp at it.
template <int W, bool CLEAR, typename Jobs>
__device__ __forceinline__ void plain_work(const Jobs &jobs, float2 *cells)
{
    // (what the sums go to waits in shared memory: the record loop needs the registers)
    __shared__ volatile uint32_t s_id[RICK_GRID_WARPS], s_slot[RICK_GRID_WARPS],
        s_item[RICK_GRID_WARPS];
    __shared__ volatile PlainWork s_work;
    const int wid = threadIdx.x >> 5;
    for (int i = threadIdx.x; i < RICK_GRID_WARPS * SubCells<W>::CELLS; i += 32 * RICK_GRID_WARPS)
        cells[i] = make_float2(0.0f, 0.0f);
    if (threadIdx.x == 0) start_work(s_work, jobs.total(false), jobs.total(true));
    s_item[wid] = ~0u;
    if (CLEAR) {
        __syncthreads();
        const GridArgs &a = jobs.args(0);
        const uint32_t warps = gridDim.x * RICK_GRID_WARPS;
        const uint32_t items = s_work.total[0] * RICK_GRID_WARPS + s_work.total[1];
        if (items >= 2 * warps) {
            if (threadIdx.x == 0) s_work.clear = (a.t.ntiles + items - 1) / items;
        } else {
            if (threadIdx.x == 0) s_work.clear = 0;
            for (uint32_t t = blockIdx.x * RICK_GRID_WARPS + wid; t < a.t.ntiles; t += warps)
                clear_empty(a, t, t + 1);
        }
    }
    float2 coef2[RICK_POLY_N];
    load_coef<W>(jobs.args(0).t.kp, coef2);
    int cur = 0;
    bool single = false;
#pragma unroll 1
    for (;;) {
        uint32_t b = 0, id, chunk, slot = ~0u;
        if (!single) {
            b = next_group<W>(jobs, s_work);
            single = b >= s_work.total[0];
        }
        if (single) {
            b = next_single(jobs.hdr(), s_work, s_item[wid]);
            if (b == ~0u) break;
            __syncwarp();
            s_item[wid] = b;
        }
        const int j = jobs.job(b, single);
        if (single) {
            const uint2 q = jobs.args(j).items[b - jobs.first(j, true)];
            id = q.x;
            chunk = q.y;
        } else {
            const uint4 q = jobs.args(j).groups[b - jobs.first(j, false)];
            id = q.x;
            chunk = q.y + wid;
            if (q.z != ~0u) slot = q.z + q.y / RICK_SUB_GROUP % rick_sub_slots(q.w);
            if (threadIdx.x == 0) {
                s_work.job = j;
                s_work.id = id;
                s_work.slot = slot;
                s_work.first = q.z;
                s_work.all = q.w;
            }
        }
        const GridArgs &a = jobs.args(j);
        if (j != cur) load_coef<W>(a.t.kp, coef2);
        cur = j;
        s_id[wid] = id;
        s_slot[wid] = slot;
        float2 *own = cells + wid * SubCells<W>::CELLS;
        grid_chunk<W>(a, id, chunk, own, coef2);
        if (single) {
            __syncwarp();
            cells_out<W>(sub_cells(a, s_id[wid]), a.t.n, own, 1, threadIdx.x & 31, 32);
        } else {
            __syncthreads();
            slot = s_slot[wid];
            cells_out<W>(slot == ~0u ? sub_cells(a, s_id[wid])
                                     : a.slots + (size_t)slot * RICK_SLOT_CELLS,
                         slot == ~0u ? a.t.n : RICK_SLOT_STRIDE, cells, RICK_GRID_WARPS,
                         threadIdx.x, 32 * RICK_GRID_WARPS);
        }
        if (CLEAR) {
            const uint32_t per = s_work.clear;
            const uint32_t i = single ? s_work.total[0] * RICK_GRID_WARPS + s_item[wid]
                                      : s_work.index * RICK_GRID_WARPS + wid;
            clear_empty(a, i * per, (i + 1) * per);
        }
        __syncwarp();
    }
}

// One job (job 0).
struct OneJob {
    const GridArgs &a;
    __device__ __forceinline__ const GridArgs &args(int) const { return a; }
    __device__ __forceinline__ WsHeader *hdr() const { return a.t.hdr; }
    __device__ __forceinline__ uint32_t total(bool single) const
    {
        return single ? a.t.hdr->n_items : a.t.hdr->n_groups;
    }
    __device__ __forceinline__ int job(uint32_t, bool) const { return 0; }
    __device__ __forceinline__ uint32_t first(int, bool) const { return 0; }
};

// Plain sums.
//
// Bound by instruction issue (62 % of cycles; long_scoreboard, the record loads,
// is the first stall).  A warp owns its cells, so a corner change costs W loads
// and stores of 8 bytes a lane, and only the groups meet at barriers; summing a
// 64 x 64 tile per CTA took 2 W compare-and-swap loops a lane there (shared memory
// has no FP32 add) and visited the records near a tile's edge once per tile they
// reach.  16 x 16 corners a subtile leave 32 warps an SM.  On a GB300, against the
// CTA tiles: 5e7 visibilities of 16 channels, W = 7: 1.92 -> 1.27 ms; 2e8 of 64,
// W = 9: 9.21 -> 6.57; 1e7 of 4: 0.68 -> 0.36; 4e6 of one: 0.61 -> 0.34; 1e6 of 4:
// 106 -> 57 us; 1e4: 58 -> 17 us.  Four CTAs an SM up to W = 10, where 64 registers
// spill: long runs want the warps, short ones do not (four / three, W = 9: 2e8 of 64
// channels 6.57 / 6.80 ms, 6e6 of 64 247 / 240 us, 4e6 of one 591 / 548, 1e7 of 16 431 /
// 419; W = 10: 634 / 588, 457 / 436).  From W = 11 three (W = 11 at four: 386 / 407).
template <int W, bool CLEAR>
__global__ void __launch_bounds__(32 * RICK_GRID_WARPS, W <= 10 ? 4 : 3)
    grid_warps_kernel(const __grid_constant__ GridArgs a)
{
    extern __shared__ float2 s_cells[];
    plain_work<W, CLEAR>(OneJob{a}, s_cells);
}

// Several imaging jobs gridded by one launch (rick_grid_sparse_batch): the jobs'
// work items form one list, job after job, taken from one counter (the first
// job's).  Every job has the same support W and tile T, and plain FP32 sums.
// RICK_GRID_BATCH_MAX (rick.h) jobs at most: the arguments travel as one
// kernel parameter.

struct GridBatchArgs {
    int n_jobs;
    GridArgs job[RICK_GRID_BATCH_MAX];
};
static_assert(sizeof(GridBatchArgs) <= 32764, "kernel parameters are limited to 32764 bytes");

// The slots of the last binning's dense subtiles zeroed, by block b of nb.
__device__ __forceinline__ void clear_slots(const WsHeader *hdr, float2 *slots, uint32_t *arrived,
                                            uint32_t nslots, uint32_t b, uint32_t nb)
{
    const uint32_t used = min(hdr->n_slots, nslots), first = b * blockDim.x + threadIdx.x;
    for (uint32_t i = first; i < used * (RICK_SLOT_CELLS / 2); i += nb * blockDim.x)
        ((float4 *)slots)[i] = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
    for (uint32_t i = first; i < used; i += nb * blockDim.x) arrived[i] = 0;
}

#define RICK_ZERO_LOOK 8

// Zero the tiles of at least `least` work items, into which the grid kernel adds,
// before it runs, and reset its counters: least = 2 for the compensated kernel
// (a tile's only item stores it), 1 for the plain one.  Where every tile has to be
// written, the grid kernels clear the tiles without records.  When gridding adds into
// existing planes nothing is cleared, and neither are the tiles flagged in touched (a
// chunk of a streamed set adds into the tiles earlier chunks gridded).
// Deterministic mode (mcacc != NULL): the int64 slots of those tiles are
// zeroed instead, accumulating or not (the slots are added into the planes
// after gridding).
__global__ void __launch_bounds__(256) zero_tiles_kernel(const uint32_t *base, uint32_t ntiles,
                                                         int nt, int log2T, int n, float2 *planes,
                                                         WsHeader *hdr, int accumulate,
                                                         const uint32_t *mcslot,
                                                         unsigned long long *mcacc,
                                                         const uint8_t *touched, uint32_t least,
                                                         float2 *slots, uint32_t *arrived,
                                                         uint32_t nslots)
{
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        hdr->grid_next = 0;
        hdr->zero_next = 0;
        hdr->group_next = 0;
    }
    if (blockIdx.x == 0 && threadIdx.x < RICK_ITEM_COUNTERS) hdr->item_next[threadIdx.x][0] = 0;
    const int lane = threadIdx.x & 31, T = 1 << log2T;
    if (nslots) clear_slots(hdr, slots, arrived, nslots, blockIdx.x, gridDim.x);
    if (!mcacc && accumulate) return;
    // a block looks at RICK_ZERO_LOOK tiles at a time, and its warps share the rows
    // of each one to clear: the tiles with records lie side by side
    for (uint32_t t0 = blockIdx.x * RICK_ZERO_LOOK; t0 < ntiles; t0 += gridDim.x * RICK_ZERO_LOOK) {
        const uint32_t tl = t0 + lane;
        unsigned m = __ballot_sync(0xffffffffu, lane < RICK_ZERO_LOOK && tl < ntiles &&
                                                    base[tl + 1] - base[tl] >= least &&
                                                    !(!mcacc && touched && touched[tl]));
        for (; m; m &= m - 1) {
            const uint32_t t = t0 + __ffs(m) - 1;
            if (!mcacc) {
                clear_tile(planes, t, nt, log2T, n, threadIdx.x, blockDim.x);
                continue;
            }
            ulonglong2 *slot = (ulonglong2 *)(mcacc + (size_t)mcslot[t] * 2 * T * T);
            for (int i = threadIdx.x; i < T * T; i += blockDim.x)
                slot[i] = make_ulonglong2(0ull, 0ull);
        }
    }
}

// The batch's tiles with records zeroed (one row of CTAs per job, blockIdx.y) and
// its item counter reset.
__global__ void __launch_bounds__(256)
    zero_tiles_batch_kernel(const __grid_constant__ GridBatchArgs ba)
{
    const GridArgs &a = ba.job[blockIdx.y];
    const TileArgs &ta = a.t;
    if (blockIdx.x == 0 && blockIdx.y == 0) {
        if (threadIdx.x == 0) ta.hdr->group_next = 0;
        if (threadIdx.x < RICK_ITEM_COUNTERS) ta.hdr->item_next[threadIdx.x][0] = 0;
    }
    const int lane = threadIdx.x & 31;
    clear_slots(ta.hdr, a.slots, a.arrived, a.nslots, blockIdx.x, gridDim.x);
    for (uint32_t t0 = blockIdx.x * RICK_ZERO_LOOK; t0 < ta.ntiles;
         t0 += gridDim.x * RICK_ZERO_LOOK) {
        const uint32_t tl = t0 + lane;
        unsigned m = __ballot_sync(0xffffffffu, lane < RICK_ZERO_LOOK && tl < ta.ntiles &&
                                                    ta.base[tl + 1] != ta.base[tl]);
        for (; m; m &= m - 1) clear_tile(a.planes, t0 + __ffs(m) - 1, ta.nt, a.log2T, ta.n, threadIdx.x,
                       blockDim.x);
    }
}

// The jobs of a batch: entry b of the jobs' lists belongs to the job j with
// cum[j] <= b < cum[j + 1] (cum: running totals of the jobs' entries), and is that job's
// entry b - cum[j].
struct BatchJobs {
    const GridBatchArgs &ba;
    const uint32_t (*cum)[RICK_GRID_BATCH_MAX + 1];
    __device__ __forceinline__ const GridArgs &args(int j) const { return ba.job[j]; }
    __device__ __forceinline__ WsHeader *hdr() const { return ba.job[0].t.hdr; }
    __device__ __forceinline__ uint32_t total(bool single) const { return cum[single][ba.n_jobs]; }
    __device__ __forceinline__ int job(uint32_t b, bool single) const
    {
        int j = 0;
        while (j + 1 < ba.n_jobs && cum[single][j + 1] <= b) ++j;
        return j;
    }
    __device__ __forceinline__ uint32_t first(int j, bool single) const { return cum[single][j]; }
};

// As grid_warps_kernel over the batch's work.
template <int W>
__global__ void __launch_bounds__(32 * RICK_GRID_WARPS, W <= 10 ? 4 : 3)
    grid_batch_kernel(const __grid_constant__ GridBatchArgs ba)
{
    extern __shared__ float2 s_cells[];
    __shared__ uint32_t s_cum[2][RICK_GRID_BATCH_MAX + 1];
    if (threadIdx.x < 2) {
        uint32_t c = 0;
        s_cum[threadIdx.x][0] = 0;
        for (int j = 0; j < ba.n_jobs; ++j) {
            const WsHeader *h = ba.job[j].t.hdr;
            c += threadIdx.x ? h->n_items : h->n_groups;
            s_cum[threadIdx.x][j + 1] = c;
        }
    }
    __syncthreads();
    plain_work<W, false>(BatchJobs{ba, s_cum}, s_cells);
}

// Deterministic mode: the tiles gridded by several work items, from their
// int64 slots into the planes (written, or added with accumulate), the
// checkerboard (-1)^(i+j) folded in.  A block per tile (a warp: 61 us for the few
// dense tiles of 2e6 visibilities).
__global__ void __launch_bounds__(256) det_mc_convert_kernel(const uint32_t *base, uint32_t ntiles,
                                                             int nt, int log2T, int n,
                                                             float2 *planes, const WsHeader *hdr,
                                                             int accumulate,
                                                             const uint32_t *mcslot,
                                                             const unsigned long long *mcacc)
{
    const int lane = threadIdx.x & 31, T = 1 << log2T;
    const float inv = hdr->fx_inv;
    for (uint32_t t0 = blockIdx.x * RICK_ZERO_LOOK; t0 < ntiles; t0 += gridDim.x * RICK_ZERO_LOOK) {
        const uint32_t tl = t0 + lane;
        unsigned m = __ballot_sync(0xffffffffu, lane < RICK_ZERO_LOOK && tl < ntiles &&
                                                    base[tl + 1] - base[tl] > 1);
        for (; m; m &= m - 1) {
            const uint32_t t = t0 + __ffs(m) - 1;
            const uint32_t tx = t % nt, ty = (t / nt) % nt, k = t / (nt * nt);
            const unsigned long long *slot = mcacc + (size_t)mcslot[t] * 2 * T * T;
            float2 *plane = planes + (size_t)k * n * n;
            for (int i = threadIdx.x; i < T * T; i += blockDim.x) {
                const int row = i >> log2T, col = i & (T - 1);
                const int gi = (int)(tx << log2T) + col, gj = (int)(ty << log2T) + row;
                float re = __ll2float_rn((long long)slot[2 * i]) * inv;
                float im = __ll2float_rn((long long)slot[2 * i + 1]) * inv;
                if ((gi + gj) & 1) {
                    re = -re;
                    im = -im;
                }
                float2 *dst = plane + (size_t)gj * n + gi;
                if (accumulate) {
                    const float2 o = *dst;
                    re += o.x;
                    im += o.y;
                }
                *dst = make_float2(re, im);
            }
        }
    }
}

// n_src: with the Hermitian mirror the inputs (records from n_src on mirror
// input i - n_src), else 0.
template <int W>
__device__ __forceinline__ void degrid_item(const DegridArgs &a, uint32_t b, uint32_t t,
                                            float2 *stage, uint32_t n_src)
{
    const TileArgs &ta = a.t;
    const uint32_t chunk = b - ta.base[t];
    const int T = 1 << a.log2T, S = T + W - 1, nt = ta.nt, n = ta.n;
    const uint32_t tx = t % nt, ty = (t / nt) % nt, k = t / (nt * nt);
    const int x0 = tx << a.log2T, y0 = ty << a.log2T;
    const uint32_t cap = ta.hdr->chunk_cap;
    const uint32_t r0 = ta.offsets[4 * t] + chunk * cap;
    const uint32_t r1 = min(ta.offsets[4 * t + 4], r0 + cap);

    const float2 *plane = a.planes + (size_t)k * n * n;
    for (int i = threadIdx.x; i < S * S; i += blockDim.x) {
        int row = i / S, col = i - row * S;
        int gi = x0 + col, gj = y0 + row;
        float2 v = make_float2(0.f, 0.f);
        if (gi < n && gj < n) {
            v = plane[(size_t)gj * n + gi];
            if ((gi + gj) & 1) {
                v.x = -v.x;
                v.y = -v.y;
            }
        }
        stage[i] = v;
    }
    __syncthreads();
    for (uint32_t r = r0 + threadIdx.x; r < r1; r += blockDim.x) {
        const float4 q = ta.rec[r];
        const float2 fr = make_float2(q.z, q.w);
        uint32_t cell = ta.rcell[r];
        int lx = (int)(cell & 0xFFFFu) - x0, ly = (int)(cell >> 16) - y0;
        float gx[W], gy[W];
        kernel_weights<W>(ta.kp, fr.x, gx);
        kernel_weights<W>(ta.kp, fr.y, gy);
        float sr = 0.f, si = 0.f;
#pragma unroll
        for (int jy = 0; jy < W; ++jy) {
            const float2 *rowp = stage + (ly + jy) * S + lx;
            float rr = 0.f, ri = 0.f;
#pragma unroll
            for (int jx = 0; jx < W; ++jx) {
                float2 c = rowp[jx];
                rr = fmaf(gx[jx], c.x, rr);
                ri = fmaf(gx[jx], c.y, ri);
            }
            sr = fmaf(gy[jy], rr, sr);
            si = fmaf(gy[jy], ri, si);
        }
        const uint32_t m = ta.perm[r];
        if (n_src == 0) {
            const float wt = a.weight ? a.weight[m] : 1.0f;
            a.vis_out[m] = make_float2(sr * wt, si * wt);
        } else {
            // the Hermitian mirror: input m' gets its record's value plus the
            // conjugate of its mirrored record's (two adds onto zero, so the
            // result does not depend on their order)
            const bool mir = m >= n_src;
            const uint32_t src = mir ? m - n_src : m;
            const float wt = a.weight ? a.weight[src] : 1.0f;
            atomicAdd(&a.vis_out[src], make_float2(sr * wt, mir ? -si * wt : si * wt));
        }
    }
}

template <int W>
__global__ void __launch_bounds__(256) degrid_kernel(DegridArgs a)
{
    extern __shared__ float2 stage[];
    __shared__ uint32_t s_b, s_tile;
    const uint32_t total = a.t.base[a.t.ntiles];
    const uint32_t n_src = a.t.hdr->mirror ? (uint32_t)a.t.hdr->n_src : 0u;
    for (;;) {
        if (threadIdx.x == 0) {
            uint32_t b = atomicAdd(&a.t.hdr->degrid_next, 1u);
            s_b = b;
            s_tile = b < total ? find_tile(a.t.base, a.t.ntiles, b) : 0u;
        }
        __syncthreads();
        const uint32_t b = s_b, t = s_tile;
        if (b >= total) break;
        degrid_item<W>(a, b, t, stage, n_src);
        __syncthreads();
    }
}

// Dropped visibilities (key == all ones) get a zero model value.  With the
// Hermitian mirror every output is zeroed: both records of an input add into it.
__global__ void degrid_zero_dropped_kernel(WsHeader *hdr, const uint32_t *key, float2 *vis_out)
{
    if (blockIdx.x == 0 && threadIdx.x == 0) hdr->degrid_next = 0;
    const bool all = hdr->mirror != 0;
    int64_t n = (int64_t)(all ? hdr->n_src : hdr->n_vis);
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n;
         i += (int64_t)gridDim.x * blockDim.x)
        if (all || key[i] == 0xFFFFFFFFu) vis_out[i] = make_float2(0.f, 0.f);
}

// ------------------------------------------------------------------------

static TileArgs make_tile_args(const rick_plan *plan, const WsPtrs &w, const uint32_t *base)
{
    const rick_params &p = plan->p;
    TileArgs t;
    t.n = p.n;
    t.n_w = p.n_w;
    t.T = p.tile;
    t.nt = p.n / p.tile;
    t.W = p.support;
    t.ntiles = (uint32_t)p.n_w * t.nt * t.nt;
    t.offsets = w.offsets;
    t.base = base;
    t.perm = w.perm;
    t.rcell = w.rcell;
    t.rec = w.rec;
    t.hdr = w.hdr;
    t.kp = plan->poly;
    return t;
}

static void set_sub_args(GridArgs &a, const rick_params &p, const WsPtrs &w, const WsLayout &L)
{
    a.sub = rick_sub_shape(&p);
    a.suboff = w.suboff;
    a.items = w.items;
    a.groups = w.groups;
    a.slots = w.slots;
    a.arrived = w.arrived;
    a.nslots = (uint32_t)L.nslots;
}

static int ilog2(int x)
{
    int l = 0;
    while ((1 << l) < x) ++l;
    return l;
}

// One wave of persistent CTAs: SMs x resident CTAs per SM.
template <typename K>
static unsigned persistent_blocks(K kernel, size_t smem, int num_sms)
{
    int per_sm = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kernel, 256, smem) != cudaSuccess ||
        per_sm < 1)
        per_sm = 1;
    return (unsigned)(per_sm * num_sms);
}

template <int W, int MODE>
static cudaError_t launch_grid_t(const GridArgs &a, int num_sms, cudaStream_t st)
{
    // float words: six T (T + 1) arrays, or four of 64-bit sums
    const int words = MODE == GM_COMP ? 6 : 4;
    size_t smem = words * (size_t)a.t.T * (a.t.T + 1) * sizeof(float);
    cudaFuncSetAttribute(grid_kernel<W, MODE>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                         (int)smem);
    grid_kernel<W, MODE><<<persistent_blocks(grid_kernel<W, MODE>, smem, num_sms), 32 * RICK_GRID_WARPS,
                              smem, st>>>(a);
    return cudaGetLastError();
}

template <int W>
static size_t warps_smem()
{
    return RICK_GRID_WARPS * sizeof(float2) * SubCells<W>::CELLS;
}

template <int W>
static cudaError_t launch_grid(const GridArgs &a, int mode, int num_sms, cudaStream_t st)
{
    if (mode == GM_COMP) return launch_grid_t<W, GM_COMP>(a, num_sms, st);
    if (mode == GM_DET) return launch_grid_t<W, GM_DET>(a, num_sms, st);
    const size_t smem = warps_smem<W>();
    const auto kernel = a.nzero ? grid_warps_kernel<W, true> : grid_warps_kernel<W, false>;
    cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)smem);
    if (e != cudaSuccess) return e;
    kernel<<<persistent_blocks(kernel, smem, num_sms), 32 * RICK_GRID_WARPS, smem, st>>>(a);
    return cudaGetLastError();
}

template <int W>
static cudaError_t launch_degrid(const DegridArgs &a, int num_sms, cudaStream_t st)
{
    size_t S = a.t.T + W - 1;
    size_t smem = S * S * sizeof(float2);
    cudaFuncSetAttribute(degrid_kernel<W>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    degrid_kernel<W><<<persistent_blocks(degrid_kernel<W>, smem, num_sms), 256, smem, st>>>(a);
    return cudaGetLastError();
}

#define RICK_W_SWITCH(W, CALL)          \
    switch (W) {                        \
    case 1: CALL(1); break;             \
    case 2: CALL(2); break;             \
    case 3: CALL(3); break;             \
    case 4: CALL(4); break;             \
    case 5: CALL(5); break;             \
    case 6: CALL(6); break;             \
    case 7: CALL(7); break;             \
    case 8: CALL(8); break;             \
    case 9: CALL(9); break;             \
    case 10: CALL(10); break;           \
    case 11: CALL(11); break;           \
    case 12: CALL(12); break;           \
    case 13: CALL(13); break;           \
    case 14: CALL(14); break;           \
    case 15: CALL(15); break;           \
    case 16: CALL(16); break;           \
    default: err = cudaErrorInvalidValue; \
    }

rick_status rick_grid_impl(rick_plan *plan, void *ws_dev, void *planes_dev, int mode,
                           void *stream, const uint8_t *touched)
{
    const int accumulate = mode == RICK_GRID_ACCUMULATE;
    if (!plan || !ws_dev || !planes_dev) return RICK_EINVAL;
    if (plan->sticky != RICK_OK) return plan->sticky;
    if (((uintptr_t)ws_dev & 255) || ((uintptr_t)planes_dev & 15)) return RICK_EINVAL;
    const rick_params &p = plan->p;
    const WsLayout L = rick_ws_layout(&p, plan->max_vis);
    WsPtrs w = rick_ws_ptrs(ws_dev, L);
    cudaStream_t st = (cudaStream_t)stream;
    GridArgs a;
    a.t = make_tile_args(plan, w, w.gbase);
    a.planes = (float2 *)planes_dev;
    a.log2T = ilog2(p.tile);
    a.accumulate = accumulate;
    a.touched = mode == RICK_GRID_CHUNK_TILES ? touched : NULL;
    a.nzero = mode != RICK_GRID_OVERWRITE ? 0u
                                          : (a.t.ntiles + RICK_ZERO_GROUP - 1) / RICK_ZERO_GROUP;
    cudaError_t err = cudaSuccess;
    const bool det = (p.options & RICK_OPT_DETERMINISTIC) != 0;
    if (det && mode == RICK_GRID_CHUNK_TILES) return RICK_EINVAL;  // its slots add per tile
    a.mcslot = det ? w.mcslot : NULL;
    a.mcacc = det ? w.mcacc : NULL;
    set_sub_args(a, p, w, L);
    const uint32_t least = rick_grid_plain(&p) ? 1u : 2u;
    zero_tiles_kernel<<<(accumulate && !det && !a.nslots) ? 1 : plan->num_sms * 8, 256, 0, st>>>(
        w.gbase, a.t.ntiles, a.t.nt, a.log2T, p.n, a.planes, w.hdr, accumulate, a.mcslot,
        a.mcacc, a.touched, least, a.slots, a.arrived, a.nslots);
    RICK_LAUNCH_CHECK(plan);
    const int gmode = det ? GM_DET : p.precision == RICK_PREC_FP32_COMPENSATED ? GM_COMP : GM_PLAIN;
#define CALL_GRID(WW) err = launch_grid<WW>(a, gmode, plan->num_sms, st)
    RICK_W_SWITCH(p.support, CALL_GRID);
#undef CALL_GRID
    ++plan->launches;
    RICK_CUDA_TRY(plan, err);
    if (det) {
        det_mc_convert_kernel<<<plan->num_sms * 8, 256, 0, st>>>(
            w.gbase, a.t.ntiles, a.t.nt, a.log2T, p.n, a.planes, w.hdr, accumulate, a.mcslot,
            a.mcacc);
        RICK_LAUNCH_CHECK(plan);
    }
    return RICK_OK;
}

extern "C" rick_status rick_grid(rick_plan *plan, void *ws_dev, void *planes_dev, void *stream)
{
    return rick_grid_impl(plan, ws_dev, planes_dev, RICK_GRID_OVERWRITE, stream);
}

extern "C" rick_status rick_grid_sparse(rick_plan *plan, void *ws_dev, void *planes_dev, void *stream)
{
    return rick_grid_impl(plan, ws_dev, planes_dev, RICK_GRID_RECORD_TILES, stream);
}

extern "C" rick_status rick_grid_accumulate(rick_plan *plan, void *ws_dev, void *planes_dev,
                                            void *stream)
{
    return rick_grid_impl(plan, ws_dev, planes_dev, RICK_GRID_ACCUMULATE, stream);
}

template <int W>
static cudaError_t launch_grid_batch(const GridBatchArgs &ba, int num_sms, cudaStream_t st)
{
    const size_t smem = warps_smem<W>();
    cudaError_t e = cudaFuncSetAttribute(grid_batch_kernel<W>,
                                         cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    grid_batch_kernel<W><<<persistent_blocks(grid_batch_kernel<W>, smem, num_sms),
                           32 * RICK_GRID_WARPS, smem, st>>>(ba);
    return cudaGetLastError();
}

extern "C" rick_status rick_grid_sparse_batch(rick_plan *const *plans, void *const *ws_dev,
                                              void *const *planes_dev, int32_t n_jobs,
                                              void *stream)
{
    if (!plans || !ws_dev || !planes_dev) return RICK_EINVAL;
    if (n_jobs < 1 || n_jobs > RICK_GRID_BATCH_MAX) return RICK_ERANGE;
    for (int j = 0; j < n_jobs; ++j) {
        const rick_plan *pl = plans[j];
        if (!pl || !ws_dev[j] || !planes_dev[j]) return RICK_EINVAL;
        if (pl->sticky != RICK_OK) return pl->sticky;
        if (((uintptr_t)ws_dev[j] & 255) || ((uintptr_t)planes_dev[j] & 15)) return RICK_EINVAL;
        if (pl->p.support != plans[0]->p.support || pl->p.tile != plans[0]->p.tile ||
            pl->device != plans[0]->device || pl->p.precision != RICK_PREC_FP32 ||
            (pl->p.options & RICK_OPT_DETERMINISTIC))
            return RICK_EINVAL;
        for (int i = 0; i < j; ++i)  // each job needs its own workspace and planes
            if (ws_dev[i] == ws_dev[j] || planes_dev[i] == planes_dev[j]) return RICK_EINVAL;
    }
    rick_plan *p0 = plans[0];
    GridBatchArgs ba;
    memset(&ba, 0, sizeof(ba));
    ba.n_jobs = n_jobs;
    int tiles_max = 0;
    for (int j = 0; j < n_jobs; ++j) {
        const rick_params &p = plans[j]->p;
        const WsLayout L = rick_ws_layout(&p, plans[j]->max_vis);
        WsPtrs w = rick_ws_ptrs(ws_dev[j], L);
        GridArgs &a = ba.job[j];
        a.t = make_tile_args(plans[j], w, w.gbase);
        a.planes = (float2 *)planes_dev[j];
        a.log2T = ilog2(p.tile);
        a.accumulate = 0;
        a.touched = NULL;
        a.nzero = 0;
        set_sub_args(a, p, w, L);
        a.mcslot = NULL;
        a.mcacc = NULL;
        tiles_max = max(tiles_max, (int)a.t.ntiles);
    }
    cudaStream_t st = (cudaStream_t)stream;
    const unsigned bx = (unsigned)max(1, min(p0->num_sms * 8 / n_jobs, (tiles_max + 7) / 8));
    zero_tiles_batch_kernel<<<dim3(bx, (unsigned)n_jobs), 256, 0, st>>>(ba);
    cudaError_t err = cudaGetLastError();
    if (err == cudaSuccess) {
#define CALL_GRID_BATCH(WW) err = launch_grid_batch<WW>(ba, p0->num_sms, st)
        RICK_W_SWITCH(p0->p.support, CALL_GRID_BATCH);
#undef CALL_GRID_BATCH
    }
    p0->launches += 2;
    if (err != cudaSuccess) {
        for (int j = 0; j < n_jobs; ++j) plans[j]->sticky = RICK_ECUDA;
        return RICK_ECUDA;
    }
    return RICK_OK;
}

extern "C" rick_status rick_degrid(rick_plan *plan, void *ws_dev, const void *planes_dev,
                                   const float *weight_dev, void *vis_out_dev, void *stream)
{
    if (!plan || !ws_dev || !planes_dev || !vis_out_dev) return RICK_EINVAL;
    if (plan->sticky != RICK_OK) return plan->sticky;
    if (((uintptr_t)ws_dev & 255) || ((uintptr_t)planes_dev & 15) || ((uintptr_t)vis_out_dev & 7) ||
        ((uintptr_t)weight_dev & 3))
        return RICK_EINVAL;
    const rick_params &p = plan->p;
    WsPtrs w = rick_ws_ptrs(ws_dev, rick_ws_layout(&p, plan->max_vis));
    cudaStream_t st = (cudaStream_t)stream;
    DegridArgs a;
    a.t = make_tile_args(plan, w, w.dbase);
    a.planes = (const float2 *)planes_dev;
    a.weight = weight_dev;
    a.vis_out = (float2 *)vis_out_dev;
    a.log2T = ilog2(p.tile);
    degrid_zero_dropped_kernel<<<plan->num_sms * 4, 256, 0, st>>>(w.hdr, w.key, a.vis_out);
    RICK_LAUNCH_CHECK(plan);
    cudaError_t err = cudaSuccess;
#define CALL_DEGRID(WW) err = launch_degrid<WW>(a, plan->num_sms, st)
    RICK_W_SWITCH(p.support, CALL_DEGRID);
#undef CALL_DEGRID
    ++plan->launches;
    RICK_CUDA_TRY(plan, err);
    return RICK_OK;
}
