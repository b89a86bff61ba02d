// rick_bin.cu -- binning of visibilities by (w-plane, uv-tile, edge class)
// (§2, gridding sub-step 1: "an array is created for each slab, concatenating
// the data with u-v coordinates inside the corresponding slab"; here the slab
// is a T x T uv-tile of one w-plane, and a visibility goes to the closest
// w-plane, §2).
//
// Passes, all stream-ordered:
//   1. w range: min / max of the finite w as order-preserving integer keys
//      (exact, deterministic), unless the range is given;
//   2. (its last block) plane width, the plane boundaries as keys, plane centres;
//   3. key: per visibility two FP64 FMAs give the grid coordinates, everything
//      else (floor, rounding, fraction, plane search) is integer work on the
//      bit patterns -- GB300 runs FP64 at a small fraction of FP32;
//      warp-aggregated histogram; deterministic weight-sum partials;
//   4. exclusive scan of the histogram -> bin offsets;
//   5. scatter: warp-aggregated cursors place each record in its bin;
//   6. work lists of the tile kernels (chunks of at most chunk_cap records).
#include <math.h>

#include <mutex>

#include "rick_common.cuh"

#define FULL 0xffffffffu

// ------------------------------------------------------------------------
// Exclusive scan of uint32 (block of 2048, recursive over block sums)

__global__ void __launch_bounds__(1024) scan_blocks_kernel(const uint32_t *in, uint32_t *out,
                                                           int64_t n, uint32_t *block_sums)
{
    __shared__ uint32_t warp_tot[32];
    int64_t base = (int64_t)blockIdx.x * 2048;
    int t = threadIdx.x, lane = t & 31, wid = t >> 5;
    int64_t i0 = base + 2 * t;
    uint32_t a = i0 < n ? in[i0] : 0u, b = i0 + 1 < n ? in[i0 + 1] : 0u;
    uint32_t s = a + b, inc = s;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        uint32_t v = __shfl_up_sync(FULL, inc, o);
        if (lane >= o) inc += v;
    }
    if (lane == 31) warp_tot[wid] = inc;
    __syncthreads();
    if (wid == 0) {
        uint32_t w = warp_tot[lane], wi = w;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            uint32_t v = __shfl_up_sync(FULL, wi, o);
            if (lane >= o) wi += v;
        }
        warp_tot[lane] = wi - w;  // exclusive prefix of the warps
        if (lane == 31) block_sums[blockIdx.x] = wi;
    }
    __syncthreads();
    uint32_t ex = warp_tot[wid] + inc - s;
    if (i0 < n) out[i0] = ex;
    if (i0 + 1 < n) out[i0 + 1] = ex + a;
}

__global__ void scan_add_kernel(uint32_t *out, int64_t n, const uint32_t *block_off)
{
    int64_t i = (int64_t)blockIdx.x * 2048 + threadIdx.x;
    uint32_t add = block_off[blockIdx.x];
    if (i < n) out[i] += add;
    if (i + 1024 < n) out[i + 1024] += add;
}

// out[i] = sum_{j < i} in[j]; in may equal out.  tmp: rick_scan_tmp(n) words.
// *launches counts the kernels enqueued.
static cudaError_t scan_u32(const uint32_t *in, uint32_t *out, int64_t n, uint32_t *tmp,
                            cudaStream_t st, unsigned long long *launches)
{
    if (n <= 0) return cudaSuccess;
    int64_t nb = (n + 2047) / 2048;
    scan_blocks_kernel<<<(unsigned)nb, 1024, 0, st>>>(in, out, n, tmp);
    ++*launches;
    if (nb == 1) return cudaGetLastError();
    cudaError_t e = scan_u32(tmp, tmp, nb, tmp + nb + 1, st, launches);
    if (e != cudaSuccess) return e;
    scan_add_kernel<<<(unsigned)nb, 1024, 0, st>>>(out, n, tmp);
    ++*launches;
    return cudaGetLastError();
}

// ------------------------------------------------------------------------
// Pass 1: w range

// Plane geometry (n_w <= 1024) from the range keys, by the threads of one block.
__device__ __forceinline__ void plane_setup(WsHeader *hdr, uint64_t lo_key, uint64_t hi_key,
                                            unsigned long long *bkey, float4 *wplane, int n_w)
{
    double wmin, wmax;
    if (lo_key == ~0ull) {  // no finite w at all
        wmin = wmax = 0.0;
    } else {
        wmin = rick_dunkey(lo_key);
        wmax = rick_dunkey(hi_key);
    }
    const double dw = (wmax - wmin) / n_w;
    if (threadIdx.x == 0) {
        hdr->dw = dw;
        hdr->stats.w_min = wmin;
        hdr->stats.w_max = wmax;
    }
    for (int j = threadIdx.x; j <= n_w; j += blockDim.x) {
        if (j >= 1 && j < n_w) bkey[j - 1] = rick_dkey(fma((double)j, dw, wmin));
        // the entry after the last plane: the plane spacing, for the phase step
        const double wk = j == n_w ? dw : dw == 0.0 ? wmin : fma(j + 0.5, dw, wmin);
        const ff f = ff_from_double(wk);
        wplane[j] = make_float4(f.hi, f.lo, (float)wk, 0.0f);
    }
}

// The header, the zeroed histogram and, where no pass over the w has to find the
// range (given, or nothing to look at), the planes.
// range_src (optional): a header whose w-range keys stand in for a given
// range (the exact range of a larger set, found by an earlier pass).
// n_vis: records (inputs, or twice the inputs with the Hermitian mirror).
__global__ void __launch_bounds__(256) bin_init_kernel(WsPtrs w, uint64_t n_vis, uint32_t chunk_cap,
                                                       int given, uint64_t wmin_key,
                                                       uint64_t wmax_key, uint32_t n_key_blocks,
                                                       const WsHeader *range_src, uint64_t n_src,
                                                       int mirror, uint32_t sub_cap, int64_t nhist,
                                                       int n_w)
{
    const int64_t n4 = nhist / 4, i0 = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    for (int64_t i = i0; i < n4; i += (int64_t)gridDim.x * blockDim.x)
        ((uint4 *)w.hist)[i] = make_uint4(0u, 0u, 0u, 0u);
    if (blockIdx.x != 0) return;
    if (threadIdx.x < nhist - 4 * n4) w.hist[4 * n4 + threadIdx.x] = 0;
    if (range_src) {
        given = 1;
        wmin_key = range_src->wmin_key;
        wmax_key = range_src->wmax_key;
    }
    if (!given) {
        wmin_key = ~0ull;
        wmax_key = 0ull;
    }
    WsHeader *hdr = w.hdr;
    if (threadIdx.x == 0) {
        hdr->sub_cap = sub_cap;
        hdr->n_items = 0;
        hdr->n_groups = 0;
        hdr->n_slots = 0;
        hdr->n_vis = n_vis;
        hdr->n_src = n_src;
        hdr->mirror = (uint32_t)mirror;
        hdr->fault = 0;
        hdr->drop_uv = 0;
        hdr->drop_w = 0;
        hdr->chunk_cap = chunk_cap;
        hdr->n_key_blocks = n_key_blocks;
        hdr->range_done = 0;
        hdr->range_given = given;
        hdr->wmin_key = wmin_key;
        hdr->wmax_key = wmax_key;
    }
    if (given || n_vis == 0) plane_setup(hdr, wmin_key, wmax_key, w.bkey, w.wplane, n_w);
}

// Launch the w-range reduction of visibilities [0, n) into hdr's range keys.
void rick_launch_wrange(const rick_plan *plan, const double *uvw, int64_t n, WsHeader *hdr,
                        cudaStream_t st, int n_chan, const double *scale);


// Fold the key of w into [lo, hi] unless w is not finite.
__device__ __forceinline__ void wrange_fold(double w, uint64_t &lo, uint64_t &hi)
{
    const uint64_t b = rick_dbits(w);
    if (((b >> 52) & 0x7FF) == 0x7FF) return;  // not finite
    const uint64_t k = rick_dkey(w);
    lo = k < lo ? k : lo;
    hi = k > hi ? k : hi;
}

// w range of visibilities [0, n).  Multi-channel input (n_chan > 0): rows of
// n_chan visibilities, w = the row's w times the channel factor.  When every
// factor is positive and finite, rounding is monotone in the factor, so a
// row's extremes are its products with the smallest and the largest factor
// (unless one of those overflows, when every channel is folded).
// MIRROR: the mirrored visibilities' -w are folded in too.
// With bkey, the block that ends last turns the range into the planes.
template <bool MIRROR>
__global__ void wrange_kernel(const double *uvw, int64_t n, WsHeader *hdr, int n_chan,
                              const double *scale, unsigned long long *bkey, float4 *wplane,
                              int n_w)
{
    __shared__ double s_min[32], s_max[32];
    __shared__ int s_ok[32];
    uint64_t lo = ~0ull, hi = 0ull;
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = blockDim.x >> 5;
    if (n_chan <= 0) {
        for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n;
             i += (int64_t)gridDim.x * blockDim.x) {
            const double w = uvw[3 * i + 2];
            wrange_fold(w, lo, hi);
            if (MIRROR) wrange_fold(-w, lo, hi);
        }
    } else {
        // smallest and largest factor, and whether all are positive and finite
        double fmin = INFINITY, fmax = 0.0;
        int ok = 1;
        for (int c = threadIdx.x; c < n_chan; c += blockDim.x) {
            const double f = scale[c];
            ok &= (f > 0.0 && f < INFINITY) ? 1 : 0;
            fmin = fmin < f ? fmin : f;
            fmax = fmax > f ? fmax : f;
        }
        for (int o = 16; o > 0; o >>= 1) {
            const double a = __shfl_xor_sync(FULL, fmin, o), b = __shfl_xor_sync(FULL, fmax, o);
            fmin = fmin < a ? fmin : a;
            fmax = fmax > b ? fmax : b;
            ok &= __shfl_xor_sync(FULL, ok, o);
        }
        if (lane == 0) {
            s_min[wid] = fmin;
            s_max[wid] = fmax;
            s_ok[wid] = ok;
        }
        __syncthreads();
        for (int k = 0; k < nw; ++k) {
            fmin = fmin < s_min[k] ? fmin : s_min[k];
            fmax = fmax > s_max[k] ? fmax : s_max[k];
            ok &= s_ok[k];
        }
        const int64_t n_rows = n / n_chan;  // whole rows (callers pass n = rows * n_chan)
        for (int64_t r = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; r < n_rows;
             r += (int64_t)gridDim.x * blockDim.x) {
            const double w0 = uvw[3 * r + 2];
            const double a = w0 * fmin, b = w0 * fmax;
            if (ok && isfinite(a) && isfinite(b)) {
                wrange_fold(a, lo, hi);
                wrange_fold(b, lo, hi);
            } else {
                for (int c = 0; c < n_chan; ++c) wrange_fold(w0 * scale[c], lo, hi);
            }
        }
    }
    for (int o = 16; o > 0; o >>= 1) {
        uint64_t l2 = __shfl_xor_sync(FULL, lo, o), h2 = __shfl_xor_sync(FULL, hi, o);
        lo = l2 < lo ? l2 : lo;
        hi = h2 > hi ? h2 : hi;
    }
    if (lane == 0) {
        if (lo != ~0ull) atomicMin(&hdr->wmin_key, (unsigned long long)lo);
        if (hi != 0ull) atomicMax(&hdr->wmax_key, (unsigned long long)hi);
    }
    if (!bkey) return;
    __shared__ bool s_last;
    __threadfence();  // this thread's minima and maxima before the block's count
    __syncthreads();
    if (threadIdx.x == 0) s_last = atomicAdd(&hdr->range_done, 1u) == gridDim.x - 1;
    __syncthreads();
    if (!s_last) return;
    __threadfence();
    plane_setup(hdr, *(volatile unsigned long long *)&hdr->wmin_key,
                *(volatile unsigned long long *)&hdr->wmax_key, bkey, wplane, n_w);
}

// Blocks of the w-range pass: four uvw rows a thread for the small sets, whose
// blocks are otherwise mostly atomics.
static int wrange_blocks(const rick_plan *plan, int64_t units)
{
    const int64_t b = (units + 1023) / 1024;
    return (int)(b < 1 ? 1 : b < plan->num_sms * 4 ? b : plan->num_sms * 4);
}

void rick_launch_wrange(const rick_plan *plan, const double *uvw, int64_t n, WsHeader *hdr,
                        cudaStream_t st, int n_chan, const double *scale)
{
    wrange_kernel<false><<<plan->num_sms * 4, 256, 0, st>>>(uvw, n, hdr, n_chan, scale, NULL, NULL,
                                                            0);
}

// ------------------------------------------------------------------------
// Pass 3: keys, histogram, weight-sum partials

struct KeyArgs {
    int64_t n_vis;
    const double *uvw;
    const float *weight;
    int n, n_w, W, log2T, nt;
    double fov, half_n;
    uint64_t key_lo, key_hi;  // rick_dkey(-0.5), rick_dkey(n + 0.5)
    int bulk;                 // uvw (and weight) 16-byte aligned: blocks stage them by bulk copy
    int n_chan;               // > 0: uvw holds rows of n_chan visibilities, scaled per channel
    int n_corr;               // correlations per visibility (weights [n_vis][n_corr])
    const double *chan_scale;
    int64_t n_src;            // inputs; records i >= n_src mirror input i - n_src (n_vis = 2 n_src)
    uint32_t wait_polls;      // limit of the wait for the block's bulk copies
    SubShape sub;
    WsPtrs ws;
};

// Dynamic shared memory of the key pass: the block's uvw and weights, then the
// plane boundary keys.
static inline size_t key_pass_smem(int n_w)
{
    return 28 * (size_t)(RICK_KEY_THREADS * RICK_KEY_ITEMS) + 8 * (size_t)(n_w > 1 ? n_w - 1 : 1);
}

__device__ __forceinline__ uint32_t plane_of(uint64_t kw, const unsigned long long *sb, int nb)
{
    int lo = 0, hi = nb;  // number of boundaries <= w
    while (lo < hi) {
        int mid = (lo + hi) >> 1;
        if (sb[mid] <= kw)
            lo = mid + 1;
        else
            hi = mid;
    }
    return (uint32_t)lo;
}

__global__ void __launch_bounds__(RICK_KEY_THREADS) bin_key_kernel(KeyArgs a)
{
    constexpr int NI = RICK_KEY_THREADS * RICK_KEY_ITEMS;
    extern __shared__ __align__(128) unsigned char s_dyn[];
    double *s_uvw = (double *)s_dyn;
    float *s_wt = (float *)(s_dyn + 24 * NI);
    unsigned long long *s_bkey = (unsigned long long *)(s_dyn + 28 * NI);
    __shared__ unsigned long long s_bar;
    __shared__ double s_wsum[RICK_KEY_THREADS / 32];
    __shared__ unsigned long long s_drop[2][RICK_KEY_THREADS / 32];
    const WsHeader *hdr = a.ws.hdr;
    const int64_t blk0 = (int64_t)blockIdx.x * NI;
    const int nitems = (int)(a.n_vis - blk0 < NI ? a.n_vis - blk0 : NI);
    // The block's 1024 uvw rows and weights are contiguous: one bulk copy each
    // (TMA) into shared memory, while the plane keys load; a ragged last block
    // or unaligned inputs take plain loads instead.
    const bool bulk = a.bulk && nitems == NI && blk0 + NI <= a.n_src;
    if (bulk && threadIdx.x == 0) {
        rick_mbar_init(&s_bar, 1);
        rick_mbar_expect_tx(&s_bar, 24 * NI + (a.weight ? 4 * NI : 0));
        rick_bulk_g2s(s_uvw, a.uvw + 3 * blk0, 24 * NI, &s_bar);
        if (a.weight) rick_bulk_g2s(s_wt, a.weight + blk0, 4 * NI, &s_bar);
    }
    int nb = a.n_w - 1;
    for (int j = threadIdx.x; j < nb; j += blockDim.x) s_bkey[j] = a.ws.bkey[j];
    if (!bulk && a.n_chan > 0) {
        // multi-channel input: the uvw of channel c of row r is the row's uvw
        // times the channel factor (one FP64 product per coordinate)
        const int64_t row0 = blk0 / a.n_chan;
        const int ch0 = (int)(blk0 - row0 * a.n_chan);
        for (int i = threadIdx.x; i < nitems; i += blockDim.x) {
            const int t = ch0 + i;
            const int64_t r = row0 + t / a.n_chan;
            const double f = a.chan_scale[t % a.n_chan];
            s_uvw[3 * i] = a.uvw[3 * r] * f;
            s_uvw[3 * i + 1] = a.uvw[3 * r + 1] * f;
            s_uvw[3 * i + 2] = a.uvw[3 * r + 2] * f;
            if (a.weight && a.n_corr == 1) s_wt[i] = a.weight[blk0 + i];
        }
    } else if (!bulk) {
        // records past the inputs mirror input i - n_src: -uvw (its weight)
        for (int i = threadIdx.x; i < nitems; i += blockDim.x) {
            const int64_t r = blk0 + i, src = r < a.n_src ? r : r - a.n_src;
            const double sg = r < a.n_src ? 1.0 : -1.0;
            s_uvw[3 * i] = sg * a.uvw[3 * src];
            s_uvw[3 * i + 1] = sg * a.uvw[3 * src + 1];
            s_uvw[3 * i + 2] = sg * a.uvw[3 * src + 2];
            if (a.weight) s_wt[i] = a.weight[src];
        }
    }
    __syncthreads();
    const bool landed = !bulk || rick_mbar_wait(&s_bar, 0, a.wait_polls);
    if (!__syncthreads_and(landed)) {
        // the copy did not complete in time (never expected): leave this block's
        // inputs out of the binning, flag the fault (reported as n_binned < 0),
        // and let the copy land before the block's shared memory is released
        if (threadIdx.x == 0) {
            atomicExch(&a.ws.hdr->fault, 1u);
            a.ws.wpart[blockIdx.x] = 0.0;
        }
        for (int i = threadIdx.x; i < nitems; i += blockDim.x) a.ws.key[blk0 + i] = 0xFFFFFFFFu;
        rick_mbar_wait(&s_bar, 0, RICK_WAIT_POLLS);  // drain: the copies land before the block ends
        return;
    }
    const bool degenerate = rick_dbits(hdr->dw) == 0;
    const bool given = hdr->range_given;
    const uint64_t wlo = hdr->wmin_key, whi = hdr->wmax_key;
    const int T = 1 << a.log2T, tmask = T - 1;
    int lane = threadIdx.x & 31;

    ff ws = {0.0f, 0.0f};  // this thread's weight sum in double-single arithmetic
    unsigned long long du = 0, dwn = 0;
    int64_t base = blk0 + threadIdx.x;
#pragma unroll 2
    for (int it = 0; it < RICK_KEY_ITEMS; ++it) {
        int64_t i = base + (int64_t)it * RICK_KEY_THREADS;
        uint32_t key = 0xFFFFFFFFu, sid = 0xFFFFFFFFu;
        const int li = it * RICK_KEY_THREADS + threadIdx.x;  // index inside the block
        if (i < a.n_vis) {
            double u = s_uvw[3 * li], v = s_uvw[3 * li + 1], w = s_uvw[3 * li + 2];
            int32_t ax, ay;
            float fx, fy;
            bool ok = rick_footprint(fma(u, a.fov, a.half_n), a.n, a.W, a.key_lo, a.key_hi, &ax,
                                     &fx) &&
                      rick_footprint(fma(v, a.fov, a.half_n), a.n, a.W, a.key_lo, a.key_hi, &ay,
                                     &fy);
            if (!ok) {
                ++du;
            } else {
                uint64_t wb = rick_dbits(w);
                uint64_t kw = rick_dkey(w);
                if (((wb >> 52) & 0x7FF) == 0x7FF || (given && (kw < wlo || kw > whi))) {
                    ++dwn;
                } else {
                    uint32_t k = degenerate ? 0u : plane_of(kw, s_bkey, nb);
                    int lx = ax & tmask, ly = ay & tmask;
                    int ex = lx > T - a.W, ey = ly > T - a.W;
                    uint32_t cls = ex ? (ey ? 2u : 1u) : (ey ? 3u : 0u);
                    key = (((k * a.nt + (uint32_t)(ay >> a.log2T)) * a.nt +
                            (uint32_t)(ax >> a.log2T)) << 2) | cls;
                    sid = rick_sub_id(a.sub, key, (uint32_t)lx, (uint32_t)ly);
                    a.ws.cell[i] = (uint32_t)ax | ((uint32_t)ay << 16);
                    a.ws.frac[i] = make_float2(fx, fy);
                    if (a.n_corr == 1) {
                        float wt = a.weight ? s_wt[li] : 1.0f;
                        ws = ff_add(ws, ff{wt, 0.0f});
                    } else {  // the visibility's weight is the sum of its correlations'
                        for (int c = 0; c < a.n_corr; ++c)
                            ws = ff_add(ws, ff{a.weight ? a.weight[i * a.n_corr + c] : 1.0f,
                                               0.0f});
                    }
                }
            }
            a.ws.key[i] = key;
        }
        // histogram: one atomic per sub-bin that the warp's 32 inputs reach.  The
        // counter's old value ranks the inputs inside the sub-bin, so the scatter
        // needs no atomics of its own.  (One per run of equal sub-bins in
        // consecutive lanes sent the core of a single-channel set to a few
        // counters nine times a warp: 4e6 visibilities, 422 -> 296 us; 5e7 of 16
        // channels, one or two runs a warp, 624 -> 604.)
        const unsigned peers = __match_any_sync(FULL, sid);
        const int first = __ffs(peers) - 1;
        uint32_t base = 0;
        if (sid != 0xFFFFFFFFu && lane == first)
            base = atomicAdd(&a.ws.hist[sid], (uint32_t)__popc(peers));
        base = __shfl_sync(FULL, base, first);
        if (i < a.n_vis) a.ws.rank[i] = base + (uint32_t)__popc(peers & ((1u << lane) - 1u));
    }
    // deterministic block reduction of the weight sum (double-single pairs in
    // the warp: GB300 issues FP64 slowly) and of the drop counts
    for (int o = 16; o > 0; o >>= 1) {
        ff other = {__shfl_xor_sync(FULL, ws.hi, o), __shfl_xor_sync(FULL, ws.lo, o)};
        ws = ff_add(ws, other);
        du += __shfl_xor_sync(FULL, du, o);
        dwn += __shfl_xor_sync(FULL, dwn, o);
    }
    int wid = threadIdx.x >> 5;
    if (lane == 0) {
        s_wsum[wid] = (double)ws.hi + (double)ws.lo;
        s_drop[0][wid] = du;
        s_drop[1][wid] = dwn;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        double t = 0.0;
        unsigned long long d0 = 0, d1 = 0;
        for (int j = 0; j < RICK_KEY_THREADS / 32; ++j) {
            t += s_wsum[j];
            d0 += s_drop[0][j];
            d1 += s_drop[1][j];
        }
        a.ws.wpart[blockIdx.x] = t;
        if (d0) atomicAdd(&a.ws.hdr->drop_uv, d0);
        if (d1) atomicAdd(&a.ws.hdr->drop_w, d1);
    }
}

// Weight sum over the block partials in a fixed order; stats.
// unit_weights > 0: no weights were given, and each kept visibility weighs
// unit_weights (its number of correlations).
// stats_out (optional): the caller's copy of the stats.
__device__ __forceinline__ void bin_finalize(WsHeader *hdr, const double *wpart, int nparts,
                                             int unit_weights, rick_bin_stats *stats_out)
{
    __shared__ double s[1024];
    double t = 0.0;
    for (int i = threadIdx.x; i < nparts; i += 1024) t += wpart[i];
    s[threadIdx.x] = t;
    __syncthreads();
    for (int o = 512; o > 0; o >>= 1) {
        if (threadIdx.x < o) s[threadIdx.x] += s[threadIdx.x + o];
        __syncthreads();
    }
    if (threadIdx.x == 0) {
        long long binned = (long long)hdr->n_vis - (long long)hdr->drop_uv - (long long)hdr->drop_w;
        if (hdr->fault) binned = -1;  // a bounded wait ran out: the binning is incomplete
        hdr->stats.n_binned = binned;
        hdr->stats.n_dropped_uv = (long long)hdr->drop_uv;
        hdr->stats.n_dropped_w = (long long)hdr->drop_w;
        hdr->stats.sum_weight = unit_weights ? (double)binned * unit_weights : s[0];
        if (stats_out) *stats_out = hdr->stats;
    }
}

__global__ void __launch_bounds__(1024) bin_finalize_kernel(WsHeader *hdr, const double *wpart,
                                                            int nparts, int unit_weights,
                                                            rick_bin_stats *stats_out)
{
    bin_finalize(hdr, wpart, nparts, unit_weights, stats_out);
}

// ------------------------------------------------------------------------
// Pass 5: scatter records into their bins

// Each thread takes RICK_SCATTER_U inputs per pass (256 apart), so that their
// load chains -- key and rank, then the (bin, sub-counter) offset, then the
// record stores -- overlap (eight chains at two CTAs per SM beat four at four
// CTAs per SM).  Positions come from the ranks the key pass took from the
// histogram counters: no atomics here.
#define RICK_SCATTER_U 8

//
// With CORR, each visibility has n_corr correlations (vis and weight
// [n_vis][n_corr]) and its record carries their weighted sum, sum_c w_c V_c.
// MIRROR: records i >= n_src (the Hermitian mirror) carry conj(V) of input
// i - n_src.
template <bool CORR, bool MIRROR>
__global__ void __launch_bounds__(256) bin_scatter_kernel(int64_t n_vis, const float2 *vis,
                                                          const float *weight, WsPtrs ws,
                                                          int n_corr, int64_t n_src,
                                                          SubShape sub)
{
    constexpr int U = RICK_SCATTER_U;
    const uint32_t tmask = (1u << sub.log2T) - 1;
    const int64_t step = (int64_t)gridDim.x * blockDim.x * U;
    for (int64_t i0 = (int64_t)blockIdx.x * blockDim.x * U; i0 < n_vis; i0 += step) {
        int64_t idx[U];
        uint32_t key[U], rk[U], cl[U];
        float2 v[U], fr[U];
        float wt[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
            idx[u] = i0 + (int64_t)u * blockDim.x + threadIdx.x;
            key[u] = 0xFFFFFFFFu;
            if (idx[u] < n_vis) {
                key[u] = ws.key[idx[u]];
                rk[u] = ws.rank[idx[u]];
                if (CORR) {
                    float2 acc = make_float2(0.0f, 0.0f);
                    for (int c = 0; c < n_corr; ++c) {
                        const float2 vc = vis[idx[u] * n_corr + c];
                        const float wc = weight ? weight[idx[u] * n_corr + c] : 1.0f;
                        acc.x = __fmaf_rn(vc.x, wc, acc.x);
                        acc.y = __fmaf_rn(vc.y, wc, acc.y);
                    }
                    v[u] = acc;
                    wt[u] = 1.0f;
                } else if (MIRROR) {
                    const bool mir = idx[u] >= n_src;
                    const int64_t src = mir ? idx[u] - n_src : idx[u];
                    v[u] = vis[src];
                    if (mir) v[u].y = -v[u].y;
                    wt[u] = weight ? weight[src] : 1.0f;
                } else {
                    v[u] = vis[idx[u]];
                    wt[u] = weight ? weight[idx[u]] : 1.0f;
                }
                fr[u] = ws.frac[idx[u]];
                cl[u] = ws.cell[idx[u]];
            }
        }
#pragma unroll
        for (int u = 0; u < U; ++u) {
            if (key[u] != 0xFFFFFFFFu) {
                const uint32_t sid = rick_sub_id(sub, key[u], cl[u] & tmask, cl[u] >> 16 & tmask);
                const uint32_t pos = ws.suboff[sid] + rk[u];
                ws.perm[pos] = (uint32_t)idx[u];
                ws.rec[pos] = make_float4(v[u].x * wt[u], v[u].y * wt[u], fr[u].x, fr[u].y);
                ws.rcell[pos] = cl[u];
            }
        }
    }
}

// Bin offsets from the sub-bin offsets: bin b starts where its first sub-bin
// starts.
__global__ void bin_offsets_kernel(const uint32_t *suboff, uint32_t *offsets, int64_t nbins,
                                   SubShape sub)
{
    for (int64_t b = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; b <= nbins;
         b += (int64_t)gridDim.x * blockDim.x)
        offsets[b] = suboff[(b >> 2) * sub.per + rick_sub_first(sub, (uint32_t)b & 3u)];
}

// Re-pack record values for new visibilities through an existing permutation,
// and sum the new weights: double-single per thread and warp, FP64 per block,
// block partials in wpart (summed in a fixed order by values_finalize_kernel).
// det: also the blocks' sums of |Re| + |Im| of the new values (the bound of the
// deterministic mode's fixed-point scale).
// RESID: the values are the gradient of chi^2 = sum w |r|^2 in the model, for the
// residuals r = vis and the gradient *grad of chi^2: -(*grad w)(2 r), in the
// roundings of that product.
template <bool RESID>
__global__ void __launch_bounds__(256) bin_values_kernel(const float2 *vis, const float *weight,
                                                         WsPtrs ws, int det, const float *grad)
{
    const float g = RESID ? -*grad : 1.0f;
    __shared__ double s_part[8];
    __shared__ float s_bound[8];
    float bound = 0.0f;
    const WsHeader *hdr = ws.hdr;
    const int64_t nb = hdr->stats.n_binned;
    ff acc = {0.0f, 0.0f};
    const int64_t n_src = (int64_t)hdr->n_src;
    for (int64_t r = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; r < nb;
         r += (int64_t)gridDim.x * blockDim.x) {
        const int64_t i0 = ws.perm[r];
        const bool mir = i0 >= n_src;  // the Hermitian mirror: conj V of input i0 - n_src
        const int64_t i = mir ? i0 - n_src : i0;
        float2 v = vis[i];
        if (mir) v.y = -v.y;
        float wt = weight ? weight[i] : 1.0f;
        if (RESID) {
            wt *= g;
            v = make_float2(2.0f * v.x, 2.0f * v.y);
        }
        float2 *val = (float2 *)&ws.rec[r];  // the value half of the record
        *val = make_float2(v.x * wt, v.y * wt);
        bound += fabsf(v.x * wt) + fabsf(v.y * wt);
        acc = ff_add(acc, ff{wt, 0.0f});
    }
    for (int o = 16; o > 0; o >>= 1) bound += __shfl_xor_sync(FULL, bound, o);
    if ((threadIdx.x & 31) == 0) s_bound[threadIdx.x >> 5] = bound;
    for (int o = 16; o > 0; o >>= 1) {
        const ff other = {__shfl_xor_sync(FULL, acc.hi, o), __shfl_xor_sync(FULL, acc.lo, o)};
        acc = ff_add(acc, other);
    }
    if ((threadIdx.x & 31) == 0) s_part[threadIdx.x >> 5] = (double)acc.hi + (double)acc.lo;
    __syncthreads();
    if (threadIdx.x == 0) {
        double t = 0.0, b = 0.0;
        for (int k = 0; k < (int)(blockDim.x >> 5); ++k) {
            t += s_part[k];
            b += s_bound[k];
        }
        ws.wpart[blockIdx.x] = t;
        if (det) ws.vpart[blockIdx.x] = b;
    }
}

__global__ void __launch_bounds__(1024) values_finalize_kernel(const double *wpart, int nparts,
                                                               int unit_weights, WsHeader *hdr,
                                                               rick_bin_stats *stats_out)
{
    __shared__ double s[1024];
    double t = 0.0;
    for (int i = threadIdx.x; i < nparts; i += 1024) t += wpart[i];
    s[threadIdx.x] = t;
    __syncthreads();
    for (int o = 512; o > 0; o >>= 1) {
        if (threadIdx.x < o) s[threadIdx.x] += s[threadIdx.x + o];
        __syncthreads();
    }
    if (threadIdx.x == 0) {
        hdr->stats.sum_weight = unit_weights ? (double)hdr->stats.n_binned : s[0];
        if (stats_out) *stats_out = hdr->stats;
    }
}

// ------------------------------------------------------------------------
// Deterministic mode (RICK_OPT_DETERMINISTIC): the ranks the key pass takes
// from atomics order a bin's records by arrival, which differs from run to
// run.  Instead, (key, input index) pairs are sorted by a stable LSD radix
// sort -- RICK_DET_DIGIT-bit digits, least significant first, over blocks of
// RICK_DET_BLOCK records -- so that the records of each bin are in input
// order, and then gathered.  A dropped record's all-ones key sorts after every
// bin in every pass.

// Per block, the count of each digit: cnt[digit * nblk + block] (digit-major,
// so that one exclusive scan gives every (digit, block) its first position).
__global__ void __launch_bounds__(256) det_hist_kernel(const uint32_t *key, int64_t n, int shift,
                                                       uint32_t *cnt, uint32_t nblk)
{
    __shared__ uint32_t h[1 << RICK_DET_DIGIT];
    for (int d = threadIdx.x; d < (1 << RICK_DET_DIGIT); d += blockDim.x) h[d] = 0;
    __syncthreads();
    const int64_t b0 = (int64_t)blockIdx.x * RICK_DET_BLOCK;
    const int lane = threadIdx.x & 31;
    for (int j = threadIdx.x; j < RICK_DET_BLOCK; j += blockDim.x) {
        const int64_t i = b0 + j;
        const uint32_t d = i < n ? (key[i] >> shift) & ((1u << RICK_DET_DIGIT) - 1) : 0xFFFFFFFFu;
        const unsigned peers = __match_any_sync(FULL, d);
        if (d != 0xFFFFFFFFu && (peers & ((1u << lane) - 1u)) == 0u)  // one add per digit
            atomicAdd(&h[d], (uint32_t)__popc(peers));
    }
    __syncthreads();
    for (int d = threadIdx.x; d < (1 << RICK_DET_DIGIT); d += blockDim.x)
        cnt[(size_t)d * nblk + blockIdx.x] = h[d];
}

// One stable pass: the block's records in rounds of 256 consecutive ones; a
// record's place is its (digit, block) start, plus the records of its digit in
// the block's earlier rounds, in earlier warps of its round and in earlier
// lanes of its warp.  idx_in NULL: the identity (the first pass).
__global__ void __launch_bounds__(256) det_scatter_kernel(const uint32_t *key_in,
                                                          const uint32_t *idx_in, int64_t n,
                                                          int shift, const uint32_t *start,
                                                          uint32_t nblk, uint32_t *key_out,
                                                          uint32_t *idx_out)
{
    constexpr int ND = 1 << RICK_DET_DIGIT;
    __shared__ uint32_t run[ND];     // next place of each digit
    __shared__ uint32_t wc[8][ND];   // this round: records of each digit per warp
    const int t = threadIdx.x, lane = t & 31, wid = t >> 5;
    for (int d = t; d < ND; d += 256) {
        run[d] = start[(size_t)d * nblk + blockIdx.x];
        for (int w = 0; w < 8; ++w) wc[w][d] = 0;
    }
    __syncthreads();
    const int64_t b0 = (int64_t)blockIdx.x * RICK_DET_BLOCK;
    for (int r = 0; r < RICK_DET_BLOCK / 256; ++r) {
        const int64_t i = b0 + r * 256 + t;
        const bool live = i < n;
        uint32_t k = 0, idx = 0, d = 0xFFFFFFFFu;
        if (live) {
            k = key_in[i];
            idx = idx_in ? idx_in[i] : (uint32_t)i;
            d = (k >> shift) & (ND - 1);
        }
        const unsigned peers = __match_any_sync(FULL, d);
        const int rank = __popc(peers & ((1u << lane) - 1u));
        if (live && rank == 0) wc[wid][d] = (uint32_t)__popc(peers);
        __syncthreads();
        if (live) {
            uint32_t pos = run[d] + (uint32_t)rank;
            for (int w = 0; w < wid; ++w) pos += wc[w][d];
            key_out[pos] = k;
            idx_out[pos] = idx;
        }
        __syncthreads();
        for (int dd = t; dd < ND; dd += 256) {
            uint32_t tot = 0;
            for (int w = 0; w < 8; ++w) {
                tot += wc[w][dd];
                wc[w][dd] = 0;
            }
            run[dd] += tot;
        }
        __syncthreads();
    }
}

// The records in sorted order: record r is input sidx[r] (records past n_src
// mirror input i - n_src; with CORR the weighted sum of the correlations).
// Each block also sums |Re| + |Im| of its record values (a fixed order: the
// grid-stride split and the reductions depend only on the sizes), the bound
// from which the fixed-point scale of the tile sums is chosen.
template <bool CORR>
__global__ void __launch_bounds__(256) det_records_kernel(const uint32_t *sidx, const float2 *vis,
                                                          const float *weight, WsPtrs ws,
                                                          int n_corr, int64_t n_src)
{
    __shared__ float s_part[8];
    const int64_t nb = ws.hdr->stats.n_binned;
    float bound = 0.0f;
    for (int64_t r = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; r < nb;
         r += (int64_t)gridDim.x * blockDim.x) {
        const uint32_t i = sidx[r];
        float2 v;
        if (CORR) {
            v = make_float2(0.0f, 0.0f);
            for (int c = 0; c < n_corr; ++c) {
                const float2 vc = vis[(int64_t)i * n_corr + c];
                const float wc = weight ? weight[(int64_t)i * n_corr + c] : 1.0f;
                v.x = __fmaf_rn(vc.x, wc, v.x);
                v.y = __fmaf_rn(vc.y, wc, v.y);
            }
        } else {
            const bool mir = (int64_t)i >= n_src;
            const int64_t src = mir ? (int64_t)i - n_src : (int64_t)i;
            v = vis[src];
            if (mir) v.y = -v.y;
            const float wt = weight ? weight[src] : 1.0f;
            v = make_float2(v.x * wt, v.y * wt);
        }
        const float2 fr = ws.frac[i];
        ws.perm[r] = i;
        ws.rec[r] = make_float4(v.x, v.y, fr.x, fr.y);
        ws.rcell[r] = ws.cell[i];
        bound += fabsf(v.x) + fabsf(v.y);
    }
    for (int o = 16; o > 0; o >>= 1) bound += __shfl_xor_sync(FULL, bound, o);
    if ((threadIdx.x & 31) == 0) s_part[threadIdx.x >> 5] = bound;
    __syncthreads();
    if (threadIdx.x == 0) {
        double t = 0.0;
        for (int k = 0; k < (int)(blockDim.x >> 5); ++k) t += s_part[k];
        ws.vpart[blockIdx.x] = t;
    }
}

// The fixed-point scale: 2^k with the sum of all |values| (each kernel weight
// is at most about 1, so every tile sum is bounded by it) below 2^60, so that
// 64-bit sums cannot overflow.
// (A fixed order of the sum; one thread took 45 us for the 977 partials of 2e6
// visibilities, 256 take 4.)
__global__ void __launch_bounds__(256) det_scale_kernel(WsHeader *hdr, const double *vpart,
                                                        int nparts)
{
    __shared__ double s[256];
    double b = 0.0;
    for (int i = threadIdx.x; i < nparts; i += 256) b += vpart[i];
    s[threadIdx.x] = b;
    __syncthreads();
    for (int o = 128; o > 0; o >>= 1) {
        if ((int)threadIdx.x < o) s[threadIdx.x] += s[threadIdx.x + o];
        __syncthreads();
    }
    if (threadIdx.x) return;
    int e = 0;
    frexp(s[0] * 1.01 + 1e-30, &e);  // the sum * 1.01 < 2^e
    int k = 60 - e;
    k = k > 100 ? 100 : (k < -100 ? -100 : k);
    hdr->fx_scale = ldexpf(1.0f, k);
    hdr->fx_inv = ldexpf(1.0f, -k);
}

// Slots of the tiles gridded by several work items (deterministic mode): a
// flag per tile, then its exclusive scan is the tile's slot.
__global__ void det_mc_flags_kernel(const uint32_t *gbase, uint32_t *slot, uint32_t ntiles)
{
    const uint32_t t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t < ntiles) slot[t] = gbase[t + 1] - gbase[t] > 1 ? 1u : 0u;
    if (t == ntiles) slot[t] = 0u;
}

__global__ void det_mc_count_kernel(WsHeader *hdr, const uint32_t *slot, uint32_t ntiles)
{
    hdr->mc_count = slot[ntiles];
}

// Enqueue the deterministic ordering and the records.  Keys of n records are
// in w.key (input order); nbins bins.
static rick_status det_sort_records(rick_plan *plan, WsPtrs w, const WsLayout &L, int64_t n,
                                    const void *vis, const float *weight, int n_corr,
                                    int64_t n_src, cudaStream_t st)
{
    const uint32_t nblk = (uint32_t)((n + RICK_DET_BLOCK - 1) / RICK_DET_BLOCK);
    int passes = 1;
    while (passes * RICK_DET_DIGIT < 32 && ((int64_t)1 << (passes * RICK_DET_DIGIT)) <= L.nbins)
        ++passes;
    // ping-pong between two (key, index) buffers; the input-order keys in
    // w.key stay (degridding and the density weights read them)
    const uint32_t *kin = w.key, *iin = NULL;
    uint32_t *kbuf[2] = {w.dkey, w.dkey2}, *ibuf[2] = {w.didx, w.rank};
    if (n > 0) {
        for (int ps = 0; ps < passes; ++ps) {
            const int shift = ps * RICK_DET_DIGIT;
            det_hist_kernel<<<nblk, 256, 0, st>>>(kin, n, shift, w.dcnt, nblk);
            RICK_LAUNCH_CHECK(plan);
            RICK_CUDA_TRY(plan, scan_u32(w.dcnt, w.dcnt, (int64_t)nblk << RICK_DET_DIGIT, w.scan,
                                         st, &plan->launches));
            uint32_t *ko = kbuf[ps & 1], *io = ibuf[ps & 1];
            det_scatter_kernel<<<nblk, 256, 0, st>>>(kin, iin, n, shift, w.dcnt, nblk, ko, io);
            RICK_LAUNCH_CHECK(plan);
            kin = ko;
            iin = io;
        }
    }
    int blocks = plan->num_sms * 8;
    if (blocks > (int)L.ndetblocks + 1) blocks = (int)L.ndetblocks + 1;
    if (n > 0) {
        if (n_corr > 1)
            det_records_kernel<true><<<blocks, 256, 0, st>>>(iin, (const float2 *)vis, weight, w,
                                                             n_corr, n);
        else
            det_records_kernel<false><<<blocks, 256, 0, st>>>(iin, (const float2 *)vis, weight,
                                                              w, 1, n_src);
        RICK_LAUNCH_CHECK(plan);
    }
    det_scale_kernel<<<1, 256, 0, st>>>(w.hdr, w.vpart, n > 0 ? blocks : 0);
    RICK_LAUNCH_CHECK(plan);
    return RICK_OK;
}

// ------------------------------------------------------------------------
// Pass 6: work lists.  The grid work of tile t covers its own bin (all four
// edge classes) plus the records of the west, north and north-west tiles
// whose footprints reach into t; degridding needs only the own bin.

// Work items (grid, degrid) of tile t; none for t = ntiles.
__device__ __forceinline__ uint2 tile_count(const uint32_t *off, uint32_t t, uint32_t ntiles, int nt,
                                            uint32_t cap)
{
    if (t >= ntiles) return make_uint2(0u, 0u);
    uint32_t tx = t % nt, ty = (t / nt) % nt;
    uint32_t own = off[4 * t + 4] - off[4 * t];
    uint32_t L = own;
    if (tx > 0) L += off[4 * (t - 1) + 3] - off[4 * (t - 1) + 1];
    if (ty > 0) L += off[4 * (t - nt) + 4] - off[4 * (t - nt) + 2];
    if (tx > 0 && ty > 0) L += off[4 * (t - nt - 1) + 3] - off[4 * (t - nt - 1) + 2];
    // tiles without records: no work item
    return make_uint2((L + cap - 1) / cap, (own + cap - 1) / cap);
}

__global__ void tile_count_kernel(const uint32_t *off, uint32_t *gcnt, uint32_t *dcnt,
                                  uint32_t ntiles, int nt, uint32_t cap)
{
    const uint32_t t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t > ntiles) return;
    const uint2 c = tile_count(off, t, ntiles, nt, cap);
    gcnt[t] = c.x;
    dcnt[t] = c.y;
}

// Room for the cnt entries of every lane in a list of *counter entries, in lane order:
// the first of each lane's, and of the warp's (total entries).  One atomic per warp.
struct Entries {
    uint32_t lane, warp, total;
};
__device__ __forceinline__ Entries reserve(uint32_t cnt, uint32_t *counter)
{
    const int lane = threadIdx.x & 31;
    uint32_t inc = cnt;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t v = __shfl_up_sync(FULL, inc, o);
        if (lane >= o) inc += v;
    }
    uint32_t at = 0;
    if (lane == 31 && inc) at = atomicAdd(counter, inc);
    at = __shfl_sync(FULL, at, 31);
    return {at + inc - cnt, at, __shfl_sync(FULL, inc, 31)};
}

// put(entry, owning lane, its number among the lane's) for the warp's entries, all lanes
// at it (put may shuffle; entries past the last are not to be stored).
template <typename Put>
__device__ __forceinline__ void each_entry(const Entries &e, Put put)
{
    for (uint32_t i0 = 0; i0 < e.total; i0 += 32) {
        // entry i belongs to the last lane whose entries start at or before it
        const uint32_t i = e.warp + i0 + (threadIdx.x & 31);
        int own = 0;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1)
            own += __shfl_sync(FULL, e.lane, own + o) <= i ? o : 0;
        put(i, own, i - __shfl_sync(FULL, e.lane, own));
    }
}

// The plain gridding kernel's work items, in no particular order: a thread per
// subtile counts its chunks (its class-0 sub-bin and, in the last column and
// row of subtiles, those of the other classes).
__device__ __forceinline__ uint32_t chunks_of(uint32_t s, uint32_t nsubtiles, const SubShape &sub,
                                              uint32_t cap, const WsPtrs &w)
{
    if (s >= nsubtiles) return 0;
    uint32_t n = 0;
#pragma unroll
    for (int g = 0; g < 4; ++g) {
        const int64_t id = rick_subtile_range(sub, s, g);
        if (id >= 0) n += w.suboff[id + 1] - w.suboff[id];
    }
    return rick_sub_chunks(n, cap);
}

// The entries of a warp's subtiles (s consecutive, with cnt chunks each) in the lists of
// groups, single items and slots, whose lengths are len.  All lanes of the warp.
struct SubEntries {
    uint32_t ng, slot;
    Entries groups, singles;
};
__device__ __forceinline__ SubEntries reserve_items(uint32_t cnt, uint32_t *len)
{
    SubEntries e = {};
    e.slot = ~0u;
    if (!__any_sync(FULL, cnt != 0)) return e;
    e.ng = cnt / RICK_SUB_GROUP;
    const uint32_t ns = rick_sub_slots(e.ng);
    if (__any_sync(FULL, ns != 0)) {
        const uint32_t at = reserve(ns, len + 2).lane;
        if (ns) e.slot = at;
    }
    e.groups = reserve(e.ng, len);
    e.singles = reserve(cnt - e.ng * RICK_SUB_GROUP, len + 1);
    return e;
}

// at: where len's lists begin.
__device__ __forceinline__ void write_items(const SubEntries &e, uint32_t s, const uint32_t *at,
                                            uint32_t nslots, const WsPtrs &w)
{
    const uint32_t s0 = s - (threadIdx.x & 31);
    uint32_t slot = e.slot;
    if (slot != ~0u) {
        slot += at[2];
        if (slot + rick_sub_slots(e.ng) > nslots) slot = ~0u;
    }
    each_entry(e.groups, [&](uint32_t i, int own, uint32_t k) {
        const uint32_t first = __shfl_sync(FULL, slot, own), all = __shfl_sync(FULL, e.ng, own);
        if (i < e.groups.warp + e.groups.total)
            w.groups[at[0] + i] = make_uint4(s0 + own, RICK_SUB_GROUP * k, first, all);
    });
    each_entry(e.singles, [&](uint32_t i, int own, uint32_t k) {
        const uint32_t c = __shfl_sync(FULL, e.ng, own) * RICK_SUB_GROUP + k;
        if (i < e.singles.warp + e.singles.total) w.items[at[1] + i] = make_uint2(s0 + own, c);
    });
}

// One atomic per list and block on the lists' lengths: they pass one by one, 3.5 ns each
// (one per warp and list: 410 us of binning, against 269 for tiles, for 1e6 visibilities
// spread over 8e6 subtiles).  U subtiles a thread, their counts in flight together: four
// for large grids, where blocks of 1024 are enough to fill the GPU.
template <int U>
__global__ void __launch_bounds__(256) sub_items_kernel(WsPtrs w, uint32_t nsubtiles, SubShape sub,
                                                        uint32_t nslots)
{
    __shared__ uint32_t s_len[3], s_at[3];
    const uint32_t s = blockIdx.x * (256 * U) + threadIdx.x, cap = w.hdr->sub_cap;
    if (threadIdx.x < 3) s_len[threadIdx.x] = 0;
    uint32_t cnt[U], any = 0;
    SubEntries e[U];
#pragma unroll
    for (int u = 0; u < U; ++u) any |= cnt[u] = chunks_of(s + 256 * u, nsubtiles, sub, cap, w);
    if (!__syncthreads_or(any != 0)) return;
#pragma unroll
    for (int u = 0; u < U; ++u) e[u] = reserve_items(cnt[u], s_len);
    __syncthreads();
    if (threadIdx.x < 3 && s_len[threadIdx.x]) {
        uint32_t *len = threadIdx.x == 0 ? &w.hdr->n_groups
                      : threadIdx.x == 1 ? &w.hdr->n_items : &w.hdr->n_slots;
        s_at[threadIdx.x] = atomicAdd(len, s_len[threadIdx.x]);
    }
    __syncthreads();
#pragma unroll
    for (int u = 0; u < U; ++u) write_items(e[u], s + 256 * u, s_at, nslots, w);
}

// Exclusive scan of n values by one CTA of 1024 threads, eight consecutive values a
// thread and round: put(i, sum of get(j < i)).
template <typename Get, typename Put>
__device__ __forceinline__ void scan_cta(int64_t n, Get get, Put put)
{
    __shared__ uint32_t s_warp[32];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    uint32_t carry = 0;
    for (int64_t b = 0; b < n; b += 8 * 1024) {
        const int64_t i0 = b + 8 * threadIdx.x;
        uint32_t v[8], sum = 0;
#pragma unroll
        for (int u = 0; u < 8; ++u) v[u] = i0 + u < n ? get(i0 + u) : 0u;
#pragma unroll
        for (int u = 0; u < 8; ++u) {
            const uint32_t x = v[u];
            v[u] = sum;
            sum += x;
        }
        uint32_t inc = sum;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t x = __shfl_up_sync(FULL, inc, o);
            if (lane >= o) inc += x;
        }
        __syncthreads();  // the last round's totals have been read
        if (lane == 31) s_warp[wid] = inc;
        __syncthreads();
        uint32_t before = 0, total = 0;
        for (int k = 0; k < 32; ++k) {
            const uint32_t x = s_warp[k];
            if (k < wid) before += x;
            total += x;
        }
        const uint32_t first = carry + before + inc - sum;
#pragma unroll
        for (int u = 0; u < 8; ++u)
            if (i0 + u < n) put(i0 + u, first + v[u]);
        carry += total;
    }
}

// Everything between the key pass and the scatter, and the work lists, by one CTA:
// for grids of few sub-bins the dozen launches of the general path cost more than
// the work (4 planes of 512^2: 31 us of GPU time and gaps against 9).
#define RICK_SMALL_SUBS 16384

struct SmallArgs {
    WsPtrs w;
    SubShape sub;
    int nparts, unit_weights, nt, plain;
    uint32_t ntiles, cap, nslots;
    int64_t nsubs, nbins;
    rick_bin_stats *stats_out;
};

__global__ void __launch_bounds__(1024) bin_small_kernel(SmallArgs a)
{
    const WsPtrs &w = a.w;
    bin_finalize(w.hdr, w.wpart, a.nparts, a.unit_weights, a.stats_out);
    scan_cta(a.nsubs + 1, [&](int64_t i) { return w.hist[i]; },
             [&](int64_t i, uint32_t v) { w.suboff[i] = v; });
    __syncthreads();
    for (int64_t b = threadIdx.x; b <= a.nbins; b += 1024)
        w.offsets[b] = w.suboff[(b >> 2) * a.sub.per + rick_sub_first(a.sub, (uint32_t)b & 3u)];
    __syncthreads();
    scan_cta((int64_t)a.ntiles + 1,
             [&](int64_t t) { return tile_count(w.offsets, (uint32_t)t, a.ntiles, a.nt, a.cap).x; },
             [&](int64_t t, uint32_t v) { w.gbase[t] = v; });
    scan_cta((int64_t)a.ntiles + 1,
             [&](int64_t t) { return tile_count(w.offsets, (uint32_t)t, a.ntiles, a.nt, a.cap).y; },
             [&](int64_t t, uint32_t v) { w.dbase[t] = v; });
    if (a.plain) {
        // the lists' lengths in shared memory until they are known
        __shared__ uint32_t s_len[3], s_at[3];
        if (threadIdx.x < 3) s_len[threadIdx.x] = s_at[threadIdx.x] = 0;
        __syncthreads();
        const uint32_t ns = a.ntiles << (2 * a.sub.lq), cap = w.hdr->sub_cap;
        for (uint32_t s = threadIdx.x; s < ((ns + 31) & ~31u); s += 1024)
            write_items(reserve_items(chunks_of(s, ns, a.sub, cap, w), s_len), s, s_at, a.nslots, w);
        __syncthreads();
        if (threadIdx.x == 0) {
            w.hdr->n_groups = s_len[0];
            w.hdr->n_items = s_len[1];
            w.hdr->n_slots = s_len[2];
        }
    }
}

// The first launch of a binning: header, histogram, planes of a given range.
static rick_status launch_init(rick_plan *plan, const WsPtrs &w, const WsLayout &L, int64_t n_vis,
                               uint32_t cap, int given, int64_t nkb, const WsHeader *range_src,
                               int64_t n_src, int mirror, cudaStream_t st)
{
    const rick_params &p = plan->p;
    const bool own = !isnan(p.w_min);
    int64_t blocks = (L.nsubs + 1 + 4 * 1024 - 1) / (4 * 1024);
    if (blocks > plan->num_sms * 8) blocks = plan->num_sms * 8;
    bin_init_kernel<<<(unsigned)blocks, 256, 0, st>>>(
        w, (uint64_t)n_vis, cap, given, own ? rick_dkey(p.w_min) : 0, own ? rick_dkey(p.w_max) : 0,
        (uint32_t)nkb, range_src, (uint64_t)n_src, mirror, rick_sub_cap(n_vis, plan->num_sms),
        L.nsubs + 1, p.n_w);
    RICK_LAUNCH_CHECK(plan);
    return RICK_OK;
}

// After the key pass: the stats and the sub-bin and bin offsets; with small also
// the work lists.
static rick_status launch_offsets(rick_plan *plan, const WsPtrs &w, const WsLayout &L,
                                  const SubShape &sub, bool small, int nparts, int unit_weights,
                                  uint32_t cap, rick_bin_stats *stats_out, cudaStream_t st)
{
    if (small) {
        const SmallArgs a = {w, sub, nparts, unit_weights, plan->p.n / plan->p.tile,
                             rick_grid_plain(&plan->p), (uint32_t)L.ntiles, cap,
                             (uint32_t)L.nslots, L.nsubs, L.nbins,
                             stats_out};
        bin_small_kernel<<<1, 1024, 0, st>>>(a);
        RICK_LAUNCH_CHECK(plan);
        return RICK_OK;
    }
    bin_finalize_kernel<<<1, 1024, 0, st>>>(w.hdr, w.wpart, nparts, unit_weights, stats_out);
    RICK_LAUNCH_CHECK(plan);
    RICK_CUDA_TRY(plan, scan_u32(w.hist, w.suboff, L.nsubs + 1, w.scan, st, &plan->launches));
    bin_offsets_kernel<<<(unsigned)((L.nbins + 256) / 256), 256, 0, st>>>(w.suboff, w.offsets,
                                                                          L.nbins, sub);
    RICK_LAUNCH_CHECK(plan);
    return RICK_OK;
}

static rick_status launch_lists(rick_plan *plan, const WsPtrs &w, const WsLayout &L, uint32_t cap,
                                cudaStream_t st)
{
    const uint32_t nt = (uint32_t)L.ntiles;
    tile_count_kernel<<<(nt + 256) / 256, 256, 0, st>>>(w.offsets, w.gbase, w.dbase, nt,
                                                        plan->p.n / plan->p.tile, cap);
    RICK_LAUNCH_CHECK(plan);
    RICK_CUDA_TRY(plan, scan_u32(w.gbase, w.gbase, L.ntiles + 1, w.scan, st, &plan->launches));
    RICK_CUDA_TRY(plan, scan_u32(w.dbase, w.dbase, L.ntiles + 1, w.scan, st, &plan->launches));
    if (!rick_grid_plain(&plan->p)) return RICK_OK;
    const SubShape sub = rick_sub_shape(&plan->p);
    const uint32_t ns = (uint32_t)(L.ntiles << (2 * sub.lq));
    if (ns > 1u << 20)
        sub_items_kernel<4><<<(ns + 1023) / 1024, 256, 0, st>>>(w, ns, sub, (uint32_t)L.nslots);
    else
        sub_items_kernel<1><<<(ns + 255) / 256, 256, 0, st>>>(w, ns, sub, (uint32_t)L.nslots);
    RICK_LAUNCH_CHECK(plan);
    return RICK_OK;
}

// ------------------------------------------------------------------------

// Rows of n_chan channels that fit a plan's capacity.
static int64_t plan_max_rows(const rick_plan *plan, int32_t n_chan)
{
    return plan && n_chan > 0 ? plan->max_vis / n_chan : 0;
}

rick_status rick_bin_impl(rick_plan *plan, int64_t n_vis, const double *uvw, const void *vis,
                          const float *weight, void *ws_dev, size_t ws_bytes,
                          rick_bin_stats *stats_dev, void *stream, const WsHeader *range_src,
                          int n_chan, const double *chan_scale, int n_corr)
{
    if (!plan || !ws_dev || n_vis < 0 || n_corr < 1 || n_corr > RICK_MAX_CORR) return RICK_EINVAL;
    if (plan->sticky != RICK_OK) return plan->sticky;
    if (n_vis > 0 && (!uvw || !vis)) return RICK_EINVAL;
    if (((uintptr_t)ws_dev & 255) || ((uintptr_t)uvw & 7) || ((uintptr_t)vis & 7) ||
        ((uintptr_t)weight & 3) || ((uintptr_t)stats_dev & 7) || ((uintptr_t)chan_scale & 7))
        return RICK_EINVAL;
    if (n_chan < 0 || (n_chan > 0 && n_vis > 0 && !chan_scale)) return RICK_EINVAL;
    if (n_vis > plan->max_vis) return RICK_ERANGE;
    const rick_params &p = plan->p;
    // the Hermitian mirror: input-order records, then the mirrored ones (per-
    // visibility input only: not with channels, correlations or streaming)
    const int mirror = (p.options & RICK_OPT_HERMITIAN_MIRROR) != 0;
    if (mirror && (n_chan > 0 || n_corr != 1 || range_src)) return RICK_EINVAL;
    const int64_t n_src = n_vis;
    n_vis = rick_n_records(&p, n_src);  // records from here on
    WsLayout L = rick_ws_layout(&p, plan->max_vis);
    if (ws_bytes < L.total) return RICK_ERANGE;
    const int64_t nkb = (n_vis + RICK_KEY_THREADS * RICK_KEY_ITEMS - 1) /
                        (RICK_KEY_THREADS * RICK_KEY_ITEMS);
    WsPtrs w = rick_ws_ptrs(ws_dev, L);
    const SubShape sub = rick_sub_shape(&p);
    cudaStream_t st = (cudaStream_t)stream;
    const bool det = (p.options & RICK_OPT_DETERMINISTIC) != 0;
    uint32_t cap = rick_chunk_cap(n_vis, plan->num_sms, rick_grid_plain(&p));
    if (det) {
        // enough records per work item that the tiles with several items fit
        // the workspace's slots (a record is visited by at most four tiles)
        const int64_t slots = rick_det_slots(&p, rick_n_records(&p, plan->max_vis));
        int64_t c = (4 * n_vis + slots - 1) / slots;
        c = (c + 255) & ~(int64_t)255;
        if (c > cap) cap = (uint32_t)c;
    }
    int given = !isnan(p.w_min) || range_src != NULL;

    const rick_status is = launch_init(plan, w, L, n_vis, cap, given, nkb, range_src, n_src, mirror,
                                       st);
    if (is != RICK_OK) return is;
    if (!given && n_vis > 0) {
        const int blocks = wrange_blocks(plan, n_chan > 0 ? n_src / n_chan : n_src);
        if (mirror)
            wrange_kernel<true><<<blocks, 256, 0, st>>>(uvw, n_src, w.hdr, n_chan, chan_scale,
                                                        w.bkey, w.wplane, p.n_w);
        else
            wrange_kernel<false><<<blocks, 256, 0, st>>>(uvw, n_src, w.hdr, n_chan, chan_scale,
                                                         w.bkey, w.wplane, p.n_w);
        RICK_LAUNCH_CHECK(plan);
    }

    if (n_vis > 0) {
        KeyArgs ka;
        ka.n_vis = n_vis;
        ka.uvw = uvw;
        ka.weight = weight;
        ka.n = p.n;
        ka.n_w = p.n_w;
        ka.W = p.support;
        ka.log2T = 0;
        while ((1 << ka.log2T) < p.tile) ++ka.log2T;
        ka.nt = p.n / p.tile;
        ka.fov = p.fov;
        ka.half_n = 0.5 * p.n;
        ka.key_lo = rick_dkey(-0.5);
        ka.key_hi = rick_dkey((double)p.n + 0.5);
        ka.ws = w;
        ka.n_chan = n_chan;
        ka.n_corr = n_corr;
        ka.chan_scale = chan_scale;
        ka.n_src = mirror ? n_src : n_vis;
        ka.wait_polls = plan->wait_polls;
        ka.sub = sub;
        ka.bulk = n_chan == 0 && n_corr == 1 && ((uintptr_t)uvw & 15) == 0 &&
                  ((uintptr_t)weight & 15) == 0;
        const size_t smem = key_pass_smem(p.n_w);
        RICK_CUDA_TRY(plan, cudaFuncSetAttribute(bin_key_kernel,
                                                 cudaFuncAttributeMaxDynamicSharedMemorySize,
                                                 (int)smem));
        bin_key_kernel<<<(unsigned)nkb, RICK_KEY_THREADS, smem, st>>>(ka);
        RICK_LAUNCH_CHECK(plan);
    }
    const bool small = !det && L.nsubs <= RICK_SMALL_SUBS;
    const rick_status os = launch_offsets(plan, w, L, sub, small, (int)nkb,
                                          weight == NULL ? n_corr : 0, cap, stats_dev, st);
    if (os != RICK_OK) return os;
    if (det) {
        rick_status ds = det_sort_records(plan, w, L, n_vis, vis, weight, n_corr,
                                          mirror ? n_src : n_vis, st);
        if (ds != RICK_OK) return ds;
    } else if (n_vis > 0) {
        int64_t blocks = (n_vis + 256 * RICK_SCATTER_U - 1) / (256 * RICK_SCATTER_U);
        if (blocks > (int64_t)plan->num_sms * 64) blocks = (int64_t)plan->num_sms * 64;
        if (n_corr > 1)
            bin_scatter_kernel<true, false><<<(unsigned)blocks, 256, 0, st>>>(
                n_vis, (const float2 *)vis, weight, w, n_corr, n_vis, sub);
        else if (mirror)
            bin_scatter_kernel<false, true><<<(unsigned)blocks, 256, 0, st>>>(
                n_vis, (const float2 *)vis, weight, w, 1, n_src, sub);
        else
            bin_scatter_kernel<false, false><<<(unsigned)blocks, 256, 0, st>>>(
                n_vis, (const float2 *)vis, weight, w, 1, n_vis, sub);
        RICK_LAUNCH_CHECK(plan);
    }
    const uint32_t nt = (uint32_t)L.ntiles;
    if (!small) {
        const rick_status ls = launch_lists(plan, w, L, cap, st);
        if (ls != RICK_OK) return ls;
    }
    if (det) {  // slots of the tiles with several grid work items
        det_mc_flags_kernel<<<(nt + 256) / 256, 256, 0, st>>>(w.gbase, w.mcslot, nt);
        RICK_LAUNCH_CHECK(plan);
        RICK_CUDA_TRY(plan, scan_u32(w.mcslot, w.mcslot, L.ntiles + 1, w.scan, st,
                                     &plan->launches));
        det_mc_count_kernel<<<1, 1, 0, st>>>(w.hdr, w.mcslot, nt);
        RICK_LAUNCH_CHECK(plan);
    }
    return RICK_OK;
}

extern "C" rick_status rick_bin(rick_plan *plan, int64_t n_vis, const double *uvw,
                                const void *vis, const float *weight, void *ws_dev,
                                size_t ws_bytes, rick_bin_stats *stats_dev, void *stream)
{
    return rick_bin_impl(plan, n_vis, uvw, vis, weight, ws_dev, ws_bytes, stats_dev, stream, NULL,
                         0, NULL, 1);
}

extern "C" rick_status rick_bin_channels(rick_plan *plan, int64_t n_rows, int32_t n_chan,
                                         const double *uvw_rows, const double *chan_scale,
                                         const void *vis, const float *weight, void *ws_dev,
                                         size_t ws_bytes, rick_bin_stats *stats_dev, void *stream)
{
    if (!plan || n_rows < 0 || n_chan < 1) return RICK_EINVAL;
    if (n_rows > 0 && !chan_scale) return RICK_EINVAL;
    if (n_rows > plan_max_rows(plan, n_chan)) return RICK_ERANGE;
    return rick_bin_impl(plan, n_rows * n_chan, uvw_rows, vis, weight, ws_dev, ws_bytes, stats_dev,
                         stream, NULL, n_chan, chan_scale, 1);
}

extern "C" rick_status rick_bin_rows(rick_plan *plan, int64_t n_rows, int32_t n_chan,
                                     int32_t n_corr, const double *uvw_rows,
                                     const double *chan_scale, const void *vis,
                                     const float *weight, void *ws_dev, size_t ws_bytes,
                                     rick_bin_stats *stats_dev, void *stream)
{
    if (!plan || n_rows < 0 || n_chan < 1 || n_corr < 1 || n_corr > RICK_MAX_CORR)
        return RICK_EINVAL;
    if (n_rows > 0 && !chan_scale) return RICK_EINVAL;
    if (n_rows > plan_max_rows(plan, n_chan)) return RICK_ERANGE;
    return rick_bin_impl(plan, n_rows * n_chan, uvw_rows, vis, weight, ws_dev, ws_bytes, stats_dev,
                         stream, NULL, n_chan, chan_scale, n_corr);
}

static rick_status bin_values_impl(rick_plan *plan, const void *vis, const float *weight,
                                   const float *grad, void *ws_dev, rick_bin_stats *stats_dev,
                                   void *stream)
{
    if (!plan || !vis || !ws_dev) return RICK_EINVAL;
    if (plan->sticky != RICK_OK) return plan->sticky;
    if (((uintptr_t)ws_dev & 255) || ((uintptr_t)vis & 7) || ((uintptr_t)weight & 3) ||
        ((uintptr_t)stats_dev & 7))
        return RICK_EINVAL;
    cudaStream_t st = (cudaStream_t)stream;
    const WsLayout L = rick_ws_layout(&plan->p, plan->max_vis);
    WsPtrs w = rick_ws_ptrs(ws_dev, L);
    // one weight partial per block: the workspace holds nkeyblocks + 1 of them
    // (and ndetblocks + 1 bound partials in deterministic mode)
    const int det = (plan->p.options & RICK_OPT_DETERMINISTIC) != 0;
    int blocks = plan->num_sms * 8;
    if (blocks > (int)L.nkeyblocks + 1) blocks = (int)L.nkeyblocks + 1;
    if (det && blocks > (int)L.ndetblocks + 1) blocks = (int)L.ndetblocks + 1;
    if (grad)
        bin_values_kernel<true><<<blocks, 256, 0, st>>>((const float2 *)vis, weight, w, det, grad);
    else
        bin_values_kernel<false><<<blocks, 256, 0, st>>>((const float2 *)vis, weight, w, det, NULL);
    RICK_LAUNCH_CHECK(plan);
    values_finalize_kernel<<<1, 1024, 0, st>>>(w.wpart, blocks, grad || !weight, w.hdr,
                                               stats_dev);
    RICK_LAUNCH_CHECK(plan);
    if (det) {  // the fixed-point scale for the new values
        det_scale_kernel<<<1, 256, 0, st>>>(w.hdr, w.vpart, blocks);
        RICK_LAUNCH_CHECK(plan);
    }
    return RICK_OK;
}

extern "C" rick_status rick_bin_values(rick_plan *plan, const void *vis, const float *weight,
                                       void *ws_dev, rick_bin_stats *stats_dev, void *stream)
{
    return bin_values_impl(plan, vis, weight, NULL, ws_dev, stats_dev, stream);
}

extern "C" rick_status rick_bin_residuals(rick_plan *plan, const void *resid, const float *weight,
                                          const float *grad, void *ws_dev,
                                          rick_bin_stats *stats_dev, void *stream)
{
    if (!weight || !grad || ((uintptr_t)grad & 3)) return RICK_EINVAL;
    return bin_values_impl(plan, resid, weight, grad, ws_dev, stats_dev, stream);
}

// chi^2 and the residuals in one pass over the visibilities (20 bytes read, 8
// written each; as torch operations the same took nine passes and their
// gradients as many: 1e7 visibilities, 450 us against 60 with the second kernel).
__global__ void __launch_bounds__(256) chi2_residuals_kernel(int64_t n, const float2 *vis,
                                                             const float *weight, float2 *model,
                                                             double *partials)
{
    __shared__ double s[8];
    double t = 0.0;
    const int64_t step = (int64_t)gridDim.x * blockDim.x;
    int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    // four visibilities in flight; their FP32 terms are added in FP32 pairs of
    // double-single first (FP64 issues at a sixty-fourth of the rate), and in plain FP32
    // for sums that are not finite, of which a pair makes NaN (inf - inf)
    ff acc = {0.0f, 0.0f};
    float plain = 0.0f;
    for (; i < n; i += 4 * step) {
        float2 o[4], m[4];
        float w[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const int64_t j = i + u * step;
            o[u] = m[u] = make_float2(0.0f, 0.0f);
            w[u] = 0.0f;
            if (j < n) {
                o[u] = vis[j];
                m[u] = model[j];
                w[u] = weight[j];
            }
        }
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const int64_t j = i + u * step;
            if (j >= n) continue;
            const float2 r = make_float2(o[u].x - m[u].x, o[u].y - m[u].y);
            model[j] = r;
            const float e = w[u] * __fadd_rn(__fmul_rn(r.x, r.x), __fmul_rn(r.y, r.y));
            acc = ff_add(acc, ff{e, 0.0f});
            plain += e;
        }
    }
    t = isfinite(acc.hi) ? (double)acc.hi + (double)acc.lo : (double)plain;
    for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(FULL, t, o);
    if ((threadIdx.x & 31) == 0) s[threadIdx.x >> 5] = t;
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int k = 1; k < 8; ++k) t += s[k];
        partials[blockIdx.x] = t;
    }
}

__global__ void __launch_bounds__(RICK_CHI2_PARTIALS) chi2_sum_kernel(const double *partials,
                                                                      int nparts, float *chi2)
{
    __shared__ double s[RICK_CHI2_PARTIALS];
    s[threadIdx.x] = (int)threadIdx.x < nparts ? partials[threadIdx.x] : 0.0;
    __syncthreads();
    for (int o = RICK_CHI2_PARTIALS / 2; o > 0; o >>= 1) {
        if ((int)threadIdx.x < o) s[threadIdx.x] += s[threadIdx.x + o];
        __syncthreads();
    }
    if (threadIdx.x == 0) *chi2 = (float)s[0];
}

extern "C" rick_status rick_chi2_residuals(rick_plan *plan, int64_t n_vis, const void *vis,
                                           const float *weight, void *model, double *partials,
                                           float *chi2, void *stream)
{
    if (!plan || n_vis < 0 || !partials || !chi2) return RICK_EINVAL;
    if (n_vis > 0 && (!vis || !weight || !model)) return RICK_EINVAL;
    if (((uintptr_t)vis & 7) || ((uintptr_t)model & 7) || ((uintptr_t)weight & 3) ||
        ((uintptr_t)partials & 7) || ((uintptr_t)chi2 & 3))
        return RICK_EINVAL;
    if (plan->sticky != RICK_OK) return plan->sticky;
    cudaStream_t st = (cudaStream_t)stream;
    int blocks = (int)((n_vis + 1023) / 1024 < RICK_CHI2_PARTIALS ? (n_vis + 1023) / 1024
                                                                   : RICK_CHI2_PARTIALS);
    if (blocks < 1) blocks = 1;
    chi2_residuals_kernel<<<blocks, 256, 0, st>>>(n_vis, (const float2 *)vis, weight,
                                                  (float2 *)model, partials);
    RICK_LAUNCH_CHECK(plan);
    chi2_sum_kernel<<<1, RICK_CHI2_PARTIALS, 0, st>>>(partials, blocks, chi2);
    RICK_LAUNCH_CHECK(plan);
    return RICK_OK;
}

// ------------------------------------------------------------------------
// rick_bin_noalloc: the binning above for callers that must not allocate
// device memory.  Its temporaries -- the per-visibility ranks and fractional
// offsets, the histogram, the scan temporaries and the weight-sum
// partials -- live in this file-scope array instead of the
// caller's workspace.  The per-visibility keys and corner cells stay in the
// caller's workspace, where rick_bin writes them: degridding and the density
// weights read them after the binning.  The array is part of the library
// image: every GPU that loads librick.so holds it (about 13.8 MB) until the
// process exits.

#define NOALLOC_MAX_VIS (1 << 18)
#define NOALLOC_MAX_BINS (1 << 17)
#define NOALLOC_FRAC (0)
#define NOALLOC_RANK (NOALLOC_FRAC + 8 * NOALLOC_MAX_VIS)
#define NOALLOC_HIST (NOALLOC_RANK + 4 * NOALLOC_MAX_VIS)
#define NOALLOC_MAX_SUBS (81 * (NOALLOC_MAX_BINS / 4))  // tile 128: 81 sub-bins per tile of 4 bins
#define NOALLOC_SCAN (NOALLOC_HIST + 4 * (NOALLOC_MAX_SUBS + 256))
#define NOALLOC_WPART (NOALLOC_SCAN + 4 * 4096)
#define NOALLOC_BYTES (NOALLOC_WPART + 8 * (NOALLOC_MAX_VIS / (RICK_KEY_THREADS * RICK_KEY_ITEMS) + 256))

static __device__ __align__(256) unsigned char g_noalloc_scratch[NOALLOC_BYTES];

// The array's device address, looked up once per device with that device
// current (a host-side name of a __device__ array is not a device address).
#define NOALLOC_MAX_DEVICES 64
static void *g_noalloc_addr[NOALLOC_MAX_DEVICES];
static std::mutex g_noalloc_mu;

static rick_status noalloc_scratch(unsigned char **out)
{
    int dev = -1;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= NOALLOC_MAX_DEVICES)
        return RICK_ECUDA;
    std::lock_guard<std::mutex> lock(g_noalloc_mu);
    if (!g_noalloc_addr[dev]) {
        void *ptr = NULL;
        if (cudaGetSymbolAddress(&ptr, g_noalloc_scratch) != cudaSuccess || !ptr) return RICK_ECUDA;
        g_noalloc_addr[dev] = ptr;
    }
    *out = (unsigned char *)g_noalloc_addr[dev];
    return RICK_OK;
}

extern "C" rick_status rick_bin_noalloc(rick_plan *plan, int64_t n_vis, const double *uvw,
                                        const void *vis, const float *weight, void *ws_dev,
                                        size_t ws_bytes, rick_bin_stats *stats_dev, void *stream)
{
    if (!plan || !ws_dev || n_vis < 0) return RICK_EINVAL;
    if (plan->sticky != RICK_OK) return plan->sticky;
    if (n_vis > 0 && (!uvw || !vis)) return RICK_EINVAL;
    if (((uintptr_t)ws_dev & 255) || ((uintptr_t)uvw & 7) || ((uintptr_t)vis & 7) ||
        ((uintptr_t)weight & 3) || ((uintptr_t)stats_dev & 7))
        return RICK_EINVAL;
    if (n_vis > plan->max_vis) return RICK_ERANGE;
    const rick_params &p = plan->p;
    if (p.options != 0) return RICK_EINVAL;  // plain binning only
    WsLayout L = rick_ws_layout(&p, plan->max_vis);
    if (ws_bytes < L.total) return RICK_ERANGE;
    // the fixed scratch bounds the problem size
    if (n_vis > NOALLOC_MAX_VIS || L.nbins > NOALLOC_MAX_BINS) return RICK_ERANGE;
    unsigned char *scratch = NULL;
    rick_status sst = noalloc_scratch(&scratch);
    if (sst != RICK_OK) {
        plan->sticky = sst;
        return sst;
    }
    const int64_t nkb = (n_vis + RICK_KEY_THREADS * RICK_KEY_ITEMS - 1) /
                        (RICK_KEY_THREADS * RICK_KEY_ITEMS);
    // outputs (records, offsets, work lists, and the keys and corner cells that
    // later calls read) in the caller's workspace, temporaries in the fixed array
    WsPtrs w = rick_ws_ptrs(ws_dev, L);
    const SubShape sub = rick_sub_shape(&p);
    w.rank = (uint32_t *)(scratch + NOALLOC_RANK);
    w.frac = (float2 *)(scratch + NOALLOC_FRAC);
    w.hist = (uint32_t *)(scratch + NOALLOC_HIST);
    w.scan = (uint32_t *)(scratch + NOALLOC_SCAN);
    w.wpart = (double *)(scratch + NOALLOC_WPART);
    cudaStream_t st = (cudaStream_t)stream;
    uint32_t cap = rick_chunk_cap(n_vis, plan->num_sms, rick_grid_plain(&p));
    int given = !isnan(p.w_min);

    // the same stages as rick_bin, in the same order; the array keeps the last
    // call's contents, and the first launch zeroes the histogram
    const rick_status is = launch_init(plan, w, L, n_vis, cap, given, nkb, NULL, n_vis, 0, st);
    if (is != RICK_OK) return is;
    if (!given && n_vis > 0) {
        wrange_kernel<false><<<wrange_blocks(plan, n_vis), 256, 0, st>>>(uvw, n_vis, w.hdr, 0, NULL,
                                                                         w.bkey, w.wplane, p.n_w);
        RICK_LAUNCH_CHECK(plan);
    }
    if (n_vis > 0) {
        KeyArgs ka;
        ka.n_vis = n_vis;
        ka.uvw = uvw;
        ka.weight = weight;
        ka.n = p.n;
        ka.n_w = p.n_w;
        ka.W = p.support;
        ka.log2T = 0;
        while ((1 << ka.log2T) < p.tile) ++ka.log2T;
        ka.nt = p.n / p.tile;
        ka.fov = p.fov;
        ka.half_n = 0.5 * p.n;
        ka.key_lo = rick_dkey(-0.5);
        ka.key_hi = rick_dkey((double)p.n + 0.5);
        ka.ws = w;
        ka.n_chan = 0;
        ka.n_corr = 1;
        ka.chan_scale = NULL;
        ka.n_src = n_vis;
        ka.wait_polls = plan->wait_polls;
        ka.sub = sub;
        ka.bulk = ((uintptr_t)uvw & 15) == 0 && ((uintptr_t)weight & 15) == 0;
        const size_t smem = key_pass_smem(p.n_w);
        RICK_CUDA_TRY(plan, cudaFuncSetAttribute(bin_key_kernel,
                                                 cudaFuncAttributeMaxDynamicSharedMemorySize,
                                                 (int)smem));
        bin_key_kernel<<<(unsigned)nkb, RICK_KEY_THREADS, smem, st>>>(ka);
        RICK_LAUNCH_CHECK(plan);
    }
    const bool small = L.nsubs <= RICK_SMALL_SUBS;
    const rick_status os = launch_offsets(plan, w, L, sub, small, (int)nkb, weight == NULL, cap,
                                          stats_dev, st);
    if (os != RICK_OK) return os;
    if (n_vis > 0) {
        int64_t blocks = (n_vis + 256 * RICK_SCATTER_U - 1) / (256 * RICK_SCATTER_U);
        if (blocks > (int64_t)plan->num_sms * 64) blocks = (int64_t)plan->num_sms * 64;
        bin_scatter_kernel<false, false><<<(unsigned)blocks, 256, 0, st>>>(
            n_vis, (const float2 *)vis, weight, w, 1, n_vis, sub);
        RICK_LAUNCH_CHECK(plan);
    }
    if (!small) return launch_lists(plan, w, L, cap, st);
    return RICK_OK;
}
