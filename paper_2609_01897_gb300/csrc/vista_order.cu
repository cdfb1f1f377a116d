// Row ordering, per-row FP64 records and the work list of the mixed path.
//
// Rows of each window are put in uv-cell order so that the stacking kernel's
// per-lane running sums absorb consecutive rows that share a cell, and the
// work list walks the cube stripe by stripe (a stripe = a few iv rows of the
// cube, sized to stay resident in L2) across all windows.
//
//   k_keys         cell of every row at the window's middle in-cube channel
//                  (from where a row's cell moves least towards both ends of
//                  the band: 3 to 11 % fewer finished runs than at the highest
//                  frequency on narrow bands, 4 % more on a 20 % wide one) ->
//                  (stripe, local cell key); stripe counts per segment of
//                  rows; a re-projected window's gridding baselines
//                  R (u, v, w) (Eq. 1)
//   k_segscan      segment offsets inside each (window, stripe) bucket (a
//                  warp scan per bucket)
//   k_slots        each row's slot in its bucket, in row order
//   k_scan         one block: per-window bucket offsets, per-bucket work-list
//                  offsets, class by class in stripe-major order (item = rows of one bucket x
//                  one chunk)
//   k_items        the work list, one thread per item
//   k_scatter      rows grouped by bucket
//   k_bucket_sort  one block per bucket: stable counting sort by local cell
//                  key (the rows of one key stay in row order), one
//                  contiguous part of the bucket per warp
//   k_rows         per row, in processing order (rows of one cell by the part
//                  of the cell they lie in, see part_order): the FP64 delay of
//                  Eq. 2 as a float-float pair, the weights, and the uv cells
//                  of each of the window's channel chunks
#include "vista_device.cuh"

namespace vista {

// Row-order slots in (window, stripe) buckets, three passes over segments of
// seg_rows rows: keys and per-segment stripe counts, an exclusive scan of the
// counts over each window's segments, then each segment's slots in row order
// (ranks within a warp from a match, warps in turn against running counts in
// shared memory).  Rows that share a bucket thus keep their row order.
constexpr uint32_t NO_BUCKET = 0xffffffffu;

struct SegRange {
    int w;
    int64_t g0, r0, r1;   // first global row of the window, rows [r0, r1) of the segment
};
__device__ __forceinline__ SegRange seg_range(const RunArgs &a, int64_t seg)
{
    SegRange sr;
    sr.w = find_owner(a.so.seg_off, a.nsrc, seg);
    sr.g0 = a.row_off[sr.w];
    sr.r0 = (seg - a.so.seg_off[sr.w]) * a.so.seg_rows;
    const int64_t n = a.srcs[sr.w].nrow;
    sr.r1 = sr.r0 + a.so.seg_rows < n ? sr.r0 + a.so.seg_rows : n;
    return sr;
}

// Pass 1: the cell of every row at the window's middle in-cube channel ->
// (stripe, local cell key), and the stripe counts of the segment.
__global__ void __launch_bounds__(256) k_keys(RunArgs a)
{
    chain_begin();
    __shared__ uint32_t cnt[MAX_STRIPES];
    const SortArgs &so = a.so;
    const int64_t seg = blockIdx.x;
    const SegRange sr = seg_range(a, seg);
    const SrcDev &S = a.srcs[sr.w];
    // a re-projected window's gridding baselines are written here (Eq. 1)
    const double *R = S.rot1 ? a.rot + 9 * (int64_t)(S.rot1 - 1) : nullptr;
    double *G = R ? const_cast<double *>(S.guvw) : nullptr;
    if (!so.sorted) {
        for (int64_t r = sr.r0 + threadIdx.x; r < sr.r1; r += blockDim.x) {
            so.slot[sr.g0 + r] = (uint32_t)r;
            so.key[sr.g0 + r] = 0u;
            if (G) rotate_row(R, S.uvw + 3 * r, G + 3 * r);
        }
        if (threadIdx.x == 0 && sr.r0 == 0) so.hist[sr.w] = (uint32_t)S.nrow;
        return;
    }
    for (int k = threadIdx.x; k < so.nstripe; k += blockDim.x) cnt[k] = 0u;
    __syncthreads();
    for (int64_t r = sr.r0 + threadIdx.x; r < sr.r1; r += blockDim.x) {
        uint32_t stripe = 0, L = 0;
        if (S.k_hi > S.k_lo) {
            double u, v;
            if (G) {
                const double2 g = rotate_row(R, S.uvw + 3 * r, G + 3 * r);
                u = g.x;
                v = g.y;
            } else {
                u = S.uvw[3 * r];
                v = S.uvw[3 * r + 1];
            }
            if (a.g.fold && (v < 0.0 || (v == 0.0 && u < 0.0))) {
                u = -u;
                v = -v;
            }
            float x = floorf((float)u * S.key_su) + (float)(a.g.nu >> 1);
            float y = floorf((float)v * S.key_sv) + (float)(a.g.nv >> 1);
            x = fminf(fmaxf(x, 0.0f), (float)(a.g.nu - 1));   // NaN -> 0
            y = fminf(fmaxf(y, 0.0f), (float)(a.g.nv - 1));
            const int iu = (int)x, iv = (int)y;
            stripe = (uint32_t)(iv / so.stripe_rows);
            L = (uint32_t)((iv % so.stripe_rows) * so.nuk + (iu >> so.ushift));
        }
        so.key[sr.g0 + r] = (stripe << 13) | L;
        atomicAdd(&cnt[stripe], 1u);
    }
    __syncthreads();
    for (int k = threadIdx.x; k < so.nstripe; k += blockDim.x) so.segcnt[seg * so.nstripe + k] = cnt[k];
}

// Pass 2: one warp per (window, stripe): the segments' first slots (an
// exclusive scan of the counts over the window's segments, 32 at a time)
// and the bucket's row count.
__global__ void __launch_bounds__(256) k_segscan(RunArgs a)
{
    chain_begin();
    const SortArgs &so = a.so;
    const int64_t t = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int lane = threadIdx.x & 31;
    if (!so.sorted || t >= (int64_t)a.nsrc * so.nstripe) return;   // whole warps
    const int w = (int)(t / so.nstripe), k = (int)(t % so.nstripe);
    const int64_t s1 = so.seg_off[w + 1];
    uint32_t run = 0;
    for (int64_t s0 = so.seg_off[w]; s0 < s1; s0 += 32) {
        const int64_t seg = s0 + lane;
        uint32_t *c = so.segcnt + seg * so.nstripe + k;
        const uint32_t n = seg < s1 ? *c : 0u;
        uint32_t incl = n;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t y = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += y;
        }
        if (seg < s1) *c = run + incl - n;
        run += __shfl_sync(0xffffffffu, incl, 31);
    }
    if (lane == 0) so.hist[t] = run;
}

// Pass 3: each segment's slots in row order.  Warp w of W takes the
// contiguous w-th part of the segment, counts its stripes into its own
// shared-memory row, the counts become offsets (the segment's first slots
// plus the earlier warps' counts), and the warp assigns its rows in order.
// Dynamic shared memory: W x nstripe words.
__global__ void __launch_bounds__(256) k_slots(RunArgs a)
{
    chain_begin();
    extern __shared__ uint32_t dsm[];
    const SortArgs &so = a.so;
    if (!so.sorted) return;
    const int64_t seg = blockIdx.x;
    const SegRange sr = seg_range(a, seg);
    const int ns = so.nstripe;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nwarps = blockDim.x >> 5;
    uint32_t *cnt = dsm + (size_t)warp * ns;
    for (int i = threadIdx.x; i < nwarps * ns; i += blockDim.x) dsm[i] = 0u;
    __syncthreads();
    const int64_t nr = sr.r1 - sr.r0;
    const int64_t p0 = sr.r0 + nr * warp / nwarps, p1 = sr.r0 + nr * (warp + 1) / nwarps;
    for (int64_t c = p0; c < p1; c += 32) {
        const int64_t r = c + lane;
        const uint32_t stripe = r < p1 ? so.key[sr.g0 + r] >> 13 : NO_BUCKET;
        const unsigned peers = __match_any_sync(0xffffffffu, stripe);
        if (stripe != NO_BUCKET && lane == __ffs(peers) - 1) cnt[stripe] += (uint32_t)__popc(peers);
    }
    __syncthreads();
    for (int k = threadIdx.x; k < ns; k += blockDim.x) {
        uint32_t run = so.segcnt[seg * ns + k];
        for (int v = 0; v < nwarps; ++v) {
            const uint32_t c = dsm[(size_t)v * ns + k];
            dsm[(size_t)v * ns + k] = run;
            run += c;
        }
    }
    __syncthreads();
    for (int64_t c = p0; c < p1; c += 32) {
        const int64_t r = c + lane;
        const uint32_t stripe = r < p1 ? so.key[sr.g0 + r] >> 13 : NO_BUCKET;
        const unsigned peers = __match_any_sync(0xffffffffu, stripe);
        const int leader = __ffs(peers) - 1;
        uint32_t b0 = 0;
        if (stripe != NO_BUCKET && lane == leader) {
            b0 = cnt[stripe];
            cnt[stripe] = b0 + (uint32_t)__popc(peers);
        }
        const uint32_t slot = __shfl_sync(0xffffffffu, b0, leader) + (uint32_t)__popc(peers & ((1u << lane) - 1u));
        if (r < p1) so.slot[sr.g0 + r] = slot;
    }
}

// Warps per block for a per-warp table of nk words in shared memory
// (tables + extra tables of nk words kept within 96 KB).
static int table_warps(int nk, int extra)
{
    int nw = (int)(96 * 1024 / (4 * (int64_t)(nk > 0 ? nk : 1))) - extra;
    return nw < 1 ? 1 : (nw > 8 ? 8 : nw);
}

// Launch a kernel that takes dynamic shared memory above the 48 KB default.
template <typename K>
static cudaError_t allow_smem(K kern, size_t smem)
{
    if (smem <= 48 * 1024) return cudaSuccess;
    return cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
}

// The window and stripe of bucket i.
struct Bucket {
    int w, s;
};
__device__ __forceinline__ Bucket bucket_at(const RunArgs &a, int64_t i)
{
    const int ns = a.so.nstripe;
    if (a.so.nclass == 1) return Bucket{(int)((uint32_t)i % (uint32_t)a.nsrc), (int)((uint32_t)i / (uint32_t)a.nsrc)};
    int c = 0;
    while (c + 1 < a.so.nclass && a.so.cls_off[c + 1] * ns <= i) ++c;
    const int w0 = (int)a.so.cls_off[c], nw = (int)a.so.cls_off[c + 1] - w0;
    const uint32_t k = (uint32_t)(i - (int64_t)w0 * ns);   // (a class has fewer than 2^31 buckets)
    return Bucket{w0 + (int)(k % (uint32_t)nw), (int)(k / (uint32_t)nw)};
}

// One block of 1024 threads.
__global__ void __launch_bounds__(1024) k_scan(RunArgs a)
{
    chain_begin();
    const SortArgs &so = a.so;
    const int nw = a.nsrc, ns = so.nstripe, R = so.rows_per_item;
    // a warp per window: its buckets' first positions, 32 stripes at a time
    const int lane = threadIdx.x & 31;
    for (int w = threadIdx.x >> 5; w < nw; w += blockDim.x >> 5) {
        uint32_t run = 0;
        for (int s0 = 0; s0 < ns; s0 += 32) {
            const int s = s0 + lane;
            const uint32_t n = s < ns ? so.hist[(size_t)w * ns + s] : 0u;
            uint32_t incl = n;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const uint32_t y = __shfl_up_sync(0xffffffffu, incl, o);
                if (lane >= o) incl += y;
            }
            if (s < ns) so.qstart[(size_t)w * ns + s] = run + incl - n;
            run += __shfl_sync(0xffffffffu, incl, 31);
        }
    }
    __syncthreads();
    // the work list: four buckets a thread at a time
    const int64_t nb = (int64_t)nw * ns;
    __shared__ long long part[32];
    long long run = 0;
    for (int64_t t0 = 0; t0 < nb; t0 += 4 * blockDim.x) {
        const int64_t i0 = t0 + 4 * threadIdx.x;
        long long cnt[4], mine = 0;
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            cnt[k] = 0;
            if (i0 + k < nb) {
                const Bucket b = bucket_at(a, i0 + k);
                const uint32_t n = so.hist[(size_t)b.w * ns + b.s];
                cnt[k] = (long long)((n + R - 1) / R) * a.srcs[b.w].nchunk;
            }
        }
#pragma unroll
        for (int k = 0; k < 4; ++k) mine += cnt[k];
        long long incl = mine;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const long long y = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += y;
        }
        if (lane == 31) part[threadIdx.x >> 5] = incl;
        __syncthreads();
        long long before = run;
        for (int v = 0; v < 32; ++v) {
            const long long x = part[v];
            if (v < (int)(threadIdx.x >> 5)) before += x;
            run += x;
        }
        __syncthreads();
        long long pos = before + incl - mine;
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            if (i0 + k < nb) so.ioff[i0 + k] = pos;
            pos += cnt[k];
        }
    }
    if (threadIdx.x == 0) {
        so.ioff[nb] = run;
        if (run > so.max_items) atomicExch(a.err, 2);   // host sizing bug: never expected
    }
    __syncthreads();
    for (int c = threadIdx.x; c <= so.nclass; c += blockDim.x)
        so.ctr[c] = (uint32_t)min(so.ioff[so.cls_off[c] * ns], so.max_items);
}

// One thread per work item: bucket i holds items [ioff[i], ioff[i+1]), rows
// in groups of rows_per_item, each group split into the window's channel
// chunks.
__global__ void __launch_bounds__(256) k_items(RunArgs a)
{
    chain_begin();
    const SortArgs &so = a.so;
    const int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const int64_t nb = (int64_t)a.nsrc * so.nstripe;
    if (p >= so.ioff[nb] || p >= so.max_items) return;
    const int i = find_owner_chained(so.ioff, (int)nb, p);
    const int R = so.rows_per_item;
    const Bucket bk = bucket_at(a, i);
    const int st = bk.s, w = bk.w;
    const SrcDev &S = a.srcs[w];
    const uint32_t local = (uint32_t)(p - so.ioff[i]), nchunk = (uint32_t)S.nchunk;   // (a list has fewer than 2^32 items)
    const uint32_t t = local / nchunk;
    const int c = (int)(local - t * nchunk);
    const int64_t n = so.hist[(size_t)w * so.nstripe + st];
    const int64_t q = so.qstart[(size_t)w * so.nstripe + st];
    const int nin = S.k_hi - S.k_lo;
    Item it;
    it.w = w;
    it.chunk = c;
    it.q0 = (int32_t)(q + (int64_t)t * R);
    it.q1 = (int32_t)min(q + n, q + ((int64_t)t + 1) * R);
    it.chf0 = S.chan_off + c * S.cw;
    it.nch = min(S.cw, nin - c * S.cw);
    it.rec0 = S.rec_off + it.q0;
    it.cell0 = S.cell_off + (int64_t)c * S.nrow + it.q0;
    it.pad = 0;
    so.items[p] = it;
}

__global__ void __launch_bounds__(256) k_scatter(RunArgs a)
{
    chain_begin();
    const int64_t g = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (g >= a.nrows_total) return;
    const SortArgs &so = a.so;
    const int w = find_owner(a.row_off, a.nsrc, g);
    const uint32_t r = (uint32_t)(g - a.row_off[w]);
    const uint32_t key = so.key[g];
    const uint32_t s = key >> 13, L = key & 0x1fffu;
    const int64_t q = (int64_t)so.qstart[(size_t)w * so.nstripe + s] + so.slot[g];
    so.tmp[a.row_off[w] + q] = ((unsigned long long)L << 32) | r;
}

// One block per (window, stripe) bucket: a stable counting sort of the
// bucket's rows by local cell key.  The rows arrive in row order (k_slots)
// and keep it within each key, so that rows of one baseline stay
// consecutive in time and, at the window's other channels, a group's cell
// changes at most once instead of alternating.  Warp w of W takes the
// contiguous w-th part of the bucket: it counts its keys into its own
// shared-memory row (no block barrier per 32 rows), the counts become
// offsets (key-major, then warp), and the warp scatters its part in order.
// Dynamic shared memory: (W + 1) x nk words.
__global__ void __launch_bounds__(256) k_bucket_sort(RunArgs a)
{
    chain_begin();
    extern __shared__ uint32_t dsm[];
    __shared__ uint32_t part[256];
    const SortArgs &so = a.so;
    const int64_t b = blockIdx.x;
    const int w = (int)(b / so.nstripe);
    const uint32_t n = so.hist[b];
    if (n == 0) return;
    const int64_t base = a.row_off[w] + so.qstart[b];
    if (!so.sorted || n == 1) {
        for (uint32_t i = threadIdx.x; i < n; i += blockDim.x) so.perm[base + i] = (uint32_t)so.tmp[base + i];
        return;
    }
    const int nk = so.stripe_rows * so.nuk;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nwarps = blockDim.x >> 5;
    uint32_t *cnt = dsm + (size_t)warp * nk;        // this warp's counts, then its offsets
    uint32_t *tot = dsm + (size_t)nwarps * nk;      // per key: all warps' counts, then the key's start
    for (int i = threadIdx.x; i < (nwarps + 1) * nk; i += blockDim.x) dsm[i] = 0u;
    __syncthreads();
    const uint32_t r0 = (uint32_t)((uint64_t)n * warp / nwarps), r1 = (uint32_t)((uint64_t)n * (warp + 1) / nwarps);
    for (uint32_t c0 = r0; c0 < r1; c0 += 32) {
        const uint32_t i = c0 + lane;
        const uint32_t L = i < r1 ? (uint32_t)(so.tmp[base + i] >> 32) : NO_BUCKET;
        const unsigned peers = __match_any_sync(0xffffffffu, L);
        if (L != NO_BUCKET && lane == __ffs(peers) - 1) cnt[L] += (uint32_t)__popc(peers);
    }
    __syncthreads();
    // per key: exclusive prefix over the warps, and the key's total
    for (int k = threadIdx.x; k < nk; k += blockDim.x) {
        uint32_t run = 0;
        for (int v = 0; v < nwarps; ++v) {
            const uint32_t c = dsm[(size_t)v * nk + k];
            dsm[(size_t)v * nk + k] = run;
            run += c;
        }
        tot[k] = run;
    }
    __syncthreads();
    // exclusive scan of the totals over the keys: contiguous slices per thread
    const int per = (nk + blockDim.x - 1) / blockDim.x;
    const int k0 = min(nk, (int)threadIdx.x * per), k1 = min(nk, k0 + per);
    uint32_t loc = 0;
    for (int k = k0; k < k1; ++k) loc += tot[k];
    part[threadIdx.x] = loc;
    __syncthreads();
    for (int off = 1; off < (int)blockDim.x; off <<= 1) {
        const uint32_t v = threadIdx.x >= (unsigned)off ? part[threadIdx.x - off] : 0u;
        __syncthreads();
        part[threadIdx.x] += v;
        __syncthreads();
    }
    uint32_t run = part[threadIdx.x] - loc;
    for (int k = k0; k < k1; ++k) {
        const uint32_t c = tot[k];
        tot[k] = run;
        run += c;
    }
    __syncthreads();
    for (int k = threadIdx.x; k < nk; k += blockDim.x) {
        const uint32_t st = tot[k];
        for (int v = 0; v < nwarps; ++v) dsm[(size_t)v * nk + k] += st;
    }
    __syncthreads();
    // each warp scatters its part in row order
    for (uint32_t c0 = r0; c0 < r1; c0 += 32) {
        const uint32_t i = c0 + lane;
        const bool valid = i < r1;
        const unsigned long long t = valid ? so.tmp[base + i] : 0ull;
        const uint32_t L = valid ? (uint32_t)(t >> 32) : NO_BUCKET;
        const unsigned peers = __match_any_sync(0xffffffffu, L);
        const int leader = __ffs(peers) - 1;
        uint32_t b0 = 0;
        if (valid && lane == leader) {
            b0 = cnt[L];
            cnt[L] = b0 + (uint32_t)__popc(peers);
        }
        const uint32_t pos = __shfl_sync(0xffffffffu, b0, leader) + (uint32_t)__popc(peers & ((1u << lane) - 1u));
        if (valid) so.perm[base + pos] = (uint32_t)t;
    }
}

// The cell scales (su, sv) of channel k of a window's table (read-only).
__device__ __forceinline__ float2 chan_scales(const ChanF *cf, int k)
{
    return __ldg(reinterpret_cast<const float2 *>(cf + k));
}

// The scales of a chunk's first and last channel: all a chunk's entry needs
// unless its cell changes inside it.
struct ChunkEnds {
    float2 s0, s1;
};
__device__ __forceinline__ ChunkEnds chunk_ends(const ChanF *cf, int nin, int cw, int c)
{
    const int e0 = c * cw, last = min(nin, e0 + cw) - 1 - e0;
    return ChunkEnds{chan_scales(cf, e0), chan_scales(cf, e0 + last)};
}

// First chunk-local channel in (lo, hi] whose floor(coord * s) differs from
// f_lo; f_hi = the floor at hi (different), x_lo, x_hi = fl32(coord * s) at
// lo and hi.  The cell is monotone in frequency.  The scales are close to
// linear in the channel index across a chunk, so the crossing is first
// estimated by linear interpolation and the floors at the estimate and the
// channel before it are evaluated (two loads issued together); they either
// settle the answer or narrow the bisection that follows, so the result is
// the exact first differing channel whatever the estimate.
__device__ int axis_step(float c32, const ChanF *cf, const ChanD *cd, int e0, int lo, int hi, const double *coord64,
                         bool neg, bool v_axis, float f_lo, float f_hi, float x_lo, float x_hi)
{
    auto f_at = [&](int k) {
        const float2 sc = chan_scales(cf, e0 + k);
        return axis_floor(c32, v_axis ? sc.y : sc.x, coord64, neg, v_axis ? &cd[e0 + k].sv : &cd[e0 + k].su);
    };
    if (hi - lo > 1) {
        const float B = f_hi > f_lo ? f_lo + 1.0f : f_lo;   // the value coord * s crosses
        const float dx = x_hi - x_lo, span = (float)(hi - lo);
        int k = (lo + hi + 1) >> 1;
        if (dx != 0.0f) {
            const float t = (B - x_lo) / dx * span;
            if (t > 0.0f && t < span) k = lo + (int)ceilf(t);   // a NaN fails both tests
        }
        k = min(max(k, lo + 1), hi);
        const float fk = f_at(k), fm = f_at(k - 1);   // k - 1 >= lo, where the floor is f_lo
        if (fk == f_lo)
            lo = k;
        else if (fm == f_lo)
            return k;
        else
            hi = k - 1;
    }
    while (hi - lo > 1) {
        const int mid = (lo + hi) >> 1;
        if (f_at(mid) == f_lo)
            lo = mid;
        else
            hi = mid;
    }
    return hi;
}

// The chunk-cell entry of chunk c of one row (coordinates uf, vf after the
// fold; uvw the row's FP64 coordinates for the exact fall-backs; ce the
// scales at the chunk's two end channels).  The cell index is monotone in
// frequency along each axis, so the cells at a chunk's two end channels
// bound every channel between.
__device__ int2 chunk_cell(const RunArgs &a, const ChanF *cf, const ChanD *cd, int nin, int cw, int c, float uf, float vf,
                           const double *uvw, bool fold, const ChunkEnds &ce)
{
    const float hu = (float)(a.g.nu >> 1), hv = (float)(a.g.nv >> 1);
    const int e0 = c * cw, last = min(nin, e0 + cw) - 1 - e0;
    const float fu0 = axis_floor(uf, ce.s0.x, uvw, fold, &cd[e0].su);
    const float fu1 = axis_floor(uf, ce.s1.x, uvw, fold, &cd[e0 + last].su);
    const float fv0 = axis_floor(vf, ce.s0.y, uvw + 1, fold, &cd[e0].sv);
    const float fv1 = axis_floor(vf, ce.s1.y, uvw + 1, fold, &cd[e0 + last].sv);
    // both ends off the grid on the same side of one axis: off throughout
    const bool offu = (fu0 < -hu && fu1 < -hu) || (fu0 >= hu && fu1 >= hu);
    const bool offv = (fv0 < -hv && fv1 < -hv) || (fv0 >= hv && fv1 >= hv);
    const bool in = fu0 >= -hu && fu0 < hu && fu1 >= -hu && fu1 < hu && fv0 >= -hv && fv0 < hv &&
                    fv1 >= -hv && fv1 < hv;
    if (offu || offv) return make_int2(-1, CC_NOCHANGE);
    if (!in || fabsf(fu1 - fu0) > 1.0f || fabsf(fv1 - fv0) > 1.0f) return make_int2(-1, CC_MIXED);
    uint32_t m = CC_NOCHANGE;
    if (fu1 != fu0) {
        const int b = axis_step(uf, cf, cd, e0, 0, last, uvw, fold, false, fu0, fu1, __fmul_rn(uf, ce.s0.x),
                                __fmul_rn(uf, ce.s1.x));
        m = (m & ~0xffu) | (uint32_t)b | (fu1 < fu0 ? 0x10000u : 0u);
    }
    if (fv1 != fv0) {
        const int b = axis_step(vf, cf, cd, e0, 0, last, uvw + 1, fold, true, fv0, fv1, __fmul_rn(vf, ce.s0.y),
                                __fmul_rn(vf, ce.s1.y));
        m = (m & ~0xff00u) | ((uint32_t)b << 8) | (fv1 < fv0 ? 0x20000u : 0u);
    }
    return make_int2(((int)fv0 + (a.g.nv >> 1)) * a.g.nu + ((int)fu0 + (a.g.nu >> 1)), (int)m);
}

// Rows of one cell by the part of the cell they lie in.  The cell rows are
// sorted by is that of one channel; at another channel the cell borders run
// through that cell, and rows that alternate between its parts end a run each
// time.  In row order they alternate or not as the data have it (the tracks
// of baselines that share a cell cross a border together when they are sampled
// densely, and then row order is the better one), so the lanes of a warp, 32
// rows in processing order, decide on what they see: with T changes of part
// from row to row inside the cells and G the fewest the parts present allow,
// the rows of each cell are put in the order of the parts if T > 2 G.  Parts
// are columns of a third of a cell, walked up and down in turn in two halves
// (so that neighbouring parts, also of the next cell, follow each other).
// Finished runs, with the key at the middle channel: compact array 4.49 -> 4.30
// per 32 rows x channels, wideband 5.49 -> 2.96, long baselines 3.58 -> 3.55,
// archive 2.34 -> 2.28, ragged 3.98 -> 3.56.  Kernel times with this and the
// middle channel's key, against the highest frequency's: compact array 1.675
// -> 1.605 ms, wideband 2.24 -> 1.90, long baselines 1.178 -> 1.141, archive
// 23.7 -> 23.2, ragged 0.157 -> 0.128; k_rows itself is within 2 %.
//
// Returns the row's place among the warp's rows (a permutation of the lanes
// `act`, 0 ... n - 1; only rows of one window and one cell change places).
__device__ __forceinline__ int part_order(unsigned act, int w, float x, float y)
{
    const int lane = threadIdx.x & 31;
    const unsigned below = (1u << lane) - 1u;
    const float cx = floorf(x), cy = floorf(y);
    const int col = min(max((int)((x - cx) * 3.0f), 0), 2), half = y - cy >= 0.5f ? 1 : 0;   // (NaN: 0)
    const int part = 2 * col + (half ^ (((int)cx + col) & 1));
    const int pw = __shfl_up_sync(act, w, 1), pp = __shfl_up_sync(act, part, 1);
    const float px = __shfl_up_sync(act, cx, 1), py = __shfl_up_sync(act, cy, 1);
    const bool head = lane == 0 || pw != w || px != cx || py != cy;
    const unsigned heads = __ballot_sync(act, head);
    const int T = __popc(__ballot_sync(act, !head && pp != part));
    if (T < 3) return lane;   // (G >= 1 if T >= 1)
    const int first = 31 - __clz(heads & (below | 1u << lane));
    const unsigned later = heads & ~(below | 1u << lane);
    unsigned same = act & ~((1u << first) - 1u) & (later ? (later & (0u - later)) - 1u : 0xffffffffu), less = 0u;
#pragma unroll
    for (int b = 4; b > 0; b >>= 1) {
        const unsigned set = __ballot_sync(act, (part & b) != 0);
        if (part & b) less |= same & ~set;
        same &= part & b ? set : ~set;
    }
    const int G = __popc(__ballot_sync(act, (same & below) == 0u)) - __popc(heads);
    return T > 2 * G ? first + __popc(less) + __popc(same & below) : lane;
}

// One thread per row, in processing order: the row record (the FP64 delay
// of Eq. 2 as a float-float pair, the weights, the row index)
// and the chunk-cell entries of all the window's chunks, laid out
// [chunk][row] per window so that an item's entries are contiguous.  The
// row's coordinates are read once for both.  The window's channel table is
// read from L2 (the tables of the windows a block's rows span do not stay
// in L1), so the end scales of chunk c + 1 are loaded before chunk c's entry
// is formed: one load latency per chunk overlaps the previous chunk's work.
__global__ void __launch_bounds__(256) k_rows(RunArgs a)
{
    chain_begin();
    const int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const unsigned act = __ballot_sync(0xffffffffu, p < a.nrows_total);
    if (p >= a.nrows_total) return;
    const int w = find_owner(a.row_off, a.nsrc, p);
    const SrcDev &S = a.srcs[w];
    const int64_t r = a.so.perm[p];
    const double *uvw = S.uvw + 3 * r;     // the stored baseline: the delay of Eq. 2
    const double *guvw = S.guvw + 3 * r;   // the gridding baseline (rotated for a re-projected window)
    const double tau = uvw[0] * S.l + uvw[1] * S.m + uvw[2] * S.n1;
    const double u = guvw[0], v = guvw[1];
    const bool fold = a.g.fold && (v < 0.0 || (v == 0.0 && u < 0.0));
    const float uf = (float)(fold ? -u : u), vf = (float)(fold ? -v : v);
    int64_t q = p - a.row_off[w];
    if (a.so.sorted) {
        const int lane = threadIdx.x & 31, place = part_order(act, w, __fmul_rn(uf, S.key_su), __fmul_rn(vf, S.key_sv));
        q += place - lane;
        if (place != lane) a.so.perm[p + place - lane] = (uint32_t)r;   // (every lane has its row)
    }
    RowRec rec;
    split_ff(fold ? -tau : tau, rec.tau_hi, rec.tau_lo);
    rec.row = (uint32_t)r;
    rec.fold = fold ? 0x80000000u : 0u;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        const int p = S.npol == 4 ? k : k >> 1;
        rec.W[k] = p < S.npol ? S.wts[r * S.npol + p] : 0.0f;
    }
    a.recs[S.rec_off + q] = rec;

    const ChanD *cd = a.chd + S.chan_off;
    const ChanF *cf = a.chf + S.chan_off;
    int2 *out = a.ccells + S.cell_off + q;
    const int nchunk = S.nchunk, nin = S.k_hi - S.k_lo, cw = S.cw;
    const int64_t nrow = S.nrow;
    if (nchunk <= 0) return;
    ChunkEnds nx = chunk_ends(cf, nin, cw, 0);
    for (int c = 0; c < nchunk; ++c) {
        const ChunkEnds ce = nx;
        if (c + 1 < nchunk) nx = chunk_ends(cf, nin, cw, c + 1);
        out[c * nrow] = chunk_cell(a, cf, cd, nin, cw, c, uf, vf, guvw, fold, ce);
    }
}

cudaError_t launch_prepare(const RunArgs &a, cudaStream_t st, int *nlaunch)
{
    const SortArgs &so = a.so;
    if (nlaunch) *nlaunch = 0;
    if (so.nseg_total == 0 || a.nrows_total == 0) return cudaErrorInvalidValue;   // (a class has rows)
    const unsigned rb = (unsigned)((a.nrows_total + 255) / 256);
    const int64_t nb = (int64_t)a.nsrc * so.nstripe;
    const int nws = table_warps(so.nstripe, 0);
    const size_t smem_s = (size_t)nws * so.nstripe * sizeof(uint32_t);
    const int nk = so.stripe_rows * so.nuk, nwb = table_warps(nk, 1);
    const size_t smem_b = (size_t)(nwb + 1) * nk * sizeof(uint32_t);
    cudaError_t e = allow_smem(k_slots, smem_s);
    if (e == cudaSuccess) e = allow_smem(k_bucket_sort, smem_b);
    if (e != cudaSuccess) return e;
    int n = 0;
    k_keys<<<(unsigned)so.nseg_total, 256, 0, st>>>(a);
    e = cudaGetLastError();
    auto next = [&](void (*kern)(RunArgs), int64_t grid, unsigned block, size_t smem) {
        if (e != cudaSuccess) return;
        e = launch_chained(kern, (unsigned)grid, block, smem, st, a);
        ++n;
    };
    ++n;
    next(k_segscan, (nb * 32 + 255) / 256, 256, 0);
    next(k_slots, so.nseg_total, 32 * (unsigned)nws, smem_s);
    next(k_scan, 1, 1024, 0);
    next(k_items, (so.max_items + 255) / 256, 256, 0);
    next(k_scatter, rb, 256, 0);
    next(k_bucket_sort, nb, 32 * (unsigned)nwb, smem_b);
    next(k_rows, rb, 256, 0);
    if (nlaunch) *nlaunch = n;
    return e;
}

}  // namespace vista
