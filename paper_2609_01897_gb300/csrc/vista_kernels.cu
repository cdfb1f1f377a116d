// libvista kernels over the cube, for sm_103a.
//
//   (the stacking kernels are in vista_stack.cuh and vista_fp64.cu)
//   debug_mixed   the mixed form's phasors and cells, exported
//   unpack        cube -> caller arrays
//   zero          the touched entries back to zero
//   sparse_*      the touched entries -> caller arrays
//   fold          FP32 partials -> FP64 master
#include "vista_cube.cuh"
#include "vista_device.cuh"

namespace vista {

// Debug export: the same phasor and cell code as stack_mixed, writing the
// phasor and the cell of every (row, channel) of one window.
template <int NS>
__global__ void debug_mixed(RunArgs a, int src, double *ph_out, int32_t *cell_out)
{
    const int lane = threadIdx.x & 31;
    const SrcDev &S = a.srcs[src];
    const int64_t nrow = S.nrow;
    const int64_t task = (int64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
    if (task >= nrow * S.nchunk) return;
    const int chunk = (int)(task / nrow);
    const int64_t i = task % nrow;
    const int c0 = S.k_lo + chunk * 32 * NS;
    const RowRec rec = a.recs[S.rec_off + i];
    const int2 cc = a.ccells[S.cell_off + (int64_t)chunk * nrow + i];
    const int64_t row = rec.row;
    const bool fold = rec.fold != 0u;
#pragma unroll
    for (int q = 0; q < NS; ++q) {
        const int kk = q * 32 + lane, k = c0 + kk;
        if (k < S.k_hi) {
            const ChanD *cd = a.chd + S.chan_off + (k - S.k_lo);
            const ChanF cf = a.chf[S.chan_off + (k - S.k_lo)];
            float2 ph = shift_phasor(rec.tau_hi, rec.tau_lo, cf.nuc_hi, cf.nuc_lo);
            if (fold) ph.y = -ph.y;   // the record's delay is negated
            // same cell path as the stacking kernel
            int cid;
            if (cc.y == CC_NOCHANGE)
                cid = cc.x;
            else if (cc.y != CC_MIXED)
                cid = chunk_cell_step(cc, kk, a.g.nu);
            else
                cid = cell_exact(S.guvw, row, fold, cd, a.g.nu, a.g.nv);
            const int iu = cid < 0 ? -1 : cid % a.g.nu, iv = cid < 0 ? -1 : cid / a.g.nu;
            const int64_t o = row * S.nchan + k;
            if (ph_out) {
                ph_out[2 * o] = (double)ph.x;
                ph_out[2 * o + 1] = (double)ph.y;
            }
            if (cell_out) {
                const bool ok = iu >= 0 && iv >= 0;
                cell_out[2 * o] = ok ? iu : -1;
                cell_out[2 * o + 1] = ok ? iv : -1;
            }
        }
    }
}

// ------------------------------------------------------------------ unpack

// Entry i's four sums (re and im of sum wV, sum w, sum w|V|^2): the FP64
// cube, or the mixed cube's float4 sums since the last checkpoint plus its
// FP64 master sums, as doubles or rounded to floats.
template <bool FP64>
struct RawEntry {
    float4 f;
    Double4 d;
    bool has_master;
    __device__ __forceinline__ void load(const void *cube, const double *master, bool has, int64_t i)
    {
        if constexpr (FP64) {
            d = load_double4(reinterpret_cast<const double *>(cube) + 4 * i);
        } else {
            f = reinterpret_cast<const float4 *>(cube)[i];
            has_master = has;
            if (has) d = load_double4(master + 4 * i);
        }
    }
    __device__ __forceinline__ void value(float (&e)[4]) const
    {
        if constexpr (FP64) {
            e[0] = narrow(d.x);
            e[1] = narrow(d.y);
            e[2] = narrow(d.z);
            e[3] = narrow(d.w);
        } else {
            const float4 q = has_master ? sum_f32(f, d) : f;
            e[0] = q.x;
            e[1] = q.y;
            e[2] = q.z;
            e[3] = q.w;
        }
    }
    __device__ __forceinline__ void value(double (&e)[4]) const
    {
        if constexpr (FP64) {
            e[0] = d.x;
            e[1] = d.y;
            e[2] = d.z;
            e[3] = d.w;
        } else {
            const Double4 m = has_master ? d : Double4{0.0, 0.0, 0.0, 0.0};
            e[0] = widen_exact(f.x) + m.x;
            e[1] = widen_exact(f.y) + m.y;
            e[2] = widen_exact(f.z) + m.z;
            e[3] = widen_exact(f.w) + m.w;
        }
    }
};

// The cube -> caller arrays.  An entry whose count is 0 has had no
// contribution, so only its count is read and zeros are written: 24 bytes an
// entry instead of 72 (mixed, FP32 sums), which is what bounds a cube that is
// touched in part, as cubes are (uv corners, gaps between tracks, rest bins
// outside the windows).  `all` reads every entry's sums (counts that may have
// wrapped, see cube_counts_exact()).  A thread takes CUBE_UNROLL entries a
// block apart, so that every access of a warp is contiguous and the counts of
// all of them are in flight together.  Before (every entry read, widened,
// added and narrowed on the FP64 pipe, which bound it) and now: 6.7e7 entries,
// 31 % touched, 1478 -> 403 us (468 with the masters that are zero read too);
// 2.7e8 entries, 2.6 % touched, 5902 -> 1392 us; 4.2e6 entries, 10 % touched, 96
// -> 23 us.  It is at the rate of its writes: streaming stores, 16-byte stores of
// four entries a thread and eight entries a thread were level or slower.  Sums
// are read only where some array of sums is asked for.  The FP64 cube has a form
// of its own: without the float sums and the moved bits it needs 64 registers
// instead of 80, and the next tile's counts are loaded under this tile's sums, which
// a call for one array, with few writes to wait for, would otherwise wait for (1.7e7
// entries of four planes, sum_w alone 138 -> 72 us, the counts alone 138 -> 29;
// all arrays 146 -> 110).  On the mixed cube the early counts cost registers
// (1392 -> 1747 us on the 2.7e8 entries).
constexpr int CUBE_THREADS = 256, CUBE_UNROLL = 4, CUBE_TILE = CUBE_THREADS * CUBE_UNROLL;
constexpr int ZERO_UNROLL = 8, ZERO_TILE = CUBE_THREADS * ZERO_UNROLL;

// The words of moved bits of a warp's entries b, b + CUBE_THREADS, ...: lane q
// loads that of the q-th 32 entries, to be passed round by shuffles.
__device__ __forceinline__ int64_t moved_at(int64_t b)
{
    const int lane = threadIdx.x & 31;
    return (b - lane + (int64_t)lane * CUBE_THREADS) >> 5;
}
template <int N>
__device__ __forceinline__ uint32_t moved_word(const uint32_t *moved, int64_t b, int64_t n)
{
    const int64_t w = moved_at(b);
    return moved && (threadIdx.x & 31) < N && 32 * w < n ? moved[w] : 0u;
}

template <typename T, bool FP64>
__global__ void __launch_bounds__(CUBE_THREADS, FP64 ? 4 : 3) unpack_kernel(const void *cube, const double *master,
                                                                            const uint32_t *moved, const uint32_t *count,
                                                                            int all, int pair, int64_t n, T *sum_wv,
                                                                            T *sum_w, T *sum_wvv, uint32_t *cnt_out)
{
    struct alignas(2 * sizeof(T)) Pair {
        T re, im;
    };
    const bool sums = sum_wv || sum_w || sum_wvv;   // (the counts alone: no entry is read)
    const int64_t step = (int64_t)gridDim.x * CUBE_TILE;
    uint32_t next[CUBE_UNROLL];
    auto load_counts = [&](int64_t b, uint32_t (&c)[CUBE_UNROLL]) {
#pragma unroll
        for (int q = 0; q < CUBE_UNROLL; ++q) {
            const int64_t i = b + q * CUBE_THREADS;
            c[q] = i < n ? count[i] : 0u;
        }
    };
    if constexpr (FP64) load_counts((int64_t)blockIdx.x * CUBE_TILE + threadIdx.x, next);
    for (int64_t b0 = (int64_t)blockIdx.x * CUBE_TILE; b0 < n; b0 += step) {
        const int64_t b = b0 + threadIdx.x;
        uint32_t c[CUBE_UNROLL], word = 0u;
        RawEntry<FP64> r[CUBE_UNROLL];
        if constexpr (FP64) {
#pragma unroll
            for (int q = 0; q < CUBE_UNROLL; ++q) c[q] = next[q];
            if (b0 + step < n) load_counts(b + step, next);
        } else {
            load_counts(b, c);
            if (sums) word = moved_word<CUBE_UNROLL>(moved, b, n);
        }
#pragma unroll
        for (int q = 0; q < CUBE_UNROLL; ++q) {
            const int64_t i = b + q * CUBE_THREADS;
            const uint32_t mv = FP64 ? 0u : __shfl_sync(0xffffffffu, word, q);
            if (sums && i < n && (all || c[q] != 0u)) r[q].load(cube, master, is_moved(mv, i), i);
        }
#pragma unroll
        for (int q = 0; q < CUBE_UNROLL; ++q) {
            const int64_t i = b + q * CUBE_THREADS;
            if (i >= n) break;
            T e[4] = {0, 0, 0, 0};
            if (sums && (all || c[q] != 0u)) r[q].value(e);
            if (sum_wv && pair) {
                reinterpret_cast<Pair *>(sum_wv)[i] = Pair{e[0], e[1]};
            } else if (sum_wv) {
                sum_wv[2 * i] = e[0];
                sum_wv[2 * i + 1] = e[1];
            }
            if (sum_w) sum_w[i] = e[2];
            if (sum_wvv) sum_wvv[i] = e[3];
            if (cnt_out) cnt_out[i] = c[q];
        }
    }
}

// Zeroes the entries whose count is not 0 (every other entry is zero
// already), and the counters: the counts are read, 20 bytes of a touched entry
// are written (mixed), and its master's 32 where its moved bit is set.  Against
// setting the whole cube to zero at the HBM peak: 6.7e7 entries, 31 % touched,
// 518 -> 221 -> 146 us (with every touched entry's master, with the moved ones
// only); 1.3e8 entries, 15 % touched, 1029 -> 268 -> 189 us; 2.7e8 entries, 2.6 %
// touched, 2053 -> 245 -> 237 us (eight entries a thread: the counts' latency;
// four 300).  A cube touched and moved throughout would cost 4 bytes in 52 more.
__global__ void __launch_bounds__(CUBE_THREADS) zero_kernel(void *cube, double *master, uint32_t *moved, uint32_t *count,
                                                            DevStats *stats, int fp64, int64_t n)
{
    if (blockIdx.x == 0 && threadIdx.x == 0) *stats = DevStats{};
    for (int64_t b0 = (int64_t)blockIdx.x * ZERO_TILE; b0 < n; b0 += (int64_t)gridDim.x * ZERO_TILE) {
        const int64_t b = b0 + threadIdx.x;
        uint32_t c[ZERO_UNROLL];
#pragma unroll
        for (int q = 0; q < ZERO_UNROLL; ++q) {
            const int64_t i = b + q * CUBE_THREADS;
            c[q] = i < n ? count[i] : 0u;
        }
        const uint32_t word = moved_word<ZERO_UNROLL>(moved, b, n);
        if (word != 0u) moved[moved_at(b)] = 0u;   // (its own lane's)
#pragma unroll
        for (int q = 0; q < ZERO_UNROLL; ++q) {
            const int64_t i = b + q * CUBE_THREADS;
            const uint32_t mv = __shfl_sync(0xffffffffu, word, q);
            if (c[q] == 0u) continue;
            if (fp64)
                store_zero32(reinterpret_cast<double *>(cube) + 4 * i);
            else
                reinterpret_cast<float4 *>(cube)[i] = make_float4(0.f, 0.f, 0.f, 0.f);
            if (is_moved(mv, i)) store_zero32(master + 4 * i);
            count[i] = 0u;
        }
    }
}

// Sparse readback: the entries with count > 0, in entry order, in three
// passes over tiles of SPARSE_TILE consecutive entries (thread t of a block
// reads entries t, t + 256, ... of its tile, so every load is coalesced):
// the touched entries of each tile; one block's exclusive scan of the tile
// counts, with the total at the end; and each tile's touched entries
// written from its offset on, in entry order (a ballot per warp and a count
// per warp in shared memory per round of 256 entries).
constexpr int SPARSE_THREADS = 256, SPARSE_ROUNDS = 16, SPARSE_TILE = SPARSE_THREADS * SPARSE_ROUNDS;
constexpr int SPARSE_WARPS = SPARSE_THREADS / 32, SCAN_THREADS = 1024;
static_assert(SPARSE_TILE == 4096, "sparse_tiles() counts tiles of 4096 entries");

__global__ void __launch_bounds__(SPARSE_THREADS) sparse_count_kernel(const uint32_t *count, int64_t n,
                                                                      uint32_t *tile_cnt)
{
    __shared__ int ws[SPARSE_WARPS];
    const int64_t base = (int64_t)blockIdx.x * SPARSE_TILE;
    int c = 0;
    for (int k = 0; k < SPARSE_ROUNDS; ++k) {
        const int64_t i = base + (int64_t)k * SPARSE_THREADS + threadIdx.x;
        c += (i < n && count[i] != 0u) ? 1 : 0;
    }
    c = __reduce_add_sync(0xffffffffu, c);
    if ((threadIdx.x & 31) == 0) ws[threadIdx.x >> 5] = c;
    __syncthreads();
    if (threadIdx.x == 0) {
        int t = 0;
        for (int w = 0; w < SPARSE_WARPS; ++w) t += ws[w];
        tile_cnt[blockIdx.x] = (uint32_t)t;
    }
}

// One block of SCAN_THREADS: thread t sums a contiguous run of tiles, the
// block scans those sums (warp shuffles, then the warps' totals), and each
// thread writes its tiles' offsets; the last thread writes the total.
__global__ void __launch_bounds__(SCAN_THREADS) sparse_scan_kernel(const uint32_t *tile_cnt, int64_t ntile,
                                                                   int64_t *tile_off, int64_t *total)
{
    __shared__ long long wtot[SCAN_THREADS / 32];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const int64_t per = (ntile + SCAN_THREADS - 1) / SCAN_THREADS;
    const int64_t t0 = min((int64_t)threadIdx.x * per, ntile), t1 = min(t0 + per, ntile);
    long long s = 0;
    for (int64_t t = t0; t < t1; ++t) s += tile_cnt[t];
    long long x = s;   // inclusive scan over the warp
    for (int o = 1; o < 32; o <<= 1) {
        const long long y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y;
    }
    if (lane == 31) wtot[wid] = x;
    __syncthreads();
    long long before = 0;
    for (int w = 0; w < wid; ++w) before += wtot[w];
    long long off = before + x - s;   // exclusive
    for (int64_t t = t0; t < t1; ++t) {
        tile_off[t] = off;
        off += tile_cnt[t];
    }
    if (threadIdx.x == SCAN_THREADS - 1) *total = before + x;
}

__global__ void __launch_bounds__(SPARSE_THREADS) sparse_write_kernel(const void *cube, const double *master,
                                                                      const uint32_t *moved, const uint32_t *count,
                                                                      int fp64, int64_t n,
                                                                      const int64_t *tile_off, int64_t cap,
                                                                      int64_t *idx_out, float *sum_wv, float *sum_w,
                                                                      float *sum_wvv, uint32_t *cnt_out)
{
    __shared__ int ws[SPARSE_WARPS];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const int64_t base = (int64_t)blockIdx.x * SPARSE_TILE;
    const bool sums = sum_wv || sum_w || sum_wvv;
    int64_t pos = tile_off[blockIdx.x];
    for (int k = 0; k < SPARSE_ROUNDS; ++k) {
        const int64_t i = base + (int64_t)k * SPARSE_THREADS + threadIdx.x;
        const uint32_t c = i < n ? count[i] : 0u;
        const unsigned bal = __ballot_sync(0xffffffffu, c != 0u);
        if (lane == 0) ws[wid] = __popc(bal);
        __syncthreads();
        int before = 0, all = 0;
        for (int w = 0; w < SPARSE_WARPS; ++w) {
            before += w < wid ? ws[w] : 0;
            all += ws[w];
        }
        if (c != 0u) {
            const int64_t q = pos + before + __popc(bal & ((1u << lane) - 1u));
            if (q < cap) {
                float e[4] = {0.f, 0.f, 0.f, 0.f};
                if (!sums) {   // (the index and the count alone)
                } else if (fp64) {
                    RawEntry<true> r;
                    r.load(cube, nullptr, false, i);
                    r.value(e);
                } else {
                    RawEntry<false> r;
                    r.load(cube, master, moved && is_moved(moved[i >> 5], i), i);
                    r.value(e);
                }
                idx_out[q] = i;
                if (sum_wv) {
                    sum_wv[2 * q] = e[0];
                    sum_wv[2 * q + 1] = e[1];
                }
                if (sum_w) sum_w[q] = e[2];
                if (sum_wvv) sum_wvv[q] = e[3];
                if (cnt_out) cnt_out[q] = c;
            }
        }
        pos += all;
        __syncthreads();   // ws is written again in the next round
    }
}

// --------------------------------------------------------------- launchers

// ------------------------------------------------------------------ fold

// Every nonzero FP32 entry of the mixed cube is added to its FP64 master
// entry and cleared (the exact widening of each component), so the FP32
// partials start again from zero.  Nothing else touches the cube meanwhile
// (the handle's stream orders it after the run's stacking).
__global__ void fold_kernel(float4 *cube, double *master, uint32_t *moved, int64_t n)
{
    const int64_t tid = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    for (int64_t b = tid & ~(int64_t)31; b < n; b += (int64_t)gridDim.x * blockDim.x) {   // 32 entries, a word, a warp
        const int64_t i = b + (tid & 31);
        const float4 c = i < n ? cube[i] : make_float4(0.f, 0.f, 0.f, 0.f);
        const bool nonzero = c.x != 0.f || c.y != 0.f || c.z != 0.f || c.w != 0.f;
        const unsigned bits = __ballot_sync(0xffffffffu, nonzero);
        if (bits != 0u && (tid & 31) == 0) moved[b >> 5] |= bits;
        if (nonzero) {
            double *m = master + 4 * i;
            m[0] += (double)c.x;
            m[1] += (double)c.y;
            m[2] += (double)c.z;
            m[3] += (double)c.w;
            cube[i] = make_float4(0.f, 0.f, 0.f, 0.f);
        }
    }
}

cudaError_t launch_fold(void *cube, double *master, uint32_t *moved, int64_t n, cudaStream_t st)
{
    if (n == 0) return cudaSuccess;
    int64_t blocks = (n + 255) / 256;
    if (blocks > 152 * 16) blocks = 152 * 16;
    fold_kernel<<<(unsigned)blocks, 256, 0, st>>>(reinterpret_cast<float4 *>(cube), master, moved, n);
    return cudaGetLastError();
}

static unsigned cube_blocks(int64_t n, int tile = CUBE_TILE)
{
    const int64_t tiles = (n + tile - 1) / tile;
    return (unsigned)(tiles < 152 * 16 ? tiles : 152 * 16);
}

cudaError_t launch_unpack(const void *cube, const double *master, const uint32_t *moved, const uint32_t *count, int fp64,
                          int all, int64_t n, void *sum_wv, void *sum_w, void *sum_wvv, uint32_t *cnt_out, int out_f64, cudaStream_t st)
{
    if (n == 0) return cudaSuccess;
    // one store per (re, im) pair, or one per value when sum_wv starts off a pair's boundary
    const int pair = ((uintptr_t)sum_wv % (out_f64 ? 16 : 8)) == 0;
    auto launch = [&](auto *kern, auto *wv, auto *w, auto *wvv) {
        kern<<<cube_blocks(n), CUBE_THREADS, 0, st>>>(cube, master, moved, count, all, pair, n, wv, w, wvv, cnt_out);
    };
    if (out_f64)
        launch(fp64 ? unpack_kernel<double, true> : unpack_kernel<double, false>, (double *)sum_wv, (double *)sum_w,
               (double *)sum_wvv);
    else
        launch(fp64 ? unpack_kernel<float, true> : unpack_kernel<float, false>, (float *)sum_wv, (float *)sum_w,
               (float *)sum_wvv);
    return cudaGetLastError();
}

cudaError_t launch_zero_touched(void *cube, double *master, uint32_t *moved, uint32_t *count, DevStats *stats, int fp64,
                                int64_t n, cudaStream_t st)
{
    if (n == 0) return cudaSuccess;
    zero_kernel<<<cube_blocks(n, ZERO_TILE), CUBE_THREADS, 0, st>>>(cube, master, moved, count, stats, fp64, n);
    return cudaGetLastError();
}

cudaError_t launch_sparse_count(const uint32_t *count, int64_t n, uint32_t *tile_cnt, int64_t *tile_off,
                                int64_t *total, cudaStream_t st)
{
    const int64_t ntile = sparse_tiles(n);
    if (ntile == 0) return cudaMemsetAsync(total, 0, sizeof(int64_t), st);
    sparse_count_kernel<<<(unsigned)ntile, SPARSE_THREADS, 0, st>>>(count, n, tile_cnt);
    sparse_scan_kernel<<<1, SCAN_THREADS, 0, st>>>(tile_cnt, ntile, tile_off, total);
    return cudaGetLastError();
}

cudaError_t launch_sparse_write(const void *cube, const double *master, const uint32_t *moved, const uint32_t *count,
                                int fp64, int64_t n,
                                const int64_t *tile_off, int64_t cap, int64_t *index, float *sum_wv, float *sum_w,
                                float *sum_wvv, uint32_t *cnt_out, cudaStream_t st)
{
    const int64_t ntile = sparse_tiles(n);
    if (ntile == 0 || cap == 0) return cudaSuccess;
    sparse_write_kernel<<<(unsigned)ntile, SPARSE_THREADS, 0, st>>>(cube, master, moved, count, fp64, n, tile_off, cap, index,
                                                                   sum_wv, sum_w, sum_wvv, cnt_out);
    return cudaGetLastError();
}

cudaError_t launch_debug(const RunArgs &a, int ns, int src, int fp64, double *ph, int32_t *cells, cudaStream_t st)
{
    SrcDev S;
    cudaError_t e = cudaMemcpyAsync(&S, a.srcs + src, sizeof(S), cudaMemcpyDeviceToHost, st);
    if (e != cudaSuccess) return e;
    e = cudaStreamSynchronize(st);
    if (e != cudaSuccess) return e;
    if (fp64) return launch_debug_fp64(a, src, S.nrow, ph, cells, st);
    const int64_t tasks = S.nrow * S.nchunk;
    if (tasks == 0) return cudaSuccess;
    const int64_t blocks = (tasks + 3) / 4;
    switch (ns) {
    case 1: debug_mixed<1><<<(unsigned)blocks, 128, 0, st>>>(a, src, ph, cells); break;
    case 2: debug_mixed<2><<<(unsigned)blocks, 128, 0, st>>>(a, src, ph, cells); break;
    case 4: debug_mixed<4><<<(unsigned)blocks, 128, 0, st>>>(a, src, ph, cells); break;
    default: return cudaErrorInvalidValue;
    }
    return cudaGetLastError();
}

}  // namespace vista
