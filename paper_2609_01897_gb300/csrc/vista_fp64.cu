// The FP64 form of the stacking kernel (VISTA_PREC_FP64): FP64 phasors,
// products, sums and an FP64 cube.
//
// GB300's FP64 pipe (about two lanes a clock and SM) bounds it, then the L2's
// rate of reductions, so it spends few FP64 operations per visibility and
// writes runs, not visibilities.  The mixed path's pre-pass orders the rows by
// uv cell and gives each (row, 32-channel chunk) its exact cells; a warp takes
// an item of that work list (rows of one window x one chunk) 32 rows at a time:
//   1. lane = row: the row's delay from its baseline, the phasor of the
//      chunk's first channel and of one channel step (sincospi), and the
//      chunk's phasors by recurrence (four operations each; re-seeded at every
//      chunk, so its error does not grow along the window; axes that are not
//      linear take a sincospi per channel), into shared memory;
//   2. lane = channel: the rows one by one, running sums in registers over
//      consecutive rows that share a uv cell (nine operations a visibility),
//      added to the cube when the cell changes.
// FP32 inputs are widened by moving their fields (integer instructions).
//
// Before (a thread per row, every visibility's bins written by FP64 atomics)
// and now, kernel time: 1.7e7 visibilities of two pols in complex128, 1254 ->
// 590 us (and about 80 us of pre-pass it did without); 3.5e7 of four pols, 3732
// -> 1023 us and 8.7e6 of one pol, 739 -> 378 us, both before the rows of a cell
// were ordered by parts (653 us then for two pols).  The FP64 pipe is 81 % busy.
#include "vista_device.cuh"

namespace vista {
namespace {

constexpr int NO_RUN64 = INT32_MIN;   // lane holds no run
constexpr int WARPS64 = 4;            // warps per block

// A float as a double, exactly.
__device__ __forceinline__ double widen_exact(float x)
{
    const uint32_t b = __float_as_uint(x), e = (b >> 23) & 0xffu;
    if (e - 1u >= 254u) return (double)x;   // zero, subnormal, infinite or NaN
    return __hiloint2double((int)((b & 0x80000000u) | ((e + 896u) << 20) | ((b & 0x7fffffu) >> 3)), (int)(b << 29));
}

// One lane's P stored values of one (row, channel), as loaded.
template <int P, int VT>
struct Raw64 {
    static constexpr int kBytes = P * VisType<VT>::kBytes;
    uint32_t w[kBytes / 4];
    __device__ __forceinline__ void load(const unsigned char *p)
    {
        if constexpr (kBytes >= 16) {
#pragma unroll
            for (int i = 0; i < kBytes / 16; ++i) {
                const uint4 q = __ldg(reinterpret_cast<const uint4 *>(p) + i);
                w[4 * i] = q.x;
                w[4 * i + 1] = q.y;
                w[4 * i + 2] = q.z;
                w[4 * i + 3] = q.w;
            }
        } else if constexpr (kBytes == 8) {
            const uint2 q = __ldg(reinterpret_cast<const uint2 *>(p));
            w[0] = q.x;
            w[1] = q.y;
        } else {
            w[0] = __ldg(reinterpret_cast<const uint32_t *>(p));
        }
    }
    // Value p as stored (16-bit types: unscaled); flip = the sign bit conjugates it.
    __device__ __forceinline__ double2 value(int p, uint32_t flip) const
    {
        if constexpr (VT == VISTA_VIS_C128) {
            return make_double2(__hiloint2double((int)w[4 * p + 1], (int)w[4 * p]),
                                __hiloint2double((int)(w[4 * p + 3] ^ flip), (int)w[4 * p + 2]));
        } else if constexpr (VT == VISTA_VIS_C64) {
            return make_double2(widen_exact(__uint_as_float(w[2 * p])), widen_exact(__uint_as_float(w[2 * p + 1] ^ flip)));
        } else {
            const float2 f = VisType<VT>::half_pair(w[p]);
            return make_double2(widen_exact(f.x), widen_exact(__uint_as_float(__float_as_uint(f.y) ^ flip)));
        }
    }
};

// P flag bytes (P-byte aligned).
template <int P>
__device__ __forceinline__ uint32_t flags64(const uint8_t *p)
{
    if constexpr (P == 4) return __ldg(reinterpret_cast<const uint32_t *>(p));
    else if constexpr (P == 2) return __ldg(reinterpret_cast<const uint16_t *>(p));
    else return __ldg(p);
}

__device__ __forceinline__ double2 phasor64(double t)   // exp(2 pi i t)
{
    double s, c;
    sincospi(2.0 * (t - floor(t)), &s, &c);
    return make_double2(c, s);
}

// The phasors of one row (delay tau) at a chunk's nch <= 32 channels, handed to
// take(k, phasor): by recurrence from the chunk's first channel where the axis is
// linear, else one by one.
template <typename F>
__device__ __forceinline__ void chunk_phasors(const SrcDev &S, const ChanD *cd, int nch, double tau, F &&take)
{
    if (S.linear) {
        double2 ph = phasor64(tau * (cd[0].nu * (1.0 / C_LIGHT)));
        const double2 st = phasor64(tau * S.step_c);
        for (int k = 0;; ++k) {
            take(k, ph);
            if (k == nch - 1) break;
            ph = make_double2(ph.x * st.x - ph.y * st.y, ph.x * st.y + ph.y * st.x);
        }
    } else {
        for (int k = 0; k < nch; ++k) take(k, phasor64(tau * (cd[k].nu * (1.0 / C_LIGHT))));
    }
}

template <int P>
struct __align__(16) Warp64 {
    double2 ph[32][33];   // [row][channel], padded: both phases' accesses are conflict-free
    double W[32][P];      // the rows' weights
    int2 cells[32];
    uint32_t row[32], fold[32];
};

template <int P, int VT>
__global__ void __launch_bounds__(32 * WARPS64, 3) stack_fp64_runs(RunArgs a)
{
    constexpr bool half = VT == VISTA_VIS_F16X2 || VT == VISTA_VIS_BF16X2;
    extern __shared__ __align__(16) unsigned char smem[];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    Warp64<P> &T = reinterpret_cast<Warp64<P> *>(smem)[wid];
    const uint32_t nitems = a.so.ctr[a.cls + 1], G = gridDim.x * WARPS64;   // end of the class's items
    const int npol_c = a.g.npol, nrest = a.g.nrest, gnu = a.g.nu, gnv = a.g.nv;
    double *cube = reinterpret_cast<double *>(a.cube);
    unsigned long long n_read = 0, n_ok = 0, n_duv = 0;

    for (uint32_t it = a.so.ctr[a.cls] + blockIdx.x * WARPS64 + wid; it < nitems; it += G) {
        const Item I = a.so.items[it];
        const SrcDev &S = a.srcs[I.w];
        const int n = I.q1 - I.q0, nch = I.nch, kc = min(lane, nch - 1);
        const ChanD *cd = a.chd + I.chf0;
        const int j0 = cd[kc].j0, nb = cd[kc].nb;
        const double w0 = cd[kc].w[0], w1 = cd[kc].w[1];
        const bool act = lane < nch && nb > 0;
        int plane[P];
#pragma unroll
        for (int p = 0; p < P; ++p) plane[p] = S.plane[p];
        const int64_t ch = S.k_lo + I.chunk * 32 + kc;
        const unsigned char *vis = reinterpret_cast<const unsigned char *>(S.vis) + (ch - S.kbase) * Raw64<P, VT>::kBytes;
        const uint64_t vrow = (uint64_t)S.vstride * Raw64<P, VT>::kBytes;
        const uint8_t *flg = S.fbase ? S.fbase + (ch - S.fk0) * P : nullptr;
        const uint64_t frow = (uint64_t)S.fpitch;
        if (act)
#pragma unroll
            for (int p = 0; p < P; ++p) n_read += plane[p] >= 0 ? (unsigned)n : 0u;

        int cell = NO_RUN64;
        double re[P], im[P], sw[P], sa[P];
        uint32_t cnt[P];
#pragma unroll
        for (int p = 0; p < P; ++p) {
            re[p] = im[p] = sw[p] = sa[p] = 0.0;
            cnt[p] = 0u;
        }
        // A lane whose cell changes adds its run to the cube: per (rest bin,
        // pol) the four sums and the count.  The 16-bit types' values were summed
        // as stored: their scale enters here, once a run.
        auto next_cell = [&](int cid) {
            if (cid == cell) return;
            if (cell >= 0) {
                for (int b = 0; b < nb; ++b) {
                    const double ww = b == 0 ? w0 : b == 1 ? w1 : cd[kc].w[b];
                    const double wv = half ? ww * (double)S.vis_scale : ww;
                    const double wvv = half ? wv * (double)S.vis_scale : ww;
                    const int64_t e0 = ((int64_t)cell * nrest + j0 + b) * npol_c;
#pragma unroll
                    for (int p = 0; p < P; ++p) {
                        if (plane[p] < 0 || cnt[p] == 0u) continue;
                        double *e = cube + 4 * (e0 + plane[p]);
                        atomicAdd(e, wv * re[p]);
                        atomicAdd(e + 1, wv * im[p]);
                        atomicAdd(e + 2, ww * sw[p]);
                        atomicAdd(e + 3, wvv * sa[p]);
                        atomicAdd(a.count + e0 + plane[p], cnt[p]);
                    }
                }
            }
#pragma unroll
            for (int p = 0; p < P; ++p) {
                const uint32_t c = plane[p] >= 0 && cell != NO_RUN64 ? cnt[p] : 0u;
                if (cell >= 0) n_ok += c;
                else n_duv += c;
                re[p] = im[p] = sw[p] = sa[p] = 0.0;
                cnt[p] = 0u;
            }
            cell = cid;
        };

        for (int t0 = 0; t0 < n; t0 += 32) {
            const int m = min(n - t0, 32);
            __syncwarp();
            if (lane < m) {
                const RowRec rec = a.recs[I.rec0 + t0 + lane];
                T.cells[lane] = a.ccells[I.cell0 + t0 + lane];
                T.row[lane] = rec.row;
                T.fold[lane] = rec.fold;
#pragma unroll
                for (int p = 0; p < P; ++p) T.W[lane][p] = widen_exact(rec.W[P == 4 ? p : 2 * p]);
                const double *x = S.uvw + 3 * (int64_t)rec.row;   // the stored baseline: the delay of Eq. 2
                const double tau = x[0] * S.l + x[1] * S.m + x[2] * S.n1;
                chunk_phasors(S, cd, nch, tau, [&](int k, double2 ph) {
                    T.ph[lane][k] = make_double2(ph.x, rec.fold ? -ph.y : ph.y);
                });
            }
            __syncwarp();
            // the rows' values and flags are loaded one row ahead
            Raw64<P, VT> nv;
            uint32_t nf = 0;
            auto fetch = [&](int i) {
                const uint64_t row = T.row[i];
                nv.load(vis + row * vrow);
                if (flg) nf = flags64<P>(flg + row * frow);
            };
            fetch(0);
            for (int i = 0; i < m; ++i) {
                const Raw64<P, VT> v = nv;
                const uint32_t F = nf, fold = T.fold[i];
                if (i + 1 < m) fetch(i + 1);
                const int2 cc = T.cells[i];
                int cid = NO_RUN64;
                if (act) {
                    if (cc.y == CC_NOCHANGE)
                        cid = cc.x;
                    else if (cc.y != CC_MIXED)
                        cid = chunk_cell_step(cc, lane, gnu);
                    else
                        cid = cell_exact(S.guvw, T.row[i], fold != 0u, cd + kc, gnu, gnv);
                }
                next_cell(cid);
                const double2 ph = T.ph[i][kc];
#pragma unroll
                for (int p = 0; p < P; ++p) {
                    if ((F >> (8 * p)) & 0xffu) continue;
                    const double2 z = v.value(p, fold);
                    const double W = T.W[i][p], wr = W * z.x, wi = W * z.y;
                    re[p] = fma(wr, ph.x, fma(-wi, ph.y, re[p]));
                    im[p] = fma(wr, ph.y, fma(wi, ph.x, im[p]));
                    sa[p] = fma(wr, z.x, fma(wi, z.y, sa[p]));
                    sw[p] += W;
                    ++cnt[p];
                }
            }
        }
        next_cell(NO_RUN64);   // the runs still open
    }
    unsigned long long c3[2] = {n_read - n_ok - n_duv, n_duv};
#pragma unroll
    for (int k = 0; k < 2; ++k)
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) c3[k] += __shfl_xor_sync(0xffffffffu, c3[k], o);
    if (lane == 0) {
        if (c3[0]) atomicAdd(&a.stats->n_flagged, c3[0]);
        if (c3[1]) atomicAdd(&a.stats->n_dropped_uv, c3[1]);
    }
}

template <int P, int VT>
cudaError_t launch_p(const RunArgs &a, cudaStream_t st)
{
    static_assert(sizeof(Warp64<P>) % 16 == 0, "warps' areas stay aligned");
    auto kern = stack_fp64_runs<P, VT>;
    const size_t smem = WARPS64 * sizeof(Warp64<P>);
    int dev = 0, sms = 0, per_sm = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e == cudaSuccess) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, 32 * WARPS64, smem);
    if (e != cudaSuccess) return e;
    kern<<<(unsigned)(sms * (per_sm < 1 ? 1 : per_sm)), 32 * WARPS64, smem, st>>>(a);
    return cudaGetLastError();
}

template <int VT>
cudaError_t launch_vt(const RunArgs &a, int npol, cudaStream_t st)
{
    switch (npol) {
    case 1: return launch_p<1, VT>(a, st);
    case 2: return launch_p<2, VT>(a, st);
    case 4: return launch_p<4, VT>(a, st);
    default: return cudaErrorInvalidValue;
    }
}

// The phasors and cells of one window, as the stacking kernel forms them, at the
// channels that reach the cube: one thread per row.
__global__ void __launch_bounds__(128) debug_fp64(RunArgs a, int src, double *ph_out, int32_t *cell_out)
{
    const SrcDev &S = a.srcs[src];
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;   // processing order
    if (i >= S.nrow) return;
    const RowRec rec = a.recs[S.rec_off + i];
    const double *x = S.uvw + 3 * (int64_t)rec.row;   // the stored baseline: the delay of Eq. 2
    const double tau = x[0] * S.l + x[1] * S.m + x[2] * S.n1;
    for (int c = 0; c < S.nchunk; ++c) {
        const int k0 = S.k_lo + 32 * c;
        const ChanD *cd = a.chd + S.chan_off + 32 * c;
        const int2 cc = a.ccells[S.cell_off + (int64_t)c * S.nrow + i];
        chunk_phasors(S, cd, min(32, S.k_hi - k0), tau, [&](int k, double2 ph) {
            if (cd[k].nb <= 0) return;
            const int64_t o = (int64_t)rec.row * S.nchan + k0 + k;
            if (ph_out) {
                ph_out[2 * o] = ph.x;
                ph_out[2 * o + 1] = ph.y;
            }
            if (cell_out) {
                const int cid = cc.y == CC_NOCHANGE ? cc.x
                                : cc.y != CC_MIXED  ? chunk_cell_step(cc, k, a.g.nu)
                                                    : cell_exact(S.guvw, rec.row, rec.fold != 0u, cd + k, a.g.nu, a.g.nv);
                cell_out[2 * o] = cid < 0 ? -1 : cid % a.g.nu;
                cell_out[2 * o + 1] = cid < 0 ? -1 : cid / a.g.nu;
            }
        });
    }
}

}  // namespace

cudaError_t launch_debug_fp64(const RunArgs &a, int src, int64_t nrow, double *ph, int32_t *cells, cudaStream_t st)
{
    if (nrow > 0) debug_fp64<<<(unsigned)((nrow + 127) / 128), 128, 0, st>>>(a, src, ph, cells);
    return cudaGetLastError();
}

cudaError_t launch_fp64(const RunArgs &a, int key, cudaStream_t st)
{
    const int npol = key & 0xff;
    switch (key >> 16) {
    case VISTA_VIS_C64: return launch_vt<VISTA_VIS_C64>(a, npol, st);
    case VISTA_VIS_C128: return launch_vt<VISTA_VIS_C128>(a, npol, st);
    case VISTA_VIS_F16X2: return launch_vt<VISTA_VIS_F16X2>(a, npol, st);
    case VISTA_VIS_BF16X2: return launch_vt<VISTA_VIS_BF16X2>(a, npol, st);
    default: return cudaErrorInvalidValue;
    }
}

}  // namespace vista
