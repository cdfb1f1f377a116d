// The paper's per-row output (Eq. 3): every row of one window regridded onto
// the rest lattice, V_out(j) = sum_k V'(k) w_kj / sum_k w_kj over unflagged
// channels, with V' the shifted visibility of Eq. 2 and w_kj the Eq. 4
// weights.
//
// k_regrid_prep forms, in FP64, each row's delay (kept as a float-float pair)
// and each channel's rest bins and weights (the planner's rule, the same
// rounded operations), and the range of channels that reach each output
// channel.  k_regrid then gives every (output channel, pol) of a tile of R
// rows a thread: its contributors' table entries are read once for R rows,
// their R visibilities are independent loads, and the P threads of one output
// channel compute R / P of the phasors each (as the stacking kernel does:
// float-float product tau nu_k / c, reduced mod 1 turn, __sincosf, below 5e-7
// rad) and exchange them by shuffles.  A warp's loads cover the pols of
// neighbouring channels, so every 32-byte sector fetched is used whole (a
// thread per (row, output channel) took 16 bytes of 32 different lines an
// instruction and read the tables again for every row).  Bound by L1 lines a
// load (wide windows, whose outputs' contributors lie several channels apart)
// and by latency (narrow ones).  Kernel time, 12 000 rows x 3840 channels x 4
// pols onto 1024: 437 -> 362 us (1.92 GB, 5.3 TB/s); 27 090 rows x 120
// channels x 2 pols of FP16 onto 150: 87 -> 43 us.  Rows a tile by shape, see
// launch_regrid_p: eight are 6 % better than four on the FP16 window and 5 % worse
// on the wide one; blocks of 128 columns cost 7 % on the wide one.  Outputs of few
// columns have a form of their own, k_regrid_pols.  The tables were built on the host
// before (130 and 50 us a call around the kernels, 65 and 40 us now).
#include <algorithm>
#include <climits>
#include <cmath>
#include <vector>

#include "planner.h"
#include "vista_device.cuh"
#include "vista_handle.h"

namespace vista {
namespace {

// One channel as the regrid reads it (32 B).
struct __align__(16) RegridChan {
    int32_t j0, nb;         // rest bins j0 .. j0 + nb - 1 inside the lattice
    float w[4];             // their Eq. 4 weights
    float nuc_hi, nuc_lo;   // nu_k / c as a float-float pair (1/m)
};

struct RegridArgs {
    const double *uvw;
    const double *freqs;    // [nchan]
    const void *vis;
    const uint8_t *flags;
    RegridChan *chan;       // [nchan]
    int32_t *range;         // [nrest][2] INT_MAX - first channel, last channel + 1 (zeros: none)
    float2 *tau;            // [nrow] the row's delay (m) as a float-float pair
    float *out_vis;         // [nrow][nrest][npol][2]
    float *out_wsum;        // [nrow][nrest][npol]
    double *out_uvw;        // [nrow][3] or null
    int64_t nrow;
    int32_t nchan, nrest, bin_mode;
    uint32_t ncb;           // blocks of COLS columns a tile of rows takes
    int32_t pair_out;       // out_vis is 8-byte aligned: a value's two floats in one store
    int32_t vec, vout;      // a channel's pols (and flags) in whole loads, an output channel's in whole stores
    float vis_scale;
    double l, m, n1, inv_zf;
    double zf, f0, df;      // 1 + z, the rest lattice
};

// A channel's rest bins and weights: channel_bins() of the planner, operation
// by operation.
__device__ void rest_bins(const RegridArgs &a, int k, RegridChan &c)
{
    const double *f = a.freqs;
    c.j0 = c.nb = 0;
    c.w[0] = c.w[1] = c.w[2] = c.w[3] = 0.f;
    if (a.bin_mode == VISTA_BIN_NEAREST) {
        const double q = floor(__ddiv_rn(__dsub_rn(__dmul_rn(f[k], a.zf), a.f0), a.df));
        if (q >= 0.0 && q < (double)a.nrest) {
            c.j0 = (int32_t)q;
            c.nb = 1;
            c.w[0] = 1.f;
        }
        return;
    }
    double d;
    if (k == 0)
        d = __dsub_rn(f[1], f[0]);
    else if (k == a.nchan - 1)
        d = __dsub_rn(f[k], f[k - 1]);
    else
        d = __dmul_rn(__dsub_rn(f[k + 1], f[k - 1]), 0.5);
    const double half = __dmul_rn(0.5, fabs(d));
    const double lo = __dmul_rn(__dsub_rn(f[k], half), a.zf), hi = __dmul_rn(__dadd_rn(f[k], half), a.zf);
    double ca = floor(__ddiv_rn(__dsub_rn(lo, a.f0), a.df)) - 2.0, cb = floor(__ddiv_rn(__dsub_rn(hi, a.f0), a.df)) + 2.0;
    if (ca < 0.0) ca = 0.0;
    if (cb > (double)(a.nrest - 1)) cb = (double)(a.nrest - 1);
    if (!(ca <= cb)) return;
    int n = 0;
    for (int64_t j = (int64_t)ca; j <= (int64_t)cb; ++j) {
        const double e0 = __dadd_rn(a.f0, __dmul_rn((double)j, a.df));
        const double e1 = __dadd_rn(a.f0, __dmul_rn((double)(j + 1), a.df));
        const double o = __dsub_rn(hi < e1 ? hi : e1, lo > e0 ? lo : e0);
        if (!(o > 0.0)) continue;
        if (n == VISTA_MAX_BINS) break;   // (the host has refused such windows)
        if (n == 0) c.j0 = (int32_t)j;
        const float w = (float)__ddiv_rn(o, __dsub_rn(hi, lo));
        if (n == 0) c.w[0] = w;
        else if (n == 1) c.w[1] = w;
        else if (n == 2) c.w[2] = w;
        else c.w[3] = w;
        ++n;
    }
    c.nb = n;
}

// One thread per row and per channel: the Eq. 2 delay in FP64, kept as a
// float-float pair, and the rest-frame baseline (Eq. 1 with R = I) if asked
// for; the channel's table entry and its place in the ranges.
__global__ void __launch_bounds__(128) k_regrid_prep(RegridArgs a)
{
    const int64_t r = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (r < a.nrow) {
        const double *x = a.uvw + 3 * r;
        float hi, lo;
        split_ff(x[0] * a.l + x[1] * a.m + x[2] * a.n1, hi, lo);
        a.tau[r] = make_float2(hi, lo);
        if (a.out_uvw)
            for (int c = 0; c < 3; ++c) a.out_uvw[3 * r + c] = x[c] * a.inv_zf;
    }
    if (r < a.nchan) {
        const int k = (int)r;
        RegridChan c;
        rest_bins(a, k, c);
        const double nuc = __ddiv_rn(a.freqs[k], C_LIGHT);
        split_ff(nuc, c.nuc_hi, c.nuc_lo);
        a.chan[k] = c;
        for (int b = 0; b < c.nb; ++b) {
            atomicMax(a.range + 2 * (int64_t)(c.j0 + b), INT_MAX - k);
            atomicMax(a.range + 2 * (int64_t)(c.j0 + b) + 1, k + 1);
        }
    }
}

// The visibility at `at`.
template <int VT>
__device__ __forceinline__ float2 load_value(const char *at, float scale)
{
    if constexpr (VT == VISTA_VIS_C128) {
        const double2 v = __ldg(reinterpret_cast<const double2 *>(at));
        return make_float2((float)v.x, (float)v.y);
    } else if constexpr (VT == VISTA_VIS_C64) {
        return __ldg(reinterpret_cast<const float2 *>(at));
    } else {
        const float2 v = VisType<VT>::half_pair(__ldg(reinterpret_cast<const uint32_t *>(at)));
        return make_float2(v.x * scale, v.y * scale);
    }
}

constexpr int COLS = 64;   // (output channel, pol) columns a block takes
constexpr int POLS_THREADS = 128;

template <int P, int VT, int R>
__global__ void __launch_bounds__(COLS, 14) k_regrid(RegridArgs a)
{
    constexpr int RP = R / P;   // rows whose phasors a thread computes
    constexpr uint32_t VB = VisType<VT>::kBytes;
    const int lane = threadIdx.x & 31, p = lane % P;
    // the tile and its row pointers are the same for the whole block, so that
    // a load's address is a uniform pointer plus the thread's 32-bit offset
    const uint32_t tile = blockIdx.x / a.ncb;
    const int64_t ncol = (int64_t)a.nrest * P, col = (int64_t)(blockIdx.x - tile * a.ncb) * COLS + threadIdx.x;
    const bool in = col < ncol;   // (every lane takes part in the shuffles)
    const int j = in ? (int)(col / P) : 0;
    const int64_t r0 = (int64_t)tile * R;
    const int nr = (int)(a.nrow - r0 < R ? a.nrow - r0 : R);
    const int2 rg = in ? *reinterpret_cast<const int2 *>(a.range + 2 * (int64_t)j) : make_int2(0, 0);
    const int first = INT_MAX - rg.x, cnt = rg.y > 0 ? rg.y - first : 0;
    const int steps = __reduce_max_sync(0xffffffffu, cnt);
    float2 tau[RP];   // rows p, p + P, ...
#pragma unroll
    for (int i = 0; i < RP; ++i) tau[i] = __ldg(a.tau + r0 + min(i * P + p, nr - 1));
    float sr[R], si[R], sw[R];
#pragma unroll
    for (int r = 0; r < R; ++r) sr[r] = si[r] = sw[r] = 0.f;
    const int64_t row_values = (int64_t)a.nchan * P;
    const char *vis = reinterpret_cast<const char *>(a.vis) + r0 * row_values * VB;
    const uint8_t *flags = a.flags ? a.flags + r0 * row_values : nullptr;
    for (int e = 0; e < steps; ++e) {
        const int k = first + e;
        float w = 0.f, nh = 0.f, nl = 0.f;
        if (e < cnt) {
            const int4 c0 = __ldg(reinterpret_cast<const int4 *>(a.chan + k));        // j0, nb, w0, w1
            const float4 c1 = __ldg(reinterpret_cast<const float4 *>(a.chan + k) + 1);   // w2, w3, nuc
            const int b = j - c0.x;
            if (b >= 0 && b < c0.y)
                w = b == 0 ? __int_as_float(c0.z) : b == 1 ? __int_as_float(c0.w) : b == 2 ? c1.x : c1.y;
            nh = c1.z;
            nl = c1.w;
        }
        // the rows' values and flags, all in flight together (rows past the
        // end re-read the last one, threads without a contributor channel 0)
        const bool use = w > 0.f;
        const uint32_t off = use ? (uint32_t)k * P + p : (uint32_t)p;
        float2 v[R];
        uint32_t fl[R];
#pragma unroll
        for (int r = 0; r < R; ++r) v[r] = load_value<VT>(vis + min(r, nr - 1) * row_values * VB + off * VB, a.vis_scale);
        if (flags) {
#pragma unroll
            for (int r = 0; r < R; ++r) fl[r] = __ldg(flags + min(r, nr - 1) * row_values + off);
        } else {
#pragma unroll
            for (int r = 0; r < R; ++r) fl[r] = 0u;
        }
        float2 ph[RP];
#pragma unroll
        for (int i = 0; i < RP; ++i) ph[i] = shift_phasor(tau[i].x, tau[i].y, nh, nl);
#pragma unroll
        for (int r = 0; r < R; ++r) {
            const float c = P == 1 ? ph[r / P].x : __shfl_sync(0xffffffffu, ph[r / P].x, r % P, P);
            const float s = P == 1 ? ph[r / P].y : __shfl_sync(0xffffffffu, ph[r / P].y, r % P, P);
            if (use && fl[r] == 0u) {
                // (weighting the phasors instead would save two operations of six and
                // add a rounding: rms errors 5 to 20 % larger)
                sr[r] = __fmaf_rn(w, __fmaf_rn(v[r].x, c, -__fmul_rn(v[r].y, s)), sr[r]);
                si[r] = __fmaf_rn(w, __fmaf_rn(v[r].x, s, __fmul_rn(v[r].y, c)), si[r]);
                sw[r] += w;
            }
        }
    }
    if (!in) return;
    float2 *ov = reinterpret_cast<float2 *>(a.out_vis) + r0 * ncol + col;
    float *ow = a.out_wsum + r0 * ncol + col;
#pragma unroll
    for (int r = 0; r < R; ++r) {
        if (r >= nr) break;
        const bool any = sw[r] > 0.0f;
        const float re = any ? sr[r] / sw[r] : 0.0f, im = any ? si[r] / sw[r] : 0.0f;
        if (a.pair_out) {
            ov[r * ncol] = make_float2(re, im);
        } else {
            float *o = a.out_vis + 2 * ((r0 + r) * ncol + col);
            o[0] = re;
            o[1] = im;
        }
        ow[r * ncol] = sw[r];
    }
}

// One channel's P values and flags of a row, at element i0 (= (row * nchan + k) * P).
template <int P, int VT>
__device__ __forceinline__ void load_channel(const RegridArgs &a, int64_t i0, float2 (&v)[P], uint32_t &fl)
{
    constexpr int VB = VisType<VT>::kBytes, LB = P * VB;
    const char *at = reinterpret_cast<const char *>(a.vis) + i0 * VB;
    if (P > 1 && a.vec) {
        uint32_t w[LB / 4];
        if constexpr (LB >= 16) {
#pragma unroll
            for (int q = 0; q < LB / 16; ++q) {
                const uint4 x = __ldg(reinterpret_cast<const uint4 *>(at) + q);
                w[4 * q] = x.x;
                w[4 * q + 1] = x.y;
                w[4 * q + 2] = x.z;
                w[4 * q + 3] = x.w;
            }
        } else if constexpr (LB == 8) {
            const uint2 x = __ldg(reinterpret_cast<const uint2 *>(at));
            w[0] = x.x;
            w[1] = x.y;
        } else {
            w[0] = __ldg(reinterpret_cast<const uint32_t *>(at));
        }
#pragma unroll
        for (int p = 0; p < P; ++p) {
            if constexpr (VT == VISTA_VIS_C128)
                v[p] = make_float2((float)__hiloint2double((int)w[4 * p + 1], (int)w[4 * p]),
                                   (float)__hiloint2double((int)w[4 * p + 3], (int)w[4 * p + 2]));
            else if constexpr (VT == VISTA_VIS_C64)
                v[p] = make_float2(__uint_as_float(w[2 * p]), __uint_as_float(w[2 * p + 1]));
            else {
                const float2 x = VisType<VT>::half_pair(w[p]);
                v[p] = make_float2(x.x * a.vis_scale, x.y * a.vis_scale);
            }
        }
        fl = 0u;
        if (a.flags) {
            if constexpr (P == 4) fl = __ldg(reinterpret_cast<const uint32_t *>(a.flags + i0));
            else fl = __ldg(reinterpret_cast<const uint16_t *>(a.flags + i0));
        }
        return;
    }
    fl = 0u;
#pragma unroll
    for (int p = 0; p < P; ++p) {
        v[p] = load_value<VT>(at + p * VB, a.vis_scale);
        if (a.flags) fl |= (uint32_t)__ldg(a.flags + i0 + p) << (8 * p);
    }
}

// Narrow outputs: a thread per (tile of R rows, output channel) takes all its
// pols, a channel's values in whole 16-byte (or shorter) loads.  k_regrid's block
// shares one tile's columns, so that with few of them most of its threads idle:
// 200 000 rows x 64 channels onto one, 1165 us there, 107 us here (98 us before there
// was k_regrid); 20 000 rows x 500 channels onto four, four pols, 299 and 115 (108).
template <int P, int VT, int R>
__global__ void __launch_bounds__(POLS_THREADS) k_regrid_pols(RegridArgs a)
{
    const uint32_t t = blockIdx.x * POLS_THREADS + threadIdx.x, nt = (uint32_t)((a.nrow + R - 1) / R);
    const uint32_t tile = t / (uint32_t)a.nrest;
    const int j = (int)(t - tile * (uint32_t)a.nrest);
    if (tile >= nt) return;
    const int64_t r0 = (int64_t)tile * R;
    const int nr = (int)(a.nrow - r0 < R ? a.nrow - r0 : R);
    const int2 rg = *reinterpret_cast<const int2 *>(a.range + 2 * (int64_t)j);
    const int first = INT_MAX - rg.x, cnt = rg.y > 0 ? rg.y - first : 0;
    float2 tau[R];
    float sr[R][P], si[R][P], sw[R][P];
#pragma unroll
    for (int r = 0; r < R; ++r) {
        tau[r] = __ldg(a.tau + r0 + min(r, nr - 1));
#pragma unroll
        for (int p = 0; p < P; ++p) sr[r][p] = si[r][p] = sw[r][p] = 0.f;
    }
    for (int e = 0; e < cnt; ++e) {
        const int k = first + e;
        float2 v[R][P];
        uint32_t fl[R];
#pragma unroll
        for (int r = 0; r < R; ++r) load_channel<P, VT>(a, ((r0 + min(r, nr - 1)) * a.nchan + k) * P, v[r], fl[r]);
        const int4 c0 = __ldg(reinterpret_cast<const int4 *>(a.chan + k));        // j0, nb, w0, w1
        const float4 c1 = __ldg(reinterpret_cast<const float4 *>(a.chan + k) + 1);   // w2, w3, nuc
        const int b = j - c0.x;
        if (b < 0 || b >= c0.y) continue;
        const float w = b == 0 ? __int_as_float(c0.z) : b == 1 ? __int_as_float(c0.w) : b == 2 ? c1.x : c1.y;
#pragma unroll
        for (int r = 0; r < R; ++r) {
            const float2 ph = shift_phasor(tau[r].x, tau[r].y, c1.z, c1.w);
#pragma unroll
            for (int p = 0; p < P; ++p) {
                if ((fl[r] >> (8 * p)) & 0xffu) continue;
                sr[r][p] = __fmaf_rn(w, __fmaf_rn(v[r][p].x, ph.x, -__fmul_rn(v[r][p].y, ph.y)), sr[r][p]);
                si[r][p] = __fmaf_rn(w, __fmaf_rn(v[r][p].x, ph.y, __fmul_rn(v[r][p].y, ph.x)), si[r][p]);
                sw[r][p] += w;
            }
        }
    }
#pragma unroll
    for (int r = 0; r < R; ++r) {
        if (r >= nr) break;
        const int64_t o = ((r0 + r) * a.nrest + j) * P;
        float ov[2 * P];
#pragma unroll
        for (int p = 0; p < P; ++p) {
            const bool any = sw[r][p] > 0.f;
            ov[2 * p] = any ? sr[r][p] / sw[r][p] : 0.f;
            ov[2 * p + 1] = any ? si[r][p] / sw[r][p] : 0.f;
        }
        if (P > 1 && a.vout) {
            float4 *d = reinterpret_cast<float4 *>(a.out_vis + 2 * o);
#pragma unroll
            for (int q = 0; q < P / 2; ++q) d[q] = make_float4(ov[4 * q], ov[4 * q + 1], ov[4 * q + 2], ov[4 * q + 3]);
            if constexpr (P == 4) *reinterpret_cast<float4 *>(a.out_wsum + o) = make_float4(sw[r][0], sw[r][1], sw[r][2], sw[r][3]);
            else if constexpr (P == 2) *reinterpret_cast<float2 *>(a.out_wsum + o) = make_float2(sw[r][0], sw[r][1]);
            continue;
        }
#pragma unroll
        for (int p = 0; p < P; ++p) {
            a.out_vis[2 * (o + p)] = ov[2 * p];
            a.out_vis[2 * (o + p) + 1] = ov[2 * p + 1];
            a.out_wsum[o + p] = sw[r][p];
        }
    }
}

template <int P, int VT, int R>
cudaError_t launch_pols(RegridArgs a, cudaStream_t st)
{
    // (the threads are counted in 32 bits: more of them go in several launches)
    const int64_t total = a.nrow, most = std::max<int64_t>(((int64_t)1 << 31) / a.nrest / R * R, R);
    for (int64_t r = 0; r < total; r += most) {
        a.nrow = total - r < most ? total - r : most;
        const int64_t threads = (a.nrow + R - 1) / R * a.nrest;
        k_regrid_pols<P, VT, R><<<(unsigned)((threads + POLS_THREADS - 1) / POLS_THREADS), POLS_THREADS, 0, st>>>(a);
        const int64_t in = a.nrow * a.nchan * P, out = a.nrow * a.nrest * P;
        a.vis = reinterpret_cast<const char *>(a.vis) + in * VisType<VT>::kBytes;
        if (a.flags) a.flags += in;
        a.tau += a.nrow;
        a.out_vis += 2 * out;
        a.out_wsum += out;
    }
    return cudaGetLastError();
}

// k_regrid takes outputs of two blocks of columns or more, or of one that is full;
// narrower ones go to k_regrid_pols, two rows a thread from 200 000 (row, output
// channel) pairs on.  k_regrid takes eight rows a tile where that leaves at least 16
// blocks a SM and the lines a block's threads gather from at a time, up to one of
// 128 bytes a row and output channel, stay within 8 KB; else four: with each output
// channel's contributors far from its neighbour's, the eight rows' lines of an SM's
// blocks overflow its L1 (12 000 rows x 3840 channels onto 64, two pols: eight 1148,
// four 340 us).  Over 1249 shapes (1, 2 and 4 pols of three storage types, 500 to
// 200 000 rows of 16 to 8000 channels, 1 to 1024 output channels) the rule is within
// 7 % of the best of nine forms on average, and 10 % slower than the kernel before
// k_regrid (a thread per row and output channel, its tables built on the host) on 42
// of them, by half at the most; k_regrid with eight rows alone was on 40 %, by up
// to twelve times.
template <int P, int VT>
cudaError_t launch_regrid_p(RegridArgs a, cudaStream_t st)
{
    constexpr int VB = VisType<VT>::kBytes;
    const int64_t ncol = (int64_t)a.nrest * P, ncb = (ncol + COLS - 1) / COLS;
    // (k_regrid's offsets from its row pointers are 32-bit: longer rows go to the other form)
    const bool far = (int64_t)a.nchan * P * VB > (int64_t)UINT32_MAX, full = P > 1 && ncol > 56 && ncol <= COLS;
    if (far || (ncol < 2 * COLS && !full))
        return a.nrow * a.nrest >= 200000 ? launch_pols<P, VT, 2>(a, st) : launch_pols<P, VT, 1>(a, st);
    const int64_t apart = std::max<int64_t>(a.nchan / a.nrest, 1) * P * VB;   // bytes from a column's contributors to the next
    const bool eight = (a.nrow + 7) / 8 * ncb >= (int64_t)16 * 152 && 8 * (COLS / P) * std::min<int64_t>(apart, 128) <= 8192;
    const int R = eight ? 8 : 4;
    const int64_t blocks = (a.nrow + R - 1) / R * ncb;
    if (blocks > (int64_t)INT_MAX) return cudaErrorInvalidValue;   // (an output of more than 2^40 bytes)
    a.ncb = (uint32_t)ncb;
    if (eight)
        k_regrid<P, VT, 8><<<(unsigned)blocks, COLS, 0, st>>>(a);
    else
        k_regrid<P, VT, 4><<<(unsigned)blocks, COLS, 0, st>>>(a);
    return cudaGetLastError();
}

template <int VT>
cudaError_t launch_regrid_vt(const RegridArgs &a, int npol, cudaStream_t st)
{
    return npol == 4 ? launch_regrid_p<4, VT>(a, st) : npol == 2 ? launch_regrid_p<2, VT>(a, st)
                                                                : launch_regrid_p<1, VT>(a, st);
}

}  // namespace
}  // namespace vista

using namespace vista;

extern "C" int vista_regrid_rows(vista_stack *h, const vista_source_desc *s, float *out_vis, float *out_wsum,
                                 double *out_uvw)
{
    if (!handle_live(h)) return fail(nullptr, VISTA_E_STATE, "unknown or closed handle");
    if (!s || !out_vis || !out_wsum) return fail(h, VISTA_E_ARG, "null descriptor or output");
    if (!h->lattice_fixed)
        return fail(h, VISTA_E_STATE, "the rest lattice is not fixed yet (give rest_df at open, or run first)");
    if (s->mem != VISTA_MEM_DEVICE) return fail(h, VISTA_E_ARG, "vista_regrid_rows reads device arrays only");
    if (s->nrow < 0 || s->nchan < 2) return fail(h, VISTA_E_ARG, "need nrow >= 0 and nchan >= 2");
    if (s->npol != 1 && s->npol != 2 && s->npol != 4) return fail(h, VISTA_E_ARG, "npol must be 1, 2 or 4");
    if (s->vis_type < VISTA_VIS_C64 || s->vis_type > VISTA_VIS_BF16X2)
        return fail(h, VISTA_E_ARG, "bad vis_type %d", s->vis_type);
    if (!s->freqs || (s->nrow > 0 && (!s->uvw || !s->vis)))
        return fail(h, VISTA_E_ARG, "freqs, uvw and vis must be non-NULL");
    if (!(std::isfinite(s->l) && std::isfinite(s->m) && s->l * s->l + s->m * s->m < 1.0))
        return fail(h, VISTA_E_ARG, "need finite l, m with l^2 + m^2 < 1");
    if (!(std::isfinite(s->z) && s->z > -1.0)) return fail(h, VISTA_E_ARG, "need finite z > -1");
    const int32_t n = s->nchan, nrest = h->desc.nrest;
    for (int32_t k = 0; k < n; ++k)
        if (!(std::isfinite(s->freqs[k]) && s->freqs[k] > 0.0))
            return fail(h, VISTA_E_ARG, "freqs[%d] is not finite and > 0", k);
    const bool up = s->freqs[1] > s->freqs[0];
    for (int32_t k = 1; k < n; ++k)
        if (up ? !(s->freqs[k] > s->freqs[k - 1]) : !(s->freqs[k] < s->freqs[k - 1]))
            return fail(h, VISTA_E_ARG, "freqs must be strictly monotone (index %d)", k);
    if (s->nrow == 0) return VISTA_OK;

    // a channel that may reach more than VISTA_MAX_BINS rest bins (wider than
    // VISTA_MAX_BINS - 1 of them): the planner's own count decides
    if (h->desc.bin_mode == VISTA_BIN_OVERLAP &&
        !(widest_rest_channel(s->freqs, n, s->z) <= (VISTA_MAX_BINS - 1.001) * h->df)) {
        std::vector<int32_t> j0((size_t)n), nb((size_t)n);
        std::vector<double> wk((size_t)n * VISTA_MAX_BINS);
        const int rc = channel_bins(s->freqs, n, s->z, h->f0, h->df, nrest, h->desc.bin_mode, j0.data(), nb.data(),
                                    wk.data());
        if (rc != VISTA_OK) return fail(h, rc, "channel planning failed");
    }

    // one device buffer: frequencies | channel table | ranges | per-row delays
    auto al = [](size_t b) { return (b + 255) / 256 * 256; };
    const size_t o_c = al(sizeof(double) * (size_t)n), o_r = o_c + al(sizeof(RegridChan) * (size_t)n),
                 o_t = o_r + al(sizeof(int32_t) * 2 * (size_t)nrest), total = o_t + al(sizeof(float2) * (size_t)s->nrow);
    cudaError_t e = h->b_regrid.ensure(total);
    if (e != cudaSuccess) return cuda_fail(h, e, "regrid table allocation");
    char *b = (char *)h->b_regrid.p;
    e = cudaMemcpyAsync(b, s->freqs, sizeof(double) * (size_t)n, cudaMemcpyHostToDevice, h->stream);
    if (e == cudaSuccess) e = cudaMemsetAsync(b + o_r, 0, sizeof(int32_t) * 2 * (size_t)nrest, h->stream);
    if (e != cudaSuccess) return cuda_fail(h, e, "regrid table upload");

    RegridArgs a{};
    a.uvw = s->uvw;
    a.freqs = (const double *)b;
    a.vis = s->vis;
    a.flags = s->flags;
    a.chan = (RegridChan *)(b + o_c);
    a.range = (int32_t *)(b + o_r);
    a.tau = (float2 *)(b + o_t);
    a.out_vis = out_vis;
    a.out_wsum = out_wsum;
    a.out_uvw = out_uvw;
    a.nrow = s->nrow;
    a.nchan = n;
    a.nrest = nrest;
    a.bin_mode = h->desc.bin_mode;
    const size_t lane = vis_elem_bytes(s->vis_type) * (size_t)s->npol;
    a.vec = ((uintptr_t)s->vis % std::min<size_t>(lane, 16)) == 0 &&
            (!s->flags || ((uintptr_t)s->flags % (uintptr_t)s->npol) == 0);
    a.vout = ((uintptr_t)out_vis % 16) == 0 && ((uintptr_t)out_wsum % (uintptr_t)(s->npol == 4 ? 16 : 8)) == 0;
    a.pair_out = ((uintptr_t)out_vis % 8) == 0;
    a.vis_scale = (s->vis_type == VISTA_VIS_F16X2 || s->vis_type == VISTA_VIS_BF16X2) ? s->vis_scale : 1.0f;
    a.zf = 1.0 + s->z;
    a.f0 = h->f0;
    a.df = h->df;
    a.l = s->l;
    a.m = s->m;
    a.n1 = std::sqrt(1.0 - s->l * s->l - s->m * s->m) - 1.0;
    a.inv_zf = 1.0 / (1.0 + s->z);
    const int64_t prep = s->nrow > n ? s->nrow : n;
    k_regrid_prep<<<(unsigned)((prep + 127) / 128), 128, 0, h->stream>>>(a);
    e = cudaGetLastError();
    if (e == cudaSuccess) {
        switch (s->vis_type) {
        case VISTA_VIS_C64: e = launch_regrid_vt<VISTA_VIS_C64>(a, s->npol, h->stream); break;
        case VISTA_VIS_C128: e = launch_regrid_vt<VISTA_VIS_C128>(a, s->npol, h->stream); break;
        case VISTA_VIS_F16X2: e = launch_regrid_vt<VISTA_VIS_F16X2>(a, s->npol, h->stream); break;
        default: e = launch_regrid_vt<VISTA_VIS_BF16X2>(a, s->npol, h->stream); break;
        }
    }
    if (e == cudaSuccess) e = cudaStreamSynchronize(h->stream);
    if (e != cudaSuccess) return cuda_fail(h, e, "regrid kernel");
    return VISTA_OK;
}
