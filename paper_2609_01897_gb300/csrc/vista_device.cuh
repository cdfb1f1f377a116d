// Device helpers shared by the libvista kernels: work-list lookups, FP32
// phasors, the guarded uv-cell rule and the visibility / flag loaders.
#pragma once
#include <cuda_bf16.h>
#include <cuda_fp16.h>

#include "vista_internal.h"

namespace vista {

// ---------------------------------------------------------------- helpers

// Largest s with off[s] <= x (off non-decreasing, off[0] = 0).  The table is
// read through the read-only path: nothing may write it while the kernel is on
// the chip (a table uploaded before the pre-pass, not one that the pre-pass forms).
__device__ __forceinline__ int find_owner(const int64_t *__restrict__ off, int n, int64_t x)
{
    int lo = 0, hi = n - 1;
    while (lo < hi) {
        int mid = (lo + hi + 1) >> 1;
        if (__ldg(off + mid) <= x)
            lo = mid;
        else
            hi = mid - 1;
    }
    return lo;
}

// The same over a table that an earlier kernel of the chain writes: ordinary
// loads (see chain_begin).
__device__ __forceinline__ int find_owner_chained(const int64_t *off, int n, int64_t x)
{
    int lo = 0, hi = n - 1;
    while (lo < hi) {
        int mid = (lo + hi + 1) >> 1;
        if (off[mid] <= x)
            lo = mid;
        else
            hi = mid - 1;
    }
    return lo;
}

// ---- programmatic dependent launch ----
//
// The pre-pass is a chain of short kernels; each is launched while the one
// before it still runs (launch_chained) and first waits for that one to end,
// its writes visible.  Only then does it let its own successor be launched,
// so that at most two kernels of the chain are on the chip and everything
// older, the caller's inputs among it, is complete.  About a microsecond a
// kernel: a test-sized stack's call 160 -> 141 us together with the readback's
// single wait.  The stacking kernels are launched as usual: their persistent
// blocks, waiting on the chip before the pre-pass has ended, cost the FP64
// form 6 % and an archive stack 1 %.
//
// A chained kernel's blocks are on the chip while the kernel before them still
// writes.  What the chain writes is therefore never read through the read-only
// path (__ldg, find_owner): such loads are only defined for data that nothing
// writes during the whole life of the kernel, waiting part included, and may
// be moved across the wait.

__device__ __forceinline__ void chain_begin()
{
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}

template <typename... KA, typename... A>
static cudaError_t launch_chained(void (*kern)(KA...), unsigned grid, unsigned block, size_t smem, cudaStream_t st,
                                  A... args)
{
    cudaLaunchAttribute at{};
    at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at.val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(block);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cfg.attrs = &at;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kern, args...);
}

// ---- TMA bulk copies into shared memory, completed on an mbarrier ----

__device__ __forceinline__ uint32_t smem_addr(const void *p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ void mbar_init(uint64_t *bar, uint32_t count)
{
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_addr(bar)), "r"(count) : "memory");
}

__device__ __forceinline__ void mbar_init_fence() { asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory"); }

__device__ __forceinline__ void fence_proxy_async() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }

__device__ __forceinline__ void mbar_expect_tx(uint64_t *bar, uint32_t bytes)
{
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_addr(bar)), "r"(bytes)
                 : "memory");
}

// 1-D bulk copy global -> shared (16-byte aligned addresses, size a multiple of 16).
__device__ __forceinline__ void tma_load_1d(void *dst, const void *src, uint32_t bytes, uint64_t *bar)
{
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
                     smem_addr(dst)),
                 "l"(src), "r"(bytes), "r"(smem_addr(bar))
                 : "memory");
}

__device__ __forceinline__ bool mbar_try_wait(uint64_t *bar, uint32_t parity)
{
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\tselp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(smem_addr(bar)), "r"(parity)
        : "memory");
    return ok != 0;
}

// Bounded wait: gives up after ~2^24 polls (seconds), records the failure in
// the error word and returns false; never traps and never spins forever.
constexpr int32_t ERR_WAIT_TIMEOUT = 1;
__device__ __forceinline__ bool mbar_wait_bounded(uint64_t *bar, uint32_t parity, int32_t *err)
{
    for (uint32_t i = 0; i < (1u << 24); ++i)
        if (mbar_try_wait(bar, parity)) return true;
    atomicExch(err, ERR_WAIT_TIMEOUT);
    return false;
}

// exp(2 pi i t) for a reduced turn count |t| <= 1/2 (|2 pi t| <= pi).
// CUDA's __sincosf has an absolute error of at most 2^-21.41 on [-pi, pi]
// (CUDA C Programming Guide, intrinsic functions), i.e. a phase error below
// 5e-7 rad, inside the 1e-5 rad budget, in two special-function-unit
// instructions.
__device__ __forceinline__ float2 turns_to_phasor(float t)
{
    float s, c;
    __sincosf(__fmul_rn(t, 6.28318530717958648f), &s, &c);
    return make_float2(c, s);
}

// exp(+2 pi i tau nu_k / c) from tau and nu_k / c given as float-float
// pairs.  The product is formed as p + e + x: p = fl(tau_hi nuc_hi), e its
// exact rounding error (one FMA), x the cross terms; tau_lo nuc_lo is below
// 2^-48 of the product and dropped.  p minus its nearest integer is exact, so
// the turns reach turns_to_phasor reduced, with an error of about 2^-25 turn
// (2e-7 rad) for phases up to 2^23 turns.
__device__ __forceinline__ float2 shift_phasor(float tau_hi, float tau_lo, float nuc_hi, float nuc_lo)
{
    const float p = __fmul_rn(tau_hi, nuc_hi);
    const float e = __fmaf_rn(tau_hi, nuc_hi, -p);
    const float x = __fmaf_rn(tau_hi, nuc_lo, __fmaf_rn(tau_lo, nuc_hi, e));
    const float r = __fsub_rn(p, rintf(p));
    return turns_to_phasor(__fadd_rn(r, x));
}

// Split a double into a float-float pair hi + lo.
__device__ __host__ __forceinline__ void split_ff(double x, float &hi, float &lo)
{
    hi = (float)x;
    lo = (float)(x - (double)hi);
}

// The floor of one axis of the uv cell rule, floor(fl64(coord * s_k)),
// decided in FP32 when fl32(c32 * s32) is at least 2^-21 |x| away
// from an integer (the FP32 product differs from the FP64 one by at most
// 3 * 2^-24 |x|), else by the exact FP64 product.
// The exact FP64 product, out of line so that the compiler cannot hoist it
// (and its FP64 work) out of the rarely taken branch below.
static __device__ __noinline__ float exact_floor_product(const double *coord64, bool neg, const double *s64)
{
    double c = *coord64;
    if (neg) c = -c;
    return (float)floor(__dmul_rn(c, *s64));
}

// floor(fl64(coord * s_k)) as a float (exact).
__device__ __forceinline__ float axis_floor(float c32, float s32, const double *coord64, bool neg,
                                            const double *s64)
{
    float x = __fmul_rn(c32, s32);
    float d = __fmaf_rn(fabsf(x), 4.76837158203125e-07f, 1e-30f);
    float fa = floorf(__fsub_rn(x, d)), fb = floorf(__fadd_rn(x, d));
    float fx = fa;
    if (__builtin_expect(fa != fb, 0)) fx = exact_floor_product(coord64, neg, s64);
    return fx;
}

__device__ __forceinline__ int axis_cell64(double c, double s, int n)
{
    double x = __dmul_rn(c, s);
    double h = (double)(n >> 1);
    if (!(x >= -h && x < h)) return -1;
    return (int)floor(x) + (n >> 1);
}

// Eq. 1: the gridding coordinates (u', v') = the first two rows of R (u, v, w)
// of one row of a re-projected window, each product and sum rounded in the
// order written (no FMA, as the oracle), so that the FP64 cell rule applied
// to them is exact.  Stored at g[0], g[1] (g[2], w', is not needed: the delay
// uses the stored baseline); returned as well.
__device__ __forceinline__ double2 rotate_row(const double *R, const double *x, double *g)
{
    const double a = x[0], b = x[1], c = x[2];
    const double u = __dadd_rn(__dadd_rn(__dmul_rn(R[0], a), __dmul_rn(R[1], b)), __dmul_rn(R[2], c));
    const double v = __dadd_rn(__dadd_rn(__dmul_rn(R[3], a), __dmul_rn(R[4], b)), __dmul_rn(R[5], c));
    g[0] = u;
    g[1] = v;
    return make_double2(u, v);
}

// The cell iv * nu + iu of channel `cd` of one row by the FP64 rule, -1 off
// the grid (the fall-back of CC_MIXED chunks; out of line, rarely run).
static __device__ __noinline__ int cell_exact(const double *uvw, int64_t row, bool fold, const ChanD *cd, int nu,
                                              int nv)
{
    double u = uvw[3 * row], v = uvw[3 * row + 1];
    if (fold) {
        u = -u;
        v = -v;
    }
    const int iu = axis_cell64(u, cd->su, nu), iv = axis_cell64(v, cd->sv, nv);
    return (iu >= 0 && iv >= 0) ? iv * nu + iu : -1;
}

// Cell of chunk-local channel kk from a chunk-cell entry that is neither
// CC_NOCHANGE nor CC_MIXED.
__device__ __forceinline__ int chunk_cell_step(int2 cc, int kk, int nu)
{
    const uint32_t m = (uint32_t)cc.y;
    int c = cc.x;
    if (kk >= (int)(m & 0xffu)) c += (m & 0x10000u) ? -1 : 1;
    if (kk >= (int)((m >> 8) & 0xffu)) c += (m & 0x20000u) ? -nu : nu;
    return c;
}

// ------------------------------------------------ stored visibility types

// Bytes of one complex value, and the 16-bit types' decoding.
template <int VT>
struct VisType {
    static constexpr int kBytes = VT == VISTA_VIS_C128 ? 16 : VT == VISTA_VIS_C64 ? 8 : 4;
    static __device__ __forceinline__ float2 half_pair(uint32_t b)
    {
        if constexpr (VT == VISTA_VIS_F16X2) {
            return __half22float2(*reinterpret_cast<__half2 *>(&b));
        } else {   // bf16 -> f32 is a 16-bit shift
            return make_float2(__uint_as_float(b << 16), __uint_as_float(b & 0xffff0000u));
        }
    }
};

// ---- shared-memory loads at a 32-bit address plus a constant ----

template <int OFF>
__device__ __forceinline__ uint32_t lds32(uint32_t at)
{
    uint32_t x;
    asm volatile("ld.shared.u32 %0, [%1+%2];" : "=r"(x) : "r"(at), "n"(OFF));
    return x;
}
template <int OFF>
__device__ __forceinline__ uint64_t lds64(uint32_t at)
{
    uint64_t x;
    asm volatile("ld.shared.b64 %0, [%1+%2];" : "=l"(x) : "r"(at), "n"(OFF));
    return x;
}
template <int OFF>
__device__ __forceinline__ ulonglong2 lds128(uint32_t at)
{
    ulonglong2 x;
    asm volatile("ld.shared.v2.b64 {%0, %1}, [%2+%3];" : "=l"(x.x), "=l"(x.y) : "r"(at), "n"(OFF));
    return x;
}

// ---- packed FP32 pairs (one instruction for both halves) ----

__device__ __forceinline__ uint64_t pack2(float x, float y)
{
    uint64_t r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(x), "f"(y));
    return r;
}
__device__ __forceinline__ float2 unpack2(uint64_t v)
{
    float2 r;
    asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(v));
    return r;
}
__device__ __forceinline__ uint64_t mul2(uint64_t a, uint64_t b)
{
    uint64_t r;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}

// A folded row's values conjugated (sign = the sign bit; 0 leaves them): with
// its delay negated in the record, the shifted visibilities come out conjugated.
template <int P>
__device__ __forceinline__ void conjugate(uint64_t (&v)[P], uint32_t sign)
{
#pragma unroll
    for (int p = 0; p < P; ++p) v[p] ^= (uint64_t)sign << 32;
}

// Adds one visibility V = (re, im), weighted WV = w V, to a lane's sums unless
// its flag byte is set: C += w V c, S += w V s (as pairs; cc = (c, c), ss =
// (s, s)), A += (w re^2, w im^2), sw += w, cnt += 1.  Predicated, so a flagged
// value (whatever it holds) never enters.
__device__ __forceinline__ void add_value(uint64_t &C, uint64_t &S, uint64_t &A, float &sw, uint32_t &cnt, uint64_t V,
                                          uint64_t WV, float w, uint64_t cc, uint64_t ss, uint32_t flag)
{
    asm("{\n\t.reg .pred p;\n\t"
        "setp.eq.u32 p, %11, 0;\n\t"
        "@p fma.rn.f32x2 %0, %6, %8, %0;\n\t"
        "@p fma.rn.f32x2 %1, %6, %9, %1;\n\t"
        "@p fma.rn.f32x2 %2, %6, %5, %2;\n\t"
        "@p add.rn.f32 %3, %3, %7;\n\t"
        "@p add.u32 %4, %4, %10;\n\t}"
        : "+l"(C), "+l"(S), "+l"(A), "+f"(sw), "+r"(cnt)
        : "l"(V), "l"(WV), "f"(w), "l"(cc), "l"(ss), "n"(1), "r"(flag));
}

// ---- asynchronous copies of one lane's visibilities into shared memory ----

__device__ __forceinline__ void cp_async_16(uint32_t dst, const void *src)
{
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async_8(uint32_t dst, const void *src)
{
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(dst), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async_4(uint32_t dst, const void *src)
{
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(dst), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory"); }

// One lane's P values of one (row, channel): kLaneBytes bytes, naturally
// aligned (a multiple of the element size), copied by cp.async in 16-, 8- or
// 4-byte pieces and decoded from shared memory.
template <int P, int VT>
struct VisAsync {
    static constexpr int kLaneBytes = P * VisType<VT>::kBytes;
    static __device__ __forceinline__ void copy(uint32_t dst, const void *src)
    {
        const char *s = reinterpret_cast<const char *>(src);
        if constexpr (kLaneBytes % 16 == 0) {
#pragma unroll
            for (int i = 0; i < kLaneBytes / 16; ++i) cp_async_16(dst + 16 * i, s + 16 * i);
        } else if constexpr (kLaneBytes == 8) {
            cp_async_8(dst, s);
        } else {
            static_assert(kLaneBytes == 4, "lane bytes");
            cp_async_4(dst, s);
        }
    }
    // The values at shared address at + OFF as (re, im) operand pairs.
    template <int OFF>
    static __device__ __forceinline__ void decode(uint32_t at, float scale, uint64_t (&v)[P])
    {
        if constexpr (VT == VISTA_VIS_C64) {
            if constexpr (P == 1) {
                v[0] = lds64<OFF>(at);
            } else {
                const ulonglong2 q = lds128<OFF>(at);
                v[0] = q.x;
                v[1] = q.y;
                if constexpr (P == 4) {
                    const ulonglong2 r = lds128<OFF + 16>(at);
                    v[2] = r.x;
                    v[3] = r.y;
                }
            }
        } else if constexpr (VT == VISTA_VIS_C128) {
            auto one = [&](ulonglong2 q) {
                return pack2((float)__longlong_as_double((long long)q.x), (float)__longlong_as_double((long long)q.y));
            };
            v[0] = one(lds128<OFF>(at));
            if constexpr (P >= 2) v[1] = one(lds128<OFF + 16>(at));
            if constexpr (P == 4) {
                v[2] = one(lds128<OFF + 32>(at));
                v[3] = one(lds128<OFF + 48>(at));
            }
        } else {
            const uint64_t s2 = pack2(scale, scale);
            auto one = [&](uint32_t b) {
                const float2 f = VisType<VT>::half_pair(b);
                return mul2(pack2(f.x, f.y), s2);
            };
            if constexpr (P == 1) {
                v[0] = one(lds32<OFF>(at));
            } else if constexpr (P == 2) {
                const uint64_t q = lds64<OFF>(at);
                v[0] = one((uint32_t)q);
                v[1] = one((uint32_t)(q >> 32));
            } else {
                const ulonglong2 q = lds128<OFF>(at);
                v[0] = one((uint32_t)q.x);
                v[1] = one((uint32_t)(q.x >> 32));
                v[2] = one((uint32_t)q.y);
                v[3] = one((uint32_t)(q.y >> 32));
            }
        }
    }
};

// P flag bytes (P-byte aligned) at shared address at + OFF, zero-extended.
template <int P, int OFF>
__device__ __forceinline__ uint32_t flag_bytes(uint32_t at)
{
    if constexpr (P == 4) {
        return lds32<OFF>(at);
    } else if constexpr (P == 2) {
        uint16_t h;
        asm volatile("ld.shared.u16 %0, [%1+%2];" : "=h"(h) : "r"(at), "n"(OFF));
        return h;
    } else {
        uint32_t f;
        asm volatile("ld.shared.u8 %0, [%1+%2];" : "=r"(f) : "r"(at), "n"(OFF));
        return f;
    }
}

// Vector reduction into one cube entry (no returned value).
__device__ __forceinline__ void red_add4(void *p, float x, float y, float z, float w)
{
    asm volatile("red.global.add.v4.f32 [%0], {%1, %2, %3, %4};" ::"l"(p), "f"(x), "f"(y), "f"(z), "f"(w) : "memory");
}

}  // namespace vista
