// The mixed-precision stacking kernel (sm_103a).  Each visibility type's
// instantiations are compiled in a translation unit of their own
// (vista_stack_<type>.cu, built in parallel); vista_stack.cu dispatches.
//
// Persistent: warp g of G takes work items g, g + G, g + 2G, ... of a list
// in stripe-major order (item = one window, up to rows_per_item rows in
// uv-cell order, a chunk of 32 x NS channels, walked 32 at a time, lane =
// channel).  While a warp processes an item, TMA bulk copies (one mbarrier
// per slot) bring the next item's row records, chunk cells, window header,
// channel table and work-list entries into the other shared-memory slot, so
// an item starts without a global round trip.  Inside an item the
// visibilities and flags of the next rows are in flight into a shared-memory
// ring (cp.async, two rows a group).  Each lane copies the 4-byte flag
// word that holds its flags (a chunk's flags start on a word, see
// flag_align_channels) and, when a lane's values are at most 16 bytes, its
// own values.  Wider values (four pols, or complex128) are copied in 16-byte
// pieces with piece i of lane L at byte 512 i + 16 L of the row's ring slot,
// so that every cp.async instruction of the warp reads 512 contiguous
// bytes (a lane copying its own 32 bytes as two pieces would make each
// instruction read half of every 32-byte sector, and fetch each sector from
// L2 twice); the warp then synchronises before a group's values are read and
// before their ring slots are refilled.
//
// The kernel is bound by the issue and latency of its instructions (57 to 64 %
// issue with 15 warps an SM) before it is bound by HBM, so it is built to spend
// few instructions per (row, 32 channels):
//  - the arithmetic is in packed FP32 pairs (one instruction per pair): with
//    (c, s) the phasor and v = (re, im) a value, the sums of W v c and W v s
//    are kept as pairs and combined (re = C.re - S.im, im = C.im + S.re) only
//    when a run ends, so a value costs a multiply and three packed FMAs;
//  - rows are taken two at a time (their phasors are independent work);
//  - a bit per row says whether any lane's cell can differ from the row
//    before (its chunk-cell entry differs, or is CC_MIXED); the cell logic
//    runs on those rows only;
//
// Per (row, channel): the FP32 phasor of Eq. 2 from the record's float-float
// delay and the channel's float-float nu_k / c, the uv cell from the chunk's
// cell entry (exact: computed by the pre-pass with the FP64 rule), rest bins
// and Eq. 4 weights from the FP64 channel table.  Per lane, running sums
// over consecutive rows that share a uv cell stay in registers.  When a
// lane's cell changes, its finished run goes to a per-warp stack in shared
// memory (slots from a warp ballot); once 32 runs wait the warp drains them
// together, one lane per run: runs of one cell that meet in a rest bin are
// added up across the lanes, then each (cell, rest bin, pol) gets one float4
// reduction and each pol pair one u64 count reduction.  The L2 takes about
// 2.2e11 32-byte sectors of reductions a second however few of their bytes
// change, and does not combine lanes of one address, so without the merging
// the reductions bound the kernel (0.49 of them per visibility on a compact
// array's stack, 0.25 merged; 0.150 and 0.019 on an archive stack; without any
// the kernel would now gain 1 to 2 %).  Runs off the grid only feed the dropped
// counter.
//
// Measured, before (values through predicated scalar arithmetic, one row at a
// time, runs written unmerged) and now, kernel time: a compact array's stack,
// two pols of complex64, 5.2e8 visibilities, 1.96 -> 1.56 ms; an archive
// stack, 1.2e10 visibilities of two and four pols, 28.5 -> 22.2 ms (5.1 TB/s);
// wideband FP16, 7.5e8 visibilities, 2.75 -> 1.89 ms; long baselines in BF16,
// 4.6e8 visibilities, 1.46 -> 1.13 ms.  Per (row, 32 channels) of two pols a
// warp issues about 78 instructions where no run ends (99 before the row loop
// lost its branches), 112 on the compact array's stack (178 before).
#pragma once
#include <climits>

#include "vista_device.cuh"

namespace vista {

constexpr int RB_MAX = 256;         // largest item (rows) the shared-memory buffers hold
constexpr int KMAX_THREADS = 128;   // blocks of at most 4 warps
constexpr uint32_t CKPT_EVERY = 8;     // 1 / probability that a drain checkpoints what it writes (a power of two)
constexpr int NO_RUN = INT_MIN;     // lane holds no run

// What a window without flags reads as its flags (every row: pitch 0).
__device__ __align__(16) uint8_t g_zero_flags[512];

// Rows between two looks at the number of staged runs, and the runs the stack
// holds: at most 31 wait before those rows, each of which may stage 32.
template <int P>
__host__ __device__ constexpr int stage_rows() { return P == 4 ? 1 : 2; }
template <int P>
__host__ __device__ constexpr int stage_cap() { return 32 * (stage_rows<P>() + 1); }

// Staged runs, field by field (every access of a warp is conflict-free).
//   acc   [P][cap]  sum W V'.re, sum W V'.im, sum W, sum W |V|^2
//   head  [cap]     x = cell iv * nu + iu (-1 off the grid); y = lane (its
//                   channel, 5 bits) | count of pol 0 << 5 | of pol 1 << 16
//   more  [cap]     four pols: counts of pols 2 and 3 << 16
// (a run has at most RB_MAX = 256 rows: a count takes 9 bits).
template <int P>
struct Stage {
    static constexpr int cap = stage_cap<P>();
    static constexpr size_t bytes = (size_t)cap * (16 * P + 8 + (P == 4 ? 4 : 0));
    float4 *acc;
    uint2 *head;
    uint32_t *more;
    __device__ explicit Stage(unsigned char *base)
    {
        acc = reinterpret_cast<float4 *>(base);
        head = reinterpret_cast<uint2 *>(acc + P * cap);
        more = reinterpret_cast<uint32_t *>(head + cap);
    }
};

// A channel-table entry as two 16-byte loads.
__device__ __forceinline__ ChanF load_chanf(const ChanF *p)
{
    const int4 a = *reinterpret_cast<const int4 *>(p);
    const float4 b = *reinterpret_cast<const float4 *>(reinterpret_cast<const char *>(p) + 16);
    ChanF c;
    c.su = __int_as_float(a.x);
    c.sv = __int_as_float(a.y);
    c.j0 = a.z;
    c.nb = a.w;
    c.w0 = b.x;
    c.w1 = b.y;
    c.nuc_hi = b.z;
    c.nuc_lo = b.w;
    return c;
}

// Weight of a third or fourth rest bin (lattices narrower than a channel;
// out of line so that its FP64 conversion is not hoisted into every drain).
static __device__ __noinline__ float far_bin_weight(const ChanD *cd, int b) { return (float)cd->w[b]; }

// A float as a double, exactly, by moving its IEEE-754 fields (integer
// instructions; the FP64 unit converts slowly).  Zero and subnormal inputs
// give zero (below 1.2e-38); infinities and NaNs stay what they are.
__device__ __forceinline__ double widen(float x)
{
    const uint32_t b = __float_as_uint(x);
    const uint32_t e = (b >> 23) & 0xffu;
    if (e == 0u) return 0.0;
    const uint32_t e64 = e == 0xffu ? 0x7ffu : e + 896u;
    const uint32_t hi = (b & 0x80000000u) | (e64 << 20) | ((b & 0x7fffffu) >> 3);
    return __hiloint2double((int)hi, (int)(b << 29));
}

// Chunk-cell entries per slot: an item's rows plus the entries that round
// its bulk copy out to 16-byte boundaries.
__host__ __device__ constexpr int cc_slot_entries(int rb) { return (rb + 3) & ~1; }

// Row records a slot holds past the item's rows: the row loop fetches that far
// ahead without a look at the item's end (they repeat the last row's index).
constexpr int REC_PAD = 10;

// One item slot in shared memory (filled by bulk copies).
__host__ __device__ constexpr size_t slot_bytes(int rb)
{
    return 2 * sizeof(Item) + sizeof(SrcDev) + (size_t)(rb + REC_PAD) * sizeof(RowRec) +
           (size_t)cc_slot_entries(rb) * sizeof(int2);
}

// Per-warp shared memory: two item slots, the ring of NG groups of two rows
// (values, flag words), the staged runs and two mbarriers.
template <int P, int VT, int NG>
__host__ __device__ constexpr size_t warp_smem_bytes(int rb)
{
    return 2 * slot_bytes(rb) + (size_t)NG * 2 * 32 * (VisAsync<P, VT>::kLaneBytes + 4) + Stage<P>::bytes +
           2 * sizeof(uint64_t);
}

// Views of one slot.
struct Slot {
    Item *self, *next;   // this item, the item after it (same warp)
    SrcDev *hdr;
    RowRec *rec;
    int2 *cells;
    __device__ Slot(unsigned char *base, int rb)
    {
        self = reinterpret_cast<Item *>(base);
        next = self + 1;
        hdr = reinterpret_cast<SrcDev *>(next + 1);
        rec = reinterpret_cast<RowRec *>(hdr + 1);
        cells = reinterpret_cast<int2 *>(rec + rb + REC_PAD);
    }
};

// Blocks of four warps an SM must hold: 128 registers a thread, or 168 for
// four pols (whose sums and shared memory allow three blocks only).
template <int P>
__host__ __device__ constexpr int min_blocks() { return P == 4 ? 3 : 4; }

template <int P, int VT, int NG>
__global__ void __launch_bounds__(KMAX_THREADS, (min_blocks<P>())) stack_mixed(RunArgs a)
{
    using VA = VisAsync<P, VT>;
    constexpr int LB = VA::kLaneBytes;          // bytes of a lane's values
    constexpr int VROW = 32 * LB;               // bytes of a row's values in the ring
    constexpr uint32_t RS = VROW + 128;         // bytes of a ring row: values, flag words
    static_assert(2 * NG <= REC_PAD, "records read past an item's end (the pair that holds row n fetches furthest)");
    extern __shared__ __align__(16) unsigned char smem[];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const int RB = a.so.rows_per_item, CW = a.cw;
    unsigned char *wsm = smem + (size_t)wid * warp_smem_bytes<P, VT, NG>(RB);
    auto slot_at = [&](int s) { return Slot(wsm + (size_t)s * slot_bytes(RB), RB); };
    unsigned char *ring = wsm + 2 * slot_bytes(RB);
    const Stage<P> stage(ring + NG * 2 * RS);
    uint64_t *bars = reinterpret_cast<uint64_t *>(ring + NG * 2 * RS + Stage<P>::bytes);
    const uint32_t ring_s = smem_addr(ring);
    if (lane == 0) {
        mbar_init(&bars[0], 1);
        mbar_init(&bars[1], 1);
        mbar_init_fence();
    }
    __syncwarp();

    const uint32_t nitems = a.so.ctr[a.cls + 1];   // end of the class's items
    const uint32_t G = gridDim.x * (blockDim.x >> 5);
    const uint32_t gw = blockIdx.x * (blockDim.x >> 5) + wid;
    const int npol_c = a.g.npol, nrest = a.g.nrest, gnu = a.g.nu, gnv = a.g.nv;
    const bool comp = a.comp != 0, folds = a.g.fold != 0;
    float4 *cube4 = reinterpret_cast<float4 *>(a.cube);
    // visibilities read, stacked (unflagged, on the grid) and dropped off the
    // grid; flagged = read - stacked - dropped
    uint32_t n_read = 0, n_ok = 0, n_duv = 0, n_red = 0;
    // state of the checkpoint schedule (a linear congruential sequence per warp)
    uint32_t rnd = gw * 2654435761u + 12345u;
    // the lane's pending checkpoint: FP32 sums taken out of the cube, to be
    // added to the master entry ck_dst
    float4 ck_took = make_float4(0.f, 0.f, 0.f, 0.f);
    double *ck_dst = nullptr;
    auto flush_ckpt = [&]() {
        if (ck_dst) {
            atomicAdd(ck_dst, widen(ck_took.x));
            atomicAdd(ck_dst + 1, widen(ck_took.y));
            atomicAdd(ck_dst + 2, widen(ck_took.z));
            atomicAdd(ck_dst + 3, widen(ck_took.w));
            const int64_t ce = (ck_dst - a.cube_master) >> 2;
            atomicOr(a.moved + (ce >> 5), 1u << (ce & 31));
            n_red += 4;
            ck_dst = nullptr;
        }
    };
    // warp sums of the counters, one atomic per counter per warp (at the
    // end, or early if a lane's count nears 2^32)
    auto flush_counters = [&]() {
        unsigned long long c3[3] = {(unsigned long long)n_read - n_ok - n_duv, n_duv, n_red};
#pragma unroll
        for (int k = 0; k < 3; ++k)
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) c3[k] += __shfl_xor_sync(0xffffffffu, c3[k], o);
        if (lane == 0) {
            if (c3[0]) atomicAdd(&a.stats->n_flagged, c3[0]);
            if (c3[1]) atomicAdd(&a.stats->n_dropped_uv, c3[1]);
            if (c3[2]) atomicAdd(&a.stats->n_reductions, c3[2]);
        }
        n_read = n_ok = n_duv = n_red = 0;
    };
    const unsigned below = (1u << lane) - 1u, above = ~below & ~(1u << lane);   // lanes below, above this one
    uint32_t phase = 0;   // bit s: parity of the next completion of slot s

    // Lane 0: bulk copies of item `it` (its entry `item`) into slot s,
    // together with the entry of the warp's following item `itn`, if any.
    auto issue = [&](int s, uint32_t it, const Item &item, uint32_t itn) {
        const Slot S = slot_at(s);
        const int n = item.q1 - item.q0;
        const int64_t e0a = item.cell0 & ~(int64_t)1;
        const uint32_t ncc = (uint32_t)((item.cell0 + n - e0a + 1) & ~(int64_t)1);
        const uint32_t b_items = (uint32_t)sizeof(Item) * (itn < nitems ? 2u : 1u);
        const uint32_t b_rec = (uint32_t)n * (uint32_t)sizeof(RowRec), b_cc = ncc * (uint32_t)sizeof(int2);
        fence_proxy_async();
        mbar_expect_tx(&bars[s], b_items + (uint32_t)sizeof(SrcDev) + b_rec + b_cc);
        tma_load_1d(S.self, a.so.items + it, (uint32_t)sizeof(Item), &bars[s]);
        if (itn < nitems) tma_load_1d(S.next, a.so.items + itn, (uint32_t)sizeof(Item), &bars[s]);
        tma_load_1d(S.hdr, a.srcs + item.w, (uint32_t)sizeof(SrcDev), &bars[s]);
        tma_load_1d(S.rec, a.recs + item.rec0, b_rec, &bars[s]);
        tma_load_1d(S.cells, a.ccells + e0a, b_cc, &bars[s]);
    };

    uint32_t it = a.so.ctr[a.cls] + gw;
    if (lane == 0 && it < nitems) {
        const Item first = a.so.items[it];
        issue(0, it, first, it + G);
    }
    int s = 0;
    for (; it < nitems; it += G, s ^= 1) {
        const int cs = s;
        __syncwarp();
        if (!mbar_wait_bounded(&bars[cs], (phase >> cs) & 1u, a.err)) {
            // the copy in flight gets one more bounded wait before the warp stops
            mbar_wait_bounded(&bars[cs], (phase >> cs) & 1u, a.err);
            break;
        }
        phase ^= 1u << cs;
        const Slot S = slot_at(cs);
        // the next item's copies run while this one is processed
        if (lane == 0 && it + G < nitems) issue(cs ^ 1, it + G, *S.next, it + 2 * G);

        // ---- one item ----
        // window fields in registers (the cube reductions could alias global
        // memory, so reads through pointers would be repeated)
        const SrcDev &H = *S.hdr;
        const int2 *cb = S.cells + (S.self->cell0 & 1);
        // (the reductions over the warp leave loop bounds in uniform registers)
        const int n = __reduce_max_sync(0xffffffffu, S.self->q1 - S.self->q0);
        const int nch = __reduce_max_sync(0xffffffffu, S.self->nch), chf0 = S.self->chf0;
        if (lane < 2 * NG) {
            S.rec[n + lane].row = S.rec[n - 1].row;
            fence_proxy_async();   // before the bulk copies that refill the slot
        }
        __syncwarp();
        const uint32_t vrow_bytes = (uint32_t)(H.vstride * LB);   // visibility bytes per row
        const uint32_t frow_bytes = H.fbase ? (uint32_t)H.fpitch : 0u;   // flag bytes per row (0: none, every row reads g_zero_flags)
        const float vscale = H.vis_scale;
        int plane[P];
#pragma unroll
        for (int p = 0; p < P; ++p) plane[p] = H.plane[p];
        // pol pairs (2k, 2k + 1) whose count entries are adjacent and 8-byte
        // aligned take one u64 reduction for both counts
        constexpr int NPK = P >= 2 ? P / 2 : 1;
        bool pk[NPK];
#pragma unroll
        for (int k = 0; k < NPK; ++k)
            pk[k] = P >= 2 && plane[2 * k] >= 0 && plane[2 * k + 1] == plane[2 * k] + 1 && !(plane[2 * k] & 1) &&
                    !(npol_c & 1);
        // every pol on its own plane, planes adjacent from an even one on (or
        // one pol): entries and count pairs at fixed distances from plane[0]'s
        bool std_planes = plane[0] >= 0, pairs = false;
#pragma unroll
        for (int k = 0; k < (P >= 2 ? P / 2 : 0); ++k) {
            std_planes = std_planes && pk[k] && plane[2 * k] == plane[0] + 2 * k;
            pairs = pairs || pk[k];
        }

        // the chunk, 32 channels at a time
        for (int k0 = 0; k0 < nch; k0 += 32) {
            // lane = channel k0 + lane of the chunk; lanes past its last channel
            // load that channel (always inside the row) and never hold a run
            const int nck = min(nch - k0, 32), lk = min(lane, nck - 1), kk = k0 + lane;
            // visibilities: the lane's source address in row 0 (wide values:
            // those of the pieces it copies, pieces past the chunk's last
            // channel re-read that channel's bytes)
            const int64_t c0 = (int64_t)(H.k_lo + S.self->chunk * CW + k0);
            const unsigned char *v0 = reinterpret_cast<const unsigned char *>(H.vis) + (c0 - H.kbase) * LB;
            constexpr int NPC = LB >= 32 ? LB / 16 : 1;
            const unsigned char *vsrc[NPC];
#pragma unroll
            for (int i = 0; i < NPC; ++i) {
                const int g = 512 * i + 16 * lane;
                vsrc[i] = LB < 32 ? v0 + lk * LB : v0 + (g / LB < nck ? g : (nck - 1) * LB + g % LB);
            }
            // flags: the word holding the lane's bytes, and their place in it
            const uint8_t *fsrc = (H.fbase ? H.fbase + (c0 - H.fk0) * P : g_zero_flags) + ((lk * P) & ~3);
            const uint32_t flag_at = ring_s + VROW + 4u * lane + ((lk * P) & 3), vis_at = ring_s + (uint32_t)(lane * LB);
            const uint32_t vdst = ring_s + (uint32_t)(LB >= 32 ? 16 * lane : LB * lane), fdst = ring_s + VROW + 4u * lane;

            // one row into the ring row at byte `to`
            auto fetch = [&](uint32_t to, uint32_t row) {
                if constexpr (LB >= 32) {
#pragma unroll
                    for (int q = 0; q < NPC; ++q)
                        cp_async_16(vdst + to + 512u * q, vsrc[q] + (uint64_t)row * vrow_bytes);
                } else {
                    VA::copy(vdst + to, vsrc[0] + (uint64_t)row * vrow_bytes);
                }
                cp_async_4(fdst + to, fsrc + (uint64_t)row * frow_bytes);
            };
#pragma unroll
            for (int d = 0; d < 2 * (NG - 1); ++d) {
                fetch(RS * d, S.rec[d].row);
                if (d & 1) cp_async_commit();
            }

            // the lane's channel, its latency under that of the first rows
            const ChanF cf = load_chanf(a.chf + chf0 + k0 + lk);
            const float nh = cf.nuc_hi, nl = cf.nuc_lo, w0 = cf.w0, w1 = cf.w1;
            const int nb = cf.nb;
            const bool act = lane < nck && nb > 0;
            if (act) {
                int npl = 0;
#pragma unroll
                for (int p = 0; p < P; ++p) npl += plane[p] >= 0;
                n_read += (uint32_t)(n * npl);
            }
            // runs merge across lanes when the planes are regular and no channel
            // reaches a third bin; the lane's first bin and (sign bit) whether it
            // has a second one; the lanes that come before it in the stack (the
            // ones with lower bins)
            const bool merge = std_planes && !__any_sync(0xffffffffu, act && nb > 2);
            const int jn = cf.j0 | (nb >= 2 ? INT_MIN : 0);
            const unsigned first = __shfl_sync(0xffffffffu, nh, 0) <= __shfl_sync(0xffffffffu, nh, nck - 1) ? below : above;
            const int64_t cell_entries = (int64_t)nrest * npol_c;
            // narrow channels: all of them lie in one rest bin or two adjacent ones
            const int jlo = __reduce_min_sync(0xffffffffu, act ? cf.j0 : INT_MAX);
            const int jhi = __reduce_max_sync(0xffffffffu, act ? cf.j0 + nb - 1 : -1);
            const bool narrow = P == 4 && merge && jhi - jlo <= 1;

            // the lane's cell in row i (NO_RUN for a lane without a channel);
            // chunk entries are shared by the warp: the branch is uniform
            auto lane_cell = [&](int i) -> int {
                const int2 cc = cb[i];
                int cid = NO_RUN;
                if (cc.y != CC_MIXED) {
                    cid = cc.x;
                    if (cc.y != CC_NOCHANGE) cid = chunk_cell_step(cc, kk, gnu);
                } else if (act) {
                    cid = cell_exact(H.guvw, S.rec[i].row, S.rec[i].fold != 0u, a.chd + chf0 + kk, gnu, gnv);
                }
                return act ? cid : NO_RUN;
            };

            int cell = lane_cell(0);
            uint64_t accC[P], accS[P], accA[P];
            float accW[P];
            uint32_t cnt[P];
            auto clear = [&]() {
#pragma unroll
                for (int p = 0; p < P; ++p) {
                    accC[p] = accS[p] = accA[p] = 0ull;
                    accW[p] = 0.f;
                    cnt[p] = 0u;
                }
            };
            clear();

            // Narrow channels: the runs of the lanes `fl`, all in cell c, added up
            // across the warp per rest bin.  Each halving of the lanes also halves
            // the 4 P sums a lane carries on, so that lane L ends with the total of
            // sum L / (32 / 4 P) and the entry's sums go out as one reduction of
            // adjacent floats; the counts of a pol pair are added as 16-bit halves.
            // Staged and drained, such runs would meet in the same entries all the
            // same, at three times the instructions (four pols: 17.3 -> 14.4 ms then on
            // the four-pol windows of an archive stack; two pols: no gain).
            auto reduce_runs = [&](int c, bool fl) {
                constexpr int N = 4 * P, LPS = 32 / N;   // sums, lanes per sum in the end
                rnd = rnd * 1664525u + 1013904223u;
                const bool service = comp && (rnd >> 16) % CKPT_EVERY == 0;
                if (fl) {
#pragma unroll
                    for (int p = 0; p < P; ++p) n_ok += cnt[p];
                }
#pragma unroll 1
                for (int j = jlo; j <= jhi; ++j) {
                    const bool in = fl && (cf.j0 == j || (nb >= 2 && cf.j0 + 1 == j));
                    if (!__any_sync(0xffffffffu, in)) continue;
                    const float ww = cf.j0 == j ? w0 : w1;
                    float x[N];
                    uint32_t m[(P + 1) / 2];
#pragma unroll
                    for (int p = 0; p < P; ++p) {
                        const float2 C = unpack2(accC[p]), D = unpack2(accS[p]), A = unpack2(accA[p]);
                        x[4 * p] = in ? ww * (C.x - D.y) : 0.f;
                        x[4 * p + 1] = in ? ww * (C.y + D.x) : 0.f;
                        x[4 * p + 2] = in ? ww * accW[p] : 0.f;
                        x[4 * p + 3] = in ? ww * (A.x + A.y) : 0.f;
                    }
#pragma unroll
                    for (int k = 0; k < (P + 1) / 2; ++k) {
                        m[k] = in ? cnt[2 * k] : 0u;
                        if constexpr (P >= 2) m[k] |= in ? cnt[2 * k + 1] << 16 : 0u;
                        m[k] = __reduce_add_sync(0xffffffffu, m[k]);
                    }
#pragma unroll
                    for (int h = N / 2, bit = 16; bit > 0; h >>= 1, bit >>= 1) {
                        if (h > 0) {
                            const bool hi = (lane & bit) != 0;
#pragma unroll
                            for (int i = 0; i < (h > 0 ? h : 1); ++i) {
                                const float keep = hi ? x[i + h] : x[i], give = hi ? x[i] : x[i + h];
                                x[i] = keep + __shfl_xor_sync(0xffffffffu, give, bit);
                            }
                        } else {
                            x[0] += __shfl_xor_sync(0xffffffffu, x[0], bit);
                        }
                    }
                    const int64_t e = (int64_t)c * cell_entries + (int64_t)j * npol_c + plane[0];
                    const int which = lane / LPS;   // the sum this lane holds: component which % 4 of pol which / 4
                    if (lane % LPS == 0) {
                        atomicAdd(reinterpret_cast<float *>(cube4 + e) + which, x[0]);
                        ++n_red;
                    }
                    if (lane < (P + 1) / 2) {
                        uint32_t mm = m[0];
                        if constexpr (P == 4) mm = lane == 0 ? m[0] : m[1];
                        if constexpr (P == 1) {
                            atomicAdd(a.count + e, mm);
                        } else {
                            atomicAdd(reinterpret_cast<unsigned long long *>(a.count + e + 2 * lane),
                                      (unsigned long long)(mm & 0xffffu) | ((unsigned long long)(mm >> 16) << 32));
                        }
                        ++n_red;
                    }
                    if (service && lane % (4 * LPS) == 0) {
                        flush_ckpt();
                        const int64_t ce = e + which / 4;
                        ck_took = atomicExch(cube4 + ce, make_float4(0.f, 0.f, 0.f, 0.f));
                        ck_dst = a.cube_master + 4 * ce;
                        ++n_red;
                    }
                }
            };

            // A lane whose cell changes stages its finished run and starts a new
            // one, in the order of the lanes' bins.
            uint32_t count = 0;   // staged runs
            auto next_cell = [&](int cid) {
                const bool fl = cid != cell;
                const unsigned bal = __ballot_sync(0xffffffffu, fl);
                if (P == 4 && narrow && __popc(bal) >= 8) {
                    // many lanes end a run, as a rule in one cell: the warp adds the
                    // runs up and writes the one or two entries itself (from how many
                    // on hardly matters, the lanes end their runs together or nearly
                    // alone: 1, 4, 8, 16 and 32 give 12.52 to 12.56 ms on the four-pol
                    // windows of an archive stack; never, 13.27 ms)
                    const int c0 = __shfl_sync(0xffffffffu, cell, __ffs(bal) - 1);
                    if (c0 >= 0 && __all_sync(0xffffffffu, !fl || cell == c0)) {
                        reduce_runs(c0, fl);
                        if (fl) {
                            cell = cid;
                            clear();
                        }
                        return;
                    }
                }
                if (fl) {
                    const uint32_t i = count + __popc(bal & first);
                    uint2 hd = make_uint2((uint32_t)cell, (uint32_t)lane | (cnt[0] << 5));
                    if constexpr (P >= 2) hd.y |= cnt[1] << 16;
                    stage.head[i] = hd;
                    if constexpr (P == 4) stage.more[i] = cnt[2] | (cnt[3] << 16);
#pragma unroll
                    for (int p = 0; p < P; ++p) {
                        const float2 C = unpack2(accC[p]), D = unpack2(accS[p]), A = unpack2(accA[p]);
                        stage.acc[p * Stage<P>::cap + i] = make_float4(C.x - D.y, C.y + D.x, accW[p], A.x + A.y);
                    }
                    cell = cid;
                    clear();
                }
                count += __popc(bal);
            };

            // The warp writes min(count, 32) staged runs to the cube, lane r the
            // r-th of the last 32.  Runs of one cell whose channels share a rest
            // bin, and the second bin of a run with the first bin of the next,
            // are added up across the lanes first (see the top of the file).  Then
            // one float4 reduction per (cell, rest bin, pol) and the counts.
            //
            // With checkpoints (comp), in one drain in CKPT_EVERY (drawn by the
            // warp's sequence) the writing lanes also move one entry each into the
            // FP64 master cube: 16-byte atomic exchange with zero, and the FP64
            // reductions of the value taken at the lane's next exchange (or at the
            // end), so nothing waits on a returned value.  The entry is one of
            // those the lane has just added to, its bin and pol drawn anew each
            // time (a bin may be no channel's first: the upper half of a channel
            // two bins wide, a window's last bin), so that every entry's FP32 sum
            // holds only the additions since its last checkpoint, about
            // CKPT_EVERY x P x (bins a lane writes) of them.
            auto drain = [&]() {
                __syncwarp();
                const uint32_t k = count < 32u ? count : 32u;
                count -= k;
                rnd = rnd * 1664525u + 1013904223u;
                const bool service = comp && (rnd >> 16) % CKPT_EVERY == 0;
                const bool have = (uint32_t)lane < k;
                const uint32_t i = count + (have ? lane : 0);
                const uint2 hd = stage.head[i];
                const int rc = (int)hd.x, src = (int)(hd.y & 31u);
                uint32_t rn[P];
                rn[0] = (hd.y >> 5) & 0x1ffu;
                if constexpr (P >= 2) rn[1] = hd.y >> 16;
                if constexpr (P == 4) {
                    const uint32_t m = stage.more[i];
                    rn[2] = m & 0xffffu;
                    rn[3] = m >> 16;
                }
                float v[P][4];
#pragma unroll
                for (int p = 0; p < P; ++p) {
                    const float4 q = stage.acc[p * Stage<P>::cap + i];
                    v[p][0] = q.x;
                    v[p][1] = q.y;
                    v[p][2] = q.z;
                    v[p][3] = q.w;
                }
                // the run's channel: its first bin, weights
                const int rjn = __shfl_sync(0xffffffffu, jn, src);
                const float r0 = __shfl_sync(0xffffffffu, w0, src), r1 = __shfl_sync(0xffffffffu, w1, src);
                const int rj = rjn & INT_MAX;
                uint32_t tot = 0;
#pragma unroll
                for (int p = 0; p < P; ++p) tot += plane[p] >= 0 ? rn[p] : 0u;
                const bool on = have && rc >= 0;
                if (have && rc < 0) n_duv += tot;
                if (on) n_ok += tot;
                const int64_t e = (int64_t)rc * cell_entries + (int64_t)rj * npol_c + (std_planes ? plane[0] : 0);
                if (merge) {
                    // z: the sums for the run's first bin, y: for its second
                    const bool two = on && rjn < 0;
                    float z[P][4], y[P][4];
                    uint32_t zn[P];
#pragma unroll
                    for (int p = 0; p < P; ++p) {
                        zn[p] = rn[p];
#pragma unroll
                        for (int c = 0; c < 4; ++c) {
                            z[p][c] = r0 * v[p][c];
                            y[p][c] = r1 * v[p][c];
                        }
                    }
                    // the lane below: same cell, and its second bin is this lane's
                    // first (up), or the same first bin (same)
                    const int pc = __shfl_up_sync(0xffffffffu, rc, 1), pj = __shfl_up_sync(0xffffffffu, rjn, 1);
                    const bool next_to = lane > 0 && on && pc == rc;
                    const bool up = next_to && pj < 0 && (pj & INT_MAX) + 1 == rj;
                    const bool same = next_to && (pj & INT_MAX) == rj;
                    const unsigned upm = __ballot_sync(0xffffffffu, up), samem = __ballot_sync(0xffffffffu, same);
                    if (upm) {
#pragma unroll
                        for (int p = 0; p < P; ++p) {
#pragma unroll
                            for (int c = 0; c < 4; ++c) {
                                const float q = __shfl_up_sync(0xffffffffu, y[p][c], 1);
                                if (up) z[p][c] += q;
                            }
                            const uint32_t q = __shfl_up_sync(0xffffffffu, rn[p], 1);
                            if (up) zn[p] += q;
                        }
                    }
                    // sums over neighbours of one first bin, to the last of them
                    if (samem) {
                        const int dist = __clz(~(samem << (31 - lane)));   // lanes below of the same bin
                        for (int d = 1; __any_sync(0xffffffffu, dist >= d); d <<= 1) {
                            const bool take = dist >= d;
#pragma unroll
                            for (int p = 0; p < P; ++p) {
#pragma unroll
                                for (int c = 0; c < 4; ++c) {
                                    const float q = __shfl_up_sync(0xffffffffu, z[p][c], d);
                                    if (take) z[p][c] += q;
                                }
                                const uint32_t q = __shfl_up_sync(0xffffffffu, zn[p], d);
                                if (take) zn[p] += q;
                            }
                        }
                    }
                    const bool emit = on && !((samem >> 1 >> lane) & 1u);          // no lane above takes it further
                    const bool emit2 = two && !((upm >> 1 >> lane) & 1u);
                    auto add = [&](int64_t at, const float (&x)[P][4], const uint32_t (&m)[P]) {
#pragma unroll
                        for (int p = 0; p < P; ++p) red_add4(cube4 + at + p, x[p][0], x[p][1], x[p][2], x[p][3]);
                        if constexpr (P == 1) {
                            atomicAdd(a.count + at, m[0]);
                        } else {
#pragma unroll
                            for (int k2 = 0; k2 < P / 2; ++k2)
                                atomicAdd(reinterpret_cast<unsigned long long *>(a.count + at + 2 * k2),
                                          (unsigned long long)m[2 * k2] | ((unsigned long long)m[2 * k2 + 1] << 32));
                        }
                        n_red += P + (P + 1) / 2;
                    };
                    if (emit) add(e, z, zn);
                    if (emit2) add(e + npol_c, y, rn);
                    if (service && (emit || emit2)) {
                        // complete the lane's previous exchange, whose value has long
                        // arrived, then take the chosen entry's FP32 sums
                        flush_ckpt();
                        const bool second = emit2 && (!emit || (rnd >> 28 & 1u));
                        const int64_t ce = e + (second ? npol_c : 0) + ((rnd >> 20) + (uint32_t)lane) % P;
                        ck_took = atomicExch(cube4 + ce, make_float4(0.f, 0.f, 0.f, 0.f));
                        ck_dst = a.cube_master + 4 * ce;
                        ++n_red;
                    }
                } else {
                    // per (rest bin, pol) the sums and, by the pair where the planes
                    // allow it, the counts.  Two loops, chosen for the whole warp:
                    // with the pairs looked for in one loop, stacks without any
                    // took 8 % longer (325 -> 351 us, 2.0e7 visibilities of two
                    // separate planes, a run each); without the pairs, channels over
                    // three bins 601 -> 700 us (two pols, 2.0e7 visibilities).
                    const int rb = __shfl_sync(0xffffffffu, nb, src);
                    const int64_t kt = chf0 + k0 + src;   // the run's channel-table entry
                    const int ck_b = (int)((rnd >> 24) % (uint32_t)max(rb, 1));
                    auto sums = [&](int b, float ww, int64_t at, int p) {
                        red_add4(cube4 + at, ww * v[p][0], ww * v[p][1], ww * v[p][2], ww * v[p][3]);
                        ++n_red;
                        if (service && b == ck_b && p == (int)(((rnd >> 20) + (uint32_t)lane) % P)) {
                            flush_ckpt();
                            ck_took = atomicExch(cube4 + at, make_float4(0.f, 0.f, 0.f, 0.f));
                            ck_dst = a.cube_master + 4 * at;
                            ++n_red;
                        }
                    };
                    for (int b = 0; on && b < rb; ++b) {
                        const float ww = b == 0 ? r0 : b == 1 ? r1 : far_bin_weight(a.chd + kt, b);
                        const int64_t e2 = (int64_t)rc * cell_entries + (int64_t)(rj + b) * npol_c;
                        if (!pairs) {
#pragma unroll
                            for (int p = 0; p < P; ++p) {
                                if (plane[p] < 0 || rn[p] == 0) continue;
                                sums(b, ww, e2 + plane[p], p);
                                atomicAdd(a.count + e2 + plane[p], rn[p]);
                                ++n_red;
                            }
                            continue;
                        }
#pragma unroll
                        for (int p = 0; p < P; ++p) {
                            if (plane[p] < 0 || rn[p] == 0) continue;
                            sums(b, ww, e2 + plane[p], p);
                            if (!(P >= 2 && pk[p / 2])) {
                                atomicAdd(a.count + e2 + plane[p], rn[p]);
                                ++n_red;
                            }
                        }
#pragma unroll
                        for (int k = 0; k < (P >= 2 ? P / 2 : 0); ++k) {
                            if (!pk[k] || (rn[2 * k] | rn[2 * k + 1]) == 0) continue;
                            atomicAdd(reinterpret_cast<unsigned long long *>(a.count + e2 + plane[2 * k]),
                                      (unsigned long long)rn[2 * k] | ((unsigned long long)rn[2 * k + 1] << 32));
                            ++n_red;
                        }
                    }
                }
                __syncwarp();
            };

            constexpr int RB_ = (int)sizeof(RowRec), AHEAD = 2 * (NG - 1) * RB_ + 8;   // 8: RowRec::row
            uint32_t rp = smem_addr(S.rec);
            uint32_t ro = 0, rf = 2 * RS * (NG - 1);   // ring bytes of the pair processed, of the one fetched
            // one row's contribution: phasor, weights, flags and values
            auto add = [&](float2 ph, ulonglong2 W, uint32_t F, const uint64_t (&V)[P]) {
                const uint64_t cc = pack2(ph.x, ph.x), ss = pack2(ph.y, ph.y);
                if constexpr (P == 4) {
                    const float2 wa = unpack2(W.x), wb = unpack2(W.y);
                    const float Wp[4] = {wa.x, wa.y, wb.x, wb.y};
#pragma unroll
                    for (int p = 0; p < P; ++p) {
                        const float2 x = unpack2(V[p]);
                        add_value(accC[p], accS[p], accA[p], accW[p], cnt[p], V[p], pack2(x.x * Wp[p], x.y * Wp[p]), Wp[p],
                                  cc, ss, F & (0xffu << (8 * p)));
                    }
                } else {
                    add_value(accC[0], accS[0], accA[0], accW[0], cnt[0], V[0], mul2(V[0], W.x), unpack2(W.x).x, cc, ss,
                              F & 0xffu);
                    if constexpr (P == 2)
                        add_value(accC[1], accS[1], accA[1], accW[1], cnt[1], V[1], mul2(V[1], W.y), unpack2(W.y).x, cc, ss,
                                  F & 0xff00u);
                }
            };
            // rows two at a time
            constexpr int END = P == 4 ? 1 : 0;   // four pols: row n too
#pragma unroll 1
            for (int b0 = 0; b0 < n + END; b0 += 32) {
                // bit r: row b0 + r may change a lane's cell (or lies past the end)
                uint32_t brk;
                {
                    const int r = b0 + lane;
                    bool b = r >= n;
                    if (r > 0 && r < n) {
                        const int2 c1 = cb[r], c0 = cb[r - 1];
                        b = c1.x != c0.x || c1.y != c0.y || c1.y == CC_MIXED;
                    }
                    brk = __reduce_or_sync(0xffffffffu, b ? 1u << lane : 0u);
                }
                const int m = min(n + END - b0, 32);
#pragma unroll 1
                for (int r = 0; r < m; r += 2) {
                    if constexpr (LB >= 32) __syncwarp();   // every lane is done with the rows refilled next
                    fetch(rf, lds32<AHEAD>(rp));
                    fetch(rf + RS, lds32<AHEAD + RB_>(rp));
                    cp_async_commit();
                    cp_async_wait<NG - 1>();
                    if constexpr (LB >= 32) __syncwarp();   // the rows' pieces were copied by other lanes
                    const uint32_t b2 = (brk >> r) & 3u;
                    // both rows' phasors and values (independent work)
                    float2 ph[2];
                    uint64_t V[2][P];
                    ulonglong2 W[2];
                    uint32_t F[2];
                    auto both = [&]() {
                        const float2 t0 = unpack2(lds64<0>(rp)), t1 = unpack2(lds64<RB_>(rp));
                        ph[0] = shift_phasor(t0.x, t0.y, nh, nl);
                        ph[1] = shift_phasor(t1.x, t1.y, nh, nl);
                        VA::template decode<0>(vis_at + ro, vscale, V[0]);
                        VA::template decode<(int)RS>(vis_at + ro, vscale, V[1]);
                        if (folds) {
                            conjugate(V[0], lds32<12>(rp));
                            conjugate(V[1], lds32<RB_ + 12>(rp));
                        }
                        W[0] = lds128<16>(rp);
                        W[1] = lds128<RB_ + 16>(rp);
                        F[0] = flag_bytes<P, 0>(flag_at + ro);
                        F[1] = flag_bytes<P, (int)RS>(flag_at + ro);
                    };
                    if constexpr (P < 4) {
                        both();
                        if (b2 == 0u) {
                            add(ph[0], W[0], F[0], V[0]);
                            add(ph[1], W[1], F[1], V[1]);
                        } else {
                            const int i = b0 + r;
                            if (b2 & 1u) next_cell(lane_cell(i));
                            add(ph[0], W[0], F[0], V[0]);
                            if (i + 1 < n) {
                                if (b2 & 2u) next_cell(lane_cell(i + 1));
                                add(ph[1], W[1], F[1], V[1]);
                            }
                            while (count >= 32u) drain();
                        }
                    } else if (b2 == 0u) {
                        both();
                        add(ph[0], W[0], F[0], V[0]);
                        add(ph[1], W[1], F[1], V[1]);
                    } else {
                        // four pols: the rows one by one in a loop, so that the code
                        // that ends runs is there once (a copy per row of the pair
                        // overflows the instruction cache: 14.4 -> 21 ms on the
                        // four-pol windows of an archive stack); row n ends the open runs
                        uint32_t rq = rp, rv = ro;
#pragma unroll 1
                        for (int i = b0 + r, d = 0; d < 2; ++d, ++i, rq += RB_, rv += RS) {
                            const float2 t = unpack2(lds64<0>(rq));
                            const float2 p1 = shift_phasor(t.x, t.y, nh, nl);
                            VA::template decode<0>(vis_at + rv, vscale, V[0]);
                            if (folds) conjugate(V[0], lds32<12>(rq));
                            if ((b2 >> d) & 1u) {
                                const bool end = i >= n;
                                next_cell(end ? NO_RUN : lane_cell(i));
                                while (count >= 32u || (end && count != 0u)) drain();
                                if (end) break;
                            }
                            add(p1, lds128<16>(rq), flag_bytes<P, 0>(flag_at + rv), V[0]);
                        }
                    }
                    rp += 2 * RB_;
                    rf = ro;
                    ro = ro == 2 * RS * (NG - 1) ? 0u : ro + 2 * RS;
                }
            }
            cp_async_wait<0>();
            __syncwarp();
            if constexpr (P < 4) {
                next_cell(NO_RUN);   // the runs still open (room: at most 31 wait)
                while (count != 0u) drain();
            }
        }
        if (__any_sync(0xffffffffu, (n_read | n_ok | n_duv | n_red) >= 0x40000000u)) flush_counters();
    }

    flush_ckpt();
    // counters (the visibilities read are also counted on the host from the
    // channel tables)
    flush_counters();
}

// --------------------------------------------------------------- launchers

static int sm_count()
{
    static int n = 0;
    if (n == 0) {
        int dev = 0;
        cudaGetDevice(&dev);
        cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev);
        if (n <= 0) n = 1;
    }
    return n;
}

template <int P, int VT, int NG>
static cudaError_t launch_persistent(const RunArgs &a, int wpc, cudaStream_t st)
{
    const int rb = a.so.rows_per_item;
    if (rb < 1 || rb > RB_MAX || a.cw < 32 || a.cw > 128) return cudaErrorInvalidValue;
    static int smem_max = 0;
    if (smem_max == 0) {
        int dev = 0;
        cudaGetDevice(&dev);
        cudaDeviceGetAttribute(&smem_max, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
    }
    // fewer warps per block when their staging buffers would not fit
    auto kern = stack_mixed<P, VT, NG>;
    const size_t wsm = warp_smem_bytes<P, VT, NG>(rb);
    if (wpc * 32 > KMAX_THREADS) wpc = KMAX_THREADS / 32;
    while (wpc > 1 && (size_t)wpc * wsm > (size_t)smem_max) wpc >>= 1;
    const size_t smem = (size_t)wpc * wsm;
    if (smem > (size_t)smem_max) return cudaErrorInvalidValue;
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    int per_sm = 0;
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, wpc * 32, smem);
    if (e != cudaSuccess) return e;
    if (per_sm < 1) per_sm = 1;
    kern<<<per_sm * sm_count(), wpc * 32, smem, st>>>(a);
    return cudaGetLastError();
}

// Rows of visibilities in flight per warp besides the two being processed
// (prefetch_rows): 2, 4 or 8.
template <int P, int VT>
static cudaError_t launch_mixed_p(const RunArgs &a, int pf, int wpc, cudaStream_t st)
{
    if (pf >= 8) return launch_persistent<P, VT, 5>(a, wpc, st);
    if (pf >= 4) return launch_persistent<P, VT, 3>(a, wpc, st);
    return launch_persistent<P, VT, 2>(a, wpc, st);
}

template <int VT>
static cudaError_t launch_mixed_vt(const RunArgs &a, int pf, int npol, int wpc, cudaStream_t st)
{
    switch (npol) {
    case 1: return launch_mixed_p<1, VT>(a, pf, wpc, st);
    case 2: return launch_mixed_p<2, VT>(a, pf, wpc, st);
    case 4: return launch_mixed_p<4, VT>(a, pf, wpc, st);
    default: return cudaErrorInvalidValue;
    }
}

// One visibility type's launchers (vista_stack_<type>.cu).
cudaError_t launch_mixed_c64(const RunArgs &a, int pf, int npol, int wpc, cudaStream_t st);
cudaError_t launch_mixed_c128(const RunArgs &a, int pf, int npol, int wpc, cudaStream_t st);
cudaError_t launch_mixed_f16(const RunArgs &a, int pf, int npol, int wpc, cudaStream_t st);
cudaError_t launch_mixed_bf16(const RunArgs &a, int pf, int npol, int wpc, cudaStream_t st);

}  // namespace vista
