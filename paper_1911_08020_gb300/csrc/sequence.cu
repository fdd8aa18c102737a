// sequence.cu -- T steps of an LSTM or GRU cell on a DARB gate matrix in one
// persistent, cooperative launch (the RNNs of Sec. 4.1 run many steps per
// input; each step is the fused step of darb_lstm_step / darb_gru_step).
//
// The batch columns are cut into tiles of bt <= 32 columns, and the CTAs into
// column groups, each of which runs the recurrence of its own tiles: columns
// are independent, so a group exchanges h only among its own CTAs, stages only
// its own columns of it, and has a barrier of its own.  Within a group every CTA owns a contiguous range
// of hidden units and all gate rows of those units (LSTM rows u, H+u, 2H+u,
// 3H+u; GRU rows u, H+u, 2H+u), so the cell of a unit needs nothing from
// another CTA.  In the prologue a CTA decodes its rows once into shared memory
// as packed (value, staged row) words and keeps them there for the whole
// sequence, so W_darb leaves HBM/L2 once instead of once per step.
//
// Per step and tile a CTA copies h_{t-1} (and x_t, unless the x parts of all
// steps were one product up front) into shared memory and forms its gate
// sums.  h_t goes to h_seq and to an exchange buffer laid out as the staged
// tile is ([row][bt], two buffers by step parity), so that staging is a few
// 1-D bulk copies whatever the batch's width and alignment.  A lane multiplies 4 columns (a
// 16-byte load of the staged row its kept weight selects), bt / 4 lanes share
// a weight, and the 128 / bt subgroups of a warp take the weights of a row in
// turn; their sums meet in a shuffle reduction that leaves each lane one
// column.  The owning CTA applies the cell.  Steps are separated by a barrier
// over the group's CTAs (arrival counter in global memory) or, where a tile of
// h is small, by the values of h themselves, which carry the number of their
// step; both are spun on with a 1 s limit (on expiry the kernel records a
// timeout, raises an abort flag that ends every other CTA's wait, and
// returns).  The launch is cooperative, so all CTAs are resident and no wait
// can starve.  No CTA touches another
// CTA's shared memory, and no CTA leaves while a copy it issued may still be
// landing.
//
// What bounds a step (cycle stamps, 6000 x 3000 bf16 at batch 20, tiles of 32,
// ~13000 cycles): the gather and its reductions 5900, the barrier 2700,
// staging 2500, the cell 1800.  One column group instead of one a tile stages
// every column in every CTA: GRU 3072 x 2048 at batch 64 took 11.0 against 8.7
// us a step.  Against one lane a column, tensor-map staging and all CTAs in one
// barrier, whole calls went from 3131 to 1491 us (that GRU, 200 steps), 507 to
// 325 (the LSTM above, 35 steps), 520 to 307 (LSTM 4096 x 1280 fp32, batch 1,
// 100 steps), and 2592 to 545 where the batch is no multiple of 4 (GRU 2100 x
// 1000, batch 37, 100 steps).
#include "darb_internal.h"
#include "kernels_common.cuh"
#include "launch.cuh"
#include "rnn_epilogue.cuh"
#include "sequence_rows.h"
#include "tma.cuh"

#include <algorithm>
#include <cstdlib>
#include <vector>

namespace darb {
namespace seq {

constexpr int kThreads = 512;
constexpr int kSeqWarps = kThreads / 32;
constexpr int kMaxCtas = 256;
constexpr size_t kSmemCap = 226 * 1024 + 512;   // dynamic shared memory, below the 227 KB opt-in with room for the static part
constexpr int kMaxLbt = 5;                // batch tiles of at most 2^5 columns
constexpr size_t kCellOnChip = 16 * 1024; // LSTM cell state kept in shared memory up to this size
constexpr int kBarWords = 32;             // words between the barrier counters of two groups (128 bytes)
constexpr size_t kTaggedBytes = 32 * 1024;  // h tiles up to this size are exchanged with tags, without barriers
constexpr int kCopies = 8;                // bulk copies a staged tile is cut into, at most

struct Ranges {
    int32_t start[kMaxCtas + 1];   // CTA q of a group owns hidden units [start[q], start[q+1])
};

// Where x_t comes from.
constexpr int kXNone = 0;    // its products are precomputed (gx)
constexpr int kXBulk = 1;    // tile-major rows (x_tiles), bulk copies
constexpr int kXPlain = 2;   // the caller's x, plain loads (there is no room for its tile-major copy)

struct SeqArgs {
    int I, H, T;
    int ngroups;            // column groups; CTA i is CTA i / ngroups of group i % ngroups
    int ntiles;             // batch tiles; group g runs tiles g, g + ngroups, ...
    int tpg;                // tiles of a group, at most
    int piece;              // kept weights per work item, at most
    int c_on_chip;          // LSTM: cell state in shared memory
    int x_mode;             // kX*
    int tagged;             // h is exchanged as (value, tag) pairs, without barriers
    // staged input rows: x_t at [0, irows), h_{t-1} from row irows on (hrows of
    // them), both rounded up to 4 rows; a zero row at irows + hrows
    int irows, hrows;
    int64_t B;
    const float *gx;        // x parts of the gate sums of every step, rows x ldgx (row r, step t, column b
                            // at r * ldgx + t * B + b), or nullptr: x_t is staged with h_{t-1} instead
    int64_t ldgx;
    const float *x;         // T x I x B (kXPlain)
    const float *x_tiles;   // T x ntiles x irows x bt (kXBulk)
    const float *c0;        // H x B (LSTM)
    const float *bias;      // LSTM [4H] or nullptr
    const float *b_ih;      // GRU [3H] or nullptr
    const float *b_hh;      // GRU [3H] or nullptr
    float *h_seq;           // T x H x B
    float *c_seq;           // T x H x B or nullptr (LSTM)
    float *c_state;         // H x B: the running cell state when it is not on chip (LSTM)
    float *c_last;          // H x B or nullptr (LSTM)
    // the exchanged h_t, [t & 1][ntiles][hrows][bt]; h0 in buffer 1 at launch.
    // Tagged: 8-byte pairs of a value and the number of the step that reads it,
    // plus 1; at launch 1 with h0, 0 in buffer 0 and ~0 in rows past H
    float *h_x;
    unsigned *bar;          // arrival counters of the groups, kBarWords apart, zero at launch
    int *abort_flag;        // zero at launch
    int32_t *status;
    unsigned long long barrier_ns;   // time limit of a wait for another CTA (kWaitLimitNs unless a test shortens it)
    int skip_cta;           // test hook: this CTA does not arrive, or publish, after the first step (-1: none)
};

// Byte offsets of the regions of a CTA's dynamic shared memory.
struct SmemPlan {
    uint32_t w_off, rowptr_off, mid_off, rowitem_off, item_off, bias_off, c_off, gx_off, in_off, part_off, total;
    int items_cap;
};

inline SmemPlan smem_plan(int64_t kept_cap, int rows_cap, int items_cap, int units_cap, bool bf16, bool gru,
                          int in_rows, int bt, int tpg, bool c_on_chip, bool pre) {
    SmemPlan p{};
    p.items_cap = items_cap;
    size_t o = 0;
    auto take = [&](size_t bytes) {
        const size_t at = o;
        o = (o + bytes + 15) / 16 * 16;
        return static_cast<uint32_t>(std::min<size_t>(at, UINT32_MAX));
    };
    p.w_off = take(size_t(kept_cap) * (bf16 ? 4 : 8));
    p.rowptr_off = take(size_t(rows_cap + 1) * 4);
    p.mid_off = take(size_t(rows_cap) * 4);
    p.rowitem_off = take(size_t(rows_cap + 1) * 4);
    p.item_off = take(size_t(items_cap) * 16);
    p.bias_off = take(size_t(rows_cap) * 2 * 4);
    p.c_off = take(c_on_chip ? size_t(units_cap) * size_t(tpg) * bt * 4 : 0);
    p.gx_off = take(pre ? size_t(rows_cap) * bt * 4 : 0);
    p.in_off = take(size_t(in_rows) * bt * 4 + 128);   // rounded up to 128 bytes in the kernel
    p.part_off = take(size_t(gru ? 2 : 1) * items_cap * bt * 4);
    p.total = static_cast<uint32_t>(std::min<size_t>(o, UINT32_MAX));
    return p;
}

// Kept weight p of the CTA: its value and the index (row * bt) of the first
// element of the staged input row it multiplies.
template <bool BF16> struct Packed;
template <> struct Packed<true> {   // bf16 bits << 16 | index
    using T = uint32_t;
    static __device__ __forceinline__ T make(uint32_t bits, uint32_t col) { return (bits << 16) | col; }
    static __device__ __forceinline__ float val(T w) { return __uint_as_float(w & 0xFFFF0000u); }
    static __device__ __forceinline__ uint32_t col(T w) { return w & 0xFFFFu; }
};
template <> struct Packed<false> {  // fp32 bits, index
    using T = uint2;
    static __device__ __forceinline__ T make(uint32_t bits, uint32_t col) { return make_uint2(bits, col); }
    static __device__ __forceinline__ float val(T w) { return __uint_as_float(w.x); }
    static __device__ __forceinline__ uint32_t col(T w) { return w.y; }
};

// On-chip layout of one row's kept weights: an x region, then an h region,
// each padded with zero weights (pointing at the zero row of the staged input)
// to a multiple of 4 so that a lane loads 4 weights at once.  Block jmid = I/m
// is the only block that can hold columns on both sides of I.
//   x parts precomputed: h region only, blocks jmid.. (an x weight of block
//     jmid becomes a zero weight);
//   GRU otherwise: blocks 0..jmid in the x region (block jmid there only if
//     its weight multiplies x), blocks jmid.. in the h region;
//   LSTM otherwise: one region of all blocks.
__host__ __device__ inline int round4(int v) { return (v + 3) & ~3; }
__host__ __device__ inline void row_regions(int n, int m, int I, bool pre, bool gru, int &xr, int &hr) {
    const int jmid = I / m;
    if (pre) {
        xr = 0;
        hr = round4(n - jmid);
    } else if (gru) {
        xr = round4(jmid + 1);
        hr = round4(n - jmid);
    } else {
        xr = round4(n);
        hr = 0;
    }
}

// How the lanes of a warp share a tile of 2^LBT columns: a lane multiplies V
// columns of a weight, L lanes share the weight, S subgroups of L lanes take
// the weights of a row in turn, KW consecutive ones at a time (one load).
template <int LBT>
struct Lanes {
    static constexpr int BT = 1 << LBT;
    static constexpr int V = BT < 4 ? BT : 4;
    static constexpr int L = BT / V;
    static constexpr int S = 32 / L;
    static constexpr int KW = S <= 4 ? 4 : S <= 8 ? 2 : 1;
};

template <class P, int KW>
__device__ __forceinline__ void load_weights(const typename P::T *p, typename P::T (&w)[KW]) {
    if constexpr (sizeof(typename P::T) == 4) {
        if constexpr (KW == 4) {
            const uint4 q = *reinterpret_cast<const uint4 *>(p);
            w[0] = q.x; w[1] = q.y; w[2] = q.z; w[3] = q.w;
        } else if constexpr (KW == 2) {
            const uint2 q = *reinterpret_cast<const uint2 *>(p);
            w[0] = q.x; w[1] = q.y;
        } else {
            w[0] = *p;
        }
    } else {
        if constexpr (KW == 1) {
            w[0] = *p;
        } else {
#pragma unroll
            for (int i = 0; i < KW; i += 2) {
                const uint4 q = *reinterpret_cast<const uint4 *>(p + i);
                w[i] = make_uint2(q.x, q.y);
                w[i + 1] = make_uint2(q.z, q.w);
            }
        }
    }
}

// Sums over kept weights [pa, pb) of the CTA (multiples of 4) against the
// tile: subgroup `sub` takes every S-th run of KW weights from pa + KW sub,
// s_inc = staged tile + the lane's first column.  The lane's V columns, each
// from U * KW accumulators.
template <class P, int LBT>
__device__ __forceinline__ void dot_range(const typename P::T *s_w, const float *s_inc, int pa, int pb, int sub,
                                          float (&acc)[Lanes<LBT>::V]) {
    using G = Lanes<LBT>;
    constexpr int V = G::V, KW = G::KW, U = KW < 4 ? 2 : 1, A = U * KW, kStep = KW * G::S;
    float4 s[A];   // (V < 4: the first V of each)
#pragma unroll
    for (int i = 0; i < A; ++i) s[i] = make_float4(0.f, 0.f, 0.f, 0.f);
    // (not unrolled further: a step runs through its code once, and the fetch of
    // more of it costs more than the overlap gives; by 2: 1 to 5% slower)
#pragma unroll 1
    for (int p = pa + KW * sub; p < pb; p += U * kStep) {
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const int q = p + u * kStep;
            if (u > 0 && q >= pb) continue;
            typename P::T w[KW];
            load_weights<P, KW>(s_w + q, w);
#pragma unroll
            for (int i = 0; i < KW; ++i) {
                const float *x = s_inc + P::col(w[i]);
                const float v = P::val(w[i]);
                float4 &d = s[u * KW + i];
                if constexpr (V == 4) {
                    fma4(d, v, *reinterpret_cast<const float4 *>(x));
                } else if constexpr (V == 2) {
                    const float2 x2 = *reinterpret_cast<const float2 *>(x);
                    d.x = fmaf(v, x2.x, d.x);
                    d.y = fmaf(v, x2.y, d.y);
                } else {
                    d.x = fmaf(v, *x, d.x);
                }
            }
        }
    }
#pragma unroll
    for (int h = A / 2; h >= 1; h /= 2)
#pragma unroll
        for (int i = 0; i < h; ++i) {
            s[i].x += s[i + h].x;
            if constexpr (V > 1) s[i].y += s[i + h].y;
            if constexpr (V > 2) s[i].z += s[i + h].z;
            if constexpr (V > 2) s[i].w += s[i + h].w;
        }
    acc[0] = s[0].x;
    if constexpr (V > 1) acc[1] = s[0].y;
    if constexpr (V > 2) acc[2] = s[0].z;
    if constexpr (V > 2) acc[3] = s[0].w;
}

// Add the subgroups' sums of an item and store them at part[0 .. BT): the
// first exchanges halve the columns a lane keeps (from V to 1), the rest add
// whole; a fixed order, so deterministic.
template <int LBT>
__device__ __forceinline__ void reduce_store(float (&acc)[Lanes<LBT>::V], int lane, float *part) {
    using G = Lanes<LBT>;
    constexpr unsigned kAll = 0xFFFFFFFFu;
    int col = (lane & (G::L - 1)) * G::V;
    float v;
    int o = 16;   // the lane bits from L up to 16 number the subgroups
    if constexpr (G::V == 4) {
        const bool up = lane & 16;
        const float s0 = up ? acc[0] : acc[2], s1 = up ? acc[1] : acc[3];
        const float k0 = (up ? acc[2] : acc[0]) + __shfl_xor_sync(kAll, s0, 16);
        const float k1 = (up ? acc[3] : acc[1]) + __shfl_xor_sync(kAll, s1, 16);
        const bool up8 = lane & 8;
        v = (up8 ? k1 : k0) + __shfl_xor_sync(kAll, up8 ? k0 : k1, 8);
        col += (up ? 2 : 0) + (up8 ? 1 : 0);
        o = 4;
    } else if constexpr (G::V == 2) {
        const bool up = lane & 16;
        v = (up ? acc[1] : acc[0]) + __shfl_xor_sync(kAll, up ? acc[0] : acc[1], 16);
        col += up ? 1 : 0;
        o = 8;
    } else {
        v = acc[0];
    }
    const int rest = 2 * o - G::L;   // lane bits still to add over: L .. o
#pragma unroll
    for (int b = o; b >= G::L; b >>= 1) v += __shfl_xor_sync(kAll, v, b);
    if ((lane & rest) == 0) part[col] = v;
}

// A warp's wait for the arrivals of its group; false if it gave up or another
// CTA did.  The CTA barrier before an arrival orders every thread's
// h_t stores before it; the arrival is a release reduction on the counter (no
// return trip, no separate fence).  An acquire that reads the final count
// synchronises with every arrival (each is a read-modify-write in the
// counter's release sequence).
__device__ __forceinline__ bool wait_arrivals(const SeqArgs &a, const unsigned *bar, unsigned target) {
    const unsigned long long t0 = global_timer_ns();
    for (unsigned spin = 0;; ++spin) {
        unsigned v;
        asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(bar) : "memory");
        if (v >= target) return true;
        if ((spin & 63) == 63) {
            if (*reinterpret_cast<volatile int *>(a.abort_flag)) return false;
            if (global_timer_ns() - t0 > a.barrier_ns) {
                atomicExch(a.abort_flag, 1);
                atomicOr(a.status, kStatusTimeout);
                return false;
            }
            __nanosleep(32);
        }
    }
}

// One (value, tag) pair of an exchanged h: a single 8-byte access, so that the
// tag vouches for the value next to it without any ordering.
__device__ __forceinline__ void put_tagged(float *h_x, int64_t i, float v, uint32_t tag) {
    const uint64_t w = (uint64_t(tag) << 32) | __float_as_uint(v);
    asm volatile("st.relaxed.gpu.global.u64 [%0], %1;" ::"l"(reinterpret_cast<uint64_t *>(h_x) + i), "l"(w) : "memory");
}
__device__ __forceinline__ ulonglong2 get_tagged2(const uint64_t *p) {
    ulonglong2 v;
    asm volatile("ld.relaxed.gpu.global.v2.u64 {%0, %1}, [%2];" : "=l"(v.x), "=l"(v.y) : "l"(p) : "memory");
    return v;
}

// Stage n2 pairs of tagged elements, waiting for each to carry `tag` (or a
// later one); false if this thread gave up or another CTA did.  A buffer is
// written again two steps later, when every CTA of the group has published the
// step in between, i.e. has read this one.  U: loads a thread has in flight.
template <int U>
__device__ __forceinline__ bool stage_tagged(const SeqArgs &a, const float *h_x, int64_t first, int n2, uint32_t tag,
                                             float *dst) {
    const uint64_t *src = reinterpret_cast<const uint64_t *>(h_x) + first;
    unsigned long long t0 = 0;
    unsigned spin = 0;
    for (int i0 = threadIdx.x; i0 < n2; i0 += kThreads * U) {
        ulonglong2 v[U];
        unsigned wanted = 0;   // bit u: element u has not come yet
#pragma unroll
        for (int u = 0; u < U; ++u)
            if (i0 + u * kThreads < n2) wanted |= 1u << u;
        const unsigned all = wanted;
        while (true) {   // all that is missing is asked for again at once
#pragma unroll
            for (int u = 0; u < U; ++u)
                if (wanted >> u & 1) v[u] = get_tagged2(src + 2 * (i0 + u * kThreads));
#pragma unroll
            for (int u = 0; u < U; ++u)
                if ((wanted >> u & 1) && uint32_t(v[u].x >> 32) >= tag && uint32_t(v[u].y >> 32) >= tag)
                    wanted &= ~(1u << u);
            if (wanted == 0) break;
            if ((++spin & 63) == 0) {
                if (*reinterpret_cast<volatile int *>(a.abort_flag)) return false;
                const unsigned long long now = global_timer_ns();
                if (t0 == 0) t0 = now;
                else if (now - t0 > a.barrier_ns) {
                    atomicExch(a.abort_flag, 1);
                    atomicOr(a.status, kStatusTimeout);
                    return false;
                }
            }
        }
#pragma unroll
        for (int u = 0; u < U; ++u)
            if (all >> u & 1)
                reinterpret_cast<float2 *>(dst)[i0 + u * kThreads] =
                    make_float2(__uint_as_float(uint32_t(v[u].x)), __uint_as_float(uint32_t(v[u].y)));
    }
    return true;
}

// A tile of `bytes` (a multiple of 16): one warp, each of its first kCopies
// lanes a bulk copy that completes on `bar` (one thread issuing all of them
// took 1400 cycles of a step).  `ready` is called by the whole warp between
// arming `bar` and the copies: what only has to be done is done before it.
template <class Ready>
__device__ __forceinline__ void copy_tile(int lane, float *dst, const float *src, uint32_t bytes, uint64_t *bar,
                                          Ready ready) {
    // every thread of this CTA is done with the previous tile (the barrier
    // that ended it); order those reads before the copies
    fence_proxy_async_smem();
    if (lane == 0) mbar_arrive_expect_tx(bar, bytes);
    const uint32_t each = (bytes / kCopies + 127) & ~127u, at = uint32_t(lane) * each;
    const bool has = lane < kCopies && at < bytes;
    const uint32_t size = lane == kCopies - 1 || bytes - at < each ? bytes - at : each;
    char *d = reinterpret_cast<char *>(dst) + at;
    const char *s = reinterpret_cast<const char *>(src) + at;
    __syncwarp();
    ready();
    fence_proxy_async_global();   // what other CTAs published by generic stores, too
    if (has) bulk_g2s(d, s, size, bar);
}

template <bool BF16, int MODE, int LBT, bool TAGGED>
__global__ void __launch_bounds__(kThreads, 1)
seq_kernel(Format f, SeqArgs a, Ranges rg, SmemPlan sp) {
    using G = Lanes<LBT>;
    constexpr int kGates = MODE == kModeLstm ? 4 : 3;
    constexpr bool kGru = MODE == kModeGru;
    constexpr int bt = G::BT;
    using P = Packed<BF16>;
    using PT = typename P::T;
    extern __shared__ __align__(16) unsigned char sm[];
    __shared__ int s_nitems, s_next, s_fail;
    __shared__ __align__(8) uint64_t s_hfull, s_xfull;   // the staged h / x rows have landed
    PT *s_w = reinterpret_cast<PT *>(sm + sp.w_off);
    int *s_rowptr = reinterpret_cast<int *>(sm + sp.rowptr_off);
    int *s_mid = reinterpret_cast<int *>(sm + sp.mid_off);          // GRU: first kept weight of a row on h
    uint32_t *s_rowitem = reinterpret_cast<uint32_t *>(sm + sp.rowitem_off);   // a row's first item | their number << 16 (>= 1)
    int4 *s_item = reinterpret_cast<int4 *>(sm + sp.item_off);      // (first, end, number (at first: local row), first on h)
    float *s_bias = reinterpret_cast<float *>(sm + sp.bias_off);    // [R] (GRU: [2R], b_ih then b_hh)
    float *s_c = reinterpret_cast<float *>(sm + sp.c_off);          // [units][tpg * bt] when on chip
    float *s_gx = reinterpret_cast<float *>(sm + sp.gx_off);        // [R][bt]: x parts of this tile
    float *s_in = reinterpret_cast<float *>(                          // [kin + 1][bt], row kin zero
        (reinterpret_cast<uintptr_t>(sm + sp.in_off) + 127) & ~uintptr_t(127));
    float *s_part = reinterpret_cast<float *>(sm + sp.part_off);    // [parts][items][bt]
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int group = int(blockIdx.x) % a.ngroups, member = int(blockIdx.x) / a.ngroups;
    const unsigned members = gridDim.x / unsigned(a.ngroups);
    unsigned *bar = a.bar + group * kBarWords;
    const int u0 = rg.start[member], nu = rg.start[member + 1] - u0;
    const int R = kGates * nu;   // local row q*nu + i is matrix row q*H + u0 + i
    const int I = a.I, H = a.H;
    const int sub = lane / G::L, col = (lane % G::L) * G::V;
    const int64_t B = a.B;
    // with the x parts precomputed only h_{t-1} is staged and only the kept
    // weights of blocks that reach column I are kept on chip (columns shifted by I)
    const bool pre = a.gx != nullptr;
    // GRU without precomputed x parts keeps the x and h sums of each item apart
    const bool split = kGru && !pre;
    const int kin = a.irows + a.hrows;
    auto grow = [&](int lr) { return (lr / nu) * H + u0 + lr % nu; };

    // ---- prologue: row sizes, biases, cell state, the zero row of the staged input
    for (int lr = tid; lr < R; lr += kThreads) {
        const int r = grow(lr);
        const Group &g = f.groups[f.rowloc[r] / kSlots];
        int xr, hr;
        row_regions(g.n, g.m, I, pre, kGru, xr, hr);
        s_rowptr[lr + 1] = xr + hr;
        s_mid[lr] = xr;   // relative until the row pointers exist
        if constexpr (kGru) {
            s_bias[lr] = a.b_ih ? a.b_ih[r] : 0.0f;
            s_bias[R + lr] = a.b_hh ? a.b_hh[r] : 0.0f;
        } else {
            s_bias[lr] = a.bias ? a.bias[r] : 0.0f;
        }
    }
    const int cw = a.tpg << LBT;   // columns of the on-chip cell state
    if constexpr (!kGru)
        if (a.c_on_chip)
            for (int i = tid; i < nu * cw; i += kThreads) {
                const int64_t b = (int64_t(group + (i % cw >> LBT) * a.ngroups) << LBT) + (i & (bt - 1));
                s_c[i] = b < B ? a.c0[int64_t(u0 + i / cw) * B + b] : 0.0f;
            }
    for (int j = tid; j < bt; j += kThreads) s_in[(kin << LBT) + j] = 0.0f;
    if (tid == 0) {
        mbar_init(&s_hfull, 1);
        mbar_init(&s_xfull, 1);
        s_fail = 0;
        fence_mbar_init();
    }
    __syncthreads();
    // row pointers and work items: every row cut into pieces of at most a.piece weights
    if (tid == 0) {
        int p = 0, ni = 0;
        for (int lr = 0; lr < R; ++lr) {
            const int n = s_rowptr[lr + 1];
            s_rowptr[lr] = p;
            s_mid[lr] += p;
            const int first = ni;
            for (int q = 0; q < n; q += a.piece) s_item[ni++] = make_int4(p + q, p + min(n, q + a.piece), lr, 0);
            s_rowitem[lr] = uint32_t(first) | uint32_t(ni - first) << 16;
            p += n;
        }
        s_rowptr[R] = p;
        s_nitems = ni;
    }
    __syncthreads();
    // zero weights everywhere, then every kept weight as (value, staged row)
    for (int p = tid; p < s_rowptr[R]; p += kThreads) s_w[p] = P::make(0u, uint32_t(kin) << LBT);
    __syncthreads();
    for (int lr = warp; lr < R; lr += kSeqWarps) {
        const int loc = f.rowloc[grow(lr)];
        const Group g = f.groups[loc / kSlots];
        const int slot = loc % kSlots;
        const int base = s_rowptr[lr], mid = s_mid[lr];
        const int jmid = I / g.m;
        for (int j = (pre ? jmid : 0) + lane; j < g.n; j += 32) {
            const int64_t rec = int64_t(j / kChunk) * kSlots + slot;
            const int q = j % kChunk;
            uint32_t bits;
            if constexpr (BF16) bits = static_cast<const uint16_t *>(f.vals)[g.val_off + rec * kChunk + q];
            else bits = static_cast<const uint32_t *>(f.vals)[g.val_off + rec * kChunk + q];
            uint32_t o;
            if (g.nib) o = (f.offs[g.off_off + rec] >> (4 * q)) & 15u;
            else o = (f.offs[g.off_off + 2 * rec + (q >> 2)] >> (8 * (q & 3))) & 255u;
            uint32_t c = uint32_t(j) * uint32_t(g.m) + o;
            const bool on_h = c >= uint32_t(I);
            int at;
            if (pre || kGru) at = on_h ? mid + j - jmid : base + j;   // h region from block jmid on
            else at = base + j;
            if (on_h) {
                c = c - uint32_t(I) + uint32_t(a.irows);   // staged row of h
            } else if (pre) {   // an x weight of block jmid: its product is in gx
                bits = 0;
                c = uint32_t(kin);
                at = mid;
            }
            s_w[at] = P::make(bits, c << LBT);   // (kin + 1) * bt floats fit in shared memory: < 2^16
        }
    }
    __syncthreads();
    const int NI = s_nitems;
    if (tid == 0) s_next = kSeqWarps;   // a warp's first item is its own index
    // the items in descending order of their weights, so that the last ones
    // handed out are short; z becomes the item's number (its partial sums)
    for (int i0 = 0; i0 < NI; i0 += kThreads) {
        const int i = i0 + tid;
        int4 it = make_int4(0, 0, 0, 0);
        int rank = 0;
        if (i < NI) {
            it = s_item[i];
            it.w = split ? max(it.x, min(it.y, s_mid[it.z])) : it.y;
            it.z = i;
            const int n = it.y - it.x;
            for (int o = 0; o < NI; ++o) {
                const int2 other = *reinterpret_cast<const int2 *>(s_item + o);
                rank += other.y - other.x > n || (other.y - other.x == n && o < i);
            }
        }
        if (NI > kThreads) break;   // too many to sort in one pass: their order stays
        __syncthreads();
        if (i < NI) s_item[rank] = it;
    }
    if (NI > kThreads)
        for (int i = tid; i < NI; i += kThreads) {
            s_item[i].w = split ? max(s_item[i].x, min(s_item[i].y, s_mid[s_item[i].z])) : s_item[i].y;
            s_item[i].z = i;
        }
    __syncthreads();

    // ---- the steps
    const uint32_t xbytes = uint32_t(a.irows) * bt * 4, hbytes = uint32_t(a.hrows) * bt * 4;
    // x_t of one tile (the last warp): its rows are free once the tile before has been multiplied
    auto copy_x = [&](int t, int tile) {
        copy_tile(lane, s_in, a.x_tiles + (int64_t(t) * a.ntiles + tile) * (int64_t(a.irows) << LBT), xbytes, &s_xfull,
                  [] {});
    };
    const bool xbulk = a.x_mode == kXBulk;
    if (xbulk && warp == kSeqWarps - 1) copy_x(0, group);
    int staged = 0;   // tiles staged so far: the parity of s_hfull and s_xfull
    float *c_run = kGru ? nullptr : (a.c_on_chip ? s_c : a.c_state + int64_t(u0) * B);
    for (int t = 0; t < a.T; ++t) {
        float *ht = a.h_seq + int64_t(t) * H * B + int64_t(u0) * B;
        float *ct = a.c_seq ? a.c_seq + int64_t(t) * H * B + int64_t(u0) * B : nullptr;
        for (int k = 0, tile = group; tile < a.ntiles; ++k, tile += a.ngroups, ++staged) {
            const int64_t b0 = int64_t(tile) << LBT;
            const int nb = static_cast<int>(B - b0 < bt ? B - b0 : bt);
            if (pre)
                for (int i = tid; i < R << LBT; i += kThreads) {
                    const int lr = i >> LBT, j = i & (bt - 1);
                    cp_async4(smem_addr(s_gx + i),
                              a.gx + int64_t(grow(lr)) * a.ldgx + int64_t(t) * B + b0 + (j < nb ? j : 0), j < nb);
                }
            if (a.x_mode == kXPlain)
                for (int i = tid; i < I << LBT; i += kThreads) {
                    const int j = i & (bt - 1);
                    s_in[i] = j < nb ? __ldg(a.x + (int64_t(t) * I + (i >> LBT)) * B + b0 + j) : 0.0f;
                }
            bool ok = true;
            if constexpr (TAGGED) {
                const int64_t first = (int64_t((t + 1) & 1) * a.ntiles + tile) * (int64_t(a.hrows) << LBT);
                const int n2 = a.hrows * bt / 2;   // up to 8 a thread (kTaggedBytes)
                float *dst = s_in + (a.irows << LBT);
                const uint32_t tag = uint32_t(t) + 1u;
                ok = n2 <= kThreads       ? stage_tagged<1>(a, a.h_x, first, n2, tag, dst)
                     : n2 <= 4 * kThreads ? stage_tagged<4>(a, a.h_x, first, n2, tag, dst)
                                          : stage_tagged<8>(a, a.h_x, first, n2, tag, dst);
            } else if (warp == 0) {
                // a wait that gives up sets s_fail; its copies are harmless and let
                // the waiting threads get there
                copy_tile(lane, s_in + (a.irows << LBT),
                          a.h_x + (int64_t((t + 1) & 1) * a.ntiles + tile) * (int64_t(a.hrows) << LBT), hbytes, &s_hfull,
                          [&] {
                              if (k == 0 && t > 0 && !wait_arrivals(a, bar, unsigned(t) * members)) s_fail = 1;
                          });
            }
            if (TAGGED || a.x_mode == kXPlain) __syncthreads();
            if (!TAGGED) ok = mbar_wait(&s_hfull, staged & 1);
            if (xbulk) ok = mbar_wait(&s_xfull, staged & 1) && ok;
            // partial gate sums of the work items, handed out to warps as they come free
            for (int ii = warp; ii < NI;) {
                int next = 0;
                if (lane == 0) next = atomicAdd(&s_next, 1);
                const int4 it = s_item[ii];
                float acc[G::V];
                dot_range<P, LBT>(s_w, s_in + col, it.x, it.w, sub, acc);
                reduce_store<LBT>(acc, lane, s_part + (it.z << LBT));
                if (split) {
                    dot_range<P, LBT>(s_w, s_in + col, it.w, it.y, sub, acc);
                    reduce_store<LBT>(acc, lane, s_part + ((NI + it.z) << LBT));
                }
                ii = __shfl_sync(0xFFFFFFFFu, next, 0);
            }
            if (pre) cp_async_wait_all();
            if (!__syncthreads_and(ok) || s_fail) {
                // a wait gave up: end the other CTAs' waits too.  Copies of this
                // CTA may still land: give them a second bounded wait before it leaves
                if (tid == 0) {
                    atomicOr(a.status, kStatusTimeout);
                    atomicExch(a.abort_flag, 1);
                    if (!TAGGED) mbar_wait(&s_hfull, staged & 1);
                    if (xbulk) mbar_wait(&s_xfull, staged & 1);
                }
                return;
            }
            if (warp == kSeqWarps - 1) {
                if (lane == 0) s_next = kSeqWarps;   // for the next tile; every warp has left the loop
                // the next tile's x rows, while the cell and the barrier run
                const bool more = tile + a.ngroups < a.ntiles;
                if (xbulk && (more || t + 1 < a.T)) copy_x(more ? t : t + 1, more ? tile + a.ngroups : group);
            }
            // the cells of the owned units for these columns
            const int64_t hx0 = ((int64_t(t & 1) * a.ntiles + tile) * a.hrows + u0) * bt;
            auto publish = [&](int i, float v) {
                if (!TAGGED) a.h_x[hx0 + i] = v;
                else if (!(int(blockIdx.x) == a.skip_cta && t == 0)) put_tagged(a.h_x, hx0 + i, v, uint32_t(t) + 2u);
            };
            // partial sums of local row lr: part 0 (everything, or the x part of a
            // split GRU row), part 1 (the h part of a split GRU row)
            auto sum = [&](int lr, int part, int j) {
                const uint32_t it = s_rowitem[lr];
                const float *sp = s_part + (((it & 0xFFFFu) + part * NI) << LBT) + j;
                float v = sp[0];
                for (uint32_t o = 1; o < it >> 16; ++o) v += sp[o << LBT];
                return v;
            };
            for (int i = tid; i < nu << LBT; i += kThreads) {
                const int ui = i >> LBT, j = i & (bt - 1);
                if (j >= nb) {
                    publish(i, 0.0f);
                    continue;
                }
                const int64_t e = int64_t(ui) * B + b0 + j;
                auto xg = [&](int lr) { return pre ? s_gx[(lr << LBT) + j] : 0.0f; };
                if constexpr (MODE == kModeLstm) {
                    auto gate = [&](int lr) { return s_bias[lr] + sum(lr, 0, j) + xg(lr); };
                    const float pi = gate(ui), pf = gate(nu + ui), pg = gate(2 * nu + ui), po = gate(3 * nu + ui);
                    const int64_t ec = a.c_on_chip ? ui * cw + (k << LBT) + j : e;
                    const float cprev = t == 0 && !a.c_on_chip ? a.c0[int64_t(u0) * B + e] : c_run[ec];
                    const float c = sigm(pf) * cprev + sigm(pi) * tanhf(pg);
                    const float hv = sigm(po) * tanhf(c);
                    publish(i, hv);
                    c_run[ec] = c;
                    if (ct) ct[e] = c;
                    ht[e] = hv;
                } else {
                    // x part (b_ih + W_x x) and h part (b_hh + W_h h) of each gate
                    auto gx_ = [&](int lr) { return s_bias[lr] + (pre ? xg(lr) : sum(lr, 0, j)); };
                    auto gh_ = [&](int lr) { return s_bias[R + lr] + sum(lr, split ? 1 : 0, j); };
                    const float rr = sigm(gx_(ui) + gh_(ui));
                    const float zz = sigm(gx_(nu + ui) + gh_(nu + ui));
                    const float nn = tanhf(gx_(2 * nu + ui) + rr * gh_(2 * nu + ui));
                    const float hv = (1.0f - zz) * nn + zz * s_in[((a.irows + u0 + ui) << LBT) + j];
                    publish(i, hv);
                    ht[e] = hv;
                }
            }
            __syncthreads();
        }
        if (!TAGGED && t + 1 < a.T && tid == 0 && !(int(blockIdx.x) == a.skip_cta && t == 0))
            asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(bar) : "memory");
    }
    if constexpr (!kGru)
        if (a.c_on_chip && a.c_last)
            for (int i = tid; i < nu * cw; i += kThreads) {
                const int64_t b = (int64_t(group + (i % cw >> LBT) * a.ngroups) << LBT) + (i & (bt - 1));
                if (b < B) a.c_last[int64_t(u0 + i / cw) * B + b] = s_c[i];
            }
}

// What a call needs in place before seq_kernel: the barrier counters zero, h0
// in the exchange buffer, and x_t of every step as tile-major rows (x_tiles)
// or as the columns of one product input (xall[k][t * B + b] = x[t][k][b]).
// A warp per row of h0 or of an x_t.
__global__ void __launch_bounds__(256) prep_kernel(SeqArgs a, int lbt, const float *h0, float *x_tiles, float *xall,
                                                   int64_t ldxall, int nwords) {
    const int64_t B = a.B;
    const int lane = threadIdx.x & 31;
    for (int i = int(blockIdx.x) * 256 + int(threadIdx.x); i < nwords; i += int(gridDim.x) * 256) a.bar[i] = 0u;
    const int bt = 1 << lbt;
    const int64_t nrows = a.H + (x_tiles || xall ? int64_t(a.T) * a.I : 0);
    if (a.tagged) {   // tags of buffer 0, and of the rows past H in both
        const int64_t n = int64_t(a.ntiles) * a.hrows << lbt;
        for (int64_t i = int64_t(blockIdx.x) * 256 + threadIdx.x; i < n; i += int64_t(gridDim.x) * 256) {
            const bool pad = (i >> lbt) % a.hrows >= a.H;
            reinterpret_cast<uint64_t *>(a.h_x)[i] = pad ? ~uint64_t(0) << 32 : 0;
            if (pad) reinterpret_cast<uint64_t *>(a.h_x)[n + i] = ~uint64_t(0) << 32;
        }
    }
    for (int64_t row = int64_t(blockIdx.x) * 8 + (threadIdx.x >> 5); row < nrows; row += int64_t(gridDim.x) * 8) {
        const PrepRow r = prep_row(row, a.H, a.I);
        const int64_t xrow = row - a.H;
        if (r.of_x && xall != nullptr) {
            for (int64_t b = lane; b < B; b += 32) xall[r.k * ldxall + r.t * B + b] = __ldg(a.x + xrow * B + b);
            continue;
        }
        const float *src = r.of_x ? a.x + xrow * B : h0 + row * B;
        const int nr = r.of_x ? a.irows : a.hrows;   // rows of a tile
        float *dst = (r.of_x ? x_tiles + ((r.t * a.ntiles * nr) << lbt) : a.h_x + ((int64_t(a.ntiles) * nr) << lbt)) +
                     (r.k << lbt);
        if (!r.of_x && a.tagged) {
            uint64_t *d = reinterpret_cast<uint64_t *>(a.h_x) + ((int64_t(a.ntiles) * nr) << lbt) + (r.k << lbt);
            for (int64_t b = lane; b < (int64_t(a.ntiles) << lbt); b += 32)
                d[(((b >> lbt) * nr) << lbt) + (b & (bt - 1))] =
                    uint64_t(1) << 32 | (b < B ? __float_as_uint(__ldg(src + b)) : 0u);
            continue;
        }
        for (int64_t b = lane; b < (int64_t(a.ntiles) << lbt); b += 32)
            dst[(((b >> lbt) * nr) << lbt) + (b & (bt - 1))] = b < B ? __ldg(src + b) : 0.0f;
    }
}

}  // namespace seq

namespace {

// Test hook for the failure path of the waits between CTAs.  With the
// environment variable DARB_TEST_BARRIER_TIMEOUT=1 a launch's waits for another
// CTA give up after 1 ms, and CTA 0 withholds its arrival at the first barrier
// (or, where h is exchanged with tags, its first values): the waits of its
// column group run out, the launch records DARB_ERR_TIMEOUT (read by
// darb_sync_status), raises the abort flag, which ends every wait, and
// ends; a CTA whose copy of x is in flight waits for it first.  The results of
// that call are not valid.  Read on every launch so that a test can set and
// clear it.
void sequence_test_hook(unsigned long long *barrier_ns, int *skip_cta) {
    const char *v = std::getenv("DARB_TEST_BARRIER_TIMEOUT");
    if (v != nullptr && v[0] == '1' && v[1] == '\0') {
        *barrier_ns = 1000000ull;
        *skip_cta = 0;
    }
}

// Contiguous unit ranges over G CTAs with about equal kept weights each.
// Returns the largest weight count and unit count of any CTA.
void split_units(const std::vector<int64_t> &kept, int G, seq::Ranges &rg, int64_t &kept_cap, int &units_cap) {
    const int H = static_cast<int>(kept.size());
    int64_t total = 0;
    for (int64_t k : kept) total += k;
    kept_cap = 0;
    units_cap = 0;
    int u = 0;
    int64_t acc = 0;   // weights of units [0, u)
    for (int q = 0; q < G; ++q) {
        rg.start[q] = u;
        const int64_t target = q + 1 == G ? total : total * (q + 1) / G;
        const int last = H - (G - 1 - q);   // leave one unit for every later CTA
        int64_t mine = 0;
        while (u < last && (acc + mine < target || mine == 0)) mine += kept[static_cast<size_t>(u++)];
        acc += mine;
        kept_cap = std::max(kept_cap, mine);
        units_cap = std::max(units_cap, u - rg.start[q]);
    }
    rg.start[G] = H;
}


// A tile width and a number of column groups to try, and what a step is
// expected to take (ns).
struct Shape {
    int lbt, ngroups, tpg;
    double ns;
};

}  // namespace

// Whether the x parts of all steps go through one darb_spmm-style product up
// front: when x_t is a large share of the stacked input the per-step staging
// and gate sums shrink by that share; the product has T*B columns.
inline bool precompute_x(int64_t T, int64_t I, int64_t H, int64_t B, size_t ws_bytes) {
    return I > 0 && 2 * I >= H && T * B >= 64 && T * B <= (int64_t(1) << 19) && ws_bytes <= (size_t(1) << 30);
}

template <bool BF16, int MODE, bool TAGGED>
static auto seq_entry(int lbt) {
    using namespace seq;
    switch (lbt) {
        case 0: return seq_kernel<BF16, MODE, 0, TAGGED>;
        case 1: return seq_kernel<BF16, MODE, 1, TAGGED>;
        case 2: return seq_kernel<BF16, MODE, 2, TAGGED>;
        case 3: return seq_kernel<BF16, MODE, 3, TAGGED>;
        case 4: return seq_kernel<BF16, MODE, 4, TAGGED>;
        default: return seq_kernel<BF16, MODE, 5, TAGGED>;
    }
}

template <bool BF16, int MODE>
static cudaError_t launch_seq_t(const Format &f, const int32_t *row_m, seq::SeqArgs a, const float *h0, float *c_last,
                                cudaStream_t stream) {
    using namespace seq;
    constexpr int kGates = MODE == kModeLstm ? 4 : 3;
    constexpr bool kGru = MODE == kModeGru;
    const int H = a.H, I = a.I;
    const int64_t B = a.B, T = a.T, rows = f.rows;
    if (f.cols > 65535) return cudaErrorNotSupported;   // columns are kept in 16 bits
    auto up = [](size_t v) { return (v + 255) / 256 * 256; };
    const int64_t ldx = (T * B + 3) / 4 * 4;   // 16-byte rows for the product's loads
    const size_t pre_bytes = up(size_t(I + H) * ldx * 4) + up(size_t(rows) * ldx * 4);
    const bool pre = precompute_x(T, I, H, B, pre_bytes);
    // kept weights on chip of a row of block size m: all, or those of the blocks
    // that reach column I.  (What follows a row's size only is worked out once
    // per size: planning runs on every call, and dividing per row and candidate
    // shape took 147 us of host time for 6000 x 3000 at batch 20, against 20)
    int32_t kept_of[DARB_MAX_BLOCK + 1] = {};
    for (int m = f.m_min; m <= f.m_max; ++m) {
        int xr, hr;
        row_regions(static_cast<int>((f.cols + m - 1) / m), m, I, pre, kGru, xr, hr);
        kept_of[m] = xr + hr;
    }
    std::vector<int64_t> kept(static_cast<size_t>(H));
    int64_t total = 0;
    for (int u = 0; u < H; ++u) {
        int64_t k = 0;
        for (int q = 0; q < kGates; ++q) k += kept_of[row_m[int64_t(q) * H + u]];
        kept[static_cast<size_t>(u)] = k;
        total += k;
    }
    a.irows = pre ? 0 : (I + 3) / 4 * 4;
    a.hrows = (H + 3) / 4 * 4;
    const int in_rows = a.irows + a.hrows + 1;
    const int cmax = std::min({sm_count(), H, kMaxCtas});
    // The tile widths and the group counts, by the time a step is expected to
    // take: per tile a fixed part (barrier, cell, latencies: 2.5 us), the
    // staging of in_rows rows and the gather of the CTA's kept weights.  A
    // narrow tile stages less but keeps more weights a CTA, each of which
    // costs its own share of a load, and a quarter-warp's staged rows then
    // share banks (cycles per weight: measured on two gate matrices only,
    // 4096 x 1280 fp32 and 6000 x 3000 bf16; of 240 sequences of other sizes, 64
    // to 1500 units at batches 1 to 128, none took longer than with one lane a
    // column behind one barrier).
    Shape shapes[(kMaxLbt + 1) * 80];
    int nshapes = 0;
    for (int lbt = 0; lbt <= kMaxLbt && (lbt == 0 || (1 << (lbt - 1)) < B); ++lbt) {
        const int bt = 1 << lbt;
        const int64_t nt = (B + bt - 1) / bt;
        static const double kCycles[kMaxLbt + 1] = {0.6, 0.75, 0.85, 1.1, 1.5, 1.9};
        int64_t last = -1;
        for (int64_t tpg = 1; tpg <= nt; tpg = tpg < 8 ? tpg + 1 : tpg * 2) {
            const int64_t ng = (nt + tpg - 1) / tpg;
            if (ng > cmax || ng == last) continue;
            last = ng;
            const int members = std::min<int>(std::max(1, sm_count() / static_cast<int>(ng)), std::min(H, kMaxCtas));
            const double mine = double(total) / members;
            const double tile = 2500.0 + double(in_rows) * bt * 4 / 150.0 + mine * kCycles[lbt] / 1.9;
            shapes[nshapes++] = {lbt, static_cast<int>(ng), static_cast<int>((nt + ng - 1) / ng),
                                 double((nt + ng - 1) / ng) * tile};
        }
        if (last != 1) shapes[nshapes++] = {lbt, 1, static_cast<int>(nt), 1e18 / bt};   // always a candidate
    }
    Ranges rg{};
    SmemPlan sp{};
    Shape s{};
    int members = 0;
    bool fits = false;
    while (nshapes > 0 && !fits) {
        // the next best; one of the first few nearly always fits
        Shape *const next =
            std::min_element(shapes, shapes + nshapes, [](const Shape &p, const Shape &q) { return p.ns < q.ns; });
        s = *next;
        *next = shapes[--nshapes];
        const int bt = 1 << s.lbt;
        members = std::max(1, std::min({sm_count() / s.ngroups, H, kMaxCtas}));
        // what no split of the units can go below: the mean of kept weights and of
        // units (and an item a row)
        const int units_min = (H + members - 1) / members;
        if (smem_plan((total + members - 1) / members, kGates * units_min, kGates * units_min, units_min, BF16,
                      kGru && !pre, in_rows, bt, s.tpg, false, pre)
                .total > kSmemCap)
            continue;
        int64_t kept_cap = 0;
        int units_cap = 0;
        split_units(kept, members, rg, kept_cap, units_cap);
        if (kept_cap > (int64_t(1) << 20)) continue;
        const bool c_on_chip = !kGru && size_t(units_cap) * size_t(s.tpg) * bt * 4 <= kCellOnChip;
        // work items: rows longer than a warp's share of the CTA's weights are
        // cut (at least 2 loads per subgroup), or none where their partial sums
        // do not fit.  Items handed out longest first balance the warps: four
        // times as many, in row order, took 7.8 us against 6.5 a step on
        // 4096 x 1280 fp32 at batch 32
        const int S = bt < 4 ? 32 : 128 / bt, KW = S <= 4 ? 4 : S <= 8 ? 2 : 1;
        for (int cut = 1; cut >= 0 && !fits; --cut) {
            a.piece = round4(static_cast<int>(
                cut ? std::max<int64_t>(2 * KW * S, (kept_cap + kSeqWarps - 1) / kSeqWarps) : kept_cap));
            int32_t items_of[DARB_MAX_BLOCK + 1] = {};   // of a row of block size m
            for (int m = f.m_min; m <= f.m_max; ++m) items_of[m] = (kept_of[m] + a.piece - 1) / a.piece;
            int items_cap = 0;
            for (int q = 0; q < members; ++q) {
                int items = 0;
                for (int g = 0; g < kGates; ++g)
                    for (int u = rg.start[q]; u < rg.start[q + 1]; ++u) items += items_of[row_m[int64_t(g) * H + u]];
                items_cap = std::max(items_cap, items);
            }
            sp = smem_plan(kept_cap, kGates * units_cap, items_cap, units_cap, BF16, kGru && !pre, in_rows, bt, s.tpg,
                           c_on_chip, pre);
            fits = sp.total <= kSmemCap;
        }
        a.c_on_chip = c_on_chip ? 1 : 0;
    }
    if (!fits) return cudaErrorNotSupported;
    const int bt = 1 << s.lbt;
    a.ngroups = s.ngroups;
    a.tpg = s.tpg;
    a.ntiles = static_cast<int>((B + bt - 1) / bt);
    a.c_last = c_last;
    // small tiles are exchanged as tagged pairs: a reader waits for the values
    // themselves, not for a barrier and then for them (us a step: LSTM 4096 x
    // 1280 at batch 1 / 8 4.2 / 4.9 -> 3.5 / 4.6, H = 200 at 13 3.5 -> 2.7); twice
    // the bytes cost more than that on tiles of 128 KB (batch 32: 6.3 -> 8.1)
    a.tagged = size_t(a.hrows) * bt * 4 <= kTaggedBytes ? 1 : 0;
    const auto kernel = a.tagged ? seq_entry<BF16, MODE, true>(s.lbt) : seq_entry<BF16, MODE, false>(s.lbt);
    const cudaError_t attr = allow_smem(kernel, kSmemCap);
    if (attr != cudaSuccess) return attr;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeCooperative;
    at[0].val.cooperative = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(static_cast<unsigned>(members * s.ngroups));
    cfg.blockDim = dim3(kThreads);
    cfg.dynamicSmemBytes = sp.total;
    cfg.stream = stream;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    // every wait is bounded by kWaitLimitNs; a test may shorten the barrier's
    // limit and hold back one CTA's first arrival (sequence_test_hook)
    a.barrier_ns = kWaitLimitNs;
    a.skip_cta = -1;
    sequence_test_hook(&a.barrier_ns, &a.skip_cta);
    // x_t is read in place when its rows are already tile-major; else from a
    // tile-major copy, or by plain loads where that copy would be too large (or
    // cannot be had, below)
    const bool x_in_place = I % 4 == 0 && B == bt && reinterpret_cast<uintptr_t>(a.x) % 16 == 0;
    const size_t xt_bytes = size_t(T) * size_t(a.ntiles) * size_t(a.irows) * bt * 4;
    a.x_mode = pre || I == 0 ? kXNone : x_in_place || xt_bytes <= (size_t(1) << 30) ? kXBulk : kXPlain;
    // workspace: barrier counters and abort flag; the cell state when it is
    // neither on chip nor in c_last; the exchanged h; the x parts and the
    // product input they come from, or the tile-major copy of x
    const int nwords = (a.ngroups + 1) * kBarWords;
    const size_t bar_bytes = up(size_t(nwords) * 4);
    const size_t cbytes = kGru || a.c_on_chip || c_last ? 0 : up(size_t(H) * size_t(B) * 4);
    const size_t hx_bytes = up(2 * size_t(a.ntiles) * size_t(a.hrows) * bt * (a.tagged ? 8 : 4));
    bool x_copy = a.x_mode == kXBulk && !x_in_place;
    const size_t base_bytes = bar_bytes + cbytes + hx_bytes + (pre ? pre_bytes : 0);
    char *ws = nullptr;
    cudaError_t e = stream_alloc(reinterpret_cast<void **>(&ws), base_bytes + (x_copy ? up(xt_bytes) : 0), stream);
    if (e == cudaErrorMemoryAllocation && x_copy) {   // no room for the copy of x: the steps read it in place
        x_copy = false;
        a.x_mode = kXPlain;
        e = stream_alloc(reinterpret_cast<void **>(&ws), base_bytes, stream);
    }
    if (e != cudaSuccess) return e;
    a.bar = reinterpret_cast<unsigned *>(ws);
    a.abort_flag = reinterpret_cast<int *>(ws + size_t(a.ngroups) * kBarWords * 4);
    a.c_state = kGru || a.c_on_chip ? nullptr : (c_last ? c_last : reinterpret_cast<float *>(ws + bar_bytes));
    a.h_x = reinterpret_cast<float *>(ws + bar_bytes + cbytes);
    float *const xws = reinterpret_cast<float *>(ws + bar_bytes + cbytes + hx_bytes);
    a.x_tiles = a.x_mode != kXBulk ? nullptr : x_in_place ? a.x : xws;
    last_sequence() = {a.tagged, bt, s.ngroups, s.tpg, a.c_on_chip, a.x_mode};
    const int64_t warps = H + (pre || x_copy ? T * I : 0);
    const unsigned grid = static_cast<unsigned>(std::min<int64_t>((warps + 7) / 8, int64_t(sm_count()) * 16));
    e = launch_ex(prep_kernel, dim3(grid), dim3(256), 0, stream, 1, false, a, s.lbt, h0, x_copy ? xws : nullptr,
                  pre ? xws : nullptr, ldx, nwords);
    if (pre) {
        float *gx = reinterpret_cast<float *>(reinterpret_cast<char *>(xws) + up(size_t(I + H) * ldx * 4));
        if (e == cudaSuccess) {
            e = launch_spmm_prefix(f, I, xws, ldx, T * B, gx, ldx, false, stream);
            if (e == cudaErrorNotSupported) {   // the whole product then: the rows of h are zero
                e = cudaMemsetAsync(xws + size_t(I) * ldx, 0, size_t(H) * ldx * 4, stream);
                if (e == cudaSuccess) e = launch_spmm(f, xws, ldx, T * B, gx, ldx, false, DARB_PATH_AUTO, stream);
            }
        }
        a.gx = gx;
        a.ldgx = ldx;
    }
    if (e == cudaSuccess) e = cudaLaunchKernelEx(&cfg, kernel, f, a, rg, sp);
    const cudaError_t ef = cudaFreeAsync(ws, stream);
    return e != cudaSuccess ? e : ef;
}

cudaError_t launch_lstm_sequence(const Format &f, const int32_t *row_m, int64_t T, int64_t I, int64_t H, int64_t B,
                                 const float *x, const float *h0, const float *c0, const float *bias, float *h_seq,
                                 float *c_seq, float *c_last, cudaStream_t stream) {
    seq::SeqArgs a{};
    a.I = static_cast<int>(I);
    a.H = static_cast<int>(H);
    a.T = static_cast<int>(T);
    a.B = B;
    a.x = x;
    a.c0 = c0;
    a.bias = bias;
    a.h_seq = h_seq;
    a.c_seq = c_seq;
    a.status = f.status;
    return f.bf16 ? launch_seq_t<true, kModeLstm>(f, row_m, a, h0, c_last, stream)
                  : launch_seq_t<false, kModeLstm>(f, row_m, a, h0, c_last, stream);
}

cudaError_t launch_gru_sequence(const Format &f, const int32_t *row_m, int64_t T, int64_t I, int64_t H, int64_t B,
                                const float *x, const float *h0, const float *b_ih, const float *b_hh, float *h_seq,
                                cudaStream_t stream) {
    seq::SeqArgs a{};
    a.I = static_cast<int>(I);
    a.H = static_cast<int>(H);
    a.T = static_cast<int>(T);
    a.B = B;
    a.x = x;
    a.b_ih = b_ih;
    a.b_hh = b_hh;
    a.h_seq = h_seq;
    a.status = f.status;
    return f.bf16 ? launch_seq_t<true, kModeGru>(f, row_m, a, h0, nullptr, stream)
                  : launch_seq_t<false, kModeGru>(f, row_m, a, h0, nullptr, stream);
}

}  // namespace darb
