// rnn_step.cuh -- one LSTM or GRU cell step, or a plain product, local
// to the CTA that owns a hidden unit or a row (Sec. 3.2, Fig. 6(b) on the
// stacked input [x_t; h_{t-1}], then the cell of Sec. 4.1; or on X).
//
// The batch columns are cut into tiles of bt columns, and the CTAs into one
// group a tile; within a group every CTA owns a contiguous range of hidden
// units with all their gate rows, so no gate sum leaves its CTA: no cluster,
// no scratch, no counters.  The ranges cost about the same (unit_split.h; with
// equal numbers of units instead, 6000 x 3000 fp32 at batch 16 with its first
// tenth of the rows in blocks of 4 and the rest of 64 took 28.0 us against 8.2,
// and rows of mixed blocks 5% more).  A CTA
//  * reads its rows' places in the format and, when the handle is complete,
//    starts on their first records before the PDL wait;
//  * stages the tile's columns of x_t and h_{t-1} whole (tensor-map boxes, or
//    16- or 4-byte asynchronous copies), with its units' c_{t-1} and biases;
//  * multiplies: bt / 4 lanes share a kept weight, 4 columns each (a 16-byte
//    load of the staged row the weight selects).  The chunks of the CTA's rows
//    form one stream that the 16 * 128 / bt lane groups share out evenly, a
//    contiguous run each, so that rows of any length balance; the records come
//    straight from L2, two chunks ahead of their use;
//  * adds the runs' partial sums of each row in order (deterministic) and
//    applies the cell.
// A GRU row is two rows of the stream, its x part and its h part (r multiplies
// only the h part of the candidate); a chunk that holds columns of both sides
// of I, or runs past the row's last block, is in each with the other side's
// weights as zeros on a zero row.
//
// What bounds it: the latency of its phases (staging, gather, cell; 3 to 4 us
// with the launch) and, for wide matrices, the gather.  A step (us, in a graph
// of steps) against the kernels whose gate sums meet through clusters, scratch
// and counters (rowlane_kernel, batch_kernel): LSTM 4096 x 1280 fp32 at batch
// 1 / 8 / 32 / 64: 6.1 / 5.7 / 7.2 / 10.4 against 7.6 / 16.9 / 25.0 / 29.4; GRU
// 3072 x 2048 bf16 at batch 64: 11.0 against 32.8; LSTM 6000 x 3000 bf16 at
// batch 20: 16.0 against 36.8, fp32 at batch 37: 23.2 against 78.5.  Those
// kernels remain for inputs too tall to stage at 4 columns (some 14000 rows),
// for more than 1024 columns, and where they are expected to be faster
// (rnn.cu): above some 3600 stacked rows the tiles are narrow.
//
// A plain product (kModeY; the rows are the units, X the whole input) takes
// this kernel from batch 5 on while it is expected to be faster than the
// kernels that stream through clusters (spmm_batch.cu), whose fixed part is
// larger but whose gather is cheaper.  us against the faster of those: 1024 x
// 1024 fp32 at batch 6 / 8 / 24 / 64: 3.6 / 3.4 / 3.6 / 4.1 against 10.7 / 4.7 /
// 6.8 / 7.6; 6000 x 3000 fp32 at 6 / 8 / 16: 8.3 / 7.1 / 8.9 against 12.9 / 13.0 /
// 13.0, but 14.8 against 11.6 at 32; 2000 x 2500 fp32 at 24 / 64: 6.0 / 8.6
// against 6.5 / 8.8; 4096 x 4096 bf16 at 8: 5.2 against 7.9, but 8.5 against 7.4
// at 16.
#pragma once

#include "kernels_common.cuh"
#include "launch.cuh"
#include "rnn_epilogue.cuh"
#include "tma.cuh"

#include <cuda.h>
#include <cudaTypedefs.h>

#include <algorithm>
#include <cstring>

namespace darb {
namespace step {

constexpr int kThreads = 512;
constexpr int kStepWarps = kThreads / 32;
constexpr size_t kSmemCap = 227 * 1024 - 256;   // dynamic shared memory, with room for the static part
constexpr int kMinLbt = 2, kMaxLbt = 5;         // batch tiles of 4, 8, 16 or 32 columns
constexpr int kAhead = 2;                       // chunks a lane group has requested ahead of its use

// A row (GRU: a side of a row) of a CTA's stream of chunks.
struct Row {
    uint32_t rec, off;   // value record (8 values) and offset word of its chunk 0
    int c0;              // first chunk in the stream
    int m_nib;           // block size | 4-bit offsets << 16
    int klo, khi;        // its columns [klo, khi)
    int at;              // position of chunk c0 in the stream
    int seg;             // partial sums: first index
};

constexpr int kStage4 = 0, kStage16 = 1, kStageBoxes = 2;

struct Plan {
    int ntiles, members;          // CTA i is CTA i / ntiles of tile i % ntiles
    int64_t ldx, ldy;             // kModeY: pitches of X and Y
    int staging, early;           // kStage*; the records may be read before the PDL wait
    int nbx, bxh, nbh, bhh;       // boxes of x and h: their number and rows (the last one ends with the matrix)
    uint32_t row_off, nseg_off, bias_off, c_off, in_off, part_off;
    int by_cost;                  // the members' units: start's ranges, else equal numbers (unit_split.h)
    int start[kMaxMembers + 1];
};

template <bool BF16, int MODE, int LBT>
__global__ void __launch_bounds__(kThreads, 1)
step_kernel(Format f, RnnArgs ra, const __grid_constant__ CUtensorMap mx, const __grid_constant__ CUtensorMap mh,
            const __grid_constant__ Plan p) {
    constexpr int kGates = MODE == kModeLstm ? 4 : MODE == kModeGru ? 3 : 1;
    constexpr bool kGru = MODE == kModeGru;
    constexpr int kSides = kGru ? 2 : 1;
    constexpr int bt = 1 << LBT, L = bt / 4, S = 32 / L, kSubs = kStepWarps * S;
    constexpr int kRowShift = LBT + 2;   // log2 of the bytes of a staged row
    extern __shared__ __align__(128) unsigned char sm[];
    __shared__ __align__(8) uint64_t s_full;
    __shared__ int s_total;
    Row *s_row = reinterpret_cast<Row *>(sm + p.row_off);      // [VR + 1]
    int *s_nseg = reinterpret_cast<int *>(sm + p.nseg_off);    // [VR]
    float *s_bias = reinterpret_cast<float *>(sm + p.bias_off);   // [VR]: GRU b_ih then b_hh
    float *s_c = reinterpret_cast<float *>(sm + p.c_off);      // [units][bt]: c_{t-1} (LSTM)
    float *s_in = reinterpret_cast<float *>(sm + p.in_off);    // [K + 1][bt], row K zero
    float *s_part = reinterpret_cast<float *>(sm + p.part_off);   // [VR + kSubs][bt]

    pdl_launch_dependents();
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int tile = int(blockIdx.x) % p.ntiles, member = int(blockIdx.x) / p.ntiles;
    const int H = ra.H, I = ra.I, K = MODE == kModeY ? I : I + H;   // kModeY: H rows, I columns
    const int64_t B = ra.B, ldx = MODE == kModeY ? p.ldx : B, b0 = int64_t(tile) << LBT;
    const int nb = static_cast<int>(B - b0 < bt ? B - b0 : bt);
    const int u0 = p.by_cost ? p.start[member] : static_cast<int>(int64_t(H) * member / p.members);
    const int nu = (p.by_cost ? p.start[member + 1] : static_cast<int>(int64_t(H) * (member + 1) / p.members)) - u0;
    const int R = kGates * nu, VR = kSides * R;   // local row q*nu + i is matrix row q*H + u0 + i
    auto grow = [&](int lr) { return (lr / nu) * H + u0 + lr % nu; };

    // ---- the rows' places in the format (immutable: before the PDL wait)
    for (int v = tid; v < VR; v += kThreads) {
        const int lr = v < R ? v : v - R;
        const int loc = f.rowloc[grow(lr)];
        const Group g = f.groups[loc / kSlots];
        const int slot = loc % kSlots;
        const bool xside = kGru && v < R, hside = kGru && v >= R;
        const int nch = (g.n + kChunk - 1) / kChunk, span = kChunk * g.m;
        Row r;
        r.rec = static_cast<uint32_t>(g.val_off / kChunk) + slot;
        r.off = static_cast<uint32_t>(g.off_off) + slot * (g.nib ? 1 : 2);
        r.m_nib = g.m | (g.nib ? 1 << 16 : 0);
        r.klo = hside ? I : 0;
        r.khi = xside ? I : K;
        r.c0 = hside ? min(nch, I / span) : 0;
        const int c1 = xside ? min(nch, (I + span - 1) / span) : nch;
        r.at = c1 > r.c0 ? c1 - r.c0 : 0;   // its chunks, until the scan below
        r.seg = 0;
        s_row[v] = r;
    }
    for (int j = tid; j < bt; j += kThreads) s_in[(K << LBT) + j] = 0.0f;
    if (tid == 0) {
        mbar_init(&s_full, 1);
        fence_mbar_init();
    }
    __syncthreads();
    if (warp == 0) {   // where each row's chunks start in the stream
        int base = 0;
        for (int v0 = 0; v0 < VR; v0 += 32) {
            const int n = v0 + lane < VR ? s_row[v0 + lane].at : 0;
            int incl = n;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int up = __shfl_up_sync(0xFFFFFFFFu, incl, o);
                if (lane >= o) incl += up;
            }
            if (v0 + lane < VR) s_row[v0 + lane].at = base + incl - n;
            base += __shfl_sync(0xFFFFFFFFu, incl, 31);
        }
        if (lane == 0) {
            s_row[VR].at = base;
            s_total = base;
        }
    }
    __syncthreads();
    const int total = s_total;
    const int N = max(1, (total + kSubs - 1) / kSubs);   // chunks of a lane group
    // the lane groups that share a row are consecutive, and group + row is
    // different for every (group, row) that meet: the index of a partial sum
    for (int v = tid; v < VR; v += kThreads) {
        const int a = s_row[v].at, b = s_row[v + 1].at;
        s_row[v].seg = a / N + v;
        s_nseg[v] = b > a ? (b - 1) / N - a / N + 1 : 0;
    }

    // ---- this lane group's run of chunks, [pos, end)
    const int sub = warp * S + lane / L;
    const uint32_t xl = smem_addr(s_in) + uint32_t(lane % L) * 16u;
    const int pos = min(total, sub * N), end = min(total, pos + N);
    constexpr int kW = BF16 ? 4 : 8;
    struct Fetch {
        uint32_t vw[kW];
        uint2 ow;
        int v;          // row of the stream (-1: none)
        int m, kb;      // its block size and the chunk's first column
        bool whole;     // all of the chunk's blocks lie inside the row's columns
    };
    Fetch buf[kAhead];
    int lv = 0;     // row of the next chunk to request
    if (pos < end) {
        int hi = VR;   // the last row that starts at or before pos
        while (hi - lv > 1) {
            const int mid = (lv + hi) / 2;
            if (s_row[mid].at <= pos) lv = mid;
            else hi = mid;
        }
    }
    // the row of the next chunk to request stays in registers (read from shared
    // memory for each chunk: GRU 3072 x 2048 at batch 64 11.5 us against 10.9)
    Row row = s_row[lv];
    int row_end = s_row[lv + 1].at;
    auto fetch = [&](int i, Fetch &b) {   // chunk i of the stream
        b.v = -1;
        if (i >= end) return;
        if (i >= row_end) {
            do row_end = s_row[++lv + 1].at;
            while (i >= row_end);
            row = s_row[lv];
        }
        const int c = row.c0 + i - row.at, m = row.m_nib & 0xFFFF;
        const bool nib = row.m_nib >> 16;
        b.v = lv;
        b.m = m;
        b.kb = c * kChunk * m;
        b.whole = b.kb >= row.klo && b.kb + kChunk * m <= row.khi;
        const uint4 *pv = static_cast<const uint4 *>(f.vals) + int64_t(row.rec + uint32_t(c) * kSlots) * (BF16 ? 1 : 2);
        const uint4 w0 = __ldg(pv);
        b.vw[0] = w0.x; b.vw[1] = w0.y; b.vw[2] = w0.z; b.vw[3] = w0.w;
        if constexpr (!BF16) {
            const uint4 w1 = __ldg(pv + 1);
            b.vw[4] = w1.x; b.vw[5] = w1.y; b.vw[6] = w1.z; b.vw[7] = w1.w;
        }
        if (nib) {
            const uint32_t w = __ldg(f.offs + row.off + uint32_t(c) * kSlots);
            const uint32_t even = w & 0x0F0F0F0Fu, odd = (w >> 4) & 0x0F0F0F0Fu;
            b.ow = make_uint2(__byte_perm(even, odd, 0x5140), __byte_perm(even, odd, 0x7362));
        } else {
            b.ow = __ldg(reinterpret_cast<const uint2 *>(f.offs + row.off + uint32_t(c) * (2 * kSlots)));
        }
    };
    if (p.early) {
#pragma unroll
        for (int i = 0; i < kAhead; ++i) fetch(pos + i, buf[i]);
    }

    // ---- the inputs
    pdl_wait_previous();
    if (LBT == 5 && p.staging == kStageBoxes) {
        if (warp == 0) {
            if (lane == 0) mbar_arrive_expect_tx(&s_full, uint32_t(p.nbx * p.bxh + p.nbh * p.bhh) << kRowShift);
            __syncwarp();
            for (int i = lane; i < p.nbx + p.nbh; i += 32) {
                const bool isx = i < p.nbx;
                const int rows = isx ? I : H, bh = isx ? p.bxh : p.bhh;
                const int y = min((isx ? i : i - p.nbx) * bh, rows - bh);
                tensor2d_g2s(s_in + (int64_t((isx ? 0 : I) + y) << LBT), isx ? &mx : &mh, int(b0), y, &s_full);
            }
        }
    } else if (p.staging == kStage16) {
        constexpr int Q = bt / 4, kStep = kThreads / Q;
        const int j = (tid & (Q - 1)) * 4;
        const bool in = j < nb;   // B is a multiple of 4
        uint32_t dst = smem_addr(s_in) + uint32_t(tid) * 16u;
        const float *const sx = ra.x + b0 + (in ? j : 0), *const sh = ra.h + b0 + (in ? j : 0);
#pragma unroll 4
        for (int k = tid / Q; k < K; k += kStep, dst += kThreads * 16)
            cp_async16(dst, MODE == kModeY || k < I ? sx + int64_t(k) * ldx : sh + int64_t(k - I) * B, in);
    } else {
        constexpr int kStep = kThreads >> LBT;
        const int j = tid & (bt - 1);
        const bool in = j < nb;
        uint32_t dst = smem_addr(s_in) + uint32_t(tid) * 4u;
        const float *const sx = ra.x + b0 + (in ? j : 0), *const sh = ra.h + b0 + (in ? j : 0);
#pragma unroll 4
        for (int k = tid >> LBT; k < K; k += kStep, dst += kThreads * 4)
            cp_async4(dst, MODE == kModeY || k < I ? sx + int64_t(k) * ldx : sh + int64_t(k - I) * B, in);
    }
    if constexpr (MODE != kModeY)
    for (int v = tid; v < VR; v += kThreads) {
        const float *b = kGru ? (v < R ? ra.b_ih : ra.b_hh) : ra.bias;
        cp_async4(smem_addr(s_bias + v), b ? b + grow(v < R ? v : v - R) : ra.h, b != nullptr);
    }
    if constexpr (MODE == kModeLstm)
        for (int i = tid; i < nu << LBT; i += kThreads) {
            const int j = i & (bt - 1);
            cp_async4(smem_addr(s_c + i), ra.c_prev + int64_t(u0 + (i >> LBT)) * B + b0 + (j < nb ? j : 0), j < nb);
        }
    if (!p.early) {
#pragma unroll
        for (int i = 0; i < kAhead; ++i) fetch(pos + i, buf[i]);
    }
    cp_async_wait_all();
    __syncthreads();
    if (LBT == 5 && p.staging == kStageBoxes && !mbar_wait(&s_full, 0)) {
        atomicOr(f.status, kStatusTimeout);
        mbar_wait(&s_full, 0);   // the boxes may still land: before this CTA can leave
    }

    // ---- the products
    float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
    int cur = -1;   // row of the sums in acc
    auto flush = [&]() {
        if (cur >= 0) reinterpret_cast<float4 *>(s_part)[(cur + sub) * L + lane % L] = acc;
    };
    auto multiply = [&](const Fetch &b) {
        if (b.v < 0) return;
        if (b.v != cur) {
            flush();
            acc = make_float4(0.f, 0.f, 0.f, 0.f);
            cur = b.v;
        }
        const int m = b.m, kb = b.kb;
        // a chunk's products are added by themselves first: the chain of fp32
        // additions of a run stays short
        float4 s0 = make_float4(0.f, 0.f, 0.f, 0.f), s1 = s0;
        auto weight = [&](int e) {
            if constexpr (BF16)
                return __uint_as_float((e & 1) ? (b.vw[e >> 1] & 0xFFFF0000u) : (b.vw[e >> 1] << 16));
            else return __uint_as_float(b.vw[e]);
        };
        auto load = [&](uint32_t ad) {
            float4 x;
            asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];"
                         : "=f"(x.x), "=f"(x.y), "=f"(x.z), "=f"(x.w) : "r"(ad));
            return x;
        };
        if (b.whole) {
            const uint32_t xb = xl + (uint32_t(kb) << kRowShift), step = uint32_t(m) << kRowShift;
            float4 x[kChunk];
#pragma unroll
            for (int e = 0; e < kChunk; ++e)
                x[e] = load(xb + uint32_t(e) * step + (((e < 4 ? b.ow.x : b.ow.y) >> (8 * (e & 3)) & 255u) << kRowShift));
#pragma unroll
            for (int e = 0; e < kChunk; ++e) fma4((e & 1) ? s1 : s0, weight(e), x[e]);
        } else {
            const int klo = s_row[b.v].klo, khi = s_row[b.v].khi;
#pragma unroll
            for (int e = 0; e < kChunk; ++e) {
                const int k = kb + e * m + int((e < 4 ? b.ow.x : b.ow.y) >> (8 * (e & 3)) & 255u);
                const bool in = k >= klo && k < khi;
                fma4((e & 1) ? s1 : s0, in ? weight(e) : 0.0f, load(xl + (uint32_t(in ? k : K) << kRowShift)));
            }
        }
        acc.x += s0.x + s1.x;
        acc.y += s0.y + s1.y;
        acc.z += s0.z + s1.z;
        acc.w += s0.w + s1.w;
    };
    for (int i = pos; i < end; i += kAhead) {
#pragma unroll
        for (int a = 0; a < kAhead; ++a) {
            const Fetch now = buf[a];
            fetch(i + a + kAhead, buf[a]);
            multiply(now);
        }
    }
    flush();
    __syncthreads();

    // ---- the cells of the owned units
    auto sum = [&](int v, int j) {
        const int seg = s_row[v].seg, n = s_nseg[v];
        float r0 = 0.0f, r1 = 0.0f;
        if constexpr (MODE != kModeY) {   // few: the lane groups' runs are long
            for (int i = 0; i < n; ++i) r0 += s_part[((seg + i) << LBT) + j];
            return r0;
        }
        for (int i = 0; i + 1 < n; i += 2) {
            r0 += s_part[((seg + i) << LBT) + j];
            r1 += s_part[((seg + i + 1) << LBT) + j];
        }
        if (n & 1) r0 += s_part[((seg + n - 1) << LBT) + j];
        return r0 + r1;
    };
    for (int i = tid; i < nu << LBT; i += kThreads) {
        const int ui = i >> LBT, j = i & (bt - 1);
        if (j >= nb) continue;
        const int64_t e = int64_t(u0 + ui) * B + b0 + j;
        if constexpr (MODE == kModeY) {
            ra.h_out[int64_t(u0 + ui) * p.ldy + b0 + j] = sum(ui, j);
        } else if constexpr (!kGru) {
            float pre[4];
#pragma unroll
            for (int q = 0; q < 4; ++q) pre[q] = sum(q * nu + ui, j) + s_bias[q * nu + ui];
            const float c = sigm(pre[1]) * s_c[i] + sigm(pre[0]) * tanhf(pre[2]);
            ra.c_out[e] = c;
            ra.h_out[e] = sigm(pre[3]) * tanhf(c);
        } else {
            float ax[3], bh[3];
#pragma unroll
            for (int q = 0; q < 3; ++q) {
                const int v = q * nu + ui;
                ax[q] = sum(v, j) + s_bias[v];
                bh[q] = sum(R + v, j) + s_bias[R + v];
            }
            const float rr = sigm(ax[0] + bh[0]);
            const float zz = sigm(ax[1] + bh[1]);
            const float nn = tanhf(ax[2] + rr * bh[2]);
            ra.h_out[e] = (1.0f - zz) * nn + zz * s_in[((I + u0 + ui) << LBT) + j];
        }
    }
}

// Boxes of at most 256 rows over n rows: their number and rows.  The last one
// ends with the matrix and repeats rows of the one before.
inline void boxes(int n, int *nbox, int *rows) {
    *rows = std::min(n, 256);
    *nbox = n > 0 ? (n + *rows - 1) / *rows : 0;
}

// Whether x and h_{t-1} (or X) can be staged by copies of 16 bytes.
inline bool aligned16(const RnnArgs &ra, bool product, int64_t ldx) {
    return ra.B % 4 == 0 && ldx % 4 == 0 && (ra.I == 0 || reinterpret_cast<uintptr_t>(ra.x) % 16 == 0) &&
           (product || reinterpret_cast<uintptr_t>(ra.h) % 16 == 0);
}

// What a tile is expected to take, ns: a fixed part (launch, latencies), the
// staged bytes by the way they are copied (4 or 16 bytes at a time, or boxes;
// 16-byte copies cost more where the last tile is ragged, or where the tile is
// part of a row), the kept weights of the busiest member (8 a chunk of its
// cost), and its outputs (cell updates of a step).  A narrow tile stages less,
// but its staged rows share banks and each CTA multiplies more weights.
struct TileCost {
    double fixed, stage4, stage16, boxes, ragged, part, weight, output;
};
// Fitted to the forced tiles of 47 product shapes (128 to 6000 rows of 300 to
// 9216 columns, block sizes mixed and in runs) at 26 batches from 5 to 256, and
// of 36 gate matrices (192 to 20000 rows, inputs of 192 to 13024 rows) at 27
// batches from 1 to 128: 6 to 9% root mean square, at worst a third off.
constexpr TileCost kProductCost[kMaxLbt - kMinLbt + 1] = {
    {3156, 0.0189, 0.0272, 0, 0, 0, 0.304, 0.358},
    {3098, 0.0173, 0.0035, 0, 0.0089, 0.0089, 0.445, 0.181},
    {3031, 0.0165, 0.0048, 0, 0.0073, 0, 0.682, 0.118},
    {3143, 0.0141, 0, 0.0039, 0.0048, 0, 1.247, 0.017}};
constexpr TileCost kStepCost[kMaxLbt - kMinLbt + 1] = {
    {4407, 0.0286, 0.0085, 0, 0, 0.0282, 0.270, 3.23},
    {4425, 0.0253, 0.0043, 0, 0.0047, 0.0123, 0.395, 1.93},
    {4509, 0.0227, 0.0043, 0, 0.0043, 0, 0.573, 1.86},
    {4389, 0.0241, 0, 0.0013, 0.0058, 0.0013, 0.768, 2.81}};

template <bool BF16, int MODE, int LBT>
cudaError_t launch_tile(const Format &f, const RnnArgs &ra, Plan p, size_t smem, cudaStream_t stream) {
    constexpr int bt = 1 << LBT;
    const auto kernel = step_kernel<BF16, MODE, LBT>;
    const cudaError_t attr = allow_smem(kernel, kSmemCap);
    if (attr != cudaSuccess) return attr;
    CUtensorMap mx, mh;
    std::memset(&mx, 0, sizeof mx);
    std::memset(&mh, 0, sizeof mh);
    // How the inputs are staged: whole 32-column tiles in tensor-map boxes (LSTM
    // 4096 x 1280 at batch 32: 7.8 us against 8.3 by 16-byte copies), other
    // aligned rows in 16-byte copies (boxes of short or ragged rows are slower:
    // batch 8 6.0 against 7.3 us, 6000 x 3000 at batch 20 17.5 against 21.6),
    // the rest 4 bytes at a time
    const int64_t ldx = MODE == kModeY ? p.ldx : ra.B;
    const bool aligned = aligned16(ra, MODE == kModeY, ldx);
    p.staging = aligned ? kStage16 : kStage4;
    if (LBT == 5 && aligned && ra.B % bt == 0 && tensor_map_encoder() != nullptr) {
        auto make = [&](CUtensorMap *m, const float *base, int rows, int boxh, int64_t ld) {
            if (rows == 0) return true;
            const cuuint64_t dims[2] = {cuuint64_t(ra.B), cuuint64_t(rows)};
            const cuuint64_t strides[1] = {cuuint64_t(ld) * 4};
            const cuuint32_t box[2] = {cuuint32_t(bt), cuuint32_t(boxh)};
            const cuuint32_t es[2] = {1, 1};
            return tensor_map_encoder()(m, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 2, const_cast<float *>(base), dims,
                                        strides, box, es, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE,
                                        CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                                        CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
        };
        boxes(ra.I, &p.nbx, &p.bxh);
        boxes(MODE == kModeY ? 0 : ra.H, &p.nbh, &p.bhh);
        if (make(&mx, ra.x, ra.I, p.bxh, ldx) && (MODE == kModeY || make(&mh, ra.h, ra.H, p.bhh, ra.B)))
            p.staging = kStageBoxes;
    }
    last_kernel() = kKernelRows;
    return launch_ex(kernel, dim3(static_cast<unsigned>(p.ntiles * p.members)), dim3(kThreads), smem, stream, 1, true,
                     f, ra, mx, mh, p);
}

// The step (or product) on this kernel, or cudaErrorNotSupported when the
// staged tile does not fit beside the CTA's rows even at 4 columns, or no tile
// width is expected to take less than limit_ns.
template <bool BF16, int MODE>
cudaError_t launch(const Format &f, const RnnArgs &ra, bool early, cudaStream_t stream, int64_t ldx, int64_t ldy,
                   double limit_ns) {
    constexpr int kGates = MODE == kModeLstm ? 4 : MODE == kModeGru ? 3 : 1;
    const int64_t K = MODE == kModeY ? ra.I : int64_t(ra.I) + ra.H;
    if (K > 60000 || ra.B > 1024 || f.nitems[0][0] <= 0) return cudaErrorNotSupported;
    // kept weights of the matrix, padded to whole groups and chunks
    if (double(f.set_prefix[0][f.nitems[0][0]]) * kSlots * kChunk > 8e9) return cudaErrorNotSupported;   // Row's indices of records and offset words are 32-bit
    const UnitSplits &splits = *f.splits[MODE == kModeLstm ? kUnitLstm : MODE == kModeGru ? kUnitGru : kUnitRow];
    const int sms = sm_count();
    const bool aligned = aligned16(ra, MODE == kModeY, MODE == kModeY ? ldx : ra.B);
    int lbt = -1, best_units = 0;
    Plan best{};
    double best_ns = limit_ns;
    // the places of a CTA's shared memory for members of up to `units` units, and
    // its bytes (0: more rows than the kernel handles)
    auto lay_out = [&](Plan &p, int units, int bt) -> size_t {
        const int vr = (MODE == kModeGru ? 2 : 1) * kGates * units, subs = kStepWarps * 128 / bt;
        if (units > 4096 || vr > 4096) return 0;
        size_t o = 0;
        auto take = [&](size_t bytes) {
            const size_t at = o;
            o = (o + bytes + 127) / 128 * 128;
            return static_cast<uint32_t>(at);
        };
        p.in_off = take(size_t(K + 1) * bt * 4);
        p.part_off = take(size_t(vr + subs) * bt * 4);
        p.row_off = take(size_t(vr + 1) * sizeof(Row));
        p.nseg_off = take(size_t(vr) * 4);
        p.bias_off = take(size_t(vr) * 4);
        p.c_off = take(MODE == kModeLstm ? size_t(units) * bt * 4 : 0);
        return o;
    };
    // The tile widths, each with the time it would take if its members' shares
    // were equal: no split goes below that, so the widths are tried in the order
    // of it, and splits are worked out (once a handle) only for those that could
    // be the best.
    struct Tile {
        int l, ntiles, members;
        double ns, staging, weight, output;
        double expected_ns(double busiest, double units) const { return staging + busiest * weight + units * output; }
    } tiles[kMaxLbt - kMinLbt + 1];
    int ntiles = 0;
    for (int l = kMinLbt; l <= kMaxLbt && (l == kMinLbt || (1 << (l - 1)) < ra.B); ++l) {
        const int bt = 1 << l;
        Tile &t = tiles[ntiles++];
        t.l = l;
        t.ntiles = static_cast<int>((ra.B + bt - 1) / bt);
        t.members = std::max(1, std::min({sms / t.ntiles, ra.H, kMaxMembers}));
        const TileCost &cost = (MODE == kModeY ? kProductCost : kStepCost)[l - kMinLbt];
        const bool ragged = ra.B % bt != 0;
        const double per_byte = !aligned            ? cost.stage4
                                : l == 5 && !ragged ? cost.boxes
                                                    : cost.stage16 + (ragged ? cost.ragged : 0) +
                                                          (t.ntiles > 1 ? cost.part : 0);
        const int waves = (t.ntiles * t.members + sms - 1) / sms;
        t.staging = cost.fixed + waves * double(K) * bt * 4 * per_byte;
        t.weight = waves * kChunk * cost.weight;
        t.output = waves * bt * cost.output;
        t.ns = t.expected_ns(double(splits.total()) / t.members, double(ra.H) / t.members);
    }
    for (; ntiles > 0; --ntiles) {
        Tile *const next =
            std::min_element(tiles, tiles + ntiles, [](const Tile &p, const Tile &q) { return p.ns < q.ns; });
        const Tile t = *next;
        *next = tiles[ntiles - 1];
        if (!(t.ns < best_ns)) break;
        UnitSplit local;
        const UnitSplit &split = splits.get(t.members, local);
        // ranges by cost give some members many light units, whose rows and partial
        // sums may not fit; equal numbers then
        for (int by_cost = split.prefer_by_cost ? 1 : 0; by_cost >= 0; --by_cost) {
            const UnitRanges &r = by_cost ? split.by_cost : split.equal;
            const size_t bytes = lay_out(best, r.most_units, 1 << t.l);
            if (bytes == 0 || bytes > kSmemCap) continue;
            const double ns = t.expected_ns(double(r.busiest), double(r.most_units));
            if (ns < best_ns) {
                best_ns = ns;
                best.ntiles = t.ntiles;
                best.members = t.members;
                best.by_cost = by_cost;
                best_units = r.most_units;
                lbt = t.l;
            }
            break;
        }
    }
    if (lbt < 0) return cudaErrorNotSupported;
    const size_t smem = lay_out(best, best_units, 1 << lbt);
    if (best.by_cost) {
        UnitSplit local;
        const UnitSplit &split = splits.get(best.members, local);
        std::copy(split.start, split.start + best.members + 1, best.start);
    }
    best.early = early ? 1 : 0;
    best.ldx = ldx;
    best.ldy = ldy;
    return lbt == 2   ? launch_tile<BF16, MODE, 2>(f, ra, best, smem, stream)
           : lbt == 3 ? launch_tile<BF16, MODE, 3>(f, ra, best, smem, stream)
           : lbt == 4 ? launch_tile<BF16, MODE, 4>(f, ra, best, smem, stream)
                      : launch_tile<BF16, MODE, 5>(f, ra, best, smem, stream);
}

}  // namespace step
}  // namespace darb
