// rnn.cu -- one LSTM or GRU cell step on a DARB gate matrix, in one kernel.
//
// The gate matrix (4H or 3H rows, I + H columns) multiplies the stacked input
// [x_t; h_{t-1}], read in place from the two caller buffers.  rnn_step.cuh
// keeps all gates of a hidden unit in one CTA.  Where its staged input does
// not fit (some 14000 rows), the batch is above 1024, or it is expected to take
// longer (large matrices, whose inputs it can stage for a few columns only),
// the product kernels of darb_spmm run in an RNN output mode
// (rnn_epilogue.cuh): each gate row's final sum is published to scratch,
// arrivals are counted per hidden unit, and the CTA that brings a unit's last
// gate applies the cell; batch <= 4 on the row-per-lane kernel (instantiated
// here), larger batches on the batch-per-lane kernel (rnn_batch.cu).  GRU keeps
// the x part and the h part of each gate sum apart (a and bh), since the reset
// gate multiplies only the h part of the candidate gate.
#include "rowlane.cuh"

namespace darb {

// An upper bound on the batch tiles any RNN kernel uses for a batch of B
// (sizes the arrival counters): one tile up to 4 columns, else at most one per
// 8 columns.
int rnn_batch_tile(int64_t B) { return B == 1 ? 1 : B == 2 ? 2 : B <= 4 ? 4 : 8; }

// What rowlane_kernel is expected to take for a step of 1 or 2 columns, ns: a
// fixed part, the kept weights (in thousands) and the longest row, which the
// CTAs of a cluster share.  Fitted to 36 gate matrices: 6 to 8% root mean
// square.  From 3 columns on the step kernel was never slower.
static double rowlane_ns(const Format &f, int64_t B) {
    if (B > 2) return 1e300;
    const double kept = double(f.set_prefix[0][f.nitems[0][0]]) * kSlots * kChunk / 1000.0;
    const double longest = double(f.nch_max) / rowlane::cluster_size(f);
    return B == 1 ? 6086.0 + (f.bf16 ? 0.975 : 1.835) * kept + 37.8 * longest
                  : 6028.0 + (f.bf16 ? 2.07 : 2.35) * kept + 61.2 * longest;
}

// The kernel that is expected to take less.  Over 473 steps of 36 gate matrices
// (192 to 20000 rows, inputs of 192 to 13024 rows) at batches from 1 to 128,
// each timed on every kernel, the choice is on average 1% above the fastest; 5
// were more than 3% above the kernels below, the worst 10%.  us, step kernel
// against those: LSTM 16384 x 8192 bf16 at batch 32 84 / 56, 4768 x 8192 at
// batch 1 13.0 / 10.7 and at 64 82 / 60; but 6000 x 3000 at 64 25 / 39, and
// batch 4 9.1 / 17.5 at 8000 x 4096.
template <int MODE>
static cudaError_t launch_step(const Format &f, const RnnArgs &ra, bool early, Kernel kernel, cudaStream_t stream) {
    if (kernel == kKernelNone || kernel == kKernelRows) {
        const double limit_ns = kernel == kKernelRows ? 1e300
                                : ra.B <= 4           ? rowlane_ns(f, ra.B)
                                                      : rnn_batch_ns(f, ra, MODE);
        const cudaError_t e = launch_rnn_step(f, ra, MODE, early, limit_ns, stream);
        if (e != cudaErrorNotSupported || kernel == kKernelRows) return e;
    } else if (kernel != (ra.B <= 4 ? kKernelRowlane : kKernelBatch)) {
        return cudaErrorNotSupported;
    }
    if (ra.counters == nullptr) return cudaErrorNotSupported;
    if (ra.B <= 4)
        return f.bf16 ? rowlane::launch_any<true, MODE>(f, nullptr, 0, ra.B, nullptr, 0, ra, early, stream)
                      : rowlane::launch_any<false, MODE>(f, nullptr, 0, ra.B, nullptr, 0, ra, early, stream);
    return launch_rnn_batch(f, ra, MODE, early, stream);
}

cudaError_t launch_lstm_step(const Format &f, int64_t I, int64_t H, int64_t B, const float *x,
                             const float *h_prev, const float *c_prev, const float *bias,
                             float *h_out, float *c_out, RnnScratch s, cudaStream_t stream, bool early,
                             Kernel kernel) {
    RnnArgs ra{};
    ra.x = x; ra.h = h_prev; ra.gx = s.gates; ra.gh = nullptr; ra.counters = s.counters;
    ra.c_prev = c_prev; ra.bias = bias; ra.h_out = h_out; ra.c_out = c_out;
    ra.I = static_cast<int>(I); ra.H = static_cast<int>(H); ra.B = B;
    return launch_step<kModeLstm>(f, ra, early, kernel, stream);
}

cudaError_t launch_gru_step(const Format &f, int64_t I, int64_t H, int64_t B, const float *x,
                            const float *h_prev, const float *b_ih, const float *b_hh,
                            float *h_out, RnnScratch s, cudaStream_t stream, bool early, Kernel kernel) {
    RnnArgs ra{};
    ra.x = x; ra.h = h_prev; ra.gx = s.gates; ra.gh = s.gates ? s.gates + f.rows * B : nullptr; ra.counters = s.counters;
    ra.b_ih = b_ih; ra.b_hh = b_hh; ra.h_out = h_out;
    ra.I = static_cast<int>(I); ra.H = static_cast<int>(H); ra.B = B;
    return launch_step<kModeGru>(f, ra, early, kernel, stream);
}

}  // namespace darb
