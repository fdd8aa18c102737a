// spmm_batch.cu -- the batch > 4 product for plain Y, on one of three kernels.
// Small and middling products take the kernel whose CTAs own rows and stage
// the whole input (rnn_step.cuh) while it is expected to be faster than the
// others, which split the columns over clusters: from 17 columns on, and for
// any batch whose X no tensor map can describe (FC6 at batch 13: 15 us against
// 26), the one with the activation tile resident in shared memory (xres.cuh)
// when the call fits it, else the streaming batch kernel (batch.cuh).  At 16
// columns or fewer xres's tile is half empty or more, and the streaming
// kernel measured faster (FC6 11.4 us against 12.6).
#include "batch.cuh"
#include "xres.cuh"

#include <algorithm>

namespace darb {

cudaError_t launch_spmm_batch(const Format &f, const float *X, int64_t ldx, int64_t batch, float *Y,
                              int64_t ldy, bool early, cudaStream_t stream) {
    // What the cluster kernels take, fitted to products of 300 to 9216 columns,
    // from the time of the gather at 128 bytes a clock and SM over whole
    // 32-column tiles.  batch_kernel: a fixed part and 1.5 times the gather (2.3
    // times for fp32 weights).  xres: the lesser of two readings, one from its
    // split (xres::expected_ns) and one of a fixed part, the load of a slice of
    // the columns (slower by plain copies) and the longer of its share of the
    // gather and of its heaviest unit, two groups of the smallest block size.
    // The rows kernel has to be expected to take 5% less.  Over 611 products of
    // 47 shapes, block sizes mixed and in runs, at 26 batches from 5 to 256,
    // each timed on every kernel, the choice is on average 2% above the fastest;
    // 9 were more than 3% above the cluster kernel, the worst 14% (700 x 6000 fp32
    // at batch 32: 9.3 us against 8.1).
    const bool aligned = reinterpret_cast<uintptr_t>(X) % 16 == 0 && ldx % 4 == 0;
    const bool streams = batch <= 16 && aligned;   // batch_kernel, else xres
    const double kept = double(f.set_prefix[0][f.nitems[0][0]]) * kSlots * kChunk;
    const double gather_ns = kept * double((batch + 31) / 32) * 128.0 / (128.0 * 2.0 * sm_count());
    const double slices = double((f.cols + 1399) / 1400);
    const double unit_ns = 0.75 * 137.0 * (2.0 * f.nch_max / slices + 12.0);
    const double others_ns =
        streams ? 4600.0 + (f.bf16 ? 1.5 : 2.3) * gather_ns
                : std::min(0.95 * (3000.0 + (aligned ? 0.0 : 2500.0) + 1.66 * double(f.cols) / slices +
                                   std::max(unit_ns, 1.6 * gather_ns)),
                           f.bf16 ? xres::expected_ns<true, 32>(f, batch, aligned)
                                  : xres::expected_ns<false, 32>(f, batch, aligned));
    cudaError_t e = launch_spmm_rows(f, X, ldx, batch, Y, ldy, early, 0.95 * others_ns, stream);
    if (e != cudaErrorNotSupported) return e;
    cudaGetLastError();
    if (!streams) {
        e = f.bf16 ? xres::launch<true, 32>(f, X, ldx, batch, Y, ldy, early, stream)
                   : xres::launch<false, 32>(f, X, ldx, batch, Y, ldy, early, stream);
        if (e != cudaErrorNotSupported) return e;
        cudaGetLastError();
    }
    const RnnArgs none{};
    return f.bf16 ? batch::launch_any<true, kModeY>(f, X, ldx, batch, Y, ldy, none, early, stream)
                  : batch::launch_any<false, kModeY>(f, X, ldx, batch, Y, ldy, none, early, stream);
}

cudaError_t launch_spmm_on(const Format &f, Kernel kernel, const float *X, int64_t ldx, int64_t batch, float *Y,
                           int64_t ldy, bool early, cudaStream_t stream) {
    const RnnArgs none{};
    switch (kernel) {
        case kKernelRows: return launch_spmm_rows(f, X, ldx, batch, Y, ldy, early, 1e300, stream);
        case kKernelBatch:
            return f.bf16 ? batch::launch_any<true, kModeY>(f, X, ldx, batch, Y, ldy, none, early, stream)
                          : batch::launch_any<false, kModeY>(f, X, ldx, batch, Y, ldy, none, early, stream);
        case kKernelXres:
            if (!xres::maps(X, ldx)) return cudaErrorNotSupported;
            return f.bf16 ? xres::launch_as<true, 32, false>(f, X, ldx, batch, Y, ldy, early, stream)
                          : xres::launch_as<false, 32, false>(f, X, ldx, batch, Y, ldy, early, stream);
        case kKernelXresPlain:
            return f.bf16 ? xres::launch_as<true, 32, true>(f, X, ldx, batch, Y, ldy, early, stream)
                          : xres::launch_as<false, 32, true>(f, X, ldx, batch, Y, ldy, early, stream);
        default: return cudaErrorNotSupported;
    }
}

cudaError_t launch_spmm_prefix(const Format &f, int64_t col_limit, const float *X, int64_t ldx, int64_t batch,
                               float *Y, int64_t ldy, bool early, cudaStream_t stream) {
    if (batch > 16 && col_limit > 0 && col_limit < f.cols) {
        // xres on a view of the matrix `col_limit` columns wide: its column slices
        // cover [0, col_limit) only, a block that reaches past it reads rows that
        // lie outside the view's tensor map, i.e. zeros, and the blocks that start
        // past it are in no slice
        Format fx = f;
        fx.cols = col_limit;
        const cudaError_t e = f.bf16 ? xres::launch<true, 32>(fx, X, ldx, batch, Y, ldy, early, stream)
                                     : xres::launch<false, 32>(fx, X, ldx, batch, Y, ldy, early, stream);
        if (e == cudaErrorNotSupported) cudaGetLastError();
        return e;
    }
    return cudaErrorNotSupported;
}

}  // namespace darb
