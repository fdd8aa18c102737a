// rnn_batch.cu -- the batch > 4 RNN steps (batch.cuh in LSTM / GRU mode).
#include "batch.cuh"

namespace darb {

cudaError_t launch_rnn_batch(const Format &f, const RnnArgs &ra, int mode, bool early, cudaStream_t stream) {
    if (mode == kModeLstm)
        return f.bf16 ? batch::launch_any<true, kModeLstm>(f, nullptr, 0, ra.B, nullptr, 0, ra, early, stream)
                      : batch::launch_any<false, kModeLstm>(f, nullptr, 0, ra.B, nullptr, 0, ra, early, stream);
    return f.bf16 ? batch::launch_any<true, kModeGru>(f, nullptr, 0, ra.B, nullptr, 0, ra, early, stream)
                  : batch::launch_any<false, kModeGru>(f, nullptr, 0, ra.B, nullptr, 0, ra, early, stream);
}

// By the tile that launch_any takes (batch.cuh): a fixed part, per tile the kept
// weights (in thousands; more for fp32 and for a GRU) and the chunks of the
// longest row, and the gate sums that go through scratch (hundreds).  Fitted to
// 36 gate matrices at 13 batches from 8 to 128: 11 to 15% root mean square (the
// LSTM's 32-column tile raised by 13%: its fit was up to 30% low near the border).
// Without tensor maps (a batch that is no multiple of 4) the kernel's one
// copying warp makes it 2 to 10 times slower: never then.
double rnn_batch_ns(const Format &f, const RnnArgs &ra, int mode) {
    struct Cost {
        double fixed, weights, f32, gru, longest, sums;
    };
    static constexpr Cost k16 = {7360, 4.26, 0.68, 0.57, 42.5, 4.63}, k32Lstm = {12700, 6.80, 10.7, 0, 116, 3.40},
                          k32Gru = {8750, 11.69, 0, 0, 113.8, 4.63}, k64 = {10880, 14.08, 3.32, 0, 30.4, 1.94};
    const bool aligned = ra.B % 4 == 0 && (ra.I == 0 || reinterpret_cast<uintptr_t>(ra.x) % 16 == 0) &&
                         reinterpret_cast<uintptr_t>(ra.h) % 16 == 0;
    if (!aligned) return 1e300;
    const bool gru = mode == kModeGru;
    const bool narrow = ra.B <= 16 || f.m_max > batch::max_block<8, 4>(true);
    const bool wide = !narrow && ra.B > 32 && !gru && f.m_max <= batch::max_block<8, 8>(true);
    const Cost &c = narrow ? k16 : wide ? k64 : gru ? k32Gru : k32Lstm;
    const int bt = narrow ? 16 : wide ? 64 : 32;
    const double tiles = double((ra.B + bt - 1) / bt);
    const double kept = double(f.set_prefix[0][f.nitems[0][0]]) * kSlots * kChunk / 1000.0;
    return c.fixed + tiles * ((c.weights + (f.bf16 ? 0 : c.f32) + (gru ? c.gru : 0)) * kept + c.longest * f.nch_max) +
           c.sums * double(f.rows) * double(ra.B) / 100.0;
}

}  // namespace darb
