// rnn_step.cu -- instantiations of the local-cell RNN step and of the product on
// the same kernel (rnn_step.cuh).
#include "rnn_step.cuh"

namespace darb {

cudaError_t launch_rnn_step(const Format &f, const RnnArgs &ra, int mode, bool early, double limit_ns,
                            cudaStream_t stream) {
    if (mode == kModeLstm)
        return f.bf16 ? step::launch<true, kModeLstm>(f, ra, early, stream, 0, 0, limit_ns)
                      : step::launch<false, kModeLstm>(f, ra, early, stream, 0, 0, limit_ns);
    return f.bf16 ? step::launch<true, kModeGru>(f, ra, early, stream, 0, 0, limit_ns)
                  : step::launch<false, kModeGru>(f, ra, early, stream, 0, 0, limit_ns);
}

cudaError_t launch_spmm_rows(const Format &f, const float *X, int64_t ldx, int64_t batch, float *Y, int64_t ldy,
                             bool early, double limit_ns, cudaStream_t stream) {
    RnnArgs ra{};
    ra.x = X;
    ra.h = X;
    ra.h_out = Y;
    ra.H = static_cast<int>(f.rows);
    ra.I = static_cast<int>(f.cols);
    ra.B = batch;
    return f.bf16 ? step::launch<true, kModeY>(f, ra, early, stream, ldx, ldy, limit_ns)
                  : step::launch<false, kModeY>(f, ra, early, stream, ldx, ldy, limit_ns);
}

}  // namespace darb
