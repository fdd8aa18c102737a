// rnn_step.cu -- instantiations of the local-cell RNN step (rnn_step.cuh).
#include "rnn_step.cuh"

namespace darb {

cudaError_t launch_rnn_step(const Format &f, const RnnArgs &ra, int mode, bool early, cudaStream_t stream) {
    if (mode == kModeLstm)
        return f.bf16 ? step::launch<true, kModeLstm>(f, ra, early, stream)
                      : step::launch<false, kModeLstm>(f, ra, early, stream);
    return f.bf16 ? step::launch<true, kModeGru>(f, ra, early, stream)
                  : step::launch<false, kModeGru>(f, ra, early, stream);
}

}  // namespace darb
