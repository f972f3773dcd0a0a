// Kernels and launchers of Q_Naive for tensors of bfloat16.
#include "qnaive.cuh"

namespace tahq {
TAHQ_INSTANTIATE_QNAIVE(true)
}
