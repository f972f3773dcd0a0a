// Kernels and launchers of Q_Naive for tensors of binary32.
#include "qnaive.cuh"

namespace tahq {
TAHQ_INSTANTIATE_QNAIVE(false)
}
