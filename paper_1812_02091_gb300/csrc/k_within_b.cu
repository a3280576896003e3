// Launcher of the pruned top-K's second stage (see k_sparse_dev.cuh); a translation unit of its
// own so that the build compiles its template instances beside the others.
#include "k_sparse_dev.cuh"

namespace emd {

cudaError_t launch_rev_within_b(int meas, int k, const QDesc* qd, const int* nq, int nb, const int32_t* row_ptr,
                                const int32_t* col, const float* val, int64_t n, int K, cudaStream_t st)
{
    if (nb <= 0 || n <= 0) return cudaSuccess;
    switch (meas) {
    case M_RWMD: return rev_within_meas_b<M_RWMD>(k, qd, nq, nb, row_ptr, col, val, n, K, st);
    case M_OMR: return rev_within_meas_b<M_OMR>(k, qd, nq, nb, row_ptr, col, val, n, K, st);
    case M_ICT: return rev_within_meas_b<M_ICT>(k, qd, nq, nb, row_ptr, col, val, n, K, st);
    default: return rev_within_meas_b<M_ACT>(k, qd, nq, nb, row_ptr, col, val, n, K, st);
    }
}

}  // namespace emd
