// knn_u8.cu -- exact k-NN: uint8 rows (a file of its own, so that the kernels
// compile side by side).
#include "knn_kernel.cuh"

namespace ann {

ann_status knn_exact_u8(const uint8_t *base, int64_t n, int dim, const uint8_t *queries, int64_t nq, int k,
                        bool exclude_self, int32_t *d_ids, void *d_dists, cudaStream_t s)
{
    return knn_by_k<uint8_t, 1>(base, n, dim, ANN_L2, queries, nq, k, exclude_self, d_ids, d_dists, s);
}

}  // namespace ann
