// knn.cu -- exact k-NN: fp32 rows, and the choice of the type.
#include "knn_kernel.cuh"

namespace ann {

ann_status knn_exact_u8(const uint8_t *base, int64_t n, int dim, const uint8_t *queries, int64_t nq, int k,
                        bool exclude_self, int32_t *d_ids, void *d_dists, cudaStream_t s);  // knn_u8.cu

ann_status knn_exact(const void *d_base, int64_t n, int dim, int dtype, int metric, const void *d_queries,
                     int64_t nq, int k, bool exclude_self, int32_t *d_ids, void *d_dists, cudaStream_t s)
{
    if (dtype == ANN_U8)
        return knn_exact_u8(static_cast<const uint8_t *>(d_base), n, dim, static_cast<const uint8_t *>(d_queries), nq,
                            k, exclude_self, d_ids, d_dists, s);
    if (dtype != ANN_F32)
        return ANN_ERR_UNSUPPORTED;
    return knn_by_k<float, 3>(static_cast<const float *>(d_base), n, dim, metric, static_cast<const float *>(d_queries),
                              nq, k, exclude_self, d_ids, d_dists, s);
}

}  // namespace ann
