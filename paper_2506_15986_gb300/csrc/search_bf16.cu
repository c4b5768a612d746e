// search_bf16.cu -- instances of the search kernel (one file per group of storage
// types, so that they compile side by side).
#include "search_kernel.cuh"

namespace ann {

ANN_SEARCH_INSTANCE(, ANN_BF16, ANN_L2)
ANN_SEARCH_INSTANCE(, ANN_BF16, ANN_IP)

}  // namespace ann
