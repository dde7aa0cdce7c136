// da_batch_traced.cu -- the batched launch's kernels that store the flipped index of every
// step (da_batch.cuh), loaded when a class with a traced item first runs.
#include "da_batch.cuh"

namespace da {

BatchKernel traced_smem_kernel_for(int wk, int V) { return batch_detail::smem_kernel_for<true>(wk, V); }
BatchKernel traced_kernel_for(int wk, int V, bool coal) { return batch_detail::kernel_for<true>(wk, V, coal); }

}  // namespace da
