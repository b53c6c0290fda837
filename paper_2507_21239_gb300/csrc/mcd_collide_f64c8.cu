// mcd_collide_f64c8.cu -- the FP64 chain variants (specialised warps) of up to
// 256 swarms, with and without the stored matrix, the fragmentation ramp and the
// tracer, in a translation unit of their own so that the build compiles the
// variants in parallel.
#include "mcd_collide_chain64.cuh"

namespace mcd {

template <>
cudaError_t collide_chain64_variant<8>(int op, int store, bool ramp, bool tracer, unsigned grid, int nthr,
                                       size_t smem, cudaStream_t st, const CollideArgs *A, int *out)
{
    switch (store) {
    case 0: return collide_chain64_store<8, 0>(op, ramp, tracer, grid, nthr, smem, st, A, out);
    case 2: return collide_chain64_store<8, 2>(op, ramp, tracer, grid, nthr, smem, st, A, out);
    default: return cudaErrorInvalidValue;
    }
}

}  // namespace mcd
