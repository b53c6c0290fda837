// mcd_collide_f32c16.cu -- the mixed-precision chain variants (specialised warps) of
// up to 512 swarms, every dv-matrix store, with and without the fragmentation ramp
// and the tracer, in a translation unit of their own so that the build
// compiles the variants in parallel.
#include "mcd_collide_chain.cuh"

namespace mcd {

template <>
cudaError_t collide_chain_variant<16, 1>(int op, int store, bool ramp, bool tracer, unsigned grid, int nthr,
                                        size_t smem, cudaStream_t st, const CollideArgs *A, int *out)
{
    switch (store) {
    case 0: return collide_chain_store<16, 1, 0>(op, ramp, tracer, grid, nthr, smem, st, A, out);
    case 1: return collide_chain_store<16, 1, 1>(op, ramp, tracer, grid, nthr, smem, st, A, out);
    case 2: return collide_chain_store<16, 1, 2>(op, ramp, tracer, grid, nthr, smem, st, A, out);
    default: return cudaErrorInvalidValue;
    }
}

}  // namespace mcd
