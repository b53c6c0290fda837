// mcd_collide_f32s1.cu -- the mixed-precision block variant with one swarm per
// thread and the shared-memory matrix (with and without the fragmentation ramp
// and the tracer).  It runs where the chain variants' ready outcomes leave no
// room for the matrix beside them (cells of about 290 to 318 swarms) and the
// shared-memory matrix is asked for.
#include "mcd_collide.cuh"

namespace mcd {

template <>
cudaError_t collide_variant<1, false>(int op, int store, bool ramp, bool tracer, unsigned grid, int nthr,
                                        size_t smem, cudaStream_t st, const CollideArgs *A, int *out)
{
    if (store != 1) return cudaErrorInvalidValue;
    return collide_variant_store<1, 1, false>(op, ramp, tracer, grid, nthr, smem, st, A, out);
}

}  // namespace mcd
