// mlb_sweep_s3.cu -- further sweeps of the half step for three species (mlb_pass1.cuh).
#include "mlb_pass1.cuh"

template <>
cudaError_t mlbi_sweep_species<3>(const mlbi_params &p, const mlbi_buffers &b, const float4 *prev, float4 *next,
                                  cudaStream_t s)
{
    return sweep_species<3>(p, b, prev, next, s);
}
