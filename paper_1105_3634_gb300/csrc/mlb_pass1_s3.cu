// mlb_pass1_s3.cu -- pass 1 for three species (mlb_pass1.cuh).
#include "mlb_pass1.cuh"

template <>
cudaError_t mlbi_pass1_species<3>(const mlbi_params &p, const mlbi_buffers &b, cudaStream_t s)
{
    return pass1_species<3>(p, b, s);
}
