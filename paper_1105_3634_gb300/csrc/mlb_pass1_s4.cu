// mlb_pass1_s4.cu -- pass 1 for four species (mlb_pass1.cuh).
#include "mlb_pass1.cuh"

template <>
cudaError_t mlbi_pass1_species<4>(const mlbi_params &p, const mlbi_buffers &b, cudaStream_t s)
{
    return pass1_species<4>(p, b, s);
}
