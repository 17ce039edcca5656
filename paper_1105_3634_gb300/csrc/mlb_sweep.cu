// mlb_sweep.cu -- further Jacobi sweeps of the half step of the semi-implicit
// forcing (Eq. evolution with the half-force shift): u* = u + a(u*)/2 solved
// at every site as (I + Gamma/2) du = (F^hc + G + F_ext + F^v)/2, where the
// velocity exchange F^v (Eqs. gammaab, viscousforce) now takes the partners'
// velocities from the previous sweep's u*.  Pass 1 is the first sweep; each
// further sweep is one more pass over the contact shells (device code in
// mlb_pass1.cuh, mode kSweep).  One and two species here, the others in
// mlb_sweep_s3.cu and mlb_sweep_s4.cu.
#include "mlb_pass1.cuh"

template <>
cudaError_t mlbi_sweep_species<1>(const mlbi_params &p, const mlbi_buffers &b, const float4 *prev, float4 *next,
                                  cudaStream_t s)
{
    return sweep_species<1>(p, b, prev, next, s);
}
template <>
cudaError_t mlbi_sweep_species<2>(const mlbi_params &p, const mlbi_buffers &b, const float4 *prev, float4 *next,
                                  cudaStream_t s)
{
    return sweep_species<2>(p, b, prev, next, s);
}

cudaError_t mlbi_launch_sweep(const mlbi_params &p, const mlbi_buffers &b, const float4 *prev, float4 *next,
                              cudaStream_t s)
{
    MLBI_DISPATCH_S(return mlbi_sweep_species<SS>(p, b, prev, next, s));
    return cudaErrorInvalidValue;
}
