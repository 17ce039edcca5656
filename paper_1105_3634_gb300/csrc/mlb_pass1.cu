// mlb_pass1.cu -- launchers of pass 1 of a time step (device code in
// mlb_pass1.cuh): the exact pass and the learned surrogate's variant, for one
// and two species; mlb_pass1_s3.cu and mlb_pass1_s4.cu hold the others (each
// species count is a compilation unit of its own, the kernels are large).
#include "mlb_pass1.cuh"

namespace {

template <int S, int R, bool DRAG, int TX = mlbi_tile_of(S, R).tx>
cudaError_t launch_pass1_group(const mlbi_group &g, cudaStream_t s)
{
    if constexpr (TX == kBX && R == 1)
        if (g.tile_x == 16) return launch_pass1_group<S, R, DRAG, 16>(g, s);
    using T = TileOf<S, R, TX>;
    auto k = k_pass1_group<S, R, DRAG, TX>;
    cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)T::bytes);
    if (e != cudaSuccess) return e;
    k<<<(unsigned)g.nblk[MLBI_GROUP_PASS1], dim3(kBX, T::NTH / kBX), T::bytes, s>>>(g.mem, g.blk[MLBI_GROUP_PASS1]);
    return cudaGetLastError();
}

template <int S, int R>
cudaError_t launch_pass1_group_r(const mlbi_group &g, cudaStream_t s)
{
    return g.drag ? launch_pass1_group<S, R, true>(g, s) : launch_pass1_group<S, R, false>(g, s);
}

}  // namespace

cudaError_t mlbi_launch_group_pass1(const mlbi_group &g, cudaStream_t s)
{
    if (g.nblk[MLBI_GROUP_PASS1] < 1) return cudaErrorInvalidValue;
    if (g.S == 1) return g.R == 1 ? launch_pass1_group_r<1, 1>(g, s) : launch_pass1_group_r<1, 2>(g, s);
    if (g.S == 2) return g.R == 1 ? launch_pass1_group_r<2, 1>(g, s) : launch_pass1_group_r<2, 2>(g, s);
    return cudaErrorInvalidValue;
}

template <>
cudaError_t mlbi_pass1_species<1>(const mlbi_params &p, const mlbi_buffers &b, cudaStream_t s)
{
    return pass1_species<1>(p, b, s);
}
template <>
cudaError_t mlbi_pass1_species<2>(const mlbi_params &p, const mlbi_buffers &b, cudaStream_t s)
{
    return pass1_species<2>(p, b, s);
}

cudaError_t mlbi_launch_pass1(const mlbi_params &p, const mlbi_buffers &b, cudaStream_t s)
{
    MLBI_DISPATCH_S(return mlbi_pass1_species<SS>(p, b, s));
    return cudaErrorInvalidValue;
}
