// mlb_pass2.cu -- launchers of pass 2 and of pass 2 fused with the collision
// (device code in mlb_pass2.cuh) for one and two species and for groups; the
// other species counts in mlb_pass2_s3.cu and mlb_pass2_s4.cu.
#include "mlb_pass2.cuh"

namespace {

template <int S>
bool collide_fits(int tile_r)
{
    if (tile_r == 1) return FusedTile<S, 1>::bytes <= kMaxSharedPerBlock;
    return tile_r == 2 && S <= 2;              // more species: one block of four warps per SM, the split launches are faster
}

template <int S, int R, bool DRAG, int TX = kBX>
cudaError_t launch_pass2_collide_group(const mlbi_group &g, int odd, cudaStream_t s)
{
    using G = TmaTile<S, R, TX>;
    if constexpr (G::bytes + sizeof(mlbi_params) > kMaxSharedPerBlock) {
        return cudaErrorInvalidValue;
    } else {
        if constexpr (TX == kBX && R == 1)
            if (g.tile_x == 16) return launch_pass2_collide_group<S, R, DRAG, 16>(g, odd, s);
        auto k = k_pass2_collide_group<S, R, DRAG, TX>;
        cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)G::bytes);
        if (e != cudaSuccess) return e;
        k<<<(unsigned)g.nblk[MLBI_GROUP_PASS2], dim3(kBX, kBY), G::bytes, s>>>(g.mem, g.blk[MLBI_GROUP_PASS2], odd);
        return cudaGetLastError();
    }
}

template <int S, int R>
cudaError_t launch_pass2_collide_group_r(const mlbi_group &g, int odd, cudaStream_t s)
{
    return g.drag ? launch_pass2_collide_group<S, R, true>(g, odd, s)
                  : launch_pass2_collide_group<S, R, false>(g, odd, s);
}

}  // namespace

MLBI_PASS2_UNIT(1)
MLBI_PASS2_UNIT(2)

cudaError_t mlbi_launch_group_pass2_collide(const mlbi_group &g, int odd, cudaStream_t s)
{
    if (g.nblk[MLBI_GROUP_PASS2] < 1) return cudaErrorInvalidValue;
    if (g.S == 1) return g.R == 1 ? launch_pass2_collide_group_r<1, 1>(g, odd, s)
                                  : launch_pass2_collide_group_r<1, 2>(g, odd, s);
    if (g.S == 2) return g.R == 1 ? launch_pass2_collide_group_r<2, 1>(g, odd, s)
                                  : launch_pass2_collide_group_r<2, 2>(g, odd, s);
    return cudaErrorInvalidValue;
}

bool mlbi_group_supported(const mlbi_params &p, const mlbi_buffers &b)
{
    if (p.S < 1 || p.S > 2 || !p.local_g || p.hc_from_attr || !b.maps || !b.maps->ok) return false;
    if (p.tile_r != 1 && p.tile_r != 2) return false;
    return mlbi_pass2_collide_supported(p);
}

void mlbi_group_grid(const mlbi_params &p, int stage, int grid[3])
{
    const int zc = (p.nz + p.zchunk - 1) / p.zchunk;
    if (stage == MLBI_GROUP_MOMENTS) {
        grid[0] = (int)grid_for(p.N);
        grid[1] = grid[2] = 1;
    } else {
        const int ty = mlbi_tile_rows(p);      // reach 1, 2: the same tiles in both passes
        grid[0] = (p.nx + p.tile_x - 1) / p.tile_x;
        grid[1] = (p.ny + ty - 1) / ty;
        grid[2] = zc;
    }
}

cudaError_t mlbi_launch_pass2(const mlbi_params &p, const mlbi_buffers &b, double *acc_out, cudaStream_t s)
{
    MLBI_DISPATCH_S(return mlbi_pass2_species<SS>(p, b, acc_out, s));
    return cudaErrorInvalidValue;
}

bool mlbi_pass2_collide_supported(const mlbi_params &p)
{
    switch (p.S) {
    case 1: return collide_fits<1>(p.tile_r);
    case 2: return collide_fits<2>(p.tile_r);
    case 3: return collide_fits<3>(p.tile_r);
    case 4: return collide_fits<4>(p.tile_r);
    default: return false;
    }
}

cudaError_t mlbi_launch_pass2_collide(const mlbi_params &p, const mlbi_buffers &b, int cur, cudaStream_t s)
{
    MLBI_DISPATCH_S(return mlbi_pass2_collide_species<SS>(p, b, cur, s));
    return cudaErrorInvalidValue;
}
