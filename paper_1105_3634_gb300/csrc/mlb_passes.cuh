// mlb_passes.cuh -- device code shared by the two force passes of a time step
// (mlb_pass1.cuh, mlb_pass2.cuh): packed FP32 pairs, the shared-memory
// z-marching tiles and the offset classes of the 3x3x3 cube.  Internal header.
#pragma once

#include "mlb_internal.h"
#include "mlb_device.cuh"

#include <type_traits>

namespace {

// ------------------------------------------------------------------ packed FP32 pairs
// Pass 1 accumulates in lane pairs so that one packed instruction (two IEEE
// FP32 operations, each rounded as the scalar one) serves two sums:
//   hf[q] = (F^hc_q, F^v_q) per component q, and the friction matrix as
//   G[0] = (xx, yy), G[1] = (zz, xy), G[2] = (xz, yz).
__device__ __forceinline__ float2 f2(float x, float y) { return make_float2(x, y); }
__device__ __forceinline__ float2 fma2(float2 a, float2 b, float2 c) { return __ffma2_rn(a, b, c); }
__device__ __forceinline__ float2 mul2(float2 a, float2 b) { return __fmul2_rn(a, b); }
__device__ __forceinline__ float2 add2(float2 a, float2 b) { return __fadd2_rn(a, b); }

// ------------------------------------------------------------------ shared-memory tiles (z marching)
// A block owns a TX x TY column of sites (TX = 32 or 16), SPLIT threads to a site, and
// marches up z through `zchunk` planes.  The stencil field of every species (float4: the
// moments in pass 1, (n - n_ref, u*) in pass 2) and the contact-value
// deviations of every pair are staged in shared memory as a ring of planes
// of (TX + 2R) x (TY + 2R) sites: 2R + 1 planes in use and one more being
// filled by cp.async while the current plane is computed.  Every shell
// neighbour is then read from shared memory.
// ALT (16-wide tiles of pass 1, the sweeps and the split pass 2; the fused tiles do
// without): a warp's two rows of 16 sites are two apart and the rows of the contact
// values 24 floats, so that their 4-byte loads meet in no bank (rows one apart at a
// pitch of 18 share 2 banks of 16, of 22 6, an extra wavefront per load): 256 x 16^3
// 0.247 -> 0.242 ms per step, three species at reach 3 (512 x 64 x 64) pass 2 1.061 -> 1.049.
template <int S, int R, int TY_ = kBY, int TX_ = kBX, int SPLIT_ = 1, bool ALT = false>
struct Tile {
    static constexpr int TX = TX_, TY = TY_, SPLIT = SPLIT_;
    static constexpr int TXH = TX + 2 * R, TYH = TY + 2 * R, PLANE = TXH * TYH;
    static_assert(!ALT || (TX == 16 && TXH <= 24 && TY % 4 == 0), "two rows per warp");
    static constexpr int GP = ALT ? 24 : TXH, GPLANE = GP * TYH;      // rows and planes of the contact values
    static constexpr int NSLOT = 2 * R + 2;
    static constexpr int NP = S * (S + 1) / 2;
    static constexpr int NT = TX * TY;                       // sites
    static constexpr int NTH = NT * SPLIT;                   // threads: `split` per site, whole warps each
    static_assert(NT % 32 == 0, "a warp has one part");
    static constexpr int J = (PLANE + NTH - 1) / NTH;        // staging sites per thread and plane
    static constexpr size_t ring = NSLOT * ((size_t)PLANE * S * sizeof(float4) + (size_t)GPLANE * NP * sizeof(float));
    static constexpr size_t bytes = ring + (size_t)(SPLIT - 1) * NT * 12 * S * sizeof(float);   // + partial sums
    // resident blocks: what the tile's shared memory allows, 16 warps (128 registers) at most
    static constexpr int by_smem = (int)((228 * 1024) / (bytes + 1024)), by_warps = NTH >= 512 ? 1 : 512 / NTH;
    static constexpr int blocks = by_smem < 1 ? 1 : (by_smem < by_warps ? by_smem : by_warps);
    // this thread's site of the tile, and its part of the site's shell sums
    static __device__ __forceinline__ int tid() { return threadIdx.y * kBX + threadIdx.x; }
    static __device__ __forceinline__ int sid() { return SPLIT == 1 ? tid() : tid() % NT; }
    static __device__ __forceinline__ int part() { return SPLIT == 1 ? 0 : tid() / NT; }
    static __device__ __forceinline__ int lx() { return TX == kBX ? threadIdx.x : sid() % TX; }
    static __device__ __forceinline__ int ly()
    {
        if (TX == kBX && SPLIT == 1) return threadIdx.y;
        const int s = sid();
        return ALT ? (s >> 6) * 4 + ((s >> 5) & 1) + ((s >> 4) & 1) * 2 : s / TX;
    }
    // the site in a staged plane of the fields and of the contact values
    static __device__ __forceinline__ int cidx() { return (ly() + R) * TXH + lx() + R; }
    static __device__ __forceinline__ int gidx() { return (ly() + R) * GP + lx() + R; }
};

// The tile of (S, R); reach 1 of one and two species also comes 16 x 8
template <int S, int R, int TX>
using TileOf = Tile<S, R, R == 1 ? 128 / TX : mlbi_tile_of(S, R).ty, TX, mlbi_tile_of(S, R).split, TX == 16>;

// The shell groups of the reach-3 tiles, staged once per block into shared
// memory after the tile where they fit (one block per SM holds the tile anyway),
// read there instead of through the L1.  Host and device agree on the size.
template <class T, int R>
__host__ __device__ inline size_t staged_table_bytes(const mlbi_params &p)
{
    if (R != 3) return 0;
    const size_t b = (size_t)p.grp[p.S - 1][7] * 2 * sizeof(mlbi_entry);
    return T::bytes + b <= MLBI_MAX_TILE_BYTES ? b : 0;
}
// copy the groups to dst (visible after the caller's next barrier); returns
// the table the shell loops read
template <class T, int R>
__device__ inline const mlbi_entry *stage_table(const mlbi_params &p, const mlbi_entry *tab, float4 *dst)
{
    tab += p.grp_at;
    if (staged_table_bytes<T, R>(p) == 0) return tab;
    for (int e = T::tid(); e < 2 * p.grp[p.S - 1][7]; e += T::NTH) dst[e] = __ldg(&tab[e]);
    return dst;
}

// (x, y) offsets x + nx y of this thread's staging sites, fixed while the
// block marches up z; -1 beyond a wall
template <class T, int R>
__device__ __forceinline__ void stage_sites(const mlbi_params &p, int x0, int y0, int (&xy)[T::J])
{
    const int tid = T::tid();
#pragma unroll
    for (int j = 0; j < T::J; ++j) {
        const int idx = tid + j * T::NTH;
        const int hx = idx % T::TXH, hy = idx / T::TXH;
        const int x = wrap_or_out(x0 - R + hx, p.nx, p.wall_axis == 0);
        const int y = wrap_or_out(y0 - R + hy, p.ny, p.wall_axis == 1);
        xy[j] = (x < 0 || y < 0) ? -1 : x + p.nx * y;
    }
}

// plane index with one periodic wrap (|overhang| <= R < extent), or -1 beyond a wall
__device__ __forceinline__ int wrap_plane(int c, int L, bool wall)
{
    if (wall) return (c < 0 || c >= L) ? -1 : c;
    return c < 0 ? c + L : (c >= L ? c - L : c);
}

// Stage plane gz of the tile into ring slot `slot`.  Sites beyond a wall get
// n = 0 (n - n_ref = -n_ref) and zero velocity; their dg is never used (every
// term carries n(r+d) = 0) and is set to 0.
template <class T, int S>
__device__ __forceinline__ void stage_plane(const mlbi_params &p, const int (&xy)[T::J], int gz, int slot,
                                            const float4 *__restrict__ fld, const float *__restrict__ dg, float4 *sf,
                                            float *sg)
{
    const long long N = p.N;
    const int tid = T::tid();
    const int z = wrap_plane(gz, p.nz, p.wall_axis == 2);
    const long long zoff = (long long)p.nx * p.ny * z;
#pragma unroll
    for (int j = 0; j < T::J; ++j) {
        const int idx = tid + j * T::NTH;
        if (j == T::J - 1 && idx >= T::PLANE) break;
        float4 *df = sf + (size_t)slot * S * T::PLANE + idx;
        float *dgs = sg + (size_t)slot * T::NP * T::GPLANE + (T::GP == T::TXH ? idx : idx / T::TXH * T::GP + idx % T::TXH);
        if (xy[j] < 0 || z < 0) {
#pragma unroll
            for (int b = 0; b < S; ++b) df[b * T::PLANE] = make_float4(-p.nref[b], 0.f, 0.f, 0.f);
#pragma unroll
            for (int q = 0; q < T::NP; ++q) dgs[q * T::GPLANE] = 0.f;
        } else {
            const long long g = zoff + xy[j];
#pragma unroll
            for (int b = 0; b < S; ++b) cp_async16(df + b * T::PLANE, fld + b * N + g);
#pragma unroll
            for (int q = 0; q < T::NP; ++q) cp_async4(dgs + q * T::GPLANE, dg + q * N + g);
        }
    }
}

// ------------------------------------------------------------------ the 3x3x3 cube
// The 13 canonical half offsets (first non-zero of (dz, dy, dx) positive).
// With reach 1 every contact shell is a union of the three classes |d|^2 = 1
// (axis), 2 (face diagonal), 3 (corner); the bit of class CL in cube_mask is
// the bit of its first offset.
__host__ __device__ constexpr int cls_bit(int cl) { return cl == 0 ? 0 : (cl == 1 ? 1 : 4); }
__host__ __device__ constexpr float cls_il(int cl)   // 1/|d|
{
    return cl == 0 ? 1.0f : (cl == 1 ? 0.70710678118654752f : 0.57735026918962576f);
}

}  // namespace

#define MLBI_DISPATCH_S(...)                                                                       \
    switch (p.S) {                                                                                 \
    case 1: { constexpr int SS = 1; __VA_ARGS__; } break;                                          \
    case 2: { constexpr int SS = 2; __VA_ARGS__; } break;                                          \
    case 3: { constexpr int SS = 3; __VA_ARGS__; } break;                                          \
    case 4: { constexpr int SS = 4; __VA_ARGS__; } break;                                          \
    default: return cudaErrorInvalidValue;                                                         \
    }
