// mlb_pass2.cuh -- pass 2 of a time step on sm_103a: the velocity exchange
// (Eqs. gammaab, viscousforce) at the predicted velocities u* of pass 1,
// completed to the acceleration a^a = frest^a + sum_points s sd (masses 1).
// Same three variants as pass 1: global memory and tile (reach 2, 3) with the
// sign groups, compile-time 3x3x3 cube (reach 1).  The tiled variants also come
// fused with the collision (k_pass2_collide): the acceleration is not stored,
// the same thread collides and streams its site right away (the collision
// needs only the site's own acceleration).
#pragma once

#include "mlb_passes.cuh"
#include "mlb_cube.cuh"
#include "mlb_groups.cuh"
#include "mlb_collide.cuh"

namespace {

template <int S>
__device__ __forceinline__ void store_acc(const mlbi_params &p, long long r, const float (&acc)[S][3],
                                          float4 *__restrict__ acc_f, double *__restrict__ acc_out)
{
    const long long N = p.N;
#pragma unroll
    for (int a = 0; a < S; ++a) {
        if (acc_out) {
#pragma unroll
            for (int q = 0; q < 3; ++q) acc_out[(a * 3 + q) * N + r] = (double)acc[a][q];
        } else {
            acc_f[a * N + r] = make_float4(acc[a][0], acc[a][1], acc[a][2], 0.f);
        }
    }
}

template <int S>
__device__ __forceinline__ void zero_acc(float (&acc)[S][3])
{
#pragma unroll
    for (int a = 0; a < S; ++a) acc[a][0] = acc[a][1] = acc[a][2] = 0.f;
}

// the rest force F^hc + G + F_ext is added after the shell sums (the same
// order in every variant, so the fused and split launches agree bit for bit)
__device__ __forceinline__ void add_rest(float (&acc)[3], const float4 fr)
{
    acc[0] = fr.x + acc[0];
    acc[1] = fr.y + acc[1];
    acc[2] = fr.z + acc[2];
}

// a^a = frest^a + vx_ab sum_{+-d} s s.[(g(r)+g(r+d))/2 n^b(r+d) (u*^b(r+d) - u*^a(r))]
// from global memory: 32 sites a block, kParts threads per site (as k_pass1).  Five
// blocks per SM, four for four species (416 bytes of spills at five, 24 at four).
constexpr int kParts2 = 4;
template <int S, bool DRAG>
__global__ void __launch_bounds__(32 * kParts2, S == 4 && !DRAG ? 4 : 5) k_pass2(const mlbi_params p, const float *__restrict__ dg,
                                                           const mlbi_entry *__restrict__ tab,
                                                           const float4 *__restrict__ frest,
                                                           const float4 *__restrict__ pst, float4 *__restrict__ acc_f,
                                                           double *__restrict__ acc_out)
{
    step_begin();
    __shared__ float red[kParts2 - 1][3 * S][32];
    const long long N = p.N, r = blockIdx.x * 32ll + threadIdx.x;
    const int part = threadIdx.y, lane = threadIdx.x;
    const bool active = r < N;
    float acc[S][3];
    zero_acc<S>(acc);
    if (active) {
        const GlobalView<S> view{p, pst, dg, (int)(r % p.nx), (int)(r / p.nx % p.ny), (int)(r / ((long long)p.nx * p.ny))};
        p2_groups<S, kParts2, DRAG>(p, tab + p.grp_at, view, part, acc);
        if (part > 0)
#pragma unroll
            for (int k = 0; k < 3 * S; ++k) red[part - 1][k][lane] = acc[k / 3][k % 3];
    }
    __syncthreads();
    if (!active || part > 0) return;
#pragma unroll
    for (int q = 0; q < kParts2 - 1; ++q)
#pragma unroll
        for (int k = 0; k < 3 * S; ++k) acc[k / 3][k % 3] += red[q][k][lane];
#pragma unroll
    for (int a = 0; a < S; ++a) add_rest(acc[a], frest[a * N + r]);
    store_acc<S>(p, r, acc, acc_f, acc_out);
}

// ------------------------------------------------------------------ tiled variants
// reach 1 (mlb_cube.cuh)
template <int S, bool DRAG, class T, int NSL = 4>
__device__ __forceinline__ void pass2_cube(const mlbi_params &p, const float4 *sf, const float *sg, int kz, int cidx,
                                           const float (&dgc)[S * (S + 1) / 2], const float (&us)[S][3],
                                           float (&acc)[S][3])
{
    const CubeView<S, T> view(sf, sg, kz, cidx, NSL);
    VA<S> ua[3], P[3];
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        ua[k] = va_make<S>([&](int a) { return us[a][k]; });
        P[k] = va_zero<S>();
    }
#pragma unroll
    for (int b = 0; b < S; ++b) p2_cube_species<S, DRAG>(p, view, b, dgc, ua, us[b], P);
#pragma unroll
    for (int a = 0; a < S; ++a)
#pragma unroll
        for (int k = 0; k < 3; ++k) acc[a][k] += va_get<S>(P[k], a);
}

// the shell sums of the acceleration of the site at ring position kz of the
// tile, added to acc (reach 2, 3: this thread's part of the groups `tab`)
template <class T, int S, int R, bool DRAG, int NSL = 2 * R + 2>
__device__ __forceinline__ void pass2_site(const mlbi_params &p, const mlbi_entry *tab, const float4 *sf,
                                           const float *sg, int kz, int cidx, float (&acc)[S][3])
{
    if constexpr (R == 1) {
        const int cs = ring(kz, NSL);
        float dgc[T::NP];
#pragma unroll
        for (int q = 0; q < T::NP; ++q) dgc[q] = sg[(cs * T::NP + q) * T::GPLANE + T::gidx()];
        float us[S][3];
#pragma unroll
        for (int a = 0; a < S; ++a) {
            const float4 v = sf[cs * S * T::PLANE + a * T::PLANE + cidx];
            us[a][0] = v.y; us[a][1] = v.z; us[a][2] = v.w;
        }
        pass2_cube<S, DRAG, T, NSL>(p, sf, sg, kz, cidx, dgc, us, acc);
    } else {
        const TileView<S, T> view{sf, sg, kz, cidx, NSL};
        p2_groups<S, T::SPLIT, DRAG>(p, tab, view, T::part(), acc);
    }
}

// One thread per site where the fused kernel also serves the lattice: the two
// agree bit for bit.
template <int S, int R, int TX>
using Tile2Of = Tile<S, R, TileOf<S, R, TX>::TY, TX, R == 2 && S <= 2 ? 1 : TileOf<S, R, TX>::SPLIT, TX == 16>;

template <int S, int R, bool DRAG, int TX>
__global__ void __launch_bounds__(Tile2Of<S, R, TX>::NTH, Tile2Of<S, R, TX>::blocks)
    k_pass2_tiled(const mlbi_params p, const float *__restrict__ dg, const mlbi_entry *__restrict__ tab,
                  const float4 *__restrict__ frest, const float4 *__restrict__ pst, float4 *__restrict__ acc_f,
                  double *__restrict__ acc_out)
{
    using T = Tile2Of<S, R, TX>;
    step_begin();
    extern __shared__ float4 smem[];
    float4 *sf = smem;
    float *sg = reinterpret_cast<float *>(smem + (size_t)T::NSLOT * S * T::PLANE);
    float *red = reinterpret_cast<float *>(reinterpret_cast<char *>(smem) + T::ring) + T::sid();   // [SPLIT - 1][3 S][NT]
    const int x0 = blockIdx.x * T::TX, y0 = blockIdx.y * T::TY, z0 = blockIdx.z * p.zchunk;
    const int z1 = min(z0 + p.zchunk, p.nz);
    const int x = x0 + T::lx(), y = y0 + T::ly();
    const bool active = x < p.nx && y < p.ny;
    const int cidx = T::cidx();
    const mlbi_entry *stab =
        stage_table<T, R>(p, tab, reinterpret_cast<float4 *>(reinterpret_cast<char *>(smem) + T::bytes));
    int xy[T::J];
    stage_sites<T, R>(p, x0, y0, xy);
    for (int k = 0; k < 2 * R + 1; ++k)
        stage_plane<T, S>(p, xy, z0 - R + k, ring(k, T::NSLOT), pst, dg, sf, sg);
    cp_async_commit();
    for (int z = z0; z < z1; ++z) {
        cp_async_wait_all();
        __syncthreads();
        const int kz = z - z0 + R;
        if (z + 1 < z1) {
            stage_plane<T, S>(p, xy, z + R + 1, ring(kz + R + 1, T::NSLOT), pst, dg, sf, sg);
            cp_async_commit();
        }
        if (T::SPLIT == 1 && !active) continue;
        const long long r = x + (long long)p.nx * (y + (long long)p.ny * z);
        float acc[S][3];
        zero_acc<S>(acc);
        if (active) pass2_site<T, S, R, DRAG>(p, stab, sf, sg, kz, cidx, acc);
        if constexpr (T::SPLIT > 1) {
            if (active && T::part() > 0) {
#pragma unroll
                for (int k = 0; k < 3 * S; ++k) red[((T::part() - 1) * 3 * S + k) * T::NT] = acc[k / 3][k % 3];
            }
            __syncthreads();
            if (!active || T::part() > 0) continue;
#pragma unroll
            for (int q = 0; q < T::SPLIT - 1; ++q)
#pragma unroll
                for (int k = 0; k < 3 * S; ++k) acc[k / 3][k % 3] += red[(q * 3 * S + k) * T::NT];
        }
#pragma unroll
        for (int a = 0; a < S; ++a) add_rest(acc[a], frest[a * p.N + r]);
        store_acc<S>(p, r, acc, acc_f, acc_out);
    }
}

// ------------------------------------------------------------------ pass 2 fused with the collision
// Per plane, each thread computes the acceleration of its site and at once
// collides and streams the site.  Its own populations and moments for the
// next plane are prefetched by cp.async into a per-thread slot of shared
// memory while this plane's shell sums run.  Two cp.async groups per plane,
// committed by every thread (empty where there is nothing to copy):
//   A(z) = halo plane z + R of the stencil ring and the site's frest(z),
//   P(z) = the site's populations and moments of plane z.
// They alternate A(z), P(z), A(z+1), P(z+1), ..., so "all but the newest
// group" is A(z) at the top of plane z and P(z) before its collision.
template <int S, int R, int TX = kBX>
struct FusedTile {
    using T = Tile<S, R, 128 / TX, TX>;
    static constexpr size_t pops_off = T::bytes;                                   // float [S*19][NT]
    static constexpr size_t mom_off = pops_off + (size_t)S * MLBI_Q * T::NT * sizeof(float);   // float4 [S][NT]
    static constexpr size_t rest_off = mom_off + (size_t)S * T::NT * sizeof(float4);           // float4 [S][NT]
    static constexpr size_t bytes = rest_off + (size_t)S * T::NT * sizeof(float4);
};

template <int S>
__device__ __forceinline__ void stage_pops(const mlbi_params &p, long long r, int tid, int nt,
                                           const float *__restrict__ fin, const float4 *__restrict__ mom, float *sF,
                                           float4 *sM)
{
#pragma unroll
    for (int a = 0; a < S; ++a) {
        cp_async16(sM + a * nt + tid, mom + a * p.N + r);
#pragma unroll
        for (int i = 0; i < MLBI_Q; ++i)
            cp_async4(sF + (a * MLBI_Q + i) * nt + tid, fin + ((long long)a * MLBI_Q + i) * p.N + r);
    }
}

template <int S>
__device__ __forceinline__ void stage_rest(const mlbi_params &p, long long r, int tid, int nt,
                                           const float4 *__restrict__ frest, float4 *sR)
{
#pragma unroll
    for (int a = 0; a < S; ++a) cp_async16(sR + a * nt + tid, frest + a * p.N + r);
}

__device__ __forceinline__ void cp_async_wait_all_but_newest() { asm volatile("cp.async.wait_group 1;\n" ::: "memory"); }

template <int S, int R, bool DRAG, int TX>
__global__ void __launch_bounds__(kBX * kBY, S <= 2 ? 3 : 2) k_pass2_collide(const mlbi_params p,
                                                                            const float *__restrict__ dg,
                                                                            const mlbi_entry *__restrict__ tab,
                                                                            const float4 *__restrict__ frest,
                                                                            const float4 *__restrict__ pst,
                                                                            const float4 *__restrict__ mom,
                                                                            const float *__restrict__ fin,
                                                                            float *__restrict__ fout)
{
    using F = FusedTile<S, R, TX>;
    using T = typename F::T;
    step_begin();
    extern __shared__ float4 smem[];
    float4 *sf = smem;
    float *sg = reinterpret_cast<float *>(smem + (size_t)T::NSLOT * S * T::PLANE);
    float *sF = reinterpret_cast<float *>(reinterpret_cast<char *>(smem) + F::pops_off);
    float4 *sM = reinterpret_cast<float4 *>(reinterpret_cast<char *>(smem) + F::mom_off);
    float4 *sR = reinterpret_cast<float4 *>(reinterpret_cast<char *>(smem) + F::rest_off);
    const int x0 = blockIdx.x * TX, y0 = blockIdx.y * T::TY, z0 = blockIdx.z * p.zchunk;
    const int z1 = min(z0 + p.zchunk, p.nz);
    const int x = x0 + T::lx(), y = y0 + T::ly();
    const int tid = T::tid();
    const bool active = x < p.nx && y < p.ny;
    const int cidx = T::cidx();
    const long long sxy = x + (long long)p.nx * y, nxy = (long long)p.nx * p.ny;
    int xy[T::J];
    stage_sites<T, R>(p, x0, y0, xy);
    for (int k = 0; k < 2 * R + 1; ++k) stage_plane<T, S>(p, xy, z0 - R + k, ring(k, T::NSLOT), pst, dg, sf, sg);
    if (active) stage_rest<S>(p, sxy + nxy * z0, tid, T::NT, frest, sR);
    cp_async_commit();                                                  // A(z0)
    if (active) stage_pops<S>(p, sxy + nxy * z0, tid, T::NT, fin, mom, sF, sM);
    cp_async_commit();                                                  // P(z0)
    float rest[S][3];
    for (int z = z0; z < z1; ++z) {
        cp_async_wait_all_but_newest();                                 // A(z) landed
        __syncthreads();
        const int kz = z - z0 + R;
        const long long r = sxy + nxy * z;
        float acc[S][3];
        zero_acc<S>(acc);
        if (active) {
#pragma unroll
            for (int a = 0; a < S; ++a) {
                const float4 v = sR[a * T::NT + tid];
                rest[a][0] = v.x; rest[a][1] = v.y; rest[a][2] = v.z;
            }
        }
        if (z + 1 < z1) {
            stage_plane<T, S>(p, xy, z + R + 1, ring(kz + R + 1, T::NSLOT), pst, dg, sf, sg);
            if (active) stage_rest<S>(p, r + nxy, tid, T::NT, frest, sR);
        }
        cp_async_commit();                                              // A(z + 1)
        if (active) {
            pass2_site<T, S, R, DRAG>(p, tab + p.grp_at, sf, sg, kz, cidx, acc);
#pragma unroll
            for (int a = 0; a < S; ++a) add_rest(acc[a], make_float4(rest[a][0], rest[a][1], rest[a][2], 0.f));
        }
        cp_async_wait_all_but_newest();                                 // P(z) landed (own slots only)
        if (active) {
            Centre<S> c;
#pragma unroll
            for (int a = 0; a < S; ++a) {
                const float4 v = sM[a * T::NT + tid];
                c.dn[a] = v.x;
                c.n[a] = p.nref[a] + v.x;
                c.u[a][0] = v.y; c.u[a][1] = v.z; c.u[a][2] = v.w;
            }
            collide_push<S>(p, x, y, z, r, c, acc, SharedPops{sF + tid, T::NT}, fout);
            if (z + 1 < z1) stage_pops<S>(p, r + nxy, tid, T::NT, fin, mom, sF, sM);
        }
        cp_async_commit();                                              // P(z + 1)
    }
    cp_async_wait_all();
}

// ------------------------------------------------------------------ fused, with bulk tensor copies
// The same per-site arithmetic as k_pass2_collide.  The site's own data of a
// plane -- its 19 S populations, moments and rest force -- arrive as three
// bulk tensor (TMA) copies of the block's 128 sites (32 x 4 or 16 x 8), issued by one thread
// at the top of the plane and waited on (mbarrier, bounded) only before the
// collision, so they land while the plane's shell sums run.  Shared layouts
// are those of the cp.async variant: population (a, i) of thread t at
// sF[(a * 19 + i) * 128 + t], moments and rest force at sM / sR[a * 128 + t].
// The stencil ring holds 2R + 1 planes only: the next plane is staged into
// the slot of plane z - R once every thread has finished plane z's shell
// sums (a second barrier per plane), and lands during the collisions.  The
// 9 KB this saves (R = 1, S = 2) and a 128-register bound give 4 resident
// blocks per SM instead of 3.
template <int S, int R, int TX = kBX>
struct TmaTile {
    using T = Tile<S, R, 128 / TX, TX>;
    static constexpr int NSL = 2 * R + 1;
    static constexpr size_t pad(size_t b) { return (b + 127) / 128 * 128; }
    static constexpr size_t ring_bytes = (size_t)NSL * T::PLANE * (S * sizeof(float4) + T::NP * sizeof(float));
    static constexpr uint32_t pops_bytes = (uint32_t)S * MLBI_Q * T::NT * 4;
    static constexpr uint32_t v4_bytes = (uint32_t)S * T::NT * 16;
    static constexpr size_t pops_off = pad(ring_bytes);
    static constexpr size_t mom_off = pops_off + pops_bytes;
    static constexpr size_t rest_off = mom_off + v4_bytes;
    static constexpr size_t bytes = rest_off + v4_bytes + 128;       // + alignment slack of the base
    static constexpr uint32_t tx_bytes = pops_bytes + 2 * v4_bytes;
};

// the tile (bx, by, bz) of the fused pass; the maps are kernel parameters or
// (grouped launches) global-memory copies the issuing thread has acquired
template <int S, int R, bool DRAG, int TX>
__device__ __forceinline__ void pass2_collide_tma_tile(const mlbi_params &p, const float *__restrict__ dg,
                                                       const mlbi_entry *__restrict__ tab,
                                                       const float4 *__restrict__ pst, float *__restrict__ fout,
                                                       unsigned int *__restrict__ flags, const CUtensorMap *map_f,
                                                       const CUtensorMap *map_mom, const CUtensorMap *map_rest,
                                                       int bx, int by, int bz)
{
    using F = TmaTile<S, R, TX>;
    using T = typename F::T;
    extern __shared__ float4 smem_raw[];
    __shared__ __align__(8) uint64_t bar_mem;
    // the bulk copies want 128-byte aligned destinations
    char *base = reinterpret_cast<char *>((reinterpret_cast<uintptr_t>(smem_raw) + 127) & ~uintptr_t(127));
    constexpr int NSL = F::NSL;
    float4 *sf = reinterpret_cast<float4 *>(base);
    float *sg = reinterpret_cast<float *>(sf + (size_t)NSL * S * T::PLANE);
    float *sF = reinterpret_cast<float *>(base + F::pops_off);
    float4 *sM = reinterpret_cast<float4 *>(base + F::mom_off);
    float4 *sR = reinterpret_cast<float4 *>(base + F::rest_off);
    __shared__ int s_fail;                                       // a wait gave up (read after a barrier)
    const uint32_t bar = smem_u32(&bar_mem);
    const int x0 = bx * TX, y0 = by * T::TY, z0 = bz * p.zchunk;
    const int z1 = min(z0 + p.zchunk, p.nz);
    const int x = x0 + T::lx(), y = y0 + T::ly();
    const int tid = T::tid();
    const bool active = x < p.nx && y < p.ny;
    const int cidx = T::cidx();
    const int sxy = x + p.nx * y, nxy = p.nx * p.ny;
    auto issue = [&](int z) {
        mbar_expect_tx(bar, F::tx_bytes);
        tma_load_4d(smem_u32(sF), map_f, bar, x0, y0, z, 0);
        tma_load_5d(smem_u32(sM), map_mom, bar, 0, x0, y0, z, 0);
        tma_load_5d(smem_u32(sR), map_rest, bar, 0, x0, y0, z, 0);
    };
    if (tid == 0) {
        mbar_init(bar, 1);
        s_fail = 0;
    }
    int xy[T::J];
    stage_sites<T, R>(p, x0, y0, xy);
    for (int k = 0; k < 2 * R + 1; ++k) stage_plane<T, S>(p, xy, z0 - R + k, ring(k, NSL), pst, dg, sf, sg);
    cp_async_commit();
    __syncthreads();                                            // the barrier is initialised
    if (tid == 0) issue(z0);
    uint32_t phase = 0;
    for (int z = z0; z < z1; ++z) {
        cp_async_wait_all();
        __syncthreads();              // ring planes up to z + R in; every thread is done with plane z - 1
        if (s_fail) break;            // uniform: read after the barrier
        if (tid == 0 && z > z0) issue(z);
        const int kz = z - z0 + R;
        float acc[S][3];
        zero_acc<S>(acc);
        if (active) pass2_site<T, S, R, DRAG, NSL>(p, tab + p.grp_at, sf, sg, kz, cidx, acc);
        __syncthreads();              // every thread is done with plane z - R: its slot takes plane z + R + 1
        if (z + 1 < z1) stage_plane<T, S>(p, xy, z + R + 1, ring(kz + R + 1, NSL), pst, dg, sf, sg);
        cp_async_commit();
        // each thread waits for the copies itself, so warps move on to their
        // collisions independently; a wait that gives up marks the block failed,
        // and every thread leaves at the next barrier
        const bool ok = mbar_wait(bar, phase);
        phase ^= 1u;
        if (!ok) {
            s_fail = 1;
            if (tid == 0) atomicOr(flags, MLBI_FLAG_TIMEOUT);
            continue;
        }
        if (active) {
            Centre<S> c;
#pragma unroll
            for (int a = 0; a < S; ++a) {
                const float4 v = sM[a * T::NT + tid];
                c.dn[a] = v.x;
                c.n[a] = p.nref[a] + v.x;
                c.u[a][0] = v.y; c.u[a][1] = v.z; c.u[a][2] = v.w;
                add_rest(acc[a], sR[a * T::NT + tid]);
            }
            collide_push<S>(p, x, y, z, sxy + nxy * z, c, acc, SharedPops{sF + tid, T::NT}, fout);
        }
    }
    cp_async_wait_all();
    if (s_fail && tid == 0) mbar_wait(bar, phase ^ 1u);       // one more bounded wait for the copy in flight
}

template <int S, int R, bool DRAG, int TX>
__global__ void __launch_bounds__(kBX * kBY, S <= 2 ? 4 : 2)
    k_pass2_collide_tma(const mlbi_params p, const float *__restrict__ dg, const mlbi_entry *__restrict__ tab,
                        const float4 *__restrict__ pst, float *__restrict__ fout, unsigned int *__restrict__ flags,
                        const __grid_constant__ CUtensorMap map_f, const __grid_constant__ CUtensorMap map_mom,
                        const __grid_constant__ CUtensorMap map_rest)
{
    step_begin();
    pass2_collide_tma_tile<S, R, DRAG, TX>(p, dg, tab, pst, fout, flags, &map_f, &map_mom, &map_rest, blockIdx.x,
                                       blockIdx.y, blockIdx.z);
}

// every member of a group (block table entries {member, bx, by, bz}); odd:
// the members read f[cur ^ 1] and write f[cur]
template <int S, int R, bool DRAG, int TX>
__global__ void __launch_bounds__(kBX * kBY, S <= 2 ? 4 : 2)
    k_pass2_collide_group(const mlbi_member *__restrict__ mem, const int4 *__restrict__ blk, int odd)
{
    __shared__ mlbi_params sp;
    const int4 e = blk[blockIdx.x];
    const mlbi_member *m = mem + e.x;
    const int rd = m->cur ^ odd;
    if (threadIdx.x == 0 && threadIdx.y == 0) {
        tensormap_acquire(&m->map_f[rd]);
        tensormap_acquire(&m->map_mom);
        tensormap_acquire(&m->map_frest);
    }
    group_params(m, sp);
    const mlbi_buffers &b = m->b;
    pass2_collide_tma_tile<S, R, DRAG, TX>(sp, b.dg, b.table, b.pst, b.f[rd ^ 1], b.flags, &m->map_f[rd], &m->map_mom,
                                       &m->map_frest, e.y, e.z, e.w);
}

template <int S, int R, bool DRAG, int TX = mlbi_tile_of(S, R).tx>
cudaError_t launch_pass2_tiled(const mlbi_params &p, const mlbi_buffers &b, double *acc_out, cudaStream_t s)
{
    if constexpr (mlbi_tile_ty(S, R) == 0) {
        return cudaErrorInvalidValue;
    } else {
        if constexpr (TX == kBX && R == 1 && S <= 2)
            if (p.tile_x == 16) return launch_pass2_tiled<S, R, DRAG, 16>(p, b, acc_out, s);
        using T = Tile2Of<S, R, TX>;
        auto k = k_pass2_tiled<S, R, DRAG, TX>;
        const size_t bytes = T::bytes + staged_table_bytes<T, R>(p);
        cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
        if (e != cudaSuccess) return e;
        const dim3 g((unsigned)((p.nx + T::TX - 1) / T::TX), (unsigned)((p.ny + T::TY - 1) / T::TY),
                     (unsigned)((p.nz + p.zchunk - 1) / p.zchunk));
        return launch_step(k, g, dim3(kBX, T::NTH / kBX), bytes, s, p, b.dg, b.table, b.frest, b.pst, b.acc, acc_out);
    }
}

template <int S, bool DRAG>
cudaError_t launch_pass2(const mlbi_params &p, const mlbi_buffers &b, double *acc_out, cudaStream_t s)
{
    if (p.tile_r == 1) return launch_pass2_tiled<S, 1, DRAG>(p, b, acc_out, s);
    if (p.tile_r == 2) return launch_pass2_tiled<S, 2, DRAG>(p, b, acc_out, s);
    if (p.tile_r == 3) return launch_pass2_tiled<S, 3, DRAG>(p, b, acc_out, s);
    return launch_step(k_pass2<S, DRAG>, (unsigned)((p.N + 31) / 32), dim3(32, kParts2), 0, s, p, b.dg, b.table, b.frest, b.pst, b.acc,
                       acc_out);
}

constexpr size_t kMaxSharedPerBlock = 227 * 1024;

template <int S, int R, bool DRAG, int TX = kBX>
cudaError_t launch_pass2_collide_tiled(const mlbi_params &p, const mlbi_buffers &b, int cur, cudaStream_t s)
{
    using F = FusedTile<S, R, TX>;
    using G = TmaTile<S, R, TX>;
    if constexpr (F::bytes > kMaxSharedPerBlock) {
        return cudaErrorInvalidValue;
    } else {
        if constexpr (TX == kBX && R == 1 && S <= 2)
            if (p.tile_x == 16) return launch_pass2_collide_tiled<S, R, DRAG, 16>(p, b, cur, s);
        const dim3 g((unsigned)((p.nx + TX - 1) / TX), (unsigned)((p.ny + F::T::TY - 1) / F::T::TY),
                     (unsigned)((p.nz + p.zchunk - 1) / p.zchunk));
        if constexpr (G::bytes <= kMaxSharedPerBlock) {
            if (b.maps && b.maps->ok) {
                auto k = k_pass2_collide_tma<S, R, DRAG, TX>;
                cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)G::bytes);
                if (e != cudaSuccess) return e;
                return launch_step(k, g, dim3(kBX, kBY), G::bytes, s, p, b.dg, b.table, b.pst, b.f[cur ^ 1], b.flags,
                                   b.maps->f[cur], b.maps->mom, b.maps->frest);
            }
        }
        auto k = k_pass2_collide<S, R, DRAG, TX>;
        cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)F::bytes);
        if (e != cudaSuccess) return e;
        return launch_step(k, g, dim3(kBX, kBY), F::bytes, s, p, b.dg, b.table, b.frest, b.pst, b.mom, b.f[cur],
                           b.f[cur ^ 1]);
    }
}

template <int S, bool DRAG>
cudaError_t launch_pass2_collide(const mlbi_params &p, const mlbi_buffers &b, int cur, cudaStream_t s)
{
    if (p.tile_r == 1) return launch_pass2_collide_tiled<S, 1, DRAG>(p, b, cur, s);
    if constexpr (S <= 2)
        if (p.tile_r == 2) return launch_pass2_collide_tiled<S, 2, DRAG>(p, b, cur, s);
    return cudaErrorInvalidValue;          // the global-memory pass 2 is not fused
}

template <int S>
cudaError_t pass2_species(const mlbi_params &p, const mlbi_buffers &b, double *acc_out, cudaStream_t s)
{
    return p.drag_only ? launch_pass2<S, true>(p, b, acc_out, s) : launch_pass2<S, false>(p, b, acc_out, s);
}
template <int S>
cudaError_t pass2_collide_species(const mlbi_params &p, const mlbi_buffers &b, int cur, cudaStream_t s)
{
    return p.drag_only ? launch_pass2_collide<S, true>(p, b, cur, s) : launch_pass2_collide<S, false>(p, b, cur, s);
}

}  // namespace

// the entry points of one species count, for the unit that holds it
#define MLBI_PASS2_UNIT(S)                                                                                             \
    template <>                                                                                                        \
    cudaError_t mlbi_pass2_species<S>(const mlbi_params &p, const mlbi_buffers &b, double *acc_out, cudaStream_t s)     \
    {                                                                                                                  \
        return pass2_species<S>(p, b, acc_out, s);                                                                     \
    }                                                                                                                  \
    template <>                                                                                                        \
    cudaError_t mlbi_pass2_collide_species<S>(const mlbi_params &p, const mlbi_buffers &b, int cur, cudaStream_t s)     \
    {                                                                                                                  \
        return pass2_collide_species<S>(p, b, cur, s);                                                                 \
    }
