// mlb_internal.h -- definitions shared by the C-ABI runtime (mlb_api.cu) and
// the sm_103a kernel units (mlb_kernels.cu, mlb_pass1.cu, mlb_pass2.cu,
// mlb_attraction.cu).  Not part of the public ABI.
#pragma once

#include <cuda.h>
#include <cuda_runtime.h>
#include <stdint.h>

#define MLBI_Q 19
#define MLBI_MAXS 4
#define MLBI_MAXP 10            // unordered species pairs for MLBI_MAXS species

// One stencil entry is two float4 in the table:
//   e0 = (x, y, z, packed d): a unit vector s_d or a kernel vector, and the
//        offset d packed as three signed 10-bit fields (see mlbi_pack);
//   e1 = (linear offset of d for this lattice as int bits, 0, 0, 0).
typedef float4 mlbi_entry;

__host__ __device__ inline int mlbi_pack(int dx, int dy, int dz)
{
    return (dx + 512) | ((dy + 512) << 10) | ((dz + 512) << 20);
}
__host__ __device__ inline void mlbi_unpack(int p, int &dx, int &dy, int &dz)
{
    dx = (p & 1023) - 512;
    dy = ((p >> 10) & 1023) - 512;
    dz = ((p >> 20) & 1023) - 512;
}

struct mlbi_pair {               // unordered pair a <= b, index a*S - a(a-1)/2 + (b - a)
    int attr_start, attr_count;      // half attraction region (entries)
    float hc_pre;                    // kT sigma_ab^2 4 pi / |S_ab|
    float vx_pre;                    // K_ab 4 pi / |S_ab|,  K_ab = 2 sigma_ab^2 sqrt(2 mu_ab kT / pi)
    float h;                         // BMCSL h_ab = sigma_a sigma_b / (sigma_a + sigma_b)
    float g_ref;                     // BMCSL contact value at the reference densities
};

struct mlbi_params {
    int nx, ny, nz, S;
    long long N;
    int wall_axis;                   // -1 periodic
    int drag_only;
    int semi_implicit;               // 1: half-force shift, 0: forward Euler
    int has_fext;
    int has_attraction;
    int npairs;
    float omega;
    float src_scale;                 // 1 - omega/2 (semi-implicit) or 1
    float nref[MLBI_MAXS];
    float xi2_coef[MLBI_MAXS];       // (pi/6) sigma^2
    float xi3_coef[MLBI_MAXS];       // (pi/6) sigma^3
    float xi2_ref, xi3_ref;
    int ball_at, ball_grp[MLBI_MAXS][8];   // smoothing balls without their centre, as sign groups (see grp)
    float ball_inv[MLBI_MAXS];
    int reach;                       // largest offset component of any stencil (>= 1)
    int local_g;                     // every smoothing ball is the single site
    int tile_r;                      // reach of the union shells if the tiled kernels serve it (1..3), else 0
    // sign groups of the union half shells (mlb_groups.cuh), two float4 each from
    // table[grp_at]: (|s_x|, |s_y|, |s_z|, mask of the species a), (X, Y, Z, 0);
    // grp[b][t] the first of type t for neighbour species b, grp[b][7] the end
    int grp_at, grp[MLBI_MAXS][8];
    int cube_mask[MLBI_MAXP];        // tile_r == 1: bit k set when half offset k of the 3x3x3 cube is in S_ab
    int attr_r;                      // reach of the attraction if the column attraction kernel serves it (1..8), else 0
    // column form of the attraction (attr_r > 0): acol_count groups of columns (+-X, +-Y),
    // (+-Y, +-X), X >= Y >= 0, one float4 each at table[acol_start] = (X, Y, E, 0) as int
    // bits, E the largest |dz| any pair reaches there; their weights k are floats per
    // (group, pair, dz = 0..attr_r) at ((float *)(table + aw_start))
    int acol_start, acol_count, aw_start;
    int tile_x;                      // tile width of the reach-1 passes of one and two species: 32 (x 4) or 16 (x 8)
    int zchunk;                      // planes per block of the tiled kernels
    int hc_from_attr;                // 1: pass 1 skips the hard-core sums and takes attr as F^hc (surrogate)
    int pair_index[MLBI_MAXS][MLBI_MAXS];
    mlbi_pair pair[MLBI_MAXP];
    float wall_lo[3], wall_hi[3];
};

// Shared-memory z-marching tiles of the stencil passes: a ring of 2R + 2
// planes of (tx + 2R) x (ty + 2R) sites, each site S float4 fields and
// S(S+1)/2 contact-value deviations.  Reach 3 tiles leave room for one block
// per SM, so `split` threads share a site there (each takes every split-th
// group of the shell table) to keep enough warps resident; their partial sums
// meet in shared memory behind the ring.  So they do at reach 2, where the rings of three
// and four species leave one block of 4 warps otherwise: three threads a site for three
// species, two for the others (four: 204 KB with two).  Per step at 64^3, 1 / 1.5 / 2 and 1 / 1.5 / 1.75
// / 2: 0.680 -> 0.279 and 1.17 -> 0.536 ms (one thread a site from global memory before).
#define MLBI_MAX_TILE_BYTES (227 * 1024)
struct mlbi_tile {
    int tx, ty, split;               // ty = 0: no tile, the global-memory passes
};
__host__ __device__ constexpr mlbi_tile mlbi_tile_of(int S, int R)
{
    return R == 1 ? mlbi_tile{32, 4, 1}
         : R == 2 ? mlbi_tile{32, 4, S == 3 ? 3 : 2}
         : R == 3 && S <= 2 ? mlbi_tile{32, 8, 2}
         : R == 3 && S == 3 ? mlbi_tile{16, 8, 3}
         : mlbi_tile{32, 0, 1};
}
__host__ __device__ constexpr int mlbi_tile_ty(int S, int R) { return mlbi_tile_of(S, R).ty; }

// ------------------------------------------------------------------ work decomposition of the tiled passes
// Tile width of the reach-1 passes (one and two species): 32 x 4 sites, or 16
// x 8 where that leaves at least a tenth fewer idle threads (nx = 16: half of a
// 32-wide tile is idle; nx = 97, ny = 61: 72 % against 83 % of the threads have
// a site).  At equal use the wide tiles stay: their rows are read in full lines, and in the
// fused tiles the contact values of a narrow warp's two rows meet in 2 banks of 16.
inline bool mlbi_narrow_tiles(int S, int tile_r, long long tiles32, long long tiles16)
{
    return S <= 2 && tile_r == 1 && 10 * tiles16 <= 9 * tiles32;
}
inline int mlbi_tile_x(int S, int tile_r, int nx, int ny)
{
    return mlbi_narrow_tiles(S, tile_r, (long long)((nx + 31) / 32) * ((ny + 3) / 4),
                             (long long)((nx + 15) / 16) * ((ny + 7) / 8))
               ? 16
               : 32;
}
// rows of a tile of pass 1 and of the fused pass 2 + collision
inline int mlbi_tile_rows(const mlbi_params &p) { return p.tile_r == 1 ? 128 / p.tile_x : mlbi_tile_ty(p.S, p.tile_r); }
inline int mlbi_tile_cols(const mlbi_params &p) { return p.tile_r == 1 ? p.tile_x : mlbi_tile_of(p.S, p.tile_r).tx; }
// tile planes (one tile of one z plane) of a lattice
inline long long mlbi_tile_planes(const mlbi_params &p)
{
    const int ty = mlbi_tile_rows(p);
    const int tx = mlbi_tile_cols(p);
    return ty < 1 ? 0 : (long long)((p.nx + tx - 1) / tx) * ((p.ny + ty - 1) / ty) * p.nz;
}
// Planes per block.  A block pays about one plane's time for filling its ring,
// and the kernel's last blocks run about one block's time with the GPU
// emptying: with W tile planes on M resident blocks the time goes as
// W (1 + 1/z)/M + z + 1, least at z = sqrt(W / M).  Measured (reach 1, planes
// per block and ms per step): 64 x 8 x 8 1: 0.020, 8: 0.056; 97 x 61 x 45 2:
// 0.094, 12: 0.177; 128^3 6: 0.387, 12: 0.397; 256 x 16^3 4: 0.436, 12: 0.521.
// M is the two-species bulk-copy kernels' (4 blocks per SM) for every kernel of reach 1: with the
// fused kernels' own 2 of three and four species 64^3 took 0.120 and 0.256 ms per step against
// 0.114 and 0.250, 128 x 128 x 96 0.564 and 1.149 against 0.569 and 1.173; with the 3 of the
// cp.async kernel (nx % 4 != 0) nothing moved.  152: the SMs of the one part this builds for.
constexpr int kMlbiSMs = 152;
inline int mlbi_planes_per_block(const mlbi_params &p, long long tile_planes)
{
    const int resident = p.tile_r == 1 ? 4 : (p.tile_r == 2 ? 2 : 1);
    int z = 1;
    while (z < 16 && (long long)(2 * z + 1) * (2 * z + 1) * kMlbiSMs * resident < 4 * tile_planes) ++z;   // nearest to the root
    const int chunks = p.nz > z ? (2 * p.nz + z) / (2 * z) : 1;
    return (p.nz + chunks - 1) / chunks;
}

// Bulk tensor (TMA) descriptors of the buffers the fused pass-2 + collision
// kernel copies plane by plane: the populations f[c] as a 4D FP32 tensor
// (x, y, z, S*19), the moments and the rest force as 5D (4 components, x,
// y, z, S).  ok = 0 (no TMA: nx not a multiple of 4, or the encode failed)
// selects the cp.async variant.
struct mlbi_maps {
    CUtensorMap f[2];
    CUtensorMap mom;
    CUtensorMap frest;
    int ok;
};

// Tables of the tensor-core attraction (mlb_attraction_tc.cu), device memory
// owned by the context: per column (dx, dy), sorted by dy then dx, the B
// operands hi and lo; the columns and the first column of every dy row; the
// BF16 hi / lo copies of n - n_ref in the layout [y][b][z / 8][x][8 planes].
struct mlbi_tc_tables {
    void *weights;                   // [ncols][hi, lo][K / 8][N][8] BF16
    int2 *cols;                      // [ncols] (dx, dy)
    int *row_start;                  // [nrows + 1]
    void *qhi, *qlo;                 // [nyp][S][nz / 8][nxp][8] BF16 each (padded, mlbi_attraction_tc_padded)
    int ncols, nrows;
    int pass3;                       // 1: compensated hi/lo product, 0: hi only
};

// Device buffers of one context (all carved from one allocation).
struct mlbi_buffers {
    float *f[2];                     // [S][19][N] populations minus w_i n_ref
    float4 *mom;                     // [S][N]  (dn, ux, uy, uz), dn = n - n_ref
    float *dg;                       // [npairs][N]  g_ab - g_ref_ab
    float4 *frest;                   // [S][N]  pass 1 -> 2: F^hc + G + F_ext
    float4 *pst;                     // [S][N]  pass 1 -> 2: (n - n_ref, u* = u + du)
    float4 *acc;                     // [S][N]  pass 2 -> collide: acceleration
    float4 *attr;                    // [S][N]  attraction G^a (column attraction kernel -> pass 1)
    float4 *fext;                    // [S][N]  external force (if any)
    const mlbi_entry *table;         // stencil entries
    double *stage;                   // [S*4*N] FP64 staging for host transfers
    double *partial;                 // [MLBI_RED_BLOCKS][S+3] FP64 block sums
    double *sums;                    // [S+3] final sums
    unsigned int *flags;             // [1] numeric fault flags
    const mlbi_maps *maps;           // host copy of the TMA descriptors (owned by the context)
    unsigned long long *first_bad;   // [3] first invalid entry of uploaded fields (n, xi3, u)
};

#define MLBI_RED_BLOCKS 1024
#define MLBI_FLAG_XI3 1u
#define MLBI_FLAG_NAN 2u
#define MLBI_FLAG_TIMEOUT 4u            // a bounded device wait gave up


// kernel launchers (one per kernel unit); each returns cudaGetLastError()
// sums: also the FP64 conservation sums of the state into b.sums (mass[S],
// mom[3]; a grid of MLBI_RED_BLOCKS blocks and the final reduction)
cudaError_t mlbi_launch_moments(const mlbi_params &p, const mlbi_buffers &b, int cur, cudaStream_t s,
                                bool sums = false);
// FP64 sums of the populations f[cur] themselves into b.sums (mass[S], mom[3];
// mlb_popsum.cuh; b.partial holds the block partials)
cudaError_t mlbi_launch_pop_sums(const mlbi_params &p, const mlbi_buffers &b, int cur, cudaStream_t s);
cudaError_t mlbi_launch_gfield(const mlbi_params &p, const mlbi_buffers &b, cudaStream_t s);
cudaError_t mlbi_launch_pass1(const mlbi_params &p, const mlbi_buffers &b, cudaStream_t s);
// one further Jacobi sweep of the half step: prev = the previous sweep's
// (n - n_ref, u*) [S][N], next receives this sweep's (must differ from prev);
// b.mom, b.dg, b.frest as left by pass 1
cudaError_t mlbi_launch_sweep(const mlbi_params &p, const mlbi_buffers &b, const float4 *prev, float4 *next,
                              cudaStream_t s);
// tensor-core attraction: whether the lattice and species suit it (S <= 2,
// reach <= 8, no walls normal to z, nz % 8 == 0), bytes of one column's B
// operands, and the launch (prep + implicit GEMM) writing b.attr
bool mlbi_attraction_tc_supported(const mlbi_params &p);
size_t mlbi_attraction_tc_column_bytes(int S);
// padded extents of the BF16 density copies (an 8-site halo in x and y, x up to whole tiles)
void mlbi_attraction_tc_padded(const mlbi_params &p, int *nxp, int *nyp);
cudaError_t mlbi_launch_attraction_tc(const mlbi_params &p, const mlbi_buffers &b, const mlbi_tc_tables &t,
                                      cudaStream_t s);
cudaError_t mlbi_launch_attraction(const mlbi_params &p, const mlbi_buffers &b, cudaStream_t s);
cudaError_t mlbi_launch_moments_g(const mlbi_params &p, const mlbi_buffers &b, int cur, cudaStream_t s,
                                  bool sums = false);
// Uploaded fields n [S][N] and u [S][3][N] (u may be NULL), FP64 in device
// memory: the per-species sums of n into b.sums[0 .. S-1], and in
// b.first_bad the first flat index of n not finite or negative, of a site with
// xi3 = sum_a v3[a] n^a >= 1, and of u not finite or |u| >= 1 (all ones where
// none; b.first_bad is reset by the launch)
cudaError_t mlbi_launch_field_check(const mlbi_params &p, const mlbi_buffers &b, const double *n, const double *u,
                                    const double *v3, cudaStream_t s);
cudaError_t mlbi_launch_pass2(const mlbi_params &p, const mlbi_buffers &b, double *acc_out, cudaStream_t s);
cudaError_t mlbi_launch_collide(const mlbi_params &p, const mlbi_buffers &b, int cur, cudaStream_t s);
// pass 2 fused with the collision and streaming of f[cur] -> f[cur ^ 1] (no acceleration
// stored); only where mlbi_pass2_collide_supported (tiled passes whose fused tile fits
// in shared memory), else cudaErrorInvalidValue
bool mlbi_pass2_collide_supported(const mlbi_params &p);
cudaError_t mlbi_launch_pass2_collide(const mlbi_params &p, const mlbi_buffers &b, int cur, cudaStream_t s);
// the passes by species count (one compilation unit per count above two)
template <int S> cudaError_t mlbi_pass1_species(const mlbi_params &p, const mlbi_buffers &b, cudaStream_t s);
template <> cudaError_t mlbi_pass1_species<1>(const mlbi_params &p, const mlbi_buffers &b, cudaStream_t s);
template <> cudaError_t mlbi_pass1_species<2>(const mlbi_params &p, const mlbi_buffers &b, cudaStream_t s);
template <> cudaError_t mlbi_pass1_species<3>(const mlbi_params &p, const mlbi_buffers &b, cudaStream_t s);
template <> cudaError_t mlbi_pass1_species<4>(const mlbi_params &p, const mlbi_buffers &b, cudaStream_t s);
template <int S> cudaError_t mlbi_sweep_species(const mlbi_params &p, const mlbi_buffers &b, const float4 *prev, float4 *next, cudaStream_t s);
template <> cudaError_t mlbi_sweep_species<1>(const mlbi_params &p, const mlbi_buffers &b, const float4 *prev, float4 *next, cudaStream_t s);
template <> cudaError_t mlbi_sweep_species<2>(const mlbi_params &p, const mlbi_buffers &b, const float4 *prev, float4 *next, cudaStream_t s);
template <> cudaError_t mlbi_sweep_species<3>(const mlbi_params &p, const mlbi_buffers &b, const float4 *prev, float4 *next, cudaStream_t s);
template <> cudaError_t mlbi_sweep_species<4>(const mlbi_params &p, const mlbi_buffers &b, const float4 *prev, float4 *next, cudaStream_t s);
template <int S> cudaError_t mlbi_pass2_species(const mlbi_params &p, const mlbi_buffers &b, double *acc_out, cudaStream_t s);
template <> cudaError_t mlbi_pass2_species<1>(const mlbi_params &p, const mlbi_buffers &b, double *acc_out, cudaStream_t s);
template <> cudaError_t mlbi_pass2_species<2>(const mlbi_params &p, const mlbi_buffers &b, double *acc_out, cudaStream_t s);
template <> cudaError_t mlbi_pass2_species<3>(const mlbi_params &p, const mlbi_buffers &b, double *acc_out, cudaStream_t s);
template <> cudaError_t mlbi_pass2_species<4>(const mlbi_params &p, const mlbi_buffers &b, double *acc_out, cudaStream_t s);
template <int S> cudaError_t mlbi_pass2_collide_species(const mlbi_params &p, const mlbi_buffers &b, int cur, cudaStream_t s);
template <> cudaError_t mlbi_pass2_collide_species<1>(const mlbi_params &p, const mlbi_buffers &b, int cur, cudaStream_t s);
template <> cudaError_t mlbi_pass2_collide_species<2>(const mlbi_params &p, const mlbi_buffers &b, int cur, cudaStream_t s);
template <> cudaError_t mlbi_pass2_collide_species<3>(const mlbi_params &p, const mlbi_buffers &b, int cur, cudaStream_t s);
template <> cudaError_t mlbi_pass2_collide_species<4>(const mlbi_params &p, const mlbi_buffers &b, int cur, cudaStream_t s);
cudaError_t mlbi_launch_init(const mlbi_params &p, const mlbi_buffers &b, int cur, const double *n,
                             const double *u, cudaStream_t s);
cudaError_t mlbi_launch_export_moments(const mlbi_params &p, const mlbi_buffers &b, double *n_out,
                                       double *u_out, cudaStream_t s);
cudaError_t mlbi_launch_import_fext(const mlbi_params &p, const mlbi_buffers &b, const double *fext,
                                    cudaStream_t s);
// float4 [S][N] (x, y, z) -> FP64 [S][3][N]
cudaError_t mlbi_launch_export_vec(const mlbi_params &p, const float4 *src, double *dst, cudaStream_t s);

// ------------------------------------------------------------------ grouped launches
// One launch of a stage steps every member of a group of independent
// lattices (mlb_batch): the members take the same kernel instantiation (same
// S, shell reach and drag mode; site-local contact values; the fused pass 2 +
// collision on bulk tensor copies), each block reads its member and tile from
// a block table, copies the member's parameters into shared memory and runs
// the stage's per-block code unchanged, so a member's arithmetic is bitwise
// that of its own launches.  Device memory; the tensor maps are the
// members' host-encoded descriptors copied to global memory.
struct mlbi_member {
    CUtensorMap map_f[2];            // populations f[0], f[1]
    CUtensorMap map_mom, map_frest;
    mlbi_params p;
    mlbi_buffers b;                  // device pointers of the member (b.maps unused)
    int cur;                         // the buffer f[cur] the member reads at the group's even steps
};
struct mlbi_group {
    const mlbi_member *mem;          // [nmem] device
    const int4 *blk[3];              // per stage: [nblk] {member, block x, block y, block z} device
    int nblk[3];                     // (moments: {member, block, blocks of the member, 0})
    int S, R, drag, tile_x;          // the shared instantiation: species, shell reach (1, 2), drag only, tile width
};
enum { MLBI_GROUP_MOMENTS = 0, MLBI_GROUP_PASS1 = 1, MLBI_GROUP_PASS2 = 2 };
// whether a member can join a group, and its stage grids (blocks per stage)
bool mlbi_group_supported(const mlbi_params &p, const mlbi_buffers &b);
void mlbi_group_grid(const mlbi_params &p, int stage, int grid[3]);
// out[i] = *flags[i] for n contexts' fault-flag words (one launch; mlb_batch)
cudaError_t mlbi_launch_gather_flags(const unsigned int *const *flags, int n, unsigned int *out, cudaStream_t s);
// odd: the group's odd step (members read f[cur ^ 1])
cudaError_t mlbi_launch_group_moments(const mlbi_group &g, int odd, cudaStream_t s);
cudaError_t mlbi_launch_group_pass1(const mlbi_group &g, cudaStream_t s);
cudaError_t mlbi_launch_group_pass2_collide(const mlbi_group &g, int odd, cudaStream_t s);

// learned surrogate of the hard-core force (mlb_surrogate.cu)
struct mlb_net;
bool mlbi_net_matches(const mlb_net *n, int nx, int ny, int nz);
// a bounded wait in the network's tensor-core kernel gave up (synchronous read)
bool mlbi_net_timed_out(mlb_net *n);
// force[S][N] = the network's F^hc from the moments' n - n_ref
cudaError_t mlbi_net_force_from_moments(mlb_net *n, const float4 *mom, float4 *force, cudaStream_t s);
// sums[0] = sum |fs - fx|^2, sums[1] = sum |fx|^2 over n4 float4 (x, y, z)
cudaError_t mlbi_force_error(long long n4, const float4 *fs, const float4 *fx, double *sums, cudaStream_t s);
