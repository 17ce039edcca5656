// mlb_pass1.cuh -- device code of pass 1 of a time step on sm_103a: the
// hard-core force (Eq. potmeanforce), the velocity exchange (Eqs. gammaab,
// viscousforce) at u, the friction matrix Gamma^a, the attraction read-in,
// and the half-step predictor du of the semi-implicit forcing.  Three
// variants of the shell sums: global memory with the sign groups (any reach),
// shared-memory tile with the sign groups (reach 2, 3), and the compile-time
// 3x3x3 cube (reach 1).  The kernels come in three modes:
//   kExact      the method's pass 1 (mlb_pass1.cu)
//   kSurrogate  F^hc taken from attr (the learned surrogate's), no hard-core sums
//   kSweep      a further Jacobi sweep of the half step u* = u + a(u*)/2: the
//               staged field holds the previous sweep's (n - n_ref, u*), the
//               centre keeps its own u (from the moments), the rest force comes
//               from frest; only the exchange and Gamma are summed (mlb_sweep.cu)
// Internal header: each including unit instantiates the kernels it launches.
#pragma once

#include "mlb_passes.cuh"
#include "mlb_cube.cuh"
#include "mlb_groups.cuh"

namespace {

constexpr int kExact = 0, kSurrogate = 1, kSweep = 2;

// Solve (I + G/2) x = b for symmetric G = (xx, yy, zz, xy, xz, yz).
__device__ __forceinline__ void solve_sym3(const float G[6], const float b[3], float x[3])
{
    float a00 = 1.f + 0.5f * G[0], a11 = 1.f + 0.5f * G[1], a22 = 1.f + 0.5f * G[2];
    float a01 = 0.5f * G[3], a02 = 0.5f * G[4], a12 = 0.5f * G[5];
    float c00 = a11 * a22 - a12 * a12;
    float c01 = a02 * a12 - a01 * a22;
    float c02 = a01 * a12 - a02 * a11;
    float c11 = a00 * a22 - a02 * a02;
    float c12 = a01 * a02 - a00 * a12;
    float c22 = a00 * a11 - a01 * a01;
    float inv = 1.f / (a00 * c00 + a01 * c01 + a02 * c02);
    x[0] = (c00 * b[0] + c01 * b[1] + c02 * b[2]) * inv;
    x[1] = (c01 * b[0] + c11 * b[1] + c12 * b[2]) * inv;
    x[2] = (c02 * b[0] + c12 * b[1] + c22 * b[2]) * inv;
}

// per species: hf[q] = (F^hc_q, F^v_q), G = friction matrix packed as
// (xx, yy), (zz, xy), (xz, yz), at = attraction
template <int S>
struct Acc1 {
    float2 hf[S][3], G[S][3];
    float at[S][3];
    __device__ __forceinline__ void zero()
    {
#pragma unroll
        for (int a = 0; a < S; ++a) {
#pragma unroll
            for (int k = 0; k < 3; ++k) {
                hf[a][k] = make_float2(0.f, 0.f);
                G[a][k] = make_float2(0.f, 0.f);
                at[a][k] = 0.f;
            }
        }
    }
    // the shell sums of (a, b): D hard core, E = sum s s^T (W+ + W-), J the
    // exchange relative to the partners' velocity u^b(r), completed by
    // Gamma_ab w, w = u^b(r) - u^a(r) (drag); K = vx_ab / 2, H = -hc_ab / 2
    template <bool DRAG, bool HC>
    __device__ __forceinline__ void add(int a, float K, float H, const float (&D)[3], const float (&E)[6],
                                        const float (&J)[3], const float (&w)[3], bool drag)
    {
        float e[6];
#pragma unroll
        for (int k = 0; k < 6; ++k) e[k] = K * E[k];
        G[a][0] = add2(G[a][0], f2(e[0], e[1]));
        G[a][1] = add2(G[a][1], f2(e[2], e[3]));
        G[a][2] = add2(G[a][2], f2(e[4], e[5]));
        if constexpr (HC)
#pragma unroll
            for (int k = 0; k < 3; ++k) hf[a][k].x = fmaf(H, D[k], hf[a][k].x);
        if constexpr (!DRAG)
#pragma unroll
            for (int k = 0; k < 3; ++k) hf[a][k].y = fmaf(K, J[k], hf[a][k].y);
        if (drag) {
            hf[a][0].y = fmaf(e[0], w[0], fmaf(e[3], w[1], fmaf(e[4], w[2], hf[a][0].y)));
            hf[a][1].y = fmaf(e[3], w[0], fmaf(e[1], w[1], fmaf(e[5], w[2], hf[a][1].y)));
            hf[a][2].y = fmaf(e[4], w[0], fmaf(e[5], w[1], fmaf(e[2], w[2], hf[a][2].y)));
        }
    }
    // the 12 partial sums per species of a part, stride n floats apart
    __device__ __forceinline__ void put(float *m, int n) const
    {
#pragma unroll
        for (int a = 0; a < S; ++a)
#pragma unroll
            for (int k = 0; k < 3; ++k) {
                m[(a * 12 + k) * n] = hf[a][k].x;
                m[(a * 12 + 3 + k) * n] = hf[a][k].y;
                m[(a * 12 + 6 + k) * n] = G[a][k].x;
                m[(a * 12 + 9 + k) * n] = G[a][k].y;
            }
    }
    __device__ __forceinline__ void take(const float *m, int n)
    {
#pragma unroll
        for (int a = 0; a < S; ++a)
#pragma unroll
            for (int k = 0; k < 3; ++k) {
                hf[a][k] = add2(hf[a][k], f2(m[(a * 12 + k) * n], m[(a * 12 + 3 + k) * n]));
                G[a][k] = add2(G[a][k], f2(m[(a * 12 + 6 + k) * n], m[(a * 12 + 9 + k) * n]));
            }
    }
};

// attraction sum_{+d} K_ab(d) (n^b(r+d) - n^b(r-d)) from global memory (G term
// of Eq. potmeanforce, RPA), for reaches the column kernel does not serve: the
// offsets that are `part` modulo PARTS
template <int S, int PARTS, bool INTERIOR>
__device__ __forceinline__ void pass1_attraction(const mlbi_params &p, const Loc &L,
                                                 const float4 *__restrict__ mom,
                                                 const mlbi_entry *__restrict__ tab, int part, float (&at)[S][3])
{
    const long long N = p.N;
#pragma unroll
    for (int a = 0; a < S; ++a) {
#pragma unroll
        for (int b = 0; b < S; ++b) {
            const mlbi_pair &pr = p.pair[pair_of(a, b, S)];
            const float *nb = reinterpret_cast<const float *>(mom + b * N);
            float s0 = 0.f, s1 = 0.f, s2 = 0.f;
#pragma unroll 4
            for (int k = pr.attr_start + part; k < pr.attr_start + pr.attr_count; k += PARTS) {
                const float4 e0 = __ldg(&tab[2 * k]);
                const float4 e1 = __ldg(&tab[2 * k + 1]);
                float vp, vm;
                if (INTERIOR) {
                    const long long o = __float_as_int(e1.x);
                    vp = nb[4 * (L.r + o)];
                    vm = nb[4 * (L.r - o)];
                } else {
                    const long long ip = nbr(p, L, e0, e1, 1), im = nbr(p, L, e0, e1, -1);
                    // beyond a wall n = 0, i.e. n - n_ref = -n_ref
                    vp = ip >= 0 ? nb[4 * ip] : -p.nref[b];
                    vm = im >= 0 ? nb[4 * im] : -p.nref[b];
                }
                const float d = vp - vm;        // deviations cancel n_ref exactly inside the fluid
                s0 += e0.x * d; s1 += e0.y * d; s2 += e0.z * d;
            }
            at[a][0] += s0; at[a][1] += s1; at[a][2] += s2;
        }
    }
}
// Added to the site's hard-core force, so that the parts add up as their shell sums
// do.  The half region has thousands of offsets for a pair of species and outweighs the
// shells, so every thread of a site takes its share.  Per step (left to the first part
// of a site -> shared; one thread per site in brackets): spheres of 4 with tails to 10
// sites, 64^3, 8.98 -> 2.32 ms (2.78); three of 2 / 2.5 / 3 to 9 sites between walls, 61 x 45 x 37,
// 23.7 -> 8.6 (9.0); two of 4 / 3, the same box, 8.85 -> 3.35 (5.3).
template <int S, int PARTS>
__device__ __forceinline__ void far_attraction(const mlbi_params &p, int x, int y, int z, long long r,
                                               const float4 *__restrict__ mom, const mlbi_entry *__restrict__ tab,
                                               int part, Acc1<S> &A)
{
    Loc L;
    L.x = x; L.y = y; L.z = z; L.r = r;
    const int R = p.reach;
    L.interior = x >= R && x < p.nx - R && y >= R && y < p.ny - R && z >= R && z < p.nz - R;
    float at[S][3];
#pragma unroll
    for (int a = 0; a < S; ++a) at[a][0] = at[a][1] = at[a][2] = 0.f;
    if (L.interior) pass1_attraction<S, PARTS, true>(p, L, mom, tab, part, at);
    else pass1_attraction<S, PARTS, false>(p, L, mom, tab, part, at);
#pragma unroll
    for (int a = 0; a < S; ++a)
#pragma unroll
        for (int k = 0; k < 3; ++k) A.hf[a][k].x += at[a][k];
}

// Finish pass 1 at one site.  rest = F^hc + G + F_ext and the exchange at u
// (the shell sums of sd) give the predictor du from (I + Gamma/2) du =
// (rest + exchange)/2: one Jacobi sweep of u* = u + a(u*)/2 with partner
// velocities held at u.  Outputs for pass 2: frest = rest, pst = (n - n_ref,
// u* = u + du).
template <int S, bool DRAG>
__device__ __forceinline__ void pass1_finish(const mlbi_params &p, long long r, const Centre<S> &c, const Acc1<S> &A,
                                             const float4 *__restrict__ fext, float4 *__restrict__ frest,
                                             float4 *__restrict__ pst)
{
    const long long N = p.N;
#pragma unroll
    for (int a = 0; a < S; ++a) {
        const float4 fe = p.has_fext ? fext[a * N + r] : make_float4(0.f, 0.f, 0.f, 0.f);
        const float fr[3] = {A.hf[a][0].x + A.at[a][0] + fe.x, A.hf[a][1].x + A.at[a][1] + fe.y,
                             A.hf[a][2].x + A.at[a][2] + fe.z};
        float d[3] = {0.f, 0.f, 0.f};
        if (p.semi_implicit) {
            const float rhs[3] = {0.5f * (fr[0] + A.hf[a][0].y), 0.5f * (fr[1] + A.hf[a][1].y),
                                  0.5f * (fr[2] + A.hf[a][2].y)};
            const float G[6] = {A.G[a][0].x, A.G[a][0].y, A.G[a][1].x, A.G[a][1].y, A.G[a][2].x, A.G[a][2].y};
            solve_sym3(G, rhs, d);
        }
        frest[a * N + r] = make_float4(fr[0], fr[1], fr[2], 0.f);
        pst[a * N + r] = make_float4(c.dn[a], c.u[a][0] + d[0], c.u[a][1] + d[1], c.u[a][2] + d[2]);
    }
}

// Finish a further sweep at one site: rest = frest (pass 1's), the exchange
// with the partners at the previous sweep's u*, the same Gamma; pst_out =
// (n - n_ref, u + du).
template <int S>
__device__ __forceinline__ void sweep_finish(const mlbi_params &p, long long r, const Centre<S> &c, const Acc1<S> &A,
                                             const float4 *__restrict__ frest, float4 *__restrict__ pst_out)
{
    const long long N = p.N;
#pragma unroll
    for (int a = 0; a < S; ++a) {
        const float4 fr = frest[a * N + r];
        const float rhs[3] = {0.5f * (fr.x + A.hf[a][0].y), 0.5f * (fr.y + A.hf[a][1].y),
                              0.5f * (fr.z + A.hf[a][2].y)};
        const float G[6] = {A.G[a][0].x, A.G[a][0].y, A.G[a][1].x, A.G[a][1].y, A.G[a][2].x, A.G[a][2].y};
        float d[3];
        solve_sym3(G, rhs, d);
        pst_out[a * N + r] = make_float4(c.dn[a], c.u[a][0] + d[0], c.u[a][1] + d[1], c.u[a][2] + d[2]);
    }
}

// the centre of a site: densities from the staged field; velocities from it
// too, except in a sweep, where the centre keeps its own u (mom_c) and the
// staged u* of the previous sweep is the partners' (ub, used by drag only)
template <int S, int MODE>
__device__ __forceinline__ void centre_of(const mlbi_params &p, const float4 (&cv)[S], const float4 *__restrict__ mom_c,
                                          long long r, Centre<S> &c, float (&ub)[S][3])
{
#pragma unroll
    for (int a = 0; a < S; ++a) {
        c.dn[a] = cv[a].x;
        c.n[a] = p.nref[a] + cv[a].x;
        ub[a][0] = cv[a].y; ub[a][1] = cv[a].z; ub[a][2] = cv[a].w;
        if constexpr (MODE == kSweep) {
            const float4 m = mom_c[a * p.N + r];
            c.u[a][0] = m.y; c.u[a][1] = m.z; c.u[a][2] = m.w;
        } else {
            c.u[a][0] = cv[a].y; c.u[a][1] = cv[a].z; c.u[a][2] = cv[a].w;
        }
    }
}

// ------------------------------------------------------------------ global memory
// Shells beyond the tiles (reach 4 and more; four species at reach 3).  A block
// takes 32 consecutive sites, each by kParts threads (one warp per part) that
// share the groups: enough warps for small lattices of large spheres (80 x 40 x
// 40 has 4000 site warps for 152 SMs), no idle lanes at ragged widths, and the
// parts read neighbouring rows at the same time.  Measured (sigma = 8 / 4, 925
// pairs a site, 80 x 40 x 40): pass 1 1.419 -> 0.429 ms, pass 2 1.043 ->
// 0.348 (one thread per site, a table entry per pair, every neighbour of a site near a
// face wrapped by itself: three quarters of the sites).  Two or eight threads a site: 0.53 and 0.53.
// Blocks per SM: two species take five, the L1 latency counts more than a few spills
// (4 blocks 0.443).  Three and four species would spill 1.0 and 2.9 KB at five (per step, 64^3,
// sigma = 6 / 4 / 3: 5 blocks 2.40 ms, 4 blocks 2.00, 3 blocks 2.08; 6 / 4 / 3 / 2: 5 blocks 8.6, 4 blocks
// 3.13, 3 blocks 3.04, 2 blocks 3.80; one thread per site 6.08 and 9.40); drag-only sums need
// fewer registers (four species of 1.5 / 2 / 2.5 / 3: 5 or 4 blocks 0.90 and 0.91, 3 blocks 0.975).  One species has the
// registers for seven (sigma = 4: 5 blocks 0.170, 7 blocks 0.164, 8 blocks 0.169).
// FAR: with an attraction beyond the columns' reach, whose loop wants warps more than
// registers (four species of 4 / 2 / 3 / 3.5 to 10 sites between walls, 61 x 45 x 37: 5 blocks 13.2
// ms, 3 blocks 16.7; one of 4 to 10 sites, 64^3: 5 blocks 2.81, 8 blocks 2.32), as a kernel of its own.
constexpr int kParts = 4;

constexpr int pass1_blocks(int S, bool drag, bool far)
{
    return S == 1 ? (far ? 8 : 7) : S == 2 || far ? 5 : drag ? (S == 4 ? 4 : 5) : (S == 3 ? 4 : 3);
}

template <int S, bool DRAG, int MODE, bool FAR>
__global__ void __launch_bounds__(32 * kParts, pass1_blocks(S, DRAG, FAR)) k_pass1(const mlbi_params p, const float4 *__restrict__ mom,
                                                          const float *__restrict__ dg,
                                                          const mlbi_entry *__restrict__ tab,
                                                          const float4 *__restrict__ fext,
                                                          const float4 *__restrict__ attr,
                                                          const float4 *__restrict__ mom_c, float4 *__restrict__ frest,
                                                          float4 *__restrict__ pst)
{
    step_begin();
    __shared__ float red[kParts - 1][12 * S][32];
    const long long N = p.N, r = blockIdx.x * 32ll + threadIdx.x;
    const int part = threadIdx.y;
    const bool active = r < N;
    const int x = (int)(r % p.nx), y = (int)(r / p.nx % p.ny), z = (int)(r / ((long long)p.nx * p.ny));
    Centre<S> c;
    Acc1<S> A;
    A.zero();
    if (active) {
        float ub[S][3];
        float4 cv[S];
#pragma unroll
        for (int a = 0; a < S; ++a) cv[a] = mom[a * N + r];
        centre_of<S, MODE>(p, cv, mom_c, r, c, ub);
        const GlobalView<S> view{p, mom, dg, x, y, z};
        p1_groups<S, kParts, DRAG, MODE == kSweep, MODE == kExact>(p, tab + p.grp_at, view, c.u, part, A);
        if constexpr (FAR) far_attraction<S, kParts>(p, x, y, z, r, mom, tab, part, A);
        if (part > 0) A.put(&red[part - 1][0][threadIdx.x], 32);
    }
    __syncthreads();
    if (!active || part > 0) return;
#pragma unroll
    for (int k = 0; k < kParts - 1; ++k) A.take(&red[k][0][threadIdx.x], 32);
    if constexpr (MODE == kSweep) {
        sweep_finish<S>(p, r, c, A, frest, pst);
        return;
    }
    if (MODE == kSurrogate || p.attr_r) {
#pragma unroll
        for (int a = 0; a < S; ++a) {
            const float4 v = attr[a * N + r];
            A.at[a][0] = v.x; A.at[a][1] = v.y; A.at[a][2] = v.z;
        }
    }
    pass1_finish<S, DRAG>(p, r, c, A, fext, frest, pst);
}

// ------------------------------------------------------------------ tiled variants
// Shell sums for reach 1 (mlb_cube.cuh), folded into the site's force sums.
// The exchange sums are relative to the partners' own velocity at r (ub):
// Gamma_ab (u^b(r) - u^a(r)) completes them.
template <int S, bool DRAG, int MODE, class T>
__device__ __forceinline__ void pass1_cube(const mlbi_params &p, const float4 *sf, const float *sg, int kz, int cidx,
                                           const Centre<S> &c, const float (&ub)[S][3],
                                           const float (&dgc)[S * (S + 1) / 2], Acc1<S> &A)
{
    constexpr bool HC = MODE == kExact;
    const CubeView<S, T> view(sf, sg, kz, cidx, T::NSLOT);
#pragma unroll
    for (int b = 0; b < S; ++b) {
        PairSums<S> s;
        p1_cube_species<S, DRAG, HC>(p, view, b, dgc, ub[b], s);
#pragma unroll
        for (int a = 0; a < S; ++a) {
            const mlbi_pair &pr = p.pair[pair_of(a, b, S)];
            float D[3], E[6], J[3];
#pragma unroll
            for (int k = 0; k < 3; ++k) {
                D[k] = va_get<S>(s.D[k], a);
                J[k] = va_get<S>(s.P[k], a);
                E[k] = va_get<S>(s.E[k], a);
                E[k + 3] = va_get<S>(s.E[k + 3], a);
            }
            const float w[3] = {ub[b][0] - c.u[a][0], ub[b][1] - c.u[a][1], ub[b][2] - c.u[a][2]};
            A.template add<DRAG, HC>(a, 0.5f * pr.vx_pre, -0.5f * pr.hc_pre, D, E, J, w, MODE == kSweep || a != b);
        }
    }
}

// MODE: kExact; kSurrogate (no hard-core sums, attr holds F^hc); kSweep (mom
// is the previous sweep's (n - n_ref, u*) field, mom_c the moments, frest is
// read, pst receives the sweep's u*)
// the tile (bx, by, bz) of the tiled pass 1
template <class T, int S, int R, bool DRAG, int MODE>
__device__ __forceinline__ void pass1_tile(const mlbi_params &p, const float4 *__restrict__ mom,
                                           const float *__restrict__ dg, const mlbi_entry *__restrict__ tab,
                                           const float4 *__restrict__ fext, const float4 *__restrict__ attr,
                                           const float4 *__restrict__ mom_c, float4 *__restrict__ frest,
                                           float4 *__restrict__ pst, int bx, int by, int bz)
{
    constexpr bool HC = MODE == kExact;
    extern __shared__ float4 smem[];
    float4 *sf = smem;                                                      // [NSLOT][S][PLANE]
    float *sg = reinterpret_cast<float *>(smem + (size_t)T::NSLOT * S * T::PLANE);   // [NSLOT][NP][GPLANE]
    float *red = reinterpret_cast<float *>(reinterpret_cast<char *>(smem) + T::ring) + T::sid();   // [SPLIT - 1][12 S][NT]
    const int x0 = bx * T::TX, y0 = by * T::TY, z0 = bz * p.zchunk;
    const int z1 = min(z0 + p.zchunk, p.nz);
    const int x = x0 + T::lx(), y = y0 + T::ly();
    const bool active = x < p.nx && y < p.ny;
    const int cidx = T::cidx();
    const mlbi_entry *stab =
        stage_table<T, R>(p, tab, reinterpret_cast<float4 *>(reinterpret_cast<char *>(smem) + T::bytes));
    int xy[T::J];
    stage_sites<T, R>(p, x0, y0, xy);
    for (int k = 0; k < 2 * R + 1; ++k)
        stage_plane<T, S>(p, xy, z0 - R + k, ring(k, T::NSLOT), mom, dg, sf, sg);
    cp_async_commit();
    for (int z = z0; z < z1; ++z) {
        cp_async_wait_all();
        __syncthreads();
        const int kz = z - z0 + R;                      // ring position of plane z
        if (z + 1 < z1) {
            stage_plane<T, S>(p, xy, z + R + 1, ring(kz + R + 1, T::NSLOT), mom, dg, sf, sg);
            cp_async_commit();
        }
        if (T::SPLIT == 1 && !active) continue;
        const int cs = ring(kz, T::NSLOT);
        const long long r = x + (long long)p.nx * (y + (long long)p.ny * z);
        Centre<S> c;
        float ub[S][3];
        Acc1<S> A;
        A.zero();
        if (active) {
            float4 cv[S];
#pragma unroll
            for (int a = 0; a < S; ++a) cv[a] = sf[cs * S * T::PLANE + a * T::PLANE + cidx];
            centre_of<S, MODE>(p, cv, mom_c, r, c, ub);
            if constexpr (R == 1) {
                float dgc[T::NP];
#pragma unroll
                for (int q = 0; q < T::NP; ++q) dgc[q] = sg[(cs * T::NP + q) * T::GPLANE + T::gidx()];
                pass1_cube<S, DRAG, MODE, T>(p, sf, sg, kz, cidx, c, ub, dgc, A);
            } else {
                const TileView<S, T> view{sf, sg, kz, cidx, T::NSLOT};
                p1_groups<S, T::SPLIT, DRAG, MODE == kSweep, HC>(p, stab, view, c.u, T::part(), A);
            }
            if constexpr (MODE == kExact)
                if (p.has_attraction && !p.attr_r) far_attraction<S, T::SPLIT>(p, x, y, z, r, mom, tab, T::part(), A);
        }
        if constexpr (T::SPLIT > 1) {
            if (active && T::part() > 0) A.put(red + (T::part() - 1) * 12 * S * T::NT, T::NT);
            __syncthreads();
            if (!active || T::part() > 0) continue;
#pragma unroll
            for (int k = 0; k < T::SPLIT - 1; ++k) A.take(red + k * 12 * S * T::NT, T::NT);
        }
        if constexpr (MODE == kSweep) {
            sweep_finish<S>(p, r, c, A, frest, pst);
            continue;
        }
        if (MODE == kSurrogate || p.attr_r) {
#pragma unroll
            for (int a = 0; a < S; ++a) {
                const float4 v = attr[a * p.N + r];
                A.at[a][0] = v.x; A.at[a][1] = v.y; A.at[a][2] = v.z;
            }
        }
        pass1_finish<S, DRAG>(p, r, c, A, fext, frest, pst);
    }
}

// Resident blocks asked for: 16 warps at most, which leaves 128 registers a
// thread, enough for the sums without spills (256^3 binary, reach 1: 4 blocks
// 0.867 ms; 5 blocks 0.892, 6 blocks 0.996, both spilling).  The grouped kernel of
// two species at reach 1 has its parameters in shared memory and spills 56 to 76 bytes.  The loads from
// shared memory bound the kernel (76 % of the L1's wavefronts at 128^3, issue
// slots 66 %).
template <int S, int R, bool DRAG, int TX, int MODE>
__global__ void __launch_bounds__(TileOf<S, R, TX>::NTH, TileOf<S, R, TX>::blocks)
    k_pass1_tiled(const mlbi_params p, const float4 *__restrict__ mom, const float *__restrict__ dg,
                  const mlbi_entry *__restrict__ tab, const float4 *__restrict__ fext, const float4 *__restrict__ attr,
                  const float4 *__restrict__ mom_c, float4 *__restrict__ frest, float4 *__restrict__ pst)
{
    step_begin();
    pass1_tile<TileOf<S, R, TX>, S, R, DRAG, MODE>(p, mom, dg, tab, fext, attr, mom_c, frest, pst, blockIdx.x,
                                                   blockIdx.y, blockIdx.z);
}

// every member of a group (block table entries {member, bx, by, bz}), the exact pass
template <int S, int R, bool DRAG, int TX>
__global__ void __launch_bounds__(TileOf<S, R, TX>::NTH, TileOf<S, R, TX>::blocks)
    k_pass1_group(const mlbi_member *__restrict__ mem, const int4 *__restrict__ blk)
{
    __shared__ mlbi_params sp;
    const int4 e = blk[blockIdx.x];
    const mlbi_member *m = mem + e.x;
    group_params(m, sp);
    const mlbi_buffers &b = m->b;
    pass1_tile<TileOf<S, R, TX>, S, R, DRAG, kExact>(sp, b.mom, b.dg, b.table, b.fext, b.attr, b.mom, b.frest, b.pst,
                                                     e.y, e.z, e.w);
}

// launch the tiled pass 1 (or sweep: fld the previous sweep's field, out the next) of a lattice
template <int S, int R, bool DRAG, int MODE, int TX = mlbi_tile_of(S, R).tx>
cudaError_t launch_tiled(const mlbi_params &p, const mlbi_buffers &b, const float4 *fld, float4 *out, cudaStream_t s)
{
    if constexpr (mlbi_tile_ty(S, R) == 0) {
        return cudaErrorInvalidValue;
    } else {
        if constexpr (TX == kBX && R == 1 && S <= 2)
            if (p.tile_x == 16) return launch_tiled<S, R, DRAG, MODE, 16>(p, b, fld, out, s);
        using T = TileOf<S, R, TX>;
        auto k = k_pass1_tiled<S, R, DRAG, TX, MODE>;
        const size_t bytes = T::bytes + staged_table_bytes<T, R>(p);
        cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
        if (e != cudaSuccess) return e;
        const dim3 g((unsigned)((p.nx + T::TX - 1) / T::TX), (unsigned)((p.ny + T::TY - 1) / T::TY),
                     (unsigned)((p.nz + p.zchunk - 1) / p.zchunk));
        return launch_step(k, g, dim3(kBX, T::NTH / kBX), bytes, s, p, fld, b.dg, b.table, b.fext, b.attr, b.mom, b.frest,
                           out);
    }
}

template <int S, int R, bool DRAG, int MODE = kExact>
cudaError_t launch_pass1_tiled(const mlbi_params &p, const mlbi_buffers &b, cudaStream_t s)
{
    return launch_tiled<S, R, DRAG, MODE>(p, b, b.mom, b.pst, s);
}

template <int S, bool DRAG>
cudaError_t launch_pass1(const mlbi_params &p, const mlbi_buffers &b, cudaStream_t s)
{
    if (p.hc_from_attr) {
        // the surrogate's case only: binary, no drag-only mode, reach 1 or 2
        if constexpr (S == 2 && !DRAG) {
            if (p.tile_r == 1) return launch_pass1_tiled<S, 1, DRAG, kSurrogate>(p, b, s);
            if (p.tile_r == 2) return launch_pass1_tiled<S, 2, DRAG, kSurrogate>(p, b, s);
        }
        return cudaErrorInvalidValue;
    }
    if (p.tile_r == 1) return launch_pass1_tiled<S, 1, DRAG>(p, b, s);
    if (p.tile_r == 2) return launch_pass1_tiled<S, 2, DRAG>(p, b, s);
    if (p.tile_r == 3) return launch_pass1_tiled<S, 3, DRAG>(p, b, s);
    const auto k = p.has_attraction && !p.attr_r ? k_pass1<S, DRAG, kExact, true> : k_pass1<S, DRAG, kExact, false>;
    return launch_step(k, (unsigned)((p.N + 31) / 32), dim3(32, kParts), 0, s, p, b.mom, b.dg, b.table, b.fext, b.attr,
                       b.mom, b.frest, b.pst);
}

template <int S>
cudaError_t pass1_species(const mlbi_params &p, const mlbi_buffers &b, cudaStream_t s)
{
    return p.drag_only ? launch_pass1<S, true>(p, b, s) : launch_pass1<S, false>(p, b, s);
}

// ------------------------------------------------------------------ further sweeps (mlb_sweep*.cu)
template <int S, int R, bool DRAG>
cudaError_t launch_sweep_tiled(const mlbi_params &p, const mlbi_buffers &b, const float4 *prev, float4 *next,
                               cudaStream_t s)
{
    return launch_tiled<S, R, DRAG, kSweep>(p, b, prev, next, s);
}

template <int S, bool DRAG>
cudaError_t launch_sweep(const mlbi_params &p, const mlbi_buffers &b, const float4 *prev, float4 *next, cudaStream_t s)
{
    if (p.tile_r == 1) return launch_sweep_tiled<S, 1, DRAG>(p, b, prev, next, s);
    if (p.tile_r == 2) return launch_sweep_tiled<S, 2, DRAG>(p, b, prev, next, s);
    if (p.tile_r == 3) return launch_sweep_tiled<S, 3, DRAG>(p, b, prev, next, s);
    return launch_step(k_pass1<S, DRAG, kSweep, false>, (unsigned)((p.N + 31) / 32), dim3(32, kParts), 0, s, p, prev, b.dg, b.table, b.fext,
                       b.attr, b.mom, b.frest, next);
}

template <int S>
cudaError_t sweep_species(const mlbi_params &p, const mlbi_buffers &b, const float4 *prev, float4 *next, cudaStream_t s)
{
    return p.drag_only ? launch_sweep<S, true>(p, b, prev, next, s) : launch_sweep<S, false>(p, b, prev, next, s);
}

}  // namespace
