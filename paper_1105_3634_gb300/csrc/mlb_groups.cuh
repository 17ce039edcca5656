// mlb_groups.cuh -- shell sums of the force passes for contact shells beyond
// the 3x3x3 cube, from a table of sign groups.  Internal header.
//
// A contact shell contains every offset of a length together with all its sign
// flips, so its half shell (one of each +-d) is cut into groups (X, Y, Z), X, Y,
// Z >= 0: one +-d pair on an axis, two in a coordinate plane, four in general
// position.  The points of a group share |s| and differ in signs only: the sums
// over s and s s^T of a group are butterflies over the pairs' scalars and one
// multiply-add per component and group, as in mlb_cube.cuh (whose header states
// what is summed), and the 8 neighbours of a group are independent loads.
// Groups are sorted by neighbour species, then by type (which components are
// non-zero): the loops over a type are compile-time in their signs.  A group's
// mask says for which species a its length lies in the shell of (a, b).
//
// Measured (sigma = 2 / 3, reach 3, 128^3, 113 pairs a site, one block of 16 warps
// per SM): pass 1 0.941 -> 0.629 ms, pass 2 0.812 -> 0.524 against one table entry
// and a multiply-add per component for each pair on 8 warps; three species (2 /
// 2.5 / 3, 512 x 64 x 64), which had no tile: 3.30 -> 1.35 and 1.81 -> 1.06 ms.
#pragma once

#include "mlb_passes.cuh"
#include "mlb_cube.cuh"

namespace {

// ------------------------------------------------------------------ group types
// 0..2 axis x, y, z; 3 xy, 4 xz, 5 yz; 6 xyz.  In pair k the last non-zero
// component is positive and the others have the signs of k's bits.
__host__ __device__ constexpr bool grp_has(int type, int c)
{
    return type < 3 ? type == c : (type == 3 ? c != 2 : (type == 4 ? c != 1 : (type == 5 ? c != 0 : true)));
}
__host__ __device__ constexpr int grp_pairs(int type) { return type < 3 ? 1 : (type < 6 ? 2 : 4); }
__host__ __device__ constexpr bool grp_neg(int type, int c, int k)
{
    return type == 6 ? (c == 0 ? (k & 1) : (c == 1 ? (k & 2) : 0)) != 0 : (k == 1 && c == (type == 5 ? 1 : 0));
}

template <int I, int N, class F>
__device__ __forceinline__ void static_for(F &&f)
{
    if constexpr (I < N) {
        f(std::integral_constant<int, I>{});
        static_for<I + 1, N>(f);
    }
}

struct Group {
    float s[3];
    int X, Y, Z, mask;
    __device__ __forceinline__ Group(const float4 *tab, int g)
    {
        const float4 a = tab[2 * g], b = tab[2 * g + 1];
        s[0] = a.x; s[1] = a.y; s[2] = a.z;
        mask = __float_as_int(a.w);
        X = __float_as_int(b.x); Y = __float_as_int(b.y); Z = __float_as_int(b.z);
    }
};

// ------------------------------------------------------------------ neighbours of a site
// A view gives the elements of a group's neighbours: f the index for field(b,
// f), g for dg(q, g), and whether the neighbour lies inside the walls.
struct Neighbour {
    int f, g;
    bool ok;
};

// the staged planes of a tile (sites beyond a wall are staged with n = 0)
template <int S, class T>
struct TileView {
    static constexpr bool kWalls = false;
    __device__ __forceinline__ bool walls() const { return false; }
    const float4 *sf;
    const float *sg;
    int kz, cidx, nsl;
    __device__ __forceinline__ Neighbour centre() const
    {
        const int pl = ring(kz, nsl);
        return {pl * S * T::PLANE + cidx, pl * T::NP * T::GPLANE + T::gidx(), true};
    }
    template <int TYPE>
    __device__ __forceinline__ void neighbours(const Group &g, Neighbour (&P)[grp_pairs(TYPE)],
                                               Neighbour (&M)[grp_pairs(TYPE)]) const
    {
        const int up = ring(kz + (grp_has(TYPE, 2) ? g.Z : 0), nsl), dn = grp_has(TYPE, 2) ? ring(kz - g.Z, nsl) : up;
        const int oy = g.Y * T::TXH, gy = g.Y * T::GP, gc = T::gidx();
        static_for<0, grp_pairs(TYPE)>([&](auto K) {
            constexpr int k = decltype(K)::value;
            int o = 0, og = 0;
            if constexpr (grp_has(TYPE, 0)) o = og = grp_neg(TYPE, 0, k) ? -g.X : g.X;
            if constexpr (grp_has(TYPE, 1)) {
                o += grp_neg(TYPE, 1, k) ? -oy : oy;
                og += grp_neg(TYPE, 1, k) ? -gy : gy;
            }
            P[k] = {up * S * T::PLANE + cidx + o, up * T::NP * T::GPLANE + gc + og, true};
            M[k] = {dn * S * T::PLANE + cidx - o, dn * T::NP * T::GPLANE + gc - og, true};
        });
    }
    __device__ __forceinline__ float4 field(int b, int f) const { return sf[f + b * T::PLANE]; }
    __device__ __forceinline__ float dg(int q, int g) const { return sg[g + q * T::GPLANE]; }
};

// global memory, for shells beyond the tiles: the coordinates of a group's 8
// neighbours are two per axis, so their wraps cost 6 minima a group instead of
// 24 selects, and every site takes the same path wherever it lies
template <int S>
struct GlobalView {
    static constexpr bool kWalls = true;
    __device__ __forceinline__ bool walls() const { return p.wall_axis >= 0; }
    const mlbi_params &p;
    const float4 *__restrict__ fld;
    const float *__restrict__ dgv;
    int x, y, z;
    __device__ __forceinline__ Neighbour centre() const
    {
        const int r = x + p.nx * (y + p.ny * z);
        return {r, r, true};
    }
    // c + d and c - d on a periodic axis of extent L (d < L): the smaller of the two
    // candidates as unsigned numbers
    static __device__ __forceinline__ int above(int c, int L) { return (int)min((unsigned)c, (unsigned)(c - L)); }
    static __device__ __forceinline__ int below(int c, int L) { return (int)min((unsigned)c, (unsigned)(c + L)); }
    // both, or on a wall axis (uniform) any site in the place of one beyond the wall
    static __device__ __forceinline__ void pair_at(int c, int d, int L, bool wall, int &up, int &dn, bool &bad_up,
                                                   bool &bad_dn)
    {
        if (wall) {
            bad_up = c + d >= L;
            bad_dn = c - d < 0;
            up = min(c + d, L - 1);
            dn = max(c - d, 0);
        } else {
            up = above(c + d, L);
            dn = below(c - d, L);
        }
    }
    template <int TYPE>
    __device__ __forceinline__ void neighbours(const Group &g, Neighbour (&P)[grp_pairs(TYPE)],
                                               Neighbour (&M)[grp_pairs(TYPE)]) const
    {
        int xp = x, xm = x, yp = y, ym = y, zp = z, zm = z;
        bool bad_up = false, bad_dn = false;               // along the wall axis
        if constexpr (grp_has(TYPE, 0)) pair_at(x, g.X, p.nx, p.wall_axis == 0, xp, xm, bad_up, bad_dn);
        if constexpr (grp_has(TYPE, 1)) pair_at(y, g.Y, p.ny, p.wall_axis == 1, yp, ym, bad_up, bad_dn);
        if constexpr (grp_has(TYPE, 2)) pair_at(z, g.Z, p.nz, p.wall_axis == 2, zp, zm, bad_up, bad_dn);
        const int nxy = p.nx * p.ny;
        const int ypr = yp * p.nx, ymr = ym * p.nx, zpr = zp * nxy, zmr = zm * nxy;
        const bool w = p.wall_axis >= 0;
        static_for<0, grp_pairs(TYPE)>([&](auto K) {
            constexpr int k = decltype(K)::value;
            constexpr int ix = grp_neg(TYPE, 0, k), iy = grp_neg(TYPE, 1, k);
            bool okp = true, okm = true;
            if (w) {
                // whether pair k's + neighbour goes down the wall axis
                const bool down = (ix && p.wall_axis == 0) || (iy && p.wall_axis == 1);
                okp = !(down ? bad_dn : bad_up);
                okm = !(down ? bad_up : bad_dn);
            }
            P[k].f = P[k].g = (ix ? xm : xp) + ((iy ? ymr : ypr) + zpr);
            M[k].f = M[k].g = (ix ? xp : xm) + ((iy ? ypr : ymr) + zmr);
            P[k].ok = okp;
            M[k].ok = okm;
        });
    }
    __device__ __forceinline__ float4 field(int b, int f) const { return (fld + b * p.N)[f]; }
    __device__ __forceinline__ float dg(int q, int g) const { return (dgv + q * p.N)[g]; }
};

// ------------------------------------------------------------------ sums over a group
// sum over the pairs of s x (odd in d), without the factors |s_c|
template <int TYPE>
__device__ __forceinline__ void grp_odd(const float (&x)[grp_pairs(TYPE)], float (&v)[3])
{
    if constexpr (TYPE < 3) {
        v[TYPE] = x[0];
    } else if constexpr (TYPE < 6) {
        v[TYPE == 5 ? 1 : 0] = x[0] - x[1];
        v[TYPE == 3 ? 1 : 2] = x[0] + x[1];
    } else {
        const float s01 = x[0] + x[1], d01 = x[0] - x[1], s23 = x[2] + x[3], d23 = x[2] - x[3];
        v[0] = d01 + d23;
        v[1] = s01 - s23;
        v[2] = s01 + s23;
    }
}
// E += sum over the pairs of s s^T x, E = (xx, yy, zz, xy, xz, yz)
template <int TYPE>
__device__ __forceinline__ void grp_even(const float (&x)[grp_pairs(TYPE)], const float (&s)[3], float (&E)[6])
{
    if constexpr (TYPE < 3) {
        E[TYPE] = fmaf(s[TYPE] * s[TYPE], x[0], E[TYPE]);
    } else if constexpr (TYPE < 6) {
        constexpr int I = TYPE == 5 ? 1 : 0, J = TYPE == 3 ? 1 : 2;
        const float sum = x[0] + x[1], dif = x[0] - x[1];
        E[I] = fmaf(s[I] * s[I], sum, E[I]);
        E[J] = fmaf(s[J] * s[J], sum, E[J]);
        E[TYPE] = fmaf(s[I] * s[J], dif, E[TYPE]);
    } else {
        const float s01 = x[0] + x[1], d01 = x[0] - x[1], s23 = x[2] + x[3], d23 = x[2] - x[3], sum = s01 + s23;
#pragma unroll
        for (int c = 0; c < 3; ++c) E[c] = fmaf(s[c] * s[c], sum, E[c]);
        E[3] = fmaf(s[0] * s[1], d01 - d23, E[3]);
        E[4] = fmaf(s[0] * s[2], d01 + d23, E[4]);
        E[5] = fmaf(s[1] * s[2], s01 - s23, E[5]);
    }
}

// +-s.v of pair k
template <int TYPE, int K>
__device__ __forceinline__ float grp_dot(const float (&s)[3], float vx, float vy, float vz, float c0)
{
    float r = c0;
    if constexpr (grp_has(TYPE, 2)) r = fmaf(s[2], vz, r);
    if constexpr (grp_has(TYPE, 1)) r = fmaf(grp_neg(TYPE, 1, K) ? -s[1] : s[1], vy, r);
    if constexpr (grp_has(TYPE, 0)) r = fmaf(grp_neg(TYPE, 0, K) ? -s[0] : s[0], vx, r);
    return r;
}

// ------------------------------------------------------------------ one group, pass 1
// The 8 neighbours and what does not depend on a come first, then each species
// a in the mask (the same for the whole block).  Scalar arithmetic: the packed
// FP32x2 instructions of the cube sums would do both species at once, but the
// groups beyond the smaller shells belong to one of them only (sigma = 2 / 3,
// reach 3, 128^3: pass 1 0.680 ms packed with a mask factor, 0.639 scalar).
template <int S>
struct GroupSums1 {
    float D[S][3], E[S][6], P[S][3];      // as PairSums of mlb_cube.cuh
};

template <int S, int b, bool DRAG, bool HC, int TYPE, class V>
__device__ __forceinline__ void p1_group(const Group &g, const V &v, float nr, const float (&Gc)[S],
                                         const float (&ub)[3], GroupSums1<S> &A)
{
    constexpr int NPR = grp_pairs(TYPE);
    Neighbour P[NPR], M[NPR];
    v.template neighbours<TYPE>(g, P, M);
    float np[NPR], nm[NPR], jp[NPR], jm[NPR], x[NPR], xo[3], t[3];
    static_for<0, NPR>([&](auto K) {
        constexpr int k = decltype(K)::value;
        float4 vp = v.field(b, P[k].f), vm = v.field(b, M[k].f);
        if (V::kWalls && v.walls()) {
            vp.x = P[k].ok ? vp.x : -nr;
            vm.x = M[k].ok ? vm.x : -nr;
        }
        np[k] = nr + vp.x;
        nm[k] = nr + vm.x;
        x[k] = vp.x - vm.x;
        if constexpr (!DRAG) {
            const float c0 = -grp_dot<TYPE, k>(g.s, ub[0], ub[1], ub[2], 0.f);
            jp[k] = grp_dot<TYPE, k>(g.s, vp.y, vp.z, vp.w, c0);
            jm[k] = grp_dot<TYPE, k>(g.s, vm.y, vm.z, vm.w, c0);
        }
    });
    grp_odd<TYPE>(x, xo);
#pragma unroll
    for (int a = 0; a < S; ++a) {
        if (S > 1 && !((g.mask >> a) & 1)) continue;
        float e[NPR], d[NPR], pj[NPR];
#pragma unroll
        for (int k = 0; k < NPR; ++k) {
            const float qp = __fmul_rn(np[k], v.dg(pair_of(a, b, S), P[k].g));
            const float qm = __fmul_rn(nm[k], v.dg(pair_of(a, b, S), M[k].g));
            const float wp = fmaf(np[k], Gc[a], qp), wm = fmaf(nm[k], Gc[a], qm);
            e[k] = wp + wm;
            if constexpr (HC) d[k] = qp - qm;
            if constexpr (!DRAG) pj[k] = fmaf(jm[k], wm, __fmul_rn(jp[k], wp));
        }
        grp_even<TYPE>(e, g.s, A.E[a]);
        if constexpr (HC) {
            grp_odd<TYPE>(d, t);
#pragma unroll
            for (int c = 0; c < 3; ++c)
                if (grp_has(TYPE, c)) A.D[a][c] = fmaf(g.s[c], fmaf(xo[c], Gc[a], t[c]), A.D[a][c]);
        }
        if constexpr (!DRAG) {
            grp_odd<TYPE>(pj, t);
#pragma unroll
            for (int c = 0; c < 3; ++c)
                if (grp_has(TYPE, c)) A.P[a][c] = fmaf(g.s[c], t[c], A.P[a][c]);
        }
    }
}

// the groups [grp[0], grp[7]) that are `part` modulo PARTS in the table, type by type
// (so a type's odd one out falls to another part than the last type's)
template <int PARTS, class F>
__device__ __forceinline__ void for_groups(const int (&grp)[8], const float4 *tab, int part, F &&f)
{
    static_for<0, 7>([&](auto TY) {
        constexpr int type = decltype(TY)::value;
        const int start = grp[type], end = grp[type + 1];
        const int first = PARTS == 1 ? 0 : (part + PARTS - start % PARTS) % PARTS;
#pragma unroll 1
        for (int k = start + first; k < end; k += PARTS) f(TY, Group(tab, k));
    });
}

// Pass 1 of a site: adds the shell sums of every pair (a, b) to A (this part's
// groups).  ua: the site's own velocities; the partners' are the staged ones.
template <int S, int PARTS, bool DRAG, bool SWEEP, bool HC, class V, class ACC>
__device__ __forceinline__ void p1_groups(const mlbi_params &p, const float4 *tab, const V &v, const float (&ua)[S][3],
                                          int part, ACC &A)
{
    static_for<0, S>([&](auto B) {
        constexpr int b = decltype(B)::value;
        const float4 cb = v.field(b, v.centre().f);
        const float ub[3] = {cb.y, cb.z, cb.w};
        float Gc[S];
        GroupSums1<S> s;
#pragma unroll
        for (int a = 0; a < S; ++a) {
            Gc[a] = fmaf(2.f, p.pair[pair_of(a, b, S)].g_ref, v.dg(pair_of(a, b, S), v.centre().g));
#pragma unroll
            for (int k = 0; k < 3; ++k) s.D[a][k] = s.P[a][k] = s.E[a][k] = s.E[a][k + 3] = 0.f;
        }
        const float nr = p.nref[b];
        for_groups<PARTS>(p.grp[b], tab, part, [&](auto TY, const Group &g) {
            p1_group<S, b, DRAG, HC, decltype(TY)::value>(g, v, nr, Gc, ub, s);
        });
#pragma unroll
        for (int a = 0; a < S; ++a) {
            const mlbi_pair &pr = p.pair[pair_of(a, b, S)];
            const float w[3] = {ub[0] - ua[a][0], ub[1] - ua[a][1], ub[2] - ua[a][2]};
            A.template add<DRAG, HC>(a, 0.5f * pr.vx_pre, -0.5f * pr.hc_pre, s.D[a], s.E[a], s.P[a], w, SWEEP || a != b);
        }
    });
}

// ------------------------------------------------------------------ one group, pass 2
template <int S, int b, bool DRAG, int TYPE, class V>
__device__ __forceinline__ void p2_group(const Group &g, const V &v, float nr, const float (&Gc)[S],
                                         const float (&w)[S][3], const float (&ub)[3], float (&F)[S][3])
{
    constexpr int NPR = grp_pairs(TYPE);
    Neighbour P[NPR], M[NPR];
    v.template neighbours<TYPE>(g, P, M);
    float np[NPR], nm[NPR], jp[NPR], jm[NPR], t[3];
    static_for<0, NPR>([&](auto K) {
        constexpr int k = decltype(K)::value;
        float4 vp = v.field(b, P[k].f), vm = v.field(b, M[k].f);
        if (V::kWalls && v.walls()) {
            vp.x = P[k].ok ? vp.x : -nr;
            vm.x = M[k].ok ? vm.x : -nr;
        }
        np[k] = nr + vp.x;
        nm[k] = nr + vm.x;
        if constexpr (!DRAG) {
            // velocities relative to the partner's own at the site
            const float c0 = -grp_dot<TYPE, k>(g.s, ub[0], ub[1], ub[2], 0.f);
            jp[k] = grp_dot<TYPE, k>(g.s, vp.y, vp.z, vp.w, c0);
            jm[k] = grp_dot<TYPE, k>(g.s, vm.y, vm.z, vm.w, c0);
        }
    });
#pragma unroll
    for (int a = 0; a < S; ++a) {
        if (S > 1 && !((g.mask >> a) & 1)) continue;                        // the same for the whole block
        float pj[NPR];
        static_for<0, NPR>([&](auto K) {
            constexpr int k = decltype(K)::value;
            const float wp = __fmul_rn(np[k], Gc[a] + v.dg(pair_of(a, b, S), P[k].g));
            const float wm = __fmul_rn(nm[k], Gc[a] + v.dg(pair_of(a, b, S), M[k].g));
            const float sw = grp_dot<TYPE, k>(g.s, w[a][0], w[a][1], w[a][2], 0.f);   // s.(u^b - u^a)(r)
            pj[k] = DRAG ? __fmul_rn(wp + wm, sw) : fmaf(wm, jm[k] + sw, __fmul_rn(wp, jp[k] + sw));
        });
        grp_odd<TYPE>(pj, t);
#pragma unroll
        for (int c = 0; c < 3; ++c)
            if (grp_has(TYPE, c)) F[a][c] = fmaf(g.s[c], t[c], F[a][c]);
    }
}

// Pass 2 of a site: adds the exchange of every pair (a, b) at the staged
// velocities to acc (this part's groups)
template <int S, int PARTS, bool DRAG, class V>
__device__ __forceinline__ void p2_groups(const mlbi_params &p, const float4 *tab, const V &v, int part,
                                          float (&acc)[S][3])
{
    static_for<0, S>([&](auto B) {
        constexpr int b = decltype(B)::value;
        const float4 cb = v.field(b, v.centre().f);
        const float ub[3] = {cb.y, cb.z, cb.w};
        float Gc[S], w[S][3], P[S][3];
#pragma unroll
        for (int a = 0; a < S; ++a) {
            Gc[a] = fmaf(2.f, p.pair[pair_of(a, b, S)].g_ref, v.dg(pair_of(a, b, S), v.centre().g));
            const float4 ca = v.field(a, v.centre().f);
            w[a][0] = ub[0] - ca.y;
            w[a][1] = ub[1] - ca.z;
            w[a][2] = ub[2] - ca.w;
            P[a][0] = P[a][1] = P[a][2] = 0.f;
        }
        const float nr = p.nref[b];
        for_groups<PARTS>(p.grp[b], tab, part, [&](auto TY, const Group &g) {
            p2_group<S, b, DRAG, decltype(TY)::value>(g, v, nr, Gc, w, ub, P);
        });
#pragma unroll
        for (int a = 0; a < S; ++a) {
            const float K = 0.5f * p.pair[pair_of(a, b, S)].vx_pre;
#pragma unroll
            for (int k = 0; k < 3; ++k) acc[a][k] = fmaf(K, P[a][k], acc[a][k]);
        }
    });
}

}  // namespace
