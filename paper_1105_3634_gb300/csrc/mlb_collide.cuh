// mlb_collide.cuh -- the moments, site-local contact values, collision and
// push streaming of one site, shared by the stand-alone kernels
// (mlb_kernels.cu) and the fused pass-2 + collision kernels (mlb_pass2.cu),
// which must agree bit for bit.  Internal header.
#pragma once

#include "mlb_internal.h"
#include "mlb_device.cuh"

namespace {

// ------------------------------------------------------------------ moments
// dn = sum_i f_i (f stored minus w_i n_ref), j = sum_i c_i f_i taken as the
// differences of opposite links first, u = j / n (the barycentric velocity
// where n is tiny), for every species.
// j: the momentum densities themselves, sum_i c_i f_i
template <int S, class Pops>
__device__ __forceinline__ void site_moments(const mlbi_params &p, const Pops &pops, float (&dn)[S], float (&u)[S][3],
                                             float (&j)[S][3])
{
    float jx[S], jy[S], jz[S], rho = 0.f, m[3] = {0.f, 0.f, 0.f};
#pragma unroll
    for (int a = 0; a < S; ++a) {
        float v[MLBI_Q];
#pragma unroll
        for (int i = 0; i < MLBI_Q; ++i) v[i] = pops(a, i);
        float m0 = v[0], mx = 0.f, my = 0.f, mz = 0.f;
#pragma unroll
        for (int i = 1; i < MLBI_Q; i += 2) {
            m0 += v[i] + v[i + 1];
            const float d = v[i] - v[i + 1];          // opposite links i, i + 1
            if (CX[i]) mx += CX[i] * d;
            if (CY[i]) my += CY[i] * d;
            if (CZ[i]) mz += CZ[i] * d;
        }
        dn[a] = m0;
        jx[a] = mx; jy[a] = my; jz[a] = mz;
        rho += p.nref[a] + m0;
        m[0] += mx; m[1] += my; m[2] += mz;
    }
    const float irho = rho > 0.f ? 1.f / rho : 0.f;
#pragma unroll
    for (int a = 0; a < S; ++a) {
        j[a][0] = jx[a]; j[a][1] = jy[a]; j[a][2] = jz[a];
        const float n = p.nref[a] + dn[a];
        const bool ok = n > kTinyDensity;
        const float in = ok ? 1.f / n : 0.f;
        u[a][0] = ok ? jx[a] * in : m[0] * irho;
        u[a][1] = ok ? jy[a] * in : m[1] * irho;
        u[a][2] = ok ? jz[a] * in : m[2] * irho;
    }
}

template <int S, class Pops>
__device__ __forceinline__ void site_moments(const mlbi_params &p, const Pops &pops, float (&dn)[S], float (&u)[S][3])
{
    float j[S][3];
    site_moments<S>(p, pops, dn, u, j);
}

// ------------------------------------------------------------------ collide + stream
// Collision toward psi_perp at u + a/2 (Eq. prefactor, Hermite-2) with the
// forcing of Eq. evolution scaled by (1 - omega/2), then push streaming:
// f(r + c_i) with periodic wrap by selects, or halfway bounce-back at walls.
// population sources: pops(a, i) = f_i^a at the site
// g_ab(xi) - g_ab(xi_ref) of the BMCSL contact value
//   g = 1/o + 3 h xi2 / o^2 + 2 h^2 xi2^2 / o^3,   o = 1 - xi3,
// expanded exactly in the deviations d2 = xi2 - xi2_ref, d3 = xi3 - xi3_ref
// so that its FP32 value is accurate relative to the deviation itself.
__device__ __forceinline__ float bmcsl_dev(float h, float xi2r, float xi3r, float d2, float d3)
{
    float orf = 1.f - xi3r;
    float o = orf - d3;
    float xi2 = xi2r + d2;
    float o2 = o * o, or2 = orf * orf;
    float dA = d3 / (o * orf);
    float dB = 3.f * h * (d2 / o2 + xi2r * d3 * (orf + o) / (o2 * or2));
    float dC = 2.f * h * h * (d2 * (xi2 + xi2r) / (o2 * o) + xi2r * xi2r * d3 * (or2 + orf * o + o2) / (o2 * o * or2 * orf));
    return dA + dB + dC;
}

// Contact values of a site whose smoothing balls are the site itself:
// dg_q = g_q(xi) - g_q(xi_ref) from the density deviations dn.  Returns
// false where xi3 >= 1.
template <int S>
__device__ __forceinline__ bool site_contact(const mlbi_params &p, const float (&dn)[S],
                                             float (&dg)[S * (S + 1) / 2])
{
    float d2 = 0.f, d3 = 0.f;
#pragma unroll
    for (int a = 0; a < S; ++a) {
        d2 += p.xi2_coef[a] * dn[a];
        d3 += p.xi3_coef[a] * dn[a];
    }
#pragma unroll
    for (int q = 0; q < S * (S + 1) / 2; ++q) dg[q] = bmcsl_dev(p.pair[q].h, p.xi2_ref, p.xi3_ref, d2, d3);
    return p.xi3_ref + d3 < 1.f;
}

struct GlobalPops {
    const float *__restrict__ f;         // f + r
    long long N;
    __device__ __forceinline__ float operator()(int a, int i) const { return __ldg(f + ((long long)a * MLBI_Q + i) * N); }
};
struct SharedPops {
    const float *f;                      // tile slot of the site, stride nt per (a, i)
    int nt;
    __device__ __forceinline__ float operator()(int a, int i) const { return f[(a * MLBI_Q + i) * nt]; }
};

// c.v for a link with components in {-1, 0, 1}, and v.w.  The collision's
// arithmetic is spelled out (fmaf, __fmul_rn, __fadd_rn) so that no kernel that
// includes it contracts it differently.
__device__ __forceinline__ float cdot(int cx, int cy, int cz, float v0, float v1, float v2)
{
    float s = 0.f;
    bool any = false;
    if (cx) s = cx > 0 ? v0 : -v0, any = true;
    if (cy) s = any ? (cy > 0 ? __fadd_rn(s, v1) : __fsub_rn(s, v1)) : (cy > 0 ? v1 : -v1), any = true;
    if (cz) s = any ? (cz > 0 ? __fadd_rn(s, v2) : __fsub_rn(s, v2)) : (cz > 0 ? v2 : -v2);
    return s;
}
__device__ __forceinline__ float dot3(float a0, float a1, float a2, float b0, float b1, float b2)
{
    return fmaf(a0, b0, fmaf(a1, b1, __fmul_rn(a2, b2)));
}

// links with a component +1 / -1 along an axis (bit i for link i)
constexpr unsigned axis_links(const int (&c)[MLBI_Q], int sign)
{
    unsigned m = 0u;
    for (int i = 0; i < MLBI_Q; ++i)
        if (c[i] == sign) m |= 1u << i;
    return m;
}
constexpr unsigned kPlusX = axis_links(CX, 1), kMinusX = axis_links(CX, -1);
constexpr unsigned kPlusY = axis_links(CY, 1), kMinusY = axis_links(CY, -1);
constexpr unsigned kPlusZ = axis_links(CZ, 1), kMinusZ = axis_links(CZ, -1);

// Sites next to a wall run the same unrolled links as the others and only
// store differently.  (With a loop over the links there, one at a time, the
// warps at a wall finished long after the others: 97 x 61 x 45 between walls,
// fused pass 2 + collision 0.058 -> 0.044 ms; 256 x 16^3, half of them channels,
// 0.310 -> 0.243 ms per step.)  Periodic lattices take a copy without walls:
// the branch per link costs 7 % of the fused kernel at 128^3.
template <int S, bool WALLS, class Pops>
__device__ __forceinline__ void collide_push_w(const mlbi_params &p, int x, int y, int z, long long r,
                                             const Centre<S> &c, const float (&acc)[S][3], const Pops &pops,
                                             float *__restrict__ fout)
{
    const long long N = p.N;
    const float half = p.semi_implicit ? 0.5f : 0.f;
    float ueq[S][3];
    float ub[3] = {0.f, 0.f, 0.f}, rho = 0.f;
#pragma unroll
    for (int a = 0; a < S; ++a) {
#pragma unroll
        for (int q = 0; q < 3; ++q) {
            ueq[a][q] = fmaf(half, acc[a][q], c.u[a][q]);
            ub[q] = fmaf(c.n[a], ueq[a][q], ub[q]);
        }
        rho += c.n[a];
    }
    const float irho = rho > 0.f ? 1.f / rho : 0.f;
#pragma unroll
    for (int q = 0; q < 3; ++q) ub[q] = __fmul_rn(ub[q], irho);
    const float ubub = dot3(ub[0], ub[1], ub[2], ub[0], ub[1], ub[2]);
    const float omega = p.omega;
    // target site of every moving link (32-bit: the lattice has fewer than
    // 2^31 sites), the same for every species: tgt[i - 1] for link i; links that
    // wrap around a periodic face move by -+ the extent
    int tgt[MLBI_Q - 1];
    const int r32 = (int)r;
    {
        const int sy = p.nx, sz = p.nx * p.ny;
        const int wxm = x == 0 ? p.nx : 0, wxp = x == p.nx - 1 ? -p.nx : 0;
        const int wym = y == 0 ? sz : 0, wyp = y == p.ny - 1 ? -sz : 0;
        const int wzm = z == 0 ? (int)N : 0, wzp = z == p.nz - 1 ? -(int)N : 0;
#pragma unroll
        for (int i = 1; i < MLBI_Q; i += 2) {
            int dp = CX[i] + CY[i] * sy + CZ[i] * sz;                  // i: +c, i + 1: -c
            int dm = -dp;
            if (CX[i] > 0) { dp += wxp; dm += wxm; }
            if (CX[i] < 0) { dp += wxm; dm += wxp; }
            if (CY[i] > 0) { dp += wyp; dm += wym; }
            if (CY[i] < 0) { dp += wym; dm += wyp; }
            if (CZ[i] > 0) { dp += wzp; dm += wzm; }
            if (CZ[i] < 0) { dp += wzm; dm += wzp; }
            tgt[i - 1] = r32 + dp;
            tgt[i] = r32 + dm;
        }
    }
    // bit i set: link i leaves through the low / high wall and bounces back
    unsigned lo = 0u, hi = 0u;
    if constexpr (WALLS) {
        const int at = p.wall_axis == 0 ? x : (p.wall_axis == 1 ? y : z);
        const int last = (p.wall_axis == 0 ? p.nx : (p.wall_axis == 1 ? p.ny : p.nz)) - 1;
        if (at == 0) lo = p.wall_axis == 0 ? kMinusX : (p.wall_axis == 1 ? kMinusY : kMinusZ);
        if (at == last) hi = p.wall_axis == 0 ? kPlusX : (p.wall_axis == 1 ? kPlusY : kPlusZ);
    }
    const bool wall_site = WALLS && (lo | hi) != 0u;
#pragma unroll
    for (int a = 0; a < S; ++a) {
        const float na = c.n[a], dna = c.dn[a];
        float *oa = fout + (long long)a * MLBI_Q * N;
        float fi[MLBI_Q];
#pragma unroll
        for (int i = 0; i < MLBI_Q; ++i) fi[i] = pops(a, i);
        const float ua0 = ueq[a][0], ua1 = ueq[a][1], ua2 = ueq[a][2];
        const float a0 = acc[a][0], a1 = acc[a][1], a2 = acc[a][2];
        const float trM = fmaf(2.f, dot3(ua0, ua1, ua2, ub[0], ub[1], ub[2]), -ubub);   // tr(ua u + u ua - u u)
        const float trS = 2.f * dot3(ub[0], ub[1], ub[2], a0, a1, a2);                   // tr(u a + a u)
        const float ks = __fmul_rn(p.src_scale, na);
        // psi_perp and the forcing split into parts even and odd in c_i:
        // direction i and its opposite share the even part and flip the odd one.
        // (Collecting the Hermite-2 terms into one quadratic form per species
        // saves arithmetic but doubles the FP32 velocity error at 500 steps
        // against the FP64 oracle: this order is kept.)
        const float om1 = 1.f - omega;
        const float K1 = fmaf(__fmul_rn(-1.5f, na), trM, dna);          // even part of psi at c = 0
        const float K2 = __fmul_rn(__fmul_rn(-1.5f, ks), trS);          // even part of the forcing at c = 0
        const float n45 = __fmul_rn(4.5f, na), k9 = __fmul_rn(9.f, ks);
        const float n3 = __fmul_rn(__fmul_rn(3.f, omega), na), k3 = __fmul_rn(3.f, ks);
        oa[r] = fmaf(om1, fi[0], __fmul_rn(WQ[0], fmaf(omega, K1, K2)));
#pragma unroll
        for (int i = 1; i < MLBI_Q; i += 2) {
            const float cu = cdot(CX[i], CY[i], CZ[i], ua0, ua1, ua2);
            const float cb = cdot(CX[i], CY[i], CZ[i], ub[0], ub[1], ub[2]);
            const float ca = cdot(CX[i], CY[i], CZ[i], a0, a1, a2);
            const float psi = fmaf(n45, __fmul_rn(cb, fmaf(2.f, cu, -cb)), K1);
            const float even = fmaf(omega, psi, fmaf(__fmul_rn(k9, cb), ca, K2));
            const float odd = fmaf(n3, cu, __fmul_rn(k3, ca));
            const float fp = fmaf(om1, fi[i], __fmul_rn(WQ[i], __fadd_rn(even, odd)));
            const float fm = fmaf(om1, fi[i + 1], __fmul_rn(WQ[i], __fsub_rn(even, odd)));
            if (!wall_site) {
                (oa + i * N)[tgt[i - 1]] = fp;
                (oa + (i + 1) * N)[tgt[i]] = fm;
            } else {
                // halfway bounce-back: a link through a wall comes back as its
                // opposite, i + 1 for i and i for i + 1, with the wall's velocity
                const bool pl = (lo >> i) & 1u, ph = (hi >> i) & 1u, ml = (lo >> (i + 1)) & 1u, mh = (hi >> (i + 1)) & 1u;
                const float wn = __fmul_rn(6.f * WQ[i], na);
                const float cl = cdot(CX[i], CY[i], CZ[i], p.wall_lo[0], p.wall_lo[1], p.wall_lo[2]);
                const float ch = cdot(CX[i], CY[i], CZ[i], p.wall_hi[0], p.wall_hi[1], p.wall_hi[2]);
                if (pl || ph) (oa + (i + 1) * N)[r] = fmaf(-wn, pl ? cl : ch, fp);
                else (oa + i * N)[tgt[i - 1]] = fp;
                if (ml || mh) (oa + i * N)[r] = fmaf(wn, ml ? cl : ch, fm);
                else (oa + (i + 1) * N)[tgt[i]] = fm;
            }
        }
    }
}

template <int S, class Pops>
__device__ __forceinline__ void collide_push(const mlbi_params &p, int x, int y, int z, long long r,
                                             const Centre<S> &c, const float (&acc)[S][3], const Pops &pops,
                                             float *__restrict__ fout)
{
    if (p.wall_axis < 0) collide_push_w<S, false>(p, x, y, z, r, c, acc, pops, fout);
    else collide_push_w<S, true>(p, x, y, z, r, c, acc, pops, fout);
}

}  // namespace
