// mlb_cube.cuh -- shell sums of the force passes for reach 1, where every
// contact shell is a union of the three offset classes of the 3x3x3 cube:
// |d|^2 = 1 (axis), 2 (face diagonal), 3 (corner).  Internal header.
//
// What is summed, for a species a against neighbour species b over the +-d
// pairs of a shell (e = d as integers, s = e / |d|):
//   q+- = n+- dg+-,  W+- = n+- (2 g_ref + dg(r)) + q+-  (twice the midpoint weight of n+-)
//   hard core  -hc/2 sum s [(2 g_ref + dg(r)) (n+ - n-) + (q+ - q-)]
//   friction    vx/2 sum s s^T (W+ + W-)                                = Gamma_ab
//   exchange    vx/2 sum s [W+ s.(u^b(r+d) - u^a(r)) + W- s.(u^b(r-d) - u^a(r))]
// Within a class the directions differ by signs only, so the sums over s and
// s s^T are sums and differences of the points' scalars (one butterfly per
// plane of face diagonals, one per set of corners) scaled once per class by
// 1/|d| and 1/|d|^2, instead of a multiply-add per component and point.  n+ -
// n- does not depend on a and is summed once per b.  Pass 1 needs Gamma_ab
// anyway, so its exchange takes the velocities relative to u^b(r), shared by
// every a, and adds Gamma_ab (u^b(r) - u^a(r)).
//
// Measured at 256^3, two species (1 / 1.5): 1419 instructions per site in pass
// 1 (1884 with a multiply-add per component and point), 1.038 -> 0.867 ms; the
// fused pass 2 + collision 1.517 -> 1.313 ms.
//
// Per-species scalars are kept as vectors over a (VA): for two species one
// packed FP32x2 instruction serves both.
#pragma once

#include "mlb_passes.cuh"

namespace {

// ------------------------------------------------------------------ vectors over the species a
template <int S>
struct VA {
    float v[S];
};
template <>
struct VA<2> {
    float2 v;
};
template <int S>
__device__ __forceinline__ float va_get(const VA<S> &x, int a)
{
    if constexpr (S == 2) return a == 0 ? x.v.x : x.v.y;
    else return x.v[a];
}
template <int S, class F>
__device__ __forceinline__ VA<S> va_make(F &&f)
{
    VA<S> r;
    if constexpr (S == 2) {
        r.v = make_float2(f(0), f(1));
    } else {
#pragma unroll
        for (int a = 0; a < S; ++a) r.v[a] = f(a);
    }
    return r;
}
template <int S>
__device__ __forceinline__ VA<S> operator+(const VA<S> &x, const VA<S> &y)
{
    VA<S> r;
    if constexpr (S == 2) r.v = add2(x.v, y.v);
    else
#pragma unroll
        for (int a = 0; a < S; ++a) r.v[a] = __fadd_rn(x.v[a], y.v[a]);
    return r;
}
template <int S>
__device__ __forceinline__ VA<S> operator-(const VA<S> &x, const VA<S> &y)
{
    VA<S> r;
    if constexpr (S == 2) r.v = add2(x.v, f2(-y.v.x, -y.v.y));
    else
#pragma unroll
        for (int a = 0; a < S; ++a) r.v[a] = __fsub_rn(x.v[a], y.v[a]);
    return r;
}
template <int S>
__device__ __forceinline__ VA<S> operator*(float k, const VA<S> &x)
{
    VA<S> r;
    if constexpr (S == 2) r.v = mul2(f2(k, k), x.v);
    else
#pragma unroll
        for (int a = 0; a < S; ++a) r.v[a] = __fmul_rn(k, x.v[a]);
    return r;
}
template <int S>
__device__ __forceinline__ VA<S> operator*(const VA<S> &x, const VA<S> &y)
{
    VA<S> r;
    if constexpr (S == 2) r.v = mul2(x.v, y.v);
    else
#pragma unroll
        for (int a = 0; a < S; ++a) r.v[a] = __fmul_rn(x.v[a], y.v[a]);
    return r;
}
template <int S>
__device__ __forceinline__ VA<S> va_fma(const VA<S> &x, const VA<S> &y, const VA<S> &z)
{
    VA<S> r;
    if constexpr (S == 2) r.v = fma2(x.v, y.v, z.v);
    else
#pragma unroll
        for (int a = 0; a < S; ++a) r.v[a] = fmaf(x.v[a], y.v[a], z.v[a]);
    return r;
}
template <int S>
__device__ __forceinline__ VA<S> va_fma(float k, const VA<S> &y, const VA<S> &z)
{
    VA<S> r;
    if constexpr (S == 2) r.v = fma2(f2(k, k), y.v, z.v);
    else
#pragma unroll
        for (int a = 0; a < S; ++a) r.v[a] = fmaf(k, y.v[a], z.v[a]);
    return r;
}
template <int S>
__device__ __forceinline__ VA<S> va_zero()
{
    return va_make<S>([](int) { return 0.f; });
}

// e.v for an integer direction with components in {-1, 0, 1}
template <int X, int Y, int Z>
__device__ __forceinline__ float edot(float vx, float vy, float vz)
{
    float r = 0.f;
    if constexpr (X != 0) r = X > 0 ? vx : -vx;
    if constexpr (Y != 0) r = X != 0 ? (Y > 0 ? __fadd_rn(r, vy) : __fsub_rn(r, vy)) : (Y > 0 ? vy : -vy);
    if constexpr (Z != 0) r = (X != 0 || Y != 0) ? (Z > 0 ? __fadd_rn(r, vz) : __fsub_rn(r, vz)) : (Z > 0 ? vz : -vz);
    return r;
}
template <int S, int X, int Y, int Z>
__device__ __forceinline__ VA<S> edot_va(const VA<S> (&u)[3])
{
    VA<S> r = va_zero<S>();
    if constexpr (X != 0) r = X > 0 ? u[0] : va_zero<S>() - u[0];
    if constexpr (Y != 0) {
        if constexpr (X != 0) r = Y > 0 ? r + u[1] : r - u[1];
        else r = Y > 0 ? u[1] : va_zero<S>() - u[1];
    }
    if constexpr (Z != 0) {
        if constexpr (X != 0 || Y != 0) r = Z > 0 ? r + u[2] : r - u[2];
        else r = Z > 0 ? u[2] : va_zero<S>() - u[2];
    }
    return r;
}

// ------------------------------------------------------------------ the site's view of the staged planes
// f[k], g[k]: element offsets of plane z - 1 + k at the site, for the float4
// field of species 0 and the contact-value deviations of pair 0
template <int S, class T>
struct CubeView {
    const float4 *sf;
    const float *sg;
    int f[3], g[3];
    __device__ __forceinline__ CubeView(const float4 *sf_, const float *sg_, int kz, int cidx, int nsl)
        : sf(sf_), sg(sg_)
    {
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            const int s = ring(kz - 1 + k, nsl);
            f[k] = s * S * T::PLANE + cidx;
            g[k] = s * T::NP * T::GPLANE + T::gidx();
        }
    }
    template <int X, int Y, int Z>
    __device__ __forceinline__ float4 field(int b) const
    {
        return sf[f[1 + Z] + b * T::PLANE + X + T::TXH * Y];
    }
    template <int X, int Y, int Z>
    __device__ __forceinline__ VA<S> dg(int b) const
    {
        return va_make<S>([&](int a) { return sg[g[1 + Z] + pair_of(a, b, S) * T::GPLANE + X + T::GP * Y]; });
    }
};

// the shells of a class that contain it, per a: 1 or 0 (cube_mask bit of the
// class); false if none does
template <int S, int CL>
__device__ __forceinline__ bool class_mask(const mlbi_params &p, int b, VA<S> &m)
{
    bool any = false;
    m = va_make<S>([&](int a) {
        const bool h = (p.cube_mask[pair_of(a, b, S)] >> cls_bit(CL)) & 1;
        any |= h;
        return h ? 1.f : 0.f;
    });
    return any;
}

// ------------------------------------------------------------------ sums over the directions of a class
template <class T>
struct Odd {
    T x, y, z;
};
// sum_e e x_e over the corners, from the sums s and differences d of x at (1,1,1), (-1,1,1)
// and at (1,-1,1), (-1,-1,1)
template <class T>
__device__ __forceinline__ Odd<T> corner_odd(const T &s01, const T &d01, const T &s23, const T &d23)
{
    return {d01 + d23, s01 - s23, s01 + s23};
}

// ------------------------------------------------------------------ pass 1
// per (a, b): hard core D = sum s [(2 g_ref + dg(r)) (n+ - n-) + (q+ - q-)],
// friction E = sum s s^T (W+ + W-), exchange P relative to u^b(r)
template <int S>
struct PairSums {
    VA<S> D[3], E[6], P[3];
};

template <int S, bool DRAG, bool HC>
struct P1Point {
    VA<S> d, e, p;       // q+ - q-, W+ + W-, W+ j+ + W- j-
    float x;             // n+ - n-
    template <int X, int Y, int Z, class V>
    __device__ __forceinline__ void at(const V &c, int b, float nr, const VA<S> &Gc, const float (&ub)[3])
    {
        const float4 vp = c.template field<X, Y, Z>(b), vm = c.template field<-X, -Y, -Z>(b);
        const VA<S> gp = c.template dg<X, Y, Z>(b), gm = c.template dg<-X, -Y, -Z>(b);
        const float np = __fadd_rn(nr, vp.x), nm = __fadd_rn(nr, vm.x);
        const VA<S> qp = np * gp, qm = nm * gm;
        const VA<S> wp = va_fma(np, Gc, qp), wm = va_fma(nm, Gc, qm);
        e = wp + wm;
        if constexpr (HC) {
            x = __fsub_rn(vp.x, vm.x);
            d = qp - qm;
        }
        if constexpr (!DRAG) {
            const float ec = edot<X, Y, Z>(ub[0], ub[1], ub[2]);
            const float jp = __fsub_rn(edot<X, Y, Z>(vp.y, vp.z, vp.w), ec);
            const float jm = __fsub_rn(edot<X, Y, Z>(vm.y, vm.z, vm.w), ec);
            p = va_fma(jm, wm, jp * wp);
        }
    }
};

// fold sum_e e (Gc X + D) of one component into the pair sums
template <int S, bool HC>
__device__ __forceinline__ void fold_d(const VA<S> &k, const VA<S> &Gc, float x, const VA<S> &d, VA<S> &D)
{
    if constexpr (HC) D = va_fma(k, va_fma(x, Gc, d), D);
}

template <int S, bool DRAG, bool HC, class V>
__device__ __forceinline__ void p1_axis(const mlbi_params &p, const V &c, int b, float nr, const VA<S> &Gc,
                                        const float (&ub)[3], PairSums<S> &A)
{
    VA<S> m;
    if (!class_mask<S, 0>(p, b, m)) return;
    P1Point<S, DRAG, HC> t;
    t.template at<1, 0, 0>(c, b, nr, Gc, ub);
    A.E[0] = va_fma(m, t.e, A.E[0]);
    fold_d<S, HC>(m, Gc, t.x, t.d, A.D[0]);
    if constexpr (!DRAG) A.P[0] = va_fma(m, t.p, A.P[0]);
    t.template at<0, 1, 0>(c, b, nr, Gc, ub);
    A.E[1] = va_fma(m, t.e, A.E[1]);
    fold_d<S, HC>(m, Gc, t.x, t.d, A.D[1]);
    if constexpr (!DRAG) A.P[1] = va_fma(m, t.p, A.P[1]);
    t.template at<0, 0, 1>(c, b, nr, Gc, ub);
    A.E[2] = va_fma(m, t.e, A.E[2]);
    fold_d<S, HC>(m, Gc, t.x, t.d, A.D[2]);
    if constexpr (!DRAG) A.P[2] = va_fma(m, t.p, A.P[2]);
}

// one plane of face diagonals: components i, j of the vectors, entry ij of the matrix
template <int S, bool DRAG, bool HC, int I, int J, class V>
__device__ __forceinline__ void p1_face(const V &c, int b, float nr, const VA<S> &Gc, const float (&ub)[3],
                                        const VA<S> &k1, const VA<S> &k2, PairSums<S> &A)
{
    constexpr int IJ = I + J + 2;                       // xy 3, xz 4, yz 5
    P1Point<S, DRAG, HC> tp, tm;
    tp.template at<I == 0, I == 1 || J == 1, J == 2>(c, b, nr, Gc, ub);
    tm.template at<I == 0 ? -1 : 0, I == 1 ? -1 : (J == 1 ? 1 : 0), J == 2>(c, b, nr, Gc, ub);
    const VA<S> es = tp.e + tm.e;
    A.E[I] = va_fma(k2, es, A.E[I]);
    A.E[J] = va_fma(k2, es, A.E[J]);
    A.E[IJ] = va_fma(k2, tp.e - tm.e, A.E[IJ]);
    if constexpr (HC) {
        fold_d<S, HC>(k1, Gc, __fsub_rn(tp.x, tm.x), tp.d - tm.d, A.D[I]);
        fold_d<S, HC>(k1, Gc, __fadd_rn(tp.x, tm.x), tp.d + tm.d, A.D[J]);
    }
    if constexpr (!DRAG) {
        A.P[I] = va_fma(k2, tp.p - tm.p, A.P[I]);
        A.P[J] = va_fma(k2, tp.p + tm.p, A.P[J]);
    }
}

template <int S, bool DRAG, bool HC, class V>
__device__ __forceinline__ void p1_corner(const mlbi_params &p, const V &c, int b, float nr, const VA<S> &Gc,
                                          const float (&ub)[3], PairSums<S> &A)
{
    VA<S> m;
    if (!class_mask<S, 2>(p, b, m)) return;
    constexpr float il = cls_il(2);
    const VA<S> k1 = il * m, k2 = (1.f / 3.f) * m;
    P1Point<S, DRAG, HC> t0, t1;
    t0.template at<1, 1, 1>(c, b, nr, Gc, ub);
    t1.template at<-1, 1, 1>(c, b, nr, Gc, ub);
    const VA<S> es01 = t0.e + t1.e, ed01 = t0.e - t1.e;
    VA<S> ds01 = va_zero<S>(), dd01 = ds01, ps01 = ds01, pd01 = ds01;
    float xs01 = 0.f, xd01 = 0.f;
    if constexpr (HC) {
        ds01 = t0.d + t1.d, dd01 = t0.d - t1.d;
        xs01 = __fadd_rn(t0.x, t1.x), xd01 = __fsub_rn(t0.x, t1.x);
    }
    if constexpr (!DRAG) ps01 = t0.p + t1.p, pd01 = t0.p - t1.p;
    t0.template at<1, -1, 1>(c, b, nr, Gc, ub);
    t1.template at<-1, -1, 1>(c, b, nr, Gc, ub);
    const VA<S> es23 = t0.e + t1.e, ed23 = t0.e - t1.e;
    const VA<S> diag = es01 + es23;
    A.E[0] = va_fma(k2, diag, A.E[0]);
    A.E[1] = va_fma(k2, diag, A.E[1]);
    A.E[2] = va_fma(k2, diag, A.E[2]);
    A.E[3] = va_fma(k2, ed01 - ed23, A.E[3]);
    A.E[4] = va_fma(k2, ed01 + ed23, A.E[4]);
    A.E[5] = va_fma(k2, es01 - es23, A.E[5]);
    if constexpr (HC) {
        const Odd<VA<S>> v = corner_odd<VA<S>>(ds01, dd01, t0.d + t1.d, t0.d - t1.d);
        const float xs23 = __fadd_rn(t0.x, t1.x), xd23 = __fsub_rn(t0.x, t1.x);
        fold_d<S, HC>(k1, Gc, __fadd_rn(xd01, xd23), v.x, A.D[0]);
        fold_d<S, HC>(k1, Gc, __fsub_rn(xs01, xs23), v.y, A.D[1]);
        fold_d<S, HC>(k1, Gc, __fadd_rn(xs01, xs23), v.z, A.D[2]);
    }
    if constexpr (!DRAG) {
        const Odd<VA<S>> v = corner_odd<VA<S>>(ps01, pd01, t0.p + t1.p, t0.p - t1.p);
        A.P[0] = va_fma(k2, v.x, A.P[0]);
        A.P[1] = va_fma(k2, v.y, A.P[1]);
        A.P[2] = va_fma(k2, v.z, A.P[2]);
    }
}

// 2 g_ref + dg(r) per a
template <int S>
__device__ __forceinline__ VA<S> twice_g(const mlbi_params &p, const float (&dgc)[S * (S + 1) / 2], int b)
{
    return va_make<S>([&](int a) { return fmaf(2.f, p.pair[pair_of(a, b, S)].g_ref, dgc[pair_of(a, b, S)]); });
}

// sums of neighbour species b
template <int S, bool DRAG, bool HC, class V>
__device__ __forceinline__ void p1_cube_species(const mlbi_params &p, const V &c, int b,
                                                const float (&dgc)[S * (S + 1) / 2], const float (&ub)[3],
                                                PairSums<S> &A)
{
    const float nr = p.nref[b];
    const VA<S> Gc = twice_g<S>(p, dgc, b);
#pragma unroll
    for (int k = 0; k < 3; ++k) A.D[k] = A.P[k] = A.E[k] = A.E[k + 3] = va_zero<S>();
    p1_axis<S, DRAG, HC>(p, c, b, nr, Gc, ub, A);
    VA<S> m;
    if (class_mask<S, 1>(p, b, m)) {
        const VA<S> k1 = cls_il(1) * m, k2 = 0.5f * m;
        p1_face<S, DRAG, HC, 0, 1>(c, b, nr, Gc, ub, k1, k2, A);
        p1_face<S, DRAG, HC, 0, 2>(c, b, nr, Gc, ub, k1, k2, A);
        p1_face<S, DRAG, HC, 1, 2>(c, b, nr, Gc, ub, k1, k2, A);
    }
    p1_corner<S, DRAG, HC>(p, c, b, nr, Gc, ub, A);
}

// ------------------------------------------------------------------ pass 2
// exchange only, at the staged velocities relative to u^a(r) (the friction
// matrix is not needed, so the relative velocity is taken per a):
// P = W+ j+ + W- j-, j+- = e.(u^b(r +- d) - u^a(r)); drag only: (W+ + W-) e.(u^b - u^a)(r)
template <int S, bool DRAG, int X, int Y, int Z, class V>
__device__ __forceinline__ VA<S> p2_point(const V &c, int b, float nr, const VA<S> &Gc,
                                          const VA<S> (&ua)[3], const float (&ub)[3])
{
    const float4 vp = c.template field<X, Y, Z>(b), vm = c.template field<-X, -Y, -Z>(b);
    const VA<S> gp = c.template dg<X, Y, Z>(b), gm = c.template dg<-X, -Y, -Z>(b);
    const float np = __fadd_rn(nr, vp.x), nm = __fadd_rn(nr, vm.x);
    const VA<S> wp = np * (Gc + gp), wm = nm * (Gc + gm);
    const VA<S> ea = edot_va<S, X, Y, Z>(ua);
    if constexpr (DRAG) {
        const float eb = edot<X, Y, Z>(ub[0], ub[1], ub[2]);
        return (wp + wm) * (va_make<S>([&](int) { return eb; }) - ea);
    } else {
        const float jp = edot<X, Y, Z>(vp.y, vp.z, vp.w), jm = edot<X, Y, Z>(vm.y, vm.z, vm.w);
        const VA<S> jpa = va_make<S>([&](int) { return jp; }) - ea, jma = va_make<S>([&](int) { return jm; }) - ea;
        return va_fma(wm, jma, wp * jpa);
    }
}

// adds to P[3] the exchange sums of neighbour species b
template <int S, bool DRAG, class V>
__device__ __forceinline__ void p2_cube_species(const mlbi_params &p, const V &c, int b,
                                                const float (&dgc)[S * (S + 1) / 2], const VA<S> (&ua)[3],
                                                const float (&ub)[3], VA<S> (&P)[3])
{
    const float nr = p.nref[b];
    const VA<S> Gc = twice_g<S>(p, dgc, b);
    const VA<S> k = va_make<S>([&](int a) { return 0.5f * p.pair[pair_of(a, b, S)].vx_pre; });
    VA<S> m;
    if (class_mask<S, 0>(p, b, m)) {
        const VA<S> km = k * m;
        P[0] = va_fma(km, p2_point<S, DRAG, 1, 0, 0>(c, b, nr, Gc, ua, ub), P[0]);
        P[1] = va_fma(km, p2_point<S, DRAG, 0, 1, 0>(c, b, nr, Gc, ua, ub), P[1]);
        P[2] = va_fma(km, p2_point<S, DRAG, 0, 0, 1>(c, b, nr, Gc, ua, ub), P[2]);
    }
    if (class_mask<S, 1>(p, b, m)) {
        const VA<S> km = 0.5f * (k * m);
        VA<S> tp = p2_point<S, DRAG, 1, 1, 0>(c, b, nr, Gc, ua, ub);
        VA<S> tm = p2_point<S, DRAG, -1, 1, 0>(c, b, nr, Gc, ua, ub);
        VA<S> vx = tp - tm, vy = tp + tm;
        tp = p2_point<S, DRAG, 1, 0, 1>(c, b, nr, Gc, ua, ub);
        tm = p2_point<S, DRAG, -1, 0, 1>(c, b, nr, Gc, ua, ub);
        vx = vx + (tp - tm);
        VA<S> vz = tp + tm;
        tp = p2_point<S, DRAG, 0, 1, 1>(c, b, nr, Gc, ua, ub);
        tm = p2_point<S, DRAG, 0, -1, 1>(c, b, nr, Gc, ua, ub);
        vy = vy + (tp - tm);
        vz = vz + (tp + tm);
        P[0] = va_fma(km, vx, P[0]);
        P[1] = va_fma(km, vy, P[1]);
        P[2] = va_fma(km, vz, P[2]);
    }
    if (class_mask<S, 2>(p, b, m)) {
        const VA<S> km = (1.f / 3.f) * (k * m);
        VA<S> t0 = p2_point<S, DRAG, 1, 1, 1>(c, b, nr, Gc, ua, ub);
        VA<S> t1 = p2_point<S, DRAG, -1, 1, 1>(c, b, nr, Gc, ua, ub);
        const VA<S> s01 = t0 + t1, d01 = t0 - t1;
        t0 = p2_point<S, DRAG, 1, -1, 1>(c, b, nr, Gc, ua, ub);
        t1 = p2_point<S, DRAG, -1, -1, 1>(c, b, nr, Gc, ua, ub);
        const Odd<VA<S>> v = corner_odd<VA<S>>(s01, d01, t0 + t1, t0 - t1);
        P[0] = va_fma(km, v.x, P[0]);
        P[1] = va_fma(km, v.y, P[1]);
        P[2] = va_fma(km, v.z, P[2]);
    }
}

}  // namespace
