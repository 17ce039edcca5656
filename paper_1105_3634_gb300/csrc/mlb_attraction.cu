// mlb_attraction.cu -- the attractive mean field of the RPA (Sec. III, G term
// of Eq. potmeanforce) as a column stencil on sm_103a.
//
// G^a(r) = sum_b sum_d K_ab(d) n^b(r + d), K_ab(d) = 6 eps_ab sigma_ab^6 d / |d|^8
// on sigma_ab <= |d| <= lambda_c sigma_ab.  K is odd, so n may be replaced by
// the deviation n - n_ref (the constant part sums to zero over the region).
//
// The kernel k(d) = 6 eps sigma^6 / |d|^8 (zero off the region) depends on |d|
// only, so the columns (dx, dy) along z come in groups that share their weights:
// (+-X, +-Y) and (+-Y, +-X), eight columns for X > Y > 0, four for Y = 0 or X = Y,
// one for (0, 0).  With the plane sums over a group
//   A = sum dx n(x + dx, y + dy, .), B = sum dy n(..), C = sum n(..)
// every output plane z takes
//   G_x += k(dz) A(z + dz), G_y += k(dz) B(z + dz),
//   G_z += dz k(dz) (C(z + dz) - C(z - dz)) for dz > 0
// whatever the number of columns (each half-plane column took four multiply-adds
// per dz and species before).
// Each thread owns Z consecutive planes of one (x, y) site and streams the
// planes: a plane's A and B are formed once and added to all Z outputs and both
// output species (packed FP32x2), C is kept for the differences.  A group's sums
// are formed by themselves and added to the running ones once: with every plane added
// straight in, several hundred terms, the error against 64 bits grew beyond that of a
// sum by columns on many fields (sigma = 2 / 3, 40 x 20 x 18, largest error over
// largest |G|, by half-plane columns / planes added straight in / this form:
// wave along x 4.1e-7 / 9.0e-7 / 2.2e-7, along z 1.2e-6 / 2.3e-7 / 1.1e-7, noise 8.1e-7 /
// 5.7e-7 / 2.6e-7).  An output's partial sum is live from its first plane to its last
// only, which keeps two species within 128 registers.  A block stages the deviations of
// one neighbour species over its (32 + 2R) x (TY + 2R) x (Z + 2R) slab in shared
// memory.  (sigma = 2 / 3, reach 7, 128^3: half-plane columns 0.868 ms, planes added
// straight in 0.707, this form 0.742.)
#include "mlb_internal.h"
#include "mlb_device.cuh"
#include "mlb_cube.cuh"

namespace {

template <int S, int R, int TY, int Z>
struct CTile {
    static constexpr int TXH = kBX + 2 * R, TYH = TY + 2 * R, TZH = Z + 2 * R;
    static constexpr int PL = TXH * TYH;                   // one slab plane
    static constexpr int NT = kBX * TY;                    // threads
    // output species per pass: pairs, an odd one out with itself (three species with tails
    // to 6 sites, 64^3: one by one 0.550 ms, 0.415 so; half-plane columns 0.590)
    static constexpr int AG = S == 1 ? 1 : 2;
    static constexpr size_t bytes = (size_t)PL * TZH * sizeof(float);
};

// stage n^b - n_ref^b of the block's slab; beyond a wall there are no particles (n = 0)
template <int S, int R, int TY, int Z>
__device__ __forceinline__ void stage_slab(const mlbi_params &p, int x0, int y0, int z0,
                                           const float4 *__restrict__ momb, float nrefb, float *slab)
{
    using T = CTile<S, R, TY, Z>;
    const int tid = threadIdx.y * kBX + threadIdx.x;
    for (int idx = tid; idx < T::PL; idx += T::NT) {
        const int hx = idx % T::TXH, hy = idx / T::TXH;
        const int x = wrap_or_out(x0 - R + hx, p.nx, p.wall_axis == 0);
        const int y = wrap_or_out(y0 - R + hy, p.ny, p.wall_axis == 1);
        const long long xy = (x < 0 || y < 0) ? -1 : x + (long long)p.nx * y;
        const long long nxy = (long long)p.nx * p.ny;
        for (int hz = 0; hz < T::TZH; ++hz) {
            const int z = wrap_or_out(z0 - R + hz, p.nz, p.wall_axis == 2);
            float *d = slab + hz * T::PL + idx;
            if (xy < 0 || z < 0) *d = -nrefb;
            else cp_async4(d, reinterpret_cast<const float *>(momb + xy + nxy * z));
        }
    }
    cp_async_commit();
}

template <int S, int R, int TY, int Z>
__global__ void __launch_bounds__(kBX * TY, 2) k_attraction_columns(const mlbi_params p,
                                                                    const float4 *__restrict__ mom,
                                                                    const float4 *__restrict__ cols,
                                                                    const float *__restrict__ wts,
                                                                    float4 *__restrict__ attr)
{
    using T = CTile<S, R, TY, Z>;
    constexpr int AG = T::AG, W = T::TZH;
    step_begin();
    extern __shared__ float slab[];                         // [TZH][TYH][TXH]
    const int x0 = blockIdx.x * kBX, y0 = blockIdx.y * TY, z0 = blockIdx.z * Z;
    const int x = x0 + threadIdx.x, y = y0 + threadIdx.y;
    const float *centre = slab + (threadIdx.y + R) * T::TXH + threadIdx.x + R;
    const int stride = p.attr_r + 1;
    for (int a0 = 0; a0 < S; a0 += AG) {
        VA<AG> acc[Z][3];
#pragma unroll
        for (int i = 0; i < Z; ++i) acc[i][0] = acc[i][1] = acc[i][2] = va_zero<AG>();
        for (int b = 0; b < S; ++b) {
            __syncthreads();                                 // the previous slab is consumed
            stage_slab<S, R, TY, Z>(p, x0, y0, z0, mom + b * p.N, p.nref[b], slab);
            cp_async_wait_all();
            __syncthreads();
            for (int c = 0; c < p.acol_count; ++c) {
                const float4 cc = __ldg(&cols[c]);
                const int X = __float_as_int(cc.x), Y = __float_as_int(cc.y), E = __float_as_int(cc.z);
                const float fx = (float)X, fy = (float)Y;
                const int yr = Y * T::TXH, xr = X * T::TXH;
                VA<AG> k[R + 1];
#pragma unroll
                for (int dz = 0; dz <= R; ++dz) {
                    const bool in = dz <= p.attr_r;          // a tier may reach beyond the region
                    k[dz] = va_make<AG>([&](int g) {
                        const int a = S % AG == 0 ? a0 + g : min(a0 + g, S - 1);
                        return in ? __ldg(&wts[(c * p.npairs + pair_of(a, b, S)) * stride + dz]) : 0.f;
                    });
                }
                // Opposite columns are subtracted first (what they share is exact to
                // cancel), then C's planes z + dz and z - dz below.
                float C[W];
                VA<AG> t[Z][2];                              // this group's share of G_x, G_y
#pragma unroll
                for (int j = 0; j < W; ++j) {
                    C[j] = 0.f;
                    if (j < Z) t[j][0] = t[j][1] = va_zero<AG>();
                    if (j >= R - E && j < R + Z + E) {              // uniform: some output reaches this plane
                        const float *v = centre + j * T::PL;
                        float A, B;
                        if (Y > 0 && X > Y) {
                            const float pp = v[X + yr], pm = v[X - yr], mp = v[-X + yr], mm = v[-X - yr];
                            const float qp = v[Y + xr], qm = v[Y - xr], rp = v[-Y + xr], rm = v[-Y - xr];
                            const float d1 = pp - mm, d2 = pm - mp, e1 = qp - rm, e2 = qm - rp;
                            A = fmaf(fx, d1 + d2, fy * (e1 + e2));
                            B = fmaf(fy, d1 - d2, fx * (e1 - e2));
                            C[j] = ((pp + mm) + (pm + mp)) + ((qp + rm) + (qm + rp));
                        } else if (Y > 0) {
                            const float pp = v[X + yr], pm = v[X - yr], mp = v[-X + yr], mm = v[-X - yr];
                            const float d1 = pp - mm, d2 = pm - mp;
                            A = fx * (d1 + d2);
                            B = fx * (d1 - d2);
                            C[j] = (pp + mm) + (pm + mp);
                        } else if (X > 0) {
                            const float xp = v[X], xm = v[-X], yp = v[xr], ym = v[-xr];
                            A = fx * (xp - xm);
                            B = fx * (yp - ym);
                            C[j] = (xp + xm) + (yp + ym);
                        } else {
                            A = B = 0.f;
                            C[j] = v[0];
                        }
#pragma unroll
                        for (int i = 0; i < Z; ++i) {
                            const int dz = j - R - i;
                            if (dz < -R || dz > R) continue;
                            const int m = dz < 0 ? -dz : dz;
                            t[i][0] = va_fma(A, k[m], t[i][0]);
                            t[i][1] = va_fma(B, k[m], t[i][1]);
                        }
                    }
                    if (j >= 2 * R) {                               // output j - 2R has all its planes
                        acc[j - 2 * R][0] = acc[j - 2 * R][0] + t[j - 2 * R][0];
                        acc[j - 2 * R][1] = acc[j - 2 * R][1] + t[j - 2 * R][1];
                    }
                }
                VA<AG> tz[Z];
#pragma unroll
                for (int i = 0; i < Z; ++i) tz[i] = va_zero<AG>();
#pragma unroll
                for (int dz = 1; dz <= R; ++dz) {
                    if (dz > E) break;
                    const VA<AG> kz = (float)dz * k[dz];
#pragma unroll
                    for (int i = 0; i < Z; ++i) tz[i] = va_fma(C[i + R + dz] - C[i + R - dz], kz, tz[i]);
                }
#pragma unroll
                for (int i = 0; i < Z; ++i) acc[i][2] = acc[i][2] + tz[i];
            }
        }
        if (x < p.nx && y < p.ny) {
#pragma unroll
            for (int g = 0; g < AG; ++g)
#pragma unroll
                for (int i = 0; i < Z; ++i) {
                    const int z = z0 + i;
                    if (z < p.nz && a0 + g < S) {
                        const long long r = x + (long long)p.nx * (y + (long long)p.ny * z);
                        attr[(a0 + g) * p.N + r] = make_float4(va_get<AG>(acc[i][0], g), va_get<AG>(acc[i][1], g),
                                                               va_get<AG>(acc[i][2], g), 0.f);
                    }
                }
        }
    }
}

}  // namespace

constexpr int kAttrTY = 8, kAttrZ = 8;

template <int S, int R>
cudaError_t launch_columns(const mlbi_params &p, const mlbi_buffers &b, cudaStream_t s)
{
    using T = CTile<S, R, kAttrTY, kAttrZ>;
    auto k = k_attraction_columns<S, R, kAttrTY, kAttrZ>;
    cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)T::bytes);
    if (e != cudaSuccess) return e;
    const dim3 g((unsigned)((p.nx + kBX - 1) / kBX), (unsigned)((p.ny + kAttrTY - 1) / kAttrTY),
                 (unsigned)((p.nz + kAttrZ - 1) / kAttrZ));
    const float4 *cols = reinterpret_cast<const float4 *>(b.table) + p.acol_start;
    const float *wts = reinterpret_cast<const float *>(reinterpret_cast<const float4 *>(b.table) + p.aw_start);
    return launch_step(k, g, dim3(kBX, kAttrTY), T::bytes, s, p, b.mom, cols, wts, b.attr);
}

// reach tiers: the smallest tier >= the attraction reach (a wider halo than
// needed is harmless: columns and weights stop at the true reach)
template <int S>
cudaError_t attraction_for_reach(const mlbi_params &p, const mlbi_buffers &b, cudaStream_t s)
{
    if (p.attr_r <= 3) return launch_columns<S, 3>(p, b, s);
    if (p.attr_r <= 5) return launch_columns<S, 5>(p, b, s);
    if (p.attr_r <= 7) return launch_columns<S, 7>(p, b, s);
    if (p.attr_r <= 8) return launch_columns<S, 8>(p, b, s);
    return cudaErrorInvalidValue;
}

cudaError_t mlbi_launch_attraction(const mlbi_params &p, const mlbi_buffers &b, cudaStream_t s)
{
    if (p.acol_count <= 0) return cudaErrorInvalidValue;
    MLBI_DISPATCH_S(return attraction_for_reach<SS>(p, b, s));
    return cudaErrorInvalidValue;
}
