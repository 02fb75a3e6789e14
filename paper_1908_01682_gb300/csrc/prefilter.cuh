// Rows of staged halo cells and the distance test of the binary32 prefilter
// of the binary64 3D density (sph.cu): which candidates a particle of a tile
// looks at before the pair sums run over the recorded ones in binary64. All
// lengths are in units of h, relative to the tile's corner.
#pragma once

#include "pair.cuh"
#include "tile.cuh"

namespace tfsph {

struct Prefilter {
    float w[3], inv_w[3];  // cell edges and their inverses
    // Largest coordinate the margins below hold for: the tile's halo. A tile
    // that stages a particle beyond it (outside the box along an open axis)
    // takes its candidates in binary64.
    float far;
    float reach2;  // squared radius of the rows
    float thr;     // squared radius of the candidates
};

// Relative coordinates are below `far`, each rounded to 2^-24 far: 2^-19 far
// covers the displacement; the rest covers the arithmetic here.
template <class T> __host__ __device__ __forceinline__ Prefilter prefilter_of(const Geo<T> &G, const TileCfg &C)
{
    Prefilter P;
    P.far = 0.0f;
    for (int d = 0; d < 3; ++d) {
        P.w[d] = (float)(G.w[d] * G.inv_h);
        P.inv_w[d] = (float)(G.inv_w[d] * G.h);
        P.far = fmaxf(P.far, (float)C.H[d] * P.w[d]);
    }
    const float reach = 2.0f + 0x1p-19f * P.far;
    P.reach2 = reach * reach * (1.0f + 0x1p-18f) + 0x1p-19f * P.far * reach;
    P.thr = reach * reach * (1.0f + 0x1p-20f);
    return P;
}

__host__ __device__ __forceinline__ bool prefilter_holds(const Prefilter &P, float x, float y, float z)
{
    return fmaxf(fmaxf(fabsf(x), fabsf(y)), fabsf(z)) <= P.far && x == x && y == y && z == z;
}

__host__ __device__ __forceinline__ float prefilter_sqrt(float x)
{
#ifdef __CUDA_ARCH__
    return approx_sqrt(x);
#else
    return sqrtf(x);
#endif
}

__host__ __device__ __forceinline__ int prefilter_floor(float x)
{
#ifdef __CUDA_ARCH__
    return floor_int(x);
#else
    return (int)floorf(x);
#endif
}

// Calls row(u0, u1) with the half-open range of halo cells, u0 <= u1, of
// every row within reach of a particle in halo cell h at fractions f of it;
// lane sub of step lanes takes its planes (first_plane). h is the rounded estimate
// of the cell, up to one off the cell the particle is stored in, and the
// margins widen the radius, so a range may end past the staged halo where 2h
// is just short of a whole number of cells; no neighbour lies there, and the
// ranges are cut to the halo.
template <class Row>
__host__ __device__ __forceinline__ void prefilter_rows(const Prefilter &P, const int R[3], const int H[3],
                                                        const int h[3], const float f[3], int sub, int step, Row &&row)
{
    const float tz = prefilter_sqrt(P.reach2) * P.inv_w[2];
    const int oz1 = min(min(R[2], max(0, prefilter_floor(f[2] + tz))), H[2] - 1 - h[2]);
    const int oz0 = max(-min(R[2], max(0, prefilter_floor(tz - f[2] + 1.0f))), -h[2]);
#pragma unroll 1
    for (int oz = first_plane(oz0, R[2], sub, step); oz <= oz1; oz += step) {
        const float sz = slab_dist(oz, f[2]) * P.w[2], dz2 = sz * sz;
        const float ty = prefilter_sqrt(fmaxf(P.reach2 - dz2, 0.0f)) * P.inv_w[1];
        const int oy1 = min(min(R[1], max(0, prefilter_floor(f[1] + ty))), H[1] - 1 - h[1]);
        const int oy0 = max(-min(R[1], max(0, prefilter_floor(ty - f[1] + 1.0f))), -h[1]);
#pragma unroll 1
        for (int oy = oy0; oy <= oy1; ++oy) {
            const float sy = slab_dist(oy, f[1]) * P.w[1];
            const float tx = prefilter_sqrt(fmaxf(P.reach2 - dz2 - sy * sy, 0.0f)) * P.inv_w[0];
            const int ohi = min(R[0], max(0, prefilter_floor(f[0] + tx)));
            const int olo = -min(R[0], max(0, prefilter_floor(tx - f[0] + 1.0f)));
            const int hrow = H[0] * ((h[1] + oy) + H[1] * (h[2] + oz));
            const int u0 = min(max(h[0] + olo, 0), H[0]);
            row(hrow + u0, hrow + max(u0, min(h[0] + ohi + 1, H[0])));
        }
    }
}

__host__ __device__ __forceinline__ bool prefilter_near(const Prefilter &P, float dx, float dy, float dz)
{
    return fmaf(dz, dz, fmaf(dy, dy, dx * dx)) < P.thr;
}

}  // namespace tfsph
