// Cell tiles staged in shared memory: a CTA owns a box of cells and stages the
// particles of the box and of its halo (the cells within the search reach R).
// The shape of the tiles and the arithmetic of their cells, shared by the gas
// pair sums and the cross-phase sums.
#pragma once

#include <algorithm>
#include <cmath>

#include "pair.cuh"

namespace tfsph {

struct TileCfg {
    int T[3];     // owned cells per axis
    int H[3];     // halo cells per axis (T + 2R)
    int nt[3];    // tiles per axis
    int nhalo;    // H0 H1 H2
    int nrows;    // T1 T2 owned rows
    int cap;      // particles that fit in shared memory
    int offset;   // byte offset of the particle arrays in shared memory
    int lanes = 1;  // lanes per owned particle (listing passes of small 3D problems)
    float invH[2];  // 1 / H0, 1 / H1
};

// Bytes of the 16-bit halo-cell offsets (nhalo + 1 of them), padded to 4.
__host__ __device__ constexpr long lstart_bytes(long nhalo) { return (2 * (nhalo + 1) + 3) / 4 * 4; }

// q = floor(x / d) for 0 <= x < 2^22 and 0 < d < 2^10 by a float multiply with
// the rounded reciprocal: (x + 1/2)/d lies at least 1/(2d) from an integer,
// more than the product's rounding error, so the truncation is exact.
__device__ __forceinline__ int small_div(int x, int d, float inv_d)
{
    return (int)(((float)x + 0.5f) * inv_d);
}

// Halo cell h -> (hx, hy, hz), without integer division.
__device__ __forceinline__ void halo_coords(int h, const TileCfg &C, int &hx, int &hy, int &hz)
{
    const int row = small_div(h, C.H[0], C.invH[0]);
    hx = h - row * C.H[0];
    hz = small_div(row, C.H[1], C.invH[1]);
    hy = row - hz * C.H[1];
}

// In-place exclusive scan of m values in shared memory by the whole block;
// a[m] receives the total, which is also returned (exact in int when the
// 16-bit form truncates the stored sums).
template <class E>
__device__ inline int block_scan_smem(E *a, int m, int *wsum)
{
    const int tid = threadIdx.x, nth = blockDim.x;
    const int chunk = (m + nth - 1) / nth;
    const int b0 = min(m, tid * chunk), b1 = min(m, b0 + chunk);
    int s = 0;
    for (int i = b0; i < b1; ++i) s += a[i];
    const int lane = tid & 31, wid = tid >> 5;
    int x = s;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y;
    }
    if (lane == 31) wsum[wid] = x;
    __syncthreads();
    if (wid == 0) {
        int t = lane < (nth >> 5) ? wsum[lane] : 0;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int y = __shfl_up_sync(0xffffffffu, t, o);
            if (lane >= o) t += y;
        }
        if (lane < (nth >> 5)) wsum[lane] = t;
    }
    __syncthreads();
    const int total = wsum[(nth >> 5) - 1];
    int run = (wid > 0 ? wsum[wid - 1] : 0) + x - s;
    for (int i = b0; i < b1; ++i) {
        const int v = a[i];
        a[i] = (E)run;
        run += v;
    }
    if (tid == nth - 1) a[m] = (E)run;
    __syncthreads();
    return total;
}

// First plane from oz0 on that belongs to lane sub of step lanes (a power of
// two), a plane's lane being its distance from plane -R modulo step: the lanes
// of a particle then share out the planes whatever window each of them takes
// (one whose list overflows walks in other arithmetic than the others).
__host__ __device__ __forceinline__ int first_plane(int oz0, int R, int sub, int step)
{
    return oz0 + ((sub - (oz0 + R)) & (step - 1));
}

// Global cell coordinate of halo coordinate hc along axis k (-1: none).
template <class T>
__device__ __forceinline__ int halo_cell(const Geo<T> &G, int k, int c0, int hc)
{
    return axis_wrap(c0 - G.R[k] + hc, G.n[k], G.per[k]);
}

// 1 if halo coordinate hc along axis k lies across the periodic seam.
template <class T>
__device__ __forceinline__ int halo_seam(const Geo<T> &G, int k, int c0, int hc)
{
    const int g = c0 - G.R[k] + hc;
    return G.per[k] && (g < 0 || g >= G.n[k]);
}

// Tile shape for a phase with `mean` particles per cell. The CTA's threads
// take the owned particles in turn; a tile holds about 7/8 of them per
// thread, or 1.97 (two nearly full passes) where the halo of R cells staged
// around it outweighs it (in 3D with R = 3: 8 halo cells per owned cell for
// 6^3 owned cells, 5.5 for 10 x 7 x 7), so that the halo is spread over more
// particles; in 1D and 2D, with cells of 2h (R = 1), the halo is small and
// the second pass would cost more than it saves. Its expected halo must fill at most 90 %
// of the shared-memory capacity (a tile whose halo exceeds it takes the
// global-memory walk; the 3D box's halos stay within 4 % of their mean).
// Returns false when an axis wraps fully.
// lanes > 1: small tiles, of one pass with that many threads per particle.
template <class T>
bool plan_tiles(const Geo<T> &G, int dim, double mean, int bytes_pp, int smem_budget, int threads, TileCfg &C,
                size_t &smem, int lanes = 1)
{
    for (int k = 0; k < dim; ++k)
        if (G.full[k]) return false;
    int Tt[3] = {1, 1, 1};
    // owned cells for about `per_thread` owned particles per thread
    auto shape = [&](double per_thread) {
        const double target_cells = std::max(1.0, per_thread * threads / std::max(mean, 1e-6));
        const int side = std::max(1, (int)std::floor(std::pow(target_cells, 1.0 / dim) + 1e-9));
        Tt[0] = Tt[1] = Tt[2] = 1;
        for (int k = 1; k < dim; ++k) Tt[k] = std::min(side, G.n[k]);
        double rest = 1.0;
        for (int k = 1; k < dim; ++k) rest *= Tt[k];
        Tt[0] = std::max(1, std::min(G.n[0], (int)std::floor(target_cells / rest + 1e-9)));
    };
    // one pass over the owned particles (7/8 of the threads) unless the halo
    // outweighs the tile (more than 3 halo cells per owned cell, as in 3D
    // with R = 3), then two nearly full passes to spread it
    shape(0.875 / lanes);
    double halo_ratio = 1.0;
    for (int k = 0; k < dim; ++k) halo_ratio *= (double)(Tt[k] + 2 * G.R[k]) / (double)Tt[k];
    if (halo_ratio > 3.0 && lanes == 1) shape(1.97);
    for (;;) {
        int H[3] = {1, 1, 1};
        long nh = 1;
        for (int k = 0; k < dim; ++k) {
            H[k] = Tt[k] + 2 * G.R[k];
            nh *= H[k];
        }
        const long nrows = (long)Tt[1] * Tt[2];
        const long nhr = (long)H[1] * H[2];
        // the halo cells' 16-bit offsets, the owned rows' prefix and starts,
        // the halo rows' starts and offsets
        const long table = lstart_bytes(nh) + 4 * (2 * nrows + 1 + 2 * nhr + 1);
        const long offset = (table + 63) / 64 * 64;
        const long cap = (smem_budget - offset) / bytes_pp;
        const double expected = mean * (double)nh;
        int kmax = 0;
        for (int k = 1; k < dim; ++k)
            if (Tt[k] > Tt[kmax]) kmax = k;
        if ((cap > 0 && expected <= 0.9 * (double)cap) || Tt[kmax] == 1) {
            if (cap <= 0 || nh >= (1L << 22) || H[0] >= 1024 || H[1] >= 1024) return false;
            for (int k = 0; k < 3; ++k) {
                C.T[k] = Tt[k];
                C.H[k] = H[k];
                C.nt[k] = k < dim ? (G.n[k] + Tt[k] - 1) / Tt[k] : 1;
            }
            C.nhalo = (int)nh;
            C.nrows = (int)nrows;
            C.invH[0] = 1.0f / (float)H[0];
            C.invH[1] = 1.0f / (float)H[1];
            C.cap = (int)cap;
            C.offset = (int)offset;
            C.lanes = lanes;
            smem = (size_t)offset + (size_t)cap * (size_t)bytes_pp;
            return true;
        }
        Tt[kmax] = (Tt[kmax] + 1) / 2;
    }
}

}  // namespace tfsph
