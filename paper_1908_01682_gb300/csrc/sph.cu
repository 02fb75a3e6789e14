// SPH pair sums over cell lists: summation density (rho^n of Eq. 19, with
// the equation of state) and the gas pressure (+ artificial viscosity)
// acceleration of the first term of Eq. 19, with the adiabatic energy rate.
//
// Tiled path (default). One CTA owns a box of cells. It stages the particles
// of the box and of its halo (the cells within the search reach R) into
// shared memory once, with a local table of cell starts, and then each thread
// takes one owned particle and walks its candidate rows in shared memory.
// Rows and row ends whose slab lies farther than 2h (plus a rounding margin)
// from the particle are skipped. The halo cells that lie across a periodic
// seam are known per row segment, so the inner loop of the common case is a
// plain difference of coordinates; seam segments use the two-sum displacement
// below. A tile whose halo does not fit in shared memory computes from global
// memory with the same arithmetic.
//
// Neighbour membership r^2 < 4h^2 is evaluated with explicitly rounded
// operations so that it is a plain IEEE decision, the same one the checker
// takes.
#include <algorithm>
#include <cmath>

#include "pair.cuh"
#include "prefilter.cuh"
#include "tile.cuh"

namespace tfsph {
namespace {

constexpr int kTileThreads = 256;
// Shared memory of a tile that stages positions only (density, isothermal
// force): 4 CTAs per SM, each with its static arrays and the 1 KB the
// hardware reserves, within the SM's 228 KB (4 x (56832 + 64 + 1024) bytes).
constexpr int kTileSmemPos = 56832;
// The same for the binary64 state in 3D, whose tiles also hold a binary32 copy
// of the positions: 2 CTAs per SM. They are bound by the binary64 pipe, which
// a few warps fill.
constexpr int kTileSmemWide = 112 * 1024;
template <class T, int DIM> constexpr bool kPrefilter = sizeof(T) == 8 && DIM == 3;

// One thread per particle, candidates from global memory.
template <class T, int DIM, int MODE>
__global__ void __launch_bounds__(128, 1)
k_pair_global(Geo<T> G, Phys<T> Ph, const V4<T> *__restrict__ pos, const V4<T> *__restrict__ vel,
              const T *__restrict__ rho, const uint32_t *__restrict__ id, const uint32_t *__restrict__ start, int n,
              T mass, T *__restrict__ out_rho, T *pr_out, V4<T> *__restrict__ out_acc, int32_t *__restrict__ cnt,
              uint64_t *__restrict__ fpr)
{
    const int a = blockIdx.x * blockDim.x + threadIdx.x;
    if (a >= n) return;
    const V4<T> pa = pos[a];
    PairAcc<T, MODE> A;
    acc_init(A, Ph, pa, vel, rho, a);
    walk_global<T, DIM, MODE>(A, G, Ph, pa, pos, vel, rho, id, start);
    acc_store(A, Ph, a, mass, vel, out_rho, pr_out, out_acc, cnt, fpr);
}

// ---------------------------------------------------------------------------
// Tiled path
// ---------------------------------------------------------------------------
// Appends the neighbours the density walk finds to the particle's list:
// entry n goes to slot n mod 4 of group n / 4 (16-bit stores; the force pass
// reads whole groups). Groups beyond cap entries go to the tile's spare
// group (never read), which keeps the store unconditional.
struct NbRec {
    unsigned long long *base;  // group 0 of the particle
    uint32_t stride;           // owned_cap ((cap + 1) * owned_cap < 2^31: slot offsets fit 32 bits)
    int gcap;                  // cap / 4: the spare group
    int n;
    __device__ __forceinline__ void push(int j, bool seam)
    {
        const uint32_t g = (uint32_t)min(n >> 2, gcap);
        reinterpret_cast<uint16_t *>(base)[((g * stride) << 2) + (uint32_t)(n & 3)] =
            (uint16_t)((uint32_t)j | (seam ? kNbSeam : 0u));
        ++n;
    }
};

template <class T, int DIM, int MODE, bool SEAM, bool REC>
__device__ __forceinline__ void walk_smem_range(PairAcc<T, MODE> &A, const Geo<T> &G, const Phys<T> &Ph,
                                                const V4<T> &pa, const V4<T> *spos, const V4<T> *svel,
                                                const T *srho, const uint32_t *sid, int j0, int j1, NbRec *rec)
{
    // a row holds a few candidates: no unrolled prologue or remainder
#pragma unroll 1
    for (int j = j0; j < j1; ++j) {
        const V4<T> pb = spos[j];
        T d[3];
        const T r2 = pair_r2<T, DIM, SEAM>(G, pa, pb, d);
        if (REC) {
            if (r2 < G.h2x4) {
                A.template add<DIM>(G, Ph, pb, nullptr, T(1), 0u, r2, d);
                rec->push(j, SEAM);
            }
        } else if (ModeUses<MODE>::vel || ModeUses<MODE>::rho) {
            if (r2 < G.h2x4)
                A.template add<DIM>(G, Ph, pb, ModeUses<MODE>::vel ? &svel[j] : nullptr,
                                    ModeUses<MODE>::rho ? srho[j] : T(1), 0u, r2, d);
        } else {
            A.template add<DIM>(G, Ph, pb, nullptr, T(1), MODE == 1 ? sid[j] : 0u, r2, d);
        }
    }
}

// Candidate walk of one owned particle over the staged tile (REC: the
// density pass recording the neighbour list; SEAMLESS: no halo cell of the
// tile lies across a periodic seam, or the tile was staged with its seam
// shifts, so every row is one plain range). Each row is walked in the order
// of its staged cells in either case.
template <class T, int DIM, int MODE, bool REC, bool SEAMLESS>
__device__ __forceinline__ void walk_tile(PairAcc<T, MODE> &A, const Geo<T> &G, const Phys<T> &Ph, const TileCfg &C,
                                          const int c0[3], const V4<T> &pa, const V4<T> &pc, const uint16_t *lstart,
                                          const V4<T> *spos, const V4<T> *svel, const T *srho, const uint32_t *sid,
                                          NbRec *rec, int sub = 0, int step = 1)
{
    // (step > 1, 3D: lane sub of step lanes, which takes its planes)
    // pa: the staged (possibly shifted) position the displacements use;
    // pc: the same position in box coordinates, for its cell and window
    T tx_, ty_ = T(0), tz_ = T(0);
    const int cx = axis_cell(pc.x, G.lo[0], G.inv_w[0], G.n[0], tx_);
    const int cy = DIM > 1 ? axis_cell(pc.y, G.lo[1], G.inv_w[1], G.n[1], ty_) : 0;
    const int cz = DIM > 2 ? axis_cell(pc.z, G.lo[2], G.inv_w[2], G.n[2], tz_) : 0;
    const T fx = tx_ - T(cx);
    const T fy = DIM > 1 ? ty_ - T(cy) : T(0);
    const T fz = DIM > 2 ? tz_ - T(cz) : T(0);
    const int hx = cx - c0[0] + G.R[0];
    const int hy = DIM > 1 ? cy - c0[1] + G.R[1] : 0;
    const int hz = DIM > 2 ? cz - c0[2] + G.R[2] : 0;
    // x seam bounds in halo coordinates: cells below sx0 or from sx1 on lie across
    const int sx0 = G.per[0] ? G.R[0] - c0[0] : -1;
    const int sx1 = G.per[0] ? G.n[0] - c0[0] + G.R[0] : C.H[0] + 1;
    // z and y offsets limited by the closed form of the x window; a row may
    // come out one cell wider than an exact slab test, which only adds
    // candidates (each pair is decided by its own r^2 < 4h^2)
    int oz0 = 0, oz1 = 0;
    if (DIM > 2) {
        const T tz = approx_sqrt(G.lim2) * G.inv_w[2];
        oz1 = min(G.R[2], max(0, floor_int(fz + tz)));
        oz0 = -min(G.R[2], max(0, floor_int(tz - fz + T(1))));
    }
#pragma unroll 1
    for (int oz = first_plane(oz0, G.R[2], sub, step); oz <= oz1; oz += step) {
        T dz2 = T(0);
        int seam_z = 0;
        if (DIM > 2) {
            const T s = slab_dist(oz, fz) * G.w[2];
            dz2 = s * s;
            if (!SEAMLESS) seam_z = halo_seam(G, 2, c0[2], hz + oz);
        }
        int oy0 = 0, oy1 = 0;
        if (DIM > 1) {
            const T ty = approx_sqrt(fmax(G.lim2 - dz2, T(0))) * G.inv_w[1];
            oy1 = min(G.R[1], max(0, floor_int(fy + ty)));
            oy0 = -min(G.R[1], max(0, floor_int(ty - fy + T(1))));
        }
#pragma unroll 1
        for (int oy = oy0; oy <= oy1; ++oy) {
            T dy2 = T(0);
            int seam_y = 0;
            if (DIM > 1) {
                const T s = slab_dist(oy, fy) * G.w[1];
                dy2 = s * s;
                if (!SEAMLESS) seam_y = halo_seam(G, 1, c0[1], hy + oy);
            }
            // x window: the cells whose slab lies within t = sqrt(rem)/w of the
            // particle, (o - fx) <= t for o > 0 and (fx + |o| - 1) <= t for o < 0
            const T t = approx_sqrt(fmax(G.lim2 - dz2 - dy2, T(0))) * G.inv_w[0];
            const int ohi = min(G.R[0], max(0, floor_int(fx + t)));
            const int olo = -min(G.R[0], max(0, floor_int(t - fx + T(1))));
            const int hrow = C.H[0] * ((hy + oy) + C.H[1] * (hz + oz));
            const int u0 = hx + olo, u1 = hx + ohi + 1;  // halo x cells [u0, u1)
            if (SEAMLESS) {
                walk_smem_range<T, DIM, MODE, false, REC>(A, G, Ph, pa, spos, svel, srho, sid, lstart[hrow + u0],
                                                          lstart[hrow + u1], rec);
                continue;
            }
            // [u0, a0) across the low seam, [a0, a1) inside, [a1, u1) across the
            // high seam, in that order (the order of the staged cells, as in the
            // tiles staged with their seam shifts); a row across a y or z seam
            // takes the two-sum displacement over its whole range
            const int a0 = min(max(u0, sx0), u1);
            const int a1 = max(min(u1, sx1), a0);
            if (seam_y | seam_z) {
                walk_smem_range<T, DIM, MODE, true, REC>(A, G, Ph, pa, spos, svel, srho, sid, lstart[hrow + u0],
                                                         lstart[hrow + u1], rec);
                continue;
            }
            if (a0 > u0)
                walk_smem_range<T, DIM, MODE, true, REC>(A, G, Ph, pa, spos, svel, srho, sid, lstart[hrow + u0],
                                                         lstart[hrow + a0], rec);
            if (a1 > a0)
                walk_smem_range<T, DIM, MODE, false, REC>(A, G, Ph, pa, spos, svel, srho, sid, lstart[hrow + a0],
                                                          lstart[hrow + a1], rec);
            if (u1 > a1)
                walk_smem_range<T, DIM, MODE, true, REC>(A, G, Ph, pa, spos, svel, srho, sid, lstart[hrow + a1],
                                                         lstart[hrow + u1], rec);
        }
    }
}

// One particle's sums by the global-memory walk, for tiles whose halo does
// not fit shared memory. Kept out of line so that the rare path does not
// weigh on the register allocation of the tiled walks.
template <class T, int DIM, int MODE>
__device__ __noinline__ void particle_global(const Geo<T> G, const Phys<T> Ph, uint32_t a,
                                             const V4<T> *__restrict__ pos, const V4<T> *__restrict__ vel,
                                             const T *__restrict__ rho, const uint32_t *__restrict__ id,
                                             const uint32_t *__restrict__ start, T mass, T *__restrict__ out_rho,
                                             T *pr_out, V4<T> *__restrict__ out_acc, int32_t *__restrict__ cnt,
                                             uint64_t *__restrict__ fpr)
{
    PairAcc<T, MODE> A;
    const V4<T> pa = pos[a];
    acc_init(A, Ph, pa, vel, rho, a);
    walk_global<T, DIM, MODE>(A, G, Ph, pa, pos, vel, rho, id, start, true);
    acc_store(A, Ph, a, mass, vel, out_rho, pr_out, out_acc, cnt, fpr);
}

// One particle's sums by the tile walk without recording, for the listing
// passes (density MODE 0, isothermal force MODE 2) when the list does not
// cover the particle; out of line for the same reason as particle_global.
// (The density pass calls it; the force pass keeps its walk inline, where
// the call's register saves cost more than they free.)
template <class T, int DIM, int MODE, bool SEAMLESS>
__device__ __noinline__ void particle_tile(const Geo<T> G, const Phys<T> Ph, const TileCfg C, int c0x, int c0y,
                                           int c0z, const V4<T> pa, const V4<T> pc, uint32_t a, const uint16_t *lstart,
                                           const V4<T> *spos, const V4<T> *__restrict__ vel, T mass,
                                           T *__restrict__ out_rho, T *pr_out, V4<T> *__restrict__ out_acc)
{
    static_assert(MODE == 0 || MODE == 2, "listing passes only");
    PairAcc<T, MODE> A;
    acc_init(A, Ph, pa, vel, static_cast<const T *>(nullptr), a);
    const int c0[3] = {c0x, c0y, c0z};
    walk_tile<T, DIM, MODE, false, SEAMLESS>(A, G, Ph, C, c0, pa, pc, lstart, spos, nullptr, nullptr, nullptr, nullptr);
    acc_store(A, Ph, a, mass, vel, out_rho, pr_out, out_acc, nullptr, nullptr);
}

// The recording walk of a binary64 particle in 3D (seamless tiles whose staged
// particles all lie within the prefilter's range): rows and candidates are
// taken in binary32 from a copy of the staged positions relative to the tile
// (sf; pf the particle's own), so that the binary64 pipe, at 2 lanes per SM
// and clock the bound of these sums, only sees the listed pairs. The margins
// over 4h^2 and the pruning radius cover the rounding of the relative
// coordinates, of the cell fractions f and of the arithmetic; a pair between
// 4h^2 and thr lies where the kernel is zero (its (2 - q) is clamped) and adds
// nothing.
__device__ __forceinline__ void record_walk_f32(const int R[3], const Prefilter &P, const TileCfg &C, const int h[3],
                                                const float f[3], const float4 pf, const uint16_t *lstart,
                                                const float4 *sf, NbRec &rec, int sub, int step)
{
    prefilter_rows(P, R, C.H, h, f, sub, step, [&](int u0, int u1) {
        const int j1 = lstart[u1];
#pragma unroll 1
        for (int j = lstart[u0]; j < j1; ++j) {
            const float4 q = sf[j];
            if (prefilter_near(P, pf.x - q.x, pf.y - q.y, pf.z - q.z)) rec.push(j, false);
        }
    });
}

// Pair sums over a particle's recorded list (groups `e[g * st]` of four
// 16-bit entries, n entries), in the recorded order (SEAMLESS: the tile
// recorded no seam flags; RO: the list was written by an earlier kernel).
template <class T, int DIM, int MODE, bool SEAMLESS, bool RO = true>
__device__ __forceinline__ void read_list(PairAcc<T, MODE> &A, const Geo<T> &G, const Phys<T> &Ph, const V4<T> &pa,
                                          const V4<T> *spos, const unsigned long long *e, size_t st, int n)
{
    auto load = [](const unsigned long long *q) { return RO ? __ldg(q) : *q; };
    auto pair = [&](uint32_t cur) {
        const V4<T> pb = spos[cur & 0x7FFFu];
        T d[3];
        const T r2 = (!SEAMLESS && (cur & kNbSeam)) ? pair_r2<T, DIM, true>(G, pa, pb, d)
                                                    : pair_r2<T, DIM, false>(G, pa, pb, d);
        A.template add<DIM, true>(G, Ph, pb, nullptr, T(1), 0u, r2, d);
    };
    auto quad = [&](unsigned long long w) {
        const uint32_t l = (uint32_t)w, h = (uint32_t)(w >> 32);
        pair(l & 0xFFFFu);
        pair(l >> 16);
        pair(h & 0xFFFFu);
        pair(h >> 16);
    };
    // full groups two at a time through the read-only path, the next two
    // loaded while the current ones are used; then the partial group
    const int ng = n >> 2;
    int g = 0;
    unsigned long long c0, c1, n0 = 0, n1 = 0;
    if (ng >= 2) {
        n0 = load(&e[0]);
        n1 = load(&e[st]);
    }
    for (; g + 2 <= ng; g += 2) {
        c0 = n0;
        c1 = n1;
        if (g + 4 <= ng) {
            n0 = load(&e[(size_t)(g + 2) * st]);
            n1 = load(&e[(size_t)(g + 3) * st]);
        }
        quad(c0);
        quad(c1);
    }
    if (g < ng) quad(load(&e[(size_t)g++ * st]));
    const int m = n & 3;
    if (m) {
        const unsigned long long w = load(&e[(size_t)g * st]);
        for (int u = 0; u < m; ++u) pair((uint32_t)(w >> (16 * u)) & 0xFFFFu);
    }
}

// SPLIT: C.lanes threads share an owned particle (each takes every lanes-th
// plane of cells (first_plane) and keeps its own part of the list), for problems whose tiles
// of a thread per particle would not fill the chip.
template <class T, int DIM, int MODE, bool SPLIT = false>
__global__ void __launch_bounds__(kTileThreads, sizeof(T) == 4 ? ((MODE == 0 || MODE == 2) ? 4 : 3)
                                                         : (kPrefilter<T, DIM> && (MODE == 0 || MODE == 2) ? 2 : 1))
k_pair_tile(Geo<T> G, Phys<T> Ph, TileCfg C, const V4<T> *__restrict__ pos, const V4<T> *__restrict__ vel,
            const T *__restrict__ rho, const uint32_t *__restrict__ id, const uint32_t *__restrict__ start, T mass,
            T *__restrict__ out_rho, T *pr_out, V4<T> *__restrict__ out_acc, int32_t *__restrict__ cnt,
            uint64_t *__restrict__ fpr, NbList nbl)
{
    extern __shared__ __align__(64) unsigned char smem[];
    __shared__ int wsum[kTileThreads / 32];
    // staged offset of every halo cell (16 bits: a staged tile holds at most
    // cap <= 0x7FFF particles), then 32-bit tables
    uint16_t *lstart = reinterpret_cast<uint16_t *>(smem);                     // nhalo + 1
    int *rowpref = reinterpret_cast<int *>(smem + lstart_bytes(C.nhalo));      // nrows + 1
    int *rowg = rowpref + C.nrows + 1;                 // nrows
    const int nhr = C.H[1] * C.H[2];                   // halo rows (along x)
    int *hr_first = rowg + C.nrows;                    // nhr: global start of a halo row
    int *hr_base = hr_first + nhr;                     // nhr + 1: its staged offset
    V4<T> *spos = reinterpret_cast<V4<T> *>(smem + C.offset);
    V4<T> *svel = spos + C.cap;                        // modes staging a second V4
    T *srho = reinterpret_cast<T *>(svel + (ModeUses<MODE>::vel ? C.cap : 0));  // modes staging a scalar
    uint32_t *sid = reinterpret_cast<uint32_t *>(spos + C.cap);  // MODE 1
    float4 *sf = reinterpret_cast<float4 *>(spos + C.cap);       // binary32 copy (kPrefilter, MODE 0)
    constexpr bool kPre = kPrefilter<T, DIM> && MODE == 0;

    const int tid = threadIdx.x;
    int b = blockIdx.x;
    const int tx = b % C.nt[0];
    b /= C.nt[0];
    const int ty = b % C.nt[1];
    const int tz = b / C.nt[1];
    const int c0[3] = {tx * C.T[0], ty * C.T[1], tz * C.T[2]};
    int ext[3];
#pragma unroll
    for (int k = 0; k < 3; ++k) ext[k] = min(C.T[k], G.n[k] - c0[k]);

    // Periodic seams. A tile whose halo crosses the low seam of axis k stages
    // its wrapped cells at x - L; one whose halo crosses the high seam stages
    // its own cells at x - L and its wrapped ones at x. With lo = 0 every such
    // subtraction is exact (Sterbenz: the coordinates lie within a factor of
    // two of L, for a high seam because the halo lies in the upper half of
    // the box), so each pair's displacement is the plain difference of staged
    // coordinates, the correctly rounded periodic displacement, and the walks
    // take the plain path. Tiles that do not meet this (lo != 0, a halo over
    // both seams) keep the per-pair seam path.
    bool seamless = true, shifted = false;
    int lowk[3] = {0, 0, 0}, highk[3] = {0, 0, 0};
    T orig[3] = {T(0), T(0), T(0)};  // what the owned particles' staged coordinates lack
    {
        bool crosses = false, ok = true;
#pragma unroll
        for (int k = 0; k < DIM; ++k) {
            if (!G.per[k]) continue;
            lowk[k] = c0[k] < G.R[k];
            highk[k] = c0[k] + ext[k] + G.R[k] > G.n[k];
            if (lowk[k] || highk[k]) {
                crosses = true;
                if (!(G.lo[k] == T(0)) || (lowk[k] && highk[k]) || (highk[k] && 2 * (c0[k] - G.R[k]) < G.n[k]))
                    ok = false;
            }
        }
        if (crosses) {
            if (ok) {
                shifted = true;
#pragma unroll
                for (int k = 0; k < DIM; ++k) orig[k] = highk[k] ? G.L[k] : T(0);
            } else {
                seamless = false;
            }
        }
    }

    // origin of the binary32 copy: the tile's corner, in staged coordinates
    T org[3] = {T(0), T(0), T(0)};
    if constexpr (kPre) {
#pragma unroll
        for (int k = 0; k < DIM; ++k) org[k] = G.lo[k] + T(c0[k]) * G.w[k] - orig[k];
    }
    // whether the tile has staged a particle beyond the prefilter's range (this thread's, then the CTA's)
    bool beyond = false;
    Prefilter pre{};
    if constexpr (kPre) pre = prefilter_of(G, C);
    auto copy32 = [&](int j, const V4<T> &q) {
        if constexpr (kPre) {
            const float4 s = make_float4((float)((q.x - org[0]) * G.inv_h), (float)((q.y - org[1]) * G.inv_h),
                                         (float)((q.z - org[2]) * G.inv_h), 0.0f);
            beyond = beyond || !prefilter_holds(pre, s.x, s.y, s.z);
            sf[j] = s;
        }
    };
    auto staged = [&] {
        if constexpr (kPre) beyond = __syncthreads_or(beyond);
        else __syncthreads();
    };

    // owned rows: global start and particle count
    for (int r = tid; r < C.nrows; r += blockDim.x) {
        const int oy = r % C.T[1], oz = r / C.T[1];
        int c = 0, g = 0;
        if (oy < ext[1] && oz < ext[2]) {
            const uint32_t rowkey =
                (uint32_t)G.n[0] * ((uint32_t)(c0[1] + oy) + (uint32_t)G.n[1] * (uint32_t)(c0[2] + oz));
            g = (int)start[rowkey + c0[0]];
            c = (int)start[rowkey + c0[0] + ext[0]] - g;
        }
        rowg[r] = g;
        rowpref[r] = c;
    }
    // a tile whose halo lies inside the grid on every axis (no wrap, no
    // cell outside): each halo row of cells is one contiguous range of the
    // sorted particles, so the rows are counted and copied whole (not for
    // the full force, whose walk then spills a register; and only where the
    // particle area can hold the halo cells' 32-bit starts meanwhile)
    bool interior = MODE != 3 && C.nhalo * 4 <= C.cap * (int)sizeof(V4<T>);
#pragma unroll
    for (int k = 0; k < 3; ++k)
        if (c0[k] < G.R[k] || c0[k] + ext[k] + G.R[k] > G.n[k]) interior = false;
    int total;
    if (interior) {
        // the particle area serves as scratch for the global starts until the copy
        int *raw = reinterpret_cast<int *>(smem + C.offset);
        const int gx0 = c0[0] - G.R[0], gy0 = c0[1] - G.R[1], gz0 = c0[2] - G.R[2];
        // global start of every halo cell and the end of each row
        for (int h = tid; h < C.nhalo; h += blockDim.x) {
            int hx, hy, hz;
            halo_coords(h, C, hx, hy, hz);
            const uint32_t key = (uint32_t)(gx0 + hx) +
                                 (uint32_t)G.n[0] * ((uint32_t)(gy0 + hy) + (uint32_t)G.n[1] * (uint32_t)(gz0 + hz));
            raw[h] = (int)start[key];
            if (hx == C.H[0] - 1) hr_base[hy + C.H[1] * hz] = (int)start[key + 1];
        }
        __syncthreads();
        for (int r = tid; r < nhr; r += blockDim.x) {
            const int f = raw[r * C.H[0]];
            hr_first[r] = f;
            hr_base[r] -= f;  // particles in the row
        }
        __syncthreads();
        total = block_scan_smem(hr_base, nhr, wsum);
        block_scan_smem(rowpref, C.nrows, wsum);
        // staged offset of every halo cell: its row's offset plus its place in the row
        for (int h = tid; h < C.nhalo; h += blockDim.x) {
            const int r = small_div(h, C.H[0], C.invH[0]);
            lstart[h] = (uint16_t)(hr_base[r] + raw[h] - hr_first[r]);
        }
        if (tid == 0) lstart[C.nhalo] = (uint16_t)total;
        __syncthreads();  // the copy overwrites the scratch
        if (total <= C.cap) {
            // half a warp per row, consecutive lanes on consecutive particles
            const int lane = tid & 15;
            for (int r = tid >> 4; r < nhr; r += (int)blockDim.x >> 4) {
                const int j0 = hr_base[r], m = hr_base[r + 1] - j0;
                const uint32_t g0 = (uint32_t)hr_first[r];
                for (int u = lane; u < m; u += 16) {
                    const uint32_t gi = g0 + (uint32_t)u;
                    const V4<T> q = pos[gi];
                    spos[j0 + u] = q;
                    copy32(j0 + u, q);
                    if (ModeUses<MODE>::vel) svel[j0 + u] = vel[gi];
                    if (ModeUses<MODE>::rho) srho[j0 + u] = rho[gi];
                    if (MODE == 1) sid[j0 + u] = id[gi];
                }
            }
        }
        staged();
    } else {
        // halo cell counts; a ragged tile needs only ext + 2R halo cells per axis,
        // which keeps every raw coordinate within (-n, 2n) so one wrap suffices
        for (int h = tid; h < C.nhalo; h += blockDim.x) {
            int hx, hy, hz;
            halo_coords(h, C, hx, hy, hz);
            const bool inside = hx < ext[0] + 2 * G.R[0] && hy < ext[1] + 2 * G.R[1] && hz < ext[2] + 2 * G.R[2];
            const int gx = inside ? halo_cell(G, 0, c0[0], hx) : -1;
            const int gy = DIM > 1 ? halo_cell(G, 1, c0[1], hy) : 0;
            const int gz = DIM > 2 ? halo_cell(G, 2, c0[2], hz) : 0;
            uint32_t c = 0;
            if (gx >= 0 && gy >= 0 && gz >= 0) {
                const uint32_t key = (uint32_t)gx + (uint32_t)G.n[0] * ((uint32_t)gy + (uint32_t)G.n[1] * (uint32_t)gz);
                c = start[key + 1] - start[key];
            }
            // a count that does not fit 16 bits makes the tile exceed cap anyway
            lstart[h] = (uint16_t)min(c, 0xFFFFu);
        }
        __syncthreads();
        total = block_scan_smem(lstart, C.nhalo, wsum);
        block_scan_smem(rowpref, C.nrows, wsum);
        if (total <= C.cap) {
            for (int h = tid; h < C.nhalo; h += blockDim.x) {
                const int j0 = lstart[h], j1 = lstart[h + 1];
                if (j1 == j0) continue;
                int hx, hy, hz;
                halo_coords(h, C, hx, hy, hz);
                const int gx = halo_cell(G, 0, c0[0], hx);
                const int gy = DIM > 1 ? halo_cell(G, 1, c0[1], hy) : 0;
                const int gz = DIM > 2 ? halo_cell(G, 2, c0[2], hz) : 0;
                const uint32_t key = (uint32_t)gx + (uint32_t)G.n[0] * ((uint32_t)gy + (uint32_t)G.n[1] * (uint32_t)gz);
                const uint32_t g0 = start[key];
                // the seam shift of this halo cell (see above)
                T sh[3] = {T(0), T(0), T(0)};
                if (shifted) {
                    const int hk[3] = {hx, hy, hz};
#pragma unroll
                    for (int k = 0; k < DIM; ++k) {
                        const int raw = c0[k] - G.R[k] + hk[k];
                        if ((highk[k] && raw < G.n[k]) || (lowk[k] && raw < 0)) sh[k] = G.L[k];
                    }
                }
                for (int j = j0; j < j1; ++j) {
                    const uint32_t gi = g0 + (uint32_t)(j - j0);
                    V4<T> q = pos[gi];
                    q.x = sub_rn(q.x, sh[0]);
                    if (DIM > 1) q.y = sub_rn(q.y, sh[1]);
                    if (DIM > 2) q.z = sub_rn(q.z, sh[2]);
                    spos[j] = q;
                    copy32(j, q);
                    if (ModeUses<MODE>::vel) svel[j] = vel[gi];
                    if (ModeUses<MODE>::rho) srho[j] = rho[gi];
                    if (MODE == 1) sid[j] = id[gi];
                }
            }
            staged();
        }
    }
    const int owned = rowpref[C.nrows];
    const bool tiled = total <= C.cap;


    const int lanes = SPLIT ? C.lanes : 1;
    for (int slot = tid; slot < owned * lanes; slot += blockDim.x) {
        const int p = SPLIT ? slot / lanes : slot, sub = SPLIT ? slot & (lanes - 1) : 0;
        // owned row of p: the last r with rowpref[r] <= p
        int lo = 0, hi = C.nrows - 1;
        while (lo < hi) {
            const int mid = (lo + hi + 1) >> 1;
            if (rowpref[mid] <= p) lo = mid; else hi = mid - 1;
        }
        const int k = p - rowpref[lo];
        const uint32_t a = (uint32_t)(rowg[lo] + k);
        if (!tiled) {
            if (SPLIT && sub != 0) continue;
            particle_global<T, DIM, MODE>(G, Ph, a, pos, vel, rho, id, start, mass, out_rho, pr_out, out_acc, cnt,
                                          fpr);
            continue;
        }
        PairAcc<T, MODE> A;
        {
            // the owned row starts at halo x = R of halo row (oy + R, oz + R)
            const int oy = lo % C.T[1], oz = lo / C.T[1];
            const int hrow = C.H[0] * ((oy + (DIM > 1 ? G.R[1] : 0)) + C.H[1] * (oz + (DIM > 2 ? G.R[2] : 0)));
            const V4<T> pa = spos[lstart[hrow + G.R[0]] + k];
            V4<T> pc = pa;  // box coordinates (adding back the shift is exact)
            if (shifted) {
                pc.x = add_rn(pa.x, orig[0]);
                if (DIM > 1) pc.y = add_rn(pa.y, orig[1]);
                if (DIM > 2) pc.z = add_rn(pa.z, orig[2]);
            }
            acc_init(A, Ph, pa, vel, rho, a);
            const bool listed = nbl.idx && slot < nbl.owned_cap;
            const size_t oc = (size_t)nbl.owned_cap;
            const size_t lbase = (size_t)blockIdx.x * (size_t)(nbl.cap / 4 + 1) * oc + (size_t)slot;
            if (kPre && listed && seamless && !beyond) {
                if constexpr (kPre) {
                    NbRec rec{nbl.idx + lbase, (uint32_t)oc, nbl.cap / 4, 0};
                    const int ja = lstart[hrow + G.R[0]] + k;
                    T t[3];
                    const int h[3] = {axis_cell(pc.x, G.lo[0], G.inv_w[0], G.n[0], t[0]) - c0[0] + G.R[0],
                                      axis_cell(pc.y, G.lo[1], G.inv_w[1], G.n[1], t[1]) - c0[1] + G.R[1],
                                      axis_cell(pc.z, G.lo[2], G.inv_w[2], G.n[2], t[2]) - c0[2] + G.R[2]};
                    float f[3];
#pragma unroll
                    for (int d = 0; d < 3; ++d) f[d] = (float)(t[d] - T(h[d] + c0[d] - G.R[d]));
                    record_walk_f32(G.R, pre, C, h, f, sf[ja], lstart, sf, rec, sub, lanes);
                    const int n = rec.n;
                    nbl.cnt[(size_t)blockIdx.x * oc + slot] = n <= nbl.cap ? (uint16_t)n : kNbNone;
                    if (SPLIT && n > nbl.cap) {
                        walk_tile<T, DIM, MODE, false, true>(A, G, Ph, C, c0, pa, pc, lstart, spos, svel, srho, sid,
                                                             nullptr, sub, lanes);
                    } else if (n > nbl.cap) {
                        particle_tile<T, DIM, MODE, true>(G, Ph, C, c0[0], c0[1], c0[2], pa, pc, a, lstart, spos, vel,
                                                          mass, out_rho, pr_out, out_acc);
                        continue;
                    } else {
                        read_list<T, DIM, MODE, true, false>(A, G, Ph, pa, spos, nbl.idx + lbase, oc, n);
                    }
                }
            } else if (MODE == 0 && listed) {
                // density pass: record the neighbours in walk order
                NbRec rec{nbl.idx + lbase, (uint32_t)oc, nbl.cap / 4, 0};
                if (seamless)
                    walk_tile<T, DIM, MODE, true, true>(A, G, Ph, C, c0, pa, pc, lstart, spos, svel, srho, sid, &rec,
                                                        sub, lanes);
                else
                    walk_tile<T, DIM, MODE, true, false>(A, G, Ph, C, c0, pa, pc, lstart, spos, svel, srho, sid, &rec,
                                                         sub, lanes);
                nbl.cnt[(size_t)blockIdx.x * oc + slot] = rec.n <= nbl.cap ? (uint16_t)rec.n : kNbNone;
            } else if (MODE == 2 && listed && nbl.cnt[(size_t)blockIdx.x * oc + slot] != kNbNone) {
                // force pass: the density pass's list of this binning, same order
                const int n = nbl.cnt[(size_t)blockIdx.x * oc + slot];
                const unsigned long long *e = nbl.idx + lbase;
                const size_t st = oc;
                if (seamless)
                    read_list<T, DIM, MODE, true>(A, G, Ph, pa, spos, e, st, n);
                else
                    read_list<T, DIM, MODE, false>(A, G, Ph, pa, spos, e, st, n);
            } else if (MODE == 0 && !SPLIT) {
                // a particle the density pass does not list (rare): out of line
                if constexpr (MODE == 0 && !SPLIT) {
                    if (seamless)
                        particle_tile<T, DIM, MODE, true>(G, Ph, C, c0[0], c0[1], c0[2], pa, pc, a, lstart, spos, vel,
                                                          mass, out_rho, pr_out, out_acc);
                    else
                        particle_tile<T, DIM, MODE, false>(G, Ph, C, c0[0], c0[1], c0[2], pa, pc, a, lstart, spos, vel,
                                                           mass, out_rho, pr_out, out_acc);
                }
                continue;
            } else if (seamless) {
                walk_tile<T, DIM, MODE, false, true>(A, G, Ph, C, c0, pa, pc, lstart, spos, svel, srho, sid, nullptr,
                                                     sub, lanes);
            } else {
                walk_tile<T, DIM, MODE, false, false>(A, G, Ph, C, c0, pa, pc, lstart, spos, svel, srho, sid, nullptr,
                                                      sub, lanes);
            }
        }
        if constexpr (SPLIT) {
            // the lanes of a particle lie in one warp and got here together
            const unsigned mask = ((1u << lanes) - 1u) << ((tid & 31) & ~(lanes - 1));
            for (int o = lanes >> 1; o > 0; o >>= 1) {
                if (MODE == 0) {
                    A.sum += __shfl_xor_sync(mask, A.sum, o);
                } else {
                    A.ax += __shfl_xor_sync(mask, A.ax, o);
                    A.ay += __shfl_xor_sync(mask, A.ay, o);
                    A.az += __shfl_xor_sync(mask, A.az, o);
                }
            }
            if (sub != 0) continue;
        }
        acc_store(A, Ph, a, mass, vel, out_rho, pr_out, out_acc, cnt, fpr);
    }
}

// ---------------------------------------------------------------------------
// Host side
// ---------------------------------------------------------------------------
template <class T, int DIM, int MODE> constexpr int tile_bytes_per_particle()
{
    return (int)sizeof(V4<T>) + (kPrefilter<T, DIM> && (MODE == 0 || MODE == 2) ? (int)sizeof(float4) : 0) + (ModeUses<MODE>::vel ? (int)sizeof(V4<T>) : 0) +
           (ModeUses<MODE>::rho ? (int)sizeof(T) : 0) + (MODE == 1 ? 4 : 0);
}

// Shared memory of the listing passes' tiles (the list belongs to their shape).
template <class T, int DIM> constexpr int tile_budget() { return kPrefilter<T, DIM> ? kTileSmemWide : kTileSmemPos; }

// Tiles of the listing passes (density and isothermal force). In 3D a problem
// of few tiles takes smaller ones, with up to eight lanes per particle, until
// there are two CTAs per SM (binary64: one, which fills its pipe). A 24^3 box:
// density 56 -> 17 us, force 24 -> 15 us; 16^3: step 254 -> 98 us; 44^3, two
// lanes: 181 -> 174 us; at 52^3, with 2.5 CTAs per SM, two lanes would lose
// (211 -> 219 us).
template <class T>
bool plan_listing(const Geo<T> &G, int dim, double mean, TileCfg &C, size_t &smem)
{
    const int bpp = dim == 3 ? tile_bytes_per_particle<T, 3, 0>() : tile_bytes_per_particle<T, 1, 0>();
    const int budget = dim == 3 ? tile_budget<T, 3>() : tile_budget<T, 1>();
    if (!plan_tiles(G, dim, mean, bpp, budget, kTileThreads, C, smem)) return false;
    const int64_t want = (int64_t)kSmCount * (sizeof(T) == 4 ? 2 : 1);
    for (int lanes = 2; dim == 3 && lanes <= 8 && (int64_t)C.nt[0] * C.nt[1] * C.nt[2] < want; lanes *= 2) {
        TileCfg S{};
        size_t sm = 0;
        if (!plan_tiles(G, dim, mean, bpp, budget, kTileThreads, S, sm, lanes)) break;
        C = S;
        smem = sm;
    }
    return true;
}

// Tiles of any pair pass (false: none, each particle walks global memory).
template <class T, int DIM, int MODE> bool plan_pass(const Geo<T> &G, double mean, TileCfg &C, size_t &smem)
{
    if constexpr (MODE == 0 || MODE == 2) return plan_listing(G, DIM, mean, C, smem);
    constexpr int budget = (ModeUses<MODE>::vel || ModeUses<MODE>::rho) ? 72 * 1024 : tile_budget<T, DIM>();
    return plan_tiles(G, DIM, mean, tile_bytes_per_particle<T, DIM, MODE>(), budget, kTileThreads, C, smem);
}

template <class T, int DIM, int MODE>
cudaError_t pair_launch(const LaunchCtx &L, const Geo<T> &G, const Phys<T> &Ph, int n, T mass, const V4<T> *pos,
                        const V4<T> *vel, const T *rho, const uint32_t *id, const uint32_t *start, T *out_rho,
                        T *pr_out, V4<T> *out_acc, int32_t *cnt, uint64_t *fpr, double mean,
                        NbList nb = NbList{})
{
    constexpr int budget = (ModeUses<MODE>::vel || ModeUses<MODE>::rho) ? 72 * 1024 : tile_budget<T, DIM>();
    constexpr bool kListing = MODE == 0 || MODE == 2;
    TileCfg C{};
    size_t smem = 0;
    if (plan_pass<T, DIM, MODE>(G, mean, C, smem)) {
        static bool attr_set = false;
        if (!attr_set) {
            cudaError_t e = cudaFuncSetAttribute(k_pair_tile<T, DIM, MODE>,
                                                 cudaFuncAttributeMaxDynamicSharedMemorySize, budget);
            if constexpr (kListing && DIM == 3)
                if (e == cudaSuccess)
                    e = cudaFuncSetAttribute(k_pair_tile<T, DIM, MODE, true>,
                                             cudaFuncAttributeMaxDynamicSharedMemorySize, budget);
            if (e != cudaSuccess) return e;
            attr_set = true;
        }
        const int blocks = C.nt[0] * C.nt[1] * C.nt[2];
        // tile-local indices must fit the list's 15 index bits
        if (C.cap > 0x7FFF) nb = NbList{};
        auto kern = k_pair_tile<T, DIM, MODE>;
        if constexpr (kListing && DIM == 3)
            if (C.lanes > 1) kern = k_pair_tile<T, DIM, MODE, true>;
        kern<<<blocks, kTileThreads, smem, L.stream>>>(G, Ph, C, pos, vel, rho, id, start, mass, out_rho, pr_out,
                                                       out_acc, cnt, fpr, nb);
    } else {
        const int threads = 128;
        k_pair_global<T, DIM, MODE><<<(n + threads - 1) / threads, threads, 0, L.stream>>>(
            G, Ph, pos, vel, rho, id, start, n, mass, out_rho, pr_out, out_acc, cnt, fpr);
    }
    return cudaGetLastError();
}

template <class T, int DIM>
cudaError_t density_t(const LaunchCtx &L, const void *geo, const void *phys, PhaseBufs &P, void *rho, bool gas,
                      int32_t *cnt, uint64_t *fprint, const NbList *nbl)
{
    if (P.n == 0) return cudaSuccess;
    const Geo<T> &G = *static_cast<const Geo<T> *>(geo);
    const Phys<T> &Ph = *static_cast<const Phys<T> *>(phys);
    auto *pos = static_cast<V4<T> *>(P.pos[P.cur]);
    auto *vel = static_cast<const V4<T> *>(P.vel[P.cur]);
    T *pr = gas ? reinterpret_cast<T *>(pos) : nullptr;
    const T mass = gas ? Ph.m_g : Ph.m_d;
    const double mean = (double)P.n / (double)G.ncells;
    // the neighbour statistics are an export: p/rho^2 of the state stays the
    // density pass's (whose sums may be split over lanes and round otherwise)
    if (cnt)
        return pair_launch<T, DIM, 1>(L, G, Ph, (int)P.n, mass, pos, vel, nullptr, P.id[P.cur], P.start,
                                      static_cast<T *>(rho), nullptr, nullptr, cnt, fprint, mean);
    return pair_launch<T, DIM, 0>(L, G, Ph, (int)P.n, mass, pos, vel, nullptr, P.id[P.cur], P.start,
                                  static_cast<T *>(rho), pr, nullptr, nullptr, nullptr, mean,
                                  (gas && nbl) ? *nbl : NbList{});
}

template <class T, int DIM>
cudaError_t force_t(const LaunchCtx &L, const void *geo, const void *phys, PhaseBufs &P, const void *rho, void *acc,
                    const NbList *nbl)
{
    if (P.n == 0) return cudaSuccess;
    const Geo<T> &G = *static_cast<const Geo<T> *>(geo);
    const Phys<T> &Ph = *static_cast<const Phys<T> *>(phys);
    auto *pos = static_cast<const V4<T> *>(P.pos[P.cur]);
    auto *vel = static_cast<const V4<T> *>(P.vel[P.cur]);
    const double mean = (double)P.n / (double)G.ncells;
    const bool full = Ph.av || Ph.eos == TFSPH_EOS_ADIABATIC;
    if (full)
        return pair_launch<T, DIM, 3>(L, G, Ph, (int)P.n, T(0), pos, vel, static_cast<const T *>(rho), P.id[P.cur],
                                      P.start, nullptr, nullptr, static_cast<V4<T> *>(acc), nullptr, nullptr, mean);
    return pair_launch<T, DIM, 2>(L, G, Ph, (int)P.n, T(0), pos, vel, static_cast<const T *>(rho), P.id[P.cur],
                                  P.start, nullptr, nullptr, static_cast<V4<T> *>(acc), nullptr, nullptr, mean,
                                  nbl ? *nbl : NbList{});
}

// lambda_A (V4, storage order) -> lambda_x (V4 .xyz) and lambda_q (.w).
template <class T, int DIM>
cudaError_t force_adjoint_t(const LaunchCtx &L, const void *geo, const void *phys, PhaseBufs &P, const void *lamA,
                            void *out)
{
    if (P.n == 0) return cudaSuccess;
    const Geo<T> &G = *static_cast<const Geo<T> *>(geo);
    const Phys<T> &Ph = *static_cast<const Phys<T> *>(phys);
    auto *pos = static_cast<const V4<T> *>(P.pos[P.cur]);
    const double mean = (double)P.n / (double)G.ncells;
    return pair_launch<T, DIM, 4>(L, G, Ph, (int)P.n, T(0), pos, static_cast<const V4<T> *>(lamA), nullptr,
                                  P.id[P.cur], P.start, nullptr, nullptr, static_cast<V4<T> *>(out), nullptr, nullptr,
                                  mean);
}

// lambda_rho (T, storage order) -> lambda_x (V4 .xyz) accumulated.
template <class T, int DIM>
cudaError_t density_adjoint_t(const LaunchCtx &L, const void *geo, const void *phys, PhaseBufs &P,
                              const void *lamrho, void *inout)
{
    if (P.n == 0) return cudaSuccess;
    const Geo<T> &G = *static_cast<const Geo<T> *>(geo);
    const Phys<T> &Ph = *static_cast<const Phys<T> *>(phys);
    auto *pos = static_cast<const V4<T> *>(P.pos[P.cur]);
    const double mean = (double)P.n / (double)G.ncells;
    return pair_launch<T, DIM, 5>(L, G, Ph, (int)P.n, T(0), pos, nullptr, static_cast<const T *>(lamrho),
                                  P.id[P.cur], P.start, nullptr, nullptr, static_cast<V4<T> *>(inout), nullptr,
                                  nullptr, mean);
}

}  // namespace

cudaError_t launch_force_adjoint(const LaunchCtx &L, const void *geo, const void *phys, PhaseBufs &G,
                                 const void *lamA, void *out)
{
    if (L.precision == TFSPH_FP64) {
        switch (L.dim) {
            case 1: return force_adjoint_t<double, 1>(L, geo, phys, G, lamA, out);
            case 2: return force_adjoint_t<double, 2>(L, geo, phys, G, lamA, out);
            default: return force_adjoint_t<double, 3>(L, geo, phys, G, lamA, out);
        }
    }
    switch (L.dim) {
        case 1: return force_adjoint_t<float, 1>(L, geo, phys, G, lamA, out);
        case 2: return force_adjoint_t<float, 2>(L, geo, phys, G, lamA, out);
        default: return force_adjoint_t<float, 3>(L, geo, phys, G, lamA, out);
    }
}

cudaError_t launch_density_adjoint(const LaunchCtx &L, const void *geo, const void *phys, PhaseBufs &G,
                                   const void *lamrho, void *inout)
{
    if (L.precision == TFSPH_FP64) {
        switch (L.dim) {
            case 1: return density_adjoint_t<double, 1>(L, geo, phys, G, lamrho, inout);
            case 2: return density_adjoint_t<double, 2>(L, geo, phys, G, lamrho, inout);
            default: return density_adjoint_t<double, 3>(L, geo, phys, G, lamrho, inout);
        }
    }
    switch (L.dim) {
        case 1: return density_adjoint_t<float, 1>(L, geo, phys, G, lamrho, inout);
        case 2: return density_adjoint_t<float, 2>(L, geo, phys, G, lamrho, inout);
        default: return density_adjoint_t<float, 3>(L, geo, phys, G, lamrho, inout);
    }
}

cudaError_t launch_density(const LaunchCtx &L, const void *geo, const void *phys, PhaseBufs &P, void *rho, bool gas,
                           int32_t *cnt, uint64_t *fprint, const NbList *nbl)
{
    if (L.precision == TFSPH_FP64) {
        switch (L.dim) {
            case 1: return density_t<double, 1>(L, geo, phys, P, rho, gas, cnt, fprint, nbl);
            case 2: return density_t<double, 2>(L, geo, phys, P, rho, gas, cnt, fprint, nbl);
            default: return density_t<double, 3>(L, geo, phys, P, rho, gas, cnt, fprint, nbl);
        }
    }
    switch (L.dim) {
        case 1: return density_t<float, 1>(L, geo, phys, P, rho, gas, cnt, fprint, nbl);
        case 2: return density_t<float, 2>(L, geo, phys, P, rho, gas, cnt, fprint, nbl);
        default: return density_t<float, 3>(L, geo, phys, P, rho, gas, cnt, fprint, nbl);
    }
}

cudaError_t launch_force(const LaunchCtx &L, const void *geo, const void *phys, PhaseBufs &G, const void *rho,
                         void *acc, const NbList *nbl)
{
    if (L.precision == TFSPH_FP64) {
        switch (L.dim) {
            case 1: return force_t<double, 1>(L, geo, phys, G, rho, acc, nbl);
            case 2: return force_t<double, 2>(L, geo, phys, G, rho, acc, nbl);
            default: return force_t<double, 3>(L, geo, phys, G, rho, acc, nbl);
        }
    }
    switch (L.dim) {
        case 1: return force_t<float, 1>(L, geo, phys, G, rho, acc, nbl);
        case 2: return force_t<float, 2>(L, geo, phys, G, rho, acc, nbl);
        default: return force_t<float, 3>(L, geo, phys, G, rho, acc, nbl);
    }
}

namespace {
template <class T>
bool nblist_layout_t(const Geo<T> &G, int dim, int64_t n, int *cap, int *owned_cap, int64_t *tiles)
{
    if (n <= 0) return false;
    double ball = 4.0 * (double)G.h;  // length, area or volume within 2h
    if (dim == 2) ball = M_PI * 4.0 * (double)G.h * (double)G.h;
    if (dim == 3) ball = 4.0 / 3.0 * M_PI * 8.0 * (double)G.h * (double)G.h * (double)G.h;
    double cellv = 1.0;
    for (int k = 0; k < dim; ++k) cellv *= (double)G.w[k];
    const double mean = (double)n / (double)G.ncells;
    const double want = 1.5 * mean * ball / cellv + 16.0;
    if (want > 1024.0) return false;
    // the density pass's tiles
    TileCfg C{};
    size_t smem = 0;
    if (!plan_listing(G, dim, mean, C, smem) || C.cap > 0x7FFF) return false;
    // a lane's part of a split particle's neighbours: the planes of cells it
    // takes, at most about 2/5 of them more than its even share
    const double part = C.lanes == 1 ? want : (want - 16.0) * std::min(1.0, 1.0 / C.lanes + 0.3) + 16.0;
    double owned = mean * C.lanes;
    for (int k = 0; k < dim; ++k) owned *= (double)C.T[k];
    const double cap_d = 32.0 * std::ceil(part / 32.0);
    const double oc_d = 32.0 * std::ceil((1.25 * owned + 32.0) / 32.0);
    // cap is a multiple of 32 (so of the 4 entries of a group); a particle's
    // 16-bit slots lie within cap * owned_cap + 4 of its first (32-bit offsets)
    if ((cap_d + 1.0) * oc_d >= 2147483648.0) return false;
    *cap = (int)cap_d;
    *owned_cap = (int)oc_d;
    *tiles = (int64_t)C.nt[0] * C.nt[1] * C.nt[2];
    return true;
}
}  // namespace

namespace {
template <class T, int DIM> bool gas_sums_tiled_t(const void *geo, int64_t n, int mode)
{
    const Geo<T> &G = *static_cast<const Geo<T> *>(geo);
    const double mean = (double)n / (double)G.ncells;
    TileCfg C{};
    size_t smem = 0;
    return mode == 3 ? plan_pass<T, DIM, 3>(G, mean, C, smem) : plan_pass<T, DIM, 0>(G, mean, C, smem);
}
}  // namespace

bool gas_sums_tiled(const void *geo, int precision, int dim, int64_t n, int mode)
{
    if (precision == TFSPH_FP64)
        return dim == 1 ? gas_sums_tiled_t<double, 1>(geo, n, mode)
                        : (dim == 2 ? gas_sums_tiled_t<double, 2>(geo, n, mode) : gas_sums_tiled_t<double, 3>(geo, n, mode));
    return dim == 1 ? gas_sums_tiled_t<float, 1>(geo, n, mode)
                    : (dim == 2 ? gas_sums_tiled_t<float, 2>(geo, n, mode) : gas_sums_tiled_t<float, 3>(geo, n, mode));
}

bool nblist_layout(const void *geo, int precision, int dim, int64_t n, int *cap, int *owned_cap, int64_t *tiles)
{
    if (precision == TFSPH_FP64)
        return nblist_layout_t(*static_cast<const Geo<double> *>(geo), dim, n, cap, owned_cap, tiles);
    return nblist_layout_t(*static_cast<const Geo<float> *>(geo), dim, n, cap, owned_cap, tiles);
}

}  // namespace tfsph
