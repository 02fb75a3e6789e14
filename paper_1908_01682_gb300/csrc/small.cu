// The whole IDIC step of a small context in one cooperative launch.
//
// A step is nine kernels; a problem of a few thousand particles leaves most
// of the chip idle in each of them and waits on the host between them (100 +
// 100 particles in FP64: 66 us a step, of which 60 us are the host's nine
// launches and 48 us kernels that run on one SM). Here the phases (count,
// scan, scatter, rank + gather, density, force, cell drag and update) run in
// one launch, separated by barriers (of a cluster for the smallest, else of
// the grid, with bounded waits), and every phase is spread over all CTAs: consecutive warps of particles go to
// different SMs. The phases compute what the kernels of bin.cu, sph.cu and
// drag.cu compute, with the sums in their order: the results are the same bit
// for bit. 1D and 2D only: in 3D the lanes of a warp would read their
// candidates from 32 places of global memory at a time (a 24^3 box: density
// 50 us against 55 us of its few tiles).
#include <algorithm>

#include "drag_ops.cuh"
#include "grid_barrier.cuh"
#include "pair.cuh"
#include "sort_ops.cuh"

namespace tfsph {
namespace {

constexpr int kSmallThreads = 512;  // most threads of a CTA
constexpr int kSmallCluster = 8;    // most CTAs of the cluster form

template <class T> struct SmallArgs {
    Geo<T> G;
    Phys<T> Ph;
    StepVals S;
    // phase state: storage a (unsorted) -> b (sorted)
    const V4<T> *gpa, *gva, *dpa, *dva;
    V4<T> *gpb, *gvb, *dpb, *dvb;
    const uint32_t *gia, *dia;
    uint32_t *gib, *dib;
    uint32_t *gkey, *dkey, *gcnt, *dcnt, *gstart, *dstart, *gsrc, *dsrc, *gtid, *dtid;
    T *rho;
    V4<T> *acc;
    int *err;
    GridBar *bar;
    long long spin;
    uint32_t ng, nd;
    int lanes;    // lanes per particle of the pair sums (1, or up to 8: binary64 in 1D)
    uint32_t cpc; // cells a CTA updates at a time
    int *counted; // nonzero: gcnt, dcnt hold the counts of the current keys (the last step left them)
    int cluster;  // the grid is one cluster
    int few;      // few candidates per particle: terms without a branch (binary64 in 1D)
    int harmonic, has_frozen, adiabatic;
};

// Exclusive scan of one value per thread over the CTA.
__device__ __forceinline__ uint32_t cta_scan(uint32_t v, uint32_t &excl, uint32_t *wtot)
{
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const int nw = blockDim.x >> 5;
    uint32_t x = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y;
    }
    __syncthreads();
    if (lane == 31) wtot[wid] = x;
    __syncthreads();
    uint32_t before = 0, total = 0;
    for (int w = 0; w < nw; ++w) {
        if (w < wid) before += wtot[w];
        total += wtot[w];
    }
    excl = before + x - v;
    return total;
}

// Cell ranges of both phases. A tile's first slot is the sum of all counts
// before it, which its CTA adds up itself (at most kSmallCells counts, four
// 16-byte loads in flight a thread): one phase instead of three.
template <class T> __device__ __forceinline__ void small_scan(const SmallArgs<T> &B, uint32_t *wtot)
{
    const uint32_t nc = B.G.ncells;
    const uint32_t tile = blockDim.x * kScanItems, ntile = (nc + tile - 1) / tile;
    for (uint32_t t = blockIdx.x; t < 2 * ntile; t += gridDim.x) {
        const bool dust = t >= ntile;
        const uint32_t first = (dust ? t - ntile : t) * tile;
        const uint32_t *cnt = dust ? B.dcnt : B.gcnt;
        uint32_t *st = dust ? B.dstart : B.gstart;
        uint32_t s = 0, e;
        const uint4 *c4 = reinterpret_cast<const uint4 *>(cnt);
#pragma unroll 4
        for (uint32_t i = threadIdx.x; i < first / 4; i += blockDim.x) {
            const uint4 v = c4[i];
            s += v.x + v.y + v.z + v.w;
        }
        const uint32_t before = cta_scan(s, e, wtot);
        const uint32_t base = first + threadIdx.x * kScanItems;
        uint32_t v[kScanItems];
        s = 0;
#pragma unroll
        for (int k = 0; k < kScanItems; ++k) {
            v[k] = base + k < nc ? cnt[base + k] : 0u;
            s += v[k];
        }
        cta_scan(s, e, wtot);
        uint32_t run = before + e;
#pragma unroll
        for (int k = 0; k < kScanItems; ++k) {
            if (base + k < nc) st[base + k] = min(run, dust ? B.nd : B.ng);  // (past n: a step that gave up)
            run += v[k];
        }
        if (first == 0 && threadIdx.x == 0) st[nc] = dust ? B.nd : B.ng;
    }
}

// Density (MODE 0) or pressure force (MODE 2, 3) of the gas, a thread per
// particle. Consecutive warps lie in different CTAs.
template <class T, int DIM, int MODE> __device__ __forceinline__ void small_pair(const SmallArgs<T> &B)
{
    const uint32_t nw = (B.ng + 31) / 32, nwarps = gridDim.x * (blockDim.x >> 5);
    const V4<T> *pos = B.gpb, *vel = B.gvb;
    const T *rho = B.rho;
    for (uint32_t w = (threadIdx.x >> 5) * gridDim.x + blockIdx.x; w < nw; w += nwarps) {
        const uint32_t a = w * 32 + (threadIdx.x & 31);
        if (a >= B.ng) continue;
        PairAcc<T, MODE> A;
        const V4<T> pa = pos[a];
        acc_init(A, B.Ph, pa, vel, rho, a);
        auto range = [&](uint32_t b0, uint32_t n, auto seam) {
            // four candidates loaded, and their distances formed, at a time
            constexpr int kAhead = 4;
            if constexpr (sizeof(T) == 8 && DIM == 1 && (MODE == 0 || MODE == 2)) {
                if (B.few) {
                    // four chains of binary64 operations in flight
#pragma unroll 1
                    for (uint32_t b = b0; b < b0 + n; b += kAhead) {
                        T s[kAhead], d[kAhead][3];
#pragma unroll
                        for (int u = 0; u < kAhead; ++u) {
                            const bool have = b + u < b0 + n;
                            const V4<T> pb = pos[have ? b + u : b];
                            const T r2 = pair_r2<T, DIM, decltype(seam)::value>(B.G, pa, pb, d[u]);
                            s[u] = pair_term<T, DIM, MODE>(A, B.G, B.Ph, pb, r2, d[u], have && r2 < B.G.h2x4);
                        }
#pragma unroll
                        for (int u = 0; u < kAhead; ++u) add_term<T, DIM, MODE>(A, s[u], d[u]);
                    }
                    return;
                }
            }
#pragma unroll 1
            for (uint32_t b = b0; b < b0 + n; b += kAhead) {
                V4<T> pb[kAhead];
#pragma unroll
                for (int u = 0; u < kAhead; ++u) pb[u] = pos[b + u < b0 + n ? b + u : b];
#pragma unroll
                for (int u = 0; u < kAhead; ++u) {
                    T d[3];
                    const T r2 = pair_r2<T, DIM, decltype(seam)::value>(B.G, pa, pb[u], d);
                    if (b + u < b0 + n && r2 < B.G.h2x4) {
                        V4<T> vb;
                        T rhob = T(1);
                        if (ModeUses<MODE>::vel) vb = vel[b + u];
                        if (ModeUses<MODE>::rho) rhob = rho[b + u];
                        A.template add<DIM, true>(B.G, B.Ph, pb[u], &vb, rhob, 0u, r2, d);
                    }
                }
            }
        };
        for_each_range<T, DIM>(B.G, B.gstart, pa.x, pa.y, pa.z, [&](uint32_t b0, uint32_t n, bool seam) {
            if (seam) range(b0, n, SeamTag<true>{});
            else range(b0, n, SeamTag<false>{});
        }, true);
        if (MODE == 0)
            acc_store<T, MODE>(A, B.Ph, a, B.Ph.m_g, vel, B.rho, reinterpret_cast<T *>(B.gpb), nullptr, nullptr,
                               nullptr);
        else
            acc_store<T, MODE>(A, B.Ph, a, T(0), vel, nullptr, nullptr, B.acc, nullptr, nullptr);
    }
}

// The same sums of a 1D binary64 gas by `lanes` lanes per particle, a
// candidate each, for problems that leave most of the chip's binary64 units
// idle (a warp's operation takes its unit 64 cycles, however many lanes it
// has, and a lone thread per particle runs some 200 of them in a row). The
// terms are added in the walk's order, so the result is the same bit for bit.
template <class T, int MODE> __device__ __forceinline__ void small_pair_lanes(const SmallArgs<T> &B)
{
    const int lanes = B.lanes, lane = threadIdx.x & 31, sub = lane & (lanes - 1), lead = lane & ~(lanes - 1);
    const uint32_t per = 32u / (uint32_t)lanes;
    const uint32_t nw = (B.ng + per - 1) / per, nwarps = gridDim.x * (blockDim.x >> 5);
    const V4<T> *pos = B.gpb;
    for (uint32_t w = (threadIdx.x >> 5) * gridDim.x + blockIdx.x; w < nw; w += nwarps) {
        const uint32_t a = w * per + (uint32_t)(lane / lanes);
        const bool live = a < B.ng;
        PairAcc<T, MODE> A;
        const V4<T> pa = pos[live ? a : 0];
        acc_init(A, B.Ph, pa, B.gvb, B.rho, live ? a : 0u);
        // up to three ranges in the walk's order
        uint32_t rb[3] = {0, 0, 0}, rn[3] = {0, 0, 0}, seams = 0;
        int nr = 0;
        if (live)
            for_each_range<T, 1>(B.G, B.gstart, pa.x, T(0), T(0), [&](uint32_t b0, uint32_t n, bool seam) {
#pragma unroll
                for (int k = 0; k < 3; ++k)
                    if (nr == k) {
                        rb[k] = b0;
                        rn[k] = n;
                    }
                seams |= (seam ? 1u : 0u) << nr;
                ++nr;
            }, true);
        const uint32_t m = rn[0] + rn[1] + rn[2];
        const uint32_t most = __reduce_max_sync(0xffffffffu, m);
        for (uint32_t c0 = 0; c0 < most; c0 += (uint32_t)lanes) {
            const uint32_t c = c0 + (uint32_t)sub;
            T s = T(0), d[3] = {T(0), T(0), T(0)};
            if (c < m) {
                const int k = c < rn[0] ? 0 : (c < rn[0] + rn[1] ? 1 : 2);
                const uint32_t b = k == 0 ? rb[0] + c : (k == 1 ? rb[1] + (c - rn[0]) : rb[2] + (c - rn[0] - rn[1]));
                const V4<T> pb = pos[b];
                const T r2 = (seams >> k) & 1u ? pair_r2<T, 1, true>(B.G, pa, pb, d)
                                               : pair_r2<T, 1, false>(B.G, pa, pb, d);
                s = pair_term<T, 1, MODE>(A, B.G, B.Ph, pb, r2, d, r2 < B.G.h2x4);
            }
            for (int u = 0; u < lanes; ++u) {
                const T su = __shfl_sync(0xffffffffu, s, lead + u);
                const T du[3] = {MODE == 0 ? T(0) : __shfl_sync(0xffffffffu, d[0], lead + u), T(0), T(0)};
                add_term<T, 1, MODE>(A, su, du);
            }
        }
        if (live && sub == 0) {
            if (MODE == 0)
                acc_store<T, MODE>(A, B.Ph, a, B.Ph.m_g, B.gvb, B.rho, reinterpret_cast<T *>(B.gpb), nullptr, nullptr,
                                   nullptr);
            else
                acc_store<T, MODE>(A, B.Ph, a, T(0), B.gvb, nullptr, nullptr, B.acc, nullptr, nullptr);
        }
    }
}

template <class T, int DIM, int MODE> __device__ __forceinline__ void small_pairs(const SmallArgs<T> &B)
{
    if constexpr (sizeof(T) == 8 && DIM == 1 && (MODE == 0 || MODE == 2)) {
        if (B.lanes > 1) {
            small_pair_lanes<T, MODE>(B);
            return;
        }
    }
    small_pair<T, DIM, MODE>(B);
}

__device__ __forceinline__ void cluster_barrier()
{
    asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}

template <class T, class A, int DIM, int FMODE>
__global__ void __launch_bounds__(kSmallThreads, 1) k_step_small(const SmallArgs<T> B)
{
    __shared__ uint32_t wtot[kSmallThreads / 32];
    __shared__ CellShared<T> cs;
    auto barrier = [&] {
        if (B.cluster) {
            cluster_barrier();
            return true;
        }
        return grid_barrier(B.bar, B.spin, B.err, 0u);
    };
    const uint32_t rank = blockIdx.x * blockDim.x + threadIdx.x, count = gridDim.x * blockDim.x;
    const uint32_t n = B.ng + B.nd;

    // The scan runs on the counts that the last step left while the words that
    // tell whether it did are on their way (0.9 us a step at 2 x 20011); else it
    // runs again behind a count. A step behind one whose barrier gave up does
    // nothing (it finds its counts and its barrier half done).
    const int err = *reinterpret_cast<volatile int *>(B.err);
    const int counted = *reinterpret_cast<volatile int *>(B.counted);
    small_scan(B, wtot);
    if (err & kErrTimeout) return;
    if (!counted) {
        for (uint32_t i = rank; i < n; i += count)
            count_add_agg(i < B.ng ? &B.gcnt[B.gkey[i]] : &B.dcnt[B.dkey[i - B.ng]]);
        if (!barrier()) return;
        small_scan(B, wtot);
    }
    if (!barrier()) return;
    for (uint32_t i = rank; i < n; i += count) {
        if (i < B.ng) scatter_one_agg(i, B.gkey, B.gia, B.gcnt, B.gstart, B.gsrc, B.gtid, B.ng, B.err);
        else scatter_one_agg(i - B.ng, B.dkey, B.dia, B.dcnt, B.dstart, B.dsrc, B.dtid, B.nd, B.err);
    }
    if (!barrier()) return;
    for (uint32_t s = rank; s < n; s += count) {
        if (s < B.ng)
            rank_move<T>(s, B.gkey, B.gstart, B.gsrc, B.gtid, B.gpa, B.gva, B.gia, B.gpb, B.gvb, B.gib, B.ng, B.err);
        else
            rank_move<T>(s - B.ng, B.dkey, B.dstart, B.dsrc, B.dtid, B.dpa, B.dva, B.dia, B.dpb, B.dvb, B.dib, B.nd,
                         B.err);
    }
    if (!barrier()) return;
    small_pairs<T, DIM, 0>(B);
    if (!barrier()) return;
    small_pairs<T, DIM, FMODE>(B);
    if (!barrier()) return;
    if (rank == 0) *B.counted = 1;
    for (uint32_t c0 = blockIdx.x * B.cpc; c0 < B.G.ncells; c0 += gridDim.x * B.cpc) {
        // the dust starts half a CTA away from the gas, so that a CTA with
        // few particles updates both at once
        const uint32_t half = blockDim.x / 2;
        const uint32_t dust_tid = threadIdx.x < half ? threadIdx.x + half : threadIdx.x - half;
        // binary64: one lane per cell unless the CTA has only a few cells
        // (four lanes repeat the scalar part of the solve)
        if (sizeof(T) == 4 || B.cpc <= 16)
            cell_update_cta<T, A, DIM, false, 4, true>(cs, B.G, B.Ph, B.S, B.harmonic, B.has_frozen, B.adiabatic, c0,
                                                       B.cpc, dust_tid, B.gpb, B.gvb, B.gib, B.gkey, B.gstart, B.acc,
                                                       B.dpb, B.dvb, B.dkey, B.dstart, B.gcnt, B.dcnt);
        else
            cell_update_cta<T, A, DIM, false, 1, true>(cs, B.G, B.Ph, B.S, B.harmonic, B.has_frozen, B.adiabatic, c0,
                                                       B.cpc, dust_tid, B.gpb, B.gvb, B.gib, B.gkey, B.gstart, B.acc,
                                                       B.dpb, B.dvb, B.dkey, B.dstart, B.gcnt, B.dcnt);
        __syncthreads();
    }
}

template <class T, class A, int DIM> void *pick_mode(bool full)
{
    return full ? (void *)k_step_small<T, A, DIM, 3> : (void *)k_step_small<T, A, DIM, 2>;
}
template <class T, class A> void *pick_dim(int dim, bool full)
{
    return dim == 1 ? pick_mode<T, A, 1>(full) : pick_mode<T, A, 2>(full);
}
void *pick(int precision, int cell_acc, int dim, bool full)
{
    if (precision == TFSPH_FP64) return pick_dim<double, double>(dim, full);
    return cell_acc == TFSPH_CELL_ACC_FP64 ? pick_dim<float, df>(dim, full) : pick_dim<float, float>(dim, full);
}

// Launch of a grid that is one cluster.
void cluster_config(cudaLaunchConfig_t &cfg, cudaLaunchAttribute attr[1], const SmallPlan &P)
{
    cfg.gridDim = dim3((unsigned)P.grid);
    cfg.blockDim = dim3((unsigned)P.threads);
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = (unsigned)P.grid;
    attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
}

template <class T>
cudaError_t small_t(const LaunchCtx &L, const void *geo, const void *phys, PhaseBufs &G, PhaseBufs &D, void *rho,
                    void *acc, const StepArgs &S, const SmallPlan &P, GridBar *bar, int *counted)
{
    SmallArgs<T> B{};
    B.G = *static_cast<const Geo<T> *>(geo);
    B.Ph = *static_cast<const Phys<T> *>(phys);
    B.S = step_vals(S.tau, S.g);
    const int og = G.cur ^ 1, od = D.cur ^ 1;
    B.gpa = static_cast<const V4<T> *>(G.pos[G.cur]);
    B.gva = static_cast<const V4<T> *>(G.vel[G.cur]);
    B.dpa = static_cast<const V4<T> *>(D.pos[D.cur]);
    B.dva = static_cast<const V4<T> *>(D.vel[D.cur]);
    B.gpb = static_cast<V4<T> *>(G.pos[og]);
    B.gvb = static_cast<V4<T> *>(G.vel[og]);
    B.dpb = static_cast<V4<T> *>(D.pos[od]);
    B.dvb = static_cast<V4<T> *>(D.vel[od]);
    B.gia = G.id[G.cur];
    B.dia = D.id[D.cur];
    B.gib = G.id[og];
    B.dib = D.id[od];
    B.gkey = G.key;
    B.dkey = D.key;
    B.gcnt = G.count;
    B.dcnt = D.count;
    B.gstart = G.start;
    B.dstart = D.start;
    B.gsrc = G.tmp_src;
    B.dsrc = D.tmp_src;
    B.gtid = G.tmp_id;
    B.dtid = D.tmp_id;
    B.rho = static_cast<T *>(rho);
    B.acc = static_cast<V4<T> *>(acc);
    B.err = L.d_err;
    B.bar = bar;
    B.spin = P.spin;
    B.ng = (uint32_t)G.n;
    B.nd = (uint32_t)D.n;
    B.lanes = P.lanes;
    B.counted = counted;
    B.cluster = P.cluster;
    B.few = (double)G.n * (2 * B.G.R[0] + 1) <= 16.0 * (double)B.G.ncells;
    // cells shared out evenly over the CTAs, at most what four lanes each allow
    B.cpc = std::min((uint32_t)P.threads / 4, std::max(1u, (B.G.ncells + (uint32_t)P.grid - 1) / (uint32_t)P.grid));
    B.harmonic = S.tstar_mode == TFSPH_TSTAR_HARMONIC;
    B.has_frozen = S.has_frozen;
    B.adiabatic = B.Ph.eos == TFSPH_EOS_ADIABATIC;
    void *args[] = {&B};
    cudaLaunchConfig_t cfg{};
    cudaLaunchAttribute attr[1];
    if (P.cluster) {
        cluster_config(cfg, attr, P);
    } else {
        cfg.gridDim = dim3((unsigned)P.grid);
        cfg.blockDim = dim3((unsigned)P.threads);
        attr[0].id = cudaLaunchAttributeCooperative;
        attr[0].val.cooperative = 1;
        cfg.attrs = attr;
        cfg.numAttrs = 1;
    }
    cfg.stream = L.stream;
    const cudaError_t e = cudaLaunchKernelExC(&cfg, P.fn, args);
    if (e != cudaSuccess) return e;
    G.cur = og;
    D.cur = od;
    return cudaSuccess;
}

}  // namespace

// Which contexts take the one-launch step. us a step, one launch against one
// per phase (2 x n particles):
//   1D FP32 waves      2 x 1000 25 | 49, 2 x 16384 37 | 50, 2 x 32768 40 | 49, 2 x 131072 58 | 59
//   1D FP64 waves      2 x 1000 31 | 64, 2 x 16384 60 | 70, 2 x 32768 67 | 70, 2 x 131072 138 | 152
//   1D FP32, 600 candidates a particle   2 x 2000 216 | 303, 2 x 20000 223 | 325
//   shocks, FP32 and FP64   2 x 16384 61 | 98 and 262 | 652
//   2D columns, FP32   2 x 900 68 | 84, 2 x 4096 70 | 93, 2 x 16384 75 | 89
//   2D columns, FP64   2 x 900 379 | 383, 2 x 4096 379 | 490, 2 x 16384 356 | 505
// The particle limit is where the gain has become small in FP64; in FP32 it
// still gains some beyond (2 x 49152 41 | 50).
bool small_plan(const void *geo, const void *phys, int precision, int cell_acc, int dim, int64_t ng, int64_t nd,
                SmallPlan *P)
{
    *P = SmallPlan{};
    const bool f64 = precision == TFSPH_FP64;
    const uint32_t ncells = f64 ? static_cast<const Geo<double> *>(geo)->ncells : static_cast<const Geo<float> *>(geo)->ncells;
    const int av = f64 ? static_cast<const Phys<double> *>(phys)->av : static_cast<const Phys<float> *>(phys)->av;
    const int eos = f64 ? static_cast<const Phys<double> *>(phys)->eos : static_cast<const Phys<float> *>(phys)->eos;
    if (dim > 2 || ng <= 0 || nd <= 0 || ng + nd > kSmallParticles || ncells > kSmallCells) return false;
    const bool full = av || eos == TFSPH_EOS_ADIABATIC;
    void *fn = pick(precision, cell_acc, dim, full);
    // The sums here run in the order of the tiled walks. Where the passes do not
    // run on tiles (cells much finer than the particles' spacing, a y axis that
    // wraps fully), their order is another one and the step keeps their form;
    // an x axis that wraps fully has one order only.
    const int full_x = f64 ? static_cast<const Geo<double> *>(geo)->full[0] : static_cast<const Geo<float> *>(geo)->full[0];
    if (!full_x && !(gas_sums_tiled(geo, precision, dim, ng, 0) && gas_sums_tiled(geo, precision, dim, ng, full ? 3 : 2)))
        return false;
    int dev = 0, sms = 0, coop = 0;
    if (cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, dev) != cudaSuccess || !coop) {
        cudaGetLastError();
        return false;
    }
    // lanes per particle, while the warps still find a binary64 unit each (four an SM)
    int lanes = 1;
    if (f64 && dim == 1)
        while (lanes < 8 && (ng * lanes * 2 + 31) / 32 <= (int64_t)4 * sms) lanes *= 2;
    P->lanes = lanes;
    // A binary64 particle of many candidates with a lane of its own: the pair
    // sums bound both forms, and the tiles have more warps, up to a tile per few
    // cells (1D, isothermal, 20,000 + 20,000 particles, one launch against
    // phases: 60 candidates 166 against 165 us a step, 90: 230 against 214, 180:
    // 393 against 348, 600: 1317 against 1753).
    const int reach = f64 ? static_cast<const Geo<double> *>(geo)->R[0] : 0;
    const double seen = (double)ng * (2 * reach + 1) / (double)ncells;
    if (f64 && dim == 1 && lanes == 1 && !full && seen > 64.0 && seen <= 400.0) return false;
    // up to one CTA an SM. Up to kSmallCluster CTAs' worth of warps: one
    // cluster, whose barrier takes 0.1 us against about 1.5 us for the grid's.
    const int64_t warps = std::max((ng * lanes + 31) / 32, (nd + 31) / 32);
    P->cluster = warps <= 4 * kSmallCluster;
    P->grid = (int)std::min<int64_t>(P->cluster ? kSmallCluster : sms, warps);
    P->threads = 128;
    while (P->threads < kSmallThreads && warps * 32 > (int64_t)P->grid * P->threads) P->threads *= 2;
    // whether the device holds the cluster, or a CTA on every SM, at once
    if (P->cluster) {
        cudaLaunchConfig_t cfg{};
        cudaLaunchAttribute attr[1];
        cluster_config(cfg, attr, *P);
        int clusters = 0;
        if (cudaOccupancyMaxActiveClusters(&clusters, fn, &cfg) != cudaSuccess || clusters < 1) {
            cudaGetLastError();
            return false;
        }
    } else {
        int per_sm = 0;
        if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, fn, P->threads, 0) != cudaSuccess ||
            (int64_t)per_sm * sms < P->grid) {
            cudaGetLastError();
            return false;
        }
    }
    P->fn = fn;
    return true;
}

cudaError_t launch_step_small(const LaunchCtx &L, const void *geo, const void *phys, PhaseBufs &G, PhaseBufs &D,
                              void *rho, void *acc, const StepArgs &S, const SmallPlan &P, void *bar, int *counted)
{
    GridBar *b = static_cast<GridBar *>(bar);
    return L.precision == TFSPH_FP64 ? small_t<double>(L, geo, phys, G, D, rho, acc, S, P, b, counted)
                                     : small_t<float>(L, geo, phys, G, D, rho, acc, S, P, b, counted);
}

}  // namespace tfsph
