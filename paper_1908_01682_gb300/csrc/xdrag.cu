// The two other drag schemes of the paper on the same binning, densities and
// gas pressure force: ISPH (Sec. 2.2, Eqs. 11-16) and MK (Sec. 2.1,
// Eqs. 8-10).
//
// Drag coefficient K = rho_d / t_stop (Eq. 7) with the per-particle stopping
// times t_j (vel.w of the dust); at a gas particle ISPH interpolates K like
// any dust field: K_a = m_d sum_j W_aj / t_j. In MK, K_aj / (rho_a,g rho_j,d)
// = 1 / (rho_a,g t_j), sigma = the dimension, eta^2 = 0.001 h^2. Frozen
// (wall) gas particles enter the density and pressure sums and take no part
// in the drag.
//
// Cross-phase sums, with the neighbour decision of the gas pair sums. In 3D
// (FP32, isothermal, no walls) a CTA stages the source particles of a tile of
// cells and its halo, 32 bytes each, and its threads take one target each
// (k_xsum_tile). Otherwise one thread per target walks the other phase's
// candidate cells in global memory (k_xsum; k_xsum_rest behind the tiles).
//   ISPH at gas a over dust:  rho^d_a = m_d sum W,  K_a,  u_a = m_d sum u_j/rho_j W
//   ISPH at dust j over gas:  rho^g_j = m_g sum W,  v_j = m_g sum_moving v_a/rho_a W,
//     e_j (adiabatic), pressure acceleration A_j = -(Q_j + q_j G_j) (Eq. 14)
//     with G_j = m_g sum grad_j W, Q_j = m_g sum q_a grad_j W, q_j = p_j/rho_j^2
//   MK at gas a:  D_a = -sigma m_d / rho_a sum_j ((v_a - u_j).d)/(r^2 + eta^2) d W / t_j
//   MK at dust j: D_j =  sigma m_g / t_j sum_a ((v_a - u_j).d)/(r^2 + eta^2) d W / rho_a
// (d = x_target - x_source; ((v_a - u_j).r) r is even in r).
// Then one thread per particle: the ISPH 2x2 implicit solve in (own velocity,
// interpolated velocity of the other phase)
//   w' = (v - u + tau A) / (1 + tau (alpha + beta)),  alpha = K/rho_g, beta = K/rho_d,
//   gas keeps v' = v + tau (A + g) - tau alpha w', dust keeps u' = u + tau g + tau beta w',
// or the MK explicit update v' = v + tau (A + D + g), u' = u + tau (D + g); then
// x' = x + tau v' (periodic wrap) and the next cell keys.
#include "pair.cuh"
#include "tile.cuh"

namespace tfsph {
namespace {

constexpr int kXThreads = 128;

enum XKind { kIsphAtGas = 0, kIsphAtDust = 1, kMkAtGas = 2, kMkAtDust = 3 };

template <class T> struct XArgs {
    // targets
    const V4<T> *tpos, *tvel;
    const uint32_t *tid;
    const T *trho;      // target density (MK gas: rho_g)
    int n;
    // sources (the other phase)
    const V4<T> *spos, *svel;
    const uint32_t *sid;
    const uint32_t *sstart, *tstart;  // cell ranges of the sources and the targets
    const T *srho;      // source density (rho_d for ISPH at gas, rho_g otherwise)
    int has_frozen;     // gas carries frozen flags (in tid for gas targets, sid for gas sources)
    // outputs
    V4<T> *out4;        // ISPH gas: (u_a, K_a); ISPH dust: (v_j, rho^g_j); MK: D
    V4<T> *out4b;       // ISPH dust: (A_j, 0)
    T *out1;            // ISPH gas: rho^d_a
    // Tiled sums: two words, one of which is set where they run (NULL: they do),
    // per tile whether its targets are left to a thread each, and whether any are.
    const int *gate = nullptr;
    uint8_t *over = nullptr;
    int *any = nullptr;
    int tile[3] = {1, 1, 1}, tiles[3] = {1, 1, 1};  // cells of a tile, tiles per axis
};

// One target's sums over its candidate cells in global memory.
template <class T, int DIM, int KIND>
__device__ __forceinline__ void xsum_global(const Geo<T> &G, const Phys<T> &Ph, const XArgs<T> &X, uint32_t t)
{
    const bool gas_target = KIND == kIsphAtGas || KIND == kMkAtGas;
    if (gas_target && X.has_frozen && (X.tid[t] & kFrozenBit)) return;
    const V4<T> pt = X.tpos[t];
    const V4<T> vt = X.tvel[t];
    const T eta2 = T(0.001) * G.h * G.h;
    T s0 = T(0), s1 = T(0);                         // rho, K (ISPH gas) / rho, e (ISPH dust)
    T a[3] = {T(0), T(0), T(0)};                    // u_a, v_j or the MK sum
    T gs[3] = {T(0), T(0), T(0)}, qs[3] = {T(0), T(0), T(0)};
    auto range = [&](uint32_t b0, uint32_t n, auto seam) {
        for (uint32_t b = b0; b < b0 + n; ++b) {
            const V4<T> pb = X.spos[b];
            T d[3];
            const T r2 = pair_r2<T, DIM, decltype(seam)::value>(G, pt, pb, d);
            if (!(r2 < G.h2x4)) continue;
            const V4<T> vb = X.svel[b];
            const T r = approx_sqrt(r2);
            const T W = kernel_w(G, r * G.inv_h);
            if (KIND == kIsphAtGas) {
                const T w = Ph.m_d * W;
                s0 += w;
                s1 += approx_div(w, vb.w);  // t_j
                const T c = approx_div(w, X.srho[b]);
                a[0] += c * vb.x;
                a[1] += c * vb.y;
                a[2] += c * vb.z;
            } else if (KIND == kIsphAtDust) {
                const T w = Ph.m_g * W;
                const T inv_rho = approx_div(T(1), X.srho[b]);
                s0 += w;
                if (Ph.eos == TFSPH_EOS_ADIABATIC) s1 += w * vb.w * inv_rho;
                if (!(X.has_frozen && (X.sid[b] & kFrozenBit))) {
                    a[0] += w * vb.x * inv_rho;
                    a[1] += w * vb.y * inv_rho;
                    a[2] += w * vb.z * inv_rho;
                }
                if (r2 > T(0)) {
                    const T F = Ph.m_g * kernel_f(G, r * G.inv_h, approx_div(G.h, r));  // m_g (1/r) dW/dr
                    const T q = pb.w;                                       // p_a / rho_a^2
                    for (int k = 0; k < 3; ++k) {
                        gs[k] += F * d[k];
                        qs[k] += q * F * d[k];
                    }
                }
            } else {
                // MK: ((v_a - u_j) . d) / (r^2 + eta^2) W, times 1/t_j (gas target) or 1/rho_a (dust target)
                if (KIND == kMkAtDust && X.has_frozen && (X.sid[b] & kFrozenBit)) continue;
                T rel;
                if (KIND == kMkAtGas) rel = (vt.x - vb.x) * d[0] + (vt.y - vb.y) * d[1] + (vt.z - vb.z) * d[2];
                else rel = (vb.x - vt.x) * d[0] + (vb.y - vt.y) * d[1] + (vb.z - vt.z) * d[2];
                const T coef = approx_div(T(1), KIND == kMkAtGas ? vb.w : X.srho[b]);
                const T f = approx_div(coef * rel, r2 + eta2) * W;
                a[0] += f * d[0];
                a[1] += f * d[1];
                a[2] += f * d[2];
            }
        }
    };
    for_each_range<T, DIM>(G, X.sstart, pt.x, pt.y, pt.z, [&](uint32_t b0, uint32_t n, bool seam) {
        if (seam) range(b0, n, SeamTag<true>{});
        else range(b0, n, SeamTag<false>{});
    });
    V4<T> o;
    if (KIND == kIsphAtGas) {
        o.x = a[0]; o.y = a[1]; o.z = a[2]; o.w = s1;
        X.out4[t] = o;
        X.out1[t] = s0;
    } else if (KIND == kIsphAtDust) {
        T qj = T(0);
        if (s0 > T(0)) qj = Ph.eos == TFSPH_EOS_ADIABATIC ? Ph.gm1 * s1 / s0 : Ph.cs2 / s0;
        o.x = a[0]; o.y = a[1]; o.z = a[2]; o.w = s0;
        X.out4[t] = o;
        V4<T> A;
        A.x = -(qs[0] + qj * gs[0]);
        A.y = -(qs[1] + qj * gs[1]);
        A.z = -(qs[2] + qj * gs[2]);
        A.w = T(0);
        X.out4b[t] = A;
    } else {
        const T sig = T(DIM);
        const T c = KIND == kMkAtGas ? -sig * Ph.m_d / X.trho[t] : sig * Ph.m_g / vt.w;
        o.x = c * a[0]; o.y = c * a[1]; o.z = c * a[2]; o.w = T(0);
        X.out4[t] = o;
    }
}

template <class T, int DIM, int KIND>
__global__ void __launch_bounds__(kXThreads, sizeof(T) == 4 ? 12 : 1) k_xsum(Geo<T> G, Phys<T> Ph, XArgs<T> X)
{
    const uint32_t t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t < (uint32_t)X.n) xsum_global<T, DIM, KIND>(G, Ph, X, t);
}

// Behind the tiled sums of both kinds (gas targets in the first gas_blocks
// CTAs): all targets where the tiled sums did not run, else those of the tiles
// left to it. One launch, which usually returns at once (4 us a step).
template <int KIND> __device__ __forceinline__ void xsum_rest(const Geo<float> &G, const Phys<float> &Ph,
                                                              const XArgs<float> &X, uint32_t t)
{
    const bool all = X.gate && !(X.gate[0] | X.gate[1]);
    if (!all && !*X.any) return;
    if (t >= (uint32_t)X.n) return;
    if (!all) {
        const float4 p = X.tpos[t];
        const int c[3] = {exact_cell(G, 0, p.x), exact_cell(G, 1, p.y), exact_cell(G, 2, p.z)};
        if (!X.over[c[0] / X.tile[0] + X.tiles[0] * (c[1] / X.tile[1] + X.tiles[1] * (c[2] / X.tile[2]))]) return;
    }
    xsum_global<float, 3, KIND>(G, Ph, X, t);
}
template <int AT_GAS, int AT_DUST>
__global__ void __launch_bounds__(kXThreads, 12)
k_xsum_rest(Geo<float> G, Phys<float> Ph, XArgs<float> Xg, XArgs<float> Xd, uint32_t gas_blocks)
{
    if (blockIdx.x < gas_blocks) xsum_rest<AT_GAS>(G, Ph, Xg, blockIdx.x * blockDim.x + threadIdx.x);
    else xsum_rest<AT_DUST>(G, Ph, Xd, (blockIdx.x - gas_blocks) * blockDim.x + threadIdx.x);
}

// ---------------------------------------------------------------------------
// Tiled sums (3D, FP32, isothermal, no walls)
// ---------------------------------------------------------------------------
// A source is staged as (x, y, z, c1) and (vx, vy, vz, c2): c1 = 1/t_j (ISPH and
// MK at gas), p/rho^2 (ISPH at dust) or 1/rho (MK at dust), c2 = 1/rho (ISPH).
//
// Walking the candidates in global memory took 20,600 instructions per warp of
// targets with 13 of 32 lanes active, each load touching up to 32 lines: the
// 60-odd instructions of a pair ran in every iteration in which any lane had a
// neighbour. Here the lanes of a warp go through the same rows of cells
// together and only test candidates; each lane puts its neighbours in a small
// queue of its own (kQueue entries in shared memory), and when a queue is half
// full every lane evaluates one entry, so that the pair arithmetic runs with
// nearly all lanes active.
__device__ __forceinline__ float approx_rcp(float x)
{
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}
constexpr int kXTileThreads = 512;
constexpr int kQueue = 8;
// 2 CTAs per SM: 2 x (112 KB + static + 1 KB reserved) of 228 KB
constexpr int kXTileSmem = 112 * 1024;
constexpr int kXQueueBytes = kQueue * kXTileThreads * 2;

// The targets of a staged tile. SEAM: displacements take the periodic image
// (tiles that could not be staged with their seam shifts).
template <int KIND, bool SEAM>
__device__ __forceinline__ void xsum_tile_walk(const Geo<float> &G, const Phys<float> &Ph, const TileCfg &C,
                                               const int c0[3], const float orig[3], const XArgs<float> &X,
                                               const uint16_t *lstart, const int *rowpref, const int *rowg,
                                               const float4 *sa, const float4 *sb, uint16_t *queue, int owned)
{
    constexpr unsigned kAll = 0xffffffffu;
    const int lane = threadIdx.x & 31;
    const float eta2 = 0.001f * G.h * G.h;
    for (int p0 = (int)threadIdx.x - lane; p0 < owned; p0 += blockDim.x) {
        const bool live = p0 + lane < owned;
        const int p = min(p0 + lane, owned - 1);
        int lo = 0, hi = C.nrows - 1;
        while (lo < hi) {
            const int mid = (lo + hi + 1) >> 1;
            if (rowpref[mid] <= p) lo = mid;
            else hi = mid - 1;
        }
        const uint32_t t = (uint32_t)(rowg[lo] + p - rowpref[lo]);
        float4 pt = X.tpos[t];
        float4 vt = make_float4(0.0f, 0.0f, 0.0f, 1.0f);
        if (KIND == kMkAtGas || KIND == kMkAtDust) vt = X.tvel[t];
        float f[3];
        int h[3];
        {
            float tc;
            h[0] = axis_cell(pt.x, G.lo[0], G.inv_w[0], G.n[0], tc);
            f[0] = tc - (float)h[0];
            h[1] = axis_cell(pt.y, G.lo[1], G.inv_w[1], G.n[1], tc);
            f[1] = tc - (float)h[1];
            h[2] = axis_cell(pt.z, G.lo[2], G.inv_w[2], G.n[2], tc);
            f[2] = tc - (float)h[2];
#pragma unroll
            for (int k = 0; k < 3; ++k) h[k] += G.R[k] - c0[k];
        }
        if (!SEAM) {
            pt.x = sub_rn(pt.x, orig[0]);
            pt.y = sub_rn(pt.y, orig[1]);
            pt.z = sub_rn(pt.z, orig[2]);
        }
        float s0 = 0.0f, s1 = 0.0f, a[3] = {0.0f, 0.0f, 0.0f};
        float gs[3] = {0.0f, 0.0f, 0.0f}, qs[3] = {0.0f, 0.0f, 0.0f};
        uint32_t head = 0, tail = 0;
        // queue positions in bytes
        constexpr uint32_t kSlot = 2 * kXTileThreads, kWrap = (kQueue - 1) * kSlot;
        unsigned char *qu = reinterpret_cast<unsigned char *>(queue + threadIdx.x);

        // every lane takes one of its neighbours; the sums leave out the
        // kernel's normalisation and the mass, applied once at the end
        auto pop = [&] {
            if (head == tail) return;
            const int j = *reinterpret_cast<const uint16_t *>(qu + (head & kWrap));
            head += kSlot;
            const float4 q = sa[j], v = sb[j];
            float d[3];
            const float r2 = pair_r2<float, 3, SEAM>(G, pt, q, d);
            if (KIND == kIsphAtDust) {
                const float inv_r = r2 >= pair_r2_min<float>() ? pair_rsqrt(r2) : 0.0f;
                const float qq = r2 * inv_r * G.inv_h;
                const float w = kernel_w4(qq);
                s0 += w;
                const float c = w * v.w;
                a[0] += c * v.x;
                a[1] += c * v.y;
                a[2] += c * v.z;
                const float e = positive_part(2.0f - qq);
                const float F = below_one(qq) ? -3.0f + 2.25f * qq : (e * e) * (Ph.hm075 * inv_r);
                const float Fq = F * q.w;
#pragma unroll
                for (int k = 0; k < 3; ++k) {
                    gs[k] += F * d[k];
                    qs[k] += Fq * d[k];
                }
            } else {
                const float w = kernel_w4(pair_sqrt(r2) * G.inv_h);
                if (KIND == kIsphAtGas) {
                    s0 += w;
                    s1 += w * q.w;
                    const float c = w * v.w;
                    a[0] += c * v.x;
                    a[1] += c * v.y;
                    a[2] += c * v.z;
                } else {
                    const float rel = (vt.x - v.x) * d[0] + (vt.y - v.y) * d[1] + (vt.z - v.z) * d[2];
                    const float c = approx_rcp(r2 + eta2) * (q.w * rel) * w;
                    a[0] += c * d[0];
                    a[1] += c * d[1];
                    a[2] += c * d[2];
                }
            }
        };

#pragma unroll 1
        for (int oz = -G.R[2]; oz <= G.R[2]; ++oz) {
            const float sz = slab_dist(oz, f[2]) * G.w[2];
            // (rows outside the halo: only where a target on a cell face is
            // placed one cell off, beyond the radius by a rounding)
            const float remz = live && (unsigned)(h[2] + oz) < (unsigned)C.H[2] ? G.lim2 - sz * sz : -1.0f;
            if (!__any_sync(kAll, remz > 0.0f)) continue;
#pragma unroll 1
            for (int oy = -G.R[1]; oy <= G.R[1]; oy += 2) {
                // two rows of cells at a time: [ja, ja + na), then [jb, jb + nb)
                int jr[2] = {0, 0}, nr[2] = {0, 0};
#pragma unroll
                for (int m = 0; m < 2; ++m) {
                    const float sy = slab_dist(oy + m, f[1]) * G.w[1];
                    const float rem = oy + m <= G.R[1] ? remz - sy * sy : -1.0f;
                    if (rem > 0.0f && (unsigned)(h[1] + oy + m) < (unsigned)C.H[1]) {
                        const float tx = pair_sqrt(rem) * G.inv_w[0];
                        const int ohi = min(G.R[0], max(0, floor_int(f[0] + tx)));
                        const int olo = -min(G.R[0], max(0, floor_int(tx - f[0] + 1.0f)));
                        const int row = C.H[0] * ((h[1] + oy + m) + C.H[1] * (h[2] + oz));
                        jr[m] = lstart[row + max(h[0] + olo, 0)];
                        nr[m] = lstart[row + min(h[0] + ohi + 1, C.H[0])] - jr[m];
                    }
                }
                const int len = nr[0] + nr[1], jump = jr[1] - nr[0] - jr[0];
                const int most = __reduce_max_sync(kAll, len);
#pragma unroll 1
                for (int k0 = 0; k0 < most; k0 += kQueue / 2) {
                    bool near[kQueue / 2];
                    int j[kQueue / 2];
#pragma unroll
                    for (int u = 0; u < kQueue / 2; ++u) {
                        const int k = k0 + u;
                        // (past a lane's candidates: some other staged word)
                        j[u] = jr[0] + k + (k >= nr[0] ? jump : 0);
                        float d[3];
                        near[u] = pair_r2<float, 3, SEAM>(G, pt, sa[j[u]], d) < G.h2x4 && k < len;
                    }
#pragma unroll
                    for (int u = 0; u < kQueue / 2; ++u)
                        if (near[u]) {
                            *reinterpret_cast<uint16_t *>(qu + (tail & kWrap)) = (uint16_t)j[u];
                            tail += kSlot;
                        }
                    // room for the next half queue in every lane
                    while (__any_sync(kAll, tail - head >= kSlot * (kQueue / 2))) pop();
                }
            }
        }
        while (__any_sync(kAll, tail != head)) pop();
        if (!live) continue;

        const float mw = (KIND == kIsphAtGas || KIND == kMkAtGas ? Ph.m_d : Ph.m_g) * Ph.wnorm4;
        if (KIND == kIsphAtGas) {
            X.out4[t] = make_float4(mw * a[0], mw * a[1], mw * a[2], mw * s1);
            X.out1[t] = mw * s0;
        } else if (KIND == kIsphAtDust) {
            s0 *= mw;
            const float qj = s0 > 0.0f ? Ph.cs2 / s0 : 0.0f, mf = -Ph.mfnorm;
            X.out4[t] = make_float4(mw * a[0], mw * a[1], mw * a[2], s0);
            X.out4b[t] = make_float4(mf * (qs[0] + qj * gs[0]), mf * (qs[1] + qj * gs[1]), mf * (qs[2] + qj * gs[2]),
                                     0.0f);
        } else {
            const float c = -3.0f * mw / (KIND == kMkAtGas ? X.trho[t] : vt.w);
            X.out4[t] = make_float4(c * a[0], c * a[1], c * a[2], 0.0f);
        }
    }
}

template <int KIND>
__global__ void __launch_bounds__(kXTileThreads, 2)
k_xsum_tile(Geo<float> G, Phys<float> Ph, TileCfg C, XArgs<float> X)
{
    if (X.gate && !(X.gate[0] | X.gate[1])) return;
    extern __shared__ __align__(64) unsigned char smem[];
    __shared__ int wsum[kXTileThreads / 32];
    uint16_t *lstart = reinterpret_cast<uint16_t *>(smem);                 // nhalo + 1
    int *rowpref = reinterpret_cast<int *>(smem + lstart_bytes(C.nhalo));  // nrows + 1
    int *rowg = rowpref + C.nrows + 1;                                     // nrows
    float4 *sa = reinterpret_cast<float4 *>(smem + C.offset);
    float4 *sb = sa + C.cap;
    uint16_t *queue = reinterpret_cast<uint16_t *>(sb + C.cap);

    const int tid = threadIdx.x;
    int b = blockIdx.x;
    const int tx = b % C.nt[0];
    b /= C.nt[0];
    const int ty = b % C.nt[1], tz = b / C.nt[1];
    const int c0[3] = {tx * C.T[0], ty * C.T[1], tz * C.T[2]};
    int ext[3];
#pragma unroll
    for (int k = 0; k < 3; ++k) ext[k] = min(C.T[k], G.n[k] - c0[k]);

    // seam shifts, as in the gas pair sums: exact where lo = 0 and the halo
    // lies over one seam of the axis only
    int low[3] = {0, 0, 0}, high[3] = {0, 0, 0};
    bool crosses = false, exact = true;
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        if (!G.per[k]) continue;
        low[k] = c0[k] < G.R[k];
        high[k] = c0[k] + ext[k] + G.R[k] > G.n[k];
        if (low[k] || high[k]) {
            crosses = true;
            if (!(G.lo[k] == 0.0f) || (low[k] && high[k]) || (high[k] && 2 * (c0[k] - G.R[k]) < G.n[k])) exact = false;
        }
    }
    const bool shifted = crosses && exact;
    float orig[3];
#pragma unroll
    for (int k = 0; k < 3; ++k) orig[k] = shifted && high[k] ? G.L[k] : 0.0f;

    for (int r = tid; r < C.nrows; r += blockDim.x) {
        const int oy = r % C.T[1], oz = r / C.T[1];
        int c = 0, g = 0;
        if (oy < ext[1] && oz < ext[2]) {
            const uint32_t key = (uint32_t)G.n[0] * ((uint32_t)(c0[1] + oy) + (uint32_t)G.n[1] * (uint32_t)(c0[2] + oz));
            g = (int)X.tstart[key + c0[0]];
            c = (int)X.tstart[key + c0[0] + ext[0]] - g;
        }
        rowg[r] = g;
        rowpref[r] = c;
    }
    // the global cell of halo cell h, or -1
    auto halo_key = [&](int h, int hk[3]) -> int {
        halo_coords(h, C, hk[0], hk[1], hk[2]);
        int g[3];
#pragma unroll
        for (int k = 0; k < 3; ++k) g[k] = hk[k] < ext[k] + 2 * G.R[k] ? halo_cell(G, k, c0[k], hk[k]) : -1;
        if (g[0] < 0 || g[1] < 0 || g[2] < 0) return -1;
        return (int)((uint32_t)g[0] + (uint32_t)G.n[0] * ((uint32_t)g[1] + (uint32_t)G.n[1] * (uint32_t)g[2]));
    };
    for (int h = tid; h < C.nhalo; h += blockDim.x) {
        int hk[3];
        const int key = halo_key(h, hk);
        // a count that does not fit 16 bits makes the tile exceed cap anyway
        lstart[h] = key < 0 ? 0 : (uint16_t)min(X.sstart[key + 1] - X.sstart[key], 0xFFFFu);
    }
    __syncthreads();
    const int total = block_scan_smem(lstart, C.nhalo, wsum);
    block_scan_smem(rowpref, C.nrows, wsum);
    const int owned = rowpref[C.nrows];
    // A halo that does not fit: the targets are left to k_xsum_rest. A tile's
    // own threads, walking global memory for them, were the last to finish by far
    // (both phases in a layer of a quarter of the box, 50^3: ISPH 3444 -> 2261 us, MK
    // 2180 -> 827; 96^3: 7560 -> 5465 and 5531 -> 3401; of half: 1287 -> 1210, 809 -> 635,
    // 4015 -> 3190, 2984 -> 2129), except where few tiles overflow a little
    // (50^3, cells of 1.5 spacings: 389 -> 424 and 290 -> 319).
    const bool later = total > C.cap;
    if (tid == 0) {
        X.over[blockIdx.x] = later;
        if (later) *X.any = 1;
    }
    if (later) return;
    for (int h = tid; h < C.nhalo; h += blockDim.x) {
        const int j0 = lstart[h], j1 = lstart[h + 1];
        if (j1 == j0) continue;
        int hk[3];
        const int key = halo_key(h, hk);
        const uint32_t g0 = X.sstart[key];
        float sh[3] = {0.0f, 0.0f, 0.0f};
        if (shifted) {
#pragma unroll
            for (int k = 0; k < 3; ++k) {
                const int raw = c0[k] - G.R[k] + hk[k];
                if ((high[k] && raw < G.n[k]) || (low[k] && raw < 0)) sh[k] = G.L[k];
            }
        }
        for (int j = j0; j < j1; ++j) {
            const uint32_t gi = g0 + (uint32_t)(j - j0);
            float4 q = X.spos[gi], v = X.svel[gi];
            const float t = v.w;
            q.x = sub_rn(q.x, sh[0]);
            q.y = sub_rn(q.y, sh[1]);
            q.z = sub_rn(q.z, sh[2]);
            if (KIND == kIsphAtGas || KIND == kMkAtGas) q.w = approx_div(1.0f, t);
            if (KIND == kMkAtDust) q.w = approx_div(1.0f, X.srho[gi]);
            if (KIND == kIsphAtGas || KIND == kIsphAtDust) v.w = approx_div(1.0f, X.srho[gi]);
            sa[j] = q;
            sb[j] = v;
        }
    }
    __syncthreads();
    if (crosses && !shifted)
        xsum_tile_walk<KIND, true>(G, Ph, C, c0, orig, X, lstart, rowpref, rowg, sa, sb, queue, owned);
    else
        xsum_tile_walk<KIND, false>(G, Ph, C, c0, orig, X, lstart, rowpref, rowg, sa, sb, queue, owned);
}

// Whether the tiled sums pay, from the places f of kSample particles of a phase
// (block 0 gas, 1 dust) inside their cells: not while both phases sit on
// lattices in step with the cells. Summed over the axes, the
// variance of f is then at most 0.03 (displacements of up to 0.17 of a
// spacing), or, wherever the lattice lies in the cells (on their faces f is
// next to 0 or 1), they hold one phase exactly: 1 - R^2 below 0.01, R the length of
// the mean of exp(2 pi i f). A lattice displaced about the faces has lanes in
// cells on both sides of them and counts as scattered (0.05 of a spacing, tiles
// against a thread per target: 96^3 ISPH 1327 against 1397 us, MK 1126 against
// 1078; 75^3 639 against 844 and 529 against 652; not displaced at all, 96^3:
// 1383 against 1021 and 1176 against 768).
constexpr int kSample = 4096;
__global__ void __launch_bounds__(512)
k_scattered(Geo<float> G, const float4 *__restrict__ gpos, uint32_t ng, const float4 *__restrict__ dpos, uint32_t nd,
            int *out)
{
    const float4 *pos = blockIdx.x == 0 ? gpos : dpos;
    const uint32_t n = blockIdx.x == 0 ? ng : nd, m = min((uint32_t)kSample, n);
    constexpr int kSums = 12;  // per axis: f, f^2, cos, sin
    float s[kSums] = {};
    for (uint32_t i = threadIdx.x; i < m; i += blockDim.x) {
        // in scattered order (evenly spaced slots may all be the first of their cell)
        const float4 p = pos[__umulhi(i * 2654435761u, n)];
        const float x[3] = {p.x, p.y, p.z};
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            const float t = (x[k] - G.lo[k]) * G.inv_w[k], f = t - floorf(t);
            s[4 * k] += f;
            s[4 * k + 1] += f * f;
            s[4 * k + 2] += cospif(2.0f * f);
            s[4 * k + 3] += sinpif(2.0f * f);
        }
    }
    __shared__ float part[16][kSums];
#pragma unroll
    for (int k = 0; k < kSums; ++k) {
        for (int o = 16; o > 0; o >>= 1) s[k] += __shfl_xor_sync(0xffffffffu, s[k], o);
        if ((threadIdx.x & 31) == 0) part[threadIdx.x >> 5][k] = s[k];
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        float spread = 0.0f, lost = 0.0f;
        for (int k = 0; k < 3; ++k) {
            float a[4] = {0.0f, 0.0f, 0.0f, 0.0f};
            for (int w = 0; w < 16; ++w)
                for (int q = 0; q < 4; ++q) a[q] += part[w][4 * k + q];
            for (int q = 0; q < 4; ++q) a[q] /= (float)m;
            spread += a[1] - a[0] * a[0];
            lost += 1.0f - (a[2] * a[2] + a[3] * a[3]);
        }
        out[blockIdx.x] = spread > 0.03f && lost > 0.01f;  // (no particles, or no numbers: 0)
    }
}

// Targets that fill the chip with one thread each (12 CTAs an SM).
constexpr int64_t kXFill = (int64_t)kSmCount * 12 * kXThreads;

// Most sources per cell of the tiled form beyond kXFill targets (cells of 1.5
// spacings, 3.4 sources: 96^3 ISPH 1435 us against 1744, MK 1058 against 1253;
// of two spacings, 8 sources: 2109 and 1645 against 1864 and 1306).
constexpr double kXMean = 5.0;

// The tiled sums of one kind, where they apply (a tile for every SM): alone when
// a thread per target would not fill the chip (50^3 targets: 69 us against
// 126-130 us on the lattice, 106 against 208 us off it); beyond, only while
// k_scattered tells that they pay. There (884,736 targets displaced by up to
// 0.35 of a spacing) they take 613 and 653 us against 702 and 898 us for ISPH
// and 625 against 711-722 us for MK, because the lanes' rows differ in length;
// on a lattice (0.05) they do not, and a thread per target takes 367-449 us
// against 426-453. False: not launched.
template <int KIND>
bool launch_xsum_tile(const LaunchCtx &L, const Geo<float> &G, const Phys<float> &Ph, XArgs<float> &X, double mean,
                      const XDragBufs &B, bool dust, cudaError_t &e)
{
    TileCfg C{};
    size_t smem = 0;
    if (X.n <= 0 || X.has_frozen || Ph.eos != TFSPH_EOS_ISOTHERMAL || (mean > kXMean && X.n > kXFill) ||
        !plan_tiles(G, 3, mean, 32, kXTileSmem - kXQueueBytes, kXTileThreads, C, smem) || C.cap > 0xFFFF ||
        (int64_t)C.nt[0] * C.nt[1] * C.nt[2] < kSmCount)
        return false;
    // (per call: the attribute belongs to the device's copy of the kernel)
    e = cudaFuncSetAttribute(k_xsum_tile<KIND>, cudaFuncAttributeMaxDynamicSharedMemorySize, kXTileSmem);
    if (e != cudaSuccess) return false;
    if (X.n > kXFill) X.gate = B.gate;
    X.over = B.over + (dust ? G.ncells : 0u);
    X.any = B.any;
    for (int k = 0; k < 3; ++k) {
        X.tile[k] = C.T[k];
        X.tiles[k] = C.nt[k];
    }
    k_xsum_tile<KIND><<<(unsigned)(C.nt[0] * C.nt[1] * C.nt[2]), kXTileThreads, smem + kXQueueBytes, L.stream>>>(G, Ph, C, X);
    return true;
}

// Both kinds of sums of a scheme.
template <class T, int DIM, int AT_GAS, int AT_DUST>
cudaError_t launch_xsums(const LaunchCtx &L, const Geo<T> &G, const Phys<T> &Ph, XArgs<T> Xg, XArgs<T> Xd, double mean_g,
                         double mean_d, const XDragBufs &B, int64_t *launches)
{
    bool gas = false, dust = false;
    cudaError_t e = cudaSuccess;
    if constexpr (sizeof(T) == 4 && DIM == 3) {
        if (std::max(Xg.n, Xd.n) > kXFill) {
            k_scattered<<<2, 512, 0, L.stream>>>(G, Xg.tpos, (uint32_t)Xg.n, Xd.tpos, (uint32_t)Xd.n, B.gate);
            ++*launches;
        }
        gas = launch_xsum_tile<AT_GAS>(L, G, Ph, Xg, mean_d, B, false, e);
        if (e == cudaSuccess) dust = launch_xsum_tile<AT_DUST>(L, G, Ph, Xd, mean_g, B, true, e);
        if (e != cudaSuccess) return e;
    }
    auto blocks = [](int n) { return (unsigned)((n + kXThreads - 1) / kXThreads); };
    if (Xg.n > 0 && !gas) k_xsum<T, DIM, AT_GAS><<<blocks(Xg.n), kXThreads, 0, L.stream>>>(G, Ph, Xg);
    if (Xd.n > 0 && !dust) k_xsum<T, DIM, AT_DUST><<<blocks(Xd.n), kXThreads, 0, L.stream>>>(G, Ph, Xd);
    if constexpr (sizeof(T) == 4 && DIM == 3) {
        if (gas || dust) {
            const unsigned bg = gas ? blocks(Xg.n) : 0u, bd = dust ? blocks(Xd.n) : 0u;
            k_xsum_rest<AT_GAS, AT_DUST><<<bg + bd, kXThreads, 0, L.stream>>>(G, Ph, Xg, Xd, bg);
            ++*launches;
        }
    }
    *launches += (Xg.n > 0) + (Xd.n > 0);  // (a sum of each, tiled or not)
    return cudaGetLastError();
}

// Per-particle updates. SCHEME: TFSPH_DRAG_ISPH or TFSPH_DRAG_MK.
template <class T, int DIM, int SCHEME>
__global__ void __launch_bounds__(256)
k_xupdate_gas(Geo<T> G, Phys<T> Ph, T tau, T g0, T g1, T g2, int has_frozen, V4<T> *__restrict__ pos,
              V4<T> *__restrict__ vel, const uint32_t *__restrict__ id, uint32_t *__restrict__ key,
              const T *__restrict__ rho, const V4<T> *__restrict__ acc, const V4<T> *__restrict__ x4,
              const T *__restrict__ x1, int n, int *__restrict__ any)
{
    const int a = blockIdx.x * blockDim.x + threadIdx.x;
    if (a == 0 && any) *any = 0;  // k_xsum_rest is done with it
    if (a >= n) return;
    V4<T> p = pos[a];
    if (has_frozen && (id[a] & kFrozenBit)) {
        key[a] = cell_key<T, DIM>(G, p.x, p.y, p.z);
        return;
    }
    V4<T> v = vel[a];
    const V4<T> A = acc[a], X = x4[a];
    const T gv[3] = {g0, g1, g2};
    T vv[3] = {v.x, v.y, v.z};
    const T AA[3] = {A.x, A.y, A.z}, XX[3] = {X.x, X.y, X.z};
    if (SCHEME == TFSPH_DRAG_ISPH) {
        const T rd = x1[a];
        if (rd > T(0)) {
            const T alpha = X.w / rho[a], beta = X.w / rd;
            const T den = T(1) + tau * (alpha + beta);
#pragma unroll
            for (int k = 0; k < DIM; ++k) {
                const T wn = (vv[k] - XX[k] + tau * AA[k]) / den;
                vv[k] = vv[k] + tau * (AA[k] + gv[k]) - tau * alpha * wn;
            }
        } else {
#pragma unroll
            for (int k = 0; k < DIM; ++k) vv[k] = vv[k] + tau * (AA[k] + gv[k]);
        }
    } else {
#pragma unroll
        for (int k = 0; k < DIM; ++k) vv[k] = vv[k] + tau * (AA[k] + XX[k] + gv[k]);
    }
    v.x = vv[0];
    p.x = p.x + tau * vv[0];
    if (G.per[0]) p.x = wrap_periodic(p.x, G.lo[0], G.L[0]);
    if (DIM > 1) {
        v.y = vv[1];
        p.y = p.y + tau * vv[1];
        if (G.per[1]) p.y = wrap_periodic(p.y, G.lo[1], G.L[1]);
    }
    if (DIM > 2) {
        v.z = vv[2];
        p.z = p.z + tau * vv[2];
        if (G.per[2]) p.z = wrap_periodic(p.z, G.lo[2], G.L[2]);
    }
    if (Ph.eos == TFSPH_EOS_ADIABATIC) v.w = v.w + tau * A.w;
    p.w = T(0);
    pos[a] = p;
    vel[a] = v;
    key[a] = cell_key<T, DIM>(G, p.x, p.y, p.z);
}

template <class T, int DIM, int SCHEME>
__global__ void __launch_bounds__(256)
k_xupdate_dust(Geo<T> G, T tau, T g0, T g1, T g2, V4<T> *__restrict__ pos, V4<T> *__restrict__ vel,
               uint32_t *__restrict__ key, const T *__restrict__ rho_d, const V4<T> *__restrict__ x4,
               const V4<T> *__restrict__ x4b, int n)
{
    const int j = blockIdx.x * blockDim.x + threadIdx.x;
    if (j >= n) return;
    V4<T> p = pos[j];
    V4<T> u = vel[j];
    const V4<T> X = x4[j];
    const T gv[3] = {g0, g1, g2};
    T uu[3] = {u.x, u.y, u.z};
    const T XX[3] = {X.x, X.y, X.z};
    if (SCHEME == TFSPH_DRAG_ISPH) {
        if (X.w > T(0)) {
            const V4<T> A = x4b[j];
            const T AA[3] = {A.x, A.y, A.z};
            const T alpha = rho_d[j] / (X.w * u.w), beta = T(1) / u.w;
            const T den = T(1) + tau * (alpha + beta);
#pragma unroll
            for (int k = 0; k < DIM; ++k) {
                const T wn = (XX[k] - uu[k] + tau * AA[k]) / den;
                uu[k] = uu[k] + tau * gv[k] + tau * beta * wn;
            }
        } else {
#pragma unroll
            for (int k = 0; k < DIM; ++k) uu[k] = uu[k] + tau * gv[k];
        }
    } else {
#pragma unroll
        for (int k = 0; k < DIM; ++k) uu[k] = uu[k] + tau * (XX[k] + gv[k]);
    }
    u.x = uu[0];
    p.x = p.x + tau * uu[0];
    if (G.per[0]) p.x = wrap_periodic(p.x, G.lo[0], G.L[0]);
    if (DIM > 1) {
        u.y = uu[1];
        p.y = p.y + tau * uu[1];
        if (G.per[1]) p.y = wrap_periodic(p.y, G.lo[1], G.L[1]);
    }
    if (DIM > 2) {
        u.z = uu[2];
        p.z = p.z + tau * uu[2];
        if (G.per[2]) p.z = wrap_periodic(p.z, G.lo[2], G.L[2]);
    }
    pos[j] = p;
    vel[j] = u;
    key[j] = cell_key<T, DIM>(G, p.x, p.y, p.z);
}

unsigned blocks_for(int64_t n, int threads) { return (unsigned)((n + threads - 1) / threads); }

template <class T, int DIM>
cudaError_t xdrag_t(const LaunchCtx &L, const void *geo, const void *phys, PhaseBufs &Gp, PhaseBufs &Dp,
                    const void *rho_g, const void *rho_d, const void *acc, const XDragBufs &B, const StepArgs &S,
                    int scheme, int64_t *launches)
{
    const Geo<T> &G = *static_cast<const Geo<T> *>(geo);
    const Phys<T> &Ph = *static_cast<const Phys<T> *>(phys);
    const int ng = (int)Gp.n, nd = (int)Dp.n;
    auto *gpos = static_cast<V4<T> *>(Gp.pos[Gp.cur]);
    auto *gvel = static_cast<V4<T> *>(Gp.vel[Gp.cur]);
    auto *dpos = static_cast<V4<T> *>(Dp.pos[Dp.cur]);
    auto *dvel = static_cast<V4<T> *>(Dp.vel[Dp.cur]);
    const T *rg = static_cast<const T *>(rho_g);
    const T *rd = static_cast<const T *>(rho_d);
    XArgs<T> at_gas{gpos, gvel, Gp.id[Gp.cur], rg, ng, dpos, dvel, Dp.id[Dp.cur], Dp.start, Gp.start, rd,
                    S.has_frozen,
                    static_cast<V4<T> *>(B.g4), nullptr, static_cast<T *>(B.g1)};
    XArgs<T> at_dust{dpos, dvel, Dp.id[Dp.cur], rd, nd, gpos, gvel, Gp.id[Gp.cur], Gp.start, Dp.start, rg,
                     S.has_frozen,
                     static_cast<V4<T> *>(B.d4), static_cast<V4<T> *>(B.d4b), nullptr};
    const bool isph = scheme == TFSPH_DRAG_ISPH;
    const double mean_g = (double)ng / (double)G.ncells, mean_d = (double)nd / (double)G.ncells;
    const cudaError_t e =
        isph ? launch_xsums<T, DIM, kIsphAtGas, kIsphAtDust>(L, G, Ph, at_gas, at_dust, mean_g, mean_d, B, launches)
             : launch_xsums<T, DIM, kMkAtGas, kMkAtDust>(L, G, Ph, at_gas, at_dust, mean_g, mean_d, B, launches);
    if (e != cudaSuccess) return e;
    const T tau = T(S.tau), g0 = T(S.g[0]), g1 = T(S.g[1]), g2 = T(S.g[2]);
    *launches += (ng > 0) + (nd > 0);
    if (ng > 0) {
        if (isph)
            k_xupdate_gas<T, DIM, TFSPH_DRAG_ISPH><<<blocks_for(ng, 256), 256, 0, L.stream>>>(
                G, Ph, tau, g0, g1, g2, S.has_frozen, gpos, gvel, Gp.id[Gp.cur], Gp.key, rg,
                static_cast<const V4<T> *>(acc), static_cast<const V4<T> *>(B.g4), static_cast<const T *>(B.g1), ng, B.any);
        else
            k_xupdate_gas<T, DIM, TFSPH_DRAG_MK><<<blocks_for(ng, 256), 256, 0, L.stream>>>(
                G, Ph, tau, g0, g1, g2, S.has_frozen, gpos, gvel, Gp.id[Gp.cur], Gp.key, rg,
                static_cast<const V4<T> *>(acc), static_cast<const V4<T> *>(B.g4), static_cast<const T *>(B.g1), ng, B.any);
    }
    if (nd > 0) {
        if (isph)
            k_xupdate_dust<T, DIM, TFSPH_DRAG_ISPH><<<blocks_for(nd, 256), 256, 0, L.stream>>>(
                G, tau, g0, g1, g2, dpos, dvel, Dp.key, rd, static_cast<const V4<T> *>(B.d4),
                static_cast<const V4<T> *>(B.d4b), nd);
        else
            k_xupdate_dust<T, DIM, TFSPH_DRAG_MK><<<blocks_for(nd, 256), 256, 0, L.stream>>>(
                G, tau, g0, g1, g2, dpos, dvel, Dp.key, rd, static_cast<const V4<T> *>(B.d4),
                static_cast<const V4<T> *>(B.d4b), nd);
    }
    return cudaGetLastError();
}

}  // namespace

cudaError_t launch_xdrag(const LaunchCtx &L, const void *geo, const void *phys, PhaseBufs &G, PhaseBufs &D,
                         const void *rho_g, const void *rho_d, const void *acc, const XDragBufs &B,
                         const StepArgs &S, int scheme, int64_t *launches)
{
    if (L.precision == TFSPH_FP64) {
        switch (L.dim) {
            case 1: return xdrag_t<double, 1>(L, geo, phys, G, D, rho_g, rho_d, acc, B, S, scheme, launches);
            case 2: return xdrag_t<double, 2>(L, geo, phys, G, D, rho_g, rho_d, acc, B, S, scheme, launches);
            default: return xdrag_t<double, 3>(L, geo, phys, G, D, rho_g, rho_d, acc, B, S, scheme, launches);
        }
    }
    switch (L.dim) {
        case 1: return xdrag_t<float, 1>(L, geo, phys, G, D, rho_g, rho_d, acc, B, S, scheme, launches);
        case 2: return xdrag_t<float, 2>(L, geo, phys, G, D, rho_g, rho_d, acc, B, S, scheme, launches);
        default: return xdrag_t<float, 3>(L, geo, phys, G, D, rho_g, rho_d, acc, B, S, scheme, launches);
    }
}

}  // namespace tfsph
