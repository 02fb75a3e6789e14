// Arithmetic of the implicit drag in cell (Sec. 2.3, Eqs. 17-21) shared by the
// single-context cell update and the batched step: the per-cell sums and
// implicit solve, and the per-particle update of each phase.
#pragma once

#include <type_traits>

#include "dfloat.cuh"
#include "tfsph_internal.cuh"

namespace tfsph {

// tau and g of a step for every accumulator type: float takes the leading
// parts, df the pairs, double the binary64 values. Filled on the host, so no
// kernel converts them.
struct StepVals {
    df tau, g[3];
    double dtau, dg[3];
};
inline StepVals step_vals(double tau, const double g[3])
{
    StepVals v;
    v.tau = df(tau);
    v.dtau = tau;
    for (int k = 0; k < 3; ++k) {
        v.g[k] = df(g[k]);
        v.dg[k] = g[k];
    }
    return v;
}
template <class A> __device__ __forceinline__ A step_val(df pair, double wide)
{
    if constexpr (std::is_same<A, df>::value) return pair;
    else if constexpr (sizeof(A) == 4) return pair.h;
    else return A(wide);
}

// One cell: N, L, sum v, sum u, sum A, sum t_j (or sum 1/t_j) in storage
// order, with accumulator type A (float, df or double), then
//   eps* = m_d L / (m_g N)                                (Eq. 17)
//   t*   = sum t_j / L   (or L / sum 1/t_j)               (Eq. 18)
//   w    = v_* - u_*                                      (Eq. 21)
//   w'   = (w + tau Abar) / (1 + tau (1 + eps*)/t*)
//   u_*' = u_* + tau g + (tau/t*) w',  v_*' = u_*' + w'
// which is the cell average of the implicit Eqs. 19-20. Returns 1 when the
// cell holds moving gas and dust (drag applies) and then sets un = u_*',
// vn = v_*', ig = 1/(1 + tau eps*/t*) and id = 1/(1 + tau/t*). With A = df it
// returns 2 where the binary32 exponent range may not hold the solve: a scalar
// outside the bounds of df_drag_fits, or a velocity so small (nonzero, below
// 2^-80) or so large that low parts are lost.
template <class T, class A, int DIM>
__device__ __forceinline__ int cell_drag_solve(const Phys<T> &Ph, const StepVals &S, int harmonic, int has_frozen,
                                               const V4<T> *__restrict__ gvel, const uint32_t *__restrict__ gid,
                                               const V4<T> *__restrict__ acc, uint32_t gs, uint32_t ge,
                                               const V4<T> *__restrict__ dvel, uint32_t ds, uint32_t de, T un_out[3],
                                               T vn_out[3], T &ig_out, T &id_out)
{
    constexpr bool kPair = std::is_same<A, df>::value;
    const A one = A(1.0f), zero = A(0.0f);
    uint32_t ng = 0, nd = 0;
    A st = zero;
    A sv[3] = {zero, zero, zero}, sa[3] = {zero, zero, zero}, su[3] = {zero, zero, zero};
    // a particle's component into a sum (df: value + float)
    auto add = [](A &s, T x) {
        if constexpr (kPair) s += (float)x;
        else s += A(x);
    };
    auto add_gas = [&](uint32_t idv, const V4<T> &v, const V4<T> &ac) {
        if (has_frozen && (idv & kFrozenBit)) return;
        ++ng;
        add(sv[0], v.x);
        add(sa[0], ac.x);
        if (DIM > 1) { add(sv[1], v.y); add(sa[1], ac.y); }
        if (DIM > 2) { add(sv[2], v.z); add(sa[2], ac.z); }
    };
    auto add_dust = [&](const V4<T> &u) {
        ++nd;
        add(su[0], u.x);
        if (DIM > 1) add(su[1], u.y);
        if (DIM > 2) add(su[2], u.z);
        if (harmonic) st += one / A(u.w);
        else add(st, u.w);
    };
    // the first gas and dust particles are loaded together (the usual cell
    // holds one or a few of each), the rest in storage order
    V4<T> v0{}, a0{}, u0{};
    uint32_t id0 = 0u;
    if (gs < ge) {
        v0 = gvel[gs];
        a0 = acc[gs];
        if (has_frozen) id0 = gid[gs];
    }
    if (ds < de) u0 = dvel[ds];
    // not unrolled: with a particle or two per cell the unrolled bodies only
    // cost registers and branches (128^3 box: 67 us against 82 unrolled)
    if (gs < ge) add_gas(id0, v0, a0);
#pragma unroll 1
    for (uint32_t a = gs + 1; a < ge; ++a) add_gas(has_frozen ? gid[a] : 0u, gvel[a], acc[a]);
    if (ds < de) add_dust(u0);
#pragma unroll 1
    for (uint32_t j = ds + 1; j < de; ++j) add_dust(dvel[j]);
    if (ng == 0 || nd == 0) return 0;
    const A tau = step_val<A>(S.tau, S.dtau);
    const A N = A(ng), L = A(nd);
    const A dust = A(Ph.m_d) * L, gas = A(Ph.m_g) * N;
    const A eps = dust / gas;
    // 1/N and 1/L from one division (N L is an exact product of counts)
    const A invNL = one / (N * L);
    const A invN = L * invNL, invL = N * invNL;
    // rt = tau / t*, with t* = st / L (mean) or L / st (harmonic mean)
    const A rt = harmonic ? tau * st * invL : tau * L / st;
    const A den = one + rt * (one + eps);
    const A invden = one / den;  // one division for the DIM components
    bool fits = true;
    if constexpr (kPair) fits = df_drag_fits(tau, st, gas, dust, rt, eps);
#pragma unroll
    for (int k = 0; k < DIM; ++k) {
        const A vs = sv[k] * invN;
        const A us = su[k] * invL;
        const A ab = sa[k] * invN;
        const A wn = ((vs - us) + tau * ab) * invden;
        const A un = us + tau * step_val<A>(S.g[k], S.dg[k]) + rt * wn;
        const A vn = un + wn;
        un_out[k] = T(un);
        vn_out[k] = T(vn);
        if constexpr (kPair) fits = fits && df_vel_fits(wn, un, vn, 0x1p100f);
    }
    // 1/(1 + rt eps) and 1/(1 + rt) from one division
    const A dg = one + rt * eps, dd = one + rt;
    const A invgd = one / (dg * dd);
    ig_out = T(dd * invgd);
    id_out = T(dg * invgd);
    return fits ? 1 : 2;
}

// The binary64 solve of a cell outside df's range (see above): rare, so out of
// line and off the register allocation of the common path.
template <class T, int DIM>
__device__ __noinline__ int cell_drag_wide(const Phys<T> Ph, const StepVals S, int harmonic, int has_frozen,
                                           const V4<T> *__restrict__ gvel, const uint32_t *__restrict__ gid,
                                           const V4<T> *__restrict__ acc, uint32_t gs, uint32_t ge,
                                           const V4<T> *__restrict__ dvel, uint32_t ds, uint32_t de, T *out)
{
    T un[3] = {T(0), T(0), T(0)}, vn[3] = {T(0), T(0), T(0)}, ig = T(0), id = T(0);
    const int r = cell_drag_solve<T, double, DIM>(Ph, S, harmonic, has_frozen, gvel, gid, acc, gs, ge, dvel, ds, de,
                                                  un, vn, ig, id);
#pragma unroll
    for (int k = 0; k < DIM; ++k) {
        out[k] = un[k];
        out[3 + k] = vn[k];
    }
    out[6] = ig;
    out[7] = id;
    return r;
}

// cell_drag_solve with df's rare cells taken in binary64.
template <class T, class A, int DIM>
__device__ __forceinline__ int cell_drag(const Phys<T> &Ph, const StepVals &S, int harmonic, int has_frozen,
                                         const V4<T> *__restrict__ gvel, const uint32_t *__restrict__ gid,
                                         const V4<T> *__restrict__ acc, uint32_t gs, uint32_t ge,
                                         const V4<T> *__restrict__ dvel, uint32_t ds, uint32_t de, T un[3], T vn[3],
                                         T &ig, T &id)
{
    int r = cell_drag_solve<T, A, DIM>(Ph, S, harmonic, has_frozen, gvel, gid, acc, gs, ge, dvel, ds, de, un, vn, ig,
                                       id);
    if constexpr (std::is_same<A, df>::value) {
        if (r == 2) {
            T o[8];
            r = cell_drag_wide<T, DIM>(Ph, S, harmonic, has_frozen, gvel, gid, acc, gs, ge, dvel, ds, de, o);
#pragma unroll
            for (int k = 0; k < DIM; ++k) {
                un[k] = o[k];
                vn[k] = o[3 + k];
            }
            ig = o[6];
            id = o[7];
        }
    }
    return r;
}

// A value of lane src of the warp (df, float or double).
template <class A> __device__ __forceinline__ A lane_value(unsigned mask, A v, int src)
{
    if constexpr (std::is_same<A, df>::value)
        return df(__shfl_sync(mask, v.h, src), __shfl_sync(mask, v.l, src));
    else return __shfl_sync(mask, v, src);
}

// The same solve by four consecutive lanes of a warp, lane k of them on
// component k (lane 3 on the stopping times), for cells holding several
// particles: four times the threads of the form above, loads of a component
// by consecutive lanes, four particles in flight per lane, and the terms of
// every sum still added in storage order by one lane, so both forms round
// alike. Lane k returns un[k], vn[k] in un, vn; ig and id come back in every
// lane. mask: the four lanes, which call it together.
template <class T, class A, int DIM>
__device__ __forceinline__ int cell_drag_lanes(const Phys<T> &Ph, const StepVals &S, int harmonic, int has_frozen,
                                               const V4<T> *__restrict__ gvel, const uint32_t *__restrict__ gid,
                                               const V4<T> *__restrict__ acc, uint32_t gs, uint32_t ge,
                                               const V4<T> *__restrict__ dvel, uint32_t ds, uint32_t de,
                                               unsigned mask, T &un_out, T &vn_out, T &ig_out, T &id_out)
{
    constexpr bool kPair = std::is_same<A, df>::value;
    const int k = threadIdx.x & 3;
    const A one = A(1.0f), zero = A(0.0f);
    auto add = [](A &s, T x) {
        if constexpr (kPair) s += (float)x;
        else s += A(x);
    };
    const T *gv = reinterpret_cast<const T *>(gvel) + k, *ga = reinterpret_cast<const T *>(acc) + k;
    const T *dv = reinterpret_cast<const T *>(dvel) + k;
    const bool axis = k < DIM, last = k == 3;
    uint32_t ng = 0, nd = de - ds;
    A sv = zero, sa = zero, su = zero;  // lane 3: su is the sum over the stopping times
    constexpr int kAhead = 4;
    for (uint32_t a = gs; a < ge; a += kAhead) {
        T v[kAhead], ac[kAhead];
        uint32_t fz[kAhead];
#pragma unroll
        for (int u = 0; u < kAhead; ++u) {
            const bool in = a + u < ge;
            v[u] = in && axis ? gv[4 * (size_t)(a + u)] : T(0);
            ac[u] = in && axis ? ga[4 * (size_t)(a + u)] : T(0);
            fz[u] = in ? (has_frozen ? gid[a + u] & kFrozenBit : 0u) : 1u;
        }
#pragma unroll
        for (int u = 0; u < kAhead; ++u)
            if (!fz[u]) {
                ++ng;
                add(sv, v[u]);
                add(sa, ac[u]);
            }
    }
    for (uint32_t j = ds; j < de; j += kAhead) {
        T w[kAhead];
#pragma unroll
        for (int u = 0; u < kAhead; ++u) w[u] = j + u < de && (axis || last) ? dv[4 * (size_t)(j + u)] : T(1);
#pragma unroll
        for (int u = 0; u < kAhead; ++u)
            if (j + u < de) {
                if (harmonic && last) su += one / A(w[u]);
                else add(su, w[u]);
            }
    }
    if (ng == 0 || nd == 0) return 0;
    const A st = lane_value(mask, su, (threadIdx.x & 31) | 3);
    const A tau = step_val<A>(S.tau, S.dtau);
    const A N = A(ng), L = A(nd);
    const A dust = A(Ph.m_d) * L, gas = A(Ph.m_g) * N;
    const A eps = dust / gas;
    const A invNL = one / (N * L);
    const A invN = L * invNL, invL = N * invNL;
    const A rt = harmonic ? tau * st * invL : tau * L / st;
    const A den = one + rt * (one + eps);
    const A invden = one / den;
    const A dg = one + rt * eps, dd = one + rt;
    const A invgd = one / (dg * dd);
    ig_out = T(dd * invgd);
    id_out = T(dg * invgd);
    bool fits = true;
    if constexpr (kPair) fits = df_drag_fits(tau, st, gas, dust, rt, eps);
    if (axis) {
        const A g = k == 0 ? step_val<A>(S.g[0], S.dg[0])
                           : (k == 1 ? step_val<A>(S.g[1], S.dg[1]) : step_val<A>(S.g[2], S.dg[2]));
        const A us = su * invL;
        const A wn = ((sv * invN - us) + tau * (sa * invN)) * invden;
        const A un = us + tau * g + rt * wn;
        const A vn = un + wn;
        un_out = T(un);
        vn_out = T(vn);
        if constexpr (kPair) fits = fits && df_vel_fits(wn, un, vn, 0x1p100f);
    }
    if constexpr (kPair) {
        if (!__all_sync(mask, fits)) return 2;
    }
    return 1;
}

// Gas particle (Eq. 19 solved for v'): v' = u_*' + (v + tau (A + g) - u_*') ig
// in a drag cell, v + tau (A + g) otherwise; e' = e + tau de/dt (adiabatic);
// x' = x + tau v' with the periodic wrap.
template <class T, int DIM>
__device__ __forceinline__ void gas_particle_update(const Geo<T> &G, T tau_t, const T gt[3], int adiabatic, V4<T> &p,
                                                    V4<T> &v, const V4<T> &ac, bool drag, const T us[3], T ig)
{
    T vn[3];
    vn[0] = v.x + tau_t * (ac.x + gt[0]);
    vn[1] = DIM > 1 ? v.y + tau_t * (ac.y + gt[1]) : T(0);
    vn[2] = DIM > 2 ? v.z + tau_t * (ac.z + gt[2]) : T(0);
    if (drag) {
#pragma unroll
        for (int k = 0; k < DIM; ++k) vn[k] = us[k] + (vn[k] - us[k]) * ig;
    }
    v.x = vn[0];
    p.x = p.x + tau_t * vn[0];
    if (G.per[0]) p.x = wrap_periodic(p.x, G.lo[0], G.L[0]);
    if (DIM > 1) {
        v.y = vn[1];
        p.y = p.y + tau_t * vn[1];
        if (G.per[1]) p.y = wrap_periodic(p.y, G.lo[1], G.L[1]);
    }
    if (DIM > 2) {
        v.z = vn[2];
        p.z = p.z + tau_t * vn[2];
        if (G.per[2]) p.z = wrap_periodic(p.z, G.lo[2], G.L[2]);
    }
    if (adiabatic) v.w = v.w + tau_t * ac.w;
    p.w = T(0);
}

// Dust particle (Eq. 20 solved for u'): u' = v_*' + (u + tau g - v_*') id in a
// drag cell, u + tau g otherwise; x' = x + tau u' with the periodic wrap.
template <class T, int DIM>
__device__ __forceinline__ void dust_particle_update(const Geo<T> &G, T tau_t, const T gt[3], V4<T> &p, V4<T> &u,
                                                     bool drag, const T vs[3], T id)
{
    T un[3];
    un[0] = u.x + tau_t * gt[0];
    un[1] = DIM > 1 ? u.y + tau_t * gt[1] : T(0);
    un[2] = DIM > 2 ? u.z + tau_t * gt[2] : T(0);
    if (drag) {
#pragma unroll
        for (int k = 0; k < DIM; ++k) un[k] = vs[k] + (un[k] - vs[k]) * id;
    }
    u.x = un[0];
    p.x = p.x + tau_t * un[0];
    if (G.per[0]) p.x = wrap_periodic(p.x, G.lo[0], G.L[0]);
    if (DIM > 1) {
        u.y = un[1];
        p.y = p.y + tau_t * un[1];
        if (G.per[1]) p.y = wrap_periodic(p.y, G.lo[1], G.L[1]);
    }
    if (DIM > 2) {
        u.z = un[2];
        p.z = p.z + tau_t * un[2];
        if (G.per[2]) p.z = wrap_periodic(p.z, G.lo[2], G.L[2]);
    }
}

// The cells [c0, c0 + cpc) and their particles, by one CTA (see drag.cu):
// phase 1 with LANES threads per cell, then the particle updates and the next
// cell keys; the dust loop starts at thread dust_tid. With COUNT the next keys
// are counted too (gcnt, dcnt: all zero before). The caller syncs before it
// reuses the shared arrays.
template <class T> struct CellShared {
    T us[3][kCellsPerCta], vs[3][kCellsPerCta], ig[kCellsPerCta], id[kCellsPerCta];
    int drag[kCellsPerCta];
    // binary64: the cells' first slots, by which a particle finds its cell
    // without the key's binary64 arithmetic
    uint32_t first[sizeof(T) == 8 ? 2 : 1][sizeof(T) == 8 ? kCellsPerCta : 1];
};
// The last of n cells whose first slot is at or before i.
__device__ __forceinline__ uint32_t slot_cell(const uint32_t *first, uint32_t n, uint32_t i)
{
    uint32_t lo = 0, hi = n - 1;
    while (lo < hi) {
        const uint32_t mid = (lo + hi + 1) >> 1;
        if (first[mid] <= i) lo = mid;
        else hi = mid - 1;
    }
    return lo;
}
template <class T, class A, int DIM, bool EST, int LANES, bool COUNT = false>
__device__ __forceinline__ void
cell_update_cta(CellShared<T> &s, const Geo<T> &G, const Phys<T> &Ph, const StepVals &S, int harmonic, int has_frozen,
                int adiabatic, uint32_t c0, uint32_t cpc, uint32_t dust_tid, V4<T> *__restrict__ gpos,
                V4<T> *__restrict__ gvel, const uint32_t *__restrict__ gid, uint32_t *__restrict__ gkey,
                const uint32_t *__restrict__ gstart, const V4<T> *__restrict__ acc, V4<T> *__restrict__ dpos,
                V4<T> *__restrict__ dvel, uint32_t *__restrict__ dkey, const uint32_t *__restrict__ dstart,
                uint32_t *__restrict__ gcnt = nullptr, uint32_t *__restrict__ dcnt = nullptr)
{
    constexpr bool kWide = sizeof(T) == 8;
    const uint32_t ncells = G.ncells;
    const uint32_t lc0 = threadIdx.x / LANES;
    const uint32_t c = c0 + lc0;

    // ---- phase 1: per-cell sums and the implicit solve ----
    int drag = 0;
    if (lc0 < cpc && c < ncells) {
        const uint32_t gs = gstart[c], ge = gstart[c + 1], ds = dstart[c], de = dstart[c + 1];
        if (kWide && (LANES == 1 || (threadIdx.x & 3) == 0)) {
            s.first[0][lc0] = gs;
            s.first[kWide ? 1 : 0][lc0] = ds;
        }
        T un[3] = {T(0), T(0), T(0)}, vn[3] = {T(0), T(0), T(0)}, ig = T(0), id = T(0);
        if constexpr (LANES == 1) {
            drag = cell_drag<T, A, DIM>(Ph, S, harmonic, has_frozen, gvel, gid, acc, gs, ge, dvel, ds, de, un, vn, ig,
                                        id);
            if (drag) {
#pragma unroll
                for (int k = 0; k < DIM; ++k) {
                    s.us[k][lc0] = un[k];
                    s.vs[k][lc0] = vn[k];
                }
                s.ig[lc0] = ig;
                s.id[lc0] = id;
            }
        } else {
            const int k = threadIdx.x & 3;
            const unsigned mask = 0xfu << (threadIdx.x & 28);
            drag = cell_drag_lanes<T, A, DIM>(Ph, S, harmonic, has_frozen, gvel, gid, acc, gs, ge, dvel, ds, de, mask,
                                              un[0], vn[0], ig, id);
            if (drag == 1) {
                if (k < DIM) {
                    s.us[k][lc0] = un[0];
                    s.vs[k][lc0] = vn[0];
                }
                if (k == 0) {
                    s.ig[lc0] = ig;
                    s.id[lc0] = id;
                }
            } else if (drag == 2) {
                if (k == 0) {
                    T o[8];
                    cell_drag_wide<T, DIM>(Ph, S, harmonic, has_frozen, gvel, gid, acc, gs, ge, dvel, ds, de, o);
                    for (int m = 0; m < DIM; ++m) {
                        s.us[m][lc0] = o[m];
                        s.vs[m][lc0] = o[3 + m];
                    }
                    s.ig[lc0] = o[6];
                    s.id[lc0] = o[7];
                }
            }
        }
    }
    if (lc0 < cpc && (LANES == 1 || (threadIdx.x & 3) == 0)) s.drag[lc0] = drag;
    __syncthreads();

    // ---- phase 2: particle updates over the CTA's storage ranges ----
    const uint32_t c1 = min(c0 + cpc, ncells);
    const T tau_t = step_val<T>(S.tau, S.dtau);
    const T gt[3] = {step_val<T>(S.g[0], S.dg[0]), step_val<T>(S.g[1], S.dg[1]), step_val<T>(S.g[2], S.dg[2])};
    {
        const uint32_t a0 = gstart[c0], a1 = gstart[c1];
        for (uint32_t a = a0 + threadIdx.x; a < a1; a += blockDim.x) {
            V4<T> p = gpos[a];
            if (has_frozen && (gid[a] & kFrozenBit)) {
                const uint32_t key = cell_key<T, DIM, EST>(G, p.x, p.y, p.z);
                gkey[a] = key;
                if (COUNT) atomicAdd(&gcnt[key], 1u);
                continue;
            }
            V4<T> v = gvel[a];
            const V4<T> ac = acc[a];
            const uint32_t lc = kWide ? slot_cell(s.first[0], c1 - c0, a)
                                      : cell_key<T, DIM, EST>(G, p.x, p.y, p.z) - c0;
            const bool dr = lc < cpc && s.drag[lc];
            T us[3] = {T(0), T(0), T(0)}, ig = T(0);
            if (dr) {
                ig = s.ig[lc];
#pragma unroll
                for (int k = 0; k < DIM; ++k) us[k] = s.us[k][lc];
            }
            gas_particle_update<T, DIM>(G, tau_t, gt, adiabatic, p, v, ac, dr, us, ig);
            gpos[a] = p;
            gvel[a] = v;
            const uint32_t key = cell_key<T, DIM, EST>(G, p.x, p.y, p.z);
            gkey[a] = key;
            if (COUNT) atomicAdd(&gcnt[key], 1u);
        }
    }
    {
        const uint32_t j0 = dstart[c0], j1 = dstart[c1];
        for (uint32_t j = j0 + dust_tid; j < j1; j += blockDim.x) {
            V4<T> p = dpos[j];
            V4<T> u = dvel[j];
            const uint32_t lc = kWide ? slot_cell(s.first[kWide ? 1 : 0], c1 - c0, j)
                                      : cell_key<T, DIM, EST>(G, p.x, p.y, p.z) - c0;
            const bool dr = lc < cpc && s.drag[lc];
            T vs[3] = {T(0), T(0), T(0)}, id = T(0);
            if (dr) {
                id = s.id[lc];
#pragma unroll
                for (int k = 0; k < DIM; ++k) vs[k] = s.vs[k][lc];
            }
            dust_particle_update<T, DIM>(G, tau_t, gt, p, u, dr, vs, id);
            dpos[j] = p;
            dvel[j] = u;
            const uint32_t key = cell_key<T, DIM, EST>(G, p.x, p.y, p.z);
            dkey[j] = key;
            if (COUNT) atomicAdd(&dcnt[key], 1u);
        }
    }
}

}  // namespace tfsph
