// Implicit drag in cell (Sec. 2.3, Eqs. 17-21) fused with the particle
// update and the next step's cell keys.
//
// One CTA owns kCellsPerCta (or fewer) consecutive cells and, because
// particles are stored in cell order, the contiguous gas and dust ranges of
// those cells.
//   Phase 1 (thread per cell, accumulator type A: float, double, or df, the
//   two-float form of double that the FP32 state takes): N, L, sum v, sum u,
//     sum A, sum t_j (or sum 1/t_j) in storage order, then
//       eps* = m_d L / (m_g N)                                (Eq. 17)
//       t*   = sum t_j / L   (or L / sum 1/t_j)               (Eq. 18)
//       w    = v_* - u_*                                      (Eq. 21)
//       w'   = (w + tau Abar) / (1 + tau (1 + eps*)/t*)
//       u_*' = u_* + tau g + (tau/t*) w',  v_*' = u_*' + w'
//     which is the cell average of the implicit Eqs. 19-20.
//   Phase 2 (thread per particle, coalesced): the particle equations of
//     Eqs. 19-20 solved for the new velocity, written in the form
//       v_a' = u_*' + (v_a + tau (A_a + g) - u_*') / (1 + tau eps*/t*)
//       u_j' = v_*' + (u_j + tau g - v_*') / (1 + tau/t*)
//     (well conditioned for tau/t* up to 1e6); explicit update in cells with
//     N = 0 or L = 0; e' = e + tau de/dt; x' = x + tau v' (periodic wrap);
//     next cell key.
// The per-cell results live in shared memory only; nothing per cell is
// written to global memory.
#include <algorithm>

#include "drag_ops.cuh"

namespace tfsph {
namespace {

// LANES: 1, a thread per cell in phase 1, or 4, four lanes per cell (cells of
// several particles, whose serial sums otherwise wait on one load at a time).
// The CTA owns blockDim.x / LANES cells.
template <class T, class A, int DIM, bool EST, int LANES>
__global__ void __launch_bounds__(kCellsPerCta, (sizeof(T) == 4 && sizeof(A) == 4) ? 12 : (sizeof(T) == 4 ? 8 : 1))
k_cell_update(Geo<T> G, Phys<T> Ph, StepVals S, int harmonic, int has_frozen, int adiabatic,
              V4<T> *__restrict__ gpos, V4<T> *__restrict__ gvel, const uint32_t *__restrict__ gid,
              uint32_t *__restrict__ gkey, const uint32_t *__restrict__ gstart, const V4<T> *__restrict__ acc,
              V4<T> *__restrict__ dpos, V4<T> *__restrict__ dvel, uint32_t *__restrict__ dkey,
              const uint32_t *__restrict__ dstart)
{
    __shared__ CellShared<T> s;
    const uint32_t cpc = blockDim.x / LANES;
    cell_update_cta<T, A, DIM, EST, LANES>(s, G, Ph, S, harmonic, has_frozen, adiabatic, blockIdx.x * cpc, cpc,
                                           threadIdx.x, gpos, gvel, gid, gkey, gstart, acc, dpos, dvel, dkey, dstart);
}

// Reverse mode of the cell drag and the particle update (isothermal gas,
// no viscosity). Inputs, in storage order: lambda of the step's outputs
// x', v' (gas) and x', u' (dust) as V4; outputs: lambda_A (gas, V4),
// lambda_v (gas, written over lgv), lambda_u (dust, over ldu) and
// lambda_t_stop (dust, added to lts). With lv = lambda_v' + tau lambda_x'
// (x' = x + tau v'), for a cell with drag:
//   v_a' = u*' + (v_a + tau (A_a + g) - u*') ig      ig = 1/(1 + rt eps)
//   u_j' = v*' + (u_j + tau g - v*') id              id = 1/(1 + rt)
//   v*' = u*' + w',  u*' = ubar + tau g + rt w',  w' = (vbar - ubar + tau Abar)/den,
//   den = 1 + rt (1 + eps),  rt = tau / t*,  t* = mean (or harmonic mean) of t_j.
struct CellRange {
    uint32_t gs, ge, ds, de;  // the cell's gas and dust slots
};
// What a cell hands its particles: ig, id, lambda_t*, t*, L, then per axis
// the lambdas of vbar, Abar (per gas particle) and ubar (per dust particle).
template <class T> struct CellLam {
    T ig, id, lt, tst, L, lv[3], lA[3], lu[3];
};

// One cell's reverse solve with accumulator A; 0 without drag, 2 when df's
// range may not hold it (the bounds of cell_drag_solve, on the lambdas too).
template <class T, class A, int DIM>
__device__ __forceinline__ int cell_adjoint_solve(const Phys<T> &Ph, const StepVals &S, int harmonic, int has_frozen,
                                                  const V4<T> *__restrict__ gvel, const uint32_t *__restrict__ gid,
                                                  const V4<T> *__restrict__ acc, const V4<T> *__restrict__ dvel,
                                                  const V4<T> *__restrict__ lgx, const V4<T> *lgv,
                                                  const V4<T> *__restrict__ ldx, const V4<T> *ldu, const CellRange &R,
                                                  CellLam<T> &O)
{
    constexpr bool kPair = std::is_same<A, df>::value;
    const A one = A(1.0f), zero = A(0.0f);
    const A tau = step_val<A>(S.tau, S.dtau);
    A gv[3];
#pragma unroll
    for (int k = 0; k < 3; ++k) gv[k] = step_val<A>(S.g[k], S.dg[k]);
    uint32_t ng = 0, nd = 0;
    A st = zero;
    A sv[3] = {zero, zero, zero}, sa[3] = {zero, zero, zero}, su[3] = {zero, zero, zero};
    auto add = [](A &s, T x) {
        if constexpr (kPair) s += (float)x;
        else s += A(x);
    };
    for (uint32_t a = R.gs; a < R.ge; ++a) {
        if (has_frozen && (gid[a] & kFrozenBit)) continue;
        const V4<T> v = gvel[a];
        const V4<T> ac = acc[a];
        ++ng;
        add(sv[0], v.x);
        add(sa[0], ac.x);
        if (DIM > 1) { add(sv[1], v.y); add(sa[1], ac.y); }
        if (DIM > 2) { add(sv[2], v.z); add(sa[2], ac.z); }
    }
    for (uint32_t j = R.ds; j < R.de; ++j) {
        const V4<T> u = dvel[j];
        ++nd;
        add(su[0], u.x);
        if (DIM > 1) add(su[1], u.y);
        if (DIM > 2) add(su[2], u.z);
        if (harmonic) st += one / A(u.w);
        else add(st, u.w);
    }
    if (ng == 0 || nd == 0) return 0;
    const A N = A(ng), L = A(nd);
    const A dust = A(Ph.m_d) * L, gas = A(Ph.m_g) * N;
    const A eps = dust / gas;
    const A tst = harmonic ? L / st : st / L;
    const A rt = tau / tst;
    const A den = one + rt * (one + eps);
    const A ig = one / (one + rt * eps), id = one / (one + rt);
    bool fits = true;
    if constexpr (kPair) fits = df_drag_fits(tau, st, gas, dust, rt, eps);
    A wn[3] = {zero, zero, zero}, un[3] = {zero, zero, zero}, vn[3] = {zero, zero, zero};
#pragma unroll
    for (int k = 0; k < DIM; ++k) {
        wn[k] = ((sv[k] / N - su[k] / L) + tau * (sa[k] / N)) / den;
        un[k] = su[k] / L + tau * gv[k] + rt * wn[k];
        vn[k] = un[k] + wn[k];
        if constexpr (kPair) fits = fits && df_vel_fits(wn[k], un[k], vn[k], 0x1p60f);
    }
    // sums over the cell's particles of the lambdas reaching u*', v*', ig, id
    A S_un[3] = {zero, zero, zero}, S_vn[3] = {zero, zero, zero}, S_ig = zero, S_id = zero;
    for (uint32_t a = R.gs; a < R.ge; ++a) {
        if (has_frozen && (gid[a] & kFrozenBit)) continue;
        const V4<T> v = gvel[a], ac = acc[a], lx = lgx[a], lv = lgv[a];
        const T vv[3] = {v.x, v.y, v.z}, aa[3] = {ac.x, ac.y, ac.z}, xx[3] = {lx.x, lx.y, lx.z},
                ll[3] = {lv.x, lv.y, lv.z};
#pragma unroll
        for (int k = 0; k < DIM; ++k) {
            const A l = A(ll[k]) + tau * A(xx[k]);
            S_un[k] += (one - ig) * l;
            S_ig += (A(vv[k]) + tau * (A(aa[k]) + gv[k]) - un[k]) * l;
        }
    }
    for (uint32_t j = R.ds; j < R.de; ++j) {
        const V4<T> u = dvel[j], lx = ldx[j], lu = ldu[j];
        const T uu[3] = {u.x, u.y, u.z}, xx[3] = {lx.x, lx.y, lx.z}, ll[3] = {lu.x, lu.y, lu.z};
#pragma unroll
        for (int k = 0; k < DIM; ++k) {
            const A l = A(ll[k]) + tau * A(xx[k]);
            S_vn[k] += (one - id) * l;
            S_id += (A(uu[k]) + tau * gv[k] - vn[k]) * l;
        }
    }
    A l_rt = zero, l_den = zero;
#pragma unroll
    for (int k = 0; k < DIM; ++k) {
        const A l_vn = S_vn[k];
        const A l_un = S_un[k] + l_vn;
        const A l_wn = l_vn + rt * l_un;
        l_rt += wn[k] * l_un;
        const A l_w = l_wn / den;
        l_den -= wn[k] * l_wn / den;
        O.lv[k] = T(l_w / N);               // lambda of vbar, per gas particle
        O.lA[k] = T(tau * l_wn / den / N);  // lambda of Abar, per gas particle
        O.lu[k] = T((l_un - l_w) / L);      // lambda of ubar, per dust particle
        if constexpr (kPair)
            fits = fits && !df_small(l_vn) && !df_small(l_un) && !df_small(l_wn) && df_in(l_un, -0x1p60f, 0x1p60f) &&
                   df_in(l_wn, -0x1p60f, 0x1p60f);
    }
    l_rt += (one + eps) * l_den;
    l_rt -= eps * ig * ig * S_ig;
    l_rt -= id * id * S_id;
    const A lt = -(rt / tst) * l_rt;
    if constexpr (kPair)
        fits = fits && !df_small(S_ig) && !df_small(S_id) && !df_small(l_rt) && df_in(l_rt, -0x1p60f, 0x1p60f) &&
               df_in(lt, -0x1p100f, 0x1p100f);
    O.lt = T(lt);  // lambda of t*
    O.ig = T(ig);
    O.id = T(id);
    O.tst = T(tst);
    O.L = T(L);
    return fits ? 1 : 2;
}

// Its binary64 form for the cells outside df's range, out of line.
template <class T, int DIM>
__device__ __noinline__ int cell_adjoint_wide(const Phys<T> Ph, const StepVals S, int harmonic, int has_frozen,
                                              const V4<T> *__restrict__ gvel, const uint32_t *__restrict__ gid,
                                              const V4<T> *__restrict__ acc, const V4<T> *__restrict__ dvel,
                                              const V4<T> *__restrict__ lgx, const V4<T> *lgv,
                                              const V4<T> *__restrict__ ldx, const V4<T> *ldu, const CellRange R,
                                              CellLam<T> *O)
{
    return cell_adjoint_solve<T, double, DIM>(Ph, S, harmonic, has_frozen, gvel, gid, acc, dvel, lgx, lgv, ldx, ldu, R,
                                              *O);
}

// The same by four consecutive lanes, lane k on component k and lane 3 on the
// stopping times (df only; a sum over the components is added up at the end,
// which two-float sums leave far below the rounding of the results). Lane k
// returns its component in lv, lA, lu; the scalars come back in every lane.
template <class T, int DIM>
__device__ __forceinline__ int cell_adjoint_lanes(const Phys<T> &Ph, const StepVals &S, int harmonic, int has_frozen,
                                                  const V4<T> *__restrict__ gvel, const uint32_t *__restrict__ gid,
                                                  const V4<T> *__restrict__ acc, const V4<T> *__restrict__ dvel,
                                                  const V4<T> *__restrict__ lgx, const V4<T> *lgv,
                                                  const V4<T> *__restrict__ ldx, const V4<T> *ldu, const CellRange &R,
                                                  unsigned mask, CellLam<T> &O)
{
    const int k = threadIdx.x & 3;
    const bool axis = k < DIM, last = k == 3;
    const df one = df(1.0f), zero = df(0.0f);
    const df tau = S.tau;
    const df g = k == 0 ? S.g[0] : (k == 1 ? S.g[1] : S.g[2]);
    auto at = [k](const V4<T> *p, uint32_t a) { return reinterpret_cast<const T *>(p + a)[k]; };
    uint32_t ng = 0;
    const uint32_t nd = R.de - R.ds;
    df sv = zero, sa = zero, su = zero;
#pragma unroll 2
    for (uint32_t a = R.gs; a < R.ge; ++a) {
        if (has_frozen && (gid[a] & kFrozenBit)) continue;
        ++ng;
        sv += at(gvel, a);
        sa += at(acc, a);
    }
#pragma unroll 2
    for (uint32_t j = R.ds; j < R.de; ++j) {
        const T u = at(dvel, j);
        if (harmonic && last) su += one / df(u);
        else su += u;
    }
    if (ng == 0 || nd == 0) return 0;
    const df st = lane_value(mask, su, (threadIdx.x & 31) | 3);
    const df N = df(ng), L = df(nd);
    const df dust = df(Ph.m_d) * L, gas = df(Ph.m_g) * N;
    const df eps = dust / gas;
    const df tst = harmonic ? L / st : st / L;
    const df rt = tau / tst;
    const df den = one + rt * (one + eps);
    const df ig = one / (one + rt * eps), id = one / (one + rt);
    bool fits = df_drag_fits(tau, st, gas, dust, rt, eps);
    df wn = zero, un = zero, vn = zero, S_un = zero, S_vn = zero, S_ig = zero, S_id = zero;
    if (axis) {
        wn = ((sv / N - su / L) + tau * (sa / N)) / den;
        un = su / L + tau * g + rt * wn;
        vn = un + wn;
        fits = fits && df_vel_fits(wn, un, vn, 0x1p60f);
        for (uint32_t a = R.gs; a < R.ge; ++a) {
            if (has_frozen && (gid[a] & kFrozenBit)) continue;
            const df l = df(at(lgv, a)) + tau * df(at(lgx, a));
            S_un += (one - ig) * l;
            S_ig += (df(at(gvel, a)) + tau * (df(at(acc, a)) + g) - un) * l;
        }
        for (uint32_t j = R.ds; j < R.de; ++j) {
            const df l = df(at(ldu, j)) + tau * df(at(ldx, j));
            S_vn += (one - id) * l;
            S_id += (df(at(dvel, j)) + tau * g - vn) * l;
        }
    }
    const df l_un = S_un + S_vn;
    const df l_wn = S_vn + rt * l_un;
    const df l_w = l_wn / den;
    O.lv[0] = T(l_w / N);               // lambda of vbar, per gas particle
    O.lA[0] = T(tau * l_wn / den / N);  // lambda of Abar, per gas particle
    O.lu[0] = T((l_un - l_w) / L);      // lambda of ubar, per dust particle
    fits = fits && !df_small(S_vn) && !df_small(l_un) && !df_small(l_wn) && df_in(l_un, -0x1p60f, 0x1p60f) &&
           df_in(l_wn, -0x1p60f, 0x1p60f);
    // over the components (lanes without one hold zeros)
    df l_rt = wn * l_un, l_den = -(wn * l_wn / den);
#pragma unroll
    for (int o = 1; o < 4; o <<= 1) {
        const int other = (threadIdx.x & 31) ^ o;
        l_rt += lane_value(mask, l_rt, other);
        l_den += lane_value(mask, l_den, other);
        S_ig += lane_value(mask, S_ig, other);
        S_id += lane_value(mask, S_id, other);
    }
    l_rt += (one + eps) * l_den;
    l_rt -= eps * ig * ig * S_ig;
    l_rt -= id * id * S_id;
    const df lt = -(rt / tst) * l_rt;
    fits = fits && !df_small(S_ig) && !df_small(S_id) && !df_small(l_rt) && df_in(l_rt, -0x1p60f, 0x1p60f) &&
           df_in(lt, -0x1p100f, 0x1p100f);
    O.lt = T(lt);  // lambda of t*
    O.ig = T(ig);
    O.id = T(id);
    O.tst = T(tst);
    O.L = T(L);
    return __all_sync(mask, fits) ? 1 : 2;
}

// LANES: as in the cell update (4 with df only).
template <class T, class A, int DIM, int LANES>
__global__ void __launch_bounds__(kCellsPerCta)
k_cell_adjoint(Geo<T> G, Phys<T> Ph, StepVals S, int harmonic, int has_frozen,
               const V4<T> *__restrict__ gvel, const uint32_t *__restrict__ gid, const uint32_t *__restrict__ gstart,
               const V4<T> *__restrict__ acc, const V4<T> *__restrict__ gpos, const V4<T> *__restrict__ dvel,
               const V4<T> *__restrict__ dpos, const uint32_t *__restrict__ dstart, const V4<T> *__restrict__ lgx,
               V4<T> *lgv, const V4<T> *__restrict__ ldx, V4<T> *ldu, V4<T> *__restrict__ lA, T *__restrict__ lts)
{
    __shared__ T s_ig[kCellsPerCta], s_id[kCellsPerCta], s_lt[kCellsPerCta], s_tst[kCellsPerCta], s_L[kCellsPerCta];
    __shared__ T s_lv[3][kCellsPerCta], s_lA[3][kCellsPerCta], s_lu[3][kCellsPerCta];
    __shared__ int s_drag[kCellsPerCta];

    const uint32_t ncells = G.ncells;
    const uint32_t cpc = kCellsPerCta / LANES;
    const uint32_t c0 = blockIdx.x * cpc;
    const uint32_t lc0 = threadIdx.x / LANES;
    const uint32_t c = c0 + lc0;
    int drag = 0;
    if (c < ncells) {
        const CellRange R{gstart[c], gstart[c + 1], dstart[c], dstart[c + 1]};
        CellLam<T> O;
        const int k = threadIdx.x & 3;
        bool all = LANES == 1;  // this thread holds every component
        if constexpr (LANES == 1)
            drag = cell_adjoint_solve<T, A, DIM>(Ph, S, harmonic, has_frozen, gvel, gid, acc, dvel, lgx, lgv, ldx, ldu,
                                                 R, O);
        else
            drag = cell_adjoint_lanes<T, DIM>(Ph, S, harmonic, has_frozen, gvel, gid, acc, dvel, lgx, lgv, ldx, ldu, R,
                                              0xfu << (threadIdx.x & 28), O);
        if constexpr (std::is_same<A, df>::value) {
            if (drag == 2 && (LANES == 1 || k == 0)) {
                CellLam<T> W;
                cell_adjoint_wide<T, DIM>(Ph, S, harmonic, has_frozen, gvel, gid, acc, dvel, lgx, lgv, ldx, ldu, R, &W);
                O = W;
                all = true;
            }
        }
        if (drag && all) {
#pragma unroll
            for (int m = 0; m < DIM; ++m) {
                s_lv[m][lc0] = O.lv[m];
                s_lA[m][lc0] = O.lA[m];
                s_lu[m][lc0] = O.lu[m];
            }
        } else if (drag == 1 && k < DIM) {
            s_lv[k][lc0] = O.lv[0];
            s_lA[k][lc0] = O.lA[0];
            s_lu[k][lc0] = O.lu[0];
        }
        if (drag && (LANES == 1 || k == 0)) {
            s_lt[lc0] = O.lt;
            s_ig[lc0] = O.ig;
            s_id[lc0] = O.id;
            s_tst[lc0] = O.tst;
            s_L[lc0] = O.L;
        }
    }
    if (LANES == 1 || (threadIdx.x & 3) == 0) s_drag[lc0] = drag;
    __syncthreads();

    const uint32_t c1 = min(c0 + cpc, ncells);
    const T tau_t = step_val<T>(S.tau, S.dtau);
    for (uint32_t a = gstart[c0] + threadIdx.x; a < gstart[c1]; a += blockDim.x) {
        V4<T> la;
        la.x = la.y = la.z = la.w = T(0);
        if (has_frozen && (gid[a] & kFrozenBit)) {
            lA[a] = la;
            continue;
        }
        const V4<T> p = gpos[a], lx = lgx[a];
        V4<T> lv = lgv[a];
        lv.x += tau_t * lx.x;
        lv.y += tau_t * lx.y;
        lv.z += tau_t * lx.z;
        const uint32_t lc = cell_key<T, DIM>(G, p.x, p.y, p.z) - c0;
        if (lc < cpc && s_drag[lc]) {
            const T ig = s_ig[lc];
            la.x = tau_t * ig * lv.x + s_lA[0][lc];
            lv.x = ig * lv.x + s_lv[0][lc];
            if (DIM > 1) { la.y = tau_t * ig * lv.y + s_lA[1][lc]; lv.y = ig * lv.y + s_lv[1][lc]; }
            if (DIM > 2) { la.z = tau_t * ig * lv.z + s_lA[2][lc]; lv.z = ig * lv.z + s_lv[2][lc]; }
        } else {
            la.x = tau_t * lv.x;
            la.y = tau_t * lv.y;
            la.z = tau_t * lv.z;
        }
        lv.w = T(0);
        lA[a] = la;
        lgv[a] = lv;
    }
    for (uint32_t j = dstart[c0] + threadIdx.x; j < dstart[c1]; j += blockDim.x) {
        const V4<T> p = dpos[j], lx = ldx[j];
        V4<T> lu = ldu[j];
        lu.x += tau_t * lx.x;
        lu.y += tau_t * lx.y;
        lu.z += tau_t * lx.z;
        const uint32_t lc = cell_key<T, DIM>(G, p.x, p.y, p.z) - c0;
        if (lc < cpc && s_drag[lc]) {
            const T id = s_id[lc];
            lu.x = id * lu.x + s_lu[0][lc];
            if (DIM > 1) lu.y = id * lu.y + s_lu[1][lc];
            if (DIM > 2) lu.z = id * lu.z + s_lu[2][lc];
            // dt*/dt_j: 1/L (arithmetic mean) or t*^2 / (L t_j^2) (harmonic mean)
            const T tj = dvel[j].w;
            const T dtdt = harmonic ? s_tst[lc] * s_tst[lc] / (s_L[lc] * tj * tj) : T(1) / s_L[lc];
            lts[j] += s_lt[lc] * dtdt;
        }
        lu.w = T(0);
        ldu[j] = lu;
    }
}

template <class T, class A, int DIM>
cudaError_t cell_adjoint_t(const LaunchCtx &L, const void *geo, const void *phys, PhaseBufs &G, PhaseBufs &D,
                           const void *acc, const StepArgs &S, const void *lgx, void *lgv, const void *ldx, void *ldu,
                           void *lA, void *lts)
{
    const Geo<T> &Gg = *static_cast<const Geo<T> *>(geo);
    const Phys<T> &Ph = *static_cast<const Phys<T> *>(phys);
    // four lanes per cell where cells hold several particles (see the update):
    // 512^2 column 62 -> 44 us
    bool lanes = false;
    auto kern = k_cell_adjoint<T, A, DIM, 1>;
    if constexpr (std::is_same<A, df>::value) {
        lanes = (double)std::max(G.n, D.n) >= 1.5 * (double)Gg.ncells;
        if (lanes) kern = k_cell_adjoint<T, A, DIM, 4>;
    }
    const uint32_t cpc = kCellsPerCta / (lanes ? 4 : 1);
    const uint32_t blocks = (Gg.ncells + cpc - 1) / cpc;
    kern<<<blocks, kCellsPerCta, 0, L.stream>>>(
        Gg, Ph, step_vals(S.tau, S.g), S.tstar_mode == TFSPH_TSTAR_HARMONIC, S.has_frozen,
        static_cast<const V4<T> *>(G.vel[G.cur]), G.id[G.cur], G.start, static_cast<const V4<T> *>(acc),
        static_cast<const V4<T> *>(G.pos[G.cur]), static_cast<const V4<T> *>(D.vel[D.cur]),
        static_cast<const V4<T> *>(D.pos[D.cur]), D.start, static_cast<const V4<T> *>(lgx), static_cast<V4<T> *>(lgv),
        static_cast<const V4<T> *>(ldx), static_cast<V4<T> *>(ldu), static_cast<V4<T> *>(lA), static_cast<T *>(lts));
    return cudaGetLastError();
}

template <class T, class A>
cudaError_t cell_adjoint_dim(const LaunchCtx &L, const void *geo, const void *phys, PhaseBufs &G, PhaseBufs &D,
                             const void *acc, const StepArgs &S, const void *lgx, void *lgv, const void *ldx, void *ldu,
                             void *lA, void *lts)
{
    switch (L.dim) {
        case 1: return cell_adjoint_t<T, A, 1>(L, geo, phys, G, D, acc, S, lgx, lgv, ldx, ldu, lA, lts);
        case 2: return cell_adjoint_t<T, A, 2>(L, geo, phys, G, D, acc, S, lgx, lgv, ldx, ldu, lA, lts);
        default: return cell_adjoint_t<T, A, 3>(L, geo, phys, G, D, acc, S, lgx, lgv, ldx, ldu, lA, lts);
    }
}

template <class T, class A, int DIM>
cudaError_t cell_update_t(const LaunchCtx &L, const void *geo, const void *phys, PhaseBufs &G, PhaseBufs &D,
                          const void *acc, const StepArgs &S)
{
    const Geo<T> &Gg = *static_cast<const Geo<T> *>(geo);
    const Phys<T> &Ph = *static_cast<const Phys<T> *>(phys);
    bool est = true;
    for (int d = 0; d < DIM; ++d) est = est && Gg.est_exact[d];
    // Four lanes per cell where cells hold several particles of a phase; with
    // binary64 sums only while the chip is not full of warps anyway (the lanes
    // repeat the scalar part of the solve on the 2-lane pipe).
    // Fewer cells per CTA, down to one warp, until every SM has two CTAs.
    const double mean = (double)std::max(G.n, D.n) / (double)Gg.ncells;
    const bool lanes = mean >= 1.5 && (sizeof(A) == 4 || std::is_same<A, df>::value || Gg.ncells < 4096u);
    const int per = lanes ? 4 : 1;
    int threads = kCellsPerCta;
    while (threads > 32 && (int64_t)Gg.ncells * per < (int64_t)threads * 2 * kSmCount) threads /= 2;
    const uint32_t cpc = (uint32_t)(threads / per);
    const uint32_t blocks = (Gg.ncells + cpc - 1) / cpc;
    auto kern = lanes ? (est ? k_cell_update<T, A, DIM, true, 4> : k_cell_update<T, A, DIM, false, 4>)
                      : (est ? k_cell_update<T, A, DIM, true, 1> : k_cell_update<T, A, DIM, false, 1>);
    kern<<<blocks, threads, 0, L.stream>>>(
        Gg, Ph, step_vals(S.tau, S.g), S.tstar_mode == TFSPH_TSTAR_HARMONIC, S.has_frozen,
        Ph.eos == TFSPH_EOS_ADIABATIC, static_cast<V4<T> *>(G.pos[G.cur]), static_cast<V4<T> *>(G.vel[G.cur]),
        G.id[G.cur], G.key, G.start, static_cast<const V4<T> *>(acc), static_cast<V4<T> *>(D.pos[D.cur]),
        static_cast<V4<T> *>(D.vel[D.cur]), D.key, D.start);
    return cudaGetLastError();
}

template <class T, class A>
cudaError_t cell_update_dim(const LaunchCtx &L, const void *geo, const void *phys, PhaseBufs &G, PhaseBufs &D,
                            const void *acc, const StepArgs &S)
{
    switch (L.dim) {
        case 1: return cell_update_t<T, A, 1>(L, geo, phys, G, D, acc, S);
        case 2: return cell_update_t<T, A, 2>(L, geo, phys, G, D, acc, S);
        default: return cell_update_t<T, A, 3>(L, geo, phys, G, D, acc, S);
    }
}

}  // namespace

cudaError_t launch_cell_adjoint(const LaunchCtx &L, const void *geo, const void *phys, PhaseBufs &G, PhaseBufs &D,
                                const void *acc, const StepArgs &S, const void *lgx, void *lgv, const void *ldx,
                                void *ldu, void *lA, void *lts)
{
    if (L.precision == TFSPH_FP64)
        return cell_adjoint_dim<double, double>(L, geo, phys, G, D, acc, S, lgx, lgv, ldx, ldu, lA, lts);
    if (S.cell_acc == TFSPH_CELL_ACC_FP64)
        return cell_adjoint_dim<float, df>(L, geo, phys, G, D, acc, S, lgx, lgv, ldx, ldu, lA, lts);
    return cell_adjoint_dim<float, float>(L, geo, phys, G, D, acc, S, lgx, lgv, ldx, ldu, lA, lts);
}

cudaError_t launch_cell_update(const LaunchCtx &L, const void *geo, const void *phys, PhaseBufs &G,
                               PhaseBufs &D, const void *acc, const StepArgs &S)
{
    if (L.precision == TFSPH_FP64) return cell_update_dim<double, double>(L, geo, phys, G, D, acc, S);
    if (S.cell_acc == TFSPH_CELL_ACC_FP64) return cell_update_dim<float, df>(L, geo, phys, G, D, acc, S);
    return cell_update_dim<float, float>(L, geo, phys, G, D, acc, S);
}

}  // namespace tfsph
