// Ligand-receptor bond kinetics (device logic): rupture, then formation,
// decided with counter-based Philox draws so that the bond history is
// reproducible and independent of thread scheduling.
//
// Paper: Coclite, arXiv 1907.00080, Sec. 2.2 (wall-particle interaction: bonds
// form below a critical separation, a forward probability governs formation
// and a reverse probability governs rupture each step) and Sec. 3 (k_f/k_r0).
// Philox4x64-10: Salmon, Moraes, Dror & Shaw, "Parallel random numbers: as easy
// as 1, 2, 3", SC'11 -- implemented here from that definition.
//
// Decisions are FP64 decisions: an FP32 estimate settles every test whose
// outcome is clear by a relative margin of 1e-5 (the estimates are accurate to
// ~1e-6), and anything closer is recomputed in FP64.
#pragma once

#include <climits>

#include "ext_real.cuh"
#include "lbib_internal.cuh"

namespace lbib {

// a scalar parameter in the compute precision (double field, or its FP32 copy)
template <typename C> __device__ __forceinline__ C par(double d, float f);
template <> __device__ __forceinline__ double par<double>(double d, float) { return d; }
template <> __device__ __forceinline__ float par<float>(double, float f) { return f; }

__device__ __forceinline__ void philox4x64_10(unsigned long long c[4], unsigned long long k0,
                                              unsigned long long k1) {
    const unsigned long long M0 = 0xD2E7470EE14C6C93ULL, M1 = 0xCA5A826395121157ULL;
    const unsigned long long W0 = 0x9E3779B97F4A7C15ULL, W1 = 0xBB67AE8584CAA73BULL;
#pragma unroll 1
    for (int r = 0; r < 10; ++r) {
        if (r > 0) {
            k0 += W0;
            k1 += W1;
        }
        const unsigned long long hi0 = __umul64hi(M0, c[0]), lo0 = M0 * c[0];
        const unsigned long long hi1 = __umul64hi(M1, c[2]), lo1 = M1 * c[2];
        const unsigned long long n0 = hi1 ^ c[1] ^ k0, n2 = hi0 ^ c[3] ^ k1;
        c[0] = n0;
        c[1] = lo1;
        c[2] = n2;
        c[3] = lo0;
    }
}

// the draw of a decision: the top 53 bits k of the first output word; the
// uniform in [0, 1) is k 2^-53
__device__ __forceinline__ unsigned long long bond_draw(const MarkerArgs& a, long long step, int lig, int rec,
                                                        int tag) {
    unsigned long long c[4] = {(unsigned long long)step, (unsigned long long)lig,
                               (unsigned long long)rec, (unsigned long long)tag};
    philox4x64_10(c, a.seed, a.instance);
    return c[0] >> 11;
}
__device__ __forceinline__ double uniform_of(unsigned long long k) { return (double)k * 0x1.0p-53; }
// k 2^-53 < t and k 2^-53 > t for an FP32 threshold t < 2: exact (t 2^53 is a
// scaling by a power of two), without the slow FP64 pipe; neither for NaN
// (0 times an overflow in the FP32 probability: the FP64 one decides)
__device__ __forceinline__ bool draw_below(unsigned long long k, float t) {
    return t > 0.f && k < __float2ull_ru(t * 0x1.0p53f);
}
__device__ __forceinline__ bool draw_above(unsigned long long k, float t) {
    return t < 0.f || (t >= 0.f && k > __float2ull_rd(t * 0x1.0p53f));
}

// forward (formation) and reverse (rupture) probabilities per step, FP64
// (kept out of line: they run only for near ties, and scalars are passed so the
// argument block is never copied)
static __device__ __noinline__ double p_form_d(double d, double y_eq, double inv_y_eq, double kf_dt, double beta_f) {
    const double z = (d - y_eq) * inv_y_eq;
    return 1.0 - exp(-kf_dt * exp(-beta_f * z * z));
}
static __device__ __noinline__ double p_rupture_d(double d, double y_eq, double inv_y_eq, double kr0_dt, double beta_r) {
    const double z = (d - y_eq) * inv_y_eq;
    return 1.0 - exp(-kr0_dt * exp(beta_r * z * z));
}
__device__ __forceinline__ double p_form(const MarkerArgs& a, double d) {
    return p_form_d(d, a.y_eq, a.inv_y_eq, a.kf_dt, a.beta_f);
}
__device__ __forceinline__ double p_rupture(const MarkerArgs& a, double d) {
    return p_rupture_d(d, a.y_eq, a.inv_y_eq, a.kr0_dt, a.beta_r);
}
constexpr float kMargin = 1e-5f;
__device__ __forceinline__ float p_form_f(const MarkerArgs& a, float d) {
    const float z = (d - a.f.y_eq) * a.f.inv_y_eq;
    return 1.0f - expf(-a.f.kf_dt * expf(-a.f.beta_f * z * z));
}
__device__ __forceinline__ float p_rupture_f(const MarkerArgs& a, float d) {
    const float z = (d - a.f.y_eq) * a.f.inv_y_eq;
    return 1.0f - expf(-a.f.kr0_dt * expf(a.f.beta_r * z * z));
}

// ligand point to receptor (rx, ry) in FP64 (periodic minimum image in x, and
// in y without walls)
static __device__ __noinline__ double lig_rec_dist_d(double rx, double ry, double cxp, double cyp, double nx,
                                              double inv_nx, double ny, double inv_ny, int walls) {
    double dx = rx - cxp;
    dx -= nx * floor(dx * inv_nx + 0.5);
    double dy = ry - cyp;
    if (!walls) dy -= ny * floor(dy * inv_ny + 0.5);
    return sqrt(dx * dx + dy * dy);
}
__device__ __forceinline__ double lig_rec_dist(const MarkerArgs& a, double cxp, double cyp, int r) {
    return lig_rec_dist_d(a.rec_xy[2 * r], a.rec_xy[2 * r + 1], cxp, cyp, (double)a.nx, a.inv_nx,
                          (double)a.ny, a.inv_ny, a.walls);
}

// Ligand point (element centroid at X^{n+1}) and its distance to receptor r:
// the estimate in the compute precision, and the FP64 value on demand.
template <typename C>
struct LigandPoint {
    typename Ext<C>::E cx, cy;
    double cxd, cyd;
    bool have_d;
    __device__ void init(typename Ext<C>::E xa, typename Ext<C>::E ya, typename Ext<C>::E xb,
                         typename Ext<C>::E yb) {
        cx = emulc(eadd(xa, xb), C(0.5));
        cy = emulc(eadd(ya, yb), C(0.5));
        have_d = false;
    }
    __device__ bool finite() const { return isfinite(ehi(cx)) && isfinite(ehi(cy)); }
    __device__ C dist_est(const MarkerArgs& a, int r) const {
        typename Ext<C>::E rx, ry;
        PosIO<C>::load(a.rec_e, r, rx, ry);
        return dist_est_at(a, rx, ry);
    }
    __device__ C dist_est_at(const MarkerArgs& a, typename Ext<C>::E rx, typename Ext<C>::E ry) const {
        const C dx = etoc(ewrap(esub(rx, cx), par<C>(a.nx, a.f.nx), par<C>(a.inv_nx, a.f.inv_nx)));
        C dy = etoc(esub(ry, cy));
        if (!a.walls) dy = etoc(ewrap(esub(ry, cy), par<C>(a.ny, a.f.ny), par<C>(a.inv_ny, a.f.inv_ny)));
        return sqrt(dx * dx + dy * dy);
    }
    __device__ double dist(const MarkerArgs& a, int r) {
        if (!have_d) {
            cxd = etod(cx);
            cyd = etod(cy);
            have_d = true;
        }
        return lig_rec_dist(a, cxd, cyd, r);
    }
};

// formation test of ligand l with receptor r at (rx, ry) (tag 0): d < d_cut and u < P_f(d)
template <typename C>
__device__ __forceinline__ bool forms(const MarkerArgs& a, LigandPoint<C>& lp, long long step, int l, int r,
                                      typename Ext<C>::E rx, typename Ext<C>::E ry) {
    if (sizeof(C) == 8) {
        const double d = lp.dist(a, r);
        if (!(d < a.d_cut)) return false;
        return uniform_of(bond_draw(a, step, l, r, 0)) < p_form(a, d);
    }
    const float df = float(lp.dist_est_at(a, rx, ry));
    const float dc = a.f.d_cut;
    if (!(df < dc * (1.f + kMargin))) return false;  // surely beyond the cut-off
    double d = -1.0;
    if (!(df < dc * (1.f - kMargin))) {
        d = lp.dist(a, r);
        if (!(d < a.d_cut)) return false;
    }
    const unsigned long long k = bond_draw(a, step, l, r, 0);
    const float pf = p_form_f(a, df);
    if (draw_below(k, pf - kMargin)) return true;
    if (draw_above(k, pf + kMargin)) return false;
    if (d < 0.0) d = lp.dist(a, r);
    return uniform_of(k) < p_form(a, d);
}

// rupture test of the bond (l, r) (tag 1): d >= d_break or u < P_r(d)
template <typename C>
__device__ __forceinline__ bool ruptures(const MarkerArgs& a, LigandPoint<C>& lp, long long step, int l, int r) {
    if (sizeof(C) == 8) {
        const double d = lp.dist(a, r);
        if (d >= a.d_break) return true;
        return uniform_of(bond_draw(a, step, l, r, 1)) < p_rupture(a, d);
    }
    const float df = float(lp.dist_est(a, r));
    const float db = a.f.d_break;
    double d = -1.0;
    if (df >= db * (1.f + kMargin)) return true;
    if (!(df < db * (1.f - kMargin))) {
        d = lp.dist(a, r);
        if (d >= a.d_break) return true;
    }
    const unsigned long long k = bond_draw(a, step, l, r, 1);
    const float pr = p_rupture_f(a, df);
    if (draw_below(k, pr - kMargin)) return true;
    if (draw_above(k, pr + kMargin)) return false;
    if (d < 0.0) d = lp.dist(a, r);
    return uniform_of(k) < p_rupture(a, d);
}

// false where no receptor can be within the cut-off of the ligand point by its
// height alone
template <typename C>
__device__ __forceinline__ bool receptors_in_reach(const MarkerArgs& a, const LigandPoint<C>& lp) {
    const float y = float(ehi(lp.cy));
    return !(y < a.f.y_reach[0] || (y > a.f.y_reach[1] && y < a.f.y_reach[2]) || y > a.f.y_reach[3]);
}

// 3x3 receptor-grid cells around a ligand point: the nine [p0, p1) ranges of
// the cell-ordered receptor arrays (empty outside the grid's rows)
template <typename C>
__device__ __forceinline__ void ligand_cells(const MarkerArgs& a, const LigandPoint<C>& lp, int p0[9], int p1[9]) {
    const float cxh = float(ehi(lp.cx)), cyh = float(ehi(lp.cy));
    const float xw = cxh - a.f.nx * floorf(cxh * a.f.inv_nx);
    int gx = (int)floorf(xw * a.f.inv_rc_w);
    gx = gx >= a.rc_nx ? a.rc_nx - 1 : (gx < 0 ? 0 : gx);
    const int gy = (int)fminf(fmaxf(floorf((cyh - a.f.rc_y0) * a.f.inv_rc_h), -4.f), float(a.rc_ny) + 4.f);
#pragma unroll
    for (int c = 0; c < 9; ++c) {
        const int qy = gy - 1 + c / 3, qx = gx - 1 + c % 3;
        p0[c] = p1[c] = 0;
        if (qy >= 0 && qy < a.rc_ny) {
            // (qx lies in -1 .. rc_nx)
            const int cell = qy * a.rc_nx + (qx < 0 ? qx + a.rc_nx : (qx >= a.rc_nx ? qx - a.rc_nx : qx));
            p0[c] = a.rcell_start[cell];
            p1[c] = a.rcell_start[cell + 1];
        }
    }
}

// The bonds at the start of this step of the ligands la, lb (-1: none): the
// settled ones, or (the previous step's decisions not yet settled) the previous
// ones changed by them: a won claim binds, else a rupture frees.  Both are
// looked up at once.
__device__ __forceinline__ void bonds_now(const MarkerArgs& a, int la, int lb, bool settled, int& ra, int& rb) {
    const int ia = la < 0 ? 0 : la, ib = lb < 0 ? 0 : lb;
    if (settled) {
        ra = a.bond_of_lig[ia];
        rb = a.bond_of_lig[ib];
    } else {
        ra = a.bond_prev[ia];
        rb = a.bond_prev[ib];
        const int ca = a.cand_prev[ia], cb = a.cand_prev[ib], xa = a.rupt_prev[ia], xb = a.rupt_prev[ib];
        if (xa >= 0) ra = -1;
        if (xb >= 0) rb = -1;
        if (ca >= 0 && a.claim_prev[ca] == ia) ra = ca;
        if (cb >= 0 && a.claim_prev[cb] == ib) rb = cb;
    }
    if (la < 0) ra = -1;
    if (lb < 0) rb = -1;
}

// Settle the decisions of the previous step, all threads of one block: the
// bonds and the step counter of this parity, the receptors' owners (by receptor
// id and in cell order), and this parity's own decisions of two steps ago
// cleared for the coming advance kernel.  A receptor that a rupture frees was
// bound at the start of that step and one that is won was free, so no receptor
// is written twice.
static __device__ __forceinline__ void settle_bonds(const MarkerArgs& a) {
    if (a.nrec > 0) {
        for (int l = threadIdx.x; l < a.nlig; l += blockDim.x) {
            const int b = a.bond_prev[l], c = a.cand_prev[l], r = a.rupt_prev[l], old = a.cand[l];
            const bool won = c >= 0 && a.claim_prev[c] == l;
            if (r >= 0) {
                a.owner[r] = -1;
                a.owner_cell[a.rcell_of_rec[r]] = -1;
            }
            if (won) {
                a.owner[c] = l;
                a.owner_cell[a.rcell_of_rec[c]] = l;
            }
            a.bond_of_lig[l] = won ? c : (r >= 0 ? -1 : b);
            if (old >= 0) a.claim[old] = INT_MAX;
            a.cand[l] = -1;
            a.rupt[l] = -1;
        }
    }
    if (threadIdx.x == 0) *a.d_step = *a.step_prev + 1;
}

}  // namespace lbib
