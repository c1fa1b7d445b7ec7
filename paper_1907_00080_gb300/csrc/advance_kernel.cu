// Interpolation, kinematic advance and bond kinetics in one kernel.
//
// One block of a.adv_threads (<= kAdvThreads) threads per unit: a chunk of up to kChunkV vertices
// of a kinematic membrane or a deformable dynamic particle, or a whole
// rigid-projected membrane or rigid dynamic particle (one vertex per thread;
// the velocities of the former are first projected on their least-squares
// rigid motion, the latter follows Newton-Euler).  Per vertex: interpolate
// u^n (Sec. 2.3), advance with Eq. kinematicPos (BDF2; forward Euler on the
// first step), refresh the repulsion boxes.  Then the ligands whose element
// starts in the unit are decided at X^{n+1} (bond_logic.cuh); a chunk whose
// last element ends in the ring's next chunk advances that one vertex too.
//
// The decisions are applied by the next force kernel (settle_bonds).  A last
// block that decided the elements across chunks and applied everything, as
// this kernel had before, was a third of its time: 6100 of 18000 cycles on the
// 640 x 160 capillary (a device-wide fence and an arrival counter, then two
// more rounds to L2).
#include "marker_common.cuh"

namespace lbib {

constexpr int kAdvThreads = 4 * kChunkV;  // most threads per unit: one vertex each of a rigid ring (<= 256)
constexpr int kMaxPairs = 512;  // (ligand, receptor) formation candidates staged per block

// receptor position p of the cell-ordered array
template <typename C>
__device__ __forceinline__ typename Ext<C>::E ehi_pos_x(const MarkerArgs& a, int p) {
    typename Ext<C>::E x, y;
    PosIO<C>::load(a.rcell_pos, p, x, y);
    return x;
}
template <typename C>
__device__ __forceinline__ typename Ext<C>::E ehi_pos_y(const MarkerArgs& a, int p) {
    typename Ext<C>::E x, y;
    PosIO<C>::load(a.rcell_pos, p, x, y);
    return y;
}

// Eqs. verletPos / verletVel of a deformable dynamic particle: the vertex moves
// by the interpolated velocity (the first tentative velocity) plus F / (2 m_v)
// (F the total force of this step, m_v = rho_P A_0 / n); its velocity is the
// backward difference 3/2 (x^{n+1} - x^n) - 1/2 (x^n - x^{n-1}) (first-order on
// the first step)
template <typename C>
__device__ __forceinline__ void verlet(const MarkerArgs& a, int m, int v, typename Ext<C>::E x,
                                       typename Ext<C>::E y, typename Ext<C>::E xp, typename Ext<C>::E yp,
                                       C Ux, C Uy, long long step, bool store_v, typename Ext<C>::E& xn,
                                       typename Ext<C>::E& yn) {
    const C* F = static_cast<const C*>(a.F);
    C* V = static_cast<C*>(a.V);
    const C mv = C(a.mem_dyn[3 * m + 2]);
    xn = eaddc(x, Ux + (C(0.5) * F[2 * (size_t)v]) / mv);
    yn = eaddc(y, Uy + (C(0.5) * F[2 * (size_t)v + 1]) / mv);
    if (!store_v) return;
    if (step == 0) {
        V[2 * (size_t)v] = etoc(esub(xn, x));
        V[2 * (size_t)v + 1] = etoc(esub(yn, y));
    } else {
        V[2 * (size_t)v] = C(1.5) * etoc(esub(xn, x)) - C(0.5) * etoc(esub(x, xp));
        V[2 * (size_t)v + 1] = C(1.5) * etoc(esub(yn, y)) - C(0.5) * etoc(esub(y, yp));
    }
}

// DYN: the context holds dynamic particles (without them their paths are not
// compiled into the kernel, which keeps its code small)
//
// advance_unit is the body for advance unit `u` of the context `a`: the
// single-context kernel runs unit blockIdx.x, the batched kernel (ensembles)
// one unit of one member per block.
//
// Everything but the velocities is read before dep_wait(): the positions,
// forces, weights and bonds were complete when the fused kernel (the
// predecessor in a chained launch) let this one start.  What needs no velocity
// is also done before it: the rigid projection's position sums, and all of a
// rigid dynamic particle, bond decisions included (the fused kernel touches
// nothing that is written here).  The kinds share one path but for what is
// their own, which keeps the instructions that a step has to fetch anew few.
template <typename C, bool DYN>
__device__ __forceinline__ void advance_unit(const MarkerArgs& a, int u) {
    using E = typename Ext<C>::E;
    const int4 u0 = a.au[3 * u], u1 = a.au[3 * u + 1], u2 = a.au[3 * u + 2];
    const int m = u0.x, k0 = u0.y, kn = u0.z, off = u0.w, n = u1.x, kind = u1.y;
    const int tid = threadIdx.x, lane = tid & 31;
    const bool body = DYN && kind == LBIB_MEMBRANE_DYNAMIC_RIGID;
    __shared__ E s_x[kAdvThreads], s_y[kAdvThreads];
    __shared__ C cred[3][4][8];
    __shared__ int s_np;  // formation candidates listed
    if (tid == 0) s_np = 0;
    const long long step = *a.d_step;
    C* U = static_cast<C*>(a.U);
    // the unit's ligand records and current bonds, fetched now so that their
    // latency overlaps the marker advance (a unit has at most one ligand per thread)
    const int lq0 = u1.z;
    const int nlq = a.nrec > 0 ? u1.w : 0;
    int4 my_rec = make_int4(-1, 0, 0, 0);
    int my_bond = -1;
    if (tid < nlq) {
        my_rec = a.au_ligs[lq0 + tid];
        my_bond = a.bond_of_lig[my_rec.x];
    }

    // ---- one vertex per thread, and one thread for the next chunk's first
    // vertex, where this unit's ligands may need it: read from the halo records,
    // nothing stored
    const bool mine = tid < kn;
    const bool next = tid == kn && nlq > 0 && kn < n;
    const bool wraps = k0 + kn == n;
    const int v = off + (mine ? k0 + tid : (next && !wraps ? k0 + kn : (next ? 0 : k0)));
    E x, y, xp, yp, xn, yn, cax, cay;
    if (n > kDirectArea) PosIO<C>::load(a.halo, 2 * (u - k0 / kChunkV), cax, cay);  // X^n of vertex 0
    if (next) {
        const int un = wraps ? u - k0 / kChunkV : u + 1;
        PosIO<C>::load(a.halo, 2 * un, x, y);
        PosIO<C>::load(a.halo, 2 * un + 1, xp, yp);
    } else {
        load_pos<C>(a, v, x, y);
        PosIO<C>::load(a.Xp, v, xp, yp);
    }
    const Shape<C> sh = load_shape<C>(a, v);
    C Ux = 0, Uy = 0;
    if (body) {
        // a rigid dynamic particle, the whole ring in this block: Eqs.
        // linearVelRig / angularVelRig.  F and its moment M about the area
        // centroid give du/dt = F/m, domega/dt = M/I; the body translates by u
        // and turns by omega about its centroid (cos omega - 1 = -2 sin^2(omega/2))
        E xr, yr, xq, yq;
        load_pos<C>(a, off, xr, yr);
        load_pos<C>(a, v + 1 == off + n ? off : v + 1, xq, yq);
        const C* F = static_cast<const C*>(a.F);
        const C fx = mine ? F[2 * (size_t)v] : C(0), fy = mine ? F[2 * (size_t)v + 1] : C(0);
        const C ax = mine ? etoc(esub(x, xr)) : C(0), ay = mine ? etoc(esub(y, yr)) : C(0);
        const C bx = mine ? etoc(esub(xq, xr)) : C(0), by = mine ? etoc(esub(yq, yr)) : C(0);
        // area centroid relative to vertex 0 from the triangles (vertex 0, k, k+1)
        const C cr = ax * by - ay * bx;
        C s3[3] = {cr, cr * (ax + bx), cr * (ay + by)};
        block_sum_c<C, 3>(s3, cred[0]);
        const C gx = s3[1] / (C(3) * s3[0]), gy = s3[2] / (C(3) * s3[0]);
        const C rx = ax - gx, ry = ay - gy;
        C f3[3] = {fx, fy, mine ? rx * fy - ry * fx : C(0)};
        block_sum_c<C, 3>(f3, cred[1]);
        // the rigid state in FP64, one component a lane of the first warp (done
        // by every warp, these operations took most of the kernel: 9000 of 20000
        // cycles for a 210-vertex carrier)
        __shared__ C s_rb[5];
        if (tid < 3) {
            double* rb = a.rb + 6 * m;
            const int now = tid < 2 ? tid : 4, before = tid < 2 ? tid + 2 : 5;
            const double s0 = rb[now], sp = rb[before];
            const double acc = double(tid == 0 ? f3[0] : (tid == 1 ? f3[1] : f3[2])) / a.mem_dyn[3 * m + (tid < 2 ? 0 : 1)];
            const double sn = step == 0 ? s0 + acc : (2.0 / 3.0) * (2.0 * s0 - 0.5 * sp + acc);
            rb[before] = s0;
            rb[now] = sn;
            s_rb[tid] = C(sn);
            if (tid == 2) {
                const C hs = sin(C(0.5) * C(sn));
                s_rb[3] = C(-2) * hs * hs;
                s_rb[4] = sin(C(sn));
            }
        }
        __syncthreads();
        const C un = s_rb[0], vn = s_rb[1], wn = s_rb[2], c1 = s_rb[3], sn = s_rb[4];
        const C drx = c1 * rx - sn * ry, dry = sn * rx + c1 * ry;
        xn = eaddc(x, un + drx);
        yn = eaddc(y, vn + dry);
        if (mine) {
            C* V = static_cast<C*>(a.V);
            V[2 * (size_t)v] = un - wn * (ry + dry);
            V[2 * (size_t)v + 1] = vn + wn * (rx + drx);
        }
    } else {
        // rigid projection (the whole ring in this block): positions about their
        // mean, from vertex 0
        const bool project = kind == LBIB_MEMBRANE_RIGID_PROJECTED;
        const C inv_n = C(1) / C(n);
        C rx = 0, ry = 0, den = 0;
        if (project) {
            E xr, yr;
            load_pos<C>(a, off, xr, yr);
            const C dx = etoc(esub(x, xr)), dy = etoc(esub(y, yr));
            C p2[2] = {mine ? dx : C(0), mine ? dy : C(0)};
            block_sum_c<C, 2>(p2, cred[0]);
            rx = dx - p2[0] * inv_n;
            ry = dy - p2[1] * inv_n;
        }
        dep_wait();
        dep_trigger();
        interp_vertex<C>(a, sh, Ux, Uy);
        if (project) {
            // least-squares rigid motion U_c + omega x (x - x_c)
            C u2s[2] = {mine ? Ux : C(0), mine ? Uy : C(0)};
            block_sum_c<C, 2>(u2s, cred[1]);
            const C mu = u2s[0] * inv_n, mv = u2s[1] * inv_n;
            C q2[2] = {mine ? rx * (Uy - mv) - ry * (Ux - mu) : C(0), mine ? rx * rx + ry * ry : C(0)};
            block_sum_c<C, 2>(q2, cred[2]);
            const C om = q2[0] / q2[1];
            Ux = mu - om * ry;
            Uy = mv + om * rx;
        }
        if (DYN && kind == LBIB_MEMBRANE_DYNAMIC) {
            verlet<C>(a, m, v, x, y, xp, yp, Ux, Uy, step, mine, xn, yn);
        } else {
            bdf2<C>(x, xp, Ux, step, xn);
            bdf2<C>(y, yp, Uy, step, yn);
        }
        if (mine) {
            U[2 * v] = Ux;
            U[2 * v + 1] = Uy;
        }
    }
    if (mine) {
        if (!isfinite(ehi(xn)) || !isfinite(ehi(yn))) atomicOr(a.status, ST_NONFINITE);
        PosIO<C>::store(a.Xp, v, x, y);
        PosIO<C>::store(a.X, v, xn, yn);
    }
    s_x[tid] = xn;
    s_y[tid] = yn;
    {
        // boxes of the unit's repulsion segments (units are segment-aligned); lanes
        // past a segment's end take its first vertex
        const int gfirst = tid & ~(kSegV - 1);
        const int sg = gfirst < kn ? u2.x + (k0 + gfirst) / kSegV : -1;
        const int gr = (tid & ~(kGroupV - 1)) < kn ? u2.y + (k0 + tid) / kGroupV : -1;
        E gx, gy;
        shfl_e(gx, xn, lane & ~(kSegV - 1));
        shfl_e(gy, yn, lane & ~(kSegV - 1));
        seg_box_regs<C>(a, sg, gr, lane, mine ? xn : gx, mine ? yn : gy);
    }
    __syncthreads();
    if (n > kDirectArea && tid < 32) {
        // the chunk's share of the ring's area at the new positions, by the first warp
        const E part = chunk_area<C>(kn, lane, cax, cay, [&](int k, E& px, E& py) {
            px = s_x[k];
            py = s_y[k];
        });
        if (lane == 0) PosIO<C>::store(a.area_part, u, part, part);
    }

    // ---- bond decisions for the ligands whose element starts in this unit.
    // (a) per ligand: rupture test of its bond; a free ligand lists the
    //     receptors of the 3x3 cells around it as (ligand, receptor) pairs;
    // (b) per pair: the formation test; each ligand keeps the lowest passing
    //     receptor id (a minimum: independent of evaluation order);
    // (c) per ligand that is free after (a): claim its receptor.
    // Receptors have to be free at the start of the step.
    if (nlq > 0) {
        __shared__ int s_pl[kMaxPairs], s_pr[kMaxPairs];
        __shared__ int s_best[kAdvThreads];
        __shared__ int4 s_lig[kAdvThreads];
        const int l = my_rec.x;  // a unit has no more ligands than threads
        bool look = false;
        if (tid < nlq) {
            LigandPoint<C> lp;
            lp.init(s_x[my_rec.y], s_y[my_rec.y], s_x[my_rec.z], s_y[my_rec.z]);
            s_lig[tid] = my_rec;
            s_best[tid] = INT_MAX;
            look = lp.finite();  // non-finite positions: reported above
            if (look && my_bond >= 0) {
                look = ruptures<C>(a, lp, step, l, my_bond);
                if (look) a.rupt[l] = my_bond;
            }
            if (look && receptors_in_reach<C>(a, lp)) {
                int p0[9], p1[9];
                ligand_cells<C>(a, lp, p0, p1);
                // every receptor of the cells becomes a pair; whether it was free at
                // the start of the step is checked per pair, in parallel
#pragma unroll
                for (int c = 0; c < 9; ++c) {
                    for (int p = p0[c]; p < p1[c]; ++p) {
                        const int slot = atomicAdd(&s_np, 1);
                        if (slot < kMaxPairs) {
                            s_pl[slot] = tid;
                            s_pr[slot] = p;
                        } else {
                            // list full: decide in place
                            const int rr = a.rcell_ids[p];
                            if (a.owner_cell[p] < 0 && forms<C>(a, lp, step, l, rr, ehi_pos_x<C>(a, p), ehi_pos_y<C>(a, p)))
                                atomicMin(&s_best[tid], rr);
                        }
                    }
                }
            }
        }
        __syncthreads();
        // (often none: no receptor near any of the unit's free ligands)
        const int np = s_np < kMaxPairs ? s_np : kMaxPairs;
        for (int t = tid; t < np; t += blockDim.x) {
            const int q = s_pl[t], p = s_pr[t];
            const int rr = a.rcell_ids[p];
            typename Ext<C>::E rx, ry;
            PosIO<C>::load(a.rcell_pos, p, rx, ry);
            if (a.owner_cell[p] >= 0) continue;  // bound at the start of the step
            const int4 rec = s_lig[q];
            LigandPoint<C> lp;
            lp.init(s_x[rec.y], s_y[rec.y], s_x[rec.z], s_y[rec.z]);
            if (forms<C>(a, lp, step, rec.x, rr, rx, ry)) atomicMin(&s_best[q], rr);
        }
        if (np > 0) __syncthreads();
        if (look && s_best[tid] != INT_MAX) {
            a.cand[l] = s_best[tid];
            atomicMin(&a.claim[s_best[tid]], l);
        }
    }
    if (body) {
        // the flow's velocity at the vertices, for the read-back
        dep_wait();
        dep_trigger();
        if (mine) {
            interp_vertex<C>(a, sh, Ux, Uy);
            U[2 * v] = Ux;
            U[2 * v + 1] = Uy;
        }
    }
}

// (Up to 128 registers, 100 in FP32.  Left to itself ptxas stops at 80, three
// blocks of 256 threads, which a single run's few blocks never are on one SM;
// what it then keeps in flight turned on unrelated edits: 640 x 160 capillary,
// 100 steps from three starts, 1255 / 1095 / 1190 us in one build, 1440 / 1220 /
// 1250 with eight bytes fewer in MarkerArgs, 1116 / 1136 / 1126 now.  Thousands
// of units lose a little by the fewer blocks that fit: 2500 rings, a step 206.5
// -> 207.1 us.)
template <typename C, bool DYN>
__global__ void __launch_bounds__(kAdvThreads, 2) k_advance(const MarkerArgs a) {
    advance_unit<C, DYN>(a, blockIdx.x);
}

// Batched form: the advance units of up to kBatchMax contexts (ensemble
// members) in one launch, one block per (member, unit).  Blocks have the threads of the widest member (idle
// threads beyond a unit's vertices, as in the single-context kernel).
template <typename C, bool DYN>
__global__ void __launch_bounds__(kAdvThreads) k_advance_batch(const __grid_constant__ MarkerBatch b) {
    __shared__ MarkerArgs s_a;
    const int m = marker_member(b, blockIdx.x);
    stage_args(&s_a, b.args + m);
    advance_unit<C, DYN>(s_a, blockIdx.x - b.off[m]);
}

template <typename C>
static auto advance_kernel(bool dyn) {
    return dyn ? k_advance<C, true> : k_advance<C, false>;
}
template <typename C>
static auto advance_batch_kernel(bool dyn) {
    return dyn ? k_advance_batch<C, true> : k_advance_batch<C, false>;
}

cudaError_t launch_advance(lbib_precision prec, const MarkerArgs& a, cudaStream_t s, bool chained) {
    if (a.adv_threads < kChunkV || a.adv_threads > kAdvThreads || a.adv_threads % 32) return cudaErrorInvalidValue;
    return launch_kernel(prec == LBIB_F64 ? advance_kernel<double>(a.has_dyn) : advance_kernel<float>(a.has_dyn), a.nau,
                         a.adv_threads, 0, s, chained, a);
}

cudaError_t launch_advance_batch(lbib_precision prec, bool dyn, const MarkerBatch& b, int threads, cudaStream_t s,
                                 bool chained) {
    if (b.n < 1 || b.n > kBatchMax) return cudaErrorInvalidValue;
    const int nunits = b.off[b.n];
    if (nunits <= 0) return cudaSuccess;
    if (threads < kChunkV || threads > kAdvThreads || threads % 32) return cudaErrorInvalidValue;
    return launch_kernel(prec == LBIB_F64 ? advance_batch_kernel<double>(dyn) : advance_batch_kernel<float>(dyn), nunits,
                         threads, 0, s, chained, b);
}

}  // namespace lbib
