// Lagrangian-side kernels: membrane forces (stretching, bending, enclosed
// area, repulsion, bond springs), the IB shape functions and the spreading of
// the marker forces; rest state, segment boxes and position conversion.
//
// Paper: Coclite, arXiv 1907.00080, Sec. 2.2 (Eqs. strainFor, bendFor,
// areaFor, repFor, adhFor; MLS exchange), Sec. 2.3 (nine Eulerian points per
// vertex).
//
// Precision: the compute type C is double in FP64 mode and float otherwise;
// positions and every cancellation-prone product use the matching extended
// type E (double, or float-float) from ext_real.cuh.
#include "marker_common.cuh"

namespace lbib {

// ---------------------------------------------------------------- rest state
// Captures, per vertex, the squared and plain rest length of the element
// (v, v+1) and the rest cross/dot products of the two edges at v (which fix the
// rest turning angle theta_0), plus A_0 per membrane -- with the arithmetic the
// force kernel repeats, so the rest shape gives exactly zero force.
template <typename C>
__global__ void k_rest(const MarkerArgs a, void* rest_v, double* A0, double* qa) {
    using E = typename Ext<C>::E;
    const int m = blockIdx.x;
    const int off = a.mem_off[m], n = a.mem_n[m];
    __shared__ E red[4];
    Rest<C>* rest = static_cast<Rest<C>*>(rest_v);
    for (int k = threadIdx.x; k < n; k += blockDim.x) {
        const int v = off + k, L = off + (k == 0 ? n - 1 : k - 1), R = off + (k == n - 1 ? 0 : k + 1);
        E xL, yL, xv, yv, xR, yR;
        load_pos<C>(a, L, xL, yL);
        load_pos<C>(a, v, xv, yv);
        load_pos<C>(a, R, xR, yR);
        const EdgeProducts<C> p = edge_products<E, C>(xL, yL, xv, yv, xR, yR);
        Rest<C> r;
        r.lsq = p.lsqR;
        r.cross = p.cross;
        r.dot = p.dot;
        r.l0 = sqrt(etoc(p.lsqR));
        rest[v] = r;
    }
    if (threadIdx.x < 64) {
        const E A = ring_area<C>(a, off, n, a.mem_au[m], 0, red, 1);
        if (threadIdx.x == 0) {
            const double A0m = etod(A);
            A0[m] = A0m;
            qa[m] = a.mem_ka[m] * (1.0 / 3.0) / A0m;  // k_a p_ref / A_0 (p_ref = 1/3)
        }
    }
}

// ---------------------------------------------------------------- forces
// Eq. adhFor on an element whose ligand is bonded to receptor r (-1: none), half
// to the vertex; positions of the element's two vertices are given
template <typename C, typename E>
__device__ __forceinline__ void bond_on_element(const MarkerArgs& a, int r, E xa, E ya, E xb, E yb, C& Fx, C& Fy) {
    if (r < 0) return;
    E rx, ry;
    PosIO<C>::load(a.rec_e, r, rx, ry);
    // receptor minus ligand point (element centroid)
    const E cx = emulc(eadd(xa, xb), C(0.5)), cy = emulc(eadd(ya, yb), C(0.5));
    const C dx = etoc(ewrap(esub(rx, cx), par<C>(a.nx, a.f.nx), par<C>(a.inv_nx, a.f.inv_nx)));
    C dy = etoc(esub(ry, cy));
    if (!a.walls) dy = etoc(ewrap(esub(ry, cy), par<C>(a.ny, a.f.ny), par<C>(a.inv_ny, a.f.inv_ny)));
    const C d = sqrt(dx * dx + dy * dy);
    const C c = par<C>(a.sigma, a.f.sigma) * (d - par<C>(a.y_eq, a.f.y_eq)) / d;
    Fx += C(0.5) * c * dx;
    Fy += C(0.5) * c * dy;
}

constexpr int kForceThreads = 256;  // threads per force block: eight warps with the roles below
constexpr int kMaxCand = 256;       // repulsion candidate segments per block
constexpr int kStageSeg = 48;       // candidate segments staged in shared memory
constexpr int kScreenIter = 3;      // group boxes per lane loaded ahead of the screen

// Geometry of a vertex from its position and its neighbours': the two edges
// with their squared lengths in the extended type, and for the bending the
// vertex normal (the normalised sum of the outward edge normals, CCW ring) and
// the moment k_b (theta - theta_0) from the rotation between the rest and the
// current edge pair, atan2(c d0 - c0 d, d d0 + c c0): no cancellation of two
// nearly equal angles.
template <typename C, typename E>
struct VertexGeo {
    C mx, my, sL, sR, nx, ny;  // moment times normal, the neighbours' shares, normal
    C eLx, eLy, eRx, eRy, lL, lR;
    E lsqL, lsqR;
};
template <typename C, typename E>
__device__ __forceinline__ VertexGeo<C, E> vertex_geometry(const Rest<C>& r0, C kb, E xL, E yL, E xv, E yv, E xR, E yR) {
    VertexGeo<C, E> g;
    const E dLx = esub(xv, xL), dLy = esub(yv, yL);
    const EdgeProducts<C> p = edge_products<E, C>(xL, yL, xv, yv, xR, yR);
    g.lsqR = p.lsqR;
    g.lsqL = eadd(emul(dLx, dLx), emul(dLy, dLy));
    const E sn = esub(emul(p.cross, r0.dot), emul(r0.cross, p.dot));
    const E cs = eadd(emul(p.dot, r0.dot), emul(p.cross, r0.cross));
    const C dth = atan2(etoc(sn), etoc(cs));
    g.eLx = etoc(dLx);
    g.eLy = etoc(dLy);
    g.eRx = etoc(esub(xR, xv));
    g.eRy = etoc(esub(yR, yv));
    g.lL = sqrt(g.eLx * g.eLx + g.eLy * g.eLy);
    g.lR = sqrt(g.eRx * g.eRx + g.eRy * g.eRy);
    const C iL = C(1) / g.lL, iR = C(1) / g.lR;
    g.nx = g.eLy * iL + g.eRy * iR;
    g.ny = -g.eLx * iL - g.eRx * iR;
    const C inn = C(1) / sqrt(g.nx * g.nx + g.ny * g.ny);
    g.nx *= inn;
    g.ny *= inn;
    const C mb = kb * dth;
    const C isum = C(1) / (g.lL + g.lR);
    g.mx = mb * g.nx;
    g.my = mb * g.ny;
    g.sL = g.lL * isum;
    g.sR = g.lR * isum;
    return g;
}

// i modulo the period n for |i| <= 1e7, without an integer division: the
// rounded quotient is off by one at most
__device__ __forceinline__ int wrap_index(int i, int n, float inv_n) {
    const int r = i - (int)floorf((float)i * inv_n) * n;
    return r < 0 ? r + n : (r >= n ? r - n : r);
}

// flag the nodes of a stencil (origin wrapped into the lattice), one word of
// three neighbouring nodes' bits at a time
__device__ __forceinline__ void flag_nodes(const MarkerArgs& a, int i0, int j0) {
    const int il = i0 == 0 ? a.nx - 1 : i0 - 1, ir = i0 + 1 == a.nx ? 0 : i0 + 1;
    const int wl = il >> 5, wm = i0 >> 5, wr = ir >> 5;
    unsigned bl = 1u << (il & 31), bm = 1u << (i0 & 31), br = 1u << (ir & 31);
    // (a row of 32 k + 1 nodes has its last node alone in a word)
    if (wr == wl) {
        bl |= br;
        br = 0u;
    }
    if (wm == wl) {
        bl |= bm;
        bm = 0u;
    } else if (wm == wr) {
        br |= bm;
        bm = 0u;
    }
#pragma unroll
    for (int b = -1; b <= 1; ++b) {
        int j = j0 + b;
        if (a.walls) {
            if (j < 0 || j >= a.ny) continue;
        } else {
            j = j < 0 ? j + a.ny : (j >= a.ny ? j - a.ny : j);
        }
        unsigned* row = a.flags + (size_t)j * a.tiles_x;
        atomicOr(row + wl, bl);
        if (br) atomicOr(row + wr, br);
        if (bm) atomicOr(row + wm, bm);
    }
}

// IB shape functions at a position: nine nearest nodes, Roma weights, MLS
// (basis 1, dx, dy) re-solved where wall rows drop out.  Node indices are
// clamped so that a runaway position still stays in range; the advance kernel
// flags non-finite positions.
template <typename C, typename E>
__device__ __forceinline__ void shape_functions(const MarkerArgs& a, E xv, E yv, C (&w)[9], int& i0, int& j0) {
    const C fi0 = fmin(fmax(C(efloor(eaddc(xv, C(0.5)))), C(-1.0e7)), C(1.0e7));
    const C fj0 = fmin(fmax(C(efloor(eaddc(yv, C(0.5)))), C(-1.0e6)), C(1.0e6));
    i0 = (int)fi0;
    j0 = (int)fj0;
    C rx[3], ry[3], wx[3], wy[3];
    bool rowok[3];
    bool all = true;
#pragma unroll
    for (int q = 0; q < 3; ++q) {
        // node minus marker, (i0 + q - 1) - x
        rx[q] = -etoc(eaddc(xv, -(fi0 + C(q - 1))));
        ry[q] = -etoc(eaddc(yv, -(fj0 + C(q - 1))));
        wx[q] = roma<C>(rx[q]);
        wy[q] = roma<C>(ry[q]);
        const int jj = j0 + q - 1;
        rowok[q] = a.walls ? (jj >= 0 && jj < a.ny) : true;
        all = all && rowok[q];
    }
#pragma unroll
    for (int b = 0; b < 3; ++b)
#pragma unroll
        for (int q = 0; q < 3; ++q) w[b * 3 + q] = rowok[b] ? wx[q] * wy[b] : C(0);
    if (!all) {
        C M00 = 0, M01 = 0, M02 = 0, M11 = 0, M12 = 0, M22 = 0, sw = 0;
#pragma unroll
        for (int b = 0; b < 3; ++b)
#pragma unroll
            for (int q = 0; q < 3; ++q) {
                const C ww = w[b * 3 + q];
                sw += ww;
                M00 += ww;
                M01 += ww * rx[q];
                M02 += ww * ry[b];
                M11 += ww * rx[q] * rx[q];
                M12 += ww * rx[q] * ry[b];
                M22 += ww * ry[b] * ry[b];
            }
        // first column of the inverse of the symmetric 3x3 moment matrix
        const C c0 = M11 * M22 - M12 * M12;
        const C c1 = -(M01 * M22 - M12 * M02);
        const C c2 = M01 * M12 - M11 * M02;
        const C det = M00 * c0 + M01 * c1 + M02 * c2;
        if (det > C(1e-10)) {
#pragma unroll
            for (int b = 0; b < 3; ++b)
#pragma unroll
                for (int q = 0; q < 3; ++q) w[b * 3 + q] = w[b * 3 + q] * (c0 + c1 * rx[q] + c2 * ry[b]) / det;
        } else if (sw > C(0)) {
#pragma unroll
            for (int q = 0; q < 9; ++q) w[q] = w[q] / sw;
        } else {
#pragma unroll
            for (int q = 0; q < 9; ++q) w[q] = C(0);
        }
    }
}

// Eq. repFor screening by one warp, in two stages: groups (32 vertices) of
// other membranes whose box comes within d_rep of this chunk's box (the union
// of its one or two groups' boxes), and of those the segments.  Hits join the
// block's candidate list in any order: the repulsion sums are over integers, and
// a pair rounds the same whether its segment is staged, listed or just walked.
// The groups cut the boxes that every block reads to a quarter (64 instead of
// 228 on the 640 x 160 capillary, one pass of the loop below).
struct Candidates {
    int* n;       // all hits
    int* seg;     // [kMaxCand] the first of them, and of the first kStageSeg also
    int* v0;      // first vertex and vertices
    int* nv;
    float4* box;
};
__device__ __forceinline__ void screen_segments(const MarkerArgs& a, int m, int own0, int kn, int lane,
                                                const Candidates& s_c) {
    const float4 o0 = a.group_box[own0];
    const float4 o1 = kn > kGroupV ? a.group_box[own0 + 1] : o0;
    const float reach = a.f.d_rep + 2e-3f;
    float ddx = wrap_half(o1.x - o0.x, a.f.nx);
    float ddy = o1.y - o0.y;
    if (!a.walls) ddy = wrap_half(ddy, a.f.ny);
    const float lo_x = fminf(-o0.z, ddx - o1.z), hi_x = fmaxf(o0.z, ddx + o1.z);
    const float lo_y = fminf(-o0.w, ddy - o1.w), hi_y = fmaxf(o0.w, ddy + o1.w);
    const float cbx = o0.x + 0.5f * (lo_x + hi_x), cby = o0.y + 0.5f * (lo_y + hi_y);
    const float rx = 0.5f * (hi_x - lo_x) + reach, ry = 0.5f * (hi_y - lo_y) + reach;
    auto near = [&](const float4& b) {
        const float dx = wrap_half(b.x - cbx, a.f.nx);
        float dy = b.y - cby;
        if (!a.walls) dy = wrap_half(dy, a.f.ny);
        return fabsf(dx) <= b.z + rx && fabsf(dy) <= b.w + ry;
    };
    for (int base = lane; base < a.ngroup; base += 32 * kScreenIter) {
        float4 bx[kScreenIter];
        int4 gi[kScreenIter];
#pragma unroll
        for (int it = 0; it < kScreenIter; ++it) {
            const int g = base + 32 * it;
            gi[it].x = m;
            if (g < a.ngroup) {
                bx[it] = a.group_box[g];
                gi[it] = a.group[g];
            }
        }
#pragma unroll
        for (int it = 0; it < kScreenIter; ++it) {
            if (gi[it].x == m || !near(bx[it])) continue;  // own membrane, or beyond the range
            const int ns = (gi[it].w + kSegV - 1) / kSegV;
            float4 sb[kGroupV / kSegV];
#pragma unroll
            for (int q = 0; q < kGroupV / kSegV; ++q)
                if (q < ns) sb[q] = a.seg_box[gi[it].y + q];
#pragma unroll
            for (int q = 0; q < kGroupV / kSegV; ++q) {
                if (q >= ns || !near(sb[q])) continue;
                const int pos = atomicAdd(s_c.n, 1);
                if (pos < kMaxCand) s_c.seg[pos] = gi[it].y + q;
                if (pos < kStageSeg) {
                    s_c.v0[pos] = gi[it].z + kSegV * q;
                    s_c.nv[pos] = min(kSegV, gi[it].w - kSegV * q);
                    s_c.box[pos] = sb[q];
                }
            }
        }
    }
}

// One block per work unit (a chunk of up to kChunkV consecutive vertices of one
// membrane).  The kernel is a chain of dependent loads and FP32 divisions and
// square roots, so the parts of a vertex's force go to different warps and
// meet only where one needs another:
//   warps 0-1  bending geometry, stretching, bending and bond forces per vertex
//   warps 2-3  IB shape functions (MLS / Roma) and stencil origins
//   warp 4     repulsion candidate segments
//   warp 5     bending geometry of the halo vertices (one on each side), halo
//              record for the advance kernel
//   warps 6-7  enclosed area of the membrane
//   between    warps 0, 1, 5 meet for the neighbours' bending shares
//   then       all: (candidate segment, vertex) pairs where there are any, four
//              threads a vertex, accumulated in fixed point (order-free);
//              warps 0-1 add the parts of a vertex up, and all spread it over
//              its nodes (of a dynamic particle: its forcing term, see
//              dynamic_kernels.cu)
// Before, ten warps met after each of four phases, the area (four warps) and
// the screening of every segment (two) ahead of the force terms: 8900 cycles a
// block on the 640 x 160 capillary, three blocks per SM in the batched form
// (four now).
//
// forces_unit is the body for force unit `unit` of the context `a`: the
// single-context kernel runs unit blockIdx.x, the batched kernel (ensembles)
// one unit of one member per block.
template <typename C>
__device__ __forceinline__ void forces_unit(const MarkerArgs& a, int unit, bool settle) {
    using E = typename Ext<C>::E;
    if (unit == a.nfu) {  // one block more than units: the previous step's bond decisions
        dep_wait();
        dep_trigger();
        if (settle) settle_bonds(a);
        return;
    }
    const int4 u0 = a.fu[3 * unit], u1 = a.fu[3 * unit + 1];
    const int m = u0.x, k0 = u0.y, kn = u0.z, off = u0.w, n = u1.x;
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    __shared__ E s_x[kChunkV], s_y[kChunkV];  // positions of the chunk
    // bending geometry of vertices k0-1 .. k0+kn (slot j <-> vertex k0 - 1 + j)
    __shared__ C s_mnx[kChunkV + 2], s_mny[kChunkV + 2], s_sL[kChunkV + 2], s_sR[kChunkV + 2];
    __shared__ C s_nx[kChunkV], s_ny[kChunkV];
    __shared__ C s_w[kChunkV][9];
    __shared__ int s_i0[kChunkV], s_j0[kChunkV];
    __shared__ unsigned long long s_rep[kChunkV];
    // force without area and repulsion, and the area term's direction
    __shared__ C s_F[kChunkV][2], s_ax[kChunkV], s_ay[kChunkV];
    __shared__ E red[4];
    __shared__ C s_ca;
    __shared__ int s_cand[kMaxCand];
    __shared__ int s_ncand;
    // staged candidate segments: box, anchor (first vertex) and the offsets of
    // their vertices from the anchor in the compute type
    __shared__ float4 s_cbox[kStageSeg];
    __shared__ E s_cax[kStageSeg], s_cay[kStageSeg];
    __shared__ __align__(16) C s_cox[kStageSeg][kSegV], s_coy[kStageSeg][kSegV];
    __shared__ int s_cn[kStageSeg], s_cv0[kStageSeg];
    const Rest<C>* rest = static_cast<const Rest<C>*>(a.rest);
    // (with dynamic particles the predecessor is the hydrodynamic kernel, which
    // started after the positions were complete: its results are waited for
    // where they are used)
    // the halo vertices' bending geometry: by the two lanes after the chunk's
    // last vertex where warps 0-1 have them, else by warp 5
    const bool halo_here = kn + 2 <= 64;
    if (wid < 2) {
        // slot of this thread's vertex: tid + 1, then the two halo vertices
        const int slot = tid < kn ? tid + 1 : (halo_here && tid == kn ? kn + 1 : 0);
        const bool mine = tid < kn;
        C Fx = C(0), Fy = C(0), mx = C(0), my = C(0);
        if (mine || (halo_here && tid < kn + 2)) {
            int k = k0 - 1 + slot;
            k = k < 0 ? k + n : (k >= n ? k - n : k);
            const int v = off + k, L = off + (k == 0 ? n - 1 : k - 1), R = off + (k == n - 1 ? 0 : k + 1);
            const Rest<C> rv = rest[v], rl = rest[L];
            const C kb = par<C>(a.mem_kb[m], float(a.mem_kb[m])), ks = par<C>(a.mem_ks[m], float(a.mem_ks[m]));
            int lig_l = -1, lig_v = -1;
            if (mine && a.nlig > 0) {
                lig_l = a.elem_lig[L];
                lig_v = a.elem_lig[v];
            }
            if (!a.has_dyn) dep_wait();
            E xl, yl, xv, yv, xR, yR;
            load_pos<C>(a, L, xl, yl);
            load_pos<C>(a, v, xv, yv);
            load_pos<C>(a, R, xR, yR);
            // Eq. adhFor on the two elements sharing v, half each
            if (lig_l >= 0 || lig_v >= 0) {
                int rec_l, rec_v;
                bonds_now(a, lig_l, lig_v, !settle, rec_l, rec_v);
                bond_on_element<C, E>(a, rec_l, xl, yl, xv, yv, Fx, Fy);
                bond_on_element<C, E>(a, rec_v, xv, yv, xR, yR, Fx, Fy);
            }
            const VertexGeo<C, E> g = vertex_geometry<C, E>(rv, kb, xl, yl, xv, yv, xR, yR);
            mx = g.mx;
            my = g.my;
            s_mnx[slot] = g.mx;
            s_mny[slot] = g.my;
            s_sL[slot] = g.sL;
            s_sR[slot] = g.sR;
            if (mine) {
                s_nx[tid] = g.nx;
                s_ny[tid] = g.ny;
                // Eq. strainFor on elements (v, R) and (L, v); l - l_0 is formed as
                // (l^2 - l_0^2) / (l + l_0) with the squares in the extended type
                const C l = sqrt(etoc(g.lsqR)), l2 = sqrt(etoc(g.lsqL));
                const C c = ks * etoc(esub(g.lsqR, rv.lsq)) / ((l + rv.l0) * l);
                Fx += c * g.eRx;
                Fy += c * g.eRy;
                const C c2 = -ks * etoc(esub(g.lsqL, rl.lsq)) / ((l2 + rl.l0) * l2);
                Fx += c2 * g.eLx;
                Fy += c2 * g.eLy;
                // Eq. areaFor's direction, half of each adjacent element
                s_ax[tid] = -etoc(esub(yR, yl));
                s_ay[tid] = etoc(esub(xR, xl));
            }
        } else if (!a.has_dyn) {
            dep_wait();
        }
        // Eq. bendFor gathered: own term plus the neighbours' shares (warps 0, 1, 5)
        asm volatile("bar.sync 1, 96;" ::: "memory");
        if (mine) {
            Fx += -mx + s_mnx[slot + 1] * s_sL[slot + 1] + s_mnx[slot - 1] * s_sR[slot - 1];
            Fy += -my + s_mny[slot + 1] * s_sL[slot + 1] + s_mny[slot - 1] * s_sR[slot - 1];
            s_F[tid][0] = Fx;
            s_F[tid][1] = Fy;
        }
    } else if (wid < 4) {
        const int j = tid - 64;
        s_rep[j] = 0ull;
        if (!a.has_dyn) dep_wait();
        if (j < kn) {
            E xv, yv;
            load_pos<C>(a, off + k0 + j, xv, yv);
            s_x[j] = xv;
            s_y[j] = yv;
            C w[9];
            int i0, j0;
            shape_functions<C, E>(a, xv, yv, w, i0, j0);
            const int v = off + k0 + j;
            C* W = static_cast<C*>(a.W);
#pragma unroll
            for (int q = 0; q < 9; ++q) {
                W[9 * (size_t)v + q] = w[q];
                s_w[j][q] = w[q];
            }
            const int i0w = wrap_index(i0, a.nx, a.f.inv_nx);
            const int j0s = a.walls ? j0 : wrap_index(j0, a.ny, a.f.inv_ny);
            reinterpret_cast<int2*>(a.stencil)[v] = make_int2(i0w, j0s);
            s_i0[j] = i0w;
            s_j0[j] = j0s;
            flag_nodes(a, i0w, j0s);
        }
    } else if (wid == 4) {
        const int own0 = a.fu[3 * unit + 2].y + k0 / kGroupV;
        if (lane == 0) s_ncand = 0;
        __syncwarp();
        if (!a.has_dyn) dep_wait();
        if (a.nmem > 1)
            screen_segments(a, m, own0, kn, lane, Candidates{&s_ncand, s_cand, s_cv0, s_cn, s_cbox});
    } else if (wid == 5) {
        if (!halo_here && lane < 2) {
            // the halo vertices k0 - 1 (slot 0) and k0 + kn (slot kn + 1)
            const int slot = lane == 1 ? kn + 1 : 0;
            int k = k0 - 1 + slot;
            k = k < 0 ? k + n : (k >= n ? k - n : k);
            const Rest<C> r0 = rest[off + k];
            const C kb = par<C>(a.mem_kb[m], float(a.mem_kb[m]));
            if (!a.has_dyn) dep_wait();
            E xl, yl, xv, yv, xR, yR;
            load_pos<C>(a, off + (k == 0 ? n - 1 : k - 1), xl, yl);
            load_pos<C>(a, off + k, xv, yv);
            load_pos<C>(a, off + (k == n - 1 ? 0 : k + 1), xR, yR);
            const VertexGeo<C, E> g = vertex_geometry<C, E>(r0, kb, xl, yl, xv, yv, xR, yR);
            s_mnx[slot] = g.mx;
            s_mny[slot] = g.my;
            s_sL[slot] = g.sL;
            s_sR[slot] = g.sR;
        } else if (!a.has_dyn) {
            dep_wait();
        }
        __syncwarp();
        asm volatile("bar.sync 1, 96;" ::: "memory");
        if (lane == 2 && u1.w >= 0 && (a.nlig > 0 || n > kDirectArea)) {
            // this chunk's first vertex for the advance of the ring's other chunks
            E xh, yh;
            load_pos<C>(a, off + k0, xh, yh);
            PosIO<C>::store(a.halo, 2 * u1.w, xh, yh);
            PosIO<C>::load(a.Xp, off + k0, xh, yh);
            PosIO<C>::store(a.halo, 2 * u1.w + 1, xh, yh);
        }
    } else {
        // Eq. areaFor with p_ref = 1/3: F_l = c_a (inward normal) l_l
        // c_a = -k_a (1 - A/A_0) p_ref = q (A - A_0), q = k_a p_ref / A_0 from set-up
        const double A0 = a.mem_A0[m], q = a.mem_qa[m];
        if (!a.has_dyn) dep_wait();
        const E A = ring_area<C>(a, off, n, u1.w - k0 / kChunkV, 6, red, 2);
        if (tid == 32 * 6) s_ca = C(q * (etod(A) - A0));
    }

    __syncthreads();
    {
        const int ncand = s_ncand;
        const bool all_segs = ncand > kMaxCand;  // list overflow: screen every segment
        if (ncand > 0) {
            // Eq. repFor against vertices of other membranes closer than d_rep, over
            // (candidate segment, vertex) pairs; the magnitudes of each vertex are
            // summed in fixed point (the direction is its own inward normal).
            // First the candidates' vertices as offsets from their first vertex
            // (the anchor)
            const int nst = all_segs ? 0 : (ncand < kStageSeg ? ncand : kStageSeg);
            for (int e = tid; e < nst * kSegV; e += kForceThreads) {
                const int ci = e / kSegV, g = e - ci * kSegV;
                const int v0 = s_cv0[ci];
                const bool there = g < s_cn[ci];
                E xa, ya, xb, yb;
                load_pos<C>(a, v0, xa, ya);
                load_pos<C>(a, v0 + (there ? g : 0), xb, yb);
                // (a segment's missing vertices: out of any range)
                s_cox[ci][g] = there ? etoc(esub(xb, xa)) : C(1e15);
                s_coy[ci][g] = there ? etoc(esub(yb, ya)) : C(1e15);
                if (g == 0) {
                    s_cax[ci] = xa;
                    s_cay[ci] = ya;
                }
            }
            __syncthreads();
            const int nscan = all_segs ? a.nseg : ncand;
            const float reach = a.f.d_rep + 2e-3f;
            const C c_rep = C(1e-4 / (8.0 * 1.4142135623730951));
            const C drep = par<C>(a.d_rep, a.f.d_rep);
            // a squared distance beyond this is surely out of range: no square root
            const C drep2 = drep * drep * C(1.00001);
            // a thread keeps its vertex and takes every fourth candidate
            const int j = tid & (kChunkV - 1);
            const E xv = s_x[j], yv = s_y[j];
            const float hx = float(ehi(xv)), hy = float(ehi(yv));
            const float xvw = hx - a.f.nx * floorf(hx * a.f.inv_nx);
            const float yvw = hy - a.f.wrap_ny * floorf(hy * a.f.inv_ny);
            bool bad = false;
            for (int ci = tid / kChunkV; ci < nscan && j < kn; ci += kForceThreads / kChunkV) {
                const bool staged = !all_segs && ci < kStageSeg;
                const int sg = all_segs ? ci : s_cand[ci];
                if (all_segs && a.seg_mem[sg] == m) continue;
                const float4 bx = staged ? s_cbox[ci] : a.seg_box[sg];
                const float ddx = wrap_half(xvw - bx.x, a.f.nx);
                float ddy = yvw - bx.y;
                if (!a.walls) ddy = wrap_half(ddy, a.f.ny);
                if (fabsf(ddx) > bx.z + reach || fabsf(ddy) > bx.w + reach) continue;
                C mags = C(0);
                if (staged) {
                    // vertex relative to the segment anchor once, then plain differences
                    const C dxa = etoc(ewrap(esub(xv, s_cax[ci]), par<C>(a.nx, a.f.nx), par<C>(a.inv_nx, a.f.inv_nx)));
                    C dya = etoc(esub(yv, s_cay[ci]));
                    if (!a.walls) dya = etoc(ewrap(esub(yv, s_cay[ci]), par<C>(a.ny, a.f.ny), par<C>(a.inv_ny, a.f.inv_ny)));
                    unsigned close = 0;
#pragma unroll
                    for (int g = 0; g < kSegV; ++g) {
                        const C dx = dxa - s_cox[ci][g], dy = dya - s_coy[ci][g];
                        if (dx * dx + dy * dy < drep2) close |= 1u << g;
                    }
                    while (close) {
                        const int g = __ffs(close) - 1;
                        close &= close - 1;
                        const C dx = dxa - s_cox[ci][g], dy = dya - s_coy[ci][g];
                        const C d = sqrt(dx * dx + dy * dy);
                        if (d < drep) mags += c_rep * sqrt(C(1) / (d * d * d * d * d));
                    }
                } else {
                    // (by the offsets from the anchor too)
                    const int nb = a.seg_n[sg], b0 = a.seg_v0[sg];
                    E xa, ya;
                    load_pos<C>(a, b0, xa, ya);
                    const C dxa = etoc(ewrap(esub(xv, xa), par<C>(a.nx, a.f.nx), par<C>(a.inv_nx, a.f.inv_nx)));
                    C dya = etoc(esub(yv, ya));
                    if (!a.walls) dya = etoc(ewrap(esub(yv, ya), par<C>(a.ny, a.f.ny), par<C>(a.inv_ny, a.f.inv_ny)));
                    for (int g = 0; g < nb; ++g) {
                        E xb, yb;
                        load_pos<C>(a, b0 + g, xb, yb);
                        const C dx = dxa - etoc(esub(xb, xa)), dy = dya - etoc(esub(yb, ya));
                        const C d = sqrt(dx * dx + dy * dy);
                        if (d < drep) mags += c_rep * sqrt(C(1) / (d * d * d * d * d));
                    }
                }
                if (mags != C(0)) {
                    mags = clamp_fix(mags, C(kFix60Limit), bad);
                    atomicAdd(&s_rep[j], (unsigned long long)to_fix60<C>(mags));
                }
            }
            if (bad) atomicOr(a.status, ST_FIXRANGE);
            __syncthreads();
        }
    }
    if (a.has_dyn) dep_wait();
    // (here rather than at the start: the fused kernel's early blocks would
    // take SMs unevenly around the force blocks; FP64 capillary step 58.6 vs
    // 63.4 us, FP32 17.0 vs 17.5 us)
    dep_trigger();

    if (tid < kn) {
        // the parts added up; what is spread, in units of the fixed-point grid
        // (2^-52: an exact scaling)
        const C ca = s_ca;
        const C mag = fix60_to_c<C>((long long)s_rep[tid]);
        C Fx = s_F[tid][0] + C(0.5) * ca * s_ax[tid], Fy = s_F[tid][1] + C(0.5) * ca * s_ay[tid];
        Fx -= mag * s_nx[tid];
        Fy -= mag * s_ny[tid];
        C Sx = Fx, Sy = Fy;
        const int v = off + k0 + tid;
        if (u1.y >= LBIB_MEMBRANE_DYNAMIC) {
            // dynamic particle (Sec. 2.4): the total force of Eq. newtonSoft adds
            // the hydrodynamic force; the fluid receives the forcing term instead
            const C* Hf = static_cast<const C*>(a.Hf);
            const C* D = static_cast<const C*>(a.Dib);
            Fx += Hf[2 * (size_t)v];
            Fy += Hf[2 * (size_t)v + 1];
            Sx = D[2 * (size_t)v];
            Sy = D[2 * (size_t)v + 1];
        }
        C* F = static_cast<C*>(a.F);
        F[2 * (size_t)v] = Fx;
        F[2 * (size_t)v + 1] = Fy;
        s_F[tid][0] = Sx * C(kFixScale);
        s_F[tid][1] = Sy * C(kFixScale);
    }
    __syncthreads();
    // spreading (Sec. 2.2, the transpose of the interpolation): w_j F_v into the
    // fixed-point force field
    for (int p = tid; p < 9 * kn; p += kForceThreads) {
        const int j = p / 9, q9 = p - 9 * j;
        const int b = q9 / 3, q = q9 - 3 * b;
        int jj = s_j0[j] + b - 1;
        if (a.walls) {
            if (jj < 0 || jj >= a.ny) continue;
        } else {
            jj = jj < 0 ? jj + a.ny : (jj >= a.ny ? jj - a.ny : jj);
        }
        int ii = s_i0[j] + q - 1;
        ii = ii < 0 ? ii + a.nx : (ii >= a.nx ? ii - a.nx : ii);
        const C wq = s_w[j][q9];
        bool bad = false;
        const C gx = clamp_fix(wq * s_F[j][0], C(kFixLimit * kFixScale), bad);
        const C gy = clamp_fix(wq * s_F[j][1], C(kFixLimit * kFixScale), bad);
        if (bad) atomicOr(a.status, ST_FIXRANGE);
        unsigned long long* gp = reinterpret_cast<unsigned long long*>(a.gsum + (size_t)jj * a.nx + ii);
        atomicAdd(gp, (unsigned long long)to_fix<C>(gx));
        atomicAdd(gp + 1, (unsigned long long)to_fix<C>(gy));
    }
}

template <typename C>
__global__ void __launch_bounds__(kForceThreads) k_forces(const MarkerArgs a, const bool settle) {
    forces_unit<C>(a, blockIdx.x, settle);
}

// Batched form: the force units of up to kBatchMax contexts (ensemble
// members) in one launch, one block per (member, unit).  The member's
// arguments are staged in shared memory.
// (FP32: four blocks per SM, the batch's thousands of blocks are limited by how
// many fit, not by one block's latency.  FP64: three.  At four the 64 registers
// spill 268 bytes of stores and 200 of loads: 64 members 94.4 us against 89.8,
// 10 members 25.5 against 24.8; 32 members 54.6 against 58.7, their whole step
// 659.4 against 658.2.)
template <typename C>
__global__ void __launch_bounds__(kForceThreads, sizeof(C) == 8 ? 3 : 4)
    k_forces_batch(const __grid_constant__ MarkerBatch b, const bool settle) {
    __shared__ MarkerArgs s_a;
    const int m = marker_member(b, blockIdx.x);
    stage_args(&s_a, b.args + m);
    forces_unit<C>(s_a, blockIdx.x - b.off[m], settle);
}

// the end of a launch sequence: the last step's bond decisions, one block per
// context
__global__ void __launch_bounds__(256) k_settle(const MarkerArgs a) {
    dep_wait();
    settle_bonds(a);
}
__global__ void __launch_bounds__(256) k_settle_batch(const MarkerArgs* args) {
    __shared__ MarkerArgs s_a;
    stage_args(&s_a, args + blockIdx.x);
    dep_wait();
    settle_bonds(s_a);
}

// ---------------------------------------------------------------- segments
// segment and group boxes alone (before the first step and after user-written
// markers): one warp per group
template <typename C>
__global__ void k_seg_boxes(const MarkerArgs a) {
    using E = typename Ext<C>::E;
    const int lane = threadIdx.x & 31;
    const int gr = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
    if (gr >= a.ngroup) return;
    const int4 g = a.group[gr];
    const int first = lane & ~(kSegV - 1);  // of this lane's segment
    E x, y;
    load_pos<C>(a, g.z + (lane < g.w ? lane : (first < g.w ? first : 0)), x, y);
    seg_box_regs<C>(a, first < g.w ? g.y + lane / kSegV : -1, gr, lane, x, y);
}

// the chunk sums of the long rings' areas, one warp per advance unit
template <typename C>
__global__ void k_area_parts(const MarkerArgs a) {
    using E = typename Ext<C>::E;
    const int4 u0 = a.au[3 * blockIdx.x], u1 = a.au[3 * blockIdx.x + 1];
    if (u1.x <= kDirectArea) return;
    E cx, cy;
    PosIO<C>::load(a.Xp, u0.w, cx, cy);
    const int v0 = u0.w + u0.y;
    const E part = chunk_area<C>(u0.z, threadIdx.x, cx, cy, [&](int k, E& x, E& y) { load_pos<C>(a, v0 + k, x, y); });
    if (threadIdx.x == 0) PosIO<C>::store(a.area_part, blockIdx.x, part, part);
}

template <typename C>
__global__ void k_areas(const MarkerArgs a, double* areas) {
    __shared__ typename Ext<C>::E red[4];
    const int m = blockIdx.x;
    const typename Ext<C>::E A = ring_area<C>(a, a.mem_off[m], a.mem_n[m], a.mem_au[m], 0, red, 1);
    if (threadIdx.x == 0) areas[blockIdx.x] = etod(A);
}

// marker positions between doubles (x0, y0, x1, ...) and the device layout
template <typename C>
__global__ void k_pos_in(const double* xy, void* X, int nv) {
    const int v = blockIdx.x * blockDim.x + threadIdx.x;
    if (v >= nv) return;
    PosIO<C>::store(X, v, from_double_e<C>(xy[2 * v]), from_double_e<C>(xy[2 * v + 1]));
}
template <typename C>
__global__ void k_pos_out(const void* X, double* xy, int nv) {
    const int v = blockIdx.x * blockDim.x + threadIdx.x;
    if (v >= nv) return;
    typename Ext<C>::E x, y;
    PosIO<C>::load(X, v, x, y);
    xy[2 * v] = etod(x);
    xy[2 * v + 1] = etod(y);
}

// ---------------------------------------------------------------- launchers
static bool is_f64(lbib_precision p) { return p == LBIB_F64; }

cudaError_t launch_rest(lbib_precision prec, const MarkerArgs& a, void* rest, double* A0, double* qa,
                        cudaStream_t s) {
    if (is_f64(prec)) k_rest<double><<<a.nmem, 256, 0, s>>>(a, rest, A0, qa);
    else k_rest<float><<<a.nmem, 256, 0, s>>>(a, rest, A0, qa);
    return cudaGetLastError();
}

cudaError_t launch_forces(lbib_precision prec, const MarkerArgs& a, bool settle, cudaStream_t s, bool chained) {
    return launch_kernel(is_f64(prec) ? k_forces<double> : k_forces<float>, a.nfu + (settle ? 1 : 0), kForceThreads, 0, s,
                         chained, a, settle);
}

cudaError_t launch_forces_batch(lbib_precision prec, const MarkerBatch& b, bool settle, cudaStream_t s, bool chained) {
    if (b.n < 1 || b.n > kBatchMax) return cudaErrorInvalidValue;
    const int nunits = b.off[b.n];
    if (nunits <= 0) return cudaSuccess;
    return launch_kernel(is_f64(prec) ? k_forces_batch<double> : k_forces_batch<float>, nunits, kForceThreads, 0, s,
                         chained, b, settle);
}

cudaError_t launch_settle(const MarkerArgs& a, cudaStream_t s) {
    return launch_kernel(k_settle, 1, 256, 0, s, true, a);
}

cudaError_t launch_settle_batch(const MarkerArgs* args, int n, cudaStream_t s) {
    return launch_kernel(k_settle_batch, n, 256, 0, s, true, args);
}

cudaError_t launch_seg_boxes(lbib_precision prec, const MarkerArgs& a, cudaStream_t s) {
    if (a.ngroup == 0) return cudaSuccess;
    const int g = (a.ngroup + 7) / 8;
    if (is_f64(prec)) k_seg_boxes<double><<<g, 256, 0, s>>>(a);
    else k_seg_boxes<float><<<g, 256, 0, s>>>(a);
    return cudaGetLastError();
}

cudaError_t launch_area_parts(lbib_precision prec, const MarkerArgs& a, cudaStream_t s) {
    if (a.nau == 0) return cudaSuccess;
    if (is_f64(prec)) k_area_parts<double><<<a.nau, 32, 0, s>>>(a);
    else k_area_parts<float><<<a.nau, 32, 0, s>>>(a);
    return cudaGetLastError();
}

cudaError_t launch_areas(lbib_precision prec, const MarkerArgs& a, double* areas, cudaStream_t s) {
    if (is_f64(prec)) k_areas<double><<<a.nmem, 64, 0, s>>>(a, areas);
    else k_areas<float><<<a.nmem, 64, 0, s>>>(a, areas);
    return cudaGetLastError();
}

cudaError_t launch_pos_in(lbib_precision prec, const double* xy, void* X, int nv, cudaStream_t s) {
    if (nv == 0) return cudaSuccess;
    if (is_f64(prec)) k_pos_in<double><<<(nv + 255) / 256, 256, 0, s>>>(xy, X, nv);
    else k_pos_in<float><<<(nv + 255) / 256, 256, 0, s>>>(xy, X, nv);
    return cudaGetLastError();
}

cudaError_t launch_pos_out(lbib_precision prec, const void* X, double* xy, int nv, cudaStream_t s) {
    if (nv == 0) return cudaSuccess;
    if (is_f64(prec)) k_pos_out<double><<<(nv + 255) / 256, 256, 0, s>>>(X, xy, nv);
    else k_pos_out<float><<<(nv + 255) / 256, 256, 0, s>>>(X, xy, nv);
    return cudaGetLastError();
}

}  // namespace lbib
