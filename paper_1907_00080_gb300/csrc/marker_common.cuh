// Device helpers shared by the Lagrangian kernels (forces / spreading and
// interpolation / advance / bonds).
#pragma once

#include <climits>

#include "bond_logic.cuh"
#include "ext_real.cuh"
#include "lbib_internal.cuh"

namespace lbib {

constexpr unsigned kFull = 0xffffffffu;

__device__ __forceinline__ float wrap_half(float d, float L) {
    return d > 0.5f * L ? d - L : (d < -0.5f * L ? d + L : d);
}

// force value, in units of the fixed-point grid of the spread field (2^-52),
// to the grid
template <typename C> __device__ __forceinline__ long long to_fix(C v);
template <> __device__ __forceinline__ long long to_fix<float>(float t) {
    // exact: t is either below 2^23 in magnitude (round it with a 32-bit
    // conversion) or an integer whose mantissa is shifted into place
    if (fabsf(t) < 8388608.0f) return (long long)__float2int_rn(t);
    const int bits = __float_as_int(t);
    const int e = ((bits >> 23) & 0xff) - 150;  // t = mant 2^e with e >= 0 here
    const long long mag = (long long)((bits & 0x7fffff) | 0x800000) << (e < 40 ? e : 40);
    return bits < 0 ? -mag : mag;
}
template <> __device__ __forceinline__ long long to_fix<double>(double t) { return __double2ll_rn(t); }

// Range of the fixed-point conversions.  The spread field holds w F per
// (vertex, node) scaled by 2^52, the repulsion accumulators one magnitude per
// (vertex, segment) scaled by 2^60, in signed 64-bit integers.  A value at or
// beyond its bound, or not finite, is clamped to the bound (NaN to 0) and
// `bad` is set; the kernel then raises ST_FIXRANGE, which the host reads as
// LBIB_E_NONFINITE.  Bounds: 64 lu of force per (vertex, node), 2^58 in the
// field, so 32 such terms fit in one node's int64; repulsion 1 per
// (vertex, segment), 2^60 in an accumulator that holds 8 (Eq. repFor reaches
// 1 at d = 9.4e-3 lu, i.e. membranes that overlap).
constexpr double kFixLimit = 64.0;
constexpr double kFix60Limit = 1.0;
template <typename C>
__device__ __forceinline__ C clamp_fix(C v, C lim, bool& bad) {
    if (fabs(v) < lim) return v;  // false for NaN
    bad = true;
    return v > C(0) ? lim : (v < C(0) ? -lim : C(0));
}

// value scaled by 2^60 to a 64-bit integer (repulsion accumulators: magnitudes
// stay below 8, resolution 2^-60), exact for the float case
template <typename C> __device__ __forceinline__ long long to_fix60(C v);
template <> __device__ __forceinline__ long long to_fix60<float>(float v) {
    const float t = v * 1.152921504606846976e18f;  // 2^60
    if (fabsf(t) < 8388608.0f) return (long long)__float2int_rn(t);
    const int bits = __float_as_int(t);
    const int e = ((bits >> 23) & 0xff) - 150;
    const long long mag = (long long)((bits & 0x7fffff) | 0x800000) << (e < 39 ? e : 39);
    return bits < 0 ? -mag : mag;
}
template <> __device__ __forceinline__ long long to_fix60<double>(double v) {
    return __double2ll_rn(v * 1.152921504606846976e18);
}
template <typename C> __device__ __forceinline__ C fix60_to_c(long long v);
template <> __device__ __forceinline__ float fix60_to_c<float>(long long v) {
    const int hi = (int)(v >> 32);
    const unsigned lo = (unsigned)(v & 0xffffffffll);
    return fmaf((float)hi, 3.7252902984619141e-09f, (float)lo * 8.6736173798840355e-19f);
}
template <> __device__ __forceinline__ double fix60_to_c<double>(long long v) {
    return __ll2double_rn(v) * 8.6736173798840355e-19;
}

// fixed-point value (scaled by 2^52) back to the compute type
template <typename C> __device__ __forceinline__ C fix_to_c(long long v);
template <> __device__ __forceinline__ float fix_to_c<float>(long long v) {
    const int hi = (int)(v >> 32);
    const unsigned lo = (unsigned)(v & 0xffffffffll);
    return fmaf((float)hi, 9.5367431640625e-07f, (float)lo * 2.220446049250313e-16f);
}
template <> __device__ __forceinline__ double fix_to_c<double>(long long v) {
    return __ll2double_rn(v) * kFixInv;
}

// Roma, Peskin & Berger three-point regularised delta
template <typename C>
__device__ __forceinline__ C roma(C r) {
    const C a = fabs(r);
    if (a <= C(0.5)) return (C(1) + sqrt(C(1) - C(3) * a * a)) / C(3);
    if (a <= C(1.5)) {
        const C b = C(1) - a;
        return (C(5) - C(3) * a - sqrt(C(1) - C(3) * b * b)) / C(6);
    }
    return C(0);
}

template <typename C>
__device__ __forceinline__ void load_pos(const MarkerArgs& a, int v, typename Ext<C>::E& x,
                                         typename Ext<C>::E& y) {
    PosIO<C>::load(a.X, v, x, y);
}

// Edge products at a vertex in the extended type from the positions of L, v, R:
// squared length of e_R = x_R - x_v, and the cross and dot products of
// e_L = x_v - x_L with e_R (their rotation from the rest pair gives theta - theta_0).
template <typename C>
struct EdgeProducts {
    typename Ext<C>::E lsqR, cross, dot;
};
template <typename E, typename C>
__device__ __forceinline__ EdgeProducts<C> edge_products(E xL, E yL, E xv, E yv, E xR, E yR) {
    const E eLx = esub(xv, xL), eLy = esub(yv, yL), eRx = esub(xR, xv), eRy = esub(yR, yv);
    EdgeProducts<C> p;
    p.lsqR = eadd(emul(eRx, eRx), emul(eRy, eRy));
    p.cross = esub(emul(eLx, eRy), emul(eLy, eRx));
    p.dot = eadd(emul(eLx, eRx), emul(eLy, eRy));
    return p;
}

// Enclosed area of a ring by the shoelace formula, summed in a fixed order, so
// that every caller gets the same bits at the same state (the rest shape of a
// ring of up to kDirectArea vertices then has exactly its rest area; a longer
// ring's while X^{n-1} of its vertex 0 is the set-up's too).
//
// Rings of up to kDirectArea vertices: about vertex 0, by the 64 lanes of two
// consecutive warps starting at `w0`: four sums, of the terms k with k / 32 mod
// 4 = 0 .. 3 (lane l of sum s takes terms 32 s + l + 128 i in order, the lanes
// are reduced by a fixed tree), added in order.  `red` holds 4 values; the
// result is valid in the first warp's lanes after the named barrier `bar` (64
// threads).
//
// Longer rings: every block of the force kernel would walk the whole ring (27
// blocks of 1700 vertices on the fine capillary, 9800 of their 18900 cycles).
// Their chunks' interior elements are summed once, by the advance kernel where
// it has the new positions at hand (chunk_area), about c = X^{n-1} of vertex 0;
// the reader adds the elements between chunks and the chunks' sums
// (ring_area_parts, one warp, result in lane 0).
constexpr int kDirectArea = 256;
template <typename E>
__device__ __forceinline__ E cross_about(E cx, E cy, E xa, E ya, E xb, E yb) {
    return esub(emul(esub(xa, cx), esub(yb, cy)), emul(esub(xb, cx), esub(ya, cy)));
}
// sum over the warp's lanes by a fixed tree, in lane 0
template <typename E>
__device__ __forceinline__ E warp_tree(E v, int lane) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        E t;
        shfl_e(t, v, (lane + o) & 31);
        v = eadd(v, t);
    }
    return v;
}
template <typename C>
__device__ typename Ext<C>::E ring_area_direct(const MarkerArgs& a, int off, int n, int w0,
                                               typename Ext<C>::E* red, int bar) {
    using E = typename Ext<C>::E;
    const int t = threadIdx.x - 32 * w0;  // 0 .. 63
    const int lane = t & 31;
    E xr, yr;
    load_pos<C>(a, off, xr, yr);
    // two rows of terms at once, t + 128 i and t + 64 + 128 i, all loads of a
    // pass issued first
    E acc[2] = {ezero<E>(), ezero<E>()};
    for (int k0 = t; k0 < n; k0 += 128) {
        E xv[2], yv[2], xR[2], yR[2];
#pragma unroll
        for (int q = 0; q < 2; ++q) {
            const int k = k0 + 64 * q;
            const int kk = k < n ? k : 0;
            load_pos<C>(a, off + kk, xv[q], yv[q]);
            load_pos<C>(a, off + (kk == n - 1 ? 0 : kk + 1), xR[q], yR[q]);
        }
#pragma unroll
        for (int q = 0; q < 2; ++q)
            if (k0 + 64 * q < n) acc[q] = eadd(acc[q], cross_about<E>(xr, yr, xv[q], yv[q], xR[q], yR[q]));
    }
    __syncwarp();
#pragma unroll
    for (int q = 0; q < 2; ++q) {
        acc[q] = warp_tree<E>(acc[q], lane);
        if (lane == 0) red[(t >> 5) + 2 * q] = acc[q];
    }
    asm volatile("bar.sync %0, 64;" ::"r"(bar) : "memory");
    return emulc(eadd(eadd(eadd(red[0], red[1]), red[2]), red[3]), C(0.5));
}
// one warp: the interior elements of a chunk of kn vertices, whose positions
// pos(k, x, y) gives, about (cx, cy); in lane 0
template <typename C, typename Pos>
__device__ __forceinline__ typename Ext<C>::E chunk_area(int kn, int lane, typename Ext<C>::E cx,
                                                         typename Ext<C>::E cy, Pos pos) {
    using E = typename Ext<C>::E;
    E acc = ezero<E>();
#pragma unroll
    for (int q = 0; q < kChunkV / 32; ++q) {
        const int k = lane + 32 * q;
        if (k + 1 < kn) {
            E xa, ya, xb, yb;
            pos(k, xa, ya);
            pos(k + 1, xb, yb);
            acc = eadd(acc, cross_about<E>(cx, cy, xa, ya, xb, yb));
        }
    }
    __syncwarp();
    return warp_tree<E>(acc, lane);
}
// one warp: area of a long ring from its chunks' sums; u0: advance unit of its
// first chunk; in lane 0
template <typename C>
__device__ typename Ext<C>::E ring_area_parts(const MarkerArgs& a, int off, int n, int u0, int lane) {
    using E = typename Ext<C>::E;
    E cx, cy;
    PosIO<C>::load(a.Xp, off, cx, cy);
    E acc = ezero<E>();
    const int nchunk = (n + kChunkV - 1) / kChunkV;
    for (int i = lane; i < nchunk; i += 32) {
        const int last = i + 1 == nchunk ? n - 1 : (i + 1) * kChunkV - 1;
        E xa, ya, xb, yb, part, unused;
        load_pos<C>(a, off + last, xa, ya);
        load_pos<C>(a, off + (last == n - 1 ? 0 : last + 1), xb, yb);
        PosIO<C>::load(a.area_part, u0 + i, part, unused);
        acc = eadd(acc, eadd(part, cross_about<E>(cx, cy, xa, ya, xb, yb)));
    }
    __syncwarp();
    return emulc(warp_tree<E>(acc, lane), C(0.5));
}
// the area of ring m by warps w0, w0 + 1 (the second only helps short rings);
// valid in lane 0 of the first; au0: advance unit of its first chunk (long rings)
template <typename C>
__device__ __forceinline__ typename Ext<C>::E ring_area(const MarkerArgs& a, int off, int n, int au0, int w0,
                                                        typename Ext<C>::E* red, int bar) {
    if (n <= kDirectArea) return ring_area_direct<C>(a, off, n, w0, red, bar);
    if ((threadIdx.x >> 5) == w0) return ring_area_parts<C>(a, off, n, au0, threadIdx.x & 31);
    return ezero<typename Ext<C>::E>();
}

// N block-wide sums in the compute type at once (every thread gets all of
// them); each by a fixed shuffle tree per warp, then every thread adds the
// warps' partials in a fixed tree of eight (blocks have at most eight warps).
// One barrier: `red` is the call's own.
template <typename C, int N>
__device__ __forceinline__ void block_sum_c(C (&v)[N], C (*red)[8]) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1)
#pragma unroll
        for (int q = 0; q < N; ++q) v[q] += __shfl_down_sync(kFull, v[q], o);
    const int w = threadIdx.x >> 5, nw = blockDim.x >> 5;
    if ((threadIdx.x & 31) == 0) {
#pragma unroll
        for (int q = 0; q < N; ++q) red[q][w] = v[q];
    }
    __syncthreads();
#pragma unroll
    for (int q = 0; q < N; ++q) {
        C t[8];
#pragma unroll
        for (int k = 0; k < 8; ++k) t[k] = k < nw ? red[q][k] : C(0);
        v[q] = ((t[0] + t[4]) + (t[2] + t[6])) + ((t[1] + t[5]) + (t[3] + t[7]));
    }
}

// Boxes of the segments and of the screening group that a warp's positions
// form: lane l holds vertex l of the group; lanes g, g + 1, .. of a segment past
// its end hold a copy of its first vertex.  FP32 offsets from the segment's
// first vertex; centre x wrapped into [0, nx), and without walls centre y into
// [0, ny) (rings may lie several periods apart).  sg: this lane's segment (-1:
// none), gr: the warp's group (-1: none).  The group's box is widened by 1e-3
// (its own roundings stay below 1e-3 of a lattice unit).  All 32 lanes call it.
template <typename C>
__device__ __forceinline__ void seg_box_regs(const MarkerArgs& a, int sg, int gr, int lane, typename Ext<C>::E x,
                                             typename Ext<C>::E y) {
    using E = typename Ext<C>::E;
    const int g0 = lane & ~(kSegV - 1);
    // first vertex of the segment, broadcast in its (hi, lo) parts
    E ax, ay, wx, wy;
    shfl_e(ax, x, g0);
    shfl_e(ay, y, g0);
    const float ox = float(etoc(esub(x, ax))), oy = float(etoc(esub(y, ay)));
    float lo_x = ox, hi_x = ox, lo_y = oy, hi_y = oy;
#pragma unroll
    for (int o = kSegV / 2; o > 0; o >>= 1) {
        lo_x = fminf(lo_x, __shfl_xor_sync(kFull, lo_x, o));
        hi_x = fmaxf(hi_x, __shfl_xor_sync(kFull, hi_x, o));
        lo_y = fminf(lo_y, __shfl_xor_sync(kFull, lo_y, o));
        hi_y = fmaxf(hi_y, __shfl_xor_sync(kFull, hi_y, o));
    }
    auto wrapped_y = [&](float cy) { return cy - a.f.wrap_ny * floorf(cy * a.f.inv_ny); };
    const float Lx = a.f.nx;
    if (sg >= 0 && lane == g0) {
        const float cx = float(ehi(ax)) + 0.5f * (lo_x + hi_x);
        a.seg_box[sg] = make_float4(cx - Lx * floorf(cx * a.f.inv_nx), wrapped_y(float(ehi(ay)) + 0.5f * (lo_y + hi_y)),
                                    0.5f * (hi_x - lo_x), 0.5f * (hi_y - lo_y));
    }
    shfl_e(wx, x, 0);
    shfl_e(wy, y, 0);
    const float dx = float(etoc(esub(ax, wx))), dy = float(etoc(esub(ay, wy)));
    lo_x = sg >= 0 ? lo_x + dx : 1e30f;
    hi_x = sg >= 0 ? hi_x + dx : -1e30f;
    lo_y = sg >= 0 ? lo_y + dy : 1e30f;
    hi_y = sg >= 0 ? hi_y + dy : -1e30f;
#pragma unroll
    for (int o = kSegV; o < kGroupV; o <<= 1) {
        lo_x = fminf(lo_x, __shfl_xor_sync(kFull, lo_x, o));
        hi_x = fmaxf(hi_x, __shfl_xor_sync(kFull, hi_x, o));
        lo_y = fminf(lo_y, __shfl_xor_sync(kFull, lo_y, o));
        hi_y = fmaxf(hi_y, __shfl_xor_sync(kFull, hi_y, o));
    }
    if (gr >= 0 && lane == 0) {
        const float cx = float(ehi(wx)) + 0.5f * (lo_x + hi_x);
        a.group_box[gr] = make_float4(cx - Lx * floorf(cx * a.f.inv_nx), wrapped_y(float(ehi(wy)) + 0.5f * (lo_y + hi_y)),
                                      0.5f * (hi_x - lo_x) + 1e-3f, 0.5f * (hi_y - lo_y) + 1e-3f);
    }
}

// interpolation U_v = sum_j phi_v(x_j) u(x_j) with the weights of this step:
// the weights and the stencil origin, read ahead of the velocities (in the
// advance kernel's prologue, beside the fused kernel that writes those)
template <typename C>
struct Shape {
    C w[9];
    int i0, j0;
};
template <typename C>
__device__ __forceinline__ Shape<C> load_shape(const MarkerArgs& a, int v) {
    const C* W = static_cast<const C*>(a.W);
    Shape<C> s;
#pragma unroll
    for (int q = 0; q < 9; ++q) s.w[q] = W[9 * (size_t)v + q];
    const int2 o = reinterpret_cast<const int2*>(a.stencil)[v];
    s.i0 = o.x;
    s.j0 = o.y;
    return s;
}
// (every node is read, rows outside the walls at the row of zeros after the
// field's last: a branch per row made three round trips of one, 3400 cycles of
// the advance kernel's chain.  The nearest fluid row would not do: for a marker
// beyond a wall no stencil flagged it, and what an earlier step left there, not
// finite perhaps, does not vanish by a weight of 0.)
template <typename C>
__device__ __forceinline__ void interp_vertex(const MarkerArgs& a, const Shape<C>& s, C& Ux, C& Uy) {
    const C* ux = static_cast<const C*>(a.ux);
    const C* uy = static_cast<const C*>(a.uy);
    int i[3];
    size_t row[3];
    bool in[3];
#pragma unroll
    for (int q = 0; q < 3; ++q) {
        i[q] = s.i0 + q - 1;
        i[q] = i[q] < 0 ? i[q] + a.nx : (i[q] >= a.nx ? i[q] - a.nx : i[q]);
        int j = s.j0 + q - 1;
        in[q] = !a.walls || (j >= 0 && j < a.ny);
        j = a.walls ? (in[q] ? j : a.ny) : (j < 0 ? j + a.ny : (j >= a.ny ? j - a.ny : j));
        row[q] = (size_t)j * a.nx;
    }
    C u[9], v[9];
#pragma unroll
    for (int k = 0; k < 9; ++k) {
        u[k] = ux[row[k / 3] + i[k % 3]];
        v[k] = uy[row[k / 3] + i[k % 3]];
    }
    C sx = C(0), sy = C(0);
#pragma unroll
    for (int k = 0; k < 9; ++k) {
        const C w = in[k / 3] ? s.w[k] : C(0);
        sx += w * u[k];
        sy += w * v[k];
    }
    Ux = sx;
    Uy = sy;
}

// Eq. kinematicPos (BDF2): x^{n+1} = 2/3 (2 x^n - 1/2 x^{n-1} + U dt);
// forward Euler on the very first step
template <typename C>
__device__ __forceinline__ void bdf2(typename Ext<C>::E x, typename Ext<C>::E xp, C U, long long step,
                                     typename Ext<C>::E& xn) {
    using E = typename Ext<C>::E;
    if (step == 0) {
        xn = eaddc(x, U);
    } else {
        xn = emul(eaddc(esub(emulc(x, C(2)), emulc(xp, C(0.5))), U), two_thirds_e<E>());
    }
}

}  // namespace lbib
