// step_kernel.cuh -- the fused LBGK time step on sm_103a.
//
// One launch performs, for every fluid node of one or more lattices (Sec. 5 of the paper, in its
// order): advection by pull (Eq. 17) with bounce-back on blocked links (Eq. 12), the moments
// (Eq. 16), the Hermite equilibrium (Eq. 15 or its 4th-order continuation), the regularized
// collision (Eqs. 18-19) or the plain BGK step (Eq. 14), an optional body force, and the store.
// The momentum given to the body is summed in FP64 by warps of its own over a list of the body's links
// (bounce-back, two buffers) or of its boundary nodes (diffuse walls, in-place streaming), in groups of
// one warp and then over the groups, always in the same order; the last group to finish writes (Fx, Fy)
// of the step.  No block ever waits for another.
//
// Storage.  Populations are kept as scaled deviations from the rest state,
//     h_i = (f_i - w_i rho0) / (w_i s),
// structure-of-arrays [Q][ny][pitch].  s = 1 for FP64/FP32 storage and s = u0 (the drive
// amplitude) for BF16/FP16, so that every direction is O(1) and far from the 16-bit subnormal
// range.  The weights cancel out of the equilibrium and collision in these units.  Arithmetic is
// FP64 for FP64 storage and FP32 otherwise; the wall force is always accumulated in FP64.
#pragma once

#include "collision.cuh"

namespace lbm {

// Eq. 17 from global memory: h_i^adv(x) = h_i(x - c_i), periodic in x and y.
template <class L, class ST, bool COH = false>
__device__ __forceinline__ void gather_global(const InstDev& P, const ST* __restrict__ src, int x, int y,
                                              typename StoreT<ST>::CT (&h)[L::Q]) {
    using S = StoreT<ST>;
    constexpr int Q = L::Q, R = L::R;
    const unsigned plane = (unsigned)P.plane;  // Q * plane < 2^32 (checked at creation)
    unsigned roff[2 * R + 1], col[2 * R + 1];
#pragma unroll
    for (int d = -R; d <= R; ++d) {
        int ys = y - d;
        ys += ys < 0 ? P.ny : 0;
        ys -= ys >= P.ny ? P.ny : 0;
        int xs = x - d;
        xs += xs < 0 ? P.nx : 0;
        xs -= xs >= P.nx ? P.nx : 0;
        roff[d + R] = (unsigned)(ys * P.pitch);
        col[d + R] = (unsigned)xs;
    }
#pragma unroll
    for (int i = 0; i < Q; ++i) {
        const int cx = cx_of<L>(i), cy = cy_of<L>(i);
        // 32-bit element offset, widened once: one multiply-add per address
        const ST* p = src + (unsigned)(i * plane + roff[cy + R] + col[cx + R]);
        h[i] = COH ? S::ldc(p) : S::ld(p);
    }
}

// Where a node's own post-collision population opposite to link i is: plane opp(i) of src (two buffers,
// OWN_OPP), or plane i (in-place AA streaming, whose even steps store directions swapped, OWN_SWAPPED).
enum OwnPlane { OWN_OPP = 0, OWN_SWAPPED = 1 };

// Momentum handed over along body links, node by node: the sum of c_i w_i v_i in FP64 with c_i w_i a
// compile-time constant.  An FP64 instruction holds its SM sub-partition's FP64 unit for 64 cycles
// however few lanes are active (predicated off included), so a link that no lane of the warp has is
// skipped by a branch.
struct LinkSum {
    double x = 0.0, y = 0.0;
    // v = a + b along link i
    template <class L, class T>
    __device__ __forceinline__ void add(int i, bool has, T a, T b = (T)0) {
        if (__builtin_expect(__any_sync(__activemask(), has), 0)) {
            const double d = has ? __dadd_rn((double)a, (double)b) : 0.0;
            if (cx_of<L>(i)) x = __fma_rn(cx_of<L>(i) * w_of<L>(i), d, x);
            if (cy_of<L>(i)) y = __fma_rn(cy_of<L>(i) * w_of<L>(i), d, y);
        }
    }
};

// What arrives at the boundary node (x, y) with the links blk blocked: pulls along the open links and, in
// the same loads, the node's own opposite population for each blocked one (Eq. 12 before the wall term):
// one memory latency.
template <class L, class ST, int OWN = OWN_OPP>
__device__ __forceinline__ void gather_boundary(const InstDev& P, const ST* __restrict__ src, int x, int y,
                                                unsigned long long blk, typename StoreT<ST>::CT (&h)[L::Q]) {
    constexpr int Q = L::Q, R = L::R;
    const unsigned plane = (unsigned)P.plane;
    const unsigned idx = (unsigned)(y * P.pitch + x);
    unsigned roff[2 * R + 1], col[2 * R + 1];
#pragma unroll
    for (int d = -R; d <= R; ++d) {
        int ys = y - d;
        ys += ys < 0 ? P.ny : 0;
        ys -= ys >= P.ny ? P.ny : 0;
        int xs = x - d;
        xs += xs < 0 ? P.nx : 0;
        xs -= xs >= P.nx ? P.nx : 0;
        roff[d + R] = (unsigned)(ys * P.pitch);
        col[d + R] = (unsigned)xs;
    }
#pragma unroll
    for (int i = 0; i < Q; ++i) {
        // two buffers: pull from plane i, own from plane opp(i); in place, directions are swapped
        const int pull = OWN == OWN_SWAPPED ? opp_of<L>(i) : i, own = OWN == OWN_SWAPPED ? i : opp_of<L>(i);
        const unsigned open = pull * plane + roff[cy_of<L>(i) + R] + col[cx_of<L>(i) + R];
        h[i] = StoreT<ST>::ld(src + ((blk >> i) & 1ull ? own * plane + idx : open));
    }
}

// Eq. 12 on the blocked links lk, whose own populations are in h: the moving-wall term
// 2 w_i rho0 c_i.U_w / theta (w_i and s divided out) on the body's links, and with 16-bit storage and
// the stream offset on the change of direction's offset.  h holds values relative to the stream on
// entry, and on exit for the regularized collision; absolute ones on exit for BGK (entry: absolute
// except on the blocked links).
template <class L, class ST, int COLL>
__device__ __forceinline__ void bb_apply(const InstDev& P, ulonglong2 lk, typename StoreT<ST>::CT (&h)[L::Q]) {
    using T = typename StoreT<ST>::CT;
    const bool off = sizeof(ST) == 2 && P.stream_off;
    if (!off && !P.moving) return;
    const unsigned long long blk = lk.x | lk.y;
#pragma unroll
    for (int i = 1; i < L::Q; ++i) {
        if ((blk >> i) & 1ull) {
            T v = h[i];
            if (off) v = vadd(v, (T)off_l<L>(P, opp_of<L>(i)));
            const int cx = cx_of<L>(i), m = cx < 0 ? -cx : cx;
            if (cx && ((lk.x >> i) & 1ull)) {
                const T term = kconst<T>(P.mw[m], P.mw_f[m]);
                v = cx > 0 ? vadd(v, term) : vsub(v, term);
            }
            h[i] = off && COLL == COLL_REG ? vsub(v, (T)off_l<L>(P, i)) : v;
        }
    }
}

// Eq. 11 on the blocked links lk: each wall returns its discrete Maxwellian at the wall velocity,
// f_i = w_i rho_w (1 + e_i(U_w)), with rho_w set so that the node gets back exactly the mass it sends
// into that wall (per wall: body = bits of .x, static wall = bits of .y).  e_i depends on c_ix only, so
// what comes back is tabulated per c_ix.  Returns the momentum handed to the body.
template <class L, class ST, int COLL>
__device__ __forceinline__ double2 ds_apply(const InstDev& P, ulonglong2 lk, double dv, float dv_f,
                                            typename StoreT<ST>::CT (&h)[L::Q]) {
    using T = typename StoreT<ST>::CT;
    constexpr int Q = L::Q, R = L::R;
    const bool off = sizeof(ST) == 2 && P.stream_off;
    const unsigned long long blk = lk.x | lk.y;
    const T rho0 = kconst<T>(P.rho0, P.rho0_f), sT = kconst<T>(P.s, P.s_f);
    const T Ub = P.moving ? kconst<T>(dv, dv_f) : (T)0;
    const T ith = (T)(1.0 / L::theta()), bb = Ub * Ub * ith;
    const bool eq4 = P.eq_order >= 4;
    T eb[2 * R + 1];  // the body's e_i, index c_ix + R
#pragma unroll
    for (int cx = -R; cx <= R; ++cx) {
        const T a = (T)cx * Ub * ith;
        T e = a + (T)0.5 * (a * a - bb);
        if (eq4) e += (a * a * a - (T)3 * a * bb) * (T)(1.0 / 6.0) +
                      (a * a * a * a - (T)6 * a * a * bb + (T)3 * bb * bb) * (T)(1.0 / 24.0);
        eb[cx + R] = e;
    }
    T in[2] = {0, 0}, mw[2] = {0, 0}, se = 0;
#pragma unroll
    for (int i = 1; i < Q; ++i) {
        if ((blk >> i) & 1ull) {
            const T w = (T)w_of<L>(i);
            if (off) h[i] += (T)off_l<L>(P, opp_of<L>(i));
            if ((lk.x >> i) & 1ull) {
                in[0] += w * h[i];
                mw[0] += w;
                se += w * eb[cx_of<L>(i) + R];
            } else {
                in[1] += w * h[i];
                mw[1] += w;
            }
        }
    }
    // rho_w - rho0 of each wall, and what comes back along a link of the body (per c_ix) and of a
    // static wall (e = 0)
    const T den = mw[0] + se;
    const T dr = den > (T)0 ? (sT * in[0] - rho0 * se) / den : (T)0;
    const T rw = rho0 + dr;
#pragma unroll
    for (int cx = 0; cx <= 2 * R; ++cx) eb[cx] = (dr + rw * eb[cx]) / sT;
    const T hw = mw[1] > (T)0 ? (sT * in[1]) / mw[1] / sT : (T)0;
    LinkSum G;
#pragma unroll
    for (int i = 1; i < Q; ++i) {
        const bool blocked = (blk >> i) & 1ull, body = (lk.x >> i) & 1ull;
        const T hadv = body ? eb[cx_of<L>(i) + R] : hw;
        G.add<L>(i, body, h[i], hadv);
        if (blocked) h[i] = off && COLL == COLL_REG ? hadv - (T)off_l<L>(P, i) : hadv;
    }
    return make_double2(__dmul_rn(-P.s, G.x), __dmul_rn(-P.s, G.y));
}

// With 16-bit storage and the stream offset on the stored values are relative to the uniform stream:
// plain BGK needs every h_i, the regularized collision only their moments (HM is added to those).
// (The blocked links blk, which hold the node's own opposite populations, are left to the wall rule.)
template <class L, class ST, int COLL, class V>
__device__ __forceinline__ void add_offset(const InstDev& P, unsigned long long blk, V (&h)[L::Q]) {
    if (sizeof(ST) == 2 && COLL == COLL_BGK && P.stream_off) {
#pragma unroll
        for (int i = 0; i < L::Q; ++i)
            if (!((blk >> i) & 1ull)) h[i] = vadds(h[i], (typename Lane<V>::T)off_l<L>(P, i));
    }
}

// Moments, collision and outputs of one node (V = float, double) or two (V2) from the populations h
// that arrived at it: emit(i, v) receives output i in storage units.
template <class L, class ST, int COLL, class V, class Emit>
__device__ __forceinline__ void collide_emit(const InstDev& P, double dv, float dv_f, const V (&h)[L::Q], Emit&& emit) {
    const auto at = [&](int i) { return h[i]; };
    const Moments<V> M = moments<L, V>(at);
    if constexpr (sizeof(ST) == 8) {
        // (plain BGK: one copy of the outputs, which read the populations)
        if (COLL == COLL_BGK) {
            const Coef<V> C = P.body_force ? coefficients<L, ST, COLL, V, 1>(P, dv, dv_f, M) : coefficients<L, ST, COLL, V, 0>(P, dv, dv_f, M);
            emit_outputs<L, ST, COLL, V>(P, C, at, emit);
        } else if (P.body_force) {
            emit_outputs<L, ST, COLL, V>(P, coefficients<L, ST, COLL, V, 1>(P, dv, dv_f, M), at, emit);
        } else {
            emit_outputs<L, ST, COLL, V>(P, coefficients<L, ST, COLL, V, 0>(P, dv, dv_f, M), at, emit);
        }
    } else {
        emit_outputs<L, ST, COLL, V>(P, coefficients<L, ST, COLL, V>(P, dv, dv_f, M), at, emit);
    }
}

// The same, stored at the node's place (element offset y pitch + x).
template <class L, class ST, int COLL>
__device__ __forceinline__ void collide_store(const InstDev& P, void* dst_v, int x, int y, double dv, float dv_f,
                                              const typename StoreT<ST>::CT (&h)[L::Q]) {
    using T = typename StoreT<ST>::CT;
    // 32-bit plane stride (Q * plane < 2^32, checked at creation): each address is the node's
    // pointer plus stride * i, one widening multiply-add
    ST* __restrict__ dst = static_cast<ST*>(dst_v) + (y * P.pitch + x);
    const unsigned plane = (unsigned)P.plane;
    collide_emit<L, ST, COLL, T>(P, dv, dv_f, h, [&](int i, T v) {
        StoreT<ST>::stg(dst + (unsigned long long)plane * (unsigned)i, v);
    });
}

// A fluid node of a tile kernel, whose tile computes its boundary nodes too (bounce-back), with the pulled
// populations in h: the own populations of the blocked links (all loaded before the first is used), then
// the wall term.
template <class L, class ST, int COLL, bool COH = false>
__device__ __forceinline__ void tile_fixup(const InstDev& P, const void* src, int x, int y, int cls,
                                           typename StoreT<ST>::CT (&h)[L::Q]) {
    using S = StoreT<ST>;
    ulonglong2 lk = make_ulonglong2(0ull, 0ull);
    if (cls == NODE_BOUNDARY) {
        const int idx = y * P.pitch + x;
        lk = P.links[idx];
        const unsigned long long blk = lk.x | lk.y;
        const ST* own = static_cast<const ST*>(src) + idx;
#pragma unroll
        for (int i = 1; i < L::Q; ++i) {
            const ST* po = own + (unsigned long long)(unsigned)P.plane * (unsigned)opp_of<L>(i);
            if ((blk >> i) & 1ull) h[i] = COH ? S::ldc(po) : S::ld(po);
        }
    }
    add_offset<L, ST, COLL>(P, lk.x | lk.y, h);
    if (cls == NODE_BOUNDARY) bb_apply<L, ST, COLL>(P, lk, h);
}

template <class L, class ST, int COLL, bool COH = false>
__device__ __forceinline__ void tile_node(const InstDev& P, const void* src, void* dst, int x, int y, int cls,
                                          double dv, float dv_f, typename StoreT<ST>::CT (&h)[L::Q]) {
    tile_fixup<L, ST, COLL, COH>(P, src, x, y, cls, h);
    collide_store<L, ST, COLL>(P, dst, x, y, dv, dv_f, h);
}

// ---------------------------------------------------------------------------------------------
// force: groups of one warp, then one sum over the groups, always in the same order
// ---------------------------------------------------------------------------------------------

// Sum of (x, y) over a warp: after the first exchange the lanes 0-15 go on with x and the lanes 16-31
// with y, so that a round costs one FP64 add instead of two.  Lane 0 returns the sum of x, lane 16 that
// of y.
__device__ __forceinline__ double warp_sum2(double x, double y, int lane) {
    const bool upper = lane & 16;
    double v = upper ? y : x;
    v = __dadd_rn(v, __shfl_xor_sync(0xffffffffu, upper ? x : y, 16));
#pragma unroll
    for (int o = 8; o; o >>= 1) v = __dadd_rn(v, __shfl_down_sync(0xffffffffu, v, o, 16));
    return v;
}

// One warp: a step's force from its group partials (group g at g stride), times scale, plus what depends
// on the geometry and the drive only.  Lanes 0-15 sum the x and lanes 16-31 the y of every 16th group.
__device__ __forceinline__ void force_sum(const InstDev& P, const double2* partials, int stride, double dv,
                                          double2* force_out, double scale, int lane) {
    const double* part = reinterpret_cast<const double*>(partials) + (lane >> 4);
    double v = 0.0;
    for (int k = lane & 15; k < P.ngroups; k += 16) v = __dadd_rn(v, __ldcg(part + 2 * stride * (size_t)k));
#pragma unroll
    for (int o = 8; o; o >>= 1) v = __dadd_rn(v, __shfl_down_sync(0xffffffffu, v, o, 16));
    if ((lane & 15) == 0) {
        const bool y = lane >> 4;
        v = __fma_rn(scale, v, __fma_rn(dv, y ? P.fmov.y : P.fmov.x, y ? P.fconst.y : P.fconst.x));
        if (!isfinite(v)) atomicOr(P.err, 1);
        reinterpret_cast<double*>(force_out)[y] = v;
    }
}

// The forces of up to kForceSteps consecutive steps, whose kernels left their partials one after another
// (step k at k ngroups) and no ticket: a warp each.  The wait for a step's last group and its sum
// (fence, atomic, sum) then stay out of every step: 64^2 D2Q37 FP32 beam 4.1 -> 2.6 us a step, 256^2
// 5.3 -> 3.9, together with boundary blocks of one warp.  The sums are the same, in the same order.
constexpr int kForceSteps = 64;
struct ForceSteps {
    double dv[kForceSteps];
    double2* force_out;
    double scale;
    int n;
};

static __global__ void __launch_bounds__(128) sum_forces(const __grid_constant__ InstDev P,
                                                         const __grid_constant__ ForceSteps F) {
    const int k = blockIdx.x * 4 + (threadIdx.x >> 5);
    pdl_wait_then_release();
    if (k < F.n)
        force_sum(P, P.partials + (size_t)k * P.ngroups, 1, F.dv[k], F.force_out + k, F.scale, threadIdx.x & 31);
}

// One warp, force group g: the lanes' parts F into the group's partial; the last group of the step to
// finish sums them all (and returns true).
template <int NF>
__device__ __forceinline__ bool group_force(const InstDev& P, int g, double2* force_out, const double2 (&F)[NF],
                                            double scale, int lane) {
#pragma unroll
    for (int f = 0; f < NF; ++f) {
        const double v = warp_sum2(F[f].x, F[f].y, lane);
        if ((lane & 15) == 0) reinterpret_cast<double*>(P.partials + (size_t)g * NF + f)[lane >> 4] = v;
    }
    if (!P.ticket) return false;  // summed for several steps at once (sum_forces)
    __threadfence();
    __syncwarp();
    unsigned t = 0;
    if (lane == 0) t = atomicAdd(P.ticket, 1u);
    const bool last = __shfl_sync(0xffffffffu, t, 0) == (unsigned)(P.ngroups - 1);
    if (last) {
        __threadfence();
#pragma unroll
        for (int f = 0; f < NF; ++f) force_sum(P, P.partials + f, NF, f == 0 ? P.dv : P.dv2, force_out + f, scale, lane);
        if (lane == 0) *P.ticket = 0u;
    }
    return last;
}

// One warp, force group g of the body's links (bounce-back): momentum c_opp h_opp in and c_i h_i^adv out
// along each, -c_i w_i s (2 h_opp + moving-wall term), of which the group sums c_i w_i h_opp: two
// FP64 multiply-adds a link.  FP64 is slow here (an instruction holds its sub-partition's unit for 64
// cycles whatever its active lanes), so a warp takes 32 links at a time, whoever their nodes are, and
// the factors and the moving-wall term (geometry only) come in once per step.  `wait` runs between the
// loads of the list and those of the populations.  Lanes past the end of the list read some body
// link's population with a weight of 0, never a place that is none's: solid nodes are not written and may hold
// NaN or infinities, which that weight would not keep out of the sum.  (The group's first link for FP64, the list's
// last else, by the registers that leaves the kernels: FP64 D2Q9 384^2 26.2 us a step with the first, 30.9 with the last,
// plain FP32 D2Q9 tiles of 1024^2 12.9 and 11.6, 256^2 FP32 D2Q37 3.8 and 3.7.)
template <class L, class ST, bool COH = false, class Wait>
__device__ __forceinline__ bool link_force(const InstDev& P, const void* src_v, int g, double2* force_out, int lane,
                                           Wait&& wait) {
    using S = StoreT<ST>;
    const ST* __restrict__ src = static_cast<const ST*>(src_v);
    const bool off = sizeof(ST) == 2 && P.stream_off;
    const uint2* list = flink_entries(P.flinks);
    const double2* weights = flink_weights(P.flinks);
    double2 F[1] = {make_double2(0.0, 0.0)};
    const long long first = (long long)g * 32 * P.glen + lane;
    for (int j0 = 0; j0 < P.glen; j0 += 4) {
        uint2 e[4];
        double2 cw[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const long long k = first + 32ll * (j0 + j);
            const bool has = j0 + j < P.glen && k < P.nfl;
            if constexpr (sizeof(ST) == 8)
                e[j] = list[has ? k : (long long)g * 32 * P.glen];
            else
                e[j] = list[k < P.nfl ? k : P.nfl - 1];
            cw[j] = has ? weights[e[j].y & 0xffu] : make_double2(0.0, 0.0);
        }
        if (j0 == 0) wait();
        typename S::CT own[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) own[j] = COH ? S::ldc(src + e[j].x) : S::ld(src + e[j].x);
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            // offset of the opposite direction: index 3 - c_x
            if (off) own[j] = vadd(own[j], (typename S::CT)P.Hl[6 - (int)(e[j].y >> 8)]);
            F[0].x = __fma_rn(cw[j].x, (double)own[j], F[0].x);
            F[0].y = __fma_rn(cw[j].y, (double)own[j], F[0].y);
        }
    }
    return group_force<1>(P, g, force_out, F, -2.0 * P.s, lane);
}

// Blocks of `threads` that hold the force groups, and the f-th of them.
__host__ __device__ inline int force_blocks(int ngroups, int threads) { return (ngroups * 32 + threads - 1) / threads; }

template <class L, class ST>
__device__ __forceinline__ void force_block(const InstDev& P, int f) {
    const int tid = threadIdx.y * blockDim.x + threadIdx.x;
    const int g = f * ((blockDim.x * blockDim.y) >> 5) + (tid >> 5);
    if (g < P.ngroups)
        link_force<L, ST>(P, P.src, g, P.force_out, tid & 31, [] { pdl_wait_then_release(); });
    else
        pdl_wait_then_release();
}

// ---------------------------------------------------------------------------------------------
// boundary blocks and bulk blocks
// ---------------------------------------------------------------------------------------------
//
// The single-instance kernels compute the fluid nodes with blocked links in blocks of their own, which
// come first in the grid, one listed node per thread; the force takes further blocks (force_block); the
// others compute bulk nodes only and need no links.  With wall rule and force inside the tiles, a
// warp next to the body took every lane's links in turn, ten FP64 instructions each, and that chain was
// the step of a small grid (256^2 D2Q37 FP32, 32 x 32 beam: 18.4 us a launch, the FP64 pipe of one SM
// 89 % busy and the chip at an IPC of 1.03).  Per step, in back-to-back launches: 64^2 13.8 -> 2.6 us,
// 256^2 15.0 -> 3.9, 512^2 19.3 -> 9.2; 32 x 4096 plate 14.9 -> 5.2, with diffuse walls (force still node
// by node) 19.2 -> 7.8.

// Boundary blocks of a grid: one warp of listed nodes each (further warps leave), since their scattered
// loads are bound by the SM's L1: four warps on one SM take four times as long as on four.
__host__ __device__ inline int boundary_blocks(int nb) { return (nb + 31) / 32; }

// The b-th boundary block: listed nodes 32 b + lane.  The list and the links (host-written) are read before
// the wait for the previous step's grid.
template <class L, class ST, int COLL, int WALL>
__device__ __forceinline__ void boundary_block(const InstDev& P, int b) {
    const int lane = threadIdx.y * blockDim.x + threadIdx.x;
    const int k = 32 * b + lane;
    const bool has = lane < 32 && k < P.nb;
    const uint2 at = has ? P.bnodes[k] : make_uint2(0u, 0u);
    const ulonglong2 lk = has ? P.blinks[k] : make_ulonglong2(0ull, 0ull);
    prepare_collision<ST>();
    pdl_wait_then_release();
    if (lane >= 32 || (!WALL && !has)) return;
    double2 F[1] = {make_double2(0.0, 0.0)};
    typename StoreT<ST>::CT h[L::Q];
    gather_boundary<L, ST>(P, static_cast<const ST*>(P.src), at.x, at.y, lk.x | lk.y, h);
    add_offset<L, ST, COLL>(P, lk.x | lk.y, h);
    if (WALL) F[0] = ds_apply<L, ST, COLL>(P, lk, P.dv, P.dv_f, h);  // whole warps: votes
    else bb_apply<L, ST, COLL>(P, lk, h);
    if (has) collide_store<L, ST, COLL>(P, P.dst, at.x, at.y, P.dv, P.dv_f, h);
    if (WALL && b < P.ngroups) group_force<1>(P, b, P.force_out, F, 1.0, lane);
}

// Blocks of a grid before the bulk tiles: boundary blocks, then force blocks.  Returns true if this block
// was one of them, else its tile.
template <class L, class ST, int COLL, int WALL>
__device__ __forceinline__ bool edge_block(const InstDev& P, int threads, int& tile) {
    const int nbb = boundary_blocks(P.nb), nfb = WALL ? 0 : force_blocks(P.ngroups, threads);
    tile = (int)blockIdx.x - nbb - nfb;
    if (tile >= 0) {
        if (P.flip) tile = P.ntiles - 1 - tile;
        return false;
    }
    if ((int)blockIdx.x < nbb) boundary_block<L, ST, COLL, WALL>(P, blockIdx.x);
    else force_block<L, ST>(P, blockIdx.x - nbb);
    return true;
}

template <int WALL>
inline dim3 edge_grid(const InstDev& P, int threads) {
    return dim3(P.ntiles + boundary_blocks(P.nb) + (WALL ? 0 : force_blocks(P.ngroups, threads)));
}

// Node (x, y) inside the grid, of class cls (already loaded), in a bulk block.  With 4- and 8-byte
// storage its pulls are issued whatever the class (the pulls of any node inside the grid are in bounds,
// so they need not wait for the class test), then a bulk node collides and stores; the others load for
// nothing, a small fraction of a grid.  The 16-bit kernels, and plain BGK in FP32, run at a register budget
// where that spills, so they test the class first.
template <class L, class ST, int COLL>
__device__ __forceinline__ void bulk_node(const InstDev& P, int x, int y, int cls) {
    if ((sizeof(ST) == 2 || (sizeof(ST) == 4 && L::Q == 37 && COLL == COLL_BGK)) && cls != NODE_BULK) return;
    typename StoreT<ST>::CT h[L::Q];
    gather_global<L, ST>(P, static_cast<const ST*>(P.src), x, y, h);
    if (cls != NODE_BULK) return;
    add_offset<L, ST, COLL>(P, 0ull, h);
    collide_store<L, ST, COLL>(P, P.dst, x, y, P.dv, P.dv_f, h);
}

// A bulk block's tile of blockDim.x x blockDim.y nodes, one thread per node.  The node's class (host-
// written) is read before the wait for the previous step's grid, the populations after it.
template <class L, class ST, int COLL>
__device__ __forceinline__ void bulk_tile(const InstDev& P, int tile) {
    const int x = (tile % P.ntx) * blockDim.x + threadIdx.x;
    const int y = (tile / P.ntx) * blockDim.y + threadIdx.y;
    const bool inside = x < P.nx && y < P.ny;
    const int cls = inside ? (int)P.cls[y * P.pitch + x] : (int)NODE_SOLID;
    prepare_collision<ST>();
    pdl_wait_then_release();
    if (inside) bulk_node<L, ST, COLL>(P, x, y, cls);
}

// Single-instance step: boundary and force blocks, then one block per tile.
template <class L, class ST, int COLL, int WALL = 0>
__global__ void __launch_bounds__(512) step_kernel(const __grid_constant__ InstDev P) {
    int tile;
    if (!edge_block<L, ST, COLL, WALL>(P, blockDim.x * blockDim.y, tile)) bulk_tile<L, ST, COLL>(P, tile);
}

using StepLaunchFn = cudaError_t (*)(const InstDev& P, dim3 block, cudaStream_t stream);

// The plain step on 32 x 4 tiles with an occupancy floor: at least MINB blocks of 128 threads per
// SM, so the compiler keeps the kernel within 65536 / (128 MINB) registers per thread.  The plain
// kernel waits on its global loads; more resident warps hide more of that latency.
template <class L, class ST, int COLL, int MINB, int WALL = 0>
__global__ void __launch_bounds__(128, MINB) step_kernel_occ(const __grid_constant__ InstDev P) {
    int tile;
    if (!edge_block<L, ST, COLL, WALL>(P, 128, tile)) bulk_tile<L, ST, COLL>(P, tile);
}

// Diffuse walls: the boundary blocks' wall rule takes 128 registers, which would leave the bulk blocks at 16
// warps per SM; on tiles of 128 nodes FP32 D2Q37 is held to six blocks (the rule spills, the bulk not)
// where the bulk is what counts: 1024^2 52.1 -> 45.5 us a step, but 512^2 FP16 12.6 -> 14.0 and 32 x 4096 7.8
// -> 9.0, so from 4096 tiles on.
template <class L, class ST, int COLL, int WALL = 0>
cudaError_t launch_step(const InstDev& P, dim3 block, cudaStream_t stream) {
    if constexpr (WALL == 1 && L::Q == 37 && sizeof(ST) < 8) {
        if (block.x * block.y == 128 && P.ntiles >= 4096)
            return launch_pdl(step_kernel_occ<L, ST, COLL, 6, 1>, edge_grid<1>(P, 128), block, 0, stream, P);
    }
    return launch_pdl(step_kernel<L, ST, COLL, WALL>, edge_grid<WALL>(P, block.x * block.y), block, 0, stream, P);
}

template <class L, class ST, int COLL, int MINB>
cudaError_t launch_step_occ(const InstDev& P, dim3 block, cudaStream_t stream) {
    return launch_pdl(step_kernel_occ<L, ST, COLL, MINB>, edge_grid<0>(P, 128), block, 0, stream, P);
}

// The same on tiles of 32 x (4 NR) nodes: each thread computes NR nodes of its column, 4 rows apart,
// one at a time, so that the block's fixed costs (tile indices, launch constants) are spread over NR
// nodes.
template <class L, class ST, int COLL, int MINB, int NR>
__global__ void __launch_bounds__(128, MINB) step_kernel_occn(const __grid_constant__ InstDev P) {
    int t;
    if (edge_block<L, ST, COLL, 0>(P, 128, t)) return;
    pdl_wait_then_release();
    const int x = (t % P.ntx) * 32 + threadIdx.x;
    const int y0 = (t / P.ntx) * (4 * NR) + threadIdx.y;
#pragma unroll 1
    for (int r = 0; r < NR; ++r) {
        const int y = y0 + 4 * r;
        if (x < P.nx && y < P.ny) bulk_node<L, ST, COLL>(P, x, y, (int)P.cls[y * P.pitch + x]);
    }
}

template <class L, class ST, int COLL, int MINB, int NR>
cudaError_t launch_step_occn(const InstDev& P, dim3, cudaStream_t stream) {
    return launch_pdl(step_kernel_occn<L, ST, COLL, MINB, NR>, edge_grid<0>(P, 128), dim3(32, 4), 0, stream, P);
}

// Launchers for (lattice Q, storage, collision); nullptr if the combination is not built.
StepLaunchFn find_step_launcher(int Q, int storage, int coll, int wall = 0);
// Plain step with an occupancy floor: variant 1 = 6 blocks of 128 per SM, 2 = 7; 3, 4 = 7 blocks with
// 2 or 4 nodes per thread (nullptr if not built).
StepLaunchFn find_occ_launcher(int Q, int storage, int coll, int variant);
// The direct kernel of a variant (1-4, 30, 31), nullptr if not built.
StepLaunchFn find_direct_launcher(int Q, int storage, int coll, int variant);

}  // namespace lbm
