// step_q9v.cuh -- the D2Q9 step with 16-bit storage, four neighbouring nodes per thread.
//
// With nine populations per node the D2Q9 step does little arithmetic per byte, so the one-node-
// per-thread kernels spend most of their instructions on addressing, per-element loads, stores and
// conversions and are bound by instruction issue, not by HBM.  Here each thread owns four
// x-neighbouring nodes (x0 .. x0 + 3, x0 a multiple of 4, so 8-byte aligned in every row of every
// plane): per direction it loads the four stored values of its source row with one 8-byte load,
// takes the value shifted in by c_x = +1 or -1 from the neighbouring lane (warp shuffle) or, at a
// warp's ends and the periodic seam, with one 2-byte load, evaluates the collision of two nodes at a
// time (V2), and stores the four outputs of each direction with one 8-byte store.  A warp covers 128
// nodes of one row, a block 128 x 4.  Nodes with blocked links are left to the boundary blocks.
#pragma once

#include "step_kernel.cuh"

namespace lbm {

// The source rows of one thread's four nodes: per direction the four stored values of its pulled
// row (w0: elements 0, 1; w1: elements 2, 3) and the value shifted in by c_x (h(x0 - 1) for
// c_x = +1, h(x0 + 4) for c_x = -1).
struct Q9Row {
    unsigned w0[9], w1[9];
    unsigned short sh[9];
};

// Loads of the row y of a thread's nodes x0 .. x0 + 3 (warp-uniform y: the shuffles need the whole
// warp; `any`: this thread owns a node inside the grid).
template <class ST>
__device__ __forceinline__ void q9v_load(const InstDev& P, int x0, int y, int lane, bool any, Q9Row& R) {
    using L = D2Q9;
    const ST* __restrict__ src = static_cast<const ST*>(P.src);
    const unsigned plane = (unsigned)P.plane;
    const int nx = P.nx, ny = P.ny, pitch = P.pitch;
    int ys[3];  // source row of c_y = -1, 0, +1
#pragma unroll
    for (int d = -1; d <= 1; ++d) {
        int r = y - d;
        r += r < 0 ? ny : 0;
        r -= r >= ny ? ny : 0;
        ys[d + 1] = r;
    }
    const int xl = x0 == 0 ? nx - 1 : x0 - 1;   // left neighbour column (periodic)
    const int xr = x0 + 4 >= nx ? x0 + 4 - nx : x0 + 4;
    const bool edge_l = lane == 0 || x0 == 0;
    const bool edge_r = lane == 31 || x0 + 4 >= nx;
#pragma unroll
    for (int i = 0; i < 9; ++i) {
        const int cx = cx_of<L>(i), cy = cy_of<L>(i);
        const unsigned rowoff = (unsigned)(i * plane + ys[cy + 1] * pitch);
        uint2 v = make_uint2(0u, 0u);
        if (any) v = *reinterpret_cast<const uint2*>(src + rowoff + x0);
        R.w0[i] = v.x;
        R.w1[i] = v.y;
        if (cx == 1) {
            const unsigned up = __shfl_up_sync(0xffffffffu, v.y, 1);
            unsigned short s = (unsigned short)(up >> 16);
            if (edge_l && any) s = *reinterpret_cast<const unsigned short*>(src + rowoff + xl);
            R.sh[i] = s;
        } else if (cx == -1) {
            const unsigned dn = __shfl_down_sync(0xffffffffu, v.x, 1);
            unsigned short s = (unsigned short)(dn & 0xffffu);
            if (edge_r && any && x0 + 4 <= nx) s = *reinterpret_cast<const unsigned short*>(src + rowoff + xr);
            R.sh[i] = s;
            if (any && x0 + 4 > nx) {
                // the row ends inside this vector: the element after its last node is column 0
                const unsigned c0 = *reinterpret_cast<const unsigned short*>(src + rowoff);
                const int r = nx - x0;  // 1..3
                if (r == 1) R.w0[i] = (R.w0[i] & 0xffffu) | (c0 << 16);
                if (r == 2) R.w1[i] = (R.w1[i] & 0xffff0000u) | c0;
                if (r == 3) R.w1[i] = (R.w1[i] & 0xffffu) | (c0 << 16);
            }
        } else {
            R.sh[i] = 0;
        }
    }
}

// Collision and store of a thread's four nodes of row y from their loaded source rows (bulk nodes only:
// a vector holding others stores its bulk nodes one by one).
template <class ST, int COLL>
__device__ __forceinline__ void q9v_compute(const InstDev& P, int x0, int y, unsigned cls4, const Q9Row& R) {
    using L = D2Q9;
    using H = Half16<ST>;
    constexpr int Q = 9;
    const unsigned plane = (unsigned)P.plane;
    ST* __restrict__ dst = static_cast<ST*>(P.dst) + (size_t)y * P.pitch + x0;
    unsigned o[2][Q];
    // value of direction i pulled to node j (0..3) of this thread
    auto pulled = [&](int i, int j) -> float {
        const int cx = cx_of<L>(i);
        const int e = j - cx;  // element of the loaded vector, -1 or 4: the shifted-in one
        if (e < 0 || e > 3) return H::lo((unsigned)R.sh[i]);
        return e == 0 ? H::lo(R.w0[i]) : e == 1 ? H::hi(R.w0[i]) : e == 2 ? H::lo(R.w1[i]) : H::hi(R.w1[i]);
    };
#pragma unroll
    for (int pr = 0; pr < 2; ++pr) {
        V2 h[Q];
#pragma unroll
        for (int i = 0; i < Q; ++i) h[i] = V2{pulled(i, 2 * pr), pulled(i, 2 * pr + 1)};
        add_offset<L, ST, COLL>(P, 0ull, h);
        collide_emit<L, ST, COLL, V2>(P, P.dv, P.dv_f, h, [&](int i, V2 v) { o[pr][i] = H::pack(v.x, v.y); });
    }
    if (cls4 == 0u) {
#pragma unroll
        for (int i = 0; i < Q; ++i) *reinterpret_cast<uint2*>(dst + (size_t)i * plane) = make_uint2(o[0][i], o[1][i]);
    } else {
#pragma unroll
        for (int i = 0; i < Q; ++i) {
            unsigned short* p = reinterpret_cast<unsigned short*>(dst + (size_t)i * plane);
#pragma unroll
            for (int j = 0; j < 4; ++j)
                if (((cls4 >> (8 * j)) & 0xffu) == NODE_BULK) p[j] = (unsigned short)(o[j >> 1][i] >> (16 * (j & 1)));
        }
    }
}

// NR rows per thread, 4 apart (tiles of 128 x 4 NR nodes): the loads of all NR rows are issued
// before the first row is computed, so that more bytes are in flight per thread.
template <class ST, int COLL, int NR, int MINB>
__global__ void __launch_bounds__(128, MINB) step_kernel_q9v(const __grid_constant__ InstDev P) {
    int t;
    if (edge_block<D2Q9, ST, COLL, 0>(P, 128, t)) return;
    const int lane = threadIdx.x;
    const int x0 = (t % P.ntx) * 128 + 4 * lane;
    const int y0 = (t / P.ntx) * (4 * NR) + threadIdx.y;
    unsigned cls4[NR];
#pragma unroll
    for (int r = 0; r < NR; ++r) {
        const int y = y0 + 4 * r;
        cls4[r] = 0x01010101u;  // NODE_SOLID x 4
        if (y < P.ny && x0 < P.nx) cls4[r] = *reinterpret_cast<const unsigned*>(P.cls + (size_t)y * P.pitch + x0);
    }
    pdl_wait_then_release();
    Q9Row R[NR];
#pragma unroll
    for (int r = 0; r < NR; ++r) {
        const int y = y0 + 4 * r;
        if (y < P.ny) q9v_load<ST>(P, x0, y, lane, x0 < P.nx, R[r]);  // warp-uniform row test
    }
#pragma unroll
    for (int r = 0; r < NR; ++r) {
        const int y = y0 + 4 * r;
        // (a row's padding is solid, so the last vector of a row never stores past it)
        if (y < P.ny && x0 < P.nx && cls4[r] != 0x01010101u) q9v_compute<ST, COLL>(P, x0, y, cls4[r], R[r]);
    }
}

template <class ST, int COLL, int NR, int MINB>
cudaError_t launch_step_q9v(const InstDev& P, dim3, cudaStream_t stream) {
    return launch_pdl(step_kernel_q9v<ST, COLL, NR, MINB>, edge_grid<0>(P, 128), dim3(32, 4), 0, stream, P);
}

}  // namespace lbm
