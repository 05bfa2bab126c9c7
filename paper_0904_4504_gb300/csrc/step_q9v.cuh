// step_q9v.cuh -- the D2Q9 step, several neighbouring nodes per thread: four with 16-bit storage, two with
// FP32.
//
// With nine populations per node the D2Q9 step does little arithmetic per byte, so the one-node-
// per-thread kernels spend most of their instructions on addressing, per-element loads, stores and
// conversions.  Here each thread owns N x-neighbouring nodes (x0 .. x0 + N - 1, x0 a multiple of N, so
// 8-byte aligned in every row of every plane): per direction it loads the N stored values of its source
// row with one 8-byte load and the value shifted in by c_x = +1 or -1 with a single one, evaluates the
// collision of two nodes at a time (V2), and stores the N outputs of each direction with one 8-byte store.  A warp
// covers 32 N nodes of one row, a block 32 N x 4.  Nodes with blocked links are left to the boundary
// blocks.
#pragma once

#include "step_kernel.cuh"

namespace lbm {

// N stored values in one 8-byte word.
template <class ST> struct Vec8 {
    static constexpr int N = 4;
    using H = Half16<ST>;
    using One = unsigned short;  // one stored value
    uint2 v;
    __device__ __forceinline__ void load(const ST* p) { v = *reinterpret_cast<const uint2*>(p); }
    static __device__ __forceinline__ float value(One o) { return H::lo((unsigned)o); }
    __device__ __forceinline__ float get(int e) const {
        return e == 0 ? H::lo(v.x) : e == 1 ? H::hi(v.x) : e == 2 ? H::lo(v.y) : H::hi(v.y);
    }
    __device__ __forceinline__ void set(int e, One o) {  // e >= 1
        if (e == 1) v.x = (v.x & 0xffffu) | (unsigned)o << 16;
        if (e == 2) v.y = (v.y & 0xffff0000u) | (unsigned)o;
        if (e == 3) v.y = (v.y & 0xffffu) | (unsigned)o << 16;
    }
    __device__ __forceinline__ void put(int pr, V2 a) { (pr == 0 ? v.x : v.y) = H::pack(a.x, a.y); }
    __device__ __forceinline__ void store(ST* p) const { *reinterpret_cast<uint2*>(p) = v; }
    __device__ __forceinline__ void store1(ST* p, int e) const {
        reinterpret_cast<One*>(p)[e] = (One)((e < 2 ? v.x : v.y) >> (16 * (e & 1)));
    }
};
template <> struct Vec8<float> {
    static constexpr int N = 2;
    using One = float;
    float2 v;
    __device__ __forceinline__ void load(const float* p) { v = *reinterpret_cast<const float2*>(p); }
    static __device__ __forceinline__ float value(One o) { return o; }
    __device__ __forceinline__ float get(int e) const { return e == 0 ? v.x : v.y; }
    __device__ __forceinline__ void set(int, One o) { v.y = o; }
    __device__ __forceinline__ void put(int, V2 a) { v = make_float2(a.x, a.y); }
    __device__ __forceinline__ void store(float* p) const { *reinterpret_cast<float2*>(p) = v; }
    __device__ __forceinline__ void store1(float* p, int e) const { p[e] = e == 0 ? v.x : v.y; }
};

// The source rows of one thread's nodes: per direction the stored values of its pulled row and the one
// shifted in by c_x (h(x0 - 1) for c_x = +1, h(x0 + N) for c_x = -1).
template <class ST>
struct Q9Row {
    Vec8<ST> w[9];
    typename Vec8<ST>::One sh[9];
};

// Loads of the row y of a thread's nodes.  The value shifted in is a load of its own, from the line the
// neighbouring lane reads anyway: no lane depends on another's load, and the seam is only another address.
template <class ST>
__device__ __forceinline__ void q9v_load(const InstDev& P, int x0, int y, Q9Row<ST>& R) {
    using L = D2Q9;
    using W = Vec8<ST>;
    using One = typename W::One;
    constexpr int N = W::N;
    const int nx = P.nx, ny = P.ny;
    const unsigned long long plane = (unsigned)P.plane;
    const int xl = x0 == 0 ? nx - 1 : x0 - 1;   // neighbour columns (periodic)
    const int xr = x0 + N >= nx ? x0 + N - nx : x0 + N;
    const bool ragged = x0 + N > nx;            // the row ends inside this vector
    const One* row[3];                          // source row of c_y = -1, 0, +1
#pragma unroll
    for (int d = -1; d <= 1; ++d) {
        int r = y - d;
        r += r < 0 ? ny : 0;
        r -= r >= ny ? ny : 0;
        row[d + 1] = static_cast<const One*>(P.src) + (unsigned)(r * P.pitch);
    }
#pragma unroll
    for (int i = 0; i < 9; ++i) {
        const int cx = cx_of<L>(i);
        const One* r = row[cy_of<L>(i) + 1];
        R.w[i].load(reinterpret_cast<const ST*>(r + x0 + plane * (unsigned)i));
        R.sh[i] = cx == 1 ? (r + xl)[plane * (unsigned)i] : cx == -1 ? (r + xr)[plane * (unsigned)i] : One{};
        if (cx == -1 && ragged) R.w[i].set(nx - x0, r[plane * (unsigned)i]);  // the element after the last node is column 0
    }
}

// Collision and store of a thread's nodes of row y from their loaded source rows; cls: their classes, a
// byte each (bulk nodes only: a vector holding others stores its bulk nodes one by one).
template <class ST, int COLL>
__device__ __forceinline__ void q9v_compute(const InstDev& P, int x0, int y, unsigned cls, const Q9Row<ST>& R) {
    using L = D2Q9;
    using W = Vec8<ST>;
    constexpr int Q = 9, N = W::N;
    const unsigned long long plane = (unsigned)P.plane;
    ST* __restrict__ dst = static_cast<ST*>(P.dst) + (unsigned)(y * P.pitch + x0);
    W o[Q];
    // value of direction i pulled to node j of this thread
    auto pulled = [&](int i, int j) -> float {
        const int e = j - cx_of<L>(i);  // element of the loaded vector, -1 or N: the shifted-in one
        return e < 0 || e >= N ? W::value(R.sh[i]) : R.w[i].get(e);
    };
#pragma unroll
    for (int pr = 0; pr < N / 2; ++pr) {
        V2 h[Q];
#pragma unroll
        for (int i = 0; i < Q; ++i) h[i] = V2{pulled(i, 2 * pr), pulled(i, 2 * pr + 1)};
        add_offset<L, ST, COLL>(P, 0ull, h);
        collide_emit<L, ST, COLL, V2>(P, P.dv, P.dv_f, h, [&](int i, V2 v) { o[i].put(pr, v); });
    }
    if (cls == 0u) {
#pragma unroll
        for (int i = 0; i < Q; ++i) o[i].store(dst + plane * (unsigned)i);
    } else {
#pragma unroll
        for (int i = 0; i < Q; ++i) {
#pragma unroll
            for (int j = 0; j < N; ++j)
                if (((cls >> (8 * j)) & 0xffu) == NODE_BULK) o[i].store1(dst + plane * (unsigned)i, j);
        }
    }
}

template <class ST, int COLL, int MINB>
__global__ void __launch_bounds__(128, MINB) step_kernel_q9v(const __grid_constant__ InstDev P) {
    constexpr int N = Vec8<ST>::N;
    constexpr unsigned solid = N == 4 ? 0x01010101u : 0x0101u;  // NODE_SOLID x N
    int t;
    if (edge_block<D2Q9, ST, COLL, 0>(P, 128, t)) return;
    const int lane = threadIdx.x;
    const int x0 = (t % P.ntx) * (32 * N) + N * lane;
    const int y = (t / P.ntx) * 4 + threadIdx.y;
    // classes (host-written; a row's padding is solid, so the last vector of a row never stores past it)
    unsigned cls = solid;
    if (y < P.ny && x0 < P.nx) {
        const uint8_t* c = P.cls + (size_t)y * P.pitch + x0;
        cls = N == 4 ? *reinterpret_cast<const unsigned*>(c) : (unsigned)*reinterpret_cast<const unsigned short*>(c);
    }
    pdl_wait_then_release();
    if (y >= P.ny || x0 >= P.nx) return;
    Q9Row<ST> R;
    q9v_load<ST>(P, x0, y, R);
    if (cls != solid) q9v_compute<ST, COLL>(P, x0, y, cls, R);
}

template <class ST, int COLL, int MINB>
cudaError_t launch_step_q9v(const InstDev& P, dim3, cudaStream_t stream) {
    return launch_pdl(step_kernel_q9v<ST, COLL, MINB>, edge_grid<0>(P, 128), dim3(32, 4), 0, stream, P);
}

}  // namespace lbm
