// step_q37v.cuh -- the D2Q37 step with 16-bit storage, two neighbouring nodes per thread.
//
// With one node per thread the 16-bit step is bound by instruction issue: 37 two-byte loads, conversions,
// address computations and two-byte stores a node around the collision, about 760 instructions a node
// where HBM leaves room for about 440 (2048^2 FP16: 141 us a step, 0.65 of the copy bandwidth, at an IPC
// of 2.8 of 4).  Here a thread owns the nodes (x0, x0 + 1), x0 even: a direction with even c_x has both
// values in one aligned word of its source row, one with odd c_x the upper half of one word and the lower
// half of the next; the collision runs on both nodes at once (V2, packed FP32 operations); an output is
// one conversion and one 4-byte store for both: about 510 instructions a node (regularized collision; plain
// BGK needs the populations again for its outputs, 168 registers, and gains nothing).
//
// Two forms.  Direct (variant 31): the 57 loads of a thread are independent and all in flight at once; 96
// registers, 20 warps per SM.  Staged (variant 32): bulk tensor copies bring a block's rows to shared
// memory; more bytes in flight, but block by block.  Measured, us a step (direct / staged / one node per
// thread): 256^2 4.6 / 5.1 / 4.7, 512^2 7.6 / 10.4 / 8.7, 768^2 13.8 / 15.8 / 17.9, 1024^2 26.8 / 27.5 / 33.6, 1280^2
// 42.2 / 40.9 / 51.7, 2048^2 105 / 94 / 142.  So a single simulation stages when its two buffers hold more than about
// 200 MB, well past the L2; a batch of instances, which keeps the SMs full whatever a launch's ramp, nearly
// always does (64 instances of 256 to 1024 a side: 757 us a step staged, 807 direct, 865 one node per thread).
// pair_variant (runtime.h) draws the lines, narrow and small grids included.
#pragma once

#include "step_tma.cuh"

namespace lbm {

// The words a thread's two nodes read: direction i of the pair is (lower, upper) half of a for even c_x,
// (upper half of a, lower half of b) for odd c_x.
template <class L>
struct PairWords {
    unsigned a[L::Q], b[L::Q];
};

template <class L, class ST>
__device__ __forceinline__ V2 pair_value(const PairWords<L>& W, int i) {
    using H = Half16<ST>;
    return cx_of<L>(i) & 1 ? V2{H::hi(W.a[i]), H::lo(W.b[i])} : V2{H::lo(W.a[i]), H::hi(W.a[i])};
}

// Plain loads, or (COH) weak loads that never take the read-only path (see StoreT::ldc).
template <bool COH>
__device__ __forceinline__ unsigned load_word(const unsigned* p) {
    if (!COH) return *p;
    unsigned v;
    asm volatile("ld.global.ca.b32 %0, [%1];" : "=r"(v) : "l"(p));
    return v;
}
template <bool COH>
__device__ __forceinline__ unsigned load_half(const unsigned short* p) {
    if (!COH) return *p;
    unsigned short v;
    asm volatile("ld.global.ca.u16 %0, [%1];" : "=h"(v) : "l"(p));
    return v;
}

// Away from the seam the words lie at compile-time offsets from the node's place in the source row, one
// widening multiply-add per direction; threads within the reach of the seam read value by value.
template <class L, class ST, bool COH = false>
__device__ __forceinline__ void pair_load(const InstDev& P, int x0, int y, PairWords<L>& W) {
    constexpr int R = L::R;
    const unsigned char* __restrict__ src = static_cast<const unsigned char*>(P.src);
    const unsigned plane2 = 2u * (unsigned)P.plane;  // bytes of a plane (Q * plane < 2^32 elements)
    const int nx = P.nx, ny = P.ny;
    const unsigned char* row[2 * R + 1];  // source row of c_y = -R..R
#pragma unroll
    for (int d = -R; d <= R; ++d) {
        int ys = y - d;
        ys += ys < 0 ? ny : 0;
        ys -= ys >= ny ? ny : 0;
        row[d + R] = src + 2ull * (unsigned)(ys * P.pitch);
    }
    if (x0 >= 4 && x0 + 6 <= nx) {
#pragma unroll
        for (int d = 0; d <= 2 * R; ++d) row[d] += 2u * (unsigned)x0;
#pragma unroll
        for (int i = 0; i < L::Q; ++i) {
            const int cx = cx_of<L>(i);
            const unsigned* w = reinterpret_cast<const unsigned*>(row[cy_of<L>(i) + R] + (unsigned long long)plane2 * (unsigned)i);
            // odd c_x: the first node's element x0 - cx is the upper half of the word before it
            W.a[i] = load_word<COH>(w + (cx & 1 ? (-cx - 1) / 2 : -cx / 2));
            W.b[i] = cx & 1 ? load_word<COH>(w + (-cx + 1) / 2) : 0u;
        }
    } else {
        unsigned xs[2 * R + 2];  // columns x0 - R .. x0 + R + 1, periodic
#pragma unroll
        for (int d = -R; d <= R + 1; ++d) {
            int e = x0 + d;
            e += e < 0 ? nx : 0;
            e -= e >= nx ? nx : 0;
            xs[d + R] = (unsigned)e;
        }
#pragma unroll
        for (int i = 0; i < L::Q; ++i) {
            const int cx = cx_of<L>(i);
            const unsigned short* r = reinterpret_cast<const unsigned short*>(row[cy_of<L>(i) + R] + (unsigned long long)plane2 * (unsigned)i);
            const unsigned v0 = load_half<COH>(r + xs[R - cx]), v1 = load_half<COH>(r + xs[R - cx + 1]);
            W.a[i] = cx & 1 ? v0 << 16 : v0 | v1 << 16;
            W.b[i] = v1;
        }
    }
}

// Collision and store of a pair of row y from its words; cls: the two classes, a byte each (bulk nodes only).
template <class L, class ST, int COLL>
__device__ __forceinline__ void pair_compute(const InstDev& P, int x0, int y, unsigned cls, const PairWords<L>& W) {
    using H = Half16<ST>;
    const bool off = COLL == COLL_BGK && P.stream_off;
    const auto at = [&](int i) {
        const V2 v = pair_value<L, ST>(W, i);
        return off ? vadds(v, off_l<L>(P, i)) : v;
    };
    const Coef<V2> C = coefficients<L, ST, COLL, V2>(P, P.dv, P.dv_f, moments<L, V2>(at));
    unsigned char* __restrict__ dst = static_cast<unsigned char*>(P.dst) + 2ull * (unsigned)(y * P.pitch + x0);
    const unsigned plane2 = 2u * (unsigned)P.plane;
    if (cls == 0u) {
        // (no memory clobber before the last store: where P lies in shared memory -- the persistent batch kernel --
        // its constants would be read again after each, 903 us a step of 64 instances instead of 881)
        emit_outputs<L, ST, COLL, V2>(P, C, at, [&](int i, V2 v) {
            asm volatile("st.global.b32 [%0], %1;" ::"l"(dst + (unsigned long long)plane2 * (unsigned)i), "r"(H::pack(v.x, v.y)));
        });
        asm volatile("" ::: "memory");
    } else {
        // one of the two is a bulk node: its half of each word
        const bool first = (cls & 0xffu) == NODE_BULK;
        emit_outputs<L, ST, COLL, V2>(P, C, at, [&](int i, V2 v) {
            const unsigned w = H::pack(v.x, v.y);
            unsigned short* p = reinterpret_cast<unsigned short*>(dst + (unsigned long long)plane2 * (unsigned)i);
            if (first) *p = (unsigned short)w;
            else p[1] = (unsigned short)(w >> 16);
        });
    }
}

// Whether a pair holds a bulk node.
__device__ __forceinline__ bool pair_bulk(unsigned cls) { return (cls & 0xffu) == NODE_BULK || cls >> 8 == NODE_BULK; }

// The words of a pair from a staged tile of box width G::BW: row j, columns 2 tx, 2 tx + 1 of the tile.
template <class G, class L>
__device__ __forceinline__ void pair_stage(const unsigned char* stage, int tx, int j, PairWords<L>& W) {
    const unsigned char* base = stage + 2 * (j * G::BW + G::PAD) + 4 * tx;
#pragma unroll
    for (int i = 0; i < L::Q; ++i) {
        const int cx = cx_of<L>(i);
        const unsigned* w = reinterpret_cast<const unsigned*>(base + i * G::SLOT);
        W.a[i] = cx & 1 ? w[(-cx - 1) / 2] : w[-cx / 2];
        W.b[i] = cx & 1 ? w[(-cx + 1) / 2] : 0u;
    }
}

// Grid: blocks along x; along y (and z, 32768 rows each) first the rows of edge blocks, then the
// grid's rows, so that a block's row is its block index and needs no division.
constexpr int kPairGridRows = 32768;
inline int pair_edge_rows(const InstDev& P, int ntx, int threads) {
    const int n = boundary_blocks(P.nb) + force_blocks(P.ngroups, threads);
    return (n + ntx - 1) / ntx;
}

template <class L, class ST, int COLL, int BT, int MINB>
__global__ void __launch_bounds__(BT, MINB) step_kernel_pair16(const __grid_constant__ InstDev P, int edge_rows) {
    const int r = blockIdx.z * kPairGridRows + blockIdx.y;
    if (r < edge_rows) {
        const int e = r * gridDim.x + blockIdx.x, nbb = boundary_blocks(P.nb);
        if (e < nbb) boundary_block<L, ST, COLL, 0>(P, e);
        else force_block<L, ST>(P, e - nbb);
        return;
    }
    const int y = P.flip ? P.ny - 1 - (r - edge_rows) : r - edge_rows;
    const int x0 = blockIdx.x * (2 * BT) + 2 * threadIdx.x;
    // classes (host-written; a row's padding is solid) before the wait for the previous step's grid
    const bool inside = x0 < P.nx && y >= 0 && y < P.ny;
    unsigned cls = 0x0101u;
    if (inside) cls = *reinterpret_cast<const unsigned short*>(P.cls + y * P.pitch + x0);
    pdl_wait_then_release();
    if (!inside) return;
    // the pulls of any node inside the grid are in bounds: they do not wait for the class
    PairWords<L> W;
    pair_load<L, ST>(P, x0, y, W);
    if (pair_bulk(cls)) pair_compute<L, ST, COLL>(P, x0, y, cls, W);
}

template <class L, class ST, int COLL, int BT, int MINB>
cudaError_t launch_pair16(const InstDev& P, cudaStream_t stream) {
    const int ntx = (P.nx + 2 * BT - 1) / (2 * BT);
    const int er = pair_edge_rows(P, ntx, BT), rows = er + P.ny;
    const dim3 grid(ntx, rows < kPairGridRows ? rows : kPairGridRows, (rows + kPairGridRows - 1) / kPairGridRows);
    return launch_pdl(step_kernel_pair16<L, ST, COLL, BT, MINB>, grid, dim3(BT), 0, stream, P, er);
}

// Rows shorter than 512 nodes take blocks of one warp (64 nodes), so that at most an eighth of the lanes
// of a long row idle (the two compared in this kernel's first form: 256^2 4.75 us a step against 5.09, 1024^2 30.3
// against 29.9).
template <class L, class ST, int COLL>
cudaError_t launch_step_pair16(const InstDev& P, dim3, cudaStream_t stream) {
    return P.nx < 512 ? launch_pair16<L, ST, COLL, 32, 20>(P, stream) : launch_pair16<L, ST, COLL, 64, 10>(P, stream);
}

// The same, staged: a block of BT threads computes NR rows of 2 BT nodes, whose populations are copied to
// shared memory by one set of Q bulk tensor copies; a pair's words then lie at compile-time offsets, and
// the copies of the resident blocks keep far more bytes in flight than registers could.  Tiles at the
// grid's edges load as above.
template <class L, class ST, int COLL, int BT, int NR, int MINB>
__global__ void __launch_bounds__(BT, MINB) step_kernel_pair16s(const __grid_constant__ InstDev P,
                                                                const __grid_constant__ CUtensorMap map, int edge_rows) {
    using G = TmaGeom<L, ST, 1, 2 * BT, NR>;
    extern __shared__ __align__(128) unsigned char smem[];
    __shared__ __align__(8) uint64_t bar;
    const int r = blockIdx.z * kPairGridRows + blockIdx.y;
    if (r < edge_rows) {
        const int e = r * gridDim.x + blockIdx.x, nbb = boundary_blocks(P.nb);
        if (e < nbb) boundary_block<L, ST, COLL, 0>(P, e);
        else force_block<L, ST>(P, e - nbb);
        return;
    }
    const int tx0 = blockIdx.x * (2 * BT), nty = (P.ny + NR - 1) / NR;
    const int y0 = (P.flip ? nty - 1 - (r - edge_rows) : r - edge_rows) * NR;
    if (y0 < 0) {  // past the last row of blocks (grids of several z)
        pdl_wait_then_release();
        return;
    }
    const int x0 = tx0 + 2 * threadIdx.x;
    const bool interior = tx0 >= L::R && tx0 + 2 * BT + L::R <= P.nx && y0 >= L::R && y0 + NR + L::R <= P.ny;
    unsigned cls[NR];
#pragma unroll
    for (int j = 0; j < NR; ++j) {
        cls[j] = 0x0101u;
        if (x0 < P.nx && y0 + j < P.ny) cls[j] = *reinterpret_cast<const unsigned short*>(P.cls + (y0 + j) * P.pitch + x0);
    }
    if (interior && threadIdx.x == 0) {
        mbar_init(&bar, 1);
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    }
    pdl_wait_then_release();
    if (interior) {
        if (threadIdx.x == 0) {
            mbar_expect_tx(&bar, (unsigned)(L::Q * G::BOX_BYTES));
#pragma unroll
            for (int i = 0; i < L::Q; ++i) tma_load_3d(smem + i * G::SLOT, &map, tx0 - G::PAD, y0 - cy_of<L>(i), i, &bar);
        }
        __syncthreads();
        const bool ok = mbar_wait(&bar, 0, kTmaWaitLimit);
        if (!__syncthreads_and(ok)) {
            if (threadIdx.x == 0) {
                atomicOr(P.err, 4);
                mbar_wait(&bar, 0, kTmaWaitLimit);
            }
            __syncthreads();
            return;
        }
    }
#pragma unroll 1
    for (int j = 0; j < NR; ++j) {
        const unsigned c = cls[0];
#pragma unroll
        for (int q = 0; q + 1 < NR; ++q) cls[q] = cls[q + 1];
        if (!pair_bulk(c)) continue;
        PairWords<L> W;
        if (interior) pair_stage<G, L>(smem, threadIdx.x, j, W);
        else pair_load<L, ST>(P, x0, y0 + j, W);
        pair_compute<L, ST, COLL>(P, x0, y0 + j, c, W);
    }
}

template <class L, class ST, int COLL, int BT, int NR, int MINB>
cudaError_t launch_step_pair16s(const InstDev& P, const CUtensorMap& map, const CUtensorMap&, cudaStream_t stream) {
    using G = TmaGeom<L, ST, 1, 2 * BT, NR>;
    static bool attr = false;
    if (!attr) {
        cudaError_t e = cudaFuncSetAttribute(step_kernel_pair16s<L, ST, COLL, BT, NR, MINB>,
                                             cudaFuncAttributeMaxDynamicSharedMemorySize, G::SMEM);
        if (e != cudaSuccess) return e;
        attr = true;
    }
    const int er = pair_edge_rows(P, P.ntx, BT), rows = er + (P.ny + NR - 1) / NR;
    const dim3 grid(P.ntx, rows < kPairGridRows ? rows : kPairGridRows, (rows + kPairGridRows - 1) / kPairGridRows);
    return launch_pdl(step_kernel_pair16s<L, ST, COLL, BT, NR, MINB>, grid, dim3(BT), G::SMEM, stream, P, map, er);
}

}  // namespace lbm
