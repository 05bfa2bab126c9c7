// step_tma.cuh -- the fused step with TMA-staged tile loads (sm_103a).
//
// A block computes a tile of BX x BY nodes.  For a tile that lies at least the lattice reach inside
// the grid, one thread issues Q bulk tensor copies (cp.async.bulk.tensor.3d, one box per direction
// plane): box i is the BY rows y0 - c_iy .. and the BX + 2 PAD columns x0 - PAD .., so it holds every
// pulled population h_i(x - c_i) of the tile.  The copies complete on an mbarrier.  Threads then read
// their populations from shared memory at compile-time offsets (no address arithmetic per direction),
// apply the wall rule to the tile's boundary nodes and run the collision of the plain kernel.  Tiles
// that touch the periodic edges use the plain wrapped global loads.  Results are the plain kernel's bit
// for bit (collision.cuh).
//
// Every wait on an mbarrier is bounded; a wait that runs out sets bit 2 of the error word, the
// CTA waits (again bounded) for its own copies in flight and returns.
#pragma once

#include <cuda.h>

#include "step_kernel.cuh"

namespace lbm {

template <class L, class ST, int STAGES_, int BX_ = 64, int BY_ = 4>
struct TmaGeom {
    static constexpr int BX = BX_, BY = BY_;
    static constexpr int THREADS = BX * BY;
    static constexpr int ES = (int)sizeof(ST);
    static constexpr int PAD = (16 / ES) >= L::R ? (16 / ES) : 2 * (16 / ES);  // 16-byte aligned, >= reach
    static constexpr int BW = BX + 2 * PAD;                                       // box width (elements)
    static constexpr int BOX_BYTES = BW * BY * ES;
    static constexpr int SLOT = (BOX_BYTES + 127) / 128 * 128;                    // one direction's box
    static constexpr int STAGE = L::Q * SLOT;
    static constexpr int STAGES = STAGES_;
    static constexpr int SMEM = STAGES * STAGE;
};

__device__ __forceinline__ uint32_t smem_u32(const void* p) {
    return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}

__device__ __forceinline__ void mbar_init(uint64_t* bar, unsigned count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count) : "memory");
}

__device__ __forceinline__ void mbar_expect_tx(uint64_t* bar, unsigned bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes)
                 : "memory");
}

__device__ __forceinline__ bool mbar_try_wait(uint64_t* bar, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred P1;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 P1, [%1], %2;\n\t"
        "selp.b32 %0, 1, 0, P1;\n\t}"
        : "=r"(ok)
        : "r"(smem_u32(bar)), "r"(parity)
        : "memory");
    return ok != 0;
}

// Bounded wait for the phase with the given parity to complete.
__device__ __forceinline__ bool mbar_wait(uint64_t* bar, uint32_t parity, long long limit) {
    const long long t0 = clock64();
    while (!mbar_try_wait(bar, parity)) {
        if (clock64() - t0 > limit) return false;
    }
    return true;
}

__device__ __forceinline__ void tma_load_3d(void* dst, const CUtensorMap* map, int c0, int c1, int c2, uint64_t* bar) {
    asm volatile(
        "cp.async.bulk.tensor.3d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4}], "
        "[%5];" ::"r"(smem_u32(dst)),
        "l"(reinterpret_cast<uint64_t>(map)), "r"(c0), "r"(c1), "r"(c2), "r"(smem_u32(bar))
        : "memory");
}

// Bulk tensor store of one box from shared memory (tracked by the thread's bulk async-group).
__device__ __forceinline__ void tma_store_3d(const CUtensorMap* map, int c0, int c1, int c2, const void* src) {
    asm volatile("cp.async.bulk.tensor.3d.global.shared::cta.tile.bulk_group [%0, {%1, %2, %3}], [%4];" ::"l"(
                     reinterpret_cast<uint64_t>(map)),
                 "r"(c0), "r"(c1), "r"(c2), "r"(smem_u32(src))
                 : "memory");
}

// Grid of a staged kernel: force blocks, then one block per tile.
inline dim3 tile_grid(const InstDev& P, int threads) { return dim3(P.ntiles + force_blocks(P.ngroups, threads)); }

constexpr long long kTmaWaitLimit = 4000000000ll;  // clock cycles (about 2 s)

// Tile t lies at least the lattice reach inside the grid (its boxes need no periodic wrap).
template <class G, class L>
__device__ __forceinline__ bool tile_interior(const InstDev& P, int t) {
    const int x0 = (t % P.ntx) * G::BX, y0 = (t / P.ntx) * G::BY;
    return x0 >= L::R && x0 + G::BX + L::R <= P.nx && y0 >= L::R && y0 + G::BY + L::R <= P.ny;
}

// Thread 0: arm the stage's barrier and issue the Q boxes of tile t.
template <class G, class L>
__device__ __forceinline__ void issue_tile(const InstDev& P, const CUtensorMap* map, int t, unsigned char* stage,
                                           uint64_t* bar) {
    const int x0 = (t % P.ntx) * G::BX, y0 = (t / P.ntx) * G::BY;
    mbar_expect_tx(bar, (unsigned)(L::Q * G::BOX_BYTES));
#pragma unroll
    for (int i = 0; i < L::Q; ++i) tma_load_3d(stage + i * G::SLOT, map, x0 - G::PAD, y0 - cy_of<L>(i), i, bar);
}

// Eq. 17 from a staged tile: h_i^adv = box_i[ty][tx + PAD - c_ix].
template <class G, class L, class ST>
__device__ __forceinline__ void gather_smem(const unsigned char* stage, int tx, int ty,
                                            typename StoreT<ST>::CT (&h)[L::Q]) {
    const ST* base = reinterpret_cast<const ST*>(stage) + ty * G::BW + tx + G::PAD;
#pragma unroll
    for (int i = 0; i < L::Q; ++i) {
        const ST* p = reinterpret_cast<const ST*>(reinterpret_cast<const unsigned char*>(base) + i * G::SLOT) -
                      cx_of<L>(i);
        h[i] = StoreT<ST>::ld(p);
    }
}

// Single-instance step, one block per tile: an interior tile is staged by one set of Q bulk
// copies, waited for and computed; latency is hidden by the other resident blocks.
template <class L, class ST, int COLL, int BX, int BY>
__global__ void __launch_bounds__(BX * BY) step_kernel_tma1(const __grid_constant__ InstDev P,
                                                            const __grid_constant__ CUtensorMap map) {
    using G = TmaGeom<L, ST, 1, BX, BY>;
    extern __shared__ __align__(128) unsigned char smem[];
    __shared__ __align__(8) uint64_t bar;
    const int t = (int)blockIdx.x - force_blocks(P.ngroups, blockDim.x * blockDim.y);
    if (t < 0) {
        force_block<L, ST>(P, blockIdx.x);
        return;
    }
    pdl_wait_then_release();  // before the tile's copies: they read the previous step's output
    const int tid = threadIdx.y * BX + threadIdx.x;
    const int x = (t % P.ntx) * BX + threadIdx.x;
    const int y = (t / P.ntx) * BY + threadIdx.y;
    const int cls = (x < P.nx && y < P.ny) ? (int)P.cls[y * P.pitch + x] : (int)NODE_SOLID;
    typename StoreT<ST>::CT h[L::Q];
    if (tile_interior<G, L>(P, t)) {
        if (tid == 0) {
            mbar_init(&bar, 1);
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            issue_tile<G, L>(P, &map, t, smem, &bar);
        }
        __syncthreads();
        const bool ok = mbar_wait(&bar, 0, kTmaWaitLimit);
        if (!__syncthreads_and(ok)) {
            if (tid == 0) {
                atomicOr(P.err, 4);
                mbar_wait(&bar, 0, kTmaWaitLimit);
            }
            __syncthreads();
            return;
        }
        if (cls != NODE_SOLID) {
            gather_smem<G, L, ST>(smem, threadIdx.x, threadIdx.y, h);
            tile_node<L, ST, COLL>(P, P.src, P.dst, x, y, cls, P.dv, P.dv_f, h);
        }
    } else if (cls != NODE_SOLID) {
        gather_global<L, ST>(P, static_cast<const ST*>(P.src), x, y, h);
        tile_node<L, ST, COLL>(P, P.src, P.dst, x, y, cls, P.dv, P.dv_f, h);
    }
}

// Single-instance step, one block per tile of BX x (NR BY) nodes: the tile is staged by one set of
// Q bulk copies, and each thread computes NR nodes of its column, one row of BY apart at a time.
// The block's fixed costs (tile indices, launch constants, the copies and their barrier, the
// force epilogue) are spread over NR nodes per thread, while only one node's populations are live.
// MINB: resident blocks per SM the register allocation must allow (the compiler would otherwise keep
// launch constants live across the rows at the price of occupancy).
template <class L, class ST, int COLL, int BX, int BY, int NR, int MINB>
__global__ void __launch_bounds__(BX * BY, MINB) step_kernel_tman(const __grid_constant__ InstDev P,
                                                            const __grid_constant__ CUtensorMap map) {
    using G = TmaGeom<L, ST, 1, BX, BY * NR>;
    extern __shared__ __align__(128) unsigned char smem[];
    __shared__ __align__(8) uint64_t bar;
    // The geometry (node classes) is written by the host only: it is read before the
    // wait for the previous step's grid, while that grid drains.
    const int t = (int)blockIdx.x - force_blocks(P.ngroups, blockDim.x * blockDim.y);
    if (t < 0) {
        force_block<L, ST>(P, blockIdx.x);
        return;
    }
    const int tid = threadIdx.y * BX + threadIdx.x;
    const int x = (t % P.ntx) * BX + threadIdx.x;
    const int yt = (t / P.ntx) * (BY * NR);
    const bool interior = tile_interior<G, L>(P, t);
    int cls[NR];
#pragma unroll
    for (int r = 0; r < NR; ++r) {
        const int y = yt + threadIdx.y + r * BY;
        cls[r] = (x < P.nx && y < P.ny) ? (int)P.cls[y * P.pitch + x] : (int)NODE_SOLID;
    }
    if (interior && tid == 0) {
        mbar_init(&bar, 1);
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    }
    pdl_wait_then_release();  // before the tile's copies: they read the previous step's output
    if (interior) {
        if (tid == 0) issue_tile<G, L>(P, &map, t, smem, &bar);
        __syncthreads();
        const bool ok = mbar_wait(&bar, 0, kTmaWaitLimit);
        if (!__syncthreads_and(ok)) {
            if (tid == 0) {
                atomicOr(P.err, 4);
                mbar_wait(&bar, 0, kTmaWaitLimit);
            }
            __syncthreads();
            return;
        }
    }
#pragma unroll 1
    for (int r = 0; r < NR; ++r) {
        const int ty = threadIdx.y + r * BY;
        const int y = yt + ty;
        const int c = cls[0];
#pragma unroll
        for (int j = 0; j + 1 < NR; ++j) cls[j] = cls[j + 1];  // rotate: stays in registers
        if (c == NODE_SOLID) continue;
        typename StoreT<ST>::CT h[L::Q];
        if (interior)
            gather_smem<G, L, ST>(smem, threadIdx.x, ty, h);
        else
            gather_global<L, ST>(P, static_cast<const ST*>(P.src), x, y, h);
        tile_node<L, ST, COLL>(P, P.src, P.dst, x, y, c, P.dv, P.dv_f, h);
    }
}

// Eq. 17 from a staged tile for the two neighbouring nodes (2 tx, 2 tx + 1) of a thread; a
// direction with even c_ix has both values in one aligned two-element word.
template <class G, class L, class ST>
__device__ __forceinline__ void gather_smem_pair(const unsigned char* stage, int tx, int ty,
                                                 typename StoreT<ST>::CT (&h0)[L::Q],
                                                 typename StoreT<ST>::CT (&h1)[L::Q]) {
    static_assert(G::PAD % 2 == 0 && G::BW % 2 == 0, "two-element words must stay aligned");
    const ST* base = reinterpret_cast<const ST*>(stage) + ty * G::BW + 2 * tx + G::PAD;
#pragma unroll
    for (int i = 0; i < L::Q; ++i) {
        const int cx = cx_of<L>(i);
        const ST* p = reinterpret_cast<const ST*>(reinterpret_cast<const unsigned char*>(base) + i * G::SLOT) - cx;
        if ((cx & 1) == 0) {
            StoreT<ST>::ld2(p, h0[i], h1[i]);
        } else {
            h0[i] = StoreT<ST>::ld(p);
            h1[i] = StoreT<ST>::ld(p + 1);
        }
    }
}

// Single-instance step, one block of TX x TY threads per tile of 2 TX x TY nodes; each thread
// updates the two neighbouring nodes (x, x + 1), x even, and stores both with one access per
// direction.  Interior tiles are staged by TMA; edge tiles read with wrapped global loads.
template <class L, class ST, int COLL, int TX, int TY>
__global__ void __launch_bounds__(TX * TY) step_kernel_pair(const __grid_constant__ InstDev P,
                                                            const __grid_constant__ CUtensorMap map) {
    using G = TmaGeom<L, ST, 1, 2 * TX, TY>;
    using S = StoreT<ST>;
    using T = typename S::CT;
    extern __shared__ __align__(128) unsigned char smem[];
    __shared__ __align__(8) uint64_t bar;
    const int t = (int)blockIdx.x - force_blocks(P.ngroups, blockDim.x * blockDim.y);
    if (t < 0) {
        force_block<L, ST>(P, blockIdx.x);
        return;
    }
    pdl_wait_then_release();  // before the tile's copies: they read the previous step's output
    const int tid = threadIdx.y * TX + threadIdx.x;
    const int x = (t % P.ntx) * (2 * TX) + 2 * threadIdx.x;
    const int y = (t / P.ntx) * TY + threadIdx.y;
    const bool row = y < P.ny;
    const int cls0 = (row && x < P.nx) ? (int)P.cls[y * P.pitch + x] : (int)NODE_SOLID;
    const int cls1 = (row && x + 1 < P.nx) ? (int)P.cls[y * P.pitch + x + 1] : (int)NODE_SOLID;
    T h0[L::Q], h1[L::Q];
    if (tile_interior<G, L>(P, t)) {
        if (tid == 0) {
            mbar_init(&bar, 1);
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            issue_tile<G, L>(P, &map, t, smem, &bar);
        }
        __syncthreads();
        const bool ok = mbar_wait(&bar, 0, kTmaWaitLimit);
        if (!__syncthreads_and(ok)) {
            if (tid == 0) {
                atomicOr(P.err, 4);
                mbar_wait(&bar, 0, kTmaWaitLimit);
            }
            __syncthreads();
            return;
        }
        gather_smem_pair<G, L, ST>(smem, threadIdx.x, threadIdx.y, h0, h1);
    } else {
        if (cls0 != NODE_SOLID) gather_global<L, ST>(P, static_cast<const ST*>(P.src), x, y, h0);
        if (cls1 != NODE_SOLID) gather_global<L, ST>(P, static_cast<const ST*>(P.src), x + 1, y, h1);
    }
    if (cls0 != NODE_SOLID || cls1 != NODE_SOLID) {
        // solid nodes keep g = 0 (a stored 0 means h = H there; solid values are never read)
        T o0[L::Q] = {}, o1[L::Q] = {};
        if (cls0 != NODE_SOLID) {
            tile_fixup<L, ST, COLL>(P, P.src, x, y, cls0, h0);
            collide_emit<L, ST, COLL, T>(P, P.dv, P.dv_f, h0, [&](int i, T v) { o0[i] = v; });
        }
        if (cls1 != NODE_SOLID) {
            tile_fixup<L, ST, COLL>(P, P.src, x + 1, y, cls1, h1);
            collide_emit<L, ST, COLL, T>(P, P.dv, P.dv_f, h1, [&](int i, T v) { o1[i] = v; });
        }
        ST* __restrict__ dst = static_cast<ST*>(P.dst) + y * P.pitch + x;
        const long long plane = P.plane;
#pragma unroll
        for (int i = 0; i < L::Q; ++i) S::st2(dst + i * plane, o0[i], o1[i]);
    }
}

template <class L, class ST, int COLL, int TX, int TY>
cudaError_t launch_step_pair(const InstDev& P, const CUtensorMap& map, const CUtensorMap&, cudaStream_t stream) {
    using G = TmaGeom<L, ST, 1, 2 * TX, TY>;
    static bool attr = false;
    if (!attr) {
        cudaError_t e = cudaFuncSetAttribute(step_kernel_pair<L, ST, COLL, TX, TY>,
                                             cudaFuncAttributeMaxDynamicSharedMemorySize, G::SMEM);
        if (e != cudaSuccess) return e;
        attr = true;
    }
    return launch_pdl(step_kernel_pair<L, ST, COLL, TX, TY>, tile_grid(P, TX * TY), dim3(TX, TY), G::SMEM, stream, P, map);
}

// Launch of a staged step: `map` addresses the source buffer with the load boxes, `store_map` the
// destination buffer with the tile's own box (used by the kernels that store through TMA).
using TmaStepLaunchFn = cudaError_t (*)(const InstDev& P, const CUtensorMap& map, const CUtensorMap& store_map,
                                        cudaStream_t stream);

template <class L, class ST, int COLL, int BX, int BY>
cudaError_t launch_step_tma1(const InstDev& P, const CUtensorMap& map, const CUtensorMap&, cudaStream_t stream) {
    using G = TmaGeom<L, ST, 1, BX, BY>;
    static bool attr = false;
    if (!attr) {
        cudaError_t e = cudaFuncSetAttribute(step_kernel_tma1<L, ST, COLL, BX, BY>,
                                             cudaFuncAttributeMaxDynamicSharedMemorySize, G::SMEM);
        if (e != cudaSuccess) return e;
        attr = true;
    }
    return launch_pdl(step_kernel_tma1<L, ST, COLL, BX, BY>, tile_grid(P, BX * BY), dim3(BX, BY), G::SMEM, stream, P, map);
}

template <class L, class ST, int COLL, int BX, int BY, int NR, int MINB>
cudaError_t launch_step_tman(const InstDev& P, const CUtensorMap& map, const CUtensorMap&, cudaStream_t stream) {
    using G = TmaGeom<L, ST, 1, BX, BY * NR>;
    static bool attr = false;
    if (!attr) {
        cudaError_t e = cudaFuncSetAttribute(step_kernel_tman<L, ST, COLL, BX, BY, NR, MINB>,
                                             cudaFuncAttributeMaxDynamicSharedMemorySize, G::SMEM);
        if (e != cudaSuccess) return e;
        attr = true;
    }
    return launch_pdl(step_kernel_tman<L, ST, COLL, BX, BY, NR, MINB>, tile_grid(P, BX * BY), dim3(BX, BY), G::SMEM, stream,
                      P, map);
}

// The staged step with staged stores: an interior tile's outputs are written to a second
// shared-memory tile at compile-time offsets, then one thread stores each direction plane with one
// bulk tensor copy (box BX x BY at the tile's origin, never negative, x a multiple of BX) and waits
// for the copies before the block exits.  Nodes of the tile that are solid are stored as zero (no
// step ever reads them).  Tiles at the periodic edges keep the plain loads and stores.
template <class L, class ST, int COLL, int BX, int BY>
struct TmaStoreGeom {
    using G = TmaGeom<L, ST, 1, BX, BY>;
    static constexpr int OSLOT = (BX * BY * (int)sizeof(ST) + 127) / 128 * 128;  // one plane of outputs
    static constexpr int SMEM = G::SMEM + L::Q * OSLOT;
};

template <class L, class ST, int COLL, int BX, int BY>
__global__ void __launch_bounds__(BX * BY) step_kernel_tma1s(const __grid_constant__ InstDev P,
                                                             const __grid_constant__ CUtensorMap map,
                                                             const __grid_constant__ CUtensorMap smap) {
    using G = TmaGeom<L, ST, 1, BX, BY>;
    using O = TmaStoreGeom<L, ST, COLL, BX, BY>;
    using S = StoreT<ST>;
    using T = typename S::CT;
    extern __shared__ __align__(128) unsigned char smem[];
    __shared__ __align__(8) uint64_t bar;
    const int t = (int)blockIdx.x - force_blocks(P.ngroups, blockDim.x * blockDim.y);
    if (t < 0) {
        force_block<L, ST>(P, blockIdx.x);
        return;
    }
    pdl_wait_then_release();  // before the tile's copies: they read the previous step's output
    const int tid = threadIdx.y * BX + threadIdx.x;
    const int x = (t % P.ntx) * BX + threadIdx.x;
    const int y = (t / P.ntx) * BY + threadIdx.y;
    const int cls = (x < P.nx && y < P.ny) ? (int)P.cls[y * P.pitch + x] : (int)NODE_SOLID;
    T h[L::Q];
    if (tile_interior<G, L>(P, t)) {
        if (tid == 0) {
            mbar_init(&bar, 1);
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            issue_tile<G, L>(P, &map, t, smem, &bar);
        }
        __syncthreads();
        const bool ok = mbar_wait(&bar, 0, kTmaWaitLimit);
        if (!__syncthreads_and(ok)) {
            if (tid == 0) {
                atomicOr(P.err, 4);
                mbar_wait(&bar, 0, kTmaWaitLimit);
            }
            __syncthreads();
            return;
        }
        unsigned char* out = smem + G::SMEM;
        const int o = threadIdx.y * BX + threadIdx.x;
        if (cls != NODE_SOLID) {
            gather_smem<G, L, ST>(smem, threadIdx.x, threadIdx.y, h);
            tile_fixup<L, ST, COLL>(P, P.src, x, y, cls, h);
            collide_emit<L, ST, COLL, T>(P, P.dv, P.dv_f, h,
                                         [&](int i, T v) { S::st(reinterpret_cast<ST*>(out + i * O::OSLOT) + o, v); });
        } else {
#pragma unroll
            for (int i = 0; i < L::Q; ++i) S::st(reinterpret_cast<ST*>(out + i * O::OSLOT) + o, (T)0);
        }
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");  // generic writes -> async proxy
        __syncthreads();
        if (tid == 0) {
            const int x0 = (t % P.ntx) * BX, y0 = (t / P.ntx) * BY;
#pragma unroll
            for (int i = 0; i < L::Q; ++i) tma_store_3d(&smap, x0, y0, i, out + i * O::OSLOT);
            asm volatile("cp.async.bulk.commit_group;" ::: "memory");
            // the block may exit once the copies have read its shared memory; the global writes
            // complete with the grid
            asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory");
        }
    } else if (cls != NODE_SOLID) {
        gather_global<L, ST>(P, static_cast<const ST*>(P.src), x, y, h);
        tile_node<L, ST, COLL>(P, P.src, P.dst, x, y, cls, P.dv, P.dv_f, h);
    }
}

template <class L, class ST, int COLL, int BX, int BY>
cudaError_t launch_step_tma1s(const InstDev& P, const CUtensorMap& map, const CUtensorMap& smap,
                              cudaStream_t stream) {
    using O = TmaStoreGeom<L, ST, COLL, BX, BY>;
    static bool attr = false;
    if (!attr) {
        cudaError_t e = cudaFuncSetAttribute(step_kernel_tma1s<L, ST, COLL, BX, BY>,
                                             cudaFuncAttributeMaxDynamicSharedMemorySize, O::SMEM);
        if (e != cudaSuccess) return e;
        attr = true;
    }
    return launch_pdl(step_kernel_tma1s<L, ST, COLL, BX, BY>, tile_grid(P, BX * BY), dim3(BX, BY), O::SMEM, stream, P, map,
                      smap);
}

}  // namespace lbm
