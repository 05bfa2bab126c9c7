// step_types.cuh -- what every step kernel needs: the launch parameters of one lattice instance, the
// storage types and programmatic dependent launch.
#pragma once

#include <cuda_bf16.h>
#include <cuda_fp16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include <utility>

#include "lattice.cuh"

namespace lbm {

enum Storage { ST_F64 = 0, ST_F32 = 1, ST_BF16 = 2, ST_F16 = 3 };
enum Collision { COLL_BGK = 0, COLL_REG = 1 };

// Node classes of the `cls` array.
enum NodeClass : uint8_t { NODE_BULK = 0, NODE_SOLID = 1, NODE_BOUNDARY = 2 };

// Everything one launch needs to know about one lattice instance.
struct InstDev {
    const void* src;             // h at step n, [Q][ny][pitch]
    void* dst;                   // h at step n+1
    const uint8_t* cls;          // [ny][pitch] NodeClass
    const ulonglong2* links;     // [ny][pitch] (tile kernels): .x bit i = link i blocked by the body (label
                                 // 1), .y bit i = blocked by a static wall (label 2)
    double2* partials;           // [ngroups] FP64 force partials of the groups (scratch)
    unsigned int* ticket;        // groups of the current step that have finished (scratch, 0 between
                                 // launches: the last one resets it)
    double2* force_out;          // force on the body during this step (written by the last group)
    int* err;                    // bit 0: non-finite force seen
    double dv;                   // drive of this step: U_w(n + 1/2) (wall) or g(n + 1/2) (body force)
    double dv2;                  // drive of the next step, n + 3/2 (in-place AA streaming only)
    // moving-wall terms 2 rho0 m U_w / (theta s) of the links with |c_x| = m, for dv and dv2 (zero unless
    // the wall moves), and their FP32 copies
    double mw[4], mw2[4];
    float mw_f[4], mw2_f[4];
    const uint2* bnodes;         // [nb] (x, y) of the fluid nodes with blocked links: the nodes with body
                                 // links first, then the others, each part in increasing node order
    const ulonglong2* blinks;    // [nb] their links, as in `links`
    const void* flinks;          // body links for the force (flink_entries)
    double2 fconst;              // geometry-only part of the force, -sum c_i 2 w_i rho0
    double2 fmov;                // moving-wall part of the force per unit drive, -sum c_i c_ix 2 w_i rho0 / theta
                                 // (body links, bounce-back, wall drive; 0 otherwise)
    int nb, nbf;                 // nodes listed, and those of them with body links
    int nfl, glen;               // body links, and links per lane of a force group
    int ngroups;                 // force groups of a step
    long long plane;             // ny * pitch
    int nx, ny, pitch;
    int ntx;                     // tiles along x
    int ntiles;
    int flip;                    // 1: the tiles are taken from the last to the first.  lbm_step alternates: the
                                 // step starts with what the previous one wrote last and is still in L2
                                 // (1024^2 D2Q37 FP32 47.7 -> 45.4 us a step, FP16 30.0 -> 27; 1001 x 777
                                 // in place 42.5 -> 34.8; 2048^2 FP32 186.9 -> 184)
    int eq_order;                // 2 or 4
    int moving;                  // 1: body links carry the moving-wall term (wall drive)
    int wall_ds;                 // 0: bounce-back (Eq. 12); 1: diffuse scattering (Eq. 11)
    int body_force;              // 1: fluid gets rho * g (body-frame drive)
    double rho0;
    double s, inv_s;             // storage scale
    double omega_c;              // 1/tau
    double reg_a, reg_a2;        // (1 - 1/tau) / (2 theta^2), and twice that
    double src_k, src_t;         // (1 - 1/(2 tau)) / theta, and tau times that
    double mw_k;                 // 2 rho0 / (theta s): moving-wall term per unit c_i.U_w
    // FP32 copies of the constants above (and of dv), so that FP32 arithmetic converts nothing per
    // node: double -> float conversions run on the FP64 pipe, which is slow on this GPU
    float dv_f, rho0_f, s_f, inv_s_f, omega_c_f, src_k_f;
    float src_t_f[2];            // src_k over omega_c_f, as the sum of two floats (collision.cuh)
    // FP32 regularization factors of P_xx, P_yy and of P_xy, each as the sum of two floats (collision.cuh)
    float reg_f[4];
    // 16-bit body-frame runs store h_i - H_i(n), with H_i(n) the (scaled) equilibrium deviation of
    // the uniform stream U(n) = sum_{k<n} g(k + 1/2) that the body force sets up; far from the body
    // the stored values are then small and so are their rounding errors.  The stream is along x, so
    // H_i depends on c_ix only: Hl (the state read) and Hs (the state written) hold it for
    // c_ix = -3..3 at index c_ix + 3.  HM: moments sum_i w_i {1, c, cc} H_i of Hl (scaled units).
    // He, Ho: the even and odd parts of Hs in c_x, He[m] = (Hs(m) + Hs(-m)) / 2 and
    // Ho[m] = (Hs(m) - Hs(-m)) / 2 for m = |c_x|; the collision folds them into its per-node
    // coefficients, so outputs leave it already relative to the stream.  All zero when stream_off
    // is clear.
    int stream_off;
    float HM[6];
    float Hl[7];
    float Hs[7];
    float He[4];
    float Ho[4];
};

// Drive of a step and what follows from it (see InstDev).
__host__ __device__ inline void set_drive(InstDev& P, double dv) {
    P.dv = dv;
    P.dv_f = (float)dv;
    for (int m = 0; m < 4; ++m) {
        P.mw[m] = P.moving ? P.mw_k * m * dv : 0.0;
        P.mw_f[m] = (float)P.mw[m];
    }
}

// Body links sorted by direction, then node: c_i w_i by direction, followed (at kFLinkTable bytes) by one
// entry per link i of a node: .x the element offset of the node's own population opposite to link i, .y the
// direction i | (c_ix + 3) << 8.
constexpr size_t kFLinkTable = 640;
__device__ __forceinline__ const double2* flink_weights(const void* f) { return static_cast<const double2*>(f); }
__device__ __forceinline__ const uint2* flink_entries(const void* f) {
    return reinterpret_cast<const uint2*>(static_cast<const unsigned char*>(f) + kFLinkTable);
}
// A force group is one warp: glen links a lane.  Four, or more where that would give more than
// kMaxForceGroups groups.
constexpr int kMaxForceGroups = 8192;
inline int force_group_len(int nfl) {
    const long long per = 32ll * kMaxForceGroups;
    const int len = (int)((nfl + per - 1) / per);
    return len > 4 ? len : 4;
}
inline int force_groups(int nfl, int len) { return (int)(((long long)nfl + 32ll * len - 1) / (32ll * len)); }

// Programmatic dependent launch.  Step kernels are launched so that the next kernel of the stream
// may be scheduled while this one drains: every step kernel first waits for the previous grid of
// its stream to complete (its outputs are this step's inputs, including the force scratch), then
// lets the next one launch.  The next grid is launched only after every block of this one has
// passed that point, so its blocks never take SM slots that this grid still needs.
__device__ __forceinline__ void pdl_wait_then_release() {
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}

// Launch a step kernel with programmatic stream serialization (disabled when the environment
// sets LBM_PDL=0: plain stream order).
bool pdl_enabled();

template <class... KArgs, class... Args>
cudaError_t launch_pdl(void (*kernel)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t stream,
                       Args&&... args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = stream;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = pdl_enabled() ? 1 : 0;
    return cudaLaunchKernelEx(&cfg, kernel, std::forward<Args>(args)...);
}

// Stream-offset constants of direction i (see InstDev): read / written state.
template <class L>
__device__ __forceinline__ float off_l(const InstDev& P, int i) { return P.Hl[cx_of<L>(i) + 3]; }
template <class L>
__device__ __forceinline__ float off_s(const InstDev& P, int i) { return P.Hs[cx_of<L>(i) + 3]; }

// A launch constant in the arithmetic type T: the double itself, or its FP32 copy.
template <class T>
__device__ __forceinline__ T kconst(double d, float f);
template <>
__device__ __forceinline__ double kconst<double>(double d, float) { return d; }
template <>
__device__ __forceinline__ float kconst<float>(double, float f) { return f; }

template <class ST> struct StoreT;
// Loads and stores of the storage type; ld2/st2 move two neighbouring values (p aligned to two
// elements) with one access; rnd(v) is v rounded to the storage type (what a store and a load give).
// st stores through a generic pointer (global or shared memory); stg stores to global memory only,
// for 16-bit storage as a streaming store (st.global.cs): the next step reads the populations back
// long after they have left L2, and marking them first to evict keeps the staged loads' shared halo
// sectors in L2 longer.
// ldc is a plain weak load (ld.global.ca), never the read-only path (ld.global.nc) that the
// compiler may pick for a const __restrict__ pointer: the persistent batch kernel reads populations
// that other blocks of the same launch wrote.  They are visible to weak loads that follow the
// acquire of their producer's release (in the block, through the block barrier), which is what the
// memory model guarantees; it guarantees nothing for the read-only path.
template <> struct StoreT<double> {
    using CT = double;
    static __device__ __forceinline__ double rnd(double v) { return v; }
    static __device__ __forceinline__ double ld(const double* p) { return *p; }
    static __device__ __forceinline__ double ldc(const double* p) {
        double v;
        asm volatile("ld.global.ca.f64 %0, [%1];" : "=d"(v) : "l"(p));
        return v;
    }
    static __device__ __forceinline__ void st(double* p, double v) { *p = v; }
    static __device__ __forceinline__ void stg(double* p, double v) { *p = v; }
    static __device__ __forceinline__ void ld2(const double* p, double& a, double& b) {
        const double2 v = *reinterpret_cast<const double2*>(p);
        a = v.x;
        b = v.y;
    }
    static __device__ __forceinline__ void st2(double* p, double a, double b) {
        *reinterpret_cast<double2*>(p) = make_double2(a, b);
    }
};
template <> struct StoreT<float> {
    using CT = float;
    static __device__ __forceinline__ float rnd(float v) { return v; }
    static __device__ __forceinline__ float ld(const float* p) { return *p; }
    static __device__ __forceinline__ float ldc(const float* p) {
        float v;
        asm volatile("ld.global.ca.f32 %0, [%1];" : "=f"(v) : "l"(p));
        return v;
    }
    static __device__ __forceinline__ void st(float* p, float v) { *p = v; }
    static __device__ __forceinline__ void stg(float* p, float v) { *p = v; }
    static __device__ __forceinline__ void ld2(const float* p, float& a, float& b) {
        const float2 v = *reinterpret_cast<const float2*>(p);
        a = v.x;
        b = v.y;
    }
    static __device__ __forceinline__ void st2(float* p, float a, float b) {
        *reinterpret_cast<float2*>(p) = make_float2(a, b);
    }
};
template <> struct StoreT<__nv_bfloat16> {
    using CT = float;
    static __device__ __forceinline__ float rnd(float v) { return __bfloat162float(__float2bfloat16_rn(v)); }
    static __device__ __forceinline__ float ld(const __nv_bfloat16* p) { return __bfloat162float(*p); }
    static __device__ __forceinline__ float ldc(const __nv_bfloat16* p) {
        unsigned short v;
        asm volatile("ld.global.ca.u16 %0, [%1];" : "=h"(v) : "l"(p));
        return __bfloat162float(__ushort_as_bfloat16(v));
    }
    static __device__ __forceinline__ void st(__nv_bfloat16* p, float v) { *p = __float2bfloat16_rn(v); }
    static __device__ __forceinline__ void stg(__nv_bfloat16* p, float v) {
        asm("st.global.cs.b16 [%0], %1;" ::"l"(p), "h"(__bfloat16_as_ushort(__float2bfloat16_rn(v))));
    }
    static __device__ __forceinline__ void ld2(const __nv_bfloat16* p, float& a, float& b) {
        const float2 v = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(p));
        a = v.x;
        b = v.y;
    }
    static __device__ __forceinline__ void st2(__nv_bfloat16* p, float a, float b) {
        *reinterpret_cast<__nv_bfloat162*>(p) = __floats2bfloat162_rn(a, b);
    }
};
template <> struct StoreT<__half> {
    using CT = float;
    static __device__ __forceinline__ float rnd(float v) { return __half2float(__float2half_rn(v)); }
    static __device__ __forceinline__ float ld(const __half* p) { return __half2float(*p); }
    static __device__ __forceinline__ float ldc(const __half* p) {
        unsigned short v;
        asm volatile("ld.global.ca.u16 %0, [%1];" : "=h"(v) : "l"(p));
        return __half2float(__ushort_as_half(v));
    }
    static __device__ __forceinline__ void st(__half* p, float v) { *p = __float2half_rn(v); }
    static __device__ __forceinline__ void stg(__half* p, float v) {
        asm("st.global.cs.b16 [%0], %1;" ::"l"(p), "h"(__half_as_ushort(__float2half_rn(v))));
    }
    static __device__ __forceinline__ void ld2(const __half* p, float& a, float& b) {
        const float2 v = __half22float2(*reinterpret_cast<const __half2*>(p));
        a = v.x;
        b = v.y;
    }
    static __device__ __forceinline__ void st2(__half* p, float a, float b) {
        *reinterpret_cast<__half2*>(p) = __floats2half2_rn(a, b);
    }
};

// Two 16-bit values in one word: the lower, the upper, and a word of two rounded FP32 values.
template <class ST> struct Half16;
template <> struct Half16<__half> {
    static __device__ __forceinline__ float lo(unsigned w) { return __low2float(*reinterpret_cast<const __half2*>(&w)); }
    static __device__ __forceinline__ float hi(unsigned w) { return __high2float(*reinterpret_cast<const __half2*>(&w)); }
    static __device__ __forceinline__ unsigned pack(float a, float b) {
        const __half2 h = __floats2half2_rn(a, b);
        return *reinterpret_cast<const unsigned*>(&h);
    }
};
template <> struct Half16<__nv_bfloat16> {
    static __device__ __forceinline__ float lo(unsigned w) { return __uint_as_float(w << 16); }
    static __device__ __forceinline__ float hi(unsigned w) { return __uint_as_float(w & 0xffff0000u); }
    static __device__ __forceinline__ unsigned pack(float a, float b) {
        const __nv_bfloat162 h = __floats2bfloat162_rn(a, b);
        return *reinterpret_cast<const unsigned*>(&h);
    }
};

}  // namespace lbm
