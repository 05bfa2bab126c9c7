// collision.cuh -- the collision of the fused step: moments (Eq. 16), Hermite equilibrium (Eq. 15 or
// its 4th-order continuation), regularized (Eqs. 18-19) or plain BGK collision (Eq. 14) and the
// body-force source, of one node (float, double) or of two nodes at once (V2).
//
// Every operation is an explicitly rounded add, multiply or fused multiply-add, so that the compiler
// contracts nothing: all kernels, whatever their tiles and however many nodes a thread computes, give
// the same bits for the same node.
//
// An output is E(c) + O(c), an even and an odd polynomial of degree 4 in the velocity (c_x, c_y)
// whose coefficients depend on the node only.  They are expanded in monomials, so that the axis parts
// are evaluated once per |c_x| and |c_y| and shared by the shells, and the four velocities
// +-(m, n), +-(m, -n) of a shell cost 14 operations together.  (Polynomials in a = c.u / theta,
// evaluated velocity by velocity, take 410 FP64 operations a node, this form 291, and 284 without a body
// force.  FP64 storage is bound by them: 725 -> 579 us a step of the 1024^2 D2Q37 box, 51 -> 38 us of a 512^2
// D2Q9 plate, plain BGK 53 -> 40 with 74 operations.)
#pragma once

#include "step_types.cuh"

namespace lbm {

// Two FP32 values, one per node; the packed FP32 operations of sm_100+ issue both lanes at once, each
// rounded like the scalar operation.  Products with compile-time constants stay scalar (an immediate
// operand costs no register pair; the FP32 pipe takes the same time either way).
struct V2 {
    float x, y;
};

__device__ __forceinline__ float vadd(float a, float b) { return __fadd_rn(a, b); }
__device__ __forceinline__ float vsub(float a, float b) { return __fsub_rn(a, b); }
__device__ __forceinline__ float vmul(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ float vfma(float a, float b, float c) { return __fmaf_rn(a, b, c); }
__device__ __forceinline__ float vneg(float a) { return -a; }
__device__ __forceinline__ float vrcp(float a) { return __frcp_rn(a); }

// FP64: on this GPU a multiply-add whose three operands are registers takes 16.9 cycles per warp and SM, but an
// add, a multiply, or a multiply-add with a constant or uniform operand 20.0 (measured, independent chains).
// So every FP64 operation below is a multiply-add of registers: an add multiplies by a 1 and a multiply adds
// a 0 that the compiler cannot know, and constants go through a register it cannot know either (their bits
// xor an unknown zero: two integer instructions, whose units idle; a zero of each lane's own, since one that is the
// same for a warp may end up in a uniform register: plain BGK 1024 x 700 D2Q37 415 -> 373 us a step).  The results are the same.  1024^2
// D2Q37 579 -> 493 us a step, 512^2 152 -> 129; 2048^2 D2Q9 558 -> 482.
static __device__ int fp64_zero_word[32] = {};
__device__ __forceinline__ double opaque(double k) {
    const int z = __ldg(&fp64_zero_word[threadIdx.x & 31]);
    return __hiloint2double(__double2hiint(k) ^ z, __double2loint(k) ^ z);
}
// Reads the unknown zero now (before a wait), so that the collision need not wait for it.
template <class ST>
__device__ __forceinline__ void prepare_collision() {
    if (sizeof(ST) == 8) asm volatile("" ::"r"(__ldg(&fp64_zero_word[threadIdx.x & 31])));
}
__device__ __forceinline__ double vadd(double a, double b) { return __fma_rn(a, opaque(1.0), b); }
__device__ __forceinline__ double vsub(double a, double b) { return __fma_rn(b, -opaque(1.0), a); }
__device__ __forceinline__ double vmul(double a, double b) { return __fma_rn(a, b, opaque(0.0)); }
__device__ __forceinline__ double vfma(double a, double b, double c) { return __fma_rn(a, b, c); }
__device__ __forceinline__ double vneg(double a) { return -a; }
__device__ __forceinline__ double vrcp(double a) { return __drcp_rn(a); }

__device__ __forceinline__ V2 vadd(V2 a, V2 b) {
    V2 d;
    asm("{\n\t.reg .b64 a, b;\n\tmov.b64 a, {%2, %3};\n\tmov.b64 b, {%4, %5};\n\tadd.rn.f32x2 a, a, b;\n\t"
        "mov.b64 {%0, %1}, a;\n\t}"
        : "=f"(d.x), "=f"(d.y)
        : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y));
    return d;
}
__device__ __forceinline__ V2 vsub(V2 a, V2 b) {
    V2 d;
    asm("{\n\t.reg .b64 a, b;\n\tmov.b64 a, {%2, %3};\n\tmov.b64 b, {%4, %5};\n\tsub.rn.f32x2 a, a, b;\n\t"
        "mov.b64 {%0, %1}, a;\n\t}"
        : "=f"(d.x), "=f"(d.y)
        : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y));
    return d;
}
__device__ __forceinline__ V2 vfma(V2 a, V2 b, V2 c) {
    V2 d;
    asm("{\n\t.reg .b64 a, b, c;\n\tmov.b64 a, {%2, %3};\n\tmov.b64 b, {%4, %5};\n\tmov.b64 c, {%6, %7};\n\t"
        "fma.rn.f32x2 a, a, b, c;\n\tmov.b64 {%0, %1}, a;\n\t}"
        : "=f"(d.x), "=f"(d.y)
        : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y), "f"(c.x), "f"(c.y));
    return d;
}
// (as a multiply-add of zero: a packed multiply would be contracted with an add that follows it)
__device__ __forceinline__ V2 vmul(V2 a, V2 b) { return vfma(a, b, V2{0.f, 0.f}); }
__device__ __forceinline__ V2 vneg(V2 a) { return V2{-a.x, -a.y}; }
__device__ __forceinline__ V2 vrcp(V2 a) { return V2{__frcp_rn(a.x), __frcp_rn(a.y)}; }

// The scalar type of V, and a scalar in every lane of V.
template <class V> struct Lane { using T = V; };
template <> struct Lane<V2> { using T = float; };
template <class V> __device__ __forceinline__ V vset(typename Lane<V>::T s) { return s; }
template <> __device__ __forceinline__ V2 vset<V2>(float s) { return V2{s, s}; }

// k b + c and k b for a scalar k (a launch constant or a compile-time constant).
template <class V>
__device__ __forceinline__ V vfmas(typename Lane<V>::T k, V b, V c) { return vfma(k, b, c); }
template <>
__device__ __forceinline__ double vfmas<double>(double k, double b, double c) { return __fma_rn(opaque(k), b, c); }
template <>
__device__ __forceinline__ V2 vfmas<V2>(float k, V2 b, V2 c) { return V2{__fmaf_rn(k, b.x, c.x), __fmaf_rn(k, b.y, c.y)}; }
template <class V>
__device__ __forceinline__ V vmuls(typename Lane<V>::T k, V b) { return vmul(k, b); }
template <>
__device__ __forceinline__ double vmuls<double>(double k, double b) { return __fma_rn(opaque(k), b, opaque(0.0)); }
template <>
__device__ __forceinline__ V2 vmuls<V2>(float k, V2 b) { return V2{__fmul_rn(k, b.x), __fmul_rn(k, b.y)}; }
template <class V>
__device__ __forceinline__ V vadds(V b, typename Lane<V>::T k) { return vadd(b, k); }
template <>
__device__ __forceinline__ double vadds<double>(double b, double k) { return __fma_rn(b, opaque(1.0), opaque(k)); }
template <>
__device__ __forceinline__ V2 vadds<V2>(V2 b, float k) { return V2{__fadd_rn(b.x, k), __fadd_rn(b.y, k)}; }
// k b + c where many of them share the launch constant k: two nodes at a time with it in registers (kv), one packed
// operation instead of two.
template <class V>
__device__ __forceinline__ V vfmac(typename Lane<V>::T k, V, V b, V c) { return vfmas<V>(k, b, c); }
template <>
__device__ __forceinline__ V2 vfmac<V2>(float, V2 kv, V2 b, V2 c) { return vfma(kv, b, c); }
// The same for compile-time constants (after inlining): a factor of 1 or -1 is an add or a subtract.
template <class V>
__device__ __forceinline__ V vfmak(double k, V b, V c) {
    if (k == 1.0) return vadd(b, c);
    if (k == -1.0) return vsub(c, b);
    return vfmas<V>((typename Lane<V>::T)k, b, c);
}
template <class V>
__device__ __forceinline__ V vmulk(double k, V b) {
    if (k == 1.0) return b;
    return vmuls<V>((typename Lane<V>::T)k, b);
}

// Sums over the weights as FP32 holds them (w_i, w_i c_i, .. rounded): what a collision and the next
// step's moments multiply mass, momentum and the kept part of the stress by, were it not corrected --
// 1 + 8e-9 and 1 + 1.5e-8 a step for mass and momentum in D2Q37, which adds up over a run.  The rest weight,
// 1/theta and the regularization factors (InstDev::reg_f) make up for it, in two parts where one float
// cannot hold them.
template <class L, class T>
__host__ __device__ constexpr double rest_weight() {  // 1 - sum of the other weights
    double s = 1.0;
    for (int k = 0; k < L::NP; ++k) s -= 2.0 * (double)(T)L::wp(k);
    return s;
}
template <class L, class T>
__host__ __device__ constexpr double inv_theta() {    // 1 / sum of w_i c_ix c_ix
    double s = 0.0;
    for (int k = 0; k < L::NP; ++k) s += 2.0 * (double)(T)(L::wp(k) * L::px(k)) * L::px(k);
    return 1.0 / s;
}
// Weight of pair k in p_xx as the moments apply it (diagonal shells in two parts).
template <class L, class T>
__host__ __device__ constexpr double weight_xx(int k) {
    const int x2 = L::px(k) * L::px(k);
    return x2 && L::py(k) ? (double)(T)L::wp(k) + (double)(T)(L::wp(k) * (x2 - 1)) : (double)(T)(L::wp(k) * x2);
}
// theta as the second moments see it: what p_xx holds of a constant, sum of w_i c_ix c_ix.
template <class L, class T>
__host__ __device__ constexpr double pressure() {
    double s = 0.0;
    for (int k = 0; k < L::NP; ++k) s += 2.0 * weight_xx<L, T>(k);
    return s;
}
// What the next step's P_xx and P_xy hold of r_xx and r_xy (exactly 2 theta^2 and theta^2).
template <class L, class T>
__host__ __device__ constexpr double reg_diag() {
    double m = 0.0;
    for (int k = 0; k < L::NP; ++k) m += 2.0 * weight_xx<L, T>(k) * (L::px(k) * L::px(k));
    return m - pressure<L, T>() * pressure<L, T>();
}
template <class L, class T>
__host__ __device__ constexpr double reg_cross() {
    double m = 0.0;
    for (int k = 0; k < L::NP; ++k) {
        const int xy = L::px(k) * L::py(k);
        m += 2.0 * (double)(T)(L::wp(k) * xy) * xy;
    }
    return m;
}

// k v for a constant k given to more digits than T holds.
template <class V>
__device__ __forceinline__ V vmulx(double k, V v) {
    using T = typename Lane<V>::T;
    if (sizeof(T) == 8) return vmulk(k, v);
    const T hi = (T)k;
    return vfmas<V>((T)(k - (double)hi), v, vmuls<V>(hi, v));
}
template <class V>
__device__ __forceinline__ V vfmax(double k, V v, V c) {
    using T = typename Lane<V>::T;
    if (sizeof(T) == 8) return vfmak(k, v, c);
    const T hi = (T)k;
    return vfmas<V>((T)(k - (double)hi), v, vfmas<V>(hi, v, c));
}

// Eq. 16 on deviations: drho = sum g_i, j = sum g_i c_i, Pi' = sum g_i c_i c_i, in the units of
// the populations (w_i divided out).  The pair tables list pairs in groups of two of one shell:
// (p_x, p_y) and (p_x, -p_y), whose sums S, D and differences Jp, Jm of the pairs' sums and
// differences go into the moments, or (m, 0) and (0, m), taken pair by pair.  A diagonal shell's w S goes
// once into a sum that m0, pxx and pyy share.
template <class V>
struct Moments {
    V m0, jx, jy, pxx, pxy, pyy;
};

// (h(i): the population that arrived along direction i.)
template <class L, class V, class H>
__device__ __forceinline__ Moments<V> moments(H&& h) {
    using T = typename Lane<V>::T;
    static_assert(L::NP % 2 == 0 && L::py(0) == 0 && L::py(2) != 0 && L::py(2) == -L::py(3),
                  "the pair tables start with the axis pairs (1, 0), (0, 1) and the diagonal shell");
    Moments<V> M;
    // what the diagonal shells give to m0, pxx and pyy alike, and what they give to pxx and pyy beyond it
    V all, xx, yy;
    bool first_xx = true;
#pragma unroll
    for (int k = 2; k < L::NP; k += 2) {
        const int m = L::px(k), n = L::py(k);
        if (n == 0) continue;
        const double w = L::wp(k);
        const V a1 = h(1 + 2 * k), b1 = h(2 + 2 * k), a2 = h(3 + 2 * k), b2 = h(4 + 2 * k);
        const V sp1 = vadd(a1, b1), dm1 = vsub(a1, b1), sp2 = vadd(a2, b2), dm2 = vsub(a2, b2);
        const V S = vadd(sp1, sp2), D = vsub(sp1, sp2), Jp = vadd(dm1, dm2), Jm = vsub(dm1, dm2);
        if (k == 2) {
            all = vmulk(w, S);
            M.jx = vmulk(w * m, Jp);
            M.jy = vmulk(w * n, Jm);
            M.pxy = vmulk(w * m * n, D);
        } else {
            all = vfmak(w, S, all);
            M.jx = vfmak(w * m, Jp, M.jx);
            M.jy = vfmak(w * n, Jm, M.jy);
            M.pxy = vfmak(w * m * n, D, M.pxy);
        }
        if (m > 1 && n > 1) {  // the (2, 2) shell comes first of those with more than `all`
            xx = yy = vmulk(w * (m * m - 1), S);
            first_xx = false;
        } else if (m > 1) {
            xx = vfmak(w * (m * m - 1), S, xx);
        } else if (n > 1) {
            yy = vfmak(w * (n * n - 1), S, yy);
        }
    }
    M.m0 = all;
    M.pxx = first_xx ? all : vadd(all, xx);
    M.pyy = first_xx ? all : vadd(all, yy);
#pragma unroll
    for (int k = 0; k < L::NP; k += 2) {
        const int m = L::px(k);
        if (L::py(k) != 0) continue;
        const double w = L::wp(k);
        const V a1 = h(1 + 2 * k), b1 = h(2 + 2 * k), a2 = h(3 + 2 * k), b2 = h(4 + 2 * k);
        const V sp1 = vadd(a1, b1), dm1 = vsub(a1, b1), sp2 = vadd(a2, b2), dm2 = vsub(a2, b2);
        M.m0 = vfmak(w, sp2, vfmak(w, sp1, M.m0));
        M.jx = vfmak(w * m, dm1, M.jx);
        M.jy = vfmak(w * m, dm2, M.jy);
        M.pxx = vfmak(w * m * m, sp1, M.pxx);
        M.pyy = vfmak(w * m * m, sp2, M.pyy);
    }
    constexpr double w0 = sizeof(T) == 8 ? L::w0() : rest_weight<L, T>();
    M.m0 = vfmax<V>(w0, h(0), M.m0);
    return M;
}

// Coefficients of a node's outputs by monomial c_x^p c_y^q, in storage units.
template <class V>
struct Coef {
    V c0, q20, q11, q02;            // even part up to second order (regularized: with Eq. 19 and the source)
    V q40, q31, q22, q13, q04;      // fourth order; q31, q13 and q22 less their factors 4, 4 and 6
    V l10, l01;                     // odd part, first order
    V c30, c21, c12, c03;           // third order; c21 and c12 less their factor 3
};

// Coefficients from the moments (storage units, relative to the stream offset with 16-bit storage and
// the offset on): Eqs. 15 and 19 and the Guo-type source.  With 16-bit storage the moments are scaled
// by s on the way in and the coefficients by 1/s on the way out.
// BODY: whether there is a body force (0, 1), or -1 to ask the launch parameters.  (FP64 asks once per node, in
// collide_emit: an FP64 instruction predicated off takes as long as one that runs.)
template <class L, class ST, int COLL, class V, int BODY = -1>
__device__ __forceinline__ Coef<V> coefficients(const InstDev& P, double dv, float dv_f, Moments<V> M) {
    using T = typename Lane<V>::T;
    constexpr bool SCALED = sizeof(ST) == 2;
    constexpr bool H4 = L::R == 3;  // the lattice carries the fourth-order equilibrium
    const bool body = BODY < 0 ? P.body_force != 0 : BODY == 1;
    Coef<V> C;
    if (SCALED) {
        if (COLL == COLL_REG && P.stream_off) {
            M.m0 = vadds(M.m0, (T)P.HM[0]); M.jx = vadds(M.jx, (T)P.HM[1]); M.jy = vadds(M.jy, (T)P.HM[2]);
            M.pxx = vadds(M.pxx, (T)P.HM[3]); M.pxy = vadds(M.pxy, (T)P.HM[4]); M.pyy = vadds(M.pyy, (T)P.HM[5]);
        }
        const T s = kconst<T>(P.s, P.s_f);
        M.m0 = vmuls<V>(s, M.m0); M.jx = vmuls<V>(s, M.jx); M.jy = vmuls<V>(s, M.jy);
        if (COLL == COLL_REG) { M.pxx = vmuls<V>(s, M.pxx); M.pxy = vmuls<V>(s, M.pxy); M.pyy = vmuls<V>(s, M.pyy); }
    }
    constexpr double TH = L::theta();
    const V rho = vadds(M.m0, kconst<T>(P.rho0, P.rho0_f));
    const V irho = vrcp(rho);
    V jx = M.jx, F = vset<V>((T)0);
    if (body) {
        F = vmuls<V>(kconst<T>(dv, dv_f), rho);
        jx = vfmak(0.5, F, jx);
    }
    const V ux = vmul(jx, irho), uy = vmul(M.jy, irho);
    constexpr double ITH = sizeof(T) == 8 ? 1.0 / TH : inv_theta<L, T>();
    const V X = vmulx<V>(ITH, ux), Y = vmulx<V>(ITH, uy);
    const V b = vfma(uy, Y, vmul(ux, X));

    // Eq. 15 (+ 4th order): g_i^eq / w_i = e0 + a^2 (e1 + a^2 e2) + a (o0 + o1 a^2), a = c_i.u/theta
    const V hr = vmulk(0.5, rho);
    V e0 = vfma(vneg(hr), b, M.m0), e1 = hr, o0 = rho, e2, o1;
    if (H4) {
        e2 = o1 = vset<V>((T)0);
        if (P.eq_order >= 4) {
            const V rb = vmul(rho, b);
            e0 = vfma(vmulk(0.125, rb), b, e0);
            e1 = vfmak(-0.25, rb, e1);
            o0 = vfmak(-0.5, rb, o0);
            e2 = vmulk(1.0 / 24.0, rho);
            o1 = vmulk(1.0 / 6.0, rho);
        }
    }
    // Guo-type source: even part kf (a c_x - u_x), odd part c_x times hf, kf (plain BGK) or F/(2 theta).  It goes
    // into the coefficients; for plain BGK, whose outputs are h + (E + O - h) / tau, it is tau times the source.
    // (Added to each output instead it took two operations a direction and the registers of its parts: 16
    // instances of 256^2 D2Q37 FP64 788 us a step against 555, 12 of D2Q9 FP16 56.5 against 50.4.)
    V kf = vset<V>((T)0);
    if (body) {
        if constexpr (COLL == COLL_REG) kf = vmuls<V>(kconst<T>(P.src_k, P.src_k_f), F);
        else if constexpr (sizeof(T) == 8) kf = vmuls<V>(P.src_t, F);
        else kf = vfmas<V>(P.src_t_f[1], F, vmuls<V>(P.src_t_f[0], F));
    }
    if (body && COLL == COLL_BGK) e0 = vfma(vneg(kf), ux, e0);
    V rxx, rxy, ryy, hf = kf, kx = kf;
    if (COLL == COLL_REG) {
        // Eq. 19: Pi^ne = Pi - Pi^eq with Pi^eq = rho theta I + rho u u (exact on these lattices)
        constexpr double THP = sizeof(T) == 8 ? TH : pressure<L, T>();
        const V rux = vmul(rho, ux), ruy = vmul(rho, uy);
        const V Pxx = vfma(vneg(rux), ux, vfmax<V>(-THP, M.m0, M.pxx));
        const V Pxy = vfma(vneg(rux), uy, M.pxy);
        const V Pyy = vfma(vneg(ruy), uy, vfmax<V>(-THP, M.m0, M.pyy));
        if constexpr (sizeof(T) == 8) {
            rxx = vmuls<V>(P.reg_a, Pxx);
            rxy = vmuls<V>(P.reg_a2, Pxy);
            ryy = vmuls<V>(P.reg_a, Pyy);
        } else {
            rxx = vfmas<V>(P.reg_f[1], Pxx, vmuls<V>(P.reg_f[0], Pxx));
            rxy = vfmas<V>(P.reg_f[3], Pxy, vmuls<V>(P.reg_f[2], Pxy));
            ryy = vfmas<V>(P.reg_f[1], Pyy, vmuls<V>(P.reg_f[0], Pyy));
        }
        e0 = vfmax<V>(-THP, vadd(rxx, ryy), e0);
        if (body) e0 = vfma(vneg(kf), ux, e0);
        hf = vmulk(0.5 / TH, F);   // first-order part: kept J^ne = -F/2 plus the source
    }
    if (SCALED) {
        // outputs are wanted in storage units (divided by s): scale the coefficients once per node
        const T is = kconst<T>(P.inv_s, P.inv_s_f);
        e0 = vmuls<V>(is, e0); e1 = vmuls<V>(is, e1); o0 = vmuls<V>(is, o0);
        if (H4) { e2 = vmuls<V>(is, e2); o1 = vmuls<V>(is, o1); }
        if (COLL == COLL_REG) {
            rxx = vmuls<V>(is, rxx); rxy = vmuls<V>(is, rxy); ryy = vmuls<V>(is, ryy);
        }
        hf = vmuls<V>(is, hf);
        kx = vmuls<V>(is, kf);
    }
    // monomials
    C.c0 = e0;
    const V eX = vmul(e1, X), eY = vmul(e1, Y), eX2 = vadd(eX, eX);
    if (COLL == COLL_REG) {
        C.q20 = vfma(eX, X, rxx);
        C.q11 = vfma(eX2, Y, rxy);
        C.q02 = vfma(eY, Y, ryy);
    } else {
        C.q20 = vmul(eX, X);
        C.q11 = vmul(eX2, Y);
        C.q02 = vmul(eY, Y);
    }
    C.l10 = BODY == 0 ? vmul(o0, X) : vfma(o0, X, hf);
    if (body) {
        C.q20 = vfma(kx, X, C.q20);
        C.q11 = vfma(kx, Y, C.q11);
    }
    C.l01 = vmul(o0, Y);
    if (H4) {
        const V X2 = vmul(X, X), XY = vmul(X, Y), Y2 = vmul(Y, Y);
        const V eXX = vmul(e2, X2), eYY = vmul(e2, Y2);
        C.q40 = vmul(eXX, X2);
        C.q31 = vmul(eXX, XY);
        C.q22 = vmul(eXX, Y2);
        C.q13 = vmul(eYY, XY);
        C.q04 = vmul(eYY, Y2);
        const V oX = vmul(o1, X), oY = vmul(o1, Y);
        C.c30 = vmul(oX, X2);
        C.c21 = vmul(oY, X2);
        C.c12 = vmul(oX, Y2);
        C.c03 = vmul(oY, Y2);
    }
    return C;
}

// The outputs of a node from its coefficients: emit(i, v) receives output i in storage units, relative to the
// stream offset of the stored state when it is on (regularized: its even and odd parts He and Ho of |c_x| leave
// the even and odd parts; plain BGK with OFFSET: off_s leaves the output).  Plain BGK reads the pulled populations h
// (absolute ones), the regularized collision does not.
template <class L, class ST, int COLL, class V, bool OFFSET, class H, class Emit>
__device__ __forceinline__ void emit_outputs_s(const InstDev& P, const Coef<V>& C, H&& h, Emit&& emit) {
    using T = typename Lane<V>::T;
    constexpr int R = L::R;
    constexpr bool H4 = R == 3;
    constexpr bool SCALED = sizeof(ST) == 2, REG = COLL == COLL_REG;
    const T om = kconst<T>(P.omega_c, P.omega_c_f);
    const V omv = vset<V>(om);
    V EA[R + 1], EB[R + 1], OX[R + 1], OY[R + 1], U[R + 1];
#pragma unroll
    for (int m = 0; m <= R; ++m) EA[m] = REG && SCALED ? vadds(C.c0, -(T)P.He[m]) : C.c0;
    // even axis parts of (m, .) and (., n); odd ones
#pragma unroll
    for (int m = 1; m <= R; ++m) {
        const double m2 = (double)m * m;
        EB[m] = vmulk(m2, H4 ? vfmak(m2, C.q04, C.q02) : C.q02);
        OX[m] = vmulk((double)m, H4 ? vfmak(m2, C.c30, C.l10) : C.l10);
        OY[m] = vmulk((double)m, H4 ? vfmak(m2, C.c03, C.l01) : C.l01);
        if (REG && SCALED) OX[m] = vadds(OX[m], -(T)P.Ho[m]);
        U[m] = H4 ? vfmak(4.0 * m2, C.q31, C.q11) : C.q11;
    }
    auto out = [&](int i, V eq) {
        if (REG) {
            emit(i, eq);
        } else {
            // Eq. 14 discretized: f - (f - f^eq)/tau, with the source in f^eq
            const V hi = h(i);
            const V v = vfmac<V>(om, omv, vsub(eq, hi), hi);
            emit(i, OFFSET ? vadds(v, -(T)off_s<L>(P, i)) : v);
        }
    };
    out(0, EA[0]);
    const V rest = EA[0];
#pragma unroll
    for (int m = 1; m <= R; ++m) EA[m] = vfmak((double)m * m, H4 ? vfmak((double)m * m, C.q40, C.q20) : C.q20, EA[m]);
#pragma unroll
    for (int k = 0; k < L::NP; k += 2) {
        const int m = L::px(k), n = L::py(k);
        const int i = 1 + 2 * k;  // +p_k, -p_k, +p_(k+1), -p_(k+1)
        if (n == 0) {
            out(i, vadd(EA[m], OX[m]));
            out(i + 1, vsub(EA[m], OX[m]));
            const V E = vadd(rest, EB[m]);
            // (0, m): c_x = 0, so the odd part holds no offset (Ho[0] = 0)
            out(i + 2, vadd(E, OY[m]));
            out(i + 3, vsub(E, OY[m]));
        } else {
            const double mn = (double)m * n, m2 = (double)m * m, n2 = (double)n * n;
            V S = vadd(EA[m], EB[n]);
            if (H4) S = vfmak(6.0 * m2 * n2, C.q22, S);
            const V M = H4 ? vfmak(4.0 * n2, C.q13, U[m]) : U[m];
            const V Ep = vfmak(mn, M, S), Em = vfmak(-mn, M, S);
            const V ox = H4 ? vfmak(3.0 * m * n2, C.c12, OX[m]) : OX[m];
            const V oy = H4 ? vfmak(3.0 * n * m2, C.c21, OY[n]) : OY[n];
            const V Op = vadd(ox, oy), Om = vsub(ox, oy);
            out(i, vadd(Ep, Op));
            out(i + 1, vsub(Ep, Op));
            out(i + 2, vadd(Em, Om));
            out(i + 3, vsub(Em, Om));
        }
    }
}

// The same; plain BGK takes its offset out where the launch has one (a branch, not predicated operations).
template <class L, class ST, int COLL, class V, class H, class Emit>
__device__ __forceinline__ void emit_outputs(const InstDev& P, const Coef<V>& C, H&& h, Emit&& emit) {
    if constexpr (COLL == COLL_BGK && sizeof(ST) == 2) {
        if (P.stream_off) {
            emit_outputs_s<L, ST, COLL, V, true>(P, C, h, emit);
            return;
        }
    }
    emit_outputs_s<L, ST, COLL, V, false>(P, C, h, emit);
}

}  // namespace lbm
