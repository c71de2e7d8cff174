// Device-side building blocks of the D2Q9 MRT pseudopotential update.
//
// Velocity order e_0..e_8 = (0,0),(1,0),(0,1),(-1,0),(0,-1),(1,1),(-1,1),(-1,-1),(1,-1);
// moment order (rho, e, zeta, j_x, q_x, j_y, q_y, p_xx, p_xy) of the standard D2Q9
// transformation matrix M (Sec. II). All constants below are written out by hand.
//
// The collision works on PAIRS of sites held in a two-lane vector: in FP32 the lanes are
// packed into one register pair and every add / subtract / multiply / fma is a single
// packed instruction of sm_100-class GPUs (__fadd2_rn, sub.rn.f32x2, __fmul2_rn,
// __ffma2_rn, each lane rounded exactly like the scalar operation); in FP64 the two lanes
// are plain scalar doubles.
#pragma once

#include <climits>

#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include "lb_internal.h"

namespace lbm {

// Storage element -> arithmetic type: BF16 storage (LB_BF16) is worked on in FP32.
template <typename T>
struct ArithOf { using type = T; };
template <>
struct ArithOf<__nv_bfloat16> { using type = float; };
template <typename T>
using Arith = typename ArithOf<T>::type;
template <typename T>
constexpr bool PLAIN_OF = std::is_same<T, __nv_bfloat16>::value;   // see collide_plain

// The update's constants as values of type C: the arithmetic type itself in kernel parameters
// (DevConsts), pairs (v, v) where a kernel keeps them in shared memory (lb_tile.cuh): a packed
// operation then takes its constant as loaded.
template <typename C>
struct ConstFields {
    C b4;                                  // Carnahan-Starling, 2/G folded in: see eos_psi
    C rtc, a2, c3;
    C psi0, rho0;
    C th_v, th_m, th_l, rho1, rho2, p_rho1, p_rho2;
    C two_over_G;
    C G, mG12, qk3;                        // G, -G/12, kappa G / 6
    // Eq. 17 coefficients of the moments as M^-1 uses them (collide): (e + 2 rho)/36,
    // (zeta - rho)/36, q/12, p/4. *_m multiplies the moment itself (1 - s); the others, in the
    // order of the terms of collide, the equilibrium, the forcing (1 - s/2) and the source.
    // Rounded once from FP64.
    C e_m, e_w, e_fs, e_ss, e_tr;
    C z_m, z_w, z_fs, z_ss, z_tr;
    C q_m, q_j, q_f;
    C v_m, v_u, v_f2, v_f4, v_q4, v_q16;
    // storage shift w_a rho_s: LB_BF16 stores f_a - w_a rho_s (zero for FP32 / FP64)
    C wshift[9];
    C rho_s;
    // nu(rho) (open-boundary kernels only): sites with rho < rho_sw relax p_xx, p_xy at
    // s_vV; the v_* coefficients for that rate
    C rho_sw, v_m_V, v_u_V, v_f2_V, v_f4_V, v_q4_V, v_q16_V;
};
// The constants of collide_plain and of its psi: Eq. 17's (1 - s), s, (1 - s/2) and source weights
// of the unscaled moments, rounded once from FP64; *_V: of the vapour's rate.
template <typename T>
struct PlainConsts {
    T a, RT, mG, kG2, sig_coef, rho_sw, rho_s;
    T e_keep, s_e, e_half, e_src, z_keep, s_z, z_half, z_src, q_keep, s_q, q_half;
    T v_keep, s_v, v_half, v_src, v_keep_V, s_v_V, v_half_V, v_src_V;
};
template <typename T>
struct DevConsts : ConstFields<T> {
    PlainConsts<T> sw;
    int stall_row;                         // test hook (lb_debug_stall_row): kernels that wait for rows,
    unsigned vain_bytes;                   // and staged tiles
    // LB_BF16 stochastic rounding: the step of the launch (the counter)
    unsigned sr_step;
};

// Per-lattice record of the batched step (lives in a device table).
template <typename T>
struct BatchLattice {
    T *g[2];              // the lattice's two population buffers
    DevConsts<T> P;
    int nx, ny, pitch;
    unsigned plane;
    int frozen;           // 1: set inactive (not stepped); its state stays in g[0]
};

template <typename T>
inline DevConsts<T> to_dev(const Consts &c) {
    DevConsts<T> d;
    d.b4 = T(c.b4);
    d.rtc = T(c.RT * c.two_over_G);
    d.a2 = T(c.a * c.two_over_G);
    d.c3 = T(c.two_over_G / 3.0);
    d.psi0 = T(c.psi0); d.rho0 = T(c.rho0);
    d.th_v = T(c.th_v); d.th_m = T(c.th_m); d.th_l = T(c.th_l);
    d.rho1 = T(c.rho1); d.rho2 = T(c.rho2); d.p_rho1 = T(c.p_rho1); d.p_rho2 = T(c.p_rho2);
    d.two_over_G = T(c.two_over_G);
    d.G = T(c.G); d.mG12 = T(-c.G / 12.0); d.qk3 = T(c.kG2 / 3.0);
    const double e_keep = 1.0 - c.s_e, e_half = 1.0 - 0.5 * c.s_e;
    d.e_m = T(e_keep / 36.0); d.e_w = T(c.s_e / 12.0);
    d.e_fs = T(e_half / 6.0); d.e_ss = T(e_half * c.sig_coef / 5184.0); d.e_tr = T(c.s_e / 24.0);
    const double z_keep = 1.0 - c.s_z, z_half = 1.0 - 0.5 * c.s_z;
    d.z_m = T(z_keep / 12.0); d.z_w = T(-c.s_z / 12.0);   // times (zeta - rho)/3 = f_0 - sum f_1..4
    d.z_fs = T(-z_half / 6.0); d.z_ss = T(-z_half * c.sig_coef / 5184.0); d.z_tr = T(-c.s_z / 24.0);
    d.q_m = T((1.0 - c.s_q) / 12.0); d.q_j = T(-c.s_q / 12.0);
    d.q_f = T(-(1.0 - 0.5 * c.s_q) / 12.0);
    auto rate_v = [](double s, T &m, T &u, T &f2, T &f4, T &q4, T &q16) {
        const double h = 1.0 - 0.5 * s;
        m = T((1.0 - s) / 4.0); u = T(s / 4.0); f2 = T(h / 2.0); f4 = T(h / 4.0);
        q4 = T(-s / 4.0); q16 = T(-s / 16.0);
    };
    rate_v(c.s_v, d.v_m, d.v_u, d.v_f2, d.v_f4, d.v_q4, d.v_q16);
    rate_v(c.s_v_vapour, d.v_m_V, d.v_u_V, d.v_f2_V, d.v_f4_V, d.v_q4_V, d.v_q16_V);
    for (int a = 0; a < 9; ++a)
        d.wshift[a] = T((a == 0 ? 4.0 / 9.0 : (a <= 4 ? 1.0 / 9.0 : 1.0 / 36.0)) * c.shift_rho);
    d.rho_s = T(c.shift_rho);
    d.rho_sw = T(c.rho_sw);
    PlainConsts<T> &w = d.sw;
    w.a = T(c.a); w.RT = T(c.RT); w.rho_s = T(c.shift_rho);
    w.mG = T(-c.G); w.kG2 = T(c.kG2); w.sig_coef = T(c.sig_coef); w.rho_sw = T(c.rho_sw);
    w.e_keep = T(1.0 - c.s_e); w.s_e = T(c.s_e); w.e_half = T(1.0 - 0.5 * c.s_e); w.e_src = T(1.5 * c.s_e);
    w.z_keep = T(1.0 - c.s_z); w.s_z = T(c.s_z); w.z_half = T(1.0 - 0.5 * c.s_z); w.z_src = T(1.5 * c.s_z);
    w.q_keep = T(1.0 - c.s_q); w.s_q = T(c.s_q); w.q_half = T(1.0 - 0.5 * c.s_q);
    w.v_keep = T(1.0 - c.s_v); w.s_v = T(c.s_v); w.v_half = T(1.0 - 0.5 * c.s_v); w.v_src = T(-c.s_v);
    w.v_keep_V = T(1.0 - c.s_v_vapour); w.s_v_V = T(c.s_v_vapour);
    w.v_half_V = T(1.0 - 0.5 * c.s_v_vapour); w.v_src_V = T(-c.s_v_vapour);
    d.stall_row = c.stall_row;
    d.vain_bytes = c.stall_row != INT_MIN ? 16 : 0;
    d.sr_step = c.step_key;
    return d;
}

// ---- scalar helpers: FP32 uses the hardware approximations (a few ulp, far inside the
// FP32 error budget), FP64 IEEE-rounded operations (its division within one ulp: the
// product with the rounded reciprocal). Every add / multiply / fma is an
// explicit round-to-nearest intrinsic, so the compiler cannot contract them differently
// at different inline sites: a site's psi is bitwise the same wherever it is computed. --
__device__ __forceinline__ float lb_exp(float v) { return __expf(v); }
__device__ __forceinline__ double lb_exp(double v) { return exp(v); }
// FP32 reciprocal and reciprocal square root: one hardware approximation each (PTX
// rcp.approx / rsqrt.approx, within two ulp), subnormal inputs and results flushed to zero
// (.ftz): the update meets no subnormal density, pressure or potential, and the
// non-flushing forms add range fix-ups around every approximation.
__device__ __forceinline__ float rcp_ftz(float v) {
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(v));
    return r;
}
__device__ __forceinline__ float rsqrt_ftz(float v) {
    float r;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(v));
    return r;
}
__device__ __forceinline__ float lb_div(float a, float b) { return __fmul_rn(a, rcp_ftz(b)); }
// FP64 a / b as a times the correctly rounded 1 / b (within one ulp of the quotient)
__device__ __forceinline__ double lb_div(double a, double b) { return __dmul_rn(a, __drcp_rn(b)); }
__device__ __forceinline__ float lb_rcp(float v) { return rcp_ftz(v); }
__device__ __forceinline__ double lb_rcp(double v) { return __drcp_rn(v); }   // = 1 / v rounded
__device__ __forceinline__ float lb_sqrt_pos(float v) { return __fmul_rn(v, rsqrt_ftz(v)); }   // v > 0
__device__ __forceinline__ double lb_sqrt_pos(double v) { return __dsqrt_rn(v); }
__device__ __forceinline__ float radd(float a, float b) { return __fadd_rn(a, b); }
__device__ __forceinline__ double radd(double a, double b) { return __dadd_rn(a, b); }
__device__ __forceinline__ float rsub(float a, float b) { return __fsub_rn(a, b); }
__device__ __forceinline__ double rsub(double a, double b) { return __dsub_rn(a, b); }
__device__ __forceinline__ float rmul(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ double rmul(double a, double b) { return __dmul_rn(a, b); }
__device__ __forceinline__ float rfma(float a, float b, float c) { return __fmaf_rn(a, b, c); }
__device__ __forceinline__ double rfma(double a, double b, double c) { return __fma_rn(a, b, c); }

// ---- stored population <-> value. FP32 / FP64 store f itself; LB_BF16 stores the FP32
// difference f_a - w_a rho_s rounded to BF16 (nearest even), and reads it back exactly
// as float(stored) + w_a rho_s (one FP32 rounding).
template <typename T>
__device__ __forceinline__ Arith<T> pop_dec(T v, int, const DevConsts<Arith<T>> &) { return v; }
template <>
__device__ __forceinline__ float pop_dec<__nv_bfloat16>(__nv_bfloat16 v, int a,
                                                         const DevConsts<float> &P) {
    return __fadd_rn(__bfloat162float(v), P.wshift[a]);
}
// MurmurHash3's 32-bit finaliser (fmix32; A. Appleby, public domain): a bijective mix of a
// 32-bit counter into well-spread bits, the generator of the stochastic rounding below.
__device__ __forceinline__ unsigned mix32(unsigned h) {
    h ^= h >> 16;
    h *= 0x85ebca6bu;
    h ^= h >> 13;
    h *= 0xc2b2ae35u;
    h ^= h >> 16;
    return h;
}

// The counter of a site pair (first column x, row y) in the step of the launch, and the 32
// random bits of its population a (16 per site of the pair): reproducible, and independent
// of the launch shape.
__device__ __forceinline__ unsigned sr_pair_key(int x, int y, unsigned step) {
    return mix32(mix32((unsigned)y * 0x9e3779b1u + (unsigned)x) ^ (step * 0x85ebca6bu));
}
__device__ __forceinline__ unsigned sr_bits(unsigned key, int a) {
    return mix32(key + (unsigned)(a + 1) * 0x9e3779b9u);
}

// BF16 of v rounded stochastically with the 16 random bits r16: r16 is added below the
// kept bits and the rest cut off, so the magnitude rounds up with probability (dropped
// bits) / 2^16 and the expected stored value is v.
__device__ __forceinline__ __nv_bfloat16 bf16_stochastic(float v, unsigned r16) {
    unsigned b = __float_as_uint(v);
    if ((b & 0x7f800000u) != 0x7f800000u) b += r16 & 0xffffu;   // not Inf / NaN
    __nv_bfloat16_raw raw;
    raw.x = (unsigned short)(b >> 16);
    return __nv_bfloat16(raw);
}

// SR: LB_BF16 with stochastic rounding, r16 its random bits; otherwise nearest even
template <typename T, bool SR = false>
__device__ __forceinline__ T pop_enc(Arith<T> v, int a, const DevConsts<Arith<T>> &P,
                                     unsigned r16 = 0) {
    if constexpr (std::is_same<T, __nv_bfloat16>::value) {
        const float d = __fsub_rn(v, P.wshift[a]);
        if constexpr (SR) return bf16_stochastic(d, r16);
        else return __float2bfloat16_rn(d);
    } else {
        (void)a; (void)P; (void)r16;
        return v;
    }
}

// a constant as a scalar, however the kernel keeps it (ConstFields)
template <typename T>
struct V2;
template <typename T>
__device__ __forceinline__ T scalar(T v) { return v; }
template <typename T>
__device__ __forceinline__ T scalar(const V2<T> &v) { return v.lo(); }

// Interaction potential psi(rho) (Sec. II): psi0 exp(-rho0/rho), or
// sqrt(2 (p_EOS - rho c_s^2) / G) with p_EOS the Carnahan-Starling EOS or Eq. 23.
// Sets `bad` when rho <= 0 or psi^2 <= 0 (the value is then not usable).
// PLAIN: psi of the BF16 steps, whose arithmetic stays as it is (see collide_plain).
template <typename T, int EOS, bool PLAIN = false, typename PT>
__device__ __forceinline__ T eos_psi(T rho, const PT &P, bool &bad) {
    if constexpr (EOS == LB_EOS_EXP) {
        bad |= !(rho > T(0));
        return rmul(scalar<T>(P.psi0), lb_exp(-lb_div(scalar<T>(P.rho0), rho)));
    } else {
        T arg;   // 2 (p_EOS - rho/3) / G
        if constexpr (EOS == LB_EOS_CS) {
            // p = rho RT (1 + eta + eta^2 - eta^3) / (1 - eta)^3 - a rho^2; with 2/G folded
            // into the constants, arg = rho RT' poly / den - a' rho^2 - 2 rho/(3G)
            const T eta = rmul(scalar<T>(P.b4), rho);
            const T om = rsub(T(1), eta);
            const T poly = rfma(eta, rfma(eta, om, T(1)), T(1));
            T rt;
            if constexpr (PLAIN) rt = P.sw.RT;
            else rt = scalar<T>(P.rtc);
            const T num = rmul(rmul(rho, rt), poly);
            const T q = rmul(num, lb_rcp(rmul(rmul(om, om), om)));
            if constexpr (PLAIN)
                arg = rmul(rsub(rsub(q, rmul(P.sw.a, rmul(rho, rho))), rmul(rho, T(1.0 / 3.0))), P.two_over_G);
            else if constexpr (std::is_same<T, float>::value)   // the three terms rounded apart: see eos_psi2
                arg = rsub(rsub(q, rmul(scalar<T>(P.a2), rmul(rho, rho))), rmul(rho, scalar<T>(P.c3)));
            else
                arg = rfma(rho, -rfma(scalar<T>(P.a2), rho, scalar<T>(P.c3)), q);
        } else {
            const T p = (rho <= scalar<T>(P.rho1)) ? rmul(rho, scalar<T>(P.th_v))
                      : (rho < scalar<T>(P.rho2)) ? rfma(rsub(rho, scalar<T>(P.rho1)), scalar<T>(P.th_m), scalar<T>(P.p_rho1))
                                       : rfma(rsub(rho, scalar<T>(P.rho2)), scalar<T>(P.th_l), scalar<T>(P.p_rho2));
            arg = rmul(rsub(p, rmul(rho, T(1.0 / 3.0))), scalar<T>(P.two_over_G));
        }
        bad |= !(arg > T(0)) || !(rho > T(0));
        return lb_sqrt_pos(arg);
    }
}

// ---- two-lane vectors ---------------------------------------------------------------
template <typename T>
struct V2;

template <>
struct V2<float> {
    float2 v;
    __device__ __forceinline__ V2() {}
    __device__ __forceinline__ V2(float2 a) : v(a) {}
    __device__ __forceinline__ V2(float a, float b) : v(make_float2(a, b)) {}
    __device__ __forceinline__ static V2 all(float a) { return V2(a, a); }
    __device__ __forceinline__ static V2 all(V2 a) { return a; }   // a constant kept as a pair
    __device__ __forceinline__ float lo() const { return v.x; }
    __device__ __forceinline__ float hi() const { return v.y; }
};
__device__ __forceinline__ V2<float> operator+(V2<float> a, V2<float> b) { return __fadd2_rn(a.v, b.v); }
__device__ __forceinline__ V2<float> operator*(V2<float> a, V2<float> b) { return __fmul2_rn(a.v, b.v); }
__device__ __forceinline__ V2<float> operator-(V2<float> a, V2<float> b) {
    // the packed subtraction (PTX sub.rn.f32x2), lane by lane the rounded a - b
    float2 r;
    asm("{\n\t.reg .b64 ra, rb, rd;\n\t"
        "mov.b64 ra, {%2, %3};\n\tmov.b64 rb, {%4, %5};\n\t"
        "sub.rn.f32x2 rd, ra, rb;\n\tmov.b64 {%0, %1}, rd;\n\t}"
        : "=f"(r.x), "=f"(r.y)
        : "f"(a.v.x), "f"(a.v.y), "f"(b.v.x), "f"(b.v.y));
    return r;
}
__device__ __forceinline__ V2<float> vfma(V2<float> a, V2<float> b, V2<float> c) {
    return __ffma2_rn(a.v, b.v, c.v);
}
__device__ __forceinline__ V2<float> operator-(V2<float> a) { return V2<float>(-a.v.x, -a.v.y); }

template <>
struct V2<double> {
    double x, y;
    __device__ __forceinline__ V2() {}
    __device__ __forceinline__ V2(double a, double b) : x(a), y(b) {}
    __device__ __forceinline__ static V2 all(double a) { return V2(a, a); }
    __device__ __forceinline__ double lo() const { return x; }
    __device__ __forceinline__ double hi() const { return y; }
};
__device__ __forceinline__ V2<double> operator+(V2<double> a, V2<double> b) {
    return {__dadd_rn(a.x, b.x), __dadd_rn(a.y, b.y)};
}
__device__ __forceinline__ V2<double> operator*(V2<double> a, V2<double> b) {
    return {__dmul_rn(a.x, b.x), __dmul_rn(a.y, b.y)};
}
__device__ __forceinline__ V2<double> operator-(V2<double> a, V2<double> b) {
    return {__dsub_rn(a.x, b.x), __dsub_rn(a.y, b.y)};
}
__device__ __forceinline__ V2<double> vfma(V2<double> a, V2<double> b, V2<double> c) {
    return {__fma_rn(a.x, b.x, c.x), __fma_rn(a.y, b.y, c.y)};
}
__device__ __forceinline__ V2<double> operator-(V2<double> a) { return {-a.x, -a.y}; }

// one site (the lane of the scalar kernels), the same operations
template <typename T>
struct V1 {
    T v;
    __device__ __forceinline__ V1() {}
    __device__ __forceinline__ V1(T a) : v(a) {}
    __device__ __forceinline__ static V1 all(T a) { return V1(a); }
};
template <typename T>
__device__ __forceinline__ V1<T> operator+(V1<T> a, V1<T> b) { return radd(a.v, b.v); }
template <typename T>
__device__ __forceinline__ V1<T> operator*(V1<T> a, V1<T> b) { return rmul(a.v, b.v); }
template <typename T>
__device__ __forceinline__ V1<T> operator-(V1<T> a, V1<T> b) { return rsub(a.v, b.v); }
template <typename T>
__device__ __forceinline__ V1<T> operator-(V1<T> a) { return V1<T>(-a.v); }
template <typename T>
__device__ __forceinline__ V1<T> vfma(V1<T> a, V1<T> b, V1<T> c) { return rfma(a.v, b.v, c.v); }

template <typename T>
__device__ __forceinline__ V2<T> vrcp(V2<T> a) { return V2<T>(lb_rcp(a.lo()), lb_rcp(a.hi())); }
template <typename T>
__device__ __forceinline__ V1<T> vrcp(V1<T> a) { return V1<T>(lb_rcp(a.v)); }
// per lane: a >= limit ? x : y
template <typename T>
__device__ __forceinline__ V2<T> pick_ge(V2<T> a, T limit, T x, T y) {
    return V2<T>(a.lo() >= limit ? x : y, a.hi() >= limit ? x : y);
}
template <typename T>
__device__ __forceinline__ V1<T> pick_ge(V1<T> a, T limit, T x, T y) {
    return V1<T>(a.v >= limit ? x : y);
}

// psi of two densities; lane by lane the same operations, in the same order and with
// the same rounding, as eos_psi (so a site's psi does not depend on which lane or which
// kernel computes it). `hi_valid` = false: the second lane is padding and is not checked.
template <typename T, int EOS, bool PLAIN = false, typename PT>
__device__ __forceinline__ V2<T> eos_psi2(V2<T> rho, const PT &P, bool hi_valid, bool &bad) {
    if constexpr (EOS == LB_EOS_CS) {
        using V = V2<T>;
        const V one = V::all(T(1));
        const V eta = V::all(P.b4) * rho;
        const V om = one - eta;
        const V poly = vfma(eta, vfma(eta, om, one), one);
        V rt;
        if constexpr (PLAIN) rt = V::all(P.sw.RT);
        else rt = V::all(P.rtc);
        const V num = (rho * rt) * poly, den = (om * om) * om;
        V q;
        if constexpr (PLAIN) q = V(lb_div(num.lo(), den.lo()), lb_div(num.hi(), den.hi()));
        else q = num * vrcp(den);
        // In FP32 the three terms are rounded one by one: arg is a small difference of terms of
        // the order of rho, and the fused form (two operations fewer) rounds 2 a rho + 2/3, twice
        // their size; the pressure it left in a liquid at 0.8 T_c doubled the error of a droplet
        // after 200 steps against FP64 (1.3e-6 against 6e-7). In FP64 the error of a run is the same
        // either way (1.1e-15 of the largest population), and two operations fewer count.
        V arg;
        if constexpr (PLAIN)
            arg = ((q - V::all(P.sw.a) * (rho * rho)) - rho * V::all(T(1.0 / 3.0))) * V::all(P.two_over_G);
        else if constexpr (std::is_same<T, float>::value)
            arg = (q - V::all(P.a2) * (rho * rho)) - rho * V::all(P.c3);
        else
            arg = vfma(rho, -vfma(V::all(P.a2), rho, V::all(P.c3)), q);
        bad |= !(arg.lo() > T(0)) || !(rho.lo() > T(0));
        if (hi_valid) bad |= !(arg.hi() > T(0)) || !(rho.hi() > T(0));
        return V(lb_sqrt_pos(arg.lo()), lb_sqrt_pos(arg.hi()));
    } else {
        bool b2 = false;
        const T lo = eos_psi<T, EOS, PLAIN>(rho.lo(), P, bad);
        const T hi = eos_psi<T, EOS, PLAIN>(rho.hi(), P, b2);
        if (hi_valid) bad |= b2;
        return V2<T>(lo, hi);
    }
}

// The collision of the steps in which a rounding decides, with the moments as they are: m* = (1 - s)
// m + s m_eq + (1 - s/2) S + C of Eq. 17, then M^-1 m*. VSW: the viscosity switch of FP32 lattices
// with open boundaries: a site whose rho lies within the rounding errors of rho_sw takes one
// viscosity or the other, which moves populations by up to 1e-3 of the largest and is carried on.
// SH: BF16 storage, where one rounding of the FP32 value sends the stored one to its other
// neighbour, and with it a reproducible run (with stochastic rounding, one of its random walks) to
// another. So the arithmetic of these stays as it is, operation by operation (collide, below, has
// 30 operations fewer and a smaller error, but another one). SH: f holds f_a - w_a rho_s; the shift
// only moves the moments rho, e and zeta (M w = (1, -2, 1, 0, ..., 0)), so those are corrected by
// rho_s, and the same is taken off m* before M^-1 gives the shifted f* that is stored.
template <typename T, bool VSW, bool SH, typename V>
__device__ __forceinline__ void collide_plain(V (&f)[9], const V (&pn)[9], const PlainConsts<T> &P) {
    const V third = V::all(T(1.0 / 3.0)), twelfth = V::all(T(1.0 / 12.0));
    const V two = V::all(T(2)), four = V::all(T(4)), half = V::all(T(0.5)), mtwo = V::all(T(-2));
    const V pc = pn[0];

    // Eq. 7 force and Eq. 19 differences
    const V dg_pp = pn[5] - pn[7], dg_mp = pn[6] - pn[8];
    const V Sx = vfma(third, pn[1] - pn[3], twelfth * (dg_pp - dg_mp));
    const V Sy = vfma(third, pn[2] - pn[4], twelfth * (dg_pp + dg_mp));
    const V mGpc = V::all(P.mG) * pc;
    const V Fx = mGpc * Sx, Fy = mGpc * Sy;
    const V dsum = vfma(V::all(T(-4)), pc, (pn[5] + pn[6]) + (pn[7] + pn[8]));
    const V qpre = V::all(P.kG2) * pc, tdsum = twelfth * dsum;
    const V Qxx = qpre * vfma(third, vfma(mtwo, pc, pn[1] + pn[3]), tdsum);
    const V Qyy = qpre * vfma(third, vfma(mtwo, pc, pn[2] + pn[4]), tdsum);
    const V Qxy = qpre * (twelfth * ((pn[5] + pn[7]) - (pn[6] + pn[8])));

    // moments m = M f
    const V ax = f[1] + f[3], ay = f[2] + f[4];
    const V d13 = f[1] - f[3], d24 = f[2] - f[4];
    const V s57 = f[5] + f[7], s68 = f[6] + f[8];
    const V d57 = f[5] - f[7], d68 = f[6] - f[8];
    const V axis = ax + ay, diag = s57 + s68;
    const V rsum = f[0] + (axis + diag);       // sum of f (of the shifted f when SH)
    const V rs = V::all(P.rho_s);
    V rho = rsum;
    if constexpr (SH) rho = rsum + rs;
    const V jx = d13 + (d57 - d68), jy = d24 + (d57 + d68);
    V m1 = vfma(two, diag, vfma(V::all(T(-4)), f[0], -axis));
    V m2 = vfma(four, f[0], vfma(mtwo, axis, diag));
    if constexpr (SH) {
        m1 = vfma(mtwo, rs, m1);
        m2 = m2 + rs;
    }
    const V m4 = vfma(mtwo, d13, d57 - d68), m6 = vfma(mtwo, d24, d57 + d68);

    // Eq. 6 velocity, Eq. 3 equilibria, Eqs. 5 and 8 forcing, Eq. 18 source
    const V rinv = vrcp(rho);
    const V vx = vfma(half, Fx, jx) * rinv, vy = vfma(half, Fy, jy) * rinv;
    const V vxx = vx * vx, vyy = vy * vy, v2 = vxx + vyy;
    const V meq1 = rho * vfma(V::all(T(3)), v2, mtwo);
    const V meq2 = rho * vfma(V::all(T(-3)), v2, V::all(T(1)));
    const V rvx = rho * vx, rvy = rho * vy;
    const V S1 = vfma(V::all(T(6)), vfma(vx, Fx, vy * Fy), V::all(P.sig_coef) * vfma(Sx, Sx, Sy * Sy));
    const V S7 = two * (vx * Fx - vy * Fy);
    const V S8 = vfma(vx, Fy, vy * Fx);
    const V tr = Qxx + Qyy;

    // Eq. 17
    V ms1 = vfma(V::all(P.e_keep), m1, vfma(V::all(P.s_e), meq1, vfma(V::all(P.e_half), S1, V::all(P.e_src) * tr)));
    V ms2 = vfma(V::all(P.z_keep), m2, vfma(V::all(P.s_z), meq2, -vfma(V::all(P.z_half), S1, V::all(P.z_src) * tr)));
    const V ms3 = jx + Fx, ms5 = jy + Fy;
    const V ms4 = vfma(V::all(P.q_keep), m4, -vfma(V::all(P.s_q), rvx, V::all(P.q_half) * Fx));
    const V ms6 = vfma(V::all(P.q_keep), m6, -vfma(V::all(P.s_q), rvy, V::all(P.q_half) * Fy));
    V vkeep = V::all(P.v_keep), vs = V::all(P.s_v), vhalf = V::all(P.v_half), vsrc = V::all(P.v_src);
    if constexpr (VSW) {
        vkeep = pick_ge(rho, P.rho_sw, P.v_keep, P.v_keep_V);
        vs = pick_ge(rho, P.rho_sw, P.s_v, P.s_v_V);
        vhalf = pick_ge(rho, P.rho_sw, P.v_half, P.v_half_V);
        vsrc = pick_ge(rho, P.rho_sw, P.v_src, P.v_src_V);
    }
    const V ms7 = vfma(vkeep, ax - ay, vfma(vs, rho * (vxx - vyy), vfma(vhalf, S7, vsrc * (Qxx - Qyy))));
    const V ms8 = vfma(vkeep, s57 - s68, vfma(vs, rvx * vy, vfma(vhalf, S8, vsrc * Qxy)));

    // f* = M^-1 m*; f*_0 from mass conservation, so that rounded constants add no mass
    if constexpr (SH) {                        // back to the moments of the shifted f*
        ms1 = vfma(two, rs, ms1);
        ms2 = ms2 - rs;
    }
    const V c18 = V::all(T(1.0 / 18.0)), c36 = V::all(T(1.0 / 36.0));
    const V c6 = V::all(T(1.0 / 6.0)), c4 = V::all(T(0.25));
    const V a0 = V::all(T(1.0 / 9.0)) * rsum;
    const V base_axis = a0 - vfma(c36, ms1, c18 * ms2);
    const V base_diag = vfma(c18, ms1, vfma(c36, ms2, a0));
    const V jx6 = c6 * ms3, qx6 = c6 * ms4, jy6 = c6 * ms5, qy6 = c6 * ms6;
    const V pxx4 = c4 * ms7, pxy4 = c4 * ms8;
    const V ax1 = jx6 - qx6, ay1 = jy6 - qy6;
    f[1] = base_axis + (ax1 + pxx4);
    f[3] = base_axis + (pxx4 - ax1);
    f[2] = base_axis + (ay1 - pxx4);
    f[4] = base_axis - (ay1 + pxx4);
    const V xp = vfma(twelfth, ms4, jx6), yp = vfma(twelfth, ms6, jy6);
    const V xy_p = xp + yp, xy_m = xp - yp;
    f[5] = base_diag + (xy_p + pxy4);
    f[6] = base_diag - (xy_m + pxy4);
    f[7] = base_diag - (xy_p - pxy4);
    f[8] = base_diag + (xy_m - pxy4);
    f[0] = rsum - (((f[1] + f[3]) + (f[2] + f[4])) + ((f[5] + f[7]) + (f[6] + f[8])));
}

// One collision for the sites of a vector V (V2: two sites, V1: one): f[9] (populations
// after streaming, pre-collision) and the potential at the sites and their neighbours
// pn[a] = psi(x + e_a) (pn[0] = psi(x)) give f*[9] in place.
//
// Arithmetic (identical in exact arithmetic to Eqs. 3, 5-8, 17-19 and f* = M^-1 m*):
//   12 S = 12 sum_a w_a psi(x+e_a) e_a,      F = -G psi(x) S                        (Eq. 7)
//   Q = kappa G/2 psi(x) sum_a w_a (psi_a - psi) e_a e_a enters only as Q_xx + Q_yy,
//   Q_xx - Q_yy and 4 Q_xy                                                         (Eq. 19)
//   rho v = j + F/2                                                                 (Eq. 6)
//   |F|^2 / psi^2 in Eq. 8 is evaluated as G^2 |S|^2 (no division by psi)
//   m*_rho = rho and m*_j = j + F for every s_j (relaxing j towards rho v = j + F/2 and
//   adding (1 - s_j/2) F cancels s_j exactly), so s_rho and s_j drop out;
//   m*_k = (1 - s_k) m_k + s_k m_eq_k + (1 - s_k/2) S_k + C_k for the other moments, formed
//   directly as (e + 2 rho)/36, (zeta - rho)/36, q/12 and p/4: the multiples that M^-1 adds
//   up, and e and zeta as departures from rest, which are small, so that their roundings are
//   too. The products with rho v are taken before the division by rho is multiplied back.
//   That is 120 operations and one reciprocal per site (FP64, whose pipe is the bound of
//   the FP64 step; the form with unscaled moments took 150: 1000 x 700 FP64 steps in 280
//   against 333 us, FP32 2048^2 1 % faster).
//   VSW: nu(rho) of Sec. V.C, the rate of p_xx, p_xy (and the weight of their source
//   terms) taken per site as s_v where rho >= rho_sw, else s_vV.
//   SH: LB_BF16, see collide_plain.
template <typename T, bool VSW = false, bool SH = false, typename V, typename PT>
__device__ __forceinline__ void collide(V (&f)[9], const V (&pn)[9], const PT &P) {
    if constexpr (SH || (VSW && std::is_same<T, float>::value)) {
        collide_plain<T, VSW, SH>(f, pn, P.sw);
        return;
    }
    const V four = V::all(T(4)), half = V::all(T(0.5)), mtwo = V::all(T(-2)), mfour = V::all(T(-4));
    const V pc = pn[0];

    // Eq. 7 neighbour sums (times 12) and the three combinations of Eq. 19
    const V dg_pp = pn[5] - pn[7];
    const V dg_mp = pn[6] - pn[8];
    const V Sx = vfma(four, pn[1] - pn[3], dg_pp - dg_mp);
    const V Sy = vfma(four, pn[2] - pn[4], dg_pp + dg_mp);
    const V gp = V::all(P.mG12) * pc;
    const V Fx = gp * Sx;
    const V Fy = gp * Sy;
    const V pa = pn[1] + pn[3], pb = pn[2] + pn[4];
    const V p57 = pn[5] + pn[7], p68 = pn[6] + pn[8];
    const V qp = V::all(P.qk3) * pc;
    const V dsum = vfma(mfour, pc, p57 + p68);
    const V tr = qp * vfma(half, dsum, vfma(mfour, pc, pa + pb));   // Q_xx + Q_yy
    const V dq = qp * (pa - pb);                                     // Q_xx - Q_yy
    const V qxy4 = qp * (p57 - p68);                                 // 4 Q_xy

    // moments m = M f
    const V ax = f[1] + f[3], ay = f[2] + f[4];
    const V d13 = f[1] - f[3], d24 = f[2] - f[4];
    const V s57 = f[5] + f[7], s68 = f[6] + f[8];
    const V d57 = f[5] - f[7], d68 = f[6] - f[8];
    const V axis = ax + ay, diag = s57 + s68;
    const V moving = axis + diag;
    const V rho = f[0] + moving;
    const V dm = d57 - d68, dp = d57 + d68;
    const V jx = d13 + dm;
    const V jy = d24 + dp;
    const V m1 = vfma(four, diag, vfma(mtwo, f[0], axis));      // e + 2 rho
    const V m2 = f[0] - axis;                                    // (zeta - rho)/3
    const V m4 = vfma(mtwo, d13, dm);
    const V m6 = vfma(mtwo, d24, dp);
    const V m7 = ax - ay;
    const V m8 = s57 - s68;

    // Eq. 6 velocity; products for Eqs. 3, 5 and 8
    const V rinv = vrcp(rho);
    const V rvx = vfma(half, Fx, jx), rvy = vfma(half, Fy, jy);
    const V vx = rvx * rinv, vy = rvy * rinv;
    const V ryy = rvy * vy;
    const V w = vfma(rvx, vx, ryy), u = vfma(rvx, vx, -ryy);     // rho (v_x^2 +- v_y^2)
    const V xy = rvx * vy;
    const V fyy = vy * Fy;
    const V fs = vfma(vx, Fx, fyy), fd = vfma(vx, Fx, -fyy);     // v_x F_x +- v_y F_y
    const V S8 = vfma(vx, Fy, vy * Fx);
    const V ss = vfma(Sx, Sx, Sy * Sy);

    // Eq. 17, scaled as M^-1 uses the moments
    const V de = vfma(V::all(P.e_m), m1, vfma(V::all(P.e_w), w, vfma(V::all(P.e_fs), fs,
                      vfma(V::all(P.e_ss), ss, V::all(P.e_tr) * tr))));
    const V dz = vfma(V::all(P.z_m), m2, vfma(V::all(P.z_w), w, vfma(V::all(P.z_fs), fs,
                      vfma(V::all(P.z_ss), ss, V::all(P.z_tr) * tr))));
    const V qx = vfma(V::all(P.q_m), m4, vfma(V::all(P.q_j), rvx, V::all(P.q_f) * Fx));
    const V qy = vfma(V::all(P.q_m), m6, vfma(V::all(P.q_j), rvy, V::all(P.q_f) * Fy));
    V vm = V::all(P.v_m), vu = V::all(P.v_u), vf2 = V::all(P.v_f2), vf4 = V::all(P.v_f4);
    V vq4 = V::all(P.v_q4), vq16 = V::all(P.v_q16);
    if constexpr (VSW) {
        vm = pick_ge(rho, P.rho_sw, P.v_m, P.v_m_V);
        vu = pick_ge(rho, P.rho_sw, P.v_u, P.v_u_V);
        vf2 = pick_ge(rho, P.rho_sw, P.v_f2, P.v_f2_V);
        vf4 = pick_ge(rho, P.rho_sw, P.v_f4, P.v_f4_V);
        vq4 = pick_ge(rho, P.rho_sw, P.v_q4, P.v_q4_V);
        vq16 = pick_ge(rho, P.rho_sw, P.v_q16, P.v_q16_V);
    }
    const V pxx = vfma(vm, m7, vfma(vu, u, vfma(vf2, fd, vq4 * dq)));
    const V pxy = vfma(vm, m8, vfma(vu, xy, vfma(vf4, S8, vq16 * qxy4)));

    // f* = M^-1 m*, M^-1 = M^T diag(1/9, 1/36, 1/36, 1/6, 1/12, 1/6, 1/12, 1/4, 1/4)
    const V c6 = V::all(T(1.0 / 6.0));
    const V base_axis = vfma(V::all(T(1.0 / 9.0)), rho, -vfma(V::all(T(2)), dz, de));
    const V base_diag = vfma(V::all(T(1.0 / 36.0)), rho, vfma(V::all(T(2)), de, dz));
    // j* = j + F as 4 (j*/6 + q/12) along the diagonals and the rest along the axes, so that a
    // rounded 1/6 (which in FP32 adds 3e-8 of the momentum at every step) does not enter it (160
    // steps of a 600 x 225 splash with this collision, error against FP64: 2.6e-7 against 1.5e-6)
    const V jxn = jx + Fx, jyn = jy + Fy;
    const V xp = vfma(c6, jxn, qx), yp = vfma(c6, jyn, qy);
    const V ax1 = vfma(mtwo, xp, half * jxn), ay1 = vfma(mtwo, yp, half * jyn);
    f[1] = base_axis + (ax1 + pxx);
    f[3] = base_axis + (pxx - ax1);
    f[2] = base_axis + (ay1 - pxx);
    f[4] = base_axis - (ay1 + pxx);
    const V xy_p = xp + yp, xy_m = xp - yp;
    f[5] = base_diag + (xy_p + pxy);
    f[6] = base_diag - (xy_m + pxy);
    f[7] = base_diag - (xy_p - pxy);
    f[8] = base_diag + (xy_m - pxy);
    // f*_0 from mass conservation instead of (m*_0 - m*_1 + m*_2)/9: with the rounded
    // constants the column sums of M^-1 are not exactly (1, 0, ..., 0), which in FP32 adds mass
    // at about 7e-9 per step. In FP32 it is f_0 plus what the moving populations lost, the two
    // sums over them formed alike: in a uniform fluid their roundings cancel, where rho - sum
    // f*_a adds the same one at every step (a 501 x 383 droplet after 200 steps, error against
    // FP64: 7.3e-7 against 1.1e-6; the unscaled moments of collide_plain had 6.2e-7 there, and more
    // than these elsewhere: a 4096 x 2048 wave 6.6e-7 / 3.0e-7, 24 droplets of 128^2 1.3e-6 / 3.7e-7).
    // In FP64 the eight f*_a sum to 4 (base_axis + base_diag) up
    // to their own unbiased roundings, two operations instead of nine.
    if constexpr (std::is_same<T, double>::value)
        f[0] = vfma(mfour, base_axis + base_diag, rho);
    else
        f[0] = f[0] + (moving - (((f[1] + f[3]) + (f[2] + f[4])) + ((f[5] + f[7]) + (f[6] + f[8]))));
}

}  // namespace lbm
