// Fused pull stream-and-collide kernels for the PR and IR Bingham models.
//
// One thread owns one cell (k_step; k_step2 runs two cells per thread with
// the collision in packed two-wide FP32).  Per fluid cell and time step it
//   1. gathers the Q incoming populations (eq. 8, pull form): population i
//      comes from the cell at x - c_i (periodic wrap) or, when that cell is
//      solid, is the cell's own outgoing population in the opposite direction
//      (halfway bounce-back, Sec. 4.3);
//   2. forms the moments rho, j, Pi (eq. MomentsLBM) in registers;
//   3. collides:
//      PR  T = Pi - rho c_s^2 I - rho u u, D = -T/(2 tau_old c_s^2)
//          (eq. LBM_strain_rate), gdot = sqrt(2 D:D), nu_app from eqs.
//          (Pap_reg_1)/(PR_interpolation), tau = 1/2 + nu_app/c_s^2
//          (eq. tau_visc), or the Newton-implicit tau of Sec. 3; TRT with
//          tau_odd from Lambda (Sec. 2.1) and the exact-difference force of
//          eq. (14);
//      IR  u = (j + F/2)/rho, T as above, the closed-form solution of
//          eq. (Vikh_main_short) (eqs. Vikh_sigmaS_formula/tensor, yield where
//          |T| >= sqrt2 sigma_y), A = -sigma_bar + s/2, and the post-collision
//          populations f_eq + w/(2 c_s^4)(cc - c_s^2 I):A + Phi/2 of
//          eqs. (Vikh_postCol)/(Vikh_f_stress)/(Vikh_force);
//   4. stores the Q outgoing populations (and, PR, the new tau in place).
//
// Populations are stored as offsets f_i - w_i from the rest state (scaled per
// direction for the 16-bit forms), so every moment is formed from small
// numbers (no cancellation against the weights).  On check steps the same
// launch also accumulates the flow-rate sums and the residual against the
// previous snapshot into per-block partials, summed in FP64 in a fixed order.
#pragma once

#include <algorithm>
#include <atomic>
#include <cstdint>
#include <type_traits>
#include <utility>

#include <cuda_bf16.h>
#include <cuda_fp16.h>
#include <cuda_runtime.h>

#include "../../include/bingham_lbm.h"
#include "lattice.cuh"
#include "lbm_internal.h"

namespace blbm {

// ---------------------------------------------------------------------------
// compile-time loop
template <int I, int N, class F>
__device__ __forceinline__ void static_for(F&& f) {
    if constexpr (I < N) {
        f(std::integral_constant<int, I>{});
        static_for<I + 1, N>(std::forward<F>(f));
    }
}

// Sums with compile-time integer coefficients.  Terms with a zero
// coefficient are left out entirely (IEEE arithmetic forbids the compiler to
// drop 0 * x or x + 0 by itself), +-1 become adds and subtracts.
template <class R, bool Started> struct CSum {
    R v;
};

template <int c, class R, bool S>
__device__ __forceinline__ auto cadd(CSum<R, S> a, R x) {
    if constexpr (c == 0) {
        return a;
    } else if constexpr (!S) {
        if constexpr (c == 1) return CSum<R, true>{x};
        else if constexpr (c == -1) return CSum<R, true>{-x};
        else return CSum<R, true>{R(c) * x};
    } else {
        if constexpr (c == 1) return CSum<R, true>{a.v + x};
        else if constexpr (c == -1) return CSum<R, true>{a.v - x};
        else return CSum<R, true>{a.v + R(c) * x};
    }
}

template <class R, bool S> __device__ __forceinline__ R cval(CSum<R, S> a) {
    if constexpr (S) return a.v;
    else return R(0);
}

// a x + b y + c z
template <int a, int b, int c, class R>
__device__ __forceinline__ R cdot(R x, R y, R z) {
    return cval(cadd<c>(cadd<b>(cadd<a>(CSum<R, false>{R(0)}, x), y), z));
}

// a x + b y + c z + d p + e q + g r
template <int a, int b, int c, int d, int e, int g, class R>
__device__ __forceinline__ R cdot6(R x, R y, R z, R p, R q, R r) {
    return cval(cadd<g>(cadd<e>(cadd<d>(cadd<c>(cadd<b>(cadd<a>(CSum<R, false>{R(0)}, x), y), z), p), q), r));
}

// ---------------------------------------------------------------------------
// Random bits for stochastic rounding.  Per cell and launch one hash of
// (cell index, launch counter) with the PCG-based hash of Jarzynski & Olano,
// "Hash Functions for GPU Rendering" (JCGT 9(3), 2020).  Population pair p
// takes that word times a distinct odd constant (a bijection of 32-bit words,
// so every pair's word is exactly as uniform as the hash; one multiply).
__device__ __forceinline__ uint32_t pcg_hash(uint32_t v) {
    const uint32_t state = v * 747796405u + 2891336453u;
    const uint32_t word = ((state >> ((state >> 28u) + 4u)) ^ state) * 277803737u;
    return (word >> 22u) ^ word;
}
template <int p>
__device__ __forceinline__ uint32_t pair_bits(uint32_t h) {
    constexpr uint32_t k = 0x9e3779b9u * uint32_t(2 * p + 1);   // odd
    return h * k;
}
// Hardware stochastic rounding of two FP32 values to a packed 16-bit pair
// (PTX cvt.rs, sm_100a and later): the high half holds `hi`, the low half
// `lo`; rbits supplies the random bits.
__device__ __forceinline__ uint32_t cvt_rs_f16x2(float hi, float lo, uint32_t rbits) {
    uint32_t d;
    asm("cvt.rs.f16x2.f32 %0, %1, %2, %3;" : "=r"(d) : "f"(hi), "f"(lo), "r"(rbits));
    return d;
}
__device__ __forceinline__ uint32_t cvt_rs_bf16x2(float hi, float lo, uint32_t rbits) {
    uint32_t d;
    asm("cvt.rs.bf16x2.f32 %0, %1, %2, %3;" : "=r"(d) : "f"(hi), "f"(lo), "r"(rbits));
    return d;
}
__device__ __forceinline__ void st_u16(void* p, uint32_t v) { *reinterpret_cast<uint16_t*>(p) = (uint16_t)v; }

// ---------------------------------------------------------------------------
// Two cells in one register pair.  F2 holds one FP32 quantity of two cells;
// its +, -, * issue the packed f32x2 forms (PTX add/sub/mul/fma .f32x2,
// sm_100a and later): one instruction for both cells.  A product stays
// unevaluated (F2P) until it is used, so a following add or subtract becomes
// one fused multiply-add, the contraction nvcc applies to scalar code.
struct F2 {
    unsigned long long v;
    F2() = default;
    __device__ __forceinline__ F2(float a) { asm("mov.b64 %0, {%1, %1};" : "=l"(v) : "f"(a)); }
    __device__ __forceinline__ F2(double a) : F2((float)a) {}
    __device__ __forceinline__ F2(int a) : F2((float)a) {}
    __device__ __forceinline__ F2(float a, float b) { asm("mov.b64 %0, {%1, %2};" : "=l"(v) : "f"(a), "f"(b)); }
    __device__ __forceinline__ float lo() const { return __uint_as_float((unsigned)v); }
    __device__ __forceinline__ float hi() const { return __uint_as_float((unsigned)(v >> 32)); }
};
__device__ __forceinline__ F2 f2_bits(unsigned long long b) {
    F2 r;
    r.v = b;
    return r;
}
__device__ __forceinline__ F2 f2_add(F2 a, F2 b) {
    unsigned long long d;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a.v), "l"(b.v));
    return f2_bits(d);
}
__device__ __forceinline__ F2 f2_sub(F2 a, F2 b) {
    unsigned long long d;
    asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a.v), "l"(b.v));
    return f2_bits(d);
}
__device__ __forceinline__ F2 f2_mul(F2 a, F2 b) {
    unsigned long long d;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a.v), "l"(b.v));
    return f2_bits(d);
}
__device__ __forceinline__ F2 f2_fma(F2 a, F2 b, F2 c) {
    unsigned long long d;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a.v), "l"(b.v), "l"(c.v));
    return f2_bits(d);
}
__device__ __forceinline__ F2 operator-(F2 a) { return f2_bits(a.v ^ 0x8000000080000000ull); }
struct F2P {   // a * b, not yet rounded
    F2 a, b;
    __device__ __forceinline__ operator F2() const { return f2_mul(a, b); }
};
__device__ __forceinline__ F2 operator+(F2 a, F2 b) { return f2_add(a, b); }
__device__ __forceinline__ F2 operator-(F2 a, F2 b) { return f2_sub(a, b); }
__device__ __forceinline__ F2P operator*(F2 a, F2 b) { return F2P{a, b}; }
__device__ __forceinline__ F2P operator*(F2P p, F2 b) { return F2P{F2(p), b}; }
__device__ __forceinline__ F2P operator*(F2 a, F2P p) { return F2P{a, F2(p)}; }
__device__ __forceinline__ F2P operator*(F2P p, F2P q) { return F2P{F2(p), F2(q)}; }
__device__ __forceinline__ F2 operator+(F2P p, F2 c) { return f2_fma(p.a, p.b, c); }
__device__ __forceinline__ F2 operator+(F2 c, F2P p) { return f2_fma(p.a, p.b, c); }
__device__ __forceinline__ F2 operator-(F2 c, F2P p) { return f2_fma(-p.a, p.b, c); }
__device__ __forceinline__ F2 operator-(F2P p, F2 c) { return f2_fma(p.a, p.b, -c); }
__device__ __forceinline__ F2 operator+(F2P p, F2P q) { return f2_fma(p.a, p.b, F2(q)); }
__device__ __forceinline__ F2 operator-(F2P p, F2P q) { return f2_fma(p.a, p.b, -F2(q)); }
__device__ __forceinline__ F2P operator-(F2P p) { return F2P{-p.a, p.b}; }
__device__ __forceinline__ F2& operator+=(F2& a, F2 b) { return a = a + b; }
__device__ __forceinline__ F2& operator-=(F2& a, F2 b) { return a = a - b; }
__device__ __forceinline__ F2& operator+=(F2& a, F2P p) { return a = a + p; }

// The scalar type of an arithmetic type, and lane access: the parts of the
// collision with no packed form (sqrt, divisions, expm1, branches) run per
// cell on the lanes.
template <class R> struct Lanes {
    using Sc = R;
    static constexpr int n = 1;
    __device__ __forceinline__ static R get(R x, int) { return x; }
    __device__ __forceinline__ static R make(const R (&v)[1]) { return v[0]; }
};
template <> struct Lanes<F2> {
    using Sc = float;
    static constexpr int n = 2;
    __device__ __forceinline__ static float get(F2 x, int k) { return k ? x.hi() : x.lo(); }
    __device__ __forceinline__ static F2 make(const float (&v)[2]) { return F2(v[0], v[1]); }
};
__device__ __forceinline__ float recip(float x) { return 1.0f / x; }
__device__ __forceinline__ double recip(double x) { return 1.0 / x; }
__device__ __forceinline__ F2 recip(F2 x) { return F2(1.0f / x.lo(), 1.0f / x.hi()); }

// Arithmetic with every rounding spelled out (mad: one, fused).  The compiler
// may neither fuse these nor take a fused one apart, so a collision written in
// them gives the same bits in every kernel it is compiled into.
__device__ __forceinline__ double add(double a, double b) { return __dadd_rn(a, b); }
__device__ __forceinline__ double sub(double a, double b) { return __dsub_rn(a, b); }
__device__ __forceinline__ double mul(double a, double b) { return __dmul_rn(a, b); }
__device__ __forceinline__ double mad(double a, double b, double c) { return __fma_rn(a, b, c); }

// a > b for numbers >= 0, whose bits order as integers: an FP64 compare would
// take its turn on the FP64 pipe like an add
__device__ __forceinline__ bool above(double a, double b) {
    return __double_as_longlong(a) > __double_as_longlong(b);
}
// x in [2^-960, 2^960), by its high word: neither x nor its reciprocal or root is
// near what the starts below flush to zero
__device__ __forceinline__ bool moderate(double x) {
    return (uint32_t)__double2hiint(x) - 0x03f00000u < 0x78000000u;
}
// Reciprocal and (reciprocal) square root of the pair-form collision: the
// hardware's approximation refined by the residual of its defining equation.
// With e = 1 - x r, 1 / x = r (1 + e + e^2 + ...); with e = 1 - x r^2, 1 / sqrt(x)
// = r (1 + e/2 + 3/8 e^2 + ...) (binomial series).  The starts read and give 20
// mantissa bits, so e stays near 2^-19 and two terms do, 3 and 5 operations on the
// FP64 pipe where the division and the root take 9 to 10.  Largest errors measured:
// 0.50 ulp of 1 / x, 0.92 of 1 / sqrt(x) (the root and the division: up to 1), 1.61
// of the root.  x has to be moderate; callers divide and root other numbers, zeros,
// infinities and NaN among them.
__device__ __forceinline__ double rcp(double x) {
    double r;
    asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(r) : "d"(x));
    const double e = mad(-x, r, 1.0);
    return mad(r, mad(e, e, e), r);
}
__device__ __forceinline__ double rcp_root(double x) {
    double r;
    asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(r) : "d"(x));
    const double e = mad(-mul(x, r), r, 1.0);
    return mad(mul(r, e), mad(0.375, e, 0.5), r);
}
__device__ __forceinline__ double root(double x) { return moderate(x) ? mul(x, rcp_root(x)) : sqrt(x); }

// ---------------------------------------------------------------------------
// storage.  R is the arithmetic type.  ld / st move population i between
// memory and registers; enc / dec convert full FP64 populations at the ABI
// (set/get populations).
//
// The 16-bit forms store the offset normalised by its lattice weight,
// (f_i - w_i) / w_i, which is O(Ma) in every direction; FP16 also scales it
// by 2^14 (exact) so offsets down to ~4e-9 stay out of FP16's subnormal range
// while |(f_i - w_i)/w_i| up to 4 stays below its largest finite value.
template <class S> struct Store;
//
// The collision works on populations in MEMORY UNITS x_i = alpha_i (f_i - w_i),
// so loads and stores need no scaling.  Three per-direction constants carry
// the units: beta_i = 1 / alpha_i turns x_i into an offset (moments),
// gam_i = alpha_i w_i scales the equilibrium-type terms (which all carry a
// factor w_i) and god_i = alpha_i 3 w_i their odd part.  For the 16-bit forms
// alpha_i is proportional to 1 / w_i, so gam_i and god_i are the same for
// every direction and the weights drop out of the collision arithmetic.
template <> struct Store<float> {
    using R = float;
    template <class L, int i> __host__ __device__ static constexpr R beta() { return 1.0f; }
    template <class L, int i> __host__ __device__ static constexpr R gam() { return R(L::w(i)); }
    template <class L, int i> __host__ __device__ static constexpr R god() { return L::w3f(i); }
    template <class L, int i> static __device__ __forceinline__ R ld(const float* p) { return *p; }
    static constexpr bool kStochastic = false;
    template <class L, int i> static __device__ __forceinline__ void st(float* p, R v, uint32_t) { *p = v; }
    template <class L, int i>
    static __device__ __forceinline__ void st2(float* pi, float* po, R vi, R vo, uint32_t) { *pi = vi; *po = vo; }
    static __device__ __forceinline__ float enc(double off, double) { return (float)off; }
    static __device__ __forceinline__ double dec(float v, double) { return (double)v; }
};
template <> struct Store<double> {
    using R = double;
    template <class L, int i> __host__ __device__ static constexpr R beta() { return 1.0; }
    template <class L, int i> __host__ __device__ static constexpr R gam() { return L::w(i); }
    template <class L, int i> __host__ __device__ static constexpr R god() { return 3.0 * L::w(i); }
    template <class L, int i> static __device__ __forceinline__ R ld(const double* p) { return *p; }
    static constexpr bool kStochastic = false;
    template <class L, int i> static __device__ __forceinline__ void st(double* p, R v, uint32_t) { *p = v; }
    template <class L, int i>
    static __device__ __forceinline__ void st2(double* pi, double* po, R vi, R vo, uint32_t) { *pi = vi; *po = vo; }
    static __device__ __forceinline__ double enc(double off, double) { return off; }
    static __device__ __forceinline__ double dec(double v, double) { return v; }
};
template <> struct Store<__half> {
    using R = float;
    static constexpr double kScale = 16384.0;   // 2^14: alpha_i = 2^14 / w_i
    template <class L, int i> __host__ __device__ static constexpr R beta() { return float(L::w(i) / kScale); }
    template <class L, int i> __host__ __device__ static constexpr R gam() { return float(kScale); }
    template <class L, int i> __host__ __device__ static constexpr R god() { return float(3.0 * kScale); }
    template <class L, int i> static __device__ __forceinline__ R ld(const __half* p) {
        return __half2float(*p);
    }
    static constexpr bool kStochastic = true;
    // stochastic rounding (unbiased: a value moves by less than half an ulp per
    // step in slowly relaxing flows, and round-to-nearest would freeze it)
    template <class L, int i> static __device__ __forceinline__ void st(__half* p, R v, uint32_t rnd) {
        st_u16(p, cvt_rs_f16x2(v, 0.0f, rnd) >> 16);
    }
    // populations i and its opposite (same weight) in one conversion
    template <class L, int i>
    // pi and po = pi + 1 are the two halves of one 4-byte-aligned word (the
    // interleaved pair layout): f_i in the low half, f_o in the high half
    static __device__ __forceinline__ void st2(__half* pi, __half*, R vi, R vo, uint32_t rnd) {
        *reinterpret_cast<uint32_t*>(pi) = cvt_rs_f16x2(vo, vi, rnd);
    }
    static __device__ __forceinline__ __half enc(double off, double w) { return __double2half(off / w * kScale); }
    static __device__ __forceinline__ double dec(__half v, double w) { return (double)__half2float(v) * (w / kScale); }
};
template <> struct Store<__nv_bfloat16> {
    using R = float;   // alpha_i = 1 / w_i
    template <class L, int i> __host__ __device__ static constexpr R beta() { return float(L::w(i)); }
    template <class L, int i> __host__ __device__ static constexpr R gam() { return 1.0f; }
    template <class L, int i> __host__ __device__ static constexpr R god() { return 3.0f; }
    template <class L, int i> static __device__ __forceinline__ R ld(const __nv_bfloat16* p) {
        return __bfloat162float(*p);
    }
    static constexpr bool kStochastic = true;
    template <class L, int i> static __device__ __forceinline__ void st(__nv_bfloat16* p, R v, uint32_t rnd) {
        st_u16(p, cvt_rs_bf16x2(v, 0.0f, rnd) >> 16);
    }
    template <class L, int i>
    static __device__ __forceinline__ void st2(__nv_bfloat16* pi, __nv_bfloat16*, R vi, R vo,
                                               uint32_t rnd) {
        *reinterpret_cast<uint32_t*>(pi) = cvt_rs_bf16x2(vo, vi, rnd);
    }
    static __device__ __forceinline__ __nv_bfloat16 enc(double off, double w) { return __double2bfloat16(off / w); }
    static __device__ __forceinline__ double dec(__nv_bfloat16 v, double w) { return (double)__bfloat162float(v) * w; }
};

// Rheology constants in the arithmetic type, derived on the host in FP64.
template <class R> struct Coef {
    R nu_p, sigma_y, m, gdot_c, inv_gc, e_c, magic;
    R g[3];
    R s2y;     // sqrt(2) sigma_y
    R ir_a;    // 1 / (1/2 + 3 nu_p)
    R ir_b;    // 1 / (1 + 6 nu_p)
    R six_nu;  // 6 nu_p
    R s2y2;    // 2 sigma_y^2, the square of the IR yield threshold
    R ir_bn;   // six_nu ir_b
    R ir_bs;   // s2y ir_b
    R ir_k;    // ir_bn - ir_a / 2 - 1
    R ir_ks;   // s2y (ir_a / 2 + ir_b)
    R hg[3];   // g / 2
    int newton;  // PR: Newton iterations of the implicit tau update
    R cg[13];   // c_i . g of direction i = 2p + 1 (PR force terms of the class form), per pair p
    R cgg[13];  // (c_i . g)^2
};

struct KArgs {
    KParams kp;
    Coef<float> cf;
    Coef<double> cd;
};

template <class R> __device__ __forceinline__ const Coef<R>& coef(const KArgs& a);
template <> __device__ __forceinline__ const Coef<float>& coef<float>(const KArgs& a) { return a.cf; }
template <> __device__ __forceinline__ const Coef<double>& coef<double>(const KArgs& a) { return a.cd; }

// Base pointer of every population plane, passed by value in the kernel
// parameters: an address is then one multiply-add of the 32-bit cell index.
// Population layout.  FP32 / FP64: plane i holds population i of every cell.
// 16-bit forms: the rest population has plane 0; an opposite pair (i, i + 1),
// i odd, shares planes i and i + 1 as one plane of 32-bit words holding f_i
// in the low and f_{i+1} in the high half of cell n's word, so the pair's
// packed stochastic-rounding result is one aligned 32-bit store.  Element
// (i, n) is at pop_base(i) + pop_step(i) n; the total is Q planes either way.
template <class S> __host__ __device__ constexpr bool pairs_interleaved() { return sizeof(S) == 2; }
template <class S> __host__ __device__ constexpr int64_t pop_base(int i, int64_t plane) {
    return (!pairs_interleaved<S>() || i == 0) ? i * plane : (i - ((i - 1) & 1)) * plane + ((i - 1) & 1);
}
template <class S> __host__ __device__ constexpr int pop_step(int i) {
    return (pairs_interleaved<S>() && i > 0) ? 2 : 1;
}

template <class S> struct SrcPlanes {
    const S* p[27];   // p[i] = buffer + pop_base(i)
    template <int i> __device__ __forceinline__ const S* at(int n) const {
        return p[i] + (int64_t)pop_step<S>(i) * n;
    }
};
template <class S> struct DstPlanes {
    S* p[27];
    template <int i> __device__ __forceinline__ S* at(int n) const {
        return p[i] + (int64_t)pop_step<S>(i) * n;
    }
};
// Planes of one buffer addressed by a stride (batched launches, where the
// pointers differ per domain), in 32-bit arithmetic (the batch admits only
// domains with Q * plane < 2^31, and every element index is below that).
template <class S> struct SrcStride {
    const S* base;
    int plane;
    template <int i> __device__ __forceinline__ const S* at(int n) const {
        return base + ((int)pop_base<S>(i, plane) + pop_step<S>(i) * n);
    }
};
template <class S> struct DstStride {
    S* base;
    int plane;
    template <int i> __device__ __forceinline__ S* at(int n) const {
        return base + ((int)pop_base<S>(i, plane) + pop_step<S>(i) * n);
    }
};

// cell index -> (x, y, z)
__device__ __forceinline__ void cell_xyz(const KParams& kp, int idx, int& x, int& y, int& z) {
    const uint32_t t = kp.div_nx.div((uint32_t)idx);
    x = idx - (int)t * kp.nx;
    z = (int)kp.div_ny.div(t);
    y = (int)t - z * kp.ny;
}

// ---------------------------------------------------------------------------
// streaming (pull) with halfway bounce-back
// 1: the gather path is chosen per warp (see gather); 0 restores the
// per-thread choice, for comparison builds.
#ifndef BLBM_WARP_UNIFORM_GATHER
#define BLBM_WARP_UNIFORM_GATHER 1
#endif
// Offsets from a cell's index to its pull sources x - c (periodic wrap):
// m for a velocity component +1, p for -1.
struct PullOffsets {
    int dxm, dxp, dym, dyp, dzm, dzp;
    template <class L, int i> __device__ __forceinline__ int of() const {
        constexpr int cx = L::cx(i), cy = L::cy(i), cz = L::cz(i);
        int off = 0;
        if constexpr (cx > 0) off += dxm;
        if constexpr (cx < 0) off += dxp;
        if constexpr (cy > 0) off += dym;
        if constexpr (cy < 0) off += dyp;
        if constexpr (cz > 0) off += dzm;
        if constexpr (cz < 0) off += dzp;
        return off;
    }
};

__device__ __forceinline__ PullOffsets pull_offsets(const KParams& kp, int idx) {
    const int nx = kp.nx, ny = kp.ny, nz = kp.nz;
    int x, y, z;
    cell_xyz(kp, idx, x, y, z);
    const int sy = nx, sz = nx * ny;
    PullOffsets o;
    o.dxm = (x == 0) ? nx - 1 : -1;
    o.dxp = (x == nx - 1) ? -(nx - 1) : 1;
    o.dym = (y == 0) ? (ny - 1) * sy : -sy;
    o.dyp = (y == ny - 1) ? -(ny - 1) * sy : sy;
    o.dzm = (z == 0) ? (nz - 1) * sz : -sz;
    o.dzp = (z == nz - 1) ? -(nz - 1) * sz : sz;
    return o;
}

// self = true loads the cell's own populations, plane by plane (all offsets
// 0; lk must be 0): the copy-through of a solid cell.
template <class L, class S, class Src>
__device__ __forceinline__ void gather(const KParams& kp, const Src& P, uint32_t lk,
                                       int idx, typename Store<S>::R (&v)[L::Q],
                                       bool self = false) {
    PullOffsets o = pull_offsets(kp, idx);
    if (self) o = PullOffsets{0, 0, 0, 0, 0, 0};
    auto offset = [&](auto I) { return o.template of<L, decltype(I)::value>(); };
    // The path is chosen per warp: a warp takes the plain pull only when none
    // of its cells has a solid neighbour.  A per-thread choice makes a warp
    // that mixes wall and interior cells run both paths one after the other,
    // which is most warps in a porous medium; the select path is exact for
    // interior cells too (their link bits are 0).
#if BLBM_WARP_UNIFORM_GATHER
    const bool plain = __all_sync(__activemask(), lk == 0u);
#else
    const bool plain = lk == 0u;
#endif
    if (plain) {
        // no solid neighbour: plain pull, no per-population selects
        static_for<0, L::Q>([&](auto I) {
            constexpr int i = decltype(I)::value;
            v[i] = Store<S>::template ld<L, i>(P.template at<i>(idx + offset(I)));
        });
    } else {
        static_for<0, L::Q>([&](auto I) {
            constexpr int i = decltype(I)::value;
            const S* p = ((lk >> i) & 1u) ? P.template at<L::opp(i)>(idx)
                                          : P.template at<i>(idx + offset(I));
            v[i] = Store<S>::template ld<L, i>(p);   // opposite planes share w_i
        });
    }
}

// ---------------------------------------------------------------------------
// moments of the offsets: d = sum df, j = sum c df, p = sum c c df
template <class R> struct Mom {
    R d, jx, jy, jz, xx, yy, zz, xy, xz, yz;
};
// symmetric second-order tensor
template <class R> struct Tens {
    R xx, yy, zz, xy, xz, yz;
};

// Which form of the collision a storage runs.  Pair form (below): FP64, whose
// step is bound by the FP64 pipe (D3Q27 IR, duct 1 x 64 x 64: 24.5 -> 19.0 us a
// step; D2Q9 PR, 80 x 80: 15.6 -> 13.5).  FP32 arithmetic keeps the class sums.  The
// pair form gained FP32 storage 0.4-3 % (its large steps are bound by HBM) and
// the 16-bit forms 5-20 %, but it rounds in another order: near a steady state the
// FP32 residual shows that, and 16-bit storage picks the other neighbour here and
// there, so that a domain would depend on which form its size, or a batch, runs.
template <class S> __host__ __device__ constexpr bool pair_form() { return sizeof(S) == 8; }

// Grouped sums: populations are added once per velocity class (c_x = +1, -1,
// 0; c_y = +-1; c_z = +-1; sign of c_x c_y, c_x c_z, c_y c_z) and the moments
// are sums and differences of those class sums.  Each class sum starts as its
// first member (no add to a zero).  f is in memory units; beta_i turns each
// value into an offset.  Where beta_i != 1 it is applied inside each class
// sum's multiply-add (one instruction per class membership, no separate
// multiply per population).
enum { kXp, kXm, kX0, kYp, kYm, kZp, kZm, kPxy, kMxy, kPxz, kMxz, kPyz, kMyz, kNumClasses };

__host__ __device__ constexpr bool in_class(int k, int cx, int cy, int cz) {
    return k == kXp ? cx == 1 : k == kXm ? cx == -1 : k == kX0 ? cx == 0
         : k == kYp ? cy == 1 : k == kYm ? cy == -1 : k == kZp ? cz == 1 : k == kZm ? cz == -1
         : k == kPxy ? cx * cy == 1 : k == kMxy ? cx * cy == -1
         : k == kPxz ? cx * cz == 1 : k == kMxz ? cx * cz == -1
         : k == kPyz ? cy * cz == 1 : cy * cz == -1;
}
template <class L> __host__ __device__ constexpr int first_in_class(int k) {
    for (int i = 0; i < L::Q; ++i)
        if (in_class(k, L::cx(i), L::cy(i), L::cz(i))) return i;
    return -1;
}

template <class L, class S, class R>
__device__ __forceinline__ Mom<R> class_moments(const R (&f)[L::Q]) {
    R acc[kNumClasses];
    static_for<0, L::Q>([&](auto I) {
        constexpr int i = decltype(I)::value;
        constexpr int cx = L::cx(i), cy = L::cy(i), cz = L::cz(i);
        constexpr auto beta = Store<S>::template beta<L, i>();
        static_for<0, kNumClasses>([&](auto K) {
            constexpr int k = decltype(K)::value;
            if constexpr (in_class(k, cx, cy, cz)) {
                if constexpr (beta == 1) {
                    if constexpr (first_in_class<L>(k) == i) acc[k] = f[i];
                    else acc[k] += f[i];
                } else {
                    if constexpr (first_in_class<L>(k) == i) acc[k] = R(f[i] * R(beta));
                    else acc[k] = acc[k] + f[i] * R(beta);
                }
            }
        });
    });
    Mom<R> m;
    m.xx = acc[kXp] + acc[kXm];
    m.jx = acc[kXp] - acc[kXm];
    m.d = m.xx + acc[kX0];
    m.yy = acc[kYp] + acc[kYm];
    m.jy = acc[kYp] - acc[kYm];
    m.xy = acc[kPxy] - acc[kMxy];
    if constexpr (L::D == 3) {
        m.zz = acc[kZp] + acc[kZm];
        m.jz = acc[kZp] - acc[kZm];
        m.xz = acc[kPxz] - acc[kMxz];
        m.yz = acc[kPyz] - acc[kMyz];
    } else {
        m.zz = R(0);
        m.jz = R(0);
        m.xz = R(0);
        m.yz = R(0);
    }
    return m;
}

// Direction families.  In the pair order of lattice.cuh the axis pairs come
// first, then the face diagonals (xy+, xy-, xz+, xz-, yz+, yz-), then the
// corners (+++), (++-), (+-+), (-++); first() is the index i of a family's
// first member, 0 where the lattice has none.  All members of a family share
// their weight.
template <class L> struct Fam {
    static constexpr int axis = 1;
    static constexpr int face = L::Q == 9 ? 5 : L::Q == 15 ? 0 : 7;
    static constexpr int corner = L::Q == 15 ? 7 : L::Q == 27 ? 19 : 0;
};
template <class L> constexpr bool fam_order() {
    auto is = [](int i, int x, int y, int z) { return L::cx(i) == x && L::cy(i) == y && L::cz(i) == z; };
    bool ok = is(1, 1, 0, 0) && is(3, 0, 1, 0) && (L::D == 2 || is(5, 0, 0, 1));
    constexpr int f = Fam<L>::face, c = Fam<L>::corner;
    if (f) ok = ok && is(f, 1, 1, 0) && is(f + 2, 1, -1, 0);
    if (f && L::D == 3)
        ok = ok && is(f + 4, 1, 0, 1) && is(f + 6, 1, 0, -1) && is(f + 8, 0, 1, 1) && is(f + 10, 0, 1, -1);
    if (c) ok = ok && is(c, 1, 1, 1) && is(c + 2, 1, 1, -1) && is(c + 4, 1, -1, 1) && is(c + 6, -1, 1, 1);
    return ok;
}
static_assert(fam_order<D2Q9>() && fam_order<D3Q15>() && fam_order<D3Q19>() && fam_order<D3Q27>(),
              "direction families");

// Parts a cell's pair-form collision can be divided into, one warp each (see
// k_step_split), by families: the axis pairs with the rest population, and the
// diagonals.  pair_part() owns pair p.
template <class L> __host__ __device__ constexpr int parts() { return L::Q >= 19 ? 4 : 2; }
template <class L> __host__ __device__ constexpr int pair_part(int p) {
    if (p < L::D) return 0;
    if (L::Q == 9 || L::Q == 15) return 1;
    if (L::Q == 19) return 1 + (p - 3) / 2;                  // a part per face plane
    return p < 7 ? 1 : p < 9 ? 2 : 3;                        // xy and xz, yz, corners
}
// pair k of a part (-1: it has fewer), and the place of pair p in its part
template <class L> __host__ __device__ constexpr int part_pair(int part, int k) {
    for (int p = 0; p < (L::Q - 1) / 2; ++p)
        if (pair_part<L>(p) == part && k-- == 0) return p;
    return -1;
}
template <class L> __host__ __device__ constexpr int part_place(int p) {
    int k = 0;
    for (int q = 0; q < p; ++q) k += pair_part<L>(q) == pair_part<L>(p);
    return k;
}

// b x and y + b x for a compile-time factor b (a plain x, y + x where it is 1)
__device__ __forceinline__ double scale(double b, double x) { return b == 1.0 ? x : mul(x, b); }
__device__ __forceinline__ double axpy(double b, double x, double y) {
    return b == 1.0 ? add(y, x) : mad(x, b, y);
}

// Pair form: f[i] = f_i + f_o and f[o] = f_i - f_o for every opposite pair
// (i, o = i + 1).  Even moments need the sums only, odd ones the differences
// only, and so do the two halves of the TRT collision.
template <class L, class R> __device__ __forceinline__ void to_pairs(R (&f)[L::Q]) {
    static_for<0, (L::Q - 1) / 2>([&](auto P) {
        constexpr int i = 2 * decltype(P)::value + 1;
        const R a = f[i], b = f[i + 1];
        f[i] = add(a, b);
        f[i + 1] = sub(a, b);
    });
}

// Moments from the pair form.  Per family the members are first combined by
// sums and differences (xx + yy against xy of a face plane; the four corners
// by one 4-point butterfly), then added to the axis terms.  On D3Q27 this takes
// 82 adds where adding every population to its velocity classes took 96, and 26
// of them are the pair sums that the TRT collision needs anyway.
template <class L, class R> __device__ __forceinline__ Mom<R> pair_moments(const R (&f)[L::Q]) {
    constexpr int F = Fam<L>::face, C = Fam<L>::corner;
    Mom<R> m;
    if constexpr (L::D == 2) {
        const R XY = add(f[F], f[F + 2]);
        m.xx = add(XY, f[1]);
        m.yy = add(XY, f[3]);
        m.d = add(m.xx, add(f[3], f[0]));
        m.xy = sub(f[F], f[F + 2]);
        m.jx = add(add(f[F + 1], f[F + 3]), f[2]);
        m.jy = add(sub(f[F + 1], f[F + 3]), f[4]);
        m.zz = R(0);
        m.jz = R(0);
        m.xz = R(0);
        m.yz = R(0);
    } else {
        R X, Y, Z, rest = add(f[3], f[5]);   // X: diagonal sums beyond the axis pairs
        R jx, jy, jz;
        if constexpr (C != 0) {
            const R ab = add(f[C], f[C + 2]), amb = sub(f[C], f[C + 2]);
            const R ce = add(f[C + 4], f[C + 6]), cme = sub(f[C + 4], f[C + 6]);
            X = add(ab, ce);
            m.xy = sub(ab, ce);
            m.xz = add(amb, cme);
            m.yz = sub(amb, cme);
            const R dp = add(f[C + 1], f[C + 3]), dq = sub(f[C + 5], f[C + 7]);
            jx = add(dp, dq);
            jy = sub(dp, dq);
            jz = add(sub(f[C + 1], f[C + 3]), add(f[C + 5], f[C + 7]));
            Y = X;
            Z = X;
        }
        if constexpr (F != 0) {
            const R sxy = add(f[F], f[F + 2]), sxz = add(f[F + 4], f[F + 6]), syz = add(f[F + 8], f[F + 10]);
            const R oxy = sub(f[F], f[F + 2]), oxz = sub(f[F + 4], f[F + 6]), oyz = sub(f[F + 8], f[F + 10]);
            const R fx = add(add(f[F + 1], f[F + 3]), add(f[F + 5], f[F + 7]));
            const R fy = add(sub(f[F + 1], f[F + 3]), add(f[F + 9], f[F + 11]));
            const R fz = add(sub(f[F + 5], f[F + 7]), sub(f[F + 9], f[F + 11]));
            const R xs = add(sxy, sxz), ys = add(sxy, syz), zs = add(sxz, syz);
            rest = add(rest, syz);
            if constexpr (C != 0) {
                X = add(X, xs);
                Y = add(Y, ys);
                Z = add(Z, zs);
                m.xy = add(m.xy, oxy);
                m.xz = add(m.xz, oxz);
                m.yz = add(m.yz, oyz);
                jx = add(jx, fx);
                jy = add(jy, fy);
                jz = add(jz, fz);
            } else {
                X = xs;
                Y = ys;
                Z = zs;
                m.xy = oxy;
                m.xz = oxz;
                m.yz = oyz;
                jx = fx;
                jy = fy;
                jz = fz;
            }
        }
        m.xx = add(X, f[1]);
        m.yy = add(Y, f[3]);
        m.zz = add(Z, f[5]);
        m.d = add(m.xx, add(rest, f[0]));
        m.jx = add(jx, f[2]);
        m.jy = add(jy, f[4]);
        m.jz = add(jz, f[6]);
    }
    return m;
}

// moments of populations in memory units (f may be overwritten)
template <class L, class S, class R = typename Store<S>::R>
__device__ __forceinline__ Mom<R> moments(R (&f)[L::Q]) {
    if constexpr (pair_form<S>()) {
        to_pairs<L>(f);
        return pair_moments<L, R>(f);
    } else {
        return class_moments<L, S, R>(f);
    }
}

// Pi - c_s^2 rho I written with offsets: Pi = c_s^2 I + p, rho = 1 + d.
template <class L, class R> __device__ __forceinline__ Tens<R> dynamic(const Mom<R>& m) {
    const R third = R(-1.0 / 3.0);
    Tens<R> t;
    t.xx = mad(m.d, third, m.xx);
    t.yy = mad(m.d, third, m.yy);
    t.xy = m.xy;
    t.zz = R(0);
    t.xz = R(0);
    t.yz = R(0);
    if constexpr (L::D == 3) {
        t.zz = mad(m.d, third, m.zz);
        t.xz = m.xz;
        t.yz = m.yz;
    }
    return t;
}

// Non-equilibrium second moment T = Pi - rho c_s^2 I - rho u u, from the first
// two terms P, p = -rho u and u.
template <class L, class R>
__device__ __forceinline__ Tens<R> noneq(const Tens<R>& P, R px, R py, R pz, R ux, R uy, R uz,
                                         uint32_t flags) {
    Tens<R> t;
    t.xx = mad(px, ux, P.xx);
    t.yy = mad(py, uy, P.yy);
    t.xy = mad(px, uy, P.xy);
    if constexpr (L::D == 3) {
        t.zz = mad(pz, uz, P.zz);
        t.xz = mad(px, uz, P.xz);
        t.yz = mad(py, uz, P.yz);
    } else {
        t.zz = R(0);
        t.xz = R(0);
        t.yz = R(0);
    }
    if (flags & LBM_FLAG_BURNETT_X) t.xx = R(0);
    return t;
}

// T:T
template <class L, class R> __device__ __forceinline__ R square(const Tens<R>& T) {
    R off = mul(T.xy, T.xy), diag = mad(T.yy, T.yy, mul(T.xx, T.xx));
    if constexpr (L::D == 3) {
        off = mad(T.yz, T.yz, mad(T.xz, T.xz, off));
        diag = mad(T.zz, T.zz, diag);
    }
    return mad(R(2), off, diag);
}

template <class L, class R> __device__ __forceinline__ R trace(const Tens<R>& t) {
    if constexpr (L::D == 3) return add(add(t.xx, t.yy), t.zz);
    return add(t.xx, t.yy);
}

// The post-collision populations of both models have the form
//   f_i = [kept part] + w_i (e0 + 9/2 c.N.c) + 3 w_i c.q
// (memory units).  The even bracket takes six numbers per cell, and the
// members of a family differ only by the signs of the off-diagonal terms: one
// sum per axis pair, two per face plane, one 4-point butterfly for the
// corners, instead of c.u, its square and c.T.c per pair (D3Q27: 23 adds
// against 150 operations).  put(i, e, cq, wo) stores pair i, its even part e
// (weighted) and its odd part wo cq.
// PART >= 0: only the pairs of that part (the compiler drops the rest).
template <class L, class S, class R, int PART = -1, class Put>
__device__ __forceinline__ void pair_terms(R e0, const Tens<R>& N, R qx, R qy, R qz, Put&& put) {
    constexpr int F = Fam<L>::face, C = Fam<L>::corner;
#define BLBM_I(n) std::integral_constant<int, (n)>{}
    // Even parts carry their weights: per family gam enters e0's sums once (the
    // axis family through its constants) and the off-diagonal terms' constant.
    constexpr R gA = Store<S>::template gam<L, 1>();
    constexpr R gF = Store<S>::template gam<L, (F ? F : 1)>();
    constexpr R gC = Store<S>::template gam<L, (C ? C : 1)>();
    constexpr R k = 4.5, kA = 4.5 * gA, kF = 9.0 * gF, kC = 9.0 * gC;
    auto pair = [&](auto I, R e, R cq) {
        constexpr int i = decltype(I)::value;
        if constexpr (PART >= 0 && pair_part<L>((i - 1) / 2) != PART) return;
        else put(I, e, cq, Store<S>::template god<L, i>());
    };
    const R eA = scale(gA, e0);
    pair(BLBM_I(1), mad(kA, N.xx, eA), qx);
    pair(BLBM_I(3), mad(kA, N.yy, eA), qy);
    const R ex = mad(k, N.xx, e0);
    const R exy = mad(k, N.yy, ex);
    const R qxpy = add(qx, qy), qxmy = sub(qx, qy);
    if constexpr (L::D == 2) {
        const R s = scale(gF, exy), b = mul(kF, N.xy);
        pair(BLBM_I(F), add(s, b), qxpy);
        pair(BLBM_I(F + 2), sub(s, b), qxmy);
    } else {
        pair(BLBM_I(5), mad(kA, N.zz, eA), qz);
        const R ez = mad(k, N.zz, e0);
        if constexpr (F != 0) {
            const R sxy = scale(gF, exy), bxy = mul(kF, N.xy);
            pair(BLBM_I(F), add(sxy, bxy), qxpy);
            pair(BLBM_I(F + 2), sub(sxy, bxy), qxmy);
            const R sxz = scale(gF, mad(k, N.zz, ex)), bxz = mul(kF, N.xz);
            pair(BLBM_I(F + 4), add(sxz, bxz), add(qx, qz));
            pair(BLBM_I(F + 6), sub(sxz, bxz), sub(qx, qz));
            const R syz = scale(gF, mad(k, N.yy, ez)), byz = mul(kF, N.yz);
            pair(BLBM_I(F + 8), add(syz, byz), add(qy, qz));
            pair(BLBM_I(F + 10), sub(syz, byz), sub(qy, qz));
        }
        if constexpr (C != 0) {
            const R e = scale(gC, mad(k, N.zz, exy));
            const R bxy = mul(kC, N.xy), bxz = mul(kC, N.xz), byz = mul(kC, N.yz);
            const R ep = add(e, byz), em = sub(e, byz), bp = add(bxy, bxz), bm = sub(bxy, bxz);
            pair(BLBM_I(C), add(ep, bp), add(qxpy, qz));
            pair(BLBM_I(C + 2), add(em, bm), sub(qxpy, qz));
            pair(BLBM_I(C + 4), sub(em, bm), add(qxmy, qz));
            pair(BLBM_I(C + 6), sub(ep, bp), sub(qz, qxmy));
        }
    }
#undef BLBM_I
}

// ---------------------------------------------------------------------------
// IR yield solve, per cell: with s = as T, sigma = asg T (eq. Vikh_sigmaS_tensor)
// from |T|^2, returns k1 = as / 2 - asg - 1 and asg.  Both factors are linear in
// 1 / |T| (-(|T| - sqrt2 sigma_y) a / |T| = sqrt2 sigma_y a / |T| - a), and so is
// k1: one reciprocal square root and two multiply-adds.
__device__ __forceinline__ void ir_yield(const Coef<double>& c, double t2, double& k1, double& asg) {
    k1 = 0.0;
    asg = -1.0;
    double it;
    if (moderate(t2)) {
        if (above(c.s2y2, t2)) return;
        it = rcp_root(t2);
    } else {
        const double tn = sqrt(t2);
        if (!(tn > 0.0 && tn >= c.s2y)) return;
        it = 1.0 / tn;
    }
    k1 = mad(c.ir_ks, it, c.ir_k);
    asg = mad(-c.ir_bs, it, -c.ir_bn);
}

// ---------------------------------------------------------------------------
// IR collision (Secs. 2.3, 3.2).  f: memory units in, memory units out.
// What the pairs need from the moments: e0, N and q of pair_terms.
template <class L, class R>
__device__ __forceinline__ void ir_terms(const Coef<typename Lanes<R>::Sc>& c, uint32_t flags,
                                         const Mom<R>& m, R& e0, Tens<R>& N, R (&q)[3], R (&ur)[3]) {
    const R rho = add(R(1), m.d);
    const R inv = moderate(rho) ? rcp(rho) : 1.0 / rho;
    const R gx = R(c.g[0]), gy = R(c.g[1]);
    R gz = R(0);
    if constexpr (L::D == 3) gz = R(c.g[2]);
    const R px = mad(rho, R(c.hg[0]), m.jx), py = mad(rho, R(c.hg[1]), m.jy);   // rho u
    R pz = R(0);
    if constexpr (L::D == 3) pz = mad(rho, R(c.hg[2]), m.jz);
    const R ux = mul(px, inv), uy = mul(py, inv);
    R uz = R(0);
    if constexpr (L::D == 3) uz = mul(pz, inv);
    const Tens<R> P = dynamic<L, R>(m);
    const Tens<R> T = noneq<L, R>(P, -px, -py, -pz, ux, uy, uz, flags);
    R k1, asg;   // k1 - 1 with the k1 below
    ir_yield(c, square<L, R>(T), k1, asg);
    // A = -sigma_bar + s/2 = k1 T + k2 I with sigma_bar = sigma - tr(sigma)/D I;
    // N = rho u u + A gives f_eq + f^sigma = w_i (d - 3/2 tr N + 9/2 c.N.c + 3 rho c.u) + w_i,
    // and rho u u = P - T
    const R k2 = mul(asg, mul(trace<L, R>(T), R(1.0 / L::D)));
    N.xx = mad(k1, T.xx, add(P.xx, k2));
    N.yy = mad(k1, T.yy, add(P.yy, k2));
    N.xy = mad(k1, T.xy, P.xy);
    N.zz = R(0);
    N.xz = R(0);
    N.yz = R(0);
    if constexpr (L::D == 3) {
        N.zz = mad(k1, T.zz, add(P.zz, k2));
        N.xz = mad(k1, T.xz, P.xz);
        N.yz = mad(k1, T.yz, P.yz);
    }
    if (flags & LBM_FLAG_BURNETT_X) N.xx = add(mul(px, ux), k2);   // T.xx was dropped
    e0 = mad(R(-1.5), trace<L, R>(N), m.d);
    // odd part: w_i (3 rho c.u + 3/2 c.F) = 3 w_i c.(j + F), since rho u = j + F/2
    q[0] = mad(rho, gx, m.jx);
    q[1] = mad(rho, gy, m.jy);
    q[2] = R(0);
    if constexpr (L::D == 3) q[2] = mad(rho, gz, m.jz);
    ur[0] = ux;
    ur[1] = uy;
    ur[2] = uz;
}

template <class L, class S, class R>
__device__ __forceinline__ void pair_collide_ir(const Coef<typename Lanes<R>::Sc>& c, uint32_t flags,
                                                R (&f)[L::Q], R& drho, R (&ur)[3]) {
    const Mom<R> m = moments<L, S, R>(f);
    R e0, q[3];
    Tens<R> N;
    ir_terms<L, R>(c, flags, m, e0, N, q, ur);
    f[0] = scale(Store<S>::template gam<L, 0>(), e0);
    pair_terms<L, S, R>(e0, N, q[0], q[1], q[2], [&](auto I, R e, R cq, auto wo) {
        constexpr int i = decltype(I)::value;
        f[i] = axpy(wo, cq, e);
        f[i + 1] = axpy(-wo, cq, e);
    });
    drho = m.d;
}

// ---------------------------------------------------------------------------
// Implicit PR update (Sec. 3, Newton iterations).  With the unknown tau the
// strain rate of eq. (LBM_strain_rate) is gdot = a / tau, a = 1.5 sqrt(2 T:T);
// tau = 1/2 + 3 nu_app(gdot).  Consistency is the root of
// H(gdot) = gdot tau(gdot) - a = gdot / 2 + 3 gdot nu_app(gdot) - a, whose
// derivative is 1/2 + 3 d(gdot nu_app)/d gdot: nu_p + (sigma_y / rho) m e^(-m gdot)
// above the cut-off, nu_0 + 2 gdot (nu_c - nu_0) / gdot_C on the linear part
// below it.  Iterates are clamped at 0, H' floored at 1/2.
template <class R>
__device__ __forceinline__ R pr_newton(const Coef<R>& c, R a, R gd, R sy_rho) {
    const R nu0 = c.nu_p + c.m * sy_rho;
    const R nuc = c.nu_p + sy_rho * c.e_c;
    for (int k = 0; k < c.newton; ++k) {
        R gnu, dgnu;   // gdot nu_app(gdot) and its derivative
        if (gd >= c.gdot_c) {
            const R em = expm1(-c.m * gd);
            gnu = c.nu_p * gd - sy_rho * em;
            dgnu = c.nu_p + sy_rho * c.m * (R(1) + em);
        } else {
            const R s = gd * c.inv_gc;
            gnu = gd * ((R(1) - s) * nu0 + s * nuc);
            dgnu = nu0 + R(2) * s * (nuc - nu0);
        }
        const R h = R(0.5) * gd + R(3) * gnu - a;
        const R dh = fmax(R(0.5) + R(3) * dgnu, R(0.5));
        gd = fmax(gd - h / dh, R(0));
    }
    return gd;
}

// ---------------------------------------------------------------------------
// PR relaxation rates, per cell: strain rate with the previous step's tau
// (or the Newton-implicit one), apparent viscosity, tau and the two TRT rates.
template <bool IMPLICIT, class R>
__device__ __forceinline__ void pr_rates(const Coef<typename Lanes<R>::Sc>& c, R tn2, R inv, R& tau,
                                         R& wp_out, R& wm_out) {
    using Sc = typename Lanes<R>::Sc;
    Sc tau_[Lanes<R>::n], wp_[Lanes<R>::n], wm_[Lanes<R>::n];
#pragma unroll
    for (int k = 0; k < Lanes<R>::n; ++k) {
        // D = -T / (2 tau_old c_s^2) = -1.5 T / tau_old ; gdot = sqrt(2 D:D)
        const Sc tt = sqrt(Sc(2) * Lanes<R>::get(tn2, k));
        Sc gd = Sc(1.5) / Lanes<R>::get(tau, k) * tt;
        const Sc sy_rho = c.sigma_y * Lanes<R>::get(inv, k);
        if constexpr (IMPLICIT) gd = pr_newton(c, Sc(1.5) * tt, gd, sy_rho);
        Sc nu;
        if (gd >= c.gdot_c) {
            nu = c.nu_p + sy_rho * (-expm1(-c.m * gd)) / gd;
        } else {
            const Sc nu0 = c.nu_p + c.m * sy_rho;
            const Sc nuc = c.nu_p + sy_rho * c.e_c;
            nu = (c.gdot_c - gd) * c.inv_gc * nu0 + gd * c.inv_gc * nuc;
        }
        const Sc tn = Sc(0.5) + Sc(3) * nu;
        wp_[k] = Sc(1) / tn;
        // 1 / tau_odd with tau_odd = 1/2 + Lambda / (tau - 1/2), as one division
        const Sc tm = tn - Sc(0.5);
        wm_[k] = tm / (Sc(0.5) * tm + c.magic);
        tau_[k] = tn;
    }
    tau = Lanes<R>::make(tau_);
    wp_out = Lanes<R>::make(wp_);
    wm_out = Lanes<R>::make(wm_);
}

// The same for the pair form.  itau: 1 / (previous step's tau).  Both rates come
// from one reciprocal, of a moderate product (all but an extreme m or Lambda).
template <bool IMPLICIT>
__device__ __forceinline__ void pair_pr_rates(const Coef<double>& c, double tn2, double inv, double itau,
                                              double& tau, double& wp, double& wm) {
    const double tt = root(mul(4.5, tn2));   // 1.5 sqrt(2 T:T)
    double gd = mul(itau, tt);
    const double sy_rho = mul(c.sigma_y, inv);
    if constexpr (IMPLICIT) gd = pr_newton(c, tt, gd, sy_rho);
    double nu;
    if (!above(c.gdot_c, gd)) {
        const double y = mul(sy_rho, -expm1(mul(-c.m, gd)));
        nu = moderate(gd) ? mad(y, rcp(gd), c.nu_p) : add(c.nu_p, y / gd);
    } else {
        const double nu0 = mad(c.m, sy_rho, c.nu_p);
        const double nuc = mad(sy_rho, c.e_c, c.nu_p);
        const double s = mul(gd, c.inv_gc);
        nu = mad(mul(sub(c.gdot_c, gd), c.inv_gc), nu0, mul(s, nuc));
    }
    tau = mad(3.0, nu, 0.5);
    // 1 / tau_odd with tau_odd = 1/2 + Lambda / (tau - 1/2) is tm / odd
    const double tm = sub(tau, 0.5);
    const double odd = mad(0.5, tm, c.magic);
    const double product = mul(tau, odd);
    if (moderate(product)) {
        const double r = rcp(product);
        wp = mul(r, odd);
        wm = mul(tm, mul(r, tau));
    } else {
        wp = 1.0 / tau;
        wm = tm / odd;
    }
}

// ---------------------------------------------------------------------------
// PR collision (Sec. 3.1 + TRT + EDM).  tau: previous step's relaxation time
// in, this step's out.  f: memory units in, memory units out (the TRT update is
// linear and opposite populations share their unit).  R as for collide_ir.
// What the pairs need from the moments: K0, N and q of pair_terms and the rates.
template <class L, bool IMPLICIT, class R>
__device__ __forceinline__ void pr_terms(const Coef<typename Lanes<R>::Sc>& c, uint32_t flags,
                                         const Mom<R>& m, R& tau, R& K0, Tens<R>& N, R (&q)[3], R& wp,
                                         R& wm, R (&ur)[3]) {
    const R rho = add(R(1), m.d);
    R inv, itau;   // 1 / rho, 1 / tau_old, of a moderate product from one reciprocal
    const R product = mul(rho, tau);
    if (moderate(product)) {
        const R both = rcp(product);
        inv = mul(both, tau);
        itau = mul(both, rho);
    } else {
        inv = 1.0 / rho;
        itau = 1.0 / tau;
    }
    const R ux = mul(m.jx, inv), uy = mul(m.jy, inv);
    R uz = R(0);
    if constexpr (L::D == 3) uz = mul(m.jz, inv);
    {
        const Tens<R> T = noneq<L, R>(dynamic<L, R>(m), -m.jx, -m.jy, -m.jz, ux, uy, uz, flags);
        pair_pr_rates<IMPLICIT>(c, square<L, R>(T), inv, itau, tau, wp, wm);
    }
    const R gx = R(c.g[0]), gy = R(c.g[1]);
    R gz = R(0);
    if constexpr (L::D == 3) gz = R(c.g[2]);
    const R Fx = mul(rho, gx), Fy = mul(rho, gy);
    R Fz = R(0);
    if constexpr (L::D == 3) Fz = mul(rho, gz);
    // Per pair (i, o = opposite), with f^+- = (f_i +- f_o) / 2:
    //   E = f^+ - wp (f^+ - f_eq^+) + F^+ = (1 - wp)/2 (f_i + f_o) + w_i (K0 + 9/2 c.N.c),
    //       N = rho (wp u u + u g + g u + g g) = j (wp u + g) + F (u + g),
    //       K0 = wp d - 3/2 tr N;
    //   O = f^- - wm (f^- - f_eq^-) + F^- = (1 - wm)/2 (f_i - f_o) + 3 w_i c.(wm j + F),
    // the odd equilibrium and force parts from j and F directly (3 w_i rho c.u
    // = 3 w_i c.j exactly).  f holds the pair sums and differences.
    {
        const R vx = mad(wp, ux, gx), vy = mad(wp, uy, gy), zx = add(ux, gx), zy = add(uy, gy);
        N.xx = mad(m.jx, vx, mul(Fx, zx));
        N.yy = mad(m.jy, vy, mul(Fy, zy));
        N.xy = mad(m.jx, vy, mul(Fx, zy));
        N.zz = R(0);
        N.xz = R(0);
        N.yz = R(0);
        if constexpr (L::D == 3) {
            const R vz = mad(wp, uz, gz), zz = add(uz, gz);
            N.zz = mad(m.jz, vz, mul(Fz, zz));
            N.xz = mad(m.jx, vz, mul(Fx, zz));
            N.yz = mad(m.jy, vz, mul(Fy, zz));
        }
    }
    K0 = mad(R(-1.5), trace<L, R>(N), mul(wp, m.d));
    q[0] = mad(wm, m.jx, Fx);
    q[1] = mad(wm, m.jy, Fy);
    q[2] = R(0);
    if constexpr (L::D == 3) q[2] = mad(wm, m.jz, Fz);
    ur[0] = mad(R(0.5), gx, ux);
    ur[1] = mad(R(0.5), gy, uy);
    ur[2] = mad(R(0.5), gz, uz);
}

template <class L, class S, bool IMPLICIT, class R>
__device__ __forceinline__ void pair_collide_pr(const Coef<typename Lanes<R>::Sc>& c, uint32_t flags,
                                                R (&f)[L::Q], R& tau, R& drho, R (&ur)[3]) {
    const Mom<R> m = moments<L, S, R>(f);
    R K0, q[3], wp, wm;
    Tens<R> N;
    pr_terms<L, IMPLICIT, R>(c, flags, m, tau, K0, N, q, wp, wm, ur);
    const R omp = mad(R(-0.5), wp, R(0.5));
    const R omm = mad(R(-0.5), wm, R(0.5));
    f[0] = axpy(Store<S>::template gam<L, 0>(), K0, mad(-wp, f[0], f[0]));
    pair_terms<L, S, R>(K0, N, q[0], q[1], q[2], [&](auto I, R e, R cq, auto wo) {
        constexpr int i = decltype(I)::value;
        const R E = mad(omp, f[i], e);
        const R O = mad(omm, f[i + 1], scale(wo, cq));
        f[i] = add(E, O);
        f[i + 1] = sub(E, O);
    });
    drho = m.d;
}

// ---------------------------------------------------------------------------
// The same two collisions on class sums, for FP32 arithmetic (see pair_form).  R is
// the arithmetic type: one cell (float) or two cells (F2).
template <class L, class R> __device__ __forceinline__ R tnorm2(const Tens<R>& T) {
    R s = T.xx * T.xx + T.yy * T.yy + R(2) * T.xy * T.xy;
    if constexpr (L::D == 3) s += T.zz * T.zz + R(2) * (T.xz * T.xz + T.yz * T.yz);
    return s;
}

template <class L, class R>
__device__ __forceinline__ Tens<R> class_noneq(const Mom<R>& m, R rho, R ux, R uy, R uz, uint32_t flags) {
    const R d3 = m.d * R(1.0 / 3.0);
    Tens<R> t;
    t.xx = m.xx - d3 - rho * ux * ux;
    t.yy = m.yy - d3 - rho * uy * uy;
    t.xy = m.xy - rho * ux * uy;
    if constexpr (L::D == 3) {
        t.zz = m.zz - d3 - rho * uz * uz;
        t.xz = m.xz - rho * ux * uz;
        t.yz = m.yz - rho * uy * uz;
    } else {
        t.zz = R(0);
        t.xz = R(0);
        t.yz = R(0);
    }
    if (flags & LBM_FLAG_BURNETT_X) t.xx = R(0);
    return t;
}

// c.T.c for a lattice velocity, from T and the doubled off-diagonals
template <int cx, int cy, int cz, class R>
__device__ __forceinline__ R ctc(const Tens<R>& T, R t2xy, R t2xz, R t2yz) {
    return cdot6<cx * cx, cy * cy, cz * cz, cx * cy, cx * cz, cy * cz>(T.xx, T.yy, T.zz, t2xy,
                                                                        t2xz, t2yz);
}

template <class R>
__device__ __forceinline__ void class_ir_yield(const Coef<typename Lanes<R>::Sc>& c, R tn2, R& as_out,
                                         R& asg_out) {
    using Sc = typename Lanes<R>::Sc;
    Sc as[Lanes<R>::n], asg[Lanes<R>::n];
#pragma unroll
    for (int k = 0; k < Lanes<R>::n; ++k) {
        const Sc tn = sqrt(Lanes<R>::get(tn2, k));
        as[k] = Sc(0);
        asg[k] = Sc(-1);
        if (tn > Sc(0) && tn >= c.s2y) {
            const Sc it = Sc(1) / tn;
            as[k] = -(tn - c.s2y) * c.ir_a * it;
            asg[k] = -(c.six_nu * tn + c.s2y) * c.ir_b * it;
        }
    }
    as_out = Lanes<R>::make(as);
    asg_out = Lanes<R>::make(asg);
}

template <class L, class S, class R>
__device__ __forceinline__ void class_collide_ir(const Coef<typename Lanes<R>::Sc>& c, uint32_t flags,
                                           R (&f)[L::Q], R& drho, R (&ur)[3]) {
    const Mom<R> m = class_moments<L, S, R>(f);
    const R rho = R(1) + m.d;
    const R inv = recip(rho);
    const R Fx = rho * R(c.g[0]), Fy = rho * R(c.g[1]);
    R Fz = R(0);
    if constexpr (L::D == 3) Fz = rho * R(c.g[2]);
    const R ux = (m.jx + R(0.5) * Fx) * inv;
    const R uy = (m.jy + R(0.5) * Fy) * inv;
    R uz = R(0);
    if constexpr (L::D == 3) uz = (m.jz + R(0.5) * Fz) * inv;
    const Tens<R> T = class_noneq<L, R>(m, rho, ux, uy, uz, flags);
    R as, asg;
    class_ir_yield<R>(c, tnorm2<L, R>(T), as, asg);
    // A = -sigma_bar + s/2 = k1 T + k2 I with sigma_bar = sigma - tr(sigma)/D I
    const R trT = T.xx + T.yy + T.zz;
    const R k1 = R(0.5) * as - asg;
    const R k2 = asg * trT * R(1.0 / L::D);
    // (c c - c_s^2 I):A = k1 (cTc - trT/3) + k2 (|c|^2 - D/3) = h0 + k1 cTc + k2 |c|^2
    const R h0 = -(k1 * trT + k2 * R(L::D)) * R(1.0 / 3.0);
    const R uu = ux * ux + uy * uy + uz * uz;
    const R base = m.d - R(1.5) * rho * uu;
    const R r45 = R(4.5) * rho;
    const R k145 = R(4.5) * k1;
    const R t2xy = R(2) * T.xy, t2xz = R(2) * T.xz, t2yz = R(2) * T.yz;
    // odd part: w_i (3 rho c.u + 3/2 c.F) = 3 w_i c.(j + F), since rho u = j + F/2
    const R qx = m.jx + Fx, qy = m.jy + Fy, qz = m.jz + Fz;
    f[0] = R(Store<S>::template gam<L, 0>()) * (base + R(4.5) * h0);
    static_for<0, (L::Q - 1) / 2>([&](auto P) {
        constexpr int i = 2 * decltype(P)::value + 1;
        constexpr int o = i + 1;
        constexpr int cx = L::cx(i), cy = L::cy(i), cz = L::cz(i);
        constexpr int c2 = cx * cx + cy * cy + cz * cz;
        const R w = R(Store<S>::template gam<L, i>());   // w_i in memory units
        // even part e = w (base + 4.5 rho cu^2 + 4.5 h) = A + B cu^2 + C cTc (per class A, B, C)
        const R A = w * (base + R(4.5) * (h0 + k2 * R(c2)));
        const R B = w * r45;
        const R C = w * k145;
        const R cu = cdot<cx, cy, cz>(ux, uy, uz);
        const R e = A + B * (cu * cu) + C * ctc<cx, cy, cz>(T, t2xy, t2xz, t2yz);
        const R od = R(Store<S>::template god<L, i>()) * cdot<cx, cy, cz>(qx, qy, qz);
        f[i] = e + od;
        f[o] = e - od;
    });
    drho = m.d;
    ur[0] = ux;
    ur[1] = uy;
    ur[2] = uz;
}

template <class L, class S, bool IMPLICIT, class R>
__device__ __forceinline__ void class_collide_pr(const Coef<typename Lanes<R>::Sc>& c, uint32_t flags,
                                           R (&f)[L::Q], R& tau, R& drho, R (&ur)[3]) {
    const Mom<R> m = class_moments<L, S, R>(f);
    const R rho = R(1) + m.d;
    const R inv = recip(rho);
    const R ux = m.jx * inv, uy = m.jy * inv;
    R uz = R(0);
    if constexpr (L::D == 3) uz = m.jz * inv;
    const Tens<R> T = class_noneq<L, R>(m, rho, ux, uy, uz, flags);
    R wp, wm;
    pr_rates<IMPLICIT, R>(c, tnorm2<L, R>(T), inv, tau, wp, wm);
    const R gx = R(c.g[0]), gy = R(c.g[1]);
    R gz = R(0);
    if constexpr (L::D == 3) gz = R(c.g[2]);
    const R Fx = rho * gx, Fy = rho * gy, Fz = rho * gz;
    const R uu = ux * ux + uy * uy + uz * uz;
    const R ug = ux * gx + uy * gy + uz * gz;
    const R gg = gx * gx + gy * gy + gz * gz;
    const R base = m.d - R(1.5) * rho * uu;                 // even part of f_eq - w, direction-free
    const R fbase = R(-1.5) * rho * (R(2) * ug + gg);      // even part of the EDM difference
    const R r45 = R(4.5) * rho;
    // Per pair (i, o = opposite), with f^+- = (f_i +- f_o) / 2:
    //   E = f^+ - wp (f^+ - f_eq^+) + F^+ = (1 - wp)/2 (f_i + f_o) + w_i (K0 + 4.5 rho t),
    //       K0 = wp base + fbase,  t = wp cu^2 + cg (2 cu + cg) = cu (wp cu + 2 cg) + cg^2;
    //   O = f^- - wm (f^- - f_eq^-) + F^- = (1 - wm)/2 (f_i - f_o) + 3 w_i c.(wm j + F),
    // the odd equilibrium and force parts from j and F directly (3 w_i rho c.u
    // = 3 w_i c.j exactly).  cg = c_i.g and cg^2 are per-launch constants.
    const R omp = R(0.5) - R(0.5) * wp;
    const R omm = R(0.5) - R(0.5) * wm;
    const R K0 = wp * base + fbase;
    const R qx = wm * m.jx + Fx, qy = wm * m.jy + Fy, qz = wm * m.jz + Fz;
    {
        const R w0 = R(Store<S>::template gam<L, 0>());
        f[0] = (R(1) - wp) * f[0] + w0 * K0;
    }
    static_for<0, (L::Q - 1) / 2>([&](auto P) {
        constexpr int p = decltype(P)::value;
        constexpr int i = 2 * p + 1;
        constexpr int o = i + 1;
        constexpr int cx = L::cx(i), cy = L::cy(i), cz = L::cz(i);
        const R w = R(Store<S>::template gam<L, i>());    // w_i and 3 w_i in memory units
        const R w3 = R(Store<S>::template god<L, i>());
        const R cu = cdot<cx, cy, cz>(ux, uy, uz);
        const R cg = R(c.cg[p]);
        const R t = cu * (wp * cu + R(2) * cg) + R(c.cgg[p]);
        const R E = omp * (f[i] + f[o]) + w * (K0 + r45 * t);
        const R O = omm * (f[i] - f[o]) + w3 * cdot<cx, cy, cz>(qx, qy, qz);
        f[i] = E + O;
        f[o] = E - O;
    });
    drho = m.d;
    ur[0] = ux + R(0.5) * gx;
    ur[1] = uy + R(0.5) * gy;
    ur[2] = uz + R(0.5) * gz;
}

template <class L, class S, class R = typename Store<S>::R>
__device__ __forceinline__ void collide_ir(const Coef<typename Lanes<R>::Sc>& c, uint32_t flags,
                                           R (&f)[L::Q], R& drho, R (&ur)[3]) {
    if constexpr (pair_form<S>()) pair_collide_ir<L, S, R>(c, flags, f, drho, ur);
    else class_collide_ir<L, S, R>(c, flags, f, drho, ur);
}

template <class L, class S, bool IMPLICIT, class R = typename Store<S>::R>
__device__ __forceinline__ void collide_pr(const Coef<typename Lanes<R>::Sc>& c, uint32_t flags,
                                           R (&f)[L::Q], R& tau, R& drho, R (&ur)[3]) {
    if constexpr (pair_form<S>()) pair_collide_pr<L, S, IMPLICIT, R>(c, flags, f, tau, drho, ur);
    else class_collide_pr<L, S, IMPLICIT, R>(c, flags, f, tau, drho, ur);
}

// ---------------------------------------------------------------------------
// deterministic block reduction of kNumStats values (fixed shuffle tree).
// The warp and block stages run in the type of v (the arithmetic type on
// check steps: at most 256 terms); each block's sums are stored as FP64
// partials and summed in FP64 in a fixed order by the finaliser.  Keeping the
// block stage off the FP64 pipe matters on GB300, whose FP64 rate is a small
// fraction of FP32: a serial FP64 shuffle chain per block made check steps
// four to five times slower than plain steps.
template <class V>
__device__ __forceinline__ void block_sum_store(V (&v)[kNumStats], double* __restrict__ out) {
    __shared__ V sm[kBlock / 32][kNumStats];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
    for (int k = 0; k < kNumStats; ++k) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) v[k] += __shfl_down_sync(0xffffffffu, v[k], o);
    }
    if (lane == 0) {
#pragma unroll
        for (int k = 0; k < kNumStats; ++k) sm[warp][k] = v[k];
    }
    __syncthreads();
    if (warp == 0) {
#pragma unroll
        for (int k = 0; k < kNumStats; ++k) {
            V t = (lane < kBlock / 32) ? sm[lane][k] : V(0);
#pragma unroll
            for (int o = 4; o > 0; o >>= 1) t += __shfl_down_sync(0xffffffffu, t, o);
            if (lane == 0) out[k] = (double)t;
        }
    }
}

// ---------------------------------------------------------------------------
// Overlapped launches.  Step kernels are launched, where it pays (launch_step),
// with programmatic stream serialisation: a kernel's blocks may start while the
// previous step drains, read what no step writes (link words, maps,
// coefficients), and wait for the
// previous step's stores before they touch anything else.  step_begin() is
// that wait; `n`, which every later address is formed from, passes through it
// so that no load can move up past it.  Only then the next launch is let in,
// so a kernel never overlaps more than the one before it, and the lines it
// reads (the ones that kernel writes) cannot sit stale in L1: the last kernel
// that read them has ended before this kernel's blocks are launched.  Every
// block calls it, also one with nothing to do (but for the compact 16-bit steps,
// which are never overlapped).  A small step is mostly launch and ramp (us a step,
// plain -> overlapped: D2Q9 FP32 IR, 128 x 128: 2.1 -> 1.6; D3Q15 FP32 PR, 45 x 47 x 43:
// 3.6 -> 3.1), a large one gains its last, partly filled wave (D3Q27 duct 256 x 128 x
// 128: FP32 PR 138.8 -> 138.5, FP16 PR 111.6 -> 111.2).
__device__ __forceinline__ void step_begin(int& n) {
    asm volatile("griddepcontrol.wait;\n\tgriddepcontrol.launch_dependents;" : "+r"(n) : : "memory");
}

// ---------------------------------------------------------------------------
// the fused step
//
// Minimum resident blocks per SM requested from the register allocator (0 =
// let it choose).  PR in FP32 arithmetic (FP32 and 16-bit storage): D3Q27
// keeps 1024 threads resident per SM at 256 and 512 threads per block (64
// registers) and 9 blocks at 128 (56 registers); a tighter cap spills.  The
// smaller lattices keep 1280 (10 x 128, 5 x 256, 2 x 512): D3Q19 PR then
// takes 48 registers without spilling and measured 7-9 % faster than at 64
// (porous box 256^3: FP32 466 -> 430 us, FP16 440 -> 401 us; duct
// 256 x 128 x 128: FP32 113.5 -> 105.7 us).  IR (40-48 registers) and FP64
// arithmetic (which these caps would make spill) are left to the allocator.
// BLBM_PR_MINB / BLBM_IR_MINB override at build time.
#ifndef BLBM_PR_MINB
#define BLBM_PR_MINB -1
#endif
#ifndef BLBM_IR_MINB
#define BLBM_IR_MINB 0
#endif
template <class L, int MODEL, class S, bool CHECK, int BLOCK> constexpr int step_min_blocks() {
    if (BLOCK < 128) return 0;   // small grids, and FP64: left to the allocator
    if (MODEL == LBM_MODEL_IR) return BLBM_IR_MINB;
    if (std::is_same<typename Store<S>::R, double>::value) return 0;
    if (BLBM_PR_MINB >= 0) return BLBM_PR_MINB;
    if (L::Q == 27 || CHECK) return BLOCK == 128 ? 9 : 1024 / BLOCK;   // check steps: no spill
    return 1280 / BLOCK;
}

// Stores one cell's outgoing populations at element n of the planes: the
// rest population, then the opposite pairs (i, i + 1), one random word each.
template <class L, class S, class Dst>
__device__ __forceinline__ void store_cell(const Dst& dst, int n,
                                           const typename Store<S>::R (&f)[L::Q], uint32_t rnd) {
    Store<S>::template st<L, 0>(dst.template at<0>(n), f[0], rnd);
    static_for<0, (L::Q - 1) / 2>([&](auto P) {
        constexpr int i = 2 * decltype(P)::value + 1;
        Store<S>::template st2<L, i>(dst.template at<i>(n), dst.template at<i + 1>(n), f[i],
                                     f[i + 1], pair_bits<decltype(P)::value + 1>(rnd));
    });
}

// A cell's check-step contributions (velocity, its change since the previous
// snapshot up, density offset, non-finite flag); its velocity becomes element
// n of the snapshot.
template <class R>
__device__ __forceinline__ void check_stats(const R (&ur)[3], const R (&up)[3], R drho,
                                            R* __restrict__ usnap, int64_t plane, int n,
                                            R (&acc)[kNumStats]) {
    R du2 = R(0), u2 = R(0);
#pragma unroll
    for (int d = 0; d < 3; ++d) {
        acc[kStatUx + d] = ur[d];
        du2 += (ur[d] - up[d]) * (ur[d] - up[d]);
        u2 += ur[d] * ur[d];
        usnap[(int64_t)d * plane + n] = ur[d];
    }
    acc[kStatDu2] = du2;
    acc[kStatU2] = u2;
    acc[kStatDrho] = drho;
    acc[kStatNonFinite] = isfinite(drho) ? R(0) : R(1);
}

// One cell of one time step: pull, collide, store; on check steps the cell's
// contributions to the flow-rate and residual sums go to acc.  Shared by the
// single-domain and the batched kernels so both do identical arithmetic.
// fluid = false copies a solid cell's populations through unchanged, the
// step's definition for solid cells: the stores of a group of cells that
// holds fluid cells then fill whole 32-byte sectors.  A sector the stores
// cover only in part costs a DRAM read before its write; at the edges of a
// porous medium's grains that doubled the reads.
template <class L, int MODEL, class S, bool CHECK, class Src, class Dst>
__device__ __forceinline__ void cell_step(const KParams& kp, const Coef<typename Store<S>::R>& c,
                                          const Src& src, const Dst& dst, uint32_t lk, int idx,
                                          typename Store<S>::R* __restrict__ tau,
                                          typename Store<S>::R* __restrict__ usnap, uint32_t rnd,
                                          typename Store<S>::R (&acc)[kNumStats],
                                          bool fluid = true) {
    using R = typename Store<S>::R;
    // check steps: the previous snapshot is read first, so its latency overlaps
    // the gather (after the population stores the compiler could not move
    // these loads up past them: the pointers may alias)
    R up[3] = {R(0), R(0), R(0)};
    if constexpr (CHECK) {
#pragma unroll
        for (int d = 0; d < 3; ++d) up[d] = usnap[(int64_t)d * kp.plane + idx];
    }
    R f[L::Q];
    gather<L, S>(kp, src, fluid ? lk : 0u, idx, f, !fluid);
    R drho = R(0), ur[3] = {R(0), R(0), R(0)};
    if (fluid) {
        if constexpr (MODEL != LBM_MODEL_IR) {
            R t = tau[idx];
            collide_pr<L, S, MODEL == kModelPRImplicit>(c, kp.flags, f, t, drho, ur);
            tau[idx] = t;
        } else {
            collide_ir<L, S>(c, kp.flags, f, drho, ur);
        }
    }
    store_cell<L, S>(dst, idx, f, rnd);
    if constexpr (CHECK) check_stats(ur, up, drho, usnap, kp.plane, idx, acc);
}

// Copy-through: the solid cells that share an aligned group of 8 consecutive
// cells (one 32-byte sector of a plane of 4-byte words) with a fluid cell run
// cell_step with fluid = false, which stores their populations unchanged, so
// the stores fill whole sectors (plain and check steps).  Groups without fluid
// cells are neither read nor written.  (The earlier rule, every solid cell of
// a warp that holds fluid cells, also moved the all-solid sectors of mixed
// warps: on a porous box of porosity 0.7 with grains of radius 6-10 it
// touched 1.43x the fluid cells' bytes, the 8-cell groups 1.27x.)  For the PR
// step of the 16-bit forms it is a per-solver choice (COPY), because there
// its path costs registers: on the D3Q27 duct, which has no warp mixing
// solid and fluid cells, it spills and the step is 6 % slower, while on a
// porous box it saves 7 % (256^3 D3Q19: 431 -> 401 us).  The solver takes it
// when at least 1 % of its warps with fluid cells also hold solid ones.
// (Solid lanes copying their raw words in a branch of their own keep the
// fluid path's registers, but a mixed warp then runs both branches one after
// the other: 40 % slower on the porous box in FP32.)
template <int MODEL, class S> __host__ __device__ constexpr bool copy_is_choice() {
    return MODEL != LBM_MODEL_IR && sizeof(S) == 2;
}

// Whether the aligned group of kCopyGroup cells holding cell idx has a fluid
// cell among the warp's active lanes.  Lane l holds cell idx - (threadIdx.x &
// 31) + l; cells of the group outside the warp count as solid (possible only
// when a launch does not start on a group boundary, a step taken in parts).
constexpr int kCopyGroup = 8;
__device__ __forceinline__ bool group_has_fluid(bool fluid, int idx) {
    const uint32_t b = __ballot_sync(__activemask(), fluid);
    const int first = (int)(threadIdx.x & 31) - (idx & (kCopyGroup - 1));   // -7 .. 31
    return ((((uint64_t)b << 32) >> (first + 32)) & ((1u << kCopyGroup) - 1u)) != 0;
}

// BLOCK: threads per block, chosen per (lattice, model, storage, size class)
// by the tuning table; check steps always run with kBlock so their reduction
// order does not depend on the tuning.
// RANGE: the launch covers cells [cell_begin, cell_end) only, one part of a
// step taken in parts (lbm_step_cells; 256 threads, plain steps).  Its own
// instantiation, so the whole-domain kernels carry no range arithmetic: under
// the 48-register budget of the smaller lattices it made the D3Q19 FP32 PR
// step spill and run 4 % slower.
template <class L, int MODEL, class S, bool CHECK, int BLOCK = kBlock, bool COPY = true,
          bool RANGE = false>
__global__ void __launch_bounds__(BLOCK, step_min_blocks<L, MODEL, S, CHECK, BLOCK>())
k_step(const KArgs a, const SrcPlanes<S> src, const DstPlanes<S> dst,
       const uint32_t* __restrict__ links, typename Store<S>::R* __restrict__ tau,
       typename Store<S>::R* __restrict__ usnap, double* __restrict__ partials,
       uint32_t* __restrict__ rng_ctr, int parity) {
    static_assert(!CHECK || BLOCK == kBlock, "check steps use the fixed block size");
    using R = typename Store<S>::R;
    const KParams& kp = a.kp;
    int idx = (RANGE ? kp.cell_begin : 0) + (int)(blockIdx.x * BLOCK + threadIdx.x);
    const bool inside = idx < (RANGE ? kp.cell_end : kp.ncells);
    uint32_t lk = kSolidBit, rnd = 0u;
    if constexpr (!Store<S>::kStochastic) {
        if (inside) lk = __ldg(links + idx);
        step_begin(idx);
    } else {
        step_begin(idx);
        // this launch reads counter[parity] and leaves counter + 1 for the next
        const uint32_t seed = rng_ctr[parity];
        if (blockIdx.x == 0 && threadIdx.x == 0) rng_ctr[parity ^ 1] = seed + 1u;
        rnd = pcg_hash(((uint32_t)idx + kp.hash_offset) ^ (seed * 0x9e3779b9u));
        // behind the hash: before it, the PR step is slower than the wait it hides
        // (FP16 duct 256 x 128 x 128, D3Q19 92.6 us against 88.8; D3Q27 at 256 threads
        // 128.4 against 119.0)
        if (inside) lk = __ldg(links + idx);
    }
    const bool active = !(lk & kSolidBit);
    R acc[kNumStats];
    if constexpr (!CHECK) {
        if constexpr (COPY) {
            // a group without fluid cells has nothing to do; in any other group
            // the solid cells inside the domain copy their populations through
            if (!group_has_fluid(active, idx) || !inside) return;
            cell_step<L, MODEL, S, false>(kp, coef<R>(a), src, dst, lk, idx, tau, usnap, rnd, acc,
                                          active);
        } else {
            if (!active) return;
            cell_step<L, MODEL, S, false>(kp, coef<R>(a), src, dst, lk, idx, tau, usnap, rnd, acc);
        }
    } else {
#pragma unroll
        for (int k = 0; k < kNumStats; ++k) acc[k] = R(0);
        if constexpr (COPY) {
            // solid cells add nothing to the sums: their velocity and snapshot are 0
            if (group_has_fluid(active, idx) && inside)
                cell_step<L, MODEL, S, true>(kp, coef<R>(a), src, dst, lk, idx, tau, usnap, rnd, acc,
                                             active);
        } else {
            if (active)
                cell_step<L, MODEL, S, true>(kp, coef<R>(a), src, dst, lk, idx, tau, usnap, rnd, acc);
        }
        block_sum_store(acc, partials + (int64_t)blockIdx.x * kNumStats);
    }
}

// ---------------------------------------------------------------------------
// Two cells per thread.  Thread t of a block works on cells base + t and
// base + t + BLOCK, so every load and store instruction of a warp stays
// contiguous; it gathers and stores each cell as cell_step does and runs one
// collision on F2 values (packed f32x2 arithmetic for both cells).  A lane
// whose cell is solid or past the end repeats the other cell's work and
// stores nothing.  Plain steps of the FP32 and 16-bit forms only.
template <class L, int MODEL, class S, class Src, class Dst>
__device__ __forceinline__ void cell_step2(const KParams& kp, const Coef<float>& c, const Src& src,
                                           const Dst& dst, const uint32_t (&lk)[2],
                                           const int (&idx)[2], const bool (&act)[2],
                                           float* __restrict__ tau, const uint32_t (&rnd)[2]) {
    float a[L::Q], b[L::Q];
    gather<L, S>(kp, src, lk[0], idx[0], a);
    gather<L, S>(kp, src, lk[1], idx[1], b);
    F2 f[L::Q];
    static_for<0, L::Q>([&](auto I) {
        constexpr int i = decltype(I)::value;
        f[i] = F2(a[i], b[i]);
    });
    F2 drho, ur[3];
    if constexpr (MODEL != LBM_MODEL_IR) {
        F2 t(tau[idx[0]], tau[idx[1]]);
        collide_pr<L, S, MODEL == kModelPRImplicit, F2>(c, kp.flags, f, t, drho, ur);
        if (act[0]) tau[idx[0]] = t.lo();
        if (act[1]) tau[idx[1]] = t.hi();
    } else {
        collide_ir<L, S, F2>(c, kp.flags, f, drho, ur);
    }
    static_for<0, 2>([&](auto K) {
        constexpr int k = decltype(K)::value;
        if (act[k]) {
            const int n = idx[k];
            Store<S>::template st<L, 0>(dst.template at<0>(n), Lanes<F2>::get(f[0], k), rnd[k]);
            static_for<0, (L::Q - 1) / 2>([&](auto P) {
                constexpr int i = 2 * decltype(P)::value + 1;
                Store<S>::template st2<L, i>(dst.template at<i>(n), dst.template at<i + 1>(n),
                                             Lanes<F2>::get(f[i], k), Lanes<F2>::get(f[i + 1], k),
                                             pair_bits<decltype(P)::value + 1>(rnd[k]));
            });
        }
    });
}

// PR: at most 128 registers a thread, so 16 warps (1024 cells) stay resident
// per SM, the memory-level parallelism of the one-cell PR kernel.  IR needs
// fewer registers unbounded.
template <int MODEL, int BLOCK> constexpr int step2_min_blocks() {
    return MODEL == LBM_MODEL_IR ? 0 : 512 / BLOCK;
}

template <class L, int MODEL, class S, int BLOCK>
__global__ void __launch_bounds__(BLOCK, step2_min_blocks<MODEL, BLOCK>())
k_step2(const KArgs a, const SrcPlanes<S> src, const DstPlanes<S> dst,
        const uint32_t* __restrict__ links, float* __restrict__ tau,
        uint32_t* __restrict__ rng_ctr, int parity) {
    static_assert(std::is_same<typename Store<S>::R, float>::value, "two-cell steps need FP32 arithmetic");
    const KParams& kp = a.kp;
    int i0 = blockIdx.x * (2 * BLOCK) + threadIdx.x;
    const uint32_t l0 = i0 < kp.ncells ? __ldg(links + i0) : kSolidBit;
    const uint32_t l1 = i0 + BLOCK < kp.ncells ? __ldg(links + i0 + BLOCK) : kSolidBit;
    step_begin(i0);
    const int i1 = i0 + BLOCK;
    uint32_t seed = 0u;
    if constexpr (Store<S>::kStochastic) {
        // this launch reads counter[parity] and leaves counter + 1 for the next
        seed = rng_ctr[parity];
        if (blockIdx.x == 0 && threadIdx.x == 0) rng_ctr[parity ^ 1] = seed + 1u;
    }
    const bool a0 = !(l0 & kSolidBit), a1 = !(l1 & kSolidBit);
    if (!a0 && !a1) return;
    const int idx[2] = {a0 ? i0 : i1, a1 ? i1 : i0};
    const uint32_t lk[2] = {a0 ? l0 : l1, a1 ? l1 : l0};
    const bool act[2] = {a0, a1};
    uint32_t rnd[2] = {0u, 0u};
    if constexpr (Store<S>::kStochastic) {
        rnd[0] = pcg_hash(((uint32_t)idx[0] + kp.hash_offset) ^ (seed * 0x9e3779b9u));
        rnd[1] = pcg_hash(((uint32_t)idx[1] + kp.hash_offset) ^ (seed * 0x9e3779b9u));
    }
    cell_step2<L, MODEL, S>(kp, a.cf, src, dst, lk, idx, act, tau, rnd);
}

// ---------------------------------------------------------------------------
// Divided FP64 steps.  An FP64 warp instruction holds its SM sub-partition's
// FP64 pipe for 64 cycles whatever it has in flight, so a small domain, one warp
// on each of a few sub-partitions, takes as long as its longest warp however
// many others idle.  Here the cells of one warp are stepped by parts<L>() warps:
// each gathers, pairs up and stores the populations of its part (see
// pair_part); the family sums that pair_moments combines go through shared
// memory, its combining adds are dealt out to the warps, and what follows from
// the moments is done by every warp for itself.  The expressions are those of
// pair_moments, ir_terms, pr_terms and pair_terms, so the results are the bits of
// the undivided step.  FP64 operations of the longest warp, D3Q27 IR: about 96
// against 215.
enum { kExFace = 0, kExCorner = 12, kExAxis = 19, kExRest = 25, kExCount = 26 };
struct SplitShared {
    double ex[kExCount][32];   // family sums: 4 per face plane, 7 of the corners, the axis pairs, f_0
    double mo[10][32];         // d, j, p
};
// f(part as a constant)
template <class L, class F> __device__ __forceinline__ void by_part(int part, F&& f) {
    if (part == 0) f(std::integral_constant<int, 0>{});
    else if (part == 1) f(std::integral_constant<int, 1>{});
    if constexpr (parts<L>() == 4) {
        if (part == 2) f(std::integral_constant<int, 2>{});
        else if (part == 3) f(std::integral_constant<int, 3>{});
    }
}
// r[2 k], r[2 k + 1]: populations (i, i + 1) of a part's pair k; f(i, place in r)
template <class L, int PART, class F> __device__ __forceinline__ void part_pops(F&& f) {
    static_for<0, 4>([&](auto K) {
        constexpr int k = decltype(K)::value, p = part_pair<L>(PART, k);
        if constexpr (p >= 0) {
            f(std::integral_constant<int, 2 * p + 1>{}, std::integral_constant<int, 2 * k>{});
            f(std::integral_constant<int, 2 * p + 2>{}, std::integral_constant<int, 2 * k + 1>{});
        }
    });
}
// pair form of a part, and its family sums
template <class L, int PART>
__device__ __forceinline__ void part_sums(double (&r)[8], double f0, SplitShared& sh, int lane) {
    static_for<0, 4>([&](auto K) {
        constexpr int k = 2 * decltype(K)::value;
        if constexpr (part_pair<L>(PART, k / 2) >= 0) {
            const double a = r[k], b = r[k + 1];
            r[k] = add(a, b);
            r[k + 1] = sub(a, b);
        }
    });
    if constexpr (PART == 0) {
#pragma unroll
        for (int d = 0; d < L::D; ++d) {
            sh.ex[kExAxis + d][lane] = r[2 * d];
            sh.ex[kExAxis + 3 + d][lane] = r[2 * d + 1];
        }
        sh.ex[kExRest][lane] = f0;
    }
    constexpr int F = Fam<L>::face, C = Fam<L>::corner;
    if constexpr (F != 0) {
        static_for<0, L::D == 2 ? 1 : 3>([&](auto J) {
            constexpr int j = decltype(J)::value, p = (F - 1) / 2 + 2 * j;
            if constexpr (pair_part<L>(p) == PART) {
                constexpr int k = 2 * part_place<L>(p);
                sh.ex[kExFace + 4 * j][lane] = add(r[k], r[k + 2]);
                sh.ex[kExFace + 4 * j + 1][lane] = sub(r[k], r[k + 2]);
                sh.ex[kExFace + 4 * j + 2][lane] = add(r[k + 1], r[k + 3]);
                sh.ex[kExFace + 4 * j + 3][lane] = sub(r[k + 1], r[k + 3]);
            }
        });
    }
    if constexpr (C != 0) {
        if constexpr (pair_part<L>((C - 1) / 2) == PART) {
            constexpr int k = 2 * part_place<L>((C - 1) / 2);
            const double ab = add(r[k], r[k + 2]), amb = sub(r[k], r[k + 2]);
            const double ce = add(r[k + 4], r[k + 6]), cme = sub(r[k + 4], r[k + 6]);
            const double dp = add(r[k + 1], r[k + 3]), dq = sub(r[k + 5], r[k + 7]);
            sh.ex[kExCorner][lane] = add(ab, ce);
            sh.ex[kExCorner + 1][lane] = sub(ab, ce);
            sh.ex[kExCorner + 2][lane] = add(amb, cme);
            sh.ex[kExCorner + 3][lane] = sub(amb, cme);
            sh.ex[kExCorner + 4][lane] = add(dp, dq);
            sh.ex[kExCorner + 5][lane] = sub(dp, dq);
            sh.ex[kExCorner + 6][lane] = add(sub(r[k + 1], r[k + 3]), add(r[k + 5], r[k + 7]));
        }
    }
}
// the combining adds of pair_moments, dealt out by moment
template <class L, int PART> __device__ __forceinline__ void part_moments(SplitShared& sh, int lane) {
    constexpr bool F = Fam<L>::face != 0, C = Fam<L>::corner != 0;
    auto e = [&](int k) { return sh.ex[k][lane]; };
    auto face = [&](int j, int k) { return e(kExFace + 4 * j + k); };   // k: sum, difference; odd ones
    if constexpr (L::D == 2) {
        if constexpr (PART == 0) {
            const double xx = add(face(0, 0), e(kExAxis));
            sh.mo[4][lane] = xx;
            sh.mo[0][lane] = add(xx, add(e(kExAxis + 1), e(kExRest)));
        } else {
            sh.mo[5][lane] = add(face(0, 0), e(kExAxis + 1));
            sh.mo[7][lane] = face(0, 1);
            sh.mo[1][lane] = add(face(0, 2), e(kExAxis + 3));
            sh.mo[2][lane] = add(face(0, 3), e(kExAxis + 4));
        }
    } else {
        // diagonal sum beyond the axis pair: corners, then the two planes of the axis
        auto diag = [&](int j, int k) {
            if constexpr (F && C) return add(e(kExCorner), add(face(j, 0), face(k, 0)));
            else if constexpr (F) return add(face(j, 0), face(k, 0));
            else return e(kExCorner);
        };
        auto off = [&](int j) {
            if constexpr (F && C) return add(e(kExCorner + 1 + j), face(j, 1));
            else if constexpr (F) return face(j, 1);
            else return e(kExCorner + 1 + j);
        };
        // odd sum of an axis: corners, then two planes' terms a and b
        auto odd = [&](int axis, int ja, int ka, int jb, int kb) {
            double v;
            if constexpr (F) {
                v = add(face(ja, ka), face(jb, kb));
                if constexpr (C) v = add(e(kExCorner + 4 + axis), v);
            } else {
                v = e(kExCorner + 4 + axis);
            }
            return add(v, e(kExAxis + 3 + axis));
        };
        constexpr bool two = parts<L>() == 2;
        if constexpr (PART == 0) {
            const double xx = add(diag(0, 1), e(kExAxis));
            double rest = add(e(kExAxis + 1), e(kExAxis + 2));
            if constexpr (F) rest = add(rest, face(2, 0));
            sh.mo[4][lane] = xx;
            sh.mo[0][lane] = add(xx, add(rest, e(kExRest)));
        }
        if constexpr (PART == 1) {
            sh.mo[5][lane] = add(diag(0, 2), e(kExAxis + 1));
            sh.mo[6][lane] = add(diag(1, 2), e(kExAxis + 2));
            sh.mo[7][lane] = off(0);
        }
        if constexpr (PART == (two ? 0 : 2)) {
            sh.mo[1][lane] = odd(0, 0, 2, 1, 2);
            sh.mo[2][lane] = odd(1, 0, 3, 2, 2);
            sh.mo[8][lane] = off(1);
        }
        if constexpr (PART == (two ? 1 : 3)) {
            sh.mo[3][lane] = odd(2, 1, 3, 2, 3);
            sh.mo[9][lane] = off(2);
        }
    }
}
// The divided collision of a warp's cells: r, f0 in and out as populations, tau in
// and out.  Every thread of the block calls it (two block barriers); `on`:
// this lane's cell collides.
template <class L, int MODEL>
__device__ __forceinline__ void split_collide(const Coef<double>& c, uint32_t flags, int part, int lane,
                                              bool on, SplitShared& sh, double (&r)[8], double& f0,
                                              double& tau) {
    if (on) by_part<L>(part, [&](auto P) { part_sums<L, decltype(P)::value>(r, f0, sh, lane); });
    __syncthreads();
    if (on) by_part<L>(part, [&](auto P) { part_moments<L, decltype(P)::value>(sh, lane); });
    __syncthreads();
    if (!on) return;
    Mom<double> m;
    m.d = sh.mo[0][lane];
    m.jx = sh.mo[1][lane];
    m.jy = sh.mo[2][lane];
    m.xx = sh.mo[4][lane];
    m.yy = sh.mo[5][lane];
    m.xy = sh.mo[7][lane];
    m.jz = L::D == 3 ? sh.mo[3][lane] : 0.0;
    m.zz = L::D == 3 ? sh.mo[6][lane] : 0.0;
    m.xz = L::D == 3 ? sh.mo[8][lane] : 0.0;
    m.yz = L::D == 3 ? sh.mo[9][lane] : 0.0;
    double e0, q[3], ur[3];
    Tens<double> N;
    if constexpr (MODEL == LBM_MODEL_IR) {
        ir_terms<L, double>(c, flags, m, e0, N, q, ur);
        by_part<L>(part, [&](auto P) {
            constexpr int PART = decltype(P)::value;
            if constexpr (PART == 0) f0 = scale(Store<double>::template gam<L, 0>(), e0);
            pair_terms<L, double, double, PART>(e0, N, q[0], q[1], q[2], [&](auto I, double e, double cq, auto wo) {
                constexpr int k = 2 * part_place<L>((decltype(I)::value - 1) / 2);
                r[k] = axpy(wo, cq, e);
                r[k + 1] = axpy(-wo, cq, e);
            });
        });
    } else {
        double wp, wm;
        pr_terms<L, false, double>(c, flags, m, tau, e0, N, q, wp, wm, ur);
        const double omp = mad(-0.5, wp, 0.5);
        const double omm = mad(-0.5, wm, 0.5);
        by_part<L>(part, [&](auto P) {
            constexpr int PART = decltype(P)::value;
            if constexpr (PART == 0)
                f0 = axpy(Store<double>::template gam<L, 0>(), e0, mad(-wp, f0, f0));
            pair_terms<L, double, double, PART>(e0, N, q[0], q[1], q[2], [&](auto I, double e, double cq, auto wo) {
                constexpr int k = 2 * part_place<L>((decltype(I)::value - 1) / 2);
                const double E = mad(omp, r[k], e);
                const double O = mad(omm, r[k + 1], scale(wo, cq));
                r[k] = add(E, O);
                r[k + 1] = sub(E, O);
            });
        });
    }
}

// Plain FP64 step, the 32 cells of a block by parts<L>() warps.
template <class L, int MODEL>
__global__ void __launch_bounds__(32 * parts<L>())
k_step_split(const KArgs a, const SrcPlanes<double> src, const DstPlanes<double> dst,
             const uint32_t* __restrict__ links, double* __restrict__ tau) {
    __shared__ SplitShared sh;
    const KParams& kp = a.kp;
    const int lane = threadIdx.x & 31, part = threadIdx.x >> 5;
    int idx = blockIdx.x * 32 + lane;
    const bool inside = idx < kp.ncells;
    const uint32_t lk = inside ? __ldg(links + idx) : kSolidBit;
    step_begin(idx);
    const bool on = !(lk & kSolidBit);
    // as k_step: the solid cells of a group with fluid copy through
    const bool go = group_has_fluid(on, idx) && inside;
    if (!__any_sync(0xffffffffu, go)) return;   // the same cells in every warp
    double r[8], f0 = 0.0, t = 0.0;
    if (go) {
        PullOffsets o{0, 0, 0, 0, 0, 0};
        if (on) o = pull_offsets(kp, idx);
        const uint32_t wall = on ? lk : 0u;
        by_part<L>(part, [&](auto P) {
            constexpr int PART = decltype(P)::value;
            if constexpr (PART == 0) f0 = *src.template at<0>(idx);
            part_pops<L, PART>([&](auto I, auto K) {
                constexpr int i = decltype(I)::value;
                r[decltype(K)::value] = ((wall >> i) & 1u) ? *src.template at<L::opp(i)>(idx)
                                                           : *src.template at<i>(idx + o.template of<L, i>());
            });
        });
        if constexpr (MODEL != LBM_MODEL_IR)
            if (on) t = tau[idx];
    }
    split_collide<L, MODEL>(a.cd, kp.flags, part, lane, on, sh, r, f0, t);
    if (!go) return;
    by_part<L>(part, [&](auto P) {
        constexpr int PART = decltype(P)::value;
        if constexpr (PART == 0) {
            *dst.template at<0>(idx) = f0;
            if constexpr (MODEL != LBM_MODEL_IR)
                if (on) tau[idx] = t;
        }
        part_pops<L, PART>([&](auto I, auto K) {
            *dst.template at<decltype(I)::value>(idx) = r[decltype(K)::value];
        });
    });
}

// ---------------------------------------------------------------------------
// Resident steps: a run of plain steps of a small domain in one launch, its
// populations held in the shared memory of one cluster.  A step of such a
// domain is almost only launch and memory latency (256 cells: 1.6 us of which
// the arithmetic is a quarter); here a step is a gather from the cluster's
// shared memory, the collision and one cluster barrier.  Thread t of block b
// owns cell b T + t for the whole run (T = blockDim.x), so where each of its
// populations comes from (a neighbour's slot, in this block or another one of
// the cluster, or at a wall its own opposite population) is worked out once.
// Arithmetic, rounding bits and results are k_step's.
//
// Most threads per block: the registers hold the source addresses and the
// populations of one cell.  FP64 is kept to one warp per SM sub-partition
// (see untuned_block).
template <class L, class S> __host__ __device__ constexpr int resident_threads() {
    return sizeof(typename Store<S>::R) == 8 ? 128 : L::Q == 9 ? 640 : 512;
}
constexpr int kResidentCluster = 16;    // blocks per cluster (non-portable above 8)

template <class S> __device__ __forceinline__ typename Store<S>::R ld_cluster(uint32_t a) {
    if constexpr (sizeof(S) == 8) {
        double v;
        asm volatile("ld.shared::cluster.f64 %0, [%1];" : "=d"(v) : "r"(a));
        return v;
    } else if constexpr (sizeof(S) == 4) {
        float v;
        asm volatile("ld.shared::cluster.f32 %0, [%1];" : "=f"(v) : "r"(a));
        return v;
    } else {
        unsigned short v;
        asm volatile("ld.shared::cluster.u16 %0, [%1];" : "=h"(v) : "r"(a));
        if constexpr (std::is_same<S, __half>::value) return __half2float(__ushort_as_half(v));
        else return __bfloat162float(__ushort_as_bfloat16(v));
    }
}
// one barrier of the cluster's threads; the writes before it are visible after it
__device__ __forceinline__ void cluster_barrier() {
    asm volatile("barrier.cluster.arrive.release;\n\tbarrier.cluster.wait.acquire;" : : : "memory");
}

template <class L, int MODEL, class S>
__global__ void __launch_bounds__(resident_threads<L, S>())
k_resident(const KArgs a, const S* src, S* dst, const uint32_t* __restrict__ links,
           typename Store<S>::R* __restrict__ tau, uint32_t* __restrict__ rng_ctr, int parity,
           int nsteps) {
    using R = typename Store<S>::R;
    extern __shared__ __align__(16) unsigned char smem[];
    const KParams& kp = a.kp;
    const int T = (int)blockDim.x, t = (int)threadIdx.x;
    int idx = (int)blockIdx.x * T + t;
    const bool inside = idx < kp.ncells;
    const uint32_t lk = inside ? __ldg(links + idx) : kSolidBit;
    const bool active = !(lk & kSolidBit);
    step_begin(idx);
    // element (i, n) of a block's buffer, as in a population buffer of T cells
    auto elem = [&](int i, int n) { return (int)pop_base<S>(i, T) + pop_step<S>(i) * n; };
    S* const buf = reinterpret_cast<S*>(smem);
    const int half = L::Q * T;               // elements of one of the two buffers
    if (inside) {
        // both buffers: a solid or ghost cell is never stepped, but may be read
        static_for<0, L::Q>([&](auto I) {
            constexpr int i = decltype(I)::value;
            const S v = src[pop_base<S>(i, kp.plane) + (int64_t)pop_step<S>(i) * idx];
            buf[elem(i, t)] = v;
            buf[half + elem(i, t)] = v;
        });
    }
    uint32_t from[L::Q];                     // shared::cluster address of each population's source
    {
        const uint32_t base = (uint32_t)__cvta_generic_to_shared(smem);
        PullOffsets o{0, 0, 0, 0, 0, 0};
        if (active) o = pull_offsets(kp, idx);
        static_for<0, L::Q>([&](auto I) {
            constexpr int i = decltype(I)::value;
            const bool wall = (lk >> i) & 1u;
            const int n = active && !wall ? idx + o.template of<L, i>() : inside ? idx : 0;
            const int b = n / T;
            const uint32_t own = base + (uint32_t)(elem(wall ? L::opp(i) : i, n - b * T) * (int)sizeof(S));
            asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(from[i]) : "r"(own), "r"(b));
        });
    }
    uint32_t seed = 0u;
    if constexpr (Store<S>::kStochastic) seed = rng_ctr[parity];
    R tc = R(0);
    if constexpr (MODEL != LBM_MODEL_IR)
        if (active) tc = tau[idx];
    cluster_barrier();
    uint32_t rd = 0u;                        // byte offset of the buffer this step reads
    const uint32_t bytes = (uint32_t)half * (uint32_t)sizeof(S);
    for (int k = 0; k < nsteps; ++k) {
        if (active) {
            R f[L::Q];
            static_for<0, L::Q>([&](auto I) {
                constexpr int i = decltype(I)::value;
                f[i] = ld_cluster<S>(from[i] + rd);
            });
            R drho, ur[3];
            if constexpr (MODEL != LBM_MODEL_IR) {
                collide_pr<L, S, false>(coef<R>(a), kp.flags, f, tc, drho, ur);
            } else if constexpr (pair_form<S>()) {
                collide_ir<L, S>(coef<R>(a), kp.flags, f, drho, ur);
            } else {
                // behind a branch of its own, as in k_step: merged with the
                // gather the compiler contracts the class sums differently
                int go = 1;
                asm volatile("" : "+r"(go));
                if (go) collide_ir<L, S>(coef<R>(a), kp.flags, f, drho, ur);
            }
            uint32_t rnd = 0u;
            if constexpr (Store<S>::kStochastic)
                rnd = pcg_hash(((uint32_t)idx + kp.hash_offset) ^ ((seed + (uint32_t)k) * 0x9e3779b9u));
            store_cell<L, S>(DstStride<S>{reinterpret_cast<S*>(smem + (bytes - rd)), T}, t, f, rnd);
        }
        rd = bytes - rd;
        cluster_barrier();
    }
    if (active) {
        const S* last = reinterpret_cast<const S*>(smem + rd);
        static_for<0, L::Q>([&](auto I) {
            constexpr int i = decltype(I)::value;
            dst[pop_base<S>(i, kp.plane) + (int64_t)pop_step<S>(i) * idx] = last[elem(i, t)];
        });
        if constexpr (MODEL != LBM_MODEL_IR) tau[idx] = tc;
    }
    if constexpr (Store<S>::kStochastic)
        // as after nsteps launches: the counter of the buffer now current
        if (blockIdx.x == 0 && t == 0) rng_ctr[parity ^ (nsteps & 1)] = seed + (uint32_t)nsteps;
}

// The FP64 run of a domain small enough to have a cluster's sub-partitions to
// spare, its collision divided (see k_step_split): blocks of T cells, T parts<L>()
// threads, warp w working on part w % parts of the 32 cells w / parts.
template <class L> struct SplitRun {
    static constexpr int np = parts<L>();
    static constexpr int most_cells = 128 / np;            // of a block: a warp per sub-partition
    static constexpr size_t bytes(int T) {
        return sizeof(double) * 2 * L::Q * (size_t)T + sizeof(SplitShared) * (size_t)(T / 32);
    }
};
template <class L, int MODEL>
__global__ void __launch_bounds__(128)
k_resident_split(const KArgs a, const double* src, double* dst, const uint32_t* __restrict__ links,
                 double* __restrict__ tau, int nsteps) {
    extern __shared__ __align__(16) unsigned char smem[];
    const KParams& kp = a.kp;
    constexpr int np = parts<L>();
    const int T = (int)blockDim.x / np;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int part = warp % np, t = (warp / np) * 32 + lane;
    int idx = (int)blockIdx.x * T + t;
    const bool inside = idx < kp.ncells;
    const uint32_t lk = inside ? __ldg(links + idx) : kSolidBit;
    const bool on = !(lk & kSolidBit);
    step_begin(idx);
    double* const buf = reinterpret_cast<double*>(smem);
    const int half = L::Q * T;
    SplitShared& sh = reinterpret_cast<SplitShared*>(smem + sizeof(double) * 2 * half)[warp / np];
    uint32_t from[8];
    const uint32_t base = (uint32_t)__cvta_generic_to_shared(smem);
    by_part<L>(part, [&](auto P) {
        constexpr int PART = decltype(P)::value;
        auto load = [&](int i) {   // both buffers, as k_resident
            if (!inside) return;
            const double v = src[(int64_t)i * kp.plane + idx];
            buf[i * T + t] = v;
            buf[half + i * T + t] = v;
        };
        if constexpr (PART == 0) load(0);
        PullOffsets o{0, 0, 0, 0, 0, 0};
        if (on) o = pull_offsets(kp, idx);
        part_pops<L, PART>([&](auto I, auto K) {
            constexpr int i = decltype(I)::value;
            load(i);
            const bool wall = (lk >> i) & 1u;
            const int n = on && !wall ? idx + o.template of<L, i>() : inside ? idx : 0;
            const int b = n / T;
            const uint32_t own = base + (uint32_t)(((wall ? L::opp(i) : i) * T + n - b * T) * (int)sizeof(double));
            asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(from[decltype(K)::value]) : "r"(own), "r"(b));
        });
    });
    double tc = 0.0;
    if constexpr (MODEL != LBM_MODEL_IR)
        if (on) tc = tau[idx];
    cluster_barrier();
    uint32_t rd = 0u;                        // byte offset of the buffer this step reads
    const uint32_t bytes = (uint32_t)half * (uint32_t)sizeof(double);
    for (int k = 0; k < nsteps; ++k) {
        double r[8], f0 = 0.0;
        if (on) {
            const double* in = reinterpret_cast<const double*>(smem + rd);
            by_part<L>(part, [&](auto P) {
                constexpr int PART = decltype(P)::value;
                if constexpr (PART == 0) f0 = in[t];
                part_pops<L, PART>([&](auto, auto K) {
                    constexpr int j = decltype(K)::value;
                    r[j] = ld_cluster<double>(from[j] + rd);
                });
            });
        }
        split_collide<L, MODEL>(a.cd, kp.flags, part, lane, on, sh, r, f0, tc);
        if (on) {
            double* out = reinterpret_cast<double*>(smem + (bytes - rd));
            by_part<L>(part, [&](auto P) {
                constexpr int PART = decltype(P)::value;
                if constexpr (PART == 0) out[t] = f0;
                part_pops<L, PART>([&](auto I, auto K) {
                    out[decltype(I)::value * T + t] = r[decltype(K)::value];
                });
            });
        }
        rd = bytes - rd;
        cluster_barrier();
    }
    if (on) {
        const double* last = reinterpret_cast<const double*>(smem + rd);
        by_part<L>(part, [&](auto P) {
            constexpr int PART = decltype(P)::value;
            if constexpr (PART == 0) {
                dst[idx] = last[t];
                if constexpr (MODEL != LBM_MODEL_IR) tau[idx] = tc;
            }
            part_pops<L, PART>([&](auto I, auto) {
                constexpr int i = decltype(I)::value;
                dst[(int64_t)i * kp.plane + idx] = last[i * T + t];
            });
        });
    }
}

// ---------------------------------------------------------------------------
// Compact layout (LBM_FLAG_COMPACT).  The population planes, the link words,
// tau and the check-step snapshot hold the stepped fluid cells only: slot k is
// the k-th fluid cell in cell-index order, cellidx[k] its cell index, and
// rank[n] the slot of cell n (negative for a solid cell).  One thread per slot, so
// every lane of a warp is a fluid cell and every store fills whole sectors,
// whereas on a porous medium the dense layout also moves the solid cells that
// share a DRAM access with fluid ones.  The pull reads population i of the
// cell at x - c_i from slot rank[x - c_i] (a solid source: the cell's own
// opposite population, as in the dense layout); the rank words a warp reads
// lie in a few rows and mostly come from L1.  Per cell the arithmetic is the
// dense step's (the same collision code, the same stochastic-rounding hash of
// the cell index); compiled into another kernel, it may differ from it by the
// compiler's multiply-add contraction, i.e. to round-off.
//
// rank[] is a running count: a fluid cell holds its slot, a solid cell ~n with
// n the number of fluid cells before it.  Slots are in cell order, so along a
// row the slots of the neighbours x - 1 and x + 1 follow from the word of the
// cell between them (one less; one more if that cell is fluid), and a gather
// reads one word per neighbouring row, 8 (D3Q15, D3Q19, D3Q27) instead of 14,
// 18 and 26.  The wrap in x is the exception: a warp that holds a cell at
// either end of a row looks every neighbour up.
//
// ROWS = false leaves the row paths out: beside them the compiler contracts some
// class sums differently, and results would move by a rounding.  So the 16-bit
// forms look every neighbour up, in a step and in a read-back alike.
template <class L> __host__ __device__ constexpr int dir_index(int cx, int cy, int cz) {
    for (int i = 0; i < L::Q; ++i)
        if (L::cx(i) == cx && L::cy(i) == cy && L::cz(i) == cz) return i;
    return -1;
}
template <class L, class S, bool ROWS = sizeof(S) != 2, class Src>
__device__ __forceinline__ void gather_compact(const KParams& kp, const Src& P, uint32_t lk,
                                               int idx, int slot, const int* __restrict__ rank,
                                               typename Store<S>::R (&v)[L::Q]) {
    const PullOffsets o = pull_offsets(kp, idx);
    // the cell's own rank word: each neighbour's is one multiply-add from it
    // (against an add and a sign-extended 64-bit address per neighbour: 2-8 %
    // faster steps on 256^3 porous boxes)
    const int* __restrict__ rk = rank + idx;
    v[0] = Store<S>::template ld<L, 0>(P.template at<0>(slot));
    if constexpr (ROWS) {
        // by rows (cy, cz): f(direction, slot of its source if that is fluid)
        auto rows = [&](bool solid_free, auto&& f) {
            static_for<0, 9>([&](auto J) {
                constexpr int cy = decltype(J)::value % 3 - 1, cz = decltype(J)::value / 3 - 1;
                constexpr int im = dir_index<L>(1, cy, cz), i0 = dir_index<L>(0, cy, cz),
                              ip = dir_index<L>(-1, cy, cz);
                if constexpr (im >= 0 || i0 >= 0 || ip >= 0) {
                    int c = slot, after = slot + 1;
                    if constexpr (cy != 0 || cz != 0) {
                        int off = 0;
                        if constexpr (cy > 0) off += o.dym;
                        if constexpr (cy < 0) off += o.dyp;
                        if constexpr (cz > 0) off += o.dzm;
                        if constexpr (cz < 0) off += o.dzp;
                        c = __ldg(rk + off);
                        if (i0 >= 0 && solid_free) {     // the row's own cell is a source, hence fluid
                            after = c + 1;
                        } else {
                            const int s = c >> 31;       // -1 for a solid cell
                            c ^= s;
                            after = c + 1 + s;
                        }
                    }
                    if constexpr (im >= 0) f(std::integral_constant<int, im>{}, c - 1);
                    if constexpr (i0 > 0) f(std::integral_constant<int, i0>{}, c);
                    if constexpr (ip >= 0) f(std::integral_constant<int, ip>{}, after);
                }
            });
        };
        const bool edge = o.dxm != -1 || o.dxp != 1;   // the x neighbours wrap
        const unsigned warp = __activemask();
        if (__all_sync(warp, lk == 0u && !edge)) {
            rows(true, [&](auto I, int k) {
                constexpr int i = decltype(I)::value;
                v[i] = Store<S>::template ld<L, i>(P.template at<i>(k));
            });
        } else if (__all_sync(warp, !edge)) {
            rows(false, [&](auto I, int k) {
                constexpr int i = decltype(I)::value;
                const S* p = ((lk >> i) & 1u) ? P.template at<L::opp(i)>(slot) : P.template at<i>(k);
                v[i] = Store<S>::template ld<L, i>(p);   // opposite planes share w_i
            });
        } else {
            static_for<1, L::Q>([&](auto I) {
                constexpr int i = decltype(I)::value;
                const S* p;
                if ((lk >> i) & 1u)
                    p = P.template at<L::opp(i)>(slot);
                else
                    p = P.template at<i>(__ldg(rk + o.template of<L, i>()));
                v[i] = Store<S>::template ld<L, i>(p);
            });
        }
    } else {
        if (__all_sync(__activemask(), lk == 0u)) {
            static_for<1, L::Q>([&](auto I) {
                constexpr int i = decltype(I)::value;
                const int k = __ldg(rk + o.template of<L, i>());
                v[i] = Store<S>::template ld<L, i>(P.template at<i>(k));
            });
        } else {
            static_for<1, L::Q>([&](auto I) {
                constexpr int i = decltype(I)::value;
                const S* p;
                if ((lk >> i) & 1u)
                    p = P.template at<L::opp(i)>(slot);
                else
                    p = P.template at<i>(__ldg(rk + o.template of<L, i>()));
                v[i] = Store<S>::template ld<L, i>(p);
            });
        }
    }
}

// One fluid cell of one time step in the compact layout (as cell_step).
template <class L, int MODEL, class S, bool CHECK, class Src, class Dst>
__device__ __forceinline__ void compact_cell(const KParams& kp, const Coef<typename Store<S>::R>& c,
                                             const Src& src, const Dst& dst, uint32_t lk, int idx,
                                             int slot, const int* __restrict__ rank,
                                             typename Store<S>::R* __restrict__ tau,
                                             typename Store<S>::R* __restrict__ usnap, uint32_t rnd,
                                             typename Store<S>::R (&acc)[kNumStats]) {
    using R = typename Store<S>::R;
    R up[3] = {R(0), R(0), R(0)};
    if constexpr (CHECK) {
#pragma unroll
        for (int d = 0; d < 3; ++d) up[d] = usnap[(int64_t)d * kp.plane + slot];
    }
    R f[L::Q];
    // so does the D3Q27 FP32 IR step (160^3 porous box: 124 us, 118 with the row paths)
    constexpr bool rows = sizeof(S) != 2 && !(sizeof(S) == 4 && L::Q == 27 && MODEL == LBM_MODEL_IR);
    gather_compact<L, S, rows>(kp, src, lk, idx, slot, rank, f);
    R drho, ur[3];
    if constexpr (MODEL != LBM_MODEL_IR) {
        R t = tau[slot];
        collide_pr<L, S, MODEL == kModelPRImplicit>(c, kp.flags, f, t, drho, ur);
        tau[slot] = t;
    } else {
        collide_ir<L, S>(c, kp.flags, f, drho, ur);
    }
    store_cell<L, S>(dst, slot, f, rnd);
    if constexpr (CHECK) check_stats(ur, up, drho, usnap, kp.plane, slot, acc);
}

// Register budget of the compact step: the dense step's (BLBM_COMPACT_MINB
// overrides it at build time for the FP32-arithmetic forms).
#ifndef BLBM_COMPACT_MINB
#define BLBM_COMPACT_MINB -1
#endif
template <class L, int MODEL, class S, bool CHECK> constexpr int compact_min_blocks() {
    if (std::is_same<typename Store<S>::R, double>::value) return 0;
    if (BLBM_COMPACT_MINB >= 0) return BLBM_COMPACT_MINB;
    // IR up to 19 velocities: 6 blocks of 256 (40 registers): on the 256^3
    // porous box, D3Q19, 378 -> 361 us (FP32) and 318 -> 302 us (FP16) against
    // the allocator's 38 registers.  D3Q27 IR: 4 blocks (64 registers; 48
    // spilled and ran slower).  PR keeps the dense step's budget (6 blocks
    // spilled and made the D3Q19 FP16 step 7 % slower).
    if (MODEL == LBM_MODEL_IR && !CHECK) return L::Q <= 19 ? 6 : 4;
    return step_min_blocks<L, MODEL, S, CHECK, kBlock>();
}

// Threads per block of the plain compact step (check steps: kBlock).  A
// block's rank words come from the rows next to its cells, so a wider block
// reuses more of them from L1; the register budget per SM stays the same.
// 256^3 porous box, D3Q19: IR (FP32) 373 / 361 / 349 us at 128 / 256 / 512
// threads; PR, whose budget at 512 threads loses occupancy, 400 / 405 / 500
// (FP32) and 331 / 338 / 406 (FP16).  D3Q27 IR, whose 64 registers allow
// only two blocks of 512 per SM: 581 us at 512 threads, 512 us at 256 (256^3
// box, porosity 0.7).  BLBM_COMPACT_BLOCK overrides it.
#ifndef BLBM_COMPACT_BLOCK
#define BLBM_COMPACT_BLOCK 0
#endif
template <class L, int MODEL> constexpr int compact_block() {
    if (BLBM_COMPACT_BLOCK > 0) return BLBM_COMPACT_BLOCK;
    if (MODEL != LBM_MODEL_IR) return 128;
    return L::Q <= 19 ? 512 : 256;
}

template <class L, int MODEL, class S, bool CHECK, int BLOCK = kBlock>
__global__ void __launch_bounds__(BLOCK, compact_min_blocks<L, MODEL, S, CHECK>() * kBlock / BLOCK)
k_step_compact(const KArgs a, const SrcPlanes<S> src, const DstPlanes<S> dst,
               const uint32_t* __restrict__ links, const int* __restrict__ cellidx,
               const int* __restrict__ rank, typename Store<S>::R* __restrict__ tau,
               typename Store<S>::R* __restrict__ usnap, double* __restrict__ partials,
               uint32_t* __restrict__ rng_ctr, int parity) {
    static_assert(!CHECK || BLOCK == kBlock, "check steps use the fixed block size");
    using R = typename Store<S>::R;
    const KParams& kp = a.kp;
    int slot = blockIdx.x * BLOCK + threadIdx.x;
    int idx = 0;
    uint32_t lk = 0u, seed = 0u;
    if constexpr (!Store<S>::kStochastic) {
        if (slot < kp.nslots) {
            idx = __ldg(cellidx + slot);
            lk = __ldg(links + slot);
        }
        step_begin(slot);
    } else {
        // this launch reads counter[parity] and leaves counter + 1 for the next
        seed = rng_ctr[parity];
        if (blockIdx.x == 0 && threadIdx.x == 0) rng_ctr[parity ^ 1] = seed + 1u;
    }
    R acc[kNumStats];
    if constexpr (CHECK) {
#pragma unroll
        for (int k = 0; k < kNumStats; ++k) acc[k] = R(0);
    }
    if (slot < kp.nslots) {
        uint32_t rnd = 0u;
        if constexpr (Store<S>::kStochastic) {
            idx = __ldg(cellidx + slot);
            lk = __ldg(links + slot);
            rnd = pcg_hash(((uint32_t)idx + kp.hash_offset) ^ (seed * 0x9e3779b9u));
        }
        compact_cell<L, MODEL, S, CHECK>(kp, coef<R>(a), src, dst, lk, idx, slot, rank, tau, usnap,
                                         rnd, acc);
    }
    if constexpr (CHECK) block_sum_store(acc, partials + (int64_t)blockIdx.x * kNumStats);
}

// Plain compact step over a persistent grid: each thread walks the slots
// slot, slot + stride, ... and loads the next slot's cell index and link word
// before it steps the current one, so of the three dependent loads of a slot
// (cell index, neighbour slots, populations) only the last two are on the
// critical path.  It pays for the IR step of the 16-bit forms (256^3 porous
// box, D3Q19 FP16: 306 -> 268 us).  The FP32 forms need more registers for it
// than their budgets hold (D3Q19 IR, 256^3 porous box: 323 us by one-slot
// threads, 349-386 by the loop); 16-bit PR gained nothing.
template <int MODEL, class S> constexpr bool compact_loop() {
    return MODEL == LBM_MODEL_IR && sizeof(S) == 2;
}
// (BLBM_COMPACT_LOOP_MINB overrides its register budget at build time.)
#ifndef BLBM_COMPACT_LOOP_MINB
#define BLBM_COMPACT_LOOP_MINB -1
#endif
// D3Q27: 4 blocks (64 registers; at 5 blocks it spills 68 bytes).
template <class L, int MODEL, class S> constexpr int compact_loop_min_blocks() {
    if (BLBM_COMPACT_LOOP_MINB >= 0) return BLBM_COMPACT_LOOP_MINB;
    if (L::Q == 27) return 4;
    return compact_min_blocks<L, MODEL, S, false>();
}

template <class L, int MODEL, class S>
__global__ void __launch_bounds__(kBlock, compact_loop_min_blocks<L, MODEL, S>())
k_step_compact_loop(const KArgs a, const SrcPlanes<S> src, const DstPlanes<S> dst,
                    const uint32_t* __restrict__ links, const int* __restrict__ cellidx,
                    const int* __restrict__ rank, typename Store<S>::R* __restrict__ tau,
                    uint32_t* __restrict__ rng_ctr, int parity) {
    using R = typename Store<S>::R;
    const KParams& kp = a.kp;
    const int n = kp.nslots, stride = gridDim.x * kBlock;
    int slot = blockIdx.x * kBlock + threadIdx.x;
    uint32_t seed = 0u;
    if constexpr (Store<S>::kStochastic) {
        // this launch reads counter[parity] and leaves counter + 1 for the next
        seed = rng_ctr[parity];
        if (blockIdx.x == 0 && threadIdx.x == 0) rng_ctr[parity ^ 1] = seed + 1u;
    }
    int idx = 0;
    uint32_t lk = 0u;
    if (slot < n) {
        idx = __ldg(cellidx + slot);
        lk = __ldg(links + slot);
    }
    R acc[kNumStats];
    for (; slot < n; slot += stride) {
        const int next = slot + stride;
        int nidx = 0;
        uint32_t nlk = 0u;
        if (next < n) {
            nidx = __ldg(cellidx + next);
            nlk = __ldg(links + next);
        }
        uint32_t rnd = 0u;
        if constexpr (Store<S>::kStochastic)
            rnd = pcg_hash(((uint32_t)idx + kp.hash_offset) ^ (seed * 0x9e3779b9u));
        compact_cell<L, MODEL, S, false>(kp, coef<R>(a), src, dst, lk, idx, slot, rank, tau,
                                         nullptr, rnd, acc);
        idx = nidx;
        lk = nlk;
    }
}

// link words of the compact layout: slot k gets the bits of cell cellidx[k]
template <class L>
__global__ void __launch_bounds__(kBlock)
k_links_compact(const KParams kp, const uint8_t* __restrict__ mask,
                const int* __restrict__ cellidx, uint32_t* __restrict__ links) {
    const int slot = blockIdx.x * kBlock + threadIdx.x;
    if (slot >= kp.nslots) return;
    const int nx = kp.nx, ny = kp.ny, nz = kp.nz;
    int x, y, z;
    cell_xyz(kp, cellidx[slot], x, y, z);
    uint32_t bits = 0;
#pragma unroll
    for (int i = 0; i < L::Q; ++i) {
        const int xs = (x - L::cx(i) + nx) % nx;
        const int ys = (y - L::cy(i) + ny) % ny;
        const int zs = (z - L::cz(i) + nz) % nz;
        if (mask[xs + nx * (ys + ny * zs)]) bits |= 1u << i;
    }
    links[slot] = bits;
}

// ---------------------------------------------------------------------------
// Batched step: all resident domains of one (lattice, model, storage) in one
// launch.  Block b works on domain block_dom[b]; each domain's blocks are
// contiguous from desc.block_begin.  The current buffer of a domain is
// phase ^ desc.parity0, so a captured graph that alternates the phase stays
// valid for every domain.
struct BatchDesc {
    KParams kp;
    Coef<float> cf;
    Coef<double> cd;
    void* f[2];
    const uint32_t* links;
    void* tau;
    void* usnap;
    uint32_t* rng;      // two launch counters (16-bit storage)
    int parity0;
    int block_begin;    // first 256-cell tile of this domain (check steps)
    int nblocks;        // its 256-cell tiles
    int slot;           // row of this domain in the batch's per-domain stats
    int pblock_begin;   // first tile of this domain in the plain-step tile map
};

template <class R> __device__ __forceinline__ const Coef<R>& bcoef(const BatchDesc& d);
template <> __device__ __forceinline__ const Coef<float>& bcoef<float>(const BatchDesc& d) { return d.cf; }
template <> __device__ __forceinline__ const Coef<double>& bcoef<double>(const BatchDesc& d) { return d.cd; }

// One check step of one tile (kBlock consecutive cells of one domain): as
// k_step's check step, with the copy-through for every form (the solid cells
// of a group with fluid cells copy their populations through).
template <class L, int MODEL, class S>
__device__ __forceinline__ void batch_tile_check(const BatchDesc& D, int tile, int phase,
                                                 double* __restrict__ partials) {
    using R = typename Store<S>::R;
    const KParams& kp = D.kp;
    const int lb = tile - D.block_begin;
    const int idx = lb * kBlock + threadIdx.x;
    const int cur = phase ^ D.parity0;
    const SrcStride<S> src{(const S*)D.f[cur], (int)kp.plane};
    const DstStride<S> dst{(S*)D.f[cur ^ 1], (int)kp.plane};
    const bool inside = idx < kp.ncells;
    uint32_t rnd = 0u;
    if constexpr (Store<S>::kStochastic) {
        // reads counter[cur], leaves counter + 1 in the other slot for the next launch
        const uint32_t seed = D.rng[cur];
        if (lb == 0 && threadIdx.x == 0) D.rng[cur ^ 1] = seed + 1u;
        rnd = pcg_hash(((uint32_t)idx + kp.hash_offset) ^ (seed * 0x9e3779b9u));
    }
    const uint32_t lk = inside ? __ldg(D.links + idx) : kSolidBit;
    const bool active = !(lk & kSolidBit);
    const bool group_fluid = group_has_fluid(active, idx);
    R acc[kNumStats];
#pragma unroll
    for (int k = 0; k < kNumStats; ++k) acc[k] = R(0);
    if (group_fluid && inside)
        cell_step<L, MODEL, S, true>(kp, bcoef<R>(D), src, dst, lk, idx, (R*)D.tau, (R*)D.usnap,
                                     rnd, acc, active);
    block_sum_store(acc, partials + (int64_t)tile * kNumStats);
}

// One plain step of one tile of T x C cells of one domain (the tile shape the
// batch schedule sets per group): thread t steps cells base + t, base + t + T,
// ... (C of them, one after the other), so every warp access stays
// contiguous.  Per cell as k_step, with the copy-through for every form.
template <class L, int MODEL, class S, int T, int C>
__device__ __forceinline__ void batch_tile_plain(const BatchDesc& D, int tile, int phase) {
    using R = typename Store<S>::R;
    const KParams& kp = D.kp;
    const int lb = tile - D.pblock_begin;
    const int cur = phase ^ D.parity0;
    const SrcStride<S> src{(const S*)D.f[cur], (int)kp.plane};
    const DstStride<S> dst{(S*)D.f[cur ^ 1], (int)kp.plane};
    uint32_t seed = 0u;
    if constexpr (Store<S>::kStochastic) {
        // reads counter[cur], leaves counter + 1 in the other slot for the next launch
        seed = D.rng[cur];
        if (lb == 0 && threadIdx.x == 0) D.rng[cur ^ 1] = seed + 1u;
    }
#pragma unroll 1
    for (int c = 0; c < C; ++c) {
        const int idx = (lb * C + c) * T + (int)threadIdx.x;
        const bool inside = idx < kp.ncells;
        uint32_t rnd = 0u;
        if constexpr (Store<S>::kStochastic) rnd = pcg_hash(((uint32_t)idx + kp.hash_offset) ^ (seed * 0x9e3779b9u));
        const uint32_t lk = inside ? __ldg(D.links + idx) : kSolidBit;
        const bool active = !(lk & kSolidBit);
        const bool group_fluid = group_has_fluid(active, idx);
        R acc[kNumStats];
        if (group_fluid && inside)
            cell_step<L, MODEL, S, false>(kp, bcoef<R>(D), src, dst, lk, idx, (R*)D.tau,
                                          (R*)D.usnap, rnd, acc, active);
    }
}

// Batch steps: the CTAs walk the tiles of every domain of the group (tile t,
// t + gridDim.x, ...).  With one CTA per tile this is the plain launch; with
// fewer CTAs it is a persistent grid.  Check-step partials are indexed by
// 256-cell tile, so check steps reduce in the same order for every grid size
// and every plain-step tile shape.
// Register budget of the batch kernels, as resident 256-thread blocks (scaled
// to the tile's threads): plain PR steps in FP32 arithmetic keep 4 (64
// registers).  Without it the 16-bit forms take 72 registers and FP32
// storage 70 (the descriptor's coefficients are loaded, not kernel-parameter
// operands), leaving 3 blocks; on a single D3Q27 duct the FP32 PR batch step
// measured 170 us without and 154 us with the budget.  Plain IR steps of the
// 16-bit forms keep 5 (48 registers; their copy-through path takes 58 and 4
// blocks otherwise).  FP32 IR, check steps and FP64 are left to the
// allocator.  BLBM_BATCH_PR_MINB (16-bit PR), BLBM_BATCH_PR32_MINB (FP32 PR)
// and BLBM_BATCH_IR16_MINB override at build time.
#ifndef BLBM_BATCH_PR_MINB
#define BLBM_BATCH_PR_MINB 4
#endif
#ifndef BLBM_BATCH_PR32_MINB
#define BLBM_BATCH_PR32_MINB 4
#endif
#ifndef BLBM_BATCH_IR16_MINB
#define BLBM_BATCH_IR16_MINB 5
#endif
template <int MODEL, class S, bool CHECK> constexpr int batch_min_blocks() {
    return CHECK ? 0
         : MODEL == LBM_MODEL_IR ? (sizeof(S) == 2 ? BLBM_BATCH_IR16_MINB : 0)
         : sizeof(S) == 2 ? BLBM_BATCH_PR_MINB
         : sizeof(S) == 4 ? BLBM_BATCH_PR32_MINB : 0;
}

// Both batch kernels read nothing in front of step_begin(): a tile's map entry,
// descriptor and first link word read there cost the rest of the tile more than
// the wait hides (16 D2Q9 domains of 256^2 cells, PR: FP16 18.7 -> 21.6 us, FP32 18.7 ->
// 20.5; D3Q27 FP32 IR 16^3: 4.5 -> 5.1).
template <class L, int MODEL, class S>
__global__ void __launch_bounds__(kBlock)
k_step_batch_check(const BatchDesc* __restrict__ descs, const int* __restrict__ block_dom,
                   int ntiles, int phase, double* __restrict__ partials) {
    int first = blockIdx.x;
    step_begin(first);
    for (int t = first; t < ntiles; t += gridDim.x) {
        batch_tile_check<L, MODEL, S>(descs[block_dom[t]], t, phase, partials);
        __syncthreads();   // block_sum_store's shared rows are reused
    }
}

template <class L, int MODEL, class S, int T, int C>
__global__ void __launch_bounds__(T, batch_min_blocks<MODEL, S, false>() * kBlock / T)
k_step_batch(const BatchDesc* __restrict__ descs, const int* __restrict__ tile_dom, int ntiles,
             int phase) {
    int first = blockIdx.x;
    step_begin(first);
    for (int t = first; t < ntiles; t += gridDim.x)
        batch_tile_plain<L, MODEL, S, T, C>(descs[tile_dom[t]], t, phase);
}

// density and velocity u = (j + F/2) / rho of gathered populations
template <class L, class S>
__device__ __forceinline__ void fields_of(const KArgs& a, typename Store<S>::R (&v)[L::Q],
                                          double& r, double (&u)[3]) {
    using R = typename Store<S>::R;
    const Mom<R> m = moments<L, S>(v);
    const Coef<R>& c = coef<R>(a);
    const R rr = R(1) + m.d;
    const R inv = R(1) / rr;
    r = (double)rr;
    u[0] = (double)((m.jx + R(0.5) * rr * c.g[0]) * inv);
    u[1] = (double)((m.jy + R(0.5) * rr * c.g[1]) * inv);
    if constexpr (L::D == 3) u[2] = (double)((m.jz + R(0.5) * rr * c.g[2]) * inv);
}

// macroscopic fields of the streamed populations (solid cells: 0)
template <class L, class S>
__global__ void __launch_bounds__(kBlock)
k_fields(const KArgs a, const SrcPlanes<S> f, const uint32_t* __restrict__ links,
         double* __restrict__ rho, double* __restrict__ ux, double* __restrict__ uy,
         double* __restrict__ uz) {
    using R = typename Store<S>::R;
    const KParams& kp = a.kp;
    const int idx = blockIdx.x * kBlock + threadIdx.x;
    if (idx >= kp.ncells) return;
    const uint32_t lk = links[idx];
    double r = 0.0, u[3] = {0.0, 0.0, 0.0};
    if (!(lk & kSolidBit)) {
        R v[L::Q];
        gather<L, S>(kp, f, lk, idx, v);
        fields_of<L, S>(a, v, r, u);
    }
    if (rho) rho[idx] = r;
    if (ux) ux[idx] = u[0];
    if (uy) uy[idx] = u[1];
    if (uz) uz[idx] = u[2];
}

// the same from the compact layout, one thread per cell of the box
template <class L, class S>
__global__ void __launch_bounds__(kBlock)
k_fields_compact(const KArgs a, const SrcPlanes<S> f, const uint32_t* __restrict__ links,
                 const int* __restrict__ rank, double* __restrict__ rho, double* __restrict__ ux,
                 double* __restrict__ uy, double* __restrict__ uz) {
    using R = typename Store<S>::R;
    const KParams& kp = a.kp;
    const int idx = blockIdx.x * kBlock + threadIdx.x;
    if (idx >= kp.ncells) return;
    const int slot = rank[idx];
    double r = 0.0, u[3] = {0.0, 0.0, 0.0};
    if (slot >= 0) {
        R v[L::Q];
        gather_compact<L, S>(kp, f, links[slot], idx, slot, rank, v);
        fields_of<L, S>(a, v, r, u);
    }
    if (rho) rho[idx] = r;
    if (ux) ux[idx] = u[0];
    if (uy) uy[idx] = u[1];
    if (uz) uz[idx] = u[2];
}

// grid-stride reductions: flow sums of u_real (gathered) or state totals,
// over the cells of the box (dense layout) or the slots (COMPACT)
template <class L, class S, int MODE, bool COMPACT>
__global__ void __launch_bounds__(kBlock)
k_reduce(const KArgs a, const SrcPlanes<S> f, const uint32_t* __restrict__ links,
         const int* __restrict__ cellidx, const int* __restrict__ rank,
         double* __restrict__ partials) {
    using R = typename Store<S>::R;
    const KParams& kp = a.kp;
    double acc[kNumStats];
#pragma unroll
    for (int k = 0; k < kNumStats; ++k) acc[k] = 0.0;
    const int stride = gridDim.x * kBlock;
    const int n_end = COMPACT ? kp.nslots : kp.ncells;
    for (int n = blockIdx.x * kBlock + threadIdx.x; n < n_end; n += stride) {
        const uint32_t lk = links[n];
        if (!COMPACT && (lk & kSolidBit)) continue;
        R v[L::Q];
        if constexpr (MODE == kReduceFlow) {
            if constexpr (COMPACT)
                gather_compact<L, S>(kp, f, lk, cellidx[n], n, rank, v);
            else
                gather<L, S>(kp, f, lk, n, v);
        } else {
            static_for<0, L::Q>([&](auto I) {
                constexpr int i = decltype(I)::value;
                v[i] = Store<S>::template ld<L, i>(f.template at<i>(n));
            });
        }
        const Mom<R> m = moments<L, S>(v);
        if constexpr (MODE == kReduceFlow) {
            const Coef<R>& c = coef<R>(a);
            const R rr = R(1) + m.d;
            const R inv = R(1) / rr;
            acc[kStatUx] += (double)((m.jx + R(0.5) * rr * c.g[0]) * inv);
            acc[kStatUy] += (double)((m.jy + R(0.5) * rr * c.g[1]) * inv);
            if constexpr (L::D == 3) acc[kStatUz] += (double)((m.jz + R(0.5) * rr * c.g[2]) * inv);
            acc[kStatDrho] += (double)m.d;
        } else {
            acc[kTotMass] += (double)m.d;
            acc[kTotJx] += (double)m.jx;
            acc[kTotJy] += (double)m.jy;
            acc[kTotJz] += (double)m.jz;
        }
    }
    block_sum_store(acc, partials + (int64_t)blockIdx.x * kNumStats);
}

// solid / bounce-back link bits: bit i set if the cell at x - c_i is solid
// (With LBM_FLAG_Z_GHOSTS the first and last z-planes are ghost planes: they
// are never stepped, like solid cells, while their mask rows, the
// neighbouring slabs' own, still set the link bits of the planes next to them.)
template <class L>
__global__ void __launch_bounds__(kBlock)
k_links(const KParams kp, const uint8_t* __restrict__ mask, uint32_t* __restrict__ links) {
    const int idx = blockIdx.x * kBlock + threadIdx.x;
    if (idx >= kp.ncells) return;
    const int nx = kp.nx, ny = kp.ny, nz = kp.nz;
    int x, y, z;
    cell_xyz(kp, idx, x, y, z);
    const bool ghost = (kp.flags & LBM_FLAG_Z_GHOSTS) && (z == 0 || z == nz - 1);
    if (mask[idx] || ghost) {
        links[idx] = kSolidBit;
        return;
    }
    uint32_t bits = 0;
#pragma unroll
    for (int i = 0; i < L::Q; ++i) {
        const int xs = (x - L::cx(i) + nx) % nx;
        const int ys = (y - L::cy(i) + ny) % ny;
        const int zs = (z - L::cz(i) + nz) % nz;
        if (mask[xs + nx * (ys + ny * zs)]) bits |= 1u << i;
    }
    links[idx] = bits;
}

// FP64 full populations <-> stored offsets, one population plane at a time.
// Compact layout (rank != nullptr): the fluid cells' values move through
// their slots; solid cells are not stored and read back as the rest state w_q.
template <class L, class S>
__global__ void __launch_bounds__(kBlock)
k_convert(const KParams kp, int q, bool to_device, S* __restrict__ f, double* __restrict__ buf,
          const int* __restrict__ rank) {
    const int idx = blockIdx.x * kBlock + threadIdx.x;
    if (idx >= kp.ncells) return;
    double w = 0.0;
#pragma unroll
    for (int i = 0; i < L::Q; ++i)
        if (i == q) w = L::w(i);
    const int n = rank ? rank[idx] : idx;
    if (n < 0) {
        if (!to_device) buf[idx] = w;
        return;
    }
    S* p = f + pop_base<S>(q, kp.plane) + (int64_t)pop_step<S>(q) * n;
    if (to_device)
        *p = Store<S>::enc(buf[idx] - w, w);
    else
        buf[idx] = Store<S>::dec(*p, w) + w;
}

// Slab faces (LBM_FLAG_Z_GHOSTS).  The populations that cross a z-face are
// those with c_z = +1 (moving up) and c_z = -1 (moving down).  side 1 packs
// the last interior plane's c_z = +1 populations (the upper neighbour's lower
// ghost plane receives them: its side 0 unpack); side 0 packs the first
// interior plane's c_z = -1 populations (the lower neighbour's side 1
// unpack, into its upper ghost plane).  buf holds the stored values (no
// conversion), [j][cell of the plane] for the j-th crossing population in the
// lattice's order.
template <class L> __host__ __device__ constexpr int face_count() {
    int n = 0;
    for (int i = 0; i < L::Q; ++i) n += L::cz(i) == 1;
    return n;
}
template <class L> __device__ __forceinline__ int face_pop(int j, int cz) {
    int n = 0;
    for (int i = 0; i < L::Q; ++i)
        if (L::cz(i) == cz && n++ == j) return i;
    return -1;
}

template <class L, class S>
__global__ void __launch_bounds__(kBlock)
k_halo(const KParams kp, S* __restrict__ f, S* __restrict__ buf, int side, bool pack) {
    const int nxy = kp.nx * kp.ny;
    const int k = blockIdx.x * kBlock + threadIdx.x;
    if (k >= face_count<L>() * nxy) return;
    const int j = k / nxy, xy = k - j * nxy;
    // pack: interior plane next to the face, populations leaving through it;
    // unpack: ghost plane of the face, populations entering through it
    const int cz = (side == 1) == pack ? 1 : -1;
    const int z = pack ? (side == 1 ? kp.nz - 2 : 1) : (side == 1 ? kp.nz - 1 : 0);
    const int i = face_pop<L>(j, cz);
    S* p = f + pop_base<S>(i, kp.plane) + (int64_t)pop_step<S>(i) * ((int64_t)z * nxy + xy);
    if (pack)
        buf[k] = *p;
    else
        *p = buf[k];
}

// full FP64 populations of listed cells: out[i * n + k] = f_i(cells[k])
// (compact layout: a solid cell reads as the rest state w_i)
template <class L, class S>
__global__ void __launch_bounds__(kBlock)
k_gather_cells(const KParams kp, const S* __restrict__ f, const int64_t* __restrict__ cells,
               int n, double* __restrict__ out, const int* __restrict__ rank) {
    const int k = blockIdx.x * kBlock + threadIdx.x;
    if (k >= n) return;
    const int64_t c = rank ? (int64_t)rank[cells[k]] : cells[k];
    static_for<0, L::Q>([&](auto I) {
        constexpr int i = decltype(I)::value;
        out[(int64_t)i * n + k] =
            c < 0 ? L::w(i)
                  : Store<S>::dec(f[pop_base<S>(i, kp.plane) + (int64_t)pop_step<S>(i) * c], L::w(i)) + L::w(i);
    });
}

// ---------------------------------------------------------------------------
// host-side helpers for the per-lattice launchers
template <class L, class R> inline void fill_force_dirs(Coef<R>& c, const KParams& kp) {
    for (int p = 0; p < 13; ++p) {
        c.cg[p] = R(0);
        c.cgg[p] = R(0);
    }
    for (int p = 0; p < (L::Q - 1) / 2; ++p) {
        const int i = 2 * p + 1;
        const double cg = L::cx(i) * kp.g[0] + L::cy(i) * kp.g[1] + L::cz(i) * kp.g[2];
        c.cg[p] = (R)cg;
        c.cgg[p] = (R)(cg * cg);
    }
}

template <class R> inline Coef<R> make_coef(const KParams& kp) {
    Coef<R> c;
    const double nu = kp.nu_p;
    c.nu_p = (R)nu;
    c.sigma_y = (R)kp.sigma_y;
    c.m = (R)kp.m;
    c.gdot_c = (R)kp.gdot_c;
    c.inv_gc = (R)(1.0 / kp.gdot_c);
    c.e_c = (R)(kp.m * kp.gdot_c > 0.0 ? -expm1(-kp.m * kp.gdot_c) / kp.gdot_c : 0.0);
    c.magic = (R)kp.magic;
    for (int d = 0; d < 3; ++d) {
        c.g[d] = (R)kp.g[d];
        c.hg[d] = (R)(0.5 * kp.g[d]);
    }
    const double s2y = 1.4142135623730951 * kp.sigma_y;
    c.s2y = (R)s2y;
    c.ir_a = (R)(1.0 / (0.5 + 3.0 * nu));
    c.ir_b = (R)(1.0 / (1.0 + 6.0 * nu));
    c.six_nu = (R)(6.0 * nu);
    c.s2y2 = (R)(2.0 * kp.sigma_y * kp.sigma_y);
    c.ir_k = (R)(6.0 * nu / (1.0 + 6.0 * nu) - 0.5 / (0.5 + 3.0 * nu) - 1.0);
    c.ir_ks = (R)(s2y * (0.5 / (0.5 + 3.0 * nu) + 1.0 / (1.0 + 6.0 * nu)));
    c.ir_bn = (R)(6.0 * nu / (1.0 + 6.0 * nu));
    c.ir_bs = (R)(s2y / (1.0 + 6.0 * nu));
    c.newton = kp.newton;
    return c;
}

template <class L> inline KArgs make_args(const KParams& kp) {
    KArgs a;
    a.kp = kp;
    a.cf = make_coef<float>(kp);
    a.cd = make_coef<double>(kp);
    fill_force_dirs<L>(a.cf, kp);
    fill_force_dirs<L>(a.cd, kp);
    return a;
}

// Coefficients of a domain of lattice `lat` (host code without the lattice
// as a template parameter: the batch tables).
template <class R> inline Coef<R> make_coef_lat(const KParams& kp, int lat) {
    Coef<R> c = make_coef<R>(kp);
    switch (lat) {
    case LBM_D2Q9: fill_force_dirs<D2Q9>(c, kp); break;
    case LBM_D3Q15: fill_force_dirs<D3Q15>(c, kp); break;
    case LBM_D3Q19: fill_force_dirs<D3Q19>(c, kp); break;
    default: fill_force_dirs<D3Q27>(c, kp); break;
    }
    return c;
}

template <class L, class S> inline SrcPlanes<S> src_planes(const void* f, int64_t plane) {
    SrcPlanes<S> P{};
    for (int i = 0; i < L::Q; ++i) P.p[i] = (const S*)f + pop_base<S>(i, plane);
    return P;
}
template <class L, class S> inline DstPlanes<S> dst_planes(void* f, int64_t plane) {
    DstPlanes<S> P{};
    for (int i = 0; i < L::Q; ++i) P.p[i] = (S*)f + pop_base<S>(i, plane);
    return P;
}

// Lanes of one warp on every FP64 pipe (152 SMs of four sub-partitions): the
// most that divided steps fill (cells times parts).
constexpr int64_t kSplitLanes = 608 * 32;

// Launch of a step kernel; overlap: over the tail of the one before (it calls
// step_begin()).
template <class... K, class... A>
inline cudaError_t launch_kernel(bool overlap, void (*kernel)(K...), int grid, int block,
                                 cudaStream_t st, A&&... args) {
    cudaLaunchAttribute attr;
    attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr.val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3((unsigned)grid);
    cfg.blockDim = dim3((unsigned)block);
    cfg.stream = st;
    cfg.attrs = &attr;
    cfg.numAttrs = overlap ? 1 : 0;
    return cudaLaunchKernelEx(&cfg, kernel, std::forward<A>(args)...);
}
template <class... K, class... A>
inline cudaError_t launch_overlapped(void (*kernel)(K...), int grid, int block, cudaStream_t st,
                                     A&&... args) {
    return launch_kernel(true, kernel, grid, block, st, std::forward<A>(args)...);
}

// Launch of a solver's step kernel, overlapped where that pays.  The blocks of a
// launch over the tail of another share the SMs with it, so two grids that fit
// together overlap whole, and of a grid of a wave and more some blocks start early.
// In between, a grid that fits alone only would start in part, and in a second
// wave.  Steps of 0.05-2 waves on D2Q9 to D3Q27, FP32 and FP16, plain over overlapped
// us: 1.03-1.31 up to half a wave, 0.72-0.95 from there to 0.8, 1.04 from 0.9 on
// (D3Q15 FP32 PR, 48^3: 3.7 plain, 4.7 overlapped; 40^3: 3.2 and 2.8).  FP64 steps in
// blocks of 256, bound by the FP64 pipe of the SMs that hold two of the blocks, are
// launched plainly: the blocks that start early take the SMs the other grid leaves
// idle first, several to an SM (a step of 256^2 cells in two parts: 39.1 -> 32.8 us).
template <auto Kernel, class R, class... A>
inline cudaError_t launch_step(int grid, int block, cudaStream_t st, A&&... args) {
    struct Wave {
        int sms = 1, per_sm = 0;   // (unknown: overlapped)
    };
    static const Wave wave = [block] {   // per instantiation, which has one block size
        Wave w;
        int dev = 0;
        if (cudaGetDevice(&dev) != cudaSuccess ||
            cudaDeviceGetAttribute(&w.sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess ||
            cudaOccupancyMaxActiveBlocksPerMultiprocessor(&w.per_sm, Kernel, block, 0) != cudaSuccess) {
            cudaGetLastError();
            return Wave();
        }
        return w;
    }();
    const bool both = 2 * ((grid + wave.sms - 1) / wave.sms) <= wave.per_sm;
    const bool waves = 10 * (int64_t)grid >= 9 * (int64_t)wave.per_sm * wave.sms;
    const bool piled = sizeof(R) == 8 && block >= kBlock;
    return launch_kernel((both || waves) && !piled, Kernel, grid, block, st, std::forward<A>(args)...);
}

// Threads per block and blocks of a resident run of ncells cells, and whether
// the domain takes it (fits one cluster): small domains of FP32 arithmetic
// share one block, larger ones spread over the cluster's 16 (D2Q9 F32 IR, us a
// step: 256 cells in one block 0.55, 512 cells in one block 0.74, 640 cells in
// 10 blocks 0.58).  Steps launched one by one take 1.35-1.55.
template <class L, class S> inline bool resident_shape(int ncells, int& threads, int& blocks) {
    constexpr int most = resident_threads<L, S>();
    const int one = sizeof(typename Store<S>::R) == 8 ? 32 : L::Q == 9 ? 256 : 64;
    const int per = ncells <= one ? ncells : (ncells + kResidentCluster - 1) / kResidentCluster;
    threads = std::max((per + 31) / 32 * 32, sizeof(typename Store<S>::R) == 8 ? 32 : 64);
    blocks = (ncells + threads - 1) / threads;
    return threads <= most;
}

// Raises the kernel's limits (shared memory and blocks per cluster above the
// defaults) and asks whether the device can hold its largest cluster; once per
// instantiation and device (the limits belong to the device's copy).
template <class L, int MODEL, class S> bool resident_ready() {
    constexpr int kDevices = 64;
    static std::atomic<int> known[kDevices];   // 0: not asked, 1: yes, 2: no
    int dev = -1;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kDevices) return false;
    if (const int k = known[dev].load()) return k == 1;
    const bool ready = [] {
        auto kernel = k_resident<L, MODEL, S>;
        constexpr int threads = resident_threads<L, S>();
        constexpr int bytes = (int)sizeof(S) * 2 * L::Q * threads;
        cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
        if (e == cudaSuccess)
            e = cudaFuncSetAttribute(kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
        cudaLaunchAttribute attr;
        attr.id = cudaLaunchAttributeClusterDimension;
        attr.val.clusterDim.x = kResidentCluster;
        attr.val.clusterDim.y = 1;
        attr.val.clusterDim.z = 1;
        cudaLaunchConfig_t cfg{};
        cfg.gridDim = dim3(kResidentCluster);
        cfg.blockDim = dim3(threads);
        cfg.dynamicSmemBytes = bytes;
        cfg.attrs = &attr;
        cfg.numAttrs = 1;
        int clusters = 0;
        if (e == cudaSuccess) e = cudaOccupancyMaxActiveClusters(&clusters, kernel, &cfg);
        if constexpr (std::is_same<S, double>::value) {
            auto divided = k_resident_split<L, MODEL>;
            cfg.blockDim = dim3(128);
            cfg.dynamicSmemBytes = SplitRun<L>::bytes(SplitRun<L>::most_cells);
            int more = 0;
            if (e == cudaSuccess)
                e = cudaFuncSetAttribute(divided, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)cfg.dynamicSmemBytes);
            if (e == cudaSuccess)
                e = cudaFuncSetAttribute(divided, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
            if (e == cudaSuccess) e = cudaOccupancyMaxActiveClusters(&more, divided, &cfg);
            clusters = std::min(clusters, more);
        }
        if (e != cudaSuccess) cudaGetLastError();
        return e == cudaSuccess && clusters > 0;
    }();
    known[dev].store(ready ? 1 : 2);
    return ready;
}

template <class L, int MODEL, class S>
cudaError_t launch_resident_t(const KParams& kp, const StepArgs& s, int nsteps, cudaStream_t st) {
    using R = typename Store<S>::R;
    auto kernel = k_resident<L, MODEL, S>;
    int threads = 0, blocks = 0;
    if (!resident_shape<L, S>(kp.ncells, threads, blocks)) return cudaErrorNotSupported;
    const KArgs a = make_args<L>(kp);
    bool divided = false;
    if constexpr (std::is_same<S, double>::value) divided = threads <= SplitRun<L>::most_cells;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    attr[1].id = cudaLaunchAttributeClusterDimension;
    attr[1].val.clusterDim.x = (unsigned)blocks;
    attr[1].val.clusterDim.y = 1;
    attr[1].val.clusterDim.z = 1;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3((unsigned)blocks);
    cfg.blockDim = dim3((unsigned)threads);
    cfg.dynamicSmemBytes = sizeof(S) * 2 * L::Q * (size_t)threads;
    cfg.stream = st;
    cfg.attrs = attr;
    cfg.numAttrs = 2;
    if constexpr (std::is_same<S, double>::value) {
        if (divided) {
            cfg.blockDim = dim3((unsigned)(threads * parts<L>()));
            cfg.dynamicSmemBytes = SplitRun<L>::bytes(threads);
            return cudaLaunchKernelEx(&cfg, k_resident_split<L, MODEL>, a, (const double*)s.fsrc,
                                      (double*)s.fdst, s.links, (double*)s.tau, nsteps);
        }
    }
    return cudaLaunchKernelEx(&cfg, kernel, a, (const S*)s.fsrc, (S*)s.fdst, s.links, (R*)s.tau,
                              s.rng_ctr, s.parity, nsteps);
}

// Left out: the Newton-implicit step, and class sums that the compiler contracts
// differently here than in k_step: IR on D3Q15 and D3Q27, 16-bit PR on D3Q19 (every
// other form gives the same bits).
template <class L, class S> constexpr bool resident_pr() {
    return pair_form<S>() || sizeof(S) == 4 || L::Q != 19;
}
template <class L, class S> constexpr bool resident_ir() {
    return pair_form<S>() || L::Q == 9 || L::Q == 19;
}

template <class L, class S>
cudaError_t launch_resident_model(int model, const KParams& kp, const StepArgs& s, int nsteps,
                                  cudaStream_t st) {
    if constexpr (resident_pr<L, S>()) {
        if (model == LBM_MODEL_PR) return launch_resident_t<L, LBM_MODEL_PR, S>(kp, s, nsteps, st);
    }
    if constexpr (resident_ir<L, S>()) return launch_resident_t<L, LBM_MODEL_IR, S>(kp, s, nsteps, st);
    return cudaErrorNotSupported;
}

template <class L>
cudaError_t launch_resident_lat(int model, int storage, const KParams& kp, const StepArgs& s,
                                int nsteps, cudaStream_t st) {
    switch (storage) {
    case LBM_F32: return launch_resident_model<L, float>(model, kp, s, nsteps, st);
    case LBM_F64: return launch_resident_model<L, double>(model, kp, s, nsteps, st);
    case LBM_F16_OFS: return launch_resident_model<L, __half>(model, kp, s, nsteps, st);
    case LBM_BF16_OFS: return launch_resident_model<L, __nv_bfloat16>(model, kp, s, nsteps, st);
    default: return cudaErrorNotSupported;
    }
}

template <class L, class S> bool resident_fits_model(int model, int ncells) {
    int threads = 0, blocks = 0;
    if (!resident_shape<L, S>(ncells, threads, blocks)) return false;
    if (model == kModelPRImplicit) return false;
    if (model == LBM_MODEL_PR) {
        if constexpr (resident_pr<L, S>()) return resident_ready<L, LBM_MODEL_PR, S>();
        return false;
    }
    if constexpr (resident_ir<L, S>()) return resident_ready<L, LBM_MODEL_IR, S>();
    return false;
}

template <class L> bool resident_fits_lat(int model, int storage, int ncells) {
    switch (storage) {
    case LBM_F32: return resident_fits_model<L, float>(model, ncells);
    case LBM_F64: return resident_fits_model<L, double>(model, ncells);
    case LBM_F16_OFS: return resident_fits_model<L, __half>(model, ncells);
    case LBM_BF16_OFS: return resident_fits_model<L, __nv_bfloat16>(model, ncells);
    default: return false;
    }
}

template <class L, int MODEL, class S, bool COPY>
cudaError_t launch_step_c(bool check, const KParams& kp, const StepArgs& s, cudaStream_t st) {
    using R = typename Store<S>::R;
    const KArgs a = make_args<L>(kp);
    const int ncell = kp.cell_end - kp.cell_begin;   // the cells this launch covers
    const SrcPlanes<S> src = src_planes<L, S>(s.fsrc, kp.plane);
    const DstPlanes<S> dst = dst_planes<L, S>(s.fdst, kp.plane);
    constexpr bool f64 = std::is_same<typename Store<S>::R, double>::value;
    // the implicit step is not in the tuning table (FP64: 64 threads, as untuned_block())
    const int block = check ? kBlock : MODEL == kModelPRImplicit ? (f64 ? 64 : kBlock) : s.block;
    if constexpr (MODEL != kModelPRImplicit && std::is_same<typename Store<S>::R, float>::value) {
        if (!check && s.cpt == 2) {   // two cells per thread
            if (block == 128)
                return launch_step<k_step2<L, MODEL, S, 128>, R>((kp.ncells + 255) / 256, 128, st, a, src,
                                                              dst, s.links, (R*)s.tau, s.rng_ctr, s.parity);
            return launch_step<k_step2<L, MODEL, S, 256>, R>((kp.ncells + 511) / 512, 256, st, a, src, dst,
                                                          s.links, (R*)s.tau, s.rng_ctr, s.parity);
        }
    }
    // (the block size and whether it is a check step, whole or in part)
    auto go = [&](auto B, auto CHECK, auto PART) {
        constexpr int b = decltype(B)::value;
        return launch_step<k_step<L, MODEL, S, decltype(CHECK)::value, b, COPY, decltype(PART)::value>, R>(
            (ncell + b - 1) / b, b, st, a, src, dst, s.links, (R*)s.tau, (R*)s.usnap, s.partials,
            s.rng_ctr, s.parity);
    };
    constexpr std::true_type yes;
    constexpr std::false_type no;
#define BLBM_B(n) std::integral_constant<int, n>{}
    if (check) return go(BLBM_B(kBlock), yes, no);
    // FP64 domains that leave sub-partitions idle
    if constexpr (f64 && MODEL != kModelPRImplicit) {
        if (s.split && kp.cell_begin == 0 && kp.cell_end == kp.ncells &&
            (int64_t)kp.ncells * parts<L>() <= kSplitLanes)
            return launch_step<k_step_split<L, MODEL>, R>((kp.ncells + 31) / 32, 32 * parts<L>(), st, a, src,
                                                       dst, s.links, (R*)s.tau);
    }
    // one part of a step taken in parts (256 threads)
    if (kp.cell_begin != 0 || kp.cell_end != kp.ncells)
        return go(BLBM_B(kBlock), no, yes);
    if constexpr (MODEL != kModelPRImplicit || f64) {
        if (block == 64) return go(BLBM_B(64), no, no);
    }
    if constexpr (MODEL != kModelPRImplicit) {
        if (block == 128) return go(BLBM_B(128), no, no);
        if (block == 512) return go(BLBM_B(512), no, no);
    }
    return go(BLBM_B(kBlock), no, no);
#undef BLBM_B
}

template <class L, int MODEL, class S>
cudaError_t launch_step_compact(bool check, const KParams& kp, const StepArgs& s, cudaStream_t st) {
    using R = typename Store<S>::R;
    const KArgs a = make_args<L>(kp);
    const SrcPlanes<S> src = src_planes<L, S>(s.fsrc, kp.plane);
    const DstPlanes<S> dst = dst_planes<L, S>(s.fdst, kp.plane);
    // The 16-bit steps are not overlapped: with their loads in front of the wait the
    // compiler orders the rest worse (D3Q27 FP16, 160^3 porous box: PR 109.3 -> 115.5 us;
    // 100^3, IR 21.7 -> 23.4) and contracts the class sums of D3Q15 and D3Q19 IR
    // differently; behind it an overlapped launch gains nothing.
    auto one = [&](auto B, auto CHECK) {
        constexpr int b = decltype(B)::value;
        constexpr auto kernel = k_step_compact<L, MODEL, S, decltype(CHECK)::value, b>;
        const int blocks = (kp.nslots + b - 1) / b;
        if constexpr (Store<S>::kStochastic)
            return launch_kernel(false, kernel, blocks, b, st, a, src, dst, s.links, s.cellidx, s.rank,
                                 (R*)s.tau, (R*)s.usnap, s.partials, s.rng_ctr, s.parity);
        else
            return launch_step<kernel, R>(blocks, b, st, a, src, dst, s.links, s.cellidx, s.rank, (R*)s.tau,
                                       (R*)s.usnap, s.partials, s.rng_ctr, s.parity);
    };
    if (check) return one(std::integral_constant<int, kBlock>{}, std::true_type{});
    if constexpr (compact_loop<MODEL, S>()) {
        // persistent: as many blocks as are resident at once, at most one per 256 slots
        static const int resident = [] {   // blocks per SM (per instantiation)
            int r = 0;
            if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&r, k_step_compact_loop<L, MODEL, S>,
                                                              kBlock, 0) != cudaSuccess) {
                cudaGetLastError();
                r = 1;
            }
            return r < 1 ? 1 : r;
        }();
        int dev = 0, sms = 0;
        cudaGetDevice(&dev);
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
        const int pgrid = std::min(step_grid(kp.nslots), std::max(1, resident * sms));
        return launch_kernel(false, k_step_compact_loop<L, MODEL, S>, pgrid, kBlock, st, a, src, dst,
                             s.links, s.cellidx, s.rank, (R*)s.tau, s.rng_ctr, s.parity);
    }
    // few slots: finer blocks spread over the SMs (see untuned_block)
    if (kp.nslots <= 8 * 152 * kBlock) return one(std::integral_constant<int, 128>{}, std::false_type{});
    return one(std::integral_constant<int, compact_block<L, MODEL>()>{}, std::false_type{});
}

// The compact layout has its own kernel.  In the dense one the copy-through
// is on for every form but the PR step of the 16-bit ones, which follows the
// solver's geometry (s.copy).
template <class L, int MODEL, class S>
cudaError_t launch_step_t(bool check, const KParams& kp, const StepArgs& s, cudaStream_t st) {
    if (s.rank) return launch_step_compact<L, MODEL, S>(check, kp, s, st);
    if constexpr (copy_is_choice<MODEL, S>()) {
        if (!s.copy) return launch_step_c<L, MODEL, S, false>(check, kp, s, st);
    }
    return launch_step_c<L, MODEL, S, true>(check, kp, s, st);
}

template <class L, class S>
cudaError_t launch_step_model(int model, bool check, const KParams& kp, const StepArgs& s,
                              cudaStream_t st) {
    if (model == kModelPRImplicit) return launch_step_t<L, kModelPRImplicit, S>(check, kp, s, st);
    if (model == LBM_MODEL_PR) return launch_step_t<L, LBM_MODEL_PR, S>(check, kp, s, st);
    return launch_step_t<L, LBM_MODEL_IR, S>(check, kp, s, st);
}

template <class L>
cudaError_t launch_step_lat(int model, int storage, bool check, const KParams& kp,
                            const StepArgs& s, cudaStream_t st) {
    switch (storage) {
    case LBM_F32: return launch_step_model<L, float>(model, check, kp, s, st);
    case LBM_F64: return launch_step_model<L, double>(model, check, kp, s, st);
    case LBM_F16_OFS: return launch_step_model<L, __half>(model, check, kp, s, st);
    case LBM_BF16_OFS: return launch_step_model<L, __nv_bfloat16>(model, check, kp, s, st);
    default: return cudaErrorNotSupported;
    }
}

// Plain-step tile shapes of the batch (threads per CTA x cells per thread);
// FP64 storage and the Newton-implicit PR step run 256 x 1 only.
template <int MODEL, class S> constexpr bool batch_shapes_all() {
    return MODEL != kModelPRImplicit && !std::is_same<S, double>::value;
}

template <class L, int MODEL, class S>
cudaError_t launch_batch_t(bool check, const BatchDesc* descs, const int* block_dom, int nblocks,
                           int grid, int phase, double* partials, int threads, int cpt,
                           cudaStream_t st) {
    using R = typename Store<S>::R;
    if (check)
        return launch_step<k_step_batch_check<L, MODEL, S>, R>(grid, kBlock, st, descs, block_dom, nblocks,
                                                               phase, partials);
    auto go = [&](auto T, auto C) {
        return launch_step<k_step_batch<L, MODEL, S, decltype(T)::value, decltype(C)::value>, R>(
            grid, threads, st, descs, block_dom, nblocks, phase);
    };
#define BLBM_I(n) std::integral_constant<int, n>{}
    if (threads == 256 && cpt == 1) return go(BLBM_I(256), BLBM_I(1));
    if constexpr (batch_shapes_all<MODEL, S>()) {
        if (threads == 128 && cpt == 1) return go(BLBM_I(128), BLBM_I(1));
        if (threads == 512 && cpt == 1) return go(BLBM_I(512), BLBM_I(1));
        if (threads == 128 && cpt == 2) return go(BLBM_I(128), BLBM_I(2));
        if (threads == 256 && cpt == 2) return go(BLBM_I(256), BLBM_I(2));
    }
#undef BLBM_I
    return cudaErrorInvalidValue;
}

template <class L, class S>
cudaError_t launch_batch_model(int model, bool check, const BatchDesc* descs, const int* block_dom,
                               int nblocks, int grid, int phase, double* partials, int threads,
                               int cpt, cudaStream_t st) {
    if (model == kModelPRImplicit)
        return launch_batch_t<L, kModelPRImplicit, S>(check, descs, block_dom, nblocks, grid, phase, partials, threads, cpt, st);
    if (model == LBM_MODEL_PR)
        return launch_batch_t<L, LBM_MODEL_PR, S>(check, descs, block_dom, nblocks, grid, phase, partials, threads, cpt, st);
    return launch_batch_t<L, LBM_MODEL_IR, S>(check, descs, block_dom, nblocks, grid, phase, partials, threads, cpt, st);
}

template <class L>
cudaError_t launch_batch_lat(int model, int storage, bool check, const BatchDesc* descs,
                             const int* block_dom, int nblocks, int grid, int phase,
                             double* partials, int threads, int cpt, cudaStream_t st) {
    switch (storage) {
    case LBM_F32: return launch_batch_model<L, float>(model, check, descs, block_dom, nblocks, grid, phase, partials, threads, cpt, st);
    case LBM_F64: return launch_batch_model<L, double>(model, check, descs, block_dom, nblocks, grid, phase, partials, threads, cpt, st);
    case LBM_F16_OFS: return launch_batch_model<L, __half>(model, check, descs, block_dom, nblocks, grid, phase, partials, threads, cpt, st);
    case LBM_BF16_OFS: return launch_batch_model<L, __nv_bfloat16>(model, check, descs, block_dom, nblocks, grid, phase, partials, threads, cpt, st);
    default: return cudaErrorNotSupported;
    }
}

template <class L>
cudaError_t launch_links_lat(const KParams& kp, const uint8_t* mask, uint32_t* links,
                             const int* cellidx, cudaStream_t st) {
    if (cellidx)
        k_links_compact<L><<<step_grid(kp.nslots), kBlock, 0, st>>>(kp, mask, cellidx, links);
    else
        k_links<L><<<step_grid(kp.ncells), kBlock, 0, st>>>(kp, mask, links);
    return cudaGetLastError();
}

template <class L, class S>
cudaError_t launch_fields_s(const KArgs& a, const void* f, const uint32_t* links, const int* rank,
                            double* rho, double* ux, double* uy, double* uz, cudaStream_t st) {
    const int grid = step_grid(a.kp.ncells);
    const SrcPlanes<S> P = src_planes<L, S>(f, a.kp.plane);
    if (rank)
        k_fields_compact<L, S><<<grid, kBlock, 0, st>>>(a, P, links, rank, rho, ux, uy, uz);
    else
        k_fields<L, S><<<grid, kBlock, 0, st>>>(a, P, links, rho, ux, uy, uz);
    return cudaGetLastError();
}

template <class L>
cudaError_t launch_fields_lat(int storage, const KParams& kp, const void* f, const uint32_t* links,
                              const int* rank, double* rho, double* ux, double* uy, double* uz,
                              cudaStream_t st) {
    const KArgs a = make_args<L>(kp);
    switch (storage) {
    case LBM_F32: return launch_fields_s<L, float>(a, f, links, rank, rho, ux, uy, uz, st);
    case LBM_F64: return launch_fields_s<L, double>(a, f, links, rank, rho, ux, uy, uz, st);
    case LBM_F16_OFS: return launch_fields_s<L, __half>(a, f, links, rank, rho, ux, uy, uz, st);
    case LBM_BF16_OFS: return launch_fields_s<L, __nv_bfloat16>(a, f, links, rank, rho, ux, uy, uz, st);
    default: return cudaErrorNotSupported;
    }
}

template <class L, class S>
cudaError_t launch_reduce_s(int mode, const KArgs& a, const void* f, const uint32_t* links,
                            const int* cellidx, const int* rank, double* partials, int nblocks,
                            cudaStream_t st) {
    const SrcPlanes<S> P = src_planes<L, S>(f, a.kp.plane);
    if (cellidx) {
        if (mode == kReduceFlow)
            k_reduce<L, S, kReduceFlow, true><<<nblocks, kBlock, 0, st>>>(a, P, links, cellidx, rank, partials);
        else
            k_reduce<L, S, kReduceTotals, true><<<nblocks, kBlock, 0, st>>>(a, P, links, cellidx, rank, partials);
    } else {
        if (mode == kReduceFlow)
            k_reduce<L, S, kReduceFlow, false><<<nblocks, kBlock, 0, st>>>(a, P, links, nullptr, nullptr, partials);
        else
            k_reduce<L, S, kReduceTotals, false><<<nblocks, kBlock, 0, st>>>(a, P, links, nullptr, nullptr, partials);
    }
    return cudaGetLastError();
}

template <class L>
cudaError_t launch_reduce_lat(int storage, int mode, const KParams& kp, const void* f,
                              const uint32_t* links, const int* cellidx, const int* rank,
                              double* partials, int nblocks, cudaStream_t st) {
    const KArgs a = make_args<L>(kp);
    switch (storage) {
    case LBM_F32: return launch_reduce_s<L, float>(mode, a, f, links, cellidx, rank, partials, nblocks, st);
    case LBM_F64: return launch_reduce_s<L, double>(mode, a, f, links, cellidx, rank, partials, nblocks, st);
    case LBM_F16_OFS: return launch_reduce_s<L, __half>(mode, a, f, links, cellidx, rank, partials, nblocks, st);
    case LBM_BF16_OFS: return launch_reduce_s<L, __nv_bfloat16>(mode, a, f, links, cellidx, rank, partials, nblocks, st);
    default: return cudaErrorNotSupported;
    }
}

template <class L>
cudaError_t launch_convert_lat(int storage, bool to_device, const KParams& kp, int q, void* f,
                               double* buf, const int* rank, cudaStream_t st) {
    const int grid = step_grid(kp.ncells);
    switch (storage) {
    case LBM_F32: k_convert<L, float><<<grid, kBlock, 0, st>>>(kp, q, to_device, (float*)f, buf, rank); break;
    case LBM_F64: k_convert<L, double><<<grid, kBlock, 0, st>>>(kp, q, to_device, (double*)f, buf, rank); break;
    case LBM_F16_OFS: k_convert<L, __half><<<grid, kBlock, 0, st>>>(kp, q, to_device, (__half*)f, buf, rank); break;
    case LBM_BF16_OFS: k_convert<L, __nv_bfloat16><<<grid, kBlock, 0, st>>>(kp, q, to_device, (__nv_bfloat16*)f, buf, rank); break;
    default: return cudaErrorNotSupported;
    }
    return cudaGetLastError();
}

template <class L>
cudaError_t launch_gather_lat(int storage, const KParams& kp, const void* f, const int64_t* cells,
                              int n, double* out, const int* rank, cudaStream_t st) {
    const int grid = (n + kBlock - 1) / kBlock;
    switch (storage) {
    case LBM_F32: k_gather_cells<L, float><<<grid, kBlock, 0, st>>>(kp, (const float*)f, cells, n, out, rank); break;
    case LBM_F64: k_gather_cells<L, double><<<grid, kBlock, 0, st>>>(kp, (const double*)f, cells, n, out, rank); break;
    case LBM_F16_OFS: k_gather_cells<L, __half><<<grid, kBlock, 0, st>>>(kp, (const __half*)f, cells, n, out, rank); break;
    case LBM_BF16_OFS: k_gather_cells<L, __nv_bfloat16><<<grid, kBlock, 0, st>>>(kp, (const __nv_bfloat16*)f, cells, n, out, rank); break;
    default: return cudaErrorNotSupported;
    }
    return cudaGetLastError();
}

template <class L>
cudaError_t launch_halo_lat(int storage, const KParams& kp, void* f, void* buf, int side,
                            bool pack, cudaStream_t st) {
    const int n = face_count<L>() * kp.nx * kp.ny;
    const int grid = (n + kBlock - 1) / kBlock;
    switch (storage) {
    case LBM_F32: k_halo<L, float><<<grid, kBlock, 0, st>>>(kp, (float*)f, (float*)buf, side, pack); break;
    case LBM_F64: k_halo<L, double><<<grid, kBlock, 0, st>>>(kp, (double*)f, (double*)buf, side, pack); break;
    case LBM_F16_OFS: k_halo<L, __half><<<grid, kBlock, 0, st>>>(kp, (__half*)f, (__half*)buf, side, pack); break;
    case LBM_BF16_OFS: k_halo<L, __nv_bfloat16><<<grid, kBlock, 0, st>>>(kp, (__nv_bfloat16*)f, (__nv_bfloat16*)buf, side, pack); break;
    default: return cudaErrorNotSupported;
    }
    return cudaGetLastError();
}

template <class L> int face_count_lat() { return face_count<L>(); }

template <class L> void lattice_table(int* c, double* w) {
    for (int i = 0; i < L::Q; ++i) {
        if (c) {
            c[3 * i] = L::cx(i);
            c[3 * i + 1] = L::cy(i);
            c[3 * i + 2] = L::cz(i);
        }
        if (w) w[i] = L::w(i);
    }
}

}  // namespace blbm

#define BLBM_DEFINE_LAUNCHERS(L)                                                               \
    namespace blbm {                                                                            \
    cudaError_t launch_step_##L(int model, int storage, bool check, const KParams& kp,         \
                                const StepArgs& a, cudaStream_t st) {                           \
        return launch_step_lat<L>(model, storage, check, kp, a, st);                            \
    }                                                                                           \
    cudaError_t launch_links_##L(const KParams& kp, const uint8_t* mask, uint32_t* links,      \
                                 const int* cellidx, cudaStream_t st) {                         \
        return launch_links_lat<L>(kp, mask, links, cellidx, st);                               \
    }                                                                                           \
    cudaError_t launch_fields_##L(int storage, const KParams& kp, const void* f,               \
                                  const uint32_t* links, const int* rank, double* rho,         \
                                  double* ux, double* uy, double* uz, cudaStream_t st) {        \
        return launch_fields_lat<L>(storage, kp, f, links, rank, rho, ux, uy, uz, st);          \
    }                                                                                           \
    cudaError_t launch_reduce_##L(int storage, int mode, const KParams& kp, const void* f,     \
                                  const uint32_t* links, const int* cellidx, const int* rank,  \
                                  double* partials, int nblocks, cudaStream_t st) {             \
        return launch_reduce_lat<L>(storage, mode, kp, f, links, cellidx, rank, partials,       \
                                    nblocks, st);                                               \
    }                                                                                           \
    cudaError_t launch_convert_##L(int storage, bool to_device, const KParams& kp, int q,      \
                                   void* f, double* plane_buf, const int* rank,                 \
                                   cudaStream_t st) {                                           \
        return launch_convert_lat<L>(storage, to_device, kp, q, f, plane_buf, rank, st);        \
    }                                                                                           \
    void lattice_table_##L(int* c, double* w) { lattice_table<L>(c, w); }                       \
    cudaError_t launch_gather_##L(int storage, const KParams& kp, const void* f,               \
                                  const int64_t* cells, int n, double* out, const int* rank,   \
                                  cudaStream_t st) {                                            \
        return launch_gather_lat<L>(storage, kp, f, cells, n, out, rank, st);                   \
    }                                                                                           \
    cudaError_t launch_halo_##L(int storage, const KParams& kp, void* f, void* buf, int side,  \
                                bool pack, cudaStream_t st) {                                   \
        return launch_halo_lat<L>(storage, kp, f, buf, side, pack, st);                         \
    }                                                                                           \
    int face_count_##L() { return face_count_lat<L>(); }                                        \
    }

// The batch kernels of a lattice, in a translation unit of their own.
#define BLBM_DEFINE_BATCH_LAUNCHERS(L)                                                         \
    namespace blbm {                                                                            \
    cudaError_t launch_step_batch_##L(int model, int storage, bool check, const BatchDesc* descs,\
                                      const int* block_dom, int nblocks, int grid, int phase,  \
                                      double* partials, int threads, int cpt, cudaStream_t st) {\
        return launch_batch_lat<L>(model, storage, check, descs, block_dom, nblocks, grid,      \
                                   phase, partials, threads, cpt, st);                          \
    }                                                                                           \
    }

// The resident runs of a lattice, in a translation unit of their own.
#define BLBM_DEFINE_RESIDENT_LAUNCHERS(L)                                                      \
    namespace blbm {                                                                            \
    cudaError_t launch_resident_##L(int model, int storage, const KParams& kp,                 \
                                    const StepArgs& a, int nsteps, cudaStream_t st) {           \
        return launch_resident_lat<L>(model, storage, kp, a, nsteps, st);                       \
    }                                                                                           \
    bool resident_fits_##L(int model, int storage, int ncells) {                                \
        return resident_fits_lat<L>(model, storage, ncells);                                           \
    }                                                                                           \
    }
