// teuk_step_common.cuh -- device building blocks of the Lax-Wendroff step kernels:
// precision policies, node loads/stores, the compensated update, the predictor
// (Eq. 13) and corrector (Eq. 14) bodies.  See teuk_step.cu for the scheme.
#pragma once
#include "teuk_df.cuh"
#include "teuk_internal.cuh"

namespace teuk {

constexpr int kMaxRows = 1024;   // a block holds one theta column of up to 1024 rows

// ---------------------------------------------------------------- complex
template <typename T>
struct Cx {
    T re, im;
    __device__ __forceinline__ static Cx zero() { return {T(0), T(0)}; }
};
template <typename T>
__device__ __forceinline__ Cx<T> operator+(Cx<T> a, Cx<T> b) { return {a.re + b.re, a.im + b.im}; }
template <typename T>
__device__ __forceinline__ Cx<T> operator-(Cx<T> a, Cx<T> b) { return {a.re - b.re, a.im - b.im}; }
template <typename T>
__device__ __forceinline__ Cx<T> operator*(T s, Cx<T> a) { return {s * a.re, s * a.im}; }
// Fused multiply-add in the type itself (a plain fma() call on floats would resolve to
// the double overload and run on the FP64 pipe).
__device__ __forceinline__ float tfma(float a, float b, float c) { return __fmaf_rn(a, b, c); }
__device__ __forceinline__ double tfma(double a, double b, double c) { return __fma_rn(a, b, c); }

// acc + (cr + i ci) * z
template <typename T>
__device__ __forceinline__ Cx<T> cmac(Cx<T> acc, T cr, T ci, Cx<T> z) {
    return {tfma(cr, z.re, tfma(-ci, z.im, acc.re)), tfma(cr, z.im, tfma(ci, z.re, acc.im))};
}
// acc + s * z (s real)
template <typename T>
__device__ __forceinline__ Cx<T> rmac(Cx<T> acc, T s, Cx<T> z) {
    return {tfma(s, z.re, acc.re), tfma(s, z.im, acc.im)};
}

// FP32 complex values in paired instructions (sm_100 and later: FADD2 / FMUL2 / FFMA2
// act on both components of a register pair).  Each component rounds exactly as the
// scalar round-to-nearest operation, so these overloads change no result, only the
// instruction count.
__device__ __forceinline__ float2 pk(Cx<float> a) { return make_float2(a.re, a.im); }
__device__ __forceinline__ Cx<float> up(float2 v) { return {v.x, v.y}; }
__device__ __forceinline__ float2 bc(float s) { return make_float2(s, s); }
__device__ __forceinline__ Cx<float> operator+(Cx<float> a, Cx<float> b) {
    return up(__fadd2_rn(pk(a), pk(b)));
}
// a - b as b * (-1) + a: the product is exact, so this rounds as the subtraction
__device__ __forceinline__ Cx<float> operator-(Cx<float> a, Cx<float> b) {
    return up(__ffma2_rn(bc(-1.0f), pk(b), pk(a)));
}
__device__ __forceinline__ Cx<float> operator*(float s, Cx<float> a) {
    return up(__fmul2_rn(bc(s), pk(a)));
}
// Complex double-float values in paired instructions: the high parts (re, im) and the
// low parts (re, im) each form a register pair, and every step of the scalar
// double-float operation (teuk_df.cuh) runs on both components at once, with the same
// roundings, so the results equal the scalar code's.
struct DF2 { float2 hi, lo; };
__device__ __forceinline__ DF2 pk2(Cx<DF> a) {
    return {make_float2(a.re.hi, a.im.hi), make_float2(a.re.lo, a.im.lo)};
}
__device__ __forceinline__ Cx<DF> up2(DF2 v) { return {DF(v.hi.x, v.lo.x), DF(v.hi.y, v.lo.y)}; }
__device__ __forceinline__ float2 p_add(float2 a, float2 b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ float2 p_sub(float2 a, float2 b) { return __ffma2_rn(bc(-1.0f), b, a); }   // exact product
__device__ __forceinline__ float2 p_neg(float2 a) { return make_float2(-a.x, -a.y); }
// s + e = a + b exactly (per component)
__device__ __forceinline__ DF2 p_two_sum(float2 a, float2 b) {
    const float2 s = p_add(a, b);
    const float2 bb = p_sub(s, a);
    return {s, p_add(p_sub(a, p_sub(s, bb)), p_sub(b, bb))};
}
// s + e = a - b exactly (two_sum with -b written out)
__device__ __forceinline__ DF2 p_two_diff(float2 a, float2 b) {
    const float2 s = p_sub(a, b);
    const float2 bb = p_sub(s, a);
    return {s, p_sub(p_sub(a, p_sub(s, bb)), p_add(b, bb))};
}
__device__ __forceinline__ DF2 p_fast_two_sum(float2 a, float2 b) {
    const float2 s = p_add(a, b);
    return {s, p_sub(b, p_sub(s, a))};
}
__device__ __forceinline__ Cx<DF> operator+(Cx<DF> x, Cx<DF> y) {
    const DF2 X = pk2(x), Y = pk2(y);
    const DF2 S = p_two_sum(X.hi, Y.hi);
    return up2(p_fast_two_sum(S.hi, p_add(S.lo, p_add(X.lo, Y.lo))));
}
__device__ __forceinline__ Cx<DF> operator-(Cx<DF> x, Cx<DF> y) {
    const DF2 X = pk2(x), Y = pk2(y);
    const DF2 S = p_two_diff(X.hi, Y.hi);
    return up2(p_fast_two_sum(S.hi, p_add(S.lo, p_sub(X.lo, Y.lo))));
}
// a * b + c per component, a given as pairs (hi, lo): the double-float tfma without its last
// normalisation (see Lin<DF> for how large lo may get)
__device__ __forceinline__ DF2 p_tfma(DF2 A, DF2 B, DF2 C) {
    const float2 p = __fmul2_rn(A.hi, B.hi);
    float2 e = __ffma2_rn(A.hi, B.hi, p_neg(p));
    e = __ffma2_rn(A.hi, B.lo, e);
    e = __ffma2_rn(A.lo, B.hi, e);
    const DF2 S = p_two_sum(p, C.hi);
    return {S.hi, p_add(S.lo, p_add(e, C.lo))};
}
__device__ __forceinline__ DF2 bc2(DF s) { return {bc(s.hi), bc(s.lo)}; }
__device__ __forceinline__ Cx<DF> operator*(DF s, Cx<DF> a) {
    const DF2 S = bc2(s), A = pk2(a);
    const float2 p = __fmul2_rn(S.hi, A.hi);
    float2 e = __ffma2_rn(S.hi, A.hi, p_neg(p));
    e = __ffma2_rn(S.hi, A.lo, e);
    e = __ffma2_rn(S.lo, A.hi, e);
    return up2(p_fast_two_sum(p, e));
}
__device__ __forceinline__ Cx<DF> rmac(Cx<DF> acc, DF s, Cx<DF> z) {
    return up2(p_tfma(bc2(s), pk2(z), pk2(acc)));
}
// same order as the generic cmac: the ci terms first, then the cr terms
__device__ __forceinline__ Cx<DF> cmac(Cx<DF> acc, DF cr, DF ci, Cx<DF> z) {
    const DF2 Z = pk2(z);
    const DF2 Zs = {make_float2(Z.hi.y, Z.hi.x), make_float2(Z.lo.y, Z.lo.x)};   // (im, re)
    const DF2 Ci = {make_float2(-ci.hi, ci.hi), make_float2(-ci.lo, ci.lo)};
    return up2(p_tfma(bc2(cr), Z, p_tfma(Ci, Zs, pk2(acc))));
}
__device__ __forceinline__ Cx<float> rmac(Cx<float> acc, float s, Cx<float> z) {
    return up(__ffma2_rn(bc(s), pk(z), pk(acc)));
}

// ---------------------------------------------------------------- precisions
// kind: the teuk_precision value; planes: 16-byte planes per state buffer (the layout
// in teuk_internal.cuh); blocks256: resident blocks per SM that the register budget of
// the step kernel for columns of up to 256 rows aims at (two: at three the FP32 paths
// fit in 80 registers but run no faster, being issue-bound)
enum PrecKind { kFP64 = 0, kFP32 = 1, kKahan = 2, kDF = 3 };
struct P64 {
    using T = double;
    static constexpr bool kahan = false;
    static constexpr int kind = kFP64, planes = 2, blocks256 = 2;
};
struct P32 {
    using T = float;
    static constexpr bool kahan = false;
    static constexpr int kind = kFP32, planes = 1, blocks256 = 2;
};
struct PK {
    using T = float;
    static constexpr bool kahan = true;
    static constexpr int kind = kKahan, planes = 2, blocks256 = 2;
};
// FP64-equivalent: double-float state, coefficients and arithmetic on the FP32 units
struct PD {
    using T = DF;
    static constexpr bool kahan = false;
    static constexpr int kind = kDF, planes = 2, blocks256 = 2;
};
template <typename T> __host__ __device__ constexpr bool uses_pairs() { return false; }
template <> __host__ __device__ constexpr bool uses_pairs<DF>() { return true; }
// the FP32 paths that form their coefficients from 1D tables
template <class P>
__host__ __device__ constexpr bool uses_1d_tables() { return P::kind == kFP32 || P::kind == kKahan; }

// Compensated add (Kahan 1965) of both components of a complex value: the represented
// value is hi - c.
__device__ __forceinline__ void kahan_add(Cx<float>& hi, Cx<float>& c, Cx<float> delta) {
    const Cx<float> y = delta - c;
    const Cx<float> t = hi + y;
    c = (t - hi) - y;
    hi = t;
}

// State of one node: Phi, Pi (and, compensated, their c parts).
template <class P>
struct NodeV {
    using T = typename P::T;
    Cx<T> F, Pp;      // hi parts (or the value)
    Cx<T> Fc, Pc;     // compensations (Kahan only; zero otherwise)
    __device__ __forceinline__ static NodeV zero() {
        NodeV n;
        n.F = n.Pp = n.Fc = n.Pc = Cx<T>::zero();
        return n;
    }
    // Phi(this) - Phi(o), accurate for compensated pairs
    __device__ __forceinline__ Cx<T> dphi(const NodeV& o) const {
        if constexpr (P::kahan) return (F - o.F) - (Fc - o.Fc);
        else return F - o.F;
    }
    // Split theta differences of Phi at this node from the rows above (a, factor ga)
    // and below (b, factor gb), given -ga and -gb: nd2 = -(ga a - 2 this + gb b) and d1 =
    // ga a - gb b.  For compensated pairs the hi differences (exact for neighbouring values
    // within a factor of two) and the c differences are combined first, so nd2 and d1 round
    // relative to their own size, not to that of the first differences.
    __device__ __forceinline__ void theta_split(T nga, const NodeV& a, T ngb, const NodeV& b,
                                                Cx<T>& nd2, Cx<T>& d1) const {
        const Cx<T> hp = rmac(F, nga, a.F);   // this - ga a
        const Cx<T> hm = rmac(F, ngb, b.F);   // this - gb b
        if constexpr (P::kahan) {
            const Cx<T> cp = rmac(Fc, nga, a.Fc);
            const Cx<T> cm = rmac(Fc, ngb, b.Fc);
            nd2 = (hp + hm) - (cp + cm);
            d1 = (hm - hp) - (cm - cp);
        } else {
            nd2 = hp + hm;
            d1 = hm - hp;
        }
    }
    __device__ __forceinline__ Cx<T> dpi(const NodeV& o) const {
        if constexpr (P::kahan) return (Pp - o.Pp) - (Pc - o.Pc);
        else return Pp - o.Pp;
    }
    __device__ __forceinline__ double2 phi64() const {
        double v[4];
        v64(v);
        return make_double2(v[0], v[1]);
    }
    // {Phi_R, Phi_I, Pi_R, Pi_I} as FP64
    __device__ __forceinline__ void v64(double* v) const {
        if constexpr (P::kind == kDF) {
            v[0] = F.re.to_double(); v[1] = F.im.to_double();
            v[2] = Pp.re.to_double(); v[3] = Pp.im.to_double();
        } else if constexpr (P::kahan) {
            v[0] = (double)F.re - (double)Fc.re; v[1] = (double)F.im - (double)Fc.im;
            v[2] = (double)Pp.re - (double)Pc.re; v[3] = (double)Pp.im - (double)Pc.im;
        } else {
            v[0] = (double)F.re; v[1] = (double)F.im; v[2] = (double)Pp.re; v[3] = (double)Pp.im;
        }
    }
    __device__ __forceinline__ void update(Cx<T> dF, Cx<T> dP) {
        if constexpr (P::kahan) {
            kahan_add(F, Fc, dF);
            kahan_add(Pp, Pc, dP);
        } else {
            F = F + dF; Pp = Pp + dP;
        }
    }
};

// Views of the planes of one ping-pong buffer.
template <class P> struct Planes;
template <> struct Planes<P64> {
    double2* phi; double2* pi;
    __device__ __forceinline__ static Planes of(const InstDev& d, int b) {
        return {(double2*)d.buf[b][0], (double2*)d.buf[b][1]};
    }
    // planes of one column copied to shared memory, `stride` nodes apart
    __device__ __forceinline__ static Planes at(void* base, unsigned stride) {
        return {(double2*)base, (double2*)base + stride};
    }
    __device__ __forceinline__ NodeV<P64> load(size_t o) const {
        NodeV<P64> n;
        double2 a = phi[o], b = pi[o];
        n.F = {a.x, a.y}; n.Pp = {b.x, b.y};
        n.Fc = n.Pc = Cx<double>::zero();
        return n;
    }
    // Phi alone (the theta neighbours of a node)
    __device__ __forceinline__ NodeV<P64> load_phi(size_t o) const {
        NodeV<P64> n = NodeV<P64>::zero();
        double2 a = phi[o];
        n.F = {a.x, a.y};
        return n;
    }
    __device__ __forceinline__ void store(size_t o, const NodeV<P64>& n) const {
        phi[o] = make_double2(n.F.re, n.F.im);
        pi[o] = make_double2(n.Pp.re, n.Pp.im);
    }
};
template <> struct Planes<P32> {
    float4* u;
    __device__ __forceinline__ static Planes of(const InstDev& d, int b) { return {(float4*)d.buf[b][0]}; }
    __device__ __forceinline__ static Planes at(void* base, unsigned) { return {(float4*)base}; }
    __device__ __forceinline__ NodeV<P32> load(size_t o) const {
        NodeV<P32> n;
        float4 a = u[o];
        n.F = {a.x, a.y}; n.Pp = {a.z, a.w};
        n.Fc = n.Pc = Cx<float>::zero();
        return n;
    }
    __device__ __forceinline__ NodeV<P32> load_phi(size_t o) const {
        NodeV<P32> n = NodeV<P32>::zero();
        float2 a = *(const float2*)(u + o);
        n.F = {a.x, a.y};
        return n;
    }
    __device__ __forceinline__ void store(size_t o, const NodeV<P32>& n) const {
        u[o] = make_float4(n.F.re, n.F.im, n.Pp.re, n.Pp.im);
    }
};
template <> struct Planes<PK> {
    float4* hi; float4* c;
    __device__ __forceinline__ static Planes of(const InstDev& d, int b) {
        return {(float4*)d.buf[b][0], (float4*)d.buf[b][1]};
    }
    __device__ __forceinline__ static Planes at(void* base, unsigned stride) {
        return {(float4*)base, (float4*)base + stride};
    }
    __device__ __forceinline__ NodeV<PK> load(size_t o) const {
        NodeV<PK> n;
        float4 a = hi[o], b = c[o];
        n.F = {a.x, a.y}; n.Pp = {a.z, a.w};
        n.Fc = {b.x, b.y}; n.Pc = {b.z, b.w};
        return n;
    }
    __device__ __forceinline__ NodeV<PK> load_phi(size_t o) const {
        NodeV<PK> n = NodeV<PK>::zero();
        float2 a = *(const float2*)(hi + o), b = *(const float2*)(c + o);
        n.F = {a.x, a.y};
        n.Fc = {b.x, b.y};
        return n;
    }
    __device__ __forceinline__ void store(size_t o, const NodeV<PK>& n) const {
        hi[o] = make_float4(n.F.re, n.F.im, n.Pp.re, n.Pp.im);
        c[o] = make_float4(n.Fc.re, n.Fc.im, n.Pc.re, n.Pc.im);
    }
};

template <> struct Planes<PD> {
    float4* hi; float4* lo;   // {Phi, Pi} high parts, low parts
    __device__ __forceinline__ static Planes of(const InstDev& d, int b) {
        return {(float4*)d.buf[b][0], (float4*)d.buf[b][1]};
    }
    __device__ __forceinline__ static Planes at(void* base, unsigned stride) {
        return {(float4*)base, (float4*)base + stride};
    }
    __device__ __forceinline__ NodeV<PD> load(size_t o) const {
        NodeV<PD> n;
        const float4 a = hi[o], b = lo[o];
        n.F = {DF(a.x, b.x), DF(a.y, b.y)};
        n.Pp = {DF(a.z, b.z), DF(a.w, b.w)};
        n.Fc = n.Pc = Cx<DF>::zero();
        return n;
    }
    __device__ __forceinline__ NodeV<PD> load_phi(size_t o) const {
        NodeV<PD> n = NodeV<PD>::zero();
        const float2 a = *(const float2*)(hi + o), b = *(const float2*)(lo + o);
        n.F = {DF(a.x, b.x), DF(a.y, b.y)};
        return n;
    }
    __device__ __forceinline__ void store(size_t o, const NodeV<PD>& n) const {
        hi[o] = make_float4(n.F.re.hi, n.F.im.hi, n.Pp.re.hi, n.Pp.im.hi);
        lo[o] = make_float4(n.F.re.lo, n.F.im.lo, n.Pp.re.lo, n.Pp.im.lo);
    }
};

// ---------------------------------------------------------------- half nodes
template <typename T>
struct Half { Cx<T> Fb, Pb, dF, dP; };

// Sums and radial differences across the half node i+1/2 (own = column i, nb = column
// i+1): Fb = Phi_i + Phi_{i+1}, Pb the same of Pi.
template <class P>
__device__ __forceinline__ Half<typename P::T> half_prep(const NodeV<P>& own, const NodeV<P>& nb) {
    using T = typename P::T;
    Half<T> h;
    if constexpr (P::kahan) {
        h.Fb = (own.F + nb.F) - (own.Fc + nb.Fc);
        h.Pb = (own.Pp + nb.Pp) - (own.Pc + nb.Pc);
    } else {
        h.Fb = own.F + nb.F;
        h.Pb = own.Pp + nb.Pp;
    }
    h.dF = nb.dphi(own);
    h.dP = nb.dpi(own);
    return h;
}

// Angular term of S_Pi, w Theta[F] - w V F (the V part sits in E3), in one of two forms:
//   expanded (FP64, double-float): ep (F_{j+1} - F_j) - em (F_j - F_{j-1}),
//   split (FP32 paths):            A (F_{j+1} - 2 F_j + F_{j-1}) + B (F_{j+1} - F_{j-1}),
//   A = s dt w / dth^2, B = s dt w cot / (2 dth)  (ep = A + B, em = A - B).
// The two are the same operator.  In FP32 the split form keeps the large coefficient
// A on the second difference, which is formed from the compensated pairs to its own
// relative accuracy; the expanded form would round ep and em separately and apply
// them to first differences, an error of order A times the first difference that the
// long-run growth of the angular modes then amplifies.
template <class P>
__host__ __device__ constexpr bool split_angular() { return P::kind == kFP32 || P::kind == kKahan; }

// ---------------------------------------------------------------- expanded form
// FP64 and double-float step (HalfX, predict_x, correct_x).  What bounds it is the number
// of operations: GB300's FP64 pipe retires one warp DFMA per SM in 16 clocks, so every
// operation counts, and a double-float operation is 8 to 16 FP32 ones.  The half-node
// state is therefore kept undivided, as 2 h = (u_i + u_{i+1}) + ..., the powers of two
// folded into the coefficient tables (exactly; teuk_setup.cu), sums and differences are
// formed once and shared, and the angular differences are taken of the sums s = Phi_i +
// Phi_{i+1} and S = 2 h_R + 2 h_L, which the neighbouring rows exchange:
//   predictor   s, sP, dF, dP (sums and differences of columns i, i+1)
//     2 h_Phi = s + (dt/2) sP - G dF
//     2 h_Pi  = sP + G dP + E1 sP + E2 dF + ep (s(j+1) - s(j)) - em (s(j) - s(j-1)) + E3 s + dt tau
//   corrector   S, SP, D, DP (sums and differences of the half nodes R, L)
//     Phi += (dt/4) SP - G D
//     Pi  += G DP + E1 SP + E2 D + ep (S(j+1) - S(j)) - em (S(j) - S(j-1)) + E3 S + dt tau
// 72 FP64 operations a node where the form in separate half-node increments had 124.  The
// rounding error against extended precision is the same (60 x 128 grid, 1000 steps: 3.89e-15
// both), because both increments of the state are formed apart and added once.  16384 x 256,
// us per step before and after: FP64 947 -> 629, double-float 262 -> 205 (681 -> 506 paired
// FP32 operations a node, and no register spills: the record of a half node is two complex
// values instead of eight); with the time steps formed on the host and the pole factor
// applied to the sign bits (85 -> 75 FP64 instructions a node, and 14 -> 0 on the
// double-float path) and double-float coefficients loaded ahead: FP64 570 to 576, double-float 148.

// Complex sums and differences.  FP64: as DFMA with a factor one that the compiler cannot
// see (DADD and DMUL take 19 clocks of the SM's FP64 pipe, DFMA 16; the rounding is the
// sum's own).  A product is formed as DFMA with a zero addend for the same reason.
template <typename T> struct Lin;
template <> struct Lin<double> {
    using C = Cx<double>;
    double one;
    __device__ __forceinline__ explicit Lin(const InstDev& d) : one(d.one) {}
    __device__ __forceinline__ C add(C a, C b) const {
        return {__fma_rn(a.re, one, b.re), __fma_rn(a.im, one, b.im)};
    }
    __device__ __forceinline__ C update(C a, C b) const { return add(a, b); }
    __device__ __forceinline__ C sub(C a, C b) const {
        return {__fma_rn(b.re, -one, a.re), __fma_rn(b.im, -one, a.im)};
    }
    __device__ __forceinline__ C mul(double s, C a) const { return {__fma_rn(s, a.re, 0.0), __fma_rn(s, a.im, 0.0)}; }
};
// Double-float: the sums, differences and products of a step's chain stay unnormalised (three
// operations saved in each; as in Ogita, Rump and Oishi's compensated dot product, the
// residues are summed apart), only the state that is stored is normalised (update).  With
// u = 2^-24, n links and M the sum of the moduli of a chain's terms, a partial sum's lo stays
// within (n + 8) u M and the error within (38 + n + 2 n (n + 8)) u^2 M, also where hi cancels
// and lo holds the rest (the bounds count M, not the sum).  Measured on 2e6 chains of n = 10,
// half of them cancelling: rms 0.51, at most 13 u^2 M; normalised 0.31 and 4.9.  In a run the
// rounding of the state outweighs it: the error against 64 bits over 36 runs of 241 x 32 to
// 16384 x 256, in proportion to the normalised form's, is on average 1.002 (state, L2), 0.994
// (state, largest), 0.966 (waveform, L2) and 0.962 (waveform, largest).
// us per step: 16384 x 256 148 -> 136 (the tables and the state alone take 129 at the
// measured copy rate), 8192 x 128 43.5 -> 37.9, 800 x 64 5.4 -> 4.8.
template <> struct Lin<DF> {
    using C = Cx<DF>;
    __device__ __forceinline__ explicit Lin(const InstDev&) {}
    __device__ __forceinline__ C update(C a, C b) const { return a + b; }
    __device__ __forceinline__ C add(C x, C y) const {
        const DF2 X = pk2(x), Y = pk2(y);
        const DF2 S = p_two_sum(X.hi, Y.hi);
        return up2({S.hi, p_add(S.lo, p_add(X.lo, Y.lo))});
    }
    __device__ __forceinline__ C sub(C x, C y) const {
        const DF2 X = pk2(x), Y = pk2(y);
        const DF2 S = p_two_diff(X.hi, Y.hi);
        return up2({S.hi, p_add(S.lo, p_sub(X.lo, Y.lo))});
    }
    __device__ __forceinline__ C mul(DF s, C a) const {
        const DF2 S = bc2(s), A = pk2(a);
        const float2 p = __fmul2_rn(S.hi, A.hi);
        float2 e = __ffma2_rn(S.hi, A.hi, p_neg(p));
        e = __ffma2_rn(S.hi, A.lo, e);
        return up2({p, __ffma2_rn(S.lo, A.hi, e)});
    }
};

template <> struct Lin<float> {   // (the FP32 paths take the split form)
    __device__ __forceinline__ explicit Lin(const InstDev&) {}
};

// 2 h_Phi and 2 h_Pi at one half node
template <typename T>
struct HalfX { Cx<T> F, P; };

// kSrc: src is a source term (else it is not read)
template <typename T, bool kSrc>
__device__ __forceinline__ HalfX<T> predict_x(const Lin<T>& A, Cx<T> F0, Cx<T> P0, Cx<T> F1, Cx<T> P1, Cx<T> s,
                                              Cx<T> s_p, Cx<T> s_m, const T* cf, T hdt, Cx<T> src) {
    const Cx<T> dF = A.sub(F1, F0), sP = A.add(P0, P1), dP = A.sub(P1, P0);
    HalfX<T> h;
    h.F = rmac(rmac(s, hdt, sP), -cf[C_G], dF);
    Cx<T> a = rmac(sP, cf[C_G], dP);
    a = cmac(a, cf[C_E1R], cf[C_E1I], sP);
    a = cmac(a, cf[C_E2R], cf[C_E2I], dF);
    a = cmac(a, cf[C_E3R], cf[C_E3I], s);
    a = rmac(a, cf[C_EP], A.sub(s_p, s));
    a = rmac(a, -cf[C_EM], A.sub(s, s_m));
    if constexpr (kSrc) a = A.add(a, src);
    h.P = a;
    return h;
}

// Eq. (14) at one node: the increments of Phi and Pi from the half nodes R and L, with S =
// R.F + L.F of this row and of the rows above and below
template <typename T, bool kSrc>
__device__ __forceinline__ void correct_x(const Lin<T>& A, const HalfX<T>& R, const HalfX<T>& L, Cx<T> S, Cx<T> S_p,
                                          Cx<T> S_m, const T* cf, T qdt, Cx<T> src, Cx<T>& dPhi, Cx<T>& dPi) {
    const Cx<T> D = A.sub(R.F, L.F), SP = A.add(R.P, L.P), DP = A.sub(R.P, L.P);
    dPhi = rmac(A.mul(qdt, SP), -cf[C_G], D);
    Cx<T> a;
    if constexpr (kSrc) a = rmac(src, cf[C_G], DP);
    else a = A.mul(cf[C_G], DP);
    a = cmac(a, cf[C_E1R], cf[C_E1I], SP);
    a = cmac(a, cf[C_E2R], cf[C_E2I], D);
    a = cmac(a, cf[C_E3R], cf[C_E3I], S);
    a = rmac(a, cf[C_EP], A.sub(S_p, S));
    a = rmac(a, -cf[C_EM], A.sub(S, S_m));
    dPi = a;
}

// A complex value as one 16-byte shared-memory entry
__device__ __forceinline__ void put16(void* e, Cx<double> v) { *(double2*)e = make_double2(v.re, v.im); }
__device__ __forceinline__ void put16(void* e, Cx<DF> v) {
    *(float4*)e = make_float4(v.re.hi, v.im.hi, v.re.lo, v.im.lo);
}
template <typename T>
__device__ __forceinline__ Cx<T> get16(const void* e) {
    if constexpr (sizeof(Cx<T>) == sizeof(double2) && !uses_pairs<T>()) {
        const double2 v = *(const double2*)e;
        return {v.x, v.y};
    } else {
        const float4 v = *(const float4*)e;
        return {T(v.x, v.z), T(v.y, v.w)};
    }
}
// +-v, by the sign bits (flip: 0 or the sign bit), without an operation on the FP64 or FMA
// pipe
__device__ __forceinline__ float flip_sign(float v, int flip) { return __int_as_float(__float_as_int(v) ^ flip); }
__device__ __forceinline__ double flip_sign(double v, int flip) {
    return __hiloint2double(__double2hiint(v) ^ flip, __double2loint(v));
}
__device__ __forceinline__ DF flip_sign(DF v, int flip) { return DF(flip_sign(v.hi, flip), flip_sign(v.lo, flip)); }
template <typename T>
__device__ __forceinline__ Cx<T> flip_sign(Cx<T> v, int flip) { return {flip_sign(v.re, flip), flip_sign(v.im, flip)}; }
// flip of the pole factor
__device__ __forceinline__ int pole_flip(const InstDev& d) { return d.ghost_f < 0.f ? (int)0x80000000 : 0; }

// The pole rows of a column (0 and n_theta - 1, distinct: n_theta >= 4) and the exchange
// entry of the ghost row beyond each (0 and n_theta + 1)
struct PoleRow {
    bool edge;
    int entry, flip;
    __device__ __forceinline__ PoleRow(const InstDev& d, int j)
        : edge(j == 0 || j == d.nth - 1), entry(j == 0 ? 0 : d.nth + 1), flip(pole_flip(d)) {}
};
// Publish this row's value (row j at entry j + 1 of x) and, for a pole row, its ghost row's
template <typename T>
__device__ __forceinline__ void publish16(unsigned char* x, int j, Cx<T> v, const PoleRow& pole, bool row_ok) {
    if (row_ok) put16(x + 16 * (j + 1), v);
    if (pole.edge) put16(x + 16 * pole.entry, flip_sign(v, pole.flip));
}

// dt/2 and dt/4 in the arithmetic type
template <typename T>
__device__ __forceinline__ T step_hdt(const InstDev& d) {
    if constexpr (uses_pairs<T>()) return T(d.hdt2.x, d.hdt2.y);
    else if constexpr (sizeof(T) == 4) return d.hdt2.x;
    else return d.hdt;
}
template <typename T>
__device__ __forceinline__ T step_qdt(const InstDev& d) {
    if constexpr (uses_pairs<T>()) return T(d.qdt2.x, d.qdt2.y);
    else if constexpr (sizeof(T) == 4) return d.qdt2.x;
    else return d.qdt;
}

// ---------------------------------------------------------------- split form
// FP32 and FP32-Kahan step.  Issue and latency bound it (some 250 instructions a node, four
// warps a scheduler), so the averages over two and four values stay undivided sums, the
// powers of two folded into the 1D tables (exactly, so that every result keeps its bits), and
// the second difference is carried with the sign it is formed with.  us per step before and
// after: FP32-Kahan 16384 x 256 47.0 -> 46.1, 8192 x 128 14.3 -> 13.8; FP32 36.5 -> 34.9, 11.2
// -> 10.7.  (Real coefficients times complex values as two scalar FMAs, to save the
// broadcast of the coefficient into a register pair: no faster, FP32 35.2.)
// s a + b, s a power of two
__device__ __forceinline__ Cx<float> sadd(float s, Cx<float> a, Cx<float> b) {
    return up(__ffma2_rn(bc(s), pk(a), pk(b)));
}

// Predictor output at one half node, plus the inputs the corrector needs from it: Fb, Pb
// (sums over the two columns), the radial differences, Dp = -(Fb(j+1) - 2 Fb(j) + Fb(j-1)),
// D1 = Fb(j+1) - Fb(j-1), and the increments hF, hP.
template <typename T>
struct HalfRec { Cx<T> Fb, Pb, dF, dP, Dp, D1, hF, hP; };

// Corrector inputs of one row, combined from the half nodes R = i+1/2 and L = i-1/2.
template <typename T>
struct CRow {
    Cx<T> Hs;        // dh_Phi_R + dh_Phi_L
    Cx<T> DpS;       // Dp_R + Dp_L
    Cx<T> D1S;       // D1_R + D1_L
    Cx<T> FC, PC;    // 4 u~, u~ = (h_R + h_L)/2 for Phi and Pi
    Cx<T> dFc, dPc;  // h_R - h_L for Phi and Pi
};

template <typename T>
__device__ __forceinline__ CRow<T> combine_lr(const HalfRec<T>& R, const HalfRec<T>& L) {
    CRow<T> c;
    c.Hs = R.hF + L.hF;
    c.DpS = R.Dp + L.Dp;
    c.D1S = R.D1 + L.D1;
    c.FC = sadd(2.f, c.Hs, R.Fb + L.Fb);
    c.PC = sadd(2.f, R.hP + L.hP, R.Pb + L.Pb);
    c.dFc = sadd(0.5f, R.dF + L.dF, R.hF - L.hF);
    c.dPc = sadd(0.5f, R.dP + L.dP, R.hP - L.hP);
    return c;
}

// Coefficients of node (i, j) from a 2D table (rows past n_theta read its padding: in
// bounds, never used)
template <typename T>
__device__ __forceinline__ void load_coefs(const void* tab, int pitch, int i, int j, T* cf) {
    const char* p = (const char*)tab + ((size_t)i * (size_t)pitch + (size_t)(j & ~31)) * (kNCoef * 8u);
    const int l = j & 31;
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        if constexpr (uses_pairs<T>()) {
            const float4 v = __ldg((const float4*)(p + 512 * q) + l);
            cf[1 + 2 * q] = T(v.x, v.y);
            cf[2 + 2 * q] = T(v.z, v.w);
        } else {
            const double2 v = __ldg((const double2*)(p + 512 * q) + l);
            cf[1 + 2 * q] = v.x;
            cf[2 + 2 * q] = v.y;
        }
    }
    if constexpr (uses_pairs<T>()) {
        const float2 v = __ldg((const float2*)(p + 2048) + l);
        cf[C_G] = T(v.x, v.y);
    } else {
        cf[C_G] = __ldg((const double*)(p + 2048) + l);
    }
}

// The theta table of one row as broadcast pairs (x, x), held in registers by its thread
// for a whole work item (FP32 paths; empty for FP64, which reads 2D tables).
struct ThPair { float2 sin2, cs, V, i2, i1; };
template <class P>
struct RowTab {
    ThPair t;
    __device__ __forceinline__ void load(const ThTab* tab, int j, bool ok) {
        if constexpr (uses_1d_tables<P>()) {
            const ThTab h = ok ? tab[j] : ThTab{};
            t = ThPair{bc(h.sin2), bc(h.cs), bc(h.V), bc(h.i2), bc(h.i1)};
        }
    }
};

// FP32 coefficients of the half node i+1/2 (.x) and of the node i (.y) of one column,
// from the column's radial table and the row's theta table (see RTab2), in paired
// instructions.
__device__ __forceinline__ void form_coefs2(const RTab2& t, const ThPair& h, float2* cf) {
    const float2 sig2 = __ffma2_rn(t.naD, h.sin2, t.R2);
    float2 rs = make_float2(rsqrtf(sig2.x), rsqrtf(sig2.y));
    // one Newton step on 1/sqrt: rs (1.5 - (sig2 / 2) rs^2)
    const float2 hr = __fmul2_rn(__fmul2_rn(bc(-0.5f), sig2), rs);
    rs = __fmul2_rn(rs, __ffma2_rn(hr, rs, bc(1.5f)));
    const float2 iS = __fmul2_rn(rs, rs);                // 1/Sigma^2 within a few ulp
    const float2 g = __fmul2_rn(t.Rd, rs);
    const float2 ctre = __fmul2_rn(t.ctr, iS);
    const float2 ctim = __fmul2_rn(__ffma2_rn(t.ctc, h.cs, t.cti), iS);
    cf[C_G] = g;
    cf[C_E1R] = __fmul2_rn(t.nsdt, ctre);
    cf[C_E1I] = __fmul2_rn(t.nsdt, ctim);
    const float2 pb = __ffma2_rn(__fmul2_rn(t.nbb, h.sin2), iS, t.pr);   // pr - bb sin^2 iS
    cf[C_E2R] = __ffma2_rn(ctre, g, __fmul2_rn(pb, iS));
    cf[C_E2I] = __ffma2_rn(ctim, g, __fmul2_rn(t.pi, iS));
    const float2 ws = __fmul2_rn(t.Ds, iS);
    cf[C_EP] = __fmul2_rn(ws, h.i2);   // A (split angular form; -A from the forward tables)
    cf[C_EM] = __fmul2_rn(ws, h.i1);   // B
    cf[C_E3R] = __fmul2_rn(__ffma2_rn(t.nDs, h.V, t.qr), iS);
    cf[C_E3I] = __fmul2_rn(t.qi, iS);
}

// FP64 or double-float coefficients of the predictor (half = true, node i+1/2) or the
// corrector (node i) at row j, from the 2D tables.
template <typename T>
__device__ __forceinline__ void coefs2d(const InstDev& d, bool half, int i, int j, T* cf) {
    load_coefs<T>(half ? d.coef_h : d.coef_i, d.pitch, i, j, cf);
}

// Eq. (13) at the own half node, as an increment on the averaged state.  Dp, D1: the second
// (negated) and two-cell theta differences of Fb; qdt = dt/4.
template <typename T>
__device__ __forceinline__ HalfRec<T> predictor(const Half<T>& h, Cx<T> Dp, Cx<T> D1, const T* cf,
                                                T qdt, Cx<T> src) {
    HalfRec<T> r;
    r.Fb = h.Fb; r.Pb = h.Pb; r.dF = h.dF; r.dP = h.dP; r.Dp = Dp; r.D1 = D1;
    r.hF = rmac(rmac(Cx<T>::zero(), -cf[C_G], h.dF), qdt, h.Pb);
    Cx<T> a = rmac(src, cf[C_G], h.dP);
    a = cmac(a, cf[C_E1R], cf[C_E1I], h.Pb);
    a = cmac(a, cf[C_E2R], cf[C_E2I], h.dF);
    a = rmac(a, cf[C_EP], Dp);
    a = rmac(a, cf[C_EM], D1);
    a = cmac(a, cf[C_E3R], cf[C_E3I], h.Fb);
    r.hP = a;
    return r;
}

// ---------------------------------------------------------------- extraction
// Waveform record between the nodes i_e (a) and i_e + 1 (b): (1 - f) a + f b, written with
// explicit roundings so that every kernel that records a level rounds it the same way.
__device__ __forceinline__ double2 wave_lerp(double2 a, double2 b, double f) {
    const double g = 1.0 - f;
    return make_double2(__fma_rn(f, b.x, __dmul_rn(g, a.x)), __fma_rn(f, b.y, __dmul_rn(g, a.y)));
}

// ---------------------------------------------------------------- corrector
// Exchange entry of one row for the corrector's theta neighbours: Hs (the first two of the
// entry's four floats).  Row j sits at entry j + 1 of its column's buffer; entries 0 and
// n_theta + 1 hold the ghost rows of the pole rule, g Hs of the pole row.
// xb: the column's buffer, mine = xb + 4 (j + 1).
__device__ __forceinline__ void xpublish(float* xb, float* mine, const CRow<float>& row, float g, bool row_ok,
                                         bool top, bool bot) {
    if (row_ok) *(float2*)mine = make_float2(row.Hs.re, row.Hs.im);
    if (top) *(float2*)(mine + 4) = make_float2(g * row.Hs.re, g * row.Hs.im);
    if (bot) *(float2*)xb = make_float2(g * row.Hs.re, g * row.Hs.im);
}

// Read the entries of the rows above and below (after the barrier that follows xpublish).
__device__ __forceinline__ void xread(const float* mine, Cx<float>& Hs_p, Cx<float>& Hs_m) {
    const float2 a = *(const float2*)(mine + 4), b = *(const float2*)(mine - 4);
    Hs_p = {a.x, a.y};
    Hs_m = {b.x, b.y};
}

// Eq. (14) at one node as increments (dPhi, dPi) from the row's combined half-node values,
// the theta neighbours' exchange entries, the node's coefficients cf and source term.
template <class P>
__device__ __forceinline__ void corrector_incr(const CRow<typename P::T>& row, Cx<typename P::T> Hs_p,
                                               Cx<typename P::T> Hs_m, const typename P::T* cf, typename P::T qdt,
                                               Cx<typename P::T> srcc, Cx<typename P::T>& dPhi,
                                               Cx<typename P::T>& dPi) {
    using C = Cx<typename P::T>;
    // second (negated) and two-cell differences of 4 u~
    const C Dplus = sadd(-2.f, (Hs_p - row.Hs) - (row.Hs - Hs_m), row.DpS);
    const C Dminus = sadd(2.f, Hs_p - Hs_m, row.D1S);
    dPhi = rmac(rmac(C::zero(), -cf[C_G], row.dFc), qdt, row.PC);
    dPi = rmac(srcc, cf[C_G], row.dPc);
    dPi = cmac(dPi, cf[C_E1R], cf[C_E1I], row.PC);
    dPi = cmac(dPi, cf[C_E2R], cf[C_E2I], row.dFc);
    dPi = rmac(dPi, cf[C_EP], Dplus);
    dPi = rmac(dPi, cf[C_EM], Dminus);
    dPi = cmac(dPi, cf[C_E3R], cf[C_E3I], row.FC);
}

// ---------------------------------------------------------------- source
// dt_sub A_n e^{-i (omega t + phase0)} at t = t_n + off * dt: the predictor's factor
// (off = 0, dt_sub = dt/2) or the corrector's (off = 1/2, dt_sub = dt); for a moving
// particle dt_sub A e^{-i m phi_p} of the step's sample (the Gaussian is tabulated)
template <bool kMov>
__device__ __forceinline__ double2 source_factor(const InstDev& d, int64_t step, double off,
                                                 double dt_sub) {
    if constexpr (kMov) {
        if (d.src.moving) {   // sample 2n (off = 0) or 2n + 1 (off = 1/2) of a sampled path
            if (step >= d.src.n_traj) return make_double2(0.0, 0.0);
            const double2 A = d.src.amp[2 * step + (off == 0.0 ? 0 : 1)];
            return make_double2(dt_sub * A.x, dt_sub * A.y);
        }
    }
    double A = (d.src.amps != nullptr && step < d.src.n_amps) ? d.src.amps[step] : 1.0;
    double t = (double)step * d.dt;
    double sn, cs;
    sincos(d.src.omega * (t + off * d.dt) + d.src.phase0, &sn, &cs);
    double h = dt_sub * A;
    return make_double2(h * cs, -h * sn);
}

// tau at a window node: factor (A e^{-i(omega t + phase0)} and the sub-step's share of
// dt) times the profile, from the column-major copy in the arithmetic type
template <typename T> struct V2T;
template <> struct V2T<float> { using V = float2; };
template <> struct V2T<double> { using V = double2; };
struct DFC { DF x, y; };   // complex double-float as stored: x.hi, x.lo, y.hi, y.lo
template <> struct V2T<DF> { using V = DFC; };

template <typename T>
__device__ __forceinline__ Cx<T> source_at(const void* q, int stride, Cx<T> fac, int a, int b) {
    const typename V2T<T>::V p = ((const typename V2T<T>::V*)q)[(size_t)a * stride + b];
    return {fac.re * p.x - fac.im * p.y, fac.re * p.y + fac.im * p.x};
}

template <typename T>
__device__ __forceinline__ Cx<T> source_half(const SourceDev& s, Cx<T> fac, int i, int j) {
    int a = i - s.h_lo, b = j - s.j_lo;
    if ((unsigned)a < (unsigned)s.nh && (unsigned)b < (unsigned)s.nj)
        return source_at<T>(s.Q_half, s.q_stride, fac, a, b);
    return Cx<T>::zero();
}

template <typename T>
__device__ __forceinline__ Cx<T> source_int(const SourceDev& s, Cx<T> fac, int i, int j) {
    int a = i - s.i_lo, b = j - s.j_lo;
    if ((unsigned)a < (unsigned)s.ni && (unsigned)b < (unsigned)s.nj)
        return source_at<T>(s.Q_int, s.q_stride, fac, a, b);
    return Cx<T>::zero();
}

}  // namespace teuk
