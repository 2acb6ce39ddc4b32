// teuk_adjoint.cu -- transpose of one Lax-Wendroff step (Eqs. 13-14), as gathers.
//
// The step is affine and complex-linear in u:  u^{n+1} = P (u^n + C(H u^n)) + A_n s_n,
// with H the predictor of Eq. (13) (integer nodes -> half nodes), C the corrector
// increment of Eq. (14) (half nodes -> integer nodes) and P the radial boundary
// condition (zero at i = 0 and i = n_rstar - 1).  With the real inner product
// <x, y> = sum Re(conj(x) y), the transpose of y += c x is x += conj(c) y.  So one
// reverse step is
//   lam'  = P lam^{n+1}
//   mu    = C^T lam'                       (half nodes)
//   lam^n = lam' + H^T mu + E^T gbar_n     (integer nodes), all in one reverse-step kernel
// and the source enters the gradients as
//   dL/dA_n  = <mu_Pi, (dt/2) e_p P_half> + <lam'_Pi, dt e_c P_int>
//   dL/dr0  += A_n (<mu_Pi, (dt/2) d(e_p P_half)/dr0> + <lam'_Pi, dt d(e_c P_int)/dr0>)
// with e_p = e^{-i(omega t_n + phase0)}, e_c the same at t_n + dt/2 (the step stores
// mu_Pi and lam'_Pi over the source window; adj_src_grad_kernel forms the sums).
// Coefficients (g, E1, E2, ep, em, E3, scaled as in teuk_setup.cu) are read from the 2D
// tables for FP64 and double-float instances and formed from the 1D tables, as the
// forward kernels form them, for FP32 instances; in
// the corrector's angular term  ep Phi~(j+1) + em Phi~(j-1) + (E3 - ep - em) Phi~(j)
// the ghost rows fold back onto rows 0 and n_theta-1 with the sign of the pole
// condition.  The co-state lam and mu are FP64 for FP64 instances; for FP32 instances
// they are FP32, lam compensated like the forward state (value hi - c, each step's
// increment added with Kahan's compensated sum), the gradient sums FP64 either way.
#include <algorithm>
#include <type_traits>

#include "teuk_df.cuh"
#include "teuk_internal.cuh"
#include "teuk_step_common.cuh"

namespace teuk {

template <typename R>
struct Z { R x, y; };
template <typename R>
__device__ __forceinline__ Z<R> zadd(Z<R> a, Z<R> b) { return {a.x + b.x, a.y + b.y}; }
template <typename R>
__device__ __forceinline__ Z<R> zscale(R s, Z<R> a) { return {s * a.x, s * a.y}; }

template <typename R> struct R2T;
template <> struct R2T<double> { using V = double2; };
template <> struct R2T<float> { using V = float2; };

template <typename R>
__device__ __forceinline__ Z<R> ldv(const void* p, size_t o) {
    const typename R2T<R>::V a = ((const typename R2T<R>::V*)p)[o];
    return {a.x, a.y};
}
template <typename R>
__device__ __forceinline__ void stv(void* p, size_t o, Z<R> z) {
    ((typename R2T<R>::V*)p)[o] = {z.x, z.y};
}
// Row j of a record's cotangent (n_theta values: the padding rows of a column have none)
template <typename R>
__device__ __forceinline__ Z<R> gld(const InstDev& d, const double2* gbar, int j) {
    if (!TK_IN(d.status, j, d.nth)) return {0, 0};
    const double2 a = gbar[j];
    return {(R)a.x, (R)a.y};
}

// Coefficients as FP64: all of node (i, j), or coefficient k alone
template <typename T>
__device__ __forceinline__ double as64(T v) {
    if constexpr (std::is_same<T, DF>::value) return v.to_double();
    else return v;
}
template <typename T>
__device__ __forceinline__ void adj_coefs(const void* tab, int pitch, int i, int j, double* c) {
    T v[kNCoef];
    load_coefs<T>(tab, pitch, i, j, v);
#pragma unroll
    for (int k = 0; k < kNCoef; ++k) c[k] = as64(v[k]);
}
template <typename T>
__device__ __forceinline__ double adj_coef(const void* tab, int pitch, int i, int j, int k) {
    return as64(((const T*)tab)[coef_index(pitch, i, j, k)]);
}

// lam = E^T gbar (the start of the reverse sweep).
template <typename R>
__global__ void adj_init_kernel(InstDev d, const double2* gbar, CoLevel out) {
    int j = blockIdx.y * blockDim.x + threadIdx.x;   // theta row
    int i = blockIdx.x;                              // r* column
    if (j >= d.pitch || i >= d.nr) return;
    size_t o = node_index(d, i, j);
    Z<double> a = {0, 0};
    if (gbar && j < d.nth && i == d.i_e) a = zscale(1.0 - d.f_e, gld<double>(d, gbar, j));
    if (gbar && j < d.nth && i == d.i_e + 1) a = zscale(d.f_e, gld<double>(d, gbar, j));
    if constexpr (sizeof(R) == 4) {
        ((float4*)out.F)[o] = make_float4((float)a.x, (float)a.y, 0.f, 0.f);
        ((float4*)out.Fc)[o] = make_float4(0.f, 0.f, 0.f, 0.f);
    } else {
        stv<R>(out.F, o, Z<R>{(R)a.x, (R)a.y});
        stv<R>(out.P, o, Z<R>{0, 0});
    }
}

// ------------------------------------------------------------------ fused reverse step
// One reverse step in one pass over the grid: lam^n = P lam^{n+1} + H^T (C^T P lam^{n+1})
// + E^T gbar.  A block holds one theta column (one thread a row) and streams along r*
// over a strip of output columns [c0, c1): at half node h it forms mu(h) = C^T lam' from
// the integer columns h and h+1 (the angular neighbours of lam'_Pi through shared
// memory), then lam^n(h) = H^T mu from the half nodes h-1 and h (the angular neighbours
// of mu_Pi through shared memory), so neither mu nor lam' is written to memory.  Over the
// source window the step also stores mu_Pi (half nodes) and lam'_Pi (integer nodes) into
// one slot of a ring, from which adj_src_grad_kernel forms the source gradients of many
// steps at once, off the step's critical path.

// Real arithmetic of the FP64 reverse step: every operation a DFMA (DADD and DMUL take 19
// clocks of the SM's FP64 pipe, DFMA 16; `one` is a factor the compiler cannot see).
struct AdjLin {
    using Zd = Z<double>;
    double one;
    __device__ __forceinline__ double sum(double a, double b) const { return __fma_rn(a, one, b); }
    __device__ __forceinline__ Zd add(Zd a, Zd b) const { return {sum(a.x, b.x), sum(a.y, b.y)}; }
    __device__ __forceinline__ Zd sub(Zd a, Zd b) const {
        return {__fma_rn(b.x, -one, a.x), __fma_rn(b.y, -one, a.y)};
    }
    // s a + b
    __device__ __forceinline__ Zd mac(Zd b, double s, Zd a) const { return {__fma_rn(s, a.x, b.x), __fma_rn(s, a.y, b.y)}; }
    // conj(cr + i ci) a + b
    __device__ __forceinline__ Zd cmac(Zd b, double cr, double ci, Zd a) const {
        return {__fma_rn(cr, a.x, __fma_rn(ci, a.y, b.x)), __fma_rn(cr, a.y, __fma_rn(-ci, a.x, b.y))};
    }
};

// b + Th^T l at row j, Th the angular and zero-order part of one sub-step, ep (F_{j+1} - F_j)
// - em (F_j - F_{j-1}) + E3 F with the ghost rows of the pole rule (flip: flip_sign of its
// factor); c: the node's coefficients; lm, l, lp: l at the rows j-1, j, j+1.
template <typename T>
__device__ __forceinline__ Z<double> theta_cot(const AdjLin& A, Z<double> b, const double* c, const void* tab,
                                               int pitch, int i, int j, int nth, Z<double> lm, Z<double> l,
                                               Z<double> lp, int flip) {
    b = A.cmac(b, __fma_rn(c[C_EM], -A.one, __fma_rn(c[C_EP], -A.one, c[C_E3R])), c[C_E3I], l);
    const bool lo = j >= 1, hi = j + 1 < nth;
    b = A.mac(b, lo ? adj_coef<T>(tab, pitch, i, j - 1, C_EP) : flip_sign(c[C_EM], flip), lo ? lm : l);
    return A.mac(b, hi ? adj_coef<T>(tab, pitch, i, j + 1, C_EM) : flip_sign(c[C_EP], flip), hi ? lp : l);
}

// The FP64 co-state of one node.
struct CoNode { Z<double> F, P; };

// Source gradients of step n.  With e = e^{-i phi} the phase of a sub-step and
// de = d e / d r0,
//   dL/dA_n  = Re( (dt/2) e_p S_h + dt e_c S_i ),
//   dL/dr0  += A_n Re( (dt/2) (de_p S_h + e_p S'_h) + dt (de_c S_i + e_c S'_i) ),
// where S_h = sum conj(mu_Pi) P_half and S'_h = sum conj(mu_Pi) dP_half over the
// half-node window, S_i and S'_i the same with lam'_Pi over the integer-node window
// (zero off the interior columns).  One block a step: the steps k0 .. k0 + count - 1 of
// a sweep (absolute step step0 + k); ring slot k % slots holds the step's half-node
// window ([nj][nh]) followed by its integer-node window ([nj][ni]).  Each
// thread sums its nodes (t, t + blockDim, ...) in FP64, the threads are added in a fixed
// tree, so the result does not depend on the scheduling.
constexpr int kSrcGradThreads = 256;

template <typename R>
__global__ void __launch_bounds__(kSrcGradThreads) adj_src_grad_kernel(InstDev d, int64_t step0, int64_t k0,
                                                                       int slots, const void* ring,
                                                                       double* gA, double* gR) {
    using V = typename R2T<R>::V;
    const SourceDev& s = d.src;
    const int64_t k = k0 + blockIdx.x, n = step0 + k;
    const size_t nhw = (size_t)s.nh * s.nj, niw = (size_t)s.ni * s.nj;
    const V* Hw = (const V*)ring + (size_t)(k % slots) * (nhw + niw);
    const V* Iw = Hw + nhw;
    double acc[8] = {0, 0, 0, 0, 0, 0, 0, 0};   // S_h, S'_h, S_i, S'_i (re, im)
    for (size_t q = threadIdx.x; q < nhw; q += blockDim.x) {
        const V m = Hw[q];
        const double lx = (double)m.x, ly = (double)m.y;
        const double2 P = s.P_half[q], dP = s.dP_half[q];
        acc[0] += lx * P.x + ly * P.y;
        acc[1] += lx * P.y - ly * P.x;
        acc[2] += lx * dP.x + ly * dP.y;
        acc[3] += lx * dP.y - ly * dP.x;
    }
    for (size_t q = threadIdx.x; q < niw; q += blockDim.x) {
        const V m = Iw[q];
        const double lx = (double)m.x, ly = (double)m.y;
        const double2 P = s.P_int[q], dP = s.dP_int[q];
        acc[4] += lx * P.x + ly * P.y;
        acc[5] += lx * P.y - ly * P.x;
        acc[6] += lx * dP.x + ly * dP.y;
        acc[7] += lx * dP.y - ly * dP.x;
    }
    __shared__ double wred[kSrcGradThreads / 32][8];
    __shared__ double S[8];
    __shared__ Z<double> ph[4];   // e_p, e_c, de_p, de_c
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
#pragma unroll
    for (int v = 0; v < 8; ++v) {
        double x = acc[v];
        for (int off = 16; off > 0; off >>= 1) x += __shfl_down_sync(0xffffffffu, x, off);
        if (lane == 0) wred[warp][v] = x;
    }
    __syncthreads();
    if (t < 8) {
        double x = 0.0;
        for (int w = 0; w < kSrcGradThreads / 32; ++w) x += wred[w][t];
        S[t] = x;
    }
    if (t == 64 || t == 96) {   // the two sub-step phases, on two other warps
        const double tt = (double)n * d.dt + (t == 64 ? 0.0 : 0.5 * d.dt);
        double sn, cs;
        sincos(s.omega * tt + s.phase0, &sn, &cs);
        const double kk = tt * s.domega + s.dphase0;   // e = (cos, -sin); de = -i k e
        const Z<double> e = {cs, -sn};
        ph[t == 64 ? 0 : 1] = e;
        ph[t == 64 ? 2 : 3] = Z<double>{kk * e.y, -kk * e.x};
    }
    __syncthreads();
    if (t != 0) return;
    const double A = (s.amps != nullptr && n < s.n_amps) ? s.amps[n] : 1.0;
    auto re_mul = [](Z<double> a, double bx, double by) { return a.x * bx - a.y * by; };
    const double hd = d.dt;   // (the window holds the cotangent of 2 h_Pi)
    gA[k] = hd * re_mul(ph[0], S[0], S[1]) + d.dt * re_mul(ph[1], S[4], S[5]);
    gR[k] = A * (hd * (re_mul(ph[2], S[0], S[1]) + re_mul(ph[0], S[2], S[3])) +
                 d.dt * (re_mul(ph[3], S[4], S[5]) + re_mul(ph[1], S[6], S[7])));
}

// Programmatic dependent launch of consecutive reverse steps: a block releases the next
// step's launch on entry; the next step's blocks set up what depends only on constant
// data and wait (griddepcontrol.wait: the previous grid has completed and its writes are
// visible) before they read the co-state or write anything to global memory.
__device__ __forceinline__ void adj_release_next() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void adj_wait_prev() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

// kMaxT: the largest block this instance serves (256: columns of up to 256 rows, with
// the register budget of several blocks per SM; 512: up to 512 rows, one block per SM;
// 1024: taller columns)
//
// The FP64 co-state (FP64 and double-float instances).  Bound by the FP64 pipe, so the
// cotangents of the undivided sums of the forward step (predict_x, correct_x) are formed
// once a node and once a half node and shared by the two neighbours they enter:
//   node i, l = lam':       cS = Th^T l_Pi, cD = -G l_Phi + conj(E2) l_Pi,
//                           cSP = (dt/4) l_Phi + conj(E1) l_Pi, cDP = G l_Pi
//     mu_Phi += cS +- cD, mu_Pi += cSP +- cDP  at the half nodes right (+) and left (-) of i
//   half node h, mu:        cs = mu_Phi + Th^T mu_Pi, cd = -G mu_Phi + conj(E2) mu_Pi,
//                           csP = (dt/2) mu_Phi + mu_Pi + conj(E1) mu_Pi, cdP = G mu_Pi
//     lam_Phi += cs +- cd, lam_Pi += csP +- cdP  at the nodes right (+) and left (-) of h
// 76 FP64 operations a node instead of 190 (4096 x 128: 195 -> 89 us a reverse step, double-float
// instances 360 -> 161).  mu here is the cotangent of
// 2 h (adj_src_grad_kernel has the factor).
template <typename T, int kMaxT>
__global__ void __launch_bounds__(kMaxT) adj_step_kernel(InstDev d, CoLevel lin, const double2* gbar,
                                                         CoLevel lout, void* wh, void* wi) {
    using Zd = Z<double>;
    extern __shared__ __align__(16) unsigned char adj_smem[];
    adj_release_next();
    Zd* LB = (Zd*)adj_smem;                    // [2][pitch] lam'_Pi of a column
    Zd* MB = LB + 2 * (size_t)d.pitch;         // [2][pitch] mu_Pi of a half node
    const int j = threadIdx.x, nth = d.nth, nr = d.nr, pitch = d.pitch;
    const bool row_ok = j < nth;
    // output columns [c0, c1): one of gridDim.x pieces of equal length to a column
    const int c0 = (int)((int64_t)blockIdx.x * nr / gridDim.x), c1 = (int)((int64_t)(blockIdx.x + 1) * nr / gridDim.x);
    const double hdt = d.hdt, qdt = d.qdt;
    const int flip = pole_flip(d);
    const AdjLin A{d.one};
    const SourceDev& s = d.src;
    const Zd zero = {0, 0};
    // wh, wi: this step's ring slot of the window co-states (null: no source)
    // lam' = P lam^{n+1} at column col (zero at the boundary columns and outside)
    auto lam_at = [&](int col) {
        CoNode z{};
        if (row_ok && col >= 1 && col <= nr - 2) {
            const size_t o = node_index(d, col, j);
            z = CoNode{ldv<double>(lin.F, o), ldv<double>(lin.P, o)};
        }
        return z;
    };
    auto nb3 = [&](const Zd* buf, int sl, Zd& lm, Zd& lp) {
        const Zd* b = buf + (size_t)sl * pitch;
        lm = j >= 1 ? b[j - 1] : zero;
        lp = j + 1 < nth ? b[j + 1] : zero;
    };
    // shares of node col (co-state L, its Pi part exchanged) of the half nodes to its right
    // (rF, rP) and left (lF, lP)
    auto node_shares = [&](const CoNode& L, int col, Zd& rF, Zd& rP, Zd& lF, Zd& lP) {
        rF = rP = lF = lP = zero;
        if (!row_ok || col < 1 || col > nr - 2) return;
        double c[kNCoef];
        adj_coefs<T>(d.coef_i, pitch, col, j, c);
        Zd lm, lp;
        nb3(LB, col & 1, lm, lp);
        const Zd cS = theta_cot<T>(A, zero, c, d.coef_i, pitch, col, j, nth, lm, L.P, lp, flip);
        const Zd cD = A.cmac(A.mac(zero, -c[C_G], L.F), c[C_E2R], c[C_E2I], L.P);
        const Zd cSP = A.cmac(A.mac(zero, qdt, L.F), c[C_E1R], c[C_E1I], L.P);
        const Zd cDP = A.mac(zero, c[C_G], L.P);
        rF = A.add(cS, cD);
        lF = A.sub(cS, cD);
        rP = A.add(cSP, cDP);
        lP = A.sub(cSP, cDP);
    };
    adj_wait_prev();
    // prologue: column c0 - 1
    CoNode l_cur = lam_at(c0 - 1), l_next;
    LB[(size_t)((c0 - 1) & 1) * pitch + j] = l_cur.P;
    __syncthreads();
    Zd muF_part, muP_part, aF_part = zero, aP_part = zero, x, y;
    node_shares(l_cur, c0 - 1, muF_part, muP_part, x, y);
    for (int h = c0 - 1; h <= c1 - 1; ++h) {
        // column h+1: lam' and its shares; mu at half node h
        l_next = lam_at(h + 1);
        LB[(size_t)((h + 1) & 1) * pitch + j] = l_next.P;
        __syncthreads();
        Zd muF_next, muP_next, muF, muP;
        node_shares(l_next, h + 1, muF_next, muP_next, muF, muP);
        const bool half_ok = row_ok && h >= 0 && h <= nr - 2;
        muF = half_ok ? A.add(muF_part, muF) : zero;
        muP = half_ok ? A.add(muP_part, muP) : zero;
        if (wh && half_ok && h >= c0) {   // half-node window: the cotangent of h_Pi (half node c0 - 1 is
                                          // the previous block's)
            const int a = h - s.h_lo, bb = j - s.j_lo;
            if ((unsigned)a < (unsigned)s.nh && (unsigned)bb < (unsigned)s.nj)
                stv<double>(wh, (size_t)bb * s.nh + a, muP);
        }
        MB[(size_t)(h & 1) * pitch + j] = muP;
        __syncthreads();
        // the shares of half node h of the nodes h (left) and h+1 (right)
        Zd tF = zero, tP = zero, nF = zero, nP = zero;
        if (half_ok) {
            double c[kNCoef];
            adj_coefs<T>(d.coef_h, pitch, h, j, c);
            Zd mm, mp;
            nb3(MB, h & 1, mm, mp);
            const Zd cs = theta_cot<T>(A, muF, c, d.coef_h, pitch, h, j, nth, mm, muP, mp, flip);
            const Zd cd = A.cmac(A.mac(zero, -c[C_G], muF), c[C_E2R], c[C_E2I], muP);
            const Zd csP = A.cmac(A.mac(muP, hdt, muF), c[C_E1R], c[C_E1I], muP);
            tF = A.sub(cs, cd);
            nF = A.add(cs, cd);
            tP = A.mac(csP, -c[C_G], muP);
            nP = A.mac(csP, c[C_G], muP);
        }
        // lam^n at column h
        if (h >= c0 && row_ok) {
            const size_t o = node_index(d, h, j);
            const bool interior = h >= 1 && h <= nr - 2;
            Zd aF = A.add(aF_part, tF), aP = A.add(aP_part, tP);
            if (interior) {
                aF = A.add(l_cur.F, aF);
                aP = A.add(l_cur.P, aP);
            }
            if (TK_IN(d.status, o, plane_elems(d))) {
                stv<double>(lout.F, o, aF);
                stv<double>(lout.P, o, aP);
            }
            if (wi) {   // integer-node window: lam'_Pi (zero off the interior columns)
                const int a = h - s.i_lo, bb = j - s.j_lo;
                if ((unsigned)a < (unsigned)s.ni && (unsigned)bb < (unsigned)s.nj)
                    stv<double>(wi, (size_t)bb * s.ni + a, interior ? l_cur.P : zero);
            }
        }
        l_cur = l_next;
        muF_part = muF_next;
        muP_part = muP_next;
        aF_part = nF;
        aP_part = nP;
    }
    // transpose of the linear extraction between i_e and i_e + 1, added to this row's own
    // values (in the loop its operations would run, predicated off, at every column)
    if (gbar && row_ok) {
        for (int e = 0; e < 2; ++e) {
            const int col = d.i_e + e;
            const size_t o = node_index(d, col, j);
            if (col < c0 || col >= c1 || !TK_IN(d.status, o, plane_elems(d))) continue;
            const double w = e ? d.f_e : 1.0 - d.f_e;
            const Zd gb = gld<double>(d, gbar, j);
            stv<double>(lout.F, o, zadd(ldv<double>(lout.F, o), zscale(w, gb)));
        }
    }
}

// The FP32 co-state (FP32 and FP32-Kahan instances): the same shares as in the FP64 kernel,
// with the coefficients formed in registers from 1D tables (form_coefs2; the adjoint's own
// tables carry the powers of two, ep = A + B and em = A - B turn the split angular form back),
// i.e. the coefficients that the forward FP32 kernels compute, and the co-state compensated
// like the forward state (value v - c, two planes of {Phi, Pi}).  Bound by instruction issue:
// each column's coefficients are formed once and each node's and half node's shares once, the
// rows exchange the products ep l and em l instead of l and their coefficients, and complex
// sums run in paired instructions.  4096 x 128: 13.7 -> 10.0 us a reverse step (10.7 with the cotangents' upload); 400 instructions a
// node instead of 588.
struct CfF { float g, e1r, e1i, e2r, e2i, ep, em, e3r, e3i; };

// columns of radial tables the FP32 reverse step stages in shared memory (pieces of up
// to kAdjRtCols - 2 columns; longer ones read the tables from global memory)
constexpr int kAdjRtCols = 64;

__device__ __forceinline__ Cx<float> conj_mac(Cx<float> b, float cr, float ci, Cx<float> a) {
    return {__fmaf_rn(cr, a.re, __fmaf_rn(ci, a.im, b.re)), __fmaf_rn(cr, a.im, __fmaf_rn(-ci, a.re, b.im))};
}

template <int kMaxT>
__global__ void __launch_bounds__(kMaxT) adj_step_kernel_f32(InstDev d, CoLevel lin, const double2* gbar,
                                                             CoLevel lout, void* wh, void* wi) {
    using C = Cx<float>;
    extern __shared__ __align__(16) unsigned char adj_smem[];
    adj_release_next();
    const int j = threadIdx.x, nth = d.nth, nr = d.nr, pitch = d.pitch;
    float4* LB = (float4*)adj_smem;                 // [2][pitch] {ep l, em l} of a column, l = lam'_Pi
    float4* MB = LB + 2 * (size_t)pitch;            // [2][pitch] the same of a half node, l = mu_Pi
    RTab2* RT = (RTab2*)(MB + 2 * (size_t)pitch);   // radial tables of columns c0-1 .. c1
    const bool row_ok = j < nth, lo_ok = j >= 1, hi_ok = j + 1 < nth;
    // output columns [c0, c1): one of gridDim.x pieces of equal length to a column
    const int c0 = (int)((int64_t)blockIdx.x * nr / gridDim.x), c1 = (int)((int64_t)(blockIdx.x + 1) * nr / gridDim.x);
    const bool rt_smem = c1 - c0 + 2 <= kAdjRtCols;
    const float hdt = d.hdt2.x, qdt = d.qdt2.x;
    const int flip = pole_flip(d);
    const SourceDev& s = d.src;
    const C zero = C::zero();
    // wh, wi: this step's ring slot of the window co-states (null: no source)
    RowTab<PK> rt;
    rt.load(d.thtab_a, j, row_ok);
    // a column as stored, loaded one column ahead of use (zero off the interior columns); plain
    // loads: the previous reverse step may still write these planes while this block is set up,
    // so they are not read-only for the kernel's life and must stay behind adj_wait_prev
    struct Node { C vF, vP, cF, cP; };
    auto load = [&](int col) {
        Node n{zero, zero, zero, zero};
        if (row_ok && col >= 1 && col <= nr - 2) {
            const size_t o = node_index(d, col, j);
            const float4 v = ((const float4*)lin.F)[o], c = ((const float4*)lin.Fc)[o];
            n = Node{{v.x, v.y}, {v.z, v.w}, {c.x, c.y}, {c.z, c.w}};
        }
        return n;
    };
    // coefficients of column col: node col (ci) and half node col+1/2 (ch)
    auto form = [&](int col, CfF& ci, CfF& ch) {
        float2 cf[kNCoef];
        if (col >= 0 && col <= nr - 1) {
            form_coefs2(rt_smem ? RT[col - (c0 - 1)] : d.rtab_a[col], rt.t, cf);
        } else {
#pragma unroll
            for (int q = 0; q < kNCoef; ++q) cf[q] = make_float2(0.f, 0.f);
        }
        const float2 ep = __fadd2_rn(cf[C_EP], cf[C_EM]), em = p_sub(cf[C_EP], cf[C_EM]);
        ch = CfF{cf[C_G].x, cf[C_E1R].x, cf[C_E1I].x, cf[C_E2R].x, cf[C_E2I].x, ep.x, em.x, cf[C_E3R].x, cf[C_E3I].x};
        ci = CfF{cf[C_G].y, cf[C_E1R].y, cf[C_E1I].y, cf[C_E2R].y, cf[C_E2I].y, ep.y, em.y, cf[C_E3R].y, cf[C_E3I].y};
    };
    // this row's products ep l and em l, published for the rows above and below
    auto publish = [&](float4* x, const CfF& c, C l) {
        const float4 p = make_float4(c.ep * l.re, c.ep * l.im, c.em * l.re, c.em * l.im);
        x[j] = p;
        return p;
    };
    // b + Th^T l from this row's products p and the neighbours' in x, as differences: a product
    // enters its own row and its neighbour's with opposite signs and the same rounding
    auto theta = [&](C b, const CfF& c, const float4* x, float4 p, C l) {
        const C ep = {p.x, p.y}, em = {p.z, p.w};
        C lo = flip_sign(em, flip), hi = flip_sign(ep, flip);
        if (lo_ok) lo = up(*(const float2*)(x + j - 1));
        if (hi_ok) hi = up(*((const float2*)(x + j + 1) + 1));
        return conj_mac(b, c.e3r, c.e3i, l) + ((lo - ep) + (hi - em));
    };
    // shares of node col (co-state lF, lP) of the half nodes to its right (rF, rP) and left (xF, xP)
    auto node_shares = [&](const CfF& c, const float4* x, float4 p, C lF, C lP, int col, C& rF, C& rP, C& xF, C& xP) {
        rF = rP = xF = xP = zero;
        if (!row_ok || col < 1 || col > nr - 2) return;
        const C cS = theta(zero, c, x, p, lP);
        const C cD = conj_mac(rmac(zero, -c.g, lF), c.e2r, c.e2i, lP);
        const C cSP = conj_mac(rmac(zero, qdt, lF), c.e1r, c.e1i, lP);
        rF = cS + cD;
        xF = cS - cD;
        rP = rmac(cSP, c.g, lP);
        xP = rmac(cSP, -c.g, lP);
    };
    // the piece's radial tables into shared memory (one broadcast read per column later)
    if (rt_smem) {
        const int ncols = c1 - c0 + 2;
        for (int q = threadIdx.x; q < ncols * 8; q += blockDim.x) {
            const int k = q >> 3, col = c0 - 1 + k;
            if (col >= 0 && col <= nr - 1) ((float4*)(RT + k))[q & 7] = __ldg((const float4*)(d.rtab_a + col) + (q & 7));
        }
        __syncthreads();
    }
    adj_wait_prev();
    // the record's cotangent and the extraction weights, once (column -2: no record)
    const int ie = gbar ? d.i_e : -2;
    float we = 0.f, we1 = 0.f;
    C gb = zero;
    if (gbar && row_ok && c0 <= ie + 1 && ie < c1) {
        const Z<float> g = gld<float>(d, gbar, j);
        gb = {g.x, g.y};
        we = (float)(1.0 - d.f_e);
        we1 = (float)d.f_e;
    }
    // prologue: column c0 - 1
    Node cur = load(c0 - 1), next = load(c0);
    C lF = cur.vF - cur.cF, lP = cur.vP - cur.cP;
    CfF ci, ch_cur, ch_n;
    form(c0 - 1, ci, ch_cur);
    float4 p = publish(LB + (size_t)((c0 - 1) & 1) * pitch, ci, lP);
    __syncthreads();
    C muF_part, muP_part, aF_part = zero, aP_part = zero, xF, xP;
    node_shares(ci, LB + (size_t)((c0 - 1) & 1) * pitch, p, lF, lP, c0 - 1, muF_part, muP_part, xF, xP);
    for (int h = c0 - 1; h <= c1 - 1; ++h) {
        // column h+1: lam' and its shares; mu at half node h
        const Node nx = next;
        next = load(h + 2);
        lF = nx.vF - nx.cF;
        const C lP_n = nx.vP - nx.cP;
        float4* lb = LB + (size_t)((h + 1) & 1) * pitch;
        form(h + 1, ci, ch_n);
        p = publish(lb, ci, lP_n);
        __syncthreads();
        C muF_next, muP_next;
        node_shares(ci, lb, p, lF, lP_n, h + 1, muF_next, muP_next, xF, xP);
        const bool half_ok = row_ok && h >= 0 && h <= nr - 2;
        const C muF = half_ok ? muF_part + xF : zero, muP = half_ok ? muP_part + xP : zero;
        if (wh && half_ok && h >= c0) {   // half-node window (half node c0 - 1 is the previous block's)
            const int a = h - s.h_lo, bb = j - s.j_lo;
            if ((unsigned)a < (unsigned)s.nh && (unsigned)bb < (unsigned)s.nj)
                ((float2*)wh)[(size_t)bb * s.nh + a] = pk(muP);
        }
        float4* mb = MB + (size_t)(h & 1) * pitch;
        p = publish(mb, ch_cur, muP);
        __syncthreads();
        // the shares of half node h of the nodes h (left) and h+1 (right)
        C tF = zero, tP = zero, nF = zero, nP = zero;
        if (half_ok) {
            const C cs = theta(muF, ch_cur, mb, p, muP);
            const C cd = conj_mac(rmac(zero, -ch_cur.g, muF), ch_cur.e2r, ch_cur.e2i, muP);
            const C csP = conj_mac(rmac(muP, hdt, muF), ch_cur.e1r, ch_cur.e1i, muP);
            tF = cs - cd;
            nF = cs + cd;
            tP = rmac(csP, -ch_cur.g, muP);
            nP = rmac(csP, ch_cur.g, muP);
        }
        // lam^n at column h
        if (h >= c0 && row_ok) {
            const size_t o = node_index(d, h, j);
            C aF = aF_part + tF;
            const C aP = aP_part + tP;
            if (h == ie) aF = rmac(aF, we, gb);
            if (h == ie + 1) aF = rmac(aF, we1, gb);
            const C lam = cur.vP - cur.cP;   // (lam'_Pi, for the window)
            kahan_add(cur.vF, cur.cF, aF);   // (a column off the interior was loaded as zero)
            kahan_add(cur.vP, cur.cP, aP);
            if (TK_IN(d.status, o, plane_elems(d))) {
                ((float4*)lout.F)[o] = make_float4(cur.vF.re, cur.vF.im, cur.vP.re, cur.vP.im);
                ((float4*)lout.Fc)[o] = make_float4(cur.cF.re, cur.cF.im, cur.cP.re, cur.cP.im);
            }
            if (wi) {   // integer-node window: lam'_Pi (zero off the interior columns)
                const int a = h - s.i_lo, bb = j - s.j_lo;
                if ((unsigned)a < (unsigned)s.ni && (unsigned)bb < (unsigned)s.nj)
                    ((float2*)wi)[(size_t)bb * s.ni + a] = pk(lam);
            }
        }
        cur = nx;
        ch_cur = ch_n;
        muF_part = muF_next;
        muP_part = muP_next;
        aF_part = nF;
        aP_part = nP;
    }
}

// Loss of the built-in |r_ext^3 W|^2: per record, lossrec[k] = r^6 sum_j |W_k[j]|^2 (j
// ascending) and gbar_k = 2 r^6 W_k.  Records are read from a ring (slot level % cap),
// gbar_k is written to slot (g0 + k) % gcap of another.
__global__ void loss_records_kernel(const double2* wave, int64_t cap, int nth, int64_t level0,
                                    int64_t count, double r6, double* lossrec, double2* gbar,
                                    int64_t gcap, int64_t g0) {
    int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (k >= count) return;
    const double2* w = wave + (size_t)((level0 + k) % cap) * nth;
    double2* g = gbar + (size_t)((g0 + k) % gcap) * nth;
    double acc = 0.0;
    for (int j = 0; j < nth; ++j) {
        double2 v = w[j];
        acc += v.x * v.x + v.y * v.y;
        g[j] = make_double2(2.0 * r6 * v.x, 2.0 * r6 * v.y);
    }
    lossrec[k] = r6 * acc;
}

// out = sum of v[0 .. n) in index order (one thread: the order is part of the result).
__global__ void ordered_sum_kernel(const double* v, int64_t n, double* out) {
    if (blockIdx.x != 0 || threadIdx.x != 0) return;
    double acc = 0.0;
    for (int64_t k = 0; k < n; ++k) acc += v[k];
    *out = acc;
}

// ------------------------------------------------------------------ launchers

void launch_adj_init(cudaStream_t st, const InstDev& d, const double2* gbar, const CoLevel& out) {
    dim3 g(d.nr, (d.pitch + 127) / 128);
    if (d.prec == 0 || d.prec == 3) adj_init_kernel<double><<<g, 128, 0, st>>>(d, gbar, out);
    else adj_init_kernel<float><<<g, 128, 0, st>>>(d, gbar, out);
}

// dynamic shared memory of the reverse-step kernels for blocks of `threads` rows
static size_t adj_smem_bytes(int prec, int threads) {
    const bool f32 = prec != 0 && prec != 3;
    return 4 * (size_t)threads * 16 + (f32 ? kAdjRtCols * sizeof(RTab2) : 0);
}

template <class K>
static int adj_resident(K kernel, int threads, size_t smem) {
    int dev = 0, sms = 0, per = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, kernel, threads, smem);
    return (per > 0 ? per : 1) * (sms > 0 ? sms : 1);
}

// f(kernel, dynamic shared memory, rows) with the reverse-step kernel built for blocks of t
// rows (up to 256, 512 or 1024: rows is the build's limit)
template <class F>
static void adj_dispatch(int prec, int t, F f) {
    const int rows = t <= 256 ? 256 : t <= 512 ? 512 : 1024;
    const size_t sm = adj_smem_bytes(prec, t);
    if (prec == 0) {
        if (rows == 256) f(adj_step_kernel<double, 256>, sm, rows);
        else if (rows == 512) f(adj_step_kernel<double, 512>, sm, rows);
        else f(adj_step_kernel<double, 1024>, sm, rows);
    } else if (prec == 3) {
        if (rows == 256) f(adj_step_kernel<DF, 256>, sm, rows);
        else if (rows == 512) f(adj_step_kernel<DF, 512>, sm, rows);
        else f(adj_step_kernel<DF, 1024>, sm, rows);
    } else {
        if (rows == 256) f(adj_step_kernel_f32<256>, sm, rows);
        else if (rows == 512) f(adj_step_kernel_f32<512>, sm, rows);
        else f(adj_step_kernel_f32<1024>, sm, rows);
    }
}

// The cut of the reverse step.  FP64 co-state: a whole number of blocks on every SM, two or
// three of them, each with the same number of columns.  It is bound by the FP64 pipe of
// the SM that has most blocks, and consecutive steps overlap (programmatic dependent
// launch), so that any other number piles the next step's blocks on the SMs that happen to
// be free: 1024 x 64 in 256 strips of 4 columns took 66 us a step, in 304 pieces 20; 2048 x
// 128 in 512 strips 85, in 304 pieces 49; 4096 x 128 in 820 strips 106, in 456 pieces 88 (304:
// 102).  More blocks have more columns at their edges computed twice; two an SM hide too
// little latency once a piece is longer than some six columns.
// FP32 co-state: a piece for every place the GPU has, or, while a piece would have less than
// three columns, half as many places (down to four an SM), capped.  us per step, one wave of
// strips of at least four columns -> this: 512 x 32 6.1 -> 3.7, 1024 x 64 9.4 -> 5.2, 2048 x 128
// 10.0 -> 9.7, 4096 x 64 9.8 -> 9.4, 4096 x 128 14.0 both (with the step then at 588 instructions a node).
AdjCut adj_step_plan(const InstDev& d) {
    int res = 1, dev = 0, sms = 0;
    adj_dispatch(d.prec, d.pitch, [&](auto kernel, size_t sm, int rows) {
        // Tall blocks, and capped ones, take more than the default 48 KB.  The limit belongs to the
        // kernel, not to this context: it is set to what the build's tallest block and its smallest
        // cap take, the same whoever calls, so that no call lowers it under another context's sweep
        cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             (int)capped_smem(4, adj_smem_bytes(d.prec, rows)));
        res = adj_resident(kernel, d.pitch, sm);
    });
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (sms < 1) sms = 1;
    const int places = std::max(1, res / sms);
    if (d.prec == 0 || d.prec == 3) {
        const int per = std::min(places, d.nr >= 6 * 3 * sms ? 3 : 2);
        return {std::max(1, std::min(per * sms, d.nr / 2)), 0};
    }
    int per = places;
    while (per > 4 && d.nr < 3 * per * sms) per = std::max(4, per / 2);
    return {std::min(per * sms, d.nr), per < places ? per : 0};
}

template <class K>
static void adj_launch(cudaStream_t st, K kernel, int nb, int t, size_t sm, const InstDev& d, const CoLevel& lin,
                       const double2* gbar, const CoLevel& lout, void* wh, void* wi) {
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(nb);
    cfg.blockDim = dim3(t);
    cfg.dynamicSmemBytes = sm;
    cfg.stream = st;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    cudaLaunchKernelEx(&cfg, kernel, d, lin, gbar, lout, wh, wi);
}

void launch_adj_step(cudaStream_t st, const InstDev& d, const CoLevel& lin, const double2* gbar,
                     const CoLevel& lout, const AdjCut& cut, void* wh, void* wi) {
    adj_dispatch(d.prec, d.pitch, [&](auto kernel, size_t sm, int) {
        if (cut.cap > 0) sm = capped_smem(cut.cap, sm);
        adj_launch(st, kernel, cut.nb, d.pitch, sm, d, lin, gbar, lout, wh, wi);
    });
}

size_t adj_window_bytes(const InstDev& d) {
    const size_t es = (d.prec == 0 || d.prec == 3) ? sizeof(double2) : sizeof(float2);
    return ((size_t)d.src.nh + d.src.ni) * d.src.nj * es;
}

void launch_adj_src_grad(cudaStream_t st, const InstDev& d, int64_t step0, int64_t k0, int64_t count,
                         int slots, const void* ring, double* gA, double* gR) {
    if (count <= 0) return;
    if (d.prec == 0 || d.prec == 3)
        adj_src_grad_kernel<double><<<(unsigned)count, kSrcGradThreads, 0, st>>>(d, step0, k0, slots, ring, gA, gR);
    else
        adj_src_grad_kernel<float><<<(unsigned)count, kSrcGradThreads, 0, st>>>(d, step0, k0, slots, ring, gA, gR);
}

void launch_loss_records(cudaStream_t st, const double2* wave, int64_t cap, int nth,
                         int64_t level0, int64_t count, double r6, double* lossrec,
                         double2* gbar, int64_t gcap, int64_t g0) {
    loss_records_kernel<<<(unsigned)((count + 127) / 128), 128, 0, st>>>(wave, cap, nth, level0, count, r6,
                                                                        lossrec, gbar, gcap, g0);
}

void launch_ordered_sum(cudaStream_t st, const double* v, int64_t n, double* out) {
    ordered_sum_kernel<<<1, 32, 0, st>>>(v, n, out);
}

}  // namespace teuk
