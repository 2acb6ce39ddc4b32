// teuk_step.cu -- the Lax-Wendroff step (Eqs. 13-14) as one fused kernel per step.
//
// Work decomposition: a thread block holds one whole theta column (thread j = row j,
// blockDim = n_theta rounded up to a warp) and streams along r* over a strip of
// columns [c0, c1).  The columns of u^n arrive in a ring of shared-memory slots, filled
// by bulk-async (TMA) copies several columns ahead of use; at each column the block
// computes the predictor (Eq. 13) at the half node just behind it and the corrector
// (Eq. 14) at the column behind that, and stores u^{n+1}.  Radial neighbours are the
// registers of the previous column; the theta neighbours of the input state (FP32 paths) are
// read from the ring slot, and those of the predictor's results through a small shared
// exchange buffer (one barrier per column).  A strip reads two extra columns, so every
// input is read from HBM about once per step.  The angular ghost
// rows of the pole condition (Sec. 2.2) mirror row 0 / row n_theta-1 with sign +1
// (even |m + s|) or -1 (odd |m + s|): on the averaged state in the predictor, on the half-node
// results in the corrector.
//
// The FP64 and double-float kernels take the expanded form of teuk_step_common.cuh
// (predict_x, correct_x), in which the rows exchange the radial sums s of the next half
// node as well as S, so that no row reads another row's slot entries.
//
// Arithmetic of the FP32 paths, in differences so that the compensated FP32 state keeps its
// accuracy (a difference of two (hi, c) pairs is formed as (hi_a - hi_b) - (c_a - c_b)
// before anything cancels):
//   predictor at (i+1/2, j), with the undivided sums Fb = Phi_i + Phi_{i+1}, Pb of Pi, the
//   differences dF = Phi_{i+1} - Phi_i, dP of Pi, and Dp = -(Fb(j+1) - 2 Fb(j) + Fb(j-1)),
//   D1 = Fb(j+1) - Fb(j-1) formed from the state's own theta differences:
//     dh_Phi = -g dF + (dt/4) Pb
//     dh_Pi  =  g dP + E1 Pb + E2 dF + A Dp + B D1 + E3 Fb + (dt/2) tau(t_n)
//   corrector at (i, j) from the half nodes R = i+1/2, L = i-1/2 (h = Fb/2 + dh):
//     h_R - h_L = (dF_R + dF_L)/2 + dh_R - dh_L,  4 u~ = Fb_R + Fb_L + 2 (dh_R + dh_L),
//     Delta Phi = -g d(h_Phi) + (dt/4) 4 Pi~
//     Delta Pi  =  g d(h_Pi) + E1 4 Pi~ + E2 d(h_Phi) + A D2 + B D1 + E3 4 Phi~ + dt tau(t_n+dt/2)
//     u^{n+1} = u^n + Delta   (Kahan-compensated for the FP32_KAHAN state)
// (D2, D1: the same theta differences of 4 u~), with the scaled coefficients of RTab2, which
// carry the powers of two of the undivided sums; A and B are the split form of the angular
// part (see split_angular).  This is Eqs. (13)-(14) with S_Pi = -c_t Pi + P* Phi_* + w
// Theta[Phi] + q Phi + tau, rearranged, not approximated.
#include <type_traits>

#include "teuk_internal.cuh"
#include "teuk_step_common.cuh"

namespace teuk {

// ---------------------------------------------------------------- column ring
// PTX wrappers: mbarrier and the bulk-async copy global -> shared (TMA, untiled form).
__device__ __forceinline__ unsigned smem_addr(const void* p) {
    return (unsigned)__cvta_generic_to_shared(p);
}
__device__ __forceinline__ void mbar_init(uint64_t* b) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_addr(b)) : "memory");
}
__device__ __forceinline__ void mbar_init_fence() {
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}
__device__ __forceinline__ void mbar_expect_tx(uint64_t* b, unsigned bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_addr(b)),
                 "r"(bytes)
                 : "memory");
}
__device__ __forceinline__ bool mbar_try_wait(uint64_t* b, unsigned parity) {
    unsigned ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(smem_addr(b)), "r"(parity)
        : "memory");
    return ok != 0;
}
__device__ __forceinline__ void bulk_copy_g2s(void* dst, const void* src, unsigned bytes,
                                              uint64_t* b) {
    asm volatile(
        "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
            smem_addr(dst)),
        "l"(src), "r"(bytes), "r"(smem_addr(b))
        : "memory");
}
// Bulk prefetch of a global range into L2 (16-byte aligned, size a multiple of 16).
__device__ __forceinline__ void bulk_prefetch_l2(const void* src, unsigned bytes) {
    asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(src), "r"(bytes) : "memory");
}
// Orders this thread's view of global memory (generic proxy) before its later bulk copies.
__device__ __forceinline__ void fence_proxy_async_global() {
    asm volatile("fence.proxy.async.global;" ::: "memory");
}
// Programmatic dependent launch: wait for the previous grid in the stream (complete and
// its memory visible; a no-op for launches without the attribute), and allow the next
// grid to launch.
__device__ __forceinline__ void griddep_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void griddep_launch_dependents() {
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}
__device__ __forceinline__ unsigned long long global_ns() {
    unsigned long long t;
    asm volatile("mov.u64 %0, %globaltimer;" : "=l"(t));
    return t;
}

constexpr unsigned long long kRingWaitNs = 1000000000ull;  // a slot wait gives up after 1 s

// Columns of the input level (every plane, plus on the FP32 paths the column's radial
// table) are copied into R shared-memory slots by one thread, R - 2 columns
// ahead of use; each slot has an mbarrier that its copy completes.  A column is read
// (own node and theta neighbours) when it arrives and its radial tables one column
// later, so its slot is refilled after the barrier two columns on, when every thread
// has finished with it.  Copies start on 16-byte boundaries with sizes in multiples of
// 16 bytes: a column is n_theta 16-byte nodes at a 512-byte aligned offset, a radial
// table 128 bytes.
template <class P, int R>
struct ColumnRing {
    static constexpr int kSlots = R;
    static constexpr bool kTabs = uses_1d_tables<P>();
    __host__ __device__ static unsigned slot_bytes(int threads) {
        return (unsigned)P::planes * (unsigned)threads * 16u + (kTabs ? (unsigned)sizeof(RTab2) : 0u);
    }

    unsigned char* base;  // R slots: planes [P::planes][stride] of 16-byte nodes, then RTab2
    uint64_t* mbar;       // [R]
    unsigned stride;      // nodes per plane in a slot (the block size)
    unsigned sbytes;
    unsigned phase;       // bit s: parity of the next completion awaited on slot s
    bool late;            // a wait gave up

    __device__ __forceinline__ ColumnRing(unsigned char* b, uint64_t* m)
        : base(b), mbar(m), stride(blockDim.x), sbytes(slot_bytes(blockDim.x)), phase(0), late(false) {}

    // One thread, once per block, before any fill; the block synchronizes afterwards.
    __device__ __forceinline__ void init() const {
        for (int k = 0; k < R; ++k) mbar_init(mbar + k);
        mbar_init_fence();
    }
    __device__ __forceinline__ unsigned char* slot(int s) const { return base + (size_t)s * sbytes; }
    __device__ __forceinline__ Planes<P> planes(int s) const { return Planes<P>::at(slot(s), stride); }
    // One thread: copy column col of buffer bin (and its radial tables) into slot s, and
    // prefetch the column's slices of the source profile into L2 (read once per step,
    // they would otherwise come from DRAM, evicted by the state streaming through L2); kSrc
    // false: the block meets no source (this thread's instructions are on every column's path:
    // FP32-Kahan 8192 x 128 13.8 -> 13.6 us per step).
    template <bool kSrc = true>
    __device__ __forceinline__ void fill(const InstDev& d, int bin, int col, int s) const {
        if (col == d.fault_col) return;   // testing aid: the slot's phase never completes
        if (!TK_IN(d.status, col, d.nr)) return;   // (checked builds; the waiters time out)
        if (kSrc && d.src.on) {
            const SourceDev& w = d.src;
            const unsigned cb = (unsigned)w.q_stride * (unsigned)sizeof(typename V2T<typename P::T>::V);
            const int a = col - w.i_lo, h = col - w.h_lo;
            if ((unsigned)a < (unsigned)w.ni) bulk_prefetch_l2((const char*)w.Q_int + (size_t)a * cb, cb);
            if ((unsigned)h < (unsigned)w.nh) bulk_prefetch_l2((const char*)w.Q_half + (size_t)h * cb, cb);
        }
        unsigned char* dst = slot(s);
        const unsigned nb = (unsigned)d.nth * 16u;
        mbar_expect_tx(mbar + s, P::planes * nb + (kTabs ? (unsigned)sizeof(RTab2) : 0u));
        const size_t off = (size_t)col * (size_t)d.pitch * 16u;
#pragma unroll
        for (int q = 0; q < P::planes; ++q)
            bulk_copy_g2s(dst + q * stride * 16u, (const unsigned char*)d.buf[bin][q] + off, nb, mbar + s);
        if constexpr (kTabs) {
            bulk_copy_g2s(dst + P::planes * stride * 16u, d.rtab + col, sizeof(RTab2), mbar + s);
        }
    }
    // Wait for the next copy into slot s.  Once a wait has given up, the thread waits
    // no more (its results are void and the status word says so).
    __device__ __forceinline__ void wait(int s) {
        const unsigned par = (phase >> s) & 1u;
        phase ^= 1u << s;
        if (mbar_try_wait(mbar + s, par) || late) return;
        const unsigned long long t0 = global_ns();
        while (!mbar_try_wait(mbar + s, par))
            if (global_ns() - t0 > kRingWaitNs) { late = true; return; }
    }
    // Radial table of the column in slot s (FP32 paths).
    __device__ __forceinline__ RTab2 tab2(int s) const {
        RTab2 t{};
        if constexpr (kTabs) {
            const float4* q = (const float4*)(slot(s) + P::planes * stride * 16u);
            float4 v[7];
#pragma unroll
            for (int k = 0; k < 7; ++k) v[k] = q[k];
            t.R2 = {v[0].x, v[0].y};   t.naD = {v[0].z, v[0].w};
            t.Rd = {v[1].x, v[1].y};   t.ctr = {v[1].z, v[1].w};
            t.cti = {v[2].x, v[2].y};  t.ctc = {v[2].z, v[2].w};
            t.pr = {v[3].x, v[3].y};   t.pi = {v[3].z, v[3].w};
            t.nbb = {v[4].x, v[4].y};  t.Ds = {v[4].z, v[4].w};
            t.nDs = {v[5].x, v[5].y};  t.qr = {v[5].z, v[5].w};
            t.qi = {v[6].x, v[6].y};   t.nsdt = {v[6].z, v[6].w};
        }
        return t;
    }
    // After a wait gave up: give every copy still in flight (bounded) time to land, so
    // the block never exits with a copy into its shared memory outstanding.
    __device__ void drain() const {
        const unsigned long long t0 = global_ns();
        for (int k = 0; k < R; ++k)
            while (!mbar_try_wait(mbar + k, ((phase >> k) & 1u) ^ 1u))
                if (global_ns() - t0 > kRingWaitNs) return;
    }
};

// Shared memory of a step block: the ring, then the exchange buffer of the predictor's
// results, [2 (column parity)][threads + 2][4] values (row j at entry j + 1; entries 0
// and n_theta + 1 hold the ghost rows of the pole rule).
template <class P, int R>
struct StepShared {
    using T = typename P::T;
    __host__ __device__ static unsigned xbuf_elems(int threads) { return 2u * ((unsigned)threads + 2u) * 4u; }
    __host__ __device__ static unsigned bytes(int threads) {
        return R * ColumnRing<P, R>::slot_bytes(threads) + xbuf_elems(threads) * (unsigned)sizeof(T);
    }
    __device__ __forceinline__ static T* xbuf(unsigned char* base) {
        return (T*)(base + R * ColumnRing<P, R>::slot_bytes(blockDim.x));
    }
};

// Slots of the ring: six for blocks of up to 512 rows, four for larger blocks (whose
// slots are up to four times bigger than those of 256 rows).
constexpr int kRingS = 6, kRingL = 4;

// Waveform record of the level in buffer bin between columns i_e and i_e + 1, one row a
// thread, read from the buffer itself.  It stands outside the column loop: in there the
// compiler ran its FP64 conversions (1 to 2 a node on the FP32 paths, on a pipe that is
// busy 16 clocks of the SM with each) at every column and discarded them (16384 x 256, us
// per step: FP32-Kahan 50.9 -> 48.0, FP32 39.0 -> 37.1).
template <class P>
__device__ __forceinline__ void record_level(const InstDev& d, int64_t step, int bin) {
    const int j = threadIdx.x;
    const Planes<P> in = Planes<P>::of(d, bin);
    const size_t wi = (size_t)(step % d.wave_cap) * d.nth + j;
    if (j >= d.nth || !TK_IN(d.status, d.i_e, d.nr - 1) || !TK_IN(d.status, wi, d.wave_cap * d.nth)) return;
    const double2 w = wave_lerp(in.load(node_index(d, d.i_e, j)).phi64(),
                                in.load(node_index(d, d.i_e + 1, j)).phi64(), d.f_e);
    d.wave[wi] = w;
    if (!isfinite(w.x) || !isfinite(w.y)) atomicOr(d.status, (unsigned)ST_NONFINITE);
}

// Columns of a work item in the expanded form (FP64, double-float), after the ring's first
// fills.  At column c the half-node sum s of c-1/2 has been exchanged already: predictor at
// c-1/2, S published together with the next half node's s (from column c+1, awaited here),
// one barrier, corrector at c-1.  A slot is read by its own rows only and is refilled after
// the next barrier, R columns ahead.  has_src: source terms meet this block; moving: from
// the moving particle's tables.
template <class P, int R, bool kMov, class SH, class SI, class MH, class MI>
__device__ __forceinline__ void strip_columns_x(const InstDev& d, int64_t step, int bin, int c0, int c1,
                                                ColumnRing<P, R>& ring, unsigned char* xb, bool has_src, bool moving,
                                                SH src_h, SI src_i, MH msrc_h, MI msrc_i) {
    using T = typename P::T;
    using C = Cx<T>;
    const Lin<T> A(d);
    const int j = threadIdx.x, nth = d.nth;
    const bool row_ok = j < nth;
    const PoleRow pole(d, j);
    const T hdt = step_hdt<T>(d), qdt = step_qdt<T>(d);
    const Planes<P> out = Planes<P>::of(d, 1 - bin);
    // exchange entries: [column parity][S, s][threads + 2] of 16 bytes
    const unsigned xs = 16u * (blockDim.x + 2u);
    auto xS = [&](int c) { return xb + (c & 1) * 2u * xs; };
    auto xs_ = [&](int c) { return xb + (c & 1) * 2u * xs + xs; };
    auto nbr = [&](const unsigned char* x, C& p, C& m) {
        p = get16<T>(x + 16 * (j + 2));
        m = get16<T>(x + 16 * j);
    };
    auto node = [&](int slot) { return ring.planes(slot).load((size_t)j); };
    // refill the slot that column col has left with column col + R
    auto refill = [&](int col, int slot) {
        if (threadIdx.x == 0 && col + R <= c1) ring.fill(d, bin, col + R, slot);
    };
    auto coefs = [&](bool half, int col, T* cf) {
        if (TK_IN(d.status, col, d.nr)) coefs2d<T>(d, half, col, j, cf);
    };
    auto term_h = [&](int h) { return kMov && moving ? msrc_h(h) : src_h(h); };
    auto term_i = [&](int i) { return kMov && moving ? msrc_i(i) : src_i(i); };

    // prologue: columns c0-1, c0, c0+1 in slots 0, 1, 2; the sums of c0-1/2 and c0+1/2
    ring.wait(0);
    NodeV<P> u_prev = node(0);
    ring.wait(1);
    NodeV<P> u_cur = node(1);
    ring.wait(2);
    NodeV<P> u_next = node(2);
    C s0 = A.add(u_prev.F, u_cur.F), s = A.add(u_cur.F, u_next.F);
    publish16<T>(xS(c0), j, s0, pole, row_ok);
    publish16<T>(xs_(c0), j, s, pole, row_ok);
    __syncthreads();
    for (int k = 0; k < 3; ++k) refill(c0 - 1 + k, k);
    HalfX<T> L;
    {
        C p, m;
        nbr(xS(c0), p, m);
        T cf[kNCoef];
        coefs(true, c0 - 1, cf);
        C src = C::zero();
        if (has_src) src = term_h(c0 - 1);
        L = predict_x<T, true>(A, u_prev.F, u_prev.Pp, u_cur.F, u_cur.Pp, s0, p, m, cf, hdt, src);
    }
    size_t o = node_index(d, c0, j);
    // two instances of the loop: blocks without source nodes carry no source code
    auto steady = [&](auto src_kind) {
        constexpr bool kSrc = decltype(src_kind)::value;
        int slot = 3 % R;   // of column c + 1
        // double-float: coefficients one phase ahead of use, the corrector's loaded before
        // the predictor, the next half node's after it (16384 x 256: 200 -> 169 us per step).
        // FP64 has the FP64 pipe to wait for and loads them where they are used (570 us
        // per step; one phase ahead 577)
        constexpr bool kAhead = P::kind == kDF;
        T cf[kNCoef], ci[kNCoef];
        if constexpr (kAhead) coefs(true, c0, cf);
#pragma unroll 2
        for (int c = c0 + 1; c <= c1; ++c) {
            // half node c-1/2 = (c-1, c): u_cur holds c-1, u_next column c
            C p, m;
            if constexpr (kAhead) coefs(false, c - 1, ci);
            else coefs(true, c - 1, cf);
            nbr(xs_(c - 1), p, m);
            C src = C::zero();
            if constexpr (kSrc) src = term_h(c - 1);
            const HalfX<T> Rh = predict_x<T, kSrc>(A, u_cur.F, u_cur.Pp, u_next.F, u_next.Pp, s, p, m, cf, hdt, src);
            if constexpr (kAhead) {
                if (c < c1) coefs(true, c, cf);
            }
            const C S = A.add(Rh.F, L.F);
            publish16<T>(xS(c), j, S, pole, row_ok);
            const NodeV<P> u = u_cur;
            u_cur = u_next;
            if (c < c1) {
                ring.wait(slot);
                u_next = node(slot);
                s = A.add(u_cur.F, u_next.F);
                publish16<T>(xs_(c), j, s, pole, row_ok);
            }
            __syncthreads();
            if (c < c1) refill(c + 1, slot);
            C S_p, S_m;
            nbr(xS(c), S_p, S_m);
            if constexpr (!kAhead) coefs(false, c - 1, ci);
            C srcc = C::zero();
            if constexpr (kSrc) srcc = term_i(c - 1);
            C dPhi, dPi;
            correct_x<T, kSrc>(A, Rh, L, S, S_p, S_m, ci, qdt, srcc, dPhi, dPi);
            if (row_ok && TK_IN(d.status, o, plane_elems(d))) {
                NodeV<P> v = u;
                v.F = A.update(v.F, dPhi);
                v.Pp = A.update(v.Pp, dPi);
                out.store(o, v);
            }
            L = Rh;
            o += d.pitch;
            slot = slot + 1 == R ? 0 : slot + 1;
        }
    };
    if (has_src) steady(std::true_type{});
    else steady(std::false_type{});
}

// One work item: the columns [c0, c1) of one instance for one step, one thread per row.
// Per column c (FP32 paths; strip_columns_x has the others): theta differences of Phi(c) from
// the ring slot; predictor at the half node c-1/2; exchange of its results with the rows
// above and below (the one barrier of the column); corrector at column c-1.  The first two columns are peeled so the steady-state loop has no
// per-column mode switches, and it is unrolled by two so the rotation of the
// previous / current column is register renaming (by two: measured faster than one,
// three or six on GB300).  Columns c0-1 .. c1 are read.
// kPerStep: the block belongs to a per-step launch (programmatic dependent launch: the
// part before griddepcontrol.wait overlaps the previous step, and the block returns at
// once when a bounded wait of an earlier launch gave up).  Returns false in that case.
// kMov: the kernel serves instances whose particle moves (per-step Gaussian tables);
// the kernels of circular orbits are compiled without that code.
// rec_here: the block that owns the extraction column takes the level's record.
template <class P, int R, bool kPerStep, bool kMov>
__device__ __forceinline__ bool strip_step(const InstDev& d, int64_t step, int bin, int c0,
                                           int c1, bool rec_here, ColumnRing<P, R>& ring,
                                           typename P::T* xbuf) {
    using T = typename P::T;
    using C = Cx<T>;
    constexpr bool kSplit = split_angular<P>();
    const int j = threadIdx.x;
    const int nth = d.nth;
    const bool row_ok = j < nth;
    const Planes<P> out = Planes<P>::of(d, 1 - bin);
    RowTab<P> rt;
    rt.load(d.thtab, j, row_ok);

    // source: this block's columns against the window
    const SourceDev& sw = d.src;
    const bool src_blk = sw.on &&
                         ((c0 - 1 < sw.i_lo + sw.ni && c1 >= sw.i_lo) ||
                          (c0 - 1 < sw.h_lo + sw.nh && c1 >= sw.h_lo));
    // the step's two source factors, computed once in FP64 (sincos) by two warps, one
    // factor each, and shared already rounded to the arithmetic type
    __shared__ T sfac[4];
    __shared__ int skip;
    if (src_blk) {
        const int w1 = blockDim.x > 32 ? 32 : 0;
        if (threadIdx.x == 0) {
            const double2 f = source_factor<kMov>(d, step, 0.0, kSplit ? 0.5 * d.dt : d.dt);
            sfac[0] = (T)f.x;
            sfac[1] = (T)f.y;
        }
        if (threadIdx.x == w1) {
            const double2 f = source_factor<kMov>(d, step, 0.5, d.dt);
            sfac[2] = (T)f.x;
            sfac[3] = (T)f.y;
        }
    }
    // Everything above reads only constant data; the state of the previous step (read
    // by the ring, overwritten by this step's stores) is touched only below.
    if constexpr (kPerStep) griddep_wait();
    if (threadIdx.x == 0) {
        // a bounded wait of an earlier launch gave up: the state is void until it is reset
        skip = kPerStep ? (*(volatile unsigned*)d.status & ST_TIMEOUT) != 0 : 0;
        if (!skip) {
            fence_proxy_async_global();
            for (int k = 0; k < c1 - c0 + 2 && k < R; ++k) ring.fill(d, bin, c0 - 1 + k, k);
        }
    }
    __syncthreads();
    if (kPerStep && skip) return false;
    C sp_fac = C::zero(), sc_fac = C::zero();
    if (src_blk) {
        sp_fac = {sfac[0], sfac[1]};
        sc_fac = {sfac[2], sfac[3]};
    }
    // moving particle: this row's angular factors join the step's factors; gr points at
    // the step's radial factors (half nodes, then integer nodes)
    const T* gr = nullptr;
    if constexpr (kMov) {
        if (src_blk && sw.moving && step < sw.n_traj) {
            const int b = j - sw.j_lo;
            T gh = T(0), gi = T(0);
            if ((unsigned)b < (unsigned)sw.nj) {
                const T* gt = (const T*)sw.gt + (size_t)step * 2 * sw.nj + b;
                gh = gt[0];
                gi = gt[sw.nj];
            }
            sp_fac = gh * sp_fac;
            sc_fac = gi * sc_fac;
            gr = (const T*)sw.gr + (size_t)step * (sw.nh + sw.ni);
        }
    }
    // the input level's waveform record, by the block that owns column i_e (block 0 also
    // between columns 0 and 1), while the ring's first copies are in flight
    if (rec_here && ((c0 <= d.i_e && d.i_e < c1) || (c0 == 1 && d.i_e == 0))) record_level<P>(d, step, bin);

    // radial boundary condition: Phi = Pi = 0 at i = 0 and i = nr - 1
    if (row_ok && c0 == 1) out.store(node_index(d, 0, j), NodeV<P>::zero());
    if (row_ok && c1 == d.nr - 1) out.store(node_index(d, d.nr - 1, j), NodeV<P>::zero());

    // source terms at the half node h and the node i (source blocks only)
    auto src_h = [&](int h) { return source_half<T>(sw, sp_fac, h, j); };
    auto src_i = [&](int i) { return source_int<T>(sw, sc_fac, i, j); };
    // the same for a moving particle: the column's radial factor joins the step's factor
    auto msrc_h = [&](int h) {
        const int a = h - sw.h_lo;
        const T g = (unsigned)a < (unsigned)sw.nh ? gr[a] : T(0);
        return source_half<T>(sw, g * sp_fac, h, j);
    };
    auto msrc_i = [&](int i) {
        const int a = i - sw.i_lo;
        const T g = (unsigned)a < (unsigned)sw.ni ? gr[sw.nh + a] : T(0);
        return source_int<T>(sw, g * sc_fac, i, j);
    };
    if constexpr (kSplit) {
        const bool bot = j == 0, top = j == nth - 1;
        // theta neighbours in the slot, the pole rows standing in for the ghost rows: row
        // nth = g * row nth-1 and row -1 = g * row 0 (-ngp, -ngm the factors)
        const int jp = j + 1 < nth ? j + 1 : j, jm = j > 0 ? j - 1 : 0;
        const T g = d.ghost_f;
        const T ngp = top ? -g : T(-1), ngm = bot ? -g : T(-1);
        const T qdt = step_qdt<T>(d);
        const unsigned xstride = 4u * (blockDim.x + 2u);
        const size_t pitch = (size_t)d.pitch;
        // own node of the column in slot s (rows past nth read slot padding: their results
        // are never stored or exchanged)
        auto node = [&](int s) { return ring.planes(s).load((size_t)j); };
        // theta differences of Phi in the column in slot s (own node u): second (negated) and
        // two-cell (see split_angular)
        auto theta_diffs = [&](int s, const NodeV<P>& u, C& dl, C& dlm) {
            const Planes<P> pl = ring.planes(s);
            const NodeV<P> dn = pl.load_phi((size_t)jp), upn = pl.load_phi((size_t)jm);
            u.theta_split(ngp, dn, ngm, upn, dl, dlm);
        };
        // predictor at the half node h between columns h (ul) and h+1 (ur)
        auto predict = [&](const NodeV<P>& ul, const NodeV<P>& ur, C dll, C dlr, C dlml, C dlmr,
                           const T* cf, C src) {
            const Half<T> hp = half_prep<P>(ul, ur);
            return predictor<T>(hp, dll + dlr, dlml + dlmr, cf, qdt, src);
        };
        // coefficients of the column whose tables are in slot: the half node to its right into
        // cfh and the node into cfi, formed together in paired instructions
        auto coefs = [&](int slot, T* cfh, T* cfi) {
            float2 cf2[kNCoef];
            form_coefs2(ring.tab2(slot), rt.t, cf2);
#pragma unroll
            for (int k = 0; k < kNCoef; ++k) {
                cfh[k] = cf2[k].x;
                cfi[k] = cf2[k].y;
            }
        };
        // corrector at a column from the half nodes L and R on its two sides; xb is the exchange
        // buffer of the column's parity, srcc the node's source term, cfi its coefficients
        auto correct = [&](const HalfRec<T>& Rh, const HalfRec<T>& Lh, const NodeV<P>& uc,
                           const T* cfi, T* xb, size_t o, C srcc) {
            const CRow<T> row = combine_lr<T>(Rh, Lh);
            // publish this row's exchange entry (the split form needs Hs alone: its averaged
            // differences are the row's own), then read the rows above and below
            T* mine = xb + 4 * (j + 1);
            xpublish(xb, mine, row, g, row_ok, top, bot);
            __syncthreads();
            C Hs_p, Hs_m;
            xread(mine, Hs_p, Hs_m);
            C dPhi, dPi;
            corrector_incr<P>(row, Hs_p, Hs_m, cfi, qdt, srcc, dPhi, dPi);
            if (row_ok && TK_IN(d.status, o, plane_elems(d))) {
                NodeV<P> u = uc;
                u.update(dPhi, dPi);
                out.store(o, u);
            }
        };
        // prologue: columns c0-1 (slot 0) and c0 (slot 1)
        C dl_prev, dlm_prev, dl, dlm;
        ring.wait(0);
        NodeV<P> u_prev = node(0);
        theta_diffs(0, u_prev, dl_prev, dlm_prev);
        ring.wait(1);
        NodeV<P> u_cur = node(1);
        theta_diffs(1, u_cur, dl, dlm);
        T cfh[kNCoef], cfi[kNCoef];
        coefs(0, cfh, cfi);
        C s_first = C::zero();
        if constexpr (kMov) {
            if (gr) s_first = msrc_h(c0 - 1);
            else if (src_blk) s_first = src_h(c0 - 1);
        } else {
            if (src_blk) s_first = src_h(c0 - 1);
        }
        HalfRec<T> L = predict(u_prev, u_cur, dl_prev, dl, dlm_prev, dlm, cfh, s_first);
        u_prev = u_cur;
        dl_prev = dl;
        dlm_prev = dlm;
        size_t o = node_index(d, c0, j);               // output offset of the corrector's column

        // steady state: column c arrives, predictor at c-1/2, corrector at c-1; the slots
        // hold columns c-2 (sf, free once the column's barrier is passed), c-1 (sp) and c (sc).
        // Three instances of the loop: blocks without source nodes carry no source code; the
        // source blocks (circular orbit: kSrc = 1, moving particle: 2) load the next
        // column's source terms one column ahead.
        auto steady = [&](auto src_kind) {
            constexpr int kSrc = decltype(src_kind)::value;
            auto load_src = [&](int c, C& h, C& i) {
                if constexpr (kSrc == 1) {
                    h = src_h(c);
                    i = src_i(c);
                } else if constexpr (kSrc == 2 && kMov) {
                    h = msrc_h(c);
                    i = msrc_i(c);
                }
            };
            C nxt_h = C::zero(), nxt_i = C::zero();
            load_src(c0, nxt_h, nxt_i);
            int sf = 0, sp = 1, sc = 2;
#pragma unroll 2
            for (int c = c0 + 1; c <= c1; ++c) {
                const C s_h = nxt_h, s_i = nxt_i;
                if constexpr (kSrc != 0) {
                    if (c < c1) load_src(c, nxt_h, nxt_i);
                }
                ring.wait(sc);
                u_cur = node(sc);
                theta_diffs(sc, u_cur, dl, dlm);
                coefs(sp, cfh, cfi);
                const HalfRec<T> Rh = predict(u_prev, u_cur, dl_prev, dl, dlm_prev, dlm, cfh, s_h);
                correct(Rh, L, u_prev, cfi, xbuf + (c & 1) * xstride, o, s_i);
                if (threadIdx.x == 0 && c - 2 + R <= c1) ring.template fill<kSrc != 0>(d, bin, c - 2 + R, sf);
                L = Rh;
                u_prev = u_cur;
                dl_prev = dl;
                dlm_prev = dlm;
                o += pitch;
                sf = sp;
                sp = sc;
                sc = sc + 1 == R ? 0 : sc + 1;
            }
        };
        if constexpr (kMov) {
            if (gr) steady(std::integral_constant<int, 2>{});
            else if (src_blk) steady(std::integral_constant<int, 1>{});
            else steady(std::integral_constant<int, 0>{});
        } else {
            if (src_blk) steady(std::integral_constant<int, 1>{});
            else steady(std::integral_constant<int, 0>{});
        }
    } else {
        strip_columns_x<P, R, kMov>(d, step, bin, c0, c1, ring, (unsigned char*)xbuf, src_blk, gr != nullptr,
                                    src_h, src_i, msrc_h, msrc_i);
    }
    if (__syncthreads_or(ring.late)) {
        if (threadIdx.x == 0) {
            ring.drain();
            atomicOr(d.status, (unsigned)ST_TIMEOUT);
        }
        __syncthreads();
        ring.late = false;
    }
    return true;
}

// Four register budgets: columns of up to 256 rows (the common case, P::blocks256
// blocks per SM), of up to 320 rows (FP32 paths, two blocks per SM, 96 registers), of
// up to 512 rows (one block per SM, 128 registers a thread) and of up to 1024 rows.
// Dynamic shared memory: StepShared<P, R>::bytes(blockDim.x).
// part (may be null): the block's columns are [part[b], part[b+1]), of `strip` pieces, instead
// of uniform strips of `strip` columns; it is written by the host before the launch sequence
// and never changes while a step runs, so it is read before griddepcontrol.wait.
template <class P, int R, bool kMov>
__device__ __forceinline__ void step_body(const InstDev& d, int64_t step, int bin, int strip,
                                          const int* part) {
    extern __shared__ __align__(128) unsigned char step_smem[];
    __shared__ uint64_t mbar[R];
    // the next step's launch may begin now: its blocks become resident as ours retire and
    // run their set-up while this step drains
    griddep_launch_dependents();
    // replayed from a graph: the step is an offset from a base that the host (before the
    // first replay) or the graph's last node (after each replay) sets; it does not change
    // while the graph's steps run
    if (d.step_base) step += *d.step_base;
    // a launch with one block more than pieces takes the record in that block
    const bool rec_apart = part ? (int)gridDim.x > strip : (int64_t)(gridDim.x - 1) * strip >= d.nr - 2;
    if (rec_apart && blockIdx.x == gridDim.x - 1) {
        griddep_wait();
        if (!(*(volatile unsigned*)d.status & ST_TIMEOUT)) record_level<P>(d, step, bin);
        return;
    }
    ColumnRing<P, R> ring(step_smem, mbar);
    if (threadIdx.x == 0) ring.init();
    __syncthreads();
    int c0, c1;
    if (part) {
        c0 = part[blockIdx.x];
        c1 = part[blockIdx.x + 1];
    } else {
        c0 = 1 + blockIdx.x * strip;
        c1 = min(d.nr - 1, c0 + strip);
    }
    strip_step<P, R, true, kMov>(d, step, bin, c0, c1, !rec_apart, ring, StepShared<P, R>::xbuf(step_smem));
}

template <class P, bool kMov>
__global__ void __launch_bounds__(256, P::blocks256) step_kernel_s(InstDev d, int64_t step, int bin, int strip,
                                                                  const int* part) {
    step_body<P, kRingS, kMov>(d, step, bin, strip, part);
}

// FP32 paths, columns of 257 to 320 rows: with 96 registers a thread
// two blocks per SM, 20 warps, where the 512-row build holds one, 10 warps.
// us per step, 3001 x 300: FP32 12.6 -> 10.6, FP32-Kahan 15.6 -> 13.2; 8192 x 288: 30.5 -> 23.9, 38.7 ->
// 30.8.  (FP64 3001 x 300 147.8 -> 145.3 but 1000 x 270 53.9 -> 55.5; double-float spills.)
constexpr int kWideRows = 320;
template <class P>
__host__ __device__ constexpr bool has_wide() { return split_angular<P>(); }
template <class P, bool kMov>
__global__ void __launch_bounds__(kWideRows, 2) step_kernel_w(InstDev d, int64_t step, int bin, int strip,
                                                             const int* part) {
    step_body<P, kRingS, kMov>(d, step, bin, strip, part);
}

template <class P, bool kMov>
__global__ void __launch_bounds__(512, 1) step_kernel_m(InstDev d, int64_t step, int bin, int strip,
                                                       const int* part) {
    step_body<P, kRingS, kMov>(d, step, bin, strip, part);
}

template <class P, bool kMov>
__global__ void __launch_bounds__(1024) step_kernel_l(InstDev d, int64_t step, int bin, int strip,
                                                     const int* part) {
    step_body<P, kRingL, kMov>(d, step, bin, strip, part);
}

__global__ void advance_step_kernel(int64_t* base, int64_t k) {
    if (threadIdx.x == 0 && blockIdx.x == 0) *base += k;
}

void launch_advance_step(cudaStream_t st, int64_t* base, int64_t k) {
    advance_step_kernel<<<1, 32, 0, st>>>(base, k);
}

// Waveform record of the state in buffer bin (time level `step`): one thread per row.
template <class P>
__global__ void extract_kernel(InstDev d, int64_t step, int bin) {
    int j = blockIdx.x * blockDim.x + threadIdx.x;
    if (j >= d.nth) return;
    if (!TK_IN(d.status, d.i_e + 1, d.nr) || !TK_IN(d.status, d.i_e, d.nr)) return;
    const Planes<P> in = Planes<P>::of(d, bin);
    double2 a = in.load(node_index(d, d.i_e, j)).phi64();
    double2 b = in.load(node_index(d, d.i_e + 1, j)).phi64();
    double f = d.f_e;
    double2 w = wave_lerp(a, b, f);
    const size_t wi = (size_t)(step % d.wave_cap) * d.nth + j;
    if (TK_IN(d.status, wi, d.wave_cap * d.nth)) d.wave[wi] = w;
    if (!isfinite(w.x) || !isfinite(w.y)) atomicOr(d.status, (unsigned)ST_NONFINITE);
}

// ---------------------------------------------------------------- batched path
__device__ __forceinline__ int ld_acquire(const int* p) {
    int v;
    asm volatile("ld.acquire.gpu.global.b32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ void st_release(int* p, int v) {
    asm volatile("st.release.gpu.global.b32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}

// Wait until the strips st-1, st, st+1 of the previous step have completed.  That
// covers what this strip reads (one column on each side) and what it overwrites (the
// buffer its neighbours read).  Threads 0..2 poll one neighbour each with acquire
// loads; a wait gives up after spin_limit polls.  Returns false on give-up or abort.
__device__ bool wait_neighbours(const BatchDev& b, const int* fl, int nstrip, int st, int64_t s,
                                int* flag_smem) {
    const int t = threadIdx.x;
    if (t == 0) *flag_smem = 1;
    __syncthreads();
    if (t < 3) {
        int q = st + t - 1;
        if (q >= 0 && q < nstrip) {
            long long it = 0;
            while (ld_acquire(fl + q) < (int)s) {
                if (++it > b.spin_limit || *(volatile int*)b.abort) {
                    *flag_smem = 0;
                    break;
                }
                __nanosleep(64);
            }
        }
    }
    __syncthreads();
    bool ok = *flag_smem != 0;
    __threadfence();
    __syncthreads();
    return ok;
}

// Persistent kernel of one block-size class: blocks grab (step, instance, strip) items
// in step order; an item waits for its radial neighbours of the previous step.  Items
// only wait on items grabbed earlier, so the launch cannot deadlock whatever the
// number of resident blocks.  kMov: some instance of the class has a moving particle.
template <class P, int kMaxThreads, int kMinBlocks, int R, bool kMov>
__global__ void __launch_bounds__(kMaxThreads, kMinBlocks) batched_step_kernel(BatchDev b) {
    extern __shared__ __align__(128) unsigned char step_smem[];
    __shared__ uint64_t mbar[R];
    __shared__ unsigned long long item;
    __shared__ int flag;
    __shared__ InstDev inst_sm;
    static_assert(sizeof(InstDev) % sizeof(int) == 0, "descriptor copied as ints");
    ColumnRing<P, R> ring(step_smem, mbar);
    typename P::T* xbuf = StepShared<P, R>::xbuf(step_smem);
    if (threadIdx.x == 0) ring.init();
    const int64_t nsteps = *b.n_steps;
    const int64_t total = b.items_per_step * nsteps;
    for (;;) {
        __syncthreads();
        if (threadIdx.x == 0) item = atomicAdd(b.counter, 1ull);
        __syncthreads();
        const unsigned long long g = item;
        if ((int64_t)g >= total || *(volatile int*)b.abort) return;
        const int64_t s = (int64_t)g / b.items_per_step, r = (int64_t)g % b.items_per_step;
        int lo = 0, hi = b.n_inst - 1;
        while (lo < hi) {
            int mid = (lo + hi + 1) >> 1;
            if (b.item_base[mid] <= r) lo = mid; else hi = mid - 1;
        }
        const int k = lo;
        const int st = (int)(r - b.item_base[k]);
        if (!TK_IN(b.status, k, b.n_inst) || !TK_IN(b.status, r, b.items_per_step)) return;
        // the item's instance descriptor in shared memory: its fields are then cheap
        // shared loads instead of global loads held in registers (the previous item's
        // readers are past the barrier that ends strip_step)
        for (int q = threadIdx.x; q < (int)(sizeof(InstDev) / sizeof(int)); q += blockDim.x)
            ((int*)&inst_sm)[q] = ((const int*)(b.inst + k))[q];
        __syncthreads();
        const InstDev& d = inst_sm;
        const int strip = b.strip[k], nstrip = b.nstrip[k];
        if (!TK_IN(b.status, st, nstrip)) return;
        int* fl = b.flags + b.item_base[k];
        if (s > 0 && !wait_neighbours(b, fl, nstrip, st, s, &flag)) {
            if (threadIdx.x == 0) {
                atomicOr(b.status, (unsigned)ST_TIMEOUT);
                atomicExch(b.abort, 1);
            }
            return;
        }
        const int c0 = 1 + st * strip;
        const int c1 = min(d.nr - 1, c0 + strip);
        strip_step<P, R, false, kMov>(d, b.base_step[k] + s, (int)((b.base_bin[k] + s) & 1), c0, c1, true, ring, xbuf);
        __threadfence();
        __syncthreads();
        if (threadIdx.x == 0 && !(s == 0 && r == b.skip_release_item))
            st_release(fl + st, (int)(s + 1));
    }
}

// Waveform record of the final level of every instance of the class (block row y).
template <class P>
__global__ void batched_extract_kernel(BatchDev b) {
    const int k = blockIdx.y;
    if (!TK_IN(b.status, k, b.n_inst)) return;
    const InstDev& d = b.inst[k];
    int j = blockIdx.x * blockDim.x + threadIdx.x;
    if (j >= d.nth) return;
    if (!TK_IN(d.status, d.i_e + 1, d.nr) || !TK_IN(d.status, d.i_e, d.nr)) return;
    const int64_t n = *b.n_steps;
    const int bin = (int)((b.base_bin[k] + n) & 1);
    const int64_t step = b.base_step[k] + n;
    const Planes<P> in = Planes<P>::of(d, bin);
    double2 a = in.load(node_index(d, d.i_e, j)).phi64();
    double2 c = in.load(node_index(d, d.i_e + 1, j)).phi64();
    double f = d.f_e;
    double2 w = wave_lerp(a, c, f);
    const size_t wi = (size_t)(step % d.wave_cap) * d.nth + j;
    if (TK_IN(d.status, wi, d.wave_cap * d.nth)) d.wave[wi] = w;
    if (!isfinite(w.x) || !isfinite(w.y)) atomicOr(d.status, (unsigned)ST_NONFINITE);
}

template <class P>
static int grid_for(int threads) {
    int dev = 0, sms = 0, per = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    // the smaller residency of the two variants (with and without moving particles)
    int per2 = 0;
    if (threads <= 256) {
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, batched_step_kernel<P, 256, P::blocks256, kRingS, false>,
                                                      threads, StepShared<P, kRingS>::bytes(threads));
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per2, batched_step_kernel<P, 256, P::blocks256, kRingS, true>,
                                                      threads, StepShared<P, kRingS>::bytes(threads));
    } else if (threads <= 512) {
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, batched_step_kernel<P, 512, 1, kRingS, false>,
                                                      threads, StepShared<P, kRingS>::bytes(threads));
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per2, batched_step_kernel<P, 512, 1, kRingS, true>,
                                                      threads, StepShared<P, kRingS>::bytes(threads));
    } else {
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, batched_step_kernel<P, 1024, 1, kRingL, false>,
                                                      threads, StepShared<P, kRingL>::bytes(threads));
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per2, batched_step_kernel<P, 1024, 1, kRingL, true>,
                                                      threads, StepShared<P, kRingL>::bytes(threads));
    }
    per = per < per2 ? per : per2;
    return (per > 0 ? per : 1) * (sms > 0 ? sms : 1);
}

int batched_grid(int prec, int threads) {
    if (prec == 0) return grid_for<P64>(threads);
    if (prec == 1) return grid_for<P32>(threads);
    if (prec == 3) return grid_for<PD>(threads);
    return grid_for<PK>(threads);
}

template <class P, bool kMov>
static void launch_batched_m(cudaStream_t st, const BatchDev& b, int grid, int threads) {
    if (threads <= 256)
        batched_step_kernel<P, 256, P::blocks256, kRingS, kMov><<<grid, threads, StepShared<P, kRingS>::bytes(threads), st>>>(b);
    else if (threads <= 512)
        batched_step_kernel<P, 512, 1, kRingS, kMov><<<grid, threads, StepShared<P, kRingS>::bytes(threads), st>>>(b);
    else
        batched_step_kernel<P, 1024, 1, kRingL, kMov><<<grid, threads, StepShared<P, kRingL>::bytes(threads), st>>>(b);
}
template <class P>
static void launch_batched_p(cudaStream_t st, const BatchDev& b, int grid, int threads, bool mov) {
    if (mov) launch_batched_m<P, true>(st, b, grid, threads);
    else launch_batched_m<P, false>(st, b, grid, threads);
}

void launch_batched_step(cudaStream_t st, int prec, const BatchDev& b, int grid, int threads,
                         bool moving) {
    if (prec == 0) launch_batched_p<P64>(st, b, grid, threads, moving);
    else if (prec == 1) launch_batched_p<P32>(st, b, grid, threads, moving);
    else if (prec == 3) launch_batched_p<PD>(st, b, grid, threads, moving);
    else launch_batched_p<PK>(st, b, grid, threads, moving);
}

void launch_batched_extract(cudaStream_t st, int prec, const BatchDev& b, int max_nth) {
    dim3 g((max_nth + 127) / 128, b.n_inst);
    if (prec == 0) batched_extract_kernel<P64><<<g, 128, 0, st>>>(b);
    else if (prec == 1) batched_extract_kernel<P32><<<g, 128, 0, st>>>(b);
    else if (prec == 3) batched_extract_kernel<PD><<<g, 128, 0, st>>>(b);
    else batched_extract_kernel<PK><<<g, 128, 0, st>>>(b);
}

size_t capped_smem(int cap, size_t own) {
    int dev = 0, sm = 0, res = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sm, cudaDevAttrMaxSharedMemoryPerMultiprocessor, dev);
    cudaDeviceGetAttribute(&res, cudaDevAttrReservedSharedMemoryPerBlock, dev);
    const int b = (sm / cap - res - 512) / 128 * 128;   // (512: the kernels' static shared memory)
    return b > (int)own ? (size_t)b : own;
}

template <class P, bool kMov>
static void launch_step_m(cudaStream_t st, const InstDev& d, int64_t step, int bin, const StepCut& cut) {
    const int strip = cut.part ? cut.nb : cut.strip;
    const int* part = cut.part;
    // a grid that leaves a block's place free takes its record in a block of its own: on
    // 800 x 64 (one-column pieces) the block that also took the record was the step's last
    // (us per step: FP32-Kahan 4.01 -> 3.49, FP32 3.35 -> 3.09); a full wave has no such
    // place, and the piece that holds the record is cut shorter (refresh_partition)
    int blocks = part ? cut.nb : (d.nr - 2 + strip - 1) / strip;
    if (blocks < cut.room) ++blocks;
    int threads = d.pitch;
    // programmatic dependent launch (see step_body)
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(blocks);
    cfg.blockDim = dim3(threads);
    cfg.stream = st;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    if (threads <= 256) {
        cfg.dynamicSmemBytes = StepShared<P, kRingS>::bytes(threads);
        if (cut.cap > 0) cfg.dynamicSmemBytes = capped_smem(cut.cap, cfg.dynamicSmemBytes);
        cudaLaunchKernelEx(&cfg, step_kernel_s<P, kMov>, d, step, bin, strip, part);
    } else if (threads <= kWideRows && has_wide<P>()) {
        cfg.dynamicSmemBytes = StepShared<P, kRingS>::bytes(threads);
        if constexpr (has_wide<P>()) cudaLaunchKernelEx(&cfg, step_kernel_w<P, kMov>, d, step, bin, strip, part);
    } else if (threads <= 512) {
        cfg.dynamicSmemBytes = StepShared<P, kRingS>::bytes(threads);
        cudaLaunchKernelEx(&cfg, step_kernel_m<P, kMov>, d, step, bin, strip, part);
    } else {
        cfg.dynamicSmemBytes = StepShared<P, kRingL>::bytes(threads);
        cudaLaunchKernelEx(&cfg, step_kernel_l<P, kMov>, d, step, bin, strip, part);
    }
}
template <class P>
static void launch_step_p(cudaStream_t st, const InstDev& d, int64_t step, int bin, const StepCut& cut) {
    if (d.src.on && d.src.moving) launch_step_m<P, true>(st, d, step, bin, cut);
    else launch_step_m<P, false>(st, d, step, bin, cut);
}

template <class P>
static int resident_p(int threads) {
    int dev = 0, sms = 0, per = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (threads <= 256)
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, step_kernel_s<P, false>, threads,
                                                      StepShared<P, kRingS>::bytes(threads));
    else if (threads <= kWideRows && has_wide<P>()) {
        if constexpr (has_wide<P>())
            cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, step_kernel_w<P, false>, threads,
                                                          StepShared<P, kRingS>::bytes(threads));
    } else if (threads <= 512)
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, step_kernel_m<P, false>, threads,
                                                      StepShared<P, kRingS>::bytes(threads));
    else
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, step_kernel_l<P, false>, threads,
                                                      StepShared<P, kRingL>::bytes(threads));
    return (per > 0 ? per : 1) * (sms > 0 ? sms : 1);
}

int step_resident_blocks(int prec, int threads) {
    if (prec == 0) return resident_p<P64>(threads);
    if (prec == 1) return resident_p<P32>(threads);
    if (prec == 3) return resident_p<PD>(threads);
    return resident_p<PK>(threads);
}

void launch_step(cudaStream_t st, const InstDev& d, int64_t step, int bin, const StepCut& cut) {
    if (d.prec == 0) launch_step_p<P64>(st, d, step, bin, cut);
    else if (d.prec == 1) launch_step_p<P32>(st, d, step, bin, cut);
    else if (d.prec == 3) launch_step_p<PD>(st, d, step, bin, cut);
    else launch_step_p<PK>(st, d, step, bin, cut);
}

// Shared memory that the batched kernels of up to 512 rows ask an SM to set aside, per cent of
// its 228 KB: 164 KB, room for the 512 threads of a plan of several classes side by side
// (plan_branches: at most 256 bytes a thread and 1.7 KB a block, of 16 blocks 155 KB).
// Left to the launches, an SM set aside what the class that came first needs; the blocks of
// the other class found no room there and joined only when it had finished.  us per step,
// FP32-Kahan 32 + 64 rows, 12000 columns each: 46.4 -> 30.4, one class after the other 33.4;
// FP64 128 + 160 rows: 210 -> 121, 128.  What the L1 loses costs nothing (one class after the
// other 1.00 in 54 batches); 100 per cent costs double-float 3 to 10 % (its tables come
// through the L1), 70 per cent leaves 132 KB, too little.
constexpr int kBatchCarveout = 72;

// Opt the step kernels of one precision in to the dynamic shared memory of their largest
// blocks (on the current device; called when a context of that precision is created).
template <class P, bool kMov>
static cudaError_t prepare_m() {
    // (a capped launch, FP64 and double-float, takes more than its blocks need)
    const unsigned need = StepShared<P, kRingS>::bytes(256);
    const int s = (int)(split_angular<P>() ? need : capped_smem(kMinCap, need)), m = (int)StepShared<P, kRingS>::bytes(512),
              l = (int)StepShared<P, kRingL>::bytes(1024);
    const cudaFuncAttribute a = cudaFuncAttributeMaxDynamicSharedMemorySize;
    cudaError_t e = cudaFuncSetAttribute(step_kernel_s<P, kMov>, a, s);
    if constexpr (has_wide<P>()) {
        if (e == cudaSuccess)
            e = cudaFuncSetAttribute(step_kernel_w<P, kMov>, a, (int)StepShared<P, kRingS>::bytes(kWideRows));
    }
    if (e == cudaSuccess) e = cudaFuncSetAttribute(step_kernel_m<P, kMov>, a, m);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(step_kernel_l<P, kMov>, a, l);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(batched_step_kernel<P, 256, P::blocks256, kRingS, kMov>, a, s);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(batched_step_kernel<P, 512, 1, kRingS, kMov>, a, m);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(batched_step_kernel<P, 1024, 1, kRingL, kMov>, a, l);
    const cudaFuncAttribute cv = cudaFuncAttributePreferredSharedMemoryCarveout;
    if (e == cudaSuccess) e = cudaFuncSetAttribute(batched_step_kernel<P, 256, P::blocks256, kRingS, kMov>, cv, kBatchCarveout);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(batched_step_kernel<P, 512, 1, kRingS, kMov>, cv, kBatchCarveout);
    return e;
}
template <class P>
static cudaError_t prepare_p() {
    cudaError_t e = prepare_m<P, false>();
    if (e == cudaSuccess) e = prepare_m<P, true>();
    return e;
}

cudaError_t prepare_step_kernels(int prec) {
    if (prec == 0) return prepare_p<P64>();
    if (prec == 1) return prepare_p<P32>();
    if (prec == 3) return prepare_p<PD>();
    return prepare_p<PK>();
}

void launch_extract(cudaStream_t st, const InstDev& d, int64_t step, int bin) {
    int blocks = (d.nth + 127) / 128;
    if (d.prec == 0) extract_kernel<P64><<<blocks, 128, 0, st>>>(d, step, bin);
    else if (d.prec == 1) extract_kernel<P32><<<blocks, 128, 0, st>>>(d, step, bin);
    else if (d.prec == 3) extract_kernel<PD><<<blocks, 128, 0, st>>>(d, step, bin);
    else extract_kernel<PK><<<blocks, 128, 0, st>>>(d, step, bin);
}

}  // namespace teuk
