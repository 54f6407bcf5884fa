// Persistent step kernels: one launch advances every instance of a uniform-N group by nsteps
// RK4IP or Strang steps with the field held in registers throughout.
#pragma once

#include <type_traits>

#include "cme_core.cuh"
#include "cme_fixed.cuh"

namespace cme {
inline namespace CME_FP32_VARIANT {

// Threads per block a kernel is compiled for: groups of P >= 64 threads run one instance per
// block (so the register file is shared by as few threads as possible); narrower groups pack
// up to 256 threads.
template <int LOGN, int R>
constexpr int max_threads() { return Plan<LOGN, R>::P >= 64 ? Plan<LOGN, R>::P : 256; }

// Per-mode propagators of the RK4IP and Strang steps: E = exp(L h/2), e1 = expm1(L h/2),
// e2 = expm1(L h).  For FP32 groups up to N = 1024 they are held in registers for the whole
// launch; otherwise they are read through the read-only cache where used.
template <typename T, int LOGN, int R, int C = 1>
struct Props {
    // cluster groups run few threads per block, so their register budget has room, and so do
    // 16-value groups of N >= 2048, whose twiddles live in shared memory
    static constexpr bool IN_REGS =
        sizeof(T) == 4 && (((LOGN <= 10 || C > 1) && R <= 8) || (LOGN >= 11 && R == 16));
    cx<T> E[IN_REGS ? R : 1], e1[IN_REGS ? R : 1], e2[IN_REGS ? R : 1];
    const cx<T>* pE;   // pointers pre-offset to (instance offset + t)
    const cx<T>* pe1;
    const cx<T>* pe2;
    const int4* pF;    // FP64: limbs of E (StepArgs::Ef)

    CME_DEV void init(const StepArgs& a, long long off, int t)
    {
        constexpr int P = Plan<LOGN, R>::P;
        pE = reinterpret_cast<const cx<T>*>(a.E) + off + t;
        pe1 = reinterpret_cast<const cx<T>*>(a.e1) + off + t;
        pe2 = reinterpret_cast<const cx<T>*>(a.e2) + off + t;
        pF = reinterpret_cast<const int4*>(a.Ef) + off + t;
        if constexpr (IN_REGS) {
#pragma unroll
            for (int j = 0; j < R; ++j) {
                E[j] = gload<T>(pE, j * P);
                e1[j] = gload<T>(pe1, j * P);
                e2[j] = gload<T>(pe2, j * P);
            }
        }
    }
    CME_DEV fl2 getF(int j) const { return fx_twiddle(pF, j * Plan<LOGN, R>::P); }
    CME_DEV cx<T> getE(int j) const
    {
        if constexpr (IN_REGS)
            return E[j];
        else
            return gload<T>(pE, j * Plan<LOGN, R>::P);
    }
    CME_DEV cx<T> get1(int j) const
    {
        if constexpr (IN_REGS)
            return e1[j];
        else
            return gload<T>(pe1, j * Plan<LOGN, R>::P);
    }
    CME_DEV cx<T> get2(int j) const
    {
        if constexpr (IN_REGS)
            return e2[j];
        else
            return gload<T>(pe2, j * Plan<LOGN, R>::P);
    }
};

// Twiddles stay in registers up to N = 1024 (FP32) / 512 (FP64).
template <typename T, int LOGN>
constexpr bool twiddles_in_regs() { return sizeof(T) == 4 ? LOGN <= 10 : LOGN <= 9; }

// The transform of a group: one block's Stockham transform, or for C > 1 the four-step
// cluster transform and its transform inside one block.
template <typename T, int LOGN, int R, int C>
struct GroupFFT {
    using CF = ClusterFFT<T, LOGN, R, C>;
    using TF = typename CF::TL;
};
template <typename T, int LOGN, int R>
struct GroupFFT<T, LOGN, R, 1> {
    using CF = void;
    using TF = Transform<T, LOGN, R, (Plan<LOGN, R>::P <= 32)>;
};

template <typename T, int LOGN, int R, int C>
CME_HD constexpr size_t cluster_smem_bytes();

// Per-thread view of one instance: the transform machinery plus the instance constants.
// C > 1: the instance is spread over the C blocks of a thread-block cluster.
template <typename T, int LOGN, int R, int C = 1>
struct Group {
    using PL = Plan<LOGN, R>;
    static constexpr int N = PL::N, P = PL::P;
    static constexpr bool WARP = (C == 1 && P <= 32);
    static constexpr bool COMP = (sizeof(T) == 4);  // compensated state in FP32
    // C > 1: the four-step cluster transform; TF is then its transform inside one block
    using CF = typename GroupFFT<T, LOGN, R, C>::CF;
    using TF = typename GroupFFT<T, LOGN, R, C>::TF;
    static constexpr int LC = ilog2(C);
    // twiddles: registers (small N), this group's shared memory (FP32 one-block groups of
    // N >= 2048), else the global table (read at stride C by the block transforms of a cluster)
    static constexpr bool TW_REGS =
        twiddles_in_regs<T, LOGN - LC>() && (C == 1 || sizeof(T) == 4);
    static constexpr bool TW_SMEM = !TW_REGS && twiddles_in_smem(sizeof(T), LOGN - LC);
    // FP64 transforms run in fixed point (cme_fixed.cuh)
    static constexpr bool FIX = sizeof(T) == 8;
    using FT = FixTransform<LOGN - LC, R, (Plan<LOGN - LC, R>::P <= 32), (C > 1)>;
    using TW = std::conditional_t<
        FIX, FixTwiddles<LOGN - LC, R, TW_REGS, C>,
        std::conditional_t<TW_SMEM, TwiddlesSmem<T, LOGN - LC, R, C>,
                           Twiddles<T, LOGN - LC, R, TW_REGS, C>>>;
    // the block's own transform leaves the Kerr term's samples (a cluster's radix-C sums follow it,
    // whose scale is chosen for them)
    static constexpr bool TO_KERR = C == 1;
    int2* red;     // FP64: reduction pairs of this group's warps (shared memory)

    int t;         // the thread holds modes t + jP
    int ts;        // this thread's slots ts + jP of per-thread scratch vectors (coalesced)
    int par;
    Xbuf<T> buf;   // first of the two ping-pong exchange buffers
    typename TF::Addr ad;
    TW tw;

    // C > 1: all-to-all state (block `rank`, thread l): this thread's slots of the receive
    // buffer 0; shared::cluster address of receive buffer 0 and of its mbarrier in every
    // block; byte offsets of this thread's stores; the twiddles of the two directions in this
    // block's shared memory (thread-major); the receive-buffer parity; the phase parities of
    // this block's two mbarriers; whether a wait gave up.
    Xbuf<T> abuf;
    uint32_t rb[C > 1 ? C : 1];
    uint32_t rmb[C > 1 ? C : 1];
    uint32_t mb;
    uint32_t om, ot;
    // (FP64: limbs; scw: the source blocks' scale words of receive buffer 0, at byte offset scw_off
    // of the receive buffers in every block)
    using TWC = std::conditional_t<sizeof(T) == 8, int4, cx<T>>;
    const TWC* twm;
    const TWC* twt;
    const int2* scw;
    uint32_t scw_off;
    int rank;
    int apar;
    uint32_t ph;
    bool timed_out;
    int fault;     // StepArgs::a2a_fault
    // polls of one all-to-all wait before it gives up (a wait normally ends within a few)
    static constexpr int WAIT_TRIES = 1 << 20;

    // a bounded wait of an all-to-all gave up (the results are then not valid)
    CME_DEV bool failed() const
    {
        if constexpr (C == 1)
            return false;
        else
            return timed_out;
    }
    // Physical modes (the zero padding of Sec. 2): of the N modes only the centred M,
    // mu = mlo .. mhi, are physical; the right-hand side is zero on the others, which stay at
    // zero.  masked = false (M = N) skips the test.
    bool masked;
    int mlo, mhi;

    CME_DEV void set_modes(int M)
    {
        masked = M < N;
        mlo = -(M / 2);
        mhi = M - M / 2 - 1;
    }
    // Is the thread's position t + jP (mode mu = p or p - N, transform order) physical?
    CME_DEV bool physical(int j) const
    {
        if (!masked)
            return true;
        const int p = t + j * P;
        const int mu = p >= N / 2 ? p - N : p;
        return mu >= mlo && mu <= mhi;
    }
    CME_DEV void mask(cx<T> (&x)[R]) const
    {
        if (masked) {
#pragma unroll
            for (int j = 0; j < R; ++j)
                if (!physical(j))
                    x[j] = cx<T>{T(0), T(0)};
        }
    }
    // Per-mode Kerr coefficient (Sec. 2: g0 need not be constant): the four-wave-mixing term
    // of output mode mu carries g0_mu instead of the instance's g0, applied as the factor
    // km[j P] of this thread's mode t + jP to the forward transform's output (the instance's g0
    // is then 1).  km = null (the default) leaves every mode at g0.
    const T* km;
    CME_DEV void set_kerr(const void* table, long long off)
    {
        km = table ? reinterpret_cast<const T*>(table) + off + t : nullptr;
    }
    // The right-hand side's output side: the per-mode Kerr factor, then the physical-mode mask.
    CME_DEV void out_modes(cx<T> (&x)[R]) const
    {
        if (km) {
#pragma unroll
            for (int j = 0; j < R; ++j)
                x[j] = cscale(x[j], __ldg(km + j * P));
        }
        mask(x);
    }

    // The step loops contain a single copy of the transform code (instruction-cache
    // footprint): the forward transform is computed as conj(inverse(conj(x))).  d = 0 takes
    // modes to time samples, d = 1 time samples to modes (the same for one block; the
    // reverse order of the stages for a cluster).
    CME_DEV void inverse(cx<T> (&x)[R], int d)
    {
        if constexpr (FIX) {
            fx X[R];
            const typename FT::Scale sc = FT::template load<false>(x, X, red, tl());
            int q = sc.q;
            bool bad = q == FT::POISON;
            fix_inverse(X, q, sc.b, bad, d);
            FT::store(X, bad ? -FT::POISON : -q, x);
        } else if constexpr (C == 1) {
            TF::template run<+1>(x, tw, buf, par, ad);
        } else {
            if (d == 1) {
                CF::radix_c(x);
                twiddle(x, twt);
                all_to_all<true>(x);
            }
            TF::template run<+1>(x, tw, buf, par, ad);
            if (d == 0) {
                twiddle(x, twm);
                all_to_all<false>(x);
                CF::radix_c(x);
            }
        }
    }
    // this thread's index among those that share a transform's block
    CME_DEV int tl() const { return C == 1 ? t : (int)threadIdx.x; }
    // The same for fixed-point values X = x 2^q of bounds b; returns the bits of the result's
    // modulus.  C > 1: every block scales by its own bounds (its modes or samples alone), and
    // every all-to-all carries each source block's scale word (q, modulus and L1 bits), by
    // which the receiver aligns that block's values: no reduction over the cluster (16 x N = 4096
    // on 8-block clusters, RK4IP: 115 us per step in FP64 instructions, see rk4ip_step).
    CME_DEV int fix_inverse(fx (&X)[R], int& q, FixBound b, bool& bad, int d)
    {
        if constexpr (C == 1) {
            int ups[FT::NS];
            const int up = FT::template lift<TO_KERR>(b, ups);
            FT::run(X, tw, buf, par, ad, ups);
            q += up - FT::OUT;
            return FT::out_bits(b) + up;
        } else {
            constexpr int G = CF::G, PC = CF::PC;
            int bits = 0;
            int qs[C], bs[C], ls[C];   // the source blocks' scale words
            if (d == 1) {
                fix_radix_c(X);
                // (slots of k1 = 0 have twiddle 1: a rounded shift has no bias, a floored product
                // by 1 has)
#pragma unroll
                for (int j = 0; j < R; ++j)
                    X[j] = j < G ? fx{fshift(X[j].re, 2), fshift(X[j].im, 2)}
                                 : fcmul4(X[j], fl2_of(twt[j * PC]));
                fix_all_to_all<true>(X, q - 2, min(b.bl, b.bm + LC) - 2, b.bl - 2, bad, qs, bs, ls);
                q = qs[0];
#pragma unroll
                for (int c = 1; c < C; ++c)
                    q = min(q, qs[c]);
                // bounds at the coarsest source's scale: every received value is a sum over
                // all sources' samples of unit-modulus multiples, so L1 is at most the sum of
                // the sources' L1 (in units of 2^(top - 20))
                int top = -1000, bm = -1000;
#pragma unroll
                for (int c = 0; c < C; ++c) {
                    top = max(top, ls[c] - (qs[c] - q));
                    bm = max(bm, bs[c] - (qs[c] - q));
                }
                unsigned cnt = 0;
#pragma unroll
                for (int c = 0; c < C; ++c)
                    cnt += (1u << 20) >> min(top - (ls[c] - (qs[c] - q)), 31);
                b = {bm, top + 32 - __clz((int)(cnt - 1)) - 20};
                const int s = FT::LIM - FT::template headroom<false>(b);
                q += s;
                b.bm += s;
                b.bl += s;
#pragma unroll
                for (int j = 0; j < R; ++j)
                    X[j] = align_to(X[j], qs[j % C] - q);
            }
            int ups[FT::NS];
            const int up = FT::template lift<TO_KERR>(b, ups);
            FT::run(X, tw, buf, par, ad, ups);
            q += up - FT::OUT;
            bits = FT::out_bits(b) + up;
            if (d == 0) {
                if (rank != 0) {   // block 0's twiddles are 1
#pragma unroll
                    for (int j = 0; j < R; ++j)
                        X[j] = fcmul4(X[j], fl2_of(twm[j * PC]));
                    q -= 2;
                    bits -= 2;
                }
                fix_all_to_all<false>(X, q, bits, 0, bad, qs, bs, ls);
                // a scale at which the C-point sums stay below 2^61
                q = 1 << 28;
#pragma unroll
                for (int c = 0; c < C; ++c)
                    q = min(q, qs[c] - max(bs[c] - (61 - LC), 0));
#pragma unroll
                for (int j = 0; j < R; ++j)
                    X[j] = align_to(X[j], qs[j / G] - q);
                fix_radix_c(X);
                bits = 61;
            }
            return bits;
        }
    }
    CME_DEV static fl2 fl2_of(int4 v) { return {{v.x, v.y}, {v.z, v.w}}; }
    // v 2^-s, to the left for s < 0 (uniform over the block)
    CME_DEV static fx align_to(fx v, int s)
    {
        if (s < 0)
            return {fshl(v.re, -s), fshl(v.im, -s)};
        s = min(s, 63);
        return {frsh(v.re, s), frsh(v.im, s)};
    }
    CME_DEV static void fix_radix_c(fx (&x)[R])
    {
        if constexpr (C > 1) {
#pragma unroll
            for (int m = 0; m < CF::G; ++m) {
                fx v[C];
#pragma unroll
                for (int c = 0; c < C; ++c)
                    v[c] = x[c * CF::G + m];
                fdft<C>(v);
#pragma unroll
                for (int c = 0; c < C; ++c)
                    x[c * CF::G + m] = v[c];
            }
        }
    }
    // all_to_all of fixed-point values with this block's scale word (q, bits of the modulus and of
    // L1, whether a value was not finite) to every block; qs, bs, ls are the sources'.
    template <bool T2M>
    CME_DEV void fix_all_to_all(fx (&X)[R], int q, int bm, int bl, bool& bad, int (&qs)[C],
                                int (&bs)[C], int (&ls)[C])
    {
        cx<double> y[R];
#pragma unroll
        for (int j = 0; j < R; ++j)
            y[j] = {__longlong_as_double(X[j].re), __longlong_as_double(X[j].im)};
        const int buffer = apar;
        if ((int)threadIdx.x < C && !timed_out) {
            const int word = ((bm & 0xfff) << 16) | ((bl & 0xfff) << 1) | (bad ? 1 : 0);
            uint32_t to = 0, tm = 0;
#pragma unroll
            for (int c = 0; c < C; ++c)
                if ((int)threadIdx.x == c) {
                    to = rb[c];
                    tm = rmb[c];
                }
            dsmem_put_async(to + scw_off + (uint32_t)(8 * (buffer * C + rank)),
                            __hiloint2double(q, word), tm + 8u * (uint32_t)buffer);
        }
        all_to_all<T2M>(y);
#pragma unroll
        for (int j = 0; j < R; ++j)
            X[j] = {__double_as_longlong(y[j].re), __double_as_longlong(y[j].im)};
#pragma unroll
        for (int c = 0; c < C; ++c) {
            const int2 w = scw[buffer * C + c];
            qs[c] = w.y;
            bs[c] = (w.x << 4) >> 20;
            ls[c] = (w.x << 19) >> 20;
            bad |= (w.x & 1) != 0;
        }
    }
    CME_DEV static void twiddle(cx<T> (&x)[R], const TWC* w)
    {
#pragma unroll
        for (int j = 0; j < R; ++j)
            x[j] = cmul(x[j], w[j * CF::PC]);
    }
    // Cluster all-to-all.  Modes to time (T2M = false): the value of local position
    // n2 = l + PC j (k1 = rank) goes to block j mod C, slot rank G + j / C.  Time to modes:
    // slot i = k1 G + m of thread (rank, l) goes to block k1, slot rank + C m.  Every thread
    // reads its slots j at l + PC j of its own buffer.
    template <bool T2M>
    CME_DEV void all_to_all(cx<T> (&x)[R])
    {
        constexpr int PC = CF::PC, G = CF::G, W = Xbuf<T>::words_per_elem;
        if (timed_out) {
            // after a wait gave up this thread stores, arrives and waits no more, so no
            // mbarrier receives an arrival or bytes beyond the phase it is stuck in
            apar ^= 1;
            return;
        }
        const uint32_t po = (uint32_t)apar * (uint32_t)(CF::N2 * 8 * W);
        const uint32_t bo = 8u * (uint32_t)apar;   // mbarrier of buffer apar
#pragma unroll
        for (int j = 0; j < R; ++j) {
            if constexpr (T2M)
                abuf.put_remote_async(rb[j / G] + ot + po + (uint32_t)(8 * PC * C * (j % G)),
                                      x[j], rmb[j / G] + bo);
            else
                abuf.put_remote_async(rb[j % C] + om + po + (uint32_t)(8 * PC * (j / C)), x[j],
                                      rmb[j % C] + bo);
        }
        // the phase ends when this block's one arrival is in and all N2 values (FP64: and the
        // C scale words) have landed
        if (threadIdx.x == 0)
            mbar_arrive_expect_tx(mb + bo, (uint32_t)(CF::N2 * 8 * W + (FIX ? 8 * C : 0) +
                                                      (fault ? 8 : 0)));
        if (!mbar_wait(mb + bo, (ph >> apar) & 1u, fault ? 1024 : WAIT_TRIES))
            timed_out = true;   // the caller reports the instance
        ph ^= 1u << apar;
        const Xbuf<T> mine = abuf.at(apar * CF::N2);
#pragma unroll
        for (int j = 0; j < R; ++j)
            x[j] = mine.get(PC * j);
        apar ^= 1;
    }

    // F(x) = pump + i (g0/N) DFT(|a|^2 a), a = inverse transform of x   (Eq. 4)
    CME_DEV void rhs(cx<T> (&x)[R], T gN, cx<T> pump) { rhs_store_a(x, gN, pump, nullptr); }

    // The same, also storing the time-domain field a at aout[j P] unless aout is null.
    CME_DEV void rhs_store_a(cx<T> (&x)[R], T gN, cx<T> pump, cx<T>* aout)
    {
        if constexpr (FIX)
            fix_rhs(x, gN, aout);
        else
            float_rhs(x, gN, aout);
#pragma unroll
        for (int j = 0; j < R; ++j)
            x[j].im = -x[j].im;
        out_modes(x);
        if (t == 0)
            x[0] = cadd(x[0], pump);
    }
    // x becomes conj(i gN DFT(|a|^2 a)): both transforms and the Kerr term in fixed point
    CME_DEV void fix_rhs(cx<T> (&x)[R], T gN, cx<T>* aout)
    {
        fx X[R];
        const typename FT::Scale sc = FT::template load<TO_KERR>(x, X, red, tl());
        int q = sc.q;
        FixBound b = sc.b;
        bool bad = q == FT::POISON;
#pragma unroll 1
        for (int d = 0; d < 2; ++d) {
            fix_inverse(X, q, b, bad, d);
            if (d == 0) {
                if (aout) {
                    FT::store(X, bad ? -FT::POISON : -q, x);
#pragma unroll
                    for (int j = 0; j < R; ++j)
                        sstore(aout + j * P, x[j]);
                }
                const typename FT::Kerr k = FT::kerr(X, q, gN, red, tl());
                bad |= k.over;
                q = k.q;
                b = k.b;
            }
        }
        FT::store(X, bad ? -FT::POISON : -q, x);
    }
    CME_DEV void float_rhs(cx<T> (&x)[R], T gN, cx<T>* aout)
    {
#pragma unroll 1
        for (int d = 0; d < 2; ++d) {
            inverse(x, d);
            if (d == 0 && aout) {
#pragma unroll
                for (int j = 0; j < R; ++j)
                    sstore(aout + j * P, x[j]);
            }
            if (d == 0) {
                // conj(i c a) with c = (g0/N) |a|^2
#pragma unroll
                for (int j = 0; j < R; ++j) {
                    const T c = gN * (x[j].re * x[j].re + x[j].im * x[j].im);
                    x[j] = {-c * x[j].im, -c * x[j].re};
                }
            }
        }
    }

    static constexpr bool ACC_SMEM = C == 1 && acc_in_smem(sizeof(T), LOGN, R);
    cx<T>* accS;   // shared-memory accumulator S (ACC_SMEM), pre-offset by t
    cx<T>* accL;   // shared-memory compensation word (ACC_SMEM, FP32), pre-offset by t

    // Block-local set-up: thread index in the group, exchange buffers, addresses, twiddles.
    CME_DEV void setup(unsigned char* smem, int g, int t_, const void* tw_table)
    {
        constexpr int W = Xbuf<T>::words_per_elem;  // 8-byte words per element
        unsigned char* gbase = smem + (size_t)g * group_smem_bytes(sizeof(T), LOGN, R);
        double* base = reinterpret_cast<double*>(gbase);
        cx<T>* acc = reinterpret_cast<cx<T>*>(gbase + (size_t)2 * W * PL::BUF * 8);
        static_assert(xbuf_bytes(sizeof(T), LOGN) == (size_t)2 * W * PL::BUF * 8, "layout");
        accS = acc + t_;
        accL = acc + N + t_;
        red = reinterpret_cast<int2*>(gbase + xbuf_bytes(sizeof(T), LOGN) +
                                      acc_bytes(sizeof(T), LOGN, R) + tw_bytes(sizeof(T), LOGN, R));
        if constexpr (sizeof(T) == 4) {
            buf.p = reinterpret_cast<float2*>(base);
        } else {
            buf.re = base;           // buffer 0: re [0, BUF), im [BUF, 2 BUF)
            buf.stride = PL::BUF;    // buffer 1 starts at 2 BUF (Xbuf::at)
        }
        t = t_;
        ts = t_;
        par = 0;
        ad = TF::make_addr(t);
        if constexpr (TW_SMEM)
            tw.init(tw_table, t,
                    reinterpret_cast<cx<T>*>(gbase + xbuf_bytes(sizeof(T), LOGN) +
                                             acc_bytes(sizeof(T), LOGN, R)));
        else
            tw.init(tw_table, t);
        set_modes(N);
        km = nullptr;
    }

    // Cluster set-up (C > 1): block `rank` of the cluster, thread l of the block.  The block's
    // dynamic shared memory holds the two exchange buffers of its N2-point transform, the two
    // all-to-all receive buffers, the two twiddle arrays of the four-step transform, (FP32,
    // N2 >= 2048) the pass twiddles of the N2-point transform, the receive buffers' two
    // mbarriers and (FP64) their scale words and the reduction pairs.
    CME_DEV void setup_cluster(unsigned char* smem, int rank_, int l, const void* tw_table,
                               int a2a_fault)
    {
        static_assert(C > 1, "cluster groups only");
        constexpr int W = Xbuf<T>::words_per_elem, PC = CF::PC, N2 = CF::N2, G = CF::G;
        unsigned char* a2a = smem + (size_t)2 * TF::BUF * 8 * W;
        TWC* tws = reinterpret_cast<TWC*>(a2a + (size_t)2 * N2 * 8 * W);
        rank = rank_;
        if constexpr (sizeof(T) == 4) {
            buf.p = reinterpret_cast<float2*>(smem);
            abuf.p = reinterpret_cast<float2*>(a2a) + l;
        } else {
            buf.re = reinterpret_cast<double*>(smem);
            buf.stride = TF::BUF;
            abuf.re = reinterpret_cast<double*>(a2a) + l;
            abuf.stride = N2;
        }
        accS = nullptr;
        accL = nullptr;
        t = rank + C * l;
        ts = rank * PC + l;
        par = 0;
        apar = 0;
        ad = TF::make_addr(l);
        if constexpr (TW_SMEM)
            tw.init(tw_table, l, reinterpret_cast<cx<T>*>(tws + 2 * N2));
        else
            tw.init(tw_table, l);
        const uint32_t a0 = smem_addr(a2a);
        mb = smem_addr(reinterpret_cast<unsigned char*>(tws + 2 * N2) +
                       (TW_SMEM ? tw_bytes(sizeof(T), LOGN - LC, R) : 0));
#pragma unroll
        for (int c = 0; c < C; ++c) {
            rb[c] = dsmem_map(a0, c);
            rmb[c] = dsmem_map(mb, c);
        }
        if constexpr (FIX) {
            red = reinterpret_cast<int2*>(smem + cluster_smem_bytes<T, LOGN, R, C>() -
                                          red_bytes(sizeof(T), PC));
            scw = red - 2 * C;
            scw_off = smem_addr(scw) - a0;
        }
        // the kernel's cluster barrier before the first all-to-all publishes the initialisation
        if (l == 0) {
            mbar_init(mb, 1);
            mbar_init(mb + 8u, 1);
            mbar_init_fence();
        }
        ph = 0;
        timed_out = false;
        fault = a2a_fault;
        om = 8u * (uint32_t)(l + PC * rank * G);
        ot = 8u * (uint32_t)(l + PC * rank);
        // exp(2 pi i n2 k1 / N): after the block transform (n2 = l + PC j, k1 = rank), and
        // after the C-point transforms (n2 = rank PC + l + P (i mod G), k1 = i / G)
        const int tp = rank * PC + l;
        TWC* wm = tws + l;
        TWC* wt = tws + N2 + l;
        const auto tab = [&](int i) -> TWC {
            if constexpr (FIX)
                return __ldg(reinterpret_cast<const int4*>(tw_table) + i);
            else
                return gload<T>(tw_table, i);
        };
#pragma unroll
        for (int j = 0; j < R; ++j) {
            wm[j * PC] = tab(((l + PC * j) * rank) & (N - 1));
            wt[j * PC] = tab(((tp + P * (j % G)) * (j / G)) & (N - 1));
        }
        twm = wm;
        twt = wt;
        set_modes(N);
        km = nullptr;
    }
};

// Dynamic shared memory of one block of a cluster group (Group::setup_cluster).
template <typename T, int LOGN, int R, int C>
CME_HD constexpr size_t cluster_smem_bytes()
{
    using CF = ClusterFFT<T, LOGN, R, C>;
    constexpr size_t W = Xbuf<T>::words_per_elem;
    return (size_t)2 * CF::TL::BUF * 8 * W + (size_t)2 * CF::N2 * 8 * W +
           (size_t)2 * CF::N2 * sizeof(cx<T>) +
           (Group<T, LOGN, R, C>::TW_SMEM ? tw_bytes(sizeof(T), LOGN - CF::LC, R) : 0) + 16 +
           (Group<T, LOGN, R, C>::FIX ? 2 * C * 8 : 0) + red_bytes(sizeof(T), CF::PC);
}

template <typename T>
struct Coef;  // step coefficients in the field precision, converted once on the host
template <>
struct Coef<float> {
    CME_DEV static float h(const StepArgs& a) { return a.hf; }
    CME_DEV static float hh(const StepArgs& a) { return a.hhf; }
    CME_DEV static float h6(const StepArgs& a) { return a.h6f; }
};
template <>
struct Coef<double> {
    CME_DEV static double h(const StepArgs& a) { return a.h; }
    CME_DEV static double hh(const StepArgs& a) { return 0.5 * a.h; }
    CME_DEV static double h6(const StepArgs& a) { return a.h / 6.0; }
};

// nsteps steps of the instances [first, first + blockDim.x / P) of the group described by a
// (group-relative indices; groups past a.ninst recompute the last instance and store nothing).
// The evolving field of one thread: hi part in registers; the compensation word Dl (FP32) and
// the Runge-Kutta accumulator S in registers, or (ACC_SMEM) in this thread's own shared-memory
// slots t + jP.
template <typename T, int LOGN, int R, int C = 1>
struct FieldState {
    using GR = Group<T, LOGN, R, C>;
    static constexpr int P = GR::P;
    static constexpr bool COMP = GR::COMP, AS = GR::ACC_SMEM;
    cx<T> Dh[R];
    cx<T> Dlr[AS ? 1 : R];
    cx<T> Sr[AS ? 1 : R];
    cx<T>* accL;
    cx<T>* accS;

    CME_DEV void bind(const GR& grp)
    {
        accL = grp.accL;
        accS = grp.accS;
    }
    CME_DEV cx<T> getL(int j) const
    {
        if constexpr (!COMP)
            return cx<T>{T(0), T(0)};
        else if constexpr (AS)
            return accL[j * P];
        else
            return Dlr[j];
    }
    CME_DEV void setL(int j, cx<T> v)
    {
        if constexpr (COMP) {
            if constexpr (AS)
                accL[j * P] = v;
            else
                Dlr[j] = v;
        }
    }
    CME_DEV cx<T> getS(int j) const
    {
        if constexpr (AS)
            return accS[j * P];
        else
            return Sr[j];
    }
    CME_DEV void setS(int j, cx<T> v)
    {
        if constexpr (AS)
            accS[j * P] = v;
        else
            Sr[j] = v;
    }
    // D += d (compensated two-sum in FP32)
    CME_DEV void add(int j, cx<T> d)
    {
        cx<T> l = getL(j);
        accumulate<T, COMP>(Dh[j], l, d);
        setL(j, l);
    }
    CME_DEV void load(const cx<T>* hi, const cx<T>* lo)
    {
#pragma unroll
        for (int j = 0; j < R; ++j) {
            Dh[j] = hi[j * P];
            if constexpr (COMP)
                setL(j, lo[j * P]);
        }
    }
    CME_DEV void store(cx<T>* hi, cx<T>* lo) const
    {
#pragma unroll
        for (int j = 0; j < R; ++j) {
            hi[j * P] = Dh[j];
            if constexpr (COMP)
                lo[j * P] = getL(j);
        }
    }
};

// Instance constants of the step loops.
template <typename T>
struct StepConsts {
    cx<T> pump;   // sqrt(kappa_ext) A_in
    cx<T> cp;     // Strang pump increment over h/2
    cx<T> cp2;    // ... over h
    T gN;         // g0 / N
    T g0h;        // g0 h / 2 (Strang half phase per |a|^2)
    T h, hh, h6;
};

// One RK4IP step (Sec. 2 "fourth-order Runge-Kutta"; Hult 2007) written as increments of D:
//   x2 = D + (e1 D + h/2 k1),  x3 = D + (e1 D + h/2 k2),  x4 = D + (e2 D + h E k3),
//   D' = D + e2 D + h/6 [E (k1 + 2 k2 + 2 k3) + k4],  k1 = E F(D),  k_i = F(x_i),
// with E = exp(L h/2), e1 = expm1(L h/2), e2 = expm1(L h).  The four stages share one copy of
// the right-hand-side code (a runtime loop).
// STAGES = true also stores, unless so is null (the adjoint's recomputation), the right-hand-side
// values y1 = F(D), k2 = F(x2), k3 = F(x3) of the thread's positions at so[st * sstride + j P],
// st = 0, 1, 2, and the time-domain fields a of the four stage inputs D, x2, x3, x4 at
// so[(3 + st) * sstride + j P], st = 0..3.
template <bool STAGES, bool CACHE = false, typename T, int LOGN, int R, int C>
CME_DEV void rk4ip_step_impl(Group<T, LOGN, R, C>& grp, FieldState<T, LOGN, R, C>& fs,
                             const Props<T, LOGN, R, C>& pr, const StepConsts<T>& c, cx<T>* so,
                             long long sstride)
{
    constexpr bool COMP = Group<T, LOGN, R, C>::COMP;
    constexpr int P = Group<T, LOGN, R, C>::P;
    constexpr bool PK = packed_twiddles(LOGN, R);
    cx<T> x[R];
    // CACHE: e1 D (stages 0, 1), then e2 D (stages 2, 3) computed once and kept in registers
    // across the stage's transforms (kernels with registers to spare); else recomputed
    cx<T> eD[CACHE ? R : 1];
#pragma unroll
    for (int j = 0; j < R; ++j)
        x[j] = fs.Dh[j];
    // one RK stage (st = 0 ... 3)
    auto stage = [&](int st) {
        if constexpr (STAGES)
            grp.rhs_store_a(x, c.gN, c.pump, so ? so + (3 + st) * sstride : nullptr);
        else
            grp.rhs(x, c.gN, c.pump);
        if constexpr (STAGES) {
            if (st < 3 && so) {
#pragma unroll
                for (int j = 0; j < R; ++j)
                    sstore(so + st * sstride + j * P, x[j]);
            }
        }
        if (st == 0) {
#pragma unroll
            for (int j = 0; j < R; ++j) {
                const cx<T> E = pr.getE(j);
                const cx<T> k1 = cmul_pk<PK>(E, x[j]);
                fs.setS(j, cmul_pk<PK>(E, k1));
                const cx<T> e1D = cmul_pk<PK>(pr.get1(j), fs.Dh[j]);
                if constexpr (CACHE)
                    eD[j] = e1D;
                x[j] = cadd(fs.Dh[j], caxpy(e1D, c.hh, k1));
            }
        } else if (st == 1) {
#pragma unroll
            for (int j = 0; j < R; ++j) {
                fs.setS(j, caxpy(fs.getS(j), T(2), cmul_pk<PK>(pr.getE(j), x[j])));
                cx<T> e1D;
                if constexpr (CACHE)
                    e1D = eD[j];
                else
                    e1D = cmul_pk<PK>(pr.get1(j), fs.Dh[j]);
                x[j] = cadd(fs.Dh[j], caxpy(e1D, c.hh, x[j]));
            }
        } else if (st == 2) {
#pragma unroll
            for (int j = 0; j < R; ++j) {
                const cx<T> Ek3 = cmul_pk<PK>(pr.getE(j), x[j]);
                fs.setS(j, caxpy(fs.getS(j), T(2), Ek3));
                const cx<T> e2D = cmul_pk<PK>(pr.get2(j), fs.Dh[j]);
                if constexpr (CACHE)
                    eD[j] = e2D;
                x[j] = cadd(fs.Dh[j], caxpy(e2D, c.h, Ek3));
            }
        } else {
#pragma unroll
            for (int j = 0; j < R; ++j) {
                const cx<T> e2 = pr.get2(j);
                cx<T> d;
                if constexpr (CACHE)
                    d = eD[j];
                else
                    d = cmul_pk<PK>(e2, fs.Dh[j]);
                if constexpr (COMP)
                    d = cadd(d, cmul_pk<PK>(e2, fs.getL(j)));
                d = caxpy(d, c.h6, cadd(fs.getS(j), x[j]));
                fs.add(j, d);
            }
        }
    };
    // One-block CACHE kernels (registers to spare) take the four stages unrolled: 51.6 -> 49.4
    // ms per headline run.  Elsewhere one copy of the stage code in a loop keeps the
    // instruction footprint small: unrolled, the 8-block cluster kernel of N = 4096 took 6.9
    // instead of 5.1 us per step.
    if constexpr (CACHE && C == 1) {
#pragma unroll
        for (int st = 0; st < 4; ++st)
            stage(st);
    } else {
#pragma unroll 1
        for (int st = 0; st < 4; ++st)
            stage(st);
    }
}

// One RK4IP step of an FP64 group with the stages in fixed point (cme_fixed.cuh).  The
// state D, its propagation and the step's increment are FP64; what only enters a right-hand side
// (the stage inputs) or the increment (the right-hand sides and their sum) stays in fixed
// point, each on its own block scale, as in
//     Y1 = h/2 F(D),    U = E D,  A = E Y1,   x2 = U + A,
//     Y2 = h/2 F(x2),   A += 2 Y2,            x3 = U + Y2,
//     Y3 = h F(x3),     A += Y3,              x4 = E (U + Y3),
//     Y4 = h/2 F(x4),   D' = D + [expm1(L h) D + (E A + Y4) / 3],
// the same step as rk4ip_step_impl.  Per mode and step that leaves 8 FP64 instructions of the 74
// outside the transforms, and one conversion from and one to FP64 instead of four each.
// N = 512 x 256: 88.5 us per step with FP64 instructions throughout (bound by their pipe), 36.8
// with only the transforms and the Kerr term in fixed point, 21.7 with the stages.  One N = 64
// instance: 19.5, 11.7 and 7.2 us.  What bounds it now is one warp per scheduler issuing dependent
// integer instructions (fixed-latency waits, 1.4 per issue).
// The error of a step against extended precision on the small modes of a comb (1e-6 beside a
// pumped mode of 1.3, h = 2e-4): 1.1e-21 at N = 512 and 1.2e-21 at 4096, from 4.9e-21 and 1.6e-21
// in FP64 instructions.  It is set by the units of the stage inputs and of the increment, so both
// keep every bit the bounds leave (fcmul1, not fcmul4, there).
// park: where the state waits in global memory during the step (groups whose registers and shared
// memory are full: ACC_SMEM), else unused.  STAGES: as in rk4ip_step_impl.
template <bool STAGES, int LOGN, int R, int C>
CME_DEV void fix_rk4ip_step(Group<double, LOGN, R, C>& grp, FieldState<double, LOGN, R, C>& fs,
                            const Props<double, LOGN, R, C>& pr, const StepConsts<double>& c,
                            cx<double>* park, cx<double>* so, long long sstride)
{
    using GR = Group<double, LOGN, R, C>;
    using FT = typename GR::FT;
    constexpr int P = GR::P;
    constexpr bool AS = GR::ACC_SMEM;
    fx X[R], U[R], Ar[AS ? 1 : R];
    auto getA = [&](int j) -> fx {
        if constexpr (AS) {
            const cx<double> v = grp.accS[j * P];
            return {__double_as_longlong(v.re), __double_as_longlong(v.im)};
        } else {
            return Ar[j];
        }
    };
    auto setA = [&](int j, fx v) {
        if constexpr (AS)
            grp.accS[j * P] = {__longlong_as_double(v.re), __longlong_as_double(v.im)};
        else
            Ar[j] = v;
    };
    const typename FT::Scale sc = FT::template load<GR::TO_KERR>(fs.Dh, X, grp.red, grp.tl());
    if constexpr (AS) {
#pragma unroll
        for (int j = 0; j < R; ++j)
            park_store(park + j * P, fs.Dh[j]);
    }
    bool bad = sc.q == FT::POISON;
    FixBound b = sc.b;
    int q = bad ? 0 : sc.q, bY = 0, qU = q, bU = min(b.bm, b.bl), qA = 0, bA = 0;
#pragma unroll
    for (int j = 0; j < R; ++j)
        U[j] = X[j];
    const double gh = c.gN * c.hh;
    const cx<double> pump = cscale(c.pump, c.hh);
    // |pump| < 2^eP (in the block that holds mode 0)
    const int eP = C > 1 && grp.rank != 0
                       ? -4000
                       : (int)(max(FT::habs(pump.re), FT::habs(pump.im)) >> 20) - 1022 + 1;
#pragma unroll 1
    for (int st = 0; st < 4; ++st) {
        // X becomes Y of this stage, scale q, modulus below 2^bY
#pragma unroll 1
        for (int d = 0; d < 2; ++d) {
            bY = grp.fix_inverse(X, q, b, bad, d);
            if (d == 0) {
                if constexpr (STAGES) {
                    if (so) {
                        cx<double> a[R];
                        FT::store(X, bad ? -FT::POISON : -q, a);
#pragma unroll
                        for (int j = 0; j < R; ++j)
                            sstore(so + (3 + st) * sstride + j * P, a[j]);
                    }
                }
                const typename FT::Kerr k = FT::kerr(X, q, gh, grp.red, grp.tl());
                bad |= k.over;
                q = k.q - (st == 2);
                b = k.b;
            }
        }
        // the sum with the pump stays below 2^62
        const int s = max(eP + (st == 2) + q, bY) - 61;
        if (s > 0) {
#pragma unroll
            for (int j = 0; j < R; ++j)
                X[j] = {frsh(X[j].re, min(s, 63)), frsh(X[j].im, min(s, 63))};
            q -= s;
            bY -= s;
        }
        bY = max(bY, eP + (st == 2) + q) + 1;
#pragma unroll
        for (int j = 0; j < R; ++j) {
            X[j].im = -X[j].im;
            if (!grp.physical(j))
                X[j] = {0, 0};
        }
        if (grp.t == 0) {
            const int c0 = 1085 - q - (st == 2);
            X[0] = fadd(X[0], {FT::template fix<true>(pump.re, c0),
                               FT::template fix<true>(pump.im, c0)});
        }
        if constexpr (STAGES) {
            if (so && st < 3) {
                cx<double> y[R];
                FT::store(X, bad ? -FT::POISON : -q, y);
                const double ih = 1.0 / (st == 2 ? c.h : c.hh);
#pragma unroll
                for (int j = 0; j < R; ++j)
                    sstore(so + st * sstride + j * P, cscale(y[j], ih));
            }
        }
        if (st == 3)
            break;
        if (st == 0) {
            qA = q - 2;
            bA = bY - 2;
            const typename FT::Align al = FT::align(qU, bU, qA, bA);
#pragma unroll
            for (int j = 0; j < R; ++j) {
                const fl2 E = pr.getF(j);
                const fx a = fcmul4(X[j], E);
                U[j] = fcmul1(U[j], E);
                setA(j, a);
                X[j] = FT::template asum<false>(U[j], a, al);
            }
            q = al.q;
        } else {
            // A += (2 or 1) Y
            const typename FT::Align aa = FT::align(qA, bA, q - (st == 1), bY);
            bA = aa.b;
            qA = aa.q;
            const typename FT::Align al = FT::align(qU, bU, q, bY);
#pragma unroll
            for (int j = 0; j < R; ++j) {
                setA(j, FT::template asum<true>(getA(j), X[j], aa));
                X[j] = FT::template asum<false>(U[j], X[j], al);
            }
            q = al.q;
            if (st == 2)
#pragma unroll
                for (int j = 0; j < R; ++j)
                    X[j] = fcmul1(X[j], pr.getF(j));
        }
        b = FT::bounds(X, grp.red, grp.tl());
        q += FT::template rescale<GR::TO_KERR>(X, b);
    }
    // the increment (E A + Y4) / 3
    // (unscaled product: the increment's unit, relative to its largest mode, is what limits the
    // accuracy of the small ones)
    const typename FT::Align al = FT::align(qA, bA, q, bY);
#pragma unroll
    for (int j = 0; j < R; ++j)
        X[j] = FT::template asum<true>(fcmul1(getA(j), pr.getF(j)), X[j], al);
    cx<double> w[R];
    FT::store(X, bad ? -FT::POISON : -al.q, w);
#pragma unroll
    for (int j = 0; j < R; ++j) {
        if constexpr (AS)
            fs.Dh[j] = park_load(park + j * P);
        const cx<double> d = cmul(pr.get2(j), fs.Dh[j]);
        fs.Dh[j] = cadd(fs.Dh[j], caxpy(d, 1.0 / 3.0, w[j]));
    }
}

// Whether a step kernel has the registers to keep e1 D / e2 D across a stage (FP32 at 8 values
// per thread, at most 256 threads per block: N = 512, 64 threads, 168 -> 192 registers), not
// in the work-list kernel, whose tiles share one register budget.
template <typename T, int LOGN, int R, int C>
CME_HD constexpr bool rk_cache_ed()
{
    return sizeof(T) == 4 && R <= 8 && Plan<LOGN, R>::P / C <= 256;
}

// The RK4IP step: FP64 in fixed point, except with per-mode Kerr factors (of any size, so without
// a common scale).
template <bool STAGES, bool CACHE, typename T, int LOGN, int R, int C>
CME_DEV void rk4ip_step(Group<T, LOGN, R, C>& grp, FieldState<T, LOGN, R, C>& fs,
                        const Props<T, LOGN, R, C>& pr, const StepConsts<T>& c, cx<T>* park,
                        cx<T>* so, long long sstride)
{
    if constexpr (sizeof(T) == 8) {
        if (!grp.km) {
            fix_rk4ip_step<STAGES>(grp, fs, pr, c, park, so, sstride);
            return;
        }
    }
    rk4ip_step_impl<STAGES, CACHE>(grp, fs, pr, c, so, sstride);
}

// sin y and cos y in FP32 for the Strang Kerr phase y = g0 |a|^2 h / 2, which is small in any
// resolved step.  For |y| <= 1/2 the Taylor series of sin (to y^9) and cos (to y^8), evaluated
// in y^2 by Horner's rule, leave truncation errors below y^11/11! <= 1.2e-11 and
// y^10/10! <= 2.7e-10, far under FP32 rounding; larger |y| (small_phase false) take sincosf.
CME_DEV void taylor_sincos(float y, float& s, float& c)
{
    const float y2 = y * y;
    s = y * (1.f + y2 * (-1.f / 6 + y2 * (1.f / 120 + y2 * (-1.f / 5040 + y2 * (1.f / 362880)))));
    c = 1.f + y2 * (-0.5f + y2 * (1.f / 24 + y2 * (-1.f / 720 + y2 * (1.f / 40320))));
}
CME_DEV bool small_phase(float y) { return fabsf(y) <= 0.5f; }   // false for NaN

// Linear and pump flow of the Strang step, exact, applied as the increment D += e D + c: over
// h/2 (full = false: e = expm1(L h/2), c = (exp(L_0 h/2) - 1)/L_0 sqrt(kappa_ext) A_in on the
// pumped mode) or over h (full = true: e = expm1(L h), c the same over h).
template <typename T, int LOGN, int R, int C>
CME_DEV void strang_linear(const Group<T, LOGN, R, C>& grp, FieldState<T, LOGN, R, C>& fs,
                           const Props<T, LOGN, R, C>& pr, const StepConsts<T>& c, bool full)
{
    constexpr bool COMP = Group<T, LOGN, R, C>::COMP;
#pragma unroll
    for (int j = 0; j < R; ++j) {
        const cx<T> e = full ? pr.get2(j) : pr.get1(j);
        cx<T> d = cmul_pk<packed_twiddles(LOGN, R)>(e, fs.Dh[j]);
        if constexpr (COMP)
            d = cadd(d, cmul_pk<packed_twiddles(LOGN, R)>(e, fs.getL(j)));
        if (j == 0 && grp.t == 0)
            d = cadd(d, full ? c.cp2 : c.cp);
        fs.add(j, d);
    }
}

// The same in fixed point (FP64): both transforms, the phase and its exponential.
template <bool STORE, int LOGN, int R, int C>
CME_DEV void fix_strang_kerr(Group<double, LOGN, R, C>& grp, FieldState<double, LOGN, R, C>& fs,
                             const StepConsts<double>& c, cx<double>* so, long long sstride)
{
    using GR = Group<double, LOGN, R, C>;
    using FT = typename GR::FT;
    constexpr int P = GR::P;
    fx X[R];
    cx<double> x[R];
    const typename FT::Scale sc = FT::template load<GR::TO_KERR>(fs.Dh, X, grp.red, grp.tl());
    FixBound b = sc.b;
    int q = sc.q;
    bool bad = q == FT::POISON;
#pragma unroll 1
    for (int d = 0; d < 2; ++d) {
        grp.fix_inverse(X, q, b, bad, d);
        if (d == 0) {
            if constexpr (STORE) {
                if (so) {
                    FT::store(X, bad ? -FT::POISON : -q, x);
#pragma unroll
                    for (int j = 0; j < R; ++j)
                        sstore(so + j * P, x[j]);
                }
            }
            const typename FT::Kerr k =
                FT::template kerr_flow<LOGN>(X, q, 2.0 * c.g0h, bad, grp.red, grp.tl());
            bad |= k.over;
            q = k.q;
            b = k.b;
        }
    }
    FT::store(X, bad ? -FT::POISON : -q, x);
    grp.mask(x);   // no Kerr increment on padding modes
#pragma unroll
    for (int j = 0; j < R; ++j)
        fs.add(j, cx<double>{x[j].re, -x[j].im});
    if constexpr (STORE) {
        if (so) {
#pragma unroll
            for (int j = 0; j < R; ++j)
                sstore(so + sstride + j * P, fs.Dh[j]);
        }
    }
}

// Exact Kerr flow of the Strang step over h.  With a = inverse transform of D the flow is
// a -> a exp(i g0 |a|^2 h); it is applied as the increment D += DFT(a expm1(i g0 |a|^2 h))/N.
// STORE = true also stores, unless so is null (the adjoint's recomputation), the time-domain
// field a at so[j P] and the state after the flow at so[sstride + j P].
template <bool STORE, typename T, int LOGN, int R, int C>
CME_DEV void strang_kerr(Group<T, LOGN, R, C>& grp, FieldState<T, LOGN, R, C>& fs,
                         const StepConsts<T>& c, cx<T>* so, long long sstride)
{
    if constexpr (sizeof(T) == 8) {
        fix_strang_kerr<STORE>(grp, fs, c, so, sstride);
    } else {
    constexpr int P = Group<T, LOGN, R, C>::P;
    constexpr T invN = (T)(1.0 / (1 << LOGN));
    cx<T> x[R];
#pragma unroll
    for (int j = 0; j < R; ++j)
        x[j] = fs.Dh[j];
#pragma unroll 1
    for (int d = 0; d < 2; ++d) {
        grp.inverse(x, d);
        if constexpr (STORE) {
            if (d == 0 && so) {
#pragma unroll
                for (int j = 0; j < R; ++j)
                    sstore(so + j * P, x[j]);
            }
        }
        if (d == 0) {
            // expm1(i phi) = (-2 sin^2(phi/2), sin(phi)), phi = g0 |a|^2 h; the forward
            // transform runs as conj(inverse(conj(.))).  FP32: the Taylor series for every
            // value, then sincosf only for values outside its range, behind one branch per
            // thread rather than one per value
            T ph2[R], sn[R], cs[R];
            bool big = false;
#pragma unroll
            for (int j = 0; j < R; ++j) {
                ph2[j] = c.g0h * (x[j].re * x[j].re + x[j].im * x[j].im);
                if constexpr (sizeof(T) == 4) {
                    taylor_sincos(ph2[j], sn[j], cs[j]);
                    big |= !small_phase(ph2[j]);
                } else {
                    sincos(ph2[j], &sn[j], &cs[j]);
                }
            }
            if constexpr (sizeof(T) == 4) {
                if (big) {
#pragma unroll
                    for (int j = 0; j < R; ++j)
                        if (!small_phase(ph2[j]))
                            sincosf(ph2[j], &sn[j], &cs[j]);
                }
            }
#pragma unroll
            for (int j = 0; j < R; ++j) {
                const cx<T> em = {T(-2) * sn[j] * sn[j] * invN, T(2) * sn[j] * cs[j] * invN};
                const cx<T> b = cmul(x[j], em);
                x[j] = {b.re, -b.im};
            }
        }
    }
    grp.mask(x);   // no Kerr increment on padding modes
#pragma unroll
    for (int j = 0; j < R; ++j)
        fs.add(j, cx<T>{x[j].re, -x[j].im});
    if constexpr (STORE) {
        if (so) {
#pragma unroll
            for (int j = 0; j < R; ++j)
                sstore(so + sstride + j * P, fs.Dh[j]);
        }
    }
    }
}

// One Strang split step (Sec. 2 "split-step Fourier method ... field in the frequency domain"):
// exact linear+pump flow over h/2, exact Kerr flow over h, exact linear+pump flow over h/2.
// The adjoint's recomputation takes the steps one by one (STORE: see strang_kerr).
template <bool STORE, typename T, int LOGN, int R, int C>
CME_DEV void strang_step_impl(Group<T, LOGN, R, C>& grp, FieldState<T, LOGN, R, C>& fs,
                              const Props<T, LOGN, R, C>& pr, const StepConsts<T>& c, cx<T>* so,
                              long long sstride)
{
    strang_linear(grp, fs, pr, c, false);
    strang_kerr<STORE>(grp, fs, c, so, sstride);
    strang_linear(grp, fs, pr, c, false);
}

// n Strang steps as the step kernels take them: the half flow that closes a step and the half
// flow that opens the next compose exactly into the flow over h (exp(L h/2)^2 = exp(L h), and
// the pump increments into the increment over h), so the n steps apply n + 1 linear flows
// instead of 2n.  The field after the n steps is that of n single steps up to rounding.
template <typename T, int LOGN, int R, int C>
CME_DEV void strang_steps(Group<T, LOGN, R, C>& grp, FieldState<T, LOGN, R, C>& fs,
                          const Props<T, LOGN, R, C>& pr, const StepConsts<T>& c, long long n)
{
    if (n <= 0)
        return;
    strang_linear(grp, fs, pr, c, false);
    for (long long k = 0; k < n; ++k) {
        strang_kerr<false>(grp, fs, c, static_cast<cx<T>*>(nullptr), 0);
        strang_linear(grp, fs, pr, c, k + 1 < n);
    }
}

template <typename T>
CME_DEV StepConsts<T> step_consts(const StepArgs& a, int inst, int N)
{
    StepConsts<T> c;
    const double2 pd = a.pump[inst];
    c.pump = {(T)pd.x, (T)pd.y};
    const double2 cpd = a.cpump[inst];
    c.cp = {(T)cpd.x, (T)cpd.y};
    const double2 cpd2 = a.cpump2 ? a.cpump2[inst] : make_double2(0.0, 0.0);
    c.cp2 = {(T)cpd2.x, (T)cpd2.y};
    c.gN = (T)(a.g0[inst] / (double)N);
    c.g0h = (T)(a.g0[inst] * a.h * 0.5);
    c.h = Coef<T>::h(a);
    c.hh = Coef<T>::hh(a);
    c.h6 = Coef<T>::h6(a);
    return c;
}

// nsteps steps of the instances [first, first + blockDim.x / P) of the group described by a
// (group-relative indices; groups past a.ninst recompute the last instance and store nothing).
// MASKABLE = false compiles the body without the physical-mode mask (every instance M = N):
// the mask test then folds away at compile time.
template <typename T, int LOGN, int R, int METHOD, bool MASKABLE = true, bool FUSED = false>
CME_DEV void step_body(const StepArgs& a, int first, unsigned char* smem)
{
    using GR = Group<T, LOGN, R>;
    constexpr int N = GR::N, P = GR::P;

    const int g = threadIdx.x / P;
    int inst = first + g;
    const bool valid = inst < a.ninst;
    if (!valid)
        inst = a.ninst - 1;  // duplicate work keeps every group in the barriers; no store
    GR grp;
    grp.setup(smem, g, threadIdx.x - g * P, a.tw);
    const long long off = a.base + (long long)inst * N;
    if constexpr (MASKABLE) {
        if (a.phys)
            grp.set_modes(a.phys[inst]);
        grp.set_kerr(a.kerr, off);
    }
    const int t = grp.t;

    cx<T>* hi = reinterpret_cast<cx<T>*>(a.hi) + off + t;
    cx<T>* lo = reinterpret_cast<cx<T>*>(a.lo) + off + t;
    FieldState<T, LOGN, R> fs;
    fs.bind(grp);
    fs.load(hi, lo);
    const StepConsts<T> c = step_consts<T>(a, inst, N);
    Props<T, LOGN, R> pr;
    pr.init(a, off, t);

    if constexpr (METHOD == METHOD_RK4IP) {
        for (long long n = 0; n < a.nsteps; ++n)
            rk4ip_step<false, !FUSED && rk_cache_ed<T, LOGN, R, 1>()>(
                grp, fs, pr, c, hi, static_cast<cx<T>*>(nullptr), 0);
    } else {
        strang_steps(grp, fs, pr, c, a.nsteps);
    }

    bool bad = false;
#pragma unroll
    for (int j = 0; j < R; ++j)
        bad |= !(isfinite(fs.Dh[j].re) && isfinite(fs.Dh[j].im));
    if (valid) {
        fs.store(hi, lo);
        if (bad)
            a.status[inst] = 1;
    }
}

// Blocks an SM has to hold (the register limit that sets): FP32 N = 1024 at 8 values per thread
// three, not the two that 190 registers leave (167, 56 bytes spilled; split step 162, none).  us per
// step before, with the packed arithmetic in it / now, RK4IP 1 instance 4.04 / 3.60, 300 5.66 / 5.09,
// 400 10.6 / 6.8, 900 16.9 / 13.5; split step 1.10 / 1.09, 1.87 / 1.65, 2.49 / 2.25, 4.89 / 4.33; with
// padding modes RK4IP 4.79 / 4.19, 6.15 / 5.64, 12.0 / 7.4, 18.3 / 14.6, split step 1.14 / 1.10,
// 1.89 / 1.68, 2.42 / 2.31, 4.74 / 4.47.
template <typename T, int LOGN, int R>
constexpr int min_blocks() { return sizeof(T) == 4 && LOGN == 10 && R == 8 ? 3 : 1; }

template <typename T, int LOGN, int R, int METHOD, bool MASKABLE>
__global__ void __launch_bounds__(max_threads<LOGN, R>(), min_blocks<T, LOGN, R>())
    step_kernel(const StepArgs a)
{
    extern __shared__ __align__(16) unsigned char smem[];
    step_body<T, LOGN, R, METHOD, MASKABLE>(a, blockIdx.x * a.G, smem);
}

// The same steps with each instance spread over a cluster of C blocks (P/C threads each);
// launched with a grid of exactly ninst * C blocks and cluster dimension C, so every block
// holds a real instance and all of them take part in every cluster barrier.
template <typename T, int LOGN, int R, int C, int METHOD>
__global__ void __launch_bounds__(Plan<LOGN, R>::P / C) cluster_step_kernel(const StepArgs a)
{
    using GR = Group<T, LOGN, R, C>;
    constexpr int N = GR::N;
    extern __shared__ __align__(16) unsigned char smem[];
    const int inst = blockIdx.x / C;
    GR grp;
    grp.setup_cluster(smem, cluster_rank(), threadIdx.x, a.tw, a.a2a_fault);
    const long long off = a.base + (long long)inst * N;
    if (a.phys)
        grp.set_modes(a.phys[inst]);
    grp.set_kerr(a.kerr, off);
    const int t = grp.t;

    cx<T>* hi = reinterpret_cast<cx<T>*>(a.hi) + off + t;
    cx<T>* lo = reinterpret_cast<cx<T>*>(a.lo) + off + t;
    FieldState<T, LOGN, R, C> fs;
    fs.bind(grp);
    fs.load(hi, lo);
    const StepConsts<T> c = step_consts<T>(a, inst, N);
    Props<T, LOGN, R, C> pr;
    pr.init(a, off, t);
    cluster_sync();   // every block of the cluster runs before the first remote store

    if constexpr (METHOD == METHOD_RK4IP) {
        for (long long n = 0; n < a.nsteps; ++n)
            rk4ip_step<false, rk_cache_ed<T, LOGN, R, C>()>(grp, fs, pr, c, hi,
                                                            static_cast<cx<T>*>(nullptr), 0);
    } else {
        strang_steps(grp, fs, pr, c, a.nsteps);
    }

    bool bad = false;
#pragma unroll
    for (int j = 0; j < R; ++j)
        bad |= !(isfinite(fs.Dh[j].re) && isfinite(fs.Dh[j].im));
    fs.store(hi, lo);
    if (bad)
        a.status[inst] = 1;
    if (grp.failed())
        a.status[inst] = 2;
    cluster_sync();   // no block leaves while a peer may still address its shared memory
}

// Diagnostics: one transform or one right-hand-side evaluation of the current field, written in
// transform order to a.diag_out (same layout as the field).
template <typename T, int LOGN, int R>
__global__ void __launch_bounds__(max_threads<LOGN, R>()) diag_kernel(const StepArgs a)
{
    using GR = Group<T, LOGN, R>;
    constexpr int N = GR::N, P = GR::P;
    extern __shared__ __align__(16) unsigned char smem[];
    const int g = threadIdx.x / P;
    int inst = blockIdx.x * a.G + g;
    const bool valid = inst < a.ninst;
    if (!valid)
        inst = a.ninst - 1;
    GR grp;
    grp.setup(smem, g, threadIdx.x - g * P, a.tw);
    const long long off = a.base + (long long)inst * N;
    if (a.phys)
        grp.set_modes(a.phys[inst]);
    grp.set_kerr(a.kerr, off);
    const int t = grp.t;
    const cx<T>* src = reinterpret_cast<const cx<T>*>(a.hi) + off + t;
    cx<T>* dst = reinterpret_cast<cx<T>*>(a.diag_out) + off + t;
    cx<T> x[R];
#pragma unroll
    for (int j = 0; j < R; ++j)
        x[j] = src[j * P];
    if (a.diag_mode == DIAG_IDFT) {
        grp.inverse(x, 0);
    } else if (a.diag_mode == DIAG_DFT) {
        if constexpr (GR::FIX) {
#pragma unroll
            for (int j = 0; j < R; ++j)
                x[j].im = -x[j].im;
            grp.inverse(x, 1);
#pragma unroll
            for (int j = 0; j < R; ++j)
                x[j].im = -x[j].im;
        } else {
            GR::TF::template run<-1>(x, grp.tw, grp.buf, grp.par, grp.ad);
        }
    } else {
        const double2 pd = a.pump[inst];
        grp.rhs(x, (T)(a.g0[inst] / (double)N), cx<T>{(T)pd.x, (T)pd.y});
    }
    if (valid) {
#pragma unroll
        for (int j = 0; j < R; ++j)
            dst[j * P] = x[j];
    }
}

}  // namespace CME_FP32_VARIANT
}  // namespace cme
