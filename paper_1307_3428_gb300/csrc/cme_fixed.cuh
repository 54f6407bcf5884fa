// FP64 transforms in 64-bit fixed point.
//
// FP64 instructions run at 1/64 of the FP32 rate on this GPU: a DADD or DFMA holds its scheduler
// for 64 to 76 cycles, where a 64-bit integer add takes 3 and a 32 x 32 -> 64 multiply about 4
// (one warp per scheduler).  A transform only adds, subtracts and rotates, and every
// intermediate value is a partial sum of unit-modulus multiples of its inputs, so its modulus is
// at most L1 = sum |x_k|.  The FP64 kernels therefore scale a group's values by one power of two
// such that this bound fits 61 bits, run the passes on integers, and convert back.  The rounding
// of a pass is then 2^-61 of the bound instead of 2^-53 of each value; against extended precision
// the transforms are 1.2 to 3 times closer than FP64 ones (N = 4 ... 4096).
// One radix-8 pass with its twiddles takes about 1100 cycles a warp (8 values per thread, one warp per
// scheduler), where its 84 FP64 instructions per thread took about 6000.
//
// Scale.  One reduction per transform gives the largest exponent and L1.  A group of unrelated
// modes has L1 ~ sqrt(N) times its 2-norm and would leave its values log2(N) bits low; so the scale
// follows the bounds after every pass, min(L1, (product of the radices so far) |x|max), less the
// two bits by which each twiddled pass scales down (FixTransform::headroom).  Both bounds are
// the group's own, powers of two, and independent of the order of the reduction.
//
// Multiplication.  A value is x = h 2^32 + l with h and l signed 32-bit ("balanced" limbs: l is
// the low word read as signed, h the high word plus its carry), so every partial product is a
// signed 32 x 32 -> 64 multiply; l l' is below one unit of the result and is dropped.
#pragma once

#include "cme_core.cuh"

namespace cme {
inline namespace CME_FP32_VARIANT {

struct fx {   // fixed-point complex value
    long long re, im;
};
struct fl {   // balanced limbs
    int h, l;
};
struct fl2 {  // limbs of a complex factor w: w 2^62
    fl re, im;
};

CME_DEV fl fsplit(long long v)
{
    const unsigned lo = (unsigned)v;
    return {(int)((unsigned)(v >> 32) + (lo >> 31)), (int)lo};
}
// a b, a b + c and v 2^s
#ifndef CME_HOST_PRIMITIVES   // (a host build supplies these, with overflow checks)
CME_DEV long long fwide(int a, int b)
{
    long long d;
    asm("mul.wide.s32 %0, %1, %2;" : "=l"(d) : "r"(a), "r"(b));
    return d;
}
CME_DEV long long fmad(int a, int b, long long c)
{
    long long d;
    asm("mad.wide.s32 %0, %1, %2, %3;" : "=l"(d) : "r"(a), "r"(b), "l"(c));
    return d;
}
CME_DEV long long fshl(long long v, int s) { return (long long)((unsigned long long)v << s); }
#endif
CME_DEV int fhi(long long v) { return (int)(v >> 32); }

// Products.  The middle sum (h l' + l h') 2^-32 is taken as the difference of two floors, whose
// biases of half a unit cancel; a constant would turn zeros into units.  It is added as a product
// with 1: the sign extension and the 64-bit add would take three instructions of the pipe that
// the rest already fills.

// (x y) 2^-64
CME_DEV long long fmulhi(fl x, fl y)
{
    const int t = fhi(fwide(x.l, y.h)) - fhi(fwide(-x.h, y.l));
    return fmad(t, 1, fwide(x.h, y.h));
}
// v 2^-s, rounded to nearest, ties to even.  (A floor alone leaves half a unit in every value,
// and rounding ties up 2^-s-1; the following passes add them up coherently: N = 4096, random
// field, right-hand side off by 1.7e-15 instead of 3.6e-16.)
CME_DEV long long fshift(long long v, int s)
{
    return (v + ((1LL << (s - 1)) - 1) + ((v >> s) & 1)) >> s;
}
// the same for s in 0 ... 63 (uniform over the group); EVEN = false rounds ties up, for shifts of
// many bits or values that only enter a right-hand side
template <bool EVEN = true>
CME_DEV long long frsh(long long v, int s)
{
    if (s == 0)
        return v;
    return EVEN ? fshift(v, s) : (v + (1LL << (s - 1))) >> s;
}
// a (w / 4): twiddled values lose two bits, which the growth of the next pass takes anyway
CME_DEV fx fcmul4(fx a, fl2 w)
{
    const fl r = fsplit(a.re), i = fsplit(a.im);
    const int nih = -i.h;
    const long long A = fmad(nih, w.im.l, fmad(r.l, w.re.h, fwide(r.h, w.re.l)));
    const long long M = fmad(i.l, w.re.h, fmad(r.l, w.im.h, fwide(r.h, w.im.l)));
    const int t = fhi(A) - fhi(fwide(i.l, w.im.h)), u = fhi(M) - fhi(fwide(nih, w.re.l));
    return {fmad(t, 1, fmad(nih, w.im.h, fwide(r.h, w.re.h))),
            fmad(u, 1, fmad(i.h, w.re.h, fwide(r.h, w.im.h)))};
}
// a w, unscaled (|a| < 2^62)
CME_DEV fx fcmul1(fx a, fl2 w)
{
    constexpr long long half = 1LL << 29;
    const fl r = fsplit(a.re), i = fsplit(a.im);
    const int nih = -i.h;
    const long long A = fmad(nih, w.im.l, fmad(r.l, w.re.h, fmad(r.h, w.re.l, half)));
    const long long M = fmad(
        i.l, w.re.h, fmad(i.h, w.re.l, fmad(r.l, w.im.h, fmad(r.h, w.im.l, half))));
    const long long hr = fmad(nih, w.im.h, fwide(r.h, w.re.h));
    const long long hi = fmad(i.h, w.re.h, fwide(r.h, w.im.h));
    return {fshl(hr, 2) + ((A - fwide(i.l, w.im.h)) >> 30), fshl(hi, 2) + (M >> 30)};
}
CME_DEV fx fadd(fx a, fx b) { return {a.re + b.re, a.im + b.im}; }
CME_DEV fx fsub(fx a, fx b) { return {a.re - b.re, a.im - b.im}; }

// z times sqrt(1/2), cos(pi/8), sin(pi/8): factors of 2^64 within +-1/2 (c - 1 for the cosines)
CME_DEV long long fmul_h(long long z) { return z + fmulhi(fsplit(z), {-1257966796, -102865788}); }
CME_DEV long long fmul_c(long long z) { return z + fmulhi(fsplit(z), {-326934918, -1804979899}); }
CME_DEV long long fmul_s(long long z) { return fmulhi(fsplit(z), {1643612827, -1163556025}); }

// z exp(2 pi i K / 16), K = 0 ... 7
template <int K>
CME_DEV fx frot16(fx z)
{
    if constexpr (K == 0)
        return z;
    else if constexpr (K == 4)
        return {-z.im, z.re};
    else if constexpr (K > 4)
        return frot16<4>(frot16<K - 4>(z));
    else if constexpr (K == 2)
        return {fmul_h(z.re - z.im), fmul_h(z.re + z.im)};
    else if constexpr (K == 1)
        return {fmul_c(z.re) - fmul_s(z.im), fmul_s(z.re) + fmul_c(z.im)};
    else
        return {fmul_s(z.re) - fmul_c(z.im), fmul_c(z.re) + fmul_s(z.im)};
}

// In-register inverse DFT of size r (natural order in and out), as dft<r, +1>.
template <int r, int span>
CME_DEV void fdft_stage(fx (&v)[r])
{
    if constexpr (span >= 1) {
#pragma unroll
        for (int blk = 0; blk < r; blk += 2 * span)
#pragma unroll
            for (int j = 0; j < span; ++j) {
                const fx a = v[blk + j], b = v[blk + j + span];
                v[blk + j] = fadd(a, b);
                v[blk + j + span] = fsub(a, b);
            }
#pragma unroll
        for (int blk = 0; blk < r; blk += 2 * span) {
            if constexpr (span >= 2)
                v[blk + span + 1] = frot16<8 / span>(v[blk + span + 1]);
            if constexpr (span >= 4) {
                v[blk + span + 2] = frot16<16 / span>(v[blk + span + 2]);
                v[blk + span + 3] = frot16<24 / span>(v[blk + span + 3]);
            }
            if constexpr (span >= 8) {
                v[blk + span + 4] = frot16<4>(v[blk + span + 4]);
                v[blk + span + 5] = frot16<5>(v[blk + span + 5]);
                v[blk + span + 6] = frot16<6>(v[blk + span + 6]);
                v[blk + span + 7] = frot16<7>(v[blk + span + 7]);
            }
        }
        fdft_stage<r, span / 2>(v);
    }
}
template <int r>
CME_DEV void fdft(fx (&v)[r])
{
    if constexpr (r > 1) {
        fdft_stage<r, r / 2>(v);
        fx t[r];
#pragma unroll
        for (int k = 0; k < r; ++k)
            t[k] = v[bitrev(k, ilog2(r))];
#pragma unroll
        for (int k = 0; k < r; ++k)
            v[k] = t[k];
    }
}

// Twiddle limbs of the FP64 table (aux_kernels.cu: exp(2 pi i k / N) 2^62 as balanced limbs).
CME_DEV fl2 fx_twiddle(const void* table, long long i)
{
    const int4 v = __ldg(reinterpret_cast<const int4*>(table) + i);
    return {{v.x, v.y}, {v.z, v.w}};
}
// the same as an FP64 value
CME_DEV cx<double> fx_twiddle_f64(const void* table, long long i)
{
    const fl2 w = fx_twiddle(table, i);
    constexpr double s = 1.0 / 4611686018427387904.0;   // 2^-62
    return {(double)(((long long)w.re.h << 32) + w.re.l) * s,
            (double)(((long long)w.im.h << 32) + w.im.l) * s};
}
template <typename T>
CME_DEV cx<T> twload(const void* table, long long i)
{
    if constexpr (sizeof(T) == 4)
        return gload<T>(table, i);
    else
        return fx_twiddle_f64(table, i);
}

// Pass twiddles of a thread, as Twiddles (registers, or read from the table where used).
template <int LOGN, int R, bool IN_REGS, int TS = 1>
struct FixTwiddles {
    using PL = Plan<LOGN, R>;
    fl2 w[IN_REGS && PL::NTW > 0 ? PL::NTW : 1];
    const void* table;
    int kst[PL::NS > 1 ? PL::NS : 1];   // (t mod L_s) N / (L_s r_s) per pass

    template <int s>
    CME_DEV void fill()
    {
        if constexpr (s < PL::NS) {
            constexpr int r = PL::radix(s), Q = R / r;
#pragma unroll
            for (int q = 0; q < Q; ++q)
#pragma unroll
                for (int j = 1; j < r; ++j)
                    w[(s - 1) * (R - 1) + q * (r - 1) + (j - 1)] = read<s>(q, j);
            fill<s + 1>();
        }
    }
    CME_DEV void init(const void* tbl, int t)
    {
        table = tbl;
#pragma unroll
        for (int s = 1; s < PL::NS; ++s) {
            const int L = PL::L(s), r = PL::radix(s);
            kst[s] = (t & (L - 1)) * (PL::N / (L * r));
        }
        if constexpr (IN_REGS)
            fill<1>();
    }
    template <int s>
    CME_DEV fl2 read(int q, int j) const
    {
        // butterfly q > 0 only occurs in the last pass, where k = t + qP exactly
        constexpr int r = PL::radix(s), L = PL::L(s), stride = PL::N / (L * r);
        return fx_twiddle(table,
                          ((j * kst[s] + j * q * PL::P * stride) & (PL::N - 1)) * TS);
    }
    template <int s>
    CME_DEV fl2 get(int q, int j) const
    {
        if constexpr (IN_REGS)
            return w[(s - 1) * (R - 1) + q * (PL::radix(s) - 1) + (j - 1)];
        else
            return read<s>(q, j);
    }
};

// (-1)^n / (2n + 1)! and (-1)^n / (2n + 2)!, times 2^62: sin(x)/x and (1 - cos(x))/x^2 in x^2.
// Templates, so that only the units whose kernels read them hold constant data: with it every launch
// of a unit's kernels takes about 0.15 us longer (four-step FP32, eight kernels a step: N = 2^13 18.4
// -> 17.2 us per step without, N = 2^14 19.5 -> 18.5).
template <int>
static __constant__ long long fx_sinc[10] = {
    4611686018427387904, -768614336404564651, 38430716820228233, -915017067148291, 12708570377060,
    -115532457973, 740592679, -3526632, 12966, -38};
template <int>
static __constant__ long long fx_cosc[10] = {
    2305843009213693952, -192153584101141163, 6405119470038039, -114377133393536, 1270857037706,
    -9627704831, 52899477, -220414, 720, -2};

// Bounds of a group's values in bits: every value's modulus is below 2^bm, L1 below 2^bl.
struct FixBound {
    int bm, bl;
};

// One pair of reductions over the P threads of a group: the largest key, then the sum of
// counts that each warp (each group, P <= 32) forms relative to its own largest key; P > 32
// combines the warps' pairs through shared memory (`red`, P / 32 pairs), where a warp whose
// key >> key_shift is d below the largest has its sum shifted right by count_shift d bits.
template <int P>
struct GroupReduce {
    static constexpr int W = P > 32 ? P / 32 : 1;
    CME_DEV static unsigned max_key(unsigned v)
    {
        if constexpr (P >= 32) {
            return __reduce_max_sync(0xffffffffu, v);
        } else {
#pragma unroll
            for (int o = P / 2; o > 0; o >>= 1)
                v = max(v, __shfl_xor_sync(0xffffffffu, v, o));
            return v;
        }
    }
    CME_DEV static unsigned sum(unsigned v)
    {
        if constexpr (P >= 32) {
            return __reduce_add_sync(0xffffffffu, v);
        } else {
#pragma unroll
            for (int o = P / 2; o > 0; o >>= 1)
                v += __shfl_xor_sync(0xffffffffu, v, o);
            return v;
        }
    }
    template <int count_shift, int key_shift = 0>
    CME_DEV static void combine(int& key, unsigned& count, int2* red, int t)
    {
        if constexpr (W > 1) {
            if ((t & 31) == 0)
                red[t >> 5] = make_int2(key, (int)count);
            __syncthreads();
            int2 v[W];
#pragma unroll
            for (int i = 0; i < W; ++i) {
                v[i] = red[i];
                key = max(key, v[i].x);
            }
            count = 0;
#pragma unroll
            for (int i = 0; i < W; ++i)
                count += ((unsigned)v[i].y >>
                          min(count_shift * ((key >> key_shift) - (v[i].x >> key_shift)), 31)) +
                         1u;
        }
    }
};

// Fixed-point transform of one group; the passes, exchanges and twiddles are those of
// Transform, inverse direction only (the forward transform is conj(inverse(conj(.)))).
template <int LOGN, int R, bool WARP, bool CLUSTER = false>
struct FixTransform {
    using PL = Plan<LOGN, R>;
    using TF = Transform<double, LOGN, R, WARP>;   // exchange layout
    static constexpr int N = PL::N, P = PL::P, NS = PL::NS;
    // A twiddled pass scales by 1/4; where many narrow passes follow one another (R <= 4) its
    // inputs are doubled first, so that 7 passes cost 7 bits and not 14.
    static constexpr int HB = R <= 4 ? 1 : 2;
    // Bits of every value's modulus: sqrt(2) 2^62 is the largest sum inside a rotation, and the
    // middle products of fcmul4 stay below 2^63.  With a single pass, which scales nothing, and with
    // narrow ones 61, the limit of samples that the Kerr term takes (SAMPLE).
    static constexpr int SAMPLE = 61;
    static constexpr int LIM = HB == 1 || NS == 1 ? 61 : 62;
    // modulus of a product of the Kerr term: room for the first pass's growth (59: its limbs')
    static constexpr int KB = LIM - ilog2(PL::radix(0)) < 59 ? LIM - ilog2(PL::radix(0)) : 59;
    using GRd = GroupReduce<P>;

    static constexpr int OUT = HB * (NS - 1);   // the result of a run is X 2^(OUT - lift)

    // Bits that an input of bounds b reaches, over the passes: at most LIM before a run.  KERR: the
    // result goes to the Kerr term, so that it counts LIM - SAMPLE bits more than the passes.  (Where
    // the last pass is the largest, on short pulses with their flat spectra, it left samples of up
    // to 2^62, and the Kerr term overflowed: error of order 1.  Other fields keep their scale.)
    // FROM: the first pass that counts.
    template <bool KERR, int FROM = 0>
    CME_DEV static int headroom(FixBound b)
    {
        int g = b.bm + ilog2(PL::radix(0)), h = FROM == 0 ? min(b.bl, g) : -(1 << 20);
#pragma unroll
        for (int s = 1; s < NS; ++s) {
            g += ilog2(PL::radix(s));
            if (s >= FROM)
                h = max(h, min(b.bl, g) - s * HB);
        }
        if constexpr (KERR && LIM > SAMPLE)
            h = max(h, min(b.bl, g) - OUT + (LIM - SAMPLE));
        return h;
    }
    // Where the bounds grow less than the passes scale down, the samples lie bits below the limit, and
    // the rounding of the last passes lies above FP64's.  Transforms of many passes, and those of a
    // cluster's blocks, therefore shift their values left before the passes s of lifts(s), by what
    // the passes from s - 1 on leave free (`up`; lift returns their sum).  Error of the modes below
    // 1e-4 after an RK4IP step of a comb (tests/test_fixed_bounds.py), relative to that of FP64
    // instructions, without and with it: N = 128 at 2 values per thread 1.4 and 0.4, N = 1024 1.7 and
    // 0.9, N = 2048 1.3 and 1.0, N = 4096 2.2 and 1.55, clusters of 2 ... 8 blocks 1.0 to 2.7 and 0.85 to
    // 1.0 at N = 2048, 2.0 to 3.7 and 1.35 to 1.45 at N = 4096; all modes together 1.00.  What is left
    // at N = 4096 is the unit of the Kerr term, set by the envelope's peak, on the samples beside it.
    // us per RK4IP step without and with: N = 128 x 300 8.5 / 8.7, N = 1024 x 300 36.2 / 36.9,
    // N = 2048 x 150 45.9 / 46.2, N = 4096 x 150 107.7 / 105.0, x 64 (clusters) 72.5 / 72.8; split step
    // N = 1024 x 76 10.05 / 9.6, N = 2048 x 150 16.7 / 17.1, N = 4096 x 150 35.4 / 36.1.
    CME_HD static constexpr bool lifts(int s)
    {
        return R == 2 ? LOGN == 7 && (s == 3 || s == 5) : (LOGN >= 10 || CLUSTER) && s >= 2;
    }
    template <bool KERR, int s = 1>
    CME_DEV static int lift(FixBound b, int (&up)[NS], int sum = 0)
    {
        if constexpr (s < NS) {
            up[s] = 0;
            if constexpr (lifts(s)) {
                up[s] = min(max(LIM - headroom<KERR, s - 1>(b) - sum, 0), 15);
                sum += up[s];
            }
            return lift<KERR, s + 1>(b, up, sum);
        } else {
            return sum;
        }
    }
    // bits of the modulus of a run's result, before its shift
    CME_DEV static int out_bits(FixBound b) { return min(b.bl, b.bm + LOGN) - OUT; }

    // up: left shift before this pass (lifts): the bits that it cleared are not lost by the floors.
    template <int s, class TW>
    CME_DEV static void pass(fx (&x)[R], const TW& tw, int up)
    {
        constexpr int r = PL::radix(s), Q = R / r;
        // Butterflies whose twiddles are all 1 (k = 0; they lead to output 0) floor their products
        // exactly, without the second floor that cancels the bias elsewhere: each value ends
        // 3/8 (HB = 1: 1/4) of a unit low.  Their first value is floored too, so that only
        // output 0 is off, by r times that (`low`), and it is corrected (not where it is 0: zeros
        // stay zeros).  Without it: output 0 of N = 4096 off by 4 to 12 times the other outputs'
        // error.
        constexpr bool fix0 = s > 0 && (HB == 2 || r > 2);
        const int low = up == 0 ? (HB == 2 ? (3 * r + 4) / 8 : r / 4) : up < HB ? r / 4 : 0;
        bool k0 = false;
        if constexpr (fix0)
            k0 = tw.kst[s] == 0;
#pragma unroll
        for (int q = 0; q < Q; ++q) {
            fx v[r];
#pragma unroll
            for (int j = 0; j < r; ++j)
                v[j] = x[q + j * Q];
            if constexpr (s > 0) {
                constexpr int half = (1 << (HB - 1)) - 1;   // ties to even
                const bool z = fix0 && k0 && q == 0;
                const int ar = z ? 0 : half + ((int)(v[0].re >> HB) & 1);
                const int ai = z ? 0 : half + ((int)(v[0].im >> HB) & 1);
                v[0] = {(v[0].re + ar) >> HB, (v[0].im + ai) >> HB};
#pragma unroll
                for (int j = 1; j < r; ++j) {
                    if constexpr (HB == 1)
                        v[j] = fadd(v[j], v[j]);
                    v[j] = fcmul4(v[j], tw.template get<s>(q, j));
                }
            }
            fdft<r>(v);
            if (fix0 && q == 0)
                v[0] = {v[0].re + (k0 && v[0].re != 0 ? low : 0),
                        v[0].im + (k0 && v[0].im != 0 ? low : 0)};
#pragma unroll
            for (int j = 0; j < r; ++j)
                x[q + j * Q] = v[j];
        }
    }
    template <int s, class TW>
    CME_DEV static void run_from(fx (&x)[R], const TW& tw, const Xbuf<double>& buf, int& par,
                                 const typename TF::Addr& ad, const int (&up)[NS])
    {
        if constexpr (lifts(s)) {
#pragma unroll
            for (int j = 0; j < R; ++j)
                x[j] = {fshl(x[j].re, up[s]), fshl(x[j].im, up[s])};
            pass<s>(x, tw, up[s]);
        } else {
            pass<s>(x, tw, 0);
        }
        if constexpr (s + 1 < NS) {
            cx<double> y[R];
#pragma unroll
            for (int j = 0; j < R; ++j)
                y[j] = {__longlong_as_double(x[j].re), __longlong_as_double(x[j].im)};
            TF::template exchange<s>(y, buf, ad, par);
#pragma unroll
            for (int j = 0; j < R; ++j)
                x[j] = {__double_as_longlong(y[j].re), __double_as_longlong(y[j].im)};
            par ^= 1;
            run_from<s + 1>(x, tw, buf, par, ad, up);
        }
    }
    template <class TW>
    CME_DEV static void run(fx (&x)[R], const TW& tw, const Xbuf<double>& buf, int& par,
                            const typename TF::Addr& ad, const int (&up)[NS])
    {
        run_from<0>(x, tw, buf, par, ad, up);
    }

    // Scale of a group's FP64 values: X = x 2^q, bounds of X.  q = POISON: a value is not finite.
    static constexpr int POISON = 1 << 20;
    struct Scale {
        int q;
        FixBound b;
    };
    CME_DEV static unsigned habs(double v) { return (unsigned)__double2hiint(v) & 0x7fffffffu; }

    // FP64 -> fixed point.  `red`: the group's reduction pairs (P > 32).  KERR: see headroom.
    template <bool KERR>
    CME_DEV static Scale load(const cx<double> (&xin)[R], fx (&X)[R], int2* red, int t)
    {
        cx<double> x[R];
        unsigned mh = 0;
#pragma unroll
        for (int j = 0; j < R; ++j) {
            x[j] = xin[j];
            mh = max(mh, max(habs(x[j].re), habs(x[j].im)));
        }
        int E = (int)(GRd::max_key(mh) >> 20);   // biased exponent (the warp's)
        // sum of |re| + |im| in units of 2^(E - 1023), from the leading 20 bits of each
        const int base = (E - 127) * (1 << 20);
        float f = 0.f;
#pragma unroll
        for (int j = 0; j < R; ++j) {
            f += __int_as_float(max((int)habs(x[j].re) - base, 0) << 3);
            f += __int_as_float(max((int)habs(x[j].im) - base, 0) << 3);
        }
        unsigned cnt = GRd::sum((unsigned)(f * 4096.f) + 1u);
        GRd::template combine<1>(E, cnt, red, t);
        int pre = 0;
        if (E < 100) {   // near the denormal range (or all zero): scale up first
            pre = 900;
            E += 900;
#pragma unroll
            for (int j = 0; j < R; ++j)
                x[j] = cscale(x[j], 8.452712498170644e270);   // 2^900
        }
        const bool bad = E == 2047;
        const int bl = 32 - __clz((int)cnt) - 12, bm = 2;
        const int B0 = headroom<KERR>({bm, bl});
        const int c0 = 62 - LIM + B0 + E;
#pragma unroll
        for (int j = 0; j < R; ++j)
            X[j] = {fix(x[j].re, c0), fix(x[j].im, c0)};
        return {bad ? POISON : LIM - B0 - E + 1023 + pre, {bm + LIM - B0, bl + LIM - B0}};
    }
    // v 2^(1085 - c0), rounded; |result| < 2^62.  SUB: c0 may be below 64, where zero and subnormal
    // numbers have to be told from normal ones of the smallest exponent; above, both round to 0.
    template <bool SUB = false>
    CME_DEV static long long fix(double v, int c0)
    {
        const unsigned hi = (unsigned)__double2hiint(v), lo = (unsigned)__double2loint(v);
        int e = (int)((hi >> 20) & 0x7ffu);
        unsigned mh = (hi & 0xfffffu) | 0x100000u;
        if (SUB && e == 0) {
            e = 1;
            mh &= 0xfffffu;
        }
        const int sh = min(c0 - 1 - e, 63);   // one more bit, rounded off
        const unsigned long long m =
            ((unsigned long long)__funnelshift_l(lo, mh, 10) << 32) | (lo << 10);
        const long long a = (long long)(((m >> sh) + 1) >> 1);
        return (int)hi < 0 ? -a : a;
    }

    // fixed point -> FP64: x = X 2^k (k <= -POISON / 2: NaN)
    // In integer arithmetic (about 22 instructions): the conversion instruction takes an FP64
    // slot of 64 cycles.
    CME_DEV static double unfix(long long v, int k)
    {
        const unsigned sg = (unsigned)fhi(v) & 0x80000000u;
        const unsigned long long a = (unsigned long long)(v < 0 ? -v : v);
        unsigned h = (unsigned)(a >> 32), l = (unsigned)a;
        int e = k + 1023 + 63 - 1;   // the leading bit of the mantissa adds the last one
        if (h == 0) {
            h = l;
            l = 0;
            e -= 32;
        }
        const int z = __clz((int)h);
        const unsigned mh = __funnelshift_l(l, h, z), ml = __funnelshift_l(0u, l, z);
        const unsigned long long d =
            ((((unsigned long long)((mh >> 11) + ((unsigned)(e - z) << 20))) << 32) |
             __funnelshift_r(ml, mh, 11)) +
            ((ml >> 10) & 1u);
        return __hiloint2double(h ? (int)((unsigned)(d >> 32) | sg) : 0, (int)(unsigned)d);
    }
    CME_DEV static void store(const fx (&X)[R], int k, cx<double> (&x)[R])
    {
        if (k > -900 && k < 900) {   // every result is a normal number
#pragma unroll
            for (int j = 0; j < R; ++j)
                x[j] = {unfix(X[j].re, k), unfix(X[j].im, k)};
        } else {   // near the ends of the FP64 range, or not finite
            const int k1 = min(max(k / 2, -1022), 1023), k2 = min(max(k - k / 2, -1022), 1023);
            const double s1 = k <= -POISON / 2 ? __longlong_as_double(0x7ff8000000000000LL)
                                               : __hiloint2double((k1 + 1023) << 20, 0);
            const double s2 = __hiloint2double((k2 + 1023) << 20, 0);
#pragma unroll
            for (int j = 0; j < R; ++j)
                x[j] = {(double)X[j].re * s1 * s2, (double)X[j].im * s1 * s2};
        }
    }

    // Scales of the Kerr term of the time samples a = X 2^-q, |X| <= 2^SAMPLE, with the coefficient g.
    // The samples are first scaled by their own largest modulus (they lie up to sqrt(N) below the
    // bound of the transform), and L1 of the product comes from the same reduction.
    struct Kerr {
        int up, ps, us;   // left shifts of the samples, of |a|^2 and of g |a|^2
        fl G;         // limbs of -g 2^(62 - eg), |g| = m 2^eg with m in [1/2, 1)
        int qc;       // -g |a|^2 is (|a|^2 G) 2^-qc before its shift
        int q;        // scale and bounds of conj(i g |a|^2 a)
        FixBound b;
        bool over;    // the largest |a|^2, at least 2^(key - 3) units of 2^80, leaves the FP64 range
    };
    CME_DEV static Kerr kerr_scale(const fx (&X)[R], int q, double g, int2* red, int t)
    {
        float mx = 0.f, f = 0.f;
#pragma unroll
        for (int j = 0; j < R; ++j) {
            const float r = hi_float(X[j].re), i = hi_float(X[j].im);
            const float p = r * r + i * i;
            mx = fmaxf(mx, p);
            f += p * (fabsf(r) + fabsf(i));
        }
        // |a|^2 below 2^(key - 1), the modulus below 2^(key / 2), units of 2^40.  A component lies up
        // to one unit above its floor: |a|^2 < p + 2 sqrt(2 p) + 2 <= 1.02 p + 102.  The samples'
        // limit of 2^21 units gives key = 43, also where 1.02 p exceeds its square.
        int key = min((int)(GRd::max_key(__float_as_uint(fmaf(mx, 1.02f, 102.f))) >> 23) - 127 + 2,
                      2 * (SAMPLE - 40) + 1);
        unsigned cnt = GRd::sum(
            (unsigned)(f * __int_as_float((127 + 12 - 3 * (key >> 1)) << 23)) + 1u);
        GRd::template combine<3, 1>(key, cnt, red, t);
        Kerr k;
        k.up = SAMPLE - 40 - (key >> 1);   // modulus below 2^61
        // |a|^2 2^-64 <= 2^58, shifted left by 4 bits, times |g| 2^(62 - eg) < 2^62 and a <= 2^61:
        // products below 2^57, and below 2^KB with g |a|^2 <= 2^60 shifted left by KB - 57 <= 2;
        // less where the next transform has no room for that; an even key leaves |a|^2 one bit
        // below its bound, so that the shift is one more
        const FixBound full = {KB, KB + 32 - __clz((int)cnt) - 12};
        const int less = max(headroom<false>(full) - LIM, 0);
        const int sh = KB - 57 - less, odd = (key & 1) ^ 1;
        k.ps = 4 + min(sh, 0);
        k.us = max(sh, 0) + odd;
        const int gh = __double2hiint(g);
        const int ge = (gh >> 20) & 0x7ff, eg = ge ? ge - 1022 : 0;
        const long long gm =
            ge ? (long long)((((unsigned long long)((gh & 0xfffff) | 0x100000) << 32) |
                              (unsigned)__double2loint(g))
                             << 9)
               : 0;
        k.G = fsplit(gh < 0 ? gm : -gm);
        const int qa = q + k.up;
        k.qc = 2 * qa - 66 + k.ps - eg;
        k.q = qa + k.qc + k.us - 64;
        k.b = {full.bm - less, full.bl - less};
        k.over = 2 * (SAMPLE - qa) - 3 >= 1024;
        return k;
    }
    // X becomes conj(i g |a|^2 a) 2^k.q; returns -g |a|^2 2^k.qc
    CME_DEV static long long kerr_term(fx& X, const Kerr& k)
    {
        const fl r = fsplit(fshl(X.re, k.up)), i = fsplit(fshl(X.im, k.up));
        const long long m = fmad(i.h, i.l, fmad(r.h, r.l, 0x40000000LL));
        const long long p2 = fshl(fmad(i.h, i.h, fmad(r.h, r.h, m >> 31)), k.ps);
        const long long pg = fmulhi(fsplit(p2), k.G);
        const fl c = fsplit(fshl(pg, k.us));
        X = {fmulhi(c, i), fmulhi(c, r)};
        return pg;
    }
    CME_DEV static Kerr kerr(fx (&X)[R], int q, double g, int2* red, int t)
    {
        const Kerr k = kerr_scale(X, q, g, red, t);
#pragma unroll
        for (int j = 0; j < R; ++j)
            kerr_term(X[j], k);
        return k;
    }
    // The exact Kerr flow's increment: X becomes conj(a expm1(i phi)) / N, phi = gh |a|^2, for
    // the next transform (scale k.q, bounds k.b).  For phi < 1 everywhere in the group
    // expm1(i phi) = i phi F with the Taylor series F = sin(phi)/phi + i (1 - cos(phi))/phi in
    // phi^2, cut where the group's largest phi leaves less than 2^-62 (5 terms at 0.06); larger
    // phases take sincos in FP64 (no reduction in that branch: groups of a block may differ).
    // 4 x N = 256 at 4 values per thread: 9.1 -> 4.8 us per split step, most of it the FP64
    // instructions of sincos (about 3500 cycles per value, against about 350).
    // LG: log2 of the instance's N (this transform's, or that of its cluster).  bad: this thread holds
    // a sample whose phase is not finite.
    template <int LG>
    CME_DEV static Kerr kerr_flow(fx (&X)[R], int q, double gh, bool& bad, int2* red, int t)
    {
        constexpr double invN = 1.0 / (1 << LG);
        Kerr k = kerr_scale(X, q, gh * invN, red, t);
        const int sh = k.qc - 62 - LG;   // |pg| < 2^60: phi 2^62 = |pg| 2^-sh < 2^(60 - sh)
        if (sh >= -2) {
            const int terms = sh < 0 ? (sh == -1 ? 8 : 10) : sh < 2 ? 7 : sh < 4 ? 5 : sh < 8 ? 4
                              : sh < 15 ? 3 : 2;
            const int rs = min(max(sh, 0), 63), ls = max(-sh, 0);
            fx S[R];
            long long ph[R];
            fl z[R];
#pragma unroll
            for (int j = 0; j < R; ++j) {
                ph[j] = fshl(-kerr_term(X[j], k), ls) >> rs;
                const fl p = fsplit(ph[j]);
                z[j] = fsplit(fshl(fmulhi(p, p), 2));
                S[j] = {0, 0};
            }
#pragma unroll 1
            for (int n = terms - 1; n >= 0; --n) {
                const long long cs = fx_sinc<0>[n], cc = fx_cosc<0>[n];
#pragma unroll
                for (int j = 0; j < R; ++j)
                    S[j] = {cs + fshl(fmulhi(fsplit(S[j].re), z[j]), 2),
                            cc + fshl(fmulhi(fsplit(S[j].im), z[j]), 2)};
            }
#pragma unroll
            for (int j = 0; j < R; ++j) {
                const long long im = fshl(fmulhi(fsplit(S[j].im), fsplit(ph[j])), 2);
                X[j] = fcmul1(X[j], {fsplit(S[j].re), fsplit(-im)});
            }
        } else {
            cx<double> a[R];
            store(X, -q, a);
#pragma unroll
            for (int j = 0; j < R; ++j) {
                const double y = 0.5 * gh * (a[j].re * a[j].re + a[j].im * a[j].im);
                double sn = 0.0, cs = 0.0;
                if (isfinite(y))
                    sincos(y, &sn, &cs);
                else
                    bad = true;
                // a times conj(expm1(i phi)) / 2, whose modulus is at most 1
                const fl2 w = {fsplit(fix(-sn * sn, 1085 - 62)), fsplit(fix(-sn * cs, 1085 - 62))};
                X[j] = fcmul1({fshl(X[j].re, k.up), -fshl(X[j].im, k.up)}, w);
            }
            // |a expm1(i phi)| / 2 <= |a| min(1, phi / 2): L1 is at most N |a|max, and at most
            // 2^(f - 1) |a|max sum (|a| / |a|max)^3 with phi < 2^f, the sum from the scale's bounds
            const int f = -2 - sh;
            k.q = q + k.up - 1 + LG;
            k.b = {SAMPLE, SAMPLE + min(LOGN, f - 1 + k.b.bl - k.b.bm)};
            const int less = max(headroom<false>(k.b) - LIM, 0);
#pragma unroll
            for (int j = 0; j < R; ++j)
                X[j] = {frsh(X[j].re, less), frsh(X[j].im, less)};
            k.q -= less;
            k.b = {k.b.bm - less, k.b.bl - less};
        }
        return k;
    }
    // Bounds of values that are below 2^62.5: the largest component and L1, from their high words.
    CME_DEV static FixBound bounds(const fx (&X)[R], int2* red, int t)
    {
        float mx = 0.f, f = 0.f;
#pragma unroll
        for (int j = 0; j < R; ++j) {
            const float r = fabsf(hi_float<9>(X[j].re)), i = fabsf(hi_float<9>(X[j].im));
            mx = fmaxf(mx, fmaxf(r, i));
            f += r + i;
        }
        // components below 2^(key + 1) units of 2^41 (each high word is up to 1 below its value)
        int key = (int)(GRd::max_key(__float_as_uint(mx + 1.f)) >> 23) - 127;
        unsigned cnt = GRd::sum(
            (unsigned)((f + 2 * R) * __int_as_float((127 + 11 - key) << 23)) + 1u);
        GRd::template combine<1>(key, cnt, red, t);
        return {41 + key + 2, 41 + key + 1 + 32 - __clz((int)cnt) - 12};
    }
    // Scale values with bounds b for a transform: right where a pass could overflow,
    // left where more than three bits would be lost.  Returns the shift (left positive).
    template <bool KERR>
    CME_DEV static int rescale(fx (&X)[R], FixBound& b)
    {
        const int s = LIM - headroom<KERR>(b);
        if (s >= 0 && s <= 3)
            return 0;
        if (s < 0) {
#pragma unroll
            for (int j = 0; j < R; ++j)
                X[j] = {frsh<false>(X[j].re, -s), frsh<false>(X[j].im, -s)};
        } else {
#pragma unroll
            for (int j = 0; j < R; ++j)
                X[j] = {fshl(X[j].re, s), fshl(X[j].im, s)};
        }
        b.bm += s;
        b.bl += s;
        return s;
    }
    // Common scale of the sum of values v 2^-q, modulus below 2^b, of two sums: the coarser of the
    // two, and coarse enough that the result's modulus stays below 2^62 (2^62.1 where one is a
    // sixteenth of the other or less, so that a value at the limit keeps its last bit).
    struct Align {
        int q, sv, sw;   // scale of the sum, right shifts of the two
        int b;           // bits of the sum
    };
    CME_DEV static Align align(int qv, int bv, int qw, int bw)
    {
        int q = min(qv, qw);
        const int cv = bv - (qv - q), cw = bw - (qw - q);
        const int top = max(cv, cw), sum = top - min(cv, cw) >= 4 ? top : top + 1;
        const int e = max(sum - 62, 0);
        q -= e;
        return {q, min(qv - q, 63), min(qw - q, 63), sum - e};
    }
    template <bool EVEN>
    CME_DEV static fx asum(fx v, fx w, const Align& a)
    {
        return {frsh<EVEN>(v.re, a.sv) + frsh<EVEN>(w.re, a.sw),
                frsh<EVEN>(v.im, a.sv) + frsh<EVEN>(w.im, a.sw)};
    }
    // v in units of 2^(32 + S), floored; below 2^22 of them
    template <int S = 8>
    CME_DEV static float hi_float(long long v)
    {
        return __int_as_float(0x4b400000 + ((int)(v >> 32) >> S)) - 12582912.f;
    }
};

}  // namespace CME_FP32_VARIANT
}  // namespace cme
