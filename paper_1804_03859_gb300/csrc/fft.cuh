// Register-resident Stockham FFT for the row and column passes of the stepper.
//
// A complex sequence of length N = 2^logN is spread over N/E threads, E = 2,
// 4 or 8 elements each (template parameter LE = log2 E): thread t of a
// sequence holds the elements t + r N/E, r < E.  Input and output have the
// same distribution and natural order, so a transform starts on values as
// they come from memory (consecutive threads, consecutive elements), a
// column pass goes from its forward transform through the diagonal operator
// into the inverse one without leaving the registers, and results are stored
// straight from the registers.  Shared memory only carries the exchange
// between two radix-E passes (one smaller radix closes a length that is no
// power of E, with several butterflies per thread on the same distribution).
// M sequences with the same index map are transformed side by side by the
// same threads: one twiddle load and one pair of barriers serve all of them.
//
// Why: the passes are bound by shared-memory and barrier latency, integer
// addressing (44% of the issued instructions in an in-place shared-memory
// form of the same radix-8 passes) and, in FP64, by the FP64 pipe.  Keeping
// the data in registers takes out the staging copies on both sides and two
// of every three shared-memory round trips of a column pass.
//
// Fewer elements per thread means more warps for the same transform, which is
// what small grids need to occupy all four SM sub-partitions (on GB300 a
// warp-wide FP64 instruction holds a sub-partition's FP64 unit for 64
// cycles, so each sub-partition needs its own warp).
//
// Shared-memory layout: element e of a sequence sits at slot sw<T>(e) = e +
// e / 2^PL with one pad slot per 128-byte bank row (2^PL = 16 float2 or 8
// 16-byte elements): the stores of the first passes (stride 2, 4 or 8 between
// neighbouring threads) and all unit-stride accesses are free of bank
// conflicts (FP64 with E = 4 has a two-way conflict in its second exchange),
// and the slots of one thread are linear in r.
//
// Twiddles come from precomputed per-pass tables (built on the host in
// extended precision) read through the read-only cache; consecutive threads
// read consecutive entries.
//
// FP64: the pipe issues 2 lane operations per clock and SM, so the number of
// FP64 instructions is the cost.  The butterflies are those of the fused
// multiply-add FFT of Linzer and Feig (IEEE Trans. Signal Processing 41, 1993):
// a twiddle w = c - i s is stored as its larger component m and the ratio tau
// of the other to it (|tau| <= 1):
// w b = m (p + tau q, q - tau p) with (p, q) = (b.x, b.y), or (b.y, -b.x)
// where |s| > |c|.  A radix-2 butterfly a +- w b is then two FMAs for the
// bracket and four for the sums, 6 instructions instead of 8, and a radix-8
// pass is three layers of such butterflies with four twiddles (w^4, w^2, w,
// w e^{-i pi/4}): 72 instructions instead of 84 (radix 4: 24 instead of 28).
// Every value passes through no more roundings than in the plain form.
//
// FP32 transforms carry every twiddle as hi + lo (lo = the FP32 rounding
// error of hi) and fold the lo product into the fused multiply-adds before
// their final rounding; the radix-8 constant 1/sqrt(2) is split the same
// way.  A twiddle rounded to FP32 makes the transform a fixed, slightly
// wrong linear map, and a time-stepper applies that same map at every step,
// so its error adds up linearly over a run (about 1e-5 relative after a few
// hundred steps, which then bounds the accuracy of the eigenvalues); with
// the split only the data-dependent rounding of the arithmetic remains.
#pragma once

#include <type_traits>

#include "common.cuh"

namespace nsstab {

// log2 of the elements per 128-byte bank row
template <class T> constexpr int kPadLog = sizeof(Cx<T>) == 8 ? 4 : 3;
template <class T> __host__ __device__ constexpr int sw(int i) { return i + (i >> kPadLog<T>); }
// slots a sequence of n elements occupies
template <class T> __host__ __device__ constexpr int padded_len(int n) { return sw<T>(n); }

// Cx<T> slots per twiddle entry: FP32 tables store hi and lo side by side.
template <class T> constexpr int kTwWidth = std::is_same<T, float>::value ? 2 : 1;
// Twiddle rows (of Ns entries each) of a pass of radix 2^LR: FP64 w^4, w^2,
// w, w e^{-i pi/4} (radix 8), w^2, w (radix 4), w (radix 2); otherwise w^r, r
// = 1 .. R-1, with w = exp(-2 pi i k / (Ns R)) for entry k.  A table is the
// rows of the passes after the first, in order: fewer than 2 N entries.
template <class T> __host__ __device__ constexpr int tw_rows(int LR) {
    return std::is_same<T, double>::value ? (LR == 3 ? 4 : LR) : (1 << LR) - 1;
}
// exponent e of row q's entry k: the twiddle is exp(-2 pi i e / (Ns R))
template <class T> inline long tw_exponent(int LR, int q, long k, long Ns) {
    if (!std::is_same<T, double>::value) return (q + 1) * k;
    if (LR == 3) return q == 0 ? 4 * k : q == 1 ? 2 * k : q == 2 ? k : k + Ns;
    if (LR == 2) return q == 0 ? 2 * k : k;
    return k;
}
// FP64: whether the twiddle of exponent e (of len per turn) is stored by its
// sine, i.e. its angle lies in the quarter turns around +-90 degrees
__host__ __device__ constexpr bool tw_by_sine(long e, long len) { return ((8 * e / len + 1) >> 1) & 1; }

template <class T> struct Consts;
template <> struct Consts<double> { static constexpr double rsqrt2 = 0.70710678118654752440084436210485; };
template <> struct Consts<float> {
    static constexpr float rsqrt2 = 0.70710678118654752440f;
    static constexpr float rsqrt2_lo = 1.21016175e-08f;   // 1/sqrt(2) - rsqrt2
};
template <> struct Consts<df64> { static constexpr df64 rsqrt2 = df64(0.70710677f, 1.21016175e-08f); };

// s / sqrt(2), with the FP32 constant's rounding error compensated
template <class T> __device__ __forceinline__ T mul_rsqrt2(T s) {
    if constexpr (std::is_same<T, float>::value) {
        return __fmaf_rn(s, Consts<float>::rsqrt2, s * Consts<float>::rsqrt2_lo);
    } else {
        return s * Consts<T>::rsqrt2;
    }
}

// forward: X_k = sum_j x_j exp(-2 pi i jk/N); INV: exp(+2 pi i jk/N), unnormalised
template <bool INV, class C> __device__ __forceinline__ void dft4(C& a0, C& a1, C& a2, C& a3) {
    const C s02 = cadd(a0, a2), d02 = csub(a0, a2);
    const C s13 = cadd(a1, a3), d13 = csub(a1, a3);
    const C t = INV ? cmul_pi(d13) : cmul_mi(d13);
    a0 = cadd(s02, s13);
    a2 = csub(s02, s13);
    a1 = cadd(d02, t);
    a3 = csub(d02, t);
}

template <bool INV, class T> __device__ __forceinline__ void dft8(Cx<T>* v) {
    // decimation in frequency: X_{2k} = DFT4(a)_k, X_{2k+1} = DFT4(b)_k with
    // a_r = v_r + v_{r+4}, b_r = (v_r - v_{r+4}) W8^r, W8 = exp(-+ 2 pi i / 8)
    Cx<T> a0 = cadd(v[0], v[4]), b0 = csub(v[0], v[4]);
    Cx<T> a1 = cadd(v[1], v[5]), b1 = csub(v[1], v[5]);
    Cx<T> a2 = cadd(v[2], v[6]), b2 = csub(v[2], v[6]);
    Cx<T> a3 = cadd(v[3], v[7]), b3 = csub(v[3], v[7]);
    if (!INV) {
        b1 = mk<T>(mul_rsqrt2<T>(b1.x + b1.y), mul_rsqrt2<T>(b1.y - b1.x));     // (1 - i)/sqrt2
        b2 = cmul_mi(b2);                                                      // -i
        b3 = mk<T>(mul_rsqrt2<T>(b3.y - b3.x), -mul_rsqrt2<T>(b3.x + b3.y));    // (-1 - i)/sqrt2
    } else {
        b1 = mk<T>(mul_rsqrt2<T>(b1.x - b1.y), mul_rsqrt2<T>(b1.x + b1.y));     // (1 + i)/sqrt2
        b2 = cmul_pi(b2);                                                      // +i
        b3 = mk<T>(-mul_rsqrt2<T>(b3.x + b3.y), mul_rsqrt2<T>(b3.x - b3.y));    // (-1 + i)/sqrt2
    }
    dft4<INV>(a0, a1, a2, a3);
    dft4<INV>(b0, b1, b2, b3);
    v[0] = a0; v[1] = b0; v[2] = a1; v[3] = b1;
    v[4] = a2; v[5] = b2; v[6] = a3; v[7] = b3;
}

// a * w_e (INV: a * conj(w_e)) for a loaded twiddle entry (FP32: hi, lo)
template <class T> struct TwEntry {
    using type = Cx<T>;
    __device__ static __forceinline__ type load(const Cx<T>* __restrict__ tw, int e) { return ldg_c(tw + e); }
};
template <> struct TwEntry<float> {
    using type = float4;
    __device__ static __forceinline__ type load(const float2* __restrict__ tw, int e) {
        return __ldg(reinterpret_cast<const float4*>(tw) + e);
    }
};
template <bool INV, class T> __device__ __forceinline__ Cx<T> twiddle(Cx<T> a, typename TwEntry<T>::type q) {
    if constexpr (std::is_same<T, float>::value) {   // hi (x, y), lo (z, w)
        float re, im;
        if (!INV) {
            const float lr = a.x * q.z - a.y * q.w, li = a.x * q.w + a.y * q.z;
            re = __fmaf_rn(a.x, q.x, __fmaf_rn(-a.y, q.y, lr));
            im = __fmaf_rn(a.x, q.y, __fmaf_rn(a.y, q.x, li));
        } else {
            const float lr = a.x * q.z + a.y * q.w, li = a.y * q.z - a.x * q.w;
            re = __fmaf_rn(a.x, q.x, __fmaf_rn(a.y, q.y, lr));
            im = __fmaf_rn(a.y, q.x, __fmaf_rn(-a.x, q.y, li));
        }
        return mk<float>(re, im);
    } else if constexpr (std::is_same<T, df64>::value) {
        return INV ? mk<df64>(df_dot2(a.x, q.x, a.y, q.y), df_dot2(a.y, q.x, -a.x, q.y))
                   : mk<df64>(df_dot2(a.x, q.x, -a.y, q.y), df_dot2(a.x, q.y, a.y, q.x));
    } else {
        return INV ? cmulc(a, q) : cmul(a, q);
    }
}

// FP64 butterfly a, b <- a + w b, a - w b (INV: conj(w)) with w = (m, tau),
// by_sine as tw_by_sine
template <bool INV>
__device__ __forceinline__ void bfly(double2& a, double2& b, double2 w, bool by_sine) {
    const double p = by_sine ? (INV ? -b.y : b.y) : b.x;
    const double q = by_sine ? (INV ? b.x : -b.x) : b.y;
    const double re = INV ? fma(-w.y, q, p) : fma(w.y, q, p);
    const double im = INV ? fma(w.y, p, q) : fma(-w.y, p, q);
    b.x = fma(-w.x, re, a.x);
    b.y = fma(-w.x, im, a.y);
    a.x = fma(w.x, re, a.x);
    a.y = fma(w.x, im, a.y);
}
// the same with w = 1
__device__ __forceinline__ void bfly1(double2& a, double2& b) {
    const double2 t = b;
    b = csub(a, t);
    a = cadd(a, t);
}
template <bool INV> __device__ __forceinline__ double2 rot(double2 b) { return INV ? cmul_pi(b) : cmul_mi(b); }

// FP64 DFT of radix 2^LR on x with its twiddles (FIRST: none); w: the pass's
// rows in order, s4 / s2: tw_by_sine of the w^4 / w^2 rows (radix 8), of the
// w^2 / w rows (radix 4), of the w row (radix 2: s4)
template <bool INV, int LR, bool FIRST>
__device__ __forceinline__ void dft_fma(double2* x, const double2* w, bool s4, bool s2) {
    if constexpr (LR == 1) {
        if (FIRST) bfly1(x[0], x[1]);
        else bfly<INV>(x[0], x[1], w[0], s4);
    } else if constexpr (LR == 2) {
        // even: x0 +- w^2 x2, odd: x1 +- w^2 x3; then w and -i w
        if (FIRST) {
            bfly1(x[0], x[2]);
            bfly1(x[1], x[3]);
            x[3] = rot<INV>(x[3]);
            bfly1(x[0], x[1]);
            bfly1(x[2], x[3]);
        } else {
            bfly<INV>(x[0], x[2], w[0], s4);
            bfly<INV>(x[1], x[3], w[0], s4);
            x[3] = rot<INV>(x[3]);
            bfly<INV>(x[0], x[1], w[1], s2);
            bfly<INV>(x[2], x[3], w[1], s2);
        }
        const double2 t = x[1];   // x = X0, X2, X1, X3
        x[1] = x[2];
        x[2] = t;
    } else {
        if (FIRST) {
#pragma unroll
            for (int r = 0; r < 4; ++r) bfly1(x[r], x[r + 4]);
            x[6] = rot<INV>(x[6]);
            x[7] = rot<INV>(x[7]);
            bfly1(x[0], x[2]);
            bfly1(x[4], x[6]);
            bfly1(x[1], x[3]);
            bfly1(x[5], x[7]);
        } else {
#pragma unroll
            for (int r = 0; r < 4; ++r) bfly<INV>(x[r], x[r + 4], w[0], s4);
            x[6] = rot<INV>(x[6]);
            x[7] = rot<INV>(x[7]);
            bfly<INV>(x[0], x[2], w[1], s2);
            bfly<INV>(x[4], x[6], w[1], s2);
            bfly<INV>(x[1], x[3], w[1], s2);
            bfly<INV>(x[5], x[7], w[1], s2);
        }
        // even part G0, G2, G1, G3 in x0, x2, x4, x6; odd part H alike in
        // x1, x3, x5, x7; X_m = G_m +- w W8^m H_m
        x[3] = rot<INV>(x[3]);
        x[7] = rot<INV>(x[7]);
        const double2 w8 = make_double2(Consts<double>::rsqrt2, 1.0);   // e^{-i pi/4} by its cosine
        if (FIRST) {
            bfly1(x[0], x[1]);
            bfly1(x[2], x[3]);
            bfly<INV>(x[4], x[5], w8, false);
            bfly<INV>(x[6], x[7], w8, false);
        } else {
            bfly<INV>(x[0], x[1], w[2], false);   // angles in [0, 45) degrees
            bfly<INV>(x[2], x[3], w[2], false);
            bfly<INV>(x[4], x[5], w[3], true);    // and in [45, 90)
            bfly<INV>(x[6], x[7], w[3], true);
        }
        // x0, x1 = X0, X4; x4, x5 = X1, X5; x2, x3 = X2, X6; x6, x7 = X3, X7
        const double2 X4 = x[1], X1 = x[4], X6 = x[3], X3 = x[6];
        x[1] = X1;
        x[3] = X3;
        x[4] = X4;
        x[6] = X6;
    }
}

template <bool INV, class T, int LR> __device__ __forceinline__ void dft_r(Cx<T>* v) {
    if (LR == 3) {
        dft8<INV, T>(v);
    } else if (LR == 2) {
        dft4<INV>(v[0], v[1], v[2], v[3]);
    } else {
        const Cx<T> a = v[0], b = v[1];
        v[0] = cadd(a, b);
        v[1] = csub(a, b);
    }
}

// One pass of radix R = 2^LR with Stockham stride Ns = 2^nsl over the E =
// 2^LE elements of each sequence: E/R butterflies, number b = t + u N/E on
// registers u + r E/R, twiddled by the pass's rows at k = b mod Ns.
template <bool INV, class T, int LE, int LR, int M, bool FIRST>
__device__ __forceinline__ void pass_regs(Cx<T> (&v)[M][1 << LE], int t, int lt, int nsl,
                                          const Cx<T>* __restrict__ tw) {
    constexpr int E = 1 << LE, R = 1 << LR, U = E / R;
    const int Ns = 1 << nsl;
#pragma unroll
    for (int u = 0; u < U; ++u) {
        const int k = (t + (u << lt)) & (Ns - 1);
        if constexpr (std::is_same<T, double>::value) {
            constexpr int Q = tw_rows<T>(LR);
            double2 w[Q];
            bool s4 = false, s2 = false;
            if (!FIRST) {
#pragma unroll
                for (int q = 0; q < Q; ++q) w[q] = ldg_c(tw + q * Ns + k);
                // the top row's angle is pi k / Ns, the next one's half of that
                s4 = (((4 * k >> nsl) + 1) >> 1) & 1;
                s2 = (2 * k >> nsl) & 1;
            }
#pragma unroll
            for (int m = 0; m < M; ++m) {
                double2 x[R];
#pragma unroll
                for (int r = 0; r < R; ++r) x[r] = v[m][u + r * U];
                dft_fma<INV, LR, FIRST>(x, w, s4, s2);
#pragma unroll
                for (int r = 0; r < R; ++r) v[m][u + r * U] = x[r];
            }
        } else {
            if (!FIRST) {
#pragma unroll
                for (int r = 1; r < R; ++r) {
                    const auto w = TwEntry<T>::load(tw, (r - 1) * Ns + k);
#pragma unroll
                    for (int m = 0; m < M; ++m) v[m][u + r * U] = twiddle<INV, T>(v[m][u + r * U], w);
                }
            }
#pragma unroll
            for (int m = 0; m < M; ++m) {
                Cx<T> x[R];
#pragma unroll
                for (int r = 0; r < R; ++r) x[r] = v[m][u + r * U];
                dft_r<INV, T, LR>(x);
#pragma unroll
                for (int r = 0; r < R; ++r) v[m][u + r * U] = x[r];
            }
        }
    }
}

// Barrier of the threads that share a sequence: one warp, or `count` threads
// (named barrier `id`, 1 .. 15), or the block (id 0).
struct SeqSync {
    bool warp;
    int id = 0, count = 0;
    __device__ __forceinline__ void operator()() const {
        if (warp) __syncwarp();
        else if (id) asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(count) : "memory");
        else __syncthreads();
    }
};

// The exchange after a pass and the next pass of fft_regs: rem factors of two
// are left, nsl are done.
template <bool INV, class T, int LE, int M>
__device__ __forceinline__ void exchange_and_pass(Cx<T> (&v)[M][1 << LE], Cx<T>* d, int ms, int t, int lt,
                                                  const Cx<T>* __restrict__& tw, SeqSync sync, int& rem, int& nsl) {
    constexpr int E = 1 << LE, PL = kPadLog<T>;
    Cx<T>* const rd = d + sw<T>(t);
    // thread t's butterfly of the last pass wrote (t - k) E + k + r Ns, k = t mod Ns
    const int Ns = 1 << nsl;
    const int k = t & (Ns - 1);
    Cx<T>* const wr = d + sw<T>(((t - k) << LE) + k);
    if (nsl == 0) {
#pragma unroll
        for (int m = 0; m < M; ++m)
#pragma unroll
            for (int r = 0; r < E; ++r) wr[m * ms + r] = v[m][r];
    } else if (LE == 1 || nsl >= PL) {
        const int st = Ns + (Ns >> PL);
#pragma unroll
        for (int m = 0; m < M; ++m)
#pragma unroll
            for (int r = 0; r < E; ++r) wr[m * ms + r * st] = v[m][r];
    } else {
        // the second exchange, Ns = E < 2^PL
#pragma unroll
        for (int m = 0; m < M; ++m)
#pragma unroll
            for (int r = 0; r < E; ++r) wr[m * ms + r * E + ((r * E) >> PL)] = v[m][r];
    }
    sync();
    const int tps = 1 << lt;
    if (lt >= PL) {
        const int st = tps + (tps >> PL);
#pragma unroll
        for (int m = 0; m < M; ++m)
#pragma unroll
            for (int r = 0; r < E; ++r) v[m][r] = rd[m * ms + r * st];
    } else {
#pragma unroll
        for (int m = 0; m < M; ++m)
#pragma unroll
            for (int r = 0; r < E; ++r) v[m][r] = rd[m * ms + (r << lt) + ((r << lt) >> PL)];
    }
    sync();
    nsl += LE;
    if (rem >= LE) {
        pass_regs<INV, T, LE, LE, M, false>(v, t, lt, nsl, tw);
        tw += kTwWidth<T> * (tw_rows<T>(LE) << nsl);
        rem -= LE;
    } else {
        if (LE == 3 && rem == 2) pass_regs<INV, T, LE, (LE == 3 ? 2 : 1), M, false>(v, t, lt, nsl, tw);
        if (rem == 1) pass_regs<INV, T, LE, 1, M, false>(v, t, lt, nsl, tw);
        rem = 0;
    }
}

// Transform M sequences held in registers (see the file comment).  d: shared
// memory of this thread's sequences, sequence m at d + m ms (padded_len(N)
// slots each); t: the thread's number in the sequence, < 2^lt = N/E; tw: the
// twiddle table of this N and LE.  All threads behind `sync` must call it; the
// shared memory is free again when it returns.  LT: lt as a constant (-1: not
// known), which unrolls the passes and makes every shared-memory and twiddle
// address of one an immediate offset.
template <bool INV, class T, int LE, int M, int LT = -1>
__device__ __forceinline__ void fft_regs(Cx<T> (&v)[M][1 << LE], Cx<T>* d, int ms, int t, int lt,
                                         const Cx<T>* __restrict__ tw, SeqSync sync) {
    if (LT >= 0) lt = LT;
    int rem = lt, nsl = 0;   // logN - LE factors of two after the first pass
    pass_regs<INV, T, LE, LE, M, true>(v, t, lt, 0, tw);
    if constexpr (LT >= 0) {
#pragma unroll
        for (int pass = 0; pass < (LT + LE - 1) / LE; ++pass) exchange_and_pass<INV, T, LE, M>(v, d, ms, t, lt, tw, sync, rem, nsl);
    } else {
#pragma unroll 1
        while (rem > 0) exchange_and_pass<INV, T, LE, M>(v, d, ms, t, lt, tw, sync, rem, nsl);
    }
}

// In-place transform of nseq sequences in shared memory, sequence f at
// seq(f) (a device functor), padded layout.  All threads of the block must
// call it; blockDim.x >= N/E.
template <bool INV, class T, int LE, class SeqPtr>
__device__ void fft_smem_seqs(SeqPtr seq, int logN, int nseq, const Cx<T>* __restrict__ tw) {
    constexpr int E = 1 << LE;
    const int lt = logN - LE, t = threadIdx.x & ((1 << lt) - 1);
    const int F = blockDim.x >> lt;             // sequences per round
    for (int f0 = 0; f0 < nseq; f0 += F) {
        const int f = f0 + (threadIdx.x >> lt);
        const bool act = f < nseq;
        Cx<T>* d = seq(act ? f : 0);
        Cx<T> v[1][E];
#pragma unroll
        for (int r = 0; r < E; ++r) v[0][r] = act ? d[sw<T>(t + (r << lt))] : mk<T>(T(0), T(0));
        // threads without a sequence of their own (act false) take part in the
        // barriers only
        constexpr int PL = kPadLog<T>;
        int rem = lt, nsl = 0;
        const Cx<T>* twp = tw;
        pass_regs<INV, T, LE, LE, 1, true>(v, t, lt, 0, twp);
        __syncthreads();
#pragma unroll 1
        while (rem > 0) {
            const int Ns = 1 << nsl, k = t & (Ns - 1);
            Cx<T>* const wr = d + sw<T>(((t - k) << LE) + k);
            if (act) {
#pragma unroll
                for (int r = 0; r < E; ++r) wr[(r << nsl) + ((r << nsl) >> PL)] = v[0][r];
            }
            __syncthreads();
            if (act) {
#pragma unroll
                for (int r = 0; r < E; ++r) v[0][r] = d[sw<T>(t + (r << lt))];
            }
            __syncthreads();
            nsl += LE;
            if (rem >= LE) {
                pass_regs<INV, T, LE, LE, 1, false>(v, t, lt, nsl, twp);
                twp += kTwWidth<T> * (tw_rows<T>(LE) << nsl);
                rem -= LE;
            } else {
                if (LE == 3 && rem == 2) pass_regs<INV, T, LE, (LE == 3 ? 2 : 1), 1, false>(v, t, lt, nsl, twp);
                if (rem == 1) pass_regs<INV, T, LE, 1, 1, false>(v, t, lt, nsl, twp);
                rem = 0;
            }
        }
        if (act) {
#pragma unroll
            for (int r = 0; r < E; ++r) d[sw<T>(t + (r << lt))] = v[0][r];
        }
        __syncthreads();
    }
}

}  // namespace nsstab
