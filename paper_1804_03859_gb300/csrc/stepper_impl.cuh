// The vorticity-streamfunction time-stepper: kernels and host driver.
//
// One time step (nonlinear or linearised, Sec. 3, Eqs. 28-30) is six
// kernels (five in FP32), alternating row passes (x-direction FFT of two real
// rows packed into one complex transform, with the finite-difference stencil
// fused into the forward pass) and column passes (y-direction FFT with the
// spectral diagonal operators fused between the forward and inverse
// transforms):
//
//   col_poisson   X1 (x-spectrum of omega)  -> Wh = FFT2(omega), X2 = x-spectrum of psi
//   row_inverse   X2                        -> P = psi
//   row_forward   RHS: W, P (+ base)        -> X1 = x-spectrum of N
//   col_update    X1, Wh, Nh                -> Nh = FFT2(N), X1/X2 = x-spectra of omega*, psi*
//   row_inverse   X1, X2                    -> W = omega*, P = psi* (where the penalisation reads it)
//   row_forward   PEN: W, P (+ SFD state Y) -> W = omega^{n+1}, X1 = its x-spectrum
//
// FP32: the right-hand side needs u' and v only at the point itself, so its
// row pass transforms the pair's u' and v spectra and uses the values in
// registers; they are never written and the second kernel drops out.
//
// FP32 steppers take three measures against error that a time-stepper
// would otherwise accumulate over hundreds of steps:
//  * they carry the velocity instead of the streamfunction: the column
//    passes form the x-spectra of u' = D_y psi and v = -D_x psi by
//    multiplying psi^ with the centred-difference symbols i sin(k h)/h (the
//    same discrete operator as the stencil on psi), and the inverse row
//    passes produce U, V (and W).  The stencil on a rounded psi loses about
//    log2(|psi| / (h |D psi|)) bits to cancellation (a per-step error near
//    7e-6 at 512x256); the spectral form keeps the velocity error at the
//    rounding of the velocity itself;
//  * the Crank-Nicolson factor A = (1 + nu dt lam/2)/(1 - nu dt lam/2),
//    within 1e-3 of 1 for the modes that carry the flow, is stored as
//    A - 1: an FP32 A is a fixed relative error of up to 3e-8 applied at
//    every step, which grows linearly over a run;
//  * their transforms split each twiddle into hi + lo (fft.cuh), for the
//    same reason.
// Together these take the FP32 propagator of 200 steps from about 1e-5 to
// about 1e-6 relative to FP64.  The FP64 and double-float steppers keep psi,
// the stencil and plain tables (their rounding is far below the parity bar),
// with 1.5x fewer row transforms.
//
// Layouts: physical fields [ny][nx] (x fastest).  The x-spectra (X1 .. X4),
// which row passes and column passes both touch, are stored [ny/4][kx][4]
// over the nx/2 packed x-wavenumbers (kXRows).  Column-major they cost the row
// passes 8 or 16 bytes of every sector: 658 us for the FP32 u', v inverse pass
// of 32 fields at 2048x1024, against 411 us for three fields now.  Full
// spectra and tables, private to the column passes, are [kx][ky].  Spectra
// are stored doubled (split_pair); the operator tables hold the half.  The x-transform of a
// real row is packed into nx/2 complex slots: slot 0 holds X[0] (real) in
// .x and X[nx/2] (real) in .y.  In the column passes the packed kx = 0
// column is the y-transform of (X0 + i XN); the spectral operators act on it
// through its Hermitian halves (see apply_packed0).
#pragma once

#include <algorithm>
#include <cmath>
#include <cstring>
#include <map>
#include <type_traits>
#include <vector>

#include "fft.cuh"
#include "stepper.cuh"

namespace nsstab {

// TAN: a trajectory (member 0, nonlinear) and a perturbation (member 1,
// linearised about member 0's state) in one launch
enum RowMode { FWD_PLAIN = 0, FWD_RHS_NL = 1, FWD_RHS_LIN = 2, FWD_PEN_NL = 3, FWD_PEN_LIN = 4, FWD_RHS_TAN = 5,
               FWD_PEN_TAN = 6 };

// The FP32 stepper's accuracy measures (see the file comment): velocities
// in place of psi, and the Crank-Nicolson factor stored as A - 1.  (Its
// transforms also split twiddles into hi + lo; see fft.cuh.)
template <class T> constexpr bool kF32 = std::is_same<T, float>::value;

constexpr int kPenChunkLog = 5;

template <class T> struct Fields {
    int nx, ny, nxh, logx, logy;
    int bper;              // members per parameter set (member m uses set m / bper)
    size_t fs, cs, ts;     // member strides: physical field, spectrum, operator table
    const unsigned char* active;   // per-member flag: inactive members skip every kernel
    T idx2, idy2;          // 1/(2 dx), 1/(2 dy)
    T Uinf;
    T scale;               // 1/(2 nx ny): normalisation of the inverse transform of spectra stored doubled (split_pair)
    T sfd_k1, sfd_k2;      // dt*chi_sfd, dt/Delta
    T* W;                  // omega (physical)
    T* P;                  // psi (physical)
    T* U; T* V;            // u' = D_y psi, v = -D_x psi (physical; FP32 steppers)
    T* Y;                  // SFD filtered state
    const T* cS;           // s/(1+s), s = dt (chi/eta + sigma)
    // FP32: dt sigma Uinf / (1+s).  Otherwise the terms of the nonlinear
    // correction that do not depend on psi*: -D_y of (cG - cS Uinf)
    const T* cG;
    // per row pair and chunk of 2^kPenChunkLog columns: bit 0, a penalisation
    // coefficient in reach of the chunk's stencils is non-zero; bit 1, such a
    // stencil reads the chunk's intermediate velocity or psi
    const unsigned char* pf;
    int logc;              // log2 of the chunks per row
    const T* Ub; const T* Vb; const T* DxOb; const T* DyOb;   // base-derived fields
    Cx<T>* X1; Cx<T>* X2;  // x-spectral, y-physical [ny/4][kx][4] (kXRows)
    Cx<T>* X3;             // x-spectrum of v (FP32 steppers)
    Cx<T>* X4;             // x-spectrum of N written by the fused row pass (FP32)
    const Cx<T>* XN;       // x-spectrum of N read by k_col_update (X1, or X4)
    Cx<T>* Wh; Cx<T>* Nh;  // full spectra [kx][ky]
    const T* tA; const T* tB; const T* tP;   // spectral operator tables [nxh+1][ny]
    const T* tDx; const T* tDy;              // sin(2 pi kx/nx)/dx [nxh+1], sin(2 pi ky/ny)/dy [ny]
    const Cx<T>* twx[4]; const Cx<T>* twy[4];   // per-pass twiddle tables for LE = 1, 2, 3
};

// Offset the member-dependent pointers to member m (and its parameter
// set).  Returns false for an inactive member: its blocks return
// at once, so independent solves of a batch can drop out or idle.
template <class T> __device__ __forceinline__ bool member_view_at(Fields<T>& f, int m) {
    if (f.active && !f.active[m]) return false;
    const int set = m / f.bper;
    const size_t fo = (size_t)m * f.fs, co = (size_t)m * f.cs, so = (size_t)set * f.fs, to = (size_t)set * f.ts;
    f.W += fo;
    f.P += fo;
    if (f.Y) f.Y += fo;
    f.X1 += co;
    f.X2 += co;
    f.XN += co;
    if (kF32<T>) {
        f.U += fo;
        f.V += fo;
        f.X3 += co;
        f.X4 += co;
    }
    f.Wh += co;
    f.Nh += co;
    f.cS += so;
    f.cG += so;
    f.pf += (size_t)set * (f.ny >> 1) << f.logc;
    if (f.Ub) {
        f.Ub += so;
        f.Vb += so;
        f.DxOb += so;
        f.DyOb += so;
    }
    f.tA += to;
    f.tB += to;
    return true;
}

template <class T> __device__ __forceinline__ bool member_view(Fields<T>& f) { return member_view_at(f, blockIdx.y); }

// Diagonal operators at (kx, ky), kx in [0, nx/2]: Crank-Nicolson A = a/b
// (FP32 steppers: A - 1), B = dt/b (both times 1/(2 nx ny): the inverse
// transform of spectra stored doubled) and the inverse Laplacian P = -1/lam
// (zero for the mean mode), read from tables
// computed on the host in FP64 and rounded once to the stepper's precision
// (a division costs ~10 FP64 instructions on GB300, and evaluating them in
// FP32 on the device adds several roundings that show in the FP32
// eigenvalues).
template <class T> struct SpecOp {
    __device__ static __forceinline__ void ab(const Fields<T>& f, int kx, int ky, T& A, T& B) {
        const size_t g = (size_t)kx * f.ny + ky;
        A = f.tA[g];
        B = f.tB[g];
    }
    __device__ static __forceinline__ T p(const Fields<T>& f, int kx, int ky) { return f.tP[(size_t)kx * f.ny + ky]; }
};

// ------------------------------------------------------------ row kernels

// Register budget: blocks of up to 512 threads at 8 elements per thread (the
// largest rows, nx = 4096, need 512), up to 1024 otherwise.
#define NS_FFT_BOUNDS __launch_bounds__(LE == 3 ? 512 : 1024)

// A row pass works on row pairs: rows a = 2 p and b = 2 p + 1 of a field are
// one complex sequence.  Thread t of a pair holds the columns t + r nx/E.
// LN: log2 nx as a constant (0: not known), see fft_regs.
template <class T, int LE, int LN = 0> struct RowUnit {
    static constexpr int kLT = LN ? LN - LE : -1;
    int q, t, lt, tps;   // sequence within the block, thread within it, log2 / number of its threads
    SeqSync sync;
    __device__ __forceinline__ explicit RowUnit(const Fields<T>& f) {
        lt = LN ? LN - LE : f.logx - LE;
        tps = 1 << lt;
        t = threadIdx.x & (tps - 1);
        q = threadIdx.x >> lt;
        sync.warp = lt <= 5;
    }
};

// Rows of an x-spectrum stored side by side, [ny/4][kx][4].  A warp of a row
// pass (one pair) reads 16-byte pieces 32 bytes apart, eight 128-byte lines;
// one of a column pass (32 values of y) eight runs of 32 bytes, eight lines.
// With 2 rows the column passes touch 16 lines an access and are bound by
// them (69-73% of the L1 wavefronts), with 8 rows the row passes are: step of
// 32 FP32 fields at 2048x1024 2486 / 2232 / 2293 us with 2 / 4 / 8.
constexpr int kXRows = 4;
template <class T> __device__ __forceinline__ size_t xs_pair(const Fields<T>& f, int pair, int kx) {
    return ((size_t)(pair >> 1) * f.nxh + kx) * kXRows + (pair & 1) * 2;
}

// Half-spectra of M real row pairs (arrays X[m], at element offset `off` of
// the pair) as the sequences A + i B in registers: the lower half is formed
// by the thread that holds it, the upper half (the conjugate part) goes
// through shared memory d, sequence m at d + m ms.  cross (M = 2): row a of
// both arrays as the first sequence, row b of both as the second, instead of
// rows a, b of each.
template <class T, int LE, int M, int LN>
__device__ __forceinline__ void merge_pairs(Cx<T> (&v)[M][1 << LE], const Cx<T>* const (&X)[M], int nx, Cx<T>* d,
                                            int ms, const RowUnit<T, LE, LN>& u, bool cross = false) {
    constexpr int E = 1 << LE, H = E / 2;
    const int nh = nx >> 1;
    Cx<T> A[M][H], B[M][H];
#pragma unroll
    for (int m = 0; m < M; ++m)
#pragma unroll
        for (int r = 0; r < H; ++r) PairIO<T>::load(X[m] + kXRows * (u.t + (r << u.lt)), A[m][r], B[m][r]);
    if (M == 2 && cross) {
#pragma unroll
        for (int r = 0; r < H; ++r) {
            const Cx<T> t = B[0][r];
            B[0][r] = A[M - 1][r];
            A[M - 1][r] = t;
        }
    }
#pragma unroll
    for (int m = 0; m < M; ++m)
#pragma unroll
        for (int r = 0; r < H; ++r) {
            const int k = u.t + (r << u.lt);
            Cx<T> lo = mk<T>(A[m][r].x - B[m][r].y, A[m][r].y + B[m][r].x);   // A + i B
            Cx<T> hi = mk<T>(A[m][r].x + B[m][r].y, B[m][r].x - A[m][r].y);   // conj(A) + i conj(B), at nx - k
            if (k == 0) {   // slot 0 packs X[0] and X[nx/2], both real
                lo = mk<T>(A[m][r].x, B[m][r].x);
                hi = mk<T>(A[m][r].y, B[m][r].y);
            }
            v[m][r] = lo;
            d[m * ms + sw<T>((nh - k) & (nh - 1))] = hi;
        }
    u.sync();
#pragma unroll
    for (int m = 0; m < M; ++m)
#pragma unroll
        for (int r = 0; r < H; ++r) v[m][H + r] = d[m * ms + sw<T>(u.t + (r << u.lt))];
    u.sync();
}

// One row of two arrays (A, B at its first element) as the sequence A + i B,
// as merge_pairs.
template <class T, int LE, int LN>
__device__ __forceinline__ void merge_rows(Cx<T>* v, const Cx<T>* XA, const Cx<T>* XB, int nx, Cx<T>* d,
                                           const RowUnit<T, LE, LN>& u) {
    constexpr int E = 1 << LE, H = E / 2;
    const int nh = nx >> 1;
    Cx<T> A[H], B[H];
#pragma unroll
    for (int r = 0; r < H; ++r) {
        A[r] = XA[kXRows * (u.t + (r << u.lt))];
        B[r] = XB[kXRows * (u.t + (r << u.lt))];
    }
#pragma unroll
    for (int r = 0; r < H; ++r) {
        const int k = u.t + (r << u.lt);
        v[r] = k ? mk<T>(A[r].x - B[r].y, A[r].y + B[r].x) : mk<T>(A[r].x, B[r].x);
        d[sw<T>((nh - k) & (nh - 1))] = k ? mk<T>(A[r].x + B[r].y, B[r].x - A[r].y) : mk<T>(A[r].y, B[r].y);
    }
    u.sync();
#pragma unroll
    for (int r = 0; r < H; ++r) v[H + r] = d[sw<T>(u.t + (r << u.lt))];
    u.sync();
}

// The reverse: a transformed pair Z = FFT(a + i b) in registers into twice
// the half-spectra of a and b (the factor is in the operator tables),
// stored to X at the pair's element offset.
template <class T, int LE, int LN>
__device__ __forceinline__ void split_pair(const Cx<T>* v, Cx<T>* X, int nx, Cx<T>* d, const RowUnit<T, LE, LN>& u) {
    constexpr int E = 1 << LE, H = E / 2;
    const int nh = nx >> 1;
#pragma unroll
    for (int r = 0; r < H; ++r) d[sw<T>(u.t + (r << u.lt))] = v[H + r];
    u.sync();
#pragma unroll
    for (int r = 0; r < H; ++r) {
        const int k = u.t + (r << u.lt);
        const Cx<T> zk = v[r], zm = d[sw<T>((nh - k) & (nh - 1))];   // Z[nx - k] (k = 0: Z[nx/2])
        Cx<T> A = mk<T>(zk.x + zm.x, zk.y - zm.y);   // Z_k + conj(Z_{nx-k})
        Cx<T> B = mk<T>(zk.y + zm.y, zm.x - zk.x);   // -i (Z_k - conj(Z_{nx-k}))
        if (k == 0) {
            A = mk<T>(T(2) * zk.x, T(2) * zm.x);
            B = mk<T>(T(2) * zk.y, T(2) * zm.y);
        }
        PairIO<T>::store(X + kXRows * k, A, B);
    }
}

// Row offsets of pair p: rows a - 2 .. b + 2 = 2 p - 2 .. 2 p + 3, periodic.
struct RowOffs {
    int am2, am1, a, b, bp1, bp2;
    __device__ __forceinline__ RowOffs(int pair, int nx, int ny) {
        const int j = 2 * pair;
        am2 = ((j - 2) & (ny - 1)) * nx;
        am1 = ((j - 1) & (ny - 1)) * nx;
        a = j * nx;
        b = (j + 1) * nx;
        bp1 = ((j + 2) & (ny - 1)) * nx;
        bp2 = ((j + 3) & (ny - 1)) * nx;
    }
};

// Where a row pass finds psi (or u', v: FP32) at row a + j, j = -2 .. 3, of
// its pair: in memory, or in the transformed pairs p - 1, p, p + 1 (and, for v,
// one more) in shared memory, S elements apart.
template <class T> struct GlobalRows {
    const Fields<T>& f;
    const RowOffs& o;
    __device__ __forceinline__ int off(int j) const {
        return j == -2 ? o.am2 : j == -1 ? o.am1 : j == 0 ? o.a : j == 1 ? o.b : j == 2 ? o.bp1 : o.bp2;
    }
    __device__ __forceinline__ T p(int j, int i) const { return f.P[off(j) + i]; }
    __device__ __forceinline__ T u(int j, int i) const { return f.U[off(j) + i]; }
    __device__ __forceinline__ T v(int j, int i) const { return f.V[off(j) + i]; }
};
template <class T> struct TileRows {
    const Cx<T>* q;
    int S;
    __device__ __forceinline__ T at(int tile, int j, int i) const {
        const Cx<T>& z = q[tile * S + sw<T>(i)];
        return (j & 1) ? z.y : z.x;
    }
    __device__ __forceinline__ T p(int j, int i) const { return at((j + 2) >> 1, j, i); }
    // u of rows a, b is the second row of tiles 1, 4, beside omega*
    __device__ __forceinline__ T u(int j, int i) const {
        return j == 0 ? at(1, 1, i) : j == 1 ? at(4, 1, i) : at((j + 2) >> 1, j, i);
    }
    __device__ __forceinline__ T v(int j, int i) const { return at(3, j, i); }
};
// psi differences of rows a, b at column i: (ua, ub) along y, (va, vb) along x
template <class T, class R>
__device__ __forceinline__ void psi_diffs(const R& q, int i, int nx, T& ua, T& ub, T& va, T& vb) {
    const int ip = (i + 1) & (nx - 1), im = (i - 1) & (nx - 1);
    ua = q.p(1, i) - q.p(-1, i);
    ub = q.p(2, i) - q.p(0, i);
    va = q.p(0, ip) - q.p(0, im);
    vb = q.p(1, ip) - q.p(1, im);
}

// Advection term of rows a, b at column i, as (N_a, N_b).  FP32: (ua, ub) =
// u', (va, vb) = v at rows a, b; otherwise the differences of psi (psi_diffs).
// LIN: N' = Ub dW_x + Vb dW_y + Ox u' + Oy v' with the scales and signs of
// k_base_fields, d the undivided centred differences.
template <class T, bool LIN>
__device__ __forceinline__ Cx<T> rhs_point(const Fields<T>& f, int i, const RowOffs& o, T ua, T ub, T va, T vb) {
    const int nx = f.nx;
    const int ip = (i + 1) & (nx - 1), im = (i - 1) & (nx - 1);
    const T* W = f.W;
    const T wa = W[o.a + i], wb = W[o.b + i];
    const T dxa = W[o.a + ip] - W[o.a + im], dxb = W[o.b + ip] - W[o.b + im];
    const T dya = wb - W[o.am1 + i], dyb = W[o.bp1 + i] - wa;
    if (LIN) {
        const T na = f.Ub[o.a + i] * dxa + f.Vb[o.a + i] * dya + ua * f.DxOb[o.a + i] + va * f.DyOb[o.a + i];
        const T nb = f.Ub[o.b + i] * dxb + f.Vb[o.b + i] * dyb + ub * f.DxOb[o.b + i] + vb * f.DyOb[o.b + i];
        return mk<T>(na, nb);
    }
    // N = -(u D_x w + v D_y w)
    if (kF32<T>) {
        return mk<T>(-((f.Uinf + ua) * (dxa * f.idx2) + va * (dya * f.idy2)),
                     -((f.Uinf + ub) * (dxb * f.idx2) + vb * (dyb * f.idy2)));
    }
    // u = Uinf + idy2 dpsi_y, v = -idx2 dpsi_x: N = idx2 (idy2 dpsi_x dw_y - u dw_x)
    const T uA = f.Uinf + f.idy2 * ua, uB = f.Uinf + f.idy2 * ub;
    return mk<T>(f.idx2 * (f.idy2 * (va * dya) - uA * dxa), f.idx2 * (f.idy2 * (vb * dyb) - uB * dxb));
}

// Advection term of the perturbation (member 1, at f) linearised about the
// trajectory (member 0, one member stride before it) at rows a, b of column i.
// FP32: uv = u', v of member 1, uv0 those of member 0, as (row a, row b).
template <class T>
__device__ __forceinline__ Cx<T> tan_point(const Fields<T>& f, int i, const RowOffs& o, Cx<T> u1, Cx<T> v1, Cx<T> u0,
                                           Cx<T> v0) {
    const int nx = f.nx;
    const int ip = (i + 1) & (nx - 1), im = (i - 1) & (nx - 1);
    const T *W = f.W, *W0 = f.W - f.fs;
    const T dxa = W[o.a + ip] - W[o.a + im], dxb = W[o.b + ip] - W[o.b + im];
    const T dya = W[o.b + i] - W[o.am1 + i], dyb = W[o.bp1 + i] - W[o.a + i];
    const T xa = W0[o.a + ip] - W0[o.a + im], xb = W0[o.b + ip] - W0[o.b + im];
    const T ya = W0[o.b + i] - W0[o.am1 + i], yb = W0[o.bp1 + i] - W0[o.a + i];
    if constexpr (kF32<T>) {
        return mk<T>(-((f.Uinf + u0.x) * (dxa * f.idx2) + v0.x * (dya * f.idy2) + u1.x * (xa * f.idx2) + v1.x * (ya * f.idy2)),
                     -((f.Uinf + u0.y) * (dxb * f.idx2) + v0.y * (dyb * f.idy2) + u1.y * (xb * f.idx2) + v1.y * (yb * f.idy2)));
    } else {
        // u = idy2 dpsi_y, v = -idx2 dpsi_x of both members
        const T *P = f.P, *P0 = f.P - f.fs;
        const T pxa = P[o.a + ip] - P[o.a + im], pxb = P[o.b + ip] - P[o.b + im];
        const T pya = P[o.b + i] - P[o.am1 + i], pyb = P[o.bp1 + i] - P[o.a + i];
        const T qxa = P0[o.a + ip] - P0[o.a + im], qxb = P0[o.b + ip] - P0[o.b + im];
        const T qya = P0[o.b + i] - P0[o.am1 + i], qyb = P0[o.bp1 + i] - P0[o.a + i];
        const T uA = f.Uinf + f.idy2 * qya, uB = f.Uinf + f.idy2 * qyb;
        return mk<T>(f.idx2 * (f.idy2 * (qxa * dya + pxa * ya - pya * xa) - uA * dxa),
                     f.idx2 * (f.idy2 * (qxb * dyb + pxb * yb - pyb * xb) - uB * dxb));
    }
}

// Correction D_x dv - D_y du of the implicit Brinkman + fringe split (du = cG
// - cS u*, dv = -cS v*) at rows a, b of column i, where some coefficient of
// the stencil is non-zero (see Fields::pf).
template <class T, bool LIN, class R>
__device__ __forceinline__ Cx<T> pen_point(const Fields<T>& f, const R& q, int i, const RowOffs& o) {
    const int nx = f.nx;
    const int ip = (i + 1) & (nx - 1), im = (i - 1) & (nx - 1);
    const T* S = f.cS;
    const T sam = S[o.am1 + i], sa = S[o.a + i], sb = S[o.b + i], sbp = S[o.bp1 + i];
    if constexpr (kF32<T>) {
        const T Ui = LIN ? T(0) : f.Uinf;
        const T dva = S[o.a + im] * q.v(0, im) - S[o.a + ip] * q.v(0, ip);
        const T dvb = S[o.b + im] * q.v(1, im) - S[o.b + ip] * q.v(1, ip);
        T dum = -sam * (Ui + q.u(-1, i)), dua = -sa * (Ui + q.u(0, i));
        T dub = -sb * (Ui + q.u(1, i)), dup = -sbp * (Ui + q.u(2, i));
        if (!LIN) {
            const T* G = f.cG;
            dum += G[o.am1 + i];
            dua += G[o.a + i];
            dub += G[o.b + i];
            dup += G[o.bp1 + i];
        }
        return mk<T>(dva * f.idx2 - (dub - dum) * f.idy2, dvb * f.idx2 - (dup - dua) * f.idy2);
    } else {
        // u* = Uinf + idy2 dpsi_y, v* = -idx2 dpsi_x; the terms without psi*
        // are the field cG
        const int ipp = (i + 2) & (nx - 1), imm = (i - 2) & (nx - 1);
        const T pa = q.p(0, i), pb = q.p(1, i);
        const T xa = S[o.a + ip] * (q.p(0, ipp) - pa) - S[o.a + im] * (pa - q.p(0, imm));
        const T xb = S[o.b + ip] * (q.p(1, ipp) - pb) - S[o.b + im] * (pb - q.p(1, imm));
        const T ya = sb * (q.p(2, i) - pa) - sam * (pa - q.p(-2, i));
        const T yb = sbp * (q.p(3, i) - pb) - sa * (pb - q.p(-1, i));
        T ca = f.idx2 * f.idx2 * xa + f.idy2 * f.idy2 * ya;
        T cb = f.idx2 * f.idx2 * xb + f.idy2 * f.idy2 * yb;
        if (!LIN) {
            ca = ca + f.cG[o.a + i];
            cb = cb + f.cG[o.b + i];
        }
        return mk<T>(ca, cb);
    }
}

// Bring the rows a right-hand-side pass reads after its inverse transforms
// into L2 (the pair's rows of W and of the base-derived fields, one 128-byte
// line per instruction), while these run: with 64 registers the pass has few
// loads in flight of its own, but twice the warps (k_row_forward).
template <class T, bool LIN>
__device__ __forceinline__ void prefetch_rows(const Fields<T>& f, int pair, int t, int tps) {
    constexpr int line = 128 / (int)sizeof(T);
    for (int c = t * line; c < 2 * f.nx; c += tps * line) {
        const size_t o = (size_t)2 * pair * f.nx + c;
        asm volatile("prefetch.global.L2 [%0];" ::"l"(f.W + o));
        if (LIN) {
            asm volatile("prefetch.global.L2 [%0];" ::"l"(f.Ub + o));
            asm volatile("prefetch.global.L2 [%0];" ::"l"(f.Vb + o));
            asm volatile("prefetch.global.L2 [%0];" ::"l"(f.DxOb + o));
            asm volatile("prefetch.global.L2 [%0];" ::"l"(f.DyOb + o));
        }
    }
}

// Forward x-transform of RP row pairs per block, with the row values made by
// MODE.  RHS modes: the advection term (FP32: first the inverse transforms of
// the pair's u' and v spectra X2, X3, whose values are used where they stand
// and never written).  PEN modes: omega^{n+1} = omega* + the penalisation
// correction (and the SFD filter), stored to W.  Writes the pair's
// half-spectra to X1 when do_fft.  m: the member (TAN modes).
template <class T, int MODE, int LE, int LN = 0>
__device__ __forceinline__ void row_forward_body(const Fields<T>& f, int m, int bx, int RP, bool sfd, bool do_fft) {
    using C = Cx<T>;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    constexpr int E = 1 << LE;
    constexpr bool RHS = (MODE == FWD_RHS_NL || MODE == FWD_RHS_LIN || MODE == FWD_RHS_TAN);
    constexpr bool LIN = (MODE == FWD_RHS_LIN || MODE == FWD_PEN_LIN);
    constexpr bool UV = RHS && kF32<T>;
    const int nx = LN ? 1 << LN : f.nx, S = padded_len<T>(nx);
    const RowUnit<T, LE, LN> u(f);
    const int pair = bx * RP + u.q;
    C* d = reinterpret_cast<C*>(smem_raw) + (size_t)u.q * (UV ? (MODE == FWD_RHS_TAN ? 4 : 2) : 1) * S;
    const RowOffs o(pair, nx, f.ny);
    C z[1][E];
    if (MODE == FWD_RHS_TAN && m == 1) {
        // FP32: u', v of the perturbation and of the trajectory, whose
        // transforms member 0's blocks make as well (no launch to wait for)
        C uv[UV ? 4 : 1][E];
        if constexpr (UV) {
            prefetch_rows<T, false>(f, pair, u.t, u.tps);
            const size_t x0 = xs_pair(f, pair, 0);
            const C* const X[4] = {f.X2 + x0, f.X3 + x0, f.X2 - f.cs + x0, f.X3 - f.cs + x0};
            merge_pairs<T, LE, 4>(uv, X, nx, d, S, u);
            fft_regs<true, T, LE, 4>(uv, d, S, u.t, u.lt, f.twx[LE], u.sync);
        }
#pragma unroll
        for (int r = 0; r < E; ++r) {
            const int i = u.t + (r << u.lt);
            if constexpr (UV) z[0][r] = tan_point<T>(f, i, o, uv[0][r], uv[1][r], uv[2][r], uv[3][r]);
            else z[0][r] = tan_point<T>(f, i, o, C{}, C{}, C{}, C{});
        }
    } else if constexpr (RHS) {
        C uv[UV ? 2 : 1][E];
        if constexpr (UV) prefetch_rows<T, LIN>(f, pair, u.t, u.tps);
        if constexpr (UV) {
            const size_t x0 = xs_pair(f, pair, 0);
            const C* const X[2] = {f.X2 + x0, f.X3 + x0};
            merge_pairs<T, LE, 2>(uv, X, nx, d, S, u);
            fft_regs<true, T, LE, 2>(uv, d, S, u.t, u.lt, f.twx[LE], u.sync);
        }
#pragma unroll
        for (int r = 0; r < E; ++r) {
            const int i = u.t + (r << u.lt);
            if constexpr (UV) z[0][r] = rhs_point<T, LIN>(f, i, o, uv[0][r].x, uv[0][r].y, uv[1][r].x, uv[1][r].y);
            else {
                T ua, ub, va, vb;
                psi_diffs<T>(GlobalRows<T>{f, o}, i, nx, ua, ub, va, vb);
                z[0][r] = rhs_point<T, LIN>(f, i, o, ua, ub, va, vb);
            }
        }
    } else if constexpr (MODE == FWD_PLAIN) {
#pragma unroll
        for (int r = 0; r < E; ++r) {
            const int i = u.t + (r << u.lt);
            z[0][r] = mk<T>(f.W[o.a + i], f.W[o.b + i]);
        }
    } else {
        const unsigned char* pf = f.pf + ((size_t)pair << f.logc);
#pragma unroll
        for (int r = 0; r < E; ++r) {
            const int i = u.t + (r << u.lt);
            z[0][r] = mk<T>(f.W[o.a + i], f.W[o.b + i]);
        }
#pragma unroll
        for (int r = 0; r < E; ++r) {
            const int i = u.t + (r << u.lt);
            if (pf[i >> kPenChunkLog] & 1) {
                const GlobalRows<T> q{f, o};
                if (MODE == FWD_PEN_TAN && m == 1) z[0][r] = cadd(z[0][r], pen_point<T, true>(f, q, i, o));
                else z[0][r] = cadd(z[0][r], pen_point<T, LIN>(f, q, i, o));
                if (!sfd) {
                    f.W[o.a + i] = z[0][r].x;
                    f.W[o.b + i] = z[0][r].y;
                }
            }
        }
        if (sfd) {
#pragma unroll
            for (int r = 0; r < E; ++r) {
                const int i = u.t + (r << u.lt);
                const T ya = f.Y[o.a + i], yb = f.Y[o.b + i];
                const T da = z[0][r].x - ya, db = z[0][r].y - yb;
                f.Y[o.a + i] = ya + f.sfd_k2 * da;
                f.Y[o.b + i] = yb + f.sfd_k2 * db;
                z[0][r] = mk<T>(z[0][r].x - f.sfd_k1 * da, z[0][r].y - f.sfd_k1 * db);
                f.W[o.a + i] = z[0][r].x;
                f.W[o.b + i] = z[0][r].y;
            }
        }
    }
    if (!do_fft) return;
    fft_regs<false, T, LE, 1, RowUnit<T, LE, LN>::kLT>(z, d, S, u.t, u.lt, f.twx[LE], u.sync);
    split_pair<T, LE>(z[0], f.X1 + xs_pair(f, pair, 0), nx, d, u);
}

// FP32 at 8 elements a thread is capped at 64 registers as well (1024-thread
// bounds): four 256-thread blocks an SM instead of two hide the loads of the
// right-hand side (32 fields of 2048x1024: 771 -> 584 us) and of the
// penalisation (274 -> 221 us).
template <class T, int MODE, int LE, int LN = 0>
__global__ void __launch_bounds__((kF32<T> ? MODE == FWD_RHS_TAN && LE >= 2 : LE == 3) ? 512 : 1024)
    k_row_forward(Fields<T> f, int RP, bool sfd, bool do_fft) {
    if (!member_view(f)) return;
    row_forward_body<T, MODE, LE, LN>(f, blockIdx.y, blockIdx.x, RP, sfd, do_fft);
}

// What an inverse row pass transforms: the row pairs of one array after
// another, ny/2 sequences each.
enum InvIO {
    INV_PSI = 0,   // X2 -> P
    INV_WP = 1,    // X1 -> W, X2 -> P
    INV_UV = 2,    // X2 -> U, X3 -> V
    // X1 -> W, X2 -> U, X3 -> V (FP32), two sequences a unit: rows a, b of W each
    // with the same row of U (ny/2 units), then two pairs of V (ny/4).  The
    // rounding error of a transform spreads evenly over its two rows, and the
    // velocity's share of it matters little: with W's rows together the error
    // of W is sqrt(2) times as large (march at 512x256, 100 steps, against 64
    // bits: 7.4e-7 instead of 7.2e-7).
    INV_WUV = 3,
};

// Inverse x-transform of RP row pairs per block, as selected by IO.  sparse:
// the velocity or psi of the intermediate state, which only the penalisation
// reads: stored where one of its stencils reaches (Fields::pf bit 1).
// PART: the last block may have units beyond the last one (wuv_plan); they
// repeat unit 0 up to the stores, so that they meet every barrier.
template <class T, int LE, int LN, bool PART>
__device__ __forceinline__ void row_inverse_wuv(const Fields<T>& f, int bx, int units) {
    using C = Cx<T>;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    constexpr int E = 1 << LE;
    const int nx = LN ? 1 << LN : f.nx, S = padded_len<T>(nx);
    const RowUnit<T, LE, LN> u(f);
    const int np = f.ny >> 1;
    int unit = bx * units + u.q;
    const bool idle = PART && unit >= np + (np >> 1);
    if (idle) unit = 0;
    const bool wu = unit < np;
    const int p0 = wu ? unit : 2 * (unit - np), p1 = wu ? unit : p0 + 1;   // pairs of the two loads
    C* d = reinterpret_cast<C*>(smem_raw) + (size_t)u.q * 2 * S;
    C v[2][E];
    const C* const Xs[2] = {(wu ? f.X1 : f.X3) + xs_pair(f, p0, 0), (wu ? f.X2 : f.X3) + xs_pair(f, p1, 0)};
    merge_pairs<T, LE, 2>(v, Xs, nx, d, S, u, wu);
    fft_regs<true, T, LE, 2, RowUnit<T, LE, LN>::kLT>(v, d, S, u.t, u.lt, f.twx[LE], u.sync);
    if (idle) return;
    // first rows of the two sequences; the second rows are at d1 beyond them
    T* const o0 = (wu ? f.W : f.V) + 2 * p0 * nx;
    T* const o1 = (wu ? f.U + 2 * p0 * nx : f.V + (2 * p0 + 1) * nx);
    const int step = wu ? nx : 2 * nx;
    const unsigned char *f0 = f.pf + ((size_t)p0 << f.logc), *f1 = f.pf + ((size_t)p1 << f.logc);
#pragma unroll
    for (int r = 0; r < E; ++r) {
        const int i = u.t + (r << u.lt);
        const bool n0 = f0[i >> kPenChunkLog] & 2, n1 = f1[i >> kPenChunkLog] & 2;
        if (wu || n0) o0[i] = v[0][r].x;
        if (n0) o1[i] = v[0][r].y;
        if (wu || n1) o0[i + step] = v[1][r].x;
        if (n1) o1[i + step] = v[1][r].y;
    }
}

template <class T, int LE, int IO, int LN = 0, bool PART = false>
__device__ __forceinline__ void row_inverse_body(const Fields<T>& f, int bx, int RP, bool sparse) {
    if constexpr (IO == INV_WUV) {
        row_inverse_wuv<T, LE, LN, PART>(f, bx, RP > 1 ? RP >> 1 : 1);
        return;
    }
    using C = Cx<T>;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    constexpr int E = 1 << LE;
    const int nx = LN ? 1 << LN : f.nx, S = padded_len<T>(nx);
    const RowUnit<T, LE, LN> u(f);
    const int unit = bx * RP + u.q;
    const int m = unit >> (f.logy - 1), pair = unit & ((f.ny >> 1) - 1);
    const C* X;
    T* dst;
    if (IO == INV_PSI) {
        X = f.X2;
        dst = f.P;
    } else if (IO == INV_WP) {
        X = m == 0 ? f.X1 : f.X2;
        dst = m == 0 ? f.W : f.P;
    } else {
        X = m == 0 ? f.X2 : f.X3;
        dst = m == 0 ? f.U : f.V;
    }
    const bool all = !sparse || m == 0;   // W is read everywhere
    C* d = reinterpret_cast<C*>(smem_raw) + (size_t)u.q * S;
    C v[1][E];
    const C* const Xs[1] = {X + xs_pair(f, pair, 0)};
    merge_pairs<T, LE, 1>(v, Xs, nx, d, S, u);
    fft_regs<true, T, LE, 1, RowUnit<T, LE, LN>::kLT>(v, d, S, u.t, u.lt, f.twx[LE], u.sync);
    const int oa = 2 * pair * nx, ob = oa + nx;
    const unsigned char* pf = f.pf + ((size_t)pair << f.logc);
#pragma unroll
    for (int r = 0; r < E; ++r) {
        const int i = u.t + (r << u.lt);
        if (all || (pf[i >> kPenChunkLog] & 2)) {
            dst[oa + i] = v[0][r].x;
            dst[ob + i] = v[0][r].y;
        }
    }
}

template <class T, int LE, int IO, int LN = 0>
__global__ void NS_FFT_BOUNDS k_row_inverse(Fields<T> f, int RP, bool sparse) {
    if (!member_view(f)) return;
    row_inverse_body<T, LE, IO, LN>(f, blockIdx.x, RP, sparse);
}

// A forward row pass together with the inverse pass before it, one row pair p
// per block: group g of tps threads transforms one sequence,
//   RHS (psi steppers)  psi of pairs p - 1, p, p + 1
//   PEN                 psi* of pairs p - 1, p, p + 1, omega* of pair p; FP32:
//                       u* of pairs p - 1, p + 1, v* of p, and rows a, b of
//                       omega* each with the same row of u* (see INV_WUV),
// into shared memory, all threads share the pointwise part, and group 0
// transforms the result.  The neighbours' transforms are made three times over
// the grid, so it is for grids that leave most of the chip idle, where a
// kernel costs its fixed 3-4 us and a chain of dependent instructions whatever
// its work: two kernels a step less and the pointwise chain spread over 3 to
// 5 times the threads.  us a step at 128x64: FP64 38.0 -> 33.6, double-float
// 28.6 -> 22.8, FP32 20.3 -> 17.5.
template <class T, int MODE> struct RowChain {
    static constexpr bool RHS = (MODE == FWD_RHS_NL || MODE == FWD_RHS_LIN);
    static constexpr bool LIN = (MODE == FWD_RHS_LIN || MODE == FWD_PEN_LIN);
    static constexpr int kGroups = RHS ? 3 : kF32<T> ? 5 : 4;
};

template <class T, int MODE, int LE>
__global__ void __launch_bounds__(1024) k_row_chain(Fields<T> f, bool sfd, bool do_fft) {
    using C = Cx<T>;
    using K = RowChain<T, MODE>;
    if (!member_view(f)) return;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    constexpr int E = 1 << LE, G = K::kGroups;
    const int nx = f.nx, S = padded_len<T>(nx), pair = blockIdx.x;
    RowUnit<T, LE> u(f);
    u.sync.count = u.tps;   // barriers of a group
    u.sync.id = 1 + u.q;
    C* const tiles = reinterpret_cast<C*>(smem_raw);
    C* const d = tiles + u.q * S;
    const RowOffs o(pair, nx, f.ny);
    if (K::RHS) prefetch_rows<T, K::LIN>(f, pair, threadIdx.x, blockDim.x);
    {
        C v[1][E];
        if (!K::RHS && kF32<T> && (u.q == 1 || u.q == 4)) {   // row a (u.q = 1) or b of omega* and u*
            const size_t x0 = xs_pair(f, pair, 0) + (u.q == 4);
            merge_rows<T, LE>(v[0], f.X1 + x0, f.X2 + x0, nx, d, u);
        } else {
            const C* X = u.q < 3 ? f.X2 : kF32<T> ? f.X3 : f.X1;
            const int pr = u.q < 3 ? (pair - 1 + u.q) & ((f.ny >> 1) - 1) : pair;
            const C* const Xs[1] = {X + xs_pair(f, pr, 0)};
            merge_pairs<T, LE, 1>(v, Xs, nx, d, S, u);
        }
        fft_regs<true, T, LE, 1>(v, d, S, u.t, u.lt, f.twx[LE], u.sync);
#pragma unroll
        for (int r = 0; r < E; ++r) d[sw<T>(u.t + (r << u.lt))] = v[0][r];
    }
    __syncthreads();
    const TileRows<T> q{tiles, S};
    C* const out = tiles + G * S;
    const unsigned char* pf = f.pf + ((size_t)pair << f.logc);
    for (int i = threadIdx.x; i < nx; i += blockDim.x) {
        C z;
        if constexpr (K::RHS) {
            T ua, ub, va, vb;
            psi_diffs<T>(q, i, nx, ua, ub, va, vb);
            z = rhs_point<T, K::LIN>(f, i, o, ua, ub, va, vb);
        } else {
            z = tiles[(kF32<T> ? 1 : G - 1) * S + sw<T>(i)];   // omega*
            if (kF32<T>) z = mk<T>(z.x, tiles[4 * S + sw<T>(i)].x);
            if (pf[i >> kPenChunkLog] & 1) {
                if (MODE == FWD_PEN_TAN && blockIdx.y == 1) z = cadd(z, pen_point<T, true>(f, q, i, o));
                else z = cadd(z, pen_point<T, K::LIN>(f, q, i, o));
            }
            if (sfd) {
                const T ya = f.Y[o.a + i], yb = f.Y[o.b + i];
                const T da = z.x - ya, db = z.y - yb;
                f.Y[o.a + i] = ya + f.sfd_k2 * da;
                f.Y[o.b + i] = yb + f.sfd_k2 * db;
                z = mk<T>(z.x - f.sfd_k1 * da, z.y - f.sfd_k1 * db);
            }
            f.W[o.a + i] = z.x;
            f.W[o.b + i] = z.y;
        }
        out[sw<T>(i)] = z;
    }
    __syncthreads();
    if (!do_fft || u.q != 0) return;
    C z[1][E];
#pragma unroll
    for (int r = 0; r < E; ++r) z[0][r] = out[sw<T>(u.t + (r << u.lt))];
    fft_regs<false, T, LE, 1>(z, d, S, u.t, u.lt, f.twx[LE], u.sync);
    split_pair<T, LE>(z[0], f.X1 + xs_pair(f, pair, 0), nx, d, u);
}

// ----------------------------------------------------------- column kernels

// A column pass handles CP neighbouring packed columns per block.  Thread t
// of a column holds y = t + r ny/E; 16 threads of a column, then 16 of the
// next one: shared-memory phases stay within a column, and the warp's
// accesses to the x-spectra fill runs of CP x 4 elements (kXRows).
template <class T, int LE, int LN = 0> struct ColUnit {
    static constexpr int kLT = LN ? LN - LE : -1;
    int c, t, lt;
    __device__ __forceinline__ ColUnit(const Fields<T>& f, int CP) {
        lt = LN ? LN - LE : f.logy - LE;
        const int lo = lt < 4 ? lt : 4, lc = 31 - __clz(CP);
        c = (threadIdx.x >> lo) & (CP - 1);
        t = (threadIdx.x & ((1 << lo) - 1)) | ((threadIdx.x >> (lo + lc)) << lo);
    }
};

// element index of (kx, y) in an x-spectrum
template <class T> __device__ __forceinline__ size_t xs_at(const Fields<T>& f, int kx, int y) {
    return ((size_t)(y / kXRows) * f.nxh + kx) * kXRows + (y & (kXRows - 1));
}

// Packed kx = 0 column: Z = FFT_y(X0 + i XN).  Applying real operators f0 to
// the kx = 0 part and fN to the kx = nx/2 part gives
//   Z'(ky) = (f0 + fN)/2 Z(ky) + (f0 - fN)/2 conj(Z(-ky)).
// The operator tables hold the half sum s in row 0 and the half difference d
// in row nx/2, which no other column reads.
template <class C, class T>
__device__ __forceinline__ C apply_packed0(C z, C zm, T s, T d) {
    return mk<T>(s * z.x + d * zm.x, s * z.y - d * zm.y);
}

// A thread takes the modes ky = k and -k of the packed column together, k = 0
// .. ny/2.  FP64: the two modes that mirror themselves, 0 and ny/2, are one
// pair too, so that at 2 elements a thread there is one pair per thread and
// no second round for thread 0.  Every round is a chain of FP64 instructions in
// the one block all others wait for: with half sums formed on the device and
// the extra round the FP64 step took 40.8 us at 128x64, with the tables alone
// 39.8, with both 38.3 (512x256: 62.7, 61.7, 60.9).  FP32 and double-float lose
// more by the registers this takes than by the round (Jacobian product at
// 512x256 FP32 26.7 -> 27.4 us a step).
template <class T> struct PackedPair {
    static constexpr bool kSelf = std::is_same<T, double>::value;
    int k, km;
    bool self;   // both modes mirror themselves
    __device__ __forceinline__ PackedPair(int k_, int ny) : k(k_) {
        self = kSelf && k == 0;
        km = self ? ny >> 1 : (ny - k) & (ny - 1);
    }
    __device__ static __forceinline__ bool more(int k, int ny) { return kSelf ? 2 * k < ny : 2 * k <= ny; }
};

template <class T, int LE> struct ColArrays {
    // sequences a thread of col_update_body carries through the inverse transforms
    static constexpr int kUpdate = kF32<T> ? 3 : 2;
};

// Forward y-transform of CP columns of X1, store Wh, psi^ = scale * tP * omega^,
// inverse y-transform into X2.  VEL: inverse y-transforms of
// u'^ = i sy psi^ into X2 and v^ = -i sx psi^ into X3 instead, with
// sy = sin(2 pi ky/ny)/dy, sx = sin(2 pi kx/nx)/dx, the symbols of the
// centred differences (zero at kx = 0 and kx = nx/2, so the packed column of
// v is zero; sy is odd in ky and acts alike on both halves of the packed
// column).
template <class T, int LE, bool VEL, int LN = 0>
__device__ __forceinline__ void col_poisson_body(const Fields<T>& f, int bx, int CP, T scale) {
    using C = Cx<T>;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    constexpr int E = 1 << LE, M = VEL ? 2 : 1;
    const int ny = LN ? 1 << LN : f.ny, S = padded_len<T>(ny);
    const ColUnit<T, LE, LN> u(f, CP);
    const int kx = bx * CP + u.c;
    C* d = reinterpret_cast<C*>(smem_raw) + (size_t)u.c * M * S;
    const SeqSync sync{false, 0, 0};
    C z[1][E];
#pragma unroll
    for (int r = 0; r < E; ++r) z[0][r] = f.X1[xs_at(f, kx, u.t + (r << u.lt))];
    fft_regs<false, T, LE, 1, ColUnit<T, LE, LN>::kLT>(z, d, S, u.t, u.lt, f.twy[LE], sync);
    const size_t g0 = (size_t)kx * ny + u.t;
#pragma unroll
    for (int r = 0; r < E; ++r) f.Wh[g0 + (r << u.lt)] = z[0][r];
    C v[M][E];
    if (bx == 0) {   // the block that holds the packed column: modes ky and -ky of it by one thread
#pragma unroll
        for (int r = 0; r < E; ++r) d[sw<T>(u.t + (r << u.lt))] = z[0][r];
        __syncthreads();
        if (kx == 0) {
#pragma unroll 1
            for (int k = u.t; PackedPair<T>::more(k, ny); k += 1 << u.lt) {
                const PackedPair<T> q(k, ny);
                const T s0 = scale * SpecOp<T>::p(f, 0, k), d0 = scale * SpecOp<T>::p(f, f.nxh, k);
                T s1 = s0, d1 = d0;   // even in ky
                if (q.self) {
                    s1 = scale * SpecOp<T>::p(f, 0, q.km);
                    d1 = scale * SpecOp<T>::p(f, f.nxh, q.km);
                }
                const C zk = d[sw<T>(k)], zm = d[sw<T>(q.km)];
                C pk = apply_packed0(zk, q.self ? zk : zm, s0, d0), pm = apply_packed0(zm, q.self ? zm : zk, s1, d1);
                if (VEL) {
                    pk = cscale(cmul_pi(pk), f.tDy[k]);
                    pm = cscale(cmul_pi(pm), f.tDy[q.km]);
                }
                d[sw<T>(k)] = pk;
                if (q.km != k) d[sw<T>(q.km)] = pm;
            }
        }
        __syncthreads();
#pragma unroll
        for (int r = 0; r < E; ++r) {
            v[0][r] = d[sw<T>(u.t + (r << u.lt))];
            if (VEL) v[M - 1][r] = mk<T>(T(0), T(0));
        }
        __syncthreads();
    }
    if (kx != 0) {
        const T dx = VEL ? f.tDx[kx] : T(0);
#pragma unroll
        for (int r = 0; r < E; ++r) {
            const int k = u.t + (r << u.lt);
            const C ps = cscale(z[0][r], scale * SpecOp<T>::p(f, kx, k));
            if (VEL) {
                v[0][r] = cscale(cmul_pi(ps), f.tDy[k]);
                v[M - 1][r] = cscale(cmul_mi(ps), dx);
            } else {
                v[0][r] = ps;
            }
        }
    }
    fft_regs<true, T, LE, M, ColUnit<T, LE, LN>::kLT>(v, d, S, u.t, u.lt, f.twy[LE], sync);
#pragma unroll
    for (int r = 0; r < E; ++r) {
        const size_t g = xs_at(f, kx, u.t + (r << u.lt));
        f.X2[g] = v[0][r];
        if (VEL) f.X3[g] = v[M - 1][r];
    }
}

template <class T, int LE, bool VEL, int LN = 0>
__global__ void NS_FFT_BOUNDS k_col_poisson(Fields<T> f, int CP, T scale) {
    if (!member_view(f)) return;
    col_poisson_body<T, LE, VEL, LN>(f, blockIdx.x, CP, scale);
}

// Forward y-transform of N (x-spectra in XN: X1, or X4 after the fused FP32
// row pass); AB2/AB1 + Crank-Nicolson update
//   omega*^ = tA omega^ + tB (c1 N^n + c0 N^{n-1}),  psi*^ = tP omega*^
// (tA, tB carry the 1/(2 nx ny) of the inverse transform); Nh <- N^n; inverse
// y-transforms of omega*^ -> X1 and psi*^ -> X2 (FP32: u*'^ -> X2 and
// v*^ -> X3, as in k_col_poisson).
template <class T, int LE, int LN = 0>
__device__ __forceinline__ void col_update_body(const Fields<T>& f, int bx, int CP, T c1, T c0, bool first) {
    using C = Cx<T>;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    constexpr int E = 1 << LE, M = ColArrays<T, LE>::kUpdate;
    const int ny = LN ? 1 << LN : f.ny, S = padded_len<T>(ny);
    const ColUnit<T, LE, LN> u(f, CP);
    const int kx = bx * CP + u.c;
    C* d = reinterpret_cast<C*>(smem_raw) + (size_t)u.c * M * S;
    const SeqSync sync{false, 0, 0};
    const size_t g0 = (size_t)kx * ny + u.t;
    C n[1][E], w[E], nh[E], v[M][E];
#pragma unroll
    for (int r = 0; r < E; ++r) n[0][r] = f.XN[xs_at(f, kx, u.t + (r << u.lt))];
#pragma unroll
    for (int r = 0; r < E; ++r) {
        w[r] = f.Wh[g0 + (r << u.lt)];
        if (!first) nh[r] = f.Nh[g0 + (r << u.lt)];
    }
    fft_regs<false, T, LE, 1, ColUnit<T, LE, LN>::kLT>(n, d, S, u.t, u.lt, f.twy[LE], sync);
    // N^n to memory, n <- the right-hand side c1 N^n + c0 N^{n-1}
#pragma unroll
    for (int r = 0; r < E; ++r) {
        f.Nh[g0 + (r << u.lt)] = n[0][r];
        n[0][r] = cscale(n[0][r], c1);
        if (!first) n[0][r] = cadd(n[0][r], cscale(nh[r], c0));
    }
    if (bx == 0) {   // the block that holds the packed column: modes ky and -ky of it by one thread
#pragma unroll
        for (int r = 0; r < E; ++r) {
            d[sw<T>(u.t + (r << u.lt))] = w[r];
            d[S + sw<T>(u.t + (r << u.lt))] = n[0][r];
        }
        __syncthreads();
        if (kx == 0) {
#pragma unroll 1
            for (int k = u.t; PackedPair<T>::more(k, ny); k += 1 << u.lt) {
                const PackedPair<T> q(k, ny);
                T As, Bs, Ad, Bd;   // half sums and differences, even in ky
                SpecOp<T>::ab(f, 0, k, As, Bs);
                SpecOp<T>::ab(f, f.nxh, k, Ad, Bd);
                const T Ps = SpecOp<T>::p(f, 0, k), Pd = SpecOp<T>::p(f, f.nxh, k);
                T As1 = As, Bs1 = Bs, Ad1 = Ad, Bd1 = Bd, Ps1 = Ps, Pd1 = Pd;
                if (q.self) {
                    SpecOp<T>::ab(f, 0, q.km, As1, Bs1);
                    SpecOp<T>::ab(f, f.nxh, q.km, Ad1, Bd1);
                    Ps1 = SpecOp<T>::p(f, 0, q.km);
                    Pd1 = SpecOp<T>::p(f, f.nxh, q.km);
                }
                const C wk = d[sw<T>(k)], wm = d[sw<T>(q.km)], nk = d[S + sw<T>(k)], nm = d[S + sw<T>(q.km)];
                C wsk = cadd(apply_packed0(wk, q.self ? wk : wm, As, Ad), apply_packed0(nk, q.self ? nk : nm, Bs, Bd));
                C wsm = cadd(apply_packed0(wm, q.self ? wm : wk, As1, Ad1), apply_packed0(nm, q.self ? nm : nk, Bs1, Bd1));
                if constexpr (kF32<T>) {   // plus scale * omega^ (tA holds scale (A - 1))
                    wsk = mk<T>(__fmaf_rn(wk.x, f.scale, wsk.x), __fmaf_rn(wk.y, f.scale, wsk.y));
                    wsm = mk<T>(__fmaf_rn(wm.x, f.scale, wsm.x), __fmaf_rn(wm.y, f.scale, wsm.y));
                }
                C pk = apply_packed0(wsk, q.self ? wsk : wsm, Ps, Pd), pm = apply_packed0(wsm, q.self ? wsm : wsk, Ps1, Pd1);
                if (kF32<T>) {
                    pk = cscale(cmul_pi(pk), f.tDy[k]);
                    pm = cscale(cmul_pi(pm), f.tDy[q.km]);
                }
                d[sw<T>(k)] = wsk;
                d[sw<T>(q.km)] = wsm;
                d[S + sw<T>(k)] = pk;
                d[S + sw<T>(q.km)] = pm;
            }
        }
        __syncthreads();
#pragma unroll
        for (int r = 0; r < E; ++r) {
            v[0][r] = d[sw<T>(u.t + (r << u.lt))];
            v[1][r] = d[S + sw<T>(u.t + (r << u.lt))];
            if (kF32<T>) v[M - 1][r] = mk<T>(T(0), T(0));
        }
        __syncthreads();
    }
    if (kx != 0) {
        const T dx = kF32<T> ? f.tDx[kx] : T(0);
#pragma unroll
        for (int r = 0; r < E; ++r) {
            const int k = u.t + (r << u.lt);
            T A, B;
            SpecOp<T>::ab(f, kx, k, A, B);
            C ws;
            if constexpr (kF32<T>) {   // tA = scale (A - 1): the small terms first, one rounding at the end
                const C t = cadd(cscale(w[r], A), cscale(n[0][r], B));
                ws = mk<T>(__fmaf_rn(w[r].x, f.scale, t.x), __fmaf_rn(w[r].y, f.scale, t.y));
            } else {
                ws = cadd(cscale(w[r], A), cscale(n[0][r], B));
            }
            v[0][r] = ws;
            const C ps = cscale(ws, SpecOp<T>::p(f, kx, k));
            if (kF32<T>) {
                v[1][r] = cscale(cmul_pi(ps), f.tDy[k]);
                v[M - 1][r] = cscale(cmul_mi(ps), dx);
            } else {
                v[1][r] = ps;
            }
        }
    }
    fft_regs<true, T, LE, M, ColUnit<T, LE, LN>::kLT>(v, d, S, u.t, u.lt, f.twy[LE], sync);
#pragma unroll
    for (int r = 0; r < E; ++r) {
        const size_t g = xs_at(f, kx, u.t + (r << u.lt));
        f.X1[g] = v[0][r];
        f.X2[g] = v[1][r];
        if (kF32<T>) f.X3[g] = v[M - 1][r];
    }
}

template <class T, int LE, int LN = 0>
__global__ void NS_FFT_BOUNDS k_col_update(Fields<T> f, int CP, T c1, T c0, bool first) {
    if (!member_view(f)) return;
    col_update_body<T, LE, LN>(f, blockIdx.x, CP, c1, c0, first);
}

// ------------------------------------------------------- pointwise kernels

// Base-derived fields of parameter set blockIdx.y, from Omega_b and Psi_b
// (FP32: the base velocity) held in member slot blockIdx.y of W and P (U, V),
// with the signs and the 1/(2 dx), 1/(2 dy) of N' = -(U_b D_x w + V_b D_y w +
// u' D_x Om_b + v' D_y Om_b) folded in: the linearised pass multiplies them
// with undivided differences (of w and psi; FP32: of w, and with u', v').
template <class T>
__global__ void k_base_fields(Fields<T> f, T* Ub, T* Vb, T* DxOb, T* DyOb) {
    const size_t n = (size_t)f.nx * f.ny;
    const size_t off = (size_t)blockIdx.y * f.fs;
    const T* P = f.P + off;   // Psi_b
    const T* W = f.W + off;   // Omega_b
    for (size_t c = blockIdx.x * (size_t)blockDim.x + threadIdx.x; c < n; c += (size_t)gridDim.x * blockDim.x) {
        const int i = (int)(c & (f.nx - 1));
        const int j = (int)(c >> f.logx);
        const int ip = (i + 1) & (f.nx - 1), im = (i - 1) & (f.nx - 1);
        const int jp = (j + 1) & (f.ny - 1), jm = (j - 1) & (f.ny - 1);
        T ub, vb;
        if (kF32<T>) {   // u', v of the base in U, V
            ub = f.Uinf + f.U[off + c];
            vb = f.V[off + c];
        } else {
            ub = f.Uinf + (P[(size_t)jp * f.nx + i] - P[(size_t)jm * f.nx + i]) * f.idy2;
            vb = -((P[(size_t)j * f.nx + ip] - P[(size_t)j * f.nx + im]) * f.idx2);
        }
        const T ox = (W[(size_t)j * f.nx + ip] - W[(size_t)j * f.nx + im]) * f.idx2;
        const T oy = (W[(size_t)jp * f.nx + i] - W[(size_t)jm * f.nx + i]) * f.idy2;
        Ub[off + c] = -(ub * f.idx2);
        Vb[off + c] = -(vb * f.idy2);
        DxOb[off + c] = kF32<T> ? -ox : -(ox * f.idy2);   // times u', or the y difference of psi'
        DyOb[off + c] = kF32<T> ? -oy : oy * f.idx2;      // times v', or the x difference (v' = -D_x psi')
    }
}

// dst[m] <- src[m] (FP64 -> T) for the members with a non-null source
template <class T>
__global__ void k_gather(const double* const* __restrict__ src, T* __restrict__ dst, size_t n, size_t fs) {
    const double* s = src[blockIdx.y];
    if (!s) return;
    T* d = dst + (size_t)blockIdx.y * fs;
    for (size_t c = blockIdx.x * (size_t)blockDim.x + threadIdx.x; c < n; c += (size_t)gridDim.x * blockDim.x)
        d[c] = (T)s[c];
}

// dst[m] <- src[m] (T -> FP64) for the members with a non-null destination
template <class T>
__global__ void k_scatter(const T* __restrict__ src, double* const* __restrict__ dst, size_t n, size_t fs) {
    double* d = dst[blockIdx.y];
    if (!d) return;
    const T* s = src + (size_t)blockIdx.y * fs;
    for (size_t c = blockIdx.x * (size_t)blockDim.x + threadIdx.x; c < n; c += (size_t)gridDim.x * blockDim.x)
        d[c] = (double)s[c];
}

// partial[m][b] = sum over block b's share of (a - b)^2 of member m, in FP64
template <class T>
__global__ void k_diff_sumsq(const T* __restrict__ a, const T* __restrict__ b, size_t n, size_t fs, double* partial) {
    a += (size_t)blockIdx.y * fs;
    b += (size_t)blockIdx.y * fs;
    partial += (size_t)blockIdx.y * gridDim.x;
    double acc = 0.0;
    for (size_t c = blockIdx.x * (size_t)blockDim.x + threadIdx.x; c < n; c += (size_t)gridDim.x * blockDim.x) {
        const double d = (double)a[c] - (double)b[c];
        acc += d * d;
    }
    for (int o = 16; o > 0; o >>= 1) acc += __shfl_down_sync(0xffffffffu, acc, o);
    __shared__ double red[32];
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = acc;
    __syncthreads();
    if (threadIdx.x < 32) {
        acc = (threadIdx.x < (blockDim.x >> 5)) ? red[threadIdx.x] : 0.0;
        for (int o = 16; o > 0; o >>= 1) acc += __shfl_down_sync(0xffffffffu, acc, o);
        if (threadIdx.x == 0) partial[blockIdx.x] = acc;
    }
}

}  // namespace nsstab

#include "rowroll.cuh"   // fused FP32 row passes (uses Fields, row modes and the FFT above)

namespace nsstab {

// ------------------------------------------------------------- host side

// One launch configuration: `per` sequences (row pairs or columns) per
// block, 2^le elements per thread in the FFT passes; grid.y = members.
struct Launch {
    int blocks = 0, threads = 0, per = 0, le = 3;
    size_t smem = 0;
    bool ok = false;
};

// the six kernels of a step, in order
enum KernelId { KCOLP = 0, KINVP = 1, KFWDR = 2, KCOLU = 3, KINVR = 4, KFWDP = 5 };
template <class T> int max_threads_for(int kid, int le);

static const int kRedBlocks = 64;           // partial sums per member
static const int kPtBlocks = 152;           // grid.x of the pointwise kernels
static const double kPi = 3.14159265358979323846;
static const int kGraphChunk = 256;         // time steps per captured graph
static const size_t kMaxSmem = 200 * 1024;

#define K_FWD_PLAIN(le) k_row_forward<T, FWD_PLAIN, le>
#define K_FWD_RNL(le) k_row_forward<T, FWD_RHS_NL, le>
#define K_FWD_RLIN(le) k_row_forward<T, FWD_RHS_LIN, le>
#define K_FWD_PNL(le) k_row_forward<T, FWD_PEN_NL, le>
#define K_FWD_PLIN(le) k_row_forward<T, FWD_PEN_LIN, le>
#define K_FWD_RTAN(le) k_row_forward<T, FWD_RHS_TAN, le>
#define K_FWD_PTAN(le) k_row_forward<T, FWD_PEN_TAN, le>
#define K_INVP(le) k_row_inverse<T, le, (kF32<T> ? INV_UV : INV_PSI)>
#define K_INVR(le) k_row_inverse<T, le, (kF32<T> ? INV_WUV : INV_WP)>
#define K_INVPSI(le) k_row_inverse<T, le, INV_PSI>
#define K_COLP(le) k_col_poisson<T, le, kF32<T>>
#define K_COLPSI(le) k_col_poisson<T, le, false>
#define K_COLU(le) k_col_update<T, le>

// FP32 passes at 8 elements a thread whose transform length is a constant of
// the kernel: call(std::integral_constant<int, log2 N>) for the lengths in
// [lo, lo + 2], else false.  Their instructions are a quarter addressing with
// the length at run time; 32 fields of 2048x1024, us a launch: column Poisson
// pass 400 -> 359, column update 579 -> 490, inverse rows 411 -> 375,
// penalisation 221 -> 195.  (The right-hand side keeps the run-time form: four
// pairs of sequences unrolled spill at its 64 registers, 613 -> 762.  FP64 and
// double-float are bound by their arithmetic.)  The lengths outside the two
// windows do without so far, at a price: 4096-point rows and 2048-, 4096-point
// columns (one field of 4096x2048 399 us a step, 334 with constants; of
// 4096x1024 188 and 169; of 2048x4096 365 and 333), 256-point rows and
// 128-point columns of a batch (64 fields of 256x128 66.0 and 58.7; of 128x128
// 43.0 and 41.5).
template <class F> bool with_length(int ln, int lo, F call) {
    switch (ln - lo) {
        case 0: call(std::integral_constant<int, 0>()); return true;
        case 1: call(std::integral_constant<int, 1>()); return true;
        case 2: call(std::integral_constant<int, 2>()); return true;
        default: return false;
    }
}
constexpr int kRowLo = 9, kColLo = 8;   // rows of 512 .. 2048 points, columns of 256 .. 1024

class RaggedF32;

template <class T>
class StepperImpl : public StepperBase {
    friend class RaggedF32;   // drives float steppers' data through the ragged launches

  public:
    using C = Cx<T>;
    StepperImpl(const nsstab_config& cfg, int nsets, const double* Re, const double* D, int per_set,
                cudaStream_t s)
        : cfg_(cfg), stream_(s), S_(nsets), bper_(per_set), B_(nsets * per_set) {
        for (int k = 0; k < nsets; ++k) {
            Re_.push_back(Re ? Re[k] : cfg.Re);
            D_.push_back(D ? D[k] : cfg.cyl_D);
        }
    }
    ~StepperImpl() override { release(); }

    int init() override;
    int members() const override { return B_; }
    int sets() const override { return S_; }
    int poisson(const double* omega, double* psi) override;
    int step_nonlinear(double* omega, int nsteps) override;
    int set_base(const double* base_omega) override;
    int set_base_ptrs(const double* const* base_omegas) override;
    int step_linear(const double* v_in, double* v_out, int nsteps) override;
    int step_linear_ptrs(const double* const* in, double* const* out, int nsteps) override;
    int tangent(const double* q, const double* v_in, double* v_out, int nsteps) override;
    int residual(const double* q, double* r) override;
    int sfd(double* omega, double chi, double Delta, double tol, long max_steps, int check_every,
            double* r, long* steps) override;
    int launches_per_step() const override {
        if (rollR_) return 4;
        return (kF32<T> ? 5 : kNumStepKernels) - (chain_threads(KFWDR) > 0) - (chain_threads(KFWDP) > 0);
    }
    int profile_linear(const double* v, int nsteps, double* ms) override;
    int autotune(int reps, int* chosen) override;
    int plan_of(int kid, int* le, int* per) const override {
        if (kid < 0 || kid >= kNumStepKernels) return NSSTAB_ERR_INVALID_ARG;
        *le = plan_[kid].le;
        *per = plan_[kid].per;
        return NSSTAB_OK;
    }
    int set_plan(int kid, int le, int per) override;
    int set_fused_rows(int R) override;
    int fused_rows() const override { return rollR_; }

  private:
    nsstab_config cfg_;
    cudaStream_t stream_;
    int S_, bper_, B_;
    std::vector<double> Re_, D_;
    cudaStream_t cap_ = nullptr;   // private stream used only to capture graphs
    Fields<T> f_{};
    int nx_ = 0, ny_ = 0, nxh_ = 0;
    size_t n_ = 0, nc_ = 0;
    std::vector<void*> allocs_;
    T* Wsave_ = nullptr;
    C* Nhsave_ = nullptr;
    double* red_ = nullptr;          // device partials [B][kRedBlocks]
    double* red_host_ = nullptr;     // pinned
    unsigned char* active_ = nullptr;
    bool xn_x4_ = false;                           // k_col_update reads N from X4 (fused row passes)
    std::vector<unsigned char> active_host_;
    const double** ptr_in_ = nullptr;   // device arrays of B member pointers
    double** ptr_out_ = nullptr;
    std::vector<const double*> pin_host_;
    std::vector<double*> pout_host_;
    bool have_base_ = false;
    Launch plan_[kNumStepKernels];
    int rollR_ = 0;                // fused FP32 row passes over strips of rollR_ rows (0: off)
    RollShape rs_{};
    struct GraphKey {
        int nsteps, flags;
        bool operator<(const GraphKey& o) const { return nsteps != o.nsteps ? nsteps < o.nsteps : flags < o.flags; }
    };
    std::map<GraphKey, cudaGraphExec_t> graphs_;

    template <class P> int dalloc(P** p, size_t count) {
        void* q = nullptr;
        cudaError_t e = cudaMalloc(&q, count * sizeof(P));
        if (e != cudaSuccess) {
            set_error(std::string("cudaMalloc: ") + cudaGetErrorString(e));
            return e == cudaErrorMemoryAllocation ? NSSTAB_ERR_OUT_OF_MEMORY : NSSTAB_ERR_CUDA;
        }
        allocs_.push_back(q);
        *p = static_cast<P*>(q);
        return NSSTAB_OK;
    }
    void clear_graphs() {
        for (auto& kv : graphs_) cudaGraphExecDestroy(kv.second);
        graphs_.clear();
    }
    void release() {
        cudaStreamSynchronize(stream_);
        clear_graphs();
        if (cap_) cudaStreamDestroy(cap_);
        cap_ = nullptr;
        for (void* p : allocs_) cudaFree(p);
        allocs_.clear();
        if (red_host_) cudaFreeHost(red_host_);
        red_host_ = nullptr;
    }
    int build_tables();
    Launch make_plan(int kid, int le, int per) const;
    Launch wuv_plan(int le, int units) const;
    Launch default_plan(int kid) const;
    int set_smem_attr(int kid, const Launch& L);

    int set_active(const std::vector<unsigned char>& a);
    int all_active() { return set_active(std::vector<unsigned char>(B_, 1)); }
    int gather(const double* const* src);                // W[m] <- src[m] (null: skip)
    int scatter(const T* from, double* const* dst);      // dst[m] <- from[m] (null: skip)
    int gather_contig(const double* src, int count);     // members 0..count-1 from [count][n]
    int scatter_contig(const T* from, double* dst);      // all members to [B][n]
    int launch(int kid, cudaStream_t st, bool linear, bool sfd, bool do_fft, bool first);
    bool launch_fixed(int kid, cudaStream_t st, bool linear, bool sfd, bool do_fft, bool first);
    int launch_tangent_row(int kid, cudaStream_t st, bool do_fft);
    int chain_threads(int kid, int le) const;
    int chain_threads(int kid) const { return chain_threads(kid, plan_[kid].le); }
    int launch_chain(int kid, cudaStream_t st, bool linear, bool sfd, bool do_fft, bool tangent);
    int launch_roll(bool pen, cudaStream_t st, bool linear, bool sfd, bool do_fft, bool write_w);
    RollShape roll_shape(int R) const;
    int launch_plain(cudaStream_t st);
    int transform_W();                                   // X1 = x-spectrum of W
    int stream_function(cudaStream_t st);                // Wh, X2 (X3), P (U, V) from X1
    int psi_function(cudaStream_t st);                   // Wh, X2, P from X1
    int issue_steps(cudaStream_t st, int nsteps, bool linear, bool sfd, bool first_ab1, bool fft_last,
                    bool tangent = false);
    int run_steps(int nsteps, bool linear, bool sfd, bool fft_last, bool first_ab1 = true, bool tangent = false);
    int alloc_base_fields();
    int sumsq_diff(const T* a, const T* b, double* out);   // out[B]
    bool may_chain(int kid) const;
    int time_kernel(int kid, const Launch& L, int reps, float* ms);
};

// ---------------------------------------------------------- launch plans

// Sequences per member of launch kid: row pairs (of every array the pass
// transforms, see InvIO) for the row passes, columns for the column passes.
template <class T> static int seq_count(int kid, int nx, int ny) {
    switch (kid) {
        case KCOLP:
        case KCOLU: return nx / 2;
        case KINVP: return kF32<T> ? ny : ny / 2;
        case KINVR: return kF32<T> ? ny + ny / 2 : ny;
        default: return ny / 2;
    }
}

template <class T> Launch StepperImpl<T>::make_plan(int kid, int le, int per) const {
    Launch L;
    const bool row = (kid == KINVP || kid == KFWDR || kid == KINVR || kid == KFWDP);
    const int N = row ? nx_ : ny_;
    const int logN = row ? ilog2(nx_) : ilog2(ny_);
    const int count = seq_count<T>(kid, nx_, ny_);
    // sequences a thread transforms side by side, each with its shared memory
    const int nseq = (kid == KCOLU) ? (kF32<T> ? 3 : 2) : ((kid == KCOLP || kid == KFWDR) && kF32<T>) ? 2 : 1;
    if (le < 1 || le > 3 || logN < le || per < 1 || !is_pow2(per) || per > count) return L;
    const int threads = per * (N >> le);
    const size_t smem = (size_t)per * nseq * padded_len<T>(N) * sizeof(C);
    if (threads > (le == 3 ? 512 : 1024) || smem > kMaxSmem) return L;
    L.per = per;
    L.le = le;
    // count / per blocks; three arrays' pairs need not divide evenly
    L.blocks = count / per;
    L.threads = threads;
    L.smem = smem;
    L.ok = count % per == 0;
    if (kid == KINVR && kF32<T>) {
        const int units = std::max(1, per / 2);
        const bool whole = L.ok && (count / 2) % units == 0;
        L = wuv_plan(le, units);
        L.per = per;
        L.ok = L.ok && whole;
    }
    return L;
}

// KINVR of an FP32 stepper: blocks of `units` units of two sequences each
// (INV_WUV), 3 ny / 4 units in all.  The last block may be partly empty (the
// PART form of row_inverse_wuv).
template <class T> Launch StepperImpl<T>::wuv_plan(int le, int units) const {
    Launch L;
    const int total = ny_ / 2 + ny_ / 4;
    L.per = 2 * units;
    L.le = le;
    L.blocks = (total + units - 1) / units;
    L.threads = units * (nx_ >> le);
    L.smem = (size_t)units * 2 * padded_len<T>(nx_) * sizeof(C);
    L.ok = L.threads <= (le == 3 ? 512 : 1024) && L.smem <= kMaxSmem;
    return L;
}

// Default: the largest elements-per-thread (fewest exchanges) that still
// gives every SM sub-partition a warp over the whole batch, down to 2 but
// with a sequence within one block (4096 points take 4), then enough
// sequences per block for at least two warps.  Below one warp per
// sub-partition the pass is a serial chain of FP64 instructions, 64 cycles
// each per warp, and halving the elements halves the chain at about the same
// instruction count (radix-2 passes 23, radix-4 22 per element at N = 256):
// FP64 step at 128x64 58 -> 40 us, at 512x256 71 -> 63 us with 2 elements
// instead of 4; at 2048x1024 8 elements are best (749 us against 784).  FP32
// stays at 4 or more: every radix-2 level twiddles, which is one rounding more
// (error of 50 steps at 128x64 against 64 bits 9.9e-7 with 2, 9.2e-7 with 4).
template <class T> Launch StepperImpl<T>::default_plan(int kid) const {
    const bool row = (kid == KINVP || kid == KFWDR || kid == KINVR || kid == KFWDP);
    const int N = row ? nx_ : ny_;
    const long count = seq_count<T>(kid, nx_, ny_);
    const long target = 4L * 152 * 32;   // one warp per SM sub-partition
    int le = 3;
    const int least = kF32<T> ? 2 : 1;
    while (le > least && (long)B_ * count * (N >> le) < target && (N >> (le - 1)) <= 1024) --le;
    if (ilog2(N) < le) le = ilog2(N);
    int per = 1;
    while (per * (N >> le) < 64 && 2 * per <= count) per *= 2;
    Launch L = make_plan(kid, le, per);
    while ((!L.ok || L.threads > max_threads_for<T>(kid, le)) && per > 1) L = make_plan(kid, le, per /= 2);
    while ((!L.ok || L.threads > max_threads_for<T>(kid, le)) && le > 1) L = make_plan(kid, --le, 1);
    return L;
}

// The dynamic shared-memory limit is an attribute of the kernel function,
// shared by every stepper in the process: each one raises it to the same
// library-wide cap (never to its own plan's size), so steppers on other
// grids running concurrently in other threads can never lower it below
// what their launches need.  A launch still requests only L.smem.
template <class T> int StepperImpl<T>::set_smem_attr(int kid, const Launch& L) {
    if (L.smem > kMaxSmem) {
        set_error("launch plan needs more shared memory than the library allows");
        return NSSTAB_ERR_INVALID_ARG;
    }
    const int sm = (int)kMaxSmem;
#define NS_ATTR(fn) NS_CUDA(cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, sm))
    if constexpr (kF32<T>) {   // the constant-length kernels of launch_fixed
        int rc = NSSTAB_OK;
        auto attr = [&](auto kernel) { rc = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, sm) == cudaSuccess ? rc : NSSTAB_ERR_CUDA; };
        with_length(f_.logy, kColLo, [&](auto i) {
            if (kid == KCOLP) attr(k_col_poisson<T, 3, true, kColLo + i>);
            if (kid == KCOLU) attr(k_col_update<T, 3, kColLo + i>);
        });
        with_length(f_.logx, kRowLo, [&](auto i) {
            if (kid == KINVR) attr(k_row_inverse<T, 3, INV_WUV, kRowLo + i>);
            if (kid == KFWDP) attr(k_row_forward<T, FWD_PEN_LIN, 3, kRowLo + i>);
            if (kid == KFWDP) attr(k_row_forward<T, FWD_PEN_NL, 3, kRowLo + i>);
        });
        if (rc != NSSTAB_OK) set_error("launch plan: cudaFuncSetAttribute failed");
        NS_TRY(rc);
    }
#define NS_ATTR_LE(KERNEL)                 \
    switch (L.le) {                        \
        case 1: NS_ATTR(KERNEL(1)); break; \
        case 2: NS_ATTR(KERNEL(2)); break; \
        default: NS_ATTR(KERNEL(3)); break; \
    }
    switch (kid) {
        case KCOLP: NS_ATTR_LE(K_COLP); NS_ATTR_LE(K_COLPSI); break;
        case KINVP: NS_ATTR_LE(K_INVP); NS_ATTR_LE(K_INVPSI); break;
        case KINVR: NS_ATTR_LE(K_INVR); break;
        case KFWDR:
            NS_ATTR_LE(K_FWD_RNL);
            NS_ATTR_LE(K_FWD_RLIN);
            NS_ATTR_LE(K_FWD_PLAIN);
            // launch_tangent_row runs at other elements a thread and with
            // more sequences' shared memory than this plan
            NS_ATTR(K_FWD_RTAN(1));
            NS_ATTR(K_FWD_RTAN(2));
            NS_ATTR(K_FWD_RTAN(3));
            break;
        case KCOLU: NS_ATTR_LE(K_COLU); break;
        default: NS_ATTR_LE(K_FWD_PNL); NS_ATTR_LE(K_FWD_PLIN); NS_ATTR_LE(K_FWD_PTAN); break;
    }
    return NSSTAB_OK;
}

// Largest block the register budget of the kernel instantiations behind
// launch `kid` with 2^le elements per thread allows.
template <class T> int max_threads_for(int kid, int le) {
    cudaFuncAttributes a;
    int m = 1024;
    auto take = [&](const void* fn) {
        if (cudaFuncGetAttributes(&a, fn) == cudaSuccess) m = std::min(m, a.maxThreadsPerBlock);
        else m = 0;
    };
#define NS_TAKE_LE(KERNEL)                            \
    switch (le) {                                     \
        case 1: take((const void*)KERNEL(1)); break;  \
        case 2: take((const void*)KERNEL(2)); break;  \
        default: take((const void*)KERNEL(3)); break; \
    }
    switch (kid) {
        case KCOLP: NS_TAKE_LE(K_COLP); NS_TAKE_LE(K_COLPSI); break;
        case KINVP: NS_TAKE_LE(K_INVP); NS_TAKE_LE(K_INVPSI); break;
        case KINVR: NS_TAKE_LE(K_INVR); break;
        case KFWDR: NS_TAKE_LE(K_FWD_RNL); NS_TAKE_LE(K_FWD_RLIN); NS_TAKE_LE(K_FWD_PLAIN); break;
        case KCOLU: NS_TAKE_LE(K_COLU); break;
        default: NS_TAKE_LE(K_FWD_PNL); NS_TAKE_LE(K_FWD_PLIN); NS_TAKE_LE(K_FWD_PTAN); break;
    }
    return m;
}

template <class T> int StepperImpl<T>::set_plan(int kid, int le, int per) {
    if (kid < 0 || kid >= kNumStepKernels) {
        set_error("set_plan: bad kernel id");
        return NSSTAB_ERR_INVALID_ARG;
    }
    const Launch L = make_plan(kid, le, per);
    if (!L.ok || L.threads > max_threads_for<T>(kid, le)) {
        set_error("set_plan: configuration not valid for this grid");
        return NSSTAB_ERR_INVALID_ARG;
    }
    NS_TRY(set_smem_attr(kid, L));
    plan_[kid] = L;
    clear_graphs();
    return NSSTAB_OK;
}

#define NS_DISPATCH_LE(L, CALL)  \
    switch ((L).le) {            \
        case 1: CALL(1); break;  \
        case 2: CALL(2); break;  \
        default: CALL(3); break; \
    }

template <class T> int StepperImpl<T>::launch_plain(cudaStream_t st) {
    const Launch& L = plan_[KFWDR];
    const dim3 g(L.blocks, B_);
#define CALL_PLAIN(le) k_row_forward<T, FWD_PLAIN, le><<<g, L.threads, L.smem, st>>>(f_, L.per, false, true)
    NS_DISPATCH_LE(L, CALL_PLAIN);
    NS_LAUNCH_CHECK();
    return NSSTAB_OK;
}

template <class T> bool StepperImpl<T>::launch_fixed(int kid, cudaStream_t st, bool linear, bool sfd, bool do_fft, bool first) {
    if constexpr (kF32<T>) {
        const Launch& L = plan_[kid];
        if (L.le != 3) return false;
        const dim3 g(L.blocks, B_);
        switch (kid) {
            case KCOLP:
                return with_length(f_.logy, kColLo, [&](auto i) {
                    k_col_poisson<T, 3, true, kColLo + i><<<g, L.threads, L.smem, st>>>(f_, L.per, f_.scale);
                });
            case KCOLU:
                return with_length(f_.logy, kColLo, [&](auto i) {
                    Fields<T> fl = f_;
                    if (xn_x4_) fl.XN = f_.X4;
                    k_col_update<T, 3, kColLo + i><<<g, L.threads, L.smem, st>>>(fl, L.per, first ? T(1) : T(1.5),
                                                                                 first ? T(0) : T(-0.5), first);
                });
            case KINVR:
                return with_length(f_.logx, kRowLo, [&](auto i) {
                    k_row_inverse<T, 3, INV_WUV, kRowLo + i><<<g, L.threads, L.smem, st>>>(f_, L.per, true);
                });
            case KFWDP:
                return with_length(f_.logx, kRowLo, [&](auto i) {
                    if (linear) k_row_forward<T, FWD_PEN_LIN, 3, kRowLo + i><<<g, L.threads, L.smem, st>>>(f_, L.per, sfd, do_fft);
                    else k_row_forward<T, FWD_PEN_NL, 3, kRowLo + i><<<g, L.threads, L.smem, st>>>(f_, L.per, sfd, do_fft);
                });
        }
    }
    return false;
}

template <class T> int StepperImpl<T>::launch(int kid, cudaStream_t st, bool linear, bool sfd, bool do_fft, bool first) {
    const Launch& L = plan_[kid];
    const dim3 g(L.blocks, B_);
    if (launch_fixed(kid, st, linear, sfd, do_fft, first)) {
        NS_LAUNCH_CHECK();
        return NSSTAB_OK;
    }
    Fields<T> fl = f_;
    switch (kid) {
        case KCOLP: {
#define CALL_COLP(le) k_col_poisson<T, le, kF32<T>><<<g, L.threads, L.smem, st>>>(fl, L.per, f_.scale)
            NS_DISPATCH_LE(L, CALL_COLP);
            break;
        }
        case KINVP: {
#define CALL_INVP(le) K_INVP(le)<<<g, L.threads, L.smem, st>>>(fl, L.per, false)
            NS_DISPATCH_LE(L, CALL_INVP);
            break;
        }
        case KFWDR: {
#define CALL_FRL(le) k_row_forward<T, FWD_RHS_LIN, le><<<g, L.threads, L.smem, st>>>(fl, L.per, false, true)
#define CALL_FRN(le) k_row_forward<T, FWD_RHS_NL, le><<<g, L.threads, L.smem, st>>>(fl, L.per, false, true)
            if (linear) {
                NS_DISPATCH_LE(L, CALL_FRL);
            } else {
                NS_DISPATCH_LE(L, CALL_FRN);
            }
            break;
        }
        case KCOLU: {
            if (xn_x4_) fl.XN = f_.X4;
            const T c1 = first ? T(1) : T(1.5), c0 = first ? T(0) : T(-0.5);
#define CALL_COLU(le) k_col_update<T, le><<<g, L.threads, L.smem, st>>>(fl, L.per, c1, c0, first)
            NS_DISPATCH_LE(L, CALL_COLU);
            break;
        }
        case KINVR: {
#define CALL_INVR(le) K_INVR(le)<<<g, L.threads, L.smem, st>>>(fl, L.per, true)
            NS_DISPATCH_LE(L, CALL_INVR);
            break;
        }
        default: {
#define CALL_FPL(le) k_row_forward<T, FWD_PEN_LIN, le><<<g, L.threads, L.smem, st>>>(fl, L.per, sfd, do_fft)
#define CALL_FPN(le) k_row_forward<T, FWD_PEN_NL, le><<<g, L.threads, L.smem, st>>>(fl, L.per, sfd, do_fft)
            if (linear) {
                NS_DISPATCH_LE(L, CALL_FPL);
            } else {
                NS_DISPATCH_LE(L, CALL_FPN);
            }
            break;
        }
    }
    NS_LAUNCH_CHECK();
    return NSSTAB_OK;
}

// Threads of a block of k_row_chain in place of KINVP + KFWDR or KINVR +
// KFWDP (0: keep the two kernels): where no SM gets more than `most` warps of
// the batch.  us a step without / with it, warps an SM at the edge: FP64
// 128x64 x 4 (8) 39.0 / 33.8, 256x128 (16) 40.2 / 43.0 (the extra transforms
// are FP64-bound there); double-float 256x128 (16) 29.8 / 27.4, 512x256 (32)
// 38.4 / 40.9; FP32 256x128 (20) 21.6 / 19.6.
template <class T> int StepperImpl<T>::chain_threads(int kid, int le) const {
    if ((kF32<T> && kid == KFWDR) || (!kF32<T> && le == 3)) return 0;
    const int groups = kid == KFWDR ? 3 : kF32<T> ? 5 : 4;
    const int threads = groups * (nx_ >> le);
    const size_t smem = (size_t)(groups + 1) * padded_len<T>(nx_) * sizeof(C);
    const long most = std::is_same<T, double>::value ? 8 : kF32<T> ? 20 : 16;
    const long per_sm = ((long)B_ * (ny_ / 2) + 151) / 152 * ((threads + 31) / 32);
    if (threads > 1024 || smem > kMaxSmem || per_sm > most) return 0;
    return threads;
}

template <class T>
int StepperImpl<T>::launch_chain(int kid, cudaStream_t st, bool linear, bool sfd, bool do_fft, bool tangent) {
    const int threads = chain_threads(kid), le = plan_[kid].le;
    const size_t smem = (size_t)((kid == KFWDR ? 3 : kF32<T> ? 5 : 4) + 1) * padded_len<T>(nx_) * sizeof(C);
    const dim3 g(ny_ / 2, B_);
    auto run = [&](auto kernel) -> int {
        if (smem > 48 * 1024)
            NS_CUDA(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kMaxSmem));
        kernel<<<g, threads, smem, st>>>(f_, sfd, do_fft);
        NS_LAUNCH_CHECK();
        return NSSTAB_OK;
    };
#define NS_CHAIN(MODE)                                          \
    do {                                                        \
        if (le == 1) return run(k_row_chain<T, MODE, 1>);       \
        if (le == 2) return run(k_row_chain<T, MODE, 2>);       \
        if constexpr (kF32<T>) return run(k_row_chain<T, MODE, 3>); \
    } while (0)
    if (kid == KFWDR) {
        if constexpr (!kF32<T>) {
            if (linear) NS_CHAIN(FWD_RHS_LIN);
            NS_CHAIN(FWD_RHS_NL);
        }
    } else {
        if (tangent) NS_CHAIN(FWD_PEN_TAN);
        if (linear) NS_CHAIN(FWD_PEN_LIN);
        NS_CHAIN(FWD_PEN_NL);
    }
    set_error("fused row pass: no such kernel");
    return NSSTAB_ERR_INVALID_ARG;
}

// The row passes of a trajectory and its perturbation (two members): FWD_RHS_TAN, FWD_PEN_TAN
template <class T> int StepperImpl<T>::launch_tangent_row(int kid, cudaStream_t st, bool do_fft) {
    Launch L = plan_[kid];
    if (kid == KFWDR) {
        if (kF32<T>) {
            // four transforms a thread (512-thread bounds): 8 elements in
            // place of 4 (27.5 us a step against 30.0 at 512x256, and 4 is
            // behind 2 or 8 on every grid from 64x32 to 2048x1024), fewer
            // pairs where the plan's block would not fit
            if (L.le == 2 && f_.logx >= 3) L = make_plan(kid, 3, L.per);
            while (L.per > 1 && (L.threads > 512 || 2 * L.smem > kMaxSmem)) L = make_plan(kid, L.le, L.per / 2);
            if (L.threads > 512) L = make_plan(kid, 3, 1);
            L.smem *= 2;
        }
        const dim3 g(L.blocks, B_);
#define CALL_RTAN(le) K_FWD_RTAN(le)<<<g, L.threads, L.smem, st>>>(f_, L.per, false, true)
        NS_DISPATCH_LE(L, CALL_RTAN);
    } else {
        const dim3 g(L.blocks, B_);
#define CALL_PTAN(le) K_FWD_PTAN(le)<<<g, L.threads, L.smem, st>>>(f_, L.per, false, do_fft)
        NS_DISPATCH_LE(L, CALL_PTAN);
    }
    NS_LAUNCH_CHECK();
    return NSSTAB_OK;
}

// Shape of the fused row passes for strips of R rows (nunits = 0: the grid
// or arithmetic does not allow it).
template <class T> RollShape StepperImpl<T>::roll_shape(int R) const {
    RollShape r{};
    if (!kF32<T> || nx_ < 64 || nx_ > kRollPoints || R < 2 || (R & 1) || R > ny_ || ny_ % R != 0) return r;
    r.R = R;
    r.G = std::min(kRollPoints / nx_, ny_ / R);
    r.upm = ny_ / (R * r.G);
    r.nunits = B_ * r.upm;
    return r;
}

template <class T> int StepperImpl<T>::set_fused_rows(int R) {
    if (R == 0) {
        rollR_ = 0;
        clear_graphs();
        return NSSTAB_OK;
    }
    const RollShape r = roll_shape(R);
    if (r.nunits == 0) {
        set_error("fused row passes need the FP32 stepper, 64 <= nx <= 2048 and an even R dividing ny");
        return NSSTAB_ERR_INVALID_ARG;
    }
    if constexpr (kF32<T>) {
        const int sm = (int)roll_smem(kRollPoints);
        NS_CUDA(cudaFuncSetAttribute(k_row_roll<FWD_RHS_NL>, cudaFuncAttributeMaxDynamicSharedMemorySize, sm));
        NS_CUDA(cudaFuncSetAttribute(k_row_roll<FWD_RHS_LIN>, cudaFuncAttributeMaxDynamicSharedMemorySize, sm));
        NS_CUDA(cudaFuncSetAttribute(k_row_roll<FWD_PEN_NL>, cudaFuncAttributeMaxDynamicSharedMemorySize, sm));
        NS_CUDA(cudaFuncSetAttribute(k_row_roll<FWD_PEN_LIN>, cudaFuncAttributeMaxDynamicSharedMemorySize, sm));
    }
    rollR_ = R;
    rs_ = r;
    clear_graphs();
    return NSSTAB_OK;
}

// One fused row pass over every active member: persistent blocks, one per
// SM at most (the pass holds 96 G nx bytes of shared memory).
template <class T>
int StepperImpl<T>::launch_roll(bool pen, cudaStream_t st, bool linear, bool sfd, bool do_fft, bool write_w) {
    if constexpr (kF32<T>) {
        RollShape r = rs_;
        r.write_w = write_w ? 1 : 0;
        r.do_fft = do_fft ? 1 : 0;
        const Fields<T>& fl = f_;
        const int blocks = std::min(r.nunits, 152);
        const size_t smem = roll_smem(r.G * nx_) ;
        if (!pen) {
            if (linear) k_row_roll<FWD_RHS_LIN><<<blocks, kRollThreads, smem, st>>>(fl, r, false);
            else k_row_roll<FWD_RHS_NL><<<blocks, kRollThreads, smem, st>>>(fl, r, false);
        } else {
            if (linear) k_row_roll<FWD_PEN_LIN><<<blocks, kRollThreads, smem, st>>>(fl, r, sfd);
            else k_row_roll<FWD_PEN_NL><<<blocks, kRollThreads, smem, st>>>(fl, r, sfd);
        }
        NS_LAUNCH_CHECK();
        return NSSTAB_OK;
    } else {
        set_error("fused row passes exist for the FP32 stepper only");
        return NSSTAB_ERR_INVALID_ARG;
    }
}

// --------------------------------------------------------------- tables

template <class T> int StepperImpl<T>::build_tables() {
    const int nx = nx_, ny = ny_, nxh = nxh_;
    const double dx = cfg_.Lx / nx, dy = cfg_.Ly / ny;
    const double dt = cfg_.dt;
    const long double two_pi = 6.283185307179586476925286766559005768L;
    // per-pass twiddle tables (see fft.cuh) in extended precision, rounded once
    auto build_tw = [&](int N, int LE, std::vector<C>& out) {
        const int logN = ilog2(N);
        out.clear();
        int nsl = 0, rem = logN;
        auto pass = [&](int LR) {
            const long Ns = 1L << nsl, len = Ns << LR;
            for (int q = 0; nsl > 0 && q < tw_rows<T>(LR); ++q)
                for (long k = 0; k < Ns; ++k) {
                    const long e = tw_exponent<T>(LR, q, k, Ns);
                    const long double a = two_pi * (long double)e / (long double)len;
                    const long double c = cosl(a), sn = sinl(a);
                    if constexpr (std::is_same<T, double>::value) {   // larger component, ratio
                        out.push_back(tw_by_sine(e, len) ? mk<T>((double)sn, (double)(-c / sn))
                                                         : mk<T>((double)c, (double)(sn / c)));
                        continue;
                    }
                    const T ch = (T)(double)c, sh = (T)(double)-sn;
                    out.push_back(mk<T>(ch, sh));
                    if (kTwWidth<T> == 2)   // FP32: the rounding errors of hi, next to it
                        out.push_back(mk<T>((T)(double)(c - (long double)(double)ch),
                                            (T)(double)(-sn - (long double)(double)sh)));
                }
            nsl += LR;
            rem -= LR;
        };
        while (rem >= LE) pass(LE);
        if (rem > 0) pass(rem);
    };
    // spectral operators over kx in [0, nx/2], ky in [0, ny): eigenvalue of
    // the periodic 5-point Laplacian lam = lx(kx) + ly(ky); tA, tB per set
    const size_t nt = (size_t)(nxh + 1) * ny;
    std::vector<T> tA(nt * S_), tB(nt * S_), tP(nt);
    // rows 0 and nx/2: the half sum and half difference of their operators (apply_packed0)
    std::vector<double> row0((size_t)(1 + 2 * S_) * ny);   // row 0 of tP, then of tA, tB per set, in FP64
    auto put = [&](std::vector<T>& t, size_t at, int kx, int ky, double* first, double v) {
        if (kx == 0) {
            first[ky] = v;
        } else if (kx < nxh) {
            t[at + (size_t)kx * ny + ky] = (T)v;
        } else {
            t[at + ky] = (T)(0.5 * (first[ky] + v));
            t[at + (size_t)nxh * ny + ky] = (T)(0.5 * (first[ky] - v));
        }
    };
    const double scale = 0.5 / ((double)nx * (double)ny);
    for (int kx = 0; kx <= nxh; ++kx) {
        const double sx = std::sin(kPi * kx / nx);
        const double lx = -(4.0 / (dx * dx)) * sx * sx;
        for (int ky = 0; ky < ny; ++ky) {
            const double sy = std::sin(kPi * ky / ny);
            const double lam = lx - (4.0 / (dy * dy)) * sy * sy;
            const bool mean = kx == 0 && ky == 0;   // the mean mode is removed: A = B = P = 0
            put(tP, 0, kx, ky, row0.data(), mean ? 0.0 : -1.0 / lam);
            for (int k = 0; k < S_; ++k) {
                const double nu = 1.0 / Re_[k];
                const double a = 1.0 + 0.5 * nu * dt * lam;
                const double b = 1.0 - 0.5 * nu * dt * lam;
                double* first = row0.data() + (size_t)(1 + 2 * k) * ny;
                // FP32: A - 1 = nu dt lam / b, formed without cancellation
                const double A = kF32<T> ? (mean ? -scale : scale * (nu * dt * lam) / b) : (mean ? 0.0 : scale * a / b);
                put(tA, k * nt, kx, ky, first, A);
                put(tB, k * nt, kx, ky, first + ny, mean ? 0.0 : scale * dt / b);
            }
        }
    }
    // penalisation coefficients from the cylinder mask and the fringe, per set
    std::vector<T> cS(n_ * S_), cG(n_ * S_);
    const int nxc = 1 << f_.logc, np = ny / 2;
    std::vector<unsigned char> pf((size_t)S_ * np * nxc);
    std::vector<double> sS(n_), sG(n_);
    std::vector<unsigned char> hit((size_t)np * nxc);
    const double w = 0.5 * cfg_.mask_cells * dx;
    const double xs = (1.0 - cfg_.sponge_frac) * cfg_.Lx;
    // periodic distances to the cylinder centre and the fringe, per column and row
    auto wrap = [](double d, double L) {
        d = std::fmod(d + 0.5 * L, L);
        return (d < 0 ? d + L : d) - 0.5 * L;
    };
    std::vector<double> ddx(nx), ddy(ny), sig(nx);
    for (int i = 0; i < nx; ++i) {
        const double x = i * dx;
        ddx[i] = wrap(x - cfg_.cyl_x, cfg_.Lx);
        if (cfg_.sponge_sigma > 0.0 && cfg_.sponge_frac > 0.0 && x >= xs) {
            const double sn = std::sin(kPi * (x - xs) / (cfg_.sponge_frac * cfg_.Lx));
            sig[i] = cfg_.sponge_sigma * sn * sn;
        }
    }
    for (int j = 0; j < ny; ++j) ddy[j] = wrap(j * dy - cfg_.cyl_y, cfg_.Ly);
    for (int k = 0; k < S_; ++k) {
        const double Dk = D_[k], R = 0.5 * Dk;
        for (int j = 0; j < ny; ++j) {
            for (int i = 0; i < nx; ++i) {
                double chi = 0.0;
                if (Dk > 0.0 && std::abs(ddx[i]) < R + w && std::abs(ddy[j]) < R + w) {
                    const double r = std::sqrt(ddx[i] * ddx[i] + ddy[j] * ddy[j]);
                    if (r <= R - w) chi = 1.0;
                    else if (r >= R + w) chi = 0.0;
                    else chi = 0.5 * (1.0 - std::sin(kPi * (r - R) / (2.0 * w)));
                }
                const size_t c = (size_t)j * nx + i;
                sS[c] = sG[c] = 0.0;
                if (chi == 0.0 && sig[i] == 0.0) continue;
                const double s = dt * (chi / cfg_.eta + sig[i]);
                sS[c] = s / (1.0 + s);
                sG[c] = dt * sig[i] * cfg_.Uinf / (1.0 + s);
            }
        }
        // chunks (rows 2 p, 2 p + 1; 2^kPenChunkLog columns) with a coefficient
        // in reach of their stencils (one column and one row to each side)
        std::fill(hit.begin(), hit.end(), (unsigned char)0);
        for (int j = 0; j < ny; ++j)
            for (int i = 0; i < nx; ++i) {
                if (sS[(size_t)j * nx + i] == 0.0 && sG[(size_t)j * nx + i] == 0.0) continue;
                for (int dj = -1; dj <= 1; ++dj)
                    for (int di = -1; di <= 1; ++di)
                        hit[(size_t)(((j + dj) & (ny - 1)) >> 1) * nxc + (((i + di) & (nx - 1)) >> kPenChunkLog)] = 1;
            }
        // those read u*, v* or psi* up to two columns and rows beyond them
        for (int p = 0; p < np; ++p)
            for (int c = 0; c < nxc; ++c) {
                int read = 0;
                for (int dp = -1; dp <= 1; ++dp)
                    for (int dc = -1; dc <= 1; ++dc)
                        read |= hit[(size_t)((p + dp) & (np - 1)) * nxc + ((c + dc) & (nxc - 1))];
                pf[((size_t)k * np + p) * nxc + c] = (unsigned char)(hit[(size_t)p * nxc + c] | (read << 1));
            }
        const double idy2 = 1.0 / (2.0 * dy), U = cfg_.Uinf;
        for (int j = 0; j < ny; ++j)
            for (int i = 0; i < nx; ++i) {
                const size_t c = (size_t)j * nx + i;
                const size_t cp = (size_t)((j + 1) & (ny - 1)) * nx + i, cm = (size_t)((j - 1) & (ny - 1)) * nx + i;
                cS[k * n_ + c] = (T)sS[c];
                cG[k * n_ + c] = kF32<T> ? (T)sG[c] : (T)(-((sG[cp] - sS[cp] * U) - (sG[cm] - sS[cm] * U)) * idy2);
            }
    }
    for (int le = 1; le <= 3; ++le) {
        std::vector<C> tx, ty;
        if (ilog2(nx) >= le) {
            build_tw(nx, le, tx);
            NS_CUDA(cudaMemcpy((void*)f_.twx[le], tx.data(), tx.size() * sizeof(C), cudaMemcpyHostToDevice));
        }
        if (ilog2(ny) >= le) {
            build_tw(ny, le, ty);
            NS_CUDA(cudaMemcpy((void*)f_.twy[le], ty.data(), ty.size() * sizeof(C), cudaMemcpyHostToDevice));
        }
    }
    NS_CUDA(cudaMemcpyAsync((void*)f_.tA, tA.data(), tA.size() * sizeof(T), cudaMemcpyHostToDevice, stream_));
    NS_CUDA(cudaMemcpyAsync((void*)f_.tB, tB.data(), tB.size() * sizeof(T), cudaMemcpyHostToDevice, stream_));
    NS_CUDA(cudaMemcpyAsync((void*)f_.tP, tP.data(), tP.size() * sizeof(T), cudaMemcpyHostToDevice, stream_));
    // centred-difference symbols: D_x <-> i sin(2 pi kx/nx)/dx, D_y alike
    std::vector<T> tDx(nxh + 1), tDy(ny);
    for (int kx = 0; kx <= nxh; ++kx) tDx[kx] = (kx == 0 || kx == nxh) ? T(0) : (T)(std::sin(2.0 * kPi * kx / nx) / dx);
    for (int ky = 0; ky < ny; ++ky) tDy[ky] = (2 * ky == ny || ky == 0) ? T(0) : (T)(std::sin(2.0 * kPi * ky / ny) / dy);
    if (f_.tDx) {
        NS_CUDA(cudaMemcpyAsync((void*)f_.tDx, tDx.data(), tDx.size() * sizeof(T), cudaMemcpyHostToDevice, stream_));
        NS_CUDA(cudaMemcpyAsync((void*)f_.tDy, tDy.data(), tDy.size() * sizeof(T), cudaMemcpyHostToDevice, stream_));
    }
    NS_CUDA(cudaMemcpyAsync((void*)f_.cS, cS.data(), cS.size() * sizeof(T), cudaMemcpyHostToDevice, stream_));
    NS_CUDA(cudaMemcpyAsync((void*)f_.cG, cG.data(), cG.size() * sizeof(T), cudaMemcpyHostToDevice, stream_));
    NS_CUDA(cudaMemcpyAsync((void*)f_.pf, pf.data(), pf.size(), cudaMemcpyHostToDevice, stream_));
    NS_CUDA(cudaStreamSynchronize(stream_));   // host vectors go out of scope
    return NSSTAB_OK;
}

template <class T> int StepperImpl<T>::init() {
    nx_ = cfg_.nx;
    ny_ = cfg_.ny;
    nxh_ = nx_ / 2;
    n_ = (size_t)nx_ * ny_;
    nc_ = (size_t)nxh_ * ny_;
    const size_t nt = (size_t)(nxh_ + 1) * ny_;
    f_.nx = nx_;
    f_.ny = ny_;
    f_.nxh = nxh_;
    f_.logx = ilog2(nx_);
    f_.logy = ilog2(ny_);
    f_.logc = std::max(0, f_.logx - kPenChunkLog);
    f_.bper = bper_;
    f_.fs = n_;
    f_.cs = nc_;
    f_.ts = nt;
    f_.idx2 = (T)(1.0 / (2.0 * cfg_.Lx / nx_));
    f_.idy2 = (T)(1.0 / (2.0 * cfg_.Ly / ny_));
    f_.Uinf = (T)cfg_.Uinf;
    f_.scale = (T)(0.5 / ((double)nx_ * (double)ny_));
    const size_t B = B_, S = S_;
    T *W, *P, *cS, *cG, *tA, *tB, *tP;
    C *X1, *X2, *Wh, *Nh;
    NS_TRY(dalloc(&W, B * n_));
    NS_TRY(dalloc(&P, B * n_));
    NS_TRY(dalloc(&X1, B * nc_));
    NS_TRY(dalloc(&X2, B * nc_));
    NS_TRY(dalloc(&Wh, B * nc_));
    NS_TRY(dalloc(&Nh, B * nc_));
    NS_TRY(dalloc(&cS, S * n_));
    NS_TRY(dalloc(&cG, S * n_));
    NS_TRY(dalloc(&tA, S * nt));
    NS_TRY(dalloc(&tB, S * nt));
    NS_TRY(dalloc(&tP, nt));
    if (kF32<T>) {
        T *U, *V, *tDx, *tDy;
        C* X3;
        NS_TRY(dalloc(&U, B * n_));
        NS_TRY(dalloc(&V, B * n_));
        NS_TRY(dalloc(&X3, B * nc_));
        C* X4;
        NS_TRY(dalloc(&X4, B * nc_));
        f_.X4 = X4;
        NS_CUDA(cudaMemsetAsync(X4, 0, B * nc_ * sizeof(C), stream_));
        NS_TRY(dalloc(&tDx, (size_t)nxh_ + 1));
        NS_TRY(dalloc(&tDy, (size_t)ny_));
        f_.U = U; f_.V = V; f_.X3 = X3; f_.tDx = tDx; f_.tDy = tDy;
        NS_CUDA(cudaMemsetAsync(U, 0, B * n_ * sizeof(T), stream_));
        NS_CUDA(cudaMemsetAsync(V, 0, B * n_ * sizeof(T), stream_));
        NS_CUDA(cudaMemsetAsync(X3, 0, B * nc_ * sizeof(C), stream_));
    }
    for (int le = 1; le <= 3; ++le) {
        C *tx, *ty;
        NS_TRY(dalloc(&tx, (size_t)2 * kTwWidth<T> * nx_));
        NS_TRY(dalloc(&ty, (size_t)2 * kTwWidth<T> * ny_));
        f_.twx[le] = tx;
        f_.twy[le] = ty;
    }
    f_.twx[0] = f_.twx[1];
    f_.twy[0] = f_.twy[1];
    unsigned char* pf;
    NS_TRY(dalloc(&pf, S * (size_t)(ny_ / 2) << f_.logc));
    f_.pf = pf;
    NS_TRY(dalloc(&red_, B * kRedBlocks));
    NS_TRY(dalloc(&active_, B));
    NS_TRY(dalloc(&ptr_in_, B));
    NS_TRY(dalloc(&ptr_out_, B));
    NS_CUDA(cudaMallocHost((void**)&red_host_, B * kRedBlocks * sizeof(double)));
    f_.W = W; f_.P = P; f_.cS = cS; f_.cG = cG;
    f_.X1 = X1; f_.X2 = X2; f_.Wh = Wh; f_.Nh = Nh;
    f_.XN = X1;
    f_.tA = tA; f_.tB = tB; f_.tP = tP;
    f_.Y = nullptr;
    f_.Ub = f_.Vb = f_.DxOb = f_.DyOb = nullptr;
    f_.active = active_;
    NS_TRY(build_tables());
    // zero the workspace so that timing runs of the autotuner see finite data
    NS_CUDA(cudaMemsetAsync(f_.W, 0, B * n_ * sizeof(T), stream_));
    NS_CUDA(cudaMemsetAsync(f_.P, 0, B * n_ * sizeof(T), stream_));
    NS_CUDA(cudaMemsetAsync(f_.X1, 0, B * nc_ * sizeof(C), stream_));
    NS_CUDA(cudaMemsetAsync(f_.X2, 0, B * nc_ * sizeof(C), stream_));
    NS_CUDA(cudaMemsetAsync(f_.Wh, 0, B * nc_ * sizeof(C), stream_));
    NS_CUDA(cudaMemsetAsync(f_.Nh, 0, B * nc_ * sizeof(C), stream_));
    NS_TRY(all_active());
    NS_CUDA(cudaStreamCreateWithFlags(&cap_, cudaStreamNonBlocking));
    for (int k = 0; k < kNumStepKernels; ++k) {
        const Launch L = default_plan(k);
        if (!L.ok) {
            set_error("grid too large for the shared-memory FFT");
            return NSSTAB_ERR_INVALID_ARG;
        }
        NS_TRY(set_plan(k, L.le, L.per));
    }

    NS_CUDA(cudaStreamSynchronize(stream_));
    return NSSTAB_OK;
}

// ------------------------------------------------- member data movement

// Host vectors are pageable: cudaMemcpyAsync stages them before returning,
// so they may be reused by the next call at once.
template <class T> int StepperImpl<T>::set_active(const std::vector<unsigned char>& a) {
    active_host_ = a;
    NS_CUDA(cudaMemcpyAsync(active_, active_host_.data(), B_, cudaMemcpyHostToDevice, stream_));
    return NSSTAB_OK;
}

template <class T> int StepperImpl<T>::gather(const double* const* src) {
    pin_host_.assign(src, src + B_);
    NS_CUDA(cudaMemcpyAsync(ptr_in_, pin_host_.data(), B_ * sizeof(double*), cudaMemcpyHostToDevice, stream_));
    k_gather<T><<<dim3(kPtBlocks, B_), 256, 0, stream_>>>(ptr_in_, f_.W, n_, n_);
    NS_LAUNCH_CHECK();
    return NSSTAB_OK;
}

template <class T> int StepperImpl<T>::scatter(const T* from, double* const* dst) {
    pout_host_.assign(dst, dst + B_);
    NS_CUDA(cudaMemcpyAsync(ptr_out_, pout_host_.data(), B_ * sizeof(double*), cudaMemcpyHostToDevice, stream_));
    k_scatter<T><<<dim3(kPtBlocks, B_), 256, 0, stream_>>>(from, ptr_out_, n_, n_);
    NS_LAUNCH_CHECK();
    return NSSTAB_OK;
}

template <class T> int StepperImpl<T>::gather_contig(const double* src, int count) {
    std::vector<const double*> p(B_, nullptr);
    for (int m = 0; m < count; ++m) p[m] = src + (size_t)m * n_;
    return gather(p.data());
}

template <class T> int StepperImpl<T>::scatter_contig(const T* from, double* dst) {
    std::vector<double*> p(B_);
    for (int m = 0; m < B_; ++m) p[m] = dst + (size_t)m * n_;
    return scatter(from, p.data());
}

// ------------------------------------------------------------- stepping

template <class T> int StepperImpl<T>::transform_W() { return launch_plain(stream_); }

template <class T> int StepperImpl<T>::stream_function(cudaStream_t st) {
    NS_TRY(launch(KCOLP, st, false, false, true, false));
    return launch(KINVP, st, false, false, true, false);
}

// P = psi from X1 for every stepper (FP32 steppers carry u', v in the step
// and form psi only here): the psi variant of the column pass, then the
// row pairs of X2, with the launch shapes of KCOLP and KINVP.
template <class T> int StepperImpl<T>::psi_function(cudaStream_t st) {
    if (!kF32<T>) return stream_function(st);
    const Launch& Lc = plan_[KCOLP];
    const dim3 gc(Lc.blocks, B_);
#define CALL_COLPSI(le) k_col_poisson<T, le, false><<<gc, Lc.threads, Lc.smem, st>>>(f_, Lc.per, f_.scale)
    NS_DISPATCH_LE(Lc, CALL_COLPSI);
    NS_LAUNCH_CHECK();
    Launch L = plan_[KINVP];   // ny rows -> ny/2 row pairs, each block at most as large
    while (L.per > ny_ / 2) L.per /= 2;
    L.blocks = (ny_ / 2) / L.per;
    L.threads = L.per * (nx_ >> L.le);
    L.smem = (size_t)L.per * padded_len<T>(nx_) * sizeof(C);
    const dim3 gr(L.blocks, B_);
#define CALL_INVPSI(le) K_INVPSI(le)<<<gr, L.threads, L.smem, st>>>(f_, L.per, false)
    NS_DISPATCH_LE(L, CALL_INVPSI);
    NS_LAUNCH_CHECK();
    return NSSTAB_OK;
}

// Enqueue nsteps time steps on `st`.  first_ab1: the first of them is AB1.
// fft_last: the last step also forms the x-spectrum of its result.
template <class T>
int StepperImpl<T>::issue_steps(cudaStream_t st, int nsteps, bool linear, bool sfd, bool first_ab1, bool fft_last,
                                bool tangent) {
    if (tangent) {
        // co-integration (members: 0 = trajectory, 1 = perturbation): the
        // steps of both in one launch per kernel, the row passes each in its
        // member's mode
        for (int s = 0; s < nsteps; ++s) {
            const bool first = first_ab1 && s == 0;
            NS_TRY(launch(KCOLP, st, false, false, true, first));
            if (!kF32<T>) NS_TRY(launch(KINVP, st, false, false, true, first));
            NS_TRY(launch_tangent_row(KFWDR, st, true));
            NS_TRY(launch(KCOLU, st, true, false, true, first));
            const bool fft = fft_last || (s + 1 < nsteps);
            if (chain_threads(KFWDP)) {
                NS_TRY(launch_chain(KFWDP, st, true, false, fft, true));
                continue;
            }
            NS_TRY(launch(KINVR, st, true, false, true, first));
            NS_TRY(launch_tangent_row(KFWDP, st, fft));
        }
        return NSSTAB_OK;
    }
    if (rollR_) {
        // four kernels: column Poisson pass, fused RHS row pass, column
        // update, fused penalisation row pass (omega to W on the last step)
        for (int s = 0; s < nsteps; ++s) {
            const bool first = first_ab1 && s == 0;
            NS_TRY(launch(KCOLP, st, false, false, true, first));
            NS_TRY(launch_roll(false, st, linear, false, true, false));
            xn_x4_ = true;
            const int rc = launch(KCOLU, st, linear, false, true, first);
            xn_x4_ = false;
            NS_TRY(rc);
            NS_TRY(launch_roll(true, st, linear, sfd, fft_last || (s + 1 < nsteps), s + 1 == nsteps));
        }
        return NSSTAB_OK;
    }
    const bool chain_r = chain_threads(KFWDR) > 0, chain_p = chain_threads(KFWDP) > 0;
    for (int s = 0; s < nsteps; ++s) {
        const bool first = first_ab1 && s == 0;
        const bool fft = fft_last || (s + 1 < nsteps);
        NS_TRY(launch(KCOLP, st, linear, false, true, first));
        if (chain_r) {
            NS_TRY(launch_chain(KFWDR, st, linear, false, true, false));
        } else {
            if (!kF32<T>) NS_TRY(launch(KINVP, st, linear, false, true, first));   // FP32: within KFWDR
            NS_TRY(launch(KFWDR, st, linear, false, true, first));
        }
        NS_TRY(launch(KCOLU, st, linear, false, true, first));
        if (chain_p) {
            NS_TRY(launch_chain(KFWDP, st, linear, sfd, fft, false));
        } else {
            NS_TRY(launch(KINVR, st, linear, false, true, first));
            NS_TRY(launch(KFWDP, st, linear, sfd, fft, first));
        }
    }
    return NSSTAB_OK;
}

// Run nsteps steps on the stepper's stream.  Long runs replay CUDA graphs of
// up to kGraphChunk steps, captured once per (length, flags) on a private
// stream and launched into the stepper's stream; the AB2 history carries
// from one chunk to the next through the workspace.  The active-member mask
// is read from device memory at run time, so graphs serve any subset.
template <class T>
int StepperImpl<T>::run_steps(int nsteps, bool linear, bool sfd, bool fft_last, bool first_ab1, bool tangent) {
    if (linear && !have_base_) {
        set_error("linearised step requested before a base flow was set");
        return NSSTAB_ERR_INVALID_ARG;
    }
    if (nsteps < 4) return issue_steps(stream_, nsteps, linear, sfd, first_ab1, fft_last, tangent);
    int done = 0;
    while (done < nsteps) {
        const int len = std::min(kGraphChunk, nsteps - done);
        const bool first = first_ab1 && done == 0;
        const bool last_fft = (done + len < nsteps) || fft_last;
        const GraphKey key{len, (linear ? 1 : 0) | (sfd ? 2 : 0) | (first ? 4 : 0) | (last_fft ? 8 : 0) |
                                    (tangent ? 16 : 0)};
        auto it = graphs_.find(key);
        if (it == graphs_.end()) {
            cudaGraph_t g = nullptr;
            NS_CUDA(cudaStreamBeginCapture(cap_, cudaStreamCaptureModeThreadLocal));
            const int rc = issue_steps(cap_, len, linear, sfd, first, last_fft, tangent);
            const cudaError_t ec = cudaStreamEndCapture(cap_, &g);
            if (rc != NSSTAB_OK) {
                if (g) cudaGraphDestroy(g);
                return rc;
            }
            NS_CUDA(ec);
            cudaGraphExec_t ex = nullptr;
            const cudaError_t ei = cudaGraphInstantiate(&ex, g, 0);
            cudaGraphDestroy(g);
            NS_CUDA(ei);
            it = graphs_.emplace(key, ex).first;
        }
        NS_CUDA(cudaGraphLaunch(it->second, stream_));
        done += len;
    }
    return NSSTAB_OK;
}

// Whether some plan of row pass kid runs with the inverse pass before it as one kernel
template <class T> bool StepperImpl<T>::may_chain(int kid) const {
    if (rollR_ || (kid != KFWDR && kid != KFWDP)) return false;
    for (int le = 1; le <= 3; ++le)
        if (chain_threads(kid, le)) return true;
    return false;
}

// Time of `reps` launches of kernel kid under plan L, replayed as a graph as
// in a step (launched one by one, kernels of 3-5 us are timed by the host).  A
// row pass that may_chain is timed together with the inverse pass before it,
// in the form the step would take; linearised once there is a base flow.
template <class T> int StepperImpl<T>::time_kernel(int kid, const Launch& L, int reps, float* ms) {
    const Launch saved = plan_[kid];
    plan_[kid] = L;
    const bool both = may_chain(kid), lin = have_base_;
    auto issue = [&]() -> int {
        if (both && chain_threads(kid)) return launch_chain(kid, cap_, lin, false, true, false);
        if (both) NS_TRY(launch(kid == KFWDR ? KINVP : KINVR, cap_, lin, false, true, false));
        return launch(kid, cap_, lin, false, true, false);
    };
    auto fail = [&](cudaError_t e) {
        set_error(std::string("autotune: ") + cudaGetErrorString(e));
        return NSSTAB_ERR_CUDA;
    };
    cudaGraph_t g = nullptr;
    cudaGraphExec_t ex = nullptr;
    cudaEvent_t e0 = nullptr, e1 = nullptr;
    int rc = NSSTAB_OK;
    cudaError_t e = cudaStreamBeginCapture(cap_, cudaStreamCaptureModeThreadLocal);
    if (e == cudaSuccess) {
        for (int r = 0; r < reps && rc == NSSTAB_OK; ++r) rc = issue();
        e = cudaStreamEndCapture(cap_, &g);
    }
    plan_[kid] = saved;
    if (rc == NSSTAB_OK) {
        if (e == cudaSuccess) e = cudaGraphInstantiate(&ex, g, 0);
        if (e == cudaSuccess) e = cudaEventCreate(&e0);
        if (e == cudaSuccess) e = cudaEventCreate(&e1);
        if (e == cudaSuccess) e = cudaGraphLaunch(ex, stream_);   // warm-up
        if (e == cudaSuccess) e = cudaEventRecord(e0, stream_);
        if (e == cudaSuccess) e = cudaGraphLaunch(ex, stream_);
        if (e == cudaSuccess) e = cudaEventRecord(e1, stream_);
        if (e == cudaSuccess) e = cudaEventSynchronize(e1);
        if (e == cudaSuccess) e = cudaEventElapsedTime(ms, e0, e1);
        if (e != cudaSuccess) rc = fail(e);
    }
    if (e0) cudaEventDestroy(e0);
    if (e1) cudaEventDestroy(e1);
    if (ex) cudaGraphExecDestroy(ex);
    if (g) cudaGraphDestroy(g);
    return rc;
}

// Measure every valid (elements per thread, sequences per block) pair of
// each kernel on this grid and batch and keep the fastest.  What is measured
// is what a step launches: with the six kernels timed one by one the choice of
// KFWDP took k_row_chain away from grids that are faster with it (double-float
// 512x64: 32.3 us a step by default, 32.7-35.9 tuned).  (KINVP of an FP32
// stepper runs outside the steps, in set_base and the like.)  Clobbers the
// workspace (never the base flow).  chosen[2k], chosen[2k+1] = (le, per).
template <class T> int StepperImpl<T>::autotune(int reps, int* chosen) {
    NS_TRY(all_active());
    for (int kid = 0; kid < kNumStepKernels; ++kid) {
        Launch best = plan_[kid];
        float best_ms = 1e30f;
        for (int le = 1; le <= 3; ++le) {
            for (int per = 1; per <= 16; per *= 2) {
                const Launch L = make_plan(kid, le, per);
                if (!L.ok || L.threads < 32 || L.threads > max_threads_for<T>(kid, le)) continue;
                NS_TRY(set_smem_attr(kid, L));
                float ms = 0.f;
                NS_TRY(time_kernel(kid, L, reps, &ms));
                if (ms < best_ms) {
                    best_ms = ms;
                    best = L;
                }
                if (may_chain(kid) && chain_threads(kid, le)) break;   // one block per pair whatever `per`
            }
        }
        NS_TRY(set_plan(kid, best.le, best.per));
        if (chosen) {
            chosen[2 * kid] = best.le;
            chosen[2 * kid + 1] = best.per;
        }
    }
    return NSSTAB_OK;
}

template <class T> int StepperImpl<T>::profile_linear(const double* v, int nsteps, double* ms) {
    if (!have_base_) {
        set_error("profile: no base flow set");
        return NSSTAB_ERR_INVALID_ARG;
    }
    cudaEvent_t ev[kNumStepKernels + 1];
    for (int k = 0; k <= kNumStepKernels; ++k) NS_CUDA(cudaEventCreate(&ev[k]));
    for (int k = 0; k < kNumStepKernels; ++k) ms[k] = 0.0;
    int rc = all_active();
    if (rc == NSSTAB_OK) rc = gather_contig(v, B_);
    if (rc == NSSTAB_OK) rc = transform_W();
    for (int s = 0; s < nsteps && rc == NSSTAB_OK; ++s) {
        const bool first = (s == 0);
        for (int k = 0; k < kNumStepKernels && rc == NSSTAB_OK; ++k) {
            cudaEventRecord(ev[k], stream_);
            if (!rollR_) {
                if (!(kF32<T> && k == KINVP)) rc = launch(k, stream_, true, false, true, first);
            }
            else if (k == KCOLP) rc = launch(k, stream_, true, false, true, first);
            else if (k == KCOLU) {
                xn_x4_ = true;
                rc = launch(k, stream_, true, false, true, first);
                xn_x4_ = false;
            }
            else if (k == KFWDR) rc = launch_roll(false, stream_, true, false, true, false);
            else if (k == KFWDP) rc = launch_roll(true, stream_, true, false, true, s + 1 == nsteps);
        }
        cudaEventRecord(ev[kNumStepKernels], stream_);
        if (rc != NSSTAB_OK) break;
        const cudaError_t e = cudaEventSynchronize(ev[kNumStepKernels]);
        if (e != cudaSuccess) {
            set_error(std::string("profile: ") + cudaGetErrorString(e));
            rc = NSSTAB_ERR_CUDA;
            break;
        }
        for (int k = 0; k < kNumStepKernels; ++k) {
            float t = 0.f;
            cudaEventElapsedTime(&t, ev[k], ev[k + 1]);
            ms[k] += t;
        }
    }
    for (int k = 0; k <= kNumStepKernels; ++k) cudaEventDestroy(ev[k]);
    return rc;
}

template <class T> int StepperImpl<T>::poisson(const double* omega, double* psi) {
    NS_TRY(all_active());
    NS_TRY(gather_contig(omega, B_));
    NS_TRY(transform_W());
    NS_TRY(psi_function(stream_));
    return scatter_contig(f_.P, psi);
}

template <class T> int StepperImpl<T>::step_nonlinear(double* omega, int nsteps) {
    NS_TRY(all_active());
    NS_TRY(gather_contig(omega, B_));
    if (nsteps > 0) {
        NS_TRY(transform_W());
        NS_TRY(run_steps(nsteps, false, false, false));
    }
    return scatter_contig(f_.W, omega);
}

template <class T> int StepperImpl<T>::set_base(const double* base_omega) {
    std::vector<const double*> p(S_);
    for (int k = 0; k < S_; ++k) p[k] = base_omega + (size_t)k * n_;
    return set_base_ptrs(p.data());
}

template <class T> int StepperImpl<T>::alloc_base_fields() {
    if (!f_.Ub) {
        T *Ub, *Vb, *DxOb, *DyOb;
        NS_TRY(dalloc(&Ub, (size_t)S_ * n_));
        NS_TRY(dalloc(&Vb, (size_t)S_ * n_));
        NS_TRY(dalloc(&DxOb, (size_t)S_ * n_));
        NS_TRY(dalloc(&DyOb, (size_t)S_ * n_));
        f_.Ub = Ub; f_.Vb = Vb; f_.DxOb = DxOb; f_.DyOb = DyOb;
        clear_graphs();   // captured kernels carry the field pointers by value
    }
    return NSSTAB_OK;
}

template <class T> int StepperImpl<T>::set_base_ptrs(const double* const* base_omegas) {
    NS_TRY(alloc_base_fields());
    // the S base flows go through member slots 0..S-1
    std::vector<unsigned char> a(B_, 0);
    std::vector<const double*> src(B_, nullptr);
    for (int k = 0; k < S_; ++k) {
        a[k] = 1;
        src[k] = base_omegas[k];
    }
    NS_TRY(set_active(a));
    NS_TRY(gather(src.data()));
    NS_TRY(transform_W());
    NS_TRY(stream_function(stream_));   // P = Psi_b (FP32: U, V = its velocity)
    k_base_fields<T><<<dim3(kPtBlocks, S_), 256, 0, stream_>>>(f_, (T*)f_.Ub, (T*)f_.Vb, (T*)f_.DxOb, (T*)f_.DyOb);
    NS_LAUNCH_CHECK();
    NS_TRY(all_active());
    have_base_ = true;
    return NSSTAB_OK;
}

template <class T> int StepperImpl<T>::step_linear(const double* v_in, double* v_out, int nsteps) {
    std::vector<const double*> pi(B_);
    std::vector<double*> po(B_);
    for (int m = 0; m < B_; ++m) {
        pi[m] = v_in + (size_t)m * n_;
        po[m] = v_out + (size_t)m * n_;
    }
    return step_linear_ptrs(pi.data(), po.data(), nsteps);
}

template <class T> int StepperImpl<T>::step_linear_ptrs(const double* const* in, double* const* out, int nsteps) {
    if (!have_base_) {
        set_error("linearised step requested before a base flow was set");
        return NSSTAB_ERR_INVALID_ARG;
    }
    std::vector<unsigned char> a(B_);
    for (int m = 0; m < B_; ++m) a[m] = in[m] != nullptr;
    NS_TRY(set_active(a));
    NS_TRY(gather(in));
    if (nsteps > 0) {
        NS_TRY(transform_W());
        NS_TRY(run_steps(nsteps, true, false, false));
    }
    return scatter(f_.W, out);
}

// dPhi_T(q)/dq v_in for the stepper's two members (one parameter set):
// member 0 marches q nonlinearly, member 1 marches v linearised about
// member 0's state of the same step (co-integration).  The base does not
// outlive the call: a later linearised step needs a new one.
template <class T> int StepperImpl<T>::tangent(const double* q, const double* v_in, double* v_out, int nsteps) {
    if (B_ != 2 || S_ != 1) {
        set_error("tangent: needs a batch of two members and one parameter set");
        return NSSTAB_ERR_INVALID_ARG;
    }
    have_base_ = false;
    NS_TRY(all_active());
    const double* src[2] = {q, v_in};
    NS_TRY(gather(src));
    if (nsteps > 0) {
        NS_TRY(transform_W());
        NS_TRY(run_steps(nsteps, false, false, false, true, true));
    }
    double* dst[2] = {nullptr, v_out};
    return scatter(f_.W, dst);
}

template <class T> int StepperImpl<T>::sumsq_diff(const T* a, const T* b, double* out) {
    k_diff_sumsq<T><<<dim3(kRedBlocks, B_), 256, 0, stream_>>>(a, b, n_, n_, red_);
    NS_LAUNCH_CHECK();
    NS_CUDA(cudaMemcpyAsync(red_host_, red_, (size_t)B_ * kRedBlocks * sizeof(double), cudaMemcpyDeviceToHost,
                            stream_));
    NS_CUDA(cudaStreamSynchronize(stream_));
    for (int m = 0; m < B_; ++m) {
        double s = 0.0;
        for (int b2 = 0; b2 < kRedBlocks; ++b2) s += red_host_[(size_t)m * kRedBlocks + b2];
        out[m] = s;
    }
    return NSSTAB_OK;
}

template <class T> int StepperImpl<T>::residual(const double* q, double* r) {
    if (!Wsave_) NS_TRY(dalloc(&Wsave_, (size_t)B_ * n_));
    NS_TRY(all_active());
    NS_TRY(gather_contig(q, B_));
    NS_CUDA(cudaMemcpyAsync(Wsave_, f_.W, (size_t)B_ * n_ * sizeof(T), cudaMemcpyDeviceToDevice, stream_));
    NS_TRY(transform_W());
    NS_TRY(run_steps(1, false, false, false));
    std::vector<double> ss(B_);
    NS_TRY(sumsq_diff(f_.W, Wsave_, ss.data()));
    const double dx = cfg_.Lx / nx_, dy = cfg_.Ly / ny_;
    for (int m = 0; m < B_; ++m) r[m] = std::sqrt(ss[m] * dx * dy) / cfg_.dt;
    return NSSTAB_OK;
}

template <class T>
int StepperImpl<T>::sfd(double* omega, double chi, double Delta, double tol, long max_steps, int check_every,
                        double* r_out, long* steps_out) {
    if (!f_.Y) {
        T* Y;
        NS_TRY(dalloc(&Y, (size_t)B_ * n_));
        f_.Y = Y;
    }
    if (!Wsave_) NS_TRY(dalloc(&Wsave_, (size_t)B_ * n_));
    if (!Nhsave_) NS_TRY(dalloc(&Nhsave_, (size_t)B_ * nc_));
    f_.sfd_k1 = (T)(cfg_.dt * chi);
    f_.sfd_k2 = (T)(cfg_.dt / Delta);
    clear_graphs();   // captured kernels carry the gains and the Y pointer by value
    NS_TRY(all_active());
    NS_TRY(gather_contig(omega, B_));
    NS_CUDA(cudaMemcpyAsync(f_.Y, f_.W, (size_t)B_ * n_ * sizeof(T), cudaMemcpyDeviceToDevice, stream_));
    NS_TRY(transform_W());
    const double dx = cfg_.Lx / nx_, dy = cfg_.Ly / ny_;
    long k = 0;
    std::vector<double> r(B_, INFINITY), ss(B_);
    int status = NSSTAB_NOT_CONVERGED;
    bool first_chunk = true;
    while (k < max_steps) {
        const long chunk = std::min<long>(check_every, max_steps - k);
        // the AB2 history continues across chunks: only the very first step is AB1
        NS_TRY(run_steps((int)chunk, false, true, true, first_chunk));
        first_chunk = false;
        k += chunk;
        // residual of the current X with one plain AB1 step, then restore the state
        NS_CUDA(cudaMemcpyAsync(Wsave_, f_.W, (size_t)B_ * n_ * sizeof(T), cudaMemcpyDeviceToDevice, stream_));
        NS_CUDA(cudaMemcpyAsync(Nhsave_, f_.Nh, (size_t)B_ * nc_ * sizeof(C), cudaMemcpyDeviceToDevice, stream_));
        NS_TRY(run_steps(1, false, false, false));
        NS_TRY(sumsq_diff(f_.W, Wsave_, ss.data()));
        bool all_ok = true, finite = true;
        for (int m = 0; m < B_; ++m) {
            r[m] = std::sqrt(ss[m] * dx * dy) / cfg_.dt;
            finite = finite && std::isfinite(r[m]);
            all_ok = all_ok && r[m] <= tol;
        }
        NS_CUDA(cudaMemcpyAsync(f_.W, Wsave_, (size_t)B_ * n_ * sizeof(T), cudaMemcpyDeviceToDevice, stream_));
        NS_CUDA(cudaMemcpyAsync(f_.Nh, Nhsave_, (size_t)B_ * nc_ * sizeof(C), cudaMemcpyDeviceToDevice, stream_));
        NS_TRY(transform_W());
        if (!finite) {
            status = NSSTAB_DIVERGED;
            break;
        }
        if (all_ok) {
            status = NSSTAB_OK;
            break;
        }
    }
    NS_TRY(scatter_contig(f_.W, omega));
    NS_CUDA(cudaStreamSynchronize(stream_));
    for (int m = 0; m < B_; ++m) r_out[m] = r[m];
    *steps_out = k;
    return status;
}

}  // namespace nsstab
