// FP64 tall-skinny kernels of the Krylov layer: the classical Gram-Schmidt
// products of Algorithm 1 (h = V^T w, w -= V h, applied twice = CGS2), norms
// and the basis contraction V Q of the Krylov-Schur truncation / Ritz vector
// assembly (Sec. 3.2.2).  The basis V is column-major: column k of length n
// starts at V + k*ldv.  Reductions use a fixed grid and a fixed summation
// order, so results are bit-reproducible run to run.
#include <algorithm>
#include <vector>

#include "stepper.cuh"

namespace nsstab {

static const int kGsThreads = 256;

// Which vectors a Gram-Schmidt launch works on: one member (V, w, n, j), or
// member b's (Vs[b], ws[b], js[b]) with j < 0 for a member that sits out and,
// where ns is given, its own length n = ldv = ns[b].
__device__ __forceinline__ bool gs_member(GsArgs& a, int b) {
    if (a.Vs) {
        a.j = a.js[b];
        if (a.j < 0) return false;
        a.V = a.Vs[b];
        a.w = a.ws[b];
        if (a.ns) a.ldv = a.n = a.ns[b];
    }
    return true;
}

// partial[(b nbx + x) ldp + c] = sum over row chunk x of V[c][i] w[i], for
// the up to 8 columns c of group blockIdx.y (the groups split j evenly).
//
// Bound: the FP64 pipe (one FMA per 8 bytes of V: 2 per clock and SM take 5
// TB/s, the HBM copy runs at 6.8).  A block keeps its 8 columns over a long
// chunk of rows (64 FMAs a thread at n = 1e6, j = 129) and folds its 8 sums
// across the lanes in 9 exchanges (each halves the columns a lane holds)
// instead of 8 x 5: with 13 rows a thread and a full fold per column and warp
// the folds were 40% of the FP64 work.  Column groups in the grid keep the
// chip full at short n and leave few partial sums.  One CGS2 (with
// k_gs_update, host call included) at n = 1000003, j = 129: 2000 -> 1095 us
// (FP64 bound 820 us); n = 131072, j = 64: 273 -> 158 us; n = 8192, j = 64:
// 220 -> 66 us.
__global__ void __launch_bounds__(kGsThreads) k_gs_dot(GsArgs a, double* __restrict__ partial, int ldp) {
    if (!gs_member(a, blockIdx.z) || a.j <= 0) return;
    const int ncg = (a.j + kGsGroup - 1) / kGsGroup, g = blockIdx.y;
    if (g >= ncg) return;
    const int c0 = g * a.j / ncg, nc = (g + 1) * a.j / ncg - c0;
    const long chunk = (a.n + gridDim.x - 1) / gridDim.x;
    const long r0 = (long)blockIdx.x * chunk, r1 = min(a.n, r0 + chunk);
    const double* __restrict__ V = a.V + (long)c0 * a.ldv;
    const double* __restrict__ w = a.w;
    double v[kGsGroup];
#pragma unroll
    for (int c = 0; c < kGsGroup; ++c) v[c] = 0.0;
    if (nc == kGsGroup) {
#pragma unroll 2
        for (long i = r0 + threadIdx.x; i < r1; i += kGsThreads) {
            const double wi = w[i];
#pragma unroll
            for (int c = 0; c < kGsGroup; ++c) v[c] = fma(V[c * a.ldv + i], wi, v[c]);
        }
    } else {
#pragma unroll 2
        for (long i = r0 + threadIdx.x; i < r1; i += kGsThreads) {
            const double wi = w[i];
#pragma unroll
            for (int c = 0; c < kGsGroup; ++c)
                if (c < nc) v[c] = fma(V[c * a.ldv + i], wi, v[c]);
        }
    }
    // lane bit 4, 3, 2 selects the upper half of the columns still held
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
    for (int h = kGsGroup / 2, o = 16; h > 0; h >>= 1, o >>= 1) {
        const bool up = lane & o;
#pragma unroll
        for (int c = 0; c < h; ++c) {
            const double send = up ? v[c] : v[c + h];
            v[c] = (up ? v[c + h] : v[c]) + __shfl_xor_sync(0xffffffffu, send, o);
        }
    }
    v[0] += __shfl_xor_sync(0xffffffffu, v[0], 2);
    v[0] += __shfl_xor_sync(0xffffffffu, v[0], 1);
    __shared__ double red[kGsGroup][kGsThreads / 32];
    // bit 4 of the lane picked columns 4..7, bit 3 the upper two, bit 2 the upper one
    if ((lane & 3) == 0) red[lane >> 2][warp] = v[0];
    __syncthreads();
    if (threadIdx.x < nc) {
        double s = 0.0;
        for (int k = 0; k < kGsThreads / 32; ++k) s += red[threadIdx.x][k];
        partial[((long)blockIdx.z * gridDim.x + blockIdx.x) * ldp + c0 + threadIdx.x] = s;
    }
}

// out[c] = sum_b partial[b * ldp + c] for c < j, over many blocks: each block
// takes 32 columns, its warps sum interleaved rows of partials, and warp 0
// adds the warp sums in a fixed order (bit-reproducible run to run).
// member blockIdx.y: partial + member * nb * ldp, out + member * ldo; js
// (optional) gives a per-member column count (<= 0: member skipped).
__global__ void k_gs_reduce_par(const double* __restrict__ partial, int nb, int ldp, int j,
                                const int* __restrict__ js, double* __restrict__ out, int ldo) {
    const int b = blockIdx.y;
    if (js) j = js[b];
    const int lane = threadIdx.x & 31, wv = threadIdx.x >> 5, nw = blockDim.x >> 5;
    const int c = blockIdx.x * 32 + lane;
    if (j <= 0 || blockIdx.x * 32 >= j) return;
    partial += (size_t)b * nb * ldp;
    __shared__ double red[32][33];
    double s = 0.0;
    if (c < j)
        for (int r = wv; r < nb; r += nw) s += partial[(long)r * ldp + c];
    red[wv][lane] = s;
    __syncthreads();
    if (wv == 0 && c < j) {
        double t = 0.0;
        for (int w = 0; w < nw; ++w) t += red[w][lane];
        out[(size_t)b * ldo + c] = t;
    }
}

// w[i] -= sum_c V[c][i] h[c]; NORM: also normp[b gridDim.x + x] = block x's
// share of sum w[i]^2 (j = 0: only that).  h: the member's row of `h`, or with
// nsum > 0 the sum of the nsum rows of `partial` (which block 0 stores to h).
// PARTS threads share a row, each a part of the columns, so that a short
// vector still fills the chip (n = 8192: 256 blocks instead of 32).
template <int PARTS, bool NORM>
__global__ void __launch_bounds__(kGsThreads) k_gs_update(GsArgs a, double* __restrict__ h, int ldh,
                                                          const double* __restrict__ partial, int nsum, int ldp,
                                                          double* __restrict__ normp) {
    constexpr int ROWS = kGsThreads / PARTS;
    extern __shared__ double hs[];
    __shared__ double red[kGsThreads];
    if (!gs_member(a, blockIdx.y) || (!NORM && a.j == 0)) return;
    h += (long)blockIdx.y * ldh;
    for (int c = threadIdx.x; c < a.j; c += kGsThreads) {
        double s = 0.0;
        if (nsum > 0) {
            for (int r = 0; r < nsum; ++r) s += partial[((long)blockIdx.y * nsum + r) * ldp + c];
            if (blockIdx.x == 0) h[c] = s;
        } else {
            s = h[c];
        }
        hs[c] = s;
    }
    __syncthreads();
    const int part = threadIdx.x / ROWS, row = threadIdx.x % ROWS;
    const int p0 = part * a.j / PARTS, p1 = (part + 1) * a.j / PARTS;
    double nrm = 0.0;
    for (long i0 = (long)blockIdx.x * ROWS; i0 < a.n; i0 += (long)gridDim.x * ROWS) {
        const long i = i0 + row;
        double acc = 0.0;
        if (i < a.n && a.j > 0) {
            const double* __restrict__ V = a.V + i;
            double acc2 = 0.0;
            int c = p0;
            for (; c + 8 <= p1; c += 8) {   // eight loads in flight
                double x[8];
#pragma unroll
                for (int q = 0; q < 8; ++q) x[q] = V[(long)(c + q) * a.ldv];
#pragma unroll
                for (int q = 0; q < 8; q += 2) {
                    acc = fma(x[q], hs[c + q], acc);
                    acc2 = fma(x[q + 1], hs[c + q + 1], acc2);
                }
            }
            for (; c < p1; ++c) acc = fma(V[(long)c * a.ldv], hs[c], acc);
            acc += acc2;
        }
        if (PARTS > 1) {
            red[threadIdx.x] = acc;
            __syncthreads();
            if (part == 0) {
#pragma unroll
                for (int q = 1; q < PARTS; ++q) acc += red[q * ROWS + row];
            }
            __syncthreads();
        }
        if (part == 0 && i < a.n) {
            const double x = a.w[i] - acc;
            if (a.j > 0) a.w[i] = x;
            if (NORM) nrm = fma(x, x, nrm);
        }
    }
    if (NORM) {
        for (int o = 16; o > 0; o >>= 1) nrm += __shfl_down_sync(0xffffffffu, nrm, o);
        if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = nrm;
        __syncthreads();
        if (threadIdx.x == 0) {
            double s = 0.0;
            for (int k = 0; k < kGsThreads / 32; ++k) s += red[k];
            normp[(long)blockIdx.y * gridDim.x + blockIdx.x] = s;
        }
    }
}

// Row chunks of the dot products of nmem members of up to j columns and n
// rows: eight blocks an SM over all members and column groups, at least four
// rows a thread.
static int gs_chunks(int nmem, int j, long n) {
    const int ncg = std::max(1, (j + kGsGroup - 1) / kGsGroup);
    const long want = (kGsGrid + (long)ncg * nmem - 1) / ((long)ncg * nmem);
    return (int)std::max<long>(1, std::min<long>(want, (n + 4 * kGsThreads - 1) / (4 * kGsThreads)));
}

int gs_norm_blocks(int nmem, long n) {
    return (int)std::max<long>(1, std::min<long>(std::max(16, kGsGrid / nmem), (n + 31) / 32));
}

template <bool NORM>
static void launch_update(const GsArgs& a, int nmem, int j, long n, double* h, int ldh, const double* partial, int nsum,
                          int ldp, double* normp, cudaStream_t stream) {
    // eight threads a row where one a row gives fewer than four blocks an SM
    const bool parts = (n + kGsThreads - 1) / kGsThreads * nmem < 4 * 152;
    const size_t sm = (size_t)std::max(j, 1) * sizeof(double);
    const dim3 g(gs_norm_blocks(nmem, n), nmem);
    if (parts) k_gs_update<8, NORM><<<g, kGsThreads, sm, stream>>>(a, h, ldh, partial, nsum, ldp, normp);
    else k_gs_update<1, NORM><<<g, kGsThreads, sm, stream>>>(a, h, ldh, partial, nsum, ldp, normp);
}

// The launches of one CGS2 over nmem members (at most j columns and n rows):
// h1, h2 (row stride ldh) and the partial sums of ||w||^2, gs_norm_blocks per
// member.  The second update also sums the squares of what it writes.  Few
// partial sums (short vectors) are added by the update that consumes them,
// which saves a launch of about 3 us.
int gs_passes(const GsArgs& a, int nmem, int j, long n, double* partial, double* h1, double* h2, int ldh, double* normp,
              cudaStream_t stream) {
    const int nbx = gs_chunks(nmem, j, n), ldp = j, nsum = nbx <= 16 ? nbx : 0;
    for (int pass = 0; pass < 2 && j > 0; ++pass) {
        double* h = pass ? h2 : h1;
        k_gs_dot<<<dim3(nbx, (j + kGsGroup - 1) / kGsGroup, nmem), kGsThreads, 0, stream>>>(a, partial, ldp);
        if (nsum == 0)
            k_gs_reduce_par<<<dim3((j + 31) / 32, nmem), 1024, 0, stream>>>(partial, nbx, ldp, j, a.js, h, ldh);
        if (pass == 0) launch_update<false>(a, nmem, j, n, h, ldh, partial, nsum, ldp, nullptr, stream);
        else launch_update<true>(a, nmem, j, n, h, ldh, partial, nsum, ldp, normp, stream);
    }
    if (j <= 0) launch_update<true>(a, nmem, 0, n, h1, ldh, partial, 0, 1, normp, stream);
    NS_LAUNCH_CHECK();
    return NSSTAB_OK;
}

// partial sums of a CGS2 over nmem members of up to j columns
static size_t gs_partial_len(int nmem, int j) { return (size_t)kGsGrid * kGsGroup + (size_t)nmem * (j + kGsGroup); }
static size_t gs_norm_len(int nmem) { return (size_t)kGsGrid + 16 * (size_t)nmem; }

// dst = a x + b y (dst may alias x or y)
__global__ void k_axpby(double* dst, double a, const double* x, double b, const double* y, long n) {
    for (long i = (long)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (long)gridDim.x * blockDim.x)
        dst[i] = a * x[i] + b * y[i];
}

__global__ void k_scale(double* __restrict__ dst, const double* __restrict__ src, long n, double s) {
    for (long i = (long)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (long)gridDim.x * blockDim.x)
        dst[i] = src[i] * s;
}

// out[c][i] = sum_k V[k][i] C[c*ldc + k], c < p  (out must not alias V)
__global__ void k_combine(const double* __restrict__ V, long ldv, long n, int m, const double* __restrict__ C,
                          int ldc, int p, double* __restrict__ out, long ldo) {
    const int G = 8;
    for (long i = (long)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (long)gridDim.x * blockDim.x) {
        for (int c0 = 0; c0 < p; c0 += G) {
            double acc[G];
#pragma unroll
            for (int g = 0; g < G; ++g) acc[g] = 0.0;
            for (int k = 0; k < m; ++k) {
                const double v = V[(long)k * ldv + i];
#pragma unroll
                for (int g = 0; g < G; ++g)
                    if (c0 + g < p) acc[g] = fma(v, __ldg(C + (long)(c0 + g) * ldc + k), acc[g]);
            }
#pragma unroll
            for (int g = 0; g < G; ++g)
                if (c0 + g < p) out[(long)(c0 + g) * ldo + i] = acc[g];
        }
    }
}

// ----------------------------------------------------- batched variants
// Member b (blockIdx.y) works on its own basis V[b] (column-major, leading
// dimension ldv), vector w[b] and column count j[b]; j[b] <= 0 leaves w[b]
// alone in the products (the norm pass uses its own count array).

__global__ void k_scale_b(double* const* __restrict__ ws, long n, const double* __restrict__ s,
                          const long* __restrict__ ns) {
    double* w = ws[blockIdx.y];
    if (!w) return;
    if (ns) n = ns[blockIdx.y];
    const double f = s[blockIdx.y];
    for (long i = (long)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (long)gridDim.x * blockDim.x) w[i] *= f;
}

// ------------------------------------------------ blocked Gram-Schmidt
// Block form of the Gram-Schmidt step for block Krylov methods: the b new
// columns W of a set are projected against its first J orthonormal basis
// columns in one tall-skinny product pair, H = V_J^T W (J x b) and
// W -= V_J H, so V is read once per pass for all b columns instead of once
// per column.  Set s = blockIdx.z (dot) / blockIdx.y (update); J[s] <= 0
// skips the set.  W's columns are ldw apart; H is stored [c * b + q].

static const int kBgsCols = 4;   // basis columns per block row of the dot product

// partial[s][blk][c * B + q] = sum over block blk's row range of V[c][i] W[q][i],
// for the kBgsCols columns c of block row blockIdx.y
template <int B>
__global__ void __launch_bounds__(256) k_bgs_dot(const double* const* __restrict__ Vs, long ldv, long n,
                                                 const int* __restrict__ Js, const double* const* __restrict__ Ws,
                                                 long ldw, double* __restrict__ partial, int ldp) {
    const int s = blockIdx.z;
    const int J = Js[s];
    const int c0 = blockIdx.y * kBgsCols;
    if (J <= 0 || c0 >= J) return;
    const double* V = Vs[s];
    const double* W = Ws[s];
    const long chunk = (n + gridDim.x - 1) / gridDim.x;
    const long r0 = (long)blockIdx.x * chunk;
    const long r1 = min(n, r0 + chunk);
    const int nc = min(kBgsCols, J - c0);
    double acc[kBgsCols][B];
#pragma unroll
    for (int cc = 0; cc < kBgsCols; ++cc)
#pragma unroll
        for (int q = 0; q < B; ++q) acc[cc][q] = 0.0;
    for (long i = r0 + threadIdx.x; i < r1; i += blockDim.x) {
        double w[B];
#pragma unroll
        for (int q = 0; q < B; ++q) w[q] = W[(long)q * ldw + i];
#pragma unroll
        for (int cc = 0; cc < kBgsCols; ++cc) {
            if (cc < nc) {
                const double v = V[(long)(c0 + cc) * ldv + i];
#pragma unroll
                for (int q = 0; q < B; ++q) acc[cc][q] = fma(v, w[q], acc[cc][q]);
            }
        }
    }
    __shared__ double red[kBgsCols * B][8];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
    for (int cc = 0; cc < kBgsCols; ++cc)
#pragma unroll
        for (int q = 0; q < B; ++q) {
            double a = acc[cc][q];
            for (int o = 16; o > 0; o >>= 1) a += __shfl_down_sync(0xffffffffu, a, o);
            if (lane == 0) red[cc * B + q][warp] = a;
        }
    __syncthreads();
    const int t = threadIdx.x;
    if (t < nc * B) {
        double sum = 0.0;
        for (int wv = 0; wv < (int)(blockDim.x >> 5); ++wv) sum += red[t][wv];
        partial[((size_t)s * gridDim.x + blockIdx.x) * ldp + (size_t)c0 * B + t] = sum;
    }
}

// W[q][i] -= sum_c V[c][i] H[c * B + q]
template <int B>
__global__ void __launch_bounds__(256) k_bgs_update(double* const* __restrict__ Ws, long ldw,
                                                    const double* const* __restrict__ Vs, long ldv, long n,
                                                    const int* __restrict__ Js, const double* __restrict__ H,
                                                    int ldh) {
    const int s = blockIdx.y;
    const int J = Js[s];
    if (J <= 0) return;
    extern __shared__ double hs[];
    for (int e = threadIdx.x; e < J * B; e += blockDim.x) hs[e] = H[(size_t)s * ldh + e];
    __syncthreads();
    double* W = Ws[s];
    const double* V = Vs[s];
    for (long i = (long)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (long)gridDim.x * blockDim.x) {
        double acc[B];
#pragma unroll
        for (int q = 0; q < B; ++q) acc[q] = 0.0;
        for (int c = 0; c < J; ++c) {
            const double v = V[(long)c * ldv + i];
#pragma unroll
            for (int q = 0; q < B; ++q) acc[q] = fma(v, hs[c * B + q], acc[q]);
        }
#pragma unroll
        for (int q = 0; q < B; ++q) W[(long)q * ldw + i] -= acc[q];
    }
}

template <int B>
static int bgs_pass(int S, const double* const* Vd, long ldv, long n, const int* Jd, int Jmax, double* const* Wd,
                    long ldw, double* partial, int nbx, int ldp, double* Hout, cudaStream_t stream) {
    const dim3 gd(nbx, (Jmax + kBgsCols - 1) / kBgsCols, S);
    k_bgs_dot<B><<<gd, 256, 0, stream>>>(Vd, ldv, n, Jd, (const double* const*)Wd, ldw, partial, ldp);
    k_gs_reduce_par<<<dim3((Jmax * B + 31) / 32, S), 256, 0, stream>>>(partial, nbx, ldp, Jmax * B, nullptr, Hout,
                                                                        ldp);
    const int ub = std::max(16, 4 * 152 / S);
    k_bgs_update<B><<<dim3(ub, S), 256, (size_t)Jmax * B * sizeof(double), stream>>>(Wd, ldw, Vd, ldv, n, Jd,
                                                                                      Hout, ldp);
    NS_LAUNCH_CHECK();
    return NSSTAB_OK;
}

int bcgs2_batch(int S, const double* const* V, long ldv, long n, const int* J, double* const* W, long ldw, int b,
                double* H, int ldh, GsBatch& ws, cudaStream_t stream) {
    if (b < 1 || b > kMaxGsBlock) {
        set_error("block Gram-Schmidt: block size out of range");
        return NSSTAB_ERR_INVALID_ARG;
    }
    int Jmax = 0;
    for (int s = 0; s < S; ++s) Jmax = std::max(Jmax, J[s]);
    if (Jmax <= 0) return NSSTAB_OK;
    const int ldp = Jmax * b;
    NS_TRY(ws.alloc(S, ldp));
    std::vector<int> jh(S);
    std::vector<const double*> ph(2 * (size_t)S);
    for (int s = 0; s < S; ++s) {
        jh[s] = J[s];
        ph[s] = V[s];
        ph[S + s] = W[s];
    }
    NS_CUDA(cudaMemcpyAsync(ws.jdev, jh.data(), S * sizeof(int), cudaMemcpyHostToDevice, stream));
    NS_CUDA(cudaMemcpyAsync(ws.ptrs, ph.data(), ph.size() * sizeof(double*), cudaMemcpyHostToDevice, stream));
    const double* const* Vd = (const double* const*)ws.ptrs;
    double* const* Wd = ws.ptrs + S;
    // partial sums [S][nbx][ldp] fit the workspace's [S][grid][max_cols]
    const int rows_of_blocks = (Jmax + kBgsCols - 1) / kBgsCols;
    const int nbx = std::max(8, std::min(ws.grid, 4 * 152 / std::max(1, rows_of_blocks * S)));
    double* h1 = ws.hdev;
    double* h2 = ws.hdev + (size_t)S * ldp;
#define NS_BGS(BB)                                                                                          \
    do {                                                                                                    \
        NS_TRY(bgs_pass<BB>(S, Vd, ldv, n, ws.jdev, Jmax, Wd, ldw, ws.partial, nbx, ldp, h1, stream));      \
        NS_TRY(bgs_pass<BB>(S, Vd, ldv, n, ws.jdev, Jmax, Wd, ldw, ws.partial, nbx, ldp, h2, stream));      \
    } while (0)
    switch (b) {
        case 1: NS_BGS(1); break;
        case 2: NS_BGS(2); break;
        case 3: NS_BGS(3); break;
        case 4: NS_BGS(4); break;
        case 5: NS_BGS(5); break;
        case 6: NS_BGS(6); break;
        case 7: NS_BGS(7); break;
        default: NS_BGS(8); break;
    }
#undef NS_BGS
    NS_CUDA(cudaMemcpyAsync(ws.hhost, ws.hdev, (size_t)2 * S * ldp * sizeof(double), cudaMemcpyDeviceToHost,
                            stream));
    NS_CUDA(cudaStreamSynchronize(stream));
    for (int s = 0; s < S; ++s)
        for (int e = 0; e < J[s] * b; ++e)
            H[(size_t)s * ldh + e] = ws.hhost[(size_t)s * ldp + e] + ws.hhost[(size_t)(S + s) * ldp + e];
    return NSSTAB_OK;
}

int GsBatch::alloc(int nmem, int cols) {
    if (nmem <= B && cols <= max_cols) return NSSTAB_OK;
    release();
    B = nmem;
    max_cols = cols;
    grid = 152;
    const size_t ph = (size_t)B * 2 * max_cols + gs_norm_len(B);
    NS_CUDA(cudaMalloc(&partial, std::max((size_t)B * grid * max_cols, gs_partial_len(B, max_cols)) * sizeof(double)));
    NS_CUDA(cudaMalloc(&hdev, ph * sizeof(double)));
    NS_CUDA(cudaMalloc(&jdev, (size_t)B * sizeof(int)));
    NS_CUDA(cudaMalloc(&ptrs, (size_t)B * 2 * sizeof(double*)));
    NS_CUDA(cudaMalloc(&sdev, (size_t)B * sizeof(double)));
    NS_CUDA(cudaMalloc(&ndev, (size_t)B * sizeof(long)));
    NS_CUDA(cudaMallocHost(&hhost, ph * sizeof(double)));
    return NSSTAB_OK;
}

void GsBatch::release() {
    if (partial) cudaFree(partial);
    if (hdev) cudaFree(hdev);
    if (jdev) cudaFree(jdev);
    if (ptrs) cudaFree(ptrs);
    if (sdev) cudaFree(sdev);
    if (ndev) cudaFree(ndev);
    if (hhost) cudaFreeHost(hhost);
    partial = hdev = sdev = hhost = nullptr;
    ndev = nullptr;
    jdev = nullptr;
    ptrs = nullptr;
    B = max_cols = 0;
}

// CGS2 of w[b] against the first j[b] columns of V[b] for every member with
// j[b] >= 0 (j[b] = 0: norm only; j[b] < 0: member skipped); h[b][0..j[b])
// and beta[b] = ||w[b]|| to the host.  One synchronisation.
int cgs2_batch(int nmem, const double* const* V, long ldv, long n, const int* j, double* const* w,
               double* h /*host [nmem][ldh]*/, int ldh, double* beta, GsBatch& ws, cudaStream_t stream,
               const long* nm) {
    int jmax = 0;
    for (int b = 0; b < nmem; ++b) jmax = std::max(jmax, j[b]);
    NS_TRY(ws.alloc(nmem, std::max(jmax, 1)));
    const long* nd = nullptr;
    if (nm) {
        NS_CUDA(cudaMemcpyAsync(ws.ndev, nm, nmem * sizeof(long), cudaMemcpyHostToDevice, stream));
        nd = ws.ndev;
    }
    std::vector<const double*> ph(2 * (size_t)nmem);
    for (int b = 0; b < nmem; ++b) {
        ph[b] = V[b];
        ph[nmem + b] = w[b];
    }
    NS_CUDA(cudaMemcpyAsync(ws.jdev, j, nmem * sizeof(int), cudaMemcpyHostToDevice, stream));
    NS_CUDA(cudaMemcpyAsync(ws.ptrs, ph.data(), ph.size() * sizeof(double*), cudaMemcpyHostToDevice, stream));
    GsArgs a{};
    a.Vs = (const double* const*)ws.ptrs;
    a.ws = ws.ptrs + nmem;
    a.js = ws.jdev;
    a.ns = nd;
    a.ldv = ldv;
    a.n = n;
    double* h1 = ws.hdev;
    double* h2 = h1 + (size_t)nmem * jmax;
    double* normp = h2 + (size_t)nmem * jmax;
    const int nnorm = gs_norm_blocks(nmem, n);
    NS_TRY(gs_passes(a, nmem, jmax, n, ws.partial, h1, h2, jmax, normp, stream));
    NS_CUDA(cudaMemcpyAsync(ws.hhost, ws.hdev, ((size_t)2 * nmem * jmax + (size_t)nmem * nnorm) * sizeof(double),
                            cudaMemcpyDeviceToHost, stream));
    NS_CUDA(cudaStreamSynchronize(stream));
    for (int b = 0; b < nmem; ++b) {
        if (j[b] < 0) continue;
        for (int c = 0; c < j[b]; ++c)
            h[(size_t)b * ldh + c] = ws.hhost[(size_t)b * jmax + c] + ws.hhost[(size_t)(nmem + b) * jmax + c];
        double s = 0.0;
        for (int k = 0; k < nnorm; ++k) s += ws.hhost[(size_t)2 * nmem * jmax + (size_t)b * nnorm + k];
        beta[b] = std::sqrt(s);
    }
    return NSSTAB_OK;
}

// w[b] *= s[b] for members with a non-null w[b]
int scale_batch(int nmem, double* const* w, long n, const double* s, GsBatch& ws, cudaStream_t stream,
                const long* nm) {
    NS_TRY(ws.alloc(nmem, 1));
    const long* nd = nullptr;
    if (nm) {
        NS_CUDA(cudaMemcpyAsync(ws.ndev, nm, nmem * sizeof(long), cudaMemcpyHostToDevice, stream));
        nd = ws.ndev;
    }
    std::vector<double*> ph(w, w + nmem);
    NS_CUDA(cudaMemcpyAsync(ws.ptrs, ph.data(), nmem * sizeof(double*), cudaMemcpyHostToDevice, stream));
    std::vector<double> sh(s, s + nmem);
    NS_CUDA(cudaMemcpyAsync(ws.sdev, sh.data(), nmem * sizeof(double), cudaMemcpyHostToDevice, stream));
    k_scale_b<<<dim3(ws.grid, nmem), kGsThreads, 0, stream>>>(ws.ptrs, n, ws.sdev, nd);
    NS_LAUNCH_CHECK();
    return NSSTAB_OK;
}

int GsWork::alloc(int max_cols_) {
    if (max_cols_ <= max_cols) return NSSTAB_OK;
    release();
    max_cols = max_cols_;
    const size_t ph = (size_t)2 * max_cols + gs_norm_len(1);
    NS_CUDA(cudaMalloc(&partial, gs_partial_len(1, max_cols) * sizeof(double)));
    NS_CUDA(cudaMalloc(&hdev, ph * sizeof(double)));
    NS_CUDA(cudaMallocHost(&hhost, ph * sizeof(double)));
    return NSSTAB_OK;
}

void GsWork::release() {
    if (partial) cudaFree(partial);
    if (hdev) cudaFree(hdev);
    if (hhost) cudaFreeHost(hhost);
    partial = hdev = hhost = nullptr;
    max_cols = 0;
}

int cgs2(const double* V, long ldv, long n, int j, double* w, double* h, double* beta, GsWork& ws,
         cudaStream_t stream) {
    NS_TRY(ws.alloc(std::max(j, 1)));
    GsArgs a{};
    a.V = V;
    a.w = w;
    a.ldv = ldv;
    a.n = n;
    a.j = j;
    double* normp = ws.hdev + 2 * (size_t)j;
    const int nnorm = gs_norm_blocks(1, n);
    NS_TRY(gs_passes(a, 1, j, n, ws.partial, ws.hdev, ws.hdev + j, j, normp, stream));
    NS_CUDA(cudaMemcpyAsync(ws.hhost, ws.hdev, ((size_t)2 * j + nnorm) * sizeof(double), cudaMemcpyDeviceToHost,
                            stream));
    NS_CUDA(cudaStreamSynchronize(stream));
    for (int c = 0; c < j; ++c) h[c] = ws.hhost[c] + ws.hhost[j + c];
    double s = 0.0;
    for (int k = 0; k < nnorm; ++k) s += ws.hhost[2 * j + k];
    *beta = std::sqrt(s);
    return NSSTAB_OK;
}

int vec_norm(const double* x, long n, double* out, GsWork& ws, cudaStream_t stream) {
    return cgs2(nullptr, n, n, 0, const_cast<double*>(x), nullptr, out, ws, stream);   // j = 0 writes nothing
}

int vec_axpby(double* dst, double a, const double* x, double b, const double* y, long n, cudaStream_t stream) {
    k_axpby<<<304, kGsThreads, 0, stream>>>(dst, a, x, b, y, n);
    NS_LAUNCH_CHECK();
    return NSSTAB_OK;
}

int vec_scale(double* dst, const double* src, long n, double s, cudaStream_t stream) {
    k_scale<<<304, kGsThreads, 0, stream>>>(dst, src, n, s);
    NS_LAUNCH_CHECK();
    return NSSTAB_OK;
}

int basis_combine(const double* V, long ldv, long n, int m, const double* C_dev, int p, double* out, long ldo,
                  cudaStream_t stream) {
    k_combine<<<608, 128, 0, stream>>>(V, ldv, n, m, C_dev, m, p, out, ldo);
    NS_LAUNCH_CHECK();
    return NSSTAB_OK;
}

}  // namespace nsstab
