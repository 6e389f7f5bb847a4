// The learned initial guess for the Newton-Krylov base-flow solve: a
// 4-level U-Net (declared in include/nsstab.h; the paper has no network).
//
// Storage: activations in bfloat16, channels innermost ([B][H][W][C]), so
// the channels of one point are one contiguous run; weights as FP32 masters
// (with Adam's moments) plus a bfloat16 copy that the convolutions read;
// every sum in FP32; gradients of activations in FP32 (bfloat16 hi + lo
// planes where a GEMM reads them).
//
// Kernels (one pass each, no im2col buffer; implicit GEMMs on the tensor
// cores, BF16 mma.sync, FP32 accumulate):
//   k_conv_halo<false>  3x3 periodic convolution + bias + ReLU by patches of
//                       128 points with their halo; the 2x2 pooling or the
//                       1x1 output layer after it in its epilogue; the level
//                       below and the skip read in place of a concatenation
//   k_conv_halo<true>   gradient of the input: the same GEMM with the
//                       channels exchanged and the taps mirrored; that of a
//                       ReLU output leaves as bfloat16 hi + lo planes
//   k_conv_bwd_w_halo   gradient of the weights and bias: per tap a GEMM
//                       reduced over points, split over the blocks of
//                       clusters, atomicAdd into the FP32 gradient
//   the adjoints of pooling and concatenation, the mean-squared loss, the
//   output layer's gradient and Adam are pointwise kernels.
// Where the patches do not apply (halo_shape: a level too small for them;
// channel counts that do not come in eights, 16-byte misaligned weights) the
// same steps are k_conv_gemm<false>, k_conv_gemm<true> and k_conv_bwd_w, one
// tap's rows a stage, with k_pool, k_up_cat, k_out_fwd and k_relu_split as
// passes of their own.
// The layer sequence and every rounding point follow the oracle's
// definition of the network (the same flat parameter layout).
#include <cooperative_groups.h>
#include <cuda_bf16.h>

#include <cmath>
#include <cstdint>
#include <initializer_list>
#include <string>
#include <vector>

#include "common.cuh"

namespace nsstab {
namespace {

using bf16 = __nv_bfloat16;
namespace cg = cooperative_groups;
constexpr int kLevels = 4;

struct ConvDesc {
    int ci = 0, co = 0, k = 3;   // k = 3 (3x3) or 1 (the output layer)
    long w_off = 0, b_off = 0;   // offsets into the flat parameter vector
};

// Neighbour (y + dy, x + dx) of point p = (b, y, x) on the periodic
// 2^lh x 2^lw grid.
__device__ __forceinline__ long nbr(long p, int lh, int lw, int dy, int dx) {
    const int W = 1 << lw, H = 1 << lh;
    const int x = (int)(p & (W - 1));
    const int y = (int)((p >> lw) & (H - 1));
    const long b = p >> (lw + lh);
    return (((b << lh) + ((y + dy) & (H - 1))) << lw) + ((x + dx) & (W - 1));
}

// ---------------------------------------------------------------------------
// The three 3x3 convolutions are implicit GEMMs on the tensor cores (BF16
// mma.sync m16n8k16, FP32 accumulation; products of bfloat16 values are
// exact in FP32, so only the order of the FP32 sums differs from a scalar
// loop).  Operands reach shared memory by 16-byte cp.async copies (VEC: all
// channel counts multiples of 8 and 16-byte aligned bases; otherwise plain
// loads), in a ring of pipeline stages, and reach the registers by ldmatrix.
// Every tile row is padded to 40 bf16 (80 bytes), which makes the ldmatrix
// reads of a warp hit 32 distinct banks.
//
// The FP32 gradient of a ReLU output enters as two bfloat16 planes
// (hi = bf16(g), lo = bf16(g - hi), written by k_relu_split), two mma steps
// per fragment: about 16 significant bits of every product, summed in FP32.
//
// The bfloat16 weight copy wt is tap-major, wt[tap][co][ci], so that a tile
// of (output, input) channels of one tap is a set of contiguous rows for
// either GEMM that reads it.
// ---------------------------------------------------------------------------
constexpr int kMmaCo = 32, kMmaK = 16;
constexpr int kStr = 40;            // padded tile row (bf16)
constexpr int kTilePts = 64;        // points per block in the forward and input-gradient GEMMs
constexpr int kRing = 4;            // pipeline depth of those GEMMs

__device__ __forceinline__ void mma_bf16(float* d, uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint32_t b0,
                                         uint32_t b1) {
    asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, "
                 "{%0,%1,%2,%3};"
                 : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
                 : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}

__device__ __forceinline__ uint32_t smem_u32(const void* p) {
    return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}
__device__ __forceinline__ void ldsm_x4(uint32_t addr, uint32_t& r0, uint32_t& r1, uint32_t& r2, uint32_t& r3) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];"
                 : "=r"(r0), "=r"(r1), "=r"(r2), "=r"(r3)
                 : "r"(addr));
}
__device__ __forceinline__ void ldsm_x4_t(uint32_t addr, uint32_t& r0, uint32_t& r1, uint32_t& r2, uint32_t& r3) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];"
                 : "=r"(r0), "=r"(r1), "=r"(r2), "=r"(r3)
                 : "r"(addr));
}
__device__ __forceinline__ void ldsm_x2(uint32_t addr, uint32_t& r0, uint32_t& r1) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x2.shared.b16 {%0,%1}, [%2];" : "=r"(r0), "=r"(r1) : "r"(addr));
}
__device__ __forceinline__ void ldsm_x2_t(uint32_t addr, uint32_t& r0, uint32_t& r1) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x2.trans.shared.b16 {%0,%1}, [%2];" : "=r"(r0), "=r"(r1) : "r"(addr));
}
// 16-byte global -> shared copy; src_bytes = 0 writes zeros
__device__ __forceinline__ void cp_async16(uint32_t dst, const void* src, int src_bytes) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(src_bytes));
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;"); }
template <int N>
__device__ __forceinline__ void cp_async_wait() {
    asm volatile("cp.async.wait_group %0;" ::"n"(N));
}

// rows x 32 channels of a [row][LD] bfloat16 array (C channels used) into a
// padded tile: row r of the tile is src_row(r) (negative: zeros), channels
// c0 .. c0 + 31 (zeros at and beyond C; VEC copies whole 8-channel groups,
// so channels C .. LD - 1 must hold zeros).  NT threads share the work.
template <bool VEC, int ROWS, int NT, class RowFn>
__device__ __forceinline__ void stage_rows(bf16 (*tile)[kStr], const bf16* __restrict__ base, int C, int LD, int c0,
                                           RowFn src_row) {
    if (VEC) {
#pragma unroll
        for (int i = 0; i < (ROWS * 4 + NT - 1) / NT; ++i) {
            const int f = threadIdx.x + i * NT;
            if (ROWS * 4 % NT != 0 && f >= ROWS * 4) break;
            const int r = f >> 2, g = f & 3;
            const long row = src_row(r);
            const bool ok = row >= 0 && c0 + 8 * g < C;
            cp_async16(smem_u32(&tile[r][8 * g]), ok ? base + row * LD + c0 + 8 * g : base, ok ? 16 : 0);
        }
    } else {
#pragma unroll 4
        for (int i = 0; i < (ROWS * kMmaCo + NT - 1) / NT; ++i) {
            const int f = threadIdx.x + i * NT;
            if (ROWS * kMmaCo % NT != 0 && f >= ROWS * kMmaCo) break;
            const int r = f / kMmaCo, c = f % kMmaCo;
            const long row = src_row(r);
            tile[r][c] = (row >= 0 && c0 + c < C) ? base[row * LD + c0 + c] : __float2bfloat16_rn(0.f);
        }
    }
}

// Forward (BWD = false): out[p][co] = relu(bias[co] + sum_{tap, ci}
//   wt[tap][co][ci] in[nbr(p, tap)][ci]) in bfloat16; rows = points,
//   columns = output channels, reduction = (tap, input channel).
// Input gradient (BWD = true): gin[q][ci] = sum_{tap, co} wt[tap][co][ci]
//   gz[q - tap offset][co] in FP32; rows = points, columns = input channels,
//   reduction = (tap, output channel), A = the gradient's hi and lo planes.
// A block of 4 warps owns 64 points x 32 columns (warp w: points 16 w .. +15,
// all 32 columns); one pipeline stage is one tap and 32 reduction channels.
// VA / VB: 16-byte copies for the A rows (row stride lda) / the weight rows.
template <bool BWD, bool VA, bool VB>
__global__ void __launch_bounds__(128) k_conv_gemm(const bf16* __restrict__ a_hi, const bf16* __restrict__ a_lo,
                                                   const bf16* __restrict__ wt, const float* __restrict__ bias,
                                                   void* __restrict__ out, long P, int lh, int lw, int Ci, int Co,
                                                   int lda) {
    constexpr int NP = BWD ? 2 : 1;   // A planes
    struct Stage {
        bf16 a[NP][kTilePts][kStr];
        bf16 b[kMmaCo][kStr];   // forward: [co][ci]; input gradient: [co][ci] read transposed
    };
    extern __shared__ __align__(16) unsigned char smem[];
    Stage* ring = reinterpret_cast<Stage*>(smem);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int Ck = BWD ? Co : Ci;   // reduction channels per tap
    const int Cn = BWD ? Ci : Co;   // output columns
    const long pb = (long)blockIdx.x * kTilePts;
    const int n0 = blockIdx.y * kMmaCo;
    const int nck = (Ck + kMmaCo - 1) / kMmaCo;
    const int nst = 9 * nck;
    auto issue = [&](int s) {
        Stage& st = ring[s % kRing];
        const int t = s % 9, kc = (s / 9) * kMmaCo;
        const int dy = BWD ? 1 - t / 3 : t / 3 - 1, dx = BWD ? 1 - t % 3 : t % 3 - 1;
        auto arow = [&](int r) -> long {
            const long p = pb + r;
            return p < P ? nbr(p, lh, lw, dy, dx) : -1;
        };
#pragma unroll
        for (int h = 0; h < NP; ++h) stage_rows<VA, kTilePts, 128>(st.a[h], h ? a_lo : a_hi, Ck, lda, kc, arow);
        if (BWD) {   // rows = output channels kc .. kc + 31 (reduction), columns = input channels
            stage_rows<VB, kMmaCo, 128>(st.b, wt + (long)t * Co * Ci, Ci, Ci, n0, [&](int r) -> long {
                return kc + r < Co ? (long)(kc + r) : -1;
            });
        } else {     // rows = output channels n0 .. n0 + 31 (columns), columns = input channels
            stage_rows<VB, kMmaCo, 128>(st.b, wt + (long)t * Co * Ci, Ci, Ci, kc, [&](int r) -> long {
                return n0 + r < Co ? (long)(n0 + r) : -1;
            });
        }
    };
    float acc[4][4];
#pragma unroll
    for (int j = 0; j < 4; ++j)
#pragma unroll
        for (int r = 0; r < 4; ++r) acc[j][r] = 0.f;
    // ldmatrix: lane = 8 i + r supplies row r of 8x8 matrix i
    const int lr = lane & 7, li = lane >> 3;
    const int a_m = warp * 16 + (li & 1) * 8 + lr, a_k = (li >> 1) * 8;        // A [point][k]
    const int bf_n = (li >> 1) * 8 + lr, bf_k = (li & 1) * 8;                  // forward B [n][k]
    const int bb_k = (li & 1) * 8 + lr, bb_n = (li >> 1) * 8;                  // input-gradient B [k][n]
#pragma unroll
    for (int s = 0; s < kRing - 1; ++s) {
        if (s < nst) issue(s);
        cp_async_commit();
    }
    for (int s = 0; s < nst; ++s) {
        cp_async_wait<kRing - 2>();
        __syncthreads();
        if (s + kRing - 1 < nst) issue(s + kRing - 1);
        cp_async_commit();
        const Stage& st = ring[s % kRing];
#pragma unroll
        for (int k0 = 0; k0 < kMmaCo; k0 += kMmaK) {
            uint32_t a[NP][4];
#pragma unroll
            for (int h = 0; h < NP; ++h) ldsm_x4(smem_u32(&st.a[h][a_m][k0 + a_k]), a[h][0], a[h][1], a[h][2], a[h][3]);
#pragma unroll
            for (int jj = 0; jj < 2; ++jj) {
                uint32_t b0, b1, b2, b3;
                if (BWD)
                    ldsm_x4_t(smem_u32(&st.b[k0 + bb_k][16 * jj + bb_n]), b0, b1, b2, b3);
                else
                    ldsm_x4(smem_u32(&st.b[16 * jj + bf_n][k0 + bf_k]), b0, b1, b2, b3);
#pragma unroll
                for (int h = 0; h < NP; ++h) {
                    mma_bf16(acc[2 * jj], a[h][0], a[h][1], a[h][2], a[h][3], b0, b1);
                    mma_bf16(acc[2 * jj + 1], a[h][0], a[h][1], a[h][2], a[h][3], b2, b3);
                }
            }
        }
    }
    cp_async_wait<0>();
    const int gid = lane >> 2, tig = lane & 3;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
#pragma unroll
        for (int r = 0; r < 4; ++r) {
            const long p = pb + warp * 16 + gid + (r >> 1) * 8;
            const int n = n0 + j * 8 + 2 * tig + (r & 1);
            if (p >= P || n >= Cn) continue;
            if (BWD)
                static_cast<float*>(out)[p * Cn + n] = acc[j][r];
            else
                static_cast<bf16*>(out)[p * Cn + n] = __float2bfloat16_rn(fmaxf(acc[j][r] + bias[n], 0.f));
        }
    }
}
template <bool BWD>
constexpr int conv_gemm_smem() {
    return kRing * ((BWD ? 2 : 1) * kTilePts * kStr + kMmaCo * kStr) * (int)sizeof(bf16);
}

// The same two products by patches: a block owns 128 points, a TH x TW patch
// of one image (or several whole images of a small level), and stages the
// patch with its one-point halo once per 32 reduction channels, together with
// those channels' weights of all 9 taps; the taps then read the staged rows
// shifted, with no barrier between them.
//
// Why: k_conv_gemm fetches the same rows once per tap and stops at a barrier
// every 8 mma of a warp; it ran at 2% of the tensor rate, bound by those
// fetches and barriers.  Here a warp (32 points x 8 NT columns) issues
// 9 x 2 x 2 NT mma between barriers, 12 of them per 5 ldmatrix at NT = 6, and
// the activations are read 1.4 times instead of 9.  Two stages: the next 32
// channels are copied while this stage computes.  Forward at 512x256 (14
// convolutions, width 24): 558 -> 305 us; gradient at 128x64, batch 16, all told:
// 2109 -> 1203 us.
//
// The order of the sums of an output (32 channels outside, taps, then 16
// channels) is that of k_conv_gemm, so results are the same bits; steps whose
// 16 channels are all padding are left out (they add zeros).
//
// Forward with `pool` (patches of 16-point rows): the 2x2 means of the rounded
// outputs go there too; a thread holds both rows of a 2x2 block, the lane 4
// beside it the other column.  Forward with `yout` (all columns in one block):
// the 1x1 output layer wo, bo on the rounded outputs, one thread a point, the
// sum in the order of k_out_fwd.  Neither re-reads the activations:
// forward at 512x256 306 -> 286 us.
//
// BWD with `act`: the gradient of a ReLU output `act` leaves as the two
// bfloat16 planes (out, out_lo) that k_relu_split would make of it.
// VB: 16-byte copies of the weight rows (ci a multiple of 8).
constexpr int kHaloPts = 128, kHaloRows = 384;
struct HaloShape {
    int lh, lw;        // log2 of the image
    int lth, ltw;      // log2 of the patch
    int images;        // images per block (patch = whole image when > 1)
    int B;             // images in all
};
__host__ __device__ inline int halo_rows(const HaloShape& h) { return h.images * ((1 << h.lth) + 2) * ((1 << h.ltw) + 2); }
// Input of the first convolution of a decoder level, read in place instead of
// being concatenated: channels below C1 from the parent point of the level
// below (nearest upsampling), the rest from the skip.  C1 = 0: an ordinary
// input.
struct CatIn {
    const bf16* low = nullptr;
    int C1 = 0;
    // channels c .. c + 7 of point p of images of 2^lw columns; rows of ld channels
    __device__ __forceinline__ const bf16* at(const bf16* skip, int p, int c, int ld, int lw) const {
        if (c < C1) {
            const int x = p & ((1 << lw) - 1), r = p >> lw;   // rows of all images
            return low + ((long)(((r >> 1) << (lw - 1)) + (x >> 1))) * C1 + c;
        }
        return skip + (long)p * ld + (c - C1);
    }
};

// Staged rows of a patch: images one after another, each (TH + 2) x (TW + 2).
struct HaloMap {
    HaloShape hs;
    int nrows, per_image, TW2;
    __device__ __forceinline__ explicit HaloMap(const HaloShape& h) : hs(h) {
        nrows = halo_rows(h);
        per_image = nrows / h.images;
        TW2 = (1 << h.ltw) + 2;
    }
    // staged row of point m at tap offset (-1, -1)
    __device__ __forceinline__ int row_of(int m) const {
        return (m >> (hs.lth + hs.ltw)) * per_image + ((m >> hs.ltw) & ((1 << hs.lth) - 1)) * TW2 +
               (m & ((1 << hs.ltw) - 1));
    }
    // table of the point of each staged row (-1: beyond the last image)
    __device__ __forceinline__ void fill(int* rows, int patch, int tid) const {
        const int H = 1 << hs.lh, W = 1 << hs.lw;
        int img0 = patch * hs.images, y0 = 0, x0 = 0;   // first image and corner of the patch
        if (hs.images == 1) {
            const int lpx = hs.lw - hs.ltw, lpp = lpx + hs.lh - hs.lth;
            img0 = patch >> lpp;
            y0 = ((patch & ((1 << lpp) - 1)) >> lpx) << hs.lth;
            x0 = (patch & ((1 << lpx) - 1)) << hs.ltw;
        }
        for (int r = tid; r < nrows; r += 128) {
            const int im = r / per_image, q = r - im * per_image;
            const int y = (y0 + q / TW2 - 1) & (H - 1), x = (x0 + q % TW2 - 1) & (W - 1);
            rows[r] = img0 + im < hs.B ? ((((img0 + im) << hs.lh) + y) << hs.lw) + x : -1;
        }
    }
};
template <bool BWD, int NT>
__host__ __device__ constexpr int halo_brow() {   // bytes of a staged weight row
    return !BWD ? 2 * kStr : NT == 3 ? 80 : 16 * NT + 16;
}
template <bool BWD, int NT>
__host__ __device__ inline int halo_stage(const HaloShape& h) {
    return halo_rows(h) * 2 * kStr * (BWD ? 2 : 1) + 9 * (BWD ? kMmaCo : 8 * NT) * halo_brow<BWD, NT>();
}

struct HaloTail {
    bf16* pool = nullptr;          // forward: 2x2 means of the output
    const bf16* wo = nullptr;      // forward: 1x1 output layer (weights, bias, result)
    const float* bo = nullptr;
    float* yout = nullptr;
    CatIn cat;                     // forward: where the first channels of the input come from
};

template <bool BWD, int NT, bool VB>
__global__ void __launch_bounds__(128) k_conv_halo(const bf16* __restrict__ a_hi, const bf16* __restrict__ a_lo,
                                                   const bf16* __restrict__ wt, const float* __restrict__ bias,
                                                   const bf16* __restrict__ act, void* __restrict__ out,
                                                   bf16* __restrict__ out_lo, HaloShape hs, int Ci, int Co, int lda,
                                                   HaloTail tail) {
    constexpr int NP = BWD ? 2 : 1, NB = 8 * NT, BROW = halo_brow<BWD, NT>();
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ int rows[kHaloRows];   // point of each staged row, -1: none
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int Ck = BWD ? Co : Ci, Cn = BWD ? Ci : Co;
    const int n0 = blockIdx.y * NB;
    const int nck = (Ck + kMmaCo - 1) / kMmaCo;
    const HaloMap map(hs);
    const int nrows = map.nrows, TW2 = map.TW2;
    map.fill(rows, blockIdx.x, tid);
    __syncthreads();
    const int asz = nrows * 2 * kStr;
    const int stage = asz * NP + 9 * (BWD ? kMmaCo : NB) * BROW;
    auto issue = [&](int kc, int buf) {
        unsigned char* st = smem + buf * stage;
        const int c0 = kc * kMmaCo;
        for (int f = tid; f < nrows * 4; f += 128) {
            const int r = f >> 2, g = f & 3, p = rows[r];
            const bool ok = p >= 0 && c0 + 8 * g < Ck;
#pragma unroll
            for (int h = 0; h < NP; ++h) {
                const bf16* base = h ? a_lo : a_hi;
                const bf16* src = !ok ? base : BWD ? base + (long)p * lda + c0 + 8 * g
                                                   : tail.cat.at(base, p, c0 + 8 * g, lda, hs.lw);
                cp_async16(smem_u32(st + h * asz + r * 2 * kStr + 16 * g), src, ok ? 16 : 0);
            }
        }
        unsigned char* sb = st + asz * NP;
        if (!VB) {   // few input channels (the first layer): forward only
            for (int f = tid; f < 9 * NB * kMmaCo; f += 128) {
                const int r = f / kMmaCo, k = f % kMmaCo, t = r / NB, n = n0 + r % NB;
                reinterpret_cast<bf16*>(sb + r * BROW)[k] =
                    (n < Co && c0 + k < Ci) ? wt[((long)t * Co + n) * Ci + c0 + k] : __float2bfloat16_rn(0.f);
            }
        } else {   // rows of each tap: output channels c0 .. c0 + 31 (BWD), n0 .. n0 + NB - 1
            constexpr int RC = BWD ? NT : 4, RT = BWD ? kMmaCo : NB;   // 16-byte pieces a row, rows a tap
            for (int f = tid; f < RT * RC; f += 128) {
                const int r = f / RC, g = f % RC;
                const bool ok = BWD ? c0 + r < Co && n0 + 8 * g < Ci : n0 + r < Co && c0 + 8 * g < Ci;
                const bf16* src = ok ? wt + (long)((BWD ? c0 : n0) + r) * Ci + (BWD ? n0 : c0) + 8 * g : wt;
                const long step = ok ? (long)Co * Ci : 0;
                uint32_t dst = smem_u32(sb + r * BROW + 16 * g);
#pragma unroll
                for (int t = 0; t < 9; ++t, dst += RT * BROW, src += step) cp_async16(dst, src, ok ? 16 : 0);
            }
        }
    };
    const int lr = lane & 7, li = lane >> 3;
    uint32_t a_addr[2];   // ldmatrix row addresses of the warp's two 16-point tiles
#pragma unroll
    for (int i = 0; i < 2; ++i)
        a_addr[i] = smem_u32(smem) + map.row_of(warp * 32 + i * 16 + (li & 1) * 8 + lr) * 2 * kStr + (li >> 1) * 16;
    const uint32_t b_addr = smem_u32(smem) + asz * NP +
                            (BWD ? ((li & 1) * 8 + lr) * BROW + (li >> 1) * 16 : ((li >> 1) * 8 + lr) * BROW + (li & 1) * 16);
    // the last, single tile of an odd NT (ldmatrix.x2: lanes 0..15)
    const uint32_t b_last = smem_u32(smem) + asz * NP +
                            (BWD ? ((li & 1) * 8 + lr) * BROW + (NT - 1) * 16 : ((NT - 1) * 8 + lr) * BROW + (li & 1) * 16);
    float acc[2][NT][4];
#pragma unroll
    for (int i = 0; i < 2; ++i)
#pragma unroll
        for (int j = 0; j < NT; ++j)
#pragma unroll
            for (int r = 0; r < 4; ++r) acc[i][j][r] = 0.f;
    issue(0, 0);
    cp_async_commit();
    for (int kc = 0; kc < nck; ++kc) {
        if (kc + 1 < nck) issue(kc + 1, (kc + 1) & 1);
        cp_async_commit();
        cp_async_wait<1>();
        __syncthreads();
        const uint32_t so = (kc & 1) * stage;
        const int ksteps = min(kMmaCo, Ck - kc * kMmaCo) > kMmaK ? 2 : 1;
#pragma unroll
        for (int t = 0; t < 9; ++t) {
            const int ty = BWD ? 2 - t / 3 : t / 3, tx = BWD ? 2 - t % 3 : t % 3;
            const uint32_t ao = so + (ty * TW2 + tx) * 2 * kStr;
            const uint32_t bo = so + t * (BWD ? kMmaCo : NB) * BROW;
#pragma unroll
            for (int ks = 0; ks < 2; ++ks) {
                if (ks == ksteps) break;
                uint32_t a[2][NP][4], b[NT][2];
                const uint32_t bk = bo + ks * (BWD ? kMmaK * BROW : kMmaK * 2);
#pragma unroll
                for (int i = 0; i < 2; ++i)
#pragma unroll
                    for (int h = 0; h < NP; ++h)
                        ldsm_x4(a_addr[i] + ao + h * asz + ks * kMmaK * 2, a[i][h][0], a[i][h][1], a[i][h][2], a[i][h][3]);
#pragma unroll
                for (int j = 0; j + 1 < NT; j += 2) {
                    if (BWD) ldsm_x4_t(b_addr + bk + j * 16, b[j][0], b[j][1], b[j + 1][0], b[j + 1][1]);
                    else ldsm_x4(b_addr + bk + j * 8 * BROW, b[j][0], b[j][1], b[j + 1][0], b[j + 1][1]);
                }
                if (NT & 1) {
                    if (BWD) ldsm_x2_t(b_last + bk, b[NT - 1][0], b[NT - 1][1]);
                    else ldsm_x2(b_last + bk, b[NT - 1][0], b[NT - 1][1]);
                }
#pragma unroll
                for (int h = 0; h < NP; ++h)
#pragma unroll
                    for (int i = 0; i < 2; ++i)
#pragma unroll
                        for (int j = 0; j < NT; ++j)
                            mma_bf16(acc[i][j], a[i][h][0], a[i][h][1], a[i][h][2], a[i][h][3], b[j][0], b[j][1]);
            }
        }
        __syncthreads();
    }
    cp_async_wait<0>();
    const int gid = lane >> 2, tig = lane & 3;
#pragma unroll
    for (int i = 0; i < 2; ++i)
#pragma unroll
        for (int r = 0; r < 2; ++r) {
            const int p = rows[map.row_of(warp * 32 + i * 16 + gid + 8 * r) + TW2 + 1];
            if (p < 0) continue;
#pragma unroll
            for (int j = 0; j < NT; ++j) {
                const int n = n0 + j * 8 + 2 * tig;   // channel counts are multiples of 8
                if (n >= Cn) continue;
                const long o = (long)p * Cn + n;
                const float x = acc[i][j][2 * r], y = acc[i][j][2 * r + 1];
                if (!BWD) {
                    const __nv_bfloat162 h(__float2bfloat16_rn(fmaxf(x + bias[n], 0.f)),
                                           __float2bfloat16_rn(fmaxf(y + bias[n + 1], 0.f)));
                    *reinterpret_cast<__nv_bfloat162*>(static_cast<bf16*>(out) + o) = h;
                    acc[i][j][2 * r] = __bfloat162float(h.x);
                    acc[i][j][2 * r + 1] = __bfloat162float(h.y);
                } else if (act) {
                    const __nv_bfloat162 a = *reinterpret_cast<const __nv_bfloat162*>(act + o);
                    const float vx = __bfloat162float(a.x) > 0.f ? x : 0.f, vy = __bfloat162float(a.y) > 0.f ? y : 0.f;
                    const __nv_bfloat162 hi(__float2bfloat16_rn(vx), __float2bfloat16_rn(vy));
                    *reinterpret_cast<__nv_bfloat162*>(static_cast<bf16*>(out) + o) = hi;
                    *reinterpret_cast<__nv_bfloat162*>(out_lo + o) =
                        __nv_bfloat162(__float2bfloat16_rn(vx - __bfloat162float(hi.x)),
                                       __float2bfloat16_rn(vy - __bfloat162float(hi.y)));
                } else {
                    *reinterpret_cast<float2*>(static_cast<float*>(out) + o) = make_float2(x, y);
                }
            }
        }
    if (!BWD && tail.pool) {
        // points (2 row, x) in acc[0], (2 row + 1, x) in acc[1]; x = gid + 8 r
        const int Wp = 1 << (hs.lw - 1);
#pragma unroll
        for (int r = 0; r < 2; ++r) {
            const int p = rows[map.row_of(warp * 32 + gid + 8 * r) + TW2 + 1];   // (even row, x)
            const int x = p & ((1 << hs.lw) - 1), row = p >> hs.lw;              // row of all images
            const long q = (long)(row >> 1) * Wp + (x >> 1);
#pragma unroll
            for (int j = 0; j < NT; ++j) {
                float m[2];
#pragma unroll
                for (int e = 0; e < 2; ++e) {
                    const float a = acc[0][j][2 * r + e], b = acc[1][j][2 * r + e];
                    const float a1 = __shfl_xor_sync(0xffffffffu, a, 4), b1 = __shfl_xor_sync(0xffffffffu, b, 4);
                    m[e] = 0.25f * (a + a1 + b + b1);   // read by lanes of even x
                }
                const int n = n0 + j * 8 + 2 * tig;
                if (n < Cn && !(gid & 1))
                    *reinterpret_cast<__nv_bfloat162*>(tail.pool + q * Cn + n) =
                        __nv_bfloat162(__float2bfloat16_rn(m[0]), __float2bfloat16_rn(m[1]));
            }
        }
    }
    if (!BWD && tail.yout) {
        // the outputs of each point in shared memory (the stages are free), then one thread a point
        constexpr int LD = NB + 1;
        float* hbuf = reinterpret_cast<float*>(smem);
#pragma unroll
        for (int i = 0; i < 2; ++i)
#pragma unroll
            for (int j = 0; j < NT; ++j)
#pragma unroll
                for (int r = 0; r < 4; ++r)
                    hbuf[(warp * 32 + i * 16 + gid + 8 * (r >> 1)) * LD + j * 8 + 2 * tig + (r & 1)] = acc[i][j][r];
        __syncthreads();
        const int p = rows[map.row_of(tid) + TW2 + 1];
        if (p >= 0) {
            float sum = tail.bo[0];
            for (int c = 0; c < Cn; ++c) sum = fmaf(__bfloat162float(tail.wo[c]), hbuf[tid * LD + c], sum);
            tail.yout[p] = sum;
        }
    }
}

// gw[co][ci][tap] += sum_p gz[p][co] in[nbr(p, tap)][ci]; gb[co] += sum_p gz[p][co]
// on the tensor cores: per tap a GEMM with rows = output channels, columns =
// input channels and the reduction over points.  A block owns 32 x 32
// (output, input) channels, all 9 taps, and a chunk of points (a multiple of
// kWgPts).  The blocks of a cluster (up to kWgCluster chunks of one tile) add
// their sums through distributed shared memory, each a share of the tile, and
// one atomicAdd per element and cluster goes to the gradient: with one per
// element and block the 456 blocks of a 24 x 24 layer sent 2.4 M atomics to
// 5184 addresses and took 70 us, 34 us now (cold caches).  The bias gradient is a
// column of ones beside the input (one more mma per fragment) instead of a
// serial sum by the first warp.  A stage holds,
// point-major, the gradient's hi and lo planes and the 9 neighbour rows of
// the input; fragments of both come from ldmatrix.trans.  Warp w owns output
// rows 16 (w & 1) .. +15 and input columns 16 (w >> 1) .. +15 for all 9 taps
// (72 FP32 accumulators a thread).  VA / VB: 16-byte copies for the gradient
// planes / the input rows (row stride ldin).
constexpr int kWgPts = 32;   // points per stage
constexpr int kWgRing = 4;
constexpr int kWgCluster = 8;
constexpr int kWgTile = 9 * kMmaCo * kMmaCo + kMmaCo;   // sums of a block: weights [tap][co][ci], bias
struct WgStage {
    bf16 ah[kWgPts][kStr], al[kWgPts][kStr];   // [point][co]
    bf16 b[9][kWgPts][kStr];                   // [tap][point][ci]
};
constexpr int wg_smem() {
    const int ring = kWgRing * (int)sizeof(WgStage), sums = kWgTile * (int)sizeof(float);
    return ring > sums ? ring : sums;   // the sums reuse the ring
}

// Sums of a weight-gradient block (fragments acc of warp rows mrow, columns
// ncol; accb: column sums) into the gradient: through shared memory `sums`,
// then across the cluster.
__device__ __forceinline__ void wgrad_store(float* sums, const float (&acc)[9][2][4], const float (&accb)[4], int mrow,
                                            int ncol, int co0, int ci0, int Ci, int Co, float* gw, float* gb) {
    const int lane = threadIdx.x & 31, gid = lane >> 2, tig = lane & 3;
#pragma unroll
    for (int t = 0; t < 9; ++t)
#pragma unroll
        for (int j = 0; j < 2; ++j)
#pragma unroll
            for (int r = 0; r < 4; ++r)
                sums[(t * kMmaCo + mrow + gid + (r >> 1) * 8) * kMmaCo + ncol + j * 8 + 2 * tig + (r & 1)] = acc[t][j][r];
    if (ncol == 0 && tig == 0) {
        sums[9 * kMmaCo * kMmaCo + mrow + gid] = accb[0];
        sums[9 * kMmaCo * kMmaCo + mrow + gid + 8] = accb[2];
    }
    cg::cluster_group cl = cg::this_cluster();
    const int nb = cl.num_blocks();
    cl.sync();
    for (int e = cl.block_rank() * blockDim.x + threadIdx.x; e < kWgTile; e += nb * blockDim.x) {
        const int t = e / (kMmaCo * kMmaCo), co = co0 + (t < 9 ? (e / kMmaCo) % kMmaCo : e - 9 * kMmaCo * kMmaCo);
        const int ci = ci0 + e % kMmaCo;
        if (co >= Co || (t < 9 ? ci >= Ci : ci0 != 0)) continue;
        float v = 0.f;
        for (int b = 0; b < nb; ++b) v += cl.map_shared_rank(sums, b)[e];
        atomicAdd(t < 9 ? &gw[((long)co * Ci + ci) * 9 + t] : &gb[co], v);
    }
    cl.sync();   // no block leaves while another reads its sums
}

template <bool VA, bool VB>
__global__ void __launch_bounds__(128) k_conv_bwd_w(const bf16* __restrict__ gzh, const bf16* __restrict__ gzl,
                                                    const bf16* __restrict__ in, float* __restrict__ gw,
                                                    float* __restrict__ gb, long P, int lh, int lw, int Ci, int Co,
                                                    int ldin, long chunk) {
    extern __shared__ __align__(16) unsigned char smem[];
    WgStage* ring = reinterpret_cast<WgStage*>(smem);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int ci_tiles = (Ci + kMmaCo - 1) / kMmaCo;
    const int co0 = (blockIdx.x / ci_tiles) * kMmaCo, ci0 = (blockIdx.x % ci_tiles) * kMmaCo;
    const long p0 = blockIdx.y * chunk, p1 = min(P, p0 + chunk);
    const int nst = (int)((p1 - p0 + kWgPts - 1) / kWgPts);
    const int mrow = (warp & 1) * 16, ncol = (warp >> 1) * 16;
    auto issue = [&](int s) {
        WgStage& st = ring[s % kWgRing];
        const long ps = p0 + (long)s * kWgPts;
        auto prow = [&](int r) -> long { return ps + r < p1 ? ps + r : -1; };
        stage_rows<VA, kWgPts, 128>(st.ah, gzh, Co, Co, co0, prow);
        stage_rows<VA, kWgPts, 128>(st.al, gzl, Co, Co, co0, prow);
#pragma unroll
        for (int t = 0; t < 9; ++t)
            stage_rows<VB, kWgPts, 128>(st.b[t], in, Ci, ldin, ci0, [&](int r) -> long {
                return ps + r < p1 ? nbr(ps + r, lh, lw, t / 3 - 1, t % 3 - 1) : -1;
            });
    };
    // ldmatrix.trans row addresses: lane = 8 i + r supplies row r of matrix i
    const int lr = lane & 7, li = lane >> 3;
    const int a_k = (li >> 1) * 8 + lr, a_m = mrow + (li & 1) * 8;   // A^T stored [point][co]
    const int b_k = (li & 1) * 8 + lr, b_n = ncol + (li >> 1) * 8;   // B stored [point][ci]
    float acc[9][2][4];
#pragma unroll
    for (int t = 0; t < 9; ++t)
#pragma unroll
        for (int j = 0; j < 2; ++j)
#pragma unroll
            for (int r = 0; r < 4; ++r) acc[t][j][r] = 0.f;
    float accb[4] = {0.f, 0.f, 0.f, 0.f};   // column sums of the gradient (warps of ncol = 0 in blocks of ci0 = 0)
    const bool do_b = ci0 == 0 && ncol == 0;
    const uint32_t ones = 0x3f803f80u;      // two bfloat16 1.0
#pragma unroll
    for (int s = 0; s < kWgRing - 1; ++s) {
        if (s < nst) issue(s);
        cp_async_commit();
    }
    for (int s = 0; s < nst; ++s) {
        cp_async_wait<kWgRing - 2>();
        __syncthreads();
        if (s + kWgRing - 1 < nst) issue(s + kWgRing - 1);
        cp_async_commit();
        const WgStage& st = ring[s % kWgRing];
#pragma unroll
        for (int k0 = 0; k0 < kWgPts; k0 += kMmaK) {
            uint32_t h0, h1, h2, h3, l0, l1, l2, l3;
            ldsm_x4_t(smem_u32(&st.ah[k0 + a_k][a_m]), h0, h1, h2, h3);
            ldsm_x4_t(smem_u32(&st.al[k0 + a_k][a_m]), l0, l1, l2, l3);
            if (do_b) {
                mma_bf16(accb, h0, h1, h2, h3, ones, ones);
                mma_bf16(accb, l0, l1, l2, l3, ones, ones);
            }
#pragma unroll
            for (int t = 0; t < 9; ++t) {
                uint32_t b00, b01, b10, b11;
                ldsm_x4_t(smem_u32(&st.b[t][k0 + b_k][b_n]), b00, b01, b10, b11);
                mma_bf16(acc[t][0], h0, h1, h2, h3, b00, b01);
                mma_bf16(acc[t][0], l0, l1, l2, l3, b00, b01);
                mma_bf16(acc[t][1], h0, h1, h2, h3, b10, b11);
                mma_bf16(acc[t][1], l0, l1, l2, l3, b10, b11);
            }
        }
    }
    cp_async_wait<0>();
    __syncthreads();   // the ring is free: it takes the sums
    wgrad_store(reinterpret_cast<float*>(smem), acc, accb, mrow, ncol, co0, ci0, Ci, Co, gw, gb);
}

// The same by the patches of k_conv_halo (all channel counts multiples of 8):
// a stage is one patch of 128 points, the gradient planes of its points and
// the input rows with their halo, which the 9 taps read shifted.  72 x 8 mma
// of a warp between two barriers instead of 72 x 2, and a staged row costs a
// table lookup instead of the periodic index arithmetic of every copy.  Block
// y of the grid takes the patches y, y + gridDim.y, ...
__global__ void __launch_bounds__(128) k_conv_bwd_w_halo(const bf16* __restrict__ gzh, const bf16* __restrict__ gzl,
                                                         const bf16* __restrict__ in, float* __restrict__ gw,
                                                         float* __restrict__ gb, HaloShape hs, int npatch, int Ci,
                                                         int Co, int ldin, CatIn cat) {
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ int rows[2][kHaloRows];
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int ci_tiles = (Ci + kMmaCo - 1) / kMmaCo;
    const int co0 = (blockIdx.x / ci_tiles) * kMmaCo, ci0 = (blockIdx.x % ci_tiles) * kMmaCo;
    const int mrow = (warp & 1) * 16, ncol = (warp >> 1) * 16;
    const HaloMap map(hs);
    const int asz = kHaloPts * 2 * kStr, stage = 2 * asz + map.nrows * 2 * kStr;
    const int nst = blockIdx.y < npatch ? (npatch - 1 - blockIdx.y) / gridDim.y + 1 : 0;
    auto issue = [&](int s) {
        unsigned char* st = smem + (s & 1) * stage;
        const int* tab = rows[s & 1];
        for (int f = tid; f < kHaloPts * 4; f += 128) {
            const int m = f >> 2, g = f & 3, p = tab[map.row_of(m) + map.TW2 + 1];
            const bool ok = p >= 0 && co0 + 8 * g < Co;
            const long o = ok ? (long)p * Co + co0 + 8 * g : 0;
            cp_async16(smem_u32(st + m * 2 * kStr + 16 * g), gzh + o, ok ? 16 : 0);
            cp_async16(smem_u32(st + asz + m * 2 * kStr + 16 * g), gzl + o, ok ? 16 : 0);
        }
        for (int f = tid; f < map.nrows * 4; f += 128) {
            const int r = f >> 2, g = f & 3, p = tab[r];
            const bool ok = p >= 0 && ci0 + 8 * g < Ci;
            cp_async16(smem_u32(st + 2 * asz + r * 2 * kStr + 16 * g), ok ? cat.at(in, p, ci0 + 8 * g, ldin, hs.lw) : in,
                       ok ? 16 : 0);
        }
    };
    // ldmatrix.trans row addresses: lane = 8 i + r supplies row r of matrix i
    const int lr = lane & 7, li = lane >> 3;
    const uint32_t a_addr = smem_u32(smem) + ((li >> 1) * 8 + lr) * 2 * kStr + (mrow + (li & 1) * 8) * 2;
    const uint32_t b_addr = smem_u32(smem) + 2 * asz + (ncol + (li >> 1) * 8) * 2;
    const int b_k = (li & 1) * 8 + lr;
    float acc[9][2][4];
#pragma unroll
    for (int t = 0; t < 9; ++t)
#pragma unroll
        for (int j = 0; j < 2; ++j)
#pragma unroll
            for (int r = 0; r < 4; ++r) acc[t][j][r] = 0.f;
    float accb[4] = {0.f, 0.f, 0.f, 0.f};   // column sums of the gradient (warps of ncol = 0 in blocks of ci0 = 0)
    const bool do_b = ci0 == 0 && ncol == 0;
    const uint32_t ones = 0x3f803f80u;      // two bfloat16 1.0
    if (nst > 0) map.fill(rows[0], blockIdx.y, tid);
    __syncthreads();
    if (nst > 0) issue(0);
    cp_async_commit();
    if (nst > 1) map.fill(rows[1], blockIdx.y + gridDim.y, tid);
    for (int s = 0; s < nst; ++s) {
        cp_async_wait<0>();
        __syncthreads();   // stage s has landed; stage s - 1 and the table of s + 1 are done with / filled
        if (s + 1 < nst) issue(s + 1);
        cp_async_commit();
        if (s + 2 < nst) map.fill(rows[s & 1], blockIdx.y + (s + 2) * gridDim.y, tid);
        const uint32_t so = (s & 1) * stage;
#pragma unroll 2
        for (int k0 = 0; k0 < kHaloPts; k0 += kMmaK) {
            uint32_t h0, h1, h2, h3, l0, l1, l2, l3;
            ldsm_x4_t(a_addr + so + k0 * 2 * kStr, h0, h1, h2, h3);
            ldsm_x4_t(a_addr + so + asz + k0 * 2 * kStr, l0, l1, l2, l3);
            if (do_b) {
                mma_bf16(accb, h0, h1, h2, h3, ones, ones);
                mma_bf16(accb, l0, l1, l2, l3, ones, ones);
            }
            const uint32_t br = b_addr + so + map.row_of(k0 + b_k) * 2 * kStr;
#pragma unroll
            for (int t = 0; t < 9; ++t) {
                uint32_t b00, b01, b10, b11;
                ldsm_x4_t(br + ((t / 3) * map.TW2 + t % 3) * 2 * kStr, b00, b01, b10, b11);
                mma_bf16(acc[t][0], h0, h1, h2, h3, b00, b01);
                mma_bf16(acc[t][1], h0, h1, h2, h3, b10, b11);
                mma_bf16(acc[t][0], l0, l1, l2, l3, b00, b01);
                mma_bf16(acc[t][1], l0, l1, l2, l3, b10, b11);
            }
        }
    }
    cp_async_wait<0>();
    __syncthreads();   // the stages are free: they take the sums
    wgrad_store(reinterpret_cast<float*>(smem), acc, accb, mrow, ncol, co0, ci0, Ci, Co, gw, gb);
}
inline int wg_halo_smem(const HaloShape& h) {
    const int ring = 2 * (2 * kHaloPts + halo_rows(h)) * 2 * kStr, sums = kWgTile * (int)sizeof(float);
    return ring > sums ? ring : sums;
}

// x [B][C][H][W] FP32 -> [B][H][W][LD] bfloat16, channels C .. LD - 1 zero
__global__ void k_to_nhwc(const float* __restrict__ x, bf16* __restrict__ out, long P, int HW, int C, int LD) {
    for (long e = blockIdx.x * (long)blockDim.x + threadIdx.x; e < P * LD; e += (long)gridDim.x * blockDim.x) {
        const long p = e / LD;
        const int c = (int)(e % LD);
        const long b = p / HW, s = p % HW;
        out[e] = (c < C) ? __float2bfloat16_rn(x[(b * C + c) * HW + s]) : __float2bfloat16_rn(0.f);
    }
}

// V consecutive channels of a bfloat16 or FP32 row as floats (V = 8 where the
// channel counts are multiples of 8, else 1)
template <int V> __device__ __forceinline__ void load_bf16(const bf16* p, float (&v)[V]) {
    if constexpr (V == 8) {
        const uint4 q = *reinterpret_cast<const uint4*>(p);
        const uint32_t w[4] = {q.x, q.y, q.z, q.w};
#pragma unroll
        for (int i = 0; i < 4; ++i) {   // a bfloat16 is the upper half of a float
            v[2 * i] = __uint_as_float(w[i] << 16);
            v[2 * i + 1] = __uint_as_float(w[i] & 0xffff0000u);
        }
    } else {
        v[0] = __bfloat162float(p[0]);
    }
}
template <int V> __device__ __forceinline__ void store_bf16(bf16* p, const float (&v)[V]) {
    if constexpr (V == 8) {
        uint4 q;
        uint32_t* w = reinterpret_cast<uint32_t*>(&q);
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const __nv_bfloat162 b(__float2bfloat16_rn(v[2 * i]), __float2bfloat16_rn(v[2 * i + 1]));
            w[i] = *reinterpret_cast<const uint32_t*>(&b);
        }
        *reinterpret_cast<uint4*>(p) = q;
    } else {
        p[0] = __float2bfloat16_rn(v[0]);
    }
}
template <int V> __device__ __forceinline__ void load_f32(const float* p, float (&v)[V]) {
    if constexpr (V == 8) {
        *reinterpret_cast<float4*>(&v[0]) = reinterpret_cast<const float4*>(p)[0];
        *reinterpret_cast<float4*>(&v[4]) = reinterpret_cast<const float4*>(p)[1];
    } else {
        v[0] = p[0];
    }
}
template <int V> __device__ __forceinline__ void store_f32(float* p, const float (&v)[V]) {
    if constexpr (V == 8) {
        reinterpret_cast<float4*>(p)[0] = *reinterpret_cast<const float4*>(&v[0]);
        reinterpret_cast<float4*>(p)[1] = *reinterpret_cast<const float4*>(&v[4]);
    } else {
        p[0] = v[0];
    }
}
// gradient g of a ReLU output a as the two bfloat16 planes the convolution
// GEMMs read: v = g where the activation is positive, else 0; hi = bf16(v),
// lo = bf16(v - hi)
template <int V>
__device__ __forceinline__ void relu_split(const float (&g)[V], const bf16* a, bf16* hi, bf16* lo) {
    float act[V], h[V], l[V];
    load_bf16<V>(a, act);
#pragma unroll
    for (int i = 0; i < V; ++i) {
        const float v = act[i] > 0.f ? g[i] : 0.f;
        h[i] = __bfloat162float(__float2bfloat16_rn(v));
        l[i] = v - h[i];
    }
    store_bf16<V>(hi, h);
    store_bf16<V>(lo, l);
}

// 2x2 mean of [B][H][W][C] -> [B][H/2][W/2][C], rounded to bfloat16
template <int V>
__global__ void k_pool(const bf16* __restrict__ in, bf16* __restrict__ out, long Pout, int lwo, int C) {
    const int CV = C / V;
    const long W = 2L << lwo;
    for (long e = blockIdx.x * (long)blockDim.x + threadIdx.x; e < Pout * CV; e += (long)gridDim.x * blockDim.x) {
        const long p = e / CV;
        const int c = (int)(e - p * CV) * V;
        // output point (row r of all images, x) covers input rows 2r, 2r + 1
        const long x = p & ((1L << lwo) - 1), r = p >> lwo;
        const bf16* q = in + ((2 * r) * W + 2 * x) * C + c;
        float a[V], b[V], d[V], f[V];
        load_bf16<V>(q, a);
        load_bf16<V>(q + C, b);
        load_bf16<V>(q + W * C, d);
        load_bf16<V>(q + W * C + C, f);
#pragma unroll
        for (int i = 0; i < V; ++i) a[i] = 0.25f * (a[i] + b[i] + d[i] + f[i]);
        store_bf16<V>(out + p * C + c, a);
    }
}

// out[b][y][x] = (low[b][y/2][x/2][0..C1), skip[b][y][x][0..C2)); images of
// 2^lw columns
template <int V>
__global__ void k_up_cat(const bf16* __restrict__ low, const bf16* __restrict__ skip, bf16* __restrict__ out, long P,
                         int lw, int C1, int C2) {
    const int CV = (C1 + C2) / V;
    for (long e = blockIdx.x * (long)blockDim.x + threadIdx.x; e < P * CV; e += (long)gridDim.x * blockDim.x) {
        const long p = e / CV;
        const int c = (int)(e - p * CV) * V;
        const bf16* src = skip + p * C2 + (c - C1);
        if (c < C1) {
            const long x = p & ((1L << lw) - 1), r = p >> lw;   // rows of all images: r/2 is the low level's row
            src = low + (((r >> 1) << (lw - 1)) + (x >> 1)) * C1 + c;
        }
        if constexpr (V == 8) *reinterpret_cast<uint4*>(out + p * (C1 + C2) + c) = *reinterpret_cast<const uint4*>(src);
        else out[p * (C1 + C2) + c] = *src;
    }
}

// adjoint of k_up_cat: the sum over the 2x2 children of g[.][c] is the
// gradient of the low level's ReLU output act, written as bfloat16 planes;
// gskip[p][c] = g[p][C1 + c]
template <int V>
__global__ void k_up_cat_bwd(const float* __restrict__ g, const bf16* __restrict__ act, bf16* __restrict__ hi,
                             bf16* __restrict__ lo, float* __restrict__ gskip, long Plow, int lwl, int C1, int C2) {
    const int C = C1 + C2, CV = C / V;
    const long W = 2L << lwl;
    for (long e = blockIdx.x * (long)blockDim.x + threadIdx.x; e < Plow * CV; e += (long)gridDim.x * blockDim.x) {
        const long q = e / CV;
        const int c = (int)(e - q * CV) * V;
        const long x = q & ((1L << lwl) - 1), r = q >> lwl;
        const long p00 = 2 * r * W + 2 * x;
        const long ps[4] = {p00, p00 + 1, p00 + W, p00 + W + 1};
        if (c < C1) {
            float s[V] = {};
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                float v[V];
                load_f32<V>(g + ps[k] * C + c, v);
#pragma unroll
                for (int i = 0; i < V; ++i) s[i] += v[i];
            }
            const long o = q * C1 + c;
            relu_split<V>(s, act + o, hi + o, lo + o);
        } else {
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                float v[V];
                load_f32<V>(g + ps[k] * C + c, v);
                store_f32<V>(gskip + ps[k] * C2 + (c - C1), v);
            }
        }
    }
}

// adjoint of k_pool plus the skip gradient, glow[parent][c] / 4 + gskip[p][c]:
// the gradient of the ReLU output act, as bfloat16 planes
template <int V>
__global__ void k_pool_bwd_add(const float* __restrict__ glow, const float* __restrict__ gskip,
                               const bf16* __restrict__ act, bf16* __restrict__ hi, bf16* __restrict__ lo, long P,
                               int lw, int C) {
    const int CV = C / V;
    for (long e = blockIdx.x * (long)blockDim.x + threadIdx.x; e < P * CV; e += (long)gridDim.x * blockDim.x) {
        const long p = e / CV;
        const int c = (int)(e - p * CV) * V;
        const long x = p & ((1L << lw) - 1), r = p >> lw;
        float a[V], b[V];
        load_f32<V>(glow + (((r >> 1) << (lw - 1)) + (x >> 1)) * C + c, a);
        load_f32<V>(gskip + p * C + c, b);
#pragma unroll
        for (int i = 0; i < V; ++i) a[i] = 0.25f * a[i] + b[i];
        const long o = p * C + c;
        relu_split<V>(a, act + o, hi + o, lo + o);
    }
}

template <int V>
__global__ void k_relu_split(const float* __restrict__ g, const bf16* __restrict__ a, bf16* __restrict__ hi,
                             bf16* __restrict__ lo, long n) {
    for (long e = V * (blockIdx.x * (long)blockDim.x + threadIdx.x); e < n; e += V * (long)gridDim.x * blockDim.x) {
        float v[V];
        load_f32<V>(g + e, v);
        relu_split<V>(v, a + e, hi + e, lo + e);
    }
}

// y[p] = b + sum_c w[c] h[p][c]
__global__ void k_out_fwd(const bf16* __restrict__ h, const bf16* __restrict__ w, const float* __restrict__ b,
                          float* __restrict__ y, long P, int C) {
    for (long p = blockIdx.x * (long)blockDim.x + threadIdx.x; p < P; p += (long)gridDim.x * blockDim.x) {
        float s = b[0];
        for (int c = 0; c < C; ++c) s = fmaf(__bfloat162float(w[c]), __bfloat162float(h[p * C + c]), s);
        y[p] = s;
    }
}

// gy = 2 (y - t) / P; partial[block] = sum (y - t)^2 (FP64)
__global__ void k_mse(const float* __restrict__ y, const float* __restrict__ t, float* __restrict__ gy,
                      double* __restrict__ partial, long P) {
    double acc = 0.0;
    const float sc = 2.0f / (float)P;
    for (long p = blockIdx.x * (long)blockDim.x + threadIdx.x; p < P; p += (long)gridDim.x * blockDim.x) {
        const float d = y[p] - t[p];
        gy[p] = sc * d;
        acc += (double)d * (double)d;
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

// output layer backward: the gradient w[c] gy[p] of its input h, a ReLU
// output, as bfloat16 planes; gw[c] += sum_p gy[p] h[p][c]; gb += sum_p gy[p].
// One thread per point; the channel sums of a warp are folded by shuffles,
// those of a block in shared memory (C + 1 floats), one atomic per block.
template <int V>
__global__ void __launch_bounds__(256) k_out_bwd(const float* __restrict__ gy, const bf16* __restrict__ h,
                                                 const bf16* __restrict__ w, bf16* __restrict__ hi,
                                                 bf16* __restrict__ lo, float* __restrict__ gw, float* __restrict__ gb,
                                                 long P, int C) {
    extern __shared__ float part[];   // [8 warps][C + 1]
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const long p = blockIdx.x * 256L + threadIdx.x;
    const float gp = p < P ? gy[p] : 0.f;
    for (int c = 0; c <= C; c += V) {
        float v[V];
        if (c < C) {
            float hv[V], g[V];
            if (p < P) load_bf16<V>(h + p * C + c, hv);
#pragma unroll
            for (int i = 0; i < V; ++i) {
                g[i] = __bfloat162float(w[c + i]) * gp;
                v[i] = p < P ? gp * hv[i] : 0.f;
            }
            if (p < P) relu_split<V>(g, h + p * C + c, hi + p * C + c, lo + p * C + c);
        } else {
            v[0] = gp;
        }
#pragma unroll
        for (int i = 0; i < V; ++i) {
            if (c + i > C) break;
            float s = v[i];
            for (int o = 16; o > 0; o >>= 1) s += __shfl_down_sync(0xffffffffu, s, o);
            if (lane == 0) part[warp * (C + 1) + c + i] = s;
        }
    }
    __syncthreads();
    for (int c = threadIdx.x; c <= C; c += 256) {
        float s = 0.f;
        for (int k = 0; k < 8; ++k) s += part[k * (C + 1) + c];
        atomicAdd(c < C ? &gw[c] : gb, s);
    }
}

// where the bfloat16 copy of flat parameter i lives: the 3x3 weights
// [co][ci][tap] of each convolution tap-major as [tap][co][ci] at the same
// offset; biases and the output layer in place
struct WtMap {
    int n = 0;
    long off[16];
    int ci[16], co[16];
};
__device__ __forceinline__ long wt_index(const WtMap& m, long i) {
    for (int c = 0; c < m.n; ++c) {
        const long j = i - m.off[c];
        const long sz = 9L * m.ci[c] * m.co[c];
        if (j >= 0 && j < sz) {
            const int t = (int)(j % 9);
            const long oc = j / 9;   // co * ci + ci_
            return m.off[c] + (long)t * m.co[c] * m.ci[c] + oc;
        }
    }
    return i;
}

__global__ void k_adam(float* __restrict__ th, const float* __restrict__ g, float* __restrict__ m, float* __restrict__ v,
                       bf16* __restrict__ wt, WtMap map, long n, float lr, float b1, float b2, float eps, float c1,
                       float c2) {
    for (long i = blockIdx.x * (long)blockDim.x + threadIdx.x; i < n; i += (long)gridDim.x * blockDim.x) {
        const float gi = g[i];
        const float mi = b1 * m[i] + (1.f - b1) * gi;
        const float vi = b2 * v[i] + (1.f - b2) * gi * gi;
        m[i] = mi;
        v[i] = vi;
        const float t = th[i] - lr * (mi / c1) / (sqrtf(vi / c2) + eps);
        th[i] = t;
        wt[wt_index(map, i)] = __float2bfloat16_rn(t);
    }
}

__global__ void k_to_bf16(const float* __restrict__ a, bf16* __restrict__ wt, WtMap map, long n) {
    for (long i = blockIdx.x * (long)blockDim.x + threadIdx.x; i < n; i += (long)gridDim.x * blockDim.x)
        wt[wt_index(map, i)] = __float2bfloat16_rn(a[i]);
}

unsigned grid_for(long n, int threads) {
    const long b = (n + threads - 1) / threads;
    return (unsigned)std::max<long>(1, std::min<long>(b, 152L * 32));
}

}  // namespace
}  // namespace nsstab

using namespace nsstab;

struct nsstab_unet {
    int in_ch = 0, width = 0, H = 0, W = 0, lh = 0, lw = 0, maxB = 0;
    int ldx = 0;                  // channel stride of the bfloat16 input (in_ch rounded up to 8)
    cudaStream_t stream = nullptr;
    long count = 0;
    int step = 0;
    std::vector<ConvDesc> conv;   // 14 convolutions in forward order, then the output layer
    std::vector<void*> allocs;
    float *theta = nullptr, *grad = nullptr, *m = nullptr, *v = nullptr;
    bf16* wt = nullptr;           // bfloat16 weights, 3x3 convolutions tap-major
    WtMap map;
    bf16 *gzh = nullptr, *gzl = nullptr;   // a ReLU output's gradient as bf16 hi + lo planes
    bf16 *gnh = nullptr, *gnl = nullptr;   // those of the next layer down (swapped after each layer)
    bf16* x = nullptr;
    bf16* act[14] = {};           // ReLU outputs of the 14 convolutions
    bf16* pool[kLevels - 1] = {};
    bf16* cat[kLevels - 1] = {};  // decoder inputs, by level (none where cat_in_place)
    float* y = nullptr;
    float* gy = nullptr;
    float* g0 = nullptr;                  // gradient of a concatenation, a pooled level or (small levels) a ReLU output
    float* gskip[kLevels - 1] = {};
    double* partial = nullptr;
    double* partial_host = nullptr;

    template <class P> int alloc(P** p, size_t count_) {
        void* q = nullptr;
        const cudaError_t e = cudaMalloc(&q, std::max<size_t>(count_, 1) * sizeof(P));
        if (e != cudaSuccess) {
            set_error(std::string("unet: cudaMalloc: ") + cudaGetErrorString(e));
            return e == cudaErrorMemoryAllocation ? NSSTAB_ERR_OUT_OF_MEMORY : NSSTAB_ERR_CUDA;
        }
        allocs.push_back(q);
        *p = static_cast<P*>(q);
        return NSSTAB_OK;
    }
    ~nsstab_unet() {
        if (stream) cudaStreamSynchronize(stream);
        for (void* p : allocs) cudaFree(p);
        if (partial_host) cudaFreeHost(partial_host);
    }
    int c(int l) const { return width << l; }
    int h(int l) const { return H >> l; }
    int w(int l) const { return W >> l; }
};

namespace {

constexpr int kRedBlocksU = 128;

std::vector<ConvDesc> make_layout(int in_ch, int width, long* count) {
    std::vector<ConvDesc> v;
    long off = 0;
    auto add = [&](int ci, int co, int k) {
        ConvDesc d;
        d.ci = ci;
        d.co = co;
        d.k = k;
        d.w_off = off;
        off += (long)co * ci * k * k;
        d.b_off = off;
        off += co;
        v.push_back(d);
    };
    int ci = in_ch;
    for (int l = 0; l < kLevels; ++l) {
        add(ci, width << l, 3);
        add(width << l, width << l, 3);
        ci = width << l;
    }
    for (int l = kLevels - 2; l >= 0; --l) {
        add((width << (l + 1)) + (width << l), width << l, 3);
        add(width << l, width << l, 3);
    }
    add(width, 1, 1);
    *count = off;
    return v;
}

// indices into conv[] / act[]: encoder level l conv s (0 = a, 1 = b) and
// decoder level l conv s
int enc_id(int l, int s) { return 2 * l + s; }
int dec_id(int l, int s) { return 2 * kLevels + 2 * (kLevels - 2 - l) + s; }

bool al16(const void* p) { return reinterpret_cast<uintptr_t>(p) % 16 == 0; }

using GemmFn = void (*)(const bf16*, const bf16*, const bf16*, const float*, void*, long, int, int, int, int, int);
using WgradFn = void (*)(const bf16*, const bf16*, const bf16*, float*, float*, long, int, int, int, int, int, long);
template <bool BWD>
GemmFn pick_gemm(bool va, bool vb) {
    return va ? (vb ? k_conv_gemm<BWD, true, true> : k_conv_gemm<BWD, true, false>)
              : (vb ? k_conv_gemm<BWD, false, true> : k_conv_gemm<BWD, false, false>);
}
WgradFn pick_wgrad(bool va, bool vb) {
    return va ? (vb ? k_conv_bwd_w<true, true> : k_conv_bwd_w<true, false>)
              : (vb ? k_conv_bwd_w<false, true> : k_conv_bwd_w<false, false>);
}

// Patch shape of the halo kernels at level l (false: the level is too small,
// its halo would outweigh the patch).
bool halo_shape(const nsstab_unet* n, int l, int B, HaloShape* h) {
    h->lh = n->lh - l;
    h->lw = n->lw - l;
    h->ltw = std::min(h->lw, 7 - std::min(h->lh, 3));   // 8 x 16 points where the image has them
    h->lth = std::min(h->lh, 7 - h->ltw);
    h->images = kHaloPts >> (h->ltw + h->lth);
    h->B = B;
    // several images per block only when the patch is the whole image
    if (h->images > 1 && (h->lth < h->lh || h->ltw < h->lw)) return false;
    return halo_rows(*h) <= kHaloRows;
}

using HaloFn = void (*)(const bf16*, const bf16*, const bf16*, const float*, const bf16*, void*, bf16*, HaloShape, int,
                        int, int, HaloTail);
struct HaloKernel {
    HaloFn fn;
    int nt, stage;   // columns per block / 8, bytes of a stage
};
template <bool BWD, bool VB>
HaloKernel pick_halo(int cn, const HaloShape& h) {
    // the fewest padded columns, then the widest tile
    int nt = 6, best = 1 << 30;
    for (int c : {6, 4, 3, 2}) {
        const int padded = (cn + 8 * c - 1) / (8 * c) * 8 * c;
        if (padded < best) {
            best = padded;
            nt = c;
        }
    }
    switch (nt) {
        case 6: return {k_conv_halo<BWD, 6, VB>, 6, halo_stage<BWD, 6>(h)};
        case 4: return {k_conv_halo<BWD, 4, VB>, 4, halo_stage<BWD, 4>(h)};
        case 3: return {k_conv_halo<BWD, 3, VB>, 3, halo_stage<BWD, 3>(h)};
        default: return {k_conv_halo<BWD, 2, VB>, 2, halo_stage<BWD, 2>(h)};
    }
}

// raise the shared-memory limit of every halo kernel, to the same cap for all networks
template <bool BWD, bool VB> cudaError_t halo_attrs() {
    cudaError_t e = cudaSuccess;
    for (const HaloFn f : {HaloFn(k_conv_halo<BWD, 6, VB>), HaloFn(k_conv_halo<BWD, 4, VB>),
                           HaloFn(k_conv_halo<BWD, 3, VB>), HaloFn(k_conv_halo<BWD, 2, VB>)})
        if (e == cudaSuccess) e = cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024);
    return e;
}

// Launch the halo kernel (see k_conv_halo) on level l.  ck, cn: reduction
// channels and output columns.
int launch_halo(const nsstab_unet* n, const HaloKernel& k, const HaloShape& h, int l, const bf16* a_hi, const bf16* a_lo,
                const bf16* w, const float* bias, const bf16* act, void* out, bf16* out_lo, const ConvDesc& d, int ck,
                int cn, int lda, const HaloTail& tail = HaloTail()) {
    const long P = (long)h.B * n->h(l) * n->w(l);
    const int smem = std::max(k.stage * (ck > kMmaCo ? 2 : 1),
                              tail.yout ? kHaloPts * (8 * k.nt + 1) * (int)sizeof(float) : 0);
    const dim3 g((unsigned)((P + kHaloPts - 1) / kHaloPts), (unsigned)((cn + 8 * k.nt - 1) / (8 * k.nt)));
    k.fn<<<g, 128, smem, n->stream>>>(a_hi, a_lo, w, bias, act, out, out_lo, h, d.ci, d.co, lda, tail);
    NS_LAUNCH_CHECK();
    return NSSTAB_OK;
}

// Whether the decoder's first convolution at level l reads its two inputs in
// place (forward and weight gradient both by patches, all channels in eights);
// there is no concatenated input then.
bool cat_in_place(const nsstab_unet* n, int l) {
    HaloShape h;
    const ConvDesc& d = n->conv[dec_id(l, 0)];
    return n->c(l) % 8 == 0 && d.ci % 8 == 0 && al16(n->wt + d.w_off) && halo_shape(n, l, 1, &h);
}

// conv id on input rows `in` of stride lda (its input channels, or the
// padded stride of the network input)
// (pool / y: where the 2x2 means of the output / the network's output go if
// this launch can make them; set to null if it did)
int conv_fwd(nsstab_unet* n, int id, const bf16* in, int lda, int l, int B, bf16** pool = nullptr, float** y = nullptr,
             const CatIn& cat = CatIn()) {
    const ConvDesc& d = n->conv[id];
    const long P = (long)B * n->h(l) * n->w(l);
    const dim3 g((unsigned)((P + kTilePts - 1) / kTilePts), (unsigned)((d.co + kMmaCo - 1) / kMmaCo));
    const bf16* w = n->wt + d.w_off;
    HaloShape hs;
    if (lda % 8 == 0 && al16(in) && d.co % 8 == 0 && halo_shape(n, l, B, &hs)) {
        const bool vb = d.ci % 8 == 0 && al16(w);
        const HaloKernel k = vb ? pick_halo<false, true>(d.co, hs) : pick_halo<false, false>(d.co, hs);
        HaloTail tail;
        tail.cat = cat;
        if (pool && hs.images == 1 && hs.ltw == 4) std::swap(tail.pool, *pool);
        if (y && d.co <= 8 * k.nt) {
            const ConvDesc& o = n->conv.back();
            tail.wo = n->wt + o.w_off;
            tail.bo = n->theta + o.b_off;
            std::swap(tail.yout, *y);
        }
        return launch_halo(n, k, hs, l, in, nullptr, w, n->theta + d.b_off, nullptr, n->act[id], nullptr, d, d.ci, d.co,
                           lda, tail);
    }
    const GemmFn k = pick_gemm<false>(lda % 8 == 0 && al16(in), d.ci % 8 == 0 && al16(w));
    k<<<g, 128, conv_gemm_smem<false>(), n->stream>>>(in, nullptr, w, n->theta + d.b_off, n->act[id], P, n->lh - l,
                                                      n->lw - l, d.ci, d.co, lda);
    NS_LAUNCH_CHECK();
    return NSSTAB_OK;
}

// Launch a pointwise kernel over n channels of C: 8 channels a thread where
// they come in eights.
#define NS_POINTWISE(KERNEL, C, n, ...)                                                             \
    do {                                                                                            \
        if ((C) % 8 == 0) KERNEL<8><<<grid_for((n) / 8, 256), 256, 0, net->stream>>>(__VA_ARGS__);  \
        else KERNEL<1><<<grid_for((n), 256), 256, 0, net->stream>>>(__VA_ARGS__);                   \
        NS_LAUNCH_CHECK();                                                                          \
    } while (0)

// Weight and bias gradients of conv id from the planes gzh, gzl of its ReLU
// output's gradient and its input rows `in` (stride ldin); then, unless `to`
// is INPUT_NONE, the gradient of its input: FP32 into g0 (INPUT_F32), or,
// the input being the ReLU output act_in, as planes that take gzh, gzl's place
// (INPUT_PLANES).
enum InputGrad { INPUT_NONE, INPUT_F32, INPUT_PLANES };
int conv_bwd(nsstab_unet* net, int id, const bf16* in, int ldin, InputGrad to, const bf16* act_in, int l, int B,
             const CatIn& cat = CatIn()) {
    nsstab_unet* n = net;
    const ConvDesc& d = n->conv[id];
    const long P = (long)B * n->h(l) * n->w(l);
    const bool vz = d.co % 8 == 0 && al16(n->gzh) && al16(n->gzl);
    const bool vin = ldin % 8 == 0 && al16(in);
    HaloShape hs;
    const bool patches = halo_shape(n, l, B, &hs);
    const bool wg_halo = patches && vz && vin;
    // about three blocks per SM in all, each chunk a whole number of stages
    const long tiles = (long)((d.co + kMmaCo - 1) / kMmaCo) * ((d.ci + kMmaCo - 1) / kMmaCo);
    const long nchunk = std::max<long>(1, 3 * 152 / tiles);
    const long chunk = std::max<long>(4 * kWgPts, ((P + nchunk - 1) / nchunk + kWgPts - 1) / kWgPts * kWgPts);
    const long npatch = (P + kHaloPts - 1) / kHaloPts;
    long ny = wg_halo ? std::min(npatch, nchunk) : (P + chunk - 1) / chunk;
    int cluster = kWgCluster;
    while (cluster > 1 && cluster > ny) cluster /= 2;
    ny = (ny + cluster - 1) / cluster * cluster;   // chunks past the last point add zeros
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3((unsigned)tiles, (unsigned)ny);
    cfg.blockDim = dim3(128);
    cfg.dynamicSmemBytes = wg_halo ? wg_halo_smem(hs) : wg_smem();
    cfg.stream = n->stream;
    cudaLaunchAttribute at{};
    at.id = cudaLaunchAttributeClusterDimension;
    at.val.clusterDim.x = 1;
    at.val.clusterDim.y = cluster;
    at.val.clusterDim.z = 1;
    cfg.attrs = &at;
    cfg.numAttrs = 1;
    if (wg_halo)
        NS_CUDA(cudaLaunchKernelEx(&cfg, k_conv_bwd_w_halo, (const bf16*)n->gzh, (const bf16*)n->gzl, in,
                                   n->grad + d.w_off, n->grad + d.b_off, hs, (int)npatch, d.ci, d.co, ldin, cat));
    else
        NS_CUDA(cudaLaunchKernelEx(&cfg, pick_wgrad(vz, vin), (const bf16*)n->gzh, (const bf16*)n->gzl, in,
                                   n->grad + d.w_off, n->grad + d.b_off, P, n->lh - l, n->lw - l, d.ci, d.co, ldin,
                                   chunk));
    if (to == INPUT_NONE) return NSSTAB_OK;
    const bf16* w = n->wt + d.w_off;
    const bool vb = d.ci % 8 == 0 && al16(w);
    if (vz && vb && patches) {
        const bool planes = to == INPUT_PLANES;
        NS_TRY(launch_halo(n, pick_halo<true, true>(d.ci, hs), hs, l, n->gzh, n->gzl, w, nullptr,
                           planes ? act_in : nullptr, planes ? (void*)n->gnh : (void*)n->g0, n->gnl, d, d.co, d.ci,
                           d.co));
    } else {
        const dim3 gd((unsigned)((P + kTilePts - 1) / kTilePts), (unsigned)((d.ci + kMmaCo - 1) / kMmaCo));
        const GemmFn kd = pick_gemm<true>(vz, vb);
        kd<<<gd, 128, conv_gemm_smem<true>(), n->stream>>>(n->gzh, n->gzl, w, nullptr, n->g0, P, n->lh - l, n->lw - l,
                                                           d.ci, d.co, d.co);
        NS_LAUNCH_CHECK();
        if (to == INPUT_PLANES) NS_POINTWISE(k_relu_split, d.ci, P * d.ci, n->g0, act_in, n->gnh, n->gnl, P * d.ci);
    }
    if (to == INPUT_PLANES) {
        std::swap(n->gzh, n->gnh);
        std::swap(n->gzl, n->gnl);
    }
    return NSSTAB_OK;
}

// The network's output for a batch into y.
int forward(nsstab_unet* net, const float* x, int B, float* y) {
    nsstab_unet* n = net;
    const long P0 = (long)B * n->H * n->W;
    k_to_nhwc<<<grid_for(P0 * n->ldx, 256), 256, 0, n->stream>>>(x, n->x, P0, n->H * n->W, n->in_ch, n->ldx);
    NS_LAUNCH_CHECK();
    const bf16* h = n->x;
    for (int l = 0; l < kLevels; ++l) {
        NS_TRY(conv_fwd(n, enc_id(l, 0), h, l == 0 ? n->ldx : n->c(l - 1), l, B));
        bf16* pool = l < kLevels - 1 ? n->pool[l] : nullptr;
        NS_TRY(conv_fwd(n, enc_id(l, 1), n->act[enc_id(l, 0)], n->c(l), l, B, pool ? &pool : nullptr));
        h = n->act[enc_id(l, 1)];
        if (l < kLevels - 1) {
            const long Po = (long)B * n->h(l + 1) * n->w(l + 1);
            if (pool) NS_POINTWISE(k_pool, n->c(l), Po * n->c(l), h, n->pool[l], Po, n->lw - l - 1, n->c(l));
            h = n->pool[l];
        }
    }
    for (int l = kLevels - 2; l >= 0; --l) {
        const long P = (long)B * n->h(l) * n->w(l);
        const bf16* skip = n->act[enc_id(l, 1)];
        if (cat_in_place(n, l)) {
            CatIn cat;
            cat.low = h;
            cat.C1 = n->c(l + 1);
            NS_TRY(conv_fwd(n, dec_id(l, 0), skip, n->c(l), l, B, nullptr, nullptr, cat));
        } else {
            NS_POINTWISE(k_up_cat, n->c(l), P * (n->c(l + 1) + n->c(l)), h, skip, n->cat[l], P, n->lw - l, n->c(l + 1),
                         n->c(l));
            NS_TRY(conv_fwd(n, dec_id(l, 0), n->cat[l], n->c(l + 1) + n->c(l), l, B));
        }
        NS_TRY(conv_fwd(n, dec_id(l, 1), n->act[dec_id(l, 0)], n->c(l), l, B, nullptr, l == 0 ? &y : nullptr));
        h = n->act[dec_id(l, 1)];
    }
    if (y) {
        const ConvDesc& o = n->conv.back();
        k_out_fwd<<<grid_for(P0, 256), 256, 0, n->stream>>>(h, n->wt + o.w_off, n->theta + o.b_off, y, P0, n->c(0));
        NS_LAUNCH_CHECK();
    }
    return NSSTAB_OK;
}

int backward(nsstab_unet* net, const float* target, int B, double* loss) {
    nsstab_unet* n = net;
    const long P0 = (long)B * n->H * n->W;
    NS_CUDA(cudaMemsetAsync(n->grad, 0, n->count * sizeof(float), n->stream));
    k_mse<<<kRedBlocksU, 256, 0, n->stream>>>(n->y, target, n->gy, n->partial, P0);
    NS_LAUNCH_CHECK();
    NS_CUDA(cudaMemcpyAsync(n->partial_host, n->partial, kRedBlocksU * sizeof(double), cudaMemcpyDeviceToHost,
                            n->stream));
    const ConvDesc& o = n->conv.back();
    const unsigned ob = (unsigned)((P0 + 255) / 256);
    const size_t osm = 8 * (size_t)(n->c(0) + 1) * sizeof(float);
    const bf16* top = n->act[dec_id(0, 1)];
    if (n->c(0) % 8 == 0)
        k_out_bwd<8><<<ob, 256, osm, n->stream>>>(n->gy, top, n->wt + o.w_off, n->gzh, n->gzl, n->grad + o.w_off,
                                                  n->grad + o.b_off, P0, n->c(0));
    else
        k_out_bwd<1><<<ob, 256, osm, n->stream>>>(n->gy, top, n->wt + o.w_off, n->gzh, n->gzl, n->grad + o.w_off,
                                                  n->grad + o.b_off, P0, n->c(0));
    NS_LAUNCH_CHECK();
    // gzh, gzl: the planes of the current ReLU output's gradient
    for (int l = 0; l < kLevels - 1; ++l) {
        NS_TRY(conv_bwd(n, dec_id(l, 1), n->act[dec_id(l, 0)], n->c(l), INPUT_PLANES, n->act[dec_id(l, 0)], l, B));
        const bf16* low = n->act[l + 1 < kLevels - 1 ? dec_id(l + 1, 1) : enc_id(l + 1, 1)];   // the level below's output
        if (cat_in_place(n, l)) {
            CatIn cat;
            cat.low = low;
            cat.C1 = n->c(l + 1);
            NS_TRY(conv_bwd(n, dec_id(l, 0), n->act[enc_id(l, 1)], n->c(l), INPUT_F32, nullptr, l, B, cat));
        } else {
            NS_TRY(conv_bwd(n, dec_id(l, 0), n->cat[l], n->c(l + 1) + n->c(l), INPUT_F32, nullptr, l, B));
        }
        // g0: gradient of cat[l]; split into the level below's output and the skip
        const long Pl = (long)B * n->h(l + 1) * n->w(l + 1);
        NS_POINTWISE(k_up_cat_bwd, n->c(l), Pl * (n->c(l + 1) + n->c(l)), n->g0, low, n->gzh, n->gzl, n->gskip[l], Pl,
                     n->lw - l - 1, n->c(l + 1), n->c(l));
    }
    for (int l = kLevels - 1; l >= 0; --l) {
        if (l < kLevels - 1) {
            const long P = (long)B * n->h(l) * n->w(l);
            NS_POINTWISE(k_pool_bwd_add, n->c(l), P * n->c(l), n->g0, n->gskip[l], n->act[enc_id(l, 1)], n->gzh, n->gzl,
                         P, n->lw - l, n->c(l));
        }
        NS_TRY(conv_bwd(n, enc_id(l, 1), n->act[enc_id(l, 0)], n->c(l), INPUT_PLANES, n->act[enc_id(l, 0)], l, B));
        const bf16* in = (l == 0) ? n->x : n->pool[l - 1];
        NS_TRY(conv_bwd(n, enc_id(l, 0), in, l == 0 ? n->ldx : n->c(l - 1), l == 0 ? INPUT_NONE : INPUT_F32, nullptr, l,
                        B));
    }
    NS_CUDA(cudaStreamSynchronize(n->stream));
    double s = 0.0;
    for (int b = 0; b < kRedBlocksU; ++b) s += n->partial_host[b];
    *loss = s / (double)P0;
    return NSSTAB_OK;
}

int check_batch(nsstab_unet* n, int B, const void* a, const void* b) {
    if (!n || !a || !b) {
        set_error("unet: null argument");
        return NSSTAB_ERR_INVALID_ARG;
    }
    if (B < 1 || B > n->maxB) {
        set_error("unet: batch must be in [1, max_batch]");
        return NSSTAB_ERR_INVALID_ARG;
    }
    return NSSTAB_OK;
}

}  // namespace

extern "C" {

long unet_param_count(int in_ch, int width) {
    if (in_ch < 1 || width < 1) return -1;
    long c = 0;
    make_layout(in_ch, width, &c);
    return c;
}

int unet_create(int in_ch, int width, int ny, int nx, int max_batch, void* stream, nsstab_unet** out) {
    if (!out) {
        set_error("unet_create: null argument");
        return NSSTAB_ERR_INVALID_ARG;
    }
    *out = nullptr;
    const int q = 1 << (kLevels - 1);
    if (in_ch < 1 || in_ch > 64 || width < 1 || width > 256 || max_batch < 1 || ny < q || nx < q ||
        !is_pow2(ny) || !is_pow2(nx) || (long)ny * nx * max_batch > (1L << 28)) {
        set_error("unet_create: need 1 <= in_ch <= 64, 1 <= width <= 256, max_batch >= 1, ny and nx powers of two "
                  ">= 8, max_batch*ny*nx <= 2^28");
        return NSSTAB_ERR_INVALID_ARG;
    }
    bool attr_ok = halo_attrs<false, true>() == cudaSuccess && halo_attrs<false, false>() == cudaSuccess &&
                   halo_attrs<true, true>() == cudaSuccess &&
                   cudaFuncSetAttribute(k_conv_bwd_w_halo, cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024) ==
                       cudaSuccess;
    for (int va = 0; va < 2; ++va)
        for (int vb = 0; vb < 2; ++vb) {
            attr_ok = attr_ok &&
                      cudaFuncSetAttribute(pick_wgrad(va, vb), cudaFuncAttributeMaxDynamicSharedMemorySize,
                                           wg_smem()) == cudaSuccess &&
                      cudaFuncSetAttribute(pick_gemm<true>(va, vb), cudaFuncAttributeMaxDynamicSharedMemorySize,
                                           conv_gemm_smem<true>()) == cudaSuccess;
        }
    if (!attr_ok) {
        set_error("unet_create: cudaFuncSetAttribute failed");
        return NSSTAB_ERR_CUDA;
    }
    nsstab_unet* n = new nsstab_unet();
    n->in_ch = in_ch;
    n->ldx = (in_ch + 7) / 8 * 8;
    n->width = width;
    n->H = ny;
    n->W = nx;
    n->lh = ilog2(ny);
    n->lw = ilog2(nx);
    n->maxB = max_batch;
    n->stream = (cudaStream_t)stream;
    n->conv = make_layout(in_ch, width, &n->count);
    for (const ConvDesc& d : n->conv)
        if (d.k == 3) {
            n->map.off[n->map.n] = d.w_off;
            n->map.ci[n->map.n] = d.ci;
            n->map.co[n->map.n] = d.co;
            ++n->map.n;
        }
    const long B = max_batch;
    int rc = NSSTAB_OK;
    auto A = [&](int r) {
        if (rc == NSSTAB_OK) rc = r;
    };
    A(n->alloc(&n->theta, n->count));
    A(n->alloc(&n->grad, n->count));
    A(n->alloc(&n->m, n->count));
    A(n->alloc(&n->v, n->count));
    A(n->alloc(&n->wt, n->count));
    A(n->alloc(&n->x, B * ny * nx * n->ldx));
    for (int l = 0; l < kLevels; ++l) {
        const long P = B * n->h(l) * n->w(l);
        A(n->alloc(&n->act[enc_id(l, 0)], P * n->c(l)));
        A(n->alloc(&n->act[enc_id(l, 1)], P * n->c(l)));
        if (l < kLevels - 1) {
            A(n->alloc(&n->act[dec_id(l, 0)], P * n->c(l)));
            A(n->alloc(&n->act[dec_id(l, 1)], P * n->c(l)));
            A(n->alloc(&n->pool[l], B * n->h(l + 1) * n->w(l + 1) * n->c(l)));
            if (!cat_in_place(n, l)) A(n->alloc(&n->cat[l], P * (n->c(l + 1) + n->c(l))));
            A(n->alloc(&n->gskip[l], P * n->c(l)));
        }
    }
    long gmax = 0;
    for (int l = 0; l < kLevels; ++l) {
        const long P = B * n->h(l) * n->w(l);
        gmax = std::max(gmax, P * (n->c(l) + (l + 1 < kLevels ? n->c(l + 1) : 0)));
        gmax = std::max(gmax, P * (long)(l == 0 ? std::max(in_ch, n->c(0)) : n->c(l - 1)));
    }
    A(n->alloc(&n->gzh, gmax));
    A(n->alloc(&n->gzl, gmax));
    A(n->alloc(&n->gnh, gmax));
    A(n->alloc(&n->gnl, gmax));
    A(n->alloc(&n->g0, gmax));
    A(n->alloc(&n->y, B * ny * nx));
    A(n->alloc(&n->gy, B * ny * nx));
    A(n->alloc(&n->partial, kRedBlocksU));
    if (rc == NSSTAB_OK && cudaMallocHost((void**)&n->partial_host, kRedBlocksU * sizeof(double)) != cudaSuccess) {
        set_error("unet_create: cudaMallocHost failed");
        rc = NSSTAB_ERR_OUT_OF_MEMORY;
    }
    for (void* z : {(void*)n->theta, (void*)n->m, (void*)n->v})
        if (rc == NSSTAB_OK && cudaMemsetAsync(z, 0, n->count * sizeof(float), n->stream) != cudaSuccess)
            rc = NSSTAB_ERR_CUDA;
    if (rc == NSSTAB_OK && cudaMemsetAsync(n->wt, 0, n->count * sizeof(bf16), n->stream) != cudaSuccess)
        rc = NSSTAB_ERR_CUDA;
    if (rc != NSSTAB_OK) {
        delete n;
        return rc;
    }
    *out = n;
    return NSSTAB_OK;
}

void unet_destroy(nsstab_unet* net) { delete net; }

int unet_set_params(nsstab_unet* net, const float* theta) {
    if (!net || !theta) {
        set_error("unet_set_params: null argument");
        return NSSTAB_ERR_INVALID_ARG;
    }
    NS_CUDA(cudaMemcpyAsync(net->theta, theta, net->count * sizeof(float), cudaMemcpyDeviceToDevice, net->stream));
    NS_CUDA(cudaMemsetAsync(net->m, 0, net->count * sizeof(float), net->stream));
    NS_CUDA(cudaMemsetAsync(net->v, 0, net->count * sizeof(float), net->stream));
    net->step = 0;
    k_to_bf16<<<grid_for(net->count, 256), 256, 0, net->stream>>>(net->theta, net->wt, net->map, net->count);
    NS_LAUNCH_CHECK();
    return NSSTAB_OK;
}

int unet_get_params(nsstab_unet* net, float* theta) {
    if (!net || !theta) {
        set_error("unet_get_params: null argument");
        return NSSTAB_ERR_INVALID_ARG;
    }
    NS_CUDA(cudaMemcpyAsync(theta, net->theta, net->count * sizeof(float), cudaMemcpyDeviceToDevice, net->stream));
    return NSSTAB_OK;
}

int unet_forward(nsstab_unet* net, const float* x, int batch, float* y) {
    NS_TRY(check_batch(net, batch, x, y));
    return forward(net, x, batch, y);
}

int unet_gradient(nsstab_unet* net, const float* x, const float* target, int batch, float* grad, double* loss) {
    NS_TRY(check_batch(net, batch, x, target));
    if (!grad || !loss) {
        set_error("unet_gradient: null argument");
        return NSSTAB_ERR_INVALID_ARG;
    }
    NS_TRY(forward(net, x, batch, net->y));
    NS_TRY(backward(net, target, batch, loss));
    NS_CUDA(cudaMemcpyAsync(grad, net->grad, net->count * sizeof(float), cudaMemcpyDeviceToDevice, net->stream));
    NS_CUDA(cudaStreamSynchronize(net->stream));
    return NSSTAB_OK;
}

int unet_train_step(nsstab_unet* net, const float* x, const float* target, int batch, float lr, float beta1,
                    float beta2, float eps, double* loss) {
    NS_TRY(check_batch(net, batch, x, target));
    if (!loss || !(lr > 0) || !(beta1 >= 0 && beta1 < 1) || !(beta2 >= 0 && beta2 < 1) || !(eps > 0)) {
        set_error("unet_train_step: need loss != NULL, lr > 0, 0 <= beta < 1, eps > 0");
        return NSSTAB_ERR_INVALID_ARG;
    }
    NS_TRY(forward(net, x, batch, net->y));
    NS_TRY(backward(net, target, batch, loss));
    net->step += 1;
    const float c1 = 1.f - std::pow(beta1, (float)net->step), c2 = 1.f - std::pow(beta2, (float)net->step);
    k_adam<<<grid_for(net->count, 256), 256, 0, net->stream>>>(net->theta, net->grad, net->m, net->v, net->wt, net->map,
                                                               net->count, lr, beta1, beta2, eps, c1, c2);
    NS_LAUNCH_CHECK();
    return NSSTAB_OK;
}

}  // extern "C"
